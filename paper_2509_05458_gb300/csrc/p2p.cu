// Near field (List 1, step 3 of Sec. 6.4) and the direct sum (Sec. 2.3,
// Eq. evaluation_problem) for 2D/3D Laplace and Helmholtz, single and double
// layer, in float64 / complex128 or in mixed precision (complex64 kernel
// arithmetic, FP32 hi/lo pair differences, compensated sums).
//
// Mixed precision: one CTA per target leaf, 128 threads = 32 targets x 4 source
// lanes; the sources of each List-1 leaf are staged through shared memory in
// chunks; the 4 partial sums of a target are combined in a fixed order, so
// results are bitwise reproducible. FP64: see k_near.
#include <algorithm>
#include <cmath>
#include <cstddef>

#include "kernels.cuh"
#include "pair64.cuh"

namespace cfmm {

// ---------------------------------------------------------------------------
// Ascending series of H_0^(1), H_1^(1) in w = -(kappa r)^2/4 (DLMF 10.2.2,
// 10.8.1), evaluated by Horner's rule with precomputed coefficients:
//   A(w) = sum w^k/(k!)^2                   J_0 = A
//   B(w) = sum w^k/(k!(k+1)!)               J_1 = (z/2) B
//   C(w) = sum_{k>=1} H_k w^k/(k!)^2        Y_0 = (2/pi)((log(z/2)+gamma) A - C)
//   D(w) = sum (psi(k+1)+psi(k+2)) w^k/(k!(k+1)!)
//                                           Y_1 = -2/(pi z) + (2/pi) log(z/2) J_1 - (z/(2pi)) D
// with H_k the harmonic numbers and psi(k+1) = -gamma + H_k. Only r^2 enters:
// log(z/2) = Log(q)/2 with q = (kappa r/2)^2, and the double layer needs
// kappa J_1/r = (kappa^2/2) B and kappa Y_1/r = -2/(pi r^2) + (kappa^2/pi) log(z/2) B
// - (kappa^2/(2 pi)) D, so the near field takes no square root.
// ---------------------------------------------------------------------------
constexpr int kSerMax = 21;
struct SeriesTab {
    double a[kSerMax + 1], b[kSerMax + 1], c[kSerMax + 1], d[kSerMax + 1];
    float af[kSerMax + 1], bf[kSerMax + 1], cf_[kSerMax + 1], df[kSerMax + 1];
};
static __constant__ SeriesTab c_ser;

static SeriesTab make_series_tab() {
    SeriesTab T;
    const double g = 0.57721566490153286061;
    double fk = 1.0, H = 0.0;   // k!, H_k
    for (int k = 0; k <= kSerMax; ++k) {
        if (k > 0) {
            fk *= k;
            H += 1.0 / k;
        }
        double fk1 = fk * (k + 1);
        T.a[k] = 1.0 / (fk * fk);
        T.b[k] = 1.0 / (fk * fk1);
        T.c[k] = H / (fk * fk);
        T.d[k] = (-2.0 * g + 2.0 * H + 1.0 / (k + 1)) / (fk * fk1);
        T.af[k] = (float)T.a[k];
        T.bf[k] = (float)T.b[k];
        T.cf_[k] = (float)T.c[k];
        T.df[k] = (float)T.d[k];
    }
    return T;
}

static __device__ PairTab d_pair;

void make_pair_tab(PairTab* T) {
    const double kPi = 3.14159265358979323846;
    for (int k = 0; k < kAngTab; ++k) {
        // the first octant's values, so that the symmetric entries agree
        int q = k / (kAngTab / 4), r = k % (kAngTab / 4);
        double c = r > kAngTab / 8 ? std::sin(2 * kPi * (kAngTab / 4 - r) / kAngTab) : std::cos(2 * kPi * r / kAngTab);
        double s = r > kAngTab / 8 ? std::cos(2 * kPi * (kAngTab / 4 - r) / kAngTab) : std::sin(2 * kPi * r / kAngTab);
        T->ang[k] = q == 0 ? make_double2(c, s) : q == 1 ? make_double2(-s, c) : q == 2 ? make_double2(-c, -s)
                                                                                       : make_double2(s, -c);
    }
    for (int k = 0; k < kExpTab; ++k) T->ex[k] = std::exp2((double)k / kExpTab);
    for (int j = 0; j < kLogRad; ++j) {
        double c = std::ldexp(std::rint(std::ldexp(1.0 / (1.0 + (j + 0.5) / kLogRad), 20)), -20);
        T->lrad[j] = make_double2(c, -std::log(c));
    }
    for (int k = 0; k < kLogAng; ++k) {
        double th = 2 * kPi * (k <= kLogAng / 2 ? k : k - kLogAng) / kLogAng;
        double c = std::ldexp(std::rint(std::ldexp(std::cos(th), 27)), -27);
        double s = std::ldexp(std::rint(std::ldexp(-std::sin(th), 27)), -27);
        T->ldir[k] = make_double2(c, s);
        // |dir|^2 - 1 is exact in FP64 (54 bits after the leading ones cancel)
        T->llog[k] = make_double2(-0.5 * std::log1p(std::fma(c, c, std::fma(s, s, -1.0))),
                                  k == kLogAng / 2 ? kPi : -std::atan2(s, c));
    }
}

const PairTab* pair_tab_device() {
    void* d = nullptr;
    CFMM_CUDA(cudaGetSymbolAddress(&d, d_pair));
    return static_cast<const PairTab*>(d);
}

Wave make_wave(double k) {
    if (!(k > 0.0)) return Wave{0.0, 0.0, 0.0, 0.0, 0.0};
    return Wave{k, 1.0 / k, std::sqrt(1.0 / k), k * 40.74366543152521, k * 369.3299304675746};   // 256/(2 pi), 256/log 2
}

void upload_lag_rule_p2p() {
    upload_lag_rule_local();
    SeriesTab T = make_series_tab();
    CFMM_CUDA(cudaMemcpyToSymbol(c_ser, &T, sizeof(T)));
    std::vector<char> buf(offsetof(PairTab, hk));
    PairTab* d = nullptr;
    CFMM_CUDA(cudaGetSymbolAddress((void**)&d, d_pair));
    make_pair_tab(reinterpret_cast<PairTab*>(buf.data()));
    CFMM_CUDA(cudaMemcpy(d, buf.data(), buf.size(), cudaMemcpyHostToDevice));
    k_pair_hankel<<<(2 * kHkGrids * kHkNx * kHkNy + 127) / 128, 128>>>(d);
    CFMM_LAUNCHED();
    CFMM_CUDA(cudaDeviceSynchronize());
}

// number of series terms for |q|^2 = aq, FP64 (truncation below 1e-18)
__device__ __forceinline__ int series_terms64(double aq) {
    return aq <= 0.0625 ? 8 : aq <= 1.0 ? 11 : aq <= 5.0625 ? 14 : aq <= 16.0 ? 16 : 21;
}
// FP32 (truncation below 1e-9)
__device__ __forceinline__ int series_terms32(float aq) {
    return aq <= 0.0625f ? 5 : aq <= 1.0f ? 7 : aq <= 5.0625f ? 9 : aq <= 16.0f ? 10 : 14;
}

// The general FP64 2D Helmholtz pair: ascending series up to |z| = 6, the
// quadrature of hankel01 beyond
static __device__ __noinline__ void helm2d_pair64_general(cd r2, double kappa, bool dlp, cd& h0, cd& g1) {
    const double kPi = 3.14159265358979323846, kG = 0.57721566490153286061;
    double k2 = kappa * kappa;
    cd q = (0.25 * k2) * r2;
    double aq = cabs2(q);
    if (aq <= 81.0) {
        cd w = -q;
        int K = series_terms64(aq);
        cd A = {c_ser.a[K], 0}, Bs = {c_ser.b[K], 0}, Cs = {c_ser.c[K], 0}, Ds = {c_ser.d[K], 0};
        for (int k = K - 1; k >= 0; --k) {
            A = A * w + cd{c_ser.a[k], 0};
            Cs = Cs * w + cd{c_ser.c[k], 0};
            if (dlp) {
                Bs = Bs * w + cd{c_ser.b[k], 0};
                Ds = Ds * w + cd{c_ser.d[k], 0};
            }
        }
        cd L = {0.25 * log(aq), 0.5 * atan2(q.y, q.x)};    // log(z/2)
        h0 = A + mul_i((2.0 / kPi) * ((L + cd{kG, 0}) * A - Cs));
        if (dlp) {
            cd ir2 = cinv(r2);
            cd y = (-2.0 / kPi) * ir2 + (k2 / kPi) * (L * Bs) - (k2 / (2.0 * kPi)) * Ds;
            g1 = (0.5 * k2) * Bs + mul_i(y);
        }
        return;
    }
    cd r = csqrt_p(r2);
    cd h1;
    hankel01(kappa * r, &h0, &h1);
    g1 = (kappa * h1) * cinv(r);
}

// sum of c[k] w^k, k <= N, real c, by the two-term recurrence in 2 Re w = s and
// |w|^2 = v (two FP64 instructions a term instead of four)
template <int N>
__device__ __forceinline__ cd real_poly(const double* c, cd w, double s, double v) {
    double b1 = fma(s, c[N], c[N - 1]), b2 = c[N];
#pragma unroll
    for (int k = N - 2; k >= 1; --k) {
        double b = fma(-v, b2, fma(s, b1, c[k]));
        b2 = b1;
        b1 = b;
    }
    return cd{fma(-v, b2, fma(w.x, b1, c[0])), w.y * b1};
}

// H_0 and kappa H_1 / r by N terms of the series, q = (kappa r/2)^2
template <int N>
__device__ __forceinline__ void helm2d_series(cd r2, cd q, double aq, double k2, bool slp, bool dlp, cd& h0, cd& g1) {
    const double kPi = 3.14159265358979323846, kG = 0.57721566490153286061;
    cd w = -q;
    double s = w.x + w.x;
    cd L = 0.5 * clog64(&d_pair, q);
    if (slp) {
        cd A = real_poly<N>(c_ser.a, w, s, aq), Cs = real_poly<N>(c_ser.c, w, s, aq);
        cd t = cmac(-Cs, cd{L.x + kG, L.y}, A);
        h0 = cd{fma(-2.0 / kPi, t.y, A.x), fma(2.0 / kPi, t.x, A.y)};
    }
    if (dlp) {
        cd Bs = real_poly<N>(c_ser.b, w, s, aq), Ds = real_poly<N>(c_ser.d, w, s, aq);
        cd t = (k2 / kPi) * (L * Bs) - (2.0 / kPi) * crcp64(r2) - (k2 / (2.0 * kPi)) * Ds;
        g1 = (0.5 * k2) * Bs + mul_i(t);
    }
}

// FP64 2D Helmholtz pair: SLP factor H_0 and DLP factor kappa H_1 / r. The series
// close to z = 0, the Taylor cells of hankel_factor beyond, outside the cells'
// sector the general evaluation. The first two cost 140 (8 terms) to 190 FP64
// instructions a combined-field pair, the general one about 670 at |z| = 3 and
// 6000 beyond 6. A warp whose lanes fall on both sides of a limit pays for both,
// and a leaf's near field spans |z| up to 2 or so in most plans; so a converged
// warp (WARP) takes the series as a whole while every lane has |z| <= 2 (11
// terms), and cells for |z| > 1/2 otherwise.
template <bool WARP>
__device__ __forceinline__ void helm2d_pair64(cd r2, const Wave& k, bool slp, bool dlp, cd& h0, cd& g1) {
    double k2 = k.k * k.k;
    cd q = (0.25 * k2) * r2;
    double aq = cabs2(q);
    if (WARP) {
        // (comparisons on the high words: an FP64 compare costs an FP64 slot)
        const int ha = __double2hiint(aq);
        if (__all_sync(0xffffffffu, ha < 0x3fb00000)) {      // aq < 1/16
            helm2d_series<8>(r2, q, aq, k2, slp, dlp, h0, g1);
            return;
        }
        if (__all_sync(0xffffffffu, ha < 0x3ff00000)) {      // aq < 1
            helm2d_series<11>(r2, q, aq, k2, slp, dlp, h0, g1);
            return;
        }
    }
    cd y = crsqrt64(r2), ds;
    int cell = hankel_cell(k.ik * y, ds);
    if (cell >= 0) {
        cd r;
        cd e = wave64(&d_pair, k, r2, y, r);
        e = e * (k.isk * crsqrt64(r));
        if (slp) h0 = e * hankel_factor(d_pair.hk[cell][0], ds);
        if (dlp) g1 = (e * hankel_factor(d_pair.hk[cell][1], ds)) * (k.k * y);
    } else if (aq <= 0.0625) {
        helm2d_series<8>(r2, q, aq, k2, slp, dlp, h0, g1);
    } else {
        helm2d_pair64_general(r2, k.k, dlp, h0, g1);
    }
}

constexpr int kP2PThreads = 128;
constexpr int kP2PTargets = 32;
constexpr int kP2PSplit = kP2PThreads / kP2PTargets;
constexpr int kP2PChunk = 128;

// r^2 = sum d_a^2 of the complex differences (3 DIM + 1 FP64 instructions). Its imaginary
// part starts from +0: a sum of zero products is +0, the upper side of the branch cut
template <int DIM>
__device__ __forceinline__ cd pair_r2(const double* dr, const double* di) {
    double x = dr[0] * dr[0], y = fma(dr[0], di[0], 0.0);
    x = fma(-di[0], di[0], x);
#pragma unroll
    for (int a = 1; a < DIM; ++a) {
        x = fma(-di[a], di[a], fma(dr[a], dr[a], x));
        y = fma(dr[a], di[a], y);
    }
    return cd{x, y + y};
}

// K(x, y) sigma + (n . grad_y K)(x, y) tau for one pair (d = x - y != 0)
template <int DIM, int KER>
__device__ __forceinline__ void pair_kernel(const double* dr, const double* di, const double* nr,
                                            const double* ni, cd sg, cd ta, bool slp, bool dlp,
                                            const Wave& k, cd& acc) {
    const double kappa = k.k;
    cd d[DIM];
    cd r2 = pair_r2<DIM>(dr, di);
#pragma unroll
    for (int a = 0; a < DIM; ++a) d[a] = cd{dr[a], di[a]};
    cd nd = {0.0, 0.0};
    if (dlp) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) nd = cmac(nd, cd{nr[a], ni[a]}, d[a]);
    }
    if (DIM == 2 && KER == CFMM_LAPLACE) {
        // log r = Log(r^2)/2 ; grad_y log r = (y - x)/r^2
        if (slp) acc = cmac(acc, 0.5 * clog64(&d_pair, r2), sg);
        if (dlp) acc = cmac(acc, -nd * crcp64(r2), ta);
    } else if (DIM == 2) {
        cd h0, g1;
        helm2d_pair64<true>(r2, k, slp, dlp, h0, g1);
        if (slp) acc = cmac(acc, h0, sg);
        if (dlp) acc = cmac(acc, g1 * nd, ta);
    } else if (KER == CFMM_LAPLACE) {
        cd ir = crsqrt64(r2);
        if (slp) acc = cmac(acc, ir, sg);
        if (dlp) acc = cmac(acc, nd * (ir * (ir * ir)), ta);
    } else {
        cd ir = crsqrt64(r2);
        cd r;
        cd g = wave64(&d_pair, k, r2, ir, r) * ir;
        if (slp) acc = cmac(acc, g, sg);
        if (dlp) acc = cmac(acc, (nd * cd{fma(kappa, r.y, 1.0), -kappa * r.x}) * (g * (ir * ir)), ta);
    }
}

// grad_x of K(x, y) sg + (n . grad_y K)(x, y) ta for one pair (d = x - y != 0),
// added to g[0..DIM-1] (Sec. 2.1: S' and D' are its normal components). With
// K = K(r): grad_x K = (K'/r) d and grad_x (n . grad_y K) = -(K'/r) n -
// ((K'' - K'/r)/r^2) (n.d) d.
template <int DIM, int KER>
__device__ __forceinline__ void pair_grad(const double* dr, const double* di, const double* nr, const double* ni,
                                          cd sg, cd ta, bool slp, bool dlp, const Wave& k, cd* g) {
    const double kappa = k.k;
    cd d[DIM];
    cd r2 = pair_r2<DIM>(dr, di);
#pragma unroll
    for (int a = 0; a < DIM; ++a) d[a] = cd{dr[a], di[a]};
    cd a1, a2;   // K'/r and (K'' - K'/r)/r^2
    if (DIM == 2 && KER == CFMM_LAPLACE) {
        cd ir2 = crcp64(r2);
        a1 = ir2;
        a2 = -2.0 * (ir2 * ir2);
    } else if (DIM == 2) {
        cd h0, g1;                      // H_0, kappa H_1 / r
        helm2d_pair64<true>(r2, k, true, true, h0, g1);
        a1 = -g1;
        a2 = (2.0 * g1 - (kappa * kappa) * h0) * crcp64(r2);
    } else if (KER == CFMM_LAPLACE) {
        cd ir = crsqrt64(r2), ir2 = ir * ir;
        cd ir3 = ir * ir2;
        a1 = -ir3;
        a2 = 3.0 * (ir3 * ir2);
    } else {
        cd ir = crsqrt64(r2), ir2 = ir * ir;
        cd r;
        cd e = wave64(&d_pair, k, r2, ir, r);
        cd ikr = mul_i(kappa * r);
        cd ir3 = ir * ir2;
        a1 = (e * (ikr - cd{1.0, 0.0})) * ir3;
        a2 = (e * (cd{3.0, 0.0} - 3.0 * ikr - (kappa * kappa) * r2)) * (ir3 * ir2);
    }
    cd cs = slp ? a1 * sg : cd{0, 0};
    cd cn = {0, 0}, cdd = {0, 0};
    if (dlp) {
        cd nd = {0.0, 0.0};
#pragma unroll
        for (int a = 0; a < DIM; ++a) nd += cd{nr[a], ni[a]} * d[a];
        cn = -(a1 * ta);
        cdd = -(a2 * (nd * ta));
    }
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        cd v = (cs + cdd) * d[a];
        if (dlp) v += cn * cd{nr[a], ni[a]};
        g[a] += v;
    }
}

// ---------------------------------------------------------------------------
// FP64 near field, its gradient and the direct sum.
//
// The FP64 pipe bounds them (pair64.cuh), so what counts is that every lane of
// an FP64 instruction holds a pair. Lanes therefore stand for sources, 32 of the
// concatenated source leaves at a time, which leaves a partial warp only at the
// end of a list; with lanes as targets of one leaf, 25 of 32 were in use (leaf
// size 128). A lane keeps its source in registers and meets the block's nt
// targets in turn, target (lane + k) mod nt at step k, so the lanes of a step add
// to different entries of the warp's accumulator row in shared memory (for nt <
// 32 the lanes beyond nt use further copies of the row). Each warp takes every
// fourth 32-source group; rows and copies are added in a fixed order at the end,
// so results are bitwise reproducible.
//
// A block takes at most kNearTargets targets of a leaf; the launch lowers that
// until the grid covers the chip, which a few dozen leaves with all their targets
// in one block each do not.
// ---------------------------------------------------------------------------
constexpr int kNearThreads = 128;
constexpr int kNearWarps = kNearThreads / 32;
constexpr int kNearTargets = 128;     // targets of a block at most
constexpr int kNearSeg = kNearThreads;   // source leaves whose ranges are staged at once

// targets and sources of a launch: index ranges per box into the sorted points,
// or a single range each (direct sum: boxes == nullptr)
struct NearLists {
    const int* boxes;
    SubRange src, trg;
    const int* l1off;
    const int* l1;
};

template <int DIM, int KER, bool GRAD>
__global__ void __launch_bounds__(kNearThreads) k_near(KParams K, NearLists L, int tb, cd* __restrict__ out) {
    constexpr int NA = GRAD ? DIM : 1;                  // complex accumulators of a target
    constexpr int kRow = kNearTargets + 32;             // nt, or copies * nt < nt + 32
    extern __shared__ double near_sm[];
    double* tx = near_sm;                               // [2 DIM][kNearTargets]
    cd* acc = reinterpret_cast<cd*>(tx + 2 * DIM * kNearTargets);   // [warps][NA][kRow]
    __shared__ int seg_pos[kNearSeg], seg_end[kNearSeg], warp_sum[kNearWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int rhs = blockIdx.y;
    const int b = L.boxes ? L.boxes[blockIdx.x] : 0;
    const Wave wave{K.kappa, K.ikappa, K.isqrt_kappa, K.kappa_ang, K.kappa_exp};
    const int qa = L.boxes ? L.l1off[b] : 0, qb = L.boxes ? L.l1off[b + 1] : 1;
    // groups of targets blockIdx.z, + gridDim.z, ..: the grid covers leaf_size
    // points a leaf; leaves at the deepest level may hold more
    const int64_t tstep = (int64_t)(L.boxes ? gridDim.z : gridDim.x) * tb, tend = L.boxes ? L.trg.en[b] : K.n_trg;
    for (int64_t t0 = L.boxes ? L.trg.st[b] + (int64_t)blockIdx.z * tb : (int64_t)blockIdx.x * tb; t0 < tend; t0 += tstep) {
    const int nt = (int)min((int64_t)tb, tend - t0);
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += kNearThreads) {
        const int64_t g = L.trg.at(t0 + i);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            tx[a * kNearTargets + i] = K.trg_re[a * K.n_trg + g];
            tx[(DIM + a) * kNearTargets + i] = K.trg_im[a * K.n_trg + g];
        }
    }
    const int copies = nt >= 32 ? 1 : (31 + nt) / nt;
    cd* row = acc + wid * NA * kRow;
    for (int i = lane; i < NA * kRow; i += 32) row[i] = cd{0.0, 0.0};
    row += (lane / nt) * (nt >= 32 ? 0 : nt);
    const int first = lane % nt;
    for (int q0 = qa; q0 < qb; q0 += kNearSeg) {
        // ranges of the next source leaves and the running total of their sizes
        int q = q0 + threadIdx.x, s0 = 0, cnt = 0;
        if (q < qb) {
            int src = L.boxes ? L.l1[q] : 0;
            s0 = L.boxes ? L.src.st[src] : 0;
            cnt = L.boxes ? L.src.en[src] - s0 : (int)K.n_src;
        }
        int sum = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, sum, o);
            if (lane >= o) sum += v;
        }
        __syncthreads();                                // the last round's ranges have been read
        if (lane == 31) warp_sum[wid] = sum;
        __syncthreads();
        for (int w = 0; w < wid; ++w) sum += warp_sum[w];
        seg_pos[threadIdx.x] = s0;
        seg_end[threadIdx.x] = sum;
        __syncthreads();
        const unsigned total = (unsigned)seg_end[kNearSeg - 1];
        for (unsigned c0 = wid * 32; c0 < total; c0 += kNearThreads) {
            const unsigned f = c0 + lane;
            const bool valid = f < total;
            double yr[DIM], yi[DIM], nr[DIM], ni[DIM];
            cd sg = {0.0, 0.0}, ta = {0.0, 0.0};
            if (valid) {
                int lo = 0, hi = kNearSeg - 1;          // first range that ends beyond f
                while (lo < hi) {
                    int m = (lo + hi) >> 1;
                    if ((unsigned)seg_end[m] > f) hi = m;
                    else lo = m + 1;
                }
                const int64_t j = L.src.at(seg_pos[lo] + (int)(f - (lo ? seg_end[lo - 1] : 0))), n = K.n_src;
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    yr[a] = K.src_re[a * n + j];
                    yi[a] = K.src_im[a * n + j];
                    nr[a] = K.dlp ? K.nrm_re[a * n + j] : 0.0;
                    ni[a] = K.dlp ? K.nrm_im[a * n + j] : 0.0;
                }
                if (K.slp) sg = K.sigma[(int64_t)rhs * K.dens_stride + j];
                if (K.dlp) ta = K.tau[(int64_t)rhs * K.dens_stride + j];
            }
            int t = first;
            for (int k = 0; k < nt; ++k) {
                __syncwarp();                           // the neighbour lane's sum of the last step
                // lanes without a source and pairs with x == y (self pair, coincident
                // point) take a harmless distance and store nothing: the warp stays whole
                double dr[DIM], di[DIM];
                int hi = 0, lo = 0;                     // the differences' bits (FP64 compares cost an FP64 slot)
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    dr[a] = tx[a * kNearTargets + t] - yr[a];
                    di[a] = tx[(DIM + a) * kNearTargets + t] - yi[a];
                    hi |= __double2hiint(dr[a]) | __double2hiint(di[a]);
                    lo |= __double2loint(dr[a]) | __double2loint(di[a]);
                }
                // (the difference of -0 and +0 is -0)
                const bool skip = !valid || ((hi & 0x7fffffff) | lo) == 0;
                if (skip) {
                    dr[0] = wave.k > 0.0 ? wave.ik : 1.0;
                    di[0] = 0.0;
#pragma unroll
                    for (int a = 1; a < DIM; ++a) dr[a] = di[a] = 0.0;
                }
                if (GRAD) {
                    cd g[DIM];
#pragma unroll
                    for (int a = 0; a < DIM; ++a) g[a] = row[a * kRow + t];
                    pair_grad<DIM, KER>(dr, di, nr, ni, sg, ta, K.slp, K.dlp, wave, g);
#pragma unroll
                    for (int a = 0; a < DIM; ++a)
                        if (!skip) row[a * kRow + t] = g[a];
                } else {
                    cd u = row[t];
                    pair_kernel<DIM, KER>(dr, di, nr, ni, sg, ta, K.slp, K.dlp, wave, u);
                    if (!skip) row[t] = u;
                }
                if (++t == nt) t = 0;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nt * NA; i += kNearThreads) {
        int a = i / nt, t = i - a * nt;
        cd s = {0.0, 0.0};
        for (int w = 0; w < kNearWarps; ++w)
            for (int c = 0; c < copies; ++c) s += acc[(w * NA + a) * kRow + c * nt + t];
        out[((int64_t)rhs * NA + a) * K.n_trg + L.trg.at(t0 + t)] = s;
    }
    }
}

template <int DIM, bool GRAD>
constexpr size_t near_smem() {
    return sizeof(double) * 2 * DIM * kNearTargets +
           sizeof(cd) * kNearWarps * (GRAD ? DIM : 1) * (kNearTargets + 32);
}

template <int DIM, int KER>
__device__ void finish_target(cd acc, cd* red, int tl, int split, bool tvalid, cd* out) {
    red[split * kP2PTargets + tl] = acc;
    __syncthreads();
    if (split == 0 && tvalid) {
        cd s = red[tl];
        for (int q = 1; q < kP2PSplit; ++q) s += red[q * kP2PTargets + tl];
        *out = s;
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Mixed precision (complex64 kernel arithmetic, compensated FP32 sums).
// Coordinates enter as FP64 offsets from a reference point of the target
// block (the first target), split into FP32 hi + lo parts; the pair
// difference (x_h - y_h) + (x_l - y_l) keeps FP32 relative accuracy even for
// near-coincident pairs (Sterbenz: x_h - y_h is exact when x_h, y_h are
// close). Sums over sources use compensated (Kahan) FP32 accumulation; the
// few partial sums of a target are combined in FP64.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void helm2d_pair32(cf r2, float kappa, bool dlp, cf& h0, cf& g1) {
    const float kPi = 3.14159265f, kG = 0.5772156649f;
    float k2 = kappa * kappa;
    cf q = (0.25f * k2) * r2;
    float aq = q.x * q.x + q.y * q.y;
    cf w = cf{-q.x, -q.y};
    int K = series_terms32(aq);
    cf A = {c_ser.af[K], 0.f}, Bs = {c_ser.bf[K], 0.f}, Cs = {c_ser.cf_[K], 0.f}, Ds = {c_ser.df[K], 0.f};
    for (int k = K - 1; k >= 0; --k) {
        A = A * w + cf{c_ser.af[k], 0.f};
        Cs = Cs * w + cf{c_ser.cf_[k], 0.f};
        if (dlp) {
            Bs = Bs * w + cf{c_ser.bf[k], 0.f};
            Ds = Ds * w + cf{c_ser.df[k], 0.f};
        }
    }
    cf L = {0.25f * logf(aq), 0.5f * atan2f(q.y, q.x)};
    cf lg = L + cf{kG, 0.f};
    h0 = A + mul_if((2.f / kPi) * (lg * A - Cs));
    if (dlp) {
        cf ir2 = cinvf(r2);
        cf y = (-2.f / kPi) * ir2 + (k2 / kPi) * (L * Bs) - (k2 / (2.f * kPi)) * Ds;
        g1 = (0.5f * k2) * Bs + mul_if(y);
    }
}

// FP32 rounding of the general FP64 evaluation, which the mixed near field is
// defined by. The quick evaluation is within 2^-42 (1 + |kappa r|/64) of it
// relative to the modulus (both are good to 2^-44 or better at |kappa r| of
// order 1 and their phases to 2^-52 |kappa r|), so both round alike except where
// a bound of that interval rounds differently: about one pair in 30,000, which
// takes the general evaluation.
__device__ __forceinline__ bool round32(cd v, double rel, cf& out) {
    double d = rel * (fabs(v.x) + fabs(v.y));
    out = cf{(float)(v.x - d), (float)(v.y - d)};
    return out.x == (float)(v.x + d) && out.y == (float)(v.y + d);
}
__device__ __forceinline__ void helm2d_round32(cd r2, const Wave& k, bool slp, bool dlp, cf& h0f, cf& g1f) {
    cd h0, g1;
    helm2d_pair64<false>(r2, k, slp, dlp, h0, g1);
    double rel = 2.2737367544323206e-13 * (1.0 + 0.015625 * k.k * sqrt(fabs(r2.x) + fabs(r2.y)));
    bool same = true;
    if (slp) same = round32(h0, rel, h0f);
    if (dlp) same = round32(g1, rel, g1f) && same;
    if (same) return;
    helm2d_pair64_general(r2, k.k, dlp, h0, g1);
    if (slp) h0f = cf{(float)h0.x, (float)h0.y};
    if (dlp) g1f = cf{(float)g1.x, (float)g1.y};
}

// Error-free transformations (Dekker, Knuth): the product and sum of two
// floats as an unevaluated hi + lo pair.
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = a * b;
    e = fmaf(a, b, -p);
}
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
// (h1 + l1) * (h2 + l2) added to the double-float accumulator (S, E)
__device__ __forceinline__ void df_fma(float h1, float l1, float h2, float l2, float sgn, float& S, float& E) {
    float p, e, t;
    two_prod(h1, h2, p, e);
    e = fmaf(h1, l2, fmaf(l1, h2, e));
    two_sum(S, sgn * p, S, t);
    E += t + sgn * e;
}

// n . d with the normal and the difference each as FP32 hi + lo: on a smooth
// curve or surface n is nearly orthogonal to d for close pairs, so n . d
// cancels; the double-float evaluation keeps its FP32 relative accuracy.
template <int DIM>
__device__ __forceinline__ cf dot_nd(const float* dh_r, const float* dl_r, const float* dh_i, const float* dl_i,
                                     const float* nh_r, const float* nl_r, const float* nh_i, const float* nl_i) {
    float Sr = 0.f, Er = 0.f, Si = 0.f, Ei = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        df_fma(nh_r[a], nl_r[a], dh_r[a], dl_r[a], 1.f, Sr, Er);
        df_fma(nh_i[a], nl_i[a], dh_i[a], dl_i[a], -1.f, Sr, Er);
        df_fma(nh_r[a], nl_r[a], dh_i[a], dl_i[a], 1.f, Si, Ei);
        df_fma(nh_i[a], nl_i[a], dh_r[a], dl_r[a], 1.f, Si, Ei);
    }
    return cf{Sr + Er, Si + Ei};
}

// The hi/lo parts of a target and a source (offsets from the block's
// reference point), for pairs that need the difference in FP64.
struct PairHL {
    const float *xhr, *xlr, *xhi, *xli;   // target
    const float *yhr, *ylr, *yhi, *yli;   // source
};

// r^2 in FP64 from the hi/lo parts (for |kappa r| beyond the complex64 range:
// the phase kappa*r needs more than FP32 relative accuracy there, and the
// FP32 difference of the hi parts is not exact for distant pairs)
template <int DIM>
__device__ __forceinline__ cd r2_from_hl(const PairHL& H) {
    cd r2 = {0.0, 0.0};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        cd d = {((double)H.xhr[a] - (double)H.yhr[a]) + ((double)H.xlr[a] - (double)H.ylr[a]),
                ((double)H.xhi[a] - (double)H.yhi[a]) + ((double)H.xli[a] - (double)H.yli[a])};
        r2 += d * d;
    }
    return r2;
}

// e^{i kappa r} and r for |kappa r| > 3 in double-float FP32 arithmetic (the
// FP32 phase would lose digits there): d = x - y as hi + lo per component
// (an exact two_sum of the hi parts plus the lo difference), r^2 in
// double-float, r = r0 + (r^2 - r0^2)/(2 r0) (one Newton step from the FP32
// root), kappa r in double-float, the phase reduced by 2 pi before sincosf.
template <int DIM>
__device__ __forceinline__ void far_phase_df(const PairHL& H, float kh, float kl, cf& e_ikr, cf& r) {
    float Sr = 0.f, Er = 0.f, Si = 0.f, Ei = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        float s, t, rh, rl, ih, il;
        two_sum(H.xhr[a], -H.yhr[a], s, t);
        two_sum(s, t + (H.xlr[a] - H.ylr[a]), rh, rl);
        two_sum(H.xhi[a], -H.yhi[a], s, t);
        two_sum(s, t + (H.xli[a] - H.yli[a]), ih, il);
        df_fma(rh, rl, rh, rl, 1.f, Sr, Er);
        df_fma(ih, il, ih, il, -1.f, Sr, Er);
        df_fma(rh, rl, ih, il, 2.f, Si, Ei);
    }
    cf r0 = csqrtf_p(cf{Sr + Er, Si + Ei});
    float Rr = Sr, ERr = Er, Ri = Si, ERi = Ei;
    df_fma(r0.x, 0.f, r0.x, 0.f, -1.f, Rr, ERr);
    df_fma(r0.y, 0.f, r0.y, 0.f, 1.f, Rr, ERr);
    df_fma(r0.x, 0.f, r0.y, 0.f, -2.f, Ri, ERi);
    cf corr = cf{Rr + ERr, Ri + ERi} * cinvf(2.f * r0);
    float th, te, dh, de;
    two_prod(kh, r0.x, th, te);
    te += fmaf(kh, corr.x, kl * r0.x);
    two_prod(kh, r0.y, dh, de);
    de += fmaf(kh, corr.y, kl * r0.y);
    const float kTwoPiH = 6.28318548202514648f;     // float(2 pi)
    const float kTwoPiL = -1.74845553e-07f;         // 2 pi - float(2 pi)
    float k = rintf(th * 0.159154943f);
    float q, qe;
    two_prod(k, kTwoPiH, q, qe);
    float red = (th - q) + ((te - qe) - k * kTwoPiL);
    float sn, cs;
    sincosf(red, &sn, &cs);
    float mag = expf(-dh) * (1.f - de);
    e_ikr = cf{mag * cs, mag * sn};
    r = r0 + corr;
}

template <int DIM, int KER>
__device__ __forceinline__ void pair_kernel32(const float* d_re, const float* d_im, const PairHL& H, cf nd, cf sg,
                                              cf ta, bool slp, bool dlp, float kappa, const Wave& k, Kahan& acc) {
    cf d[DIM];
    cf r2 = {0.f, 0.f};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        d[a] = cf{d_re[a], d_im[a]};
        r2 = r2 + d[a] * d[a];
    }
    cf v = {0.f, 0.f};
    if (DIM == 2 && KER == CFMM_LAPLACE) {
        if (slp) v = cf{0.25f * logf(r2.x * r2.x + r2.y * r2.y), 0.5f * atan2f(r2.y, r2.x)} * sg;
        if (dlp) v = v - (nd * cinvf(r2)) * ta;
    } else if (DIM == 2) {
        float k2 = kappa * kappa;
        cf q = (0.25f * k2) * r2;
        // complex64 series only for |kappa r| <= 3 (|q| <= 2.25), where its
        // terms stay below ~1.3x the result; beyond, the FP64 evaluation
        if (q.x * q.x + q.y * q.y <= 5.0625f) {
            cf h0, g1;
            helm2d_pair32(r2, kappa, dlp, h0, g1);
            if (slp) v = h0 * sg;
            if (dlp) v = v + (g1 * nd) * ta;
        } else {
            // |kappa r| > 3: FP64 r^2 and the FP64 evaluation, result rounded to FP32
            cf h0 = {0.f, 0.f}, g1 = {0.f, 0.f};
            helm2d_round32(r2_from_hl<DIM>(H), k, slp, dlp, h0, g1);
            if (slp) v = h0 * sg;
            if (dlp) v = v + (g1 * nd) * ta;
        }
    } else if (KER == CFMM_LAPLACE) {
        cf r = csqrtf_p(r2);
        cf ir = cinvf(r);
        if (slp) v = ir * sg;
        if (dlp) v = v + (nd * (ir * ir * ir)) * ta;
    } else {
        cf r = csqrtf_p(r2);
        cf g;
        float k4 = kappa * kappa * kappa * kappa;
        if (k4 * (r2.x * r2.x + r2.y * r2.y) <= 81.f) {    // |kappa r| <= 3
            float e = expf(-kappa * r.y), sn, cs;
            sincosf(kappa * r.x, &sn, &cs);
            g = cf{e * cs, e * sn} * cinvf(r);
        } else {
            // |kappa r| > 3: double-float phase
            cf e;
            far_phase_df<DIM>(H, kappa, (float)(k.k - (double)kappa), e, r);
            g = e * cinvf(r);
        }
        cf ir = cinvf(r);
        if (slp) v = g * sg;
        if (dlp) v = v + (nd * (cf{1.f, 0.f} - mul_if(kappa * r)) * g * (ir * ir)) * ta;
    }
    acc.add(v);
}

struct SrcTileF {
    float hr[kP2PChunk][3], lr[kP2PChunk][3], hi[kP2PChunk][3], li[kP2PChunk][3];
    float nhr[kP2PChunk][3], nlr[kP2PChunk][3], nhi[kP2PChunk][3], nli[kP2PChunk][3];
    cf sg[kP2PChunk], ta[kP2PChunk];
};

__device__ __forceinline__ void split_hl(double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
}

template <int DIM, int KER>
__device__ void accumulate_sources32(SrcTileF& S, const KParams& K, int rhs, int s, int e, bool tvalid,
                                     const double* ref_re, const double* ref_im, const float* xh_r,
                                     const float* xl_r, const float* xh_i, const float* xl_i, Kahan& acc,
                                     int split) {
    const int64_t n = K.n_src;
    float kap = (float)K.kappa;
    for (int c0 = s; c0 < e; c0 += kP2PChunk) {
        int cn = min(kP2PChunk, e - c0);
        __syncthreads();
        for (int j = threadIdx.x; j < cn; j += blockDim.x) {
            int g = c0 + j;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                split_hl(K.src_re[a * n + g] - ref_re[a], S.hr[j][a], S.lr[j][a]);
                split_hl(K.src_im[a * n + g] - ref_im[a], S.hi[j][a], S.li[j][a]);
                if (K.dlp) {
                    split_hl(K.nrm_re[a * n + g], S.nhr[j][a], S.nlr[j][a]);
                    split_hl(K.nrm_im[a * n + g], S.nhi[j][a], S.nli[j][a]);
                }
            }
            if (K.slp) {
                cd v = K.sigma[(int64_t)rhs * K.dens_stride + g];
                S.sg[j] = cf{(float)v.x, (float)v.y};
            }
            if (K.dlp) {
                cd v = K.tau[(int64_t)rhs * K.dens_stride + g];
                S.ta[j] = cf{(float)v.x, (float)v.y};
            }
        }
        __syncthreads();
        if (tvalid) {
            for (int j = split; j < cn; j += kP2PSplit) {
                float dr[DIM], di[DIM], hr[DIM], lr[DIM], hi[DIM], li[DIM];
                bool zero = true;
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    hr[a] = xh_r[a] - S.hr[j][a];
                    lr[a] = xl_r[a] - S.lr[j][a];
                    hi[a] = xh_i[a] - S.hi[j][a];
                    li[a] = xl_i[a] - S.li[j][a];
                    zero = zero && hr[a] == 0.f && lr[a] == 0.f && hi[a] == 0.f && li[a] == 0.f;
                    dr[a] = hr[a] + lr[a];
                    di[a] = hi[a] + li[a];
                }
                if (zero) continue;
                cf nd = {0.f, 0.f};
                if (K.dlp) nd = dot_nd<DIM>(hr, lr, hi, li, S.nhr[j], S.nlr[j], S.nhi[j], S.nli[j]);
                PairHL H{xh_r, xl_r, xh_i, xl_i, S.hr[j], S.lr[j], S.hi[j], S.li[j]};
                pair_kernel32<DIM, KER>(dr, di, H, nd, K.slp ? S.sg[j] : cf{0, 0}, K.dlp ? S.ta[j] : cf{0, 0},
                                        K.slp, K.dlp, kap, Wave{K.kappa, K.ikappa, K.isqrt_kappa, K.kappa_ang, K.kappa_exp}, acc);
            }
        }
    }
}

template <int DIM, int KER>
__device__ __forceinline__ void load_target32(const KParams& K, int ti, bool tvalid, const double* ref_re,
                                              const double* ref_im, float* xh_r, float* xl_r, float* xh_i,
                                              float* xl_i) {
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        double vr = tvalid ? K.trg_re[a * K.n_trg + ti] - ref_re[a] : 0.0;
        double vi = tvalid ? K.trg_im[a * K.n_trg + ti] - ref_im[a] : 0.0;
        split_hl(vr, xh_r[a], xl_r[a]);
        split_hl(vi, xh_i[a], xl_i[a]);
    }
}

template <int DIM, int KER>
__global__ void __launch_bounds__(kP2PThreads) k_p2p32(KParams K, const int* __restrict__ leaf_boxes,
                                                       const int* __restrict__ bst, const int* __restrict__ sen,
                                                       const int* __restrict__ ten,
                                                       const int* __restrict__ l1off, const int* __restrict__ l1,
                                                       cd* __restrict__ out) {
    __shared__ SrcTileF S;
    __shared__ cd red[kP2PThreads];
    int b = leaf_boxes[blockIdx.x];
    int rhs = blockIdx.y;
    int tl = threadIdx.x % kP2PTargets, split = threadIdx.x / kP2PTargets;
    int ts = bst[b], te = ten[b];
    double ref_re[DIM], ref_im[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        ref_re[a] = K.trg_re[a * K.n_trg + ts];
        ref_im[a] = K.trg_im[a * K.n_trg + ts];
    }
    for (int t0 = ts; t0 < te; t0 += kP2PTargets) {
        int ti = t0 + tl;
        bool tvalid = ti < te;
        float xh_r[DIM], xl_r[DIM], xh_i[DIM], xl_i[DIM];
        load_target32<DIM, KER>(K, ti, tvalid, ref_re, ref_im, xh_r, xl_r, xh_i, xl_i);
        Kahan acc;
        for (int q = l1off[b]; q < l1off[b + 1]; ++q) {
            int a = l1[q];
            accumulate_sources32<DIM, KER>(S, K, rhs, bst[a], sen[a], tvalid, ref_re, ref_im, xh_r, xl_r, xh_i,
                                           xl_i, acc, split);
        }
        finish_target<DIM, KER>(acc.value(), red, tl, split, tvalid, out + (int64_t)rhs * K.n_trg + ti);
    }
}

template <int DIM, int KER>
__global__ void __launch_bounds__(kP2PThreads) k_direct32(KParams K, cd* __restrict__ out) {
    __shared__ SrcTileF S;
    __shared__ cd red[kP2PThreads];
    int rhs = blockIdx.y;
    int tl = threadIdx.x % kP2PTargets, split = threadIdx.x / kP2PTargets;
    int t0 = blockIdx.x * kP2PTargets;
    int ti = t0 + tl;
    bool tvalid = ti < K.n_trg;
    double ref_re[DIM], ref_im[DIM];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        ref_re[a] = K.trg_re[a * K.n_trg + t0];
        ref_im[a] = K.trg_im[a * K.n_trg + t0];
    }
    float xh_r[DIM], xl_r[DIM], xh_i[DIM], xl_i[DIM];
    load_target32<DIM, KER>(K, ti, tvalid, ref_re, ref_im, xh_r, xl_r, xh_i, xl_i);
    Kahan acc;
    accumulate_sources32<DIM, KER>(S, K, rhs, 0, (int)K.n_src, tvalid, ref_re, ref_im, xh_r, xl_r, xh_i, xl_i,
                                   acc, split);
    finish_target<DIM, KER>(acc.value(), red, tl, split, tvalid, out + (int64_t)rhs * K.n_trg + ti);
}

// ---------------------------------------------------------------------------
// Mixed-precision 3D Helmholtz near field on a power-of-two grid.
//
// Every coordinate v of a List-1 pair (real and imaginary parts, offsets from
// the target leaf's first point) is split as v = h + l with h = g rint(v/g)
// on a grid of step g = 2^e >= R/1024, R = 1.5 (k+1) w the per-axis reach of
// the near field of a leaf of width w at separation k (List-1 leaves differ
// by at most one level), and l = v - h, |l| <= g/2, rounded to FP32. Then the
// differences dh = x_h - y_h are multiples of g below 2048 g and are exact in
// FP32, as are their products and the sums of three of them (below 2^24 g^2):
//   r^2 = S_h + S_l,  S_h = sum dh_re^2 - dh_im^2 + 2 i dh_re dh_im  (exact),
//   S_l = sum (2 dh + dl) dl terms                           (FP32, small),
// so r^2 is known as an unevaluated FP32 pair to ~2^-24 g |r| absolute. The
// root r0 of the rounded sum is refined by one Newton step computed from
// that pair (r = r0 + (r^2 - r0^2)/(2 r0), with r0^2 formed by exact
// products), and kappa r is formed in double-float, so the phase and the
// decay exp(-kappa Im r) keep absolute errors near kappa g 2^-24 at any
// kappa r. The phase is reduced by 2 pi before sincosf. Sources are staged
// as float4 quadruples; the sum over sources is compensated (Kahan).
// ---------------------------------------------------------------------------
struct SrcTileG {
    float4 q0[kP2PChunk], q1[kP2PChunk], q2[kP2PChunk], dn[kP2PChunk];   // coordinates, densities
    float4 n0[kP2PChunk], n1[kP2PChunk], n2[kP2PChunk];                  // normals (double layer)
};

// v = h + l on the grid of step g (h exact in FP32 for |v| < 2^23 g)
__device__ __forceinline__ void split_grid(double v, double g, double ig, float& h, float& l) {
    double hv = g * rint(v * ig);
    h = (float)hv;
    l = (float)(v - hv);
}

// (re hi x3, im hi x3, re lo x3, im lo x3) <-> three float4
__device__ __forceinline__ void pack12(const float* a, float4& q0, float4& q1, float4& q2) {
    q0 = make_float4(a[0], a[1], a[2], a[3]);
    q1 = make_float4(a[4], a[5], a[6], a[7]);
    q2 = make_float4(a[8], a[9], a[10], a[11]);
}

// grid step for a target leaf of width w at separation k: 2^ceil(log2(R/1024))
__device__ __forceinline__ double near_grid_step(double w, int sep) {
    double R = 1.5 * (sep + 1) * w;
    int e;
    frexp(R / 1024.0, &e);     // R/1024 = f 2^e, f in [0.5, 1)
    return ldexp(1.0, e);
}

__global__ void __launch_bounds__(kP2PThreads) k_p2p32g_h3(KParams K, const int* __restrict__ leaf_boxes, NearRanges R,
                                                           const int* __restrict__ l1off,
                                                           const int* __restrict__ l1,
                                                           const int* __restrict__ blevel, double W, int sep,
                                                           cd* __restrict__ out) {
    __shared__ SrcTileG S;
    __shared__ cd red[kP2PThreads];
    const int64_t n = K.n_src;
    int b = leaf_boxes[blockIdx.x];
    int rhs = blockIdx.y;
    int tl = threadIdx.x % kP2PTargets, split = threadIdx.x / kP2PTargets;
    int ts = R.trg.st[b], te = R.trg.en[b];
    const int first = R.first[b];   // (ts, the same point, costs 92 registers instead of 80 and 46 ms instead of 44)
    double g = near_grid_step(ldexp(W, -blevel[b]), sep), ig = 1.0 / g;
    double ref_re[3], ref_im[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ref_re[a] = K.trg_re[a * K.n_trg + first];
        ref_im[a] = K.trg_im[a * K.n_trg + first];
    }
    const float kh = (float)K.kappa, kl = (float)(K.kappa - (double)kh);
    const float kTwoPiH = 6.28318548202514648f;     // float(2 pi)
    const float kTwoPiL = -1.74845553e-07f;         // 2 pi - float(2 pi)
    for (int t0 = ts; t0 < te; t0 += kP2PTargets) {
        bool tvalid = t0 + tl < te;
        const int64_t ti = tvalid ? R.trg.at(t0 + tl) : 0;
        // target: x[0..2] re hi, x[3..5] im hi, x[6..8] re lo, x[9..11] im lo
        float x[12];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            double vr = tvalid ? K.trg_re[a * K.n_trg + ti] - ref_re[a] : 0.0;
            double vi = tvalid ? K.trg_im[a * K.n_trg + ti] - ref_im[a] : 0.0;
            split_grid(vr, g, ig, x[a], x[6 + a]);
            split_grid(vi, g, ig, x[3 + a], x[9 + a]);
        }
        Kahan acc;
        for (int q = l1off[b]; q < l1off[b + 1]; ++q) {
            int src = l1[q];
            int s0 = R.src.st[src], s1 = R.src.en[src];
            for (int c0 = s0; c0 < s1; c0 += kP2PChunk) {
                int cn = min(kP2PChunk, s1 - c0);
                __syncthreads();
                for (int j = threadIdx.x; j < cn; j += blockDim.x) {
                    const int64_t gi = R.src.at(c0 + j);
                    float y[12];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        split_grid(K.src_re[a * n + gi] - ref_re[a], g, ig, y[a], y[6 + a]);
                        split_grid(K.src_im[a * n + gi] - ref_im[a], g, ig, y[3 + a], y[9 + a]);
                    }
                    pack12(y, S.q0[j], S.q1[j], S.q2[j]);
                    float4 dn = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (K.slp) {
                        cd v = K.sigma[(int64_t)rhs * K.dens_stride + gi];
                        dn.x = (float)v.x;
                        dn.y = (float)v.y;
                    }
                    if (K.dlp) {
                        cd v = K.tau[(int64_t)rhs * K.dens_stride + gi];
                        dn.z = (float)v.x;
                        dn.w = (float)v.y;
                        float nv[12];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            split_hl(K.nrm_re[a * n + gi], nv[a], nv[6 + a]);
                            split_hl(K.nrm_im[a * n + gi], nv[3 + a], nv[9 + a]);
                        }
                        pack12(nv, S.n0[j], S.n1[j], S.n2[j]);
                    }
                    S.dn[j] = dn;
                }
                __syncthreads();
                if (!tvalid) continue;
                for (int j = split; j < cn; j += kP2PSplit) {
                    float4 a0 = S.q0[j], a1 = S.q1[j], a2 = S.q2[j];
                    // dh: re 0..2, im 0..2 (exact); dl likewise
                    float hr0 = x[0] - a0.x, hr1 = x[1] - a0.y, hr2 = x[2] - a0.z;
                    float hi0 = x[3] - a0.w, hi1 = x[4] - a1.x, hi2 = x[5] - a1.y;
                    float lr0 = x[6] - a1.z, lr1 = x[7] - a1.w, lr2 = x[8] - a2.x;
                    float li0 = x[9] - a2.y, li1 = x[10] - a2.z, li2 = x[11] - a2.w;
                    unsigned nz = (__float_as_uint(hr0) | __float_as_uint(hr1) | __float_as_uint(hr2) |
                                   __float_as_uint(hi0) | __float_as_uint(hi1) | __float_as_uint(hi2) |
                                   __float_as_uint(lr0) | __float_as_uint(lr1) | __float_as_uint(lr2) |
                                   __float_as_uint(li0) | __float_as_uint(li1) | __float_as_uint(li2)) &
                                  0x7fffffffu;
                    if (nz == 0u) continue;   // x == y: self pair / coincident point
                    // r^2 = (Srh + Srl) + i (Sih + Sil)
                    float Srh = hr0 * hr0;
                    Srh = fmaf(hr1, hr1, Srh);
                    Srh = fmaf(hr2, hr2, Srh);
                    Srh = fmaf(-hi0, hi0, Srh);
                    Srh = fmaf(-hi1, hi1, Srh);
                    Srh = fmaf(-hi2, hi2, Srh);
                    float Sih = hr0 * hi0;
                    Sih = fmaf(hr1, hi1, Sih);
                    Sih = fmaf(hr2, hi2, Sih);
                    Sih = 2.f * Sih;
                    float Srl = fmaf(2.f, hr0, lr0) * lr0;
                    Srl = fmaf(fmaf(2.f, hr1, lr1), lr1, Srl);
                    Srl = fmaf(fmaf(2.f, hr2, lr2), lr2, Srl);
                    Srl = fmaf(-fmaf(2.f, hi0, li0), li0, Srl);
                    Srl = fmaf(-fmaf(2.f, hi1, li1), li1, Srl);
                    Srl = fmaf(-fmaf(2.f, hi2, li2), li2, Srl);
                    float Sil = fmaf(hr0, li0, lr0 * (hi0 + li0));
                    Sil = fmaf(hr1, li1, fmaf(lr1, hi1 + li1, Sil));
                    Sil = fmaf(hr2, li2, fmaf(lr2, hi2 + li2, Sil));
                    Sil = 2.f * Sil;
                    float ra = Srh + Srl, rb = Sih + Sil;
                    // r0 = principal sqrt(ra + i rb) in FP32 (refined below)
                    float m = sqrtf(fmaf(ra, ra, rb * rb));
                    float t2 = 0.5f * (fabsf(ra) + m);
                    float rt = rsqrtf(t2);
                    float t = t2 * rt, u = 0.5f * rb * rt;
                    float a0r = ra >= 0.f ? t : fabsf(u);
                    float b0r = ra >= 0.f ? u : copysignf(t, rb);
                    // Newton step: delta = (r^2 - r0^2)/(2 r0), r0^2 from exact products
                    float p = a0r * a0r, e1 = fmaf(a0r, a0r, -p);
                    float qq = b0r * b0r, e2 = fmaf(b0r, b0r, -qq);
                    float hs, ls;
                    two_sum(p, -qq, hs, ls);
                    float dre = ((Srh - hs) - ls) + ((Srl - e1) + e2);
                    float pi_ = a0r * b0r, e3 = fmaf(a0r, b0r, -pi_);
                    float dim = ((Sih - 2.f * pi_) - 2.f * e3) + Sil;
                    float i2m = __fdividef(0.5f, m);
                    float der = fmaf(dre, a0r, dim * b0r) * i2m;
                    float dei = fmaf(dim, a0r, -dre * b0r) * i2m;
                    // kappa r in double-float: (th + te) + i (dh + de)
                    float th, tq, dh, dq;
                    two_prod(kh, a0r, th, tq);
                    tq = fmaf(kh, der, fmaf(kl, a0r, tq));
                    two_prod(kh, b0r, dh, dq);
                    dq = fmaf(kh, dei, fmaf(kl, b0r, dq));
                    float kk = rintf(th * 0.159154943f);
                    float q2, q2e;
                    two_prod(kk, kTwoPiH, q2, q2e);
                    float ph = (th - q2) + ((tq - q2e) - kk * kTwoPiL);
                    float sn, cs;
                    sincosf(ph, &sn, &cs);
                    float mag = expf(-dh) * (1.f - dq);
                    // 1/r with r = r0 + delta rounded to FP32
                    float rr = a0r + der, ri = b0r + dei;
                    float id = __frcp_rn(fmaf(rr, rr, ri * ri));
                    float irr = rr * id, iri = -ri * id;
                    cf gk = cf{mag * cs, mag * sn} * cf{irr, iri};   // e^{i kappa r}/r
                    float4 dn = S.dn[j];
                    cf v = {0.f, 0.f};
                    if (K.slp) v = gk * cf{dn.x, dn.y};
                    if (K.dlp) {
                        float4 b0 = S.n0[j], b1 = S.n1[j], b2 = S.n2[j];
                        const float dh_r[3] = {hr0, hr1, hr2}, dl_r[3] = {lr0, lr1, lr2};
                        const float dh_i[3] = {hi0, hi1, hi2}, dl_i[3] = {li0, li1, li2};
                        const float nh_r[3] = {b0.x, b0.y, b0.z}, nh_i[3] = {b0.w, b1.x, b1.y};
                        const float nl_r[3] = {b1.z, b1.w, b2.x}, nl_i[3] = {b2.y, b2.z, b2.w};
                        cf nd = dot_nd<3>(dh_r, dl_r, dh_i, dl_i, nh_r, nl_r, nh_i, nl_i);
                        cf ir = {irr, iri};
                        cf kr = {kh * rr, kh * ri};
                        v = v + (nd * (cf{1.f, 0.f} - mul_if(kr)) * gk * (ir * ir)) * cf{dn.z, dn.w};
                    }
                    acc.add(v);
                }
            }
        }
        finish_target<3, CFMM_HELMHOLTZ>(acc.value(), red, tl, split, tvalid, out + (int64_t)rhs * K.n_trg + ti);
    }
}

static KParams with_wave(KParams K) {
    Wave w = make_wave(K.kappa);
    K.ikappa = w.ik;
    K.isqrt_kappa = w.isk;
    K.kappa_ang = w.ka;
    K.kappa_exp = w.kb;
    return K;
}

// nleaves target leaves of at most leaf_size points each (List 1 in L), or,
// without boxes, all targets against all sources. Blocks differ in work, so a
// large near field is cut down to 16 targets a block while an SM gets fewer than
// 32 blocks (8,224 instead of 1,028 blocks of the 1e5-point 3D Helmholtz surface:
// 37.9 -> 36.1 ms). A small one runs beside the far field, whose first kernels
// wait for free SMs: two blocks an SM, of at least 4 targets (70 leaves of a
// 3,001-point 2D Helmholtz matvec: 0.62 -> 0.21 ms). The direct sum has the chip
// to itself.
template <int DIM, int KER, bool GRAD>
static void launch_near(const KParams& K, const NearLists& L, int nleaves, int leaf_size, cd* out, int nrhs,
                        cudaStream_t st) {
    int dev = 0, nsm = 0;
    CFMM_CUDA(cudaGetDevice(&dev));
    CFMM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    // (nrhs stays out of the rule: the order of a target's sum depends on tb, and a
    // right-hand side's result is the same alone and among others)
    int64_t per = L.boxes ? leaf_size : K.n_trg, rows = L.boxes ? nleaves : 1;
    int tb = (int)std::min<int64_t>(kNearTargets, per);
    auto blocks = [&] { return rows * ((per + tb - 1) / tb); };
    if (rows * per >= 32768)
        while (tb > 16 && blocks() < 32 * nsm) tb = std::max(16, tb / 2);
    while (tb > 4 && blocks() < (L.boxes ? 2 : 8) * nsm) tb = std::max(4, tb / 2);
    unsigned groups = (unsigned)((per + tb - 1) / tb);
    dim3 grid = L.boxes ? dim3((unsigned)nleaves, nrhs, groups) : dim3(groups, nrhs);
    k_near<DIM, KER, GRAD><<<grid, kNearThreads, near_smem<DIM, GRAD>(), st>>>(K, L, tb, out);
    CFMM_LAUNCHED();
}

template <int DIM, int KER>
static void launch_p2p_t(const KParams& K, const int* leaf_boxes, int nleaves, const NearRanges& R,
                         const int* l1off, const int* l1, cd* out, int nrhs, bool mixed, cudaStream_t st,
                         int leaf_size) {
    if (nleaves == 0) return;
    dim3 grid(nleaves, nrhs);
    if (mixed) {
        k_p2p32<DIM, KER><<<grid, kP2PThreads, 0, st>>>(K, leaf_boxes, R.first, R.src.en, R.trg.en, l1off, l1, out);
        CFMM_LAUNCHED();
    } else {
        launch_near<DIM, KER, false>(K, NearLists{leaf_boxes, R.src, R.trg, l1off, l1}, nleaves, leaf_size, out, nrhs, st);
    }
}

void launch_p2p(int dim, int ker, const KParams& K0, const int* leaf_boxes, int nleaves, const NearRanges& R,
                const int* l1off, const int* l1, cd* out, int nrhs, cudaStream_t st,
                bool mixed, int leaf_size, const int* blevel, double W, int sep) {
    const KParams K = with_wave(K0);
    if (mixed && dim == 3 && ker == CFMM_HELMHOLTZ && blevel && nleaves > 0) {
        dim3 grid(nleaves, nrhs);
        k_p2p32g_h3<<<grid, kP2PThreads, 0, st>>>(K, leaf_boxes, R, l1off, l1, blevel, W, sep, out);
        CFMM_LAUNCHED();
        return;
    }
    if (dim == 2 && ker == CFMM_LAPLACE) launch_p2p_t<2, CFMM_LAPLACE>(K, leaf_boxes, nleaves, R, l1off, l1, out, nrhs, mixed, st, leaf_size);
    else if (dim == 2) launch_p2p_t<2, CFMM_HELMHOLTZ>(K, leaf_boxes, nleaves, R, l1off, l1, out, nrhs, mixed, st, leaf_size);
    else if (ker == CFMM_LAPLACE) launch_p2p_t<3, CFMM_LAPLACE>(K, leaf_boxes, nleaves, R, l1off, l1, out, nrhs, mixed, st, leaf_size);
    else launch_p2p_t<3, CFMM_HELMHOLTZ>(K, leaf_boxes, nleaves, R, l1off, l1, out, nrhs, mixed, st, leaf_size);
}

template <int DIM, int KER>
static void launch_p2p_grad_t(const KParams& K, const int* leaf_boxes, int nleaves, const NearRanges& R,
                              const int* l1off, const int* l1, cd* g, int nrhs, cudaStream_t st, int leaf_size) {
    if (nleaves == 0) return;
    launch_near<DIM, KER, true>(K, NearLists{leaf_boxes, R.src, R.trg, l1off, l1}, nleaves, leaf_size, g, nrhs, st);
}

void launch_p2p_grad(int dim, int ker, const KParams& K0, const int* leaf_boxes, int nleaves, const NearRanges& R,
                     const int* l1off, const int* l1, cd* g, int nrhs, cudaStream_t st,
                     int leaf_size) {
    const KParams K = with_wave(K0);
    if (dim == 2 && ker == CFMM_LAPLACE) launch_p2p_grad_t<2, CFMM_LAPLACE>(K, leaf_boxes, nleaves, R, l1off, l1, g, nrhs, st, leaf_size);
    else if (dim == 2) launch_p2p_grad_t<2, CFMM_HELMHOLTZ>(K, leaf_boxes, nleaves, R, l1off, l1, g, nrhs, st, leaf_size);
    else if (ker == CFMM_LAPLACE) launch_p2p_grad_t<3, CFMM_LAPLACE>(K, leaf_boxes, nleaves, R, l1off, l1, g, nrhs, st, leaf_size);
    else launch_p2p_grad_t<3, CFMM_HELMHOLTZ>(K, leaf_boxes, nleaves, R, l1off, l1, g, nrhs, st, leaf_size);
}

template <int DIM, int KER>
static void launch_direct_t(const KParams& K, cd* out, int nrhs, bool mixed, cudaStream_t st) {
    if (!mixed) {
        launch_near<DIM, KER, false>(K, NearLists{}, 0, 0, out, nrhs, st);
        return;
    }
    dim3 grid((unsigned)((K.n_trg + kP2PTargets - 1) / kP2PTargets), nrhs);
    k_direct32<DIM, KER><<<grid, kP2PThreads, 0, st>>>(K, out);
    CFMM_LAUNCHED();
}

void launch_direct(int dim, int ker, const KParams& K0, cd* out, int nrhs, cudaStream_t st, bool mixed) {
    const KParams K = with_wave(K0);
    if (K.n_trg == 0) return;
    if (dim == 2 && ker == CFMM_LAPLACE) launch_direct_t<2, CFMM_LAPLACE>(K, out, nrhs, mixed, st);
    else if (dim == 2) launch_direct_t<2, CFMM_HELMHOLTZ>(K, out, nrhs, mixed, st);
    else if (ker == CFMM_LAPLACE) launch_direct_t<3, CFMM_LAPLACE>(K, out, nrhs, mixed, st);
    else launch_direct_t<3, CFMM_HELMHOLTZ>(K, out, nrhs, mixed, st);
}

}  // namespace cfmm

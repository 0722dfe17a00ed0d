// 3D translations (M2M, M2L, L2L), Laplace and Helmholtz: point-and-shoot (the
// scheme, operators and recurrences of helm3d.cu's file comment) with 32 pairs on
// the lanes of a warp.
//
// The FP64 pipe bounds them (one warp instruction per 16 SM cycles), so the work
// is arranged to issue as few FP64 instructions as the operators allow, each with
// 32 lanes in use:
//   * a lane is a pair. Every lane does the same (n, m, m') at the same time: no
//     partial warps at the ends of rows and orders, rotation table entries are
//     uniform, per-pair factors sit in [..][32] rows that load as 512 bytes.
//   * both directions of a List-2 pair (a <- b, b <- a) share the shift's length
//     and so the coaxial operator T: it is built once per unordered pair and each
//     entry, once loaded, serves 4 vectors (two directions, +m and -m). The
//     reversed shift has e' = -e and e_a' = -1/e_a.
//   * a shift with d3 = 0 (boxes in one layer, equal Im of the third centre
//     coordinate; most List-2 pairs of a flat surface) has e_a = i exactly, and the
//     rotation D^T E(i) D between the diagonal factors is the fixed matrix D
//     itself: one real matrix pass and one diagonal scaling instead of two each.
// Stages, each reading and writing the pair vectors V[rhs, dir][tile][coef][32]:
//   k_pair_pre    powers e^m, e_a^m and the radial sequence of each pair
//   k_pair_tri    coaxial triangles T (Helmholtz)
//   k_pair_fwd    gather the source expansion, rotate (per order n)
//   k_pair_coax   coaxial product (per m), in place
//   k_pair_bwd    rotate back (per order n), in place
//   k_pair_sum    add the vectors of a box's List 2 (children, parent) in order
// Per List-2 pair and direction at order 16: 25k FP64 lane instructions + 4k for T,
// against 65k issued by one-block-per-box translation (153 coefficient items on
// 256 threads, both rotations in full, T per direction). V costs 5 passes over
// 16 (P+1)^2 bytes a pair, about a tenth of the time at HBM rate.
#include <algorithm>

#include "cfmm_special.cuh"
#include "kernels.cuh"
#include "pairs3d.cuh"

namespace cfmm {

namespace {

constexpr int kPairFlat = 0, kPairGeneral = 1, kPairIso = 2;   // kPairIso + k: fixed frame Q_k
constexpr double kDegenTol = 1e-8;   // |d1^2 + d2^2| <= this * sum |d_i|^2: fixed-frame translation
constexpr int kPairThreads = 128;
constexpr size_t kPairBudget = (size_t)6 << 30;   // bytes of T and V of a launch range

__device__ __forceinline__ int nmi(int n, int m) { return n * n + n + m; }
__device__ __forceinline__ cd ipow(int e, cd x) {
    switch (e & 3) {
        case 0: return x;
        case 1: return cd{-x.y, x.x};
        case 2: return cd{-x.x, -x.y};
        default: return cd{x.y, -x.x};
    }
}
__device__ __forceinline__ cd sgn(int m, cd x) { return (m & 1) ? -x : x; }
__device__ __forceinline__ double coax_g(int c) { return (c & 1) ? -(2.0 * c + 1.0) : (2.0 * c + 1.0); }
__host__ __device__ inline size_t tri_off(int P, int m) {      // entries of the triangles r <= P before m
    size_t a = (size_t)(P + 1) * (P + 2) * (P + 3) / 6, b = (size_t)(P - m + 1) * (P - m + 2) * (P - m + 3) / 6;
    return a - b;
}

// shift c_a - c_b (destination a), turned into the fixed frame for isotropic pairs
__device__ int pair_shift(const double* cre, const double* cim, int a, int b, cd* d) {
    for (int k = 0; k < 3; ++k) d[k] = cd{cre[3 * a + k] - cre[3 * b + k], cim[3 * a + k] - cim[3 * b + k]};
    cd s2 = d[0] * d[0] + d[1] * d[1];
    double n2 = cabs2(d[0]) + cabs2(d[1]) + cabs2(d[2]);
    bool xy = d[0].x != 0.0 || d[0].y != 0.0 || d[1].x != 0.0 || d[1].y != 0.0;
    if (xy && cabs2(s2) <= (kDegenTol * n2) * (kDegenTol * n2)) {
        // Q_0 d = (-d3, d2, d1), Q_1 d = (-d3, -d1, d2): the one with the larger |(Q d)_1^2 + (Q d)_2^2|
        cd a0 = d[2] * d[2] + d[1] * d[1], a1 = d[2] * d[2] + d[0] * d[0];
        int k = cabs2(a0) >= cabs2(a1) ? 0 : 1;
        cd q1 = k == 0 ? d[1] : -d[0], q2 = k == 0 ? d[0] : d[1];
        d[0] = -d[2];
        d[1] = q1;
        d[2] = q2;
        return kPairIso + k;
    }
    return xy && d[2].x == 0.0 && d[2].y == 0.0 ? kPairFlat : kPairGeneral;
}

// A warp per box a over its List-2 entries (a, b), a < b, in list order. Flat pairs fill
// their level's slots from the front, the others from the back, so a tile holds one sort
// only and a pair's arithmetic does not depend on its slot. The first call (box_a null)
// counts a box's pairs, cnt[a] flat and cnt[nbox + a] others; the second takes the slots
// from the counts' scan: they follow from the lists alone, so that the order in which a
// box's terms are added is the same for every plan of a geometry. With separate targets
// (src.map), a pair gets a slot only where one box holds a source and the other a target.
// (50,007 targets of 200,000 Laplace sources, order 16: M2L 39.3 -> 13.8 ms.)
__global__ void k_pair_slots(int nbox, const int* __restrict__ loff, const int* __restrict__ lent,
                             const int* __restrict__ level, const int* __restrict__ level_off,
                             const int* __restrict__ tile0, const double* __restrict__ cre,
                             const double* __restrict__ cim, SubRange src, SubRange trg, int* __restrict__ cnt,
                             const int* __restrict__ pos, int* __restrict__ box_a, int* __restrict__ box_b,
                             signed char* __restrict__ kind, int* __restrict__ slot) {
    const int a = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (a >= nbox) return;
    const int l = level[a], q1 = loff[a + 1];
    const bool a_src = !src.map || src.st[a] < src.en[a], a_trg = !src.map || trg.st[a] < trg.en[a];
    int nf = 0, no = 0;
    if (box_a) {
        nf = 32 * tile0[l] + pos[a] - pos[level_off[l]];
        no = 32 * tile0[l + 1] - 1 - (pos[nbox + a] - pos[nbox + level_off[l]]);
    }
    for (int q0 = loff[a]; q0 < q1; q0 += 32) {
        const int q = q0 + lane, b = q < q1 ? lent[q] : -1;
        const bool mine = b > a;
        const bool use = mine && (!src.map || (a_src && trg.st[b] < trg.en[b]) || (a_trg && src.st[b] < src.en[b]));
        cd d[3];
        const int kd = use ? pair_shift(cre, cim, a, b, d) : kPairFlat;
        const unsigned mf = __ballot_sync(0xffffffffu, use && kd == kPairFlat),
                       mo = __ballot_sync(0xffffffffu, use && kd != kPairFlat), below = (1u << lane) - 1u;
        if (box_a && mine) {
            int lo = loff[b], hi = loff[b + 1] - 1;       // a in the list of b (sorted; List 2 is symmetric)
            while (lo < hi) {
                int m = (lo + hi) >> 1;
                if (lent[m] < a) lo = m + 1;
                else hi = m;
            }
            if (!use) {
                slot[q] = slot[lo] = -1;
            } else {
                const int p = kd == kPairFlat ? nf + __popc(mf & below) : no - __popc(mo & below);
                box_a[p] = a;
                box_b[p] = b;
                kind[p] = (signed char)kd;
                slot[q] = 2 * p;
                slot[lo] = 2 * p + 1;
            }
        }
        nf += __popc(mf);
        no += box_a ? -__popc(mo) : __popc(mo);
    }
    if (!box_a && lane == 0) {
        cnt[a] = nf;
        cnt[nbox + a] = no;
        if (a == 0) cnt[2 * nbox] = 0;
    }
}

// pairs before each level: out[l] flat, out[nlev + 1 + l] others
__global__ void k_pair_levels(int nlev, int nbox, const int* __restrict__ level_off, const int* __restrict__ pos,
                              int* __restrict__ out) {
    for (int l = threadIdx.x; l <= nlev; l += blockDim.x) {
        out[l] = pos[level_off[l]];
        out[nlev + 1 + l] = pos[nbox + level_off[l]];
    }
}

// mode 0: M2M (a = parent <- b = child), 1: M2L (both directions), 2: L2L (b <- a)
struct PairArgs {
    const double *cre, *cim;
    const int *box_a, *box_b;     // slots (M2L); nullptr: pair p is child box lo + p and its parent
    const int* parent;
    signed char* kind;
    int lo, hi;                   // children (M2M, L2L)
    Tr3Tables T;
    const int64_t* eoff;
    int64_t ncoef;
    int mode, Pi, Po, Pm, Pn;     // source and destination order, their maximum and minimum
    int t0, ntile;                // tiles [t0, t0 + ntile) of the slots
    double kappa;
    cd *pw, *fl, *tri, *vec;      // of this range
    // diagonal factors of the Laplace stages (solid-harmonic and Y basis, see k_pair_coax)
    const double *s_in, *s_mid, *s_out, *s_fin;

    __device__ int a(int p) const {
        if (box_a) return box_a[32 * t0 + p];
        return lo + p < hi ? parent[lo + p] : -1;
    }
    __device__ int b(int p) const {
        if (box_a) return box_b[32 * t0 + p];
        return lo + p < hi ? lo + p : -1;
    }
    // direction and right-hand side of vector v
    __device__ int dir(int v) const { return mode == 1 ? v & 1 : mode >> 1; }
    __device__ int rhs(int v) const { return mode == 1 ? v >> 1 : v; }
    __host__ __device__ size_t K() const { return (size_t)(Pm + 1) * (Pm + 1); }
};

// e^m, e_a^m (m = -Pm..Pm) and the radial sequence, rows [..][32], one thread per
// pair. Helmholtz: h_l(kappa t) (M2L) or j_l(kappa t), l <= Pi + Po. Laplace, along
// the z-axis in the solid-harmonic basis: l!/t^{l+1} (M2L), (-t)^l/l! (M2M), t^l/l!
// (L2L), l <= 2P.
template <bool LAP>
__global__ void k_pair_pre(PairArgs A) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 32 * A.ntile) return;
    const int P = A.Pm, NR = A.Pi + A.Po, a = A.a(p);
    if (a < 0) return;
    size_t tile = p >> 5;
    int lane = p & 31;
    cd d[3];
    int kd = pair_shift(A.cre, A.cim, a, A.b(p), d);
    if (A.mode != 1) {
        if (kd == kPairFlat) kd = kPairGeneral;
        A.kind[p] = (signed char)kd;
    }
    cd s2 = d[0] * d[0] + d[1] * d[1];
    cd t = csqrt_p(s2 + d[2] * d[2]);
    cd sq = {0, 0}, e = {1, 0};
    if (!(s2.x == 0.0 && s2.y == 0.0)) {
        sq = csqrt_p(s2);
        e = (d[0] + mul_i(d[1])) / sq;
    }
    cd* pw = A.pw + tile * (4 * P + 2) * 32 + lane;
    for (int q = 0; q < (kd == kPairFlat ? 1 : 2); ++q) {
        cd x = q ? (d[2] + mul_i(sq)) / t : e, ix = cinv(x), v = {1, 0}, iv = {1, 0};
        cd* dst = pw + (size_t)(q * (2 * P + 1) + P) * 32;
        dst[0] = v;
        for (int m = 1; m <= P; ++m) {
            v = v * x;
            iv = iv * ix;
            dst[m * 32] = v;
            dst[-m * 32] = iv;
        }
    }
    cd* f = A.fl + tile * (NR + 1) * 32 + lane;
    if (LAP) {
        cd x = A.mode == 1 ? cinv(t) : A.mode == 0 ? -t : t, v = A.mode == 1 ? x : cd{1, 0};
        const double* c = A.mode == 1 ? A.T.fact : A.T.ifact;
        for (int j = 0; j <= NR; ++j) {
            f[j * 32] = __ldg(c + j) * v;
            v = v * x;
        }
    } else if (A.mode == 1) {
        // h_n of cfmm_special.cuh's sph_h_seq, written row by row
        cd z = A.kappa * t, ez = cexp_i(z), zi = cinv(z);
        cd h0 = -mul_i(ez * zi), h1 = -(ez * (z + cd{0.0, 1.0})) * (zi * zi);
        f[0] = h0;
        if (NR > 0) f[32] = h1;
        for (int n = 1; n < NR; ++n) {
            cd h2 = rmac(-h0, 2.0 * n + 1.0, zi * h1);
            f[(n + 1) * 32] = h2;
            h0 = h1;
            h1 = h2;
        }
    } else {
        cd j[2 * kMaxP3Top + 1];
        sph_j_seq(A.kappa * t, NR, j);
        for (int n = 0; n <= NR; ++n) f[n * 32] = j[n];
    }
}

// Coaxial triangles T'_{rc} = g_c T_{rc}^m, m <= c <= r, r <= Pm, c <= Pn, g_c =
// (-1)^c (2c+1), of a tile: entries at tri_off(Pm, m) + (r-m)(r-m+1)/2 + c - m, rows
// [..][32]. The block's warps take the rows r of a column; the sectorial column and
// the two before the next one live in shared memory, the buffers changing roles.
// With T_{rc} = gamma_c U_{rc}, gamma_{c+1} = gamma_c / be_c, the recurrence of
// helm3d.cu has no division:
//   U_{r,c+1} = al_c be_{c-1} U_{r,c-1} - al_{r+1} U_{r+1,c} + be_{r-1} U_{r-1,c},
// 6 FP64 instructions a row and 2 for the rows kept (T' = cg_c U, cg = g gamma; the
// products of coefficients are tabulated), which bound it (with 8 + 2 and six more a
// column 3.86 instead of 2.86 ms at order 23, 32,000 pairs). The 3 (NR+2)
// rows of 512 bytes leave 4 blocks an SM at order 16 and 1 at 63, and a block's
// warps alone keep most of the FP64 pipe busy.
//
// A launch of few tiles (a coarse level: high orders, few pairs) would leave SMs
// idle and walk all m in one block: there k_pair_sect writes the sectorial columns
// of every m first and the grid takes (tile, m) (52 tiles at order 60: 7.2 -> 2.1
// ms). With four tiles an SM the columns stay in the block.
__global__ void __launch_bounds__(256) k_pair_sect(PairArgs A, cd* __restrict__ out) {
    extern __shared__ cd sm[];
    const int NR = A.Pi + A.Po, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t tile = blockIdx.x, L = (size_t)(NR + 2) * 32;
    cd *sect = sm + lane, *b1 = sect + L;
    const cd* f = A.fl + tile * (NR + 1) * 32 + lane;
    for (int m = 0; m <= A.Pn; ++m) {
        cd* o = out + (tile * (A.Pn + 1) + m) * (NR + 1) * 32 + lane;
        for (int r = m + w; r <= NR - m; r += nw) {
            // T^m_{r,m} from T^{m-1}_{r+-1,m-1}
            cd v = m == 0 ? coax_g(r) * f[r * 32]
                          : rmac(__ldg(A.T.smu + nmi(r, m)) * sect[(r + 1) * 32], __ldg(A.T.snu + nmi(r, m)),
                                 sect[(r - 1) * 32]);
            b1[r * 32] = v;
            o[(size_t)r * 32] = v;
        }
        cd* x = sect;
        sect = b1;
        b1 = x;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k_pair_tri(PairArgs A, const cd* __restrict__ sect_all) {
    extern __shared__ cd sm[];
    const int Pm = A.Pm, Pn = A.Pn, NR = A.Pi + A.Po;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t tile = blockIdx.x, L = (size_t)(NR + 2) * 32;
    const Tr3Tables& C = A.T;
    cd *sect = sm + lane, *b1 = sect + L, *b2 = b1 + L;
    const cd* f = A.fl + tile * (NR + 1) * 32 + lane;
    cd* T = A.tri + tile * tri_off(Pm, Pm + 1) * 32 + lane;
    const int m_lo = sect_all ? blockIdx.y : 0, m_hi = sect_all ? m_lo : Pn;
    for (int m = m_lo; m <= m_hi; ++m) {
        if (sect_all) {
            const cd* g = sect_all + (tile * (Pn + 1) + m) * (NR + 1) * 32 + lane;
            for (int r = m + w; r <= NR - m; r += nw) sect[r * 32] = g[(size_t)r * 32];
        } else if (m == 0) {
            for (int r = w; r <= NR; r += nw) sect[r * 32] = coax_g(r) * f[r * 32];
        } else {
            // T^m_{r,m} from T^{m-1}_{r+-1,m-1}
            for (int r = m + w; r <= NR - m; r += nw)
                b1[r * 32] = rmac(__ldg(C.smu + nmi(r, m)) * sect[(r + 1) * 32], __ldg(C.snu + nmi(r, m)),
                                  sect[(r - 1) * 32]);
            cd* x = sect;
            sect = b1;
            b1 = x;
        }
        cd* Tm = T + tri_off(Pm, m) * 32;
        __syncthreads();
        double g = __ldg(C.cg + nmi(m, m));
        for (int r = m + w; r <= Pm; r += nw) Tm[(size_t)(r - m) * (r - m + 1) / 2 * 32] = g * sect[r * 32];
        cd *prv = nullptr, *cur = sect;
        for (int c = m; c < Pn; ++c) {
            // the next column goes over the one before the current (a row reads only its
            // own entry of that), but the sectorial one stays for the next m
            cd* nxt = c == m ? b1 : c == m + 1 ? b2 : prv;
            double ab = __ldg(C.ab + nmi(c, m));
            g = __ldg(C.cg + nmi(c + 1, m));
            for (int r = c + 1 + w; r <= NR - c - 1; r += nw) {
                cd v = __ldg(C.be + nmi(r - 1, m)) * cur[(r - 1) * 32];
                v = rmac(v, -__ldg(C.al + nmi(r + 1, m)), cur[(r + 1) * 32]);
                if (c > m) v = rmac(v, ab, prv[r * 32]);
                nxt[r * 32] = v;
                if (r <= Pm) Tm[((size_t)(r - m) * (r - m + 1) / 2 + (c + 1 - m)) * 32] = g * v;
            }
            __syncthreads();
            prv = cur;
            cur = nxt;
        }
        __syncthreads();
    }
}

// The fixed matrices satisfy D[-m][m'] = D[m][-m'] = (-1)^{n+m+m'} D[m][m']. With
// w+-_{m'} = x_{m'} +- (-1)^{m'} x_{-m'} (m' > 0), rows +-m of D x follow from one
// half-row pass over m' > 0, E and O the sums over even and odd m':
//   n+m even:  y_{+-m} = D[m][0] x_0 + E +- O  (with w+)
//   n+m odd:   y_m = E + O,  y_{-m} = O - E    (with w-; D[m][0] = 0)
// y = D x for order n from w+- of x (w+ in rows n .. 2n of buf, w- in rows n-1 ..
// 0), rows +-m handed to emit(m, y_m, y_-m). The warps
// take the rows of one parity of n + m each, four rows at a time: one 512-byte row
// of w+- and four uniform table entries feed 8 FP64 instructions.
template <class F>
__device__ __forceinline__ void rot_rows(const double* __restrict__ D, const cd* buf, int n, int w, int nw, F emit) {
    const int N1 = n + 1, odd = w & 1, nsub = nw >> 1;
    for (int i0 = w >> 1; ((n + odd) & 1) + 2 * i0 <= n; i0 += 4 * nsub) {
        int m[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) m[k] = ((n + odd) & 1) + 2 * (i0 + k * nsub);
        const int last = m[3] <= n ? 4 : m[2] <= n ? 3 : m[1] <= n ? 2 : 1;
        cd E[4], O[4];
        const cd* wv = buf + n * 32;
        if (odd) {
#pragma unroll
            for (int k = 0; k < 4; ++k) E[k] = cd{0, 0};
        } else {
            cd x0 = wv[0];
#pragma unroll
            for (int k = 0; k < 4; ++k) E[k] = __ldg(D + min(m[k], n)) * x0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) O[k] = cd{0, 0};
        const int st = odd ? -32 : 32;
        auto body = [&](auto cnt) {
            constexpr int R = decltype(cnt)::value;
#pragma unroll 2
            for (int mp = 1; mp < n; mp += 2) {
                cd u = wv[mp * st], v = wv[(mp + 1) * st];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    O[k] = rmac(O[k], __ldg(D + mp * N1 + m[k]), u);
                    E[k] = rmac(E[k], __ldg(D + (mp + 1) * N1 + m[k]), v);
                }
            }
            if (n & 1) {
                cd u = wv[n * st];
#pragma unroll
                for (int k = 0; k < R; ++k) O[k] = rmac(O[k], __ldg(D + n * N1 + m[k]), u);
            }
#pragma unroll
            for (int k = 0; k < R; ++k) emit(m[k], E[k] + O[k], odd ? O[k] - E[k] : E[k] - O[k]);
        };
        if (last == 4) body(std::integral_constant<int, 4>{});
        else if (last == 3) body(std::integral_constant<int, 3>{});
        else if (last == 2) body(std::integral_constant<int, 2>{});
        else body(std::integral_constant<int, 1>{});
    }
}

// w+- of x_{+-m} into the rows of buf
__device__ __forceinline__ void put_w(cd* buf, int n, int m, cd xp, cd xm) {
    if (m == 0) {
        buf[n * 32] = xp;
        return;
    }
    xm = sgn(m, xm);
    buf[(n + m) * 32] = xp + xm;
    buf[(n - m) * 32] = xp - xm;
}

// Forward rotation. Grid (rhs x direction, tile, order group): orders n = Pi - g,
// Pi - g - groups, .. Two buffers of 2Pm+1 rows in shared memory. For Helmholtz the
// last matrix pass uses Dg, so that V holds a_n (-1)^n/(2n+1), the vector the
// coaxial product wants.
template <bool LAP>
__global__ void __launch_bounds__(256) k_pair_fwd(PairArgs A, const cd* __restrict__ mp) {
    extern __shared__ cd sm[];
    const int P = A.Pm, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int dir = A.dir(blockIdx.x), rhs = A.rhs(blockIdx.x);
    const size_t tile = blockIdx.y, K = A.K();
    const int p = 32 * (int)tile + lane;
    const int src = dir ? A.a(p) : A.b(p), kd = src < 0 ? kPairFlat : A.kind[32 * A.t0 + p];
    const bool flat = __all_sync(0xffffffffu, kd == kPairFlat), iso = __any_sync(0xffffffffu, kd >= kPairIso);
    const cd* c = mp + (int64_t)rhs * A.ncoef + (src < 0 ? 0 : A.eoff[src]);
    const cd* pe = A.pw + (tile * (4 * P + 2) + P) * 32 + lane;      // e^m at pe[32 m]
    const cd* pa = pe + (2 * P + 1) * 32;
    cd* V = A.vec + ((size_t)blockIdx.x * A.ntile + tile) * K * 32 + lane;
    cd *b1 = sm + lane, *b2 = b1 + (size_t)(2 * P + 1) * 32;
    auto load = [&](int n, int m) -> cd {
        if (src < 0) return cd{0, 0};
        cd v = c[nmi(n, m)];
        return LAP ? __ldg(A.s_in + nmi(n, m)) * v : v;
    };
    // powers of this direction's e (e' = -e) and e_a (e_a' = -1/e_a)
    auto ep = [&](int m) -> cd { return src < 0 ? cd{0, 0} : dir ? sgn(m, pe[m * 32]) : pe[m * 32]; };
    auto ap = [&](int m) -> cd { return src < 0 ? cd{0, 0} : dir ? sgn(m, pa[-m * 32]) : pa[m * 32]; };
    for (int n = A.Pi - (int)blockIdx.z; n >= 0; n -= gridDim.z) {
        const double* D = A.T.Dh + __ldg(A.T.Dhoff + n);
        const double* Dl = LAP ? D : A.T.Dg + __ldg(A.T.Dhoff + n);
        auto out = [&](int m, cd yp, cd ym) {
            V[(size_t)nmi(n, m) * 32] = yp;
            if (m > 0) V[(size_t)nmi(n, -m) * 32] = ym;
        };
        __syncthreads();
        if (iso) {
            // isotropic pairs: into the frame of Q_k first (D E(i^k) c), left in b2
            for (int m = w; m <= n; m += nw) {
                int k = kd >= kPairIso ? kd - kPairIso : 0;
                put_w(b1, n, m, ipow(k * m, load(n, m)), ipow(-k * m, load(n, -m)));
            }
            __syncthreads();
            rot_rows(D, b1, n, w, nw, [&](int m, cd yp, cd ym) {
                b2[(n + m) * 32] = kd >= kPairIso ? yp : load(n, m);
                if (m > 0) b2[(n - m) * 32] = kd >= kPairIso ? ym : load(n, -m);
            });
            __syncthreads();
        }
        for (int m = w; m <= n; m += nw) {
            cd xp = iso ? b2[(n + m) * 32] : load(n, m), xm = iso ? b2[(n - m) * 32] : load(n, -m);
            xp = xp * ep(m);
            xm = xm * ep(-m);
            if (flat) put_w(b1, n, m, xp, xm);
            else put_w(b1, n, m, ipow(m, xp), ipow(-m, xm));
        }
        __syncthreads();
        if (flat) {
            rot_rows(Dl, b1, n, w, nw, out);
            continue;
        }
        rot_rows(D, b1, n, w, nw, [&](int m, cd yp, cd ym) {
            put_w(b2, n, m, sgn(m, yp * ap(m)), sgn(m, ym * ap(-m)));
        });
        __syncthreads();
        rot_rows(Dl, b2, n, w, nw, [&](int m, cd yp, cd ym) { out(m, ipow(m, yp), ipow(-m, ym)); });
    }
}

// Backward rotation, in place: flat E(1/e) S D S c', else E(1/e) i^m D S E(1/e_a) D
// Phi c', and isotropic pairs out of their frame at the end (E(i^-k) S D S).
template <bool LAP>
__global__ void __launch_bounds__(256) k_pair_bwd(PairArgs A) {
    extern __shared__ cd sm[];
    const int P = A.Pm, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int dir = A.dir(blockIdx.x);
    const size_t tile = blockIdx.y, K = A.K();
    const int p = 32 * (int)tile + lane;
    const bool none = A.a(p) < 0;
    const int kd = none ? kPairFlat : A.kind[32 * A.t0 + p];
    const bool flat = __all_sync(0xffffffffu, kd == kPairFlat), iso = __any_sync(0xffffffffu, kd >= kPairIso);
    const cd* pe = A.pw + (tile * (4 * P + 2) + P) * 32 + lane;
    const cd* pa = pe + (2 * P + 1) * 32;
    cd* V = A.vec + ((size_t)blockIdx.x * A.ntile + tile) * K * 32 + lane;
    cd *b1 = sm + lane, *b2 = b1 + (size_t)(2 * P + 1) * 32;
    auto epi = [&](int m) -> cd { return none ? cd{0, 0} : dir ? sgn(m, pe[-m * 32]) : pe[-m * 32]; };
    auto api = [&](int m) -> cd { return none ? cd{0, 0} : dir ? sgn(m, pa[m * 32]) : pa[-m * 32]; };
    for (int n = A.Po - (int)blockIdx.z; n >= 0; n -= gridDim.z) {
        const double* D = A.T.Dh + __ldg(A.T.Dhoff + n);
        auto out = [&](int m, cd yp, cd ym) {
            V[(size_t)nmi(n, m) * 32] = yp;
            if (m > 0) V[(size_t)nmi(n, -m) * 32] = ym;
        };
        __syncthreads();
        for (int m = w; m <= n; m += nw) {
            // (no entries beyond |m| = Pi)
            cd xp = {0, 0}, xm = {0, 0};
            if (m <= A.Pn) {
                xp = V[(size_t)nmi(n, m) * 32];
                xm = V[(size_t)nmi(n, -m) * 32];
            }
            if (flat) put_w(b1, n, m, sgn(m, xp), sgn(m, xm));
            else put_w(b1, n, m, ipow(m, xp), ipow(-m, xm));
        }
        __syncthreads();
        if (flat) {
            rot_rows(D, b1, n, w, nw, [&](int m, cd yp, cd ym) { out(m, sgn(m, yp * epi(m)), sgn(m, ym * epi(-m))); });
            continue;
        }
        rot_rows(D, b1, n, w, nw, [&](int m, cd yp, cd ym) {
            put_w(b2, n, m, sgn(m, yp * api(m)), sgn(m, ym * api(-m)));
        });
        __syncthreads();
        rot_rows(D, b2, n, w, nw, [&](int m, cd yp, cd ym) {
            yp = ipow(m, yp) * epi(m);
            ym = ipow(-m, ym) * epi(-m);
            if (iso) put_w(b1, n, m, sgn(m, yp), sgn(m, ym));
            if (kd < kPairIso) out(m, yp, ym);
        });
        if (!iso) continue;
        __syncthreads();
        rot_rows(D, b1, n, w, nw, [&](int m, cd yp, cd ym) {
            int k = kd - kPairIso;
            if (kd >= kPairIso) out(m, sgn(m, ipow(-k * m, yp)), sgn(m, ipow(k * m, ym)));
        });
    }
}

// Coaxial product at one m <= Pn of a tile, in place: out_n = sum_k T'_{max(n,k),
// min(n,k)} a_k, n <= Po, k <= Pi, for the NV vectors of the tile (M2L: two
// directions, +m and -m). Laplace in the solid-harmonic basis (s_mid, s_out turn the
// Y-basis coefficients into it and back), f the radial rows:
//   M2L out_n = (-1)^{n+m} sum_k f_{n+k} a_k,  M2M sum_{k<=n} f_{n-k} a_k,  L2L sum_{k>=n} f_{k-n} a_k.
// Grid (rhs, tile, m): the right-hand sides of a tile's T run side by side. The
// block's vectors sit in shared memory; a warp takes every fourth n, four at a time,
// so a loaded entry feeds 4 NV FP64 instructions.
template <bool LAP, int MODE>
__global__ void __launch_bounds__(kPairThreads) k_pair_coax(PairArgs A) {
    extern __shared__ cd sm[];
    constexpr int NV = MODE == 1 ? 4 : 2, ND = NV / 2;
    const int m = blockIdx.z, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kPairThreads / 32;
    const size_t tile = blockIdx.y, K = A.K();
    const int rhs = blockIdx.x, nk = A.Pi - m + 1, n1 = A.Po - m + 1;
    cd* V[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) V[d] = A.vec + ((size_t)(ND * rhs + d) * A.ntile + tile) * K * 32 + lane;
    cd* a = sm + lane;                                  // [nk][NV]: +m, -m per direction
    for (int k = w; k < nk; k += nw) {
        double sp = LAP ? __ldg(A.s_mid + nmi(m + k, m)) : 1.0, sn = LAP ? __ldg(A.s_mid + nmi(m + k, -m)) : 1.0;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            cd vp = V[d][(size_t)nmi(m + k, m) * 32], vm = m ? V[d][(size_t)nmi(m + k, -m) * 32] : cd{0, 0};
            a[(NV * k + 2 * d) * 32] = LAP ? sp * vp : vp;
            a[(NV * k + 2 * d + 1) * 32] = LAP ? sn * vm : vm;
        }
    }
    __syncthreads();
    const cd* T = LAP ? A.fl + tile * (A.Pi + A.Po + 1) * 32 + lane
                      : A.tri + (tile * tri_off(A.Pm, A.Pm + 1) + tri_off(A.Pm, m)) * 32 + lane;
    auto entry = [&](int i, int k) -> cd {              // rows n = m + i and m + k
        if (LAP) {
            if (MODE == 1) return T[(size_t)(2 * m + i + k) * 32];
            int j = MODE == 0 ? i - k : k - i;
            return j >= 0 ? T[(size_t)j * 32] : cd{0, 0};
        }
        int hi = max(i, k), lo = min(i, k);
        return T[(size_t)(hi * (hi + 1) / 2 + lo) * 32];
    };
    for (int i0 = w; i0 < n1; i0 += 4 * nw) {
        auto body = [&](auto cnt) {
            constexpr int R = decltype(cnt)::value;
            cd s[R][NV];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int v = 0; v < NV; ++v) s[r][v] = cd{0, 0};
            // Laplace M2M and L2L: the terms beyond the triangle are zero
            int k0 = LAP && MODE == 2 ? i0 : 0, k1 = LAP && MODE == 0 ? min(nk, i0 + (R - 1) * nw + 1) : nk;
            for (int k = k0; k < k1; ++k) {
                cd t[R];
#pragma unroll
                for (int r = 0; r < R; ++r) t[r] = entry(i0 + r * nw, k);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    if (m == 0 && (v & 1)) continue;
                    cd x = a[(NV * k + v) * 32];
#pragma unroll
                    for (int r = 0; r < R; ++r) s[r][v] = cmac(s[r][v], t[r], x);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int n = m + i0 + r * nw;
                double gp = 1.0, gn = 1.0;
                if (LAP) {
                    double e = MODE == 1 && ((n + m) & 1) ? -1.0 : 1.0;
                    gp = e * __ldg(A.s_out + nmi(n, m));
                    gn = e * __ldg(A.s_out + nmi(n, -m));
                }
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    if (m == 0 && (v & 1)) continue;
                    V[v >> 1][(size_t)nmi(n, (v & 1) ? -m : m) * 32] = LAP ? ((v & 1) ? gn : gp) * s[r][v] : s[r][v];
                }
            }
        };
        int rows = (n1 - i0 + nw - 1) / nw;
        if (rows >= 4) body(std::integral_constant<int, 4>{});
        else if (rows == 3) body(std::integral_constant<int, 3>{});
        else if (rows == 2) body(std::integral_constant<int, 2>{});
        else body(std::integral_constant<int, 1>{});
    }
}

// Destination boxes lo + blockIdx.x. M2L: out (+)= sum over the box's List-2 entries
// whose slot is in the range; M2M: out = sum over the children of a box (a leaf keeps
// its P2M expansion); L2L: out += the parent's vector.
template <bool LAP>
__global__ void k_pair_sum(PairArgs A, int lo, const int* __restrict__ q_beg, const int* __restrict__ q_end,
                           const int* __restrict__ slot, const int* __restrict__ leaf, int first,
                           cd* __restrict__ out) {
    const int b = lo + blockIdx.x, rhs = blockIdx.y, K = (A.Po + 1) * (A.Po + 1);
    if (A.mode == 0 && leaf[b]) return;
    int q0 = A.mode == 2 ? b : q_beg[b], q1 = A.mode == 2 ? b + 1 : q_end[b];
    if (A.mode == 0) {
        // children of the range; a box's sum starts with its first child's range
        first = q0 >= A.lo;
        q0 = max(q0, A.lo);
        q1 = min(q1, A.hi);
        if (q0 >= q1) return;
    }
    const size_t KV = A.K();
    cd* o = out + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int k = blockIdx.z * blockDim.x + threadIdx.x; k < K; k += gridDim.z * blockDim.x) {
        cd s = {0, 0};
#pragma unroll 4
        for (int q = q0; q < q1; ++q) {
            int v = rhs, p = q - A.lo;
            if (A.mode == 1) {
                int u = slot[q] - 64 * A.t0;
                if (u < 0 || u >= 64 * A.ntile) continue;
                v = 2 * rhs + (u & 1);
                p = u >> 1;
            }
            s += A.vec[(((size_t)v * A.ntile + (p >> 5)) * KV + k) * 32 + (p & 31)];
        }
        if (LAP) s = __ldg(A.s_fin + k) * s;
        o[k] = first ? s : o[k] + s;
    }
}

// shared memory of the stages
constexpr size_t kPairRow = 32 * sizeof(cd);
constexpr size_t rot_bytes(int Pm) { return 2 * (size_t)(2 * Pm + 1) * kPairRow; }
constexpr size_t tri_bytes(int NR) { return 3 * (size_t)(NR + 2) * kPairRow; }
constexpr size_t sect_bytes(int NR) { return 2 * (size_t)(NR + 2) * kPairRow; }
constexpr size_t coax_bytes(int mode, int Pi) { return (mode == 1 ? 4 : 2) * (size_t)(Pi + 1) * kPairRow; }

// blocks of twice the warps where shared memory leaves one or two an SM
constexpr int pair_threads(int Pm) { return Pm > 40 ? 2 * kPairThreads : kPairThreads; }

}  // namespace

void init_pairs3d() {
    constexpr int P = kMaxP3Top;
    auto set = [](const void* f, size_t smem) {
        CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    };
    for (auto f : {(const void*)k_pair_fwd<true>, (const void*)k_pair_fwd<false>, (const void*)k_pair_bwd<true>,
                   (const void*)k_pair_bwd<false>})
        set(f, rot_bytes(P));
    set((const void*)k_pair_tri, tri_bytes(2 * P));
    set((const void*)k_pair_sect, sect_bytes(2 * P));
    for (auto f : {(const void*)k_pair_coax<true, 1>, (const void*)k_pair_coax<false, 1>}) set(f, coax_bytes(1, P));
    for (auto f : {(const void*)k_pair_coax<true, 0>, (const void*)k_pair_coax<false, 0>,
                   (const void*)k_pair_coax<true, 2>, (const void*)k_pair_coax<false, 2>})
        set(f, coax_bytes(0, P));
}

void pair_slots_build(cfmm_plan_s* P, PairSlots* S, const std::vector<int>& l2off, int l0) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    const int nent = l2off[T.nboxes];
    const int nb = T.nboxes, nlev = T.nlevels;
    S->tile0.assign(nlev + 1, 0);
    S->d_tile0.alloc(nlev + 1);
    int *cnt = nullptr, *pos = nullptr;
    auto slots = [&](int* box_a, int* box_b, signed char* kind, int* slot) {
        k_pair_slots<<<(unsigned)(((int64_t)nb * 32 + 127) / 128), 128, 0, st>>>(
            nb, T.loff[1].get(), T.lent[1].get(), T.level.get(), T.d_level_off.get(), S->d_tile0.get(), T.cen_re.get(),
            T.cen_im.get(), source_range(P), target_range(P), cnt, pos, box_a, box_b, kind, slot);
        CFMM_LAUNCHED();
    };
    std::vector<int> off(2 * (nlev + 1), 0);
    if (nent > 0) {
        cnt = plan_scratch().take_n<int>(2 * (size_t)nb + 1);
        pos = plan_scratch().take_n<int>(2 * (size_t)nb + 1);
        slots(nullptr, nullptr, nullptr, nullptr);
        scan_exclusive_async(cnt, pos, 2 * nb + 1, st);
        if (P->n_trg > 0) {
            int* d_off = plan_scratch().take_n<int>(off.size());
            k_pair_levels<<<1, 64, 0, st>>>(nlev, nb, T.d_level_off.get(), pos, d_off);
            CFMM_LAUNCHED();
            CFMM_CUDA(cudaMemcpyAsync(off.data(), d_off, sizeof(int) * off.size(), cudaMemcpyDeviceToHost, st));
            CFMM_CUDA(cudaStreamSynchronize(st));
        }
    }
    auto tiles = [](int n) { return (n + 31) / 32; };
    for (int l = 0; l < nlev; ++l) {
        const int pairs = (l2off[T.level_off[l + 1]] - l2off[T.level_off[l]]) / 2;
        // flat and other pairs each end with a partial tile
        S->tile0[l + 1] = S->tile0[l] + (l < l0         ? 0
                                         : P->n_trg > 0 ? tiles(off[l + 1] - off[l]) + tiles(off[nlev + 2 + l] - off[nlev + 1 + l])
                                         : pairs        ? tiles(pairs) + 1
                                                        : 0);
    }
    S->nslot = (int64_t)32 * S->tile0[nlev];
    if (nent <= 0) return;
    S->slot.alloc(nent);
    S->box_a.alloc(std::max<int64_t>(1, S->nslot));
    S->box_b.alloc(std::max<int64_t>(1, S->nslot));
    S->kind.alloc(std::max<int64_t>(1, S->nslot));
    CFMM_CUDA(cudaMemsetAsync(S->box_a.get(), 0xff, sizeof(int) * S->nslot, st));
    CFMM_CUDA(cudaMemsetAsync(S->box_b.get(), 0xff, sizeof(int) * S->nslot, st));
    upload(S->d_tile0.get(), S->tile0.data(), sizeof(int) * (nlev + 1), st);
    slots(S->box_a.get(), S->box_b.get(), S->kind.get(), S->slot.get());
}

namespace {

// right-hand sides of a range whose vectors fit beside its operators
int range_rhs(bool lap, const PairArgs& A, int per_rhs, int nrhs) {
    const size_t tile = (lap ? 0 : tri_off(A.Pm, A.Pm + 1)) * kPairRow, v = (size_t)per_rhs * A.K() * kPairRow;
    const size_t nt = std::max(1, A.ntile), left = kPairBudget > nt * tile ? kPairBudget - nt * tile : 0;
    return (int)std::max<size_t>(1, std::min<size_t>(nrhs, left / (nt * v)));
}

// one range of tiles of A: the pairs' powers, radial rows and operators
template <bool LAP, int MODE>
void launch_pairs(PairArgs& A, PairSlots* S, int batch, int nsm, cudaStream_t st) {
    const int nt = A.ntile, NR = A.Pi + A.Po;
    if (nt <= 0) return;
    const size_t K = A.K();
    S->pw.alloc((size_t)nt * (4 * A.Pm + 2) * 32);
    S->fl.alloc((size_t)nt * (NR + 1) * 32);
    S->vec.alloc((size_t)nt * batch * (MODE == 1 ? 2 : 1) * K * 32);
    if (!LAP) S->tri.alloc((size_t)nt * tri_off(A.Pm, A.Pm + 1) * 32);
    if (MODE != 1) {
        S->kind_c.alloc((size_t)nt * 32);
        A.kind = S->kind_c.get();
    }
    A.pw = S->pw.get();
    A.fl = S->fl.get();
    A.vec = S->vec.get();
    A.tri = S->tri.get();
    k_pair_pre<LAP><<<(nt + 3) / 4, 128, 0, st>>>(A);
    CFMM_LAUNCHED();
    if (!LAP) {
        const bool split = nt < 4 * nsm;
        if (split) {
            S->sect.alloc((size_t)nt * (A.Pn + 1) * (NR + 1) * 32);
            k_pair_sect<<<nt, 256, sect_bytes(NR), st>>>(A, S->sect.get());
            CFMM_LAUNCHED();
        }
        k_pair_tri<<<dim3(nt, split ? A.Pn + 1 : 1), pair_threads(A.Pm), tri_bytes(NR), st>>>(A, split ? S->sect.get() : nullptr);
        CFMM_LAUNCHED();
    }
}

// the vectors of `nrhs` right-hand sides through them: everything but the sum
template <bool LAP, int MODE>
void launch_vectors(const PairArgs& A, const cd* in, int nrhs, int nsm, cudaStream_t st) {
    const int nt = A.ntile, nv = nrhs * (MODE == 1 ? 2 : 1), wide = pair_threads(A.Pm);
    if (nt <= 0) return;
    const size_t rot_smem = rot_bytes(A.Pm), cx_smem = coax_bytes(MODE, A.Pi);
    // small launches: one thread block per order as well
    auto groups = [&](int P) {
        return (unsigned)std::min<int64_t>(P + 1, std::max<int64_t>(1, (int64_t)8 * nsm / ((int64_t)nt * nv)));
    };
    k_pair_fwd<LAP><<<dim3(nv, nt, groups(A.Pi)), wide, rot_smem, st>>>(A, in);
    CFMM_LAUNCHED();
    k_pair_coax<LAP, MODE><<<dim3(nrhs, nt, A.Pn + 1), kPairThreads, cx_smem, st>>>(A);
    CFMM_LAUNCHED();
    k_pair_bwd<LAP><<<dim3(nv, nt, groups(A.Po)), wide, rot_smem, st>>>(A);
    CFMM_LAUNCHED();
}

// Tiles of a range: T (Helmholtz) and V of kPairRhs right-hand sides within the budget.
// The number of right-hand sides has no part in it: where a box's pairs fall into several
// ranges, the cuts decide the order of its sum, and a right-hand side's result is the same
// alone and among others. (4: a single one leaves half the budget unused, and T is read
// once for every four of several.)
constexpr int kPairRhs = 4;
int range_tiles(bool lap, int Pm, int per_rhs) {
    const size_t K = (size_t)(Pm + 1) * (Pm + 1);
    const size_t per = ((lap ? 0 : tri_off(Pm, Pm + 1)) + (size_t)(kPairRhs * per_rhs) * K) * kPairRow;
    return (int)std::max<size_t>(1, std::min<size_t>(kPairBudget / per, 65535));
}

template <bool LAP>
void launch_sum(const PairArgs& A, int lo, int nb, const int* q_beg, const int* q_end, const int* slot, const int* leaf,
                bool first, cd* out, int nrhs, int nsm, cudaStream_t st) {
    const int K = (A.Po + 1) * (A.Po + 1);
    dim3 g(nb, nrhs, (unsigned)std::max(1, std::min((K + 127) / 128, 8 * nsm / nb)));
    k_pair_sum<LAP><<<g, 128, 0, st>>>(A, lo, q_beg, q_end, slot, leaf, first ? 1 : 0, out);
    CFMM_LAUNCHED();
}

PairArgs pair_args(cfmm_plan_s* P, const Tr3Tables& T, int mode, int Pi, int Po, double kappa, const int64_t* eoff,
                   int64_t ncoef) {
    TreeDev& Tr = P->tree;
    PairArgs A{};
    A.cre = Tr.cen_re.get();
    A.cim = Tr.cen_im.get();
    A.parent = Tr.parent.get();
    A.T = T;
    A.eoff = eoff;
    A.ncoef = ncoef;
    A.mode = mode;
    A.Pi = Pi;
    A.Po = Po;
    A.Pm = std::max(Pi, Po);
    A.Pn = std::min(Pi, Po);
    A.kappa = kappa;
    // Y basis: eps s M (multipole), eps L / s (local)
    A.s_in = mode == 2 ? T.lsd : T.lsm;
    A.s_mid = mode == 2 ? T.lsm : T.lsd;
    A.s_out = mode == 0 ? T.lsm : T.lsd;
    A.s_fin = mode == 0 ? T.lsd : T.lsm;
    return A;
}

int sm_count(cfmm_plan_s* P) {
    int nsm = 0;
    CFMM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, P->device));
    return nsm;
}

template <bool LAP>
void launch_m2l(cfmm_plan_s* P, PairSlots* S, PairArgs A, int l_lo, int l_hi, const cd* mp, cd* lc, int nrhs) {
    TreeDev& Tr = P->tree;
    const int lo = Tr.level_off[l_lo], nb = Tr.level_off[l_hi] - lo, nsm = sm_count(P);
    if (nb <= 0) return;
    A.box_a = S->box_a.get();
    A.box_b = S->box_b.get();
    A.kind = S->kind.get();
    const int cap = range_tiles(LAP, A.Pm, 2), end = S->tile0[l_hi];
    bool first = true;
    A.t0 = S->tile0[l_lo];
    do {                       // (also without pairs: the boxes' expansions become zero)
        A.ntile = std::min(cap, end - A.t0);
        const int batch = range_rhs(LAP, A, 2, nrhs);
        launch_pairs<LAP, 1>(A, S, batch, nsm, P->stream);
        for (int r = 0; r < nrhs; r += batch) {
            const int nr = std::min(batch, nrhs - r);
            launch_vectors<LAP, 1>(A, mp + (int64_t)r * A.ncoef, nr, nsm, P->stream);
            launch_sum<LAP>(A, lo, nb, Tr.loff[1].get(), Tr.loff[1].get() + 1, S->slot.get(), nullptr, first,
                            lc + (int64_t)r * A.ncoef, nr, nsm, P->stream);
        }
        first = false;
        A.t0 += A.ntile;
    } while (A.t0 < end);
}

// M2M of the boxes of level l from their children (mode 0), L2L of the boxes of level
// l + 1 from their parents (mode 2), in ranges of children that fit the budget
template <bool LAP, int MODE>
void launch_child(cfmm_plan_s* P, PairSlots* S, PairArgs A, int l, const cd* in, cd* out, int nrhs) {
    TreeDev& Tr = P->tree;
    const int c0 = Tr.level_off[l + 1], c1 = Tr.level_off[l + 2], nsm = sm_count(P);
    const int64_t need = ((int64_t)(c1 - c0) + 31) / 32;
    const int cap = range_tiles(LAP, A.Pm, 1);
    for (int64_t t = 0; t < need; t += cap) {
        A.ntile = (int)std::min<int64_t>(cap, need - t);
        A.lo = c0 + (int)(32 * t);
        A.hi = (int)std::min<int64_t>(c1, (int64_t)A.lo + 32 * (int64_t)A.ntile);
        const int batch = range_rhs(LAP, A, 1, nrhs);
        launch_pairs<LAP, MODE>(A, S, batch, nsm, P->stream);
        for (int r = 0; r < nrhs; r += batch) {
            const int nr = std::min(batch, nrhs - r);
            const int64_t at = (int64_t)r * A.ncoef;
            launch_vectors<LAP, MODE>(A, in + at, nr, nsm, P->stream);
            if (MODE == 0)
                launch_sum<LAP>(A, Tr.level_off[l], Tr.level_off[l + 1] - Tr.level_off[l], Tr.cbeg.get(), Tr.cend.get(),
                                nullptr, Tr.leaf.get(), true, out + at, nr, nsm, P->stream);
            else
                launch_sum<LAP>(A, A.lo, A.hi - A.lo, nullptr, nullptr, nullptr, nullptr, false, out + at, nr, nsm,
                                P->stream);
        }
    }
}

}  // namespace

void pairs3d_m2l(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l_lo, int l_hi, int Pord, double kappa,
                 const int64_t* eoff, int64_t ncoef, const cd* mp, cd* lc, int nrhs) {
    PairArgs A = pair_args(P, T, 1, Pord, Pord, kappa, eoff, ncoef);
    if (kappa == 0.0) launch_m2l<true>(P, S, A, l_lo, l_hi, mp, lc, nrhs);
    else launch_m2l<false>(P, S, A, l_lo, l_hi, mp, lc, nrhs);
}

void pairs3d_m2m(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l, int Pc, int Pp, double kappa,
                 const int64_t* eoff, int64_t ncoef, cd* mp, int nrhs) {
    PairArgs A = pair_args(P, T, 0, Pc, Pp, kappa, eoff, ncoef);
    if (kappa == 0.0) launch_child<true, 0>(P, S, A, l, mp, mp, nrhs);
    else launch_child<false, 0>(P, S, A, l, mp, mp, nrhs);
}

void pairs3d_l2l(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l, int Pp, int Pc, double kappa,
                 const int64_t* eoff, int64_t ncoef, cd* lc, int nrhs) {
    PairArgs A = pair_args(P, T, 2, Pp, Pc, kappa, eoff, ncoef);
    if (kappa == 0.0) launch_child<true, 2>(P, S, A, l, lc, lc, nrhs);
    else launch_child<false, 2>(P, S, A, l, lc, lc, nrhs);
}

}  // namespace cfmm

// 3D M2L (List 2), Laplace and Helmholtz: point-and-shoot translation (the
// scheme, operators and recurrences of helm3d.cu's file comment) with 32 pairs
// on the lanes of a warp.
//
// The FP64 pipe bounds it (one warp instruction per 16 SM cycles), so the work
// is arranged to issue as few FP64 instructions as the operators allow, each with
// 32 lanes in use:
//   * a lane is a pair. Every lane does the same (n, m, m') at the same time: no
//     partial warps at the ends of rows and orders, rotation table entries are
//     uniform, per-pair factors sit in [..][32] rows that load as 512 bytes.
//   * both directions of a pair (a <- b, b <- a) share the shift's length and so
//     the coaxial operator T: it is built once per unordered pair and each entry,
//     once loaded, serves 4 vectors (two directions, +m and -m). The reversed
//     shift has e' = -e and e_a' = -1/e_a.
//   * a shift with d3 = 0 (boxes in one layer, equal Im of the third centre
//     coordinate; most pairs of a flat surface) has e_a = i exactly, and the
//     rotation D^T E(i) D between the diagonal factors is the fixed matrix D
//     itself: one real matrix pass and one diagonal scaling instead of two each.
// Stages, each reading and writing the pair vectors V[dir][tile][coef][32]:
//   k_pair_pre    powers e^m, e_a^m and the radial sequence of each pair
//   k_pair_tri    coaxial triangles T (Helmholtz)
//   k_pair_fwd    gather the source expansion, rotate (per order n)
//   k_pair_coax   coaxial product (per m), in place
//   k_pair_bwd    rotate back (per order n), in place
//   k_pair_sum    add the vectors of a box's List 2 in list order
// Per pair and direction at order 16: 25k FP64 lane instructions + 5k for T,
// against 65k issued by one-block-per-box translation (153 coefficient items on
// 256 threads, both rotations in full, T per direction). V costs 5 passes over
// 16 (P+1)^2 bytes a pair, about a tenth of the time at HBM rate.
#include <algorithm>

#include "cfmm_special.cuh"
#include "m2l3d.cuh"

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
__host__ __device__ inline size_t tri_off(int P, int m) {      // entries of the triangles before m
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

// One thread per List-2 entry (a, b), a < b. Flat pairs fill their level's slots
// from the front, the others from the back, so a tile holds one sort only and a
// pair's arithmetic does not depend on its slot.
__global__ void k_pair_slots(int nent, const int* __restrict__ loff, const int* __restrict__ lent, int nbox,
                             const int* __restrict__ level, const int* __restrict__ tile0,
                             const double* __restrict__ cre, const double* __restrict__ cim, int* __restrict__ count,
                             int* __restrict__ box_a, int* __restrict__ box_b, signed char* __restrict__ kind,
                             int* __restrict__ slot) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nent) return;
    int lo = 0, hi = nbox - 1;                    // owner: last box with loff <= q
    while (lo < hi) {
        int m = (lo + hi + 1) >> 1;
        if (loff[m] <= q) lo = m;
        else hi = m - 1;
    }
    int a = lo, b = lent[q];
    if (b <= a) return;
    lo = loff[b];                                 // a in the list of b (sorted; List 2 is symmetric)
    hi = loff[b + 1] - 1;
    while (lo < hi) {
        int m = (lo + hi) >> 1;
        if (lent[m] < a) lo = m + 1;
        else hi = m;
    }
    cd d[3];
    int kd = pair_shift(cre, cim, a, b, d), l = level[a];
    int i = atomicAdd(count + 2 * l + (kd == kPairFlat ? 0 : 1), 1);
    int p = kd == kPairFlat ? 32 * tile0[l] + i : 32 * tile0[l + 1] - 1 - i;
    box_a[p] = a;
    box_b[p] = b;
    kind[p] = (signed char)kd;
    slot[q] = 2 * p;
    slot[lo] = 2 * p + 1;
}

struct PairArgs {
    const double *cre, *cim;
    const int *box_a, *box_b;
    const signed char* kind;
    Tr3Tables T;
    const int64_t* eoff;
    int64_t ncoef;
    int P, t0, ntile;         // tiles [t0, t0 + ntile) of the slots
    double kappa;
    cd *pw, *fl, *tri, *vec;  // of this range
};

// e^m, e_a^m (m = -P..P) and, Helmholtz, h_l(kappa t), l <= 2P, or, Laplace,
// l!/t^{l+1}, l <= 2P; one thread per pair, rows [..][32]
template <bool LAP>
__global__ void k_pair_pre(PairArgs A) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 32 * A.ntile) return;
    int P = A.P, a = A.box_a[32 * A.t0 + p];
    if (a < 0) return;
    size_t tile = p >> 5;
    int lane = p & 31;
    cd d[3];
    int kd = pair_shift(A.cre, A.cim, a, A.box_b[32 * A.t0 + p], d);
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
    cd* f = A.fl + tile * (2 * P + 1) * 32 + lane;
    if (LAP) {
        cd it = cinv(t), v = it;
        for (int j = 0; j <= 2 * P; ++j) {
            f[j * 32] = __ldg(A.T.fact + j) * v;
            v = v * it;
        }
    } else {
        // h_n of cfmm_special.cuh's sph_h_seq, written row by row
        cd z = A.kappa * t, ez = cexp_i(z), zi = cinv(z);
        cd h0 = -mul_i(ez * zi), h1 = -(ez * (z + cd{0.0, 1.0})) * (zi * zi);
        f[0] = h0;
        if (P > 0) f[32] = h1;
        for (int n = 1; n < 2 * P; ++n) {
            cd h2 = rmac(-h0, 2.0 * n + 1.0, zi * h1);
            f[(n + 1) * 32] = h2;
            h0 = h1;
            h1 = h2;
        }
    }
}

// Coaxial triangles T'_{rc} = g_c T_{rc}^m, m <= c <= r <= P, g_c = (-1)^c (2c+1),
// of a tile: entries at tri_off(P, m) + (r-m)(r-m+1)/2 + c - m, rows [..][32].
// The block's warps take the rows of a column; the sectorial column and the two
// before the next one live in shared memory, the buffers changing roles:
// T_{r,c+1} = ibe_c (al_c T_{r,c-1} - al_{r+1} T_{r+1,c} + be_{r-1} T_{r-1,c}).
// 8 FP64 instructions a row (10 for the rows kept) bound it; the 3 (2P+2) rows of
// 512 bytes leave 4 blocks an SM at order 16 and 1 at 63, and a block's 4 warps
// alone keep most of the FP64 pipe busy.
__global__ void __launch_bounds__(256) k_pair_tri(PairArgs A) {
    extern __shared__ cd sm[];
    const int P = A.P, NR = 2 * P, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t tile = blockIdx.x, L = (size_t)(NR + 2) * 32;
    cd *sect = sm + lane, *b1 = sect + L, *b2 = b1 + L;
    const cd* f = A.fl + tile * (NR + 1) * 32 + lane;
    cd* T = A.tri + tile * tri_off(P, P + 1) * 32 + lane;
    for (int m = 0; m <= P; ++m) {
        const Tr3Tables& C = A.T;
        if (m == 0) {
            for (int r = w; r <= NR; r += nw) sect[r * 32] = (((r & 1) ? -1.0 : 1.0) * (2.0 * r + 1.0)) * f[r * 32];
        } else {
            // T^m_{r,m} from T^{m-1}_{r+-1,m-1}
            double inu = 1.0 / __ldg(C.nu + nmi(m - 1, m - 1));
            for (int r = m + w; r <= NR - m; r += nw) {
                double mu1 = inu * __ldg(C.mu + nmi(r + 1, m - 1)), nu1 = inu * __ldg(C.nu + nmi(r - 1, m - 1));
                b1[r * 32] = rmac(mu1 * sect[(r + 1) * 32], nu1, sect[(r - 1) * 32]);
            }
            cd* x = sect;
            sect = b1;
            b1 = x;
        }
        cd* Tm = T + tri_off(P, m) * 32;
        __syncthreads();
        for (int r = m + w; r <= P; r += nw) Tm[(size_t)(r - m) * (r - m + 1) / 2 * 32] = coax_g(m) * sect[r * 32];
        cd *prv = nullptr, *cur = sect;
        for (int c = m; c < P; ++c) {
            // the next column goes over the one before the current (a row reads only its
            // own entry of that), but the sectorial one stays for the next m
            cd* nxt = c == m ? b1 : c == m + 1 ? b2 : prv;
            double ib = __ldg(C.ibe + nmi(c, m)), ac = ib * __ldg(C.al + nmi(c, m)), g = coax_g(c + 1);
            for (int r = c + 1 + w; r <= NR - c - 1; r += nw) {
                cd v = (-__ldg(C.al + nmi(r + 1, m))) * cur[(r + 1) * 32];
                if (r - 1 >= m) v = rmac(v, __ldg(C.be + nmi(r - 1, m)), cur[(r - 1) * 32]);
                v = ib * v;
                if (c > m) v = rmac(v, ac, prv[r * 32]);
                nxt[r * 32] = v;
                if (r <= P) Tm[((size_t)(r - m) * (r - m + 1) / 2 + (c + 1 - m)) * 32] = g * v;
            }
            __syncthreads();
            prv = cur;
            cur = nxt;
        }
    }
}

// y = D x for order n from w+- of x (w+ in rows n .. 2n of buf, w- in rows n-1 ..
// 0; see w_pass of helm3d.cu), rows +-m handed to emit(m, y_m, y_-m). The warps
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

// Forward rotation. Grid (rhs x direction, tile, order group): orders n = P - g,
// P - g - groups, .. Two buffers of 2P+1 rows in shared memory. For Helmholtz the
// last matrix pass uses Dg, so that V holds a_n (-1)^n/(2n+1), the vector the
// coaxial product wants.
template <bool LAP>
__global__ void __launch_bounds__(256) k_pair_fwd(PairArgs A, const cd* __restrict__ mp) {
    extern __shared__ cd sm[];
    const int P = A.P, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int dir = blockIdx.x & 1, rhs = blockIdx.x >> 1;
    const size_t tile = blockIdx.y, K = (size_t)(P + 1) * (P + 1);
    const int p = 32 * (A.t0 + (int)tile) + lane;
    const int src = dir ? A.box_a[p] : A.box_b[p], kd = src < 0 ? kPairFlat : A.kind[p];
    const bool flat = __all_sync(0xffffffffu, kd == kPairFlat), iso = __any_sync(0xffffffffu, kd >= kPairIso);
    const cd* c = mp + (int64_t)rhs * A.ncoef + (src < 0 ? 0 : A.eoff[src]);
    const cd* pe = A.pw + (tile * (4 * P + 2) + P) * 32 + lane;      // e^m at pe[32 m]
    const cd* pa = pe + (2 * P + 1) * 32;
    cd* V = A.vec + ((size_t)blockIdx.x * A.ntile + tile) * K * 32 + lane;
    cd *b1 = sm + lane, *b2 = b1 + (size_t)(2 * P + 1) * 32;
    auto load = [&](int n, int m) -> cd {
        if (src < 0) return cd{0, 0};
        cd v = c[nmi(n, m)];
        return LAP ? __ldg(A.T.lsm + nmi(n, m)) * v : v;
    };
    // powers of this direction's e (e' = -e) and e_a (e_a' = -1/e_a)
    auto ep = [&](int m) -> cd { return src < 0 ? cd{0, 0} : dir ? sgn(m, pe[m * 32]) : pe[m * 32]; };
    auto ap = [&](int m) -> cd { return src < 0 ? cd{0, 0} : dir ? sgn(m, pa[-m * 32]) : pa[m * 32]; };
    for (int n = P - (int)blockIdx.z; n >= 0; n -= gridDim.z) {
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
    const int P = A.P, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int dir = blockIdx.x & 1;
    const size_t tile = blockIdx.y, K = (size_t)(P + 1) * (P + 1);
    const int p = 32 * (A.t0 + (int)tile) + lane;
    const bool none = A.box_a[p] < 0;
    const int kd = none ? kPairFlat : A.kind[p];
    const bool flat = __all_sync(0xffffffffu, kd == kPairFlat), iso = __any_sync(0xffffffffu, kd >= kPairIso);
    const cd* pe = A.pw + (tile * (4 * P + 2) + P) * 32 + lane;
    const cd* pa = pe + (2 * P + 1) * 32;
    cd* V = A.vec + ((size_t)blockIdx.x * A.ntile + tile) * K * 32 + lane;
    cd *b1 = sm + lane, *b2 = b1 + (size_t)(2 * P + 1) * 32;
    auto epi = [&](int m) -> cd { return none ? cd{0, 0} : dir ? sgn(m, pe[-m * 32]) : pe[-m * 32]; };
    auto api = [&](int m) -> cd { return none ? cd{0, 0} : dir ? sgn(m, pa[m * 32]) : pa[-m * 32]; };
    for (int n = P - (int)blockIdx.z; n >= 0; n -= gridDim.z) {
        const double* D = A.T.Dh + __ldg(A.T.Dhoff + n);
        auto out = [&](int m, cd yp, cd ym) {
            V[(size_t)nmi(n, m) * 32] = yp;
            if (m > 0) V[(size_t)nmi(n, -m) * 32] = ym;
        };
        __syncthreads();
        for (int m = w; m <= n; m += nw) {
            cd xp = V[(size_t)nmi(n, m) * 32], xm = V[(size_t)nmi(n, -m) * 32];
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

// Coaxial product at one m of a tile, in place: out_n = sum_k T'_{max(n,k), min(n,k)}
// a_k for the 4 vectors (two directions, +m and -m); Laplace has T_{nk} =
// (-1)^{n+m} lsd_n lsd_k (n+k)!/t^{n+k+1}. Grid (rhs, tile, m): the right-hand
// sides of a tile's T run side by side. The block's vectors sit in shared memory;
// a warp takes every fourth n, four at a time, so an entry loaded feeds 16 FP64
// instructions.
template <bool LAP>
__global__ void __launch_bounds__(kPairThreads) k_pair_coax(PairArgs A) {
    extern __shared__ cd sm[];
    const int P = A.P, m = blockIdx.z, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kPairThreads / 32;
    const size_t tile = blockIdx.y, K = (size_t)(P + 1) * (P + 1);
    const int rhs = blockIdx.x, n1 = P - m + 1;
    cd* V[2];
    for (int dir = 0; dir < 2; ++dir) V[dir] = A.vec + ((size_t)(2 * rhs + dir) * A.ntile + tile) * K * 32 + lane;
    cd* a = sm + lane;                                  // [n1][4]: direction 0 +m, -m, direction 1 +m, -m
    for (int k = w; k < n1; k += nw) {
        double s = LAP ? __ldg(A.T.lsd + nmi(m + k, m)) : 1.0, sm_ = LAP ? __ldg(A.T.lsd + nmi(m + k, -m)) : 1.0;
        for (int dir = 0; dir < 2; ++dir) {
            cd vp = V[dir][(size_t)nmi(m + k, m) * 32], vm = m ? V[dir][(size_t)nmi(m + k, -m) * 32] : cd{0, 0};
            a[(4 * k + 2 * dir) * 32] = LAP ? s * vp : vp;
            a[(4 * k + 2 * dir + 1) * 32] = LAP ? sm_ * vm : vm;
        }
    }
    __syncthreads();
    const cd* T = LAP ? A.fl + tile * (2 * P + 1) * 32 + lane
                      : A.tri + (tile * tri_off(P, P + 1) + tri_off(P, m)) * 32 + lane;
    auto entry = [&](int i, int k) -> cd {              // rows n = m + i and m + k
        if (LAP) return T[(size_t)(2 * m + i + k) * 32];
        int hi = max(i, k), lo = min(i, k);
        return T[(size_t)(hi * (hi + 1) / 2 + lo) * 32];
    };
    for (int i0 = w; i0 < n1; i0 += 4 * nw) {
        auto body = [&](auto cnt) {
            constexpr int R = decltype(cnt)::value;
            cd s[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int v = 0; v < 4; ++v) s[r][v] = cd{0, 0};
            for (int k = 0; k < n1; ++k) {
                cd t[R];
#pragma unroll
                for (int r = 0; r < R; ++r) t[r] = entry(i0 + r * nw, k);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (m == 0 && (v & 1)) continue;
                    cd x = a[(4 * k + v) * 32];
#pragma unroll
                    for (int r = 0; r < R; ++r) s[r][v] = cmac(s[r][v], t[r], x);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int n = m + i0 + r * nw;
                double g = 1.0, gm = 1.0;
                if (LAP) {
                    double e = ((n + m) & 1) ? -1.0 : 1.0;
                    g = e * __ldg(A.T.lsd + nmi(n, m));
                    gm = e * __ldg(A.T.lsd + nmi(n, -m));
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (m == 0 && (v & 1)) continue;
                    V[v >> 1][(size_t)nmi(n, (v & 1) ? -m : m) * 32] = LAP ? ((v & 1) ? gm : g) * s[r][v] : s[r][v];
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

// out[b] (+)= sum over the List-2 entries of b whose slot is in the range
template <bool LAP>
__global__ void k_pair_sum(PairArgs A, int lo, const int* __restrict__ loff, const int* __restrict__ slot,
                           int first, cd* __restrict__ out) {
    const int b = lo + blockIdx.x, rhs = blockIdx.y, K = (A.P + 1) * (A.P + 1);
    const int q0 = loff[b], q1 = loff[b + 1];
    cd* o = out + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int k = blockIdx.z * blockDim.x + threadIdx.x; k < K; k += gridDim.z * blockDim.x) {
        cd s = {0, 0};
#pragma unroll 4
        for (int q = q0; q < q1; ++q) {
            int u = slot[q] - 64 * A.t0;
            if (u < 0 || u >= 64 * A.ntile) continue;
            s += A.vec[(((size_t)(2 * rhs + (u & 1)) * A.ntile + (u >> 6)) * K + k) * 32 + ((u >> 1) & 31)];
        }
        if (LAP) s = __ldg(A.T.lsm + k) * s;
        o[k] = first ? s : o[k] + s;
    }
}

}  // namespace

void pair_slots_build(cfmm_plan_s* P, PairSlots* S, const std::vector<int>& l2off, int l0) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    S->tile0.assign(T.nlevels + 1, 0);
    for (int l = 0; l < T.nlevels; ++l) {
        int64_t pairs = l < l0 ? 0 : (l2off[T.level_off[l + 1]] - l2off[T.level_off[l]]) / 2;
        // flat and other pairs each end with a partial tile
        S->tile0[l + 1] = S->tile0[l] + (pairs ? (int)((pairs + 31) / 32) + 1 : 0);
    }
    S->nslot = (int64_t)32 * S->tile0[T.nlevels];
    const int nent = l2off[T.nboxes];
    if (nent <= 0) return;
    S->box_a.alloc(S->nslot);
    S->box_b.alloc(S->nslot);
    S->kind.alloc(S->nslot);
    S->slot.alloc(nent);
    S->count.alloc(3 * T.nlevels + 1);
    CFMM_CUDA(cudaMemsetAsync(S->box_a.get(), 0xff, sizeof(int) * S->nslot, st));
    CFMM_CUDA(cudaMemsetAsync(S->box_b.get(), 0xff, sizeof(int) * S->nslot, st));
    CFMM_CUDA(cudaMemsetAsync(S->count.get(), 0, sizeof(int) * 2 * T.nlevels, st));
    int* t0 = S->count.get() + 2 * T.nlevels;
    upload(t0, S->tile0.data(), sizeof(int) * (T.nlevels + 1), st);
    k_pair_slots<<<(nent + 127) / 128, 128, 0, st>>>(nent, T.loff[1].get(), T.lent[1].get(), T.nboxes, T.level.get(),
                                                    t0, T.cen_re.get(), T.cen_im.get(), S->count.get(),
                                                    S->box_a.get(), S->box_b.get(), S->kind.get(), S->slot.get());
    CFMM_LAUNCHED();
}

void m2l3d_launch(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l_lo, int l_hi, int Pord, double kappa,
                  const int64_t* eoff, int64_t ncoef, const cd* mp, cd* lc, int nrhs) {
    TreeDev& Tr = P->tree;
    cudaStream_t st = P->stream;
    const bool lap = kappa == 0.0;
    const int lo = Tr.level_off[l_lo], nb = Tr.level_off[l_hi] - lo;
    if (nb <= 0) return;
    const size_t K = (size_t)(Pord + 1) * (Pord + 1), row = 32 * sizeof(cd);
    const int tiles = S->tile0[l_hi] - S->tile0[l_lo];
    const size_t rot_smem = 2 * (size_t)(2 * Pord + 1) * row, cx_smem = 4 * (size_t)(Pord + 1) * row,
                 tri_smem = 3 * (size_t)(2 * Pord + 2) * row;
    // blocks of twice the warps where shared memory leaves one or two an SM
    const int wide = Pord > 40 ? 2 * kPairThreads : kPairThreads;
    if (tiles > 0) {
        for (auto f : {lap ? (const void*)k_pair_fwd<true> : (const void*)k_pair_fwd<false>,
                       lap ? (const void*)k_pair_bwd<true> : (const void*)k_pair_bwd<false>,
                       lap ? (const void*)k_pair_coax<true> : (const void*)k_pair_coax<false>,
                       (const void*)k_pair_tri})
            CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)std::max(rot_smem, std::max(cx_smem, tri_smem))));
    }
    int nsm = 0;
    CFMM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, P->device));
    // tiles of a range: T (Helmholtz) and V within the budget
    const size_t tri_row = lap ? 0 : tri_off(Pord, Pord + 1), per = (tri_row + 2 * (size_t)nrhs * K) * row;
    const int cap = (int)std::max<size_t>(1, std::min<size_t>(kPairBudget / per, 65535));
    PairArgs A{Tr.cen_re.get(), Tr.cen_im.get(), S->box_a.get(), S->box_b.get(), S->kind.get(), T, eoff, ncoef,
               Pord, 0, 0, kappa, nullptr, nullptr, nullptr, nullptr};
    int t0 = S->tile0[l_lo];
    bool first = true;
    do {
        const int nt = std::min(cap, S->tile0[l_hi] - t0);
        A.t0 = t0;
        A.ntile = nt;
        if (nt > 0) {
            S->pw.alloc((size_t)nt * (4 * Pord + 2) * 32);
            S->fl.alloc((size_t)nt * (2 * Pord + 1) * 32);
            S->vec.alloc((size_t)nt * 2 * nrhs * K * 32);
            if (!lap) S->tri.alloc((size_t)nt * tri_row * 32);
            A.pw = S->pw.get();
            A.fl = S->fl.get();
            A.vec = S->vec.get();
            A.tri = S->tri.get();
            // small launches: one thread block per order as well
            int groups = (int)std::min<int64_t>(Pord + 1, std::max<int64_t>(1, (int64_t)8 * nsm / ((int64_t)nt * 2 * nrhs)));
            dim3 gr(2 * nrhs, nt, groups), gc(nrhs, nt, Pord + 1);
            if (lap) {
                k_pair_pre<true><<<(nt + 3) / 4, 128, 0, st>>>(A);
                CFMM_LAUNCHED();
                k_pair_fwd<true><<<gr, wide, rot_smem, st>>>(A, mp);
                CFMM_LAUNCHED();
                k_pair_coax<true><<<gc, kPairThreads, cx_smem, st>>>(A);
                CFMM_LAUNCHED();
                k_pair_bwd<true><<<gr, wide, rot_smem, st>>>(A);
                CFMM_LAUNCHED();
            } else {
                k_pair_pre<false><<<(nt + 3) / 4, 128, 0, st>>>(A);
                CFMM_LAUNCHED();
                k_pair_tri<<<nt, wide, tri_smem, st>>>(A);
                CFMM_LAUNCHED();
                k_pair_fwd<false><<<gr, wide, rot_smem, st>>>(A, mp);
                CFMM_LAUNCHED();
                k_pair_coax<false><<<gc, kPairThreads, cx_smem, st>>>(A);
                CFMM_LAUNCHED();
                k_pair_bwd<false><<<gr, wide, rot_smem, st>>>(A);
                CFMM_LAUNCHED();
            }
        }
        // (also without pairs: the boxes' expansions become zero)
        dim3 gs(nb, nrhs, (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)(K + 127) / 128, 8 * nsm / nb)));
        if (lap) k_pair_sum<true><<<gs, 128, 0, st>>>(A, lo, Tr.loff[1].get(), S->slot.get(), first ? 1 : 0, lc);
        else k_pair_sum<false><<<gs, 128, 0, st>>>(A, lo, Tr.loff[1].get(), S->slot.get(), first ? 1 : 0, lc);
        CFMM_LAUNCHED();
        first = false;
        t0 += nt;
    } while (t0 < S->tile0[l_hi]);
}

}  // namespace cfmm

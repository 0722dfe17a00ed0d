// 2D complex-coordinate FMM: expansions and translations (Sec. 4, Sec. 6.4).
//
// Notation: for a complex displacement d = (d1, d2) put zeta = d1 + i d2,
// eta = d1 - i d2 (r^2 = zeta*eta, e^{+-i phi} = zeta/r, eta/r; Def. 3.1).
//
// 2D Laplace (Sec. 4.2) -- coefficient layout [c0, c_1..c_P, c_{P+1}..c_{2P}]:
//   multipole  u = M0 log r + sum Mp_n eta^-n + sum Mm_n zeta^-n
//              Mp_n = -(1/2n) sum eta_j^n s_j ;  Mm_n likewise in zeta
//   local      u = L0 + sum Lp_n zeta^n + sum Lm_n eta^n
//   M2M/M2L/L2L: the binomial re-expansions of Lemma 4.2.4 in zeta and eta
//   separately; the M0 term of M2L is -(1/2k) zeta0^-k M0 (derived from
//   log(1 - z) = -sum z^k/k).
//   Stored in units of the box's level: Mp_n / s^n, Mm_n / s^n, Lp_n s^n, Lm_n s^n with
//   s = 2^(we - l), W = f 2^we, 1/2 <= f < 1. The scaling is exact, every power is then
//   one of a number of order 1, and deep boxes neither underflow nor overflow (unscaled
//   z^40 at level 26 of a unit domain is below the smallest double).
// 2D Helmholtz (Sec. 4.3) -- layout [c_{-P} .. c_P]: with
//   G_n(d) = J_n(kappa r) e^{in phi}, S_n(d) = H_n^(1)(kappa r) e^{in phi}
//   and Graf's theorem (Thm 3.2.1): for expansions about c re-centred at c',
//   P2M  M_n = sum G_{-n}(c - y) s      M2P  u = sum M_n S_n(x - c)
//   M2M  M'_m = sum G_{n-m}(c' - c) M_n M2L  L_j = sum S_{n-j}(c' - c) M_n
//   L2L  L'_m = sum G_{n-m}(c' - c) L_n P2L  L_j = sum S_{-j}(c' - y) s
//   L2P  u = sum L_n G_n(x - c').
// Double layer: source-side terms differentiated along the caller's normal,
//   n.grad_y = nu d/dzeta + nut d/deta (nu = n1 + i n2, nut = n1 - i n2),
//   d/dzeta G_n = (kappa/2) G_{n-1}, d/deta G_n = -(kappa/2) G_{n+1}.
//
// Helmholtz translation tables depend only on the geometry and are built
// once per plan (one table per List-2 pair and per child box).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <mutex>

#include "kernels.cuh"
#include "pair64.cuh"

namespace cfmm {

// 1/k (an FP64 division costs ten FP64 instructions)
constexpr int kInvTab = 128;
static __constant__ double c_inv[kInvTab];
__device__ __forceinline__ double inv_of(int k) { return k < kInvTab ? c_inv[k] : 1.0 / k; }

void upload_lag_rule_fmm2d() {
    upload_lag_rule_local();
    double inv[kInvTab] = {0.0};
    for (int k = 1; k < kInvTab; ++k) inv[k] = 1.0 / k;
    CFMM_CUDA(cudaMemcpyToSymbol(c_inv, inv, sizeof(inv)));
}

constexpr int kExpThreads = 64;
constexpr int kP2eThreads = 128;   // k_point_to_exp
// its accumulator entries at orders up to P
static size_t p2e_acc(int P) { return std::max<size_t>(2 * (size_t)P + 1, kP2eThreads); }
constexpr int kMaxSmem = 200 * 1024;

// per-plan constants of the 2D expansions
struct Fmm2dState {
    int ker;
    int l0, nlev;
    std::vector<int> Plev;                 // host
    DevBuf<int> dPlev;
    DevBuf<int64_t> exp_off;               // per box (coefficient offset), -1 below l0
    int64_t ncoef = 0;
    int maxP = 0;
    // Laplace, (maxP+1)^2 by [n][k]: C(k-1, n-1) 2^-n, C(n+k-1, k) and C(n, k) 2^-k (a
    // child's unit is half its parent's)
    DevBuf<double> cm2m, cm2l, cl2l;
    int we = 0;                            // exponent of the root width: box units 2^(we - l)
    // Helmholtz translation tables
    DevBuf<cd> t_m2l;                      // per List-2 entry: S_j(c_t - c_s), j = -2P..2P
    std::vector<int64_t> m2l_base;         // per level: table base (complex units)
    std::vector<int> m2l_q0;               // per level: first List-2 entry index
    DevBuf<int64_t> d_m2l_base;
    DevBuf<int> d_m2l_q0;
    DevBuf<cd> t_shift;                    // per child box: G_j(c_parent - c_child), j = -(Pc+Pp)..(Pc+Pp)
    // Helmholtz: per point, the regular row T_m(c - y), m = -P-1..P+1 (P of
    // the point's leaf, index m + P + 1, stride RL), c its leaf's centre; P2M
    // of the leaf and L2P at the point both use it (geometry only)
    DevBuf<cd> lrow;
    int RL = 0;
    DevBuf<int64_t> shift_off;             // per box, -1 when none
    // work lists
    std::vector<int> leaves_l0;            // leaves at level >= l0
    DevBuf<int> d_leaves_l0;
    int maxP_leaf = 0;                     // largest order at a leaf level (P2M)
    int maxP_fine = 0;                     // largest order at or below the coarsest leaf level (M2P, L2P)
    bool rows_side = false;                // the row table is being built on the side stream
    int n_p2l = 0;                         // boxes with a non-empty List 4
    DevBuf<int> d_p2l_boxes;
    // Helmholtz M2L work split: chunks of at most kM2LChunk List-2 entries
    DevBuf<int> chunk_box, chunk_q0, chunk_q1, box_chunk0;   // box_chunk0: [nboxes+1]
    DevBuf<int64_t> chunk_part;            // per chunk: its partial sum's first slot
    int nchunk = 0;
    int64_t npart = 0;                     // partial-sum slots per rhs
    DevBuf<cd> part;
};


// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void zeta_eta(cd d0, cd d1, cd& z, cd& e) {
    z = d0 + mul_i(d1);
    e = d0 - mul_i(d1);
}

// 2^k, |k| <= 1000
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// tables and wavenumber constants of the quick Hankel functions (pair64.cuh)
struct HankelArgs {
    const PairTab* T;
    Wave w;
};

// H_0^(1), H_1^(1) of kappa r, r^2 given: the Taylor cells of pair64.cuh (about 150
// FP64 instructions), or hankel01 outside them (its quadrature beyond |z| = 6 takes
// 6000, which a lone warp issues in 0.2 ms)
__device__ void hankel01_r2(const HankelArgs& H, cd r2, cd* h0, cd* h1) {
    cd y = crsqrt64(r2), ds;
    int cell = hankel_cell(H.w.ik * y, ds);
    if (cell < 0) {
        hankel01(H.w.k * csqrt_p(r2), h0, h1);
        return;
    }
    cd r;
    cd e = wave64(H.T, H.w, r2, y, r);
    e = e * (H.w.isk * crsqrt64(r));
    *h0 = e * hankel_factor(H.T->hk[cell][0], ds);
    *h1 = e * hankel_factor(H.T->hk[cell][1], ds);
}

// Fill row[0 .. 2P+2] with T_m(d), m = -P-1..P+1 (index m + P + 1), where
// T = G (kind 0, regular) or S (kind 1, singular) of the displacement d.
__device__ void cyl_row(int kind, cd zeta, cd eta, const HankelArgs& H, int P, cd* row) {
    const double kappa = H.w.k;
    cd r2 = zeta * eta;
    cd r = csqrt_p(r2);
    int M = P + 1;
    cd* pos = row + M;   // pos[m] = T_m for m >= 0
    if (kind == 0) {
        if (r.x == 0.0 && r.y == 0.0) {
            for (int m = -M; m <= M; ++m) row[m + M] = cd{m == 0 ? 1.0 : 0.0, 0.0};
            return;
        }
        bessel_j_seq(kappa * r, M, pos);
    } else {
        cd h0, h1;
        cd z = kappa * r;
        hankel01_r2(H, r2, &h0, &h1);
        pos[0] = h0;
        if (M >= 1) pos[1] = h1;
        cd zi = cinv(z);
        for (int m = 1; m < M; ++m) pos[m + 1] = rmac(-pos[m - 1], 2.0 * m, zi * pos[m]);
    }
    cd ir = cinv(r);
    cd u = zeta * ir, v = eta * ir;
    cd up = u, vp = v;
    for (int m = 1; m <= M; ++m) {
        cd f = pos[m];
        cd neg = (m & 1) ? -f : f;
        row[M - m] = neg * vp;
        pos[m] = f * up;
        up = up * u;
        vp = vp * v;
    }
}

// Regular rows of every point about its leaf's centre (plan time): block per
// leaf, thread per point.
__global__ void k_leaf_rows(const int* __restrict__ leaves, const int* __restrict__ blevel,
                            const int* __restrict__ bst, const int* __restrict__ ben, const int* __restrict__ Plev,
                            const double* __restrict__ xr, const double* __restrict__ xi, int64_t n,
                            const double* __restrict__ cre, const double* __restrict__ cim, HankelArgs H, int RL,
                            cd* __restrict__ lrow) {
    int b = leaves[blockIdx.x];
    int P = Plev[blevel[b]];
    cd cen0 = {cre[2 * b], cim[2 * b]}, cen1 = {cre[2 * b + 1], cim[2 * b + 1]};
    for (int j = bst[b] + threadIdx.x; j < ben[b]; j += blockDim.x) {
        cd y0 = {xr[j], xi[j]}, y1 = {xr[n + j], xi[n + j]};
        cd z, e;
        zeta_eta(cen0 - y0, cen1 - y1, z, e);   // D = c - y
        cyl_row(0, z, e, H, P, lrow + (int64_t)j * RL);
    }
}

// ---------------------------------------------------------------------------
// P2M (step 1) and P2L (step 6): point terms reduced per coefficient
// ---------------------------------------------------------------------------
struct ExpArgs {
    const double* xr;
    const double* xi;
    const double* nr;
    const double* ni;
    int64_t n;
    const cd* sigma;
    const cd* tau;
    int64_t dstride;
    bool slp, dlp;
    double kappa;
    const int* blevel;
    SubRange src, trg;
    const double* cre;
    const double* cim;
    const int* Plev;
    const int64_t* eoff;
    int64_t ncoef;
    HankelArgs H;
    int we;
};

// term row (Laplace) for a source at d = y - c, regular (P2M) or singular (P2L):
//   P2M  row_k = -s eta^k/(2k) - nut t eta^{k-1}/2          (k <= P; P + k: zeta, nu)
//   P2L  row_k = -s zeta^-k/(2k) + nu t zeta^{-k-1}/2       (P + k: eta, nut)
// as two running products a series, 10 FP64 instructions a term; iu = 1 / the box's unit
__device__ void lap_terms(const PairTab* T, double iu, bool sing, cd zeta, cd eta, cd s, cd t, cd nu, cd nut, int P,
                          bool slp, bool dlp, cd* row) {
    nu = iu * nu;
    nut = iu * nut;
    cd x = iu * eta, y = iu * zeta, nx = nut, ny = nu;   // series 1..P in x, P+1..2P in y
    double h = -0.5;
    cd v0 = slp ? s : cd{0, 0};
    if (sing) {
        x = crcp64(iu * zeta);
        y = crcp64(iu * eta);
        nx = nu;
        ny = nut;
        h = 0.5;
        v0 = slp ? (0.5 * clog64(T, zeta * eta)) * s : cd{0, 0};
        if (dlp) v0 = cmac(v0, 0.5 * (nu * x + nut * y), t);
    }
    row[0] = v0;
    cd ax = -0.5 * (s * x), ay = -0.5 * (s * y), bx = h * (nx * t), by = h * (ny * t);
    if (sing) {
        bx = bx * x * x;
        by = by * y * y;
    }
    for (int k = 1; k <= P; ++k) {
        double ik = inv_of(k);
        cd a = dlp ? bx : cd{0, 0}, b = dlp ? by : cd{0, 0};
        if (slp) {
            a = rmac(a, ik, ax);
            b = rmac(b, ik, ay);
            ax = ax * x;
            ay = ay * y;
        }
        row[k] = a;
        row[P + k] = b;
        if (dlp) {
            bx = bx * x;
            by = by * y;
        }
    }
}

// One CTA per target box; sources = the box's own points (P2M, list == null)
// or the points of the List-4 leaves (P2L), taken `chunk` at a time over the whole
// list (leaves of a point or two share a chunk: a source's row is a chain of 700
// FP64 instructions). Thread (c, s) owns coefficient c for every S-th source: with
// one thread per coefficient 41 of 64 lanes were in use at order 20. Result added to
// (P2L) or stored in (P2M) out[rhs][eoff[b] + c].
template <int KER>
__global__ void k_point_to_exp(ExpArgs A, const int* __restrict__ boxes, const int* __restrict__ loff,
                               const int* __restrict__ lent, int sing, cd* __restrict__ out, int chunk,
                               const cd* __restrict__ lrow, int RL) {
    extern __shared__ cd sm[];
    int b = boxes[blockIdx.x];
    int rhs = blockIdx.y;
    int P = A.Plev[A.blevel[b]];
    int nc = 2 * P + 1;
    int R = KER == CFMM_LAPLACE ? nc : nc + 2;
    const int S = max(1, min((int)blockDim.x / nc, 4));
    cd* acc = sm;                              // [S][nc]
    cd* rows = sm + S * nc;
    cd* wts = rows + (size_t)chunk * R;        // Helmholtz: per source (s, -k/2 nu t, k/2 nu~ t)
    for (int c = threadIdx.x; c < S * nc; c += blockDim.x) acc[c] = cd{0, 0};
    cd cen0 = {A.cre[2 * b], A.cim[2 * b]}, cen1 = {A.cre[2 * b + 1], A.cim[2 * b + 1]};
    // first source of the next chunk: point j0 of list entry qn
    int qn = loff ? loff[b] : 0, j0 = 0;
    const int qb = loff ? loff[b + 1] : 1;
    while (qn < qb) {
        // the thread's source, and (the same for all) where the chunk ends
        int64_t j = -1;
        int cn = 0, q = qn, jn = j0;
        while (q < qb && cn < chunk) {
            const int src = loff ? lent[q] : b;
            const int s0 = A.src.st[src] + jn, m = min(A.src.en[src] - s0, chunk - cn);
            if ((int)threadIdx.x >= cn && (int)threadIdx.x < cn + m) j = A.src.at(s0 + (threadIdx.x - cn));
            cn += m;
            if (s0 + m == A.src.en[src]) {
                ++q;
                jn = 0;
            } else {
                jn += m;
            }
        }
        __syncthreads();
        if (j >= 0) {
            cd y0 = {A.xr[j], A.xi[j]}, y1 = {A.xr[A.n + j], A.xi[A.n + j]};
            cd s = A.slp ? A.sigma[rhs * A.dstride + j] : cd{0, 0};
            cd t = A.dlp ? A.tau[rhs * A.dstride + j] : cd{0, 0};
            cd nu = {0, 0}, nut = {0, 0};
            if (A.dlp) {
                cd n0 = {A.nr[j], A.ni[j]}, n1 = {A.nr[A.n + j], A.ni[A.n + j]};
                nu = n0 + mul_i(n1);
                nut = n0 - mul_i(n1);
            }
            cd* row = rows + (size_t)threadIdx.x * R;
            cd z, e;
            if (KER == CFMM_LAPLACE) {
                zeta_eta(y0 - cen0, y1 - cen1, z, e);   // d = y - c
                lap_terms(A.H.T, pow2(A.blevel[b] - A.we), sing != 0, z, e, s, t, nu, nut, P, A.slp, A.dlp, row);
            } else {
                if (!lrow || sing) {
                    zeta_eta(cen0 - y0, cen1 - y1, z, e);   // D = c - y
                    cyl_row(sing ? 1 : 0, z, e, A.H, P, row);
                }
                double hk = 0.5 * A.kappa;
                cd* w = wts + 3 * threadIdx.x;
                w[0] = s;
                w[1] = (-hk) * (nu * t);
                w[2] = hk * (nut * t);
            }
        }
        // the plan's rows of the points about their own leaf (this box), a warp a row
        if (KER == CFMM_HELMHOLTZ && lrow && !sing)
            for (int tt = threadIdx.x >> 5; tt < cn; tt += blockDim.x >> 5) {
                const cd* src = lrow + A.src.at(A.src.st[b] + j0 + tt) * RL;
                for (int i = threadIdx.x & 31; i < R; i += 32) rows[(size_t)tt * R + i] = src[i];
            }
        __syncthreads();
        for (int i = threadIdx.x; i < S * nc; i += blockDim.x) {
            const int sl = i / nc, c = i - sl * nc;
            cd a = acc[i];
            if (KER == CFMM_LAPLACE) {
                for (int tt = sl; tt < cn; tt += S) a += rows[(size_t)tt * R + c];
            } else {
                // coefficient n = c - P: s T_{-n} - (k/2)(nu T_{-n-1} - nu~ T_{-n+1}) t,
                // T_k at row index k + P + 1
                int i0 = 2 * P + 1 - c;
                if (A.dlp) {
                    for (int tt = sl; tt < cn; tt += S) {
                        const cd* r = rows + (size_t)tt * R + i0;
                        const cd* w = wts + 3 * tt;
                        a = cmac(cmac(cmac(a, w[0], r[0]), w[1], r[-1]), w[2], r[1]);
                    }
                } else {
                    for (int tt = sl; tt < cn; tt += S) a = cmac(a, wts[3 * tt], rows[(size_t)tt * R + i0]);
                }
            }
            acc[i] = a;
        }
        qn = q;
        j0 = jn;
    }
    __syncthreads();
    cd* o = out + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        cd v = acc[c];
        for (int sl = 1; sl < S; ++sl) v += acc[sl * nc + c];
        if (sing) o[c] += v;
        else o[c] = v;
    }
}

// ---------------------------------------------------------------------------
// M2M (step 2) and L2L (step 7): one CTA per target box at one level
// ---------------------------------------------------------------------------
struct TransArgs {
    const int* blevel;
    const int* parent;
    const int* cbeg;
    const int* cend;
    const double* cre;
    const double* cim;
    const int* Plev;
    const int64_t* eoff;
    int64_t ncoef;
    int we;
    const cd* tshift;
    const int64_t* shoff;
};

// The Laplace translations with the binomials as real matrices between diagonal
// scalings (z = zeta or eta of the shift, per series):
//   M2M  M'_k = z^k (sum_{n<=k} C(k-1,n-1) z^-n M_n - M_0/(2k))
//   M2L  L_k  = z^-k (sum_n C(n+k-1,k) (-z)^-n M_n - M_0/(2k))
//   L2L  L'_k = z^-k sum_{n>=k} C(n,k) z^n L_n
// with z in the parent's unit (M2M, L2L) or the level's; the factors 2^-n and 2^-k
// between a child's and its parent's unit are in the tables. 2 FP64 instructions a term instead of 8. What bounds a level is the chain of FP64
// instructions one warp issues (one in 64 cycles), so threads are (shift, k): a
// group of warps takes a shift (its last warp the constant coefficient), and the
// groups of a block work side by side.
__device__ __forceinline__ cd cpow_k(cd z, int k) {
    cd r = {1, 0};
    for (; k; k >>= 1) {
        if (k & 1) r = r * z;
        if (k > 1) z = z * z;
    }
    return r;
}
__host__ __device__ inline int lap_group(int P) { return (2 * P + 31) / 32 * 32 + 32; }   // threads of a shift

// M2M: parent b gathers its children
__global__ void k_m2m_lap(TransArgs T, int lo, const cd* __restrict__ mp_in, cd* __restrict__ mp_out,
                          const int* __restrict__ leaf, int P, const double* __restrict__ cm2m) {
    extern __shared__ cd sm[];
    const int b = lo + blockIdx.x, rhs = blockIdx.y, nc = 2 * P + 1;
    if (leaf[b]) return;
    const int gs = lap_group(P), ng = blockDim.x / gs, g = threadIdx.x / gs, i = threadIdx.x - g * gs;
    cd *x = sm + g * nc, *red = sm + ng * nc + g * nc;
    const int c = i < 2 * P ? i + 1 : 0, k = c > P ? c - P : c;
    const double iu = pow2(T.blevel[b] - T.we);
    cd acc = {0, 0};
    for (int c0 = T.cbeg[b]; c0 < T.cend[b]; c0 += ng) {
        const int ch = c0 + g;
        const bool on = ch < T.cend[b];
        cd pk = {1, 0}, m0 = {0, 0};
        bool nz = true;
        __syncthreads();
        if (on) {
            const cd* m = mp_in + (int64_t)rhs * T.ncoef + T.eoff[ch];
            m0 = m[0];
            if (c) {
                // a = c_child - c_parent
                cd z, e;
                zeta_eta(cd{T.cre[2 * ch] - T.cre[2 * b], T.cim[2 * ch] - T.cim[2 * b]},
                         cd{T.cre[2 * ch + 1] - T.cre[2 * b + 1], T.cim[2 * ch + 1] - T.cim[2 * b + 1]}, z, e);
                z = iu * (c <= P ? e : z);
                nz = z.x != 0.0 || z.y != 0.0;
                if (nz) pk = cpow_k(z, k);
                x[c] = nz ? m[c] * crcp64(pk) : m[c];
            }
        }
        __syncthreads();
        if (on && c) {
            const cd* xs = x + (c > P ? P : 0);
            if (nz) {
                cd y = (-0.5 * inv_of(k)) * m0;
                for (int n = 1; n <= P; ++n) y = rmac(y, __ldg(cm2m + n * (P + 1) + k), xs[n]);   // 0 for n > k
                acc = cmac(acc, pk, y);
            } else {
                acc += pow2(-k) * xs[k];
            }
        } else if (on && i == 2 * P) {
            acc += m0;
        }
    }
    __syncthreads();
    if (c || i == 2 * P) red[c] = acc;
    __syncthreads();
    cd* o = mp_out + (int64_t)rhs * T.ncoef + T.eoff[b];
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
        cd v = sm[ng * nc + q];
        for (int j = 1; j < ng; ++j) v += sm[(ng + j) * nc + q];
        o[q] = v;
    }
}

// L2L: child b (at level lo..) receives its parent's local expansion
__global__ void k_l2l_lap(TransArgs T, int lo, cd* __restrict__ loc, int P, const double* __restrict__ cl2l) {
    extern __shared__ cd sm[];
    const int b = lo + blockIdx.x, rhs = blockIdx.y, p = T.parent[b], i = threadIdx.x;
    const int c = i < 2 * P ? i + 1 : 0, k = c > P ? c - P : c;
    const cd* lp = loc + (int64_t)rhs * T.ncoef + T.eoff[p];
    cd* o = loc + (int64_t)rhs * T.ncoef + T.eoff[b];
    cd pk = {1, 0};
    bool nz = true;
    if (c) {
        // powers of -zeta0, -eta0 with a = c_parent - c_child: of the child's offset
        cd z, e;
        zeta_eta(cd{T.cre[2 * b] - T.cre[2 * p], T.cim[2 * b] - T.cim[2 * p]},
                 cd{T.cre[2 * b + 1] - T.cre[2 * p + 1], T.cim[2 * b + 1] - T.cim[2 * p + 1]}, z, e);
        z = pow2(T.blevel[p] - T.we) * (c > P ? e : z);
        nz = z.x != 0.0 || z.y != 0.0;
        if (nz) pk = cpow_k(z, k);
        // (a zero shift leaves the coefficients; they do not reach L_0)
        sm[c] = pk * lp[c];
        sm[2 * P + c] = nz ? sm[c] : cd{0, 0};
    }
    __syncthreads();
    if (c) {
        const cd* xs = sm + (c > P ? P : 0);
        if (nz) {
            cd y = {0, 0};
            for (int n = 1; n <= P; ++n) y = rmac(y, __ldg(cl2l + n * (P + 1) + k), xs[n]);   // 0 for n < k
            o[c] = cmac(o[c], crcp64(pk), y);
        } else {
            o[c] += pow2(-k) * xs[k];
        }
    } else if (i >= (int)blockDim.x - 32) {
        // the constant: the last warp sums L_0 and every scaled coefficient
        const int lane = i & 31;
        cd v = {0, 0};
        for (int q = 1 + lane; q <= 2 * P; q += 32) v += sm[2 * P + q];
        for (int d = 16; d > 0; d >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, d);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, d);
        }
        if (lane == 0) o[0] += lp[0] + v;
    }
}

// The Helmholtz M2M and L2L: Toeplitz products with the plan's tables; item (c, s)
// takes every S-th term of coefficient c, so that a block's warps share the chain.
__global__ void k_m2m_helm(TransArgs T, int lo, const cd* __restrict__ mp_in, cd* __restrict__ mp_out,
                           const int* __restrict__ leaf, int Pc, int Pp, int S) {
    extern __shared__ cd sm[];
    const int b = lo + blockIdx.x, rhs = blockIdx.y, ncp = 2 * Pp + 1, ncc = 2 * Pc + 1, off = Pc + Pp;
    if (leaf[b]) return;
    cd *src = sm, *pw = src + ncc, *red = pw + 2 * off + 1;
    for (int i = threadIdx.x; i < S * ncp; i += blockDim.x) red[i] = cd{0, 0};
    for (int ch = T.cbeg[b]; ch < T.cend[b]; ++ch) {
        __syncthreads();
        const cd* m = mp_in + (int64_t)rhs * T.ncoef + T.eoff[ch];
        const cd* tb = T.tshift + T.shoff[ch];
        for (int q = threadIdx.x; q < ncc; q += blockDim.x) src[q] = m[q];
        for (int q = threadIdx.x; q < 2 * off + 1; q += blockDim.x) pw[q] = tb[q];
        __syncthreads();
        for (int i = threadIdx.x; i < S * ncp; i += blockDim.x) {
            const int s = i / ncp, c = i - s * ncp;
            cd a = red[i];
            for (int q = s; q < ncc; q += S) a = cmac(a, pw[q - Pc - (c - Pp) + off], src[q]);
            red[i] = a;
        }
    }
    __syncthreads();
    cd* o = mp_out + (int64_t)rhs * T.ncoef + T.eoff[b];
    for (int q = threadIdx.x; q < ncp; q += blockDim.x) {
        cd v = red[q];
        for (int j = 1; j < S; ++j) v += red[j * ncp + q];
        o[q] = v;
    }
}

__global__ void k_l2l_helm(TransArgs T, int lo, cd* __restrict__ loc, int Pp, int Pc, int S) {
    extern __shared__ cd sm[];
    const int b = lo + blockIdx.x, rhs = blockIdx.y, p = T.parent[b], ncp = 2 * Pp + 1, ncc = 2 * Pc + 1, off = Pc + Pp;
    cd *src = sm, *pw = src + ncp, *red = pw + 2 * off + 1;
    const cd* lp = loc + (int64_t)rhs * T.ncoef + T.eoff[p];
    // table holds G_j(c_parent - c_child); L2L needs G_j(c_child - c_parent) = (-1)^j G_j(...)
    const cd* tb = T.tshift + T.shoff[b];
    for (int q = threadIdx.x; q < ncp; q += blockDim.x) src[q] = lp[q];
    for (int q = threadIdx.x; q < 2 * off + 1; q += blockDim.x) pw[q] = ((q - off) & 1) ? -tb[q] : tb[q];
    __syncthreads();
    for (int i = threadIdx.x; i < S * ncc; i += blockDim.x) {
        const int s = i / ncc, c = i - s * ncc;
        cd a = {0, 0};
        for (int q = s; q < ncp; q += S) a = cmac(a, pw[q - Pp - (c - Pc) + off], src[q]);
        red[i] = a;
    }
    __syncthreads();
    cd* o = loc + (int64_t)rhs * T.ncoef + T.eoff[b];
    for (int q = threadIdx.x; q < ncc; q += blockDim.x) {
        cd v = red[q];
        for (int j = 1; j < S; ++j) v += red[j * ncc + q];
        o[q] += v;
    }
}

// ---------------------------------------------------------------------------
// M2L (step 4) over List 2, all levels >= l0 in one launch
// ---------------------------------------------------------------------------
struct M2LArgs {
    const int* blevel;
    const double* cre;
    const double* cim;
    const int* Plev;
    const int64_t* eoff;
    int64_t ncoef;
    const int* loff;
    const int* lent;
    const cd* tab;
    const int64_t* tbase;
    const int* tq0;
    int we;
};

// Laplace M2L (see the comment above k_m2m_lap): a block per box, groups of warps
// side by side on its List-2 entries
__global__ void k_m2l_lap(M2LArgs A, int first_box, const cd* __restrict__ mp, cd* __restrict__ loc, int P,
                          const double* __restrict__ cm2l, const PairTab* __restrict__ T, int add) {
    extern __shared__ cd sm[];
    const int b = first_box + blockIdx.x, rhs = blockIdx.y, nc = 2 * P + 1;
    const int gs = lap_group(P), ng = blockDim.x / gs, g = threadIdx.x / gs, i = threadIdx.x - g * gs;
    cd *x = sm + g * nc, *red = sm + ng * nc + g * nc;
    const int c = i < 2 * P ? i + 1 : 0, k = c > P ? c - P : c, q1 = A.loff[b + 1];
    const bool last = i >= gs - 32;                     // the group's last warp: the constant
    const double iu = pow2(A.blevel[b] - A.we);
    cd acc = {0, 0};
    for (int q0 = A.loff[b]; q0 < q1; q0 += ng) {
        const bool on = q0 + g < q1;
        cd pk = {0, 0}, m0 = {0, 0}, z = {1, 0}, e = {1, 0};
        __syncthreads();
        if (on) {
            const int s = A.lent[q0 + g];
            const cd* m = mp + (int64_t)rhs * A.ncoef + A.eoff[s];
            m0 = m[0];
            // a = c_s - c_t
            zeta_eta(cd{A.cre[2 * s] - A.cre[2 * b], A.cim[2 * s] - A.cim[2 * b]},
                     cd{A.cre[2 * s + 1] - A.cre[2 * b + 1], A.cim[2 * s + 1] - A.cim[2 * b + 1]}, z, e);
            if (c) {
                // L_1.. in zeta from the source's zeta series (entries P+1..), L_P+1.. in eta from 1..P
                pk = cpow_k(crcp64(iu * (c <= P ? z : e)), k);
                cd v = pk * m[c <= P ? P + c : c - P];
                x[c] = (k & 1) ? -v : v;
            }
        }
        __syncthreads();
        if (!on) continue;
        if (c) {
            const cd* xs = x + (c > P ? P : 0);
            cd y = (-0.5 * inv_of(k)) * m0;
            for (int n = 1; n <= P; ++n) y = rmac(y, __ldg(cm2l + n * (P + 1) + k), xs[n]);
            acc = cmac(acc, pk, y);
        } else if (last) {
            for (int n = 1 + (i & 31); n <= 2 * P; n += 32) acc += x[n];
            if (i == gs - 1) acc = cmac(acc, 0.5 * clog64(T, z * e), m0);
        }
    }
    __syncthreads();
    if (last) {
        for (int d = 16; d > 0; d >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, d);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, d);
        }
    }
    if (c || i == gs - 1) red[c] = acc;
    __syncthreads();
    cd* o = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int q = threadIdx.x; q < nc; q += blockDim.x) {
        cd v = sm[ng * nc + q];
        for (int j = 1; j < ng; ++j) v += sm[(ng + j) * nc + q];
        o[q] = add ? o[q] + v : v;
    }
}

// Helmholtz M2L of orders beyond the chunked kernel's block: one block per box
__global__ void k_m2l_helm(M2LArgs A, int first_box, const cd* __restrict__ mp, cd* __restrict__ loc, int add) {
    extern __shared__ cd sm[];
    int b = first_box + blockIdx.x;
    int rhs = blockIdx.y;
    int l = A.blevel[b];
    int P = A.Plev[l];
    int nc = 2 * P + 1;
    cd* acc = sm;
    cd* src = sm + nc;
    cd* tb = src + nc;     // 4P+1
    for (int c = threadIdx.x; c < nc; c += blockDim.x) acc[c] = cd{0, 0};
    for (int q = A.loff[b]; q < A.loff[b + 1]; ++q) {
        int s = A.lent[q];
        __syncthreads();
        const cd* m = mp + (int64_t)rhs * A.ncoef + A.eoff[s];
        for (int c = threadIdx.x; c < nc; c += blockDim.x) src[c] = m[c];
        const cd* t = A.tab + A.tbase[l] + (int64_t)(q - A.tq0[l]) * (4 * P + 1);
        for (int c = threadIdx.x; c < 4 * P + 1; c += blockDim.x) tb[c] = t[c];
        __syncthreads();
        for (int c = threadIdx.x; c < nc; c += blockDim.x) {
            cd a = acc[c];
            int j = c - P;
            for (int nn = -P; nn <= P; ++nn) a = cmac(a, tb[nn - j + 2 * P], src[nn + P]);
            acc[c] = a;
        }
    }
    __syncthreads();
    cd* o = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) o[c] = add ? o[c] + acc[c] : acc[c];
}

// Helmholtz M2L split into chunks of List-2 entries: one CTA per chunk, thread
// (c, s) owns output c for source lane s; the S lanes' sums are combined in a
// fixed order into one partial sum per chunk, and k_m2l_reduce adds the chunks
// of a box in chunk order (bitwise reproducible, and the long all-pairs lists
// of the top level are spread over many CTAs).
constexpr int kM2LChunk = 32;

// All levels share one launch (the orders and so the split over S come from the
// box's level): the coarse levels' few, long blocks run beside the fine levels'.
__host__ __device__ inline int m2l_lanes(int nc, int threads) { return nc > threads ? 1 : threads / nc < 8 ? threads / nc : 8; }

__global__ void k_m2l_chunk(M2LArgs A, const int* __restrict__ chunk_box, const int* __restrict__ cq0,
                            const int* __restrict__ cq1, const int64_t* __restrict__ cpart, cd* __restrict__ part,
                            int64_t part_stride, const cd* __restrict__ mp) {
    extern __shared__ cd sm[];
    int ch = blockIdx.x;
    int rhs = blockIdx.y;
    int b = chunk_box[ch];
    int l = A.blevel[b];
    const int P = A.Plev[l];
    int nc = 2 * P + 1, nt = 4 * P + 1;
    const int S = m2l_lanes(nc, blockDim.x);
    int t = threadIdx.x;
    int c = t % nc, sl = t / nc;
    bool act = sl < S;
    cd* msrc = sm;                         // [S][nc]
    cd* mtab = sm + (size_t)S * nc;        // [S][nt]
    cd acc = {0, 0};
    int q0 = cq0[ch], q1 = cq1[ch];
    for (int qb = q0; qb < q1; qb += S) {
        __syncthreads();
        int nsrc = min(S, q1 - qb);
        for (int i = t; i < nsrc * nc; i += blockDim.x) {
            int ss = i / nc, cc = i - ss * nc;
            int src = A.lent[qb + ss];
            msrc[(size_t)ss * nc + cc] = mp[(int64_t)rhs * A.ncoef + A.eoff[src] + cc];
        }
        for (int i = t; i < nsrc * nt; i += blockDim.x) {
            int ss = i / nt, cc = i - ss * nt;
            int q = qb + ss;
            mtab[(size_t)ss * nt + cc] = A.tab[A.tbase[l] + (int64_t)(q - A.tq0[l]) * nt + cc];
        }
        __syncthreads();
        if (act && sl < nsrc) {
            const cd* ms = msrc + (size_t)sl * nc;
            const cd* tb = mtab + (size_t)sl * nt + (nc - 1 - c);   // T[n - c + 2P] = tb[n]
            cd a = acc;
            for (int nn = 0; nn < nc; ++nn) a = cmac(a, tb[nn], ms[nn]);
            acc = a;
        }
    }
    __syncthreads();
    cd* red = sm;                          // [S][nc]
    if (act) red[(size_t)sl * nc + c] = acc;
    __syncthreads();
    if (t < nc) {
        cd v = red[t];
        for (int ss = 1; ss < S; ++ss) v += red[(size_t)ss * nc + t];
        part[(int64_t)rhs * part_stride + cpart[ch] + t] = v;
    }
}

// chunk sums of a box in order, added to what P2L left there (add) or stored
__global__ void k_m2l_reduce(int first_box, const int* __restrict__ blevel, const int* __restrict__ Plev,
                             const int* __restrict__ box_chunk0, const int64_t* __restrict__ cpart,
                             const cd* __restrict__ part, int64_t part_stride, const int64_t* __restrict__ eoff,
                             int64_t ncoef, int add, cd* __restrict__ loc) {
    int b = first_box + blockIdx.x;
    int rhs = blockIdx.y;
    int c0 = box_chunk0[b], c1 = box_chunk0[b + 1], nc = 2 * Plev[blevel[b]] + 1;
    cd* out = loc + (int64_t)rhs * ncoef + eoff[b];
    const cd* pp = part + (int64_t)rhs * part_stride;
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        cd v = {0, 0};
        for (int k = c0; k < c1; ++k) v += pp[cpart[k] + c];
        out[c] = add ? out[c] + v : v;
    }
}

// ---------------------------------------------------------------------------
// M2P (step 5, List 3) and L2P (step 8): one CTA per leaf, one thread per target
// ---------------------------------------------------------------------------
template <int KER>
__global__ void k_eval(ExpArgs A, const int* __restrict__ leaves, const int* __restrict__ l3off,
                       const int* __restrict__ l3, const cd* __restrict__ mp, const cd* __restrict__ loc,
                       cd* __restrict__ u, int maxP, const cd* __restrict__ lrow, int RL, int do_l2p) {
    extern __shared__ cd sm[];
    int b = leaves[blockIdx.x];
    int rhs = blockIdx.y;
    int P = A.Plev[A.blevel[b]];
    int nc = 2 * P + 1;
    cd* coef = sm;                                  // 2*maxP+1
    cd* rows = sm + 2 * maxP + 1;                   // per thread: maxP+2 (Helmholtz L2P), 1 (M2P)
    int s0 = A.trg.st[b], s1 = A.trg.en[b];
    for (int t0 = s0; t0 < s1; t0 += blockDim.x) {
        bool valid = t0 + (int)threadIdx.x < s1;
        const int64_t i = valid ? A.trg.at(t0 + threadIdx.x) : 0;
        cd x0 = {0, 0}, x1 = {0, 0};
        if (valid) {
            x0 = cd{A.xr[i], A.xi[i]};
            x1 = cd{A.xr[A.n + i], A.xi[A.n + i]};
        }
        cd acc = {0, 0};
        // M2P over List 3: items (entry, target), a thread each, so that the entries
        // of a leaf of few points (a chain of 700 FP64 instructions each) run side by
        // side; a target adds its items in list order
        const int nt = min((int)blockDim.x, s1 - t0), q0 = l3off[b], items = (l3off[b + 1] - q0) * nt;
        for (int base = 0; base < items; base += blockDim.x) {
            const int item = base + threadIdx.x;
            cd v = {0, 0};
            if (item < items) {
                const int s = l3[q0 + item / nt], Ps = A.Plev[A.blevel[s]];
                const int64_t it = A.trg.at(t0 + item % nt);
                const cd* m = mp + (int64_t)rhs * A.ncoef + A.eoff[s];
                cd z, e;
                zeta_eta(cd{A.xr[it], A.xi[it]} - cd{A.cre[2 * s], A.cim[2 * s]},
                         cd{A.xr[A.n + it], A.xi[A.n + it]} - cd{A.cre[2 * s + 1], A.cim[2 * s + 1]}, z, e);
                if (KER == CFMM_LAPLACE) {
                    // Horner in 1/eta and 1/zeta
                    const double iu = pow2(A.blevel[s] - A.we);
                    cd iz = crcp64(iu * z), ie = crcp64(iu * e), vz = m[2 * Ps], ve = m[Ps];
                    for (int nn = Ps - 1; nn >= 1; --nn) {
                        ve = cmac(m[nn], ve, ie);
                        vz = cmac(m[Ps + nn], vz, iz);
                    }
                    v = cmac(cmac((0.5 * clog64(A.H.T, z * e)) * m[0], ve, ie), vz, iz);
                } else {
                    // S_n(x - c) by forward recurrence in registers
                    cd r = csqrt_p(z * e);
                    cd zz = A.kappa * r;
                    cd h0, h1;
                    hankel01_r2(A.H, z * e, &h0, &h1);
                    cd ir = cinv(r), uu = z * ir, vv = e * ir, zi = cinv(zz);
                    v = m[Ps] * h0;
                    cd hm = h0, hn = h1, up = uu, vp = vv;
                    for (int nn = 1; nn <= Ps; ++nn) {
                        cd neg = (nn & 1) ? -hn : hn;
                        v = cmac(cmac(v, m[Ps + nn], hn * up), m[Ps - nn], neg * vp);
                        cd hp = rmac(-hm, 2.0 * nn, zi * hn);
                        hm = hn;
                        hn = hp;
                        up = up * uu;
                        vp = vp * vv;
                    }
                }
            }
            __syncthreads();
            rows[threadIdx.x] = v;
            __syncthreads();
            // the pass's items of this target: base + k with (base + k) % nt == its index
            if ((int)threadIdx.x < nt)
                for (int k = ((int)threadIdx.x - base % nt + nt) % nt; k < (int)blockDim.x && base + k < items; k += nt)
                    acc += rows[k];
            __syncthreads();
        }
        if (!do_l2p) {
            // M2P only (the L2P runs in complex64): leaves without List 3 add nothing
            if (valid && l3off[b + 1] > l3off[b]) u[(int64_t)rhs * A.n + i] += acc;
            continue;
        }
        // L2P
        __syncthreads();
        const cd* lc = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
        for (int c = threadIdx.x; c < nc; c += blockDim.x) coef[c] = lc[c];
        __syncthreads();
        if (valid) {
            cd z, e;
            zeta_eta(x0 - cd{A.cre[2 * b], A.cim[2 * b]}, x1 - cd{A.cre[2 * b + 1], A.cim[2 * b + 1]}, z, e);
            if (KER == CFMM_LAPLACE) {
                const double iu = pow2(A.blevel[b] - A.we);
                z = iu * z;
                e = iu * e;
                cd vz = coef[P], ve = coef[2 * P];
                for (int nn = P - 1; nn >= 1; --nn) {
                    vz = cmac(coef[nn], vz, z);
                    ve = cmac(coef[P + nn], ve, e);
                }
                acc += cmac(cmac(coef[0], vz, z), ve, e);
            } else if (lrow) {
                // T_k(x - c) = (-1)^k T_k(c - x), the plan's row of this point
                const cd* t = lrow + (int64_t)i * RL + (P + 1);
                acc += coef[P] * t[0];
                for (int nn = 1; nn <= P; ++nn) {
                    cd tp = t[nn], tm = t[-nn];
                    if (nn & 1) {
                        tp = -tp;
                        tm = -tm;
                    }
                    acc = cmac(cmac(acc, coef[P + nn], tp), coef[P - nn], tm);
                }
            } else {
                cd* row = rows + (size_t)threadIdx.x * (maxP + 2);
                cd r = csqrt_p(z * e);
                if (r.x == 0.0 && r.y == 0.0) {
                    acc += coef[P];
                } else {
                    bessel_j_seq(A.kappa * r, P, row);
                    cd ir = cinv(r), uu = z * ir, vv = e * ir, up = uu, vp = vv;
                    acc += coef[P] * row[0];
                    for (int nn = 1; nn <= P; ++nn) {
                        cd jn = row[nn];
                        cd neg = (nn & 1) ? -jn : jn;
                        acc += coef[P + nn] * (jn * up) + coef[P - nn] * (neg * vp);
                        up = up * uu;
                        vp = vp * vv;
                    }
                }
            }
            u[(int64_t)rhs * A.n + i] += acc;
        }
    }
}

// ---------------------------------------------------------------------------
// Target gradients of M2P (List 3) and L2P (FP64), added to g [rhs][2][n]:
// d/dx1 = d/dzeta + d/deta, d/dx2 = i (d/dzeta - d/deta), with
//   Laplace  u = M0 log(zeta eta)/2 + sum Mp_n eta^-n + Mm_n zeta^-n:
//            d/dzeta = M0/(2 zeta) - sum n Mm_n zeta^-n-1 (likewise eta);
//            u = L0 + sum Lp_n zeta^n + Lm_n eta^n: d/dzeta = sum n Lp_n zeta^n-1;
//   Helmholtz d/dzeta T_n = (kappa/2) T_{n-1}, d/deta T_n = -(kappa/2) T_{n+1}
//            for T = S (M2P) and G (L2P).
// ---------------------------------------------------------------------------
template <int KER>
__global__ void k_eval_grad(ExpArgs A, const int* __restrict__ leaves, const int* __restrict__ l3off,
                            const int* __restrict__ l3, const cd* __restrict__ mp, const cd* __restrict__ loc,
                            cd* __restrict__ g, int maxP) {
    extern __shared__ cd sm[];
    int b = leaves[blockIdx.x];
    int rhs = blockIdx.y;
    int P = A.Plev[A.blevel[b]];
    cd* coef = sm;                                  // 2*maxP+1
    cd* rows = sm + 2 * maxP + 1;                   // per thread: 2*maxP+3 (Helmholtz rows n = -P-1..P+1)
    int s0 = A.trg.st[b], s1 = A.trg.en[b];
    const double kh = 0.5 * A.kappa;
    for (int t0 = s0; t0 < s1; t0 += blockDim.x) {
        bool valid = t0 + (int)threadIdx.x < s1;
        const int64_t i = valid ? A.trg.at(t0 + threadIdx.x) : 0;
        cd x0 = {0, 0}, x1 = {0, 0};
        if (valid) {
            x0 = cd{A.xr[i], A.xi[i]};
            x1 = cd{A.xr[A.n + i], A.xi[A.n + i]};
        }
        cd dz = {0, 0}, de = {0, 0};
        cd* row = rows + (size_t)threadIdx.x * (2 * maxP + 3);
        for (int q = l3off[b]; q < l3off[b + 1]; ++q) {
            int s = l3[q];
            int Ps = A.Plev[A.blevel[s]];
            __syncthreads();
            const cd* m = mp + (int64_t)rhs * A.ncoef + A.eoff[s];
            for (int c = threadIdx.x; c < 2 * Ps + 1; c += blockDim.x) coef[c] = m[c];
            __syncthreads();
            if (!valid) continue;
            cd z, e;
            zeta_eta(x0 - cd{A.cre[2 * s], A.cim[2 * s]}, x1 - cd{A.cre[2 * s + 1], A.cim[2 * s + 1]}, z, e);
            if (KER == CFMM_LAPLACE) {
                const double iu = pow2(A.blevel[s] - A.we);
                cd iz = cinv(iu * z), ie = cinv(iu * e);
                dz += 0.5 * (coef[0] * (iu * iz));
                de += 0.5 * (coef[0] * (iu * ie));
                cd zp = iu * (iz * iz), ep = iu * (ie * ie);   // zeta^-n-1
                for (int nn = 1; nn <= Ps; ++nn) {
                    dz -= (double)nn * (coef[Ps + nn] * zp);
                    de -= (double)nn * (coef[nn] * ep);
                    zp = zp * iz;
                    ep = ep * ie;
                }
            } else {
                cyl_row(1, z, e, A.H, Ps, row);          // S_n, n = -Ps-1..Ps+1
                for (int nn = -Ps; nn <= Ps; ++nn) {
                    cd c = coef[Ps + nn];
                    dz = cmac(dz, c, row[nn + Ps + 1 - 1]);
                    de = cmac(de, c, row[nn + Ps + 1 + 1]);
                }
            }
        }
        __syncthreads();
        const cd* lc = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
        for (int c = threadIdx.x; c < 2 * P + 1; c += blockDim.x) coef[c] = lc[c];
        __syncthreads();
        if (!valid) continue;
        cd z, e;
        zeta_eta(x0 - cd{A.cre[2 * b], A.cim[2 * b]}, x1 - cd{A.cre[2 * b + 1], A.cim[2 * b + 1]}, z, e);
        cd lz = {0, 0}, le = {0, 0};
        if (KER == CFMM_LAPLACE) {
            const double iu = pow2(A.blevel[b] - A.we);
            z = iu * z;
            e = iu * e;
            cd zp = {iu, 0}, ep = {iu, 0};   // zeta^n-1
            for (int nn = 1; nn <= P; ++nn) {
                lz += (double)nn * (coef[nn] * zp);
                le += (double)nn * (coef[P + nn] * ep);
                zp = zp * z;
                ep = ep * e;
            }
        } else {
            cyl_row(0, z, e, A.H, P, row);               // G_n, n = -P-1..P+1
            for (int nn = -P; nn <= P; ++nn) {
                cd c = coef[P + nn];
                lz = cmac(lz, c, row[nn + P + 1 - 1]);
                le = cmac(le, c, row[nn + P + 1 + 1]);
            }
        }
        if (KER == CFMM_LAPLACE) {
            dz += lz;
            de += le;
        } else {
            dz = kh * (dz + lz);
            de = (-kh) * (de + le);
        }
        cd* go = g + (int64_t)rhs * 2 * A.n + i;
        go[0] += dz + de;
        go[A.n] += mul_i(dz - de);
    }
}

// ---------------------------------------------------------------------------
// L2P in complex64 arithmetic (mixed precision). With zeta~ = zeta/rho_b,
// eta~ = eta/rho_b (rho_b = sqrt(2)/2 w, the leaf's radius):
//   Laplace    u = L^_0 + sum L^_n zeta~^n + L^'_n eta~^n,  L^_n = L_n rho_b^n (rho_b in
//              the box's unit, as L_n is)
//   Helmholtz  u = sum_n Jh_n(k r) (L^_n zeta~^n + L^_-n eta~^n),
//              L^_n = L_n (k rho_b/2)^n/n!,  L^_-n = (-1)^n L_-n (k rho_b/2)^n/n!
// (G_n = J_n(k r) (zeta/r)^n, G_-n = (-1)^n J_n(k r) (eta/r)^n), where
//   Jh_n(z) = J_n(z) n! (2/z)^n
// is entire in w = z^2 = (k rho_b)^2 zeta~ eta~ with Jh_n(0) = 1. From
// J_{n-1} + J_{n+1} = (2n/z) J_n,  Jh_{n-1} = Jh_n - (w/4) Jh_{n+1}/(n(n+1)),
// so the ratios q_n = Jh_n/Jh_{n-1} = 1/(1 - (w/4) q_{n+1}/(n(n+1))) follow by
// Miller's backward recurrence from q = 1, and Jh_0 = J_0 from
// exp(-+ i z) = J_0 + 2 sum (-+ i)^k J_k = Jh_0 (1 + 2 sum (-+ i z/2)^k/k! prod q).
// Coefficients are scaled in FP64 per leaf and rounded; the terms are added
// in a compensated (Kahan) FP32 sum.
// ---------------------------------------------------------------------------
constexpr int kL2p2fMaxP = 128;

template <int KER>
__global__ void __launch_bounds__(kExpThreads) k_l2p2f(ExpArgs A, const int* __restrict__ leaves,
                                                        const cd* __restrict__ loc, cd* __restrict__ u, double W) {
    extern __shared__ cf coef2[];
    int b = leaves[blockIdx.x];
    int rhs = blockIdx.y;
    int lev = A.blevel[b];
    int P = A.Plev[lev];
    int nc = 2 * P + 1;
    double rb = 0.70710678118654752440 * ldexp(W, -lev);
    const cd* lc = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        // Laplace layout [c0, zeta^1..zeta^P, eta^1..eta^P]; Helmholtz [c_-P .. c_P]
        int n = KER == CFMM_LAPLACE ? (c <= P ? c : c - P) : abs(c - P);
        double s = 1.0, g = KER == CFMM_LAPLACE ? pow2(lev - A.we) * rb : 0.5 * A.kappa * rb;
        for (int j = 1; j <= n; ++j) s *= KER == CFMM_LAPLACE ? g : g / j;
        if (KER != CFMM_LAPLACE && c < P && (n & 1)) s = -s;
        coef2[c] = to_cf(s * lc[c]);
    }
    __syncthreads();
    double irb = 1.0 / rb;
    cd c0 = {A.cre[2 * b], A.cim[2 * b]}, c1 = {A.cre[2 * b + 1], A.cim[2 * b + 1]};
    cf G[kL2p2fMaxP + 1];
    for (int k = A.trg.st[b] + threadIdx.x; k < A.trg.en[b]; k += blockDim.x) {
        const int64_t i = A.trg.at(k);
        cd d0 = irb * (cd{A.xr[i], A.xi[i]} - c0), d1 = irb * (cd{A.xr[A.n + i], A.xi[A.n + i]} - c1);
        cf zt = to_cf(d0 + mul_i(d1)), et = to_cf(d0 - mul_i(d1));
        Kahan acc;
        if (KER == CFMM_LAPLACE) {
            acc.add(coef2[0]);
            cf zp = zt, ep = et;
            for (int nn = 1; nn <= P; ++nn) {
                acc.add(cmacf(coef2[nn] * zp, coef2[P + nn], ep));
                zp = zp * zt;
                ep = ep * et;
            }
        } else {
            float kr = (float)(A.kappa * rb);
            cf w = (kr * kr) * (zt * et);
            cf zz = csqrtf_p(w);
            float big = fmaxf((float)P, hypotf(zz.x, zz.y));
            int N = (int)big + 12 + (int)sqrtf(8.f * big);
            bool up = zz.y >= 0.f;
            cf a = 0.5f * (up ? cf{zz.y, -zz.x} : cf{-zz.y, zz.x});   // -+ i z / 2
            cf q = {1.f, 0.f}, H = {1.f, 0.f};
            for (int nn = N; nn >= 1; --nn) {
                float den = 0.25f / ((float)nn * (float)(nn + 1));
                q = cinvf(cf{1.f, 0.f} - (den * w) * q);
                if (nn <= P) G[nn] = q;
                H = cf{1.f, 0.f} + (1.f / (float)nn) * (a * (q * H));
            }
            float ex = expf(2.f * a.x), sn, cs;
            sincosf(2.f * a.y, &sn, &cs);
            cf g = cf{ex * cs, ex * sn} * cinvf(2.f * H - cf{1.f, 0.f});
            acc.add(coef2[P] * g);
            cf zp = zt, ep = et;
            for (int nn = 1; nn <= P; ++nn) {
                g = g * G[nn];
                acc.add(g * cmacf(coef2[P + nn] * zp, coef2[P - nn], ep));
                zp = zp * zt;
                ep = ep * et;
            }
        }
        u[(int64_t)rhs * A.n + i] += acc.value();
    }
}

// table kernels (plan time)
__global__ void k_tab_m2l(int nq, const int* __restrict__ qbox, const int* __restrict__ lent,
                          const int* __restrict__ blevel, const int* __restrict__ Plev, const int64_t* __restrict__ tbase,
                          const int* __restrict__ tq0, const double* __restrict__ cre, const double* __restrict__ cim,
                          HankelArgs H, cd* __restrict__ tab, int q_first) {
    int qi = blockIdx.x * blockDim.x + threadIdx.x;
    if (qi >= nq) return;
    int q = q_first + qi;
    int b = qbox[qi], s = lent[q];
    int l = blevel[b];
    int P = Plev[l];
    cd* t = tab + tbase[l] + (int64_t)(q - tq0[l]) * (4 * P + 1);
    // S_j(c_t - c_s), j = -2P..2P, stored at j + 2P
    cd z, e;
    zeta_eta(cd{cre[2 * b] - cre[2 * s], cim[2 * b] - cim[2 * s]},
             cd{cre[2 * b + 1] - cre[2 * s + 1], cim[2 * b + 1] - cim[2 * s + 1]}, z, e);
    cd r = csqrt_p(z * e);
    cd zz = H.w.k * r;
    cd h0, h1;
    hankel01_r2(H, z * e, &h0, &h1);
    cd ir = cinv(r), uu = z * ir, vv = e * ir, zi = cinv(zz);
    int M = 2 * P;
    t[M] = h0;
    cd hm = h0, hn = h1, up = uu, vp = vv;
    for (int j = 1; j <= M; ++j) {
        cd neg = (j & 1) ? -hn : hn;
        t[M + j] = hn * up;
        t[M - j] = neg * vp;
        cd hp = (2.0 * j) * (zi * hn) - hm;
        hm = hn;
        hn = hp;
        up = up * uu;
        vp = vp * vv;
    }
}

// per child box: G_j(c_parent - c_child), j = -(Pc+Pp)..(Pc+Pp); scratch row per thread
__global__ void k_tab_shift(int lo, int hi, const int* __restrict__ parent, const int* __restrict__ blevel,
                            const int* __restrict__ Plev, const int64_t* __restrict__ shoff,
                            const double* __restrict__ cre, const double* __restrict__ cim, double kappa,
                            cd* __restrict__ tab) {
    int b = lo + blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= hi) return;
    int p = parent[b];
    int Pc = Plev[blevel[b]], Pp = Plev[blevel[p]];
    int M = Pc + Pp;
    cd* t = tab + shoff[b];
    cd z, e;
    zeta_eta(cd{cre[2 * p] - cre[2 * b], cim[2 * p] - cim[2 * b]},
             cd{cre[2 * p + 1] - cre[2 * b + 1], cim[2 * p + 1] - cim[2 * b + 1]}, z, e);
    cd r = csqrt_p(z * e);
    // J_0..J_M into the positive half, then the angular factors
    bessel_j_seq(kappa * r, M, t + M);
    if (r.x == 0.0 && r.y == 0.0) {
        for (int j = 1; j <= M; ++j) t[M - j] = cd{0, 0};
        return;
    }
    cd ir = cinv(r), uu = z * ir, vv = e * ir, up = uu, vp = vv;
    for (int j = 1; j <= M; ++j) {
        cd f = t[M + j];
        cd neg = (j & 1) ? -f : f;
        t[M - j] = neg * vp;
        t[M + j] = f * up;
        up = up * uu;
        vp = vp * vv;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct PlanExt {
    cfmm_plan_s* P;
    Fmm2dState* S;
};
static std::mutex g_ext_mu;
static std::vector<PlanExt>& exts() {
    static std::vector<PlanExt> v;
    return v;
}

static Fmm2dState* state(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_ext_mu);
    for (auto& e : exts())
        if (e.P == P) return e.S;
    return nullptr;
}

void fmm2d_release(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_ext_mu);
    auto& v = exts();
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i].P == P) {
            delete v[i].S;
            v.erase(v.begin() + i);
            return;
        }
}

// Sec. 6.3: expansion order per level (prefactors dropped, one digit of headroom)
static int nterms_laplace(int dim, int k, double eps) {
    double ratio = (std::sqrt((double)dim) * 0.5) / (k + 0.5);
    double t = 1.0;
    int n = 0;
    for (;;) {
        ++n;
        t *= ratio;
        if (t <= eps) return n;
    }
}

static int nterms_helm2d_upto(int k, double eps, double kappa, double w, int pmax) {
    double R = (k + 0.5) * w, r = std::sqrt(2.0) * 0.5 * w;
    std::vector<cd> J(pmax + 4), H(pmax + 4);
    bessel_j_seq(cd{kappa * r, 0.0}, pmax + 3, J.data());
    cd zR = {kappa * R, 0.0};
    hankel01(zR, &H[0], &H[1]);
    cd zi = cinv(zR);
    for (int m = 1; m < pmax + 3; ++m) H[m + 1] = (2.0 * m) * (zi * H[m]) - H[m - 1];
    std::vector<char> ok(pmax + 4);
    for (int m = 0; m < pmax + 4; ++m) {
        cd v = H[m] * J[m];
        double a = std::sqrt(cabs2(v));
        ok[m] = std::isfinite(a) && a <= eps;
    }
    for (int n = 1; n < pmax; ++n)
        if (ok[n] && ok[n + 1] && ok[n + 2] && ok[n + 3]) return n;
    return -1;
}

// smallest n with |H_n(kR) J_n(kr)| <= eps for n..n+3 (search up to 2000; a
// short search range first, since the answer is near k R for large k R and
// O(log eps) otherwise)
static int nterms_helm2d(int k, double eps, double kappa, double w) {
    int guess = (int)(kappa * (k + 0.5) * w) + 80;
    if (guess < 2000) {
        int n = nterms_helm2d_upto(k, eps, kappa, w, guess);
        if (n > 0) return n;
    }
    int n = nterms_helm2d_upto(k, eps, kappa, w, 2000);
    return n > 0 ? n : 2000;
}

// the criterion is applied at eps * headroom: one digit for Laplace, two for
// Helmholtz (|H_n(kR) J_n(kr)| carries an extra 1/(n pi) against (r/R)^n)
constexpr double kPHeadroom = 0.1;
constexpr double kPHeadroomHelm = 0.01;

static HankelArgs hankel_args(double kappa) { return HankelArgs{pair_tab_device(), make_wave(kappa)}; }

// First part of the setup, run before the lists are built: orders, offsets,
// the leaves and (Helmholtz) the per-point row table and the children's shift
// tables, launched on the side stream so that they overlap the construction of the
// lists.
void fmm2d_presetup(cfmm_plan_s* P) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    PhaseTimer pt(st);
    Fmm2dState* S = new Fmm2dState();
    {
        std::lock_guard<std::mutex> lk(g_ext_mu);
        exts().push_back(PlanExt{P, S});
    }
    S->ker = P->kernel;
    S->l0 = T.l0;
    S->nlev = T.nlevels;
    std::frexp(P->W, &S->we);
    S->we = std::min(900, std::max(-900, S->we));
    S->Plev.assign(T.nlevels, 0);
    for (int l = 0; l < T.nlevels; ++l) {
        if (P->kernel == CFMM_LAPLACE) S->Plev[l] = nterms_laplace(2, P->sep, P->eps * kPHeadroom);
        // Helmholtz levels above the top expansion level carry no expansions:
        // their (large, host-evaluated) orders are not computed and read 0
        else if (l >= S->l0 || T.nboxes <= 1)
            S->Plev[l] = nterms_helm2d(P->sep, P->eps * kPHeadroomHelm, P->kappa, std::ldexp(P->W, -l));
    }
    P->P = S->Plev;
    pt.mark("setup:orders");
    if (T.nboxes <= 1) return;   // single leaf: near field only
    int maxP = 0;
    for (int l = S->l0; l < T.nlevels; ++l) maxP = std::max(maxP, S->Plev[l]);
    CFMM_REQUIRE(maxP <= 1000, CFMM_EUNSUPPORTED, "expansion order above 1000 at the top expansion level");
    S->maxP = maxP;
    P->maxP = maxP;
    S->dPlev.alloc(T.nlevels);
    upload(S->dPlev.get(), S->Plev.data(), sizeof(int) * T.nlevels, st);
    // coefficient offsets
    std::vector<int64_t> off(T.nboxes, -1);
    int64_t tot = 0;
    for (int l = S->l0; l < T.nlevels; ++l)
        for (int b = T.level_off[l]; b < T.level_off[l + 1]; ++b) {
            off[b] = tot;
            tot += 2 * S->Plev[l] + 1;
        }
    S->ncoef = tot;
    P->ncoef = tot;
    S->exp_off.alloc(T.nboxes);
    upload(S->exp_off.get(), off.data(), sizeof(int64_t) * T.nboxes, st);
    // leaves at level >= l0 (all leaves when the tree has more than one box);
    // boxes are level-major, so a box's level follows from the level offsets
    auto level_of = [&](int b) {
        return (int)(std::upper_bound(T.level_off.begin(), T.level_off.end(), b) - T.level_off.begin()) - 1;
    };
    S->maxP_leaf = 0;
    int lmin = T.nlevels;
    for (int b : T.leaf_boxes) {
        int lb = level_of(b);
        if (lb >= S->l0) {
            S->leaves_l0.push_back(b);
            S->maxP_leaf = std::max(S->maxP_leaf, S->Plev[lb]);
            lmin = std::min(lmin, lb);
        }
    }
    // a leaf's List 3 boxes lie below its level: their orders and the leaf's
    // own are at most the largest order at or below the coarsest leaf level
    S->maxP_fine = 0;
    for (int l = lmin; l < T.nlevels; ++l) S->maxP_fine = std::max(S->maxP_fine, S->Plev[l]);
    S->d_leaves_l0.alloc(S->leaves_l0.size());
    upload(S->d_leaves_l0.get(), S->leaves_l0.data(), sizeof(int) * S->leaves_l0.size(), st);
    pt.mark("setup:leaves");
    if (P->kernel == CFMM_HELMHOLTZ) {   // (a tree of several boxes has leaves below l0)
        // on the side stream, beside the lists: the rows and the shift tables
        S->RL = 2 * S->maxP_leaf + 3;
        S->lrow.alloc((size_t)P->n * S->RL);
        S->rows_side = true;
        // (its offsets are uploaded on the plan's stream, before the fork)
        std::vector<int64_t> so(T.nboxes, -1);
        int64_t sb = 0;
        for (int l = S->l0 + 1; l < T.nlevels; ++l)
            for (int b = T.level_off[l]; b < T.level_off[l + 1]; ++b) {
                so[b] = sb;
                sb += 2 * (S->Plev[l] + S->Plev[l - 1]) + 1;
            }
        S->t_shift.alloc(sb > 0 ? sb : 1);
        S->shift_off.alloc(T.nboxes);
        upload(S->shift_off.get(), so.data(), sizeof(int64_t) * T.nboxes, st);
        cudaStream_t side = near_fork(P);
        if (!S->leaves_l0.empty())
            k_leaf_rows<<<(unsigned)S->leaves_l0.size(), 64, 0, side>>>(
            S->d_leaves_l0.get(), T.level.get(), T.start.get(), T.end.get(), S->dPlev.get(), P->xr.get(),
            P->xi.get(), P->n, T.cen_re.get(), T.cen_im.get(), hankel_args(P->kappa), S->RL, S->lrow.get());
        CFMM_LAUNCHED();
        // translation tables of the child boxes (levels > l0)
        int lo = T.level_off[std::min(S->l0 + 1, T.nlevels)], hi = T.nboxes;
        if (hi > lo) {
            k_tab_shift<<<(hi - lo + 31) / 32, 32, 0, side>>>(lo, hi, T.parent.get(), T.level.get(), S->dPlev.get(),
                                                             S->shift_off.get(), T.cen_re.get(), T.cen_im.get(),
                                                             P->kappa, S->t_shift.get());
            CFMM_LAUNCHED();
        }
    }
}

// The rest of the setup, once the lists exist: P2L boxes, translation tables,
// List-2 chunks; joins the side stream's row table at the end.
void fmm2d_setup(cfmm_plan_s* P) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    if (!state(P)) fmm2d_presetup(P);
    Fmm2dState* S = state(P);
    PhaseTimer pt(st);
    if (T.nboxes <= 1) return;   // single leaf: near field only
    int maxP = S->maxP;
    // boxes that receive P2L contributions
    {
        const std::vector<int>& l4 = T.hloff[3];
        std::vector<int> boxes;
        for (int b = T.level_off[S->l0]; b < T.nboxes; ++b)
            if (l4[b + 1] > l4[b]) boxes.push_back(b);
        S->n_p2l = (int)boxes.size();
        S->d_p2l_boxes.alloc(boxes.size());
        if (!boxes.empty())
            upload(S->d_p2l_boxes.get(), boxes.data(), sizeof(int) * boxes.size(), st);
    }
    pt.mark("setup:p2l");
    if (P->kernel == CFMM_LAPLACE) {
        // binomials C(n, k), n < 2 maxP (exact integers up to 2^53, then rounded)
        const size_t w = maxP + 1, nb = 2 * (size_t)maxP;
        std::vector<double> bt(nb * nb, 0.0), a(w * w, 0.0), c(w * w, 0.0), d(w * w, 0.0);
        for (size_t n = 0; n < nb; ++n) {
            bt[n * nb] = 1.0;
            for (size_t k = 1; k <= n; ++k) bt[n * nb + k] = bt[(n - 1) * nb + k - 1] + bt[(n - 1) * nb + k];
        }
        for (size_t n = 1; n < w; ++n)
            for (size_t k = 1; k < w; ++k) {
                if (n <= k) a[n * w + k] = std::ldexp(bt[(k - 1) * nb + n - 1], -(int)n);
                c[n * w + k] = bt[(n + k - 1) * nb + k];
                if (n >= k) d[n * w + k] = std::ldexp(bt[n * nb + k], -(int)k);
            }
        for (auto t : {std::make_pair(&S->cm2m, &a), std::make_pair(&S->cm2l, &c), std::make_pair(&S->cl2l, &d)}) {
            t.first->alloc(w * w);
            upload(t.first->get(), t.second->data(), sizeof(double) * w * w, st);
        }
    }
    if (P->kernel == CFMM_HELMHOLTZ) {
        // M2L tables, level-major like List 2 itself
        const std::vector<int>& loff = T.hloff[1];
        S->m2l_base.assign(T.nlevels, 0);
        S->m2l_q0.assign(T.nlevels, 0);
        int64_t base = 0;
        for (int l = 0; l < T.nlevels; ++l) {
            int q0 = loff[T.level_off[l]], q1 = loff[T.level_off[l + 1]];
            S->m2l_base[l] = base;
            S->m2l_q0[l] = q0;
            if (l >= S->l0) base += (int64_t)(q1 - q0) * (4 * S->Plev[l] + 1);
        }
        S->t_m2l.alloc(base > 0 ? base : 1);
        S->d_m2l_base.alloc(T.nlevels);
        S->d_m2l_q0.alloc(T.nlevels);
        upload(S->d_m2l_base.get(), S->m2l_base.data(), sizeof(int64_t) * T.nlevels, st);
        upload(S->d_m2l_q0.get(), S->m2l_q0.data(), sizeof(int) * T.nlevels, st);
        // owner box of every List-2 entry at levels >= l0
        int qf = loff[T.level_off[S->l0]], ql = loff[T.nboxes];
        if (ql > qf) {
            std::vector<int> qbox(ql - qf);
            for (int b = T.level_off[S->l0]; b < T.nboxes; ++b)
                for (int q = loff[b]; q < loff[b + 1]; ++q) qbox[q - qf] = b;
            int* dq = plan_scratch().take_n<int>(qbox.size());
            upload(dq, qbox.data(), sizeof(int) * qbox.size(), st);
            int nq = ql - qf;
            // one warp per block: the few thousand pairs (one thread each) spread over
            // every SM instead of filling a fraction of them with larger blocks
            k_tab_m2l<<<(nq + 31) / 32, 32, 0, st>>>(nq, dq, T.lent[1].get(), T.level.get(), S->dPlev.get(),
                                                       S->d_m2l_base.get(), S->d_m2l_q0.get(), T.cen_re.get(),
                                                       T.cen_im.get(), hankel_args(P->kappa), S->t_m2l.get(), qf);
            CFMM_LAUNCHED();
        }
        pt.mark("setup:m2ltab");
        // List-2 chunks per box (levels >= l0)
        {
            std::vector<int> cb, c0v, c1v, bc0(T.nboxes + 1, 0);
            std::vector<int64_t> cp;
            int64_t pslot = 0;
            for (int l = 0; l < T.nlevels; ++l) {
                // chunks of kM2LChunk entries (shorter chunks fill more SMs at a coarse
                // top level but spread each block's fixed per-coefficient work over
                // fewer sources: measured slower)
                int clen = kM2LChunk;
                for (int b = T.level_off[l]; b < T.level_off[l + 1]; ++b) {
                    bc0[b] = (int)cb.size();
                    if (l < S->l0) continue;
                    for (int q = loff[b]; q < loff[b + 1]; q += clen) {
                        cb.push_back(b);
                        c0v.push_back(q);
                        c1v.push_back(std::min(q + clen, loff[b + 1]));
                        cp.push_back(pslot);
                        pslot += 2 * S->Plev[l] + 1;
                    }
                }
            }
            S->nchunk = (int)cb.size();
            bc0[T.nboxes] = (int)cb.size();
            S->npart = pslot;
            S->chunk_box.alloc(cb.size());
            S->chunk_q0.alloc(cb.size());
            S->chunk_q1.alloc(cb.size());
            S->chunk_part.alloc(cb.size());
            S->box_chunk0.alloc(T.nboxes + 1);
            if (!cb.empty()) {
                upload(S->chunk_box.get(), cb.data(), sizeof(int) * cb.size(), st);
                upload(S->chunk_q0.get(), c0v.data(), sizeof(int) * cb.size(), st);
                upload(S->chunk_q1.get(), c1v.data(), sizeof(int) * cb.size(), st);
                upload(S->chunk_part.get(), cp.data(), sizeof(int64_t) * cp.size(), st);
            }
            upload(S->box_chunk0.get(), bc0.data(), sizeof(int) * (T.nboxes + 1), st);
        }
        pt.mark("setup:chunks");
    }
    if (S->rows_side) near_join(P);
    pt.mark("setup:rowsjoin");
}

void init_fmm2d() {
    for (auto f : {(const void*)k_point_to_exp<CFMM_LAPLACE>, (const void*)k_point_to_exp<CFMM_HELMHOLTZ>,
                   (const void*)k_m2m_lap, (const void*)k_m2m_helm, (const void*)k_l2l_lap, (const void*)k_l2l_helm,
                   (const void*)k_m2l_lap, (const void*)k_m2l_helm,
                   (const void*)k_m2l_chunk,
                   (const void*)k_eval<CFMM_LAPLACE>, (const void*)k_eval<CFMM_HELMHOLTZ>,
                   (const void*)k_eval_grad<CFMM_LAPLACE>, (const void*)k_eval_grad<CFMM_HELMHOLTZ>})
        CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
}

template <int KER>
static void apply_t(cfmm_plan_s* P, Fmm2dState* S, const cd* sigma, const cd* tau, int64_t dstride, cd* u, int nrhs,
                    cd* g) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    auto rec = [&](int i) {
        if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev[i], st));
    };
    KParams K{P->xr.get(), P->xi.get(), P->nr.get(), P->ni.get(), P->xr.get(), P->xi.get(), P->n, P->n,
              sigma, tau, dstride, P->slp, P->dlp, P->kappa};
    if (T.nboxes <= 1) {
        for (int i = 2; i <= 6; ++i) rec(i);
        launch_p2p(2, KER, K, T.d_leaf_boxes.get(), T.nleaves, near_ranges(P), T.loff[0].get(),
                   T.lent[0].get(), u, nrhs, st, P->precision == CFMM_MIXED, P->leaf_size);
        if (g)
            launch_p2p_grad(2, KER, K, T.d_leaf_boxes.get(), T.nleaves, near_ranges(P), T.loff[0].get(),
                            T.lent[0].get(), g, nrhs, st, P->leaf_size);
        rec(7);
        rec(8);
        return;
    }
    size_t need = (size_t)S->ncoef * nrhs;
    P->mpole.alloc(need);
    P->local.alloc(need);
    cd* mp = P->mpole.get();
    cd* lc = P->local.get();
    ExpArgs A{P->xr.get(), P->xi.get(), P->nr.get(), P->ni.get(), P->n, sigma, tau, dstride, P->slp, P->dlp,
              P->kappa, T.level.get(), source_range(P), target_range(P), T.cen_re.get(), T.cen_im.get(),
              S->dPlev.get(), S->exp_off.get(), S->ncoef, hankel_args(P->kappa), S->we};
    int maxP = S->maxP;
    // (6) P2L over List 4, added to the local expansions
    auto p2l = [&](cudaStream_t s) {
        if (S->n_p2l == 0) return;
        int R = KER == CFMM_LAPLACE ? 2 * maxP + 1 : 2 * maxP + 3;
        int chunk = std::max(1, std::min(kExpThreads, (int)((96 * 1024) / ((R + 3) * sizeof(cd)))));
        size_t smem = sizeof(cd) * (p2e_acc(maxP) + (size_t)chunk * (R + 3));
        k_point_to_exp<KER><<<dim3(S->n_p2l, nrhs), kP2eThreads, smem, s>>>(
            A, S->d_p2l_boxes.get(), T.loff[3].get(), T.lent[3].get(), 1, lc, chunk, nullptr, 0);
        CFMM_LAUNCHED();
    };
    // (5) M2P over List 3, added to u
    bool l2p32 = P->precision == CFMM_MIXED && S->maxP_leaf <= kL2p2fMaxP;
    // P2L and (mixed) M2P are short chains on a few blocks that need nothing of the
    // M2L: they run on the side stream, P2L into zeroed expansions before the near
    // field and M2P after it (0.08 and 0.13 of 1.43 ms of a 100,000-point mixed 2D
    // Helmholtz apply). An FP64 near field of more than 2^21 pairs (1 ms) is itself the
    // longer branch, and P2L stays in its place.
    const bool side_work = !(P->timing && P->serial);
    const bool p2l_first = side_work && S->n_p2l > 0 && (P->precision == CFMM_MIXED || P->p2p_pairs <= (1 << 21));
    const bool m2p_side = side_work && l2p32 && T.llen[2] > 0;
    auto eval = [&](cudaStream_t s, int do_l2p) {
        // with the plan's rows, L2P needs no per-thread row space
        size_t smem = sizeof(cd) * ((size_t)(2 * maxP + 1) + (size_t)kExpThreads * (S->lrow.get() ? 1 : maxP + 2));
        dim3 gr((unsigned)S->leaves_l0.size(), nrhs);
        k_eval<KER><<<gr, kExpThreads, smem, s>>>(A, S->d_leaves_l0.get(), T.loff[2].get(), T.lent[2].get(), mp, lc, u,
                                                 maxP, S->lrow.get(), S->RL, do_l2p);
        CFMM_LAUNCHED();
    };
    // (3) P2P over List 1 (writes u) on the side stream, beside the far field
    cudaStream_t ns = near_fork(P);
    {
        if (p2l_first) {
            P->p2l_side = true;
            if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev_side[0], ns));
            CFMM_CUDA(cudaMemsetAsync(lc, 0, sizeof(cd) * need, ns));
            p2l(ns);
            CFMM_CUDA(cudaEventRecord(P->ev_far[0], ns));
            if (P->timing) {
                CFMM_CUDA(cudaEventRecord(P->ev_side[1], ns));
                CFMM_CUDA(cudaEventRecord(P->ev_p2p[0], ns));    // the near field begins here
            }
        }
        launch_p2p(2, KER, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P),
                   T.loff[0].get(), T.lent[0].get(), u, nrhs, ns, P->precision == CFMM_MIXED, P->leaf_size);
        if (g)
            launch_p2p_grad(2, KER, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P),
                            T.loff[0].get(), T.lent[0].get(), g, nrhs, ns, P->leaf_size);
    }
    near_launched(P);
    // (1) P2M (shared memory sized by the leaves' orders)
    {
        int PL = S->maxP_leaf;
        int R = KER == CFMM_LAPLACE ? 2 * PL + 1 : 2 * PL + 3;
        int chunk = std::max(1, std::min(kExpThreads, (int)((96 * 1024) / ((R + 3) * sizeof(cd)))));
        size_t smem = sizeof(cd) * (p2e_acc(PL) + (size_t)chunk * (R + 3));
        dim3 g((unsigned)S->leaves_l0.size(), nrhs);
        if (g.x) {
            k_point_to_exp<KER><<<g, kP2eThreads, smem, st>>>(A, S->d_leaves_l0.get(), nullptr, nullptr, 0, mp, chunk,
                                                             S->lrow.get(), S->RL);
            CFMM_LAUNCHED();
        }
    }
    rec(2);
    // (2) M2M, finest level first
    TransArgs TA{T.level.get(), T.parent.get(), T.cbeg.get(), T.cend.get(), T.cen_re.get(), T.cen_im.get(),
                 S->dPlev.get(), S->exp_off.get(), S->ncoef, S->we, S->t_shift.get(),
                 S->shift_off.get()};
    // Helmholtz: parts of a coefficient's sum, threads of a block
    auto split = [](int nc) { return std::max(1, std::min(8, 512 / nc)); };
    auto threads = [](int nc, int S2) { return std::min(512, (nc * S2 + 31) / 32 * 32); };
    for (int l = T.nlevels - 2; l >= S->l0; --l) {
        int lo = T.level_off[l], nb = T.level_off[l + 1] - lo;
        int Pp = S->Plev[l], Pc = S->Plev[l + 1];
        dim3 g(nb, nrhs);
        if (KER == CFMM_LAPLACE) {
            const int ng = 2;
            k_m2m_lap<<<g, ng * lap_group(Pp), sizeof(cd) * 2 * ng * (2 * Pp + 1), st>>>(TA, lo, mp, mp, T.leaf.get(),
                                                                                      Pp, S->cm2m.get());
        } else {
            const int S2 = split(2 * Pp + 1);
            k_m2m_helm<<<g, threads(2 * Pp + 1, S2), sizeof(cd) * ((2 * Pc + 1) + 2 * (Pc + Pp) + 1 + S2 * (2 * Pp + 1)),
                         st>>>(TA, lo, mp, mp, T.leaf.get(), Pc, Pp, S2);
        }
        CFMM_LAUNCHED();
    }
    rec(3);
    if (m2p_side) {
        CFMM_CUDA(cudaEventRecord(P->ev_far[1], st));
        CFMM_CUDA(cudaStreamWaitEvent(ns, P->ev_far[1], 0));
        P->m2p_side = true;
        if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev_side[2], ns));
        eval(ns, 0);
        if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev_side[3], ns));
    }
    if (p2l_first) CFMM_CUDA(cudaStreamWaitEvent(st, P->ev_far[0], 0));
    // (4) M2L over List 2 (all levels >= l0)
    {
        M2LArgs MA{T.level.get(), T.cen_re.get(), T.cen_im.get(), S->dPlev.get(), S->exp_off.get(), S->ncoef,
                   T.loff[1].get(), T.lent[1].get(), S->t_m2l.get(), S->d_m2l_base.get(), S->d_m2l_q0.get(), S->we};
        int first = T.level_off[S->l0], nb = T.nboxes - first;
        if (KER == CFMM_HELMHOLTZ && maxP <= 255) {
            // chunks of List-2 entries, then the per-box reduction of the chunk sums
            P->m2l_part.alloc((size_t)S->npart * nrhs + 1);
            cd* part = P->m2l_part.get();
            if (S->nchunk > 0) {
                int threads = std::max(256, (2 * maxP + 1 + 31) / 32 * 32);
                size_t smem = 0;
                for (int l = S->l0; l < T.nlevels; ++l) {
                    int ncl = 2 * S->Plev[l] + 1;
                    smem = std::max(smem, sizeof(cd) * (size_t)m2l_lanes(ncl, threads) * (ncl + 4 * S->Plev[l] + 1));
                }
                k_m2l_chunk<<<dim3(S->nchunk, nrhs), threads, smem, st>>>(MA, S->chunk_box.get(), S->chunk_q0.get(),
                                                                        S->chunk_q1.get(), S->chunk_part.get(), part,
                                                                        S->npart, mp);
                CFMM_LAUNCHED();
            }
            k_m2l_reduce<<<dim3(nb, nrhs), 64, 0, st>>>(first, T.level.get(), S->dPlev.get(), S->box_chunk0.get(),
                                                       S->chunk_part.get(), part, S->npart, S->exp_off.get(), S->ncoef,
                                                       p2l_first ? 1 : 0, lc);
            CFMM_LAUNCHED();
        } else {
            dim3 g(nb, nrhs);
            if (KER == CFMM_LAPLACE) {
                const int ng = 3;
                k_m2l_lap<<<g, ng * lap_group(maxP), sizeof(cd) * 2 * ng * (2 * maxP + 1), st>>>(
                    MA, first, mp, lc, maxP, S->cm2l.get(), pair_tab_device(), p2l_first ? 1 : 0);
            } else {
                size_t smem = sizeof(cd) * (2 * (2 * maxP + 1) + 4 * maxP + 3);
                k_m2l_helm<<<g, 128, smem, st>>>(MA, first, mp, lc, p2l_first ? 1 : 0);
            }
            CFMM_LAUNCHED();
        }
    }
    rec(4);
    if (!p2l_first) p2l(st);   // (6)
    rec(5);
    // (7) L2L, coarsest level first
    for (int l = S->l0 + 1; l < T.nlevels; ++l) {
        int lo = T.level_off[l], nb = T.level_off[l + 1] - lo;
        int Pp = S->Plev[l - 1], Pc = S->Plev[l];
        dim3 g(nb, nrhs);
        if (KER == CFMM_LAPLACE) {
            k_l2l_lap<<<g, lap_group(Pc), sizeof(cd) * (4 * Pc + 1), st>>>(TA, lo, lc, Pc, S->cl2l.get());
        } else {
            const int S2 = split(2 * Pc + 1);
            k_l2l_helm<<<g, threads(2 * Pc + 1, S2), sizeof(cd) * ((2 * Pp + 1) + 2 * (Pc + Pp) + 1 + S2 * (2 * Pc + 1)),
                         st>>>(TA, lo, lc, Pp, Pc, S2);
        }
        CFMM_LAUNCHED();
    }
    rec(6);
    rec(7);
    near_join(P);   // the near field has written u
    // (5) M2P and (8) L2P (add to u; L2P in complex64 in mixed precision)
    {
        dim3 gr((unsigned)S->leaves_l0.size(), nrhs);
        if (!m2p_side && !(l2p32 && T.llen[2] == 0)) eval(st, l2p32 ? 0 : 1);
        if (l2p32 && gr.x) {
            k_l2p2f<KER><<<gr, kExpThreads, sizeof(cf) * (2 * S->maxP_leaf + 1), st>>>(A, S->d_leaves_l0.get(), lc,
                                                                                        u, P->W);
            CFMM_LAUNCHED();
        }
        if (g && gr.x) {
            int Pg = S->maxP_fine;
            size_t gsm = sizeof(cd) * ((size_t)(2 * Pg + 1) + (size_t)kExpThreads * (2 * Pg + 3));
            CFMM_REQUIRE(gsm <= (size_t)kMaxSmem, CFMM_EUNSUPPORTED,
                         "2D gradient: leaf-level expansion order too large for the evaluation kernel");
            k_eval_grad<KER><<<gr, kExpThreads, gsm, st>>>(A, S->d_leaves_l0.get(), T.loff[2].get(), T.lent[2].get(),
                                                            mp, lc, g, Pg);
            CFMM_LAUNCHED();
        }
    }
    rec(8);
}

void fmm2d_apply(cfmm_plan_s* P, const cd* sigma, const cd* tau, int64_t dstride, cd* u, int nrhs, cd* g) {
    Fmm2dState* S = state(P);
    CFMM_REQUIRE(S, CFMM_EINVAL, "plan has no 2D state");
    if (P->kernel == CFMM_LAPLACE) apply_t<CFMM_LAPLACE>(P, S, sigma, tau, dstride, u, nrhs, g);
    else apply_t<CFMM_HELMHOLTZ>(P, S, sigma, tau, dstride, u, nrhs, g);
}

}  // namespace cfmm

// FP64 expansions of and at points in 3D, Laplace and Helmholtz: P2M and P2L (their own
// comment below), M2P over List 3 and L2P, potential and target gradient.
//
// The expansion functions (file comments of fmm3d.cu and helm3d.cu) share their
// dependence on z and rho^2 between +m and -m:
//   H_n^{+-m}(x) = F_n xi_{+-}^m q_n^m,  q_m^m = D_m,  q_n^m = A_n^m (zeta q_{n-1}^m) - B_n^m (w q_{n-2}^m),
//   Helmholtz      zeta = z, w = rho^2, xi+- = x+-,            F_n = f_n(kappa rho)/rho^n  (q from Z)
//   Laplace L2P    zeta = z, w = rho^2, xi+ = x+, xi- = -x-,   F_n = 1                     (q from U)
//   Laplace M2P    the same over rho^2, w = 1/rho^2,           F_n = 1/rho                 (q from T)
// so sum c_n^{+-m} H_n^{+-m} = sum_m xi+^m (sum_n F_n q_n c_n^m) + xi-^m (sum_n F_n q_n
// c_n^{-m}): 24 FP64 instructions per (n, m >= 0) for both signs instead of 20 for
// each, which is what bounds it (the FP64 pipe).
//
// A warp evaluates one expansion (a leaf's own, or one List-3 entry) at up to 32
// targets of a leaf. Fewer targets leave room for groups of lanes that take every
// G-th m each (a shell of leaves of one or two points has most List-3 entries of a
// small surface: 2.4 of 32 lanes were in use with a thread per target and a block
// per leaf, and the entries of a leaf ran one after the other). Each result goes to
// its own slot and k_eval3_sum adds a target's slots in list order.
#include <algorithm>
#include <cmath>

#include "eval3d.cuh"
#include "pair64.cuh"

namespace cfmm {

namespace {

__host__ __device__ __forceinline__ int nmi(int n, int m) { return n * n + n + m; }

__device__ __forceinline__ cd ldc(const cd* p) {
    double2 v = __ldg(reinterpret_cast<const double2*>(p));
    return cd{v.x, v.y};
}

constexpr int kEvalWarps = 4;
constexpr int64_t kEvalItems = (int64_t)1 << 27;   // slots of a launch over all right-hand sides, about
constexpr int64_t kEvalSlots = (int64_t)1 << 22;   // slots of a range of leaves (more than one only if they fit)

struct EvalK {
    const double *xr, *xi;
    int64_t n;
    Eval3Args E;
    SubRange trg;
    const int *l3off, *l3, *blevel;
    const double *cre, *cim;
    const int64_t* ioff;
    const int* own;
    EvalRange R;                  // the leaves of this launch
    int64_t nslot;                // its slots per right-hand side (and component): a target's L2P, then the items
    int l2p;                      // 0: List 3 only
    Eval3Tables T;
    const cd* gco;                // Helmholtz gradient: derived coefficients [3][2][ncoef] (multipole, local)
    cd* val;                      // [rhs][1 or 3][nslot]
    int nleaf_tasks, ntask;
};

// F_n = f_n(kappa rho)/rho^n, n = 0..N, of one lane into rows F[ld n]: h by forward
// recurrence, j by Miller's (both as in cfmm_special.cuh; the overflow test reads the
// exponent bits)
__device__ void radial_rows(bool sing, double kappa, cd r2, int N, cd* F, int ld = 32) {
    cd rho = csqrt_p(r2);
    if (rho.x == 0.0 && rho.y == 0.0) {
        double v = 1.0;
        for (int n = 0; n <= N; ++n) {
            F[n * ld] = cd{v, 0};
            v *= kappa / (2.0 * n + 3.0);
        }
        return;
    }
    cd z = kappa * rho, ir = cinv(rho), p = {1, 0};
    if (sing) {
        cd e = cexp_i(z), zi = cinv(z);
        cd h0 = -mul_i(e * zi), h1 = -(e * (z + cd{0.0, 1.0})) * (zi * zi);
        double c = 3.0;
        for (int n = 0; n <= N; ++n, c += 2.0) {
            F[n * ld] = h0 * p;
            p = p * ir;
            cd h2 = rmac(-h0, c, zi * h1);
            h0 = h1;
            h1 = h2;
        }
        return;
    }
    double az = hypot(z.x, z.y);
    double big = az > (double)N ? az : (double)N;
    int N0 = az <= 2.0 ? N + 13 + (int)(4.0 * az) : (int)big + 24 + (int)sqrt(32.0 * big);
    bool up = z.y >= 0.0;
    cd zi = cinv(z), fp = {0.0, 0.0}, f = {1e-200, 0.0}, S = {0.0, 0.0};
    double c2 = 2.0 * N0 + 1.0;
    for (int n = N0; n >= 1; --n, c2 -= 2.0) {
        if (n <= N) F[n * ld] = f;
        // (-+i)^n f
        int r = up ? n & 3 : (4 - n) & 3;
        cd w = r == 0 ? f : r == 1 ? cd{f.y, -f.x} : r == 2 ? -f : cd{-f.y, f.x};
        S = rmac(S, c2, w);
        cd fm = rmac(-fp, c2, zi * f);
        fp = f;
        f = fm;
        // |f| beyond 2^500: everything so far is scaled down
        unsigned hx = (unsigned)__double2hiint(f.x) & 0x7fffffffu, hy = (unsigned)__double2hiint(f.y) & 0x7fffffffu;
        if (max(hx, hy) >= 0x5f300000u) {
            const double sc = 3.0549363634996047e-151;     // 2^-500
            f = sc * f;
            fp = sc * fp;
            S = sc * S;
            for (int m = n; m <= min(N, N0); ++m) F[m * ld] = sc * F[m * ld];
        }
    }
    F[0] = f;
    S += f;
    cd s = (up ? cexp_i(-z) : cexp_i(z)) / S;
    for (int n = 0; n <= N; ++n) {
        F[n * ld] = F[n * ld] * s;
        s = s * ir;
    }
}

// Columns m = g, g + G, .. of the sums of one target. POT: u = sum c H. GRAD, Laplace:
// dz, dp, dm from the shifted coefficients (d+ U_n^m = -U_{n-1}^{m-1}/2 etc.), order
// Q = P - 1 (L2P) or P + 1 (M2P); Helmholtz: dz, dp, dm, b of eval with F_{n+1} from
// the derived coefficients (k_grad_coef).
template <bool LAP, bool GRAD>
__device__ __forceinline__ void eval_columns(const QTables& q, bool sing, cd zeta, cd w, cd xp, cd xm, int P,
                                             const cd* __restrict__ F, const cd* __restrict__ c,
                                             const cd* __restrict__ dc, int64_t dstride, int g, int G, cd* out) {
    constexpr int NS = !GRAD ? 1 : LAP ? 3 : 4;        // sums
    const int Q = GRAD && LAP ? (sing ? P + 1 : P - 1) : P;
    cd pp = {1, 0}, pm = {1, 0}, sp = {1, 0}, sm = {1, 0};
    for (int i = 0; i < G; ++i) {
        if (i == g) {
            pp = sp;
            pm = sm;
        }
        sp = sp * xp;
        sm = sm * xm;
    }
    for (int m = g; m <= Q; m += G) {
        cd a[NS], b[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) a[k] = b[k] = cd{0, 0};
        cd q2 = {0, 0}, q1 = {__ldg(q.D + m), 0};
        for (int n = m; n <= Q; ++n) {
            if (GRAD && LAP) {
                // H_n^{+-m} meets c_k^{+-m}, c_k^{+-m+1}, c_k^{+-m-1} with k = n + 1 (L2P) or n - 1
                const int k = sing ? n - 1 : n + 1;
                auto at = [&](int mm) -> cd { return k >= 0 && mm <= k && -mm <= k ? ldc(c + nmi(k, mm)) : cd{0, 0}; };
                a[0] = cmac(a[0], q1, at(m));
                a[1] = cmac(a[1], q1, at(m + 1));
                a[2] = cmac(a[2], q1, at(m - 1));
                b[0] = cmac(b[0], q1, at(-m));
                b[1] = cmac(b[1], q1, at(-m + 1));
                b[2] = cmac(b[2], q1, at(-m - 1));
            } else if (GRAD) {
                cd t = F[(n + 1) * 32] * q1;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    a[k] = cmac(a[k], t, ldc(dc + k * dstride + nmi(n, m)));
                    b[k] = cmac(b[k], t, ldc(dc + k * dstride + nmi(n, -m)));
                }
                a[3] = cmac(a[3], t, ldc(c + nmi(n, m)));
                b[3] = cmac(b[3], t, ldc(c + nmi(n, -m)));
            } else {
                cd t = LAP ? q1 : F[n * 32] * q1;
                a[0] = cmac(a[0], t, ldc(c + nmi(n, m)));
                b[0] = cmac(b[0], t, ldc(c + nmi(n, -m)));
            }
            if (n == Q) break;
            double A = __ldg(q.A + nmi(n + 1, m)), B = __ldg(q.B + nmi(n + 1, m));
            cd v = rmac(A * (zeta * q1), -B, w * q2);
            q2 = q1;
            q1 = v;
        }
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            out[k] = cmac(out[k], pp, a[k]);
            if (m > 0) out[k] = cmac(out[k], pm, b[k]);
        }
        pp = pp * sp;
        pm = pm * sm;
    }
}

// One warp per (task, 32 targets): tasks are the leaves (L2P) and then the List-3
// entries. Grid (tasks / warps, target groups, rhs).
template <bool LAP, bool GRAD>
__global__ void __launch_bounds__(kEvalWarps * 32) k_eval3_items(EvalK A) {
    extern __shared__ cd sm[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, rhs = blockIdx.z;
    const int task = blockIdx.x * kEvalWarps + wid;
    if (task >= A.ntask) return;
    const bool sing = task >= A.nleaf_tasks;
    int b, s, li;
    int64_t slot;
    if (!sing) {
        li = A.R.leaf0 + task;
        b = s = A.E.leaves[li];
        slot = A.trg.st[b] - A.R.t0;
    } else {
        const int e = task - A.nleaf_tasks;
        li = A.own[e];
        if (li < A.R.leaf0 || li >= A.R.leaf1) return;
        b = A.E.leaves[li];
        s = A.l3[e];
        slot = A.R.nt + (A.ioff[li] - A.ioff[A.R.leaf0]) + (int64_t)(e - A.l3off[b]) * (A.trg.en[b] - A.trg.st[b]);
    }
    const int P = A.E.Plev[A.blevel[s]], t0 = A.trg.st[b], cnt = A.trg.en[b] - t0;
    const int64_t co = (int64_t)rhs * A.E.ncoef + A.E.eoff[s];
    const cd* c = (sing ? A.E.mp : A.E.loc) + co;
    cd* F = sm + (size_t)wid * (A.E.maxP + 2) * 32;
    const cd cen[3] = {{A.cre[3 * s], A.cim[3 * s]}, {A.cre[3 * s + 1], A.cim[3 * s + 1]},
                       {A.cre[3 * s + 2], A.cim[3 * s + 2]}};
    for (int k0 = blockIdx.y * 32; k0 < cnt; k0 += gridDim.y * 32) {
        const int nt = min(32, cnt - k0), G = min(32 / nt, P + 1), g = lane / nt, t = lane - g * nt;
        const bool on = g < G;
        const int64_t i = A.trg.at(t0 + k0 + t);
        cd x[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) x[a] = cd{A.xr[a * A.n + i], A.xi[a * A.n + i]} - cen[a];
        cd xp = x[0] + mul_i(x[1]), xm = x[0] - mul_i(x[1]), zeta = x[2];
        cd w = xp * xm + zeta * zeta, ir = {1, 0};
        if (LAP) {
            xm = -xm;
            if (sing) {
                ir = cinv(csqrt_p(w));
                w = cinv(w);
                xp = xp * w;
                xm = xm * w;
                zeta = zeta * w;
            }
        } else {
            __syncwarp();
            if (g == 0) radial_rows(sing, A.E.kappa, w, GRAD ? P + 1 : P, F + t);
            __syncwarp();
        }
        constexpr int NS = !GRAD ? 1 : LAP ? 3 : 4;
        cd o[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) o[k] = cd{0, 0};
        if (on)
            eval_columns<LAP, GRAD>(LAP ? (sing ? A.T.T : A.T.U) : A.T.Z, sing, zeta, w, xp, xm, P, F + t, c,
                                    GRAD && !LAP ? A.gco + (sing ? 0 : A.E.ncoef) + (int64_t)rhs * 6 * A.E.ncoef + A.E.eoff[s]
                                                 : nullptr,
                                    2 * A.E.ncoef, g, G, o);
        // the groups' sums in order
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            cd sum = o[k];
            for (int j = 1; j < G; ++j) {
                double px = __shfl_sync(0xffffffffu, o[k].x, min(31, t + j * nt));
                double py = __shfl_sync(0xffffffffu, o[k].y, min(31, t + j * nt));
                sum += cd{px, py};
            }
            o[k] = sum;
        }
        if (lane >= nt) continue;
        cd* v = A.val + (int64_t)rhs * (GRAD ? 3 : 1) * A.nslot + slot + k0 + t;
        if (!GRAD) {
            v[0] = LAP ? ir * o[0] : o[0];
        } else if (LAP) {
            // dz U_n = U_{n-1}, d+ U_n^m = -U_{n-1}^{m-1}/2, d- U_n^m = U_{n-1}^{m+1}/2; dz T has the other sign
            cd dz = ir * o[0], dp = -0.5 * (ir * o[1]), dm = 0.5 * (ir * o[2]);
            v[0] = dp + dm;
            v[A.nslot] = mul_i(dp - dm);
            v[2 * A.nslot] = sing ? -dz : dz;
        } else {
            const double k = A.E.kappa;
            v[0] = o[1] + o[2] - k * (x[0] * o[3]);
            v[A.nslot] = mul_i(o[1] - o[2]) - k * (x[1] * o[3]);
            v[2 * A.nslot] = o[0] - k * (x[2] * o[3]);
        }
    }
}

// Derived coefficients of the Helmholtz gradient, one block per box of [lo, lo + grid):
// dz_n^m = g3(n+1,m) c_{n+1}^m, dp_n^m = -gp(n+1,m+1) c_{n+1}^{m+1}, dm_n^m =
// gm(n+1,m-1) c_{n+1}^{m-1} (0 for n = P), for the multipole (x) and local expansion;
// out [rhs][3][2][ncoef]
__global__ void k_grad_coef(EvalK A, int lo, cd* __restrict__ out) {
    const int b = lo + blockIdx.x, rhs = blockIdx.y, kind = blockIdx.z, P = A.E.Plev[A.blevel[b]];
    const cd* c = (kind ? A.E.loc : A.E.mp) + (int64_t)rhs * A.E.ncoef + A.E.eoff[b];
    cd* o = out + (int64_t)rhs * 6 * A.E.ncoef + kind * A.E.ncoef + A.E.eoff[b];
    const int64_t st = 2 * A.E.ncoef;
    for (int k = threadIdx.x; k < (P + 1) * (P + 1); k += blockDim.x) {
        int n = (int)sqrtf((float)k);
        while (n * n > k) --n;
        while ((n + 1) * (n + 1) <= k) ++n;
        const int m = k - n * n - n, n1 = n + 1;
        const bool in = n1 <= P;
        auto at = [&](const double* f, int mm) -> cd {
            return in && mm <= n1 && -mm <= n1 ? __ldg(f + nmi(n1, mm)) * c[nmi(n1, mm)] : cd{0, 0};
        };
        o[k] = at(A.T.g3, m);
        o[st + k] = -at(A.T.gp, m + 1);
        o[2 * st + k] = at(A.T.gm, m - 1);
    }
}

__global__ void k_eval3_own(int nleaf, const int* __restrict__ leaves, const int* __restrict__ l3off,
                            int* __restrict__ own) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nleaf) return;
    int b = leaves[i];
    for (int e = l3off[b]; e < l3off[b + 1]; ++e) own[e] = i;
}

// u [rhs][comp][n] += the slots of each target: L2P and its leaf's List 3 in order
__global__ void k_eval3_sum(EvalK A, int ncomp, cd* __restrict__ u) {
    const int li = A.R.leaf0 + blockIdx.x, row = blockIdx.y, b = A.E.leaves[li];
    const int t0 = A.trg.st[b], cnt = A.trg.en[b] - t0, ne = A.l3off[b + 1] - A.l3off[b];
    if (!A.l2p && ne == 0) return;
    const cd* v = A.val + (int64_t)row * A.nslot;
    const int64_t l0 = t0 - A.R.t0, first = A.R.nt + (A.ioff[li] - A.ioff[A.R.leaf0]);
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        cd s = A.l2p ? v[l0 + t] : cd{0, 0};
        for (int e = 0; e < ne; ++e) s += v[first + (int64_t)e * cnt + t];
        u[(int64_t)row * A.n + A.trg.at(t0 + t)] += s;
    }
}

// ---------------------------------------------------------------------------
// P2M and P2L, single and double layer. With the harmonics H_n^mu = F_n xi^|mu| q_n
// of the source's offset y, the expansions need four sums over the sources, each
// over all (n, mu):
//   W = sum s F_n Z - k t (y.nu) F_{n+1} Z   (Laplace sum s H),
//   C3, C+, C- = sum t n3 G, t nu+ G, t nu- G,  G = F_{n+1} Z (Laplace H),
// from which (mu = -m)
//   Helmholtz    M_n^m = ik(2n+1) [W_n^mu + g3 C3_{n-1}^mu - gp C+_{n-1}^{mu-1} + gm C-_{n-1}^{mu+1}]
//   Laplace P2M  M_n^m = (-1)^m [W_n^mu + C3_{n-1}^mu - C+_{n-1}^{mu-1}/2 + C-_{n-1}^{mu+1}/2]
//   Laplace P2L  L_n^m = (-1)^m [W_n^mu - C3_{n+1}^mu - C+_{n+1}^{mu-1}/2 + C-_{n+1}^{mu+1}/2]
// (g3, gp, gm the tables of the gradient): the double layer's derivative costs three
// products a coefficient once per box instead of per source, and a source 4 FP64
// instructions per sum and coefficient beside its own harmonics, which +-m share.
// The FP64 pipe bounds it: 32 instructions per (n, m >= 0) pair and source for a single
// layer. Sum over the leaves, before -> after: 1e5-point 3D Helmholtz single layer,
// orders 23 and 36, 5.8 -> 3.6 ms; 3e4 points 1.2 -> 0.76 ms; 2e5-point 3D Laplace
// single and double layer, order 16, 12.1 -> 3.6 ms.
//
// A block per box. The sources (of the whole List 4) come in groups of 32 (or 8), whose
// offsets, radial functions and weights one warp computes, and in chunks of `cs` of
// them: first the harmonics (a warp takes cs sources and 32 / cs columns m), then the
// sums (thread = sum and (n, mu), consecutive lanes on consecutive entries of a
// source's table). Where the sums do not fit in shared memory together (a double
// layer at orders above 38, Laplace 46 for P2M and 45 for P2L), each product is a pass of
// its own.
// ---------------------------------------------------------------------------
constexpr int kP2xThreads = 256;
constexpr size_t kP2xSmem = 220 * 1024;

struct P2xK {
    const double *xr, *xi, *nr, *ni;
    int64_t n;
    const cd *sigma, *tau;        // nullptr: no such layer
    int64_t dstride;
    const int* boxes;
    const int *loff, *lent;       // List 4 (P2L) or nullptr (P2M)
    SubRange src;
    const int *Plev, *blevel;
    const double *cre, *cim;
    const int64_t* eoff;
    int64_t ncoef;
    double kappa;
    Eval3Tables T;
    int cs, gs;                   // sources of a chunk and of a group
    bool all;                     // all sums in one pass, or one product a pass
    cd* out;
};

// order of the harmonics
__host__ __device__ inline int p2x_order(bool lap, bool sing, bool dlp, int P) { return lap && sing && dlp ? P + 1 : P; }

template <bool LAP>
__global__ void __launch_bounds__(kP2xThreads) k_p2x3(P2xK A) {
    extern __shared__ cd sm[];
    const int b = A.boxes[blockIdx.x], rhs = blockIdx.y, P = A.Plev[A.blevel[b]];
    const bool sing = A.loff != nullptr, slp = A.sigma != nullptr, dlp = A.tau != nullptr;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int qb = sing ? A.loff[b] : 0, qe = sing ? A.loff[b + 1] : 1;
    if (sing) {
        int q = qb;
        while (q < qe && A.src.st[A.lent[q]] == A.src.en[A.lent[q]]) ++q;
        if (q == qe) return;
    }
    const int Q = p2x_order(LAP, sing, dlp, P), KQ = (Q + 1) * (Q + 1), cs = A.cs;
    const bool both = !LAP && dlp && A.all;
    const int nsum = dlp && A.all ? 4 : 1, gs = A.gs;
    cd* acc = sm;                                       // [nsum][KQ]
    cd* Y0 = acc + nsum * KQ;                           // [cs][KQ] F_n Z (Laplace H)
    cd* Y1 = Y0 + (both ? (size_t)cs * KQ : 0);         // [cs][KQ] F_{n+1} Z (Helmholtz double layer)
    cd* F = Y1 + (size_t)cs * KQ;                       // Helmholtz [P + 2][gs]
    cd* geo = F + (LAP ? 0 : (size_t)(P + 2) * gs);     // [5][32]: x+, x-, zeta, w, radial factor
    cd* wt = geo + 5 * 32;                              // [32][5]: s, -k t (y.nu), t n3, t nu+, t nu-
    const QTables& q = LAP ? (sing ? A.T.T : A.T.U) : A.T.Z;
    cd* o = A.out + (int64_t)rhs * A.ncoef + A.eoff[b];
    // the columns of a warp: the four schedulers of an SM get equal shares
    const int per = 32 / cs, src = lane & (cs - 1), col = (wid < 4 ? wid : 11 - wid) * per + lane / cs;
    // products of a weight and a table: s F_n Z and -k t (y.nu) F_{n+1} Z into W, the
    // others into C3, C+, C-
    const int p0 = slp ? 0 : LAP ? 2 : 1, p1 = dlp ? 5 : 1;
    for (int pass = p0; pass < p1; pass += A.all ? 5 : LAP && pass == 0 ? 2 : 1) {
    const int off = !LAP && !both && pass > 0 ? 1 : 0;  // F_{n+1} in the one table
    __syncthreads();
    for (int i = threadIdx.x; i < nsum * KQ; i += kP2xThreads) acc[i] = cd{0, 0};
    int qn = qb, j0 = 0;
    while (qn < qe) {
        // the lane's source of the next 32, and where these end
        int64_t j = -1;
        int gn = 0;
        while (qn < qe && gn < gs) {
            const int box = sing ? A.lent[qn] : b;
            const int k0 = A.src.st[box] + j0, m = min(A.src.en[box] - k0, gs - gn);
            if (lane >= gn && lane < gn + m) j = A.src.at(k0 + (lane - gn));
            gn += m;
            if (k0 + m == A.src.en[box]) {
                ++qn;
                j0 = 0;
            } else {
                j0 += m;
            }
        }
        __syncthreads();                                // the last group has been used
        if (wid == 0 && j >= 0) {
            cd y[3];
            for (int a = 0; a < 3; ++a)
                y[a] = cd{A.xr[a * A.n + j], A.xi[a * A.n + j]} - cd{A.cre[3 * b + a], A.cim[3 * b + a]};
            cd xp = y[0] + mul_i(y[1]), xm = y[0] - mul_i(y[1]), zeta = y[2], w = xp * xm + zeta * zeta, f0 = {1, 0};
            if (LAP) {
                xm = -xm;
                if (sing) {
                    f0 = crcp_general(csqrt_p(w));
                    w = crcp_general(w);
                    xp = xp * w;
                    xm = xm * w;
                    zeta = zeta * w;
                }
            } else {
                radial_rows(sing, A.kappa, w, P + 1, F + lane, gs);
            }
            geo[lane] = xp;
            geo[32 + lane] = xm;
            geo[64 + lane] = zeta;
            geo[96 + lane] = w;
            geo[128 + lane] = f0;
            cd* v = wt + 5 * lane;
            v[0] = slp ? A.sigma[(int64_t)rhs * A.dstride + j] : cd{0, 0};
            if (dlp) {
                cd t = A.tau[(int64_t)rhs * A.dstride + j], nn[3];
                for (int a = 0; a < 3; ++a) nn[a] = cd{A.nr[a * A.n + j], A.ni[a * A.n + j]};
                v[1] = (-A.kappa) * ((y[0] * nn[0] + y[1] * nn[1] + y[2] * nn[2]) * t);
                v[2] = nn[2] * t;
                v[3] = (nn[0] + mul_i(nn[1])) * t;
                v[4] = (nn[0] - mul_i(nn[1])) * t;
            }
        }
        for (int g0 = 0; g0 < gn; g0 += cs) {
            const int cn = min(cs, gn - g0), s = g0 + src;
            __syncthreads();                            // group ready, last chunk summed
            if (src < cn) {
                const cd xp = geo[s], xm = geo[32 + s], zeta = geo[64 + s], w = geo[96 + s], f0 = geo[128 + s];
                cd *y0 = Y0 + (size_t)src * KQ, *y1 = Y1 + (size_t)src * KQ;
                for (int m = col; m <= Q; m += kP2xThreads / cs) {
                    cd pp = f0, pm = f0, bp = xp, bm = xm;
                    for (int e = m; e; e >>= 1) {
                        if (e & 1) {
                            pp = pp * bp;
                            pm = pm * bm;
                        }
                        if (e > 1) {
                            bp = bp * bp;
                            bm = bm * bm;
                        }
                    }
                    cd q2 = {0, 0}, q1 = {__ldg(q.D + m), 0};
                    for (int n = m; n <= Q; ++n) {
                        cd t = LAP ? q1 : F[(n + off) * gs + s] * q1;
                        y0[nmi(n, m)] = t * pp;
                        if (m) y0[nmi(n, -m)] = t * pm;
                        if (both) {
                            t = F[(n + 1) * gs + s] * q1;
                            y1[nmi(n, m)] = t * pp;
                            if (m) y1[nmi(n, -m)] = t * pm;
                        }
                        if (n == Q) break;
                        cd v = rmac(__ldg(q.A + nmi(n + 1, m)) * (zeta * q1), -__ldg(q.B + nmi(n + 1, m)), w * q2);
                        q2 = q1;
                        q1 = v;
                    }
                }
            }
            __syncthreads();
            const cd* wc = wt + 5 * g0;
            for (int i = threadIdx.x; i < nsum * KQ; i += kP2xThreads) {
                const int sum = i / KQ, k = i - sum * KQ;
                cd a = acc[i];
                if (!A.all) {
                    for (int s2 = 0; s2 < cn; ++s2) a = cmac(a, wc[5 * s2 + pass], Y0[(size_t)s2 * KQ + k]);
                } else if (sum == 0) {
                    if (slp)
                        for (int s2 = 0; s2 < cn; ++s2) a = cmac(a, wc[5 * s2], Y0[(size_t)s2 * KQ + k]);
                    if (both)
                        for (int s2 = 0; s2 < cn; ++s2) a = cmac(a, wc[5 * s2 + 1], Y1[(size_t)s2 * KQ + k]);
                } else {
                    const cd* Y = LAP ? Y0 : Y1;
                    for (int s2 = 0; s2 < cn; ++s2) a = cmac(a, wc[5 * s2 + 1 + sum], Y[(size_t)s2 * KQ + k]);
                }
                acc[i] = a;
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (P + 1) * (P + 1); k += kP2xThreads) {
        int n = (int)sqrtf((float)k);
        while (n * n > k) --n;
        while ((n + 1) * (n + 1) <= k) ++n;
        const int m = k - n * n - n, mu = -m, nn = LAP && sing ? n + 1 : n - 1;
        auto at = [&](int sum, int mm) -> cd {
            const int nx = sum ? nn : n;
            if (!A.all && sum != max(pass - 1, 0)) return cd{0, 0};
            if (nx < 0 || mm > nx || -mm > nx) return cd{0, 0};
            return acc[(A.all ? sum * KQ : 0) + nmi(nx, mm)];
        };
        cd v = at(0, mu);
        if (dlp) {
            const double g3 = LAP ? (sing ? -1.0 : 1.0) : __ldg(A.T.g3 + nmi(n, mu));
            const double gp = LAP ? 0.5 : __ldg(A.T.gp + nmi(n, mu)), gm = LAP ? 0.5 : __ldg(A.T.gm + nmi(n, mu));
            v += g3 * at(1, mu) - gp * at(2, mu - 1) + gm * at(3, mu + 1);
        }
        if (LAP) v = (m & 1) ? -v : v;
        else v = mul_i(A.kappa * (2.0 * n + 1.0) * v);
        o[k] = sing || pass > p0 ? o[k] + v : v;
    }
    }
}

// shared memory of k_eval3_items, Helmholtz
constexpr size_t items_bytes(int maxP) { return sizeof(cd) * kEvalWarps * (size_t)(maxP + 2) * 32; }

template <bool LAP, bool GRAD>
void launch_items(EvalK A, cudaStream_t st, int nrhs, int groups) {
    const size_t smem = LAP ? 0 : items_bytes(A.E.maxP);
    if (A.ntask <= 0) return;
    dim3 g((unsigned)((A.ntask + kEvalWarps - 1) / kEvalWarps), groups, nrhs);
    k_eval3_items<LAP, GRAD><<<g, kEvalWarps * 32, smem, st>>>(A);
    CFMM_LAUNCHED();
}

}  // namespace

void init_eval3d() {
    for (auto f : {(const void*)k_eval3_items<false, false>, (const void*)k_eval3_items<false, true>})
        CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)items_bytes(kMaxP3Top)));
    for (auto f : {(const void*)k_p2x3<true>, (const void*)k_p2x3<false>})
        CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kP2xSmem));
}

void eval3_qtable(int kind, int N, double* A, double* B, double* D) {
    double d = 1.0;
    for (int m = 0; m <= N; ++m) {
        if (m > 0) d *= kind == 0 ? -std::sqrt((2.0 * m - 1.0) / (2.0 * m)) : kind == 1 ? -0.5 / m : -(2.0 * m - 1.0);
        D[m] = d;
        for (int n = m; n <= N; ++n) {
            double& a = A[nmi(n, m)];
            double& b = B[nmi(n, m)];
            a = b = 0.0;
            if (n == m) continue;
            double nn = (double)(n - m) * (n + m);
            a = kind == 0 ? (2.0 * n - 1.0) / std::sqrt(nn) : kind == 1 ? (2.0 * n - 1.0) / nn : 2.0 * n - 1.0;
            if (n >= m + 2)
                b = kind == 0 ? std::sqrt((double)(n - m - 1) * (n + m - 1) / nn) : kind == 1 ? 1.0 / nn
                                                                                   : (double)(n - 1) * (n - 1) - (double)m * m;
        }
    }
}

void eval3_build(Eval3* E, const std::vector<int>& leaves, const std::vector<int>& l3off, const std::vector<int>& st,
                 const std::vector<int>& en, const int* d_leaves, const int* d_l3off, cudaStream_t stream) {
    std::vector<int64_t> off(leaves.size() + 1, 0);
    for (size_t i = 0; i < leaves.size(); ++i) {
        int b = leaves[i];
        off[i + 1] = off[i] + (int64_t)(l3off[b + 1] - l3off[b]) * (en[b] - st[b]);
    }
    // leaves in Morton order: a range's targets are one interval
    for (size_t i = 0; i < leaves.size();) {
        EvalRange R{(int)i, (int)i, st[leaves[i]], 0, 0};
        for (; i < leaves.size(); ++i) {
            CFMM_REQUIRE(i == 0 || st[leaves[i]] >= en[leaves[i - 1]], CFMM_ECUDA, "leaves out of Morton order");
            const int64_t nt = en[leaves[i]] - R.t0, slots = nt + off[i + 1] - off[R.leaf0];
            if (slots > kEvalSlots && R.leaf1 > R.leaf0) break;
            R.leaf1 = (int)i + 1;
            R.nt = nt;
            R.slots = slots;
        }
        E->max_slots = std::max(E->max_slots, R.slots);
        E->ranges.push_back(R);
    }
    E->ioff.alloc(off.size());
    upload(E->ioff.get(), off.data(), sizeof(int64_t) * off.size(), stream);
    if (l3off.back() == 0) return;
    E->own.alloc(l3off.back());
    k_eval3_own<<<((int)leaves.size() + 127) / 128, 128, 0, stream>>>((int)leaves.size(), d_leaves, d_l3off, E->own.get());
    CFMM_LAUNCHED();
}

bool p2x3_apply(cfmm_plan_s* P, const Eval3Tables& T, const P2x3Args& A, const cd* sigma, const cd* tau, int64_t dstride,
                cd* out, int nrhs) {
    if (A.cnt <= 0) return true;
    TreeDev& Tr = P->tree;
    const bool lap = A.kappa == 0.0, dlp = tau != nullptr;
    const int Q = p2x_order(lap, A.sing, dlp, A.P);
    const size_t KQ = (size_t)(Q + 1) * (Q + 1);
    P2xK K{P->xr.get(), P->xi.get(), P->nr.get(), P->ni.get(), P->n, sigma, tau, dstride, A.boxes,
           A.sing ? Tr.loff[3].get() : nullptr, A.sing ? Tr.lent[3].get() : nullptr, source_range(P), A.Plev,
           Tr.level.get(), Tr.cen_re.get(), Tr.cen_im.get(), A.eoff, A.ncoef, A.kappa, T, 0, 32, true, out};
    auto bytes = [&](bool all, int cs, int gs) {
        return sizeof(cd) * ((all && dlp ? 4 : 1) * KQ + cs * (all && dlp && !lap ? 2 : 1) * KQ +
                             (lap ? 0 : (size_t)(A.P + 2) * gs) + 10 * 32);
    };
    auto fit = [&](size_t limit, bool all, int gs, int least) {
        for (int cs = gs; cs >= least && !K.cs; cs /= 2)
            if (bytes(all, cs, gs) <= limit) {
                K.cs = cs;
                K.gs = gs;
                K.all = all;
            }
    };
    // the largest chunk that leaves two blocks an SM, or one; a product a pass where
    // the sums leave no room for two sources; the least that any order needs
    fit(kP2xSmem / 2, true, 32, 4);
    fit(kP2xSmem, true, 32, 2);
    fit(kP2xSmem, false, 32, 2);
    fit(kP2xSmem, !dlp, 8, 1);
    if (!K.cs) return false;
    const size_t smem = bytes(K.all, K.cs, K.gs);
    dim3 g(A.cnt, nrhs);
    if (lap) k_p2x3<true><<<g, kP2xThreads, smem, P->stream>>>(K);
    else k_p2x3<false><<<g, kP2xThreads, smem, P->stream>>>(K);
    CFMM_LAUNCHED();
    return true;
}

void eval3_apply(cfmm_plan_s* P, Eval3* E, const Eval3Tables& T, const Eval3Args& A, bool l2p, cd* u, cd* g, int nrhs) {
    TreeDev& Tr = P->tree;
    cudaStream_t st = P->stream;
    if (A.nleaf == 0) return;
    const bool lap = A.kappa == 0.0;
    const int nl3 = Tr.hloff[2].back();
    EvalK K{P->xr.get(), P->xi.get(), P->n, A, target_range(P), Tr.loff[2].get(), Tr.lent[2].get(),
            Tr.level.get(), Tr.cen_re.get(), Tr.cen_im.get(), E->ioff.get(), E->own.get(), EvalRange{}, 0, 0, T, nullptr,
            nullptr, 0, 0};
    const int groups = std::max(1, std::min(64, (P->leaf_size + 31) / 32));
    const bool pot = u && (l2p || nl3 > 0);
    // right-hand sides whose slots fit (a range of one leaf may hold more on its own)
    const int ncomp = g ? 3 : 1;
    const int64_t per = std::max<int64_t>(1, std::max(E->max_slots * ncomp, g && !lap ? 6 * A.ncoef : 0));
    const int batch = (int)std::max<int64_t>(1, std::min<int64_t>(nrhs, kEvalItems / per));
    if (pot) E->val.alloc((size_t)batch * E->max_slots);
    if (g) E->gval.alloc((size_t)batch * 3 * E->max_slots);
    if (g && !lap) E->gco.alloc((size_t)6 * A.ncoef * batch);
    for (int r = 0; r < nrhs; r += batch) {
        const int nr = std::min(batch, nrhs - r);
        K.E.mp = A.mp + (int64_t)r * A.ncoef;
        K.E.loc = A.loc + (int64_t)r * A.ncoef;
        if (g && !lap) {
            const int lo = Tr.level_off[Tr.l0];
            k_grad_coef<<<dim3(Tr.nboxes - lo, nr, 2), 128, 0, st>>>(K, lo, E->gco.get());
            CFMM_LAUNCHED();
            K.gco = E->gco.get();
        }
        for (const EvalRange& R : E->ranges) {
            const int nl = R.leaf1 - R.leaf0;
            K.R = R;
            K.nslot = R.slots;
            if (pot) {
                K.val = E->val.get();
                K.l2p = l2p ? 1 : 0;
                K.nleaf_tasks = l2p ? nl : 0;
                K.ntask = K.nleaf_tasks + nl3;
                if (lap) launch_items<true, false>(K, st, nr, groups);
                else launch_items<false, false>(K, st, nr, groups);
                k_eval3_sum<<<dim3(nl, nr), 64, 0, st>>>(K, 1, u + (int64_t)r * P->n);
                CFMM_LAUNCHED();
            }
            if (!g) continue;
            K.val = E->gval.get();
            K.l2p = 1;
            K.nleaf_tasks = nl;
            K.ntask = K.nleaf_tasks + nl3;
            if (lap) launch_items<true, true>(K, st, nr, groups);
            else launch_items<false, true>(K, st, nr, groups);
            k_eval3_sum<<<dim3(nl, 3 * nr), 64, 0, st>>>(K, 3, g + (int64_t)r * 3 * P->n);
            CFMM_LAUNCHED();
        }
    }
}

}  // namespace cfmm

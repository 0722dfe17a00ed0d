// 3D complex-coordinate Helmholtz FMM: expansions and translations (Sec. 5.3,
// Sec. 6.4), FP64.
//
// Expansion functions of a complex 3-vector x (x+ = x1 + i x2, x- = x1 - i x2,
// x3, rho^2 = x.x, rho the principal root; no angle is formed):
//   Z_n^m(x) = rho^n Y_n^m, Y the Schmidt semi-normalised harmonics of Sec. 3.2,
//     Z_0^0 = 1,  Z_m^m = -x+ sqrt((2m-1)/(2m)) Z_{m-1}^{m-1},  Z_{m+1}^m = sqrt(2m+1) x3 Z_m^m,
//     Z_n^m = A_n^m x3 Z_{n-1}^m - B_n^m rho^2 Z_{n-2}^m,
//     A_n^m = (2n-1)/sqrt((n-m)(n+m)),  B_n^m = sqrt((n-m-1)(n+m-1)/((n-m)(n+m))),
//     Z_n^{-m} = Z_n^m with x+ and x- exchanged;
//   R_n^m = j_n(k rho) rho^-n Z_n^m (entire),  S_n^m = h_n(k rho) rho^-n Z_n^m.
// Gegenbauer's addition theorem with Eq. sphaddition gives, for the
// constant-free kernel e^{ik r}/r = ik h_0(kr),
//   e^{ik|x-y|}/|x-y| = ik sum (2n+1) R_n^{-m}(y) S_n^m(x),
// hence (Thms 5.3.1, 5.3.2)
//   P2M  M_n^m = ik(2n+1) sum_j s_j R_n^{-m}(y_j - c)     M2P  u = sum M_n^m S_n^m(x - c)
//   P2L  L_n^m = ik(2n+1) sum_j s_j S_n^{-m}(y_j - c)     L2P  u = sum L_n^m R_n^m(x - c)
// and the double layer differentiates the source side along the normal:
//   grad(f_n rho^-n Z) = f_n rho^-n grad Z - k f_{n+1} rho^-(n+1) Z x,
//   n.grad Z_n^m = n3 c3 Z_{n-1}^m - nu+ s+ c+ Z_{n-1}^{m-1} + nu- s- c- Z_{n-1}^{m+1},
//   c3 = sqrt((n-m)(n+m)), c+ = sqrt((n+m)(n+m-1))/2, c- = sqrt((n-m)(n-m-1))/2,
//   s+ = 1 (m >= 1) else -1, s- = 1 (m >= 0) else -1, nu+- = n1 +- i n2.
//
// Translations by a complex shift d = c_new - c_old ("point and shoot",
// Sec. 5.3 translation operators):
//   1. rotate to the z-axis. e = (d1 + i d2)/s, s = sqrt(d1^2 + d2^2) (e = 1 if
//      s^2 = 0); t = sqrt(d.d); e_a = (d3 + i s)/t. The complex rotation
//      x' = R_y(a) R_z(-b) x carries d to (0, 0, t) and maps coefficients by
//        c' = Phi^-1 D^T E(e_a) D Phi E(e) c,   Phi = diag(i^m), E(e) = diag(e^m),
//      with D_n the real (2n+1)x(2n+1) matrix of the fixed rotation
//      x -> R_x(pi/2) x conjugated by Phi: the y-rotation of Eq. mp_y_rot
//      factored into two fixed rotations around a diagonal z-rotation.
//      D is built on the host by projecting onto the equator exactly as
//      Eq. mp_y_rot does (real rotation, so F_n is a trigonometric polynomial
//      and 2n+1 samples are exact);
//   2. re-expand along z with the exact coaxial coefficients
//        W_{n'}^m(x + t e3) = sum_n T^m_{n n'}(t) V_n^m(x)
//      (W = S, V = R for M2L, f = h; W = V = R or S, f = j for L2L and M2M),
//      generated per shift by the recurrences that follow from
//        d3 W_n^m = k(alpha_n^m W_{n-1}^m - beta_n^m W_{n+1}^m),
//        d- W_n^m = k(mu_n^m W_{n-1}^{m+1} + nu_n^m W_{n+1}^{m+1})  (m >= 0),
//        alpha = sqrt((n-m)(n+m))/(2n+1), beta = sqrt((n+1-m)(n+1+m))/(2n+1),
//        mu = sqrt((n-m)(n-m-1))/(2(2n+1)), nu = sqrt((n+m+1)(n+m+2))/(2(2n+1)):
//        T^0_{n,0} = (2n+1)(-1)^n f_n(kt),
//        T^m_{n,m} = [mu_{n+1}^{m-1} T^{m-1}_{n+1,m-1} + nu_{n-1}^{m-1} T^{m-1}_{n-1,m-1}] / nu_{m-1}^{m-1},
//        T_{n,n'+1} = [alpha_{n'} T_{n,n'-1} - alpha_{n+1} T_{n+1,n'} + beta_{n-1} T_{n-1,n'}] / beta_{n'},
//      the last only for n > n' (the stable direction); the rest from
//        T_{n',n} = (2n'+1)/(2n+1) (-1)^{n+n'} T_{n,n'},   T^{-m} = T^m.
//      These are the translations the paper's projection step approximates
//      (its Gauss-Legendre projection recovers T up to aliasing);
//   3. rotate back: c = E(1/e) Phi^-1 D^T E(1/e_a) D Phi c'.
#include <algorithm>
#include <cmath>
#include <map>
#include <memory>
#include <mutex>

#include "cfmm_special.cuh"
#include "eval3d.cuh"
#include "kernels.cuh"
#include "pairs3d.cuh"

namespace cfmm {

namespace {

__host__ __device__ __forceinline__ int nmi(int n, int m) { return n * n + n + m; }

constexpr int kH3MaxP = kMaxP3Top;   // expansion order limit of this path
constexpr int kH3Smem = 220 * 1024;  // dynamic shared memory ceiling per block

// ---------------------------------------------------------------------------
// Per-device tables shared by all plans: D_n (row-major, n <= Pmax), the Z
// recurrence coefficients and the coaxial recurrence coefficients.
// ---------------------------------------------------------------------------
struct H3Tables {
    int Pmax = -1;
    DevBuf<double> Dh;       // D_n[m][m'] for m, m' >= 0, column-major per order
    DevBuf<double> Dg;       // the same scaled by (-1)^n/(2n+1)
    DevBuf<int64_t> Dhoff;   // [Pmax+2]
    DevBuf<double> al, be, ab, cg, smu, snu;   // coaxial recurrence coefficients (see Tr3Tables)
    DevBuf<double> g3, gp, gm;           // gradient coefficients c3, s+ c+, s- c- by nmi(n, m), all m
    DevBuf<int> knm;         // k -> n * 256 + (m + 128), k < (Pmax+1)^2
    DevBuf<double> lsm, lsd; // eps_m s_n^m and eps_m / s_n^m, s = sqrt((n-|m|)! (n+|m|)!)
    DevBuf<double> fact, ifact;  // j! and 1/j!, j <= 2 Pmax + 2
    DevBuf<double> q[3][3];  // A, B, D of Z, U, T (eval3d.cuh), orders <= Pmax + 2
    // FP32, mixed P2M and L2P: Z recurrence by nmi(n, m), m >= 0; sqrt((2m-1)/(2m)), sqrt(2m+1), m <= Pmax+1
    DevBuf<float> zAf, zBf, dgf, s21f;
};

// Tables only grow: a larger order builds a new set and the older sets stay
// alive, since plans that hold them may be running on other streams.
static std::mutex g_tab_mu;
static std::map<int, std::vector<H3Tables*>>& tab_map() {
    static std::map<int, std::vector<H3Tables*>> m;
    return m;
}

// Z_n^m at a complex point (host), n <= P, all m
static void host_ztable(int P, cd x0, cd x1, cd x2, std::vector<cd>& Z) {
    Z.assign((size_t)(P + 1) * (P + 1), cd{0, 0});
    cd xp = x0 + mul_i(x1), xm = x0 - mul_i(x1), z = x2;
    cd r2 = xp * xm + z * z;
    for (int sgn = 0; sgn < 2; ++sgn) {
        cd xs = sgn ? xm : xp;
        cd d = {1, 0};
        for (int m = 0; m <= P; ++m) {
            if (m > 0) d = (-std::sqrt((2.0 * m - 1.0) / (2.0 * m))) * (xs * d);
            if (sgn == 1 && m == 0) continue;
            int mi = sgn ? -m : m;
            Z[nmi(m, mi)] = d;
            if (m + 1 > P) continue;
            cd p2 = d, p1 = std::sqrt(2.0 * m + 1.0) * (z * d);
            Z[nmi(m + 1, mi)] = p1;
            for (int n = m + 2; n <= P; ++n) {
                double A = (2.0 * n - 1.0) / std::sqrt((double)(n - m) * (n + m));
                double B = std::sqrt((double)(n - m - 1) * (n + m - 1) / ((double)(n - m) * (n + m)));
                cd cur = A * (z * p1) - B * (r2 * p2);
                Z[nmi(n, mi)] = cur;
                p2 = p1;
                p1 = cur;
            }
        }
    }
}

// D_n for n <= P (real, row-major by (m + n, m' + n)); see the file comment.
static void host_rotation_tables(int P, std::vector<double>& D, std::vector<int64_t>& off) {
    const double kPi = 3.14159265358979323846;
    off.assign(P + 2, 0);
    for (int n = 0; n <= P; ++n) off[n + 1] = off[n] + (int64_t)(2 * n + 1) * (2 * n + 1);
    D.assign(off[P + 1], 0.0);
    std::vector<cd> Z, ab;
    // a_n^m = Y_n^m(e1), b_n^m = d_theta Y_n^m at (pi/2, 0) = -sqrt((n-m)(n+m)) Z_{n-1}^m(e1)
    host_ztable(P, cd{1, 0}, cd{0, 0}, cd{0, 0}, ab);
    std::vector<cd> F, G;
    for (int n = 0; n <= P; ++n) {
        int N = 2 * n + 1;
        // samples of Z_n^{m'} at p_j = X^T-rotated equator points and their
        // theta-derivative: frame x1 = Q x with Q = R_x(-pi/2)^T, so the
        // samples are taken at Q^T e_j = (cos phi, 0, -sin phi) along
        // Q^T (0, 0, -1) = (0, -1, 0) (v+ = -i, v- = i)
        F.assign((size_t)N * N, cd{0, 0});
        G.assign((size_t)N * N, cd{0, 0});
        for (int j = 0; j < N; ++j) {
            double ph = 2.0 * kPi * j / N;
            host_ztable(n, cd{std::cos(ph), 0}, cd{0, 0}, cd{-std::sin(ph), 0}, Z);
            for (int mp = -n; mp <= n; ++mp) {
                F[(size_t)j * N + (mp + n)] = Z[nmi(n, mp)];
                // grad Z . v = -i d+ Z + i d- Z
                cd g = {0, 0};
                if (n >= 1) {
                    if (std::abs(mp - 1) <= n - 1) {
                        double sp = mp >= 1 ? 1.0 : -1.0;
                        cd dp = (-0.5 * sp * std::sqrt((double)(n + mp) * (n + mp - 1))) * Z[nmi(n - 1, mp - 1)];
                        g = g - mul_i(dp);
                    }
                    if (std::abs(mp + 1) <= n - 1) {
                        double sm = mp >= 0 ? 1.0 : -1.0;
                        cd dm = (0.5 * sm * std::sqrt((double)(n - mp) * (n - mp - 1))) * Z[nmi(n - 1, mp + 1)];
                        g = g + mul_i(dm);
                    }
                }
                G[(size_t)j * N + (mp + n)] = g;
            }
        }
        for (int m = -n; m <= n; ++m) {
            double a = ab[nmi(n, m)].x;
            double b = 0.0;
            if (std::abs(m) <= n - 1) b = -std::sqrt((double)(n - m) * (n + m)) * ab[nmi(n - 1, m)].x;
            double den = a * a + b * b;
            for (int mp = -n; mp <= n; ++mp) {
                cd Fh = {0, 0}, Gh = {0, 0};
                for (int j = 0; j < N; ++j) {
                    double ph = 2.0 * kPi * j / N;
                    cd w = {std::cos(m * ph) / N, -std::sin(m * ph) / N};
                    Fh = Fh + w * F[(size_t)j * N + (mp + n)];
                    Gh = Gh + w * G[(size_t)j * N + (mp + n)];
                }
                cd da = (a * Fh + b * Gh) * (1.0 / den);
                // D = Phi DA Phi^-1: multiply by i^m i^-m'
                int e = ((m - mp) % 4 + 4) % 4;
                cd ph = e == 0 ? cd{1, 0} : e == 1 ? cd{0, 1} : e == 2 ? cd{-1, 0} : cd{0, -1};
                cd v = ph * da;
                CFMM_REQUIRE(std::fabs(v.y) <= 1e-10 * (1.0 + std::fabs(v.x)), CFMM_ECUDA,
                             "3D Helmholtz rotation table is not real");
                D[off[n] + (int64_t)(m + n) * N + (mp + n)] = v.x;
            }
        }
    }
}

static Tr3Tables tr3_tables(const H3Tables* T) {
    return Tr3Tables{T->Dh.get(), T->Dg.get(), T->Dhoff.get(), T->al.get(), T->be.get(), T->ab.get(), T->cg.get(),
                     T->smu.get(), T->snu.get(), T->lsm.get(), T->lsd.get(), T->fact.get(), T->ifact.get()};
}

static Eval3Tables eval3_tables(const H3Tables* T) {
    auto q = [&](int k) { return QTables{T->q[k][0].get(), T->q[k][1].get(), T->q[k][2].get()}; };
    return Eval3Tables{q(0), q(1), q(2), T->g3.get(), T->gp.get(), T->gm.get()};
}

static H3Tables* tables(int P) {
    int dev = 0;
    CFMM_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_tab_mu);
    auto& sets = tab_map()[dev];
    if (!sets.empty() && sets.back()->Pmax >= P) return sets.back();
    auto owned = std::make_unique<H3Tables>();
    H3Tables* T = owned.get();
    int Pm = std::max(P, 16);
    std::vector<double> D;
    std::vector<int64_t> off;
    host_rotation_tables(Pm, D, off);
    int NN = 2 * Pm + 3;
    size_t NT = (size_t)NN * NN;
    std::vector<double> zA(NT, 0.0), zB(NT, 0.0), al(NT, 0.0), be(NT, 0.0), mu(NT, 0.0),
        nu(NT, 0.0), g3(NT, 0.0), gp(NT, 0.0), gm(NT, 0.0), dg(Pm + 2, 0.0), s21(Pm + 2, 0.0);
    for (int n = 0; n < NN; ++n) {
        for (int m = 0; m <= n; ++m) {
            int k = nmi(n, m);
            if (n >= m + 2) {
                zA[k] = (2.0 * n - 1.0) / std::sqrt((double)(n - m) * (n + m));
                zB[k] = std::sqrt((double)(n - m - 1) * (n + m - 1) / ((double)(n - m) * (n + m)));
            }
            al[k] = std::sqrt((double)(n - m) * (n + m)) / (2.0 * n + 1.0);
            be[k] = std::sqrt((double)(n + 1 - m) * (n + 1 + m)) / (2.0 * n + 1.0);
            mu[k] = std::sqrt((double)(n - m) * std::max(n - m - 1, 0)) / (2.0 * (2.0 * n + 1.0));
            nu[k] = std::sqrt((double)(n + m + 1) * (n + m + 2)) / (2.0 * (2.0 * n + 1.0));
        }
        for (int m = -n; m <= n; ++m) {
            int k = nmi(n, m);
            g3[k] = std::sqrt((double)(n - m) * (n + m));
            gp[k] = (m >= 1 ? 0.5 : -0.5) * std::sqrt((double)(n + m) * std::max(n + m - 1, 0));
            gm[k] = (m >= 0 ? 0.5 : -0.5) * std::sqrt((double)(n - m) * std::max(n - m - 1, 0));
        }
    }
    for (int m = 1; m <= Pm + 1; ++m) dg[m] = std::sqrt((2.0 * m - 1.0) / (2.0 * m));
    for (int m = 0; m <= Pm + 1; ++m) s21[m] = std::sqrt(2.0 * m + 1.0);
    std::vector<int> knm((size_t)(Pm + 1) * (Pm + 1));
    for (int n = 0; n <= Pm; ++n)
        for (int m = -n; m <= n; ++m) knm[nmi(n, m)] = n * 256 + (m + 128);
    std::vector<int64_t> hoff(Pm + 2, 0);
    for (int n = 0; n <= Pm; ++n) hoff[n + 1] = hoff[n] + (int64_t)(n + 1) * (n + 1);
    std::vector<double> Dh(hoff[Pm + 1]);
    for (int n = 0; n <= Pm; ++n) {
        int N = 2 * n + 1;
        for (int m = 0; m <= n; ++m)
            for (int mp = 0; mp <= n; ++mp) Dh[hoff[n] + (int64_t)mp * (n + 1) + m] = D[off[n] + (int64_t)(m + n) * N + (mp + n)];
    }
    // products of the coaxial recurrence (see Tr3Tables)
    std::vector<double> ab(NT, 0.0), cg(NT, 0.0), smu(NT, 0.0), snu(NT, 0.0);
    for (int m = 0; m < NN; ++m) {
        double gam = 1.0;
        for (int n = m; n < NN; ++n) {
            cg[nmi(n, m)] = ((n & 1) ? -(2.0 * n + 1.0) : 2.0 * n + 1.0) * gam;
            gam /= be[nmi(n, m)];
            if (n > m) ab[nmi(n, m)] = al[nmi(n, m)] * be[nmi(n - 1, m)];
            if (m > 0 && n + 1 < NN) {
                smu[nmi(n, m)] = mu[nmi(n + 1, m - 1)] / nu[nmi(m - 1, m - 1)];
                snu[nmi(n, m)] = nu[nmi(n - 1, m - 1)] / nu[nmi(m - 1, m - 1)];
            }
        }
    }
    auto up = [](DevBuf<double>& b, const std::vector<double>& v) {
        b.alloc(v.size());
        CFMM_CUDA(cudaMemcpy(b.get(), v.data(), sizeof(double) * v.size(), cudaMemcpyHostToDevice));
    };
    up(T->Dh, Dh);
    for (int n = 0; n <= Pm; ++n)
        for (int64_t k = hoff[n]; k < hoff[n + 1]; ++k) Dh[k] *= ((n & 1) ? -1.0 : 1.0) / (2.0 * n + 1.0);
    up(T->Dg, Dh);
    T->Dhoff.alloc(hoff.size());
    CFMM_CUDA(cudaMemcpy(T->Dhoff.get(), hoff.data(), sizeof(int64_t) * hoff.size(), cudaMemcpyHostToDevice));
    up(T->al, al);
    up(T->be, be);
    up(T->ab, ab);
    up(T->cg, cg);
    up(T->smu, smu);
    up(T->snu, snu);
    up(T->g3, g3);
    up(T->gp, gp);
    up(T->gm, gm);
    {
        std::vector<double> f(2 * Pm + 3), fi(2 * Pm + 3), lm(knm.size()), ld(knm.size());
        f[0] = 1.0;
        for (int j = 1; j < (int)f.size(); ++j) f[j] = f[j - 1] * j;
        for (size_t j = 0; j < f.size(); ++j) fi[j] = 1.0 / f[j];
        for (int n = 0; n <= Pm; ++n)
            for (int m = -n; m <= n; ++m) {
                int am = std::abs(m);
                double sv = std::sqrt(f[n - am] * f[n + am]);
                double e = (m < 0 && (am & 1)) ? -1.0 : 1.0;
                lm[nmi(n, m)] = e * sv;
                ld[nmi(n, m)] = e / sv;
            }
        up(T->fact, f);
        up(T->ifact, fi);
        up(T->lsm, lm);
        up(T->lsd, ld);
    }
    for (int kind = 0; kind < 3; ++kind) {
        int N = Pm + 2;
        std::vector<double> A((size_t)(N + 1) * (N + 1), 0.0), B = A, Dq(N + 1, 0.0);
        eval3_qtable(kind, N, A.data(), B.data(), Dq.data());
        up(T->q[kind][0], A);
        up(T->q[kind][1], B);
        up(T->q[kind][2], Dq);
    }
    T->knm.alloc(knm.size());
    CFMM_CUDA(cudaMemcpy(T->knm.get(), knm.data(), sizeof(int) * knm.size(), cudaMemcpyHostToDevice));
    {
        auto upf = [](DevBuf<float>& b, const std::vector<double>& v) {
            std::vector<float> f(v.begin(), v.end());
            b.alloc(f.size());
            CFMM_CUDA(cudaMemcpy(b.get(), f.data(), sizeof(float) * f.size(), cudaMemcpyHostToDevice));
        };
        upf(T->zAf, zA);
        upf(T->zBf, zB);
        upf(T->dgf, dg);
        upf(T->s21f, s21);
    }
    T->Pmax = Pm;
    sets.push_back(owned.release());
    return T;
}

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void nm_tab(const int* knm, int k, int& n, int& m) {
    int v = __ldg(knm + k);
    n = v >> 8;
    m = (v & 255) - 128;
}

// ---------------------------------------------------------------------------
// L2P in complex64 arithmetic (mixed precision), 3D Helmholtz and Laplace.
//
// With x~ = (x - c)/rho_b (rho_b = sqrt(3)/2 w, the leaf's radius) the local
// expansion is evaluated as
//   Helmholtz  u = sum L^_n^m jh_n(k rho) Z_n^m(x~),  L^ = L_n^m (k rho_b)^n/(2n+1)!!
//   Laplace    u = sum L^_n^m Z_n^m(x~),              L^ = L_n^m lsd_n^m rho_b^n
// (Z_n^m(x) = rho_b^n Z_n^m(x~); U_n^m = lsd_n^m Z_n^m), where
//   jh_n(z) = j_n(z) (2n+1)!!/z^n
// is entire in w = z^2 with jh_n(0) = 1, so every factor stays O(1) in FP32
// at any leaf size. From j_{n-1} + j_{n+1} = (2n+1)/z j_n,
//   jh_{n-1} = jh_n - w jh_{n+1}/((2n+1)(2n+3)),
// and the ratios q_n = jh_n/jh_{n-1} = 1/(1 - w q_{n+1}/((2n+1)(2n+3))) follow
// by Miller's backward recurrence from q = 1 far above P; jh_0 = j_0 comes
// from the plane-wave normalisation exp(-+ i z) = sum (2n+1) (-+ i)^n j_n =
// jh_0 sum (-+ i z)^n/(2n-1)!! prod_{k<=n} q_k (sign with |exp| >= 1, as in
// the FP64 Miller recurrence). The coefficients are formed in FP64 per leaf
// and rounded; each harmonic column is summed in FP32 and the columns in a
// compensated (Kahan) FP32 sum.
// ---------------------------------------------------------------------------
struct L2p3fArgs {
    const double* xr;
    const double* xi;
    int64_t n;
    const int* blevel;
    SubRange pts;                // sources (Exp3hArgs, k_p2m3f) or targets (k_l2p3f)
    const double* cre;
    const double* cim;
    const int* Plev;
    const int64_t* eoff;
    int64_t ncoef;
    double kappa;
    double W;            // root box width
    const float* zA;     // FP32 Z recurrence coefficients by nmi(n, m >= 0)
    const float* zB;
    const float* dg;
    const float* s21;
    const int* knm;
    const double* lsd;   // Laplace: e_m / s_n^m by nmi(n, m)
};

// jh_n(z) = j_n(z) (2n+1)!!/z^n, n = 0..P, in complex64 from w = z^2 (see
// the comment above k_l2p3f): ratios by Miller's backward recurrence from 1,
// jh_0 from the plane-wave normalisation.
__device__ __forceinline__ void jhat_seq(cf w, int P, cf* G) {
    cf zz = csqrtf_p(w);
    float big = fmaxf((float)P, hypotf(zz.x, zz.y));
    int N = (int)big + 12 + (int)sqrtf(8.f * big);
    bool up = zz.y >= 0.f;                           // exp(-i z), |.| >= 1
    cf a = up ? cf{zz.y, -zz.x} : cf{-zz.y, zz.x};   // -+ i z
    cf q = {1.f, 0.f}, H = {1.f, 0.f};
    for (int nn = N; nn >= 1; --nn) {
        float den = 1.f / ((2.f * nn + 1.f) * (2.f * nn + 3.f));
        q = cinvf(cf{1.f, 0.f} - (den * w) * q);
        if (nn <= P) G[nn] = q;
        H = cf{1.f, 0.f} + (1.f / (2.f * nn - 1.f)) * (a * (q * H));
    }
    // jh_0 = exp(a) / H
    float ex = expf(a.x), sn, cs;
    sincosf(a.y, &sn, &cs);
    cf g = cf{ex * cs, ex * sn} * cinvf(H);
    G[0] = g;
    for (int nn = 1; nn <= P; ++nn) {
        g = g * G[nn];
        G[nn] = g;
    }
}

template <bool HELM>
__global__ void __launch_bounds__(128) k_l2p3f(L2p3fArgs A, const int* __restrict__ leaves,
                                                const cd* __restrict__ loc, cd* __restrict__ u) {
    extern __shared__ unsigned char smraw[];
    int b = leaves[blockIdx.x];
    int rhs = blockIdx.y;
    int lev = A.blevel[b];
    int P = A.Plev[lev];
    int nc = (P + 1) * (P + 1);
    double rb = 0.86602540378443864676 * ldexp(A.W, -lev);
    double* scl = reinterpret_cast<double*>(smraw);              // P + 1
    cf* coef = reinterpret_cast<cf*>(scl + (P + 1));             // (P + 1)^2
    if (threadIdx.x == 0) {
        double f = 1.0, g = HELM ? A.kappa * rb : rb;
        for (int n = 0; n <= P; ++n) {
            scl[n] = f;
            f *= HELM ? g / (2.0 * n + 3.0) : g;
        }
    }
    __syncthreads();
    const cd* lc = loc + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        int n, m;
        nm_tab(A.knm, c, n, m);
        double s = scl[n];
        if (!HELM) s *= __ldg(A.lsd + c);
        coef[c] = to_cf(s * lc[c]);
    }
    __syncthreads();
    double irb = 1.0 / rb;
    cd cen[3];
    for (int a = 0; a < 3; ++a) cen[a] = cd{A.cre[3 * b + a], A.cim[3 * b + a]};
    cf G[kH3MaxP + 1];
    for (int k = A.pts.st[b] + threadIdx.x; k < A.pts.en[b]; k += blockDim.x) {
        const int64_t i = A.pts.at(k);
        cf x[3];
        for (int a = 0; a < 3; ++a)
            x[a] = to_cf(irb * (cd{A.xr[a * A.n + i], A.xi[a * A.n + i]} - cen[a]));
        cf xp = x[0] + mul_if(x[1]), xm = x[0] - mul_if(x[1]), z = x[2];
        cf r2 = xp * xm + z * z;
        if (HELM) {
            // w = (k rho)^2 = (k rho_b)^2 x~.x~
            float kr = (float)(A.kappa * rb);
            jhat_seq((kr * kr) * r2, P, G);
        }
        Kahan acc;
        for (int sgn = 0; sgn < 2; ++sgn) {
            cf xs = sgn ? xm : xp;
            cf d = {1.f, 0.f};
            for (int m = 0; m <= P; ++m) {
                if (m > 0) d = (-__ldg(A.dg + m)) * (xs * d);
                if (sgn == 1 && m == 0) continue;
                int mi = sgn ? -m : m;
                cf col = coef[nmi(m, mi)] * (HELM ? G[m] * d : d);
                if (m + 1 <= P) {
                    cf p2 = d, p1 = __ldg(A.s21 + m) * (z * d);
                    col = cmacf(col, coef[nmi(m + 1, mi)], HELM ? G[m + 1] * p1 : p1);
                    for (int n = m + 2; n <= P; ++n) {
                        int k = nmi(n, m);
                        cf cur = __ldg(A.zA + k) * (z * p1) - __ldg(A.zB + k) * (r2 * p2);
                        col = cmacf(col, coef[nmi(n, mi)], HELM ? G[n] * cur : cur);
                        p2 = p1;
                        p1 = cur;
                    }
                }
                acc.add(col);
            }
        }
        u[(int64_t)rhs * A.n + i] += acc.value();
    }
}

// Single-layer P2M in complex64 products (mixed precision), 3D Helmholtz and
// Laplace. With y~ = (y - c)/rho_b,
//   Helmholtz  M_n^m = i k (2n+1) (k rho_b)^n/(2n+1)!! sum s jh_n(k rho) Z_n^{-m}(y~)
//   Laplace    M_n^m = lsd_n^m rho_b^n sum s Z_n^{-m}(y~)
// (scaled as in k_l2p3f). Each warp stages 32
// sources (their jh table, x+, x-, x3 and density) and then takes (source,
// harmonic column) items in rounds of 32, one per lane; a column owns the
// coefficients (n, -mu), n >= |mu|, so with 2P+1 >= 32 columns the lanes of a
// round write disjoint coefficients (fewer columns: one source at a time, a
// lane per column). Products are complex64 and each warp's accumulator row is
// a compensated (Kahan) complex64 sum; the rows are summed in warp order in
// FP64 and scaled in FP64.
constexpr int kP2m3fWarps = 4;

template <bool HELM>
__global__ void __launch_bounds__(kP2m3fWarps * 32) k_p2m3f(L2p3fArgs A, const int* __restrict__ boxes,
                                                             const cd* __restrict__ sigma, int64_t dstride,
                                                             cd* __restrict__ out) {
    extern __shared__ unsigned char smraw[];
    int b = boxes[blockIdx.x];
    int rhs = blockIdx.y;
    int lev = A.blevel[b];
    int P = A.Plev[lev];
    int nc = (P + 1) * (P + 1), C = 2 * P + 1;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4* acc = reinterpret_cast<float4*>(smraw);                         // [nwarp][nc]: sum, compensation
    cf* Gs = reinterpret_cast<cf*>(acc + (size_t)kP2m3fWarps * nc);         // [nwarp][32][P+1]
    cf* Ys = Gs + (size_t)kP2m3fWarps * 32 * (P + 1);                       // [nwarp][32][4]
    float4* accw = acc + (size_t)wid * nc;
    cf* Gw = Gs + (size_t)wid * 32 * (P + 1);
    cf* Yw = Ys + (size_t)wid * 32 * 4;
    for (int c = lane; c < nc; c += 32) accw[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    auto kadd = [&](int k, cf t) {
        float4 a = accw[k];
        float yx = t.x - a.z, tx = a.x + yx;
        float yy = t.y - a.w, ty = a.y + yy;
        accw[k] = make_float4(tx, ty, (tx - a.x) - yx, (ty - a.y) - yy);
    };
    double rb = 0.86602540378443864676 * ldexp(A.W, -lev), irb = 1.0 / rb;
    cd cen[3];
    for (int a = 0; a < 3; ++a) cen[a] = cd{A.cre[3 * b + a], A.cim[3 * b + a]};
    float kr = (float)(A.kappa * rb);
    int s0 = A.pts.st[b], s1 = A.pts.en[b];
    for (int base = s0 + wid * 32; base < s1; base += kP2m3fWarps * 32) {
        int cnt = min(32, s1 - base);
        __syncwarp();
        if (lane < cnt) {
            const int64_t j = A.pts.at(base + lane);
            cf y[3];
            for (int a = 0; a < 3; ++a) y[a] = to_cf(irb * (cd{A.xr[a * A.n + j], A.xi[a * A.n + j]} - cen[a]));
            cf xp = y[0] + mul_if(y[1]), xm = y[0] - mul_if(y[1]);
            Yw[lane * 4 + 0] = xp;
            Yw[lane * 4 + 1] = xm;
            Yw[lane * 4 + 2] = y[2];
            Yw[lane * 4 + 3] = to_cf(sigma[rhs * dstride + j]);
            if (HELM) jhat_seq((kr * kr) * (xp * xm + y[2] * y[2]), P, Gw + lane * (P + 1));
        }
        __syncwarp();
        int items = cnt * C;
        int step = C >= 32 ? 32 : C;
        for (int r0 = 0; r0 < items; r0 += step) {
            int it = r0 + lane;
            if (lane < step && it < items) {
                int js = it / C, col = it - js * C;
                cf xp = Yw[js * 4 + 0], xm = Yw[js * 4 + 1], z = Yw[js * 4 + 2], d = Yw[js * 4 + 3];
                cf r2 = xp * xm + z * z;
                const cf* G = Gw + js * (P + 1);
                int am = col <= P ? col : col - P;
                bool neg = col > P;
                int m = neg ? am : -am;
                cf xs = neg ? xm : xp;
                for (int i = 1; i <= am; ++i) d = (-__ldg(A.dg + i)) * (xs * d);
                kadd(nmi(am, m), HELM ? G[am] * d : d);
                if (am + 1 <= P) {
                    cf p2 = d, p1 = __ldg(A.s21 + am) * (z * d);
                    kadd(nmi(am + 1, m), HELM ? G[am + 1] * p1 : p1);
                    for (int n = am + 2; n <= P; ++n) {
                        int kk = nmi(n, am);
                        cf cur = __ldg(A.zA + kk) * (z * p1) - __ldg(A.zB + kk) * (r2 * p2);
                        kadd(nmi(n, m), HELM ? G[n] * cur : cur);
                        p2 = p1;
                        p1 = cur;
                    }
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    cd* o = out + (int64_t)rhs * A.ncoef + A.eoff[b];
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        cd v = {0.0, 0.0};
        for (int w = 0; w < kP2m3fWarps; ++w) {
            float4 a = acc[(size_t)w * nc + c];
            v += cd{(double)a.x - (double)a.z, (double)a.y - (double)a.w};
        }
        int n, m;
        nm_tab(A.knm, c, n, m);
        double sc = 1.0, g = HELM ? A.kappa * rb : rb;
        for (int j = 1; j <= n; ++j) sc *= HELM ? g / (2.0 * j + 1.0) : g;
        if (HELM) o[c] = mul_i((A.kappa * (2.0 * n + 1.0) * sc) * v);
        else o[c] = (__ldg(A.lsd + c) * sc) * v;
    }
}

// shared memory of k_p2m3f at order P
static size_t p2m3f_smem(int P) {
    size_t nc = (size_t)(P + 1) * (P + 1);
    return sizeof(float4) * kP2m3fWarps * nc + sizeof(cf) * (size_t)kP2m3fWarps * 32 * (P + 1 + 4);
}

static void launch_p2m3f(H3Tables* TB, bool helm, cfmm_plan_s* P, const int* boxes, int cnt, int PL,
                         const int* dPlev, const int64_t* eoff, int64_t ncoef, const cd* sigma, int64_t dstride,
                         cd* out, int nrhs) {
    if (cnt <= 0) return;
    TreeDev& T = P->tree;
    L2p3fArgs A{P->xr.get(), P->xi.get(), P->n, T.level.get(), source_range(P), T.cen_re.get(),
                T.cen_im.get(), dPlev, eoff, ncoef, P->kappa, P->W, TB->zAf.get(), TB->zBf.get(),
                TB->dgf.get(), TB->s21f.get(), TB->knm.get(), TB->lsd.get()};
    size_t smem = p2m3f_smem(PL);
    dim3 g((unsigned)cnt, nrhs);
    if (helm) {
        k_p2m3f<true><<<g, kP2m3fWarps * 32, smem, P->stream>>>(A, boxes, sigma, dstride, out);
    } else {
        k_p2m3f<false><<<g, kP2m3fWarps * 32, smem, P->stream>>>(A, boxes, sigma, dstride, out);
    }
    CFMM_LAUNCHED();
}

static void launch_l2p3f(H3Tables* TB, bool helm, cfmm_plan_s* P, const int* leaves, int cnt, int maxP,
                         const int* dPlev, const int64_t* eoff, int64_t ncoef, const cd* loc, cd* u, int nrhs) {
    if (cnt == 0) return;
    TreeDev& T = P->tree;
    L2p3fArgs A{P->xr.get(), P->xi.get(), P->n, T.level.get(), target_range(P), T.cen_re.get(),
                T.cen_im.get(), dPlev, eoff, ncoef, P->kappa, P->W, TB->zAf.get(), TB->zBf.get(),
                TB->dgf.get(), TB->s21f.get(), TB->knm.get(), TB->lsd.get()};
    size_t smem = sizeof(double) * (size_t)(maxP + 1) + sizeof(cf) * (size_t)(maxP + 1) * (maxP + 1);
    dim3 g((unsigned)cnt, nrhs);
    if (helm) k_l2p3f<true><<<g, 128, smem, P->stream>>>(A, leaves, loc, u);
    else k_l2p3f<false><<<g, 128, smem, P->stream>>>(A, leaves, loc, u);
    CFMM_LAUNCHED();
}

}  // namespace

void init_helm3d() {
    for (auto f : {(const void*)k_p2m3f<true>, (const void*)k_p2m3f<false>})
        CFMM_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kH3Smem));
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct Helm3dState {
    int l0 = 1, nlev = 0, maxP = 0;
    std::vector<int> Plev;
    DevBuf<int> dPlev;
    DevBuf<int64_t> exp_off;
    int64_t ncoef = 0;
    std::vector<int> leaves_l0;
    DevBuf<int> d_leaves_l0;
    std::vector<int> p2m_off;    // leaves by level: [p2m_off[l], p2m_off[l+1]) in d_p2m
    DevBuf<int> d_p2m;
    std::vector<int> p2l_off;    // List-4 targets by level, likewise
    int n_p2l = 0;
    DevBuf<int> d_p2l_boxes;
    H3Tables* tab = nullptr;
    PairSlots pairs;             // List-2 pairs, workspaces of the translations
    Eval3 eval;                  // M2P, L2P
    int maxP_eval = 0;           // largest order at a leaf's level
};

static std::mutex g_mu;
static std::vector<std::pair<cfmm_plan_s*, Helm3dState*>>& exts() {
    static std::vector<std::pair<cfmm_plan_s*, Helm3dState*>> v;
    return v;
}
static Helm3dState* state(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto& e : exts())
        if (e.first == P) return e.second;
    return nullptr;
}
void helm3d_release(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_mu);
    auto& v = exts();
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i].first == P) {
            delete v[i].second;
            v.erase(v.begin() + i);
            return;
        }
}

// smallest n with |h_n(kR) j_n(kr)| <= eps for n..n+3 (Eq. nterms_criteria_3d),
// R = (k + 1/2) w, r = sqrt(3)/2 w; a short search first, then up to 2000
static int nterms_helm3d_upto(int k, double eps, double kappa, double w, int pmax) {
    double R = (k + 0.5) * w, r = std::sqrt(3.0) * 0.5 * w;
    std::vector<cd> J(pmax + 4), H(pmax + 4);
    sph_j_seq(cd{kappa * r, 0.0}, pmax + 3, J.data());
    sph_h_seq(cd{kappa * R, 0.0}, pmax + 3, H.data());
    std::vector<char> ok(pmax + 4);
    for (int m = 0; m < pmax + 4; ++m) {
        double a = std::sqrt(cabs2(H[m] * J[m]));
        ok[m] = std::isfinite(a) && a <= eps;
    }
    for (int n = 1; n < pmax; ++n)
        if (ok[n] && ok[n + 1] && ok[n + 2] && ok[n + 3]) return n;
    return -1;
}

int nterms_helm3d(int k, double eps, double kappa, double w) {
    int guess = (int)(kappa * (k + 0.5) * w) + 80;
    if (guess < 2000) {
        int n = nterms_helm3d_upto(k, eps, kappa, w, guess);
        if (n > 0) return n;
    }
    int n = nterms_helm3d_upto(k, eps, kappa, w, 2000);
    return n > 0 ? n : 2000;
}

void helm3d_setup(cfmm_plan_s* P) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    Helm3dState* S = new Helm3dState();
    {
        std::lock_guard<std::mutex> lk(g_mu);
        exts().push_back({P, S});
    }
    S->l0 = T.l0;
    S->nlev = T.nlevels;
    S->Plev.resize(T.nlevels);
    for (int l = 0; l < T.nlevels; ++l) S->Plev[l] = nterms_helm3d(P->sep, P->eps * 0.01, P->kappa, P->W / (double)(1 << l));
    P->P = S->Plev;
    if (T.nboxes <= 1) return;
    int maxP = 0;
    for (int l = S->l0; l < T.nlevels; ++l) maxP = std::max(maxP, S->Plev[l]);
    CFMM_REQUIRE(maxP <= kH3MaxP, CFMM_EUNSUPPORTED,
                 "3D Helmholtz: expansion order above 63 at the top expansion level (raise top_level or eps)");
    S->maxP = maxP;
    S->tab = tables(maxP);
    S->dPlev.alloc(T.nlevels);
    CFMM_CUDA(cudaMemcpyAsync(S->dPlev.get(), S->Plev.data(), sizeof(int) * T.nlevels, cudaMemcpyHostToDevice, st));
    std::vector<int64_t> off(T.nboxes, -1);
    int64_t tot = 0;
    for (int l = S->l0; l < T.nlevels; ++l)
        for (int b = T.level_off[l]; b < T.level_off[l + 1]; ++b) {
            off[b] = tot;
            tot += (int64_t)(S->Plev[l] + 1) * (S->Plev[l] + 1);
        }
    S->ncoef = tot;
    P->ncoef = tot;
    S->exp_off.alloc(T.nboxes);
    CFMM_CUDA(cudaMemcpyAsync(S->exp_off.get(), off.data(), sizeof(int64_t) * T.nboxes, cudaMemcpyHostToDevice, st));
    std::vector<int> lvl(T.nboxes), l4(T.nboxes + 1), boxes;
    CFMM_CUDA(cudaMemcpyAsync(lvl.data(), T.level.get(), sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaMemcpyAsync(l4.data(), T.loff[3].get(), sizeof(int) * (T.nboxes + 1), cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaStreamSynchronize(st));
    for (int b : T.leaf_boxes)
        if (lvl[b] >= S->l0) S->leaves_l0.push_back(b);
    pair_slots_build(P, &S->pairs, T.hloff[1], S->l0);
    S->d_leaves_l0.alloc(S->leaves_l0.size());
    CFMM_CUDA(cudaMemcpyAsync(S->d_leaves_l0.get(), S->leaves_l0.data(), sizeof(int) * S->leaves_l0.size(),
                              cudaMemcpyHostToDevice, st));
    std::vector<int> byl = S->leaves_l0;
    std::stable_sort(byl.begin(), byl.end(), [&](int x, int y) { return lvl[x] < lvl[y]; });
    S->p2m_off.assign(T.nlevels + 1, 0);
    for (int b : byl) S->p2m_off[lvl[b] + 1]++;
    for (int l = 0; l < T.nlevels; ++l) S->p2m_off[l + 1] += S->p2m_off[l];
    S->d_p2m.alloc(byl.size());
    CFMM_CUDA(cudaMemcpyAsync(S->d_p2m.get(), byl.data(), sizeof(int) * byl.size(), cudaMemcpyHostToDevice, st));
    S->p2l_off.assign(T.nlevels + 1, 0);
    for (int b = T.level_off[S->l0]; b < T.nboxes; ++b)
        if (l4[b + 1] > l4[b]) {
            boxes.push_back(b);
            S->p2l_off[lvl[b] + 1]++;
        }
    for (int l = 0; l < T.nlevels; ++l) S->p2l_off[l + 1] += S->p2l_off[l];
    S->n_p2l = (int)boxes.size();
    {
        std::vector<int> tst(T.nboxes), ten(T.nboxes);
        const SubRange tr = target_range(P);
        CFMM_CUDA(cudaMemcpyAsync(tst.data(), tr.st, sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
        CFMM_CUDA(cudaMemcpyAsync(ten.data(), tr.en, sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
        CFMM_CUDA(cudaStreamSynchronize(st));
        eval3_build(&S->eval, S->leaves_l0, T.hloff[2], tst, ten, S->d_leaves_l0.get(), T.loff[2].get(), st);
        for (int b : S->leaves_l0) S->maxP_eval = std::max(S->maxP_eval, S->Plev[lvl[b]]);
    }
    S->d_p2l_boxes.alloc(boxes.size());
    if (!boxes.empty())
        CFMM_CUDA(cudaMemcpyAsync(S->d_p2l_boxes.get(), boxes.data(), sizeof(int) * boxes.size(),
                                  cudaMemcpyHostToDevice, st));
    CFMM_CUDA(cudaStreamSynchronize(st));
}

void helm3d_apply(cfmm_plan_s* P, const cd* sigma, const cd* tau, int64_t dstride, cd* u, int nrhs, cd* g) {
    Helm3dState* S = state(P);
    CFMM_REQUIRE(S, CFMM_EINVAL, "plan has no 3D Helmholtz state");
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    auto rec = [&](int i) {
        if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev[i], st));
    };
    KParams K{P->xr.get(), P->xi.get(), P->nr.get(), P->ni.get(), P->xr.get(), P->xi.get(), P->n, P->n,
              sigma, tau, dstride, P->slp, P->dlp, P->kappa};
    bool mixed = P->precision == CFMM_MIXED;
    if (T.nboxes <= 1) {
        for (int i = 2; i <= 6; ++i) rec(i);
        launch_p2p(3, P->kernel, K, T.d_leaf_boxes.get(), T.nleaves, near_ranges(P), T.loff[0].get(),
                   T.lent[0].get(), u, nrhs, st, mixed, P->leaf_size);
        if (g)
            launch_p2p_grad(3, P->kernel, K, T.d_leaf_boxes.get(), T.nleaves, near_ranges(P), T.loff[0].get(), T.lent[0].get(), g, nrhs, st, P->leaf_size);
        rec(7);
        rec(8);
        return;
    }
    size_t need = (size_t)S->ncoef * nrhs;
    P->mpole.alloc(need);
    P->local.alloc(need);
    cd* mp = P->mpole.get();
    cd* lc = P->local.get();
    H3Tables* TB = S->tab;
    int maxP = S->maxP;
    // (3) P2P (writes u) on the side stream, beside the far field
    {
        cudaStream_t ns = near_fork(P);
        launch_p2p(3, P->kernel, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P), T.loff[0].get(), T.lent[0].get(), u, nrhs, ns, mixed, P->leaf_size, T.level.get(), P->W,
                   P->sep);
        if (g)
            launch_p2p_grad(3, P->kernel, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P), T.loff[0].get(), T.lent[0].get(), g, nrhs, ns, P->leaf_size);
    }
    near_launched(P);
    bool slp_only = P->slp && !P->dlp;
    auto p2x = [&](int l, bool sing, const int* boxes, int cnt, cd* dst) {
        P2x3Args X{boxes, cnt, sing, S->Plev[l], S->dPlev.get(), S->exp_off.get(), S->ncoef, P->kappa};
        CFMM_REQUIRE(p2x3_apply(P, eval3_tables(TB), X, sigma, tau, dstride, dst, nrhs), CFMM_EUNSUPPORTED,
                     "3D Helmholtz P2M/P2L exceeds shared memory");
    };
    // (1) P2M, one launch per level (shared memory sized by that level's P)
    for (int l = S->l0; l < T.nlevels; ++l) {
        int cnt = S->p2m_off[l + 1] - S->p2m_off[l];
        if (cnt <= 0) continue;
        if (slp_only && mixed && p2m3f_smem(S->Plev[l]) <= (size_t)kH3Smem) {
            // complex64 products, FP64 sums
            launch_p2m3f(TB, true, P, S->d_p2m.get() + S->p2m_off[l], cnt, S->Plev[l], S->dPlev.get(),
                         S->exp_off.get(), S->ncoef, sigma, dstride, mp, nrhs);
            continue;
        }
        p2x(l, false, S->d_p2m.get() + S->p2m_off[l], cnt, mp);
    }
    rec(2);
    const Tr3Tables tr = tr3_tables(TB);
    // (2) M2M: parents at level l from children at l + 1
    for (int l = T.nlevels - 2; l >= S->l0; --l)
        pairs3d_m2m(P, &S->pairs, tr, l, S->Plev[l + 1], S->Plev[l], P->kappa, S->exp_off.get(), S->ncoef, mp, nrhs);
    rec(3);
    // (4) M2L per level (overwrites L at levels >= l0)
    for (int l = S->l0; l < T.nlevels; ++l)
        pairs3d_m2l(P, &S->pairs, tr, l, l + 1, S->Plev[l], P->kappa, S->exp_off.get(), S->ncoef, mp, lc, nrhs);
    rec(4);
    // (6) P2L, per level
    for (int l = S->l0; l < T.nlevels; ++l) {
        int cnt = S->p2l_off[l + 1] - S->p2l_off[l];
        if (cnt <= 0) continue;
        p2x(l, true, S->d_p2l_boxes.get() + S->p2l_off[l], cnt, lc);
    }
    rec(5);
    // (7) L2L
    for (int l = S->l0; l + 1 < T.nlevels; ++l)
        pairs3d_l2l(P, &S->pairs, tr, l, S->Plev[l], S->Plev[l + 1], P->kappa, S->exp_off.get(), S->ncoef, lc, nrhs);
    rec(6);
    rec(7);
    near_join(P);   // the near field has written u
    // (5) M2P, (8) L2P (complex64 in mixed precision)
    {
        Eval3Args E{S->d_leaves_l0.get(), (int)S->leaves_l0.size(), S->dPlev.get(), S->maxP_eval, S->exp_off.get(),
                    S->ncoef, P->kappa, mp, lc};
        eval3_apply(P, &S->eval, eval3_tables(TB), E, !mixed, u, g, nrhs);
        if (mixed) launch_l2p3f(TB, true, P, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), maxP, S->dPlev.get(),
                                S->exp_off.get(), S->ncoef, lc, u, nrhs);
    }
    rec(8);
}

// ---------------------------------------------------------------------------
// 3D Laplace translations (used by fmm3d.cu)
// ---------------------------------------------------------------------------
struct Lap3Tr {
    H3Tables* tab = nullptr;
    int Pord = 0;
    PairSlots pairs;
};

Lap3Tr* lap3_tr_create(cfmm_plan_s* P, int Pord) {
    TreeDev& T = P->tree;
    auto L = std::make_unique<Lap3Tr>();
    L->tab = tables(Pord);
    L->Pord = Pord;
    pair_slots_build(P, &L->pairs, T.hloff[1], T.l0);
    return L.release();
}

void lap3_p2x(Lap3Tr* L, cfmm_plan_s* P, const P2x3Args& A, const cd* sigma, const cd* tau, int64_t dstride, cd* out,
              int nrhs) {
    CFMM_REQUIRE(p2x3_apply(P, eval3_tables(L->tab), A, sigma, tau, dstride, out, nrhs), CFMM_EUNSUPPORTED,
                 "3D Laplace P2M/P2L exceeds shared memory");
}

bool lap3_p2m32(Lap3Tr* L, cfmm_plan_s* P, const int* leaves, int cnt, int maxP, const int* dPlev,
                const int64_t* eoff, int64_t ncoef, const cd* sigma, int64_t dstride, cd* out, int nrhs) {
    if (maxP > L->tab->Pmax || p2m3f_smem(maxP) > (size_t)kH3Smem) return false;
    launch_p2m3f(L->tab, false, P, leaves, cnt, maxP, dPlev, eoff, ncoef, sigma, dstride, out, nrhs);
    return true;
}

void lap3_l2p32(Lap3Tr* L, cfmm_plan_s* P, const int* leaves, int cnt, int maxP, const int* dPlev,
                const int64_t* eoff, int64_t ncoef, const cd* loc, cd* u, int nrhs) {
    CFMM_REQUIRE(maxP <= L->tab->Pmax, CFMM_ECUDA, "3D Laplace L2P: order beyond the tables");
    launch_l2p3f(L->tab, false, P, leaves, cnt, maxP, dPlev, eoff, ncoef, loc, u, nrhs);
}

void lap3_tr_destroy(Lap3Tr* L) { delete L; }

void lap3_m2l(Lap3Tr* L, cfmm_plan_s* P, int l_lo, int l_hi, int Pord, const int64_t* eoff, int64_t ncoef, const cd* mp,
              cd* lc, int nrhs) {
    pairs3d_m2l(P, &L->pairs, tr3_tables(L->tab), l_lo, l_hi, Pord, 0.0, eoff, ncoef, mp, lc, nrhs);
}

void lap3_eval(Lap3Tr* L, cfmm_plan_s* P, Eval3* E, const Eval3Args& A, bool l2p, cd* u, cd* g, int nrhs) {
    eval3_apply(P, E, eval3_tables(L->tab), A, l2p, u, g, nrhs);
}

void lap3_m2m(Lap3Tr* L, cfmm_plan_s* P, int l, int Pord, const int64_t* eoff, int64_t ncoef, cd* mp, int nrhs) {
    pairs3d_m2m(P, &L->pairs, tr3_tables(L->tab), l, Pord, Pord, 0.0, eoff, ncoef, mp, nrhs);
}

void lap3_l2l(Lap3Tr* L, cfmm_plan_s* P, int l, int Pord, const int64_t* eoff, int64_t ncoef, cd* lc, int nrhs) {
    pairs3d_l2l(P, &L->pairs, tr3_tables(L->tab), l, Pord, Pord, 0.0, eoff, ncoef, lc, nrhs);
}

}  // namespace cfmm

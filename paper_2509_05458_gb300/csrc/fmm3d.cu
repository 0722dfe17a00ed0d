// 3D complex-coordinate Laplace FMM: expansions and translations (Sec. 5.2,
// Sec. 6.4), FP64.
//
// Solid harmonics of a complex 3-vector x (x+ = x1 + i x2, x- = x1 - i x2,
// z = x3, rho^2 = x+ x- + z^2 = x.x):
//   regular   U_n^m = rho^n P_n^m(cos theta) e^{im phi}/(n+m)!
//   irregular T_n^m = (n-m)! P_n^m(cos theta) e^{im phi}/rho^{n+1}
// by their three-term recurrences (entire in x; no angle is formed);
// U_n^{-m} = (-1)^m U_n^m[x+ <-> x-], likewise T. With
//   1/|x - y| = sum (-1)^m U_n^{-m}(y) T_n^m(x)             (Lemma 5.2.1, Eq. sphaddition)
//   U_n^m(a + b) = sum U_k^l(a) U_{n-k}^{m-l}(b)
//   T_n^m(x - y) = sum (-1)^l U_k^{-l}(y) T_{n+k}^{m+l}(x)
// the operators are (coefficients at n*n + n + m):
//   P2M  M_n^m = sum s (-1)^m U_n^{-m}(y - c)          M2P  u = sum M_n^m T_n^m(x - c)
//   M2M  M_n^m(c) = sum (-1)^l U_k^l(c' - c) M_{n-k}^{m+l}(c')
//   M2L  L_k^l = (-1)^{k+l} sum M_n^m T_{n+k}^{m-l}(c_t - c_s)
//   L2L  L'_k^l = sum L_n^m U_{n-k}^{m-l}(c' - c)
//   P2L  L_k^l = sum s (-1)^l T_k^{-l}(y - c)          L2P  u = sum L_k^l U_k^l(x - c)
// The translations run as point-and-shoot (rotate the shift onto the z-axis,
// translate along it, rotate back; O(P^3)), in pairs3d.cu.
// Double layer: n.grad = nu+ d+ + nu- d- + n3 dz (nu+- = n1 +- i n2),
//   d+ U_n^m = -U_{n-1}^{m-1}/2, d- U_n^m = U_{n-1}^{m+1}/2, dz U_n^m = U_{n-1}^m,
//   d+ T_n^m = -T_{n+1}^{m-1}/2, d- T_n^m = T_{n+1}^{m+1}/2, dz T_n^m = -T_{n+1}^m.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "cfmm_special.cuh"
#include "eval3d.cuh"
#include "kernels.cuh"

namespace cfmm {

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct Fmm3dState {
    int l0 = 1, nlev = 0, maxP = 0;
    std::vector<int> Plev;
    DevBuf<int> dPlev;
    DevBuf<int64_t> exp_off;
    int64_t ncoef = 0;
    std::vector<int> leaves_l0;
    DevBuf<int> d_leaves_l0;
    int n_p2l = 0;
    DevBuf<int> d_p2l_boxes;
    Lap3Tr* tr = nullptr;
    Eval3 eval;                  // M2P, L2P
    ~Fmm3dState() { lap3_tr_destroy(tr); }
};

static std::mutex g_mu3;
static std::vector<std::pair<cfmm_plan_s*, Fmm3dState*>>& exts3() {
    static std::vector<std::pair<cfmm_plan_s*, Fmm3dState*>> v;
    return v;
}
static Fmm3dState* state3(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_mu3);
    for (auto& e : exts3())
        if (e.first == P) return e.second;
    return nullptr;
}
void fmm3d_release(cfmm_plan_s* P) {
    std::lock_guard<std::mutex> lk(g_mu3);
    auto& v = exts3();
    for (size_t i = 0; i < v.size(); ++i)
        if (v[i].first == P) {
            delete v[i].second;
            v.erase(v.begin() + i);
            return;
        }
}

static int nterms_laplace3(int k, double eps) {
    double ratio = (std::sqrt(3.0) * 0.5) / (k + 0.5);
    double t = 1.0;
    int n = 0;
    for (;;) {
        ++n;
        t *= ratio;
        if (t <= eps) return n;
    }
}

void fmm3d_setup(cfmm_plan_s* P) {
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    Fmm3dState* S = new Fmm3dState();
    {
        std::lock_guard<std::mutex> lk(g_mu3);
        exts3().push_back({P, S});
    }
    S->l0 = T.l0;
    S->nlev = T.nlevels;
    S->Plev.assign(T.nlevels, nterms_laplace3(P->sep, P->eps * 0.1));
    P->P = S->Plev;
    // 3D Helmholtz: the tree and lists are built; the apply reports that its
    // translations are not (unless the tree is a single leaf)
    if (T.nboxes <= 1 || P->kernel != CFMM_LAPLACE) return;
    int maxP = S->Plev[0];
    CFMM_REQUIRE(maxP <= 63, CFMM_EUNSUPPORTED, "3D Laplace: expansion order above 63 (eps too small)");
    S->maxP = maxP;
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
    std::vector<int> lvl(T.nboxes), l4(T.nboxes + 1), hst(T.nboxes), hen(T.nboxes), boxes;
    const SubRange tr = target_range(P);
    CFMM_CUDA(cudaMemcpyAsync(hst.data(), tr.st, sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaMemcpyAsync(hen.data(), tr.en, sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaMemcpyAsync(lvl.data(), T.level.get(), sizeof(int) * T.nboxes, cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaMemcpyAsync(l4.data(), T.loff[3].get(), sizeof(int) * (T.nboxes + 1), cudaMemcpyDeviceToHost, st));
    CFMM_CUDA(cudaStreamSynchronize(st));
    for (int b : T.leaf_boxes)
        if (lvl[b] >= S->l0) S->leaves_l0.push_back(b);
    S->d_leaves_l0.alloc(S->leaves_l0.size());
    CFMM_CUDA(cudaMemcpyAsync(S->d_leaves_l0.get(), S->leaves_l0.data(), sizeof(int) * S->leaves_l0.size(),
                              cudaMemcpyHostToDevice, st));
    for (int b = T.level_off[S->l0]; b < T.nboxes; ++b)
        if (l4[b + 1] > l4[b]) boxes.push_back(b);
    S->n_p2l = (int)boxes.size();
    S->d_p2l_boxes.alloc(boxes.size());
    if (!boxes.empty())
        CFMM_CUDA(cudaMemcpyAsync(S->d_p2l_boxes.get(), boxes.data(), sizeof(int) * boxes.size(),
                                  cudaMemcpyHostToDevice, st));
    CFMM_CUDA(cudaStreamSynchronize(st));
    eval3_build(&S->eval, S->leaves_l0, T.hloff[2], hst, hen, S->d_leaves_l0.get(), T.loff[2].get(), st);
    S->tr = lap3_tr_create(P, maxP);
}

void fmm3d_apply(cfmm_plan_s* P, const cd* sigma, const cd* tau, int64_t dstride, cd* u, int nrhs, cd* g) {
    Fmm3dState* S = state3(P);
    CFMM_REQUIRE(S, CFMM_EINVAL, "plan has no 3D state");
    TreeDev& T = P->tree;
    cudaStream_t st = P->stream;
    auto rec = [&](int i) {
        if (P->timing) CFMM_CUDA(cudaEventRecord(P->ev[i], st));
    };
    KParams K{P->xr.get(), P->xi.get(), P->nr.get(), P->ni.get(), P->xr.get(), P->xi.get(), P->n, P->n,
              sigma, tau, dstride, P->slp, P->dlp, P->kappa};
    bool mixed = P->precision == CFMM_MIXED;
    CFMM_REQUIRE(T.nboxes <= 1 || P->kernel == CFMM_LAPLACE, CFMM_EUNSUPPORTED,
                 "3D Helmholtz translations are not built yet");
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
    int maxP = S->maxP;
    // (3) P2P (writes u) on the side stream, beside the far field
    {
        cudaStream_t ns = near_fork(P);
        launch_p2p(3, P->kernel, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P), T.loff[0].get(), T.lent[0].get(), u, nrhs, ns, mixed, P->leaf_size);
        if (g)
            launch_p2p_grad(3, P->kernel, K, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), near_ranges(P), T.loff[0].get(), T.lent[0].get(), g, nrhs, ns, P->leaf_size);
    }
    near_launched(P);
    // (1) P2M (single layer: complex64 products with FP64 sums in mixed precision)
    bool slp1 = P->slp && !P->dlp;
    bool p2m_done = slp1 && mixed &&
                    lap3_p2m32(S->tr, P, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), maxP, S->dPlev.get(),
                               S->exp_off.get(), S->ncoef, sigma, dstride, mp, nrhs);
    P2x3Args X{S->d_leaves_l0.get(), (int)S->leaves_l0.size(), false, maxP, S->dPlev.get(), S->exp_off.get(), S->ncoef,
               0.0};
    if (!p2m_done) lap3_p2x(S->tr, P, X, sigma, tau, dstride, mp, nrhs);
    rec(2);
    int Pu = S->Plev[0];
    // (2) M2M
    for (int l = T.nlevels - 2; l >= S->l0; --l)
        lap3_m2m(S->tr, P, l, Pu, S->exp_off.get(), S->ncoef, mp, nrhs);
    rec(3);
    // (4) M2L
    lap3_m2l(S->tr, P, S->l0, T.nlevels, Pu, S->exp_off.get(), S->ncoef, mp, lc, nrhs);
    rec(4);
    // (6) P2L
    X.boxes = S->d_p2l_boxes.get();
    X.cnt = S->n_p2l;
    X.sing = true;
    lap3_p2x(S->tr, P, X, sigma, tau, dstride, lc, nrhs);
    rec(5);
    // (7) L2L
    for (int l = S->l0; l + 1 < T.nlevels; ++l)
        lap3_l2l(S->tr, P, l, Pu, S->exp_off.get(), S->ncoef, lc, nrhs);
    rec(6);
    rec(7);
    near_join(P);   // the near field has written u
    // (5) M2P, (8) L2P (complex64 in mixed precision)
    {
        Eval3Args E{S->d_leaves_l0.get(), (int)S->leaves_l0.size(), S->dPlev.get(), maxP, S->exp_off.get(), S->ncoef,
                    0.0, mp, lc};
        lap3_eval(S->tr, P, &S->eval, E, !mixed, u, g, nrhs);
        if (mixed) lap3_l2p32(S->tr, P, S->d_leaves_l0.get(), (int)S->leaves_l0.size(), maxP, S->dPlev.get(),
                              S->exp_off.get(), S->ncoef, lc, u, nrhs);
    }
    rec(8);
}

}  // namespace cfmm

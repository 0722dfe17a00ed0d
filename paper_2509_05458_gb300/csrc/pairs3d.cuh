// 3D translations with the pairs on the lanes (pairs3d.cu).
#pragma once

#include "kernels.cuh"

namespace cfmm {

// Device tables of the 3D translations (helm3d.cu builds and owns them)
struct Tr3Tables {
    const double* Dh;       // D_n[m][m'], m, m' >= 0, column-major per order
    const double* Dg;       // D_n scaled by (-1)^n/(2n+1)
    const int64_t* Dhoff;
    const double *al, *be;  // coaxial recurrence coefficients by nmi(n, m >= 0)
    const double* ab;       // al_n^m be_{n-1}^m
    const double* cg;       // g_n gamma_n^m, g_n = (-1)^n (2n+1), gamma_m = 1, gamma_{n+1} = gamma_n / be_n
    const double *smu, *snu;   // mu_{n+1}^{m-1}, nu_{n-1}^{m-1} over nu_{m-1}^{m-1} (sectorial columns)
    const double *lsm, *lsd;   // eps_m s_n^m, eps_m / s_n^m by nmi(n, m)
    const double *fact, *ifact;   // j!, 1/j!
};

// The unordered List-2 pairs of a plan in slots of 32-lane tiles: level l owns
// the tiles [tile0[l], tile0[l+1]). With one order at every level (Laplace) all
// levels are translated in one go.
struct PairSlots {
    std::vector<int> tile0;
    int64_t nslot = 0;
    DevBuf<int> box_a, box_b;     // the pair's boxes (a < b), -1 for an empty slot
    DevBuf<signed char> kind;     // kPairFlat, kPairGeneral, kPairIso + k
    DevBuf<int> slot;             // per List-2 entry: 2 slot + (0: owner is box_a, 1: box_b)
    DevBuf<int> d_tile0;
    // workspaces of an apply; an apply recorded in a graph keeps the pointers, and no size
    // here grows when the right-hand sides become fewer
    DevBuf<cd> pw, fl, sect, tri, vec;
    DevBuf<signed char> kind_c;   // M2M, L2L: kind of each child's shift
};

// Builds the slots of the plan's List 2 (device work on the plan's stream)
void pair_slots_build(cfmm_plan_s* P, PairSlots* S, const std::vector<int>& l2off, int l0);

// M2L of the boxes of levels [l_lo, l_hi) at order Pord, all right-hand sides:
// local expansions of those boxes are overwritten. Laplace when kappa == 0.
void pairs3d_m2l(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l_lo, int l_hi, int Pord, double kappa,
                 const int64_t* eoff, int64_t ncoef, const cd* mp, cd* lc, int nrhs);
// M2M into the non-leaf boxes of level l (order Pp) from level l + 1 (order Pc)
void pairs3d_m2m(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l, int Pc, int Pp, double kappa,
                 const int64_t* eoff, int64_t ncoef, cd* mp, int nrhs);
// L2L from level l (order Pp), added to the boxes of level l + 1 (order Pc)
void pairs3d_l2l(cfmm_plan_s* P, PairSlots* S, const Tr3Tables& T, int l, int Pp, int Pc, double kappa,
                 const int64_t* eoff, int64_t ncoef, cd* lc, int nrhs);

}  // namespace cfmm

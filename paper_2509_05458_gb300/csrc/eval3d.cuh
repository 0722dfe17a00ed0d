// FP64 expansions of and at points, 3D: P2M, P2L, M2P (List 3), L2P and gradients of
// the last two (eval3d.cu).
#pragma once

#include "kernels.cuh"

namespace cfmm {

// q_n^m = A_n^m (zeta q_{n-1}^m) - B_n^m (w q_{n-2}^m), q_m^m = D_m: the part of a
// harmonic that +m and -m share (see eval3d.cu); A, B by nmi(n, m), m >= 0
struct QTables {
    const double *A, *B, *D;
};
struct Eval3Tables {
    QTables Z, U, T;             // Helmholtz; Laplace regular and irregular
    const double *g3, *gp, *gm;  // Helmholtz gradient coefficients by nmi(n, m), all m
};
// host tables of q for orders <= N (kind 0: Z, 1: U, 2: T), A and B of (N+1)^2 entries, D of N+1
void eval3_qtable(int kind, int N, double* A, double* B, double* D);

// Per plan: items (List-3 entry, target) of each leaf, and the buffers of an apply. An
// apply takes ranges of leaves whose slots fit a budget (a graded cloud has far more items
// than points).
struct EvalRange {
    int leaf0, leaf1;             // leaves of the list
    int64_t t0, nt;               // their targets
    int64_t slots;                // nt, then the items
};
struct Eval3 {
    std::vector<EvalRange> ranges;
    int64_t max_slots = 0;        // of a range
    DevBuf<int64_t> ioff;         // first item of each leaf of the plan's list
    DevBuf<int> own;              // leaf (position in the list) of each List-3 entry
    DevBuf<cd> val;               // slots of the potential; an apply recorded in a graph keeps the pointer,
    DevBuf<cd> gval, gco;         // so a gradient has slots of its own, and derived coefficients
};
// leaves: box index of each leaf of the plan's list; l3off, st, en: host copies of
// the List-3 offsets and the boxes' target ranges
void eval3_build(Eval3* E, const std::vector<int>& leaves, const std::vector<int>& l3off, const std::vector<int>& st,
                 const std::vector<int>& en, const int* d_leaves, const int* d_l3off, cudaStream_t stream);

struct Eval3Args {
    const int* leaves;            // device list of the leaves
    int nleaf;
    const int* Plev;              // orders by level (device)
    int maxP;                     // largest order of a leaf's or a List-3 box's expansion
    const int64_t* eoff;
    int64_t ncoef;
    double kappa;                 // 0: Laplace
    const cd *mp, *loc;
};
// P2M of `cnt` leaves (written), or P2L into `cnt` boxes over their List 4 (added), FP64,
// single layer (sigma) and/or double layer (tau); P: the largest order among the boxes
struct P2x3Args {
    const int* boxes;
    int cnt;
    bool sing;                    // P2L
    int P;
    const int* Plev;
    const int64_t* eoff;
    int64_t ncoef;
    double kappa;                 // 0: Laplace
};
bool p2x3_apply(cfmm_plan_s* P, const Eval3Tables& T, const P2x3Args& A, const cd* sigma, const cd* tau, int64_t dstride,
                cd* out, int nrhs);
// u [rhs][n] += M2P, and L2P when l2p; g [rhs][3][n] += gradients of both (either may be null)
void eval3_apply(cfmm_plan_s* P, Eval3* E, const Eval3Tables& T, const Eval3Args& A, bool l2p, cd* u, cd* g, int nrhs);

}  // namespace cfmm

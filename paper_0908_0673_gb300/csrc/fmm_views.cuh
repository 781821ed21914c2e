// Kernel-argument views of a plan, shared by the product's translation units.
#pragma once

#include "bem_internal.cuh"

namespace bem {

struct Tabs {
    const int *m, *n, *k, *idx3;
    const double *fact;
    int p, np;                          // largest order, and the coefficient count (array stride)
    const int *lev_p;                   // order of each tree level (nullptr: p everywhere)
};

// number of multi-indices of degree <= q (the coefficients of order q)
__host__ __device__ __forceinline__ int np_of(int q) { return (q + 1) * (q + 2) * (q + 3) / 6; }
__device__ __forceinline__ int order_of(const Tabs &tb, int level) { return tb.lev_p ? tb.lev_p[level] : tb.p; }

struct TreeView {
    const int *level, *ix, *iy, *iz, *parent, *child0, *nchild, *nb, *ne, *eb, *ee, *leaves;
    const int *near_ptr, *near_idx, *inter_ptr, *inter_idx, *node_perm, *reach;
    const double *cx, *cy, *cz, *r, *tx, *ty, *tz;
    double side;
};

struct QuadView {
    const double *x, *y, *z, *nx, *ny, *nz, *w;
    const float *fx, *fy, *fz, *fnx, *fny, *fnz, *fw;
    const float *lx, *ly, *lz, *lnx, *lny, *lnz;     // float64 plans: low parts of the pairs (fx, lx) ...
};

Tabs tabs_of(const bem_plan *P);
TreeView view_of(const bem_plan *P);
QuadView quad_of(const bem_plan *P);

// float64 near field in float32 pairs (near_f64.cu)
constexpr int ND_SLOTS = 32;            // targets per work item
int near_pairs_prepare(bem_plan *P);
bool near_pairs_apply(const bem_plan *P, int C, double kwave);
template <int C>
int launch_near_pairs(bem_plan *P, int op, double kwave, const double *f, double *ytmp, cudaStream_t s);

// P2M of float64 plans in float32 pairs (p2m_f64.cu)
int p2m_pairs_prepare();
template <int C>
int launch_p2m_pairs(bem_plan *P, bool dl, const double *f, double *M, cudaStream_t s);

}  // namespace bem

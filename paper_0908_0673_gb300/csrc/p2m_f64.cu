// P2M of float64 plans (Eq. 6) in float32 pairs (dfloat.cuh): one block, or a
// cluster of blocks sharing the points, per leaf.
//
// The on-the-fly float64 form took three products and an accumulation per
// (point, coefficient) on a pipe with 1/64 of the float32 rate: 593 us for
// 61,236 points at p = 10 (double layer), 164 us for 8,960 at p = 8 on 56
// blocks.  Here a thread holds a row (m, n) and all its k in registers, for
// every second, third, ... pair of points: the row's factors x^m y^n and
// their normal derivative are formed once per point, then each k costs two pair
// multiply-adds (one for the single layer), packed over two points.  Powers come
// from shared memory, built per 64 points; strengths are folded into the x
// powers (real) at a power-of-two scale taken from the block's largest.  Offsets
// are taken in units of the edge x 2^box_reach, so that the powers stay in
// float32's range; the factor returns with the float64 sums.
// Measured: 61,236 points, p = 10, double layer 593 -> 98 us; 31,500 points,
// single layer 205 -> 37; 20,160 points, Helmholtz double layer 399 -> 68; 8,960
// points, p = 8 (56 leaves, four blocks each) 164 -> 23.  About 9,300 float32
// operations a point at p = 10, 40 % of the float32 pipe: the rows of a warp
// differ in length (60 % of its lanes busy), and power tables cost the rest.
#include <algorithm>
#include <cmath>

#include "cluster.cuh"
#include "dfloat.cuh"
#include "fmm_views.cuh"

namespace bem {

namespace {

constexpr int PP_T = 256, PP_B = 64, PP_S = PP_B + 2;   // threads, points per round, their stride
constexpr int PP_MAXC = 4;                              // blocks per cluster at most

// power tables: [axis][P h, P l, Q h, Q l][p + 1][PP_S]; strengths [C][h, l][PP_S]
__host__ __device__ constexpr size_t pp_tab(int p, int C) { return (size_t)(12 * (p + 1) + 2 * C) * PP_S; }
__host__ __device__ inline size_t pp_smem(int p, int C) {
    const size_t np = (size_t)(p + 1) * (p + 2) * (p + 3) / 6, nrow = (size_t)(p + 1) * (p + 2) / 2;
    const size_t groups = PP_T / nrow > 0 ? PP_T / nrow : 1;
    const size_t tab = sizeof(float) * pp_tab(p, C), red = sizeof(float2) * groups * np * C;
    return ((tab > red ? tab : red) + 7) / 8 * 8 + sizeof(double) * np * C;   // + this block's share
}

__device__ __forceinline__ P2 ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }

struct D2 {                             // pairs of two points
    P2 h, l;
};
__device__ __forceinline__ D2 dmul(D2 a, D2 b) {
    const P2 p = pmul(a.h, b.h);
    P2 e = pfma(a.h, b.h, pneg(p));
    e = pfma(a.h, b.l, e);
    e = pfma(a.l, b.h, e);
    return D2{p, e};
}
__device__ __forceinline__ D2 dadd(D2 a, D2 b) {
    D2 r;
    P2 e;
    two_sum(a.h, b.h, r.h, e);
    r.l = padd(padd(a.l, b.l), e);
    return r;
}
__device__ __forceinline__ void dacc(D2 &acc, D2 a, D2 b) { acc = dadd(acc, dmul(a, b)); }

// scalar pair product, for the power tables
__device__ __forceinline__ void df_mul(float &h, float &l, float bh, float bl) {
    const float p = __fmul_rn(h, bh);
    l = fmaf(l, bh, fmaf(h, bl, fmaf(h, bh, -p)));
    h = p;
}

template <int C, bool DL, int KM>
__global__ void __launch_bounds__(PP_T, KM <= 11 && C == 1 ? 2 : 1) k_p2m_pairs(int ns, Tabs tb, TreeView tv, QuadView qv, const double *__restrict__ f,
                                                    double *__restrict__ M, const int *__restrict__ skip) {
    if (skip && *skip) return;                          // every block of the cluster reads the same word
    extern __shared__ __align__(16) float pp_sm[];
    __shared__ int wexp[PP_T / 32];
    const int rank = ns > 1 ? (int)cluster_rank() : 0;
    const int b = tv.leaves[blockIdx.x / ns], tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np = tb.np, p = order_of(tb, tv.level[b]), npl = np_of(p), P1 = p + 1, nrow = P1 * (p + 2) / 2;
    const int groups = max(1, PP_T / nrow), grp = tid / nrow;
    double *share = (double *)((char *)pp_sm + (pp_smem(tb.p, C) - sizeof(double) * np * C));
    // this block's points, and the exponent of its largest strength
    const int qa = tv.eb[b] * NQ, nq = (tv.ee[b] - tv.eb[b]) * NQ;
    const int q0 = qa + (int)((long long)nq * rank / ns), q1 = qa + (int)((long long)nq * (rank + 1) / ns);
    int E = 1;
    for (int i = q0 * C + tid; i < q1 * C; i += PP_T) E = max(E, (int)((unsigned)__double2hiint(f[i]) >> 20) & 0x7ff);
#pragma unroll
    for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    if (lane == 0) wexp[warp] = E;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < PP_T / 32; w++) E = max(E, wexp[w]);
    E = min(E, 2046);                                   // an infinity or NaN carries itself
    // offsets and normals in units of the leaf's edge x 2^reach
    const int es = ilogb(tv.side), reach = tv.reach[b];
    float uh, ul;                                       // 2^es / unit: the plan's pairs hold offsets x 2^-es
    df_split(1.0 / scalbn(tv.side, reach - tv.level[b] - es), uh, ul);
    // row of this thread, in order of m + n (rows of a warp have about the same length)
    const bool worker = grp < groups;
    int deg = 0, r = tid - grp * nrow;
    while (r > deg) r -= ++deg;
    const int n = r, m = deg - r, len = worker ? P1 - deg : 0;
    D2 acc[KM][C];
#pragma unroll
    for (int k = 0; k < KM; k++)
#pragma unroll
        for (int c = 0; c < C; c++) acc[k][c] = D2{p2(0.f), p2(0.f)};
    float *tab = pp_sm, *str = pp_sm + (size_t)12 * P1 * PP_S;
    auto at = [&](int ax, int w, int e) { return tab + ((size_t)(ax * 4 + w) * P1 + e) * PP_S; };
    for (int base = q0; base < q1; base += PP_B) {
        const int nb = min(PP_B, q1 - base);
        __syncthreads();
        if (tid < 3 * PP_B) {
            const int ax = tid / PP_B, pt = tid % PP_B, o = base + pt;
            const bool on = pt < nb;
            float dh = 0.f, dl = 0.f, ch = 0.f, cl = 0.f, vh = 1.f, vl = 0.f;
            if (on) {
                dh = ax == 0 ? qv.fx[o] : ax == 1 ? qv.fy[o] : qv.fz[o];
                dl = ax == 0 ? qv.lx[o] : ax == 1 ? qv.ly[o] : qv.lz[o];
                df_mul(dh, dl, uh, ul);
                if (DL) {
                    ch = ax == 0 ? qv.fnx[o] : ax == 1 ? qv.fny[o] : qv.fnz[o];
                    cl = ax == 0 ? qv.lnx[o] : ax == 1 ? qv.lny[o] : qv.lnz[o];
                    df_mul(ch, cl, uh, ul);
                }
            }
            if (ax == 0) {                              // the strength: folded into x (real), kept beside (complex)
                float fh[C], fl[C];
#pragma unroll
                for (int c = 0; c < C; c++) {
                    fh[c] = fl[c] = 0.f;
                    if (on) df_bits(f[(size_t)o * C + c], E, fh[c], fl[c]);
                    if (C == 2) {
                        str[(2 * c) * PP_S + pt] = fh[c];
                        str[(2 * c + 1) * PP_S + pt] = fl[c];
                    }
                }
                if (C == 1) {
                    vh = fh[0];
                    vl = fl[0];
                }
            }
            float qh = 0.f, ql = 0.f;                   // e (n / h) d^(e-1)
            for (int e = 0; e < P1; e++) {
                at(ax, 0, e)[pt] = vh;
                at(ax, 1, e)[pt] = vl;
                if (DL) {
                    at(ax, 2, e)[pt] = qh;
                    at(ax, 3, e)[pt] = ql;
                    // next: (e + 1) c v
                    float ah = (float)(e + 1) * ch, al = fmaf((float)(e + 1), ch, -ah) + (float)(e + 1) * cl;
                    df_mul(ah, al, vh, vl);
                    qh = ah;
                    ql = al;
                }
                df_mul(vh, vl, dh, dl);
            }
        }
        __syncthreads();
        if (worker)
            for (int i = 2 * grp; i < nb; i += 2 * groups) {   // points i, i + 1 (strength 0 beyond nb)
                const D2 X{ld2(at(0, 0, m) + i), ld2(at(0, 1, m) + i)}, Y{ld2(at(1, 0, n) + i), ld2(at(1, 1, n) + i)};
                const D2 A = dmul(X, Y);
                D2 B{};
                if (DL) {
                    const D2 XQ{ld2(at(0, 2, m) + i), ld2(at(0, 3, m) + i)}, YQ{ld2(at(1, 2, n) + i), ld2(at(1, 3, n) + i)};
                    B = dadd(dmul(XQ, Y), dmul(X, YQ));
                }
                D2 Af[C], Bf[C];
#pragma unroll
                for (int c = 0; c < C; c++) {
                    if (C == 1) {
                        Af[c] = A;
                        Bf[c] = B;
                    } else {
                        const D2 F{ld2(str + (2 * c) * PP_S + i), ld2(str + (2 * c + 1) * PP_S + i)};
                        Af[c] = dmul(A, F);
                        if (DL) Bf[c] = dmul(B, F);
                    }
                }
#pragma unroll
                for (int k = 0; k < KM; k++) {
                    if (k >= len) break;
                    const D2 Z{ld2(at(2, 0, k) + i), ld2(at(2, 1, k) + i)};
                    if (DL) {
                        const D2 ZQ{ld2(at(2, 2, k) + i), ld2(at(2, 3, k) + i)};
#pragma unroll
                        for (int c = 0; c < C; c++) {
                            dacc(acc[k][c], Af[c], ZQ);
                            dacc(acc[k][c], Bf[c], Z);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < C; c++) dacc(acc[k][c], Af[c], Z);
                    }
                }
            }
    }
    // the groups' sums of every coefficient, then the cluster's
    __syncthreads();
    float2 *red = (float2 *)pp_sm;                      // [group][coefficient][C]
    if (worker)
#pragma unroll
        for (int k = 0; k < KM; k++) {
            if (k >= len) break;
            const int d = deg + k, idx = (d > 0 ? np_of(d - 1) : 0) + (d - m) * (d - m + 1) / 2 + (d - m - n);
#pragma unroll
            for (int c = 0; c < C; c++) {
                float h = acc[k][c].h.x, l = acc[k][c].l.x;
                df_add(h, l, acc[k][c].h.y, acc[k][c].l.y);
                red[((size_t)grp * npl + idx) * C + c] = make_float2(h, l);
            }
        }
    __syncthreads();
    const double unit = scalbn(1.0, E - 1023 - (DL ? es : 0));   // normals were taken over the unit x 2^-es
    // back from the unit to the edge: 2^(reach |a|)
    auto in_edges = [&](double v, int i) {
        return reach ? scalbn(v, reach * (tb.m[i / C] + tb.n[i / C] + tb.k[i / C])) : v;
    };
    for (int i = tid; i < npl * C; i += PP_T) {
        float h = 0.f, l = 0.f;
        for (int g = 0; g < groups; g++) {
            const float2 v = red[(size_t)g * npl * C + i];
            df_add(h, l, v.x, v.y);
        }
        const double v = ((double)h + (double)l) * unit;
        if (ns > 1) share[i] = v;
        else M[(size_t)b * np * C + i] = in_edges(v, i);
    }
    if (ns > 1) {
        cluster_sync();
        if (rank == 0)
            for (int i = tid; i < npl * C; i += PP_T) {
                double v = share[i];
                for (int q = 1; q < ns; q++) v += peer_double(share + i, q);
                M[(size_t)b * np * C + i] = in_edges(v, i);
            }
        cluster_sync();                                 // no block leaves while block 0 reads its share
    }
}

template <int C, bool DL>
int launch(bem_plan *P, const double *f, double *M, cudaStream_t s) {
    const int nl = P->t.nleaf, p = P->mi.p;
    if (nl == 0) return BEM_OK;
    int ns = 1;                                         // two blocks per SM where there are fewer leaves
    while (ns < PP_MAXC && nl * ns < 2 * P->sm_count) ns *= 2;
    const size_t sm = pp_smem(p, C);
    if (p <= 10)
        return launch_cluster(k_p2m_pairs<C, DL, 11>, (unsigned)(nl * ns), PP_T, sm, ns, s, ns, tabs_of(P), view_of(P),
                              quad_of(P), f, M, (const int *)P->skip);
    return launch_cluster(k_p2m_pairs<C, DL, PMAX + 1>, (unsigned)(nl * ns), PP_T, sm, ns, s, ns, tabs_of(P), view_of(P),
                          quad_of(P), f, M, (const int *)P->skip);
}

template <class K>
int allow(K k, int C, int p) {
    BEM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pp_smem(p, C)));
    return BEM_OK;
}

}  // namespace

int p2m_pairs_prepare() {
    BEM_TRY(allow(k_p2m_pairs<1, true, 11>, 1, 10));
    BEM_TRY(allow(k_p2m_pairs<1, false, 11>, 1, 10));
    BEM_TRY(allow(k_p2m_pairs<2, true, 11>, 2, 10));
    BEM_TRY(allow(k_p2m_pairs<2, false, 11>, 2, 10));
    BEM_TRY(allow(k_p2m_pairs<1, true, PMAX + 1>, 1, PMAX));
    BEM_TRY(allow(k_p2m_pairs<1, false, PMAX + 1>, 1, PMAX));
    BEM_TRY(allow(k_p2m_pairs<2, true, PMAX + 1>, 2, PMAX));
    BEM_TRY(allow(k_p2m_pairs<2, false, PMAX + 1>, 2, PMAX));
    return BEM_OK;
}

template <int C>
int launch_p2m_pairs(bem_plan *P, bool dl, const double *f, double *M, cudaStream_t s) {
    return dl ? launch<C, true>(P, f, M, s) : launch<C, false>(P, f, M, s);
}
template int launch_p2m_pairs<1>(bem_plan *, bool, const double *, double *, cudaStream_t);
template int launch_p2m_pairs<2>(bem_plan *, bool, const double *, double *, cudaStream_t);

const void *kernel_of_p2m_f64() { return (const void *)k_p2m_pairs<1, true, 11>; }

}  // namespace bem

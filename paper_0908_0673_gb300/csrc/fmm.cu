// One fast matrix multiplication (Section 3.6, steps 1-4) on the device:
//
//   P2Q  quadrature-point strengths f_q = w_q J_q sum_a L_a(xi_q) x_idx(e,a)
//   P2M  leaf moments I_alpha = sum_q f_q (x_q - c)^alpha            (Eq. 6, monopoles)
//        or sum_q f_q n_q . grad (x_q - c)^alpha                       (dipoles)
//   M2M  coefficient shift child -> parent                            (Eq. 8)
//   M2L  local expansion from the interaction list                     (Eq. 7)
//   L2L  expansion shift parent -> child, with binomials               (Eq. 9)
//   P2P  the regular-rule sum over the elements of the near-field boxes
//   the stored special-pair correction and the diagonal C
//   L2P  local expansion at every vertex of a leaf; it adds the parts up.
//
// Moments and locals are stored scaled by powers of the box edge h:
// Ms_alpha = I_alpha / h^|alpha|, Ls_beta = F_beta h^|beta|, so that every
// shift factor is an exact power of two and float32 storage stays in range.
// Green's-function derivatives come from Tausch's recursions (Section 3.3)
// evaluated per interaction pair at r / h_t.
//
// Templates: R = double (BEM_F64) or float (BEM_MIXED); C = 1 (real, Laplace)
// or 2 (complex, Helmholtz); DL selects dipole (op A) or monopole (op B)
// sources.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "cluster.cuh"
#include "dfloat.cuh"
#include "fmm_views.cuh"

namespace bem {

__constant__ double c_Lq[2][NQ][6];   // shape values at the 7 rule points (tri3, tri6)

// ---------------------------------------------------------------------------
// P2Q
// ---------------------------------------------------------------------------
template <class R, int C>
__global__ void k_p2q(int Q, int npe, const int *__restrict__ el_idx, const double *__restrict__ w,
                      const void *const *__restrict__ xslot, R *__restrict__ f, const int *__restrict__ skip) {
    if (skip && *skip) return;
    int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= Q) return;
    const double *x = (const double *)*xslot;
    int i = o / NQ, q = o - i * NQ, t6 = npe == 6;
    double acc[C];
#pragma unroll
    for (int c = 0; c < C; c++) acc[c] = 0.0;
    for (int a = 0; a < npe; a++) {
        double L = c_Lq[t6][q][a];
        int j = el_idx[(size_t)i * npe + a];
#pragma unroll
        for (int c = 0; c < C; c++) acc[c] += L * x[(size_t)j * C + c];
    }
    double ww = w[o];
#pragma unroll
    for (int c = 0; c < C; c++) f[(size_t)o * C + c] = (R)(ww * acc[c]);
}

// ---------------------------------------------------------------------------
// P2M of float32 plans: one block per leaf, threads over multi-indices, sources
// in batches of 32 (float64 plans: p2m_f64.cu)
// ---------------------------------------------------------------------------
constexpr int P2M_T = 128, P2M_B = 32;
// index slots per thread (NS >= ceil(n_p / P2M_T)): instantiated for orders
// up to 11 (3), 16 (8) and 20 (14)
constexpr int p2m_slots(int np) { return np <= 3 * P2M_T ? 3 : np <= 8 * P2M_T ? 8 : 14; }

// WEIGHTS: instead of the moments, write each point's row of P2M weights
// W[o][a] (the value that multiplies f[o] in moment a) for the stored form.
//
// Per batch of points, shared memory holds for every point and axis the pairs
// (d^e, e n d^(e-1) / h) (d = offset / h, n the normal's component), so a
// monopole coefficient is Px Py Pz and a double-layer one, the normal
// derivative of the monomial, (Qx Py + Px Qy) Pz + Px Py Qz: three paired
// loads and no branches per (point, coefficient).
template <int C, bool DL, bool WEIGHTS, int NS>
__global__ void __launch_bounds__(P2M_T) k_p2m(int nleaf, Tabs tb, TreeView tv, QuadView qv, const float *__restrict__ f,
                                               float *__restrict__ M, const int *__restrict__ skip, float *__restrict__ W = nullptr) {
    using R = float;
    using R2 = float2;
    if (skip && *skip) return;
    const int li = blockIdx.x;
    if (li >= nleaf) return;
    const int b = tv.leaves[li];
    const int np = tb.np, tid = threadIdx.x;
    const int p = order_of(tb, tv.level[b]), npl = np_of(p);   // this leaf's order; np is the stride
    __shared__ R2 pq[3][P2M_B][PMAX + 1];            // [axis][point][power]: (d^e, e n d^(e-1) / h)
    __shared__ R sf[P2M_B][C];
    const double h = scalbn(tv.side, -tv.level[b]);
    const R hinv = (R)(1.0 / h);
    int am[NS], an[NS], ak[NS];
    R acc[NS][C];
#pragma unroll
    for (int s = 0; s < NS; s++) {
        int a = tid + s * P2M_T;
        am[s] = a < npl ? tb.m[a] : 0;
        an[s] = a < npl ? tb.n[a] : 0;
        ak[s] = a < npl ? tb.k[a] : 0;
#pragma unroll
        for (int c = 0; c < C; c++) acc[s][c] = (R)0;
    }
    const int q0 = tv.eb[b] * NQ, q1 = tv.ee[b] * NQ;
    for (int base = q0; base < q1; base += P2M_B) {
        const int nb = min(P2M_B, q1 - base);
        __syncthreads();
        if (tid < 3 * P2M_B) {
            int pt = tid % P2M_B, ax = tid / P2M_B;
            R d = (R)0, nd = (R)0;
            if (pt < nb) {
                int o = base + pt;
                // offsets from the owning leaf (this box) centre
                d = (ax == 0 ? qv.fx[o] : (ax == 1 ? qv.fy[o] : qv.fz[o])) * hinv;
                if (DL) nd = ax == 0 ? qv.fnx[o] : (ax == 1 ? qv.fny[o] : qv.fnz[o]);
            }
            nd *= hinv;
            R v = (R)1, vm = (R)0;                    // d^e, d^(e-1)
            for (int e = 0; e <= p; e++) {
                R2 t;
                t.x = v;
                t.y = DL ? (R)e * nd * vm : (R)0;
                pq[ax][pt][e] = t;
                vm = v;
                v *= d;
            }
        } else if (!WEIGHTS && tid < 3 * P2M_B + P2M_B) {
            int pt = tid - 3 * P2M_B;
            int o = base + pt;
#pragma unroll
            for (int c = 0; c < C; c++) sf[pt][c] = pt < nb ? f[(size_t)o * C + c] : (R)0;
        }
        __syncthreads();
        for (int pt = 0; pt < nb; pt++) {
#pragma unroll
            for (int s = 0; s < NS; s++) {
                if (tid + s * P2M_T >= npl) break;
                const R2 X = pq[0][pt][am[s]], Y = pq[1][pt][an[s]], Z = pq[2][pt][ak[s]];
                const R xy = X.x * Y.x;
                R val;
                if (!DL) val = xy * Z.x;
                else val = xy * Z.y + (X.y * Y.x + X.x * Y.y) * Z.x;
                if (WEIGHTS) {
                    W[(size_t)(base + pt) * np + tid + s * P2M_T] = val;
                } else {
#pragma unroll
                    for (int c = 0; c < C; c++) acc[s][c] += val * sf[pt][c];
                }
            }
        }
    }
    if (WEIGHTS) return;
#pragma unroll
    for (int s = 0; s < NS; s++) {
        int a = tid + s * P2M_T;
        if (a < npl)
#pragma unroll
            for (int c = 0; c < C; c++) M[((size_t)b * np + a) * C + c] = acc[s][c];
    }
}

// ---------------------------------------------------------------------------
// P2M from stored weights (float32 double-layer moments): M[a] = sum over the
// leaf's points of W[o][a] f[o] with W the values the on-the-fly form builds;
// each product only streams the weight rows (coalesced across the indices a),
// two halves of the block taking alternate chunks of points to keep more
// loads in flight.
// ---------------------------------------------------------------------------
constexpr int P2S_T = 2 * P2M_T, P2S_U = 8;           // two halves of P2M_T threads; points per chunk

template <int C, int NS>
__global__ void __launch_bounds__(P2S_T) k_p2m_stored(int nleaf, int np, TreeView tv, const float *__restrict__ W,
                                                      const float *__restrict__ f, float *__restrict__ M,
                                                      const int *__restrict__ skip) {
    if (skip && *skip) return;
    const int li = blockIdx.x;
    if (li >= nleaf) return;
    __shared__ float part[NS][C][P2M_T];
    const int b = tv.leaves[li], half = threadIdx.x / P2M_T, tid = threadIdx.x % P2M_T;
    const int q0 = tv.eb[b] * NQ, q1 = tv.ee[b] * NQ;
    float acc[NS][C];
#pragma unroll
    for (int s = 0; s < NS; s++)
#pragma unroll
        for (int c = 0; c < C; c++) acc[s][c] = 0.f;
    // chunks of P2S_U points alternate between the halves; within a half the
    // points are summed in order, then half 1's sums are added to half 0's
    for (int o0 = q0 + half * P2S_U; o0 < q1; o0 += 2 * P2S_U) {
        const int n = min(P2S_U, q1 - o0);
        float w[P2S_U][NS], fv[P2S_U][C];
#pragma unroll
        for (int u = 0; u < P2S_U; u++) {
            const bool on = u < n;
#pragma unroll
            for (int c = 0; c < C; c++) fv[u][c] = on ? __ldg(f + (size_t)(o0 + u) * C + c) : 0.f;
#pragma unroll
            for (int s = 0; s < NS; s++) {
                const int a = tid + s * P2M_T;
                w[u][s] = on && a < np ? __ldg(W + (size_t)(o0 + u) * np + a) : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < P2S_U; u++)
#pragma unroll
            for (int s = 0; s < NS; s++)
#pragma unroll
                for (int c = 0; c < C; c++) acc[s][c] += w[u][s] * fv[u][c];
    }
    if (half == 1)
#pragma unroll
        for (int s = 0; s < NS; s++)
#pragma unroll
            for (int c = 0; c < C; c++) part[s][c][tid] = acc[s][c];
    __syncthreads();
    if (half == 0)
#pragma unroll
        for (int s = 0; s < NS; s++) {
            const int a = tid + s * P2M_T;
            if (a < np)
#pragma unroll
                for (int c = 0; c < C; c++) M[((size_t)b * np + a) * C + c] = acc[s][c] + part[s][c][tid];
        }
}


// P2M launches with the slot count of the plan's largest order
template <int C, bool DL, bool WEIGHTS = false>
static void launch_p2m(int nleaf, const Tabs &tb, const TreeView &tv, const QuadView &qv, const float *f, float *M,
                       const int *skip, cudaStream_t s, float *W = nullptr) {
    const int ns = p2m_slots(tb.np);
    if (ns == 3) (k_p2m<C, DL, WEIGHTS, 3><<<nleaf, P2M_T, 0, s>>>(nleaf, tb, tv, qv, f, M, skip, W), ::bem::count_launch());
    else if (ns == 8) (k_p2m<C, DL, WEIGHTS, 8><<<nleaf, P2M_T, 0, s>>>(nleaf, tb, tv, qv, f, M, skip, W), ::bem::count_launch());
    else (k_p2m<C, DL, WEIGHTS, 14><<<nleaf, P2M_T, 0, s>>>(nleaf, tb, tv, qv, f, M, skip, W), ::bem::count_launch());
}

template <int C>
static void launch_p2m_stored(int nleaf, int np, const TreeView &tv, const float *W, const float *f, float *M,
                              const int *skip, cudaStream_t s) {
    const int ns = p2m_slots(np);
    if (ns == 3) (k_p2m_stored<C, 3><<<nleaf, P2S_T, 0, s>>>(nleaf, np, tv, W, f, M, skip), ::bem::count_launch());
    else if (ns == 8) (k_p2m_stored<C, 8><<<nleaf, P2S_T, 0, s>>>(nleaf, np, tv, W, f, M, skip), ::bem::count_launch());
    else (k_p2m_stored<C, 14><<<nleaf, P2S_T, 0, s>>>(nleaf, np, tv, W, f, M, skip), ::bem::count_launch());
}

// ---------------------------------------------------------------------------
// near field (regular rule over the near-list boxes), float64 arithmetic:
// Helmholtz plans whose phases exceed the table of the float32-pair kernel
// (near_f64.cu), which takes every other float64 product
// ---------------------------------------------------------------------------
constexpr int NF_T = 256, NF_TGT = 64, NF_SL = NF_T / NF_TGT, NF_TILE = 256;

template <bool DL>
__device__ __forceinline__ void pair_f64(double rx, double ry, double rz, double nx, double ny, double nz,
                                         const double *fv, double kw, double *acc) {
    const double r2 = rx * rx + ry * ry + rz * rz, inv = rsqrt(r2), R1 = r2 * inv;
    double sn, cs, gr, gi;
    sincos(kw * R1, &sn, &cs);
    if (DL) {
        const double kr = kw * R1, rn = (rx * nx + ry * ny + rz * nz) * inv * inv * inv;
        gr = (cs + kr * sn) * rn;
        gi = (sn - kr * cs) * rn;
    } else {
        gr = cs * inv;
        gi = sn * inv;
    }
    acc[0] += gr * fv[0] - gi * fv[1];
    acc[1] += gr * fv[1] + gi * fv[0];
}

template <bool DL>
__global__ void __launch_bounds__(NF_T) k_near(int nleaf, TreeView tv, QuadView qv, double kw,
                                               const double *__restrict__ f, double *__restrict__ ytmp,
                                               const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int C = 2;
    const int li = blockIdx.x;
    if (li >= nleaf) return;
    const int b = tv.leaves[li];
    const int tid = threadIdx.x, tt = tid % NF_TGT, sl = tid / NF_TGT;
    __shared__ double sx[NF_TILE], sy[NF_TILE], sz[NF_TILE], snx[NF_TILE], sny[NF_TILE], snz[NF_TILE];
    __shared__ double sf[NF_TILE][C];
    __shared__ double red[NF_T][C];
    const double cbx = tv.cx[b], cby = tv.cy[b], cbz = tv.cz[b];
    for (int t0 = tv.nb[b]; t0 < tv.ne[b]; t0 += NF_TGT) {
        const int tk = t0 + tt;
        const bool active = tk < tv.ne[b];
        const double tx = active ? tv.tx[tk] : cbx, ty = active ? tv.ty[tk] : cby, tz = active ? tv.tz[tk] : cbz;
        double acc[C] = {0.0, 0.0};
        for (int u = tv.near_ptr[b]; u < tv.near_ptr[b + 1]; u++) {
            const int s = tv.near_idx[u];
            const int q0 = tv.eb[s] * NQ, q1 = tv.ee[s] * NQ;
            double part[C] = {0.0, 0.0};
            for (int base = q0; base < q1; base += NF_TILE) {
                const int nt = min(NF_TILE, q1 - base);
                __syncthreads();
                if (tid < nt) {
                    const int o = base + tid;
                    sx[tid] = qv.x[o]; sy[tid] = qv.y[o]; sz[tid] = qv.z[o];
                    if (DL) { snx[tid] = qv.nx[o]; sny[tid] = qv.ny[o]; snz[tid] = qv.nz[o]; }
                    sf[tid][0] = f[(size_t)o * C];
                    sf[tid][1] = f[(size_t)o * C + 1];
                }
                __syncthreads();
                if (active)
                    for (int j = sl; j < nt; j += NF_SL)
                        pair_f64<DL>(tx - sx[j], ty - sy[j], tz - sz[j], DL ? snx[j] : 0.0, DL ? sny[j] : 0.0,
                                     DL ? snz[j] : 0.0, sf[j], kw, part);
            }
            acc[0] += part[0];
            acc[1] += part[1];
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < C; c++) red[tid][c] = acc[c] * (0.25 / M_PI);
        __syncthreads();
        if (sl == 0 && active) {
            double s[C] = {red[tid][0], red[tid][1]};
            for (int u = 1; u < NF_SL; u++)
#pragma unroll
                for (int c = 0; c < C; c++) s[c] += red[tid + u * NF_TGT][c];
            const int node = tv.node_perm[tk];
#pragma unroll
            for (int c = 0; c < C; c++) ytmp[(size_t)node * C + c] = s[c];
        }
    }
}


// ---------------------------------------------------------------------------
// near field, float32 form.  A block takes one leaf and up to 64 of
// its targets per pass: G = ceil(targets / U) target groups x (256 / G)
// source slices, each thread holding U targets (8 real, 4 complex) so that
// every source read from shared memory serves U pairs.  The near-list
// sources are packed into full tiles across box boundaries; each staged
// source is rebased to the target leaf's centre (box offset in float64,
// rounded once).  Pairs run two targets to a packed instruction.  For the real
// double layer the strength is folded into the staged normal, so a pair costs 3
// subtractions, two 3-term dot products, one reciprocal square root and three
// multiplies.  Complex pairs (33 packed operations) take e^{jkr} from a table of
// the unit circle and the first two terms of the rest (sincosf cost more than
// the rest of the pair: sphere of 20,480 tri6 738 -> 573 us, of 81,920 3142 ->
// 2290, FMA pipe 65 % busy).  Tile partial sums are added with compensation,
// slices as float32 pairs.
// ---------------------------------------------------------------------------
constexpr int NF2_T = 256, NF2_ENT = 256, NF2_SLOTS = 64, NF2_MAXC = 8;
__host__ __device__ constexpr int nf2_u(int C) { return C == 1 ? 8 : 4; }
// Complex pairs take e^{jkr} from a table of the unit circle (TAB): 1,024 steps
// leave an angle below 3.1e-3, whose sine is itself to 2^-27.  k r in table steps
// must stay below 2^22, where adding 1.5 2^23 still rounds to the index; plans
// beyond it (k x side above 1,600) take sincosf.
constexpr int NF2_TAB = 1024;
constexpr double NF2_MAXPHASE = 4194304.0;
// A cluster of up to NF2_MAXC blocks shares an item's sources and expansion terms
// where items would not fill two waves of three blocks per SM (59 -> 34 us for 72
// leaves, 121 -> 76 for 56 complex ones); the kernel without the cluster's code
// is the faster one where they do (429 against 444 us for 1,180 items).
constexpr int NF2_WAVES = 2;
// sources staged per round, and float4 of each: packed forms hold every value
// twice, for the two targets of a float2 operation.  Real: 1024 per round, three
// blocks per SM (0.437 ms against 0.456 for 640 at four blocks on the cube
// workload, the rounds' barriers and staging halved).
__host__ __device__ constexpr int nf2_tile(int C, bool TAB) { return C == 2 && TAB ? 640 : 1024; }
__host__ __device__ constexpr int nf2_stage(int C, bool TAB) { return nf2_tile(C, TAB) * (C == 1 ? 3 : TAB ? 4 : 2); }

// Work items of the near field: one per (leaf, pass of up to NF2_SLOTS targets,
// ND_SLOTS in float64 plans), ordered by decreasing pair count (targets x near sources, ties in
// leaf order), so the largest blocks start first and the last wave is made of
// the smallest.  Each target is summed by one block whatever the order.  Uploads
// go to the stream of the first product (the diagonal's; pageable sources, staged
// before the calls return).
int build_near_items(bem_plan *P, cudaStream_t s) {
    const Tree &t = P->t;
    std::vector<int> nptr(t.nbox + 1), nidx(std::max<int64_t>(1, t.n_near)), nb(t.nbox), ne(t.nbox), eb(t.nbox),
        ee(t.nbox), lv(t.nleaf);
    BEM_CUDA(cudaMemcpy(nptr.data(), t.near_ptr, sizeof(int) * (t.nbox + 1), cudaMemcpyDeviceToHost));
    if (t.n_near) BEM_CUDA(cudaMemcpy(nidx.data(), t.near_idx, sizeof(int) * t.n_near, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(nb.data(), t.nb, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(ne.data(), t.ne, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(eb.data(), t.eb, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(ee.data(), t.ee, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(lv.data(), t.leaves, sizeof(int) * t.nleaf, cudaMemcpyDeviceToHost));
    // A literal list (leaf_descend = 0) may hold non-leaf boxes.  The float64
    // near field takes a source's position from its own leaf's centre, so such
    // an entry becomes its subtree's leaves, in element order.
    if (!P->prm.leaf_descend) {
        std::vector<int> child0(t.nbox), nchild(t.nbox), ptr(t.nbox + 1, 0), idx, stack;
        BEM_CUDA(cudaMemcpy(child0.data(), t.child0, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
        BEM_CUDA(cudaMemcpy(nchild.data(), t.nchild, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
        for (int b = 0; b < t.nbox; b++) {
            if (nchild[b] == 0)                       // only leaves are targets
                for (int u = nptr[b]; u < nptr[b + 1]; u++) {
                    stack.push_back(nidx[u]);
                    while (!stack.empty()) {
                        const int s = stack.back();
                        stack.pop_back();
                        if (nchild[s] == 0) idx.push_back(s);
                        for (int q = nchild[s] - 1; q >= 0; q--) stack.push_back(child0[s] + q);
                    }
                }
            ptr[b + 1] = (int)idx.size();
        }
        BEM_TRY(P->arena.alloc(&P->leaf_near_ptr, ptr.size()));
        BEM_TRY(P->arena.alloc(&P->leaf_near_idx, idx.size()));
        BEM_CUDA(cudaMemcpyAsync(P->leaf_near_ptr, ptr.data(), sizeof(int) * ptr.size(), cudaMemcpyHostToDevice, s));
        if (!idx.empty())
            BEM_CUDA(cudaMemcpyAsync(P->leaf_near_idx, idx.data(), sizeof(int) * idx.size(), cudaMemcpyHostToDevice, s));
    }
    int64_t pairs = 0;
    std::vector<int64_t> src(t.nleaf);
    for (int li = 0; li < t.nleaf; li++) {
        const int b = lv[li];
        int64_t n = 0;
        for (int u = nptr[b]; u < nptr[b + 1]; u++) n += (int64_t)(ee[nidx[u]] - eb[nidx[u]]) * NQ;
        src[li] = n;
        pairs += n * (ne[b] - nb[b]);
    }
    P->near_pairs = pairs;
    // real items for every plan (the diagonal's product is Laplace), complex
    // ones for Helmholtz plans only
    for (int v = 0; v < (P->green == BEM_HELMHOLTZ ? 2 : 1); v++) {
        const int slots = P->prm.precision == BEM_MIXED ? NF2_SLOTS : ND_SLOTS;
        std::vector<int2> items;
        std::vector<int64_t> cost;
        for (int li = 0; li < t.nleaf; li++) {
            const int b = lv[li];
            for (int t0 = nb[b]; t0 < ne[b]; t0 += slots) {
                items.push_back(make_int2(li, t0));
                cost.push_back((int64_t)std::min(slots, ne[b] - t0) * src[li]);
            }
        }
        std::vector<int> ord(items.size());
        for (size_t i = 0; i < ord.size(); i++) ord[i] = (int)i;
        std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return cost[x] > cost[y]; });
        std::vector<int2> sorted(std::max<size_t>(1, items.size()));
        for (size_t i = 0; i < ord.size(); i++) sorted[i] = items[ord[i]];
        BEM_TRY(P->arena.alloc(&P->near_items[v], sorted.size()));
        BEM_CUDA(cudaMemcpyAsync(P->near_items[v], sorted.data(), sizeof(int2) * sorted.size(), cudaMemcpyHostToDevice, s));
        P->near_nitems[v] = (int)items.size();
    }
    return BEM_OK;
}

// 1 / sqrt(x) as the single hardware approximation (flush-to-zero form: the
// squared distances of near-field pairs are never subnormal)
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int C, bool DL>
__device__ __forceinline__ void pair_f32(float rx, float ry, float rz, const float4 &sa, const float4 &sb, float kw,
                                         float *acc) {
    const float r2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
    const float inv = rsqrt_ftz(r2);
    if (C == 1) {
        if (DL) {   // sb = strength * normal
            const float dot = fmaf(rx, sb.x, fmaf(ry, sb.y, rz * sb.z));
            acc[0] = fmaf(dot * inv, inv * inv, acc[0]);
        } else {
            acc[0] = fmaf(sa.w, inv, acc[0]);
        }
    } else {
        const float R1 = r2 * inv;
        float sn, cs;
        sincosf(kw * R1, &sn, &cs);
        float gr, gi;
        if (DL) {
            const float kr = kw * R1, rn = fmaf(rx, sb.x, fmaf(ry, sb.y, rz * sb.z)) * inv * inv * inv;
            gr = (cs + kr * sn) * rn;
            gi = (sn - kr * cs) * rn;
        } else {
            gr = cs * inv;
            gi = sn * inv;
        }
        acc[0] += gr * sa.w - gi * sb.w;
        acc[C - 1] += gr * sb.w + gi * sa.w;
    }
}

// compensated float32 accumulation (Kahan): GB300's float64 pipe is a small
// fraction of its float32 pipe, so long sums stay in float32 with a carried
// error term instead of being promoted
struct KahanF {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c, t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

// shared memory of the float32 near field beyond its static part: the staged
// sources (sa, sb) and the per-thread compensated sums
__host__ __device__ constexpr size_t nf2_dyn_bytes(int C, bool TAB) {
    return (size_t)nf2_stage(C, TAB) * sizeof(float4) + 2 * (size_t)nf2_u(C) * C * NF2_T * sizeof(float) +
           (C == 2 && TAB ? NF2_TAB * sizeof(float2) : 0);
}

template <int C, bool DL, bool TAB, bool CL>
__global__ void __launch_bounds__(NF2_T, C == 1 || TAB ? 3 : 4)
    k_near_f32(int ns_, const int2 *__restrict__ items, TreeView tv, QuadView qv, double kwave,
               const float *__restrict__ f, double *__restrict__ ytmp,
               const float *__restrict__ wave, const int *__restrict__ skip) {
    constexpr int U = nf2_u(C);                       // targets per thread
    constexpr int SLOTS = NF2_SLOTS;                  // targets per pass (at most SLOTS / U groups)
    constexpr int UC = U * C;
    constexpr int TILE = nf2_tile(C, TAB);            // sources staged per round
    if (skip && *skip) return;                        // every block of the cluster reads the same word
    const int ns = CL ? ns_ : 1, rank = CL ? (int)cluster_rank() : 0;
    const int2 item = items[blockIdx.x / ns];         // (leaf, first target of the pass)
    const int b = tv.leaves[item.x];
    const int tid = threadIdx.x, lane = tid & 31;
    // The staged-source region is reused for the slices' sums once the sources are done.
    extern __shared__ float4 near_tile[];
    float4 *sa = near_tile, *sb = near_tile + TILE;                     // sincosf form: position | Re f, normal | Im f
    float4 *s0 = near_tile, *s1 = s0 + TILE, *s2 = s1 + TILE, *s3 = s2 + TILE;   // packed forms (see the staging)
    float *ks = (float *)(near_tile + nf2_stage(C, TAB));   // [UC][NF2_T] compensated sums
    float *kc = ks + UC * NF2_T;                      // [UC][NF2_T] their carries
    float *red = (float *)near_tile;                  // [slice][slot][C]
    __shared__ int pref[NF2_ENT + 1];
    __shared__ int ebase[NF2_ENT];                    // first quadrature point of each entry's box
    __shared__ float eoff[NF2_ENT][3];                // entry box centre - target leaf centre
    __shared__ float toff[SLOTS][3];                  // target - target leaf centre
    __shared__ double share[SLOTS][C];                // this block's sums, for the cluster's first
    const double cbx = tv.cx[b], cby = tv.cy[b], cbz = tv.cz[b];
    const float kw = (float)kwave;
    float *sw = kc + UC * NF2_T;                      // the unit circle: cosines, then sines
    const double ktd = kwave * (NF2_TAB / (2.0 * M_PI));
    const float kt = (float)ktd, ktl = (float)(ktd - (double)kt);   // k in table steps per length
    if (C == 2 && TAB)
        for (int i = tid; i < 2 * NF2_TAB; i += NF2_T) sw[i] = wave[i];
    const int t0 = item.y, nt = min(SLOTS, tv.ne[b] - t0);
    const int G = (nt + U - 1) / U, S = NF2_T / G, tg = tid % G, sl = tid / G;
    const bool worker = sl < S;
    if (tid < SLOTS) {
        const int k = t0 + tid;
        const bool on = tid < nt;
        toff[tid][0] = on ? (float)(tv.tx[k] - cbx) : 0.f;
        toff[tid][1] = on ? (float)(tv.ty[k] - cby) : 0.f;
        toff[tid][2] = on ? (float)(tv.tz[k] - cbz) : 1.f;   // off targets stay away from every source
    }
    for (int i = tid; i < 2 * UC * NF2_T; i += NF2_T) ks[i] = 0.f;
    __syncthreads();
    float tx[U], ty[U], tz[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int slot = tg + G * u;                 // < G U <= SLOTS
        tx[u] = toff[slot][0];
        ty[u] = toff[slot][1];
        tz[u] = toff[slot][2];
    }
    for (int e0 = tv.near_ptr[b]; e0 < tv.near_ptr[b + 1]; e0 += NF2_ENT) {
        const int ne_ = min(NF2_ENT, tv.near_ptr[b + 1] - e0);
        __syncthreads();
        if (tid < 32) {                               // quadrature-point offsets of the entries (warp scan)
            int carry = 0;
            for (int i0 = 0; i0 < ne_; i0 += 32) {
                const int i = i0 + lane;
                int x = 0;
                if (i < ne_) {
                    const int s = tv.near_idx[e0 + i];
                    x = (tv.ee[s] - tv.eb[s]) * NQ;
                    ebase[i] = tv.eb[s] * NQ;
                    eoff[i][0] = (float)(tv.cx[s] - cbx);
                    eoff[i][1] = (float)(tv.cy[s] - cby);
                    eoff[i][2] = (float)(tv.cz[s] - cbz);
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (i < ne_) pref[i + 1] = carry + x;
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) pref[0] = 0;
        }
        __syncthreads();
        // this block's share of the chunk's sources
        const int j0 = (int)((long long)pref[ne_] * rank / ns), j1 = (int)((long long)pref[ne_] * (rank + 1) / ns);
        for (int base = j0; base < j1; base += TILE) {
            __syncthreads();
            int lo = 0;                               // entry holding j: pref[lo] <= j < pref[lo + 1]
            if (base + tid < j1) {
                int hi = ne_ - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pref[mid] <= base + tid) lo = mid; else hi = mid - 1;
                }
            }
            for (int jj = tid; jj < TILE; jj += NF2_T) {
                const int j = base + jj;
                if (j >= j1) break;
                while (pref[lo + 1] <= j) lo++;       // j grows with jj: the entry only moves forward
                const int o = ebase[lo] + (j - pref[lo]);
                const float4 xa = make_float4(eoff[lo][0] + qv.fx[o], eoff[lo][1] + qv.fy[o], eoff[lo][2] + qv.fz[o], 0.f);
                if constexpr (C == 1) {
                    // packed layout: each value twice, for the two targets of a float2
                    // operation; positions negated so that r = t + (-a)
                    const float fo = f[o];
                    s0[jj] = make_float4(-xa.x, -xa.x, -xa.y, -xa.y);
                    if (DL) {
                        const float nx = fo * qv.fnx[o], ny = fo * qv.fny[o], nz = fo * qv.fnz[o];
                        s1[jj] = make_float4(-xa.z, -xa.z, nx, nx);
                        s2[jj] = make_float4(ny, ny, nz, nz);
                    } else {
                        s1[jj] = make_float4(-xa.z, -xa.z, fo, fo);
                    }
                } else if constexpr (TAB) {
                    const float fr = f[(size_t)o * C], fi = f[(size_t)o * C + 1];
                    s0[jj] = make_float4(-xa.x, -xa.x, -xa.y, -xa.y);
                    s1[jj] = make_float4(-xa.z, -xa.z, fr, fr);
                    if (DL) {
                        const float nx = qv.fnx[o], ny = qv.fny[o], nz = qv.fnz[o];
                        s2[jj] = make_float4(fi, fi, nx, nx);
                        s3[jj] = make_float4(ny, ny, nz, nz);
                    } else {
                        s2[jj] = make_float4(fi, fi, 0.f, 0.f);
                    }
                } else {
                    sa[jj] = make_float4(xa.x, xa.y, xa.z, f[(size_t)o * C]);
                    sb[jj] = make_float4(DL ? qv.fnx[o] : 0.f, DL ? qv.fny[o] : 0.f, DL ? qv.fnz[o] : 0.f,
                                         C == 2 ? f[(size_t)o * C + C - 1] : 0.f);
                }
            }
            __syncthreads();
            const int nq = min(TILE, j1 - base);
            float part[U][C];
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int c = 0; c < C; c++) part[u][c] = 0.f;
            if constexpr (C == 1) {
                // two targets per packed float32 operation (__fadd2 / __fmul2 / __ffma2):
                // half the issue slots of the scalar form, same roundings in the same order
                float2 t2x[U / 2], t2y[U / 2], t2z[U / 2], p2[U / 2];
#pragma unroll
                for (int v = 0; v < U / 2; v++) {
                    t2x[v] = make_float2(tx[2 * v], tx[2 * v + 1]);
                    t2y[v] = make_float2(ty[2 * v], ty[2 * v + 1]);
                    t2z[v] = make_float2(tz[2 * v], tz[2 * v + 1]);
                    p2[v] = make_float2(0.f, 0.f);
                }
                auto source = [&](int q) {
                    const float4 a0 = s0[q], a1 = s1[q];
                    const float2 mx = make_float2(a0.x, a0.y), my = make_float2(a0.z, a0.w), mz = make_float2(a1.x, a1.y);
                    float2 nx, ny, nz;
                    if (DL) {
                        const float4 a2 = s2[q];
                        nx = make_float2(a1.z, a1.w);
                        ny = make_float2(a2.x, a2.y);
                        nz = make_float2(a2.z, a2.w);
                    }
#pragma unroll
                    for (int v = 0; v < U / 2; v++) {
                        const float2 rx = __fadd2_rn(t2x[v], mx), ry = __fadd2_rn(t2y[v], my), rz = __fadd2_rn(t2z[v], mz);
                        float2 r2 = __fmul2_rn(rz, rz);
                        r2 = __ffma2_rn(ry, ry, r2);
                        r2 = __ffma2_rn(rx, rx, r2);
                        const float2 inv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
                        if (DL) {
                            float2 dot = __fmul2_rn(rz, nz);
                            dot = __ffma2_rn(ry, ny, dot);
                            dot = __ffma2_rn(rx, nx, dot);
                            p2[v] = __ffma2_rn(__fmul2_rn(dot, inv), __fmul2_rn(inv, inv), p2[v]);
                        } else {
                            p2[v] = __ffma2_rn(make_float2(a1.z, a1.w), inv, p2[v]);
                        }
                    }
                };
                if (worker) {
                    int q = sl;
                    for (; q + S < nq; q += 2 * S) {
                        source(q);
                        source(q + S);
                    }
                    if (q < nq) source(q);
                }
#pragma unroll
                for (int v = 0; v < U / 2; v++) {
                    part[2 * v][0] = p2[v].x;
                    part[2 * v + 1][0] = p2[v].y;
                }
            } else if constexpr (TAB) {
                // packed as the real form; e^{jkr} = table entry times the small rest
                float2 t2x[U / 2], t2y[U / 2], t2z[U / 2], pr[U / 2], pi[U / 2];
#pragma unroll
                for (int v = 0; v < U / 2; v++) {
                    t2x[v] = make_float2(tx[2 * v], tx[2 * v + 1]);
                    t2y[v] = make_float2(ty[2 * v], ty[2 * v + 1]);
                    t2z[v] = make_float2(tz[2 * v], tz[2 * v + 1]);
                    pr[v] = pi[v] = make_float2(0.f, 0.f);
                }
                if (worker)
                    for (int q = sl; q < nq; q += S) {
                        const float4 a0 = s0[q], a1 = s1[q], a2 = s2[q];
                        const float2 mx = make_float2(a0.x, a0.y), my = make_float2(a0.z, a0.w), mz = make_float2(a1.x, a1.y),
                                     fr = make_float2(a1.z, a1.w), fi = make_float2(a2.x, a2.y);
                        float2 nx, ny, nz;
                        if (DL) {
                            const float4 a3 = s3[q];
                            nx = make_float2(a2.z, a2.w);
                            ny = make_float2(a3.x, a3.y);
                            nz = make_float2(a3.z, a3.w);
                        }
#pragma unroll
                        for (int v = 0; v < U / 2; v++) {
                            const float2 rx = padd(t2x[v], mx), ry = padd(t2y[v], my), rz = padd(t2z[v], mz);
                            const float2 r2 = pfma(rx, rx, pfma(ry, ry, pmul(rz, rz)));
                            const float2 inv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)), R1 = pmul(r2, inv);
                            // k r = j + d table steps, both exact products: adding 1.5 2^23 rounds to j
                            const float2 jf = pfma(p2(kt), R1, p2(12582912.f)), nj = psub(p2(12582912.f), jf);
                            const float2 d = pfma(p2(ktl), R1, pfma(p2(kt), R1, nj));
                            const int i0 = __float_as_int(jf.x) & (NF2_TAB - 1), i1 = __float_as_int(jf.y) & (NF2_TAB - 1);
                            const float2 Cs = make_float2(sw[i0], sw[i1]), Sn = make_float2(sw[NF2_TAB + i0], sw[NF2_TAB + i1]);
                            // e^{jg} = (1 - g^2 / 2) + j g to 2^-27, g = d 2 pi / 1024
                            constexpr float st = (float)(2.0 * M_PI / NF2_TAB);
                            const float2 g = pmul(d, p2(st)), q1 = pfma(pmul(d, d), p2(-0.5f * st * st), p2(1.f));
                            const float2 cs = pfma(Cs, q1, pmul(Sn, pxneg(g))), sn = pfma(Sn, q1, pmul(Cs, g));
                            // H = (1 - j k r) (r . n) / r^3 f, or f / r; then times cs + j sn
                            float2 hr, hi;
                            if (DL) {
                                const float2 dot = pfma(rx, nx, pfma(ry, ny, pmul(rz, nz)));
                                const float2 w = pmul(pmul(dot, inv), pmul(inv, inv));
                                const float2 gr = pmul(fr, w), gi = pmul(fi, w), kr = pmul(p2(kw), R1);
                                hr = pfma(kr, gi, gr);
                                hi = pfma(kr, pxneg(gr), gi);
                            } else {
                                hr = pmul(fr, inv);
                                hi = pmul(fi, inv);
                            }
                            pr[v] = pfma(cs, hr, pr[v]);
                            pi[v] = pfma(cs, hi, pi[v]);
                            pr[v] = pfma(pxneg(sn), hi, pr[v]);
                            pi[v] = pfma(sn, hr, pi[v]);
                        }
                    }
#pragma unroll
                for (int v = 0; v < U / 2; v++) {
                    part[2 * v][0] = pr[v].x;
                    part[2 * v + 1][0] = pr[v].y;
                    part[2 * v][C - 1] = pi[v].x;
                    part[2 * v + 1][C - 1] = pi[v].y;
                }
            } else if (worker) {
                // two sources per iteration (fewer loop instructions, more independent work)
                const float4 *pa = sa + sl, *pb = sb + sl;
                int q = sl;
                for (; q + S < nq; q += 2 * S, pa += 2 * S, pb += 2 * S) {
                    const float4 A0 = pa[0], B0 = pb[0], A1 = pa[S], B1 = pb[S];
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        pair_f32<C, DL>(tx[u] - A0.x, ty[u] - A0.y, tz[u] - A0.z, A0, B0, kw, part[u]);
                        pair_f32<C, DL>(tx[u] - A1.x, ty[u] - A1.y, tz[u] - A1.z, A1, B1, kw, part[u]);
                    }
                }
                if (q < nq) {
                    const float4 A = pa[0], Bv = pb[0];
#pragma unroll
                    for (int u = 0; u < U; u++)
                        pair_f32<C, DL>(tx[u] - A.x, ty[u] - A.y, tz[u] - A.z, A, Bv, kw, part[u]);
                }
            }
            // tile partials into the compensated sums (Kahan), kept in shared memory
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int c = 0; c < C; c++) {
                    const int i = (u * C + c) * NF2_T + tid;
                    const float s = ks[i], y = part[u][c] - kc[i], t = s + y;
                    kc[i] = (t - s) - y;
                    ks[i] = t;
                }
        }
    }
    __syncthreads();                                  // sources done: their region is reused below
    if (worker)
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
            for (int c = 0; c < C; c++) red[((size_t)sl * G * U + tg + G * u) * C + c] = ks[(u * C + c) * NF2_T + tid];
    __syncthreads();
    {
        // four threads per target add every fourth slice (target t0 + slot sits in
        // place slot = tg + G u of each), then each other's sums
        static_assert(NF2_T == 4 * SLOTS, "four threads per target");
        const int slot = tid >> 2, q0 = tid & 3;
#pragma unroll
        for (int c = 0; c < C; c++) {
            KahanF k;
            if (slot < nt)
                for (int q = q0; q < S; q += 4) k.add(red[((size_t)q * G * U + slot) * C + c]);
            // float32 pairs (few float64 operations: 1 / 64 of the rate)
            float h = k.s, l = -k.c;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1)
                df_add(h, l, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
            if (q0 == 0) share[slot][c] = ((double)h + (double)l) * (0.25 / M_PI);
        }
    }
    if (CL) cluster_sync(); else __syncthreads();
    if (rank == 0 && tid < nt) {
        const int node = tv.node_perm[t0 + tid];
#pragma unroll
        for (int c = 0; c < C; c++) {
            double y = share[tid][c];
            for (int q = 1; q < ns; q++) y += peer_double(&share[tid][c], q);
            ytmp[(size_t)node * C + c] = y;
        }
    }
    if (CL) cluster_sync();                           // no block leaves while block 0 reads its share
}

// ---------------------------------------------------------------------------
// L2P: the local expansion at the targets of a leaf (the near field's work
// items).  256 / SLOTS threads per target share its rows (m, n) of polynomials
// in z (Horner), float32 rows added with compensation.  It ends a product and
// alone writes its output, which may be the input's memory, when every other
// part has been summed from the input:
//   out = corr - (near + far)
// (out null: near += far, the diagonal's regular sums).
// ---------------------------------------------------------------------------
constexpr int L2P_T = 256;
template <class R, int C, int SLOTS>
__global__ void __launch_bounds__(L2P_T) k_l2p(const int2 *__restrict__ items, Tabs tb, TreeView tv,
                                               const int *__restrict__ mexp, double inv_side, const R *__restrict__ L,
                                               double *__restrict__ near, const double *__restrict__ corr,
                                               void *const *__restrict__ yslot, const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int PARTS = L2P_T / SLOTS, W = sizeof(R) == sizeof(float) ? 2 : 1;
    extern __shared__ __align__(16) unsigned char l2p_sm[];
    __shared__ R px[PMAX + 1][SLOTS], py[PMAX + 1][SLOTS], pz[SLOTS];
    __shared__ R red[PARTS][SLOTS][C][W];
    R *sL = (R *)l2p_sm;                              // [np of the leaf's order][C], row (m, n) by row, k ascending
    __shared__ short rows[(PMAX + 1) * (PMAX + 2) / 2][2];   // m | n << 8, first coefficient
    const int2 item = items[blockIdx.x];
    const int b = tv.leaves[item.x], tid = threadIdx.x, slot = tid % SLOTS, part = tid / SLOTS;
    const int t0 = item.y, nt = min(SLOTS, tv.ne[b] - t0), k = t0 + (slot < nt ? slot : 0);
    const int p = order_of(tb, tv.level[b]), npl = np_of(p);
    auto row_at = [&](int m, int n) { return npl - np_of(p - m) + n * (p - m + 1) - n * (n - 1) / 2; };
    for (int i = tid; i < npl; i += L2P_T) {
        const int e = __ldg(mexp + i), m = e & 255, n = e >> 8 & 255, at = row_at(m, n) + (e >> 16 & 255);
#pragma unroll
        for (int c = 0; c < C; c++) sL[at * C + c] = L[((size_t)b * tb.np + i) * C + c];
        if ((e >> 16 & 255) == 0) {                   // rows in order of m, then n
            const int r = m * (p + 1) - m * (m - 1) / 2 + n;
            rows[r][0] = (short)(m | n << 8);
            rows[r][1] = (short)at;
        }
    }
    if (part < 3) {
        const double ih = scalbn(inv_side, tv.level[b]);      // 1 / edge of the leaf
        const R d = (R)((part == 0 ? tv.tx[k] - tv.cx[b] : part == 1 ? tv.ty[k] - tv.cy[b] : tv.tz[k] - tv.cz[b]) * ih);
        if (part == 2) {
            pz[slot] = d;
        } else {
            R (*pw)[SLOTS] = part ? py : px, v = (R)1;
            for (int e = 0; e <= p; e++) {
                pw[e][slot] = v;
                v *= d;
            }
        }
    }
    __syncthreads();
    const R z = pz[slot];
    const int nrow = (p + 1) * (p + 2) / 2;
    R sum[C], car[C];
#pragma unroll
    for (int c = 0; c < C; c++) sum[c] = car[c] = (R)0;
    for (int r = part; r < nrow; r += PARTS) {
        const int mn = rows[r][0], m = mn & 255, n = mn >> 8;
        const R *a = sL + rows[r][1] * C;
        R v[C];
#pragma unroll
        for (int c = 0; c < C; c++) v[c] = (R)0;
#pragma unroll 4
        for (int e = p - m - n; e >= 0; e--)
#pragma unroll
            for (int c = 0; c < C; c++) v[c] = fma(v[c], z, a[e * C + c]);
        const R xy = px[m][slot] * py[n][slot];
#pragma unroll
        for (int c = 0; c < C; c++) {
            if constexpr (sizeof(R) == sizeof(float)) {
                const R a = __fmaf_rn(v[c], xy, -car[c]), t = __fadd_rn(sum[c], a);
                car[c] = __fsub_rn(__fsub_rn(t, sum[c]), a);
                sum[c] = t;
            } else {
                sum[c] = fma(v[c], xy, sum[c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < C; c++) {
        red[part][slot][c][0] = sum[c];
        if constexpr (W == 2) red[part][slot][c][1] = -car[c];
    }
    __syncthreads();
    double *out = yslot ? (double *)*yslot : nullptr;
    for (int i = tid; i < nt * C; i += L2P_T) {
        const size_t at = (size_t)tv.node_perm[t0 + i / C] * C + i % C;
        double v;
        if constexpr (W == 2) {                       // float32 pairs
            float h = red[0][i / C][i % C][0], l = red[0][i / C][i % C][1];
#pragma unroll
            for (int q = 1; q < PARTS; q++) df_add(h, l, red[q][i / C][i % C][0], red[q][i / C][i % C][1]);
            v = (double)h + (double)l;
        } else {
            v = red[0][i / C][i % C][0];
#pragma unroll
            for (int q = 1; q < PARTS; q++) v += red[q][i / C][i % C][0];
        }
        v += near[at];
        if (out) out[at] = corr[at] - v;
        else near[at] = v;
    }
}

// ---------------------------------------------------------------------------
// correction SpMV + diagonal, a product's part from the input vector alone, into
// a buffer of the plan's:
//   op A: y = C x - K_D x;  op B: y = -K_S x
//
// A warp walks a row's nonzeros, four per lane in flight; the lanes' sums go to
// shared memory, eight threads add a row's, and one thread per row (all lanes of
// a warp, for 32 rows a block) takes the float64 end.  With a shuffle reduction
// and one lane's float64 end per row the float64 pipe (two operations a cycle
// and SM, whatever the lanes) was 80 % busy: Helmholtz mixed, 40,962 rows,
// 7.5M nonzeros 64 -> 39 us (with the copy of x), 163,842 rows, 30M nonzeros
// 214 -> 88.
// ---------------------------------------------------------------------------
constexpr int CB_T = 256;

// a row's end
template <int C, bool OPA>
__device__ __forceinline__ void row_end(int row, int c, double s, const double *Cdiag, const double *x, double *y) {
    const size_t i = (size_t)row * C + c;
    y[i] = OPA ? Cdiag[row] * x[i] - s : -s;
}

template <int C, bool OPA, int RW>
__global__ void __launch_bounds__(CB_T) k_corr(int N, const int *__restrict__ ptr, const int *__restrict__ col,
                                                  const double *__restrict__ val, const double *__restrict__ Cdiag,
                                                  const void *const *__restrict__ xslot, double *__restrict__ y,
                                                  const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int ROWS = CB_T / 32 * RW;
    __shared__ double part[ROWS][C][33], total[ROWS][C];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row0 = blockIdx.x * ROWS;
    const double *x = (const double *)*xslot;
    int p[RW + 1];
#pragma unroll
    for (int r = 0; r <= RW; r++) p[r] = ptr[min(N, row0 + warp * RW + r)];
#pragma unroll
    for (int r = 0; r < RW; r++) {
        double s[C];
#pragma unroll
        for (int c = 0; c < C; c++) s[c] = 0.0;
        auto term = [&](int q, int j) {
            if (C == 1) {
                s[0] += val[q] * x[j];
            } else {
                const double vr = val[2 * (size_t)q], vi = val[2 * (size_t)q + 1];
                const double xr = x[2 * (size_t)j], xi = x[2 * (size_t)j + 1];
                s[0] += vr * xr - vi * xi;
                s[C - 1] += vr * xi + vi * xr;
            }
        };
        // four of a lane's columns loaded ahead, nonzeros summed in order
        constexpr int CU = 4;
        const int qe = p[r + 1];
        int q = p[r] + lane;
        for (; q + 32 * (CU - 1) < qe; q += 32 * CU) {
            int j[CU];
#pragma unroll
            for (int u = 0; u < CU; u++) j[u] = col[q + 32 * u];
#pragma unroll
            for (int u = 0; u < CU; u++) term(q + 32 * u, j[u]);
        }
        for (; q < qe; q += 32) term(q, col[q]);
#pragma unroll
        for (int c = 0; c < C; c++) part[warp * RW + r][c][lane] = s[c];
    }
    __syncthreads();
    for (int i = tid; i < ROWS * C * 8; i += CB_T) {  // whole groups of eight threads
        const int rc = i >> 3, j = i & 7;
        const double *v = part[rc / C][rc % C] + 4 * j;
        double s = (v[0] + v[1]) + (v[2] + v[3]);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (j == 0) total[rc / C][rc % C] = s;
    }
    __syncthreads();
    for (int i = tid; i < ROWS * C; i += CB_T)
        if (row0 + i / C < N) row_end<C, OPA>(row0 + i / C, i % C, total[i / C][i % C], Cdiag, x, y);
}

// float32 correction product (mixed plans): the vector is first copied to
// float32 (one conversion per entry instead of one per nonzero), each lane sums
// its nonzeros with compensation, the lanes' sums combine as float32 pairs.
__global__ void k_x_float(int64_t n, const void *const *__restrict__ xslot, float *__restrict__ xf,
                          const int *__restrict__ skip) {
    if (skip && *skip) return;
    const double *x = (const double *)*xslot;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        xf[i] = (float)x[i];
}

template <int C, bool OPA, int RW>
__global__ void __launch_bounds__(CB_T) k_corr_f(int N, const int *__restrict__ ptr, const int *__restrict__ col,
                                                    const float *__restrict__ val, const float *__restrict__ xf,
                                                    const double *__restrict__ Cdiag, const void *const *__restrict__ xslot,
                                                    double *__restrict__ y, const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int ROWS = CB_T / 32 * RW;
    __shared__ float2 part[ROWS][C][33], total[ROWS][C];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row0 = blockIdx.x * ROWS;
    int p[RW + 1];
#pragma unroll
    for (int r = 0; r <= RW; r++) p[r] = ptr[min(N, row0 + warp * RW + r)];
    auto ldv = [&](int q) {
        return C == 1 ? make_float2(__ldg(val + q), 0.f) : __ldg(reinterpret_cast<const float2 *>(val) + q);
    };
    auto ldx = [&](int j) {
        return C == 1 ? make_float2(__ldg(xf + j), 0.f) : __ldg(reinterpret_cast<const float2 *>(xf) + j);
    };
#pragma unroll
    for (int r = 0; r < RW; r++) {
        KahanF k[C];
        auto term = [&](float2 v, float2 x) {
            if (C == 1) {
                k[0].add(v.x * x.x);
            } else {
                k[0].add(fmaf(v.x, x.x, -v.y * x.y));
                k[C - 1].add(fmaf(v.x, x.y, v.y * x.x));
            }
        };
        // four of a lane's nonzeros in flight at a time (columns, values, then
        // the vector entries), summed in the same order as one at a time
        constexpr int CU = 4;
        const int qe = p[r + 1];
        int q = p[r] + lane;
        for (; q + 32 * (CU - 1) < qe; q += 32 * CU) {
            int j[CU];
            float2 v[CU], x[CU];
#pragma unroll
            for (int u = 0; u < CU; u++) {
                j[u] = __ldg(col + q + 32 * u);
                v[u] = ldv(q + 32 * u);
            }
#pragma unroll
            for (int u = 0; u < CU; u++) x[u] = ldx(j[u]);
#pragma unroll
            for (int u = 0; u < CU; u++) term(v[u], x[u]);
        }
        // the rest the same way, entries beyond the row's end as zeros
        {
            int j[CU];
            float2 v[CU], x[CU];
#pragma unroll
            for (int u = 0; u < CU - 1; u++) {
                const bool on = q + 32 * u < qe;
                j[u] = on ? __ldg(col + q + 32 * u) : -1;
                v[u] = on ? ldv(q + 32 * u) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < CU - 1; u++) x[u] = j[u] >= 0 ? ldx(j[u]) : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < CU - 1; u++)
                if (j[u] >= 0) term(v[u], x[u]);
        }
#pragma unroll
        for (int c = 0; c < C; c++) part[warp * RW + r][c][lane] = make_float2(k[c].s, -k[c].c);
    }
    __syncthreads();
    for (int i = tid; i < ROWS * C * 8; i += CB_T) {  // whole groups of eight threads
        const int rc = i >> 3, j = i & 7;
        const float2 *v = part[rc / C][rc % C] + 4 * j;
        float h = v[0].x, l = v[0].y;
#pragma unroll
        for (int u = 1; u < 4; u++) df_add(h, l, v[u].x, v[u].y);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
            df_add(h, l, oh, ol);
        }
        if (j == 0) total[rc / C][rc % C] = make_float2(h, l);
    }
    __syncthreads();
    const double *x = (const double *)*xslot;
    for (int i = tid; i < ROWS * C; i += CB_T)
        if (row0 + i / C < N) {
            const float2 s = total[i / C][i % C];
            row_end<C, OPA>(row0 + i / C, i % C, (double)s.x + (double)s.y, Cdiag, x, y);
        }
}

// C_i = 1 + (regular Laplace double layer of phi = 1) + (correction row sum),
// and 1 / C_i for the solver's diagonal preconditioner
__global__ void k_finish_diag(int N, const double *__restrict__ ytmp, double *Cdiag, double *dinv) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) {
        const double c = 1.0 + ytmp[i] + Cdiag[i];
        Cdiag[i] = c;
        dinv[i] = 1.0 / c;
    }
}

__global__ void k_fill(int64_t n, double v, double *a) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = v;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
void MIndex::init(int p_) {
    p = p_;
    np = (p + 1) * (p + 2) * (p + 3) / 6;
    m.clear(); n.clear(); k.clear();
    idx3.assign((size_t)(p + 1) * (p + 1) * (p + 1), -1);
    deg_off.assign(p + 2, 0);
    int c = 0;
    for (int h = 0; h <= p; h++) {
        deg_off[h] = c;
        for (int a = h; a >= 0; a--)
            for (int b = h - a; b >= 0; b--) {
                int cc = h - a - b;
                m.push_back(a); n.push_back(b); k.push_back(cc);
                idx3[((size_t)a * (p + 1) + b) * (p + 1) + cc] = c++;
            }
    }
    deg_off[p + 1] = c;
}

Tabs tabs_of(const bem_plan *P) {
    return Tabs{P->d_m, P->d_n, P->d_k, P->d_idx3, P->d_fact, P->mi.p, P->mi.np,
                P->lev_var ? P->d_lev_p : nullptr};
}

TreeView view_of(const bem_plan *P) {
    const Tree &t = P->t;
    return TreeView{t.level, t.ix, t.iy, t.iz, t.parent, t.child0, t.nchild, t.nb, t.ne, t.eb, t.ee, t.leaves,
                    t.near_ptr, t.near_idx, t.inter_ptr, t.inter_idx, t.node_perm, t.reach, t.cx, t.cy, t.cz, t.r,
                    t.tx, t.ty, t.tz, t.side};
}

QuadView quad_of(const bem_plan *P) {
    const Quad &q = P->q;
    return QuadView{q.x, q.y, q.z, q.nx, q.ny, q.nz, q.w, q.fx, q.fy, q.fz, q.fnx, q.fny, q.fnz, q.fw,
                    q.lx, q.ly, q.lz, q.lnx, q.lny, q.lnz};
}

// Shape-function values at the 7 rule points, in constant memory.  Written
// once per device (under a lock): plans are built from several host threads
// while kernels of other plans that read the table are running.
static int init_shape_table(int device) {
    static std::mutex mu;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (device < 0 || device >= 64) { set_error("device %d out of range", device); return BEM_EINVAL; }
    if (done[device]) return BEM_OK;
    double Lq[2][NQ][6] = {};
    {
        const double q = std::sqrt(15.0);
        const double a = (6.0 - q) / 21.0, b = (9.0 + 2.0 * q) / 21.0;
        const double c = (6.0 + q) / 21.0, d = (9.0 - 2.0 * q) / 21.0;
        const double S[7] = {1.0 / 3.0, a, b, a, c, d, c}, T[7] = {1.0 / 3.0, a, a, b, c, c, d};
        for (int r = 0; r < NQ; r++) {
            double l0 = 1.0 - S[r] - T[r], l1 = S[r], l2 = T[r];
            Lq[0][r][0] = l0; Lq[0][r][1] = l1; Lq[0][r][2] = l2;
            Lq[1][r][0] = l0 * (2 * l0 - 1); Lq[1][r][1] = l1 * (2 * l1 - 1); Lq[1][r][2] = l2 * (2 * l2 - 1);
            Lq[1][r][3] = 4 * l0 * l1; Lq[1][r][4] = 4 * l1 * l2; Lq[1][r][5] = 4 * l2 * l0;
        }
    }
    BEM_CUDA(cudaMemcpyToSymbol(c_Lq, Lq, sizeof(Lq)));
    BEM_COPIES_DONE();
    done[device] = true;
    return BEM_OK;
}

// The unit circle at 2 pi j / 1024 for the float32 Helmholtz near field, filled
// once per device (under a lock, as the shape table).
__device__ float g_wave[2 * NF2_TAB];
static int wave_table(int device, const float **out) {
    static std::mutex mu;
    static const float *addr[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (device < 0 || device >= 64) { set_error("device %d out of range", device); return BEM_EINVAL; }
    if (!addr[device]) {
        std::vector<float> t(2 * NF2_TAB);
        for (int j = 0; j < NF2_TAB; j++) {
            t[j] = (float)std::cos(2.0 * M_PI * j / NF2_TAB);
            t[NF2_TAB + j] = (float)std::sin(2.0 * M_PI * j / NF2_TAB);
        }
        void *p = nullptr;
        BEM_CUDA(cudaGetSymbolAddress(&p, g_wave));
        BEM_CUDA(cudaMemcpy(p, t.data(), sizeof(float) * t.size(), cudaMemcpyHostToDevice));
        BEM_COPIES_DONE();
        addr[device] = (const float *)p;
    }
    *out = addr[device];
    return BEM_OK;
}

// the float32 near-field kernels stage their source tile in dynamic shared
// memory above the 48 KB default (set outside any graph capture)
static void set_near_attributes() {
    const int big = 100 * 1024;
    cudaFuncSetAttribute(k_near_f32<1, true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<1, true, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<1, false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<1, false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, true, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, true, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, true, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, true, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_near_f32<2, false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
}

int alloc_fmm(bem_plan *P, cudaStream_t s) {
    Arena &A = P->arena;
    MIndex &mi = P->mi;
    mi.init(P->prm.p);
    // order of each level: L_l = min(p, p_min + l_max - l) (Section 3.6), or p
    {
        const int nlev = std::max(1, P->t.nlev), lmax = nlev - 1;
        P->lev_p.assign(nlev, P->prm.p);
        P->lev_var = false;
        if (P->prm.p_min > 0)
            for (int l = 0; l < nlev; l++) {
                P->lev_p[l] = std::min(P->prm.p, P->prm.p_min + lmax - l);
                if (P->lev_p[l] != P->prm.p) P->lev_var = true;
            }
        BEM_TRY(A.alloc(&P->d_lev_p, nlev));
        BEM_CUDA(cudaMemcpyAsync(P->d_lev_p, P->lev_p.data(), sizeof(int) * nlev, cudaMemcpyHostToDevice, s));
    }
    const int np = mi.np, nbox = P->t.nbox, C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    BEM_TRY(A.alloc(&P->d_m, np));
    BEM_TRY(A.alloc(&P->d_n, np));
    BEM_TRY(A.alloc(&P->d_k, np));
    BEM_TRY(A.alloc(&P->d_idx3, mi.idx3.size()));
    BEM_CUDA(cudaMemcpyAsync(P->d_m, mi.m.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
    BEM_CUDA(cudaMemcpyAsync(P->d_n, mi.n.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
    BEM_CUDA(cudaMemcpyAsync(P->d_k, mi.k.data(), sizeof(int) * np, cudaMemcpyHostToDevice, s));
    BEM_CUDA(cudaMemcpyAsync(P->d_idx3, mi.idx3.data(), sizeof(int) * mi.idx3.size(), cudaMemcpyHostToDevice, s));
    std::vector<double> fact(2 * PMAX + 2);
    fact[0] = 1.0;
    for (int i = 1; i < (int)fact.size(); i++) fact[i] = fact[i - 1] * i;
    BEM_TRY(A.alloc(&P->d_fact, fact.size()));
    BEM_CUDA(cudaMemcpyAsync(P->d_fact, fact.data(), sizeof(double) * fact.size(), cudaMemcpyHostToDevice, s));
    BEM_TRY(init_shape_table(P->device));
    const bool mx = P->prm.precision == BEM_MIXED;
    if (mx) {
        BEM_TRY(A.alloc(&P->ff, (size_t)P->Q * C));
        BEM_TRY(A.alloc(&P->fM, (size_t)nbox * np * C));
        BEM_TRY(A.alloc(&P->fL, (size_t)nbox * np * C));
    } else {
        BEM_TRY(A.alloc(&P->f, (size_t)P->Q * C));
        BEM_TRY(A.alloc(&P->M, (size_t)nbox * np * C));
        BEM_TRY(A.alloc(&P->L, (size_t)nbox * np * C));
    }
    BEM_TRY(A.alloc(&P->ytmp, (size_t)P->N * C));
    BEM_TRY(A.alloc(&P->xptr, 2));
    BEM_TRY(A.alloc(&P->yptr, 2));
    if (mx) BEM_TRY(A.alloc(&P->xf, (size_t)std::max(P->N, P->nchi) * C));
    if (!P->diag_mode) BEM_TRY(A.alloc(&P->ycor, (size_t)P->N * C));
    if (mx && !P->diag_mode && !P->lev_var) {
        // stored P2M weights of the double layer (op A, every product of a solve)
        BEM_TRY(A.alloc(&P->p2m_W, (size_t)P->Q * np));
        const Tree &t = P->t;
        launch_p2m<1, true, true>(t.nleaf, tabs_of(P), view_of(P), quad_of(P), nullptr, nullptr, nullptr, s,
                                         P->p2m_W);
        BEM_LAUNCH_CHECK();
    }
    set_translation_attributes();
    set_near_attributes();
    if (mx && P->green == BEM_HELMHOLTZ) BEM_TRY(wave_table(P->device, &P->wave));
    if (!mx) {
        BEM_TRY(near_pairs_prepare(P));
        BEM_TRY(p2m_pairs_prepare());
    }
    BEM_TRY(build_translation_tables(P, s));
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// near-field sums of every node into ytmp
template <class R, int C>
static int launch_near(bem_plan *P, int op, double kwave, const R *f, double *ytmp, cudaStream_t s) {
    const TreeView tv = view_of(P);
    const QuadView qv = quad_of(P);
    const Tree &t = P->t;
    const int *sk = P->skip;
    if constexpr (sizeof(R) == sizeof(float)) {
        const int ni = P->near_nitems[C - 1];
        const int2 *it = P->near_items[C - 1];
        if (ni == 0) return BEM_OK;
        // blocks per item
        int ns = 1;
        while (ns < NF2_MAXC && ni * ns < NF2_WAVES * 3 * P->sm_count) ns *= 2;
        auto near = [&](auto shared, auto alone, size_t sm) {
            return launch_cluster(ns > 1 ? shared : alone, (unsigned)(ni * ns), NF2_T, sm, ns, s, ns, it, tv, qv, kwave, f,
                                  ytmp, P->wave, sk);
        };
#define BEM_NEAR(C_, DL_, TAB_) \
    return near(k_near_f32<C_, DL_, TAB_, true>, k_near_f32<C_, DL_, TAB_, false>, nf2_dyn_bytes(C_, TAB_))
        // (two points of one near field are at most some 4 sides apart; see near_pairs_apply)
        if (C == 2 && kwave * t.side * 8.0 * (NF2_TAB / (2.0 * M_PI)) >= NF2_MAXPHASE) {
            if (op == BEM_OP_A) BEM_NEAR(2, true, false);
            BEM_NEAR(2, false, false);
        }
        if (op == BEM_OP_A) BEM_NEAR(C, true, true);
        BEM_NEAR(C, false, true);
#undef BEM_NEAR
    } else {
        if (near_pairs_apply(P, C, kwave)) return launch_near_pairs<C>(P, op, kwave, f, ytmp, s);
        if constexpr (C == 2) {
            if (op == BEM_OP_A) (k_near<true><<<t.nleaf, NF_T, 0, s>>>(t.nleaf, tv, qv, kwave, f, ytmp, sk), ::bem::count_launch());
            else (k_near<false><<<t.nleaf, NF_T, 0, s>>>(t.nleaf, tv, qv, kwave, f, ytmp, sk), ::bem::count_launch());
            BEM_LAUNCH_CHECK();
        }
        return BEM_OK;
    }
}

// the correction's part of a product into ycor
template <class R, int C>
static int launch_correction(bem_plan *P, int op, cudaStream_t s) {
    const int N = (int)P->N;
    const Correction &K = P->corr;
    // four rows a warp where that still makes eight blocks per SM
    const bool four = N >= 32 * 8 * P->sm_count;
    const int blocks = four ? (N + 31) / 32 : (N + 7) / 8;
    const bool a = op == BEM_OP_A;
    const int *ptr = a ? K.ptrD : K.ptrS, *col = a ? K.colD : K.colS;
    if constexpr (sizeof(R) == sizeof(float)) {
        const int64_t nx = (int64_t)(a ? N : P->nchi) * C;
        (k_x_float<<<(int)std::min<int64_t>((nx + 255) / 256, 4096), 256, 0, s>>>(nx, P->xptr, P->xf, P->skip),
         ::bem::count_launch());
        auto go = [&](auto kernel) {
            (kernel<<<blocks, CB_T, 0, s>>>(N, ptr, col, a ? K.fvalD : K.fvalS, P->xf, P->C, P->xptr, P->ycor, P->skip),
             ::bem::count_launch());
        };
        if (four) a ? go(k_corr_f<C, true, 4>) : go(k_corr_f<C, false, 4>);
        else a ? go(k_corr_f<C, true, 1>) : go(k_corr_f<C, false, 1>);
    } else {
        auto go = [&](auto kernel) {
            (kernel<<<blocks, CB_T, 0, s>>>(N, ptr, col, a ? K.valD : K.valS, P->C, P->xptr, P->ycor, P->skip),
             ::bem::count_launch());
        };
        if (four) a ? go(k_corr<C, true, 4>) : go(k_corr<C, false, 4>);
        else a ? go(k_corr<C, true, 1>) : go(k_corr<C, false, 1>);
    }
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// ev (optional, BEM_NSTAGES + 1 events): ev[0] recorded before P2Q, ev[i] after
// stage i, and the last event before the correction, which comes first; for
// per-stage timing outside graphs.
//
// Under a capture the correction (memory-bound, needs the input vector alone) and
// the near field (arithmetic, needs the strengths alone) take branches of their
// own beside the expansions; L2P ends the product when all three are done, and
// no kernel before it writes the output.
template <class R, int C>
static int run_fmm(bem_plan *P, int op, double kwave, R *f, R *M, R *L, double *ytmp, int with_diag, cudaStream_t s,
                   cudaEvent_t *ev, cudaStream_t fork) {
    if (ev) BEM_CUDA(cudaEventRecord(ev[BEM_NSTAGES], s));
    if (with_diag) {
        if (fork) {
            BEM_CUDA(cudaEventRecord(P->fork_ev[0], s));
            BEM_CUDA(cudaStreamWaitEvent(P->corr_stream, P->fork_ev[0], 0));
        }
        BEM_TRY((launch_correction<R, C>(P, op, fork ? P->corr_stream : s)));
        if (fork) BEM_CUDA(cudaEventRecord(P->fork_ev[1], P->corr_stream));
    }
    if (ev) BEM_CUDA(cudaEventRecord(ev[0], s));
    const Tabs tb = tabs_of(P);
    const TreeView tv = view_of(P);
    const QuadView qv = quad_of(P);
    const Tree &t = P->t;
    const int np = tb.np, p = tb.p;
    const int *sk = P->skip;
    const int *el = op == BEM_OP_A ? t.el_phi : t.el_chi;
    const int Q = (int)P->Q;
    (k_p2q<R, C><<<(Q + 255) / 256, 256, 0, s>>>(Q, P->npe, el, P->q.w, P->xptr, f, sk), ::bem::count_launch());
    if (ev) BEM_CUDA(cudaEventRecord(ev[1], s));
    auto near = [&](cudaStream_t ns) -> int { return launch_near<R, C>(P, op, kwave, f, ytmp, ns); };
    if (fork) {
        BEM_CUDA(cudaEventRecord(P->fork_ev[2], s));
        BEM_CUDA(cudaStreamWaitEvent(fork, P->fork_ev[2], 0));
    }
    if constexpr (sizeof(R) == sizeof(float)) {
        if (op == BEM_OP_A && P->p2m_W)
            launch_p2m_stored<C>(t.nleaf, np, tv, P->p2m_W, f, M, sk, s);
        else if (op == BEM_OP_A) launch_p2m<C, true>(t.nleaf, tb, tv, qv, f, M, sk, s);
        else launch_p2m<C, false>(t.nleaf, tb, tv, qv, f, M, sk, s);
    } else {
        BEM_TRY(launch_p2m_pairs<C>(P, op == BEM_OP_A, f, M, s));
    }
    BEM_LAUNCH_CHECK();
    if (fork) {
        BEM_TRY(near(fork));
        BEM_CUDA(cudaEventRecord(P->fork_ev[3], fork));
    }
    if (ev) BEM_CUDA(cudaEventRecord(ev[2], s));
    BEM_TRY((launch_translations<R, C>(P, M, L, s, ev)));
    if (!fork) BEM_TRY(near(s));
    if (fork) {
        if (with_diag) BEM_CUDA(cudaStreamWaitEvent(s, P->fork_ev[1], 0));
        BEM_CUDA(cudaStreamWaitEvent(s, P->fork_ev[3], 0));
    }
    const int ni = P->near_nitems[C - 1];
    constexpr int SLOTS = sizeof(R) == sizeof(float) ? NF2_SLOTS : ND_SLOTS;
    if (ni > 0)
        (k_l2p<R, C, SLOTS><<<ni, L2P_T, sizeof(R) * np * C, s>>>(P->near_items[C - 1], tb, tv, P->sy_mexp, 1.0 / tv.side, L,
                                                                 ytmp, P->ycor, with_diag ? P->yptr : nullptr, sk),
         ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    if (ev) BEM_CUDA(cudaEventRecord(ev[6], s));
    return BEM_OK;
}

// Moments for the field evaluation: double-layer moments of phi minus
// single-layer moments of chi at the leaves (the local buffer serves as
// scratch), then shifted up the tree.
template <class R>
__global__ void k_sub_moments(size_t n, R *__restrict__ M, const R *__restrict__ B) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) M[i] -= B[i];
}

template <class R, int C>
static int field_moments_t(bem_plan *P, const void *phi, const void *chi, R *f, R *M, R *Bm, cudaStream_t s) {
    const Tabs tb = tabs_of(P);
    const TreeView tv = view_of(P);
    const QuadView qv = quad_of(P);
    const Tree &t = P->t;
    const int Q = (int)P->Q;
    const int *sk = P->skip;
    // strengths in float64 for the direct part, and in the plan's precision for
    // the moments (float64 plans: the same array)
    for (int part = 0; part < 2; part++) {
        double *str = P->fd_str + (size_t)part * Q * C;
        const int *el = part ? t.el_chi : t.el_phi;
        BEM_TRY(set_slots(P, part ? chi : phi, nullptr, s));
        (k_p2q<double, C><<<(Q + 255) / 256, 256, 0, s>>>(Q, P->npe, el, P->q.w, P->xptr, str, sk), ::bem::count_launch());
        if constexpr (sizeof(R) == sizeof(double)) {
            BEM_TRY(launch_p2m_pairs<C>(P, !part, str, part ? Bm : M, s));
        } else {
            (k_p2q<R, C><<<(Q + 255) / 256, 256, 0, s>>>(Q, P->npe, el, P->q.w, P->xptr, f, sk), ::bem::count_launch());
            if (part) launch_p2m<C, false>(t.nleaf, tb, tv, qv, f, Bm, sk, s);
            else if (P->p2m_W) launch_p2m_stored<C>(t.nleaf, P->mi.np, tv, P->p2m_W, f, M, sk, s);
            else launch_p2m<C, true>(t.nleaf, tb, tv, qv, f, M, sk, s);
        }
    }
    const size_t n = (size_t)t.nbox * P->mi.np * C;
    (k_sub_moments<R><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, M, Bm), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return launch_m2m<R, C>(P, M, s);
}

int field_moments(bem_plan *P, const void *phi, const void *chi, cudaStream_t s) {
    const bool mx = P->prm.precision == BEM_MIXED, helm = P->green == BEM_HELMHOLTZ;
    if (mx) return helm ? field_moments_t<float, 2>(P, phi, chi, P->ff, P->fM, P->fL, s)
                        : field_moments_t<float, 1>(P, phi, chi, P->ff, P->fM, P->fL, s);
    return helm ? field_moments_t<double, 2>(P, phi, chi, P->f, P->M, P->L, s)
                : field_moments_t<double, 1>(P, phi, chi, P->f, P->M, P->L, s);
}

// Enqueues one product on stream s.  The input and output vectors are read
// from the device slots P->xptr[0] / P->yptr[0].  with_diag = 0 leaves the
// regular far + near sums in the regular-sum buffer (used for the diagonal).
// wb (optional) names the work buffers of this product; NULL = the plan's.
// fork (optional, under a capture only): a second stream for the near field, and
// corr_stream takes the correction.
int enqueue_matvec_raw(bem_plan *P, int op, int green, double kwave, int with_diag, cudaStream_t s,
                       cudaEvent_t *ev, const WorkBufs *wb, cudaStream_t fork) {
    const int C = green == BEM_HELMHOLTZ ? 2 : 1;
    const bool mx = P->prm.precision == BEM_MIXED;
    WorkBufs w;
    if (wb) w = *wb;
    else if (mx) w = WorkBufs{P->ff, P->fM, P->fL, P->ytmp};
    else w = WorkBufs{P->f, P->M, P->L, P->ytmp};
    if (!mx) {
        double *f = (double *)w.f, *M = (double *)w.M, *L = (double *)w.L;
        if (C == 1) BEM_TRY((run_fmm<double, 1>(P, op, kwave, f, M, L, w.ytmp, with_diag, s, ev, fork)));
        else BEM_TRY((run_fmm<double, 2>(P, op, kwave, f, M, L, w.ytmp, with_diag, s, ev, fork)));
    } else {
        float *f = (float *)w.f, *M = (float *)w.M, *L = (float *)w.L;
        if (C == 1) BEM_TRY((run_fmm<float, 1>(P, op, kwave, f, M, L, w.ytmp, with_diag, s, ev, fork)));
        else BEM_TRY((run_fmm<float, 2>(P, op, kwave, f, M, L, w.ytmp, with_diag, s, ev, fork)));
    }
    return BEM_OK;
}

// Diagonal: C_i = 1 + sum_j D0_ij with D0 the Laplace double layer.  The
// correction row sums are already in P->C; one regular Laplace double-layer
// product on phi = 1 adds the rest.  For a constant density the far-field
// contributions add up coherently, so the expansions' relative error shows
// in full; this one product therefore runs in float64 at the largest
// supported order (error ~ eta^-(p+1)), on the same tree and lists, before
// the buffers are sized for the plan's own order and precision.
// The order, precision and Green's function of the diagonal's product.
struct DiagSwap {
    int p, precision, green, p_min;
};
// the diagonal's product runs at one order for every level: float64 plans at
// DIAG_P, where its truncation error is below the float64 diagonal's stated
// 5e-8; mixed plans at p + 2, at most DIAG_P: there float32 rounding, not the
// truncation, sets the diagonal's error (its difference from the float64
// plan's diagonal is the same at p + 2, p + 3 and p + 4)
constexpr int DIAG_P = 16;
static DiagSwap diag_fields(const bem_plan *P) {
    const bool mixed = P->prm.precision == BEM_MIXED;
    return DiagSwap{mixed ? std::min(DIAG_P, P->prm.p + 2) : DIAG_P, mixed ? BEM_MIXED : BEM_F64, BEM_LAPLACE, 0};
}
static DiagSwap swap_fields(bem_plan *P, const DiagSwap &d) {
    const DiagSwap old{P->prm.p, P->prm.precision, P->green, P->prm.p_min};
    P->prm.p = d.p;
    P->prm.precision = d.precision;
    P->green = d.green;
    P->prm.p_min = d.p_min;
    return old;
}

// Three steps, so that the product can run on its own stream beside the
// correction: prepare (buffers and tables at the diagonal's order, built into
// the plan and then moved to diag_state; all allocations happen here),
// product (phi = 1, into the diagonal's ytmp), finish (C += that ytmp once the
// correction's row sums are in C, then the diagonal's buffers are released).
// The plan's own order is built between product and finish, while the product
// runs.  The plan's fields are switched only while each step runs.
static void swap_state(bem_plan *P) { std::swap(static_cast<FmmState &>(*P), P->diag_state); }

int diagonal_prepare(bem_plan *P, cudaStream_t s) {
    const DiagSwap keep = swap_fields(P, diag_fields(P));
    P->diag_mode = true;                              // no stored weights at the diagonal's order
    int rc = alloc_fmm(P, s);
    P->diag_mode = false;
    if (rc == BEM_OK) rc = P->arena.alloc(&P->diag_ones, P->N);
    swap_state(P);                                    // the plan's own state is empty until alloc_fmm
    swap_fields(P, keep);
    return rc;
}

int diagonal_product(bem_plan *P, cudaStream_t s) {
    const int N = (int)P->N;
    const DiagSwap keep = swap_fields(P, diag_fields(P));
    swap_state(P);
    (k_fill<<<(N + 255) / 256, 256, 0, s>>>(N, 1.0, P->diag_ones), ::bem::count_launch());
    int rc = set_slots(P, P->diag_ones, nullptr, s);
    if (rc == BEM_OK) rc = enqueue_matvec_raw(P, BEM_OP_A, BEM_LAPLACE, 0.0, 0, s, nullptr);
    swap_state(P);
    swap_fields(P, keep);
    return rc;
}

int diagonal_finish(bem_plan *P, cudaStream_t s) {
    const int N = (int)P->N;
    BEM_TRY(P->arena.alloc(&P->dinv, P->N));
    (k_finish_diag<<<(N + 255) / 256, 256, 0, s>>>(N, P->diag_state.ytmp, P->C, P->dinv), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    BEM_CUDA(cudaStreamSynchronize(s));
    P->arena.release(P->diag_ones);
    P->diag_ones = nullptr;
    swap_state(P);
    free_fmm(P);
    swap_state(P);
    return BEM_OK;
}

// releases what alloc_fmm allocated
void free_fmm(bem_plan *P) {
    free_translation_tables(P);
    Arena &A = P->arena;
    for (void *q : {(void *)P->d_m, (void *)P->d_n, (void *)P->d_k, (void *)P->d_idx3, (void *)P->d_fact,
                    (void *)P->f, (void *)P->M, (void *)P->L, (void *)P->ff, (void *)P->fM,
                    (void *)P->fL, (void *)P->ytmp, (void *)P->xptr, (void *)P->yptr, (void *)P->p2m_W, (void *)P->xf, (void *)P->ycor, (void *)P->d_lev_p})
        A.release(q);
    P->p2m_W = nullptr;
    P->xf = nullptr;
    P->ycor = nullptr;
    P->d_lev_p = nullptr;
    P->lev_var = false;
    P->d_m = P->d_n = P->d_k = P->d_idx3 = nullptr;
    P->d_fact = nullptr;
    P->f = P->M = P->L = P->ytmp = nullptr;
    P->ff = P->fM = P->fL = nullptr;
    P->xptr = nullptr;
    P->yptr = nullptr;
}


// ---------------------------------------------------------------------------
// A product that allocates nothing
//
// Callers that cannot allocate device memory when they need a product --
// real-time loops where an allocation (which may synchronise the device) is
// not allowed, or hosts whose device memory all belongs to another allocator
// (a framework's pool) that forbids stray cudaMalloc calls -- can use
// bem_matvec_noalloc.  It launches the same kernels as bem_matvec, directly
// (no graph is instantiated), and keeps the per-product scratch (quadrature
// strengths, moments, local expansions, regular sums) in the file-scope array
// below instead of the plan's own buffers: the array's pieces go to the
// launches as arguments (WorkBufs), and no field of the plan is changed, so
// other host threads see the plan as it was.  The array is NOALLOC_BYTES long
// and every GPU that loads this library holds it until the process exits.
// Its device address is looked up once per device, on the first call made
// on that device (so that first call should come before any stream capture).
// All calls share the array and it keeps the last call's contents; no part of
// it needs to start at zero (every stage writes its output before it is read).
// Calls that overlap on the GPU -- on different streams, or for different
// plans at the same time -- race on the array.
// ---------------------------------------------------------------------------
constexpr size_t NOALLOC_BYTES = (size_t)48 << 20;   // 48 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];
static void *g_noalloc_addr[64];                     // per device ordinal, 0 until looked up

static size_t noalloc_round(size_t b) { return (b + 255) & ~(size_t)255; }

const void *kernel_of_fmm() { return (const void *)k_fill; }

}  // namespace bem

extern "C" int bem_matvec_noalloc(bem_plan *P, int op, const void *x_dev, void *y_dev, void *cuda_stream) {
    using namespace bem;
    if (!P || !x_dev || !y_dev) { set_error("bem_matvec_noalloc: NULL argument"); return BEM_EINVAL; }
    if (op != BEM_OP_A && op != BEM_OP_B) { set_error("bem_matvec_noalloc: bad op %d", op); return BEM_EINVAL; }
    if (P->device < 0 || P->device >= 64) { set_error("bem_matvec_noalloc: device %d out of range", P->device); return BEM_EINVAL; }
    const int C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    const bool mx = P->prm.precision == BEM_MIXED;
    const size_t rb = mx ? sizeof(float) : sizeof(double);
    const size_t bf = noalloc_round((size_t)P->Q * C * rb);
    const size_t bm = noalloc_round((size_t)P->t.nbox * P->mi.np * C * rb);
    const size_t by = noalloc_round((size_t)P->N * C * sizeof(double));
    const size_t need = bf + 2 * bm + by;
    if (need > NOALLOC_BYTES) {
        set_error("bem_matvec_noalloc: this plan needs %zu bytes of scratch, the fixed array holds %zu",
                  need, NOALLOC_BYTES);
        return BEM_EINVAL;
    }
    int prev_dev = -1;
    BEM_CUDA(cudaGetDevice(&prev_dev));
    BEM_CUDA(cudaSetDevice(P->device));
    int rc = BEM_OK;
    if (!g_noalloc_addr[P->device]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) rc = cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)", __FILE__, __LINE__);
        else g_noalloc_addr[P->device] = ptr;
    }
    if (rc == BEM_OK) {
        // this product's work buffers are carved from the scratch and passed to
        // the launches as arguments; the plan's own fields are not touched
        unsigned char *base = (unsigned char *)g_noalloc_addr[P->device];
        const WorkBufs w{base, base + bf, base + bf + bm, (double *)(base + bf + 2 * bm)};
        cudaStream_t s = (cudaStream_t)cuda_stream;
        rc = set_slots(P, x_dev, y_dev, s);
        if (rc == BEM_OK) {
            cudaError_t e = cudaMemsetAsync(P->skip, 0, sizeof(int), s);
            rc = e == cudaSuccess ? BEM_OK : cuda_fail(e, "cudaMemsetAsync", __FILE__, __LINE__);
        }
        if (rc == BEM_OK) rc = enqueue_matvec_raw(P, op, P->green, P->k, 1, s, nullptr, &w);
        P->fence.mark(s);
    }
    cudaSetDevice(prev_dev);
    return rc;
}



// Translation operators of the fast method:
//
//   M2M  coefficient shift (Eq. 8):  Ms'_a = sum_{b<=a} C(a,b) s^b 2^-(|a|+|b|) Ms_{a-b}
//   L2L  expansion shift (Eq. 9):    Ls'_b += sum_g C(b+g,b) s^g 2^-(2|g|+|b|) Ls_{b+g}
//   M2L  local expansion (Eq. 7):    Ls_t[b] = 1/(h_t b!) sum_a D[a+b] (-1)^|a| (h_s/h_t)^|a| Ms_s[a] / a!
//
// Moments / locals are scaled by the box edge (Ms = I / h^|a|, Ls = F h^|b|),
// so a child's offset from its parent is +-1/4 of the parent edge per axis and
// every shift coefficient is a product of per-axis binomials and powers of
// two; the octant only flips signs.
//
// M2L: the derivatives D[g] = d^g Ghat(rho) (Tausch's recursions, Section
// 3.3) depend only on rho = (c_t - c_s) / h_t, the level difference and, for
// Helmholtz, k h_t.  Boxes sit on dyadic lattices, so every interaction pair
// falls into one of a small number of exact offset classes, and these reduce
// further to canonical classes under the signed axis permutations
// (m2l_tc.cu).  This file builds the exact classes and the FP64 derivative
// tables; the contraction runs on the tensor cores (m2l_tc.cu) or as a SIMT
// GEMM (m2l_simt.cu).
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <map>
#include <thread>
#include <tuple>
#include <unordered_map>
#include <vector>

#include "cluster.cuh"

namespace bem {

constexpr int TT = 128;                   // threads per block of the translation kernels

template <class R, int C>
__device__ __forceinline__ void cmac(R *acc, R cf, const R *v) {
#pragma unroll
    for (int c = 0; c < C; c++) acc[c] += cf * v[c];
}

// ---------------------------------------------------------------------------
// Shifts as three one-dimensional passes.  With box-scaled expansions every
// shift coefficient is a product of per-axis factors,
//   M2M  M'_a = 2^-|a| sum_{g <= a} prod_i binom(a_i, g_i) 2^-g_i s_i^g_i  M_{a-g},
//   L2L  L'_b = 2^-|b| sum_{|b|+|g| <= p} prod_i binom(b_i+g_i, b_i) 4^-g_i s_i^g_i  L_{b+g},
// (s_i = -1 where the child lies on the low side of axis i), so each shift is
// done axis by axis: an output of one pass sums at most p + 1 terms, and the
// degree bound |.| <= p carries through the passes unchanged.  Multi-index
// table and per-axis factors sit in shared memory.  One child per block either
// way.  Deterministic.
//
// A level is bound by its blocks' latency (it takes as long for one parent as
// for hundreds), so a block does little one after the other: its coefficients,
// the packed multi-indices and the factors come in one round of loads, and the
// eight children of a parent go to the eight blocks of a cluster, whose sums
// are added in child order through distributed shared memory.  With the
// children in one block and the factors computed there, M2M of the cube of 24,300
// tri6 (float32, four levels) took 57 us, now 36, of 8,748 (float64) 137, now
// 40; L2L 31 -> 21 and 33 -> 20.
// ---------------------------------------------------------------------------
constexpr int MM_T = 320, MM_CL = 8;      // threads; blocks per parent (M2M)

// shared-memory bytes of the shift tables at order p: factors [P1][P1], index
// of every multi-index of degree <= p (the only ones a pass looks up) at
// (m (p + 1) + n) (p + 1) + k, packed multi-indices [np]
template <class R>
__host__ __device__ inline size_t shift_tab_bytes(int p, int np) {
    const int P1 = p + 1;
    return (((size_t)sizeof(R) * P1 * P1 + sizeof(short) * P1 * P1 * P1 + 15) / 16) * 16 + 4 * (size_t)np + 16;
}

// The tables and the block's nt source values, all loads of a thread in flight
// before the first is stored.  G: factors [a][g] of stride Pm1 for the pass
// direction; mexp: packed multi-indices.
template <class R, int U>
__device__ __forceinline__ void shift_load(int p, int np, int Pm1, const R *__restrict__ G, const int *__restrict__ mexp,
                                           const R *src, int nt, short *sIdx, R *sG, int *sMNK, R *sA) {
    const int P1 = p + 1, tid = threadIdx.x;
    R v[U];
    int e[2];
#pragma unroll
    for (int u = 0; u < U; u++) v[u] = tid + u * MM_T < nt ? src[tid + u * MM_T] : (R)0;
#pragma unroll
    for (int u = 0; u < 2; u++) e[u] = tid + u * MM_T < np ? __ldg(mexp + tid + u * MM_T) : 0;
    const R g0 = tid < P1 * P1 ? G[tid / P1 * Pm1 + tid % P1] : (R)0;
#pragma unroll
    for (int u = 0; u < 2; u++) {
        const int a = tid + u * MM_T;
        if (a < np) {
            sMNK[a] = e[u];
            sIdx[((e[u] & 255) * P1 + (e[u] >> 8 & 255)) * P1 + (e[u] >> 16 & 255)] = (short)a;
        }
    }
    for (int a = tid + 2 * MM_T; a < np; a += MM_T) {
        const int x = __ldg(mexp + a);
        sMNK[a] = x;
        sIdx[((x & 255) * P1 + (x >> 8 & 255)) * P1 + (x >> 16 & 255)] = (short)a;
    }
    if (tid < P1 * P1) sG[tid] = g0;
    for (int i = tid + MM_T; i < P1 * P1; i += MM_T) sG[i] = G[i / P1 * Pm1 + i % P1];
#pragma unroll
    for (int u = 0; u < U; u++)
        if (tid + u * MM_T < nt) sA[tid + u * MM_T] = v[u];
    for (int t = tid + U * MM_T; t < nt; t += MM_T) sA[t] = src[t];
}

// one axis pass: out[a] = sum_g G[a_ax][g] s^g in[a -/+ g e_ax]
template <class R, int C, bool DOWN>
__device__ __forceinline__ void shift_pass(int ax, int p, int np, const int *sMNK, const short *sIdx, const R *sG,
                                           int mask, const R *in, R *out) {
    const int P1 = p + 1, st = ax == 0 ? P1 * P1 : ax == 1 ? P1 : 1;
    const R sg = (mask >> ax) & 1 ? (R)-1 : (R)1;
    for (int a = threadIdx.x; a < np; a += MM_T) {
        const int mnk = sMNK[a], e = mnk >> (8 * ax) & 255, rest = p - (mnk >> 24);
        const short *id = sIdx + ((mnk & 255) * P1 + (mnk >> 8 & 255)) * P1 + (mnk >> 16 & 255);
        const R *Ge = sG + e * P1;
        R acc[C];
#pragma unroll
        for (int c = 0; c < C; c++) acc[c] = (R)0;
        R gs = (R)1;
        const int ng = DOWN ? e : rest;          // M2M: g <= a_ax;  L2L: |a| + g <= p
#pragma unroll 4
        for (int g = 0; g <= ng; g++, gs *= sg) cmac<R, C>(acc, gs * Ge[g], in + id[DOWN ? -g * st : g * st] * C);
#pragma unroll
        for (int c = 0; c < C; c++) out[(size_t)a * C + c] = acc[c];
    }
}

// 2^-|a| of the coefficient with packed multi-index mnk
template <class R>
__device__ __forceinline__ R deg_scale(int mnk) {
    const int d = mnk >> 24;
    if constexpr (sizeof(R) == sizeof(float)) return ldexpf(1.f, -d);
    else return ldexp(1.0, -d);
}

// block 8 i + j of the grid: child j of the level's i-th box
template <class R, int C>
__global__ void __launch_bounds__(MM_T) __cluster_dims__(MM_CL, 1, 1)
    k_m2m_sep(int off, const int *__restrict__ child0, const int *__restrict__ nchild, const int *__restrict__ ix,
              const int *__restrict__ iy, const int *__restrict__ iz, int p, int np, int nps, int npc, int Pm1,
              const R *__restrict__ G, const int *__restrict__ mexp, R *__restrict__ M, const int *__restrict__ skip) {
    if (skip && *skip) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = p + 1;
    R *sA = (R *)smem_raw;                                  // [np][C]
    R *sB = sA + (size_t)np * C;                             // [np][C]
    R *sG = sB + (size_t)np * C;                             // [P1][P1]
    short *sIdx = (short *)(sG + P1 * P1);                   // [P1^3]
    int *sMNK = (int *)((unsigned char *)sG + (shift_tab_bytes<R>(p, np) - 4 * (size_t)np - 16));   // [np]
    const int b = off + blockIdx.x / MM_CL, j = blockIdx.x % MM_CL, nch = nchild[b], tid = threadIdx.x;
    if (nch == 0) return;                                    // all blocks of the cluster
    if (j < nch) {
        // the child (consecutive boxes, row stride nps) holds npc coefficients; the rest enter as zero
        const int c = child0[b] + j, nt = npc * C;
        for (int t = nt + tid; t < np * C; t += MM_T) sA[t] = (R)0;
        // a child on the low side of an axis has offset -1/4 of the parent edge
        const int mask = ((ix[c] & 1) ? 0 : 1) | ((iy[c] & 1) ? 0 : 2) | ((iz[c] & 1) ? 0 : 4);
        shift_load<R, 2 * C>(p, np, Pm1, G, mexp, M + (size_t)c * nps * C, min(nt, np * C), sIdx, sG, sMNK, sA);
        __syncthreads();
        shift_pass<R, C, true>(0, p, np, sMNK, sIdx, sG, mask, sA, sB);
        __syncthreads();
        shift_pass<R, C, true>(1, p, np, sMNK, sIdx, sG, mask, sB, sA);
        __syncthreads();
        shift_pass<R, C, true>(2, p, np, sMNK, sIdx, sG, mask, sA, sB);
    }
    cluster_sync();
    if (j < nch)                                             // these hold the multi-indices
        for (int t = j * MM_T + tid; t < np * C; t += nch * MM_T) {
            R v[MM_CL];
#pragma unroll
            for (int q = 0; q < MM_CL; q++) v[q] = q < nch ? peer_load(sB + t, q) : (R)0;
            R sum = (R)0;
#pragma unroll
            for (int q = 0; q < MM_CL; q++)
                if (q < nch) sum += v[q];
            M[(size_t)b * nps * C + t] = sum * deg_scale<R>(sMNK[t / C]);
        }
    cluster_sync();                                          // no block leaves while others read its sums
}

template <class R, int C>
__global__ void __launch_bounds__(MM_T) k_l2l_sep(int off, const int *__restrict__ parent, const int *__restrict__ ix,
                                                  const int *__restrict__ iy, const int *__restrict__ iz, int p, int np,
                                                  int nps, int npo, int Pm1, const R *__restrict__ G,
                                                  const int *__restrict__ mexp, R *__restrict__ L,
                                                  const int *__restrict__ skip) {
    if (skip && *skip) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P1 = p + 1;
    R *sA = (R *)smem_raw;                                  // [np][C]
    R *sB = sA + (size_t)np * C;                             // [np][C]
    R *sG = sB + (size_t)np * C;                             // [P1][P1]
    short *sIdx = (short *)(sG + P1 * P1);                   // [P1^3]
    int *sMNK = (int *)((unsigned char *)sG + (shift_tab_bytes<R>(p, np) - 4 * (size_t)np - 16));   // [np]
    const int b = off + blockIdx.x, tid = threadIdx.x;
    const int mask = ((ix[b] & 1) ? 0 : 1) | ((iy[b] & 1) ? 0 : 2) | ((iz[b] & 1) ? 0 : 4);
    shift_load<R, 2 * C>(p, np, Pm1, G, mexp, L + (size_t)parent[b] * nps * C, np * C, sIdx, sG, sMNK, sA);
    __syncthreads();
    shift_pass<R, C, false>(2, p, np, sMNK, sIdx, sG, mask, sA, sB);
    __syncthreads();
    shift_pass<R, C, false>(1, p, np, sMNK, sIdx, sG, mask, sB, sA);
    __syncthreads();
    shift_pass<R, C, false>(0, p, np, sMNK, sIdx, sG, mask, sA, sB);
    __syncthreads();
    for (int t = tid; t < npo * C; t += MM_T)        // the child keeps its own order's npo coefficients (npo <= np)
        L[(size_t)b * nps * C + t] += sB[t] * deg_scale<R>(sMNK[t / C]);
}

// ---------------------------------------------------------------------------
// M2L derivative tables, one block per offset class (FP64)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(TT) k_m2l_tables(int ncls, int p, int np, int C, const int *__restrict__ tm,
                                                   const int *__restrict__ tn, const int *__restrict__ tk,
                                                   const int *__restrict__ idx3, const double *__restrict__ rho,
                                                   const double *__restrict__ kh, double *__restrict__ D,
                                                   float *__restrict__ Df) {
    extern __shared__ unsigned char smem_raw[];
    const int cls = blockIdx.x, tid = threadIdx.x, P1 = p + 1;
    if (cls >= ncls) return;
    double *Gh = (double *)smem_raw;             // [(p+2)][2]
    double *up = Gh + 2 * (p + 2), *cur = up + 2 * np;
    const double rx = rho[3 * cls], ry = rho[3 * cls + 1], rz = rho[3 * cls + 2];
    if (tid == 0) {
        // G^(h) = (R^-1 d/dR)^h Ghat at |rho|; Laplace: G^(h+1) = -(2h+1) G^(h) / R^2;
        // Helmholtz adds -khat^2 G^(h-1) / R^2 with G^(-1) = -j e^{j khat R} / (4 pi khat)
        const double r2 = rx * rx + ry * ry + rz * rz, r1 = sqrt(r2), inv4pi = 0.25 / M_PI;
        if (C == 1) {
            double g = inv4pi / r1;
            for (int h = 0; h <= p; h++) {
                Gh[2 * h] = g;
                Gh[2 * h + 1] = 0.0;
                g = -(2.0 * h + 1.0) * g / r2;
            }
        } else {
            const double k = kh[cls];
            double sn, cs;
            sincos(k * r1, &sn, &cs);
            double pr = sn * inv4pi / k, pi = -cs * inv4pi / k, cr = cs * inv4pi / r1, ci = sn * inv4pi / r1;
            for (int h = 0; h <= p; h++) {
                Gh[2 * h] = cr;
                Gh[2 * h + 1] = ci;
                const double nr = -((2.0 * h + 1.0) * cr + k * k * pr) / r2;
                const double ni = -((2.0 * h + 1.0) * ci + k * k * pi) / r2;
                pr = cr; pi = ci; cr = nr; ci = ni;
            }
        }
        up[0] = Gh[2 * p];
        up[1] = Gh[2 * p + 1];
    }
    __syncthreads();
    const double rr[3] = {rx, ry, rz};
    for (int h = p - 1; h >= 0; h--) {
        const int top = p - h, n = (top + 1) * (top + 2) * (top + 3) / 6;
        for (int u = tid; u < n; u += TT) {
            const int m = tm[u], nn = tn[u], k = tk[u];
            double v0, v1;
            if (m + nn + k == 0) {
                v0 = Gh[2 * h];
                v1 = Gh[2 * h + 1];
            } else {
                const int ax = m > 0 ? 0 : (nn > 0 ? 1 : 2);
                const int g = ax == 0 ? m : (ax == 1 ? nn : k);
                const int m1 = m - (ax == 0), n1 = nn - (ax == 1), k1 = k - (ax == 2);
                const int i1 = idx3[(m1 * P1 + n1) * P1 + k1];
                v0 = rr[ax] * up[2 * i1];
                v1 = rr[ax] * up[2 * i1 + 1];
                if (g > 1) {
                    const int i2 = idx3[((m1 - (ax == 0)) * P1 + (n1 - (ax == 1))) * P1 + (k1 - (ax == 2))];
                    v0 += (g - 1) * up[2 * i2];
                    v1 += (g - 1) * up[2 * i2 + 1];
                }
            }
            cur[2 * u] = v0;
            cur[2 * u + 1] = v1;
        }
        __syncthreads();
        double *sw = up; up = cur; cur = sw;
        __syncthreads();
    }
    for (int u = tid; u < np; u += TT)
        for (int c = 0; c < C; c++) {
            const double v = up[2 * u + c];
            D[((size_t)cls * np + u) * C + c] = v;
            if (Df) Df[((size_t)cls * np + u) * C + c] = (float)v;
        }
}

// ---------------------------------------------------------------------------
// host: tables
// ---------------------------------------------------------------------------

// Offset classes: key (dl, level for Helmholtz, K).  Offsets of interacting
// boxes are small integers, so the key packs into 64 bits (17 bits per K
// component, biased) and goes into a flat open-addressing table (Fibonacci
// hashing: the product's top bits depend on every bit of the key; the table
// starts small and doubles at half load, so it stays in cache); a key that
// does not pack goes to an ordered map.  Per class its offset vector, level
// difference and key level, in order of first appearance.  The level field holds
// the source's box_reach (float64 plans) in its bits from 8 on; such keys do not pack.
struct ClassSet {
    std::vector<unsigned long long> tkey = std::vector<unsigned long long>(4096, 0ull);
    std::vector<int> tval = std::vector<int>(4096, -1);
    size_t tmask = 4095, tused = 0;
    int tbits = 12;
    std::map<std::tuple<int, int, long long, long long, long long>, int> wide;
    std::vector<int> dls, levs;
    std::vector<long long> kvec;
    int find_or_add(long long kx, long long ky, long long kz, int dl, int lv) {
        constexpr int KB = 17;
        constexpr long long KMAX = (1ll << (KB - 1)) - 1;
        if (std::llabs(kx) <= KMAX && std::llabs(ky) <= KMAX && std::llabs(kz) <= KMAX && dl > -64 && dl < 64 && lv < 64) {
            const unsigned long long key =
                1ull + (((unsigned long long)(kx + KMAX)) | ((unsigned long long)(ky + KMAX) << KB) |
                        ((unsigned long long)(kz + KMAX) << (2 * KB)) | ((unsigned long long)(dl + 64) << (3 * KB)) |
                        ((unsigned long long)lv << (3 * KB + 7)));
            unsigned long long *tk = tkey.data();
            size_t h = (size_t)((key * 0x9E3779B97F4A7C15ull) >> (64 - tbits));
            while (tk[h] != 0ull && tk[h] != key) h = (h + 1) & tmask;
            if (tk[h] == key) return tval[h];
            if (2 * (tused + 1) > tmask + 1) {
                grow();
                tk = tkey.data();
                h = (size_t)((key * 0x9E3779B97F4A7C15ull) >> (64 - tbits));
                while (tk[h] != 0ull) h = (h + 1) & tmask;
            }
            tk[h] = key;
            tused++;
            return tval[h] = add(kx, ky, kz, dl, lv);
        }
        auto wk = std::make_tuple(dl, lv, kx, ky, kz);
        auto it = wide.find(wk);
        if (it == wide.end()) it = wide.emplace(wk, add(kx, ky, kz, dl, lv)).first;
        return it->second;
    }
    int add(long long kx, long long ky, long long kz, int dl, int lv) {
        dls.push_back(dl);
        levs.push_back(lv);
        kvec.push_back(kx);
        kvec.push_back(ky);
        kvec.push_back(kz);
        return (int)dls.size() - 1;
    }
    void grow() {
        std::vector<unsigned long long> ok;
        std::vector<int> ov;
        ok.swap(tkey);
        ov.swap(tval);
        tmask = 2 * (tmask + 1) - 1;
        tbits++;
        tkey.assign(tmask + 1, 0ull);
        tval.assign(tmask + 1, -1);
        for (size_t i = 0; i < ok.size(); i++)
            if (ok[i]) {
                size_t h = (size_t)((ok[i] * 0x9E3779B97F4A7C15ull) >> (64 - tbits));
                while (tkey[h] != 0ull) h = (h + 1) & tmask;
                tkey[h] = ok[i];
                tval[h] = ov[i];
            }
    }
};

// the classes of the pairs of boxes [b0, b1), in a set of their own
static void number_classes(int b0, int b1, bool by_level, const int *reach, const int *lev, const int *ix, const int *iy, const int *iz,
                           const int *ip, const int *ii, int *pair_cls, ClassSet &S) {
    for (int b = b0; b < b1; b++) {
        const int lb = lev[b], xb = ix[b], yb = iy[b], zb = iz[b], lv = by_level ? lb : 0;
        for (int u = ip[b]; u < ip[b + 1]; u++) {
            const int s = ii[u], dl = lb - lev[s], e = std::max(0, -dl);
            // 2 rho 2^e = (2 i_t + 1) 2^e - (2 i_s + 1) 2^(dl + e), an integer vector
            const long long ft = 1ll << e, fs = 1ll << (dl + e);
            pair_cls[u] = S.find_or_add((2ll * xb + 1) * ft - (2ll * ix[s] + 1) * fs, (2ll * yb + 1) * ft - (2ll * iy[s] + 1) * fs,
                                        (2ll * zb + 1) * ft - (2ll * iz[s] + 1) * fs, dl, lv | reach[s] << 8);
        }
    }
}

// Offset classes of the interaction pairs (independent of the order p).
int build_m2l_classes(bem_plan *P) {
    const Tree &t = P->t;
    std::vector<int> lev(t.nbox), ix(t.nbox), iy(t.nbox), iz(t.nbox), ip(t.nbox + 1), ii(t.n_inter);
    BEM_CUDA(cudaMemcpy(lev.data(), t.level, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(ix.data(), t.ix, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(iy.data(), t.iy, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(iz.data(), t.iz, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    BEM_CUDA(cudaMemcpy(ip.data(), t.inter_ptr, sizeof(int) * (t.nbox + 1), cudaMemcpyDeviceToHost));
    if (t.n_inter) BEM_CUDA(cudaMemcpy(ii.data(), t.inter_idx, sizeof(int) * t.n_inter, cudaMemcpyDeviceToHost));
    std::vector<int> reach(t.nbox, 0);
    if (P->prm.precision == BEM_F64)
        BEM_CUDA(cudaMemcpy(reach.data(), t.reach, sizeof(int) * t.nbox, cudaMemcpyDeviceToHost));
    const bool helm = P->green == BEM_HELMHOLTZ;
    const bool by_level = helm || P->prm.p_min > 0;   // the target level enters the key
    // Classes are numbered in order of first appearance over the pairs in list
    // order.  The boxes are cut into up to three ranges of about equal pair
    // counts, numbered on threads of their own (number_classes); the ranges'
    // classes are then numbered together in range order, which is the
    // numbering of one pass over all pairs.
    const int64_t npair = t.n_inter;
    const int nth = (int)std::max<int64_t>(1, std::min<int64_t>(3, npair / 32768));
    std::vector<int> bcut(nth + 1, t.nbox);
    bcut[0] = 0;
    for (int k = 1, b = 0; k < nth; k++) {
        while (b < t.nbox && (int64_t)ip[b] * nth < npair * k) b++;
        bcut[k] = b;
    }
    std::vector<int> pair_cls(std::max<int64_t>(1, npair));
    std::vector<ClassSet> sets(nth);
    {
        std::vector<std::thread> th;
        for (int k = 1; k < nth; k++)
            th.emplace_back(number_classes, bcut[k], bcut[k + 1], by_level, reach.data(), lev.data(), ix.data(), iy.data(),
                            iz.data(), ip.data(), ii.data(), pair_cls.data(), std::ref(sets[k]));
        number_classes(bcut[0], bcut[1], by_level, reach.data(), lev.data(), ix.data(), iy.data(), iz.data(), ip.data(), ii.data(),
                       pair_cls.data(), sets[0]);
        for (auto &x : th) x.join();
    }
    // the first range's numbers are already global; later ranges' are mapped
    ClassSet &all = sets[0];
    for (int k = 1; k < nth; k++) {
        const ClassSet &R = sets[k];
        std::vector<int> to(R.dls.size());
        for (size_t c = 0; c < R.dls.size(); c++)
            to[c] = all.find_or_add(R.kvec[3 * c], R.kvec[3 * c + 1], R.kvec[3 * c + 2], R.dls[c], R.levs[c]);
        for (int u = ip[bcut[k]]; u < ip[bcut[k + 1]]; u++) pair_cls[u] = to[pair_cls[u]];
    }
    const std::vector<int> &dls = all.dls, &levs = all.levs;
    const std::vector<long long> &kvec = all.kvec;
    P->m2l_src_lmin = P->m2l_tgt_lmin = t.nlev;
    for (int b = 0; b < t.nbox; b++)
        if (ip[b + 1] > ip[b]) P->m2l_tgt_lmin = std::min(P->m2l_tgt_lmin, lev[b]);
    for (int64_t u = 0; u < t.n_inter; u++) P->m2l_src_lmin = std::min(P->m2l_src_lmin, lev[ii[u]]);
    return build_m2l_sym(P, pair_cls, kvec, dls, levs, ii, ip);
}

// derivative tables of ncls offset classes (rho: [class][3]; kh: [class], Helmholtz only)
int launch_m2l_derivs(bem_plan *P, int ncls, const double *rho, const double *kh, double *D, float *fD,
                      cudaStream_t s) {
    if (ncls <= 0) return BEM_OK;
    const int p = P->mi.p, np = P->mi.np, C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    const size_t sm = sizeof(double) * (2 * (p + 2) + 4 * (size_t)np) + 64;
    (k_m2l_tables<<<ncls, TT, sm, s>>>(ncls, p, np, C, P->d_m, P->d_n, P->d_k, P->d_idx3, rho, kh, D, fD),
     ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// M2L tables for the current order (called by alloc_fmm).
int build_translation_tables(bem_plan *P, cudaStream_t s) {
    // per-axis shift factors [M2M, L2L][a][g], in the plan's precision
    const int n = P->mi.p + 1;
    std::vector<double> b((size_t)(2 * n) * (2 * n), 0.0), G(2 * (size_t)n * n, 0.0);   // binomials, exact
    for (int i = 0; i < 2 * n; i++)
        for (int j = 0; j <= i; j++) b[i * 2 * n + j] = j == 0 || j == i ? 1.0 : b[(i - 1) * 2 * n + j - 1] + b[(i - 1) * 2 * n + j];
    for (int a = 0; a < n; a++)
        for (int g = 0; g < n; g++) {
            if (g <= a) G[a * n + g] = std::ldexp(b[a * 2 * n + g], -g);
            G[n * n + a * n + g] = std::ldexp(b[(a + g) * 2 * n + a], -2 * g);
        }
    const bool mx = P->prm.precision == BEM_MIXED;
    const std::vector<float> Gf(G.begin(), G.end());
    const size_t bytes = (mx ? sizeof(float) : sizeof(double)) * G.size();
    BEM_TRY(P->arena.alloc((char **)&P->shift_G, bytes));
    // (pageable source: staged before the call returns)
    BEM_CUDA(cudaMemcpyAsync(P->shift_G, mx ? (const void *)Gf.data() : (const void *)G.data(), bytes, cudaMemcpyHostToDevice, s));
    return build_sym_tables(P, s);
}

void free_translation_tables(bem_plan *P) {
    P->arena.release(P->shift_G);
    P->shift_G = nullptr;
    free_sym_tables(P);
}

// ---------------------------------------------------------------------------
// host: launchers
// ---------------------------------------------------------------------------
static int np_host(int q) { return (q + 1) * (q + 2) * (q + 3) / 6; }
static int level_order(const bem_plan *P, int l) {
    return l < (int)P->lev_p.size() ? P->lev_p[l] : P->mi.p;
}

// upward pass: moments of every parent from its children, level by level,
// up to level lmin (coarser moments are not formed)
template <class R, int C>
int launch_m2m(bem_plan *P, R *M, cudaStream_t s, int lmin) {
    const Tree &t = P->t;
    const int nps = P->mi.np;
    const int *sk = P->skip;
    for (int l = t.nlev - 2; l >= std::max(0, lmin); l--) {
        const int off = t.lev_off[l], cnt = t.lev_off[l + 1] - off;
        const int p = level_order(P, l), np = np_host(p), npc = np_host(level_order(P, l + 1));
        const size_t sm = sizeof(R) * 2 * np * C + shift_tab_bytes<R>(p, np);
        (k_m2m_sep<R, C><<<cnt * MM_CL, MM_T, sm, s>>>(off, t.child0, t.nchild, t.ix, t.iy, t.iz, p, np, nps, npc,
                                                       P->mi.p + 1, (const R *)P->shift_G, P->sy_mexp, M, sk),
         ::bem::count_launch());
    }
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

template <class R, int C>
int launch_translations(bem_plan *P, R *M, R *L, cudaStream_t s, cudaEvent_t *ev) {
    const Tree &t = P->t;
    const int np = P->mi.np;
    const int *sk = P->skip;
    // M2L reads moments at levels >= m2l_src_lmin only, and every local
    // coarser than m2l_tgt_lmin is zero (the gathers write each box's local),
    // so the upward pass stops at the first and the downward one starts below
    // the second
    BEM_TRY((launch_m2m<R, C>(P, M, s, P->m2l_src_lmin)));
    BEM_LAUNCH_CHECK();
    if (ev) BEM_CUDA(cudaEventRecord(ev[3], s));
    if (std::is_same<R, float>::value && C == 1 && P->sy_tc) {
        BEM_TRY(launch_m2l_tc(P, (const float *)M, (float *)L, s));
    } else {
        BEM_TRY((launch_m2l_sy<R, C>(P, M, L, s)));
    }
    BEM_LAUNCH_CHECK();
    if (ev) BEM_CUDA(cudaEventRecord(ev[4], s));
    for (int l = std::max(1, P->m2l_tgt_lmin + 1); l < t.nlev; l++) {
        // the shift runs at the parent's order; the child keeps its own order's terms
        const int off = t.lev_off[l], cnt = t.lev_off[l + 1] - off;
        const int p = level_order(P, l - 1), pnp = np_host(p), npo = np_host(level_order(P, l));
        const size_t tab_sm = shift_tab_bytes<R>(p, pnp);
        const int n = P->mi.p + 1;
        (k_l2l_sep<R, C><<<cnt, MM_T, sizeof(R) * 2 * pnp * C + tab_sm, s>>>(off, t.parent, t.ix, t.iy, t.iz, p, pnp, np, npo,
                                                                           n, (const R *)P->shift_G + n * n, P->sy_mexp,
                                                                           L, sk),
         ::bem::count_launch());
    }
    BEM_LAUNCH_CHECK();
    if (ev) BEM_CUDA(cudaEventRecord(ev[5], s));
    return BEM_OK;
}

// large dynamic shared memory for every instantiation (outside any capture)
void set_translation_attributes() {
    const int big = 220 * 1024;
    cudaFuncSetAttribute(k_m2l_tables, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_m2m_sep<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_m2m_sep<double, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_m2m_sep<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_m2m_sep<float, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_l2l_sep<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_l2l_sep<double, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_l2l_sep<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    cudaFuncSetAttribute(k_l2l_sep<float, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    set_tc_attributes();
    set_sy_attributes();
}

template int launch_m2m<double, 1>(bem_plan *, double *, cudaStream_t, int);
template int launch_m2m<double, 2>(bem_plan *, double *, cudaStream_t, int);
template int launch_m2m<float, 1>(bem_plan *, float *, cudaStream_t, int);
template int launch_m2m<float, 2>(bem_plan *, float *, cudaStream_t, int);
template int launch_translations<double, 1>(bem_plan *, double *, double *, cudaStream_t, cudaEvent_t *);
template int launch_translations<double, 2>(bem_plan *, double *, double *, cudaStream_t, cudaEvent_t *);
template int launch_translations<float, 1>(bem_plan *, float *, float *, cudaStream_t, cudaEvent_t *);
template int launch_translations<float, 2>(bem_plan *, float *, float *, cudaStream_t, cudaEvent_t *);

const void *kernel_of_translate() { return (const void *)k_m2l_tables; }

}  // namespace bem

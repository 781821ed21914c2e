// M2L (Eq. 7) on the canonical offset classes on the float32 pipe: every
// product the tensor-core form does not take (float32 Helmholtz, float64 of
// either Green's function, level-dependent orders and orders beyond the
// tensor-core tables).
//
// A tile holds up to 64 pairs of one canonical class and its block computes
//     Lhat[pair][b] = sum_a T[b][a] Mhat[pair][a],
//     T[b][a] = Dhat[a + b] (-1)^|a| 2^(dl |a|) / (a! b!)   (|a| + |b| <= p),
// with Mhat the sign-permuted moments of the pair's source box.  A value is a
// number of float32 words: one per real component in float32 plans, a pair
// (h, l) of 48 bits (dfloat.cuh) in float64 plans, whose float64 arithmetic
// would run at 1/64 of the rate.
//
// What bounds it: 8,008 multiply-adds a pair at p = 10 (four times as many
// complex ones; 13 operations each in pairs), in a triangle: column a reaches
// the rows |b| <= p - |a|, 286 of them for the first column and one for each of
// the last 66.  So (1) a warp holds rows, two to a packed operand, its lanes
// pairs (two each): a T value is one broadcast shared-memory read for 64 pairs
// and every warp walks only the columns that reach its rows, with no
// divergence; rows go round the warps in blocks of two, so all have about the
// same work.  (2) The columns that reach only a few rows (the last three
// degrees, 166 of 286 columns with 9 % of the products) are dealt out to the
// warps instead, each computing all their rows, and the warps' sums are added
// in warp order.  (3) T is laid out once per plan in the order it is consumed,
// the moments are permuted once per product so that they load in whole rows,
// and both come with cp.async, 16 columns a stage, three stages in flight; a
// lane applies its pairs' reflection signs as it reads them.
//
// Measured, M2L stage: Helmholtz in float32 on a sphere of 20,480 tri6
// (241,778 pairs) 2433 -> 790 us, on 81,920 (858,978) 7957 -> 2710; float64 on a
// cube of 8,748 tri6 1656 -> 228, Helmholtz on 2,880 1528 -> 325, the level-3
// sphere 268 -> 48.  58,800 complex pairs take 184 us, FMA pipe 39 % busy, issue
// slots 62 %: each (warp, column) visit costs some 20 instructions beside its
// packed multiply-adds.  Not kept: 18 row blocks a warp and half the warps
// (fewer visits, 28 % fewer instructions, but 283 us: too few warps to cover
// latency), 9 blocks at two blocks per SM (230), 4 at four (190), unpacked
// multiply-adds (261), packing over the pairs (275: T copied twice into
// registers).  The form before rebuilt T for every tile and walked every column
// in every warp (FMA pipe 23 % busy).
// In float64 plans a source box with box_reach e > 0 enters with its moments x
// 2^(-e |a|), and the class's dl (part of its key) holds e beside the level
// difference.
// Rows go to a buffer pair by pair and a gather sums each target's in list
// order: deterministic, no atomics.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dfloat.cuh"
#include "fmm_views.cuh"

namespace bem {

namespace {

// SY_PERMS as two bits per entry, for device code
constexpr unsigned long long pack_perms() {
    unsigned long long v = 0;
    for (int q = 0; q < 6; q++)
        for (int i = 0; i < 3; i++) v |= (unsigned long long)SY_PERMS[q][i] << (8 * q + 2 * i);
    return v;
}
// canonical axis of a pair's axis i under axis permutation q
__device__ __forceinline__ int sy_perm(int q, int i) {
    constexpr unsigned long long packed = pack_perms();
    return (int)(packed >> (8 * q + 2 * i)) & 3;
}

constexpr int MG_T = 256, MG_W = MG_T / 32;   // threads, warps (row groups)
constexpr int MG_PT = 64;                     // pairs per tile
constexpr int MG_KA = 16;                     // columns per stage
constexpr int MG_ST = 3;                      // stages in flight
constexpr int MG_TILE = 128;                  // pairs per tile of the plan's tables

// A row block: RB rows of WC words, in row pairs (one packed operand per word):
// float2 (row 0, row 1) of each word in turn; VB float4.
__host__ __device__ constexpr int mg_rb(int WC) { return WC == 1 ? 4 : 2; }
__host__ __device__ constexpr int mg_vb(int WC) { return mg_rb(WC) * WC / 4; }
// row blocks per warp (48, 72 or 64 accumulators a thread, for three blocks per
// SM in float32 and two in pairs) and per row chunk
__host__ __device__ constexpr int mg_nb(int W, int C) { return W == 1 ? 6 : C == 1 ? 9 : 4; }
__host__ __device__ constexpr int mg_cb(int W, int C) { return MG_W * mg_nb(W, C); }
__host__ __device__ constexpr int mg_rows(int W, int C) { return mg_cb(W, C) * mg_rb(W * C); }
__host__ __device__ constexpr int mg_kstride(int WC) { return WC * MG_PT + 4; }   // floats per staged moment column
__host__ __device__ constexpr int mg_tstride(int W, int C) { return mg_cb(W, C) * mg_vb(W * C); }   // float4 per staged T column
// shared memory: the T and moment stages, reused for the warps' partial sums
// and for the output rows, then the column table
__host__ __device__ constexpr size_t mg_t_bytes(int W, int C) { return sizeof(float4) * MG_ST * MG_KA * mg_tstride(W, C); }
__host__ __device__ constexpr size_t mg_work(int W, int C) {
    const int WC = W * C;
    const size_t st = mg_t_bytes(W, C) + sizeof(float) * MG_ST * MG_KA * mg_kstride(WC);
    const size_t part = sizeof(float2) * mg_cb(W, C) * mg_rb(WC) * WC * 32;
    const size_t out = sizeof(float) * MG_PT * (mg_rows(W, C) * WC + 1);
    const size_t m = st > part ? (st > out ? st : out) : (part > out ? part : out);
    return (m + 15) / 16 * 16;
}
static size_t mg_smem(int W, int C, int np) { return mg_work(W, C) + 9 * (size_t)((np + MG_KA + 7) / 8 * 8); }

__host__ __device__ __forceinline__ int n_upto(int q) { return q < 0 ? 0 : (q + 1) * (q + 2) * (q + 3) / 6; }

struct GemmArgs {
    int np, ldp, ldq, u0, kt;                 // kt: first column of the dealt-out tail of row chunk 0
    int cls0;                                 // class of the first image held
    size_t img_vec;                           // float4 of a class's image
    const int *tile_cls, *tile_start, *tile_cnt;
    const int *src, *sig, *pair;
    const int *colx;                          // [np] (row blocks a column reaches | end of its degree << 16, first float4 in the image)
    const int *mexp;                          // [np] exponents m | n << 8 | k << 16 | degree << 24
    const float4 *img;                        // [class - cls0][img_vec]
    const float *Mq;                          // [box][6][ldq][WC]
    float *Lp;                                // [pair][ldp][WC]
    const int *skip;
};

template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// words t of a row pair times a pair's moment words m (nm: their negatives)
template <int W, int C>
__device__ __forceinline__ void row_mac(const P2 *t, const P2 *m, const P2 *nm, P2 *acc) {
    auto mac = [](P2 th, P2 tl, P2 mh, P2 nmh, P2 ml, P2 &h, P2 &l) {
        const P2 p = pmul(th, mh);
        P2 e = pfma(th, mh, pmul(th, nmh)), s, r;
        e = pfma(th, ml, e);
        e = pfma(tl, mh, e);
        two_sum(h, p, s, r);
        h = s;
        l = padd(l, padd(r, e));
    };
    if constexpr (W == 1 && C == 1) {
        acc[0] = pfma(t[0], m[0], acc[0]);
    } else if constexpr (W == 1 && C == 2) {
        acc[0] = pfma(t[0], m[0], acc[0]);
        acc[1] = pfma(t[0], m[1], acc[1]);
        acc[0] = pfma(t[1], nm[1], acc[0]);
        acc[1] = pfma(t[1], m[0], acc[1]);
    } else if constexpr (C == 1) {
        mac(t[0], t[1], m[0], nm[0], m[1], acc[0], acc[1]);
    } else {                                  // words re h, re l, im h, im l
        mac(t[0], t[1], m[0], nm[0], m[1], acc[0], acc[1]);
        mac(t[0], t[1], m[2], nm[2], m[3], acc[2], acc[3]);
        mac(t[2], t[3], nm[2], m[2], nm[3], acc[0], acc[1]);
        mac(t[2], t[3], m[0], nm[0], m[1], acc[2], acc[3]);
    }
}

// n columns, every cs-th, against N row blocks, every step-th.  par: the
// columns' exponent parities; s0, s1: this lane's two pairs' signs by parity.
template <int W, int C, int N, int NA>
__device__ __forceinline__ void run_columns(int n, int cs, int step, const float4 *T, const float *M,
                                            const unsigned char *par, unsigned s0, unsigned s1,
                                            P2 (&acc)[mg_nb(W, C)][2][NA]) {
    constexpr int WC = W * C, VB = mg_vb(WC), KS = mg_kstride(WC), TS = mg_tstride(W, C), RP = mg_rb(WC) / 2;
    constexpr int U = W == 2 ? 1 : (N >= 4 ? 1 : (N >= 2 ? 2 : 4));   // columns in flight
    auto columns = [&](auto u_const) {
        constexpr int V = decltype(u_const)::value;
        float4 t[V][N * VB];
        float mv[V][2][WC];
        unsigned pb[V];
#pragma unroll
        for (int u = 0; u < V; u++) {
            const float *q = M + u * cs * KS;
            pb[u] = par[u * cs];
            if constexpr (WC == 1) {
                const float2 x = *reinterpret_cast<const float2 *>(q);
                mv[u][0][0] = x.x; mv[u][1][0] = x.y;
            } else {
#pragma unroll
                for (int w = 0; w < 2 * WC; w += 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(q + w);
                    mv[u][w / WC][w % WC] = x.x;
                    mv[u][w / WC][w % WC + 1] = x.y;
                    mv[u][(w + 2) / WC][(w + 2) % WC] = x.z;
                    mv[u][(w + 2) / WC][(w + 2) % WC + 1] = x.w;
                }
            }
#pragma unroll
            for (int i = 0; i < N; i++)
#pragma unroll
                for (int v = 0; v < VB; v++) t[u][i * VB + v] = T[u * cs * TS + i * step * VB + v];
        }
#pragma unroll
        for (int u = 0; u < V; u++)
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const unsigned sg = ((j ? s1 : s0) << (31 - pb[u])) & 0x80000000u;
                P2 m[WC], nm[WC];
#pragma unroll
                for (int w = 0; w < WC; w++) {
                    m[w] = p2(__uint_as_float(__float_as_uint(mv[u][j][w]) ^ sg));
                    nm[w] = p2(__uint_as_float(__float_as_uint(mv[u][j][w]) ^ sg ^ 0x80000000u));
                }
#pragma unroll
                for (int i = 0; i < N; i++) {
                    P2 tv[VB * 2];
#pragma unroll
                    for (int v = 0; v < VB; v++) {
                        tv[2 * v] = make_float2(t[u][i * VB + v].x, t[u][i * VB + v].y);
                        tv[2 * v + 1] = make_float2(t[u][i * VB + v].z, t[u][i * VB + v].w);
                    }
#pragma unroll
                    for (int r = 0; r < RP; r++) row_mac<W, C>(tv + r * WC, m, nm, acc[i][j] + r * WC);
                }
            }
        T += V * cs * TS;
        M += V * cs * KS;
        par += V * cs;
    };
    int k = 0;
    for (; k + U <= n; k += U) columns(std::integral_constant<int, U>{});
    if constexpr (U > 1)
        for (; k < n; k++) columns(std::integral_constant<int, 1>{});
}

template <int W, int C>
__global__ void __launch_bounds__(MG_T, W == 1 ? 3 : 2) k_m2l_gemm(const __grid_constant__ GemmArgs a) {
    if (a.skip && *a.skip) return;
    constexpr int WC = W * C, RB = mg_rb(WC), VB = mg_vb(WC), NB = mg_nb(W, C), CB = mg_cb(W, C), KS = mg_kstride(WC),
                  TS = mg_tstride(W, C), OS = mg_rows(W, C) * WC + 1, NA = RB / 2 * WC;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int sSrc[MG_PT], sPair[MG_PT];
    __shared__ unsigned sSgn[MG_PT];
    const int tile = blockIdx.x >> 1, half = blockIdx.x & 1;
    const int cnt = min(MG_PT, a.tile_cnt[tile] - half * MG_PT);
    if (cnt <= 0) return;
    const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
    const int cls = a.tile_cls[tile], st = a.tile_start[tile] + half * MG_PT;
    float4 *sT = (float4 *)smem;                          // [MG_ST][MG_KA][TS]
    float *sM = (float *)(smem + mg_t_bytes(W, C));       // [MG_ST][MG_KA][KS]: [pair][word]
    float2 *sP = (float2 *)smem;                          // [warp][block][pair][value][lane]
    float *sO = (float *)smem;                            // [pair][OS]
    int2 *sCol = (int2 *)(smem + mg_work(W, C));          // [np]
    unsigned char *sPar = (unsigned char *)(sCol + (a.np + MG_KA + 7) / 8 * 8);   // [np] exponent parities
    for (int k = tid; k < a.np; k += MG_T) {
        sCol[k] = __ldg((const int2 *)a.colx + k);
        const int e = __ldg(a.mexp + k);
        sPar[k] = (unsigned char)((e & 1) | (e >> 7 & 2) | (e >> 14 & 4));
    }
    if (tid < MG_PT) {
        const int j = st + (tid < cnt ? tid : 0);         // off slots repeat the first pair
        const int sig = a.sig[j], q = sig >> 3, sb = sig & 7;
        sSrc[tid] = a.src[j] * 6 + q;
        sPair[tid] = a.pair[j] - a.u0;
        // sign of a canonical column: the parity of its exponents under the
        // pair's reflections, taken to the canonical axes (canonical axis
        // perm(i) is the pair's axis i), as one bit per exponent parity
        int cb = 0;
#pragma unroll
        for (int i = 0; i < 3; i++)
            if (sb >> i & 1) cb |= 1 << sy_perm(q, i);
        unsigned tab = 0;
#pragma unroll
        for (int e = 0; e < 8; e++) tab |= (unsigned)(__popc(cb & e) & 1) << e;
        sSgn[tid] = tab;
    }
    __syncthreads();
    const unsigned s0 = sSgn[2 * lane], s1 = sSgn[2 * lane + 1];
    const float4 *img = a.img + (size_t)(cls - a.cls0) * a.img_vec;
    // starts a stage's copies: the moments of its columns (whole row segments),
    // T blocks [b0, b0 + CB) and the columns' parities
    auto copy = [&](int k0, int b0, int buf) {
        const int c = tid & (MG_KA - 1);
        float *d = sM + ((size_t)buf * MG_KA + c) * KS;
#pragma unroll
        for (int i = 0; i < MG_KA * MG_PT / MG_T; i++) {
            const int j = tid / MG_KA + (MG_T / MG_KA) * i;
            cp_async<4 * WC>(d + j * WC, a.Mq + ((size_t)sSrc[j] * a.ldq + k0 + c) * WC);
        }
        for (int q = g; q < MG_KA; q += MG_W) {
            const int k = k0 + q;
            if (k >= a.np) break;
            const int nv = min(CB, (sCol[k].x & 0xffff) - b0) * VB;
            const float4 *s = img + sCol[k].y + b0 * VB;
            float4 *t = sT + ((size_t)buf * MG_KA + q) * TS;
            for (int i = lane; i < nv; i += 32) cp_async<16>(t + i, s + i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    P2 acc[NB][2][NA];                                    // [block][pair][row pair, word]
    // columns [kb, ke) of the stages from k0 on: in the tail a warp takes every
    // eighth column with all its rows, otherwise every column with its own rows
    auto walk = [&](int kb, int ke, int b0, bool tail) {
        const int f = kb / MG_KA, n = (ke + MG_KA - 1) / MG_KA - f;
        if (n <= 0) return;
#pragma unroll
        for (int i = 0; i < MG_ST - 1; i++) {
            if (i < n) copy((f + i) * MG_KA, b0, i);
            else asm volatile("cp.async.commit_group;" ::: "memory");
        }
        for (int s = 0; s < n; s++) {
            asm volatile("cp.async.wait_group %0;" ::"n"(MG_ST - 2) : "memory");
            __syncthreads();                              // stage s is there; stage s - 1 is consumed
            if (s + MG_ST - 1 < n) copy((f + s + MG_ST - 1) * MG_KA, b0, (s + MG_ST - 1) % MG_ST);
            else asm volatile("cp.async.commit_group;" ::: "memory");
            const int buf = s % MG_ST, off = (f + s) * MG_KA;
            const float4 *T = sT + (size_t)buf * MG_KA * TS;
            const float *M = sM + (size_t)buf * MG_KA * KS + 2 * lane * WC;
            const int k1 = min(ke, off + MG_KA), step = tail ? 1 : MG_W;
            // columns of one degree reach the same rows: one run of this
            // warp's block count after the other
            for (int k = max(kb, off); k < k1;) {
                const int cx = sCol[k].x, kend = min(k1, cx >> 16), blocks = min(CB, (cx & 0xffff) - b0);
                const int nb = tail ? blocks : (blocks - g + MG_W - 1) / MG_W;   // this warp's blocks
                const int k0 = tail ? k + ((g - k) & (MG_W - 1)) : k, cs = tail ? MG_W : 1;
                const int nc = tail ? (kend - k0 + MG_W - 1) / MG_W : kend - k0;
                const float4 *t = T + (k0 - off) * TS + (tail ? 0 : g * VB);
                const float *m = M + (k0 - off) * KS;
                const unsigned char *par = sPar + k0;
#define MG_RUN(N_)                                                                                              \
    case N_:                                                                                                    \
        if constexpr (N_ <= NB) run_columns<W, C, N_, NA>(nc, cs, step, t, m, par, s0, s1, acc);                \
        break;
                switch (nb) {
                    MG_RUN(1) MG_RUN(2) MG_RUN(3) MG_RUN(4) MG_RUN(5) MG_RUN(6) MG_RUN(7) MG_RUN(8) MG_RUN(9)
                default: break;
                }
#undef MG_RUN
                k = kend;
            }
        }
        __syncthreads();                                  // the stages are free
    };
    for (int b0 = 0; b0 * RB < a.np; b0 += CB) {
#pragma unroll
        for (int i = 0; i < NB; i++)
#pragma unroll
            for (int r = 0; r < 2 * NA; r++) acc[i][r / NA][r % NA] = p2(0.f);
        // columns that reach this chunk (the rows reached fall with the column)
        int ke = a.np;
        if (b0 > 0) {
            int lo = 0, hi = a.np;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((sCol[mid].x & 0xffff) > b0) lo = mid + 1; else hi = mid;
            }
            ke = lo;
        }
        if (b0 == 0 && a.kt < ke) {
            walk(a.kt, ke, 0, true);
            // the warps' sums of the tail's rows, added by the rows' owners
#pragma unroll
            for (int i = 0; i < NB; i++)
#pragma unroll
                for (int r = 0; r < 2 * NA; r++) sP[((g * NB + i) * 2 * NA + r) * 32 + lane] = acc[i][r / NA][r % NA];
            __syncthreads();
#pragma unroll
            for (int i = 0; i < NB; i++) {
                const int b = g + MG_W * i;
#pragma unroll
                for (int r = 0; r < 2 * NA; r++) acc[i][r / NA][r % NA] = p2(0.f);
                if (b < NB)
                    for (int w = 0; w < MG_W; w++) {
                        const float2 *q = sP + (size_t)((w * NB + b) * 2 * NA) * 32 + lane;
#pragma unroll
                        for (int r = 0; r < 2 * NA; r += W) {
                            P2 *d = &acc[i][r / NA][r % NA];
                            if constexpr (W == 1) {
                                d[0] = padd(d[0], q[r * 32]);
                            } else {
                                P2 h, e;
                                two_sum(d[0], q[r * 32], h, e);
                                d[0] = h;
                                d[1] = padd(d[1], padd(e, q[(r + 1) * 32]));
                            }
                        }
                    }
            }
            __syncthreads();
            ke = a.kt;
        }
        walk(0, ke, b0, false);
        // rows to shared memory pair by pair, then whole rows out
#pragma unroll
        for (int i = 0; i < NB; i++)
#pragma unroll
            for (int j = 0; j < 2; j++) {
                float *d = sO + (size_t)(2 * lane + j) * OS + (g + MG_W * i) * RB * WC;
#pragma unroll
                for (int r = 0; r < NA; r++) {            // row pair r / WC, word r % WC
                    d[(r / WC * 2) * WC + r % WC] = acc[i][j][r].x;
                    d[(r / WC * 2 + 1) * WC + r % WC] = acc[i][j][r].y;
                }
            }
        __syncthreads();
        const int n = min(mg_rows(W, C), a.np - b0 * RB) * WC;
        for (int j = g; j < cnt; j += MG_W) {
            float *o = a.Lp + ((size_t)sPair[j] * a.ldp + b0 * RB) * WC;
            for (int i = lane; i < n; i += 32) o[i] = sO[(size_t)j * OS + i];
        }
        __syncthreads();
    }
}

// Moments under each axis permutation, in words, one block per box; float64
// plans scale each box's by a power of two (its largest exponent, to E[box]),
// and by 2^(-reach |a|) where its points reach far beyond its edge
template <class R, int C>
__global__ void __launch_bounds__(256) k_m2l_words(int np, int ldq, const unsigned short *__restrict__ fwd,
                                                   const int *__restrict__ mexp, const int *__restrict__ reach_of,
                                                   const R *__restrict__ M, float *__restrict__ Mq, int *__restrict__ Eb,
                                                   const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int WC = (sizeof(R) == 8 ? 2 : 1) * C;
    const size_t box = blockIdx.x;
    const R *m = M + box * np * C;
    const int reach = sizeof(R) == 8 ? __ldg(reach_of + box) : 0;
    auto moment = [&](int i) -> R {                       // i = coefficient x C + component
        if constexpr (sizeof(R) == 8)
            if (reach) return scalbn(m[i], -reach * (__ldg(mexp + i / C) >> 24));
        return m[i];
    };
    int E = 1;
    if constexpr (sizeof(R) == 8) {
        __shared__ int we[8];
        for (int i = threadIdx.x; i < np * C; i += 256) E = max(E, (int)((unsigned)__double2hiint(moment(i)) >> 20) & 0x7ff);
#pragma unroll
        for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
        if ((threadIdx.x & 31) == 0) we[threadIdx.x >> 5] = E;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; w++) E = max(E, we[w]);
        E = min(E, 2046);                                 // an infinity or NaN carries itself
        if (threadIdx.x == 0) Eb[box] = E;
    }
    for (int i = threadIdx.x; i < 6 * ldq; i += 256) {
        const int q = i / ldq, k = i - q * ldq;
        float v[WC];
#pragma unroll
        for (int w = 0; w < WC; w++) v[w] = 0.f;
        if (k < np) {
            const int f = __ldg(fwd + (size_t)q * 8 * np + k) & 0x7fff;
#pragma unroll
            for (int c = 0; c < C; c++) {
                if constexpr (sizeof(R) == 8) df_bits(moment(f * C + c), E, v[2 * c], v[2 * c + 1]);
                else v[c] = m[f * C + c];
            }
        }
        float *d = Mq + (box * 6 * ldq + i) * WC;
#pragma unroll
        for (int w = 0; w < WC; w++) d[w] = v[w];
    }
}

// L_t[b] = (1 / h_t) sum over t's interaction list, in list order, of
// sign * Lhat_u[b o pi_u^-1].  A block takes 96 rows of one target and
// splits the list into four interleaved parts, added in order (one thread per
// row walked the list alone before: 15 % of the warps resident, bound by load
// latency).  float64 plans: rows are pairs at their source box's scale, summed
// as pairs at the largest scale in the list.
constexpr int GA_R = 96, GA_S = 4, GA_LIST = 256;
template <class R, int C>
__global__ void __launch_bounds__(GA_R *GA_S) k_m2l_gather_sy(int t0, const int *__restrict__ level, double side,
                                                              const int *__restrict__ lev_p, const int *__restrict__ inter_ptr,
                                                              const int *__restrict__ inter_idx, const int *__restrict__ Eb,
                                                              int u0r, int np, int ldp, const int *__restrict__ sig_u,
                                                              const int *__restrict__ inv, const float *__restrict__ Lp,
                                                              R *__restrict__ L, const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int W = sizeof(R) == 8 ? 2 : 1, WC = W * C;
    __shared__ int sOff[GA_LIST];
    __shared__ float sSc[GA_LIST];
    __shared__ float red[GA_S][GA_R][WC];
    __shared__ int we[GA_R * GA_S / 32];
    const int t = t0 + blockIdx.x, tid = threadIdx.x, r = tid % GA_R, sl = tid / GA_R;
    const int u0 = inter_ptr[t], u1 = inter_ptr[t + 1];
    const int npt = lev_p ? n_upto(lev_p[level[t]]) : np;   // the target's own coefficients
    if ((int)blockIdx.y * GA_R >= npt) return;
    const int b = blockIdx.y * GA_R + r;
    int E = 1;
    if constexpr (W == 2) {
        for (int u = u0 + tid; u < u1; u += GA_R * GA_S) E = max(E, Eb[inter_idx[u]]);
#pragma unroll
        for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
        if ((tid & 31) == 0) we[tid >> 5] = E;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < GA_R * GA_S / 32; w++) E = max(E, we[w]);
    }
    float sum[WC];
#pragma unroll
    for (int w = 0; w < WC; w++) sum[w] = 0.f;
    for (int base = u0; base < u1; base += GA_LIST) {
        const int n = min(GA_LIST, u1 - base);
        __syncthreads();
        for (int i = tid; i < n; i += GA_R * GA_S) {
            sOff[i] = sig_u[base + i] * np;
            // 2^(e - E), zero when below float32's range
            if constexpr (W == 2) {
                const int e = Eb[inter_idx[base + i]] - E + 127;
                sSc[i] = e > 0 ? __uint_as_float((unsigned)e << 23) : 0.f;
            }
        }
        __syncthreads();
        if (b < npt) {
            constexpr int U = WC == 4 ? 4 : 8;            // rows in flight
            for (int i0 = sl; i0 < n; i0 += GA_S * U) {
                int f[U];
                float v[U][WC];
#pragma unroll
                for (int q = 0; q < U; q++) {
                    const int i = i0 + GA_S * q;
                    f[q] = i < n ? __ldg(inv + sOff[i] + b) : 0;
                }
#pragma unroll
                for (int q = 0; q < U; q++) {
                    const int i = i0 + GA_S * q;
#pragma unroll
                    for (int w = 0; w < WC; w++) v[q][w] = 0.f;
                    if (i < n) {
                        const float *p = Lp + ((size_t)(base + i - u0r) * ldp + (f[q] & 0x7fffffff)) * WC;
                        if constexpr (WC == 1) {
                            v[q][0] = __ldg(p);
                        } else if constexpr (WC == 2) {
                            const float2 x = __ldg((const float2 *)p);
                            v[q][0] = x.x; v[q][1] = x.y;
                        } else {
                            const float4 x = __ldg((const float4 *)p);
                            v[q][0] = x.x; v[q][1] = x.y; v[q][WC - 2] = x.z; v[q][WC - 1] = x.w;
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < U; q++) {
                    const int i = i0 + GA_S * q;
                    if (i >= n) break;
                    const unsigned sg = (unsigned)f[q] & 0x80000000u;
                    if constexpr (W == 1) {
#pragma unroll
                        for (int c = 0; c < C; c++) sum[c] += __uint_as_float(__float_as_uint(v[q][c]) ^ sg);
                    } else {
                        const float sc = __uint_as_float(__float_as_uint(sSc[i]) ^ sg);
#pragma unroll
                        for (int c = 0; c < C; c++) df_add(sum[2 * c], sum[2 * c + 1], v[q][2 * c] * sc, v[q][2 * c + 1] * sc);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int w = 0; w < WC; w++) red[sl][r][w] = sum[w];
    __syncthreads();
    if (sl == 0 && b < npt) {
        for (int q = 1; q < GA_S; q++) {
            if constexpr (W == 1) {
#pragma unroll
                for (int c = 0; c < C; c++) sum[c] += red[q][r][c];
            } else {
#pragma unroll
                for (int c = 0; c < C; c++) df_add(sum[2 * c], sum[2 * c + 1], red[q][r][2 * c], red[q][r][2 * c + 1]);
            }
        }
        const double ih = 1.0 / scalbn(side, -level[t]);
#pragma unroll
        for (int c = 0; c < C; c++) {
            if constexpr (W == 1) L[((size_t)t * np + b) * C + c] = sum[c] * (R)ih;
            else L[((size_t)t * np + b) * C + c] = ((double)sum[2 * c] + (double)sum[2 * c + 1]) * scalbn(ih, E - 1023);
        }
    }
}

// T of every class in image order: column a (blockIdx.y), rows by thread
template <int W, int C>
__global__ void __launch_bounds__(256) k_m2l_image(int cls0, int np, int p, size_t img_vec, const int *__restrict__ colx,
                                                   const int *__restrict__ mexp, const int *__restrict__ idx3,
                                                   const double *__restrict__ invf, const double *__restrict__ D,
                                                   const int *__restrict__ dl, const int *__restrict__ ord, float *img,
                                                   const int *__restrict__ skip) {
    if (skip && *skip) return;
    constexpr int WC = W * C;
    const int cls = cls0 + blockIdx.x, a = blockIdx.y, P1 = p + 1;
    const int ps = ord[2 * cls], pt = ord[2 * cls + 1], pm = max(ps, pt);
    const int ea = mexp[a], da = ea >> 24;
    const double fa = ((da & 1) ? -1.0 : 1.0) * ldexp(invf[a], dl[cls] * da);
    constexpr int RB = mg_rb(WC);
    float *out = img + ((size_t)blockIdx.x * img_vec + colx[2 * a + 1]) * 4;
    for (int b = threadIdx.x; b < (colx[2 * a] & 0xffff) * RB; b += 256) {
        float v[WC];
#pragma unroll
        for (int w = 0; w < WC; w++) v[w] = 0.f;
        if (b < np) {
            const int eb = mexp[b], db = eb >> 24;
            // moments |a| <= ps, locals |b| <= pt, |a| + |b| <= max(ps, pt)
            if (da <= ps && db <= pt && da + db <= pm) {
                const int m = (ea & 0xff) + (eb & 0xff), n = ((ea >> 8) & 0xff) + ((eb >> 8) & 0xff),
                          k = ((ea >> 16) & 0xff) + ((eb >> 16) & 0xff);
                const double f = fa * invf[b];
                const double *d = D + ((size_t)cls * np + idx3[(m * P1 + n) * P1 + k]) * C;
#pragma unroll
                for (int c = 0; c < C; c++) {
                    if constexpr (W == 1) v[c] = (float)(d[c] * f);
                    else df_split(d[c] * f, v[2 * c], v[2 * c + 1]);
                }
            }
        }
#pragma unroll
        for (int w = 0; w < WC; w++)
            out[(size_t)(b / RB) * RB * WC + (b % RB / 2 * WC + w) * 2 + (b & 1)] = v[w];
    }
}

}  // namespace

static int launch_images(bem_plan *P, int cls0, int n, const int *skip, cudaStream_t s) {
    const bool mx = P->prm.precision == BEM_MIXED, cx = P->green == BEM_HELMHOLTZ;
    auto go = [&](auto kernel) {
        (kernel<<<dim3(n, P->mi.np), 256, 0, s>>>(cls0, P->mi.np, P->mi.p, P->sg_vec, P->sg_colx, P->sy_mexp, P->d_idx3,
                                                  P->sy_invf, P->sy_D, P->sy_dl, P->sy_ord, (float *)P->sg_img, skip),
         ::bem::count_launch());
    };
    if (mx) cx ? go(k_m2l_image<1, 2>) : go(k_m2l_image<1, 1>);
    else cx ? go(k_m2l_image<2, 2>) : go(k_m2l_image<2, 1>);
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// The SIMT form's tables of the current order: column extents, class images,
// permuted-moment buffer.  The images stay for the plan's life when they fit
// SG_IMG_BYTES + SG_IMG_NODE per node (71 KB a class at p = 10 in float64);
// else (high orders: 640 KB a class at the float64 diagonal's p = 16) they are
// built per product, as many classes at a time as fit.
constexpr size_t SG_IMG_BYTES = (size_t)48 << 20, SG_IMG_NODE = 4096;

int build_simt_tables(bem_plan *P, cudaStream_t s) {
    const MIndex &mi = P->mi;
    const int p = mi.p, np = mi.np, C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    const int W = P->prm.precision == BEM_MIXED ? 1 : 2, WC = W * C, RB = mg_rb(WC), VB = mg_vb(WC);
    Arena &A = P->arena;
    std::vector<int> colx(2 * (size_t)np);
    size_t off = 0;
    P->sg_kt = np;
    for (int a = 0; a < np; a++) {
        const int deg = mi.m[a] + mi.n[a] + mi.k[a], blocks = (n_upto(p - deg) + RB - 1) / RB;
        colx[2 * a] = blocks | n_upto(deg) << 16;
        colx[2 * a + 1] = (int)off;
        off += (size_t)blocks * VB;
        if (blocks <= mg_nb(W, C) && P->sg_kt == np) P->sg_kt = a;
    }
    P->sg_vec = off;
    P->sg_ldq = (np + MG_KA - 1) / MG_KA * MG_KA;
    BEM_TRY(A.alloc(&P->sg_colx, colx.size()));
    BEM_CUDA(cudaMemcpyAsync(P->sg_colx, colx.data(), sizeof(int) * colx.size(), cudaMemcpyHostToDevice, s));
    const int nc = P->sy_ncls;
    const size_t cap = (SG_IMG_BYTES + SG_IMG_NODE * (size_t)P->N) / (sizeof(float4) * off);
    P->sg_batch = (int)std::max<size_t>(1, std::min<size_t>(std::max(1, nc), cap));
    BEM_TRY(A.alloc((float4 **)&P->sg_img, (size_t)P->sg_batch * off));
    BEM_TRY(A.alloc(&P->sg_Mq, std::max<size_t>(1, (size_t)P->t.nbox * 6 * P->sg_ldq * WC)));
    if (W == 2) BEM_TRY(A.alloc(&P->sg_E, P->t.nbox));
    if (nc > 0 && P->sg_batch >= nc) BEM_TRY(launch_images(P, 0, nc, nullptr, s));
    return BEM_OK;
}

template <class R, int C>
int launch_m2l_sy(bem_plan *P, const R *M, R *L, cudaStream_t s) {
    constexpr int W = sizeof(R) == 8 ? 2 : 1, WC = W * C;
    const Tree &t = P->t;
    if (t.nbox == 0 || P->sy_bt.size() < 2) return BEM_OK;
    GemmArgs a{};
    a.np = P->mi.np;
    a.ldp = P->sy_ldp;
    a.ldq = P->sg_ldq;
    a.kt = P->sg_kt;
    a.img_vec = P->sg_vec;
    a.src = P->sy_src;
    a.sig = P->sy_sig;
    a.pair = P->sy_pair;
    a.colx = P->sg_colx;
    a.mexp = P->sy_mexp;
    a.img = (const float4 *)P->sg_img;
    a.Mq = P->sg_Mq;
    a.Lp = (float *)P->sy_Lp;
    a.skip = P->skip;
    const size_t sm = mg_smem(W, C, a.np);
    if (P->sy_ntile > 0)
        (k_m2l_words<R, C><<<t.nbox, 256, 0, s>>>(a.np, a.ldq, P->sy_fwd, P->sy_mexp, t.reach, M, P->sg_Mq,
                                                  P->sg_E, P->skip),
         ::bem::count_launch());
    // one run of targets at a time: its tiles, then the gather of its targets
    for (size_t r = 0; r + 1 < P->sy_bt.size(); r++) {
        const int bt0 = P->sy_bt[r], nt = P->sy_bt[r + 1] - bt0, tg0 = P->sy_bb[r], ntg = P->sy_bb[r + 1] - tg0;
        a.u0 = P->sy_bu[r];
        const bool kept = P->sg_batch >= P->sy_ncls;
        for (int i = 0; i < nt;) {                        // tiles are in class order
            int j = nt;
            a.cls0 = 0;
            if (!kept) {
                a.cls0 = P->sy_htile[bt0 + i];
                const int n = std::min(P->sg_batch, P->sy_ncls - a.cls0);
                for (j = i; j < nt && P->sy_htile[bt0 + j] < a.cls0 + n;) j++;
                BEM_TRY(launch_images(P, a.cls0, n, P->skip, s));
            }
            a.tile_cls = P->sy_tile_cls + bt0 + i;
            a.tile_start = P->sy_tile_start + bt0 + i;
            a.tile_cnt = P->sy_tile_cnt + bt0 + i;
            (k_m2l_gemm<W, C><<<(j - i) * (MG_TILE / MG_PT), MG_T, sm, s>>>(a), ::bem::count_launch());
            i = j;
        }
        if (ntg > 0)
            (k_m2l_gather_sy<R, C><<<dim3(ntg, (a.np + GA_R - 1) / GA_R), GA_R * GA_S, 0, s>>>(
                 tg0, t.level, t.side, P->lev_var ? P->d_lev_p : nullptr, t.inter_ptr, t.inter_idx, P->sg_E, a.u0, a.np,
                 a.ldp, P->sy_sig_u, P->sy_inv, (const float *)P->sy_Lp, L, P->skip),
             ::bem::count_launch());
    }
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

void set_sy_attributes() {
    const int n = n_upto(PMAX);
    cudaFuncSetAttribute(k_m2l_gemm<1, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mg_smem(1, 1, n));
    cudaFuncSetAttribute(k_m2l_gemm<1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mg_smem(1, 2, n));
    cudaFuncSetAttribute(k_m2l_gemm<2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mg_smem(2, 1, n));
    cudaFuncSetAttribute(k_m2l_gemm<2, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mg_smem(2, 2, n));
}

template int launch_m2l_sy<float, 1>(bem_plan *, const float *, float *, cudaStream_t);
template int launch_m2l_sy<float, 2>(bem_plan *, const float *, float *, cudaStream_t);
template int launch_m2l_sy<double, 1>(bem_plan *, const double *, double *, cudaStream_t);
template int launch_m2l_sy<double, 2>(bem_plan *, const double *, double *, cudaStream_t);

const void *kernel_of_m2l_simt() { return (const void *)k_m2l_gemm<1, 1>; }

}  // namespace bem

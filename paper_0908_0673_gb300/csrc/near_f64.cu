// Near field (regular rule over the near-list boxes) of float64 plans, in
// float32 pairs (dfloat.cuh).
//
// In float64 arithmetic a pair of the double layer is about 17 instructions on
// a pipe with 1/64 of the float32 rate, which bound the whole product.  In
// pairs it is about 107 float32 operations (73 single layer, 243 Helmholtz),
// all packed two targets per instruction, one hardware reciprocal square root
// as the seed of one third-order Newton step, and for Helmholtz a 2,048-entry
// table of the unit circle with a short Taylor step.  Measured (one product's
// near field + L2P): cube of 8,748 tri6, double layer, 263M pairs, 29.06 ->
// 0.96 ms; ellipsoid of 4,500, single layer, 114M pairs, 7.45 -> 0.37 ms;
// sphere of 2,880, Helmholtz, 70M pairs, 30.87 -> 0.74 ms; level-3 sphere of
// 1,280 tri3, 5M pairs, 1.57 -> 0.063 ms.  It is bound by the float32 pipe:
// 2.9e13 of the 3.9e13 operations per second the chip issues (Helmholtz 2.3e13,
// whose table reads share the issue slots).  Products differ from the float64
// kernel's by 5e-15 (Laplace) and 5e-14 (Helmholtz) of their norm; their error
// against the exact sums, the expansions' truncation (6e-8 at p = 10), is the
// same to every digit compared.
//
// Positions: everything is taken relative to the target leaf's centre and
// scaled by a power of two so that all points of the leaf's near field lie in
// [-1, 1].  A position is H + L1 + L2 with H on the grid 2^-22 and L1 on the
// grid 2^-44, so the differences of two H and of two L1 are exact float32
// subtractions and the pair's offset keeps its 48 bits however close the two
// points are: seven operations per component (two words, four operations, left
// an error of 2^-45 of the near field's extent, 1e-10 of a product).  Strengths
// are scaled by a power of two taken from the largest one the block reads; both
// scales return in float64 at the end.
//
// Layout as the float32 kernel (fmm.cu): a work item is one leaf and up to 32
// of its targets; G = ceil(targets / U) target groups x (256 / G) source
// slices, sources staged in shared memory in rounds of 512.  A cluster of 1 to
// 8 blocks shares an item (each takes a contiguous share of its sources) and
// block 0 adds the shares in rank order through distributed shared memory: small
// trees have fewer items than the chip has SMs.  Deterministic for a given plan.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "cluster.cuh"
#include "dfloat.cuh"
#include "fmm_views.cuh"

namespace bem {

namespace {

constexpr int ND_T = 256;               // threads
constexpr int ND_TILE = 512;            // sources per staged round
constexpr int ND_ENT = 256;             // near-list entries per chunk
constexpr int ND_TAB = 2048;            // unit-circle table entries
constexpr int ND_MAXC = 8;              // blocks per cluster at most
// phases above this many table steps lose the exact rounding to an index
// (1.5 2^23 + j must keep j): the plan then takes the float64 kernel
constexpr double ND_MAXPHASE = 2097152.0;

__host__ __device__ constexpr int nd_u(int C) { return C == 1 ? 4 : 2; }            // targets per thread
__host__ __device__ constexpr int nd_vec(int C, bool DL) { return C == 1 ? (DL ? 4 : 3) : (DL ? 5 : 4); }   // float4 per staged source
constexpr size_t nd_dyn_bytes(int C, bool DL) {
    return sizeof(float4) * ((size_t)ND_TILE * nd_vec(C, DL) + (C == 2 ? ND_TAB : 0));
}

template <int C, bool DL>
struct Src {                            // one source: minus its position's words, normal (x strength when real), strength
    float mh[3], m1[3], m2[3], nh[3], nl[3], fh[C], fl[C];
};

struct Wave {                           // wavenumber pair, and in table steps per length
    float kh, kl, th, tl;
};

__device__ __forceinline__ float rsqrt_seed(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// h + l + m + k (decreasing words) as H (grid 2^-22), L1 (grid 2^-44) and L2,
// for |h| <= 1
__device__ __forceinline__ void on_grid(float h, float l, float m, float k, float &H, float &L1, float &L2) {
    H = __fsub_rn(__fadd_rn(h, 3.f), 3.f);
    float a, b, e;
    two_sum(__fsub_rn(h, H), l, a, b);
    two_sum(a, m, a, e);
    L1 = __fsub_rn(__fadd_rn(a, 0x1.8p-21f), 0x1.8p-21f);
    L2 = __fadd_rn(__fsub_rn(a, L1), __fadd_rn(__fadd_rn(b, e), k));
}

// a float64 value as three float32 words
__device__ __forceinline__ void split3(double x, float &h, float &l, float &m) {
    h = (float)x;
    const double r = x - (double)h;
    l = (float)r;
    m = (float)(r - (double)l);
}

// acc += (xh + xl) (fh + fl), nxh = -xh
__device__ __forceinline__ void pmacc(P2 xh, P2 nxh, P2 xl, float fh, float fl, P2 &ah, P2 &al) {
    const P2 p = pmul(xh, p2(fh)), n = pmul(nxh, p2(fh));
    P2 lo = pfma(xh, p2(fh), n), s, t;
    lo = pfma(xh, p2(fl), lo);
    lo = pfma(xl, p2(fh), lo);
    two_sum(ah, p, s, t);
    ah = s;
    al = padd(al, padd(t, lo));
}

// one source against two targets: acc += kernel x strength
template <int C, bool DL>
__device__ __forceinline__ void pair_step(const P2 (&tH)[3], const P2 (&t1)[3], const P2 (&t2)[3], const Src<C, DL> &s, const Wave &kw,
                                          const float4 *tab, P2 (&ah)[C], P2 (&al)[C]) {
    const P2 one = p2(1.f), two = p2(2.f);
    P2 h[3], l[3], g[3], p[3], ne[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        // exact differences; H is 0 or at least as large as L1, so the fast sum is exact too
        const P2 d0 = padd(tH[c], p2(s.mh[c])), d1 = padd(t1[c], p2(s.m1[c]));
        h[c] = padd(d0, d1);
        l[c] = padd(psub(d1, psub(h[c], d0)), padd(t2[c], p2(s.m2[c])));
        g[c] = pneg(h[c]);
        p[c] = pmul(h[c], h[c]);
        ne[c] = pfma(g[c], h[c], p[c]);             // minus the product's rounding error
    }
    // r^2 = R + rho
    const P2 cr = pfma(l[0], h[0], pfma(l[1], h[1], pmul(l[2], h[2])));
    P2 s1, r1, R, r2;
    two_sum(p[0], p[1], s1, r1);
    two_sum(s1, p[2], R, r2);
    const P2 rho = psub(pfma(cr, two, padd(r1, r2)), padd(padd(ne[0], ne[1]), ne[2]));
    // 1 / r = y (1 - e)^(-1/2) with y the hardware seed and e = 1 - r^2 y^2 (about 2^-22)
    const P2 y = make_float2(rsqrt_seed(R.x), rsqrt_seed(R.y)), m = pneg(y);
    const P2 q = pmul(y, y), nq = pmul(m, y), nqe = pfma(m, y, q);
    P2 e = pfma(R, nq, one);
    e = pfma(rho, nq, e);
    e = pfma(R, nqe, e);
    P2 Wh, Wl;                                      // (r . n) / r^3 or 1 / r
    if (DL) {
        P2 pd[3], nd[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            pd[c] = pmul(h[c], p2(s.nh[c]));
            nd[c] = pfma(g[c], p2(s.nh[c]), pd[c]);
        }
        P2 dl = pmul(h[0], p2(s.nl[0]));
        dl = pfma(l[0], p2(s.nh[0]), dl);
        dl = pfma(h[1], p2(s.nl[1]), dl);
        dl = pfma(l[1], p2(s.nh[1]), dl);
        dl = pfma(h[2], p2(s.nl[2]), dl);
        dl = pfma(l[2], p2(s.nh[2]), dl);
        P2 s2, u1, D, u2;
        two_sum(pd[0], pd[1], s2, u1);
        two_sum(s2, pd[2], D, u2);
        const P2 Dl = psub(padd(padd(u1, u2), dl), padd(padd(nd[0], nd[1]), nd[2]));
        const P2 c3 = pmul(q, y), m3 = pmul(q, m);  // y^3
        P2 c3l = pfma(q, y, m3);
        c3l = pfma(nqe, m, c3l);
        const P2 g3 = pmul(e, pfma(e, p2(1.875f), p2(1.5f)));      // (1 - e)^(-3/2) - 1
        Wh = pmul(D, c3);
        Wl = pfma(D, c3, pmul(D, m3));
        Wl = pfma(D, c3l, Wl);
        Wl = pfma(Dl, c3, Wl);
        Wl = pfma(Wh, g3, Wl);
    }
    const P2 corr = pmul(e, pfma(e, p2(0.375f), p2(0.5f)));        // (1 - e)^(-1/2) - 1
    if (C == 1) {
        if (DL) {                                   // the strength is in the normal
            P2 a, t;
            two_sum(ah[0], Wh, a, t);
            ah[0] = a;
            al[0] = padd(al[0], padd(t, Wl));
        } else {
            pmacc(y, m, pmul(y, corr), s.fh[0], s.fl[0], ah[0], al[0]);
        }
        return;
    }
    if (!DL) {
        Wh = y;
        Wl = pmul(y, corr);
    }
    const P2 rh = pmul(R, y);
    P2 rl = pfma(R, y, pmul(R, m));
    rl = pfma(rho, y, rl);
    rl = pfma(rh, corr, rl);
    // k r in table steps = j + d, |d| <= 1/2
    const P2 th = pmul(p2(kw.th), rh);
    P2 tl = pfma(p2(kw.th), rh, pmul(p2(-kw.th), rh));
    tl = pfma(p2(kw.th), rl, tl);
    tl = pfma(p2(kw.tl), rh, tl);
    const P2 jf = padd(th, p2(12582912.f));
    P2 d = psub(th, padd(jf, p2(-12582912.f))), dlo;
    two_sum(d, tl, d, dlo);
    const float4 e0 = tab[__float_as_int(jf.x) & (ND_TAB - 1)], e1 = tab[__float_as_int(jf.y) & (ND_TAB - 1)];
    const P2 Ch = make_float2(e0.x, e1.x), Cl = make_float2(e0.y, e1.y), Sh = make_float2(e0.z, e1.z),
             Sl = make_float2(e0.w, e1.w);
    // the remaining angle in radians, g = gh + gl; cos g - 1 = cm, sin g = gh + sl
    const float sh = 0x1.921fb6p-9f, sl_ = -0x1.777a5cp-34f;       // 2 pi / 2048 as a pair
    const P2 gh = pmul(d, p2(sh)), ngh = pmul(d, p2(-sh));
    P2 gl = pfma(d, p2(sh), ngh);
    gl = pfma(d, p2(sl_), gl);
    gl = pfma(dlo, p2(sh), gl);
    const P2 a2 = pmul(gh, gh);
    P2 cm = pmul(a2, pfma(a2, p2(1.f / 24.f), p2(-0.5f)));
    cm = pfma(ngh, gl, cm);
    const P2 sl = pfma(pmul(gh, a2), p2(-1.f / 6.f), gl), nsl = pneg(sl);
    P2 ch, cl, sn, snl, t;
    {
        const P2 p1 = pmul(Sh, gh), n1 = pmul(Sh, ngh);
        two_sum(Ch, n1, ch, t);
        cl = padd(padd(t, Cl), pfma(Sh, ngh, p1));
        cl = pfma(Ch, cm, cl);
        cl = pfma(Sh, nsl, cl);
        cl = pfma(Sl, ngh, cl);
        const P2 p3 = pmul(Ch, gh), n3 = pmul(Ch, ngh);
        two_sum(Sh, p3, sn, t);
        snl = padd(padd(t, Sl), pfma(Ch, gh, n3));
        snl = pfma(Sh, cm, snl);
        snl = pfma(Ch, sl, snl);
        snl = pfma(Cl, gh, snl);
    }
    P2 grh = ch, grl = cl, gih = sn, gil = snl;     // e^{jkr}, times (1 - j k r) for the double layer
    if (DL) {
        const P2 Kh = pmul(p2(kw.kh), rh), nKh = pmul(p2(-kw.kh), rh);
        P2 Kl = pfma(p2(kw.kh), rh, nKh);
        Kl = pfma(p2(kw.kh), rl, Kl);
        Kl = pfma(p2(kw.kl), rh, Kl);
        const P2 pa = pmul(Kh, sn);
        P2 ea = pfma(Kh, sn, pmul(nKh, sn));
        ea = pfma(Kh, snl, ea);
        ea = pfma(Kl, sn, ea);
        two_sum(ch, pa, grh, t);
        grl = padd(padd(t, ea), cl);
        const P2 pb = pmul(Kh, ch), nb = pmul(nKh, ch);
        P2 eb = pfma(nKh, ch, pb);
        eb = pfma(nKh, cl, eb);
        eb = pfma(pneg(Kl), ch, eb);
        two_sum(sn, nb, gih, t);
        gil = padd(padd(t, eb), snl);
    }
    const P2 nW = pneg(Wh);
    const P2 A = pmul(Wh, grh), nA = pmul(nW, grh), B = pmul(Wh, gih), nB = pmul(nW, gih);
    P2 Al = pfma(Wh, grh, nA), Bl = pfma(Wh, gih, nB);
    Al = pfma(Wh, grl, Al);
    Al = pfma(Wl, grh, Al);
    Bl = pfma(Wh, gil, Bl);
    Bl = pfma(Wl, gih, Bl);
    pmacc(A, nA, Al, s.fh[0], s.fl[0], ah[0], al[0]);
    pmacc(B, nB, Bl, -s.fh[C - 1], -s.fl[C - 1], ah[0], al[0]);
    pmacc(A, nA, Al, s.fh[C - 1], s.fl[C - 1], ah[C - 1], al[C - 1]);
    pmacc(B, nB, Bl, s.fh[0], s.fl[0], ah[C - 1], al[C - 1]);
}

template <int C, bool DL>
__global__ void __launch_bounds__(ND_T, 2) k_near_pairs(int ns, const int2 *__restrict__ items, TreeView tv, QuadView qv,
                                                        double kwave, const double *__restrict__ f, double *__restrict__ ytmp,
                                                        const float4 *__restrict__ circle, const int *__restrict__ skip) {
    if (skip && *skip) return;                       // every block of the cluster reads the same word
    constexpr int U = nd_u(C);
    constexpr int SLOTS = ND_SLOTS;
    extern __shared__ float4 nd_smem[];
    float4 *stage = nd_smem, *tab = nd_smem + ND_TILE * nd_vec(C, DL);
    __shared__ int pref[ND_ENT + 1], ebase[ND_ENT];
    __shared__ float eoff[ND_ENT][9];                // entry box centre - target leaf centre, scaled, three words
    __shared__ float tpos[SLOTS][9];                 // target - target leaf centre: H, L1, L2
    __shared__ double share[SLOTS][C];
    __shared__ float wmax[ND_T / 32];
    __shared__ int wexp[ND_T / 32];
    const int rank = ns > 1 ? (int)cluster_rank() : 0;
    const int2 item = items[blockIdx.x / ns];
    const int b = tv.leaves[item.x], tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double cb[3] = {tv.cx[b], tv.cy[b], tv.cz[b]};
    const int t0 = item.y, nt = min(SLOTS, tv.ne[b] - t0);
    const int G = (nt + U - 1) / U, S = ND_T / G, tg = tid % G, sl = tid / G;
    const bool worker = sl < S;
    const int n0 = tv.near_ptr[b], n1 = tv.near_ptr[b + 1];
    // power-of-two scale: float pairs of the plan hold x 2^-es (es of the root
    // cube, so that any body's coordinates fit float32); M bounds every offset
    // from the leaf's centre, and 2^-em takes it into [-1, 1]
    const int es = ilogb(tv.side);
    float mx = (float)scalbn(tv.r[b], -es);
    for (int u = n0 + tid; u < n1; u += ND_T) {
        const int s = tv.near_idx[u];
        const double dx = fabs(tv.cx[s] - cb[0]), dy = fabs(tv.cy[s] - cb[1]), dz = fabs(tv.cz[s] - cb[2]);
        mx = fmaxf(mx, (float)scalbn(fmax(dx, fmax(dy, dz)) + tv.r[s], -es));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) wmax[warp] = mx;
    if (C == 2)
        for (int i = tid; i < ND_TAB; i += ND_T) tab[i] = circle[i];
    __syncthreads();
#pragma unroll
    for (int w = 0; w < ND_T / 32; w++) mx = fmaxf(mx, wmax[w]);
    const int em = ilogbf(fmaxf(mx, 1e-30f) * 1.0001f) + 1;         // 2^em > every offset
    const float sc = scalbnf(1.f, -em);
    const double kunit = kwave * scalbn(1.0, es + em);
    Wave kw{};
    if (C == 2) {
        df_split(kunit, kw.kh, kw.kl);
        df_split(kunit * (ND_TAB / (2.0 * M_PI)), kw.th, kw.tl);
    }
    if (tid < SLOTS) {
        const int k = t0 + (tid < nt ? tid : 0);     // off targets repeat the first
        const double x[3] = {tv.tx[k] - cb[0], tv.ty[k] - cb[1], tv.tz[k] - cb[2]};
#pragma unroll
        for (int c = 0; c < 3; c++) {
            float h, l, m;
            split3(scalbn(x[c], -es - em), h, l, m);
            on_grid(h, l, m, 0.f, tpos[tid][c], tpos[tid][3 + c], tpos[tid][6 + c]);
        }
    }
    __syncthreads();
    P2 tH[U / 2][3], t1[U / 2][3], t2[U / 2][3], ah[U / 2][C], al[U / 2][C];
#pragma unroll
    for (int v = 0; v < U / 2; v++) {
        const int i0 = tg + G * (2 * v), i1 = tg + G * (2 * v + 1);   // slots < G U <= SLOTS
#pragma unroll
        for (int c = 0; c < 3; c++) {
            tH[v][c] = make_float2(tpos[i0][c], tpos[i1][c]);
            t1[v][c] = make_float2(tpos[i0][3 + c], tpos[i1][3 + c]);
            t2[v][c] = make_float2(tpos[i0][6 + c], tpos[i1][6 + c]);
        }
#pragma unroll
        for (int c = 0; c < C; c++) ah[v][c] = al[v][c] = p2(0.f);
    }
    int E = 1;                                       // biased exponent of the strengths' scale
    for (int c0 = n0; c0 < n1; c0 += ND_ENT) {
        const int ne = min(ND_ENT, n1 - c0);
        __syncthreads();
        if (tid < 32) {                              // quadrature-point offsets of the entries (warp scan)
            int carry = 0;
            for (int i0 = 0; i0 < ne; i0 += 32) {
                const int i = i0 + lane;
                int x = 0;
                if (i < ne) {
                    const int s = tv.near_idx[c0 + i];
                    x = (tv.ee[s] - tv.eb[s]) * NQ;
                    ebase[i] = tv.eb[s] * NQ;
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (i < ne) pref[i + 1] = carry + x;
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) pref[0] = 0;
        } else {
            for (int i = tid - 32; i < ne; i += ND_T - 32) {
                const int s = tv.near_idx[c0 + i];
                const double d[3] = {tv.cx[s] - cb[0], tv.cy[s] - cb[1], tv.cz[s] - cb[2]};
#pragma unroll
                for (int c = 0; c < 3; c++) split3(scalbn(d[c], -es - em), eoff[i][c], eoff[i][3 + c], eoff[i][6 + c]);
            }
        }
        __syncthreads();
        // this block's share of the chunk's sources, and the largest strength in it
        const int total = pref[ne], j0 = (int)((long long)total * rank / ns), j1 = (int)((long long)total * (rank + 1) / ns);
        int ex = 0;
        for (int i = warp; i < ne; i += ND_T / 32) {
            const int a = max(pref[i], j0), z = min(pref[i + 1], j1);
            const double *fp = f + (size_t)ebase[i] * C;
            for (int j = (a - pref[i]) * C + lane; j < (z - pref[i]) * C; j += 32)
                ex = max(ex, (int)((unsigned)__double2hiint(__ldg(fp + j)) >> 20) & 0x7ff);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
        if (lane == 0) wexp[warp] = ex;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < ND_T / 32; w++) ex = max(ex, wexp[w]);
        ex = min(ex, 2046);                          // an infinity or NaN carries itself
        if (ex > E) {                                // earlier chunks go to the larger scale
            const int dn = max(-252, E - ex);
            const P2 sa = p2(scalbnf(1.f, dn / 2)), sb = p2(scalbnf(1.f, dn - dn / 2));
#pragma unroll
            for (int v = 0; v < U / 2; v++)
#pragma unroll
                for (int c = 0; c < C; c++) {
                    ah[v][c] = pmul(pmul(ah[v][c], sa), sb);
                    al[v][c] = pmul(pmul(al[v][c], sa), sb);
                }
            E = ex;
        }
        for (int base = j0; base < j1; base += ND_TILE) {
            __syncthreads();
            int lo = 0;                              // entry holding j: pref[lo] <= j < pref[lo + 1]
            if (base + tid < j1) {
                int hi = ne - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pref[mid] <= base + tid) lo = mid; else hi = mid - 1;
                }
            }
            for (int jj = tid; jj < ND_TILE; jj += ND_T) {
                const int j = base + jj;
                if (j >= j1) break;
                while (pref[lo + 1] <= j) lo++;      // j grows with jj: the entry only moves forward
                const int o = ebase[lo] + (j - pref[lo]);
                const float xh[3] = {qv.fx[o], qv.fy[o], qv.fz[o]}, xl[3] = {qv.lx[o], qv.ly[o], qv.lz[o]};
                float H[3], L1[3], L2[3];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    float s, e, l, m;
                    two_sum(eoff[lo][c], xh[c] * sc, s, e);
                    two_sum(eoff[lo][3 + c], xl[c] * sc, l, m);
                    on_grid(s, e, l, m + eoff[lo][6 + c], H[c], L1[c], L2[c]);
                }
                float fh[C], fl[C];
#pragma unroll
                for (int c = 0; c < C; c++) df_bits(f[(size_t)o * C + c], E, fh[c], fl[c]);
                float4 *d = stage + jj;
                d[0] = make_float4(-H[0], -H[1], -H[2], -L1[0]);
                d[ND_TILE] = make_float4(-L1[1], -L1[2], -L2[0], -L2[1]);
                if constexpr (C == 1 && DL) {        // strength x normal
                    const float nh[3] = {qv.fnx[o], qv.fny[o], qv.fnz[o]}, nl[3] = {qv.lnx[o], qv.lny[o], qv.lnz[o]};
                    float ph[3], pl[3];
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        ph[c] = __fmul_rn(fh[0], nh[c]);
                        pl[c] = fmaf(fl[0], nh[c], fmaf(fh[0], nl[c], fmaf(fh[0], nh[c], -ph[c])));
                    }
                    d[2 * ND_TILE] = make_float4(-L2[2], ph[0], ph[1], ph[2]);
                    d[3 * ND_TILE] = make_float4(pl[0], pl[1], pl[2], 0.f);
                } else {
                    d[2 * ND_TILE] = make_float4(-L2[2], fh[0], fl[0], fh[C - 1]);
                    if constexpr (C == 2)
                        d[3 * ND_TILE] = make_float4(fl[1], DL ? qv.fnx[o] : 0.f, DL ? qv.fny[o] : 0.f, DL ? qv.fnz[o] : 0.f);
                    if constexpr (C == 2 && DL) d[4 * ND_TILE] = make_float4(qv.lnx[o], qv.lny[o], qv.lnz[o], 0.f);
                }
            }
            __syncthreads();
            const int nq = min(ND_TILE, j1 - base);
            if (worker)
                for (int q = sl; q < nq; q += S) {
                    const float4 a = stage[q], c = stage[ND_TILE + q], e = stage[2 * ND_TILE + q];
                    Src<C, DL> s{};
                    s.mh[0] = a.x; s.mh[1] = a.y; s.mh[2] = a.z;
                    s.m1[0] = a.w; s.m1[1] = c.x; s.m1[2] = c.y;
                    s.m2[0] = c.z; s.m2[1] = c.w; s.m2[2] = e.x;
                    if constexpr (C == 1 && DL) {
                        const float4 g = stage[3 * ND_TILE + q];
                        s.nh[0] = e.y; s.nh[1] = e.z; s.nh[2] = e.w;
                        s.nl[0] = g.x; s.nl[1] = g.y; s.nl[2] = g.z;
                    } else {
                        s.fh[0] = e.y;
                        s.fl[0] = e.z;
                        if constexpr (C == 2) {
                            const float4 g = stage[3 * ND_TILE + q];
                            s.fh[1] = e.w;
                            s.fl[1] = g.x;
                            s.nh[0] = g.y; s.nh[1] = g.z; s.nh[2] = g.w;
                        }
                        if constexpr (C == 2 && DL) {
                            const float4 n = stage[4 * ND_TILE + q];
                            s.nl[0] = n.x; s.nl[1] = n.y; s.nl[2] = n.z;
                        }
                    }
#pragma unroll
                    for (int v = 0; v < U / 2; v++) pair_step<C, DL>(tH[v], t1[v], t2[v], s, kw, tab, ah[v], al[v]);
                }
        }
    }
    __syncthreads();                                 // sources done: the staged region is reused below
    // slices: eight threads per target add every eighth slice, then each other's sums
    float2 *red = (float2 *)stage;                   // [C][slot][S]
    if (worker)
#pragma unroll
        for (int v = 0; v < U / 2; v++)
#pragma unroll
            for (int c = 0; c < C; c++) {
                red[(c * G * U + tg + G * (2 * v)) * S + sl] = make_float2(ah[v][c].x, al[v][c].x);
                red[(c * G * U + tg + G * (2 * v + 1)) * S + sl] = make_float2(ah[v][c].y, al[v][c].y);
            }
    __syncthreads();
    {
        static_assert(ND_T == 8 * SLOTS, "eight threads per target");
        const int slot = tid >> 3;
        // kernel units: 1 / length^2 (double layer) or 1 / length, strengths 2^(E - 1023)
        const double unit = scalbn(0.25 / M_PI, E - 1023 - (DL ? 2 : 1) * (es + em));
#pragma unroll
        for (int c = 0; c < C; c++) {
            float sh = 0.f, sll = 0.f;
            if (slot < nt)
                for (int q = tid & 7; q < S; q += 8) {
                    const float2 x = red[(c * G * U + slot) * S + q];
                    df_add(sh, sll, x.x, x.y);
                }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, sh, o), ol = __shfl_xor_sync(0xffffffffu, sll, o);
                df_add(sh, sll, oh, ol);
            }
            if ((tid & 7) == 0) share[slot][c] = ((double)sh + (double)sll) * unit;
        }
    }
    if (ns > 1) cluster_sync(); else __syncthreads();
    if (rank == 0 && tid < nt) {
        const int node = tv.node_perm[t0 + tid];
#pragma unroll
        for (int c = 0; c < C; c++) {
            double y = share[tid][c];
            for (int q = 1; q < ns; q++) y += peer_double(&share[tid][c], q);
            ytmp[(size_t)node * C + c] = y;
        }
    }
    if (ns > 1) cluster_sync();                      // no block leaves while block 0 reads its share
}

// The unit circle at 2 pi j / 2048, cosine and sine as float pairs.
__device__ float4 g_circle[ND_TAB];

// address of the table on the current device, filled once per device (under a
// lock: plans are built from several host threads)
int circle_table(int device, const float4 **out) {
    static std::mutex mu;
    static const float4 *addr[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (device < 0 || device >= 64) { set_error("device %d out of range", device); return BEM_EINVAL; }
    if (!addr[device]) {
        std::vector<float4> t(ND_TAB);
        for (int j = 0; j < ND_TAB; j++) {
            const double a = 2.0 * M_PI * j / ND_TAB, c = std::cos(a), s = std::sin(a);
            const float ch = (float)c, sh = (float)s;
            t[j] = make_float4(ch, (float)(c - ch), sh, (float)(s - sh));
        }
        void *p = nullptr;
        BEM_CUDA(cudaGetSymbolAddress(&p, g_circle));
        BEM_CUDA(cudaMemcpy(p, t.data(), sizeof(float4) * ND_TAB, cudaMemcpyHostToDevice));
        BEM_COPIES_DONE();
        addr[device] = (const float4 *)p;
    }
    *out = addr[device];
    return BEM_OK;
}

template <int C, bool DL>
int launch(bem_plan *P, double kwave, const double *f, double *ytmp, cudaStream_t s) {
    const int ni = P->near_nitems[C - 1];
    if (ni == 0) return BEM_OK;
    // blocks per item: the smallest power of two that fills two blocks per SM
    // four times over (a last wave of small shares), at most a portable cluster
    int ns = 1;
    while (ns < ND_MAXC && ni * ns < 8 * P->sm_count) ns *= 2;
    TreeView tv = view_of(P);
    if (P->leaf_near_ptr) {                          // every entry a leaf, the sources' own box
        tv.near_ptr = P->leaf_near_ptr;
        tv.near_idx = P->leaf_near_idx;
    }
    BEM_TRY(launch_cluster(k_near_pairs<C, DL>, (unsigned)(ni * ns), ND_T, nd_dyn_bytes(C, DL), ns, s, ns,
                           (const int2 *)P->near_items[C - 1], tv, quad_of(P), kwave, f, ytmp, P->circle,
                           (const int *)P->skip));
    return BEM_OK;
}

}  // namespace

// Whether the pairs kernel takes a product: Helmholtz phases must stay within
// the table index (the points of one near field are at most 2 sqrt(3) (side +
// root radius) apart, and the root radius is at most the side for meshes whose
// curved sides stay near their nodes; 8 sides cover both with a margin).
bool near_pairs_apply(const bem_plan *P, int C, double kwave) {
    return C == 1 || kwave * P->t.side * 8.0 * (ND_TAB / (2.0 * M_PI)) < ND_MAXPHASE;
}

int near_pairs_prepare(bem_plan *P) {
    if (P->green == BEM_HELMHOLTZ) BEM_TRY(circle_table(P->device, &P->circle));
    const int b = 100 * 1024;
    BEM_CUDA(cudaFuncSetAttribute(k_near_pairs<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BEM_CUDA(cudaFuncSetAttribute(k_near_pairs<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BEM_CUDA(cudaFuncSetAttribute(k_near_pairs<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    BEM_CUDA(cudaFuncSetAttribute(k_near_pairs<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
    return BEM_OK;
}

template <int C>
int launch_near_pairs(bem_plan *P, int op, double kwave, const double *f, double *ytmp, cudaStream_t s) {
    return op == BEM_OP_A ? launch<C, true>(P, kwave, f, ytmp, s) : launch<C, false>(P, kwave, f, ytmp, s);
}
template int launch_near_pairs<1>(bem_plan *, int, double, const double *, double *, cudaStream_t);
template int launch_near_pairs<2>(bem_plan *, int, double, const double *, double *, cudaStream_t);

const void *kernel_of_near_f64() { return (const void *)k_near_pairs<1, true>; }

}  // namespace bem

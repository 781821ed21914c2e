// Accelerated field evaluation (Section 2.2, "Accelerated field evaluation"):
// the field of known surface data at points off the surface,
//     u(x) = sum over the surface of  phi dG/dn1 - G chi      (C(x) = 1 outside),
// by descending the box tree from the root for every field point: a box whose
// centre is farther than eta r_C from the point contributes its multipole
// expansion; otherwise a parent is opened and a leaf is integrated directly
// over its elements (7-point rule, or the parametric subdivision of the
// near-singular rule when the point is within tau h_e of an element).
// Everything after the moments is float64.
//
// One warp per point.  The descent tests up to 32 boxes at a time, one per
// lane; far boxes, near leaves and near-singular elements go to small queues in
// shared memory that are worked off 32 items at a time, so lanes do the same
// thing side by side and nothing recurses.
//
// Far boxes.  The expansion is a(d) G(x - c) with the polynomial a(xi) =
// sum_g (-1)^|g| I_g xi^g / g!.  Splitting a into |xi|^(2j) Y_nm(xi) with solid
// harmonics Y (orthogonal under the product <P, Q> = P(d) Q) and using
// |d|^2 G = -k^2 G and Hobson's theorem Y_n(d) f(r) = Y_n(x) (1/r d/dr)^n f
// leaves  sum_n G^(n)(r) sum_m b_nm Y_nm(x),  G^(n) = (1/r d/dr)^n G:
// (p + 1)^2 = 121 coefficients at p = 10 instead of 286 derivatives from an
// O(p^4) recursion, and a lane evaluates a whole box with three-term recurrences
// in registers.  The coefficients b are formed once per call and box; the sum is
// the same polynomial, so the truncation is unchanged.
//
// Near elements.  The 7-point rule reads the plan's quadrature points and
// strengths formed once per call; the subdivision takes the element's map and
// data as six monomial coefficients each (formed once per call), its pieces as
// integer codes.
//
// Before, a warp ran the O(p^4) recursion for every (point, box) with serial
// divisions on one lane, and every lane integrated whole elements with its own
// stack of triangles in local memory: 65.9 ms for 10,000 points around a sphere
// of 5,120 tri6 (p = 10).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "fmm_views.cuh"

namespace bem {

namespace {

constexpr int FW = 4;                   // warps (field points) per block
constexpr int FSTACK = 768;             // descent stack entries per warp
constexpr int FQ = 64;                  // queue capacity (worked off from 32)
constexpr int FPIECE = 256;             // subdivision pieces per warp
constexpr int FUNIT = 10;               // piece corners in units of 2^-10 (max_subdiv is at most 10)

// Harmonic parts of the monomials of every degree d <= PMAX: row (j, n = d - 2j,
// m, cos | sin), column g of degree d (the order of MIndex), value
// y_g / <|xi|^2j Y, |xi|^2j Y> with y the coefficients of |xi|^2j Y_nm.
// Degree d starts at harm_off(d), [column][row], n_d = (d+1)(d+2)/2 of each.
constexpr int harm_n(int d) { return (d + 1) * (d + 2) / 2; }
constexpr int harm_size(int d) {
    int s = 0;
    for (int e = 0; e < d; e++) s += harm_n(e) * harm_n(e);
    return s;
}
__device__ double g_harm[harm_size(PMAX + 1)];
__constant__ int c_harm_off[PMAX + 1];
__constant__ double c_rec[(PMAX + 1) * (PMAX + 1)];    // [n][m] (n^2 - m^2) / (4 n^2 - 1)

struct FieldArgs {
    double k, eta, iside, tau2;
    int maxdepth, p, npe;
    const double *cx, *cy, *cz, *r;
    const int *level, *child0, *nchild, *eb, *ee;
    const double *qx, *qy, *qz, *qnx, *qny, *qnz;
    const double *sphi, *schi;          // [Q][C] strengths w J phi, w J chi
    const double *harm;                 // [box][coefficients][2 C]
    const double *elem;                 // [E][18 + 12 C] monomial coefficients of map, phi, chi
    const double *cen;                  // [E][4] centroid image, (tau h)^2
    const float4 *fcen;                 // [E] the same in float32, tau h rounded up
    int *err;
};

__host__ __device__ constexpr int coef_count(int p) { return (p + 1) * (p + 2) / 2; }

// ---------------------------------------------------------------------------
// per call: harmonic coefficients of every box, monomial form of every element
// ---------------------------------------------------------------------------

// b_nm of one box from its scaled moments Ms = I / h^|g|, in units of the box
// edge, stored m by m, n ascending: (cos, sin) x C
template <class R, int C>
__global__ void __launch_bounds__(128) k_field_harm(int p_max, int np, const int *__restrict__ lev_p,
                                                    const int *__restrict__ level, double side, double k,
                                                    const R *__restrict__ M, double *__restrict__ H) {
    extern __shared__ double sm[];                       // [np][C]
    const int b = blockIdx.x, p = lev_p ? lev_p[level[b]] : p_max;
    for (int i = threadIdx.x; i < np_of(p) * C; i += blockDim.x) sm[i] = (double)M[(size_t)b * np * C + i];
    __syncthreads();
    const double kh = C == 2 ? k * scalbn(side, -level[b]) : 0.0, k2 = -kh * kh;
    const int nc = coef_count(p_max);
    for (int i = threadIdx.x; i < nc * 2; i += blockDim.x) {
        const int trig = i & 1;
        int m = 0, first = 0;                            // coefficients of m start at first
        while (i / 2 - first >= p_max + 1 - m) first += p_max + 1 - m++;
        const int n = m + i / 2 - first;
        double v[C];
#pragma unroll
        for (int c = 0; c < C; c++) v[c] = 0.0;
        if (!(m == 0 && trig)) {
            double f = (n & 1) ? -1.0 : 1.0;             // (-1)^d (-k^2)^j, d = n + 2 j
            for (int j = 0, d = n; d <= p && (C == 2 || j == 0); j++, d += 2) {
                const int nd = harm_n(d);
                // rows of degree d: those of n' = d, d - 2, ..., each 2 n' + 1 (m = 0, then cos, sin)
                int row = m == 0 ? 0 : 2 * m - 1 + trig;
                for (int e = d; e > n; e -= 2) row += 2 * e + 1;
                const double *W = g_harm + c_harm_off[d] + row, *x = sm + (d > 0 ? np_of(d - 1) : 0) * C;
                double s[C];
#pragma unroll
                for (int c = 0; c < C; c++) s[c] = 0.0;
                for (int g = 0; g < nd; g++) {
                    const double w = W[(size_t)g * nd];
#pragma unroll
                    for (int c = 0; c < C; c++) s[c] = fma(w, x[g * C + c], s[c]);
                }
#pragma unroll
                for (int c = 0; c < C; c++) v[c] += f * s[c];
                f *= k2;
            }
        }
#pragma unroll
        for (int c = 0; c < C; c++) H[((size_t)b * nc * 2 + i) * C + c] = v[c];
    }
}

// monomial coefficients over 1, s, t, s^2, s t, t^2 of a quantity with nodal values f
__device__ __forceinline__ void monomials(int npe, const double *f, double *a) {
    if (npe == 3) {
        a[0] = f[0]; a[1] = f[1] - f[0]; a[2] = f[2] - f[0];
        a[3] = a[4] = a[5] = 0.0;
        return;
    }
    a[0] = f[0];
    a[1] = 4.0 * f[3] - 3.0 * f[0] - f[1];
    a[2] = 4.0 * f[5] - 3.0 * f[0] - f[2];
    a[3] = 2.0 * (f[0] + f[1]) - 4.0 * f[3];
    a[4] = 4.0 * (f[0] - f[3] + f[4] - f[5]);
    a[5] = 2.0 * (f[0] + f[2]) - 4.0 * f[5];
}

template <int C>
__global__ void __launch_bounds__(128) k_field_elems(int E, int npe, double tau, const double *__restrict__ nodes,
                                                     const int *__restrict__ el_phi, const int *__restrict__ el_chi,
                                                     const double *__restrict__ phi, const double *__restrict__ chi,
                                                     double *__restrict__ elem, double *__restrict__ cen,
                                                     float4 *__restrict__ fcen) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= E) return;
    const int *ep = el_phi + (size_t)e * npe, *ec = el_chi + (size_t)e * npe;
    double *out = elem + (size_t)e * (18 + 12 * C);
    double f[6], a[6], c[3], h2 = 0.0, x[3][3], big = 0.0;
    for (int d = 0; d < 3; d++) {
        for (int q = 0; q < npe; q++) f[q] = nodes[3 * (size_t)ep[q] + d];
        for (int q = 0; q < 3; q++) x[q][d] = f[q];
        monomials(npe, f, a);
        for (int q = 0; q < 6; q++) out[q * 3 + d] = a[q];
        const double t = 1.0 / 3.0;
        c[d] = a[0] + t * (a[1] + a[2]) + t * t * (a[3] + a[4] + a[5]);
        big = fmax(big, fabs(c[d]));
    }
    for (int q = 0; q < 3; q++) {
        double s = 0.0;
        for (int d = 0; d < 3; d++) s += (x[q][d] - x[(q + 1) % 3][d]) * (x[q][d] - x[(q + 1) % 3][d]);
        h2 = fmax(h2, s);
    }
    for (int w = 0; w < C; w++) {
        for (int q = 0; q < npe; q++) f[q] = phi[(size_t)ep[q] * C + w];
        monomials(npe, f, a);
        for (int q = 0; q < 6; q++) out[18 + q * C + w] = a[q];
        for (int q = 0; q < npe; q++) f[q] = chi[(size_t)ec[q] * C + w];
        monomials(npe, f, a);
        for (int q = 0; q < 6; q++) out[18 + 6 * C + q * C + w] = a[q];
    }
    for (int d = 0; d < 3; d++) cen[4 * (size_t)e + d] = c[d];
    cen[4 * (size_t)e + 3] = tau * tau * h2;
    // float32 filter: a point farther than this in float32 is not near-singular
    // (rounding of the centre and of the three differences: 2^-21 of the coordinates)
    fcen[e] = make_float4((float)c[0], (float)c[1], (float)c[2], (float)((tau * sqrt(h2) + 5e-7 * big) * (1.0 + 1e-6)));
}

// ---------------------------------------------------------------------------
// the evaluation
// ---------------------------------------------------------------------------
template <int C>
struct WarpShared {
    int stack[FSTACK];
    int far[FQ], leaf[FQ], sing[FQ];
    int pref[33], base[32];
    int2 piece[FPIECE], leaves[FQ];
};

// kernel of one quadrature point: w (phi dG/dn - chi G) with the weighted
// strengths (sp, sc), rn = (x - y) . n and r^2
template <int C>
__device__ __forceinline__ void add_point(double k, double r2, double rn, const double *sp, const double *sc, double *acc) {
    const double ir = rsqrt(r2);
    if constexpr (C == 1) {
        acc[0] += ir * (sp[0] * rn * ir * ir - sc[0]);
    } else {
        const double kr = k * (r2 * ir);
        double sn, cs;
        sincos(kr, &sn, &cs);
        const double d = rn * ir * ir;                   // e^{jkr} [(1 - jkr) d phi - chi] / r
        const double dr = d, di = -kr * d;
        const double vr = sp[0] * dr - sp[1] * di - sc[0], vi = sp[0] * di + sp[1] * dr - sc[1];
        acc[0] += ir * (cs * vr - sn * vi);
        acc[1] += ir * (cs * vi + sn * vr);
    }
}

// multipole expansion of box b (one per lane) at the point; gs: this lane's
// column of [p + 1][C][32]
template <int C>
__device__ __forceinline__ void far_box(const FieldArgs &a, int b, const double *x, double *gs, double *acc) {
    const int p = a.p;
    const double ih = scalbn(a.iside, a.level[b]);       // 1 / edge
    const double rx = (x[0] - a.cx[b]) * ih, ry = (x[1] - a.cy[b]) * ih, rz = (x[2] - a.cz[b]) * ih;
    const double r2 = rx * rx + ry * ry + rz * rz, ir = rsqrt(r2), ir2 = ir * ir;
    // G^(n): G^(n+1) = -((2n + 1) G^(n) + k^2 G^(n-1)) / r^2
    if constexpr (C == 1) {
        double g = ir;
        for (int n = 0; n <= p; n++) {
            gs[32 * n] = g;
            g *= -(2.0 * n + 1.0) * ir2;
        }
    } else {
        const double kh = a.k / ih, k2 = kh * kh;
        double sn, cs;
        sincos(kh * (r2 * ir), &sn, &cs);
        double pr = sn / kh, pi = -cs / kh, cr = cs * ir, ci = sn * ir;
        for (int n = 0; n <= p; n++) {
            gs[64 * n] = cr;
            gs[64 * n + 32] = ci;
            const double f = -(2.0 * n + 1.0), nr = (f * cr - k2 * pr) * ir2, ni = (f * ci - k2 * pi) * ir2;
            pr = cr; pi = ci; cr = nr; ci = ni;
        }
    }
    const double *h = a.harm + (size_t)b * coef_count(p) * 2 * C;
    double cm = 1.0, sm = 0.0, sum[C];                   // Re, Im (rx + j ry)^m
#pragma unroll
    for (int c = 0; c < C; c++) sum[c] = 0.0;
    for (int m = 0; m <= p; m++) {
        double B = 1.0, Bp = 0.0, ac[C], as[C];
#pragma unroll
        for (int c = 0; c < C; c++) ac[c] = as[c] = 0.0;
        for (int n = m; n <= p; n++) {
            if constexpr (C == 1) {
                const double2 v = *reinterpret_cast<const double2 *>(h);
                const double gB = gs[32 * n] * B;
                ac[0] = fma(gB, v.x, ac[0]);
                as[0] = fma(gB, v.y, as[0]);
            } else {
                const double2 v = *reinterpret_cast<const double2 *>(h), w = *reinterpret_cast<const double2 *>(h + 2);
                const double gr = gs[64 * n] * B, gi = gs[64 * n + 32] * B;
                ac[0] += gr * v.x - gi * v.y;
                ac[C - 1] += gr * v.y + gi * v.x;
                as[0] += gr * w.x - gi * w.y;
                as[C - 1] += gr * w.y + gi * w.x;
            }
            h += 2 * C;
            const double Bn = rz * B - c_rec[n * (PMAX + 1) + m] * r2 * Bp;
            Bp = B;
            B = Bn;
        }
#pragma unroll
        for (int c = 0; c < C; c++) sum[c] += cm * ac[c] + sm * as[c];
        const double t = cm * rx - sm * ry;
        sm = cm * ry + sm * rx;
        cm = t;
    }
#pragma unroll
    for (int c = 0; c < C; c++) acc[c] += sum[c] * ih;
}

__device__ __forceinline__ void map_at(const double *A, double s, double t, double *y) {
    const double ss = s * s, st = s * t, tt = t * t;
#pragma unroll
    for (int c = 0; c < 3; c++)
        y[c] = A[c] + s * A[3 + c] + t * A[6 + c] + ss * A[9 + c] + st * A[12 + c] + tt * A[15 + c];
}

// edge vectors u_f, v_f = u_(f+1) of a piece's frame, in units of its edge: (1,0)
// (0,1) (-1,1) (-1,0) (0,-1) (1,-1); the middle piece of a 4-way split has the
// next frame (u' = v / 2, v' = (v - u) / 2), the corner pieces keep it
__device__ __forceinline__ void frame_uv(int f, int *u, int *v) {
    constexpr int s = 2 | 1 << 2 | 0 << 4 | 0 << 6 | 1 << 8 | 2 << 10 | 2 << 12;   // components + 1, two bits each
    constexpr int t = 1 | 2 << 2 | 2 << 4 | 1 << 6 | 0 << 8 | 0 << 10 | 1 << 12;
    u[0] = (s >> 2 * f & 3) - 1;
    u[1] = (t >> 2 * f & 3) - 1;
    v[0] = (s >> 2 * (f + 1) & 3) - 1;
    v[1] = (t >> 2 * (f + 1) & 3) - 1;
}

template <int C>
__global__ void __launch_bounds__(FW * 32) k_field(int64_t npts, const double *__restrict__ pts, double *__restrict__ u,
                                                   const FieldArgs a) {
    extern __shared__ __align__(16) double fsm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t gsz = (size_t)(a.p + 1) * 32 * C;
    double *gs = fsm + (gsz + (sizeof(WarpShared<C>) + 7) / 8) * warp + lane;
    WarpShared<C> &S = *reinterpret_cast<WarpShared<C> *>(fsm + (gsz + (sizeof(WarpShared<C>) + 7) / 8) * warp + gsz);
    const int64_t ip = (int64_t)blockIdx.x * FW + warp;
    if (ip >= npts) return;                              // warp-uniform
    const double x[3] = {pts[3 * ip], pts[3 * ip + 1], pts[3 * ip + 2]};
    const float xf[3] = {(float)x[0], (float)x[1], (float)x[2]};
    const float xmargin = 5e-7f * fmaxf(fabsf(xf[0]), fmaxf(fabsf(xf[1]), fabsf(xf[2])));
    const unsigned below = (1u << lane) - 1u;
    double acc[C];
#pragma unroll
    for (int c = 0; c < C; c++) acc[c] = 0.0;
    int nst = 1, nfar = 0, nleaf = 0, nsing = 0;

    // pieces of the near-singular elements in the queue
    auto subdivide = [&]() {
        int np = nsing, nlv = 0;
        for (int i = lane; i < np; i += 32) S.piece[i] = make_int2(0, S.sing[i]);
        nsing = 0;
        __syncwarp();
        // piece: x = corner s | corner t << 11 | frame << 22 | depth << 25, y = element
        auto integrate = [&](int n) {
            for (int i = lane; i < 7 * n; i += 32) {
                const int2 pc = S.leaves[i / 7];
                const int f = pc.x >> 22 & 7, depth = pc.x >> 25 & 15;
                int fu[2], fv[2];
                frame_uv(f, fu, fv);
                const double un = 1.0 / (1 << FUNIT), w0 = scalbn(1.0, -depth);
                double s, t, w;
                radon7(i % 7, s, t, w);
                const double ps = un * (pc.x & 2047) + w0 * (s * fu[0] + t * fv[0]),
                             pt = un * (pc.x >> 11 & 2047) + w0 * (s * fu[1] + t * fv[1]);
                const double *A = a.elem + (size_t)pc.y * (18 + 12 * C);
                double y[3], ts[3], tt[3];
                map_at(A, ps, pt, y);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    ts[c] = A[3 + c] + 2.0 * ps * A[9 + c] + pt * A[12 + c];
                    tt[c] = A[6 + c] + ps * A[12 + c] + 2.0 * pt * A[15 + c];
                }
                const double nx = ts[1] * tt[2] - ts[2] * tt[1], ny = ts[2] * tt[0] - ts[0] * tt[2],
                             nz = ts[0] * tt[1] - ts[1] * tt[0];
                const double rx = x[0] - y[0], ry = x[1] - y[1], rz = x[2] - y[2];
                const double wq = w * w0 * w0, J = sqrt(nx * nx + ny * ny + nz * nz);
                const double ss = ps * ps, st = ps * pt, t2 = pt * pt;
                double sp[C], sc[C];
#pragma unroll
                for (int c = 0; c < C; c++) {
                    const double *F = A + 18 + c, *X = A + 18 + 6 * C + c;
                    sp[c] = wq * (F[0] + ps * F[C] + pt * F[2 * C] + ss * F[3 * C] + st * F[4 * C] + t2 * F[5 * C]);
                    sc[c] = wq * J * (X[0] + ps * X[C] + pt * X[2 * C] + ss * X[3 * C] + st * X[4 * C] + t2 * X[5 * C]);
                }
                add_point<C>(a.k, rx * rx + ry * ry + rz * rz, rx * nx + ry * ny + rz * nz, sp, sc, acc);
            }
            __syncwarp();
        };
        while (np > 0) {
            // a pass adds at most 3 n; one at a time (depth first, 30 more) when nearly full
            const int n = min(min(32, np), max(1, (FPIECE - 40 - np) / 3));
            const bool on = lane < n;
            const int2 pc = on ? S.piece[np - 1 - lane] : make_int2(0, 0);
            __syncwarp();
            np -= n;
            bool split = false;
            const int f = pc.x >> 22 & 7, depth = pc.x >> 25 & 15, as = pc.x & 2047, at = pc.x >> 11 & 2047;
            int fu[2], fv[2];
            frame_uv(f, fu, fv);
            const int len = 1 << (FUNIT - depth);
            if (on && depth < a.maxdepth) {
                const double *A = a.elem + (size_t)pc.y * (18 + 12 * C), un = 1.0 / (1 << FUNIT);
                double ya[3], yb[3], yc[3], ym[3];
                map_at(A, un * as, un * at, ya);
                map_at(A, un * (as + len * fu[0]), un * (at + len * fu[1]), yb);
                map_at(A, un * (as + len * fv[0]), un * (at + len * fv[1]), yc);
                map_at(A, un * (as + len * (fu[0] + fv[0]) / 3.0), un * (at + len * (fu[1] + fv[1]) / 3.0), ym);
                double dab = 0.0, dbc = 0.0, dca = 0.0, dx = 0.0;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    dab += (ya[c] - yb[c]) * (ya[c] - yb[c]);
                    dbc += (yb[c] - yc[c]) * (yb[c] - yc[c]);
                    dca += (yc[c] - ya[c]) * (yc[c] - ya[c]);
                    dx += (x[c] - ym[c]) * (x[c] - ym[c]);
                }
                split = dx < a.tau2 * fmax(dab, fmax(dbc, dca));
            }
            const unsigned ms = __ballot_sync(0xffffffffu, split), ml = __ballot_sync(0xffffffffu, on && !split);
            if (split) {
                int2 *q = S.piece + np + 4 * __popc(ms & below);
                const int hl = len >> 1, d = (depth + 1) << 25;
                auto put = [&](int i, int s, int t, int fr) { q[i] = make_int2(s | t << 11 | fr << 22 | d, pc.y); };
                put(0, as, at, f);
                put(1, as + hl * fu[0], at + hl * fu[1], f);
                put(2, as + hl * fv[0], at + hl * fv[1], f);
                put(3, as + hl * fu[0], at + hl * fu[1], f == 5 ? 0 : f + 1);    // (ab, bc, ca): u' = v / 2, v' = (v - u) / 2
            }
            np += 4 * __popc(ms);
            if (on && !split) S.leaves[nlv + __popc(ml & below)] = pc;
            nlv += __popc(ml);
            __syncwarp();
            if (nlv >= 32) {
                integrate(nlv);
                nlv = 0;
            }
        }
        if (nlv > 0) integrate(nlv);
    };

    // sources of the near leaves in the queue, one per lane
    auto direct = [&]() {
        {
            const int b = lane < nleaf ? S.leaf[lane] : -1;
            int n = b >= 0 ? (a.ee[b] - a.eb[b]) * NQ : 0;
            S.base[lane] = b >= 0 ? a.eb[b] * NQ : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, n, o);
                if (lane >= o) n += y;
            }
            S.pref[lane + 1] = n;
            if (lane == 0) S.pref[0] = 0;
        }
        nleaf = 0;
        __syncwarp();
        const int total = S.pref[32];
        for (int j0 = 0; j0 < total; j0 += 32) {
            const int j = j0 + lane;
            bool near = false;
            int e = 0, o = 0;
            if (j < total) {
                int lo = 0, hi = 31;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (S.pref[mid] <= j) lo = mid; else hi = mid - 1;
                }
                o = S.base[lo] + j - S.pref[lo];
                e = o / NQ;
                const float4 fc = a.fcen[e];
                const float fx = xf[0] - fc.x, fy = xf[1] - fc.y, fz = xf[2] - fc.z, lim = fc.w + xmargin;
                if (fx * fx + fy * fy + fz * fz <= lim * lim) {
                    const double *c = a.cen + 4 * (size_t)e;
                    const double dx = x[0] - c[0], dy = x[1] - c[1], dz = x[2] - c[2];
                    near = dx * dx + dy * dy + dz * dz < c[3];
                }
                if (!near) {
                    const double rx = x[0] - a.qx[o], ry = x[1] - a.qy[o], rz = x[2] - a.qz[o];
                    add_point<C>(a.k, rx * rx + ry * ry + rz * rz, rx * a.qnx[o] + ry * a.qny[o] + rz * a.qnz[o],
                                 a.sphi + (size_t)o * C, a.schi + (size_t)o * C, acc);
                }
            }
            const unsigned mn = __ballot_sync(0xffffffffu, near && o % NQ == 0);
            if (near && o % NQ == 0) S.sing[nsing + __popc(mn & below)] = e;
            nsing += __popc(mn);
            __syncwarp();
            if (nsing >= 32) subdivide();
        }
    };

    if (lane == 0) S.stack[0] = 0;                       // the root
    __syncwarp();
    while (nst > 0) {
        // a pass adds at most 7 n; one at a time (depth first, 140 more) when nearly full
        const int n = min(min(32, nst), max(1, (FSTACK - 160 - nst) / 7));
        const bool on = lane < n;
        const int b = on ? S.stack[nst - 1 - lane] : 0;
        __syncwarp();
        nst -= n;
        bool is_far = false;
        int nch = 0;
        if (on) {
            const double dx = x[0] - a.cx[b], dy = x[1] - a.cy[b], dz = x[2] - a.cz[b];
            is_far = sqrt(dx * dx + dy * dy + dz * dz) > a.eta * a.r[b];
            nch = is_far ? 0 : a.nchild[b];
        }
        const bool is_leaf = on && !is_far && nch == 0;
        const unsigned mf = __ballot_sync(0xffffffffu, is_far), ml = __ballot_sync(0xffffffffu, is_leaf);
        if (is_far) S.far[nfar + __popc(mf & below)] = b;
        if (is_leaf) S.leaf[nleaf + __popc(ml & below)] = b;
        nfar += __popc(mf);
        nleaf += __popc(ml);
        int off = nch;                                   // inclusive scan of the children
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, off, o);
            if (lane >= o) off += y;
        }
        const int push = __shfl_sync(0xffffffffu, off, 31);
        for (int q = 0; q < nch; q++) {
            const int at = nst + off - nch + q;
            if (at < FSTACK) S.stack[at] = a.child0[b] + q;
            else atomicOr(a.err, 2);                     // stack full: this branch is skipped
        }
        nst = min(FSTACK, nst + push);
        __syncwarp();
        if (nfar >= 32) {
            far_box<C>(a, S.far[nfar - 32 + lane], x, gs, acc);
            nfar -= 32;
        }
        if (nleaf >= 32) {
            // keep the first 32 for the pass, move the rest down
            const int more = nleaf - 32, keep = lane < more ? S.leaf[32 + lane] : 0;
            nleaf = 32;
            direct();
            if (lane < more) S.leaf[lane] = keep;
            nleaf = more;
            __syncwarp();
        }
    }
    if (lane < nfar) far_box<C>(a, S.far[lane], x, gs, acc);
    __syncwarp();
    if (nleaf > 0) direct();
    if (nsing > 0) subdivide();
#pragma unroll
    for (int c = 0; c < C; c++) {
        for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
        if (lane == 0) u[ip * C + c] = acc[c] * (0.25 / M_PI);
    }
}

// ---------------------------------------------------------------------------
// host: the harmonic table
// ---------------------------------------------------------------------------

// coefficients of a homogeneous polynomial of degree d, by (m, n) exponents of
// x and y in the order of MIndex within a degree
struct Poly {
    int d;
    std::vector<double> c;
    explicit Poly(int d_) : d(d_), c(harm_n(d_), 0.0) {}
    static int at(int d, int m, int n) { return (d - m) * (d - m + 1) / 2 + (d - m - n); }   // m descending, then n
    double &operator()(int m, int n) { return c[at(d, m, n)]; }
    double operator()(int m, int n) const { return c[at(d, m, n)]; }
};

Poly mul_axis(const Poly &a, int ax) {
    Poly r(a.d + 1);
    for (int m = 0; m <= a.d; m++)
        for (int n = 0; m + n <= a.d; n++) r(m + (ax == 0), n + (ax == 1)) += a(m, n);
    return r;
}
Poly mul_r2(const Poly &a) {
    Poly r(a.d + 2);
    for (int m = 0; m <= a.d; m++)
        for (int n = 0; m + n <= a.d; n++) {
            r(m + 2, n) += a(m, n);
            r(m, n + 2) += a(m, n);
            r(m, n) += a(m, n);
        }
    return r;
}
Poly axpy(const Poly &a, double s, const Poly &b) {
    Poly r = a;
    for (size_t i = 0; i < r.c.size(); i++) r.c[i] += s * b.c[i];
    return r;
}
double rec_coef(int n, int m) { return (double)(n * n - m * m) / (4.0 * n * n - 1.0); }

// degrees [d0, d1] of the table
std::vector<double> harmonic_table(int d0, int d1) {
    double fact[PMAX + 1];
    fact[0] = 1.0;
    for (int i = 1; i <= PMAX; i++) fact[i] = fact[i - 1] * i;
    // Y[n][row]: m = 0, then (cos, sin) of m = 1..n
    std::vector<std::vector<Poly>> Y(d1 + 1);
    Poly C(0), S(0);
    C(0, 0) = 1.0;
    for (int n = 0; n <= d1; n++) Y[n].assign(2 * n + 1, Poly(n));
    for (int m = 0; m <= d1; m++) {
        for (int trig = 0; trig < (m ? 2 : 1); trig++) {
            const int row = m ? 2 * m - 1 + trig : 0;
            Y[m][row] = trig ? S : C;
            for (int n = m; n < d1; n++) {
                Poly q = mul_axis(Y[n][row], 2);
                if (n > m) q = axpy(q, -rec_coef(n, m), mul_r2(Y[n - 1][row]));
                Y[n + 1][row] = q;
            }
        }
        // (C + j S) (x + j y)
        Poly c = axpy(mul_axis(C, 0), -1.0, mul_axis(S, 1)), s = axpy(mul_axis(C, 1), 1.0, mul_axis(S, 0));
        C = c;
        S = s;
    }
    std::vector<double> out;
    std::vector<Poly> rows;
    for (int d = d0; d <= d1; d++) {
        rows.clear();
        for (int n = d; n >= 0; n -= 2)
            for (const Poly &y : Y[n]) {
                Poly q = y;
                for (int j = n; j < d; j += 2) q = mul_r2(q);
                rows.push_back(q);
            }
        const int nd = harm_n(d);
        const size_t base = out.size();
        out.resize(base + (size_t)nd * nd);
        for (int r = 0; r < nd; r++) {
            double norm = 0.0;
            for (int m = 0; m <= d; m++)
                for (int n = 0; m + n <= d; n++) norm += fact[m] * fact[n] * fact[d - m - n] * rows[r](m, n) * rows[r](m, n);
            for (int g = 0; g < nd; g++) out[base + (size_t)g * nd + r] = rows[r].c[g] / norm;
        }
    }
    return out;
}

}  // namespace

template <int C>
static size_t field_smem(int p) {
    return FW * (((size_t)(p + 1) * 32 * C + (sizeof(WarpShared<C>) + 7) / 8) * sizeof(double));
}

// The table of degrees <= p on the plan's device (filled once per device and
// degree, under a lock) and the workspaces of a field evaluation.
int field_prepare(bem_plan *P) {
    static std::mutex mu;
    static int have[64];                                 // degrees on the device: [0, have)
    const int p = P->mi.p, C = P->green == BEM_HELMHOLTZ ? 2 : 1, dev = P->device;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (dev < 0 || dev >= 64) { set_error("device %d out of range", dev); return BEM_EINVAL; }
        if (have[dev] == 0) {
            int off[PMAX + 1];
            std::vector<double> rec((PMAX + 1) * (PMAX + 1), 0.0);
            for (int d = 0; d <= PMAX; d++) off[d] = harm_size(d);
            for (int n = 1; n <= PMAX; n++)
                for (int m = 0; m < n; m++) rec[n * (PMAX + 1) + m] = rec_coef(n, m);
            BEM_CUDA(cudaMemcpyToSymbol(c_harm_off, off, sizeof(off)));
            BEM_CUDA(cudaMemcpyToSymbol(c_rec, rec.data(), sizeof(double) * rec.size()));
        }
        if (have[dev] <= p) {
            const std::vector<double> t = harmonic_table(have[dev], p);
            BEM_CUDA(cudaMemcpyToSymbol(g_harm, t.data(), sizeof(double) * t.size(), sizeof(double) * harm_size(have[dev])));
            BEM_COPIES_DONE();
            have[dev] = p + 1;
        }
    }
    // one value for every order: plans of different orders evaluate fields on
    // different threads, and one must not lower another's limit before its launch
    BEM_CUDA(cudaFuncSetAttribute(k_field<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)field_smem<1>(PMAX)));
    BEM_CUDA(cudaFuncSetAttribute(k_field<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)field_smem<2>(PMAX)));
    Arena &A = P->arena;
    BEM_TRY(A.alloc(&P->fd_str, 2 * (size_t)P->Q * C));
    BEM_TRY(A.alloc(&P->fd_elem, (size_t)P->E * (18 + 12 * C)));
    BEM_TRY(A.alloc(&P->fd_cen, 4 * (size_t)P->E));
    BEM_TRY(A.alloc((float4 **)&P->fd_fcen, (size_t)P->E));
    BEM_TRY(A.alloc(&P->fd_harm, (size_t)P->t.nbox * coef_count(p) * 2 * C));
    return BEM_OK;
}

template <class R, int C>
static int launch_field(bem_plan *P, int64_t npts, const double *pts, double *u, const double *phi, const double *chi,
                        const R *M, cudaStream_t s) {
    const Tree &t = P->t;
    const int E = (int)P->E, p = P->mi.p;
    (k_field_harm<R, C><<<t.nbox, 128, sizeof(double) * P->mi.np * C, s>>>(
         p, P->mi.np, P->lev_var ? P->d_lev_p : nullptr, t.level, t.side, P->k, M, P->fd_harm),
     ::bem::count_launch());
    (k_field_elems<C><<<(E + 127) / 128, 128, 0, s>>>(E, P->npe, P->prm.tau_near, P->nodes, t.el_phi, t.el_chi, phi, chi,
                                                      P->fd_elem, P->fd_cen, (float4 *)P->fd_fcen),
     ::bem::count_launch());
    FieldArgs a{};
    a.k = P->k;
    a.eta = P->prm.eta;
    a.iside = 1.0 / t.side;
    a.tau2 = P->prm.tau_near * P->prm.tau_near;
    a.maxdepth = P->prm.max_subdiv;
    a.p = p;
    a.npe = P->npe;
    a.cx = t.cx; a.cy = t.cy; a.cz = t.cz; a.r = t.r;
    a.level = t.level; a.child0 = t.child0; a.nchild = t.nchild; a.eb = t.eb; a.ee = t.ee;
    a.qx = P->q.x; a.qy = P->q.y; a.qz = P->q.z;
    a.qnx = P->q.nx; a.qny = P->q.ny; a.qnz = P->q.nz;
    a.sphi = P->fd_str;
    a.schi = P->fd_str + (size_t)P->Q * C;
    a.harm = P->fd_harm;
    a.elem = P->fd_elem;
    a.cen = P->fd_cen;
    a.fcen = (const float4 *)P->fd_fcen;
    a.err = P->dev_err;
    const size_t sm = field_smem<C>(p);
    const int64_t nblk = (npts + FW - 1) / FW;
    if (nblk > 0) (k_field<C><<<(unsigned)nblk, FW * 32, sm, s>>>(npts, pts, u, a), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

const void *kernel_of_field() { return (const void *)k_field_harm<float, 1>; }

}  // namespace bem

using namespace bem;

extern "C" int bem_field(bem_plan *P, const void *phi_dev, const void *chi_dev, int64_t npts, const double *pts_dev,
                         void *u_dev, void *cuda_stream) {
    if (!P || !phi_dev || !chi_dev || npts < 0 || (npts > 0 && (!pts_dev || !u_dev))) {
        set_error("bem_field: bad argument");
        return BEM_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    BEM_CUDA(cudaSetDevice(P->device));
    BEM_CUDA(cudaMemsetAsync(P->skip, 0, sizeof(int), s));
    struct Mark {                                        // also where a call below fails
        bem_plan *P;
        cudaStream_t s;
        ~Mark() { P->fence.mark(s); }
    } mark{P, s};
    BEM_TRY(field_moments(P, phi_dev, chi_dev, s));
    const double *ph = (const double *)phi_dev, *ch = (const double *)chi_dev;
    double *u = (double *)u_dev;
    const bool helm = P->green == BEM_HELMHOLTZ;
    if (P->prm.precision == BEM_MIXED)
        return helm ? launch_field<float, 2>(P, npts, pts_dev, u, ph, ch, P->fM, s)
                    : launch_field<float, 1>(P, npts, pts_dev, u, ph, ch, P->fM, s);
    return helm ? launch_field<double, 2>(P, npts, pts_dev, u, ph, ch, P->M, s)
                : launch_field<double, 1>(P, npts, pts_dev, u, ph, ch, P->M, s);
}

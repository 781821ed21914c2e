// Restarted GMRES on A phi = b (b = B chi from one product), device resident:
// float64 Arnoldi with classical Gram-Schmidt applied twice (CGS2), Givens
// rotations on the Hessenberg column, and the true residual b - A x at every
// restart.  Vectors are real or complex (interleaved pairs).  A device flag
// set by the rotation step makes every later kernel of the cycle a no-op once
// the estimated residual reaches the tolerance, so a whole cycle is enqueued
// (or replayed as one captured graph) and the host synchronises once per
// cycle.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <chrono>
#include <new>
#include <vector>

#include "bem_internal.cuh"

namespace bem {

constexpr int GM_T = 256;
constexpr int GM_BLK = 304;     // partial-sum blocks at most (2 per SM on a 152-SM part)
constexpr int GM_MAXV = 201;    // Krylov vectors of a cycle at most (restart <= 200)
static int gm_blocks(int n) { return std::max(1, std::min(GM_BLK, (n + GM_T - 1) / GM_T)); }

// partial[i][blk][c] = sum over this block's rows of conj(V_i) w, i < nv.  Eight
// real values at a time: each thread sums its rows, a transposing butterfly
// leaves one value per four lanes (nine float64 additions a warp where eight
// separate reductions take forty: the pipe does two a cycle and SM), and eight
// threads add the warps' values.
template <int C>
__device__ __forceinline__ void block_dots(int n, int nv, const double *V, size_t ld, const double *w, double *partial,
                                           double (*red)[8]) {
    constexpr int B = 8 / C;                          // vectors per batch
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nblk = gridDim.x;
    for (int i0 = 0; i0 < nv; i0 += B) {
        double s[8];
#pragma unroll
        for (int q = 0; q < 8; q++) s[q] = 0.0;
        for (int r = blockIdx.x * GM_T + tid; r < n; r += nblk * GM_T) {
            if constexpr (C == 1) {
                const double x = w[r];
#pragma unroll
                for (int q = 0; q < B; q++)
                    if (i0 + q < nv) s[q] += V[(size_t)(i0 + q) * ld + r] * x;
            } else {
                const double2 x = *reinterpret_cast<const double2 *>(w + 2 * (size_t)r);
#pragma unroll
                for (int q = 0; q < B; q++)
                    if (i0 + q < nv) {
                        const double2 v = *reinterpret_cast<const double2 *>(V + (size_t)(i0 + q) * ld + 2 * (size_t)r);
                        s[2 * q] += v.x * x.x + v.y * x.y;
                        s[2 * q + 1] += v.x * x.y - v.y * x.x;
                    }
            }
        }
#pragma unroll
        for (int h = 4, off = 16; h >= 1; h >>= 1, off >>= 1) {
            const bool up = lane & off;
#pragma unroll
            for (int q = 0; q < h; q++) {
                const double keep = up ? s[q + h] : s[q], send = up ? s[q] : s[q + h];
                s[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        }
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        __syncthreads();                              // the previous batch is read
        if ((lane & 3) == 0) red[warp][(lane >> 4 & 1) * 4 + (lane >> 3 & 1) * 2 + (lane >> 2 & 1)] = s[0];
        __syncthreads();
        if (tid < 8 && i0 + tid / C < nv) {
            double t = red[0][tid];
#pragma unroll
            for (int k = 1; k < GM_T / 32; k++) t += red[k][tid];
            partial[((size_t)(i0 + tid / C) * nblk + blockIdx.x) * C + tid % C] = t;
        }
    }
}

template <int C>
__global__ void __launch_bounds__(GM_T) k_mdot(int n, int nv, const double *__restrict__ V, size_t ld,
                                               const double *__restrict__ w, double *__restrict__ partial,
                                               const int *__restrict__ skip) {
    if (skip && *skip) return;
    __shared__ double red[GM_T / 32][8];
    block_dots<C>(n, nv, V, ld, w, partial, red);
}

// out[i] (+)= sum_blk partial[i][blk], one warp per i; fixed order
template <int C>
__global__ void k_mdot_final(int nv, const double *__restrict__ partial, double *out, int accumulate,
                             const int *__restrict__ skip) {
    if (skip && *skip) return;
    const int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x & 31;
    if (i >= nv) return;
    double s[C];
#pragma unroll
    for (int c = 0; c < C; c++) s[c] = 0.0;
    for (int b = lane; b < GM_BLK; b += 32)
#pragma unroll
        for (int c = 0; c < C; c++) s[c] += partial[((size_t)i * GM_BLK + b) * C + c];
#pragma unroll
    for (int c = 0; c < C; c++)
        for (int off = 16; off; off >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], off);
    if (lane == 0)
#pragma unroll
        for (int c = 0; c < C; c++) out[(size_t)i * C + c] = (accumulate ? out[(size_t)i * C + c] : 0.0) + s[c];
}

// One Gram-Schmidt update with its reduction: h_i = sum_blk partial[i][blk]
// (every block sums the partials itself, in one fixed order; block 0 stores h),
// then w -= sum_i h_i V_i on this block's rows.  LAST: the block also leaves the
// sum of |w|^2 over its rows in npart[block].  Otherwise it goes on to the next
// pass's partial sums of the same rows (partial2).
template <int C, bool LAST>
__global__ void __launch_bounds__(GM_T) k_orth_fused(int n, int nv, const double *__restrict__ V, size_t ld,
                                                     const double *__restrict__ partial, double *hout, double *w,
                                                     double *partial2, double *npart, const int *__restrict__ skip) {
    if (skip && *skip) return;
    __shared__ double hs[GM_MAXV * C];
    __shared__ double red[GM_T / 32][8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nblk = gridDim.x;
    for (int i = warp; i < nv; i += GM_T / 32) {
        double t[C];
#pragma unroll
        for (int c = 0; c < C; c++) t[c] = 0.0;
        for (int b = lane; b < nblk; b += 32)
#pragma unroll
            for (int c = 0; c < C; c++) t[c] += partial[((size_t)i * nblk + b) * C + c];
#pragma unroll
        for (int c = 0; c < C; c++)
            for (int off = 16; off; off >>= 1) t[c] += __shfl_xor_sync(0xffffffffu, t[c], off);
        if (lane == 0)
#pragma unroll
            for (int c = 0; c < C; c++) {
                hs[i * C + c] = t[c];
                if (blockIdx.x == 0) hout[(size_t)i * C + c] = t[c];
            }
    }
    __syncthreads();
    double sq = 0.0;
    for (int r = blockIdx.x * GM_T + tid; r < n; r += nblk * GM_T) {
        double a[C];
#pragma unroll
        for (int c = 0; c < C; c++) a[c] = w[(size_t)r * C + c];
#pragma unroll 4
        for (int i = 0; i < nv; i++) {
            const double *v = V + (size_t)i * ld;
            if (C == 1) {
                a[0] -= hs[i] * v[r];
            } else {
                double hr = hs[2 * i], hi = hs[2 * i + 1], vr = v[2 * (size_t)r], vi = v[2 * (size_t)r + 1];
                a[0] -= hr * vr - hi * vi;
                a[C - 1] -= hr * vi + hi * vr;
            }
        }
#pragma unroll
        for (int c = 0; c < C; c++) {
            w[(size_t)r * C + c] = a[c];
            sq += a[c] * a[c];
        }
    }
    if constexpr (LAST) {
        for (int off = 16; off; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
        if (lane == 0) red[warp][0] = sq;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int k = 0; k < GM_T / 32; k++) t += red[k][0];
            npart[blockIdx.x] = t;
        }
    } else {
        block_dots<C>(n, nv, V, ld, w, partial2, red);   // each thread reads back the rows it wrote
    }
}

template <int C>
__global__ void k_nrm2_partial(int n, const double *__restrict__ v, double *partial, const int *__restrict__ skip) {
    if (skip && *skip) return;
    __shared__ double red[GM_T];
    double s = 0.0;
    for (int r = blockIdx.x * GM_T + threadIdx.x; r < n * C; r += GM_BLK * GM_T) s += v[r] * v[r];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int off = GM_T / 2; off; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_nrm2_final(const double *__restrict__ partial, double *out, const int *__restrict__ skip) {
    if (skip && *skip) return;
    double s = 0.0;
    for (int b = threadIdx.x; b < GM_BLK; b += 32) s += partial[b];
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) *out = sqrt(s);
}

// r = b - r (r holds A x on entry) and the partial sums of |r|^2
template <int C>
__global__ void k_resid_nrm2(int n, const double *__restrict__ b, double *r, double *partial, const int *__restrict__ skip) {
    if (skip && *skip) return;
    __shared__ double red[GM_T];
    double s = 0.0;
    for (int i = blockIdx.x * GM_T + threadIdx.x; i < n * C; i += GM_BLK * GM_T) {
        const double v = b[i] - r[i];
        r[i] = v;
        s += v * v;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int off = GM_T / 2; off; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}
// before a product: the stop flag back to the halt flag, the product's slots
__global__ void k_arm(int *st, const void **xptr, void **yptr, void *const *src, void *y) {
    st[0] = st[2];
    xptr[0] = *src;
    yptr[0] = y;
}

// Targets of a mixed-precision solve.  The float32 operator's rounding leaves
// a true (float64) residual floor of 2-5e-8.  Arnoldi steps go on until the
// estimated residual reaches TAU_MIXED_CYCLE, just above that floor, and a
// true residual up to TAU_MIXED is accepted: the cycle that reaches the
// estimate ends the solve, instead of a second, one-step cycle taken to push
// the true residual from just above the floor to just below it.
constexpr double TAU_MIXED = 1e-7;
constexpr double TAU_MIXED_CYCLE = 5e-8;
// A mixed solve that stops because a restart cycle failed to halve the true
// residual has converged only if that residual is at most max(tol, TAU_STALL).
// The second-kind collocation equation is well conditioned (condition numbers
// of order 10 on the sphere and cube), so a relative residual of 1e-6 bounds
// the solution's relative error near the 1e-5 that every solution must meet;
// the float32 operator's own floor (about 2e-8) lies fifty times below it, so
// a stall above TAU_STALL is the iteration's (a short restart, a system near
// an interior resonance), not rounding, and is reported as BEM_ENOCONV.
constexpr double TAU_STALL = 1e-6;
}  // namespace bem

extern "C" int bem_solve_stop_rule(int precision, double tol, int restarts, double rel, double prev_rel, int iters,
                                   int max_iter, int *status) {
    using namespace bem;
    const bool mixed = precision == BEM_MIXED;
    const double target = mixed ? std::max(tol, TAU_MIXED) : tol;
    int st = BEM_OK, end = 0;
    if (rel <= target) end = 1;
    else if (mixed && restarts > 1 && rel > 0.5 * prev_rel) {
        end = 1;
        st = rel <= std::max(tol, TAU_STALL) ? BEM_OK : BEM_ENOCONV;
    } else if (iters >= max_iter) {
        end = 1;
        st = BEM_ENOCONV;
    }
    if (status && end) *status = st;
    return end;
}

namespace bem {

__global__ void k_set_scalar(double *p, double v) { *p = v; }

static int set_scalar(double *p, double v, cudaStream_t s) {
    (k_set_scalar<<<1, 1, 0, s>>>(p, v), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

struct GmState {
    // scalars: [0] ||b||, [1] beta, [2] |g_{j+1}| / ||b||, [3] tol, [4] ||w||
    double *sc;
    // [0] stop flag (the cycle's kernels return at once; set by the step that
    // converges), [1] steps done in the cycle, [2] halt (the solve has ended:
    // every kernel of it returns), [4 + (j & 1)] the stop flag as step j finds it,
    // written by the step before: a step's last kernel raises [0] while its other
    // blocks start, so they read this word instead ([3] is the plan's dev_err)
    int *st;
    double *H;      // [(m+1)][m] complex pairs
    double *cs, *sn, *g, *y;
    double *hcol;   // [m+1] first Gram-Schmidt pass coefficients
    double *hcol2;  // [m+1] second pass coefficients
};

// sum of the nblk block sums of |w|^2, the same in every block (256 threads)
__device__ __forceinline__ double norm2_of(const double *__restrict__ npart, int nblk, double *red) {
    const int tid = threadIdx.x, lane = tid & 31;
    double t = 0.0;
    if (tid < 32) {
        for (int b = tid; b < nblk; b += 32) t += npart[b];
        for (int off = 16; off; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0) *red = t;
    }
    __syncthreads();
    return *red;
}

// The end of an Arnoldi step.  Blocks below the last: V_{j+1} = w / ||w|| (0 if
// that is 0) and z = M^-1 V_{j+1}, the next product's input.  The last block:
// Hessenberg column j: fold in h (from CGS2) and ||w||, apply the previous
// rotations, compute the new one, update g and the residual estimate (a serial
// chain on one thread, from values its block has brought to shared memory).
template <int C>
__global__ void __launch_bounds__(GM_T) k_step_end(int n, GmState S, int m, int j, const double *__restrict__ npart, int nblk,
                                                   const double *__restrict__ w, double *vout,
                                                   const double *__restrict__ dinv, double *z) {
    int *const next = S.st + 4 + ((j + 1) & 1);
    if (S.st[4 + (j & 1)]) {                          // no block of this launch writes that word
        if (blockIdx.x + 1 == gridDim.x && threadIdx.x == 0) *next = 1;
        return;
    }
    __shared__ double nrm, sc[GM_MAXV], ss[2 * GM_MAXV], Hc[2 * (GM_MAXV + 1)];
    const int tid = threadIdx.x;
    if (blockIdx.x + 1 < gridDim.x) {
        const int r = blockIdx.x * GM_T + tid;
        double x[C], di = 0.0;
#pragma unroll
        for (int c = 0; c < C; c++) x[c] = r < n ? w[(size_t)r * C + c] : 0.0;
        if (r < n) di = dinv[r];
        const double d = sqrt(norm2_of(npart, nblk, &nrm));
        if (r < n)
#pragma unroll
            for (int c = 0; c < C; c++) {
                const double v = d > 0.0 ? x[c] / d : 0.0;
                vout[(size_t)r * C + c] = v;
                z[(size_t)r * C + c] = di * v;
            }
        return;
    }
    for (int i = tid; i < j; i += GM_T) {
        sc[i] = S.cs[i];
        ss[2 * i] = S.sn[2 * i];
        ss[2 * i + 1] = S.sn[2 * i + 1];
    }
    for (int i = tid; i <= j; i += GM_T) {
        Hc[2 * i] = S.hcol[i * C] + S.hcol2[i * C];
        Hc[2 * i + 1] = C == 2 ? S.hcol[i * C + 1] + S.hcol2[i * C + 1] : 0.0;
    }
    double *const Hg = S.H + (size_t)j * (m + 1) * 2;   // column j, rows 0..j+1, complex pairs
    const double g0r = S.g[2 * j], g0i = S.g[2 * j + 1], bnorm = S.sc[0], tol = S.sc[3];
    const double wn = sqrt(norm2_of(npart, nblk, &nrm));
    if (tid == 0) {
        S.sc[4] = wn;
        double ar = Hc[0], ai = Hc[1];                // the entry the next rotation turns
        for (int i = 0; i < j; i++) {
            const double c = sc[i], sr = ss[2 * i], si = ss[2 * i + 1], br = Hc[2 * i + 2], bi = Hc[2 * i + 3];
            // t = c a + s b ; b' = -conj(s) a + c b
            Hc[2 * i] = c * ar + (sr * br - si * bi);
            Hc[2 * i + 1] = c * ai + (sr * bi + si * br);
            const double nbr = -(sr * ar + si * ai) + c * br, nbi = -(sr * ai - si * ar) + c * bi;
            ar = nbr;
            ai = nbi;
        }
        const double b = wn;                          // real, >= 0
        const double aa = hypot(ar, ai), rho = hypot(aa, b);
        double c, sr, si;
        if (rho == 0.0) { c = 1.0; sr = 0.0; si = 0.0; }
        else if (aa == 0.0) { c = 0.0; sr = 1.0; si = 0.0; }
        else {
            c = aa / rho;
            sr = (ar / aa) * b / rho;
            si = (ai / aa) * b / rho;
        }
        S.cs[j] = c; S.sn[2 * j] = sr; S.sn[2 * j + 1] = si;
        Hc[2 * j] = c * ar + sr * b;
        Hc[2 * j + 1] = c * ai + si * b;
        Hc[2 * j + 2] = 0.0;
        Hc[2 * j + 3] = 0.0;
        // g_{j+1} = -conj(s) g_j, g_j = c g_j
        const double g1r = -(sr * g0r + si * g0i), g1i = -(sr * g0i - si * g0r);
        S.g[2 * j + 2] = g1r;
        S.g[2 * j + 3] = g1i;
        S.g[2 * j] = c * g0r;
        S.g[2 * j + 1] = c * g0i;
        const double est = hypot(g1r, g1i) / bnorm;
        S.sc[2] = est;
        S.st[1] = j + 1;
        const bool stop = est <= tol || wn == 0.0;
        if (stop) S.st[0] = 1;
        *next = stop;
    }
    __syncthreads();
    for (int i = tid; i < 2 * (j + 2); i += GM_T) Hg[i] = Hc[i];
}

// back substitution H y = g over the steps of the cycle, then the solver
// writes x += V y
template <int C>
__global__ void k_backsolve(GmState S, int m) {
    if (S.st[2]) return;
    const int k = S.st[1];
    for (int i = k - 1; i >= 0; i--) {
        double sr = S.g[2 * i], si = S.g[2 * i + 1];
        for (int l = i + 1; l < k; l++) {
            const double *Hl = S.H + (size_t)l * (m + 1) * 2;
            double hr = Hl[2 * i], hi = Hl[2 * i + 1], yr = S.y[2 * l], yi = S.y[2 * l + 1];
            sr -= hr * yr - hi * yi;
            si -= hr * yi + hi * yr;
        }
        const double *Hi = S.H + (size_t)i * (m + 1) * 2;
        double dr = Hi[2 * i], di = Hi[2 * i + 1], den = dr * dr + di * di;
        S.y[2 * i] = (sr * dr + si * di) / den;
        S.y[2 * i + 1] = (si * dr - sr * di) / den;
    }
}

// x += M^-1 sum_{i<k} y_i V_i  (right preconditioner M = diag(C): dinv = 1 / C)
template <int C>
__global__ void k_xupdate(int n, const double *__restrict__ V, size_t ld, GmState S, double *const *xslot,
                          const double *__restrict__ dinv) {
    if (S.st[2]) return;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    double *x = *xslot;
    const int k = S.st[1];
    double a[C];
#pragma unroll
    for (int c = 0; c < C; c++) a[c] = 0.0;
    for (int i = 0; i < k; i++) {
        const double *v = V + (size_t)i * ld;
        if (C == 1) {
            a[0] += S.y[2 * i] * v[r];
        } else {
            double yr = S.y[2 * i], yi = S.y[2 * i + 1], vr = v[2 * (size_t)r], vi = v[2 * (size_t)r + 1];
            a[0] += yr * vr - yi * vi;
            a[C - 1] += yr * vi + yi * vr;
        }
    }
#pragma unroll
    for (int c = 0; c < C; c++) x[(size_t)r * C + c] += dinv[r] * a[c];
}

// The start of a cycle: V_0 = r / ||r|| and M^-1 V_0 for the first product;
// block 0 also resets the small system and points every product of the cycle at
// z and w.  (One launch; the three parts had one each.)
template <int C>
__global__ void k_cycle_begin(int n, GmState S, int m, double *v0, const double *__restrict__ dinv, double *z, double *w,
                              const void **xptr, void **yptr) {
    const bool halted = S.st[2] != 0;
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) {
            S.st[0] = S.st[4] = S.st[5] = S.st[2];
            S.st[1] = 0;
            xptr[0] = z;
            yptr[0] = w;
        }
        if (!halted)
            for (int i = threadIdx.x; i < 2 * (m + 1); i += blockDim.x) S.g[i] = i == 0 ? S.sc[1] : 0.0;   // beta
    }
    if (halted) return;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const double d = S.sc[1], di = dinv[r];
#pragma unroll
    for (int c = 0; c < C; c++) {
        const double v = d > 0.0 ? v0[(size_t)r * C + c] / d : 0.0;
        v0[(size_t)r * C + c] = v;
        z[(size_t)r * C + c] = di * v;
    }
}

// pointer slots of a solve: [0] chi (Neumann data), [1] x (the solution)
__global__ void k_set_ptrs(void **slot, const void *chi, void *x) {
    slot[0] = (void *)chi;
    slot[1] = x;
}
__global__ void k_set_ptrs_tab(void **slot, const void *const *chi_tab, void *const *x_tab, int i) {
    slot[0] = (void *)chi_tab[i];
    slot[1] = x_tab[i];
}
// x = 0 through a solve slot
__global__ void k_zero_slot(void *const *slot, size_t n, const int *__restrict__ skip) {
    if (skip && *skip) return;
    double *x = (double *)*slot;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        x[i] = 0.0;
}

// ---------------------------------------------------------------------------
// The solve as a state machine.  Every transition enqueues device work on the
// solve's own stream plus an asynchronous read-back (pinned memory) of the
// few scalars the host decides on -- ||b||, ||r||, the steps of a cycle -- and
// records an event.  bem_solve drives one solve to the end, waiting on each
// event; the batch API advances many solves of different plans together,
// querying events without blocking, so their device work overlaps.  The
// device work of each transition (start, true residual, restart cycle) is a
// fixed kernel sequence that reads x and chi through the solve's pointer
// slots, so a group of plans can also capture it once into one graph.
// ---------------------------------------------------------------------------
struct GmSolver {
    bem_plan *P = nullptr;
    const double *chi = nullptr;   // Neumann data (chi index space), device
    double *x = nullptr;           // solution, device
    bem_solve_params sp{};
    cudaStream_t s = nullptr;
    cudaEvent_t ev = nullptr;
    int phase = 0;                 // 0 start, 1 residual in flight, 2 cycle steps, 3 done, 4 cycle end in flight
    bool waiting = false;
    // cycle steps go out in chunks, at most two in flight; each chunk reports
    // the device's converged flag, and once one has, no further chunk is sent
    cudaEvent_t evc[2] = {nullptr, nullptr};
    int cyc_steps = 0, j_next = 0, nfly = 0, chunk_seq = 0;
    bool stop = false;
    int iters = 0, restarts = 0, status = BEM_ENOCONV;
    double rel = 1.0, prev_rel = 2.0, tol = 0.0;
};

static int gm_workspace(bem_plan *P, int m) {
    const int C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    if (m < 1 || m > 200) { set_error("bem_solve: restart %d outside [1, 200]", m); return BEM_EINVAL; }
    const size_t ne = (size_t)P->N * C;
    if (P->gm_restart != m) {
        if (P->V) { P->arena.release(P->V); P->arena.release(P->H); P->arena.release(P->gs); }
        BEM_TRY(P->arena.alloc(&P->V, (size_t)(m + 1) * ne));
        BEM_TRY(P->arena.alloc(&P->H, (size_t)(m + 1) * m * 2));
        BEM_TRY(P->arena.alloc(&P->gs, (size_t)12 * (m + 2)));
        P->gm_restart = m;
    }
    if (!P->w) {
        BEM_TRY(P->arena.alloc(&P->w, ne));
        BEM_TRY(P->arena.alloc(&P->zbuf, ne));
        BEM_TRY(P->arena.alloc(&P->npart, GM_BLK));
        BEM_TRY(P->arena.alloc(&P->bvec, ne));
        BEM_TRY(P->arena.alloc(&P->scal, 16 + 2 * (size_t)GM_BLK * 2 * (GM_MAXV + 1)));
        BEM_TRY(P->arena.alloc(&P->gm_slot, 2));
    }
    if (!P->hostbuf) BEM_CUDA(cudaHostAlloc((void **)&P->hostbuf, 64, cudaHostAllocDefault));
    return BEM_OK;
}

template <int C>
static GmState gm_state(bem_plan *P) {
    const int m = P->gm_restart;
    double *g0 = P->gs;
    return GmState{P->scal, P->istate, P->H, g0, g0 + m, g0 + 3 * m, g0 + 5 * m + 2, g0 + 7 * m + 2, g0 + 9 * m + 4};
}

// the product inside a solve: a replay of the plan's graph, or (inside a
// group capture) its kernels
static int gm_product(bem_plan *P, int op, cudaStream_t s, bool raw) {
    if (raw) return enqueue_matvec_raw(P, op, P->green, P->k, 1, s);
    return enqueue_matvec(P, op, P->green, P->k, s);
}

// b = B chi, ||b||, tolerance, x = 0
template <int C>
static int gm_k_start(bem_plan *P, double tol, cudaStream_t s, bool raw) {
    const int n = (int)P->N;
    double *partial = P->scal + 16;
    GmState S = gm_state<C>(P);
    int *skip = P->istate;
    (k_arm<<<1, 1, 0, s>>>(P->istate, P->xptr, P->yptr, (void *const *)P->gm_slot, P->bvec), ::bem::count_launch());
    BEM_TRY(gm_product(P, BEM_OP_B, s, raw));
    (k_nrm2_partial<C><<<GM_BLK, GM_T, 0, s>>>(n, P->bvec, partial, skip), ::bem::count_launch());
    (k_nrm2_final<<<1, 32, 0, s>>>(partial, S.sc + 0, skip), ::bem::count_launch());
    BEM_TRY(set_scalar(S.sc + 3, tol, s));
    (k_zero_slot<<<GM_BLK, 256, 0, s>>>((void *const *)P->gm_slot + 1, (size_t)n * C, skip), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// true residual r = b - A x into V_0 (unscaled), beta = ||r||
template <int C>
static int gm_k_residual(bem_plan *P, cudaStream_t s, bool raw) {
    const int n = (int)P->N;
    double *V = P->V, *partial = P->scal + 16;
    GmState S = gm_state<C>(P);
    int *skip = P->istate;
    (k_arm<<<1, 1, 0, s>>>(P->istate, P->xptr, P->yptr, (void *const *)P->gm_slot + 1, V), ::bem::count_launch());
    BEM_TRY(gm_product(P, BEM_OP_A, s, raw));
    (k_resid_nrm2<C><<<GM_BLK, GM_T, 0, s>>>(n, P->bvec, V, partial, skip), ::bem::count_launch());
    (k_nrm2_final<<<1, 32, 0, s>>>(partial, S.sc + 1, skip), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

// one restart cycle: Arnoldi (CGS2) + Givens for up to `steps` steps, then
// x += V y.  Begin, one step, end: the solver enqueues steps in chunks, the
// captured group graphs the whole cycle.
template <int C>
static int gm_k_cycle_begin(bem_plan *P, cudaStream_t s) {
    const int n = (int)P->N, nb = (n + 255) / 256;
    GmState S = gm_state<C>(P);
    (k_cycle_begin<C><<<nb, 256, 0, s>>>(n, S, P->gm_restart, P->V, P->dinv, P->zbuf, P->w, P->xptr, P->yptr),
     ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

template <int C>
static int gm_k_step(bem_plan *P, int j, cudaStream_t s, bool raw) {
    const int n = (int)P->N, m = P->gm_restart, ne = n * C;
    const size_t ld = (size_t)ne;
    double *V = P->V, *w = P->w, *partial = P->scal + 16, *partial2 = partial + (size_t)GM_BLK * 2 * (GM_MAXV + 1);
    GmState S = gm_state<C>(P);
    const int nb = (n + 255) / 256, ng = gm_blocks(n);
    int *skip = P->istate;
    // the product of M^-1 V_j (zbuf, written with V_j) into w
    BEM_TRY(gm_product(P, BEM_OP_A, s, raw));
    // CGS2: two classical Gram-Schmidt passes against V_0..V_j.  Partial sums; an
    // update that reduces them itself and forms the second pass's; the second
    // update, which sums |w|^2 per block; then the scaling of V_{j+1} beside the
    // rotation step.  Four kernels (six before, 54 us a step on 48,602 rows: the
    // dot products reduced vector by vector and the rotation walked a chain of
    // global loads)
    (k_mdot<C><<<ng, GM_T, 0, s>>>(n, j + 1, V, ld, w, partial, skip), ::bem::count_launch());
    (k_orth_fused<C, false><<<ng, GM_T, 0, s>>>(n, j + 1, V, ld, partial, S.hcol, w, partial2, nullptr, skip), ::bem::count_launch());
    (k_orth_fused<C, true><<<ng, GM_T, 0, s>>>(n, j + 1, V, ld, partial2, S.hcol2, w, nullptr, P->npart, skip), ::bem::count_launch());
    (k_step_end<C><<<nb + 1, GM_T, 0, s>>>(n, S, m, j, P->npart, ng, w, V + (size_t)(j + 1) * ld, P->dinv, P->zbuf),
     ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

template <int C>
static int gm_k_cycle_end(bem_plan *P, cudaStream_t s) {
    const int n = (int)P->N;
    GmState S = gm_state<C>(P);
    (k_backsolve<C><<<1, 1, 0, s>>>(S, P->gm_restart), ::bem::count_launch());
    (k_xupdate<C><<<(n + 255) / 256, 256, 0, s>>>(n, P->V, (size_t)n * C, S, (double *const *)P->gm_slot + 1, P->dinv),
     ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

template <int C>
static int gm_k_cycle(bem_plan *P, int steps, cudaStream_t s, bool raw) {
    BEM_TRY(gm_k_cycle_begin<C>(P, s));
    for (int j = 0; j < steps; j++) BEM_TRY(gm_k_step<C>(P, j, s, raw));
    return gm_k_cycle_end<C>(P, s);
}

static double gm_tol(const bem_plan *P, double tol) {
    // the Arnoldi estimate's target; the true residual's is bem_solve_stop_rule's
    return P->prm.precision == BEM_MIXED ? std::max(tol, TAU_MIXED_CYCLE) : tol;
}


// host decision after a true residual: returns true when the solve has ended
static bool gm_after_residual(GmSolver &g, double bnorm, double beta) {
    g.restarts++;
    g.rel = bnorm > 0.0 ? beta / bnorm : 0.0;
    int status = BEM_OK;
    const bool end = bem_solve_stop_rule(g.P->prm.precision, g.sp.tol, g.restarts, g.rel, g.prev_rel, g.iters,
                                         g.sp.max_iter, &status) != 0;
    g.prev_rel = g.rel;
    if (end) g.status = status;
    return end;
}

template <int C>
static int gm_enqueue_residual(GmSolver &g) {
    bem_plan *P = g.P;
    GmState S = gm_state<C>(P);
    BEM_TRY(gm_k_residual<C>(P, g.s, false));
    BEM_CUDA(cudaMemcpyAsync(P->hostbuf, S.sc, sizeof(double) * 2, cudaMemcpyDeviceToHost, g.s));
    BEM_CUDA(cudaEventRecord(g.ev, g.s));
    g.waiting = true;
    g.phase = 1;
    return BEM_OK;
}

// The first residual of a solve: x = 0, so r = b and beta = ||b|| (the
// product of the zero vector is exactly zero and is not formed).
template <int C>
static int gm_enqueue_start(GmSolver &g) {
    bem_plan *P = g.P;
    GmState S = gm_state<C>(P);
    g.tol = gm_tol(P, g.sp.tol);
    BEM_CUDA(cudaMemsetAsync(P->istate, 0, sizeof(int) * 3, g.s));
    (k_set_ptrs<<<1, 1, 0, g.s>>>((void **)P->gm_slot, g.chi, g.x), ::bem::count_launch());
    BEM_TRY(gm_k_start<C>(P, g.tol, g.s, false));
    BEM_CUDA(cudaMemcpyAsync(P->V, P->bvec, sizeof(double) * (size_t)P->N * C, cudaMemcpyDeviceToDevice, g.s));
    BEM_CUDA(cudaMemcpyAsync(S.sc + 1, S.sc, sizeof(double), cudaMemcpyDeviceToDevice, g.s));
    BEM_CUDA(cudaMemcpyAsync(P->hostbuf, S.sc, sizeof(double) * 2, cudaMemcpyDeviceToHost, g.s));
    BEM_CUDA(cudaEventRecord(g.ev, g.s));
    g.waiting = true;
    g.phase = 1;
    return BEM_OK;
}

constexpr int GM_CHUNK = 1;         // Arnoldi steps per chunk (two chunks in flight: at most one step too many)

template <int C>
static int gm_enqueue_cycle(GmSolver &g) {
    BEM_TRY(gm_k_cycle_begin<C>(g.P, g.s));
    g.cyc_steps = std::min(g.P->gm_restart, g.sp.max_iter - g.iters);
    g.j_next = g.nfly = g.chunk_seq = 0;
    g.stop = false;
    g.waiting = false;
    g.phase = 2;
    return BEM_OK;
}

// Sends chunks of cycle steps (at most two in flight) and reads their
// converged flags; once every chunk has finished, the cycle's end.  Returns
// with phase 2 when a chunk is pending and the call does not block.
template <int C>
static int gm_cycle_steps(GmSolver &g, bool blocking) {
    bem_plan *P = g.P;
    GmState S = gm_state<C>(P);
    for (;;) {
        if (!g.stop && g.j_next < g.cyc_steps && g.nfly < 2) {
            const int j1 = std::min(g.cyc_steps, g.j_next + GM_CHUNK), k = (g.chunk_seq + g.nfly) & 1;
            for (int j = g.j_next; j < j1; j++) BEM_TRY(gm_k_step<C>(P, j, g.s, false));
            BEM_CUDA(cudaMemcpyAsync(P->hostbuf + 4 + k, S.st, sizeof(int), cudaMemcpyDeviceToHost, g.s));
            BEM_CUDA(cudaEventRecord(g.evc[k], g.s));
            g.j_next = j1;
            g.nfly++;
            continue;
        }
        if (g.nfly == 0) break;
        const int k = g.chunk_seq & 1;             // the oldest chunk in flight
        cudaError_t e = blocking ? cudaEventSynchronize(g.evc[k]) : cudaEventQuery(g.evc[k]);
        if (e == cudaErrorNotReady) return BEM_OK;
        if (e != cudaSuccess) return cuda_fail(e, "GMRES chunk event", __FILE__, __LINE__);
        int conv;
        memcpy(&conv, P->hostbuf + 4 + k, sizeof(int));
        g.nfly--;
        g.chunk_seq++;
        if (conv) g.stop = true;
    }
    BEM_TRY(gm_k_cycle_end<C>(P, g.s));
    BEM_CUDA(cudaMemcpyAsync(P->hostbuf + 2, S.st + 1, sizeof(int), cudaMemcpyDeviceToHost, g.s));
    BEM_CUDA(cudaEventRecord(g.ev, g.s));
    g.waiting = true;
    g.phase = 4;
    return BEM_OK;
}

// Advances the solve as far as finished device work allows.  blocking: wait
// for each pending event; otherwise return as soon as one is still pending.
template <int C>
static int gm_advance(GmSolver &g, bool blocking) {
    while (g.phase != 3) {
        if (g.phase == 0) {
            BEM_TRY(gm_enqueue_start<C>(g));
            continue;
        }
        if (g.phase == 2) {
            BEM_TRY(gm_cycle_steps<C>(g, blocking));
            if (g.phase == 2) return BEM_OK;          // a chunk is still running
            continue;
        }
        if (g.waiting) {
            cudaError_t e = blocking ? cudaEventSynchronize(g.ev) : cudaEventQuery(g.ev);
            if (e == cudaErrorNotReady) return BEM_OK;
            if (e != cudaSuccess) return cuda_fail(e, "GMRES event", __FILE__, __LINE__);
            g.waiting = false;
        }
        const double *h = g.P->hostbuf;
        if (g.phase == 1) {
            if (gm_after_residual(g, h[0], h[1])) {
                g.phase = 3;
                break;
            }
            BEM_TRY(gm_enqueue_cycle<C>(g));
        } else {
            int steps;
            memcpy(&steps, g.P->hostbuf + 2, sizeof(int));
            g.iters += steps;
            if (steps == 0) {
                g.status = BEM_ENOCONV;
                g.phase = 3;
                break;
            }
            BEM_TRY(gm_enqueue_residual<C>(g));
        }
    }
    return BEM_OK;
}

// the event a solver is waiting for (the oldest chunk while steps are out)
static cudaEvent_t gm_pending_event(const GmSolver &g) {
    return g.phase == 2 && g.nfly > 0 ? g.evc[g.chunk_seq & 1] : g.ev;
}

static void gm_release(GmSolver &g) {
    if (g.ev) cudaEventDestroy(g.ev);
    for (auto &e : g.evc)
        if (e) cudaEventDestroy(e);
    g.ev = g.evc[0] = g.evc[1] = nullptr;
}

static int gm_init(GmSolver &g, bem_plan *P, const double *chi, double *x, const bem_solve_params *sp, cudaStream_t s) {
    g = GmSolver{};
    g.P = P;
    g.chi = chi;
    g.x = x;
    g.sp = *sp;
    g.s = s;
    BEM_TRY(gm_workspace(P, sp->restart));
    BEM_CUDA(cudaEventCreateWithFlags(&g.ev, cudaEventDisableTiming));
    for (auto &e : g.evc) BEM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return BEM_OK;
}

static int gm_run(GmSolver &g, bool blocking) {
    return g.P->green == BEM_HELMHOLTZ ? gm_advance<2>(g, blocking) : gm_advance<1>(g, blocking);
}

// ---------------------------------------------------------------------------
// BiCGStab (the paper's solver, Section 4), device resident in float64:
//   rho = rh^H r, beta = (rho / rho_prev)(alpha / omega), p = r + beta (p - omega v),
//   v = A p, alpha = rho / (rh^H v), s = r - alpha v, t = A s,
//   omega = (t^H s) / (t^H t), x += alpha p + omega s, r = s - omega t,
// with rh the residual at the (re)start.  The iteration stops on the device
// (the shared skip flag) once ||r|| / ||b|| reaches the tolerance or a
// denominator vanishes; the host then evaluates the true residual b - A x and
// restarts from it (rh = r) while it is above the tolerance, with the same
// stopping rule as GMRES (mixed plans: max(tol, TAU_MIXED), or a restart that
// fails to halve the true residual).  Steps go out in chunks of GM_CHUNK with
// at most two in flight, each chunk reading back the flag.
// ---------------------------------------------------------------------------
struct BcState {
    // scalars (complex as pairs): [0] rho, [2] rho_prev, [4] alpha, [6] omega,
    // [8] rh^H v, [10] t^H s, [12] ||t||, [13] ||r||, [14] ||r|| / ||b||
    double *sc;
    int *st;                            // [0] steps since the (re)start, [1] breakdown
    double *r, *rh, *p, *v, *s, *t;
    const double *bn, *tol;             // ||b|| and the tolerance (GMRES scalars 0 and 3)
};

static int bc_workspace(bem_plan *P) {
    const int C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    if (!P->bc_vec) {
        BEM_TRY(P->arena.alloc(&P->bc_vec, (size_t)6 * P->N * C));
        BEM_TRY(P->arena.alloc(&P->bc_sc, 32));
        BEM_TRY(P->arena.alloc(&P->bc_st, 4));
    }
    return BEM_OK;
}

static BcState bc_state(bem_plan *P, int C) {
    const size_t ne = (size_t)P->N * C;
    double *b = P->bc_vec;
    return BcState{P->bc_sc, P->bc_st, b, b + ne, b + 2 * ne, b + 3 * ne, b + 4 * ne, b + 5 * ne, P->scal, P->scal + 3};
}

__device__ __forceinline__ void cmul(double ar, double ai, double br, double bi, double &cr, double &ci) {
    cr = ar * br - ai * bi;
    ci = ar * bi + ai * br;
}
__device__ __forceinline__ void cdiv(double ar, double ai, double br, double bi, double &cr, double &ci) {
    const double d = br * br + bi * bi;
    cr = (ar * br + ai * bi) / d;
    ci = (ai * br - ar * bi) / d;
}

// at a (re)start: rh = r, p = v = 0, rho_prev = alpha = omega = 1
template <int C>
__global__ void k_bc_reset(int ne, BcState B) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ne) {
        B.rh[i] = B.r[i];
        B.p[i] = 0.0;
        B.v[i] = 0.0;
    }
    if (i == 0) {
        B.sc[2] = 1.0; B.sc[3] = 0.0; B.sc[4] = 1.0; B.sc[5] = 0.0; B.sc[6] = 1.0; B.sc[7] = 0.0;
        B.st[0] = 0;
        B.st[1] = 0;
    }
}

// p = r + beta (p - omega v)
template <int C>
__global__ void k_bc_p(int n, BcState B, const int *__restrict__ skip) {
    if (*skip) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double q0, q1, br, bi;
    cdiv(B.sc[0], C == 2 ? B.sc[1] : 0.0, B.sc[2], C == 2 ? B.sc[3] : 0.0, q0, q1);
    double a0, a1;
    cdiv(B.sc[4], C == 2 ? B.sc[5] : 0.0, B.sc[6], C == 2 ? B.sc[7] : 0.0, a0, a1);
    cmul(q0, q1, a0, a1, br, bi);
    if (C == 1) {
        B.p[i] = B.r[i] + br * (B.p[i] - B.sc[6] * B.v[i]);
    } else {
        double wr, wi;
        cmul(B.sc[6], B.sc[7], B.v[2 * i], B.v[2 * i + 1], wr, wi);
        const double dr = B.p[2 * i] - wr, di = B.p[2 * i + 1] - wi;
        double er, ei;
        cmul(br, bi, dr, di, er, ei);
        B.p[2 * i] = B.r[2 * i] + er;
        B.p[2 * i + 1] = B.r[2 * i + 1] + ei;
    }
}

// alpha = rho / (rh^H v), s = r - alpha v; a vanishing denominator stops the run
template <int C>
__global__ void k_bc_s(int n, BcState B, int *skip) {
    if (*skip) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double sr = B.sc[8], si = C == 2 ? B.sc[9] : 0.0;
    if (sr == 0.0 && si == 0.0) {
        if (i == 0) B.st[1] = 1;
        return;
    }
    double ar, ai;
    cdiv(B.sc[0], C == 2 ? B.sc[1] : 0.0, sr, si, ar, ai);
    if (i == 0) { B.sc[4] = ar; B.sc[5] = ai; }
    if (i >= n) return;
    if (C == 1) {
        B.s[i] = B.r[i] - ar * B.v[i];
    } else {
        double wr, wi;
        cmul(ar, ai, B.v[2 * i], B.v[2 * i + 1], wr, wi);
        B.s[2 * i] = B.r[2 * i] - wr;
        B.s[2 * i + 1] = B.r[2 * i + 1] - wi;
    }
}

// omega = (t^H s) / ||t||^2, x += alpha p + omega s, r = s - omega t
template <int C>
__global__ void k_bc_xr(int n, BcState B, void *const *xslot, const int *skip) {
    if (*skip || B.st[1]) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double tt = B.sc[12] * B.sc[12];
    double wr = 0.0, wi = 0.0;
    if (tt > 0.0) {
        wr = B.sc[10] / tt;
        wi = C == 2 ? B.sc[11] / tt : 0.0;
    }
    if (i == 0) { B.sc[6] = wr; B.sc[7] = wi; }
    if (i >= n) return;
    double *x = (double *)*xslot;
    const double ar = B.sc[4], ai = C == 2 ? B.sc[5] : 0.0;
    if (C == 1) {
        x[i] += ar * B.p[i] + wr * B.s[i];
        B.r[i] = B.s[i] - wr * B.t[i];
    } else {
        double pr, pi, qr, qi, tr, ti;
        cmul(ar, ai, B.p[2 * i], B.p[2 * i + 1], pr, pi);
        cmul(wr, wi, B.s[2 * i], B.s[2 * i + 1], qr, qi);
        cmul(wr, wi, B.t[2 * i], B.t[2 * i + 1], tr, ti);
        x[2 * i] += pr + qr;
        x[2 * i + 1] += pi + qi;
        B.r[2 * i] = B.s[2 * i] - tr;
        B.r[2 * i + 1] = B.s[2 * i + 1] - ti;
    }
}

// end of a step: residual estimate, step count, stop flag
__global__ void k_bc_check(BcState B, int *skip, int max_steps) {
    if (*skip) return;
    const double bn = *B.bn;
    const double est = bn > 0.0 ? B.sc[13] / bn : 0.0;
    B.sc[14] = est;
    B.st[0] += 1;
    B.sc[2] = B.sc[0];
    B.sc[3] = B.sc[1];
    const bool wzero = B.sc[6] == 0.0 && B.sc[7] == 0.0;
    if (B.st[1] || wzero) B.st[1] = 1;
    if (est <= *B.tol || B.st[1] || B.st[0] >= max_steps) *skip = 1;
}

template <int C>
static int bc_k_step(bem_plan *P, const BcState &B, int max_steps, cudaStream_t s) {
    const int n = (int)P->N, nb = (n + 255) / 256;
    const size_t ld = (size_t)n * C;
    double *partial = P->scal + 16;
    int *skip = P->istate;
    (k_mdot<C><<<GM_BLK, GM_T, 0, s>>>(n, 1, B.rh, ld, B.r, partial, skip), ::bem::count_launch());
    (k_mdot_final<C><<<1, 32, 0, s>>>(1, partial, B.sc + 0, 0, skip), ::bem::count_launch());
    (k_bc_p<C><<<nb, 256, 0, s>>>(n, B, skip), ::bem::count_launch());
    BEM_TRY(set_slots(P, B.p, B.v, s));
    BEM_TRY(gm_product(P, BEM_OP_A, s, false));
    (k_mdot<C><<<GM_BLK, GM_T, 0, s>>>(n, 1, B.rh, ld, B.v, partial, skip), ::bem::count_launch());
    (k_mdot_final<C><<<1, 32, 0, s>>>(1, partial, B.sc + 8, 0, skip), ::bem::count_launch());
    (k_bc_s<C><<<nb, 256, 0, s>>>(n, B, skip), ::bem::count_launch());
    BEM_TRY(set_slots(P, B.s, B.t, s));
    BEM_TRY(gm_product(P, BEM_OP_A, s, false));
    (k_mdot<C><<<GM_BLK, GM_T, 0, s>>>(n, 1, B.t, ld, B.s, partial, skip), ::bem::count_launch());
    (k_mdot_final<C><<<1, 32, 0, s>>>(1, partial, B.sc + 10, 0, skip), ::bem::count_launch());
    (k_nrm2_partial<C><<<GM_BLK, GM_T, 0, s>>>(n, B.t, partial, skip), ::bem::count_launch());
    (k_nrm2_final<<<1, 32, 0, s>>>(partial, B.sc + 12, skip), ::bem::count_launch());
    (k_bc_xr<C><<<nb, 256, 0, s>>>(n, B, (void *const *)P->gm_slot + 1, skip), ::bem::count_launch());
    (k_nrm2_partial<C><<<GM_BLK, GM_T, 0, s>>>(n, B.r, partial, skip), ::bem::count_launch());
    (k_nrm2_final<<<1, 32, 0, s>>>(partial, B.sc + 13, skip), ::bem::count_launch());
    (k_bc_check<<<1, 1, 0, s>>>(B, skip, max_steps), ::bem::count_launch());
    BEM_LAUNCH_CHECK();
    return BEM_OK;
}

template <int C>
static int bicgstab_one(bem_plan *P, const double *chi, double *x, const bem_solve_params &sp, bem_solve_info *info,
                        cudaStream_t s) {
    BEM_TRY(gm_workspace(P, P->gm_restart > 0 ? P->gm_restart : 1));
    BEM_TRY(bc_workspace(P));
    const BcState B = bc_state(P, C);
    const size_t ne = (size_t)P->N * C;
    const double tol = gm_tol(P, sp.tol);
    cudaEvent_t ev[2];
    for (auto &e : ev) BEM_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    auto done = [&](int rc) {
        for (auto &e : ev) cudaEventDestroy(e);
        return rc;
    };
    BEM_CUDA(cudaMemsetAsync(P->istate, 0, sizeof(int) * 3, s));
    (k_set_ptrs<<<1, 1, 0, s>>>((void **)P->gm_slot, chi, x), ::bem::count_launch());
    BEM_TRY(gm_k_start<C>(P, tol, s, false));                    // b, ||b||, x = 0
    BEM_CUDA(cudaMemcpyAsync(B.r, P->bvec, sizeof(double) * ne, cudaMemcpyDeviceToDevice, s));
    BEM_CUDA(cudaMemcpyAsync(P->hostbuf, P->scal, sizeof(double), cudaMemcpyDeviceToHost, s));
    BEM_CUDA(cudaStreamSynchronize(s));
    const double bnorm = P->hostbuf[0];
    int iters = 0, restarts = 0, status = BEM_ENOCONV;
    double rel = bnorm > 0.0 ? 1.0 : 0.0, prev = 2.0;
    if (bnorm == 0.0) status = BEM_OK;
    while (status != BEM_OK && iters < sp.max_iter) {
        const int budget = sp.max_iter - iters;
        BEM_CUDA(cudaMemsetAsync(P->istate, 0, sizeof(int), s));
        (k_bc_reset<C><<<(int)((ne + 255) / 256), 256, 0, s>>>((int)ne, B), ::bem::count_launch());
        // chunks of steps, at most two in flight, each reading back the stop flag
        int sent = 0, nfly = 0, seq = 0;
        bool stop = false;
        for (;;) {
            if (!stop && sent < budget && nfly < 2) {
                const int j1 = std::min(budget, sent + GM_CHUNK), k = (seq + nfly) & 1;
                for (int j = sent; j < j1; j++) BEM_TRY(bc_k_step<C>(P, B, budget, s));
                BEM_CUDA(cudaMemcpyAsync(P->hostbuf + 4 + k, P->istate, sizeof(int), cudaMemcpyDeviceToHost, s));
                BEM_CUDA(cudaEventRecord(ev[k], s));
                sent = j1;
                nfly++;
                continue;
            }
            if (nfly == 0) break;
            const int k = seq & 1;
            BEM_CUDA(cudaEventSynchronize(ev[k]));
            int flag;
            memcpy(&flag, P->hostbuf + 4 + k, sizeof(int));
            nfly--;
            seq++;
            if (flag) stop = true;
        }
        int st[2];
        BEM_CUDA(cudaMemcpyAsync(st, B.st, sizeof(int) * 2, cudaMemcpyDeviceToHost, s));
        // true residual r = b - A x (into V_0), its norm; the next run starts from it
        BEM_TRY(gm_k_residual<C>(P, s, false));
        BEM_CUDA(cudaMemcpyAsync(P->hostbuf, P->scal, sizeof(double) * 2, cudaMemcpyDeviceToHost, s));
        BEM_CUDA(cudaMemcpyAsync(B.r, P->V, sizeof(double) * ne, cudaMemcpyDeviceToDevice, s));
        BEM_CUDA(cudaStreamSynchronize(s));
        iters += st[0];
        restarts++;
        rel = P->hostbuf[1] / bnorm;
        int rs = BEM_OK;
        if (bem_solve_stop_rule(P->prm.precision, sp.tol, restarts, rel, prev, iters, sp.max_iter, &rs)) {
            status = rs;
            break;
        }
        if (st[0] == 0) break;                               // no progress from this residual
        prev = rel;
    }
    if (info) *info = bem_solve_info{iters, restarts, rel, status};
    return done(status);
}

static int bicgstab(bem_plan *P, const void *chi, void *phi, int nrhs, const bem_solve_params *sp,
                    bem_solve_info *info, cudaStream_t s) {
    const int C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    const size_t nchi = (size_t)P->nchi * C, ne = (size_t)P->N * C;
    int worst = BEM_OK;
    for (int r = 0; r < nrhs; r++) {
        const double *c = (const double *)chi + r * nchi;
        double *x = (double *)phi + r * ne;
        const int rc = C == 2 ? bicgstab_one<2>(P, c, x, *sp, info ? info + r : nullptr, s)
                              : bicgstab_one<1>(P, c, x, *sp, info ? info + r : nullptr, s);
        if (rc == BEM_ENOCONV) worst = BEM_ENOCONV;
        else if (rc != BEM_OK) return rc;
    }
    return worst;
}

int solve(bem_plan *P, const void *chi, void *phi, int nrhs, const bem_solve_params *sp, bem_solve_info *info,
          cudaStream_t s) {
    if (sp->method == BEM_BICGSTAB) return bicgstab(P, chi, phi, nrhs, sp, info, s);
    const int C = P->green == BEM_HELMHOLTZ ? 2 : 1;
    int worst = BEM_OK;
    const size_t nchi = (size_t)P->nchi * C, ne = (size_t)P->N * C;
    for (int r = 0; r < nrhs; r++) {
        GmSolver g;
        BEM_TRY(gm_init(g, P, (const double *)chi + r * nchi, (double *)phi + r * ne, sp, s));
        int rc = gm_run(g, true);
        gm_release(g);
        if (rc != BEM_OK) return rc;
        if (info) info[r] = bem_solve_info{g.iters, g.restarts, g.rel, g.status};
        if (g.status == BEM_ENOCONV) worst = BEM_ENOCONV;
    }
    return worst;
}

// ---------------------------------------------------------------------------
// Group solves: many plans (meshes of any size, either Green's function,
// either precision) advanced in lock step, every restart cycle of every
// member one launch of a single captured graph (members are parallel
// branches; a member that has ended is halted and its branch returns at once).
// ---------------------------------------------------------------------------
__global__ void k_apply_halt(int n, int *const *ist, const int *__restrict__ halt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ist[i][0] = ist[i][2] = halt[i];
}
__global__ void k_gather_read(int n, double *const *sc, int *const *ist, double *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[3 * i] = sc[i][0];
    out[3 * i + 1] = sc[i][1];
    out[3 * i + 2] = (double)ist[i][1];
}

}  // namespace bem

struct bem_group {
    int device = 0, n = 0, m = 0;
    double tol = -1.0;
    std::vector<bem_plan *> plans;
    std::vector<cudaStream_t> st;
    std::vector<cudaEvent_t> ev;
    cudaStream_t s0 = nullptr;
    cudaEvent_t e0 = nullptr;
    cudaGraphExec_t gstart = nullptr, gcycle = nullptr;
    long long kstart = 0, kcycle = 0;   // kernels per graph launch
    std::vector<const void *> captured; // members' Krylov bases the graphs were captured with
    bem::Arena arena;
    const void **d_chi = nullptr;
    void **d_x = nullptr;
    int *d_halt = nullptr;
    int **d_ist = nullptr;
    double **d_sc = nullptr;
    double *d_read = nullptr;
    void *h_pin = nullptr;              // pinned: chi ptrs, x ptrs, halt, read-back
    ~bem_group() {
        if (gstart) cudaGraphExecDestroy(gstart);
        if (gcycle) cudaGraphExecDestroy(gcycle);
        for (auto e : ev) if (e) cudaEventDestroy(e);
        for (auto s : st) if (s) cudaStreamDestroy(s);
        if (e0) cudaEventDestroy(e0);
        if (s0) cudaStreamDestroy(s0);
        if (h_pin) cudaFreeHost(h_pin);
    }
};

namespace bem {

// Captures one graph: (apply halts) -> per member on its stream
// [pointer slots, body] -> gather of (||b||, beta, steps) of every member.
template <class Body>
static int group_capture(bem_group *G, cudaGraphExec_t *out, long long *kernels, Body body) {
    if (*out) { cudaGraphExecDestroy(*out); *out = nullptr; }
    cudaGraph_t gr = nullptr;
    BEM_CUDA(cudaStreamBeginCapture(G->s0, cudaStreamCaptureModeThreadLocal));
    long long count = 0;
    tl_capture_count = &count;
    int rc = BEM_OK;
    (k_apply_halt<<<(G->n + 127) / 128, 128, 0, G->s0>>>(G->n, G->d_ist, G->d_halt), ::bem::count_launch());
    if (cudaEventRecord(G->e0, G->s0) != cudaSuccess) rc = BEM_ECUDA;
    for (int i = 0; i < G->n && rc == BEM_OK; i++) {
        bem_plan *P = G->plans[i];
        cudaStream_t s = G->st[i];
        if (cudaStreamWaitEvent(s, G->e0, 0) != cudaSuccess) { rc = BEM_ECUDA; break; }
        (k_set_ptrs_tab<<<1, 1, 0, s>>>((void **)P->gm_slot, G->d_chi, G->d_x, i), ::bem::count_launch());
        rc = body(P, s);
        if (rc == BEM_OK && (cudaEventRecord(G->ev[i], s) != cudaSuccess || cudaStreamWaitEvent(G->s0, G->ev[i], 0) != cudaSuccess))
            rc = BEM_ECUDA;
    }
    if (rc == BEM_OK)
        (k_gather_read<<<(G->n + 127) / 128, 128, 0, G->s0>>>(G->n, G->d_sc, G->d_ist, G->d_read), ::bem::count_launch());
    tl_capture_count = nullptr;
    cudaError_t e = cudaStreamEndCapture(G->s0, &gr);
    if (rc != BEM_OK || e != cudaSuccess) {
        if (gr) cudaGraphDestroy(gr);
        cudaGetLastError();
        if (rc == BEM_OK) rc = cuda_fail(e, "group capture", __FILE__, __LINE__);
        else set_error("group capture failed");
        return rc;
    }
    e = cudaGraphInstantiate(out, gr, 0);
    cudaGraphDestroy(gr);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate", __FILE__, __LINE__);
    *kernels = count;
    return BEM_OK;
}

const void *kernel_of_gmres() { return (const void *)k_backsolve<1>; }

}  // namespace bem

// ---------------------------------------------------------------------------
// Batch of concurrent solves (each on its own stream), for request serving
// ---------------------------------------------------------------------------
struct bem_batch {
    int device = 0, nslot = 0;
    std::vector<bem::GmSolver> slot;
    std::vector<int> used;              // 0 free, 1 active, 2 finished
    std::vector<cudaStream_t> streams;
    ~bem_batch() {
        for (auto &g : slot) bem::gm_release(g);
        for (auto s : streams)
            if (s) cudaStreamDestroy(s);
    }
};

using namespace bem;

extern "C" {

int bem_batch_create(bem_ctx *ctx, int max_slots, bem_batch **out) {
    if (!ctx || !out || max_slots < 1 || max_slots > 4096) {
        set_error("bem_batch_create: bad argument");
        return BEM_EINVAL;
    }
    *out = nullptr;
    BEM_CUDA(cudaSetDevice(ctx->device));
    bem_batch *b = new (std::nothrow) bem_batch;
    if (!b) { set_error("bem_batch_create: out of host memory"); return BEM_ENOMEM; }
    b->device = ctx->device;
    b->nslot = max_slots;
    b->slot.resize(max_slots);
    b->used.assign(max_slots, 0);
    b->streams.assign(max_slots, nullptr);
    for (int i = 0; i < max_slots; i++) {
        cudaError_t e = cudaStreamCreateWithFlags(&b->streams[i], cudaStreamNonBlocking);
        if (e != cudaSuccess) { delete b; return cuda_fail(e, "cudaStreamCreate", __FILE__, __LINE__); }
    }
    *out = b;
    return BEM_OK;
}

void bem_batch_destroy(bem_batch *b) {
    if (!b) return;
    cudaSetDevice(b->device);
    for (auto s : b->streams)
        if (s) cudaStreamSynchronize(s);
    delete b;
}

int bem_batch_submit(bem_batch *b, bem_plan *P, const void *chi_dev, void *phi_dev, const bem_solve_params *params,
                     int *slot_out) {
    if (!b || !P || !chi_dev || !phi_dev || !slot_out) { set_error("bem_batch_submit: NULL argument"); return BEM_EINVAL; }
    bem_solve_params sp;
    bem_solve_params_default(&sp);
    if (params) sp = *params;
    if (sp.method != BEM_GMRES) { set_error("bem_batch_submit: batched solves use GMRES"); return BEM_EINVAL; }
    int free_slot = -1;
    for (int i = 0; i < b->nslot; i++) {
        if (b->used[i] == 0 && free_slot < 0) free_slot = i;
        if (b->used[i] && b->slot[i].P == P) { set_error("bem_batch_submit: the plan already has a solve in the batch"); return BEM_EBUSY; }
    }
    if (free_slot < 0) { set_error("bem_batch_submit: no free slot"); return BEM_EBUSY; }
    BEM_CUDA(cudaSetDevice(b->device));
    GmSolver &g = b->slot[free_slot];
    gm_release(g);
    BEM_TRY(gm_init(g, P, (const double *)chi_dev, (double *)phi_dev, &sp, b->streams[free_slot]));
    b->used[free_slot] = 1;
    int rc = gm_run(g, false);
    P->fence.mark(g.s);
    if (rc != BEM_OK) { b->used[free_slot] = 2; g.status = rc; g.phase = 3; }
    *slot_out = free_slot;
    return rc;
}

int bem_batch_progress(bem_batch *b, int *n_active) {
    if (!b) { set_error("bem_batch_progress: NULL batch"); return BEM_EINVAL; }
    BEM_CUDA(cudaSetDevice(b->device));
    int act = 0, worst = BEM_OK;
    for (int i = 0; i < b->nslot; i++) {
        if (b->used[i] != 1) continue;
        GmSolver &g = b->slot[i];
        int rc = gm_run(g, false);
        if (rc != BEM_OK) { g.status = rc; g.phase = 3; worst = rc; }
        if (g.phase == 3) {
            b->used[i] = 2;
            g.P->fence.mark(g.s);
        } else {
            act++;
        }
    }
    if (n_active) *n_active = act;
    return worst;
}

int bem_batch_poll(bem_batch *b, int slot, int *done, bem_solve_info *info) {
    if (!b || slot < 0 || slot >= b->nslot || !done) { set_error("bem_batch_poll: bad argument"); return BEM_EINVAL; }
    *done = b->used[slot] == 2;
    if (*done && info) {
        const GmSolver &g = b->slot[slot];
        *info = bem_solve_info{g.iters, g.restarts, g.rel, g.status};
    }
    return BEM_OK;
}

int bem_batch_wait(bem_batch *b, int slot, double timeout_s) {
    if (!b || slot < 0 || slot >= b->nslot || b->used[slot] == 0) { set_error("bem_batch_wait: bad slot"); return BEM_EINVAL; }
    const auto t0 = std::chrono::steady_clock::now();
    while (b->used[slot] == 1) {
        BEM_TRY(bem_batch_progress(b, nullptr));
        if (b->used[slot] != 1) break;
        const double el = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        if (el > timeout_s) { set_error("bem_batch_wait: slot %d not finished after %g s", slot, timeout_s); return BEM_ETIMEOUT; }
        cudaEventSynchronize(gm_pending_event(b->slot[slot]));   // sleep until this slot's next step is done
    }
    return BEM_OK;
}

int bem_batch_release(bem_batch *b, int slot) {
    if (!b || slot < 0 || slot >= b->nslot) { set_error("bem_batch_release: bad slot"); return BEM_EINVAL; }
    if (b->used[slot] == 1) { set_error("bem_batch_release: slot %d is still running", slot); return BEM_EBUSY; }
    BEM_CUDA(cudaSetDevice(b->device));
    BEM_CUDA(cudaStreamSynchronize(b->streams[slot]));
    b->used[slot] = 0;
    b->slot[slot].P = nullptr;
    return BEM_OK;
}

void *bem_batch_stream(bem_batch *b, int slot) {
    if (!b || slot < 0 || slot >= b->nslot) return nullptr;
    return (void *)b->streams[slot];
}


int bem_group_create(bem_ctx *ctx, bem_plan *const *plans, int nplans, bem_group **out) {
    if (!ctx || !plans || !out || nplans < 1 || nplans > 65536) { set_error("bem_group_create: bad argument"); return BEM_EINVAL; }
    *out = nullptr;
    for (int i = 0; i < nplans; i++) {
        if (!plans[i]) { set_error("bem_group_create: plan %d is NULL", i); return BEM_EINVAL; }
        for (int j = 0; j < i; j++)
            if (plans[j] == plans[i]) { set_error("bem_group_create: plan %d appears twice", i); return BEM_EINVAL; }
    }
    BEM_CUDA(cudaSetDevice(ctx->device));
    bem_group *G = new (std::nothrow) bem_group;
    if (!G) { set_error("bem_group_create: out of host memory"); return BEM_ENOMEM; }
    G->device = ctx->device;
    G->n = nplans;
    G->plans.assign(plans, plans + nplans);
    G->st.assign(nplans, nullptr);
    G->ev.assign(nplans, nullptr);
    auto fail = [&](cudaError_t e, const char *what) { delete G; return cuda_fail(e, what, __FILE__, __LINE__); };
    cudaError_t e = cudaStreamCreateWithFlags(&G->s0, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->e0, cudaEventDisableTiming);
    for (int i = 0; i < nplans && e == cudaSuccess; i++) {
        e = cudaStreamCreateWithFlags(&G->st[i], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&G->ev[i], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) return fail(e, "bem_group_create");
    int rc = G->arena.alloc(&G->d_chi, nplans);
    if (rc == BEM_OK) rc = G->arena.alloc(&G->d_x, nplans);
    if (rc == BEM_OK) rc = G->arena.alloc(&G->d_halt, nplans);
    if (rc == BEM_OK) rc = G->arena.alloc(&G->d_ist, nplans);
    if (rc == BEM_OK) rc = G->arena.alloc(&G->d_sc, nplans);
    if (rc == BEM_OK) rc = G->arena.alloc(&G->d_read, 3 * (size_t)nplans);
    if (rc != BEM_OK) { delete G; return rc; }
    const size_t pin = sizeof(void *) * 2 * nplans + sizeof(int) * nplans + sizeof(double) * 3 * nplans + 64;
    e = cudaHostAlloc(&G->h_pin, pin, cudaHostAllocDefault);
    if (e != cudaSuccess) return fail(e, "cudaHostAlloc");
    *out = G;
    return BEM_OK;
}

void bem_group_destroy(bem_group *G) {
    if (!G) return;
    cudaSetDevice(G->device);
    cudaStreamSynchronize(G->s0);
    delete G;
}

int bem_group_solve(bem_group *G, const void *const *chis, void *const *phis, const bem_solve_params *params,
                    bem_solve_info *info, long long *launches) {
    if (!G || !chis || !phis) { set_error("bem_group_solve: NULL argument"); return BEM_EINVAL; }
    bem_solve_params sp;
    bem_solve_params_default(&sp);
    if (params) sp = *params;
    if (!(sp.tol > 0.0) || sp.max_iter < 1) { set_error("bem_group_solve: tol must be > 0 and max_iter >= 1"); return BEM_EINVAL; }
    if (sp.method != BEM_GMRES) { set_error("bem_group_solve: group solves use GMRES"); return BEM_EINVAL; }
    BEM_CUDA(cudaSetDevice(G->device));
    const int n = G->n;
    const void **h_chi = (const void **)G->h_pin;
    void **h_x = (void **)(h_chi + n);
    int *h_halt = (int *)(h_x + n);
    double *h_read = (double *)(((uintptr_t)(h_halt + n) + 15) & ~(uintptr_t)15);
    std::vector<GmSolver> gs(n);
    std::vector<int> ist_ok(n);
    std::vector<int *> ist(n);
    std::vector<double *> sc(n);
    for (int i = 0; i < n; i++) {
        bem_plan *P = G->plans[i];
        gs[i] = GmSolver{};
        gs[i].P = P;
        gs[i].sp = sp;
        gs[i].chi = (const double *)chis[i];
        gs[i].x = (double *)phis[i];
        gs[i].tol = gm_tol(P, sp.tol);
        BEM_TRY(gm_workspace(P, sp.restart));
        ist[i] = P->istate;
        sc[i] = P->scal;
        h_chi[i] = chis[i];
        h_x[i] = phis[i];
        h_halt[i] = chis[i] && phis[i] ? 0 : 1;          // a member without data sits this solve out
        gs[i].phase = h_halt[i] ? 3 : 0;
        gs[i].status = BEM_OK;
    }
    cudaStream_t s0 = G->s0;
    struct Mark {                          // a solve that ends with an error may leave work behind
        bem_group *G;
        bool done;
        ~Mark() {
            if (!done)
                for (bem_plan *P : G->plans) P->fence.mark(G->s0);
        }
    } mark{G, false};
    BEM_CUDA(cudaMemcpyAsync(G->d_ist, ist.data(), sizeof(int *) * n, cudaMemcpyHostToDevice, s0));
    BEM_CUDA(cudaMemcpyAsync(G->d_sc, sc.data(), sizeof(double *) * n, cudaMemcpyHostToDevice, s0));
    BEM_CUDA(cudaMemcpyAsync(G->d_chi, h_chi, sizeof(void *) * n, cudaMemcpyHostToDevice, s0));
    BEM_CUDA(cudaMemcpyAsync(G->d_x, h_x, sizeof(void *) * n, cudaMemcpyHostToDevice, s0));
    BEM_CUDA(cudaMemcpyAsync(G->d_halt, h_halt, sizeof(int) * n, cudaMemcpyHostToDevice, s0));
    BEM_CUDA(cudaStreamSynchronize(s0));   // tables in place (the pinned copies are rewritten below)
    // graphs are captured once per (restart, tolerance) and read pointers from the tables
    std::vector<const void *> bases(n);
    for (int i = 0; i < n; i++) bases[i] = G->plans[i]->V;
    if (!G->gstart || !G->gcycle || G->m != sp.restart || G->tol != sp.tol || G->captured != bases) {
        for (int i = 0; i < n; i++)
            BEM_CUDA(cudaMemsetAsync(G->plans[i]->istate, 0, sizeof(int) * 3, s0));
        BEM_CUDA(cudaStreamSynchronize(s0));
        BEM_TRY(group_capture(G, &G->gstart, &G->kstart, [&](bem_plan *P, cudaStream_t s) -> int {
            const double tol = gm_tol(P, sp.tol);
            if (P->green == BEM_HELMHOLTZ) {
                BEM_TRY(gm_k_start<2>(P, tol, s, true));
                return gm_k_residual<2>(P, s, true);
            }
            BEM_TRY(gm_k_start<1>(P, tol, s, true));
            return gm_k_residual<1>(P, s, true);
        }));
        BEM_TRY(group_capture(G, &G->gcycle, &G->kcycle, [&](bem_plan *P, cudaStream_t s) -> int {
            if (P->green == BEM_HELMHOLTZ) {
                BEM_TRY(gm_k_cycle<2>(P, P->gm_restart, s, true));
                return gm_k_residual<2>(P, s, true);
            }
            BEM_TRY(gm_k_cycle<1>(P, P->gm_restart, s, true));
            return gm_k_residual<1>(P, s, true);
        }));
        G->m = sp.restart;
        G->tol = sp.tol;
        G->captured = bases;
    }
    long long nlaunch = 0;
    auto launch = [&](cudaGraphExec_t ge, long long k) -> int {
        BEM_CUDA(cudaMemcpyAsync(G->d_halt, h_halt, sizeof(int) * n, cudaMemcpyHostToDevice, s0));
        BEM_CUDA(cudaGraphLaunch(ge, s0));
        count_launch(k);
        nlaunch += k;
        BEM_CUDA(cudaMemcpyAsync(h_read, G->d_read, sizeof(double) * 3 * n, cudaMemcpyDeviceToHost, s0));
        BEM_CUDA(cudaStreamSynchronize(s0));
        return BEM_OK;
    };
    BEM_TRY(launch(G->gstart, G->kstart));
    int active = 0;
    for (int i = 0; i < n; i++) {
        if (gs[i].phase == 3) continue;
        if (gm_after_residual(gs[i], h_read[3 * i], h_read[3 * i + 1])) { gs[i].phase = 3; h_halt[i] = 1; }
        else active++;
    }
    while (active > 0) {
        BEM_TRY(launch(G->gcycle, G->kcycle));
        active = 0;
        for (int i = 0; i < n; i++) {
            if (gs[i].phase == 3) continue;
            const int steps = (int)h_read[3 * i + 2];
            gs[i].iters += steps;
            if (steps == 0) {
                gs[i].status = BEM_ENOCONV;
                gs[i].phase = 3;
            } else if (gm_after_residual(gs[i], h_read[3 * i], h_read[3 * i + 1])) {
                gs[i].phase = 3;
            }
            if (gs[i].phase == 3) h_halt[i] = 1;
            else active++;
        }
    }
    int worst = BEM_OK;
    for (int i = 0; i < n; i++) {
        if (info) info[i] = bem_solve_info{gs[i].iters, gs[i].restarts, gs[i].rel, gs[i].status};
        if (gs[i].status == BEM_ENOCONV) worst = BEM_ENOCONV;
    }
    if (launches) *launches = nlaunch;
    mark.done = true;                      // (synchronised after every launch)
    return worst;
}

}  // extern "C"

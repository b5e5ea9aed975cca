// CPR two-stage preconditioner (Section "CPR-like Preconditioners").
//
// Pressure stage: quasi-IMPES decoupling (named in the numerical experiments;
// diagonal reading: with D = A_cc, w_c = (1, -D01/D11, -D02/D22)), the
// restriction Pi_r f = (w_c . f_c)_c, and the pressure matrix
// (A_pp)_cn = sum_r w_c[r] A_cn[r][0] (the pressure column of the weighted
// block row), a seven-point scalar stencil.  It is solved approximately by
// one geometric-multigrid V-cycle standing in for the paper's AMG (Section
// "Algebraic Multigrid Methods": R = P^T, A_{l+1} = R A_l P, pre-smoother,
// residual, restriction, recursion, prolongation, post-smoother, exact
// coarsest solve):
//   * P is piecewise constant on 2x2x2 boxes (coarse dims ceil(d/2)), so the
//     Galerkin operator stays seven-point: entry (I, J) sums the fine
//     couplings from box I to box J, couplings inside a box add to I's centre;
//   * smoothing is red-black Gauss-Seidel, colour (i+j+k) mod 2, red then
//     black before the recursion and black then red after it;
//   * the coarsest level (at most gmg_max_coarse cells) is solved with its
//     explicit inverse, computed at setup from a partial-pivoting LU.
// Full stage (CPR-PF, two-stage multiplicative): x = Pi_p p; r = f - A x;
// x = x + ILU0^{-1} r, with Pi_p p = (p_c, 0, 0)_c.
//
// Stencil storage: a7[s][c] (slot-major, coalesced), slots -z, -y, -x,
// centre, +x, +y, +z; absent faces hold 0.
#include <algorithm>

#include "common.cuh"

namespace rsv {
namespace {

__device__ __forceinline__ bool gated(const int *done) { return done && *(volatile const int *)done; }

struct G3 {
    int nx, ny, nz;
    __host__ __device__ int64_t n() const { return (int64_t)nx * ny * nz; }
};

__device__ __forceinline__ void ijk(int64_t c, G3 g, int &i, int &j, int &k) {
    i = (int)(c % g.nx);
    j = (int)((c / g.nx) % g.ny);
    k = (int)(c / ((int64_t)g.nx * g.ny));
}

// The divisors of the smoother's index arithmetic, built on the host (Div32): ny and the
// colour slots of a grid row, ceil(nx / 2) (a level has < 2^31 cells).
struct G3Div {
    Div32 dy, dh;
    static G3Div of(const G3 &g) { return {Div32::of(g.ny), Div32::of((g.nx + 1) / 2)}; }
};


__constant__ int kDI[7] = {0, 0, -1, 0, 1, 0, 0};
__constant__ int kDJ[7] = {0, -1, 0, 0, 0, 1, 0};
__constant__ int kDK[7] = {-1, 0, 0, 0, 0, 0, 1};

__device__ __forceinline__ int slot_of(int di, int dj, int dk) {
    return dk < 0 ? 0 : dj < 0 ? 1 : di < 0 ? 2 : di > 0 ? 4 : dj > 0 ? 5 : dk > 0 ? 6 : 3;
}

// Quasi-IMPES weights and the pressure stencil of the block row of cell c.
template <typename Tv>
__global__ void qi_setup_kernel(G3 g, const int32_t *__restrict__ rp, const Tv *__restrict__ v, int decoupling,
                                const double *__restrict__ acc, double *__restrict__ w, double *__restrict__ a7,
                                int *status) {
    const int64_t n = g.n();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= n) return;
    int i, j, k;
    ijk(c, g, i, j, k);
    const bool has[7] = {k > 0, j > 0, i > 0, true, i < g.nx - 1, j < g.ny - 1, k < g.nz - 1};
    int slot_pos[7], q = 0;
    for (int s = 0; s < 7; ++s) slot_pos[s] = has[s] ? q++ : -1;
    const Tv *dv = v + 9 * ((int64_t)rp[c] + slot_pos[3]);
    double d[9];
    if (decoupling == 2)  // true-IMPES: the cell's accumulation block instead of A's diagonal block
        for (int q = 0; q < 9; ++q) d[q] = acc[9 * c + q];
    else
        for (int q = 0; q < 9; ++q) d[q] = exact_double(dv[q]);
    double w0, w1, w2;
    if (decoupling == 1 || decoupling == 2) {
        // ABF / true-IMPES: the first row of D^{-1} = adj(D) / det(D), from the cofactors of D's first column
        const double c0 = d[4] * d[8] - d[5] * d[7];
        const double det = d[0] * c0 + d[1] * (d[5] * d[6] - d[3] * d[8]) + d[2] * (d[3] * d[7] - d[4] * d[6]);
        if (!(fabs(det) > 1e-300)) {
            atomicCAS(status, 0, (int)RSV_ESINGULAR);
            return;
        }
        w0 = c0 / det;
        w1 = (d[2] * d[7] - d[1] * d[8]) / det;
        w2 = (d[1] * d[5] - d[2] * d[4]) / det;
    } else {
        // quasi-IMPES: keep the pressure equation, cancel the diagonal coupling of the other two
        if (!(fabs(d[4]) > 1e-300) || !(fabs(d[8]) > 1e-300)) {
            atomicCAS(status, 0, (int)RSV_ESINGULAR);
            return;
        }
        w0 = 1.0;
        w1 = -d[1] / d[4];
        w2 = -d[2] / d[8];
    }
    w[3 * c] = w0;
    w[3 * c + 1] = w1;
    w[3 * c + 2] = w2;
    for (int s = 0; s < 7; ++s) {
        double val = 0.0;
        if (has[s]) {
            const Tv *blk = v + 9 * ((int64_t)rp[c] + slot_pos[s]);
            val = w0 * exact_double(blk[0]) + w1 * exact_double(blk[3]) + w2 * exact_double(blk[6]);
        }
        a7[(int64_t)s * n + c] = val;
    }
}

// Galerkin coarse operator P^T A P for piecewise-constant P: one thread per
// coarse cell sums the couplings of its children (children and slots in a
// fixed order, so the result is deterministic).
__global__ void gmg_coarsen_kernel(G3 f, const double *__restrict__ af, G3 cg, double *__restrict__ ac) {
    const int64_t nc = cg.n(), nf = f.n();
    const int64_t C = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (C >= nc) return;
    int I, J, K;
    ijk(C, cg, I, J, K);
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int dk = 0; dk < 2; ++dk)
        for (int dj = 0; dj < 2; ++dj)
            for (int di = 0; di < 2; ++di) {
                const int i = 2 * I + di, j = 2 * J + dj, k = 2 * K + dk;
                if (i >= f.nx || j >= f.ny || k >= f.nz) continue;
                const int64_t c = (int64_t)k * f.nx * f.ny + (int64_t)j * f.nx + i;
                for (int s = 0; s < 7; ++s) {
                    const int ii = i + kDI[s], jj = j + kDJ[s], kk = k + kDK[s];
                    if (ii < 0 || jj < 0 || kk < 0 || ii >= f.nx || jj >= f.ny || kk >= f.nz) continue;
                    acc[slot_of(ii / 2 - I, jj / 2 - J, kk / 2 - K)] += af[(int64_t)s * nf + c];
                }
            }
    for (int s = 0; s < 7; ++s) ac[(int64_t)s * nc + C] = acc[s];
}

__global__ void cast_stencil(int64_t n, const double *__restrict__ a, float *__restrict__ b) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = round_float(a[i]);
}

// Dense matrix of the coarsest stencil, row-major n x n; M is cleared before.
__global__ void coarse_dense_kernel(G3 g, const double *__restrict__ a7, double *__restrict__ M) {
    const int64_t n = g.n();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= n) return;
    int i, j, k;
    ijk(c, g, i, j, k);
    for (int s = 0; s < 7; ++s) {
        const int ii = i + kDI[s], jj = j + kDJ[s], kk = k + kDK[s];
        if (ii < 0 || jj < 0 || kk < 0 || ii >= g.nx || jj >= g.ny || kk >= g.nz) continue;
        M[c * n + (int64_t)kk * g.nx * g.ny + (int64_t)jj * g.nx + ii] = a7[(int64_t)s * n + c];
    }
}

// The coarsest level's inverse from an LU factorisation with partial pivoting, kLuB columns (a panel) at a time, and
// triangular solves for the unit vectors.  Every entry sees the operations of the plain row-by-row elimination in that
// order (a - l u as one fused operation, l a true quotient), so neither the rounding nor which matrices are found
// singular depends on the panels.  A Gauss-Jordan inverse rounds differently, and with pivot rows scaled by rounded
// reciprocals an exactly singular operator can pass.
// FP64 arithmetic bounds it: one SM adds and multiplies 1.7 values per clock, so only the panel's own columns stay in
// one CTA (lu_panel); the other columns are updated by the whole chip (lu_update), and columns of the inverse are solved
// for side by side (lu_columns), bound by the chain of 2 n steps, n of them with a division.
// A one-level CPR setup of 8x8x4 cells (n = 256) takes 0.86 ms and of 10x10x5 2.1 ms; with elimination and solves by
// single CTAs 4.6 and 22.6 ms, with Gauss-Jordan 0.58 and 1.6 ms.
constexpr int kLuB = 8;
constexpr int kLuRows = 1024;  // rows that one thread each of the panel CTA holds in registers

// The largest key of the warp and the smallest row that has it (keys: bits of |value|, which order like the
// values; integer reductions keep the search off the FP64 pipe).
__device__ __forceinline__ void warp_largest(unsigned long long &key, int &at) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32) == hi ? (unsigned)key : 0u);
    const unsigned long long best = (unsigned long long)hi << 32 | lo;
    at = (int)__reduce_min_sync(0xffffffffu, key == best ? (unsigned)at : 0x7fffffffu);
    key = best;
}
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// One panel: elimination steps k0 .. k0 + kLuB - 1 on those columns of the n x n matrix A, rows k0 and below (m of them).
// Thread r holds row k0 + r of the panel in registers.  Q [m][kLuB]: the panel afterwards, L below the diagonal and U
// on and above it.  perm[i], i >= k0: the row of A that the pivoting moved to row i.  Largest |pivot| first, the smallest row
// on ties; |pivot| <= 1e-300 reports RSV_ESINGULAR.
__global__ void __launch_bounds__(kLuRows) lu_panel(int n, int k0, const double *__restrict__ A, double *__restrict__ Q,
                                                    int *__restrict__ perm, int *status) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    __shared__ unsigned long long wmax[32];
    __shared__ double prow[kLuB], trow[kLuB];
    __shared__ int widx[32], sidx[2];
    const int r = threadIdx.x, lane = r & 31, warp = r >> 5, nw = (int)(blockDim.x >> 5);
    const int m = n - k0, nk = min(kLuB, m);
    double a[kLuB];
#pragma unroll
    for (int c = 0; c < kLuB; ++c) a[c] = r < m && c < nk ? A[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
    int src = k0 + r;
#pragma unroll
    for (int t = 0; t < kLuB; ++t) {
        if (t >= nk) break;
        const bool in = r >= t && r < m;
        unsigned long long key = in ? abs_bits(a[t]) : 0ull;
        int at = in ? r : m;  // m: no candidate, behind every row of the same key
        warp_largest(key, at);
        if (lane == 0) {
            wmax[warp] = key;
            widx[warp] = at;
        }
        __syncthreads();
        key = lane < nw ? wmax[lane] : 0ull;
        at = lane < nw ? widx[lane] : m;
        warp_largest(key, at);
        const int p = at;
        if (r == t) {
#pragma unroll
            for (int c = 0; c < kLuB; ++c) trow[c] = a[c];
            sidx[0] = src;
            if (!(__longlong_as_double((long long)key) > 1e-300)) atomicCAS(status, 0, (int)RSV_ESINGULAR);
        }
        if (r == p) {
#pragma unroll
            for (int c = 0; c < kLuB; ++c) prow[c] = a[c];
            sidx[1] = src;
        }
        __syncthreads();
        if (r == p) {
#pragma unroll
            for (int c = 0; c < kLuB; ++c) a[c] = trow[c];
            src = sidx[0];
        }
        if (r == t) {
#pragma unroll
            for (int c = 0; c < kLuB; ++c) a[c] = prow[c];
            src = sidx[1];
        } else if (in) {
            const double l = a[t] / prow[t];
            a[t] = l;
#pragma unroll
            for (int c = t + 1; c < kLuB; ++c) a[c] = fma(-l, prow[c], a[c]);
        }
    }
    if (r < m) {
#pragma unroll
        for (int c = 0; c < kLuB; ++c) Q[r * kLuB + c] = a[c];
        perm[k0 + r] = src;
    }
}

// The same for more rows than a CTA has threads (few levels on a large grid): the panel lives in Q, the row
// order in perm.
__global__ void __launch_bounds__(kLuRows) lu_panel_large(int n, int k0, const double *__restrict__ A, double *Q, int *perm,
                                                          int *status) {
    pdl_wait();
    pdl_trigger();
    __shared__ unsigned long long wmax[32];
    __shared__ int widx[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = n - k0, nk = min(kLuB, m);
    for (int r = threadIdx.x; r < m; r += kLuRows) {
        for (int c = 0; c < kLuB; ++c) Q[(int64_t)r * kLuB + c] = c < nk ? A[(int64_t)(k0 + r) * n + k0 + c] : 0.0;
        perm[k0 + r] = k0 + r;
    }
    __syncthreads();
    for (int t = 0; t < nk; ++t) {
        unsigned long long key = 0ull;
        int at = m;
        for (int r = t + threadIdx.x; r < m; r += kLuRows) {
            const unsigned long long v = abs_bits(Q[(int64_t)r * kLuB + t]);
            if (at == m || v > key) {
                key = v;
                at = r;
            }
        }
        warp_largest(key, at);
        if (lane == 0) {
            wmax[warp] = key;
            widx[warp] = at;
        }
        __syncthreads();
        key = wmax[lane];
        at = widx[lane];
        warp_largest(key, at);
        const int p = at;
        if (threadIdx.x == 0 && !(__longlong_as_double((long long)key) > 1e-300)) atomicCAS(status, 0, (int)RSV_ESINGULAR);
        if (threadIdx.x < kLuB && p != t) {
            const int c = threadIdx.x;
            const double v = Q[(int64_t)p * kLuB + c];
            Q[(int64_t)p * kLuB + c] = Q[t * kLuB + c];
            Q[t * kLuB + c] = v;
            if (c == 0) {
                const int sp = perm[k0 + p];
                perm[k0 + p] = perm[k0 + t];
                perm[k0 + t] = sp;
            }
        }
        __syncthreads();
        for (int r = t + 1 + threadIdx.x; r < m; r += kLuRows) {
            double *q = Q + (int64_t)r * kLuB;
            const double l = q[t] / Q[t * kLuB + t];
            q[t] = l;
            for (int c = t + 1; c < nk; ++c) q[c] = fma(-l, Q[t * kLuB + c], q[c]);
        }
        __syncthreads();
    }
}

// B = A with the panel's rows moved, its columns from Q, and the columns right of it updated.  A CTA takes 16 rows of 32
// columns; one warp forms the columns' part of U (28 dependent FP64 operations), which the others' rows need.  Tracks the
// row order (order_out = order_in through perm).  The last panel writes B transposed.
__global__ void __launch_bounds__(256) lu_update(int n, int k0, const double *__restrict__ A, const double *__restrict__ Q,
                                                 const int *__restrict__ perm, const int *__restrict__ order_in,
                                                 int *__restrict__ order_out, double *__restrict__ B) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    __shared__ double u[kLuB][32];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, i0 = blockIdx.y * 16, j = blockIdx.x * 32 + tx;
    const int k1 = min(k0 + kLuB, n);
    const bool right = j >= k1 && j < n;  // then the panel is a full one
    double v[2];
    int src[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = i0 + ty + 8 * h;
        src[h] = i < k0 || i >= n ? i : perm[i];
        v[h] = i < n && j < n ? A[(int64_t)src[h] * n + j] : 0.0;
    }
    if (ty == 0 && right && i0 + 16 > k0) {
        double w[kLuB];
#pragma unroll
        for (int t = 0; t < kLuB; ++t) w[t] = A[(int64_t)perm[k0 + t] * n + j];
#pragma unroll
        for (int t = 0; t < kLuB; ++t) {
#pragma unroll
            for (int s = 0; s < t; ++s) w[t] = fma(-Q[t * kLuB + s], w[s], w[t]);
            u[t][tx] = w[t];
        }
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = i0 + ty + 8 * h;
        if (i >= n || j >= n) continue;
        if (j == 0) order_out[i] = order_in ? order_in[src[h]] : src[h];
        double r = v[h];
        if (i >= k0 && j >= k0) {
            const double *l = Q + (int64_t)(i - k0) * kLuB;
            if (j < k1) {
                r = l[j - k0];
            } else if (i < k1) {
                r = u[i - k0][tx];
            } else {
#pragma unroll
                for (int t = 0; t < kLuB; ++t) r = fma(-l[t], u[t][tx], r);
            }
        }
        B[k1 < n ? (int64_t)i * n + j : (int64_t)j * n + i] = r;
    }
}

// Columns j = C b .. C b + C - 1 of the inverse by CTA b: L U x = P e_j, T the transpose of L and U.  At most kLuRows rows, x
// in registers (row threadIdx.x + q blockDim.x at q); a step's x_k travel through shared memory, and T is read four
// steps ahead.  The quotients of a step are formed by one lane each: a division in one lane holds the FP64 pipe as
// long as one in all of them.
constexpr int kLuOwn = 4;
template <int C>
__global__ void __launch_bounds__(kLuRows / kLuOwn, C == 1 ? 2 : 1) lu_columns(int n, const double *__restrict__ T,
                                                               const int *__restrict__ order, double *__restrict__ Minv) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    __shared__ double xk[2][C];
    __shared__ int start;  // x is zero above its unit entries: the first group of four steps that has one
    const int j0 = blockIdx.x * C, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    double x[kLuOwn][C], now[4][kLuOwn], next[4][kLuOwn], dnow[4], dnext[4];
    if (tid == 0) start = n;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kLuOwn; ++q) {
        const int i = tid + q * nt, at = i < n ? order[i] - j0 : -1;
#pragma unroll
        for (int c = 0; c < C; ++c) x[q][c] = at == c ? 1.0 : 0.0;
        if (at >= 0 && at < C) atomicMin(&start, i & ~3);
    }
    __syncthreads();
    // columns k .. k + 3 of T, rows below (or above) the diagonal only
    auto fetch = [&](int k, bool below, double(&l)[4][kLuOwn], double(&d)[4]) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const bool in = k >= 0 && k + s < n;
            d[s] = in && !below ? T[(int64_t)(k + s) * n + k + s] : 1.0;
#pragma unroll
            for (int q = 0; q < kLuOwn; ++q) {
                const int i = tid + q * nt;
                l[s][q] = in && (below ? i > k + s && i < n : i < k + s) ? T[(int64_t)(k + s) * n + i] : 0.0;
            }
        }
    };
    // the unit lower triangle
    fetch(start, true, next, dnext);
#pragma unroll
    for (int o = 0; o < kLuOwn; ++o)
        for (int k = max(o * nt, start); k < min((o + 1) * nt, n); k += 4) {
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int q = 0; q < kLuOwn; ++q) now[s][q] = next[s][q];
            fetch(k + 4, true, next, dnext);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (k + s >= n) break;
                if (tid == k + s - o * nt)
#pragma unroll
                    for (int c = 0; c < C; ++c) xk[s & 1][c] = x[o][c];
                __syncthreads();
#pragma unroll
                for (int q = o; q < kLuOwn; ++q) {
                    const int i = tid + q * nt;
                    if (i > k + s && i < n)
#pragma unroll
                        for (int c = 0; c < C; ++c) x[q][c] = fma(-now[s][q], xk[s & 1][c], x[q][c]);
                }
            }
        }
    __syncthreads();
    // the upper triangle
    const int last = (n - 1) / 4 * 4;
    fetch(last, false, next, dnext);
#pragma unroll
    for (int o = kLuOwn - 1; o >= 0; --o)
        for (int k = min((o + 1) * nt - 4, last); k >= o * nt; k -= 4) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                dnow[s] = dnext[s];
#pragma unroll
                for (int q = 0; q < kLuOwn; ++q) now[s][q] = next[s][q];
            }
            fetch(k - 4, false, next, dnext);
#pragma unroll
            for (int s = 3; s >= 0; --s) {
                if (k + s >= n) continue;
                const int at = k + s - o * nt;  // the thread that owns row k + s
                if (C == 1) {
                    if (tid == at) xk[s & 1][0] = x[o][0] /= dnow[s];
                } else if (warp == at >> 5) {
                    double v = 0.0;
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const double t = __shfl_sync(0xffffffffu, x[o][c], at & 31);
                        if (lane == c) v = t;
                    }
                    if (lane < C) xk[s & 1][lane] = v / dnow[s];
                }
                __syncthreads();
                if (C > 1 && tid == at)
#pragma unroll
                    for (int c = 0; c < C; ++c) x[o][c] = xk[s & 1][c];
#pragma unroll
                for (int q = 0; q <= o; ++q)
                    if (tid + q * nt < k + s)
#pragma unroll
                        for (int c = 0; c < C; ++c) x[q][c] = fma(-now[s][q], xk[s & 1][c], x[q][c]);
            }
        }
#pragma unroll
    for (int q = 0; q < kLuOwn; ++q) {
        const int i = tid + q * nt;
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (i < n && j0 + c < n) Minv[(int64_t)i * n + j0 + c] = x[q][c];
    }
}

// The same for more rows: x in row j of `work`.
__global__ void __launch_bounds__(256) lu_columns_large(int n, const double *__restrict__ T, const int *__restrict__ order,
                                                        double *__restrict__ Minv, double *work) {
    pdl_wait();
    pdl_trigger();
    const int j = blockIdx.x;
    double *x = work + (int64_t)j * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) x[i] = order[i] == j ? 1.0 : 0.0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        const double xk = x[k];
        for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) x[i] = fma(-T[(int64_t)k * n + i], xk, x[i]);
        __syncthreads();
    }
    for (int k = n - 1; k >= 0; --k) {
        if (threadIdx.x == 0) x[k] /= T[(int64_t)k * n + k];
        __syncthreads();
        const double xk = x[k];
        for (int i = threadIdx.x; i < k; i += blockDim.x) x[i] = fma(-T[(int64_t)k * n + i], xk, x[i]);
        __syncthreads();
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) Minv[(int64_t)i * n + j] = x[i];
}

// Minv = inverse of the n x n matrix in `dense` (overwritten).  work: n (n + kLuB) doubles; index: 3 n ints.
cudaError_t coarse_inverse(cudaStream_t st, int n, double *dense, double *work, int *index, double *Minv, int *status) {
    double *X[2] = {dense, work}, *Q = work + (int64_t)n * n;
    int *perm = index, *order[2] = {index + n, index + 2 * n};
    cudaError_t e = cudaSuccess;
    int q = 0;
    for (int k0 = 0; k0 < n && e == cudaSuccess; k0 += kLuB, q ^= 1) {
        const int m = n - k0;
        count_launches(2);
        e = m <= kLuRows ? launch_pdl(lu_panel, dim3(1), dim3((m + 31) / 32 * 32), 0, st, n, k0, X[q], Q, perm, status)
                         : launch_pdl(lu_panel_large, dim3(1), dim3(kLuRows), 0, st, n, k0, X[q], Q, perm, status);
        if (e == cudaSuccess)
            e = launch_pdl(lu_update, dim3((n + 31) / 32, (n + 15) / 16), dim3(256), 0, st, n, k0, X[q], Q, perm,
                           k0 ? order[q] : nullptr, order[q ^ 1], X[q ^ 1]);
    }
    if (e != cudaSuccess) return e;
    count_launches(1);
    if (n > kLuRows)
        return launch_pdl(lu_columns_large, dim3(n), dim3(256), 0, st, n, X[q], order[q], Minv, X[q ^ 1]);
    // two CTAs are resident per SM with one column each, one with four: as many columns as one wave takes
    const dim3 block(std::min((n + 31) / 32 * 32, kLuRows / kLuOwn));
    return n <= 2 * 152 ? launch_pdl(lu_columns<1>, dim3(n), block, 0, st, n, X[q], order[q], Minv)
                        : launch_pdl(lu_columns<4>, dim3((n + 3) / 4), block, 0, st, n, X[q], order[q], Minv);
}

// x = Minv b (one warp per row), b and x in T, arithmetic in FP64.
template <typename T>
__global__ void coarse_apply_kernel(int n, const double *__restrict__ Minv, const T *__restrict__ b, T *__restrict__ x,
                                    const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    double s = 0.0;
    for (int q = lane; q < n; q += 32) s += Minv[(int64_t)row * n + q] * (double)b[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) x[row] = (T)s;
}

// Colour-split position of the cell (2 h + parity, j, k) of colour `colour` in grid row
// row = j + ny k: the row's red cells first (i ascending), then its black cells.  A row
// starting with a red cell ((j + k) even) holds ceil(nx / 2) red cells, else floor(nx / 2).
__device__ __forceinline__ int64_t split_pos(G3 g, int64_t row, int j, int k, int h, int colour) {
    const int nred = (g.nx + 1 - ((j + k) & 1)) >> 1;
    return row * g.nx + (colour == 0 ? h : nred + h);
}

// a7s[s][split_pos(c)] = a7[s][c] (converted to T).
template <typename T>
__global__ void split_stencil_kernel(G3 g, const double *__restrict__ a7, T *__restrict__ a7s) {
    const int64_t n = g.n();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= n) return;
    int i, j, k;
    ijk(c, g, i, j, k);
    const int64_t ps = split_pos(g, c / g.nx, j, k, i >> 1, (i + j + k) & 1);
    for (int s = 0; s < 7; ++s) a7s[(int64_t)s * n + ps] = (T)a7[(int64_t)s * n + c];
}

// One red-black Gauss-Seidel half sweep over the cells of colour (i+j+k) mod 2;
// one thread per cell of that colour (a row of nx cells holds ceil(nx/2) or
// floor(nx/2) of them).  Cells of one colour couple only to the other colour,
// so the update x_c = (b_c - sum_n a_cn x_n) / a_cc reads only cells this
// launch does not write.  MODE selects what the neighbours hold:
//   0  x as stored;
//   1  zero (the first half sweep of a V-cycle level from a zero guess:
//      x_c = b_c / a_cc, and x need not be cleared first);
//   2  x + P xc (the first half sweep after the coarse correction: the
//      prolongation x += P xc is applied to the neighbours on the fly; this
//      colour's own cells are overwritten, so the correction need not be
//      stored for them, and the other colour's cells are overwritten by the
//      next half sweep, which reads only this colour).
// Each variant rounds exactly as the separate zeroing / prolongation kernels
// followed by the plain half sweep.
//
// The coefficients come from a colour-split copy a7s (see split_pos): the cells
// of one colour in a grid row are contiguous there, so a half sweep reads
// only its own colour's coefficients, coalesced.
// Each thread takes CELLS cells of the colour, blockDim.x colour slots apart (coalesced per
// slot), and issues all their loads before any store: same-colour cells never read one
// another.  On large levels the loads in flight per thread, not bandwidth, bound the
// one-cell form (finest level of 256x256x128: 47 us per half sweep, 38 us with four cells);
// small levels and the prolongating sweep (MODE 2) keep one cell per thread.
template <typename T, int MODE, int CELLS>
__global__ void rbgs_kernel(G3 g, G3Div gd, const T *__restrict__ a7s, const T *__restrict__ b, T *__restrict__ x,
                            int colour, const T *__restrict__ xc, G3 cg, const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int64_t n = g.n();
    const int half = (g.nx + 1) >> 1;
    const int rows = g.ny * g.nz;
    const int64_t sy = g.nx, sz = (int64_t)g.nx * g.ny;
    T res[CELLS];
    int64_t cell[CELLS];
#pragma unroll
    for (int u = 0; u < CELLS; ++u) {
        cell[u] = -1;
        const int q = (blockIdx.x * CELLS + u) * blockDim.x + threadIdx.x;
        const int row = gd.dh(q);  // row = j + ny k
        if (row >= rows) continue;
        const int k = gd.dy(row), j = row - k * g.ny;
        const int h = q - row * half;
        const int i = 2 * h + ((colour + j + k) & 1);
        if (i >= g.nx) continue;
        const int64_t c = (int64_t)row * g.nx + i;
        const T *a7 = a7s + split_pos(g, row, j, k, h, colour);  // slot s at a7[s * n]
        T s = b[c];
        if (MODE != 1) {
            auto nbr = [&](int64_t o, int ii, int jj, int kk) -> T {
                T v = x[o];
                if (MODE == 2) v += xc[(int64_t)(kk >> 1) * cg.nx * cg.ny + (int64_t)(jj >> 1) * cg.nx + (ii >> 1)];
                return v;
            };
            if (k > 0) s -= a7[0 * n] * nbr(c - sz, i, j, k - 1);
            if (j > 0) s -= a7[1 * n] * nbr(c - sy, i, j - 1, k);
            if (i > 0) s -= a7[2 * n] * nbr(c - 1, i - 1, j, k);
            if (i < g.nx - 1) s -= a7[4 * n] * nbr(c + 1, i + 1, j, k);
            if (j < g.ny - 1) s -= a7[5 * n] * nbr(c + sy, i, j + 1, k);
            if (k < g.nz - 1) s -= a7[6 * n] * nbr(c + sz, i, j, k + 1);
        }
        res[u] = s / a7[3 * n];
        cell[u] = c;
    }
#pragma unroll
    for (int u = 0; u < CELLS; ++u)
        if (cell[u] >= 0) x[cell[u]] = res[u];
}

// b_coarse[C] = sum over the children f of C of (b_f - (A x)_f): residual and
// restriction R = P^T fused.
template <typename T>
__global__ void residual_restrict_kernel(G3 f, const T *__restrict__ a7, const T *__restrict__ b,
                                         const T *__restrict__ x, G3 cg, T *__restrict__ bc, const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int64_t nc = cg.n(), n = f.n();
    const int64_t C = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (C >= nc) return;
    int I, J, K;
    ijk(C, cg, I, J, K);
    const int64_t sy = f.nx, sz = (int64_t)f.nx * f.ny;
    T acc = T(0);
    for (int dk = 0; dk < 2; ++dk)
        for (int dj = 0; dj < 2; ++dj)
            for (int di = 0; di < 2; ++di) {
                const int i = 2 * I + di, j = 2 * J + dj, k = 2 * K + dk;
                if (i >= f.nx || j >= f.ny || k >= f.nz) continue;
                const int64_t c = (int64_t)k * sz + (int64_t)j * sy + i;
                T r = b[c] - a7[3 * n + c] * x[c];
                if (k > 0) r -= a7[0 * n + c] * x[c - sz];
                if (j > 0) r -= a7[1 * n + c] * x[c - sy];
                if (i > 0) r -= a7[2 * n + c] * x[c - 1];
                if (i < f.nx - 1) r -= a7[4 * n + c] * x[c + 1];
                if (j < f.ny - 1) r -= a7[5 * n + c] * x[c + sy];
                if (k < f.nz - 1) r -= a7[6 * n + c] * x[c + sz];
                acc += r;
            }
    bc[C] = acc;
}

// x_fine += P x_coarse (injection of the box value).
template <typename T>
__global__ void prolong_add_kernel(G3 f, const T *__restrict__ xc, G3 cg, T *__restrict__ x, const int *done) {
    if (gated(done)) return;
    const int64_t n = f.n();
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= n) return;
    int i, j, k;
    ijk(c, f, i, j, k);
    x[c] += xc[(int64_t)(k / 2) * cg.nx * cg.ny + (int64_t)(j / 2) * cg.nx + i / 2];
}

// x += P xc on a large level, four consecutive cells of a grid row per thread (all loads
// before the stores).  dq divides by the row's quads, ceil(nx / 4); dy by ny.  Each cell's
// sum is the one prolong_add_kernel forms.
template <typename T>
__global__ void prolong_add_rows(G3 f, Div32 dq, Div32 dy, const T *__restrict__ xc, G3 cg, T *__restrict__ x,
                                 const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int quads = (f.nx + 3) >> 2;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const int row = dq(q);
    if (row >= f.ny * f.nz) return;
    const int k = dy(row), j = row - k * f.ny, i0 = 4 * (q - row * quads);
    T *xr = x + (int64_t)row * f.nx;
    const T *cr = xc + (int64_t)(k >> 1) * cg.nx * cg.ny + (int64_t)(j >> 1) * cg.nx;
    if constexpr (sizeof(T) == 4) {
        if ((f.nx & 3) == 0 && (((uintptr_t)x) & 15) == 0) {  // one 16-byte access per quad
            float4 v = *reinterpret_cast<const float4 *>(xr + i0);
            const T p0 = cr[i0 >> 1], p1 = cr[(i0 >> 1) + 1];
            v.x += p0;
            v.y += p0;
            v.z += p1;
            v.w += p1;
            *reinterpret_cast<float4 *>(xr + i0) = v;
            return;
        }
    }
    T v[4], p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (i0 + u < f.nx) {
            v[u] = xr[i0 + u];
            p[u] = cr[(i0 + u) >> 1];
        }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (i0 + u < f.nx) xr[i0 + u] = v[u] + p[u];
}

template <typename T>
__global__ void zero_kernel(int64_t n, T *x, const int *done) {
    if (gated(done)) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = T(0);
}

// p_c = w_c . f_c
template <typename T>
__global__ void restrict_pressure_kernel(int64_t nb, const T *__restrict__ w, const T *__restrict__ f,
                                         T *__restrict__ p, const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= nb) return;
    p[c] = w[3 * c] * f[3 * c] + w[3 * c + 1] * f[3 * c + 1] + w[3 * c + 2] * f[3 * c + 2];
}

// The same for FP32 with 16-byte accesses: four cells per thread (three float4 loads of w and
// of f, one float4 store), each cell's products and sums written as above.  Needs nb % 4 == 0
// and 16-byte aligned w, f and p.
__global__ void restrict_pressure_v4(int64_t nb4, const float4 *__restrict__ w, const float4 *__restrict__ f,
                                     float4 *__restrict__ p, const int *done) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    if (gated(done)) return;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nb4) return;
    const float4 w0 = w[3 * t], w1 = w[3 * t + 1], w2 = w[3 * t + 2];
    const float4 f0 = f[3 * t], f1 = f[3 * t + 1], f2 = f[3 * t + 2];
    float4 o;
    o.x = w0.x * f0.x + w0.y * f0.y + w0.z * f0.z;
    o.y = w0.w * f0.w + w1.x * f1.x + w1.y * f1.y;
    o.z = w1.z * f1.z + w1.w * f1.w + w2.x * f2.x;
    o.w = w2.y * f2.y + w2.z * f2.z + w2.w * f2.w;
    p[t] = o;
}

// x_c = (p_c, 0, 0) and r = f (the copy the stage-two residual starts from)
template <typename T>
__global__ void prolong_pressure_kernel(int64_t nb, const T *__restrict__ p, const T *__restrict__ f,
                                        T *__restrict__ x, T *__restrict__ r, const int *done) {
    if (gated(done)) return;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= nb) return;
    x[3 * c] = p[c];
    x[3 * c + 1] = T(0);
    x[3 * c + 2] = T(0);
    r[3 * c] = f[3 * c];
    r[3 * c + 1] = f[3 * c + 1];
    r[3 * c + 2] = f[3 * c + 2];
}

// The pressure column of every block, apc[3 q + e] = A_q[e][0] (in the solver's precision).
template <typename Tv, typename T>
__global__ void pressure_columns_kernel(int64_t nnzb, const Tv *__restrict__ v, T *__restrict__ apc) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nnzb; q += (int64_t)gridDim.x * blockDim.x) {
        apc[3 * q] = (T)v[9 * q];
        apc[3 * q + 1] = (T)v[9 * q + 3];
        apc[3 * q + 2] = (T)v[9 * q + 6];
    }
}

// x_c += (p_c, 0, 0): a pressure-stage correction added to the iterate
template <typename T>
__global__ void prolong_add_pressure_kernel(int64_t nb, const T *__restrict__ p, T *__restrict__ x, const int *done) {
    if (gated(done)) return;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c >= nb) return;
    x[3 * c] += p[c];
}

template <typename T>
__global__ void add_kernel(int64_t n, const T *__restrict__ z, T *__restrict__ x, const int *done) {
    if (gated(done)) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += z[i];
}

unsigned blocks(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

}  // namespace

void free_cpr(Cpr *P) {
    amg_free(P);
    for (int l = 0; l < kMaxLevels; ++l)
        for (void *p : {(void *)P->a7[l], P->a7f[l], P->a7s[l], P->x[l], P->b[l]})
            if (p) cudaFree(p);
    for (void *p : {(void *)P->w64, P->w, (void *)P->minv, (void *)P->dense, (void *)P->piv, (void *)P->work,
                    P->r, P->z, P->xp, P->apc})
        if (p) cudaFree(p);
    *P = Cpr();
}

cudaError_t cpr_setup(const rsv_mat *A, cudaStream_t st, bool mixed, int max_levels, int max_coarse, int sweeps,
                      int decoupling, const double *acc, int coarsening, Cpr *P, int *status) {
    const size_t es = mixed ? sizeof(float) : sizeof(double);
    amg_free(P);
    if (coarsening == 1) max_levels = 1;  // the geometric part keeps only the finest level
    // level sizes: halve (ceil) each dimension while the level has more than max_coarse cells
    int dims[kMaxLevels][3];
    G3 g{A->nx, A->ny, A->nz};
    int nl = 0;
    dims[nl][0] = g.nx, dims[nl][1] = g.ny, dims[nl][2] = g.nz;
    ++nl;
    max_levels = std::min(std::max(max_levels, 1), kMaxLevels);
    while (nl < max_levels && g.n() > max_coarse) {
        g = G3{(g.nx + 1) / 2, (g.ny + 1) / 2, (g.nz + 1) / 2};
        dims[nl][0] = g.nx, dims[nl][1] = g.ny, dims[nl][2] = g.nz;
        ++nl;
    }
    const int64_t nb = A->nb;
    const int nc = (int)g.n();
    const int64_t ncd = coarsening == 1 ? 1 : nc;  // the algebraic hierarchy keeps its own coarsest inverse
    // a new setup of the same hierarchy (the usual case: new values, same grid) reuses the buffers
    bool same = P->w64 && P->mixed == mixed && P->nlev == nl && P->ndense == ncd;
    for (int l = 0; same && l < nl; ++l)
        for (int d = 0; d < 3; ++d) same = same && P->dims[l][d] == dims[l][d];
    if (!same) free_cpr(P);
    P->mixed = mixed;
    P->sweeps = sweeps;
    for (int l = 0; l < nl; ++l)
        for (int d = 0; d < 3; ++d) P->dims[l][d] = dims[l][d];
    P->nlev = nl;
    P->ncoarse = nc;
    P->ndense = ncd;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess && !same) e = cudaMalloc(p, std::max<size_t>(bytes, 16));
    };
    alloc((void **)&P->w64, sizeof(double) * 3 * nb);
    alloc(&P->w, es * 3 * nb);
    for (int l = 0; l < nl; ++l) {
        const int64_t n = (int64_t)P->dims[l][0] * P->dims[l][1] * P->dims[l][2];
        alloc((void **)&P->a7[l], sizeof(double) * 7 * n);
        if (mixed) alloc(&P->a7f[l], sizeof(float) * 7 * n);
        if (l + 1 < nl) alloc(&P->a7s[l], es * 7 * n);
        alloc(&P->x[l], es * n);
        alloc(&P->b[l], es * n);
    }
    alloc((void **)&P->dense, sizeof(double) * ncd * ncd);
    alloc((void **)&P->minv, sizeof(double) * ncd * ncd);
    alloc((void **)&P->work, sizeof(double) * ncd * (ncd + kLuB));
    alloc((void **)&P->piv, sizeof(int) * 3 * ncd);
    alloc(&P->r, es * 3 * nb);
    alloc(&P->z, es * 3 * nb);
    alloc(&P->xp, es * 3 * nb);
    alloc(&P->apc, es * 3 * (size_t)A->nnzb + 64);  // tail room: the residual kernels stage whole 16-byte units
    if (e != cudaSuccess) {
        free_cpr(P);  // else the next setup would take the buffers for complete
        return e;
    }
    G3 g0{A->nx, A->ny, A->nz};
    count_launches(1);
    if (mixed)
        qi_setup_kernel<float><<<blocks(nb), 256, 0, st>>>(g0, A->d_rp, A->d_v32, decoupling, acc, P->w64, P->a7[0],
                                                           status);
    else
        qi_setup_kernel<double><<<blocks(nb), 256, 0, st>>>(g0, A->d_rp, A->d_v, decoupling, acc, P->w64, P->a7[0],
                                                            status);
    for (int l = 0; l + 1 < nl; ++l) {
        G3 f{P->dims[l][0], P->dims[l][1], P->dims[l][2]}, c{P->dims[l + 1][0], P->dims[l + 1][1], P->dims[l + 1][2]};
        count_launches(1);
        gmg_coarsen_kernel<<<blocks(c.n()), 256, 0, st>>>(f, P->a7[l], c, P->a7[l + 1]);
    }
    if (coarsening != 1) {
        G3 gc{P->dims[nl - 1][0], P->dims[nl - 1][1], P->dims[nl - 1][2]};
        count_launches(1);
        if ((e = cudaMemsetAsync(P->dense, 0, sizeof(double) * nc * nc, st)) != cudaSuccess) return e;
        coarse_dense_kernel<<<blocks(nc, 64), 64, 0, st>>>(gc, P->a7[nl - 1], P->dense);
        if ((e = coarse_inverse(st, nc, P->dense, P->work, P->piv, P->minv, status)) != cudaSuccess) return e;
    }
    const unsigned pcb = (unsigned)std::min<int64_t>(blocks(A->nnzb), 152 * 32);
    count_launches(1);
    if (mixed)
        pressure_columns_kernel<float, float><<<pcb, 256, 0, st>>>(A->nnzb, A->d_v32, (float *)P->apc);
    else
        pressure_columns_kernel<double, double><<<pcb, 256, 0, st>>>(A->nnzb, A->d_v, (double *)P->apc);
    for (int l = 0; l + 1 < nl; ++l) {  // the smoothed levels' colour-split coefficients
        G3 g{P->dims[l][0], P->dims[l][1], P->dims[l][2]};
        count_launches(1);
        if (mixed)
            split_stencil_kernel<float><<<blocks(g.n()), 256, 0, st>>>(g, P->a7[l], (float *)P->a7s[l]);
        else
            split_stencil_kernel<double><<<blocks(g.n()), 256, 0, st>>>(g, P->a7[l], (double *)P->a7s[l]);
    }
    if (mixed) {
        count_launches(1 + nl);
        cast_stencil<<<blocks(3 * nb), 256, 0, st>>>(3 * nb, P->w64, (float *)P->w);
        for (int l = 0; l < nl; ++l) {
            const int64_t n = (int64_t)P->dims[l][0] * P->dims[l][1] * P->dims[l][2];
            cast_stencil<<<blocks(7 * n), 256, 0, st>>>(7 * n, P->a7[l], (float *)P->a7f[l]);
        }
    } else {
        e = cudaMemcpyAsync(P->w, P->w64, sizeof(double) * 3 * nb, cudaMemcpyDeviceToDevice, st);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

// One V-cycle on level l from a zero initial guess: x[l] = V(b[l]).
template <typename T>
static cudaError_t vcycle(const Cpr &P, int l, cudaStream_t st, const int *done) {
    if (l == 0 && P.amg) return amg_vcycle<T>(P, st, done);
    const T *a7 = P.mixed ? (const T *)P.a7f[l] : (const T *)P.a7[l];
    const T *a7s = (const T *)P.a7s[l];  // colour-split copy for the smoother
    T *x = (T *)P.x[l], *b = (T *)P.b[l];
    G3 g{P.dims[l][0], P.dims[l][1], P.dims[l][2]};
    const int64_t n = g.n();
    // The cycle's kernels are launched as programmatic dependents (launch_pdl): each waits for
    // its predecessor on the device, so the launch latency of most levels' small kernels overlaps
    // the kernel before.
    if (l == P.nlev - 1) {
        count_launches(1);
        return launch_pdl(coarse_apply_kernel<T>, dim3(blocks(n * 32)), dim3(256), 0, st, (int)n, P.minv, b, x,
                          done);
    }
    G3 c{P.dims[l + 1][0], P.dims[l + 1][1], P.dims[l + 1][2]};
    const T *xc = (const T *)P.x[l + 1];
    const int64_t slots = (int64_t)((g.nx + 1) / 2) * g.ny * g.nz;  // colour slots of a half sweep
    const bool wide = slots >= (1 << 20);                             // four cells per thread
    const dim3 hb(blocks(slots)), hb4(blocks(slots, 256 * 4)), t256(256);
    const G3Div gd = G3Div::of(g);
    cudaError_t e = cudaSuccess;
    auto sweep = [&](auto kern, dim3 grid, int colour) {
        if (e == cudaSuccess) e = launch_pdl(kern, grid, t256, 0, st, g, gd, a7s, b, x, colour, xc, c, done);
    };
    auto half_sweep0 = [&](int colour) {
        if (wide)
            sweep(rbgs_kernel<T, 0, 4>, hb4, colour);
        else
            sweep(rbgs_kernel<T, 0, 1>, hb, colour);
    };
    // pre-smoothing from x = 0: red, black, `sweeps` times (the first red half sweep reads no neighbour)
    count_launches(P.sweeps > 0 ? 2 * P.sweeps : 1);
    if (P.sweeps == 0) zero_kernel<T><<<blocks(n), 256, 0, st>>>(n, x, done);
    for (int s = 0; s < P.sweeps; ++s) {
        if (s > 0)
            half_sweep0(0);
        else if (wide)
            sweep(rbgs_kernel<T, 1, 4>, hb4, 0);
        else
            sweep(rbgs_kernel<T, 1, 1>, hb, 0);
        half_sweep0(1);
    }
    count_launches(1);
    if (e == cudaSuccess)
        e = launch_pdl(residual_restrict_kernel<T>, dim3(blocks(c.n())), t256, 0, st, g, a7, b, x, c, (T *)P.b[l + 1],
                       done);
    if (e == cudaSuccess) e = vcycle<T>(P, l + 1, st, done);
    if (e != cudaSuccess) return e;
    // coarse correction x += P xc and post-smoothing black, red, `sweeps` times (the first black half
    // sweep applies the correction to the red values it reads)
    count_launches(P.sweeps > 0 ? 2 * P.sweeps : 1);
    if (P.sweeps == 0) prolong_add_kernel<T><<<blocks(n), 256, 0, st>>>(g, xc, c, x, done);
    for (int s = 0; s < P.sweeps; ++s) {
        if (s > 0) {
            half_sweep0(1);
        } else if (wide) {
            // on a large level the correction pass and a four-cell sweep beat the one-cell
            // prolongating sweep (finest level of 256x256x128: 68 us for MODE 2)
            count_launches(1);
            const int64_t quads = (int64_t)((g.nx + 3) / 4) * g.ny * g.nz;
            if (e == cudaSuccess)
                e = launch_pdl(prolong_add_rows<T>, dim3(blocks(quads)), t256, 0, st, g, Div32::of((g.nx + 3) / 4),
                               Div32::of(g.ny), xc, c, x, done);
            half_sweep0(1);
        } else {
            sweep(rbgs_kernel<T, 2, 1>, hb, 1);
        }
        half_sweep0(0);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Stage one, first half: the restricted right-hand side P.b[0] = Pi_r f.
template <typename T>
cudaError_t cpr_restrict(const rsv_mat *A, const Cpr &P, const T *f, const int *done) {
    count_launches(1);
    const bool v4 = sizeof(T) == 4 && A->nb % 4 == 0 && ((((uintptr_t)P.w) | ((uintptr_t)f) | ((uintptr_t)P.b[0])) & 15) == 0;
    if (v4)
        return launch_pdl(restrict_pressure_v4, dim3(blocks(A->nb / 4)), dim3(256), 0, A->stream, A->nb / 4,
                          (const float4 *)P.w, (const float4 *)f, (float4 *)P.b[0], done);
    return launch_pdl(restrict_pressure_kernel<T>, dim3(blocks(A->nb)), dim3(256), 0, A->stream, A->nb,
                      (const T *)P.w, f, (T *)P.b[0], done);
}

// The pressure solve P.x[0] = V-cycle(P.b[0]); kernels skip when *gate != 0.
template <typename T>
cudaError_t cpr_pressure_vcycle(const rsv_mat *A, const Cpr &P, const int *gate) {
    return vcycle<T>(P, 0, A->stream, gate);
}

// Stage one's prolongation x = Pi_p P.x[0], then stage two: x += ILU0^{-1}(f - A x).  Fused:
// r = f - A Pi_p p from the pressure columns alone, then x = ILU0^{-1} r + Pi_p p (the same
// sums, in the same order, as forming x = Pi_p p, r = f - A x and x += ILU0^{-1} r).
template <typename T>
cudaError_t cpr_finish(const rsv_mat *A, const Cpr &P, const IluTiles &tiles, const T *f, T *x, const int *done,
                       int *status, unsigned long long timeout_ns) {
    T *r = (T *)P.r;
    const T *p = (const T *)P.x[0];
    cudaError_t e = launch_pressure_residual<T>(A, (const T *)P.apc, p, f, r, done, status, timeout_ns);
    if (e != cudaSuccess) return e;
    // x = ILU0^{-1} r, and x_c[0] += p_c as the backward sweep stores x: p_c rides in the pad slot
    // of the sweeps' tile-order vectors, so no step of the sweeps waits on a load of p
    return launch_ilu_apply_tiles<T>(A, tiles, r, x, done, status, timeout_ns, p);
}

template <typename T>
cudaError_t cpr_apply(const rsv_mat *A, const Cpr &P, const IluTiles &tiles, const T *f, T *x, const int *done,
                      int *status, unsigned long long timeout_ns) {
    cudaError_t e = cpr_restrict<T>(A, P, f, done);
    if (e == cudaSuccess) e = vcycle<T>(P, 0, A->stream, done);
    if (e == cudaSuccess) e = cpr_finish<T>(A, P, tiles, f, x, done, status, timeout_ns);
    return e;
}

// The CPR orders of Section "CPR-like preconditioners" (Algorithms CPR-FP, CPR-PF,
// CPR-FPF, CPR-FFPF) as a string of stages.  The first stage writes x from f;
// every later stage forms r = f - A x (a copy of f and one SpMV) and adds its
// correction: F adds ILU0^{-1} r, P adds Pi_p V-cycle(Pi_r r).
template <typename T>
cudaError_t cpr_apply_order(const rsv_mat *A, const Cpr &P, const IluTiles &tiles, const char *stages, const T *f,
                            T *x, const int *done, int *status, unsigned long long timeout_ns) {
    cudaStream_t st = A->stream;
    const int64_t nb = A->nb;
    T *r = (T *)P.r, *z = (T *)P.z;
    cudaError_t e = cudaSuccess;
    for (int q = 0; stages[q] && e == cudaSuccess; ++q) {
        const T *src = f;
        if (q > 0) {
            e = cudaMemcpyAsync(r, f, sizeof(T) * 3 * nb, cudaMemcpyDeviceToDevice, st);
            if (e == cudaSuccess)
                e = (sizeof(T) == 8) ? launch_spmv_f64(A, -1.0, (const double *)x, 1.0, (double *)r, done, status, timeout_ns)
                                     : launch_spmv_f32(A, -1.0f, (const float *)x, 1.0f, (float *)r, done, status,
                                                       timeout_ns);
            src = r;
        }
        if (e != cudaSuccess) break;
        if (stages[q] == 'F') {
            e = launch_ilu_apply_tiles<T>(A, tiles, src, q == 0 ? x : z, done, status, timeout_ns);
            if (e == cudaSuccess && q > 0) {
                count_launches(1);
                add_kernel<T><<<blocks(3 * nb), 256, 0, st>>>(3 * nb, z, x, done);
                e = cudaGetLastError();
            }
        } else {
            e = cpr_restrict<T>(A, P, src, done);
            if (e == cudaSuccess) e = vcycle<T>(P, 0, st, done);
            if (e == cudaSuccess) {
                count_launches(1);
                if (q == 0)
                    prolong_pressure_kernel<T><<<blocks(nb), 256, 0, st>>>(nb, (const T *)P.x[0], f, x, r, done);
                else
                    prolong_add_pressure_kernel<T><<<blocks(nb), 256, 0, st>>>(nb, (const T *)P.x[0], x, done);
                e = cudaGetLastError();
            }
        }
    }
    return e;
}

template <typename T>
cudaError_t cpr_vcycle(const rsv_mat *A, const Cpr &P, const T *b, T *x) {
    const int64_t n = A->nb;
    cudaError_t e = cudaMemcpyAsync(P.b[0], b, sizeof(T) * n, cudaMemcpyDeviceToDevice, A->stream);
    if (e == cudaSuccess) e = vcycle<T>(P, 0, A->stream, nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(x, P.x[0], sizeof(T) * n, cudaMemcpyDeviceToDevice, A->stream);
    return e;
}

template cudaError_t cpr_apply<double>(const rsv_mat *, const Cpr &, const IluTiles &, const double *, double *,
                                       const int *, int *, unsigned long long);
template cudaError_t cpr_apply<float>(const rsv_mat *, const Cpr &, const IluTiles &, const float *, float *,
                                      const int *, int *, unsigned long long);
template cudaError_t cpr_apply_order<double>(const rsv_mat *, const Cpr &, const IluTiles &, const char *,
                                             const double *, double *, const int *, int *, unsigned long long);
template cudaError_t cpr_apply_order<float>(const rsv_mat *, const Cpr &, const IluTiles &, const char *,
                                            const float *, float *, const int *, int *, unsigned long long);
template cudaError_t cpr_vcycle<double>(const rsv_mat *, const Cpr &, const double *, double *);
template cudaError_t cpr_restrict<double>(const rsv_mat *, const Cpr &, const double *, const int *);
template cudaError_t cpr_pressure_vcycle<double>(const rsv_mat *, const Cpr &, const int *);
template cudaError_t cpr_finish<double>(const rsv_mat *, const Cpr &, const IluTiles &, const double *, double *,
                                        const int *, int *, unsigned long long);
template cudaError_t cpr_vcycle<float>(const rsv_mat *, const Cpr &, const float *, float *);

}  // namespace rsv

// Batched solves: many independent reservoir systems of uneven grid sizes.
//
// The systems of a batch matrix (rsv_mat_create_batch) form one
// block-diagonal BSR matrix, so one SpMV launch and one cooperative launch of
// each block-ILU(0) tile sweep serve every system at once.  The Krylov
// method runs per system: right-preconditioned BiCGSTAB (Section "Solvers")
// with each system's own scalars (rho, alpha, omega, beta), its own
// convergence test and iteration count.  A converged system freezes: the
// vector updates, the sweeps and the products skip its rows.  Segmented reductions give every system its
// own FP64-accurate dot products, deterministically (per system, the last CTA
// to finish adds the partial sums of fixed chunks in a fixed pattern).
//
// One loop pass (two preconditioner applications, two SpMVs, four segmented
// reductions and the scalar steps) is captured once into a CUDA graph holding
// kGraphIters passes; the host replays the graph and reads a single
// "systems done" counter between replays.
//
// Mixed precision: an FP64 refinement loop per system (r = b - A x in FP64,
// per-system norms), FP32 inner BiCGSTAB on r / ||r|| to the inner
// tolerance, x += ||r|| d; systems that meet the outer tolerance stop.
//
// The SpMV tile shape (block rows per CTA) is picked by timing the candidates
// on the batch matrix at preconditioner setup.
#include <cmath>
#include <vector>

#include "reduce.cuh"
#include "solver.cuh"

namespace rsv {
namespace {

constexpr int kChunk = 8192;      // elements per reduction work item
constexpr int kGraphIters = 4;    // BiCGSTAB passes per graph replay
constexpr int kSegThreads = 256;
constexpr int kStallPasses = 30;  // FP32 inner solves: passes without progress before handing back

struct SegItem {
    int sys;
    int pad;
    int64_t begin, end;
};

// Per-system state of the batched BiCGSTAB (arrays of nsys).
struct BatchDev {
    double *rho, *rho1, *alpha, *omega, *beta, *tol, *rhn, *scale, *bnorm, *best;
    double *red;     // [8][nsys]: 0 <rh,r> 1 <rh,v> 2 ||v|| 3 ||s|| 4 <t,s> 5 <t,t> 6 ||r|| 7 spare
    int *done, *status, *iters, *half, *outer, *stall;
    int *ndone;      // systems done (single counter)
    unsigned *ticket;  // [4][nsys] reduction tickets
    double *partial;   // [2][nitems]
};

struct BatchState {
    int nsys = 0, nitems = 0;
    SegItem *items = nullptr;
    int *item_begin = nullptr;  // per system: first item; item_begin[nsys] = nitems
    BatchDev dv{};
    void *dev_block = nullptr;  // one allocation behind dv
    void *vec = nullptr;        // 8 Krylov vectors in the inner precision
    void *xin = nullptr;        // inner solution (FP64 mode: copy of x; mixed: the FP32 correction)
    void *rin = nullptr;        // inner right-hand side
    int *h_ndone = nullptr;     // pinned
    cudaGraphExec_t graph[2] = {nullptr, nullptr};  // [0] FP64, [1] FP32
    size_t graph_nodes[2] = {0, 0};
    uint64_t graph_version = ~0ull;
    bool graph_ok[2] = {true, true};
    bool tuned = false;
    cudaStream_t own = nullptr;  // capture-capable stream used when the caller's is the legacy default
};

// Runs the batched solve on the solver's own stream when the caller's stream
// is the legacy default stream (which cannot be captured into a graph):
// the caller's stream is synchronised first and the handles point at the
// own stream until the solve returns.
struct StreamSwap {
    rsv_solver *s;
    cudaStream_t saved;
    bool active = false;
    StreamSwap(rsv_solver *s_, cudaStream_t own) : s(s_), saved(s_->st) {
        if (saved == nullptr || saved == cudaStreamLegacy) {
            cudaStreamSynchronize(saved);
            s->st = own;
            s->A->stream = own;
            active = true;
        }
    }
    ~StreamSwap() {
        if (active) {
            cudaStreamSynchronize(s->st);
            s->st = saved;
            s->A->stream = saved;
        }
    }
};

// Calls f4(i) for the 16-byte groups of a work item and f1(i) for the elements beside them, over the CTA's threads.
// Groups start at multiples of 16 bytes of the vectors (ok: every vector's base is 16-byte aligned).
template <typename T, typename F4, typename F1>
__device__ __forceinline__ void over_item(const SegItem &w, bool ok, F4 f4, F1 f1) {
    constexpr int N = Vec<T>::N;
    const int64_t g0 = ok ? min((w.begin + N - 1) / N * N, w.end) : w.end, g1 = ok ? max(w.end / N * N, g0) : w.end;
    const int64_t head = ok ? g0 : w.end;
#pragma unroll 4
    for (int64_t i = g0 + N * (int64_t)threadIdx.x; i < g1; i += N * (int64_t)blockDim.x) f4(i);
    for (int64_t i = w.begin + threadIdx.x; i < head; i += blockDim.x) f1(i);
    for (int64_t i = g1 + threadIdx.x; i < w.end; i += blockDim.x) f1(i);
}
template <typename T> __device__ __forceinline__ typename Vec<T>::V ld_vec(const T *p) {
    return *reinterpret_cast<const typename Vec<T>::V *>(p);
}
template <typename T> __device__ __forceinline__ void st_vec(T *p, const typename Vec<T>::V &v) {
    *reinterpret_cast<typename Vec<T>::V *>(p) = v;
}
__device__ __forceinline__ float scalar(double v, float) { return (float)v; }
__device__ __forceinline__ double scalar(double v, double) { return v; }

__device__ __forceinline__ void finish_sys(BatchDev d, int s, int code) {
    if (code && d.status[s] == 0) d.status[s] = code;
    if (!d.done[s]) {
        d.done[s] = 1;
        atomicAdd(d.ndone, 1);
    }
}

// BiCGSTAB scalar steps of system s.
__device__ __forceinline__ void step_beta(BatchDev d, int nsys, int s, double btol) {
    if (d.done[s]) return;
    const double rho1 = d.red[0 * nsys + s];
    if (!isfinite(rho1)) return finish_sys(d, s, RSV_ENAN);
    if (fabs(rho1) <= btol * d.rhn[s] * d.red[6 * nsys + s]) return finish_sys(d, s, RSV_EBREAKDOWN);
    d.rho1[s] = rho1;
    d.beta[s] = (rho1 / d.rho[s]) * (d.alpha[s] / d.omega[s]);
}
__device__ __forceinline__ void step_alpha(BatchDev d, int nsys, int s, double btol) {
    if (d.done[s]) return;
    const double rv = d.red[1 * nsys + s], vn = sqrt(fmax(d.red[2 * nsys + s], 0.0));
    if (!isfinite(rv)) return finish_sys(d, s, RSV_ENAN);
    if (fabs(rv) <= btol * d.rhn[s] * vn) return finish_sys(d, s, RSV_EBREAKDOWN);
    d.alpha[s] = d.rho1[s] / rv;
}
__device__ __forceinline__ void step_check_s(BatchDev d, int nsys, int s) {
    if (d.done[s]) return;
    d.iters[s] += 1;
    const double sn = d.red[3 * nsys + s];
    if (!isfinite(sn)) return finish_sys(d, s, RSV_ENAN);
    if (sn <= d.tol[s]) {
        d.half[s] = 1;  // x += alpha ph pending
        finish_sys(d, s, 0);
    }
}
__device__ __forceinline__ void step_omega(BatchDev d, int nsys, int s, double btol) {
    if (d.half[s] == 1) d.half[s] = 2;  // b_half_x has run
    if (d.done[s]) return;
    const double ts = d.red[4 * nsys + s], tt = d.red[5 * nsys + s];
    if (!isfinite(tt)) return finish_sys(d, s, RSV_ENAN);
    if (!(tt > 0.0)) return finish_sys(d, s, RSV_EBREAKDOWN);
    const double om = ts / tt;
    if (fabs(om) <= btol) return finish_sys(d, s, RSV_EBREAKDOWN);
    d.omega[s] = om;
}
// stall_limit > 0 (FP32 inner solves of refinement): a system whose residual
// has not dropped below 0.99 of its best for stall_limit passes ends its
// inner solve; FP32 BiCGSTAB can stagnate above the inner tolerance on an
// ill-conditioned system, and the FP64 outer step continues from there.
__device__ __forceinline__ void step_finish(BatchDev d, int nsys, int s, int maxit, int stall_limit) {
    if (d.done[s]) return;
    d.rho[s] = d.rho1[s];
    const double rn = d.red[6 * nsys + s];
    if (!isfinite(rn)) return finish_sys(d, s, RSV_ENAN);
    if (rn <= d.tol[s]) return finish_sys(d, s, 0);
    if (d.iters[s] >= maxit) return finish_sys(d, s, RSV_ENOCONV);
    if (stall_limit > 0) {
        if (rn < 0.99 * d.best[s]) {
            d.best[s] = rn;
            d.stall[s] = 0;
        } else if (++d.stall[s] >= stall_limit) {
            return finish_sys(d, s, 0);
        }
    }
}

// The scalar step that follows a reduction, run by the thread that finishes a system's sums.
enum class After { none, alpha, check_s, omega, finish };
struct Scalars {
    BatchDev d;
    int nsys;
    double btol;
    int maxit, stall_limit;
};

// out1[s] = <x, y1> (or its sqrt) and, when y2, out2[s] = <x, y2>, per system s, then the scalar step `after`
// of system s.  HBM should bound it; what did was one thread per system adding the items' partial sums one
// after another, an FP64 tree in every warp and scalar loads (24 systems, 7 M FP32 unknowns: 72 -> 27 us).  Now items are
// read in 16-byte groups, half a warp adds an item's sums (each lane a fixed strided subset, then a tree), and a warp adds
// the items' partial sums in the same manner: FP64 throughout, and still deterministic.  (A tree of double-float pairs in
// every warp takes 4 us less, but keeps 46 bits of the 53.)
template <typename T>
__global__ void __launch_bounds__(kSegThreads) seg_dot_kernel(const SegItem *__restrict__ items, int nitems,
                                                              const int *__restrict__ item_begin,
                                                              const T *__restrict__ x, const T *__restrict__ y1,
                                                              const T *__restrict__ y2, double *out1, double *out2,
                                                              int sqrt1, double *partial, unsigned *ticket,
                                                              const int *done, After after, Scalars sc) {
    __shared__ double sm[2][kSegThreads];
    __shared__ bool last;
    const bool ok = ((((uintptr_t)x) | ((uintptr_t)y1) | ((uintptr_t)y2)) & 15) == 0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const SegItem w = items[it];
        Acc<T> a1, a2;
        const bool frozen = done && done[w.sys];
        if (!frozen)
            over_item<T>(
                w, ok,
                [&](int64_t i) {
                    const auto xv = ld_vec(x + i), yv = ld_vec(y1 + i);
#pragma unroll
                    for (int q = 0; q < Vec<T>::N; ++q) a1.add(Vec<T>::get(xv, q), Vec<T>::get(yv, q));
                    if (y2) {
                        const auto zv = ld_vec(y2 + i);
#pragma unroll
                        for (int q = 0; q < Vec<T>::N; ++q) a2.add(Vec<T>::get(xv, q), Vec<T>::get(zv, q));
                    }
                },
                [&](int64_t i) {
                    a1.add(x[i], y1[i]);
                    if (y2) a2.add(x[i], y2[i]);
                });
        sm[0][threadIdx.x] = a1.value();
        if (y2) sm[1][threadIdx.x] = a2.value();
        __syncthreads();
        if (warp == 0) {  // lanes 0-15 add the first product's sums, lanes 16-31 the second's
            const int half = lane >> 4, l = lane & 15;
            double s1 = 0.0;
            if (half == 0 || y2)
#pragma unroll
                for (int q = 0; q < kSegThreads; q += 16) s1 += sm[half][q + l];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            if (l == 0) partial[(size_t)half * nitems + it] = s1;
            __syncwarp();
            if (lane == 0) {
                __threadfence();  // both partial sums before the ticket
                const unsigned nit = (unsigned)(item_begin[w.sys + 1] - item_begin[w.sys]);
                last = atomicAdd(&ticket[w.sys], 1u) == nit - 1;
            }
        }
        __syncthreads();
        if (last && warp == 0) {
            __threadfence();
            double s1 = 0.0, s2 = 0.0;
            for (int q = item_begin[w.sys] + lane; q < item_begin[w.sys + 1]; q += 32) {
                s1 += __ldcg(&partial[q]);
                if (y2) s2 += __ldcg(&partial[nitems + q]);
            }
            s1 = warp_sum(s1);
            if (y2) s2 = warp_sum(s2);
            if (lane == 0) {
                if (!(done && done[w.sys])) {
                    out1[w.sys] = sqrt1 ? sqrt(s1) : s1;
                    if (out2) out2[w.sys] = s2;
                }
                ticket[w.sys] = 0u;
                switch (after) {
                case After::none: break;
                case After::alpha: step_alpha(sc.d, sc.nsys, w.sys, sc.btol); break;
                case After::check_s: step_check_s(sc.d, sc.nsys, w.sys); break;
                case After::omega: step_omega(sc.d, sc.nsys, w.sys, sc.btol); break;
                case After::finish:  // and the next pass's beta
                    step_finish(sc.d, sc.nsys, w.sys, sc.maxit, sc.stall_limit);
                    step_beta(sc.d, sc.nsys, w.sys, sc.btol);
                    break;
                }
            }
        }
        __syncthreads();
    }
}

// The first pass's beta, one thread per system.
__global__ void b_beta(BatchDev d, int nsys, double btol) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nsys) step_beta(d, nsys, s, btol);
}

// Vector updates, one CTA per work item: a system's scalars are loaded and rounded once per item (once per element
// bound these kernels by the FP64 pipe's conversions), and a frozen system's items return at once.
template <typename T>
__global__ void __launch_bounds__(kSegThreads) b_update_p(const SegItem *__restrict__ items, BatchDev d, const T *r, const T *v,
                                                          T *p) {
    const SegItem w = items[blockIdx.x];
    if (d.done[w.sys]) return;
    const T beta = scalar(d.beta[w.sys], T(0)), om = scalar(d.omega[w.sys], T(0));
    over_item<T>(
        w, true,
        [&](int64_t i) {
            const auto rv = ld_vec(r + i), vv = ld_vec(v + i);
            auto pv = ld_vec(p + i);
#pragma unroll
            for (int q = 0; q < Vec<T>::N; ++q)
                Vec<T>::set(pv, q, Vec<T>::get(rv, q) + beta * (Vec<T>::get(pv, q) - om * Vec<T>::get(vv, q)));
            st_vec(p + i, pv);
        },
        [&](int64_t i) { p[i] = r[i] + beta * (p[i] - om * v[i]); });
}

template <typename T>
__global__ void __launch_bounds__(kSegThreads) b_update_s(const SegItem *__restrict__ items, BatchDev d, const T *r, const T *v,
                                                          T *sv) {
    const SegItem w = items[blockIdx.x];
    if (d.done[w.sys]) return;
    const T al = scalar(d.alpha[w.sys], T(0));
    over_item<T>(
        w, true,
        [&](int64_t i) {
            const auto rv = ld_vec(r + i), vv = ld_vec(v + i);
            auto o = rv;
#pragma unroll
            for (int q = 0; q < Vec<T>::N; ++q) Vec<T>::set(o, q, Vec<T>::get(rv, q) - al * Vec<T>::get(vv, q));
            st_vec(sv + i, o);
        },
        [&](int64_t i) { sv[i] = r[i] - al * v[i]; });
}

template <typename T>
__global__ void __launch_bounds__(kSegThreads) b_half_x(const SegItem *__restrict__ items, BatchDev d, const T *ph, T *x) {
    const SegItem w = items[blockIdx.x];
    if (d.half[w.sys] != 1) return;
    const T al = scalar(d.alpha[w.sys], T(0));
    for (int64_t i = w.begin + threadIdx.x; i < w.end; i += blockDim.x) x[i] += al * ph[i];
}

template <typename T>
__global__ void __launch_bounds__(kSegThreads) b_update_xr(const SegItem *__restrict__ items, BatchDev d, const T *ph, const T *sh,
                                                           const T *sv, const T *t, T *x, T *r) {
    const SegItem w = items[blockIdx.x];
    if (d.done[w.sys]) return;
    const T al = scalar(d.alpha[w.sys], T(0)), om = scalar(d.omega[w.sys], T(0));
    over_item<T>(
        w, true,
        [&](int64_t i) {
            const auto pv = ld_vec(ph + i), hv = ld_vec(sh + i), sw = ld_vec(sv + i), tv = ld_vec(t + i);
            auto xv = ld_vec(x + i), rv = sw;
#pragma unroll
            for (int q = 0; q < Vec<T>::N; ++q) {
                Vec<T>::set(xv, q, Vec<T>::get(xv, q) + (al * Vec<T>::get(pv, q) + om * Vec<T>::get(hv, q)));
                Vec<T>::set(rv, q, Vec<T>::get(sw, q) - om * Vec<T>::get(tv, q));
            }
            st_vec(x + i, xv);
            st_vec(r + i, rv);
        },
        [&](int64_t i) {
            x[i] += al * ph[i] + om * sh[i];
            r[i] = sv[i] - om * t[i];
        });
}

// Start of an inner solve: per-system tolerance and scalars; systems marked
// finished by the outer loop stay frozen.
__global__ void b_init(BatchDev d, int nsys, double rtol_or_inner, int mixed, double rtol) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsys) return;
    d.rho[s] = d.alpha[s] = d.omega[s] = 1.0;
    d.half[s] = 0;
    d.rhn[s] = d.red[6 * nsys + s];
    // FP64 mode: tol = rtol ||b||.  Mixed: the inner right-hand side has unit norm; the
    // inner tolerance is inner_rtol, or less strict on the system's last outer step,
    // which only needs ||r|| below rtol ||b|| (factor 2 of margin).
    if (mixed) {
        const double rn = d.red[7 * nsys + s];
        double t = rtol_or_inner;
        if (rn > 0.0) t = fmax(t, 0.5 * rtol * d.bnorm[s] / rn);
        d.tol[s] = t;
    } else {
        d.tol[s] = rtol_or_inner * d.bnorm[s];
    }
    d.done[s] = d.outer[s];
    d.best[s] = d.red[6 * nsys + s];
    d.stall[s] = 0;
}

__global__ void b_count_done(BatchDev d, int nsys) {
    int c = 0;
    for (int s = threadIdx.x; s < nsys; s += blockDim.x) c += d.done[s];
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    __shared__ int sm[32];
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += sm[q];
        *d.ndone = t;
    }
}

// Outer-loop bookkeeping: systems whose FP64 residual meets rtol ||b|| are finished.
__global__ void b_outer_check(BatchDev d, int nsys, double rtol, const double *rn, int max_outer, int maxit) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsys || d.outer[s]) return;
    if (!isfinite(rn[s])) {
        d.outer[s] = 1;
        if (d.status[s] == 0) d.status[s] = RSV_ENAN;
    } else if (rn[s] <= rtol * d.bnorm[s]) {
        d.outer[s] = 1;
        d.status[s] = 0;
    } else if (d.scale[s] >= max_outer || d.iters[s] >= maxit) {
        d.outer[s] = 1;
        if (d.status[s] == 0 || d.status[s] == RSV_ENOCONV) d.status[s] = RSV_ENOCONV;
    } else {
        d.status[s] = 0;  // an inner breakdown or maxit leaves a usable correction
    }
}

template <typename T>
__global__ void __launch_bounds__(kSegThreads) b_scaled_copy(const SegItem *__restrict__ items, BatchDev d,
                                                             const double *__restrict__ r64,
                                                             const double *__restrict__ rn, T *__restrict__ out) {
    const SegItem w = items[blockIdx.x];
    const bool skip = d.outer[w.sys] != 0;
    const double n = rn[w.sys];
    for (int64_t i = w.begin + threadIdx.x; i < w.end; i += blockDim.x) out[i] = skip ? T(0) : (T)(r64[i] / n);
}

__global__ void __launch_bounds__(kSegThreads) b_add_scaled(const SegItem *__restrict__ items, BatchDev d,
                                                            const float *__restrict__ df, const double *__restrict__ rn,
                                                            double *__restrict__ x) {
    const SegItem w = items[blockIdx.x];
    if (d.outer[w.sys]) return;
    const double n = rn[w.sys];
    for (int64_t i = w.begin + threadIdx.x; i < w.end; i += blockDim.x) x[i] += n * (double)df[i];
}

__global__ void b_bump_outer(BatchDev d, int nsys) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < nsys && !d.outer[s]) d.scale[s] += 1.0;  // outer steps taken (kept as a double)
}

unsigned sgrid(int nsys) { return (unsigned)((nsys + 127) / 128); }

template <typename T>
cudaError_t seg_dot(rsv_solver *s, BatchState *B, const T *x, const T *y1, const T *y2, double *o1, double *o2,
                    int sqrt1, int slot, const int *done, After after = After::none) {
    count_launches(1);
    const int grid = std::min(B->nitems, 8 * 152);
    const Scalars sc{B->dv, B->nsys, s->p.btol, s->p.maxit, sizeof(T) == 4 ? kStallPasses : 0};
    seg_dot_kernel<T><<<grid, kSegThreads, 0, s->st>>>(B->items, B->nitems, B->item_begin, x, y1, y2, o1, o2, sqrt1,
                                                       B->dv.partial, B->dv.ticket + (size_t)slot * B->nsys, done,
                                                       after, sc);
    return cudaGetLastError();
}

template <typename T>
T *vecs(BatchState *B, int64_t ldv, int q) {
    return (T *)B->vec + (size_t)q * ldv;
}

// z = M^{-1} r and y = A z for the systems that still run: the sweeps' tiles and the product's rows of finished ones
// are skipped (nothing reads them any more).  24 systems of 16 to 96 cells a side, FP32, to 1e-12: 330 -> 291 ms.
template <typename T>
cudaError_t apply_live(rsv_solver *s, const int *done, const T *r, T *z, T *y) {
    const unsigned long long limit = (unsigned long long)s->p.watchdog * 1000ull;
    cudaError_t e = s->pc_type == RSV_PC_BILU0
                        ? launch_ilu_apply_tiles<T>(s->A, s->tiles, r, z, nullptr, &s->ds->status, limit, nullptr, done)
                        : pc_apply<T>(s, r, z, nullptr);
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 8)
        return launch_spmv_f64(s->A, 1.0, z, 0.0, y, nullptr, &s->ds->status, limit, done);
    else
        return launch_spmv_f32(s->A, 1.f, z, 0.f, y, nullptr, &s->ds->status, limit, done);
}

// kGraphIters BiCGSTAB passes for all systems (the body that is captured).
template <typename T>
cudaError_t bicg_passes(rsv_solver *s, BatchState *B, T *x) {
    const int64_t ldv = s->ldv;
    const int nsys = B->nsys;
    const BatchDev d = B->dv;
    T *r = vecs<T>(B, ldv, 0), *rh = vecs<T>(B, ldv, 1), *p = vecs<T>(B, ldv, 2), *v = vecs<T>(B, ldv, 3),
      *ph = vecs<T>(B, ldv, 4), *sh = vecs<T>(B, ldv, 5), *sv = vecs<T>(B, ldv, 6), *t = vecs<T>(B, ldv, 7);
    const int g = B->nitems;
    cudaError_t e = cudaSuccess;
    for (int it = 0; it < kGraphIters && e == cudaSuccess; ++it) {
        count_launches(4);
        b_update_p<T><<<g, kSegThreads, 0, s->st>>>(B->items, d, r, v, p);
        if ((e = apply_live<T>(s, d.done, p, ph, v)) != cudaSuccess) break;
        if ((e = seg_dot<T>(s, B, v, rh, v, d.red + 1 * nsys, d.red + 2 * nsys, 0, 1, d.done, After::alpha)) !=
            cudaSuccess)
            break;
        b_update_s<T><<<g, kSegThreads, 0, s->st>>>(B->items, d, r, v, sv);
        if ((e = seg_dot<T>(s, B, sv, sv, (const T *)nullptr, d.red + 3 * nsys, nullptr, 1, 2, d.done,
                            After::check_s)) != cudaSuccess)
            break;
        b_half_x<T><<<g, kSegThreads, 0, s->st>>>(B->items, d, ph, x);
        if ((e = apply_live<T>(s, d.done, sv, sh, t)) != cudaSuccess) break;
        if ((e = seg_dot<T>(s, B, t, sv, t, d.red + 4 * nsys, d.red + 5 * nsys, 0, 3, d.done, After::omega)) !=
            cudaSuccess)
            break;
        b_update_xr<T><<<g, kSegThreads, 0, s->st>>>(B->items, d, ph, sh, sv, t, x, r);
        // ||r|| of the new residual and <rh, r> for the next pass, in one sweep
        if ((e = seg_dot<T>(s, B, r, r, rh, d.red + 6 * nsys, d.red + 0 * nsys, 1, 0, d.done, After::finish)) !=
            cudaSuccess)
            break;
        e = cudaGetLastError();
    }
    return e;
}

// Inner batched BiCGSTAB on A_T x = rhs (rhs, x in precision T), x from zero.
template <typename T>
rsv_status bicg_inner(rsv_solver *s, BatchState *B, const T *rhs, T *x, double tol_param, int mixed) {
    const int64_t n = s->n, ldv = s->ldv;
    const int nsys = B->nsys;
    const BatchDev d = B->dv;
    T *r = vecs<T>(B, ldv, 0), *rh = vecs<T>(B, ldv, 1), *p = vecs<T>(B, ldv, 2), *v = vecs<T>(B, ldv, 3);
    RSV_CUDA_TRY(cudaMemsetAsync(x, 0, sizeof(T) * n, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(r, rhs, sizeof(T) * n, cudaMemcpyDeviceToDevice, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(rh, rhs, sizeof(T) * n, cudaMemcpyDeviceToDevice, s->st));
    RSV_CUDA_TRY(cudaMemsetAsync(p, 0, sizeof(T) * n, s->st));
    RSV_CUDA_TRY(cudaMemsetAsync(v, 0, sizeof(T) * n, s->st));
    // ||r|| and <rh, r> of the starting residual (no system is frozen yet for this sweep)
    RSV_CUDA_TRY(seg_dot<T>(s, B, r, r, rh, d.red + 6 * nsys, d.red + 0 * nsys, 1, 0, nullptr));
    count_launches(3);
    b_init<<<sgrid(nsys), 128, 0, s->st>>>(d, nsys, tol_param, mixed, s->p.rtol);
    b_count_done<<<1, 256, 0, s->st>>>(d, nsys);
    b_beta<<<sgrid(nsys), 128, 0, s->st>>>(d, nsys, s->p.btol);
    RSV_CUDA_TRY(cudaGetLastError());
    const int gi = sizeof(T) == 8 ? 0 : 1;
    // (re)capture the graph of kGraphIters passes when the preconditioner changed
    if (B->graph_version != s->pc_version) {
        for (int q = 0; q < 2; ++q)
            if (B->graph[q]) {
                cudaGraphExecDestroy(B->graph[q]);
                B->graph[q] = nullptr;
            }
        B->graph_ok[0] = B->graph_ok[1] = true;
        B->graph_version = s->pc_version;
    }
    if (!B->graph[gi] && B->graph_ok[gi]) {
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(s->st, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            const cudaError_t eb = bicg_passes<T>(s, B, x);
            e = cudaStreamEndCapture(s->st, &g);
            if (eb != cudaSuccess) e = eb;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&B->graph[gi], g, 0);
        if (e == cudaSuccess) e = cudaGraphGetNodes(g, nullptr, &B->graph_nodes[gi]);
        if (g) cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            // a stream that cannot be captured: launch the passes directly
            B->graph[gi] = nullptr;
            B->graph_ok[gi] = false;
            cudaGetLastError();
        }
    }
    const int max_rounds = s->p.maxit / kGraphIters + 2;
    for (int round = 0; round < max_rounds; ++round) {
        RSV_CUDA_TRY(cudaMemcpyAsync(B->h_ndone, d.ndone, sizeof(int), cudaMemcpyDeviceToHost, s->st));
        RSV_CUDA_TRY(cudaStreamSynchronize(s->st));
        if (*B->h_ndone >= nsys) break;
        if (B->graph[gi]) {
            count_launches(B->graph_nodes[gi]);
            RSV_CUDA_TRY(cudaGraphLaunch(B->graph[gi], s->st));
        } else
            RSV_CUDA_TRY(bicg_passes<T>(s, B, x));
    }
    return RSV_OK;
}

// Segmented work items of the batch matrix (chunks of each system's unknowns).
rsv_status batch_init(rsv_solver *s, BatchState **out) {
    const rsv_mat *A = s->A;
    BatchState *B = new (std::nothrow) BatchState();
    if (!B) return RSV_ENOMEM;
    B->nsys = A->nsys;
    std::vector<SegItem> items;
    std::vector<int> ibeg;
    for (int q = 0; q < A->nsys; ++q) {
        ibeg.push_back((int)items.size());
        const int64_t b0 = 3 * A->h_sys[q].cell0;
        const int64_t b1 = (q + 1 < A->nsys) ? 3 * A->h_sys[q + 1].cell0 : 3 * A->nb;
        for (int64_t c = b0; c < b1; c += kChunk) items.push_back(SegItem{q, 0, c, std::min(c + kChunk, b1)});
    }
    ibeg.push_back((int)items.size());
    B->nitems = (int)items.size();
    const int ns = A->nsys;
    const size_t nd = 10 + 8;  // scalar double arrays + red[8]
    const size_t bytes = sizeof(double) * (nd * ns + 2 * (size_t)B->nitems) + sizeof(int) * (6 * ns + 4) +
                         sizeof(unsigned) * 4 * ns + 256;
    const size_t es = s->mixed ? sizeof(float) : sizeof(double);
    cudaError_t e = cudaSuccess;
    if ((e = cudaMalloc((void **)&B->items, sizeof(SegItem) * items.size())) == cudaSuccess &&
        (e = cudaMalloc((void **)&B->item_begin, sizeof(int) * ibeg.size())) == cudaSuccess &&
        (e = cudaMalloc(&B->dev_block, bytes)) == cudaSuccess &&
        (e = cudaMalloc(&B->vec, 8 * (size_t)s->ldv * es)) == cudaSuccess &&
        (e = cudaMalloc(&B->xin, (size_t)s->ldv * es)) == cudaSuccess &&
        (e = cudaMalloc(&B->rin, (size_t)s->ldv * es)) == cudaSuccess &&
        (e = cudaMallocHost((void **)&B->h_ndone, sizeof(int))) == cudaSuccess &&
        (e = cudaMemcpyAsync(B->items, items.data(), sizeof(SegItem) * items.size(), cudaMemcpyHostToDevice,
                             s->st)) == cudaSuccess &&
        (e = cudaMemcpyAsync(B->item_begin, ibeg.data(), sizeof(int) * ibeg.size(), cudaMemcpyHostToDevice,
                             s->st)) == cudaSuccess &&
        (e = cudaMemsetAsync(B->dev_block, 0, bytes, s->st)) == cudaSuccess) {
        char *p = (char *)B->dev_block;
        auto take_d = [&](size_t cnt) { double *q = (double *)p; p += sizeof(double) * cnt; return q; };
        BatchDev &d = B->dv;
        d.rho = take_d(ns); d.rho1 = take_d(ns); d.alpha = take_d(ns); d.omega = take_d(ns); d.beta = take_d(ns);
        d.tol = take_d(ns); d.rhn = take_d(ns); d.scale = take_d(ns); d.bnorm = take_d(ns); d.best = take_d(ns);
        d.red = take_d(8 * (size_t)ns);
        d.partial = take_d(2 * (size_t)B->nitems);
        int *ip = (int *)p;
        d.done = ip; d.status = ip + ns; d.iters = ip + 2 * ns; d.half = ip + 3 * ns; d.outer = ip + 4 * ns;
        d.stall = ip + 5 * ns;
        d.ndone = ip + 6 * ns;
        d.ticket = (unsigned *)(ip + 6 * ns + 4);
        e = cudaStreamSynchronize(s->st);
    }
    if (e != cudaSuccess) {
        BatchState *tmp = B;
        s->batch = tmp;
        free_batch(s);
        return cuda_status(e);
    }
    *out = B;
    return RSV_OK;
}

}  // namespace

void free_batch(rsv_solver *s) {
    BatchState *B = (BatchState *)s->batch;
    if (!B) return;
    for (int q = 0; q < 2; ++q)
        if (B->graph[q]) cudaGraphExecDestroy(B->graph[q]);
    for (void *p : {(void *)B->items, (void *)B->item_begin, B->dev_block, B->vec, B->xin, B->rin})
        if (p) cudaFree(p);
    if (B->h_ndone) cudaFreeHost(B->h_ndone);
    if (B->own) cudaStreamDestroy(B->own);
    delete B;
    s->batch = nullptr;
}

}  // namespace rsv

using namespace rsv;

extern "C" rsv_status rsv_solve_batched(rsv_solver *s, const rsv_vec *b, rsv_vec *x, rsv_solve_info *infos) {
    if (!s || !b || !x) return RSV_EINVAL;
    if (b->prec != RSV_PREC_FP64 || x->prec != RSV_PREC_FP64 || b->n != s->n || x->n != s->n) return RSV_EINVAL;
    if (b->data == x->data && s->n > 0) return RSV_EINVAL;
    return rsv_solve_batched_ptr(s, (const double *)b->data, (double *)x->data, 1, infos);
}

extern "C" rsv_status rsv_solve_batched_ptr(rsv_solver *s, const double *b, double *x, int on_device,
                                            rsv_solve_info *infos) {
    if (!s || !b || !x) return RSV_EINVAL;
    if (s->pc_type < 0 || s->pc_version != s->A->version) return RSV_EINVAL;
    if (s->p.solver != RSV_BICGSTAB) return RSV_ENOTSUP;
    if (s->pc_type != RSV_PC_NONE && s->pc_type != RSV_PC_BJACOBI && s->pc_type != RSV_PC_BILU0) return RSV_ENOTSUP;
    rsv_mat *A = s->A;
    const int nsys = A->nsys;
    const int64_t n = s->n;
    if (!s->batch) RSV_TRY(batch_init(s, (BatchState **)&s->batch));
    BatchState *B = (BatchState *)s->batch;
    if (!B->own) RSV_CUDA_TRY(cudaStreamCreateWithFlags(&B->own, cudaStreamNonBlocking));
    StreamSwap swap(s, B->own);
    if (!B->tuned) {
        RSV_CUDA_TRY(spmv_autotune(A));
        B->tuned = true;
    }
    const BatchDev d = B->dv;
    RSV_CUDA_TRY(cudaEventRecord(s->e0, s->st));
    const double *db = b;
    double *dx = x;
    if (!on_device) {
        RSV_CUDA_TRY(cudaMemcpyAsync(s->d_b, b, sizeof(double) * n, cudaMemcpyHostToDevice, s->st));
        RSV_CUDA_TRY(cudaMemcpyAsync(s->d_x, x, sizeof(double) * n, cudaMemcpyHostToDevice, s->st));
        db = s->d_b;
        dx = s->d_x;
    }
    // per-system state from scratch; ||b|| per system
    RSV_CUDA_TRY(cudaMemsetAsync(d.done, 0, sizeof(int) * (6 * nsys + 4), s->st));
    RSV_CUDA_TRY(cudaMemsetAsync(d.scale, 0, sizeof(double) * nsys, s->st));
    RSV_CUDA_TRY(seg_dot<double>(s, B, db, db, (const double *)nullptr, d.bnorm, nullptr, 1, 0, nullptr));
    if (!s->mixed) {
        // FP64: BiCGSTAB on A x = b from the given x (solve for the correction of b - A x0)
        double *r0 = s->r64;
        RSV_CUDA_TRY(cudaMemcpyAsync(r0, db, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->st));
        RSV_CUDA_TRY(launch_spmv_f64(A, -1.0, dx, 1.0, r0, nullptr, &s->ds->status, (unsigned long long)s->p.watchdog * 1000ull));
        RSV_TRY(bicg_inner<double>(s, B, r0, (double *)B->xin, s->p.rtol, 0));
        RSV_CUDA_TRY(launch_axpby<double>(s->st, n, 1.0, (const double *)B->xin, 1.0, dx, dx));
    } else {
        double *rn = d.red + 7 * nsys;  // outer residual norms
        for (int outer = 0; outer <= s->p.max_outer; ++outer) {
            RSV_CUDA_TRY(cudaMemcpyAsync(s->r64, db, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->st));
            RSV_CUDA_TRY(launch_spmv_f64(A, -1.0, dx, 1.0, s->r64, nullptr, &s->ds->status, (unsigned long long)s->p.watchdog * 1000ull));
            RSV_CUDA_TRY(seg_dot<double>(s, B, s->r64, s->r64, (const double *)nullptr, rn, nullptr, 1, 0, nullptr));
            count_launches(1);
            b_outer_check<<<sgrid(nsys), 128, 0, s->st>>>(d, nsys, s->p.rtol, rn, s->p.max_outer, s->p.maxit);
            // all finished?
            count_launches(1);
            BatchDev od = d;
            od.done = d.outer;  // count the systems the outer loop has finished
            b_count_done<<<1, 256, 0, s->st>>>(od, nsys);
            RSV_CUDA_TRY(cudaMemcpyAsync(B->h_ndone, d.ndone, sizeof(int), cudaMemcpyDeviceToHost, s->st));
            RSV_CUDA_TRY(cudaStreamSynchronize(s->st));
            if (*B->h_ndone >= nsys) break;
            count_launches(2);
            b_scaled_copy<float><<<B->nitems, kSegThreads, 0, s->st>>>(B->items, d, s->r64, rn, (float *)B->rin);
            b_bump_outer<<<sgrid(nsys), 128, 0, s->st>>>(d, nsys);
            RSV_TRY(bicg_inner<float>(s, B, (const float *)B->rin, (float *)B->xin, s->p.inner_rtol, 1));
            count_launches(1);
            b_add_scaled<<<B->nitems, kSegThreads, 0, s->st>>>(B->items, d, (const float *)B->xin, rn, dx);
            RSV_CUDA_TRY(cudaGetLastError());
        }
    }
    // FP64 true residual per system
    double *rn = d.red + 7 * nsys;
    RSV_CUDA_TRY(cudaMemcpyAsync(s->r64, db, sizeof(double) * n, cudaMemcpyDeviceToDevice, s->st));
    RSV_CUDA_TRY(launch_spmv_f64(A, -1.0, dx, 1.0, s->r64, nullptr, &s->ds->status, (unsigned long long)s->p.watchdog * 1000ull));
    RSV_CUDA_TRY(seg_dot<double>(s, B, s->r64, s->r64, (const double *)nullptr, rn, nullptr, 1, 0, nullptr));
    std::vector<double> h_rn(nsys), h_bn(nsys), h_outer(nsys);
    std::vector<int> h_iters(nsys), h_status(nsys);
    RSV_CUDA_TRY(cudaMemcpyAsync(h_rn.data(), rn, sizeof(double) * nsys, cudaMemcpyDeviceToHost, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(h_bn.data(), d.bnorm, sizeof(double) * nsys, cudaMemcpyDeviceToHost, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(h_outer.data(), d.scale, sizeof(double) * nsys, cudaMemcpyDeviceToHost, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(h_iters.data(), d.iters, sizeof(int) * nsys, cudaMemcpyDeviceToHost, s->st));
    RSV_CUDA_TRY(cudaMemcpyAsync(h_status.data(), d.status, sizeof(int) * nsys, cudaMemcpyDeviceToHost, s->st));
    if (!on_device) RSV_CUDA_TRY(cudaMemcpyAsync(x, s->d_x, sizeof(double) * n, cudaMemcpyDeviceToHost, s->st));
    RSV_CUDA_TRY(cudaEventRecord(s->e1, s->st));
    RSV_CUDA_TRY(cudaStreamSynchronize(s->st));
    float ms = 0.f;
    RSV_CUDA_TRY(cudaEventElapsedTime(&ms, s->e0, s->e1));
    rsv_status worst = RSV_OK;
    for (int q = 0; q < nsys; ++q) {
        const double rel = h_bn[q] > 0 ? h_rn[q] / h_bn[q] : h_rn[q];
        int st = h_status[q];
        if (st == RSV_OK && !(rel <= s->p.rtol || h_rn[q] <= s->p.atol)) st = RSV_ENOCONV;
        if (st == RSV_EBREAKDOWN && (rel <= s->p.rtol)) st = RSV_OK;
        if (infos) {
            infos[q].iters = h_iters[q];
            infos[q].restarts = 0;
            infos[q].outer_iters = (int)h_outer[q];
            infos[q].status = st;
            infos[q].true_relres = rel;
            infos[q].ms_setup = s->ms_setup;
            infos[q].ms_solve = ms;
            infos[q].fallback_iter = -1;
        }
        if (st != RSV_OK && worst == RSV_OK) worst = (rsv_status)st;
    }
    return worst;
}

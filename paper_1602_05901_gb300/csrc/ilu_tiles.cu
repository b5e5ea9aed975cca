// Block ILU(0) triangular sweeps as one persistent launch per sweep.
//
// The forward sweep y_c = D_c^{-1} (r_c - A_{c,-z} y_{-z} - A_{c,-y} y_{-y} -
// A_{c,-x} y_{-x}) has the i+j+k wavefront as its dependency structure
// (Section "Restricted Additive Schwarz Method": L y = b is solved row by
// row); the backward sweep z_c = y_c - D_c^{-1} (A_{c,+x} z_{+x} + A_{c,+y} z_{+y} +
// A_{c,+z} z_{+z}) is its mirror image.  What bounds a sweep is the chain of
// nx+ny+nz-2 dependent steps, then (on large grids) HBM, then (FP64) the FP64 pipe: one
// warp-wide DFMA occupies a quarter of an SM for 63 cycles (76 with all four busy).
//
// The factor is packed as C_q = -D_c^{-1} A_{c,q}: three 3x3 blocks per cell and sweep.
// A step is then y_c = v_c + C_x y_x + C_y y_y + C_z y_z with v = D^{-1} r formed for the
// whole vector before the sweep (off the chain), and z_c = y_c + C_x z_x + C_y z_y + C_z z_z:
// 27 multiply-adds on the chain instead of 36 and 6 additions, and 27 + 27 + 9 values per cell
// and application instead of 36 + 36.
//
// Instead of one launch per hyperplane, a tile of 8 (j) x 4 (k) pencils walks along x.  Lane
// (a, b) holds pencil (a, b) counted from the corner the sweep starts at, and visits its
// cell i at step s = i + a + b (backward: x is counted from the far end too, so both sweeps
// are the same code on mirrored coordinates).  Its y and z neighbours are the results that lanes
// (a-1, b) and (a, b-1) left one step earlier in a shared-memory array with a halo; the
// halo of the tile's low faces comes from the neighbouring tiles through small edge buffers in
// global memory, indexed by the step at which they are needed.  The buffers hold a
// signalling-NaN sentinel until written (arithmetic never produces one), so a reader that
// finds the sentinel re-reads until the value appears; the wait is bounded by a time limit
// that ends the sweep with RSV_ETIMEOUT.  A published value travels as itself (relaxed stores and
// loads of words that are checked one by one), so no fence is needed.
//
// A tile is one CTA: compute warps that do nothing but the recurrence, an edge warp that
// collects the halo values a window of steps at a time, and a data warp that keeps the factor rows and the input
// vector in a shared-memory ring ahead of them (TMA bulk copies); the two announce their progress by counters.
//   FP32: one compute warp, all three components of a cell per lane.  A step issues about 60 instructions.
//   FP64: three, warp e computing component e of all 32 cells, so a step's products occupy
//   three quarters of an SM for 10 x 63 cycles instead of one for 30 x 63; they exchange results
//   through the array with one barrier per step.
// Measured (one apply = gather + two sweeps; one warp per tile with 36 values per cell and every edge read and
// wait in that warp -> this form):
//   256x8x4 (a lone tile) FP32 155 -> 76 us; 100x100x50 FP32 360 -> 179 us; 256x256x128 FP32 1031 -> 912 us;
//   256x8x4 FP64 958 -> 283 us; 75x61x37 FP64 864 -> 256 us; 128x128x64 FP64 1594 -> 518 us.
// Where a sweep's 85 us go on 100x100x50 in FP32 (169 tiles, times and waits noted by each tile in a build for that;
// noting them adds 0.02 us per step): the last tile starts after 60 us and runs for 24.  Up to there lie 12 hand-offs in j
// and 12 in k, each 8 or 4 steps of the tile before and then 1.0 us until the next tile steps (store, L2, poll, halo); a
// lone tile steps in 0.13 us, tiles in the thick of the wavefront in 0.16 to 0.2, for each waits about 34 times for its
// neighbours' values, 150 to 500 cycles a time: the edge warp brings at most WIN steps per round trip.  No
// tile waits for the factor or the input.
// Independent FP32 tiles, 4 per SM, stream at 0.83 of the measured HBM rate.  Also measured:
// factor rows by register loads several steps ahead instead of the ring (a lone tile's step 0.36 us instead
// of 0.13: loads in flight share six scoreboards, and a wait on one waits for younger loads); one service warp for
// edges and data (hand-off 3 us); edge windows of 8 and 16 steps (100x100x50: 181 and 219 us against 176) and of 2
// (229 us); L2 prefetches ahead of the ring (no change).
//
// Tiles are processed in order of their distance from the sweep's first plane (backward: reverse order); all of a launch's CTAs are
// co-resident (cooperative launch), and a tile only ever waits for tiles earlier in
// its order, so the waits cannot form a cycle.
#include <algorithm>

#include "common.cuh"

namespace rsv {
namespace {

constexpr int TJ = 8, TK = 4;
constexpr int kTailRows = 16;  // rows behind the last tile's: the edge windows read past a tile's end

template <typename T> struct Bits;
template <> struct Bits<double> {
    using U = unsigned long long;
    static constexpr U SENT = 0xFFF4C0DE5A17E7A1ull;  // signalling NaN
    static constexpr int GS = 1;                      // steps per data group
    static constexpr int WIN = 2;                     // steps per edge window
    static constexpr int RD = 4;                      // steps of results kept (ring of halo'd arrays)
    static constexpr int MIN_NG = 3, MAX_NG = 8;      // groups in the data ring
};
template <> struct Bits<float> {
    using U = unsigned int;
    static constexpr U SENT = 0x7FA5C0DEu;
    static constexpr int GS = 2;
    static constexpr int WIN = 4;
    static constexpr int RD = 16;
    static constexpr int MIN_NG = 3, MAX_NG = 8;
};

// Packed arrays, per step row of a tile:
//   FP32  factor [7][32] float4 (lane's 27 values and a zero), input [32] float4 (value x 3, pad),
//         edges [TK] and [TJ] float4;
//   FP64  factor [3 components][4][32] double2 | [32] double (component e's 9 values), input
//         [4][32] (three components, pad), edges [3][TK] and [3][TJ];
//   both  D^{-1} [9][32] for the transform of the input.
// The pad carries CPR-PF's pressure correction from the input to the output.
template <typename T> struct Row {
    static constexpr int F = sizeof(T) == 4 ? 7 * 32 * 4 : 27 * 32;
    static constexpr int V = 32 * 4;
    static constexpr int EJ = sizeof(T) == 4 ? TK * 4 : TK * 3;
    static constexpr int EK = sizeof(T) == 4 ? TJ * 4 : TJ * 3;
    static constexpr int D = 9 * 32;
};

// Results of one step with their halo: position (b + 1) kHaloW + a + 1; FP32 float4 entries, FP64
// one plane per component.
constexpr int kHaloW = TJ + 1;
constexpr int kHalo = kHaloW * (TK + 1);
template <typename T> constexpr int kSlot = (sizeof(T) == 4 ? 4 : 3) * kHalo;  // values per step

struct Control {      // shared between the warps of a CTA
    int ready;        // steps whose halo is complete
    int loaded;       // steps whose data have landed (one more than the tile's steps once all have)
    int steps;        // steps the compute warps have finished
    int abort;
};

// Shared memory: data ring [NG][GS][F | V ... as factor of GS steps, then their inputs] | result ring | control | barriers
template <typename T> constexpr size_t group_bytes() { return (size_t)Bits<T>::GS * (Row<T>::F + Row<T>::V) * sizeof(T); }
template <typename T> constexpr size_t fixed_bytes() {
    return (size_t)Bits<T>::RD * kSlot<T> * sizeof(T) + sizeof(Control) + Bits<T>::MAX_NG * sizeof(uint64_t);
}
template <typename T> constexpr size_t sweep_smem(int ng) { return ng * group_bytes<T>() + fixed_bytes<T>(); }

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t global_timer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
// Control words: the writer's earlier shared-memory accesses are done when a reader sees the new value.
__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int *p, int v) {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_volatile(const int *p) { return *(volatile const int *)p; }
__device__ __forceinline__ void st_volatile(int *p, int v) { *(volatile int *)p = v; }
// Shared-memory accesses that stay in program order (volatile): the results of a step travel between the
// lanes of one warp as a store followed by loads, and the look-ahead loads have their place behind them.
__device__ __forceinline__ float4 lds4(unsigned p) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p));
    return v;
}
__device__ __forceinline__ double2 lds2d(unsigned p) {
    double2 v;
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(p));
    return v;
}
__device__ __forceinline__ double ldsd(unsigned p) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(p));
    return v;
}
__device__ __forceinline__ void sts4(unsigned p, float x, float y, float z) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(x), "f"(y), "f"(z), "f"(0.f));
}
__device__ __forceinline__ void stsd(unsigned p, double x) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(p), "d"(x)); }
// Predicated stores: a branch around a store costs the step more than the store.
__device__ __forceinline__ void st_if(bool on, float4 *p, float x, float y, float z, float w) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q st.global.v4.f32 [%0], {%1, %2, %3, %4};\n}" ::"l"(p),
                 "f"(x), "f"(y), "f"(z), "f"(w), "r"((unsigned)on));
}
__device__ __forceinline__ void st_if(bool on, float *p, float x) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.f32 [%0], %1;\n}" ::"l"(p), "f"(x), "r"((unsigned)on));
}
__device__ __forceinline__ void st_if(bool on, double *p, double x) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.f64 [%0], %1;\n}" ::"l"(p), "d"(x), "r"((unsigned)on));
}
__device__ __forceinline__ void st_relaxed_if(bool on, float4 *p, float x, float y, float z) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n @q st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};\n}" ::"l"(p),
                 "f"(x), "f"(y), "f"(z), "f"(0.f), "r"((unsigned)on));
}
__device__ __forceinline__ void st_relaxed_if(bool on, double *p, double x) {
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.relaxed.gpu.global.f64 [%0], %1;\n}" ::"l"(p), "d"(x), "r"((unsigned)on));
}
// Two FMAs in one instruction: (a.x b.x + c.x, a.y b.y + c.y).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mov.b64 c, {%6, %7};\n"
        " fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mul.rn.f32x2 d, a, b;\n"
        " mov.b64 {%0, %1}, d;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 lo(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 ld_relaxed(const float4 *p) {
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_relaxed(const double *p) {
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ bool is_sent(double v) {
    return (unsigned long long)__double_as_longlong(v) == Bits<double>::SENT;
}
__device__ __forceinline__ bool is_sent(const float4 &v) {
    return __float_as_uint(v.x) == Bits<float>::SENT || __float_as_uint(v.y) == Bits<float>::SENT ||
           __float_as_uint(v.z) == Bits<float>::SENT;
}

// One halo entry (a cell's three values) on its way from an edge buffer to the result ring.
template <typename T> struct Entry;
template <> struct Entry<float> {
    float4 v;
    __device__ __forceinline__ void load(const float *g, int) { v = ld_relaxed(reinterpret_cast<const float4 *>(g)); }
    __device__ __forceinline__ bool missing() const { return is_sent(v); }
    __device__ __forceinline__ void put_if(bool on, float *slot, int pos) const {
        asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %4, 0;\n @q st.shared.v4.f32 [%0], {%1, %2, %3, %3};\n}" ::"r"(
                         smem_u32(slot) + pos * 16),
                     "f"(v.x), "f"(v.y), "f"(v.z), "r"((unsigned)on));
    }
};
template <> struct Entry<double> {
    double v[3];
    __device__ __forceinline__ void load(const double *g, int plane) {
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = ld_relaxed(g + c * plane);
    }
    __device__ __forceinline__ bool missing() const { return is_sent(v[0]) || is_sent(v[1]) || is_sent(v[2]); }
    __device__ __forceinline__ void put_if(bool on, double *slot, int pos) const {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.shared.f64 [%0], %1;\n}" ::"r"(
                             smem_u32(slot) + (c * kHalo + pos) * 8),
                         "d"(v[c]), "r"((unsigned)on));
    }
};

template <typename T>
struct SweepArgs {
    int nT, NG;                // tiles of all grids; groups in the data ring
    const TileSys *tsys;       // per grid
    const int *tile_sys;       // position -> grid
    const int64_t *tile_row0;  // position -> first step row of the tile in the packed arrays
    const int2 *order;         // position -> tile (J, K) inside its grid
    const int *pos_of;         // grid's poff + J * nTK + K -> position
    const T *F;          // factor rows
    const T *V;          // input vector in tile order
    T *Vnext;            // forward: y in the backward sweep's tile order; backward: null
    T *z;                // backward: output in natural order; forward: null
    T *EJ, *EK;          // edge buffers this sweep publishes and reads
    int has_add;         // the pads hold a correction
    const int *done;
    const int *frozen;   // per grid: its tiles are skipped (null: none)
    int *status;
    unsigned long long timeout_ns;
    // Whether tile t of the sweep's order is skipped.
    __device__ __forceinline__ bool skip(bool fwd, int t) const { return frozen && frozen[tile_sys[fwd ? t : nT - 1 - t]]; }
};

// A tile of a sweep, seen from the corner the sweep starts at.
struct Tile {
    int nx, Sp, S;
    int pj, pk;          // positions of the tiles before this one in j and k (-1: none)
    int64_t row0, rowj, rowk;
    int64_t cell;        // this lane's pencil: its first cell visited is at cell, the next at cell +- 1
    bool jk_ok;          // the pencil exists
};
template <typename T, bool FWD>
__device__ __forceinline__ Tile tile_of(const SweepArgs<T> &P, int t, int a, int b) {
    const int tt = FWD ? t : (P.nT - 1 - t);
    const TileSys G = P.tsys[P.tile_sys[tt]];
    const int2 JK = P.order[tt];
    Tile r;
    r.nx = G.nx;
    r.S = G.S;
    r.Sp = G.Sp;
    const int dj = FWD ? -1 : 1;
    const int J = JK.x + dj, K = JK.y + dj;
    r.pj = J >= 0 && J < G.nTJ ? P.pos_of[G.poff + J * G.nTK + JK.y] : -1;
    r.pk = K >= 0 && K < G.nTK ? P.pos_of[G.poff + JK.x * G.nTK + K] : -1;
    r.row0 = P.tile_row0[tt];
    r.rowj = r.pj >= 0 ? P.tile_row0[r.pj] : 0;
    r.rowk = r.pk >= 0 ? P.tile_row0[r.pk] : 0;
    const int j = JK.x * TJ + (FWD ? a : TJ - 1 - a), k = JK.y * TK + (FWD ? b : TK - 1 - b);
    r.jk_ok = j < G.ny && k < G.nz;
    r.cell = G.cell0 + ((int64_t)k * G.ny + j) * G.nx + (FWD ? 0 : G.nx - 1);
    return r;
}

// The data warp of a tile (one lane): keeps the ring of data groups full and announces the steps that have
// landed.  group0: groups the ring has carried before this tile.  When a wait runs out, or another
// warp gave up, it raises ctl->abort; it returns with no copy in flight.
template <typename T>
__device__ void feed_tile(const SweepArgs<T> &P, const Tile &tl, T *ring, Control *ctl, uint64_t *full, int group0,
                          uint64_t deadline) {
    using R = Row<T>;
    using B = Bits<T>;
    constexpr int GSIZE = B::GS * (R::F + R::V);
    const int ngr = tl.Sp / B::GS;
    const T *Fp = P.F + tl.row0 * R::F, *Vp = P.V + tl.row0 * R::V;
    int issued = 0, landed = 0;
    int si = group0 % P.NG, sl = si;  // ring stages of the next group to issue and to land
    unsigned parity = (group0 / P.NG) & 1, spins = 0;
    uint64_t limit = deadline;
    bool failed = false;
    while (landed < (failed ? issued : ngr)) {
        if (!failed && issued < ngr && (issued - P.NG + 1) * B::GS <= ld_acquire(&ctl->steps)) {
            T *dst = ring + (size_t)si * GSIZE;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&full[si])),
                         "r"((unsigned)(GSIZE * sizeof(T)))
                         : "memory");
            tma_load_1d(dst, Fp, B::GS * R::F * sizeof(T), &full[si]);
            tma_load_1d(dst + B::GS * R::F, Vp, B::GS * R::V * sizeof(T), &full[si]);
            Fp += B::GS * R::F;
            Vp += B::GS * R::V;
            if (++si == P.NG) si = 0;
            ++issued;
            spins = 0;
        }
        if (landed < issued && mbar_test(&full[sl], parity)) {
            if (++sl == P.NG) {
                sl = 0;
                parity ^= 1u;
            }
            ++landed;
            st_release(&ctl->loaded, landed == ngr ? tl.Sp + 1 : landed * B::GS);
            spins = 0;
        } else if ((++spins & 63u) == 0) {
            if (failed) {
                if (global_timer() > limit) break;
            } else if (ld_acquire(&ctl->abort) || global_timer() > deadline) {
                failed = true;
                st_release(&ctl->abort, 1);
                limit = global_timer() + 1000000000ull;  // copies in flight land first (bounded)
            }
        }
    }
}

// The edge warp of a tile: collects the halo of a window of steps from the edge buffers, hands over those that
// have arrived and announces them.
template <typename T>
__device__ void fetch_edges(const SweepArgs<T> &P, const Tile &tl, T *results, Control *ctl, uint64_t deadline) {
    using R = Row<T>;
    using B = Bits<T>;
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // lanes 0..TK-1 collect the j halo, lanes 8..8+TJ-1 the k halo
    const bool jl = lane < TK, kl = lane >= 8 && lane < 8 + TJ;
    const int off = jl ? lane : lane - 8;  // the consuming lane's a + b
    const bool exists = __shfl_sync(ALL, (int)tl.jk_ok, jl ? lane * 8 : (lane - 8) & 31) != 0;
    const bool on = exists && ((jl && tl.pj >= 0) || (kl && tl.pk >= 0));
    constexpr int E = sizeof(T) == 4 ? 4 : 1;  // values per entry in a buffer row
    const T *g = jl ? P.EJ + tl.rowj * R::EJ + off * E : P.EK + tl.rowk * R::EK + off * E;
    const int rstep = jl ? R::EJ : R::EK, plane = jl ? TK : TJ;
    const int hp = jl ? (off + 1) * kHaloW : off + 1;  // halo position
    int q0 = 0;
    unsigned spins = 0;
    while (q0 < tl.Sp) {
        const int room = ld_volatile(&ctl->steps) + B::RD;  // the halo of step q goes to the slot of step q - 1, last read at step q - RD
        Entry<T> en[B::WIN];
#pragma unroll
        for (int w = 0; w < B::WIN; ++w)
            if (on) en[w].load(g + w * rstep, plane);
        // leading steps of the window that are complete in every lane (branch-free: this loop's length is most of
        // what a hand-off costs)
        int n = 0;
        bool more = true;
#pragma unroll
        for (int w = 0; w < B::WIN; ++w) {
            more = more && !(on && (unsigned)(q0 + w - off) < (unsigned)tl.nx && en[w].missing());
            n += more;
        }
        // room, too, as the lane that saw the fewest steps: the lanes read the counter one by one
        n = min(__reduce_min_sync(ALL, min(n, room - q0)), tl.Sp - q0);
#pragma unroll
        for (int w = 0; w < B::WIN; ++w)
            en[w].put_if(w < n && on && (unsigned)(q0 + w - off) < (unsigned)tl.nx,
                         results + ((q0 + w - 1) & (B::RD - 1)) * kSlot<T>, hp);
        if (n > 0) {
            __syncwarp();
            q0 += n;
            g += n * rstep;
            if (lane == 0) st_release(&ctl->ready, q0);
            spins = 0;
        } else if ((++spins & 7u) == 0 && __any_sync(ALL, ld_acquire(&ctl->abort) != 0 || global_timer() > deadline)) {
            if (lane == 0) st_release(&ctl->abort, 1);
            break;
        }
    }
}

// A compute warp's wait for the halo of step s and the data of the step behind it: returns the number of steps
// that may run, or 0 when the time is up or another warp gave up (the same for the whole warp).
__device__ __forceinline__ int wait_step(Control *ctl, int s, uint64_t deadline) {
    unsigned spins = 0;
    for (;;) {
        // the lanes read one by one, so the counters may move between them: the least of what they saw
        const int n = __reduce_min_sync(0xffffffffu, min(ld_acquire(&ctl->ready), ld_acquire(&ctl->loaded) - 1));
        if (s < n) return n;
        if ((++spins & 63u) == 0 && __any_sync(0xffffffffu, ld_acquire(&ctl->abort) != 0 || global_timer() > deadline))
            return 0;
    }
}

// Shared memory of a CTA.
template <typename T> struct Smem {
    T *ring, *results;
    Control *ctl;
    uint64_t *full;
    __device__ __forceinline__ Smem(unsigned char *raw, int ng) {
        ring = reinterpret_cast<T *>(raw);
        results = ring + (size_t)ng * Bits<T>::GS * (Row<T>::F + Row<T>::V);
        full = reinterpret_cast<uint64_t *>(results + Bits<T>::RD * kSlot<T>);
        ctl = reinterpret_cast<Control *>(full + Bits<T>::MAX_NG);
    }
    // Once per CTA.
    __device__ __forceinline__ void init(int ng) const {
        if (threadIdx.x) return;
        for (int q = 0; q < ng; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[q])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        ctl->abort = 0;
    }
    // Before each tile, by the whole CTA; false when a warp gave up.  Faces without a producer read zeros.
    __device__ __forceinline__ bool begin(const Tile &tl) const {
        __syncthreads();  // every warp is done with the previous tile
        if (ld_volatile(&ctl->abort)) return false;
        for (int q = threadIdx.x; q < Bits<T>::RD * kSlot<T>; q += blockDim.x) results[q] = T(0);
        if (threadIdx.x == 0) {
            ctl->ready = tl.pj < 0 && tl.pk < 0 ? tl.Sp : 0;
            ctl->loaded = ctl->steps = 0;
        }
        __syncthreads();
        return true;
    }
};

// FP32: warp 0 computes, warp 1 fetches the edges, warp 2 the data.
//
// The products of a cell's components 0 and 1 of each neighbour are packed FMAs (fma.rn.f32x2): a step takes 9
// of them and 9 scalar ones.  The factor row is stored in the order the packed operands need (put_row).
template <bool FWD>
__global__ void __launch_bounds__(96, 5) ilu_sweep_f32(SweepArgs<float> P) {
    using R = Row<float>;
    using B = Bits<float>;
    constexpr int GSIZE = B::GS * (R::F + R::V);
    static_assert(B::GS == 2, "the two steps of a group alternate the look-ahead registers");
    if (P.done && *(volatile const int *)P.done) return;
    extern __shared__ __align__(128) unsigned char smem[];
    const Smem<float> sm(smem, P.NG);
    Control *ctl = sm.ctl;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int a = lane & 7, b = lane >> 3;
    const uint64_t deadline = global_timer() + P.timeout_ns;
    sm.init(P.NG);
    int group0 = 0;  // data groups of the tiles before this one
    for (int t = blockIdx.x; t < P.nT; t += gridDim.x) {
        if (P.skip(FWD, t)) continue;
        const Tile tl = tile_of<float, FWD>(P, t, a, b);
        if (!sm.begin(tl)) break;
        const int ngr = tl.Sp / B::GS;
        if (warp == 1) {
            if (tl.pj >= 0 || tl.pk >= 0) fetch_edges<float>(P, tl, sm.results, ctl, deadline);
        } else if (warp == 2) {
            if (lane == 0) feed_tile<float>(P, tl, sm.ring, ctl, sm.full, group0, deadline);
        } else {
            const unsigned res = smem_u32(sm.results) + ((b + 1) * kHaloW + a + 1) * 16;
            // this tile's edge entries: a result of step s is needed TJ - 1 (TK - 1) steps earlier in the next tile's count
            float4 *pubj = reinterpret_cast<float4 *>(P.EJ + (tl.row0 - (TJ - 1)) * R::EJ) + b;
            float4 *pubk = reinterpret_cast<float4 *>(P.EK + (tl.row0 - (TK - 1)) * R::EK) + a;
            // forward: y goes to row S - 1 - s of the backward order, where this lane's pencil is lane 31 - lane
            float4 *yout = FWD ? reinterpret_cast<float4 *>(P.Vnext + (tl.row0 + tl.S - 1) * R::V) + (31 - lane) : nullptr;
            float *zout = FWD ? nullptr : P.z + 3 * (tl.cell + (a + b));  // cell of step 0 (before the pencil's start)
            const unsigned nx = tl.jk_ok ? tl.nx : 0;
            const bool pj = a == TJ - 1, pk = b == TK - 1;
            int i = -(a + b);  // cells visited so far; in the grid when 0 <= i < nx
            float2 p01 = make_float2(0.f, 0.f);  // the lane's previous result
            float p2 = 0.f;
            float4 f[2][7], v[2];
            const unsigned ring0 = smem_u32(sm.ring) + lane * 16, ring1 = ring0 + P.NG * GSIZE * 4;
            unsigned stage = ring0 + (group0 % P.NG) * (GSIZE * 4);
            auto fetch = [&](float4(&fo)[7], float4 &vo, int u) {
#pragma unroll
                for (int q = 0; q < 7; ++q) fo[q] = lds4(stage + (u * 7 + q) * 512);
                vo = lds4(stage + (B::GS * 7 + u) * 512);
            };
            // One step from the results at `in` to those at `out`, its data in f, v.
            auto step = [&](const float4(&f)[7], const float4 &v, const float4 &J, const float4 &K, unsigned out, int u) {
                const bool valid = (unsigned)i < nx;
                const float2 J01 = make_float2(J.x, J.y), K01 = make_float2(K.x, K.y);
                float2 s0 = mul2(lo(f[0]), p01), s1 = mul2(hi(f[1]), p01), s2 = mul2(lo(f[3]), p01);
                float r0 = f[4].z * p2, r1 = f[5].y * p2, r2 = f[6].x * p2;
                s0 = fma2(hi(f[0]), J01, s0);
                s1 = fma2(lo(f[2]), J01, s1);
                s2 = fma2(hi(f[3]), J01, s2);
                r0 = fmaf(f[4].w, J.z, r0);
                r1 = fmaf(f[5].z, J.z, r1);
                r2 = fmaf(f[6].y, J.z, r2);
                s0 = fma2(lo(f[1]), K01, s0);
                s1 = fma2(hi(f[2]), K01, s1);
                s2 = fma2(lo(f[4]), K01, s2);
                r0 = fmaf(f[5].x, K.z, r0);
                r1 = fmaf(f[5].w, K.z, r1);
                r2 = fmaf(f[6].z, K.z, r2);
                // v last: starting the sums from it costs a rounding at its magnitude per product (error of
                // an apply against 64 bits 9e-8 instead of 6e-8)
                r0 = v.x + ((r0 + s0.y) + s0.x);
                r1 = v.y + ((r1 + s1.y) + s1.x);
                r2 = v.z + ((r2 + s2.y) + s2.x);
                p01 = make_float2(valid ? r0 : 0.f, valid ? r1 : 0.f);
                p2 = valid ? r2 : 0.f;
                sts4(out, p01.x, p01.y, p2);
                __syncwarp();
                st_relaxed_if(valid && pj, pubj + u * TK, r0, r1, r2);
                st_relaxed_if(valid && pk, pubk + u * TJ, r0, r1, r2);
                if (FWD) {
                    st_if(valid, yout - u * 32, r0, r1, r2, v.w);
                } else {
                    st_if(valid, zout - 3 * u, r0 + v.w);
                    st_if(valid, zout - 3 * u + 1, r1);
                    st_if(valid, zout - 3 * u + 2, r2);
                }
                ++i;
            };
            int n = wait_step(ctl, 0, deadline);
            if (n) fetch(f[0], v[0], 0);
            unsigned prev = res + (B::RD - 1) * kHalo * 16;  // results of the step before
            for (int s = 0; n && s < tl.Sp; s += 2) {
                const unsigned out = res + (s & (B::RD - 1)) * (kHalo * 16);
                if (s >= n && !(n = wait_step(ctl, s, deadline))) break;
                {
                    const float4 J = lds4(prev - 16), K = lds4(prev - kHaloW * 16);
                    fetch(f[1], v[1], 1);
                    step(f[0], v[0], J, K, out, 0);
                }
                if (s + 1 >= n && !(n = wait_step(ctl, s + 1, deadline))) break;
                {
                    const float4 J = lds4(out - 16), K = lds4(out - kHaloW * 16);
                    stage += GSIZE * 4;
                    if (stage == ring1) stage = ring0;
                    fetch(f[0], v[0], 0);  // behind the tile's last group: a stale stage, unused
                    prev = out + kHalo * 16;
                    step(f[1], v[1], J, K, prev, 1);
                }
                if (lane == 0) st_volatile(&ctl->steps, s + 2);  // the group's values are in registers and used
                pubj += 2 * TK;
                pubk += 2 * TJ;
                if (FWD)
                    yout -= 2 * 32;
                else
                    zout -= 6;
            }
            if (!n && lane == 0) st_release(&ctl->abort, 1);
        }
        group0 += ngr;
    }
    __syncthreads();
    if (threadIdx.x == 0 && ld_volatile(&ctl->abort)) atomicCAS(P.status, 0, (int)RSV_ETIMEOUT);
}

// FP64: three compute warps, one per component; the edge warp on the fourth quarter of the SM; the data warp.
template <bool FWD>
__global__ void __launch_bounds__(160) ilu_sweep_f64(SweepArgs<double> P) {
    using R = Row<double>;
    using B = Bits<double>;
    constexpr int GSIZE = R::F + R::V;
    static_assert(B::GS == 1, "a data group is one step");
    if (P.done && *(volatile const int *)P.done) return;
    extern __shared__ __align__(128) unsigned char smem[];
    const Smem<double> sm(smem, P.NG);
    Control *ctl = sm.ctl;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // component (3: edges, 4: data); which quarter of the SM has none differs between CTAs that share an SM
    const int e = warp < 4 ? (warp + blockIdx.x / 152) & 3 : 4;
    const int a = lane & 7, b = lane >> 3;
    const uint64_t deadline = global_timer() + P.timeout_ns;
    sm.init(P.NG);
    int group0 = 0;
    for (int t = blockIdx.x; t < P.nT; t += gridDim.x) {
        if (P.skip(FWD, t)) continue;
        const Tile tl = tile_of<double, FWD>(P, t, a, b);
        if (!sm.begin(tl)) break;
        if (e == 3) {
            if (tl.pj >= 0 || tl.pk >= 0) fetch_edges<double>(P, tl, sm.results, ctl, deadline);
        } else if (e == 4) {
            if (lane == 0) feed_tile<double>(P, tl, sm.ring, ctl, sm.full, group0, deadline);
        } else {
            const unsigned res = smem_u32(sm.results) + ((b + 1) * kHaloW + a + 1) * 8;
            double *pubj = P.EJ + (tl.row0 - (TJ - 1)) * R::EJ + e * TK + b;
            double *pubk = P.EK + (tl.row0 - (TK - 1)) * R::EK + e * TJ + a;
            double *yout = FWD ? P.Vnext + (tl.row0 + tl.S - 1) * R::V + (31 - lane) : nullptr;
            double *zout = FWD ? nullptr : P.z + 3 * (tl.cell + (a + b)) + e;
            const unsigned nx = tl.jk_ok ? tl.nx : 0;
            const bool pj = a == TJ - 1, pk = b == TK - 1;
            const bool pads = P.has_add && e == 0;  // warp 0 carries the pads
            int i = -(a + b);
            double2 f[2][4];
            double f8[2], v[2], pad[2] = {0.0, 0.0};
            double zlate = 0.0;  // backward, warp 0 with pads: the step before's z_c[0] + p_c, stored one step late
            bool late = false;
            const unsigned ring0 = smem_u32(sm.ring), ring1 = ring0 + P.NG * GSIZE * 8;
            unsigned stage = ring0 + (group0 % P.NG) * (GSIZE * 8);
            auto fetch = [&](int u) {
#pragma unroll
                for (int q = 0; q < 4; ++q) f[u][q] = lds2d(stage + e * 2304 + q * 512 + lane * 16);
                f8[u] = ldsd(stage + e * 2304 + 2048 + lane * 8);
                v[u] = ldsd(stage + R::F * 8 + e * 256 + lane * 8);
                if (pads) pad[u] = ldsd(stage + R::F * 8 + 768 + lane * 8);
            };
            int n = wait_step(ctl, 0, deadline);
            bool ok = n > 0, stop = false;
            fetch(0);
            unsigned prev = res + (B::RD - 1) * kSlot<double> * 8;
            for (int s0 = 0; !stop && s0 < tl.Sp; s0 += 2) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int s = s0 + u;
                    if (s >= n && ok) {
                        n = wait_step(ctl, s, deadline);
                        ok = n > 0;
                    }
                    const unsigned out = res + (s & (B::RD - 1)) * (kSlot<double> * 8);
                    // the other two components' own results, then the neighbours'
                    double x[9];
#pragma unroll
                    for (int c = 0; c < 3; ++c) x[c] = ldsd(prev + c * (kHalo * 8));
#pragma unroll
                    for (int c = 0; c < 3; ++c) x[3 + c] = ldsd(prev + c * (kHalo * 8) - 8);
#pragma unroll
                    for (int c = 0; c < 3; ++c) x[6 + c] = ldsd(prev + c * (kHalo * 8) - kHaloW * 8);
                    stage += GSIZE * 8;
                    if (stage == ring1) stage = ring0;
                    fetch(u ^ 1);
                    const bool valid = (unsigned)i < nx;
                    double r = f[u][0].x * x[0];
                    r = fma(f[u][0].y, x[1], r);
                    r = fma(f[u][1].x, x[2], r);
                    r = fma(f[u][1].y, x[3], r);
                    r = fma(f[u][2].x, x[4], r);
                    r = fma(f[u][2].y, x[5], r);
                    r = fma(f[u][3].x, x[6], r);
                    r = fma(f[u][3].y, x[7], r);
                    r = v[u] + fma(f8[u], x[8], r);  // v last: as in FP32
                    if (!FWD) st_if(late, zout + 3, zlate);
                    stsd(out + e * (kHalo * 8), valid ? r : 0.0);
                    st_relaxed_if(valid && pj, pubj, r);
                    st_relaxed_if(valid && pk, pubk, r);
                    if (u == 0) {
                        asm volatile("barrier.cta.sync 1, 96;" ::: "memory");
                    } else {
                        // also: did any warp's wait run out in these two steps
                        unsigned any;
                        asm volatile(
                            "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, 96, p;\n"
                            " selp.u32 %0, 1, 0, q;\n}"
                            : "=r"(any)
                            : "r"((unsigned)!ok)
                            : "memory");
                        stop = any != 0;
                    }
                    if (e == 0 && lane == 0) st_volatile(&ctl->steps, s + 1);  // every warp is past the step
                    if (FWD) {
                        st_if(valid, yout + e * 32, r);
                        if (pads) st_if(valid, yout + 96, pad[u]);
                        yout -= R::V;
                    } else {
                        st_if(valid && !pads, zout, r);
                        if (pads) {
                            late = valid;
                            zlate = r + pad[u];
                        }
                        zout -= 3;
                    }
                    ++i;
                    pubj += R::EJ;
                    pubk += R::EK;
                    prev = out;
                }
            }
            if (!FWD) st_if(late && !stop, zout + 3, zlate);
            if (stop && lane == 0) st_release(&ctl->abort, 1);
        }
        group0 += tl.Sp;
    }
    __syncthreads();
    if (threadIdx.x == 0 && ld_volatile(&ctl->abort)) atomicCAS(P.status, 0, (int)RSV_ETIMEOUT);
}

// Storage of a cell's factor row: value n = 9 e + 3 q + f is C_q[e][f], q = 0 (x), 1 (y), 2 (z).  FP32: the
// pairs f = 0, 1 of (e, q) = (0, 0), (0, 1), ..., (2, 2), then f = 2 of the same.
__device__ __forceinline__ void put_row(float *F, int64_t row, int lane, const float c[27]) {
    float w[28];
#pragma unroll
    for (int n = 0; n < 9; ++n) {
        w[2 * n] = c[3 * n];
        w[2 * n + 1] = c[3 * n + 1];
        w[18 + n] = c[3 * n + 2];
    }
    w[27] = 0.f;
    float4 *o = reinterpret_cast<float4 *>(F + row * Row<float>::F) + lane;
#pragma unroll
    for (int q = 0; q < 7; ++q) o[q * 32] = make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}
__device__ __forceinline__ void put_row(double *F, int64_t row, int lane, const double c[27]) {
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        double *o = F + row * Row<double>::F + e * 288;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            reinterpret_cast<double2 *>(o)[q * 32 + lane] = make_double2(c[9 * e + 2 * q], c[9 * e + 2 * q + 1]);
        o[256 + lane] = c[9 * e + 8];
    }
}

// One entry -sum_m d[m] A[m] of a packed block.  FP64, or rounded to FP32 from a double-float sum: d as two
// floats (48 bits), exact products and two-sums, about 44 bits before the one rounding; in FP64 the products and
// conversions are what bounded the packing (128x128x64: 799 us with 36 unmultiplied values, 589 us with
// FP64 products, 152 us now).
template <typename T> struct Row3;  // three entries of a row of D^{-1}
template <> struct Row3<double> {
    double d[3];
    __device__ __forceinline__ explicit Row3(const double *p) : d{p[0], p[1], p[2]} {}
    __device__ __forceinline__ double times(const double *A) const {
        return -(d[0] * A[0] + d[1] * A[3] + d[2] * A[6]);
    }
    __device__ __forceinline__ double at(int m) const { return d[m]; }
};
template <> struct Row3<float> {
    float h[3], l[3];
    __device__ __forceinline__ explicit Row3(const double *p) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            h[m] = round_float(p[m]);
            l[m] = round_float(p[m] - exact_double(h[m]));
        }
    }
    __device__ __forceinline__ float times(const float *A) const {
        float hi = 0.f, lo = 0.f;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const float p = __fmul_rn(h[m], A[3 * m]);
            const float e = __fmaf_rn(l[m], A[3 * m], __fmaf_rn(h[m], A[3 * m], -p));  // h A = p + its rounding; + l A
            const float s = __fadd_rn(hi, p), bp = __fsub_rn(s, hi);
            lo = __fadd_rn(lo, __fadd_rn(e, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(p, bp))));
            hi = s;
        }
        return -__fadd_rn(hi, lo);
    }
    __device__ __forceinline__ float at(int m) const { return h[m]; }
};

// The packed factor of both sweeps and D^{-1} in tile order.  One thread per (tile, step, lane) of the
// forward order; its cell sits at step S - 1 - s, lane 31 - lane of the backward order.  Block values come
// from `v` (FP64, or the FP32 copy for mixed precision), D^{-1} from the FP64 factor.  Entries without a cell
// are never read as values.
template <typename T>
__global__ void __launch_bounds__(256) pack_tiles(const TileSys *__restrict__ tsys, const int *__restrict__ tile_sys,
                           const int64_t *__restrict__ tile_row0, const int2 *__restrict__ order,
                           const int32_t *__restrict__ rp, const T *__restrict__ v,
                           const double *__restrict__ dinv, T *__restrict__ Ff, T *__restrict__ Fb, T *__restrict__ D) {
    const int t = blockIdx.y;
    const TileSys G = tsys[tile_sys[t]];
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = (int)(gid & 31);
    const int s = (int)(gid >> 5);
    const int a = lane & 7, b = lane >> 3;
    const int2 JK = order[t];
    const int i = s - a - b, j = JK.x * TJ + a, k = JK.y * TK + b;
    if (j >= ny || k >= nz || i < 0 || i >= nx) return;
    const int64_t c = G.cell0 + (int64_t)k * nx * ny + (int64_t)j * nx + i;
    const int64_t row = tile_row0[t] + s, rowb = tile_row0[t] + (G.S - 1 - s);
    const Row3<T> d[3] = {Row3<T>(dinv + 9 * c), Row3<T>(dinv + 9 * c + 3), Row3<T>(dinv + 9 * c + 6)};
#pragma unroll
    for (int e = 0; e < 9; ++e) D[row * Row<T>::D + e * 32 + lane] = d[e / 3].at(e % 3);
    // blocks of the row: -z, -y, -x, self, +x, +y, +z (absent faces skipped)
    const bool has[6] = {i > 0, j > 0, k > 0, i < nx - 1, j < ny - 1, k < nz - 1};
    const int before[6] = {has[2] + has[1], has[2], 0, 1, 1 + has[3], 1 + has[3] + has[4]};
    const T *lo = v + 9 * (int64_t)rp[c], *hi = lo + 9 * (has[0] + has[1] + has[2]);
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
        T o[27];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int n = 3 * dir + q;
            T A[9];
            const T *blk = (dir == 0 ? lo : hi) + 9 * before[n];
#pragma unroll
            for (int e = 0; e < 9; ++e) A[e] = has[n] ? blk[e] : T(0);
#pragma unroll
            for (int e = 0; e < 3; ++e)
#pragma unroll
                for (int f = 0; f < 3; ++f) o[9 * e + 3 * q + f] = d[e].times(A + f);
        }
        if (dir == 0)
            put_row(Ff, row, lane, o);
        else
            put_row(Fb, rowb, 31 - lane, o);
    }
}

// Tile-order entry of the sweeps' input: three values and the pad.
__device__ __forceinline__ void put_input(float *V, int64_t row, int lane, const float v[3], float pad, bool) {
    reinterpret_cast<float4 *>(V + row * Row<float>::V)[lane] = make_float4(v[0], v[1], v[2], pad);
}
__device__ __forceinline__ void put_input(double *V, int64_t row, int lane, const double v[3], double pad, bool has) {
    double *o = V + row * Row<double>::V + lane;
    o[0] = v[0];
    o[32] = v[1];
    o[64] = v[2];
    if (has) o[96] = pad;
}
// `rows` rows of an edge buffer (per values each) to the sentinel, by one warp in 16-byte stores.
template <typename T>
__device__ __forceinline__ void reset_rows(T *E, int64_t row, int rows, int per, int lane) {
    constexpr int N = 16 / sizeof(T);
    typename Bits<T>::U w[N];
#pragma unroll
    for (int q = 0; q < N; ++q) w[q] = Bits<T>::SENT;
    uint4 *o = reinterpret_cast<uint4 *>(E + row * per);
    for (int q = lane; q < rows * per / N; q += 32) o[q] = *reinterpret_cast<const uint4 *>(w);
}

// Before a forward sweep: v = D^{-1} r in tile order, and the edge buffers of both sweeps to
// the sentinel.  One thread per (tile, lane) and kGatherSteps consecutive steps:
// its cells are consecutive along x, and all their loads are issued before the
// stores (one load per thread left the gather latency-bound).  The pad
// takes add[c] (or 0).
constexpr int kGatherSteps = 4;
template <typename T>
__global__ void __launch_bounds__(256) gather_tiles(const TileSys *__restrict__ tsys, const int *__restrict__ tile_sys,
                             const int64_t *__restrict__ tile_row0, const int2 *__restrict__ order,
                             const T *__restrict__ r, const T *__restrict__ add, const T *__restrict__ D,
                             T *__restrict__ Vt, T *__restrict__ EJf, T *__restrict__ EKf, T *__restrict__ EJb,
                             T *__restrict__ EKb, const int *frozen) {
    pdl_wait();  // launched with launch_pdl: the previous kernel may still be running
    pdl_trigger();
    using R = Row<T>;
    const int t = blockIdx.y;
    if (frozen && frozen[tile_sys[t]]) return;
    const TileSys G = tsys[tile_sys[t]];
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = (int)(gid & 31);
    const int s0 = (int)(gid >> 5) * kGatherSteps;
    if (s0 >= G.Sp) return;
    const int a = lane & 7, b = lane >> 3;
    const int2 JK = order[t];
    const int j = JK.x * TJ + a, k = JK.y * TK + b;
    const bool jk_ok = j < ny && k < nz;
    const int64_t pencil = G.cell0 + (int64_t)k * nx * ny + (int64_t)j * nx;
    const int64_t row = tile_row0[t] + s0;
    T x[kGatherSteps][4], d[kGatherSteps][9];
    bool ok[kGatherSteps];
#pragma unroll
    for (int u = 0; u < kGatherSteps; ++u) {
        const int i = s0 + u - a - b;
        ok[u] = jk_ok && i >= 0 && i < nx;
        if (ok[u]) {
            const int64_t c = pencil + i;
            x[u][0] = r[3 * c];
            x[u][1] = r[3 * c + 1];
            x[u][2] = r[3 * c + 2];
            x[u][3] = add ? add[c] : T(0);
#pragma unroll
            for (int e = 0; e < 9; ++e) d[u][e] = D[(row + u) * R::D + e * 32 + lane];
        }
    }
    const int rows = min(kGatherSteps, G.Sp - s0);
    reset_rows(EJf, row, rows, R::EJ, lane);
    reset_rows(EKf, row, rows, R::EK, lane);
    reset_rows(EJb, row, rows, R::EJ, lane);
    reset_rows(EKb, row, rows, R::EK, lane);
#pragma unroll
    for (int u = 0; u < kGatherSteps; ++u)
        if (ok[u]) {
            T v[3];
#pragma unroll
            for (int e = 0; e < 3; ++e)
                v[e] = fma(d[u][3 * e + 2], x[u][2], fma(d[u][3 * e + 1], x[u][1], d[u][3 * e] * x[u][0]));
            put_input(Vt, row + u, lane, v, x[u][3], add != nullptr);
        }
}

template <typename T> constexpr const void *sweep_kernel(bool fwd) {
    if constexpr (sizeof(T) == 4)
        return fwd ? (const void *)ilu_sweep_f32<true> : (const void *)ilu_sweep_f32<false>;
    else
        return fwd ? (const void *)ilu_sweep_f64<true> : (const void *)ilu_sweep_f64<false>;
}
template <typename T> constexpr int kSweepThreads = sizeof(T) == 4 ? 96 : 160;

// Gives back what was allocated so far unless `whole` is set: the next setup must not take it for complete.
struct FreeUnlessWhole {
    IluTiles *Tl;
    bool whole = false;
    ~FreeUnlessWhole() {
        if (!whole) free_tiles(Tl);
    }
};

}  // namespace

template <typename T>
cudaError_t tiles_setup(const rsv_mat *A, const double *dinv, IluTiles *Tl) {
    using R = Row<T>;
    cudaError_t e = cudaSuccess;
    if (!Tl->Ff || Tl->elem != (int)sizeof(T)) {
        free_tiles(Tl);
        FreeUnlessWhole guard{Tl};
        // Tiles of every grid in order of TJ J + TK K, the planes its start lies behind the grid's first cell: a
        // CTA that is free takes the tile that can start soonest, in every grid of a batch at once.  (One grid after
        // another left CTAs waiting in the far tiles of the first grids: 24 grids of 16 to 96 cells a side, 220 -> 157 us
        // per sweep.)
        struct Place {
            int key, g, J, K;
        };
        std::vector<TileSys> sys;
        std::vector<Place> places;
        int64_t rows = 0;
        int maxS = 0;
        for (int g = 0; g < A->nsys; ++g) {
            const SysGrid &sg = A->h_sys[g];
            TileSys ts;
            ts.nx = sg.nx;
            ts.ny = sg.ny;
            ts.nz = sg.nz;
            ts.nTJ = (sg.ny + TJ - 1) / TJ;
            ts.nTK = (sg.nz + TK - 1) / TK;
            ts.S = sg.nx + TJ + TK - 2;
            ts.Sp = (ts.S + 1) / 2 * 2;  // the steps are unrolled by two
            ts.cell0 = sg.cell0;
            ts.poff = (int)places.size();
            maxS = std::max(maxS, ts.Sp);
            for (int J = 0; J < ts.nTJ; ++J)
                for (int K = 0; K < ts.nTK; ++K) places.push_back(Place{TJ * J + TK * K, g, J, K});
            sys.push_back(ts);
        }
        std::stable_sort(places.begin(), places.end(), [](const Place &a, const Place &b) { return a.key < b.key; });
        std::vector<int2> order;
        std::vector<int> tile_sys, pos(places.size());
        std::vector<int64_t> row0;
        for (const Place &q : places) {
            pos[sys[q.g].poff + q.J * sys[q.g].nTK + q.K] = (int)order.size();
            order.push_back(make_int2(q.J, q.K));
            tile_sys.push_back(q.g);
            row0.push_back(rows);
            rows += sys[q.g].Sp;
        }
        const int nT = (int)order.size();
        if (nT > 65535) return cudaErrorInvalidConfiguration;  // tiles index blockIdx.y of the pack/gather grids
        Tl->nT = nT;
        Tl->maxS = maxS;
        Tl->rows = rows;
        Tl->elem = (int)sizeof(T);
        const size_t all = (size_t)(rows + kTailRows) * sizeof(T);
        auto alloc = [&](void **p, size_t bytes) {
            if (e == cudaSuccess) e = cudaMalloc(p, std::max<size_t>(bytes, 16));
        };
        alloc(&Tl->Ff, all * R::F);
        alloc(&Tl->Fb, all * R::F);
        alloc(&Tl->D, all * R::D);
        alloc(&Tl->Vf, all * R::V);
        alloc(&Tl->Vb, all * R::V);
        alloc(&Tl->EJf, all * R::EJ);
        alloc(&Tl->EKf, all * R::EK);
        alloc(&Tl->EJb, all * R::EJ);
        alloc(&Tl->EKb, all * R::EK);
        alloc((void **)&Tl->order, sizeof(int2) * nT);
        alloc((void **)&Tl->pos_of, sizeof(int) * nT);
        alloc((void **)&Tl->tile_sys, sizeof(int) * nT);
        alloc((void **)&Tl->tile_row0, sizeof(int64_t) * nT);
        alloc((void **)&Tl->tsys, sizeof(TileSys) * sys.size());
        if (e != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(Tl->order, order.data(), sizeof(int2) * nT, cudaMemcpyHostToDevice, A->stream)) !=
                cudaSuccess ||
            (e = cudaMemcpyAsync(Tl->pos_of, pos.data(), sizeof(int) * nT, cudaMemcpyHostToDevice, A->stream)) !=
                cudaSuccess ||
            (e = cudaMemcpyAsync(Tl->tile_sys, tile_sys.data(), sizeof(int) * nT, cudaMemcpyHostToDevice,
                                 A->stream)) != cudaSuccess ||
            (e = cudaMemcpyAsync(Tl->tile_row0, row0.data(), sizeof(int64_t) * nT, cudaMemcpyHostToDevice,
                                 A->stream)) != cudaSuccess ||
            (e = cudaMemcpyAsync(Tl->tsys, sys.data(), sizeof(TileSys) * sys.size(), cudaMemcpyHostToDevice,
                                 A->stream)) != cudaSuccess ||
            (e = cudaStreamSynchronize(A->stream)) != cudaSuccess)
            return e;
        int dev = 0, sms = 0, most = 0, per_f = 0, per_b = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
        // Groups in the data ring: as many as leave room for every tile to be resident, at most MAX_NG (a
        // deeper ring hides more of the memory latency from a lone tile), at least MIN_NG.
        const int want = std::max(1, (nT + sms - 1) / sms);  // tiles per SM
        const int64_t room = (int64_t)most / want - 1024 - (int64_t)fixed_bytes<T>();
        Tl->ng = (int)std::max<int64_t>(Bits<T>::MIN_NG, std::min<int64_t>(Bits<T>::MAX_NG, room / (int64_t)group_bytes<T>()));
        const size_t smem = Tl->smem = sweep_smem<T>(Tl->ng);
        for (bool fwd : {true, false})
            if ((e = cudaFuncSetAttribute(sweep_kernel<T>(fwd), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)sweep_smem<T>(Bits<T>::MAX_NG))) != cudaSuccess ||
                (e = cudaFuncSetAttribute(sweep_kernel<T>(fwd), cudaFuncAttributePreferredSharedMemoryCarveout,
                                          100)) != cudaSuccess)
                return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_f, sweep_kernel<T>(true), kSweepThreads<T>, smem)) !=
                cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_b, sweep_kernel<T>(false), kSweepThreads<T>, smem)) !=
                cudaSuccess)
            return e;
        Tl->grid = std::max(1, std::min(nT, sms * std::min(per_f, per_b)));
        guard.whole = true;
    }
    const dim3 g((unsigned)((Tl->maxS * 32 + 255) / 256), (unsigned)Tl->nT);
    rsv::count_launches(1);
    const T *v = sizeof(T) == 8 ? (const T *)A->d_v : (const T *)A->d_v32;
    pack_tiles<T><<<g, 256, 0, A->stream>>>(Tl->tsys, Tl->tile_sys, Tl->tile_row0, Tl->order, A->d_rp, v, dinv,
                                            (T *)Tl->Ff, (T *)Tl->Fb, (T *)Tl->D);
    return cudaGetLastError();
}

void free_tiles(IluTiles *Tl) {
    for (void *p : {Tl->Ff, Tl->Fb, Tl->D, Tl->Vf, Tl->Vb, Tl->EJf, Tl->EKf, Tl->EJb, Tl->EKb, (void *)Tl->order,
                    (void *)Tl->pos_of, (void *)Tl->tile_sys, (void *)Tl->tile_row0, (void *)Tl->tsys})
        if (p) cudaFree(p);
    *Tl = IluTiles();
}

template <typename T>
cudaError_t launch_ilu_apply_tiles(const rsv_mat *A, const IluTiles &Tl, const T *r, T *z, const int *done,
                                   int *status, unsigned long long timeout_ns, const T *add0, const int *frozen) {
    rsv::count_launches(3);
    const int groups = (Tl.maxS + kGatherSteps - 1) / kGatherSteps;
    const dim3 g((unsigned)((groups * 32 + 255) / 256), (unsigned)Tl.nT);
    cudaError_t e = launch_pdl(gather_tiles<T>, g, dim3(256), 0, A->stream, Tl.tsys, Tl.tile_sys, Tl.tile_row0,
                               Tl.order, r, add0, (const T *)Tl.D, (T *)Tl.Vf, (T *)Tl.EJf, (T *)Tl.EKf, (T *)Tl.EJb,
                               (T *)Tl.EKb, frozen);
    if (e != cudaSuccess) return e;
    const int has_add = add0 != nullptr;
    SweepArgs<T> f{Tl.nT, Tl.ng, Tl.tsys, Tl.tile_sys, Tl.tile_row0, Tl.order, Tl.pos_of, (const T *)Tl.Ff,
                   (const T *)Tl.Vf, (T *)Tl.Vb, nullptr, (T *)Tl.EJf, (T *)Tl.EKf, has_add, done, frozen, status, timeout_ns};
    SweepArgs<T> bw{Tl.nT, Tl.ng, Tl.tsys, Tl.tile_sys, Tl.tile_row0, Tl.order, Tl.pos_of, (const T *)Tl.Fb,
                    (const T *)Tl.Vb, nullptr, z, (T *)Tl.EJb, (T *)Tl.EKb, has_add, done, frozen, status, timeout_ns};
    void *fa[] = {&f};
    void *ba[] = {&bw};
    e = cudaLaunchCooperativeKernel(sweep_kernel<T>(true), dim3(Tl.grid), dim3(kSweepThreads<T>), fa, Tl.smem,
                                    A->stream);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(sweep_kernel<T>(false), dim3(Tl.grid), dim3(kSweepThreads<T>), ba, Tl.smem,
                                       A->stream);
}

template cudaError_t tiles_setup<double>(const rsv_mat *, const double *, IluTiles *);
template cudaError_t tiles_setup<float>(const rsv_mat *, const double *, IluTiles *);
template cudaError_t launch_ilu_apply_tiles<double>(const rsv_mat *, const IluTiles &, const double *, double *,
                                                    const int *, int *, unsigned long long, const double *,
                                                    const int *);
template cudaError_t launch_ilu_apply_tiles<float>(const rsv_mat *, const IluTiles &, const float *, float *,
                                                   const int *, int *, unsigned long long, const float *,
                                                   const int *);

}  // namespace rsv

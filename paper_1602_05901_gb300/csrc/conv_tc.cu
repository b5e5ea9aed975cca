// 3x3x3 (and 1x1x1) convolutions of the learned pressure stage as implicit
// GEMMs on the tcgen05 tensor cores: BF16 operands staged by TMA, FP32
// accumulators in TMEM, fused epilogues.
//
// Volumes are channels-last BF16, [nz][ny][nx][ld] with the layer's channels
// at the start of each voxel's row of ld values.  A 3x3x3 weight is
// w[co][t][ci] with tap t = 9(dz+1) + 3(dy+1) + (dx+1); the layer computes
// the cross-correlation y[v, co] = sum_t sum_ci w[co,t,ci] x[v + off_t, ci]
// with zeros outside the grid.
//
// Forward (and the input gradient, which is the same correlation with the
// taps mirrored and the channel roles swapped):
//   M = 128 voxels of one tile (a box of bw x bh x bd voxels), N = output
//   channels, K = taps x input channels.  Each K step is one tap and one
//   block of BK channels: TMA copies the tap-shifted box of the input volume
//   (zero fill outside the grid gives the padding exactly) and the matching
//   weight slice; four (BK = 64) or two (BK = 32) MMAs of K = 16 consume it.
// Weight gradient:
//   gw[co][t][ci] = sum_v gy[v, co] x[v + off_t, ci] reduces over voxels, so
//   K = voxels; CTAs split the voxels and write FP32 partial sums that a
//   second kernel adds in a fixed order.  Three forms:
//   * 3x3x3 with rows of at most 128 voxels: whole rows of a plane, the three
//     y taps from one box (conv_wgrad_rows).
//   * boxes of 64 voxels read from the channels-last tensors (conv_wgrad_mn):
//     1x1x1 layers and longer rows.
//   * otherwise (no such box, or a leading dimension that TMA cannot take)
//     both operands are first copied voxel-major (one row of voxels per
//     channel) into a flat layout padded by one zero slice in z and one zero
//     row in y on each side, so that the dz and dy shifts of a tap are plain
//     offsets of the flat TMA coordinate.  The dx shift cannot be such an
//     offset (the innermost TMA coordinate must stay 16-byte aligned), so the
//     input is copied three times, pre-shifted by dx = -1, 0, +1.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "conv.cuh"
#include "tc.cuh"

namespace rsv {

using namespace tc;

// ------------------------------------------------------------------ host: tensor maps
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// BF16 tensor map of rank r: dims/box innermost first, strides in bytes for dims 1..r-1.
rsv_status make_map(CUtensorMap *m, const void *base, int rank, const uint64_t *dims, const uint64_t *strides,
                    const uint32_t *box, int swz) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return RSV_ENOTSUP;
    if (((uintptr_t)base) & 15) return RSV_EINVAL;
    for (int i = 0; i < rank - 1; ++i)
        if (strides[i] % 16) return RSV_EINVAL;
    cuuint64_t d[5], s[4];
    cuuint32_t b[5], e[5];
    for (int i = 0; i < rank; ++i) {
        d[i] = dims[i];
        b[i] = box[i];
        e[i] = 1;
        if (i < rank - 1) s[i] = strides[i];
    }
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void *>(base), d, s, b, e,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swz == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? RSV_OK : RSV_EINVAL;
}

constexpr int kStages = 4;
constexpr int kThreads = 128;

__device__ __forceinline__ void raise(int *err, int code) {
    if (err) atomicCAS(err, 0, code);
}

// ------------------------------------------------------------------ forward / input-gradient kernel
struct FwdArgs {
    int nx, ny, nz;
    int bw, bh, bd;       // voxel box of one M tile
    int tx, ty;           // tiles along x and y
    int taps, nkb, ci;    // taps (27 or 1), channel blocks per tap, input channels
    int n_total;          // output channels
    const float *bias;    // [n_total] or null
    int relu;
    const __nv_bfloat16 *mask;  // multiply by (mask > 0): [V][ldm] or null
    int ldm;
    __nv_bfloat16 *y;     // [V][ldy] or null
    int ldy;
    float *y32;           // [V][n_total] or null
    int *err;
    uint64_t timeout_ns;
    const int *gate;      // skip the launch when *gate != 0 (may be null)
};

// Epilogue of 16 output channels n .. n + 15 of voxel v: bias (at n of a.bias), ReLU, mask (its 16 values), FP32 and BF16
// stores.
__device__ __forceinline__ void load_mask16(const FwdArgs &a, int64_t v, int n, uint4 mv[2]) {
    const uint4 *mp = (const uint4 *)(a.mask + v * a.ldm + n);
    mv[0] = mp[0];
    mv[1] = mp[1];
}
__device__ __forceinline__ void store16(const FwdArgs &a, int64_t v, int n, float acc[16], const float *bias, const uint4 mv[2]) {
    if (bias) {
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] += bias[i];
    }
    if (a.relu) {
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = fmaxf(acc[i], 0.0f);
    }
    if (a.mask) {
        const __nv_bfloat16 *mb = (const __nv_bfloat16 *)mv;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (!(__bfloat162float(mb[i]) > 0.0f)) acc[i] = 0.0f;
    }
    if (a.y32) {
        float4 *o = (float4 *)(a.y32 + v * a.n_total + n);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    }
    if (a.y) {
        uint4 ov[2];
        __nv_bfloat162 *ob = (__nv_bfloat162 *)ov;
#pragma unroll
        for (int i = 0; i < 8; ++i) ob[i] = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
        uint4 *o = (uint4 *)(a.y + v * a.ldy + n);
        o[0] = ov[0];
        o[1] = ov[1];
    }
}

template <int BK, int BN>
struct FwdSmem {
    static constexpr uint32_t A = 128 * BK * 2, B = BN * BK * 2, STAGE = A + B;
    static constexpr uint32_t BARS = kStages * STAGE;
    static constexpr uint32_t BYTES = BARS + 256 + 1024;  // + barriers/slots + alignment slack
};

template <int BK, int BN>
__global__ void __launch_bounds__(kThreads, 1)
    conv_fwd_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const FwdArgs a) {
    if (a.gate && *a.gate) return;  // uniform across the CTA, before any barrier or allocation
    using L = FwdSmem<BK, BN>;
    constexpr int SWZ = BK * 2;  // 128 or 64
    constexpr uint32_t TCOLS = tmem_cols_for(BN);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = (uint64_t *)(sm + L::BARS);
    uint64_t *empty = full + kStages;
    uint64_t *done = empty + kStages;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *flags = (int *)(tmem_slot + 1);  // [0] failed, [1] loads issued, [2] loads consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x;
    const int x0 = (tile % a.tx) * a.bw;
    const int y0 = ((tile / a.tx) % a.ty) * a.bh;
    const int z0 = (tile / (a.tx * a.ty)) * a.bd;
    const int n0 = blockIdx.y * BN;
    const int nk = a.taps * a.nkb;
    const uint64_t deadline = now_ns() + a.timeout_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == 2) tmem_alloc(tmem_slot, TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // TMA producer
        prefetch_map(&tmA);
        prefetch_map(&tmB);
        const uint32_t bytes = (uint32_t)(a.bw * a.bh * a.bd) * BK * 2 + (uint32_t)BN * BK * 2;
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % kStages;
            if (kk >= kStages && !mbar_wait(&empty[s], ((kk / kStages) + 1) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            const int tap = kk / a.nkb, cb = kk % a.nkb;
            int dz = 0, dy = 0, dx = 0;
            if (a.taps == 27) {
                dz = tap / 9 - 1;
                dy = (tap / 3) % 3 - 1;
                dx = tap % 3 - 1;
            }
            uint8_t *st = sm + s * L::STAGE;
            mbar_expect_tx(&full[s], bytes);
            tma_load_4d(st, &tmA, cb * BK, x0 + dx, y0 + dy, z0 + dz, &full[s]);
            tma_load_2d(st + L::A, &tmB, tap * a.ci + cb * BK, n0, &full[s]);
        }
        flags[1] = kk;
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        constexpr uint32_t idesc = idesc_bf16(128, BN);
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % kStages;
            if (!mbar_wait(&full[s], (kk / kStages) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            fence_after_sync();
            const uint32_t sa = smem_u32(sm + s * L::STAGE), sb = sa + L::A;
#pragma unroll
            for (int j = 0; j < BK / 16; ++j)
                mma_bf16(tmem, kmajor_desc(sa + j * 32, SWZ), kmajor_desc(sb + j * 32, SWZ), idesc,
                         (kk > 0 || j > 0) ? 1u : 0u);
            mma_commit(&empty[s]);
        }
        flags[2] = kk;
        mma_commit(done);
    }
    __syncwarp();

    // Epilogue: warp w owns TMEM lanes 32w..32w+31, i.e. tile rows (voxels) 32w + lane.
    const bool ok = mbar_wait(done, 0, deadline + a.timeout_ns);
    fence_after_sync();
    const int row = warp * 32 + lane;
    const int rx = row % a.bw, ry = (row / a.bw) % a.bh, rz = row / (a.bw * a.bh);
    const int x = x0 + rx, y = y0 + ry, z = z0 + rz;
    const bool valid = ok && rz < a.bd && x < a.nx && y < a.ny && z < a.nz && !flags[0];
    const int64_t v = ((int64_t)z * a.ny + y) * a.nx + x;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        float acc[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, acc);
        if (!valid) continue;
        uint4 mv[2];
        if (a.mask) load_mask16(a, v, n0 + c0, mv);
        store16(a, v, n0 + c0, acc, a.bias ? a.bias + n0 + c0 : nullptr, mv);
    }

    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && (flags[0] || !ok)) {
        raise(a.err, RSV_ETIMEOUT);
        // let copies still in flight land before the shared memory is released
        for (int kk = flags[2]; kk < flags[1]; ++kk)
            mbar_wait(&full[kk % kStages], (kk / kStages) & 1, now_ns() + a.timeout_ns);
    }
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, TCOLS);
}

// ------------------------------------------------------------------ forward, x taps folded into N
// For narrow layers (32 or 64 output channels) the kernel above is bound by L2: every tile reads its 27 shifted
// neighbourhoods.  Here the three x taps of a (dz, dy) pair become columns of one product: with
// P_dx[u] = sum over dz, dy, channels of w[dz, dy, dx] x[u + (dz, dy)] (N = 3 co columns), y[v] = P_-1[v - 1] +
// P_0[v] + P_+1[v + 1], added in the epilogue from the neighbouring TMEM lanes; a tile's rows span the whole
// x extent, so no neighbour lies outside it but the zero padding.  The y taps share one box: two M tiles
// stacked in y read one box of 2 bh + 2 rows per dz, each (tile, dy) an operand that starts a multiple
// of nx rows into it.  Per 128 voxels and 32 input channels that is 48 KB of operands from L2 instead of 216, and a
// third of the MMAs.
// A CTA takes consecutive pairs along z.  With one block of channels (32, or 64 where ci is a multiple of 64) it keeps
// the boxes of three planes, so each is loaded once instead of three times ("march").  The weights stay in shared memory
// when they fit beside the boxes (32 -> 32 and 32 -> 64 channels); else the 3 co rows of one (dz, dy) at a time pass
// through a ring.  With 32 output channels the epilogue of a pair of tiles overlaps the next pair's MMAs (two
// accumulator sets of 192 columns).
// What bounds it: with 32 output channels the issue of the MMAs, 75 cycles each where the tensor core takes 61 (N = 96),
// and the epilogue of about the same length beside it; with 64 the MMAs (102 cycles, N = 192) and then the epilogue.
// Kernel, 128x128x64: 32 -> 32 channels 175 us with a box per tap, 67 with three boxes per pair, descriptors by one lane
// and eight epilogue warps, 57 now; 64x64x32: 64 -> 64 56, 40, 34.  Calls: 128x128x64, 64 -> 64 243 -> 207 us, 96 -> 32
// 171 either way; 104x77x40, 64 -> 32 70 -> 61; 32x32x16 and below the call's fixed 30.
struct FoldArgs {
    FwdArgs f;              // bw = nx, bh rows per tile, bd = 1, ty: pairs along y
    int nz, pairs;          // planes; pairs of tiles
    int S, SB;              // slots for input boxes; for the weights of one (dz, channel block, dy), 0: all resident
    int march;
    uint32_t boxA, strideA; // bytes of an input box, and its room (a tile's 128 rows may pass the box's end)
    uint32_t offA, offBar;  // shared-memory offsets (the weights come first)
};

// Producer, MMA issuer, and four epilogue warps for each half of the channels of each tile of the pair: with four for
// all channels the epilogue, a chain of latencies, took as long as the MMAs (32 channels), or 5,400 cycles between them
// (64).
constexpr int kFoldThreads = 576;
constexpr uint32_t kFoldTail = 512 + 256 + 4096;  // barriers, bias, the epilogue's exchange
constexpr int kFoldMaxStages = 6, kFoldMaxWeights = 16;

// Whether `ok` holds for all four warps at named barrier `bar`.
__device__ __forceinline__ bool all_of_128(int bar, bool ok) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, %2, 128, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)ok), "r"(bar)
        : "memory");
    return r != 0;
}

// y taps per slot of the weights' ring.  A wait and a release per slot cost the issuing warp about as much as two MMAs:
// the smallest weights (32 rows of 32 channels, four MMAs per y tap) take all three (96 -> 32 channels on 128x128x64:
// 219 us a call with one each, 171 so).
__host__ __device__ constexpr int fold_dys(int co, int bk) { return co == 32 && bk == 32 ? 3 : 1; }

// A position in a ring: slot and the parity of its current phase.
struct RingPos {
    int s = 0;
    unsigned parity = 0;
    __device__ __forceinline__ void next(int S) {
        if (++s == S) {
            s = 0;
            parity ^= 1u;
        }
    }
};

// The pairs of tiles of a CTA.  March: consecutive ones, z fastest.  Else every gridDim-th, y fastest: neighbours in y,
// which share rows, run at the same time and find them in L2 (64 -> 32 channels on 128x128x64: 132 us a call with
// consecutive pairs, 120 so).
struct FoldWalk {
    int p0, step, n, ty, nz;
    __device__ __forceinline__ explicit FoldWalk(const FoldArgs &g) : ty(g.f.ty), nz(g.nz) {
        if (g.march) {
            p0 = (int)((int64_t)blockIdx.x * g.pairs / gridDim.x);
            n = (int)((int64_t)(blockIdx.x + 1) * g.pairs / gridDim.x) - p0;
            step = 0;
        } else {
            p0 = blockIdx.x;
            step = gridDim.x;
            n = (g.pairs - p0 + step - 1) / step;
        }
    }
    __device__ __forceinline__ void at(int it, int &yp, int &z) const {
        if (step) {
            const int p = p0 + it * step;
            z = p / ty;
            yp = p - z * ty;
        } else {
            yp = (p0 + it) / nz;
            z = p0 + it - yp * nz;
        }
    }
};

template <int CO, int BK>
__global__ void __launch_bounds__(kFoldThreads, 1)
    conv_fold_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const FoldArgs g) {
    const FwdArgs &a = g.f;
    if (a.gate && *a.gate) return;  // uniform across the CTA, before any barrier or allocation
    constexpr int BN = 3 * CO, SWZ = 2 * BK;       // SWZ: bytes of an operand row
    constexpr int NBUF = CO == 32 ? 2 : 1;         // accumulator sets
    constexpr uint32_t BDY = BN * SWZ;             // weight bytes of one (dz, channel block, dy)
    constexpr int DYS = fold_dys(CO, BK);          // y taps in a weight slot
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = (uint64_t *)(sm + g.offBar);
    uint64_t *empty = full + kFoldMaxStages, *accfull = empty + kFoldMaxStages, *accempty = accfull + 2;
    uint64_t *bfull = accempty + 2, *bempty = bfull + kFoldMaxWeights, *done = bempty + kFoldMaxWeights;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *flags = (int *)(tmem_slot + 1);  // [0] failed, [1] boxes and [2] weight loads issued
    float *sbias = (float *)(sm + g.offBar + 512);
    float *xch = sbias + 64;  // [tile, half][2][4 warps][2][16]: boundary lanes' values of a chunk
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint64_t deadline = now_ns() + a.timeout_ns;
    const int nk = 3 * a.nkb;  // boxes (dz, channel block) that a pair reads
    const FoldWalk walk(g);

    if (threadIdx.x == 0) {
        for (int s = 0; s < g.S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < max(g.SB, 1); ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accfull[b], 1);
            mbar_init(&accempty[b], 16);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    if (a.bias && warp == 2)
        for (int c = lane; c < CO; c += 32) sbias[c] = a.bias[c];
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        prefetch_map(&tmA);
        prefetch_map(&tmB);
        int boxes = 0, loads = 0;
        bool ok = true;
        if (!g.SB) {  // rows (dz, channel block, dy, dx, output channel)
            mbar_expect_tx(&bfull[0], (uint32_t)nk * 3 * BDY);
            for (int q = 0; q < nk; ++q)
                for (int dy = 0; dy < 3; dy += DYS)
                    tma_load_3d(sm + (q * 3 + dy) * BDY, &tmB, (q % a.nkb) * BK, 0, (q / a.nkb) * 9 + dy * 3, &bfull[0]);
            loads = 1;
        }
        // everything in the order in which the MMAs use it
        RingPos box, wt;
        for (int it = 0; ok && it < walk.n; ++it) {
            int yp, z;
            walk.at(it, yp, z);
            const bool start = it == 0 || z == 0;
            int dz = 0, cb = 0;
            for (int q = 0; ok && q < nk; ++q) {
                if (!g.march || start || q == 2) {
                    if (boxes >= g.S && !(ok = mbar_wait(&empty[box.s], box.parity ^ 1u, deadline))) break;
                    mbar_expect_tx(&full[box.s], g.boxA);
                    tma_load_4d(sm + g.offA + box.s * g.strideA, &tmA, cb * BK, 0, yp * 2 * a.bh - 1, z + dz - 1, &full[box.s]);
                    box.next(g.S);
                    ++boxes;
                }
                for (int dy = 0; g.SB && dy < 3; dy += DYS) {
                    if (loads >= g.SB && !(ok = mbar_wait(&bempty[wt.s], wt.parity ^ 1u, deadline))) break;
                    mbar_expect_tx(&bfull[wt.s], DYS * BDY);
                    tma_load_3d(sm + wt.s * (DYS * BDY), &tmB, cb * BK, 0, dz * 9 + dy * 3, &bfull[wt.s]);
                    wt.next(g.SB);
                    ++loads;
                }
                if (++cb == a.nkb) {
                    cb = 0;
                    ++dz;
                }
            }
        }
        if (!ok) flags[0] = 1;
        flags[1] = boxes;
        flags[2] = loads;
    } else if (warp == 1) {  // in step; one lane issues
        const uint32_t lead = elect_one();
        constexpr uint32_t idesc = idesc_bf16(128, BN);
        const uint32_t hi = (uint32_t)(kmajor_desc(0, SWZ) >> 32);
        const uint32_t lo_a = (uint32_t)kmajor_desc(smem_u32(sm + g.offA), SWZ), lo_b = (uint32_t)kmajor_desc(smem_u32(sm), SWZ);
        uint32_t off[2][3];  // (tile, dy) in an input box
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) off[m][dy] = (uint32_t)((m * a.bh + dy) * a.bw) * (SWZ / 16);
        const bool march = g.march;
        const int S = g.S;
        RingPos box, wt;
        bool ok = g.SB || warp_wait(&bfull[0], 0, deadline);
        for (int it = 0; ok && it < walk.n; ++it) {
            const int buf = it % NBUF;
            const uint32_t acc = tmem + buf * (2 * BN);
            if (it >= NBUF && !(ok = warp_wait(&accempty[buf], ((it / NBUF) + 1) & 1, deadline))) break;
            fence_after_sync();
            const bool last = it + 1 == walk.n || (walk.p0 + it + 1) % walk.nz == 0;  // the next pair, if any, starts with new boxes
            for (int q = 0; ok && q < nk; ++q) {
                RingPos b = box;  // march: the planes z - 1, z, z + 1 lie one after another in the ring
                if (march && (b.s += q) >= S) {
                    b.s -= S;
                    b.parity ^= 1u;
                }
                if (!(ok = warp_wait(&full[b.s], b.parity, deadline))) break;
                const uint32_t da = lo_a + b.s * (g.strideA >> 4);
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    if (dy % DYS == 0) {
                        if (g.SB && !(ok = warp_wait(&bfull[wt.s], wt.parity, deadline))) break;
                        fence_after_sync();
                    }
                    const uint32_t db = lo_b + ((g.SB ? wt.s * DYS + dy % DYS : q * 3 + dy)) * (BDY >> 4);
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int j = 0; j < BK / 16; ++j)
                            mma_bf16(lead, acc + m * BN, da + off[m][dy] + 2 * j, hi, db + 2 * j, hi, idesc,
                                     (q > 0 || dy > 0 || j > 0) ? 1u : 0u);
                    if (g.SB && dy % DYS == DYS - 1) {
                        mma_commit(lead, &bempty[wt.s]);
                        wt.next(g.SB);
                    }
                }
                if (!march || q == 0 || last) mma_commit(lead, &empty[b.s]);
                if (!march) box.next(S);
            }
            if (march)
                for (int i = 0; i < (last ? 3 : 1); ++i) box.next(S);
            if (ok) mma_commit(lead, &accfull[buf]);
        }
        if (!ok && lane == 0) flags[0] = 1;
        mma_commit(lead, done);
    } else if (warp >= 2) {
        // a warp reads the quarter of the TMEM lanes that its index allows
        constexpr int NCH = CO / 32;  // chunks of 16 channels per warp
        const int quarter = warp & 3, row = quarter * 32 + lane, grp = (warp - 2) >> 2, m = grp >> 1, n0 = (grp & 1) * (CO / 2);
        const int rx = row % a.bw, ry = row / a.bw;
        const bool left = rx > 0, right = rx < a.bw - 1;
        float *const mine = xch + grp * 256 + quarter * 32;
        unsigned chunk = 0;
        for (int it = 0; it < walk.n; ++it) {
            const int buf = it % NBUF;
            int yp, z;
            walk.at(it, yp, z);
            const int y = (yp * 2 + m) * a.bh + ry;
            const bool valid = ry < a.bh && y < a.ny;
            const int64_t v = ((int64_t)z * a.ny + y) * a.nx + rx;
            uint4 mv[NCH][2];
            if (a.mask && valid)  // under the MMAs
#pragma unroll
                for (int u = 0; u < NCH; ++u) load_mask16(a, v, n0 + 16 * u, mv[u]);
            // the four warps of a group share barriers: they go on, or give up, together
            if (!all_of_128(1 + grp, mbar_wait(&accfull[buf], (it / NBUF) & 1, deadline))) break;
            fence_after_sync();
            const uint32_t acc0 = tmem + buf * (2 * BN) + m * BN + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
            for (int u = 0; u < NCH; ++u, ++chunk) {
                const int n = n0 + 16 * u;
                uint32_t pm[16], pc[16], pp[16];
                tmem_ld16_start(acc0 + n, pm);
                tmem_ld16_start(acc0 + CO + n, pc);
                tmem_ld16_start(acc0 + 2 * CO + n, pp);
                tmem_ld_wait();
                tmem_landed(pm);
                tmem_landed(pc);
                tmem_landed(pp);
                float *slot = mine + (chunk & 1) * 128;
                if (lane == 31)
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *(uint4 *)(slot + i) = make_uint4(pm[i], pm[i + 1], pm[i + 2], pm[i + 3]);
                if (lane == 0)
#pragma unroll
                    for (int i = 0; i < 16; i += 4)
                        *(uint4 *)(slot + 16 + i) = make_uint4(pp[i], pp[i + 1], pp[i + 2], pp[i + 3]);
                if (u == NCH - 1) {  // the accumulators are in registers: the next pair may overwrite them
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&accempty[buf]);
                }
                asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
                float acc[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    float before = __uint_as_float(__shfl_up_sync(0xffffffffu, pm[i], 1));
                    float after = __uint_as_float(__shfl_down_sync(0xffffffffu, pp[i], 1));
                    if (lane == 0 && quarter > 0) before = slot[i - 32];
                    if (lane == 31 && quarter < 3) after = slot[i + 48];
                    acc[i] = ((left ? before : 0.0f) + __uint_as_float(pc[i])) + (right ? after : 0.0f);
                }
                if (valid) store16(a, v, n, acc, a.bias ? sbias + n : nullptr, mv[u]);
            }
        }
    }
    __syncwarp();
    const bool ok = mbar_wait(done, 0, deadline + a.timeout_ns);
    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && (flags[0] || !ok)) {
        raise(a.err, RSV_ETIMEOUT);
        // let copies still in flight land before the shared memory is released
        for (int kk = max(0, flags[1] - g.S); kk < flags[1]; ++kk)
            mbar_wait(&full[kk % g.S], (kk / g.S) & 1, now_ns() + a.timeout_ns);
        const int SB = max(g.SB, 1);
        for (int kk = max(0, flags[2] - SB); kk < flags[2]; ++kk)
            mbar_wait(&bfull[kk % SB], (kk / SB) & 1, now_ns() + a.timeout_ns);
    }
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ weight-gradient kernel
struct WgArgs {
    int nchunks, cps;          // 64-voxel K chunks in the padded volume; chunks per split
    int taps, ci, cblk, tpt, ncb;  // tap-group rows: tpt taps x cblk channels; ncb = ci / cblk
    int plane, row;            // flat shift of dz and dy in the padded layout
    int co;                    // output channels (N total)
    float *partial;            // [splits][taps][ci][co]
    int *err;
    uint64_t timeout_ns;
};

template <int BN>
struct WgSmem {
    static constexpr uint32_t A = 128 * 128, B = BN * 128, STAGE = A + B;
    static constexpr uint32_t BARS = kStages * STAGE;
    static constexpr uint32_t BYTES = BARS + 256 + 1024;
};

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    conv_wgrad_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const WgArgs a) {
    using L = WgSmem<BN>;
    constexpr uint32_t TCOLS = tmem_cols_for(BN);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = (uint64_t *)(sm + L::BARS);
    uint64_t *empty = full + kStages;
    uint64_t *done = empty + kStages;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *flags = (int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tg = blockIdx.x / a.ncb, cb = blockIdx.x % a.ncb;
    const int n0 = blockIdx.y * BN;
    const int q0 = blockIdx.z * a.cps;
    const int q1 = min(a.nchunks, q0 + a.cps);
    const int nk = max(0, q1 - q0);
    const int ntap = min(a.tpt, a.taps - tg * a.tpt);
    const uint64_t deadline = now_ns() + a.timeout_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == 2) tmem_alloc(tmem_slot, TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        prefetch_map(&tmA);
        prefetch_map(&tmB);
        const uint32_t bytes = (uint32_t)ntap * a.cblk * 128 + (uint32_t)BN * 128;
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % kStages;
            if (kk >= kStages && !mbar_wait(&empty[s], ((kk / kStages) + 1) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            const int f0 = (q0 + kk) * 64;
            uint8_t *st = sm + s * L::STAGE;
            mbar_expect_tx(&full[s], bytes);
            for (int g = 0; g < ntap; ++g) {
                const int tap = tg * a.tpt + g;
                int dz = 0, dy = 0, dxi = 0;
                if (a.taps == 27) {
                    dz = tap / 9 - 1;
                    dy = (tap / 3) % 3 - 1;
                    dxi = tap % 3;
                }
                tma_load_3d(st + g * a.cblk * 128, &tmA, f0 + dz * a.plane + dy * a.row, cb * a.cblk, dxi, &full[s]);
            }
            tma_load_2d(st + L::A, &tmB, f0, n0, &full[s]);
        }
        flags[1] = kk;
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(128, BN);
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % kStages;
            if (!mbar_wait(&full[s], (kk / kStages) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            fence_after_sync();
            const uint32_t sa = smem_u32(sm + s * L::STAGE), sb = sa + L::A;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                mma_bf16(tmem, kmajor_desc(sa + j * 32, 128), kmajor_desc(sb + j * 32, 128), idesc,
                         (kk > 0 || j > 0) ? 1u : 0u);
            mma_commit(&empty[s]);
        }
        flags[2] = kk;
        mma_commit(done);
    }
    __syncwarp();

    const bool ok = mbar_wait(done, 0, deadline + a.timeout_ns);
    fence_after_sync();
    const int row = warp * 32 + lane;
    const int g = row / a.cblk, c = row % a.cblk;
    const int tap = tg * a.tpt + g;
    const bool valid = ok && g < ntap && !flags[0];
    float *out = a.partial + (((int64_t)blockIdx.z * a.taps + tap) * a.ci + cb * a.cblk + c) * a.co + n0;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        float acc[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, acc);
        if (!valid) continue;
        if (nk == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
        }
        float4 *o = (float4 *)(out + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    }

    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && (flags[0] || !ok)) {
        raise(a.err, RSV_ETIMEOUT);
        for (int kk = flags[2]; kk < flags[1]; ++kk)
            mbar_wait(&full[kk % kStages], (kk / kStages) & 1, now_ns() + a.timeout_ns);
    }
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, TCOLS);
}

// ------------------------------------------------------------------ weight gradient, MN-major operands
// The same reduction over voxels as conv_wgrad_tc, read straight from the
// channels-last tensors: a TMA box of 64 voxels x (32 or 64) channels lands
// in shared memory as 64 rows (K = voxels) of consecutive channels (M or N),
// i.e. an MN-major operand.  Every tap shift (dz, dy, dx) is a plain TMA
// coordinate offset on the voxel axes, with zero fill outside the grid, so no
// copy of the activations is made.
//   A columns: tpt taps x cblk channels = 128 rows of M, in columns of colA
//   (64 or 32) channels; B columns: BN output channels in columns of colB.
struct WgMnArgs {
    int bw, bh, bd;                  // voxel box of one K chunk (bw * bh * bd = 64)
    int kcx, kcy, nchunks, cps;      // chunk grid (x, y; z implied), chunks per split
    int taps, ci, cblk, tpt, ncb, colA;  // ci: channels of the row (tap-shifted) operand
    int co, colB;                    // co: channels of the column operand
    int sgn;                         // +1: rows read at v + off_t; -1: at v - off_t
    float *partial;                  // [splits][taps][ci][co] in the row / column channel roles
    int *err;
    uint64_t timeout_ns;
};

// Pipeline depth per N tile: the deepest ring that still lets two CTAs share an SM.
template <int BN>
struct WgMnSmem {
    static constexpr uint32_t A = 128 * 64 * 2, B = BN * 64 * 2, STAGE = A + B;
    static constexpr int S = STAGE * 4 <= 100 * 1024 ? 4 : STAGE * 3 <= 100 * 1024 ? 3 : 2;
    static constexpr uint32_t BARS = S * STAGE;
    static constexpr uint32_t BYTES = BARS + 256 + 1024;
};

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    conv_wgrad_mn(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG, const WgMnArgs a) {
    using L = WgMnSmem<BN>;
    constexpr uint32_t TCOLS = tmem_cols_for(BN);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = (uint64_t *)(sm + L::BARS);
    uint64_t *empty = full + L::S;
    uint64_t *done = empty + L::S;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *flags = (int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tg = blockIdx.x / a.ncb, cb = blockIdx.x % a.ncb;
    const int n0 = blockIdx.y * BN;
    const int q0 = blockIdx.z * a.cps;
    const int q1 = min(a.nchunks, q0 + a.cps);
    const int nk = max(0, q1 - q0);
    const int ntap = min(a.tpt, a.taps - tg * a.tpt);
    const int colsA = 128 / a.colA, colsB = BN / a.colB;  // columns per operand
    const int colsPerTap = a.cblk / a.colA;
    const uint32_t rowA = a.colA * 2, rowB = a.colB * 2;  // bytes per K row of a column
    const uint64_t deadline = now_ns() + a.timeout_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < L::S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == 2) tmem_alloc(tmem_slot, TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        prefetch_map(&tmX);
        prefetch_map(&tmG);
        const uint32_t bytes = (uint32_t)(ntap * colsPerTap) * 64 * rowA + (uint32_t)colsB * 64 * rowB;
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % L::S;
            if (kk >= L::S && !mbar_wait(&empty[s], ((kk / L::S) + 1) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            const int q = q0 + kk;
            const int x0 = (q % a.kcx) * a.bw, y0 = ((q / a.kcx) % a.kcy) * a.bh, z0 = (q / (a.kcx * a.kcy)) * a.bd;
            uint8_t *st = sm + s * L::STAGE;
            mbar_expect_tx(&full[s], bytes);
            for (int g = 0; g < ntap; ++g) {
                const int tap = tg * a.tpt + g;
                int dz = 0, dy = 0, dx = 0;
                if (a.taps == 27) {
                    dz = tap / 9 - 1;
                    dy = (tap / 3) % 3 - 1;
                    dx = tap % 3 - 1;
                }
                for (int j = 0; j < colsPerTap; ++j)
                    tma_load_4d(st + (g * colsPerTap + j) * 64 * rowA, &tmX, cb * a.cblk + j * a.colA,
                                x0 + a.sgn * dx, y0 + a.sgn * dy, z0 + a.sgn * dz, &full[s]);
            }
            for (int j = 0; j < colsB; ++j)
                tma_load_4d(st + L::A + j * 64 * rowB, &tmG, n0 + j * a.colB, x0, y0, z0, &full[s]);
        }
        flags[1] = kk;
    } else if (warp == 1 && lane == 0) {
        constexpr uint32_t idesc = idesc_bf16(128, BN, true, true);
        const int swzA = a.colA == 64 ? 128 : 64, swzB = a.colB == 64 ? 128 : 64;
        const uint32_t colbA = 64 * rowA, colbB = 64 * rowB, grpA = 8 * rowA, grpB = 8 * rowB;
        (void)colsA;
        int kk = 0;
        for (; kk < nk; ++kk) {
            const int s = kk % L::S;
            if (!mbar_wait(&full[s], (kk / L::S) & 1, deadline)) {
                flags[0] = 1;
                break;
            }
            fence_after_sync();
            const uint32_t sa = smem_u32(sm + s * L::STAGE), sb = sa + L::A;
#pragma unroll
            for (int j = 0; j < 4; ++j)  // 4 x K = 16 rows = the 64 voxels of the chunk
                mma_bf16(tmem, mnmajor_desc(sa + j * 2 * grpA, swzA, colbA, grpA),
                         mnmajor_desc(sb + j * 2 * grpB, swzB, colbB, grpB), idesc, (kk > 0 || j > 0) ? 1u : 0u);
            mma_commit(&empty[s]);
        }
        flags[2] = kk;
        mma_commit(done);
    }
    __syncwarp();

    const bool ok = mbar_wait(done, 0, deadline + a.timeout_ns);
    fence_after_sync();
    const int row = warp * 32 + lane;
    const int g = row / a.cblk, c = row % a.cblk;
    const int tap = tg * a.tpt + g;
    const bool valid = ok && g < ntap && !flags[0];
    float *out = a.partial + (((int64_t)blockIdx.z * a.taps + tap) * a.ci + cb * a.cblk + c) * a.co + n0;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
        float acc[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, acc);
        if (!valid) continue;
        if (nk == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
        }
        float4 *o = (float4 *)(out + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    }

    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && (flags[0] || !ok)) {
        raise(a.err, RSV_ETIMEOUT);
        for (int kk = flags[2]; kk < flags[1]; ++kk)
            mbar_wait(&full[kk % L::S], (kk / L::S) & 1, now_ns() + a.timeout_ns);
    }
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, TCOLS);
}

// ------------------------------------------------------------------ weight gradient, rows of a plane shared by the y taps
// The MN-major form above reads every tap's shifted box of the activations from L2, 2 taps of 64 channels per 24 KB,
// and that is what bounds it (32 bytes per cycle and SM).  Here one K step is R whole rows of a plane, K = nx R voxels
// in (y, x) order, and its column operand comes from one box of R + 2 rows: the three y taps are the same box read
// nx shared-memory rows apart, 3 x 64 (or 32) columns of one product.  The row operand holds 128 rows: the other
// tensor at two (of 64 channels; four of 32; one of 128) of the nine (dz, dx) shifts.  An MMA's time does
// not depend on N up to 192, so the wider N is free.  The column operand is unshifted in x and z: a voxel pair
// counts where both are in the grid, and boxes read zeros outside.
// An FP32 accumulator's error grows with the number of MMAs that it takes one after another.  So the MMAs of a K step go to
// wgrad_sets(CN) accumulators in turn, as many as TMEM holds, which the epilogue adds; and the voxels are split until no
// accumulator takes more of them than one of the form above would (wg_row_plan).  With one accumulator and a single wave
// the error of 256 -> 256 channels on 16x16x8 was 2.4 times that form's, of 96 -> 32 on 128x128x64 2.9 times; now 0.6 and
// 0.65, and 0.2 to 0.8 on every shape tried.
// Kernel (ncu), boxes' form -> this: 64x64x32, 64 -> 64 channels 74 -> 27 us; 128x128x64, 32 -> 32 383 -> 116, 96 -> 32
// 403 -> 348; 32x32x16, 384 -> 128 54 -> 43; 16x16x8, 256 -> 256 22.1 -> 20.4.
struct WgRowArgs {
    int nx, R, kcy, nchunks, cps;  // rows per K step, steps per plane, steps, steps per split
    int cm, variants, nmb;         // channels per row block, shifts per MMA, channel blocks
    int ca, cb;                    // channels of the row and column operand
    int sgn;                       // +1: rows = gradient, columns = input; -1: the reverse
    int S;                         // stages
    uint32_t offN, stride, offBar;
    float *partial;                // [splits][27][ca][cb]
    int *err;
    uint64_t timeout_ns;
};

__host__ __device__ constexpr int wgrad_sets(int cn) { return cn == 64 ? 2 : 4; }

template <int CN>
__global__ void __launch_bounds__(kThreads, 1)
    conv_wgrad_rows(const __grid_constant__ CUtensorMap tmM, const __grid_constant__ CUtensorMap tmN, const WgRowArgs a) {
    constexpr int N = 3 * CN, SETS = wgrad_sets(CN);
    constexpr uint32_t TCOLS = tmem_cols_for(SETS * N);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint64_t *full = (uint64_t *)(sm + a.offBar);
    uint64_t *empty = full + a.S;
    uint64_t *done = empty + a.S;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *flags = (int *)(tmem_slot + 1);  // a wait ran out; steps issued; steps consumed

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int vg = blockIdx.x / a.nmb, mb = blockIdx.x % a.nmb;
    const int q0 = blockIdx.z * a.cps;
    const int nk = max(0, min(a.nchunks, q0 + a.cps) - q0);
    const int nv = min(a.variants, 9 - vg * a.variants);
    const int colA = min(a.cm, 64), K = a.nx * a.R;
    const uint32_t rowA = colA * 2, rowB = CN * 2, boxA = K * rowA;
    const uint64_t deadline = now_ns() + a.timeout_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        flags[0] = flags[1] = flags[2] = 0;
        fence_mbar_init();
    }
    if (warp == 2) tmem_alloc(tmem_slot, TCOLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        prefetch_map(&tmM);
        prefetch_map(&tmN);
        const int cols = a.cm / colA;
        const uint32_t bytes = (uint32_t)(nv * cols) * boxA + (uint32_t)(a.nx * (a.R + 2)) * rowB;
        int kk = 0, s = 0;
        unsigned parity = 1;
        for (; kk < nk; ++kk) {
            if (kk >= a.S && !mbar_wait(&empty[s], parity, deadline)) {
                flags[0] = 1;
                break;
            }
            const int z = (q0 + kk) / a.kcy, y = ((q0 + kk) % a.kcy) * a.R;
            uint8_t *st = sm + s * a.stride;
            mbar_expect_tx(&full[s], bytes);
            tma_load_4d(st + a.offN, &tmN, blockIdx.y * CN, 0, y - 1, z, &full[s]);
            for (int v = 0; v < nv; ++v) {
                const int sh = vg * a.variants + v, dz = sh / 3 - 1, dx = sh % 3 - 1;
                for (int j = 0; j < cols; ++j)
                    tma_load_4d(st + (v * cols + j) * boxA, &tmM, mb * a.cm + j * colA, -a.sgn * dx, y, z - a.sgn * dz,
                                &full[s]);
            }
            if (++s == a.S) {
                s = 0;
                parity ^= 1u;
            }
        }
        flags[1] = kk;
    } else if (warp == 1) {  // in step; one lane issues
        const uint32_t lead = elect_one();
        constexpr uint32_t idesc = idesc_bf16(128, N, true, true);
        const uint64_t a0 = mnmajor_desc(smem_u32(sm), colA == 64 ? 128 : 64, boxA, 8 * rowA);
        const uint64_t b0 = mnmajor_desc(smem_u32(sm + a.offN), CN == 64 ? 128 : 64, a.nx * rowB, 8 * rowB);
        const uint32_t ahi = (uint32_t)(a0 >> 32), bhi = (uint32_t)(b0 >> 32);
        int kk = 0, s = 0;
        unsigned parity = 0;
        for (; kk < nk; ++kk) {
            if (!warp_wait(&full[s], parity, deadline)) {
                if (lane == 0) flags[0] = 1;
                break;
            }
            fence_after_sync();
            uint32_t da = (uint32_t)a0 + s * (a.stride >> 4), db = (uint32_t)b0 + s * (a.stride >> 4);
#pragma unroll 4
            for (int k = 0; k < K; k += 16) {  // 16 voxels on: 16 rows of the operand's bytes
                mma_bf16(lead, tmem + (k / 16 % SETS) * N, da, ahi, db, bhi, idesc, (kk > 0 || k >= 16 * SETS) ? 1u : 0u);
                da += rowA;
                db += rowB;
            }
            mma_commit(lead, &empty[s]);
            if (++s == a.S) {
                s = 0;
                parity ^= 1u;
            }
        }
        if (lane == 0) flags[2] = kk;
        mma_commit(lead, done);
    }
    __syncwarp();

    const bool ok = mbar_wait(done, 0, deadline + a.timeout_ns);
    fence_after_sync();
    const int row = warp * 32 + lane;
    const int v = row / a.cm, c = row % a.cm, sh = vg * a.variants + v;
    const bool valid = ok && v < nv && !flags[0];
    float *out = a.partial + ((int64_t)blockIdx.z * 27 * a.ca + mb * a.cm + c) * a.cb + blockIdx.y * CN;
    const int nset = min(SETS, K / 16);
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 16) {
        uint32_t part[SETS][16];
#pragma unroll
        for (int q = 0; q < SETS; ++q)
            if (q < nset) tmem_ld16_start(tmem + ((uint32_t)(warp * 32) << 16) + q * N + c0, part[q]);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < SETS; ++q) tmem_landed(part[q]);
        float acc[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            acc[i] = __uint_as_float(part[0][i]);
#pragma unroll
            for (int q = 1; q < SETS; ++q)
                if (q < nset) acc[i] += __uint_as_float(part[q][i]);
        }
        if (!valid) continue;
        if (nk == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = 0.0f;
        }
        const int dy = a.sgn * (c0 / CN - 1);
        const int tap = 9 * (sh / 3) + 3 * (dy + 1) + sh % 3;
        float4 *o = (float4 *)(out + (int64_t)tap * a.ca * a.cb + c0 % CN);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
    }

    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0 && (flags[0] || !ok)) {
        raise(a.err, RSV_ETIMEOUT);
        // copies still in flight land before the shared memory is given up (bounded)
        for (int kk = flags[2]; kk < flags[1]; ++kk)
            mbar_wait(&full[kk % a.S], (kk / a.S) & 1, now_ns() + a.timeout_ns);
    }
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, TCOLS);
}

// gb[c] partial sums from the channels-last gradient: CTA b sums its chunk of voxels, a thread eight channels (16
// bytes) of every slots-th voxel.  part[b][co].  Bound by the loads in flight: 2-byte loads took 14.5 us on
// 64x64x32 voxels of 64 channels, these 8.
__global__ void __launch_bounds__(256) bias_grad_cl(const __nv_bfloat16 *__restrict__ gy, int ld, int co, int64_t V,
                                                    float *__restrict__ part) {
    __shared__ float red[256 * 8];
    const int64_t len = (V + gridDim.x - 1) / gridDim.x;
    const int64_t v0 = blockIdx.x * len, v1 = min(V, v0 + len);
    for (int c0 = 0; c0 < co; c0 += 2048) {  // channels that 256 threads cover
        const int pieces = min(256, (co - c0) / 8), slots = 256 / pieces;
        const int piece = threadIdx.x % pieces, slot = threadIdx.x / pieces;
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (slot < slots) {
            const __nv_bfloat16 *g = gy + c0 + piece * 8;
#pragma unroll 4
            for (int64_t v = v0 + slot; v < v1; v += slots) {
                const uint4 w = *reinterpret_cast<const uint4 *>(g + v * ld);
                const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    acc[2 * q] += __uint_as_float(u[q] << 16);
                    acc[2 * q + 1] += __uint_as_float(u[q] & 0xffff0000u);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) red[slot * pieces * 8 + piece * 8 + q] = acc[q];
        }
        __syncthreads();
        for (int c = threadIdx.x; c < pieces * 8; c += 256) {
            float t = 0.0f;
            for (int q = 0; q < slots; ++q) t += red[q * pieces * 8 + c];
            part[(int64_t)blockIdx.x * co + c0 + c] = t;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ helper kernels
// Voxel-major copy of a channels-last volume into the zero-padded flat layout
// of the weight gradient: out[d][c][f], f = ((z+1)(ny+2) + (y+1)) nx + x over
// z in [-1, nz], y in [-1, ny]; out[d][c][f] = x[z, y, x + d - 1, c] when
// nshift = 3 (d = 0, 1, 2), x[z, y, x, c] when nshift = 1; zero outside the grid.
// One CTA per (padded row, 32 channels, 128-voxel chunk of the row): the chunk
// and a one-voxel halo are read once, coalesced along the channels, and
// written nshift times, coalesced along x.
constexpr int kVmChunk = 128;
__global__ void __launch_bounds__(256)
    to_voxel_major(const __nv_bfloat16 *__restrict__ src, int ld, int nch, int nx, int ny, int nz, int nshift,
                   int64_t vpad, __nv_bfloat16 *__restrict__ dst) {
    __shared__ __nv_bfloat16 tile[kVmChunk + 2][33];
    const int row = blockIdx.x;  // padded row index (zp * (ny + 2) + yp)
    const int c0 = blockIdx.y * 32;
    const int x0 = blockIdx.z * kVmChunk;
    const int zp = row / (ny + 2), yp = row - zp * (ny + 2);
    const int z = zp - 1, y = yp - 1;
    const int w = min(kVmChunk, nx - x0);
    const bool real = z >= 0 && z < nz && y >= 0 && y < ny;
    const __nv_bfloat16 zero = __float2bfloat16(0.0f);
    if (real) {
        const int64_t base = ((int64_t)z * ny + y) * nx;
        for (int i = threadIdx.x; i < (w + 2) * 32; i += 256) {
            const int xl = i >> 5, c = i & 31;
            const int x = x0 + xl - 1;
            __nv_bfloat16 v = zero;
            if (x >= 0 && x < nx && c0 + c < nch) v = src[(base + x) * ld + c0 + c];
            tile[xl][c] = v;
        }
    }
    __syncthreads();
    const int64_t f0 = (int64_t)row * nx + x0;
    for (int d = 0; d < nshift; ++d) {
        const int sh = nshift == 3 ? d - 1 : 0;
        for (int i = threadIdx.x; i < 32 * w; i += 256) {
            const int c = i / w, xl = i - c * w;
            if (c0 + c >= nch) continue;
            const __nv_bfloat16 v = real ? tile[xl + 1 + sh][c] : zero;
            dst[((int64_t)d * nch + c0 + c) * vpad + f0 + xl] = v;
        }
    }
}

// gw[co][t][ci] = sum over splits of the partials, in split order.  The partials are
// [s][t][ci][co] (swap = 0), or [s][t][co][ci] (swap = 1: rows were output channels).  The blocks behind the first
// wblocks add the bias gradient's nblk partial sums (bias_grad_cl), one warp per channel: lane l the blocks l,
// l + 32, ... in order, then a fixed shuffle tree.
__global__ void __launch_bounds__(256) wgrad_reduce(const float *__restrict__ partial, int splits, int taps, int ci, int co,
                                                    float *__restrict__ gw, int swap, int wblocks,
                                                    const float *__restrict__ bpart, int nblk, float *__restrict__ gb) {
    if ((int)blockIdx.x >= wblocks) {
        const int c = ((int)blockIdx.x - wblocks) * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (c >= co) return;
        float t = 0.0f;
        for (int b = lane; b < nblk; b += 32) t += bpart[(int64_t)b * co + c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) gb[c] = t;
        return;
    }
    const int64_t total = (int64_t)taps * ci * co;
    const int ra = swap ? co : ci, rb = swap ? ci : co;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)wblocks * blockDim.x) {
        const int o = (int)(i / ((int64_t)taps * ci));
        const int t = (int)((i / ci) % taps);
        const int c = (int)(i % ci);
        const int row = swap ? o : c, col = swap ? c : o;
        const float *p = partial + ((int64_t)t * ra + row) * rb + col;
        float s = 0.0f;
#pragma unroll 8
        for (int q = 0; q < splits; ++q) s += p[q * total];
        gw[i] = s;
    }
}

// gb[c] = sum over the padded voxel-major row c (pads are zero): each CTA sums one
// of kBgChunks chunks of a row (fixed tree order), then bias_grad_final adds
// the chunks in order.
constexpr int kBgChunks = 32;
__global__ void __launch_bounds__(256) bias_grad(const __nv_bfloat16 *__restrict__ gyt, int64_t vpad,
                                                 float *__restrict__ part) {
    __shared__ float red[256];
    const __nv_bfloat16 *r = gyt + (int64_t)blockIdx.x * vpad;
    const int64_t len = (vpad + kBgChunks - 1) / kBgChunks;
    const int64_t a = blockIdx.y * len, b = min(vpad, a + len);
    float s = 0.0f;
    for (int64_t f = a + threadIdx.x; f < b; f += 256) s += __bfloat162float(r[f]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x * kBgChunks + blockIdx.y] = red[0];
}
__global__ void bias_grad_final(const float *__restrict__ part, int co, float *__restrict__ gb) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= co) return;
    float s = 0.0f;
    for (int k = 0; k < kBgChunks; ++k) s += part[c * kBgChunks + k];
    gb[c] = s;
}

// Weights of the input gradient: wt[ci][t][co] = w[co][26 - t][ci].
__global__ void flip_weights(const __nv_bfloat16 *__restrict__ w, int ci, int co, __nv_bfloat16 *__restrict__ wt) {
    const int64_t total = (int64_t)ci * 27 * co;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(i / (27 * co));
        const int t = (int)((i / co) % 27);
        const int o = (int)(i % co);
        wt[i] = w[((int64_t)o * 27 + (26 - t)) * ci + c];
    }
}

}  // namespace

// ------------------------------------------------------------------ host launchers
namespace {

int pick_bn(int n) {
    for (int b : {256, 192, 128, 96, 64, 32})
        if (n % b == 0) return b;
    return 0;
}

template <typename K>
cudaError_t set_smem(K kernel, uint32_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int BK, int BN>
cudaError_t launch_fwd_t(cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb, const FwdArgs &a) {
    using L = FwdSmem<BK, BN>;
    static cudaError_t attr = set_smem(conv_fwd_tc<BK, BN>, L::BYTES);
    if (attr != cudaSuccess) return attr;
    conv_fwd_tc<BK, BN><<<grid, kThreads, L::BYTES, st>>>(ma, mb, a);
    return cudaGetLastError();
}

template <int BK>
cudaError_t launch_fwd_bk(int bn, cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb,
                          const FwdArgs &a) {
    switch (bn) {
        case 32: return launch_fwd_t<BK, 32>(st, grid, ma, mb, a);
        case 64: return launch_fwd_t<BK, 64>(st, grid, ma, mb, a);
        case 96: return launch_fwd_t<BK, 96>(st, grid, ma, mb, a);
        case 128: return launch_fwd_t<BK, 128>(st, grid, ma, mb, a);
        case 192: return launch_fwd_t<BK, 192>(st, grid, ma, mb, a);
        default: return launch_fwd_t<BK, 256>(st, grid, ma, mb, a);
    }
}

template <int BN>
cudaError_t launch_wg_t(cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb, const WgArgs &a) {
    using L = WgSmem<BN>;
    static cudaError_t attr = set_smem(conv_wgrad_tc<BN>, L::BYTES);
    if (attr != cudaSuccess) return attr;
    conv_wgrad_tc<BN><<<grid, kThreads, L::BYTES, st>>>(ma, mb, a);
    return cudaGetLastError();
}

cudaError_t launch_wg(int bn, cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb,
                      const WgArgs &a) {
    switch (bn) {
        case 32: return launch_wg_t<32>(st, grid, ma, mb, a);
        case 64: return launch_wg_t<64>(st, grid, ma, mb, a);
        case 96: return launch_wg_t<96>(st, grid, ma, mb, a);
        case 128: return launch_wg_t<128>(st, grid, ma, mb, a);
        case 192: return launch_wg_t<192>(st, grid, ma, mb, a);
        default: return launch_wg_t<256>(st, grid, ma, mb, a);
    }
}

template <int BN>
cudaError_t launch_wgmn_t(cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb,
                          const WgMnArgs &a) {
    using L = WgMnSmem<BN>;
    static cudaError_t attr = set_smem(conv_wgrad_mn<BN>, L::BYTES);
    if (attr != cudaSuccess) return attr;
    conv_wgrad_mn<BN><<<grid, kThreads, L::BYTES, st>>>(ma, mb, a);
    return cudaGetLastError();
}

cudaError_t launch_wgmn(int bn, cudaStream_t st, dim3 grid, const CUtensorMap &ma, const CUtensorMap &mb,
                        const WgMnArgs &a) {
    switch (bn) {
        case 32: return launch_wgmn_t<32>(st, grid, ma, mb, a);
        case 64: return launch_wgmn_t<64>(st, grid, ma, mb, a);
        case 96: return launch_wgmn_t<96>(st, grid, ma, mb, a);
        case 128: return launch_wgmn_t<128>(st, grid, ma, mb, a);
        case 192: return launch_wgmn_t<192>(st, grid, ma, mb, a);
        default: return launch_wgmn_t<256>(st, grid, ma, mb, a);
    }
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

struct WgPlan {
    int64_t vpad;
    int nchunks, cblk, tpt, ncb, mtiles, bn, ntiles, splits, cps, nshift;
    size_t xt_bytes, gyt_bytes, part_bytes, bias_bytes;
    bool mn;                 // MN-major path: operands read straight from the channels-last tensors
    bool swap;               // MN path with rows = (tap, output channel): the gradient is the shifted operand
    int bw, bh, bd, kcx, kcy;
};

constexpr int kBiasBlocks = 304;

size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

WgPlan wg_plan(ConvVol v, int taps, int ci, int co) {
    WgPlan p{};
    p.bw = std::min(v.nx, 64);
    p.bh = std::min(v.ny, 64 / p.bw);
    p.bd = 64 / (p.bw * p.bh);
    p.mn = p.bw * p.bh * p.bd == 64 && p.bd <= v.nz;
    p.vpad = (int64_t)(v.nz + 2) * (v.ny + 2) * v.nx;
    if (p.mn) {
        p.kcx = (v.nx + p.bw - 1) / p.bw;
        p.kcy = (v.ny + p.bh - 1) / p.bh;
        p.nchunks = p.kcx * p.kcy * ((v.nz + p.bd - 1) / p.bd);
    } else {
        p.nchunks = (int)((p.vpad + 63) / 64);
    }
    // the wider channel count becomes the MMA's N when both operands are read channels-last
    p.swap = p.mn && ci > co;
    const int ra = p.swap ? co : ci, rb = p.swap ? ci : co;
    p.cblk = ra % 128 == 0 ? 128 : ra % 64 == 0 ? 64 : 32;
    p.tpt = 128 / p.cblk;
    p.ncb = ra / p.cblk;
    p.mtiles = ((taps + p.tpt - 1) / p.tpt) * p.ncb;
    p.bn = pick_bn(rb);
    p.ntiles = p.bn ? rb / p.bn : 0;
    const int ctas = std::max(1, p.mtiles * p.ntiles);
    // two resident CTAs per SM: split the voxels so that the grid is at most one wave of 2 x 152
    // (a second, nearly empty wave would double the time)
    int splits = std::max(1, std::min(p.nchunks, (2 * 152) / ctas));
    p.cps = (p.nchunks + splits - 1) / splits;
    p.splits = (p.nchunks + p.cps - 1) / p.cps;
    p.nshift = taps == 27 ? 3 : 1;
    p.xt_bytes = p.mn ? 0 : round256((size_t)p.nshift * ci * p.vpad * 2);
    p.gyt_bytes = p.mn ? 0 : round256((size_t)co * p.vpad * 2);
    p.part_bytes = round256((size_t)p.splits * taps * ci * co * 4);
    p.bias_bytes = round256((size_t)kBiasBlocks * co * 4);
    return p;
}

// The form with whole rows of a plane, or S = 0 where it does not apply: 27 taps, rows of at most 128 voxels, and
// two stages of shared memory.
struct WgRowPlan {
    int S, swap, R, kcy, nchunks, cps, splits, cm, cn, variants, groups, nmb, nnb;
    uint32_t offN, stride;
    size_t part_bytes;
};

WgRowPlan wg_row_plan(ConvVol v, int taps, int ci, int co) {
    WgRowPlan p{};
    if (taps != 27 || v.nx > 128 || v.nx % 8 || ci % 32 || co % 32) return p;
    // the roles with fewer MMAs: rows a (in blocks of 128, 64 or 32 channels), columns b (of 64 or 32)
    auto block = [](int a) { return a % 128 == 0 ? 128 : a % 64 == 0 ? 64 : 32; };
    auto mmas = [&](int a, int b) {
        const int cm = block(a), var = 128 / cm;
        return (int64_t)(a / cm) * ((9 + var - 1) / var) * (b / std::min(block(b), 64));
    };
    p.swap = mmas(ci, co) < mmas(co, ci);  // rows = input, columns = gradient
    const int a = p.swap ? ci : co, b = p.swap ? co : ci;
    p.cm = block(a);
    p.variants = 128 / p.cm;
    p.groups = (9 + p.variants - 1) / p.variants;
    p.nmb = a / p.cm;
    // Rows per step: the two rows of halo cost less the more there are, up to 256 voxels with three stages.  Two rows
    // of 120 voxels with 64 columns leave room for one stage only: 32 columns then.
    const int even = v.nx % 16 ? 2 : 1;  // K is a multiple of 16 voxels
    const int most = std::min((v.ny + even - 1) / even * even, std::max(256 / v.nx, even) / even * even);
    const uint32_t room = 227 * 1024 - 1024 - 1024;  // less alignment and barriers
    for (int cn = std::min(block(b), 64); cn >= 32 && !p.S; cn /= 2)
        for (int least : {3, 2})
            for (int R = most; R >= even && !p.S; R -= even) {
                const uint32_t offN = (uint32_t)v.nx * R * 256;
                const uint32_t stride = (offN + (uint32_t)v.nx * (R + 2) * cn * 2 + 1023u) & ~1023u;
                const int S = (int)std::min<uint32_t>(8, room / stride);
                if (S < least) continue;
                p.S = S;
                p.R = R;
                p.cn = cn;
                p.offN = offN;
                p.stride = stride;
            }
    if (!p.S) return p;
    p.nnb = b / p.cn;
    p.kcy = (v.ny + p.R - 1) / p.R;
    p.nchunks = p.kcy * v.nz;
    const int ctas = p.groups * p.nmb * p.nnb;
    // One CTA per SM, in as few waves as keep the voxels that an accumulator takes at or below those of the boxes' form.
    const int64_t most_voxels = (int64_t)wg_plan(v, taps, ci, co).cps * 64;
    const int sets = wgrad_sets(p.cn), per_step = (v.nx * p.R / 16 + sets - 1) / sets * 16;
    for (int waves = 1;; ++waves) {
        const int splits = (int)std::max<int64_t>(1, std::min<int64_t>(p.nchunks, (int64_t)waves * 152 / ctas));
        p.cps = (p.nchunks + splits - 1) / splits;
        if (p.cps == 1 || (int64_t)p.cps * per_step <= most_voxels) break;
    }
    p.splits = (p.nchunks + p.cps - 1) / p.cps;
    p.part_bytes = round256((size_t)p.splits * 27 * ci * co * 4);
    return p;
}

template <int CN>
cudaError_t launch_wgrow(cudaStream_t st, dim3 grid, const CUtensorMap &mm, const CUtensorMap &mn, const WgRowArgs &a) {
    static cudaError_t attr = set_smem(conv_wgrad_rows<CN>, 227 * 1024);
    if (attr != cudaSuccess) return attr;
    conv_wgrad_rows<CN><<<grid, kThreads, a.offBar + 1024 + 1024, st>>>(mm, mn, a);
    return cudaGetLastError();
}

// Shared memory of the folded kernel for this shape, or 0 where it is not the one to use: 27 taps, 32 or 64 output
// channels, rows of nx voxels that tile a 128-voxel tile's start addresses (nx a multiple of 8, at most 128) and at
// least half fill it, and a second tile in y.
size_t fold_plan(ConvVol v, int taps, int ci, int co, FoldArgs *g) {
    if (taps != 27 || (co != 32 && co != 64) || v.nx % 8 || v.nx > 128) return 0;
    const int bh = std::min(v.ny, 128 / v.nx);
    if (bh * v.nx < 64 || v.ny <= bh) return 0;
    const int BK = ci % 64 == 0 ? 64 : 32, rb = 2 * BK, nkb = ci / BK;
    const int dys = fold_dys(co, BK);
    const uint32_t slot = 3u * co * rb * dys, all = 9u * nkb / dys * slot;
    g->boxA = (uint32_t)v.nx * (2 * bh + 2) * rb;
    g->strideA = (g->boxA + (uint32_t)(128 - bh * v.nx) * rb + 1023u) & ~1023u;
    const uint32_t room = 227 * 1024 - 1024 - kFoldTail;  // less alignment
    // weight slots that cover a load's latency: a slot's MMAs take 410 (co = 64, BK = 32) to 820 cycles
    const int least = dys == 3 ? 2 : co == 64 && BK == 64 ? 3 : 4;
    g->S = 0;
    for (int march = nkb == 1; march >= 0 && !g->S; --march) {
        // boxes: three planes; else two, or as many as there is room for with their weights
        const int least_boxes = march ? 3 : 2;
        const int boxes = march ? 3 : std::max(2, std::min<int>(kFoldMaxStages, room / (g->strideA + 3 / dys * slot)));
        if (all + least_boxes * g->strideA <= room) {
            g->SB = 0;
            g->S = (int)std::min<uint32_t>(kFoldMaxStages, (room - all) / g->strideA);
            g->offA = all;
        } else if (boxes * g->strideA + least * slot <= room) {
            g->SB = (int)std::min<uint32_t>(kFoldMaxWeights, (room - boxes * g->strideA) / slot);
            g->S = (int)std::min<uint32_t>(kFoldMaxStages, (room - g->SB * slot) / g->strideA);
            g->offA = g->SB * slot;
        }
        g->march = march;
    }
    if (!g->S) return 0;
    g->offBar = g->offA + g->S * g->strideA;
    g->f.bh = bh;
    g->f.ty = (v.ny + 2 * bh - 1) / (2 * bh);
    g->nz = v.nz;
    g->pairs = g->f.ty * v.nz;
    return g->offBar + kFoldTail + 1024;
}

template <int CO, int BK>
cudaError_t launch_fold(cudaStream_t st, size_t smem, const CUtensorMap &ma, const CUtensorMap &mb, const FoldArgs &g) {
    static cudaError_t attr = set_smem(conv_fold_tc<CO, BK>, 227 * 1024);
    if (attr != cudaSuccess) return attr;
    conv_fold_tc<CO, BK><<<std::min(g.pairs, 152), kFoldThreads, smem, st>>>(ma, mb, g);
    return cudaGetLastError();
}

}  // namespace

rsv_status conv_fwd(cudaStream_t st, ConvVol v, int taps, int ci, int co, const __nv_bfloat16 *x, int ldx,
                    const __nv_bfloat16 *w, const float *bias, int relu, const __nv_bfloat16 *mask, int ldm,
                    __nv_bfloat16 *y, int ldy, float *y32, int *err, uint64_t timeout_ns, const int *gate) {
    if (v.nx <= 0 || v.ny <= 0 || v.nz <= 0 || (taps != 1 && taps != 27) || ci <= 0 || ci % 32 || co <= 0 ||
        co % 32 || !x || !w || (!y && !y32) || ldx < ci || ldx % 8 || (y && (ldy < co || ldy % 8)) ||
        (mask && (ldm < co || ldm % 8)))
        return RSV_EINVAL;
    if (!aligned16(x) || !aligned16(w) || (y && !aligned16(y)) || (y32 && !aligned16(y32)) ||
        (mask && !aligned16(mask)))
        return RSV_EINVAL;
    const int BK = ci % 64 == 0 ? 64 : 32;
    const int BN = pick_bn(co);
    FwdArgs a{};
    a.nx = v.nx;
    a.ny = v.ny;
    a.nz = v.nz;
    a.bw = std::min(v.nx, 128);
    a.bh = std::min(v.ny, 128 / a.bw);
    a.bd = std::min(v.nz, 128 / (a.bw * a.bh));
    a.tx = (v.nx + a.bw - 1) / a.bw;
    a.ty = (v.ny + a.bh - 1) / a.bh;
    const int tz = (v.nz + a.bd - 1) / a.bd;
    a.taps = taps;
    a.nkb = ci / BK;
    a.ci = ci;
    a.n_total = co;
    a.bias = bias;
    a.relu = relu;
    a.mask = mask;
    a.ldm = ldm;
    a.y = y;
    a.ldy = ldy;
    a.y32 = y32;
    a.err = err;
    a.timeout_ns = timeout_ns;
    a.gate = gate;
    CUtensorMap ma, mb;
    FoldArgs g{};
    if (const size_t smem = fold_plan(v, taps, ci, co, &g)) {
        const int bh = g.f.bh, ty = g.f.ty;
        g.f = a;
        g.f.bw = v.nx;
        g.f.bh = bh;
        g.f.bd = 1;
        g.f.ty = ty;
        g.f.nkb = ci / BK;
        const uint64_t dims[4] = {(uint64_t)ci, (uint64_t)v.nx, (uint64_t)v.ny, (uint64_t)v.nz};
        const uint64_t strides[3] = {(uint64_t)ldx * 2, (uint64_t)v.nx * ldx * 2, (uint64_t)v.nx * v.ny * ldx * 2};
        const uint32_t box[4] = {(uint32_t)BK, (uint32_t)v.nx, (uint32_t)(2 * bh + 2), 1u};
        RSV_TRY(make_map(&ma, x, 4, dims, strides, box, BK * 2));
        const uint64_t wdims[3] = {(uint64_t)ci, (uint64_t)co, (uint64_t)taps};
        const uint64_t wstrides[2] = {(uint64_t)taps * ci * 2, (uint64_t)ci * 2};
        const uint32_t wbox[3] = {(uint32_t)BK, (uint32_t)co, 3u * fold_dys(co, BK)};  // the x taps of one or three (dz, dy)
        RSV_TRY(make_map(&mb, w, 3, wdims, wstrides, wbox, BK * 2));
        RSV_CUDA_TRY(co == 32 ? (BK == 32 ? launch_fold<32, 32>(st, smem, ma, mb, g) : launch_fold<32, 64>(st, smem, ma, mb, g))
                              : (BK == 32 ? launch_fold<64, 32>(st, smem, ma, mb, g) : launch_fold<64, 64>(st, smem, ma, mb, g)));
        count_launches(1);
        return RSV_OK;
    }
    {
        const uint64_t dims[4] = {(uint64_t)ci, (uint64_t)v.nx, (uint64_t)v.ny, (uint64_t)v.nz};
        const uint64_t strides[3] = {(uint64_t)ldx * 2, (uint64_t)v.nx * ldx * 2, (uint64_t)v.nx * v.ny * ldx * 2};
        const uint32_t box[4] = {(uint32_t)BK, (uint32_t)a.bw, (uint32_t)a.bh, (uint32_t)a.bd};
        RSV_TRY(make_map(&ma, x, 4, dims, strides, box, BK * 2));
    }
    {
        const uint64_t dims[2] = {(uint64_t)taps * ci, (uint64_t)co};
        const uint64_t strides[1] = {(uint64_t)taps * ci * 2};
        const uint32_t box[2] = {(uint32_t)BK, (uint32_t)BN};
        RSV_TRY(make_map(&mb, w, 2, dims, strides, box, BK * 2));
    }
    const dim3 grid(a.tx * a.ty * tz, co / BN);
    RSV_CUDA_TRY(BK == 64 ? launch_fwd_bk<64>(BN, st, grid, ma, mb, a) : launch_fwd_bk<32>(BN, st, grid, ma, mb, a));
    count_launches(1);
    return RSV_OK;
}

rsv_status conv_flip(cudaStream_t st, int ci, int co, const __nv_bfloat16 *w, __nv_bfloat16 *wt) {
    if (ci <= 0 || co <= 0 || !w || !wt) return RSV_EINVAL;
    const int64_t total = (int64_t)ci * 27 * co;
    flip_weights<<<(int)std::min<int64_t>((total + 255) / 256, 4096), 256, 0, st>>>(w, ci, co, wt);
    RSV_CUDA_TRY(cudaGetLastError());
    count_launches(1);
    return RSV_OK;
}

size_t conv_wgrad_scratch(ConvVol v, int taps, int ci, int co) {
    const WgPlan p = wg_plan(v, taps, ci, co);
    return std::max(p.xt_bytes + p.gyt_bytes + p.part_bytes, wg_row_plan(v, taps, ci, co).part_bytes) + p.bias_bytes;
}

rsv_status conv_wgrad(cudaStream_t st, ConvVol v, int taps, int ci, int co, const __nv_bfloat16 *x, int ldx,
                      const __nv_bfloat16 *gy, int ldgy, float *gw, float *gb, void *scratch, int *err,
                      uint64_t timeout_ns) {
    if (v.nx <= 0 || v.ny <= 0 || v.nz <= 0 || v.nx % 8 || (taps != 1 && taps != 27) || ci <= 0 || ci % 32 ||
        co <= 0 || co % 32 || !x || !gy || !gw || !scratch || ldx < ci || ldgy < co)
        return RSV_EINVAL;
    const WgPlan p = wg_plan(v, taps, ci, co);
    if (!aligned16(scratch)) return RSV_EINVAL;
    const bool aligned = aligned16(x) && aligned16(gy) && ldx % 8 == 0 && ldgy % 8 == 0;
    if (p.mn && !aligned) return RSV_EINVAL;
    const int64_t V = (int64_t)v.nx * v.ny * v.nz, total = (int64_t)taps * ci * co;
    const int wblocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
    // the partial sums of both gradients, added in a fixed order
    auto reduce = [&](const float *part, int splits, int swap, float *bpart) -> rsv_status {
        if (gb) {
            bias_grad_cl<<<kBiasBlocks, 256, 0, st>>>(gy, ldgy, co, V, bpart);
            RSV_CUDA_TRY(cudaGetLastError());
        }
        wgrad_reduce<<<wblocks + (gb ? (co + 7) / 8 : 0), 256, 0, st>>>(part, splits, taps, ci, co, gw, swap, wblocks,
                                                                      bpart, kBiasBlocks, gb);
        RSV_CUDA_TRY(cudaGetLastError());
        count_launches(gb ? 3 : 2);
        return RSV_OK;
    };
    const WgRowPlan rp = aligned ? wg_row_plan(v, taps, ci, co) : WgRowPlan{};
    if (rp.S) {
        WgRowArgs a{};
        a.nx = v.nx;
        a.R = rp.R;
        a.kcy = rp.kcy;
        a.nchunks = rp.nchunks;
        a.cps = rp.cps;
        a.cm = rp.cm;
        a.variants = rp.variants;
        a.nmb = rp.nmb;
        a.ca = rp.swap ? ci : co;
        a.cb = rp.swap ? co : ci;
        a.sgn = rp.swap ? -1 : 1;
        a.S = rp.S;
        a.offN = rp.offN;
        a.stride = rp.stride;
        a.offBar = rp.S * rp.stride;
        a.partial = (float *)scratch;
        a.err = err;
        a.timeout_ns = timeout_ns;
        CUtensorMap mm, mn;
        auto map = [&](CUtensorMap *m, bool input, int cols, int rows) {
            const __nv_bfloat16 *base = input ? x : gy;
            const uint64_t ld = input ? ldx : ldgy;
            const uint64_t dims[4] = {(uint64_t)(input ? ci : co), (uint64_t)v.nx, (uint64_t)v.ny, (uint64_t)v.nz};
            const uint64_t strides[3] = {ld * 2, (uint64_t)v.nx * ld * 2, (uint64_t)v.nx * v.ny * ld * 2};
            const uint32_t box[4] = {(uint32_t)cols, (uint32_t)v.nx, (uint32_t)rows, 1u};
            return make_map(m, base, 4, dims, strides, box, cols * 2);
        };
        RSV_TRY(map(&mm, rp.swap, std::min(rp.cm, 64), rp.R));
        RSV_TRY(map(&mn, !rp.swap, rp.cn, rp.R + 2));
        const dim3 grid(rp.groups * rp.nmb, rp.nnb, rp.splits);
        RSV_CUDA_TRY(rp.cn == 64 ? launch_wgrow<64>(st, grid, mm, mn, a) : launch_wgrow<32>(st, grid, mm, mn, a));
        return reduce(a.partial, rp.splits, rp.swap ? 0 : 1, (float *)((char *)scratch + rp.part_bytes));
    }
    if (p.mn) {
        float *part = (float *)((char *)scratch + p.xt_bytes + p.gyt_bytes);
        float *bpart = (float *)((char *)part + p.part_bytes);
        WgMnArgs a{};
        a.bw = p.bw;
        a.bh = p.bh;
        a.bd = p.bd;
        a.kcx = p.kcx;
        a.kcy = p.kcy;
        a.nchunks = p.nchunks;
        a.cps = p.cps;
        a.taps = taps;
        a.ci = p.swap ? co : ci;
        a.cblk = p.cblk;
        a.tpt = p.tpt;
        a.ncb = p.ncb;
        a.colA = p.cblk >= 64 ? 64 : 32;
        a.co = p.swap ? ci : co;
        a.colB = p.bn % 64 == 0 ? 64 : 32;
        a.sgn = p.swap ? -1 : 1;
        a.partial = part;
        a.err = err;
        a.timeout_ns = timeout_ns;
        // row operand: the tap-shifted one (x, or gy when swapped); column operand: the other
        const __nv_bfloat16 *rowp = p.swap ? gy : x, *colp = p.swap ? x : gy;
        const int rowld = p.swap ? ldgy : ldx, colld = p.swap ? ldx : ldgy;
        CUtensorMap mx, mg;
        {
            const uint64_t dims[4] = {(uint64_t)a.ci, (uint64_t)v.nx, (uint64_t)v.ny, (uint64_t)v.nz};
            const uint64_t strides[3] = {(uint64_t)rowld * 2, (uint64_t)v.nx * rowld * 2,
                                         (uint64_t)v.nx * v.ny * rowld * 2};
            const uint32_t box[4] = {(uint32_t)a.colA, (uint32_t)p.bw, (uint32_t)p.bh, (uint32_t)p.bd};
            RSV_TRY(make_map(&mx, rowp, 4, dims, strides, box, a.colA * 2));
        }
        {
            const uint64_t dims[4] = {(uint64_t)a.co, (uint64_t)v.nx, (uint64_t)v.ny, (uint64_t)v.nz};
            const uint64_t strides[3] = {(uint64_t)colld * 2, (uint64_t)v.nx * colld * 2,
                                         (uint64_t)v.nx * v.ny * colld * 2};
            const uint32_t box[4] = {(uint32_t)a.colB, (uint32_t)p.bw, (uint32_t)p.bh, (uint32_t)p.bd};
            RSV_TRY(make_map(&mg, colp, 4, dims, strides, box, a.colB * 2));
        }
        RSV_CUDA_TRY(launch_wgmn(p.bn, st, dim3(p.mtiles, p.ntiles, p.splits), mx, mg, a));
        return reduce(part, p.splits, p.swap ? 1 : 0, bpart);
    }
    __nv_bfloat16 *xt = (__nv_bfloat16 *)scratch;
    __nv_bfloat16 *gyt = (__nv_bfloat16 *)((char *)scratch + p.xt_bytes);
    float *part = (float *)((char *)scratch + p.xt_bytes + p.gyt_bytes);
    const int prow = (v.nz + 2) * (v.ny + 2), xchunks = (v.nx + kVmChunk - 1) / kVmChunk;
    to_voxel_major<<<dim3(prow, ci / 32, xchunks), 256, 0, st>>>(x, ldx, ci, v.nx, v.ny, v.nz, p.nshift, p.vpad, xt);
    RSV_CUDA_TRY(cudaGetLastError());
    to_voxel_major<<<dim3(prow, co / 32, xchunks), 256, 0, st>>>(gy, ldgy, co, v.nx, v.ny, v.nz, 1, p.vpad, gyt);
    RSV_CUDA_TRY(cudaGetLastError());
    CUtensorMap ma, mb;
    {
        const uint64_t dims[3] = {(uint64_t)p.vpad, (uint64_t)ci, (uint64_t)p.nshift};
        const uint64_t strides[2] = {(uint64_t)p.vpad * 2, (uint64_t)ci * p.vpad * 2};
        const uint32_t box[3] = {64u, (uint32_t)p.cblk, 1u};
        RSV_TRY(make_map(&ma, xt, 3, dims, strides, box, 128));
    }
    {
        const uint64_t dims[2] = {(uint64_t)p.vpad, (uint64_t)co};
        const uint64_t strides[1] = {(uint64_t)p.vpad * 2};
        const uint32_t box[2] = {64u, (uint32_t)p.bn};
        RSV_TRY(make_map(&mb, gyt, 2, dims, strides, box, 128));
    }
    WgArgs a{};
    a.nchunks = p.nchunks;
    a.cps = p.cps;
    a.taps = taps;
    a.ci = ci;
    a.cblk = p.cblk;
    a.tpt = p.tpt;
    a.ncb = p.ncb;
    a.plane = (v.ny + 2) * v.nx;
    a.row = v.nx;
    a.co = co;
    a.partial = part;
    a.err = err;
    a.timeout_ns = timeout_ns;
    RSV_CUDA_TRY(launch_wg(p.bn, st, dim3(p.mtiles, p.ntiles, p.splits), ma, mb, a));
    wgrad_reduce<<<wblocks, 256, 0, st>>>(part, p.splits, taps, ci, co, gw, 0, wblocks, nullptr, 0, nullptr);
    RSV_CUDA_TRY(cudaGetLastError());
    int n = 4;
    if (gb) {
        // the partial sums of the weight gradient are consumed: reuse their buffer
        bias_grad<<<dim3(co, kBgChunks), 256, 0, st>>>(gyt, p.vpad, part);
        bias_grad_final<<<(co + 127) / 128, 128, 0, st>>>(part, co, gb);
        RSV_CUDA_TRY(cudaGetLastError());
        n = 6;
    }
    count_launches(n);
    return RSV_OK;
}

}  // namespace rsv

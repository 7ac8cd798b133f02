// cnn.cu -- a10 learned clutter filter: a 4-layer 3D convolutional network
// (2 -> 32 -> 32 -> 32 -> 2 channels, 5 frames x 3 x 3 pixel kernels, zero
// "same" padding, ReLU between layers) applied to the normalised IQ
// ensemble, its training step (forward, backward, Adam) and the power
// Doppler of its output.  The paper proposes filters learned from simulated
// ensembles as future work (Sec. 1, Sec. 4); this is that filter's hot path.
//
// Layout: activations channels-last, [N][F][Z][X][32] BF16 (the 2-channel
// input and output are zero-padded to 32 channels, so every layer is one
// shape).  Forward convolution = implicit GEMM on the tcgen05 tensor cores
// (conv_kernel below): one tile is 128 voxels of one frame x 32 output
// channels; K runs over 45 taps x 32 input channels.  The weights (90 KB) stay
// resident in shared memory for the CTA's lifetime; TMA's zero fill outside
// the volume is the "same" padding.  Epilogues: bias + ReLU -> BF16, bias ->
// FP32 (last layer), or gradient x ReLU mask -> BF16 (backward).
//
// The data gradient of a layer is the same convolution with the kernel
// flipped in all three axes and its channel roles swapped; the weight
// gradient (a reduction over voxels) runs on the warp-level tensor cores
// with FP32 accumulators held in registers (wgrad_kernel).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstring>

#include "fq_internal.cuh"
#include "tc.cuh"

using namespace fqtc;

namespace {

constexpr int C = 32;                 // channels of every activation tensor
constexpr int NTAP = 45;              // 5 x 3 x 3
constexpr int TILE_M = 128;           // voxels per tile: 4 depth rows x 32 lateral
constexpr int TILE_Z = 4, TILE_X = 32;
constexpr int ROWB = C * 2;           // 64 bytes per operand row
constexpr int W_TAP_BYTES = C * ROWB;         // 2 KB per tap
constexpr int W_BYTES = NTAP * W_TAP_BYTES;   // 90 KB
constexpr int CONV_THREADS = 192;     // warp 0 TMA, warp 1 MMA + TMEM owner, warps 2-5 epilogue

enum Epi { EPI_RELU_BF16 = 0, EPI_LINEAR_F32 = 1, EPI_MASK_BF16 = 2 };

struct ConvDims {
    int N, F, Z, X;
    int run;           // frames per work unit of the convolutions
    int zb, xb;        // depth and lateral blocks of a frame, the last one possibly ragged
    int walk_tiles;    // N zb xb F: tile = column * F + frame
};

struct Column {
    int n, z0, x0;
};

__device__ __forceinline__ Column column_at(const ConvDims &d, int col)
{
    Column c;
    c.x0 = (col % d.xb) * TILE_X;
    col /= d.xb;
    c.z0 = (col % d.zb) * TILE_Z;
    c.n = col / d.zb;
    return c;
}

// The tiles of a CTA are a contiguous range; a segment is its part in one
// column: output frames fa .. fb - 1.
__device__ __forceinline__ int range_begin(int tiles) { return (int)((int64_t)tiles * blockIdx.x / gridDim.x); }
__device__ __forceinline__ int range_end(int tiles) { return (int)((int64_t)tiles * (blockIdx.x + 1) / gridDim.x); }

// Epilogue of one accumulator row (32 channels of voxel `vox`).
template <int EPI>
__device__ __forceinline__ void epilogue_store(const float (&v)[32], const float *s_bias, int64_t vox, void *out,
                                               const __nv_bfloat16 *mask)
{
    if (EPI == EPI_LINEAR_F32) {
        float4 *o = reinterpret_cast<float4 *>((float *)out + vox * C);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            o[i] = make_float4(v[4 * i] + s_bias[4 * i], v[4 * i + 1] + s_bias[4 * i + 1],
                               v[4 * i + 2] + s_bias[4 * i + 2], v[4 * i + 3] + s_bias[4 * i + 3]);
    } else {
        float m[32];
        if (EPI == EPI_MASK_BF16) {
            const uint4 *mp = reinterpret_cast<const uint4 *>(mask + vox * C);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint4 u = mp[i];
                const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float2 fl = __bfloat1622float2(h[k]);
                    m[8 * i + 2 * k] = fl.x;
                    m[8 * i + 2 * k + 1] = fl.y;
                }
            }
        }
        uint4 packed[4];
        __nv_bfloat162 *pb = reinterpret_cast<__nv_bfloat162 *>(packed);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            float a0 = v[2 * k], a1 = v[2 * k + 1];
            if (EPI == EPI_RELU_BF16) {
                a0 = fmaxf(a0 + s_bias[2 * k], 0.0f);
                a1 = fmaxf(a1 + s_bias[2 * k + 1], 0.0f);
            } else {
                a0 = m[2 * k] > 0.0f ? a0 : 0.0f;
                a1 = m[2 * k + 1] > 0.0f ? a1 : 0.0f;
            }
            pb[k] = __floats2bfloat162_rn(a0, a1);
        }
        uint4 *o = reinterpret_cast<uint4 *>((__nv_bfloat16 *)out + vox * C);
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = packed[i];
    }
}

// ------------------------------------------------------------ convolution --
// A CTA takes work units (one 128-voxel tile of a frame x a run of frames)
// and walks the input frames of a unit in order through a ring of
// shared-memory slots, each one frame of the tile with its halo.
//
// An MMA of 32 output channels is bound by its operand reads (4 KB of A for
// 65k products: at most 57% of the tensor rate), so input frame g goes into
// all five outputs f = g - 2 .. g + 2 it reaches at once: their weights stand
// side by side (N = 160, block b of 32 for f = g - 2 + b, dt = 2 - b), and
// their accumulators are consecutive 32-column slots of a ring of 16 in tensor
// memory (two MMAs where the ring wraps; a ring of 8 wraps twice as often,
// 5.74 against 5.34 ms for the whole filter).  Each input frame is loaded and
// read once per unit instead of five times; the other accumulators leave the
// epilogue its time.  200 x 256 x 256, the filter with its packing and power
// Doppler: 10.9 ms with one output per MMA, 5.34 ms now (0.9 PFLOP/s of the
// padded products, tensor pipe 40-46%); a training step's seven convolutions
// (4 x 64 x 32 x 32) 1.24 -> 0.26 ms.
//
// Two tiles:
//  WIDE (Z not a multiple of 4, X of 128): 128 pixels of one depth row.  A slot holds
//    rows z - 1 .. z + 1 x pixels x0 - 1 .. x0 + 128 in 4 chunks of 8
//    channels, each a [3][130] array of 16-byte rows (one TMA box per chunk;
//    zero fill outside the volume).  In this no-swizzle K-major layout rows
//    sit 16 bytes apart, so the operand of tap (dz, dx) is the slot at row
//    offset (1 + dz) 130 + 1 + dx: a descriptor.
//  otherwise (X a multiple of 32): 4 depth rows x 32 pixels (the same time as
//    WIDE where both fit).  A slot holds
//    three copies, shifted by dx, of rows z0 - 1 .. z0 + 4 x 32 pixels, 64
//    bytes a voxel with the 64-byte swizzle (one TMA box each): the operand
//    of (dz, dx) is copy dx from row 32 (1 + dz) on, a whole number of swizzle
//    atoms.  Three boxes of 12 KB a frame where one box per tap took 45 of 8.
template <bool WIDE>
struct Tile {
    static constexpr int Z = WIDE ? 1 : TILE_Z, X = WIDE ? 128 : TILE_X;
    static constexpr int W = X + 2;                               // WIDE: with the lateral halo
    static constexpr int BOX = WIDE ? 3 * W * 16 : (TILE_Z + 2) * TILE_X * ROWB;
    static constexpr int NBOX = WIDE ? 4 : 3;
    static constexpr int STRIDE = (BOX + 127) / 128 * 128;        // of the boxes in a slot
    static constexpr int SLOT = NBOX * STRIDE;                    // 25088 or 36864 bytes
    static constexpr int SLOTS = WIDE ? 5 : 3;
    static constexpr int SMEM = W_BYTES + SLOTS * SLOT + 1024;
};

// K-major shared-memory matrix descriptor without swizzle: 8-row core
// matrices of 16-byte rows; `lbo` = bytes between core matrices along K,
// `sbo` = bytes between 8-row groups.
__device__ __forceinline__ uint64_t nosw_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version; layout type 0 = no swizzle
    return d;
}

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

struct RingUnit {
    int n, z0, x0, fa, fb;
};

template <bool WIDE>
__device__ __forceinline__ RingUnit ring_unit(const ConvDims &d, int u)
{
    const int nfc = (d.F + d.run - 1) / d.run, nxb = d.X / Tile<WIDE>::X, nzb = d.Z / Tile<WIDE>::Z;
    RingUnit r;
    const int fc = u % nfc;
    u /= nfc;
    r.x0 = (u % nxb) * Tile<WIDE>::X;
    u /= nxb;
    r.z0 = (u % nzb) * Tile<WIDE>::Z;
    r.n = u / nzb;
    r.fa = fc * d.run;
    r.fb = min(d.F, r.fa + d.run);
    return r;
}

constexpr int RING_ACC = 16;                         // accumulators of 32 columns in tensor memory
constexpr int RING_TMEM = RING_ACC * C;
constexpr int RING_WTAP = 5 * W_TAP_BYTES;           // weights of one (dz, dx), all dt
constexpr int RING_WCHUNK = RING_WTAP / 4;           // WIDE: of 8 input channels
constexpr uint32_t kRingIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TILE_M >> 4) << 24);  // | N / 8 << 17

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// input frames of a unit: those in the volume that reach its outputs (a frame
// outside contributes nothing)
__device__ __forceinline__ int ring_g0(const RingUnit &r) { return max(0, r.fa - 2); }
__device__ __forceinline__ int ring_g1(const RingUnit &r, int F) { return min(F - 1, r.fb + 1); }

template <int EPI, bool WIDE>
__global__ void __launch_bounds__(CONV_THREADS, 1)
    conv_kernel(const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap w_map,
                const __nv_bfloat16 *__restrict__ wchunk, const ConvDims d, int units, const float *__restrict__ bias, void *__restrict__ out,
                const __nv_bfloat16 *__restrict__ mask, int *__restrict__ status)
{
    using T = Tile<WIDE>;
    constexpr int RING_SLOTS = T::SLOTS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *w_s = base;
    unsigned char *ring = base + W_BYTES;
    __shared__ __align__(8) uint64_t slot_full[RING_SLOTS], slot_free[RING_SLOTS], acc_full[RING_ACC], acc_empty[RING_ACC], w_bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;
    __shared__ float s_bias[C];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < RING_SLOTS; ++s) {
            mbar_init(&slot_full[s], 1);
            mbar_init(&slot_free[s], 1);
        }
        for (int b = 0; b < RING_ACC; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        mbar_init(&w_bar, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < C) s_bias[threadIdx.x] = bias ? bias[threadIdx.x] : 0.0f;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(RING_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            // ---- producer: weights once, then the frames of each unit in order,
            // load i into slot i % RING_SLOTS
            mbar_expect_tx(&w_bar, W_BYTES);
            if constexpr (WIDE) {
                // [tap][4 chunks][32 rows][8] to [dz, dx][chunk][2 - dt][row][8]
                for (int t = 0; t < NTAP; ++t)
                    for (int c = 0; c < 4; ++c)
                        bulk_load(w_s + (t % 9) * RING_WTAP + c * RING_WCHUNK + (4 - t / 9) * (RING_WCHUNK / 5),
                                  (const unsigned char *)wchunk + (t * 4 + c) * (W_TAP_BYTES / 4), W_TAP_BYTES / 4, &w_bar);
            } else {
                for (int t = 0; t < NTAP; ++t)  // tap (dt, dz, dx) to block 2 - dt of (dz, dx)
                    tma_load_2d(w_s + ((t % 9) * 5 + 4 - t / 9) * W_TAP_BYTES, &w_map, &w_bar, 0, t * C);
            }
            uint32_t i = 0;
            bool fail = false;
            for (int u = blockIdx.x; u < units && !fail; u += gridDim.x) {
                const RingUnit r = ring_unit<WIDE>(d, u);
                for (int g = ring_g0(r); g <= ring_g1(r, d.F); ++g, ++i) {
                    const int s = i % RING_SLOTS;
                    if (!mbar_wait(&slot_free[s], ((i / RING_SLOTS) & 1u) ^ 1u)) {
                        fail = true;
                        break;
                    }
                    mbar_expect_tx(&slot_full[s], T::NBOX * T::BOX);
                    unsigned char *dst = ring + s * T::SLOT;
                    for (int k = 0; k < T::NBOX; ++k)
                        tma_load_5d(dst + k * T::STRIDE, &in_map, &slot_full[s], WIDE ? 8 * k : 0,
                                    WIDE ? r.x0 - 1 : r.x0 - 1 + k, r.z0 - 1, g, r.n);
                }
            }
            if (fail) s_fail = 1;
            // let issued copies land before the CTA can exit, whoever gave up
            for (uint32_t k = i > RING_SLOTS ? i - RING_SLOTS : 0; k < i; ++k)
                mbar_wait(&slot_full[k % RING_SLOTS], (k / RING_SLOTS) & 1u);
            mbar_wait(&w_bar, 0);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer.  Descriptors: one base per operand array; a tap's
            // operand is the base plus its byte offset / 16 in the start-address
            // field (addresses stay below 256 KB, so the field never carries).
            bool fail = !mbar_wait(&w_bar, 0);
            tc_fence_after();
            uint32_t i = 0, jb = 0;  // loads consumed; outputs of the units before this one
            const uint64_t ring_d = WIDE ? nosw_desc(smem_u32(ring), T::STRIDE, 128) : sw64_desc(smem_u32(ring));
            const uint64_t w_d = WIDE ? nosw_desc(smem_u32(w_s), RING_WCHUNK, 128) : sw64_desc(smem_u32(w_s));
            constexpr int BLOCK = WIDE ? C * 16 : W_TAP_BYTES;  // weight bytes between outputs
            for (int u = blockIdx.x; u < units && !fail; u += gridDim.x) {
                const RingUnit r = ring_unit<WIDE>(d, u);
                const int g0 = ring_g0(r), g1 = ring_g1(r, d.F);
                for (int g = g0; g <= g1; ++g, ++i) {
                    // outputs lo .. hi take frame g; from `fresh` on for the first time
                    const int lo = max(r.fa, g - 2), hi = min(r.fb - 1, g + 2);
                    const int fresh = g == g0 ? lo : g + 2;
                    for (int f = fresh; f <= hi && !fail; ++f) {
                        const uint32_t j = jb + (uint32_t)(f - r.fa);
                        if (!mbar_wait(&acc_empty[j % RING_ACC], ((j / RING_ACC) & 1u) ^ 1u)) fail = true;
                    }
                    const int s = i % RING_SLOTS;
                    if (fail || !mbar_wait(&slot_full[s], (i / RING_SLOTS) & 1u)) { fail = true; break; }
                    tc_fence_after();
                    const uint64_t a0 = ring_d + (uint64_t)((s * T::SLOT) >> 4);
                    // K step 0 or steps 1 .. 17 (step = 2 tap + half of the channels) of
                    // outputs fa .. fb, in two runs where the accumulator ring wraps
                    auto run = [&](int fa, int fb, bool first) {
                        const uint32_t c0 = (jb + (uint32_t)(fa - r.fa)) % RING_ACC;
                        const int n = fb - fa + 1, n1 = min(n, RING_ACC - (int)c0);
                        for (int part = 0; part < 2; ++part) {
                            const int m = part ? n - n1 : n1;
                            if (m <= 0) break;
                            const uint32_t acc = part ? tmem : tmem + c0 * C;
                            const uint32_t idesc = kRingIdesc | ((uint32_t)(m * C / 8) << 17);
                            const uint64_t bd = w_d + (uint64_t)(((fa - (g - 2) + (part ? n1 : 0)) * BLOCK) >> 4);
                            if (first) {
                                mma_bf16(acc, a0, bd, idesc, fa >= fresh ? 0u : 1u);
                                continue;
                            }
#pragma unroll
                            for (int k = 1; k < 18; ++k) {
                                const int dz = k / 6, dx = (k / 2) % 3, kk = k & 1;
                                // second 16 channels: two chunks on, or 32 bytes on in the row
                                const int ao = WIDE ? (dz * T::W + dx) * 16 + kk * 2 * T::STRIDE
                                                    : dx * T::STRIDE + dz * TILE_X * ROWB + kk * 32;
                                const int bo = (k / 2) * RING_WTAP + kk * (WIDE ? 2 * RING_WCHUNK : 32);
                                mma_bf16(acc, a0 + (uint64_t)(ao >> 4), bd + (uint64_t)(bo >> 4), idesc, 1u);
                            }
                        }
                    };
                    if (lo < fresh) run(lo, min(hi, fresh - 1), true);
                    if (fresh <= hi) run(fresh, hi, true);
                    run(lo, hi, false);
                    mma_commit(&slot_free[s]);
                    // outputs that frame g completes
                    for (int f = lo; f <= hi; ++f)
                        if (f == g - 2 || g == g1) mma_commit(&acc_full[(jb + (uint32_t)(f - r.fa)) % RING_ACC]);
                }
                jb += (uint32_t)(r.fb - r.fa);
            }
            if (fail) s_fail = 1;
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = pixels x0 + 32 (w % 4) + lane (WIDE)
        // or depth row z0 + w % 4
        const int q = warp & 3;
        uint32_t j = 0;
        bool stop = false;
        for (int u = blockIdx.x; u < units && !stop; u += gridDim.x) {
            const RingUnit r = ring_unit<WIDE>(d, u);
            for (int f = r.fa; f < r.fb; ++f, ++j) {
                const uint32_t buf = j % RING_ACC;
                if (!warp_wait(&acc_full[buf], (j / RING_ACC) & 1u)) {
                    if (lane == 0) s_fail = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + buf * C, v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[buf]);
                const int64_t vox = (((int64_t)r.n * d.F + f) * d.Z + r.z0 + (WIDE ? 0 : q)) * d.X + r.x0 + (WIDE ? q * 32 : 0) + lane;
                epilogue_store<EPI>(v, s_bias, vox, out, mask);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(RING_TMEM) : "memory");
    }
    if (threadIdx.x == 0 && s_fail) atomicExch(status, (int)FQ_ERR_TIMEOUT);
}

// ------------------------------------------------------------ small kernels --
// Master FP32 weights [45][32 in][32 out] -> BF16 tap tiles for the forward
// pass (rows = out channel, 32 in channels each) and for the data gradient
// (kernel flipped in all three axes: tap 44 - t; rows = in channel).
// The chunked images hold the same tiles as [tap][K chunk of 8][row][8]
// (16-byte core-matrix rows) for the WIDE tile.
__global__ void pack_weights_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wf,
                                    __nv_bfloat16 *__restrict__ wb, __nv_bfloat16 *__restrict__ wfc,
                                    __nv_bfloat16 *__restrict__ wbc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NTAP * C * C) return;
    const int t = i / (C * C), ci = (i / C) % C, co = i % C;
    const __nv_bfloat16 v = __float2bfloat16_rn(w[i]);
    const int tb = NTAP - 1 - t;
    wf[((size_t)t * C + co) * C + ci] = v;
    wb[((size_t)tb * C + ci) * C + co] = v;
    wfc[(((size_t)t * 4 + ci / 8) * C + co) * 8 + ci % 8] = v;
    wbc[(((size_t)tb * 4 + co / 8) * C + ci) * 8 + co % 8] = v;
}

// Packing of a Casorati ensemble [P][F][2] (pixel p = x + X z) for the
// network.  Pass 1 (one thread per pixel): the pixel's temporal mean (when
// removing it) and its sum of squared deviations, accumulated per CTA.
__global__ void casorati_stats_kernel(const float *__restrict__ iq, int F, int64_t P, int remove_mean,
                                      float2 *__restrict__ mean, double *__restrict__ part)
{
    __shared__ double red[8];
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double ss = 0.0;
    if (p < P) {
        const float2 *s = reinterpret_cast<const float2 *>(iq) + p * F;
        float mr = 0.0f, mi = 0.0f;
        if (remove_mean) {
            for (int f = 0; f < F; ++f) {
                mr += s[f].x;
                mi += s[f].y;
            }
            mr /= (float)F;
            mi /= (float)F;
        }
        mean[p] = make_float2(mr, mi);
        for (int f = 0; f < F; ++f) {
            const float a = s[f].x - mr, b = s[f].y - mi;
            ss += (double)a * a + (double)b * b;
        }
    }
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// scale = 1 / RMS of the deviations over the whole ensemble (real and
// imaginary parts counted separately), into *scale.
__global__ void casorati_scale_kernel(const double *__restrict__ part, int n, int64_t count, float *__restrict__ scale)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) s += part[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *scale = s > 0.0 ? (float)(1.0 / sqrt(s / (double)count)) : 1.0f;
}

// Pass 2: (s - mean) * scale * gain into the BF16 volume [F][Z][X][32]
// (channels 0, 1; the rest 0) and / or the FP32 target [F][Z][X][2].  Four
// threads per pixel, each 16 of a voxel's 64 bytes (a warp's store is 512
// contiguous bytes), kPackFrames frames a CTA: 145 us for 65536 pixels x 200
// frames, 6.5 TB/s; one thread per pixel over all frames took 285 us.
constexpr int kPackFrames = 32;
__global__ void casorati_pack_kernel(const float *__restrict__ iq, int F, int64_t P, const float2 *__restrict__ mean,
                                     const float *__restrict__ scale, float gain, __nv_bfloat16 *__restrict__ vol,
                                     float *__restrict__ tgt)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, p = t >> 2;
    const int k = (int)(t & 3);
    if (p >= P) return;
    const float g = *scale * gain;
    const float2 m = mean[p];
    const float2 *s = reinterpret_cast<const float2 *>(iq) + p * F;
    for (int64_t f0 = (int64_t)blockIdx.y * kPackFrames; f0 < F; f0 += (int64_t)gridDim.y * kPackFrames) {
        const int f1 = (int)(f0 + kPackFrames < F ? f0 + kPackFrames : F);
#pragma unroll 8
        for (int f = (int)f0; f < f1; ++f) {
            const float2 v = s[f];
            const float a = (v.x - m.x) * g, b = (v.y - m.y) * g;
            const int64_t i = (int64_t)f * P + p;
            if (vol) {
                uint4 out = make_uint4(0, 0, 0, 0);
                if (k == 0) *reinterpret_cast<__nv_bfloat162 *>(&out) = __floats2bfloat162_rn(a, b);
                reinterpret_cast<uint4 *>(vol + i * C)[k] = out;
            }
            if (tgt && k == 0) reinterpret_cast<float2 *>(tgt)[i] = make_float2(a, b);
        }
    }
}

// MSE loss of channels 0, 1 of y [V][32] against t [V][2]: gradient
// 2 (y - t) / (2 V) into dy [V][32] BF16 (other channels 0) and per-block
// partial sums of the squared error.
__global__ void mse_grad_kernel(const float *__restrict__ y, const float *__restrict__ t, int64_t V,
                                __nv_bfloat16 *__restrict__ dy, double *__restrict__ part)
{
    __shared__ double red[8];
    const float inv = 1.0f / (float)(2 * V);
    double acc = 0.0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
        const float e0 = y[v * C] - t[2 * v], e1 = y[v * C + 1] - t[2 * v + 1];
        acc += (double)e0 * e0 + (double)e1 * e1;
        uint4 out[4] = {};
        __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(out);
        h[0] = __floats2bfloat162_rn(2.0f * e0 * inv, 2.0f * e1 * inv);
        uint4 *o = reinterpret_cast<uint4 *>(dy + v * C);
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = out[k];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        part[blockIdx.x] = s;
    }
}

__global__ void sum_parts_kernel(const double *__restrict__ part, int n, int64_t count, float *__restrict__ loss)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) s += part[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *loss = (float)(s / (double)count);
}

// Weight gradient: dW[t][ci][co] = sum_v x[v + d_t][ci] dy[v][co], a
// contraction over voxels with 45 x 32 x 32 results, on the warp-level
// tensor cores (mma.sync m16n8k16, BF16 operands, FP32 accumulators).  A
// CTA keeps the whole result in registers: warp (dt, dz) holds the three
// taps dx = -1, 0, 1 (96 accumulators per lane) and walks the CTA's
// contiguous range of tiles (4 depth rows x 32 pixels of a frame) column by
// column, frame by frame.  Frames of x with their halo (6 rows x 34 pixels)
// and tiles of dy arrive by TMA (64-byte swizzle, zero fill outside the
// volume) in rings of 7 and 8 slots, so each is loaded once per CTA while
// up to five frames' warps use it; operands come out of shared memory with
// transposing ldmatrix (both are voxel-major, the K direction), conflict
// free under the swizzle.  A CTA writes one partial (kWgVals floats); the
// partials are summed in order by wgrad_reduce_kernel.
//
// The tensor core's accumulation truncates, a bias that grows with the steps
// of a running sum (1.2e-6 of the gradients at 1.7k voxels a CTA, 1.5e-4 at
// 86k), so an accumulator runs over the 32 voxels of a row only, from zero, and
// is added to the running sum in FP32: 5.4e-8 and 7.9e-8, for 0.03 ms of a
// training step (every 16 voxels: 5.6e-8, 0.07 ms).
//
// Why: one thread per four results on the CUDA cores with a shared-memory
// step of 64 voxels re-read x and dy for each of the 45 taps (3.3 ms a
// layer), and its reduction summed db in one CTA (1.5 ms).  Four layers of a
// training step of 4 volumes of 64 x 32 x 32 voxels: 19.1 -> 0.29 ms; bound by
// the mma.sync rate (24 per 16 voxels and warp) and the additions.  tcgen05
// would need 4 taps per M = 128 operand at unequal row offsets, which its
// descriptors cannot express.
constexpr int kHaloX = TILE_X + 2, kHaloZ = TILE_Z + 2;
constexpr int kWgWarps = 15;                    // (dt, dz)
constexpr int kWgThreads = 32 * (kWgWarps + 1);  // and the TMA warp
constexpr int kWgXSlots = 7, kWgDySlots = 8;
constexpr int kWgXBytes = kHaloX * kHaloZ * C * 2;           // 13056
constexpr int kWgXSlotB = (kWgXBytes + 1023) & ~1023;
constexpr int kWgDyB = TILE_M * C * 2;                        // 8192
constexpr int kWgSmem = kWgXSlots * kWgXSlotB + kWgDySlots * kWgDyB + 1024;
constexpr int kWgVals = NTAP * C * C + C;                     // dW, then db
constexpr int kWgMaxParts = 152;                              // one CTA per SM

__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// t += A B
__device__ __forceinline__ void mma16816(float (&t)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(t[0]), "+f"(t[1]), "+f"(t[2]), "+f"(t[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// t = A B
__device__ __forceinline__ void mma16816z(float (&t)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}

// byte offset of 16-byte chunk c of 64-byte row q under the 64-byte swizzle
__device__ __forceinline__ uint32_t sw64_off(int q, int c)
{
    return (uint32_t)(q * 64 + ((c ^ ((q >> 1) & 3)) << 4));
}

// NT: 8-channel blocks of dy that can be non-zero (1 for the last layer)
template <int NT>
__global__ void __launch_bounds__(kWgThreads, 1)
    wgrad_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap dy_map,
                 const ConvDims d, float *__restrict__ part, int *__restrict__ status)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char *xs = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *gs = xs + kWgXSlots * kWgXSlotB;
    __shared__ __align__(8) uint64_t x_full[kWgXSlots], x_free[kWgXSlots], g_full[kWgDySlots], g_free[kWgDySlots];
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWgXSlots; ++s) {
            mbar_init(&x_full[s], 1);
            mbar_init(&x_free[s], kWgWarps);
        }
        for (int s = 0; s < kWgDySlots; ++s) {
            mbar_init(&g_full[s], 1);
            mbar_init(&g_free[s], kWgWarps);
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int t0 = range_begin(d.walk_tiles), t1 = range_end(d.walk_tiles);

    if (warp == kWgWarps) {
        if (lane == 0) {
            int jx = 0, jg = 0;
            bool ok = true;
            for (int t = t0; t < t1 && ok;) {
                const int col = t / d.F, fa = t - col * d.F, fb = min(d.F, fa + t1 - t);
                const Column cl = column_at(d, col);
                for (int g = fa - 2; g <= fb + 1; ++g, ++jx) {
                    const int s = jx % kWgXSlots, use = jx / kWgXSlots;
                    if (use > 0 && !mbar_wait(&x_free[s], (uint32_t)(use - 1) & 1u)) { ok = false; break; }
                    mbar_expect_tx(&x_full[s], kWgXBytes);
                    tma_load_5d(xs + s * kWgXSlotB, &x_map, &x_full[s], 0, cl.x0 - 1, cl.z0 - 1, g, cl.n);
                    const int f = g + 2;  // the tile of dy first used with this frame
                    if (f >= fb) continue;
                    const int sg = jg % kWgDySlots, useg = jg / kWgDySlots;
                    ++jg;
                    if (useg > 0 && !mbar_wait(&g_free[sg], (uint32_t)(useg - 1) & 1u)) { ok = false; ++jx; --jg; break; }
                    mbar_expect_tx(&g_full[sg], kWgDyB);
                    tma_load_5d(gs + sg * kWgDyB, &dy_map, &g_full[sg], 0, cl.x0, cl.z0, f, cl.n);
                }
                t += fb - fa;
            }
            if (!ok) s_fail = 1;
            // let issued copies land before the CTA can exit, whoever gave up
            for (int k = 1; k <= kWgXSlots && jx - k >= 0; ++k)
                mbar_wait(&x_full[(jx - k) % kWgXSlots], (uint32_t)((jx - k) / kWgXSlots) & 1u);
            for (int k = 1; k <= kWgDySlots && jg - k >= 0; ++k)
                mbar_wait(&g_full[(jg - k) % kWgDySlots], (uint32_t)((jg - k) / kWgDySlots) & 1u);
        }
    } else {
        const int dti = warp / 3, dzi = warp % 3;  // dt + 2, dz + 1
        float acc[3][2][NT][4];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[a][m][n][k] = 0.0f;
        float db[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) db[n] = 0.0f;
        // ldmatrix rows of this lane: A (x): row = lane % 8 + 8 (lane / 16), chunk = (lane / 8) % 2;
        // B (dy): row = lane % 8 + 8 ((lane / 8) % 2), chunk = lane / 16
        const int a_row = (lane & 7) + ((lane >> 4) << 3), a_ch = (lane >> 3) & 1;
        const int b_row = (lane & 7) + (((lane >> 3) & 1) << 3), b_ch = lane >> 4;
        int jx = 0, jg0 = 0;
        bool ok = true;
        for (int t = t0; t < t1 && ok;) {
            const int col = t / d.F, fa = t - col * d.F, nf = min(d.F - fa, t1 - t);
            for (int j = 0; j < nf + 4; ++j, ++jx) {
                const int s = jx % kWgXSlots;
                if (!warp_wait(&x_full[s], (uint32_t)(jx / kWgXSlots) & 1u)) { ok = false; break; }
                const int i = j - dti;  // tile of dy: frame fa + i reads x frame fa + i + dt
                if (i >= 0 && i < nf) {
                    const int jg = jg0 + i, sg = jg % kWgDySlots;
                    if (!warp_wait(&g_full[sg], (uint32_t)(jg / kWgDySlots) & 1u)) { ok = false; break; }
                    const uint32_t xb = smem_u32(xs + s * kWgXSlotB), gb = smem_u32(gs + sg * kWgDyB);
#pragma unroll 1
                    for (int ks = 0; ks < TILE_M / 16; ks += 2) {  // the 32 pixels of a row
                        uint32_t b[2][(NT + 1) / 2][4];
#pragma unroll
                        for (int q = 0; q < 2; ++q)
#pragma unroll
                            for (int n = 0; n < (NT + 1) / 2; ++n)
                                ldsm4t(gb + sw64_off(16 * (ks + q) + b_row, 2 * n + b_ch), b[q][n]);
                        const int q0 = ((ks >> 1) + dzi) * kHaloX + a_row;
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                            for (int m = 0; m < 2; ++m) {
                                uint32_t a0[4], a1[4];
                                ldsm4t(xb + sw64_off(q0 + dx, 2 * m + a_ch), a0);
                                ldsm4t(xb + sw64_off(q0 + 16 + dx, 2 * m + a_ch), a1);
#pragma unroll
                                for (int n = 0; n < NT; ++n) {
                                    float t[4];
                                    mma16816z(t, a0, b[0][n / 2][2 * (n & 1)], b[0][n / 2][2 * (n & 1) + 1]);
                                    mma16816(t, a1, b[1][n / 2][2 * (n & 1)], b[1][n / 2][2 * (n & 1) + 1]);
#pragma unroll
                                    for (int i = 0; i < 4; ++i) acc[dx][m][n][i] += t[i];
                                }
                            }
                        }
                        if (warp == 0) {
#pragma unroll
                            for (int n = 0; n < NT; ++n)
#pragma unroll
                                for (int q = 0; q < 2; ++q) {
                                    const float2 u = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b[q][n / 2][2 * (n & 1)]));
                                    const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&b[q][n / 2][2 * (n & 1) + 1]));
                                    db[n] += (u.x + u.y) + (v.x + v.y);
                                }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&g_free[sg]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&x_free[s]);
            }
            jg0 += nf;
            t += nf;
        }
        if (!ok && lane == 0) s_fail = 1;
        // accumulator element (row, col): rows ci = 16 m + lane / 4 (+ 8), cols co = 8 n + 2 (lane % 4) (+ 1)
        float *o = part + (size_t)blockIdx.x * kWgVals;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
            float *ot = o + (size_t)((dti * 3 + dzi) * 3 + dx) * C * C;
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    const int ci = 16 * m + (lane >> 2), co = 8 * n + 2 * (lane & 3);
                    float2 lo = make_float2(0.0f, 0.0f), hi = lo;
                    if (n < NT) {
                        lo = make_float2(acc[dx][m][n < NT ? n : 0][0], acc[dx][m][n < NT ? n : 0][1]);
                        hi = make_float2(acc[dx][m][n < NT ? n : 0][2], acc[dx][m][n < NT ? n : 0][3]);
                    }
                    *reinterpret_cast<float2 *>(ot + ci * C + co) = lo;
                    *reinterpret_cast<float2 *>(ot + (ci + 8) * C + co) = hi;
                }
        }
        if (warp == 0) {  // b0 holds (k = 2 (lane % 4) .. + 1, n = lane / 4): sum the four lanes of a column
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                float v = n < NT ? db[n < NT ? n : 0] : 0.0f;
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                if ((lane & 3) == 0) o[NTAP * C * C + 8 * n + (lane >> 2)] = v;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_fail) atomicExch(status, (int)FQ_ERR_TIMEOUT);
}

// Sum the partials, in order, into dW [45][32][32] and db [32]: one warp
// per 32 values, the partials of a value dealt to 8 warps.
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float *__restrict__ part, int n_parts,
                                                           float *__restrict__ dw, float *__restrict__ db)
{
    __shared__ float red[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;  // kWgVals is a multiple of 32
    float s = 0.0f;
    for (int c = w; c < n_parts; c += 8) s += part[(size_t)c * kWgVals + i];
    red[w][lane] = s;
    __syncthreads();
    if (w) return;
    for (int k = 1; k < 8; ++k) s += red[k][lane];
    if (i < NTAP * C * C) dw[i] = s;
    else db[i - NTAP * C * C] = s;
}

// Adam on a flat FP32 parameter array.
__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    }
}

// PD of the network output y [F][Z][X][32] (channels 0, 1): mean over
// frames of |y|^2, divided by scale^2 (undoing the input normalisation).
__global__ void cnn_pd_kernel(const float *__restrict__ y, int F, int Z, int X, float inv_scale2, float *__restrict__ pd)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)Z * X) return;
    float s = 0.0f;
    for (int f = 0; f < F; ++f) {
        const float *q = y + ((int64_t)f * Z * X + p) * C;
        s += q[0] * q[0] + q[1] * q[1];
    }
    pd[p] = s / (float)F * inv_scale2;
}

// ------------------------------------------------------------------- host --
struct ParamLayout {   // offsets in floats inside the parameter block
    size_t w[4], b[4], m, v, n_train;  // master weights/biases, then Adam m and v over the same span
    size_t wf_bytes_off, wb_bytes_off;   // 64-byte-row tap tiles (narrow tile)
    size_t wfc_bytes_off, wbc_bytes_off; // 16-byte-chunk tap tiles (WIDE tile)
    size_t total_bytes;
};

ParamLayout param_layout()
{
    ParamLayout L;
    size_t o = 0;
    for (int l = 0; l < 4; ++l) { L.w[l] = o; o += (size_t)NTAP * C * C; }
    for (int l = 0; l < 4; ++l) { L.b[l] = o; o += C; }
    L.n_train = o;
    L.m = o; o += L.n_train;
    L.v = o; o += L.n_train;
    size_t bytes = (o * 4 + 255) & ~(size_t)255;
    L.wf_bytes_off = bytes; bytes += (size_t)4 * NTAP * C * C * 2;
    L.wb_bytes_off = bytes; bytes += (size_t)4 * NTAP * C * C * 2;
    L.wfc_bytes_off = bytes; bytes += (size_t)4 * NTAP * C * C * 2;
    L.wbc_bytes_off = bytes; bytes += (size_t)4 * NTAP * C * C * 2;
    L.total_bytes = bytes;
    return L;
}

struct ActLayout {
    size_t act[3], out, dy[2], part, loss_part, total;
    int wg_parts;
};

int64_t tile_count(int N, int F, int Z, int X)
{
    return (int64_t)N * F * ((Z + TILE_Z - 1) / TILE_Z) * ((X + TILE_X - 1) / TILE_X);
}

ActLayout act_layout(int N, int F, int Z, int X)
{
    ActLayout L;
    const size_t V = (size_t)N * F * Z * X;
    size_t o = 0;
    for (int i = 0; i < 3; ++i) { L.act[i] = o; o += (V * C * 2 + 255) & ~(size_t)255; }
    L.out = o; o += (V * C * 4 + 255) & ~(size_t)255;
    for (int i = 0; i < 2; ++i) { L.dy[i] = o; o += (V * C * 2 + 255) & ~(size_t)255; }
    const int64_t tiles = tile_count(N, F, Z, X);
    L.wg_parts = tiles < kWgMaxParts ? (int)tiles : kWgMaxParts;
    L.part = o; o += ((size_t)L.wg_parts * kWgVals * 4 + 255) & ~(size_t)255;
    L.loss_part = o; o += 1024 * 8;
    L.total = o;
    return L;
}

fq_status encode_act_map(CUtensorMap *map, const void *p, int N, int F, int Z, int X, bool ring)
{
    auto enc = (PFN_cuTensorMapEncodeTiled_v12000)fqi::tensor_map_encoder_ptr();
    FQ_REQUIRE(enc, FQ_ERR_CUDA, "cnn: cuTensorMapEncodeTiled unavailable");
    std::memset(map, 0, sizeof *map);
    cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)X, (cuuint64_t)Z, (cuuint64_t)F, (cuuint64_t)N};
    cuuint64_t strides[4] = {(cuuint64_t)C * 2, (cuuint64_t)X * C * 2, (cuuint64_t)Z * X * C * 2,
                             (cuuint64_t)F * Z * X * C * 2};
    // 32 channels x 32 pixels x 6 rows, 64-byte swizzle; WIDE: 8 channels x 130
    // pixels x 3 rows, no swizzle
    cuuint32_t box_tap[5] = {(cuuint32_t)C, (cuuint32_t)TILE_X, (cuuint32_t)TILE_Z + 2, 1, 1};
    cuuint32_t box_ring[5] = {8, (cuuint32_t)Tile<true>::W, 3, 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(p), dims, strides,
                     ring ? box_ring : box_tap, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     ring ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    FQ_REQUIRE(r == CUDA_SUCCESS, FQ_ERR_CUDA, "cnn: activation tensor map (%d)", (int)r);
    return FQ_OK;
}

// 64-byte swizzled boxes of all 32 channels: `halo` 34 pixels x 6 rows (x of
// the weight gradient), else 32 x 4 (dy).
fq_status encode_wg_map(CUtensorMap *map, const void *p, const ConvDims &d, bool halo)
{
    auto enc = (PFN_cuTensorMapEncodeTiled_v12000)fqi::tensor_map_encoder_ptr();
    FQ_REQUIRE(enc, FQ_ERR_CUDA, "cnn: cuTensorMapEncodeTiled unavailable");
    std::memset(map, 0, sizeof *map);
    cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)d.X, (cuuint64_t)d.Z, (cuuint64_t)d.F, (cuuint64_t)d.N};
    cuuint64_t strides[4] = {(cuuint64_t)C * 2, (cuuint64_t)d.X * C * 2, (cuuint64_t)d.Z * d.X * C * 2,
                             (cuuint64_t)d.F * d.Z * d.X * C * 2};
    cuuint32_t box[5] = {(cuuint32_t)C, (cuuint32_t)(halo ? kHaloX : TILE_X), (cuuint32_t)(halo ? kHaloZ : TILE_Z), 1,
                         1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(p), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    FQ_REQUIRE(r == CUDA_SUCCESS, FQ_ERR_CUDA, "cnn: activation tensor map (%d)", (int)r);
    return FQ_OK;
}

fq_status encode_w_map(CUtensorMap *map, const void *p)
{
    auto enc = (PFN_cuTensorMapEncodeTiled_v12000)fqi::tensor_map_encoder_ptr();
    FQ_REQUIRE(enc, FQ_ERR_CUDA, "cnn: cuTensorMapEncodeTiled unavailable");
    std::memset(map, 0, sizeof *map);
    cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)NTAP * C};
    cuuint64_t strides[1] = {(cuuint64_t)C * 2};
    cuuint32_t box[2] = {(cuuint32_t)C, (cuuint32_t)C};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(p), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    FQ_REQUIRE(r == CUDA_SUCCESS, FQ_ERR_CUDA, "cnn: weight tensor map (%d)", (int)r);
    return FQ_OK;
}

int num_sms()
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms < 1) sms = 1;
    }
    return sms;
}

// Frames per work unit: a run of L output frames walks L + 4 input frames (the
// first and last with part of the outputs), so few long runs cost least and
// enough runs for every SM the least time.
int conv_run(int columns, int F, int sms)
{
    int best = F;
    double cost = 1e300;
    for (int runs = 1; runs <= F; ++runs) {
        const int len = (F + runs - 1) / runs, units = columns * ((F + len - 1) / len);
        const double c = (double)((units + sms - 1) / sms) * (len + 3.0);
        if (c < cost) { cost = c; best = len; }
    }
    return best;
}

// One convolution of layer `layer` (forward or data-gradient kernel).
template <bool WIDE>
fq_status launch_conv(int epi, const CUtensorMap &in_map, const CUtensorMap &w_map, const __nv_bfloat16 *wc, ConvDims d,
                      const float *bias, void *out, const __nv_bfloat16 *mask, int *status, cudaStream_t st)
{
    using T = Tile<WIDE>;
    const int columns = d.N * (d.Z / T::Z) * (d.X / T::X);
    d.run = conv_run(columns, d.F, num_sms());
    const int units = columns * ((d.F + d.run - 1) / d.run);
    const int grid = units < num_sms() ? units : num_sms();
    auto launch = [&](auto kern) -> fq_status {
        fq_status r = fqi::cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEM),
                                      "cnn: smem attribute");
        if (r) return r;
        kern<<<grid, CONV_THREADS, T::SMEM, st>>>(in_map, w_map, wc, d, units, bias, out, mask, status);
        return fqi::launch_check("cnn: conv");
    };
    if (epi == EPI_RELU_BF16) return launch(conv_kernel<EPI_RELU_BF16, WIDE>);
    if (epi == EPI_LINEAR_F32) return launch(conv_kernel<EPI_LINEAR_F32, WIDE>);
    return launch(conv_kernel<EPI_MASK_BF16, WIDE>);
}

fq_status conv(int epi, const void *in, const void *params, int layer, bool backward, const float *bias, void *out,
               const __nv_bfloat16 *mask, const ConvDims &d, int *status, cudaStream_t st)
{
    const ParamLayout L = param_layout();
    const char *pb = (const char *)params;
    const size_t lo = (size_t)layer * NTAP * C * C * 2;
    const bool wide = d.Z % TILE_Z != 0;  // then X is a multiple of 128
    CUtensorMap in_map, w_map;
    fq_status s = encode_act_map(&in_map, in, d.N, d.F, d.Z, d.X, wide);
    if (!s) s = encode_w_map(&w_map, pb + (backward ? L.wb_bytes_off : L.wf_bytes_off) + lo);
    if (s) return s;
    const __nv_bfloat16 *wc = (const __nv_bfloat16 *)(pb + (backward ? L.wbc_bytes_off : L.wfc_bytes_off) + lo);
    return wide ? launch_conv<true>(epi, in_map, w_map, wc, d, bias, out, mask, status, st)
                : launch_conv<false>(epi, in_map, w_map, wc, d, bias, out, mask, status, st);
}

template <int NT>
fq_status launch_wgrad(const void *x, const void *dy, const ConvDims &d, int n_parts, float *part, float *dw, float *db,
                       int *status, cudaStream_t st)
{
    CUtensorMap x_map, dy_map;
    fq_status r = encode_wg_map(&x_map, x, d, true);
    if (r) return r;
    r = encode_wg_map(&dy_map, dy, d, false);
    if (r) return r;
    auto kern = wgrad_kernel<NT>;
    r = fqi::cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem),
                        "cnn: smem attribute");
    if (r) return r;
    kern<<<n_parts, kWgThreads, kWgSmem, st>>>(x_map, dy_map, d, part, status);
    wgrad_reduce_kernel<<<kWgVals / 32, 256, 0, st>>>(part, n_parts, dw, db);
    return fqi::launch_check("fq_cnn_backward: weight gradient");
}

fq_status check_dims(int N, int F, int Z, int X, const char *who)
{
    FQ_REQUIRE(N >= 1 && F >= 1 && Z >= 1 && X >= TILE_X, FQ_ERR_SHAPE, "%s: bad volume size", who);
    FQ_REQUIRE(X % Tile<true>::X == 0 || (Z % TILE_Z == 0 && X % TILE_X == 0), FQ_ERR_SHAPE,
               "%s: X must be a multiple of 128, or of 32 with Z a multiple of 4 (got Z %d, X %d)", who, Z, X);
    FQ_REQUIRE(tile_count(N, F, Z, X) < ((int64_t)1 << 31), FQ_ERR_SHAPE, "%s: too many tiles",
               who);
    return FQ_OK;
}

ConvDims make_dims(int N, int F, int Z, int X)
{
    ConvDims d;
    d.N = N; d.F = F; d.Z = Z; d.X = X;
    d.run = F;
    d.zb = (Z + TILE_Z - 1) / TILE_Z;
    d.xb = X / TILE_X;
    d.walk_tiles = (int)tile_count(N, F, Z, X);
    return d;
}

}  // namespace

extern "C" {

size_t fq_cnn_param_bytes(void) { return param_layout().total_bytes; }

size_t fq_cnn_prep_bytes(int32_t Z, int32_t X)
{
    const int64_t P = (int64_t)Z * X;
    const int64_t blocks = (P + 255) / 256;
    return (((size_t)P * 8 + 255) & ~(size_t)255) + (size_t)blocks * 8 + 256;
}

size_t fq_cnn_act_bytes(int32_t n_vol, int32_t F, int32_t Z, int32_t X)
{
    if (n_vol < 1 || F < 1 || Z < 1 || X < 1) return 0;
    return act_layout(n_vol, F, Z, X).total;
}

fq_status fq_cnn_pack(void *params, void *stream)
{
    FQ_REQUIRE(params && fqi::aligned(params, 256), FQ_ERR_INVALID_ARG, "fq_cnn_pack: null or unaligned params");
    const ParamLayout L = param_layout();
    cudaStream_t st = (cudaStream_t)stream;
    float *pf = (float *)params;
    char *pb = (char *)params;
    for (int l = 0; l < 4; ++l) {
        __nv_bfloat16 *wf = (__nv_bfloat16 *)(pb + L.wf_bytes_off) + (size_t)l * NTAP * C * C;
        __nv_bfloat16 *wb = (__nv_bfloat16 *)(pb + L.wb_bytes_off) + (size_t)l * NTAP * C * C;
        __nv_bfloat16 *wfc = (__nv_bfloat16 *)(pb + L.wfc_bytes_off) + (size_t)l * NTAP * C * C;
        __nv_bfloat16 *wbc = (__nv_bfloat16 *)(pb + L.wbc_bytes_off) + (size_t)l * NTAP * C * C;
        pack_weights_kernel<<<(NTAP * C * C + 255) / 256, 256, 0, st>>>(pf + L.w[l], wf, wb, wfc, wbc);
    }
    return fqi::launch_check("fq_cnn_pack");
}

fq_status fq_cnn_from_casorati(const float *iq, int32_t F, int32_t Z, int32_t X, int32_t remove_mean,
                               const float *scale_in, float *scale_out, float gain, void *vol, float *target,
                               void *workspace, size_t workspace_bytes, void *stream)
{
    FQ_REQUIRE(iq && (vol || target) && F >= 1 && Z >= 1 && X >= 1 && workspace, FQ_ERR_INVALID_ARG,
               "fq_cnn_from_casorati: bad arguments");
    FQ_REQUIRE(scale_in || scale_out, FQ_ERR_INVALID_ARG, "fq_cnn_from_casorati: needs scale_in or scale_out");
    FQ_REQUIRE(fqi::aligned(iq, 8) && fqi::aligned(vol, 16) && fqi::aligned(target, 8) &&
                   fqi::aligned(workspace, 256),
               FQ_ERR_ALIGN, "fq_cnn_from_casorati: alignment");
    const int64_t P = (int64_t)Z * X;
    const int blocks = (int)((P + 255) / 256);
    const size_t need = fq_cnn_prep_bytes(Z, X);
    FQ_REQUIRE(workspace_bytes >= need, FQ_ERR_WORKSPACE, "fq_cnn_from_casorati: workspace needs %zu bytes", need);
    float2 *mean = (float2 *)workspace;
    double *part = (double *)((char *)workspace + (((size_t)P * 8 + 255) & ~(size_t)255));
    cudaStream_t st = (cudaStream_t)stream;
    casorati_stats_kernel<<<blocks, 256, 0, st>>>(iq, F, P, remove_mean, mean, part);
    const float *scale = scale_in;
    if (!scale_in) {
        casorati_scale_kernel<<<1, 32, 0, st>>>(part, blocks, 2 * P * F, scale_out);
        scale = scale_out;
    }
    const unsigned runs = (unsigned)F / kPackFrames + (F % kPackFrames != 0);
    const dim3 pack((unsigned)((4 * P + 255) / 256), runs < 65535 ? runs : 65535);
    casorati_pack_kernel<<<pack, 256, 0, st>>>(iq, F, P, mean, scale, gain, (__nv_bfloat16 *)vol, target);
    return fqi::launch_check("fq_cnn_from_casorati");
}

fq_status fq_cnn_conv(int32_t mode, const void *in, const void *params, int32_t layer, int32_t backward,
                      void *out, const void *mask, int32_t n_vol, int32_t F, int32_t Z, int32_t X, int32_t *status,
                      void *stream)
{
    fq_status s = check_dims(n_vol, F, Z, X, "fq_cnn_conv");
    if (s) return s;
    FQ_REQUIRE(in && params && out && status && layer >= 0 && layer < 4 && mode >= 0 && mode <= 2 &&
                   (mode != EPI_MASK_BF16 || mask),
               FQ_ERR_INVALID_ARG, "fq_cnn_conv: bad arguments");
    FQ_REQUIRE(fqi::aligned(in, 16) && fqi::aligned(out, 16) && fqi::aligned(mask, 16) && fqi::aligned(params, 256),
               FQ_ERR_ALIGN, "fq_cnn_conv: alignment");
    const ParamLayout L = param_layout();
    const float *bias = backward ? nullptr : (const float *)params + L.b[layer];
    return conv(mode, in, params, layer, backward != 0, bias, out, (const __nv_bfloat16 *)mask,
                make_dims(n_vol, F, Z, X), (int *)status, (cudaStream_t)stream);
}

fq_status fq_cnn_forward(const void *params, const void *vol, int32_t n_vol, int32_t F, int32_t Z, int32_t X,
                         void *acts, size_t act_bytes, int32_t *status, void *stream)
{
    fq_status s = check_dims(n_vol, F, Z, X, "fq_cnn_forward");
    if (s) return s;
    const ActLayout A = act_layout(n_vol, F, Z, X);
    FQ_REQUIRE(params && vol && acts && status, FQ_ERR_INVALID_ARG, "fq_cnn_forward: null argument");
    FQ_REQUIRE(act_bytes >= A.total, FQ_ERR_WORKSPACE, "fq_cnn_forward: activations need %zu bytes", A.total);
    FQ_REQUIRE(fqi::aligned(acts, 256) && fqi::aligned(vol, 16) && fqi::aligned(params, 256), FQ_ERR_ALIGN,
               "fq_cnn_forward: alignment");
    const ParamLayout L = param_layout();
    char *ab = (char *)acts;
    const ConvDims d = make_dims(n_vol, F, Z, X);
    cudaStream_t st = (cudaStream_t)stream;
    const void *in = vol;
    for (int l = 0; l < 4; ++l) {
        const float *bias = (const float *)params + L.b[l];
        void *out = l < 3 ? (void *)(ab + A.act[l]) : (void *)(ab + A.out);
        s = conv(l < 3 ? EPI_RELU_BF16 : EPI_LINEAR_F32, in, params, l, false, bias, out, nullptr, d, (int *)status,
                 st);
        if (s) return s;
        in = out;
    }
    return FQ_OK;
}

fq_status fq_cnn_backward(const void *params, const void *vol, const float *target, int32_t n_vol, int32_t F,
                          int32_t Z, int32_t X, void *acts, size_t act_bytes, float *grads, float *loss,
                          int32_t *status, void *stream)
{
    fq_status s = check_dims(n_vol, F, Z, X, "fq_cnn_backward");
    if (s) return s;
    const ActLayout A = act_layout(n_vol, F, Z, X);
    FQ_REQUIRE(params && vol && target && acts && grads && loss && status, FQ_ERR_INVALID_ARG,
               "fq_cnn_backward: null argument");
    FQ_REQUIRE(act_bytes >= A.total, FQ_ERR_WORKSPACE, "fq_cnn_backward: activations need %zu bytes", A.total);
    const ParamLayout L = param_layout();
    char *ab = (char *)acts;
    const ConvDims d = make_dims(n_vol, F, Z, X);
    const int64_t V = (int64_t)n_vol * F * Z * X;
    cudaStream_t st = (cudaStream_t)stream;
    const __nv_bfloat16 *act_in[4] = {(const __nv_bfloat16 *)vol, (const __nv_bfloat16 *)(ab + A.act[0]),
                                      (const __nv_bfloat16 *)(ab + A.act[1]), (const __nv_bfloat16 *)(ab + A.act[2])};
    __nv_bfloat16 *dy[2] = {(__nv_bfloat16 *)(ab + A.dy[0]), (__nv_bfloat16 *)(ab + A.dy[1])};
    double *lp = (double *)(ab + A.loss_part);
    int lb = (int)((V + 255) / 256);
    if (lb > 1024) lb = 1024;
    mse_grad_kernel<<<lb, 256, 0, st>>>((const float *)(ab + A.out), target, V, dy[0], lp);
    sum_parts_kernel<<<1, 32, 0, st>>>(lp, lb, 2 * V, loss);
    s = fqi::launch_check("fq_cnn_backward: loss");
    if (s) return s;
    int cur = 0;
    for (int l = 3; l >= 0; --l) {
        // weight and bias gradients of layer l from its input and output gradient
        float *part = (float *)(ab + A.part);
        const __nv_bfloat16 *x = act_in[l];
        if (!fqi::aligned(x, 16)) {  // the caller's volume, whose copy can use the other gradient buffer now
            s = fqi::cuda_check(cudaMemcpyAsync(dy[cur ^ 1], x, (size_t)V * C * 2, cudaMemcpyDeviceToDevice, st),
                                "fq_cnn_backward: volume");
            if (s) return s;
            x = dy[cur ^ 1];
        }
        if (l == 3) s = launch_wgrad<1>(x, dy[cur], d, A.wg_parts, part, grads + L.w[l], grads + L.b[l], status, st);
        else s = launch_wgrad<4>(x, dy[cur], d, A.wg_parts, part, grads + L.w[l], grads + L.b[l], status, st);
        if (s) return s;
        if (l == 0) break;
        // data gradient through layer l, masked by the ReLU of layer l - 1
        s = conv(EPI_MASK_BF16, dy[cur], params, l, true, nullptr, dy[cur ^ 1], act_in[l], d, (int *)status, st);
        if (s) return s;
        cur ^= 1;
    }
    return FQ_OK;
}

fq_status fq_cnn_adam(void *params, const float *grads, float lr, int32_t step, void *stream)
{
    FQ_REQUIRE(params && grads && step >= 1 && lr > 0.0f, FQ_ERR_INVALID_ARG, "fq_cnn_adam: bad arguments");
    const ParamLayout L = param_layout();
    float *pf = (float *)params;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, step)));
    cudaStream_t st = (cudaStream_t)stream;
    adam_kernel<<<152 * 4, 256, 0, st>>>(pf, grads, pf + L.m, pf + L.v, (int64_t)L.n_train, lr, b1, b2, eps, c1, c2);
    fq_status s = fqi::launch_check("fq_cnn_adam");
    if (s) return s;
    return fq_cnn_pack(params, stream);
}

fq_status fq_cnn_power_doppler(const float *out, int32_t F, int32_t Z, int32_t X, float scale, float *pd,
                               void *stream)
{
    FQ_REQUIRE(out && pd && F >= 1 && Z >= 1 && X >= 1 && scale > 0.0f, FQ_ERR_INVALID_ARG,
               "fq_cnn_power_doppler: bad arguments");
    const int64_t P = (int64_t)Z * X;
    cnn_pd_kernel<<<(unsigned)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(out, F, Z, X,
                                                                                 1.0f / (scale * scale), pd);
    return fqi::launch_check("fq_cnn_power_doppler");
}

size_t fq_cnn_act_offset(int32_t which, int32_t n_vol, int32_t F, int32_t Z, int32_t X)
{
    if (n_vol < 1 || F < 1 || Z < 1 || X < 1 || which < 0 || which > 3) return (size_t)-1;
    const ActLayout A = act_layout(n_vol, F, Z, X);
    return which < 3 ? A.act[which] : A.out;
}

size_t fq_cnn_param_offset(int32_t what, int32_t layer)
{
    const ParamLayout L = param_layout();
    if (layer < 0 || layer > 3) return (size_t)-1;
    switch (what) {
    case 0: return L.w[layer] * 4;
    case 1: return L.b[layer] * 4;
    case 2: return L.m * 4;
    case 3: return L.v * 4;
    case 4: return L.n_train * 4;
    default: return (size_t)-1;
    }
}

}  // extern "C"

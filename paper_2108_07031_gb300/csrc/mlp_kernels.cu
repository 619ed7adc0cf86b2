// Warm-start surrogate: a coordinate/condition MLP trained and evaluated on
// the GPU with hand-written BF16 tensor-core kernels (FP32 accumulation).
//
// Network (include/lskum_mlp.h): 21 input features (zero-padded to 32) ->
// 5 hidden layers of 256 (tanh) -> 4 outputs (linear): six linear layers.
// Z_l = X_l W_l^T + b_l, X_{l+1} = tanh(Z_l). Weights are kept in FP32
// (Adam master copy) and in BF16 (W) for the GEMMs;
// activations are stored FP32 (for tanh') and BF16 (GEMM input).
//
// A prediction is one kernel (k_forward, or k_forward_mma where the handle's owner
// chooses mma.sync), loss and gradients four: k_forward, k_backward,
// k_weight_grads, k_reduce_grads. Every sum has a fixed order.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <algorithm>
#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "../../include/lskum_mlp.h"
#include "lskum_internal.h"

namespace mlpk {

constexpr int kLayers = LSKUM_MLP_LAYERS;
constexpr int kWidth = LSKUM_MLP_WIDTH;
constexpr int kIn = LSKUM_MLP_IN_PADDED;
constexpr int kOut = LSKUM_MLP_OUT;

__host__ __device__ inline int layer_in(int l) { return l == 0 ? kIn : kWidth; }
__host__ __device__ inline int layer_out(int l) { return l == kLayers - 1 ? kOut : kWidth; }

// Offsets of W_l and b_l in the flat parameter vector, and the BF16 copies.
struct LayerPtrs {
    int64_t w_off[kLayers];
    int64_t b_off[kLayers];
    __nv_bfloat16* W[kLayers];
};

// Raised when a bounded wait of a pass runs out: the passes' bits on the device,
// where the kernels that change the parameters read them, and 1 in pinned
// memory, where the host looks after it has synchronised.
enum Pass { kPassForward = 1, kPassBackward = 2, kPassWeightGrads = 4 };
struct ErrFlag {
    int* dev;
    int* host;
};
__device__ __forceinline__ void raise(const ErrFlag f, Pass pass) {
    atomicOr(f.dev, int(pass));
    *f.host = 1;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return uint32_t(__cvta_generic_to_shared(p));
}

// ------------------------------------------------- fused forward pass
// All six layers of a 128-row tile in one CTA on the fifth-generation tensor
// cores: the activations stay in shared memory as BF16 A operands, the weights
// stream from L2 through a ring of four 32 KB slots (64 of a layer's 256 k
// each, laid out beforehand as the operand image, one bulk copy a slot), and
// a layer's products accumulate in 256 columns of tensor memory, two layers'
// accumulators side by side. Sixteen warps turn the accumulators into the next
// layer's operand (bias, tanh, BF16), 64 columns at a time; the MMAs of those
// 64 k start as soon as they are written, so they run under the tanh of the
// next 64. One warp issues the MMAs, one the copies. The 4-wide output layer
// is FP32 FMAs on the same BF16 values, in the last epilogue.
//
// What bounds it: tanhf first, 163,840 a tile on an SM's FP32 pipes (~25
// instructions each: 15.5 of the 27 us that a wave of tiles takes); the MMAs of a
// tile are 69 MFLOP, 5.5 us at the SM's share of the BF16 rate, mostly under it;
// the rest is the chain through a tile, five layers that each begin with the last
// one's first 64 columns. A launch per layer wrote and re-read the
// activations (1.5 KB a row and layer) and filled the chip for 2 us of work:
// 16,384 samples 176 us a prediction, now 46 (27 in the kernel).
//
// Operand layout: the no-swizzle K-major canonical form of the matrix
// descriptors: core matrices of 8 rows x 16 bytes (8 BF16 along K) as 128
// contiguous bytes, neighbours along K 128 bytes apart (LBO), 8-row groups SBO
// bytes apart; one MMA (K 16) reads two core matrices along K.
constexpr int kFwdRows = 128;               // rows of a tile (MMA M)
constexpr int kFwdSlots = 4;                // weight ring
constexpr int kFwdSlotBytes = 256 * 64 * 2; // 256 outputs x 64 k
constexpr int kFwdIn0Bytes = 256 * 32 * 2;  // the first layer's one chunk
constexpr int kFwdChunks = 1 + 4 * 4;       // chunks of a tile: layer 0, then 4 each of 4 layers
constexpr int kFwdParts = 4;                // threads of a row, 16 of a chunk's 64 columns each
constexpr int kFwdCols = 64 / kFwdParts;
constexpr int kFwdEpi = kFwdRows * kFwdParts;  // epilogue threads
constexpr int kFwdMmaWarp = kFwdEpi / 32, kFwdCopyWarp = kFwdMmaWarp + 1;
constexpr int kFwdThreads = kFwdEpi + 64;   // and the MMA and the copy warp
constexpr int kFwdABytes = kFwdRows * 256 * 2;
constexpr int kFwdHidden = kLayers - 1;
// shared memory: A, ring, biases, output layer (weights as float4 a column), row partials, barriers
constexpr int kFwdOffRing = kFwdABytes;
constexpr int kFwdOffBias = kFwdOffRing + kFwdSlots * kFwdSlotBytes;
constexpr int kFwdOffW5 = kFwdOffBias + kFwdHidden * 256 * 4;
constexpr int kFwdOffPart = kFwdOffW5 + 256 * 16;
constexpr int kFwdOffBar = kFwdOffPart + (kFwdParts - 1) * kFwdRows * 16;
constexpr int kFwdSmem = kFwdOffBar + 128;
static_assert(kFwdSmem <= 227 * 1024, "one CTA's shared memory");

// Byte offset of W_l(n, k) in the operand images, one layer after the other.
__host__ __device__ inline int64_t packed_offset(int l, int n, int k) {
    if (l == 0) return (n / 8) * 512 + (k / 8) * 128 + (n % 8) * 16 + (k % 8) * 2;
    return kFwdIn0Bytes + int64_t(l - 1) * 4 * kFwdSlotBytes + (k / 64) * kFwdSlotBytes + (n / 8) * 1024 +
           (k % 64 / 8) * 128 + (n % 8) * 16 + (k % 8) * 2;
}

// The backward pass's images: W_l transposed (row k, contraction over n) of
// layers 4, 3, 2, 1 in the order it takes them.
__host__ __device__ inline int64_t packed_offset_t(int l, int n, int k) {
    return int64_t(kLayers - 2 - l) * 4 * kFwdSlotBytes + (n / 64) * kFwdSlotBytes + (k / 8) * 1024 +
           (n % 64 / 8) * 128 + (k % 8) * 16 + (n % 8) * 2;
}

// What the passes leave for one another, by tiles of 128 samples, with a tile's
// 128 rows next to one another so that a warp's 32 rows are one access: 16-byte
// granules of eight BF16 units (A_l, dZ_l) or of four FP32 ones (A_l for tanh'),
// [tile][granule][row]. A BF16 tile is at the same time the MMA operand of the
// weight gradients, whose contraction runs over the rows (core matrices of
// eight rows of a granule). Rows past n are written too (dZ = 0 there).
__host__ __device__ inline int64_t granule(int64_t tile, int per_tile, int g, int row) {
    return (tile * per_tile + g) * kFwdRows + row;
}

// SM100 shared-memory matrix descriptor: bits [0,14) start address >> 4,
// [16,30) leading-dimension byte offset >> 4, [32,46) stride-dimension byte
// offset >> 4, [46,48) descriptor version 1, [61,64) layout 0 (no swizzle).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return uint64_t((saddr >> 4) & 0x3FFFu) | (uint64_t((lbo >> 4) & 0x3FFFu) << 16) |
           (uint64_t((sbo >> 4) & 0x3FFFu) << 32) | (uint64_t(1) << 46);
}

// Instruction descriptor of kind::f16: D FP32 (bits [4,6) = 1), A and B BF16
// (bits [7,10) and [10,13) = 1), both K-major (bits 15, 16 = 0), N >> 3 at
// bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}

// Waits for phase `parity` of the mbarrier at shared address `bar`, polling a
// limited number of times (about half a second; the waits here take
// microseconds); false when the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (int i = 0; i < (1 << 22); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (i > 256) __nanosleep(128);
    }
    return false;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {  // arrives when the MMAs issued so far are done
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}

// A bulk copy of `bytes` from global to shared memory that counts on `bar`; and
// with the arrival that expects it.
__device__ __forceinline__ void bulk_copy_only(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
    bulk_copy_only(dst, src, bytes, bar);
}

// `steps` MMAs of K 16 of a 128-row A chunk (sbo 4096) and a 256-row B chunk into
// the accumulator columns at `acc`; the first overwrites unless `add`.
__device__ __forceinline__ void mma_chunk(uint32_t acc, uint32_t A, uint32_t B, uint32_t sbo, int steps, bool add) {
    constexpr uint32_t idesc = umma_idesc_bf16_f32(kFwdRows, 256);
    for (int ks = 0; ks < steps; ++ks)
        asm volatile(
            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc),
            "l"(umma_desc(A + uint32_t(ks) * 256, 128, 4096)), "l"(umma_desc(B + uint32_t(ks) * 256, 128, sbo)),
            "r"(idesc), "r"(int(add) + ks));
}

// tcgen05.ld of 32 (16) consecutive FP32 accumulator columns of this thread's
// tensor-memory lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
        "%28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// feat: n x 32 FP32; Wp: the operand images (packed_offset); p: the FP32
// parameters (biases; L's offsets), W5: the output layer's BF16 weights 4 x 256.
// out: n x 4. TRAIN: also Af[l], Ab[l] of the hidden layers, and Ab[0], in granules.
// `err` is raised if a wait ran out (the outputs are then incomplete).
struct FwdStore {
    float* Af[kLayers];
    __nv_bfloat16* Ab[kLayers];
};

template <bool TRAIN>
__global__ void __launch_bounds__(kFwdThreads, 1)
    k_forward(const float* __restrict__ feat, int64_t n, const unsigned char* __restrict__ Wp,
              const float* __restrict__ p, LayerPtrs L, float* __restrict__ out, FwdStore st,
              ErrFlag err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sA = smem_u32(smem), sRing = sA + kFwdOffRing;
    float* s_bias = reinterpret_cast<float*>(smem + kFwdOffBias);
    float4* s_w5 = reinterpret_cast<float4*>(smem + kFwdOffW5);
    float4* s_part = reinterpret_cast<float4*>(smem + kFwdOffPart);
    // barriers: full[4], empty[4], chunk of A ready [4], accumulators ready, row
    // parts ready; then the tensor-memory address
    const uint32_t bar = sA + kFwdOffBar, full = bar, empty = bar + 32, a_ready = bar + 64,
                   acc_ready = bar + 96, part_ready = bar + 104, tslot = bar + 112;
    const int64_t tiles = (n + kFwdRows - 1) / kFwdRows;

    if (tid == 0) {
        for (int i = 0; i < 4; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(full + 8 * i));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(empty + 8 * i));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(a_ready + 8 * i), "r"(kFwdEpi));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(acc_ready));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(part_ready), "r"((kFwdParts - 1) * kFwdRows));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == kFwdMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(tslot));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    for (int i = tid; i < kFwdHidden * 256; i += kFwdThreads) s_bias[i] = p[L.b_off[i >> 8] + (i & 255)];
    for (int i = tid; i < 256; i += kFwdThreads)
        s_w5[i] = make_float4(__bfloat162float(L.W[kLayers - 1][i]), __bfloat162float(L.W[kLayers - 1][256 + i]),
                              __bfloat162float(L.W[kLayers - 1][512 + i]),
                              __bfloat162float(L.W[kLayers - 1][768 + i]));
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem) : "r"(tslot));
    bool ok = true;

    if (warp == kFwdCopyWarp) {  // weight copies
        if (lane == 0) {
            int64_t g = 0;  // chunk counter
            for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                const unsigned char* src = Wp;
                for (int c = 0; c < kFwdChunks; ++c, ++g) {
                    const int slot = int(g % kFwdSlots);
                    const uint32_t bytes = c == 0 ? kFwdIn0Bytes : kFwdSlotBytes;
                    if (g >= kFwdSlots) ok = mbar_wait(empty + 8 * slot, uint32_t(g / kFwdSlots - 1) & 1u);
                    if (!ok) break;
                    bulk_copy(sRing + uint32_t(slot * kFwdSlotBytes), src, bytes, full + 8 * slot);
                    src += bytes;
                }
            }
            // no copy may be in flight when the CTA ends
            for (int64_t i = max(int64_t(0), g - kFwdSlots); i < g; ++i)
                ok = mbar_wait(full + 8 * int(i % kFwdSlots), uint32_t(i / kFwdSlots) & 1u) && ok;
        }
    } else if (warp == kFwdMmaWarp) {  // MMAs
        if (lane == 0) {
            int64_t g = 0, t = 0;
            for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++t) {
                for (int c = 0; c < kFwdChunks && ok; ++c, ++g) {
                    const int l = c == 0 ? 0 : (c + 3) / 4, kc = c == 0 ? 0 : (c - 1) % 4;
                    const int slot = int(g % kFwdSlots);
                    // the chunk of A: layer 0 fills only chunk 0
                    const int64_t phase = kc == 0 ? t * kFwdHidden + l : t * (kFwdHidden - 1) + l - 1;
                    ok = mbar_wait(a_ready + 8 * kc, uint32_t(phase) & 1u) &&
                         mbar_wait(full + 8 * slot, uint32_t(g / kFwdSlots) & 1u);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    mma_chunk(tmem + uint32_t(l & 1) * 256, sA + uint32_t(kc * 1024),
                              sRing + uint32_t(slot * kFwdSlotBytes), c == 0 ? 512u : 1024u, c == 0 ? 2 : 4,
                              kc > 0);
                    mma_commit(empty + 8 * slot);
                    if (c == 0 || kc == 3) mma_commit(acc_ready);
                }
            }
        }
    } else {  // epilogue
        const int quarter = warp & 3, part = warp >> 2;
        const int row = quarter * 32 + lane;  // of the tile; this thread's tensor-memory lane
        int64_t t = 0;
        for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++t) {
            const int64_t m = tile * kFwdRows + row;
            const bool live = m < n;
            {   // the features as BF16, eight a thread
                static_assert(kIn / kFwdParts == 8, "a 16-byte granule");
                uint32_t v[4];
                const float4* f = reinterpret_cast<const float4*>(feat + m * kIn + part * 8);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float4 x = live ? f[i] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
                    v[2 * i] = *reinterpret_cast<const uint32_t*>(&a);
                    v[2 * i + 1] = *reinterpret_cast<const uint32_t*>(&b);
                }
                const uint4 b = make_uint4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<uint4*>(smem + (row >> 3) * 4096 + part * 128 + (row & 7) * 16) = b;
                if (TRAIN) reinterpret_cast<uint4*>(st.Ab[0])[granule(tile, kIn / 8, part, row)] = b;
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                mbar_arrive(a_ready);
            }
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int l = 0; l < kFwdHidden; ++l) {
                ok = __all_sync(0xffffffffu, mbar_wait(acc_ready, uint32_t(t * kFwdHidden + l) & 1u));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const float* bias = s_bias + l * 256;
                for (int kc = 0; kc < 4; ++kc) {  // 64 columns: the next layer's chunk of k
                    const int c0 = kc * 64 + part * kFwdCols;
                    float v[kFwdCols];
                    tmem_ld16(tmem + (uint32_t(quarter * 32) << 16) + uint32_t((l & 1) * 256 + c0), v);
                    uint32_t b[kFwdCols / 2];
#pragma unroll
                    for (int j = 0; j < kFwdCols; j += 4) {
                        const float4 bj = *reinterpret_cast<const float4*>(bias + c0 + j);
                        v[j] = tanhf(v[j] + bj.x);
                        v[j + 1] = tanhf(v[j + 1] + bj.y);
                        v[j + 2] = tanhf(v[j + 2] + bj.z);
                        v[j + 3] = tanhf(v[j + 3] + bj.w);
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(v[j], v[j + 1]),
                                             hi = __floats2bfloat162_rn(v[j + 2], v[j + 3]);
                        b[j / 2] = *reinterpret_cast<const uint32_t*>(&lo);
                        b[j / 2 + 1] = *reinterpret_cast<const uint32_t*>(&hi);
                    }
                    if (l < kFwdHidden - 1) {
                        unsigned char* dst = smem + (row >> 3) * 4096 + (c0 >> 3) * 128 + (row & 7) * 16;
#pragma unroll
                        for (int j = 0; j < kFwdCols / 8; ++j)
                            *reinterpret_cast<uint4*>(dst + j * 128) =
                                make_uint4(b[4 * j], b[4 * j + 1], b[4 * j + 2], b[4 * j + 3]);
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                        mbar_arrive(a_ready + 8 * kc);
                    } else {
#pragma unroll
                        for (int j = 0; j < kFwdCols; ++j) {
                            const uint32_t w = b[j / 2];
                            const float x = __uint_as_float(j & 1 ? w & 0xffff0000u : w << 16);
                            const float4 w5 = s_w5[c0 + j];
                            y.x = fmaf(x, w5.x, y.x);
                            y.y = fmaf(x, w5.y, y.y);
                            y.z = fmaf(x, w5.z, y.z);
                            y.w = fmaf(x, w5.w, y.w);
                        }
                    }
                    if (TRAIN) {
                        float4* of = reinterpret_cast<float4*>(st.Af[l + 1]) + granule(tile, 64, c0 / 4, row);
                        uint4* ob = reinterpret_cast<uint4*>(st.Ab[l + 1]) + granule(tile, 32, c0 / 8, row);
#pragma unroll
                        for (int j = 0; j < kFwdCols / 4; ++j)
                            of[j * kFwdRows] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
#pragma unroll
                        for (int j = 0; j < kFwdCols / 8; ++j)
                            ob[j * kFwdRows] = make_uint4(b[4 * j], b[4 * j + 1], b[4 * j + 2], b[4 * j + 3]);
                    }
                }
            }
            if (!ok) break;
            // a row's parts are added by its first thread (another one writes its
            // next part only after every thread has passed the next tile's layers)
            if (part > 0) {
                s_part[(part - 1) * kFwdRows + row] = y;
                mbar_arrive(part_ready);
                continue;
            }
            ok = __all_sync(0xffffffffu, mbar_wait(part_ready, uint32_t(t) & 1u));
            if (ok && live) {
                const float* b5 = p + L.b_off[kLayers - 1];
#pragma unroll
                for (int i = 0; i < kFwdParts - 1; ++i) {
                    const float4 z = s_part[i * kFwdRows + row];
                    y = make_float4(y.x + z.x, y.y + z.y, y.z + z.z, y.w + z.w);
                }
                reinterpret_cast<float4*>(out)[m] = make_float4(y.x + b5[0], y.y + b5[1], y.z + b5[2], y.w + b5[3]);
            }
        }
    }
    if (!ok && lane == 0) raise(err, kPassForward);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    __syncwarp();
    if (warp == kFwdMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// ------------------------------------------------- forward pass on mma.sync
// The same pass with warp-level products (mma.sync m16n8k16) and no wait that could
// run out, for handles that choose LSKUM_MLP_GEMM_MMA_SYNC. A CTA takes 64 rows: their
// activations stay in shared memory, the weights come through two buffers of 64
// k by cp.async, the next one while a chunk is multiplied; a warp has 32 outputs of
// all 64 rows. The products of a row are added in the order of k, 16 at a time.
// 16,384 samples: 77 us a prediction, where a launch for each layer took 179 and the
// tcgen05 pass takes 46.
constexpr int kMmaRows = 64, kMmaThreads = 256;
constexpr int kMmaLdA = 256 + 8, kMmaLdW = 64 + 8;  // BF16 a row: eight rows 16 bytes apart in the banks
constexpr int kMmaSmem = (kMmaRows * kMmaLdA + 2 * 256 * kMmaLdW) * 2;
static_assert(kFwdRows % kMmaRows == 0, "a CTA's rows lie in one tile");

// Four 8 x 8 BF16 matrices: lane i gives the address of row i % 8 of matrix i / 8.
__device__ __forceinline__ void ldmatrix4(uint32_t r[4], const __nv_bfloat16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p))
                 : "memory");
}

__device__ __forceinline__ void mma_16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Chunk c of the weights (as k_forward counts them) into a buffer.
__device__ __forceinline__ void load_weights(const LayerPtrs& L, int c, __nv_bfloat16* to) {
    const int l = c == 0 ? 0 : (c + 3) / 4, k0 = c == 0 ? 0 : (c - 1) % 4 * 64, per_row = c == 0 ? 4 : 8;
    const __nv_bfloat16* W = L.W[l] + k0;
    for (int i = threadIdx.x; i < 256 * per_row; i += kMmaThreads) {
        const int n = i / per_row, g = i % per_row;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(to + n * kMmaLdW + g * 8)),
                     "l"(W + int64_t(n) * layer_in(l) + g * 8)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

template <bool TRAIN>
__global__ void __launch_bounds__(kMmaThreads)
    k_forward_mma(const float* __restrict__ feat, int64_t n, const float* __restrict__ p, LayerPtrs L,
                  float* __restrict__ out, FwdStore st) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __nv_bfloat16* sA = reinterpret_cast<__nv_bfloat16*>(smem);
    __nv_bfloat16* sW = sA + kMmaRows * kMmaLdA;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t m0 = int64_t(blockIdx.x) * kMmaRows, tile = m0 / kFwdRows;
    const int row0 = int(m0 % kFwdRows);  // of the tile
    load_weights(L, 0, sW);
    for (int i = tid; i < kMmaRows * kIn / 2; i += kMmaThreads) {  // the features as BF16; rows past n are zero
        const int r = i / (kIn / 2), k = i % (kIn / 2) * 2;
        const float2 x = m0 + r < n ? *reinterpret_cast<const float2*>(feat + (m0 + r) * kIn + k) : make_float2(0.f, 0.f);
        const __nv_bfloat162 b = __floats2bfloat162_rn(x.x, x.y);
        *reinterpret_cast<__nv_bfloat162*>(sA + r * kMmaLdA + k) = b;
        if (TRAIN)
            *reinterpret_cast<__nv_bfloat162*>(st.Ab[0] + granule(tile, kIn / 8, k / 8, row0 + r) * 8 + k % 8) = b;
    }
    float acc[4][4][4];  // 16 rows x 8 outputs each
    for (int c = 0; c < kFwdChunks; ++c) {
        const int l = c == 0 ? 0 : (c + 3) / 4, kc = c == 0 ? 0 : (c - 1) % 4;
        const __nv_bfloat16* W = sW + (c & 1) * 256 * kMmaLdW;
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();  // chunk c and A are there; the other buffer has been multiplied
        if (c + 1 < kFwdChunks) load_weights(L, c + 1, sW + (~c & 1) * 256 * kMmaLdW);
        if (kc == 0) {
#pragma unroll
            for (int i = 0; i < 64; ++i) acc[i / 16][i / 4 % 4][i % 4] = 0.f;
        }
        for (int ks = 0; ks < (c == 0 ? kIn : 64); ks += 16) {
            uint32_t b[2][4];  // per 16 outputs: {0-7 | k 0-7}, {0-7 | 8-15}, {8-15 | 0-7}, {8-15 | 8-15}
#pragma unroll
            for (int j = 0; j < 2; ++j)
                ldmatrix4(b[j], W + (warp * 32 + j * 16 + (lane >> 4) * 8 + (lane & 7)) * kMmaLdW + ks +
                                    (lane >> 3 & 1) * 8);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t a[4];
                ldmatrix4(a, sA + (i * 16 + (lane & 15)) * kMmaLdA + kc * 64 + ks + (lane >> 4) * 8);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_16816(acc[i][j], a, b[j / 2][j % 2 * 2], b[j / 2][j % 2 * 2 + 1]);
            }
        }
        if (c != 0 && kc != 3) continue;
        __syncthreads();  // A has been read
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int o = warp * 32 + j * 8 + (lane & 3) * 2;
                const float2 bias = *reinterpret_cast<const float2*>(p + L.b_off[l] + o);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = i * 16 + h * 8 + (lane >> 2);
                    const float2 v = make_float2(tanhf(acc[i][j][2 * h] + bias.x), tanhf(acc[i][j][2 * h + 1] + bias.y));
                    const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
                    *reinterpret_cast<__nv_bfloat162*>(sA + r * kMmaLdA + o) = b;
                    if (TRAIN) {
                        *reinterpret_cast<float2*>(st.Af[l + 1] + granule(tile, 64, o / 4, row0 + r) * 4 + o % 4) = v;
                        *reinterpret_cast<__nv_bfloat162*>(st.Ab[l + 1] + granule(tile, 32, o / 8, row0 + r) * 8 + o % 8) = b;
                    }
                }
            }
    }
    __syncthreads();
    const int r = tid / kOut, o = tid % kOut;  // the output layer: a thread an output
    const __nv_bfloat16 *x = sA + r * kMmaLdA, *w = L.W[kLayers - 1] + o * 256;
    float y = 0.f;
#pragma unroll 8
    for (int k = 0; k < 256; ++k) y = fmaf(__bfloat162float(x[k]), __bfloat162float(w[k]), y);
    if (m0 + r < n) out[(m0 + r) * kOut + o] = y + p[L.b_off[kLayers - 1] + o];
}

// Sums over the lanes of v[0..31]: lane j ends with element j's in v[0].
__device__ __forceinline__ void sum_lanes(float v[32], const int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < o; ++j) {
            const float keep = lane & o ? v[j + o] : v[j], give = lane & o ? v[j] : v[j + o];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
}

// Of v[0..15] likewise: lanes j and j + 16 end with element j's.
__device__ __forceinline__ void sum_lanes16(float v[16], const int lane) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < o; ++j) {
            const float keep = lane & o ? v[j + o] : v[j], give = lane & o ? v[j] : v[j + o];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// ------------------------------------------------- fused backward pass
// The error signals of a 128-row tile from the output to the first layer in one
// CTA, as k_forward runs forwards (8,192 samples: loss and gradients 659 us with
// a launch for each layer's product, sum and tanh', now 114): dZ_4 = (dY W_5) (1 - A_5^2) by FP32 FMAs, then
// dZ_(l-1) = (dZ_l W_l) (1 - A_l^2) for l = 4..1 with the products on the tensor
// cores. Stores each layer's dZ in BF16 (the weight gradients' operand), the
// column sums of the FP32 dZ (the bias gradients; one row of partial sums for
// each CTA and tensor-memory quarter) and the squared error.
constexpr int kBwdSums = kFwdHidden * kWidth;  // columns of a partial row; then dY's 4

struct BwdArgs {
    const float* Y;  // n x 4 outputs and targets
    const float* T;
    const float* Af[kLayers];      // A_l, l = 1..5, in granules
    __nv_bfloat16* dZb[kLayers];   // dZ_l, l = 0..4 in granules, 5 n x 4
    const unsigned char* Wt;       // transposed operand images
    const __nv_bfloat16* W5;       // 4 x 256
    float* sums;                   // [4 gridDim][kBwdSums + 4]
    double* sq;                    // [4 gridDim]
};

__global__ void __launch_bounds__(kFwdThreads, 1) k_backward(const BwdArgs a, int64_t n, ErrFlag err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sA = smem_u32(smem), sRing = sA + kFwdOffRing;
    float4* s_w5 = reinterpret_cast<float4*>(smem + kFwdOffW5);
    const uint32_t bar = sA + kFwdOffBar, full = bar, empty = bar + 32, a_ready = bar + 64,
                   acc_ready = bar + 96, tslot = bar + 112;
    const int64_t tiles = (n + kFwdRows - 1) / kFwdRows;
    constexpr int kSteps = kFwdHidden - 1;  // layers on the tensor cores

    if (tid == 0) {
        for (int i = 0; i < 4; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(full + 8 * i));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(empty + 8 * i));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(a_ready + 8 * i), "r"(kFwdEpi));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(acc_ready));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == kFwdMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(tslot));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    for (int i = tid; i < 256; i += kFwdThreads)
        s_w5[i] = make_float4(__bfloat162float(a.W5[i]), __bfloat162float(a.W5[256 + i]),
                              __bfloat162float(a.W5[512 + i]), __bfloat162float(a.W5[768 + i]));
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem) : "r"(tslot));
    bool ok = true;

    if (warp == kFwdCopyWarp) {  // weight copies
        if (lane == 0) {
            int64_t g = 0;
            for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                const unsigned char* src = a.Wt;
                for (int c = 0; c < 4 * kSteps; ++c, ++g, src += kFwdSlotBytes) {
                    const int slot = int(g % kFwdSlots);
                    if (g >= kFwdSlots) ok = mbar_wait(empty + 8 * slot, uint32_t(g / kFwdSlots - 1) & 1u);
                    if (!ok) break;
                    bulk_copy(sRing + uint32_t(slot * kFwdSlotBytes), src, kFwdSlotBytes, full + 8 * slot);
                }
            }
            for (int64_t i = max(int64_t(0), g - kFwdSlots); i < g; ++i)
                ok = mbar_wait(full + 8 * int(i % kFwdSlots), uint32_t(i / kFwdSlots) & 1u) && ok;
        }
    } else if (warp == kFwdMmaWarp) {  // MMAs
        if (lane == 0) {
            int64_t g = 0;
            for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                for (int c = 0; c < 4 * kSteps && ok; ++c, ++g) {
                    const int kc = c % 4, slot = int(g % kFwdSlots);
                    ok = mbar_wait(a_ready + 8 * kc, uint32_t(g / 4) & 1u) &&
                         mbar_wait(full + 8 * slot, uint32_t(g / kFwdSlots) & 1u);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    mma_chunk(tmem + uint32_t(c / 4 & 1) * 256, sA + uint32_t(kc * 1024),
                              sRing + uint32_t(slot * kFwdSlotBytes), 1024, 4, kc > 0);
                    mma_commit(empty + 8 * slot);
                    if (kc == 3) mma_commit(acc_ready);
                }
            }
        }
    } else {  // epilogue
        const int quarter = warp & 3, part = warp >> 2;
        const int row = quarter * 32 + lane;
        const float scale = float(n * kOut);
        float db[kFwdHidden][4] = {};  // this lane's columns: layer, chunk
        float4 db5 = make_float4(0.f, 0.f, 0.f, 0.f);
        double sq = 0.0;
        int64_t t = 0;
        for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++t) {
            const int64_t m = tile * kFwdRows + row;
            const bool live = m < n;
            // dY = 2 (Y - T) / (4 n), and its BF16 rounding
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (live) {
                const float* y = a.Y + m * kOut;
                const float* g = a.T + m * kOut;
                d = make_float4(y[0] - g[0], y[1] - g[1], y[2] - g[2], y[3] - g[3]);
            }
            const float4 dy = make_float4(2.0f * d.x / scale, 2.0f * d.y / scale, 2.0f * d.z / scale,
                                          2.0f * d.w / scale);
            const __nv_bfloat162 b01 = __floats2bfloat162_rn(dy.x, dy.y), b23 = __floats2bfloat162_rn(dy.z, dy.w);
            const float2 r01 = __bfloat1622float2(b01), r23 = __bfloat1622float2(b23);
            if (part == 0) {
                sq += double(d.x) * d.x + double(d.y) * d.y + double(d.z) * d.z + double(d.w) * d.w;
                db5.x += dy.x;
                db5.y += dy.y;
                db5.z += dy.z;
                db5.w += dy.w;
                if (live)
                    reinterpret_cast<uint2*>(a.dZb[kLayers - 1])[m] =
                        make_uint2(*reinterpret_cast<const uint32_t*>(&b01), *reinterpret_cast<const uint32_t*>(&b23));
            }
#pragma unroll
            for (int i = 0; i < kFwdHidden; ++i) {  // dZ_l, l = 4 - i
                const int l = kFwdHidden - 1 - i;
                if (i > 0) {
                    ok = __all_sync(0xffffffffu, mbar_wait(acc_ready, uint32_t(t * kSteps + i - 1) & 1u));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                }
                const float4* act = reinterpret_cast<const float4*>(a.Af[l + 1]) + granule(tile, 64, 0, row);
                uint4* to = reinterpret_cast<uint4*>(a.dZb[l]) + granule(tile, 32, 0, row);
#pragma unroll
                for (int kc = 0; kc < 4; ++kc) {
                    const int c0 = kc * 64 + part * kFwdCols;
                    float v[kFwdCols];
                    if (i == 0) {
#pragma unroll
                        for (int j = 0; j < kFwdCols; ++j) {
                            const float4 w = s_w5[c0 + j];
                            v[j] = fmaf(r23.y, w.w, fmaf(r23.x, w.z, fmaf(r01.y, w.y, r01.x * w.x)));
                        }
                    } else {
                        tmem_ld16(tmem + (uint32_t(quarter * 32) << 16) + uint32_t(((i - 1) & 1) * 256 + c0), v);
                    }
                    uint32_t b[kFwdCols / 2];
#pragma unroll
                    for (int j = 0; j < kFwdCols; j += 4) {
                        const float4 x = act[(c0 + j) / 4 * kFwdRows];
                        v[j] *= 1.0f - x.x * x.x;
                        v[j + 1] *= 1.0f - x.y * x.y;
                        v[j + 2] *= 1.0f - x.z * x.z;
                        v[j + 3] *= 1.0f - x.w * x.w;
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(v[j], v[j + 1]),
                                             hi = __floats2bfloat162_rn(v[j + 2], v[j + 3]);
                        b[j / 2] = *reinterpret_cast<const uint32_t*>(&lo);
                        b[j / 2 + 1] = *reinterpret_cast<const uint32_t*>(&hi);
                    }
                    if (l > 0) {
                        unsigned char* dst = smem + (row >> 3) * 4096 + (c0 >> 3) * 128 + (row & 7) * 16;
#pragma unroll
                        for (int j = 0; j < kFwdCols / 8; ++j)
                            *reinterpret_cast<uint4*>(dst + j * 128) =
                                make_uint4(b[4 * j], b[4 * j + 1], b[4 * j + 2], b[4 * j + 3]);
                        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                        mbar_arrive(a_ready + 8 * kc);
                    }
#pragma unroll
                    for (int j = 0; j < kFwdCols / 8; ++j)
                        to[(c0 / 8 + j) * kFwdRows] = make_uint4(b[4 * j], b[4 * j + 1], b[4 * j + 2], b[4 * j + 3]);
                    sum_lanes16(v, lane);  // the warp's 32 rows: lanes j, j + 16 end with column j
                    db[l][kc] += v[0];
                }
            }
        }
        // partial sums: one row for each CTA and quarter
        const int64_t r = int64_t(blockIdx.x) * 4 + quarter;
        float* out = a.sums + r * (kBwdSums + kOut);
#pragma unroll
        for (int l = 0; l < kFwdHidden; ++l)
#pragma unroll
            for (int kc = 0; kc < 4; ++kc)
                if (lane < kFwdCols) out[l * kWidth + kc * 64 + part * kFwdCols + lane] = db[l][kc];
        if (part == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sq += __shfl_xor_sync(0xffffffffu, sq, o);
                db5.x += __shfl_xor_sync(0xffffffffu, db5.x, o);
                db5.y += __shfl_xor_sync(0xffffffffu, db5.y, o);
                db5.z += __shfl_xor_sync(0xffffffffu, db5.z, o);
                db5.w += __shfl_xor_sync(0xffffffffu, db5.w, o);
            }
            if (lane == 0) {
                a.sq[r] = sq;
                out[kBwdSums] = db5.x;
                out[kBwdSums + 1] = db5.y;
                out[kBwdSums + 2] = db5.z;
                out[kBwdSums + 3] = db5.w;
            }
        }
    }
    if (!ok && lane == 0) raise(err, kPassBackward);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    __syncwarp();
    if (warp == kFwdMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// All weight gradients of a slice of the tiles, dW_l = dZ_l^T A_l, in one launch:
// blockIdx.x 0..7 the layers 1..4 in halves of 128 outputs, 8 and 9 the first
// layer's halves. Slice z goes to part + z * np, a whole parameter vector, each
// half in granules of four columns by output unit, so that a
// warp's store of 32 units is one access. A tile's operands are contiguous
// (granules): one bulk copy each, two tiles in flight, eight MMAs (M 128, N 256
// or 32, K 16 rows) with both operands' contraction index the slower one; the
// accumulator goes out once a slice. Meanwhile the epilogue's four warps take
// the output layer's gradient by FP32 FMAs, three or four of its 32 column
// granules a block: as blocks of their own those were the last to end. Bound by
// the copies, 96 KB a tile and half layer from L2, in one wave of at most 150
// blocks (8,192 samples 14 us; mma.sync tiles that re-read both operands 36).
struct DwArgs {
    const __nv_bfloat16* dZb[kLayers];
    const __nv_bfloat16* X[kLayers];
    LayerPtrs L;
    float* part;
    int64_t np;
};
constexpr int kDwThreads = 192;  // four epilogue warps, an MMA and a copy warp
constexpr int kDwA = 16 * kFwdRows * 16, kDwB = 32 * kFwdRows * 16;  // bytes a tile
constexpr int kDwOffBar = 2 * (kDwA + kDwB);
constexpr int kDwSmem = kDwOffBar + 64;
static_assert(kDwSmem <= 227 * 1024, "one CTA's shared memory");

__global__ void __launch_bounds__(kDwThreads, 1) k_weight_grads(const DwArgs a, int n, int tiles_per_slice,
                                                                ErrFlag err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles = (n + kFwdRows - 1) / kFwdRows;
    const int t0 = int(blockIdx.z) * tiles_per_slice, t1 = min(tiles, t0 + tiles_per_slice);
    const int l = blockIdx.x < 8 ? int(blockIdx.x) / 2 + 1 : 0, half = blockIdx.x & 1;
    const int K = layer_in(l), bytesB = K / 8 * kFwdRows * 16;
    const uint32_t sA = smem_u32(smem), sB = sA + 2 * kDwA;
    const uint32_t bar = sA + kDwOffBar, full = bar, empty = bar + 16, done = bar + 32, tslot = bar + 40;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(full + 8 * i));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(empty + 8 * i));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(done));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;\n" ::"r"(tslot));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    uint32_t tmem;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(tmem) : "r"(tslot));
    bool ok = true;
    if (warp == 5) {  // copies
        if (lane == 0) {
            int i = 0;
            for (int t = t0; t < t1; ++t, ++i) {
                const int s = i & 1;
                if (i >= 2) ok = mbar_wait(empty + 8 * s, uint32_t(i / 2 - 1) & 1u);
                if (!ok) break;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(full + 8 * s),
                             "r"(kDwA + bytesB)
                             : "memory");
                bulk_copy_only(sA + uint32_t(s * kDwA),
                               reinterpret_cast<const uint4*>(a.dZb[l]) + granule(t, kWidth / 8, half * 16, 0), kDwA,
                               full + 8 * s);
                bulk_copy_only(sB + uint32_t(s * kDwB), reinterpret_cast<const uint4*>(a.X[l]) + granule(t, K / 8, 0, 0),
                               bytesB, full + 8 * s);
            }
            for (int j = max(0, i - 2); j < i; ++j) ok = mbar_wait(full + 8 * (j & 1), uint32_t(j / 2) & 1u) && ok;
        }
    } else if (warp == 4) {  // MMAs: both operands with the contraction (rows) as the slower index
        if (lane == 0) {
            const uint32_t idesc = umma_idesc_bf16_f32(kFwdRows, K) | (1u << 15) | (1u << 16);
            int i = 0;
            for (int t = t0; t < t1 && ok; ++t, ++i) {
                const int s = i & 1;
                ok = mbar_wait(full + 8 * s, uint32_t(i / 2) & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                for (int ks = 0; ks < kFwdRows / 16; ++ks)
                    asm volatile(
                        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                        "l"(umma_desc(sA + uint32_t(s * kDwA + ks * 256), 128, kFwdRows * 16)),
                        "l"(umma_desc(sB + uint32_t(s * kDwB + ks * 256), 128, kFwdRows * 16)), "r"(idesc),
                        "r"(i + ks));
                mma_commit(empty + 8 * s);
            }
            if (ok) mma_commit(done);
        }
    } else {
        const int g = int(blockIdx.x) + 10 * warp;  // 4 x 8 of the output layer's: lanes take the rows
        if (g < kWidth / 8) {
            constexpr int o = kLayers - 1;
            const uint4* X = reinterpret_cast<const uint4*>(a.X[o]);
            const uint2* dz = reinterpret_cast<const uint2*>(a.dZb[o]);
            float v[32] = {};  // [output][column]
            for (int t = t0; t < t1; ++t)
#pragma unroll
                for (int r = lane; r < kFwdRows; r += 32) {
                    const int64_t m = int64_t(t) * kFwdRows + r;
                    const uint4 x = X[granule(t, kWidth / 8, g, r)];
                    const uint2 d = m < n ? dz[m] : make_uint2(0u, 0u);
                    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ds[2] = {d.x, d.y};
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const uint32_t xw = xs[j % 8 / 2], dw = ds[j / 16];
                        v[j] = fmaf(__uint_as_float(j & 1 ? xw & 0xffff0000u : xw << 16),
                                    __uint_as_float(j & 8 ? dw & 0xffff0000u : dw << 16), v[j]);
                    }
                }
            sum_lanes(v, lane);
            a.part[int64_t(blockIdx.z) * a.np + a.L.w_off[o] + (lane / 8) * kWidth + g * 8 + lane % 8] = v[0];
        }
        // the slice's sums: a thread an output unit
        ok = __all_sync(0xffffffffu, mbar_wait(done, 0));
        if (ok) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            float4* to = reinterpret_cast<float4*>(a.part + int64_t(blockIdx.z) * a.np + a.L.w_off[l] +
                                                   int64_t(half) * 128 * K) + warp * 32 + lane;
            for (int c = 0; c < K; c += 32) {
                float v[32];
                tmem_ld32(tmem + (uint32_t(warp * 32) << 16) + uint32_t(c), v);
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    to[(c + j) / 4 * 128] = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
        }
    }
    if (!ok && lane == 0) raise(err, kPassWeightGrads);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    __syncwarp();
    if (warp == 4) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;\n" ::"r"(tmem));
}

// The gradient vector from the slices (in slice order) and the partial column
// sums, and the loss: mean squared error. The first kBiasBlocks blocks take 32
// columns of the sums each (eight threads a column, added in order), the next
// one the loss, the others 256 weights each.
constexpr int kBiasBlocks = (kBwdSums + kOut + 31) / 32;

__global__ void __launch_bounds__(256) k_reduce_grads(const DwArgs a, int slices, const float* __restrict__ sums,
                                                      const double* __restrict__ sq, int rows, double count,
                                                      float* __restrict__ g, double* __restrict__ loss) {
    const int tid = threadIdx.x;
    if (blockIdx.x < kBiasBlocks) {
        __shared__ float part[8][32];
        const int c = int(blockIdx.x) * 32 + tid % 32;
        float s = 0.f;
        if (c < kBwdSums + kOut) {
#pragma unroll 8
            for (int r = tid / 32; r < rows; r += 8) s += sums[int64_t(r) * (kBwdSums + kOut) + c];
        }
        part[tid / 32][tid % 32] = s;
        __syncthreads();
        if (tid < 32 && c < kBwdSums + kOut) {
            float t = 0.f;
            for (int k = 0; k < 8; ++k) t += part[k][tid];
            g[a.L.b_off[c / kWidth] + c % kWidth] = t;  // kBwdSums is a multiple of kWidth
        }
    } else if (blockIdx.x == kBiasBlocks) {
        __shared__ double part[256];
        double s = 0.0;
        for (int r = tid; r < rows; r += 256) s += sq[r];
        part[tid] = s;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (tid < o) part[tid] += part[tid + o];
            __syncthreads();
        }
        if (tid == 0) *loss = part[0] / count;
    } else {
        const int64_t e = int64_t(blockIdx.x - kBiasBlocks - 1) * 256 + tid;
        if (e >= a.np) return;
        int l = kLayers - 1;
        while (e < a.L.w_off[l]) --l;
        if (e >= a.L.b_off[l]) return;  // a bias
        float s = 0.f;
#pragma unroll 8
        for (int z = 0; z < slices; ++z) s += a.part[int64_t(z) * a.np + e];
        const int i = int(e - a.L.w_off[l]), K = layer_in(l), half = i / (128 * K), q = i % (128 * K);
        g[l == kLayers - 1 ? e : a.L.w_off[l] + (half * 128 + q / 4 % 128) * K + q / 512 * 4 + q % 4] = s;
    }
}

// Features: per sample raw (x, y, wall distance, M, alpha_deg) ->
// [x/10, y/10, log(d + 1e-3)/5, (M - 0.55)/0.25, (alpha - 1)/5,
//  sin(P (x, y)), cos(P (x, y)) (8 projections each), 0 x 11 padding],
// stored FP32 (the caller-visible encoding) and BF16 (GEMM input).
__global__ void k_features(const float* __restrict__ raw, int64_t n, const float* __restrict__ proj,
                           float* __restrict__ feat) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* r = raw + 5 * i;
    float* f = feat + int64_t(kIn) * i;
    const float x = r[0], y = r[1];
    f[0] = x * 0.1f;
    f[1] = y * 0.1f;
    f[2] = logf(r[2] + 1e-3f) * 0.2f;
    f[3] = (r[3] - 0.55f) * 4.0f;
    f[4] = (r[4] - 1.0f) * 0.2f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float t = proj[2 * k] * x + proj[2 * k + 1] * y;
        f[5 + k] = sinf(t);
        f[13 + k] = cosf(t);
    }
#pragma unroll
    for (int k = 21; k < kIn; ++k) f[k] = 0.f;
}

// Adam on the flat FP32 parameter vector; the BF16 copies are refreshed after it.
// Nothing changes once a wait has run out in this step or one before it; *done
// receives the number of an applied step.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2, const int* __restrict__ err, int64_t step, int64_t* done) {
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n || *err) return;
    if (i == 0) *done = step;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// BF16 copies of the weights: row-major, and as the operand images of the fused
// forward and backward passes. (Parameters that Adam left alone give the same
// copies again.)
__global__ void k_weights_bf16(const float* __restrict__ p, LayerPtrs L, unsigned char* __restrict__ Wp,
                               unsigned char* __restrict__ Wt) {
    const int l = blockIdx.y;
    const int K = layer_in(l), N = layer_out(l);
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= int64_t(K) * N) return;
    const int row = int(e / K), k = int(e % K);
    float w = p[L.w_off[l] + e];
    if (l == 0 && k >= 21) w = 0.f;  // padded inputs carry no weight
    const __nv_bfloat16 b = __float2bfloat16(w);
    L.W[l][e] = b;
    if (l < kLayers - 1) *reinterpret_cast<__nv_bfloat16*>(Wp + packed_offset(l, row, k)) = b;
    if (l > 0 && l < kLayers - 1) *reinterpret_cast<__nv_bfloat16*>(Wt + packed_offset_t(l, row, k)) = b;
}

}  // namespace mlpk

// ------------------------------------------------------------------ C ABI

using namespace mlpk;

struct lskum_mlp {
    cudaStream_t stream = nullptr;      // stream the handle's work runs on
    cudaStream_t own_stream = nullptr;  // the handle's own (created, destroyed by it)
    int64_t cap = 0;  // samples per call
    int64_t nparam = 0;
    LayerPtrs L{};
    float* p = nullptr;   // FP32 master parameters
    float* g = nullptr;   // gradients
    float* m = nullptr;   // Adam moments
    float* v = nullptr;
    float* proj = nullptr;  // 8 x 2 Fourier projection
    int64_t step = 0;
    int gemm_path = LSKUM_MLP_GEMM_TCGEN05;  // forward pass
    // activations in granules: Af[l] (FP32, l = 1..5) and Ab[l] (BF16, l = 0..5;
    // l = 0: features); Af[0] staged features, Af[kLayers] outputs
    float* Af[kLayers + 1] = {nullptr};
    __nv_bfloat16* Ab[kLayers + 1] = {nullptr};
    __nv_bfloat16* dZb[kLayers] = {nullptr};  // error signals (BF16)
    float* slices = nullptr;  // partial weight gradients: a parameter vector for each slice
    float* sums = nullptr;    // partial bias gradients: a row for each CTA and quarter
    double* partial = nullptr;  // and squared errors
    double* loss_dev = nullptr;
    unsigned char* Wp = nullptr;  // operand images of the weights: forward pass
    unsigned char* Wt = nullptr;  // and backward pass
    int sms = 0;
    ErrFlag err{};          // raised by a pass one of whose waits ran out
    int64_t* done = nullptr;  // pinned: the last step that Adam applied
    std::vector<void*> allocs;
};

namespace {

int fail(int code, const std::string& m) {
    lskum::set_last_error(m);
    return code;
}

#define MLP_CUDA(x)                                                                    \
    do {                                                                               \
        cudaError_t e_ = (x);                                                          \
        if (e_ != cudaSuccess) return fail(LSKUM_ERR_CUDA, std::string(#x) + ": " +     \
                                                           cudaGetErrorString(e_));    \
    } while (0)

template <typename T>
cudaError_t alloc(lskum_mlp* h, T** p, int64_t count) {
    void* raw = nullptr;
    cudaError_t e = cudaMalloc(&raw, sizeof(T) * size_t(count > 0 ? count : 1));
    if (e == cudaSuccess) h->allocs.push_back(raw);
    *p = static_cast<T*>(raw);
    return e;
}

inline unsigned blocks(int64_t n, int b) { return unsigned((n + b - 1) / b); }

constexpr int kMaxSlices = 15;  // of ten blocks: one wave

// After a synchronising call: LSKUM_ERR_TIMEOUT if a pass gave up one of its waits.
// The steps queued from that pass on were not applied; they are not counted, and
// with the flag cleared the handle goes on from the last applied one.
int check_passes(lskum_mlp* h) {
    if (!*static_cast<volatile int*>(h->err.host)) return LSKUM_OK;
    int passes = 0;
    MLP_CUDA(cudaMemcpyAsync(&passes, h->err.dev, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->err.dev, 0, sizeof(int), h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    *h->err.host = 0;
    h->step = *static_cast<volatile int64_t*>(h->done);
    std::string which;
    for (const auto& [bit, name] : {std::pair(kPassForward, "forward pass"), std::pair(kPassBackward, "backward pass"),
                                    std::pair(kPassWeightGrads, "weight gradients")})
        if (passes & bit) which += std::string(which.empty() ? "" : ", ") + name;
    return fail(LSKUM_ERR_TIMEOUT, which + ": a wait ran out");
}

// Forward pass from features (FP32 n x 32) to out (n x 4); train: the hidden
// activations are kept for the backward pass.
int forward(lskum_mlp* h, const float* feat, int64_t n, float* out, bool train) {
    const int64_t tiles = (n + kFwdRows - 1) / kFwdRows;
    const unsigned grid = unsigned(std::min<int64_t>(tiles, h->sms));
    FwdStore st;
    for (int l = 0; l < kLayers; ++l) {
        st.Af[l] = h->Af[l];
        st.Ab[l] = h->Ab[l];
    }
    if (h->gemm_path == LSKUM_MLP_GEMM_MMA_SYNC) {
        const unsigned ctas = unsigned(tiles * (kFwdRows / kMmaRows));  // whole tiles
        if (train)
            k_forward_mma<true><<<ctas, kMmaThreads, kMmaSmem, h->stream>>>(feat, n, h->p, h->L, out, st);
        else
            k_forward_mma<false><<<ctas, kMmaThreads, kMmaSmem, h->stream>>>(feat, n, h->p, h->L, out, st);
    } else if (train)
        k_forward<true><<<grid, kFwdThreads, kFwdSmem, h->stream>>>(feat, n, h->Wp, h->p, h->L, out, st, h->err);
    else
        k_forward<false><<<grid, kFwdThreads, kFwdSmem, h->stream>>>(feat, n, h->Wp, h->p, h->L, out, st, h->err);
    MLP_CUDA(cudaGetLastError());
    return LSKUM_OK;
}

// The features where the forward pass can read them with 16-byte loads while
// `out` is written: the caller's, or a copy of them.
int stage_features(lskum_mlp* h, const float* feat, int64_t n, const float* out, const float** use) {
    const uintptr_t f = reinterpret_cast<uintptr_t>(feat), o = reinterpret_cast<uintptr_t>(out);
    const bool apart = !out || o >= f + sizeof(float) * n * kIn || f >= o + sizeof(float) * n * kOut;
    *use = feat;
    if (!(f & 15) && apart) return LSKUM_OK;
    MLP_CUDA(cudaMemcpyAsync(h->Af[0], feat, sizeof(float) * n * kIn, cudaMemcpyDeviceToDevice, h->stream));
    *use = h->Af[0];
    return LSKUM_OK;
}

// backward from targets T (device n x 4): gradients into h->g, loss into loss_dev
int backward(lskum_mlp* h, const float* T, int64_t n) {
    const int64_t tiles = (n + kFwdRows - 1) / kFwdRows;
    const unsigned grid = unsigned(std::min<int64_t>(tiles, h->sms));
    BwdArgs b;
    DwArgs w;
    b.Y = h->Af[kLayers];
    b.T = T;
    for (int l = 0; l < kLayers; ++l) {
        b.Af[l] = h->Af[l];
        b.dZb[l] = h->dZb[l];
        w.dZb[l] = h->dZb[l];
        w.X[l] = h->Ab[l];
    }
    b.Wt = h->Wt;
    b.W5 = h->L.W[kLayers - 1];
    b.sums = h->sums;
    b.sq = h->partial;
    w.L = h->L;
    w.part = h->slices;
    w.np = h->nparam;
    k_backward<<<grid, kFwdThreads, kFwdSmem, h->stream>>>(b, n, h->err);
    MLP_CUDA(cudaGetLastError());
    // at most kMaxSlices slices of whole tiles
    const int per_slice = int((tiles + kMaxSlices - 1) / kMaxSlices);
    const int slices = int((tiles + per_slice - 1) / per_slice);
    k_weight_grads<<<dim3(10, 1, slices), kDwThreads, kDwSmem, h->stream>>>(w, int(n), per_slice, h->err);
    MLP_CUDA(cudaGetLastError());
    k_reduce_grads<<<kBiasBlocks + 1 + blocks(h->nparam, 256), 256, 0, h->stream>>>(w, slices, h->sums, h->partial, int(grid) * 4,
                                                                  double(n * kOut), h->g, h->loss_dev);
    MLP_CUDA(cudaGetLastError());
    return LSKUM_OK;
}

int check_n(lskum_mlp* h, int64_t n) {
    if (n < 1 || n > h->cap)
        return fail(LSKUM_ERR_INVALID_ARG, "n = " + std::to_string(n) + " outside [1, " +
                                               std::to_string(h->cap) + "]");
    return LSKUM_OK;
}

}  // namespace

extern "C" {

int64_t lskum_mlp_num_params(void) {
    int64_t s = 0;
    for (int l = 0; l < kLayers; ++l) s += int64_t(layer_in(l)) * layer_out(l) + layer_out(l);
    return s;
}

int lskum_mlp_create(int64_t capacity, const float* proj, lskum_mlp** out) {
    if (!out || !proj || capacity < 1 || capacity > (int64_t(1) << 24))
        return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_create: invalid argument");
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0)
        return fail(LSKUM_ERR_CUDA, "lskum_mlp_create: no usable CUDA device");
    lskum_mlp* h = new lskum_mlp();
    h->cap = capacity;
    h->nparam = lskum_mlp_num_params();
    auto bail = [&](cudaError_t e) {
        for (void* p : h->allocs) cudaFree(p);
        if (h->err.host) cudaFreeHost(h->err.host);
        if (h->done) cudaFreeHost(h->done);
        if (h->own_stream) cudaStreamDestroy(h->own_stream);
        delete h;
        return fail(LSKUM_ERR_CUDA, std::string("lskum_mlp_create: ") + cudaGetErrorString(e));
    };
    cudaError_t e;
    if ((e = cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking)) != cudaSuccess) return bail(e);
    h->stream = h->own_stream;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return bail(e);
    int64_t off = 0;
    for (int l = 0; l < kLayers; ++l) {
        h->L.w_off[l] = off;
        off += int64_t(layer_in(l)) * layer_out(l);
        h->L.b_off[l] = off;
        off += layer_out(l);
        if ((e = alloc(h, &h->L.W[l], int64_t(layer_in(l)) * layer_out(l))) != cudaSuccess) return bail(e);
    }
    if ((e = alloc(h, &h->p, h->nparam)) != cudaSuccess || (e = alloc(h, &h->g, h->nparam)) != cudaSuccess ||
        (e = alloc(h, &h->m, h->nparam)) != cudaSuccess || (e = alloc(h, &h->v, h->nparam)) != cudaSuccess ||
        (e = alloc(h, &h->proj, 16)) != cudaSuccess ||
        (e = alloc(h, &h->slices, kMaxSlices * h->nparam)) != cudaSuccess ||
        (e = alloc(h, &h->sums, 4 * int64_t(h->sms) * (kBwdSums + kOut))) != cudaSuccess ||
        (e = alloc(h, &h->partial, 4 * int64_t(h->sms))) != cudaSuccess ||
        (e = alloc(h, &h->Wt, packed_offset_t(0, 0, 0))) != cudaSuccess ||
        (e = alloc(h, &h->loss_dev, 1)) != cudaSuccess ||
        (e = alloc(h, &h->Wp, packed_offset(kLayers - 1, 0, 0))) != cudaSuccess ||
        (e = alloc(h, &h->err.dev, 1)) != cudaSuccess ||
        (e = cudaMallocHost(&h->err.host, sizeof(int))) != cudaSuccess ||
        (e = cudaMallocHost(&h->done, sizeof(int64_t))) != cudaSuccess ||
        (e = cudaMemset(h->err.dev, 0, sizeof(int))) != cudaSuccess)
        return bail(e);
    *h->err.host = 0;
    *h->done = 0;
    if ((e = cudaFuncSetAttribute(k_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_weight_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_forward<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_forward_mma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_forward_mma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaSmem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_forward<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem)) !=
            cudaSuccess)
        return bail(e);
    const int64_t rows = (capacity + kFwdRows - 1) / kFwdRows * kFwdRows;  // whole tiles
    for (int l = 0; l <= kLayers; ++l) {
        const int w = l == 0 ? kIn : (l == kLayers ? kOut : kWidth);
        if ((e = alloc(h, &h->Af[l], rows * w)) != cudaSuccess ||
            (l < kLayers && (e = alloc(h, &h->Ab[l], rows * w)) != cudaSuccess))
            return bail(e);
        if (l < kLayers && (e = alloc(h, &h->dZb[l], rows * layer_out(l))) != cudaSuccess) return bail(e);
    }
    if ((e = cudaMemcpy(h->proj, proj, 16 * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemset(h->p, 0, sizeof(float) * h->nparam)) != cudaSuccess ||
        (e = cudaMemset(h->m, 0, sizeof(float) * h->nparam)) != cudaSuccess ||
        (e = cudaMemset(h->v, 0, sizeof(float) * h->nparam)) != cudaSuccess)
        return bail(e);
    *out = h;
    return LSKUM_OK;
}

void lskum_mlp_destroy(lskum_mlp* h) {
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    for (void* p : h->allocs) cudaFree(p);
    cudaFreeHost(h->err.host);
    cudaFreeHost(h->done);
    cudaStreamDestroy(h->own_stream);
    delete h;
}

int lskum_mlp_set_params(lskum_mlp* h, const float* params, int64_t n) {
    if (!h || !params || n != h->nparam) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_set_params: size");
    MLP_CUDA(cudaMemcpyAsync(h->p, params, sizeof(float) * n, cudaMemcpyHostToDevice, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->m, 0, sizeof(float) * n, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->v, 0, sizeof(float) * n, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->err.dev, 0, sizeof(int), h->stream));  // new parameters: earlier steps no longer count
    MLP_CUDA((k_weights_bf16<<<dim3(blocks(int64_t(kWidth) * kWidth, 256), kLayers), 256, 0, h->stream>>>(h->p, h->L,
                                                                                                      h->Wp, h->Wt),
              cudaGetLastError()));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    *h->err.host = 0;
    *h->done = 0;
    h->step = 0;
    return LSKUM_OK;
}

int lskum_mlp_get_params(lskum_mlp* h, float* params, int64_t n) {
    if (!h || !params || n != h->nparam) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_get_params: size");
    MLP_CUDA(cudaMemcpyAsync(params, h->p, sizeof(float) * n, cudaMemcpyDeviceToHost, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LSKUM_OK;
}

int lskum_mlp_features(lskum_mlp* h, const float* raw, int64_t n, float* feat) {
    if (!h || !raw || !feat) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_features: null");
    if (n < 1) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_features: n < 1");
    MLP_CUDA((k_features<<<blocks(n, 256), 256, 0, h->stream>>>(raw, n, h->proj, feat), cudaGetLastError()));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LSKUM_OK;
}

int lskum_mlp_predict(lskum_mlp* h, const float* feat, int64_t n, float* out) {
    if (!h || !feat || !out) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_predict: null");
    int rc = check_n(h, n);
    if (rc) return rc;
    float* to = reinterpret_cast<uintptr_t>(out) & 15 ? h->Af[kLayers] : out;  // 16-byte stores
    const float* f = nullptr;
    if ((rc = stage_features(h, feat, n, to, &f)) || (rc = forward(h, f, n, to, false))) return rc;
    if (to != out)
        MLP_CUDA(cudaMemcpyAsync(out, to, sizeof(float) * n * kOut, cudaMemcpyDeviceToDevice, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return check_passes(h);
}

int lskum_mlp_gradients(lskum_mlp* h, const float* feat, const float* target, int64_t n, float* grads,
                        double* loss) {
    if (!h || !feat || !target) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_gradients: null");
    int rc = check_n(h, n);
    if (rc) return rc;
    const float* f = nullptr;
    if ((rc = stage_features(h, feat, n, nullptr, &f)) || (rc = forward(h, f, n, h->Af[kLayers], true)) ||
        (rc = backward(h, target, n)))
        return rc;
    if (grads) MLP_CUDA(cudaMemcpyAsync(grads, h->g, sizeof(float) * h->nparam, cudaMemcpyDeviceToHost, h->stream));
    if (loss) MLP_CUDA(cudaMemcpyAsync(loss, h->loss_dev, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return check_passes(h);
}

int lskum_mlp_train_step(lskum_mlp* h, const float* feat, const float* target, int64_t n, float lr,
                         double* loss) {
    if (!h || !feat || !target || !(lr > 0.f)) return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_train_step: argument");
    int rc = check_n(h, n);
    if (rc) return rc;
    const float* f = nullptr;
    if ((rc = stage_features(h, feat, n, nullptr, &f)) || (rc = forward(h, f, n, h->Af[kLayers], true)) ||
        (rc = backward(h, target, n)))
        return rc;
    h->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f / (1.f - powf(b1, float(h->step)));
    const float c2 = 1.f / (1.f - powf(b2, float(h->step)));
    MLP_CUDA((k_adam<<<blocks(h->nparam, 256), 256, 0, h->stream>>>(h->p, h->g, h->m, h->v, h->nparam, lr, b1, b2,
                                                                     1e-8f, c1, c2, h->err.dev, h->step, h->done),
              cudaGetLastError()));
    MLP_CUDA((k_weights_bf16<<<dim3(blocks(int64_t(kWidth) * kWidth, 256), kLayers), 256, 0, h->stream>>>(h->p, h->L,
                                                                                                      h->Wp, h->Wt),
              cudaGetLastError()));
    if (loss) {
        MLP_CUDA(cudaMemcpyAsync(loss, h->loss_dev, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
        MLP_CUDA(cudaStreamSynchronize(h->stream));
        return check_passes(h);
    }
    return LSKUM_OK;
}

int lskum_mlp_sync(lskum_mlp* h) {
    if (!h) return fail(LSKUM_ERR_INVALID_ARG, "null");
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return check_passes(h);
}

int lskum_mlp_set_gemm(lskum_mlp* h, int path) {
    if (!h || (path != LSKUM_MLP_GEMM_MMA_SYNC && path != LSKUM_MLP_GEMM_TCGEN05))
        return fail(LSKUM_ERR_INVALID_ARG, "lskum_mlp_set_gemm: unknown path");
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    h->gemm_path = path;
    return LSKUM_OK;
}

int lskum_mlp_set_stream(lskum_mlp* h, void* stream) {
    if (!h) return fail(LSKUM_ERR_INVALID_ARG, "null");
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    h->stream = stream ? static_cast<cudaStream_t>(stream) : h->own_stream;
    return LSKUM_OK;
}

}  // extern "C"

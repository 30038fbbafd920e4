// ENCODE of whole prompts on the tensor cores (the step before the decode path: building the
// signature cache of Section 4.1 "Implementation" for n tokens at once; the paper names these
// matrix multiplications as the latency bottleneck at short contexts, Section 5.2).
//
// F = 128 -> 128 -> 128 -> 32 (Eq. 2) for a tile of 128 tokens is a chain of three small GEMMs.
// A warp owns 16 tokens and keeps their activations in registers from layer to layer: the fp32
// accumulator fragment of mma.m16n8k16 has exactly the layout of the next layer's A fragment, so
// nothing but the input tile and the weights ever touches shared memory.  Inputs and weights are
// bf16 and therefore exact operands; the fp32 hidden activations are fed to the next layer as a
// bf16 pair hi + lo (hi = round(h), lo = round(h - hi): 16 significant bits), two mma per product.
//
// Numerics: the sums are formed by the tensor cores in their own order and from 16-bit
// activations, not by the fp32 fused-multiply-add chain that defines the decode-step signatures.
// A bit can therefore differ from the chain's wherever the last layer's output is within ~1e-5 of
// zero; everywhere else the signatures are identical (the parity tests bound this by the margin of
// the exact output).  The chain-exact kernels in ha_encode.cu remain the reference for the decode
// step and are what ha_encode uses.
#include "ha_attn_dev.cuh"
#include "ha_encode_dev.cuh"

#include <cstring>
#include <type_traits>
#include <cuda.h>   // CUtensorMap (types only; the encoder is fetched through the runtime)

namespace ha {

constexpr int kTcTile = 128;                       // tokens per tile
constexpr int kTcThreads = 256;                    // 8 warps x 16 tokens
constexpr int kTcRow = kD * 2 + 16;                // padded row of the token tile and of W1 / W2 (bytes)
constexpr int kTcRow3 = kBits * 2 + 16;            // padded row of W3 (bytes)
constexpr int kTcW12Bytes = kD * kTcRow;           // 34816
constexpr int kTcW3Bytes = kHid * kTcRow3;         // 10240
constexpr int kTcXBytes = kTcTile * kTcRow;        // 34816
constexpr int kTcSmem = 2 * kTcW12Bytes + kTcW3Bytes + 2 * kTcXBytes;   // 149504

// hi / lo bf16 pair of two fp32 values after ReLU, packed for an A fragment register
__device__ __forceinline__ void split_relu(float v0, float v1, uint32_t &hi, uint32_t &lo) {
    v0 = fmaxf(v0, 0.0f);
    v1 = fmaxf(v1, 0.0f);
    const float h0 = bf16_round(v0), h1 = bf16_round(v1);
    hi = pack_bf16(h0, h1);
    lo = pack_bf16(v0 - h0, v1 - h1);
}

__global__ void __launch_bounds__(kTcThreads, 1) encode_tc_kernel(MapView map, int heads_per_kv, TensorView x, int B,
                                                                 int H, int T, uint32_t *__restrict__ codes,
                                                                 long long c_sb, long long c_sh) {
    extern __shared__ __align__(128) unsigned char tsm[];
    unsigned char *sW1 = tsm, *sW2 = sW1 + kTcW12Bytes, *sW3 = sW2 + kTcW12Bytes, *sX = sW3 + kTcW3Bytes;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, c = lane & 3;
    const int tiles_per_row = (T + kTcTile - 1) / kTcTile;
    const long long n_work = (long long)H * B * tiles_per_row;   // order: head-major, so that a CTA keeps its weights
    // contiguous range of work items per CTA
    const long long w_lo = n_work * blockIdx.x / gridDim.x, w_hi = n_work * (blockIdx.x + 1) / gridDim.x;
    if (w_lo >= w_hi) return;

    auto decode = [&](long long w, int &h, int &b, int &t0) {
        const long long per_head = (long long)B * tiles_per_row;
        h = (int)(w / per_head);
        const long long r = w - (long long)h * per_head;
        b = (int)(r / tiles_per_row);
        t0 = (int)(r - (long long)b * tiles_per_row) * kTcTile;
    };
    auto load_x = [&](long long w, int buf) {   // 128 rows x 16 chunks of 16 bytes; rows past T are zero-filled
        int h, b, t0;
        decode(w, h, b, t0);
        const unsigned char *src = reinterpret_cast<const unsigned char *>(x.ptr + (long long)b * x.sb + (long long)h * x.sh);
        const uint32_t dst = smem_u32(sX + buf * kTcXBytes);
#pragma unroll
        for (int i = 0; i < kTcTile * 16 / kTcThreads; ++i) {
            const int e = tid + i * kTcThreads, row = e >> 4, ch = e & 15;
            const bool ok = t0 + row < T;
            cp_async16(dst + row * kTcRow + ch * 16, src + (long long)(ok ? t0 + row : 0) * x.sn * 2 + ch * 16, ok ? 16u : 0u);
        }
    };
    auto load_weights = [&](int net) {
        const unsigned char *g1 = reinterpret_cast<const unsigned char *>(map.w1 + (size_t)net * kD * kHid);
        const unsigned char *g2 = reinterpret_cast<const unsigned char *>(map.w2 + (size_t)net * kHid * kHid);
        const unsigned char *g3 = reinterpret_cast<const unsigned char *>(map.w3 + (size_t)net * kHid * kBits);
        for (int e = tid; e < kD * 16; e += kTcThreads) {
            cp_async16(smem_u32(sW1) + (e >> 4) * kTcRow + (e & 15) * 16, g1 + (size_t)e * 16, 16u);
            cp_async16(smem_u32(sW2) + (e >> 4) * kTcRow + (e & 15) * 16, g2 + (size_t)e * 16, 16u);
        }
        for (int e = tid; e < kHid * 4; e += kTcThreads)
            cp_async16(smem_u32(sW3) + (e >> 2) * kTcRow3 + (e & 3) * 16, g3 + (size_t)e * 16, 16u);
    };

    // ldmatrix lane offsets.  A (token tile, row-major): matrix j = lane/8 -> rows (j&1)*8 + lane%8, k block j/2.
    const uint32_t a_off = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * kTcRow + (lane >> 4) * 16);
    // B (weights [k][n], transposed on load): matrix j -> k rows (j&1)*8 + lane%8, n block j/2.
    const uint32_t b_off12 = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * kTcRow + (lane >> 4) * 16);
    const uint32_t b_off3 = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * kTcRow3 + (lane >> 4) * 16);

    int cur_net = -1;
    load_x(w_lo, 0);
    cp_async_commit();
    int buf = 0;
    for (long long w = w_lo; w < w_hi; ++w, buf ^= 1) {
        int h, b, t0;
        decode(w, h, b, t0);
        const int net = h / heads_per_kv;
        if (net != cur_net) {   // CTA-uniform; the previous tile's math is behind the barrier at the end of the loop
            load_weights(net);
            cur_net = net;
        }
        cp_async_commit();      // group of the weights (empty when they stay)
        if (w + 1 < w_hi) load_x(w + 1, buf ^ 1);
        cp_async_commit();      // group of the next tile (empty after the last one)
        cp_async_wait<1>();     // everything but the next tile has landed: this tile and the weights
        __syncthreads();

        const float *bias1 = map.b1 ? map.b1 + net * kHid : nullptr;
        const float *bias2 = map.b2 ? map.b2 + net * kHid : nullptr;
        const float *bias3 = map.b3 ? map.b3 + net * kBits : nullptr;
        const uint32_t xs = smem_u32(sX + buf * kTcXBytes) + warp * 16 * kTcRow + a_off;

        // ---- layer 1: acc1[nt] = bias + X W1, n tile nt covers outputs 8 nt .. 8 nt + 7
        float acc1[16][4];
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
            const float b0 = bias1 ? __ldg(bias1 + 8 * nt + 2 * c) : 0.0f, b1 = bias1 ? __ldg(bias1 + 8 * nt + 2 * c + 1) : 0.0f;
            acc1[nt][0] = b0; acc1[nt][1] = b1; acc1[nt][2] = b0; acc1[nt][3] = b1;
        }
#pragma unroll
        for (int kt = 0; kt < 8; ++kt) {
            uint32_t a[4];
            ldmatrix_x4(a, xs + kt * 32);
#pragma unroll
            for (int np = 0; np < 8; ++np) {
                uint32_t bw[4];
                ldmatrix_x4_trans(bw, smem_u32(sW1) + kt * 16 * kTcRow + np * 32 + b_off12);
                mma_bf16_16816(acc1[2 * np], a[0], a[1], a[2], a[3], bw[0], bw[1]);
                mma_bf16_16816(acc1[2 * np + 1], a[0], a[1], a[2], a[3], bw[2], bw[3]);
            }
        }
        // ---- layer 2: A fragments straight from acc1 (ReLU, hi + lo)
        float acc2[16][4];
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
            const float b0 = bias2 ? __ldg(bias2 + 8 * nt + 2 * c) : 0.0f, b1 = bias2 ? __ldg(bias2 + 8 * nt + 2 * c + 1) : 0.0f;
            acc2[nt][0] = b0; acc2[nt][1] = b1; acc2[nt][2] = b0; acc2[nt][3] = b1;
        }
#pragma unroll
        for (int kt = 0; kt < 8; ++kt) {
            uint32_t ah[4], al[4];
            split_relu(acc1[2 * kt][0], acc1[2 * kt][1], ah[0], al[0]);
            split_relu(acc1[2 * kt][2], acc1[2 * kt][3], ah[1], al[1]);
            split_relu(acc1[2 * kt + 1][0], acc1[2 * kt + 1][1], ah[2], al[2]);
            split_relu(acc1[2 * kt + 1][2], acc1[2 * kt + 1][3], ah[3], al[3]);
#pragma unroll
            for (int np = 0; np < 8; ++np) {
                uint32_t bw[4];
                ldmatrix_x4_trans(bw, smem_u32(sW2) + kt * 16 * kTcRow + np * 32 + b_off12);
                mma_bf16_16816(acc2[2 * np], ah[0], ah[1], ah[2], ah[3], bw[0], bw[1]);
                mma_bf16_16816(acc2[2 * np], al[0], al[1], al[2], al[3], bw[0], bw[1]);
                mma_bf16_16816(acc2[2 * np + 1], ah[0], ah[1], ah[2], ah[3], bw[2], bw[3]);
                mma_bf16_16816(acc2[2 * np + 1], al[0], al[1], al[2], al[3], bw[2], bw[3]);
            }
        }
        // ---- layer 3: 32 outputs
        float acc3[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float b0 = bias3 ? __ldg(bias3 + 8 * nt + 2 * c) : 0.0f, b1 = bias3 ? __ldg(bias3 + 8 * nt + 2 * c + 1) : 0.0f;
            acc3[nt][0] = b0; acc3[nt][1] = b1; acc3[nt][2] = b0; acc3[nt][3] = b1;
        }
#pragma unroll
        for (int kt = 0; kt < 8; ++kt) {
            uint32_t ah[4], al[4];
            split_relu(acc2[2 * kt][0], acc2[2 * kt][1], ah[0], al[0]);
            split_relu(acc2[2 * kt][2], acc2[2 * kt][3], ah[1], al[1]);
            split_relu(acc2[2 * kt + 1][0], acc2[2 * kt + 1][1], ah[2], al[2]);
            split_relu(acc2[2 * kt + 1][2], acc2[2 * kt + 1][3], ah[3], al[3]);
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                uint32_t bw[4];
                ldmatrix_x4_trans(bw, smem_u32(sW3) + kt * 16 * kTcRow3 + np * 32 + b_off3);
                mma_bf16_16816(acc3[2 * np], ah[0], ah[1], ah[2], ah[3], bw[0], bw[1]);
                mma_bf16_16816(acc3[2 * np], al[0], al[1], al[2], al[3], bw[0], bw[1]);
                mma_bf16_16816(acc3[2 * np + 1], ah[0], ah[1], ah[2], ah[3], bw[2], bw[3]);
                mma_bf16_16816(acc3[2 * np + 1], al[0], al[1], al[2], al[3], bw[2], bw[3]);
            }
        }
        // ---- sign bits: this lane holds outputs 8 nt + 2c, 8 nt + 2c + 1 of rows g and g + 8
        uint32_t m_lo = 0u, m_hi = 0u;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int bit = 8 * nt + 2 * c;
            m_lo |= (acc3[nt][0] > 0.0f ? 1u : 0u) << bit;
            m_lo |= (acc3[nt][1] > 0.0f ? 1u : 0u) << (bit + 1);
            m_hi |= (acc3[nt][2] > 0.0f ? 1u : 0u) << bit;
            m_hi |= (acc3[nt][3] > 0.0f ? 1u : 0u) << (bit + 1);
        }
        m_lo |= __shfl_xor_sync(0xffffffffu, m_lo, 1);
        m_lo |= __shfl_xor_sync(0xffffffffu, m_lo, 2);
        m_hi |= __shfl_xor_sync(0xffffffffu, m_hi, 1);
        m_hi |= __shfl_xor_sync(0xffffffffu, m_hi, 2);
        if (c == 0) {
            uint32_t *cb = codes + (long long)b * c_sb + (long long)h * c_sh + t0 + warp * 16;
            if (t0 + warp * 16 + g < T) cb[g] = m_lo;
            if (t0 + warp * 16 + g + 8 < T) cb[g + 8] = m_hi;
        }
        __syncthreads();   // every warp is done with this token buffer (and these weights) before they are overwritten
    }
}

cudaError_t launch_encode_tc(const MapView &map, int heads_per_kv, TensorView x, int B, int H, int T, uint32_t *codes,
                             long long c_sb, long long c_sh, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(encode_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
    if (e != cudaSuccess) return e;
    const long long n_work = (long long)H * B * ((T + kTcTile - 1) / kTcTile);
    if (n_work <= 0) return cudaSuccess;
    const int grid = (int)((n_work < sm_count()) ? n_work : sm_count());
    encode_tc_kernel<<<grid, kTcThreads, kTcSmem, st>>>(map, heads_per_kv, x, B, H, T, codes, c_sb, c_sh);
    count_launch();
    return cudaGetLastError();
}


// ------------------------------------------------------------------ tcgen05 version
//
// The same chain of three GEMMs on the fifth-generation tensor cores.  A tile of 128 tokens is
// M = 128 rows = the 128 lanes of tensor memory; threads r, r + 128, r + 256 and r + 384 convert row r.
//   layer 1  D[128 x 128] = X W1 + b1   A = token tile in shared memory (K-major core matrices),
//                                       B = W1 in shared memory (N-major core matrices), 8 x K16;
//                                       the bias is one more K16 step: A = a constant tile whose
//                                       rows are (1, 1, 0, ...), B = two rows holding b1 as a bf16
//                                       pair hi + lo
//   epilogue threads read their quarter of a row of D (tcgen05.ld), apply ReLU, split into a bf16 pair hi + lo
//            (cvt.rn.bf16x2) and write both to tensor memory as the next A operand (tcgen05.st)
//   layer 2  D = A_hi W2 + A_lo W2 + b2  A from tensor memory, 16 x K16 + the bias step
//   layer 3  D[128 x 32] likewise; the epilogue packs the 32 sign bits of a row into its code.
// Activations never leave tensor memory and registers.
// Bound: the tensor pipe (43 MMAs of 64 cycles or less per tile, 1.16 us), if the hand-offs of a tile (MMAs -> mbarrier ->
// tcgen05.ld -> split -> tcgen05.st -> mbarrier -> next layer's MMAs) stay off its path.  So:
//  * two tiles (groups A and B) are in flight, half a tile apart, each with a warp of its own that issues its MMAs and its TMA;
//  * all 16 other warps convert every layer of either tile together, in the fixed order A1 B2 A2 B3 B1' A3, so that a conversion
//    takes half as long as it would by the eight warps of a group and runs under the other tile's MMAs;
//  * a tile has two regions of 128 tensor-memory columns and the hi / lo pairs overwrite the accumulators they come from, 32
//    columns by 32 columns: layer 1 fills P, layer 2 reads P and fills Q, layer 3 reads Q and puts its 32 columns into P, the
//    next tile starts in Q.  A tile never waits for the sign bits of the one before;
//  * layers 2 and 3 are issued in halves of 64 inputs: they start when half of the inputs are converted.
// Measured, 8 heads x 32768 keys: 36.9 us under ncu (523 TFLOP/s of algorithmic work) against 50.5 us with the MMAs issued by a thread of
// the converting warps and eight warps per tile.  What is left is the chain of hand-offs of two tiles in flight (6600 cycles per
// pair of tiles, 4000 of them with the tensor pipe busy); a third tile does not fit tensor memory.  The operands' swizzle made
// no difference by itself: an MMA of 128 x 128 x 16 takes 65 cycles either way when nothing else runs.
// A CTA stays with one network: its weights are loaded once.  Every wait is bounded: on a timeout the waiter raises
// HA_DEV_TIMEOUT in the status word, every role stops, and the CTA frees its tensor memory and returns.

constexpr int kU_Convert = 512;                   // four threads per token row: each converts a quarter of the columns
constexpr int kU_Threads = kU_Convert + 64;       // and one issuing warp per group
// Shared-memory operands.  Token tile (A, K-major) and W1, W2 (B, N-major) in the 128-byte swizzle:
//   token tile: two halves of 64 inputs, each 128 rows of 128 bytes;
//   W1, W2:     two halves of 64 outputs, each kU_WRows rows (inputs; then the bias step) of 128 bytes;
// 16-byte piece c of a row r lies at c ^ (r % 8).  W3 and the tile of ones stay in unswizzled 8 x 16-byte core matrices.
constexpr int kU_WRows = kD + 16;                 // 128 inputs and the 16 rows of the bias step
constexpr int kU_WHalf = kU_WRows * 128;          // 18432
constexpr int kU_WBytes = 2 * kU_WHalf;           // 36864
constexpr int kU_W3Bytes = (kD / 8 + 2) * 512;    // 9216: k-groups of 8 rows x 4 n-blocks x (8 x 16 B)
constexpr int kU_OnesBytes = 4096;                // [128 rows x 16 k] tile of (1, 1, 0, ...) rows
constexpr int kU_XHalf = kTcTile * 128;           // 16384
constexpr int kU_XBytes = 2 * kU_XHalf;           // 32768
// token tiles and W1 / W2 start on 1024-byte boundaries: the order is X, W1, W2, ones, W3
constexpr int kU_OffX = 0, kU_OffW1 = 4 * kU_XBytes, kU_OffW2 = kU_OffW1 + kU_WBytes, kU_OffOnes = kU_OffW2 + kU_WBytes,
              kU_OffW3 = kU_OffOnes + kU_OnesBytes;
constexpr int kU_Smem = kU_OffW3 + kU_W3Bytes;    // 218112
static_assert(kU_WHalf % 1024 == 0 && kU_OffW2 % 1024 == 0 && kU_OffW3 % 1024 == 0, "swizzle atoms are 1024 bytes");
constexpr uint32_t kU_TmemCols = 512;
constexpr uint32_t kU_SlotCols = 256, kU_Region = 128;   // columns of a group: two regions

// 64-bit shared-memory matrix descriptor, no swizzle: start address, leading and stride byte offsets
// in 16-byte units, descriptor version 1 (bits 46-47), layout type 0 (bits 61-63).
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((smem_addr >> 4) & 0x3fffu) | ((uint64_t)((lbo_bytes >> 4) & 0x3fffu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3fffu) << 32) | (1ull << 46);
}
// the same with the 128-byte swizzle (layout type 2); the swizzle atom is 8 rows of 128 bytes
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return umma_desc(smem_addr, lbo_bytes, sbo_bytes) | (2ull << 61);
}
// 32-bit instruction descriptor of kind::f16: fp32 accumulate (bits 4-5 = 1), A and B bf16 (bits 7-9 and
// 10-12 = 1), A K-major (bit 15 = 0), B N-major (bit 16 = 1), N / 8 in bits 17-22, M / 16 in bits 24-28.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// one lane of a converged warp: unlike a test of the lane number it lets the compiler keep the operands of the instructions
// behind it in uniform registers
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0u;
}
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 32 consecutive 32-bit columns of this thread's lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
                   "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
                   "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
                 ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                   "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }

// ReLU + split of two fp32 values into packed bf16 pairs: hi = round(max(v, 0)), lo = round(max(v, 0) - hi);
// the remainder keeps its sign (hi may have been rounded up).  Low half = first value.
__device__ __forceinline__ void relu_split_pair(float v0, float v1, uint32_t &hi, uint32_t &lo) {
    v0 = fmaxf(v0, 0.0f);
    v1 = fmaxf(v1, 0.0f);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(v1), "f"(v0));
    float r0, r1;   // both differences in one instruction
    asm("{\n\t.reg .b64 v, h, r;\n\tmov.b64 v, {%2, %3};\n\tmov.b64 h, {%4, %5};\n\tsub.rn.f32x2 r, v, h;\n\tmov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r0), "=f"(r1) : "f"(v0), "f"(v1), "f"(__uint_as_float(hi << 16)), "f"(__uint_as_float(hi & 0xffff0000u)));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(r1), "f"(r0));
}

// A whole token tile through the tensor map of x seen as [B][H][2 halves][T][64]: the box of 64 x 128 x 2 elements lands half
// after half, each as 128 rows of 128 bytes in the 128-byte swizzle.  One instruction per tile.
__device__ __forceinline__ void tma_load_tile(uint32_t dst, const CUtensorMap *tmap, int t0, int h, int b, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                 ::"r"(dst), "l"(tmap), "r"(0), "r"(t0), "r"(0), "r"(h), "r"(b), "r"(bar) : "memory");
}

// kTma: token tiles arrive through TMA (a group's issuing warp issues one box copy and the tile's mbarrier
// counts the bytes); otherwise the converting threads copy 16-byte pieces with cp.async.
template <bool kTma>
__global__ void __launch_bounds__(kU_Threads, 1) encode_umma_kernel(const __grid_constant__ CUtensorMap tmap, MapView map,
                                                                   int heads_per_kv, TensorView x, int B, int H, int T,
                                                                   int ctas_per_net, uint32_t *__restrict__ codes,
                                                                   long long c_sb, long long c_sh,
                                                                   uint32_t *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char usm[];
    unsigned char *sX = usm + kU_OffX, *sW1 = usm + kU_OffW1, *sW2 = usm + kU_OffW2, *sW3 = usm + kU_OffW3, *sOnes = usm + kU_OffOnes;
    __shared__ __align__(8) unsigned long long s_xbar[2][2];   // [group][buffer]: a token tile has landed
    __shared__ __align__(8) unsigned long long s_dbar[2];      // [group]: a hidden layer is summed
    __shared__ __align__(8) unsigned long long s_abar[2][2];   // [group][half]: 64 columns of it are converted (8 warps arrive)
    __shared__ __align__(8) unsigned long long s_obar[2];      // [group]: the 32 outputs are summed
    __shared__ __align__(8) unsigned long long s_start;        // group 0's first hidden layer is converted; completes once
    __shared__ uint32_t s_tmem_base;
    __shared__ volatile int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int row = tid & 127, quarter = tid >> 7;   // thread (row, quarter) converts columns 32 quarter .. 32 quarter + 31 of its row
    const bool issuer = warp >= kU_Convert / 32;
    const int tiles_per_row = (T + kTcTile - 1) / kTcTile;
    const int net = blockIdx.x / ctas_per_net, part = blockIdx.x % ctas_per_net;
    // tiles of this network in the order (head of the network, sequence, tile); this CTA takes a contiguous share
    const long long n_net = (long long)heads_per_kv * B * tiles_per_row;
    const long long w_lo = n_net * part / ctas_per_net, w_hi = n_net * (part + 1) / ctas_per_net;
    if (w_lo >= w_hi) return;

    auto xbuf = [&](int g, int buf) -> uint32_t { return smem_u32(sX + (g * 2 + buf) * kU_XBytes); };
    auto xbar = [&](int g, int buf) -> uint32_t { return smem_u32(&s_xbar[g][buf]); };
    const long long n_cta = w_hi - w_lo;
    auto tiles_of = [&](int g) -> int { return (int)((n_cta + 1 - g) / 2); };   // group g takes tiles w_lo + g, w_lo + g + 2, ...
    // (a network has fewer than 2^32 tiles: 64-bit divisions would cost the issuing thread 1500 cycles per pair of tiles)
    const uint32_t per_head = (uint32_t)B * (uint32_t)tiles_per_row;
    auto decode = [&](long long w, int &h, int &b, int &t0) {
        const uint32_t hh = (uint32_t)w / per_head, r = (uint32_t)w - hh * per_head, bb = r / (uint32_t)tiles_per_row;
        h = net * heads_per_kv + (int)hh;
        b = (int)bb;
        t0 = (int)(r - bb * (uint32_t)tiles_per_row) * kTcTile;
    };
    // token tile by TMA: one box copy; rows past T are filled with zeros by the tensor map
    auto tma_x = [&](int g, long long w, int buf) {
        int h, b, t0;
        decode(w, h, b, t0);
        mbar_expect_tx(xbar(g, buf), kTcTile * kD * 2);
        tma_load_tile(xbuf(g, buf), &tmap, t0, h, b, xbar(g, buf));
    };
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) {
            mbar_init(smem_u32(&s_xbar[0][0]) + 8 * i, kTma ? 1 : kU_Convert);
            mbar_init(smem_u32(&s_abar[0][0]) + 8 * i, 8);
        }
        mbar_init(smem_u32(&s_dbar[0]), 1);
        mbar_init(smem_u32(&s_dbar[1]), 1);
        mbar_init(smem_u32(&s_obar[0]), 1);
        mbar_init(smem_u32(&s_obar[1]), 1);
        mbar_init(smem_u32(&s_start), kU_Convert / 32);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    __syncwarp();
    // ---- weights, the bias rows k = 128 (hi) and 129 (lo) behind them, and the constant tile of ones
    {
        const unsigned char *g1 = reinterpret_cast<const unsigned char *>(map.w1 + (size_t)net * kD * kHid);
        const unsigned char *g2 = reinterpret_cast<const unsigned char *>(map.w2 + (size_t)net * kHid * kHid);
        const unsigned char *g3 = reinterpret_cast<const unsigned char *>(map.w3 + (size_t)net * kHid * kBits);
        for (int e = tid; e < kD * 16; e += kU_Threads) {   // 16 pieces of 8 outputs per row k
            const int k = e >> 4, nb = e & 15;
            const uint32_t off = (nb >> 3) * kU_WHalf + k * 128 + (((nb & 7) ^ (k & 7)) << 4);
            cp_async16(smem_u32(sW1) + off, g1 + (size_t)e * 16, 16u);
            cp_async16(smem_u32(sW2) + off, g2 + (size_t)e * 16, 16u);
        }
        // W3, N-major core matrices: element (k, n) at (k/8) * 512 + (n/8) * 128 + (k%8) * 16 + (n%8) * 2
        for (int e = tid; e < kHid * 4; e += kU_Threads) {  // 4 pieces per row k
            const int k = e >> 2, nb = e & 3;
            cp_async16(smem_u32(sW3) + (k >> 3) * 512 + nb * 128 + (k & 7) * 16, g3 + (size_t)e * 16, 16u);
        }
        cp_async_commit();
        // Nothing of the kernel in front is read, and nothing written, before this point: its end overlaps the launch, the barriers
        // and the fetch of the weights (us per call, 40 calls back to back over four inputs, 8 heads of 32768 keys 34.9 -> 33.2, of
        // 8192 16.5 -> 13.9, of 256 10.3 -> 9.1; the kernel by itself takes what it took).  The kernels behind start when this one has
        // ended, as they read signatures before their own wait.  The tensor memory is allocated behind the wait: a kernel in front may
        // still want it for itself.
        pdl_wait();
        if (warp == 0) {   // one warp allocates the tensor memory and passes the allocation right on
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(kU_TmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (kTma && tid == 0) {   // the first tiles are on their way while the biases are laid out
            tma_x(0, w_lo, 0);
            if (tiles_of(1) > 0) tma_x(1, w_lo + 1, 0);
        }
        __syncwarp();
        // rows 128 .. 143 (W3: k-groups 16 and 17): zero, then the bias pair in the first two
        for (int i = tid; i < 2048 / 16; i += kU_Threads) {
#pragma unroll
            for (int nh = 0; nh < 2; ++nh) {
                reinterpret_cast<uint4 *>(sW1 + nh * kU_WHalf + kD * 128)[i] = make_uint4(0u, 0u, 0u, 0u);
                reinterpret_cast<uint4 *>(sW2 + nh * kU_WHalf + kD * 128)[i] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        for (int i = tid; i < kU_OnesBytes / 16; i += kU_Threads) reinterpret_cast<uint4 *>(sOnes)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = tid; i < 1024 / 16; i += kU_Threads) reinterpret_cast<uint4 *>(sW3 + 16 * 512)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        auto bias_pair = [&](const float *bias, int n, uint16_t &hi, uint16_t &lo) {
            const float v = bias ? __ldg(bias + n) : 0.0f;
            const float h = bf16_round(v);
            const __nv_bfloat16 bh = __float2bfloat16_rn(h), bl = __float2bfloat16_rn(v - h);
            hi = *reinterpret_cast<const uint16_t *>(&bh);
            lo = *reinterpret_cast<const uint16_t *>(&bl);
        };
        auto put_bias = [&](unsigned char *w, const float *bias, int n) {   // rows 128 and 129 are rows 0 and 1 of their swizzle atom
            uint16_t hi, lo;
            bias_pair(bias, n, hi, lo);
            unsigned char *p = w + (n >> 6) * kU_WHalf + kD * 128 + (n & 7) * 2;
            const int c = (n >> 3) & 7;
            *reinterpret_cast<uint16_t *>(p + (c << 4)) = hi;
            *reinterpret_cast<uint16_t *>(p + 128 + ((c ^ 1) << 4)) = lo;
        };
        if (tid < kHid) {
            put_bias(sW1, map.b1 ? map.b1 + net * kHid : nullptr, tid);
            put_bias(sW2, map.b2 ? map.b2 + net * kHid : nullptr, tid);
            // ones tile, K-major: row r at (r/8) * 128 + (r%8) * 16 of k-chunk 0 holds (1, 1, 0, 0, 0, 0, 0, 0)
            *reinterpret_cast<uint32_t *>(sOnes + (tid >> 3) * 128 + (tid & 7) * 16) = 0x3f803f80u;
        }
        if (tid < kBits) {
            uint16_t hi, lo;
            bias_pair(map.b3 ? map.b3 + net * kBits : nullptr, tid, hi, lo);
            unsigned char *p = sW3 + 16 * 512 + (tid >> 3) * 128 + (tid & 7) * 2;
            *reinterpret_cast<uint16_t *>(p) = hi;
            *reinterpret_cast<uint16_t *>(p + 16) = lo;
        }
    }
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // ordinary writes -> visible to the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem_base;
    // by the threads: a half-warp copies one 256-byte row
    auto copy_x = [&](int g, long long w, int buf) {
        int h, b, t0;
        decode(w, h, b, t0);
        const uint32_t dst = xbuf(g, buf);
        const unsigned char *src = reinterpret_cast<const unsigned char *>(x.ptr + (long long)b * x.sb + (long long)h * x.sh);
#pragma unroll
        for (int i = 0; i < kTcTile * 16 / kU_Convert; ++i) {
            const int e = tid + i * kU_Convert, r = e >> 4, ch = e & 15;
            const bool ok = t0 + r < T;
            cp_async16(dst + (ch >> 3) * kU_XHalf + r * 128 + (((ch & 7) ^ (r & 7)) << 4),
                       src + (long long)(ok ? t0 + r : 0) * x.sn * 2 + ch * 16, ok ? 16u : 0u);
        }
        cp_async_commit();
    };
    auto copied_x = [&](int g, int buf) {   // this thread's pieces have landed and the tensor cores may see them
        cp_async_wait<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(xbar(g, buf));
    };
    // a bounded wait that fails soon after another role has given up
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
        if (mbar_test(bar, parity)) return true;
        if (!mbar_wait_parity(bar, parity)) {
            s_fail = 1;
            if (status) atomicOr(status, HA_DEV_TIMEOUT);
            return false;
        }
        return s_fail == 0;
    };
    if (issuer) {
        // The whole warp takes these steps; one elected lane issues.  One warp per group, because what a step costs the issuer
        // is its waits (a satisfied one 80 - 300 cycles), not its MMAs (40 each).
        // (the shuffles tell the compiler that the group and the addresses are the same in every lane: uniform registers)
        const int g = __shfl_sync(0xffffffffu, warp - kU_Convert / 32, 0), n_tiles = tiles_of(g);
        constexpr uint32_t kIdesc128 = umma_idesc(128, 128), kIdesc32 = umma_idesc(128, 32);
        const uint32_t smem0 = smem_u32(usm), cols = __shfl_sync(0xffffffffu, tmem, 0) + g * kU_SlotCols;
        const uint32_t dbar = smem_u32(&s_dbar[g]), abar0 = smem_u32(&s_abar[g][0]), obar = smem_u32(&s_obar[g]);
        const uint64_t ones_desc = umma_desc(smem0 + kU_OffOnes, 2048, 128);
        // ---- layer 1: D = X W1 + b1 (operands from shared memory), one MMA per 16 values of k
        auto layer1 = [&](uint32_t d, int buf) {
            tc_fence_after();
            if (elect_one()) {
                uint64_t ad = umma_desc_sw128(smem0 + kU_OffX + (g * 2 + buf) * kU_XBytes, 16, 1024), bd = umma_desc_sw128(smem0 + kU_OffW1, kU_WHalf, 1024);
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) umma_ss(d, ad + j * (32 >> 4), bd + j * (2048 >> 4), kIdesc128, (kh | j) ? 1u : 0u);
                    ad += kU_XHalf >> 4;
                    bd += 4 * 2048 >> 4;
                }
                umma_ss(d, ones_desc, bd, kIdesc128, 1u);
                umma_commit(dbar);
            }
            __syncwarp();
        };
        // ---- layers 2 and 3: D = A_hi W + A_lo W + b, A from tensor memory; bd: descriptor of the first 16 inputs, step: to the
        // next 16 (constants of the code: every instruction between two MMAs delays the tensor pipe while 16 warps convert).  The A operand of 32 inputs is 32 columns: 16 of hi, 16 of lo.
        auto layer23 = [&](auto third, uint32_t d, uint32_t ar, uint32_t parity, uint32_t done) -> bool {
            constexpr bool k3 = decltype(third)::value;
            constexpr uint32_t step = (k3 ? 1024 : 2048) >> 4, idesc = k3 ? kIdesc32 : kIdesc128;
            const uint64_t bd = k3 ? umma_desc(smem0 + kU_OffW3, 512, 128) : umma_desc_sw128(smem0 + kU_OffW2, kU_WHalf, 1024);
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {   // half `kh` of the inputs is converted
                if (!wait(abar0 + 8 * kh, parity)) return false;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t a = ar + kh * 64;
                    const uint64_t b = bd + (uint64_t)(kh * 4 * step);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint32_t aq = a + (q >> 1) * 32 + (q & 1) * 8;
                        umma_ts(d, aq, b + q * step, idesc, (kh | q) ? 1u : 0u);
                        umma_ts(d, aq + 16, b + q * step, idesc, 1u);
                    }
                    if (kh == 1) {
                        umma_ss(d, ones_desc, b + 4 * step, idesc, 1u);
                        umma_commit(done);
                    }
                }
                __syncwarp();
            }
            return true;
        };
        auto load = [&](int i) {
            if (kTma && i < n_tiles && elect_one()) tma_x(g, w_lo + g + 2LL * i, i & 1);
            __syncwarp();
        };
        // the groups work half a tile apart, or both would multiply and both would convert at the same time: group 1 starts when
        // group 0 has converted its first hidden layer.  The barrier has that one phase: group 0 does not wait for group 1, and a
        // barrier that it completes a second time reads "not complete" again to a warp that looks late.
        bool ok = g == 0 || n_tiles == 0 || wait(smem_u32(&s_start), 0u);
        int i = 0;
        for (; ok && i < n_tiles; ++i) {
            const uint32_t p = cols + (i & 1) * kU_Region, q = cols + ((i & 1) ^ 1) * kU_Region;
            ok = wait(xbar(g, i & 1), (uint32_t)(i >> 1) & 1u);
            if (ok && i > 0) ok = wait(obar, (uint32_t)(i - 1) & 1u);   // region p is what the last tile's layer 3 reads
            if (!ok) break;
            layer1(p, i & 1);
            load(i + 1);   // into the buffer that the last tile's layer 1 read
            ok = layer23(std::false_type{}, q, p, 0u, dbar);
            if (!ok) break;
            ok = layer23(std::true_type{}, p, q, 1u, obar);
            if (!ok) break;
        }
        if (!ok && kTma)   // never seen: give the tiles in flight one more bounded wait before the CTA gives up its memory
            for (int j = i; j <= i + 1 && j < n_tiles; ++j) mbar_wait_parity(xbar(g, j & 1), (uint32_t)(j >> 1) & 1u);
        // the last MMAs are complete before the tensor memory is given back
        if (n_tiles > 0) mbar_wait_parity(obar, (uint32_t)(n_tiles - 1) & 1u);
        __syncwarp();
    } else {
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;   // this warp's 32 lanes (four warps share them)
        auto region = [&](int g, int i) -> uint32_t { return tmem + g * kU_SlotCols + (i & 1) * kU_Region + lanes; };
        // this thread's 32 columns of a region, when layer 1 (phase 0) or 2 (phase 1) of the group's tile is summed: ReLU, hi / lo,
        // in place (32 columns of sums -> 16 of hi and 16 of lo)
        auto convert = [&](int g, uint32_t cols, uint32_t phase) -> bool {
            if (!wait(smem_u32(&s_dbar[g]), phase)) return false;
            tc_fence_after();
            const uint32_t c0 = cols + quarter * 32;
            uint32_t v[32], hi[16], lo[16];
            tmem_ld32(c0, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) relu_split_pair(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]), hi[i], lo[i]);
            tmem_st16(c0, hi);
            tmem_st16(c0 + 16, lo);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive(smem_u32(&s_abar[g][quarter >> 1]));
            return true;
        };
        // the sign bits of tile i of group g, by the quarter g of the threads.  Layer 2 of the group's next tile overwrites the
        // sums, and starts after these threads have converted that tile's layer 1 (both are in the first half of the columns).
        auto sign_bits = [&](int g, int i) -> bool {
            if (!wait(smem_u32(&s_obar[g]), (uint32_t)i & 1u)) return false;
            tc_fence_after();
            uint32_t v[32];
            tmem_ld32(region(g, i), v);
            tmem_wait_ld();
            tc_fence_before();
            uint32_t code = 0u;
#pragma unroll
            for (int o = 0; o < 32; ++o) code |= (__uint_as_float(v[o]) > 0.0f ? 1u : 0u) << o;
            int h, b, t0;
            decode(w_lo + g + 2LL * i, h, b, t0);
            if (t0 + row < T) codes[(long long)b * c_sb + (long long)h * c_sh + t0 + row] = code;
            return true;
        };
        const int na = tiles_of(0), nb = tiles_of(1);
        if (!kTma) {
            for (int g = 0; g < 2; ++g)
                if (tiles_of(g) > 0) { copy_x(g, w_lo + g, 0); copied_x(g, 0); }
        }
        // layer 1 of tile i of group g; without TMA also the copy of the group's next tile, into the buffer that its last layer 1 read
        auto first_layer = [&](int g, int i) -> bool {
            const bool copy = !kTma && i + 1 < tiles_of(g);
            if (copy) copy_x(g, w_lo + g + 2LL * (i + 1), (i + 1) & 1);
            if (!convert(g, region(g, i), 0u)) return false;
            if (g == 0 && i == 0 && (tid & 31) == 0) mbar_arrive(smem_u32(&s_start));
            if (copy) copied_x(g, (i + 1) & 1);
            return true;
        };
        for (int i = 0; i <= na; ++i) {   // na == nb or nb + 1
            const bool a = i < na, b = i > 0 && i - 1 < nb;
            if (a && !first_layer(0, i)) break;
            if (b && !convert(1, region(1, i), 1u)) break;          // layer 2 of tile i - 1 lies in its other region
            if (a && !convert(0, region(0, i + 1), 1u)) break;
            if (b && quarter == 1 && !sign_bits(1, i - 1)) break;   // warp-uniform
            if (i < nb && !first_layer(1, i)) break;
            if (a && quarter == 0 && !sign_bits(0, i)) break;
        }
    }
    cp_async_wait<0>();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem_base), "r"(kU_TmemCols) : "memory");
    }
}

// Tensor map of x [B][H][T][128] (bf16, strides in elements) seen as [B][H][2][T][64], with boxes of
// 64 x 128 x 2 elements; false if the driver entry point is missing or the strides do not fit a tensor map.
static bool make_x_tensor_map(CUtensorMap *tm, TensorView x, int B, int H, int T) {
    typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                 const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
        else
            cudaGetLastError();
        looked = true;
    }
    if (!fn) return false;
    const cuuint64_t dims[5] = {64u, (cuuint64_t)T, 2u, (cuuint64_t)H, (cuuint64_t)B};
    const cuuint64_t strides[4] = {(cuuint64_t)x.sn * 2, 128u, (cuuint64_t)x.sh * 2, (cuuint64_t)x.sb * 2};   // bytes
    const cuuint32_t box[5] = {64u, (cuuint32_t)kTcTile, 2u, 1u, 1u}, estr[5] = {1u, 1u, 1u, 1u, 1u};
    for (int i = 0; i < 4; ++i)
        if (strides[i] == 0 || (strides[i] & 15)) return false;
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<uint16_t *>(x.ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_encode_umma(const MapView &map, int heads_per_kv, TensorView x, int B, int H, int T, uint32_t *codes,
                               long long c_sb, long long c_sh, uint32_t *status, cudaStream_t st) {
    const int n_nets = H / heads_per_kv;
    const long long n_net = (long long)heads_per_kv * B * ((T + kTcTile - 1) / kTcTile);   // tiles per network
    if (n_net <= 0 || n_nets <= 0) return cudaSuccess;
    long long per = sm_count() / n_nets;                 // CTAs per network: a CTA never changes its weights
    if (per < 1) per = 1;
    if (per > (n_net + 1) / 2) per = (n_net + 1) / 2;    // at least two tiles (one per group) for a CTA to be worth it
    if (per < 1) per = 1;
    CUtensorMap tm;
    memset(&tm, 0, sizeof(tm));
    const bool tma = make_x_tensor_map(&tm, x, B, H, T);
    cudaError_t e = tma ? cudaFuncSetAttribute(encode_umma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kU_Smem)
                        : cudaFuncSetAttribute(encode_umma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kU_Smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(n_nets * per));
    e = tma ? launch_pdl(encode_umma_kernel<true>, grid, dim3(kU_Threads), kU_Smem, st, tm, map, heads_per_kv, x, B, H, T, (int)per, codes, c_sb, c_sh, status)
            : launch_pdl(encode_umma_kernel<false>, grid, dim3(kU_Threads), kU_Smem, st, tm, map, heads_per_kv, x, B, H, T, (int)per, codes, c_sb, c_sh, status);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

} // namespace ha

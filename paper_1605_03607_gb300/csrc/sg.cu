// sg.cu -- surrogate hardness model: message-passing network over the Chimera
// coupler graph that predicts log10 TTS (C ABI: sg_* in include/pt.h).
//
// The paper has no surrogate; it is this library's way to spend PT evaluations
// (Sec. II TTS inside Algorithm 1) only on promising coupler moves.  Network:
//   h0_i = X[u_i], e0_e = Jt[idx(J_e)]                      (u: orientation)
//   per layer: m_i = sum_{j in N(i)} relu(Wm [h_j, e_ij] + bm)
//              h_i += relu(Wu [h_i, m_i] + bu)
//              e_ij += relu(We [e_ij, h_i + h_j] + be)        (updated h)
//   readout:   y = w2 . relu(W1 mean_i(h_i) + b1) + b2
// Hidden width 64.  Weights and activations are BF16, accumulation FP32; the
// three per-layer linear maps (K = 128 -> 64 outputs over every message,
// node or edge row), their input gradients and their weight gradients run on
// the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor
// memory).  Gradients are FP32 buffers; master weights and Adam moments are
// FP32.  Every reduction runs in a fixed order (no floating-point atomics), so
// a training step is bit-reproducible.
//
// Bound: memory and L2 traffic of the row-wise data (a batch of 256 C_8 graphs has
// 753,664 message, 131,072 node and 376,832 edge rows of 64; the linear maps need
// 0.13 ms of tensor time), and launch gaps for small batches.  So per layer 3 forward
// and 4 backward kernels, each a linear map with everything around it, and no message
// row in memory.  Measured against one kernel per step with FP32 messages, pre-activations
// and masked gradients in memory (97 launches, 35 now): gradient of 256 C_8 graphs 3.95 ->
// 2.24 ms, of 128 C_4 graphs 1.01 -> 0.59 ms, 64 C_8 predictions 0.42 -> 0.26 ms.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/pt.h"
#include "pt_internal.h"

namespace {

constexpr int HD = 64;      // hidden width
constexpr int KIN = 128;    // input width of every linear map: [64 | 64]
constexpr int MAXDEG = 6;
typedef __nv_bfloat16 bf16;

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ uint32_t pack_bf2(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack_bf2(uint32_t u)
{
    __nv_bfloat162 v = *reinterpret_cast<__nv_bfloat162*>(&u);
    return __bfloat1622float2(v);
}

// Floats of one CTA's weight-gradient partial: dW [64][128] then db [64].
constexpr int WPART = HD * KIN + HD;

// ------------------------------------------- tcgen05 (5th-generation tensor core) GEMMs
// The forward maps Z = X W^T + b (128 rows x K = 128 -> 64 outputs per tile),
// the input gradient dX = dZ W (128 rows x K = 64 -> 64 inputs at a time) and the
// weight gradient dW^T += X^T dZ (K = 128 rows) run on tcgen05.mma with the
// accumulator in tensor memory:
//   * persistent CTAs over 128-row tiles; one thread issues the MMAs and
//     commits them to an mbarrier;
//   * operands in shared memory in the canonical layout without swizzle, built
//     from 8-row x 16-byte core matrices; a descriptor's leading byte offset
//     steps between core matrices along K, its stride byte offset along M or N.
//     With the two the other way round every address would still lie inside the
//     CTA's shared memory;
//   * the weights, pre-packed in that layout (pack_weights_kernel), arrive by
//     one bulk asynchronous copy; gathered rows by 16-byte cp.async;
//   * after the commit each warp reads its 32 accumulator rows (TMEM lanes
//     32w .. 32w+31) with tcgen05.ld, one row per thread, for the epilogue;
//   * every mbarrier wait is bounded: on a timeout the CTA records it in
//     *err, stops taking tiles, frees its tensor memory and returns.
constexpr uint32_t TC_WAIT_LIMIT = 1u << 22;
constexpr int TC_ROWS = 128;
// CTAs of 256 threads: all 8 warps stage a tile; in the epilogue warps w and
// w + 4 read the same 32 tensor-memory lanes (a warp reaches lanes
// 32 (w mod 4) .. + 31) and split the columns, and each warp's stores pass
// through a 4 KB slice of the consumed operand buffer.  The dynamic shared
// memory (forward: A 32 KB + W 16 KB; backward below) bounds the resident CTAs,
// so that their tensor memory (64 columns forward, 128 backward) never exceeds an
// SM's 512 columns; the persistent grids use exactly that many.
constexpr int TC_THREADS = 256;
constexpr int TC_A_FWD = TC_ROWS * KIN * 2;
constexpr int TC_SMEM_FWD = TC_A_FWD + HD * KIN * 2;
constexpr int TC_CTAS_FWD = 4;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of tcgen05.mma: start address, leading and
// stride byte offsets (all >> 4), descriptor version 1 (bits 46-47), no
// swizzle (layout type 0 in bits 61-63), base offset 0.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor, kind::f16: F32 accumulator (bits 4-5 = 1), BF16 A
// and B (bits 7-9, 10-12 = 1), both K-major, N >> 3 in bits 17-22, M >> 4 in
// bits 24-28.
__host__ __device__ constexpr uint32_t tc_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity)
{
    for (uint32_t i = 0; i < TC_WAIT_LIMIT; ++i) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(smem_u32(bar)), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}

// One bulk asynchronous copy global -> shared of `bytes` (a multiple of 16,
// both addresses 16-byte aligned), completing on `bar`.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                 ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
                 : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Epilogue stores of one warp's 32 accumulator rows (lane l holds row l),
// staged through a 4 KB slice of shared memory so that each global store
// instruction writes whole rows: 4 rows x 128 bytes (32 FP32 columns) or 8
// rows x 64 bytes (32 BF16 columns) instead of one 16-byte piece of each of
// 32 rows.  Row l's 16-byte chunk c sits at slot c ^ (l & 7) (FP32) or
// c ^ ((l >> 1) & 3) (BF16) of its row, so neither the row-wise writes nor
// the chunk-wise reads of a warp meet a bank conflict.  flush_* writes the
// staged block: g points at the warp's first row and first column, ld is the
// row pitch in elements, and only rows < nvalid are written.
__device__ __forceinline__ void stage_f32(unsigned char* stage, int lane, int c, float4 v)
{
    *reinterpret_cast<float4*>(stage + lane * 128 + ((c ^ (lane & 7)) << 4)) = v;
}

__device__ __forceinline__ void flush_f32x32(const unsigned char* stage, float* g, int ld, int nvalid, int lane)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int row = k * 4 + (lane >> 3), c = lane & 7;
        const float4 x = *reinterpret_cast<const float4*>(stage + row * 128 + ((c ^ (row & 7)) << 4));
        if (row < nvalid) *reinterpret_cast<float4*>(g + (size_t)row * ld + c * 4) = x;
    }
    __syncwarp();
}

// The same, added to g's rows.
__device__ __forceinline__ void flush_add_f32x32(const unsigned char* stage, float* g, int ld, int nvalid, int lane)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int row = k * 4 + (lane >> 3), c = lane & 7;
        float4 x = *reinterpret_cast<const float4*>(stage + row * 128 + ((c ^ (row & 7)) << 4));
        if (row < nvalid) {
            float4* gp = reinterpret_cast<float4*>(g + (size_t)row * ld + c * 4);
            const float4 o = *gp;
            x.x += o.x;
            x.y += o.y;
            x.z += o.z;
            x.w += o.w;
            *gp = x;
        }
    }
    __syncwarp();
}

// Adds the sums of staged row pairs (2p, 2p + 1), in that order, to row p of g, or
// (set) puts them there (16 pairs x 32 FP32 columns; only pairs < npairs).
__device__ __forceinline__ void flush_pairs_f32x32(const unsigned char* stage, float* g, int ld, int npairs, int lane,
                                                   bool set)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int p = k * 4 + (lane >> 3), c = lane & 7, ra = 2 * p, rb = ra + 1;
        const float4 a = *reinterpret_cast<const float4*>(stage + ra * 128 + ((c ^ (ra & 7)) << 4));
        const float4 b = *reinterpret_cast<const float4*>(stage + rb * 128 + ((c ^ (rb & 7)) << 4));
        if (p < npairs) {
            float4* gp = reinterpret_cast<float4*>(g + (size_t)p * ld + c * 4);
            float4 o = set ? make_float4(0.f, 0.f, 0.f, 0.f) : *gp;
            o.x += a.x + b.x;
            o.y += a.y + b.y;
            o.z += a.z + b.z;
            o.w += a.w + b.w;
            *gp = o;
        }
    }
    __syncwarp();
}

__device__ __forceinline__ void stage_bf16(unsigned char* stage, int lane, int c, uint4 v)
{
    *reinterpret_cast<uint4*>(stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) = v;
}

__device__ __forceinline__ void flush_bf16x32(const unsigned char* stage, bf16* g, int ld, int nvalid, int lane)
{
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int row = k * 8 + (lane >> 2), c = lane & 3;
        const uint4 x = *reinterpret_cast<const uint4*>(stage + row * 64 + ((c ^ ((row >> 1) & 3)) << 4));
        if (row < nvalid) *reinterpret_cast<uint4*>(g + (size_t)row * ld + c * 8) = x;
    }
    __syncwarp();
}

// A 32-column BF16 block packed in 16 words (2 per column pair) through the staging slice.
__device__ __forceinline__ void store_bf16x32(unsigned char* stage, const uint32_t (&w)[16], bf16* g, int ld,
                                              int nvalid, int lane)
{
#pragma unroll
    for (int c = 0; c < 4; ++c) stage_bf16(stage, lane, c, make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]));
    flush_bf16x32(stage, g, ld, nvalid, lane);
}

// Common prologue: tensor memory (ncols columns, warp 0), the two mbarriers,
// and the packed weights (bytes) by one bulk copy.  Returns false (for every
// thread) if the weights did not arrive within the wait limit.
__device__ __forceinline__ bool tc_setup(uint32_t* tmem_sh, uint64_t* bar_w, uint64_t* bar_mma, uint32_t ncols,
                                         void* Ws, const void* Wpk, uint32_t bytes)
{
    const int tid = threadIdx.x;
    if ((tid >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_sh)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(bar_w, 1);
        mbar_init(bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (bytes == 0) return true;
    if (tid == 0) bulk_g2s(Ws, Wpk, bytes, bar_w);
    bool ok = mbar_wait(bar_w, 0);
    if (!ok) ok = mbar_wait(bar_w, 0);         // second bounded wait for the copy still in flight
    return !__syncthreads_or(!ok);
}

__device__ __forceinline__ void tc_teardown(uint32_t tmem, uint32_t ncols, bool failed, int* err)
{
    tc_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    }
    if (failed && threadIdx.x == 0) atomicExch(err, 1);
}

// ------------------------------------------------------------- layer kernels
// Rows of a tile are gathered while they are staged, and everything elementwise
// around a linear map runs in its staging or its epilogue, so that per layer only
// node and edge features (BF16), their gradients (FP32) and one bit per activation
// go through memory:
//   * the backward needs a pre-activation's sign only: the forward keeps it as a
//     bit (z > 0 after rounding to BF16), 8 bytes per row of 64;
//   * messages are computed target by target, 21 nodes of 6 slots per tile, and
//     summed in the epilogue (in the order of the node's slots); their gradient
//     with respect to the source node source by source, the same way;
//   * a map's input gradient and weight gradient share the staged tile.
// Row r of a tile sits in 8-row core matrices: chunk (row group r / 8, column chunk
// of 8) is 8 rows x 16 bytes.  Read along its columns that is a K-major operand,
// read along its rows an MN-major one; only the two descriptor strides differ (the
// leading offset steps along K, the stride offset along M or N), so the dZ tile is
// the A operand of the input gradient and the B operand of the weight gradient.
constexpr int NODE_ROWS = 6, TILE_NODES = TC_ROWS / NODE_ROWS;        // 21 nodes, 126 rows

// z's sign bit of the backward's mask: positive after rounding to BF16 (2^-133 is
// the smallest BF16 number; 2^-134 and below round to zero).
__device__ __forceinline__ uint32_t positive_bf16(float z) { return z > 0x1p-134f ? 1u : 0u; }

// 8 BF16 values (one 16-byte chunk) with the columns whose mask bit is 0 cleared.
__device__ __forceinline__ uint4 mask_bf16x8(uint4 v, uint32_t bits)
{
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] &= ((bits >> (2 * i)) & 1u ? 0xFFFFu : 0u) | ((bits >> (2 * i + 1)) & 1u ? 0xFFFF0000u : 0u);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ uint32_t mask_byte(const uint2* mask, size_t row, int kc)
{
    return (reinterpret_cast<const uint8_t*>(mask + row))[kc];
}

// Messages: rows [h[src] | e[edge]] of 21 target nodes, m = sum over a node's slots of
// relu(z) (FP32, slot order) as BF16, and the mask bits of row (node, slot).
// in_tab [N][6]: (source node, edge) of every slot, -1 where empty.
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_FWD)
msg_fwd_kernel(int nodes, int N, int E, const int2* __restrict__ in_tab, const bf16* __restrict__ h, const bf16* __restrict__ e,
               const bf16* __restrict__ Wpk, const float* __restrict__ bias, bf16* __restrict__ m, uint2* __restrict__ mask,
               int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char* As = tc_smem;                         // [16 row groups][16 k-chunks][8 rows][16 B], then FP32 rows
    unsigned char* Ws = tc_smem + TC_A_FWD;              // [8 output groups][16 k-chunks][8 outputs][16 B]
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ const unsigned char* rowp[2][2][TC_ROWS]; // gathered row halves of this and the next tile (NULL: no row)
    __shared__ float bias_sm[HD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < HD) bias_sm[tid] = bias[tid];
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 64, Ws, Wpk, HD * KIN * 2);
    const uint32_t tmem = tmem_sh;
    constexpr uint32_t IDESC = tc_idesc_bf16(TC_ROWS, HD);
    const int ntiles = (nodes + TILE_NODES - 1) / TILE_NODES;
    uint32_t phase = 0;
    auto lookup = [&](int t, int buf) {
        const int row = tid & (TC_ROWS - 1), hf = tid >> 7, k = row / NODE_ROWS, n = t * TILE_NODES + k;
        const unsigned char* p = nullptr;
        if (k < TILE_NODES && n < nodes) {
            const int b = n / N, l = n - b * N;
            const int2 s = in_tab[l * NODE_ROWS + row - k * NODE_ROWS];
            if (s.x >= 0)
                p = reinterpret_cast<const unsigned char*>(hf == 0 ? h + ((size_t)b * N + s.x) * HD : e + ((size_t)b * E + s.y) * HD);
        }
        rowp[buf][hf][row] = p;
    };
    if (blockIdx.x < ntiles) lookup(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, buf ^= 1) {
        __syncthreads();                                    // this tile's row pointers staged; the last epilogue done
        for (int i = tid; i < 16 * TC_ROWS; i += TC_THREADS) {   // chunk i: row (i >> 7) * 8 + (i & 7), k-chunk (i >> 3) & 15
            const int kc = (i >> 3) & 15, row = ((i >> 7) << 3) | (i & 7);
            const unsigned char* p = rowp[buf][kc >> 3][row];
            cp_async16(As + i * 16, p ? p + (kc & 7) * 16 : reinterpret_cast<const unsigned char*>(Wpk), p != nullptr);
        }
        if (tile + (int)gridDim.x < ntiles) lookup(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // visible to the tensor core
        tc_fence_before();
        __syncthreads();                                    // also: the previous tile's TMEM reads are done
        tc_fence_after();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < KIN / 16; ++ks)
                tc_mma(tmem, tc_desc(smem_u32(As) + ks * 256, 128, 16 * 128), tc_desc(smem_u32(Ws) + ks * 256, 128, 16 * 128),
                       IDESC, ks > 0 ? 1u : 0u);
            tc_commit(&bar_mma);
        }
        const bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        tc_fence_after();
        // warp w: accumulator rows 32 (w mod 4) .. + 31, columns 32 (w / 4) .. + 31: relu(z) to the consumed
        // operand tile as FP32 rows of 256 bytes (16-byte chunks swizzled by row)
        const int q = warp & 3, cb = (warp >> 2) * (HD / 2), row = q * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
        uint32_t bits = 0u;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int c0 = cb + 16 * hh;
            float z[16];
            tmem_ld16(tl + c0, z);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                z[i] += bias_sm[c0 + i];
                bits |= positive_bf16(z[i]) << (16 * hh + i);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4*>(As + row * 256 + ((((c0 >> 2) + c) ^ (row & 7)) << 4)) =
                    make_float4(fmaxf(z[4 * c], 0.f), fmaxf(z[4 * c + 1], 0.f), fmaxf(z[4 * c + 2], 0.f), fmaxf(z[4 * c + 3], 0.f));
        }
        if (mask && rowp[buf][0][row])
            reinterpret_cast<uint32_t*>(mask + (size_t)tile * TILE_NODES * NODE_ROWS + row)[warp >> 2] = bits;
        __syncthreads();
        for (int i = tid; i < TILE_NODES * (HD / 2); i += TC_THREADS) {      // node i / 32 of the tile, column pair i mod 32
            const int k = i >> 5, cp = i & 31, n = tile * TILE_NODES + k;
            if (n >= nodes) break;
            float x = 0.f, y = 0.f;
#pragma unroll
            for (int s = 0; s < NODE_ROWS; ++s) {
                const int r = k * NODE_ROWS + s;
                if (!rowp[buf][0][r]) continue;
                const float2 v = *reinterpret_cast<const float2*>(As + r * 256 + (((cp >> 1) ^ (r & 7)) << 4) + (cp & 1) * 8);
                x += v.x;
                y += v.y;
            }
            reinterpret_cast<uint32_t*>(m + (size_t)n * HD)[cp] = pack_bf2(x, y);
        }
    }
    tc_teardown(tmem, 64, failed, err);
}

// Sum of two BF16 rows' chunk, rounded to BF16.
__device__ __forceinline__ uint4 add_bf16x8(uint4 a, uint4 b)
{
    const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 p = unpack_bf2(x[i]), q = unpack_bf2(y[i]);
        w[i] = pack_bf2(p.x + q.x, p.y + q.y);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Node and edge updates: Y = P0 + relu([P0 | second] W^T + bias) as BF16 and the mask
// bits.  Nodes: second = m (rows of P1).  Edges (EDGE): second = h[i] + h[j], the sum
// of the edge's end rows of P1 = h, formed while staging.
template <bool EDGE>
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_FWD)
upd_fwd_kernel(int rows, const bf16* __restrict__ P0, const bf16* __restrict__ P1, const int2* __restrict__ ends, int N, int E,
               const bf16* __restrict__ Wpk, const float* __restrict__ bias, bf16* __restrict__ Yout, uint2* __restrict__ mask,
               int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char* As = tc_smem;                         // [16 row groups][16 k-chunks][8 rows][16 B]
    unsigned char* Ws = tc_smem + TC_A_FWD;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ const uint4* endp[2][2][TC_ROWS];         // EDGE: the two end rows of this and the next tile's edges
    __shared__ float bias_sm[HD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < HD) bias_sm[tid] = bias[tid];
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 64, Ws, Wpk, HD * KIN * 2);
    const uint32_t tmem = tmem_sh;
    constexpr uint32_t IDESC = tc_idesc_bf16(TC_ROWS, HD);
    const int ntiles = (rows + TC_ROWS - 1) / TC_ROWS;
    uint32_t phase = 0;
    auto lookup = [&](int t, int buf) {
        if (!EDGE) return;
        const int row = tid & (TC_ROWS - 1), which = tid >> 7, r = t * TC_ROWS + row;
        const uint4* p = nullptr;
        if (r < rows) {
            const int b = r / E, l = r - b * E;
            const int2 ij = ends[l];
            p = reinterpret_cast<const uint4*>(P1 + ((size_t)b * N + (which == 0 ? ij.x : ij.y)) * HD);
        }
        endp[buf][which][row] = p;
    };
    if (blockIdx.x < ntiles) lookup(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, buf ^= 1) {
        const int r0 = tile * TC_ROWS;
        __syncthreads();
        if (EDGE) {
            for (int i = tid; i < 8 * TC_ROWS; i += TC_THREADS) {        // first half: chunk kc of row, consecutive rows of P0
                const int kc = (i >> 3) & 7, row = ((i >> 6) << 3) | (i & 7), r = r0 + row;
                cp_async16(As + (((row >> 3) * 16 + kc) * 8 + (row & 7)) * 16, P0 + (size_t)(r < rows ? r : 0) * HD + kc * 8, r < rows);
            }
#pragma unroll
            for (int j = 0; j < 8 * TC_ROWS / TC_THREADS; ++j) {         // second half: the sum of the end rows
                const int i = tid + j * TC_THREADS, kc = (i >> 3) & 7, row = ((i >> 6) << 3) | (i & 7);
                const uint4 *p = endp[buf][0][row], *q = endp[buf][1][row];
                *reinterpret_cast<uint4*>(As + (((row >> 3) * 16 + 8 + kc) * 8 + (row & 7)) * 16) =
                    p ? add_bf16x8(p[kc], q[kc]) : make_uint4(0u, 0u, 0u, 0u);
            }
        } else {
            for (int i = tid; i < 16 * TC_ROWS; i += TC_THREADS) {
                const int kc = (i >> 3) & 15, row = ((i >> 7) << 3) | (i & 7), r = r0 + row;
                cp_async16(As + i * 16, (kc < 8 ? P0 : P1) + (size_t)(r < rows ? r : 0) * HD + (kc & 7) * 8, r < rows);
            }
        }
        if (tile + (int)gridDim.x < ntiles) lookup(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < KIN / 16; ++ks)
                tc_mma(tmem, tc_desc(smem_u32(As) + ks * 256, 128, 16 * 128), tc_desc(smem_u32(Ws) + ks * 256, 128, 16 * 128),
                       IDESC, ks > 0 ? 1u : 0u);
            tc_commit(&bar_mma);
        }
        const bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        tc_fence_after();
        const int q = warp & 3, cb = (warp >> 2) * (HD / 2), row0 = r0 + q * 32, row = q * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
        unsigned char* stage = As + warp * 4096;
        uint32_t yw[HD / 4], bits = 0u;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int c0 = cb + 16 * hh;
            float z[16];
            tmem_ld16(tl + c0, z);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                z[i] += bias_sm[c0 + i];
                bits |= positive_bf16(z[i]) << (16 * hh + i);
            }
            // the residual input is half 0 of this row, already staged: k-chunks c0/8 and c0/8 + 1
#pragma unroll
            for (int kc = 0; kc < 2; ++kc) {
                const uint4 b4 = *reinterpret_cast<const uint4*>(As + (((row >> 3) * 16 + (c0 >> 3) + kc) * 128) + (row & 7) * 16);
                const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 bb = unpack_bf2(bw[i]);
                    yw[8 * hh + 4 * kc + i] = pack_bf2(bb.x + fmaxf(z[8 * kc + 2 * i], 0.f), bb.y + fmaxf(z[8 * kc + 2 * i + 1], 0.f));
                }
            }
        }
        if (mask && r0 + row < rows) reinterpret_cast<uint32_t*>(mask + r0 + row)[warp >> 2] = bits;
        __syncthreads();                                   // every residual read before any slice is overwritten
        store_bf16x32(stage, yw, Yout + (size_t)row0 * HD + cb, HD, rows - row0, lane);
    }
    tc_teardown(tmem, 64, failed, err);
}

// ---- backward: input gradient dX = dZ W and weight gradient dW += dZ^T X of a tile
// Shared memory: X [16 input groups][16 row groups][8 rows][16 B] (32 KB, the weight
// gradient's A operand), dZ [16 row groups][8 k-chunks][8 rows][16 B] (16 KB), W^T
// (one or both 8 KB halves of 64 inputs).  Tensor memory: columns 0..63 dW^T
// accumulated over the CTA's tiles, 64..127 the current half of dX.  db: a thread
// stages one 8-column chunk of every eighth row group and adds it up on the way.
constexpr int BW_X = TC_ROWS * KIN * 2, BW_Z = TC_ROWS * HD * 2, BW_W = HD * HD * 2;
constexpr int TC_SMEM_UPD_BWD = BW_X + BW_Z + 2 * BW_W, TC_SMEM_EDGE_BWD = BW_X + BW_Z + BW_W;
constexpr int TC_CTAS_UPD_BWD = 3, TC_CTAS_EDGE_BWD = 3;

__device__ __forceinline__ void bwd_mma_wgrad(uint32_t tmem, const unsigned char* Xs, const unsigned char* Zs, bool first)
{
    constexpr uint32_t IDESC = tc_idesc_bf16(KIN, HD) | (1u << 15) | (1u << 16);   // M = 128 inputs, N = 64, both MN-major
#pragma unroll
    for (int ks = 0; ks < TC_ROWS / 16; ++ks)
        tc_mma(tmem, tc_desc(smem_u32(Xs) + ks * 256, 128, 16 * 128), tc_desc(smem_u32(Zs) + ks * 2048, 1024, 128), IDESC,
               first && ks == 0 ? 0u : 1u);
}

__device__ __forceinline__ void bwd_mma_input(uint32_t tmem, const unsigned char* Zs, const unsigned char* Wh)
{
    constexpr uint32_t IDESC = tc_idesc_bf16(TC_ROWS, HD);                         // one half: 64 inputs
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks)
        tc_mma(tmem + HD, tc_desc(smem_u32(Zs) + ks * 256, 128, 8 * 128), tc_desc(smem_u32(Wh) + ks * 256, 128, 8 * 128), IDESC,
               ks > 0 ? 1u : 0u);
}

// Adds the 8 BF16 values of a staged dZ chunk to this thread's column sums.
__device__ __forceinline__ void add_db(float (&db)[8], uint4 z)
{
    const uint32_t w[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 v = unpack_bf2(w[i]);
        db[2 * i] += v.x;
        db[2 * i + 1] += v.y;
    }
}

// The CTA's partials: dW [64][128] from tensor memory (lane = input), db [64] from the
// threads' column sums (thread: chunk kc of 8 columns; the 32 threads of a chunk in
// thread order), through `sm` (8 KB of shared memory).
__device__ __forceinline__ void bwd_partials(uint32_t tmem, float* P, const float (&db)[8], int kc, float* sm)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp < 4) {
        const int in = warp * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll
        for (int c0 = 0; c0 < HD; c0 += 16) {
            float d[16];
            tmem_ld16(tl + c0, d);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) P[(c0 + i) * KIN + in] = d[i];
        }
    }
    __syncthreads();                                        // the last tile's staging slices are read
    // threads of chunk kc: 8 per warp in the 4 warps with warp & 1 == kc >> 2
    const int slot = (warp >> 1) * 8 + (lane & 7);
#pragma unroll
    for (int i = 0; i < 8; ++i) sm[(kc * 8 + i) * 32 + slot] = db[i];
    __syncthreads();
    if (tid < HD) {
        float s = 0.f;
        for (int j = 0; j < 32; ++j) s += sm[tid * 32 + j];
        P[HD * KIN + tid] = s;
    }
}

// Node and edge updates.  EDGE: dZ = de & mask, de += dX[:, :64] in place, ds = dX[:, 64:]
// (FP32); X = [e | h_i + h_j].  Nodes: dh += sum over the node's edges of ds (inc order; inc NULL: none),
// dZ = dh & mask, dh += dX[:, :64], dm = dX[:, 64:] rounded to BF16 (the one form that
// the messages' dZ = dm & mask takes it in); X = [h | m].
template <bool EDGE>
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_UPD_BWD)
upd_bwd_kernel(int rows, int N, int E, const uint2* __restrict__ mask, float* g, const bf16* __restrict__ P0,
               const bf16* __restrict__ P1, const int2* __restrict__ ends, const int* __restrict__ inc, float* ds,
               bf16* __restrict__ dm, const bf16* __restrict__ WTpk, float* __restrict__ part, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *Xs = tc_smem, *Zs = tc_smem + BW_X, *Ws = Zs + BW_Z;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 128, Ws, WTpk, 2 * BW_W);
    const uint32_t tmem = tmem_sh;
    const int ntiles = (rows + TC_ROWS - 1) / TC_ROWS;
    const int r8 = lane & 7, q4 = lane >> 3, kz = (warp & 1) * 4 + q4;     // a warp stages 8 rows x 4 chunks at a time
    float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t phase = 0;
    bool first = true;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x) {
        const int r0 = tile * TC_ROWS;
#pragma unroll
        for (int j = 0; j < 8; ++j) {                       // X
            const int u = warp + 8 * j, rg = u >> 2, kc = (u & 3) * 4 + q4, row = rg * 8 + r8, r = r0 + row;
            unsigned char* dst = Xs + (kc * 16 + rg) * 128 + r8 * 16;
            const bool v = r < rows;
            if (!EDGE || (u & 2) == 0) {
                cp_async16(dst, (kc < 8 ? P0 : P1) + (size_t)(v ? r : 0) * HD + (kc & 7) * 8, v);
            } else {
                uint4 s = make_uint4(0u, 0u, 0u, 0u);
                if (v) {
                    const int b = r / E;
                    const int2 ij = ends[r - b * E];
                    s = add_bf16x8(*reinterpret_cast<const uint4*>(P1 + ((size_t)b * N + ij.x) * HD + (kc & 7) * 8),
                                   *reinterpret_cast<const uint4*>(P1 + ((size_t)b * N + ij.y) * HD + (kc & 7) * 8));
                }
                *reinterpret_cast<uint4*>(dst) = s;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {                       // dZ: chunk kz of row groups (warp >> 1) + 4 j
            const int rg = (warp >> 1) + 4 * j, row = rg * 8 + r8, r = r0 + row;
            uint4 z = make_uint4(0u, 0u, 0u, 0u);
            if (r < rows) {
                float4* gp = reinterpret_cast<float4*>(g + (size_t)r * HD + kz * 8);
                float4 a = gp[0], b = gp[1];
                if (!EDGE && inc) {
                    const int bi = r / N;
                    const int* il = inc + (r - bi * N) * NODE_ROWS;
                    float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
#pragma unroll
                    for (int s = 0; s < NODE_ROWS; ++s) {
                        const int ed = il[s];
                        if (ed < 0) continue;
                        const float4* dp = reinterpret_cast<const float4*>(ds + ((size_t)bi * E + ed) * HD + kz * 8);
                        const float4 x = dp[0], y = dp[1];
                        s0.x += x.x; s0.y += x.y; s0.z += x.z; s0.w += x.w;
                        s1.x += y.x; s1.y += y.y; s1.z += y.z; s1.w += y.w;
                    }
                    a.x += s0.x; a.y += s0.y; a.z += s0.z; a.w += s0.w;
                    b.x += s1.x; b.y += s1.y; b.z += s1.z; b.w += s1.w;
                    gp[0] = a;                              // the epilogue adds dX to it
                    gp[1] = b;
                }
                z = mask_bf16x8(make_uint4(pack_bf2(a.x, a.y), pack_bf2(a.z, a.w), pack_bf2(b.x, b.y), pack_bf2(b.z, b.w)),
                                mask_byte(mask, r, kz));
            }
            add_db(db, z);
            *reinterpret_cast<uint4*>(Zs + (rg * 8 + kz) * 128 + r8 * 16) = z;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const int q = warp & 3, row0 = r0 + q * 32, cb = (warp >> 2) * (HD / 2);
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + HD + cb;
        unsigned char* stage = Xs + warp * 4096;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (tid == 0) {
                bwd_mma_input(tmem, Zs, Ws + half * BW_W);
                if (half == 0) bwd_mma_wgrad(tmem, Xs, Zs, first);
                tc_commit(&bar_mma);
            }
            const bool ok = mbar_wait(&bar_mma, phase);
            phase ^= 1u;
            if (__syncthreads_or(!ok)) {
                failed = true;
                break;
            }
            tc_fence_after();
            uint32_t w[16];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                float d[16];
                tmem_ld16(tl + 16 * hh, d);
                tmem_ld_wait();
                if (half == 0 || EDGE) {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        stage_f32(stage, lane, 4 * hh + c, make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]));
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) w[8 * hh + i] = pack_bf2(d[2 * i], d[2 * i + 1]);
                }
            }
            if (half == 0) flush_add_f32x32(stage, g + (size_t)row0 * HD + cb, HD, rows - row0, lane);
            else if (EDGE) flush_f32x32(stage, ds + (size_t)row0 * HD + cb, HD, rows - row0, lane);
            else store_bf16x32(stage, w, dm + (size_t)row0 * HD + cb, HD, rows - row0, lane);
            tc_fence_before();
            __syncthreads();                                // dX read, the slices free: the next half or tile
            tc_fence_after();
        }
        first = false;
    }
    if (!failed) bwd_partials(tmem, part + (size_t)blockIdx.x * WPART, db, kz, reinterpret_cast<float*>(Xs));
    tc_teardown(tmem, 128, failed, err);
}

// Messages, edge half: rows 2e and 2e + 1 are the two directions of edge e; dZ = dm[tgt]
// & mask, de[e] += dX[2e][64:] + dX[2e + 1][64:] (set: =), weight gradient with X = [h[src] | e].
// msg_tab [2E]: (source node, mask row = target node * 6 + slot).
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_EDGE_BWD)
msg_bwd_edge_kernel(int rows, int N, int E, const int2* __restrict__ msg_tab, const uint2* __restrict__ mask,
                    const bf16* __restrict__ dm, const bf16* __restrict__ h, const bf16* __restrict__ e,
                    const bf16* __restrict__ WTpk, float* de, int set, float* __restrict__ part, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *Xs = tc_smem, *Zs = tc_smem + BW_X, *Ws = Zs + BW_Z;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ int4 rowt[2][TC_ROWS];                       // this and the next tile: source row, edge row, target row, mask row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 128, Ws, WTpk + HD * HD, BW_W);
    const uint32_t tmem = tmem_sh;
    const int ntiles = (rows + TC_ROWS - 1) / TC_ROWS;
    const int r8 = lane & 7, q4 = lane >> 3, kz = (warp & 1) * 4 + q4;
    float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t phase = 0;
    bool first = true;
    auto lookup = [&](int t, int buf) {
        if (tid >= TC_ROWS) return;
        const int r = t * TC_ROWS + tid;
        int4 v = make_int4(-1, 0, 0, 0);
        if (r < rows) {
            const int b = r / (2 * E), l = r - b * 2 * E;
            const int2 s = msg_tab[l];
            v = make_int4(b * N + s.x, b * E + (l >> 1), b * N + s.y / NODE_ROWS, b * N * NODE_ROWS + s.y);
        }
        rowt[buf][tid] = v;
    };
    if (blockIdx.x < ntiles) lookup(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, buf ^= 1) {
        const int r0 = tile * TC_ROWS;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int u = warp + 8 * j, rg = u >> 2, kc = (u & 3) * 4 + q4;
            const int4 t = rowt[buf][rg * 8 + r8];
            const bf16* p = kc < 8 ? h + (size_t)(t.x < 0 ? 0 : t.x) * HD : e + (size_t)t.y * HD;
            cp_async16(Xs + (kc * 16 + rg) * 128 + r8 * 16, p + (kc & 7) * 8, t.x >= 0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int rg = (warp >> 1) + 4 * j;
            const int4 t = rowt[buf][rg * 8 + r8];
            uint4 z = make_uint4(0u, 0u, 0u, 0u);
            if (t.x >= 0)
                z = mask_bf16x8(*reinterpret_cast<const uint4*>(dm + (size_t)t.z * HD + kz * 8), mask_byte(mask, t.w, kz));
            add_db(db, z);
            *reinterpret_cast<uint4*>(Zs + (rg * 8 + kz) * 128 + r8 * 16) = z;
        }
        if (tile + (int)gridDim.x < ntiles) lookup(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            bwd_mma_input(tmem, Zs, Ws);
            bwd_mma_wgrad(tmem, Xs, Zs, first);
            tc_commit(&bar_mma);
        }
        first = false;
        const bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        tc_fence_after();
        const int q = warp & 3, row0 = r0 + q * 32, cb = (warp >> 2) * (HD / 2);
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + HD + cb;
        unsigned char* stage = Xs + warp * 4096;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float d[16];
            tmem_ld16(tl + 16 * hh, d);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 4; ++c)
                stage_f32(stage, lane, 4 * hh + c, make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]));
        }
        // a warp's 32 rows are 16 whole edges (row0 is even)
        flush_pairs_f32x32(stage, de + (size_t)(row0 / 2) * HD + cb, HD, (rows - row0) / 2, lane, set != 0);
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    if (!failed) bwd_partials(tmem, part + (size_t)blockIdx.x * WPART, db, kz, reinterpret_cast<float*>(Xs));
    tc_teardown(tmem, 128, failed, err);
}

// Messages, node half: the rows of 21 source nodes (out_tab [N][6]: mask row of the
// message in a slot, -1 where empty); dh[n] += sum over n's slots of dX[:, :64].
// dZ (16 KB), then the FP32 rows over it (32 KB); W^T half; 12 KB unused, so that 4 CTAs fit and no fifth
constexpr int TC_SMEM_NODE_BWD = TC_ROWS * HD * 4 + BW_W + 12 * 1024;
constexpr int TC_CTAS_NODE_BWD = 4;
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_NODE_BWD)
msg_bwd_node_kernel(int nodes, int N, const int* __restrict__ out_tab, const uint2* __restrict__ mask,
                    const bf16* __restrict__ dm, const bf16* __restrict__ WTpk, float* dh, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *Zs = tc_smem, *Ws = tc_smem + TC_ROWS * HD * 4;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ int rowm[2][TC_ROWS];                        // this and the next tile: mask row (-1: none)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 128, Ws, WTpk, BW_W);
    const uint32_t tmem = tmem_sh;
    const int ntiles = (nodes + TILE_NODES - 1) / TILE_NODES;
    const int r8 = lane & 7, q4 = lane >> 3, kz = (warp & 1) * 4 + q4;
    uint32_t phase = 0;
    auto lookup = [&](int t, int buf) {
        if (tid >= TC_ROWS) return;
        const int k = tid / NODE_ROWS, n = t * TILE_NODES + k;
        int v = -1;
        if (k < TILE_NODES && n < nodes) {
            const int b = n / N, s = out_tab[(n - b * N) * NODE_ROWS + tid - k * NODE_ROWS];
            if (s >= 0) v = b * N * NODE_ROWS + s;
        }
        rowm[buf][tid] = v;
    };
    if (blockIdx.x < ntiles) lookup(blockIdx.x, 0);
    int buf = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, buf ^= 1) {
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int rg = (warp >> 1) + 4 * j, t = rowm[buf][rg * 8 + r8];
            uint4 z = make_uint4(0u, 0u, 0u, 0u);
            if (t >= 0)
                z = mask_bf16x8(*reinterpret_cast<const uint4*>(dm + (size_t)(t / NODE_ROWS) * HD + kz * 8), mask_byte(mask, t, kz));
            *reinterpret_cast<uint4*>(Zs + (rg * 8 + kz) * 128 + r8 * 16) = z;
        }
        if (tile + (int)gridDim.x < ntiles) lookup(tile + gridDim.x, buf ^ 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
            bwd_mma_input(tmem, Zs, Ws);
            tc_commit(&bar_mma);
        }
        const bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        if (__syncthreads_or(!ok)) {
            failed = true;
            break;
        }
        tc_fence_after();
        const int q = warp & 3, cb = (warp >> 2) * (HD / 2), row = q * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + HD + cb;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float d[16];
            tmem_ld16(tl + 16 * hh, d);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4*>(Zs + row * 256 + ((((cb + 16 * hh) >> 2) + c) ^ (row & 7)) * 16) =
                    make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]);
        }
        tc_fence_before();
        __syncthreads();
        for (int i = tid; i < TILE_NODES * (HD / 2); i += TC_THREADS) {
            const int k = i >> 5, cp = i & 31, n = tile * TILE_NODES + k;
            if (n >= nodes) break;
            float x = 0.f, y = 0.f;
#pragma unroll
            for (int s = 0; s < NODE_ROWS; ++s) {
                const int r = k * NODE_ROWS + s;
                if (rowm[buf][r] < 0) continue;
                const float2 v = *reinterpret_cast<const float2*>(Zs + r * 256 + (((cp >> 1) ^ (r & 7)) << 4) + (cp & 1) * 8);
                x += v.x;
                y += v.y;
            }
            float2* p = reinterpret_cast<float2*>(dh + (size_t)n * HD) + cp;
            float2 o = *p;
            o.x += x;
            o.y += y;
            *p = o;
        }
    }
    tc_teardown(tmem, 128, failed, err);
}

// dW += sum over a map's CTA partials, db likewise, for all maps at once (blockIdx.y):
// four interleaved sums added in a fixed order.
struct WMaps {
    float *dW[24], *db[24];
    int n[24];                       // partials of the map
};
__global__ void wgrad_reduce_kernel(WMaps maps, size_t stride, const float* __restrict__ part)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (i >= WPART) return;
    const float* p = part + k * stride + i;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    int b = 0;
    for (; b + 4 <= maps.n[k]; b += 4)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] += p[(size_t)(b + j) * WPART];
    for (int j = 0; b < maps.n[k]; ++b, ++j) s[j] += p[(size_t)b * WPART];
    const float t = (s[0] + s[1]) + (s[2] + s[3]);
    if (i < HD * KIN) maps.dW[k][i] += t;
    else maps.db[k][i - HD * KIN] += t;
}

// Packs the BF16 matrix W [64 outputs][128 inputs] of every layer map into the
// tcgen05 operand layouts: Wpk [8 output groups][16 k-chunks][8][8] (forward,
// B = W, K = inputs) and WTpk [16 input groups][8 k-chunks][8][8] (input
// gradient, B = W^T, K = outputs).  One thread per packed element.
__global__ void pack_weights_kernel(int nmat, const bf16* const* __restrict__ Ws, bf16* __restrict__ out)
{
    const int per = HD * KIN;
    const int64_t total = (int64_t)nmat * 2 * per;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / (2 * per)), which = (int)((i / per) & 1), e = (int)(i % per);
        const bf16* W = Ws[m];
        const int j = e & 7, r8 = (e >> 3) & 7;
        bf16 v;
        if (which == 0) {                    // output n = (e >> 10) * 8 + r8, input k = ((e >> 6) & 15) * 8 + j
            const int n = ((e >> 10) << 3) | r8, k = (((e >> 6) & 15) << 3) | j;
            v = W[n * KIN + k];
        } else {                             // input n = (e >> 9) * 8 + r8, output k = ((e >> 6) & 7) * 8 + j
            const int n = ((e >> 9) << 3) | r8, k = (((e >> 6) & 7) << 3) | j;
            v = W[k * KIN + n];
        }
        out[i] = v;
    }
}

// ------------------------------------------------------- elementwise kernels
// h0[b][n] = X[u_n]; e0[b][e] = Jt[idx(J)]; a thread converts 8 columns of a row
__global__ void embed_kernel(int B, int N, int E, const int* __restrict__ u, const int8_t* __restrict__ J,
                             const float* __restrict__ Xemb, const float* __restrict__ Jemb, bf16* h, bf16* e)
{
    const size_t nN = (size_t)B * N, total = (nN + (size_t)B * E) * (HD / 8);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t row = i / (HD / 8);
        const int c = (int)(i % (HD / 8));
        const float* src;
        bf16* dst;
        if (row < nN) {
            src = Xemb + u[row % N] * HD;
            dst = h + row * HD;
        } else {
            const int j = J[row - nN];
            src = Jemb + (j < 0 ? j + 3 : j + 2) * HD;      // -3,-2,-1,1,2,3 -> 0..5
            dst = e + (row - nN) * HD;
        }
        const float4 a = reinterpret_cast<const float4*>(src)[2 * c], b = reinterpret_cast<const float4*>(src)[2 * c + 1];
        reinterpret_cast<uint4*>(dst)[c] = make_uint4(pack_bf2(a.x, a.y), pack_bf2(a.z, a.w), pack_bf2(b.x, b.y), pack_bf2(b.z, b.w));
    }
}

// readout forward + loss gradient (one block of 256 threads per graph).  The node mean is
// summed node by node (64 threads, a column each) from rows that the block stages 64 at a
// time, the next 64 on their way meanwhile.
constexpr int RO_ROWS = 64, RO_THREADS = 256;
__global__ void __launch_bounds__(RO_THREADS) readout_kernel(int N, const bf16* __restrict__ h, const float* __restrict__ W1, const float* __restrict__ b1,
                               const float* __restrict__ w2, const float* __restrict__ b2, float* y, float* gbuf,
                               float* zbuf, const float* __restrict__ target, float inv_B, float* dybuf,
                               float* sqbuf, float* dh)
{
    __shared__ __align__(16) float gs[HD];
    __shared__ float as[HD], red[HD], dz[HD];
    __shared__ __align__(16) bf16 rows[RO_ROWS][HD];
    const int b = blockIdx.x, tid = threadIdx.x, c = tid;
    const uint4* src = reinterpret_cast<const uint4*>(h + (size_t)b * N * HD);
    constexpr int PER = RO_ROWS * HD / 8 / RO_THREADS;      // 16-byte pieces per thread
    uint4 v[PER];
    auto fetch = [&](int n0) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int i = tid + j * RO_THREADS;
            v[j] = n0 + i / (HD / 8) < N ? src[(size_t)n0 * (HD / 8) + i] : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    fetch(0);
    float acc = 0.f;
    for (int n0 = 0; n0 < N; n0 += RO_ROWS) {
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PER; ++j) reinterpret_cast<uint4*>(&rows[0][0])[tid + j * RO_THREADS] = v[j];
        __syncthreads();
        if (n0 + RO_ROWS < N) fetch(n0 + RO_ROWS);
        if (c < HD) {
            const int m = min(RO_ROWS, N - n0);
#pragma unroll 8
            for (int n = 0; n < m; ++n) acc += __bfloat162float(rows[n][c]);
        }
    }
    if (c < HD) gs[c] = acc / (float)N;
    __syncthreads();
    float z = 0.f;
    if (c < HD) {
        z = b1[c];
        for (int k = 0; k < HD; ++k) z += W1[c * HD + k] * gs[k];
        as[c] = fmaxf(z, 0.f);
        red[c] = as[c] * w2[c];
        gbuf[b * HD + c] = gs[c];
        zbuf[b * HD + c] = z;
    }
    __syncthreads();
    for (int s = HD / 2; s > 0; s >>= 1) {
        if (c < s) red[c] += red[c + s];
        __syncthreads();
    }
    const float yb = red[0] + b2[0];
    if (c == 0) y[b] = yb;
    if (!target) return;
    const float dy = 2.f * (yb - target[b]) * inv_B;
    if (c == 0) {                                  // this graph's loss term and output gradient (summed in order
        dybuf[b] = dy;                             // over graphs by readout_grad_kernel)
        sqbuf[b] = (yb - target[b]) * (yb - target[b]) * inv_B;
    }
    if (c < HD) dz[c] = z > 0.f ? dy * w2[c] : 0.f;
    __syncthreads();
    if (c < HD) {
        float dg = 0.f;
        for (int o = 0; o < HD; ++o) dg += dz[o] * W1[o * HD + c];
        dg /= (float)N;
        gs[c] = dg;
    }
    __syncthreads();
    const float4 d = reinterpret_cast<const float4*>(gs)[tid & (HD / 4 - 1)];
    float4* out = reinterpret_cast<float4*>(dh + (size_t)b * N * HD);
    for (int i = tid; i < N * (HD / 4); i += RO_THREADS) out[i] = d;
}

// Readout parameter gradients and the loss, summed over the B graphs in graph
// order (bit-reproducible): block c < 64, thread k: dW1[c][k] += sum_b dz_b[c]
// g_b[k] with dz_b[c] = dy_b w2[c] where z_b[c] > 0, and (thread 0) db1[c],
// dw2[c]; block 64: db2 and the loss.
__global__ void readout_grad_kernel(int B, const float* __restrict__ gbuf, const float* __restrict__ zbuf,
                                    const float* __restrict__ dybuf, const float* __restrict__ sqbuf,
                                    const float* __restrict__ w2, float* loss, float* dW1, float* db1, float* dw2,
                                    float* db2)
{
    const int c = blockIdx.x, k = threadIdx.x;
    if (c < HD) {
        const float w = w2[c];
        float acc = 0.f, a1 = 0.f, a2 = 0.f;
        for (int b = 0; b < B; ++b) {
            const float z = zbuf[b * HD + c], dy = dybuf[b];
            const float dz = z > 0.f ? dy * w : 0.f;
            acc += dz * gbuf[b * HD + k];
            a1 += dz;
            a2 += dy * fmaxf(z, 0.f);
        }
        dW1[c * HD + k] += acc;
        if (k == 0) {
            db1[c] += a1;
            dw2[c] += a2;
        }
    } else if (k == 0) {
        float s2 = 0.f, l = 0.f;
        for (int b = 0; b < B; ++b) {
            s2 += dybuf[b];
            l += sqbuf[b];
        }
        db2[0] += s2;
        *loss += l;
    }
}

// Embedding gradients: dX[o] += sum of dh over the nodes of orientation o, dJt[v] += sum of de over
// the edges of coupler value v.  A thread owns column c of a strided set of rows and keeps its 2 + 6
// class sums in registers; the block adds its 4 lanes' sums in lane order and writes them as its
// partial part[block][8][64] (classes: orientations 0, 1, coupler values -3..3 without 0), and
// embed_bwd_reduce adds the partials in block order (bit-reproducible).  256 threads per block.
__global__ void embed_bwd_kernel(int B, int N, int E, const int* __restrict__ u, const int8_t* __restrict__ J,
                                 const float* __restrict__ dh, const float* __restrict__ de, float* __restrict__ part)
{
    __shared__ float sp[4][8][HD];
    const int c = threadIdx.x % HD, lane = threadIdx.x / HD, lanes = blockDim.x / HD;
    const size_t nN = (size_t)B * N, nE = (size_t)B * E, stride = (size_t)gridDim.x * lanes;
    const size_t first = blockIdx.x * (size_t)lanes + lane;
    float ax0 = 0.f, ax1 = 0.f, aj[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (size_t row = first; row < nN; row += stride) {
        const float v = dh[row * HD + c];
        if (u[row % N]) ax1 += v;
        else ax0 += v;
    }
    for (size_t re = first; re < nE; re += stride) {
        const int j = J[re];
        const int k = j < 0 ? j + 3 : j + 2;                 // -3,-2,-1,1,2,3 -> 0..5
        const float v = de[re * HD + c];
#pragma unroll
        for (int q = 0; q < 6; ++q) aj[q] += k == q ? v : 0.f;
    }
    sp[lane][0][c] = ax0;
    sp[lane][1][c] = ax1;
#pragma unroll
    for (int q = 0; q < 6; ++q) sp[lane][2 + q][c] = aj[q];
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * HD; i += blockDim.x) {
        float t = 0.f;
        for (int l = 0; l < lanes; ++l) t += sp[l][i / HD][i % HD];
        part[(size_t)blockIdx.x * 8 * HD + i] = t;
    }
}

__global__ void embed_bwd_reduce(int nblocks, const float* __restrict__ part, float* dX, float* dJt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 8 * HD) return;
    float t = 0.f;
    for (int b = 0; b < nblocks; ++b) t += part[(size_t)b * 8 * HD + i];
    if (i < 2 * HD) dX[i] += t;
    else dJt[i - 2 * HD] += t;
}

__global__ void adam_kernel(int64_t n, float* theta, const float* __restrict__ g, float* m, float* v, float lr,
                            float b1, float b2, float c1, float c2, float eps)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void to_bf16_kernel(int64_t n, const float* __restrict__ x, bf16* y)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

int grid_for(size_t work, int block = 256)
{
    const size_t b = (work + block - 1) / block;
    return (int)(b > 8192 ? 8192 : (b < 1 ? 1 : b));
}

}  // namespace

// ==========================================================================
// host runtime
// ==========================================================================
struct sg_model {
    int layers = 4;
    int64_t nparams = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    float *theta = nullptr, *grad = nullptr, *mom1 = nullptr, *mom2 = nullptr, *dloss = nullptr;
    bf16* wbf = nullptr;          // BF16 copy of theta
    bf16* wpk = nullptr;          // per layer map: W and W^T in the tcgen05 operand layouts (2 x 8192 BF16 each)
    const bf16** d_wptr = nullptr;// device array: the BF16 matrices of every layer map (pack_weights_kernel input)
    int* d_err = nullptr;         // set by a tensor-core kernel whose bounded wait ran out
    int sms = 0;                  // SMs of the device (persistent grids)
    int64_t step = 0;
    // offsets into theta
    int64_t oX = 0, oJ = 0, oW1 = 0, ob1 = 0, ow2 = 0, ob2 = 0;
    std::vector<int64_t> oWm, obm, oWu, obu, oWe, obe;
    // graph + activation buffers for the current (L, Bcap)
    int L = 0, N = 0, E = 0, Bcap = 0;
    int *d_u = nullptr, *d_inc = nullptr, *d_out_tab = nullptr;   // topology tables (see the kernels)
    int2 *d_ends = nullptr, *d_in_tab = nullptr, *d_msg_tab = nullptr;
    int8_t* d_J = nullptr;
    float *d_t = nullptr, *d_y = nullptr, *d_g = nullptr, *d_z = nullptr;
    float *d_dy = nullptr, *d_sq = nullptr;   // per graph: output gradient, loss term (readout)
    float* d_epart = nullptr;                 // embedding-gradient block partials [4 x SMs][8][64]
    std::vector<bf16*> h, e, m;
    std::vector<uint2*> mm, mu, me;   // per layer: sign bits of the message, node and edge pre-activations
    float *dh = nullptr, *de = nullptr, *ds = nullptr;
    bf16* dm = nullptr;
    float* wpart = nullptr;       // weight-gradient partials: [3 layers maps][wcap CTAs][WPART]
    int wcap = 0;
    uint64_t launches = 0;
    std::string err = "no error";
};

namespace {

int sfail(sg_model* m, int code, const std::string& msg)
{
    if (m) m->err = msg;
    else ptg::set_global_error(msg.c_str());
    return code;
}

#define SK(call, what)                                                                              \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess)                                                                      \
            return sfail(M, e_ == cudaErrorMemoryAllocation ? PT_ERR_OOM : PT_ERR_CUDA,             \
                         std::string(what) + ": " + cudaGetErrorString(e_));                        \
    } while (0)

template <class T>
cudaError_t salloc(T** p, size_t n)
{
    return cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * (n ? n : 1));
}

void free_graph(sg_model* M)
{
    cudaFree(M->d_u); cudaFree(M->d_inc); cudaFree(M->d_out_tab);
    cudaFree(M->d_ends); cudaFree(M->d_in_tab); cudaFree(M->d_msg_tab);
    M->d_u = M->d_inc = M->d_out_tab = nullptr;
    M->d_ends = M->d_in_tab = M->d_msg_tab = nullptr;
    cudaFree(M->d_J); M->d_J = nullptr;
    float** fl[] = {&M->d_t, &M->d_y, &M->d_g, &M->d_z, &M->d_dy, &M->d_sq, &M->d_epart, &M->dh, &M->de, &M->ds, &M->wpart};
    for (float** p : fl) { cudaFree(*p); *p = nullptr; }
    cudaFree(M->dm); M->dm = nullptr;
    for (auto* v : {&M->h, &M->e, &M->m}) {
        for (bf16* p : *v) cudaFree(p);
        v->clear();
    }
    for (auto* v : {&M->mm, &M->mu, &M->me}) {
        for (uint2* p : *v) cudaFree(p);
        v->clear();
    }
    M->L = M->Bcap = 0;
}

// Persistent CTAs for `rows` rows in tiles of `per` at ctas_per_sm residents.
int tc_grid(const sg_model* M, int rows, int ctas_per_sm, int per = TC_ROWS)
{
    const int tiles = (rows + per - 1) / per, cap = ctas_per_sm * M->sms;
    return tiles < cap ? (tiles > 0 ? tiles : 1) : cap;
}

// Builds the Chimera C_L topology in the coupler order of pt.h and sizes the
// activation buffers for B graphs.
int prepare(sg_model* M, int L, int B)
{
    if (M->L == L && M->Bcap >= B) return PT_OK;
    free_graph(M);
    const int N = 8 * L * L, E = 16 * L * L + 8 * L * (L - 1);
    std::vector<int> ei, ej;
    auto idx = [L](int r, int c, int u, int k) { return 8 * (r * L + c) + 4 * u + k; };
    for (int r = 0; r < L; ++r)
        for (int c = 0; c < L; ++c)
            for (int k = 0; k < 4; ++k)
                for (int kp = 0; kp < 4; ++kp) { ei.push_back(idx(r, c, 0, k)); ej.push_back(idx(r, c, 1, kp)); }
    for (int r = 0; r + 1 < L; ++r)
        for (int c = 0; c < L; ++c)
            for (int k = 0; k < 4; ++k) { ei.push_back(idx(r, c, 0, k)); ej.push_back(idx(r + 1, c, 0, k)); }
    for (int r = 0; r < L; ++r)
        for (int c = 0; c + 1 < L; ++c)
            for (int k = 0; k < 4; ++k) { ei.push_back(idx(r, c, 1, k)); ej.push_back(idx(r, c + 1, 1, k)); }
    // message row 2e: source ej -> target ei; row 2e+1: source ei -> target ej.  A node's incoming and
    // outgoing rows and its edges fill its 6 slots in ascending order
    std::vector<int> u(N), inc(N * MAXDEG, -1), out_tab(N * MAXDEG, -1);
    std::vector<int2> ends(E), in_tab(N * MAXDEG, make_int2(-1, -1)), msg_tab(2 * E);
    std::vector<int> cin(N, 0), cout(N, 0), cinc(N, 0);
    for (int i = 0; i < N; ++i) u[i] = (i >> 2) & 1;
    for (int e2 = 0; e2 < E; ++e2) {
        ends[e2] = make_int2(ei[e2], ej[e2]);
        for (int d = 0; d < 2; ++d) {
            const int src = d == 0 ? ej[e2] : ei[e2], tgt = d == 0 ? ei[e2] : ej[e2];
            const int slot = tgt * MAXDEG + cin[tgt]++;
            in_tab[slot] = make_int2(src, e2);
            msg_tab[2 * e2 + d] = make_int2(src, slot);
            out_tab[src * MAXDEG + cout[src]++] = slot;
        }
        inc[ei[e2] * MAXDEG + cinc[ei[e2]]++] = e2;
        inc[ej[e2] * MAXDEG + cinc[ej[e2]]++] = e2;
    }
    auto up = [&](auto** d, const auto& v) -> cudaError_t {
        cudaError_t r = salloc(d, v.size());
        if (r != cudaSuccess) return r;
        return cudaMemcpy(*d, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice);
    };
    SK(up(&M->d_u, u), "upload topology");
    SK(up(&M->d_inc, inc), "upload topology");
    SK(up(&M->d_out_tab, out_tab), "upload topology");
    SK(up(&M->d_ends, ends), "upload topology");
    SK(up(&M->d_in_tab, in_tab), "upload topology");
    SK(up(&M->d_msg_tab, msg_tab), "upload topology");
    const size_t nN = (size_t)B * N, nE = (size_t)B * E;
    SK(salloc(&M->d_J, nE), "cudaMalloc J");
    SK(salloc(&M->d_t, (size_t)B), "cudaMalloc t");
    SK(salloc(&M->d_y, (size_t)B), "cudaMalloc y");
    SK(salloc(&M->d_g, (size_t)B * HD), "cudaMalloc g");
    SK(salloc(&M->d_z, (size_t)B * HD), "cudaMalloc z");
    SK(salloc(&M->d_dy, (size_t)B), "cudaMalloc dy");
    SK(salloc(&M->d_sq, (size_t)B), "cudaMalloc sq");
    SK(salloc(&M->d_epart, (size_t)4 * M->sms * 8 * HD), "cudaMalloc embedding partials");
    M->h.assign(M->layers + 1, nullptr);
    for (auto* v : {&M->e, &M->m}) v->assign(M->layers, nullptr);
    for (auto* v : {&M->mm, &M->mu, &M->me}) v->assign(M->layers, nullptr);
    for (int l = 0; l <= M->layers; ++l) SK(salloc(&M->h[l], nN * HD), "cudaMalloc h");
    for (int l = 0; l < M->layers; ++l) {
        SK(salloc(&M->e[l], nE * HD), "cudaMalloc e");
        SK(salloc(&M->m[l], nN * HD), "cudaMalloc m");
        SK(salloc(&M->mm[l], nN * MAXDEG), "cudaMalloc message mask");
        SK(salloc(&M->mu[l], nN), "cudaMalloc node mask");
        if (l + 1 < M->layers) SK(salloc(&M->me[l], nE), "cudaMalloc edge mask");
    }
    M->wcap = tc_grid(M, B * 2 * E, TC_CTAS_UPD_BWD > TC_CTAS_EDGE_BWD ? TC_CTAS_UPD_BWD : TC_CTAS_EDGE_BWD);
    SK(salloc(&M->wpart, (size_t)3 * M->layers * M->wcap * WPART), "cudaMalloc wpart");
    SK(salloc(&M->dh, nN * HD), "cudaMalloc dh");
    SK(salloc(&M->dm, nN * HD), "cudaMalloc dm");
    SK(salloc(&M->de, nE * HD), "cudaMalloc de");
    SK(salloc(&M->ds, nE * HD), "cudaMalloc ds");
    M->L = L; M->N = N; M->E = E; M->Bcap = B;
    return PT_OK;
}

// The tcgen05 operand copies of every layer matrix follow the BF16 weights.
void pack_weights(sg_model* M)
{
    pack_weights_kernel<<<grid_for((size_t)M->layers * 3 * 2 * HD * KIN), 256, 0, M->stream>>>(M->layers * 3,
                                                                                                  M->d_wptr, M->wpk);
    M->launches++;
}

// Packed operands of layer l's map `which` (0 messages, 1 node update, 2 edge update).
const bf16* wpk_fwd(const sg_model* M, int l, int which) { return M->wpk + ((size_t)(l * 3 + which) * 2) * HD * KIN; }
const bf16* wpk_bwd(const sg_model* M, int l, int which) { return wpk_fwd(M, l, which) + HD * KIN; }

// The last layer updates no edges: nothing after it reads them.
void forward(sg_model* M, int B, bool train)
{
    const int N = M->N, E = M->E;
    cudaStream_t st = M->stream;
    embed_kernel<<<grid_for((size_t)B * (N + E) * (HD / 8)), 256, 0, st>>>(B, N, E, M->d_u, M->d_J, M->theta + M->oX,
                                                                             M->theta + M->oJ, M->h[0], M->e[0]);
    M->launches++;
    for (int l = 0; l < M->layers; ++l) {
        msg_fwd_kernel<<<tc_grid(M, B * N, TC_CTAS_FWD, TILE_NODES), TC_THREADS, TC_SMEM_FWD, st>>>(
            B * N, N, E, M->d_in_tab, M->h[l], M->e[l], wpk_fwd(M, l, 0), M->theta + M->obm[l], M->m[l], train ? M->mm[l] : nullptr,
            M->d_err);
        upd_fwd_kernel<false><<<tc_grid(M, B * N, TC_CTAS_FWD), TC_THREADS, TC_SMEM_FWD, st>>>(
            B * N, M->h[l], M->m[l], nullptr, N, E, wpk_fwd(M, l, 1), M->theta + M->obu[l], M->h[l + 1], train ? M->mu[l] : nullptr,
            M->d_err);
        M->launches += 2;
        if (l + 1 == M->layers) break;
        upd_fwd_kernel<true><<<tc_grid(M, B * E, TC_CTAS_FWD), TC_THREADS, TC_SMEM_FWD, st>>>(
            B * E, M->e[l], M->h[l + 1], M->d_ends, N, E, wpk_fwd(M, l, 2), M->theta + M->obe[l], M->e[l + 1],
            train ? M->me[l] : nullptr, M->d_err);
        M->launches++;
    }
}

// Gradient of the mean squared error into M->grad (zeroed first); loss into M->dloss.
int backward_all(sg_model* M, int B)
{
    const int N = M->N, E = M->E;
    cudaStream_t st = M->stream;
    float* G = M->grad;
    SK(cudaMemsetAsync(G, 0, sizeof(float) * M->nparams, st), "zero grad");
    SK(cudaMemsetAsync(M->dloss, 0, sizeof(float), st), "zero loss");
    readout_kernel<<<B, RO_THREADS, 0, st>>>(N, M->h[M->layers], M->theta + M->oW1, M->theta + M->ob1, M->theta + M->ow2,
                                             M->theta + M->ob2, M->d_y, M->d_g, M->d_z, M->d_t, 1.f / (float)B, M->d_dy,
                                             M->d_sq, M->dh);
    readout_grad_kernel<<<HD + 1, HD, 0, st>>>(B, M->d_g, M->d_z, M->d_dy, M->d_sq, M->theta + M->ow2, M->dloss,
                                               G + M->oW1, G + M->ob1, G + M->ow2, G + M->ob2);
    M->launches += 2;
    WMaps maps;
    int nmaps = 0;
    const size_t stride = (size_t)M->wcap * WPART;
    auto map = [&](int64_t oW, int64_t ob, int n) {      // the next map's partials
        maps.dW[nmaps] = G + oW;
        maps.db[nmaps] = G + ob;
        maps.n[nmaps] = n;
        return M->wpart + stride * nmaps++;
    };
    for (int l = M->layers - 1; l >= 0; --l) {
        const bool last = l + 1 == M->layers;             // its edge update has no gradient
        if (!last) {
            const int g = tc_grid(M, B * E, TC_CTAS_UPD_BWD);
            upd_bwd_kernel<true><<<g, TC_THREADS, TC_SMEM_UPD_BWD, st>>>(B * E, N, E, M->me[l], M->de, M->e[l], M->h[l + 1],
                                                                         M->d_ends, nullptr, M->ds, nullptr, wpk_bwd(M, l, 2),
                                                                         map(M->oWe[l], M->obe[l], g), M->d_err);
            M->launches++;
        }
        int g = tc_grid(M, B * N, TC_CTAS_UPD_BWD);
        upd_bwd_kernel<false><<<g, TC_THREADS, TC_SMEM_UPD_BWD, st>>>(B * N, N, E, M->mu[l], M->dh, M->h[l], M->m[l], nullptr,
                                                                      last ? nullptr : M->d_inc, M->ds, M->dm, wpk_bwd(M, l, 1),
                                                                      map(M->oWu[l], M->obu[l], g), M->d_err);
        g = tc_grid(M, B * 2 * E, TC_CTAS_EDGE_BWD);
        msg_bwd_edge_kernel<<<g, TC_THREADS, TC_SMEM_EDGE_BWD, st>>>(B * 2 * E, N, E, M->d_msg_tab, M->mm[l], M->dm, M->h[l],
                                                                     M->e[l], wpk_bwd(M, l, 0), M->de, last ? 1 : 0,
                                                                     map(M->oWm[l], M->obm[l], g), M->d_err);
        msg_bwd_node_kernel<<<tc_grid(M, B * N, TC_CTAS_NODE_BWD, TILE_NODES), TC_THREADS, TC_SMEM_NODE_BWD, st>>>(
            B * N, N, M->d_out_tab, M->mm[l], M->dm, wpk_bwd(M, l, 0), M->dh, M->d_err);
        M->launches += 3;
    }
    wgrad_reduce_kernel<<<dim3((WPART + 255) / 256, nmaps), 256, 0, st>>>(maps, stride, M->wpart);
    embed_bwd_kernel<<<4 * M->sms, 256, 0, st>>>(B, N, E, M->d_u, M->d_J, M->dh, M->de, M->d_epart);
    embed_bwd_reduce<<<(8 * HD + 255) / 256, 256, 0, st>>>(4 * M->sms, M->d_epart, G + M->oX, G + M->oJ);
    M->launches += 3;
    return PT_OK;
}

// A tensor-core kernel whose bounded mbarrier wait ran out leaves 1 in d_err
// (its CTA stopped and freed its tensor memory): the call reports a timeout
// and the word is cleared for the next call.
int tc_status(sg_model* M, int terr)
{
    if (!terr) return PT_OK;
    SK(cudaMemsetAsync(M->d_err, 0, sizeof(int), M->stream), "clear status");
    SK(cudaStreamSynchronize(M->stream), "sync status");
    return sfail(M, PT_ERR_TIMEOUT, "a tensor-core kernel's mbarrier wait ran out (results of this call are invalid)");
}

int load_batch(sg_model* M, int L, int B, const int8_t* J, const float* t)
{
    if (L < 1 || L > ptg::MAX_L || B < 1 || B > 4096 || !J) return sfail(M, PT_ERR_ARG, "need 1 <= L <= 16, 1 <= B <= 4096");
    const int E = 16 * L * L + 8 * L * (L - 1);
    unsigned bad = 0u;                                // no early exit: the compiler vectorises the scan
    for (size_t i = 0; i < (size_t)B * E; ++i) bad |= (unsigned)(J[i] == 0) | (unsigned)(J[i] < -3) | (unsigned)(J[i] > 3);
    if (bad) return sfail(M, PT_ERR_ARG, "surrogate couplers must be in {+-1, +-2, +-3}");
    int rc = prepare(M, L, B);
    if (rc) return rc;
    SK(cudaMemcpyAsync(M->d_J, J, (size_t)B * E, cudaMemcpyHostToDevice, M->stream), "upload J");
    if (t) SK(cudaMemcpyAsync(M->d_t, t, sizeof(float) * B, cudaMemcpyHostToDevice, M->stream), "upload targets");
    return PT_OK;
}

}  // namespace

extern "C" {

const char* sg_last_error(const sg_model* m) { return m ? m->err.c_str() : pt_last_error(nullptr); }

int sg_create(sg_model** out, int32_t hidden, int32_t layers, void* stream)
{
    sg_model* M = nullptr;
    if (!out) return sfail(nullptr, PT_ERR_ARG, "NULL argument");
    *out = nullptr;
    if (hidden != HD || layers < 1 || layers > 8) return sfail(nullptr, PT_ERR_ARG, "hidden must be 64, layers in [1, 8]");
    M = new (std::nothrow) sg_model();
    if (!M) return sfail(nullptr, PT_ERR_OOM, "host allocation failed");
    M->layers = layers;
    int64_t o = 0;
    M->oX = o; o += 2 * HD;
    M->oJ = o; o += 6 * HD;
    for (int l = 0; l < layers; ++l) {
        M->oWm.push_back(o); o += HD * KIN;
        M->obm.push_back(o); o += HD;
        M->oWu.push_back(o); o += HD * KIN;
        M->obu.push_back(o); o += HD;
        M->oWe.push_back(o); o += HD * KIN;
        M->obe.push_back(o); o += HD;
    }
    M->oW1 = o; o += HD * HD;
    M->ob1 = o; o += HD;
    M->ow2 = o; o += HD;
    M->ob2 = o; o += 1;
    M->nparams = o;
    auto bail = [&](int code) { std::string msg = M->err; sg_destroy(M); return sfail(nullptr, code, msg); };
    if (stream) M->stream = (cudaStream_t)stream;
    else {
        cudaError_t e = cudaStreamCreateWithFlags(&M->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) { M->err = std::string("cudaStreamCreate: ") + cudaGetErrorString(e); return bail(PT_ERR_CUDA); }
        M->own_stream = true;
    }
    if (salloc(&M->theta, o) != cudaSuccess || salloc(&M->grad, o) != cudaSuccess || salloc(&M->mom1, o) != cudaSuccess ||
        salloc(&M->mom2, o) != cudaSuccess || salloc(&M->wbf, o) != cudaSuccess || salloc(&M->dloss, 1) != cudaSuccess) {
        M->err = "cudaMalloc parameters failed";
        return bail(PT_ERR_OOM);
    }
    cudaMemset(M->theta, 0, sizeof(float) * o);
    cudaMemset(M->mom1, 0, sizeof(float) * o);
    cudaMemset(M->mom2, 0, sizeof(float) * o);
    cudaMemset(M->wbf, 0, sizeof(bf16) * o);
    {
        // tcgen05 operand copies of the layer matrices, their source pointers, the timeout word
        std::vector<const bf16*> ptrs;
        for (int l = 0; l < layers; ++l) {
            ptrs.push_back(M->wbf + M->oWm[l]);
            ptrs.push_back(M->wbf + M->oWu[l]);
            ptrs.push_back(M->wbf + M->oWe[l]);
        }
        int dev = 0, sms = 0;
        if (salloc(&M->wpk, (size_t)layers * 3 * 2 * HD * KIN) != cudaSuccess ||
            salloc(&M->d_wptr, ptrs.size()) != cudaSuccess || salloc(&M->d_err, 1) != cudaSuccess) {
            M->err = "cudaMalloc tensor-core operands failed";
            return bail(PT_ERR_OOM);
        }
        cudaError_t e = cudaMemcpy(M->d_wptr, ptrs.data(), sizeof(bf16*) * ptrs.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(M->wpk, 0, sizeof(bf16) * (size_t)layers * 3 * 2 * HD * KIN);
        if (e == cudaSuccess) e = cudaMemset(M->d_err, 0, sizeof(int));
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const struct { const void* k; int smem; } tk[] = {
            {(const void*)msg_fwd_kernel, TC_SMEM_FWD},
            {(const void*)upd_fwd_kernel<false>, TC_SMEM_FWD},
            {(const void*)upd_fwd_kernel<true>, TC_SMEM_FWD},
            {(const void*)upd_bwd_kernel<false>, TC_SMEM_UPD_BWD},
            {(const void*)upd_bwd_kernel<true>, TC_SMEM_UPD_BWD},
            {(const void*)msg_bwd_edge_kernel, TC_SMEM_EDGE_BWD},
            {(const void*)msg_bwd_node_kernel, TC_SMEM_NODE_BWD}};
        for (const auto& t : tk)
            if (e == cudaSuccess) e = cudaFuncSetAttribute(t.k, cudaFuncAttributeMaxDynamicSharedMemorySize, t.smem);
        if (e != cudaSuccess) {
            M->err = std::string("tensor-core set-up: ") + cudaGetErrorString(e);
            return bail(PT_ERR_CUDA);
        }
        M->sms = sms;
    }
    *out = M;
    return PT_OK;
}

void sg_destroy(sg_model* M)
{
    if (!M) return;
    if (M->stream) cudaStreamSynchronize(M->stream);
    free_graph(M);
    cudaFree(M->theta); cudaFree(M->grad); cudaFree(M->mom1); cudaFree(M->mom2); cudaFree(M->wbf); cudaFree(M->dloss);
    cudaFree(M->wpk); cudaFree(M->d_wptr); cudaFree(M->d_err);
    if (M->own_stream && M->stream) cudaStreamDestroy(M->stream);
    delete M;
}

int64_t sg_num_params(const sg_model* M) { return M ? M->nparams : 0; }

int sg_set_params(sg_model* M, const float* theta)
{
    if (!M || !theta) return sfail(M, PT_ERR_ARG, "NULL argument");
    SK(cudaMemcpyAsync(M->theta, theta, sizeof(float) * M->nparams, cudaMemcpyHostToDevice, M->stream), "upload params");
    SK(cudaMemsetAsync(M->mom1, 0, sizeof(float) * M->nparams, M->stream), "zero moments");
    SK(cudaMemsetAsync(M->mom2, 0, sizeof(float) * M->nparams, M->stream), "zero moments");
    to_bf16_kernel<<<grid_for((size_t)M->nparams), 256, 0, M->stream>>>(M->nparams, M->theta, M->wbf);
    M->launches++;
    pack_weights(M);
    M->step = 0;
    SK(cudaStreamSynchronize(M->stream), "sync set_params");
    return PT_OK;
}

int sg_get_params(sg_model* M, float* theta)
{
    if (!M || !theta) return sfail(M, PT_ERR_ARG, "NULL argument");
    SK(cudaMemcpyAsync(theta, M->theta, sizeof(float) * M->nparams, cudaMemcpyDeviceToHost, M->stream), "download params");
    SK(cudaStreamSynchronize(M->stream), "sync get_params");
    return PT_OK;
}

int sg_forward(sg_model* M, int32_t L, int32_t B, const int8_t* J, float* y)
{
    if (!M || !y) return sfail(M, PT_ERR_ARG, "NULL argument");
    int rc = load_batch(M, L, B, J, nullptr);
    if (rc) return rc;
    forward(M, B, false);
    readout_kernel<<<B, RO_THREADS, 0, M->stream>>>(M->N, M->h[M->layers], M->theta + M->oW1, M->theta + M->ob1,
                                            M->theta + M->ow2, M->theta + M->ob2, M->d_y, M->d_g, M->d_z, nullptr,
                                            0.f, nullptr, nullptr, nullptr);
    M->launches++;
    SK(cudaGetLastError(), "forward kernels");
    SK(cudaMemcpyAsync(y, M->d_y, sizeof(float) * B, cudaMemcpyDeviceToHost, M->stream), "download y");
    int terr = 0;
    SK(cudaMemcpyAsync(&terr, M->d_err, sizeof(int), cudaMemcpyDeviceToHost, M->stream), "download status");
    SK(cudaStreamSynchronize(M->stream), "sync forward");
    return tc_status(M, terr);
}

int sg_grad(sg_model* M, int32_t L, int32_t B, const int8_t* J, const float* t, float* loss, float* grad)
{
    if (!M || !t) return sfail(M, PT_ERR_ARG, "NULL argument");
    int rc = load_batch(M, L, B, J, t);
    if (rc) return rc;
    forward(M, B, true);
    if ((rc = backward_all(M, B))) return rc;
    SK(cudaGetLastError(), "gradient kernels");
    if (grad) SK(cudaMemcpyAsync(grad, M->grad, sizeof(float) * M->nparams, cudaMemcpyDeviceToHost, M->stream), "download grad");
    float lv = 0.f;
    int terr = 0;
    SK(cudaMemcpyAsync(&lv, M->dloss, sizeof(float), cudaMemcpyDeviceToHost, M->stream), "download loss");
    SK(cudaMemcpyAsync(&terr, M->d_err, sizeof(int), cudaMemcpyDeviceToHost, M->stream), "download status");
    SK(cudaStreamSynchronize(M->stream), "sync grad");
    if (loss) *loss = lv;
    return tc_status(M, terr);
}

int sg_adam(sg_model* M, float lr)
{
    if (!M) return PT_ERR_ARG;
    M->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - (float)std::pow(0.9, (double)M->step), c2 = 1.f - (float)std::pow(0.999, (double)M->step);
    adam_kernel<<<grid_for((size_t)M->nparams), 256, 0, M->stream>>>(M->nparams, M->theta, M->grad, M->mom1, M->mom2,
                                                                        lr, b1, b2, c1, c2, 1e-8f);
    to_bf16_kernel<<<grid_for((size_t)M->nparams), 256, 0, M->stream>>>(M->nparams, M->theta, M->wbf);
    M->launches += 2;
    pack_weights(M);
    SK(cudaGetLastError(), "adam kernels");
    SK(cudaStreamSynchronize(M->stream), "sync adam");
    return PT_OK;
}

int sg_train_step(sg_model* M, int32_t L, int32_t B, const int8_t* J, const float* t, float lr, float* loss)
{
    int rc = sg_grad(M, L, B, J, t, loss, nullptr);
    if (rc) return rc;
    return sg_adam(M, lr);
}

uint64_t sg_launch_count(const sg_model* M) { return M ? M->launches : 0; }

}  // extern "C"

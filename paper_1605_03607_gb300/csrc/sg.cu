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
// 0.13 ms of tensor time), above all its gathers into the SMs, and launch gaps for small
// batches.  So per layer 2 forward and 2 backward kernels, each with every linear map of
// its rows and everything around them, no message row in memory, and rows that a tile
// gathers several times taken from L1.  Measured against one kernel per step with FP32
// messages, pre-activations and masked gradients in memory (97 launches, 18 now):
// gradient of 256 C_8 graphs 3.95 -> 1.16 ms, of 128 C_4 graphs 1.01 -> 0.28 ms, 64 C_8
// predictions 0.42 -> 0.14 ms.  (With a kernel per map and message rows of 21 nodes
// summed through shared memory: 2.24, 0.59 and 0.26 ms.)
#include <algorithm>
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
//   * persistent CTAs over tiles of 128 rows (nodes or edges); one thread issues the
//     MMAs and commits them to an mbarrier;
//   * operands in shared memory in the canonical layout without swizzle, built
//     from 8-row x 16-byte core matrices; a descriptor's leading byte offset
//     steps between core matrices along K, its stride byte offset along M or N.
//     With the two the other way round every address would still lie inside the
//     CTA's shared memory;
//   * the weights, pre-packed in that layout (pack_weights_kernel), arrive by
//     bulk asynchronous copies; gathered rows by 16-byte cp.async;
//   * after the commit each warp reads its 32 accumulator rows (TMEM lanes
//     32w .. 32w+31) with tcgen05.ld, one row per thread, for the epilogue;
//   * every mbarrier wait is bounded: on a timeout the CTA records it in
//     *err, stops taking tiles, frees its tensor memory and returns.
constexpr uint32_t TC_WAIT_LIMIT = 1u << 22;
constexpr int TC_ROWS = 128;
// CTAs of 256 threads.  In the epilogue warps w and w + 4 read the same 32 tensor-memory
// lanes (a warp reaches lanes 32 (w mod 4) .. + 31) and split the columns.
constexpr int TC_THREADS = 256;

// A staged operand: columns ("chunks") of 8 BF16 x 128 rows, 16 bytes a row, CH bytes
// apart.  A warp's load or copy takes 4 whole rows of 128 bytes (8 lanes x 16 bytes a
// row): half the L1 wavefronts of 8 half rows, which had the L1 data pipe 45-80 % busy.
// The 16 bytes beyond 128 rows put the 8 chunks of a row into different banks.  Read
// along its columns a tile is a K-major operand, along its rows an MN-major one: the dZ
// tile is the A operand of the input gradient and the B operand of the weight gradient.
constexpr int CH = TC_ROWS * 16 + 16;
constexpr int OP64 = 8 * CH;                  // operand of 64 columns; one of 128 is two, adjacent
constexpr int W64 = HD * HD * 2;              // 64 x 64 weights

__device__ __forceinline__ unsigned char* op_at(unsigned char* t, int kc, int row) { return t + kc * CH + row * 16; }

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

// Bulk asynchronous copies global -> shared of n0 and n1 bytes (multiples of 16, 0: none;
// addresses 16-byte aligned) to adjacent places, completing on `bar`.
__device__ __forceinline__ void bulk_g2s(unsigned char* dst, const void* src0, uint32_t n0, const void* src1, uint32_t n1, uint64_t* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(n0 + n1) : "memory");
    if (n0)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(dst)), "l"(src0), "r"(n0), "r"(smem_u32(bar))
                     : "memory");
    if (n1)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(dst + n0)), "l"(src1), "r"(n1), "r"(smem_u32(bar))
                     : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

// The same through L1: rows that several rows of a tile gather.
__device__ __forceinline__ void cp_async16_l1(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid, bool l1)
{
    if (l1) cp_async16_l1(dst, src, valid);
    else cp_async16(dst, src, valid);
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

// A warp's 32 accumulator rows (lane l holds row l), 32 BF16 columns packed in 16 words
// each, through a 2 KB slice of shared memory so that each global store instruction
// writes whole pieces of rows: 8 rows x 64 bytes.  Row l's 16-byte chunk c sits at slot
// c ^ ((l >> 1) & 3) of its row, so neither the row-wise writes nor the chunk-wise reads
// meet a bank conflict.  g points at the warp's first row and first column; only rows
// < nvalid are written.
__device__ __forceinline__ void store_bf16x32(unsigned char* stage, const uint32_t (&w)[16], bf16* g, int nvalid, int lane)
{
#pragma unroll
    for (int c = 0; c < 4; ++c)
        *reinterpret_cast<uint4*>(stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) =
            make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int row = k * 8 + (lane >> 2), c = lane & 3;
        const uint4 x = *reinterpret_cast<const uint4*>(stage + row * 64 + ((c ^ ((row >> 1) & 3)) << 4));
        if (row < nvalid) *reinterpret_cast<uint4*>(g + (size_t)row * HD + c * 8) = x;
    }
    __syncwarp();
}

// FP32 tile of 128 rows x 64 columns over consumed operands (32 KB): 16-byte chunk c of
// row r at slot c ^ (r & 7), so that neither a warp that writes chunk c of 32 rows nor one
// that reads 8 chunks of 4 rows meets a bank conflict.
__device__ __forceinline__ float4* tile_f32(unsigned char* t, int row, int c)
{
    return reinterpret_cast<float4*>(t + row * 256 + ((c ^ (row & 7)) << 4));
}

// 64 accumulator columns from tensor memory to an FP32 tile.
__device__ __forceinline__ void tmem_to_tile(unsigned char* t, uint32_t tcol, int warp, int lane)
{
    const int q = warp & 3, cb = (warp >> 2) * (HD / 2);
    const uint32_t tl = tcol + ((uint32_t)(q * 32) << 16) + cb;
    float d[2][16];
    tmem_ld16(tl, d[0]);
    tmem_ld16(tl + 16, d[1]);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float* v = &d[c >> 2][4 * (c & 3)];
        *tile_f32(t, q * 32 + lane, (cb >> 2) + c) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// Common prologue: tensor memory (ncols columns, warp 0), the two mbarriers, and the
// packed weights by bulk copies.  Returns false (for every thread) if the weights did not
// arrive within the wait limit.
__device__ __forceinline__ bool tc_setup(uint32_t* tmem_sh, uint64_t* bar_w, uint64_t* bar_mma, uint32_t ncols, unsigned char* Ws,
                                         const void* W0, uint32_t n0, const void* W1, uint32_t n1)
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
    if (tid == 0) bulk_g2s(Ws, W0, n0, W1, n1, bar_w);
    bool ok = mbar_wait(bar_w, 0);
    if (!ok) ok = mbar_wait(bar_w, 0);         // second bounded wait for the copies still in flight
    return !__syncthreads_or(!ok);
}

// Launches of a pass are programmatically dependent: a kernel may start while the one before
// still runs, sets up (weights, topology tables: not written by any kernel of a pass) and
// waits here for it to end before it touches what it computed (pointers to that are not
// __restrict__: such loads may move across the wait).  Lets the next kernel start.
// 128 C_4 graphs: gradient 358 -> 319 us.
__device__ __forceinline__ void pass_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The staged operands are complete: this thread's copies have landed and its stores are
// visible to the tensor core; tensor-memory reads before it are ordered before the MMAs
// after it.  True (for every thread) if any thread's last wait failed.
__device__ __forceinline__ bool tc_ready(bool failed)
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    const bool f = __syncthreads_or(failed);
    tc_fence_after();
    return f;
}

// Z = A W^T: A 128 columns, W [8 output groups][16 k-chunks][8 outputs][16 B]
__device__ __forceinline__ void mma_forward(uint32_t tmem, const unsigned char* As, const unsigned char* Ws)
{
    const uint64_t a = tc_desc(smem_u32(As), CH, 128), b = tc_desc(smem_u32(Ws), 128, 16 * 128);     // + bytes / 16: a later start
#pragma unroll
    for (int ks = 0; ks < KIN / 16; ++ks)
        tc_mma(tmem, a + ks * 2 * CH / 16, b + ks * 16, tc_idesc_bf16(TC_ROWS, HD), ks > 0 ? 1u : 0u);
}

// dX (+)= dZ W over nin (64 or 128) inputs: W^T [nin / 8 input groups][8 k-chunks][8][16 B]
template <int NIN>
__device__ __forceinline__ void mma_input(uint32_t tmem, const unsigned char* Zs, const unsigned char* Ws, bool add)
{
    const uint64_t a = tc_desc(smem_u32(Zs), CH, 128), b = tc_desc(smem_u32(Ws), 128, 8 * 128);
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks)
        tc_mma(tmem, a + ks * 2 * CH / 16, b + ks * 16, tc_idesc_bf16(TC_ROWS, NIN), add || ks > 0 ? 1u : 0u);
}

// dW^T (+)= X^T dZ: X 128 columns (M), dZ 64 (N), K = 128 rows; both MN-major
__device__ __forceinline__ void mma_wgrad(uint32_t tmem, const unsigned char* Xs, const unsigned char* Zs, bool add)
{
    constexpr uint32_t IDESC = tc_idesc_bf16(KIN, HD) | (1u << 15) | (1u << 16);
    const uint64_t a = tc_desc(smem_u32(Xs), 128, CH), b = tc_desc(smem_u32(Zs), 128, CH);
#pragma unroll
    for (int ks = 0; ks < TC_ROWS / 16; ++ks) tc_mma(tmem, a + ks * 16, b + ks * 16, IDESC, add || ks > 0 ? 1u : 0u);
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
// Rows are gathered while they are staged, everything elementwise around a linear map
// runs in its staging or its epilogue, and maps that work on the same rows share a
// kernel: forward, a layer's messages with its node update, then its edge update;
// backward, a layer's messages with the updates of the layer below, edges then nodes.
// Only node and edge features (BF16), their gradients (FP32) and one bit per activation
// go through memory:
//   * the backward needs a pre-activation's sign only: the forward keeps it as a
//     bit (z > 0 after rounding to BF16), 8 bytes per row of 64; messages' bits are kept
//     slot by slot [6][nodes];
//   * a tile is 128 nodes, whose messages are computed slot by slot, or 128 edges, whose
//     messages are computed direction by direction.  So a thread sums relu(z) of its node
//     in registers, and the input gradients of a node's (edge's) messages add up in
//     tensor memory;
//   * a map's input gradient and weight gradient share the staged tile, and an edge's two
//     source rows of the messages are the end rows of the edge update below.
// The first layer's features are rows of the embedding tables (BF16 parameters): node
// orientations (bit 2 of the node, X [2][64]) and coupler values (Jt [6][64]).  Its kernels
// gather them there (J non-NULL), mostly from L1, and no feature of it is in memory:
// gradient of 256 C_8 graphs 1.24 -> 1.20 ms, 64 C_8 predictions 156 -> 150 us.
// Thread mapping of staged rows: q8 = lane mod 8 is the 16-byte chunk, the row is
// 4 warp + lane / 8 + 32 j, j = 0 .. 3.
constexpr int SLOTS = MAXDEG;

__device__ __forceinline__ int orientation(int node) { return (node >> 2) & 1; }
__device__ __forceinline__ int coupler_class(int j) { return j < 0 ? j + 3 : j + 2; }      // -3,-2,-1,1,2,3 -> 0..5

// z's sign bit of the backward's mask: positive after rounding to BF16 (2^-133 is
// the smallest BF16 number; 2^-134 and below round to zero).
// Appends it to `bits` from below.
__device__ __forceinline__ uint32_t push_positive(uint32_t bits, float z)
{
    return __funnelshift_l(__float_as_uint(0x1p-134f - z), bits, 1);       // the sign bit of a NaN result is 0
}

// 8 BF16 values (one 16-byte chunk) with the columns whose mask bit is 0 cleared.
__device__ __forceinline__ uint4 mask_bf16x8(uint4 v, uint32_t bits)
{
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] &= ((bits >> (2 * i)) & 1u ? 0xFFFFu : 0u) | ((bits >> (2 * i + 1)) & 1u ? 0xFFFF0000u : 0u);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// 4 FP32 values rounded to BF16, the columns whose mask bit is 0 cleared.
__device__ __forceinline__ uint2 mask_f32x4(float4 v, uint32_t bits)
{
    uint32_t a = pack_bf2(v.x, v.y), b = pack_bf2(v.z, v.w);
    a &= (bits & 1u ? 0xFFFFu : 0u) | (bits & 2u ? 0xFFFF0000u : 0u);
    b &= (bits & 4u ? 0xFFFFu : 0u) | (bits & 8u ? 0xFFFF0000u : 0u);
    return make_uint2(a, b);
}

__device__ __forceinline__ uint32_t mask_byte(const uint2* mask, size_t row, int kc)
{
    return (reinterpret_cast<const uint8_t*>(mask + row))[kc];
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

// Node stage of a layer: m = sum over a node's slots of relu(Wm [h[src] | e] + bm) (FP32, slot
// order) rounded to BF16, then hout = h + relu(Wu [h | m] + bu).  7 steps a tile (6
// slots, the update), each staged while the step before is computed: two operand
// buffers, a barrier a step.  in_tab [6][N]: (source node, edge) of every slot, -1 where
// empty.  m non-NULL (training): m and the mask bits mm, mu are kept.
constexpr int TC_SMEM_NODE_FWD = 4 * OP64 + 4 * W64 + 2 * SLOTS * TC_ROWS * 8, TC_CTAS_NODE_FWD = 2;
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_NODE_FWD)
node_fwd_kernel(int nodes, int N, int E, const int2* __restrict__ in_tab, const bf16* h, const bf16* e,
                const bf16* __restrict__ Wm, const float* __restrict__ bm, const bf16* __restrict__ Wu, const float* __restrict__ bu,
                bf16* __restrict__ hout, bf16* __restrict__ m, uint2* __restrict__ mm, uint2* __restrict__ mu,
                const int8_t* __restrict__ J, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char* const Ws = tc_smem + 4 * OP64;
    // rows of h and e (-1: none) of this and the next tile's slots [2][6][128]
    int2* const tab = reinterpret_cast<int2*>(Ws + 4 * W64);
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ float bias[2][HD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q8 = lane & 7, srow = warp * 4 + (lane >> 3);
    if (tid < HD) bias[0][tid] = bm[tid];
    else if (tid < 2 * HD) bias[1][tid - HD] = bu[tid - HD];
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 64, Ws, Wm, 2 * W64, Wu, 2 * W64);
    const uint32_t tmem = tmem_sh;
    const int ntiles = (nodes + TC_ROWS - 1) / TC_ROWS;
    const int q = warp & 3, row = q * 32 + lane, cb = (warp >> 2) * (HD / 2);       // epilogue: accumulator row, first column
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + cb;
    auto lookup = [&](int t, int which) {
        if (t >= ntiles) return;
        const int n = t * TC_ROWS + (tid & (TC_ROWS - 1)), b = n / N, l = n - b * N;
#pragma unroll
        for (int s = tid >> 7; s < SLOTS; s += 2) {
            int2 v = n < nodes ? in_tab[s * N + l] : make_int2(-1, -1);
            if (v.x >= 0) v = J ? make_int2(orientation(v.x), coupler_class(J[b * E + v.y])) : make_int2(b * N + v.x, b * E + v.y);
            tab[(which * SLOTS + s) * TC_ROWS + (tid & (TC_ROWS - 1))] = v;
        }
    };
    int lt = blockIdx.x, ls = 0, lw = 0;                    // what is staged next: tile, step, its table
    auto stage = [&](int buf) {
        if (lt >= ntiles) return;
        unsigned char* A = tc_smem + buf * 2 * OP64;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = srow + 32 * j;
            if (ls < SLOTS) {
                const int2 v = tab[(lw * SLOTS + ls) * TC_ROWS + r];
                cp_async16_l1(op_at(A, q8, r), h + (size_t)max(v.x, 0) * HD + q8 * 8, v.x >= 0);
                cp_async16(op_at(A, 8 + q8, r), e + (size_t)max(v.y, 0) * HD + q8 * 8, v.x >= 0, J != nullptr);
            } else {
                const int n = lt * TC_ROWS + r;
                cp_async16(op_at(A, q8, r), h + (size_t)(n >= nodes ? 0 : J ? orientation(n) : n) * HD + q8 * 8, n < nodes,
                           J != nullptr);
            }
        }
        if (++ls > SLOTS) { ls = 0; lt += gridDim.x; lw ^= 1; }
    };
    lookup(blockIdx.x, 0);
    __syncthreads();
    pass_begin();
    if (!failed) stage(0);
    uint32_t phase = 0;
    int buf = 0, which = 0;
    bool ok = true;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, which ^= 1) {
        const int r0 = tile * TC_ROWS;
        float acc[HD / 2];
#pragma unroll
        for (int i = 0; i < HD / 2; ++i) acc[i] = 0.f;
        for (int s = 0; s < SLOTS; ++s, buf ^= 1) {
            if ((failed = tc_ready(!ok))) break;
            unsigned char* const A = tc_smem + buf * 2 * OP64;
            if (tid == 0) {
                mma_forward(tmem, A, Ws);
                tc_commit(&bar_mma);
            }
            stage(buf ^ 1);
            if (s == 1) lookup(tile + gridDim.x, which ^ 1);      // the other table's last row was staged a barrier ago
            ok = mbar_wait(&bar_mma, phase);
            phase ^= 1u;
            tc_fence_after();
            const bool v = tab[(which * SLOTS + s) * TC_ROWS + row].x >= 0;
            float z[2][16];
            tmem_ld16(tl, z[0]);
            tmem_ld16(tl + 16, z[1]);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) z[i >> 4][i & 15] += bias[0][cb + i];
            if (m) {
                uint32_t bits = 0u;
#pragma unroll
                for (int i = 31; i >= 0; --i) bits = push_positive(bits, z[i >> 4][i & 15]);
                if (r0 + row < nodes) reinterpret_cast<uint32_t*>(mm + (size_t)s * nodes + r0 + row)[warp >> 2] = bits;
            }
            if (v)
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] += fmaxf(z[i >> 4][i & 15], 0.f);
        }
        if (failed) break;
        // m: into the update's operand, and (training) to memory through the last slot's consumed operand
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = pack_bf2(acc[2 * i], acc[2 * i + 1]);
        unsigned char* const A = tc_smem + buf * 2 * OP64;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(op_at(A, 8 + (cb >> 3) + c, row)) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
        if (m)
            store_bf16x32(tc_smem + (buf ^ 1) * 2 * OP64 + warp * 2048, w, m + (size_t)(r0 + q * 32) * HD + cb, nodes - r0 - q * 32, lane);
        if ((failed = tc_ready(!ok))) break;
        if (tid == 0) {
            mma_forward(tmem, A, Ws + 2 * W64);
            tc_commit(&bar_mma);
        }
        stage(buf ^ 1);
        ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        tc_fence_after();
        uint32_t bits = 0u;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int c0 = cb + 16 * hh;
            float z[16];
            tmem_ld16(tl + 16 * hh, z);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] += bias[1][c0 + i];
            uint32_t part = 0u;
#pragma unroll
            for (int i = 15; i >= 0; --i) part = push_positive(part, z[i]);
            bits |= part << (16 * hh);
#pragma unroll
            for (int kc = 0; kc < 2; ++kc) {                // the residual input is staged: chunks c0 / 8 and c0 / 8 + 1
                const uint4 b4 = *reinterpret_cast<const uint4*>(op_at(A, (c0 >> 3) + kc, row));
                const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 bb = unpack_bf2(bw[i]);
                    w[8 * hh + 4 * kc + i] = pack_bf2(bb.x + fmaxf(z[8 * kc + 2 * i], 0.f), bb.y + fmaxf(z[8 * kc + 2 * i + 1], 0.f));
                }
            }
        }
        if (m && r0 + row < nodes) reinterpret_cast<uint32_t*>(mu + r0 + row)[warp >> 2] = bits;
        // through the consumed half of m; the next step's barrier comes before this buffer is staged again
        store_bf16x32(A + OP64 + warp * 2048, w, hout + (size_t)(r0 + q * 32) * HD + cb, nodes - r0 - q * 32, lane);
        buf ^= 1;
    }
    failed = __syncthreads_or(failed || !ok);
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_teardown(tmem, 64, failed, err);
}

// Edge update: Y = P0 + relu([P0 | h[i] + h[j]] W^T + bias) as BF16 and the mask bits;
// the sum of the edge's end rows is formed while staging.  3 CTAs an SM up to 12 tiles an
// SM, 4 above: the fewer have more L1 for the gathered rows (64 C_8 predictions 166 ->
// 157 us), the more hide more latency (256: 434 -> 414 us).
constexpr int TC_SMEM_EDGE_FWD = 2 * OP64 + 2 * W64, EDGE_FWD_FEW = 12;
template <int CTAS>
__global__ void __launch_bounds__(TC_THREADS, CTAS)
edge_fwd_kernel(int rows, const bf16* P0, const bf16* h, const int2* __restrict__ ends, int N, int E,
                const bf16* __restrict__ W, const float* __restrict__ bias, bf16* __restrict__ Yout, uint2* __restrict__ mask,
                const int8_t* __restrict__ J, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *const As = tc_smem, *const Ws = tc_smem + 2 * OP64;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    __shared__ int2 endn[2][TC_ROWS];                       // the two end nodes of this and the next tile's edges, -1: no row
    __shared__ int prow[2][TC_ROWS];                        // and the row of P0
    __shared__ float bias_sm[HD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q8 = lane & 7, srow = warp * 4 + (lane >> 3);
    if (tid < HD) bias_sm[tid] = bias[tid];
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 64, Ws, W, 2 * W64, nullptr, 0);
    const uint32_t tmem = tmem_sh;
    const int ntiles = (rows + TC_ROWS - 1) / TC_ROWS;
    const int q = warp & 3, row = q * 32 + lane, cb = (warp >> 2) * (HD / 2);
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16) + cb;
    uint32_t phase = 0;
    auto lookup = [&](int t, int buf) {
        if (t >= ntiles || tid >= TC_ROWS) return;
        const int r = t * TC_ROWS + tid;
        int2 ij = make_int2(-1, -1);
        if (r < rows) {
            const int b = r / E;
            ij = ends[r - b * E];
            ij.x += b * N;
            ij.y += b * N;
        }
        endn[buf][tid] = ij;
        prow[buf][tid] = r >= rows ? 0 : J ? coupler_class(J[r]) : r;
    };
    lookup(blockIdx.x, 0);
    __syncthreads();
    pass_begin();
    int buf = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, buf ^= 1) {
        const int r0 = tile * TC_ROWS;
        uint4 a[4], b[4];                                   // every load before the first use
        int2 ij[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) ij[j] = endn[buf][srow + 32 * j];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            a[j] = b[j] = make_uint4(0u, 0u, 0u, 0u);
            if (ij[j].x >= 0) {
                a[j] = *reinterpret_cast<const uint4*>(h + (size_t)ij[j].x * HD + q8 * 8);
                b[j] = *reinterpret_cast<const uint4*>(h + (size_t)ij[j].y * HD + q8 * 8);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = srow + 32 * j;
            const bool v = ij[j].x >= 0;
            cp_async16(op_at(As, q8, r), P0 + (size_t)prow[buf][r] * HD + q8 * 8, v, J != nullptr);
        }
        lookup(tile + gridDim.x, buf ^ 1);
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(op_at(As, 8 + q8, srow + 32 * j)) = add_bf16x8(a[j], b[j]);
        tc_ready(false);
        if (tid == 0) {
            mma_forward(tmem, As, Ws);
            tc_commit(&bar_mma);
        }
        const bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        tc_fence_after();
        uint32_t yw[16], bits = 0u;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int c0 = cb + 16 * hh;
            float z[16];
            tmem_ld16(tl + 16 * hh, z);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] += bias_sm[c0 + i];
            uint32_t part = 0u;
#pragma unroll
            for (int i = 15; i >= 0; --i) part = push_positive(part, z[i]);
            bits |= part << (16 * hh);
#pragma unroll
            for (int kc = 0; kc < 2; ++kc) {                // the residual input is staged: chunks c0 / 8 and c0 / 8 + 1
                const uint4 b4 = *reinterpret_cast<const uint4*>(op_at(As, (c0 >> 3) + kc, row));
                const uint32_t bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 bb = unpack_bf2(bw[i]);
                    yw[8 * hh + 4 * kc + i] = pack_bf2(bb.x + fmaxf(z[8 * kc + 2 * i], 0.f), bb.y + fmaxf(z[8 * kc + 2 * i + 1], 0.f));
                }
            }
        }
        if (mask && r0 + row < rows) reinterpret_cast<uint32_t*>(mask + r0 + row)[warp >> 2] = bits;
        store_bf16x32(As + OP64 + warp * 2048, yw, Yout + (size_t)(r0 + q * 32) * HD + cb, rows - r0 - q * 32, lane);
        failed = __syncthreads_or(!ok);                     // the operand is consumed
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_teardown(tmem, 64, failed, err);
}

// ---- backward
// Adds the BF16 values of a staged dZ chunk to this thread's column sums.
__device__ __forceinline__ void add_db(float* db, uint32_t a, uint32_t b)
{
    const float2 x = unpack_bf2(a), y = unpack_bf2(b);
    db[0] += x.x;
    db[1] += x.y;
    db[2] += y.x;
    db[3] += y.y;
}

__device__ __forceinline__ void add_f4(float* s, float4 v)
{
    s[0] += v.x;
    s[1] += v.y;
    s[2] += v.z;
    s[3] += v.w;
}

// A CTA's partial of a bias gradient: a thread's 8 column sums are those of chunk q8
// (f32 false) or of the 4 columns from 4 q8 and from 32 + 4 q8 (true); the 32 threads of a
// column in thread order, through 8 KB of shared memory.
__device__ __forceinline__ void db_partial(float* P, const float (&db)[8], bool f32, float* sm)
{
    const int tid = threadIdx.x, q8 = tid & 7, slot = tid >> 3;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) sm[(f32 ? (i >> 2) * 32 + q8 * 4 + (i & 3) : q8 * 8 + i) * 32 + (slot ^ (q8 << 2))] = db[i];
    __syncthreads();
    if (tid < HD) {
        float s = 0.f;
        const int x = (f32 ? (tid & 31) >> 2 : tid >> 3) << 2;
        for (int j = 0; j < 32; ++j) s += sm[tid * 32 + (j ^ x)];
        P[HD * KIN + tid] = s;
    }
}

// A CTA's partial of dW [64][128] from tensor memory (lane = input).
__device__ __forceinline__ void dw_partial(uint32_t tcol, float* P, int warp, int lane)
{
    const int q = warp & 3, in = q * 32 + lane, cb = (warp >> 2) * (HD / 2);
    const uint32_t tl = tcol + ((uint32_t)(q * 32) << 16) + cb;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        float d[16];
        tmem_ld16(tl + 16 * hh, d);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) P[(cb + 16 * hh + i) * KIN + in] = d[i];
    }
}

constexpr int TC_CTAS_BWD = 2;

// Nodes.  PRE, messages of a layer: dh[n] += sum over the messages that n sends of
// (dm[target] & mask) Wm[:, :64], slot by slot (out_tab [6][N]: target node * 8 + its slot,
// -1 where empty).
// Both: dh[n] += the sums of the edge updates' gradients over n's edges, dc[n] for those in
// its cell, ds of the up to two between cells (inter [2][N]: their number in the graph, -1
// where empty).
// POST, node update of the layer below: dZ = dh & mu, dh += dX[:, :64], dmo = dX[:, 64:]
// rounded to BF16 (the one form that the messages' dZ = dm & mask takes it in), weight
// gradient with X = [h | m].  Slots go in two groups of three operand buffers: a step's
// fence, barrier and load latency cost more than its MMAs (256 C_8 graphs, a launch: 74
// us, slot by slot 82).  Without PRE (the last layer) every node of a graph starts
// from the readout's gradient dg [graphs][64]; without POST (the first) dh is not kept,
// only its sums over the nodes of either orientation, part [CTA][2][64].
constexpr int TC_SMEM_NODE_BWD = 5 * OP64 + 3 * W64 + 2 * (SLOTS + 2) * TC_ROWS * 4;
template <bool PRE, bool POST>
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_BWD)
node_bwd_kernel(int nodes, int N, int E, const int* __restrict__ out_tab, const uint2* mm, const bf16* dm,
                const bf16* __restrict__ WmT, const int* __restrict__ inter, const float* dc, const float* ds, const float* dg,
                float* dh, const uint2* mu, const bf16* h, const bf16* m, const bf16* __restrict__ WuT,
                bf16* __restrict__ dmo, float* __restrict__ part, int first_layer, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *const Zs = tc_smem, *const Xs = tc_smem + 3 * OP64, *const Ws = tc_smem + 5 * OP64;     // Ws: Wm^T (h half), Wu^T
    // of this and the next tile, -1: none: target row * 8 + its slot [2][6][128], rows of ds [2][2][128]
    int *const otab = reinterpret_cast<int*>(Ws + 3 * W64), *const itab = otab + 2 * SLOTS * TC_ROWS;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q8 = lane & 7, srow = warp * 4 + (lane >> 3);
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 256, Ws, WmT, PRE ? W64 : 0, WuT, POST ? 2 * W64 : 0);
    const uint32_t tmem = tmem_sh, tdw = tmem + KIN;        // dX: columns 0..127, dW^T: 128..191
    const int ntiles = (nodes + TC_ROWS - 1) / TC_ROWS;
    float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t phase = 0;
    bool first = true;
    auto lookup = [&](int t, int which) {
        if (!PRE || t >= ntiles) return;
        const int r = tid & (TC_ROWS - 1), n = t * TC_ROWS + r, b = n / N, l = n - b * N;
#pragma unroll
        for (int s = tid >> 7; s < SLOTS; s += 2) {
            const int o = n < nodes ? out_tab[s * N + l] : -1;
            otab[(which * SLOTS + s) * TC_ROWS + r] = o < 0 ? -1 : b * N * 8 + o;
        }
        if (POST) {
            const int s = tid >> 7, i = n < nodes ? inter[s * N + l] : -1;
            itab[(which * 2 + s) * TC_ROWS + r] = i < 0 ? -1 : b * (E - 2 * N) + i;
        }
    };
    lookup(blockIdx.x, 0);
    __syncthreads();
    pass_begin();
    int which = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, which ^= 1) {
        float4 ga[4], gb[4];                                // dh: columns 4 q8 .. and 32 + 4 q8 ..
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = tile * TC_ROWS + srow + 32 * j;
            const bool v = n < nodes;
            if (POST) {
                cp_async16(op_at(Xs, q8, srow + 32 * j), h + (size_t)(!v ? 0 : first_layer ? orientation(n) : n) * HD + q8 * 8, v,
                           first_layer != 0);
                cp_async16(op_at(Xs, 8 + q8, srow + 32 * j), m + (size_t)(v ? n : 0) * HD + q8 * 8, v);
            }
            ga[j] = gb[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!PRE && v) {
                ga[j] = reinterpret_cast<const float4*>(dg + (size_t)(n / N) * HD)[q8];
                gb[j] = reinterpret_cast<const float4*>(dg + (size_t)(n / N) * HD)[8 + q8];
            }
        }
        bool ok = true;
        if (PRE) {
            constexpr int GRP = SLOTS / 2;
            uint4 z[GRP][4];
            uint32_t mk[GRP][4];
            auto load = [&](int s0) {
#pragma unroll
                for (int i = 0; i < GRP; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int t = otab[(which * SLOTS + s0 + i) * TC_ROWS + srow + 32 * j];
                        z[i][j] = make_uint4(0u, 0u, 0u, 0u);
                        mk[i][j] = 0u;
                        if (t >= 0) {
                            const size_t n = t >> 3;
                            z[i][j] = *reinterpret_cast<const uint4*>(dm + n * HD + q8 * 8);
                            mk[i][j] = mask_byte(mm, (size_t)(t & 7) * nodes + n, q8);
                        }
                    }
            };
            load(0);
#pragma unroll
            for (int grp = 0; grp < 2; ++grp) {
                if (grp > 0) {                              // the first group's MMAs are done
                    ok = mbar_wait(&bar_mma, phase);
                    phase ^= 1u;
                }
#pragma unroll
                for (int i = 0; i < GRP; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<uint4*>(op_at(Zs + i * OP64, q8, srow + 32 * j)) = mask_bf16x8(z[i][j], mk[i][j]);
                // (the copies of X are not waited for here)
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                tc_fence_before();
                __syncthreads();
                tc_fence_after();
                if (tid == 0) {
#pragma unroll
                    for (int i = 0; i < GRP; ++i) mma_input<HD>(tmem, Zs + i * OP64, Ws, grp + i > 0);
                    tc_commit(&bar_mma);
                }
                if (grp == 0) load(GRP);
            }
            lookup(tile + gridDim.x, which ^ 1);
            // the node's FP32 rows: ds twice, dc, dh
#pragma unroll
            for (int s = POST ? 0 : 3; s < 4; ++s) {
                float4 x[4], y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = tile * TC_ROWS + srow + 32 * j;
                    const int r = s < 2 ? itab[(which * 2 + s) * TC_ROWS + srow + 32 * j] : n < nodes ? n : -1;
                    const float4* rp = reinterpret_cast<const float4*>((s < 2 ? ds : s == 2 ? dc : dh) + (size_t)max(r, 0) * HD);
                    x[j] = y[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r >= 0) {
                        x[j] = rp[q8];
                        y[j] = rp[8 + q8];
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    ga[j] = add4(ga[j], x[j]);
                    gb[j] = add4(gb[j], y[j]);
                }
            }
            ok = mbar_wait(&bar_mma, phase) && ok;
            phase ^= 1u;
            if ((failed = __syncthreads_or(!ok))) break;
            tc_fence_after();
            tmem_to_tile(Zs, tmem, warp, lane);
            tc_fence_before();
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ga[j] = add4(ga[j], *tile_f32(Zs, srow + 32 * j, q8));
                gb[j] = add4(gb[j], *tile_f32(Zs, srow + 32 * j, 8 + q8));
            }
            __syncthreads();
        }
        if (POST) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int n = tile * TC_ROWS + srow + 32 * j;
                const uint2 mk = n < nodes ? mu[n] : make_uint2(0u, 0u);
                const uint2 a = mask_f32x4(ga[j], mk.x >> (4 * q8)), b = mask_f32x4(gb[j], mk.y >> (4 * q8));
                add_db(db, a.x, a.y);
                add_db(db + 4, b.x, b.y);
                *reinterpret_cast<uint2*>(op_at(Zs, q8 >> 1, srow + 32 * j) + (q8 & 1) * 8) = a;
                *reinterpret_cast<uint2*>(op_at(Zs, 4 + (q8 >> 1), srow + 32 * j) + (q8 & 1) * 8) = b;
            }
            tc_ready(false);
            if (tid == 0) {
                mma_input<KIN>(tmem, Zs, Ws + (PRE ? W64 : 0), false);
                mma_wgrad(tdw, Xs, Zs, !first);
                tc_commit(&bar_mma);
            }
            first = false;
            ok = mbar_wait(&bar_mma, phase);
            phase ^= 1u;
            if ((failed = __syncthreads_or(!ok))) break;
            tc_fence_after();
            tmem_to_tile(Xs, tmem, warp, lane);
            tmem_to_tile(Zs, tmem + HD, warp, lane);
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = srow + 32 * j, n = tile * TC_ROWS + r;
                ga[j] = add4(ga[j], *tile_f32(Xs, r, q8));
                gb[j] = add4(gb[j], *tile_f32(Xs, r, 8 + q8));
                const float4 a = *tile_f32(Zs, r, q8), b = *tile_f32(Zs, r, 8 + q8);
                if (n >= nodes) continue;
                reinterpret_cast<uint2*>(dmo + (size_t)n * HD)[q8] = make_uint2(pack_bf2(a.x, a.y), pack_bf2(a.z, a.w));
                reinterpret_cast<uint2*>(dmo + (size_t)n * HD)[8 + q8] = make_uint2(pack_bf2(b.x, b.y), pack_bf2(b.z, b.w));
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = tile * TC_ROWS + srow + 32 * j;
            if (n >= nodes) continue;
            if (POST) {
                reinterpret_cast<float4*>(dh + (size_t)n * HD)[q8] = ga[j];
                reinterpret_cast<float4*>(dh + (size_t)n * HD)[8 + q8] = gb[j];
            } else {                                        // orientation of n: bit 2, this warp's lowest
                add_f4(db, ga[j]);
                add_f4(db + 4, gb[j]);
            }
        }
        __syncthreads();                                    // the tiles are read: the next staging
    }
    if (POST && !failed) {
        dw_partial(tdw, part + (size_t)blockIdx.x * WPART, warp, lane);
        db_partial(part + (size_t)blockIdx.x * WPART, db, true, reinterpret_cast<float*>(Xs));
    }
    if (!POST && !failed) {
        float* const sm = reinterpret_cast<float*>(Zs);     // [orientation][column][16 threads]
#pragma unroll
        for (int i = 0; i < 8; ++i)
            sm[((warp & 1) * HD + (i >> 2) * 32 + q8 * 4 + (i & 3)) * 17 + (warp >> 1) * 4 + (lane >> 3)] = db[i];
        __syncthreads();
        if (tid < 2 * HD) {
            float t = 0.f;
            for (int j = 0; j < 16; ++j) t += sm[tid * 17 + j];
            part[(size_t)blockIdx.x * 2 * HD + tid] = t;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_teardown(tmem, 256, failed, err);
}

// Edges.  Messages of a layer, edge half, both directions d of an edge (msg_tab [E]: source
// node and target node * 8 + its slot of either): dZ_d = dm[target] & mask,
// de += sum_d dX_d[:, 64:] (set: =), weight gradient with X_d = [h[src_d] | e].
// POST, edge update of the layer below: dZ = de & me, de += dX[:, :64], weight gradient with
// X = [eb | h_i + h_j], whose end rows are the messages' source rows.  dX[:, 64:] (FP32) goes to
// the edge's two nodes: a tile is 8 cells (16 edges each) or 128 edges between cells;
// the former sums it for its 64 nodes (dc), the latter keeps its rows (ds), so that
// node_bwd_kernel reads 3 rows a node instead of 6.
// Operands R0 | R1 | R2: h[src_0], e, h[src_1], then (POST) eb in R1 and the sum in R2.
// J: couplers, where e (without POST) or eb is the first layer's, else NULL.
// The two directions' weight gradients differ in the order of their halves ([R0 | R1] and
// [R1 | R2]) and are kept apart in tensor memory.  Without POST (the first layer) de is not
// kept, only its sums over the edges of every coupler value, epart
// [CTA][6][64]: the finished tile goes back to shared memory and a thread adds up a
// column of 32 rows, a row's class being the same for the whole warp.
__host__ __device__ inline int edge_tiles_in(int graphs, int N) { return (graphs * (N / 8) + 7) / 8; }
__host__ __device__ inline int edge_tiles_between(int graphs, int N, int E) { return (graphs * (E - 2 * N) + TC_ROWS - 1) / TC_ROWS; }
constexpr int TC_SMEM_EDGE_BWD = 5 * OP64 + 3 * W64;
template <bool POST>
__global__ void __launch_bounds__(TC_THREADS, TC_CTAS_BWD)
edge_bwd_kernel(int graphs, int N, int E, const int4* __restrict__ msg_tab, const uint2* mm, const bf16* dm,
                const bf16* h, const bf16* e, const bf16* __restrict__ WmT, float* de, int set,
                const uint2* me, const bf16* eb, const bf16* __restrict__ WeT, float* __restrict__ ds, float* __restrict__ dc,
                float* __restrict__ partm, float* __restrict__ parte, const int8_t* __restrict__ J, float* __restrict__ epart, int* err)
{
    extern __shared__ __align__(128) unsigned char tc_smem[];
    unsigned char *const R0 = tc_smem, *const R1 = R0 + OP64, *const R2 = R1 + OP64, *const Zs = R2 + OP64, *const Ws = Zs + 2 * OP64;
    __shared__ __align__(8) uint64_t bar_w, bar_mma;
    __shared__ uint32_t tmem_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q8 = lane & 7, srow = warp * 4 + (lane >> 3);
    bool failed = !tc_setup(&tmem_sh, &bar_w, &bar_mma, 256, Ws, WmT, W64, WeT, POST ? 2 * W64 : 0);
    const uint32_t tmem = tmem_sh;                          // dX, then dWm^T of direction 0 and 1, dWe^T: 64 columns each
    const int nin = edge_tiles_in(graphs, N), ntiles = nin + edge_tiles_between(graphs, N, E), nodes = graphs * N;
    // this and the next tile: source row, target row * 8 + slot, twice; edge row, -1: none
    __shared__ int4 tab[2][TC_ROWS];
    __shared__ int erow[2][TC_ROWS];
    __shared__ int xrow[2][TC_ROWS];                        // row of e (without POST: the first layer's, a coupler class) or of eb
    float sj[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float dbm[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, dbe[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t phase = 0;
    bool first = true;
    auto lookup = [&](int t, int which) {
        if (t >= ntiles || tid >= TC_ROWS) return;
        const bool in = t < nin;
        const int per = in ? N / 8 : E - 2 * N, g = in ? t * 8 + (tid >> 4) : (t - nin) * TC_ROWS + tid;     // cells, edges between them
        int4 v = make_int4(0, 0, 0, 0);
        int r = -1;
        if (g < graphs * per) {
            const int b = g / per, l = in ? (g - b * per) * 16 + (tid & 15) : 2 * N + g - b * per;
            v = msg_tab[l];
            v = make_int4(POST ? b * N + v.x : orientation(v.x), b * N * 8 + v.y, POST ? b * N + v.z : orientation(v.z), b * N * 8 + v.w);
            r = b * E + l;
        }
        tab[which][tid] = v;
        erow[which][tid] = r;
        xrow[which][tid] = r < 0 ? 0 : J ? coupler_class(J[r]) : r;
    };
    lookup(blockIdx.x, 0);
    __syncthreads();
    pass_begin();
    int which = 0;
    for (int tile = blockIdx.x; !failed && tile < ntiles; tile += gridDim.x, which ^= 1) {
        int4 ent[4];
        int er[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            ent[j] = tab[which][srow + 32 * j];
            er[j] = erow[which][srow + 32 * j];
        }
        lookup(tile + gridDim.x, which ^ 1);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int row = srow + 32 * j;
            const bool v = er[j] >= 0;
            cp_async16_l1(op_at(R0, q8, row), h + (size_t)ent[j].x * HD + q8 * 8, v);
            cp_async16(op_at(R1, q8, row), e + (size_t)(POST ? max(er[j], 0) : xrow[which][row]) * HD + q8 * 8, v, !POST);
            cp_async16_l1(op_at(R2, q8, row), h + (size_t)ent[j].z * HD + q8 * 8, v);
        }
        uint4 z0[4], z1[4];                                 // every load before the first use
        uint32_t m0[4], m1[4];
        float4 ga[4], gb[4];                                // de: columns 4 q8 .. and 32 + 4 q8 ..
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            z0[j] = z1[j] = make_uint4(0u, 0u, 0u, 0u);
            m0[j] = m1[j] = 0u;
            ga[j] = gb[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (er[j] >= 0) {
                const size_t r = er[j], n0 = ent[j].y >> 3, n1 = ent[j].w >> 3;
                z0[j] = *reinterpret_cast<const uint4*>(dm + n0 * HD + q8 * 8);
                z1[j] = *reinterpret_cast<const uint4*>(dm + n1 * HD + q8 * 8);
                m0[j] = mask_byte(mm, (size_t)(ent[j].y & 7) * nodes + n0, q8);
                m1[j] = mask_byte(mm, (size_t)(ent[j].w & 7) * nodes + n1, q8);
                if (!set) {
                    ga[j] = reinterpret_cast<const float4*>(de + r * HD)[q8];
                    gb[j] = reinterpret_cast<const float4*>(de + r * HD)[8 + q8];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            z0[j] = mask_bf16x8(z0[j], m0[j]);
            z1[j] = mask_bf16x8(z1[j], m1[j]);
            add_db(dbm, z0[j].x, z0[j].y);
            add_db(dbm + 4, z0[j].z, z0[j].w);
            add_db(dbm, z1[j].x, z1[j].y);
            add_db(dbm + 4, z1[j].z, z1[j].w);
            *reinterpret_cast<uint4*>(op_at(Zs, q8, srow + 32 * j)) = z0[j];
            *reinterpret_cast<uint4*>(op_at(Zs + OP64, q8, srow + 32 * j)) = z1[j];
        }
        tc_ready(false);
        if (tid == 0) {
            mma_input<HD>(tmem, Zs, Ws, false);
            mma_input<HD>(tmem, Zs + OP64, Ws, true);
            mma_wgrad(tmem + HD, R0, Zs, !first);
            mma_wgrad(tmem + 2 * HD, R1, Zs + OP64, !first);
            tc_commit(&bar_mma);
        }
        bool ok = mbar_wait(&bar_mma, phase);
        phase ^= 1u;
        if ((failed = __syncthreads_or(!ok))) break;
        tc_fence_after();
        if (POST) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = srow + 32 * j;
                cp_async16(op_at(R1, q8, row), eb + (size_t)xrow[which][row] * HD + q8 * 8, er[j] >= 0, J != nullptr);
                uint4* const s = reinterpret_cast<uint4*>(op_at(R2, q8, row));
                *s = add_bf16x8(*reinterpret_cast<const uint4*>(op_at(R0, q8, row)), *s);
            }
        }
        tmem_to_tile(Zs, tmem, warp, lane);
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            ga[j] = add4(ga[j], *tile_f32(Zs, srow + 32 * j, q8));
            gb[j] = add4(gb[j], *tile_f32(Zs, srow + 32 * j, 8 + q8));
        }
        if (POST) {
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = srow + 32 * j;
                const uint2 k = er[j] >= 0 ? me[er[j]] : make_uint2(0u, 0u);
                const uint2 a = mask_f32x4(ga[j], k.x >> (4 * q8)), b = mask_f32x4(gb[j], k.y >> (4 * q8));
                add_db(dbe, a.x, a.y);
                add_db(dbe + 4, b.x, b.y);
                *reinterpret_cast<uint2*>(op_at(Zs, q8 >> 1, row) + (q8 & 1) * 8) = a;
                *reinterpret_cast<uint2*>(op_at(Zs, 4 + (q8 >> 1), row) + (q8 & 1) * 8) = b;
            }
            tc_ready(false);
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (tid == 0) {
                    mma_input<HD>(tmem, Zs, Ws + (1 + half) * W64, false);
                    if (half == 0) mma_wgrad(tmem + 3 * HD, R1, Zs, !first);
                    tc_commit(&bar_mma);
                }
                ok = mbar_wait(&bar_mma, phase);
                phase ^= 1u;
                if ((failed = __syncthreads_or(!ok))) break;      // also: the other half's tile is read
                tc_fence_after();
                tmem_to_tile(R0, tmem, warp, lane);
                tc_fence_before();
                __syncthreads();
                tc_fence_after();
                if (half == 0) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        ga[j] = add4(ga[j], *tile_f32(R0, srow + 32 * j, q8));
                        gb[j] = add4(gb[j], *tile_f32(R0, srow + 32 * j, 8 + q8));
                    }
                } else if (tile < nin) {                    // node 8 c + 4 u + k of the tile: edges 16 c + 4 k + k' (u = 0), 16 c + 4 k' + k
                    const int c = tid & 15;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int nd = (tid >> 4) + 16 * i, step = nd & 4 ? 4 : 1, first_row = (nd >> 3) * 16 + (nd & 3) * (nd & 4 ? 1 : 4);
                        float4 x = *tile_f32(R0, first_row, c);
#pragma unroll
                        for (int k = 1; k < 4; ++k) x = add4(x, *tile_f32(R0, first_row + k * step, c));
                        if (tile * 64 + nd < nodes) reinterpret_cast<float4*>(dc + (size_t)(tile * 64 + nd) * HD)[c] = x;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int row = srow + 32 * j;
                        const float4 a = *tile_f32(R0, row, q8), b = *tile_f32(R0, row, 8 + q8);
                        if (er[j] < 0) continue;
                        float4* const dp = reinterpret_cast<float4*>(ds + ((size_t)(tile - nin) * TC_ROWS + row) * HD);
                        dp[q8] = a;
                        dp[8 + q8] = b;
                    }
                }
            }
            if (failed) break;
        }
        first = false;
        if (POST) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (er[j] >= 0) {
                    reinterpret_cast<float4*>(de + (size_t)er[j] * HD)[q8] = ga[j];
                    reinterpret_cast<float4*>(de + (size_t)er[j] * HD)[8 + q8] = gb[j];
                }
        } else {
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {                   // the places that this thread has read
                *tile_f32(Zs, srow + 32 * j, q8) = er[j] >= 0 ? ga[j] : zero;
                *tile_f32(Zs, srow + 32 * j, 8 + q8) = er[j] >= 0 ? gb[j] : zero;
            }
            __syncthreads();
            const int c = tid & (HD - 1);
#pragma unroll 8
            for (int i = 0; i < 32; ++i) {
                const int row = (tid >> 6) * 32 + i, k = xrow[which][row];
                const float v = reinterpret_cast<const float*>(tile_f32(Zs, row, c >> 2))[c & 3];
#pragma unroll
                for (int q = 0; q < 6; ++q) sj[q] += k == q ? v : 0.f;
            }
        }
        __syncthreads();                                    // the tiles are read: the next staging
    }
    if (!POST && !failed) {
        float* const sm = reinterpret_cast<float*>(Zs);     // [row group][value][column]
#pragma unroll
        for (int q = 0; q < 6; ++q) sm[((tid >> 6) * 6 + q) * HD + (tid & (HD - 1))] = sj[q];
        __syncthreads();
        for (int i = tid; i < 6 * HD; i += TC_THREADS)
            epart[(size_t)blockIdx.x * 6 * HD + i] = (sm[i] + sm[6 * HD + i]) + (sm[12 * HD + i] + sm[18 * HD + i]);
    }
    if (!failed) {
        // dWm^T: direction 1 has its halves (TMEM lanes) exchanged; it goes through shared memory, [column][input]
        float* const P = partm + (size_t)blockIdx.x * WPART;
        float* const sm = reinterpret_cast<float*>(tc_smem);     // R0, R1: not the sums above
        const int q = warp & 3, in = q * 32 + lane, cb = (warp >> 2) * (HD / 2);
        const uint32_t tl = tmem + HD + ((uint32_t)(q * 32) << 16) + cb;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float d[16];
            tmem_ld16(tl + HD + 16 * hh, d);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) sm[(cb + 16 * hh + i) * KIN + (in ^ HD)] = d[i];
        }
        __syncthreads();
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float d[16];
            tmem_ld16(tl + 16 * hh, d);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) P[(cb + 16 * hh + i) * KIN + in] = d[i] + sm[(cb + 16 * hh + i) * KIN + in];
        }
        db_partial(P, dbm, false, sm);
        if (POST) {
            dw_partial(tmem + 3 * HD, parte + (size_t)blockIdx.x * WPART, warp, lane);
            db_partial(parte + (size_t)blockIdx.x * WPART, dbe, true, sm);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_teardown(tmem, 256, failed, err);
}

// Every sum over CTAs or graphs that is left of a gradient, in one launch (blockIdx.y): the
// partials of up to 26 parameter blocks (weight maps with their biases, embeddings; no
// partials: 0), then the readout's.  16 columns of 16 bytes x 16 threads that each take
// every 16th partial, added in a fixed order (bit-reproducible).  11 maps of 304 partials
// (110 MB, 256 C_8 graphs) in 26 us with the readout's sums; one thread per output in order
// took 35 us, the readout's 18 us and the embeddings' 117 us in launches of their own.
constexpr int MAXPARTS = 27;
struct Parts {
    float* dst[MAXPARTS];
    const float* src[MAXPARTS];
    int n[MAXPARTS], count[MAXPARTS];        // partials; floats of one
    int blocks;
};
// Readout: dW1[c][k] = sum_b dz_b[c] g_b[k] with dz_b[c] = dy_b w2[c] where z_b[c] > 0, db1[c],
// dw2[c] (block c < 64); db2 and the loss (block 64).
struct ReadoutGrad {
    int B;
    const float *g, *z, *dy, *sq, *w2;
    float *loss, *dW1, *db1, *dw2, *db2;
};

__device__ void readout_grad(const ReadoutGrad& r, float* sm)
{
    const int c = blockIdx.x, tid = threadIdx.x, k = tid & (HD - 1), grp = tid >> 6;
    if (c < HD) {
        const float w = r.w2[c];
        float acc = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll 4
        for (int b = grp; b < r.B; b += 4) {
            const float z = r.z[b * HD + c], dy = r.dy[b];
            const float dz = z > 0.f ? dy * w : 0.f;
            acc += dz * r.g[b * HD + k];
            a1 += dz;
            a2 += dy * fmaxf(z, 0.f);
        }
        sm[tid] = acc;
        if (k == 0) {
            sm[256 + grp] = a1;
            sm[260 + grp] = a2;
        }
        __syncthreads();
        if (tid < HD) r.dW1[c * HD + k] = (sm[k] + sm[64 + k]) + (sm[128 + k] + sm[192 + k]);
        if (tid == 0) {
            r.db1[c] = (sm[256] + sm[257]) + (sm[258] + sm[259]);
            r.dw2[c] = (sm[260] + sm[261]) + (sm[262] + sm[263]);
        }
    } else if (c == HD && tid < 2) {         // in graph order
        const float* x = tid == 0 ? r.dy : r.sq;
        float t = 0.f;
#pragma unroll 8
        for (int b = 0; b < r.B; ++b) t += x[b];
        *(tid == 0 ? r.db2 : r.loss) = t;
    }
}

constexpr int RED_THREADS = 256, RED_COLS = 16, RED_PER = RED_THREADS / RED_COLS;
__global__ void __launch_bounds__(RED_THREADS) reduce_kernel(Parts p, ReadoutGrad r)
{
    __shared__ float4 sm[RED_PER][RED_COLS + 1];
    const int k = blockIdx.y;
    pass_begin();
    if (k == p.blocks) {
        readout_grad(r, reinterpret_cast<float*>(sm));
        return;
    }
    const int q = p.count[k] / 4, c = threadIdx.x % RED_COLS, g = threadIdx.x / RED_COLS, i = blockIdx.x * RED_COLS + c, n = p.n[k];
    if (blockIdx.x * RED_COLS >= q) return;
    float4 s[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < q) {
        const float4* src = reinterpret_cast<const float4*>(p.src[k]) + i;
        int b = g;
        for (; b + 3 * RED_PER < n; b += 4 * RED_PER) {
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = src[(size_t)(b + j * RED_PER) * q];
#pragma unroll
            for (int j = 0; j < 4; ++j) s[j] = add4(s[j], v[j]);
        }
        for (; b < n; b += RED_PER) s[0] = add4(s[0], src[(size_t)b * q]);
    }
    sm[g][c] = add4(add4(s[0], s[1]), add4(s[2], s[3]));
    __syncthreads();
    if (g == 0 && i < q) {
        float4 t = sm[0][c];
#pragma unroll
        for (int j = 1; j < RED_PER; ++j) t = add4(t, sm[j][c]);
        reinterpret_cast<float4*>(p.dst[k])[i] = t;
    }
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
// readout forward + loss gradient dg, the same for every node of a graph (one block of 256
// threads per graph).  The node mean is summed node by node (64 threads, a column each) from
// rows that the block stages 64 at a time, the next 64 on their way meanwhile; W1 is staged
// while the last layer runs.  64 C_8 predictions 150 -> 140 us with W1 and the rows' second
// buffer (a barrier per 64 rows), of which W1 8 us.
constexpr int RO_ROWS = 64, RO_THREADS = 256;
__global__ void __launch_bounds__(RO_THREADS) readout_kernel(int N, const bf16* h, const float* __restrict__ W1, const float* __restrict__ b1,
                               const float* __restrict__ w2, const float* __restrict__ b2, float* y, float* gbuf,
                               float* zbuf, const float* __restrict__ target, float inv_B, float* dybuf,
                               float* sqbuf, float* dgbuf, const volatile int* err)
{
    __shared__ __align__(16) float gs[HD];
    __shared__ float as[HD], red[HD], dz[HD];
    __shared__ __align__(16) bf16 rows[2][RO_ROWS][HD];
    __shared__ float W[HD][HD + 1];                         // W1, loaded before the wait for the last layer
    const int b = blockIdx.x, tid = threadIdx.x, c = tid;
    for (int i = tid; i < HD * HD; i += RO_THREADS) W[i / HD][i % HD] = W1[i];
    const float b1c = c < HD ? b1[c] : 0.f, w2c = c < HD ? w2[c] : 0.f, b20 = b2[0];
    pass_begin();
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
    for (int n0 = 0, buf = 0; n0 < N; n0 += RO_ROWS, buf ^= 1) {
#pragma unroll
        for (int j = 0; j < PER; ++j) reinterpret_cast<uint4*>(&rows[buf][0][0])[tid + j * RO_THREADS] = v[j];
        __syncthreads();                                    // the other buffer's rows are summed
        if (n0 + RO_ROWS < N) fetch(n0 + RO_ROWS);
        if (c < HD) {
            const int m = min(RO_ROWS, N - n0);
#pragma unroll 8
            for (int n = 0; n < m; ++n) acc += __bfloat162float(rows[buf][n][c]);
        }
    }
    if (c < HD) gs[c] = acc / (float)N;
    __syncthreads();
    float z = 0.f;
    if (c < HD) {
        z = b1c;
        for (int k = 0; k < HD; ++k) z += W[c][k] * gs[k];
        as[c] = fmaxf(z, 0.f);
        red[c] = as[c] * w2c;
        gbuf[b * HD + c] = gs[c];
        zbuf[b * HD + c] = z;
    }
    __syncthreads();
    for (int s = HD / 2; s > 0; s >>= 1) {
        if (c < s) red[c] += red[c + s];
        __syncthreads();
    }
    const float yb = red[0] + b20;
    if (c == 0) y[b] = yb;
    if (b == 0 && c == 1) reinterpret_cast<int*>(y)[gridDim.x] = *err;      // the status of the kernels before
    if (!target) return;
    const float dy = 2.f * (yb - target[b]) * inv_B;
    if (c == 0) {                                  // this graph's loss term and output gradient (summed in order
        dybuf[b] = dy;                             // over graphs by readout_grad)
        sqbuf[b] = (yb - target[b]) * (yb - target[b]) * inv_B;
    }
    if (c < HD) dz[c] = z > 0.f ? dy * w2c : 0.f;
    __syncthreads();
    if (c < HD) {
        float dg = 0.f;
        for (int o = 0; o < HD; ++o) dg += dz[o] * W[o][c];
        dgbuf[b * HD + c] = dg / (float)N;
    }
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
    int* d_err = nullptr;         // the word after dloss, set by a tensor-core kernel whose bounded wait ran out
    int sms = 0;                  // SMs of the device (persistent grids)
    int64_t step = 0;
    // offsets into theta
    int64_t oX = 0, oJ = 0, oW1 = 0, ob1 = 0, ow2 = 0, ob2 = 0;
    std::vector<int64_t> oWm, obm, oWu, obu, oWe, obe;
    // graph + activation buffers for the current (L, Bcap)
    int L = 0, N = 0, E = 0, Bcap = 0;
    int *d_inter = nullptr, *d_out_tab = nullptr;   // topology tables (see the kernels)
    int2 *d_ends = nullptr, *d_in_tab = nullptr;
    int4* d_msg_tab = nullptr;
    int8_t* d_J = nullptr;
    float *d_t = nullptr, *d_y = nullptr, *d_g = nullptr, *d_z = nullptr;
    float *d_dy = nullptr, *d_sq = nullptr;   // per graph: output gradient, loss term (readout)
    float* d_dg = nullptr;                    // per graph: readout's gradient of a node [64]
    float* d_epart = nullptr;                 // embedding-gradient partials: edges [CTAs][6][64], then nodes [CTAs][2][64]
    std::vector<bf16*> h, e, m;
    std::vector<uint2*> mm, mu, me;   // per layer: sign bits of the message, node and edge pre-activations
    float *dh = nullptr, *de = nullptr, *ds = nullptr, *dc = nullptr;
    bf16* dm[2] = {nullptr, nullptr};         // messages' gradient of this layer and of the one below
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
    cudaFree(M->d_inter); cudaFree(M->d_out_tab);
    cudaFree(M->d_ends); cudaFree(M->d_in_tab); cudaFree(M->d_msg_tab);
    M->d_inter = M->d_out_tab = nullptr;
    M->d_ends = M->d_in_tab = nullptr;
    M->d_msg_tab = nullptr;
    cudaFree(M->d_J); M->d_J = nullptr;
    float** fl[] = {&M->d_t, &M->d_y, &M->d_g, &M->d_z, &M->d_dy, &M->d_sq, &M->d_dg, &M->d_epart, &M->dh, &M->de, &M->ds, &M->dc, &M->wpart};
    for (float** p : fl) { cudaFree(*p); *p = nullptr; }
    for (bf16*& p : M->dm) { cudaFree(p); p = nullptr; }
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

// Persistent CTAs for `rows` rows at ctas_per_sm residents.
int tc_grid(const sg_model* M, int rows, int ctas_per_sm)
{
    const int tiles = (rows + TC_ROWS - 1) / TC_ROWS, cap = ctas_per_sm * M->sms;
    return tiles < cap ? (tiles > 0 ? tiles : 1) : cap;
}

int edge_grid(const sg_model* M, int B, int N, int E)
{
    return tc_grid(M, (edge_tiles_in(B, N) + edge_tiles_between(B, N, E)) * TC_ROWS, TC_CTAS_BWD);
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
    // messages 2e: source ej -> target ei, 2e + 1: source ei -> target ej.  A node's incoming and outgoing
    // messages fill its 6 slots in ascending order, its edges between cells (numbers 16 L^2 and up) 2;
    // tables are slot-major [6][N], [2][N]
    std::vector<int> inter(2 * N, -1), out_tab(N * MAXDEG, -1);
    std::vector<int2> ends(E), in_tab(N * MAXDEG, make_int2(-1, -1));
    std::vector<int4> msg_tab(E);
    std::vector<int> cin(N, 0), cout(N, 0), cinc(N, 0);
    for (int e2 = 0; e2 < E; ++e2) {
        ends[e2] = make_int2(ei[e2], ej[e2]);
        int at[2];
        for (int d = 0; d < 2; ++d) {
            const int src = d == 0 ? ej[e2] : ei[e2], tgt = d == 0 ? ei[e2] : ej[e2], slot = cin[tgt]++;
            in_tab[slot * N + tgt] = make_int2(src, e2);
            at[d] = tgt * 8 + slot;
            out_tab[cout[src]++ * N + src] = at[d];
        }
        msg_tab[e2] = make_int4(ej[e2], at[0], ei[e2], at[1]);
        if (e2 < 2 * N) continue;
        inter[cinc[ei[e2]]++ * N + ei[e2]] = e2 - 2 * N;
        inter[cinc[ej[e2]]++ * N + ej[e2]] = e2 - 2 * N;
    }
    auto up = [&](auto** d, const auto& v) -> cudaError_t {
        cudaError_t r = salloc(d, v.size());
        if (r != cudaSuccess) return r;
        return cudaMemcpy(*d, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice);
    };
    SK(up(&M->d_inter, inter), "upload topology");
    SK(up(&M->d_out_tab, out_tab), "upload topology");
    SK(up(&M->d_ends, ends), "upload topology");
    SK(up(&M->d_in_tab, in_tab), "upload topology");
    SK(up(&M->d_msg_tab, msg_tab), "upload topology");
    const size_t nN = (size_t)B * N, nE = (size_t)B * E;
    SK(salloc(&M->d_J, nE), "cudaMalloc J");
    SK(salloc(&M->d_t, (size_t)B), "cudaMalloc t");
    SK(salloc(&M->d_y, (size_t)B + 1), "cudaMalloc y");
    SK(salloc(&M->d_g, (size_t)B * HD), "cudaMalloc g");
    SK(salloc(&M->d_z, (size_t)B * HD), "cudaMalloc z");
    SK(salloc(&M->d_dy, (size_t)B), "cudaMalloc dy");
    SK(salloc(&M->d_sq, (size_t)B), "cudaMalloc sq");
    SK(salloc(&M->d_dg, (size_t)B * HD), "cudaMalloc dg");
    M->h.assign(M->layers + 1, nullptr);
    for (auto* v : {&M->e, &M->m}) v->assign(M->layers, nullptr);
    for (auto* v : {&M->mm, &M->mu, &M->me}) v->assign(M->layers, nullptr);
    for (int l = 1; l <= M->layers; ++l) SK(salloc(&M->h[l], nN * HD), "cudaMalloc h");      // the first layer's are embedding rows
    for (int l = 0; l < M->layers; ++l) {
        if (l > 0) SK(salloc(&M->e[l], nE * HD), "cudaMalloc e");
        SK(salloc(&M->m[l], nN * HD), "cudaMalloc m");
        SK(salloc(&M->mm[l], nN * MAXDEG), "cudaMalloc message mask");
        SK(salloc(&M->mu[l], nN), "cudaMalloc node mask");
        if (l + 1 < M->layers) SK(salloc(&M->me[l], nE), "cudaMalloc edge mask");
    }
    M->wcap = edge_grid(M, B, N, E);
    SK(salloc(&M->d_epart, (size_t)M->wcap * 8 * HD), "cudaMalloc embedding partials");
    SK(salloc(&M->wpart, (size_t)3 * M->layers * M->wcap * WPART), "cudaMalloc wpart");
    SK(salloc(&M->dh, nN * HD), "cudaMalloc dh");
    for (bf16*& p : M->dm) SK(salloc(&p, nN * HD), "cudaMalloc dm");
    SK(salloc(&M->de, nE * HD), "cudaMalloc de");
    SK(salloc(&M->ds, (size_t)B * (E - 2 * N) * HD), "cudaMalloc ds");
    SK(salloc(&M->dc, nN * HD), "cudaMalloc dc");
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

// Features that enter layer l; the first layer's are the embedding tables.
const bf16* feat_h(const sg_model* M, int l) { return l == 0 ? M->wbf + M->oX : M->h[l]; }
const bf16* feat_e(const sg_model* M, int l) { return l == 0 ? M->wbf + M->oJ : M->e[l]; }

// Just over half of the 228 KB of an SM with the 1 KB that every CTA takes, so that a CTA of the edge kernel still
// fits beside it (see launch): gradient of 32 C_8 graphs 325 -> 292 us.
constexpr int TC_SMEM_ALONE = 113 * 1024;
// One launch of a pass (see pass_begin); errors are left for cudaGetLastError.
template <class... Params, class... Args>
void launch(sg_model* M, void (*kernel)(Params...), dim3 grid, int threads, int smem, Args... args)
{
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    // CTAs that may start while the kernel before drains go where there is room first: a grid of at most one
    // CTA per SM would share SMs and leave others idle, so it takes more than half of an SM's shared memory
    c.dynamicSmemBytes = smem > 0 && 2 * (int)grid.x > M->sms && (int)grid.x <= M->sms ? std::max(smem, TC_SMEM_ALONE) : smem;
    c.stream = M->stream;
    c.attrs = &a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, args...);
    M->launches++;
}

// The last layer updates no edges: nothing after it reads them.
void forward(sg_model* M, int B, bool train)
{
    const int N = M->N, E = M->E;
    for (int l = 0; l < M->layers; ++l) {
        launch(M, node_fwd_kernel, tc_grid(M, B * N, TC_CTAS_NODE_FWD), TC_THREADS, TC_SMEM_NODE_FWD,
            B * N, N, E, M->d_in_tab, feat_h(M, l), feat_e(M, l), wpk_fwd(M, l, 0), M->theta + M->obm[l], wpk_fwd(M, l, 1), M->theta + M->obu[l],
            M->h[l + 1], train ? M->m[l] : nullptr, M->mm[l], M->mu[l], l == 0 ? M->d_J : nullptr,
            M->d_err);
        if (l + 1 == M->layers) break;
        const bool few = (B * E + TC_ROWS - 1) / TC_ROWS <= EDGE_FWD_FEW * M->sms;
        launch(M, few ? edge_fwd_kernel<3> : edge_fwd_kernel<4>, tc_grid(M, B * E, few ? 3 : 4), TC_THREADS, TC_SMEM_EDGE_FWD,
            B * E, feat_e(M, l), M->h[l + 1], M->d_ends, N, E, wpk_fwd(M, l, 2), M->theta + M->obe[l], M->e[l + 1],
            train ? M->me[l] : nullptr, l == 0 ? M->d_J : nullptr, M->d_err);
    }
}

// Predictions; train: also the loss terms and the gradient of every graph's nodes.
void readout(sg_model* M, int B, bool train)
{
    launch(M, readout_kernel, B, RO_THREADS, 0, M->N, M->h[M->layers], M->theta + M->oW1, M->theta + M->ob1, M->theta + M->ow2,
           M->theta + M->ob2, M->d_y, M->d_g, M->d_z, train ? M->d_t : nullptr, 1.f / (float)B, M->d_dy, M->d_sq, M->d_dg, M->d_err);
}

// Gradient of the mean squared error into M->grad; loss into M->dloss.
void backward_all(sg_model* M, int B)
{
    const int N = M->N, E = M->E;
    float* G = M->grad;
    readout(M, B, true);
    Parts parts;
    parts.blocks = 0;
    auto sum = [&](int64_t o, const float* src, int n, int count) {
        parts.dst[parts.blocks] = G + o;
        parts.src[parts.blocks] = src;
        parts.n[parts.blocks] = n;
        parts.count[parts.blocks++] = count;
    };
    int nmaps = 0;
    auto map = [&](int64_t oW, int n) {                  // the next map's partials: the matrix, then its bias
        float* p = M->wpart + (size_t)M->wcap * WPART * nmaps++;
        sum(oW, p, n, WPART);
        return p;
    };
    // layer l's node update; then per layer its messages with the updates of the layer below
    const int top = M->layers - 1, gn = tc_grid(M, B * N, TC_CTAS_BWD), ge = edge_grid(M, B, N, E);
    const size_t nodes = (size_t)B * N;
    float* const nepart = M->d_epart + (size_t)M->wcap * 6 * HD;
    auto node = [&](int l, auto kernel, int smem) {      // messages of layer l (if any), update of layer l - 1 (if any)
        const bool pre = l <= top, post = l > 0;
        launch(M, kernel, gn, TC_THREADS, smem,
            (int)nodes, N, E, pre ? M->d_out_tab : nullptr, pre ? M->mm[l] : nullptr, M->dm[l & 1], pre ? wpk_bwd(M, l, 0) : nullptr,
            pre && post ? M->d_inter : nullptr, M->dc, M->ds, M->d_dg, M->dh, post ? M->mu[l - 1] : nullptr, post ? feat_h(M, l - 1) : nullptr,
            post ? M->m[l - 1] : nullptr, post ? wpk_bwd(M, l - 1, 1) : nullptr, M->dm[(l & 1) ^ 1],
            post ? map(M->oWu[l - 1], gn) : nepart, l == 1 ? 1 : 0, M->d_err);
    };
    auto edge = [&](int l, auto kernel, int smem) {
        const bool post = l > 0;
        float* pm = map(M->oWm[l], ge);
        launch(M, kernel, ge, TC_THREADS, smem,
            B, N, E, M->d_msg_tab, M->mm[l], M->dm[l & 1], feat_h(M, l), feat_e(M, l), wpk_bwd(M, l, 0) + HD * HD, M->de, l == top ? 1 : 0,
            post ? M->me[l - 1] : nullptr, post ? feat_e(M, l - 1) : nullptr, post ? wpk_bwd(M, l - 1, 2) : nullptr, M->ds, M->dc, pm,
            post ? map(M->oWe[l - 1], ge) : nullptr, l <= 1 ? M->d_J : nullptr, M->d_epart, M->d_err);
    };
    node(top + 1, node_bwd_kernel<false, true>, TC_SMEM_NODE_BWD);
    for (int l = top; l > 0; --l) {
        edge(l, edge_bwd_kernel<true>, TC_SMEM_EDGE_BWD);
        node(l, node_bwd_kernel<true, true>, TC_SMEM_NODE_BWD);
    }
    edge(0, edge_bwd_kernel<false>, TC_SMEM_EDGE_BWD);
    node(0, node_bwd_kernel<true, false>, TC_SMEM_NODE_BWD);
    sum(M->oX, nepart, gn, 2 * HD);
    sum(M->oJ, M->d_epart, ge, 6 * HD);
    sum(M->oWe[top], nullptr, 0, WPART);
    const ReadoutGrad ro = {B, M->d_g, M->d_z, M->d_dy, M->d_sq, M->theta + M->ow2, M->dloss, G + M->oW1, G + M->ob1, G + M->ow2, G + M->ob2};
    launch(M, reduce_kernel, dim3((WPART / 4 + RED_COLS - 1) / RED_COLS, parts.blocks + 1), RED_THREADS, 0, parts, ro);
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
        salloc(&M->mom2, o) != cudaSuccess || salloc(&M->wbf, o) != cudaSuccess || salloc(&M->dloss, 2) != cudaSuccess) {
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
            salloc(&M->d_wptr, ptrs.size()) != cudaSuccess) {
            M->err = "cudaMalloc tensor-core operands failed";
            return bail(PT_ERR_OOM);
        }
        cudaError_t e = cudaMemcpy(M->d_wptr, ptrs.data(), sizeof(bf16*) * ptrs.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(M->wpk, 0, sizeof(bf16) * (size_t)layers * 3 * 2 * HD * KIN);
        M->d_err = reinterpret_cast<int*>(M->dloss + 1);
        if (e == cudaSuccess) e = cudaMemset(M->d_err, 0, sizeof(int));
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const struct { const void* k; int smem; } tk[] = {
            {(const void*)node_fwd_kernel, TC_SMEM_NODE_FWD},
            {(const void*)edge_fwd_kernel<3>, TC_SMEM_EDGE_FWD},
            {(const void*)edge_fwd_kernel<4>, TC_SMEM_EDGE_FWD},
            {(const void*)node_bwd_kernel<false, true>, TC_SMEM_NODE_BWD},
            {(const void*)node_bwd_kernel<true, true>, TC_SMEM_NODE_BWD},
            {(const void*)node_bwd_kernel<true, false>, TC_SMEM_NODE_BWD},
            {(const void*)edge_bwd_kernel<true>, TC_SMEM_EDGE_BWD},
            {(const void*)edge_bwd_kernel<false>, TC_SMEM_EDGE_BWD}};
        for (const auto& t : tk)
            if (e == cudaSuccess) e = cudaFuncSetAttribute(t.k, cudaFuncAttributeMaxDynamicSharedMemorySize, std::max(t.smem, TC_SMEM_ALONE));
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
    cudaFree(M->wpk); cudaFree(M->d_wptr);
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
    readout(M, B, false);
    SK(cudaGetLastError(), "forward kernels");
    float out[4096 + 1];                             // the predictions and the status word (load_batch: B <= 4096)
    SK(cudaMemcpyAsync(out, M->d_y, sizeof(float) * ((size_t)B + 1), cudaMemcpyDeviceToHost, M->stream), "download y");
    SK(cudaStreamSynchronize(M->stream), "sync forward");
    std::memcpy(y, out, sizeof(float) * B);
    int terr = 0;
    std::memcpy(&terr, out + B, sizeof terr);
    return tc_status(M, terr);
}

int sg_grad(sg_model* M, int32_t L, int32_t B, const int8_t* J, const float* t, float* loss, float* grad)
{
    if (!M || !t) return sfail(M, PT_ERR_ARG, "NULL argument");
    int rc = load_batch(M, L, B, J, t);
    if (rc) return rc;
    forward(M, B, true);
    backward_all(M, B);
    SK(cudaGetLastError(), "gradient kernels");
    if (grad) SK(cudaMemcpyAsync(grad, M->grad, sizeof(float) * M->nparams, cudaMemcpyDeviceToHost, M->stream), "download grad");
    struct { float loss; int status; } res = {0.f, 0};
    SK(cudaMemcpyAsync(&res, M->dloss, sizeof res, cudaMemcpyDeviceToHost, M->stream), "download loss and status");
    SK(cudaStreamSynchronize(M->stream), "sync grad");
    if (loss) *loss = res.loss;
    return tc_status(M, res.status);
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

// pt_lane.cuh -- the replica-lane sweep kernel (included by pt_kernels.cu).
//
// One lane = one replica (configuration buffer) of a run, at the temperature of
// the slot that holds it.  A warp updates one cell's 4 spins of a colour in 32
// replicas at once (a "warp word"), so everything that belongs to the cell is
// warp-uniform: its coupler tables, its neighbours' addresses, and the products
// of the Philox call that do not depend on the replica.  What that buys over a
// lane per cell (pt_sweep_kernel), per 4-spin word:
//   * the local fields come from three 16-entry tables (16 entries lie in 16
//     banks: no conflicts) and one add, instead of 8 dp4a on couplers loaded
//     per word;
//   * the threshold's shared address is one dp4a (byte extraction, row pitch and
//     the slot's column in one instruction), and a slot's thresholds lie in its
//     own bank; a field k <= 0 accepts through the sign of its byte;
//   * 16 wide multiplies per Philox call instead of 17, the round keys in uniform
//     registers;
//   * 2 x 2 cells a step: half of the neighbours are loaded once for two cells, and
//     loop and address instructions are shared.
// Bound: warp instruction issue.  A wide multiply holds the dispatch of its
// sub-partition for two cycles (4 on its pipe).  Measured, C_8 x 32 slots, 1024 runs
// as 16 candidates, exchange every sweep: 83.3 instructions a word with everything
// around it, 16 of them wide multiplies, so 99.3 dispatch cycles of the 122 clocks
// that a word takes on the 147 SMs in use (slot-major 4/32/1: 118 instructions, 199
// clocks); 13.2 us per sweep, 1.27e12 attempts/s (20.7 us, 8.1e11); one C_8 instance
// of 64 runs: 2.7 us per sweep (cell-major default: 11.7).
// Measured and left: 1 or 2 cells a step instead of 4 (1 % slower), keys as immediates
// (recomputed per round, 7 more uniform instructions a word), accept flags by LOP3
// instead of adds (1 % slower), by selects (2 % slower).
#pragma once

namespace ptg {
namespace {

// The terms of a group's Philox call that depend on (sweep, group) only.
__device__ __forceinline__ uint4 lane_pre(uint32_t s, int col, int q, int L, uint32_t k0, uint32_t k1)
{
    const int r = q / L, c = q - r * L, u = (r + c + col) & 1;
    const PhiloxPre p = philox_pre(s, (uint32_t)(2 * q + u), k0, k1);
    return make_uint4(p.x0b, p.z2x, p.z3, 0u);
}

// The 16 entries of one field table: `which` 0 the cell's opposite group (with the bias of 128 per byte),
// 1 / 2 the minus / plus neighbour; entry `nib` for the mask of that group's negative spins.  v: the
// group's 4 words of negated couplers (InstDesc::jw), those inside the cell for which = 0, those between
// cells otherwise, so the three entries of an update add up to 128 - h_i in byte i.  A spin's sign moves
// an entry by twice its couplers, whatever the others are: 15 additions (modulo 2^32, as the sum of the
// three) instead of 16 sums.
__device__ __forceinline__ void lane_table(uint4* out, const uint4 v, int which)
{
    uint32_t base = which == 0 ? 0x80808080u : 0u, d[4] = {0u, 0u, 0u, 0u};
    const uint32_t jw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (which == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t j = (uint32_t)(int)(int8_t)(jw[k] >> (8 * i)) << (8 * k);
                base += j;
                d[i] -= 2u * j;
            }
        } else {
            const uint32_t j = (uint32_t)(int)(int8_t)(jw[k] >> (16 * (k & 1) + 8 * (which - 1))) << (8 * k);
            base += j;
            d[k] -= 2u * j;
        }
    }
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const uint32_t e = base + (n & 1 ? d[2] : 0u) + (n & 2 ? d[3] : 0u);
        out[n] = make_uint4(e, e + d[0], e + d[1], e + d[0] + d[1]);
    }
}

// 0xFF in every byte of x whose sign bit is set, 0 in the others.
__device__ __forceinline__ uint32_t byte_signs(uint32_t x)
{
    uint32_t m;
    asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(m) : "r"(x));
    return m;
}

// The field tables of an instance.
__device__ __forceinline__ void make_tables(uint4* lut, const uint4* jw, int L2)
{
    for (int i = threadIdx.x; i < 6 * L2; i += blockDim.x) {
        const int cq = i / 3, which = i - cq * 3, c = cq >= L2, q = cq - c * L2;
        lane_table(lut + 4 * i, __ldg(jw + 4 * q + 2 * c + (which > 0)), which);
    }
}

// The thresholds, a column per slot (the columns beyond them are not used).
__device__ __forceinline__ void make_thresholds(uint32_t* out, const uint32_t* thr, int NT, int kt)
{
    for (int i = threadIdx.x; i < NT * kt; i += blockDim.x) {
        const int k = i / NT, t = i - k * NT;
        out[((t >> 5) * kt + k) * 32 + (t & 31)] = __ldg(thr + t * kt + k);
    }
}

// The same as functions of their own, for the kernels whose sweeps are faster without them in their midst (the
// compiler orders the sweep loop by what surrounds it).  Sweeps inline / apart: tables, C_4 1.27 / 1.32 us, C_16 with
// 48 slots 16.98 / 16.72; thresholds, C_4 1.27 / 1.32, C_7 2.62 / 2.61, C_13 12.37 / 12.23.
__device__ __noinline__ void make_tables_apart(uint4* lut, const uint4* jw, int L2) { make_tables(lut, jw, L2); }
__device__ __noinline__ void make_thresholds_apart(uint32_t* out, const uint32_t* thr, int NT, int kt) { make_thresholds(out, thr, NT, kt); }

// Spins of whole runs (cell by cell, buffer by buffer) between memory, where a cell has two words (orientation
// 0 and 1), and the columns of consecutive groups: word u has colour (row + column + u) & 1.  All runs at once, where
// run by run each waits for its own loads: for the small lattices, whose CTAs hold many runs (one sweep of 1000 C_2
// runs of 16 slots 23.3 -> 19.0 us).  On the others it took more from the sweep loop than it gave (C_16 with 48
// slots 15.45 -> 15.65 us a sweep).
__device__ __forceinline__ unsigned char* spin_at(unsigned char* columns, int i, int L, int per, int group_bytes, int col_bytes, int& odd)
{
    const int L2 = L * L, rb = i / L2, q = i - rb * L2, g = rb / per, p = rb - g * per, y = q / L;
    odd = (y + q - y * L) & 1;
    return columns + g * group_bytes + (p >> 5) * col_bytes + (q + L) * 32 + (p & 31);
}

__device__ __noinline__ void load_spins(unsigned char* columns, const uint2* words, int cells, int L, int per, int group_bytes, int col_bytes)
{
    constexpr int AHEAD = 4;                    // loads in flight
    for (int i0 = threadIdx.x; i0 < cells; i0 += AHEAD * blockDim.x) {
        uint2 v[AHEAD];
#pragma unroll
        for (int j = 0; j < AHEAD; ++j)
            if (i0 + j * (int)blockDim.x < cells) v[j] = words[i0 + j * (int)blockDim.x];
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) {
            const int i = i0 + j * (int)blockDim.x;
            if (i >= cells) break;
            int odd;
            unsigned char* const at = spin_at(columns, i, L, per, group_bytes, col_bytes, odd);
            at[odd ? col_bytes / 2 : 0] = (unsigned char)(((v[j].x & 0x80808080u) * 0x00204081u) >> 26);
            at[odd ? 0 : col_bytes / 2] = (unsigned char)(((v[j].y & 0x80808080u) * 0x00204081u) >> 26);
        }
    }
}

__device__ __noinline__ void store_spins(unsigned char* columns, uint2* words, int cells, int L, int per, int group_bytes, int col_bytes)
{
    for (int i = threadIdx.x; i < cells; i += blockDim.x) {
        int odd;
        const unsigned char* const at = spin_at(columns, i, L, per, group_bytes, col_bytes, odd);
        const uint32_t a = at[0], b = at[col_bytes / 2];                   // colours 0 and 1
        words[i] = make_uint2(byte_signs((odd ? b : a) * 0x04081020u) | 0x01010101u,
                              byte_signs((odd ? a : b) * 0x04081020u) | 0x01010101u);   // 0xFF or 1
    }
}

struct LaneConst {
    uint32_t c1, y2x, y1k;           // Philox: run and slot word, terms of the sweep
    uint32_t ka[7], kb[7];           // round keys of rounds 3..9
    uint32_t tcol;                   // shared address of this slot's threshold column, row k = -127
    int kt;
};

// U cells of one colour, their 4 spins each: `o` their bytes (replaced), `hb` the packed
// 128 - h_i, `pr` the cells' Philox terms.  Step by step over the cells, so that their
// chains of dependent instructions overlap.
template <int U>
__device__ __forceinline__ void lane_words(uint32_t (&o)[U], const uint32_t (&hb)[U], const uint4 (&pr)[U],
                                           const LaneConst& lc, uint32_t& dk, uint32_t& pc)
{
    uint32_t kb[U], a0[U], a1[U], a2[U], a3[U], th[U][4];
#pragma unroll
    for (int i = 0; i < U; ++i) {
        // byte j of m: 0xFF where spin j is -1 (its mask bit moved to the byte's sign, which is replicated)
        const uint32_t m = byte_signs(o[i] * 0x04081020u);
        kb[i] = (hb[i] ^ m) - (~m & 0x01010101u);                 // 127 + k, k = -s h: dE = 2 k
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // shared address of row k of the slot's column: byte j of kb times 128 plus the column
            uint32_t a = __dp4a(kb[i], 0x80u << (8 * j), lc.tcol);
#ifdef PT_DEBUG
            const int k = (int)((kb[i] >> (8 * j)) & 255u) - 127;
            if (k >= lc.kt || k <= -lc.kt) { atomicCAS(&g_pt_debug_code, 0u, 1u); a = lc.tcol + 127u * 128u; }
#endif
            asm("ld.shared.u32 %0, [%1];" : "=r"(th[i][j]) : "r"(a));
        }
    }
    // the Philox call (philox_slot) from the cell's and the sweep's terms
#pragma unroll
    for (int i = 0; i < U; ++i) {
        const uint64_t C = (uint64_t)PHILOX_M0 * (pr[i].x ^ lc.c1);
        const uint64_t F = (uint64_t)PHILOX_M1 * ((uint32_t)(C >> 32) ^ lc.y2x);
        a0[i] = (uint32_t)(F >> 32) ^ lc.y1k;
        a1[i] = (uint32_t)F;
        a2[i] = pr[i].y ^ (uint32_t)C;
        a3[i] = pr[i].z;
    }
#pragma unroll
    for (int r = 0; r < 7; ++r)
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const uint64_t p0 = (uint64_t)PHILOX_M0 * a0[i], p1 = (uint64_t)PHILOX_M1 * a2[i];
            a0[i] = (uint32_t)(p1 >> 32) ^ a1[i] ^ lc.ka[r];
            a2[i] = (uint32_t)(p0 >> 32) ^ a3[i] ^ lc.kb[r];
            a1[i] = (uint32_t)p1;
            a3[i] = (uint32_t)p0;
        }
#pragma unroll
    for (int i = 0; i < U; ++i) {
        uint32_t f = 0u;
        if (a0[i] < th[i][0]) f += 0x00000080u;
        if (a1[i] < th[i][1]) f += 0x00008000u;
        if (a2[i] < th[i][2]) f += 0x00800000u;
        if (a3[i] < th[i][3]) f += 0x80000000u;
        f = (f | ~kb[i]) & 0x80808080u;                           // k <= 0: accepted
        dk = __dp4a(kb[i], f, dk);                                // += 128 (k + 127) per accepted flip
        pc = __dp4a(f, 0x01010101u, pc);                          // += 128 per accepted flip
        o[i] ^= (f * 0x00204081u) >> 26;                          // the four flags to bits 2..5
    }
}

__device__ __forceinline__ uint32_t lane_fields(const unsigned char* lut, uint32_t in, uint32_t mn, uint32_t pl)
{
    return *reinterpret_cast<const uint32_t*>(lut + in) + *reinterpret_cast<const uint32_t*>(lut + 64 + mn) +
           *reinterpret_cast<const uint32_t*>(lut + 128 + pl);
}

// The pair of cells q, q + 1 (U = 2; q alone for U = 1) of one colour, odd L.  V = 0:
// cell q has its neighbours above and below (`up` bytes away), cell q + 1 to its left
// and right; V = 1: the other way round.  Pointers are to cell q.
template <int U, int V>
__device__ __forceinline__ void lane_pair(const unsigned char* lut, unsigned char* own, const unsigned char* opp, int up,
                                          const uint4* pre, const LaneConst& lc, uint32_t& dk, uint32_t& pc)
{
    uint32_t o[U], hb[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
        const int d = (i ^ V) & 1 ? 32 : up;
        o[i] = own[i * 32];
        hb[i] = lane_fields(lut + i * 192, opp[i * 32], opp[i * 32 - d], opp[i * 32 + d]);
    }
    uint4 pr[U];
#pragma unroll
    for (int i = 0; i < U; ++i) pr[i] = pre[i];
    lane_words<U>(o, hb, pr, lc, dk, pc);
#pragma unroll
    for (int i = 0; i < U; ++i) own[i * 32] = (unsigned char)o[i];
}

// A block of 2 x 2 cells, even row and column first: cells q, q + 1, q + L, q + L + 1.
// Two of them have their neighbours above and below, two to the left and right, and
// half of these neighbours lie in the block.
template <int COL>
__device__ __forceinline__ void lane_block(const unsigned char* lut, unsigned char* own, const unsigned char* opp, int L,
                                           const uint4* pre, const LaneConst& lc, uint32_t& dk, uint32_t& pc)
{
    const int at[4] = {0, 1, L, L + 1};
    // neighbours outside the block: of the first, second, third and fourth cell
    const int ext[4] = {COL ? -1 : -L, COL ? 1 - L : 2, COL ? 2 * L : L - 1, COL ? L + 2 : 2 * L + 1};
    uint32_t o[4], b[4], x[4], hb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o[i] = own[at[i] * 32];
        b[i] = opp[at[i] * 32];
        x[i] = opp[ext[i] * 32];
    }
    hb[0] = lane_fields(lut, b[0], x[0], COL ? b[1] : b[2]);
    hb[1] = COL ? lane_fields(lut + 192, b[1], x[1], b[3]) : lane_fields(lut + 192, b[1], b[0], x[1]);
    hb[2] = COL ? lane_fields(lut + 192 * L, b[2], b[0], x[2]) : lane_fields(lut + 192 * L, b[2], x[2], b[3]);
    hb[3] = lane_fields(lut + 192 * (L + 1), b[3], COL ? b[2] : b[1], x[3]);
    uint4 pr[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) pr[i] = pre[at[i]];
    lane_words<4>(o, hb, pr, lc, dk, pc);
#pragma unroll
    for (int i = 0; i < 4; ++i) own[at[i] * 32] = (unsigned char)o[i];
}

// One colour of a column: this warp's share of the cells.
template <int LT, int COL>
__device__ __forceinline__ void lane_phase(const unsigned char* lut, unsigned char* own, const unsigned char* opp,
                                           const uint4* pre, int w, int W, int Lr, const LaneConst& lc, uint32_t& dk,
                                           uint32_t& pc)
{
    const int L = LT ? LT : Lr;
    if (L & 1) {                                // cells alternate in orientation over all rows
        const int n = L * L / 2;
        int j = w;
        for (; j < n; j += W)
            lane_pair<2, COL>(lut + j * 384, own + j * 64, opp + j * 64, 32 * L, pre + 2 * j, lc, dk, pc);
        if (j == n) lane_pair<1, COL>(lut + j * 384, own + j * 64, opp + j * 64, 32 * L, pre + 2 * j, lc, dk, pc);
        return;
    }
    const unsigned hl = (unsigned)L / 2u;
    for (unsigned j = w; j < hl * hl; j += W) {
        const unsigned r = j / hl, q = 2u * (j + r * hl);    // block (r, j - r hl): cell (2 r, 2 (j - r hl))
        lane_block<COL>(lut + q * 192, own + q * 32, opp + q * 32, L, pre + q, lc, dk, pc);
    }
}

// The ascending exchange sweep of one run by all 32 lanes of a warp (TWO: 32 < NT <= 64,
// lane l holds slots l and l + 32).  Going up from slot 0 a configuration of energy x is
// carried along; pair p is rejected, and the configuration of slot p + 1 carried on
// instead, when its bound b_p = E_{p+1} - 2 c_p exceeds x.  What each slot then holds follows
// from the rejected pairs in parallel: slot s takes the old content of slot s + 1 when
// pair s was accepted, and otherwise the configuration carried into it, which came from
// the lowest slot of the run of accepted pairs that ends at pair s - 1.
// The rejected pairs: what is carried on from a rejection does not depend on what came
// before it, so with up to 32 slots every lane finds where its slot's configuration would
// be rejected next (31 compares, none waiting for another), and 5 doublings follow the
// chain from slot 0.  Against one chain of 31 compares and selects, run by all lanes
// alike, a sweep takes 3.4 % less with one C_8 run an SM, 2 % with full SMs, 1 % on C_4.
// With more slots that chain stays (two words of candidates would cost more than it).
// xp: scratch, padded with pairs that are never rejected.  Returns the lowest slot energy.
template <bool TWO>
__device__ __forceinline__ int lane_exchange(int32_t* Es, uint8_t* perm, uint8_t* inv, uint32_t* xacc, const int32_t* cc,
                                             int2* xp, int NT, int lane)
{
    constexpr int H = TWO ? 2 : 1;
    const int np = NT - 1, npad = (np + 7) & ~7;
    int m = INT_MAX;
    // up to 32 slots: a lane's energy, configuration and swap counter are loaded before the chain and exchanged by
    // shuffles after it, while every other warp of the group waits
    int held = 0, own = 0;
    if (!TWO) held = lane < NT ? perm[lane] : 0;
    uint32_t rej[H], count[H];
#pragma unroll
    for (int h = 0; h < H; ++h) count[h] = !TWO && lane < np ? xacc[lane] : 0u;
    if (!TWO) {
        // lane p: the energy carried on from a rejection of pair p, lane 31 the one carried into pair 0; where it is
        // rejected next; then the set of rejections that lane 31 reaches, doubling the number of hops
        int* const crit = reinterpret_cast<int*>(xp);
        own = lane < NT ? Es[lane] : INT_MAX;
        const int e = Es[lane < np ? lane + 1 : 0];                      // lane 31: Es[0]
        crit[lane] = lane < np ? e - 2 * cc[lane] : INT_MIN;
        m = __reduce_min_sync(FULL, own);
        __syncwarp();
        uint32_t hit[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int4 v = reinterpret_cast<const int4*>(crit)[i];
            if (e < v.x) hit[i & 3] |= 1u << (4 * i);
            if (e < v.y) hit[i & 3] |= 2u << (4 * i);
            if (e < v.z) hit[i & 3] |= 4u << (4 * i);
            if (e < v.w) hit[i & 3] |= 8u << (4 * i);
        }
        uint32_t later = (hit[0] | hit[1]) | (hit[2] | hit[3]);
        if (lane < 31) later &= 0xFFFFFFFEu << lane;
        int next = later ? __ffs((int)later) - 1 : 32;
        uint32_t set = lane < 31 ? 1u << lane : 0u;
#pragma unroll
        for (int r = 0; r < 4; ++r) {                                    // sets of 16 hops; the last doubling for lane 31 alone
            const uint32_t s2 = __shfl_sync(FULL, set, next);
            const int n2 = __shfl_sync(FULL, next, next);
            if (next < 32) { set |= s2; next = n2; }
        }
        const int n31 = __shfl_sync(FULL, next, 31);
        const uint32_t s31 = __shfl_sync(FULL, set, 31), far = __shfl_sync(FULL, set, n31);
        rej[0] = n31 < 32 ? s31 | far : s31;
    } else {
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int s = lane + 32 * h;
            if (s < NT) m = min(m, Es[s]);
            if (s < npad) {
                const int e = s < np ? Es[s + 1] : 0;
                xp[s] = make_int2(s < np ? e - 2 * cc[s] : INT_MIN, e);
            }
        }
        __syncwarp();
        int x = Es[0];
        const int4* x4 = reinterpret_cast<const int4*>(xp);
        int4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = x4[i];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            rej[h] = 0u;
            for (int p0 = 0; p0 < 32 && 32 * h + p0 < np; p0 += 8) {
                int4 nx[4];                        // the next eight pairs (the scratch is followed by room for them)
#pragma unroll
                for (int i = 0; i < 4; ++i) nx[i] = x4[16 * h + p0 / 2 + 4 + i];
                uint32_t r8 = 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (x < v[i].x) { x = v[i].y; r8 |= 1u << (2 * i); }
                    if (x < v[i].z) { x = v[i].w; r8 |= 2u << (2 * i); }
                }
                rej[h] |= r8 << p0;
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = nx[i];
            }
        }
    }
    // accepted pairs (pairs np and above: none)
    uint32_t acc[H];
    acc[0] = ~rej[0] & (np >= 32 ? 0xFFFFFFFFu : (1u << np) - 1u);
    if (TWO) acc[H - 1] = ~rej[H - 1] & ((1u << (np - 32)) - 1u);
    int e_new[H], b_new[H], src[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int s = lane + 32 * h;
        uint32_t below = ~acc[h] & ((1u << lane) - 1u);           // rejected pairs under s, this word
        src[h] = 32 * h + 32 - __clz((int)below);
        if (TWO && h == 1 && below == 0u) src[h] = 32 - __clz((int)~acc[0]);
        if ((acc[h] >> lane) & 1u) src[h] = s + 1;
        e_new[h] = b_new[h] = 0;
        if (s < NT) {
            e_new[h] = TWO ? Es[src[h]] : 0;
            b_new[h] = TWO ? perm[src[h]] : 0;
        }
    }
    if (TWO) m = __reduce_min_sync(FULL, m);
    else {
        e_new[0] = __shfl_sync(FULL, own, src[0]);
        b_new[0] = __shfl_sync(FULL, held, src[0]);
    }
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int s = lane + 32 * h;
        if (s < NT) {
            Es[s] = e_new[h];
            perm[s] = (uint8_t)b_new[h];
            inv[b_new[h]] = (uint8_t)s;
            if (s < np) xacc[s] = (TWO ? xacc[s] : count[h]) + ((acc[h] >> lane) & 1u);
        }
    }
    __syncwarp();
    return m;
}

// walk_update by all lanes of a warp: the hot half's copies are distinct.
__device__ __forceinline__ void walk_update_warp(const uint8_t* perm, uint32_t* whot, uint32_t* wtr, uint8_t* wst, int NT,
                                                 int lane)
{
    for (int t = NT - NT / 2 + lane; t < NT; t += 32) whot[perm[t]] += 1u;
    if (lane == 0) {
        const int c = perm[0];
        if (wst[c] == 2) wtr[c] += 1u;
        wst[c] = 1;
        const int h = perm[NT - 1];
        if (wst[h] == 1) wst[h] = 2;
    }
    __syncwarp();
}

// SWEEP: nsweeps sweeps with their exchanges, from counter sweep0 + 1 on; else one exchange with counter sweep0, which
// needs neither field and threshold tables nor spins (C_12, 24 slots, 16 runs: a call 39.5 -> 14.5 us, and the sweeps
// without its branches 2 to 3 % faster on C_4 and C_8).
template <int LT, bool SWEEP>
__device__ void process_bundle_lane(const InstDesc* __restrict__ insts, const Bundle bd, uint32_t sweep0, int nsweeps,
                                    int xevery, unsigned char* smem)
{
    const InstDesc& in0 = insts[bd.inst];
#ifdef PT_DEBUG
    if (LT && in0.L != LT) {                    // uniform per CTA: the whole CTA skips the bundle
        if (threadIdx.x == 0) atomicCAS(&g_pt_debug_code, 0u, 9u);
        return;
    }
#endif
    const int L = LT ? LT : in0.L, NT = in0.NT, L2 = L * L, N = 8 * L2, NW = 2 * L2, W = bd.sp, gr = -bd.team;
    const int ng1 = (bd.nitems + gr - 1) / gr, ngroups = ng1 + (bd.nitems2 + gr - 1) / gr, nruns = bd.nitems + bd.nitems2;
    const bool walk = in0.wstate != nullptr;
    const int kt = in0.kt;
    const LaneLayout lay = lane_layout(L, NT, kt, gr, ngroups, walk, bd.nitems2 > 0 ? 2 : 1);
    const ItemLayout rl = item_layout(0, NT, 0, walk);
    const int tid = threadIdx.x, lane = tid & 31;
    // read through a warp reduction: warp-uniform for the compiler too
    const int wid = (int)__reduce_or_sync(FULL, (unsigned)(tid >> 5));
    // this warp's group, its place in it, its column and its share of the cells
    const int gw = W * lay.ncols, grp = wid / gw, gwid = wid - grp * gw, col = gwid / W, w = gwid - col * W;
    const bool active = grp < ngroups, second = grp >= ng1 && active;
    const InstDesc& in = second ? insts[bd.inst2] : in0;
    const uint32_t k0 = __reduce_or_sync(FULL, in.seed), k1 = __reduce_or_sync(FULL, in.uid);
    const int done = (second ? grp - ng1 : grp) * gr;                // its instance's runs before the group's
    const int nit = active ? min(gr, (second ? bd.nitems2 : bd.nitems) - done) : 0;      // runs of the group
    const int rep = col * 32 + lane;
    const bool valid = rep < nit * NT, busy = col * 32 < nit * NT;   // busy: the column holds a replica
    const int item = valid ? rep / NT : 0, buf = valid ? rep - item * NT : 0;

    auto group_base = [&](int g) { return smem + lay.groups + g * lay.group_bytes; };
    auto run_base = [&](int g, int i) { return group_base(g) + lay.runs + i * lay.run_bytes; };
    unsigned char* const gb = group_base(active ? grp : 0);
    const int grun = (second ? 0 : bd.run0) + done;                  // the group's first run
    int32_t* xoff_sm = reinterpret_cast<int32_t*>(smem + lay.xtab);
    uint4* pre = reinterpret_cast<uint4*>(gb);
    auto gsync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(gw * 32) : "memory"); };
    const int n_iter = SWEEP ? nsweeps : 1;
    const uint32_t s_first = SWEEP ? sweep0 + 1u : sweep0;
    const uint32_t* const xthr = in0.xthr;
    // sweeps to the next exchange, counted down from sweep s_first on (0: exchange after that sweep)
    const bool xon = NT > 1 && (!SWEEP || xevery > 0);
    const uint32_t xper = !SWEEP || xevery < 1 ? 1u : (uint32_t)xevery;
    uint32_t xwait = (xper - s_first % xper) % xper;
    if (!SWEEP) xwait = 0u;

    // run r of the bundle: its instance, its run there, and its place in shared memory
    auto inst_of = [&](int r) -> const InstDesc& { return r < bd.nitems ? in0 : insts[bd.inst2]; };
    auto run_of = [&](int r) { return r < bd.nitems ? bd.run0 + r : r - bd.nitems; };
    auto slot_of = [&](int r) { return r < bd.nitems ? r : ng1 * gr + r - bd.nitems; };      // group * gr + place

    // ---- tables, then this bundle's runs
    for (int p = tid; p < NT; p += blockDim.x) {
        xoff_sm[p] = in0.xoff[p];
        reinterpret_cast<float*>(xoff_sm + NT)[p] = p < NT - 1 ? in0.xhint[p] : 0.0f;
    }
    constexpr bool FLAT = LT == 2;              // staging over all groups and runs at once
    if (SWEEP) {
        uint4* lut = reinterpret_cast<uint4*>(smem + lay.lut);
        for (int s = 0; s < (bd.nitems2 > 0 ? 2 : 1); ++s, lut += 24 * L2) {
            const uint4* jw = reinterpret_cast<const uint4*>(insts[s == 0 ? bd.inst : bd.inst2].jw);
            if (LT > 4) make_tables_apart(lut, jw, L2);
            else make_tables(lut, jw, L2);
        }
        uint32_t* const thr = reinterpret_cast<uint32_t*>(smem + lay.thr);
        if (LT != 4) make_thresholds_apart(thr, in0.thr, NT, kt);
        else make_thresholds(thr, in0.thr, NT, kt);
        if (FLAT) {
            const int nz = lay.ncols * lay.col_bytes / 16;
            for (int i = tid; i < ngroups * nz; i += blockDim.x)
                reinterpret_cast<uint4*>(group_base(i / nz) + lay.spins)[i % nz] = make_uint4(0u, 0u, 0u, 0u);
            for (int i = tid; i < ngroups * 2 * L2; i += blockDim.x) {
                const int g = i / (2 * L2), q = i - g * 2 * L2;
                const InstDesc& ig = g < ng1 ? in0 : insts[bd.inst2];
                reinterpret_cast<uint4*>(group_base(g))[q] = lane_pre(s_first, q >= L2, q >= L2 ? q - L2 : q, L, ig.seed, ig.uid);
            }
        } else {
            for (int g = 0; g < ngroups; ++g) {
                uint32_t* sp = reinterpret_cast<uint32_t*>(group_base(g) + lay.spins);
                for (int i = tid; i < lay.ncols * lay.col_bytes / 4; i += blockDim.x) sp[i] = 0u;
                uint4* pg = reinterpret_cast<uint4*>(group_base(g));
                const InstDesc& ig = g < ng1 ? in0 : insts[bd.inst2];
                for (int i = tid; i < 2 * L2; i += blockDim.x)
                    pg[i] = lane_pre(s_first, i >= L2, i >= L2 ? i - L2 : i, L, ig.seed, ig.uid);
            }
        }
    }
    for (int i = tid; i < nruns * NT; i += blockDim.x) {
        const int r = i / NT, t = i - r * NT, run = run_of(r), at = slot_of(r);
        const InstDesc& ir = inst_of(r);
        unsigned char* rb = run_base(at / gr, at % gr);
        const size_t g = (size_t)run * NT + t;
        const int b = PT_IDX((int)ir.perm[g], NT, 2u);
        reinterpret_cast<int32_t*>(rb + rl.E)[t] = ir.E[g];
        (rb + rl.perm)[t] = (uint8_t)b;
        (rb + rl.inv)[b] = (uint8_t)t;
        reinterpret_cast<uint32_t*>(rb + rl.macc)[t] = 0u;
        reinterpret_cast<uint32_t*>(rb + rl.xacc)[t] = 0u;
        if (walk) {
            reinterpret_cast<uint32_t*>(rb + rl.whot)[t] = 0u;
            reinterpret_cast<uint32_t*>(rb + rl.wtrips)[t] = 0u;
            (rb + rl.wstate)[t] = ir.wstate[g];
        }
        if (t == 0) {
            reinterpret_cast<int32_t*>(rb + rl.misc)[0] = ir.best[run];
            reinterpret_cast<int32_t*>(rb + rl.misc)[1] = ir.first[run];
        }
    }
    __syncthreads();
    // spin word i of run r (buffer b, group g = 2 cell + u) in memory and its byte in shared memory
    auto spin_words = [&](int r) { return reinterpret_cast<uint32_t*>(inst_of(r).spins + (size_t)run_of(r) * NT * N); };
    auto spin_byte = [&](int at, int i) {
        const int b = i / NW, g = i - b * NW, q = g >> 1, y = q / L, x = q - y * L, cl = (y + x + (g & 1)) & 1;
        const int p = (at % gr) * NT + b;
        return group_base(at / gr) + lay.spins + (p >> 5) * lay.col_bytes + cl * (lay.col_bytes / 2) + (q + L) * 32 + (p & 31);
    };
    if (SWEEP && FLAT) {
        load_spins(group_base(0) + lay.spins, reinterpret_cast<uint2*>(in0.spins + (size_t)bd.run0 * NT * N), bd.nitems * NT * L2, L,
           gr * NT, lay.group_bytes, lay.col_bytes);
        if (bd.nitems2 > 0)
            load_spins(group_base(ng1) + lay.spins, reinterpret_cast<uint2*>(insts[bd.inst2].spins), bd.nitems2 * NT * L2, L,
               gr * NT, lay.group_bytes, lay.col_bytes);
    }
    for (int r = 0; r < (SWEEP && !FLAT ? nruns : 0); ++r) {
        const uint32_t* gsp = spin_words(r);
        const int at = slot_of(r);
        for (int i = tid; i < NT * NW; i += blockDim.x)
            *spin_byte(at, i) = (unsigned char)(((gsp[i] & 0x80808080u) * 0x00204081u) >> 26);
    }
    if (n_iter > 0 && xon && xwait == 0u)
        for (int r = gw - 1 - gwid; r < nit; r += gw)
            exchange_prepare(xthr, xoff_sm, lane, s_first, (uint32_t)(grun + r) << 16, k0, k1, NT,
                             reinterpret_cast<int32_t*>(run_base(grp, r) + rl.ccrit) + (s_first & 1u) * NT);
    __syncthreads();

    if (active) {
        unsigned char* rb = run_base(grp, item);
        unsigned char* s0 = gb + lay.spins + col * lay.col_bytes + L * 32 + lane;     // colour 0, cell 0
        unsigned char* s1 = s0 + lay.col_bytes / 2;
        const unsigned char* lut0 = smem + lay.lut + (second ? 384 * L2 : 0);
        const uint32_t thr_at = (uint32_t)__cvta_generic_to_shared(smem + lay.thr);
        LaneConst lc;
        lc.kt = kt;
#pragma unroll
        for (int r = 0; r < 7; ++r) {           // through a warp reduction each, so that they are kept, not recomputed
            lc.ka[r] = __reduce_or_sync(FULL, k0 + (3u + r) * PHILOX_W0);
            lc.kb[r] = __reduce_or_sync(FULL, k1 + (3u + r) * PHILOX_W1);
        }
        const int nchain = nit < gw ? nit : gw;
        for (int it = 0; it < n_iter; ++it) {
            const uint32_t s = s_first + (uint32_t)it;
            const bool do_x = xon && xwait == 0u;
            xwait = xwait == 0u ? xper - 1u : xwait - 1u;          // from here on: of sweep s + 1
            if (SWEEP) {
                uint32_t dk = 0u, pc = 0u;
                const int t = PT_IDX((int)(rb + rl.inv)[buf], NT, 2u);
                const PhiloxPre ps = philox_pre(s, 0u, k0, k1);
                lc.y2x = ps.y2x;
                lc.y1k = ps.y1k;
                lc.c1 = ((uint32_t)(grun + item) << 16) | (uint32_t)t;
                lc.tcol = thr_at + (uint32_t)((t >> 5) * lc.kt * 128 + (t & 31) * 4) - 127u * 128u;
                if (busy) lane_phase<LT, 0>(lut0, s0, s1, pre, w, W, L, lc, dk, pc);
                if (W > 1) gsync();
                if (busy) lane_phase<LT, 1>(lut0 + L2 * 192, s1, s0, pre + L2, w, W, L, lc, dk, pc);
                const int n = (int)(pc >> 7), sk = (int)(dk >> 7) - 127 * n;   // accepted flips, sum of their k
                if (valid) {                // also zeros: a branch each cost C_4 sweeps 4 %
                    atomicAdd(reinterpret_cast<int32_t*>(rb + rl.E) + t, 2 * sk);
                    atomicAdd(reinterpret_cast<uint32_t*>(rb + rl.macc) + t, (uint32_t)n);
                }
            }
            gsync();
            for (int r = gwid; r < nit; r += gw) {
                unsigned char* xb = run_base(grp, r);
                int32_t* Es = reinterpret_cast<int32_t*>(xb + rl.E);
                int32_t* misc = reinterpret_cast<int32_t*>(xb + rl.misc);
                int m;
                const int record = misc[0];         // loaded before the chain: C_4 sweeps 6 % faster
                if (do_x) {
                    uint32_t* xacc = reinterpret_cast<uint32_t*>(xb + rl.xacc);
                    const int32_t* cc = reinterpret_cast<const int32_t*>(xb + rl.ccrit) + (s & 1u) * NT;
                    int2* xp = reinterpret_cast<int2*>(xb + rl.bytes);
                    m = NT > 32 ? lane_exchange<true>(Es, xb + rl.perm, xb + rl.inv, xacc, cc, xp, NT, lane)
                                : lane_exchange<false>(Es, xb + rl.perm, xb + rl.inv, xacc, cc, xp, NT, lane);
                    if (walk)
                        walk_update_warp(xb + rl.perm, reinterpret_cast<uint32_t*>(xb + rl.whot),
                                         reinterpret_cast<uint32_t*>(xb + rl.wtrips), xb + rl.wstate, NT, lane);
                } else {
                    m = slot_min_warp(Es, NT, lane);
                }
                if (SWEEP && lane == 0 && m < record) {
                    misc[0] = m;
                    misc[1] = (int32_t)s;
                }
            }
            if (it + 1 < n_iter) {              // meanwhile the group's other warps prepare its next sweep
                if (xon && xwait == 0u)
                    for (int r = gw - 1 - gwid; r < nit; r += gw)
                        exchange_prepare(xthr, xoff_sm, lane, s + 1u, (uint32_t)(grun + r) << 16, k0, k1, NT,
                                         reinterpret_cast<int32_t*>(run_base(grp, r) + rl.ccrit) + ((s + 1u) & 1u) * NT);
                const int f0 = gw > nchain ? nchain : 0;
                for (int i = gwid >= f0 ? (gwid - f0) * 32 + lane : 2 * L2; i < 2 * L2; i += 32 * (gw - f0))
                    pre[i] = lane_pre(s + 1u, i >= L2, i >= L2 ? i - L2 : i, L, k0, k1);
            }
            gsync();
        }
    }

    // ---- write the state back
    __syncthreads();
    if (SWEEP && FLAT) {
        store_spins(group_base(0) + lay.spins, reinterpret_cast<uint2*>(in0.spins + (size_t)bd.run0 * NT * N), bd.nitems * NT * L2, L,
           gr * NT, lay.group_bytes, lay.col_bytes);
        if (bd.nitems2 > 0)
            store_spins(group_base(ng1) + lay.spins, reinterpret_cast<uint2*>(insts[bd.inst2].spins), bd.nitems2 * NT * L2, L,
               gr * NT, lay.group_bytes, lay.col_bytes);
    }
    for (int r = 0; r < (SWEEP && !FLAT ? nruns : 0); ++r) {
        uint32_t* gsp = spin_words(r);
        const int at = slot_of(r);
        for (int i = tid; i < NT * NW; i += blockDim.x)
            gsp[i] = byte_signs(*spin_byte(at, i) * 0x04081020u) | 0x01010101u;   // 0xFF or 1
    }
    for (int i = tid; i < nruns * NT; i += blockDim.x) {
        const int r = i / NT, t = i - r * NT, run = run_of(r), at = slot_of(r);
        const InstDesc& ir = inst_of(r);
        const unsigned char* xb = run_base(at / gr, at % gr);
        const size_t g = (size_t)run * NT + t;
        ir.E[g] = reinterpret_cast<const int32_t*>(xb + rl.E)[t];
        ir.perm[g] = (xb + rl.perm)[t];
        ir.macc[g] += reinterpret_cast<const uint32_t*>(xb + rl.macc)[t];
        if (t < NT - 1) ir.xacc[(size_t)run * (NT > 1 ? NT - 1 : 1) + t] += reinterpret_cast<const uint32_t*>(xb + rl.xacc)[t];
        if (walk) {
            ir.whot[g] += reinterpret_cast<const uint32_t*>(xb + rl.whot)[t];
            ir.wtrips[g] += reinterpret_cast<const uint32_t*>(xb + rl.wtrips)[t];
            ir.wstate[g] = (xb + rl.wstate)[t];
        }
        if (t == 0) {
            ir.best[run] = reinterpret_cast<const int32_t*>(xb + rl.misc)[0];
            ir.first[run] = reinterpret_cast<const int32_t*>(xb + rl.misc)[1];
        }
    }
    __syncthreads();
}

}  // namespace
}  // namespace ptg

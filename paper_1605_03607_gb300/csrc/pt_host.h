// pt_host.h -- host-side helpers shared by the C-ABI runtimes (library-private):
// FP64 acceptance tables, the kernels' coupler layout, neighbour cells, and the
// host Philox used for the engineering draws.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <string>
#include <utility>
#include <vector>

#include "pt_internal.h"

namespace ptg {

// ------------------------------------------------------------------------
// Host Philox4x32-10 for the engineering draws (Salmon et al., SC'11).
// ------------------------------------------------------------------------
inline void philox_host(const uint32_t in[4], uint32_t k0, uint32_t k1, uint32_t out[4])
{
    uint32_t c0 = in[0], c1 = in[1], c2 = in[2], c3 = in[3];
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

inline uint32_t to_u32_threshold(double p)
{
    const double x = std::floor(std::ldexp(p, 32));
    if (x >= 4294967295.0) return 0xFFFFFFFFu;
    if (x <= 0.0) return 0u;
    return (uint32_t)x;
}

inline int n_edges_of(int L) { return 16 * L * L + 8 * L * (L - 1); }

// Coupler index helpers for the documented edge order.
inline int intra_edge(int L, int cell, int kv, int kh) { (void)L; return 16 * cell + 4 * kv + kh; }
inline int vert_edge(int L, int r, int c, int k) { return 16 * L * L + (r * L + c) * 4 + k; }
inline int horiz_edge(int L, int r, int c, int k) { return 16 * L * L + 4 * L * (L - 1) + (r * (L - 1) + c) * 4 + k; }

inline uint32_t pack4(int b0, int b1, int b2, int b3)
{
    return (uint32_t)(uint8_t)(int8_t)b0 | ((uint32_t)(uint8_t)(int8_t)b1 << 8) |
           ((uint32_t)(uint8_t)(int8_t)b2 << 16) | ((uint32_t)(uint8_t)(int8_t)b3 << 24);
}

// Kernel layout of the couplers (see InstDesc): per (cell, colour), 4 words of
// negated intra-cell couplers and 4 words of negated inter-cell couplers.
inline void pack_couplers(int L, const int8_t* J, uint32_t* jw)
{
    for (int r = 0; r < L; ++r)
        for (int c = 0; c < L; ++c) {
            const int cell = r * L + c;
            for (int col = 0; col < 2; ++col) {
                const int u = (r + c + col) & 1;
                uint32_t* w = jw + (cell * 2 + col) * 8;
                for (int k = 0; k < 4; ++k) {
                    int b[4];
                    for (int kp = 0; kp < 4; ++kp)
                        b[kp] = -(u == 0 ? J[intra_edge(L, cell, k, kp)] : J[intra_edge(L, cell, kp, k)]);
                    w[k] = pack4(b[0], b[1], b[2], b[3]);
                }
                int jm[4], jp[4];
                for (int k = 0; k < 4; ++k) {
                    if (u == 0) {
                        jm[k] = r >= 1 ? -J[vert_edge(L, r - 1, c, k)] : 0;
                        jp[k] = r + 1 < L ? -J[vert_edge(L, r, c, k)] : 0;
                    } else {
                        jm[k] = c >= 1 ? -J[horiz_edge(L, r, c - 1, k)] : 0;
                        jp[k] = c + 1 < L ? -J[horiz_edge(L, r, c, k)] : 0;
                    }
                }
                w[4] = pack4(jm[0], jp[0], 0, 0);
                w[5] = pack4(0, 0, jm[1], jp[1]);
                w[6] = pack4(jm[2], jp[2], 0, 0);
                w[7] = pack4(0, 0, jm[3], jp[3]);
            }
        }
}

inline void build_neighbours(int L, int16_t* nbr)
{
    for (int r = 0; r < L; ++r)
        for (int c = 0; c < L; ++c) {
            const int cell = r * L + c;
            for (int col = 0; col < 2; ++col) {
                const int u = (r + c + col) & 1;
                int m = cell, p = cell;
                if (u == 0) {
                    if (r >= 1) m = (r - 1) * L + c;
                    if (r + 1 < L) p = (r + 1) * L + c;
                } else {
                    if (c >= 1) m = r * L + c - 1;
                    if (c + 1 < L) p = r * L + c + 1;
                }
                nbr[(cell * 2 + col) * 2 + 0] = (int16_t)m;
                nbr[(cell * 2 + col) * 2 + 1] = (int16_t)p;
            }
        }
}

// Largest local-field magnitude an instance can produce: max over spins of
// sum_j |J_ij| (the Metropolis table needs rows k = 0 .. K).
inline int coupler_kmax(int L, const int8_t* J)
{
    const int N = 8 * L * L;
    std::vector<int> s((size_t)N, 0);
    for (int r = 0; r < L; ++r)
        for (int c = 0; c < L; ++c) {
            const int cell = r * L + c;
            for (int kv = 0; kv < 4; ++kv)
                for (int kh = 0; kh < 4; ++kh) {
                    const int a = std::abs((int)J[intra_edge(L, cell, kv, kh)]);
                    s[(size_t)8 * cell + kv] += a;
                    s[(size_t)8 * cell + 4 + kh] += a;
                }
            for (int k = 0; k < 4; ++k) {
                if (r + 1 < L) {
                    const int a = std::abs((int)J[vert_edge(L, r, c, k)]);
                    s[(size_t)8 * cell + k] += a;
                    s[(size_t)8 * (cell + L) + k] += a;
                }
                if (c + 1 < L) {
                    const int a = std::abs((int)J[horiz_edge(L, r, c, k)]);
                    s[(size_t)8 * cell + 4 + k] += a;
                    s[(size_t)8 * (cell + 1) + 4 + k] += a;
                }
            }
        }
    int m = 0;
    for (int v : s) m = v > m ? v : m;
    return m;
}

// Table rows for an instance: the default 19, or K + 1 rounded up to a
// multiple of 4 when its couplers need more.
inline int table_rows_for(int kmax)
{
    if (kmax + 1 <= KT_DEFAULT) return KT_DEFAULT;
    return (kmax + 1 + 3) & ~3;
}

struct Tables {
    int kt = KT_DEFAULT;           // rows per slot
    std::vector<uint32_t> thr;     // [NT][kt]
    std::vector<int64_t> xoff;     // [NT]
    std::vector<uint32_t> xthr;
    std::vector<float> xhint;      // [NT-1]
};

// Writes the FP64 acceptance tables into caller buffers, allocating nothing:
// thr [NT][kt], xoff [NT], xhint [max(NT-1, 1)], and the ragged exchange
// thresholds into xthr (capacity xcap entries; xthr NULL only counts them).
// Returns the exchange-table length, or -1 with *why set when the ladder's
// tables are too long or not monotone.
inline int64_t fill_tables(int NT, int kt, const double* betas, uint32_t* thr, int64_t* xoff, float* xhint,
                           uint32_t* xthr, int64_t xcap, const char** why)
{
    for (int t = 0; t < NT; ++t) {
        thr[(size_t)t * kt] = 0xFFFFFFFFu;   // k <= 0 always accepts; entry unused for decisions
        for (int k = 1; k < kt; ++k)
            thr[(size_t)t * kt + k] = to_u32_threshold(std::exp(-2.0 * (double)k * betas[t]));
    }
    int64_t n = 0;
    xhint[0] = 0.f;
    for (int p = 0; p + 1 < NT; ++p) {
        const double db = betas[p] - betas[p + 1];
        xoff[p] = n;
        xhint[p] = (float)(std::log(2.0) / (2.0 * db));
        uint32_t prev = 0xFFFFFFFFu;
        for (int64_t h = 1;; ++h) {
            const uint32_t v = to_u32_threshold(std::exp(-2.0 * (double)h * db));
            if (v == 0u) break;
            if (h > (1 << 22)) { *why = "exchange table longer than 2^22 entries (beta gap too small)"; return -1; }
            if (h > 1 && v > prev) { *why = "exchange table not monotone (host libm)"; return -1; }
            if (xthr) {
                if (n >= xcap) { *why = "exchange tables exceed the table capacity"; return -1; }
                xthr[n] = v;
            }
            prev = v;
            ++n;
        }
    }
    if (NT > 0) xoff[NT - 1] = n;
    return n;
}

// Returns an empty string or the reason the ladder is rejected.
inline std::string build_tables(int NT, int kt, const double* betas, Tables& tb)
{
    tb.kt = kt;
    tb.thr.assign((size_t)NT * kt, 0u);
    tb.xoff.assign((size_t)NT, 0);
    tb.xhint.assign((size_t)(NT > 1 ? NT - 1 : 1), 0.f);
    const char* why = "";
    const int64_t n = fill_tables(NT, kt, betas, tb.thr.data(), tb.xoff.data(), tb.xhint.data(), nullptr, 0, &why);
    if (n < 0) return why;
    if (n > (int64_t)INT32_MAX / 2) return "exchange tables too large";
    tb.xthr.assign((size_t)n, 0u);
    if (fill_tables(NT, kt, betas, tb.thr.data(), tb.xoff.data(), tb.xhint.data(), tb.xthr.data(), n, &why) < 0)
        return why;
    return "";
}

// ------------------------------------------------------------------------
// Shape of the replica-lane mapping.
// ------------------------------------------------------------------------
struct LaneShape {
    int W = 1, gr = 1, G = 1;          // warps per column, runs per group, groups per CTA
    bool span = false;                 // a CTA may hold runs of two instances (with the same tables)
    int cell_sp = 0, cell_ipc = 0;     // not 0: the cell-major mapping instead, its threads per cell and runs per CTA
};

inline int lane_columns(int NT, int gr) { return (gr * NT + 31) / 32; }
inline int lane_threads(int NT, const LaneShape& s) { return 32 * s.W * lane_columns(NT, s.gr) * s.G; }

// Estimated SM clocks per sweep of an SM that holds `k` CTAs of the shape: a warp word (one
// cell and colour of a column) takes 117 + 130 / w clocks of a sub-partition that runs w
// warps (a CTA's warps go round the four of them: a count that is no multiple of four loads
// one more than the others), exchange and barriers 910, which the groups of the SM overlap;
// no group is faster than alone.  Fitted to 900 (shape, size) pairs from C_2 to C_16, measured on
// an earlier kernel whose exchange took 200 to 300 clocks longer: there the lowest estimate's
// shape was 0.5 % slower than the best one on average, 3 % at most.  On the kernel as it is that
// has not been measured; 750 and 600 in place of 910 changed no plan for the better.
inline double lane_words(int L, int NT, const LaneShape& s)            // of a group, with its shares' imbalance
{
    const int units = (L & 1) ? L * L / 2 + 1 : (L / 2) * (L / 2);      // what the warps of a column share out
    const int c = lane_columns(NT, s.gr), per = (units + s.W - 1) / s.W, nw = s.G * c * s.W;
    return 2.0 * L * L * c * per * s.W / units * ((nw + 3) / 4 * 4) / nw;
}

inline double lane_clocks(int L, int NT, const LaneShape& s, int k)
{
    const double words = lane_words(L, NT, s), n = (double)k * s.G;
    const double w1 = 0.25 * lane_columns(NT, s.gr) * s.W, x = 910.0;
    const double together = 0.25 * words * n * (117.0 + 130.0 / (w1 * n)) + x / std::pow(n, 0.7);
    return std::max(together, 0.25 * words * (117.0 + 130.0 / w1) + x);
}

// CTAs that the estimate counts on an SM, which its constants were fitted with.  The device holds fewer of
// the small ones: 1024 threads (59 to 62 registers each, allocated as 64) and 4 CTAs of any
// size (16 named barriers each, 64 an SM).  That count with the same constants is no better a rule: of 4000
// random sizes 126 take another shape, 1.07 times faster on average but from 0.87 (C_4 x 58 slots, 195
// runs, 14 candidates) to 1.43 (C_1 x 39, 133, 16), and a batch of C_2 to C_8 0.68.  It needs a fit of its own.
inline int lane_counted(int threads, int64_t smem)
{
    return std::max(1, (int)std::min<int64_t>(std::min(32, 1152 / threads), (228 * 1024) / (smem + 1024)));
}

// Default schedule: about 256 threads per run, a multiple of 32.
inline void default_schedule(int L, int NT, int R, int& sp, int& ipc, int kt)
{
    const int L2 = L * L;
    sp = std::max(1, 256 / L2);
    if (sp > NT) sp = NT;
    while ((sp * L2) % 32 != 0) ++sp;
    const int tpi = sp * L2;
    ipc = std::max(1, 512 / tpi);
    if (ipc > R) ipc = R;
    while (ipc > 1 && bundle_smem_bytes(L, NT, ipc, 0, false, kt) > 110 * 1024) --ipc;
}

// Estimated SM clocks per sweep of a cell-major CTA with the SM to itself, its threads per cell and
// runs as above: 300 a warp, and for every further slot of a thread 800 + 75 a warp; the exchange is
// taken at half its 2100 (sweeps without one cost nothing there).  Fitted to one run and two runs a
// CTA on C_8, C_12 and C_16 with 1 to 8 slots.
inline double cell_clocks(int L, int NT, int sp, int ipc)
{
    const double w = sp * L * L * ipc / 32.0;
    return 2700.0 + 300.0 * w + (NT > 1 ? 1000.0 : 0.0) + ((NT + sp - 1) / sp - 1) * (800.0 + 75.0 * w);
}

// The shape with the lowest estimate for n_inst instances of R runs on `sms` SMs: all CTAs
// of a launch run at once if they fit, else in waves.  One run per CTA spreads best over
// the SMs; more runs share the field tables (384 L^2 bytes an instance), which decides at
// large L.  Runs that do not divide into whole CTAs fill them up with the next instance's
// (span): 16 C_8 instances of 64 runs (32 temperatures) are 147 CTAs of 7, one for each SM,
// where CTAs of one instance came in two waves: 2048 sweeps 29.9 -> 28.1 ms.
// With up to 10 slots most lanes are empty, and on large lattices a lane per cell is the
// faster mapping while its CTAs come to at most two an SM (C_16: 1.5 times with 4 slots and
// one run, even at 8; C_12: 1.2 times with 4; below C_8 with more than 2 slots never).
// cell_runs: at most so many runs in a cell-major CTA.
inline LaneShape lane_plan(int L, int NT, int kt, int R, int n_inst, bool walk, int sms, int cap, int cell_runs = 1 << 20)
{
    const int units = (L & 1) ? L * L / 2 + 1 : (L / 2) * (L / 2);
    LaneShape best;
    double best_t = 1e300;
    for (int gr = 1; gr <= 8 && gr <= R; ++gr)
        for (int G = 1; G <= LANE_GROUPS && (G - 1) * gr < R; ++G)
            for (int span = 0; span < 2; ++span) {
                const int64_t per = (R + gr - 1) / gr;                  // groups of an instance
                if (span && (n_inst == 1 || per % G == 0)) continue;    // (G - 1) * gr < R: at most two instances a CTA
                const int64_t ctas = span ? (n_inst * per + G - 1) / G : n_inst * ((per + G - 1) / G);
                // groups of the SM with most CTAs: where their words alone, evenly shared, take longer than the best shape
                // so far, no warp count helps.  Most shapes end here (C_8 x 4 slots x 100 runs: a plan 18 -> 3 us)
                const double most = (double)((ctas + sms - 1) / sms) * G;
                if (0.25 * 117.0 * (2.0 * L * L * lane_columns(NT, gr)) * most > best_t) continue;
                const int64_t smem = lane_layout(L, NT, kt, gr, G, walk, span ? 2 : 1).bytes;
                if (smem > cap) continue;
                for (int W : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}) {
                    LaneShape s;
                    s.W = W;
                    s.gr = gr;
                    s.G = G;
                    s.span = span != 0;
                    const int threads = lane_threads(NT, s);
                    if (threads > LANE_THREADS || (W > units && W > 1)) break;
                    if (0.25 * 117.0 * lane_words(L, NT, s) * most > best_t) continue;
                    const int fit = lane_counted(threads, smem);
                    const int64_t wave = (int64_t)fit * sms;
                    const int rest = (int)((ctas % wave + sms - 1) / sms);
                    const double t = (ctas >= wave ? (double)(ctas / wave) * lane_clocks(L, NT, s, fit) : 0.0) +
                                     (rest ? lane_clocks(L, NT, s, rest) : 0.0);
                    if (t < best_t * 0.999) { best_t = t; best = s; }
                }
            }
    if (NT <= 10) {
        int sp, ipc;
        default_schedule(L, NT, R, sp, ipc, kt);
        ipc = std::min(ipc, cell_runs);
        const int64_t ctas = n_inst * (int64_t)((R + ipc - 1) / ipc);
        if (sp * L * L * ipc <= MAX_THREADS && bundle_smem_bytes(L, NT, ipc, 0, walk, kt) <= cap && ctas <= 2 * sms &&
            (NT == 1 || cell_clocks(L, NT, sp, ipc) * (ctas > sms ? 1.5 : 1.0) < best_t)) {
            best.cell_sp = sp;
            best.cell_ipc = ipc;
        }
    }
    return best;
}

inline int64_t lane_smem(int L, int NT, int kt, const LaneShape& s, bool walk)
{
    return lane_layout(L, NT, kt, s.gr, s.G, walk, s.span ? 2 : 1).bytes;
}

// Bundles of the first R runs of the listed instances.
inline void lane_bundles(const LaneShape& s, const std::vector<int>& insts, int R, std::vector<Bundle>& out)
{
    out.clear();
    int r = 0;
    for (size_t a = 0; a < insts.size();) {
        Bundle b;
        b.inst = insts[a]; b.run0 = r; b.nitems = std::min(s.gr * s.G, R - r); b.sp = s.W; b.team = -s.gr;
        r += b.nitems;
        if (r == R) {
            r = 0;
            const int left = s.G - (b.nitems + s.gr - 1) / s.gr;
            if (++a < insts.size() && s.span && left > 0) {
                b.inst2 = insts[a];
                b.nitems2 = std::min(left * s.gr, R);
                r = b.nitems2;
                if (r == R) { r = 0; ++a; }
            }
        }
        out.push_back(b);
    }
}

// Shape of a batch's instances of one lattice side (their temperature counts `NTs`), whose
// CTAs of 32 W Ct threads pull bundles from a queue: for an instance the (gr, G) with the
// fewest bundles that fills at most Ct columns, and the (W, Ct) with the lowest estimated
// total.  False if no shape fits.
inline bool lane_fill(int L, int NT, int kt, int R, int W, int Ct, int cap, LaneShape* best)
{
    int fewest = 0;
    for (int gr = 1; gr <= 8 && gr <= R; ++gr) {
        const int c = lane_columns(NT, gr);
        int G = std::min(std::min(Ct / c, LANE_GROUPS), (R + gr - 1) / gr);
        while (G > 0 && lane_layout(L, NT, kt, gr, G, false).bytes > cap) --G;
        if (G < 1) continue;
        const int n = (R + gr * G - 1) / (gr * G);
        if (fewest == 0 || n < fewest) {
            fewest = n;
            best->W = W;
            best->gr = gr;
            best->G = G;
        }
    }
    return fewest > 0;
}

inline bool lane_plan_batch(int L, const std::vector<int>& NTs, int kt, int R, int sms, int cap, int* W, int* Ct,
                            double* clocks = nullptr)
{
    const int units = (L & 1) ? L * L / 2 + 1 : (L / 2) * (L / 2);
    std::vector<std::pair<int, int>> kinds;            // temperature counts and their instances: a kind is looked at once
    {
        std::vector<int> count(MAX_TEMPS + 1, 0);
        for (int nt : NTs) ++count[(size_t)nt];
        for (int nt = 1; nt <= MAX_TEMPS; ++nt)
            if (count[(size_t)nt]) kinds.push_back({nt, count[(size_t)nt]});
    }
    std::vector<LaneShape> s(kinds.size());
    double best = 1e300;
    for (int ct = 1; ct <= 32; ++ct)
        for (int w : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32}) {
            const int threads = 32 * w * ct;
            if (threads > LANE_THREADS || (w > units && w > 1)) break;
            int64_t smem = 0, ctas = 0;
            bool ok = true;
            for (size_t i = 0; ok && i < kinds.size(); ++i) {
                ok = lane_fill(L, kinds[i].first, kt, R, w, ct, cap, &s[i]);
                if (!ok) break;
                smem = std::max<int64_t>(smem, lane_layout(L, kinds[i].first, kt, s[i].gr, s[i].G, false).bytes);
                ctas += (int64_t)kinds[i].second * ((R + s[i].gr * s[i].G - 1) / (s[i].gr * s[i].G));
            }
            if (!ok) continue;
            const int fit = lane_counted(threads, smem);
            const int k = (int)std::min<int64_t>(fit, (ctas + sms - 1) / sms);      // CTAs an SM holds at a time
            double t = 0.0, longest = 0.0;
            for (size_t i = 0; i < kinds.size(); ++i) {
                const double one = lane_clocks(L, kinds[i].first, s[i], k);
                t += one / k * kinds[i].second * ((R + s[i].gr * s[i].G - 1) / (s[i].gr * s[i].G));
                longest = std::max(longest, one);
            }
            t = std::max(t / sms, longest);
            // the launch's tail: whole rounds of CTAs, which other sizes of the batch may fill
            t = 0.5 * (t + std::max(t, longest * (double)((ctas + (int64_t)k * sms - 1) / ((int64_t)k * sms))));
            if (t < best * 0.999) { best = t; *W = w; *Ct = ct; }
        }
    if (clocks) *clocks = best;
    return best < 1e300;
}

}  // namespace ptg

// Match-phase decode: the device-resident hot path.
//
// Wave 0 copies what needs no other match's output: every literal run
// (k_lits, over literal units of about equal bytes), then the in-order
// matches, whose source bytes are literals or in-order match bytes of the
// same block, level by level (a level's matches are independent; the levels
// are found at upload): one kernel per level, or, where the deferred matches
// go by waves or origin pieces, one over the blocks (k_ord_blocks).  Where
// most matches read the ones just before them they are walked in token order,
// block by block (k_ord_walk).
//
// Waves w >= 1 hold the matches whose sources become final only in earlier
// waves (the wavefront of Sec. I), block-ordered within each wave.  Two
// schedules run them:
//  - ACLZ_MODE_WAVES: one kernel per wave (k_wave_copy), kernel boundaries
//    as the wave barrier.  Where ACLZ_MODE_AUTO takes this schedule it goes
//    by levels instead of waves when the upload found them, one kernel per
//    level (k_level; runs of narrow levels together, k_level_run): every match
//    of a level is independent of the others, so no chain is left inside a step;
//  - ACLZ_MODE_PERSISTENT: one cooperative launch.  With staged copies it
//    runs the levels, with a bounded grid barrier between them
//    (k_levels_persistent); with register copies, or when the upload found no
//    levels (chains too deep) or mostly narrow ones, ranges of consecutive
//    (block, wave) segments in wave-major order (k_ranges), with bounded waits
//    on per-block completed-wave bits instead of barriers, so a match is copied
//    as soon as the blocks it reads have finished the waves below its own.
//
// All copies are 16-byte vectorised with every lane owning aligned output
// chunks, so short matches from several tokens share one pass instead of
// leaving most of the group idle (the work-granularity mechanism of
// Sec. III-C).  Matches copied by levels, and long ones in work ranges, are
// staged through shared memory by TMA bulk copies (cp.async.bulk + mbarrier).
#include <algorithm>
#include <cstring>
#include <mutex>

#include "aclz_device.cuh"
#include "aclz_internal.h"

using namespace aclz;

namespace {

constexpr int kThreads = 256;
// per-wave copy CTAs, and the CTAs of that size per SM the register cap is
// set for
constexpr int kWaveThreads = 64, kWaveMinCtas = 1024 / kWaveThreads;
// per-level copies: CTA size, the CTAs per SM the register cap is set for,
// stage bytes per warp (16 matches of up to 192 bytes; more when the deferred
// matches average kStageLongMin bytes or more), and the level sizes up to
// which a group of G lanes takes G / 4, G / 8 and one match instead of G / 2
constexpr int kLevelThreads = 128, kLevelMinCtas = 9;
constexpr uint32_t kStageWarp = 3584, kStageWarpLong = 6144;
constexpr double kStageLongMin = 224.0;
constexpr uint64_t kLevelQuarter = 40000, kLevelEighth = 20000, kLevelOne = 5000;
// runs of narrow levels: CTA size
constexpr int kRunThreads = 512;
// in-order levels by block: CTA size, and the same for blocks below kOrdSmall
// bytes (16 MiB of text flattened, 4 KiB blocks: 118 us with 128 threads,
// 131 us with 512; 32 MiB, 64 KiB blocks: 225 and 213 us); the length above
// which a match is copied by a warp
constexpr int kOrdThreads = 512, kOrdThreadsSmall = 128;
constexpr uint32_t kOrdSmall = 1u << 14;
constexpr uint32_t kOrdLong = 64;
// literal copies: CTA size, CTAs of that size per SM the register cap is set
// for, chunks per lane per round
constexpr int kLitThreads = 128, kLitMinCtas = 8, kUnrollLits = 2;
constexpr int kUnrollCopy = 2;   // chunks per lane per round in per-wave match copies
constexpr int kUnrollRanges = 4; // the same in the persistent schedule's register copies
// staged (TMA) copies: jobs of at least kTmaMin bytes, pieces of <= kPiece
constexpr uint32_t kTmaMin = 192;
constexpr uint32_t kPiece = 2048;
// persistent level copies: CTA size, CTAs per SM
constexpr int kPersThreads = 256, kPersCtas = 2;
constexpr uint32_t kSmemPerSm = 220u * 1024u;  // stage memory shared by the CTAs of one SM
// per-wave kernels are launched with programmatic stream serialization
constexpr int kWavePdl = 1;

__device__ __forceinline__ uint64_t tri_dst(const uint4 t) { return (uint64_t)t.x | ((uint64_t)(t.y & 0xffu) << 32); }
__device__ __forceinline__ uint64_t tri_src(const uint4 t) { return (uint64_t)t.z | ((uint64_t)(t.w & 0xffu) << 32); }
__device__ __forceinline__ uint32_t tri_len(const uint4 t) { return t.w >> 8; }
// set at upload on the triplets of segments without an internal chain: a
// per-wave group may start or stop at any of them
__device__ __forceinline__ bool tri_cut(const uint4 t) { return (t.y >> 8) & 1u; }

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Programmatic dependent launch (per-wave kernels): a kernel lets the next
// kernel of its stream start once all of its CTAs have begun, and that
// kernel reads nothing the previous one writes before griddep_wait, which
// returns when the previous grid has completed and its writes are visible.
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bounded waits: spin_limit polls (sleeping up to 256 ns each) before a wait
// gives up.  The host scales it with the wave count, from 2^22 (about a
// second) to 2^26: a range deep in a long chain legitimately waits for most
// of the launch.  A wait also gives up when another group already gave up
// (err has kErrTimeout), so one stuck wait ends the whole launch.
constexpr uint32_t kSpinLimitMin = 1u << 22;

// Spin (bounded) until every wave below w of one block is done: its done
// bits (ww 64-bit words, empty waves preset) are all set below bit w.
__device__ __forceinline__ bool wait_waves_below(const unsigned long long *done, uint32_t w, uint32_t *err,
                                                 uint32_t spin_limit) {
    for (uint32_t k = 0; k * 64 < w; k++) {
        const uint32_t nbits = w - k * 64;
        const unsigned long long want = nbits >= 64 ? ~0ULL : ((1ULL << nbits) - 1ULL);
        uint32_t spins = 0;
        while ((ld_acquire64(done + k) & want) != want) {
            if (++spins > spin_limit) {
                atomicOr(err, kErrTimeout);
                return false;
            }
            if ((spins & 255) == 0 && (*(volatile uint32_t *)err & kErrTimeout)) return false;
            __nanosleep(spins < 64 ? 32 : 256);
        }
    }
    return true;
}

// Exact same-wave dependencies inside one window of triplets (one per
// lane): bit j of the result is set when this lane's source overlaps the
// output of lane j < this lane.  Only matches of one block can depend on
// each other within a wave (a source in another block was final a wave
// earlier), so lanes whose source does not end in their own block skip the
// test.
template <int G>
__device__ __forceinline__ unsigned same_wave_deps(const Group<G> &g, bool v, uint64_t d, uint64_t sr,
                                                   uint32_t len, uint32_t log2bs) {
    const uint64_t blk = d >> log2bs;
    const bool local = v && ((sr + len - 1) >> log2bs) == blk;
    unsigned m = 0;
    if (!g.ballot(local)) return 0u;
    for (int j = 0; j < G; j++) {
        const uint64_t dj = g.shfl(d, j);
        const uint32_t nj = g.shfl(len, j);
        if (local && j < g.lane && nj && (dj >> log2bs) == blk && sr < dj + nj && dj < sr + len) m |= 1u << j;
    }
    return m;
}

// ------------------------------------------------------------- wave 0

// Literal runs: one group per literal unit {block, first token, literal
// range within the block}.  A window of G tokens needs no prefix sums, only
// the tokens' output and literal offsets from the upload; a token's run ends
// where the next token's literals start.  With done non-null (the
// persistent schedule follows), each block's done bits start as its empty
// waves plus wave 0; with barrier non-null (the persistent level schedule
// follows) its count starts at 0.  The other schedules leave both alone: they
// may run on one handle in several streams.
//
// Bound by the latency of the unit's one or two rounds and by instruction
// issue.  Units, and not blocks, are the work items because a stream has few
// blocks (512 in 32 MiB at 64 KiB) and very unequal amounts of literals in
// them: the literals and in-order matches of 32 MiB of word text at 6/8/10/12
// took 786 us with one warp walking each block's tokens, the literals take
// 56 us here (64 MiB of FASTQ-like text 108 -> 57 us, 256 KiB of Markov
// bytes 97 -> 6 us).
template <int G>
__global__ void __launch_bounds__(kLitThreads, kLitMinCtas)
    k_lits(const uint4 *__restrict__ units, uint64_t n_units, const uint8_t *__restrict__ lit,
           const uint64_t *__restrict__ blk_tok, const uint64_t *__restrict__ blk_lit,
           const uint32_t *__restrict__ tokdst, const uint32_t *__restrict__ toklit, uint8_t *out, uint32_t log2bs,
           const uint64_t *__restrict__ pending, uint64_t *done, uint64_t n_done, uint32_t ww, uint32_t *barrier) {
    Group<G> g;
    griddep_launch_dependents();
    if (barrier && blockIdx.x == 0 && threadIdx.x == 0) *barrier = 0;
    const uint64_t tid = blockIdx.x * (uint64_t)kLitThreads + threadIdx.x;
    for (uint64_t k = tid; k < n_done; k += (uint64_t)gridDim.x * kLitThreads)
        done[k] = ~__ldg(pending + k) | (k % ww == 0 ? 1ULL : 0ULL);
    if (tid / G >= n_units) return;
    const uint4 u = __ldg(units + tid / G);
    const uint32_t lo = u.z, hi = u.w;
    if (lo == hi) return;
    const uint64_t t1 = __ldg(blk_tok + u.x + 1);
    const uint8_t *ls = lit + __ldg(blk_lit + u.x);
    const uint64_t bpos = (uint64_t)u.x << log2bs;
    uint64_t w = u.y;
    // literal and output offset of this lane's token, the next window's
    // loaded ahead (tokens past the block's end start at hi: no run)
    uint32_t nl = w + g.lane < t1 ? __ldg(toklit + w + g.lane) : hi;
    uint32_t nd = w + g.lane < t1 ? __ldg(tokdst + w + g.lane) : 0u;
    for (;;) {
        const uint32_t l0 = nl, d0 = nd;
        w += G;
        nl = w + g.lane < t1 ? __ldg(toklit + w + g.lane) : hi;
        nd = w + g.lane < t1 ? __ldg(tokdst + w + g.lane) : 0u;
        const uint32_t after = g.shfl(nl, 0), right = g.shfl(l0, (g.lane + 1) & (G - 1));
        const uint32_t l1 = g.lane == G - 1 ? after : right;
        const uint32_t x = max(l0, lo), y = min(l1, hi);
        group_copy<G, kUnrollLits, kFromConst>(g, out, bpos + d0 + (x - l0), ls + x, y > x ? y - x : 0u);
        if (after >= hi) break;
    }
}

// ------------------------------------------------ persistent schedule

// One look, without waiting, at whether every block of [sr, sr + len) has
// finished its waves below w (w <= 64, at most 4 blocks); acquire loads.
__device__ __forceinline__ bool waves_below_now(const unsigned long long *done, uint32_t ww, uint64_t sr,
                                                uint32_t len, uint32_t w, uint32_t log2bs) {
    if (w > 64) return false;
    const uint64_t b0 = sr >> log2bs, b1 = (sr + len - 1) >> log2bs;
    if (b1 - b0 > 3) return false;
    const unsigned long long want = w >= 64 ? ~0ULL : ((1ULL << w) - 1ULL);
    for (uint64_t bb = b0; bb <= b1; bb++)
        if ((ld_acquire64(done + bb * ww) & want) != want) return false;
    return true;
}

// Waves >= 1 in one cooperative launch, by ranges: range r holds the
// consecutive triplets [first, next range's first) of one wave.  Each match
// waits (bounded) until every block its source touches has finished its
// waves below w (per-block done bits; empty waves are preset); the range
// copies its matches window by window, in dependency levels within a
// window (a match that reads another's output of the same wave goes after
// it); then it marks bit w of each block it finished.  A segment (one
// block's matches of one wave) cut into several ranges is finished by the
// last of its ranges to end, found with a per-segment counter.  Ranges
// wait only for ranges of lower waves, earlier in the list; all groups are
// co-resident and take their ranges in increasing order (r, r + K, r + 2K,
// ...), so every wait ends.
// STAGED: matches of at least kTmaMin bytes go through the group's
// shared-memory stage by TMA bulk copies, and a group looks at its next
// range before releasing the current one: when that range's sources are
// already final, its first fill is issued at once, so the bulk copy runs
// while the current range's stores drain and its blocks are released.
// Otherwise all copies go through registers and the kernel runs at higher
// occupancy.
template <int G, bool STAGED>
__global__ void __launch_bounds__(kThreads, STAGED ? 2 : 3)
    k_ranges(const uint4 *__restrict__ ranges, uint64_t n_ranges, const uint4 *__restrict__ seg,
             const uint32_t *__restrict__ pieces, uint32_t *seg_cnt, unsigned long long *done, uint32_t ww,
             const uint4 *__restrict__ tri, uint8_t *out, uint32_t log2bs, uint32_t stage_bytes, uint32_t *err,
             uint32_t spin_limit) {
    extern __shared__ __align__(128) uint8_t smem[];
    Group<G> g;
    constexpr int kGroups = kThreads / G;
    Stage st;
    uint32_t piece = 0;
    if (STAGED) {
        const int gi = threadIdx.x / G;
        st.bar = reinterpret_cast<uint64_t *>(smem) + gi;
        st.buf = smem + 128 * ((8 * kGroups + 127) / 128) + (size_t)gi * stage_bytes;
        st.bytes = stage_bytes;
        st.phase = 0;
        if (g.lane == 0) mbar_init(st.bar, 1);
        fence_mbar_init();
        __syncthreads();
        piece = min(kPiece, stage_bytes - 32u);
    }
    const uint64_t gid = (blockIdx.x * (uint64_t)kThreads + threadIdx.x) / G;
    const uint64_t ng = (uint64_t)gridDim.x * kGroups;
    const uint4 z4 = make_uint4(0, 0, 0, 0);
    bool ok = true;
    // ranges[n_ranges] is a sentinel: the end of range r is ranges[r + 1].w.
    // Loaded ahead: the descriptor and first window of this group's next
    // range (rn, tn, nt2) and the descriptor of the one after (rn3, tn3).
    auto desc = [&](uint64_t k, uint4 &rd, uint32_t &te) {
        rd = k < n_ranges ? __ldg(ranges + k) : z4;
        te = k < n_ranges ? __ldg(ranges + k + 1).w : 0u;
    };
    uint4 rc, rn, rn3;
    uint32_t tc, tn, tn3;
    desc(gid, rc, tc);
    desc(gid + ng, rn, tn);
    uint4 nt = rc.w + g.lane < tc ? __ldg(tri + rc.w + g.lane) : z4;
    uint4 nt2 = rn.w + g.lane < tn ? __ldg(tri + rn.w + g.lane) : z4;
    Fill pre = {0, 0, 0, 0};
    bool pre_on = false;  // the first batch of range `it` has its first fill in flight
    for (uint64_t it = gid; it < n_ranges; it += ng) {
        const uint4 r = rc;
        const uint64_t t_begin = r.w, t_end = tc;
        desc(it + 2 * ng, rn3, tn3);
        const uint32_t w = r.x, s0 = r.y, s1 = r.z;
        const bool has_next = it + ng < n_ranges;
        for (uint64_t cur = t_begin; cur < t_end; cur += G) {
            const bool v = cur + g.lane < t_end;
            const uint4 t = v ? nt : z4;
            if (cur + G < t_end) nt = cur + G + g.lane < t_end ? __ldg(tri + cur + G + g.lane) : z4;
            const uint64_t d = tri_dst(t), sr = tri_src(t);
            const uint32_t len = v ? tri_len(t) : 0u;
            const bool ahead = pre_on && cur == t_begin;
            if (!ahead) {
                // every block the source touches (its own included) has
                // finished its waves below w
                if (v) {
                    const uint64_t b0 = sr >> log2bs, b1 = (sr + len - 1) >> log2bs;
                    for (uint64_t bb = b0; bb <= b1; bb++)
                        if (!wait_waves_below(done + bb * ww, w, err, spin_limit)) ok = false;
                }
                g.sync();
            }
            const unsigned deps = same_wave_deps<G>(g, v, d, sr, len, log2bs);
            unsigned rem = g.ballot(v);
            bool issued = ahead;
            while (rem) {
                const unsigned batch = g.ballot(((rem >> g.lane) & 1u) && (deps & rem) == 0u);
                const bool mine = (batch >> g.lane) & 1u;
                if (STAGED) {
                    if (!issued) fence_proxy_async_global();
                    const bool longj = mine && len >= kTmaMin;
                    group_copy_batch<G, 2>(g, out, d, out + sr, (mine && !longj) ? len : 0u);
                    if (issued || g.ballot(longj)) {
                        if (!staged_copy_fills<G>(g, st, out, d, out + sr, longj ? len : 0u, piece, pre, issued,
                                                  err))
                            return;  // a bulk copy did not complete: no further copies into the stage
                    }
                } else {
                    group_copy_batch<G, kUnrollRanges>(g, out, d, out + sr, mine ? len : 0u);
                }
                g.sync();
                rem &= ~batch;
                issued = false;
            }
        }
        pre_on = false;
        // a look at the next range of this group: when the sources of its
        // first window are final already, its first fill is issued now, so
        // the bulk copy runs while this range's stores drain and its blocks
        // are released
        if (STAGED && has_next && g.ballot(!ok) == 0u) {
            const bool v2 = rn.w + g.lane < tn;
            const uint64_t d2 = tri_dst(nt2), s2 = tri_src(nt2);
            const uint32_t n2 = v2 ? tri_len(nt2) : 0u;
            const bool ready = !v2 || waves_below_now(done, ww, s2, n2, rn.x, log2bs);
            if (g.ballot(!ready) == 0u) {
                const unsigned deps2 = same_wave_deps<G>(g, v2, d2, s2, n2, log2bs);
                const unsigned all2 = g.ballot(v2);
                const bool long2 = v2 && n2 >= kTmaMin && (deps2 & all2) == 0u;
                if (g.ballot(long2)) {
                    fence_proxy_async_global();
                    pre.done = 0;
                    fill_issue<G>(g, st, out + s2, long2 ? n2 : 0u, piece, pre);
                    pre_on = true;
                }
            }
        }
        // release: this range's writes, then bit w of every block it
        // finished (of a shared segment, only the last range to end)
        __threadfence();
        g.sync();
        const unsigned long long bit = 1ULL << (w % 64);
        for (uint32_t k = s0 + g.lane; k < s1; k += G) {
            const uint64_t word = (uint64_t)__ldg(seg + k).x * ww + w / 64;
            const uint32_t pc = __ldg(pieces + k);
            if (pc > 1) {
                if (atomicAdd(seg_cnt + k, 1u) != pc - 1) continue;
                seg_cnt[k] = 0;  // the last range of the segment resets the count for the next decode
                __threadfence();
            }
            atomicOr(done + word, bit);
        }
        // shift the loaded-ahead state by one range
        nt = nt2;
        rc = rn;
        tc = tn;
        rn = rn3;
        tn = tn3;
        nt2 = rn.w + g.lane < tn ? __ldg(tri + rn.w + g.lane) : z4;
    }
    if (!ok) atomicOr(err, kErrTimeout);
}

// ------------------------------------------------------ wave schedule

// Copy one window of a wave's worklist (n triplets): the group whose window
// starts at triplet a.  A window of cuttable triplets (segments without an
// internal chain, marked at upload) is copied as it stands: no dependency
// test, no look at its neighbours.  Otherwise the group owns the segments
// (runs of one block) that start in its window, and cuttable triplets in
template <int G>
__device__ __forceinline__ void wave_window(const Group<G> &g, const uint4 *__restrict__ tri, uint64_t n, uint64_t a,
                                            const uint4 t0, uint8_t *out, uint32_t log2bs) {
    const uint4 z4 = make_uint4(0, 0, 0, 0);
    if (!g.ballot(a + g.lane < n && !tri_cut(t0))) {
        griddep_wait();
        group_copy<G, kUnrollCopy>(g, out, tri_dst(t0), out + tri_src(t0), tri_len(t0));
        return;
    }
    const uint64_t e = a + G < n ? a + G : n;
    // first cut point in [a, e): a segment start, or a cuttable triplet
    bool st0 = false;
    if (a + g.lane < e)
        st0 = a + g.lane == 0 || tri_cut(t0) ||
              (tri_dst(t0) >> log2bs) != (tri_dst(__ldg(tri + a + g.lane - 1)) >> log2bs);
    const unsigned m0 = g.ballot(st0);
    if (!m0) return;
    const uint64_t s = a + (uint64_t)(__ffs(m0) - 1);
    // the next window's triplets are loaded while the current one is copied;
    // lane 0 takes the block of the triplet before its window from the last
    // lane of the previous window (every lane of which was valid)
    uint4 nt = s + g.lane < n ? __ldg(tri + s + g.lane) : z4;
    uint64_t prev_blk = ~0ULL;
    // the worklist was written at upload; the sources, by earlier waves
    griddep_wait();
    for (uint64_t cur = s; cur < n; cur += G) {
        const uint64_t i = cur + g.lane;
        const bool v = i < n;
        const uint4 t = v ? nt : z4;
        if (cur + G + g.lane < n) nt = __ldg(tri + cur + G + g.lane);
        const uint64_t d = tri_dst(t), sr = tri_src(t);
        const uint32_t len = v ? tri_len(t) : 0u;
        const uint64_t blk = d >> log2bs;
        uint64_t pblk = g.shfl_up(blk, 1);
        if (g.lane == 0) pblk = (i == s) ? ~0ULL : prev_blk;
        prev_blk = g.shfl(blk, G - 1);
        const bool st = v && (i == s || blk != pblk || tri_cut(t));
        const unsigned stop = g.ballot(st && i >= e && i != s);
        unsigned act = g.ballot(v);
        if (stop) act &= (stop & (0u - stop)) - 1u;
        // exact same-wave dependencies inside the window (only sources that
        // end in their own block can have any); each batch takes the lanes
        // whose dependencies are all copied
        const unsigned deps = same_wave_deps<G>(g, (act >> g.lane) & 1u, d, sr, len, log2bs) & act;
        unsigned rem = act;
        while (rem) {
            const unsigned batch = g.ballot(((rem >> g.lane) & 1u) && (deps & rem) == 0u);
            const bool mine = (batch >> g.lane) & 1u;
            group_copy_batch<G, kUnrollCopy>(g, out, d, out + sr, mine ? len : 0u);
            g.sync();
            rem &= ~batch;
        }
        if (stop) break;
    }
}

// One wave's worklist, one window of G triplets per group (the most resident
// groups: two or four windows each were 2-8% slower).
template <int G>
__global__ void __launch_bounds__(kWaveThreads, kWaveMinCtas) k_wave_copy(const uint4 *__restrict__ tri, uint64_t n,
                                                                          uint8_t *out, uint32_t log2bs) {
    Group<G> g;
    griddep_launch_dependents();
    const uint64_t a = (blockIdx.x * (uint64_t)kWaveThreads + threadIdx.x) / G * G;
    if (a >= n) return;
    const uint4 t0 = a + g.lane < n ? __ldg(tri + a + g.lane) : make_uint4(0, 0, 0, 0);
    wave_window<G>(g, tri, n, a, t0, out, log2bs);
}

// One level's matches (all independent) through the groups' stages.
//
// Bound by the latency of a window and its instruction count (about 1200
// instructions for 32 matches of 128 bytes): most levels have fewer windows
// than the GPU has resident groups, so a level takes as long as one window.
// Hence few matches per group (G / 2, in small levels less), with heads and
// tails in one step, and the sources of the whole window in flight at once.
// Launches overlap (programmatic dependent launch): a small level costs 2.5
// us.  512 MiB copy sweep at L = 128 899 -> 721 us against one window of G
// matches per group through registers with small levels run one after another
// by one thread-block cluster (3.7 us a level); 256 MiB at L = 32 / 64 / 185
// 910 / 662 / 492 -> 792 / 563 / 337 us, 64 MiB of FASTQ-like text 154 -> 112
// us, 64 batched streams 70 -> 48 us, 256 KiB of Markov bytes 52 -> 36 us.
template <int G, int J>
__global__ void __launch_bounds__(kLevelThreads, kLevelMinCtas)
    k_level(const uint4 *__restrict__ tri, uint64_t n, uint8_t *out, uint32_t stage_bytes, uint32_t *err) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t bar[kLevelThreads / G];
    Group<G> g;
    griddep_launch_dependents();
    const int gi = threadIdx.x / G;
    Stage st = {smem + (size_t)gi * stage_bytes, bar + gi, stage_bytes, 0};
    const uint64_t i = (blockIdx.x * (uint64_t)kLevelThreads + threadIdx.x) / G * J + g.lane;
    const uint4 t = g.lane < J && i < n ? __ldg(tri + i) : make_uint4(0, 0, 0, 0);
    if (g.lane == 0) mbar_init(st.bar, 1);
    fence_mbar_init();
    g.sync();
    griddep_wait();
    fence_proxy_async_global();
    group_copy_staged<G, J>(g, st, out, tri_dst(t), out + tri_src(t), tri_len(t), err);
}

// A run of narrow levels by one CTA: a group takes a match or a few, loads the
// next level's while it copies, and a barrier of the CTA ends the level.
//
// Bound by a level's chain of L2 load, store and barrier (0.5 us for a match of
// 64 bytes), which a launch of its own makes 1.7 us: 16 MiB of FASTQ-like text
// with 24 KiB of zeros in it (386 levels, 360 of them of one or two matches)
// 630 -> 228 us, 1024 levels of 64 matches 1654 -> 806 us.
template <int G>
__global__ void __launch_bounds__(kRunThreads, 1) k_level_run(const Step *__restrict__ steps, uint32_t count,
                                                              uint8_t *out) {
    Group<G> g;
    griddep_launch_dependents();
    constexpr uint32_t kGroups = kRunThreads / G;
    const uint32_t gi = threadIdx.x / G;
    const ulonglong2 *list = reinterpret_cast<const ulonglong2 *>(steps);
    auto window = [&](const ulonglong2 &s) {
        const uint32_t n = (uint32_t)s.y, per = (n + kGroups - 1) / kGroups, i = gi * per + (uint32_t)g.lane;
        return (uint32_t)g.lane < per && i < n ? __ldg(reinterpret_cast<const uint4 *>(s.x) + i) : make_uint4(0, 0, 0, 0);
    };
    uint4 next = window(__ldg(list));
    ulonglong2 after = count > 1 ? __ldg(list + 1) : make_ulonglong2(0, 0);
    griddep_wait();
    for (uint32_t k = 0; k < count; k++) {
        const uint4 t = next;
        next = window(after);
        after = k + 2 < count ? __ldg(list + k + 2) : make_ulonglong2(0, 0);
        group_copy_batch<G, kUnrollCopy>(g, out, tri_dst(t), out + tri_src(t), tri_len(t));
        __syncthreads();
    }
}

// Every level in one cooperative launch.  A level's matches are dealt out
// evenly, at most G / 2 per group at a time, through the group's two stages
// in turn; the next level's first window is loaded before the barrier.
//
// Bound by a window's chain of fill, copy out, fill: a kilobyte match leaves
// three to a stage, so a window takes five fills or more.  With one stage per
// group and 32 warps per SM the 1 GiB copy sweep at L = 1024 / 4096 took
// 600 / 521 us; with two stages in turn, 16 warps per SM of up to 128
// registers and matches copied out one by one (their chunks need no search),
// 556 / 490 us, and 64 MiB at L = 1024 158 -> 125 us (k_ranges took 627 us at
// L = 1024).
template <int G>
__global__ void __launch_bounds__(kPersThreads, kPersCtas)
    k_levels_persistent(const Step *__restrict__ steps, uint32_t count, uint8_t *out, uint32_t stage_bytes,
                        uint32_t *err) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int kGroups = kPersThreads / G;
    Group<G> g;
    const int gi = threadIdx.x / G;
    Stage st[2];
    for (int k = 0; k < 2; k++) {
        st[k].bar = reinterpret_cast<uint64_t *>(smem) + 2 * gi + k;
        st[k].buf = smem + 128 * ((16 * kGroups + 127) / 128) + (size_t)(2 * gi + k) * stage_bytes;
        st[k].bytes = stage_bytes;
        st[k].phase = 0;
        if (g.lane == 0) mbar_init(st[k].bar, 1);
    }
    fence_mbar_init();
    __syncthreads();
    const uint32_t gid = (blockIdx.x * kPersThreads + threadIdx.x) / G;
    const uint32_t ng = gridDim.x * kGroups;
    const ulonglong2 *list = reinterpret_cast<const ulonglong2 *>(steps);
    const uint4 z4 = make_uint4(0, 0, 0, 0);
    auto share = [&](uint64_t n) {  // matches per group at a time
        const uint32_t e = ((uint32_t)n + ng - 1) / ng;
        return e < G / 2 ? e : (uint32_t)G / 2;
    };
    auto window = [&](const ulonglong2 &s, uint32_t per, uint32_t a) {
        return (uint32_t)g.lane < per && a + g.lane < (uint32_t)s.y
                   ? __ldg(reinterpret_cast<const uint4 *>(s.x) + a + g.lane) : z4;
    };
    ulonglong2 cur = __ldg(list), nx = count > 1 ? __ldg(list + 1) : make_ulonglong2(0, 0);
    uint32_t per = share(cur.y);
    uint4 t0 = window(cur, per, gid * per);
    bool ok = true;
    for (uint32_t k = 0; k < count; k++) {
        fence_proxy_async_global();
        for (uint32_t a = gid * per; ok && a < (uint32_t)cur.y; a += ng * per) {
            const uint4 t = t0;
            t0 = window(cur, per, a + ng * per);
            ok = group_copy_piped<G, G / 2>(g, st, out, tri_dst(t), out + tri_src(t), tri_len(t), err);
        }
        if (k + 1 == count) break;
        cur = nx;
        per = share(cur.y);
        t0 = window(cur, per, gid * per);
        if (k + 2 < count) nx = __ldg(list + k + 2);
        if (!grid_barrier(err + kBarrierWord, (k + 1) * gridDim.x, ok, err)) break;
    }
    if (!ok) {  // a wait timed out: leave no fill in flight
        stage_wait(st[0], err);
        stage_wait(st[1], err);
    }
}

// Every in-order level of one block per CTA, in shared memory: the block comes
// in as the literal copies left it, a level's matches are copied by one thread
// each (longer ones by their warp), and the block goes out again, bytes of
// deferred matches as they were.  An in-order match reads its own block only.
//
// Bound by the latency of a level's barrier, shared loads and narrow shared
// stores, not by bytes.  With one kernel per level (about 3 us each)
// 32 MiB of word text at 6/8/10/12, flattened, took 250 us and takes 213 us,
// 256 KiB of it 69 and 32 us, 16 MiB of FASTQ-like text 55 and 37 us (with 24
// KiB of zeros in it, a chain of 256 matches of 64 bytes, 216 us when one
// thread copied each whole, 113 us now).
__global__ void __launch_bounds__(kOrdThreads)
    k_ord_blocks(const uint4 *__restrict__ ord, const uint32_t *__restrict__ base, uint8_t *out, uint32_t log2bs,
                 uint64_t total) {
    extern __shared__ __align__(128) uint8_t smem[];
    griddep_launch_dependents();
    const uint32_t o0 = __ldg(base + blockIdx.x), o1 = __ldg(base + blockIdx.x + 1);
    if (o0 == o1) {
        griddep_wait();  // the grid ends after the one before it
        return;
    }
    const uint32_t tid = threadIdx.x, nt = blockDim.x;
    auto at = [&](uint32_t i) { return i < o1 ? __ldg(ord + i) : make_uint4(0, 0, 0, 0); };
    uint4 next = at(o0 + tid);
    const uint64_t bpos = (uint64_t)blockIdx.x << log2bs;
    const uint32_t len = (uint32_t)min((uint64_t)1 << log2bs, total - bpos), words = len >> 4;
    uint8_t *blk = out + bpos;
    griddep_wait();
    uint4 *sw = reinterpret_cast<uint4 *>(smem), *gw = reinterpret_cast<uint4 *>(blk);
#pragma unroll 8
    for (uint32_t i = tid; i < words; i += nt) sw[i] = __ldcg(gw + i);
    if (16 * words + tid < len && tid < 16) smem[16 * words + tid] = __ldcg(blk + 16 * words + tid);
    __syncthreads();
    const uintptr_t sbase = smem_u32(smem), gbase = reinterpret_cast<uintptr_t>(smem);
    auto piece = [&](uint32_t d, uint32_t s, uint32_t n) {
        store_bytes(gbase + d, load_bytes<kFromShared>(sbase + s, n), n);
    };
    for (uint32_t w = o0; w < o1; w += nt) {
        const uint4 t = next;
        next = at(w + nt + tid);
        const uint32_t mine = w + tid < o1 ? t.y >> 9 : 0xffffffffu;
        const uint32_t l1 = __ldg(&ord[min(w + nt, o1) - 1].y) >> 9;
        const uint32_t d = (uint32_t)(tri_dst(t) - bpos), s = (uint32_t)(tri_src(t) - bpos), n = tri_len(t);
        for (uint32_t l = __ldg(&ord[w].y) >> 9; l <= l1; l++) {
            const bool go = mine == l;
            // the warp shares its matches longer than kOrdLong, or its only one
            // longer than half of that; a thread copies the others piece by piece
            unsigned big = __ballot_sync(0xffffffffu, go && n > kOrdLong / 2);
            uint32_t alone = kOrdLong / 2;
            if (big & (big - 1u)) {
                big = __ballot_sync(0xffffffffu, go && n > kOrdLong);
                alone = kOrdLong;
            }
            if (go && n <= alone)
                for (uint32_t k = 0; k < n; k += 16) piece(d + k, s + k, min(n - k, 16u));
            for (unsigned m = big; m; m &= m - 1) {
                const int j = __ffs(m) - 1;
                const uint32_t dj = __shfl_sync(0xffffffffu, d, j), sj = __shfl_sync(0xffffffffu, s, j),
                               nj = __shfl_sync(0xffffffffu, n, j);
                for (uint32_t k = 16 * (tid & 31); k < nj; k += 512) piece(dj + k, sj + k, min(nj - k, 16u));
            }
            __syncthreads();
        }
    }
#pragma unroll 8
    for (uint32_t i = tid; i < words; i += nt) gw[i] = sw[i];
    if (16 * words + tid < len && tid < 16) blk[16 * words + tid] = smem[16 * words + tid];
}

// The in-order matches of one block per group, in token order: windows of G
// tokens, each copied in batches that read nothing a match still to be copied
// writes.  For blocks whose matches mostly read the ones just before them, or
// whose levels are too many to list: a step of a chain takes 0.4 us here (a
// store, a load of it from L2), 1.7 us as a level of its own.  12 CTAs per SM
// (80 registers): with 16 it spills.
template <int G>
__global__ void __launch_bounds__(kWaveThreads, 12)
    k_ord_walk(const uint4 *__restrict__ tok, const uint64_t *__restrict__ blk_tok, const uint32_t *__restrict__ tokdst,
               uint8_t *out, uint32_t nb, uint32_t log2bs) {
    Group<G> g;
    griddep_launch_dependents();
    const uint64_t b = (blockIdx.x * (uint64_t)kWaveThreads + threadIdx.x) / G;
    if (b >= nb) return;
    const uint64_t t0 = __ldg(blk_tok + b), t1 = __ldg(blk_tok + b + 1), bpos = b << log2bs;
    const uint4 z4 = make_uint4(0, 0, 0, 0);
    uint4 nt = t0 + g.lane < t1 ? __ldg(tok + t0 + g.lane) : z4;
    uint32_t nd = t0 + g.lane < t1 ? __ldg(tokdst + t0 + g.lane) : 0u;
    griddep_wait();
    for (uint64_t w = t0; w < t1; w += G) {
        const uint4 t = nt;
        const uint64_t d = bpos + nd + t.x;
        const bool more = w + G + g.lane < t1;
        nt = more ? __ldg(tok + w + G + g.lane) : z4;
        nd = more ? __ldg(tokdst + w + G + g.lane) : 0u;
        const uint64_t src = (uint64_t)t.z | ((uint64_t)(t.w & 0xffu) << 32);
        const bool mine = t.y && !(t.w >> 8);
        unsigned rem = g.ballot(mine);
        if (!rem) continue;
        const unsigned deps = same_wave_deps<G>(g, mine, d, src, t.y, log2bs) & rem;
        while (rem) {
            const bool now = ((rem >> g.lane) & 1u) && (deps & rem) == 0u;
            const unsigned batch = g.ballot(now);
            group_copy_batch<G, kUnrollCopy>(g, out, d, out + src, now ? t.y : 0u);
            g.sync();
            rem &= ~batch;
        }
    }
}

// Launch of one step kernel with programmatic stream serialization: its CTAs
// may start (and load their worklist) while the previous kernel's last ones
// finish.
template <class... P, class... A>
int launch_step(void (*k)(P...), uint64_t n, unsigned per_cta, unsigned threads, size_t smem, cudaStream_t st,
                A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = kWavePdl;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)((n + per_cta - 1) / per_cta));
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = 1;
    if (cudaError_t e = cudaLaunchKernelEx(&lc, k, static_cast<P>(args)...); e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

// Levels from `first` on that go in one launch as a run of narrow ones (0: the
// level goes by itself).
uint32_t narrow_run(const std::vector<Step> &levels, uint32_t first, uint32_t count, const void *d_steps) {
    uint32_t e = first;
    while (d_steps && e < count && levels[e].n <= kRunMost) e++;
    return e - first >= kRunMin ? e - first : 0;
}

// Launches of launch_levels.
uint32_t level_launches(const std::vector<Step> &levels, uint32_t count, const void *d_steps) {
    uint32_t n = 0;
    for (uint32_t i = 0; i < count; i += std::max(1u, narrow_run(levels, i, count, d_steps))) n++;
    return n;
}

// Levels: one kernel each (a run of narrow ones one kernel together), fewer
// matches per group in the small ones, whose
// groups are all resident at once and take as long as their own window.  Up
// to kLevelOne (about the warps resident at a time) a group takes one match:
// 64 MiB copy sweep at L = 900 137 -> 115 us, 256 KiB of Markov bytes 38.5 ->
// 36 us, 64 MiB of FASTQ-like text 120 -> 116 us; up to 20000 instead the
// 512 MiB sweep at L = 128 goes from 756 to 780 us.
template <int G>
int launch_levels(const aclz_handle *h, const std::vector<Step> &levels, uint32_t count, const void *d_steps,
                  uint8_t *out, cudaStream_t st) {
    const uint32_t stage = (h->mean_deferred_len >= kStageLongMin ? kStageWarpLong : kStageWarp) / 32 * G;
    constexpr int gpc = kLevelThreads / G;
    for (uint32_t i = 0; i < count; i++) {
        if (const uint32_t run = narrow_run(levels, i, count, d_steps)) {
            if (int rc = launch_step(k_level_run<G>, 1, 1, kRunThreads, 0, st, (const Step *)d_steps + i, run, out))
                return rc;
            i += run - 1;
            continue;
        }
        const uint64_t n = levels[i].n;
        const int part = n <= kLevelOne ? G : n <= kLevelEighth ? 8 : n <= kLevelQuarter ? 4 : 2;
        auto k = part == G ? k_level<G, 1> : part == 8 ? k_level<G, G / 8> : part == 4 ? k_level<G, G / 4> : k_level<G, G / 2>;
        if (int rc = launch_step(k, n, kLevelThreads / part, kLevelThreads, (size_t)gpc * stage, st,
                                 (const uint4 *)levels[i].tri, n, out, stage, h->d_err))
            return rc;
    }
    return ACLZ_OK;
}

// The in-order matches: walked, or by levels, by block where the handle lists
// them so.
template <int G>
int launch_order(const aclz_handle *h, uint8_t *out, cudaStream_t st) {
    if (h->walk)
        return launch_step(k_ord_walk<G>, h->n_blocks, kWaveThreads / G, kWaveThreads, 0, st, (const uint4 *)h->d_tok,
                           h->d_blk_tok, h->d_tokdst, out, h->n_blocks, h->log2_bs);
    if (!h->d_ord) return launch_levels<G>(h, h->steps, h->n_ord_steps, h->d_steps, out, st);
    const size_t smem = std::max<size_t>(h->block_size, 16);
    // the attribute is the largest any call needs, the same on every call
    if (cudaError_t e = cudaFuncSetAttribute(k_ord_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize, 1 << 17);
        e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    const int threads = h->block_size < kOrdSmall ? kOrdThreadsSmall : kOrdThreads;
    return launch_step(k_ord_blocks, h->n_blocks, 1, threads, smem, st, (const uint4 *)h->d_ord,
                       (const uint32_t *)h->d_ord_base, out, h->log2_bs, h->total_len);
}

// Waves >= 1: one kernel each.
template <int G>
int launch_wave_steps(const aclz_handle *h, uint8_t *out, cudaStream_t st) {
    for (size_t i = h->n_ord_steps; i < h->steps.size(); i++)
        if (int rc = launch_step(k_wave_copy<G>, h->steps[i].n, kWaveThreads, kWaveThreads, 0, st,
                                 (const uint4 *)h->steps[i].tri, h->steps[i].n, out, h->log2_bs))
            return rc;
    return ACLZ_OK;
}

template <int G>
int launch_lits(aclz_handle *h, uint8_t *out, cudaStream_t st, bool ranges, bool levels) {
    constexpr int gpc = kLitThreads / G;
    const uint64_t n_done = ranges ? (uint64_t)h->n_blocks * h->n_wave_words : 0;
    const unsigned grid = (unsigned)((h->n_lunits + gpc - 1) / gpc);
    k_lits<G><<<grid, kLitThreads, 0, st>>>((const uint4 *)h->d_lunits, h->n_lunits, h->d_lit, h->d_blk_tok,
                                            h->d_blk_lit, h->d_tokdst, h->d_toklit, out, h->log2_bs, h->d_pending,
                                            h->d_done, n_done, h->n_wave_words, levels ? h->d_err + kBarrierWord : nullptr);
    if (cudaError_t e = cudaGetLastError(); e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

// By levels where the caller left the mode open and the upload found them;
// else the in-order levels, then one kernel per wave.
template <int G>
int launch_waves(aclz_handle *h, uint8_t *out, cudaStream_t st, cudaEvent_t phase, bool by_level) {
    if (int rc = launch_lits<G>(h, out, st, false, false)) return rc;
    if (by_level) return launch_levels<G>(h, h->lsteps, (uint32_t)h->lsteps.size(), h->d_lsteps, out, st);
    if (int rc = launch_order<G>(h, out, st)) return rc;
    if (phase) cudaEventRecord(phase, st);
    return launch_wave_steps<G>(h, out, st);
}

struct Occ {
    int per_sm = 0;
    uint32_t stage_bytes = 0;
    size_t smem = 0;
};

// Dynamic shared memory limit last set on each staged kernel instance.
template <int G, bool STAGED>
size_t &smem_attr() {
    static size_t v = 0;
    return v;
}

// Persistent mode: the literal kernel initialises the per-block done bits;
// after the in-order levels one cooperative launch runs every range of
// waves >= 1.
template <int G, bool STAGED>
int launch_persistent(aclz_handle *h, uint8_t *out, uint32_t ctas_per_sm, cudaStream_t st, cudaEvent_t phase) {
    constexpr int gpc = kThreads / G;
    if (int rc = launch_lits<G>(h, out, st, true, false)) return rc;
    if (int rc = launch_order<G>(h, out, st)) return rc;
    if (phase) cudaEventRecord(phase, st);
    if (!h->n_ranges) return launch_wave_steps<G>(h, out, st);  // none, or no memory for the ranges
    auto fn = k_ranges<G, STAGED>;
    static int sms = 0;
    static Occ occ[5][33];  // [ctas_per_sm request 0..4][G]
    // the occupancy cache and the kernel's shared-memory attribute are
    // process-wide: host threads take turns from the lookup to the launch
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    const uint32_t req = std::min<uint32_t>(ctas_per_sm, 4);
    Occ &o = occ[req][G];
    if (!o.per_sm) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (STAGED) {
            cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
            const uint32_t cps = req ? req : 1;
            const size_t bar = 128 * ((8 * gpc + 127) / 128);
            o.stage_bytes = (uint32_t)(((kSmemPerSm / cps - bar) / gpc) & ~127u);
            o.smem = bar + (size_t)gpc * o.stage_bytes;
            if (cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)o.smem);
                e != cudaSuccess) {
                note_cuda_error(e);
                return ACLZ_E_CUDA;
            }
            smem_attr<G, STAGED>() = o.smem;
        }
        int m = 0;
        if (cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, fn, kThreads, o.smem);
            e != cudaSuccess) {
            note_cuda_error(e);
            return ACLZ_E_CUDA;
        }
        if (!STAGED && req && (int)req < m) m = (int)req;
        o.per_sm = m > 0 ? m : -1;
    }
    if (o.per_sm < 1) return ACLZ_E_UNSUPPORTED;
    if (STAGED && smem_attr<G, STAGED>() != o.smem) {
        if (cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)o.smem);
            e != cudaSuccess) {
            note_cuda_error(e);
            return ACLZ_E_CUDA;
        }
        smem_attr<G, STAGED>() = o.smem;
    }
    const uint64_t need = (h->n_ranges + gpc - 1) / gpc;
    unsigned grid = (unsigned)std::min<uint64_t>((uint64_t)o.per_sm * sms, need ? need : 1);
    const uint4 *ranges = (const uint4 *)h->d_ranges;
    uint64_t n_ranges = h->n_ranges;
    const uint4 *seg = (const uint4 *)h->d_seg;
    const uint32_t *pieces = h->d_seg_pieces;
    uint32_t *seg_cnt = h->d_seg_cnt;
    unsigned long long *done = (unsigned long long *)h->d_done;
    uint32_t ww = h->n_wave_words;
    const uint4 *tri = (const uint4 *)h->d_tri;
    uint32_t log2bs = h->log2_bs;
    uint32_t sb = o.stage_bytes;
    uint32_t *err = h->d_err;
    uint32_t spin_limit =
        (uint32_t)std::min<uint64_t>(kSpinLimitMax, (uint64_t)kSpinLimitMin * std::max<uint32_t>(1u, h->n_waves / 256));
    void *args[] = {&ranges, &n_ranges, &seg, &pieces, &seg_cnt, &done, &ww, &tri, &out, &log2bs, &sb, &err, &spin_limit};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)fn, dim3(grid), dim3(kThreads), args, o.smem, st);
    if (e == cudaErrorCooperativeLaunchTooLarge && o.per_sm > 1) {
        // fewer co-resident CTAs than the occupancy estimate: one per SM
        cudaGetLastError();
        o.per_sm = 1;
        grid = (unsigned)std::min<uint64_t>((uint64_t)sms, need ? need : 1);
        e = cudaLaunchCooperativeKernel((const void *)fn, dim3(grid), dim3(kThreads), args, o.smem, st);
    }
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

// Staged persistent mode by levels: the literal kernel, then every level in
// one cooperative launch.
template <int G>
int launch_levels_persistent(aclz_handle *h, uint8_t *out, uint32_t ctas_per_sm, cudaStream_t st, cudaEvent_t phase) {
    if (int rc = launch_lits<G>(h, out, st, false, true)) return rc;
    if (h->d_ord || h->walk)
        if (int rc = launch_order<G>(h, out, st)) return rc;
    if (phase) cudaEventRecord(phase, st);
    constexpr int gpc = kPersThreads / G;
    const uint32_t ctas = ctas_per_sm ? std::min<uint32_t>(ctas_per_sm, kPersCtas) : kPersCtas;
    constexpr uint32_t bar = 128 * ((16 * gpc + 127) / 128);
    uint32_t stage = ((kSmemPerSm / ctas - bar) / (2 * gpc)) & ~127u;
    const size_t smem = bar + (size_t)2 * gpc * stage;
    int sms = 0;
    auto fn = k_levels_persistent<G>;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
    // the attribute is the largest any call needs, the same on every call
    constexpr uint32_t most = ((kSmemPerSm - bar) / (2 * gpc)) & ~127u;
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(bar + (size_t)2 * gpc * most));
    const Step *steps = (const Step *)h->d_levels;
    uint32_t count = h->n_levels, *err = h->d_err;
    void *args[] = {&steps, &count, &out, &stage, &err};
    if (e == cudaSuccess)
        e = cudaLaunchCooperativeKernel((const void *)fn, dim3((unsigned)sms * ctas), dim3(kPersThreads), args, smem, st);
    if (e == cudaErrorCooperativeLaunchTooLarge && ctas > 1) {
        cudaGetLastError();
        e = cudaLaunchCooperativeKernel((const void *)fn, dim3((unsigned)sms), dim3(kPersThreads), args, smem, st);
    }
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

template <int G>
int launch_persistent_auto(aclz_handle *h, uint8_t *out, const aclz_decode_cfg &c, cudaStream_t st,
                           cudaEvent_t phase) {
    bool staged = h->mean_deferred_len >= (double)kTmaMin;
    if (c.flags & ACLZ_FLAG_STAGED) staged = true;
    if (c.flags & ACLZ_FLAG_REGISTERS) staged = false;
    // levels hold in-order and deferred matches: no place for the event then
    if (staged && h->n_levels && !(phase && h->n_ord_steps))
        return launch_levels_persistent<G>(h, out, c.ctas_per_sm, st, phase);
    return staged ? launch_persistent<G, true>(h, out, c.ctas_per_sm, st, phase)
                  : launch_persistent<G, false>(h, out, c.ctas_per_sm, st, phase);
}

}  // namespace

namespace {

// Levels take the place of waves only when the caller left the mode open (an
// explicit ACLZ_MODE_WAVES is one kernel per wave) and no event goes between
// the phases.
bool goes_by_level(const aclz_handle *h, const aclz_decode_cfg *cfg, bool phase) {
    return h->by_level && !phase && (!cfg || cfg->mode == ACLZ_MODE_AUTO) && h->mean_deferred_len < kPersistentMin;
}

// Checks cfg and resolves ACLZ_MODE_AUTO for this handle; phase: an event is
// recorded between the phases.
int resolve_cfg(const aclz_handle *h, const aclz_decode_cfg *cfg, bool phase, aclz_decode_cfg &c) {
    c = {32, ACLZ_MODE_AUTO, 0, 0};
    if (cfg) c = *cfg;
    if (c.G != 8 && c.G != 16 && c.G != 32) return ACLZ_E_INVAL;
    if (c.mode != ACLZ_MODE_WAVES && c.mode != ACLZ_MODE_PERSISTENT && c.mode != ACLZ_MODE_AUTO)
        return ACLZ_E_INVAL;
    if (c.mode == ACLZ_MODE_AUTO) {
        // long deferred matches: one persistent launch with TMA staging;
        // short ones: by levels (or waves)
        const double least = (h->by_level && !phase) || h->flat ? kPersistentMin : kPersistentMinWaves;
        c.mode = h->mean_deferred_len < least ? ACLZ_MODE_WAVES : ACLZ_MODE_PERSISTENT;
        if (c.mode == ACLZ_MODE_PERSISTENT && !(c.flags & ACLZ_FLAG_REGISTERS)) c.flags |= ACLZ_FLAG_STAGED;
    }
    if ((c.flags & ACLZ_FLAG_STAGED) && (c.flags & ACLZ_FLAG_REGISTERS)) return ACLZ_E_INVAL;
    if (c.mode == ACLZ_MODE_PERSISTENT && !(c.flags & (ACLZ_FLAG_STAGED | ACLZ_FLAG_REGISTERS)))
        c.flags |= h->mean_deferred_len >= (double)kTmaMin ? ACLZ_FLAG_STAGED : ACLZ_FLAG_REGISTERS;
    return ACLZ_OK;
}

}  // namespace

extern "C" int aclz_decode_plan(const aclz_handle *h, const aclz_decode_cfg *cfg, aclz_decode_cfg *resolved,
                                uint32_t *launches) {
    if (!h) return ACLZ_E_INVAL;
    aclz_decode_cfg c;
    if (int rc = resolve_cfg(h, cfg, false, c)) return rc;
    uint32_t n = 0;
    if (h->n_blocks) {
        const uint32_t order = level_launches(h->steps, h->n_ord_steps, h->d_steps);
        if (c.mode == ACLZ_MODE_PERSISTENT)
            n = (c.flags & ACLZ_FLAG_STAGED) && h->n_levels ? 2
                : 1 + order + (h->n_ranges ? 1 : (uint32_t)h->steps.size() - h->n_ord_steps);
        else if (goes_by_level(h, cfg, false))
            n = 1 + level_launches(h->lsteps, (uint32_t)h->lsteps.size(), h->d_lsteps);
        else
            n = 1 + order + (uint32_t)h->steps.size() - h->n_ord_steps;
        if (h->d_ord || h->walk) n++;
    }
    if (resolved) *resolved = c;
    if (launches) *launches = n;
    return ACLZ_OK;
}

extern "C" int aclz_decode_all_ev(aclz_handle *h, void *d_out, uint64_t cap, const aclz_decode_cfg *cfg,
                                  void *stream, void *phase_event) {
    if (!h || (!d_out && h->total_len)) return ACLZ_E_INVAL;
    if (cap < h->total_len) return ACLZ_E_CAPACITY;
    if (reinterpret_cast<uintptr_t>(d_out) & 15) return ACLZ_E_INVAL;
    aclz_decode_cfg c;
    if (int rc = resolve_cfg(h, cfg, phase_event != nullptr, c)) return rc;
    if (h->n_blocks == 0) return ACLZ_OK;
    cudaStream_t st = (cudaStream_t)stream;
    cudaEvent_t ev = (cudaEvent_t)phase_event;
    uint8_t *out = (uint8_t *)d_out;
    if (c.mode == ACLZ_MODE_PERSISTENT) {
        switch (c.G) {
            case 8: return launch_persistent_auto<8>(h, out, c, st, ev);
            case 16: return launch_persistent_auto<16>(h, out, c, st, ev);
            default: return launch_persistent_auto<32>(h, out, c, st, ev);
        }
    }
    const bool by_level = goes_by_level(h, cfg, ev != nullptr);
    switch (c.G) {
        case 8: return launch_waves<8>(h, out, st, ev, by_level);
        case 16: return launch_waves<16>(h, out, st, ev, by_level);
        default: return launch_waves<32>(h, out, st, ev, by_level);
    }
}

extern "C" int aclz_decode_all(aclz_handle *h, void *d_out, uint64_t cap, const aclz_decode_cfg *cfg,
                               void *stream) {
    return aclz_decode_all_ev(h, d_out, cap, cfg, stream, nullptr);
}

namespace {

// One group waits, bounded, for wave bit 0 of a block whose bits nothing
// sets: the wait the persistent decode does on a stuck source.
__global__ void k_wait_selftest(const unsigned long long *done, uint32_t spin_limit, uint32_t *err) {
    wait_waves_below(done, 1u, err, spin_limit);
}

}  // namespace

extern "C" int aclz_selftest_wait(uint32_t spin_limit, void *stream) {
    if (spin_limit == 0 || spin_limit > kSpinLimitMin) return ACLZ_E_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    void *buf = nullptr;
    if (cudaError_t e = cudaMalloc(&buf, 64); e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_NOMEM;
    }
    uint32_t err = 0;
    cudaError_t e = cudaMemsetAsync(buf, 0, 64, st);
    if (e == cudaSuccess) {
        k_wait_selftest<<<1, 32, 0, st>>>((const unsigned long long *)buf, spin_limit, (uint32_t *)buf + 8);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&err, (uint32_t *)buf + 8, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(buf);
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return (err & kErrTimeout) ? ACLZ_E_TIMEOUT : ACLZ_OK;
}

extern "C" int aclz_device_status(aclz_handle *h, void *stream) {
    if (!h) return ACLZ_E_INVAL;
    uint32_t e = 0;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(&e, h->d_err, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return ACLZ_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return ACLZ_E_CUDA;
    if (e) {
        // a failed persistent decode may leave segment counts mid-way
        cudaMemsetAsync(h->d_err, 0, 4, st);
        if (h->d_seg_cnt) cudaMemsetAsync(h->d_seg_cnt, 0, 4 * h->n_seg, st);
        cudaStreamSynchronize(st);
    }
    if (e & kErrTimeout) return ACLZ_E_TIMEOUT;
    if (e) return ACLZ_E_DEVICE;
    return ACLZ_OK;
}

// ------------------------------------------------------------- graphs

struct aclz_graph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

extern "C" int aclz_graph_create(aclz_handle *h, void *d_out, uint64_t cap, const aclz_decode_cfg *cfg,
                                 void *stream, aclz_graph **out) {
    if (!h || !out) return ACLZ_E_INVAL;
    *out = nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    // one plain decode first: sets kernel attributes and occupancy caches
    int rc = aclz_decode_all(h, d_out, cap, cfg, stream);
    if (rc) return rc;
    if (cudaStreamSynchronize(st) != cudaSuccess) return ACLZ_E_CUDA;
    cudaStream_t cs;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return ACLZ_E_CUDA;
    aclz_graph *g = new aclz_graph();
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        rc = aclz_decode_all(h, d_out, cap, cfg, cs);
        e = cudaStreamEndCapture(cs, &g->graph);
        if (e == cudaSuccess && rc == ACLZ_OK) e = cudaGraphInstantiate(&g->exec, g->graph, 0);
    }
    cudaStreamDestroy(cs);
    if (e != cudaSuccess || rc != ACLZ_OK) {
        if (e != cudaSuccess) note_cuda_error(e);
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->graph) cudaGraphDestroy(g->graph);
        delete g;
        return rc ? rc : ACLZ_E_CUDA;
    }
    *out = g;
    return ACLZ_OK;
}

extern "C" int aclz_graph_launch(aclz_graph *g, void *stream) {
    if (!g) return ACLZ_E_INVAL;
    cudaError_t e = cudaGraphLaunch(g->exec, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

extern "C" int aclz_graph_free(aclz_graph *g) {
    if (!g) return ACLZ_E_INVAL;
    if (g->exec) cudaGraphExecDestroy(g->exec);
    if (g->graph) cudaGraphDestroy(g->graph);
    delete g;
    return ACLZ_OK;
}

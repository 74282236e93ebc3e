// Greedy parse on the GPU: the container the host encoder writes (greedy
// longest match over exact 4-byte-prefix chains, nearest on ties, minimum
// length by distance class), built from the input bytes by kernels.
//
// The chains do not depend on the parse: every earlier position with the
// same 4-byte prefix is a candidate, nearest first.  Sorting the positions
// by (prefix, position) therefore lays every chain out contiguously, so the
// candidates of position p are the entries just before p in that order.
// What a position's best match is does not depend on the parse either, only
// whether the walk stops there does, so every position is scored at once;
// the walk, sequential within an LZ block (a match never crosses its
// block's end), then only steps from match to match.
//
//  1. k_keys          prefix of every position with 4 bytes left
//  2. radix sort      stable, 8-bit digits: k_rs_hist, exclusive scan,
//                     k_rs_scatter (4 passes)
//  3. k_best          best match of every position, one thread each, in
//                     sorted order
//  4. k_parse_blocks  one warp per block: greedy walk, tokens to a per-block
//                     slot array
//  5. scans of the per-block token and literal counts, then k_emit writes
//     the directory, the tokens and the literal bytes of the container
#include <algorithm>
#include <cstring>
#include <vector>

#include "aclz_device.cuh"
#include "aclz_internal.h"
#include "aclz_mem.h"

using namespace aclz;

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr uint32_t kSortPerWarp = 512;                        // 16 chunks of 32
constexpr uint32_t kSortTile = kSortWarps * kSortPerWarp;    // 4096 elements per CTA

__global__ void k_keys(const uint8_t *__restrict__ x, uint64_t m, uint32_t *__restrict__ key,
                       uint32_t *__restrict__ val) {
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m;
         p += (uint64_t)gridDim.x * blockDim.x) {
        key[p] = (uint32_t)x[p] | ((uint32_t)x[p + 1] << 8) | ((uint32_t)x[p + 2] << 16) |
                 ((uint32_t)x[p + 3] << 24);
        val[p] = (uint32_t)p;
    }
}

// Digit counts of one tile, digit-major: hist[d * ntiles + tile].
__global__ void __launch_bounds__(kSortThreads) k_rs_hist(const uint32_t *__restrict__ key, uint64_t m, int shift,
                                                          uint32_t ntiles, uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t a = (uint64_t)blockIdx.x * kSortTile;
    for (uint32_t k = threadIdx.x; k < kSortTile; k += kSortThreads)
        if (a + k < m) atomicAdd(&h[(key[a + k] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(uint64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of one tile: element i of the tile goes to
// base[digit][tile] + (number of earlier elements of the tile with the same
// digit).  Each warp owns 512 consecutive elements, walked 32 at a time in
// order; equal digits within 32 are ranked by lane.
__global__ void __launch_bounds__(kSortThreads) k_rs_scatter(const uint32_t *__restrict__ key,
                                                             const uint32_t *__restrict__ val, uint64_t m, int shift,
                                                             uint32_t ntiles, const uint32_t *__restrict__ base,
                                                             uint32_t *__restrict__ key_out,
                                                             uint32_t *__restrict__ val_out) {
    __shared__ uint32_t cnt[kSortWarps][256];
    const int w = threadIdx.x / 32, lane = threadIdx.x & 31;
    for (int d = lane; d < 256; d += 32) cnt[w][d] = 0;
    __syncwarp();
    const uint64_t a = (uint64_t)blockIdx.x * kSortTile + (uint64_t)w * kSortPerWarp;
    // digit counts of this warp's elements
    for (uint32_t c = 0; c < kSortPerWarp; c += 32) {
        const uint64_t i = a + c + lane;
        const bool v = i < m;
        const uint32_t d = v ? (key[i] >> shift) & 255u : 256u + lane;  // invalid lanes get private keys
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (v && lane == __ffs(peers) - 1) cnt[w][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over warps, per digit, plus the tile's global base
    {
        const uint32_t d = threadIdx.x;
        uint32_t run = base[(uint64_t)d * ntiles + blockIdx.x];
        for (int k = 0; k < kSortWarps; k++) {
            const uint32_t c = cnt[k][d];
            cnt[k][d] = run;
            run += c;
        }
    }
    __syncthreads();
    for (uint32_t c = 0; c < kSortPerWarp; c += 32) {
        const uint64_t i = a + c + lane;
        const bool v = i < m;
        const uint32_t kk = v ? key[i] : 0u;
        const uint32_t d = v ? (kk >> shift) & 255u : 256u + lane;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (v) {
            const uint32_t dst = cnt[w][d] + __popc(peers & ((1u << lane) - 1u));
            key_out[dst] = kk;
            val_out[dst] = val[i];
        }
        __syncwarp();
        if (v && lane == __ffs(peers) - 1) cnt[w][d] += __popc(peers);
        __syncwarp();
    }
}

// 8 bytes at a (little endian) from two aligned words; needs a + 16 <= the
// padded end of the buffer.
__device__ __forceinline__ uint64_t ld8u(const uint8_t *a) {
    const uintptr_t u = reinterpret_cast<uintptr_t>(a);
    const uint64_t *w = reinterpret_cast<const uint64_t *>(u & ~(uintptr_t)7);
    const uint32_t sh = (uint32_t)(u & 7) * 8;
    const uint64_t lo = w[0];
    if (!sh) return lo;
    return (lo >> sh) | (w[1] << (64 - sh));
}

// Common prefix of x[q..] and x[p..], at most lim bytes (q < p).
__device__ __forceinline__ uint32_t common_len(const uint8_t *x, uint64_t q, uint64_t p, uint32_t lim) {
    uint32_t len = 0;
    while (len + 8 <= lim) {
        const uint64_t a = ld8u(x + q + len), b = ld8u(x + p + len);
        if (a != b) return len + (uint32_t)(__ffsll((long long)(a ^ b)) - 1) / 8;
        len += 8;
    }
    while (len < lim && x[q + len] == x[p + len]) len++;
    return len;
}

__device__ __forceinline__ int dclass(uint64_t d) { return d < 128 ? 0 : d < 16384 ? 1 : d < 2097152 ? 2 : 3; }

// Match lengths of kCap and more are left to the walk (kLong): scoring them
// for every position of a long repeat would cost its length squared.
constexpr uint32_t kCap = 64, kLong = 255;
constexpr int kBestThreads = 256;
constexpr uint32_t kHalo = 64;             // candidates per round
constexpr uint32_t kLenWindow = 32 * 16;  // positions a warp of the walk holds

__device__ __forceinline__ uint32_t class_min(uint32_t d, uint32_t T) {
    return (T >> (8 * dclass(d))) & 255u;
}

// Best match of every position: thread r takes the position p of rank r.
// Its candidates are the entries of rank r - 1, r - 2, ... while their
// prefix is p's, at most depth of them and no farther than window; the
// longest whose length (capped at the distance and the block end) meets its
// distance class minimum wins, the nearest on ties.  best_len[p] receives
// the length (0, as cleared before, when there is none) and best_src[p] the
// source; best_len[p] = kLong and best_src[p] = r when a candidate matches
// kCap bytes.
//
// Neighbouring ranks share their candidates, so a CTA stages the entries of
// its ranks and of the kHalo before them (prefix, position and the 32 bytes
// after the prefix) in shared memory.  A round first tests its candidates
// against the bytes any match must have (a 64-bit compare each, no branch),
// then scores those that passed, each lane its own; only candidates that
// match all 36 staged bytes go back to the input.  Issue-bound; 16 MiB of
// word text at depth 64 is scored in 0.93 ms (1.6 ms when each candidate was
// tested and scored in turn with 16 bytes staged; 135 ms with one warp per
// block scoring one position at a time).
__global__ void __launch_bounds__(kBestThreads) k_best(const uint8_t *__restrict__ x, uint64_t n, uint64_t m,
                                                       uint32_t log2bs, const uint32_t *__restrict__ key_s,
                                                       const uint32_t *__restrict__ val_s, const uint8_t *mm,
                                                       const uint8_t *__restrict__ block_mm, uint32_t depth,
                                                       uint64_t window, uint8_t *__restrict__ best_len,
                                                       uint32_t *__restrict__ best_src) {
    __shared__ uint32_t skey[kBestThreads + kHalo], spos[kBestThreads + kHalo];
    __shared__ unsigned long long swin[4][kBestThreads + kHalo];  // the 32 bytes after the prefix
    const uint64_t r0 = (uint64_t)blockIdx.x * kBestThreads;
    const uint64_t r = r0 + threadIdx.x;
    bool live = r < m;
    uint32_t kp = 0, p = 0, T = 0, rem = 0, need = 0, blen = 0, bsrc = 0;
    unsigned long long own[4] = {0, 0, 0, 0}, mask = 0;
    // bytes 4 .. need - 1 of a candidate must match (up to 12 of them)
    auto set_need = [&](uint32_t v) {
        need = v;
        mask = v >= 12 ? ~0ULL : (v <= 4 ? 0ULL : (1ULL << (8 * (v - 4))) - 1ULL);
    };
    for (uint32_t kb = 0; kb < depth; kb += kHalo) {
        for (uint32_t i = threadIdx.x; i < kBestThreads + kHalo; i += kBestThreads) {
            const long long rr = (long long)r0 - (long long)kb - (long long)kHalo + (long long)i;
            uint32_t k = 0, q = 0;  // places before rank 0 are never looked at
            if (rr >= 0 && (uint64_t)rr < m) {
                k = __ldg(key_s + rr);
                q = __ldg(val_s + rr);
            }
            skey[i] = k;
            spos[i] = q;
            // 32 bytes from five aligned words (the input is readable, zero,
            // for 64 bytes past its end)
            const uintptr_t at = reinterpret_cast<uintptr_t>(x + q + 4);
            const uint64_t *w = reinterpret_cast<const uint64_t *>(at & ~(uintptr_t)7);
            const uint32_t sh = (uint32_t)(at & 7) * 8;
            uint64_t a = __ldg(w);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint64_t b = __ldg(w + j + 1);
                swin[j][i] = sh ? (a >> sh) | (b << (64 - sh)) : a;
                a = b;
            }
        }
        __syncthreads();
        if (kb == 0 && live) {
            kp = skey[threadIdx.x + kHalo];
            p = spos[threadIdx.x + kHalo];
#pragma unroll
            for (int j = 0; j < 4; j++) own[j] = swin[j][threadIdx.x + kHalo];
            const uint32_t b = p >> log2bs;
            const uint64_t bend = min((uint64_t)(b + 1) << log2bs, n);
            rem = (uint32_t)(bend - p);
            const uint8_t *Tp = block_mm ? block_mm + 4 * (uint64_t)b : mm;
            T = (uint32_t)Tp[0] | ((uint32_t)Tp[1] << 8) | ((uint32_t)Tp[2] << 16) | ((uint32_t)Tp[3] << 24);
            set_need(min(min((uint32_t)Tp[0], (uint32_t)Tp[1]), min((uint32_t)Tp[2], (uint32_t)Tp[3])));
            if (rem < need) live = false;
        }
        // candidates of this round: the entries with this prefix (the keys are
        // in order from rank 0 on, so they are a run that ends just before the
        // own entry; a live position has rank kb or more)
        uint32_t kn = 0;
        if (live) {
            const uint32_t top = threadIdx.x + kHalo;  // entry of rank r - kb
            const uint32_t rank0 = kb + kHalo > r0 ? (uint32_t)(kb + kHalo - r0) : 0u;  // entry of rank 0
            uint32_t lo = max(top - kHalo, rank0), hi = top;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (skey[mid] == kp) hi = mid; else lo = mid + 1;
            }
            kn = top - lo;
            live = kn == kHalo;  // the chain may go on past this round
            if (kn > depth - kb) kn = depth - kb;
        }
        // bit k: candidate k (rank r - 1 - (kb + k)) has the bytes it needs
        unsigned long long hits = 0;
#pragma unroll 16
        for (int k = 0; k < (int)kHalo; k++)
            if (!((swin[0][threadIdx.x + kHalo - 1 - k] ^ own[0]) & mask)) hits |= 1ULL << k;
        if (kn < kHalo) hits &= (1ULL << kn) - 1ULL;
        for (; hits; hits &= hits - 1) {
            const uint32_t e = threadIdx.x + kHalo - (uint32_t)__ffsll((long long)hits);
            const uint32_t q = spos[e], d = p - q;
            if ((uint64_t)d > window) {
                live = false;
                break;
            }
            const uint32_t lim = d < rem ? d : rem;
            if (((swin[0][e] ^ own[0]) & mask) || lim < need) continue;
            uint32_t len = 4;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const unsigned long long xj = swin[j][e] ^ own[j];
                if (xj) {
                    len += (uint32_t)(__ffsll((long long)xj) - 1) / 8;
                    break;
                }
                len += 8;
            }
            if (len == 36) {
                const uint32_t cap = lim < kCap ? lim : kCap;
                if (cap > 36) len = 36 + common_len(x, (uint64_t)q + 36, (uint64_t)p + 36, cap - 36);
                if (len >= kCap) {
                    blen = kLong;
                    bsrc = (uint32_t)r;
                    live = false;
                    break;
                }
            }
            len = len < lim ? len : lim;
            if (len >= need && len >= class_min(d, T)) {
                blen = len;
                bsrc = q;
                set_need(len + 1 > need ? len + 1 : need);
                if (need > rem) {  // no longer match fits the block
                    live = false;
                    break;
                }
            }
        }
        if (!__syncthreads_or(live && kb + kHalo < depth)) break;
    }
    if (blen) {
        best_len[p] = (uint8_t)blen;
        best_src[p] = bsrc;
    }
}

struct TokOut {
    uint32_t lit, len;
    uint64_t src;
};

// Best match of position p (rank r) whatever its length, lanes scoring 32
// candidates at a time by the rule of k_best; *len 0 when there is none.
__device__ __forceinline__ void best_long(const uint8_t *__restrict__ x, const uint32_t *__restrict__ key_s,
                                          const uint32_t *__restrict__ val_s, uint64_t p, uint64_t bend, uint32_t r,
                                          uint32_t T, uint32_t depth, uint64_t window, int lane, uint32_t *len_out,
                                          uint32_t *src_out) {
    const uint32_t kp = __ldg(key_s + r);
    uint32_t best_len = 0, best_src = 0;
    bool more = true;
    for (uint32_t k0 = 0; k0 < depth && more; k0 += 32) {
        const uint32_t k = k0 + lane;
        // candidate k exists when it is in the chain, in the window and
        // among the first depth
        bool ok = k < depth && r >= k + 1;
        uint64_t q = 0;
        if (ok) {
            const uint32_t rr = r - 1 - k;
            ok = __ldg(key_s + rr) == kp;
            q = __ldg(val_s + rr);
            ok = ok && p - q <= window;
        }
        uint32_t len = 0;
        if (ok) {
            const uint64_t d = p - q;
            const uint64_t lim = d < bend - p ? d : bend - p;
            len = common_len(x, q, p, (uint32_t)lim);
            if (len < class_min((uint32_t)d, T)) len = 0;
        }
        // longest, then nearest (smallest k): one 64-bit key per lane
        unsigned long long key = len ? ((unsigned long long)len << 32) | (0xffffffffu - k) : 0ULL;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
            key = other > key ? other : key;
        }
        if (key) {
            const uint32_t l = (uint32_t)(key >> 32);
            const uint32_t kk = 0xffffffffu - (uint32_t)key;
            if (l > best_len) {  // an earlier round keeps its ties (nearer)
                best_len = l;
                best_src = __ldg(val_s + (r - 1 - kk));
            }
        }
        more = __all_sync(0xffffffffu, !(k < depth) || ok);  // the chain went on past this round
    }
    *len_out = best_len;
    *src_out = best_src;
}

// One warp per block: the greedy walk over the best matches of k_best.  The
// warp holds the lengths of kLenWindow positions, 16 to a lane, with the
// next window loaded ahead; a step finds the first position with a match
// at or after p, emits its token and moves past it.  Lane i keeps token i of
// the current 32 and looks its source up when they are written.  Tokens go
// to slots[b * cap_tok ...], the place of every 32nd one to starts; ntok[b]
// and nlit[b] receive the counts.  best_len is readable, zero, for two windows past the input.
__global__ void __launch_bounds__(256) k_parse_blocks(const uint8_t *__restrict__ x, uint64_t n, uint32_t bs,
                                                      uint32_t nb, const uint32_t *__restrict__ key_s,
                                                      const uint32_t *__restrict__ val_s,
                                                      const uint8_t *__restrict__ best_len,
                                                      const uint32_t *__restrict__ best_src, const uint8_t *mm,
                                                      const uint8_t *__restrict__ block_mm, uint32_t depth,
                                                      uint64_t window, uint32_t cap_tok, TokOut *__restrict__ slots,
                                                      uint2 *__restrict__ starts, uint32_t *__restrict__ ntok,
                                                      uint32_t *__restrict__ nlit) {
    const uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nb) return;
    const uint8_t *Tp = block_mm ? block_mm + 4 * (uint64_t)b : mm;
    const uint32_t T = (uint32_t)Tp[0] | ((uint32_t)Tp[1] << 8) | ((uint32_t)Tp[2] << 16) | ((uint32_t)Tp[3] << 24);
    const uint64_t bstart = (uint64_t)b * bs;
    const uint64_t bend = bstart + bs < n ? bstart + bs : n;
    TokOut *out = slots + (uint64_t)b * cap_tok;
    uint2 *win = starts + (uint64_t)b * (cap_tok / 32 + 1);
    uint64_t p = bstart, lit_start = bstart;
    uint32_t cnt = 0, lits = 0;
    if (lane == 0) win[0] = make_uint2(0u, 0u);
    // this lane's token of the current 32: literals, length, source (or the
    // position whose source is still to be looked up)
    uint32_t t_lit = 0, t_len = 0, t_src = 0;
    bool t_at = false;
    auto flush = [&](uint32_t k) {  // the first k tokens of the current 32
        if ((uint32_t)lane < k)
            out[(cnt - k) + lane] = TokOut{t_lit, t_len, t_at ? (uint64_t)__ldg(best_src + t_src) : (uint64_t)t_src};
    };
    auto emit = [&](uint32_t lit, uint32_t len, uint32_t src, bool at) {
        if ((uint32_t)lane == (cnt & 31u)) {
            t_lit = lit;
            t_len = len;
            t_src = src;
            t_at = at;
        }
        lits += lit;
        cnt++;
        if (!(cnt & 31u)) {
            flush(32);
            // where the next 32 tokens start, in the block and in its literals
            if (lane == 0) win[cnt / 32] = make_uint2((uint32_t)(lit_start + lit + len - bstart), lits);
        }
    };
    auto load = [&](uint64_t at) { return __ldg(reinterpret_cast<const uint4 *>(best_len + at) + lane); };
    // bit i: position 16 * lane + i of the window has a match
    auto nonzero = [](const uint4 &v) {
        auto four = [](uint32_t w) {
            const uint32_t t = ((w & 0x7f7f7f7fu) + 0x7f7f7f7fu) | w;  // bit 7 of each byte that is not 0
            return ((t >> 7) & 1u) | ((t >> 14) & 2u) | ((t >> 21) & 4u) | ((t >> 28) & 8u);
        };
        return four(v.x) | (four(v.y) << 4) | (four(v.z) << 8) | (four(v.w) << 12);
    };
    uint64_t base = p & ~(uint64_t)(kLenWindow - 1);
    uint4 cur = load(base), nxt = load(base + kLenWindow);
    uint32_t bits = nonzero(cur);
    while (p < bend) {
        const int below = (int)(p - base) - 16 * lane;  // positions of this lane before p
        const uint32_t left = below <= 0 ? bits : (below >= 16 ? 0u : bits & (0xffffu << below));
        const unsigned have = __ballot_sync(0xffffffffu, left != 0);
        if (have) {
            const uint32_t at = (uint32_t)__ffs(left) - 1u;
            const uint32_t word = at & 8 ? (at & 4 ? cur.w : cur.z) : (at & 4 ? cur.y : cur.x);
            const uint32_t mine = ((word >> (8 * (at & 3))) & 255u) | (at << 8);
            const int f = __ffs(have) - 1;
            const uint32_t got = __shfl_sync(0xffffffffu, mine, f);
            const uint64_t q = base + 16 * (uint32_t)f + (got >> 8);
            if (q >= bend) break;
            uint32_t len = got & 255u, src = (uint32_t)q;
            const bool lng = len == kLong;
            if (lng) best_long(x, key_s, val_s, q, bend, __ldg(best_src + q), T, depth, window, lane, &len, &src);
            if (!len) {
                p = q + 1;
            } else {
                emit((uint32_t)(q - lit_start), len, src, !lng);
                p = q + len;
                lit_start = p;
            }
        } else {
            p = base + kLenWindow;
        }
        if (p - base >= kLenWindow) {
            const uint64_t nbase = p & ~(uint64_t)(kLenWindow - 1);
            if (p < bend) {
                cur = nbase == base + kLenWindow ? nxt : load(nbase);
                nxt = load(nbase + kLenWindow);
                bits = nonzero(cur);
            }
            base = nbase;
        }
    }
    if (lit_start < bend || cnt == 0) emit((uint32_t)(bend - lit_start), 0u, 0u, false);
    flush(cnt & 31u);
    if (lane == 0) {
        ntok[b] = cnt;
        nlit[b] = lits;
    }
}

// One CTA per block: directory entry, tokens and literal bytes of the
// container (tok_off / lit_off: exclusive scans of the counts; starts: place
// of every 32nd token), 32 tokens a warp at a time.
__global__ void __launch_bounds__(256) k_emit(const uint8_t *__restrict__ x, uint32_t bs,
                                              const TokOut *__restrict__ slots, const uint2 *__restrict__ starts,
                                              uint32_t cap_tok, const uint32_t *__restrict__ ntok,
                                              const uint32_t *__restrict__ tok_off,
                                              const uint32_t *__restrict__ lit_off, const uint8_t *mm,
                                              const uint8_t *__restrict__ block_mm, uint8_t *__restrict__ dir,
                                              uint8_t *__restrict__ tok, uint8_t *__restrict__ lit) {
    Group<32> g;
    const uint32_t b = blockIdx.x;
    const uint32_t nt = ntok[b];
    const uint64_t t0 = tok_off[b], l0 = lit_off[b];
    if (threadIdx.x < 8) {
        // tok_off u64, lit_off u64, n_tok u32, max_wave u16 0, flags u16 0,
        // min_match[4], pad u32 0: 32 bytes as eight words
        const uint8_t *T = block_mm ? block_mm + 4 * (uint64_t)b : mm;
        uint32_t v = 0;
        switch (threadIdx.x) {
            case 0: v = (uint32_t)t0; break;
            case 1: v = (uint32_t)(t0 >> 32); break;
            case 2: v = (uint32_t)l0; break;
            case 3: v = (uint32_t)(l0 >> 32); break;
            case 4: v = nt; break;
            case 6: v = (uint32_t)T[0] | ((uint32_t)T[1] << 8) | ((uint32_t)T[2] << 16) | ((uint32_t)T[3] << 24); break;
            default: v = 0; break;
        }
        reinterpret_cast<uint32_t *>(dir + 32 * (uint64_t)b)[threadIdx.x] = v;
    }
    const TokOut *in = slots + (uint64_t)b * cap_tok;
    const uint2 *win = starts + (uint64_t)b * (cap_tok / 32 + 1);
    for (uint32_t w = 32 * (threadIdx.x / 32); w < nt; w += 256) {
        const uint32_t i = w + g.lane;
        const bool v = i < nt;
        const uint2 at = win[w / 32];
        const TokOut t = v ? in[i] : TokOut{0u, 0u, 0ULL};
        // place of this token's literals in the block and in its literals:
        // those of the window plus the lengths of the tokens before it
        const uint32_t incl = g.scan_incl(t.lit + t.len), lincl = g.scan_incl(t.lit);
        if (v) {
            uint32_t *tw = reinterpret_cast<uint32_t *>(tok + 16 * (t0 + i));
            tw[0] = t.lit;
            tw[1] = t.len;
            tw[2] = t.len ? (uint32_t)t.src : 0u;
            tw[3] = t.len ? (uint32_t)(t.src >> 32) & 0xffu : 0u;
        }
        const uint64_t from = (uint64_t)b * bs + at.x + incl - (t.lit + t.len);
        group_copy<32, 2, kFromConst>(g, lit, l0 + at.y + lincl - t.lit, x + from, t.lit);
    }
}

}  // namespace

int aclz::device_sort_pairs(uint32_t **k0, uint32_t **v0, uint32_t **k1, uint32_t **v1, uint64_t n, int passes,
                            void *stream) {
    if (!n) return ACLZ_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t ntiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
    const uint64_t hn = 256ULL * ntiles;
    uint32_t *hist = nullptr;
    cudaError_t e = dev_alloc((void **)&hist, 4 * (hn + 4), st);
    int rc = ACLZ_OK;
    for (int pass = 0; pass < passes && e == cudaSuccess && rc == ACLZ_OK; pass++) {
        const int shift = 8 * pass;
        k_rs_hist<<<ntiles, kSortThreads, 0, st>>>(*k0, n, shift, ntiles, hist);
        rc = device_excl_scan(hist, hn, hist + hn, st);
        if (rc) break;
        k_rs_scatter<<<ntiles, kSortThreads, 0, st>>>(*k0, *v0, n, shift, ntiles, hist, *k1, *v1);
        e = cudaGetLastError();
        std::swap(*k0, *k1);
        std::swap(*v0, *v1);
    }
    dev_free(hist, st);
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return e == cudaErrorMemoryAllocation ? ACLZ_E_NOMEM : ACLZ_E_CUDA;
    }
    return rc;
}

extern "C" int aclz_encode_gpu(const void *host_src, uint64_t n, const aclz_encode_params *p,
                               const uint8_t *block_min_match, void *stream, void *host_out, uint64_t cap,
                               uint64_t *out_size) {
    if (!p || !out_size || (n && !host_src)) return ACLZ_E_INVAL;
    const uint32_t bs = p->block_size;
    if (!is_pow2(bs) || bs < kMinBlock || bs > kMaxBlock) return ACLZ_E_INVAL;
    for (int i = 0; i < 4; i++)
        if (p->min_match[i] < 4) return ACLZ_E_INVAL;
    // positions, ranks and counts are 32-bit here
    if (n >= (1ULL << 32) - 64) return ACLZ_E_UNSUPPORTED;
    const uint32_t nb = (uint32_t)((n + bs - 1) / bs);
    if (block_min_match)
        for (uint64_t i = 0; i < 4ULL * nb; i++)
            if (block_min_match[i] < 4) return ACLZ_E_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t m = n >= 4 ? n - 3 : 0;
    const uint32_t cap_tok = bs / 4 + 1;
    int rc = ACLZ_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == ACLZ_OK) {
            note_cuda_error(e);
            rc = e == cudaErrorMemoryAllocation ? ACLZ_E_NOMEM : ACLZ_E_CUDA;
        }
        return rc == ACLZ_OK;
    };
    Scratch dx, dk0, dv0, dk1, dv1, dlen, dslots, dstarts, dntok, dnlit, dtoff, dloff, dmm, dbmm, dcont;
    // the input with 64 zero bytes after it (the 8-byte compares read whole
    // aligned words, the staging of k_best 40 bytes from a prefix on)
    const uint64_t tail = n & ~(uint64_t)15;
    if (!ck(dx.alloc(n + 64, st)) || !ck(cudaMemsetAsync((uint8_t *)dx.p + tail, 0, n + 64 - tail, st)) ||
        (n && !ck(cudaMemcpyAsync(dx.p, host_src, n, cudaMemcpyHostToDevice, st))))
        return rc;
    const uint64_t mm1 = m ? m : 1;
    if (!ck(dk0.alloc(4 * mm1, st)) || !ck(dv0.alloc(4 * mm1, st)) || !ck(dk1.alloc(4 * mm1, st)) ||
        !ck(dv1.alloc(4 * mm1, st)) || !ck(dlen.alloc(n + 3 * kLenWindow, st)))
        return rc;
    uint32_t *k0 = (uint32_t *)dk0.p, *v0 = (uint32_t *)dv0.p, *k1 = (uint32_t *)dk1.p, *v1 = (uint32_t *)dv1.p;
    if (m) {
        const unsigned g = (unsigned)std::min<uint64_t>(8192, (m + 255) / 256);
        k_keys<<<g, 256, 0, st>>>((const uint8_t *)dx.p, m, k0, v0);
        ck(cudaGetLastError());
        if (rc || (rc = device_sort_pairs(&k0, &v0, &k1, &v1, m, 4, st))) return rc;
    }
    // thresholds
    if (!ck(dmm.alloc(16, st)) || !ck(cudaMemcpyAsync(dmm.p, p->min_match, 4, cudaMemcpyHostToDevice, st)))
        return rc;
    if (block_min_match && (!ck(dbmm.alloc(4ULL * nb, st)) ||
                            !ck(cudaMemcpyAsync(dbmm.p, block_min_match, 4ULL * nb, cudaMemcpyHostToDevice, st))))
        return rc;
    if (!ck(dslots.alloc(sizeof(TokOut) * (uint64_t)cap_tok * (nb ? nb : 1), st)) ||
        !ck(dstarts.alloc(sizeof(uint2) * (uint64_t)(cap_tok / 32 + 1) * (nb ? nb : 1), st)) ||
        !ck(dntok.alloc(4ULL * nb + 16, st)) || !ck(dnlit.alloc(4ULL * nb + 16, st)) ||
        !ck(dtoff.alloc(4ULL * nb + 16, st)) || !ck(dloff.alloc(4ULL * nb + 16, st)))
        return rc;
    const uint64_t window = p->window;
    if (nb) {
        // k1 and v1 are free after the sort; v1 holds the sources
        if (!ck(cudaMemsetAsync(dlen.p, 0, n + 3 * kLenWindow, st))) return rc;
        if (m)
            k_best<<<(unsigned)((m + kBestThreads - 1) / kBestThreads), kBestThreads, 0, st>>>(
                (const uint8_t *)dx.p, n, m, log2u(bs), k0, v0, (const uint8_t *)dmm.p, (const uint8_t *)dbmm.p,
                p->chain_depth, window, (uint8_t *)dlen.p, v1);
        k_parse_blocks<<<(nb + 7) / 8, 256, 0, st>>>((const uint8_t *)dx.p, n, bs, nb, k0, v0,
                                                     (const uint8_t *)dlen.p, v1, (const uint8_t *)dmm.p,
                                                     (const uint8_t *)dbmm.p, p->chain_depth, window, cap_tok,
                                                     (TokOut *)dslots.p, (uint2 *)dstarts.p, (uint32_t *)dntok.p,
                                                     (uint32_t *)dnlit.p);
        if (!ck(cudaGetLastError())) return rc;
        ck(cudaMemcpyAsync(dtoff.p, dntok.p, 4ULL * nb, cudaMemcpyDeviceToDevice, st));
        ck(cudaMemcpyAsync(dloff.p, dnlit.p, 4ULL * nb, cudaMemcpyDeviceToDevice, st));
        if (rc) return rc;
        if ((rc = device_excl_scan((uint32_t *)dtoff.p, nb, (uint32_t *)dtoff.p + nb, st))) return rc;
        if ((rc = device_excl_scan((uint32_t *)dloff.p, nb, (uint32_t *)dloff.p + nb, st))) return rc;
    }
    uint32_t tot[2] = {0, 0};
    if (nb) {
        ck(cudaMemcpyAsync(&tot[0], (uint32_t *)dtoff.p + nb, 4, cudaMemcpyDeviceToHost, st));
        ck(cudaMemcpyAsync(&tot[1], (uint32_t *)dloff.p + nb, 4, cudaMemcpyDeviceToHost, st));
        ck(cudaStreamSynchronize(st));
        if (rc) return rc;
    }
    const uint64_t nt = tot[0], nl = tot[1];
    const uint64_t need = kHdr + (uint64_t)kDirent * nb + (uint64_t)kTok * nt + nl;
    *out_size = need;
    if (!host_out) return ACLZ_OK;
    if (cap < need) return ACLZ_E_CAPACITY;
    if (!ck(dcont.alloc(need ? need : 16, st))) return rc;
    uint8_t *c = (uint8_t *)dcont.p;
    if (nb) {
        k_emit<<<nb, 256, 0, st>>>((const uint8_t *)dx.p, bs, (const TokOut *)dslots.p, (const uint2 *)dstarts.p,
                                   cap_tok, (const uint32_t *)dntok.p, (const uint32_t *)dtoff.p,
                                   (const uint32_t *)dloff.p, (const uint8_t *)dmm.p, (const uint8_t *)dbmm.p, c + kHdr,
                                   c + kHdr + (uint64_t)kDirent * nb,
                                   c + kHdr + (uint64_t)kDirent * nb + (uint64_t)kTok * nt);
        if (!ck(cudaGetLastError())) return rc;
    }
    // header: "ACLZ", v1, no tags, sizes, thresholds, distance bounds
    uint8_t h[kHdr];
    std::memset(h, 0, kHdr);
    h[0] = 'A'; h[1] = 'C'; h[2] = 'L'; h[3] = 'Z';
    wr16(h + 4, 1);
    wr16(h + 6, 0);
    wr64(h + 8, n);
    wr32(h + 16, bs);
    wr32(h + 20, nb);
    wr64(h + 24, nt);
    wr64(h + 32, nl);
    wr32(h + 40, 0);
    std::memcpy(h + 44, p->min_match, 4);
    const uint32_t bounds[3] = {128, 16384, 2097152};
    for (int i = 0; i < 3; i++) wr32(h + 48 + 4 * i, bounds[i]);
    std::memcpy(host_out, h, kHdr);
    if (need > kHdr) ck(cudaMemcpyAsync((uint8_t *)host_out + kHdr, c + kHdr, need - kHdr, cudaMemcpyDeviceToHost, st));
    ck(cudaStreamSynchronize(st));
    return rc;
}

// Device-side building blocks of the decode kernels: G-lane groups
// (G in {8, 16, 32} lanes of one warp cooperate on one LZ block, Sec. II),
// group scans and ballots, and the packed 16-byte-vectorised copy that deals
// the aligned 16-byte output chunks of several jobs to the group's lanes
// (Sec. III-C: short matches leave lanes idle unless several are packed into
// one pass).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace aclz {

// device status bits latched in a handle's error word
constexpr uint32_t kErrTimeout = 1u;
constexpr uint32_t kErrCorrupt = 2u;

// most polls of any bounded wait
constexpr uint32_t kSpinLimitMax = 1u << 26;

// Bounded grid barrier of a cooperative launch: the CTA's writes are visible
// to every CTA that leaves it.  target: CTAs times barriers so far (*count
// starts at 0).  One release and one acquire on one word: every further hop
// (a flag set by the last arrival, a tree of counters) cost 0.8 us more than
// it saved.  False, on every thread, when a thread of the CTA comes with ok
// false, when the wait ran out, or when another CTA already gave up.
__device__ __forceinline__ bool grid_barrier(uint32_t *count, uint32_t target, bool ok, uint32_t *err) {
    if (__syncthreads_or(!ok)) return false;
    bool out = false;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        uint32_t spins = 0, v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            if (v >= target) break;
            if (++spins > kSpinLimitMax) {
                atomicOr(err, kErrTimeout);
                out = true;
                break;
            }
            if ((spins & 255) == 0 && (*(volatile uint32_t *)err & kErrTimeout)) {
                out = true;
                break;
            }
            if (spins > 64) __nanosleep(64);
        }
    }
    return !__syncthreads_or(out);
}

template <int G>
struct Group {
    static_assert(G == 8 || G == 16 || G == 32, "G must be 8, 16 or 32");
    unsigned mask;  // this group's lanes within the warp
    int lane;       // 0..G-1
    int shift;      // first warp lane of the group

    __device__ __forceinline__ Group() {
        const int wl = threadIdx.x & 31;
        lane = wl & (G - 1);
        shift = wl - lane;
        mask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << shift);
    }
    __device__ __forceinline__ void sync() const { __syncwarp(mask); }
    __device__ __forceinline__ unsigned ballot(bool p) const {
        return (__ballot_sync(mask, p) & mask) >> shift;
    }
    template <typename T>
    __device__ __forceinline__ T shfl(T v, int src) const { return __shfl_sync(mask, v, src, G); }
    template <typename T>
    __device__ __forceinline__ T shfl_up(T v, int d) const { return __shfl_up_sync(mask, v, d, G); }
    // inclusive prefix sum over the group's lanes
    template <typename T>
    __device__ __forceinline__ T scan_incl(T v) const {
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            T t = shfl_up(v, o);
            if (lane >= o) v += t;
        }
        return v;
    }
    __device__ __forceinline__ unsigned lanemask_lt() const { return (1u << lane) - 1u; }
    // bitwise or over the group's lanes
    __device__ __forceinline__ unsigned or_all(unsigned v) const {
        if constexpr (G == 32) {
            return __reduce_or_sync(0xffffffffu, v);
        } else {
#pragma unroll
            for (int o = 1; o < G; o <<= 1) v |= __shfl_xor_sync(mask, v, o, G);
            return v;
        }
    }
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint4 lds16_u32(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");  // not before the stores, waits and barriers ahead of it
    return v;
}

// Bytes [r, r + 16) of the 32-byte little-endian concatenation a || b.
__device__ __forceinline__ uint4 window16(uint4 a, uint4 b, uint32_t r) {
    const bool two = r & 8, one = r & 4;
    const uint32_t sh = (r & 3) * 8;
    const uint32_t y0 = two ? a.z : a.x, y1 = two ? a.w : a.y, y2 = two ? b.x : a.z, y3 = two ? b.y : a.w,
                   y4 = two ? b.z : b.x, y5 = two ? b.w : b.y;
    const uint32_t z0 = one ? y1 : y0, z1 = one ? y2 : y1, z2 = one ? y3 : y2, z3 = one ? y4 : y3,
                   z4 = one ? y5 : y4;
    uint4 o;
    o.x = __funnelshift_r(z0, z1, sh);
    o.y = __funnelshift_r(z1, z2, sh);
    o.z = __funnelshift_r(z2, z3, sh);
    o.w = __funnelshift_r(z3, z4, sh);
    return o;
}

// Where a copy reads: L2 (bytes other kernels wrote), the non-coherent L1
// path (bytes nobody writes during the kernel), or shared memory (addresses
// in the shared window).
enum Source { kFromL2, kFromConst, kFromShared };

// One aligned source word.
template <Source SRC>
__device__ __forceinline__ uint4 ld_word(uintptr_t a) {
    if (SRC == kFromShared) return lds16_u32((uint32_t)a);
    return SRC == kFromConst ? __ldg(reinterpret_cast<const uint4 *>(a)) : __ldcg(reinterpret_cast<const uint4 *>(a));
}

// The 16 bytes from s on, of which the first n (1 <= n <= 16) are wanted:
// only the aligned words holding wanted bytes are read.
template <Source SRC>
__device__ __forceinline__ uint4 load_bytes(uintptr_t s, uint32_t n) {
    const uint32_t r = (uint32_t)s & 15u;
    const uintptr_t base = s & ~(uintptr_t)15;
    uint4 a = ld_word<SRC>(base), b = a;
    if (r + n > 16) b = ld_word<SRC>(base + 16);
    return window16(a, b, r);
}

// The first n (0 <= n <= 16) bytes of v to p, as naturally aligned stores:
// 1, 2 and 4 bytes up to the next 8-byte boundary, then 8, 8, 4, 2 and 1 as
// they fit (what is left after a skipped step is shorter than that step).
__device__ __forceinline__ void store_bytes(uintptr_t p, uint4 v, uint32_t n) {
    if ((p & 1) && n) {
        *reinterpret_cast<uint8_t *>(p) = (uint8_t)v.x;
        v.x = __funnelshift_r(v.x, v.y, 8);
        v.y = __funnelshift_r(v.y, v.z, 8);
        v.z = __funnelshift_r(v.z, v.w, 8);
        v.w >>= 8;
        p += 1;
        n -= 1;
    }
    if ((p & 2) && n >= 2) {
        *reinterpret_cast<uint16_t *>(p) = (uint16_t)v.x;
        v.x = __funnelshift_r(v.x, v.y, 16);
        v.y = __funnelshift_r(v.y, v.z, 16);
        v.z = __funnelshift_r(v.z, v.w, 16);
        v.w >>= 16;
        p += 2;
        n -= 2;
    }
    if ((p & 4) && n >= 4) {
        *reinterpret_cast<uint32_t *>(p) = v.x;
        v.x = v.y;
        v.y = v.z;
        v.z = v.w;
        p += 4;
        n -= 4;
    }
    if (n >= 8) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(v.x, v.y);
        v.x = v.z;
        v.y = v.w;
        p += 8;
        n -= 8;
        if (n >= 8) {
            *reinterpret_cast<uint2 *>(p) = make_uint2(v.x, v.y);
            n -= 8;  // 0: n was 16
        }
    }
    if (n >= 4) {
        *reinterpret_cast<uint32_t *>(p) = v.x;
        v.x = v.y;
        p += 4;
    }
    if (n & 2) {
        *reinterpret_cast<uint16_t *>(p) = (uint16_t)v.x;
        v.x >>= 16;
        p += 2;
    }
    if (n & 1) *reinterpret_cast<uint8_t *>(p) = (uint8_t)v.x;
}

// Lane of the group's o-th set bit of m (o < popc(m)).
template <int G>
__device__ __forceinline__ int select_bit(unsigned m, uint32_t o) {
    int pos = 0;
#pragma unroll
    for (int w = G / 2; w; w >>= 1)
        if ((uint32_t)__popc(m & ((1u << (pos + w)) - 1u)) <= o) pos += w;
    return pos;
}

// The full 16-byte output chunks of the group's jobs (P: output address of
// a job's first full chunk, S: source address of its first byte, c: chunks),
// numbered in lane order and dealt to the lanes, U per lane per round, loads
// before stores.  The job of a chunk is found from the starts of the jobs
// within the slot of G chunks: one bit per start, or-reduced over the group,
// counted up to the own lane.
template <int G, int U, Source SRC>
__device__ __forceinline__ void copy_full_chunks(const Group<G> &g, uintptr_t P, uintptr_t S, uint32_t c,
                                                 unsigned have) {
    if (have & (have + 1u)) {  // bring the jobs to the lowest lanes
        const uint32_t nj = __popc(have);
        const bool v = (uint32_t)g.lane < nj;
        const int from = v ? select_bit<G>(have, (uint32_t)g.lane) : 0;
        P = (uintptr_t)g.shfl((unsigned long long)P, from);
        S = (uintptr_t)g.shfl((unsigned long long)S, from);
        c = g.shfl(c, from);
        if (!v) c = 0;
    }
    const uint32_t incl = g.scan_incl(c);
    const uint32_t total = g.shfl(incl, G - 1);
    const uint32_t ex = incl - c;
    P -= 16 * (uint64_t)ex;
    S -= 16 * (uint64_t)ex;
    uint32_t before = 0;  // jobs that start in earlier slots
    for (uint32_t base = 0; base < total; base += (uint32_t)G * U) {
        uintptr_t dst[U];
        uint4 a[U], b[U];
        uint32_t r[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t k0 = base + (uint32_t)u * G;  // the same on every lane
            dst[u] = 0;
            if (k0 >= total) continue;
            const uint32_t k = k0 + (uint32_t)g.lane;
            const uint32_t t = ex - k0;
            const unsigned starts = g.or_all((c && t < (uint32_t)G) ? 1u << t : 0u);
            const int j = (int)(before + (uint32_t)__popc(starts & ((2u << g.lane) - 1u)) - 1u);
            before += (uint32_t)__popc(starts);
            const uintptr_t dj = (uintptr_t)g.shfl((unsigned long long)P, j) + 16 * (uint64_t)k;
            const uintptr_t sj = (uintptr_t)g.shfl((unsigned long long)S, j) + 16 * (uint64_t)k;
            if (k < total) {
                dst[u] = dj;
                r[u] = (uint32_t)sj & 15u;
                const uintptr_t w = sj & ~(uintptr_t)15;
                a[u] = ld_word<SRC>(w);
                if (r[u]) b[u] = ld_word<SRC>(w + 16);
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (dst[u]) *reinterpret_cast<uint4 *>(dst[u]) = window16(a[u], b[u], r[u]);
    }
}

// Packed group copy.  Each lane holds one job (p: output address, q:
// source address, n: length; n == 0 for none).  A job of at most 16 bytes is copied
// by its own lane; of a longer one the lane copies the bytes before the
// first and after the last 16-byte boundary of the output, and the full
// chunks between are dealt to the whole group (copy_full_chunks).  Jobs must
// be independent: no job's source may overlap another job's output in the
// same call.
//
// The copy is issue-bound, so it is built to take few instructions.  Against
// a form that searched every chunk's job by shuffles and cut its partial
// chunks from 64-bit fields (about 235 instructions for 32 chunks), whole
// decodes on GB300: 32 MiB of word text at 6/8/10/12, flattened (pieces of
// 3 bytes), 1217 -> 911 us; the 512 MiB copy sweep at L = 128 1096 -> 1038 us;
// 64 MiB of FASTQ-like text at 12/16/24/32 244 -> 230 us.
template <int G, int U, Source SRC>
__device__ __forceinline__ void group_copy_from(const Group<G> &g, uintptr_t p, uintptr_t q, uint32_t n) {
    const uint32_t head = n <= 16 ? n : (0u - (uint32_t)p) & 15u;
    const uint32_t rest = n - head;           // of a job longer than 16 bytes
    const uint32_t tail = rest & 15u, c = rest >> 4;
    uint4 hv = make_uint4(0, 0, 0, 0), tv = hv;
    if (head) hv = load_bytes<SRC>(q, head);
    if (tail) tv = load_bytes<SRC>(q + n - tail, tail);
    const unsigned have = g.ballot(c > 0);
    if (have) copy_full_chunks<G, U, SRC>(g, p + head, q + head, c, have);
    if (g.ballot(head > 0)) store_bytes(p, hv, head);
    if (g.ballot(tail > 0)) store_bytes(p + n - tail, tv, tail);
}

template <int G, int U, Source SRC = kFromL2>
__device__ __forceinline__ void group_copy(const Group<G> &g, uint8_t *out, uint64_t d, const uint8_t *s,
                                           uint32_t n) {
    group_copy_from<G, U, SRC>(g, reinterpret_cast<uintptr_t>(out) + d, reinterpret_cast<uintptr_t>(s), n);
}

// The same for one batch of a chain, where the next batch waits for this one:
// a single job (lane j's) is dealt to the lanes by its chunks at once, without
// the search for every chunk's job.  A step of a chain of 64-byte matches
// takes 0.38 us instead of 0.80 us (0.59 us with a packed copy that found every
// chunk's job by shuffles): 1 MiB of zeros in one block 13.2 -> 6.3 ms, 256 KiB
// in 16 KiB blocks by waves 3.11 -> 1.57 ms, by ranges 3.55 -> 1.88 ms.
template <int G, int U, Source SRC = kFromL2>
__device__ __forceinline__ void group_copy_batch(const Group<G> &g, uint8_t *out, uint64_t d, const uint8_t *s,
                                                 uint32_t n) {
    const unsigned jobs = g.ballot(n > 0);
    if (jobs & (jobs - 1u)) {
        group_copy<G, U, SRC>(g, out, d, s, n);
        return;
    }
    const int j = __ffs(jobs) - 1;
    if (j < 0) return;
    const uintptr_t p = (uintptr_t)g.shfl((unsigned long long)(reinterpret_cast<uintptr_t>(out) + d), j);
    const uintptr_t q = (uintptr_t)g.shfl((unsigned long long)reinterpret_cast<uintptr_t>(s), j);
    const uint32_t m = g.shfl(n, j);
    // stretches of the output between 16-byte boundaries, one a lane
    const uint32_t lead = (uint32_t)p & 15u;
    for (uint32_t k = g.lane; 16 * k < lead + m; k += G) {
        const uint32_t a = k ? 16 * k - lead : 0u, e = min(16 * k + 16 - lead, m);
        const uint4 v = load_bytes<SRC>(q + a, e - a);
        if (e - a == 16)
            *reinterpret_cast<uint4 *>(p + a) = v;
        else
            store_bytes(p + a, v, e - a);
    }
}

// Bytes [r, r + 16) of a || b for a shift r that is the same on every lane
// (a uniform branch picks the word offset).
__device__ __forceinline__ uint4 window16_uniform(const uint4 &a, const uint4 &b, uint32_t q, uint32_t sh) {
    uint32_t w0, w1, w2, w3, w4;
    switch (q) {
        case 0: w0 = a.x; w1 = a.y; w2 = a.z; w3 = a.w; w4 = b.x; break;
        case 1: w0 = a.y; w1 = a.z; w2 = a.w; w3 = b.x; w4 = b.y; break;
        case 2: w0 = a.z; w1 = a.w; w2 = b.x; w3 = b.y; w4 = b.z; break;
        default: w0 = a.w; w1 = b.x; w2 = b.y; w3 = b.z; w4 = b.w; break;
    }
    uint4 o;
    o.x = __funnelshift_r(w0, w1, sh);
    o.y = __funnelshift_r(w1, w2, sh);
    o.z = __funnelshift_r(w2, w3, sh);
    o.w = __funnelshift_r(w3, w4, sh);
    return o;
}

// ------------------------------------------------------- TMA staging

// Per-group staging area for 1-D bulk copies (cp.async.bulk) from global
// memory into shared memory, tracked by one mbarrier (transaction bytes).
struct Stage {
    uint8_t *buf;
    uint64_t *bar;
    uint32_t bytes;
    uint32_t phase;
};

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// orders this thread's view of global memory (including data acquired from
// other threads) before its later bulk-copy reads
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void tma_load_1d(void *dst_smem, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst_smem)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

constexpr uint32_t kMbarSpinLimit = 1u << 26;

// Wait for the stage's current phase (bounded; sets kErrTimeout on err).
// A false return means the bulk copy may still be writing the stage: the
// caller must issue no further copies into it and end the launch.
__device__ __forceinline__ bool stage_wait(Stage &st, uint32_t *err) {
    uint32_t spins = 0;
    while (!mbar_try_wait(st.bar, st.phase)) {
        if (++spins > kMbarSpinLimit) {
            atomicOr(err, kErrTimeout);
            return false;
        }
    }
    st.phase ^= 1u;
    return true;
}

// Realign-and-store of one staged job: output [d, d + n) from the shared
// copy at s (congruent to the global source mod 16).  The partial head and
// tail words go out as single bytes, one per lane, in one pass (a chain of
// narrow stores from one lane is far slower); the aligned 16-byte body
// words go to consecutive lanes, two per lane per round, each built from
// two aligned shared words and one shift common to the whole job.
template <int G>
__device__ __forceinline__ void store_staged_job(const Group<G> &g, uint8_t *out, uint64_t d,
                                                 const uint8_t *s, uint32_t n) {
    const uint64_t e = d + n;
    uint64_t a0 = (d + 15) & ~(uint64_t)15;  // first aligned body word
    uint64_t a1 = e & ~(uint64_t)15;         // end of the aligned body
    if (a0 > e) a0 = e;
    if (a1 < a0) a1 = a0;
    const uint32_t nh = (uint32_t)(a0 - d), nt = (uint32_t)(e - a1);
    for (uint32_t t = g.lane; t < nh + nt; t += G) {
        const uint32_t o = t < nh ? t : (uint32_t)(a1 - d) + (t - nh);
        out[d + o] = s[o];
    }
    if (a1 <= a0) return;
    // body: source of output word a0 + 16k is shared byte sa + (a0 - d) + 16k
    const uint32_t sb = smem_u32(s) + (uint32_t)(a0 - d);
    const uint32_t r = sb & 15u, base = sb & ~15u, q = r >> 2, sh = (r & 3u) * 8u;
    const uint32_t nw = (uint32_t)((a1 - a0) >> 4);
    uint8_t *ob = out + a0;
    for (uint32_t k = g.lane; k < nw; k += 2 * G) {
        const uint32_t k2 = k + G;
        uint4 x0 = lds16_u32(base + 16 * k), y0 = make_uint4(0, 0, 0, 0);
        uint4 x1 = make_uint4(0, 0, 0, 0), y1 = make_uint4(0, 0, 0, 0);
        if (r) y0 = lds16_u32(base + 16 * k + 16);
        if (k2 < nw) {
            x1 = lds16_u32(base + 16 * k2);
            if (r) y1 = lds16_u32(base + 16 * k2 + 16);
        }
        *reinterpret_cast<uint4 *>(ob + 16 * (uint64_t)k) = r ? window16_uniform(x0, y0, q, sh) : x0;
        if (k2 < nw) *reinterpret_cast<uint4 *>(ob + 16 * (uint64_t)k2) = r ? window16_uniform(x1, y1, q, sh) : x1;
    }
}

// One fill of a group's stage, split in two steps so that a fill can be
// issued ahead (while the group finishes other work) and consumed later.
// Per lane: done = bytes of its job written by earlier fills, off = stage
// offset of its aligned source span in the fill in flight, len = bytes of
// its piece in that fill (0: none), head = offset of the piece's first byte
// within the span.
struct Fill {
    uint32_t done, off, len, head;
};

// Issue one fill for every lane's job (s, n) from f.done on: pieces of at
// most `piece` bytes packed in lane order while they fit, one bulk copy per
// piece.  Returns false, issuing nothing, when no lane has bytes left.  The
// caller has made the sources final and visible to bulk copies.
template <int G>
__device__ __forceinline__ bool fill_issue(const Group<G> &g, Stage &st, const uint8_t *s, uint32_t n,
                                           uint32_t piece, Fill &f) {
    const uint32_t rem = n - f.done;
    f.len = 0;
    if (!g.ballot(rem > 0)) return false;
    const uint32_t len = rem < piece ? rem : piece;
    const uintptr_t ps = reinterpret_cast<uintptr_t>(s) + f.done;
    const uintptr_t sa = ps & ~(uintptr_t)15;
    const uint32_t span = rem ? (uint32_t)(((ps + len + 15) & ~(uintptr_t)15) - sa) : 0u;
    const uint32_t incl = g.scan_incl(span);
    const bool take = rem > 0 && incl <= st.bytes;
    const unsigned tm = g.ballot(take);
    const uint32_t tx = g.shfl(incl, 31 - __clz(tm));
    if (g.lane == 0) mbar_expect_tx(st.bar, tx);
    g.sync();
    f.off = incl - span;
    f.head = (uint32_t)(ps - sa);
    if (take) {
        tma_load_1d(st.buf + f.off, reinterpret_cast<const void *>(sa), span, st.bar);
        f.len = len;
    }
    return true;
}

// Wait for the fill in flight and write its pieces to out[d + done, ...),
// one job after another (store_staged_job).  False, on every lane of the
// group, when a lane's wait timed out (see stage_wait).
template <int G>
__device__ __forceinline__ bool fill_consume(const Group<G> &g, Stage &st, uint8_t *out, uint64_t d, Fill &f,
                                             uint32_t *err) {
    const bool waited = stage_wait(st, err);
    if (g.ballot(!waited)) return false;
    const uint8_t *src = st.buf + f.off + f.head;
    for (unsigned m = g.ballot(f.len > 0); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const uint64_t dj = g.shfl(d + f.done, j);
        const uint8_t *sj = reinterpret_cast<const uint8_t *>(g.shfl(reinterpret_cast<unsigned long long>(src), j));
        const uint32_t nj = g.shfl(f.len, j);
        store_staged_job<G>(g, out, dj, sj, nj);
    }
    g.sync();
    fence_proxy_async_shared();
    f.done += f.len;
    f.len = 0;
    return true;
}

// Staged copy of every lane's job (d, s, n) through fills; `issued` says
// that the first fill of these jobs (f.done = 0) is already in flight.
template <int G>
__device__ __forceinline__ bool staged_copy_fills(const Group<G> &g, Stage &st, uint8_t *out, uint64_t d,
                                                  const uint8_t *s, uint32_t n, uint32_t piece, Fill &f,
                                                  bool issued, uint32_t *err) {
    if (!issued) {
        f.done = 0;
        if (!fill_issue<G>(g, st, s, n, piece, f)) return true;
    }
    for (;;) {
        if (!fill_consume<G>(g, st, out, d, f, err)) return false;
        if (!fill_issue<G>(g, st, s, n, piece, f)) return true;
    }
}

// The full chunks of the group's jobs from shared memory (S: shared address),
// one job after another: for jobs of about G chunks or more, whose chunks
// need no search for their job and share one shift.
template <int G>
__device__ __forceinline__ void copy_full_by_job(const Group<G> &g, uintptr_t P, uint32_t S, uint32_t c,
                                                 unsigned have) {
    for (; have; have &= have - 1) {
        const int j = __ffs(have) - 1;
        uint8_t *pj = reinterpret_cast<uint8_t *>((uintptr_t)g.shfl((unsigned long long)P, j));
        const uint32_t sj = g.shfl(S, j), cj = g.shfl(c, j);
        const uint32_t r = sj & 15u, base = sj & ~15u, q = r >> 2, sh = (r & 3u) * 8u;
        auto word = [&](uint32_t k) {
            const uint4 x = lds16_u32(base + 16 * k);
            return r ? window16_uniform(x, lds16_u32(base + 16 * k + 16), q, sh) : x;
        };
        uint32_t k = g.lane, left = cj;
        for (; left > G; k += 2 * G, left = left > 2 * G ? left - 2 * G : 0) {  // two a lane
            const uint4 v = word(k);
            const bool two = k + G < cj;
            const uint4 v2 = word(two ? k + G : k);
            *reinterpret_cast<uint4 *>(pj + 16 * (uint64_t)k) = v;
            if (two) *reinterpret_cast<uint4 *>(pj + 16 * (uint64_t)(k + G)) = v2;
        }
        if (g.lane < left) *reinterpret_cast<uint4 *>(pj + 16 * (uint64_t)k) = word(k);
    }
}

// Jobs of at least this many full chunks (of 32 lanes; in proportion for
// narrower groups) are copied out one by one: below it more than a third of
// the lanes would idle.  1 GiB copy sweep at L = 384 / 512 / 1000 (23, 31 and
// 61 chunks) by level kernels 802 / 685 / 617 us packed and 790 / 663 / 577 us
// one by one; at L = 256 (15 chunks) 944 and 960 us.
constexpr uint32_t kByJobMin = 20;

// Packed group copy of at most J <= G / 2 jobs, in the lowest lanes (n == 0
// in the others), from shared memory: the next J lanes copy what the first
// ones have after their jobs' last 16-byte boundary, so that heads and tails
// take one step together.
template <int G, int J>
__device__ __forceinline__ void group_copy_few(const Group<G> &g, uintptr_t p, uintptr_t q, uint32_t n) {
    const uint32_t head = n <= 16 ? n : (0u - (uint32_t)p) & 15u;
    const uint32_t rest = n - head, c = rest >> 4;
    const int from = g.lane & (J - 1);
    const uintptr_t pe = (uintptr_t)g.shfl((unsigned long long)(p + n), from);
    const uint32_t qe = g.shfl((uint32_t)q + n, from), tail = g.shfl(rest & 15u, from);
    const bool second = g.lane >= J;
    const uintptr_t ep = second ? pe - tail : p, eq = second ? qe - tail : (uint32_t)q;
    const uint32_t en = !second ? head : g.lane < 2 * J ? tail : 0u;
    // job by job when every job fills most of the lanes by itself
    const unsigned have = g.ballot(c > 0);
    if (have && !g.ballot(c > 0 && c < kByJobMin * G / 32))
        copy_full_by_job<G>(g, p + head, (uint32_t)q + head, c, have);
    else if (have)
        copy_full_chunks<G, 1, kFromShared>(g, p + head, q + head, c, have);
    if (en) store_bytes(ep, load_bytes<kFromShared>(eq, en), en);
}

// Copy of at most J <= G / 2 jobs (in the lowest lanes) through the group's
// stage: every job's aligned source span by one bulk copy, as many jobs at a
// time as the stage holds (a job larger than the stage in pieces), then the
// packed copy from shared memory.  All of a window's source bytes are in
// flight at once and each is fetched once, where the copy through registers
// has U rounds of chunks in flight and reads every word of an unaligned
// source twice.  The sources are final and visible to bulk copies, and the
// stage is free for them.  False when a wait timed out (see stage_wait).
template <int G, int J>
__device__ __forceinline__ bool group_copy_staged(const Group<G> &g, Stage &st, uint8_t *out, uint64_t d,
                                                  const uint8_t *s, uint32_t n, uint32_t *err) {
    uintptr_t p = reinterpret_cast<uintptr_t>(out) + d, q = reinterpret_cast<uintptr_t>(s);
    while (g.ballot(n > 0)) {
        uint32_t m = n < st.bytes - 32 ? n : st.bytes - 32;  // this fill's piece of the job
        const uint32_t lead = (uint32_t)q & 15u, span = m ? (lead + m + 15u) & ~15u : 0u;
        const uint32_t incl = g.scan_incl(span), off = incl - span;
        const bool take = m > 0 && incl <= st.bytes;
        const uint32_t tx = g.shfl(incl, 31 - __clz(g.ballot(take)));
        if (g.lane == 0) mbar_expect_tx(st.bar, tx);
        g.sync();
        if (take)
            tma_load_1d(st.buf + off, reinterpret_cast<const void *>(q - lead), span, st.bar);
        else
            m = 0;
        if (g.ballot(!stage_wait(st, err))) return false;
        group_copy_few<G, J>(g, p, smem_u32(st.buf) + off + lead, m);
        p += m;
        q += m;
        n -= m;
        if (g.ballot(n > 0)) {  // the stage is filled again
            g.sync();
            fence_proxy_async_shared();
        }
    }
    return true;
}

// The same with two stages in turn: the next fill is in flight while the
// current one is copied out (jobs of a kilobyte take several fills a window).
// After a wait that timed out the next fill may be in flight: the caller
// drains both stages before it returns.
template <int G, int J>
__device__ __forceinline__ bool group_copy_piped(const Group<G> &g, Stage (&st)[2], uint8_t *out, uint64_t d,
                                                 const uint8_t *s, uint32_t n, uint32_t *err) {
    uintptr_t p = reinterpret_cast<uintptr_t>(out) + d, q = reinterpret_cast<uintptr_t>(s);
    // a fill of stage t: its piece of this lane's job (at, from, m)
    uintptr_t at = 0, at2 = 0;
    uint32_t from = 0, m = 0, from2 = 0, m2 = 0;
    auto issue = [&](Stage &t, uintptr_t &a, uint32_t &f, uint32_t &k) {
        k = n < t.bytes - 32 ? n : t.bytes - 32;
        const uint32_t lead = (uint32_t)q & 15u, span = k ? (lead + k + 15u) & ~15u : 0u;
        const uint32_t incl = g.scan_incl(span);
        const bool take = k > 0 && incl <= t.bytes;
        const uint32_t tx = g.shfl(incl, 31 - __clz(g.ballot(take)));
        if (g.lane == 0) mbar_expect_tx(t.bar, tx);
        g.sync();
        a = p;
        f = smem_u32(t.buf) + incl - span + lead;
        if (take)
            tma_load_1d(t.buf + (incl - span), reinterpret_cast<const void *>(q - lead), span, t.bar);
        else
            k = 0;
        p += k;
        q += k;
        n -= k;
    };
    if (!g.ballot(n > 0)) return true;
    issue(st[0], at, from, m);
    for (;;) {
#pragma unroll
        for (int b = 0; b < 2; b++) {
            const bool next = g.ballot(n > 0) != 0;
            if (next) issue(st[b ^ 1], at2, from2, m2);
            if (g.ballot(!stage_wait(st[b], err))) return false;
            group_copy_few<G, J>(g, at, from, m);
            g.sync();
            fence_proxy_async_shared();  // the stage may be filled again
            if (!next) {
                if (b == 0) {  // the stages keep their order
                    const Stage t = st[0];
                    st[0] = st[1];
                    st[1] = t;
                }
                return true;
            }
            at = at2;
            from = from2;
            m = m2;
        }
    }
}

}  // namespace aclz

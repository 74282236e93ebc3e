// Range decode (seek): out = decode(x)[lo, hi) without decoding the rest.
//
// Absolute back-references make any output byte resolvable on its own
// (abstract; Sec. I: a region of the stream can be read without decoding
// the whole of it).  A byte inside a match at position p comes from
// src + (p - dst); following that chain always moves strictly backwards and
// ends in a literal.  The range is cut into units, one warp each.  The warp
// walks the unit's tokens 32 at a time, copies the literal pieces straight
// from the literal array and puts the match pieces, remapped to their
// sources, on a stack in shared memory; then every lane chases a piece of
// its own: it finds the token covering the piece's first byte, copies what
// is literal, follows what is a match, and puts back what lies past the
// token.  On a flattened handle a deferred match is followed through its
// pieces, whose bytes are final after wave 0, so a chain has at most the
// in-order levels left.  Only literals are ever read, so requests never wait
// on one another or on a full decode.
//
// A window of tokens with more match bytes than the stack has room for is
// cut to that many output bytes.
//
// The token covering a position is found from the cell table of the upload
// (the token of every 2^k-th position): one load, then a short search among
// the tokens of that cell.
//
// Stack bound: a piece put on the stack covers bytes of the window that no
// other piece covers, so there are never more pieces than the window has
// match bytes.
#include <algorithm>
#include <cstring>
#include <vector>

#include "aclz_device.cuh"
#include "aclz_internal.h"

using namespace aclz;

namespace {

constexpr int kSeekThreads = 128;
constexpr int kSeekWarps = kSeekThreads / 32;
// unit bytes: large ones keep windows whole and amortise the search for their
// first token, small ones spread a short range over more warps
constexpr uint32_t kUnitLog2Max = 13, kUnitLog2Min = 8;
constexpr uint32_t kStackLog2 = 10, kStack = 1u << kStackLog2;
constexpr uint32_t kSample = 256;  // request starts held in shared memory

// One request: output [lo, hi) into out; seg_base = units of the requests
// before it.
struct SeekReq {
    uint64_t lo, hi;
    uint8_t *out;
    uint64_t seg_base;
};

struct SeekIndex {
    const uint4 *tok;
    const uint8_t *lit;
    const uint64_t *blk_tok, *blk_lit;
    const uint32_t *tokdst, *toklit, *cell;
    const uint32_t *slot;  // flattened handle: first piece of a deferred match; else null
    const uint4 *tri;
    uint64_t n_tok, n_cells, n_tri;
    uint32_t log2bs, log2c;
};

// Token covering output position a (a lane's own search).
__device__ __forceinline__ uint32_t token_at(const SeekIndex &ix, uint64_t a) {
    const uint64_t c = a >> ix.log2c, next = (c + 1) << ix.log2c;
    uint32_t lo = __ldg(ix.cell + c), hi = __ldg(ix.cell + c + 1);
    // the next cell starts with a token of the next block, or past the end
    if (!(next & ((1ULL << ix.log2bs) - 1)) || c + 1 == ix.n_cells) hi--;
    const uint32_t rel = (uint32_t)(a & ((1ULL << ix.log2bs) - 1));
    while (lo < hi) {
        const uint32_t mid = lo + ((hi - lo + 1) >> 1);
        if (__ldg(ix.tokdst + mid) <= rel) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Where the bytes from a on of match token t (m0: its first byte, of n
// wanted bytes from a) come from: the source of a, and *n cut to the bytes
// that come from there on.
__device__ __forceinline__ uint64_t source_of(const SeekIndex &ix, uint32_t t, const uint4 tk, uint64_t m0, uint64_t a,
                                              uint32_t *n) {
    if (!ix.slot || !(tk.w >> 8)) return ((uint64_t)tk.z | ((uint64_t)(tk.w & 0xffu) << 32)) + (a - m0);
    // the token's pieces follow one another from its slot on, without gaps:
    // the last one that starts at or before a, by doubling steps, then
    // halving (piece i + k starts k bytes or more after piece i, and the
    // pieces after the token's start past a)
    const uint64_t i = __ldg(ix.slot + t);
    auto dst = [&](uint64_t k) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(ix.tri + i + k));
        return (uint64_t)v.x | ((uint64_t)(v.y & 0xffu) << 32);
    };
    uint4 pc = __ldg(ix.tri + i);
    uint64_t d = (uint64_t)pc.x | ((uint64_t)(pc.y & 0xffu) << 32);
    if (d + (pc.w >> 8) <= a) {
        uint64_t lo = 0, hi = a - d < ix.n_tri - 1 - i ? a - d : ix.n_tri - 1 - i, step = 1;
        while (step <= hi && dst(step) <= a) {
            lo = step;
            step <<= 1;
        }
        if (step <= hi) hi = step - 1;
        while (lo < hi) {
            const uint64_t mid = (lo + hi + 1) >> 1;
            if (dst(mid) <= a) lo = mid; else hi = mid - 1;
        }
        pc = __ldg(ix.tri + i + lo);
        d = (uint64_t)pc.x | ((uint64_t)(pc.y & 0xffu) << 32);
    }
    const uint64_t left = d + (pc.w >> 8) - a;
    if (*n > left) *n = (uint32_t)left;
    return ((uint64_t)pc.z | ((uint64_t)(pc.w & 0xffu) << 32)) + (a - d);
}

// A piece on the stack: source position, bytes (1 .. kStack), offset in the
// unit.
__device__ __forceinline__ unsigned long long pack_piece(uint64_t a, uint32_t n, uint32_t oo) {
    static_assert(40 + kStackLog2 + kUnitLog2Max <= 64, "a piece fits 64 bits");
    return a | ((unsigned long long)(n - 1u) << 40) | ((unsigned long long)oo << (40 + kStackLog2));
}

// Bound by the latency of a hop (cell, token offset, token, piece: dependent
// loads) times the depth of the chain, so the lanes of a warp each follow a
// chain of their own, 32 tokens' pieces at a time.  Against one chain per
// warp, started from 256 output bytes and found by a search of the block's
// tokens, on flattened word text at 12/16/24/32 (the depth of the chains
// differs from text to text, both sides on the same): one 16 KiB range 54 to
// 103 -> 16 to 23 us, 64 ranges of 16 KiB to 4 MiB (50 MB) 1.3 to 3.4 ms ->
// 0.17 to 0.26 ms.  6 CTAs
// per SM (80 registers): 5 and 7 were 2% slower; units up to 8 KiB: with 1
// KiB units and no windows 0.31 ms.
__global__ void __launch_bounds__(kSeekThreads, 6) k_seek(const SeekReq *__restrict__ reqs, SeekReq one,
                                                          uint32_t nreq, uint64_t nseg, uint32_t log2u, SeekIndex ix) {
    __shared__ unsigned long long stack[kSeekWarps][kStack];
    __shared__ uint64_t sample[kSample];
    Group<32> g;
    const int wl = threadIdx.x >> 5;
    unsigned long long *stk = stack[wl];
    // every stride-th request's first unit: the table itself may lie in
    // pinned host memory, where a search would pay its latency each step
    const uint32_t stride = (nreq + kSample - 1) / kSample, ns = (nreq + stride - 1) / stride;
    if (nreq > 1) {
        for (uint32_t i = threadIdx.x; i < ns; i += kSeekThreads) sample[i] = reqs[(uint64_t)i * stride].seg_base;
        __syncthreads();
    }
    const uint64_t nw = (uint64_t)gridDim.x * kSeekWarps;
    for (uint64_t gs = blockIdx.x * (uint64_t)kSeekWarps + wl; gs < nseg; gs += nw) {
        // the request holding unit gs
        SeekReq rq = one;
        if (nreq > 1) {
            uint32_t lo = 0, hi = ns - 1;
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (sample[mid] <= gs) lo = mid; else hi = mid - 1;
            }
            lo *= stride;
            hi = min(lo + stride, nreq) - 1;
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (__ldg(&reqs[mid].seg_base) <= gs) lo = mid; else hi = mid - 1;
            }
            rq = reqs[lo];
        }
        const uint64_t a0 = rq.lo + ((gs - rq.seg_base) << log2u);
        const uint64_t b0 = min(a0 + ((uint64_t)1 << log2u), rq.hi);
        uint8_t *out = rq.out + (a0 - rq.lo);
        uint64_t at = a0, bp = a0 >> ix.log2bs;
        for (uint64_t t = token_at(ix, a0); at < b0;) {
            // the next 32 tokens
            const uint64_t ti = t + (uint64_t)g.lane;
            bool v = ti < ix.n_tok;
            uint64_t bb = bp, ts = ~0ULL, te = 0;
            uint4 tk = make_uint4(0, 0, 0, 0);
            if (v) {
                while (ti >= __ldg(ix.blk_tok + bb + 1)) bb++;
                ts = (bb << ix.log2bs) + __ldg(ix.tokdst + ti);
                tk = __ldg(ix.tok + ti);
                te = ts + tk.x + tk.y;
                v = ts < b0;
            }
            uint64_t wend = min(b0, g.shfl(te, 31 - __clz(g.ballot(v))));
            const uint64_t m0 = ts + tk.x, x = max(m0, at);
            uint64_t y = min(te, wend);
            const uint32_t mb = v && tk.y && y > x ? (uint32_t)(y - x) : 0u;
            if (__reduce_add_sync(0xffffffffu, mb) > kStack) {
                wend = min(wend, at + kStack);
                y = min(te, wend);
            }
            uint32_t ln = 0;
            uint64_t ld = 0;
            const uint8_t *ls = ix.lit;
            if (v && tk.x) {
                const uint64_t lx = max(ts, at), ly = min(m0, wend);
                if (ly > lx) {
                    ln = (uint32_t)(ly - lx);
                    ld = lx - a0;
                    ls = ix.lit + __ldg(ix.blk_lit + bb) + __ldg(ix.toklit + ti) + (lx - ts);
                }
            }
            group_copy<32, 1, kFromConst>(g, out, ld, ls, ln);
            // what a match covers of the window, its first stretch from one
            // source, is the lane's own piece; the rest waits on the stack
            uint64_t a = 0;
            uint32_t n = 0, oo = 0, rest = 0, sp = 0;
            if (v && tk.y && y > x) {
                n = rest = (uint32_t)(y - x);
                oo = (uint32_t)(x - a0);
                a = source_of(ix, (uint32_t)ti, tk, m0, x, &n);
                rest -= n;
            }
            unsigned rm = g.ballot(rest > 0);
            if (rest) stk[__popc(rm & g.lanemask_lt())] = pack_piece(x + n, rest, oo + n);
            sp = __popc(rm);
            __syncwarp();
            // chase the pieces, one per lane, newest first
            for (;;) {
                const unsigned idle = g.ballot(n == 0);
                const uint32_t rank = __popc(idle & g.lanemask_lt()), want = __popc(idle), take = want < sp ? want : sp;
                if (n == 0 && rank < take) {
                    const unsigned long long e = stk[sp - 1 - rank];
                    a = e & ((1ULL << 40) - 1);
                    n = ((uint32_t)(e >> 40) & (kStack - 1)) + 1u;
                    oo = (uint32_t)(e >> (40 + kStackLog2));
                }
                sp -= take;
                __syncwarp();
                if (!g.ballot(n > 0)) break;
                uint32_t cl = 0, co = oo;
                uint64_t from = a;
                const uint8_t *cs = ix.lit;
                rest = n;
                if (n) {
                    const uint32_t pt = token_at(ix, a);
                    const uint64_t pb = a >> ix.log2bs;
                    const uint4 pk = __ldg(ix.tok + pt);
                    const uint64_t ps = (pb << ix.log2bs) + __ldg(ix.tokdst + pt), pm = ps + pk.x;
                    if (a < pm) {
                        cl = pm - a < n ? (uint32_t)(pm - a) : n;
                        cs = ix.lit + __ldg(ix.blk_lit + pb) + __ldg(ix.toklit + pt) + (a - ps);
                        n = 0;
                    } else {
                        const uint64_t pe = pm + pk.y;
                        if (pe - a < n) n = (uint32_t)(pe - a);
                        a = source_of(ix, pt, pk, pm, a, &n);
                    }
                    const uint32_t done = cl ? cl : n;  // bytes this lane copies or keeps
                    rest -= done;
                    from += done;
                }
                rm = g.ballot(rest > 0);
                if (rest) stk[sp + __popc(rm & g.lanemask_lt())] = pack_piece(from, rest, co + (cl ? cl : n));
                sp += __popc(rm);
                if (g.ballot(cl > 0)) group_copy<32, 1, kFromConst>(g, out, co, cs, cl);
                __syncwarp();
            }
            at = wend;
            const uint32_t gone = __popc(g.ballot(v && te <= at));  // tokens the walk is past
            bp = g.shfl(bb, gone < 32 ? (int)gone : 31);
            t += gone;
        }
    }
}

// Units of 2^k bytes for a launch of these many output bytes: the largest
// that give every resident warp a few.
uint32_t unit_log2(uint64_t bytes) {
    uint32_t k = kUnitLog2Max;
    while (k > kUnitLog2Min && (bytes >> k) < 152ull * 24 * 2) k--;
    return k;
}

int seek_launch(aclz_handle *h, const SeekReq *d_reqs, const SeekReq &one, uint32_t nreq, uint64_t nseg,
                uint32_t log2u, cudaStream_t st) {
    if (!nseg) return ACLZ_OK;
    // SM count and resident CTAs, found once (thread-safe static init)
    static const uint64_t slots = [] {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_seek, kSeekThreads, 0);
        return (uint64_t)std::max(sms, 1) * (uint64_t)std::max(per_sm, 1);
    }();
    const uint64_t need = (nseg + kSeekWarps - 1) / kSeekWarps;
    const unsigned grid = (unsigned)std::min<uint64_t>(slots, need);
    SeekIndex ix;
    ix.tok = (const uint4 *)h->d_tok;
    ix.lit = h->d_lit;
    ix.blk_tok = h->d_blk_tok;
    ix.blk_lit = h->d_blk_lit;
    ix.tokdst = h->d_tokdst;
    ix.toklit = h->d_toklit;
    ix.cell = h->d_cell;
    ix.slot = h->flat && h->n_matches_deferred ? h->d_slot : nullptr;
    ix.tri = (const uint4 *)h->d_tri;
    ix.n_tok = h->n_tokens;
    ix.n_tri = h->n_deferred;
    ix.n_cells = h->n_cells;
    ix.log2bs = h->log2_bs;
    ix.log2c = h->log2_cell;
    k_seek<<<grid, kSeekThreads, 0, st>>>(d_reqs, one, nreq, nseg, log2u, ix);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        note_cuda_error(e);
        return ACLZ_E_CUDA;
    }
    return ACLZ_OK;
}

}  // namespace

extern "C" int aclz_decode_range(aclz_handle *h, uint64_t lo, uint64_t hi, void *d_out, void *stream) {
    if (!h) return ACLZ_E_INVAL;
    if (lo > hi || hi > h->total_len) return ACLZ_E_INVAL;
    if (hi == lo) return ACLZ_OK;
    if (!d_out || (reinterpret_cast<uintptr_t>(d_out) & 15)) return ACLZ_E_INVAL;
    if (hi - lo >= (1ULL << 32)) return ACLZ_E_UNSUPPORTED;
    SeekReq one;
    one.lo = lo;
    one.hi = hi;
    one.out = (uint8_t *)d_out;
    one.seg_base = 0;
    const uint32_t lu = unit_log2(hi - lo);
    const uint64_t nseg = (hi - lo + (1ULL << lu) - 1) >> lu;
    return seek_launch(h, nullptr, one, 1, nseg, lu, (cudaStream_t)stream);
}

extern "C" int aclz_ranges_scratch_bytes(uint32_t n_requests, uint64_t *out) {
    if (!out) return ACLZ_E_INVAL;
    *out = (uint64_t)n_requests * sizeof(SeekReq);
    return ACLZ_OK;
}

extern "C" int aclz_decode_ranges(aclz_handle *h, uint32_t n, const uint64_t *host_lo, const uint64_t *host_hi,
                                  void *const *host_out, void *d_scratch, uint64_t scratch_cap, void *stream) {
    if (!h || (n && (!host_lo || !host_hi || !host_out))) return ACLZ_E_INVAL;
    if (n == 0) return ACLZ_OK;
    if ((uint64_t)n * sizeof(SeekReq) > scratch_cap) return ACLZ_E_CAPACITY;
    if (!d_scratch || (reinterpret_cast<uintptr_t>(d_scratch) & 15)) return ACLZ_E_INVAL;
    std::vector<SeekReq> rq;
    rq.reserve(n);
    uint64_t bytes = 0, nseg = 0;
    for (uint32_t i = 0; i < n; i++) bytes += host_hi[i] > host_lo[i] ? host_hi[i] - host_lo[i] : 0;
    const uint32_t lu = unit_log2(bytes);
    for (uint32_t i = 0; i < n; i++) {
        const uint64_t lo = host_lo[i], hi = host_hi[i];
        if (lo > hi || hi > h->total_len) return ACLZ_E_INVAL;
        if (hi - lo >= (1ULL << 32)) return ACLZ_E_UNSUPPORTED;
        if (hi > lo && (!host_out[i] || (reinterpret_cast<uintptr_t>(host_out[i]) & 15))) return ACLZ_E_INVAL;
        SeekReq r;
        r.lo = lo;
        r.hi = hi;
        r.out = (uint8_t *)host_out[i];
        r.seg_base = nseg;
        nseg += (hi - lo + (1ULL << lu) - 1) >> lu;
        rq.push_back(r);
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(d_scratch, rq.data(), sizeof(SeekReq) * n, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return ACLZ_E_CUDA;
    // the host table must outlive the copy
    if (cudaStreamSynchronize(st) != cudaSuccess) return ACLZ_E_CUDA;
    return seek_launch(h, (const SeekReq *)d_scratch, rq[0], n, nseg, lu, st);
}

extern "C" int aclz_decode_ranges_async(aclz_handle *h, uint32_t n, aclz_range_req *reqs, void *stream) {
    static_assert(sizeof(aclz_range_req) == sizeof(SeekReq), "request layout");
    if (!h || (n && !reqs)) return ACLZ_E_INVAL;
    if (n == 0) return ACLZ_OK;
    uint64_t bytes = 0, nseg = 0;
    for (uint32_t i = 0; i < n; i++) bytes += reqs[i].hi > reqs[i].lo ? reqs[i].hi - reqs[i].lo : 0;
    const uint32_t lu = unit_log2(bytes);
    for (uint32_t i = 0; i < n; i++) {
        aclz_range_req &r = reqs[i];
        if (r.lo > r.hi || r.hi > h->total_len) return ACLZ_E_INVAL;
        if (r.hi - r.lo >= (1ULL << 32)) return ACLZ_E_UNSUPPORTED;
        if (r.hi > r.lo && (!r.d_out || (reinterpret_cast<uintptr_t>(r.d_out) & 15))) return ACLZ_E_INVAL;
        r.seg_base = nseg;
        nseg += (r.hi - r.lo + (1ULL << lu) - 1) >> lu;
    }
    const SeekReq *dev = reinterpret_cast<const SeekReq *>(reqs);
    SeekReq first;
    std::memcpy(&first, reqs, sizeof(first));
    return seek_launch(h, dev, first, n, nseg, lu, (cudaStream_t)stream);
}

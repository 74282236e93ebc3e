// Index of wave 0: what a decode can do before any deferred match.
//
//  - Literal units: the literal array cut at multiples of a unit size and at
//    block boundaries, each unit with the token its first byte belongs to,
//    so that literals are copied by as many groups as their bytes ask for,
//    whatever the number of blocks.  Unit ids need no scan: the unit of
//    block b holding the k-th stretch of the literal array is k + b (k never
//    falls and b rises from block to block); ids nothing maps to stay empty.
//  - Matches by level: level 1 reads literals only, level l + 1 matches of
//    level l and below.  The matches of one level are independent of each
//    other, in every block at once.  The list holds the in-order matches
//    (tag 0: every source byte is a literal or an in-order match byte of the
//    same block), for every schedule; where the levels of all matches are
//    known it holds the deferred ones too and is a schedule of its own: the fewest
//    dependent steps there are (a wave hides its chains within a block:
//    4 MiB of FASTQ-like text at 12/16/24/32 has 9 waves with chains adding
//    up to 42 steps, and 14 levels).
#include <algorithm>
#include <cstring>
#include <vector>

#include "aclz_device.cuh"
#include "aclz_internal.h"
#include "aclz_mem.h"

using namespace aclz;

namespace {

int rc_of(cudaError_t e) {
    if (e == cudaSuccess) return ACLZ_OK;
    note_cuda_error((int)e);
    return e == cudaErrorMemoryAllocation ? ACLZ_E_NOMEM : ACLZ_E_CUDA;
}

#define W0CK(x)                  \
    do {                         \
        int _rc = rc_of(x);      \
        if (_rc) return _rc;     \
    } while (0)

__device__ __forceinline__ uint64_t t_dst(const uint4 t) { return (uint64_t)t.x | ((uint64_t)(t.y & 0xffu) << 32); }
__device__ __forceinline__ uint64_t t_src(const uint4 t) { return (uint64_t)t.z | ((uint64_t)(t.w & 0xffu) << 32); }
__device__ __forceinline__ uint32_t t_len(const uint4 t) { return t.w >> 8; }

// units[k + b] = {block b, first token, literal range within the block}, one
// warp per block
__global__ void __launch_bounds__(256) k_lit_units(const uint64_t *__restrict__ blk_tok,
                                                   const uint64_t *__restrict__ blk_lit,
                                                   const uint32_t *__restrict__ toklit, uint32_t nb, uint32_t log2u,
                                                   uint4 *__restrict__ units) {
    const uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nb) return;
    const uint64_t l0 = blk_lit[b], l1 = blk_lit[b + 1];
    if (l1 == l0) return;
    for (uint64_t k = (l0 >> log2u) + lane; k <= (l1 - 1) >> log2u; k += 32) {
        const uint64_t x = max(l0, k << log2u), y = min(l1, (k + 1) << log2u);
        const uint32_t lo = (uint32_t)(x - l0);
        // last token whose literals start at or before lo: they hold lo
        uint64_t a = blk_tok[b], e = blk_tok[b + 1] - 1;
        while (a < e) {
            const uint64_t mid = (a + e + 1) >> 1;
            if (__ldg(toklit + mid) <= lo) a = mid; else e = mid - 1;
        }
        units[k + b] = make_uint4(b, (uint32_t)a, lo, (uint32_t)(y - l0));
    }
}

// A match longer than kLevelPiece goes into the list as several, which groups copy
// side by side (at L = 16000 a level has few matches: the 1 GiB copy sweep takes
// 496 us instead of 826; pieces of 512 bytes cost 10% at L = 1024).

// cnt[b] = triplets of block b for the list (of its in-order matches, or all)
__global__ void __launch_bounds__(256) k_lev_count(const uint4 *__restrict__ tok, const uint64_t *__restrict__ blk_tok,
                                                   uint32_t nb, bool all, uint32_t *cnt) {
    const uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nb) return;
    uint32_t c = 0;
    for (uint64_t i = blk_tok[b] + lane; i < blk_tok[b + 1]; i += 32) {
        const uint4 t = __ldg(tok + i);
        if (all || !(t.w >> 8)) c += (t.y + kLevelPiece - 1) / kLevelPiece;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) cnt[b] = c;
}

// those triplets in token order (base: exclusive scan of the
// counts), which may all be cut anywhere (bit 8 of .y), and with val their
// sort keys 2 (level - 1) + deferred
__global__ void __launch_bounds__(256) k_lev_build(const uint4 *__restrict__ tok, const uint64_t *__restrict__ blk_tok,
                                                   const uint32_t *__restrict__ tokdst, uint32_t nb, uint32_t log2bs,
                                                   const uint32_t *__restrict__ base, bool all,
                                                   const unsigned long long *__restrict__ val, uint4 *__restrict__ tri,
                                                   uint32_t *__restrict__ key, uint32_t *__restrict__ idx) {
    const uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= nb) return;
    uint32_t at = base[b];
    if (base[b + 1] == at) return;
    const uint64_t bstart = (uint64_t)b << log2bs, t1 = blk_tok[b + 1];
    for (uint64_t w = blk_tok[b]; w < t1; w += 32) {
        const uint64_t i = w + lane;
        const uint4 t = i < t1 ? __ldg(tok + i) : make_uint4(0, 0, 0, 0);
        const uint32_t c = all || !(t.w >> 8) ? (t.y + kLevelPiece - 1) / kLevelPiece : 0u;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (c) {
            const uint64_t d = bstart + __ldg(tokdst + i) + t.x;
            const uint64_t src = (uint64_t)t.z | ((uint64_t)(t.w & 0xffu) << 32);
            const uint32_t kk = val ? 2u * ((uint32_t)(__ldg(val + i) >> 32) - 1u) + ((t.w >> 8) ? 1u : 0u) : 0u;
            for (uint32_t q = 0; q < c; q++) {
                const uint32_t k = at + incl - c + q, n = min(t.y - q * kLevelPiece, kLevelPiece);
                const uint64_t pd = d + (uint64_t)q * kLevelPiece, ps = src + (uint64_t)q * kLevelPiece;
                tri[k] = make_uint4((uint32_t)pd, (uint32_t)(pd >> 32) | 0x100u, (uint32_t)ps,
                                    (uint32_t)(ps >> 32) | (n << 8));
                if (val) key[k] = kk;
                idx[k] = k;
            }
        }
        at += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// Levels of the in-order matches, one CTA per block: windows of one match a
// thread in token order, each iterated to its fixed point (a match reads
// earlier ones only, so levels before the window are final and those in it
// only grow).  Ends early once a level is past kOrdLevelsMost: a level takes
// 0.4 us here and its launch 1.7 us in every decode, a step of the walk 0.4 to
// 0.5 us (one block of 16384 levels: upload 10.4 ms and decode 26.5 ms by
// levels, 1.4 and 6.3 ms by the walk; 1024 levels of 64 matches: decode 1.7 ms
// by levels, 4.1 ms by a walk).
constexpr int kLevelThreads = 256;
constexpr uint32_t kOrdLevelsMost = 1024;
__global__ void __launch_bounds__(kLevelThreads) k_ord_levels(const uint4 *__restrict__ tri,
                                                              const uint32_t *__restrict__ base, uint32_t *lvl,
                                                              uint32_t *maxlvl, uint32_t *key) {
    const uint32_t o0 = base[blockIdx.x], o1 = base[blockIdx.x + 1];
    uint32_t mx = 0;
    for (uint32_t w = o0; w < o1; w += kLevelThreads) {
        const uint32_t i = w + threadIdx.x;
        const bool v = i < o1;
        uint64_t s = 0, e = 0;
        uint32_t jl = i, cur = 1;
        if (v) {
            const uint4 t = __ldg(tri + i);
            s = t_src(t);
            e = s + t_len(t);
            // first earlier match that ends past s
            uint32_t lo = o0, hi = i;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                const uint4 y = __ldg(tri + mid);
                if (t_dst(y) + t_len(y) > s) hi = mid; else lo = mid + 1;
            }
            jl = lo;
            __stcg(lvl + i, 1u);
        }
        bool pending = v;
        __syncthreads();
        for (;;) {
            bool changed = false;
            if (pending) {
                uint32_t lv = 1;
                bool inwin = false;
                for (uint32_t j = jl; j < i && t_dst(__ldg(tri + j)) < e; j++) {
                    lv = max(lv, __ldcg(lvl + j) + 1u);
                    inwin = inwin || j >= w;
                }
                changed = lv != cur;
                cur = lv;
                if (changed) __stcg(lvl + i, cur);
                pending = inwin;
            }
            if (!__syncthreads_or(changed)) break;
        }
        if (v) {
            mx = max(mx, cur);
            key[i] = 2u * (cur - 1u);
        }
        const bool past = mx > kOrdLevelsMost || __ldcg(maxlvl) > kOrdLevelsMost;
        if (__syncthreads_or(past)) break;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(maxlvl, mx);
}

// triplets in key order, and the first of each key present
__global__ void k_lev_gather(const uint4 *__restrict__ tri, const uint32_t *__restrict__ key,
                             const uint32_t *__restrict__ idx, uint64_t n, uint4 *__restrict__ out,
                             uint32_t *__restrict__ start) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        out[i] = __ldg(tri + idx[i]);
        if (i == 0 || key[i] != key[i - 1]) start[key[i]] = (uint32_t)i;
    }
}

// The in-order matches of the level list in one order (level after level): a
// level is the last one whose first place is at most i.
__device__ __forceinline__ uint32_t level_of(const uint2 *__restrict__ lev, uint32_t n_lev, uint32_t i) {
    uint32_t lo = 0, hi = n_lev - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (__ldg(&lev[mid].x) <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// key[i] = block of the i-th of them
__global__ void k_ord_keys(const uint4 *__restrict__ list, const uint2 *__restrict__ lev, uint32_t n_lev, uint32_t n,
                           uint32_t log2bs, uint32_t *__restrict__ key, uint32_t *__restrict__ idx) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint2 l = __ldg(lev + level_of(lev, n_lev, i));
        key[i] = (uint32_t)(t_dst(__ldg(list + l.y + (i - l.x))) >> log2bs);
        idx[i] = i;
    }
}

// their triplets in block order, the level from bit 9 of .y on, and every
// block's first place (base: nb + 1 entries)
__global__ void k_ord_gather(const uint4 *__restrict__ list, const uint2 *__restrict__ lev, uint32_t n_lev, uint32_t n,
                             const uint32_t *__restrict__ key, const uint32_t *__restrict__ idx, uint32_t nb,
                             uint4 *__restrict__ out, uint32_t *__restrict__ base) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t at = idx[i], k = level_of(lev, n_lev, at);
        const uint2 l = __ldg(lev + k);
        uint4 t = __ldg(list + l.y + (at - l.x));
        t.y = (t.y & 0x1ffu) | (k << 9);
        out[i] = t;
        for (uint32_t b = i ? key[i - 1] + 1 : 0; b <= key[i]; b++) base[b] = i;
        if (i + 1 == n)
            for (uint32_t b = key[i] + 1; b <= nb; b++) base[b] = n;
    }
}

// In-order levels from which their matches are listed by block: one kernel
// over the blocks then takes their place (k_ord_blocks).  It moves every block
// in and out of shared memory, about what three level kernels take.  Blocks up
// to kOrdBlockMax bytes are held there.
constexpr uint32_t kOrdLevelsMin = 4;
constexpr uint32_t kOrdBlockMax = 1u << 17;

// The list by block.  Without memory for it the levels stay as they are.
int build_ord_blocks(aclz_handle *h, cudaStream_t st) {
    const std::vector<uint64_t> &ls = h->lev_start;
    std::vector<uint2> lev;  // {first place, first triplet} of every level with in-order matches
    uint64_t n = 0;
    for (size_t k = 0; k + 2 < ls.size(); k += 2)
        if (ls[k + 1] > ls[k]) {
            lev.push_back(make_uint2((uint32_t)n, (uint32_t)ls[k]));
            n += ls[k + 1] - ls[k];
        }
    if (lev.size() < kOrdLevelsMin || lev.size() >= 1u << 23 || h->block_size > kOrdBlockMax || n >= 1ULL << 31)
        return ACLZ_OK;
    Scratch dl, key, idx, key2, idx2, out, base;
    const uint32_t nb = h->n_blocks, n_lev = (uint32_t)lev.size();
    for (cudaError_t e : {dl.alloc(8 * lev.size(), st), key.alloc(4 * n, st), idx.alloc(4 * n, st),
                          key2.alloc(4 * n, st), idx2.alloc(4 * n, st), out.alloc(16 * n, st),
                          base.alloc(4 * ((uint64_t)nb + 1), st)})
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? ACLZ_OK : rc_of(e);
        }
    W0CK(cudaMemcpyAsync(dl.p, lev.data(), 8 * lev.size(), cudaMemcpyHostToDevice, st));
    W0CK(cudaStreamSynchronize(st));  // lev is this call's
    uint32_t *k0 = key.as<uint32_t>(), *v0 = idx.as<uint32_t>(), *k1 = key2.as<uint32_t>(), *v1 = idx2.as<uint32_t>();
    const unsigned grid = (unsigned)std::min<uint64_t>(4096, (n + 255) / 256);
    k_ord_keys<<<grid, 256, 0, st>>>((const uint4 *)h->d_lev, dl.as<uint2>(), n_lev, (uint32_t)n, h->log2_bs, k0, v0);
    W0CK(cudaGetLastError());
    const int passes = nb <= 256 ? 1 : nb <= 65536 ? 2 : nb <= (1u << 24) ? 3 : 4;
    if (int rc = device_sort_pairs(&k0, &v0, &k1, &v1, n, passes, st)) return rc;
    k_ord_gather<<<grid, 256, 0, st>>>((const uint4 *)h->d_lev, dl.as<uint2>(), n_lev, (uint32_t)n, k0, v0, nb,
                                       out.as<uint4>(), base.as<uint32_t>());
    W0CK(cudaGetLastError());
    h->d_ord = out.p;
    out.p = nullptr;
    h->d_ord_base = base.as<uint32_t>();
    base.p = nullptr;
    return ACLZ_OK;
}

}  // namespace

void aclz::free_wave0(aclz_handle *h, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    for (void **pp : {&h->d_lunits, &h->d_lev, &h->d_levels, &h->d_ord, (void **)&h->d_ord_base, &h->d_steps,
                      &h->d_lsteps}) {
        dev_free(*pp, st);
        *pp = nullptr;
    }
    h->n_lunits = 0;
    h->lev_start.clear();
    h->by_level = h->walk = false;
    h->steps.clear();
    h->lsteps.clear();
    h->n_levels = 0;
}

int aclz::count_levels(aclz_handle *h, bool all, uint32_t *d_cnt, uint32_t *d_total, void *stream) {
    const uint32_t nb = h->n_blocks;
    k_lev_count<<<(nb + 7) / 8, 256, 0, (cudaStream_t)stream>>>((const uint4 *)h->d_tok, h->d_blk_tok, nb, all, d_cnt);
    W0CK(cudaGetLastError());
    if (int rc = device_excl_scan(d_cnt, nb, d_cnt + nb, stream)) return rc;
    return rc_of(cudaMemcpyAsync(d_total, d_cnt + nb, 4, cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
}

int aclz::build_units(aclz_handle *h, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t nb = h->n_blocks;
    // units of 2 KiB, smaller in a short stream so that there are about 32
    // of them per SM, down to 256 bytes
    uint32_t lu = 11;
    while (lu > 8 && (h->n_literals >> lu) < 152 * 32) lu--;
    h->n_lunits = (h->n_literals >> lu) + nb + 1;
    W0CK(dev_alloc(&h->d_lunits, 16 * h->n_lunits, st));
    W0CK(cudaMemsetAsync(h->d_lunits, 0, 16 * h->n_lunits, st));
    k_lit_units<<<(nb + 7) / 8, 256, 0, st>>>(h->d_blk_tok, h->d_blk_lit, h->d_toklit, nb, lu, (uint4 *)h->d_lunits);
    return rc_of(cudaGetLastError());
}

int aclz::build_levels(aclz_handle *h, const unsigned long long *d_val, uint32_t maxlvl, bool all,
                       const uint32_t *d_cnt, uint32_t n, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t nb = h->n_blocks;
    Scratch work, tri, key, idx, key2, idx2, start;
    if (!n) return ACLZ_OK;
    W0CK(tri.alloc(16 * (uint64_t)n, st));
    W0CK(key.alloc(4 * (uint64_t)n, st));
    W0CK(idx.alloc(4 * (uint64_t)n, st));
    k_lev_build<<<(nb + 7) / 8, 256, 0, st>>>((const uint4 *)h->d_tok, h->d_blk_tok, h->d_tokdst, nb, h->log2_bs,
                                              d_cnt, all, d_val, (uint4 *)tri.p, key.as<uint32_t>(), idx.as<uint32_t>());
    W0CK(cudaGetLastError());
    W0CK(key2.alloc(4 * (uint64_t)n, st));
    if (!d_val) {
        W0CK(work.alloc(16, st));
        W0CK(cudaMemsetAsync(work.p, 0, 16, st));
        k_ord_levels<<<nb, kLevelThreads, 0, st>>>((const uint4 *)tri.p, d_cnt, key2.as<uint32_t>(), work.as<uint32_t>(), key.as<uint32_t>());
        W0CK(cudaGetLastError());
        W0CK(cudaMemcpyAsync(&maxlvl, work.p, 4, cudaMemcpyDeviceToHost, st));
        W0CK(cudaStreamSynchronize(st));
        if (maxlvl > kOrdLevelsMost) {
            h->walk = true;
            return ACLZ_OK;
        }
    }
    const uint64_t keys = 2 * (uint64_t)maxlvl;
    W0CK(idx2.alloc(4 * (uint64_t)n, st));
    W0CK(start.alloc(4 * keys, st));
    W0CK(cudaMemsetAsync(start.p, 0xff, 4 * keys, st));
    W0CK(dev_alloc(&h->d_lev, 16 * (uint64_t)n, st));
    uint32_t *k0 = key.as<uint32_t>(), *v0 = idx.as<uint32_t>(), *k1 = key2.as<uint32_t>(), *v1 = idx2.as<uint32_t>();
    const int passes = keys <= 256 ? 1 : keys <= 65536 ? 2 : keys <= (1u << 24) ? 3 : 4;
    if (int rc = device_sort_pairs(&k0, &v0, &k1, &v1, n, passes, st)) return rc;
    const unsigned grid = (unsigned)std::min<uint64_t>(4096, ((uint64_t)n + 255) / 256);
    k_lev_gather<<<grid, 256, 0, st>>>((const uint4 *)tri.p, k0, v0, n, (uint4 *)h->d_lev, start.as<uint32_t>());
    W0CK(cudaGetLastError());
    std::vector<uint32_t> hs(keys);
    W0CK(cudaMemcpyAsync(hs.data(), start.p, 4 * keys, cudaMemcpyDeviceToHost, st));
    W0CK(cudaStreamSynchronize(st));
    h->by_level = all;
    h->lev_start.assign(keys + 1, n);
    for (uint64_t k = keys; k-- > 0;) h->lev_start[k] = hs[k] == 0xffffffffu ? h->lev_start[k + 1] : hs[k];
    return ACLZ_OK;
}

namespace {

// Whether the staged persistent launch is left to the work ranges: many narrow
// levels, three quarters of all or more.  Its grid barrier makes each of them
// take 2 us (16 MiB of FASTQ-like text with 24 KiB of zeros in it, 380 narrow
// levels of 386: 792 us by levels, 228 us by ranges; 4 MiB of word text with
// the zeros, 240 of 387: 965 and 1404 us).
constexpr uint32_t kNarrowMost = 64;
bool mostly_narrow(const std::vector<Step> &v) {
    const size_t n = std::count_if(v.begin(), v.end(), [](const Step &s) { return s.n <= kRunMost; });
    return n > kNarrowMost && 4 * n >= 3 * v.size();
}

// The first count steps on the device, when they hold a run of narrow levels.
// Without memory for them every level is a launch.
int copy_runs(const std::vector<Step> &v, uint32_t count, void **d, cudaStream_t st) {
    dev_free(*d, st);
    *d = nullptr;
    uint32_t run = 0, most = 0;
    for (uint32_t i = 0; i < count; i++) {
        run = v[i].n <= kRunMost ? run + 1 : 0;
        most = std::max(most, run);
    }
    if (most < kRunMin) return ACLZ_OK;
    if (cudaError_t e = dev_alloc(d, sizeof(Step) * count, st); e != cudaSuccess)
        return e == cudaErrorMemoryAllocation ? ACLZ_OK : rc_of(e);
    return rc_of(cudaMemcpyAsync(*d, v.data(), sizeof(Step) * count, cudaMemcpyHostToDevice, st));
}

}  // namespace

int aclz::build_steps(aclz_handle *h, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    h->steps.clear();
    h->lsteps.clear();
    auto add = [](std::vector<Step> &v, const void *tri, uint64_t a, uint64_t b) {
        if (b > a) v.push_back({(uint64_t)((const uint4 *)tri + a), b - a});
    };
    const std::vector<uint64_t> &ls = h->lev_start;
    dev_free(h->d_ord, st);
    dev_free(h->d_ord_base, st);
    h->d_ord = nullptr;
    h->d_ord_base = nullptr;
    if (!h->by_level && h->d_lev)
        if (int rc = build_ord_blocks(h, st); rc && rc != ACLZ_E_NOMEM) return rc;
    for (size_t k = 0; k + 2 < ls.size(); k += 2) {
        if (!h->d_ord) add(h->steps, h->d_lev, ls[k], ls[k + 1]);
        if (h->by_level) add(h->lsteps, h->d_lev, ls[k], ls[k + 2]);
    }
    h->n_ord_steps = (uint32_t)h->steps.size();
    for (uint32_t w = 1; w < h->n_waves && h->d_tri; w++)
        add(h->steps, h->d_tri, h->wave_start[w], h->wave_start[w + 1]);
    if (int rc = copy_runs(h->steps, h->n_ord_steps, &h->d_steps, st)) return rc;
    if (int rc = copy_runs(h->lsteps, (uint32_t)h->lsteps.size(), &h->d_lsteps, st)) return rc;
    dev_free(h->d_levels, st);
    h->d_levels = nullptr;
    const std::vector<Step> &list = h->by_level ? h->lsteps : h->steps;
    h->n_levels = 0;
    uint32_t n = h->by_level || h->flat ? (uint32_t)list.size() : 0;
    for (const Step &x : list)
        if (x.n >= 1ULL << 31) n = 0;  // the kernel over them counts in 32 bits
    if (mostly_narrow(list)) n = 0;
    if (n) {  // without memory for it the persistent launch goes by ranges
        cudaError_t e = dev_alloc(&h->d_levels, sizeof(Step) * list.size(), st);
        if (e == cudaErrorMemoryAllocation) n = 0;
        else W0CK(e);
    }
    if (n) W0CK(cudaMemcpyAsync(h->d_levels, list.data(), sizeof(Step) * list.size(), cudaMemcpyHostToDevice, st));
    W0CK(cudaStreamSynchronize(st));
    h->n_levels = n;
    return ACLZ_OK;
}

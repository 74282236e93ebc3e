// Tile entropy stage in front of the match phase (Sec. II places an ANS
// stage on 64 KB tiles, many in parallel, ahead of the match kernel).
//
// An ACLE container holds a v1 container's header and block directory raw
// and its 16 token byte planes and literal bytes as order-0 rANS tiles of
// 64 KiB: per tile a frequency table summing to 2^12, 32 interleaved coder
// states (byte i of the tile on state i mod 32) in [2^16, 2^32), and one
// stream of 16-bit renormalisation words, taken in increasing lane order
// within each step of 32 bytes.  One warp decodes one tile: lane k owns
// state k, a table of the 4096 slots and a ring of words sit in shared
// memory, and every step writes 32 consecutive bytes.  The planes are then transposed
// into 16-byte tokens and the upload continues as for a v1 container.
#include <algorithm>
#include <cstring>
#include <vector>

#include "aclz_device.cuh"
#include "aclz_internal.h"
#include "aclz_mem.h"

using namespace aclz;

namespace {

constexpr uint32_t kTile = 65536;
constexpr uint32_t kStreams = 17;
constexpr uint32_t kProbBits = 12, kProb = 1u << kProbBits;
constexpr uint32_t kStateLow = 1u << 16;
constexpr uint32_t kTileHeader = 512 + 4 * 32 + 4;  // freq[256], state[32], n_words
constexpr int kWarps = 1;                             // tiles per CTA (12 of them per SM)
constexpr uint32_t kGroup = 128, kRing = 4 * kGroup;  // words: a group, the ring of them
constexpr uint32_t kWarpSmem = 4 * kProb + 2 * kRing; // slot table, ring

struct TileDesc {
    uint64_t payload;  // offset in the payload area
    uint64_t dst;      // offset in [planes | literals]
    uint32_t m;        // bytes in the tile
    uint32_t n_words;
    uint32_t pad[2];
};

uint32_t rd32le(const uint8_t *p) {
    return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}
uint64_t rd64le(const uint8_t *p) { return (uint64_t)rd32le(p) | ((uint64_t)rd32le(p + 4) << 32); }

// A tile is a chain of up to 2048 steps, each depending on the one before,
// and there are few tiles per SM (1035 of them in 64 MiB of FASTQ-like text),
// so the kernel is bound by the latency of a step: one shared-memory load
// (symbol, frequency and offset of a slot packed in a word), a multiply-add,
// a ballot and a load of the word.  The words come through a ring of four
// groups in shared memory, filled by asynchronous copies three groups (some
// 50 steps) ahead; four steps take at most one group, so the ring is looked
// after once every four steps.  With separate symbol, frequency and offset
// tables and words loaded from global memory one step took 360 ns, 85 ns
// now: the tiles of 64 MiB of FASTQ-like text 740 -> 203 us, of 1 GiB 1.90 ->
// 1.69 ms (12 tiles per SM at a time; 4 tiles per CTA 1.84 ms).  Words in
// registers, shuffled, were no faster than 390 us: a register queue waits
// for its newest load at every move.
__global__ void __launch_bounds__(kWarps * 32) k_ans_tiles(const uint8_t *__restrict__ pay,
                                                          const TileDesc *__restrict__ td, uint64_t n_tiles,
                                                          uint8_t *planes, uint64_t plane_bytes, uint8_t *lits,
                                                          uint32_t *err) {
    extern __shared__ __align__(16) uint8_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t t = (uint64_t)blockIdx.x * kWarps + warp;
    if (t >= n_tiles) return;
    uint32_t *lut = reinterpret_cast<uint32_t *>(sm + warp * kWarpSmem);
    const TileDesc d = td[t];
    const uint8_t *p = pay + d.payload;
    // frequencies: 8 per lane, cumulative by a warp scan
    const uint4 fv = __ldg(reinterpret_cast<const uint4 *>(p) + lane);
    const uint32_t fw[4] = {fv.x, fv.y, fv.z, fv.w};
    uint32_t local = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) local += (fw[k >> 1] >> (16 * (k & 1))) & 0xffffu;
    uint32_t incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total != kProb) {  // checked on the host; never fill the table from a bad one
        if (lane == 0) atomicOr(err, kErrCorrupt);
        return;
    }
    uint32_t x = __ldg(reinterpret_cast<const uint32_t *>(p + 512) + lane);  // little-endian
    // the ring holds the payload from its last aligned 16 bytes before the
    // words on: word i is at place i + kLead of that stream
    constexpr uint32_t kLead = (kTileHeader & 15u) / 2;
    uint8_t *ring = sm + warp * kWarpSmem + 4 * kProb;
    const uint8_t *stream = p + (kTileHeader & ~15u);
    const uint32_t stream_bytes = 2 * (d.n_words + kLead);
    // one group (8 bytes per lane), whole copies that start inside the
    // payload: they end inside the padded buffer
    auto fetch = [&](uint32_t group) {
        const uint32_t at = group * 2 * kGroup + 8 * lane;
        if (at < stream_bytes)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(ring + (at & (2 * kRing - 1)))),
                         "l"(stream + at)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (uint32_t k = 0; k < 4; k++) fetch(k);
    // slot r of symbol s: (r - cum) | s << 12 | (freq - 1) << 20
    uint32_t c = incl - local;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t f = (fw[k >> 1] >> (16 * (k & 1))) & 0xffffu;
        for (int l = 0; l < 32; l++) {
            const uint32_t fl = __shfl_sync(0xffffffffu, f, l), cl = __shfl_sync(0xffffffffu, c, l);
            const uint32_t e = ((uint32_t)(8 * l + k) << 12) | ((fl - 1u) << 20);
            for (uint32_t j = lane; j < fl; j += 32) lut[cl + j] = e | j;
        }
        c += f;
    }
    __syncwarp();
    uint8_t *out = d.dst < plane_bytes ? planes + d.dst : lits + (d.dst - plane_bytes);
    uint32_t pos = kLead, group = 0;  // next word's place, and the group it lies in
    bool bad = x < kStateLow;
    const unsigned below = (1u << lane) - 1u;
    const uint32_t ring_at = smem_u32(ring);
    // one step: the state's symbol, and a word for every lane whose state
    // fell below kStateLow, in lane order (past the end it takes whatever the
    // ring holds; the count at the end then differs)
    auto step = [&](uint8_t *to, bool act) {
        const uint32_t e = lut[x & (kProb - 1)], xh = x >> kProbBits;
        const uint32_t y = (e >> 20) * xh + (xh + (e & (kProb - 1)));
        const bool need = act && y < kStateLow;
        const unsigned bm = __ballot_sync(0xffffffffu, need);
        const uint32_t o = pos + (uint32_t)__popc(bm & below);
        uint16_t w;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(w) : "r"(ring_at + ((2 * o) & (2 * kRing - 1))));
        if (act) *to = (uint8_t)(e >> 12);
        x = act ? (need ? (y << 16) | w : y) : x;
        pos += (uint32_t)__popc(bm);
    };
    // the groups of the next four steps have landed: all but the newest two
    auto look = [&]() {
        if (pos / kGroup != group) {
            __syncwarp();  // every lane is past the group that is overwritten
            fetch(group + 4);
            group++;
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            __syncwarp();
        }
    };
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncwarp();
    uint8_t *to = out + lane;
    const uint32_t whole = d.m >> 5;
    uint32_t i = 0;
    for (; i + 4 <= whole; i += 4, to += 128) {
        step(to, true);
        step(to + 32, true);
        step(to + 64, true);
        step(to + 96, true);
        look();
    }
    for (; i < whole; i++, to += 32) step(to, true);
    if (d.m & 31u) step(to, (uint32_t)lane < (d.m & 31u));
    if (pos != d.n_words + kLead || x != kStateLow) bad = true;  // every state back where encoding began
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(err, kErrCorrupt);
}

// 16 byte planes -> 16-byte tokens (byte k of token t is plane k, entry t).
__global__ void k_planes_to_tokens(const uint8_t *__restrict__ planes, uint64_t nt, uint4 *tok) {
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < nt; t += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < 16; k++) w[k >> 2] |= (uint32_t)__ldg(planes + (uint64_t)k * nt + t) << (8 * (k & 3));
        tok[t] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

struct AcleCtx {
    const uint8_t *pay = nullptr;  // host payload area
    uint64_t pay_bytes = 0;
    std::vector<TileDesc> tiles;
    uint64_t plane_bytes = 0;
    cudaEvent_t ev_begin = nullptr, ev_end = nullptr;  // optional: around the tile decode
};

int fill_from_acle(aclz_handle *h, const View &v, const void *ctx, void *stream) {
    const AcleCtx &a = *static_cast<const AcleCtx *>(ctx);
    cudaStream_t st = (cudaStream_t)stream;
    uint8_t *d_pay = nullptr, *d_planes = nullptr;
    TileDesc *d_td = nullptr;
    uint32_t *d_err = nullptr;
    int rc = ACLZ_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == ACLZ_OK) {
            note_cuda_error(e);
            rc = e == cudaErrorMemoryAllocation ? ACLZ_E_NOMEM : ACLZ_E_CUDA;
        }
        return rc == ACLZ_OK;
    };
    const uint64_t nt = a.tiles.size();
    if (ck(dev_alloc((void **)&d_pay, a.pay_bytes + 16, st)) &&
        ck(dev_alloc((void **)&d_td, sizeof(TileDesc) * (nt ? nt : 1), st)) &&
        ck(dev_alloc((void **)&d_planes, a.plane_bytes ? a.plane_bytes : 16, st)) && ck(dev_alloc((void **)&d_err, 4, st)) &&
        ck(cudaMemsetAsync(d_err, 0, 4, st)) &&
        (!a.pay_bytes || ck(cudaMemcpyAsync(d_pay, a.pay, a.pay_bytes, cudaMemcpyHostToDevice, st))) &&
        (!nt || ck(cudaMemcpyAsync(d_td, a.tiles.data(), sizeof(TileDesc) * nt, cudaMemcpyHostToDevice, st)))) {
        if (a.ev_begin) ck(cudaEventRecord(a.ev_begin, st));
        if (nt && ck(cudaFuncSetAttribute(k_ans_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          kWarps * kWarpSmem))) {
            const unsigned grid = (unsigned)((nt + kWarps - 1) / kWarps);
            k_ans_tiles<<<grid, kWarps * 32, kWarps * kWarpSmem, st>>>(d_pay, d_td, nt, d_planes, a.plane_bytes,
                                                                         h->d_lit, d_err);
            ck(cudaGetLastError());
        }
        if (rc == ACLZ_OK && v.n_tokens) {
            const unsigned grid = (unsigned)std::min<uint64_t>((v.n_tokens + 255) / 256, 65535u);
            k_planes_to_tokens<<<grid, 256, 0, st>>>(d_planes, v.n_tokens, (uint4 *)h->d_tok);
            ck(cudaGetLastError());
        }
        if (a.ev_end) ck(cudaEventRecord(a.ev_end, st));
        uint32_t err = 0;
        if (rc == ACLZ_OK && ck(cudaMemcpyAsync(&err, d_err, 4, cudaMemcpyDeviceToHost, st)) &&
            ck(cudaStreamSynchronize(st)) && err)
            rc = ACLZ_E_CORRUPT;
    }
    cudaStreamSynchronize(st);
    for (void *q : {(void *)d_pay, (void *)d_td, (void *)d_planes, (void *)d_err})
        dev_free(q, st);
    return rc;
}

}  // namespace

extern "C" int aclz_upload_acle_ev(const void *host_buf, uint64_t n, uint32_t flags, void *stream, aclz_handle **out,
                                   void *ev_begin, void *ev_end) {
    if (!host_buf || !out) return ACLZ_E_INVAL;
    *out = nullptr;
    if (flags & ~(uint32_t)ACLZ_UPLOAD_FLATTEN) return ACLZ_E_INVAL;
    const uint8_t *e = static_cast<const uint8_t *>(host_buf);
    if (n < 64 || std::memcmp(e, "ACLE", 4) != 0 || rd32le(e + 4) != 1) return ACLZ_E_CORRUPT;
    const uint64_t size = rd64le(e + 8), prefix = rd64le(e + 16);
    const uint64_t n_tok = rd64le(e + 32), n_lit = rd64le(e + 40), n_tiles = rd64le(e + 48);
    const uint64_t pay_off = rd64le(e + 56);
    if (rd32le(e + 24) != kStreams || rd32le(e + 28) != kTile) return ACLZ_E_CORRUPT;
    if (prefix < 64 || prefix > n - 64 || n_tok > size / 16 || n_lit > size || prefix + 16 * n_tok + n_lit != size)
        return ACLZ_E_CORRUPT;
    // the raw v1 header and directory (tokens and literals come from the
    // tiles): the directory must lie inside the stored prefix before it is
    // walked, since the v1 size above only says what the fields claim
    if (64 + 32 * (uint64_t)rd32le(e + 64 + 20) != prefix) return ACLZ_E_CORRUPT;
    View v;
    int rc = parse_container(e + 64, size, &v, true);
    if (rc) return rc;
    if (64 + 32 * (uint64_t)v.n_blocks != prefix || v.n_tokens != n_tok || v.n_literals != n_lit)
        return ACLZ_E_CORRUPT;
    const uint64_t st_off = 64 + ((prefix + 15) & ~(uint64_t)15);
    const uint64_t tt_off = st_off + 16 * kStreams;
    if (tt_off > n || n_tiles > (n - tt_off) / 16 || tt_off + 16 * n_tiles != pay_off || pay_off > n)
        return ACLZ_E_CORRUPT;
    AcleCtx a;
    a.pay = e + pay_off;
    a.pay_bytes = n - pay_off;
    a.plane_bytes = 16 * n_tok;
    a.tiles.reserve(n_tiles);
    for (uint32_t k = 0; k < kStreams; k++) {
        const uint64_t len = rd64le(e + st_off + 16 * k), first = rd64le(e + st_off + 16 * k + 8);
        const uint64_t cnt = (len + kTile - 1) / kTile;
        if (len != (k < 16 ? n_tok : n_lit) || first != a.tiles.size() || first + cnt > n_tiles)
            return ACLZ_E_CORRUPT;
        for (uint64_t j = 0; j < cnt; j++) {
            const uint8_t *te = e + tt_off + 16 * (first + j);
            const uint64_t po = rd64le(te);
            const uint32_t sz = rd32le(te + 8), m = rd32le(te + 12);
            const uint64_t want = std::min<uint64_t>(kTile, len - j * kTile);
            if (m != want || po % 16 || sz < kTileHeader || po > a.pay_bytes || sz > a.pay_bytes - po)
                return ACLZ_E_CORRUPT;
            const uint8_t *tp = a.pay + po;
            // sum of the 256 little-endian 16-bit frequencies, four at a time
            uint64_t lo = 0, hi = 0;
            for (int q = 0; q < 64; q++) {
                const uint64_t w = rd64le(tp + 8 * q);
                lo += w & 0x0000ffff0000ffffULL;
                hi += (w >> 16) & 0x0000ffff0000ffffULL;
            }
            const uint64_t fsum = (lo & 0xffffffffULL) + (lo >> 32) + (hi & 0xffffffffULL) + (hi >> 32);
            const uint32_t nw = rd32le(tp + 512 + 128);
            if (fsum != kProb || (uint64_t)kTileHeader + 2ull * nw != sz) return ACLZ_E_CORRUPT;
            TileDesc d{};
            d.payload = po;
            d.dst = (k < 16 ? (uint64_t)k * n_tok : 16 * n_tok) + j * kTile;
            d.m = m;
            d.n_words = nw;
            a.tiles.push_back(d);
        }
    }
    if (a.tiles.size() != n_tiles) return ACLZ_E_CORRUPT;
    a.ev_begin = (cudaEvent_t)ev_begin;
    a.ev_end = (cudaEvent_t)ev_end;
    return upload_view(v, flags, stream, fill_from_acle, &a, out);
}

extern "C" int aclz_upload_acle(const void *host_buf, uint64_t n, uint32_t flags, void *stream, aclz_handle **out) {
    return aclz_upload_acle_ev(host_buf, n, flags, stream, out, nullptr, nullptr);
}

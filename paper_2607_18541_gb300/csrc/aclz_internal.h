// Internal declarations shared by the translation units of libaclz.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

#include "../../include/aclz.h"

namespace aclz {

constexpr uint32_t kHdr = 64;
constexpr uint32_t kDirent = 32;
constexpr uint32_t kTok = 16;
constexpr uint64_t kSrcMask = (1ULL << 40) - 1;
constexpr uint32_t kMaxWave = (1u << 24) - 1;
constexpr uint16_t kFlagWaves = 1;
constexpr uint32_t kMinBlock = 64;
constexpr uint32_t kMaxBlock = 1u << 24;

// little-endian field access in host buffers
inline uint16_t rd16(const uint8_t *p) { return (uint16_t)(p[0] | (p[1] << 8)); }
inline uint32_t rd32(const uint8_t *p) {
    return (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
}
inline uint64_t rd64(const uint8_t *p) { return (uint64_t)rd32(p) | ((uint64_t)rd32(p + 4) << 32); }
inline void wr16(uint8_t *p, uint16_t v) { p[0] = (uint8_t)v; p[1] = (uint8_t)(v >> 8); }
inline void wr32(uint8_t *p, uint32_t v) {
    for (int i = 0; i < 4; i++) p[i] = (uint8_t)(v >> (8 * i));
}
inline void wr64(uint8_t *p, uint64_t v) {
    for (int i = 0; i < 8; i++) p[i] = (uint8_t)(v >> (8 * i));
}

inline bool is_pow2(uint64_t v) { return v && !(v & (v - 1)); }
inline uint32_t log2u(uint64_t v) {
    uint32_t k = 0;
    while ((1ULL << k) < v) k++;
    return k;
}

// Parsed header plus pointers into a host container.
struct View {
    uint64_t total_len = 0, n_tokens = 0, n_literals = 0;
    uint32_t block_size = 0, n_blocks = 0, n_waves = 0;
    uint16_t flags = 0;
    uint8_t mm[4] = {0, 0, 0, 0};
    const uint8_t *dir = nullptr, *tok = nullptr, *lit = nullptr;
};

// Header and directory checks on the host (O(n_blocks)); per-token checks
// run on the device during upload.
int parse_container(const uint8_t *c, uint64_t n, View *v, bool check_directory);

// Remember the last CUDA runtime error for aclz_last_cuda_error().
void note_cuda_error(int cuda_error_code);

// Exclusive scan of n u32 in place on the device, the total to *d_total
// (device); stream-ordered, temporary storage allocated on the stream.
int device_excl_scan(uint32_t *d, uint64_t n, uint32_t *d_total, void *stream);

// Stable sort of n (key, value) pairs by the low 8 * passes bits of the key;
// k1 and v1 are scratch of the same size, and on return k0 and v0 point to
// the sorted pairs (the pointers are exchanged when passes is odd).
int device_sort_pairs(uint32_t **k0, uint32_t **v0, uint32_t **k1, uint32_t **v1, uint64_t n, int passes,
                      void *stream);

}  // namespace aclz

struct aclz_handle;

namespace aclz {

// Wave 0's index (aclz_wave0.cu).  build_units: literal units.  count_levels:
// the triplets of the level list of every block (of its in-order matches, or
// with all of every match), scanned into d_cnt (n_blocks + 1 words), their
// total to *d_total.  build_levels: the list from that scan (n triplets).
// d_val: {level, tag} of every token and maxlvl the largest level, or null
// when the levels are not known (the in-order ones are then found block by
// block).  Where there are more than kOrdLevelsMost of those, it leaves the
// in-order matches to the walk, without a list.  build_steps: the step lists,
// once the worklists are final; synchronizes the stream.
// list_counts_fit: the list of nt tokens with total bytes, however they are
// cut, has fewer than 2^32 triplets (its counts and places are 32-bit).
constexpr uint32_t kLevelPiece = 1024;  // a longer match goes into the list as several
constexpr bool list_counts_fit(uint64_t nt, uint64_t total) { return nt + total / kLevelPiece < 0xffffffffULL; }
static_assert(list_counts_fit(1ULL << 31, 1ULL << 40) && !list_counts_fit(3500000000ULL, 1ULL << 40) &&
                  list_counts_fit(0xfffffffeULL, 1023) && !list_counts_fit(0xfffffffeULL, 1024),
              "a terabyte of kilobyte pieces takes 2^30 of the triplets");
int build_units(aclz_handle *h, void *stream);
int count_levels(aclz_handle *h, bool all, uint32_t *d_cnt, uint32_t *d_total, void *stream);
int build_levels(aclz_handle *h, const unsigned long long *d_val, uint32_t maxlvl, bool all, const uint32_t *d_cnt,
                 uint32_t n, void *stream);
int build_steps(aclz_handle *h, void *stream);
void free_wave0(aclz_handle *h, void *stream);

// Deferred matches of at least this mean length are decoded by the persistent
// schedule under ACLZ_MODE_AUTO, shorter ones by levels (or, of a flattened
// handle, as one wave), one kernel each: 1 GiB copy sweep at L = 384 / 512 /
// 768 / 1000 873 / 717 / 639 / 570 us persistent and 794 / 665 / 617 / 580 us
// by level kernels, which meet at a kilobyte; at 64 MiB the level kernels are
// ahead at L = 900 too (115 us, 136 us persistent).
constexpr double kPersistentMin = 1024.0;
// The same where the deferred matches go by waves: no levels (chains too deep
// or too narrow for them), or an event between the phases.  600 blocks of
// 16 KiB, each copied from the one before at L = 256: 3.2 ms by waves, 1.9 ms
// by ranges; 16 MiB copy sweep at L = 512 with the event: 411 us by waves, 108
// us by levels in the persistent launch (it has no in-order matches).
constexpr double kPersistentMinWaves = 192.0;

// A handle's status array: the status word and, on a line of its own, the
// count of the grid barrier.
constexpr uint32_t kBarrierWord = 32, kErrBytes = 256;

// A list of matches that may be copied once everything before it is final:
// device address of its triplets, and their number.
struct Step {
    uint64_t tri, n;
};

// Levels of at most kRunMost matches are narrow; kRunMin or more of them in a
// row go in one launch, by one CTA.
constexpr uint64_t kRunMost = 64;
constexpr uint32_t kRunMin = 8;

// Decode index of h from its device tokens (validation, offsets, wave tags,
// worklists, schedule); see aclz_index.cu.
int build_index(aclz_handle *h, bool has_tags, uint32_t given_waves, bool flat_local, void *stream);

// Upload from a parsed container view: allocates the handle's arrays, has
// fill(h, v, ctx, stream) place the token array in h->d_tok and the literal
// bytes in h->d_lit (stream-ordered), then builds the decode index as
// aclz_upload_ex does.
using FillFn = int (*)(aclz_handle *h, const View &v, const void *ctx, void *stream);
int upload_view(const View &v, uint32_t flags, void *stream, FillFn fill, const void *ctx, aclz_handle **out);

// Ranges per SM a small wave is cut into (about one per resident group).
constexpr uint32_t kRangesPerSm = 16;

// Matches per work range for a target byte size of deferred matches.
inline uint32_t range_matches(uint32_t range_bytes, double mean_len) {
    double t = mean_len > 0 ? (double)range_bytes / mean_len : 16.0;
    if (t < 8) t = 8;
    if (t > 4096) t = 4096;
    return (uint32_t)t;
}

}  // namespace aclz

// Library handle: device copies of a container plus its decode index.
struct aclz_handle {
    int device = 0;
    uint64_t total_len = 0, n_tokens = 0, n_literals = 0, n_deferred = 0;
    uint32_t block_size = 0, log2_bs = 0, n_blocks = 0, n_waves = 0;
    uint16_t flags = 0;
    uint8_t mm[4] = {0, 0, 0, 0};
    // device arrays (owned)
    void *d_tok = nullptr;        // n_tokens x 16 B, tags filled in
    uint8_t *d_lit = nullptr;     // n_literals + 32 zero bytes of padding
    uint64_t *d_blk_tok = nullptr;  // n_blocks + 1 token offsets
    uint64_t *d_blk_lit = nullptr;  // n_blocks + 1 literal offsets
    uint32_t *d_slot = nullptr;   // per token: triplet slot of a deferred match (flattened: of its first piece), else ~0u
    uint32_t *d_tokdst = nullptr; // per token: block-relative offset of its first byte
    uint32_t *d_toklit = nullptr; // per token: block-relative offset of its first literal
    // cell c: the token covering output position c << log2_cell; one entry
    // more holds n_tokens.  Cells are as many as tokens or fewer, and no
    // larger than a block.
    uint32_t *d_cell = nullptr;
    uint64_t n_cells = 0;
    uint32_t log2_cell = 0;
    void *d_tri = nullptr;        // n_deferred x 16 B triplets (dst, src, len), built at upload
    uint32_t *d_err = nullptr;    // latched device status bits; word kBarrierWord: a persistent decode's grid barrier
    std::vector<uint64_t> wave_start;  // n_waves + 1 entries into the triplet array
    // wave 0: literal units {block, first token, literal range}
    void *d_lunits = nullptr;
    uint64_t n_lunits = 0;
    // level list: triplets sorted by level, the in-order matches of a level
    // before its deferred ones (which it holds only when by_level).  Level l
    // (from 1) starts at lev_start[2l - 2], its deferred part at
    // lev_start[2l - 1]; one entry more ends the list.
    void *d_lev = nullptr;
    std::vector<uint64_t> lev_start;
    bool by_level = false;
    // the in-order matches have no list: each block's are walked in token
    // order (most matches read the ones just before them, or the levels are
    // too many, or the list does not fit)
    bool walk = false;
    // the same list's in-order matches by block and level (level from bit 9 of
    // .y on), and each block's first: they take the place of the in-order
    // levels' steps where they are built
    void *d_ord = nullptr;
    uint32_t *d_ord_base = nullptr;
    // what follows the literals, in order: in steps the in-order levels
    // (n_ord_steps of them), then the non-empty waves; in lsteps every
    // level.  d_levels is, on the device, the list whose steps hold
    // independent matches only: lsteps, or the steps of a flattened handle
    // (n_levels 0: there is none).
    std::vector<aclz::Step> steps, lsteps;
    void *d_levels = nullptr;
    uint32_t n_levels = 0;
    uint32_t n_ord_steps = 0;
    // the two lists on the device, where they hold runs of narrow levels
    void *d_steps = nullptr, *d_lsteps = nullptr;
    // persistent-mode schedule.  A segment is the run of one block's
    // matches in one wave's worklist: seg[s] = {block, wave, triplet offset,
    // count}, wave-major then block order.  A range is a run of consecutive
    // triplets of one wave: range[r] = {wave, first segment, end segment,
    // first triplet}, with a sentinel after the last.  Ranges hold up to
    // range_T triplets in large waves and fewer in small ones; they may cut
    // a segment in pieces unless one of its matches reads another's output.
    // seg_pieces[s] counts the ranges that share segment s, and seg_cnt[s]
    // counts the finished ones during a decode (reset by the last).
    void *d_seg = nullptr;
    void *d_ranges = nullptr;
    uint32_t *d_seg_pieces = nullptr;
    uint32_t *d_seg_cnt = nullptr;
    uint64_t n_seg = 0, n_ranges = 0;
    uint32_t range_T = 16;         // matches per range in large waves (from range_bytes / mean length)
    uint32_t range_bytes = 20480;
    double mean_deferred_len = 0;  // mean length of the deferred matches
    // per block, n_wave_words 64-bit words: bit w of pending = block has work
    // in wave w (bit 0 always); done = waves finished (empty waves preset)
    uint32_t n_wave_words = 0;
    uint64_t *d_pending = nullptr;
    uint64_t *d_done = nullptr;
    // set by aclz_flatten: the deferred work items are origin pieces in one
    // wave, built at flatten time
    bool flat = false;
    // set when the (wave, block) tables of the plain schedule would be too
    // large (deep copy chains): the upload then flattens
    bool needs_flatten = false;
    // the stored tags are the 0/1 "in order or not" tags of the flattening
    // upload, not a legal wave tagging of the container
    bool local_tags = false;
    uint64_t n_matches_deferred = 0;  // deferred matches before flattening
};


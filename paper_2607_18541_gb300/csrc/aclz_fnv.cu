// Chunked FNV-1a 64 of a device buffer (verification hash; the paper
// checks every GPU result by FNV, abstract and Sec. II).  Each 64 KiB chunk
// is hashed on its own; the chunk hashes are then hashed in order, 8
// little-endian bytes each, followed by the length.
//
// FNV-1a is a serial chain, h <- (h ^ byte) * P, but only its low byte is
// not linear.  Write h = D + l with l = h mod 256: (h ^ b) * P = P * D +
// (l ^ b) * P, so over a run of n bytes
//     D_out = P^n * D_in + (F(l_in) & ~255),   l_out = F(l_in) & 255,
// where F(l_in) is the plain FNV of the run started from the state l_in.
// Given the low byte at its start, every run is independent of the others
// and the runs combine by multiplications with powers of P.  The low bytes
// come from l <- (l ^ b) * 0xb3 mod 256, in which bit k of the product is
// bit k of the operand xor a function of its lower bits: with the bits
// below k known at every position, bit k is a prefix xor over the
// positions.  Eight such scans, one per bit, give the low byte anywhere.
//
// One CTA hashes one tile of 64 bytes per thread: bytes transposed into
// eight bit planes of two 32-bit words, a prefix xor per plane (in the word,
// across the warp by a ballot, across warps through shared memory), then
// each thread's own 64-byte run and a reduction with powers of P.  Measured
// per call on GB300 against one thread per chunk: 64 KiB 787 -> 40 us,
// 32 MiB 893 -> 62 us, 1 GiB 3.0 -> 0.87 ms (1236 GB/s).
#include <mutex>

#include "aclz_device.cuh"
#include "aclz_internal.h"
#include "aclz_mem.h"

using namespace aclz;

namespace {

constexpr uint64_t kBasis = 14695981039346656037ULL;
constexpr uint64_t kPrime = 1099511628211ULL;
constexpr uint64_t kChunk = 65536;
constexpr int kFnvThreads = 1024;
constexpr uint32_t kRun = 64;                       // bytes per thread
constexpr uint32_t kFnvTile = kFnvThreads * kRun;  // bytes per CTA pass
constexpr int kFnvWarps = kFnvThreads / 32;
static_assert(kFnvTile == kChunk, "a CTA hashes one chunk in one pass");

// P^e mod 2^64
__host__ __device__ constexpr uint64_t fnv_pow(uint64_t e) {
    uint64_t r = 1, b = kPrime;
    for (; e; e >>= 1, b *= b)
        if (e & 1) r *= b;
    return r;
}

__device__ __forceinline__ uint32_t maj(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// inclusive prefix xor of the bits of x, from bit 0 up
__device__ __forceinline__ uint32_t prefix_xor(uint32_t x) {
    x ^= x << 1;
    x ^= x << 2;
    x ^= x << 4;
    x ^= x << 8;
    x ^= x << 16;
    return x;
}

// exchange the bits of a selected by m << s with those of b selected by m
__device__ __forceinline__ void swap_bits(uint32_t &a, uint32_t &b, int s, uint32_t m) {
    const uint32_t t = ((a >> s) ^ b) & m;
    b ^= t;
    a ^= t << s;
}

// Bit planes of 32 bytes: pl[k] bit p = bit k of byte p (w: the bytes,
// little endian).  Word j is first made of the bytes j, j + 8, j + 16 and
// j + 24, so that exchanging the word index with the bit index within a
// byte leaves the positions in order.
__device__ __forceinline__ void bit_planes(const uint32_t *w, uint32_t *pl) {
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const uint32_t a = w[q], b = w[q + 2], c = w[q + 4], d = w[q + 6];
        const uint32_t ab0 = __byte_perm(a, b, 0x5140), ab1 = __byte_perm(a, b, 0x7362);
        const uint32_t cd0 = __byte_perm(c, d, 0x5140), cd1 = __byte_perm(c, d, 0x7362);
        pl[4 * q + 0] = __byte_perm(ab0, cd0, 0x5410);
        pl[4 * q + 1] = __byte_perm(ab0, cd0, 0x7632);
        pl[4 * q + 2] = __byte_perm(ab1, cd1, 0x5410);
        pl[4 * q + 3] = __byte_perm(ab1, cd1, 0x7632);
    }
#pragma unroll
    for (int j = 0; j < 4; j++) swap_bits(pl[j], pl[j + 4], 4, 0x0f0f0f0fu);
#pragma unroll
    for (int j = 0; j < 8; j++)
        if (!(j & 2)) swap_bits(pl[j], pl[j + 2], 2, 0x33333333u);
#pragma unroll
    for (int j = 0; j < 8; j += 2) swap_bits(pl[j], pl[j + 1], 1, 0x55555555u);
}

// FNV state after one tile of kFnvTile bytes (16 words a thread, thread
// order), from the state h; `skip` bytes at the front of the tile are not
// part of the input (0 for a full tile).  Every thread of the CTA calls it;
// the result is valid on thread 0.  sm_bits and sm_d are free for reuse
// after the __syncthreads that the caller puts before its next tile.
template <bool RAGGED>
__device__ uint64_t fnv_tile(const uint32_t (&w)[16], uint64_t h, uint32_t skip, uint32_t (*sm_bits)[32],
                             uint64_t *sm_d) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t A[8], B[8];  // planes: the bytes' bits, then those of low byte ^ byte
    bit_planes(w, A);
    bit_planes(w + 8, B);
    uint32_t ma = ~0u, mb = ~0u, first = 0;  // positions that hold input
    if (RAGGED) {
        const uint32_t at = (uint32_t)tid * kRun;
        first = skip > at ? (skip - at < kRun ? skip - at : kRun) : 0u;
        ma = first >= 32 ? 0u : ~0u << first;
        mb = first <= 32 ? ~0u : (first >= 64 ? 0u : ~0u << (first - 32));
    }
    uint32_t l0 = 0;  // low byte of the state at this thread's first byte
    // carries of x + 2x (a), + 16x (b), + 32x (c); the multiplier is
    // 0xb3 = 1 + 2 + 16 + 32 + 128
    uint32_t aA = 0, aB = 0, bA = 0, bB = 0, cA = 0, cB = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        uint32_t eA = aA ^ bA ^ cA, eB = aB ^ bB ^ cB;
        if (k >= 1) { eA ^= A[k - 1]; eB ^= B[k - 1]; }
        if (k >= 4) { eA ^= A[k - 4]; eB ^= B[k - 4]; }
        if (k >= 5) { eA ^= A[k - 5]; eB ^= B[k - 5]; }
        if (k == 7) { eA ^= A[0]; eB ^= B[0]; }
        const uint32_t yA = prefix_xor((A[k] ^ eA) & ma), yB = prefix_xor((B[k] ^ eB) & mb);
        const uint32_t bal = __ballot_sync(0xffffffffu, (yA ^ yB) >> 31);
        if (lane == 0) sm_bits[k][warp] = __popc(bal) & 1u;
        __syncthreads();
        const uint32_t wb = __ballot_sync(0xffffffffu, lane < kFnvWarps && sm_bits[k][lane]);
        const uint32_t in = (uint32_t)__popc(bal & ((1u << lane) - 1u)) + (uint32_t)__popc(wb & ((1u << warp) - 1u)) +
                            (uint32_t)(h >> k);
        const uint32_t cin = 0u - (in & 1u), cmid = cin ^ (0u - (yA >> 31));
        l0 |= (in & 1u) << k;
        const uint32_t xA = A[k] ^ (yA << 1) ^ cin, xB = B[k] ^ (yB << 1) ^ cmid;
        if (k < 7) {
            // sum bits and carries of bit k; all but the last are used above
            const uint32_t p1A = k >= 1 ? A[k - 1] : 0u, p1B = k >= 1 ? B[k - 1] : 0u;
            const uint32_t p4A = k >= 4 ? A[k - 4] : 0u, p4B = k >= 4 ? B[k - 4] : 0u;
            const uint32_t p5A = k >= 5 ? A[k - 5] : 0u, p5B = k >= 5 ? B[k - 5] : 0u;
            const uint32_t tA = xA ^ p1A ^ aA, tB = xB ^ p1B ^ aB;
            const uint32_t uA = tA ^ p4A ^ bA, uB = tB ^ p4B ^ bB;
            aA = maj(xA, p1A, aA);
            aB = maj(xB, p1B, aB);
            bA = maj(tA, p4A, bA);
            bB = maj(tB, p4B, bB);
            cA = maj(uA, p5A, cA);
            cB = maj(uB, p5B, cB);
        }
        A[k] = xA;
        B[k] = xB;
    }
    // this thread's run from its low byte
    uint64_t f = l0;
#pragma unroll
    for (int j = 0; j < 16; j++) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint64_t nf = (f ^ ((w[j] >> (8 * k)) & 0xffu)) * kPrime;
            f = (!RAGGED || (uint32_t)(4 * j + k) >= first) ? nf : f;
        }
    }
    const uint32_t l_out = (uint32_t)f & 255u;
    // an empty run has no high part of its own (f is then the low byte)
    uint64_t d = f & ~255ULL;
    constexpr uint64_t pw[5] = {fnv_pow(kRun), fnv_pow(2 * kRun), fnv_pow(4 * kRun), fnv_pow(8 * kRun),
                                fnv_pow(16 * kRun)};
#pragma unroll
    for (int s = 0; s < 5; s++) d = d * pw[s] + __shfl_down_sync(0xffffffffu, d, 1 << s);
    if (lane == 0) sm_d[warp] = d;
    if (tid == kFnvThreads - 1) sm_d[kFnvWarps] = l_out;
    __syncthreads();
    uint64_t r = 0;
    if (warp == 0) {
        constexpr uint64_t pv[5] = {fnv_pow(32 * kRun), fnv_pow(64 * kRun), fnv_pow(128 * kRun), fnv_pow(256 * kRun),
                                    fnv_pow(512 * kRun)};
        d = lane < kFnvWarps ? sm_d[lane] : 0ULL;
#pragma unroll
        for (int s = 0; s < 5; s++)
            if ((1 << s) < kFnvWarps) d = d * pv[s] + __shfl_down_sync(0xffffffffu, d, 1 << s);
        constexpr uint64_t full = fnv_pow(kFnvTile);
        const uint64_t pn = RAGGED ? fnv_pow(kFnvTile - skip) : full;
        r = pn * (h & ~255ULL) + d + sm_d[kFnvWarps];
    }
    return r;
}

// hashes[c] = FNV-1a of chunk c, one CTA per chunk.  Integer issue bounds
// it: about 15 instructions a byte (transpose and planes 8, the runs 6).
__global__ void __launch_bounds__(kFnvThreads) k_fnv_chunks(const uint8_t *__restrict__ buf, uint64_t n,
                                                            uint64_t *__restrict__ hashes) {
    __shared__ uint32_t sm_bits[8][32];
    __shared__ uint64_t sm_d[kFnvWarps + 1];
    const uint64_t lo = (uint64_t)blockIdx.x * kChunk;
    const uint32_t len = (uint32_t)(n - lo < kChunk ? n - lo : kChunk);
    uint32_t w[16];
    uint64_t h;
    if (len == kChunk) {
        // buf is 16-byte aligned and lo is a multiple of 64 KiB
        const uint4 *q = reinterpret_cast<const uint4 *>(buf + lo) + 4 * threadIdx.x;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint4 v = __ldg(q + k);
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
        h = fnv_tile<false>(w, kBasis, 0, sm_bits, sm_d);
    } else {
        // the last, short chunk ends at the tile's end
        const uint32_t skip = kFnvTile - len;
#pragma unroll
        for (int j = 0; j < 16; j++) {
            w[j] = 0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t at = threadIdx.x * kRun + 4 * j + k;
                if (at >= skip) w[j] |= (uint32_t)__ldg(buf + lo + (at - skip)) << (8 * k);
            }
        }
        h = fnv_tile<true>(w, kBasis, skip, sm_bits, sm_d);
    }
    if (threadIdx.x == 0) hashes[blockIdx.x] = h;
}

// *out = FNV-1a of the chunk hashes followed by n, 8 bytes each, by one
// CTA, tile after tile; the first tile is the short one.
__global__ void __launch_bounds__(kFnvThreads) k_fnv_combine(const uint64_t *__restrict__ hashes, uint64_t nchunks,
                                                             uint64_t n, uint64_t *out) {
    __shared__ uint32_t sm_bits[8][32];
    __shared__ uint64_t sm_d[kFnvWarps + 1];
    __shared__ uint64_t sm_h;
    constexpr uint32_t kWords = kFnvTile / 8;
    const uint64_t words = nchunks + 1;
    const uint64_t tiles = (words + kWords - 1) / kWords;
    const uint64_t pad = tiles * kWords - words;  // words before the input
    uint64_t h = kBasis;
    for (uint64_t t = 0; t < tiles; t++) {
        uint32_t w[16];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const uint64_t at = t * kWords + threadIdx.x * 8 + j;
            uint64_t v = 0;
            if (at >= pad) v = at - pad < nchunks ? hashes[at - pad] : n;
            w[2 * j] = (uint32_t)v;
            w[2 * j + 1] = (uint32_t)(v >> 32);
        }
        h = fnv_tile<true>(w, h, t ? 0u : (uint32_t)pad * 8u, sm_bits, sm_d);
        if (threadIdx.x == 0) sm_h = h;
        __syncthreads();
        h = sm_h;
    }
    if (threadIdx.x == 0) *out = h;
}

}  // namespace

namespace aclz {

// Enqueue the two FNV kernels with caller-provided scratch of
// 8 * (nchunks + 1) bytes; the result lands in scratch[nchunks].
int fnv_enqueue(const uint8_t *d_buf, uint64_t n, uint64_t *scratch, cudaStream_t st) {
    const uint64_t nchunks = (n + kChunk - 1) / kChunk;
    if (nchunks) {
        k_fnv_chunks<<<(unsigned)nchunks, kFnvThreads, 0, st>>>(d_buf, n, scratch);
    }
    k_fnv_combine<<<1, kFnvThreads, 0, st>>>(scratch, nchunks, n, scratch + nchunks);
    return cudaGetLastError() == cudaSuccess ? ACLZ_OK : ACLZ_E_CUDA;
}

}  // namespace aclz

extern "C" int aclz_fnv(const void *d_buf, uint64_t n, uint64_t *out_hash, void *stream) {
    if (!out_hash || (n && !d_buf)) return ACLZ_E_INVAL;
    if (reinterpret_cast<uintptr_t>(d_buf) & 15) return ACLZ_E_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const uint64_t nchunks = (n + kChunk - 1) / kChunk;
    uint64_t *scratch = nullptr;
    cudaError_t e = dev_alloc((void **)&scratch, 8 * (nchunks + 1), st);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? ACLZ_E_NOMEM : ACLZ_E_CUDA;
    int rc = fnv_enqueue((const uint8_t *)d_buf, n, scratch, st);
    uint64_t hv = 0;
    if (rc == ACLZ_OK &&
        cudaMemcpyAsync(&hv, scratch + nchunks, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        rc = ACLZ_E_CUDA;
    dev_free(scratch, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) rc = ACLZ_E_CUDA;
    if (rc == ACLZ_OK) *out_hash = hv;
    return rc;
}

// ---------------------------------------------------------------------
// Allocation-free variant of aclz_fnv.
//
// Some callers cannot allocate device memory at the moment they want a
// verification hash: code that runs while the device is nearly full and a
// failed allocation would abort a long pipeline, code whose device memory
// is owned by an arena or pool manager that forbids out-of-band
// allocations, and latency-critical paths that must not enter the CUDA
// allocator (which may synchronize or block).  For them the chunk hashes
// live in one fixed array in the library's device memory instead of
// stream-ordered scratch.
//
// kNoAllocChunks bounds the input: 65536 chunks of 64 KiB, i.e. 4 GiB.  The
// array (512 KiB + 8 bytes) is held on every device that loads the library
// until the process exits.  All calls share it and it keeps the previous
// call's contents; nothing in it needs to start at zero, because every
// call rewrites every entry it reads.  Calls whose work overlaps on the GPU
// (different streams, or different host threads, without ordering between
// them) race on the array and can return wrong hashes.
constexpr uint64_t kNoAllocChunks = 65536;
static __device__ __align__(256) uint64_t g_fnv_noalloc_scratch[kNoAllocChunks + 1];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
uint64_t *g_noalloc_ptr[kMaxDevices] = {};

// Device address of the fixed array on the current device, looked up once
// per device (the host-side symbol is only a stand-in, never a device
// address).
int noalloc_scratch(uint64_t **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ACLZ_E_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return ACLZ_E_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_fnv_noalloc_scratch);
        if (e != cudaSuccess || !p) return ACLZ_E_CUDA;
        g_noalloc_ptr[dev] = (uint64_t *)p;
    }
    *out = g_noalloc_ptr[dev];
    return ACLZ_OK;
}

}  // namespace

extern "C" int aclz_fnv_noalloc(const void *d_buf, uint64_t n, uint64_t *out_hash, void *stream) {
    if (!out_hash || (n && !d_buf)) return ACLZ_E_INVAL;
    if (reinterpret_cast<uintptr_t>(d_buf) & 15) return ACLZ_E_INVAL;
    const uint64_t nchunks = (n + kChunk - 1) / kChunk;
    if (nchunks > kNoAllocChunks) return ACLZ_E_CAPACITY;
    uint64_t *scratch = nullptr;
    int rc = noalloc_scratch(&scratch);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    rc = fnv_enqueue((const uint8_t *)d_buf, n, scratch, st);
    uint64_t hv = 0;
    if (rc == ACLZ_OK &&
        cudaMemcpyAsync(&hv, scratch + nchunks, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        rc = ACLZ_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) rc = ACLZ_E_CUDA;
    if (rc == ACLZ_OK) *out_hash = hv;
    return rc;
}

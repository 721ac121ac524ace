// pk_derive.cu -- key derivation kernels (sm_103a).
//
//   descriptor digests  d_j = SHA-256(enc_j)                       (Eq. 3, H over enc)
//   chunk offsets       key_off = exclusive scan of floor(T_r / C)  (full chunks only, Sec. 4.4)
//   chunk digests       c_i = SHA-256(LE int32 tokens of chunk i)  (the content part of f(x, .))
//   chain               k_i = SHA-256(k_{i-1} || d || c_i)         (the digest folded into every key)
//
// SHA-256 is plain 32-bit integer work: funnel-shift rotates, 3-input logic
// and 3-input adds, no tensor cores.  The chunk digests are fully parallel
// (one thread per chunk with the message words in registers, or, when there
// are few, two lanes of a pair of warps); the chain is serial per request (one
// or two lanes of a pair of warps).  The chunk digests are staged in the
// output key buffer and overwritten in place by the chain, so derivation needs
// no scratch memory.
#include <cuda_runtime.h>

#include <mutex>

#include "pk_device.cuh"
#include "pk_internal.h"
#include "pk_pair.cuh"
#include "pk_sha256.cuh"

namespace {

using pk::set_status;

// A digest to a 16-byte aligned 32-byte slot.
__device__ __forceinline__ void store_digest(uint8_t *dst, const uint32_t st[8]) {
    uint4 *q = reinterpret_cast<uint4 *>(dst);
    q[0] = make_uint4(pk::bswap32(st[0]), pk::bswap32(st[1]), pk::bswap32(st[2]), pk::bswap32(st[3]));
    q[1] = make_uint4(pk::bswap32(st[4]), pk::bswap32(st[5]), pk::bswap32(st[6]), pk::bswap32(st[7]));
}

// ---------------------------------------------------------------------------
// Descriptor digests: one warp per descriptor.  The warp copies the encoding
// into shared memory with coalesced byte loads (32 bytes per round trip), then
// one lane hashes it.  Encodings longer than the staging area are hashed from
// global memory.  Two forms:
//   hash_descriptor        pads the encoding in shared memory and hashes its
//                          words with the 16-round code: where the descriptors
//                          set the time, in small batches (key derivation of
//                          512 chunks of 16 tokens under 16 descriptors of about
//                          200 bytes 26.1 -> 24.8 us);
//   hash_descriptor_bytes  takes it byte by byte, in straight-line rounds: in the
//                          launch of a large batch, whose chunk digests hide it
//                          and compile to slower code beside a third copy of the
//                          16-round code (small-block key derivation 613.8 against
//                          616.1 us).
// ---------------------------------------------------------------------------
constexpr int kDescWarps = 4;
constexpr int kDescStage = 2048;

// The calling warp hashes descriptor j (all 32 lanes call).
__device__ __forceinline__ void hash_descriptor_bytes(uint8_t *stage, const uint8_t *enc, uint64_t enc_bytes,
                                                      const int64_t *enc_off, uint32_t j,
                                                      uint8_t *digests, int32_t *status) {
    const uint32_t lane = threadIdx.x & 31;
    const int64_t a = __ldcg(enc_off + j), b = __ldcg(enc_off + j + 1);
    if (a < 0 || b < a || (uint64_t)b > enc_bytes) {
        if (lane == 0) set_status(status, PK_ERR_ARG);
        return;
    }
    const int64_t len = b - a;
    const bool staged = len <= kDescStage;
    if (staged) {
#pragma unroll 4
        for (int64_t i = lane; i < len; i += 32) stage[i] = __ldcg(enc + a + i);
    }
    __syncwarp();
    if (lane == 0) pk::sha256_bytes(staged ? stage : enc + a, (uint64_t)len, digests + 32ull * j);
}

// stage: kDescStage bytes, 16-byte aligned; sK: the round constants; kAligned: digests is 16-byte aligned (else it
// may lie anywhere).
template <bool kAligned>
__device__ __forceinline__ void hash_descriptor(uint8_t *stage, const uint32_t *sK, const uint8_t *enc, uint64_t enc_bytes,
                                                const int64_t *enc_off, uint32_t j,
                                                uint8_t *digests, int32_t *status) {
    const uint32_t lane = threadIdx.x & 31;
    const int64_t a = __ldcg(enc_off + j), b = __ldcg(enc_off + j + 1);
    if (a < 0 || b < a || (uint64_t)b > enc_bytes) {
        if (lane == 0) set_status(status, PK_ERR_ARG);
        return;
    }
    const int64_t len = b - a, blocks = (len + 8) / 64 + 1;
    if (64 * blocks > kDescStage) {
        if (lane == 0) pk::sha256_bytes(enc + a, (uint64_t)len, digests + 32ull * j);
        return;
    }
    uint32_t *words = reinterpret_cast<uint32_t *>(stage);
    for (int64_t i = (len >> 2) + lane; i < 16 * blocks; i += 32) words[i] = 0u;
    __syncwarp();
#pragma unroll 4
    for (int64_t i = lane; i < len; i += 32) stage[i] = __ldcg(enc + a + i);
    if (lane == 0) {
        stage[len] = 0x80u;
        words[16 * blocks - 1] = pk::bswap32((uint32_t)len * 8u);  // (len < 2^11)
    }
    __syncwarp();
    if (lane == 0) {
        uint32_t st[8], w[16];
        pk::init_state(st);
#pragma unroll 1
        for (int64_t blk = 0; blk < blocks; ++blk) {
#pragma unroll
            for (int t = 0; t < 16; ++t) w[t] = pk::bswap32(words[16 * blk + t]);
            pk::compress_rolled(st, w, sK);
        }
        uint8_t *d = digests + 32ull * j;
        if (kAligned || (reinterpret_cast<uintptr_t>(d) & 15) == 0) {
            store_digest(d, st);
        } else {
#pragma unroll
            for (int t = 0; t < 32; ++t) d[t] = (uint8_t)(st[t / 4] >> (24 - 8 * (t % 4)));
        }
    }
}

__global__ void __launch_bounds__(32 * kDescWarps)
k_digest_descriptors(const uint8_t *enc, uint64_t enc_bytes, const int64_t *enc_off,
                     uint32_t D, uint8_t *digests, int32_t *status) {
    __shared__ __align__(16) uint8_t stage[kDescWarps][kDescStage];
    __shared__ uint32_t sK[64];
    for (int i = threadIdx.x; i < 64; i += blockDim.x) sK[i] = pk::kSha256K[i];
    __syncthreads();
    pk::pdl_launch_dependents();
    pk::pdl_wait(enc, enc_off, digests, status);
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t j = blockIdx.x * kDescWarps + warp;
    if (j < D) hash_descriptor<false>(stage[warp], sK, enc, enc_bytes, enc_off, j, digests, status);
}

// ---------------------------------------------------------------------------
// Chunk offsets: one block per tile of kScanThreads * kScanItems requests.
// Each block scans its own tile (kScanItems consecutive requests per thread)
// and sums the requests of every other tile with independent, coalesced loads:
// those before it give its first offset, all of them the checks.  No block waits
// for another and none scans the tiles one after the other (key derivation of
// 16,384 prompts of 32 tokens 37.6 -> 29.1 us, of 100,000 171 -> 100 us), but
// every block reads every request, so the loads grow with the square of R: above
// kScanTiles tiles one block walks the tiles instead (k_chunk_offsets_walk).
// This launch alone, every block reading all | one block, in us, R = 2^17:
// 43.9 | 138, 2^20: 627 | 1093, 1.48 M: 1319 | 1544, 2^21: 2473 | 2178,
// 2^23: 38332 | 9082.  Any invalid request (offsets decreasing, negative or
// past n_tokens, descriptor index >= D) or a total above key_capacity makes all
// offsets zero and reports PK_ERR_ARG.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr uint32_t kScanTile = kScanThreads * kScanItems;
constexpr uint32_t kScanTiles = 360;  // (1.47 M requests)

// Full chunks of the request [a, b) with descriptor index di; bad is set if it is invalid.
__device__ __forceinline__ long long request_chunks(int64_t a, int64_t b, uint32_t di, uint64_t n_tokens, uint32_t C,
                                                    uint32_t D, bool &bad) {
    if (a < 0 || b < a || (uint64_t)b > n_tokens || di >= D) {
        bad = true;
        return 0;
    }
    const uint64_t len = (uint64_t)(b - a);  // 32-bit division when the request fits (64-bit is a long library sequence)
    return len >> 32 ? (long long)(len / C) : (long long)((uint32_t)len / C);
}

// The requests r0 .. r0 + kScanItems - 1 of a thread: their offsets and descriptor indices.
__device__ __forceinline__ void load_requests(const int64_t *tok_off, const uint32_t *desc_idx, uint32_t R, uint64_t r0,
                                              int64_t to[kScanItems + 1], uint32_t di[kScanItems]) {
#pragma unroll
    for (int j = 0; j <= kScanItems; ++j) to[j] = r0 + j <= R ? tok_off[r0 + j] : 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) di[j] = r0 + j < R ? desc_idx[r0 + j] : 0u;
}

__device__ __forceinline__ long long warp_sum(long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Inclusive sum over the lanes.
__device__ __forceinline__ long long warp_scan(long long x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) >= o) x += v;
    }
    return x;
}

template <bool kTiles>  // false: one tile
__global__ void __launch_bounds__(kScanThreads)
k_chunk_offsets(const int64_t *tok_off, uint32_t R, uint64_t n_tokens, uint32_t C,
                const uint32_t *desc_idx, uint32_t D, uint64_t key_capacity,
                int64_t *key_off, int32_t *status) {
    __shared__ long long warp_sums[kScanThreads / 32], warp_before[kScanThreads / 32], warp_after[kScanThreads / 32];
    __shared__ long long sh_total;
    pk::pdl_wait(tok_off, desc_idx, key_off, status);
    // The chunk digests are released only here, when every earlier kernel of the stream is done: released at the
    // start, their CTAs came up beside the previous batch's last kernels and stacked on the SMs those left free,
    // two and more on one SM with others empty, where a small batch needs a lone warp per sub-partition.  Batches
    // enqueued back to back, per step: 900 ragged prompts 435 -> 188 us, multi-adapter 94.5 -> 71.9 us, long
    // context 1056 -> 947 us (both sides with the two-lane chain).
    pk::pdl_launch_dependents();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile, r0 = base + (uint64_t)tid * kScanItems;
    bool bad = false;
    int64_t to[kScanItems + 1];
    uint32_t di[kScanItems];
    load_requests(tok_off, desc_idx, R, r0, to, di);
    long long before = 0, after = 0;  // chunks of the tiles before and after this one
    for (uint64_t other = 0; kTiles && other < R; other += kScanTile) {
        if (other == base) continue;
        int64_t a[kScanItems], b[kScanItems];
        uint32_t d[kScanItems];
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            const uint64_t r = other + j * kScanThreads + tid;
            a[j] = r < R ? tok_off[r] : 0;
            b[j] = r < R ? tok_off[r + 1] : 0;
            d[j] = r < R ? desc_idx[r] : 0u;
        }
        long long sum = 0;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j)
            if (other + j * kScanThreads + tid < R) sum += request_chunks(a[j], b[j], d[j], n_tokens, C, D, bad);
        if (other < base) before += sum;
        else after += sum;
    }
    long long n[kScanItems];
    long long local = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        n[j] = r0 + j < R ? request_chunks(to[j], to[j + 1], di[j], n_tokens, C, D, bad) : 0;
        local += n[j];
    }
    // block exclusive scan of the per-thread sums, and the other tiles' totals
    const long long incl = warp_scan(local);
    if (lane == 31) warp_sums[warp] = incl;
    if (kTiles) {
        before = warp_sum(before);
        after = warp_sum(after);
        if (lane == 0) {
            warp_before[warp] = before;
            warp_after[warp] = after;
        }
    }
    bad = __syncthreads_or(bad);
    if (warp == 0) {
        const long long ws = warp_sums[lane], wincl = warp_scan(ws);
        const long long first = kTiles ? warp_sum(warp_before[lane]) : 0;
        const long long rest = kTiles ? warp_sum(warp_after[lane]) : 0;
        warp_sums[lane] = first + wincl - ws;
        if (lane == 31) sh_total = first + wincl + rest;
    }
    __syncthreads();
    bad |= (unsigned long long)sh_total > key_capacity;
    long long run = warp_sums[warp] + incl - local;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        run += n[j];
        if (r0 + j < R) key_off[r0 + j + 1] = bad ? 0 : run;
    }
    if (blockIdx.x == 0 && tid == 0) {
        key_off[0] = 0;
        if (bad) set_status(status, PK_ERR_ARG);
    }
}

// One block, tile after tile, a running carry linking them and each tile's loads in flight during the scan before it.
__global__ void __launch_bounds__(kScanThreads)
k_chunk_offsets_walk(const int64_t *tok_off, uint32_t R, uint64_t n_tokens, uint32_t C,
                     const uint32_t *desc_idx, uint32_t D, uint64_t key_capacity,
                     int64_t *key_off, int32_t *status) {
    __shared__ long long warp_sums[kScanThreads / 32];
    __shared__ long long tile_total;
    pk::pdl_wait(tok_off, desc_idx, key_off, status);
    pk::pdl_launch_dependents();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) key_off[0] = 0;
    bool bad = false;
    long long carry = 0;
    int64_t to[kScanItems + 1], to_next[kScanItems + 1] = {};
    uint32_t di[kScanItems], di_next[kScanItems] = {};
    load_requests(tok_off, desc_idx, R, (uint64_t)tid * kScanItems, to, di);
    for (uint64_t base = 0; base < R; base += kScanTile) {
        const uint64_t r0 = base + (uint64_t)tid * kScanItems;
        if (base + kScanTile < R) load_requests(tok_off, desc_idx, R, r0 + kScanTile, to_next, di_next);
        long long n[kScanItems];
        long long local = 0;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            n[j] = r0 + j < R ? request_chunks(to[j], to[j + 1], di[j], n_tokens, C, D, bad) : 0;
            local += n[j];
        }
        const long long incl = warp_scan(local);
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const long long ws = warp_sums[lane], wincl = warp_scan(ws);
            warp_sums[lane] = wincl - ws;
            if (lane == 31) tile_total = wincl;
        }
        __syncthreads();
        long long run = carry + warp_sums[warp] + incl - local;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            run += n[j];
            if (r0 + j < R) key_off[r0 + j + 1] = run;
        }
        carry += tile_total;
        __syncthreads();  // warp_sums and tile_total are written again by the next tile
#pragma unroll
        for (int j = 0; j <= kScanItems; ++j) to[j] = to_next[j];
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) di[j] = di_next[j];
    }
    bad = __syncthreads_or(bad);
    if (bad || (unsigned long long)carry > key_capacity) {
        for (uint64_t r = tid; r < R; r += kScanThreads) key_off[r + 1] = 0;
        if (tid == 0) set_status(status, PK_ERR_ARG);
    }
}

// 16 message words of one 64-byte block of int32 tokens (little-endian bytes,
// read by SHA-256 as big-endian words), straight from global memory.
__device__ __forceinline__ void load_block_global(const int32_t *src, uint32_t w[16]) {
#pragma unroll
    for (int t = 0; t < 16; ++t) w[t] = pk::bswap32((uint32_t)__ldcg(src + t));
}

// Asynchronous 64-byte copy global -> shared (4 x 16 B; both 16-byte aligned).
__device__ __forceinline__ void cp_async_block(uint32_t *smem_dst, const int32_t *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
#pragma unroll
    for (int v = 0; v < 4; ++v)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * v), "l"(src + 4 * v) : "memory");
}
// The first `bytes` (1 to 16) of a 16-byte unit, the rest of it zero-filled.
__device__ __forceinline__ void cp_async_head(uint32_t *smem_dst, const int32_t *src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
                 "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Round constants and the padding block's schedule in shared memory.
struct PadKW {
    uint32_t kw[64];  // K_t + W_t of the final block of a message of 64k bytes (padding only)
};

__device__ __forceinline__ void load_tables(uint32_t *sK, uint32_t *sPad, const PadKW &pad) {
    for (int i = threadIdx.x; i < 64; i += blockDim.x) {
        sK[i] = pk::kSha256K[i];
        sPad[i] = pad.kw[i];
    }
}

// ---------------------------------------------------------------------------
// Chunk digests: one thread per chunk, 32 consecutive chunks per warp.  Token
// blocks are staged through a 3-deep shared-memory ring with cp.async, so the
// load of block b+2 overlaps the compression of block b (a chunk's tokens need
// only be 4-byte aligned).  For chunk sizes that
// are multiples of 16 tokens the final block is pure padding, identical for
// every chunk: it runs as rounds only on a schedule precomputed on the host.
// ---------------------------------------------------------------------------
constexpr int kDigestBlock = 128;
constexpr int kStages = 3;

constexpr int kRingRow = 20;  // words per thread and stage: 16, and 4 so that a quarter warp's 16-byte rows differ in bank
typedef uint32_t RingStage[kDigestBlock][kRingRow];

// c = SHA-256 of chunk g (request r), written to keys[g] if `mine` (all 32
// lanes call, those past the batch with its last chunk).  F is the round
// form (pk_sha256.cuh: kAddsFma when several warps share each sub-partition).
// Prompts packed back to back start at any 4-byte address: the ring then
// holds the 16-byte aligned pieces that cover the chunk, and block b is read
// from pieces b and b + 1 at the chunk's word offset: 900 ragged prompts of
// chunks of 256, key derivation 175 -> 142 us.  (Read with 4-byte
// loads straight from global memory, one warp instruction touched 32 sectors
// for 128 bytes and nothing was in flight during a compression.)
template <int F>
__device__ __forceinline__ void digest_chunk(const int32_t *tokens, const int64_t *tok_off,
                                             const int64_t *key_off, uint32_t r, int64_t g, uint32_t C,
                                             const uint32_t *sK, const uint32_t *sPad, RingStage *ring, uint8_t *keys,
                                             uint32_t one, bool mine) {
    const int64_t i = g - __ldcg(key_off + r);
    const int32_t *src = tokens + __ldcg(tok_off + r) + i * (int64_t)C;
    const uint32_t o = (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15) / 4;  // the chunk's offset in its first 16 bytes
    const int32_t *base = src - o;

    uint32_t st[8];
    pk::init_state(st);
    const uint32_t nfull = C / 16;
    uint32_t w[16];
    if (__all_sync(0xffffffffu, base >= tokens)) {
        const bool shifted = __any_sync(0xffffffffu, o != 0);
        // Pieces 0 .. nfull - 1 lie inside the chunk; of piece nfull the last block needs o words.
        auto load_piece = [&](uint32_t b, uint32_t stage) {
            if (b < nfull) cp_async_block(ring[stage][threadIdx.x], base + 16 * b);
            else if (b == nfull && o) cp_async_head(ring[stage][threadIdx.x], base + 16 * b, 4 * o);
            cp_async_commit();
        };
#pragma unroll
        for (uint32_t b = 0; b < kStages - 1; ++b) load_piece(b, b);
        // one loop per case, so that the rounds need not wait for the last word of the block
        if (shifted) {
#pragma unroll 1
            for (uint32_t b = 0; b < nfull; ++b) {
                load_piece(b + kStages - 1, (b + kStages - 1) % kStages);
                cp_async_wait<kStages - 2>();  // pieces b and b + 1 have landed
                const uint32_t *A = ring[b % kStages][threadIdx.x] + o, *B = ring[(b + 1) % kStages][threadIdx.x] + o;
#pragma unroll
                for (int t = 0; t < 16; ++t)  // word o + t of the two pieces (o <= 3)
                    w[t] = pk::bswap32(t < 13 || o + t < 16 ? A[t] : B[t - 16]);
                pk::compress_rolled<F>(st, w, sK, one);
            }
        } else {
#pragma unroll 1
            for (uint32_t b = 0; b < nfull; ++b) {
                load_piece(b + kStages - 1, (b + kStages - 1) % kStages);
                cp_async_wait<kStages - 1>();  // piece b has landed
                const uint4 *q = reinterpret_cast<const uint4 *>(ring[b % kStages][threadIdx.x]);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint4 x = q[v];
                    w[4 * v + 0] = pk::bswap32(x.x);
                    w[4 * v + 1] = pk::bswap32(x.y);
                    w[4 * v + 2] = pk::bswap32(x.z);
                    w[4 * v + 3] = pk::bswap32(x.w);
                }
                pk::compress_rolled<F>(st, w, sK, one);
            }
        }
        cp_async_wait<0>();
    } else {  // the token buffer itself starts inside these 16 bytes
#pragma unroll 1
        for (uint32_t b = 0; b < nfull; ++b) {
            load_block_global(src + 16 * b, w);
            pk::compress_rolled<F>(st, w, sK, one);
        }
    }
    const uint64_t bits = (uint64_t)C * 32u;
    const int rem = (int)(C % 16);
    if (rem == 0) {
        pk::compress_kw<F>(st, sPad, one);
    } else {
        const int32_t *tail = src + 16 * nfull;
#pragma unroll
        for (int t = 0; t < 16; ++t)
            w[t] = t < rem ? pk::bswap32((uint32_t)__ldcg(tail + t)) : (t == rem ? 0x80000000u : 0u);
        if (rem <= 13) {
            w[14] = (uint32_t)(bits >> 32);
            w[15] = (uint32_t)bits;
            pk::compress_rolled<F>(st, w, sK, one);
        } else {
            pk::compress_rolled<F>(st, w, sK, one);
#pragma unroll
            for (int t = 0; t < 16; ++t) w[t] = 0;
            w[14] = (uint32_t)(bits >> 32);
            w[15] = (uint32_t)bits;
            pk::compress_rolled<F>(st, w, sK, one);
        }
    }
    if (mine) store_digest(keys + 32 * g, st);
}

// Optional descriptor work for the same launch (fused a0): the first
// desc_blocks blocks hash descriptor encodings instead, one warp each.
struct DescWork {
    const uint8_t *enc;
    uint64_t enc_bytes;
    const int64_t *enc_off;
    uint32_t D;
    uint8_t *digests;
    int32_t *status;
    uint32_t desc_blocks;
};

// `one` is the run-time constant 1 of the multiply-add round form.
template <int F>
__global__ void __launch_bounds__(kDigestBlock)
k_chunk_digest(const int32_t *tokens, const int64_t *tok_off,
               const int64_t *key_off, uint32_t R, uint32_t C, const __grid_constant__ PadKW pad,
               uint8_t *keys, const __grid_constant__ DescWork dw, uint32_t one) {
    __shared__ uint32_t sK[64], sPad[64];
    __shared__ __align__(16) RingStage ring[kStages];
    // The successor (the chain) is released as each block finishes, not at its start: released early,
    // its waiting CTAs, and those of the kernel after it, would sit on the SMs during the whole digest.
    if (blockIdx.x < dw.desc_blocks) {
        const uint8_t *enc = dw.enc;
        const int64_t *enc_off = dw.enc_off;
        uint8_t *digests = dw.digests;
        int32_t *dstatus = dw.status;
        pk::pdl_wait(enc, enc_off, digests, dstatus);
        const uint32_t warp = threadIdx.x >> 5;
        const uint32_t j = blockIdx.x * (kDigestBlock / 32) + warp;
        uint8_t *stage = reinterpret_cast<uint8_t *>(ring[0]) + warp * kDescStage;  // 4 x 2 KiB of the ring
        if (j < dw.D) hash_descriptor_bytes(stage, enc, dw.enc_bytes, enc_off, j, digests, dstatus);
        pk::pdl_launch_dependents();
        return;
    }
    load_tables(sK, sPad, pad);
    __syncthreads();
    pk::pdl_wait(tokens, tok_off, key_off, keys);
    if (R == 0) return;
    // all chunks, in tiles of one block, grid-strided
    // (the warp index from a shuffle and the chunk clamped to the batch: uniform control flow, see lane_request_guess)
    const int64_t g_end = __ldcg(key_off + R);
    const uint32_t nblocks = gridDim.x - dw.desc_blocks;
    const uint32_t warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    for (int64_t g0 = (int64_t)(blockIdx.x - dw.desc_blocks) * kDigestBlock + 32 * warp; g0 < g_end;
         g0 += (int64_t)nblocks * kDigestBlock) {
        const int64_t g = g0 + lane < g_end ? g0 + lane : g_end - 1;
        const uint32_t r = pk::lane_request_guess(key_off, R, g0, g_end, g);
        digest_chunk<F>(tokens, tok_off, key_off, r, g, C, sK, sPad, ring, keys, one, g0 + lane < g_end);
    }
    pk::pdl_launch_dependents();
}

// The chunk digests of a batch of few chunks, by pairs of warps (pk_pair.cuh): 16 chunks per pair.  CTA c of the
// work CTAs serves pairs [c * P / ctas, (c + 1) * P / ctas), at most three.
struct ChunkWords {
    const int32_t *src;  // the chunk's tokens (nullptr: a lane without a chunk)
    uint32_t C;
    uint32_t last;  // the block that holds the length
    __device__ __forceinline__ bool inside(uint32_t b) const { return src && 16 * b + 16 <= C; }
    __device__ __forceinline__ const uint32_t *block(uint32_t b) const {
        return reinterpret_cast<const uint32_t *>(src) + 16 * b;
    }
    __device__ __forceinline__ uint32_t load(uint32_t b, uint32_t t) const {
        const uint32_t i = 16 * b + t;
        return src && i < C ? (uint32_t)__ldcg(src + i) : 0u;
    }
    __device__ __forceinline__ int tail(uint32_t) const { return -1; }
    __device__ __forceinline__ uint32_t tail_word(uint32_t) const { return 0u; }
    __device__ __forceinline__ uint32_t word(uint32_t b, uint32_t t, uint32_t x) const {
        const uint32_t i = 16 * b + t;
        if (i < C) return pk::bswap32(x);
        const uint64_t bits = (uint64_t)C * 32u;
        if (b == last && t >= 14) return t == 14 ? (uint32_t)(bits >> 32) : (uint32_t)bits;
        return i == C ? 0x80000000u : 0u;
    }
};

__global__ void __launch_bounds__(pk::kPairThreads)
k_chunk_digest_pairs(const int32_t *tokens, const int64_t *tok_off, const int64_t *key_off, uint32_t R, uint32_t C,
                     const __grid_constant__ PadKW pad, uint8_t *keys, const __grid_constant__ DescWork dw, uint32_t one) {
    extern __shared__ __align__(16) uint8_t pair_smem[];
    pk::PairSmem &sm = *reinterpret_cast<pk::PairSmem *>(pair_smem);
    static_assert(sizeof(sm.ring) >= (size_t)kDescStage * kDescWarps, "descriptor staging fits in the rings");
    if (blockIdx.x < dw.desc_blocks) {
        const uint8_t *enc = dw.enc;
        const int64_t *enc_off = dw.enc_off;
        uint8_t *digests = dw.digests;
        int32_t *dstatus = dw.status;
        uint32_t *sK = sm.zero;  // (not otherwise used by this CTA)
        for (uint32_t i = threadIdx.x; i < 64; i += blockDim.x) sK[i] = pk::kSha256K[i];
        __syncthreads();
        pk::pdl_wait(enc, enc_off, digests, dstatus);
        const uint32_t warp = threadIdx.x >> 5;
        const uint32_t j = blockIdx.x * kDescWarps + warp;
        uint8_t *stage = reinterpret_cast<uint8_t *>(sm.ring) + warp * kDescStage;
        if (warp < kDescWarps && j < dw.D) hash_descriptor<true>(stage, sK, enc, dw.enc_bytes, enc_off, j, digests, dstatus);
        pk::pdl_launch_dependents();
        return;
    }
    pair_tables(sm, pad.kw);
    __syncthreads();
    pk::pdl_wait(tokens, tok_off, key_off, keys);
    const int64_t total = __ldcg(key_off + R);
    const int64_t P = (total + pk::kPairMsgs - 1) / pk::kPairMsgs;
    const int64_t ctas = gridDim.x - dw.desc_blocks, c = blockIdx.x - dw.desc_blocks;
    const pk::PairRole role = pk::pair_role();
    const int64_t p = c * P / ctas + role.pair;
    if (role.pair < pk::kPairs && p < (c + 1) * P / ctas) {
        const pk::SplitLane l = pk::split_lane(one);
        const int64_t g0 = p * pk::kPairMsgs, g = g0 + ((threadIdx.x & 31) >> 1);
        const bool pad_block = C % 16 == 0;
        const uint32_t blocks = pad_block ? C / 16 : (C * 4ull + 9 + 63) / 64;
        if (role.sched) {
            const uint32_t r = pk::lane_request_guess(key_off, R, g0, total, g);
            const int32_t *src = nullptr;
            if (g < total) src = tokens + __ldcg(tok_off + r) + (g - __ldcg(key_off + r)) * (int64_t)C;
            pair_schedule(sm, role.pair, l, blocks, ChunkWords{src, C, pad_block ? blocks : blocks - 1});
        } else {
            uint32_t st[4];
            pair_rounds(sm, role.pair, l, blocks, pad_block, st);
            if (g < total) pair_store(keys + 32 * g, l, st);
        }
    }
    pk::pdl_launch_dependents();
    __syncthreads();  // stay resident until every pair's barriers are through
}

// ---------------------------------------------------------------------------
// Chain: k_i = SHA-256(k_{i-1} || d || c_i), serial in i for each request.
//
// A group of requests is served by a pair of warps:
//   rounds warp:   holds the state; runs the 64 rounds of block 1
//                  (k_{i-1} || d) and of block 2 (c_i || padding)
//   schedule warp: writes K_t + W_t for both blocks to shared memory:
//                  block 2's schedule depends on c_i only and is made one
//                  step ahead; block 1's depends on k_{i-1} and is made as
//                  soon as k_{i-1} is published.
// Two forms:
//   k_chain_split  two lanes per request (split rounds of pk_sha256.cuh), 16
//                  requests per pair: the shortest chain step, while the SM
//                  sub-partitions have room (up to four pairs per SM);
//   k_chain        one lane per request, 32 requests per pair, four pairs per
//                  CTA and one CTA per SM: the fewest ALU cycles per key, for
//                  batches that fill every sub-partition.
// Block 1's schedule is published in two slices, t = 16..31 and 32..63 (the
// rounds warp's rounds 16..31 overlap the making of the rest; small-block key
// derivation 654 -> 641 us in k_chain, three slices 646).  Named barriers of
// pair p (count 64, producer arrives, consumer syncs): 1 + 3p block-1 slice 1,
// and block 2 of the step (written before it); 2 + 3p block-1 slice 2; 3 + 3p
// k_i published.  Four pairs stay within the 16 named barriers.
// Per pair both warps run the same number of steps (the lanes' maximum), so
// every phase of every barrier gets exactly one arrive and one sync; the
// schedule warp signals the block-1 barriers of step i only after it has
// passed the k barrier of step i-1, so after the rounds warp's block-1 syncs
// of step i-1: it never arrives twice on a barrier the rounds warp has not
// yet synced.  Block 2's buffer for step i + 1 is written after the k barrier
// of step i - 1, when the rounds warp has finished the block 2 that last used
// it.  Lanes past their own request's last chunk keep computing (masked) so
// that the warps stay aligned.
// ---------------------------------------------------------------------------
constexpr int kChainLanes = 32;

// The largest n >= 0 of the warp, by reductions whose result the compiler knows to be uniform (see
// lane_request_guess: the chains' loops over it then count in uniform registers).
__device__ __forceinline__ int64_t warp_max(int64_t n) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)((uint64_t)n >> 32));
    const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)((uint64_t)n >> 32) == hi ? (uint32_t)n : 0u);
    return (int64_t)((uint64_t)hi << 32 | lo);
}

__device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// K+W words pass between the two warps four to a 16-byte vector ([t / 4][lane]): one shared-memory
// instruction per four words on either side.
struct ChainSmem {
    uint4 kw1[16][kChainLanes];     // block-1 K+W, t = 16..63 used
    uint4 kw2[2][16][kChainLanes];  // block-2 K+W, double-buffered by step parity
    uint4 kpub[2][kChainLanes];     // k_{i-1} for the schedule warp
    uint8_t order[2][4 * kChainLanes];  // longest_first's, of the rounds and of the schedule warp
};

// 16 schedule words t = 16q .. 16q+15 of the ring w (in place), K_t + W_t -> out[t / 4][lane]
// (F: round form of pk_sha256.cuh, `one` its run-time 1)
template <int F>
__device__ __forceinline__ void schedule16(uint32_t w[16], uint4 (*out)[kChainLanes], int q, uint32_t lane,
                                           uint32_t one) {
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        pk::sched_word<F>(w, j, one);
        o[j & 3] = pk::add2<F>(pk::kSha256K[16 * q + j], w[j], one);
        if ((j & 3) == 3) out[4 * q + (j >> 2)][lane] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// rounds t = 16q .. 16q+15 with K+W from shared memory
// (the 16 words are read into registers before the first round: a lone warp
// runs 64 rounds in 1917 instead of 2184 cycles, in the late form 1830 instead
// of 2233, when no round waits on its shared-memory read)
template <int F>
__device__ __forceinline__ void rounds16_kw(uint32_t v[8], const uint4 (*kw)[kChainLanes], int q, uint32_t lane,
                                            uint32_t one) {
    uint32_t a = v[0], b = v[1], c = v[2], d = v[3], e = v[4], f = v[5], g = v[6], h = v[7];
    uint32_t x[16];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const uint4 y = kw[4 * q + m][lane];
        x[4 * m] = y.x;
        x[4 * m + 1] = y.y;
        x[4 * m + 2] = y.z;
        x[4 * m + 3] = y.w;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) pk::round_kw<F>(a, b, c, d, e, f, g, h, x[j], one);
    v[0] = a; v[1] = b; v[2] = c; v[3] = d; v[4] = e; v[5] = f; v[6] = g; v[7] = h;
}

// Request `at` of a CTA's m, from r0 on: its first key, number of keys (0: none or out of order) and descriptor.
__device__ __forceinline__ void chain_request(const int64_t *key_off, const uint32_t *desc_idx, uint32_t D, uint32_t r0,
                                              uint32_t m, uint32_t at, int64_t &a, int64_t &n, uint32_t &di) {
    a = n = 0;
    di = 0;
    if (at >= m) return;
    const uint64_t r = (uint64_t)r0 + at;
    a = key_off[r];
    n = key_off[r + 1] - a;
    di = desc_idx[r];
    if (n < 0 || di >= D) n = 0;
}

// A pair runs as many steps as its longest request has chunks, and a step is the longer the more of the CTA's pairs
// still run.  So a CTA hands its requests to its pairs longest first: short pairs end early and leave their
// sub-partitions to the long ones, whose rounds and schedule share them with other pairs (with both warps of a pair on
// one sub-partition the long pair gains nothing).  Key derivation, lookup and store of R prompts whose chunk counts
// spread evenly in the logarithm over a factor of 16, in us before and after: R = 5000 of up to 255 chunks (three pairs)
// 602 and 553, 8000 of 125 (four) 359 and 324, 16384 of 128 (k_chain) 491 and 441.  Equal prompts take the order that
// they have, found by a vote over the counts, which are read beside the request's own: 8000 prompts 438 and 443.5
// (the schedules' places; next to the rounds of pair p + 1 or p - 1 449 and 451), 5000 753.0 and 754, 16384 651.1 and
// 652.5.
//
// Which of a CTA's m <= N requests, from r0 on, is at position `pos` when the longest come first (equal ones in their
// own order); at least m where there is none.  Every warp finds it by itself; `order` (N bytes) is its own.
template <int N>
__device__ __forceinline__ uint32_t longest_first(const int64_t *key_off, uint32_t r0, uint32_t m, uint32_t pos,
                                                  uint8_t *order) {
    constexpr int kPerLane = (N + 31) / 32;
    const uint32_t lane = threadIdx.x & 31;
    int32_t n[kPerLane];  // chunks, limited to 32 bits (the order only sets which requests share a pair); none: -1
    bool equal = true;
#pragma unroll
    for (int h = 0; h < kPerLane; ++h) {
        const uint32_t j = lane + 32 * h;
        const int64_t c = j < m ? key_off[(uint64_t)r0 + j + 1] - key_off[(uint64_t)r0 + j] : -1;
        n[h] = (int32_t)(c > INT32_MAX ? INT32_MAX : c < 0 ? -1 : c);
        const int32_t n0 = __shfl_sync(0xffffffffu, n[0], 0);
        equal = equal && (j >= m || n[h] == n0);
    }
    if (__all_sync(0xffffffffu, equal)) return pos;
    uint32_t rank[kPerLane] = {};
#pragma unroll
    for (int g = 0; g < kPerLane; ++g) {
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            const int32_t o = __shfl_sync(0xffffffffu, n[g], j);
#pragma unroll
            for (int h = 0; h < kPerLane; ++h) rank[h] += o > n[h] || (o == n[h] && 32 * g + j < (int)lane + 32 * h);
        }
    }
#pragma unroll
    for (int h = 0; h < kPerLane; ++h)
        if (rank[h] < N) order[rank[h]] = (uint8_t)(lane + 32 * h);
    __syncwarp();
    return order[pos];
}

// At most 64 registers (no spills): uncapped, the compiler took 81 and a small-block step whose
// lookup-and-store launch overlaps the chain's tail ran 910 -> 955 us.  `groups` = ceil(R / 32); CTA c serves
// groups [c * groups / gridDim.x, (c + 1) * groups / gridDim.x), at most four.  Pair p is rounds warp p and
// schedule warp 4 + (p + 2) % 4: a sub-partition holds the rounds of one pair and the schedule of another, which fills
// the issue slots that the rounds' dependency chain leaves idle.
// FS1, FS2: the forms (pk_sha256.cuh) of the schedule warp's additions for block 1 and block 2, `one` their
// run-time 1.  The rounds warp's dependency chain sets the step time, and a multiply-add's longer latency there made
// the chain slower (small-block key derivation 674 -> 718 us with every addition on the FMA pipe); it takes the late
// form, one add on the ALU after the rotations (580.9 -> 572.5 us against the compiler's form; both with uniform
// loops and warp roles, without them 605.4 and 613.9).  The schedule warp's two blocks differ:
// block 1's schedule (k_{i-1} || d) can start only when k_{i-1} is published, and the rounds warp waits for
// it after its 16th round, so it keeps the short-latency form; block 2's (c_i || padding) is made a step
// ahead, off the critical path, and its additions go to the FMA pipe, where they do not compete with the
// rounds warp's logic.  Small-block key derivation, measured: 683.7 us with both blocks in one loop and all
// schedule additions on the FMA pipe; 674.8 with all on the ALU; 661.9 with the blocks in two loops, all on
// the ALU; 655.8 as here.  Moving the small sigmas' shifts or rotations to the FMA pipe as well (mul.hi /
// mad.lo by 2^(32-n): 4 and 6 cycles per warp instruction there) lost on either block (666-707 us): the
// rounds warp's own multiply-adds queue behind them.  Block 2's first 16 words (K_t + W_t, set by
// block2_head) and step 0's whole block 2, made before the loop, take FS1: 668 -> 654 us against FS2.
constexpr int kChainPairs = 4;

template <int FS1, int FS2>
__global__ void __launch_bounds__(2 * kChainLanes * kChainPairs, 4)
k_chain(const int64_t *key_off, const uint32_t *desc_idx,
        const uint8_t *digests, uint32_t R, uint32_t D, uint8_t *keys, uint32_t groups, uint32_t one) {
    extern __shared__ __align__(16) uint8_t chain_smem[];
    pk::pdl_wait(key_off, desc_idx, digests, keys);  // successor released at the last step (see k_chunk_digest)
    const uint32_t lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const bool sched = warp >= (uint32_t)kChainPairs;
    const uint32_t pair = (sched ? warp + kChainPairs / 2 : warp) & (kChainPairs - 1);
    ChainSmem &sm = reinterpret_cast<ChainSmem *>(chain_smem)[pair];
    const uint32_t r0 = (uint32_t)((uint64_t)blockIdx.x * groups / gridDim.x) * kChainLanes;
    const uint64_t r1 = (uint64_t)(blockIdx.x + 1) * groups / gridDim.x * kChainLanes;
    const uint32_t m = (uint32_t)(r1 < R ? r1 : R) - r0;
    const uint32_t at = pair * kChainLanes + lane;
    const int bar_s1 = 1 + 3 * (int)pair;   // block-1 schedule (first slice), and block 2 of the step
    const int bar_s1b = 2 + 3 * (int)pair;  // block-1 schedule (second slice)
    const int bar_k = 3 + 3 * (int)pair;    // k_i published
    int64_t a, n;
    uint32_t di;
    chain_request(key_off, desc_idx, D, r0, m, at, a, n, di);
    const uint32_t pos = longest_first<kChainPairs * kChainLanes>(key_off, r0, m, at, sm.order[sched]);
    if (pos != at) chain_request(key_off, desc_idx, D, r0, m, pos, a, n, di);
    const int64_t nmax = warp_max(n);  // identical in both warps of the pair: they cover the same requests
    if (nmax == 0) {  // uniform over the pair
        pk::pdl_launch_dependents();
        __syncthreads();
        return;
    }

    uint32_t dw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (n > 0) {
        const uint4 *dq = reinterpret_cast<const uint4 *>(digests + 32ull * di);
        const uint4 d_lo = __ldcg(dq), d_hi = __ldcg(dq + 1);
        dw[0] = pk::bswap32(d_lo.x); dw[1] = pk::bswap32(d_lo.y); dw[2] = pk::bswap32(d_lo.z);
        dw[3] = pk::bswap32(d_lo.w); dw[4] = pk::bswap32(d_hi.x); dw[5] = pk::bswap32(d_hi.y);
        dw[6] = pk::bswap32(d_hi.z); dw[7] = pk::bswap32(d_hi.w);
    }
    uint4 *kq = reinterpret_cast<uint4 *>(keys + 32ull * a);

    if (sched) {  // ---------------- schedule warp ----------------
        // block 2 of step i: W = c_i (8 words) || 0x80000000, 0 x 6, 768; words 0..15 stored as K + W
        auto block2_head = [&](int64_t i, int buf, uint32_t w[16]) {
            if (i < n) {
                const uint4 lo = kq[2 * i], hi = kq[2 * i + 1];
                w[0] = pk::bswap32(lo.x); w[1] = pk::bswap32(lo.y); w[2] = pk::bswap32(lo.z); w[3] = pk::bswap32(lo.w);
                w[4] = pk::bswap32(hi.x); w[5] = pk::bswap32(hi.y); w[6] = pk::bswap32(hi.z); w[7] = pk::bswap32(hi.w);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) w[j] = 0;
            }
            w[8] = 0x80000000u;
#pragma unroll
            for (int j = 9; j < 15; ++j) w[j] = 0;
            w[15] = 96u * 8u;
#pragma unroll
            for (int m = 0; m < 4; ++m)
                sm.kw2[buf][m][lane] = make_uint4(
                    pk::add2<FS1>(pk::kSha256K[4 * m], w[4 * m], one), pk::add2<FS1>(pk::kSha256K[4 * m + 1], w[4 * m + 1], one),
                    pk::add2<FS1>(pk::kSha256K[4 * m + 2], w[4 * m + 2], one),
                    pk::add2<FS1>(pk::kSha256K[4 * m + 3], w[4 * m + 3], one));
        };
        {
            uint32_t w[16];
            block2_head(0, 0, w);
#pragma unroll 1
            for (int q = 1; q < 4; ++q) schedule16<FS1>(w, sm.kw2[0], q, lane, one);
        }
#pragma unroll 1
        for (int64_t i = 0; i < nmax; ++i) {
            if (i + 1 == nmax) pk::pdl_launch_dependents();
            uint32_t w[16];
            if (i == 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j) w[j] = 0;  // k_{-1} = 0^32
            } else {
                bar_sync(bar_k);  // k_{i-1} published; the rounds warp has finished step i-1
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const uint4 y = sm.kpub[m][lane];
                    w[4 * m] = y.x;
                    w[4 * m + 1] = y.y;
                    w[4 * m + 2] = y.z;
                    w[4 * m + 3] = y.w;
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) w[8 + j] = dw[j];
            const int buf = (int)((i + 1) & 1);
            schedule16<FS1>(w, sm.kw1, 1, lane, one);
            bar_arrive(bar_s1);  // also: block 2 of step i ready
#pragma unroll 1
            for (int sl = 2; sl <= 3; ++sl) schedule16<FS1>(w, sm.kw1, sl, lane, one);
            bar_arrive(bar_s1b);
            if (i + 1 < nmax) {
                block2_head(i + 1, buf, w);
#pragma unroll 1
                for (int sl = 1; sl <= 3; ++sl) schedule16<FS2>(w, sm.kw2[buf], sl, lane, one);
            }
        }
        __syncthreads();  // stay resident until the rounds warp has consumed every phase
        return;
    }

    // ---------------- rounds warp ----------------
    uint32_t p[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // k_{-1} = 0^32
    uint32_t kd[8];                            // K_t + d_{t-8}, t = 8..15
#pragma unroll
    for (int j = 0; j < 8; ++j) kd[j] = pk::kSha256K[8 + j] + dw[j];
#pragma unroll 1
    for (int64_t i = 0; i < nmax; ++i) {
        if (i + 1 == nmax) pk::pdl_launch_dependents();
        uint32_t v[8] = {PK_IV0, PK_IV1, PK_IV2, PK_IV3, PK_IV4, PK_IV5, PK_IV6, PK_IV7};
        {   // block 1, rounds 0..15: W = k_{i-1} || d
            uint32_t a_ = v[0], b_ = v[1], c_ = v[2], d_ = v[3], e_ = v[4], f_ = v[5], g_ = v[6], h_ = v[7];
#pragma unroll
            for (int j = 0; j < 8; ++j) pk::round_kw<pk::kAddsLate>(a_, b_, c_, d_, e_, f_, g_, h_, pk::kSha256K[j] + p[j], one);
#pragma unroll
            for (int j = 0; j < 8; ++j) pk::round_kw<pk::kAddsLate>(a_, b_, c_, d_, e_, f_, g_, h_, kd[j], one);
            v[0] = a_; v[1] = b_; v[2] = c_; v[3] = d_; v[4] = e_; v[5] = f_; v[6] = g_; v[7] = h_;
        }
        bar_sync(bar_s1);
        rounds16_kw<pk::kAddsLate>(v, sm.kw1, 1, lane, one);
        bar_sync(bar_s1b);
        rounds16_kw<pk::kAddsLate>(v, sm.kw1, 2, lane, one);
        rounds16_kw<pk::kAddsLate>(v, sm.kw1, 3, lane, one);
        uint32_t st[8] = {PK_IV0 + v[0], PK_IV1 + v[1], PK_IV2 + v[2], PK_IV3 + v[3],
                          PK_IV4 + v[4], PK_IV5 + v[5], PK_IV6 + v[6], PK_IV7 + v[7]};
        const uint4 (*kw2)[kChainLanes] = sm.kw2[i & 1];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = st[j];
#pragma unroll 1
        for (int q = 0; q < 4; ++q) rounds16_kw<pk::kAddsLate>(v, kw2, q, lane, one);
#pragma unroll
        for (int j = 0; j < 8; ++j) p[j] = st[j] + v[j];
        if (i < n) store_digest(keys + 32ull * (a + i), p);
        if (i + 1 < nmax) {
#pragma unroll
            for (int m = 0; m < 2; ++m) sm.kpub[m][lane] = make_uint4(p[4 * m], p[4 * m + 1], p[4 * m + 2], p[4 * m + 3]);
            bar_arrive(bar_k);
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Chain with two lanes per request (split rounds and split schedule of
// pk_sha256.cuh): 16 requests per pair of warps.  The chain of one request is
// serial, so with few requests a step's latency is all that counts: a step is
// 132 slots of about 24 cycles.  With one pair per CTA the two warps run on
// different sub-partitions; with three, the rounds warps have a sub-partition
// each and the schedule warps share the fourth; with four, pair p is rounds
// warp p and schedule warp 4 + (p + 2) % 4, as in k_chain.  The rounds are straight-line code (block 2
// as a loop of 16 rounds: long-context key derivation 938 -> 1013 us), each
// 16 words of K + W read while the 16 rounds before them run, and each barrier synced
// some slots before the words it guards are needed.  The schedule warp's work
// still costs the rounds warp about 5% (865 -> 824 us with its arithmetic removed):
// its shared-memory traffic is kept to 16-byte vectors (938 -> 924 us) and its
// slices run one copy of the code.  Long-context key derivation (64 chains of
// 512 steps) 1060 -> 925 us against one lane per request, 865 us with the
// select's P on the FMA pipe.
// ---------------------------------------------------------------------------
constexpr int kSplitReq = 16;                // requests per pair
// A request's K+W row: its 32 even words, then (kSplitOdd) its 32 odd ones, each as 16-byte vectors.  The
// schedule warp's lane stores four words of its parity at once; the row stride puts the vectors of a quarter
// warp on distinct banks on either side.
constexpr int kSplitOdd = 36;
constexpr int kSplitRow = 72;
struct SplitSmem {
    uint32_t kw1[kSplitReq][kSplitRow];      // block-1 K+W, t = 16..63 used
    uint32_t kw2[2][kSplitReq][kSplitRow];   // block-2 K+W, double-buffered by step parity
    uint32_t zero[kSplitRow];                // the odd lanes' K+W
    uint32_t kpub[kSplitReq][2][4];          // k_{i-1}: its even words, its odd words
    uint32_t kpar[2][32];                    // K of the even and of the odd t
    uint8_t order[2][4 * kSplitReq];         // longest_first's, of the rounds and of the schedule warp
};

// K+W of rounds 16s .. 16s + 15
__device__ __forceinline__ void ld16(uint32_t k[16], const uint32_t *row, int s) {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const uint4 y = *reinterpret_cast<const uint4 *>(row + kSplitOdd * par + 8 * s + 4 * m);
            k[8 * m + par] = y.x;
            k[8 * m + 2 + par] = y.y;
            k[8 * m + 4 + par] = y.z;
            k[8 * m + 6 + par] = y.w;
        }
    }
}

// Warps of a CTA of kPairs pairs: with three pairs the rounds warps are warps 0, 1, 2 and the schedule warps 3, 7,
// 11 (warps 4-6 and 8-10 do nothing).
constexpr int split_warps(int pairs) { return pairs == 3 ? 12 : 2 * pairs; }

template <int kPairs>
__global__ void __launch_bounds__(32 * split_warps(kPairs))
k_chain_split(const int64_t *key_off, const uint32_t *desc_idx, const uint8_t *digests, uint32_t R, uint32_t D,
              uint8_t *keys, uint32_t groups, uint32_t one) {
    extern __shared__ __align__(16) uint8_t chain_smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool sched = kPairs == 3 ? (warp & 3) == 3 : warp >= (uint32_t)kPairs;
    const uint32_t pair = kPairs == 1 ? 0u : !sched ? warp : kPairs == 3 ? warp >> 2 : (warp + 2) & 3;
    if (kPairs == 3 && pair >= 3) {
        __syncthreads();
        return;
    }
    const uint32_t q = lane >> 1, par = lane & 1;
    SplitSmem &sm = reinterpret_cast<SplitSmem *>(chain_smem)[pair];
    if (sched) {
        sm.kpar[lane & 1][lane >> 1] = pk::kSha256K[lane];
        sm.kpar[lane & 1][16 + (lane >> 1)] = pk::kSha256K[32 + lane];
    } else {
        for (int t = lane; t < kSplitRow; t += 32) sm.zero[t] = 0u;
    }
    __syncwarp();
    pk::pdl_wait(key_off, desc_idx, digests, keys);  // successor released at the last step (see k_chunk_digest)
    uint32_t r0 = blockIdx.x * kSplitReq, m = R - r0, at = q;
    if (kPairs > 1) {
        r0 = (uint32_t)((uint64_t)blockIdx.x * groups / gridDim.x) * kSplitReq;
        const uint64_t r1 = (uint64_t)(blockIdx.x + 1) * groups / gridDim.x * kSplitReq;
        m = (uint32_t)(r1 < R ? r1 : R) - r0;
        at = pair * kSplitReq + q;
    }
    const int bar_s1 = 1 + 3 * (int)pair;   // block-1 schedule t = 16..31, and block 2 of the step
    const int bar_s1b = 2 + 3 * (int)pair;  // block-1 schedule t = 32..63
    const int bar_k = 3 + 3 * (int)pair;    // k_i published
    int64_t a, n;
    uint32_t di;
    chain_request(key_off, desc_idx, D, r0, m, at, a, n, di);
    if (kPairs > 1) {
        const uint32_t pos = longest_first<kPairs * kSplitReq>(key_off, r0, m, at, sm.order[sched]);
        if (pos != at) chain_request(key_off, desc_idx, D, r0, m, pos, a, n, di);
    }
    const int64_t nmax = warp_max(n);  // identical in both warps of the pair: they cover the same requests
    if (nmax == 0) {  // uniform over the pair
        pk::pdl_launch_dependents();
        if (kPairs > 1) __syncthreads();
        return;
    }
    uint32_t dw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (n > 0) {
        const uint4 *dq = reinterpret_cast<const uint4 *>(digests + 32ull * di);
        const uint4 lo = __ldcg(dq), hi = __ldcg(dq + 1);
        dw[0] = pk::bswap32(lo.x); dw[1] = pk::bswap32(lo.y); dw[2] = pk::bswap32(lo.z); dw[3] = pk::bswap32(lo.w);
        dw[4] = pk::bswap32(hi.x); dw[5] = pk::bswap32(hi.y); dw[6] = pk::bswap32(hi.z); dw[7] = pk::bswap32(hi.w);
    }
    const pk::SplitLane l = pk::split_lane(one);
    uint4 *kq = reinterpret_cast<uint4 *>(keys + 32ull * a);

    if (sched) {  // ---------------- schedule warp ----------------
        // c_i, loaded a step ahead of the schedule made from it
        uint4 c_lo = make_uint4(0, 0, 0, 0), c_hi = c_lo;
        auto fetch = [&](int64_t i) {
            if (i < n) {
                c_lo = __ldcg(kq + 2 * i);
                c_hi = __ldcg(kq + 2 * i + 1);
            }
        };
        // constant words t = 8..15 of block 2, in both buffers
#pragma unroll
        for (int i = 4; i < 8; ++i) {
            const uint32_t t = 2 * i + par;
            const uint32_t w = t == 8 ? 0x80000000u : t == 15 ? 96u * 8u : 0u;
            sm.kw2[0][q][kSplitOdd * par + i] = sm.kpar[par][i] + w;
            sm.kw2[1][q][kSplitOdd * par + i] = sm.kpar[par][i] + w;
        }
        uint32_t own[8], far[8], down[4], dfar[5];
#pragma unroll
        for (int j = 0; j < 4; ++j) {  // block 1: own[4 + j] = down[j], far[3 + j] = dfar[j]
            down[j] = par ? dw[2 * j + 1] : dw[2 * j];
            dfar[j + 1] = par ? (j < 3 ? dw[2 * j + 2] : 0u) : dw[2 * j + 1];
        }
        dfar[0] = dw[0];
        // next 16 words t = 16s .. 16s + 15 of the ring -> K + W in row
        auto slice = [&](uint32_t *row, int s) {
            const uint4 *kp = reinterpret_cast<const uint4 *>(&sm.kpar[par][8 * s]);
            const uint4 ka = kp[0], kb = kp[1];
            uint4 *o = reinterpret_cast<uint4 *>(row + kSplitOdd * par + 8 * s);
            pk::split_sched8(own, far, l);
            o[0] = make_uint4(own[0] + ka.x, own[1] + ka.y, own[2] + ka.z, own[3] + ka.w);
            o[1] = make_uint4(own[4] + kb.x, own[5] + kb.y, own[6] + kb.z, own[7] + kb.w);
        };
        auto block2 = [&](int64_t i, int buf) {  // words of block 2 of step i: c_i || 0x80000000, 0 x 6, 768
            const uint32_t c[8] = {pk::bswap32(c_lo.x), pk::bswap32(c_lo.y), pk::bswap32(c_lo.z), pk::bswap32(c_lo.w),
                                   pk::bswap32(c_hi.x), pk::bswap32(c_hi.y), pk::bswap32(c_hi.z), pk::bswap32(c_hi.w)};
            fetch(i + 1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                own[j] = par ? c[2 * j + 1] : c[2 * j];
                far[j] = par ? (j < 3 ? c[2 * j + 2] : 0x80000000u) : c[2 * j + 1];
            }
            const uint4 ka = *reinterpret_cast<const uint4 *>(sm.kpar[par]);
            *reinterpret_cast<uint4 *>(sm.kw2[buf][q] + kSplitOdd * par) =
                make_uint4(own[0] + ka.x, own[1] + ka.y, own[2] + ka.z, own[3] + ka.w);
            own[4] = par ? 0u : 0x80000000u;
            own[5] = own[6] = 0u;
            own[7] = par ? 96u * 8u : 0u;
            far[4] = far[5] = far[6] = far[7] = 0u;
        };
        *reinterpret_cast<uint4 *>(sm.kpub[q][par]) = make_uint4(0, 0, 0, 0);  // k_{-1} = 0^32
        __syncwarp();
        fetch(0);
        block2(0, 0);
#pragma unroll 1
        for (int s = 1; s < 4; ++s) slice(sm.kw2[0][q], s);
#pragma unroll 1
        for (int64_t i = 0; i < nmax; ++i) {
            if (i + 1 == nmax) pk::pdl_launch_dependents();
            if (i > 0) bar_sync(bar_k);  // k_{i-1} published; the rounds warp has finished step i-1
            {
                const uint4 x = *reinterpret_cast<const uint4 *>(sm.kpub[q][par]);
                const uint4 y = *reinterpret_cast<const uint4 *>(sm.kpub[q][par ^ 1]);
                own[0] = x.x; own[1] = x.y; own[2] = x.z; own[3] = x.w;
                far[0] = par ? y.y : y.x;
                far[1] = par ? y.z : y.y;
                far[2] = par ? y.w : y.z;
                far[3] = par ? dfar[0] : y.w;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    own[4 + j] = down[j];
                    far[4 + j] = dfar[j + 1];
                }
            }
            const int buf = (int)((i + 1) & 1);
            const int slices = i + 1 < nmax ? 6 : 3;
#pragma unroll 1
            for (int s = 1; s <= slices; ++s) {  // one copy of the slice body
                if (s == 4) block2(i + 1, buf);
                slice(s <= 3 ? sm.kw1[q] : sm.kw2[buf][q], s <= 3 ? s : s - 3);
                if (s == 1) bar_arrive(bar_s1);
                else if (s == 3) bar_arrive(bar_s1b);
            }
        }
        __syncthreads();  // stay resident until the rounds warp has consumed every phase
        return;
    }

    // ---------------- rounds warp ----------------
    const uint32_t iv[4] = {l.even ? PK_IV4 : PK_IV0, l.even ? PK_IV5 : PK_IV1, l.even ? PK_IV6 : PK_IV2,
                            l.even ? PK_IV7 : PK_IV3};
    const uint32_t mA = l.even ? 1u : 0u;
    uint32_t kc[8], kd[8];  // K_t, t = 0..7, and K_t + d_{t-8}, t = 8..15, in the even lanes
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        kc[j] = l.even ? pk::kSha256K[j] : 0u;
        kd[j] = l.even ? pk::kSha256K[8 + j] + dw[j] : 0u;
    }
    const uint32_t *row1 = l.even ? sm.kw1[q] : sm.zero;
    uint32_t p[4] = {0, 0, 0, 0};  // k_{-1} = 0^32 (even lane: words 4..7, odd lane: words 0..3)
    __syncwarp();
#pragma unroll 1
    for (int64_t i = 0; i < nmax; ++i) {
        if (i + 1 == nmax) pk::pdl_launch_dependents();
        uint32_t k[16], kn[16], cd[2];
        uint32_t st[4] = {iv[0], iv[1], iv[2], iv[3]};
        pk::SplitState v;
        pk::split_start(v, l, st, PK_IV2, PK_IV3);
        // block 1, rounds 0..15: W = k_{i-1} || d
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, p[j], 1);
            k[j] = pk::mad1(o, mA, kc[j]);
            k[4 + j] = pk::mad1(p[j], mA, kc[4 + j]);
        }
        pk::split_slot<true>(v, l, k[0], st[1]);
        pk::split_slot<true>(v, l, k[1], st[0]);
#pragma unroll
        for (int j = 2; j < 8; ++j) pk::split_slot(v, l, k[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) pk::split_slot(v, l, kd[j]);
        bar_sync(bar_s1);
        ld16(kn, row1, 1);
#pragma unroll
        for (int j = 4; j < 8; ++j) pk::split_slot(v, l, kd[j]);
#pragma unroll
        for (int j = 0; j < 12; ++j) pk::split_slot(v, l, kn[j]);
        bar_sync(bar_s1b);
        ld16(k, row1, 2);
#pragma unroll
        for (int j = 12; j < 16; ++j) pk::split_slot(v, l, kn[j]);
        ld16(kn, row1, 3);
#pragma unroll
        for (int j = 0; j < 16; ++j) pk::split_slot(v, l, k[j]);
        const uint32_t *r2 = l.even ? sm.kw2[i & 1][q] : sm.zero;
        ld16(k, r2, 0);
#pragma unroll
        for (int j = 0; j < 16; ++j) pk::split_slot(v, l, kn[j]);
        pk::split_end(v, l, st, cd);
        // block 2
        pk::split_start(v, l, st, PK_IV2 + cd[0], PK_IV3 + cd[1]);
        ld16(kn, r2, 1);
        pk::split_slot<true>(v, l, k[0], st[1]);
        pk::split_slot<true>(v, l, k[1], st[0]);
#pragma unroll
        for (int j = 2; j < 16; ++j) pk::split_slot(v, l, k[j]);
        ld16(k, r2, 2);
#pragma unroll
        for (int j = 0; j < 16; ++j) pk::split_slot(v, l, kn[j]);
        ld16(kn, r2, 3);
#pragma unroll
        for (int j = 0; j < 16; ++j) pk::split_slot(v, l, k[j]);
#pragma unroll
        for (int j = 0; j < 16; ++j) pk::split_slot(v, l, kn[j]);
        pk::split_end(v, l, st, cd);
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = st[j];
        const uint32_t half = l.even ? 1u : 0u;  // the even lane holds the second half of the key
        if (i + 1 < nmax) {
            *reinterpret_cast<uint2 *>(&sm.kpub[q][0][2 * half]) = make_uint2(p[0], p[2]);
            *reinterpret_cast<uint2 *>(&sm.kpub[q][1][2 * half]) = make_uint2(p[1], p[3]);
            bar_arrive(bar_k);
        }
        if (i < n)
            kq[2 * i + half] = make_uint4(pk::bswap32(p[0]), pk::bswap32(p[1]), pk::bswap32(p[2]), pk::bswap32(p[3]));
    }
    __syncthreads();
}

unsigned grid_for(uint64_t n, unsigned block) { return (unsigned)((n + block - 1) / block); }

// Dynamic shared memory of the kernels whose CTAs must not stack on an SM: padded past half of an SM's, or past a
// third for two per SM (a launch that becomes resident while its predecessor drains otherwise stacks CTAs on the SMs
// that free up first).  The price: while such a CTA runs, a CTA of another stream's kernel comes up on its SM only if
// it needs no more shared memory than is left (227 KB less 116, or less one or two times 76).
constexpr size_t kOnePerSm = 116 * 1024;
constexpr size_t kTwoPerSm = 76 * 1024;
static_assert(kOnePerSm >= kChainPairs * sizeof(ChainSmem) && kOnePerSm >= 4 * sizeof(SplitSmem) &&
                  kTwoPerSm >= sizeof(SplitSmem) && kOnePerSm >= sizeof(pk::PairSmem),
              "the kernels' shared memory fits");

// Raise those kernels' shared-memory limit, once per device.
cudaError_t raise_smem_limits() {
    static std::mutex mu;
    static bool done[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    auto raise = [&](auto *kernel) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOnePerSm);
    };
    raise(k_chunk_digest_pairs);
    raise(k_chain_split<1>);
    raise(k_chain_split<3>);
    raise(k_chain_split<4>);
    raise(k_chain<pk::kAddsPlain, pk::kAddsFma>);
    done[dev] = e == cudaSuccess;
    return e;
}

}  // namespace

cudaError_t pk_launch_digest_descriptors(const uint8_t *enc, uint64_t enc_bytes, const int64_t *enc_off,
                                         uint32_t D, uint8_t *digests, int32_t *status, cudaStream_t s) {
    if (D == 0) return cudaSuccess;
    const cudaError_t e =
        pk_launch(k_digest_descriptors, grid_for(D, kDescWarps), 32 * kDescWarps, s, enc, enc_bytes, enc_off, D,
                  digests, status);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t pk_launch_derive(const pk_ctx *ctx, const int32_t *tokens, uint64_t n_tokens,
                             const int64_t *tok_off, uint32_t R, const uint32_t *desc_idx,
                             const uint8_t *digests, uint32_t D, int64_t *key_off, uint8_t *keys,
                             uint64_t key_capacity, int32_t *status, cudaStream_t s) {
    return pk_launch_derive_enc(ctx, tokens, n_tokens, tok_off, R, desc_idx, nullptr, 0, nullptr, D,
                                const_cast<uint8_t *>(digests), key_off, keys, key_capacity, status, s);
}

cudaError_t pk_launch_derive_enc(const pk_ctx *ctx, const int32_t *tokens, uint64_t n_tokens,
                                 const int64_t *tok_off, uint32_t R, const uint32_t *desc_idx, const uint8_t *enc,
                                 uint64_t enc_bytes, const int64_t *enc_off, uint32_t D, uint8_t *digests,
                                 int64_t *key_off, uint8_t *keys, uint64_t key_capacity, int32_t *status,
                                 cudaStream_t s) {
    static_assert(kDigestBlock / 32 * kDescStage <= (int)sizeof(RingStage) * kStages,
                  "descriptor staging fits in the token ring");
    const uint32_t C = ctx->chunk_tokens;
    const uint32_t tiles = grid_for(R, kScanTile);
    cudaError_t e = pk_launch(tiles <= 1             ? k_chunk_offsets<false>
                              : tiles <= kScanTiles ? k_chunk_offsets<true>
                                                    : k_chunk_offsets_walk,
                              tiles > kScanTiles || tiles == 0 ? 1 : tiles, kScanThreads, s, tok_off, R, n_tokens, C,
                              desc_idx, D, key_capacity, key_off, status);
    if (e != cudaSuccess) return e;
    DescWork dw = {enc, enc_bytes, enc_off, D, digests, status, 0};
    if (enc_off) dw.desc_blocks = grid_for(D, kDigestBlock / 32);
    PadKW pad;
    for (int t = 0; t < 64; ++t) pad.kw[t] = ctx->pad_kw[t];
    const uint64_t most = n_tokens / C;  // chunks of the batch at most (the caller's buffers may hold many more)
    const bool chunks = R > 0 && most > 0;
    const uint32_t one = 1u;
    if (chunks) e = raise_smem_limits();
    if (e != cudaSuccess) return e;
    if (!chunks) {
        if (dw.desc_blocks)
            e = pk_launch(k_chunk_digest<pk::kAddsPlain>, dw.desc_blocks, kDigestBlock, s, tokens, tok_off,
                          (const int64_t *)key_off, 0u, C, pad, keys, dw, one);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    // The multiply-add round form from more than one warp of chunks per SM sub-partition (two warps 4610 against 5334
    // cycles per compression each; long-context key derivation, 1.7 warps per sub-partition, 870.7 -> 868.1 us).  Below
    // the line the two forms are close: key derivation at half a warp per sub-partition, compiler's form | multiply-add,
    // in us: chunks of 16 23.6 | 23.8, of 64 28.1 | 28.0, of 256 57.8 | 56.6; at one warp 26.3 | 25.9, 35.2 | 33.8,
    // 78.7 | 73.3.  With an unknown SM count the compiler's form is kept.
    const uint64_t warps = (most + 31) / 32;
    const bool fma = ctx->sm_count > 0 && warps > 4ull * ctx->sm_count;
    const unsigned grid = grid_for(most, kDigestBlock) + dw.desc_blocks;
    // Few chunks: pairs of warps, at most three per SM, on the SMs that the descriptors and the offsets kernel, still
    // running when this launch comes up, leave free.  Key derivation of N chunks (8 per request), one lane per chunk |
    // pairs, in us: chunks of 256, N = 16: 38.0 | 31.4, 2400: 45.4 | 39.2, 7000: 45.6 | 44.6; chunks of 64: 21.1 |
    // 20.9, 28.0 | 27.5, 28.3 | 28.9; chunks of 16: 19.7 | 17.5, 26.2 | 24.8, 26.7 | 25.3.
    const uint32_t desc_sms = enc_off ? grid_for(D, kDescWarps) : 0;
    const uint32_t work = ctx->sm_count > desc_sms + 1 ? ctx->sm_count - desc_sms - 1 : 0;
    if (C <= 1u << 30 && most <= (uint64_t)pk::kPairMsgsPerSm * work) {
        dw.desc_blocks = desc_sms;
        const uint64_t pairs = (most + pk::kPairMsgs - 1) / pk::kPairMsgs;
        e = pk_launch_smem(k_chunk_digest_pairs, (unsigned)(pairs < work ? pairs : work) + desc_sms, pk::kPairThreads,
                           kOnePerSm, s, tokens, tok_off, (const int64_t *)key_off, R, C, pad, keys, dw, one);
    } else if (fma) {
        e = pk_launch(k_chunk_digest<pk::kAddsFma>, grid, kDigestBlock, s, tokens, tok_off, (const int64_t *)key_off, R, C,
                      pad, keys, dw, one);
    } else {
        e = pk_launch(k_chunk_digest<pk::kAddsPlain>, grid, kDigestBlock, s, tokens, tok_off, (const int64_t *)key_off, R, C,
                      pad, keys, dw, one);
    }
    if (e != cudaSuccess) return e;
    // Chains, by pairs of 16 requests per SM (rounded up).  Key derivation of R prompts of 32 chunks of 16
    // tokens, measured, in us, for: two lanes per request, one pair per CTA | three | four | one lane per request:
    // R = 2432 (1 pair per SM) 73 | - | 94 | 112;  4864 (2) 83 | - | 103 | 121;  7296 (3) 134 | 110 | 114 | 131;
    // 9728 (4) 145 | - | 126 | 143;  11000 (5) 197 | - | 201 | 148;  16384 (7) 263 | - | 225 | 172.
    const uint32_t groups = grid_for(R, kSplitReq);
    const uint32_t sms = ctx->sm_count;
    const uint32_t per_sm = sms ? grid_for(groups, sms) : 1;
    if (per_sm <= 2) {
        // Shared memory padded so that no SM takes more than its share of the CTAs (R = 4864 without: 123 us).
        const size_t smem = per_sm == 1 ? kOnePerSm : kTwoPerSm;
        e = pk_launch_smem(k_chain_split<1>, groups, 64, smem, s, (const int64_t *)key_off, desc_idx,
                               (const uint8_t *)digests, R, D, keys, groups, one);
    } else if (per_sm == 3) {
        e = pk_launch_smem(k_chain_split<3>, sms, 32 * split_warps(3), kOnePerSm, s, (const int64_t *)key_off,
                               desc_idx, (const uint8_t *)digests, R, D, keys, groups, one);
    } else if (per_sm == 4) {
        e = pk_launch_smem(k_chain_split<4>, sms, 32 * split_warps(4), kOnePerSm, s, (const int64_t *)key_off, desc_idx,
                               (const uint8_t *)digests, R, D, keys, groups, one);
    } else {
        const uint32_t g32 = grid_for(R, kChainLanes);
        const uint32_t grid = g32 <= 4 * sms ? sms : grid_for(g32, 4);
        e = pk_launch_smem(k_chain<pk::kAddsPlain, pk::kAddsFma>, grid, 8 * kChainLanes, kOnePerSm, s,
                               (const int64_t *)key_off, desc_idx, (const uint8_t *)digests, R, D, keys, g32, one);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

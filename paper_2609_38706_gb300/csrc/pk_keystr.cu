// pk_keystr.cu -- connector key strings of a key batch (Sec. 5.3, connector
// integration).  A connector whose wire format is a fixed-width text field
// carries the 128-bit digest as twenty-two base64 characters: the standard
// alphabet of RFC 4648, Sec. 4, with the two "=" of padding dropped (16 bytes
// give 21 full 6-bit groups and 2 leftover bits, the last character's low
// four bits zero).  Row i of the output is
//     prefix || base64(first 16 bytes of k_i) || zero bytes up to the row width
// where the prefix (the connector's fixed fields and the model tag) is the
// same for every row.
//
// Output bytes dominate the traffic (the row width against 16 key bytes read
// per row), so the kernel is built to write at HBM speed: a persistent grid,
// each CTA holding two tiles of 256 rows in shared memory, laid out exactly
// as in the output (256 * width bytes, a multiple of 16) and filled once with
// the prefix and zeros: 16 rows are written one byte column per thread, the
// rest is copied from them 16 bytes at a time, so that no store depends on the
// width for its bank conflicts.  (A row per thread, byte by byte, took 2 us of
// a 4 us launch of 1,000 rows of 150 bytes, and 14 us at 240 bytes, where the
// rows of a warp fall on few banks.)  Per tile only the 22 characters of each
// row change: each thread encodes its key into its row, then one thread hands
// the whole tile to the TMA engine as a single bulk store (cp.async.bulk,
// shared to global).  The two tiles alternate, so encoding the next tile
// overlaps the store of the previous one, and each thread's next key is loaded
// a tile ahead.  10^6 rows of 150 bytes: 31.4 us before this fill, 30.4 now
// (5.4 TB/s; a plain fill of the output's bytes takes 43 us).
//
// At row widths that are multiples of 64 bytes a store of one character per
// row falls on one or two banks; there a warp encodes its 32 rows 32
// neighbouring characters at a time, from the keys in shared memory
// (encode_rows).  That is more instructions per character, so only there.
// 10^6 rows, one row per thread against by warp: 44.8 and 30.4 us at 64 bytes,
// 84.1 and 32.8 at 128, 87.6 and 53.5 at 256.  500,000 rows at 32 bytes: 13.8
// and 15.7, at 96 17.1 and 18.8, at 150 15.5 and above 20.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "pk_device.cuh"
#include "pk_internal.h"

namespace {

constexpr uint32_t kRows = 256;  // rows per tile; one thread per row
constexpr uint32_t kChars = PK_KEY_STRING_CHARS;
static_assert(PK_KEY_STRING_MAX_WIDTH <= kRows, "one thread per byte of a row");

struct KeyStrArgs {
    uint32_t plen;   // prefix bytes
    uint32_t width;  // row width in bytes, plen + 22 <= width <= PK_KEY_STRING_MAX_WIDTH
    uint32_t prefix[PK_KEY_STRING_MAX_WIDTH / 4];  // little-endian, zeros behind the prefix
};

// Character of a 6-bit value: 'A' + v with the gaps of ASCII between the alphabet's ranges.
__device__ __forceinline__ uint8_t b64_char(uint32_t v) {
    uint32_t c = 'A' + v;
    if (v > 25) c += 'a' - 'Z' - 1;
    if (v > 51) c -= 'z' - '0' + 1;
    if (v == 62) c = '+';
    if (v == 63) c = '/';
    return (uint8_t)c;
}

__device__ __forceinline__ uint32_t bswap32(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

// Bulk copy of `bytes` (a multiple of 16) from shared to global memory,
// tracked in this thread's bulk group.
__device__ __forceinline__ void bulk_store(void *gdst, const void *ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 :
                 : "l"(gdst), "r"((uint32_t)__cvta_generic_to_shared(ssrc)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// At most one bulk group of this thread still reading shared memory.
__device__ __forceinline__ void bulk_wait_read_1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// Every bulk group of this thread complete.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Shared-memory writes of this thread visible to the TMA engine (async proxy).
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void encode_row(const uint4 &k, uint8_t *c) {
    // The 16 bytes as a 128-bit big-endian integer (hi, lo); character q is
    // bits [6q, 6q + 6) counted from the most significant bit.
    const uint64_t hi = ((uint64_t)bswap32(k.x) << 32) | bswap32(k.y);
    const uint64_t lo = ((uint64_t)bswap32(k.z) << 32) | bswap32(k.w);
#pragma unroll
    for (uint32_t q = 0; q < kChars; ++q) {
        const uint32_t s = 6 * q;  // <= 126
        const uint64_t top = s == 0 ? hi : s < 64 ? (hi << s) | (lo >> (64 - s)) : lo << (s - 64);
        c[q] = b64_char((uint32_t)(top >> 58));
    }
}

// The characters of a warp's 32 rows (the first `rows` of them), 32 neighbouring ones at a time.  keys: the rows' key
// bytes in shared memory, kKeyStage apart, a zero byte after each; dst: the first row's first character.
constexpr uint32_t kKeyStage = 20;

__device__ __forceinline__ void encode_rows(const uint8_t *keys, uint8_t *dst, uint32_t width, uint32_t rows) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t row = lane >= kChars, c = lane - row * kChars;
#pragma unroll 2
    for (uint32_t it = 0; it < kChars; ++it) {
        // character c is bits [6c, 6c + 6) of the key, counted from the most significant bit of its first byte
        const uint8_t *k = keys + row * kKeyStage + (3 * c >> 2);
        const uint32_t v = ((uint32_t)k[0] << 8 | k[1]) >> (10 - (6 * c & 7)) & 63u;
        if (row < rows) dst[row * width + c] = b64_char(v);
        const bool wrap = c + 32 % kChars >= kChars;  // 32 characters on: one row and 10, or two rows
        row += wrap ? 2 : 1;
        c = wrap ? c + 32 % kChars - kChars : c + 32 % kChars;
    }
}

template <bool kByWarp>
__global__ void __launch_bounds__(kRows) k_key_strings(const uint8_t *keys, uint64_t n, KeyStrArgs a, uint8_t *out) {
    extern __shared__ __align__(128) uint8_t sm[];  // two tiles of kRows * width bytes
    __shared__ __align__(16) uint8_t stage[kByWarp ? kRows : 1][kKeyStage];
    const uint32_t t = threadIdx.x;
    const uint32_t tile_bytes = kRows * a.width;
    const uint64_t n_tiles = (n + kRows - 1) / kRows;
    // The tiles that this CTA uses, every row the prefix and zeros.
    const uint32_t units = a.width;  // 16-byte units of 16 rows
    if (t < a.width) {
        uint32_t w = 0;  // (a lookup by t would read the parameters one lane at a time)
        for (uint32_t q = 0; 4 * q < a.plen; ++q) w = q == t / 4 ? a.prefix[q] : w;
        const uint8_t b = (uint8_t)(w >> 8 * (t & 3));
#pragma unroll
        for (uint32_t r = 0; r < 16; ++r) sm[r * a.width + t] = b;
    }
    if (kByWarp) *reinterpret_cast<uint32_t *>(&stage[t][16]) = 0u;
    __syncthreads();
    {
        uint4 *sm4 = reinterpret_cast<uint4 *>(sm);
        const uint32_t all = (n_tiles > (uint64_t)blockIdx.x + gridDim.x ? 2u : 1u) * (tile_bytes / 16);
        const uint32_t step = kRows % units;
        uint32_t from = t % units;
        for (uint32_t i = units + t; i < all; i += kRows) {
            sm4[i] = sm4[from];
            from += step;
            if (from >= units) from -= units;
        }
    }
    pk::pdl_wait(keys, out);
    uint64_t tile = blockIdx.x;
    uint4 k = make_uint4(0, 0, 0, 0);
    if (tile * kRows + t < n) k = __ldcg(reinterpret_cast<const uint4 *>(keys + 32 * (tile * kRows + t)));
    for (uint32_t it = 0; tile < n_tiles; tile += gridDim.x, ++it) {
        uint8_t *buf = sm + (it & 1) * tile_bytes;
        const uint64_t row0 = tile * kRows;
        const uint32_t rows = (uint32_t)min((uint64_t)kRows, n - row0);
        const uint64_t next = row0 + (uint64_t)gridDim.x * kRows + t;  // this thread's key of the next tile
        uint4 k_next = make_uint4(0, 0, 0, 0);
        if (next < n) k_next = __ldcg(reinterpret_cast<const uint4 *>(keys + 32 * next));
        if (kByWarp) {
            uint32_t *st = reinterpret_cast<uint32_t *>(stage[t]);  // (4-byte stores: kKeyStage is no multiple of 16)
            st[0] = k.x;
            st[1] = k.y;
            st[2] = k.z;
            st[3] = k.w;
        }
        if (t == 0) bulk_wait_read_1();  // the store that last used `buf` has read it
        __syncthreads();
        if (kByWarp) {
            const uint32_t first = t & ~31u;
            if (first < rows) encode_rows(stage[first], buf + first * a.width + a.plen, a.width, rows - first);
        } else if (t < rows) {
            encode_row(k, buf + t * a.width + a.plen);
        }
        fence_proxy_async_smem();
        __syncthreads();
        const uint32_t bytes = rows * a.width;
        const uint32_t b16 = bytes & ~15u;
        uint8_t *dst = out + row0 * a.width;  // 16-byte aligned: 256 * width is a multiple of 16
        if (t == 0 && b16) bulk_store(dst, buf, b16);
        for (uint32_t j = b16 + t; j < bytes; j += kRows) dst[j] = buf[j];  // the last tile's final bytes
        k = k_next;
    }
    pk::pdl_launch_dependents();
    if (t == 0) bulk_wait_all();  // shared memory stays allocated until the TMA engine has read it
}

bool by_warp(uint32_t width) { return width % 64 == 0; }  // 16 or 32 rows of a warp on one bank

auto kernel_of(uint32_t width) { return by_warp(width) ? k_key_strings<true> : k_key_strings<false>; }

}  // namespace

// Resident CTAs of k_key_strings for a row width (SMs x CTAs per SM), computed
// once per device and width; the first call also raises the kernels' dynamic
// shared-memory limit to the largest width's two tiles.
static cudaError_t keystr_resident(int dev, uint32_t width, uint64_t *out) {
    static std::mutex mu;
    static uint32_t sms[256] = {};
    static uint16_t per_sm[256][PK_KEY_STRING_MAX_WIDTH + 1] = {};
    if (dev < 0 || dev >= 256 || width > PK_KEY_STRING_MAX_WIDTH) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (!sms[dev]) {
        int n = 0;
        cudaError_t e = cudaFuncSetAttribute(k_key_strings<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(2 * kRows * PK_KEY_STRING_MAX_WIDTH));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_key_strings<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(2 * kRows * PK_KEY_STRING_MAX_WIDTH));
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        sms[dev] = (uint32_t)n;
    }
    if (!per_sm[dev][width]) {
        int b = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel_of(width), kRows, 2ull * kRows * width);
        if (e != cudaSuccess) return e;
        per_sm[dev][width] = (uint16_t)(b < 1 ? 1 : b);
    }
    *out = (uint64_t)sms[dev] * per_sm[dev][width];
    return cudaSuccess;
}

cudaError_t pk_launch_key_strings(const uint8_t *keys, uint64_t n, const uint8_t *prefix, uint32_t plen,
                                  uint32_t width, uint8_t *out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    KeyStrArgs a;
    a.plen = plen;
    a.width = width;
    memset(a.prefix, 0, sizeof(a.prefix));
    for (uint32_t j = 0; j < plen; ++j) a.prefix[j / 4] |= (uint32_t)prefix[j] << 8 * (j % 4);
    const size_t smem = 2ull * kRows * width;  // <= 128 KiB
    int dev = 0;
    uint64_t resident = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = keystr_resident(dev, width, &resident);
    if (e != cudaSuccess) return e;
    const uint64_t tiles = (n + kRows - 1) / kRows;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles < resident ? tiles : resident));
    cfg.blockDim = dim3(kRows);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel_of(width), keys, n, a, out);
    return e != cudaSuccess ? e : cudaGetLastError();
}

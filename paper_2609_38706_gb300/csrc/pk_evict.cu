// pk_evict.cu -- eviction under a fixed budget (Sec. 6.5, eviction under a
// fixed budget: binding provenance keeps one copy per provenance, so a store
// of fixed size evicts more, and thrashes once the distinct working set
// exceeds it).
//
// Budget mode keeps a last-use stamp per table entry, (epoch << 32) | e:
// the store call's number and the key's index in that call, raised by every
// call that finds or inserts the key (pk_table.cu, examine).  Stamps of
// different entries differ, except the zero stamp of entries never used
// since the stamps were attached.  When the table holds more than `budget`
// entries, pk_evict keeps the entries whose stamp is above v, the (keep+1)-th
// largest stamp, and removes the rest: exactly the least recently used
// entries down to `keep`, the whole group of equal stamps when they tie.
//
// One cooperative launch, every CTA resident, in phases separated by
// bounded grid barriers:
//   1. every CTA reads the entry count and returns at once when it is within
//      the budget (the common step costs one short launch);
//   2. gather: one bit per entry (occupied), one byte with its distance from
//      home, the numbers of entries with and without a stamp, the range of
//      the stamps, and a histogram of their age in store calls
//      (an eviction replayed from a CUDA graph has the call number of its
//      capture: calls after that count as age 0);
//   3. the threshold v: the age histogram gives the call in which the last
//      entry to go was used; if every entry of that call and the calls before
//      it goes, v is known (a store that evicts whole batches, the common
//      case).  Otherwise the stamps of that call are split by their key
//      index, 8 bits per pass over the stamp array, until the entries to go
//      end with a bucket;
//   4. every position with a stamp <= v goes into an evicted bitmap and its
//      slot into the output (buffered in shared memory), and the table is
//      compacted in place, one thread per cluster (maximal run of occupied
//      entries, from the bitmap of phase 2): in probe order, an evicted entry
//      is cleared; a kept entry moves to the first empty position between its
//      home and its own, so that every kept key stays reachable by linear
//      probing.  Clusters are disjoint, so no two threads touch the same entry.
// Every phase but the last streams over the table or the stamps and is bound
// by loads in flight: two CTAs of 512 threads per SM, four positions per
// thread (a bulk prefetch into L2 of the next iteration changed nothing).
// 2^22 entries, 1.84 M stored, 262,144 evicted (one call's): 190 -> 86 us
// (gather 37, threshold 5, bitmap and slots 17, compaction 26), against
// compacting stamps and slots into a list, selecting over it in 5 passes and
// two more passes for the slots and the bitmap, with one CTA per SM.
// 2^14 entries, 512 of 5,120 evicted: 54 -> 18 us (before the parts of k_evict).
#include <cuda_runtime.h>

#include <mutex>

#include "pk_device.cuh"
#include "pk_internal.h"

namespace {

constexpr uint32_t kEvThreads = 512;
constexpr uint32_t kEvBlocks = 2;  // CTAs per SM
constexpr uint32_t kEvRows = 512;  // table entries per CTA below which no further CTA is launched
constexpr uint32_t kPasses = 7;    // histogram rows of the passes within a call, used in turn
constexpr uint32_t kSpinLimit = 1u << 23;  // polls of about 230 ns: a barrier gives up after about 2 s

struct EvictHeader {  // zeroed by the host before every launch
    unsigned int arrive;             // CTAs that have arrived at the grid barriers so far
    unsigned int unused;
    unsigned long long n_stamped;    // entries with a stamp
    unsigned long long n_unstamped;  // entries without (stamp 0)
    unsigned long long n_evicted;    // entries removed
    unsigned long long inv_min;      // ~(smallest non-zero stamp)
    unsigned long long max;          // largest stamp
    unsigned int max_index;          // largest key index (low half) of a stamp
    unsigned int age[256];           // stamped entries by age in calls, 255: that and older
    unsigned int hist[kPasses][256];
};
constexpr uint64_t kHeaderBytes = (sizeof(EvictHeader) + 255) & ~255ull;

uint64_t bitmap_bytes(uint64_t capacity) { return ((capacity + 31) / 32 * 4 + 255) & ~255ull; }

__device__ __forceinline__ bool is_zero(const uint4 &v) { return (v.x | v.y | v.z | v.w) == 0u; }

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The bound of a launch's barrier waits, and the CTA that withholds its
// arrival at the first barrier (none in a normal launch; the timeout test
// names one, so that the others' waits run out).
struct BarrierBound {
    uint32_t spin_limit;
    uint32_t withheld_cta;
};

// Grid-wide barrier number `k` (from 0) of the launch, with a bounded wait: a
// barrier is passed once (k + 1) x gridDim arrivals are counted, so that
// arriving and seeing the last arrival take one round trip to L2 each (a
// generation word read before and written after the count: 3.4 us a barrier
// of 32 CTAs instead of 1.7).  Returns false (in every thread of the CTA)
// when the wait gave up; the status word then holds PK_ERR_TIMEOUT.  A
// withheld CTA returns false without arriving.
__device__ bool grid_sync(EvictHeader *h, uint32_t k, int32_t *status, const BarrierBound &bb) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = blockIdx.x != bb.withheld_cta;
        if (ok) {
            __threadfence();
            atomicAdd(&h->arrive, 1u);
            const unsigned int all = (k + 1) * gridDim.x;
            uint32_t it = 0;
            while (ld_acquire(&h->arrive) < all) {
                if (++it > bb.spin_limit) {
                    ok = 0;
                    pk::set_status(status, PK_ERR_TIMEOUT);
                    break;
                }
                __nanosleep(20);
            }
            __threadfence();
        }
    }
    __syncthreads();
    return ok != 0;
}

constexpr uint32_t kPer = 4;  // elements per thread per iteration of the strided loops (loads in flight)
constexpr uint32_t kWarps = kEvThreads / 32;
constexpr uint32_t kSlotBuf = 512;  // slots of evicted entries that a warp collects before it writes them out

// The bucket of a 256-bin histogram (in global memory, complete) that holds ascending `rank`, by warp 0;
// every thread of the CTA calls it.  sel[0]: the bucket, sel[1]: the rank within it, sel[2]: its count.
__device__ __forceinline__ void pick_bucket(const unsigned int *hist, bool descending, unsigned long long rank,
                                            unsigned long long *sel) {
    const uint32_t lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {  // 8 buckets per lane, then a warp scan
        unsigned long long c[8], sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t b = lane * 8 + u;
            c[u] = __ldcg(hist + (descending ? 255 - b : b));
            sum += c[u];
        }
        unsigned long long incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        unsigned long long excl = incl - sum;
        if (rank >= excl && rank < incl) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (rank >= excl && rank < excl + c[u]) {
                    const uint32_t b = lane * 8 + u;
                    sel[0] = descending ? 255 - b : b;
                    sel[1] = rank - excl;
                    sel[2] = c[u];
                }
                excl += c[u];
            }
        }
    }
    __syncthreads();
}

// Shared-memory histogram increment of `bin` (256: none), one atomic per distinct bin of the warp.
__device__ __forceinline__ void count_bin(unsigned int *sh_hist, uint32_t bin) {
    const uint32_t peers = __match_any_sync(0xffffffffu, bin);
    if (bin < 256 && (peers & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicAdd(&sh_hist[bin], __popc(peers));
}

__device__ __forceinline__ bool bit(const uint32_t *bm, uint64_t i) { return (__ldcg(bm + (i >> 5)) >> (i & 31)) & 1u; }

// Length of the run of occupied positions (bitmap) starting at s, wrapping
// around the table; at most `capacity`.
__device__ uint64_t run_length(const uint32_t *bitmap, uint64_t s, uint64_t capacity) {
    uint64_t L = 0, p = s;
    while (L < capacity) {
        const uint32_t off = (uint32_t)(p & 31);
        const uint64_t left = min((uint64_t)(32 - off), capacity - p);  // valid bits of this word from p
        const uint32_t wd = __ldcg(bitmap + (p >> 5)) >> off;
        const uint32_t ones = (uint32_t)min((uint64_t)(__ffs(~wd) ? __ffs(~wd) - 1 : 32), left);
        L += ones;
        if (ones < left) break;
        p = (p + ones) & (capacity - 1);
    }
    return L < capacity ? L : capacity;
}

// Compaction of one cluster by one thread, serial form: in probe order an
// evicted entry is cleared, a kept entry moves to the first empty position
// from its home.  Any length; used for clusters longer than kPlanMax.
__device__ __noinline__ void compact_walk(pk_entry *table, unsigned long long *stamps, uint64_t s, uint64_t L, uint64_t mask,
                             unsigned long long v) {
    for (uint64_t step = 0; step < L; ++step) {
        const uint64_t pos = (s + step) & mask;
        uint4 *ep = reinterpret_cast<uint4 *>(&table[pos]);
        const uint4 k = __ldcg(ep), meta = __ldcg(ep + 1);
        const unsigned long long sp = __ldcg(stamps + pos);
        if (sp <= v) {
            __stcg(ep, make_uint4(0, 0, 0, 0));
            __stcg(ep + 1, make_uint4(0, 0, 0, 0));
            __stcg(stamps + pos, 0ull);
            continue;
        }
        const uint64_t home = (((uint64_t)k.y << 32) | k.x) & mask;
        const uint64_t dist = (pos - home) & mask;
        for (uint64_t q = 0; q < dist; ++q) {
            const uint64_t t = (home + q) & mask;
            uint4 *tp = reinterpret_cast<uint4 *>(&table[t]);
            if (is_zero(__ldcg(tp))) {  // first empty position from the home: move there
                __stcg(tp + 1, meta);
                __stcg(tp, k);
                __stcg(stamps + t, sp);
                __stcg(ep, make_uint4(0, 0, 0, 0));
                __stcg(ep + 1, make_uint4(0, 0, 0, 0));
                __stcg(stamps + pos, 0ull);
                break;
            }
        }
    }
}

// Pending moves of one thread, flushed four at a time: the sources' entries
// and stamps are all loaded before any target is stored.  Sources come in
// ascending order and every target lies below its source, so no source is
// overwritten before it is read.
struct MoveRing {
    uint32_t src[4], dst[4];  // positions relative to the cluster start
    uint32_t n = 0;
    __device__ __forceinline__ void flush(pk_entry *table, unsigned long long *stamps, uint64_t s0, uint64_t mask) {
        uint4 kk[4], mm[4];
        unsigned long long ss[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            if (u < n) {
                const uint64_t pos = (s0 + src[u]) & mask;
                const uint4 *ep = reinterpret_cast<const uint4 *>(&table[pos]);
                kk[u] = __ldcg(ep);
                mm[u] = __ldcg(ep + 1);
                ss[u] = __ldcg(stamps + pos);
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            if (u < n) {
                const uint64_t t = (s0 + dst[u]) & mask;
                uint4 *tp = reinterpret_cast<uint4 *>(&table[t]);
                __stcg(tp + 1, mm[u]);
                __stcg(tp, kk[u]);
                __stcg(stamps + t, ss[u]);
            }
        }
        n = 0;
    }
};

constexpr uint32_t kPlanMax = 1024;  // longest cluster compact_planned takes

// Compaction of one cluster of L <= kPlanMax entries starting at table
// position s0 (capacity >= 64), planned as in k_evict's window: kept entries in
// probe order take the first free position at or after their home, from the
// evicted bits and distance bytes, 32 positions at a time.  A saturated
// distance (255) is replaced by the exact one, from the entry's key.
__device__ __noinline__ void compact_planned(pk_entry *table, unsigned long long *stamps, const uint32_t *evbm, const uint8_t *dist,
                                uint64_t s0, uint32_t L, uint64_t mask) {
    uint64_t taken[kPlanMax / 64];
    for (uint32_t q = 0; q < kPlanMax / 64; ++q) taken[q] = 0;
    const uint64_t n_words = (mask + 1) / 32;
    MoveRing ring;
    for (uint32_t c = 0; c < L; c += 32) {
        const uint64_t p0 = (s0 + c) & mask;
        const uint32_t off = (uint32_t)(p0 & 31);
        const uint64_t wi = p0 >> 5;
        uint32_t evb = __ldcg(evbm + wi) >> off;
        if (off) evb |= __ldcg(evbm + (wi + 1) % n_words) << (32 - off);
        uint8_t d[32];
#pragma unroll
        for (uint32_t k = 0; k < 32; ++k) d[k] = __ldcg(dist + ((p0 + k) & mask));
        for (uint32_t k = 0; k < 32 && c + k < L; ++k) {
            const uint32_t j = c + k;
            if ((evb >> k) & 1u) continue;
            uint64_t dd = d[k];
            if (dd == 255) {  // saturated: the exact distance from the key (position j is not yet overwritten)
                const uint64_t pos = (s0 + j) & mask;
                const uint4 kj = __ldcg(reinterpret_cast<const uint4 *>(table[pos].k));
                dd = (pos - ((((uint64_t)kj.y << 32) | kj.x) & mask)) & mask;
            }
            const uint32_t hh = dd <= j ? j - (uint32_t)dd : j;
            uint32_t t = j;  // position j itself is free
            for (uint32_t q = hh >> 6; q <= (j >> 6); ++q) {
                uint64_t fr = ~taken[q];
                if (q == (hh >> 6)) fr &= ~0ull << (hh & 63);
                if (fr) {
                    t = q * 64 + __ffsll((long long)fr) - 1;
                    break;
                }
            }
            taken[t >> 6] |= 1ull << (t & 63);
            if (t != j) {
                ring.src[ring.n] = j;
                ring.dst[ring.n] = t;
                if (++ring.n == 4) ring.flush(table, stamps, s0, mask);
            }
        }
    }
    ring.flush(table, stamps, s0, mask);
    for (uint32_t q = 0; q * 64 < L; ++q) {  // positions left empty
        uint64_t z = ~taken[q];
        if (L - q * 64 < 64) z &= (1ull << (L - q * 64)) - 1ull;
        while (z) {
            const uint32_t p = q * 64 + __ffsll((long long)z) - 1;
            z &= z - 1;
            const uint64_t pos = (s0 + p) & mask;
            uint4 *ep = reinterpret_cast<uint4 *>(&table[pos]);
            __stcg(ep, make_uint4(0, 0, 0, 0));
            __stcg(ep + 1, make_uint4(0, 0, 0, 0));
            __stcg(stamps + pos, 0ull);
        }
    }
}

// kParts: 2^parts_log2 threads share a bitmap word in the compaction, each for the clusters that start in its part.  A
// thread's moves follow one another, loads and stores in turn, so it pays where the grid has threads to spare.
// The call between two events, without and with parts, in us: 2^20 entries, 600,000 kept, 60,000 evicted 106 and 91 (2
// parts); 2^18, 64,000 and 16,000, 50 and 45 (8); 2^16, 12,000 and 3,000, 32 and 26; 2^14, 4,800 and 800, 29 and 22;
// 2^14, 12,000 and 3,000 (long clusters) 293 and 219.  A step of 64 requests under a budget with 512 evictions (2^14):
// 77.5 and 71.5.  2^21 entries with two parts: 200,000 evicted of 1,000,000 91 and 86, but 100,000 of 700,000 68 and 72.
// A table that uses most of the grid takes the other form, which is the code without parts (with them 2^22 entries,
// one part per word, churn of 262,144 keys 173.0 -> 177.5 us).
template <bool kParts>
__global__ void __launch_bounds__(kEvThreads, kEvBlocks)
k_evict(pk_entry *table, unsigned long long *stamps, uint64_t capacity, unsigned long long *counter, uint64_t budget,
        uint64_t keep, unsigned long long epoch, EvictHeader *h, uint32_t *bitmap, uint32_t *evbm, uint8_t *dist,
        uint32_t *evicted, uint64_t evicted_cap, unsigned long long *n_evicted_out, int32_t *status, BarrierBound bb,
        uint32_t parts_log2) {
    __shared__ unsigned int sh_hist[256];
    __shared__ unsigned long long sh_sel[3];
    __shared__ unsigned long long sh_count[2];
    __shared__ unsigned long long sh_base;
    __shared__ uint32_t sh_at[kWarps + 1];
    __shared__ uint32_t sh_slots[kWarps][kSlotBuf];
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + tid;
    const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t mask = capacity - 1;
    const uint32_t kFull = 0xffffffffu;
    // grid-uniform strided loops: an iteration covers kPer positions per thread, one per pass of the grid
    const uint64_t span = nthreads * kPer;

    // 1. within the budget: nothing to do
    const unsigned long long count = __ldcg(counter);
    if (count <= budget) {
        if (gtid == 0 && n_evicted_out) *n_evicted_out = 0;
        return;
    }
    const bool by_age = epoch >> 32 == 0;  // (a stamp holds 32 bits of its call's number)
    if (tid < 256) sh_hist[tid] = 0;
    if (tid < 2) sh_count[tid] = 0;
    __syncthreads();

    // 2. gather: occupancy bitmap, distances, counts, stamp range, age histogram
    unsigned long long lo = ~0ull, hi = 0;
    uint32_t max_index = 0, stamped = 0, unstamped = 0;
    for (uint64_t base = 0; base < capacity; base += span) {
        uint4 k[kPer];
        unsigned long long st[kPer];
#pragma unroll
        for (uint32_t u = 0; u < kPer; ++u) {  // every load of the iteration at once (empty entries: stamp 0)
            const uint64_t i = base + u * nthreads + gtid;
            k[u] = make_uint4(0, 0, 0, 0);
            st[u] = 0;
            if (i < capacity) {
                k[u] = __ldcg(reinterpret_cast<const uint4 *>(&table[i]));
                st[u] = __ldcg(stamps + i);
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < kPer; ++u) {
            const uint64_t i = base + u * nthreads + gtid;
            const bool occ = !is_zero(k[u]);
            const uint32_t word = __ballot_sync(kFull, occ);
            if (lane == 0 && i < capacity) bitmap[i >> 5] = word;
            if (i < capacity) {  // distance from the home position, saturated at 255
                const uint64_t d = (i - ((((uint64_t)k[u].y << 32) | k[u].x) & mask)) & mask;
                dist[i] = occ ? (uint8_t)(d < 255 ? d : 255) : (uint8_t)0;
            }
            uint32_t bin = 256;
            if (occ && st[u]) {
                const unsigned long long call = st[u] >> 32, age = call < epoch ? epoch - call : 0ull;
                bin = by_age && age < 255 ? (uint32_t)age : 255u;
                ++stamped;
                lo = st[u] < lo ? st[u] : lo;
                hi = st[u] > hi ? st[u] : hi;
                max_index = (uint32_t)st[u] > max_index ? (uint32_t)st[u] : max_index;
            } else if (occ) {
                ++unstamped;
            }
            count_bin(sh_hist, bin);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l2 = __shfl_xor_sync(kFull, lo, o), h2 = __shfl_xor_sync(kFull, hi, o);
        lo = l2 < lo ? l2 : lo;
        hi = h2 > hi ? h2 : hi;
    }
    max_index = __reduce_max_sync(kFull, max_index);
    stamped = __reduce_add_sync(kFull, stamped);
    unstamped = __reduce_add_sync(kFull, unstamped);
    if (lane == 0) {
        if (stamped) {
            atomicMax(&h->inv_min, ~lo);
            atomicMax(&h->max, hi);
            atomicMax(&h->max_index, max_index);
            atomicAdd_block(&sh_count[0], (unsigned long long)stamped);
        }
        if (unstamped) atomicAdd_block(&sh_count[1], (unsigned long long)unstamped);
    }
    __syncthreads();
    if (tid < 256 && sh_hist[tid]) atomicAdd(&h->age[tid], sh_hist[tid]);
    if (tid == 0 && sh_count[0]) atomicAdd(&h->n_stamped, sh_count[0]);
    if (tid == 0 && sh_count[1]) atomicAdd(&h->n_unstamped, sh_count[1]);
    uint32_t barrier = 0;
    if (!grid_sync(h, barrier++, status, bb)) return;
    if (tid == 0) sh_count[0] = 0;  // from here: entries this CTA has removed
    __syncthreads();

    const unsigned long long n0 = __ldcg(&h->n_unstamped), n = n0 + __ldcg(&h->n_stamped);
    unsigned long long v = 0;  // every stamp <= v goes (0: the entries without a stamp, as one group)
    if (n > keep) {
        // 3. v, from the ascending rank n - keep - 1 of the last stamp to go
        if (n - keep > n0) {
            const unsigned long long smin = ~__ldcg(&h->inv_min), smax = __ldcg(&h->max);
            pick_bucket(h->age, true, n - keep - 1 - n0, sh_sel);  // oldest first
            const unsigned long long age = sh_sel[0];
            unsigned long long rank = sh_sel[1], left = sh_sel[2];
            // the candidates' range [clo, chi] (age 0: the call `epoch` and the calls after it)
            unsigned long long clo = age < 255 ? (epoch - age) << 32 : 0ull;
            unsigned long long chi = age == 0 ? smax
                                     : age < 255 ? clo | __ldcg(&h->max_index)
                                     : by_age    ? ((epoch - 254) << 32) - 1
                                                 : ~0ull;
            clo = clo > smin ? clo : smin;
            chi = chi < smax ? chi : smax;
            __syncthreads();
            for (uint32_t p = 0; rank + 1 < left && clo < chi; ++p) {  // the bucket goes only in part: split it
                const int bits = 64 - __clzll((long long)(chi - clo));
                const int shift = bits > 8 ? bits - 8 : 0;
                unsigned int *hist = h->hist[p % kPasses];
                if (tid < 256) sh_hist[tid] = 0;
                __syncthreads();
                for (uint64_t base = 0; base < capacity; base += span) {
                    unsigned long long x[kPer];
#pragma unroll
                    for (uint32_t u = 0; u < kPer; ++u) {
                        const uint64_t i = base + u * nthreads + gtid;
                        x[u] = i < capacity ? __ldcg(stamps + i) : 0ull;
                    }
#pragma unroll
                    for (uint32_t u = 0; u < kPer; ++u)  // (stamps of the candidates are not zero: clo >= smin)
                        count_bin(sh_hist, x[u] >= clo && x[u] <= chi ? (uint32_t)((x[u] - clo) >> shift) : 256u);
                }
                __syncthreads();
                if (tid < 256 && sh_hist[tid]) atomicAdd(&hist[tid], sh_hist[tid]);
                if (!grid_sync(h, barrier++, status, bb)) return;
                pick_bucket(hist, false, rank, sh_sel);
                clo += sh_sel[0] << shift;
                const unsigned long long top = clo + ((1ull << shift) - 1);
                chi = top < chi ? top : chi;
                rank = sh_sel[1];
                left = sh_sel[2];
                // a row is used again kPasses passes later: cleared two barriers before that, when every CTA has read it
                if (p + 2 >= kPasses && blockIdx.x == 0 && tid < 256) h->hist[(p + 2) % kPasses][tid] = 0;
                __syncthreads();
            }
            v = chi;
        }

        // 4a. the evicted positions as a bitmap, and their slots, collected per warp in shared memory
        const uint32_t warp = tid >> 5;
        unsigned long long removed = 0;
        uint32_t have = 0;  // slots in this warp's buffer
        auto put = [&](unsigned long long first) {  // the warp's buffer to evicted[first ..)
            __syncwarp();
            for (uint32_t j = lane; j < have; j += 32) {
                if (first + j < evicted_cap) evicted[first + j] = sh_slots[warp][j];
                else if (evicted) pk::set_status(status, PK_ERR_ARG);
            }
            __syncwarp();
        };
        for (uint64_t base = 0; base < capacity; base += span) {
            unsigned long long st[kPer];
            uint32_t wd[kPer], sl[kPer];
            bool ev[kPer];
#pragma unroll
            for (uint32_t u = 0; u < kPer; ++u) {
                const uint64_t i = base + u * nthreads + gtid;
                st[u] = i < capacity ? __ldcg(stamps + i) : ~0ull;
                wd[u] = i < capacity ? __ldcg(bitmap + (i >> 5)) : 0u;
            }
#pragma unroll
            for (uint32_t u = 0; u < kPer; ++u) {
                const uint64_t i = base + u * nthreads + gtid;
                ev[u] = ((wd[u] >> lane) & 1u) && st[u] <= v;
                sl[u] = ev[u] ? __ldcg(&table[i].slot) : 0u;
            }
#pragma unroll
            for (uint32_t u = 0; u < kPer; ++u) {
                const uint64_t i = base + u * nthreads + gtid;
                const uint32_t word = __ballot_sync(kFull, ev[u]);
                if (lane == 0 && i < capacity) evbm[i >> 5] = word;
                if (ev[u]) sh_slots[warp][have + __popc(word & ((1u << lane) - 1u))] = sl[u];
                have += __popc(word);
            }
            if (have + 32 * kPer > kSlotBuf) {  // the next iteration may not fit
                unsigned long long first = 0;
                if (lane == 0) first = atomicAdd(&h->n_evicted, (unsigned long long)have);
                put(__shfl_sync(kFull, first, 0));
                removed += have;
                have = 0;
            }
        }
        // what is left in the buffers: one atomic per CTA
        if (lane == 0) sh_at[warp] = have;
        if (lane == 0 && removed) atomicAdd_block(&sh_count[0], removed);
        __syncthreads();
        if (tid == 0) {
            uint32_t total = 0;
            for (uint32_t u = 0; u < kWarps; ++u) {
                const uint32_t x = sh_at[u];
                sh_at[u] = total;
                total += x;
            }
            sh_base = total ? atomicAdd(&h->n_evicted, (unsigned long long)total) : 0ull;
            const unsigned long long gone = sh_count[0] + total;
            if (gone) atomicAdd(counter, (unsigned long long)(-(long long)gone));
        }
        __syncthreads();
        put(sh_base + sh_at[warp]);
    }
    if (!grid_sync(h, barrier++, status, bb)) return;
    if (gtid == 0 && n_evicted_out) *n_evicted_out = __ldcg(&h->n_evicted);
    if (n > keep) {
        // 4b. compaction: one thread per bitmap word or part of one, for the clusters that start in it and lose an entry.  Clusters
        // that end within the 64 positions of the word and the next one are planned in registers
        // from the occupancy, evicted and distance bytes; the word's moves then go out four loads
        // at a time.  Longer clusters take compact_planned (the same plan, 32 positions at a time),
        // tables below 64 entries and clusters beyond kPlanMax compact_walk.
        const uint64_t n_words = (capacity + 31) / 32;
        // 32 neighbouring words, or parts of words (kParts), per warp, the warps in turn over the CTAs (a small table's
        // words spread over the SMs)
        const uint64_t x = ((uint64_t)(tid >> 5) * gridDim.x + blockIdx.x) * 32 + lane;
        const uint32_t log2 = kParts ? parts_log2 : 0;
        const uint32_t part = (0xffffffffu >> (32u - (32u >> log2))) << (((uint32_t)x & ((1u << log2) - 1u)) << (5 - log2));
        for (uint64_t w = x >> log2; w < n_words; w += nthreads) {
            const uint32_t occ_lo = __ldcg(bitmap + w);
            if (!occ_lo) continue;
            const uint32_t before = bit(bitmap, (w * 32 + mask) & mask);  // the position before bit 0
            uint32_t starts = occ_lo & ~((occ_lo << 1) | before);
            if (kParts) {
                starts &= part;
                if (!starts) continue;
            }
            if (capacity < 64) {
                while (starts) {
                    const uint32_t b = __ffs(starts) - 1;
                    starts &= starts - 1;
                    compact_walk(table, stamps, w * 32 + b, run_length(bitmap, w * 32 + b, capacity), mask, v);
                }
                continue;
            }
            const uint64_t w1 = (w + 1) % n_words;  // the next word (wrapping)
            const uint64_t occ = occ_lo | ((uint64_t)__ldcg(bitmap + w1) << 32);
            const uint64_t evw = __ldcg(evbm + w) | ((uint64_t)__ldcg(evbm + w1) << 32);
            if (!evw && (~occ >> 32)) continue;  // nothing goes in the window, and no cluster of it leaves the window
            uint32_t dv[16];
            {
                const uint4 *d0 = reinterpret_cast<const uint4 *>(dist + w * 32);
                const uint4 *d1 = reinterpret_cast<const uint4 *>(dist + w1 * 32);
                const uint4 a0 = __ldcg(d0), a1 = __ldcg(d0 + 1), b0 = __ldcg(d1), b1 = __ldcg(d1 + 1);
                dv[0] = a0.x, dv[1] = a0.y, dv[2] = a0.z, dv[3] = a0.w, dv[4] = a1.x, dv[5] = a1.y, dv[6] = a1.z;
                dv[7] = a1.w, dv[8] = b0.x, dv[9] = b0.y, dv[10] = b0.z, dv[11] = b0.w, dv[12] = b1.x;
                dv[13] = b1.y, dv[14] = b1.z, dv[15] = b1.w;
            }
            // window position p (0..63) is table position (w * 32 + p) & mask
            uint64_t zero = 0, msrc = 0;
            uint8_t dst_of[64];
            while (starts) {
                const uint32_t b = __ffs(starts) - 1;
                starts &= starts - 1;
                const uint64_t rest = ~(occ >> b);
                const uint32_t run = rest ? __ffsll((long long)rest) - 1 : 64 - b;
                if (b + run < 64) {  // the cluster ends inside the window
                    if (!((evw >> b) & ((1ull << run) - 1ull))) continue;  // and keeps every entry
                    uint64_t taken = 0;  // relative to b
                    for (uint32_t j = 0; j < run; ++j) {
                        const uint32_t p = b + j;
                        if ((evw >> p) & 1u) continue;
                        const uint32_t d = (dv[p >> 2] >> (8 * (p & 3))) & 255u;
                        const uint32_t hh = d <= j ? j - d : j;
                        const uint32_t t = __ffsll((long long)(~taken & (~0ull << hh))) - 1;
                        taken |= 1ull << t;
                        if (t != j) {
                            msrc |= 1ull << p;
                            dst_of[p] = (uint8_t)(b + t);
                        }
                    }
                    zero |= (((1ull << run) - 1ull) & ~taken) << b;
                } else {  // a longer cluster
                    const uint64_t L = run_length(bitmap, w * 32 + b, capacity);
                    if (L <= kPlanMax)
                        compact_planned(table, stamps, evbm, dist, w * 32 + b, (uint32_t)L, mask);
                    else
                        compact_walk(table, stamps, w * 32 + b, L, mask, v);
                }
            }
            // moves in ascending order, four loads before their stores: a target is below its
            // source, so every source is read before anything overwrites it
            while (msrc) {
                uint32_t src[4];
                uint4 kk[4], mm[4];
                unsigned long long ss[4];
                uint32_t cnt = 0;
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                    if (msrc) {
                        src[u] = __ffsll((long long)msrc) - 1;
                        msrc &= msrc - 1;
                        const uint64_t pos = (w * 32 + src[u]) & mask;
                        const uint4 *ep = reinterpret_cast<const uint4 *>(&table[pos]);
                        kk[u] = __ldcg(ep);
                        mm[u] = __ldcg(ep + 1);
                        ss[u] = __ldcg(stamps + pos);
                        cnt = u + 1;
                    }
                }
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                    if (u < cnt) {
                        const uint64_t t = (w * 32 + dst_of[src[u]]) & mask;
                        uint4 *tp = reinterpret_cast<uint4 *>(&table[t]);
                        __stcg(tp + 1, mm[u]);
                        __stcg(tp, kk[u]);
                        __stcg(stamps + t, ss[u]);
                    }
                }
            }
            while (zero) {  // positions left empty: evicted, or vacated and not retaken
                const uint32_t p = __ffsll((long long)zero) - 1;
                zero &= zero - 1;
                const uint64_t pos = (w * 32 + p) & mask;
                uint4 *ep = reinterpret_cast<uint4 *>(&table[pos]);
                __stcg(ep, make_uint4(0, 0, 0, 0));
                __stcg(ep + 1, make_uint4(0, 0, 0, 0));
                __stcg(stamps + pos, 0ull);
            }
        }
    }
}

}  // namespace

// (12 bytes per entry, once a list of stamps and slots, are not used: the size that callers allocate by is kept)
uint64_t pk_evict_scratch_bytes_impl(uint64_t capacity) {
    return kHeaderBytes + 2 * bitmap_bytes(capacity) + 8 * capacity + 4 * capacity + ((capacity + 255) & ~255ull);
}

// Resident CTAs of k_evict on a device, in either form (SMs x CTAs per SM), computed once per device.
static cudaError_t evict_resident(int dev, uint64_t *out) {
    static std::mutex mu;
    static uint64_t cache[256] = {};
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!cache[dev]) {
        int sms = 0, per_sm = 0, with_parts = 0;
        cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_evict<false>, kEvThreads, 0);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&with_parts, k_evict<true>, kEvThreads, 0);
        if (e != cudaSuccess) return e;
        if (with_parts < per_sm) per_sm = with_parts;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        cache[dev] = (uint64_t)sms * per_sm;
    }
    *out = cache[dev];
    return cudaSuccess;
}

cudaError_t pk_launch_evict(const pk_ctx *ctx, uint64_t budget, uint64_t keep, void *scratch, uint32_t *evicted,
                            uint64_t evicted_cap, unsigned long long *n_evicted, int32_t *status, cudaStream_t s,
                            uint32_t spin_limit, bool withhold_first_cta) {
    int dev = 0;
    uint64_t resident = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = evict_resident(dev, &resident);
    if (e != cudaSuccess) return e;
    // every CTA resident (the barriers need it); no more CTAs than the table has rows of kEvRows entries
    const uint64_t want = (ctx->capacity + kEvRows - 1) / kEvRows;
    const unsigned grid = (unsigned)(want < resident ? want : resident);
    uint8_t *base = static_cast<uint8_t *>(scratch);
    EvictHeader *h = reinterpret_cast<EvictHeader *>(base);
    uint32_t *bitmap = reinterpret_cast<uint32_t *>(base + kHeaderBytes);
    const uint64_t bmb = bitmap_bytes(ctx->capacity);
    uint32_t *evbm = reinterpret_cast<uint32_t *>(base + kHeaderBytes + bmb);
    uint8_t *dist = base + kHeaderBytes + 2 * bmb;
    e = cudaMemsetAsync(h, 0, sizeof(EvictHeader), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kEvThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const BarrierBound bb{spin_limit == 0 || spin_limit > kSpinLimit ? kSpinLimit : spin_limit,
                          withhold_first_cta ? 0u : 0xffffffffu};
    // At least half of the threads stay without a part, so a thread has one at most.
    const uint64_t n_words = (ctx->capacity + 31) / 32, threads = (uint64_t)grid * kEvThreads;
    uint32_t parts_log2 = 0;
    while (parts_log2 < 3 && n_words << (parts_log2 + 2) <= threads) ++parts_log2;
    e = cudaLaunchKernelEx(&cfg, parts_log2 ? k_evict<true> : k_evict<false>, ctx->table, ctx->stamps, ctx->capacity,
                           ctx->counter_dev, budget, keep, ctx->epoch, h, bitmap, evbm, dist, evicted, evicted_cap,
                           n_evicted, status, bb, parts_log2);
    return e != cudaSuccess ? e : cudaGetLastError();
}

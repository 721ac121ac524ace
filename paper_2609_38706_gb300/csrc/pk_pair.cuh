// pk_pair.cuh -- SHA-256 of independent messages by pairs of warps, for
// launches of few messages.
//
// A pair serves 16 messages with two lanes each (split rounds and schedule of
// pk_sha256.cuh): the schedule warp loads the message words a block ahead and
// writes K_t + W_t of each block to a two-deep ring in shared memory, the
// rounds warp runs the 64 rounds.  Nothing flows back but the ring's empty
// marks, so the schedule stays ahead and a block costs the rounds alone.
//
// With few messages the SM sub-partitions have room and a message's serial
// blocks set the time: one lane per message, schedule in the same thread,
// takes a lone warp 2719 to 2926 cycles per 64-byte block by the form of its
// additions, a pair alone on its SM 1793, each of two pairs 2204, of three 2414
// (their schedule warps share a sub-partition).
// A CTA holds up to three pairs, their rounds warps (0, 1, 2) on a
// sub-partition each and their schedule warps (3, 7, 11) on the fourth; warps
// 4-6 and 8-10 do nothing.  Beyond 48 messages per SM the pairs would share
// sub-partitions and one lane per message is faster.
#pragma once
#include <stdint.h>

#include "pk_sha256.cuh"

namespace pk {

constexpr int kPairMsgs = 16;                     // messages per pair
constexpr int kPairs = 3;                         // pairs per CTA
constexpr int kPairThreads = 384;
constexpr uint32_t kPairMsgsPerSm = kPairMsgs * kPairs;

// A message's K+W row: its 32 even words, then (kPairOdd) its 32 odd ones, as 16-byte vectors; the strides put the
// vectors of a quarter warp on distinct banks on either side.
constexpr int kPairOdd = 36;
constexpr int kPairRow = 72;

__device__ __forceinline__ void pair_bar_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void pair_bar_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// K+W of rounds 16s .. 16s + 15 of a row
__device__ __forceinline__ void pair_ld16(uint32_t k[16], const uint32_t *row, int s) {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const uint4 y = *reinterpret_cast<const uint4 *>(row + kPairOdd * par + 8 * s + 4 * m);
            k[8 * m + par] = y.x;
            k[8 * m + 2 + par] = y.y;
            k[8 * m + 4 + par] = y.z;
            k[8 * m + 6 + par] = y.w;
        }
    }
}

struct PairRing {
    uint32_t kw[2][kPairMsgs][kPairRow];
};
struct PairSmem {
    PairRing ring[kPairs];
    uint32_t zero[kPairRow];  // the odd lanes' K+W
    uint32_t pad[kPairRow];   // K+W of the constant last block
    uint32_t kpar[2][32];     // K of the even and of the odd t
};

// Role of a warp: which pair, and which half of it (pair >= kPairs: none).
struct PairRole {
    uint32_t pair;
    bool sched;
};
__device__ __forceinline__ PairRole pair_role() {
    const uint32_t warp = threadIdx.x >> 5;
    const bool sched = (warp & 3) == 3;
    return PairRole{sched ? warp >> 2 : warp, sched};
}

// The CTA's constant rows (all threads; a __syncthreads must follow).
__device__ __forceinline__ void pair_tables(PairSmem &sm, const uint32_t *pad_kw) {
    for (uint32_t t = threadIdx.x; t < 64; t += kPairThreads) {
        sm.kpar[t & 1][t >> 1] = kSha256K[t];
        sm.pad[kPairOdd * (t & 1) + (t >> 1)] = pad_kw[t];
    }
    for (uint32_t t = threadIdx.x; t < kPairRow; t += kPairThreads) sm.zero[t] = 0u;
}

// Named barriers of pair p: 1 + 4p, 2 + 4p a ring stage filled, 3 + 4p, 4 + 4p a stage read.  Of the kernels that use
// the pairs, the warps without a part release the successor at once, which becomes resident as far as the pairs leave
// room and waits there.
//
// Schedule warp: K+W of `blocks` blocks.  src.load(b, t) is word t (0..15) of
// block b of this lane's message in memory (0 past its last whole word;
// src.tail, src.tail_word: the bytes after that), src.word(b, t, x)
// the big-endian message word made of it (when the load has arrived, a block
// later); src.inside(b): every word of the block can be read at src.block(b),
// plain loads that all stay in flight.  The even lane of a message takes
// words 2i and 2i + 1 (own, far), the odd lane 2i + 1 and 2i + 2.
template <typename Src>
__device__ __forceinline__ void pair_schedule(PairSmem &sm, uint32_t pair, const SplitLane &l, uint32_t blocks, Src src) {
    const uint32_t lane = threadIdx.x & 31, q = lane >> 1, par = lane & 1;
    const int bar = 1 + 4 * (int)pair;
    uint32_t raw_own[8], raw_far[7], own[8], far[8];
    auto load = [&](uint32_t b) {
        if (__all_sync(0xffffffffu, src.inside(b))) {
            const uint32_t *p = src.block(b) + par;
#pragma unroll
            for (int i = 0; i < 8; ++i) raw_own[i] = __ldcg(p + 2 * i);
#pragma unroll
            for (int i = 0; i < 7; ++i) raw_far[i] = __ldcg(p + 2 * i + 1);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) raw_own[i] = src.load(b, 2 * i + par);
#pragma unroll
            for (int i = 0; i < 7; ++i) raw_far[i] = src.load(b, 2 * i + 1 + par);
            const int tail = src.tail(b);  // the word that the message ends inside of, else -1
            if (__any_sync(0xffffffffu, tail >= 0)) {
                const uint32_t x = tail >= 0 ? src.tail_word(b) : 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (tail == 2 * i + (int)par) raw_own[i] = x;
#pragma unroll
                for (int i = 0; i < 7; ++i)
                    if (tail == 2 * i + 1 + (int)par) raw_far[i] = x;
            }
        }
    };
    if (blocks) load(0);
#pragma unroll 1
    for (uint32_t b = 0; b < blocks; ++b) {
#pragma unroll
        for (int i = 0; i < 8; ++i) own[i] = src.word(b, 2 * i + par, raw_own[i]);
#pragma unroll
        for (int i = 0; i < 7; ++i) far[i] = src.word(b, 2 * i + 1 + par, raw_far[i]);
        far[7] = 0u;  // (delivered by the first step of split_sched8)
        if (b + 1 < blocks) load(b + 1);
        if (b >= 2) pair_bar_sync(bar + 2 + (int)(b & 1));
        uint4 *o = reinterpret_cast<uint4 *>(sm.ring[pair].kw[b & 1][q] + kPairOdd * par);
        const uint4 *kp = reinterpret_cast<const uint4 *>(sm.kpar[par]);
#pragma unroll 1
        for (int s = 0; s < 4; ++s) {
            if (s) split_sched8(own, far, l);
            const uint4 ka = kp[2 * s], kb = kp[2 * s + 1];
            o[2 * s] = make_uint4(own[0] + ka.x, own[1] + ka.y, own[2] + ka.z, own[3] + ka.w);
            o[2 * s + 1] = make_uint4(own[4] + kb.x, own[5] + kb.y, own[6] + kb.z, own[7] + kb.w);
        }
        pair_bar_arrive(bar + (int)(b & 1));
    }
}

// Rounds warp: `blocks` blocks from the ring, then (pad) the constant last block.  st: the digest, words 4..7 in the
// even lane, 0..3 in the odd lane.
__device__ __forceinline__ void pair_rounds(PairSmem &sm, uint32_t pair, const SplitLane &l, uint32_t blocks, bool pad,
                                            uint32_t st[4]) {
    const uint32_t q = (threadIdx.x & 31) >> 1;
    const int bar = 1 + 4 * (int)pair;
    const uint32_t total = blocks + (pad ? 1 : 0);
    st[0] = l.even ? PK_IV4 : PK_IV0;
    st[1] = l.even ? PK_IV5 : PK_IV1;
    st[2] = l.even ? PK_IV6 : PK_IV2;
    st[3] = l.even ? PK_IV7 : PK_IV3;
    uint32_t c = PK_IV2, d = PK_IV3;  // the even lane's copies of the state's third and fourth word
    if (total == 0) return;
    uint32_t k[16], kn[16];
    const uint32_t *row = nullptr;
    auto next = [&](uint32_t b) {  // block b's row, and its first 16 words into k
        if (b < blocks) pair_bar_sync(bar + (int)(b & 1));
        row = !l.even ? sm.zero : b < blocks ? sm.ring[pair].kw[b & 1][q] : sm.pad;
        pair_ld16(k, row, 0);
    };
    next(0);
    // straight-line rounds, each 16 words of K+W read while the 16 rounds before them run (as a loop of 16 rounds, a
    // block takes 0.4 us more)
#pragma unroll 1
    for (uint32_t b = 0; b < total; ++b) {
        SplitState v;
        uint32_t cd[2];
        split_start(v, l, st, c, d);
        pair_ld16(kn, row, 1);
        split_slot<true>(v, l, k[0], st[1]);
        split_slot<true>(v, l, k[1], st[0]);
#pragma unroll
        for (int j = 2; j < 16; ++j) split_slot(v, l, k[j]);
        pair_ld16(k, row, 2);
#pragma unroll
        for (int j = 0; j < 16; ++j) split_slot(v, l, kn[j]);
        pair_ld16(kn, row, 3);
#pragma unroll
        for (int j = 0; j < 16; ++j) split_slot(v, l, k[j]);
        if (b + 1 < total) next(b + 1);
#pragma unroll
        for (int j = 0; j < 16; ++j) split_slot(v, l, kn[j]);
        if (b + 2 < blocks) pair_bar_arrive(bar + 2 + (int)(b & 1));
        split_end(v, l, st, cd);
        c += cd[0];
        d += cd[1];
    }
}

// This lane's half of the digest to a 16-byte aligned 32-byte slot.
__device__ __forceinline__ void pair_store(uint8_t *dst, const SplitLane &l, const uint32_t st[4]) {
    reinterpret_cast<uint4 *>(dst)[l.even ? 1 : 0] =
        make_uint4(bswap32(st[0]), bswap32(st[1]), bswap32(st[2]), bswap32(st[3]));
}

}  // namespace pk

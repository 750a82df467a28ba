// plan.cuh -- a replica's shared-memory layout and the choice of kernel variant
// and scratch size.  Plain host C++: what it needs to know of the GPU comes
// through its arguments, so that the choice can be checked for every shape on a
// machine without one.
#pragma once

#include <cstddef>
#include <cstdint>

namespace mt {

constexpr int kWarpsPerBlock = 2;
constexpr uint32_t kInstBytes = 52;    // an instance's scalars (InstRec)
constexpr uint32_t kTotCount = 7;      // a replica's rarely changing counters
constexpr uint32_t kParamBytes = 288;  // the block's copy of the kernel parameters
constexpr uint32_t kMagicBytes = 528;  // ceil(2^64 / d) for d = 0..64, rounded up to 16 bytes
// The block's dynamic shared memory: a copy of the parameters (for out-of-line
// functions, which cannot reach the kernel's own), the table of ceil(2^64 / d),
// then each warp's replica state: its layout, the running-request records if
// they are in shared memory, and the scratch.
constexpr uint32_t kHeadBytes = kParamBytes + kMagicBytes;

// The per-warp scratch of variants with several instances per lane, log2 of its
// bytes: a window's distinct event times are counted in it, a tick's ranking and
// the list of a window's formations are kept there (scratch_need).  Small where
// many warps share an SM's shared memory (choose_plan).
constexpr int kSetBitsShared = 12, kSetBits = 11, kSetBitsMany = 10;

struct Layout {
    uint32_t inst;              // [N] x InstRec
    uint32_t cnt;               // [N*K] x 2 B
    uint32_t head, tail, hinfo; // [N*K] x 4 B
    uint32_t h;                 // [K] x 4 B
    uint32_t hist;              // [N*TH] x 1 B
    uint32_t mslot;             // [N] x 16 B
    uint32_t tot;               // [TOT_COUNT] x 4 B
    uint32_t bytes;
};

inline int lanes_c(int N) { return N <= 32 ? 1 : N <= 64 ? 2 : N <= 128 ? 4 : 8; }

// Bytes per instance of the growth histogram: T rounded up to an odd number
// of words, so lanes reading one entry of consecutive instances hit distinct
// banks (1,024-replica workload +0.8 %; the same odd stride for the bucket
// arrays, as one {head, tail, info, count} record per tier, was 3 % slower
// on the 16,384-replica workload).
inline int hist_stride(int T) { return (((T + 3) >> 2) | 1) << 2; }

inline Layout make_layout(int N, int K, int T) {
    Layout L;
    uint32_t o = 0;
    auto take = [&](uint32_t bytes, uint32_t align) {
        o = (o + align - 1) / align * align;
        const uint32_t at = o;
        o += bytes;
        return at;
    };
    L.inst = take(kInstBytes * N, 16);
    L.head = take(4u * N * K, 16);
    L.tail = take(4u * N * K, 16);
    L.hinfo = take(4u * N * K, 16);
    L.h = take(4u * K, 16);
    L.cnt = take(2u * N * K, 16);
    L.hist = take((uint32_t)N * hist_stride(T), 16);
    L.mslot = take(16u * N, 16);
    L.tot = take(4u * kTotCount, 16);
    L.bytes = (o + 15u) & ~15u;
    return L;
}

// Running-request records go to shared memory while a replica's take at most this many bytes.
constexpr uint32_t kSmemSlotLimit = 24u * 1024u;
inline bool slots_in_shared(int N, int Bmax) { return (uint32_t)N * (uint32_t)Bmax * 16u <= kSmemSlotLimit; }

// The least scratch in bytes: the ranking of a tick (ranked_tick) takes a key
// and two indices per instance, 6 bytes for N rounded up to a multiple of 4, and
// the list of a window's formations (list_own) 8 bytes per instance where a
// lane owns several.
inline uint32_t scratch_need(int N) {
    const uint32_t rank = 6u * (((uint32_t)N + 3u) & ~3u), list = lanes_c(N) > 1 ? 8u * (uint32_t)N : 0u;
    return ((rank > list ? rank : list) + 15u) & ~15u;
}

struct Plan {
    int c = 1;         // instances per lane
    bool sms = false;  // running-request records in shared memory
    bool many = false; // the loop of many replicas
    int set_bits = 0;  // the part of the scratch that counts event times, log2 of its bytes
    uint32_t scratch = 0;  // scratch of a warp, bytes
    size_t smem = 0;   // dynamic shared memory of a block
};

// Chooses the kernel variant and the scratch for R replicas on sms_count SMs
// whose blocks can have max_smem bytes of dynamic shared memory.  resident(plan)
// gives the blocks of the plan's kernel variant that fit on an SM with its
// dynamic shared memory (at most max_smem), or a negative value on an error,
// which choose_plan returns.  Otherwise it returns the resident blocks of the
// plan chosen; 0: the state does not fit.
template <class Resident>
int choose_plan(int R, int N, int Bmax, const Layout &L, int sms_count, size_t max_smem, Resident resident, Plan &out) {
    const long long want = ((long long)R + kWarpsPerBlock - 1) / kWarpsPerBlock;
    // scratch of a given number of bits (0: event times are not counted in it)
    auto scratch_of = [&](int bits) { return bits > 0 ? 1u << bits : scratch_need(N); };
    auto smem_of = [&](bool sms, int bits) {
        return kHeadBytes +
               (size_t)kWarpsPerBlock * (L.bytes + (sms ? (uint32_t)N * (uint32_t)Bmax * 16u : 0u) + scratch_of(bits));
    };
    int least = lanes_c(N) > 1 ? kSetBitsMany : 0;
    while (scratch_of(least) < scratch_need(N)) ++least;
    // the records stay in HBM where the state leaves no room for them (254 or more
    // instances with 16 tiers and about 50 tokens per block)
    const bool sms = slots_in_shared(N, Bmax) && smem_of(true, least) <= max_smem;
    out.c = lanes_c(N);
    out.sms = sms;
    auto with_bits = [&](int bits) {
        out.set_bits = bits;
        out.scratch = scratch_of(bits);
        out.smem = smem_of(sms, bits);
        return out.smem <= max_smem ? resident(out) : 0;
    };
    // Which main loop (see k_run): that of many replicas above 10 (C = 1) or 14
    // (C = 2) per SM.  1,500 requests per replica, records in HBM, loop of many /
    // of few, ms: 32 instances, 304 replicas 9.2 / 7.9, 1,216 9.9 / 9.0, 1,824 10.7 /
    // 11.5, 2,432 11.4 / 20.1; 64 instances, 304 replicas 15.5 / 12.0, 1,824 18.8 /
    // 15.7, 2,432 20.1 / 28.0 (14 warps of the loop of few fit on an SM).  With
    // records in shared memory only where at least 5 blocks fit: 8,192 replicas x 8
    // x 400 requests 15.9 / 21.6, 8,192 x 16 x 500 26.0 / 28.3 (5 blocks), 6,000 x
    // 24 x 400 27.7 / 24.4 (3 blocks).
    out.many = (sms ? out.c == 1 : out.c <= 2) && R > (sms ? 10 : out.c == 1 ? 10 : 14) * sms_count;
    if (out.many && sms) {
        const int n = with_bits(0);
        if (n < 0) return n;
        out.many = n >= 5;
    }
    // The scratch with several instances per lane: 4 KB holds a window of the
    // default `base` of 4 ms directly.  Where two instances per lane share an SM
    // with 17 other warps it has 2 KB, and 1 KB, with two warps more, for sweeps of
    // several waves (8,192 x 64: 110.2 against 112.5 ms).  Elsewhere it shrinks where
    // that makes every replica resident; more warps of several waves alone gain
    // nothing there (2,048 x 100 x 500: 26.3 against 23.9 ms).  It never goes below
    // what the shape's other uses take.
    if (out.c == 1) return with_bits(0);
    if (out.many) return with_bits(R > 26 * sms_count ? kSetBitsMany : kSetBits);
    int bits = kSetBitsShared;
    while (bits > least && smem_of(sms, bits) > max_smem) --bits;
    for (int b = bits; b >= least; --b) {
        const int n = with_bits(b);
        if (n < 0) return n;
        if ((long long)n * sms_count >= want) return n;
    }
    return with_bits(bits);
}

}  // namespace mt

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
    bool many = false; // the variant for many replicas
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
    auto waves = [&](int n) { return n > 0 ? (want + (long long)n * sms_count - 1) / ((long long)n * sms_count) : 1ll << 40; };
    // The plan of one main loop, which out keeps: its scratch and its resident
    // blocks.  With several instances per lane 4 KB of scratch hold a window of the
    // default `base` of 4 ms directly.  The loop of few takes less where that makes
    // every replica resident (more warps of several waves alone gain nothing: 2,048 x
    // 100 x 500 26.3 against 23.9 ms).  The loop of many has 2 KB, and for sweeps of
    // several waves 1 KB where more blocks then fit (8,192 x 64 with 4 tiers, ten
    // blocks instead of nine: 110.2 against 112.5 ms; with 6 tiers eight blocks either
    // way).  Never less than the shape's other uses take.
    auto plan_loop = [&](bool many) {
        out.many = many;
        if (out.c == 1) return with_bits(0);
        if (many && out.c == 2) {
            const int n = with_bits(kSetBits);
            if (n < 0 || R <= 26 * sms_count) return n;
            const int n2 = with_bits(kSetBitsMany);
            return n2 < 0 || n2 > n ? n2 : with_bits(kSetBits);
        }
        int bits = kSetBitsShared;
        while (bits > least && smem_of(sms, bits) > max_smem) --bits;
        for (int b = bits; b >= least; --b) {
            const int n = with_bits(b);
            if (n < 0 || waves(n) == 1) return n;
        }
        return with_bits(bits);
    };
    // Which main loop (see k_run).
    if (out.c == 1 && sms) {
        // Records in shared memory: both loops have about the same residency, and the
        // loop of many scales better with the warps that share an SM's instruction
        // cache, the sooner the fewer instances share a window.  Loop of few / of many,
        // ms, at 0.85 load: 4 instances, 912 replicas 16.3 / 17.0, 1,216 19.3 / 17.2; 8,
        // 912 13.5 / 14.5, 1,216 15.9 / 14.7; 12, 1,216 9.2 / 9.8, 1,520 10.8 / 10.3; 16,
        // 1,216 16.5 / 17.2, 1,520 19.7 / 18.4 (800 requests 5.4 / 6.1, 8,000 41.5 / 35.7);
        // one instance, 1,520 6.7 / 7.7.  At 0.3 to 0.4 load the lines lie about 1
        // replica per SM higher.  Only where at least 5 blocks fit (6,000 x 24 x 400,
        // 3 blocks: 24.4 / 27.7).
        const int per_sm = N == 1 ? 12 : N <= 8 ? 7 : 10;
        if (R > per_sm * sms_count) {
            const int n = plan_loop(true);
            if (n < 0 || n >= 5) return n;
        }
    } else if (out.c <= 2 && !sms) {
        // Records in HBM: a wave of the loop of few takes less time than one of the
        // loop of many, which holds more replicas.  Loop of few / of many, ms: 64
        // instances, 4 tiers (12 and 18 to 20 warps per SM), 1,824 replicas 13.8 / 18.2,
        // 2,000 23.7 / 19.2, 3,648 21.6 / 26.8, 4,000 37.9 / 37.2; 16 tiers (8 and 10
        // warps) 2,432 18.5 / 25.1, 4,000 34.0 / 37.2; 40 instances 1,824 13.1 / 15.5, 2,000
        // 21.5 / 16.6; 32 instances (12 and 16 warps) 1,824 9.0 / 10.0, 2,128 15.3 / 10.7,
        // 3,648 17.6 / 19.5, 4,864 24.8 / 20.9.  Past three waves the rate of a full SM
        // decides: 16,384 x 64 x 400 with 4, 8, 13 and 16 tiers (20, 14, 12 and 10 warps of
        // the loop of many) 81.7 / 65.9, 83.6 / 79.2, 90.3 / 87.2, 93.1 / 100.1.
        const int few = plan_loop(false);
        if (few < 0) return few;
        const int many = plan_loop(true);
        if (many < 0) return many;
        if (waves(few) > 3 ? many >= 6 : (out.c == 1 ? 11 : 14) * waves(many) < 10 * waves(few)) return many;
    }
    const int few = plan_loop(false);
    if (few < 0 || out.c != 4 || sms || waves(few) == 1) return few;
    // Four instances per lane, records in HBM: the same loop with 12 warps per SM
    // instead of 8 where that saves a wave.  8 / 12 warps, ms: 1,500 x 128 x 500 21.9 /
    // 15.5, 1,824 x 100 x 500 21.0 / 16.1, 4,096 x 100 44.7 / 41.2; 2,048 x 100 x 3,000,
    // two waves either way, 48.4 / 54.0; 2 x 74 x 1,279 14.8 / 15.3.
    const int many = plan_loop(true);
    return many < 0 || waves(many) < waves(few) ? many : plan_loop(false);
}

}  // namespace mt

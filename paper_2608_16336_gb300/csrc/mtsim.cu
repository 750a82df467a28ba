// mtsim.cu -- batched simulation of the multi-tier Llumnix-style scheduler
// ("Beyond Binary Priorities: Multi-Tier SLA Scheduling for LLM Serving",
// Sec. 3) for sm_103a, behind the C ABI declared in mtsim.h.
//
// Execution model
//   One warp simulates one replica.  A persistent grid pulls replicas from an
//   atomic work counter.  While a warp owns a replica, the replica's instance
//   state (per-instance scalars, per-(instance, tier) queue heads/tails and
//   request counts, headroom table) lives in shared memory, and so do the
//   running-request slots when they fit; everything is written back to HBM
//   when the warp stops (step limit or completion), so sim_run can be resumed.
//   Instance i belongs to lane i mod 32, C = ceil(N/32) instances per lane (C
//   is a template parameter, rounded up to a power of two); where the order of
//   instances matters, it is taken from their indices.  Per-request state stays in HBM: the read-only trace
//   (SoA), the 16-byte result record and a 16-byte queue node that threads a
//   waiting request into its (instance, tier) FCFS bucket.  A running request
//   is a 16-byte slot record that is written when it joins a batch and read
//   only on events; batch advance is lazy (see the slot record below), so an
//   iteration end and a batch formation without events cost O(1).
//   Between global events (arrivals, migration ticks) the instances that are
//   in no migration do not interact, and the two ends of a migration only with
//   each other, so the lanes advance them through a window in which each ends
//   at most one iteration; global events are stepped by the whole warp in the
//   oracle's order.  The next 32 arrivals are held in registers, one per lane.
//
// Exactness
//   Everything is integer.  Freeness F = (M - U) / max(B, 1) (Sec. 3.2 Eq. 1-2)
//   is kept per instance as an order-preserving 32-bit key
//   floor((M - U) * 4096 / max(B, 1)): for batch sizes up to 64, two distinct
//   fractions differ by at least 1/4032, so the floored keys order every pair
//   of freeness values exactly as the fractions do and equal fractions get
//   equal keys.  The floor division by B is the high half of the product
//   with a per-block table entry ceil(2^64 / B), exact for every 32-bit
//   numerator.  The
//   arg-max/arg-min of dispatch and migration pairing are therefore one warp
//   __reduce_{max,min}_sync plus a ballot (lowest index on ties).  The
//   migration threshold max F - min F >= theta is checked exactly by 64-bit
//   cross-multiplication.  Since free + sum(running blocks) + inbound
//   reservation = M on every instance, M - U reduces to
//   free - HoL demand - sum of present-tier headroom.
//
// Safety
//   No kernel waits on another warp, block or launch: there are no spin
//   loops.  Every loop is bounded by the trace length, the batch size, or the
//   per-call step limit.  Index checks on queue links and slot positions turn
//   an inconsistency into SIM_ERR_INTERNAL for that replica instead of an
//   out-of-bounds access.
#include "mtsim.h"
#include "latency.cuh"
#include "plan.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstddef>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

// A condition that rarely holds: its code is laid out away from the hot loop,
// which several warps at different points share through the instruction cache.
#define MT_RARE(c) (__builtin_expect(!!(c), 0))

namespace mt {

constexpr uint32_t kNone = 0xFFFFFFFFu;  // idle instance / no pending event / nil link
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr int kKeyShift = 12;            // keys are floor(num * 4096 / den)
constexpr int kMaxKeyRange = 1 << 19;    // |num| < 2^19 keeps num * 4096 below 2^31
constexpr int kMagicShift = 40;          // floor(n / T) = (n * ceil(2^40 / T)) >> 40 for n < 2^20, T <= 65535
constexpr int kMaxBlockTokens = 64;      // T limit of the per-instance growth histogram

enum : int { MIG_NONE = 0, MIG_SRC = 1, MIG_DST = 2 };

// A running request is a 16-byte slot record, written when it joins an
// instance's running list and read only on events (finish, preemption,
// migration, first token):
//   x = request id (index in the replica's trace)
//   y = phi: number of the instance's first formation that includes it
//   z = c | left << 16: its context length P + g and its remaining output O - g at formation phi
//   w = tier | rho << 16, rho = (c - phi) mod T
// With nf formations done and pc = 1 after the iteration that followed the
// last one (0 before), the request has advanced adv = nf - phi + pc tokens
// (0 if phi > nf) and holds ceil((c + nf - phi) / T) KV blocks: every
// formation grows each surviving request to exactly its need, one block at a
// time because contexts grow by one token per iteration.  So the number of
// requests that need a new block at the next formation is the count of
// running requests with rho == -nf (mod T), and a request finishes at the
// iteration that follows formation phi + left - 1.

// A waiting request's queue node (16 bytes, indexed by request) carries what
// admitting it needs: x = next, y = info of next, z = prev, w = own info, with
// info = context (P + g) | remaining output (O - g) << 16.  The info of each
// bucket's head is also kept in shared memory, so admission and the HoL demand
// need no dependent HBM reads.

// An instance's scalars, one record per instance: every field sits at a
// fixed offset from the record, so the accesses to one instance share one
// address.  13 words: lanes reading one field of consecutive instances hit
// distinct shared-memory banks.
struct InstRec {
    uint32_t busy;                // end of the running iteration, or kNone when idle
    int free_, resv, hol, hr;     // free KV blocks; reserved for inbound copies; HoL demand; present headroom
    int key;                      // freeness key (dispatch, rebalancing)
    uint32_t mreq;                // request being copied out (migration source)
    int mcopied;                  // its blocks copied so far
    uint32_t nf, minfin, drain;   // formations done; next finishing formation; drain start
    uint16_t wmask;               // non-empty tier buckets
    uint8_t nrun, pc, phase;      // running requests; iteration-ended flag; nf mod T
    uint8_t mrole, mpeer, mpend;  // migration role and peer; phase of a log record held back in mslot, or 0
};
static_assert(sizeof(InstRec) == 52 && sizeof(InstRec) == kInstBytes, "InstRec is 13 words");

// x.busy[i] and the like: field F of instance i's record.
template <typename T, int OFF>
struct Field {
    unsigned char *base;  // the replica's record array
    __device__ __forceinline__ T &operator[](int i) const {
        return *reinterpret_cast<T *>(base + i * (int)sizeof(InstRec) + OFF);
    }
};
#define MT_FIELD(T, f) Field<T, (int)offsetof(InstRec, f)> f

// A replica's rarely changing counters, kept with its instance state so that
// they hold no registers: log records, migrations, preemptions, migration
// starts and aborts, scale-out and scale-in signals.  Several lanes at once may
// add to TOT_PRE, TOT_ABORT and TOT_MIG (atomics), one lane at a time to the
// others.
enum : int { TOT_LOG = 0, TOT_MIG, TOT_PRE, TOT_START, TOT_ABORT, TOT_OUT, TOT_IN, TOT_COUNT };
static_assert(TOT_COUNT == kTotCount, "counters of the layout");

// Per-replica scalars persisted between sim_run calls.
struct RepState {
    uint32_t t, cursor, finished, log_events;
    uint32_t next_tick, pad0;
    uint64_t steps, iterations, member_iterations, events;
    uint32_t migrations, preemptions, starts, aborts;
    uint32_t scale_out, scale_in;
    int32_t status;
    uint32_t pad1;
};

struct Params {
    int R, N, M, T, TH, Bmax, K, S, cap, enable_mig, theta_num, theta_den;
    uint32_t interval, max_steps;
    unsigned long long magT;      // ceil(2^40 / T)
    int base, a, b;
    int ticks;                    // ticks happen (migration or the auto-scaling signal is on)
    int autoscale, scale_out_num, scale_in_num, scale_den;
    int drains;                   // a drain schedule is loaded
    unsigned long long lcm_lo, lcm_hi;  // lcm(1, ..., Bmax) as two 64-bit halves
    Layout L;
    int set_bits;                 // scratch of distinct_times (several instances per lane), log2 of its bytes
    uint32_t scratch;             // per-warp scratch, bytes
    const long long *offsets;
    const uint32_t *drain_src;    // [R][N] drain start times, or NULL
    const uint32_t *arrival;
    const uint16_t *plen, *olen;
    const uint8_t *tier;
    uint4 *node;                  // queue node per request: next, info of next, prev, own info
    sim_request_result_t *res;
    long long res_off;            // bytes from a request's queue node to its result record
    unsigned char *blobs;
    uint4 *slots;                 // [R][N][Bmax]
    RepState *rep;
    sim_migration_event_t *log;
    int *work;
    const int *order;             // [R] start order of the replicas, or NULL (trace order)
};

// Per-warp view of the replica being simulated: instance state in shared
// memory, request state in HBM, slot records in either; scalars are warp-uniform
// except t while lanes advance their own instances.
struct Ctx {
    MT_FIELD(uint32_t, busy);
    MT_FIELD(int, free_);
    MT_FIELD(int, resv);
    MT_FIELD(int, hol);
    MT_FIELD(int, hr);
    MT_FIELD(int, key);
    MT_FIELD(uint32_t, mreq);
    MT_FIELD(int, mcopied);
    MT_FIELD(uint32_t, nf);
    MT_FIELD(uint32_t, minfin);
    MT_FIELD(uint32_t, drain);
    MT_FIELD(uint16_t, wmask);
    MT_FIELD(uint8_t, nrun);
    MT_FIELD(uint8_t, pc);
    MT_FIELD(uint8_t, phase);
    MT_FIELD(uint8_t, mrole);
    MT_FIELD(uint8_t, mpeer);
    MT_FIELD(uint8_t, mpend);
    uint32_t *head, *tail, *hinfo;
    int *h;
    uint16_t *cnt;
    uint8_t *hist;
    uint4 *mslot;                     // record of the request a migration source is copying out
    uint4 *slots;
    uint32_t *tset;                   // scratch: event times, a tick's ranking, a window's formations (scratch_need)
    const unsigned long long *magic;  // [65]: ceil(2^64 / d) for d >= 2
    uint32_t *tot;                    // TOT_* counters
    uint4 *node;                      // the replica's queue nodes
    int r;                            // the replica
    unsigned long long magT;
    int N, K, T, TH, Bmax, S, lane, drains, set_bits;
    uint32_t Q, t;
    bool hold;                        // inside a window: log records are held back until it closes

    // Copies of kernel parameters (they hold no registers), and from them the
    // first trace record of the replica, its result records and its log.
    const uint32_t *arrival;
    const uint16_t *plen, *olen;
    const uint8_t *tier;
    const uint4 *node0;
    sim_migration_event_t *log0;
    long long res_off;
    int cap;
    __device__ __forceinline__ long long first() const { return node - node0; }
    __device__ __forceinline__ sim_request_result_t *res(uint32_t q) const {
        return reinterpret_cast<sim_request_result_t *>(reinterpret_cast<unsigned char *>(node + q) + res_off);
    }
    __device__ __forceinline__ uint4 *log(uint32_t k) const {
        return reinterpret_cast<uint4 *>(log0) + (size_t)r * cap + k;
    }
};

// Counters of this launch.  `iterations` and `member_iterations` are summed over
// the lanes when the warp leaves the replica; `finished` is the replica's total
// on every lane; a status below 0 on any lane ends the run.
struct Cnt {
    uint32_t finished, steps, iterations;
    uint64_t member_iterations;
    int status;
    bool held;  // this lane has held back a log record in the open window
};

static_assert(((sizeof(Params) + 15u) & ~15u) == kParamBytes, "parameter copy of the block's shared memory");

__device__ __forceinline__ void bind_blob(Ctx &x, const Layout &L, unsigned char *blob) {
    unsigned char *ib = blob + L.inst;
    x.busy.base = x.free_.base = x.resv.base = x.hol.base = x.hr.base = x.key.base = ib;
    x.mreq.base = x.mcopied.base = x.nf.base = x.minfin.base = x.drain.base = ib;
    x.wmask.base = x.nrun.base = x.pc.base = x.phase.base = x.mrole.base = x.mpeer.base = x.mpend.base = ib;
    x.cnt = reinterpret_cast<uint16_t *>(blob + L.cnt);
    x.head = reinterpret_cast<uint32_t *>(blob + L.head);
    x.tail = reinterpret_cast<uint32_t *>(blob + L.tail);
    x.hinfo = reinterpret_cast<uint32_t *>(blob + L.hinfo);
    x.h = reinterpret_cast<int *>(blob + L.h);
    x.hist = blob + L.hist;
    x.mslot = reinterpret_cast<uint4 *>(blob + L.mslot);
    x.tot = reinterpret_cast<uint32_t *>(blob + L.tot);
}

// The view of replica r that this warp is simulating, at time t.  BITS: the
// scratch is 2^set_bits bytes (several instances per lane); taken from there the
// loop of many is faster than from the parameter (4,096 x 64 x 10,000 requests 150.8
// -> 149.1 ms).
template <bool SMS, bool BITS = false>
__device__ __forceinline__ void bind_ctx(Ctx &x, const Params &p, unsigned char *smem, uint4 *node, uint32_t Q, int r,
                                         uint32_t t) {
    const uint32_t slot_bytes = SMS ? (uint32_t)p.N * (uint32_t)p.Bmax * 16u : 0u;
    unsigned char *blob =
        smem + kHeadBytes + (size_t)(threadIdx.x >> 5) * (p.L.bytes + slot_bytes + (BITS ? 1u << p.set_bits : p.scratch));
    bind_blob(x, p.L, blob);
    x.slots = SMS ? reinterpret_cast<uint4 *>(blob + p.L.bytes) : p.slots + (size_t)r * p.N * p.Bmax;
    x.tset = reinterpret_cast<uint32_t *>(blob + p.L.bytes + slot_bytes);
    x.set_bits = p.set_bits;
    x.Q = Q;
    x.node = node;
    x.r = r;
    x.arrival = p.arrival;
    x.plen = p.plen;
    x.olen = p.olen;
    x.tier = p.tier;
    x.node0 = p.node;
    x.log0 = p.log;
    x.res_off = p.res_off;
    x.cap = p.cap;
    x.magic = reinterpret_cast<const unsigned long long *>(smem + kParamBytes);
    x.magT = p.magT;
    x.N = p.N;
    x.K = p.K;
    x.T = p.T;
    x.TH = p.TH;
    x.Bmax = p.Bmax;
    x.S = p.S;
    x.lane = (int)(threadIdx.x & 31);
    x.drains = p.drains;
    x.t = t;
    x.hold = false;
}

__device__ __forceinline__ int blocks_for(const Ctx &x, uint32_t tokens) {
    return (int)(((unsigned long long)(tokens + (uint32_t)x.T - 1u) * x.magT) >> kMagicShift);
}
__device__ __forceinline__ uint32_t mod_t(const Ctx &x, uint32_t v) {  // v mod T for v < 2^20
    const uint32_t q = (uint32_t)(((unsigned long long)v * x.magT) >> kMagicShift);
    const uint32_t r = v - q * (uint32_t)x.T;
    return r >= (uint32_t)x.T ? r - (uint32_t)x.T : r;
}

// floor(v / d) for v < 2^32 and 1 <= d <= 64: the high half of v * ceil(2^64 / d).
__device__ __forceinline__ uint32_t div_small(const Ctx &x, uint32_t v, int d) {
    const uint32_t q = (uint32_t)__umul64hi((unsigned long long)v, x.magic[d]);
    return d == 1 ? v : q;
}

// SELECT: without branches.  Where instruction fetch bounds (two instances per
// lane, many replicas) the other form is faster: 8,192 x 64 108.8 against 112.0
// ms, in its steady state (4,096 x 10,000 requests) 151 against 157 ms.
template <bool SELECT = true>
__device__ __forceinline__ int make_key(const Ctx &x, int num, int nrun) {
    if constexpr (!SELECT) {
        const int d = nrun > 0 ? nrun : 1;
        if (num >= 0) return (int)(d == 1 ? (uint32_t)num << kKeyShift : div_small(x, (uint32_t)num << kKeyShift, d));
        const uint32_t v = ((uint32_t)(-num) << kKeyShift) + (uint32_t)(d - 1);
        return -(int)(d == 1 ? v : div_small(x, v, d));
    }
    // one division of the magnitude, rounded down or (negative) up, without
    // branches (64 x 256 58.8 -> 56.9 ms, 1,024 x 16 8.75 -> 8.60)
    const int d = max(nrun, 1);
    const uint32_t mag = ((uint32_t)abs(num) << kKeyShift) + (num < 0 ? (uint32_t)(d - 1) : 0u);
    const int q = (int)div_small(x, mag, d);
    return num < 0 ? -q : q;
}

__device__ __forceinline__ int fnum(const Ctx &x, int i) { return x.free_[i] - x.hol[i] - x.hr[i]; }

template <bool SELECT>
__device__ __forceinline__ void set_key(const Ctx &x, int i) {
    x.key[i] = make_key<SELECT>(x, fnum(x, i), x.nrun[i]);
}

// Instance j of a lane (j < C) and back.  Consecutive lanes own consecutive
// instances, so their records (13 words each) lie in different shared-memory
// banks.  (With C consecutive instances per lane they were C x 13 words apart,
// a 2- to 8-way conflict for every access of all lanes: 64 x 256 63.0 -> 59.2
// ms, 256 x 128 41.6 -> 40.8, 97 x 33 10.6 -> 10.1; 8,192 x 64 108.8 -> 109.3.)
__device__ __forceinline__ int inst_at(int lane, int j) { return lane + 32 * j; }
__device__ __forceinline__ int lane_of(int i) { return i & 31; }
__device__ __forceinline__ int num_of(int i) { return i >> 5; }

template <int C>
__device__ __forceinline__ void refresh_keys(const Ctx &x) {
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (i < x.N) set_key<C != 2>(x, i);
    }
    __syncwarp();
}

template <int C>
__device__ __forceinline__ uint32_t own_mask(const Ctx &x) {
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < C; ++j)
        if (inst_at(x.lane, j) < x.N) m |= 1u << j;
    return m;
}

// Arg-max (want_max) or arg-min of the freeness key over the instances whose
// bit is set in `el` (bit j = the lane's instance j), excluding `excl`; lowest
// index on ties; -1 if none.  Collective.
template <int C>
__device__ __forceinline__ int arg_ext(const Ctx &x, uint32_t el, bool want_max, int excl) {
    int bv = want_max ? INT_MIN : INT_MAX, bi = -1;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (((el >> j) & 1u) && i != excl) {
            const int k = x.key[i];
            if (bi < 0 || (want_max ? k > bv : k < bv)) { bv = k; bi = i; }
        }
    }
    const int m = want_max ? __reduce_max_sync(kFull, bv) : __reduce_min_sync(kFull, bv);
    // lowest instance among those at the extreme (INT_MAX: none)
    const int best = __reduce_min_sync(kFull, (bi >= 0 && bv == m) ? bi : INT_MAX);
    return best == INT_MAX ? -1 : best;
}

// ---- single-thread instance logic (no collectives inside) -------------------
__device__ __forceinline__ void cnt_inc(const Ctx &x, int i, int k) {
    if (x.cnt[i * x.K + k]++ == 0) x.hr[i] += x.h[k];
}
__device__ __forceinline__ void cnt_dec(const Ctx &x, int i, int k) {
    if (--x.cnt[i * x.K + k] == 0) x.hr[i] -= x.h[k];
}
__device__ __forceinline__ void push_back(const Ctx &x, int i, int k, uint32_t r, uint32_t info) {
    const int b = i * x.K + k;
    const uint32_t tl = x.tail[b];
    x.node[r] = make_uint4(kNone, 0u, tl, info);
    if (tl != kNone) *reinterpret_cast<uint2 *>(&x.node[tl]) = make_uint2(r, info);
    else { x.head[b] = r; x.hinfo[b] = info; }
    x.tail[b] = r;
    x.wmask[i] |= (uint16_t)(1u << k);
}
__device__ __forceinline__ void push_front(const Ctx &x, int i, int k, uint32_t r, uint32_t info) {
    const int b = i * x.K + k;
    const uint32_t hd = x.head[b];
    x.node[r] = make_uint4(hd, hd != kNone ? x.hinfo[b] : 0u, kNone, info);
    if (hd != kNone) x.node[hd].z = r; else x.tail[b] = r;
    x.head[b] = r;
    x.hinfo[b] = info;
    x.wmask[i] |= (uint16_t)(1u << k);
}
// Removes the tail of bucket (i, k) and returns its info in `info`.
__device__ __forceinline__ uint32_t pop_back(const Ctx &x, int i, int k, uint32_t &info, int &status) {
    const int b = i * x.K + k;
    const uint32_t r = x.tail[b];
    if (r >= x.Q) { status = SIM_ERR_INTERNAL; return kNone; }
    const uint4 nd = x.node[r];
    info = nd.w;
    x.tail[b] = nd.z;
    if (nd.z != kNone) *reinterpret_cast<uint2 *>(&x.node[nd.z]) = make_uint2(kNone, 0u);
    else { x.head[b] = kNone; x.wmask[i] &= (uint16_t)~(1u << k); }
    return r;
}
// HoL demand: KV blocks the head of the highest-priority non-empty bucket needs.
__device__ __forceinline__ void refresh_hol(const Ctx &x, int i) {
    const uint32_t wm = x.wmask[i];
    x.hol[i] = wm ? blocks_for(x, x.hinfo[i * x.K + (__ffs(wm) - 1)] & 0xFFFFu) : 0;
}
__device__ __forceinline__ void log_ev(const Ctx &x, int kind, uint32_t r, int s, int d, int blocks) {
    const uint32_t k = x.tot[TOT_LOG]++;
    if (k < (uint32_t)x.cap)
        *x.log(k) = make_uint4(x.t, r, (uint32_t)(blocks & 0xFFFF) | ((uint32_t)s << 16) | ((uint32_t)d << 24),
                               (uint32_t)kind);
}
// The record that ends the migration out of source s (phase 1: copy stage or
// finish, phase 4: preemption in batch formation).  In a window the pairs of
// migrating instances advance independently of one another, so the record is
// held back in the source's slot copy, which nothing needs any more, and
// flush_held writes the window's records in the order of time, phase and
// instance.  A migration starts only at a tick, so a source has at most one.
__device__ __forceinline__ void log_end(const Ctx &x, Cnt &cn, int kind, uint32_t r, int s, int d, int blocks, int ph) {
    if (x.hold) {
        x.mslot[s] = make_uint4(x.t, r, (uint32_t)(blocks & 0xFFFF) | ((uint32_t)s << 16) | ((uint32_t)d << 24),
                                (uint32_t)kind);
        x.mpend[s] = (uint8_t)ph;
        cn.held = true;
    } else {
        log_ev(x, kind, r, s, d, blocks);
    }
}
// Writes the records held back in a window that some lane has, and returns
// whether some instance is still in a migration (one ends only with such a
// record).  Collective.
template <int C>
__device__ __forceinline__ bool flush_held(const Ctx &x, Cnt &cn) {
    uint32_t left = 0;
    bool mig = false;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (i < x.N && x.mpend[i] != 0) left |= 1u << j;
        if (i < x.N && x.mrole[i] != MIG_NONE) mig = true;
    }
    mig = __any_sync(kFull, mig);
#pragma unroll 1
    while (__any_sync(kFull, left != 0)) {
        uint32_t bt = kNone;
#pragma unroll
        for (int j = 0; j < C; ++j)
            if ((left >> j) & 1u) bt = min(bt, x.mslot[inst_at(x.lane, j)].x);
        const uint32_t t = __reduce_min_sync(kFull, bt);
        uint32_t bk = kNone;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int i = inst_at(x.lane, j);
            if (((left >> j) & 1u) && x.mslot[i].x == t) bk = min(bk, ((uint32_t)x.mpend[i] << 16) | (uint32_t)i);
        }
        const int s = (int)(__reduce_min_sync(kFull, bk) & 0xFFFFu);
        if (x.lane == lane_of(s)) {
            left &= ~(1u << num_of(s));
            x.mpend[s] = 0;
        }
        if (x.lane == 0) {
            const uint32_t k = x.tot[TOT_LOG]++;
            if (k < (uint32_t)x.cap) *x.log(k) = x.mslot[s];
        }
    }
    cn.held = false;
    __syncwarp();
    return mig;
}
// The result record's last word holds n_preemptions (low half) and
// n_migrations (high half), both modulo 2^16.  A migration adds 1 << 16: a
// wrap carries out of the word, so nothing waits on the add.  A preemption
// adds 1 to the low half and gets the old word back; when the low half
// wrapped, the carry into n_migrations is taken back (pre_fix).
__device__ __forceinline__ unsigned int *count_word(const Ctx &x, uint32_t r) {
    return reinterpret_cast<unsigned int *>(reinterpret_cast<unsigned char *>(x.res(r)) + 12);
}
__device__ __forceinline__ void bump_mig(const Ctx &x, uint32_t r) { atomicAdd(count_word(x, r), 1u << 16); }
__device__ __forceinline__ unsigned int bump_pre(const Ctx &x, uint32_t r) { return atomicAdd(count_word(x, r), 1u); }
__device__ __forceinline__ void pre_fix(const Ctx &x, uint32_t r, unsigned int old) {
    if ((old & 0xFFFFu) == 0xFFFFu) atomicSub(count_word(x, r), 1u << 16);
}
__device__ __forceinline__ void clear_mig(const Ctx &x, int s, int d) {
    x.mrole[s] = MIG_NONE;
    x.mrole[d] = MIG_NONE;
    x.mreq[s] = kNone;
    x.mcopied[s] = 0;
}
// Abandon the staged copy out of source s: the destination releases what was copied.
__device__ __forceinline__ void abort_mig(const Ctx &x, Cnt &cn, int s, int ph) {
    const int d = x.mpeer[s];
    const int cp = x.mcopied[s];
    x.free_[d] += cp;
    x.resv[d] -= cp;
    log_end(x, cn, SIM_EV_ABORT, x.mreq[s], s, d, cp, ph);
    atomicAdd(&x.tot[TOT_ABORT], 1u);
    clear_mig(x, s, d);
}

// Derived quantities of a slot record on instance i.
__device__ __forceinline__ uint32_t sl_c(const uint4 &sl) { return sl.z & 0xFFFFu; }
__device__ __forceinline__ uint32_t sl_left(const uint4 &sl) { return sl.z >> 16; }
__device__ __forceinline__ uint32_t sl_tier(const uint4 &sl) { return sl.w & 0xFFu; }
__device__ __forceinline__ uint32_t sl_rho(const uint4 &sl) { return sl.w >> 16; }
__device__ __forceinline__ uint32_t sl_fin(const uint4 &sl) { return sl.y + sl_left(sl) - 1u; }
__device__ __forceinline__ uint32_t sl_adv(const Ctx &x, int i, const uint4 &sl) {
    const uint32_t nf = x.nf[i];
    return sl.y <= nf ? nf - sl.y + x.pc[i] : 0u;
}
__device__ __forceinline__ int sl_blocks(const Ctx &x, int i, const uint4 &sl) {
    return blocks_for(x, sl_c(sl) + x.nf[i] - sl.y);
}
__device__ __forceinline__ uint4 *slot_ptr(const Ctx &x, int i, int s) { return x.slots + i * x.Bmax + s; }

// A request joins instance i's running list at position n with context c and
// remaining output left; its first formation there will be number nf + 1.
__device__ __forceinline__ void slot_join_at(const Ctx &x, int i, int n, uint32_t r, uint32_t c, uint32_t left,
                                             uint32_t tier, uint32_t nf, uint32_t ph) {
    const uint32_t phi = nf + 1u;
    const uint32_t pm = ph + 1u == (uint32_t)x.T ? 0u : ph + 1u;  // phi mod T
    const uint32_t cm = mod_t(x, c);
    const uint32_t rho = cm >= pm ? cm - pm : cm + (uint32_t)x.T - pm;
    *slot_ptr(x, i, n) = make_uint4(r, phi, c | (left << 16), tier | (rho << 16));
    x.hist[i * x.TH + rho]++;
    x.minfin[i] = min(x.minfin[i], phi + left - 1u);
}
__device__ __forceinline__ void slot_join(const Ctx &x, int i, int n, uint32_t r, uint32_t c, uint32_t left,
                                          uint32_t tier) {
    slot_join_at(x, i, n, r, c, left, tier, x.nf[i], x.phase[i]);
}

// Books the commit of the fully copied running request of source s at its
// destination (Sec. 3.5, Fig. 4), on one lane.  The warp has already taken the
// slot out of s's running list (order kept); fm is the new minimum finishing
// formation of what is left there.
__device__ __forceinline__ void commit_book(const Ctx &x, Cnt &cn, int s, uint32_t fm) {
    const uint4 sl = x.mslot[s];  // slot records do not change while they run
    const int d = x.mpeer[s];
    const int blocks = sl_blocks(x, s, sl);
    const uint32_t adv = sl_adv(x, s, sl);
    x.nrun[s] = (uint8_t)(x.nrun[s] - 1);
    x.hist[s * x.TH + sl_rho(sl)]--;
    x.minfin[s] = fm;
    x.free_[s] += blocks;
    x.resv[d] -= x.mcopied[s];
    const uint32_t tr = sl_tier(sl);
    cnt_dec(x, s, (int)tr);
    cnt_inc(x, d, (int)tr);
    const int nd = x.nrun[d];
    slot_join(x, d, nd, sl.x, sl_c(sl) + adv, sl_left(sl) - adv, tr);
    x.nrun[d] = (uint8_t)(nd + 1);
    bump_mig(x, sl.x);
    atomicAdd(&x.tot[TOT_MIG], 1u);
    log_end(x, cn, SIM_EV_COMMIT, sl.x, s, d, blocks, 1);
    clear_mig(x, s, d);
}

// Phase 1, first part, single thread: the iteration of instance i ends at
// x.t (Sec. 2.1 token accounting; first tokens were recorded when the
// prefill iteration was scheduled).  Returns whether some running request
// finishes now (then coop_finish must run before anything else touches i).
__device__ __forceinline__ bool inst_complete_head(const Ctx &x, int i) {
    x.busy[i] = kNone;
    x.pc[i] = 1;
    return x.minfin[i] == x.nf[i];
}

// Phase 1, second part, whole warp: the requests of instance i whose output
// is complete finish at x.t and free their KV (an in-flight migration of one
// of them is abandoned).  Lane l looks at slots l and 32 + l.
__device__ __forceinline__ void coop_finish(const Ctx &x, Cnt &cn, int i) {
    const int n = x.nrun[i];
    const uint32_t nf = x.nf[i];
    uint4 *p = slot_ptr(x, i, 0);
    const int q0 = x.lane, q1 = x.lane + 32;
    const bool v0 = q0 < n, v1 = q1 < n;
    const uint4 a0 = v0 ? p[q0] : make_uint4(0, 0, 0, 0);
    const uint4 a1 = v1 ? p[q1] : make_uint4(0, 0, 0, 0);
    const bool f0 = v0 && sl_fin(a0) == nf, f1 = v1 && sl_fin(a1) == nf;
    if (f0) { x.res(a0.x)->finish_us = x.t; x.res(a0.x)->final_instance = (uint16_t)i; }
    if (f1) { x.res(a1.x)->finish_us = x.t; x.res(a1.x)->final_instance = (uint16_t)i; }
    const uint32_t m0 = __ballot_sync(kFull, f0), m1 = __ballot_sync(kFull, f1);
    // each finishing request is booked by the lane that holds it, in turn
#pragma unroll 1
    for (uint64_t m = ((uint64_t)m1 << 32) | m0; m; m &= m - 1) {
        const int l = __ffsll((long long)m) - 1;
        if (x.lane == (l & 31)) {
            const uint4 a = l & 32 ? a1 : a0;
            x.free_[i] += sl_blocks(x, i, a);
            cnt_dec(x, i, (int)sl_tier(a));
            x.hist[i * x.TH + sl_rho(a)]--;
            if (MT_RARE(x.mrole[i] == MIG_SRC && x.mreq[i] == a.x)) abort_mig(x, cn, i, 1);
        }
        __syncwarp();
    }
    const bool k0 = v0 && !f0, k1 = v1 && !f1;
    // places of the survivors: their old ones less the finishers before them
    const uint32_t below = (1u << x.lane) - 1u;
    const int p0 = q0 - __popc(m0 & below), p1 = q1 - __popc(m0) - __popc(m1 & below);
    const uint32_t fm = __reduce_min_sync(kFull, min(k0 ? sl_fin(a0) : kNone, k1 ? sl_fin(a1) : kNone));
    __syncwarp();
    if (k0 && p0 != q0) p[p0] = a0;  // only the records that move are written
    if (k1 && p1 != q1) p[p1] = a1;
    const uint32_t nfin = __popc(m0) + __popc(m1);
    cn.finished += nfin;
    if (x.lane == 0) {
        x.nrun[i] = (uint8_t)(n - (int)nfin);
        x.minfin[i] = fm;
    }
    __syncwarp();
}

// One copy stage at the end of an iteration of migration source s (nothing
// to do if a finish has just abandoned its migration), single thread: up to S
// of the request's blocks are reserved on the destination (abandoning the
// migration if they do not fit).  Returns whether all of them are copied and
// the request can commit there now (Sec. 3.5, Fig. 4): coop_commit must follow.
__device__ __forceinline__ bool stage_copy(const Ctx &x, Cnt &cn, int s) {
    if (x.mrole[s] != MIG_SRC) return false;
    const int d = x.mpeer[s];
    const int blocks = sl_blocks(x, s, x.mslot[s]);
    const int cp = x.mcopied[s];
    const int cc = min(x.S, blocks - cp);
    if (MT_RARE(x.free_[d] < cc)) {
        abort_mig(x, cn, s, 1);
        return false;
    }
    x.free_[d] -= cc;
    x.resv[d] += cc;
    x.mcopied[s] = cp + cc;
    return cp + cc == blocks && (int)x.nrun[d] < x.Bmax;
}

// The running records of instance s, lane l holding slots l and 32 + l.
struct Slots2 {
    uint4 a0, a1;
};
__device__ __forceinline__ Slots2 load_slots(const Ctx &x, int s) {
    const int n = x.nrun[s];
    const uint4 *p = slot_ptr(x, s, 0);
    const uint4 none = make_uint4(kNone, 0, 0, 0);
    return Slots2{x.lane < n ? p[x.lane] : none, x.lane + 32 < n ? p[x.lane + 32] : none};
}

// Commits the fully copied request of source s, whole warp: finds its slot
// among the records `v`, closes the gap and takes the survivors' minimum; the
// lane that owns s books.
__device__ __forceinline__ void coop_commit(const Ctx &x, Cnt &cn, int s, int owner, const Slots2 &v) {
    const uint32_t rid = x.mreq[s];
    const int n = x.nrun[s];
    uint4 *p = slot_ptr(x, s, 0);
    const int q0 = x.lane, q1 = x.lane + 32;
    const uint32_t h0 = __ballot_sync(kFull, q0 < n && v.a0.x == rid);
    const uint32_t h1 = __ballot_sync(kFull, q1 < n && v.a1.x == rid);
    const int pos = h0 ? __ffs(h0) - 1 : (h1 ? 32 + __ffs(h1) - 1 : -1);
    if (MT_RARE(pos < 0)) {
        if (x.lane == 0) cn.status = SIM_ERR_INTERNAL;
    } else {
        const uint32_t fm = __reduce_min_sync(
            kFull, min(q0 < n && q0 != pos ? sl_fin(v.a0) : kNone, q1 < n && q1 != pos ? sl_fin(v.a1) : kNone));
        if (q0 < n && q0 > pos) p[q0 - 1] = v.a0;
        if (q1 < n && q1 > pos) p[q1 - 1] = v.a1;
        if (x.lane == owner) commit_book(x, cn, s, fm);
    }
    __syncwarp();
}

// Copy stage of source s, then its commit if it is due, whole warp (steps at
// one time, where the oracle orders instances by index).
__device__ __forceinline__ void coop_stage(const Ctx &x, Cnt &cn, int s) {
    int commit = 0;
    if (x.lane == 0) commit = stage_copy(x, cn, s) ? 1 : 0;
    if (__shfl_sync(kFull, commit, 0)) coop_commit(x, cn, s, 0, load_slots(x, s));
}

// a[j] for a run-time j without dynamic indexing (the array stays in registers)
template <int C>
__device__ __forceinline__ uint32_t pick_c(const uint32_t (&a)[C], int j) {
    uint32_t v = a[0];
#pragma unroll
    for (int k = 1; k < C; ++k)
        if (j == k) v = a[k];
    return v;
}

// The copy stages of the own sources in `src`, each at its own time et[j]: the
// lanes reserve or abandon together, then the requests that are due commit one
// after another by the whole warp, the next source's records loaded while one
// commits.  Pairs share no state and the log records are held back, so the
// order does not matter.  (256 replicas x 128 instances: a copy takes about
// five stages, 32 pairs per tick; staged one by one they took a third of the
// time.)  Collective.
template <int C>
__device__ __forceinline__ void stage_all(Ctx &x, Cnt &cn, uint32_t src, const uint32_t (&et)[C]) {
    uint32_t due = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        if (!((src >> j) & 1u)) continue;
        x.t = et[j];
        if (stage_copy(x, cn, inst_at(x.lane, j))) due |= 1u << j;
    }
    __syncwarp();
    uint32_t lanes = __ballot_sync(kFull, due != 0), h = 0;
    int l = 0;
    auto next = [&]() -> int {  // the next source that is due, or -1
        if (h == 0) {
            if (lanes == 0) return -1;
            l = __ffs(lanes) - 1;
            lanes &= lanes - 1;
            h = C == 1 ? 1u : __shfl_sync(kFull, due, l);
        }
        const int j = __ffs(h) - 1;
        h &= h - 1;
        return inst_at(l, j);
    };
    int s = next();
    if (s < 0) return;
    Slots2 v = load_slots(x, s);
#pragma unroll 1
    for (;;) {
        const int s2 = next();
        Slots2 v2;
        if (s2 >= 0) v2 = load_slots(x, s2);
        if (C > 1 && x.lane == lane_of(s)) x.t = pick_c<C>(et, num_of(s));
        coop_commit(x, cn, s, lane_of(s), v);
        if (s2 < 0) break;
        s = s2;
        v = v2;
    }
}

// Recompute-style preemption of running request `sl` (holding `blocks` KV
// blocks) on instance i: its KV is freed, it keeps its generated tokens and
// goes back to the front of its tier's bucket.  The caller drops its slot.
__device__ __forceinline__ unsigned int preempt_book(const Ctx &x, Cnt &cn, int i, const uint4 &sl, int blocks) {
    const uint32_t r = sl.x;
    const int tr = (int)sl_tier(sl);
    const uint32_t adv = sl_adv(x, i, sl);
    x.free_[i] += blocks;
    const uint32_t old = x.wmask[i];
    push_front(x, i, tr, r, (sl_c(sl) + adv) | ((sl_left(sl) - adv) << 16));
    if ((old & ((1u << tr) - 1u)) == 0) x.hol[i] = blocks_for(x, sl_c(sl) + adv);  // now head of line
    x.hist[i * x.TH + sl_rho(sl)]--;
    const unsigned int word = bump_pre(x, r);
    atomicAdd(&x.tot[TOT_PRE], 1u);
    if (x.mrole[i] == MIG_SRC && x.mreq[i] == r) abort_mig(x, cn, i, 4);
    return word;  // for pre_fix, which the caller runs later so that nothing waits here
}

// The rare paths below are functions of their own, so that their code and
// registers stay out of the main loop (which instruction fetch and the
// registers per resident warp bound); they rebuild the replica's view from
// shared memory instead of taking it in registers.

// KV growth at the formation of instance i when the running requests need more
// blocks than are free (Sec. 2.2, 3.1).  Single thread.
__device__ __forceinline__ void grow_slow(const Ctx &x, Cnt &cn, int i) {
    const int n = x.nrun[i], fr = x.free_[i];
    const uint32_t ph = x.phase[i], nf = x.nf[i];
    // In running order, a request that needs a block (at most one)
    // takes a free one or preempts the lowest-priority newest running
    // request, possibly itself.  Positions are the list's before this
    // step; removals are applied afterwards.
    uint4 *p = slot_ptr(x, i, 0);
    const uint64_t all = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
    uint64_t alive = all, needs = 0, granted = 0;
    // The requests that need a block now are those whose context reaches
    // a block boundary: rho == -nf (mod T), the ones hist counts.
    const uint32_t target = ph == 0 ? 0u : (uint32_t)x.T - ph;
    // the same pass finds the first victim (lowest priority, then newest):
    // more requests need a block than there are free blocks, so there is one
    int v1 = -1;
    uint32_t vt1 = 0, vr1 = 0;
#pragma unroll 4
    for (int q = 0; q < n; ++q) {
        const uint4 sl = p[q];
        needs |= (uint64_t)(sl_rho(sl) == target) << q;
        const uint32_t ts = sl_tier(sl);
        if (v1 < 0 || ts > vt1 || (ts == vt1 && sl.x > vr1)) { v1 = q; vt1 = ts; vr1 = sl.x; }
    }
    int fb = fr;
    uint32_t pr = kNone;  // the last preempted request and its counter word before the add
    unsigned int pold = 0;
#pragma unroll 1
    for (int q = 0; q < n; ++q) {
        if (!((alive & needs) >> q & 1ull)) continue;
        for (;;) {
            if (fb > 0) { --fb; granted |= 1ull << q; break; }
            int v = -1;
            if (alive == all) {
                v = v1;  // nobody preempted yet: the victim found by the scan
            } else {
                uint32_t vt = 0, vr = 0;
#pragma unroll 1
                for (uint64_t m = alive; m; m &= m - 1) {
                    const int s2 = __ffsll((long long)m) - 1;
                    const uint32_t ts = sl_tier(p[s2]), rs = p[s2].x;
                    if (v < 0 || ts > vt || (ts == vt && rs > vr)) { v = s2; vt = ts; vr = rs; }
                }
            }
            const int vb = blocks_for(x, sl_c(p[v]) + nf - p[v].y) + (int)((granted >> v) & 1ull);
            alive &= ~(1ull << v);
            x.free_[i] = fb;
            if (pr != kNone) pre_fix(x, pr, pold);
            pr = p[v].x;
            pold = preempt_book(x, cn, i, p[v], vb);
            fb = x.free_[i];
            if (v == q) break;
        }
    }
    x.free_[i] = fb;
    int w = 0;
    uint32_t fm = kNone;  // the survivors' next finishing formation
#pragma unroll 1
    for (int q = 0; q < n; ++q) {
        if ((alive >> q) & 1ull) {
            const uint4 sl = p[q];
            if (w != q) p[w] = sl;
            ++w;
            fm = min(fm, sl_fin(sl));
        }
    }
    x.nrun[i] = (uint8_t)w;
    x.minfin[i] = fm;
    if (pr != kNone) pre_fix(x, pr, pold);
}

template <bool SMS>
__device__ __noinline__ bool grow_call(uint4 *node, uint32_t Q, int r, uint32_t t, int i, bool hold) {
    extern __shared__ __align__(16) unsigned char smem[];
    Ctx x;
    bind_ctx<SMS>(x, *reinterpret_cast<const Params *>(smem), smem, node, Q, r, t);
    x.hold = hold;
    Cnt cn;
    cn.held = false;
    grow_slow(x, cn, i);
    return cn.held;
}

// Phase 4: batch formation at idle instance i at x.t (Sec. 2.2, Sec. 3.1):
// (i) KV growth of the running requests, preempting the lowest-priority newest
// one when out of blocks; (ii) admission in (tier, FCFS) order while the head
// of line fits; (iii) the iteration starts.
template <bool SMS, bool LEAN>
__device__ __forceinline__ void inst_form(Ctx &x, Cnt &cn, int i, const Params &p) {
    // the instance's scalars, read together up front (the code below would
    // otherwise reload them after every shared-memory store)
    int n = x.nrun[i];
    int fr = x.free_[i];
    const uint32_t ph = x.phase[i];
    const uint32_t nf = x.nf[i];
    uint32_t wm = x.wmask[i];
    int need = x.hol[i];
    if (!LEAN || n > 0) {  // (nothing is counted where nothing runs)
        const int deficit = x.hist[i * x.TH + (ph == 0 ? 0u : (uint32_t)x.T - ph)];
        if (!MT_RARE(deficit > fr)) {
            fr -= deficit;  // every request that needs a block gets it
        } else {
            if (LEAN) {
                grow_slow(x, cn, i);
            } else {
                cn.held |= grow_call<SMS>(x.node, x.Q, x.r, x.t, i, x.hold);
            }
            n = x.nrun[i];  // preemptions changed the running list, the free blocks, queues and head of line
            fr = x.free_[i];
            wm = x.wmask[i];
            need = x.hol[i];
        }
    }
    // (ii) admission; the waiting mask and the HoL demand follow in registers
    const int n_decode = n;
    int prefill = 0;
#pragma unroll 1
    while (LEAN ? n < x.Bmax : (n < x.Bmax) & (wm != 0u) & (need <= fr)) {
        if (LEAN && !wm) break;
        if (LEAN && need > fr) break;
        const int k = __ffs(wm) - 1;
        const int b = i * x.K + k;
        const uint32_t info = x.hinfo[b];
        const uint32_t r = x.head[b];
        if (MT_RARE(r >= x.Q)) { cn.status = SIM_ERR_INTERNAL; break; }
        const uint4 nd = x.node[r];  // the head leaves its bucket; nd.x is the new head
        x.head[b] = nd.x;
        const uint32_t c = info & 0xFFFFu;
        slot_join_at(x, i, n, r, c, info >> 16, (uint32_t)k, nf, ph);
        ++n;
        fr -= need;
        prefill += (int)c;
        uint32_t hinfo;  // info of the new head of line
        if (nd.x != kNone) {
            x.node[nd.x].z = kNone;
            x.hinfo[b] = nd.y;
            hinfo = nd.y;
        } else {
            x.tail[b] = kNone;
            wm &= ~(1u << k);
            x.wmask[i] = (uint16_t)wm;
            hinfo = wm ? x.hinfo[i * x.K + (__ffs(wm) - 1)] : 0u;
        }
        need = wm ? blocks_for(x, hinfo & 0xFFFFu) : 0;
        x.hol[i] = need;
    }
    x.nrun[i] = (uint8_t)n;
    x.free_[i] = fr;
    // (iii) the iteration starts
    if (n > 0) {
        const long long end = (long long)x.t + p.base + (long long)p.a * prefill + (long long)p.b * n_decode;
        if (MT_RARE(end > 0xFFFFFFFELL)) {
            cn.status = SIM_ERR_OVERFLOW;
            return;
        }
        x.busy[i] = (uint32_t)end;
        const uint4 *sp = slot_ptr(x, i, 0);
#pragma unroll 1
        for (int q = n_decode; q < n; ++q) atomicMin(&x.res(sp[q].x)->first_token_us, (uint32_t)end);
        x.nf[i] = nf + 1u;
        x.phase[i] = ph + 1u == (uint32_t)x.T ? (uint8_t)0 : (uint8_t)(ph + 1u);
        x.pc[i] = 0;
        cn.iterations++;
        cn.member_iterations += (uint64_t)n;
    }
}

// ---- cooperative steps ----------------------------------------------------------
// Lane 0 appends arriving request r (tier k, prompt P, output O) to instance
// best's bucket and updates the instance (Sec. 3.4); the key store is needed
// only if another arrival at the same time is dispatched next.
__device__ __forceinline__ void dispatch_to(const Ctx &x, int best, uint32_t r, int k, uint32_t P,
                                            uint32_t O, bool store_key) {
    if (x.lane == 0) {
        // the destination's scalars, read together; the new key is computed from them
        const int b = best * x.K + k;
        const uint32_t old = x.wmask[best];
        const uint32_t tl = x.tail[b];
        const uint32_t c0 = x.cnt[b];
        int hol = x.hol[best];
        int hr = x.hr[best];
        const int fr = x.free_[best];
        const int nr = x.nrun[best];
        const int hk = x.h[k];
        const uint32_t info = P | (O << 16);
        x.node[r] = make_uint4(kNone, 0u, tl, info);  // appended to bucket (best, k), as push_back
        if (tl != kNone) *reinterpret_cast<uint2 *>(&x.node[tl]) = make_uint2(r, info);
        else { x.head[b] = r; x.hinfo[b] = info; }
        x.tail[b] = r;
        x.wmask[best] = (uint16_t)(old | (1u << k));
        x.cnt[b] = (uint16_t)(c0 + 1u);
        if (c0 == 0) x.hr[best] = hr += hk;                    // tier k now present (Eq. 4)
        if ((old & ((2u << k) - 1u)) == 0) x.hol[best] = hol = blocks_for(x, P);  // becomes head of line
        x.res(r)->dispatch_instance = (uint16_t)best;
        if (store_key) x.key[best] = make_key<false>(x, fr - hol - hr, nr);
    }
}

// Dispatch one arriving request r of tier k with prompt length P (Sec. 3.4).
template <int C>
__device__ __forceinline__ void dispatch_one(const Ctx &x, uint32_t r, int k, uint32_t P, uint32_t O,
                                             uint32_t all) {
    const int best = arg_ext<C>(x, all, true, -1);
    dispatch_to(x, best, r, k, P, O, true);
    __syncwarp();
}

// The next 32 trace records, one per lane: index pb + lane.
struct ArrBuf {
    uint32_t pb, time, tier, po;  // po: prompt length | output length << 16
};

__device__ __forceinline__ void arr_refill(const Ctx &x, ArrBuf &ab, uint32_t cursor) {
    ab.pb = cursor;
    const uint32_t idx = cursor + (uint32_t)x.lane;
    const bool in = idx < x.Q;
    const long long at = x.first() + idx;
    ab.time = in ? x.arrival[at] : kNone;
    ab.tier = in ? (uint32_t)x.tier[at] : 0u;
    ab.po = in ? (uint32_t)x.plen[at] | ((uint32_t)x.olen[at] << 16) : 0u;
}

// Dispatches all arrivals at t, from trace record `cursor` on, tier by tier to
// the instances in `all`; returns their number.  Collective.
template <int C>
__device__ __forceinline__ uint32_t dispatch_many(const Ctx &x, uint32_t cursor, uint32_t all) {
    refresh_keys<C>(x);
    const long long at = x.first();
    uint32_t m = 0;
#pragma unroll 1
    for (;;) {
        const uint32_t j2 = cursor + m + (uint32_t)x.lane;
        const bool in2 = j2 < x.Q;
        const uint32_t e2 = __ballot_sync(kFull, in2 && x.arrival[at + j2] == x.t);
        m += (uint32_t)__popc(e2);
        if (e2 != kFull) break;
    }
#pragma unroll 1
    for (int k = 0; k < x.K; ++k) {
#pragma unroll 1
        for (uint32_t base = 0; base < m; base += 32) {
            const uint32_t j2 = cursor + base + (uint32_t)x.lane;
            const bool mine = base + (uint32_t)x.lane < m;
            const uint32_t tr = mine ? x.tier[at + j2] : 0u;
            const uint32_t P = mine ? x.plen[at + j2] : 0u;
            const uint32_t O = mine ? x.olen[at + j2] : 0u;
            uint32_t bits = __ballot_sync(kFull, mine && tr == (uint32_t)k);
#pragma unroll 1
            while (bits) {
                const int l = __ffs(bits) - 1;
                bits &= bits - 1;
                dispatch_one<C>(x, cursor + base + (uint32_t)l, k, __shfl_sync(kFull, P, l),
                                __shfl_sync(kFull, O, l), all);
            }
        }
    }
    return m;
}

template <int C, bool SMS>
__device__ __noinline__ uint32_t dispatch_call(uint4 *node, uint32_t Q, int r, uint32_t t, uint32_t cursor,
                                               uint32_t all) {
    extern __shared__ __align__(16) unsigned char smem[];
    Ctx x;
    bind_ctx<SMS>(x, *reinterpret_cast<const Params *>(smem), smem, node, Q, r, t);
    return dispatch_many<C>(x, cursor, all);
}

// Phase 2: arrivals at t, tier 0 first, FCFS (trace order) within a tier.
// EXT: draining instances may exist.  Returns the destination of a lone
// arrival, or -1 after several.
template <int C, bool SMS, bool EXT, bool LEAN>
__device__ __forceinline__ int dispatch_phase(Ctx &x, uint32_t &cursor, uint32_t &next_arr, ArrBuf &ab,
                                              const Params &p) {
    uint32_t all = own_mask<C>(x);
    if (EXT && x.drains) {
        // Draining instances (infinite virtual usage, Sec. 3.5) get no
        // dispatch unless every instance drains; then the freest of them
        // does (Sec. 3.4: the least loaded draining one).
        uint32_t live = 0;
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (((all >> j) & 1u) && x.drain[inst_at(x.lane, j)] > x.t) live |= 1u << j;
        if (__any_sync(kFull, live != 0)) all = live;
    }
    int dest = -1;
    const uint32_t off = cursor - ab.pb;
    const uint32_t eq = __ballot_sync(kFull, (uint32_t)x.lane >= off && ab.time == x.t);
    // (an arrival in the buffer's last place may have others at t behind it)
    if (!MT_RARE((eq >> 31) != 0u || (eq & (eq - 1u)) != 0u)) {
        // one arrival at t (the usual case): no tier ordering to do
        const int l = __ffs(eq) - 1;
        const uint32_t k1 = __shfl_sync(kFull, ab.tier, l);
        const uint32_t po = __shfl_sync(kFull, ab.po, l);
        // the freest instance from keys computed in registers (nothing reads
        // the key array before the next refresh)
        int bv = INT_MIN, bi = -1;
#pragma unroll
        for (int j = 0; j < C; ++j) {
            const int i = inst_at(x.lane, j);
            if ((all >> j) & 1u) {
                const int kk = make_key<!LEAN>(x, fnum(x, i), x.nrun[i]);
                if (bi < 0 || kk > bv) { bv = kk; bi = i; }
            }
        }
        const int m = __reduce_max_sync(kFull, bv);
        const int best = __reduce_min_sync(kFull, (bi >= 0 && bv == m) ? bi : INT_MAX);
        dispatch_to(x, best, ab.pb + (uint32_t)l, (int)k1, po & 0xFFFFu, po >> 16, false);
        __syncwarp();
        dest = best;
        cursor += 1u;
    } else {
        if (LEAN) {
            cursor += dispatch_many<C>(x, cursor, all);
        } else {
            cursor += dispatch_call<C, SMS>(x.node, x.Q, x.r, x.t, cursor, all);
        }
    }
    if (MT_RARE(cursor - ab.pb >= 32u)) arr_refill(x, ab, cursor);
    next_arr = __shfl_sync(kFull, ab.time, (int)(cursor - ab.pb));
    return dest;
}

// Auto-scaling signal at a tick (Sec. 3.6): the mean normal-priority freeness
// (Eq. 1 without the headroom term, Sec. 3.4) over the instances that are not
// draining, compared exactly with scale_out_num / scale_den and
// scale_in_num / scale_den.  Each F_normal = (free - HoL) / max(B, 1) is scaled
// by L = lcm(1, ..., Bmax), so S = L * sum F_normal is an exact 128-bit
// integer (|S| < 2^117), and mean < x / D  <=>  S * D < x * n * L.  Collective.
template <int C>
__device__ __forceinline__ void autoscale_tick(const Ctx &x, const Params &p) {
    const __int128 L = (__int128)(((unsigned __int128)p.lcm_hi << 64) | p.lcm_lo);
    __int128 sum = 0;
    int n = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (i < x.N && !(x.drains && x.drain[i] <= x.t)) {
            const int num = x.free_[i] - x.hol[i];
            const int den = max((int)x.nrun[i], 1);
            sum += (__int128)num * (L / den);
            ++n;
        }
    }
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
        const unsigned long long lo = __shfl_xor_sync(kFull, (unsigned long long)sum, sh);
        const unsigned long long hi = __shfl_xor_sync(kFull, (unsigned long long)((unsigned __int128)sum >> 64), sh);
        sum += (__int128)(((unsigned __int128)hi << 64) | lo);
    }
    n = __reduce_add_sync(kFull, n);
    if (x.lane == 0 && n > 0) {
        const __int128 lhs = sum * p.scale_den;
        if (lhs < (__int128)p.scale_out_num * n * L) {
            x.tot[TOT_OUT]++;
            log_ev(x, SIM_EV_SCALE_OUT, kNone, 255, 255, 0);
        } else if (lhs > (__int128)p.scale_in_num * n * L) {
            x.tot[TOT_IN]++;
            log_ev(x, SIM_EV_SCALE_IN, kNone, 255, 255, 0);
        }
    }
    __syncwarp();
}

// Whether the freeness of d exceeds that of s by at least theta (Sec. 3.5).
__device__ __forceinline__ bool over_theta(const Ctx &x, int s, int d, int theta_num, int theta_den) {
    const long long ns = fnum(x, s), ds = max((int)x.nrun[s], 1);
    const long long nd = fnum(x, d), dd = max((int)x.nrun[d], 1);
    return (long long)theta_den * (nd * ds - ns * dd) >= (long long)theta_num * dd * ds;
}

// The newest request of the lowest-priority bucket of s, which has waiting
// requests, moves to d at once (no KV to copy).  Single thread; k: its place in the log.
__device__ __forceinline__ void move_queued(const Ctx &x, Cnt &cn, int s, int d, uint32_t k) {
    const int tr = 31 - __clz((unsigned)x.wmask[s]);
    uint32_t info = 0;
    const uint32_t r = pop_back(x, s, tr, info, cn.status);
    if (MT_RARE(r == kNone)) return;
    refresh_hol(x, s);
    cnt_dec(x, s, tr);
    const uint32_t old = x.wmask[d];
    push_back(x, d, tr, r, info);
    cnt_inc(x, d, tr);
    if ((old & ((2u << tr) - 1u)) == 0) x.hol[d] = blocks_for(x, info & 0xFFFFu);
    bump_mig(x, r);
    if (k < (uint32_t)x.cap) *x.log(k) = make_uint4(x.t, r, ((uint32_t)s << 16) | ((uint32_t)d << 24), SIM_EV_QUEUED);
}

// The running request of s (its records: v) with the lowest priority, then the
// fewest blocks, then the newest, starts its staged copy to d if its blocks
// fit there.  Collective; k: its place in the log.
__device__ __forceinline__ bool start_copy(const Ctx &x, int s, int d, const Slots2 &v, uint32_t k) {
    const int n = x.nrun[s];
    const bool v0 = x.lane < n, v1 = x.lane + 32 < n;
    const int k0 = v0 ? (int)((sl_tier(v.a0) << 16) | (0xFFFFu - (uint32_t)sl_blocks(x, s, v.a0))) : -1;
    const int k1 = v1 ? (int)((sl_tier(v.a1) << 16) | (0xFFFFu - (uint32_t)sl_blocks(x, s, v.a1))) : -1;
    const int km = __reduce_max_sync(kFull, max(k0, k1));
    if (km < 0) return false;  // nothing runs there
    const int blocks = (int)(0xFFFFu - ((uint32_t)km & 0xFFFFu));
    if (MT_RARE(x.free_[d] < blocks)) return false;
    const bool c0 = k0 == km, c1 = k1 == km;
    const uint32_t rid = __reduce_max_sync(kFull, max(c0 ? v.a0.x : 0u, c1 ? v.a1.x : 0u));
    const bool b0 = c0 && v.a0.x == rid;
    if (b0 || (c1 && v.a1.x == rid)) {  // the lane that holds it books
        x.mrole[s] = MIG_SRC;
        x.mpeer[s] = (uint8_t)d;
        x.mreq[s] = rid;
        x.mcopied[s] = 0;
        x.mslot[s] = b0 ? v.a0 : v.a1;
        x.mrole[d] = MIG_DST;
        x.mpeer[d] = (uint8_t)s;
        if (k < (uint32_t)x.cap)
            *x.log(k) = make_uint4(x.t, rid, (uint32_t)(blocks & 0xFFFF) | ((uint32_t)s << 16) | ((uint32_t)d << 24),
                                   SIM_EV_START);
    }
    return true;
}

// Phase 3 with theta > 0 and nothing draining: the freeness order is fixed for
// the tick, so every lane ranks its instances by ascending (sources) and
// descending freeness (destinations, lowest index first among equals in both)
// once, and pair r is then (source r, destination r) as long as the threshold
// holds; theta > 0 keeps the two sides apart.  The threshold and the moves of
// queued requests are done by one lane per pair, up to 32 at once; running
// candidates are found pair by pair by the whole warp, the next source's
// records loaded meanwhile.  A source whose candidate does not fit leaves its
// destination to the next source.  Returns whether a staged copy started.
// (A serial search took about 2,500 cycles per pair, two reductions for each
// side, the threshold and one memory round trip; 256 replicas x 128 instances
// start 32 copies per tick.)
template <int C>
__device__ __forceinline__ bool ranked_tick(const Ctx &x, Cnt &cn, int theta_num, int theta_den) {
    int *sk = reinterpret_cast<int *>(x.tset);
    const int np = (x.N + 3) & ~3;
    uint8_t *lo = reinterpret_cast<uint8_t *>(sk + np), *hi = lo + np;
    int key[C], lt[C], eqb[C], eqa[C];
    uint32_t el = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        key[j] = INT_MIN;  // below every freeness key: not eligible
        if (i < x.N && x.mrole[i] == MIG_NONE) {
            key[j] = make_key<C != 2>(x, fnum(x, i), x.nrun[i]);
            el |= 1u << j;
        }
        if (i < np) sk[i] = key[j];
        lt[j] = eqb[j] = eqa[j] = 0;
    }
    const int nel = __reduce_add_sync(kFull, __popc(el));
    __syncwarp();
    if (nel < 2) return false;
#pragma unroll 1
    for (int m = 0; m < np; m += 4) {
        const uint4 w = *reinterpret_cast<const uint4 *>(sk + m);
        const int kk[4] = {(int)w.x, (int)w.y, (int)w.z, (int)w.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                lt[j] += kk[u] < key[j] ? 1 : 0;
                if (kk[u] == key[j]) {
                    eqb[j] += m + u < inst_at(x.lane, j) ? 1 : 0;
                    eqa[j] += m + u > inst_at(x.lane, j) ? 1 : 0;
                }
            }
    }
#pragma unroll
    for (int j = 0; j < C; ++j)
        if ((el >> j) & 1u) {
            const int below = lt[j] - (np - nel);  // eligible ones
            lo[below + eqb[j]] = (uint8_t)inst_at(x.lane, j);
            hi[nel - 1 - below - eqa[j]] = (uint8_t)inst_at(x.lane, j);
        }
    __syncwarp();
    bool started = false;
    int k = 0, q = 0;  // next source and destination
#pragma unroll 1
    for (;;) {
        int s = 0, d = 0;
        bool ok = k + x.lane < nel;  // q <= k
        if (ok) {
            s = lo[k + x.lane];
            d = hi[q + x.lane];
            ok = sk[s] < sk[d] && over_theta(x, s, d, theta_num, theta_den);  // by the first: not moved yet
        }
        const uint32_t okm = __ballot_sync(kFull, ok);
        const int cnt = okm == kFull ? 32 : __ffs(~okm) - 1;
        if (cnt == 0) break;
        const bool waits = x.lane < cnt && x.wmask[s] != 0;
        const uint32_t wm = __ballot_sync(kFull, waits);
        uint32_t run = (cnt == 32 ? kFull : (1u << cnt) - 1u) & ~wm;
        const uint32_t base = x.tot[TOT_LOG];
        int done = cnt;  // pairs of this batch that move
        if (run) {
            Slots2 v = load_slots(x, lo[k + __ffs(run) - 1]);
#pragma unroll 1
            do {
                const int e = __ffs(run) - 1;
                run &= run - 1;
                Slots2 v2;
                if (C != 2 && run) v2 = load_slots(x, lo[k + __ffs(run) - 1]);
                if (!start_copy(x, lo[k + e], hi[q + e], v, base + (uint32_t)e)) {
                    done = e;
                    break;
                }
                started = true;
                if (C == 2 && run) v2 = load_slots(x, lo[k + __ffs(run) - 1]);
                v = v2;
            } while (run);
        }
        if (waits && x.lane < done) move_queued(x, cn, s, d, base + (uint32_t)x.lane);
        __syncwarp();
        if (x.lane == 0) {
            const uint32_t moved = done == 32 ? kFull : (1u << done) - 1u;
            x.tot[TOT_LOG] = base + (uint32_t)done;
            x.tot[TOT_MIG] += (uint32_t)__popc(wm & moved);
            x.tot[TOT_START] += (uint32_t)__popc(~wm & moved);
        }
        __syncwarp();
        if (done == cnt && cnt < 32) break;
        q += done;
        k += done < cnt ? done + 1 : cnt;
    }
    return started;
}

// Phase 3: periodic rebalancing between low- and high-freeness instances
// (Sec. 3.5).  Returns whether a staged copy started.
template <int C, bool EXT>
__device__ __forceinline__ bool migration_tick(const Ctx &x, Cnt &cn, int theta_num, int theta_den) {
    if (!MT_RARE(theta_num == 0) && !(EXT && x.drains)) return ranked_tick<C>(x, cn, theta_num, theta_den);
    // Pair by pair: draining instances come first and without the threshold,
    // and with theta = 0 equal freeness pairs up too.
    refresh_keys<C>(x);
    uint32_t el = 0, dr = 0;  // eligible (not migrating); draining
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (i < x.N && x.mrole[i] == MIG_NONE) el |= 1u << j;
        if (EXT && i < x.N && x.drains && x.drain[i] <= x.t) dr |= 1u << j;
    }
    bool started = false;
    for (;;) {
        const int nel = __reduce_add_sync(kFull, __popc(el));
        if (nel < 2) break;
        // A draining instance has infinite virtual usage (Sec. 3.5): it is the
        // least free (lowest index among several), passes the threshold
        // against any other instance, and is never a destination.
        int s;
        const uint32_t dl = EXT ? __ballot_sync(kFull, (el & dr) != 0) : 0u;
        if (dl) {
            const uint32_t bits = el & dr;
            s = __reduce_min_sync(kFull, bits ? inst_at(x.lane, __ffs(bits) - 1) : INT_MAX);
        } else {
            s = arg_ext<C>(x, el, false, -1);
        }
        const int d = arg_ext<C>(x, el & ~dr, true, s);
        if (d < 0) break;
        if (!dl && !over_theta(x, s, d, theta_num, theta_den)) break;
        const bool has_wait = x.wmask[s] != 0;
        const uint32_t at = x.tot[TOT_LOG];
        const Slots2 v = load_slots(x, s);
        __syncwarp();
        bool moved = has_wait;
        if (has_wait) {
            if (x.lane == 0) {
                move_queued(x, cn, s, d, at);
                x.tot[TOT_MIG]++;
            }
        } else if (start_copy(x, s, d, v, at)) {
            if (x.lane == 0) x.tot[TOT_START]++;
            moved = started = true;
        }
        if (moved && x.lane == 0) x.tot[TOT_LOG] = at + 1u;
        if (x.lane == lane_of(s)) el &= ~(1u << num_of(s));
        if (moved && x.lane == lane_of(d)) el &= ~(1u << num_of(d));
        __syncwarp();
    }
    return started;
}

// The tick as a function of its own: bit 0, a staged copy started; bit 1, an
// inconsistency on this lane.
template <int C, bool SMS, bool EXT>
__device__ __noinline__ int tick_call(uint4 *node, uint32_t Q, int r, uint32_t t) {
    extern __shared__ __align__(16) unsigned char smem[];
    const Params &p = *reinterpret_cast<const Params *>(smem);
    Ctx x;
    bind_ctx<SMS>(x, p, smem, node, Q, r, t);
    Cnt cn;
    cn.status = SIM_REPLICA_RUNNING;
    const bool started = migration_tick<C, EXT>(x, cn, p.theta_num, p.theta_den);
    return (started ? 1 : 0) | (cn.status < 0 ? 2 : 0);
}

// The number of distinct times et[j] < t1 over the warp, for a window
// [tb, t1), in two parts: distinct_times when it opens, distinct_count when it
// closes.  Collective.  One instance per lane: the lanes that share a time form a
// group (match), which nothing waits for until the window closes.  (A count in
// shared memory, as below, cost 4 KB or 1 KB per warp and 160 instructions more:
// 1,024 x 16 at 0.85 load with 20,000 requests 82.6 -> 78.4 ms, 1,024 x 24, four
// blocks per SM instead of three, 19.3 -> 10.7 ms, one 4-instance cluster 42.2 ->
// 40.1 ms, 3,840 x 32 16.9 -> 16.4 ms.)  Several: every instance writes its index
// into a byte that its time selects and reads it back: one index per byte wins
// and counts, nothing needs clearing.  When the scratch has a byte for every
// microsecond of the window the others have the winner's time; in a longer window
// the byte is hashed, the winner's time is compared, and the instances that met
// another time try again without the winners (at least one per byte leaves each
// round).
template <int C>
__device__ __forceinline__ uint32_t distinct_times(const Ctx &x, uint32_t tb, uint32_t t1, const uint32_t (&et)[C]) {
    if constexpr (C == 1) return __match_any_sync(kFull, et[0] < t1 ? et[0] : kNone);
    uint8_t *set = reinterpret_cast<uint8_t *>(x.tset);
    uint32_t fresh = 0;
    if (!MT_RARE(t1 - tb > 1u << x.set_bits)) {
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (et[j] < t1) set[et[j] - tb] = (uint8_t)inst_at(x.lane, j);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (et[j] < t1) fresh += set[et[j] - tb] == (uint8_t)inst_at(x.lane, j) ? 1u : 0u;
    } else {
        uint32_t todo = 0, at[C], win[C];
#pragma unroll
        for (int j = 0; j < C; ++j) {
            todo |= (et[j] < t1 ? 1u : 0u) << j;
            at[j] = ((et[j] - tb) * 0x9E3779B1u) >> (32 - x.set_bits);
        }
#pragma unroll 1
        while (__any_sync(kFull, todo != 0)) {
#pragma unroll
            for (int j = 0; j < C; ++j)
                if ((todo >> j) & 1u) set[at[j]] = (uint8_t)inst_at(x.lane, j);
            __syncwarp();
#pragma unroll
            for (int j = 0; j < C; ++j) {
                win[j] = ((todo >> j) & 1u) ? set[at[j]] : 0u;
                if (((todo >> j) & 1u) && win[j] == (uint32_t)inst_at(x.lane, j)) {
                    ++fresh;
                    todo &= ~(1u << j);
                }
            }
#pragma unroll
            for (int j = 0; j < C; ++j)
#pragma unroll
                for (int k = 0; k < C; ++k) {  // instance win[j] is number k of its lane
                    const uint32_t tw = __shfl_sync(kFull, et[k], lane_of((int)win[j]));
                    if (num_of((int)win[j]) == k && tw == et[j]) todo &= ~(1u << j);
                }
        }
    }
    return __reduce_add_sync(kFull, fresh);
}

// The count; in: the lane's instance had an event in the window (C = 1).
template <int C>
__device__ __forceinline__ uint32_t distinct_count(const Ctx &x, uint32_t u, bool in) {
    return C == 1 ? (uint32_t)__popc(__ballot_sync(kFull, in && __ffs(u) - 1 == x.lane)) : u;
}

__device__ __forceinline__ void copy16(unsigned char *dst, const unsigned char *src, uint32_t bytes, int lane) {
#pragma unroll 1
    for (uint32_t o = (uint32_t)lane * 16u; o < bytes; o += 512u)
        *reinterpret_cast<uint4 *>(dst + o) = *reinterpret_cast<const uint4 *>(src + o);
}

// Phase 1 at x.t for the instances in `mask` (bit j = the lane's instance j)
// whose iteration ends now, ascending index.  Collective.
template <int C>
__device__ __forceinline__ void complete_all(const Ctx &x, Cnt &cn, uint32_t mask) {
    uint32_t hits = 0;
#pragma unroll
    for (int j = 0; j < C; ++j)
        if (((mask >> j) & 1u) && x.busy[inst_at(x.lane, j)] == x.t) hits |= 1u << j;
#pragma unroll 1
    for (int j = 0; j < C; ++j)
        for (uint32_t lanes = __ballot_sync(kFull, (hits >> j) & 1u); lanes; lanes &= lanes - 1) {
            const int i = inst_at(__ffs(lanes) - 1, j);
            int fp = 0;
            if (x.lane == 0) fp = inst_complete_head(x, i);
            const bool src = x.mrole[i] == MIG_SRC;
            if (__shfl_sync(kFull, fp, 0)) coop_finish(x, cn, i);
            if (src) coop_stage(x, cn, i);
        }
}

// Phase 4 at x.t for the idle instances in `mask` that have work, ascending
// index, on lane 0.  Collective.
template <int C, bool SMS, bool LEAN>
__device__ __forceinline__ void form_all(Ctx &x, Cnt &cn, uint32_t mask, const Params &p) {
    uint32_t want = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int i = inst_at(x.lane, j);
        if (((mask >> j) & 1u) && x.busy[i] == kNone && (x.nrun[i] | x.wmask[i]) != 0) want |= 1u << j;
    }
#pragma unroll 1
    for (int j = 0; j < C; ++j)
        for (uint32_t lanes = __ballot_sync(kFull, (want >> j) & 1u); lanes; lanes &= lanes - 1)
            if (x.lane == 0) inst_form<SMS, LEAN>(x, cn, inst_at(__ffs(lanes) - 1, j), p);
    __syncwarp();
}

// The events of a window [tb, t1) that can be taken in the next round, bit j =
// the lane's instance j, at time et[j].  A window is short enough that every
// instance ends at most one iteration, and instances interact only as the two
// ends of a migration: the source's event (finish, copy stage, commit or
// abort) reads and changes the destination, the destination's event changes
// nothing at the source.  So the instances outside migrations and the earlier
// event of every pair are taken together, each at its own time (`first`), and
// the later events of the pairs in a second round (`later`: there are some).
// A pair whose two iterations end at the same time (`same`) is stepped as the
// oracle orders one time: both ends, then both formations.  `wake_lo`,
// `wake_hi`: idle destinations of a source in `first`, which may be able to
// form a batch once the source's event is done, before the source forms its
// own (lower index) or after it.
template <int C>
struct Window {
    uint32_t first, same, wake_lo, wake_hi;
    bool later;
};
template <int C>
__device__ __forceinline__ Window<C> classify(const Ctx &x, uint32_t t1, uint32_t (&et)[C]) {
    Window<C> w{0, 0, 0, 0, false};
#pragma unroll
    for (int j = 0; j < C; ++j) {
        // without branches, the peer's busy time read in any case: a divergent branch
        // costs more than the read (256 x 128 40.8 -> 39.1 ms, 1,024 x 16 9.12 -> 8.74)
        const int i = inst_at(x.lane, j), ii = i < x.N ? i : 0;
        const int role = x.mrole[ii], peer = x.mpeer[ii];
        const uint32_t pb = x.busy[peer], t = et[j];
        const bool in = i < x.N && t < t1, pair = role != MIG_NONE;
        const bool wake = i < x.N && t == kNone && role == MIG_DST && pb < t1;
        w.first |= (in && (!pair || pb > t) ? 1u : 0u) << j;
        w.same |= (in && pair && pb == t ? 1u : 0u) << j;
        w.later = w.later || (in && pair && pb < t);
        w.wake_lo |= (wake && i < peer ? 1u : 0u) << j;
        w.wake_hi |= (wake && i > peer ? 1u : 0u) << j;
        et[j] = wake ? pb : t;
    }
    return w;
}

// Lists the own instances in `sel` of all lanes, ascending, with their times
// et[j], in the scratch of distinct_times ({time, instance}); returns their
// number.  Collective.  Formations are taken from the list, so that 32 lanes
// share them evenly whichever lanes own the instances: with two instances
// per lane and a dozen formations in a window, two of them usually share a
// lane, with eight per lane four or five do (97 x 33 11.1 -> 10.6 ms, 256 x 128
// 43.3 -> 41.7 ms, 64 x 256 65.1 -> 63.8 ms).  The loop of many replicas does
// without: 112.5 -> 118.5 ms on 8,192 x 64.
template <int C>
__device__ __forceinline__ uint32_t list_own(const Ctx &x, uint32_t sel, const uint32_t (&et)[C]) {
    const uint32_t below = (1u << x.lane) - 1u;
    uint32_t pos = 0, total = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const uint32_t m = __ballot_sync(kFull, (sel >> j) & 1u);
        pos += (uint32_t)__popc(m & below);
        total += (uint32_t)__popc(m);
    }
    uint2 *list = reinterpret_cast<uint2 *>(x.tset);
#pragma unroll
    for (int j = 0; j < C; ++j)
        if ((sel >> j) & 1u) list[pos++] = make_uint2(et[j], (uint32_t)inst_at(x.lane, j));
    __syncwarp();
    return total;
}

// Advances the instances (one per lane, in no migration) through windows in
// which every iteration that ends is a quiet one, with the instances' state in
// registers: nothing finishes, the running requests get the blocks they need,
// and no waiting request can join, so the next iteration takes the same time
// with the same members.  Stops at the first window with another event, at tg
// or near the step limit, and returns the earliest iteration end then.
// Collective.  A window takes a reduction, two votes and three shared accesses
// instead of the phases below: one lightly loaded 4-instance cluster (2,000
// requests), most of whose windows are quiet, went from 59.9 to 45.4 ms.
__device__ __forceinline__ uint32_t run_quiet(const Ctx &x, Cnt &cn, uint32_t &busy, uint32_t tb, uint32_t tg,
                                              uint32_t max_steps, uint32_t &tmax, const Params &p) {
    const int i = x.lane < x.N ? x.lane : 0;
    const uint32_t n = x.nrun[i], minfin = x.minfin[i], dur = (uint32_t)p.base + (uint32_t)p.b * n;
    const bool waits = x.wmask[i] != 0 && (int)n < x.Bmax;
    const int need = x.hol[i];
    const uint8_t *hist = x.hist + i * x.TH;
    uint32_t nf = x.nf[i], ph = x.phase[i], done = 0;
    int fr = x.free_[i], grow = 0;
    bool quiet = false;
    // whether the end of the running iteration is quiet, and the blocks its successor takes
    auto look = [&]() {
        grow = hist[ph == 0 ? 0u : (uint32_t)x.T - ph];
        quiet = (nf != minfin) & (grow <= fr) & !(waits & (need <= fr - grow)) & (busy < 0xFFFFFFFEu - dur);
    };
    look();
    while (tb < tg && max_steps - cn.steps > (uint32_t)x.N) {
        const uint32_t t1 = (uint32_t)min((unsigned long long)tg, (unsigned long long)tb + (uint32_t)p.base);
        const bool ends = busy < t1;
        if (__any_sync(kFull, ends && !quiet)) break;
        const uint32_t et[1] = {busy};
        const uint32_t group = distinct_times<1>(x, tb, t1, et);
        if (ends) {
            ++done;
            tmax = max(tmax, busy);
            fr -= grow;
            ++nf;
            ph = ph + 1u == (uint32_t)x.T ? 0u : ph + 1u;
            busy += dur;
            look();
        }
        cn.steps += distinct_count<1>(x, group, ends);
        tb = __reduce_min_sync(kFull, busy);
    }
    if (done) {
        x.busy[i] = busy;
        x.free_[i] = fr;
        x.nf[i] = nf;
        x.phase[i] = (uint8_t)ph;
        cn.iterations += done;
        cn.member_iterations += (uint64_t)done * n;
    }
    __syncwarp();
    return tb;
}

// The persistent simulation kernel: each warp repeatedly takes a replica and
// advances it by up to p.max_steps event times; C = instances per lane.
//
// Between two global events (the next arrival, the next migration tick) the
// instances that are in no migration do not interact, and an iteration lasts
// at least `base` microseconds.  So in a window [tmin, min(T_g, tmin + base))
// every instance ends at most one iteration, and each lane advances its own
// instances (an O(1) iteration end + batch formation), the two ends of a
// migration in the order of their events (classify); every step at a global
// event is advanced by the warp in the oracle's order.
//
// EXT: the variant that also handles draining instances and the auto-scaling
// signal (the other variant compiles that code out).  MANY: the loop for more
// replicas than a few warps per SM (choose_plan).  What bounds the two differs:
// with few warps each replica's dependent chain, so the loop without MANY has
// a straight path per kind of pass; with many, instruction fetch and registers
// (64 instances: 14 % less code took 161 to 131 ms, 18 instead of 16 warps
// another 14 %), so the MANY loop has one copy of every phase.
//
// Resident warps against registers, same-box A/B.  Two instances per lane,
// records in HBM: a bound of 10 blocks compiles to 96 registers (few spills),
// and shared memory then holds 9 blocks of two warps: 113.6 ms on 8,192
// replicas x 64 instances x 4,000 requests, against 131.0 ms with 8 blocks at
// 124 registers.  (10 resident blocks, with 1 KB less of scratch per warp:
// 110.4 ms; 12 blocks would need 80 registers, which spills.)  One instance
// per lane: 8 blocks (128 registers); 10 and 12 blocks were 5 % slower on 3,840 x
// 32 x 1,000.  Four per lane, records in HBM: the loop of few takes 181 registers
// (8 warps per SM); MANY is the same loop at a bound of 6 blocks (168 registers, 12
// warps), for the replica counts that take fewer waves then (choose_plan).
template <int C, bool SMS, bool EXT, bool MANY>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, !MANY ? 4 : C == 4 ? 6 : C == 2 ? 10 : 8) k_run(Params p) {
    // At 96 registers there is no room for values kept across calls: the rare
    // paths stay inline (116 ms instead of 196 on the 64-instance sweep), and
    // copy stages go source by source.
    constexpr bool LEAN = MANY && C == 2;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *magic = reinterpret_cast<unsigned long long *>(smem + kParamBytes);
    for (int d = threadIdx.x; d <= 64; d += blockDim.x)
        magic[d] = d < 2 ? 0ull : ~0ull / (unsigned long long)d + 1ull;
    if (threadIdx.x == 0) *reinterpret_cast<Params *>(smem) = p;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t slot_bytes = SMS ? (uint32_t)p.N * (uint32_t)p.Bmax * 16u : 0u;
    for (;;) {
        int r = 0;
        if (lane == 0) {
            r = atomicAdd(p.work, 1);
            if (p.order && r < p.R) r = p.order[r];
        }
        r = __shfl_sync(kFull, r, 0);
        if (r >= p.R) break;
        if (p.rep[r].status != SIM_REPLICA_RUNNING) continue;
        unsigned char *gblob = p.blobs + (size_t)r * p.L.bytes;
        const long long o = p.offsets[r];
        Ctx x;
        // The state's address stays in a register (the compiler would rather
        // compute it again at every use: 130 instead of 116 ms on the 64-instance
        // sweep, 9.54 instead of 9.43 ms on 1,024 x 16).
        uint32_t zero = 0;
        asm volatile("" : "+r"(zero));
        bind_ctx<SMS, (C > 1)>(x, p, smem + zero, p.node + o, (uint32_t)(p.offsets[r + 1] - o), r, p.rep[r].t);
        if (!EXT) x.drains = 0;
        unsigned char *blob = x.busy.base - p.L.inst;
        uint4 *g_slots = p.slots + (size_t)r * p.N * p.Bmax;
        copy16(blob, gblob, p.L.bytes, lane);
        if (SMS)
            copy16(reinterpret_cast<unsigned char *>(x.slots), reinterpret_cast<const unsigned char *>(g_slots),
                   slot_bytes, lane);
        __syncwarp();
        uint32_t tmax = x.t;  // latest event time this lane has processed (the replica's: max over lanes)
        Cnt cn;
        cn.finished = p.rep[r].finished;
        cn.steps = 0;
        cn.iterations = 0;
        cn.member_iterations = 0;
        cn.status = SIM_REPLICA_RUNNING;
        cn.held = false;
        uint32_t cursor = p.rep[r].cursor;
        uint32_t next_tick = p.rep[r].next_tick;
        x.hold = false;
        // whether some instance may be in a migration (kept current: set by a tick
        // that starts one, taken back when a window closes without any)
        bool mig = false;
        for (int i = lane; i < x.N; i += 32) mig = mig || x.mrole[i] != MIG_NONE;
        mig = __any_sync(kFull, mig);
        ArrBuf ab;
        arr_refill(x, ab, cursor);
        uint32_t next_arr = __shfl_sync(kFull, ab.time, 0);
        if constexpr (MANY && C <= 2) {
            const uint32_t max_steps = p.max_steps;
            const uint32_t all = own_mask<C>(x);
            const bool ticks = EXT ? p.ticks != 0 : p.enable_mig != 0;
            // Every pass of the loop below is one of four modes, which share one
            // copy of each phase (iteration ends; finishes and copy stages;
            // dispatch and tick; batch formation), so the hot loop stays small:
            //   0: a window [tb, t1) in which every instance ends at most one
            //      iteration: each lane ends and re-forms its own instances, each
            //      at its own time, the later events of migrating pairs in a
            //      second pass (classify);
            //   1: one step, at the next time tc < t1, of the window's pairs whose
            //      two iterations end at the same time;
            //   2: one step at the next global event (arrival, tick), or near the
            //      step limit, over all instances;
            //   3: nothing left of mode 1: the window closes.
            bool any_b = false, in_cm = false;  // second events / mode-1 steps of the window remain
            uint32_t t1 = 0, cm = 0;            // window end; own instances stepped in mode 1
            uint32_t ucount = 0;                // distinct event times of the window
            bool in_window = false;             // the own instance has an event in it (C = 1)
            for (;;) {
                int mode;
                uint32_t et[C];      // event time of each own instance in this pass
                uint32_t heads = 0;  // own instances whose iteration ends in this pass
                uint32_t wake_lo = 0, wake_hi = 0;  // own idle instances to form in a window pass
                bool any_wake = false, ends = true;
                uint32_t tstep = 0;  // step time (modes 1 and 2)
                bool tick = false;
                if (MT_RARE(in_cm && !any_b)) {
                    uint32_t cb = kNone;
#pragma unroll
                    for (int j = 0; j < C; ++j)
                        if ((cm >> j) & 1u) cb = min(cb, x.busy[inst_at(lane, j)]);
                    tstep = __reduce_min_sync(kFull, cb);
                    mode = tstep < t1 ? 1 : 3;
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        et[j] = tstep;
                        if (mode == 1 && ((cm >> j) & 1u) && x.busy[inst_at(lane, j)] == tstep) heads |= 1u << j;
                    }
                } else {
                    if (!any_b) {
                        if (cn.finished == x.Q) { cn.status = SIM_REPLICA_DONE; break; }
                        if (cn.steps == max_steps) break;
                    }
                    uint32_t mb = kNone;
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        const int i = inst_at(lane, j);
                        et[j] = i < x.N ? x.busy[i] : kNone;
                        mb = min(mb, et[j]);
                    }
                    uint32_t tb = 0, tg = kNone;
                    if (!any_b) {
                        tb = __reduce_min_sync(kFull, mb);
                        tg = ticks ? min(next_arr, next_tick) : next_arr;
                        if (C == 1 && !mig && tb < tg)
                            tb = run_quiet(x, cn, et[0], tb, tg, max_steps, tmax, p);
                    }
                    if (any_b || (tb < tg && max_steps - cn.steps > (uint32_t)x.N)) {
                        mode = 0;
                        if (!any_b) {
                            t1 = (uint32_t)min((unsigned long long)tg, (unsigned long long)tb + (uint32_t)p.base);
                            // distinct event times of the window, and the latest
                            ucount = distinct_times<C>(x, tb, t1, et);
                            in_window = et[0] < t1;
#pragma unroll
                            for (int j = 0; j < C; ++j)
                                if (et[j] < t1) tmax = max(tmax, et[j]);
                        }
                        if (!mig) {
#pragma unroll
                            for (int j = 0; j < C; ++j) heads |= (et[j] < t1 ? 1u : 0u) << j;
                        } else {
                            const Window<C> w = classify<C>(x, t1, et);
                            heads = w.first;
                            wake_lo = w.wake_lo;
                            wake_hi = w.wake_hi;
                            cm = w.same;
                            const uint32_t any = __reduce_or_sync(kFull, (w.later ? 1u : 0u) | (cm != 0 ? 2u : 0u) |
                                                                             ((wake_lo | wake_hi) != 0 ? 4u : 0u));
                            any_wake = any & 4u;
                            any_b = any & 1u;
                            in_cm = any & 2u;
                            x.hold = true;
                        }
                    } else {
                        mode = 2;
                        const uint32_t tc = min(tb, next_arr);
                        if (tc == kNone) { cn.status = SIM_ERR_DEADLOCK; break; }
                        tick = ticks && next_tick <= tc;
                        tstep = tick ? next_tick : tc;
                        ends = tb == tstep;
                        tmax = max(tmax, tstep);
                        ++cn.steps;
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            if (et[j] == tstep) heads |= 1u << j;
                            et[j] = tstep;
                        }
                    }
                }
                // ---- 1. iteration ends, finishes and copy stages: in mode 0 those of
                // every instance together, in modes 1 and 2 instance by instance in
                // ascending order ----
                uint32_t todo = heads;
                bool go = LEAN || mode == 0 || __any_sync(kFull, todo != 0);
#pragma unroll 1
                while (go) {
                    uint32_t sel = todo;
                    if (!LEAN && mode != 0) {  // the lowest instance left
                        const int i = __reduce_min_sync(kFull, todo ? inst_at(lane, __ffs(todo) - 1) : INT_MAX);
                        sel = lane == lane_of(i) ? 1u << num_of(i) : 0u;
                    }
                    todo &= ~sel;
                    uint32_t fz = 0, src = 0;  // own instances with a finishing request; sources
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        if (!((sel >> j) & 1u)) continue;
                        const int i = inst_at(lane, j);
                        if (inst_complete_head(x, i)) fz |= 1u << j;
                        if (mig && x.mrole[i] == MIG_SRC) src |= 1u << j;
                    }
                    __syncwarp();
                    if (LEAN) fz |= src << C;
#pragma unroll 1
                    for (int j = 0; j < C; ++j)
                        for (uint32_t fl = __ballot_sync(kFull, (fz >> j) & (LEAN ? 1u | 1u << C : 1u)); fl; fl &= fl - 1) {
                            const int l = __ffs(fl) - 1, i = inst_at(l, j);
                            const uint32_t fzl = LEAN ? __shfl_sync(kFull, fz >> j, l) : 1u;
                            x.t = __shfl_sync(kFull, pick_c<C>(et, j), l);
                            if (!LEAN || (fzl & 1u)) coop_finish(x, cn, i);
                            if (LEAN && (fzl & (1u << C))) coop_stage(x, cn, i);
                        }
                    if (!LEAN && mig) stage_all<C>(x, cn, src, et);
                    go = !LEAN && mode != 0 && __any_sync(kFull, todo != 0);
                }
                int dest = -1;
                if (mode == 2) {
                    x.t = tstep;
                    if (next_arr == tstep) dest = dispatch_phase<C, SMS, EXT, LEAN>(x, cursor, next_arr, ab, p);  // 2. dispatch
                    if (MT_RARE(tick)) {  // 3. auto-scaling signal and migration tick
                        const uint32_t nt = next_tick + p.interval;
                        next_tick = nt < next_tick ? kNone : nt;  // saturate: no tick beyond 2^32 - 1
                        if (EXT && p.autoscale) autoscale_tick<C>(x, p);
                        if (p.enable_mig) {
                            if (LEAN) {
                                mig = migration_tick<C, EXT>(x, cn, p.theta_num, p.theta_den) || mig;
                            } else {
                                const int did = tick_call<C, SMS, EXT>(x.node, x.Q, x.r, x.t);
                                mig = mig || (did & 1);
                                if (MT_RARE(did & 2)) cn.status = SIM_ERR_INTERNAL;
                            }
                        }
                    }
                }
                // ---- 4. batch formation: in mode 0 every lane forms its own
                // instances at their own times; otherwise the idle instances with
                // work are formed on lane 0 in ascending order (their preemptions
                // may abort migrations, whose log records are lane 0's) ----
                // After a lone arrival only its destination can have become able to form
                // (an instance that stayed idle had nothing that fits, and nothing
                // else changed).
                uint32_t want = 0;
                if (mode == 0) {
                    want = any_wake ? wake_lo : heads;
                } else if (dest < 0 || ends || tick || x.busy[dest] == kNone) {
                    const uint32_t mask = mode == 1 ? cm : all;
#pragma unroll
                    for (int j = 0; j < C; ++j) {
                        const int i = inst_at(lane, j);
                        if (((mask >> j) & 1u) && x.busy[i] == kNone && (x.nrun[i] | x.wmask[i]) != 0) want |= 1u << j;
                    }
                }
                // (mode 0 with destinations to wake: three rounds, the lower wakes, the
                // instances whose iterations ended, the higher wakes)
#pragma unroll 1
                for (int j0 = 0; j0 < (mode == 0 ? 1 : C); ++j0) {
                    for (uint32_t fl = mode != 0 ? __ballot_sync(kFull, (want >> j0) & 1u) : any_wake ? 7u : 1u; fl;
                         fl &= fl - 1) {
                        const int l = __ffs(fl) - 1;
                        const uint32_t hl = mode == 0 ? want : 1u << j0;
                        const int owner = mode == 0 ? lane : l;
                        if (mode == 0 || lane == 0) {
                            for (uint32_t h = hl; h; h &= h - 1) {
                                const int j = __ffs(h) - 1;
                                x.t = mode == 0 ? pick_c<C>(et, j) : tstep;
                                inst_form<SMS, LEAN>(x, cn, inst_at(owner, j), p);
                            }
                        }
                        if (mode == 0) want = l == 0 ? heads : wake_hi;
                        __syncwarp();
                    }
                }
                // ---- step accounting ----
                if (mode == 0 || mode == 3) {
                    if (mode == 0 && (any_b || in_cm)) continue;
                    // the window closes
                    in_cm = false;
                    x.hold = false;
                    cn.steps += distinct_count<C>(x, ucount, in_window);
                }
                if (__any_sync(kFull, cn.held || cn.status < 0)) {
                    if (mode == 0 || mode == 3) mig = flush_held<C>(x, cn);
                    if (MT_RARE(__any_sync(kFull, cn.status < 0))) break;
                }
            }
            __syncwarp();
        } else {
            const uint32_t max_steps = p.max_steps;
            const uint32_t all = own_mask<C>(x);
            for (;;) {
                if (cn.finished == x.Q) { cn.status = SIM_REPLICA_DONE; break; }
                if (cn.steps == max_steps) break;
                uint32_t bz[C];
                uint32_t mb = kNone;
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const int i = inst_at(lane, j);
                    bz[j] = i < x.N ? x.busy[i] : kNone;
                    mb = min(mb, bz[j]);
                }
                uint32_t tb = __reduce_min_sync(kFull, mb);
                const bool ticks = EXT ? p.ticks != 0 : p.enable_mig != 0;
                const uint32_t tg = ticks ? min(next_arr, next_tick) : next_arr;
                if (C == 1 && !mig && tb < tg) tb = run_quiet(x, cn, bz[0], tb, tg, max_steps, tmax, p);
                if (tb < tg && max_steps - cn.steps > (uint32_t)x.N) {
                    // ---- window [tb, t1): at most one iteration end per instance ----
                    const uint32_t t1 =
                        (uint32_t)min((unsigned long long)tg, (unsigned long long)tb + (uint32_t)p.base);
                    // distinct event times of the window, and the latest
                    const uint32_t ucount = distinct_times<C>(x, tb, t1, bz);
                    const bool in_window = bz[0] < t1;
#pragma unroll
                    for (int j = 0; j < C; ++j)
                        if (bz[j] < t1) tmax = max(tmax, bz[j]);
                    // The iterations of the own instances in `sel` end; finishes follow, one
                    // instance at a time by the whole warp (each touches only its own
                    // pair, so their order does not matter), then copy stages.
                    auto ends = [&](uint32_t sel, bool stages) {
                        uint32_t fz = 0, src = 0;  // own instances with a finishing request; sources
#pragma unroll
                        for (int j = 0; j < C; ++j) {
                            if (!((sel >> j) & 1u)) continue;
                            const int i = inst_at(lane, j);
                            if (inst_complete_head(x, i)) fz |= 1u << j;
                            if (stages && x.mrole[i] == MIG_SRC) src |= 1u << j;
                        }
                        __syncwarp();
                        for (uint32_t fl = __ballot_sync(kFull, fz != 0); fl; fl &= fl - 1) {
                            const int l = __ffs(fl) - 1;
                            for (uint32_t h = C == 1 ? 1u : __shfl_sync(kFull, fz, l); h; h &= h - 1) {
                                const int j = __ffs(h) - 1;
                                x.t = __shfl_sync(kFull, pick_c<C>(bz, j), l);
                                coop_finish(x, cn, inst_at(l, j));
                            }
                        }
                        if (stages) stage_all<C>(x, cn, src, bz);
                    };
                    // Every lane forms its own instances' next batches.
                    auto forms = [&](uint32_t sel) {
                        if (C == 1) {
                            if (sel) {
                                x.t = bz[0];
                                inst_form<SMS, false>(x, cn, lane, p);
                            }
                        } else {
                            const uint32_t total = list_own<C>(x, sel, bz);
#pragma unroll 1
                            for (uint32_t q = (uint32_t)lane; q < total; q += 32) {
                                const uint2 e = reinterpret_cast<const uint2 *>(x.tset)[q];
                                x.t = e.x;
                                inst_form<SMS, false>(x, cn, (int)e.y, p);
                            }
                        }
                        __syncwarp();
                    };
                    if (!mig) {
                        uint32_t sel = 0;
#pragma unroll
                        for (int j = 0; j < C; ++j) sel |= (bz[j] < t1 ? 1u : 0u) << j;
                        ends(sel, false);
                        forms(sel);
                    } else {
                        x.hold = true;
                        uint32_t same, any;
                        do {
                            const Window<C> w = classify<C>(x, t1, bz);
                            any = __reduce_or_sync(kFull, (w.later ? 1u : 0u) | (w.same != 0 ? 2u : 0u) |
                                                              ((w.wake_lo | w.wake_hi) != 0 ? 4u : 0u));
                            same = w.same;
                            ends(w.first, true);
                            // idle destinations to wake form before or after the others, by index
                            uint32_t sel = (any & 4u) ? w.wake_lo : w.first;
#pragma unroll 1
                            for (int sub = (any & 4u) ? 3 : 1;;) {
                                forms(sel);
                                if (--sub == 0) break;
                                sel = sub == 2 ? w.first : w.wake_hi;
                            }
                            if (any & 1u) {
#pragma unroll
                                for (int j = 0; j < C; ++j)
                                    bz[j] = inst_at(lane, j) < x.N ? x.busy[inst_at(lane, j)] : kNone;
                            }
                        } while (any & 1u);
                        // pairs whose two iterations end at the same time: whole steps
                        // in time order
                        while (any & 2u) {
                            uint32_t cb = kNone;
#pragma unroll
                            for (int j = 0; j < C; ++j)
                                if ((same >> j) & 1u) cb = min(cb, x.busy[inst_at(lane, j)]);
                            const uint32_t tc = __reduce_min_sync(kFull, cb);
                            if (tc >= t1) break;
                            x.t = tc;
                            complete_all<C>(x, cn, same);
                            form_all<C, SMS, false>(x, cn, same, p);
                            if (MT_RARE(__any_sync(kFull, cn.status < 0))) break;
                        }
                        x.hold = false;
                    }
                    cn.steps += distinct_count<C>(x, ucount, in_window);
                    if (__any_sync(kFull, cn.held || cn.status < 0)) {
                        mig = flush_held<C>(x, cn);
                        if (MT_RARE(__any_sync(kFull, cn.status < 0))) break;
                    }
                    continue;
                }
                // ---- one step at the next event time (global events, or near the step limit) ----
                const uint32_t tc = min(tb, next_arr);
                if (tc == kNone) { cn.status = SIM_ERR_DEADLOCK; break; }
                const bool tick = ticks && next_tick <= tc;
                x.t = tick ? next_tick : tc;
                tmax = max(tmax, x.t);
                ++cn.steps;
                if (tb == x.t) complete_all<C>(x, cn, all);  // 1. iteration ends
                int dest = -1;
                if (next_arr == x.t) dest = dispatch_phase<C, SMS, EXT, false>(x, cursor, next_arr, ab, p);  // 2. dispatch
                if (MT_RARE(tick)) {  // 3. auto-scaling signal and migration tick
                    const uint32_t nt = next_tick + p.interval;
                    next_tick = nt < next_tick ? kNone : nt;  // saturate: no tick beyond 2^32 - 1
                    if (EXT && p.autoscale) autoscale_tick<C>(x, p);
                    if (p.enable_mig) {
                        const int did = tick_call<C, SMS, EXT>(x.node, x.Q, x.r, x.t);
                        mig = mig || (did & 1);
                        if (MT_RARE(did & 2)) cn.status = SIM_ERR_INTERNAL;
                    }
                }
                // 4. batch formation.  After a lone arrival only its destination can
                // have become able to form (an instance that stayed idle had nothing
                // that fits, and nothing else changed).
                if (tb == x.t || tick || dest < 0 || x.busy[dest] == kNone) form_all<C, SMS, false>(x, cn, all, p);
                if (MT_RARE(__any_sync(kFull, cn.status < 0))) break;
            }
            __syncwarp();
        }
        // fold the other lanes' counters into lane 0's (status: DONE or RUNNING on
        // every lane, or an error on some)
        cn.status = __reduce_min_sync(kFull, cn.status);
        const uint32_t tfin = __reduce_max_sync(kFull, tmax);
        const uint32_t a_it = __reduce_add_sync(kFull, cn.iterations);
        uint64_t a_mi = cn.member_iterations;
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) a_mi += __shfl_xor_sync(kFull, a_mi, sh);
        copy16(gblob, blob, p.L.bytes, lane);
        if (SMS)
            copy16(reinterpret_cast<unsigned char *>(g_slots), reinterpret_cast<const unsigned char *>(x.slots),
                   slot_bytes, lane);
        if (lane == 0) {
            RepState o2 = p.rep[r];  // this warp's until the launch ends
            o2.t = tfin;
            o2.cursor = cursor;
            o2.finished = cn.finished;
            o2.log_events = x.tot[TOT_LOG];
            o2.next_tick = next_tick;
            o2.steps += cn.steps;
            o2.iterations += a_it;
            o2.member_iterations += a_mi;
            o2.migrations = x.tot[TOT_MIG];
            o2.preemptions = x.tot[TOT_PRE];
            o2.starts = x.tot[TOT_START];
            o2.aborts = x.tot[TOT_ABORT];
            o2.scale_out = x.tot[TOT_OUT];
            o2.scale_in = x.tot[TOT_IN];
            o2.events = (uint64_t)cursor + cn.finished + o2.migrations + o2.preemptions;
            o2.status = cn.status;
            p.rep[r] = o2;
        }
        __syncwarp();
    }
}

// ---- set-up and export kernels ----------------------------------------------
__global__ void k_init_state(Params p, const int *rep_table, const int *tbl_k, const int *tbl_h) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < p.R; r += warps) {
        unsigned char *b = p.blobs + (size_t)r * p.L.bytes;
        const Layout &L = p.L;
        const int N = p.N, NK = p.N * p.K;
        const int tb = rep_table[r];
        const int K = tbl_k[tb];
        for (int i = lane; i < N; i += 32) {
            InstRec v;
            memset(&v, 0, sizeof v);
            v.busy = kNone;
            v.free_ = p.M;
            v.mreq = kNone;
            v.minfin = kNone;
            v.drain = p.drain_src ? p.drain_src[(size_t)r * N + i] : kNone;
            v.mrole = MIG_NONE;
            reinterpret_cast<InstRec *>(b + L.inst)[i] = v;
        }
        for (int q = lane; q < N * p.TH; q += 32) b[L.hist + q] = 0;
        if (lane < TOT_COUNT) reinterpret_cast<uint32_t *>(b + L.tot)[lane] = 0;
        for (int i = lane; i < NK; i += 32) {
            reinterpret_cast<uint16_t *>(b + L.cnt)[i] = 0;
            reinterpret_cast<uint32_t *>(b + L.head)[i] = kNone;
            reinterpret_cast<uint32_t *>(b + L.tail)[i] = kNone;
            reinterpret_cast<uint32_t *>(b + L.hinfo)[i] = 0;
        }
        for (int k = lane; k < p.K; k += 32)
            reinterpret_cast<int *>(b + L.h)[k] = k < K ? tbl_h[tb * p.K + k] : 0;
        if (lane == 0) {
            RepState s;
            memset(&s, 0, sizeof s);
            s.next_tick = p.interval;
            s.status = (p.offsets[r + 1] == p.offsets[r]) ? SIM_REPLICA_DONE : SIM_REPLICA_RUNNING;
            p.rep[r] = s;
        }
    }
}

// New headroom tables (adaptive headroom, sim_set_headroom): each replica's
// H[k] from its table, and every instance's present-tier headroom sum
// recomputed from its per-tier request counts (Sec. 3.3 Eq. 4: H_k once per
// tier present).  One warp per replica.
__global__ void k_set_headroom(Params p, const int *rep_table, const int *tbl_k, const int *tbl_h) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < p.R; r += warps) {
        unsigned char *b = p.blobs + (size_t)r * p.L.bytes;
        const int tb = rep_table[r];
        const int K = tbl_k[tb];
        const int *hn = tbl_h + (size_t)tb * p.K;
        for (int k = lane; k < p.K; k += 32) reinterpret_cast<int *>(b + p.L.h)[k] = k < K ? hn[k] : 0;
        const uint16_t *cnt = reinterpret_cast<const uint16_t *>(b + p.L.cnt);
        for (int i = lane; i < p.N; i += 32) {
            int sum = 0;
            for (int k = 0; k < K; ++k)
                if (cnt[i * p.K + k] > 0) sum += hn[k];
            reinterpret_cast<InstRec *>(b + p.L.inst)[i].hr = sum;
        }
    }
}

__global__ void k_init_requests(sim_request_result_t *res, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        reinterpret_cast<uint4 *>(res)[i] = make_uint4(0xFFFFFFFFu, kNone, kNone, 0u);
}

// Trace validation: bit 0 unsorted, 1 tier >= K, 2 zero length, 3 too long, 4 bad arrival.
__global__ void k_validate(const long long *offsets, int R, const uint32_t *arrival, const uint16_t *plen,
                           const uint16_t *olen, const uint8_t *tier, const int *rep_table, const int *tbl_k,
                           long long lim, long long n, int *flags) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = R - 1;  // replica r with offsets[r] <= i < offsets[r+1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (offsets[mid] <= i) lo = mid; else hi = mid - 1;
        }
        int f = 0;
        if (i > offsets[lo] && arrival[i] < arrival[i - 1]) f |= 1;
        if ((int)tier[i] >= tbl_k[rep_table[lo]]) f |= 2;
        if (plen[i] == 0 || olen[i] == 0) f |= 4;
        if ((long long)plen[i] + olen[i] > lim) f |= 8;
        if (arrival[i] == kNone) f |= 16;
        if (f) atomicOr(flags, f);
    }
}

// Per replica, the number of requests that have a first token; the simulation
// kernel records first tokens without counting them (see inst_form), so the
// exported event count adds these.
__global__ void k_first_tokens(const long long *offsets, int R, const sim_request_result_t *res, uint32_t *count) {
    __shared__ uint32_t part[32];
    for (int r = blockIdx.x; r < R; r += gridDim.x) {
        uint32_t c = 0;
        for (long long i = offsets[r] + threadIdx.x; i < offsets[r + 1]; i += blockDim.x)
            c += res[i].first_token_us != kNone ? 1u : 0u;
        c = __reduce_add_sync(kFull, c);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
            count[r] = t;
        }
        __syncthreads();
    }
}

__global__ void k_export_stats(const RepState *rep, sim_replica_stats_t *out, int R, int *unfinished,
                               const uint32_t *first_tokens) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < R; r += gridDim.x * blockDim.x) {
        const RepState s = rep[r];
        if (out) {
            sim_replica_stats_t o;
            o.steps = s.steps;
            o.iterations = s.iterations;
            o.member_iterations = s.member_iterations;
            o.events = s.events + (first_tokens ? first_tokens[r] : 0u);
            o.migrations = s.migrations;
            o.preemptions = s.preemptions;
            o.migration_starts = s.starts;
            o.migration_aborts = s.aborts;
            o.log_events = s.log_events;
            o.finished = s.finished;
            o.last_time_us = s.t;
            o.status = s.status;
            o.scale_out_signals = s.scale_out;
            o.scale_in_signals = s.scale_in;
            out[r] = o;
        }
        if (unfinished && s.status != SIM_REPLICA_DONE) atomicAdd(unfinished, 1);
    }
}

// ---- launch configuration ---------------------------------------------------
typedef void (*RunKernel)(Params);

template <bool EXT>
RunKernel pick(int c, bool sms, bool many) {  // c = instances per lane
    if (many && sms) return k_run<1, true, EXT, true>;
    if (many) return c == 1 ? k_run<1, false, EXT, true> : c == 2 ? k_run<2, false, EXT, true> : k_run<4, false, EXT, true>;
    switch (c) {
        case 1: return sms ? k_run<1, true, EXT, false> : k_run<1, false, EXT, false>;
        case 2: return sms ? k_run<2, true, EXT, false> : k_run<2, false, EXT, false>;
        case 4: return sms ? k_run<4, true, EXT, false> : k_run<4, false, EXT, false>;
        default: return sms ? k_run<8, true, EXT, false> : k_run<8, false, EXT, false>;
    }
}

// fn / grid: the plain variant; fn_ext / grid_ext: the one with draining and
// the auto-scaling signal (same shared memory).
struct Launch {
    RunKernel fn = nullptr, fn_ext = nullptr;
    int grid = 0, grid_ext = 0;
    int per_sm = 0, per_sm_ext = 0;  // resident blocks per SM of each variant
    int c = 1;                       // instances per lane
    bool sms = false;                // running-request records in shared memory
    int set_bits = 0;                // scratch of distinct_times, log2 of its bytes
    uint32_t scratch = 0;            // scratch of a warp, bytes
    size_t smem = 0;
};

// Chooses the kernel variant and grid for a problem; cudaSuccess or the error.
inline cudaError_t plan_launch(int R, int N, int Bmax, const Layout &L, Launch &out) {
    int dev = 0, sms_count = 0, max_smem = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms_count, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    auto resident = [&](RunKernel fn, size_t smem) -> int {
        int per_sm = 0;
        // The limit belongs to the kernel, not to a launch: it is always set to the
        // device's, so that no plan lowers it for an object that launches later.
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * kWarpsPerBlock, smem);
        return e == cudaSuccess ? per_sm : -1;
    };
    Plan plan;
    const int fits = choose_plan(R, N, Bmax, L, sms_count, (size_t)max_smem, [&](const Plan &q) {
        return resident(pick<false>(q.c, q.sms, q.many), q.smem);
    }, plan);
    if (fits < 1) return fits < 0 ? e : cudaErrorInvalidConfiguration;
    out.c = plan.c;
    out.sms = plan.sms;
    out.set_bits = plan.set_bits;
    out.scratch = plan.scratch;
    out.smem = plan.smem;
    out.fn = pick<false>(plan.c, plan.sms, plan.many);
    out.fn_ext = pick<true>(plan.c, plan.sms, plan.many);
    const long long want = ((long long)R + kWarpsPerBlock - 1) / kWarpsPerBlock;
    for (int v = 0; v < 2; ++v) {
        const int per_sm = resident(v ? out.fn_ext : out.fn, out.smem);
        if (per_sm < 0) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        (v ? out.grid_ext : out.grid) = (int)std::min<long long>(want, (long long)sms_count * per_sm);
        (v ? out.per_sm_ext : out.per_sm) = per_sm;
    }
    return cudaSuccess;
}

inline unsigned long long magic40(unsigned d) { return ((1ull << kMagicShift) + d - 1ull) / d; }

}  // namespace mt

// ============================================================================
// Host side: the C ABI.
// ============================================================================
struct sim {
    sim_cluster_t cl;
    sim_policy_t pol;
    int K = 0, ntables = 0;
    std::vector<int> tbl_k, tbl_h, rep_table;
    cudaStream_t stream = nullptr;
    sim_allocator_t al{};
    bool use_al = false;
    mt::Layout L{};
    mt::Launch launch{};
    struct Buf { void *p; size_t n; };
    std::vector<Buf> bufs;
    size_t dev_bytes = 0;
    int *d_rep_table = nullptr, *d_tbl_k = nullptr, *d_tbl_h = nullptr;
    unsigned char *d_blobs = nullptr;
    uint4 *d_slots = nullptr;
    mt::RepState *d_rep = nullptr;
    sim_migration_event_t *d_log = nullptr;
    int *d_work = nullptr;  // [0] work counter, [1] validation flags, [2] unfinished count
    int64_t qtot = 0, qcap = -1;
    bool loaded = false;
    std::vector<int64_t> h_off;
    long long *d_off = nullptr;
    uint32_t *d_arrival = nullptr;
    uint16_t *d_plen = nullptr, *d_olen = nullptr;
    uint8_t *d_tier = nullptr;
    uint4 *d_node = nullptr;
    sim_request_result_t *d_res = nullptr;
    uint32_t *d_drain = nullptr;  // [R][N] drain start times (sim_set_drain), or NULL
    int *d_order = nullptr;       // [R] replica start order (sim_set_order), or NULL
    uint32_t *d_ftc = nullptr;    // [R] first-token counts for sim_metrics
    sim_latency_stats_t *d_lat = nullptr;  // device staging of sim_latency_stats for host output
    int *d_lat_rep = nullptr;              // chunk table of sim_latency_stats: replica and first record
    long long *d_lat_b0 = nullptr;
    uint4 *d_lat_sel = nullptr;            // percentile selection scratch of sim_latency_stats
    uint32_t *d_lat_bins = nullptr;
    int lat_nchunks = -1;                  // -1: to be built for the loaded trace
    int sms = 0;
    std::string err;
};

namespace {

thread_local std::string g_create_err;

int fail(sim_t *s, int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (s) s->err = buf; else g_create_err = buf;
    return code;
}

int cuda_fail(sim_t *s, cudaError_t e, const char *what) {
    return fail(s, SIM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

void *dalloc(sim_t *s, size_t n) {
    if (n == 0) n = 16;
    n = (n + 255) & ~(size_t)255;
    void *p = nullptr;
    if (s->use_al) {
        p = s->al.alloc(s->al.ctx, n, (void *)s->stream);
    } else if (cudaMallocAsync(&p, n, s->stream) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
    if (p) {
        s->bufs.push_back({p, n});
        s->dev_bytes += n;
    }
    return p;
}

void dfree(sim_t *s, void *p) {
    if (!p) return;
    for (size_t i = 0; i < s->bufs.size(); ++i) {
        if (s->bufs[i].p == p) {
            if (s->use_al) s->al.free(s->al.ctx, p, s->bufs[i].n, (void *)s->stream);
            else cudaFreeAsync(p, s->stream);
            s->dev_bytes -= s->bufs[i].n;
            s->bufs.erase(s->bufs.begin() + i);
            return;
        }
    }
}

// Fills the scalar part of the kernel parameters (pointers are set by the caller).
void fill_scalars(mt::Params &p, const sim_cluster_t &cl, const sim_policy_t &pol, int K, int cap,
                  const mt::Layout &L, long long max_steps) {
    p.R = cl.num_replicas;
    p.N = cl.num_instances;
    p.M = cl.blocks_per_instance;
    p.T = cl.tokens_per_block;
    p.Bmax = cl.max_batch;
    p.TH = mt::hist_stride(cl.tokens_per_block);
    p.K = K;
    p.S = pol.migrate_blocks_per_iter;
    p.cap = cap;
    p.enable_mig = pol.enable_migration;
    p.theta_num = pol.theta_num;
    p.theta_den = pol.theta_den;
    p.interval = (uint32_t)pol.migrate_interval_us;
    p.max_steps = (uint32_t)std::min<long long>(max_steps, 0xFFFFFFFFLL);
    p.magT = mt::magic40((unsigned)cl.tokens_per_block);
    p.base = (int)pol.iter_base_us;
    p.a = (int)pol.iter_us_per_prefill_token;
    p.b = (int)pol.iter_us_per_decode_seq;
    p.ticks = pol.enable_migration || pol.autoscale;
    p.autoscale = pol.autoscale;
    p.scale_out_num = pol.scale_out_num;
    p.scale_in_num = pol.scale_in_num;
    p.scale_den = pol.scale_den;
    unsigned __int128 l = 1;  // lcm(1, ..., Bmax): every max(B, 1) divides it
    for (unsigned d = 2; d <= (unsigned)cl.max_batch; ++d) {
        unsigned a = d, b = (unsigned)(l % d);
        while (b) { const unsigned t = a % b; a = b; b = t; }
        l = l / a * d;
    }
    p.lcm_lo = (unsigned long long)l;
    p.lcm_hi = (unsigned long long)(l >> 64);
    p.L = L;
}

mt::Params make_params(const sim_t *s, long long max_steps) {
    mt::Params p;
    memset(&p, 0, sizeof p);
    fill_scalars(p, s->cl, s->pol, s->K, s->pol.event_log_capacity, s->L, max_steps);
    p.offsets = s->d_off;
    p.drain_src = s->d_drain;
    p.drains = s->d_drain != nullptr;
    p.arrival = s->d_arrival;
    p.plen = s->d_plen;
    p.olen = s->d_olen;
    p.tier = s->d_tier;
    p.node = s->d_node;
    p.res = s->d_res;
    p.res_off = (const char *)s->d_res - (const char *)s->d_node;
    p.blobs = s->d_blobs;
    p.slots = s->d_slots;
    p.rep = s->d_rep;
    p.log = s->d_log;
    p.work = s->d_work;
    p.order = s->d_order;
    p.set_bits = s->launch.set_bits;
    p.scratch = s->launch.scratch;
    return p;
}

int check_launch(sim_t *s, const char *what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(s, e, what);
    return SIM_OK;
}

int reset_state(sim_t *s) {
    mt::Params p = make_params(s, 0);
    const int R = s->cl.num_replicas;
    mt::k_init_state<<<(R + 7) / 8, 256, 0, s->stream>>>(p, s->d_rep_table, s->d_tbl_k, s->d_tbl_h);
    int rc = check_launch(s, "k_init_state");
    if (rc) return rc;
    if (s->qtot > 0) {
        const long long nb = std::min<long long>((s->qtot + 255) / 256, 65535LL * 16);
        mt::k_init_requests<<<(unsigned)nb, 256, 0, s->stream>>>(s->d_res, (long long)s->qtot);
        rc = check_launch(s, "k_init_requests");
    }
    return rc;
}

// The limits every entry point enforces on cluster, tier tables and policy.
int validate_config(sim_t *s, const sim_cluster_t *cl, const sim_tier_table_t *tt, const sim_policy_t *pol) {
    if (!cl || !tt || !pol) return fail(s, SIM_ERR_ARG, "cluster, tiers and policy are required");
    if (cl->num_replicas < 1) return fail(s, SIM_ERR_ARG, "num_replicas must be >= 1");
    if (cl->num_instances < 1 || cl->num_instances > SIM_MAX_INSTANCES)
        return fail(s, SIM_ERR_ARG, "num_instances must be in [1, %d]", SIM_MAX_INSTANCES);
    if (cl->blocks_per_instance < 1 || cl->blocks_per_instance > SIM_MAX_BLOCKS)
        return fail(s, SIM_ERR_ARG, "blocks_per_instance must be in [1, %d]", SIM_MAX_BLOCKS);
    if (cl->tokens_per_block < 1 || cl->tokens_per_block > mt::kMaxBlockTokens)
        return fail(s, SIM_ERR_ARG, "tokens_per_block must be in [1, %d]", mt::kMaxBlockTokens);
    if (cl->max_batch < 1 || cl->max_batch > SIM_MAX_BATCH)
        return fail(s, SIM_ERR_ARG, "max_batch must be in [1, %d]", SIM_MAX_BATCH);
    if (tt->num_tables < 1 || tt->max_tiers < 1 || tt->max_tiers > SIM_MAX_TIERS)
        return fail(s, SIM_ERR_ARG, "need num_tables >= 1 and max_tiers in [1, %d]", SIM_MAX_TIERS);
    if (!tt->num_tiers || !tt->headroom_blocks || !tt->replica_table)
        return fail(s, SIM_ERR_ARG, "tier table pointers must not be NULL");
    for (int t = 0; t < tt->num_tables; ++t) {
        const int K = tt->num_tiers[t];
        if (K < 1 || K > tt->max_tiers) return fail(s, SIM_ERR_ARG, "table %d: num_tiers out of range", t);
        long long sum = 0;
        for (int k = 0; k < K; ++k) {
            const int h = tt->headroom_blocks[t * tt->max_tiers + k];
            if (h < 0) return fail(s, SIM_ERR_ARG, "table %d: negative headroom", t);
            sum += h;
        }
        if (cl->blocks_per_instance + sum >= mt::kMaxKeyRange)
            return fail(s, SIM_ERR_ARG, "table %d: M + sum of headroom must be below 2^19", t);
    }
    for (int r = 0; r < cl->num_replicas; ++r)
        if (tt->replica_table[r] < 0 || tt->replica_table[r] >= tt->num_tables)
            return fail(s, SIM_ERR_ARG, "replica %d: table index out of range", r);
    if (pol->policy != SIM_POLICY_LLUMNIX_MT) return fail(s, SIM_ERR_ARG, "unknown policy %d", pol->policy);
    if (pol->enable_migration != 0 && pol->enable_migration != 1)
        return fail(s, SIM_ERR_ARG, "enable_migration must be 0 or 1");
    const long long lim24 = 1LL << 24;
    if (pol->iter_base_us < 1 || pol->iter_base_us > lim24 || pol->iter_us_per_prefill_token < 0 ||
        pol->iter_us_per_prefill_token > lim24 || pol->iter_us_per_decode_seq < 0 || pol->iter_us_per_decode_seq > lim24)
        return fail(s, SIM_ERR_ARG, "iteration-time base must be in [1, 2^24], the other coefficients in [0, 2^24]");
    if (pol->migrate_blocks_per_iter < 1 || pol->migrate_blocks_per_iter > 65535)
        return fail(s, SIM_ERR_ARG, "migrate_blocks_per_iter must be in [1, 65535]");
    if (pol->theta_den < 1 || pol->theta_num < 0 || pol->theta_num > (1 << 20) || pol->theta_den > (1 << 20))
        return fail(s, SIM_ERR_ARG, "theta must be num/den with num in [0, 2^20], den in [1, 2^20]");
    if (pol->event_log_capacity < 0 || pol->event_log_capacity > (1 << 24))
        return fail(s, SIM_ERR_ARG, "event_log_capacity must be in [0, 2^24]");
    if (pol->migrate_interval_us < 1 || pol->migrate_interval_us > (1LL << 31))
        return fail(s, SIM_ERR_ARG, "migrate_interval_us must be in [1, 2^31]");
    if (pol->autoscale != 0 && pol->autoscale != 1) return fail(s, SIM_ERR_ARG, "autoscale must be 0 or 1");
    if (pol->autoscale && (pol->scale_den < 1 || pol->scale_den > 64 || pol->scale_out_num < -4096 ||
                           pol->scale_in_num > 4096 || pol->scale_out_num >= pol->scale_in_num))
        return fail(s, SIM_ERR_ARG,
                    "auto-scaling thresholds must be num/den with den in [1, 64], numerators in [-4096, 4096] "
                    "and scale_out_num < scale_in_num");
    return SIM_OK;
}

}  // namespace

extern "C" {

const char *sim_strerror(int code) {
    switch (code) {
        case SIM_OK: return "ok";
        case SIM_ERR_ARG: return "invalid argument";
        case SIM_ERR_TRACE: return "malformed trace";
        case SIM_ERR_STATE: return "call out of order";
        case SIM_ERR_OOM: return "device allocation failed";
        case SIM_ERR_OVERFLOW: return "32-bit time or counter overflow";
        case SIM_ERR_CUDA: return "CUDA runtime error";
        case SIM_ERR_INTERNAL: return "device-side consistency check failed";
        case SIM_ERR_DEADLOCK: return "no pending event while requests are unfinished";
        case SIM_ERR_UNFINISHED: return "some replica did not finish";
        default: return "unknown error";
    }
}

const char *sim_last_error(const sim_t *s) { return s ? s->err.c_str() : g_create_err.c_str(); }

size_t sim_device_bytes(const sim_t *s) { return s ? s->dev_bytes : 0; }

int sim_launch_info(const sim_t *s, sim_launch_info_t *out) {
    if (!s || !out) return SIM_ERR_ARG;
    const bool ext = s->d_drain != nullptr || s->pol.autoscale != 0;
    out->grid_blocks = ext ? s->launch.grid_ext : s->launch.grid;
    out->block_threads = 32 * mt::kWarpsPerBlock;
    out->blocks_per_sm = ext ? s->launch.per_sm_ext : s->launch.per_sm;
    out->instances_per_lane = s->launch.c;
    out->slots_in_shared = s->launch.sms ? 1 : 0;
    out->extended = ext ? 1 : 0;
    out->shared_bytes = (int64_t)s->launch.smem;
    return SIM_OK;
}

int sim_create(const sim_cluster_t *cl, const sim_tier_table_t *tt, const sim_policy_t *pol, void *cuda_stream,
               const sim_allocator_t *allocator, sim_t **out) {
    if (!out) return fail(nullptr, SIM_ERR_ARG, "out is NULL");
    *out = nullptr;
    int rc = validate_config(nullptr, cl, tt, pol);
    if (rc) return rc;
    if (allocator && (!allocator->alloc || !allocator->free))
        return fail(nullptr, SIM_ERR_ARG, "allocator needs both alloc and free");

    sim_t *s = new (std::nothrow) sim_t();
    if (!s) return fail(nullptr, SIM_ERR_OOM, "host allocation failed");
    s->cl = *cl;
    s->pol = *pol;
    s->K = tt->max_tiers;
    s->ntables = tt->num_tables;
    s->tbl_k.assign(tt->num_tiers, tt->num_tiers + tt->num_tables);
    s->tbl_h.assign(tt->headroom_blocks, tt->headroom_blocks + (size_t)tt->num_tables * tt->max_tiers);
    s->rep_table.assign(tt->replica_table, tt->replica_table + cl->num_replicas);
    s->stream = (cudaStream_t)cuda_stream;
    if (allocator) { s->al = *allocator; s->use_al = true; }
    s->L = mt::make_layout(cl->num_instances, s->K, cl->tokens_per_block);

    const size_t R = (size_t)cl->num_replicas, NB = (size_t)cl->num_instances * cl->max_batch;
    s->d_rep_table = (int *)dalloc(s, R * 4);
    s->d_tbl_k = (int *)dalloc(s, (size_t)s->ntables * 4);
    s->d_tbl_h = (int *)dalloc(s, (size_t)s->ntables * s->K * 4);
    s->d_blobs = (unsigned char *)dalloc(s, R * s->L.bytes);
    s->d_slots = (uint4 *)dalloc(s, R * NB * 16);
    s->d_rep = (mt::RepState *)dalloc(s, R * sizeof(mt::RepState));
    s->d_log = (sim_migration_event_t *)dalloc(s, R * (size_t)pol->event_log_capacity * sizeof(sim_migration_event_t));
    s->d_work = (int *)dalloc(s, 16);
    if (!s->d_rep_table || !s->d_tbl_k || !s->d_tbl_h || !s->d_blobs || !s->d_slots || !s->d_rep ||
        !s->d_log || !s->d_work) {
        const size_t held = s->dev_bytes;
        sim_destroy(s);
        return fail(nullptr, SIM_ERR_OOM, "device allocation failed (%zu bytes held when it failed)", held);
    }
    cudaError_t e = cudaMemcpyAsync(s->d_rep_table, s->rep_table.data(), R * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->d_tbl_k, s->tbl_k.data(), (size_t)s->ntables * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->d_tbl_h, s->tbl_h.data(), s->tbl_h.size() * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);  // host vectors may be pageable
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = mt::plan_launch(cl->num_replicas, cl->num_instances, cl->max_batch, s->L, s->launch);
    if (e != cudaSuccess) {
        cudaGetLastError();
        rc = e == cudaErrorInvalidConfiguration
                 ? fail(nullptr, SIM_ERR_ARG, "per-replica state (%u bytes) does not fit in shared memory", s->L.bytes)
                 : cuda_fail(nullptr, e, "sim_create");
        sim_destroy(s);
        return rc;
    }
    *out = s;
    return SIM_OK;
}

int sim_load_trace(sim_t *s, const int64_t *off, const uint32_t *arrival, const uint16_t *plen, const uint16_t *olen,
                   const uint8_t *tier, int on_device) {
    if (!s) return SIM_ERR_ARG;
    if (!off) return fail(s, SIM_ERR_ARG, "replica_offsets is NULL");
    const int R = s->cl.num_replicas;
    if (off[0] != 0) return fail(s, SIM_ERR_TRACE, "replica_offsets[0] must be 0");
    for (int r = 0; r < R; ++r) {
        const int64_t q = off[r + 1] - off[r];
        if (q < 0) return fail(s, SIM_ERR_TRACE, "replica_offsets must be non-decreasing (replica %d)", r);
        if (q > (int64_t)0xFFFFFFFEll) return fail(s, SIM_ERR_TRACE, "replica %d has more than 2^32-2 records", r);
    }
    const int64_t n = off[R];
    if (n > 0 && (!arrival || !plen || !olen || !tier)) return fail(s, SIM_ERR_ARG, "trace arrays must not be NULL");
    s->loaded = false;
    if (n > s->qcap) {
        dfree(s, s->d_arrival); dfree(s, s->d_plen); dfree(s, s->d_olen); dfree(s, s->d_tier);
        dfree(s, s->d_node); dfree(s, s->d_res);
        s->d_arrival = nullptr; s->d_plen = s->d_olen = nullptr; s->d_tier = nullptr;
        s->d_node = nullptr; s->d_res = nullptr;
        s->qcap = -1;
        const size_t m = (size_t)std::max<int64_t>(n, 1);
        s->d_arrival = (uint32_t *)dalloc(s, m * 4);
        s->d_plen = (uint16_t *)dalloc(s, m * 2);
        s->d_olen = (uint16_t *)dalloc(s, m * 2);
        s->d_tier = (uint8_t *)dalloc(s, m);
        s->d_node = (uint4 *)dalloc(s, m * 16);
        s->d_res = (sim_request_result_t *)dalloc(s, m * 16);
        if (!s->d_arrival || !s->d_plen || !s->d_olen || !s->d_tier || !s->d_node || !s->d_res)
            return fail(s, SIM_ERR_OOM, "device allocation for %lld trace records failed", (long long)n);
        s->qcap = n;
    }
    if (!s->d_off) {
        s->d_off = (long long *)dalloc(s, ((size_t)R + 1) * 8);
        if (!s->d_off) return fail(s, SIM_ERR_OOM, "device allocation failed");
    }
    s->h_off.assign(off, off + R + 1);
    s->lat_nchunks = -1;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    cudaError_t e = cudaMemcpyAsync(s->d_off, s->h_off.data(), ((size_t)R + 1) * 8, cudaMemcpyHostToDevice, s->stream);
    if (n > 0) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_arrival, arrival, (size_t)n * 4, kind, s->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_plen, plen, (size_t)n * 2, kind, s->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_olen, olen, (size_t)n * 2, kind, s->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(s->d_tier, tier, (size_t)n, kind, s->stream);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_work, 0, 16, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_load_trace copy");
    s->qtot = n;
    if (n > 0) {
        const long long lim = std::min<long long>((long long)s->cl.blocks_per_instance * s->cl.tokens_per_block, 65536);
        const long long nb = std::min<long long>((n + 255) / 256, (long long)s->sms * 32);
        mt::k_validate<<<(unsigned)std::max<long long>(nb, 1), 256, 0, s->stream>>>(
            s->d_off, R, s->d_arrival, s->d_plen, s->d_olen, s->d_tier, s->d_rep_table, s->d_tbl_k, lim, n,
            s->d_work + 1);
        int rc = check_launch(s, "k_validate");
        if (rc) return rc;
    }
    int flags = 0;
    e = cudaMemcpyAsync(&flags, s->d_work + 1, 4, cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_load_trace validation");
    if (flags) {
        return fail(s, SIM_ERR_TRACE, "malformed trace:%s%s%s%s%s", (flags & 1) ? " unsorted arrivals;" : "",
                    (flags & 2) ? " tier >= K;" : "", (flags & 4) ? " zero prompt or output length;" : "",
                    (flags & 8) ? " prompt + output longer than min(M*T, 65536);" : "",
                    (flags & 16) ? " arrival time 0xFFFFFFFF;" : "");
    }
    int rc = reset_state(s);
    if (rc) return rc;
    s->loaded = true;
    return SIM_OK;
}

int sim_reset(sim_t *s) {
    if (!s) return SIM_ERR_ARG;
    if (!s->loaded) return fail(s, SIM_ERR_STATE, "sim_reset before sim_load_trace");
    return reset_state(s);
}

static_assert(sizeof(sim_latency_stats_t) == 32 + 4 * SIM_HIST_BUCKETS, "sim_latency_stats_t layout");

int sim_latency_stats(sim_t *s, sim_latency_stats_t *out, int on_device) {
    if (!s) return SIM_ERR_ARG;
    if (!out) return fail(s, SIM_ERR_ARG, "out is NULL");
    if (on_device != 0 && on_device != 1) return fail(s, SIM_ERR_ARG, "on_device must be 0 or 1");
    if (!s->loaded) return fail(s, SIM_ERR_STATE, "sim_latency_stats before sim_load_trace");
    const int R = s->cl.num_replicas, KT = s->K;
    const size_t n = (size_t)R * KT * 3;
    sim_latency_stats_t *d = out;
    if (!on_device) {
        if (!s->d_lat) {
            s->d_lat = (sim_latency_stats_t *)dalloc(s, n * sizeof(sim_latency_stats_t));
            if (!s->d_lat) return fail(s, SIM_ERR_OOM, "device allocation of the latency statistics failed");
        }
        d = s->d_lat;
    }
    // Replicas whose values fit in a block's shared memory (about 15,000 requests
    // with 4 tiers) take one kernel, larger ones the streaming passes.  One
    // kernel / streaming, us back to back: 1 replica x 64 requests 17 / 45, 1 x 14,000
    // 57 / 74, 1,024 x 5,000 161 / 240, 1,000 x 8,000 245 / 279, 3,840 x 1,000 with 10
    // tiers 388 / 730, 700 x 4,000 with 16 tiers 231 / 370.  Slower are only the largest
    // replicas just past a wave (153 x 15,900 122 / 111, 153 x 10,500 with 16 tiers 193
    // / 167) and thousands of tiny replicas beside such a one (1 tier, 8,192 x 10 +
    // 15,000 requests 305 / 222).
    long long qmax = 0;
    for (int r = 0; r < R; ++r) qmax = std::max<long long>(qmax, s->h_off[r + 1] - s->h_off[r]);
    bool done = false;
    cudaError_t e = mtlat::launch_replicas(R, qmax, s->d_off, KT, s->d_arrival, s->d_olen, s->d_tier, s->d_res, d,
                                           s->sms, s->stream, &done);
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_latency_stats");
    if (!done) {
        if (s->lat_nchunks < 0) {  // chunk table of the loaded trace
            std::vector<int> rep;
            std::vector<long long> b0;
            for (int r = 0; r < R; ++r)
                for (long long b = s->h_off[r]; b < s->h_off[r + 1]; b += mtlat::kChunk) {
                    rep.push_back(r);
                    b0.push_back(b);
                }
            const int nc = (int)rep.size();
            dfree(s, s->d_lat_rep);
            dfree(s, s->d_lat_b0);
            s->d_lat_rep = nullptr;
            s->d_lat_b0 = nullptr;
            if (nc > 0) {
                s->d_lat_rep = (int *)dalloc(s, (size_t)nc * 4);
                s->d_lat_b0 = (long long *)dalloc(s, (size_t)nc * 8);
                if (!s->d_lat_rep || !s->d_lat_b0) return fail(s, SIM_ERR_OOM, "device allocation of the chunk table failed");
                e = cudaMemcpyAsync(s->d_lat_rep, rep.data(), (size_t)nc * 4, cudaMemcpyHostToDevice, s->stream);
                if (e == cudaSuccess)
                    e = cudaMemcpyAsync(s->d_lat_b0, b0.data(), (size_t)nc * 8, cudaMemcpyHostToDevice, s->stream);
                if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);  // the host vectors go out of scope
                if (e != cudaSuccess) return cuda_fail(s, e, "sim_latency_stats chunk table");
            }
            s->lat_nchunks = nc;
        }
        if (!s->d_lat_sel) {
            s->d_lat_sel = (uint4 *)dalloc(s, mtlat::select_state_bytes((long long)n));
            s->d_lat_bins = (uint32_t *)dalloc(s, mtlat::select_bin_bytes((long long)n));
            if (!s->d_lat_sel || !s->d_lat_bins)
                return fail(s, SIM_ERR_OOM, "device allocation of the percentile selection scratch failed");
        }
        e = mtlat::launch(s->d_lat_rep, s->d_lat_b0, s->lat_nchunks, s->d_off, KT, s->d_arrival, s->d_olen, s->d_tier,
                          s->d_res, d, (long long)n, s->d_lat_sel, s->d_lat_bins, s->sms, s->stream);
    }
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_latency_stats");
    if (!on_device) {
        e = cudaMemcpyAsync(out, d, n * sizeof(sim_latency_stats_t), cudaMemcpyDeviceToHost, s->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
        if (e != cudaSuccess) return cuda_fail(s, e, "sim_latency_stats copy");
    }
    return SIM_OK;
}

int sim_set_drain(sim_t *s, const uint32_t *drain_start_us, int on_device) {
    if (!s) return SIM_ERR_ARG;
    if (on_device != 0 && on_device != 1) return fail(s, SIM_ERR_ARG, "on_device must be 0 or 1");
    if (!drain_start_us) {
        dfree(s, s->d_drain);
        s->d_drain = nullptr;
        return SIM_OK;
    }
    const size_t bytes = (size_t)s->cl.num_replicas * (size_t)s->cl.num_instances * 4u;
    if (!s->d_drain) {
        s->d_drain = (uint32_t *)dalloc(s, bytes);
        if (!s->d_drain) return fail(s, SIM_ERR_OOM, "device allocation of the drain schedule failed");
    }
    cudaError_t e = cudaMemcpyAsync(s->d_drain, drain_start_us, bytes,
                                    on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess && !on_device) e = cudaStreamSynchronize(s->stream);  // the host buffer may be reused
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_set_drain copy");
    return SIM_OK;
}

int sim_set_headroom(sim_t *s, const int32_t *headroom_blocks) {
    if (!s) return SIM_ERR_ARG;
    if (!headroom_blocks) return fail(s, SIM_ERR_ARG, "headroom_blocks is NULL");
    const int K = s->K;
    for (int t = 0; t < s->ntables; ++t) {
        long long sum = 0;
        for (int k = 0; k < s->tbl_k[t]; ++k) {
            const int h = headroom_blocks[(size_t)t * K + k];
            if (h < 0) return fail(s, SIM_ERR_ARG, "table %d: negative headroom", t);
            sum += h;
        }
        if (s->cl.blocks_per_instance + sum >= mt::kMaxKeyRange)
            return fail(s, SIM_ERR_ARG, "table %d: M + sum of headroom must be below 2^19", t);
    }
    for (int t = 0; t < s->ntables; ++t)
        for (int k = 0; k < K; ++k)
            s->tbl_h[(size_t)t * K + k] = k < s->tbl_k[t] ? headroom_blocks[(size_t)t * K + k] : 0;
    cudaError_t e = cudaMemcpyAsync(s->d_tbl_h, s->tbl_h.data(), s->tbl_h.size() * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);  // the host vector may change at the next call
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_set_headroom copy");
    if (s->loaded) {
        mt::Params p = make_params(s, 0);
        const int R = s->cl.num_replicas;
        mt::k_set_headroom<<<(R + 7) / 8, 256, 0, s->stream>>>(p, s->d_rep_table, s->d_tbl_k, s->d_tbl_h);
        return check_launch(s, "k_set_headroom");
    }
    return SIM_OK;
}

int sim_set_order(sim_t *s, const int32_t *order) {
    if (!s) return SIM_ERR_ARG;
    if (!order) {
        dfree(s, s->d_order);
        s->d_order = nullptr;
        return SIM_OK;
    }
    const int R = s->cl.num_replicas;
    std::vector<char> seen((size_t)R, 0);
    for (int k = 0; k < R; ++k) {
        const int32_t r = order[k];
        if (r < 0 || r >= R || seen[(size_t)r])
            return fail(s, SIM_ERR_ARG, "order is not a permutation of 0..%d (entry %d = %d)", R - 1, k, (int)r);
        seen[(size_t)r] = 1;
    }
    if (!s->d_order) {
        s->d_order = (int *)dalloc(s, (size_t)R * 4);
        if (!s->d_order) return fail(s, SIM_ERR_OOM, "device allocation of the replica order failed");
    }
    cudaError_t e = cudaMemcpyAsync(s->d_order, order, (size_t)R * 4, cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);  // the host buffer may be reused
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_set_order copy");
    return SIM_OK;
}

int sim_run(sim_t *s, int64_t max_steps, int64_t *num_unfinished) {
    if (!s) return SIM_ERR_ARG;
    if (!s->loaded) return fail(s, SIM_ERR_STATE, "sim_run before sim_load_trace");
    if (max_steps < 1) return fail(s, SIM_ERR_ARG, "max_steps_per_replica must be >= 1");
    cudaError_t e = cudaMemsetAsync(s->d_work, 0, 4, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_run");
    mt::Params p = make_params(s, (long long)max_steps);
    if (p.drains || p.autoscale)
        s->launch.fn_ext<<<s->launch.grid_ext, 32 * mt::kWarpsPerBlock, s->launch.smem, s->stream>>>(p);
    else
        s->launch.fn<<<s->launch.grid, 32 * mt::kWarpsPerBlock, s->launch.smem, s->stream>>>(p);
    int rc = check_launch(s, "k_run");
    if (rc) return rc;
    if (num_unfinished) {
        int cnt = 0;
        e = cudaMemsetAsync(s->d_work + 2, 0, 4, s->stream);
        if (e != cudaSuccess) return cuda_fail(s, e, "sim_run");
        const int R = s->cl.num_replicas;
        mt::k_export_stats<<<(R + 255) / 256, 256, 0, s->stream>>>(s->d_rep, nullptr, R, s->d_work + 2, nullptr);
        rc = check_launch(s, "k_export_stats");
        if (rc) return rc;
        e = cudaMemcpyAsync(&cnt, s->d_work + 2, 4, cudaMemcpyDeviceToHost, s->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
        if (e != cudaSuccess) return cuda_fail(s, e, "sim_run");
        *num_unfinished = cnt;
    }
    return SIM_OK;
}

int sim_metrics(sim_t *s, sim_request_result_t *per_request, sim_replica_stats_t *per_replica,
                sim_migration_event_t *events, int on_device) {
    if (!s) return SIM_ERR_ARG;
    if (!s->loaded) return fail(s, SIM_ERR_STATE, "sim_metrics before sim_load_trace");
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    const int R = s->cl.num_replicas;
    cudaError_t e = cudaSuccess;
    if (per_request && s->qtot > 0)
        e = cudaMemcpyAsync(per_request, s->d_res, (size_t)s->qtot * sizeof(sim_request_result_t), kind, s->stream);
    if (e == cudaSuccess && per_replica) {
        sim_replica_stats_t *dst = per_replica;
        sim_replica_stats_t *tmp = nullptr;
        if (!on_device) {
            tmp = (sim_replica_stats_t *)dalloc(s, (size_t)R * sizeof(sim_replica_stats_t));
            if (!tmp) return fail(s, SIM_ERR_OOM, "device allocation failed");
            dst = tmp;
        }
        if (!s->d_ftc) {
            s->d_ftc = (uint32_t *)dalloc(s, (size_t)R * 4);
            if (!s->d_ftc) return fail(s, SIM_ERR_OOM, "device allocation failed");
        }
        mt::k_first_tokens<<<std::max(1, std::min(R, s->sms * 8)), 256, 0, s->stream>>>(s->d_off, R, s->d_res, s->d_ftc);
        int rc = check_launch(s, "k_first_tokens");
        if (rc) return rc;
        mt::k_export_stats<<<(R + 255) / 256, 256, 0, s->stream>>>(s->d_rep, dst, R, nullptr, s->d_ftc);
        rc = check_launch(s, "k_export_stats");
        if (rc) return rc;
        if (tmp) {
            e = cudaMemcpyAsync(per_replica, tmp, (size_t)R * sizeof(sim_replica_stats_t), cudaMemcpyDeviceToHost,
                                s->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
            dfree(s, tmp);
        }
    }
    if (e == cudaSuccess && events && s->pol.event_log_capacity > 0)
        e = cudaMemcpyAsync(events, s->d_log, (size_t)R * s->pol.event_log_capacity * sizeof(sim_migration_event_t),
                            kind, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "sim_metrics");
    return SIM_OK;
}

void sim_destroy(sim_t *s) {
    if (!s) return;
    cudaStreamSynchronize(s->stream);
    while (!s->bufs.empty()) dfree(s, s->bufs.back().p);
    cudaStreamSynchronize(s->stream);
    cudaGetLastError();
    delete s;
}

}  // extern "C"

// ============================================================================
// Allocation-free entry point: the whole simulation state in one file-scope
// device array (see sim_run_static in mtsim.h).
// ============================================================================
static __device__ __align__(256) unsigned char g_static_scratch[SIM_STATIC_SCRATCH_BYTES];

namespace {

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" int sim_run_static(const sim_cluster_t *cl, const sim_tier_table_t *tt, const sim_policy_t *pol,
                              const int64_t *off, const uint32_t *arrival, const uint16_t *plen,
                              const uint16_t *olen, const uint8_t *tier, sim_request_result_t *per_request,
                              sim_replica_stats_t *per_replica, sim_migration_event_t *events, void *cuda_stream) {
    int rc = validate_config(nullptr, cl, tt, pol);
    if (rc) return rc;
    if (!off) return fail(nullptr, SIM_ERR_ARG, "replica_offsets is NULL");
    const int R = cl->num_replicas;
    if (off[0] != 0) return fail(nullptr, SIM_ERR_TRACE, "replica_offsets[0] must be 0");
    for (int r = 0; r < R; ++r) {
        const int64_t q = off[r + 1] - off[r];
        if (q < 0 || q > (int64_t)0xFFFFFFFEll)
            return fail(nullptr, SIM_ERR_TRACE, "replica_offsets invalid at replica %d", r);
    }
    const int64_t n = off[R];
    if (n > 0 && (!arrival || !plen || !olen || !tier || !per_request))
        return fail(nullptr, SIM_ERR_ARG, "trace and per_request pointers must not be NULL");
    if (!per_replica) return fail(nullptr, SIM_ERR_ARG, "per_replica must not be NULL");
    const int cap = events ? pol->event_log_capacity : 0;

    // Carve the scratch array.
    const int N = cl->num_instances, K = tt->max_tiers;
    const mt::Layout L = mt::make_layout(N, K, cl->tokens_per_block);
    size_t o = 0;
    const size_t o_blobs = o; o = align256(o + (size_t)R * L.bytes);
    const size_t o_slots = o; o = align256(o + (size_t)R * N * cl->max_batch * 16);
    const size_t o_rep = o; o = align256(o + (size_t)R * sizeof(mt::RepState));
    const size_t o_node = o; o = align256(o + (size_t)n * 16);
    const size_t o_off = o; o = align256(o + ((size_t)R + 1) * 8);
    const size_t o_rt = o; o = align256(o + (size_t)R * 4);
    const size_t o_tk = o; o = align256(o + (size_t)tt->num_tables * 4);
    const size_t o_th = o; o = align256(o + (size_t)tt->num_tables * K * 4);
    const size_t o_work = o; o = align256(o + 16);
    const size_t o_ftc = o; o = align256(o + (size_t)R * 4);
    if (o > (size_t)SIM_STATIC_SCRATCH_BYTES)
        return fail(nullptr, SIM_ERR_ARG, "problem needs %zu bytes of scratch; sim_run_static holds %u bytes", o,
                    (unsigned)SIM_STATIC_SCRATCH_BYTES);

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(nullptr, SIM_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    // The array's device address on the current device, looked up on every
    // call: a cached address would be stale after a cudaDeviceReset (the
    // module is loaded again), and nothing shared is written here.
    void *scratch = nullptr;
    e = cudaGetSymbolAddress(&scratch, g_static_scratch);
    if (e != cudaSuccess || !scratch)
        return fail(nullptr, SIM_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    unsigned char *base = (unsigned char *)scratch;
    cudaStream_t st = (cudaStream_t)cuda_stream;

    mt::Launch lc;
    e = mt::plan_launch(R, N, cl->max_batch, L, lc);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e == cudaErrorInvalidConfiguration
                   ? fail(nullptr, SIM_ERR_ARG, "per-replica state does not fit in shared memory")
                   : fail(nullptr, SIM_ERR_CUDA, "sim_run_static launch set-up: %s", cudaGetErrorString(e));
    }
    mt::Params p;
    memset(&p, 0, sizeof p);
    fill_scalars(p, *cl, *pol, K, cap, L, 1LL << 62);
    p.offsets = (const long long *)(base + o_off);
    p.arrival = arrival;
    p.plen = plen;
    p.olen = olen;
    p.tier = tier;
    p.node = (uint4 *)(base + o_node);
    p.res = per_request;
    p.res_off = (const char *)p.res - (const char *)p.node;
    p.blobs = base + o_blobs;
    p.slots = (uint4 *)(base + o_slots);
    p.rep = (mt::RepState *)(base + o_rep);
    p.log = events;
    p.work = (int *)(base + o_work);
    p.set_bits = lc.set_bits;
    p.scratch = lc.scratch;
    int *rt = (int *)(base + o_rt), *tk = (int *)(base + o_tk), *th = (int *)(base + o_th);

    // Inputs the kernels read from device memory; the work counter and flags start at zero.
    e = cudaMemcpyAsync((void *)p.offsets, off, ((size_t)R + 1) * 8, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(rt, tt->replica_table, (size_t)R * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(tk, tt->num_tiers, (size_t)tt->num_tables * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(th, tt->headroom_blocks, (size_t)tt->num_tables * K * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(p.work, 0, 16, st);
    if (e != cudaSuccess) return fail(nullptr, SIM_ERR_CUDA, "sim_run_static copy: %s", cudaGetErrorString(e));
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return fail(nullptr, SIM_ERR_CUDA, "sim_run_static: %s", cudaGetErrorString(e));
    if (n > 0) {
        const long long lim = std::min<long long>((long long)p.M * p.T, 65536);
        const long long nb = std::min<long long>((n + 255) / 256, (long long)sms * 32);
        mt::k_validate<<<(unsigned)std::max<long long>(nb, 1), 256, 0, st>>>(p.offsets, R, arrival, plen, olen, tier,
                                                                              rt, tk, lim, n, p.work + 1);
        int flags = 0;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&flags, p.work + 1, 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess)
            return fail(nullptr, SIM_ERR_CUDA, "sim_run_static validation: %s", cudaGetErrorString(e));
        if (flags) return fail(nullptr, SIM_ERR_TRACE, "malformed trace (validation flags 0x%x)", flags);
    }
    mt::k_init_state<<<(R + 7) / 8, 256, 0, st>>>(p, rt, tk, th);
    if (n > 0) {
        const long long nb = std::min<long long>((n + 255) / 256, 65535LL * 16);
        mt::k_init_requests<<<(unsigned)nb, 256, 0, st>>>(per_request, (long long)n);
    }
    if (p.autoscale)
        lc.fn_ext<<<lc.grid_ext, 32 * mt::kWarpsPerBlock, lc.smem, st>>>(p);
    else
        lc.fn<<<lc.grid, 32 * mt::kWarpsPerBlock, lc.smem, st>>>(p);
    uint32_t *ftc = (uint32_t *)(base + o_ftc);
    mt::k_first_tokens<<<std::max(1, std::min(R, sms * 8)), 256, 0, st>>>(p.offsets, R, per_request, ftc);
    // work[2] (zeroed above) counts the replicas that did not finish
    mt::k_export_stats<<<(R + 255) / 256, 256, 0, st>>>(p.rep, per_replica, R, p.work + 2, ftc);
    int unfinished = 0;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&unfinished, p.work + 2, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(nullptr, SIM_ERR_CUDA, "sim_run_static: %s", cudaGetErrorString(e));
    if (unfinished > 0)
        return fail(nullptr, SIM_ERR_UNFINISHED, "%d of %d replicas did not finish; see per_replica[r].status",
                    unfinished, R);
    return SIM_OK;
}

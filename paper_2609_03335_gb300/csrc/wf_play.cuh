// Device code shared by the sweeps (wf_sweep.cu, wf_batch.cu), the exact int64
// path (wf_eval.cu) and the constructor: the residency queue, the unit records
// and their producer, the finish-time slots, and the p95 selection by a warp.
#pragma once

#include "wf_internal.cuh"

namespace {

__host__ __device__ __forceinline__ uint32_t round16(uint32_t x) { return (x + 15u) & ~15u; }

// A type, or a number, as an argument (the choice of a kernel's instantiation).
template <typename T> struct Ty { using type = T; };
template <int V> struct Iv { static constexpr int value = V; };

__device__ __forceinline__ uint32_t bit_of_g(const uint32_t *row, int32_t n)
{
    return (__ldg(row + (n >> 5)) >> (n & 31)) & 1u;
}

// Dispatch positions of a chunk, the unit in which the stages hand records on;
// a producer warp covers two plans' chunks at once.
constexpr int kChunk = 16;
constexpr int kPlansPerIter = 32 / kChunk;  // plans a producer warp covers per iteration
constexpr int kRecWords = 6;

// Resident models of one device as a queue of 4-bit model ids, least
// recently used in nibble 0; nibbles at and above the count are zero.  A
// 32-bit word holds up to 8 models, a 64-bit word up to 16.
template <typename Q>
struct Lru;

template <>
struct Lru<uint32_t> {
    static constexpr uint32_t kOnes = 0x11111111u, kHigh = 0x88888888u;
    static constexpr int kSlots = 8;
    __device__ static __forceinline__ int32_t find(uint32_t q, uint32_t n, uint32_t m)
    {
        const uint32_t x = q ^ (kOnes * m);
        const uint32_t t = (x - kOnes) & ~x & kHigh;  // lowest zero nibble
        const int32_t k = t ? (__ffs((int)t) - 1) >> 2 : kSlots;
        return k < (int32_t)n ? k : (int32_t)n;
    }
    __device__ static __forceinline__ uint32_t remove(uint32_t q, int32_t k)
    {
        const uint32_t low = q & ((1u << (4 * k)) - 1u);
        const uint32_t high = k < kSlots - 1 ? ((q >> (4 * k + 4)) << (4 * k)) : 0u;
        return low | high;
    }
};

template <>
struct Lru<uint64_t> {
    static constexpr uint64_t kOnes = 0x1111111111111111ull, kHigh = 0x8888888888888888ull;
    static constexpr int kSlots = 16;
    __device__ static __forceinline__ int32_t find(uint64_t q, uint32_t n, uint32_t m)
    {
        const uint64_t x = q ^ (kOnes * m);
        const uint64_t t = (x - kOnes) & ~x & kHigh;
        const int32_t k = t ? (__ffsll((long long)t) - 1) >> 2 : kSlots;
        return k < (int32_t)n ? k : (int32_t)n;
    }
    __device__ static __forceinline__ uint64_t remove(uint64_t q, int32_t k)
    {
        const uint64_t low = k ? (q & ((1ull << (4 * k)) - 1)) : 0ull;
        const uint64_t high = k < kSlots - 1 ? ((q >> (4 * k + 4)) << (4 * k)) : 0ull;
        return low | high;
    }
};

// Unit record (one per plan and dispatch position):
//   w0 run time of the unit (sum over the fused chain, Eq. 4) plus the grant,
//      saturated at 2^32 - 1 (a saturated unit sends its plan to the int64 path)
//   w1 KV admission of the unit (largest on the chain, Eq. 4); the residency
//      stage overwrites it with the load time the unit waits for (0 on a hit)
//   w2 arrival time of the unit's session
//   w3 device | model << 5 | prefetch << 9 | reclaim << 10 | writes << 11 | skip << 14
//      | first write code << 16; the residency stage clears the prefetch bit
//      on a hit and sets kWasEmpty (bit 10) and kEmptied (bit 15) for timing
//   w4 second write code | third write code << 16
//   w5 the unit's last member | release slot code << 16 (bit 31: accumulator;
//      0xFFFF: none); in the batched producer's records the low half holds
//      the fourth write code instead when the unit writes exactly four (with
//      five or more, the timing stage reads the last member's list)
constexpr uint32_t kSkip = 1u << 14;
constexpr uint32_t kPrefetch = 1u << 9;
constexpr uint32_t kDrop = 1u << 10;       // before residency: the unit's model leaves when it ends (retain bit 0)
constexpr uint32_t kWasEmpty = 1u << 10;   // after residency: a miss on an empty device
constexpr uint32_t kEmptied = 1u << 15;    // after residency: the unit's reclaim empties the device
constexpr uint32_t kRunCap = 0xFFFFFFFFu;  // saturation of w0
// The writes field: 0 for up to two codes (which every record holds), 4 for
// three, 5 for four, 6 for more; kMany tests for more than two.
constexpr uint32_t kMany = 1u << 13;
constexpr uint32_t kWrites4 = 5;
// A plan's open word in shared memory: the devices still occupied at its end
// (residency, low bits) and, from bit kOpenBad, the placement status bits
// (WF_ST_DEVICE, WF_ST_CAPACITY) its producers found.
constexpr int kOpenBad = 24;


// One unit on its device under least-recently-used reclamation (Eq. 11,
// Section 3.5): q / n / u_d are the device's queue, resident count and
// resident weights.  The unit's own model leaves the queue first; the
// victims are then exactly the queue's first entries (least recently used
// first), and the unit's model goes back in as the most recently used.
// Returns the record's rewritten (w1, w3): the load the unit waits for (none
// on a hit, Eq. 5) and the occupancy changes of section 4.3.
template <typename Q>
__device__ __forceinline__ uint2 settle_lru(Q &q, uint32_t &n, uint32_t &u_d, uint32_t capd, uint32_t r1,
                                            uint32_t r3, const int32_t *weight, const int32_t *load, int32_t D,
                                            int *err, bool &missed)
{
    const int32_t d = (int32_t)(r3 & 31u);
    const uint32_t m = (r3 >> 5) & 15u;
    const uint32_t wm = (uint32_t)weight[m];
    const bool was_empty = n == 0;
    const int32_t kq = Lru<Q>::find(q, n, m);
    const bool hit = kq < (int32_t)n;
    missed = !hit;
    q = hit ? Lru<Q>::remove(q, hit ? kq : 0) : q;  // (an index below the queue length)
    n -= hit ? 1u : 0u;
    const uint32_t need = hit ? r1 : wm + r1;  // used + need <= cap + peak < 2^32
    uint32_t e = 0;
    while (u_d + need > capd && e < n) {
        u_d -= (uint32_t)weight[(uint32_t)(q >> (4 * e)) & 15u];
        ++e;
    }
    if (u_d + need > capd) atomicExch(err, 2);  // unreachable for a valid plan
    q = e < (uint32_t)Lru<Q>::kSlots ? (q >> (4 * e)) : (Q)0;
    n -= e;
    q |= (Q)m << (4 * n);
    n += 1;
    u_d += hit ? 0u : wm;
    uint32_t emptied = 0;
    if ((r3 >> 10) & 1u) {  // retain bit 0: reclaim at the end of the unit
        q &= ~((Q)0xF << (4 * (n - 1)));
        n -= 1;
        u_d -= wm;
        emptied = n == 0;
    }
    return make_uint2(hit ? 0u : (uint32_t)load[m * D + d],
                      (r3 & ~(kPrefetch | kWasEmpty)) | (hit ? 0u : (r3 & kPrefetch)) |
                          (was_empty ? kWasEmpty : 0u) | (emptied ? kEmptied : 0u));
}

// Residency of one device under least-recently-used reclamation in one
// word (shared memory in the sweeps, a lane's registers on the int64 path): the queue of 4-bit model ids, least recently used in
// nibble 0, empty places 0xF, and the free capacity (capacity minus resident
// weights); up to 8 models the queue says its own length (no id has bit 3
// set), beyond it is kept beside.  settle() plays a unit's admission (Eq. 11,
// Section 3.5): the unit's own model leaves the queue first, the victims are
// then its first entries, and the model goes back in last.  The first three
// victims' weights are read at once and taken without branching (a loop over
// victims waited for one weight at a time: about 130 instructions a unit with
// it, half of that without); kRare: where few lanes settle at once and a unit
// seldom evicts, that is skipped.  weight holds 16 entries, 0 beyond the models.
// Returns the record's rewritten (w1, w3): the
// load the unit waits for (none on a hit, Eq. 5) and the occupancy changes.
template <typename Q>
struct DevState;

// The victims: from `need` and the free capacity f, the shift that drops the
// evicted entries from queue q (at most n4 / 4 of them).
template <typename Q>
__device__ __forceinline__ int evict(Q q, uint32_t need, uint32_t &f, int n4, const int32_t *weight)
{
    const uint32_t w0 = (uint32_t)weight[(uint32_t)q & 15u], w1 = (uint32_t)weight[(uint32_t)(q >> 4) & 15u],
                   w2 = (uint32_t)weight[(uint32_t)(q >> 8) & 15u];
    int e4 = 0;
    if (need > f) { f += w0; e4 = 4; }
    if (need > f) { f += w1; e4 = 8; }
    if (need > f) { f += w2; e4 = 12; }
    for (; need > f && e4 < n4; e4 += 4) f += (uint32_t)weight[(uint32_t)(q >> e4) & 15u];
    return min(e4, n4);
}

__device__ __forceinline__ uint2 settled(uint32_t r3, bool hit, uint32_t ld, bool was_empty, bool emptied)
{
    return make_uint2(hit ? 0u : ld, (r3 & ~(hit ? kPrefetch | kWasEmpty : kWasEmpty)) | (was_empty ? kWasEmpty : 0u) |
                                         (emptied ? kEmptied : 0u));
}

template <>
struct DevState<uint32_t> {
    uint2 v;  // queue, free capacity
    __device__ __forceinline__ void init(uint32_t cap) { v = make_uint2(~0u, cap); }
    __device__ __forceinline__ bool occupied() const { return v.x != ~0u; }
    template <bool kRare = false>
    __device__ __forceinline__ uint2 settle(uint32_t r1, uint32_t r3, const int32_t *weight, const int32_t *load,
                                            int32_t D, int *err, bool &missed)
    {
        const uint32_t m = (r3 >> 5) & 15u, wm = (uint32_t)weight[m], ld = (uint32_t)load[m * D + (r3 & 31u)];
        uint32_t q = v.x, f = v.y;
        const bool was_empty = q == ~0u;
        const uint32_t x = q ^ (0x11111111u * m);
        const uint32_t z = (x - 0x11111111u) & ~x & 0x88888888u;  // its lowest bit: the nibble equal to m
        const bool hit = z != 0;
        missed = !hit;
        const uint32_t below = ((z & (0u - z)) >> 3) - 1u;  // the bits below that nibble (all when there is none)
        q = (q & below) | ((q >> 4) & ~below) | 0xF0000000u;
        const uint32_t need = hit ? r1 : wm + r1;  // at most the capacity
        int e4 = 0;
        if (!kRare || need > f) e4 = evict(q, need, f, 32, weight);
        if (need > f) atomicExch(err, 2);  // unreachable for a valid plan
        q = __funnelshift_rc(q, ~0u, e4);
        const uint32_t gap = q & 0x88888888u;
        const uint32_t at = (gap & (0u - gap)) >> 3;  // 1 << 4 n: the first empty place
        const uint32_t with = q - (15u - m) * at;     // 0xF there becomes m
        f -= hit ? 0u : wm;
        bool emptied = false;
        if (r3 & kDrop) {  // the model leaves when the unit ends
            f += wm;
            emptied = q == ~0u;
        } else {
            q = with;
        }
        v = make_uint2(q, f);
        return settled(r3, hit, ld, was_empty, emptied);
    }
};

template <>
struct DevState<uint64_t> {
    uint4 v;  // queue (low, high), free capacity, models held
    __device__ __forceinline__ void init(uint32_t cap) { v = make_uint4(~0u, ~0u, cap, 0u); }
    __device__ __forceinline__ bool occupied() const { return v.w != 0; }
    template <bool kRare = false>
    __device__ __forceinline__ uint2 settle(uint32_t r1, uint32_t r3, const int32_t *weight, const int32_t *load,
                                            int32_t D, int *err, bool &missed)
    {
        const uint32_t m = (r3 >> 5) & 15u, wm = (uint32_t)weight[m], ld = (uint32_t)load[m * D + (r3 & 31u)];
        uint64_t q = ((uint64_t)v.y << 32) | v.x;
        uint32_t f = v.z, n = v.w;
        const bool was_empty = n == 0;
        const uint64_t x = q ^ (0x1111111111111111ull * m);
        const uint64_t z = (x - 0x1111111111111111ull) & ~x & 0x8888888888888888ull;
        const uint64_t low = (z & (0ull - z)) >> 3;
        // (with 16 models the empty places match the last one)
        const bool hit = low != 0 && (uint32_t)__popcll(low - 1) < 4 * n;
        missed = !hit;
        const uint64_t below = hit ? low - 1 : ~0ull;
        q = (q & below) | ((q >> 4) & ~below) | (hit ? 0xFull << 60 : 0ull);
        n -= hit ? 1u : 0u;
        const uint32_t need = hit ? r1 : wm + r1;
        int e4 = 0;
        if (!kRare || need > f) e4 = evict(q, need, f, (int)(4 * n), weight);
        if (need > f) atomicExch(err, 2);  // unreachable for a valid plan
        q = e4 < 64 ? (q >> e4) | ~(~0ull >> e4) : ~0ull;
        n -= (uint32_t)e4 >> 2;
        f -= hit ? 0u : wm;
        bool emptied = false;
        if (r3 & kDrop) {
            f += wm;
            emptied = n == 0;
        } else {
            q ^= (uint64_t)(15u ^ m) << (4 * n);
            n += 1;
        }
        v = make_uint4((uint32_t)q, (uint32_t)(q >> 32), f, n);
        return settled(r3, hit, ld, was_empty, emptied);
    }
};

// The r-th smallest (0-based) of n values a.get(i), by a whole warp.  The p95's rank is near the top (the
// (n - r)-th largest: 4th of 64, 13th of 256), so the warp takes maxima: the
// largest value up to a bound, first ~0 and then one below the last maximum,
// and how many equal it, until the count reaches n - r.  (Every step counts at
// least one value, whatever the values are: when the maximum is 0, all that
// are left are 0, and enough of them.)  For a rank further down, a radix selection from the
// highest bit set in any value, each bit decided by a ballot.  Up to 32
// kCache values are read once into registers (a column of the slot array is
// a strided read with bank conflicts); more are read again for every step.
template <int kCache, typename SA, typename F>
__device__ __forceinline__ void each_value(const SA &a, int32_t n, bool cached, const uint64_t (&c)[kCache], F &&f)
{
    const int lane = threadIdx.x & 31;
    if (cached) {
#pragma unroll
        for (int j = 0; j < kCache; ++j)
            if (32 * j < n) f(c[j], 32 * j + lane < n);
    } else {
        for (int32_t i0 = 0; i0 < n; i0 += 32) {
            const int32_t i = i0 + lane;
            f(i < n ? (uint64_t)a.get(i) : 0ull, i < n);
        }
    }
}

template <int kCache = 8, typename SA>
__device__ uint64_t warp_select(const SA &a, int32_t n, int32_t r)
{
    constexpr int32_t kMaxSteps = 32;
    const int lane = threadIdx.x & 31;
    const bool cached = n <= 32 * kCache;
    uint64_t c[kCache];  // the values, 0 beyond n (never above the answer when taking maxima)
#pragma unroll
    for (int j = 0; j < kCache; ++j) {
        const int32_t i = 32 * j + lane;
        c[j] = cached && i < n ? (uint64_t)a.get(i) : 0ull;
    }
    if (n - r <= kMaxSteps) {
        int32_t need = n - r;  // the need-th largest of the values up to top
        uint64_t top = ~0ull;
        for (;;) {
            uint64_t mx = 0;
            each_value(a, n, cached, c, [&](uint64_t v, bool) {
                if (v <= top) mx = max(mx, v);
            });
            const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(mx >> 32));
            const uint32_t lo = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(mx >> 32) == hi ? (uint32_t)mx : 0u);
            const uint64_t m = ((uint64_t)hi << 32) | lo;
            int32_t cnt = 0;
            each_value(a, n, cached, c, [&](uint64_t v, bool in) {
                cnt += __popc(__ballot_sync(0xFFFFFFFFu, in && v == m));
            });
            if (cnt >= need) return m;
            need -= cnt;
            top = m - 1;
        }
    }
    uint64_t any = 0;
    each_value(a, n, cached, c, [&](uint64_t v, bool) { any |= v; });
    any = ((uint64_t)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)(any >> 32)) << 32) |
          __reduce_or_sync(0xFFFFFFFFu, (uint32_t)any);
    uint64_t prefix = 0;
    for (int bit = any ? 63 - __clzll((long long)any) : -1; bit >= 0; --bit) {
        int32_t zeros = 0;  // values that match prefix above bit and have a 0 there
        each_value(a, n, cached, c, [&](uint64_t v, bool in) {
            zeros += __popc(__ballot_sync(0xFFFFFFFFu, in && ((v ^ prefix) >> bit) == 0));
        });
        if (r >= zeros) {
            r -= zeros;
            prefix |= 1ull << bit;
        }
    }
    return prefix;
}

// Two extra slots follow a plan's nslots slots: a sink that absorbs writes
// with no reader (index nslots) and a slot that always holds 0 (nslots + 1),
// the release slot of a node without predecessors.  With them every unit
// reads one release slot and writes its first two codes without branching;
// the host encodes both into the per-node records (hrec).

// Storage of the finish-time slots, [slot][plan]: TT words, or (Split40, for
// u64 times whose every value stays below 2^40 us) a 32-bit low word per
// slot and an 8-bit high byte in an array of its own: 5 bytes instead of 8,
// so more plans fit an SM.
struct Split40 {};

// No time of any plan of the window can reach 2^40 us (the context's horizon
// bounds every finish: even a plan that plays its units one by one, each
// waiting for a load).
inline bool below40(const wf_dev_problem &dp) { return dp.horizon < ((int64_t)1 << 40); }

template <typename ST>
struct SlotBytes {
    static constexpr uint32_t kLo = sizeof(ST), kHi = 0;
};
template <>
struct SlotBytes<Split40> {
    static constexpr uint32_t kLo = 4, kHi = 1;
};
template <typename TT, typename ST, int kS>
struct SlotArr {  // plain words
    TT *v;
    __device__ __forceinline__ TT get(uint32_t i) const { return v[i * kS]; }
    __device__ __forceinline__ void set(uint32_t i, TT x) const { v[i * kS] = x; }
};
template <int kS>
struct SlotArr<uint64_t, Split40, kS> {
    uint32_t *lo;
    uint8_t *hi;
    __device__ __forceinline__ uint64_t get(uint32_t i) const
    {
        return ((uint64_t)hi[i * kS] << 32) | lo[i * kS];
    }
    __device__ __forceinline__ void set(uint32_t i, uint64_t x) const
    {
        lo[i * kS] = (uint32_t)x;
        hi[i * kS] = (uint8_t)(x >> 32);
    }
};

__device__ __forceinline__ void named_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void named_arrive(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Row of one plan for the batched producer: placement and dispatch rows, and
// the byte offset of its fusion / prefetch / retain bit rows.
struct RowPtrs {
    const uint8_t *place;
    const uint16_t *order;
    int64_t boff;
};

__device__ __forceinline__ const uint32_t *bits_row(const uint32_t *base, int64_t boff)
{
    return (const uint32_t *)((const uint8_t *)base + boff);
}

// Bulk prefetch of [p, p + bytes) into L2 (p 16-byte aligned, bytes a
// multiple of 16); no completion to wait for.
__device__ __forceinline__ void l2_prefetch(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// A record that starts no unit, which the timing stages may also play: no run
// time, no load, device 0, the zero slot read and the sink written.
template <int kPitch>
__device__ __forceinline__ void skip_record(uint2 *dst, uint32_t sink)
{
    dst[0] = make_uint2(0u, 0u);
    dst[1 * kChunk * kPitch] = make_uint2(0u, kSkip | (sink << 16));
    dst[2 * kChunk * kPitch] = make_uint2(sink | (sink << 16), (sink + 1) << 16);
}

// The records of kI (plan, position) pairs at once, with the gathers of all
// pairs issued together in three dependent rounds: the head's own tables
// (placement, node record, fusion / prefetch / retain words, third and
// fourth write codes); then its run time and KV on its device and the placement and fusion
// bit of its fusible neighbours; then the rare fused chain, walked as in
// produce().  Each record goes to the ring as soon as it is complete; act[j]
// false leaves a skip record.  dev[j] is the unit's device (all ones for a
// skip record).
template <int kI, int kPitch>
__device__ __forceinline__ void produce_batch(const wf_dev_problem &dp, const wf_plans &pl, const RowPtrs *rp,
                                              const bool *act, const int32_t *hh, uint2 *rb, int pos,
                                              const int *qq, uint32_t *dev, uint32_t *open)
{
    const int32_t D = dp.D;
    uint32_t d[kI], fw[kI], pw[kI], rw[kI], c2[kI], bad[kI];
    uint4 hr[kI];
#pragma unroll
    for (int j = 0; j < kI; ++j) {
        const int32_t h = hh[j];
        d[j] = act[j] ? __ldg(rp[j].place + h) : 0u;
        hr[j] = act[j] ? __ldg(dp.hrec + h) : make_uint4(0xFFFFFFFFu, 0, 0, 0);
        fw[j] = act[j] ? __ldg(bits_row(pl.fuse, rp[j].boff) + (h >> 5)) : 0u;
        pw[j] = act[j] ? __ldg(bits_row(pl.prefetch, rp[j].boff) + (h >> 5)) : 0u;
        rw[j] = act[j] && pl.retain ? __ldg(bits_row(pl.retain, rp[j].boff) + (h >> 5)) : 0xFFFFFFFFu;
        c2[j] = act[j] ? __ldg(dp.wc23 + h) : 0u;
    }
    // Placement and fit (Eq. 8) of every position's activation: a device
    // index beyond D here, a device it does not fit (KV entry -1 in lk) with
    // the next gathers.  A plan with either gets the status bits, and the
    // record a skip, so no later stage indexes by it.
#pragma unroll
    for (int j = 0; j < kI; ++j) {
        bad[j] = act[j] && d[j] >= (uint32_t)D ? (uint32_t)WF_ST_DEVICE : 0u;
        if (bad[j]) d[j] = 0u;
    }
    int2 lk0[kI];
    uint32_t pprev[kI], fnx[kI], pnx[kI];
#pragma unroll
    for (int j = 0; j < kI; ++j) {
        const uint32_t fp = hr[j].x & 0xFFFFu, s = hr[j].x >> 16;
        lk0[j] = act[j] ? __ldg(dp.lk + hh[j] * D + (int32_t)d[j]) : make_int2(0, 0);
        pprev[j] = act[j] && fp != 0xFFFFu ? __ldg(rp[j].place + fp) : 0xFFFFFFFFu;  // never a device
        fnx[j] = act[j] && s != 0xFFFFu ? __ldg(bits_row(pl.fuse, rp[j].boff) + (s >> 5)) : 0u;
        pnx[j] = act[j] && s != 0xFFFFu ? __ldg(rp[j].place + s) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int j = 0; j < kI; ++j) {
        dev[j] = 0xFFFFFFFFu;
        if (qq[j] < 0) continue;  // a lane beyond the CTA's plans
        uint2 *dst = rb + pos * kPitch + qq[j];
        const int32_t h = hh[j];
        const uint32_t s0 = hr[j].x >> 16;
        if (act[j] && !bad[j] && lk0[j].y < 0) bad[j] = (uint32_t)WF_ST_CAPACITY;  // (d was cleared for a bad device)
        if (bad[j]) atomicOr(open + qq[j], bad[j] << kOpenBad);
        if (!act[j] || bad[j] || (((fw[j] >> (h & 31)) & 1u) && pprev[j] == d[j])) {  // no unit, or inside its head's
            skip_record<kPitch>(dst, (uint32_t)dp.nslots);
            continue;
        }
        uint32_t run = (uint32_t)lk0[j].x + (uint32_t)dp.grant, ovf = 0;  // both < 2^31: no wrap
        int32_t kv = lk0[j].y, tail = h;
        uint32_t ty = hr[j].y, tw = hr[j].w, c2t = c2[j], rwt = rw[j];
        uint32_t cbad = 0;  // a member that does not fit the head's device
        if (s0 != 0xFFFFu && ((fnx[j] >> (s0 & 31)) & 1u) && pnx[j] == d[j]) {  // Eq. 3 chain
            const uint32_t *fuse = bits_row(pl.fuse, rp[j].boff);
            for (uint32_t s = s0; s != 0xFFFFu;) {
                if (s != s0 && (!bit_of_g(fuse, s) || __ldg(rp[j].place + s) != d[j])) break;
                const int2 lk = __ldg(dp.lk + s * D + d[j]);
                cbad |= lk.y < 0;
                const uint4 sr = __ldg(dp.hrec + s);
                const uint32_t r2 = run + (uint32_t)lk.x;
                ovf |= r2 < run;
                run = r2;
                kv = max(kv, lk.y);
                tail = (int32_t)s;
                ty = sr.y;
                tw = sr.w;
                s = sr.x >> 16;
            }
            c2t = __ldg(dp.wc23 + tail);
            rwt = pl.retain ? __ldg(bits_row(pl.retain, rp[j].boff) + (tail >> 5)) : 0xFFFFFFFFu;
        }
        if (cbad) {  // (the member's own position flags the plan as well)
            atomicOr(open + qq[j], (uint32_t)WF_ST_CAPACITY << kOpenBad);
            skip_record<kPitch>(dst, (uint32_t)dp.nslots);
            continue;
        }
        const uint32_t nwl = (ty >> 20) & 7u, rs = hr[j].y & 0xFFFFu;
        // A code naming the accumulator that this unit reads and resets finds 0 there: a plain write.
        if ((tw & 0xFFFFu) == rs) tw &= 0xFFFF7FFFu;
        if ((tw >> 16) == rs) tw &= 0x7FFFFFFFu;
        const uint32_t pf = (pw[j] >> (h & 31)) & 1u;
        const uint32_t reclaim = ((rwt >> (tail & 31)) & 1u) ^ 1u;
        dst[0] = make_uint2(ovf ? kRunCap : run, hr[j].z);
        dst[1 * kChunk * kPitch] = make_uint2(
            (uint32_t)kv, d[j] | (((hr[j].y >> 16) & 15u) << 5) | (pf << 9) | (reclaim << 10) | (nwl << 11) | (tw << 16));
        dst[2 * kChunk * kPitch] = make_uint2((tw >> 16) | (c2t << 16),
                                              (nwl == kWrites4 ? c2t >> 16 : (uint32_t)tail) | (hr[j].y << 16));
        dev[j] = d[j];
    }
}

// a + b on 32 bits; the carry is counted in ovf.
__device__ __forceinline__ uint32_t add_carry(uint32_t a, uint32_t b, uint32_t &ovf)
{
    uint32_t c;
    asm("add.cc.u32 %0, %2, %3;\n\taddc.u32 %1, %1, 0;" : "=r"(c), "+r"(ovf) : "r"(a), "r"(b));
    return c;
}

// A finish time into a slot: an accumulator keeps the latest of its
// writers, any other slot takes the value.
template <typename TT, typename SA>
__device__ __forceinline__ void publish(const SA &slots, uint32_t code, TT c)
{
    const uint32_t i = code & 0x7FFFu;
    slots.set(i, (code & 0x8000u) ? max(slots.get(i), c) : c);
}

}  // namespace

// Replica batch limit B_q (Eq. 11 over the running units, Section 3.5; the
// reading of the oracle's simulate_batched): producer warps build the unit
// records, and play warps settle each unit's admission and timing together --
// under the limit an admission waits for running units to end, so residency
// cannot be settled ahead of the times.
//
// A play warp holds 32 / kL plans, kL lanes each (8 or 16 by the device
// count); lane g of a plan is its device g, and beyond 16 devices its device g
// + 16 as well, and keeps that device's state in registers: the current replica's model, the last admission, the residency
// queue, resident weights and count, the occupancy balance and, up to four of
// them, the running slots (beyond, those are in shared memory, in the lane's
// own column).  Every lane walks the chunk's positions; a unit is played by
// its device's lane, so the plans of a warp play side by side and nothing is
// indexed by device.  Finish slots are shared by the plan's lanes.
//
// Times are u32 first: a plan that leaves 32 bits is listed, and a second
// instantiation with u64 times plays the list (or, once a context has seen
// most plans leave 32 bits, the whole batch).  A unit whose summed run time
// saturates 32 bits sends its plan on to the exact int64 path.
//
// Bound by the length of a unit's play (one dependent chain, with both ways
// an admission can go when the warp's plans differ) times the plans an SM
// holds.  Burst window, 16,384 plans, B_q = 4: 11.16 ms with a lane per plan
// and all state in shared memory, 7.52 ms with a lane per device on u64 times
// and slots in shared memory (108 warp instructions per plan-position),
// 4.48 ms with u32 times and the running slots in registers (65, in 39 % of
// the issue slots).
#include <algorithm>

#include "wf_play.cuh"

namespace {

constexpr int kBqPlans = 8;   // plans per CTA
constexpr int kBqIters = 2;   // plan pairs per producer warp
constexpr int kBqProducers = kBqPlans / (kPlansPerIter * kBqIters);
constexpr int kBqBuffers = 4;
constexpr int kBqPitch = kBqPlans | 1;
constexpr int kBqFull = 1, kBqEmpty = kBqFull + kBqBuffers;  // named barriers
constexpr int kBqRegs = 4;    // running slots kept in registers
static_assert(kBqEmpty + kBqBuffers <= 16, "named barriers");

template <int kL, int kDev, int kB>
struct BqShape {
    static constexpr int kPlay = kBqPlans * kL / 32;  // play warps
    static constexpr int kWarps = kPlay + kBqProducers;
    // Six CTAs of 8-device plans share an SM at 2,000 activations.  With two
    // devices a lane three CTAs do where both devices' running slots are
    // registers (92 to 96 a thread), else four.  65,536 plans of N = 32, D = 32, B_q =
    // 1, 4, 8, us: 32 lanes a plan, a device each, 575, 577, 768; 16 lanes, two
    // devices each, 437, 442, 503 (a lane a plan with its state in shared
    // memory 487, 537, 751).
    static constexpr int kMinBlocks = kL == 8 ? 6 : kDev == 1 ? 4 : kB ? 3 : 4;
};

struct BqLayout {
    uint32_t weight, cap, load, arr, ring, slots, slots_hi, se, sk, open, total;
};

// Shared memory of a CTA: TT times in ST slots, NS finish slots per plan; the
// running slots' columns when they exceed the registers (or TT is u64).
template <typename TT, typename ST>
__host__ __device__ inline BqLayout bq_layout(int32_t D, int32_t M, int32_t W, int32_t B, int32_t NS)
{
    constexpr uint32_t P = kBqPlans;
    const uint32_t cols = sizeof(TT) == 4 && B <= kBqRegs ? 0u : (uint32_t)(B * D) * P;
    BqLayout l;
    uint32_t o = 0;
    l.weight = o; o += round16(4u * M);
    l.cap = o; o += round16(4u * D);
    l.load = o; o += round16(4u * M * D);
    l.arr = o; o += round16(4u * W);
    l.ring = o; o += round16(8u * kBqBuffers * 3 * kChunk * kBqPitch);
    l.slots = o; o += round16(SlotBytes<ST>::kLo * (uint32_t)NS * P);
    l.slots_hi = o; o += round16(SlotBytes<ST>::kHi * (uint32_t)NS * P);
    l.se = o; o += (uint32_t)sizeof(TT) * cols;
    l.sk = o; o += 4u * cols;
    l.open = o; o += round16(4u * P);
    l.total = o;
    return l;
}

template <typename T>
__device__ __forceinline__ void exchange_if(bool c, T &a, T &b)
{
    const T t = a;
    a = c ? b : a;
    b = c ? t : b;
}

// The running slots of one device: each one's end and KV (0 and 0 when free).
template <typename TT, int kB>
struct Running {  // in registers, B <= kB of them
    TT e[kB];
    uint32_t kv[kB];
    __device__ __forceinline__ void init(int, TT *, uint32_t *, int)
    {
#pragma unroll
        for (int j = 0; j < kB; ++j) { e[j] = 0; kv[j] = 0; }
    }
    // f(slot, end, KV) over the B slots in order.
    template <typename F>
    __device__ __forceinline__ void each(int B, F &&f) const
    {
#pragma unroll
        for (int j = 0; j < kB; ++j)
            if (j < B) f(j, e[j], kv[j]);
    }
    __device__ __forceinline__ void reset(int, TT t)
    {
#pragma unroll
        for (int j = 0; j < kB; ++j) { e[j] = t; kv[j] = 0; }
    }
    __device__ __forceinline__ void put(int slot, TT t, uint32_t k)
    {
#pragma unroll
        for (int j = 0; j < kB; ++j)
            if (j == slot) { e[j] = t; kv[j] = k; }
    }
    __device__ __forceinline__ void swap_if(bool c, Running &o)
    {
#pragma unroll
        for (int j = 0; j < kB; ++j) { exchange_if(c, e[j], o.e[j]); exchange_if(c, kv[j], o.kv[j]); }
    }
};
template <typename TT>
struct Running<TT, 0> {  // in the lane's column of shared memory
    TT *e;
    uint32_t *kv;
    int cols;
    __device__ __forceinline__ void init(int B, TT *se, uint32_t *sk, int c)
    {
        e = se; kv = sk; cols = c;
        for (int j = 0; j < B; ++j) { e[j * cols] = 0; kv[j * cols] = 0; }
    }
    template <typename F>
    __device__ __forceinline__ void each(int B, F &&f) const
    {
        for (int j = 0; j < B; ++j) f(j, e[j * cols], kv[j * cols]);
    }
    __device__ __forceinline__ void reset(int B, TT t)
    {
        for (int j = 0; j < B; ++j) { e[j * cols] = t; kv[j * cols] = 0; }
    }
    __device__ __forceinline__ void put(int slot, TT t, uint32_t k)
    {
        e[slot * cols] = t;
        kv[slot * cols] = k;
    }
    __device__ __forceinline__ void swap_if(bool c, Running &o) { exchange_if(c, e, o.e); exchange_if(c, kv, o.kv); }
};

// The device of a lane that is not being played, when it has two.
template <typename Q, typename TT, int kB>
struct OtherDevice {
    Q queue = 0;
    uint32_t n = 0, used = 0, cur = 0xFFFFFFFFu, cap = 0;
    TT ladm = 0;
    Running<TT, kB> slots;
};

// Groups of kBqPlans plans: every plan of the batch (in_list null, a CTA per
// group) or the listed ones (CTAs walk over groups).
template <typename Q, int kL, int kDev, typename TT, typename ST, int kB>
__global__ void __launch_bounds__(32 * BqShape<kL, kDev, kB>::kWarps, BqShape<kL, kDev, kB>::kMinBlocks)
bq_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, const int32_t *in_list, const int32_t *in_count,
          int32_t *ovf_list, int32_t *ovf_count)
{
    constexpr int kP = kBqPlans, kPitch = kBqPitch;
    constexpr int kPlay = BqShape<kL, kDev, kB>::kPlay;
    constexpr int kThreads = 32 * BqShape<kL, kDev, kB>::kWarps;
    constexpr bool kNarrow = sizeof(TT) == 4;
    extern __shared__ __align__(128) uint8_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W, B = dp.batch;
    const BqLayout L = bq_layout<TT, ST>(D, M, W, B, dp.nslots + 2);
    const int64_t total = in_list ? (int64_t)*in_count : pl.P;
    if ((int64_t)blockIdx.x * kP >= total) return;  // the whole CTA: no plan
    uint2 *ring = (uint2 *)(sm + L.ring);
    const int32_t chunks = (N + kChunk - 1) / kChunk;
    int32_t *weight = (int32_t *)(sm + L.weight);
    int32_t *cap = (int32_t *)(sm + L.cap);
    int32_t *load = (int32_t *)(sm + L.load);
    uint32_t *arrival = (uint32_t *)(sm + L.arr);
    uint32_t *open = (uint32_t *)(sm + L.open);  // placement status bits from the producers (bit kOpenBad on)
    for (int32_t k = threadIdx.x; k < M; k += blockDim.x) weight[k] = __ldg(dp.weight + k);
    for (int32_t k = threadIdx.x; k < D; k += blockDim.x) cap[k] = __ldg(dp.cap + k);
    for (int32_t k = threadIdx.x; k < M * D; k += blockDim.x) load[k] = __ldg(dp.load + k);
    for (int32_t k = threadIdx.x; k < W; k += blockDim.x) arrival[k] = (uint32_t)__ldg(dp.arrival + k);

  for (int64_t j0 = (int64_t)blockIdx.x * kP; j0 < total; j0 += (int64_t)gridDim.x * kP) {
    const int ng = (int)(total - j0 < kP ? total - j0 : kP);
    const auto plan_of = [&](int q) { return in_list ? (int64_t)__ldg(in_list + j0 + q) : j0 + q; };
    if (threadIdx.x < kP) open[threadIdx.x] = 0;

    if (warp >= kPlay) {
        // ---------------- producers: lane = dispatch position (as in pc_kernel) ----------------
        __syncthreads();
        const int pw = warp - kPlay;
        const int pos = lane % kChunk, sub = lane / kChunk;
        RowPtrs rp[kBqIters];
        int qq[kBqIters];
        bool ok[kBqIters];
        int32_t h0[kBqIters];
        const uint32_t place_bytes = (uint32_t)((N + 15) & ~15), bits_bytes = (uint32_t)((((N + 31) >> 5) * 4 + 15) & ~15);
#pragma unroll
        for (int j = 0; j < kBqIters; ++j) {
            const int q = (pw * kBqIters + j) * kPlansPerIter + sub;  // one plan per half-warp
            qq[j] = q;
            ok[j] = q < ng;
            rp[j].place = nullptr;
            rp[j].order = nullptr;
            rp[j].boff = 0;
            if (ok[j]) {
                const int64_t pq = plan_of(q);
                ok[j] = __ldg(out.status + pq) == 0;
                rp[j].place = pl.place + pq * pl.place_stride;
                rp[j].order = (const uint16_t *)((const uint8_t *)pl.order + pq * pl.order_stride);
                rp[j].boff = pq * pl.bits_stride;
            }
            if (pos == 0 && ok[j]) {
                l2_prefetch(rp[j].place, place_bytes);
                l2_prefetch(bits_row(pl.fuse, rp[j].boff), bits_bytes);
                l2_prefetch(bits_row(pl.prefetch, rp[j].boff), bits_bytes);
            }
            h0[j] = ok[j] && pos < N ? (int32_t)__ldg(rp[j].order + pos) : 0;
        }
        for (int32_t c = 0; c < chunks; ++c) {
            const int b = c % kBqBuffers;
            if (c >= kBqBuffers) named_sync(kBqEmpty + b, kThreads);  // the play warps released buffer b
            uint2 *rb = ring + b * 3 * kChunk * kPitch;
            const int32_t i = c * kChunk + pos;
            int32_t h1[kBqIters];
            bool act[kBqIters];
#pragma unroll
            for (int j = 0; j < kBqIters; ++j) {
                h1[j] = ok[j] && i + kChunk < N ? (int32_t)__ldg(rp[j].order + i + kChunk) : 0;
                act[j] = ok[j] && i < N;
            }
            uint32_t dev[kBqIters];
            produce_batch<kBqIters, kPitch>(dp, pl, rp, act, h0, rb, pos, qq, dev, open);
#pragma unroll
            for (int j = 0; j < kBqIters; ++j) h0[j] = h1[j];
            named_arrive(kBqFull + b, kThreads);  // buffer b is full
        }
        for (int32_t c = chunks; c < chunks + kBqBuffers; ++c)
            if (c >= kBqBuffers) named_sync(kBqEmpty + c % kBqBuffers, kThreads);
    } else {
    // ---------------- play: lane = (plan, device), admission and timing together ----------------
    const int col = warp * 32 + lane;
    const int q = col / kL, g = col % kL;
    const int64_t p = q < ng ? plan_of(q) : 0;
    const bool live = q < ng && out.status[p] == 0;
    const auto slots_of = [&](int plan) {
        SlotArr<TT, ST, kP> a;
        if constexpr (SlotBytes<ST>::kHi) {
            a.lo = (uint32_t *)(sm + L.slots) + plan;
            a.hi = sm + L.slots_hi + plan;
        } else {
            a.v = (TT *)(sm + L.slots) + plan;
        }
        return a;
    };
    const auto slots = slots_of(q);
    Running<TT, kB> run_slots;  // [slot][plan, device] when in shared memory (lanes g >= D own none)
    run_slots.init(g < D ? B : 0, (TT *)(sm + L.se) + q * D + g, (uint32_t *)(sm + L.sk) + q * D + g, kP * D);
    for (int32_t k = g; k < dp.nslots + 2; k += kL) slots.set(k, 0);
    __syncthreads();
    const uint32_t trash = (uint32_t)dp.nslots;
    uint32_t capd = g < D ? (uint32_t)cap[g] : 0u;
    Q queue = 0;                    // resident models, least recently used first
    uint32_t n = 0, used = 0;       // their count and weights
    uint32_t cur = 0xFFFFFFFFu;     // model of the current replica
    int dev = g;                    // the device whose state this is (of g and g + kL)
    OtherDevice<Q, TT, kB> other;   // the other one's
    if constexpr (kDev == 2) {
        other.slots.init(g + kL < D ? B : 0, (TT *)(sm + L.se) + q * D + g + kL, (uint32_t *)(sm + L.sk) + q * D + g + kL, kP * D);
        other.cap = g + kL < D ? (uint32_t)cap[g + kL] : 0u;
    }
    TT ladm = 0, end = 0;           // last admission; latest finish of the lane's units
    int64_t gsum = 0;               // closed occupancy minus the open interval's start
    uint32_t ovf = 0;
    for (int32_t c = 0; c < chunks; ++c) {
        const int b = c % kBqBuffers;
        named_sync(kBqFull + b, kThreads);
        const uint2 *rb = ring + b * 3 * kChunk * kPitch + q;
        const int32_t kmax = min(kChunk, N - c * kChunk);
        // The flag words of the next position are read while this one plays.
        uint2 w1 = rb[(1 * kChunk) * kPitch];
        for (int32_t k = 0; k < kmax; ++k) {
            const uint2 nw1 = rb[(1 * kChunk + (k + 1 < kmax ? k + 1 : k)) * kPitch];
            const uint32_t r3 = w1.y;
            if (!(r3 & kSkip) && (int)((r3 & 31u) % (kDev == 1 ? 32 : kL)) == g) {
                if constexpr (kDev == 2) {  // (by selects: lanes that exchange play together with those that do not)
                    const bool c = (int)(r3 & 31u) != dev;
                    exchange_if(c, queue, other.queue);
                    exchange_if(c, n, other.n);
                    exchange_if(c, used, other.used);
                    exchange_if(c, cur, other.cur);
                    exchange_if(c, capd, other.cap);
                    exchange_if(c, ladm, other.ladm);
                    run_slots.swap_if(c, other.slots);
                    dev = (int)(r3 & 31u);
                }
                const uint2 w0 = rb[(0 * kChunk + k) * kPitch], w2 = rb[(2 * kChunk + k) * kPitch];
                const uint32_t m = (r3 >> 5) & 15u, kv = w1.x;
                const TT arr = w0.y, run = w0.x;  // run includes the grant
                const uint32_t r4 = w2.x, r5 = w2.y;
                // Release (Eq. 2, Eq. 7); an accumulator slot is reset by its reader.
                const uint32_t rs = r5 >> 16;
                const TT rel = max(arr, slots.get(rs & 0x7FFFu));
                slots.set((rs & 0x8000u) ? (rs & 0x7FFFu) : trash, 0);
                // The slot that frees first, and when the device drains.
                TT first = ~(TT)0, drain = 0;
                int slot = 0;
                run_slots.each(B, [&](int j, TT e, uint32_t) {
                    if (e < first) { first = e; slot = j; }
                    drain = max(drain, e);
                });
                const uint32_t wm = (uint32_t)weight[m];
                const bool join = m == cur;  // (the current replica's model is resident)
                const bool was_empty = n == 0;
                const int32_t kq = Lru<Q>::find(queue, n, m);
                const bool hit = kq < (int32_t)n;
                queue = hit ? Lru<Q>::remove(queue, hit ? kq : 0) : queue;
                n -= hit ? 1u : 0u;
                // Join: no earlier than the last admission (dispatch order),
                // and Eq. 11 with the running units' KV; idle models go first
                // (the head of the queue), then the admission waits for the
                // next running unit to end.  Another model: the device
                // drains, then the unit hits or loads.  Every sum of memory
                // stays below 2^32: resident weights and the running units'
                // KV fit the capacity, and so does a unit's own need alone.
                TT adm = join ? max(max(rel, first), ladm) : drain;
                const uint32_t need = hit ? kv : wm + kv;
                for (;;) {
                    uint32_t want = need;
                    if (join)
                        run_slots.each(B, [&](int, TT e, uint32_t v) { want += e > adm ? v : 0u; });
                    while (used + want > capd && n > 0) {
                        used -= (uint32_t)weight[(uint32_t)queue & 15u];
                        queue >>= 4;
                        n -= 1;
                    }
                    if (used + want <= capd) break;
                    TT next = ~(TT)0;  // the next running unit to end
                    if (join) run_slots.each(B, [&](int, TT e, uint32_t) { next = e > adm ? min(next, e) : next; });
                    if (next == ~(TT)0) {  // unreachable for a valid plan whose times fit
                        if (kNarrow) ovf = 1;
                        else atomicExch(dp.err, 2);
                        break;
                    }
                    adm = next;
                }
                TT start = adm;
                if (!join) {
                    const TT ls = max(drain, (!hit && (r3 & kPrefetch)) ? arr : rel);
                    const TT le = ls + (hit ? 0u : (uint32_t)load[m * D + dev]);
                    if (kNarrow) ovf |= le < ls;
                    start = max(le, rel);
                    adm = ls;
                    if (!hit) {
                        used += wm;
                        if (was_empty) gsum -= (int64_t)ls;
                    }
                    run_slots.reset(B, hit ? drain : le);
                    slot = 0;
                    cur = m;
                }
                queue |= (Q)m << (4 * n);  // the unit's model is now the most recently used
                n += 1;
                const TT cfin = start + run;
                // u32 times: a sum carried out (a saturated run makes the
                // finish carry, or 2^32 - 1).  u64: a saturated chain run.
                ovf |= kNarrow ? (uint32_t)(cfin < start) : (uint32_t)(w0.x == kRunCap);
                publish<TT>(slots, r3 >> 16, cfin);  // the sink when the unit writes nothing
                publish<TT>(slots, r4 & 0xFFFFu, cfin);
                const uint32_t nwl = (r3 >> 11) & 7u;
                if (r3 & kMany) {
                    publish<TT>(slots, r4 >> 16, cfin);
                    if (nwl == kWrites4) {
                        publish<TT>(slots, r5 & 0xFFFFu, cfin);
                    } else if (nwl > kWrites4) {  // five or more codes: the list from global memory
                        const int4 wr = __ldg(dp.noderec + 2 * (int32_t)(r5 & 0xFFFFu) + 1);
                        for (int32_t e = 3; e < wr.y; ++e) publish<TT>(slots, __ldg(dp.wl + wr.x + e), cfin);
                    }
                }
                run_slots.put(slot, cfin, kv);
                ladm = adm;
                end = max(end, cfin);
                if (r3 & kDrop) {  // retain bit 0 (B_q = 1 only): the model leaves after the unit
                    queue &= ~((Q)0xF << (4 * (n - 1)));
                    n -= 1;
                    used -= wm;
                    cur = 0xFFFFFFFFu;
                    if (n == 0) gsum += (int64_t)cfin;
                }
            }
            __syncwarp();  // the next unit's lane sees this one's slots
            w1 = nw1;
        }
        named_arrive(kBqEmpty + b, kThreads);  // buffer b may be refilled
    }
    // The plan's results from its lanes.
    int64_t g_all = gsum;
    uint32_t n_open = (n != 0) + (kDev == 2 && other.n != 0), o_all = ovf;
    if (kNarrow) o_all |= end == (TT)kRunCap;
#pragma unroll
    for (int o = kL / 2; o; o >>= 1) {
        end = max(end, __shfl_xor_sync(0xFFFFFFFFu, end, o));
        g_all += __shfl_xor_sync(0xFFFFFFFFu, g_all, o);
        n_open += __shfl_xor_sync(0xFFFFFFFFu, n_open, o);
        o_all |= __shfl_xor_sync(0xFFFFFFFFu, o_all, o);
    }
    const uint32_t bad = live ? open[q] >> kOpenBad : 0u;  // placement bits found by the producers
    const bool done = live && !bad && !o_all;
    if (done)
        for (int32_t w = g; w < W; w += kL) slots.set(w, slots.get(w) - arrival[w]);  // session completion latency
    if (g == 0) {
        if (bad) {
            out.status[p] = bad;
            out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
        } else if (live && o_all) {
            ovf_list[atomicAdd(ovf_count, 1)] = (int32_t)p;
        } else if (live) {
            out.makespan_us[p] = (int64_t)end - dp.first_arrival;
            out.gpu_us[p] = g_all + (int64_t)n_open * (int64_t)end;
        }
    }
    __syncwarp();  // every lane reads the latencies that a plan's lanes wrote
    // The p95 (Section 4.2, nearest rank) of the warp's plans, one after the other.
    const int32_t rank = (int32_t)((95 * (int64_t)W + 99) / 100 - 1);
    for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, done && g == 0); todo; todo &= todo - 1) {
        const int plan = (warp * 32 + __ffs((int)todo) - 1) / kL;
        const uint64_t v = warp_select(slots_of(plan), W, rank);
        if (lane == 0) out.p95_us[plan_of(plan)] = (int64_t)v;
    }
    }
    __syncthreads();  // the group's shared state is free for the next group
  }
}

size_t bytes32(const wf_dev_problem &dp)
{
    return bq_layout<uint32_t, uint32_t>(dp.D, dp.M, dp.W, dp.batch, dp.nslots + 2).total;
}

size_t bytes64(const wf_dev_problem &dp)
{
    const int32_t NS = dp.nslots + 2;
    return below40(dp) ? bq_layout<uint64_t, Split40>(dp.D, dp.M, dp.W, dp.batch, NS).total
                       : bq_layout<uint64_t, uint64_t>(dp.D, dp.M, dp.W, dp.batch, NS).total;
}

// Launches the instantiation for this problem over the batch, or over the
// listed plans (of unknown number: at most `most` CTAs).
template <typename TT, typename ST, int kB>
int launch_bq(const wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, size_t smem, const int32_t *in_list,
              const int32_t *in_count, int32_t *list, int32_t *count, cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    int64_t blocks = (pl->P + kBqPlans - 1) / kBqPlans;
    if (in_list) blocks = std::min<int64_t>(blocks, (int64_t)ctx->sms * 6);
    auto go = [&](auto q, auto l, auto n) {
        constexpr int kL = decltype(l)::value, kDev = decltype(n)::value;
        const auto k = bq_kernel<typename decltype(q)::type, kL, kDev, TT, ST, kB>;
        int rc = wf_cuda_check(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                               "batch sweep smem attribute");
        // The whole of the SM's memory as shared memory: by default four
        // CTAs were resident where six fit.
        if (!rc) rc = wf_cuda_check(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                         cudaSharedmemCarveoutMaxShared), "batch sweep carve-out");
        if (rc) return rc;
        k<<<(unsigned)blocks, 32 * BqShape<kL, kDev, kB>::kWarps, smem, st>>>(dp, *pl, *out, in_list, in_count, list, count);
        return wf_cuda_check(cudaGetLastError(), "batch sweep launch");
    };
    auto by_q = [&](auto l, auto n) { return dp.M <= 8 ? go(Ty<uint32_t>{}, l, n) : go(Ty<uint64_t>{}, l, n); };
    return dp.D <= 8 ? by_q(Iv<8>{}, Iv<1>{}) : dp.D <= 16 ? by_q(Iv<16>{}, Iv<1>{}) : by_q(Iv<16>{}, Iv<2>{});
}

int launch_bq64(const wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, size_t smem, const int32_t *in_list,
                const int32_t *in_count, int32_t *list, int32_t *count, cudaStream_t st)
{
    return below40(ctx->dp)
               ? launch_bq<uint64_t, Split40, 0>(ctx, pl, out, smem, in_list, in_count, list, count, st)
               : launch_bq<uint64_t, uint64_t, 0>(ctx, pl, out, smem, in_list, in_count, list, count, st);
}

}  // namespace

// Whether the replica-batch sweep can run this problem (the same slot and
// size limits as the sweep, plus room for every device's B_q slots); else
// the caller uses the int64 path.  Both time widths or neither: the u64 one
// needs more shared memory.
wf_batch_cfg wf_batch_config(const wf_dev_problem &dp)
{
    wf_batch_cfg c = {};
    if (dp.batch < 1 || dp.S != 0 || dp.nslots <= 0 || dp.nslots > 32765 || dp.max_arrival >= (int64_t)1 << 32 ||
        dp.M > 16 || dp.N > 65534 || dp.phi_life || dp.reclaim)
        return c;
    const size_t s64 = bytes64(dp);
    if (s64 > 227 * 1024) return c;
    c.smem32 = bytes32(dp);
    c.smem64 = s64;
    return c;
}

// Status pass (placement left to the producers), then the replica-batch
// sweep on u32 times and its hand-offs on u64 times, or (wide_first) every
// plan on u64 times; plans with a saturated chain run are left for the int64
// path.
int wf_launch_batch(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, const wf_batch_cfg &cfg, bool wide_first,
                    int32_t *counts, int32_t *list1, int32_t *list2, cudaStream_t st, const int32_t **rest_list,
                    const int32_t **rest_count)
{
    int rc = wf_launch_status(ctx, pl, out, st, false);
    if (!rc && !wide_first) {
        rc = ctx->dp.batch <= kBqRegs
                 ? launch_bq<uint32_t, uint32_t, kBqRegs>(ctx, pl, out, cfg.smem32, nullptr, nullptr, list1, counts, st)
                 : launch_bq<uint32_t, uint32_t, 0>(ctx, pl, out, cfg.smem32, nullptr, nullptr, list1, counts, st);
        if (!rc) rc = launch_bq64(ctx, pl, out, cfg.smem64, list1, counts, list2, counts + 1, st);
    } else if (!rc) {
        rc = launch_bq64(ctx, pl, out, cfg.smem64, nullptr, nullptr, list2, counts + 1, st);
    }
    *rest_list = list2;
    *rest_count = counts + 1;
    return rc;
}

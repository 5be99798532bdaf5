// Plan evaluation in shared memory.
//
// Deterministic plans (pc_kernel): a CTA plays 16 plans as a three-stage warp
// pipeline over 16 dispatch positions at a time.  Producer warps turn each
// (plan, position) into a unit record (Eq. 3-4 chain, write list, release
// slot); two residency warps settle LRU model residency under capacity
// (Eq. 11) with four lanes per plan, each playing its own devices' units;
// one timing warp plays releases, loads, starts and finishes (Eq. 2, 5, 7,
// 10) with lane = plan.  Records pass through a ring of four buffers guarded
// by named barriers.  Per-plan state lives in shared memory:
//   - finish-time slots (u32 microseconds) assigned statically from the DAG
//     (wf_slots.cpp) instead of one word per activation, [slot][plan];
//   - per device: free time [device][plan]; resident weights, count and LRU
//     queue [device][plan].
// Status bits (Eq. 8-10) come first from status_kernel, a warp per plan.
//
// Times: the deterministic sweep first plays u32 times and lists a plan whose
// times reach 2^32 us; a second instantiation with u64 times plays the listed
// plans, with 16, 6 or 3 plans per CTA by occupancy and finish slots of 40
// bits (a u32 word and a byte) while no time can reach 2^40 us.  Once a
// context has seen most plans leave 32 bits, a third instantiation (Rel32)
// plays the whole batch on u32 times counted from a per-plan base that rises
// with the plan's devices' free times, and lists for the u64 sweep only what
// leaves 32 bits even so.  Only a unit whose summed run time saturates 32
// bits goes on to the exact int64 path in wf_eval.cu.
//
// A compile-time variant (kPhi) also returns the window terms of Eq. 12's
// ranking key: residency marks a reload (a model its device held before) in
// bit 31 of the record's load word, and timing counts the timely prefetches
// and sums each unit's load delay plus its reload time.
#include <algorithm>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "wf_play.cuh"

namespace {

// CTA shape, a three-stage pipeline over kChunk dispatch positions at a time:
// the last kProducers warps prepare the unit records of kP plans (lane =
// position) into a ring of kBuffers buffers; warps 1..kRes settle model
// residency (lane = plan and device group: hits, reclamations, occupancy
// changes); warp 0 plays the timing (lane = plan: releases, starts,
// finishes, slots).  With u32 times and 16 plans per CTA, four CTAs share an
// SM at 2,000 activations; the u64 variant holds fewer plans per CTA when its
// slots need the room.
constexpr int kPlans32 = 16;                // plans per CTA of the u32 sweep
// Record buffers of the ring: four, or three under reclamation by next use,
// whose state per model would otherwise cost a CTA per SM at 2,000
// activations.  Named barriers: kFullP + b (producers -> residency), kFullR +
// b (residency -> timing), kEmpty + b (timing -> producers) for buffer b;
// kOpen (residency -> timing, once at the end).
//
// kReclaim, the reclamation order and who settles it: least recently used
// (kLru), by next use with a lane per model (kNuModel), or by next use with a
// lane per plan (kNuPlan, short windows in large batches).
enum { kLru = 0, kNuModel = 1, kNuPlan = 2 };
template <int kReclaim>
struct Ring {
    static constexpr int kBuffers = kReclaim == kNuModel ? 3 : 4;
    static constexpr int kFullP = 1, kFullR = kFullP + kBuffers, kEmpty = kFullR + kBuffers, kOpen = kEmpty + kBuffers;
    static_assert(kOpen < 16, "named barriers");
};

// The ring holds a record as word pairs (8-byte shared-memory accesses):
// (w0, w2) for timing, (w1, w3) read and rewritten by residency, (w4, w5)
// for timing; under reclamation by next use the unit's next use is beside it
// (u16: as a fourth pair it cost a CTA per SM at 2,000 activations).
constexpr int kPairs = 3;

// Lanes per plan of the residency stage under reclamation by next use: kPer
// models a lane, of the 4, 8 or 16 that a sweep is compiled for (Q: a word of
// as many 4-bit model ids).
template <typename Q>
constexpr int kPer = sizeof(Q) <= 4 ? 1 : 2;
template <typename Q>
constexpr int kModelLanes = 2 * (int)sizeof(Q) / kPer<Q>;

template <int kP, int kReclaim = 0, typename Q = uint32_t>
struct PcShape {
    static constexpr int kProducers = kP >= 32 ? 8 : kP >= 16 ? 4 : kP >= 6 ? 3 : 2;
    static constexpr int kRes = kReclaim == kNuModel ? (kP * kModelLanes<Q> + 31) / 32 : kReclaim == kNuPlan ? 2 : kP >= 32 ? 4 : kP >= 16 ? 2 : 1;  // residency warps
    static constexpr int kWarps = 1 + kRes + kProducers;
    // Four 16-plan CTAs share an SM (shared memory allows it at 2,000
    // activations), or four 6-plan CTAs at 8,192, which bounds the registers
    // per thread (large window with three of the latter, at 106 registers:
    // 56.0 ms, with four 47.4).
    static constexpr int kMinBlocks = kP >= 32 ? 2 : kP < 6 ? 1 : kP < 16 ? 4 : kReclaim == kNuModel && sizeof(Q) == 8 ? 3 : kReclaim == kNuPlan ? 4 : 4;
    // Elements (8-byte word pairs) per (pair, position) row of the ring.  A
    // producer store covers 16 positions x 2 plans in two halves of 16
    // lanes; an odd pitch puts each half's 16 pairs on 32 distinct banks, and
    // the consumers' plan-major loads are contiguous.
    static constexpr int kPitch = kP | 1;
    static_assert(kChunk == 16 && kP >= 1 && kP <= 32, "ring pitch assumes 16 positions per chunk");
};

// Residency lanes per plan under least-recently-used reclamation: a device
// group each (d = g mod kG), with a state per [device][plan].  Under
// reclamation by next use the lanes are a plan's models, every device is
// played by all of them (one group), and the state is [device][lane].
template <int kP, int kReclaim, typename Q>
struct PcGroups {
    using S = PcShape<kP, kReclaim, Q>;
    static constexpr int kG = kReclaim ? 1 : (32 * S::kRes) / kP;
    static constexpr int kRow = kReclaim == kNuModel ? 32 * S::kRes : kP;  // row length of the state
    static_assert(kG >= 1 && kG * kP <= 32 * S::kRes, "residency lanes");
};

// Relative 32-bit times (slot storage Rel32, with TT = uint32_t): every time
// the timing stage keeps (finish slots, device free times, the plan's end)
// counts from a per-plan base B, which it raises now and then to one below
// the smallest device free time.  That is exact: every later unit starts at
// or after its device's free time, so a stored finish or arrival below B can
// be read as B without changing any start (Eq. 2, 5, 7).  A session slot
// that would fall below B keeps its exact value in global memory instead,
// for the p95.
struct Rel32 {};
template <typename ST>
struct IsRel {
    static constexpr bool value = false;
};
template <>
struct IsRel<Rel32> {
    static constexpr bool value = true;
};
template <>
struct SlotBytes<Rel32> {
    static constexpr uint32_t kLo = 4, kHi = 0;
};

constexpr uint32_t kRebaseAt = 3u << 30;   // a plan's end above this raises its base ...
constexpr uint32_t kRebaseMin = 1u << 28;  // ... by at least this much, else not at all

// Up to this many sessions the timing lane selects its plan's p95 itself;
// beyond, a warp per plan does after the sweep (warp_select).
constexpr int32_t kLaneSelect = 32;

// Slots 2i and 2i + 1 of a 32-bit slot array read as one 64-bit value i (the
// relative sweep's session latencies at the end of a plan).
template <int kS>
struct PairArr {
    uint32_t *v;
    __device__ __forceinline__ uint64_t get(uint32_t i) const
    {
        return ((uint64_t)v[(2 * i + 1) * kS] << 32) | v[2 * i * kS];
    }
    __device__ __forceinline__ void set(uint32_t i, uint64_t x) const
    {
        v[2 * i * kS] = (uint32_t)x;
        v[(2 * i + 1) * kS] = (uint32_t)(x >> 32);
    }
};

struct PcLayout {
    uint32_t weight, load, rcost, wsum, arr, ring, next, slots, slots_hi, tfree, free, queue, open, flag, gmask, everl, nres, nuse, rcnt, total;
};

// Shared memory of a CTA of kP plans with TT times and NS slots per plan;
// with reclamation by next use (kReclaim) the next uses lie beside the ring
// and each plan keeps per (device, model) the next use and the last use
// of the resident copy, and per device the free capacity; with the window
// terms of Eq. 12 (kPhi) each plan keeps per device the models it ever
// held (by next use: in a register, per model the devices).
template <int kP, typename TT, typename Q, int kReclaim = 0, bool kPhi = false, typename ST = TT>
__host__ __device__ inline PcLayout pc_layout_q(int32_t D, int32_t M, int32_t W, int32_t NS)
{
    using G = PcGroups<kP, kReclaim, Q>;
    constexpr uint32_t t = sizeof(TT);
    PcLayout l;
    uint32_t o = 0;
    l.weight = o; o += 4u * 16;  // (zeros beyond M: read for the queue's empty places)
    l.load = o; o += round16(4u * M * D);
    l.rcost = o; o += kReclaim == kNuModel ? round16(4u * M * D) : 0u;
    l.wsum = o; o += kReclaim == kNuModel ? 256u * (uint32_t)sizeof(Q) : 0u;  // (the sums of each set of eight models; with Q of 16 bits more than the 16 used)
    l.arr = o; o += round16(4u * W);
    l.ring = o; o += round16(8u * Ring<kReclaim>::kBuffers * kPairs * kChunk * PcShape<kP>::kPitch);
    l.next = o; o += kReclaim ? round16(2u * Ring<kReclaim>::kBuffers * kChunk * PcShape<kP>::kPitch) : 0u;
    l.slots = o; o += round16(SlotBytes<ST>::kLo * (uint32_t)NS * kP);
    l.slots_hi = o; o += round16(SlotBytes<ST>::kHi * (uint32_t)NS * kP);
    l.tfree = o; o += round16(t * D * kP);
    const uint32_t rs = (uint32_t)(D * G::kRow);
    // Residency state: a word per device (DevState), or under reclamation by
    // next use a word per (device, model), and the free capacity apart.
    using State = std::conditional_t<kReclaim == kNuModel, uint32_t[kPer<Q>], std::conditional_t<kReclaim == kNuPlan, Q, DevState<Q>>>;
    l.queue = o; o += round16((uint32_t)sizeof(State) * rs);
    l.free = o; o += kReclaim ? round16(4u * D * kP) : 0u;
    l.open = o;
    l.flag = o + 4u * kP; o += round16(4u * kP + 4u);
    l.gmask = o; o += kReclaim == kNuModel ? 0u : round16(2u * Ring<kReclaim>::kBuffers * G::kG * kP);
    l.everl = o; o += kPhi && kReclaim != kNuModel ? round16(2u * rs) : 0u;
    l.nres = o; o += kReclaim == kNuPlan ? round16(rs) : 0u;
    l.nuse = o; o += kReclaim == kNuPlan ? round16(2u * M * rs) : 0u;
    l.rcnt = o; o += kReclaim == kNuPlan ? round16((uint32_t)M * kP) : 0u;
    l.total = o;
    return l;
}

template <int kP, typename TT, int kReclaim = 0, bool kPhi = false, typename ST = TT>
inline PcLayout pc_layout(int32_t D, int32_t M, int32_t W, int32_t NS)
{
    if constexpr (kReclaim == kNuModel)
        if (M <= 4) return pc_layout_q<kP, TT, uint16_t, kReclaim, kPhi, ST>(D, M, W, NS);
    return M <= 8 ? pc_layout_q<kP, TT, uint32_t, kReclaim, kPhi, ST>(D, M, W, NS)
                  : pc_layout_q<kP, TT, uint64_t, kReclaim, kPhi, ST>(D, M, W, NS);
}


// The r-th smallest (0-based) of slots 0 .. n-1 of a slot array (one thread).
template <typename TT, typename SA>
__device__ TT select_slots(const SA &v, int32_t n, int32_t r)
{
    int32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        const TT pivot = v.get(lo + (hi - lo) / 2);
        int32_t i = lo, j = hi;
        while (i <= j) {
            while (v.get(i) < pivot) ++i;
            while (v.get(j) > pivot) --j;
            if (i <= j) { const TT t = v.get(i); v.set(i, v.get(j)); v.set(j, t); ++i; --j; }
        }
        if (r <= j) hi = j;
        else if (r >= i) lo = i;
        else return v.get(r);
    }
    return v.get(r);
}

// The sweep of groups of kP plans: every plan of the batch (in_list NULL, plan
// = group * kP + q) or the listed ones (plan = in_list[group * kP + q] below
// *in_count).  CTA b plays groups b, b + gridDim.x, ...  TT = uint32_t: a plan whose times leave 32 bits is appended to
// ovf_list; once every plan of a CTA has, its stages run on without loads.
// TT = uint64_t: only a unit whose summed run time reaches 2^32 - 1 sends its
// plan to ovf_list.
template <typename Q, typename TT, int kP, int kReclaim, bool kPhi, typename ST>
__global__ void __launch_bounds__(32 * PcShape<kP, kReclaim, Q>::kWarps, PcShape<kP, kReclaim, Q>::kMinBlocks)
pc_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, const int32_t *in_list, const int32_t *in_count,
          int32_t *ovf_list, int32_t *ovf_count)
{
    constexpr int kRW = kPairs;  // word pairs per record in the ring
    using S = PcShape<kP, kReclaim, Q>;
    constexpr int kPitch = S::kPitch;
    constexpr int kProdThreads = 32 * S::kProducers;
    constexpr int kResThreads = 32 * S::kRes;
    constexpr bool kNarrow = sizeof(TT) == 4;
    constexpr bool kRel = IsRel<ST>::value;  // relative 32-bit times
    static_assert(!kRel || (kNarrow && kReclaim == 0 && !kPhi), "relative times: u32, least recently used");
    constexpr int kG = PcGroups<kP, kReclaim, Q>::kG;  // residency lanes per plan (by next use: one mask for all of them)
    using RG = Ring<kReclaim>;
    constexpr int kBuffers = RG::kBuffers, kFullP = RG::kFullP, kFullR = RG::kFullR, kEmpty = RG::kEmpty,
                  kOpen = RG::kOpen;
    extern __shared__ __align__(128) uint8_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W;
    const int32_t rank = (int32_t)((95 * (int64_t)W + 99) / 100 - 1);  // the p95's nearest rank (Section 4.2)
    const PcLayout L = pc_layout_q<kP, TT, Q, kReclaim, kPhi, ST>(D, M, W, dp.nslots + 2);
    const int64_t total = in_list ? (int64_t)*in_count : pl.P;
    if ((int64_t)blockIdx.x * kP >= total) return;  // the whole CTA: no plan
    uint2 *ring = (uint2 *)(sm + L.ring);
    uint16_t *next = (uint16_t *)(sm + L.next);  // [buffer][position][plan] (by next use)
    const int32_t chunks = (N + kChunk - 1) / kChunk;
    volatile uint32_t *gave_up = (volatile uint32_t *)(sm + L.flag);

    int32_t *weight = (int32_t *)(sm + L.weight);
    int32_t *load = (int32_t *)(sm + L.load);
    uint32_t *arrival = (uint32_t *)(sm + L.arr);
    uint32_t *open = (uint32_t *)(sm + L.open);
    uint16_t *gmask = (uint16_t *)(sm + L.gmask);  // [buffer][device group][plan]
    if (threadIdx.x < 16) weight[threadIdx.x] = (int)threadIdx.x < M ? __ldg(dp.weight + threadIdx.x) : 0;
    for (int32_t k = threadIdx.x; k < M * D; k += blockDim.x) load[k] = __ldg(dp.load + k);
    if (kReclaim == kNuModel) {
        for (uint32_t k = threadIdx.x; k < 64u * sizeof(Q); k += blockDim.x) {
            uint32_t w = 0;
            for (int32_t m = 0; m < 8; ++m)
                if ((k >> m) & 1u) w += 8 * (int32_t)(k >> 8) + m < M ? (uint32_t)__ldg(dp.weight + 8 * (k >> 8) + m) : 0u;
            ((uint32_t *)(sm + L.wsum))[k] = w;
        }
        for (int32_t k = threadIdx.x; k < M * D; k += blockDim.x)
            ((float *)(sm + L.rcost))[k] = 1.0f / (float)max(__ldg(dp.load + k), 1);
    }
    for (int32_t k = threadIdx.x; k < W; k += blockDim.x) arrival[k] = (uint32_t)__ldg(dp.arrival + k);
    // (each role's first __syncthreads below publishes these tables)

  for (int64_t j0 = (int64_t)blockIdx.x * kP; j0 < total; j0 += (int64_t)gridDim.x * kP) {
    const int ng = (int)(total - j0 < kP ? total - j0 : kP);
    if (threadIdx.x == 0) *gave_up = 0;
    if (threadIdx.x < kP) open[threadIdx.x] = 0;

    if (warp > S::kRes) {
        // ---------------- producers: lane = dispatch position ----------------
        __syncthreads();
        const int pw = warp - 1 - S::kRes;
        const int pos = lane % kChunk, sub = lane / kChunk;
        // The plans this lane serves, fixed for the whole sweep: row pointers
        // and whether the plan is live, resolved once.
        constexpr int kStep = S::kProducers * kPlansPerIter;
        constexpr int kIters = (kP + kStep - 1) / kStep;
        RowPtrs rp[kIters];
        bool okq[kIters];
        int qq[kIters];
        int64_t qplan[kIters];
#pragma unroll
        for (int j = 0; j < kIters; ++j) {
            const int q = pw * kPlansPerIter + j * kStep + sub;
            qq[j] = q < kP ? q : -1;
            okq[j] = q < kP && q < ng;
            qplan[j] = 0;
            rp[j].place = nullptr;
            rp[j].order = nullptr;
            rp[j].boff = 0;
            if (okq[j]) {
                const int64_t pq = in_list ? (int64_t)__ldg(in_list + j0 + q) : j0 + q;
                qplan[j] = pq;
                okq[j] = __ldg(out.status + pq) == 0;
                rp[j].place = pl.place + pq * pl.place_stride;
                rp[j].order = (const uint16_t *)((const uint8_t *)pl.order + pq * pl.order_stride);
                rp[j].boff = pq * pl.bits_stride;
            }
        }
        // The node-indexed rows (placement, fusion and prefetch bits) are
        // gathered all through the sweep; one bulk L2 prefetch per row up
        // front streams them in rather than sector by sector.  (Rows are
        // 16-byte aligned, and their 16-byte-rounded sizes fit the strides.)
        const uint32_t place_bytes = (uint32_t)((N + 15) & ~15), bits_bytes = (uint32_t)((((N + 31) >> 5) * 4 + 15) & ~15);
#pragma unroll
        for (int j = 0; j < kIters; ++j)
            if (pos == 0 && okq[j]) {
                l2_prefetch(rp[j].place, place_bytes);
                l2_prefetch(bits_row(pl.fuse, rp[j].boff), bits_bytes);
                l2_prefetch(bits_row(pl.prefetch, rp[j].boff), bits_bytes);
            }
        // Dispatch entries are read one chunk ahead of their use.
        int32_t h0[kIters];
#pragma unroll
        for (int j = 0; j < kIters; ++j) h0[j] = okq[j] && pos < N ? __ldg(rp[j].order + pos) : 0;
        // The timing stage's give-up flag, read a chunk before it is used so
        // that no load of this chunk waits for it.
        bool quit = false;
        for (int32_t c = 0; c < chunks; ++c) {
            const int b = c % kBuffers;
            if (c >= kBuffers) named_sync(kEmpty + b, kProdThreads + 32);  // timing released buffer b
            uint2 *rb = ring + b * kRW * kChunk * kPitch;
            const int32_t i = c * kChunk + pos;
            int32_t h1[kIters];
            bool act[kIters];
#pragma unroll
            for (int j = 0; j < kIters; ++j) {
                h1[j] = okq[j] && i + kChunk < N && !quit ? __ldg(rp[j].order + i + kChunk) : 0;
                act[j] = okq[j] && i < N && !quit;
                if (kReclaim && qq[j] >= 0)  // the next use of this unit's model on its device
                    next[(b * kChunk + pos) * kPitch + qq[j]] = act[j] ? __ldg(dp.nextuse + qplan[j] * (int64_t)N + i) : (uint16_t)0xFFFFu;
            }
            uint32_t dev[kIters];
            produce_batch<kIters, kPitch>(dp, pl, rp, act, h0, rb, pos, qq, dev, open);
            // For each residency lane, the chunk's units on its devices: one
            // ballot per device group; each half-warp holds one plan.
#pragma unroll
            for (int j = 0; j < kIters && kReclaim != kNuModel; ++j) {
                const uint32_t key = dev[j] == 0xFFFFFFFFu ? (uint32_t)kG : dev[j] % kG;
#pragma unroll
                for (int gg = 0; gg < kG; ++gg) {
                    const uint32_t bal = __ballot_sync(0xFFFFFFFFu, key == (uint32_t)gg);
                    if (pos == gg && qq[j] >= 0) gmask[(b * kG + gg) * kP + qq[j]] = (uint16_t)(bal >> (kChunk * sub));
                }
            }
#pragma unroll
            for (int j = 0; j < kIters; ++j) h0[j] = h1[j];
            quit = kNarrow && *gave_up;
            named_arrive(kFullP + b, kProdThreads + kResThreads);  // buffer b is full
        }
        // Match the timing stage's releases of the last buffers.
        for (int32_t c = chunks; c < chunks + kBuffers; ++c)
            if (c >= kBuffers) named_sync(kEmpty + c % kBuffers, kProdThreads + 32);
    } else if (warp >= 1) {
        // ---------------- residency (Eq. 11, Section 3.5) ----------------
        const int rl = (warp - 1) * 32 + lane;
        constexpr int kRow = PcGroups<kP, kReclaim, Q>::kRow;
        if constexpr (kReclaim == kLru) {
        // Lane (plan, device group): kG lanes per plan, and lane g plays the
        // plan's units on the devices d = g (mod kG) in dispatch order:
        // under least-recently-used reclamation devices do not interact.  The
        // producers leave each lane's units of the chunk as a mask (gmask).
        // (plans side by side: the lanes' states lie in banks of their own)
        const int qp = rl % kP, g = rl / kP;
        const bool rmine = g < kG;
        const int64_t p = (rmine && qp < ng) ? (in_list ? (int64_t)in_list[j0 + qp] : j0 + qp) : 0;
        const bool live = rmine && qp < ng && out.status[p] == 0;
        DevState<Q> *state = (DevState<Q> *)(sm + L.queue) + qp;  // [device][plan]
        uint16_t *everl = (uint16_t *)(sm + L.everl) + qp;        // [device][plan], bit m: m was held (kPhi)
        if (rmine)
            for (int32_t d = g; d < D; d += kG) {
                state[d * kRow].init((uint32_t)__ldg(dp.cap + d));
                if (kPhi) everl[d * kRow] = 0;
            }
        __syncthreads();
        for (int32_t c = 0; c < chunks; ++c) {
            const int b = c % kBuffers;
            named_sync(kFullP + b, kProdThreads + kResThreads);
            uint2 *rb = ring + b * kRW * kChunk * kPitch + qp;
            uint32_t todo = live ? gmask[(b * kG + g) * kP + qp] : 0u;
            // The ring words of the lane's next unit are read while this one
            // plays (pair 1: w1 | w3).
            int32_t k = todo ? __ffs((int)todo) - 1 : 0;
            uint2 v = todo ? rb[(1 * kChunk + k) * kPitch] : make_uint2(0u, 0u);
            while (todo) {
                todo &= todo - 1;
                const int32_t kn = todo ? __ffs((int)todo) - 1 : k;
                const uint2 nv = rb[(1 * kChunk + kn) * kPitch];
                const uint32_t r1 = v.x, r3 = v.y;
                const int32_t d = (int32_t)(r3 & 31u);
                DevState<Q> ds = state[d * kRow];
                bool missed;
                uint2 w = ds.settle(r1, r3, weight, load, D, dp.err, missed);
                if (kPhi && missed) {  // a reload of a model this device held before: bit 31 of the load word
                    const uint32_t m = (r3 >> 5) & 15u, e = everl[d * kRow];
                    w.x |= ((e >> m) & 1u) << 31;
                    everl[d * kRow] = (uint16_t)(e | (1u << m));
                }
                state[d * kRow] = ds;
                rb[(1 * kChunk + k) * kPitch] = w;
                k = kn;
                v = nv;
            }
            named_arrive(kFullR + b, kResThreads + 32);
        }
        if (live) {  // devices still occupied at the end
            uint32_t o = 0;
            for (int32_t d = g; d < D; d += kG) o += state[d * kRow].occupied();
            if (o) atomicAdd(open + qp, o);
        }
        } else if constexpr (kReclaim == kNuPlan) {
        // By next use with a lane per plan: the same rules as below, a victim at
        // a time, each found by a scan of the device's queue.  A longer chain
        // for one plan, but fewer instructions in all (lane_per_plan says where).
        constexpr int kEvery = 32 * S::kRes / kP;  // the lanes that play, spread over the residency warps
        const int qp = rl / kEvery;
        const bool rmine = rl % kEvery == 0;
        const int64_t p = (rmine && qp < ng) ? (in_list ? (int64_t)in_list[j0 + qp] : j0 + qp) : 0;
        const bool live = rmine && qp < ng && out.status[p] == 0;
        Q *queue = (Q *)(sm + L.queue) + qp;               // [device][plan]: resident models, least recently used first
        uint8_t *nres = sm + L.nres + qp;                  // [device][plan]: how many
        uint32_t *room = (uint32_t *)(sm + L.free) + qp;   // [device][plan]: free capacity
        uint16_t *nuse = (uint16_t *)(sm + L.nuse) + qp;   // [device][model][plan]: next use of the copy there
        uint8_t *copies = sm + L.rcnt + qp;                // [model][plan]: devices that hold it
        uint16_t *everl = (uint16_t *)(sm + L.everl) + qp; // [device][plan], bit m: m was held (kPhi)
        if (rmine) {
            for (int32_t d = 0; d < D; ++d) {
                queue[d * kP] = 0;
                nres[d * kP] = 0;
                room[d * kP] = (uint32_t)__ldg(dp.cap + d);
                if (kPhi) everl[d * kP] = 0;
            }
            for (int32_t m = 0; m < M; ++m) copies[m * kP] = 0;
        }
        __syncthreads();
        for (int32_t c = 0; c < chunks; ++c) {
            const int b = c % kBuffers;
            named_sync(kFullP + b, kProdThreads + kResThreads);
            uint2 *rb = ring + b * kRW * kChunk * kPitch + (rmine ? qp : 0);
            const uint16_t *nb = next + b * kChunk * kPitch + (rmine ? qp : 0);
            for (uint32_t todo = live ? gmask[b * kP + qp] : 0u; todo; todo &= todo - 1) {
                const int32_t k = __ffs((int)todo) - 1, here = c * kChunk + k;
                const uint2 v = rb[(1 * kChunk + k) * kPitch];
                const uint32_t r1 = v.x, r3 = v.y, m = (r3 >> 5) & 15u, wm = (uint32_t)weight[m];
                const int32_t d = (int32_t)(r3 & 31u);
                Q q = queue[d * kP];
                uint32_t n = nres[d * kP], f = room[d * kP];
                const bool was_empty = n == 0;
                const int32_t at = Lru<Q>::find(q, n, m);
                const bool hit = at < (int32_t)n;
                q = hit ? Lru<Q>::remove(q, hit ? at : 0) : q;
                n -= hit ? 1u : 0u;
                const uint32_t need = hit ? r1 : wm + r1;  // at most the capacity
                while (need > f && n > 0) {
                    // A copy also held elsewhere goes first, then an infinite
                    // quotient, then the larger one (exact products), then the
                    // earlier entry.
                    int32_t best = 0, bdist = 0, bcost = 0;
                    uint32_t bclass = 0;
#pragma unroll
                    for (int32_t e = 0; e < Lru<Q>::kSlots; ++e) {
                        if (e >= (int32_t)n) break;
                        const uint32_t x = (uint32_t)(q >> (4 * e)) & 15u;
                        const int32_t nu = nuse[(d * M + x) * kP], cost = load[x * D + d], dist = nu - here;
                        const bool inf = nu == 0xFFFF || cost == 0;
                        const uint32_t cls = (copies[x * kP] > 1 ? 2u : 0u) | (inf ? 1u : 0u);
                        if (e == 0 || cls > bclass || (cls == bclass && !inf && (int64_t)dist * bcost > (int64_t)bdist * cost)) {
                            best = e; bclass = cls; bdist = dist; bcost = cost;
                        }
                    }
                    const uint32_t x = (uint32_t)(q >> (4 * best)) & 15u;
                    f += (uint32_t)weight[x];
                    copies[x * kP] -= 1;
                    q = Lru<Q>::remove(q, best);
                    n -= 1;
                }
                if (need > f) atomicExch(dp.err, 2);  // unreachable for a valid plan
                uint2 w = settled(r3, hit, (uint32_t)load[m * D + d], was_empty, (r3 & kDrop) != 0 && n == 0);
                if (kPhi && !hit) {
                    const uint32_t e = everl[d * kP];
                    w.x |= ((e >> m) & 1u) << 31;
                    everl[d * kP] = (uint16_t)(e | (1u << m));
                }
                if (r3 & kDrop) {  // the model leaves when the unit ends
                    f += hit ? wm : 0u;
                    copies[m * kP] -= hit ? 1 : 0;
                } else {
                    f -= hit ? 0u : wm;
                    copies[m * kP] += hit ? 0 : 1;
                    nuse[(d * M + m) * kP] = nb[k * kPitch];
                    q |= (Q)m << (4 * n);
                    n += 1;
                }
                queue[d * kP] = q;
                nres[d * kP] = (uint8_t)n;
                room[d * kP] = f;
                rb[(1 * kChunk + k) * kPitch] = w;
            }
            named_arrive(kFullR + b, kResThreads + 32);
        }
        if (live) {  // devices still occupied at the end
            uint32_t o = 0;
            for (int32_t d = 0; d < D; ++d) o += nres[d * kP] != 0;
            if (o) atomicAdd(open + qp, o);
        }
        } else {
        // Reclamation by next use counts a model's copies over all devices, so
        // a plan's units are played one after another, by kL lanes that each
        // stand for a model, or beyond eight models for two (l and l + kL): a
        // lane keeps the number of each one's copies and, in shared memory, per device the copy's next use
        // and its last use (0: not resident).  Victims go one at a time: a copy
        // also resident elsewhere first, then the largest (next use -
        // position) / reload cost (no next use or a free reload: infinite),
        // then the least recently used.  None of that changes while one
        // admission evicts, so a lane ranks its copies among the others' at
        // once, by a float quotient, and a copy goes if those before it do
        // not make room enough; where the float cannot tell two quotients
        // apart (its error is below 2^-21) exact products decide.  The stage
        // is bound by issue (about 200 instructions a unit of four plans).  Nine
        // warps in four CTAs leave 56 registers a thread up to eight models, of
        // which the producers' and this loop spill 120 bytes; three producer warps
        // (64 registers) spill 240 and take 2,706, two 3,345, three CTAs 2,992.
        // 16,384 plans of N = 2,000, D = M = 8, us a step: a lane per plan, which
        // scanned the queue for each victim, 4,095; a lane per model 2,629; two
        // models a lane (270 instructions for eight plans, half the warps) 3,010;
        // a lane per model with a loop that takes one victim at a time 3,172.
        // Up to four models half the lanes would idle: four lanes a plan, two
        // residency warps.  56,387 plans of N = 376, D = 4, M = 2: a lane per plan
        // 963, eight lanes 1,171, four 897; 5,629 of N = 2,250, D = 2, M = 3: 760,
        // 912, 734.
        constexpr int kL = kModelLanes<Q>;
        constexpr int kI = kPer<Q>;
        constexpr uint32_t kAll = (1u << kL) - 1u;
        constexpr uint32_t kNear = 8;  // units in the last place: two quotients' errors are below 6
        const int qp = rl / kL, ml = rl % kL, shift = lane & ~(kL - 1);
        const bool rmine = qp < kP;
        const int64_t p = (rmine && qp < ng) ? (in_list ? (int64_t)in_list[j0 + qp] : j0 + qp) : 0;
        const bool live = rmine && qp < ng && out.status[p] == 0;
        uint32_t *tab = (uint32_t *)(sm + L.queue) + kI * rl;           // [device][lane][l, l + kL]: next use | last use + 1 << 16
        uint32_t *room = (uint32_t *)(sm + L.free) + (rmine ? qp : 0);  // [device][plan]: free capacity
        const float *rcost = (const float *)(sm + L.rcost);             // [model][device]: 1 / load time
        const uint32_t *wsum = (const uint32_t *)(sm + L.wsum);         // the weight of each set of eight models
        int mrow[kI];
#pragma unroll
        for (int i = 0; i < kI; ++i) mrow[i] = (ml + i * kL < M ? ml + i * kL : 0) * D;
        auto row_of = [&](uint32_t d, uint32_t (&x)[kI]) {
            if constexpr (kI == 2) {
                const uint2 u = *(const uint2 *)(tab + 2 * d * kRow);
                x[0] = u.x; x[1] = u.y;
            } else {
                x[0] = tab[d * kRow];
            }
        };
        auto set_row = [&](uint32_t d, const uint32_t (&x)[kI]) {
            if constexpr (kI == 2) *(uint2 *)(tab + 2 * d * kRow) = make_uint2(x[0], x[1]);
            else tab[d * kRow] = x[0];
        };
        const uint32_t none[kI] = {};
        for (int32_t d = 0; d < D; ++d) {
            set_row(d, none);
            if (rmine && ml == 0) room[d * kP] = (uint32_t)__ldg(dp.cap + d);
        }
        __syncthreads();
        uint32_t wx[kL][kI];  // the models' weights, of lane l ^ o
#pragma unroll
        for (int o = 0; o < kL; ++o)
#pragma unroll
            for (int i = 0; i < kI; ++i) wx[o][i] = (uint32_t)weight[(ml ^ o) + i * kL];
        uint32_t copies[kI] = {}, ever[kI] = {};  // of the lane's models; ever: the devices that held it (kPhi)
        for (int32_t c = 0; c < chunks; ++c) {
            const int b = c % kBuffers;
            named_sync(kFullP + b, kProdThreads + kResThreads);
            uint2 *rb = ring + b * kRW * kChunk * kPitch + (rmine ? qp : 0);
            const uint16_t *nb = next + b * kChunk * kPitch + (rmine ? qp : 0);
            const int32_t kmax = min(kChunk, N - c * kChunk);
            uint2 v = rb[1 * kChunk * kPitch];
            uint32_t nu = nb[0];
#pragma unroll 1
            for (int32_t k = 0; k < kmax; ++k) {
                const int32_t kn = min(k + 1, kChunk - 1);
                const uint2 nv = rb[(1 * kChunk + kn) * kPitch];
                const uint32_t nnu = nb[kn * kPitch];
                const bool act = live && !(v.y & kSkip);
                const uint32_t r1 = v.x, r3 = act ? v.y : 0u, m = (r3 >> 5) & 15u, d = r3 & 31u;
                uint32_t x[kI];
                row_of(d, x);
                uint32_t f = room[d * kP];
                const uint32_t wm = (uint32_t)weight[m], ld = (uint32_t)load[m * D + d];
                const int32_t here = c * kChunk + k;
                uint32_t held = 0;  // the models on the device
#pragma unroll
                for (int i = 0; i < kI; ++i) held |= ((__ballot_sync(0xFFFFFFFFu, x[i] >> 16) >> shift) & kAll) << (i * kL);
                const bool was_empty = held == 0, hit = (held >> m) & 1u;
                held &= ~(1u << m);
                const uint32_t need = hit ? r1 : wm + r1;  // at most the capacity
                if (__any_sync(0xFFFFFFFFu, act && need > f)) {
                    int32_t cost[kI], dist[kI];  // cost 0 (and distance 1): infinite
                    uint32_t key[kI], ahead[kI], nearest[kI];
#pragma unroll
                    for (int i = 0; i < kI; ++i) {
                        cost[i] = load[mrow[i] + d];
                        const uint32_t nuse = x[i] & 0xFFFFu;
                        const bool inf = nuse == 0xFFFFu || cost[i] == 0;
                        dist[i] = inf ? 1 : (int32_t)nuse - here;
                        // (infinite: in the order of last use, and too far apart to be called near)
                        const uint32_t q = inf ? 0x7F800000u + ((0xFFFFu - (x[i] >> 16)) << 4)
                                               : __float_as_uint((float)dist[i] * rcost[mrow[i] + d]);
                        key[i] = (held >> (ml + i * kL)) & 1u ? (copies[i] > 1 ? 0x80000000u : 0u) | q : 0u;
                        cost[i] = inf ? 0 : cost[i];
                    }
                    // The weight of the copies that go before each of this lane's, and how near the nearest quotient is.
                    if constexpr (kI == 2) {
                        ahead[0] = key[1] > key[0] ? wx[0][1] : 0u;
                        ahead[1] = key[0] > key[1] ? wx[0][0] : 0u;
                        nearest[0] = key[1] - key[0] + kNear;
                        nearest[1] = key[0] - key[1] + kNear;
                    } else {
                        ahead[0] = 0;
                        nearest[0] = ~0u;
                    }
#pragma unroll
                    for (int o = 1; o < kL; ++o)
#pragma unroll
                        for (int j = 0; j < kI; ++j) {
                            const uint32_t pk = __shfl_xor_sync(0xFFFFFFFFu, key[j], o);
#pragma unroll
                            for (int i = 0; i < kI; ++i) {
                                if (pk > key[i]) ahead[i] += wx[o][j];
                                nearest[i] = min(nearest[i], pk - key[i] + kNear);
                            }
                        }
                    bool close = false;
#pragma unroll
                    for (int i = 0; i < kI; ++i) close |= key[i] && nearest[i] <= 2 * kNear;
                    if (__any_sync(0xFFFFFFFFu, close && act && need > f)) {
#pragma unroll
                        for (int i = 0; i < kI; ++i) ahead[i] = 0;
                        for (int o = 0; o < kL; ++o)
#pragma unroll
                            for (int j = 0; j < kI; ++j) {
                                const uint32_t pk = __shfl_xor_sync(0xFFFFFFFFu, key[j], o), ps = __shfl_xor_sync(0xFFFFFFFFu, x[j] >> 16, o);
                                const int32_t pd = __shfl_xor_sync(0xFFFFFFFFu, dist[j], o), pc = __shfl_xor_sync(0xFFFFFFFFu, cost[j], o);
#pragma unroll
                                for (int i = 0; i < kI; ++i) {
                                    bool before = pk > key[i];
                                    if (key[i] && pk - key[i] + kNear <= 2 * kNear) {
                                        const int64_t l = (int64_t)pd * cost[i], r = (int64_t)dist[i] * pc;
                                        before = l > r || (l == r && ps < x[i] >> 16);  // (never before itself)
                                    }
                                    if (before) ahead[i] += (uint32_t)weight[(ml ^ o) + j * kL];
                                }
                            }
                    }
                    uint32_t gone = 0;
#pragma unroll
                    for (int i = 0; i < kI; ++i) {
                        const bool goes = act && key[i] && need > f + ahead[i];
                        gone |= ((__ballot_sync(0xFFFFFFFFu, goes) >> shift) & kAll) << (i * kL);
                        if (goes) { x[i] = 0; copies[i] -= 1; }
                    }
                    held &= ~gone;
                    f += wsum[gone & 255u];
                    if (sizeof(Q) > 4) f += wsum[256 + (gone >> 8)];
                    if (act && need > f) atomicExch(dp.err, 2);  // unreachable for a valid plan
                }
                const bool drop = (r3 & kDrop) != 0;  // the model leaves when the unit ends
                if (!hit && !drop) f -= wm;
                if (hit && drop) f += wm;
                if (act) {
                    const uint32_t mine = drop ? 0u : nu | ((uint32_t)(here + 1) << 16);
                    const uint32_t more = (hit ? 0u : 1u) - (drop ? 1u : 0u);
                    uint32_t reload = 0;
#pragma unroll
                    for (int i = 0; i < kI; ++i)
                        if ((uint32_t)(ml + i * kL) == m) {
                            copies[i] += more;
                            x[i] = mine;
                            if (kPhi && !hit) {
                                reload = ((ever[i] >> d) & 1u) << 31;
                                ever[i] |= 1u << d;
                            }
                        }
                    if ((uint32_t)ml == m % kL) {
                        uint2 w = settled(r3, hit, ld, was_empty, drop && held == 0);
                        if (kPhi) w.x |= reload;
                        room[d * kP] = f;
                        rb[(1 * kChunk + k) * kPitch] = w;
                    }
                    set_row(d, x);
                }
                __syncwarp();  // the free capacity is written
                v = nv;
                nu = nnu;
            }
            named_arrive(kFullR + b, kResThreads + 32);
        }
        uint32_t o = 0;  // devices still occupied at the end
        for (int32_t d = 0; d < D; ++d) {
            uint32_t x[kI], any = 0;
            row_of(d, x);
#pragma unroll
            for (int i = 0; i < kI; ++i) any |= x[i] >> 16;
            o += ((__ballot_sync(0xFFFFFFFFu, any) >> shift) & kAll) != 0;
        }
        if (live && ml == 0 && o) atomicAdd(open + qp, o);
        }
        named_arrive(kOpen, kResThreads + 32);
    } else {
    // ---------------- timing: lane = plan (Eq. 2, 5, 7, 10) ----------------
    const bool mine = lane < kP;  // lanes at or beyond kP own no plan and touch no per-plan state
    const int64_t p = (mine && lane < ng) ? (in_list ? (int64_t)in_list[j0 + lane] : j0 + lane) : 0;
    const bool live = mine && lane < ng && out.status[p] == 0;
    SlotArr<TT, ST, kP> slots;
    if constexpr (SlotBytes<ST>::kHi) {
        slots.lo = (uint32_t *)(sm + L.slots) + lane;
        slots.hi = sm + L.slots_hi + lane;
    } else {
        slots.v = (TT *)(sm + L.slots) + lane;
    }
    TT *tfree = (TT *)(sm + L.tfree) + lane;
    if (mine) {
        for (int32_t k = 0; k < dp.nslots + 2; ++k) slots.set(k, 0);
        for (int32_t d = 0; d < D; ++d) tfree[d * kP] = 0;
    }
    __syncthreads();
    const uint32_t trash = (uint32_t)dp.nslots;
    // u32 times: a plan is handed on when a sum carries out, or when a finish
    // reaches 2^32 - 1 (which a saturated w0 forces).  u64 times cannot wrap;
    // only a saturated w0 is handed on.
    TT end = 0;
    uint32_t ovf = 0;
    int64_t gsum = 0;
    uint32_t ph_timely = 0;  // Eq. 12 window terms (kPhi)
    uint64_t ph_life = 0;
    // Relative times (kRel): the base, the base saturated to 32 bits (for the
    // arrivals), emptied minus newly occupied devices so far (gsum counts
    // from the base), and the rebases so far.
    uint64_t base = 0;
    uint32_t bc = 0;
    int32_t net = 0, nreb = 0;
    const int64_t rcol = (int64_t)blockIdx.x * kP + lane, rstride = (int64_t)gridDim.x * kP;
    for (int32_t c = 0; c < chunks; ++c) {
        const int b = c % kBuffers;
        named_sync(kFullR + b, kResThreads + 32);
        if constexpr (kRel) {
            // Raise the base of every plan whose end nears 2^32.  The whole
            // warp walks the CTA's slot words ([slot][plan], 32 at a time,
            // word x of plan x % kP), each lowered by its plan's rise.
            if (__any_sync(0xFFFFFFFFu, live && !ovf && end > kRebaseAt)) {
                uint32_t m = 0xFFFFFFFFu;
                if (live && !ovf)
                    for (int32_t d = 0; d < D; ++d) m = min(m, tfree[d * kP]);
                const uint32_t dl = live && !ovf && m > kRebaseMin ? m - 1 : 0u;
                uint32_t *sw = (uint32_t *)(sm + L.slots);
                __syncwarp();  // every lane's slot writes are seen by the others
                const int32_t nw = W * kP, nall = (dp.nslots + 2) * kP;
                for (int32_t x0 = 0; x0 < nw; x0 += 32) {  // session slots: keep what falls below the base
                    const int32_t x = x0 + lane, q = x % kP;
                    const uint32_t dq = __shfl_sync(0xFFFFFFFFu, dl, q);
                    const uint64_t bq = __shfl_sync(0xFFFFFFFFu, base, q);
                    const int32_t rq = __shfl_sync(0xFFFFFFFFu, nreb, q);
                    if (x < nw && dq) {
                        const uint32_t v = sw[x];
                        uint64_t *r = dp.rel_ret + (int64_t)(x / kP) * rstride + (int64_t)blockIdx.x * kP + q;
                        const uint64_t keep = v && v <= dq ? bq + v : 0ull;
                        *r = rq ? max(*r, keep) : keep;
                        sw[x] = v > dq ? v - dq : 0u;
                    }
                }
                for (int32_t x0 = nw; x0 < nall; x0 += 32) {
                    const int32_t x = x0 + lane;
                    const uint32_t dq = __shfl_sync(0xFFFFFFFFu, dl, x % kP);
                    if (x < nall && dq) {
                        const uint32_t v = sw[x];
                        sw[x] = v > dq ? v - dq : 0u;
                    }
                }
                if (dl) {
                    for (int32_t d = 0; d < D; ++d) tfree[d * kP] -= dl;
                    end -= dl;
                    gsum -= (int64_t)net * dl;
                    base += dl;
                    bc = base < 0xFFFFFFFFull ? (uint32_t)base : 0xFFFFFFFFu;
                    ++nreb;
                }
                __syncwarp();
            }
        }
        const uint2 *rb = ring + b * kRW * kChunk * kPitch + lane;
        if (live) {
            // The ring words of the next position are read while this one
            // plays.  A skip record plays as a unit that changes nothing (no
            // run time, no load, the zero slot, the sink), so every lane
            // plays every position of the chunk without branching.
            uint2 w[3];
#pragma unroll
            for (int x = 0; x < 3; ++x) w[x] = rb[(x * kChunk) * kPitch];
#pragma unroll 4
            for (int32_t k = 0; k < kChunk; ++k) {
                const int32_t kn = min(k + 1, kChunk - 1);
                uint2 nw[3];
#pragma unroll
                for (int x = 0; x < 3; ++x) nw[x] = rb[(x * kChunk + kn) * kPitch];
                const uint32_t r3 = w[1].y;
                const uint32_t run = w[0].x, arr = kRel ? max(w[0].y, bc) - bc : w[0].y, r4 = w[2].x, r5 = w[2].y;
                const uint32_t ld = kPhi ? w[1].x & 0x7FFFFFFFu : w[1].x;  // bit 31: a reload (kPhi)
                TT *tf_d = tfree + (r3 & 31u) * kP;
                // Every slot of the unit is read before any is written (the
                // producers took the accumulator bit off a code that names
                // the slot which this unit resets).
                const uint32_t rs = r5 >> 16, i0 = (r3 >> 16) & 0x7FFFu, i1 = r4 & 0x7FFFu;
                const TT rel = max((TT)arr, slots.get(rs & 0x7FFFu));  // release (Eq. 2, Eq. 7)
                const TT tf = *tf_d, old0 = slots.get(i0), old1 = slots.get(i1);
                // A miss loads on this device first (ld > 0 only on a miss); a
                // prefetched load waits only for the arrival (Eq. 5).  On a hit
                // the residency stage cleared the prefetch bit and ld is 0.
                const TT ls = max(tf, (r3 & kPrefetch) ? (TT)arr : rel);
                TT le, start, cfin;
                if constexpr (kNarrow) {
                    le = add_carry(ls, ld, ovf);
                    start = max(le, rel);
                    cfin = add_carry(start, run, ovf);
                } else {
                    le = ls + ld;
                    start = max(le, rel);
                    cfin = start + run;
                    ovf |= run == kRunCap;
                }
                if (kPhi) {
                    // A prefetched load (the bit survives residency only on a
                    // miss) that starts before the release and ends by it is
                    // timely; every unit adds the delay its load puts on its
                    // start, and a reload its load time.
                    ph_timely += (r3 & kPrefetch) && ls < rel && le <= rel;
                    ph_life += (uint64_t)(start - max(tf, rel)) + (w[1].x >> 31 ? (uint64_t)ld : 0ull);
                }
                end = max(end, cfin);
                slots.set((rs & 0x8000u) ? (rs & 0x7FFFu) : trash, 0);  // an accumulator is reset by its reader
                slots.set(i0, (r3 & 0x80000000u) ? max(old0, cfin) : cfin);  // the sink when the unit writes nothing
                slots.set(i1, (r4 & 0x8000u) ? max(old1, cfin) : cfin);
                *tf_d = cfin;
                if (r3 & (kMany | kWasEmpty | kEmptied)) {
                    if (r3 & kWasEmpty) {  // an empty device becomes occupied
                        gsum -= (int64_t)ls;
                        if (kRel) --net;
                    }
                    if (r3 & kEmptied) {  // the device empties after the unit
                        gsum += (int64_t)cfin;
                        if (kRel) ++net;
                    }
                    if (r3 & kMany) {
                        publish<TT>(slots, r4 >> 16, cfin);
                        const uint32_t nwl = (r3 >> 11) & 7u;
                        if (nwl == kWrites4) {
                            publish<TT>(slots, r5 & 0xFFFFu, cfin);
                        } else if (nwl > kWrites4) {  // five or more codes: the list from global memory
                            const int4 wr = __ldg(dp.noderec + 2 * (int32_t)(r5 & 0xFFFFu) + 1);
                            for (int32_t e = 3; e < wr.y; ++e) publish<TT>(slots, __ldg(dp.wl + wr.x + e), cfin);
                        }
                    }
                }
#pragma unroll
                for (int x = 0; x < 3; ++x) w[x] = nw[x];
            }
        }
        // Once every plan of the CTA has left 32 bits, the producers stop
        // loading (they see the flag a chunk or two later).
        if (kNarrow && __all_sync(0xFFFFFFFFu, !live || ovf) && lane == 0) *gave_up = 1;
        named_arrive(kEmpty + b, kProdThreads + 32);  // buffer b may be refilled
    }
    if (kNarrow) ovf |= end == (TT)kRunCap;
    named_sync(kOpen, kResThreads + 32);  // the residency stage's final device counts
    const uint32_t bad = live ? open[lane] >> kOpenBad : 0u;  // placement bits found by the producers
    if (bad) {  // an invalid plan: its status bits and INT64_MAX metrics
        out.status[p] = bad;
        out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
        if (kPhi) dp.phi_timely[p] = dp.phi_life[p] = WF_INF64;
    } else if (live && ovf) {  // handed to the next path
        const int32_t kk = atomicAdd(ovf_count, 1);
        ovf_list[kk] = (int32_t)p;
    } else if (live && kRel) {
        // Back to absolute times: the session latencies as 64-bit values in
        // slot pairs (written from the last session down, so that no pair
        // overwrites a session slot not yet read).
        const int64_t nopen = open[lane];
        const uint64_t eabs = base + end;
        const PairArr<kP> lat{(uint32_t *)(sm + L.slots) + lane};
        for (int32_t w = W - 1; w >= 0; --w) {
            const uint32_t v = slots.get(w);
            uint64_t cw = v ? base + v : 0ull;
            if (nreb) cw = max(cw, dp.rel_ret[(int64_t)w * rstride + rcol]);
            lat.set(w, cw - arrival[w]);
        }
        out.makespan_us[p] = (int64_t)eabs - dp.first_arrival;
        out.gpu_us[p] = gsum + (int64_t)net * (int64_t)base + nopen * (int64_t)eabs;
        if (W <= kLaneSelect) out.p95_us[p] = (int64_t)select_slots<uint64_t>(lat, W, rank);
    } else if (live) {
        const int64_t nopen = open[lane];
        for (int32_t w = 0; w < W; ++w) slots.set(w, slots.get(w) - arrival[w]);  // session completion latency
        out.makespan_us[p] = (int64_t)end - dp.first_arrival;
        out.gpu_us[p] = gsum + nopen * (int64_t)end;
        if (W <= kLaneSelect) out.p95_us[p] = (int64_t)select_slots<TT>(slots, W, rank);
        if (kPhi) {
            dp.phi_timely[p] = ph_timely;
            dp.phi_life[p] = (int64_t)ph_life;
        }
    }
    // A plan whose p95 is still to be selected (more than kLaneSelect sessions).
    if (mine) open[lane] = live && !bad && !ovf && W > kLaneSelect;
    }
    __syncthreads();  // every stage is done with the group
    // The p95 of every plan played to the end with more than kLaneSelect
    // sessions (Section 4.2, nearest rank): the whole CTA, a warp per plan,
    // over the session latencies the timing stage left in the plan's slots.
    for (int q = warp; q < kP && W > kLaneSelect; q += S::kWarps) {
        if (!open[q]) continue;
        uint64_t v;
        if constexpr (kRel) {
            v = warp_select(PairArr<kP>{(uint32_t *)(sm + L.slots) + q}, W, rank);
        } else {
            SlotArr<TT, ST, kP> sq;
            if constexpr (SlotBytes<ST>::kHi) {
                sq.lo = (uint32_t *)(sm + L.slots) + q;
                sq.hi = sm + L.slots_hi + q;
            } else {
                sq.v = (TT *)(sm + L.slots) + q;
            }
            v = warp_select(sq, W, rank);
        }
        if (lane == 0) out.p95_us[in_list ? (int64_t)in_list[j0 + q] : j0 + q] = (int64_t)v;
    }
    __syncthreads();  // the group's shared state is free for the next group
  }
}

// Next use, for reclamation by next use: for every dispatch position i that
// starts a unit, the next position that starts a unit on the same device with
// the same model (0xFFFF: none).  A warp per plan walks its positions from the
// end, 32 at a time; lanes with equal (device, model) keys find each other
// with __match_any_sync, and a shared table carries the first occurrence of
// each key to the chunk before.  On windows of several chunks (kDeep) three
// chunks of gathers are in flight ahead of the one being settled; one or two
// chunks have nothing to run ahead of, and what bounds those is the plans an
// SM holds: 32 registers instead of 48, no read for a position that is not
// there.  39,692 plans of N = 22, us: 18.3 with the deep form, 12.5 without; the
// call on 30,000 plans of N = 32, D = M = 8 137 and 134, of N = 64 212 and 209, and
// from N = 128 on the deep form is ahead (355 and 359).
constexpr int kNuWarps = 4;
constexpr int32_t kNuShort = 64;  // activations

template <bool kDeep>
__global__ void __launch_bounds__(32 * kNuWarps)
nextuse_kernel(wf_dev_problem dp, wf_plans pl, const uint32_t *status, uint16_t *table)
{
    extern __shared__ __align__(16) uint8_t nsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t N = dp.N, D = dp.D, M = dp.M;
    uint16_t *last = (uint16_t *)nsm + warp * D * M;
    for (int64_t p = (int64_t)blockIdx.x * kNuWarps + warp; p < pl.P; p += (int64_t)gridDim.x * kNuWarps) {
        if (__ldg(status + p) != 0) continue;  // uniform over the warp
        const uint8_t *place = pl.place + p * pl.place_stride;
        const uint16_t *order = (const uint16_t *)((const uint8_t *)pl.order + p * pl.order_stride);
        const uint32_t *fuse = (const uint32_t *)((const uint8_t *)pl.fuse + p * pl.bits_stride);
        uint16_t *out = table + p * (int64_t)N;
        for (int32_t k = lane; k < D * M; k += 32) last[k] = 0xFFFFu;
        __syncwarp();
        // The chunks ahead: dispatch entries, then their nodes' placement,
        // record and fusion word, then the placement of their fusible
        // predecessors.
        const int32_t top = ((N - 1) / 32) * 32 + lane;
        auto entry = [&](int32_t j) { return j >= 0 && j < N ? (int32_t)__ldg(order + j) : 0; };
        struct Node {
            uint32_t d, x, links, model, fw;
        };
        auto node = [&](int32_t h) {
            const uint4 hr = __ldg(dp.hrec + h);
            return Node{__ldg(place + h), (uint32_t)h, hr.x, (hr.y >> 16) & 15u, __ldg(fuse + (h >> 5))};
        };
        auto before = [&](const Node &n) { return (n.links & 0xFFFFu) != 0xFFFFu ? (uint32_t)__ldg(place + (n.links & 0xFFFFu)) : ~0u; };
        Node n1, n2;
        uint32_t p1 = 0;
        int32_t h3 = 0;
        if constexpr (kDeep) {
            n1 = node(entry(top));
            n2 = node(entry(top - 32));
            p1 = before(n1);
            h3 = entry(top - 64);
        }
        for (int32_t base = ((N - 1) / 32) * 32; base >= 0; base -= 32) {
            const int32_t j = base + lane;
            uint32_t key = 0xFFFFFFFFu;  // not the start of a unit
            if constexpr (kDeep) {
                const Node n = n1;
                const uint32_t pn = p1;
                n1 = n2;
                p1 = before(n1);
                n2 = node(h3);
                h3 = entry(j - 96);
                if (j < N && !(((n.fw >> (n.x & 31)) & 1u) && pn == n.d)) key = n.d * M + n.model;
            } else if (j < N) {
                const int32_t x = __ldg(order + j);
                const uint32_t d = __ldg(place + x);
                const uint4 hr = __ldg(dp.hrec + x);
                const uint32_t fp = hr.x & 0xFFFFu;
                if (fp == 0xFFFFu || !bit_of_g(fuse, x) || __ldg(place + fp) != d) key = d * M + ((hr.y >> 16) & 15u);
            }
            const uint32_t same = __match_any_sync(0xFFFFFFFFu, key);
            const uint32_t above = lane == 31 ? 0u : (same & (0xFFFFFFFFu << (lane + 1)));
            if (key != 0xFFFFFFFFu) out[j] = above ? (uint16_t)(base + __ffs((int)above) - 1) : last[key];
            __syncwarp();
            if (key != 0xFFFFFFFFu && lane == __ffs((int)same) - 1) last[key] = (uint16_t)j;
            __syncwarp();
        }
    }
}

// Status bits of every plan (Eq. 8-10), one warp per plan.  Four nodes per
// lane check placement and fit (one fit mask per node); the warp scatters the
// inverse of the dispatch sequence (u16 positions) into empty cells of shared
// memory: a repeated node leaves a cell empty, so every in-range sequence
// that fills them all is a permutation.  (Reading the sequence again and
// comparing every entry: 60.5 us at 16,384 plans of N = 2,000; so 50.8.)
// The edges (pred | succ << 16) are then checked 32 at a time.  Invalid plans
// get INT64_MAX metrics here; the sweep skips them.
__host__ __device__ inline uint32_t status_warp_bytes(int32_t N)
{
    return round16(2u * (uint32_t)N);
}

// kByte: every device index is below 8, so one byte per node holds its fit
// mask (fit8): a quarter of the table reads of the 32-bit masks.
template <bool kByte, int kU, bool kPlace>
__global__ void __launch_bounds__(128)
status_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out)
{
    extern __shared__ __align__(16) uint8_t ssm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int32_t N = dp.N, D = dp.D, E = dp.E;
    uint16_t *pos = (uint16_t *)(ssm + (size_t)warp * status_warp_bytes(N));
    // Plans are visited from the last to the first: the rows read last stay
    // in L2, and they are those of the sweep's first wave of CTAs (the
    // lowest plan indices), which then re-reads them from L2 rather than DRAM.
    for (int64_t k = (int64_t)blockIdx.x * warps + warp; k < pl.P; k += (int64_t)gridDim.x * warps) {
        const int64_t p = pl.P - 1 - k;
        const uint8_t *place = pl.place + p * pl.place_stride;
        const uint16_t *order = (const uint16_t *)((const uint8_t *)pl.order + p * pl.order_stride);
        uint32_t st = 0;
        // Rows start 16-byte aligned and their strides are multiples of 16
        // bytes, so 16-byte reads at multiples of 16 bytes below N stay in
        // the row; lanes mask the entries at or beyond N.  The fit masks are
        // padded to 16 entries.
        // Every loop issues kU 16-byte reads per lane before it uses any: on
        // long rows a warp keeps a plan's reads in flight rather than one
        // round trip per 512 bytes (kU = 1 on short rows, whose loops run once).
        // The inverse permutation, 8 dispatch entries a lane at a time, into
        // cells that held no position before: N entries leave a cell empty
        // exactly when one repeats another (or is out of range).
        for (int32_t b8 = 8 * lane; b8 < N; b8 += 256) *(uint4 *)(pos + b8) = make_uint4(~0u, ~0u, ~0u, ~0u);
        __syncwarp();
        for (int32_t b8 = 8 * lane; b8 < N; b8 += kU * 256) {
            uint4 ow[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                ow[u] = b8 + 256 * u < N ? __ldg((const uint4 *)(order + b8 + 256 * u)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int32_t i8 = b8 + 256 * u;
                const uint32_t w[4] = {ow[u].x, ow[u].y, ow[u].z, ow[u].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t h = (w[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
                    if (i8 + j < N) {
                        if (h < (uint32_t)N) pos[h] = (uint16_t)(i8 + j);
                        else st |= WF_ST_PERMUTATION;
                    }
                }
            }
        }
        __syncwarp();
        for (int32_t b8 = 8 * lane; b8 < N; b8 += 256) {
            const uint4 c = *(const uint4 *)(pos + b8);
            const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // (cells at and beyond N stay empty; a position is below 0xFFFF)
                const bool lo = (w[j] & 0xFFFFu) == 0xFFFFu && b8 + 2 * j < N, hi = (w[j] >> 16) == 0xFFFFu && b8 + 2 * j + 1 < N;
                if (lo || hi) st |= WF_ST_PERMUTATION;
            }
        }
        st = __reduce_or_sync(0xFFFFFFFFu, st);
        if (!(st & WF_ST_PERMUTATION)) {
            for (int32_t b4 = 4 * lane; b4 < E; b4 += kU * 128) {  // edges padded to 4
                uint4 uv[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    uv[u] = b4 + 128 * u < E ? __ldg((const uint4 *)(dp.edges + b4 + 128 * u)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t e4 = b4 + 128 * u;
                    const uint32_t w[4] = {uv[u].x, uv[u].y, uv[u].z, uv[u].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (e4 + j < E && pos[w[j] & 0xFFFFu] > pos[w[j] >> 16]) st |= WF_ST_TOPOLOGY;
                }
            }
            st = __reduce_or_sync(0xFFFFFFFFu, st);
        }
        // Placement and fit (Eq. 8): here when asked (kPlace), else only for
        // a plan whose order is already invalid; the sweep's producers check
        // the placement of every other plan as they read it.
        if (kPlace || st) {
            for (int32_t b16 = 16 * lane; b16 < N; b16 += kU * 512) {
                uint4 pw[kU], fb[kU], fm[kU][4];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t n16 = b16 + 512 * u;
                    const bool in = n16 < N;
                    pw[u] = in ? __ldg((const uint4 *)(place + n16)) : make_uint4(0u, 0u, 0u, 0u);
                    if (kByte) {
                        fb[u] = in ? __ldg((const uint4 *)(dp.fit8 + n16)) : make_uint4(0u, 0u, 0u, 0u);
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            fm[u][q] = in ? __ldg((const uint4 *)(dp.fitmask + n16 + 4 * q)) : make_uint4(0u, 0u, 0u, 0u);
                    }
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t n16 = b16 + 512 * u;
                    const uint32_t pws[4] = {pw[u].x, pw[u].y, pw[u].z, pw[u].w};
                    if (kByte) {
                        const uint32_t fbs[4] = {fb[u].x, fb[u].y, fb[u].z, fb[u].w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t d = (pws[q] >> (8 * j)) & 255u, f = (fbs[q] >> (8 * j)) & 255u;
                                if (n16 + 4 * q + j < N)
                                    st |= d >= (uint32_t)D ? WF_ST_DEVICE
                                                           : (((f >> (d & 7u)) & 1u) ? 0u : WF_ST_CAPACITY);
                            }
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t f[4] = {fm[u][q].x, fm[u][q].y, fm[u][q].z, fm[u][q].w};
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint32_t d = (pws[q] >> (8 * j)) & 255u;
                                if (n16 + 4 * q + j < N)
                                    st |= d >= (uint32_t)D ? WF_ST_DEVICE : (((f[j] >> d) & 1u) ? 0u : WF_ST_CAPACITY);
                            }
                        }
                    }
                }
            }
        }
        st = __reduce_or_sync(0xFFFFFFFFu, st);
        if (lane == 0) {
            out.status[p] = st;
            if (st) out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
            if (st && dp.phi_life) dp.phi_timely[p] = dp.phi_life[p] = WF_INF64;
        }
        __syncwarp();  // pos[] is reused by the warp's next plan
    }
}

template <bool kByte, int kU, bool kPlace>
int launch_status_as(const wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    const size_t wbytes = status_warp_bytes(dp.N);
    const int swarps = (int)std::max<size_t>(1, std::min<size_t>(4, (227 * 1024) / wbytes));
    const size_t ssmem = wbytes * swarps;
    int rc = wf_cuda_check(cudaFuncSetAttribute(status_kernel<kByte, kU, kPlace>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem),
                           "status smem attribute");
    if (rc) return rc;
    const int64_t sblocks = std::min<int64_t>((pl->P + swarps - 1) / swarps, (int64_t)ctx->sms * 16);
    status_kernel<kByte, kU, kPlace><<<(unsigned)sblocks, 32 * swarps, ssmem, st>>>(dp, *pl, *out);
    return WF_OK;
}

template <bool kPlace>
int launch_status_p(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, cudaStream_t st)
{
    const bool byte = ctx->dp.D <= 8, wide = ctx->dp.N >= 1024;
    if (wide)
        return byte ? launch_status_as<true, 4, kPlace>(ctx, pl, out, st)
                    : launch_status_as<false, 4, kPlace>(ctx, pl, out, st);
    return byte ? launch_status_as<true, 1, kPlace>(ctx, pl, out, st)
                : launch_status_as<false, 1, kPlace>(ctx, pl, out, st);
}

}  // namespace

// The status pass; with place false the placement and fit checks of a plan
// whose order is valid are left to the deterministic sweep's producers.
int wf_launch_status(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, cudaStream_t st, bool place)
{
    return place ? launch_status_p<true>(ctx, pl, out, st) : launch_status_p<false>(ctx, pl, out, st);
}

namespace {

bool sweep_usable(const wf_dev_problem &dp)
{
    return dp.nslots > 0 && dp.nslots <= 32765 && dp.max_arrival < ((int64_t)1 << 32) && dp.M <= 16 &&
           dp.N <= 65534;
}

// The 64-bit sweep keeps its slots in 40 bits when no time of the window can
// reach 2^40 us (the context's horizon bounds every finish) and reclamation
// is least recently used.
bool split40(const wf_dev_problem &dp) { return below40(dp) && dp.reclaim == 0; }

// The relative-time sweep: least recently used, no window terms, and room
// for the sessions' 64-bit latencies in slot pairs at the end of a plan.
bool rel32(const wf_dev_problem &dp)
{
    return sweep_usable(dp) && dp.reclaim == 0 && !dp.phi_life && 2 * (int64_t)dp.W <= (int64_t)dp.nslots + 2;
}

template <typename Q, typename TT, int kP, int kR, bool kF, typename ST = TT>
int launch_pc(const wf_dev_problem &dp, int sms, int resident, const wf_plans *pl, const wf_eval_out *out,
              size_t smem, const int32_t *in_list, const int32_t *in_count, int32_t *list, int32_t *count, cudaStream_t st)
{
    int rc = wf_cuda_check(cudaFuncSetAttribute(pc_kernel<Q, TT, kP, kR, kF, ST>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                           "sweep smem attribute");
    if (rc) return rc;
    // Every plan: a CTA per group.  A list (of unknown length): at most as
    // many CTAs as are resident at once, each walking over groups.
    int64_t blocks = (pl->P + kP - 1) / kP;
    if (in_list) blocks = std::min<int64_t>(blocks, (int64_t)std::max(1, resident) * sms);
    pc_kernel<Q, TT, kP, kR, kF, ST><<<(unsigned)blocks, 32 * PcShape<kP, kR, Q>::kWarps, smem, st>>>(
        dp, *pl, *out, in_list, in_count, list, count);
    return wf_cuda_check(cudaGetLastError(), "sweep launch");
}

// Calls f(Ty<Q>{}, Iv<kP>{}, Ty<ST>{}) for the sweep instantiation that this
// problem and CTA shape take: Q the LRU word (up to 8 models pack in 32 bits),
// kP the plans per CTA, ST the finish-slot storage.
template <typename TT, int kR, typename F>
int pc_visit(const wf_dev_problem &dp, int kp, F &&f)
{
    auto by_q = [&](auto p, auto s) {
        if constexpr (kR == kNuModel)
            if (dp.M <= 4) return f(Ty<uint16_t>{}, p, s);
        return dp.M <= 8 ? f(Ty<uint32_t>{}, p, s) : f(Ty<uint64_t>{}, p, s);
    };
    if constexpr (sizeof(TT) == 4) {  // the u32 sweep has one shape
        (void)kp;
        return by_q(Iv<kPlans32>{}, Ty<TT>{});
    } else {
        auto by_p = [&](auto s) {
            if constexpr (kR != 0)
                if (kp == 2) return by_q(Iv<2>{}, s);
            return kp == 16 ? by_q(Iv<16>{}, s) : kp == 6 ? by_q(Iv<6>{}, s) : by_q(Iv<3>{}, s);
        };
        if constexpr (kR == 0)
            if (split40(dp)) return by_p(Ty<Split40>{});
        return by_p(Ty<TT>{});
    }
}

template <typename TT, int kR, bool kF>
int launch_pc_r(const wf_ctx *ctx, int kp, int resident, const wf_plans *pl, const wf_eval_out *out, size_t smem,
                const int32_t *in_list, const int32_t *in_count, int32_t *list, int32_t *count, cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    return pc_visit<TT, kR>(dp, kp, [&](auto q, auto p, auto s) {
        return launch_pc<typename decltype(q)::type, TT, decltype(p)::value, kR, kF, typename decltype(s)::type>(
            dp, ctx->sms, resident, pl, out, smem, in_list, in_count, list, count, st);
    });
}

// CTAs of the sweep instantiation resident on one SM at this shared-memory
// size: registers and shared memory both count (0 = it does not fit).
template <typename TT, int kR, bool kF>
int resident_r(const wf_dev_problem &dp, int kp, size_t smem)
{
    if (smem > 227 * 1024) return 0;
    return pc_visit<TT, kR>(dp, kp, [&](auto q, auto p, auto s) {
        const auto k = pc_kernel<typename decltype(q)::type, TT, decltype(p)::value, kR, kF, typename decltype(s)::type>;
        int n = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &n, k, 32 * PcShape<decltype(p)::value, kR, typename decltype(q)::type>::kWarps, smem) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        return n;
    });
}

template <typename TT>
int resident(const wf_dev_problem &dp, int kp, size_t smem)
{
    if (dp.phi_life)
        return dp.reclaim ? resident_r<TT, 1, true>(dp, kp, smem) : resident_r<TT, 0, true>(dp, kp, smem);
    return dp.reclaim ? resident_r<TT, 1, false>(dp, kp, smem) : resident_r<TT, 0, false>(dp, kp, smem);
}

// The relative-time sweep's shapes: 16 or 6 plans per CTA.
template <typename F>
int rel_visit(const wf_dev_problem &dp, int kp, F &&f)
{
    auto by_q = [&](auto p) {
        return dp.M <= 8 ? f(Ty<uint32_t>{}, p) : f(Ty<uint64_t>{}, p);
    };
    return kp == 16 ? by_q(Iv<16>{}) : by_q(Iv<6>{});
}

int resident_rel(const wf_dev_problem &dp, int kp, size_t smem)
{
    if (smem > 227 * 1024) return 0;
    return rel_visit(dp, kp, [&](auto q, auto p) {
        const auto k = pc_kernel<typename decltype(q)::type, uint32_t, decltype(p)::value, 0, false, Rel32>;
        int n = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32 * PcShape<decltype(p)::value>::kWarps, smem) !=
                cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        return n;
    });
}

// Every plan of the batch, in at most as many CTAs as are resident at once
// and as the evaluation scratch holds session rows for (each CTA walks
// over groups); the plans that leave 32 bits go to list.
int64_t rel_blocks(const wf_ctx *ctx, const wf_sweep_cfg &cfg, int64_t P)
{
    if (!cfg.smemRel) return 0;
    const int kp = cfg.plansRel;
    const int64_t rows = (int64_t)(ctx->eval_scratch_bytes / (8 * (size_t)std::max(ctx->dp.W, 1)));
    return std::min<int64_t>(std::min<int64_t>((P + kp - 1) / kp, (int64_t)std::max(1, cfg.resRel) * ctx->sms),
                             rows / kp);
}

int launch_rel(wf_ctx *ctx, const wf_sweep_cfg &cfg, int64_t blocks, const wf_plans *pl, const wf_eval_out *out,
               int32_t *list, int32_t *count, cudaStream_t st)
{
    wf_dev_problem dp = ctx->dp;
    dp.rel_ret = (uint64_t *)ctx->eval_scratch;
    return rel_visit(dp, cfg.plansRel, [&](auto q, auto p) {
        const auto k = pc_kernel<typename decltype(q)::type, uint32_t, decltype(p)::value, 0, false, Rel32>;
        int rc = wf_cuda_check(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.smemRel),
                               "sweep smem attribute");
        if (rc) return rc;
        k<<<(unsigned)blocks, 32 * PcShape<decltype(p)::value>::kWarps, cfg.smemRel, st>>>(dp, *pl, *out, nullptr,
                                                                                           nullptr, list, count);
        return wf_cuda_check(cudaGetLastError(), "sweep launch");
    });
}

template <typename TT>
int launch_pc_q(const wf_ctx *ctx, int kp, int resident, const wf_plans *pl, const wf_eval_out *out, size_t smem,
                const int32_t *in_list, const int32_t *in_count, int32_t *list, int32_t *count, cudaStream_t st)
{
    if (ctx->dp.phi_life)
        return ctx->dp.reclaim
                   ? launch_pc_r<TT, 1, true>(ctx, kp, resident, pl, out, smem, in_list, in_count, list, count, st)
                   : launch_pc_r<TT, 0, true>(ctx, kp, resident, pl, out, smem, in_list, in_count, list, count, st);
    return ctx->dp.reclaim
               ? launch_pc_r<TT, 1, false>(ctx, kp, resident, pl, out, smem, in_list, in_count, list, count, st)
               : launch_pc_r<TT, 0, false>(ctx, kp, resident, pl, out, smem, in_list, in_count, list, count, st);
}

}  // namespace

// Whether reclamation by next use settles with a lane per plan: short windows in
// batches large enough that the instructions of all plans bound the sweep and
// not the chain of one.  A model's lanes cost the same whether a unit evicts or
// not, a plan's lane the more the fewer devices share the models: the more
// devices, the longer the windows that it wins.  us with a lane per model and
// with a lane per plan, 30,000 and 90,000 plans: D = 8, M = 8, N = 24 123 and 122, 273 and
// 261; N = 64 214 and 235, 521 and 551.  D = 14, M = 5, N = 40 149 and 148, 348 and 330;
// N = 64 196 and 203, 476 and 474.  D = 8, M = 12, N = 64 294 and 290, 750 and 698; N = 128
// 575 and 611, 1,549 and 1,516.  D = 16, M = 12, N = 128 571 and 574, 1,534 and 1,418.  4,000
// plans of D = 8, M = 12, N = 64: 82 and 93; 8,000: 121 and 103.  (All with about 20
// activations a session.)  Long sessions, whose chains keep to few models, evict
// less too: D = 3, M = 6, N = 64 in one session 166 and 164, 397 and 376, N = 80 in two
// 198 and 198, 487 and 465, but N = 64 in three 209 and 244, 505 and 571; M = 5,
// D = 3, N = 80 in two 480 and 462.  Up to four models four
// lanes a plan win from N = 24 on, and lose 2 % below.
//
// Beyond eight models lanes per model have registers for three CTAs an SM, a
// lane per plan for four: a batch that fills a fourth of each SM and no more
// is one wave instead of two.  8,500 plans of D = 8, M = 12, N = 163, 400, 1,000:
// 268, 593, 1,445 and 233, 541, 1,274; N = 2,000, of which shared memory holds three CTAs,
// 2,825 and 4,508.
// Returns the shared memory of such a CTA, 0 for a lane per model.
static size_t lane_per_plan(const wf_ctx *ctx, int64_t P)
{
    const wf_dev_problem &dp = ctx->dp;
    if (!dp.reclaim || dp.M <= 4 || P <= 40 * (int64_t)ctx->sms) return 0;
    const size_t smem = dp.phi_life ? pc_layout<kPlans32, uint32_t, kNuPlan, true>(dp.D, dp.M, dp.W, dp.nslots + 2).total
                                    : pc_layout<kPlans32, uint32_t, kNuPlan, false>(dp.D, dp.M, dp.W, dp.nslots + 2).total;
    const bool four = 4 * (smem + 1024) <= 228 * 1024;  // CTAs an SM
    const int64_t ctas = (P + kPlans32 - 1) / kPlans32;
    if (dp.M > 8 && four && ctas > 3 * (int64_t)ctx->sms && ctas <= 4 * (int64_t)ctx->sms) return smem;
    return dp.N <= (dp.M > 8 ? 32 + 8 * dp.D : dp.N >= 32 * dp.W ? 96 : 24 + 2 * dp.D) ? smem : 0;
}

int wf_launch_nextuse(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    const size_t smem = (size_t)kNuWarps * dp.D * dp.M * sizeof(uint16_t);
    const int64_t blocks = std::min<int64_t>((pl->P + kNuWarps - 1) / kNuWarps, (int64_t)ctx->sms * 16);
    const auto k = dp.N > kNuShort ? nextuse_kernel<true> : nextuse_kernel<false>;
    k<<<(unsigned)blocks, 32 * kNuWarps, smem, st>>>(dp, *pl, out->status, dp.nextuse);
    return wf_cuda_check(cudaGetLastError(), "next-use launch");
}

// Shared memory of a sweep CTA for this problem, its reclamation order and
// whether the window terms of Eq. 12 are wanted.
template <int kP, typename TT>
size_t layout_bytes(const wf_dev_problem &dp)
{
    const int32_t NS = dp.nslots + 2;
    if (sizeof(TT) == 8 && split40(dp))
        return dp.phi_life ? pc_layout<kP, TT, 0, true, Split40>(dp.D, dp.M, dp.W, NS).total
                           : pc_layout<kP, TT, 0, false, Split40>(dp.D, dp.M, dp.W, NS).total;
    if (dp.phi_life)
        return dp.reclaim ? pc_layout<kP, TT, 1, true>(dp.D, dp.M, dp.W, NS).total
                          : pc_layout<kP, TT, 0, true>(dp.D, dp.M, dp.W, NS).total;
    return dp.reclaim ? pc_layout<kP, TT, 1, false>(dp.D, dp.M, dp.W, NS).total
                      : pc_layout<kP, TT, 0, false>(dp.D, dp.M, dp.W, NS).total;
}

namespace {

// The shape choice depends on these fields of the problem only (and on the
// device, whose registers and shared memory bound the resident CTAs).
struct CfgKey {
    int dev;
    int32_t D, M, W, nslots;
    bool usable, split, reclaim, phi;
    bool operator==(const CfgKey &o) const
    {
        return dev == o.dev && D == o.D && M == o.M && W == o.W && nslots == o.nslots && usable == o.usable &&
               split == o.split && reclaim == o.reclaim && phi == o.phi;
    }
};

// The windows that take reclamation by next use, no more and no fewer: those of
// which three plans fit a CTA with a lane's state per plan and device (16-bit
// next uses, a queue word).  The state per model is up to 8 KB larger, so near
// that limit the 64-bit sweep plays two plans a CTA.
bool next_use_window(const wf_dev_problem &dp)
{
    const int32_t D = dp.D, M = dp.M;
    const size_t o = round16(4u * M) + round16(4u * D) + round16(4u * M * D) + round16(4u * dp.W) + 4608 + round16(24u * (dp.nslots + 2)) +
                     round16(24u * D) + round16((M <= 8 ? 12u : 24u) * D) + round16(12u * D) + round16(3u * D) + 32 +
                     round16(6u * D * M) + round16(3u * M) + 48 + (dp.phi_life ? round16(6u * D) : 0u);
    return o <= 227 * 1024;
}

wf_sweep_cfg choose(const wf_dev_problem &dp)
{
    wf_sweep_cfg c = {};
    if (!sweep_usable(dp) || (dp.reclaim && !next_use_window(dp))) return c;
    const size_t s32 = layout_bytes<kPlans32, uint32_t>(dp);
    c.res32 = resident<uint32_t>(dp, kPlans32, s32);
    if (c.res32 > 0) c.smem32 = s32;
    // The u64 sweep: 16, 6 or 3 plans per CTA, whichever keeps the most plans
    // resident per SM, registers and shared memory both counted.  Ties go to
    // the larger CTA, whose producer and residency warps serve more plans.
    const int shapes[3] = {16, 6, 3};
    int best = 0;
    for (int kp : shapes) {
        const size_t sm = kp == 16 ? layout_bytes<16, uint64_t>(dp)
                          : kp == 6 ? layout_bytes<6, uint64_t>(dp)
                                    : layout_bytes<3, uint64_t>(dp);
        const int n = resident<uint64_t>(dp, kp, sm);
        if (n > 0 && kp * n > best) {
            best = kp * n;
            c.smem64 = sm;
            c.plans64 = kp;
            c.res64 = n;
        }
    }
    if (!c.smem64 && dp.reclaim) {
        const size_t sm = layout_bytes<2, uint64_t>(dp);
        c.res64 = resident<uint64_t>(dp, 2, sm);
        if (c.res64 > 0) {
            c.smem64 = sm;
            c.plans64 = 2;
        }
    }
    // The relative-time sweep (for contexts whose plans leave 32 bits): 6 or
    // 16 plans per CTA, whichever keeps more plans resident per SM; ties go
    // to the smaller CTA, whose timing warp (the chain that paces the sweep)
    // has fewer plans to play (large window: 6-plan CTAs 72.7 ms, 8-plan CTAs
    // at the same 24 plans per SM 78.0 ms).
    if (c.smem64 && rel32(dp)) {
        const int rshapes[2] = {6, 16};
        int rbest = 0;
        for (int kp : rshapes) {
            const int32_t NS = dp.nslots + 2;
            const size_t sm = kp == 16 ? pc_layout<16, uint32_t, 0, false, Rel32>(dp.D, dp.M, dp.W, NS).total
                                       : pc_layout<6, uint32_t, 0, false, Rel32>(dp.D, dp.M, dp.W, NS).total;
            const int n = resident_rel(dp, kp, sm);
            if (n > 0 && kp * n > rbest) {
                rbest = kp * n;
                c.smemRel = sm;
                c.plansRel = kp;
                c.resRel = n;
            }
        }
    }
    return c;
}

}  // namespace

wf_sweep_cfg wf_sweep_config(const wf_dev_problem &dp)
{
    static std::mutex mu;
    static std::vector<std::pair<CfgKey, wf_sweep_cfg>> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return wf_sweep_cfg{};
    }
    const CfgKey key = {dev, dp.D, dp.M, dp.W, dp.nslots, sweep_usable(dp), split40(dp), dp.reclaim != 0,
                        dp.phi_life != 0};
    std::lock_guard<std::mutex> lock(mu);
    for (const auto &e : cache)
        if (e.first == key) return e.second;
    const wf_sweep_cfg c = choose(dp);
    if (cache.size() >= 64) cache.erase(cache.begin());
    cache.emplace_back(key, c);
    return c;
}

int wf_launch_sweep(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, const wf_sweep_cfg &cfg,
                    bool wide_first, int32_t *counts, int32_t *list1, int32_t *list2, cudaStream_t st,
                    const int32_t **rest_list, const int32_t **rest_count)
{
    // The next-use pass reads every plan's placement before the sweep, so
    // under that policy the status pass checks placement itself.
    int rc = wf_launch_status(ctx, pl, out, st, ctx->dp.reclaim != 0);
    if (!rc && ctx->dp.reclaim) rc = wf_launch_nextuse(ctx, pl, out, st);
    if (rc) return rc;
    const int64_t rblocks = wide_first && ctx->start_path != WF_PATH_WIDE ? rel_blocks(ctx, cfg, pl->P) : 0;
    if (rblocks > 0) {
        // Relative u32 times for every plan; the plans that leave 32 bits
        // even so go on to the u64 sweep.
        rc = launch_rel(ctx, cfg, rblocks, pl, out, list1, counts, st);
        if (!rc) rc = launch_pc_q<uint64_t>(ctx, cfg.plans64, cfg.res64, pl, out, cfg.smem64, list1, counts, list2,
                                            counts + 1, st);
    } else if (cfg.smem32 && !(wide_first && cfg.smem64)) {
        // u32 times for every plan; the plans that leave 32 bits go on to the
        // u64 sweep, and from there (or straight) to the int64 path.
        const wf_dev_problem &dp = ctx->dp;
        const size_t by_plan = lane_per_plan(ctx, pl->P);
        if (by_plan)
            rc = dp.phi_life ? launch_pc_r<uint32_t, kNuPlan, true>(ctx, kPlans32, 1, pl, out, by_plan, nullptr, nullptr, list1, counts, st)
                             : launch_pc_r<uint32_t, kNuPlan, false>(ctx, kPlans32, 1, pl, out, by_plan, nullptr, nullptr, list1, counts, st);
        else
            rc = launch_pc_q<uint32_t>(ctx, kPlans32, cfg.res32, pl, out, cfg.smem32, nullptr, nullptr, list1, counts, st);
        if (rc) return rc;
        if (!cfg.smem64) { *rest_list = list1; *rest_count = counts; return WF_OK; }
        rc = launch_pc_q<uint64_t>(ctx, cfg.plans64, cfg.res64, pl, out, cfg.smem64, list1, counts, list2, counts + 1, st);
    } else {
        rc = launch_pc_q<uint64_t>(ctx, cfg.plans64, cfg.res64, pl, out, cfg.smem64, nullptr, nullptr, list2, counts + 1, st);
    }
    *rest_list = list2;
    *rest_count = counts + 1;
    return rc;
}

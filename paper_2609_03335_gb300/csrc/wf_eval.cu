// Plan evaluation: status bits, then a list-schedule play of
// each plan over the window with fused chains (Eq. 3-4), releases (Eq. 2,
// Eq. 7), per-device order (Eq. 10), LRU residency under capacity (Eq. 11),
// loads / prefetches on the consumer's device (Eq. 5, Eq. 9), retain /
// reclaim and the metrics of Section 4.2-4.3.
//
// Mapping: a warp plays a deterministic plan (warp_play); for
// wf_eval_plans_phi it also returns the window terms of Eq. 12's ranking key
// (timely prefetches, lifecycle overhead).  One thread plays one (plan, sample)
// of a stochastic window, one plan under the replica batch limit, or one plan
// of a large batch of short windows on few devices: its
// mutable state (chain-tail finish times, per-device and per-session state)
// lives in a scratch row of the context, and plans beyond the number of rows
// are taken in rounds.
#include <algorithm>
#include <mutex>

#include "wf_play.cuh"

namespace {

constexpr int kEvalThreads = 128;
constexpr int kSampleThreads = 64;
constexpr int64_t kNone = INT64_MIN;

struct PlanRows {
    const uint8_t *place;
    const uint16_t *order;
    const uint32_t *fuse;
    const uint32_t *prefetch;
    const uint32_t *retain;  // NULL = all retained
};

__device__ __forceinline__ bool bit_at(const uint32_t *row, int32_t n)
{
    return (__ldg(row + (n >> 5)) >> (n & 31)) & 1u;
}

__device__ __forceinline__ PlanRows plan_rows(const wf_plans &pl, int64_t p)
{
    PlanRows r;
    r.place = pl.place + p * pl.place_stride;
    r.order = (const uint16_t *)((const uint8_t *)pl.order + p * pl.order_stride);
    r.fuse = (const uint32_t *)((const uint8_t *)pl.fuse + p * pl.bits_stride);
    r.prefetch = (const uint32_t *)((const uint8_t *)pl.prefetch + p * pl.bits_stride);
    r.retain = pl.retain ? (const uint32_t *)((const uint8_t *)pl.retain + p * pl.bits_stride) : nullptr;
    return r;
}

// Scratch row of one simulation.
struct Row {
    int64_t *ctail;   // [N] finish time of chain tails (also holds int32 positions for the status check)
    int64_t *tfree;   // [D] device free time
    int64_t *occ;     // [D] start of the current occupancy interval, kNone if empty
    int64_t *gpu;     // [D] closed occupancy
    int64_t *comp;    // [W] latest finish per session
    int32_t *used;    // [D] resident weights
    int32_t *nres;    // [D] resident model count
    int32_t *stamp;   // [D][M] last dispatch position + 1 using the model, 0 = not resident
    // With a replica batch limit B = dp.batch (only then laid out):
    int64_t *slot_end;  // [D][B] when each slot of the device's current replica frees
    int64_t *slot_kv;   // [D][B] KV need of the unit in each slot
    int64_t *last_adm;  // [D] the device's latest admission
    int32_t *cur;       // [D] model of the device's current replica, -1 for none
};

__device__ __forceinline__ size_t up8(size_t x) { return (x + 7) & ~(size_t)7; }

__device__ __forceinline__ Row row_at(const wf_dev_problem &dp, uint8_t *base)
{
    Row r;
    size_t o = 0;
    r.ctail = (int64_t *)(base + o); o += up8(8 * (size_t)dp.N);
    r.tfree = (int64_t *)(base + o); o += 8 * (size_t)dp.D;
    r.occ = (int64_t *)(base + o); o += 8 * (size_t)dp.D;
    r.gpu = (int64_t *)(base + o); o += 8 * (size_t)dp.D;
    r.comp = (int64_t *)(base + o); o += 8 * (size_t)dp.W;
    r.used = (int32_t *)(base + o); o += up8(4 * (size_t)dp.D);
    r.nres = (int32_t *)(base + o); o += up8(4 * (size_t)dp.D);
    r.stamp = (int32_t *)(base + o); o += up8(4 * (size_t)dp.D * dp.M);
    o += up8(4 * (size_t)dp.D);  // (spare: the row's size is part of the static entry point's contract)
    if (dp.batch > 0) {
        r.slot_end = (int64_t *)(base + o); o += 8 * (size_t)dp.D * dp.batch;
        r.slot_kv = (int64_t *)(base + o); o += 8 * (size_t)dp.D * dp.batch;
        r.last_adm = (int64_t *)(base + o); o += 8 * (size_t)dp.D;
        r.cur = (int32_t *)(base + o);
    } else {
        r.slot_end = r.slot_kv = r.last_adm = nullptr;
        r.cur = nullptr;
    }
    return r;
}

// Status bits (Eq. 8-10).  Uses the ctail area as an int32 position table.
__device__ uint32_t plan_status(const wf_dev_problem &dp, const PlanRows &pr, Row &row)
{
    const int32_t N = dp.N, D = dp.D;
    uint32_t st = 0;
    for (int32_t n = 0; n < N; ++n) {
        const int32_t d = pr.place[n];
        if (d >= D) st |= WF_ST_DEVICE;
        else if (dp.peak[(int64_t)n * D + d] > dp.cap[d]) st |= WF_ST_CAPACITY;
    }
    int32_t *pos = (int32_t *)row.ctail;
    for (int32_t n = 0; n < N; ++n) pos[n] = -1;
    for (int32_t i = 0; i < N; ++i) {
        const int32_t h = pr.order[i];
        if (h >= N || pos[h] >= 0) { st |= WF_ST_PERMUTATION; continue; }
        pos[h] = i;
    }
    if (!(st & WF_ST_PERMUTATION)) {
        for (int32_t v = 0; v < N && !(st & WF_ST_TOPOLOGY); ++v)
            for (int32_t e = dp.pred_off[v]; e < dp.pred_off[v + 1]; ++e)
                if (pos[dp.pred_idx[e]] > pos[v]) { st |= WF_ST_TOPOLOGY; break; }
    }
    return st;
}

// SplitMix64 output function (Steele, Lea, Flood 2014).
__device__ __forceinline__ uint64_t splitmix(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// Run time of activation n on device d; in a latency sample (kStoch) scaled by
// the multiplier drawn from (plan, sample, n) through the integer Box-Muller
// tables (an arithmetic right shift of the signed product is the floor).
template <bool kStoch>
__device__ __forceinline__ int64_t run_time(const wf_dev_problem &dp, int32_t n, int32_t d, uint64_t key)
{
    const int64_t base = dp.lat[(int64_t)n * dp.D + d];
    if (!kStoch) return base;
    const uint64_t h = splitmix(key ^ (uint64_t)n);
    const int64_t r = dp.bm_r[h & (uint64_t)(dp.bm_rn - 1)];
    const int64_t c = dp.bm_c[(h >> 32) & (uint64_t)(dp.bm_cn - 1)];
    const int64_t zq = (r * c) >> 18;
    const int64_t mult = dp.bm_e[zq + ((dp.bm_en - 1) >> 1)];
    return (base * mult + 32768) >> 16;
}

// One play of a valid plan (kStoch: for one latency sample) by one thread.
// Returns makespan, counted from dp.first_arrival, and GPU time; per-session
// completion latencies are left in row.comp.
template <bool kStoch>
__device__ void play(const wf_dev_problem &dp, const PlanRows &pr, Row &row, uint64_t key,
                     int64_t *makespan, int64_t *gpu_total)
{
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W;
    for (int32_t d = 0; d < D; ++d) {
        row.tfree[d] = 0; row.occ[d] = kNone; row.gpu[d] = 0; row.used[d] = 0; row.nres[d] = 0;
    }
    for (int32_t k = 0; k < D * M; ++k) row.stamp[k] = 0;
    for (int32_t w = 0; w < W; ++w) row.comp[w] = kNone;
    int64_t end = 0;

    for (int32_t i = 0; i < N; ++i) {
        const int32_t h = pr.order[i];
        const int32_t d = pr.place[h];
        // A chain member runs inside its head's unit (Eq. 3, Eq. 9).
        const int32_t fp = dp.fprev[h];
        if (fp >= 0 && bit_at(pr.fuse, h) && pr.place[fp] == d) continue;

        const int32_t m = dp.model[h];
        const int32_t w = dp.session[h];
        const int64_t arr = dp.arrival[w];
        int64_t rel = arr;  // Eq. 2 / Eq. 7: the heads' predecessors are chain tails
        for (int32_t e = dp.pred_off[h]; e < dp.pred_off[h + 1]; ++e)
            rel = max(rel, row.ctail[dp.pred_idx[e]]);

        // Extend the chain; admission KV is the largest on it, run time the sum (Eq. 4).
        const int32_t wm = dp.weight[m];
        int32_t tail = h;
        int64_t kv = dp.peak[(int64_t)h * D + d] - wm;
        int64_t run = run_time<kStoch>(dp, h, d, key);
        for (int32_t s = dp.fnext[h]; s >= 0 && bit_at(pr.fuse, s) && pr.place[s] == d; s = dp.fnext[s]) {
            kv = max(kv, (int64_t)dp.peak[(int64_t)s * D + d] - wm);
            run += run_time<kStoch>(dp, s, d, key);
            tail = s;
        }

        // Eq. 11 with LRU reclamation of other models.
        int32_t *st = row.stamp + d * M;
        const bool hit = st[m] != 0;
        const int64_t need = hit ? kv : wm + kv;
        while (row.used[d] + need > dp.cap[d]) {
            int32_t victim = -1, vs = INT32_MAX;
            for (int32_t k = 0; k < M; ++k)
                if (k != m && st[k] != 0 && st[k] < vs) { vs = st[k]; victim = k; }
            if (victim < 0) { atomicExch(dp.err, 2); break; }  // unreachable for a valid plan
            row.used[d] -= dp.weight[victim];
            row.nres[d] -= 1;
            st[victim] = 0;
        }
        const int64_t tf = row.tfree[d];
        int64_t start;
        if (hit) {
            start = max(tf, rel);
        } else {
            const int64_t ls = max(tf, bit_at(pr.prefetch, h) ? arr : rel);
            if (row.occ[d] == kNone) row.occ[d] = ls;
            row.used[d] += wm;
            row.nres[d] += 1;
            const int64_t le = ls + dp.load[m * D + d];
            start = max(le, rel);
        }
        const int64_t c = start + dp.grant + run;
        row.ctail[tail] = c;
        row.tfree[d] = c;
        st[m] = i + 1;
        end = max(end, c);
        row.comp[w] = max(row.comp[w], c);
        if (pr.retain && !bit_at(pr.retain, tail)) {
            row.used[d] -= wm;
            row.nres[d] -= 1;
            st[m] = 0;
            if (row.nres[d] == 0) {
                row.gpu[d] += c - row.occ[d];
                row.occ[d] = kNone;
            }
        }
    }
    int64_t g = 0;
    for (int32_t d = 0; d < D; ++d) {
        if (row.occ[d] != kNone) row.gpu[d] += end - row.occ[d];
        g += row.gpu[d];
    }
    for (int32_t w = 0; w < W; ++w) row.comp[w] -= dp.arrival[w];
    *makespan = end - dp.first_arrival;
    *gpu_total = g;
}

// One play with the replica batch limit B_q (Eq. 11 over every active unit,
// Section 3.5): a device runs units of one replica (a resident model) at a
// time, up to B = dp.batch of them at once.  Units are admitted in dispatch
// order.  A unit of the device's current replica takes the slot that frees
// earliest, no earlier than its release and the device's latest admission,
// once resident weights + the KV of the units still running + its own KV
// fit (idle least-recently-used models are reclaimed first; if that is not
// enough the unit waits for the next running unit to end).  A unit of
// another model waits for the device to drain and then hits or loads as
// without the limit; its other slots free when the model is ready.  B = 1
// gives the results without it.  Deterministic times; retain rows only with B = 1.
__device__ void play_batched(const wf_dev_problem &dp, const PlanRows &pr, Row &row, int64_t *makespan,
                             int64_t *gpu_total)
{
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W, B = dp.batch;
    for (int32_t d = 0; d < D; ++d) {
        row.occ[d] = kNone; row.gpu[d] = 0; row.used[d] = 0; row.nres[d] = 0;
        row.last_adm[d] = 0; row.cur[d] = -1;
        for (int32_t j = 0; j < B; ++j) { row.slot_end[d * B + j] = 0; row.slot_kv[d * B + j] = 0; }
    }
    for (int32_t k = 0; k < D * M; ++k) row.stamp[k] = 0;
    for (int32_t w = 0; w < W; ++w) row.comp[w] = kNone;
    int64_t end = 0;

    for (int32_t i = 0; i < N; ++i) {
        const int32_t h = pr.order[i];
        const int32_t d = pr.place[h];
        const int32_t fp = dp.fprev[h];
        if (fp >= 0 && bit_at(pr.fuse, h) && pr.place[fp] == d) continue;  // inside its head's unit
        const int32_t m = dp.model[h];
        const int32_t w = dp.session[h];
        const int64_t arr = dp.arrival[w];
        int64_t rel = arr;
        for (int32_t e = dp.pred_off[h]; e < dp.pred_off[h + 1]; ++e)
            rel = max(rel, row.ctail[dp.pred_idx[e]]);
        const int32_t wm = dp.weight[m];
        int32_t tail = h;
        int64_t kv = dp.peak[(int64_t)h * D + d] - wm;
        int64_t run = dp.lat[(int64_t)h * D + d];
        for (int32_t s = dp.fnext[h]; s >= 0 && bit_at(pr.fuse, s) && pr.place[s] == d; s = dp.fnext[s]) {
            kv = max(kv, (int64_t)dp.peak[(int64_t)s * D + d] - wm);
            run += dp.lat[(int64_t)s * D + d];
            tail = s;
        }
        int32_t *st = row.stamp + d * M;
        int64_t *se = row.slot_end + d * B, *sk = row.slot_kv + d * B;
        const int64_t cap = dp.cap[d];
        int64_t adm, start;
        int32_t slot = 0;
        if (m == row.cur[d]) {
            // Join the current replica (Eq. 11 with the running units' KV).
            for (int32_t j = 1; j < B; ++j)
                if (se[j] < se[slot]) slot = j;
            adm = max(max(rel, se[slot]), row.last_adm[d]);
            for (;;) {
                int64_t running = 0;
                for (int32_t j = 0; j < B; ++j) running += se[j] > adm ? sk[j] : 0;
                while (row.used[d] + running + kv > cap) {  // idle models, least recently used first
                    int32_t victim = -1, vs = INT32_MAX;
                    for (int32_t k = 0; k < M; ++k)
                        if (k != m && st[k] != 0 && st[k] < vs) { vs = st[k]; victim = k; }
                    if (victim < 0) break;
                    row.used[d] -= dp.weight[victim];
                    row.nres[d] -= 1;
                    st[victim] = 0;
                }
                if (row.used[d] + running + kv <= cap) break;
                int64_t next = kNone;  // the next running unit to end
                for (int32_t j = 0; j < B; ++j)
                    if (se[j] > adm && (next == kNone || se[j] < next)) next = se[j];
                if (next == kNone) { atomicExch(dp.err, 2); break; }  // unreachable for a valid plan
                adm = next;
            }
            start = adm;
        } else {
            // Another model: the device drains, then the unit hits or loads.
            int64_t drain = 0;
            for (int32_t j = 0; j < B; ++j) drain = max(drain, se[j]);
            const bool hit = st[m] != 0;
            const int64_t need = hit ? kv : wm + kv;
            while (row.used[d] + need > cap) {
                int32_t victim = -1, vs = INT32_MAX;
                for (int32_t k = 0; k < M; ++k)
                    if (k != m && st[k] != 0 && st[k] < vs) { vs = st[k]; victim = k; }
                if (victim < 0) { atomicExch(dp.err, 2); break; }  // unreachable for a valid plan
                row.used[d] -= dp.weight[victim];
                row.nres[d] -= 1;
                st[victim] = 0;
            }
            int64_t ready;
            if (hit) {
                adm = start = max(drain, rel);
                ready = drain;
            } else {
                const int64_t ls = max(drain, bit_at(pr.prefetch, h) ? arr : rel);
                if (row.occ[d] == kNone) row.occ[d] = ls;
                row.used[d] += wm;
                row.nres[d] += 1;
                const int64_t le = ls + dp.load[m * D + d];
                adm = ls;
                start = max(le, rel);
                ready = le;
            }
            for (int32_t j = 0; j < B; ++j) { se[j] = ready; sk[j] = 0; }
            row.cur[d] = m;
        }
        const int64_t c = start + dp.grant + run;
        row.ctail[tail] = c;
        se[slot] = c;
        sk[slot] = kv;
        row.last_adm[d] = adm;
        st[m] = i + 1;
        end = max(end, c);
        row.comp[w] = max(row.comp[w], c);
        if (pr.retain && !bit_at(pr.retain, tail)) {  // B = 1 only
            row.used[d] -= wm;
            row.nres[d] -= 1;
            st[m] = 0;
            row.cur[d] = -1;
            if (row.nres[d] == 0) {
                row.gpu[d] += c - row.occ[d];
                row.occ[d] = kNone;
            }
        }
    }
    int64_t g = 0;
    for (int32_t d = 0; d < D; ++d) {
        if (row.occ[d] != kNone) row.gpu[d] += end - row.occ[d];
        g += row.gpu[d];
    }
    for (int32_t w = 0; w < W; ++w) row.comp[w] -= dp.arrival[w];
    *makespan = end - dp.first_arrival;
    *gpu_total = g;
}

// r-th smallest (0-based) of v[0..n), reordering v (Hoare quickselect).
__device__ int64_t select_rank(int64_t *v, int32_t n, int32_t r)
{
    int32_t lo = 0, hi = n - 1;
    while (lo < hi) {
        const int64_t pivot = v[lo + (hi - lo) / 2];
        int32_t i = lo, j = hi;
        while (i <= j) {
            while (v[i] < pivot) ++i;
            while (v[j] > pivot) --j;
            if (i <= j) { int64_t t = v[i]; v[i] = v[j]; v[j] = t; ++i; --j; }
        }
        if (r <= j) hi = j;
        else if (r >= i) lo = i;
        else return v[r];
    }
    return v[r];
}

__device__ __forceinline__ int32_t p95_rank(int64_t n) { return (int32_t)((95 * n + 99) / 100 - 1); }

// ---------------------------------------------------------------------------
// A deterministic plan by one warp.  32 dispatch positions at a time:
//   A  lane = position: the unit that starts there (Eq. 3-4 chain, its
//      predecessors, session and arrival), all gathers of a chunk in flight
//      together;
//   B  lane = device: residency of the chunk's units in dispatch order
//      (Eq. 11), the device's queue, weights and count in registers -- the
//      devices' units are settled side by side;
//   C  the units one after the other, each by its own position's lane, whose
//      registers hold the record: releases, loads, starts and finishes (Eq.
//      2, 5, 7, 10) through finish times and device free times in shared
//      memory.
// Step C is the serial chain that bounds a plan; the SM hides it behind the
// other plans' warps.  Times are TT: u64 on the int64 path; the static entry
// point plays u32 first, with half the memory and a third of the instructions
// per maximum, and again on u64 only the plans that leave 32 bits.  1,900
// plans of N = 2,000 in wf_eval_plans_static: 14.2 ms with a thread per plan
// and its state in global memory, 0.81 ms with a warp per plan on 64-bit
// times, 0.57 ms on u32 times, 0.53 ms with the devices' state in one word
// each (73 warp instructions per plan-position; 93 on 64-bit times).
// ---------------------------------------------------------------------------

// The warp's working memory: B's answers for C [32], the models' weights [16],
// device free times [D], finish times of unit tails [N] and one more entry
// that stays 0 (the predecessor of a node without one), and the sessions' last
// finishes [W].  Times count from 1, so that 0 is none yet.
template <typename TT>
struct WarpMem {
    uint2 *res;
    int32_t *weight;
    TT *tfree, *ctail, *comp;
};

constexpr size_t kWarpHead = 32 * sizeof(uint2) + 16 * sizeof(int32_t);
__host__ __device__ inline size_t warp_small_bytes(int32_t D) { return kWarpHead + 8 * (size_t)D; }
template <typename TT>
__host__ __device__ inline size_t warp_full_bytes(const wf_dev_problem &dp)
{
    return warp_small_bytes(dp.D) + sizeof(TT) * ((size_t)dp.N + 1 + (size_t)dp.W);
}

// big: the finish and session times, behind the small part in shared memory
// or in a row of global scratch.
template <typename TT>
__device__ __forceinline__ WarpMem<TT> warp_mem(const wf_dev_problem &dp, uint8_t *sm, uint8_t *big)
{
    WarpMem<TT> w;
    w.res = (uint2 *)sm;
    w.weight = (int32_t *)(sm + 32 * sizeof(uint2));
    w.tfree = (TT *)(sm + kWarpHead);
    w.ctail = (TT *)big;
    w.comp = w.ctail + dp.N + 1;
    return w;
}

// Status bits (Eq. 8-10) by a warp, as plan_status; pos: u16 [N].
__device__ uint32_t warp_status(const wf_dev_problem &dp, const PlanRows &pr, uint16_t *pos)
{
    const int lane = threadIdx.x & 31;
    const int32_t N = dp.N, D = dp.D;
    uint32_t st = 0;
#pragma unroll 4
    for (int32_t n = lane; n < N; n += 32) {
        const int32_t d = __ldg(pr.place + n);
        if (d >= D) st |= WF_ST_DEVICE;
        else if (__ldg(dp.peak + (int64_t)n * D + d) > __ldg(dp.cap + d)) st |= WF_ST_CAPACITY;
    }
#pragma unroll 4
    for (int32_t i = lane; i < N; i += 32) {
        const int32_t h = __ldg(pr.order + i);
        if (h < N) pos[h] = (uint16_t)i;
        else st |= WF_ST_PERMUTATION;
    }
    __syncwarp();
    // A repeated node leaves some position with another position's entry.
#pragma unroll 4
    for (int32_t i = lane; i < N; i += 32) {
        const int32_t h = __ldg(pr.order + i);
        if (h < N && pos[h] != (uint16_t)i) st |= WF_ST_PERMUTATION;
    }
    st = __reduce_or_sync(0xFFFFFFFFu, st);
    if (!(st & WF_ST_PERMUTATION)) {
#pragma unroll 4
        for (int32_t v = lane; v < N; v += 32) {
            const uint16_t pv = pos[v];
            const int32_t e1 = __ldg(dp.pred_off + v + 1);
            for (int32_t e = __ldg(dp.pred_off + v); e < e1; ++e)
                if (pos[__ldg(dp.pred_idx + e)] > pv) st |= WF_ST_TOPOLOGY;
        }
        st = __reduce_or_sync(0xFFFFFFFFu, st);
    }
    __syncwarp();  // pos shares memory with the finish times
    return st;
}

// The sessions' completion latencies as ordered unsigned values (sign bit
// flipped), for warp_select.
template <typename TT>
struct LatencyArr {
    const TT *comp;
    const int64_t *arrival;
    __device__ __forceinline__ uint64_t get(int32_t w) const
    {
        const uint64_t c = comp[w];
        return ((c ? c - 1 : (uint64_t)kNone) - (uint64_t)__ldg(arrival + w)) ^ (1ull << 63);
    }
};

__device__ __forceinline__ int64_t warp_sum(int64_t v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ uint64_t warp_max(uint64_t v)
{
    const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
    return ((uint64_t)hi << 32) | __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
}

struct PlayResult {
    int64_t mk, p95, gpu, timely, life;
};

// One play of a valid plan; every lane returns the results (mk still counts
// from 0, not from the first arrival).  kPhi adds the window terms of Eq. 12;
// Q is the residency queue's word; kShort walks step C over the lanes that
// start a unit instead of over all 32, unrolled.  With u32 times, false when some time
// leaves 32 bits (the results are then void).
template <typename TT, typename Q, bool kPhi, bool kShort>
__device__ bool warp_play(const wf_dev_problem &dp, const PlanRows &pr, const WarpMem<TT> &wm, PlayResult &r)
{
    constexpr bool kNarrow = sizeof(TT) == 4;
    const int lane = threadIdx.x & 31;
    const int32_t N = dp.N, D = dp.D, W = dp.W;
    for (int32_t w = lane; w < W; w += 32) wm.comp[w] = 0;
    for (int32_t d = lane; d < D; d += 32) wm.tfree[d] = 0;
    if (lane == 0) wm.ctail[N] = 0;
    if (lane < 16) wm.weight[lane] = lane < dp.M ? __ldg(dp.weight + lane) : 0;
    // The lane's device, and the models it ever held.
    DevState<Q> ds;
    ds.init(lane < D ? (uint32_t)__ldg(dp.cap + lane) : 0u);
    uint32_t ever = 0;
    int64_t gsum = 0, timely = 0, life = 0;
    bool ovf = false;
    __syncwarp();
    for (int32_t c0 = 0; c0 < N; c0 += 32) {
        // A: the unit that starts at this lane's position.
        const bool in = c0 + lane < N;
        const int32_t h = in ? __ldg(pr.order + c0 + lane) : 0;
        const int32_t d = __ldg(pr.place + h);
        const int32_t fp = __ldg(dp.fprev + h), fn = __ldg(dp.fnext + h);
        const int32_t m = __ldg(dp.model + h), w = __ldg(dp.session + h);
        const int32_t e0 = __ldg(dp.pred_off + h), np = __ldg(dp.pred_off + h + 1) - e0;
        const bool fused = bit_at(pr.fuse, h), pf = bit_at(pr.prefetch, h);
        const bool unit = in && !(fp >= 0 && fused && __ldg(pr.place + fp) == d);
        const int64_t arr64 = __ldg(dp.arrival + w);
        const int32_t wgt = __ldg(dp.weight + m);
        const int32_t p0 = np > 0 ? __ldg(dp.pred_idx + e0) : N, p1 = np > 1 ? __ldg(dp.pred_idx + e0 + 1) : N;
        int64_t run64 = (int64_t)dp.grant + __ldg(dp.lat + (int64_t)h * D + d);
        int32_t kv = __ldg(dp.peak + (int64_t)h * D + d) - wgt, tail = h;
        if (unit)
            for (int32_t s = fn; s >= 0 && bit_at(pr.fuse, s) && __ldg(pr.place + s) == d; s = __ldg(dp.fnext + s)) {
                run64 += __ldg(dp.lat + (int64_t)s * D + d);
                kv = max(kv, __ldg(dp.peak + (int64_t)s * D + d) - wgt);
                tail = s;
            }
        const TT arr = (TT)(arr64 + 1), run = (TT)run64;
        if (kNarrow) ovf |= unit && (((arr64 + 1) | run64) >> 32) != 0;
        const bool drop = unit && pr.retain && !bit_at(pr.retain, tail);
        const uint32_t w3 = (uint32_t)d | ((uint32_t)m << 5) | (pf ? kPrefetch : 0u) | (drop ? kDrop : 0u);
        // B: residency of the chunk's units on the lane's device.
        uint32_t mine = 0;
        for (int32_t dd = 0; dd < D; ++dd) {
            const uint32_t on = __ballot_sync(0xFFFFFFFFu, unit && d == dd);
            if (lane == dd) mine = on;
        }
        while (__any_sync(0xFFFFFFFFu, mine)) {
            const int k = mine ? __ffs((int)mine) - 1 : 0;
            const uint32_t r1 = __shfl_sync(0xFFFFFFFFu, (uint32_t)kv, k), r3 = __shfl_sync(0xFFFFFFFFu, w3, k);
            if (mine) {
                bool missed;
                uint2 x = ds.template settle<true>(r1, r3, wm.weight, dp.load, D, dp.err, missed);
                if (kPhi && missed) {  // a reload of a model this device held before: bit 31 of the load word
                    const uint32_t mk = (r3 >> 5) & 15u;
                    x.x |= ((ever >> mk) & 1u) << 31;
                    ever |= 1u << mk;
                }
                wm.res[k] = x;
                mine &= mine - 1;
            }
        }
        __syncwarp();
        // C: the units in turn, each by its own lane.
        const uint2 x = wm.res[lane];
        const TT ld = kPhi ? x.x & 0x7FFFFFFFu : x.x;
        const int turn = unit ? lane : 32;
        TT *const tfree = wm.tfree + d, *const done = wm.ctail + tail, *const comp = wm.comp + w;
        const TT *const pred0 = wm.ctail + p0, *const pred1 = wm.ctail + p1;
        const auto play_unit = [&](int k) {
            if (turn == k) {
                const TT tf = *tfree;
                TT rel = max(arr, max(*pred0, *pred1));  // Eq. 2, Eq. 7
                for (int32_t e = 2; e < np; ++e) rel = max(rel, wm.ctail[__ldg(dp.pred_idx + e0 + e)]);
                // (on a hit the load time is 0 and the prefetch bit cleared)
                const TT ls = max(tf, (x.y & kPrefetch) ? arr : rel), le = ls + ld;
                const TT start = max(le, rel), c = start + run;
                if (kNarrow) ovf |= le < ls || c < start;
                *done = c;
                *tfree = c;
                *comp = max(*comp, c);
                if (x.y & (kWasEmpty | kEmptied)) {
                    if (x.y & kWasEmpty) gsum -= (int64_t)ls;
                    if (x.y & kEmptied) gsum += (int64_t)c;
                }
                if (kPhi) {
                    timely += (x.y & kPrefetch) && ls < rel && le <= rel;
                    life += (int64_t)(start - max(tf, rel) + (x.x >> 31 ? ld : 0));
                }
            }
            __syncwarp();
        };
        if constexpr (kShort) {
#pragma unroll 1
            for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, unit); todo; todo &= todo - 1) play_unit(__ffs((int)todo) - 1);
        } else {
#pragma unroll 4
            for (int k = 0; k < 32; ++k) play_unit(k);
        }
        if (kNarrow && __any_sync(0xFFFFFFFFu, ovf)) return false;
    }
    const int64_t open = __popc(__ballot_sync(0xFFFFFFFFu, lane < D && ds.occupied()));  // devices occupied to the end
    const int64_t end = (int64_t)warp_max(lane < D ? wm.tfree[lane] : (TT)0);
    r.mk = end - 1;
    r.gpu = warp_sum(gsum) + open * end;
    r.timely = kPhi ? warp_sum(timely) : 0;
    r.life = kPhi ? warp_sum(life) : 0;
    const LatencyArr<TT> lat{wm.comp, dp.arrival};
    r.p95 = (int64_t)((W <= 32 ? warp_select<1>(lat, W, p95_rank(W)) : warp_select<8>(lat, W, p95_rank(W))) ^ (1ull << 63));
    __syncwarp();  // the memory is free for the next plan
    return true;
}

// Plan p's results, by lane 0 (r's makespan counted from 0; first: the first arrival).
__device__ __forceinline__ void put_result(const wf_dev_problem &dp, const wf_eval_out &out, int64_t p, uint32_t st,
                                           const PlayResult &r, int64_t first)
{
    if ((threadIdx.x & 31) != 0) return;
    out.status[p] = st;
    out.makespan_us[p] = st ? WF_INF64 : r.mk - first;
    out.p95_us[p] = st ? WF_INF64 : r.p95;
    out.gpu_us[p] = st ? WF_INF64 : r.gpu;
    if (dp.phi_life) {
        dp.phi_timely[p] = st ? WF_INF64 : r.timely;
        dp.phi_life[p] = st ? WF_INF64 : r.life;
    }
}

constexpr size_t kSmemMax = 227 * 1024;

// How the warps that play a plan each are launched.
//   kFour  four warps a CTA on 64 registers, so that 32 plans are resident on
//          an SM; step C only over the lanes that start a unit
//   kSolo  a warp a CTA, finish times in shared memory
//   kRows  a warp a CTA, finish times in a row of global scratch, which L2
//          holds for the most part
enum WarpShape { kFour, kSolo, kRows };
__host__ __device__ constexpr int warps_of(WarpShape s) { return s == kFour ? 4 : 1; }
constexpr int kSolo64 = 12, kSolo32 = 16;  // CTAs of kSolo that registers allow an SM, on u64 and on u32 times

// Shared memory of a warp.
template <typename TT>
__host__ __device__ inline size_t warp_bytes(const wf_dev_problem &dp, WarpShape s)
{
    return ((s == kRows ? warp_small_bytes(dp.D) : warp_full_bytes<TT>(dp)) + 15) & ~(size_t)15;
}

// The shape for P plans of a window whose warps take `bytes` each with finish
// times in shared memory; solo: the most CTAs of kSolo an SM holds.
//   kFour where 32 such warps fit an SM and there are more plans than kSolo
//   holds at once.  Short windows in large batches are bound by issue, a CTA of
//   one warp at a time leaves its registers' share of the SM idle: 40,000 plans of N =
//   14, D = 7, M = 12 in wf_eval_plans_static, us: a thread per plan 142, kSolo
//   153, kFour 101; 65,536 of N = 40 on the int64 path 319, 452, 314; 3,700 of
//   N = 1,000 in the static call 7,385, 535, 426.
//   kRows where shared memory holds fewer warps than registers do, once the
//   plans exceed those (and where it holds none).  On the int64 path, ms in
//   shared memory and in rows: N = 8,192, 256 plans 1.90 and 2.21, 4,096 plans 17.2 and
//   6.60; N = 20,000, 152 plans (one an SM) 4.46 and 4.62, 512 plans 17.1 and
//   4.75, 4,096 plans 119 and 12.6 (a thread per plan: 134).
WarpShape warp_shape(int sms, int64_t P, size_t bytes, int solo)
{
    if (bytes > kSmemMax) return kRows;
    if (32 * bytes <= kSmemMax && P > kSolo32 * (int64_t)sms) return kFour;
    const int64_t fit = (int64_t)(kSmemMax / bytes);
    return fit < solo && P > fit * sms ? kRows : kSolo;
}

// Whether large batches of short windows on few devices play with a thread per
// plan instead: a warp settles the devices' units side by side, and with up to
// four devices it mostly waits for one of them, while N and D that small keep
// a thread's row in L1 and L2.  60,000 plans in wf_eval_plans_static, us, a
// warp and a thread per plan: D = 2, N = 14 144 and 94, N = 39 270 and 175, N = 64
// 332 and 323, N = 100 367 and 427; D = 3, N = 39 223 and 186, N = 64 230 and 277; D = 4,
// N = 24 146 and 130, N = 39 184 and 214; D = 5, N = 14 102 and 106.  22,076 plans of D = 2,
// N = 39 about the same either way: a thread's chain is longer.  On 64-bit times
// (wide) a warp gains less: 60,000 plans of D = 4, N = 39 297 and 242.
bool thread_per_plan(const wf_dev_problem &dp, int sms, int64_t P, bool wide)
{
    return dp.D <= 4 && (int64_t)dp.N * dp.D <= (wide ? 160 : 120) && P > 160 * (int64_t)sms;
}

// Every plan of the batch, or (list) the plans whose times a sweep could not
// hold, on int64 times; a warp walks over plans.
template <typename Q, bool kPhi, WarpShape kShape>
__global__ void __launch_bounds__(32 * warps_of(kShape), kShape == kFour ? 8 : kSolo64)
eval_warp_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, uint8_t *scratch, size_t row_bytes,
                 const int32_t *list, const int32_t *count)
{
    extern __shared__ __align__(16) uint8_t esm[];
    constexpr int kW = warps_of(kShape);
    const int64_t n = list ? (int64_t)*count : pl.P, k0 = (int64_t)blockIdx.x * kW + (threadIdx.x >> 5);
    uint8_t *sm = esm + (threadIdx.x >> 5) * warp_bytes<uint64_t>(dp, kShape);
    uint8_t *big = kShape == kRows ? scratch + (size_t)k0 * row_bytes : sm + warp_small_bytes(dp.D);
    const WarpMem<uint64_t> wm = warp_mem<uint64_t>(dp, sm, big);
    for (int64_t k = k0; k < n; k += (int64_t)gridDim.x * kW) {
        const int64_t p = list ? (int64_t)list[k] : k;
        const PlanRows pr = plan_rows(pl, p);
        const uint32_t st = warp_status(dp, pr, (uint16_t *)big);
        PlayResult r = {};
        if (!st) warp_play<uint64_t, Q, kPhi, kShape == kFour>(dp, pr, wm, r);
        put_result(dp, out, p, st, r, dp.first_arrival);
    }
}

// A thread per plan on the int64 path, rows of global scratch; every plan, or
// the listed ones: the replica batch limit (kBatched), or thread_per_plan().
template <bool kBatched>
__global__ void __launch_bounds__(kEvalThreads)
eval_thread_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, uint8_t *scratch, size_t row_bytes,
                    int64_t rows, const int32_t *list, const int32_t *count)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n = list ? (int64_t)*count : pl.P;
    if (t >= rows || t >= n) return;
    Row row = row_at(dp, scratch + (size_t)t * row_bytes);
    for (int64_t k = t; k < n; k += rows) {
        const int64_t p = list ? (int64_t)list[k] : k;
        const PlanRows pr = plan_rows(pl, p);
        const uint32_t st = plan_status(dp, pr, row);
        out.status[p] = st;
        if (st) {
            out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
            continue;
        }
        int64_t mk, g;
        if (kBatched) play_batched(dp, pr, row, &mk, &g);
        else play<false>(dp, pr, row, 0, &mk, &g);
        out.makespan_us[p] = mk;
        out.gpu_us[p] = g;
        out.p95_us[p] = select_rank(row.comp, dp.W, p95_rank(dp.W));
    }
}

// Stochastic latencies: one CTA per plan, one thread per sample; the pooled
// S x W completions of the plan go to a per-CTA pool for the p95 selection.
__global__ void __launch_bounds__(kSampleThreads)
eval_stoch_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, uint8_t *scratch, size_t row_bytes,
                  int64_t *pool_base, int64_t ctas, const int32_t *list, const int32_t *list_len)
{
    __shared__ unsigned long long s_mk, s_gpu;
    __shared__ uint32_t s_status;
    __shared__ uint32_t s_hist[256];
    __shared__ uint64_t s_prefix;
    __shared__ int32_t s_rank;
    const int64_t cta = blockIdx.x;
    const int32_t S = dp.S, W = dp.W;
    Row row = row_at(dp, scratch + (size_t)(cta * blockDim.x + threadIdx.x) * row_bytes);
    int64_t *pool = pool_base + cta * (int64_t)S * W;
    // Every plan of the batch, or only those listed (plans whose times left
    // the 32-bit range of the shared-memory sweep).
    const int64_t total = list ? (int64_t)*list_len : pl.P;
    for (int64_t j = cta; j < total; j += ctas) {
        const int64_t p = list ? (int64_t)list[j] : j;
        const PlanRows pr = plan_rows(pl, p);
        if (threadIdx.x == 0) {
            s_mk = 0; s_gpu = 0;
            s_status = plan_status(dp, pr, row);
        }
        __syncthreads();
        const uint32_t st = s_status;
        if (st) {
            if (threadIdx.x == 0) {
                out.status[p] = st;
                out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
            }
            __syncthreads();
            continue;
        }
        const uint64_t gp = (uint64_t)(pl.plan_base + p);
        for (int32_t s = threadIdx.x; s < S; s += blockDim.x) {
            const uint64_t key = splitmix(splitmix(dp.seed ^ gp) ^ (uint64_t)s);
            int64_t mk, g;
            play<true>(dp, pr, row, key, &mk, &g);
            atomicAdd(&s_mk, (unsigned long long)mk);
            atomicAdd(&s_gpu, (unsigned long long)g);
            for (int32_t w = 0; w < W; ++w) pool[(int64_t)s * W + w] = row.comp[w];
        }
        __syncthreads();
        // Nearest-rank p95 of the pooled non-negative completions: radix
        // select, 8 bits per pass from the most significant byte.
        const int64_t n = (int64_t)S * W;
        if (threadIdx.x == 0) { s_prefix = 0; s_rank = p95_rank(n); }
        __syncthreads();
        for (int shift = 56; shift >= 0; shift -= 8) {
            for (int b = threadIdx.x; b < 256; b += blockDim.x) s_hist[b] = 0;
            __syncthreads();
            const uint64_t hi_mask = shift == 56 ? 0 : (~0ull << (shift + 8));
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
                const uint64_t v = (uint64_t)pool[i];
                if ((v & hi_mask) == s_prefix) atomicAdd(&s_hist[(v >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                int32_t r = s_rank;
                int b = 0;
                while ((int32_t)s_hist[b] <= r) { r -= s_hist[b]; ++b; }
                s_rank = r;
                s_prefix |= (uint64_t)b << shift;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            out.status[p] = 0;
            out.makespan_us[p] = (int64_t)(s_mk / (unsigned long long)S);
            out.gpu_us[p] = (int64_t)(s_gpu / (unsigned long long)S);
            out.p95_us[p] = (int64_t)s_prefix;
        }
        __syncthreads();
    }
}

}  // namespace

size_t wf_eval_row_bytes(const wf_dev_problem &dp)
{
    size_t b = ((8 * (size_t)dp.N + 7) & ~(size_t)7) + 8 * 3 * (size_t)dp.D + 8 * (size_t)dp.W +
               2 * ((4 * (size_t)dp.D + 7) & ~(size_t)7) + ((4 * (size_t)dp.D * dp.M + 7) & ~(size_t)7) +
               4 * (size_t)dp.D;
    if (dp.batch > 0) b += 4 + 16 * (size_t)dp.D * dp.batch + 12 * (size_t)dp.D;  // (4: padding after loaded)
    return (b + 127) & ~(size_t)127;
}

static size_t sample_cta_bytes(const wf_dev_problem &dp)
{
    const size_t pool = (8 * (size_t)dp.S * dp.W + 127) & ~(size_t)127;
    return kSampleThreads * wf_eval_row_bytes(dp) + pool;
}

size_t wf_eval_scratch_bytes(const wf_dev_problem &dp, int64_t max_P, int64_t *units)
{
    const size_t budget = (size_t)1 << 30;
    const size_t unit = dp.S == 0 ? wf_eval_row_bytes(dp) : sample_cta_bytes(dp);
    const int64_t floor_units = dp.S == 0 ? 1024 : 16;
    *units = std::min<int64_t>(max_P, std::max<int64_t>((int64_t)(budget / unit), floor_units));
    return unit * (size_t)*units;
}

namespace {

// The int64 path over every plan (list null) or the listed ones.
int launch_int64(wf_ctx *ctx, const wf_plans *plans, const wf_eval_out *out, const int32_t *list, const int32_t *count,
                 cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    uint8_t *scratch = (uint8_t *)ctx->eval_scratch;
    const int64_t units = std::min<int64_t>(ctx->eval_threads, plans->P);
    if (dp.batch > 0 || (!list && !dp.phi_life && thread_per_plan(dp, ctx->sms, plans->P, true))) {
        const int64_t blocks = (units + kEvalThreads - 1) / kEvalThreads;
        const auto kernel = dp.batch > 0 ? eval_thread_kernel<true> : eval_thread_kernel<false>;
        kernel<<<(unsigned)blocks, kEvalThreads, 0, st>>>(dp, *plans, *out, scratch, ctx->eval_row_bytes, units, list, count);
    } else {
        const size_t bytes = warp_bytes<uint64_t>(dp, kSolo);
        // A list is most often empty: few CTAs where that can be.
        const WarpShape shape = list && 32 * bytes <= kSmemMax ? kFour : warp_shape(ctx->sms, plans->P, bytes, kSolo64);
        const size_t smem = warps_of(shape) * warp_bytes<uint64_t>(dp, shape);
        const auto by_phi = [&](auto q, auto s) {
            using Q = typename decltype(q)::type;
            constexpr WarpShape kS = (WarpShape)decltype(s)::value;
            return dp.phi_life ? eval_warp_kernel<Q, true, kS> : eval_warp_kernel<Q, false, kS>;
        };
        const auto by_shape = [&](auto q) {
            return shape == kFour ? by_phi(q, Iv<kFour>{}) : shape == kSolo ? by_phi(q, Iv<kSolo>{}) : by_phi(q, Iv<kRows>{});
        };
        const auto kernel = dp.M <= 8 ? by_shape(Ty<uint32_t>{}) : by_shape(Ty<uint64_t>{});
        const int rc = wf_cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)smem), "int64 path smem attribute");
        if (rc) return rc;
        // A warp per plan, or for a list about as many as fit the chip at
        // once; with rows, a row per CTA.
        int64_t blocks = (plans->P + warps_of(shape) - 1) / warps_of(shape);
        if (list) blocks = std::min<int64_t>(blocks, (int64_t)ctx->sms * (kSolo64 / warps_of(shape)));
        if (shape == kRows) blocks = std::min<int64_t>(blocks, units);
        kernel<<<(unsigned)blocks, 32 * warps_of(shape), smem, st>>>(dp, *plans, *out, scratch, ctx->eval_row_bytes, list, count);
    }
    return wf_cuda_check(cudaGetLastError(), "int64 pass launch");
}

}  // namespace

int wf_launch_eval(wf_ctx *ctx, const wf_plans *plans, const wf_eval_out *out, cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    uint8_t *scratch = (uint8_t *)ctx->eval_scratch;
    const int64_t units = std::min<int64_t>(ctx->eval_threads, plans->P);
    if (dp.batch > 1 && plans->retain)
        return wf_set_error(WF_EINVAL, "retain rows are modelled with a replica batch limit of 1 only");
    if (dp.batch > 0 && dp.phi_life)
        return wf_set_error(WF_EINVAL, "the window terms of Eq. 12 are not modelled with a replica batch limit");
    if (dp.S == 0) {
        // The replica batch limit has a sweep of its own.  Windows that no
        // sweep holds play on the int64 path.
        wf_batch_cfg bcfg = {};
        wf_sweep_cfg cfg = {};
        if (!ctx->force_int64) {
            if (dp.batch > 0) bcfg = wf_batch_config(dp);
            else cfg = wf_sweep_config(dp);
        }
        const bool batch = bcfg.smem64 != 0;
        const bool narrow = batch || cfg.smem32, wide = batch || cfg.smem64;
        if (dp.reclaim && !cfg.smem64)
            return wf_set_error(WF_EINVAL, "reclamation by next use runs only in the shared-memory sweep");
        if (narrow || wide) {
            // Under stream capture (a CUDA graph) nothing but launches on the
            // stream may happen: the path choice stays as it is.
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            int rc0 = wf_cuda_check(cudaStreamIsCapturing(st, &cs), "stream capture status");
            if (rc0) return rc0;
            const bool capturing = cs != cudaStreamCaptureStatusNone;
            // Path choice: the u32 sweep's hand-off count of an earlier call,
            // if it has arrived (never waited for).
            if (ctx->wide_pending && !capturing) {
                const cudaError_t q = cudaEventQuery(ctx->ovf_event);
                if (q == cudaSuccess) {
                    ctx->prefer_wide = 2 * (int64_t)*ctx->h_ovf > ctx->wide_P;
                    ctx->wide_pending = false;
                } else if (q == cudaErrorNotReady) {
                    (void)cudaGetLastError();
                } else {
                    return wf_cuda_check(q, "overflow count event");
                }
            }
            const bool wide_first = (ctx->prefer_wide || ctx->start_path >= WF_PATH_WIDE) && wide;
            // Two pairs of counts, taken by calls in turn, so that a call
            // issued before an earlier call's read-back has run does not
            // reset the count it reads; a call that comes back to a pair
            // whose read-back is still pending waits for that copy first.
            const int q = capturing ? ctx->ovf_pair : (ctx->ovf_pair ^= 1);
            int32_t *counts = ctx->ovf_count + 2 * q;
            int rc = WF_OK;
            if (!capturing && ctx->wide_pending && ctx->rb_pair == q)
                rc = wf_cuda_check(cudaStreamWaitEvent(st, ctx->ovf_event, 0), "overflow read-back wait");
            if (!rc) rc = wf_cuda_check(cudaMemsetAsync(counts, 0, 2 * sizeof(int32_t), st), "reset overflow counts");
            const int32_t *rest = nullptr, *rest_count = nullptr;
            if (!rc)
                rc = batch ? wf_launch_batch(ctx, plans, out, bcfg, wide_first, counts, ctx->ovf_list, ctx->ovf_list2, st,
                                             &rest, &rest_count)
                           : wf_launch_sweep(ctx, plans, out, cfg, wide_first, counts, ctx->ovf_list, ctx->ovf_list2, st,
                                             &rest, &rest_count);
            if (rc) return rc;
            if (narrow && !wide_first && !ctx->wide_pending && !capturing) {
                // The read-back runs on the context's side stream after the
                // sweeps, so the caller's stream never waits for it; the
                // value only picks the path, never a result.
                rc = wf_cuda_check(cudaEventRecord(ctx->sweep_done, st), "sweep event");
                if (!rc) rc = wf_cuda_check(cudaStreamWaitEvent(ctx->side, ctx->sweep_done, 0), "side stream wait");
                if (!rc) rc = wf_cuda_check(cudaMemcpyAsync(ctx->h_ovf, counts, sizeof(int32_t),
                                                            cudaMemcpyDeviceToHost, ctx->side),
                                            "overflow count read-back");
                if (!rc) rc = wf_cuda_check(cudaEventRecord(ctx->ovf_event, ctx->side), "overflow count event");
                if (rc) return rc;
                ctx->wide_pending = true;
                ctx->wide_P = plans->P;
                ctx->rb_pair = q;
            }
            return launch_int64(ctx, plans, out, rest, rest_count, st);
        }
        return launch_int64(ctx, plans, out, nullptr, nullptr, st);
    } else {
        // Per-thread rows of every CTA first, then one completion pool per CTA.
        int64_t *pool = (int64_t *)(scratch + (size_t)units * kSampleThreads * ctx->eval_row_bytes);
        if (!ctx->force_int64 && wf_stoch_usable(dp)) {
            int rc = wf_cuda_check(cudaMemsetAsync(ctx->ovf_count, 0, sizeof(int32_t), st), "reset overflow count");
            if (!rc) rc = wf_launch_stoch(ctx, plans, out, ctx->ovf_list, ctx->ovf_count, st);
            if (rc) return rc;
            const int64_t lunits = std::min<int64_t>(units, (int64_t)ctx->sms * 4);
            eval_stoch_kernel<<<(unsigned)lunits, kSampleThreads, 0, st>>>(dp, *plans, *out, scratch,
                                                                           ctx->eval_row_bytes, pool, lunits,
                                                                           ctx->ovf_list, ctx->ovf_count);
        } else {
            eval_stoch_kernel<<<(unsigned)units, kSampleThreads, 0, st>>>(dp, *plans, *out, scratch,
                                                                          ctx->eval_row_bytes, pool, units,
                                                                          nullptr, nullptr);
        }
    }
    return wf_cuda_check(cudaGetLastError(), "eval launch");
}

// ---------------------------------------------------------------------------
// Allocation-free entry point: wf_eval_plans_static.
//
// Some callers cannot allocate device memory when they want to score plans:
// a scheduler that runs inside a serving engine which reserved nearly all of
// the GPU's memory up front for model weights and KV cache (an extra
// cudaMalloc there fails, or takes memory the engine's cache counts on), or a
// process whose device memory belongs to another allocator that must not be
// bypassed.  For them this entry point evaluates a deterministic batch with
// no context and no allocation: the caller passes the problem tables, the
// plans and the outputs as device pointers, and every piece of scratch lives
// in the file-scope array below, which each GPU that loads this library holds
// until the process exits.
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kStaticScratchBytes = (size_t)32 << 20;  // 32 MiB
constexpr size_t kStaticHeader = 256;                     // first arrival, error word

static __device__ __align__(256) uint8_t g_static_scratch[kStaticScratchBytes];

__host__ __device__ __forceinline__ size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Layout: header | succ count [N] | fusible successor [N] | fusible predecessor [N] | rows [P]
struct StaticLayout {
    size_t nsucc, fnext, fprev, rows, total;
};

__host__ __device__ __forceinline__ StaticLayout static_layout(int32_t N, int64_t P, size_t row)
{
    StaticLayout l;
    l.nsucc = kStaticHeader;
    l.fnext = l.nsucc + up256(4 * (size_t)N);
    l.fprev = l.fnext + up256(4 * (size_t)N);
    l.rows = l.fprev + up256(4 * (size_t)N);
    l.total = l.rows + (size_t)P * row;
    return l;
}

// Error word of the static array (header offset 8): 0, or kStaticBadTables
// when the problem tables failed the device check (bits 8.. name the first
// check that failed), or the evaluation's own error codes.
constexpr int kStaticBadTables = 4;

// Everything the derived tables start from: zero successor counts, no links,
// the first arrival at +infinity, a clear error word.
__global__ void static_init_kernel(uint8_t *s, int32_t N, StaticLayout l)
{
    const int32_t n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n == 0) {
        *(int64_t *)s = WF_INF64;
        *(int *)(s + 8) = 0;
    }
    if (n < N) {
        ((int32_t *)(s + l.nsucc))[n] = 0;
        ((int32_t *)(s + l.fnext))[n] = -1;
        ((int32_t *)(s + l.fprev))[n] = -1;
    }
}

// The device check of the caller's tables (one thread per node, model,
// device, session and (model, device) pair), before any of them indexes
// another table.  A failure sets the error word; the kernels after it then
// index nothing.
__global__ void static_check_kernel(uint8_t *s, wf_dev_problem dp)
{
    const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W;
    int bad = 0;
    if (v < N) {
        const int32_t a = dp.pred_off[v], b = dp.pred_off[v + 1];
        if ((v == 0 && a != 0) || b < a) bad = 1;
        else
            for (int32_t e = a; e < b; ++e) {
                const int32_t u = dp.pred_idx[e];
                if (u < 0 || u >= N || u == v) { bad = 2; break; }
            }
        const uint32_t m = dp.model[v];
        const int32_t w = dp.session[v];
        if (m >= (uint32_t)M) bad = 3;
        else if (w < 0 || w >= W) bad = 4;
        else
            for (int32_t d = 0; d < D; ++d)
                if (dp.lat[(int64_t)v * D + d] < 0 || dp.peak[(int64_t)v * D + d] < dp.weight[m]) { bad = 5; break; }
    }
    if (v < M && dp.weight[v] < 1) bad = 6;
    if (v < D && dp.cap[v] < 1) bad = 7;
    if (v < M * D && dp.load[v] < 0) bad = 8;
    if (v < W && dp.arrival[v] < 0) bad = 9;
    if (bad) atomicCAS((int *)(s + 8), 0, kStaticBadTables | (bad << 8));
}

__global__ void static_count_kernel(uint8_t *s, wf_dev_problem dp, StaticLayout l)
{
    if (*(volatile int *)(s + 8)) return;  // the tables failed the check
    const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < dp.W) atomicMin((long long *)s, (long long)dp.arrival[v]);
    if (v >= dp.N) return;
    int32_t *nsucc = (int32_t *)(s + l.nsucc);
    for (int32_t e = dp.pred_off[v]; e < dp.pred_off[v + 1]; ++e) atomicAdd(&nsucc[dp.pred_idx[e]], 1);
}

// Eq. 3: (u, v) fusible iff succ(u) = {v}, pred(v) = {u}, same model.
__global__ void static_link_kernel(uint8_t *s, wf_dev_problem dp, StaticLayout l)
{
    if (*(volatile int *)(s + 8)) return;  // the tables failed the check
    const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= dp.N || dp.pred_off[v + 1] - dp.pred_off[v] != 1) return;
    const int32_t u = dp.pred_idx[dp.pred_off[v]];
    if (((const int32_t *)(s + l.nsucc))[u] == 1 && dp.model[u] == dp.model[v]) {
        ((int32_t *)(s + l.fnext))[u] = v;
        ((int32_t *)(s + l.fprev))[v] = u;
    }
}

// The deterministic evaluation, a warp per plan, with the first
// arrival taken from the static header: on u32 times in shared memory, and
// on u64 times in the plan's scratch row when those do not hold the plan or
// the window does not fit (kRows).
template <typename Q, WarpShape kShape>
__global__ void __launch_bounds__(32 * warps_of(kShape), kShape == kFour ? 8 : kSolo32)
eval_static_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, uint8_t *s, StaticLayout l,
                   size_t row_bytes)
{
    extern __shared__ __align__(16) uint8_t esm[];
    const int64_t p = (int64_t)blockIdx.x * warps_of(kShape) + (threadIdx.x >> 5);
    if (p >= pl.P) return;  // the whole warp
    if ((*(volatile int *)(s + 8) & 0xFF) == kStaticBadTables) {  // nothing is evaluated
        if ((threadIdx.x & 31) == 0) {
            out.status[p] = WF_ST_TABLES;
            out.makespan_us[p] = out.p95_us[p] = out.gpu_us[p] = WF_INF64;
        }
        return;
    }
    uint8_t *sm = esm + (threadIdx.x >> 5) * warp_bytes<uint32_t>(dp, kShape);
    uint8_t *row = s + l.rows + (size_t)p * row_bytes, *big = kShape == kRows ? row : sm + warp_small_bytes(dp.D);
    const PlanRows pr = plan_rows(pl, p);
    const uint32_t st = warp_status(dp, pr, (uint16_t *)big);
    PlayResult r = {};
    constexpr bool kShort = kShape == kFour;
    if (!st && !(kShape != kRows && warp_play<uint32_t, Q, false, kShort>(dp, pr, warp_mem<uint32_t>(dp, sm, big), r)))
        warp_play<uint64_t, Q, false, kShort>(dp, pr, warp_mem<uint64_t>(dp, sm, row), r);
    put_result(dp, out, p, st, r, *(const int64_t *)s);
}

// The same with a thread per plan (thread_per_plan), in the plan's scratch row.
__global__ void __launch_bounds__(kEvalThreads)
eval_static_thread_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, uint8_t *s, StaticLayout l, size_t row_bytes)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= pl.P) return;
    uint32_t st = WF_ST_TABLES;
    int64_t mk = WF_INF64, p95 = WF_INF64, g = WF_INF64;
    if ((*(volatile int *)(s + 8) & 0xFF) != kStaticBadTables) {  // (else nothing is evaluated)
        wf_dev_problem d = dp;
        d.first_arrival = *(const int64_t *)s;
        Row row = row_at(d, s + l.rows + (size_t)p * row_bytes);
        const PlanRows pr = plan_rows(pl, p);
        st = plan_status(d, pr, row);
        if (!st) {
            play<false>(d, pr, row, 0, &mk, &g);
            p95 = select_rank(row.comp, d.W, p95_rank(d.W));
        }
    }
    out.status[p] = st;
    out.makespan_us[p] = mk;
    out.p95_us[p] = p95;
    out.gpu_us[p] = g;
}

// Device address of the static array per device, from the last lookup
// outside stream capture.
uint8_t *g_static_addr[64];
bool g_static_ready[64];
std::mutex g_static_mu;

}  // namespace

extern "C" int wf_eval_plans_static(const wf_problem *pb, const wf_plans *pl, const wf_eval_out *out,
                                    void *stream)
{
    if (!pb || !pl || !out) return wf_set_error(WF_EINVAL, "NULL argument");
    const int32_t N = pb->N, D = pb->D, M = pb->M, W = pb->W;
    if (N < 1 || N > 65535 || D < 1 || D > 32 || M < 1 || M > 16 || W < 1)
        return wf_set_error(WF_EINVAL, "sizes outside N 1..65535, D 1..32, M 1..16, W >= 1");
    if (pb->S != 0) return wf_set_error(WF_EINVAL, "wf_eval_plans_static evaluates deterministic problems (S = 0) only");
    if (pb->margin_mib != 0)
        return wf_set_error(WF_EINVAL, "wf_eval_plans_static takes no admission margin (fold it into peak_mib)");
    if (!pb->pred_off || !pb->model || !pb->session || !pb->arrival_us || !pb->lat_us || !pb->peak_mib ||
        !pb->weight_mib || !pb->load_us || !pb->cap_mib || pb->grant_us < 0)
        return wf_set_error(WF_EINVAL, "a problem table pointer is NULL or grant_us < 0");
    if (pl->P < 1 || !pl->place || !pl->order || !pl->fuse || !pl->prefetch || pl->plan_base < 0)
        return wf_set_error(WF_EINVAL, "empty batch or NULL plan array");
    if (!out->makespan_us || !out->p95_us || !out->gpu_us || !out->status)
        return wf_set_error(WF_EINVAL, "NULL output array");
    const int64_t words = ((int64_t)N + 31) / 32;
    if (pl->place_stride < N || pl->place_stride % 16 || pl->order_stride < 2 * (int64_t)N ||
        pl->order_stride % 16 || pl->bits_stride < 4 * words || pl->bits_stride % 16)
        return wf_set_error(WF_EINVAL, "plan strides must be multiples of 16 covering N");
    const uintptr_t mis = (uintptr_t)pl->place | (uintptr_t)pl->order | (uintptr_t)pl->fuse |
                          (uintptr_t)pl->prefetch | (uintptr_t)pl->retain;
    if (mis & 15u) return wf_set_error(WF_EINVAL, "plan arrays must be 16-byte aligned");

    wf_dev_problem dp = {};
    dp.N = N; dp.D = D; dp.M = M; dp.W = W;
    dp.grant = pb->grant_us;
    dp.pred_off = pb->pred_off;
    dp.pred_idx = pb->pred_idx;
    dp.model = pb->model;
    dp.session = pb->session;
    dp.arrival = pb->arrival_us;
    dp.lat = pb->lat_us;
    dp.peak = pb->peak_mib;
    dp.weight = pb->weight_mib;
    dp.load = pb->load_us;
    dp.cap = pb->cap_mib;
    const size_t row = wf_eval_row_bytes(dp);
    const StaticLayout l = static_layout(N, pl->P, row);
    if (l.total > kStaticScratchBytes) {
        const int64_t fit = (int64_t)((kStaticScratchBytes - l.rows) / row);
        return wf_set_error(WF_EINVAL,
                            "batch needs %zu bytes of scratch but the static array holds %zu; at most "
                            "%lld plans of this window per call", l.total, kStaticScratchBytes,
                            (long long)fit);
    }

    int dev = 0;
    int rc = wf_cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
    if (rc) return rc;
    if (dev < 0 || dev >= 64) return wf_set_error(WF_EINVAL, "device ordinal %d >= 64", dev);
    cudaStream_t st = (cudaStream_t)stream;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    rc = wf_cuda_check(cudaStreamIsCapturing(st, &cs), "stream capture status");
    if (rc) return rc;
    uint8_t *s = nullptr;
    {
        // Outside capture the address is looked up with the current device
        // (valid in the current context, also after a device reset); under
        // capture the last such lookup on this device is reused.
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (cs == cudaStreamCaptureStatusNone) {
            void *p = nullptr;
            rc = wf_cuda_check(cudaGetSymbolAddress(&p, g_static_scratch), "cudaGetSymbolAddress");
            if (rc) return rc;
            g_static_addr[dev] = (uint8_t *)p;
            g_static_ready[dev] = true;
        } else if (!g_static_ready[dev]) {
            return wf_set_error(WF_EINVAL, "the first wf_eval_plans_static call on a device must not be captured");
        }
        s = g_static_addr[dev];
    }
    dp.fnext = (const int32_t *)(s + l.fnext);
    dp.fprev = (const int32_t *)(s + l.fprev);
    dp.err = (int *)(s + 8);

    const int32_t span = std::max(N, W);
    const unsigned grid = (unsigned)((span + 255) / 256);
    const int32_t cspan = std::max(span, M * D);
    static_init_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(s, N, l);
    static_check_kernel<<<(unsigned)((cspan + 255) / 256), 256, 0, st>>>(s, dp);
    static_count_kernel<<<grid, 256, 0, st>>>(s, dp, l);
    static_link_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(s, dp, l);
    int sms = 0;
    rc = wf_cuda_check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
    if (rc) return rc;
    if (thread_per_plan(dp, sms, pl->P, false)) {
        eval_static_thread_kernel<<<(unsigned)((pl->P + kEvalThreads - 1) / kEvalThreads), kEvalThreads, 0, st>>>(
            dp, *pl, *out, s, l, row);
        return wf_cuda_check(cudaGetLastError(), "static evaluation launch");
    }
    const WarpShape shape = warp_shape(sms, pl->P, warp_bytes<uint32_t>(dp, kSolo), kSolo32);
    const size_t smem = warps_of(shape) * warp_bytes<uint32_t>(dp, shape);
    const auto by_shape = [&](auto q) {
        using Q = typename decltype(q)::type;
        return shape == kFour ? eval_static_kernel<Q, kFour> : shape == kSolo ? eval_static_kernel<Q, kSolo> : eval_static_kernel<Q, kRows>;
    };
    const auto kernel = M <= 8 ? by_shape(Ty<uint32_t>{}) : by_shape(Ty<uint64_t>{});
    rc = wf_cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                       "static evaluation smem attribute");
    if (rc) return rc;
    const unsigned blocks = (unsigned)((pl->P + warps_of(shape) - 1) / warps_of(shape));
    kernel<<<blocks, 32 * warps_of(shape), smem, st>>>(dp, *pl, *out, s, l, row);
    return wf_cuda_check(cudaGetLastError(), "static evaluation launch");
}

extern "C" int wf_static_status(void *stream)
{
    int rc = wf_cuda_check(cudaStreamSynchronize((cudaStream_t)stream), "cudaStreamSynchronize");
    if (rc) return rc;
    int err = 0;
    rc = wf_cuda_check(cudaMemcpyFromSymbol(&err, g_static_scratch, sizeof(int), 8), "read the static error word");
    if (rc) return rc;
    if (!err) return WF_OK;
    const int zero = 0;
    rc = wf_cuda_check(cudaMemcpyToSymbol(g_static_scratch, &zero, sizeof(int), 8), "clear the static error word");
    if (rc) return rc;
    if ((err & 0xFF) == kStaticBadTables) {
        static const char *what[] = {"", "pred_off does not start at 0 or decreases",
                                     "a pred_idx entry is out of range or a self-loop", "a model id is >= M",
                                     "a session id is out of range", "a run time is negative or a peak below its weight",
                                     "a weight is below 1", "a capacity is below 1", "a load time is negative",
                                     "an arrival is negative"};
        const int k = err >> 8;
        return wf_set_error(WF_EINVAL, "the problem tables failed the device check: %s",
                            k >= 1 && k <= 9 ? what[k] : "unknown");
    }
    return wf_set_error(WF_ECUDA, "device error word %d in the static evaluation", err);
}

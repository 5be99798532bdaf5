// Plan construction: the paper's per-tick scheduler (Algorithm 1) read as a
// list scheduler over the whole window.
//
//   RankReady            a node is ready once every graph predecessor is
//                        dispatched; the ready node with the smallest
//                        (release + jitter, id) goes next (aging)
//   BestFeasibleBinding  the device, among those whose capacity holds the
//                        node (Eq. 8), with the smallest predicted finish
//                        (resident model: no load; missing model: loaded on
//                        the device, prefetched if the device would idle
//                        before the release) plus jitter; ties: lower device
//   units                the node's fusible chain (Eq. 3) follows it on that
//                        device while each next member fits (fuse bit 1)
//   PlanPrefetch         the head's prefetch bit when its model is missing
//                        and the device is free before the release
//
// Each unit is played forward with the evaluation rules (admission and LRU
// reclamation, Eq. 11; loads, Eq. 5; starts and finishes, Eq. 2, 7, 10), so
// the constructor's timeline is the one wf_eval_plans reports for its plan.
//
// A plan is built by a group of 8, 16 or 32 lanes (at least the device
// count), so a warp builds 4, 2 or 1 plans side by side: a plan's steps are a
// serial chain of small parallel parts -- the ready set's minimum, a score per
// device, a few successors -- which fill 8 lanes and leave most of 32 idle.  A
// batch that leaves the chip's warps idle takes more lanes instead, which
// shorten the chain (lanes_of).  Lane g
// keeps device g's state in registers (free time, residency queue, resident
// weights).  Control flow is uniform over the warp: a loop runs until every
// plan of the warp is through.  Bound by integer issue (64-bit hashes, keys
// and times).  16,384 plans of the burst window (N = 2,000, D = 8, jitter
// 0.2 s): 17.9 ms with a warp per plan (13.7 G warp instructions), 6.34 ms with 8
// lanes per plan (4.8 G, 63 % of the issue slots).
#include <algorithm>

#include "wf_play.cuh"

namespace {

constexpr int kWarps = 4;          // warps per CTA
constexpr int kCtasPerSm = 7;      // resident CTAs per SM (72 registers per thread)
constexpr int kWarpsPerSm = kWarps * kCtasPerSm;

// Lanes per plan.  The chain of one plan is shorter on more lanes (a warp's
// minimum is two reductions, a longer ready set takes fewer rounds), the
// chip's issue slots hold more plans on fewer.  N = 1,000, D = 3, us with 8,
// 16, 32 lanes: 512 plans 1,267, 1,128, 928; 1,024: 1,278, 1,130, 988; 1,766: 16
// lanes 1,220, 32 lanes 1,113; 2,048: 1,291, 1,234, 1,311; 3,072: 1,535, 1,450, 1,804; 4,096: 1,588, 1,676, 2,075.  N = 40 to
// 2,000 with 3 and 8 devices change sides at the same batches, 12 and 24 plans an
// SM.
int lanes_of(int32_t D, int64_t P, int sms)
{
    const int least = D <= 8 ? 8 : D <= 16 ? 16 : 32;
    return std::max(least, P <= 12 * (int64_t)sms ? 32 : P <= 24 * (int64_t)sms ? 16 : 8);
}

__device__ __forceinline__ uint64_t mix64(uint64_t x)  // SplitMix64 output function
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// x mod d for 2 <= d < 2^63 and every 64-bit x (Barrett reduction): with
// M = floor((2^64 - 1) / d), which is at least 2^64 / d - 1, the quotient
// floor(x M / 2^64) is floor(x / d) or one less, so one conditional
// subtraction completes the remainder.
struct Mod64 {
    uint64_t M, d;
};

__device__ __forceinline__ uint64_t mod64(uint64_t x, const Mod64 &m)
{
    const uint64_t r = x - __umul64hi(x, m.M) * m.d;
    return r >= m.d ? r - m.d : r;
}

// Per-plan state in global scratch.  Only a node with several predecessors
// keeps a count and the latest finish among those seen; a node with one is
// ready when that one finishes, at its finish.
struct Scratch {
    uint64_t *key;   // [N] ready keys (rank << 16 | node), unordered
    int64_t *last;   // [N] latest finish among the predecessors seen (valid once seen > 0)
    uint16_t *seen;  // [N] predecessors finished
};

__host__ __device__ inline size_t scratch_bytes(int32_t N)
{
    return ((8 + 8 + 2) * (size_t)N + 255) & ~(size_t)255;
}

// Minimum of a 64-bit key over the kL lanes of a group.
// A whole warp: the high halves, then the low halves of those that hold it
// (five shuffles of 64 bits instead: 16,384 plans of N = 1,000, D = 32 in
// 9.07 ms, so 7.94).
template <int kL>
__device__ __forceinline__ uint64_t group_min(uint64_t key)
{
    if constexpr (kL == 32) {
        const uint32_t hi = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(key >> 32));
        const uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(key >> 32) == hi ? (uint32_t)key : 0xFFFFFFFFu);
        return ((uint64_t)hi << 32) | lo;
    }
#pragma unroll
    for (int o = kL / 2; o; o >>= 1) {
        const uint64_t other = __shfl_xor_sync(0xFFFFFFFFu, key, o);
        key = other < key ? other : key;
    }
    return key;
}

// Q: the residency queue's word (Lru); kL: lanes per plan.
template <typename Q, int kL>
__global__ void __launch_bounds__(32 * kWarps, kCtasPerSm)
construct_kernel(wf_dev_problem dp, wf_plans out, uint64_t seed, int64_t jitter, Mod64 jm, uint8_t *scratch,
                 int64_t slots)
{
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    constexpr int kPer = 32 / kL;  // plans per warp
    constexpr uint32_t kGroup = kL == 32 ? kAll : (1u << (kL & 31)) - 1u;
    const int lane = threadIdx.x & 31, g = lane % kL, shift = lane - g;
    const int64_t w = ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * kPer;  // the warp's first slot
    if (w >= slots) return;
    const int64_t slot = w + lane / kL;
    const int32_t N = dp.N, D = dp.D;
    const int32_t words = (N + 31) / 32;
    // (a slot beyond the scratch builds nothing and touches nothing)
    uint8_t *base = scratch + (size_t)(slot < slots ? slot : 0) * scratch_bytes(N);
    Scratch s;
    s.key = (uint64_t *)base;
    s.last = (int64_t *)(s.key + N);
    s.seen = (uint16_t *)(s.last + N);
    const bool dev = g < D;
    const uint32_t capd = dev ? (uint32_t)__ldg(dp.cap + g) : 0u;
    // Appends this lane's key to the plan's ready set if take.
    int32_t nready = 0;
    const auto append = [&](bool take, uint64_t key) {
        const uint32_t bal = (__ballot_sync(kAll, take) >> shift) & kGroup;
        if (take) s.key[nready + __popc(bal & ((1u << g) - 1u))] = key;
        nready += __popc(bal);
    };
    // Jitter draws are taken mod (jitter + 1); none when jitter = 0.
    const auto rank_jitter = [&](uint64_t h) { return jitter > 0 ? mod64(h, jm) : 0ull; };
    for (int64_t p0 = w; p0 < out.P; p0 += slots) {
        const int64_t p = p0 + lane / kL;
        const bool live = p < out.P && slot < slots;
        const uint64_t hp = mix64(seed ^ (uint64_t)(out.plan_base + p));
        const int64_t pr = live ? p : 0;
        uint8_t *place = (uint8_t *)out.place + pr * out.place_stride;
        uint16_t *order = (uint16_t *)((uint8_t *)out.order + pr * out.order_stride);
        uint32_t *fuse = (uint32_t *)((uint8_t *)out.fuse + pr * out.bits_stride);
        uint32_t *prefetch = (uint32_t *)((uint8_t *)out.prefetch + pr * out.bits_stride);
        for (int32_t k = g; live && k < words; k += kL) { fuse[k] = 0; prefetch[k] = 0; }
        if (out.retain && live) {
            uint32_t *retain = (uint32_t *)((uint8_t *)out.retain + p * out.bits_stride);
            for (int32_t k = g; k < words; k += kL)
                retain[k] = (k + 1 < words || (N & 31) == 0) ? 0xFFFFFFFFu : ((1u << (N & 31)) - 1u);
        }
        // Device state of lane g.
        Q queue = 0;
        uint32_t n = 0, used = 0;
        int64_t tfree = 0;
        nready = 0;
        for (int32_t v0 = 0; v0 < N; v0 += kL) {
            const int32_t v = v0 + g;
            bool take = false;
            uint64_t key = 0;
            if (live && v < N) {
                s.seen[v] = 0;
                if (__ldg(dp.pred_off + v + 1) == __ldg(dp.pred_off + v)) {
                    const int64_t arr = __ldg(dp.arrival + __ldg(dp.session + v));
                    key = (((uint64_t)arr + rank_jitter(mix64(hp ^ (uint64_t)v))) << 16) | (uint64_t)v;
                    take = true;
                }
            }
            append(take, key);
        }
        __syncwarp();
        int32_t pos = 0;
        while (__any_sync(kAll, nready > 0)) {
            const bool act = nready > 0;
            // RankReady: the smallest key (keys are unique).  Its lane then
            // holds its place, which takes the last entry.  (When it was the
            // last entry nothing moves: the successors' keys go there below,
            // from other lanes.)
            uint64_t best = ~0ull;
            int32_t at = 0;
            for (int32_t i = g; i < nready; i += 4 * kL) {
                uint64_t k[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) k[j] = i + j * kL < nready ? s.key[i + j * kL] : ~0ull;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (k[j] < best) { best = k[j]; at = i + j * kL; }
            }
            const uint64_t mine = best;
            best = group_min<kL>(best);
            if (act) --nready;
            const uint64_t tail_key = act ? s.key[nready] : 0ull;
            __syncwarp();
            if (act && mine == best && at != nready) s.key[at] = tail_key;
            const int32_t u = act ? (int32_t)(best & 0xFFFFu) : 0;
            const uint64_t hu = mix64(hp ^ (uint64_t)u);
            const int64_t rel = (int64_t)((best >> 16) - rank_jitter(hu));
            const int32_t m = __ldg(dp.model + u);
            const int64_t arr = __ldg(dp.arrival + __ldg(dp.session + u));
            const uint32_t fit_u = __ldg(dp.fitmask + u);

            // BestFeasibleBinding: a device per lane, then the smallest
            // (score, device); scores stay below 2^49.
            const int32_t kq = Lru<Q>::find(queue, n, (uint32_t)m);
            const bool hit = kq < (int32_t)n;
            const bool pf = !hit && tfree < rel;
            int64_t ld = 0, start = 0;
            int2 lk = make_int2(0, 0);
            uint64_t score = ~0ull;
            if (dev && ((fit_u >> g) & 1u)) {
                lk = __ldg(dp.lk + u * D + g);
                ld = hit ? 0 : (int64_t)__ldg(dp.load + m * D + g);
                start = max(max(tfree, pf ? arr : rel) + ld, rel);
                const int64_t fin = start + dp.grant + (int64_t)lk.x;
                score = ((uint64_t)(fin + (jitter > 0 ? (int64_t)mod64(mix64(hu ^ (uint64_t)(g + 1)), jm) : 0)) << 5) |
                        (uint64_t)g;
            }
            score = group_min<kL>(score);
            if (act && score == ~0ull) {  // unreachable: every node fits somewhere
                if (g == 0) atomicExch(dp.err, 4);
                nready = 0;
            }
            const bool on = act && score != ~0ull;
            const int32_t d = (int32_t)(score & 31u);
            const bool own = on && g == d;  // the unit's device

            // The unit: u and its fusible chain while the members fit on d.
            if (on && g == 0) { place[u] = (uint8_t)d; order[pos] = (uint16_t)u; }
            if (own && pf) atomicOr(prefetch + (u >> 5), 1u << (u & 31));
            if (on) ++pos;
            int32_t tail = u;
            int32_t kv = lk.y;
            int64_t run = (int64_t)dp.grant + lk.x;
            for (int32_t x = on ? __ldg(dp.fnext + u) : -1;
                 x >= 0 && ((__ldg(dp.fitmask + x) >> d) & 1u); x = __ldg(dp.fnext + x)) {
                if (g == 0) {
                    place[x] = (uint8_t)d;
                    order[pos] = (uint16_t)x;
                    atomicOr(fuse + (x >> 5), 1u << (x & 31));
                }
                ++pos;
                const int2 lx = __ldg(dp.lk + x * D + d);
                kv = max(kv, lx.y);
                run += lx.x;
                tail = x;
            }

            // Play it forward on its device's lane: admission with LRU
            // reclamation (Eq. 11; the unit's own model leaves the queue
            // first, then the victims are the queue's head), load, run.
            if (own) {
                const uint32_t wm = (uint32_t)__ldg(dp.weight + m);
                if (hit) { queue = Lru<Q>::remove(queue, kq); n -= 1; }
                const uint32_t need = hit ? (uint32_t)kv : wm + (uint32_t)kv;  // used + need <= cap + peak < 2^32
                while (used + need > capd && n > 0) {
                    used -= (uint32_t)__ldg(dp.weight + ((uint32_t)queue & 15u));
                    queue >>= 4;
                    n -= 1;
                }
                if (used + need > capd) atomicExch(dp.err, 4);  // unreachable: the unit fits on d
                queue |= (Q)m << (4 * n);
                n += 1;
                if (!hit) used += wm;
                tfree = start + run;
            }
            const int64_t fin = __shfl_sync(kAll, tfree, d, kL);

            // Successors of the unit's last member, one per lane: the last
            // predecessor to finish makes one ready, released at the latest
            // finish (never before the session's arrival, which every unit
            // of the session waits for).
            int32_t e = 0, e1 = 0;
            if (on) { e = __ldg(dp.succ_off + tail) + g; e1 = __ldg(dp.succ_off + tail + 1); }
            __syncwarp();  // (orders the move above before the appended keys)
            do {
                bool take = false;
                uint64_t key = 0;
                if (e < e1) {
                    const int32_t y = __ldg(dp.succ_idx + e);
                    const int32_t np = __ldg(dp.pred_off + y + 1) - __ldg(dp.pred_off + y);
                    int64_t r = fin;
                    take = true;
                    if (np > 1) {
                        const int32_t before = s.seen[y];
                        if (before > 0) r = max(r, s.last[y]);
                        take = before + 1 == np;
                        if (!take) { s.seen[y] = (uint16_t)(before + 1); s.last[y] = r; }
                    }
                    if (take) key = (((uint64_t)r + rank_jitter(mix64(hp ^ (uint64_t)y))) << 16) | (uint64_t)y;
                    e += kL;
                }
                append(take, key);
            } while (__any_sync(kAll, e < e1));
            __syncwarp();
        }
    }
}

// Plans built at once by the largest batch: as many as are resident, as far as
// 1 GiB of scratch goes (112 plans per SM up to N of about 3,500), and at least
// 60 per SM beyond that (more than a batch on more lanes holds at all).
int64_t plans_at_once(const wf_ctx *c)
{
    const int64_t fit = ((int64_t)1 << 30) / (int64_t)scratch_bytes(c->dp.N);
    const int64_t resident = (int64_t)kWarpsPerSm * (32 / lanes_of(c->dp.D, c->max_P, c->sms));
    return std::min<int64_t>(c->max_P, std::min<int64_t>(c->sms * resident, std::max<int64_t>(fit, (int64_t)c->sms * 60)));
}

// Calls f(kernel) for this problem's instantiation with l lanes per plan.
template <typename F>
int construct_visit(const wf_dev_problem &dp, int l, F &&f)
{
    if (dp.M <= 8)
        return l == 8 ? f(construct_kernel<uint32_t, 8>) : l == 16 ? f(construct_kernel<uint32_t, 16>)
                                                                   : f(construct_kernel<uint32_t, 32>);
    return l == 8 ? f(construct_kernel<uint64_t, 8>) : l == 16 ? f(construct_kernel<uint64_t, 16>)
                                                               : f(construct_kernel<uint64_t, 32>);
}

}  // namespace

extern "C" int wf_construct_plans(wf_ctx *c, const wf_plans *out, uint64_t seed, int64_t jitter_us, void *stream)
{
    if (!c || !out) return wf_set_error(WF_EINVAL, "NULL argument");
    int rc = wf_check_plans(c, out, "plans");
    if (rc) return rc;
    if (jitter_us < 0) return wf_set_error(WF_EINVAL, "jitter_us < 0");
    // Ranks (release + jitter) are packed above a 16-bit node id.
    if (c->dp.horizon + jitter_us >= ((int64_t)1 << 47))
        return wf_set_error(WF_EINVAL, "window horizon %lld us + jitter exceeds 2^47 us", (long long)c->dp.horizon);
    rc = wf_select_device(c);
    if (rc) return rc;
    const wf_dev_problem &dp = c->dp;
    if (!c->construct_scratch) {
        // First call: per-plan state for as many plans as are built at once.
        c->construct_threads = plans_at_once(c);
        rc = wf_cuda_check(cudaMalloc(&c->construct_scratch, scratch_bytes(dp.N) * c->construct_threads),
                           "cudaMalloc(constructor scratch)");
        if (rc) { c->construct_scratch = nullptr; return rc; }
    }
    const int64_t slots = std::min<int64_t>(out->P, c->construct_threads);
    const int lanes = lanes_of(dp.D, out->P, c->sms);
    const int64_t per_cta = kWarps * (32 / lanes);
    const unsigned blocks = (unsigned)((slots + per_cta - 1) / per_cta);
    const uint64_t jd = (uint64_t)jitter_us + 1;
    const Mod64 jm = {~0ull / jd, jd};
    return construct_visit(dp, lanes, [&](auto k) {
        k<<<blocks, 32 * kWarps, 0, (cudaStream_t)stream>>>(dp, *out, seed, jitter_us, jm,
                                                            (uint8_t *)c->construct_scratch, slots);
        return wf_cuda_check(cudaGetLastError(), "construct launch");
    });
}

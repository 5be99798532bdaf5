// Stochastic latencies: the plans of a window with S latency
// samples, each sample's times on u32; the floor means over the samples and the
// nearest-rank p95 of all their sessions' latencies.
//
// A team plays a plan at a time: a helper warp turns 32 dispatch positions at
// once into unit records (lane = position; Eq. 3-4), settles their residency,
// which is the same for every sample (lane = device; Eq. 11), and leaves the
// units side by side in a ring of two buffers; the timing warps play them
// (Eq. 2, 5, 7, 10) with kV samples a lane, each drawing its run-time multipliers
// from (plan, sample, node) through SplitMix64 and the integer Box-Muller
// tables.  Helper and timing meet at one barrier a chunk.  A CTA holds as many
// teams as its shared memory does, and one copy of the Box-Muller tables for
// them all; a team walks over plans.
//
// What bounds it is a timing lane's dependent chain and its ALU instructions
// (about 100 a sample and position: a 64-bit hash, three table reads, the
// times), not bandwidth.  Hence two samples a lane, which share a record's
// decoding and overlap their chains; the next unit's multiplier drawn while this
// one plays; every slot of a unit read before any is written; and the tables in
// shared memory, where 32 random reads take about 4 cycles (through L1 they
// take one for each line they touch).  8,192 plans of N = 500 with 64 samples,
// us a call: 1,318 against 2,504 for a plan per CTA of four warps with its
// tables in L1; a sample a lane and two timing warps a team 1,366; six teams a CTA
// where seven fit (the histogram in the free times' place) 1,490; the timing
// loop unrolled twice 1,390.
#include <algorithm>

#include "wf_play.cuh"

namespace {

constexpr int kPos = 32;            // positions a chunk
constexpr int kMaxThreads = 512;    // of a CTA: 128 registers a thread
constexpr int kMaxTiming = 4;       // timing warps of a team
constexpr size_t kSmemCta = 227 * 1024;

struct StochShape {
    int32_t teams, tw;   // teams a CTA, timing warps a team
    int32_t cols;        // samples rounded up to kV: the row length of slots and device free times
    uint32_t weight, cap, load, arr, tab_r, tab_c, tab_e, team0;  // byte offsets of the CTA's tables and its first team
    uint32_t ring, slots, tfree, red, team;                 // offsets within a team, and its size
};

inline uint32_t shape_layout(const wf_dev_problem &dp, StochShape &s, bool tab, int v)
{
    s.cols = (dp.S + v - 1) / v * v;
    uint32_t o = 0;
    s.weight = o; o += 4u * 16;
    s.cap = o; o += round16(4u * dp.D);
    s.load = o; o += round16(4u * dp.M * dp.D);
    s.arr = o; o += round16(4u * dp.W);
    s.tab_r = o; o += tab ? round16(2u * dp.bm_rn) : 0u;
    s.tab_c = o; o += tab ? round16(2u * dp.bm_cn) : 0u;
    s.tab_e = o; o += tab ? round16(4u * dp.bm_en) : 0u;
    s.team0 = o;
    uint32_t t = 0;
    s.ring = t; t += 2 * 32u * kPos + 16;                    // two buffers of 32-byte records; {units, open devices} of each
    s.red = t; t += 16u * kMaxTiming + 16;                   // partial sums of the timing warps; prefix, rank, overflow
    s.tfree = t; t += round16(std::max(4u * dp.D * s.cols, 4u * 256));  // (at a plan's end: the selection's histogram)
    s.slots = t; t += round16(4u * (uint32_t)(dp.nslots + 2) * s.cols);
    s.team = t + 8u * kPos;                                  // (the helper's residency results at the end)
    return o;
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// kV consecutive words of shared memory.
template <int kV>
__device__ __forceinline__ void get(const uint32_t *p, uint32_t (&x)[kV])
{
    if constexpr (kV == 2) {
        const uint2 u = *(const uint2 *)p;
        x[0] = u.x; x[1] = u.y;
    } else {
        x[0] = *p;
    }
}
template <int kV>
__device__ __forceinline__ void put(uint32_t *p, const uint32_t (&x)[kV])
{
    if constexpr (kV == 2) *(uint2 *)p = make_uint2(x[0], x[1]);
    else *p = x[0];
}

// The Box-Muller tables: radius and angle as int16 copies in shared memory
// (kTab), or the problem's int32 tables in global memory (values beyond 16 bits, or
// tables too long for shared memory).
template <bool kTab>
struct Tables;
template <>
struct Tables<true> {
    const int16_t *r, *c;
    const int32_t *e;  // at multiplier 0's place
    uint32_t rmask, cmask;
    __device__ __forceinline__ uint32_t mult(uint64_t h) const
    {
        const int32_t prod = (int32_t)r[(uint32_t)h & rmask] * (int32_t)c[(uint32_t)(h >> 32) & cmask];
        return (uint32_t)e[prod >> 18];
    }
};
template <>
struct Tables<false> {
    const int32_t *r, *c;
    const int32_t *e;
    uint32_t rmask, cmask;
    __device__ __forceinline__ uint32_t mult(uint64_t h) const
    {
        const int64_t prod = (int64_t)__ldg(r + ((uint32_t)h & rmask)) * (int64_t)__ldg(c + ((uint32_t)(h >> 32) & cmask));
        return (uint32_t)__ldg(e + (prod >> 18));
    }
};

// A unit's record, two 16-byte words:
//   a: head | last member << 16; the head's run time on the device; the arrival; device | kRare | prefetch << 9 |
//      kWasEmpty | writes << 11 | kEmptied | first code << 16
//   b: second code | third << 16; fourth code | release slot code << 16; load time (0 on a hit); 0
// A code that names the release slot which the unit itself resets is stored
// without its accumulator bit: what it finds there is 0.
// kRare: the unit changes its device's occupancy or writes more than two slots.
constexpr uint32_t kRare = 1u << 5;

template <typename Q, int kV, bool kTab>
__global__ void __launch_bounds__(kMaxThreads, 1)
stoch_kernel(wf_dev_problem dp, wf_plans pl, wf_eval_out out, StochShape sh, int32_t *ovf_list, int32_t *ovf_count)
{
    extern __shared__ __align__(128) uint8_t sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t N = dp.N, D = dp.D, M = dp.M, W = dp.W, S = dp.S;
    int32_t *weight = (int32_t *)(sm + sh.weight);
    int32_t *load = (int32_t *)(sm + sh.load);
    uint32_t *arrival = (uint32_t *)(sm + sh.arr);
    for (int32_t k = threadIdx.x; k < M; k += blockDim.x) weight[k] = __ldg(dp.weight + k);
    for (int32_t k = threadIdx.x; k < M * D; k += blockDim.x) load[k] = __ldg(dp.load + k);
    for (int32_t k = threadIdx.x; k < W; k += blockDim.x) arrival[k] = (uint32_t)__ldg(dp.arrival + k);
    if constexpr (kTab) {
        for (int32_t k = threadIdx.x; k < dp.bm_rn; k += blockDim.x) ((int16_t *)(sm + sh.tab_r))[k] = __ldg(dp.bm_r16 + k);
        for (int32_t k = threadIdx.x; k < dp.bm_cn; k += blockDim.x) ((int16_t *)(sm + sh.tab_c))[k] = __ldg(dp.bm_c16 + k);
        for (int32_t k = threadIdx.x; k < dp.bm_en; k += blockDim.x) ((int32_t *)(sm + sh.tab_e))[k] = __ldg(dp.bm_e + k);
    }
    __syncthreads();

    // Warps: every team's timing warps first, then the helpers, so that the
    // timing warps spread over the SM's four schedulers.
    const int tw = sh.tw, timing_warps = sh.teams * tw;
    const bool helper = warp >= timing_warps;
    const int team = helper ? warp - timing_warps : warp / tw;
    const int bar = 1 + team, bar_timing = 1 + sh.teams + team;  // (named barriers; the second with several timing warps)
    const int team_threads = 32 * (tw + 1);
    uint8_t *tm = sm + sh.team0 + (size_t)team * sh.team;
    uint4 *ring = (uint4 *)(tm + sh.ring);  // [buffer][unit][2]
    uint32_t *head_of = (uint32_t *)(tm + sh.ring + 2 * 32 * kPos);  // [buffer]{units, open devices}
    const int32_t chunks = (N + kPos - 1) / kPos;
    const int64_t step = (int64_t)gridDim.x * sh.teams;

    if (helper) {
        uint2 *res = (uint2 *)(tm + sh.team - 8 * kPos);  // by position: load time, flags
        const uint32_t capd = lane < D ? (uint32_t)__ldg(dp.cap + lane) : 0u;
        const uint32_t cols_zero = (uint32_t)dp.nslots + 1;
        int buf = 0;
        for (int64_t p = (int64_t)blockIdx.x * sh.teams + team; p < pl.P; p += step) {
            if (__ldg(out.status + p) != 0) continue;  // the status kernel marked the plan invalid
            const uint8_t *place = pl.place + p * pl.place_stride;
            const uint16_t *order = (const uint16_t *)((const uint8_t *)pl.order + p * pl.order_stride);
            const uint32_t *fuse = bits_row(pl.fuse, p * pl.bits_stride), *prefetch = bits_row(pl.prefetch, p * pl.bits_stride);
            const uint32_t *retain = pl.retain ? bits_row(pl.retain, p * pl.bits_stride) : nullptr;
            Q queue = 0;  // this lane's device
            uint32_t nres = 0, used = 0;
            int32_t h = lane < N ? __ldg(order + lane) : 0;
            for (int32_t c = 0; c < chunks; ++c, buf ^= 1) {
                const int32_t i = c * kPos + lane;
                const int32_t hn = i + kPos < N ? __ldg(order + i + kPos) : 0;  // a chunk ahead
                // The unit that starts at this lane's position, if one does.
                bool unit = i < N;
                uint32_t d = 0, tail = (uint32_t)h, kv = 0, lat = 0, w3 = 0, r4 = 0, c4 = 0;
                uint4 hr = make_uint4(0xFFFFFFFFu, cols_zero, 0, 0);
                if (unit) {
                    d = __ldg(place + h);
                    hr = __ldg(dp.hrec + h);
                    const uint32_t pw = __ldg(prefetch + (h >> 5)), fp = hr.x & 0xFFFFu;
                    if (fp != 0xFFFFu && bit_of_g(fuse, h) && __ldg(place + fp) == d) unit = false;  // inside its head's unit
                    else {
                        const int2 lk0 = __ldg(dp.lk + h * D + (int32_t)d);
                        lat = (uint32_t)lk0.x;
                        int32_t need = lk0.y;
                        uint32_t ty = hr.y, tcodes = hr.w;
                        for (uint32_t s = hr.x >> 16; s != 0xFFFFu;) {  // Eq. 3 chain
                            if (!bit_of_g(fuse, (int32_t)s) || __ldg(place + s) != d) break;
                            need = max(need, __ldg(&dp.lk[(int32_t)s * D + (int32_t)d].y));
                            const uint4 sr = __ldg(dp.hrec + s);
                            tail = s;
                            ty = sr.y;
                            tcodes = sr.w;
                            s = sr.x >> 16;
                        }
                        kv = (uint32_t)need;
                        const uint32_t c23 = __ldg(dp.wc23 + tail), rs = hr.y & 0xFFFFu;
                        uint32_t c0 = tcodes & 0xFFFFu, c1 = tcodes >> 16;
                        if (c0 == rs) c0 &= 0x7FFFu;  // (both accumulators: reset by this unit, so 0)
                        if (c1 == rs) c1 &= 0x7FFFu;
                        const uint32_t drop = retain ? !bit_of_g(retain, (int32_t)tail) : 0u;
                        w3 = d | (((hr.y >> 16) & 15u) << 5) | (((pw >> (h & 31)) & 1u) << 9) | (drop << 10) |
                             (((ty >> 20) & 7u) << 11) | (c0 << 16);
                        r4 = c1 | (c23 << 16);
                        c4 = c23 >> 16;
                    }
                }
                // Residency: lane = device, its units of the chunk in order.
                uint32_t mine = 0;
                const int32_t du = unit ? (int32_t)d : -1;
                for (int32_t dd = 0; dd < D; ++dd) {
                    const uint32_t on = __ballot_sync(0xFFFFFFFFu, du == dd);
                    if (lane == dd) mine = on;
                }
                while (__any_sync(0xFFFFFFFFu, mine != 0)) {
                    const int k = mine ? __ffs((int)mine) - 1 : 0;
                    const uint32_t r1 = __shfl_sync(0xFFFFFFFFu, kv, k), r3 = __shfl_sync(0xFFFFFFFFu, w3, k);
                    if (mine) {
                        bool missed;
                        res[k] = settle_lru<Q>(queue, nres, used, capd, r1, r3, weight, load, D, dp.err, missed);
                        mine &= mine - 1;
                    }
                }
                __syncwarp();
                const uint32_t units = __ballot_sync(0xFFFFFFFFu, unit);
                if (unit) {
                    const uint2 x = res[lane];
                    uint4 *dst = ring + 2 * (buf * kPos + __popc(units & ((1u << lane) - 1u)));
                    const bool rare = (x.y & (kWasEmpty | kEmptied)) || (x.y & kMany);
                    dst[0] = make_uint4((uint32_t)h | (tail << 16), lat, hr.z, (x.y & ~(15u << 5)) | (rare ? kRare : 0u));
                    dst[1] = make_uint4(r4, c4 | (hr.y << 16), x.x, 0u);
                }
                const uint32_t open = __ballot_sync(0xFFFFFFFFu, lane < D && nres != 0);
                if (lane == 0) {
                    head_of[2 * buf] = (uint32_t)__popc(units);
                    head_of[2 * buf + 1] = (uint32_t)__popc(open);
                }
                h = hn;
                __syncwarp();
                named_sync(bar, team_threads);  // this buffer is full; timing is done with the other
            }
        }
        return;
    }

    // ---------------- timing: kV samples a lane ----------------
    const int tt = 32 * (warp % tw) + lane;  // within the team
    const int32_t s0 = kV * tt, cols = sh.cols;
    const bool on = s0 < S;  // (the last lane's second sample may be one too many: played, not counted)
    uint32_t *slots = (uint32_t *)(tm + sh.slots) + (on ? s0 : 0);
    uint32_t *tfree = (uint32_t *)(tm + sh.tfree) + (on ? s0 : 0);
    uint32_t *hist = (uint32_t *)(tm + sh.tfree);
    int64_t *red = (int64_t *)(tm + sh.red);                                     // [timing warp]{makespan, GPU time}
    uint32_t *sel = (uint32_t *)(tm + sh.red + 16 * kMaxTiming);                 // prefix, rank, overflow
    auto sync_timing = [&] {
        if (tw == 1) __syncwarp();
        else named_sync(bar_timing, 32 * tw);
    };
    Tables<kTab> tab;
    if constexpr (kTab) {
        tab.r = (const int16_t *)(sm + sh.tab_r);
        tab.c = (const int16_t *)(sm + sh.tab_c);
        tab.e = (const int32_t *)(sm + sh.tab_e) + ((dp.bm_en - 1) >> 1);
    } else {
        tab.r = dp.bm_r;
        tab.c = dp.bm_c;
        tab.e = dp.bm_e + ((dp.bm_en - 1) >> 1);
    }
    tab.rmask = (uint32_t)dp.bm_rn - 1u;
    tab.cmask = (uint32_t)dp.bm_cn - 1u;
    const uint32_t grant = (uint32_t)dp.grant;
    const int64_t pool = (int64_t)S * W, rank = (95 * pool + 99) / 100 - 1;
    int buf = 0;
    for (int64_t p = (int64_t)blockIdx.x * sh.teams + team; p < pl.P; p += step) {
        if (__ldg(out.status + p) != 0) continue;
        uint64_t key[kV];
        uint32_t end[kV], ovf[kV], zero[kV];
        int64_t gsum[kV];
        const uint64_t pkey = splitmix64(dp.seed ^ (uint64_t)(pl.plan_base + p));
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            key[v] = splitmix64(pkey ^ (uint64_t)(s0 + v));
            end[v] = ovf[v] = zero[v] = 0;
            gsum[v] = 0;
        }
        if (on) {
            for (int32_t k = 0; k < dp.nslots + 2; ++k) put<kV>(slots + k * cols, zero);
            for (int32_t d = 0; d < D; ++d) put<kV>(tfree + d * cols, zero);
        }
        // A member's sampled run time, added to run (Eq. 4).
        auto draw = [&](uint32_t j, uint32_t lat, uint32_t (&run)[kV]) {
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                const uint64_t x = (uint64_t)lat * tab.mult(splitmix64(key[v] ^ (uint64_t)j)) + 32768u;
                ovf[v] |= (uint32_t)(x >> 48);
                run[v] = add_carry(run[v], (uint32_t)(x >> 16), ovf[v]);
            }
        };
        auto rest_of_chain = [&](uint32_t ends, uint32_t d, uint32_t (&run)[kV]) {  // the members after the head
            for (uint32_t j = ends & 0xFFFFu, t = ends >> 16; j != t;) {
                j = __ldg(dp.links + j) >> 16;
                draw(j, (uint32_t)__ldg(&dp.lk[(int32_t)j * D + (int32_t)d].x), run);
            }
        };
        uint32_t open = 0;
        for (int32_t c = 0; c < chunks; ++c, buf ^= 1) {
            named_sync(bar, team_threads);
            const int32_t cnt = (int32_t)head_of[2 * buf];
            open = head_of[2 * buf + 1];
            if (on && cnt) {
                const uint4 *rb = ring + 2 * buf * kPos;
                uint4 a = rb[0], b = rb[1];
                uint32_t run[kV];
#pragma unroll
                for (int v = 0; v < kV; ++v) run[v] = grant;
                draw(a.x & 0xFFFFu, a.y, run);
                rest_of_chain(a.x, a.w & 31u, run);
#pragma unroll 1
                for (int32_t k = 0; k < cnt; ++k) {
                    const int32_t kn = min(k + 1, cnt - 1);
                    const uint4 na = rb[2 * kn], nb = rb[2 * kn + 1];
                    const uint32_t rs = b.y >> 16, arr = a.z;
                    uint32_t *s_rel = slots + (int32_t)(rs & 0x7FFFu) * cols, *s0p = slots + (int32_t)((a.w >> 16) & 0x7FFFu) * cols,
                             *s1p = slots + (int32_t)(b.x & 0x7FFFu) * cols, *s_tf = tfree + (int32_t)(a.w & 31u) * cols;
                    uint32_t rel[kV], tf[kV], o0[kV], o1[kV], cfin[kV], nrun[kV], ls[kV];
                    get<kV>(s_rel, rel);
                    get<kV>(s_tf, tf);
                    get<kV>(s0p, o0);
                    get<kV>(s1p, o1);
#pragma unroll
                    for (int v = 0; v < kV; ++v) nrun[v] = grant;
                    draw(na.x & 0xFFFFu, na.y, nrun);  // (a chunk's last unit is drawn twice: a branch here would part the two chains)
#pragma unroll
                    for (int v = 0; v < kV; ++v) {
                        const uint32_t r = max(arr, rel[v]);                                // Eq. 2, Eq. 7
                        ls[v] = max(tf[v], (a.w & kPrefetch) ? arr : r);                    // Eq. 5
                        const uint32_t start = max(add_carry(ls[v], b.z, ovf[v]), r);
                        cfin[v] = add_carry(start, run[v], ovf[v]);
                        o0[v] = (a.w >> 31) ? max(o0[v], cfin[v]) : cfin[v];
                        o1[v] = (b.x & 0x8000u) ? max(o1[v], cfin[v]) : cfin[v];
                    }
                    if (rs & 0x8000u) put<kV>(s_rel, zero);  // an accumulator is reset by its reader
                    put<kV>(s_tf, cfin);
                    put<kV>(s0p, o0);
                    put<kV>(s1p, o1);
                    if (a.w & kRare) {
#pragma unroll
                        for (int v = 0; v < kV; ++v) {
                            if (a.w & kWasEmpty) gsum[v] -= (int64_t)ls[v];
                            if (a.w & kEmptied) gsum[v] += (int64_t)cfin[v];
                        }
                        auto publish_at = [&](uint32_t code) {
                            uint32_t *sp = slots + (int32_t)(code & 0x7FFFu) * cols;
                            uint32_t x[kV];
                            get<kV>(sp, x);
#pragma unroll
                            for (int v = 0; v < kV; ++v) x[v] = (code & 0x8000u) ? max(x[v], cfin[v]) : cfin[v];
                            put<kV>(sp, x);
                        };
                        const uint32_t nwl = (a.w >> 11) & 7u;
                        if (a.w & kMany) publish_at(b.x >> 16);
                        if (nwl >= kWrites4) publish_at(b.y & 0xFFFFu);
                        if (nwl > kWrites4) {
                            const int4 wr = __ldg(dp.noderec + 2 * (int32_t)(a.x >> 16) + 1);
                            for (int32_t e = 4; e < wr.y; ++e) publish_at(__ldg(dp.wl + wr.x + e));
                        }
                    }
                    if (k + 1 < cnt) rest_of_chain(na.x, na.w & 31u, nrun);
                    a = na;
                    b = nb;
#pragma unroll
                    for (int v = 0; v < kV; ++v) run[v] = nrun[v];
                }
            }
            __syncwarp();
        }
        // Per-sample results: sums over the samples, and the sessions' latencies.
        // (a plan's end: its devices' last finishes)
        if (on)
            for (int32_t d = 0; d < D; ++d) {
                uint32_t x[kV];
                get<kV>(tfree + d * cols, x);
#pragma unroll
                for (int v = 0; v < kV; ++v) end[v] = max(end[v], x[v]);
            }
        int64_t mk = 0, gp = 0;
        uint32_t bad = 0;
#pragma unroll
        for (int v = 0; v < kV; ++v)
            if (s0 + v < S) {
                mk += (int64_t)end[v] - dp.first_arrival;
                gp += gsum[v] + (int64_t)open * (int64_t)end[v];
                bad |= ovf[v];
            }
        for (int o = 16; o; o >>= 1) {
            mk += __shfl_xor_sync(0xFFFFFFFFu, mk, o);
            gp += __shfl_xor_sync(0xFFFFFFFFu, gp, o);
        }
        bad = __any_sync(0xFFFFFFFFu, bad != 0);
        if (tt == 0) sel[2] = 0;
        if (lane == 0) {
            red[2 * (warp % tw)] = mk;
            red[2 * (warp % tw) + 1] = gp;
        }
        if (tw > 1) {
            sync_timing();
            if (lane == 0 && bad) sel[2] = 1;
            sync_timing();
            bad = sel[2];
        }
        if (bad) {  // some sample's times leave 32 bits: the int64 path plays the plan
            if (tt == 0) ovf_list[atomicAdd(ovf_count, 1)] = (int32_t)p;
            sync_timing();
            continue;
        }
        if (on)
            for (int32_t w = 0; w < W; ++w) {
                uint32_t x[kV];
                get<kV>(slots + w * cols, x);
#pragma unroll
                for (int v = 0; v < kV; ++v) x[v] -= arrival[w];
                put<kV>(slots + w * cols, x);
            }
        sync_timing();  // the histogram takes the free times' place
        // Nearest-rank p95 of the S x W latencies: radix selection, 8 bits a
        // pass; the first warp scans the histogram, 8 buckets a lane.
        uint32_t prefix = 0, left = (uint32_t)rank;
        for (int shift = 24; shift >= 0; shift -= 8) {
            for (int k = tt; k < 256; k += 32 * tw) hist[k] = 0;
            sync_timing();
            const uint32_t hi = shift == 24 ? 0u : (~0u << (shift + 8));
            if (on)
                for (int32_t w = 0; w < W; ++w) {
                    uint32_t x[kV];
                    get<kV>(slots + w * cols, x);
#pragma unroll
                    for (int v = 0; v < kV; ++v)
                        if (s0 + v < S && (x[v] & hi) == prefix) atomicAdd(&hist[(x[v] >> shift) & 255u], 1u);
                }
            sync_timing();
            if (tt < 32) {
                uint32_t b8[8], sum = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) { b8[k] = hist[8 * lane + k]; sum += b8[k]; }
                uint32_t upto = sum;
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
                    if (lane >= o) upto += y;
                }
                const int at = __ffs((int)__ballot_sync(0xFFFFFFFFu, upto > left)) - 1;
                uint32_t before = upto - sum;
                int bin = 0;
                while (bin < 7 && before + b8[0] <= left) {
                    before += b8[0];
#pragma unroll
                    for (int k = 0; k < 7; ++k) b8[k] = b8[k + 1];
                    ++bin;
                }
                before = __shfl_sync(0xFFFFFFFFu, before, at);
                bin = __shfl_sync(0xFFFFFFFFu, bin, at);
                prefix |= (uint32_t)(8 * at + bin) << shift;
                left -= before;
                if (lane == 0) { sel[0] = prefix; sel[1] = left; }
            }
            sync_timing();
            prefix = sel[0];
            left = sel[1];
        }
        if (tt == 0) {
            int64_t smk = 0, sg = 0;
            for (int k = 0; k < tw; ++k) { smk += red[2 * k]; sg += red[2 * k + 1]; }
            out.makespan_us[p] = smk / S;
            out.gpu_us[p] = sg / S;
            out.p95_us[p] = (int64_t)prefix;
        }
        sync_timing();  // slots, histogram and sums are free for the next plan
    }
}

// The shape for a problem and batch: as many teams a CTA as shared memory and
// threads allow, no more than spread the plans over the SMs; the tables in shared
// memory where they fit beside a team.
bool choose_shape(const wf_dev_problem &dp, StochShape &s, bool &tab, int &v, size_t &smem)
{
    if (dp.nslots <= 0 || dp.nslots > 32765 || dp.max_arrival >= (int64_t)1 << 32 || dp.M > 16 || dp.N > 65534 || dp.S < 1)
        return false;
    v = dp.S <= 32 ? 1 : 2;  // (one warp of single samples where half of it would have none)
    s.tw = (dp.S + 32 * v - 1) / (32 * v);
    if (s.tw > kMaxTiming || (int64_t)dp.S * dp.W > INT32_MAX) return false;
    const int most = kMaxThreads / (32 * (s.tw + 1));
    for (int t = dp.bm_r16 ? 1 : 0; t >= 0; --t) {
        tab = t != 0;
        if (tab && 2 * ((int64_t)dp.bm_rn + dp.bm_cn) + 4 * (int64_t)dp.bm_en > 128 * 1024) continue;
        const uint32_t common = shape_layout(dp, s, tab, v);
        if ((size_t)common + s.team > kSmemCta) continue;
        s.teams = (int32_t)std::min<size_t>(most, (kSmemCta - common) / s.team);
        smem = common + (size_t)s.teams * s.team;
        return true;
    }
    return false;
}

template <typename Q, int kV, bool kTab>
int stoch_launch(const wf_ctx *ctx, const StochShape &s, size_t smem, const wf_plans *pl, const wf_eval_out *out,
                 int32_t *ovf_list, int32_t *ovf_count, cudaStream_t st)
{
    const auto k = stoch_kernel<Q, kV, kTab>;
    const int threads = 32 * s.teams * (s.tw + 1);
    int rc = wf_cuda_check(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                           "stochastic smem attribute");
    int n = 0;
    if (!rc) rc = wf_cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem), "stochastic occupancy");
    if (rc) return rc;
    const int64_t blocks = std::min<int64_t>((pl->P + s.teams - 1) / s.teams, (int64_t)std::max(1, n) * ctx->sms);
    k<<<(unsigned)blocks, threads, smem, st>>>(ctx->dp, *pl, *out, s, ovf_list, ovf_count);
    return wf_cuda_check(cudaGetLastError(), "stochastic launch");
}

}  // namespace

bool wf_stoch_usable(const wf_dev_problem &dp)
{
    StochShape s;
    bool tab;
    int v;
    size_t smem;
    return choose_shape(dp, s, tab, v, smem);
}

int wf_launch_stoch(wf_ctx *ctx, const wf_plans *pl, const wf_eval_out *out, int32_t *ovf_list, int32_t *ovf_count,
                    cudaStream_t st)
{
    const wf_dev_problem &dp = ctx->dp;
    StochShape s;
    bool tab;
    int v;
    size_t smem;
    if (!choose_shape(dp, s, tab, v, smem)) return wf_set_error(WF_EINVAL, "no stochastic sweep for this problem");
    int rc = wf_launch_status(ctx, pl, out, st, true);
    if (rc) return rc;
    // A small batch: fewer teams a CTA, so that it spreads over the SMs.
    const int32_t spread = (int32_t)std::max<int64_t>(1, (pl->P + ctx->sms - 1) / ctx->sms);
    if (spread < s.teams) {
        smem -= (size_t)(s.teams - spread) * s.team;
        s.teams = spread;
    }
    auto go = [&](auto q, auto vv) {
        using Q = typename decltype(q)::type;
        constexpr int kV = decltype(vv)::value;
        return tab ? stoch_launch<Q, kV, true>(ctx, s, smem, pl, out, ovf_list, ovf_count, st)
                   : stoch_launch<Q, kV, false>(ctx, s, smem, pl, out, ovf_list, ovf_count, st);
    };
    if (dp.M <= 8) return v == 1 ? go(Ty<uint32_t>{}, Iv<1>{}) : go(Ty<uint32_t>{}, Iv<2>{});
    return v == 1 ? go(Ty<uint64_t>{}, Iv<1>{}) : go(Ty<uint64_t>{}, Iv<2>{});
}

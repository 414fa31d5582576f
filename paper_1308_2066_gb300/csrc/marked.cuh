// marked.cuh -- the analysis stage (Basic Algorithm, Section II-B) over the
// register-rows kernels' rows, reading a row only for the occurrences whose
// event can add to its trial.
//
// Most occurrences add nothing: at 1M events x 16 ELTs of 20,000 entries 73%
// of the events are in no ELT, and the occurrence retention leaves 3% with a
// loss.  Reading a row for each of them is bound by the L1 unit (one line
// lookup per occurrence, about one per SM clock whatever the row's size).
// So the table build marks the events whose occurrence loss is not 0, one
// bit per catalog event (tile_rows.cu; event e's is bit 31 - e % 32 of word
// e / 32, so a rotation by e brings it to the top), and the trial pass looks each occurrence up
// in the marks first, held in shared memory; an unmarked event's loss is 0
// in the same arithmetic, so leaving it out of the sum changes nothing.
//
// Mapping (GB300).  One block of 32 warps per SM, its shared memory the marks
// (a catalog past kMaxMarkWords folds two events onto a bit) and a list of
// ids per warp.  A warp takes a contiguous range of trials and walks a trial
// in passes of up to 512 events:
//   1. every lane holds up to 16 ids, loaded a pass ahead, looks them up in
//      the marks and collects the bits in a mask (two shifts and one
//      shared-memory read per id);
//   2. the marked ids are packed into the list, lane by lane, so the rows are
//      read with full warps however the marks fall;
//   3. the listed events' rows are read, one per lane, and their occurrence
//      losses formed (steps 1 to 3) and summed (step 4).
// A list holds 256 ids (a pass with more marks goes through it in quarters):
// L1 keeps 92 KB beside the marks of a 1M-event catalog, and every
// load in flight, of ids or rows, takes a 128-byte line of it.  (With lists of
// a whole pass, 70 KB, the 2M-event catalog's pass below took 1.69 ms; with
// the ids copied to shared memory by cp.async, 2.46.)
//
// Kahan sums keep the register-rows kernels' order: event i of a trial
// belongs to the lane that holds it there, and that lane adds its events'
// losses in order, from the list, once the rows are read: the same sum bit
// for bit.  The other sums are exact (fixed.cuh), in any order; marked ids
// left over are carried from pass to pass of a trial until 32 fill a warp.
//
// At 1M trials x 1000 events x 16 ELTs of 20,000 entries: Kahan sums 0.89 ms
// (every row 3.48), FP64 0.86 (3.79); 400,000 ragged trials over a 2M-event
// catalog without terms, FP64 sums of FP32 losses: 0.96 ms (1.69).  What is
// left is the L1 data pipe, 75-80% busy: 32 random words of the marks take
// 3.5 of its cycles (bank conflicts), 0.4 ms of a paper-scale pass; then the
// id stream, 0.6 ms at the copy bandwidth.
#pragma once

#include <cuda_runtime.h>

#include <string>
#include <type_traits>

#include "are_internal.cuh"
#include "fixed.cuh"
#include "rows.cuh"

namespace are {
namespace marked {

using rows::kFull;

// Warps of a block: 32 leave 64 registers a thread, which the exact sums and
// the ragged walk spill; 28 leave 72.  1M trials x 1000 events x 16 ELTs:
// Kahan sums 0.89 ms with 32 and 0.94 with 28, FP64 0.91 and 0.86 (24: 0.93).
constexpr int kMaxWarps = 32;
__host__ __device__ constexpr int pass_warps(bool kahan, bool fixed) { return kahan && fixed ? 32 : 28; }
constexpr int kSlots = 16;                       // ids per lane and pass
constexpr int kPass = 32 * kSlots;               // events per pass
constexpr int kList = 256;                       // at least fewer than 32 carried ids and a quarter of a pass
// The most marks: with the lists they leave L1 60 KB of the SM's 256.
constexpr size_t kMarkSmem = 195 * 1024;
static_assert(sizeof(uint32_t) * ((size_t)kMaxMarkWords + kMaxWarps * kList) <= kMarkSmem, "marks and lists fit");
static_assert(kList >= 31 + kPass / 4, "a quarter of a pass fits the list");

// ---------------------------------------------------------------------------
// an event's occurrence loss by one lane, in the arithmetic and order of the
// register-rows bodies (rows.cuh)
// ---------------------------------------------------------------------------

// Dense FP32 rows of JP = 8 or 16 terms.
template <int JP>
struct DenseF32 {
    static constexpr bool PACKED = false;
    static constexpr int R = JP / 8;             // lanes a row takes in the register-rows kernel
    using Occ = float;
    const float *table;
    float occ_r, occ_l;
    struct Row {
        rows::F8 v[R];
    };
    __device__ __forceinline__ Row load(uint32_t e) const
    {
        Row r;
#pragma unroll
        for (int i = 0; i < R; ++i) r.v[i] = rows::load8(table + (size_t)e * JP + i * 8);
        return r;
    }
    __device__ __forceinline__ float loss(const Row &r, uint32_t) const
    {
        float g = rows::sum8(r.v[0]);
        if constexpr (R == 2) g = __fadd_rn(g, rows::sum8(r.v[1]));
        return fminf(fmaxf(__fsub_rn(g, occ_r), 0.f), occ_l);
    }
};

// Packed FP32 rows of PW = 8 or 16 words (the format above
// rows::BodyPackedF32).
template <int PW>
struct PackedF32 {
    static constexpr bool PACKED = true;
    static constexpr int R = PW / 8, SLOTS = PW - 1;
    using Occ = float;
    const float *table;
    const float *ovf;
    float occ_r, occ_l;
    struct Row {
        rows::F8 v[R];
    };
    __device__ __forceinline__ Row load(uint32_t e) const
    {
        Row r;
#pragma unroll
        for (int i = 0; i < R; ++i) r.v[i] = rows::load8(table + (size_t)e * PW + i * 8);
        return r;
    }
    __device__ __forceinline__ float loss(Row r, uint32_t e) const
    {
        const int cnt = __popc(__float_as_uint(r.v[0].v[0]));
        r.v[0].v[0] = 0.f;
        float g = rows::sum8(r.v[0]);
        if constexpr (R == 2) g = __fadd_rn(g, rows::sum8(r.v[1]));
        if (cnt > SLOTS) {   // rare: the inline terms, then the rest from the overflow
            const uint32_t *w = reinterpret_cast<const uint32_t *>(table) + (size_t)e * PW;
            float t = 0.f;
            for (int i = 1; i < SLOTS; ++i) t = __fadd_rn(t, __uint_as_float(__ldg(w + i)));
            const float *o = ovf + __ldg(w + SLOTS);
            for (int i = 0; i < cnt - (SLOTS - 1); ++i) t = __fadd_rn(t, __ldg(o + i));
            g = t;
        }
        return fminf(fmaxf(__fsub_rn(g, occ_r), 0.f), occ_l);
    }
};

// Packed FP64 rows of RW = 4 or 8 words (the format above rows::BodyP64):
// the oracle's occurrence loss bit for bit.
template <int RW>
struct PackedF64 {
    static constexpr int R = 1, CAP = RW - 1;
    using Occ = double;
    const unsigned long long *table;
    const double *ovf;
    double occ_r, occ_l;
    struct Row {
        rows::W4 v;              // the mask and the first three terms
    };
    __device__ __forceinline__ Row load(uint32_t e) const { return Row{rows::load4w(table + (size_t)e * RW)}; }
    __device__ __forceinline__ double loss(const Row &r, uint32_t e) const
    {
        const unsigned long long h = r.v.w[0];
        const int cnt = __popc((uint32_t)h);
        double g = rows::dbl(r.v.w[1]);
        if (cnt >= 2) g = rows::vadd(g, rows::dbl(r.v.w[2]));
        if (cnt >= 3) {
            const unsigned long long *w = table + (size_t)e * RW;
            const double *o = ovf + (uint32_t)(h >> 32);
            for (int i = 2; i < cnt; ++i)
                g = rows::vadd(g, cnt <= CAP || i < CAP ? rows::dbl(__ldg(w + 1 + i)) : __ldg(o + i));
        }
        double out = 0.0;
        if (rows::bits(g) > rows::bits(occ_r)) {
            const unsigned long long d = rows::bits(rows::vsub(g, occ_r));
            out = rows::dbl(d < rows::bits(occ_l) ? d : rows::bits(occ_l));
        }
        return out;
    }
};

// An occurrence loss x >= 0 as a fixed-point integer (fixed.cuh); a float on
// the integer pipes alone.
__device__ __forceinline__ void to_fixed(double x, int s, unsigned long long &lo, unsigned long long &hi)
{
    fixed::to_fixed(x, s, lo, hi);
}
__device__ __forceinline__ void to_fixed(float x, int s, unsigned long long &lo, unsigned long long &hi)
{
    const uint32_t u = __float_as_uint(x);
    const int be = (int)(u >> 23);
    const uint32_t m = be ? (u & 0x7fffffu) | 0x800000u : u;
    fixed::shifted(m, (be ? be : 1) - 150 + s, lo, hi);   // x * 2^s = m * 2^(e + s)
}

// ---------------------------------------------------------------------------
// the trial pass
// ---------------------------------------------------------------------------

struct PassArgs {
    rows::Trials t;
    const uint32_t *marks;   // words (a multiple of 4), one bit per catalog event, folded past `bits`
    int32_t words;
    uint32_t bits;           // FOLD: events at and past this one share the bits from 0 on
    int32_t scale;           // fixed-point scale of the exact sums
    int64_t n_trials;
};

// Where a warp is in its trials: the pass at hand starts at id p of trial t
// (numbered from the warp's first), which has `left` more events.  A trial's
// ids follow the one before, so only the lengths of ragged trials are read:
// lane i holds that of trial w + i of a window of 32 trials.
template <bool FIXED>
struct Walk {
    using Count = typename std::conditional<FIXED, int32_t, int64_t>::type;
    const int32_t *p;
    const int64_t *off;      // of the warp's first trial
    Count left, len;         // len: FIXED: events per trial
    int32_t t = 0, n;

    __device__ __forceinline__ Walk(const rows::Trials &a, int64_t t0, int64_t t1, int lane) : n((int32_t)(t1 - t0))
    {
        const int64_t first = a.trial_begin + t0;
        if constexpr (FIXED) {
            p = a.ids + first * a.k;
            off = nullptr;
            len = left = a.k;
        } else {
            off = a.off + first;
            p = a.ids + __ldg(off);
            len = 0;
            trial(lane);
        }
    }
    __device__ __forceinline__ void trial(int lane)
    {
        if constexpr (FIXED) {
            left = len;
        } else {
            if ((t & 31) == 0) len = t + lane < n ? __ldg(off + t + lane + 1) - __ldg(off + t + lane) : 0;
            left = __shfl_sync(kFull, len, t & 31);
        }
    }
    // Events of the pass at hand (0: a trial without events).
    __device__ __forceinline__ int count() const { return left < kPass ? (int)left : kPass; }
    __device__ __forceinline__ bool last() const { return left <= kPass; }
    __device__ __forceinline__ void next(int cnt, int lane)
    {
        p += cnt;
        left -= cnt;
        if (left == 0) {
            ++t;
            if (t < n) trial(lane);
        }
    }
};

// The pass's ids, slot u the event 32 u + at of the pass, in quarters as far
// as the pass reaches.  Slots past the pass hold ids of the events after it
// (their marks are masked out), or 0 where a quarter might end past the ids
// (`whole` false).
__device__ __forceinline__ void load_ids(uint32_t (&id)[kSlots], const int32_t *p, int cnt, int at, bool whole)
{
    p += at;
    if (whole) {
#pragma unroll
        for (int q = 0; q < kSlots / 4; ++q)
            if (q * 128 < cnt) {
#pragma unroll
                for (int u = 4 * q; u < 4 * q + 4; ++u) id[u] = (uint32_t)__ldcs(p + 32 * u);
            }
    } else {
#pragma unroll
        for (int u = 0; u < kSlots; ++u) id[u] = 32 * u + at < cnt ? (uint32_t)__ldcs(p + 32 * u) : 0u;
    }
}

// Whether quarters of a pass may be read past the last event of the warp's
// trials (up to t1): where the ids reach that far (to the end of the launch's
// range, and kIdPad further).
template <bool FIXED>
__device__ __forceinline__ bool whole_quarters(const PassArgs &a, int64_t t1)
{
    const int64_t end = a.t.trial_begin + a.n_trials, own = a.t.trial_begin + t1;
    return (FIXED ? (end - own) * (int64_t)a.t.k : __ldg(a.t.off + end) - __ldg(a.t.off + own)) + kIdPad >= 128;
}

// The marks of the lane's ids in a pass of cnt events, bit u for slot u (the
// event 32 u + at).
template <bool FOLD>
__device__ __forceinline__ uint32_t marks_of(const uint32_t (&id)[kSlots], const uint32_t *marks, uint32_t bits, int cnt,
                                             int at)
{
    uint32_t mask = 0;
#pragma unroll
    for (int q = kSlots / 4 - 1; q >= 0; --q)
        if (q * 128 < cnt) {
#pragma unroll
            for (int u = 4 * q + 3; u >= 4 * q; --u) {
                const uint32_t e = FOLD ? min(id[u], id[u] - bits) : id[u];
                const uint32_t word = marks[e >> 5];
                mask = __funnelshift_l(__funnelshift_l(word, word, e), mask, 1);
            }
        }
    const int mine = cnt > at ? (cnt - at + 31) >> 5 : 0;   // the lane's events in the pass
    return mask & ((1u << mine) - 1u);
}

// Where a lane's n <= 16 entries start in the warp's list of them all, lane
// by lane, and their total: from the bits of the counts by ballots (shuffles
// would take turns with the shared-memory reads).
__device__ __forceinline__ void offsets(uint32_t n, uint32_t &before, uint32_t &total)
{
    uint32_t lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    before = 0;
    total = 0;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const unsigned v = __ballot_sync(kFull, (n >> b) & 1u);
        before += (uint32_t)__popc(v & lt) << b;
        total += (uint32_t)__popc(v) << b;
    }
    if (__any_sync(kFull, n > 3u)) {
#pragma unroll
        for (int b = 2; b < 5; ++b) {
            const unsigned v = __ballot_sync(kFull, (n >> b) & 1u);
            before += (uint32_t)__popc(v & lt) << b;
            total += (uint32_t)__popc(v) << b;
        }
    }
}

// The trials' totals: a lane's sum of each trial goes in, and each 32 trials'
// losses are written together (rows::end_trial).
//
// Kahan pairs: the lanes merge as rows::SumKahan::warp_merge does, two trials
// at a time: from the first step on, half the lanes work for each (a merge
// gives both its lanes the same pair).
template <int ACC>
struct Totals {
    float s = 0.f, c = 0.f;      // the lane's sum of the even trial before an odd one
    float ks = 0.f, kc = 0.f;    // the totals of 32 trials, one per lane
    __device__ __forceinline__ static void merge(float &s, float &c, float s2, float c2)
    {
        const float t = __fadd_rn(s, s2);
        const float bp = __fsub_rn(t, s);
        const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
        c = __fsub_rn(__fadd_rn(c, c2), err);
        s = t;
    }
    __device__ __forceinline__ void end(const rows::SumKahan &x, int32_t t, bool done, int lane, const PassArgs &a,
                                        double *ylt)
    {
        const bool odd = (t & 1) != 0;
        if (!odd && !done) {
            s = x.s;
            c = x.c;
            return;
        }
        // lanes 0 .. 15: the even trial, 16 .. 31: the odd one (or, with
        // `done` on an even trial, that trial and nothing)
        const bool up = (lane & 16) != 0;
        const float s0 = odd ? s : x.s, c0 = odd ? c : x.c, s1 = x.s, c1 = x.c;
        float v = up ? s1 : s0, w = up ? c1 : c0;
        merge(v, w, __shfl_xor_sync(kFull, up ? s0 : s1, 16), __shfl_xor_sync(kFull, up ? c0 : c1, 16));
#pragma unroll
        for (int m = 8; m > 0; m >>= 1)
            merge(v, w, __shfl_xor_sync(kFull, v, m), __shfl_xor_sync(kFull, w, m));
        const int slot = t & 31;
        const float gs = __shfl_sync(kFull, v, (lane & 1) << 4), gc = __shfl_sync(kFull, w, (lane & 1) << 4);
        if (lane >> 1 == slot >> 1) {
            ks = gs;
            kc = gc;
        }
        if (slot == 31 || done)
            if (lane <= slot)
                ylt[t - slot + lane] = rows::clamp_d(__dsub_rn((double)ks, (double)kc), a.t.agg_r, a.t.agg_l);
    }
};

// Exact sums: six 27-bit limbs, each summed over the lanes by one redux (32
// lanes' limbs sum below 2^32); a trial's limb sums stay with its lane.
template <>
struct Totals<ARE_FP64> {
    uint32_t k[6];
    __device__ __forceinline__ void end(const rows::SumFixed &x, int32_t t, bool done, int lane, const PassArgs &a,
                                        double *ylt)
    {
        constexpr uint32_t M = (1u << 27) - 1u;
        const unsigned long long lo = x.a.lo, hi = x.a.hi;
        const uint32_t limb[6] = {(uint32_t)lo & M,
                                  (uint32_t)(lo >> 27) & M,
                                  (uint32_t)((lo >> 54) | (hi << 10)) & M,
                                  (uint32_t)(hi >> 17) & M,
                                  (uint32_t)((hi >> 44) | ((unsigned long long)x.a.top << 20)) & M,
                                  x.a.top >> 7};
        const int slot = t & 31;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const uint32_t r = __reduce_add_sync(kFull, limb[i]);
            if (lane == slot) k[i] = r;
        }
        if (slot == 31 || done)
            if (lane <= slot) {
                fixed::Acc s;
                s.lo = k[0];
                s.add((unsigned long long)k[1] << 27, 0, 0);
                s.add((unsigned long long)k[2] << 54, k[2] >> 10, 0);
                s.add(0, (unsigned long long)k[3] << 17, 0);
                s.add(0, (unsigned long long)k[4] << 44, k[4] >> 20);
                s.top += k[5] << 7;
                ylt[t - slot + lane] = rows::clamp_d(fixed::to_double(s, a.scale), a.t.agg_r, a.t.agg_l);
            }
    }
};

// Kahan sums in the register-rows kernels' order (ACC = ARE_FP32_KAHAN), or
// exact sums (ARE_FP64).
template <typename Rows, int ACC, bool FIXED, bool FOLD>
__global__ void __launch_bounds__(32 * pass_warps(ACC == ARE_FP32_KAHAN, FIXED), 1)
    k_marked(const PassArgs a, const Rows rows_)
{
    constexpr bool KAHAN = ACC == ARE_FP32_KAHAN;
    constexpr int kWarps = pass_warps(KAHAN, FIXED), kThreads = 32 * kWarps;
    constexpr int R = KAHAN ? Rows::R : 1, RPW = 32 / R;
    using Sum = typename std::conditional<KAHAN, rows::SumKahan, rows::SumFixed>::type;
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t *bm = smem;
    uint32_t *list = smem + a.words + wib * kList;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.marks);
        uint4 *dst = reinterpret_cast<uint4 *>(smem);
        for (int i = threadIdx.x; i < a.words / 4; i += kThreads) dst[i] = __ldg(src + i);
        __syncthreads();
    }
    const int64_t nw = (int64_t)gridDim.x * kWarps, w = (int64_t)blockIdx.x * kWarps + wib;
    const int64_t t0 = w * a.n_trials / nw, t1 = (w + 1) * a.n_trials / nw;
    if (t0 >= t1) return;
    const bool whole = whole_quarters<FIXED>(a, t1);
    const int at = (lane % R) * RPW + lane / R;   // the lane's event of each group of 32
    double *const ylt = a.t.ylt + t0;

    Sum acc;
    Totals<ACC> totals;
    uint32_t have = 0;                            // listed ids not yet read
    uint32_t held = 0, held_at = 0;               // Kahan: the lane's marks of the pass they are from, and their place
    auto add = [&](typename Rows::Occ o) {        // exact sums
        if constexpr (!KAHAN) {
            if (o != 0) {
                unsigned long long lo, hi;
                to_fixed(o, a.scale, lo, hi);
                acc.a.add(lo, hi, 0u);
            }
        }
    };

    Walk<FIXED> walk(a.t, t0, t1, lane);
    uint32_t id[kSlots];
    load_ids(id, walk.p, walk.count(), at, whole);
    for (bool more = true; more;) {
        const int cnt = walk.count();
        const int32_t tc = walk.t;
        const bool last = walk.last();
        const uint32_t mask = marks_of<FOLD>(id, bm, a.bits, cnt, at);   // 1. the marks of the lane's ids
        if constexpr (KAHAN)
            if (have == 0 && cnt > 0 && !(mask & 1u) && acc.c != 0.f) acc.add(0.f);   // (a later pass's slot 0)
        uint32_t m = mask, before, total;
        offsets(__popc(m), before, total);
        int part = 4;                             // the quarters listed, with this one
        if (have + total > kList) {               // too many marks: a quarter at a time
            part = 1;
            m = mask & 0xfu;
            offsets(__popc(m), before, total);
        }
        while (true) {
            // 2. the marked ids into the list
            const uint32_t first = have + before, n = have + total;
            {
                uint32_t *p = list + first;
#pragma unroll
                for (int q = 0; q < kSlots / 4; ++q)
                    if (q * 128 < cnt) {
#pragma unroll
                        for (int u = 4 * q; u < 4 * q + 4; ++u)
                            if (m & (1u << u)) *p++ = id[u];
                    }
            }
            if (part == 4) {   // the next pass's ids are on their way while this one's rows are read
                walk.next(cnt, lane);
                more = walk.t < walk.n;
                if (more) load_ids(id, walk.p, walk.count(), at, whole);
            }
            __syncwarp();
            // 3. the listed events' rows and losses
            if constexpr (KAHAN) {
                // few marks: they wait for the trial's next pass, which lists
                // at least a quarter of a pass at a time
                if (!last && have == 0 && part == 4 && n <= kList - kPass / 4) {
                    held = m;
                    held_at = first;
                    have = n;
                    break;
                }
                // the loss in the id's place, then the lane's own in order
                for (uint32_t j = lane; j < n; j += 32) {
                    const uint32_t e = list[j];
                    list[j] = __float_as_uint(rows_.loss(rows_.load(e), e));
                }
                __syncwarp();
                // The sum as the register-rows kernel forms it: an unmarked
                // event adds a 0, which leaves s - c as it is but may round s
                // again (once: a second 0 changes nothing, and none does while
                // c is 0), and so do the slots past the trial of its last
                // group of 32.  (That is the register-rows kernels' default,
                // one group per batch.  Two pad an odd number of groups with
                // one more 0: the same sum in another pair, whose merge may
                // round its last bits otherwise.)  Bits 0 .. 15: the pass that
                // waited.
                const int slots = kSlots + ((cnt + 31) >> 5);
                const uint32_t all = mask << kSlots | held;
                const uint32_t skip = first - held_at - __popc(held);
                uint32_t i = held_at;
                for (uint32_t d = m << kSlots | held; d; d &= d - 1) {
                    const int u = __ffs(d);
                    acc.add(__uint_as_float(list[u > kSlots ? i + skip : i]));
                    ++i;
                    if (acc.c != 0.f && u < slots && !((all >> u) & 1u)) acc.add(0.f);
                }
                held = held_at = have = 0;
            } else {
                have = n;
                while (have >= 32) {
                    have -= 32;
                    const uint32_t e = list[have + lane];
                    add(rows_.loss(rows_.load(e), e));
                }
                if (last && part == 4) {
                    if (lane < have) {
                        const uint32_t e = list[lane];
                        add(rows_.loss(rows_.load(e), e));
                    }
                    have = 0;
                }
            }
            __syncwarp();
            if (part == 4) break;
            m = mask & (0xfu << (4 * part));
            ++part;
            offsets(__popc(m), before, total);
        }
        if (last) {
            totals.end(acc, tc, !more, lane, a, ylt);
            acc = Sum{};
        }
    }
}

template <typename Rows, int ACC, bool FIXED, bool FOLD>
void launch_pass_t(const PassArgs &a, const Rows &rows_, int num_sms, cudaStream_t s)
{
    constexpr int warps = pass_warps(ACC == ARE_FP32_KAHAN, FIXED);
    auto kern = k_marked<Rows, ACC, FIXED, FOLD>;
    fit_blocks(reinterpret_cast<const void *>(kern), 32 * warps, kMarkSmem);   // raises the shared-memory limit
    const size_t smem = sizeof(uint32_t) * ((size_t)a.words + warps * kList);
    const int64_t blocks = a.n_trials < num_sms ? a.n_trials : num_sms;
    kern<<<(unsigned)blocks, 32 * warps, smem, s>>>(a, rows_);
    ARE_CUDA_TRY(cudaGetLastError());
}

inline PassArgs pass_args(const SimArgs &a, const MarkMap &m, int scale)
{
    PassArgs p;
    p.t.ids = a.ids;
    p.t.off = a.off;
    p.t.k = a.k;
    p.t.trial_begin = a.trial_begin;
    p.t.ylt = a.ylt;
    p.t.agg_r = a.agg_r;
    p.t.agg_l = a.agg_l;
    p.marks = m.d;
    p.words = m.words;
    p.bits = m.bits;
    p.scale = scale;
    p.n_trials = a.n_trials;
    return p;
}

// fn(rows) for the layer's FP32 rows: packed rows of 8 or 16 words with their
// overflow terms, or dense rows of 8 or 16 terms.
template <typename F>
auto with_rows32(const void *table, const void *ovf, bool packed, int row_words, const TermsF32 &tm, F &&fn)
{
    auto go = [&](auto r) {
        r.table = static_cast<const float *>(table);
        if constexpr (decltype(r)::PACKED) r.ovf = static_cast<const float *>(ovf);
        r.occ_r = tm.occ_r;
        r.occ_l = tm.occ_l;
        return fn(r);
    };
    if (packed && row_words == 8) return go(PackedF32<8>{});
    if (packed && row_words == 16) return go(PackedF32<16>{});
    if (!packed && row_words == 8) return go(DenseF32<8>{});
    if (!packed && row_words == 16) return go(DenseF32<16>{});
    throw Error{ARE_EINVAL, "no marked FP32 rows of " + std::to_string(row_words) + " words"};
}

// fn(rows) for the layer's packed FP64 rows of 4 or 8 words.
template <typename F>
auto with_rows64(const void *table, const void *ovf, int row_words, const TermsF64 &tm, F &&fn)
{
    auto go = [&](auto r) {
        r.table = static_cast<const unsigned long long *>(table);
        r.ovf = static_cast<const double *>(ovf);
        r.occ_r = tm.occ_r;
        r.occ_l = tm.occ_l;
        return fn(r);
    };
    if (row_words == 4) return go(PackedF64<4>{});
    if (row_words == 8) return go(PackedF64<8>{});
    throw Error{ARE_EINVAL, "no marked FP64 rows of " + std::to_string(row_words) + " words"};
}

template <typename Rows, int ACC>
void launch_pass(const SimArgs &a, const MarkMap &m, const Rows &rows_, int scale, int num_sms, cudaStream_t s)
{
    const PassArgs p = pass_args(a, m, scale);
    if (a.off)
        m.fold ? launch_pass_t<Rows, ACC, false, true>(p, rows_, num_sms, s)
               : launch_pass_t<Rows, ACC, false, false>(p, rows_, num_sms, s);
    else
        m.fold ? launch_pass_t<Rows, ACC, true, true>(p, rows_, num_sms, s)
               : launch_pass_t<Rows, ACC, true, false>(p, rows_, num_sms, s);
}

}  // namespace marked
}  // namespace are

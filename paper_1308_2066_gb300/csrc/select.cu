// select.cu -- filters on the YLT (Section II-C): PML and TVaR.
//
// The paper names PML and TVaR (Section I) without defining them; the
// library reads PML at return period RP as the m-th largest trial loss,
// m = ceil(N / RP), and TVaR at level a as the mean of the m = ceil(N(1-a))
// largest.  Both need only the m-th largest value and the sum of the values
// above it, so no sort is done: an MSB-first radix select over an
// order-preserving 64-bit key of each double finds the m-th largest key
// exactly (8 passes of 8 bits, every target rank in the same pass), then one
// more pass adds the values above it.
//
// Two forms.  are_risk_measures, the batched call and the pricing server run
// one cooperative launch that counts 13 and 11 bits and finishes on the few
// keys left (details above k_select_coop).  The allocation-free call launches
// the radix passes one kernel at a time.
//
// GB300 choices.  Each histogram pass ends with the pick of the next digit,
// done by whichever block of the pass finishes last (a counter and memory
// fences, no waiting), so a radix selection is 10 launches.  Histogram counts are
// aggregated per warp (lanes with the digit of the warp's first active lane
// add once), since early passes send most values to one or two bins.  The tail sum avoids FP64
// arithmetic, which GB300 issues at a small fraction of its integer rate:
// each value above the selected one is scaled by a power of two taken from
// the largest magnitude of the YLT and added as 32-bit limbs to integer
// accumulators, so the sum is exact, and it is rounded to double once.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <mutex>

#include "are_internal.cuh"

namespace are {
namespace {

namespace cg = cooperative_groups;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kBins = 256;
constexpr int kThreads = 256;
constexpr int kLimbs = 3;                      // 32-bit limbs of one scaled value (< 2^96)
constexpr int kAccWords = 2 * kLimbs + 1;      // per target: positive limbs, negative limbs, count
constexpr int kCtrlWords = 4;                  // blocks arrived, top word of the largest |value|
constexpr int kPre = 8;                        // values a lane loads before it processes them

__device__ __forceinline__ uint64_t key_of(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double value_of(uint64_t k)
{
    const uint64_t b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

struct Ranks {
    long long m[kMaxTargets];
};

// The radix form's YLT and scratch.
struct Sel {
    const double *ylt;
    uint32_t *hist;              // kMaxTargets x 256 counts
    unsigned long long *state;   // kMaxTargets x (key prefix, rank left)
    unsigned int *ctrl;          // kCtrlWords
    unsigned long long *acc;     // kMaxTargets x kAccWords
    double *result;              // kMaxTargets x (m-th largest, mean of the m largest)
    int blocks;                  // blocks of the histogram and tail passes
};

// ---------------------------------------------------------------------------
// multi-word integers
// ---------------------------------------------------------------------------

struct U192 {
    unsigned long long w0 = 0, w1 = 0, w2 = 0;
};
__device__ __forceinline__ void add192(U192 &a, unsigned long long b0, unsigned long long b1,
                                       unsigned long long b2)
{
    asm("add.cc.u64 %0, %0, %3;\n\t"
        "addc.cc.u64 %1, %1, %4;\n\t"
        "addc.u64 %2, %2, %5;"
        : "+l"(a.w0), "+l"(a.w1), "+l"(a.w2)
        : "l"(b0), "l"(b1), "l"(b2));
}
__device__ __forceinline__ void sub192(U192 &a, const U192 &b)
{
    asm("sub.cc.u64 %0, %0, %3;\n\t"
        "subc.cc.u64 %1, %1, %4;\n\t"
        "subc.u64 %2, %2, %5;"
        : "+l"(a.w0), "+l"(a.w1), "+l"(a.w2)
        : "l"(b.w0), "l"(b.w1), "l"(b.w2));
}
__device__ __forceinline__ bool less192(const U192 &a, const U192 &b)
{
    if (a.w2 != b.w2) return a.w2 < b.w2;
    if (a.w1 != b.w1) return a.w1 < b.w1;
    return a.w0 < b.w0;
}

// |x| * 2^s as a 96-bit integer (lo 64 bits, hi 32 bits), rounding half up
// below the last bit; |x| < 2^(95 - s) keeps it below 2^96.
__device__ __forceinline__ void scaled(double x, int s, unsigned long long &lo, unsigned long long &hi)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    const int be = (int)(b >> 52);
    unsigned long long m = b & ((1ull << 52) - 1);
    if (be) m |= 1ull << 52;
    const int sh = (be ? be : 1) - 1075 + s;   // |x| = m * 2^(sh - s)
    lo = 0;
    hi = 0;
    if (sh >= 64) {
        hi = m << (sh - 64);
    } else if (sh > 0) {
        lo = m << sh;
        hi = m >> (64 - sh);
    } else if (sh == 0) {
        lo = m;
    } else if (sh >= -53) {
        const int k = -sh;
        lo = (m >> k) + ((m >> (k - 1)) & 1ull);
    }
}

// a * 2^-s rounded once to the nearest double.
__device__ __forceinline__ double to_double(const U192 &a, int s)
{
    int L;
    if (a.w2) L = 192 - __clzll((long long)a.w2);
    else if (a.w1) L = 128 - __clzll((long long)a.w1);
    else if (a.w0) L = 64 - __clzll((long long)a.w0);
    else return 0.0;
    if (L <= 64) return ldexp(__ull2double_rn(a.w0), -s);
    const int r = L - 64;                      // 1 .. 128
    unsigned long long w, sticky;
    if (r < 64) {
        w = (a.w0 >> r) | (a.w1 << (64 - r));
        sticky = a.w0 & ((1ull << r) - 1);
    } else if (r == 64) {
        w = a.w1;
        sticky = a.w0;
    } else if (r < 128) {
        const int q = r - 64;
        w = (a.w1 >> q) | (a.w2 << (64 - q));
        sticky = a.w0 | (a.w1 & ((1ull << q) - 1));
    } else {
        w = a.w2;
        sticky = a.w0 | a.w1;
    }
    // w has its top bit set and a double keeps 53 of its 64 bits: a sticky
    // bit in bit 0 makes the conversion's one rounding the right one
    return ldexp(__ull2double_rn(w | (sticky ? 1ull : 0ull)), r - s);
}

// Scale of a YLT: s = 95 - floor(log2(largest |value|)), from the top 32
// bits of the largest magnitude's bit pattern.
__device__ __forceinline__ int tail_scale(unsigned int mag_hi)
{
    int e = (int)((mag_hi >> 20) & 0x7ff) - 1023;
    if (e < -1022) e = -1022;
    return 95 - e;
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

// state[2t] = key prefix decided so far, state[2t+1] = rank still to find
// among the keys that share the prefix (1 = the largest of them).
__global__ void k_init(Sel s, Ranks r, int nt)
{
    uint32_t *hist = s.hist;
    unsigned long long *state = s.state, *acc = s.acc;
    for (int i = threadIdx.x; i < nt * kBins; i += blockDim.x) hist[i] = 0;
    for (int i = threadIdx.x; i < nt * kAccWords; i += blockDim.x) acc[i] = 0;
    if (threadIdx.x < kCtrlWords) s.ctrl[threadIdx.x] = 0;
    if (threadIdx.x < nt) {
        state[2 * threadIdx.x] = 0ull;
        state[2 * threadIdx.x + 1] = (unsigned long long)r.m[threadIdx.x];
    }
}

// Adds the lanes with `on` set to bin `bin` of h: the lanes whose bin is the
// first active lane's add once together (the common case: early passes send
// most values to one bin), the others one by one.  Every lane of the warp
// must call it.
__device__ __forceinline__ void hist_add(uint32_t *h, bool on, uint32_t bin, int lane)
{
    const unsigned act = __ballot_sync(kFull, on);
    if (!act) return;
    const int leader = __ffs(act) - 1;
    const uint32_t b0 = __shfl_sync(kFull, bin, leader);
    const unsigned same = __ballot_sync(kFull, on && bin == b0);
    if (lane == leader) atomicAdd(h + b0, (uint32_t)__popc(same));
    else if (on && bin != b0) atomicAdd(h + bin, 1u);
}

// One warp: find the bucket of h (256 counts in global, or SHARED, memory) that holds the wanted rank,
// counting down from the top bucket, and extend the target's prefix.
template <bool SHARED = false>
__device__ __forceinline__ void pick(const uint32_t *h, unsigned long long *st, int shift, int lane)
{
    uint32_t c[8];
    unsigned long long lane_sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t *at = h + kBins - 1 - (lane * 8 + i);   // lane 0 holds the top buckets
        c[i] = SHARED ? *at : __ldcg(at);
        lane_sum += c[i];
    }
    unsigned long long incl = lane_sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long o = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += o;
    }
    const unsigned long long excl = incl - lane_sum;
    const unsigned long long r = st[1];
    if (excl < r && r <= incl) {
        unsigned long long above = excl;
        int b = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (above + c[i] >= r) {
                b = kBins - 1 - (lane * 8 + i);
                break;
            }
            above += c[i];
        }
        st[0] |= (unsigned long long)b << shift;
        st[1] = r - above;
    }
}

// Histogram pass `pass` (digit bits 56 - 8 pass .. 63 - 8 pass) over the keys
// that share each target's prefix; pass 0 counts every key once for all
// targets and records the largest magnitude.  The last block to finish picks
// every target's digit and clears the histogram for the next pass.
__global__ void __launch_bounds__(kThreads) k_hist(Sel s, int64_t n, int nt, int pass)
{
    const double *__restrict__ v = s.ylt;
    unsigned long long *state = s.state;
    uint32_t *hist = s.hist;
    unsigned int *ctrl = s.ctrl;
    __shared__ uint32_t h[kMaxTargets * kBins];
    __shared__ unsigned int s_mag;
    __shared__ int s_last;
    const int rows = pass == 0 ? 1 : nt;
    for (int i = threadIdx.x; i < rows * kBins; i += blockDim.x) h[i] = 0;
    if (threadIdx.x == 0) s_mag = 0;
    const int shift = 56 - 8 * pass;
    uint64_t pre[kMaxTargets];
#pragma unroll
    for (int t = 0; t < kMaxTargets; ++t)   // pass 0 has no prefix yet
        pre[t] = (pass > 0 && t < nt) ? state[2 * t] >> (shift + 8) : 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    unsigned int mag = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform loop: every lane takes part in the warp's histogram adds;
    // kPre values per lane are loaded before the first is counted
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n;
         base += stride * kPre) {
        double xs[kPre];
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            const int64_t i = base + u * stride + lane;
            xs[u] = i < n ? v[i] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            const bool ok = base + u * stride + lane < n;
            const double x = xs[u];
            const uint64_t k = key_of(x);
            const uint32_t d = (uint32_t)(k >> shift) & 0xffu;
            if (pass == 0) {
                hist_add(h, ok, d, lane);
                const unsigned int m32 =
                    (unsigned int)(((unsigned long long)__double_as_longlong(x) >> 32) & 0x7fffffffu);
                mag = m32 > mag ? m32 : mag;
            } else {
#pragma unroll
                for (int t = 0; t < kMaxTargets; ++t) {
                    if (t >= nt) break;
                    hist_add(h + t * kBins, ok && (k >> (shift + 8)) == pre[t], d, lane);
                }
            }
        }
    }
    if (pass == 0) {
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            const unsigned int o = __shfl_xor_sync(kFull, mag, off);
            mag = o > mag ? o : mag;
        }
        if (lane == 0) atomicMax(&s_mag, mag);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < rows * kBins; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
    if (pass == 0 && threadIdx.x == 0 && s_mag) atomicMax(&ctrl[1], s_mag);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctrl[0], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int t = threadIdx.x >> 5;
    if (t < nt) pick(hist + (pass == 0 ? 0 : t) * kBins, state + 2 * t, shift, lane);
    __syncthreads();
    for (int i = threadIdx.x; i < rows * kBins; i += blockDim.x) hist[i] = 0;
    if (threadIdx.x == 0) ctrl[0] = 0;
}

// Tail pass: every value whose key is above a target's selected key is
// added, scaled, to the target's integer accumulators (positive and
// negative values apart) and counted.  The last block to finish forms each
// target's sum of the m largest -- the values above plus (m - count) times
// the selected value -- and writes (value, sum / m).
__global__ void __launch_bounds__(kThreads) k_tail(Sel s, int64_t n, int nt, Ranks r)
{
    const double *__restrict__ v = s.ylt;
    const unsigned long long *state = s.state;
    unsigned int *ctrl = s.ctrl;
    unsigned long long *acc = s.acc;
    __shared__ unsigned long long a[kMaxTargets * kAccWords];
    __shared__ int s_last;
    for (int i = threadIdx.x; i < nt * kAccWords; i += blockDim.x) a[i] = 0;
    uint64_t kt[kMaxTargets];
    uint64_t kmin = ~0ull;
#pragma unroll
    for (int t = 0; t < kMaxTargets; ++t) {
        kt[t] = t < nt ? state[2 * t] : ~0ull;
        kmin = kt[t] < kmin ? kt[t] : kmin;
    }
    const int sc = tail_scale(ctrl[1]);
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += stride * kPre) {
        double xs[kPre];   // kPre values loaded before the first is added
#pragma unroll
        for (int u = 0; u < kPre; ++u) xs[u] = i0 + u * stride < n ? v[i0 + u * stride] : 0.0;
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            if (i0 + u * stride >= n) break;
            const double x = xs[u];
            const uint64_t k = key_of(x);
            if (k > kmin) {
                unsigned long long lo, hi;
                scaled(x, sc, lo, hi);
                const int sign = x < 0.0 ? kLimbs : 0;
                const unsigned long long l0 = lo & 0xffffffffull, l1 = lo >> 32, l2 = hi;
#pragma unroll
                for (int t = 0; t < kMaxTargets; ++t) {
                    if (t < nt && k > kt[t]) {
                        unsigned long long *p = a + t * kAccWords;
                        atomicAdd(p + sign, l0);
                        atomicAdd(p + sign + 1, l1);
                        atomicAdd(p + sign + 2, l2);
                        atomicAdd(p + 2 * kLimbs, 1ull);
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nt * kAccWords; i += blockDim.x)
        if (a[i]) atomicAdd(&acc[i], a[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctrl[0], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x < nt) {
        const int t = threadIdx.x;
        const unsigned long long *p = acc + t * kAccWords;
        U192 pos, neg;
        // limb sums -> 192-bit integers: sum_l A_l * 2^(32 l)
        for (int g = 0; g < 2; ++g) {
            U192 &z = g ? neg : pos;
            const unsigned long long A0 = __ldcg(p + g * kLimbs), A1 = __ldcg(p + g * kLimbs + 1),
                                     A2 = __ldcg(p + g * kLimbs + 2);
            add192(z, A0, 0, 0);
            add192(z, A1 << 32, A1 >> 32, 0);
            add192(z, 0, A2, 0);
        }
        const unsigned long long c = __ldcg(p + 2 * kLimbs);
        const double vt = value_of(kt[t]);
        const unsigned long long q = (unsigned long long)r.m[t] - c;   // >= 1: ties at the m-th value
        unsigned long long lo, hi;
        scaled(vt, sc, lo, hi);
        U192 &z = vt < 0.0 ? neg : pos;
        // (hi:lo) * q with hi < 2^32 and q < 2^32
        add192(z, lo * q, __umul64hi(lo, q), 0);
        add192(z, 0, hi * q, __umul64hi(hi, q));
        double sum;
        if (less192(pos, neg)) {
            sub192(neg, pos);
            sum = -to_double(neg, sc);
        } else {
            sub192(pos, neg);
            sum = to_double(pos, sc);
        }
        double *res = s.result;
        res[2 * t] = vt;
        res[2 * t + 1] = __ddiv_rn(sum, (double)r.m[t]);
    }
    if (threadIdx.x == 0) ctrl[0] = 0;
}

// ---------------------------------------------------------------------------
// The selection in one cooperative launch
// ---------------------------------------------------------------------------
//
// One kernel whose blocks are all resident (a cooperative launch), with a
// grid-wide barrier where the radix form has a launch boundary.  The blocks
// form groups, one YLT to a group at a time:
// A. the top 13 key bits (sign, exponent and a mantissa bit: half an octave)
//    counted in 8192 bins; every block finds every target's bin itself;
// B. the next 11 bits of the targets' bins (2^-12 of an octave) counted;
// C. the keys of each target's 24-bit bin kept, up to kCand of them with
//    their multiplicities (a run of ties is one key: each block counts the
//    first candidate it meets apart), and the values of higher bins added to
//    the exact tail sums of the targets that want a mean;
// D. a block per target finds the key among the kept ones and adds those above
//    it.  If some bin keeps more than kCand keys, five radix passes over the
//    whole YLT take the place of D.
// Three barriers, where eight 8-bit digits would need eight; the bins are
// narrow enough that D is a few dozen keys.
//
// Three targets of 1M losses take 43 us (two 8-bit digits and up to 16384
// kept keys: 83), eight 78 us (302), eight with a run of ties of 2% 79 us
// (463: it took the radix passes); 1000 losses 18 us in one block (34); 64 YLTs
// of 100,000 at a time 360 us (ten launches: 549).  What is left is latency:
// the launch, three barriers and the chains between them.
//
// The scratch of a group is left ready for the next YLT: histogram A is
// cleared in C (its readers are past the barrier before), histogram B in A and
// the counters and sums of C and D in B (their readers are past a barrier and
// their next writers behind one), the magnitudes by turns.

constexpr int kCand = 1024;             // keys kept per target
constexpr int kCoopThreads = 1024;
constexpr int kBitsA = 13, kBinsA = 1 << kBitsA;
constexpr int kBitsB = 11, kBinsB = 1 << kBitsB;
constexpr int kShiftA = 64 - kBitsA, kShiftB = kShiftA - kBitsB;
static_assert(kShiftB == 40, "the radix passes go on with the fourth digit of 8 bits");
constexpr size_t kCoopSmem = sizeof(uint32_t) * kMaxTargets * kBinsB;
constexpr int64_t kOneBlock = 8192;     // values that one block selects from by itself: 8 a thread
static_assert(kCoopSmem >= sizeof(uint32_t) * kBinsA && kCoopSmem >= kCand * 12ull, "what the passes share");

// One group's scratch, zero before its first use.
struct CoopScratch {
    uint32_t a[kBinsA];
    uint32_t b[kMaxTargets * kBinsB];
    uint32_t c[3 * kMaxTargets * kBins];             // the radix passes'
    unsigned long long acc[kMaxTargets * kAccWords];
    unsigned long long key[kMaxTargets * kCand];
    uint32_t times[kMaxTargets * kCand];
    uint32_t kept[kMaxTargets];
    unsigned int mag[2];                             // top word of the largest |value|, by turns
    unsigned int over[2];                            // the launch's (first group): a bin over kCand
    double result[2 * kMaxTargets];                  // value, mean of the m largest
};

struct CoopArgs {
    const double *single;        // the YLT when there is one
    const double *const *many;   // device array of YLT pointers, or nullptr
    int n_ylt;
    int per;                     // blocks of a group
    int64_t n;
    int nt;
    uint32_t means;              // bit t: target t's mean is wanted
    long long m[kMaxTargets];
    CoopScratch *scratch;        // per group
    double *results;             // per YLT: 2 * kMaxTargets, or nullptr: the scratch's
    double *out[kMaxTargets];    // per target: where its value (or, means: its mean) goes too, or nullptr
};

// Adds `times` x (scaled by 2^sc) to the accumulator words a (positive and
// negative limbs apart, then a count) in shared memory for the lanes with
// `on` set: few lanes one by one, many summed over the warp first.  Every lane
// must call it.
__device__ __forceinline__ void acc_add(unsigned long long *a, bool on, double x, uint32_t times, int sc, int lane)
{
    const unsigned act = __ballot_sync(kFull, on);
    if (!act) return;
    unsigned long long lo = 0, hi = 0;
    if (on) scaled(x, sc, lo, hi);
    const unsigned long long w[kLimbs] = {(lo & 0xffffffffull) * times, (lo >> 32) * times, hi * times};
    if (__popc(act) <= 4) {
        if (on) {
            unsigned long long *p = a + (x < 0.0 ? kLimbs : 0);
#pragma unroll
            for (int i = 0; i < kLimbs; ++i) atomicAdd(p + i, w[i]);
            atomicAdd(a + 2 * kLimbs, (unsigned long long)times);
        }
        return;
    }
    for (int g = 0; g < 2; ++g) {   // positive, then negative values
        const bool mine = on && ((x < 0.0) == (g == 1));
        if (!__any_sync(kFull, mine)) continue;
        unsigned long long v[kLimbs + 1];
#pragma unroll
        for (int i = 0; i < kLimbs; ++i) v[i] = mine ? w[i] : 0;
        v[kLimbs] = mine ? times : 0;
#pragma unroll
        for (int off = 16; off; off >>= 1)
#pragma unroll
            for (int i = 0; i <= kLimbs; ++i) v[i] += __shfl_xor_sync(kFull, v[i], off);
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < kLimbs; ++i) atomicAdd(a + g * kLimbs + i, v[i]);
            atomicAdd(a + 2 * kLimbs, v[kLimbs]);
        }
    }
}

// (value of key kt, mean of the m largest) from the accumulator words A of
// the values above kt (sum and count, scaled by 2^sc).
__device__ void tail_result(const unsigned long long (&A)[kAccWords], uint64_t kt, long long m, int sc, bool mean,
                            double *res)
{
    const double vt = value_of(kt);
    res[0] = vt;
    if (!mean) return;
    U192 pos, neg;
    for (int g = 0; g < 2; ++g) {
        U192 &z = g ? neg : pos;
        const unsigned long long A0 = A[g * kLimbs], A1 = A[g * kLimbs + 1], A2 = A[g * kLimbs + 2];
        add192(z, A0, 0, 0);
        add192(z, A1 << 32, A1 >> 32, 0);
        add192(z, 0, A2, 0);
    }
    const unsigned long long c = A[2 * kLimbs];
    const unsigned long long q = (unsigned long long)m - c;   // >= 1: ties at the m-th value
    unsigned long long lo, hi;
    scaled(vt, sc, lo, hi);
    U192 &z = vt < 0.0 ? neg : pos;
    add192(z, lo * q, __umul64hi(lo, q), 0);
    add192(z, 0, hi * q, __umul64hi(hi, q));
    double sum;
    if (less192(pos, neg)) {
        sub192(neg, pos);
        sum = -to_double(neg, sc);
    } else {
        sub192(pos, neg);
        sum = to_double(pos, sc);
    }
    res[1] = __ddiv_rn(sum, (double)m);
}

// Calls f(key, value, in range) for the group's share of the YLT, whole warps
// at a time, kPre values per lane loaded before the first call.
template <typename F>
__device__ __forceinline__ void for_values(const double *v, int64_t n, int rank, int per, F &&f)
{
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)per * kCoopThreads;
    for (int64_t base = (int64_t)rank * kCoopThreads + (threadIdx.x & ~31); base < n; base += stride * kPre) {
        double xs[kPre];
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            const int64_t i = base + u * stride + lane;
            xs[u] = i < n ? v[i] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            if (base + u * stride >= n) break;
            f(key_of(xs[u]), xs[u], base + u * stride + lane < n);
        }
    }
}

// ONE: a single YLT of few values by one block, its counts, sums and keys in
// shared memory and its barriers the block's.
struct KeptKeys {
    unsigned long long key[kMaxTargets * kCand];
    uint32_t times[kMaxTargets * kCand];
    uint32_t kept[kMaxTargets];
    unsigned int over;
};

template <bool ONE>
__global__ void __launch_bounds__(kCoopThreads) k_select_coop(const __grid_constant__ CoopArgs args)
{
    extern __shared__ __align__(16) uint32_t h[];        // kCoopSmem (ONE: and KeptKeys)
    auto barrier = [] {
        if constexpr (ONE) __syncthreads();
        else cg::this_grid().sync();
    };
    __shared__ unsigned long long st[2 * kMaxTargets];   // per target: key prefix, rank left (the same in every block)
    __shared__ unsigned long long acc[kMaxTargets * kAccWords];
    __shared__ uint64_t rep[kMaxTargets];                // per target: the block's first candidate, ~0: none; then its key
    __shared__ uint32_t rep_times[kMaxTargets];
    __shared__ uint32_t warp_sum[kCoopThreads / 32];
    __shared__ unsigned int s_mag;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = ONE ? 1 : args.per, group = blockIdx.x / per, rank = blockIdx.x % per, groups = gridDim.x / per;
    const int nt = args.nt;
    const int64_t n = args.n;
    CoopScratch &S = args.scratch[group];
    KeptKeys &K = *reinterpret_cast<KeptKeys *>(h + kCoopSmem / sizeof(uint32_t));   // ONE
    unsigned long long *const cand_key = ONE ? K.key : S.key;
    uint32_t *const cand_times = ONE ? K.times : S.times, *const kept = ONE ? K.kept : S.kept;
    unsigned int *const over = ONE ? &K.over : args.scratch[0].over;
    // counts and counters of the scratch: past L1 in global memory
    auto get = [](const auto *x) { return ONE ? *x : __ldcg(x); };
    [[maybe_unused]] auto mine = [&](int i) { return i * per + rank; };   // a block's share of the group's clearing
    for (int y0 = 0, round = 0; y0 < args.n_ylt; y0 += groups, ++round) {
        const int y = y0 + group, turn = ONE ? 0 : round & 1;
        const bool on = y < args.n_ylt;
        const bool final_round = y0 + groups >= args.n_ylt;
        const double *__restrict__ v = on ? (args.many ? args.many[y] : args.single) : nullptr;
        // A. the top bits
        if (tid < nt) {
            st[2 * tid] = 0;
            st[2 * tid + 1] = (uint64_t)args.m[tid];
        }
        if (tid == 0) s_mag = 0;
        for (int i = tid; i < kBinsA; i += kCoopThreads) h[i] = 0;
        if constexpr (!ONE)
            for (int i = mine(tid); i < kMaxTargets * kBinsB; i += per * kCoopThreads) S.b[i] = 0;
        if (blockIdx.x == 0 && tid == 0) over[turn] = 0;
        __syncthreads();
        if (on) {
            unsigned int mag = 0;
            for_values(v, n, rank, per, [&](uint64_t k, double x, bool ok) {
                hist_add(h, ok, (uint32_t)(k >> kShiftA), lane);
                const unsigned int m32 =
                    (unsigned int)(((unsigned long long)__double_as_longlong(x) >> 32) & 0x7fffffffu);
                if (ok) mag = m32 > mag ? m32 : mag;
            });
#pragma unroll
            for (int off = 16; off; off >>= 1) {
                const unsigned int o = __shfl_xor_sync(kFull, mag, off);
                mag = o > mag ? o : mag;
            }
            if (lane == 0 && mag) atomicMax(&s_mag, mag);
        }
        __syncthreads();
        if constexpr (!ONE) {
            for (int i = tid; i < kBinsA; i += kCoopThreads)
                if (h[i]) atomicAdd(&S.a[i], h[i]);
            if (tid == 0 && s_mag) atomicMax(&S.mag[turn], s_mag);
            barrier();
        }
        // every block finds every target's bin: thread i holds 8 bins, the
        // top ones first
        {
            constexpr int bins = kBinsA / kCoopThreads;
            const uint32_t *const counts = ONE ? h : S.a;
            uint32_t c[bins], sum = 0;
#pragma unroll
            for (int i = 0; i < bins; ++i) {
                c[i] = get(counts + kBinsA - 1 - (tid * bins + i));
                sum += c[i];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += o;
            }
            if (lane == 31) warp_sum[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                uint32_t s = warp_sum[lane];
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(kFull, s, d);
                    if (lane >= d) s += o;
                }
                warp_sum[lane] = s;
            }
            __syncthreads();
            if (warp) incl += warp_sum[warp - 1];
            const uint32_t excl = incl - sum;
            for (int t = 0; t < nt; ++t) {
                const uint64_t r = (uint64_t)args.m[t];
                if (excl < r && r <= incl) {
                    uint64_t above = excl;
                    int i = 0;
                    while (above + c[i] < r) above += c[i++];
                    st[2 * t] = (uint64_t)(kBinsA - 1 - (tid * bins + i)) << kShiftA;
                    st[2 * t + 1] = r - above;
                }
            }
            __syncthreads();
        }
        // B. the next bits of the targets' bins (a bin shared by targets once)
        for (int i = tid; i < nt * kBinsB; i += kCoopThreads) h[i] = 0;
        if (rank == 0) {
            if constexpr (!ONE)
                for (int i = tid; i < kMaxTargets * kAccWords; i += kCoopThreads) S.acc[i] = 0;
            if (tid < kMaxTargets) kept[tid] = 0;
        }
        __syncthreads();
        uint32_t PA[kMaxTargets];
        int first[kMaxTargets];   // the first target with the same bin
#pragma unroll
        for (int t = 0; t < kMaxTargets; ++t) {
            PA[t] = t < nt ? (uint32_t)(st[2 * t] >> kShiftA) : ~0u;
            first[t] = t;
#pragma unroll
            for (int q = kMaxTargets - 1; q >= 0; --q)
                if (q < t && PA[q] == PA[t]) first[t] = q;
        }
        if (on)
            for_values(v, n, rank, per, [&](uint64_t k, double, bool ok) {
                const uint32_t p = (uint32_t)(k >> kShiftA);
#pragma unroll
                for (int t = 0; t < kMaxTargets; ++t)
                    if (t < nt && first[t] == t)
                        hist_add(h + t * kBinsB, ok && p == PA[t], (uint32_t)(k >> kShiftB) & (kBinsB - 1), lane);
            });
        __syncthreads();
        if constexpr (!ONE) {
            for (int i = tid; i < nt * kBinsB; i += kCoopThreads)
                if (h[i]) atomicAdd(&S.b[i], h[i]);
            barrier();
        }
        if (warp < nt) {   // warp t: lane i holds 64 bins, the top ones first
            int q = 0;
#pragma unroll
            for (int t = 0; t < kMaxTargets; ++t)
                if (t == warp) q = first[t];
            const uint32_t *b = (ONE ? h : S.b) + q * kBinsB;
            constexpr int bins = kBinsB / 32;
            uint32_t sum = 0;
#pragma unroll 32
            for (int i = 0; i < bins; ++i) sum += get(b + kBinsB - 1 - (lane * bins + i));
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += o;
            }
            const uint32_t excl = incl - sum;
            const uint64_t r = st[2 * warp + 1];
            // the lane whose bins hold the rank, then its bins, two per lane
            const int l = __ffs(__ballot_sync(kFull, excl < r && r <= incl)) - 1;
            static_assert(bins == 64, "two bins per lane");
            const uint64_t left = r - __shfl_sync(kFull, excl, l);
            const int i0 = l * bins + 2 * lane;
            const uint32_t c0 = get(b + kBinsB - 1 - i0), c1 = get(b + kBinsB - 2 - i0);
            uint32_t run = c0 + c1;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(kFull, run, d);
                if (lane >= d) run += o;
            }
            const uint32_t before = run - c0 - c1;
            if (before < left && left <= run) {
                const bool second = left > (uint64_t)before + c0;
                st[2 * warp] |= (uint64_t)(kBinsB - 1 - i0 - second) << kShiftB;
                st[2 * warp + 1] = left - before - (second ? c0 : 0u);
            }
        }
        if (tid < kMaxTargets) {
            rep[tid] = ~0ull;
            rep_times[tid] = 0;
        }
        for (int i = tid; i < kMaxTargets * kAccWords; i += kCoopThreads) acc[i] = 0;
        __syncthreads();
        // C. the keys of the targets' bins, and the tail sums above them
        const int sc = tail_scale(ONE ? s_mag : __ldcg(&S.mag[turn]));
        uint32_t P[kMaxTargets];
#pragma unroll
        for (int t = 0; t < kMaxTargets; ++t) {
            P[t] = t < nt ? (uint32_t)(st[2 * t] >> kShiftB) : ~0u;
            first[t] = t;
#pragma unroll
            for (int q = kMaxTargets - 1; q >= 0; --q)
                if (q < t && P[q] == P[t]) first[t] = q;
        }
        auto keep = [&](int t, uint64_t k, uint32_t times) {
            const uint32_t at = atomicAdd(&kept[t], 1u);
            if (at < kCand) {
                cand_key[t * kCand + at] = k;
                cand_times[t * kCand + at] = times;
            }
        };
        if (on)
            for_values(v, n, rank, per, [&](uint64_t k, double x, bool ok) {
                const uint32_t p = (uint32_t)(k >> kShiftB);
#pragma unroll
                for (int t = 0; t < kMaxTargets; ++t) {
                    if (t >= nt) break;
                    if (first[t] == t) {
                        const bool in = ok && p == P[t];
                        if (__any_sync(kFull, in)) {
                            const bool same = in && *(volatile uint64_t *)&rep[t] == k;
                            const unsigned b = __ballot_sync(kFull, same);
                            if (b && lane == __ffs(b) - 1) atomicAdd(&rep_times[t], (uint32_t)__popc(b));
                            if (in && !same) {
                                const uint64_t was = atomicCAS((unsigned long long *)&rep[t], ~0ull, (unsigned long long)k);
                                if (was == ~0ull || was == k) atomicAdd(&rep_times[t], 1u);
                                else keep(t, k, 1u);
                            }
                        }
                    }
                    if ((args.means >> t) & 1u)
                        acc_add(acc + t * kAccWords, ok && p > P[t], x, 1u, sc, lane);
                }
            });
        if constexpr (!ONE) {
            for (int i = mine(tid); i < kBinsA; i += per * kCoopThreads) S.a[i] = 0;
            if (rank == 0 && tid == 0) S.mag[turn ^ 1] = 0;
        }
        __syncthreads();
        if (tid < nt && rep_times[tid]) keep(tid, rep[tid], rep_times[tid]);
        if constexpr (!ONE)
            for (int i = tid; i < nt * kAccWords; i += kCoopThreads)
                if (acc[i]) atomicAdd(&S.acc[i], acc[i]);
        __syncthreads();
        if (tid < nt && get(&kept[tid]) > kCand) atomicExch(over + turn, 1u);
        barrier();
        double *const res = args.results ? args.results + (size_t)y * 2 * kMaxTargets : S.result;
        const bool fits = get(over + turn) == 0;
        if (fits && on) {
            // D. block j of the group: targets j, j + per, ..., a warp each where
            // a block has several
            const bool warps = ONE || per < nt;
            constexpr int kWarpCand = 512;   // keys that a warp keeps in shared memory
            static_assert(kMaxTargets * kWarpCand * 12 <= kCoopSmem, "each target's keys");
            const int width = warps ? 32 : kCoopThreads, at = warps ? lane : tid;
            auto join = [&] {
                if (warps) __syncwarp();
                else __syncthreads();
            };
            const int t = warps ? warp : rank;
            if (t < nt && (!warps || t % per == rank)) {
                int q = 0;
#pragma unroll
                for (int i = 0; i < kMaxTargets; ++i)
                    if (i == t) q = first[i];
                const int c = (int)get(&kept[q]);
                const unsigned long long *keys = cand_key + q * kCand;
                const uint32_t *times = cand_times + q * kCand;
                unsigned long long *const sk = reinterpret_cast<unsigned long long *>(h) + (warps ? t * kWarpCand : 0);
                uint32_t *const sn = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned long long *>(h) +
                                                                  (warps ? kMaxTargets * kWarpCand : kCand)) +
                                     (warps ? t * kWarpCand : 0);
                unsigned long long *const sum = acc + (warps ? t * kAccWords : 0);
                if (!ONE && (!warps || c <= kWarpCand)) {
                    for (int i = at; i < c; i += width) {
                        sk[i] = __ldcg(keys + i);
                        sn[i] = __ldcg(times + i);
                    }
                    keys = sk;
                    times = sn;
                }
                if (!ONE && at < kAccWords) sum[at] = 0;   // (ONE: on with the sums of C)
                join();
                // the key with fewer than r values above it and r or more at or above
                const uint64_t r = st[2 * t + 1];
                for (int i = at; i < c; i += width) {
                    const uint64_t k = keys[i];
                    uint64_t above = 0, equal = 0;
                    for (int j = 0; j < c; ++j) {
                        const uint64_t o = keys[j];
                        above += o > k ? times[j] : 0u;
                        equal += o == k ? times[j] : 0u;
                    }
                    if (above < r && r <= above + equal) rep[t] = k;   // (equal keys write the same)
                }
                join();
                const uint64_t kt = rep[t];
                if ((args.means >> t) & 1u)
                    for (int base = at & ~31; base < c; base += width) {
                        const int i = base + lane;
                        const bool up = i < c && keys[i] > kt;
                        acc_add(sum, up, up ? value_of(keys[i]) : 0.0, up ? times[i] : 0u, sc, lane);
                    }
                join();
                if (at == 0) {
                    unsigned long long A[kAccWords];
                    for (int i = 0; i < kAccWords; ++i) A[i] = sum[i] + (ONE ? 0ull : __ldcg(&S.acc[t * kAccWords + i]));
                    tail_result(A, kt, args.m[t], sc, (args.means >> t) & 1u, res + 2 * t);
                    if (args.out[t]) *args.out[t] = res[2 * t + ((args.means >> t) & 1u)];
                }
            }
        } else if (!fits) {
            // a bin of more than kCand keys somewhere: five radix passes over
            // the YLT, then the bins' values above the keys
            for (int pass = 3; pass < 8; ++pass) {
                const int shift = 56 - 8 * pass;
                uint32_t *gh = ONE ? h : S.c + (size_t)(pass % 3) * kMaxTargets * kBins;
                for (int i = tid; i < nt * kBins; i += kCoopThreads) h[i] = 0;
                if (!ONE && rank == 0 && pass >= 5) {   // the buffer of pass - 2, read by every block already
                    uint32_t *old = S.c + (size_t)((pass - 2) % 3) * kMaxTargets * kBins;
                    for (int i = tid; i < kMaxTargets * kBins; i += kCoopThreads) old[i] = 0;
                }
                __syncthreads();
                uint64_t pre[kMaxTargets];
#pragma unroll
                for (int t = 0; t < kMaxTargets; ++t) pre[t] = t < nt ? st[2 * t] >> (shift + 8) : 0ull;
                if (on)
                    for_values(v, n, rank, per, [&](uint64_t k, double, bool ok) {
#pragma unroll
                        for (int t = 0; t < kMaxTargets; ++t) {
                            if (t >= nt) break;
                            hist_add(h + t * kBins, ok && (k >> (shift + 8)) == pre[t], (uint32_t)(k >> shift) & 0xffu,
                                     lane);
                        }
                    });
                __syncthreads();
                if constexpr (!ONE) {
                    for (int i = tid; i < nt * kBins; i += kCoopThreads)
                        if (h[i]) atomicAdd(&gh[i], h[i]);
                    barrier();
                }
                if (on && warp < nt) pick<ONE>(gh + warp * kBins, st + 2 * warp, shift, lane);
                __syncthreads();
            }
            if constexpr (!ONE)   // (ONE: on with the sums of C)
                for (int i = tid; i < nt * kAccWords; i += kCoopThreads) acc[i] = 0;
            __syncthreads();
            uint64_t kt[kMaxTargets];
#pragma unroll
            for (int t = 0; t < kMaxTargets; ++t) kt[t] = t < nt ? st[2 * t] : ~0ull;
            if (on)
                for_values(v, n, rank, per, [&](uint64_t k, double x, bool ok) {
#pragma unroll
                    for (int t = 0; t < kMaxTargets; ++t) {
                        if (t >= nt) break;
                        if ((args.means >> t) & 1u)
                            acc_add(acc + t * kAccWords, ok && (uint32_t)(k >> kShiftB) == P[t] && k > kt[t], x, 1u, sc,
                                    lane);
                    }
                });
            __syncthreads();
            if constexpr (!ONE) {
                for (int i = tid; i < nt * kAccWords; i += kCoopThreads)
                    if (acc[i]) atomicAdd(&S.acc[i], acc[i]);
                barrier();
            }
            if (on && rank == 0) {
                if (tid < nt) {
                    unsigned long long A[kAccWords];
                    for (int i = 0; i < kAccWords; ++i) A[i] = ONE ? acc[tid * kAccWords + i] : __ldcg(&S.acc[tid * kAccWords + i]);
                    tail_result(A, st[2 * tid], args.m[tid], sc, (args.means >> tid) & 1u, res + 2 * tid);
                    if (args.out[tid]) *args.out[tid] = res[2 * tid + ((args.means >> tid) & 1u)];
                }
                if constexpr (!ONE)
                    for (int i = tid; i < 3 * kMaxTargets * kBins; i += kCoopThreads) S.c[i] = 0;
            }
        }
        if (!ONE && final_round && rank == 0 && tid == 0) S.mag[0] = S.mag[1] = 0;
        __syncthreads();
    }
}

// One launch over n_ylt YLTs: `args` but for the groups.
cudaError_t enqueue_coop(CoopArgs args, int max_groups, int num_sms, cudaStream_t st)
{
    if (args.n_ylt == 1 && args.n <= kOneBlock) {
        constexpr size_t smem = kCoopSmem + sizeof(KeptKeys);
        args.per = 1;
        fit_blocks(reinterpret_cast<const void *>(k_select_coop<true>), kCoopThreads, smem);
        k_select_coop<true><<<1, kCoopThreads, smem, st>>>(args);
        return cudaGetLastError();
    }
    const int per_sm = fit_blocks(reinterpret_cast<const void *>(k_select_coop<false>), kCoopThreads, kCoopSmem);
    const int64_t resident = (int64_t)num_sms * per_sm;
    // blocks that a YLT can use, kPre values per thread each
    const int64_t useful = std::max<int64_t>(1, (args.n + kCoopThreads * kPre - 1) / (kCoopThreads * kPre));
    const int64_t groups = std::min<int64_t>({(int64_t)args.n_ylt, (int64_t)max_groups, resident});
    args.per = (int)std::min(useful, resident / groups);
    void *p[] = {&args};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_select_coop<false>), dim3((unsigned)(groups * args.per)),
                                       dim3(kCoopThreads), p, kCoopSmem, st);
}

int blocks_for(int64_t n, int cap)
{
    int64_t b = (n + kThreads * 8 - 1) / (kThreads * 8);
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

CoopArgs coop_args(int64_t n, const int64_t *ranks, int nt, int n_values)
{
    CoopArgs a{};
    a.n = n;
    a.nt = nt;
    for (int t = 0; t < nt; ++t) a.m[t] = ranks[t];
    for (int t = n_values; t < nt; ++t) a.means |= 1u << t;
    return a;
}

}  // namespace

size_t select_bytes(int groups) { return sizeof(CoopScratch) * (size_t)groups; }

// s over select_bytes(groups) of device memory at d, for selections on `st`.
void select_use(SelectScratch &s, void *d, int groups, cudaStream_t st)
{
    s.coop = d;
    s.groups = groups;
    s.result = static_cast<CoopScratch *>(d)->result;
    ARE_CUDA_TRY(cudaMemsetAsync(d, 0, select_bytes(groups), st));
}

void select_alloc(SelectScratch &s, int groups)
{
    ARE_CUDA_TRY(cudaMalloc(&s.coop, sizeof(CoopScratch) * (size_t)groups));
    ARE_CUDA_TRY(cudaMemset(s.coop, 0, sizeof(CoopScratch) * (size_t)groups));
    ARE_CUDA_TRY(cudaStreamSynchronize(nullptr));   // before any stream's selection
    s.groups = groups;
    s.result = static_cast<CoopScratch *>(s.coop)->result;
}

void select_free(SelectScratch &s)
{
    cudaFree(s.coop);
    s = SelectScratch{};
}

int launch_select(const double *ylt, int64_t n, const int64_t *ranks, int nt, int n_values, double *const *out,
                  SelectScratch &s, int num_sms, cudaStream_t st)
{
    CoopArgs a = coop_args(n, ranks, nt, n_values);
    a.single = ylt;
    a.n_ylt = 1;
    a.scratch = static_cast<CoopScratch *>(s.coop);
    for (int t = 0; t < nt && out; ++t) a.out[t] = out[t];
    ARE_CUDA_TRY(enqueue_coop(a, 1, num_sms, st));
    return 1;
}

int launch_select_multi(const double *const *ylts, int n_ylt, int64_t n, const int64_t *ranks, int nt, int n_values,
                        double *results, SelectScratch &s, int num_sms, cudaStream_t st)
{
    CoopArgs a = coop_args(n, ranks, nt, n_values);
    a.many = ylts;
    a.n_ylt = n_ylt;
    a.scratch = static_cast<CoopScratch *>(s.coop);
    a.results = results;
    ARE_CUDA_TRY(enqueue_coop(a, s.groups, num_sms, st));
    return 1;
}

}  // namespace are

// ---------------------------------------------------------------------------
// Allocation-free PML/TVaR: the same kernels, with their scratch in a
// fixed-size array that lives in the library's device image.
// ---------------------------------------------------------------------------

namespace {

constexpr size_t kStaticHist = 0;                                    // 8 x 256 words
constexpr size_t kStaticState = kStaticHist + sizeof(uint32_t) * are::kMaxTargets * 256;
constexpr size_t kStaticCtrl = kStaticState + 256;                   // 4 words
constexpr size_t kStaticAcc = kStaticCtrl + 256;                     // 8 x 7 words
constexpr size_t kStaticResult = kStaticAcc + 512;                   // 2 x 8 words
static_assert(kStaticResult + 256 <= ARE_STATIC_SCRATCH_BYTES, "static scratch too small");
static_assert(sizeof(unsigned long long) * are::kMaxTargets * 7 <= 512, "accumulator slot too small");

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[ARE_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void *g_static_addr[kMaxDevices];   // device address of g_static_scratch, per device
int g_static_sms[kMaxDevices];
thread_local char t_static_error[192];

are_status static_fail(are_status code, const char *msg)
{
    std::snprintf(t_static_error, sizeof t_static_error, "%s", msg);
    return code;
}

}  // namespace

namespace are {
const char *static_last_error() { return t_static_error; }
}

extern "C" are_status are_risk_measures_static(const double *ylt, int64_t n,
                                               const double *return_periods, int32_t n_rp,
                                               double *pml_out, const double *tvar_levels,
                                               int32_t n_tv, double *tvar_out, void *stream)
{
    using namespace are;
    t_static_error[0] = '\0';
    if (!ylt || n <= 0) return static_fail(ARE_EINVAL, "need a device YLT of n > 0 losses");
    if (n >= (int64_t)UINT32_MAX)
        return static_fail(ARE_EINVAL, "YLT too long for the selection counters");
    if (n_rp < 0 || n_tv < 0 || (n_rp > 0 && (!return_periods || !pml_out)) ||
        (n_tv > 0 && (!tvar_levels || !tvar_out)))
        return static_fail(ARE_EINVAL, "bad PML or TVaR arrays");
    if (n_rp + n_tv > kMaxTargets)
        return static_fail(ARE_EINVAL,
                           "at most 8 return periods and TVaR levels together per call");
    if (n_rp + n_tv == 0) return ARE_OK;
    int64_t ranks[kMaxTargets];
    for (int32_t r = 0; r < n_rp; ++r)
        if ((ranks[r] = rank_for_return_period(n, return_periods[r])) < 1)
            return static_fail(ARE_EINVAL, "return period must be finite and >= 1");
    for (int32_t r = 0; r < n_tv; ++r)
        if ((ranks[n_rp + r] = rank_for_level(n, tvar_levels[r])) < 1)
            return static_fail(ARE_EINVAL, "TVaR level must lie in (0, 1)");

    int dev = 0;
    cudaPointerAttributes attr;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return static_fail(ARE_ECUDA, "no usable current CUDA device");
    }
    if (cudaPointerGetAttributes(&attr, ylt) != cudaSuccess) {
        cudaGetLastError();
        return static_fail(ARE_EINVAL, "ylt is not a CUDA pointer");
    }
    if (attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged)
        return static_fail(ARE_EINVAL, "ylt must be device memory of the current device");
    if (attr.type == cudaMemoryTypeDevice && attr.device != dev)
        return static_fail(ARE_EINVAL, "ylt must be device memory of the current device");

    // Set-up, once per device with that device current: the device address
    // of the scratch array (its name is only a host-side stand-in).
    {
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_addr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return static_fail(ARE_ECUDA, "cudaGetSymbolAddress of the static scratch failed");
            }
            int sms = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                cudaGetLastError();
                return static_fail(ARE_ECUDA, "cannot query the SM count");
            }
            g_static_sms[dev] = sms;
            g_static_addr[dev] = p;
        }
    }
    unsigned char *base = static_cast<unsigned char *>(g_static_addr[dev]);
    Sel sc;
    sc.ylt = ylt;
    sc.hist = reinterpret_cast<uint32_t *>(base + kStaticHist);
    sc.state = reinterpret_cast<unsigned long long *>(base + kStaticState);
    sc.ctrl = reinterpret_cast<unsigned int *>(base + kStaticCtrl);
    sc.acc = reinterpret_cast<unsigned long long *>(base + kStaticAcc);
    sc.result = reinterpret_cast<double *>(base + kStaticResult);
    sc.blocks = blocks_for(n, g_static_sms[dev] * 4);

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nt = n_rp + n_tv;
    double res[2 * kMaxTargets];
    Ranks r{};
    for (int t = 0; t < nt; ++t) r.m[t] = ranks[t];
    k_init<<<1, kThreads, 0, st>>>(sc, r, nt);
    for (int pass = 0; pass < 8; ++pass) k_hist<<<sc.blocks, kThreads, 0, st>>>(sc, n, nt, pass);
    k_tail<<<sc.blocks, kThreads, 0, st>>>(sc, n, nt, r);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(res, sc.result, sizeof(double) * 2 * nt, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        std::snprintf(t_static_error, sizeof t_static_error, "CUDA error: %s",
                      cudaGetErrorString(e));
        return ARE_ECUDA;
    }
    for (int32_t r = 0; r < n_rp; ++r) pml_out[r] = res[2 * r];
    for (int32_t r = 0; r < n_tv; ++r) tvar_out[r] = res[2 * (n_rp + r) + 1];
    return ARE_OK;
}

// tile_rows.cu -- preprocessing (Section II-B, stage 1): a layer's rows and
// marks built in one launch, a tile of 256 catalog events per block.
//
// An ELT's entries are stored bucket by bucket, one bucket per tile (are_load_elt),
// with the offsets of the buckets, so a block finds its tile's entries of
// every ELT at once: it forms their terms, collects each event's column mask,
// places the terms at their ranks in rows held in shared memory, tells which
// events have an occurrence loss, and writes the tile's rows and marks whole.
// Nothing is cleared first, and no pass waits for another to finish.
//
// The three passes over the entries that this replaces (repack.cu, still used
// for ids past the buckets' range) read and wrote rows all over the table,
// each behind a launch, after clearing it: 33 us at 1M events x 16 ELTs of
// 20,000 entries, and 10 more for the marks.  This takes 17 us with the marks
// (the 32 MB of rows alone are 5 us at the copy bandwidth); for the 10,000
// events and 4 ELTs of a small layer 6 us instead of 23.
#include <cuda_runtime.h>

#include <string>

#include "are_internal.cuh"
#include "elt_tile.cuh"
#include "rows.cuh"

namespace are {
namespace {

constexpr int kTile = kEltTile;            // events of a block, one per thread
constexpr int kStash = 2 * kTile;          // entries whose terms are kept between the passes
constexpr unsigned kFull = 0xffffffffu;

// What a block knows of its tile.
struct Tile : EltTile {
    uint32_t ovf;                          // overflow terms handed out
    uint32_t mask[kTile];                  // per event: the ELTs whose term is not 0
};

// Packed FP32 rows of PW words (the format above rows::BodyPackedF32).
template <int PW>
struct FormPacked32 {
    using V = float;
    using W = uint32_t;
    static constexpr int WORDS = PW;
    static constexpr bool PACKED = true;
    static __device__ __forceinline__ V value(double x) { return (float)x; }
    static __device__ __forceinline__ bool nonzero(V v) { return __float_as_uint(v) != 0u; }
    static __device__ __forceinline__ W bits(V v) { return __float_as_uint(v); }
    // a term of rank r in a row of cnt terms
    static __device__ __forceinline__ void place(W *row, V *ovf, Tile &t, V v, int cnt, int r)
    {
        const int inl = cnt > PW - 1 ? PW - 2 : cnt;
        if (r < inl) {
            row[1 + r] = bits(v);
        } else if (r == inl) {
            const uint32_t off = t.base + atomicAdd(&t.ovf, (uint32_t)(cnt - inl));
            row[PW - 1] = off;
            ovf[off] = v;
        }
    }
    static __device__ __forceinline__ void place_over(const W *row, V *ovf, V v, int cnt, int r)
    {
        if (cnt > PW - 1 && r > PW - 2) ovf[row[PW - 1] + (r - (PW - 2))] = v;
    }
    static __device__ __forceinline__ void head(W *row, uint32_t mask) { row[0] = mask; }
    // whether the event has an occurrence loss (or an overflow, which may)
    static __device__ __forceinline__ bool loss(const W *row, uint32_t mask, const TermsF32 &o, const TermsF64 &)
    {
        if (__popc(mask) > PW - 1) return true;
        float g = 0.f;
#pragma unroll
        for (int h = 0; h < PW / 8; ++h) {
            rows::F8 x;
#pragma unroll
            for (int i = 0; i < 8; ++i) x.v[i] = 8 * h + i ? __uint_as_float(row[8 * h + i]) : 0.f;
            g = h ? __fadd_rn(g, rows::sum8(x)) : rows::sum8(x);
        }
        return fminf(fmaxf(__fsub_rn(g, o.occ_r), 0.f), o.occ_l) != 0.f;
    }
};

// Dense FP32 rows of JP terms.
template <int JP>
struct FormDense32 {
    using V = float;
    using W = uint32_t;
    static constexpr int WORDS = JP;
    static constexpr bool PACKED = false;
    static __device__ __forceinline__ V value(double x) { return (float)x; }
    static __device__ __forceinline__ bool nonzero(V v) { return __float_as_uint(v) != 0u; }
    static __device__ __forceinline__ W bits(V v) { return __float_as_uint(v); }
    static __device__ __forceinline__ bool loss(const W *row, uint32_t, const TermsF32 &o, const TermsF64 &)
    {
        float p[JP / 8];
#pragma unroll
        for (int h = 0; h < JP / 8; ++h) {
            rows::F8 x;
#pragma unroll
            for (int i = 0; i < 8; ++i) x.v[i] = __uint_as_float(row[8 * h + i]);
            p[h] = rows::sum8(x);
        }
        float g = p[0];
        if constexpr (JP == 16) g = __fadd_rn(p[0], p[1]);
        if constexpr (JP == 32) g = __fadd_rn(__fadd_rn(p[0], p[2]), __fadd_rn(p[1], p[3]));
        return fminf(fmaxf(__fsub_rn(g, o.occ_r), 0.f), o.occ_l) != 0.f;
    }
};

// Packed FP64 rows of RW words (the format above rows::BodyP64).
template <int RW>
struct FormPacked64 {
    using V = double;
    using W = unsigned long long;
    static constexpr int WORDS = RW;
    static constexpr bool PACKED = true;
    static __device__ __forceinline__ V value(double x) { return x; }
    static __device__ __forceinline__ bool nonzero(V v) { return rows::bits(v) != 0; }
    static __device__ __forceinline__ W bits(V v) { return rows::bits(v); }
    static __device__ __forceinline__ void place(W *row, V *, Tile &t, V v, int cnt, int r)
    {
        if (r < RW - 1) row[1 + r] = bits(v);
        if (cnt > RW - 1 && r == 0) row[0] = (W)(t.base + atomicAdd(&t.ovf, (uint32_t)cnt)) << 32;
    }
    static __device__ __forceinline__ void place_over(const W *row, V *ovf, V v, int cnt, int r)
    {
        if (cnt > RW - 1) ovf[(uint32_t)(row[0] >> 32) + r] = v;
    }
    static __device__ __forceinline__ void head(W *row, uint32_t mask) { row[0] |= mask; }
    static __device__ __forceinline__ bool loss(const W *row, uint32_t mask, const TermsF32 &, const TermsF64 &o)
    {
        const int cnt = __popc(mask);
        if (cnt > RW - 1) return true;
        double g = rows::dbl(row[1]);
        for (int i = 1; i < cnt; ++i) g = rows::vadd(g, rows::dbl(row[1 + i]));
        return rows::bits(g) > rows::bits(o.occ_r) && rows::bits(o.occ_l) != 0;
    }
};

struct BuildArgs {
    ScatterArgs elts;
    int32_t catalog;
    void *rows;
    void *ovf;               // packed rows: room for every entry
    MarkMap marks;           // d null: none
    TermsF32 o32;
    TermsF64 o64;
};

// One launch: 2.2 KB of parameters, a block per tile.  Bound by the writes of
// the rows (32 MB at 1M events in 32-byte rows).
template <typename F>
__global__ void __launch_bounds__(kTile) k_tile_rows(const __grid_constant__ BuildArgs a)
{
    using V = typename F::V;
    using W = typename F::W;
    __shared__ __align__(16) W row[kTile * F::WORDS];
    __shared__ Tile t;
    __shared__ V stash[kStash];
    __shared__ uint16_t stash_ej[kStash];
    const int tid = threadIdx.x, tile = blockIdx.x;
    const uint32_t e0 = (uint32_t)tile * kTile;
    V *const ovf = static_cast<V *>(a.ovf);
    if (tid < 32) t.find(a.elts, tile, tid);
    if (tid == 0) t.ovf = 0;
    t.mask[tid] = 0;
    {
        uint4 *z = reinterpret_cast<uint4 *>(row);
#pragma unroll
        for (int i = 0; i < (int)(sizeof(W) * F::WORDS / 16); ++i) z[i * kTile + tid] = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    const uint32_t n = t.start[32];
    // entry i of the tile: its event, ELT and term
    auto entry = [&](uint32_t i, uint32_t &e, int &j) -> V {
        const int32_t at = t.entry(a.elts, i, e0, e, j);
        return F::value(fin_term(a.elts.loss[j][at], a.elts.fx[j], a.elts.ded[j], a.elts.lim[j], a.elts.share[j]));
    };
    auto again = [&](uint32_t i, uint32_t &e, int &j) -> V {
        if (i >= kStash) return entry(i, e, j);
        e = stash_ej[i] & 255u;
        j = stash_ej[i] >> 8;
        return stash[i];
    };
    for (uint32_t i = tid; i < n; i += kTile) {
        uint32_t e;
        int j;
        const V v = entry(i, e, j);
        if constexpr (!F::PACKED) {
            row[e * F::WORDS + j] = F::bits(v);
        } else {
            if (F::nonzero(v)) atomicOr(&t.mask[e], 1u << j);
            if (i < kStash) {
                stash[i] = v;
                stash_ej[i] = (uint16_t)(e | (uint32_t)j << 8);
            }
        }
    }
    __syncthreads();
    if constexpr (F::PACKED) {
        for (int over = 0; over < 2; ++over) {   // the terms at their ranks, then the rest of the longer rows
            for (uint32_t i = tid; i < n; i += kTile) {
                uint32_t e;
                int j;
                const V v = again(i, e, j);
                if (!F::nonzero(v)) continue;
                const uint32_t mask = t.mask[e];
                const int cnt = __popc(mask), r = __popc(mask & ((1u << j) - 1u));
                if (!over) F::place(row + e * F::WORDS, ovf, t, v, cnt, r);
                else F::place_over(row + e * F::WORDS, ovf, v, cnt, r);
            }
            __syncthreads();
            if (t.ovf == 0) break;
        }
        F::head(row + tid * F::WORDS, t.mask[tid]);
    }
    const bool in = e0 + tid < (uint32_t)a.catalog;
    if (a.marks.d) {   // a warp's 32 events are one word
        const bool on = in && F::loss(row + tid * F::WORDS, t.mask[tid], a.o32, a.o64);
        const uint32_t b = __brev(__ballot_sync(kFull, on));
        uint32_t w = (e0 + tid) >> 5;
        if ((tid & 31) == 0) {
            if (a.marks.fold) {
                w = min(w, w - (uint32_t)a.marks.words);
                if (b) atomicOr(a.marks.d + w, b);
            } else if (w < (uint32_t)a.marks.words) {
                a.marks.d[w] = b;
            }
        }
    }
    __syncthreads();
    const uint32_t left = (uint32_t)a.catalog - e0;
    const uint32_t pieces = (left < kTile ? left : kTile) * (uint32_t)(sizeof(W) * F::WORDS / 16);
    uint4 *dst = reinterpret_cast<uint4 *>(static_cast<W *>(a.rows) + (size_t)e0 * F::WORDS);
    const uint4 *src = reinterpret_cast<const uint4 *>(row);
    for (uint32_t i = tid; i < pieces; i += kTile) dst[i] = src[i];
}

// An ELT's entries into buckets, one per tile of events.
// 1. One block counts the buckets and scans the counts in its shared memory,
//    kRead entries per thread in flight.  off[i + 1] receives where bucket i
//    starts; with FILL (few entries) where it ends, and the block fills the
//    buckets too.
constexpr int kBucketThreads = 1024;
template <bool FILL>
__global__ void __launch_bounds__(kBucketThreads)
    k_bucket_offsets(const int32_t *__restrict__ ids, const double *__restrict__ loss, int32_t n, int32_t tiles,
                     int32_t *__restrict__ off, int32_t *__restrict__ out_ids, double *__restrict__ out_loss)
{
    extern __shared__ int32_t count[];
    __shared__ int32_t sums[kBucketThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int i = tid; i < tiles; i += kBucketThreads) count[i] = 0;
    __syncthreads();
    constexpr int kRead = 8;
    for (int64_t i0 = tid; i0 < n; i0 += kRead * kBucketThreads) {
        int32_t id[kRead];
#pragma unroll
        for (int k = 0; k < kRead; ++k) id[k] = i0 + k * kBucketThreads < n ? ids[i0 + k * kBucketThreads] : -1;
#pragma unroll
        for (int k = 0; k < kRead; ++k)
            if (id[k] >= 0) atomicAdd(count + id[k] / kEltTile, 1);
    }
    __syncthreads();
    // exclusive scan, a run of tiles per thread
    const int per = (tiles + kBucketThreads - 1) / kBucketThreads, b = tid * per;
    int32_t own = 0;
    for (int i = b; i < b + per && i < tiles; ++i) own += count[i];
    int32_t incl = own;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t o = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) sums[w] = incl;
    __syncthreads();
    if (w == 0) {
        int32_t v = sums[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t o = __shfl_up_sync(kFull, v, d);
            if (lane >= d) v += o;
        }
        sums[lane] = v;
    }
    __syncthreads();
    int32_t run = incl - own + (w ? sums[w - 1] : 0);
    for (int i = b; i < b + per && i < tiles; ++i) {
        const int32_t c = count[i];
        count[i] = run;
        run += c;
    }
    __syncthreads();
    if constexpr (FILL) {
        for (int32_t i = tid; i < n; i += kBucketThreads) {
            const int32_t id = ids[i], at = atomicAdd(count + id / kEltTile, 1);
            out_ids[at] = id;
            out_loss[at] = loss[i];
        }
        __syncthreads();
    }
    for (int i = tid; i < tiles; i += kBucketThreads) off[i + 1] = count[i];
    if (tid == 0) off[0] = 0;
}

// 2. The entries to their buckets, off[i + 1] counted up to where bucket i ends
//    and the next starts.  (One block doing this too took 64 us for 50,000
//    entries: a store of 32 scattered words occupies the SM for 32 cycles.)
__global__ void k_bucket_fill(const int32_t *__restrict__ ids, const double *__restrict__ loss, int32_t n,
                              int32_t *__restrict__ off, int32_t *__restrict__ out_ids, double *__restrict__ out_loss)
{
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t id = ids[i], at = atomicAdd(off + 1 + id / kEltTile, 1);
    out_ids[at] = id;
    out_loss[at] = loss[i];
}

template <typename F>
void launch_t(const BuildArgs &a, cudaStream_t s)
{
    k_tile_rows<F><<<(unsigned)(((int64_t)a.catalog + kTile - 1) / kTile), kTile, 0, s>>>(a);
    ARE_CUDA_TRY(cudaGetLastError());
}

}  // namespace

// The entries of an ELT into buckets: the offsets (off, tiles + 1 of them) once
// the ids are at hand, then the rest; up to kFewEntries of them are both one
// launch, the second (2000 entries in host memory load in 38 us, in two
// launches 40; 100 entries 32 and 35).  ids and loss: device memory, or pinned
// host memory.
constexpr int32_t kFewEntries = 2048;
namespace {
template <bool FILL>
void launch_offsets(const int32_t *ids, const double *loss, int32_t n, int32_t tiles, int32_t *off, int32_t *out_ids,
                    double *out_loss, cudaStream_t s)
{
    constexpr size_t most = sizeof(int32_t) * (kMaxBucketedId / kEltTile);
    static_assert(most <= 200 * 1024, "the bucket counts fit a block");
    fit_blocks(reinterpret_cast<const void *>(k_bucket_offsets<FILL>), kBucketThreads, most);   // raises the limit
    k_bucket_offsets<FILL><<<1, kBucketThreads, sizeof(int32_t) * (size_t)tiles, s>>>(ids, loss, n, tiles, off, out_ids,
                                                                                      out_loss);
    ARE_CUDA_TRY(cudaGetLastError());
}
}  // namespace

int launch_bucket_offsets(const int32_t *ids, int32_t n, int32_t tiles, int32_t *off, cudaStream_t s)
{
    if (n <= kFewEntries) return 0;
    launch_offsets<false>(ids, nullptr, n, tiles, off, nullptr, nullptr, s);
    return 1;
}

int launch_bucket_fill(const int32_t *ids, const double *loss, int32_t n, int32_t tiles, int32_t *out_ids,
                       double *out_loss, int32_t *off, cudaStream_t s)
{
    if (n <= kFewEntries) {
        launch_offsets<true>(ids, loss, n, tiles, off, out_ids, out_loss, s);
    } else {
        k_bucket_fill<<<(unsigned)(((int64_t)n + 255) / 256), 256, 0, s>>>(ids, loss, n, off, out_ids, out_loss);
        ARE_CUDA_TRY(cudaGetLastError());
    }
    return 1;
}

// The rows of a layer (and its marks, where marks.d is set), every ELT's
// entries in buckets (elts_bucketed).  packed: rows of `words` 32-bit (fp32)
// or 64-bit words and their overflow; else dense FP32 rows of `words` terms.
int launch_tile_rows(const ScatterArgs &elts, int32_t catalog, bool fp32, bool packed, int words, void *rows, void *ovf,
                     const MarkMap &marks, const TermsF32 &o32, const TermsF64 &o64, cudaStream_t s)
{
    BuildArgs a;
    a.elts = elts;
    a.catalog = catalog;
    a.rows = rows;
    a.ovf = ovf;
    a.marks = marks;
    a.o32 = o32;
    a.o64 = o64;
    if (marks.d && marks.fold) ARE_CUDA_TRY(cudaMemsetAsync(marks.d, 0, sizeof(uint32_t) * (size_t)marks.words, s));
    if (fp32 && packed && words == 8) launch_t<FormPacked32<8>>(a, s);
    else if (fp32 && packed && words == 16) launch_t<FormPacked32<16>>(a, s);
    else if (fp32 && !packed && words == 8) launch_t<FormDense32<8>>(a, s);
    else if (fp32 && !packed && words == 16) launch_t<FormDense32<16>>(a, s);
    else if (fp32 && !packed && words == 32) launch_t<FormDense32<32>>(a, s);
    else if (!fp32 && packed && words == 4) launch_t<FormPacked64<4>>(a, s);
    else if (!fp32 && packed && words == 8) launch_t<FormPacked64<8>>(a, s);
    else throw Error{ARE_EINVAL, "no tile builder for rows of " + std::to_string(words) + " words"};
    return 1;
}

}  // namespace are

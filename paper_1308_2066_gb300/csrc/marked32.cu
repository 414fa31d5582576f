// marked32.cu -- the trial pass over marked events (marked.cuh) with FP32
// rows, packed or dense.
#include <cuda_runtime.h>

#include <string>

#include "are_internal.cuh"
#include "marked.cuh"

namespace are {
namespace {

// The layer's rows by their form: packed rows of 8 or 16 words (a.table the
// rows, a.table2 the overflow terms), or dense rows of 8 or 16 terms.
template <typename F>
auto with_rows(const void *table, const void *ovf, bool packed, int row_words, const TermsF32 &tm, F &&fn)
{
    auto go = [&](auto r) {
        r.table = static_cast<const float *>(table);
        if constexpr (decltype(r)::PACKED) r.ovf = static_cast<const float *>(ovf);
        r.occ_r = tm.occ_r;
        r.occ_l = tm.occ_l;
        return fn(r);
    };
    if (packed && row_words == 8) return go(marked::PackedF32<8>{});
    if (packed && row_words == 16) return go(marked::PackedF32<16>{});
    if (!packed && row_words == 8) return go(marked::DenseF32<8>{});
    if (!packed && row_words == 16) return go(marked::DenseF32<16>{});
    throw Error{ARE_EINVAL, "no marked FP32 rows of " + std::to_string(row_words) + " words"};
}

}  // namespace

int launch_marked32(const SimArgs &a, const MarkMap &m, are_precision prec, bool packed, int row_words,
                    const TermsF32 &t, int scale, int num_sms, cudaStream_t s)
{
    if (a.n_trials <= 0) return 0;
    with_rows(a.table, a.table2, packed, row_words, t, [&](auto r) {
        using Rows = decltype(r);
        if (prec == ARE_FP32_KAHAN) marked::launch_pass<Rows, ARE_FP32_KAHAN>(a, m, r, scale, num_sms, s);
        else marked::launch_pass<Rows, ARE_FP64>(a, m, r, scale, num_sms, s);
        return 0;
    });
    return 1;
}

}  // namespace are

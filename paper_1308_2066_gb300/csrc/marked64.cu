// marked64.cu -- the trial pass over marked events (marked.cuh) with packed
// FP64 rows.
#include <cuda_runtime.h>

#include <string>

#include "are_internal.cuh"
#include "marked.cuh"

namespace are {
namespace {

template <typename F>
auto with_rows(const void *table, const void *ovf, int row_words, const TermsF64 &tm, F &&fn)
{
    auto go = [&](auto r) {
        r.table = static_cast<const unsigned long long *>(table);
        r.ovf = static_cast<const double *>(ovf);
        r.occ_r = tm.occ_r;
        r.occ_l = tm.occ_l;
        return fn(r);
    };
    if (row_words == 4) return go(marked::PackedF64<4>{});
    if (row_words == 8) return go(marked::PackedF64<8>{});
    throw Error{ARE_EINVAL, "no marked FP64 rows of " + std::to_string(row_words) + " words"};
}

}  // namespace

int launch_marked64(const SimArgs &a, const MarkMap &m, int row_words, const TermsF64 &t, int scale, int num_sms,
                    cudaStream_t s)
{
    if (a.n_trials <= 0) return 0;
    with_rows(a.table, a.table2, row_words, t, [&](auto r) {
        marked::launch_pass<decltype(r), ARE_FP64>(a, m, r, scale, num_sms, s);
        return 0;
    });
    return 1;
}

}  // namespace are

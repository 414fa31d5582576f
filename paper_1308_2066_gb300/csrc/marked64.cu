// marked64.cu -- the trial pass over marked events (marked.cuh) with packed
// FP64 rows.
#include <cuda_runtime.h>

#include "are_internal.cuh"
#include "marked.cuh"

namespace are {

int launch_marked64(const SimArgs &a, const MarkMap &m, int row_words, const TermsF64 &t, int scale, int num_sms,
                    cudaStream_t s)
{
    if (a.n_trials <= 0) return 0;
    return marked::with_rows64(a.table, a.table2, row_words, t, [&](auto r) {
        marked::launch_pass<decltype(r), ARE_FP64>(a, m, r, scale, num_sms, s);
        return 1;
    });
}

}  // namespace are

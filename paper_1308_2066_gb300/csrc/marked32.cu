// marked32.cu -- the trial pass over marked events (marked.cuh) with FP32
// rows, packed or dense.
#include <cuda_runtime.h>

#include "are_internal.cuh"
#include "marked.cuh"

namespace are {

int launch_marked32(const SimArgs &a, const MarkMap &m, are_precision prec, bool packed, int row_words,
                    const TermsF32 &t, int scale, int num_sms, cudaStream_t s)
{
    if (a.n_trials <= 0) return 0;
    return marked::with_rows32(a.table, a.table2, packed, row_words, t, [&](auto r) {
        using Rows = decltype(r);
        if (prec == ARE_FP32_KAHAN) marked::launch_pass<Rows, ARE_FP32_KAHAN>(a, m, r, scale, num_sms, s);
        else marked::launch_pass<Rows, ARE_FP64>(a, m, r, scale, num_sms, s);
        return 1;
    });
}

}  // namespace are

// fft_kernels_mr_fwd_fold_b.cu -- composite-radix line passes, forward:
// strided lines in tiles of several outer indices.
#include "fft_p2.cuh"
#include "fft_mr.cuh"
#include "mr_lengths.h"

namespace fbfft {

LineKernel line_kernel_mr_fwd_fold_b(int L)
{
    switch (L) {
#define FB_MR_CASE(N) \
    case N: return mr_fold_entry<true, N>();
        FB_MR_LENGTHS_B(FB_MR_CASE)
    default: return LineKernel{nullptr, 0, false, 0, 0};
    }
}

}  // namespace fbfft

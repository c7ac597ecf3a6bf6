// Two-step local-potential passes (fft_two_step.cuh), double-FP32: grid edges 128, 108, 90, 54.
#include "fft_two_step.cuh"

namespace lg {
int fft2_df_4(const Fft2Args<df64f, double> &a) {
    switch (a.g->N) {
        case 128: return f2s::run<df64f, double, 128, 8>(a);
        case 108: return f2s::run<df64f, double, 108, 9>(a);
        case 90: return f2s::run<df64f, double, 90, 6>(a);
        case 54: return f2s::run<df64f, double, 54, 6>(a);
        default: return 1;
    }
}
}  // namespace lg

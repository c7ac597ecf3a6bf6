// Two-step local-potential passes (fft_two_step.cuh), double-FP32: grid edges 120, 72, 36, 24.
#include "fft_two_step.cuh"

namespace lg {
int fft2_df_1(const Fft2Args<df64f, double> &a) {
    switch (a.g->N) {
        case 120: return f2s::run<df64f, double, 120, 8>(a);
        case 72: return f2s::run<df64f, double, 72, 8>(a);
        case 36: return f2s::run<df64f, double, 36, 6>(a);
        case 24: return f2s::run<df64f, double, 24, 8>(a);
        default: return 1;
    }
}
}  // namespace lg

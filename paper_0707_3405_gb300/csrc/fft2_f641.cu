// Two-step local-potential passes (fft_two_step.cuh), FP64: grid edges 120, 72, 36, 24.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f64_1(const Fft2Args<double, double> &a) {
    switch (a.g->N) {
        case 120: return f2s::run<double, double, 120, 8>(a);
        case 72: return f2s::run<double, double, 72, 8>(a);
        case 36: return f2s::run<double, double, 36, 6>(a);
        case 24: return f2s::run<double, double, 24, 8>(a);
        default: return 1;
    }
}
}  // namespace lg

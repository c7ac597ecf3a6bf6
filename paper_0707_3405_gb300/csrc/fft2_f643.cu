// Two-step local-potential passes (fft_two_step.cuh), FP64: grid edges 160, 80, 40, 100.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f64_3(const Fft2Args<double, double> &a) {
    switch (a.g->N) {
        case 160: return f2s::run<double, double, 160, 16>(a);
        case 80: return f2s::run<double, double, 80, 8>(a);
        case 40: return f2s::run<double, double, 40, 8>(a);
        case 100: return f2s::run<double, double, 100, 10>(a);
        default: return 1;
    }
}
}  // namespace lg

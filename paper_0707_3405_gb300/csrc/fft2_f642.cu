// Two-step local-potential passes (fft_two_step.cuh), FP64: grid edges 96, 48, 64, 60.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f64_2(const Fft2Args<double, double> &a) {
    switch (a.g->N) {
        case 96: return f2s::run<double, double, 96, 8>(a);
        case 48: return f2s::run<double, double, 48, 8>(a);
        case 64: return f2s::run<double, double, 64, 8>(a);
        case 60: return f2s::run<double, double, 60, 6>(a);
        default: return 1;
    }
}
}  // namespace lg

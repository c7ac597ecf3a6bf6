// Two-step local-potential passes (fft_two_step.cuh), FP32: grid edges 120.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f32_1(const Fft2Args<float, float> &a) {
    switch (a.g->N) {
        case 120: return f2s::run<float, float, 120, 8>(a);
        default: return 1;
    }
}
}  // namespace lg

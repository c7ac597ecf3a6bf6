// Two-step local-potential passes (fft_two_step.cuh), FP32: grid edges 160, 80, 40, 100.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f32_3(const Fft2Args<float, float> &a) {
    switch (a.g->N) {
        case 160: return f2s::run<float, float, 160, 16>(a);
        case 80: return f2s::run<float, float, 80, 8>(a);
        case 40: return f2s::run<float, float, 40, 8>(a);
        case 100: return f2s::run<float, float, 100, 10>(a);
        default: return 1;
    }
}
}  // namespace lg

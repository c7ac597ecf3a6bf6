// Two-step local-potential passes (fft_two_step.cuh), FP32: grid edges 128, 108, 90, 54.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f32_4(const Fft2Args<float, float> &a) {
    switch (a.g->N) {
        case 128: return f2s::run<float, float, 128, 8>(a);
        case 108: return f2s::run<float, float, 108, 9>(a);
        case 90: return f2s::run<float, float, 90, 6>(a);
        case 54: return f2s::run<float, float, 54, 6>(a);
        default: return 1;
    }
}
}  // namespace lg

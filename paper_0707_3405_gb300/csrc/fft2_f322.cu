// Two-step local-potential passes (fft_two_step.cuh), FP32: grid edges 96, 60.
#include "fft_two_step.cuh"

namespace lg {
int fft2_f32_2(const Fft2Args<float, float> &a) {
    switch (a.g->N) {
        case 96: return f2s::run<float, float, 96, 8>(a);
        case 60: return f2s::run<float, float, 60, 6>(a);
        default: return 1;
    }
}
}  // namespace lg

// Double-FP32 local-potential passes (fft_df.cuh): grid edges 160, 80, 40, 100.
#include "fft_df.cuh"

namespace lg {
int fft_df_apply_3(const FFTGeom &g, const z64 *X, int ldx, z64 *Y, int ldy, int nb, const double *kin, const df64f *vt,
                   const z64 *tw, cx<df64f> *T2, int nbatch, int smem_max, cudaStream_t s) {
    switch (g.N) {
        case 160: return fdf::run<160, 16>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 80: return fdf::run<80, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 40: return fdf::run<40, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 100: return fdf::run<100, 10>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        default: return 1;
    }
}
}  // namespace lg

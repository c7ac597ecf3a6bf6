// Double-FP32 local-potential passes (fft_df.cuh): grid edges 128, 108, 90, 54.
#include "fft_df.cuh"

namespace lg {
int fft_df_apply_4(const FFTGeom &g, const z64 *X, int ldx, z64 *Y, int ldy, int nb, const double *kin, const df64f *vt,
                   const z64 *tw, cx<df64f> *T2, int nbatch, int smem_max, cudaStream_t s) {
    switch (g.N) {
        case 128: return fdf::run<128, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 108: return fdf::run<108, 9>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 90: return fdf::run<90, 6>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 54: return fdf::run<54, 6>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        default: return 1;
    }
}
}  // namespace lg

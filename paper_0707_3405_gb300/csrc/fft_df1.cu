// Double-FP32 local-potential passes (fft_df.cuh): grid edges 120, 72, 36, 24.
#include "fft_df.cuh"

namespace lg {
int fft_df_apply_1(const FFTGeom &g, const z64 *X, int ldx, z64 *Y, int ldy, int nb, const double *kin, const df64f *vt,
                   const z64 *tw, cx<df64f> *T2, int nbatch, int smem_max, cudaStream_t s) {
    switch (g.N) {
        case 120: return fdf::run<120, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 72: return fdf::run<72, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 36: return fdf::run<36, 6>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 24: return fdf::run<24, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        default: return 1;
    }
}
}  // namespace lg

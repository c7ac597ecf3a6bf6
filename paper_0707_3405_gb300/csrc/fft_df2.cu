// Double-FP32 local-potential passes (fft_df.cuh): grid edges 96, 48, 64, 60.
#include "fft_df.cuh"

namespace lg {
int fft_df_apply_2(const FFTGeom &g, const z64 *X, int ldx, z64 *Y, int ldy, int nb, const double *kin, const df64f *vt,
                   const z64 *tw, cx<df64f> *T2, int nbatch, int smem_max, cudaStream_t s) {
    switch (g.N) {
        case 96: return fdf::run<96, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 48: return fdf::run<48, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 64: return fdf::run<64, 8>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        case 60: return fdf::run<60, 6>(g, X, ldx, Y, ldy, nb, kin, vt, tw, T2, nbatch, smem_max, s);
        default: return 1;
    }
}
}  // namespace lg

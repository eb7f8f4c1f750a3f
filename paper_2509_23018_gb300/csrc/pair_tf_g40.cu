// Two-float pair kernel and band setup instantiated for the 40^3 grid.
#include "pair_tf_ct.cuh"

namespace gw {

cudaError_t launch_pair_tf_g40(const float4 *a, const float4 *b, int nc, int64_t p0, int64_t count,
                               const PairPlan &pp, const TfConsts &kc, tf inv, double2 *M, cudaStream_t st)
{
    return launch_pair_tf_cube<40>(a, b, nc, p0, count, pp, kc, inv, M, st);
}

cudaError_t pair_tf_slots_g40(const PairPlan &pp, int *nslots) { return pair_tf_cube_slots<40>(pp, nslots); }

cudaError_t launch_pair_tf_from_f_g40(const CUtensorMap &tmF, const CUtensorMap &tmS, int64_t R, int cb, int64_t sv,
                                      int64_t sc, const PairPlan &pp, const TfConsts &kc, tf inv, double2 *M,
                                      cudaStream_t st)
{
    return launch_pair_tf_from_f_cube<40>(tmF, tmS, R, cb, sv, sc, pp, kc, inv, M, st);
}

cudaError_t launch_band_fft_tf_g40(float4 *psi, int nb, const FftAxis *ax, const TfConsts &kc, int m0, int m1,
                                  cudaStream_t st)
{
    return launch_band_fft_tf_ct<40>(psi, nb, ax, kc, m0, m1, st);
}

} // namespace gw

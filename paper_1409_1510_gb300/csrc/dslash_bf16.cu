// Dslash instantiations for BF16 storage.
#include "dslash_launch.cuh"

namespace hisq {

template <>
cudaError_t launch_dslash_prec<HISQ_BF16>(const KArgs &a, int recon, int epi, int R, int S, int threads, size_t smem,
                                        int num_sms, cudaStream_t s, int *grid) {
    if (recon == 13) return launch_epi<HISQ_BF16, 13>(a, epi, R, S, threads, smem, num_sms, s, grid);
    if (recon == 9) return launch_epi<HISQ_BF16, 9>(a, epi, R, S, threads, smem, num_sms, s, grid);
    return launch_epi<HISQ_BF16, 18>(a, epi, R, S, threads, smem, num_sms, s, grid);
}

template <>
cudaError_t launch_dslash_mma<HISQ_BF16>(const KArgs &a, const MmaField &fat, const MmaField &naik, int epi, size_t smem,
                                         int num_sms, cudaStream_t s, int *grid) {
    if (epi == EPI_PLAIN) return launch_mma_one<HISQ_BF16, EPI_PLAIN>(a, fat, naik, smem, num_sms, s, grid);
    return launch_mma_one<HISQ_BF16, EPI_AOP>(a, fat, naik, smem, num_sms, s, grid);
}

}  // namespace hisq

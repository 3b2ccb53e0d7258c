// tc_softmax.cu -- instantiations of the fused vocabulary GEMM + online softmax / top-k
// epilogue (section 4.1.1 base logits and the section 4.1.2 W2 term in one accumulator).
#include "tc_pair.cuh"

namespace dm {

cudaError_t launch_tc_vocab_pair(int kmax, const CUtensorMap* maps, const TcParams& p, int grid, cudaStream_t s) {
  if (kmax == 8) return launch_tc_vocab_pair_k8(maps, p, grid, s);
  if (kmax == 16) return launch_tc_vocab_pair_instance<16>(maps, p, grid, s);
  if (kmax == 32) return launch_tc_vocab_pair_instance<32>(maps, p, grid, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_tc_softmax(int bn, bool swap, int kmax, const CUtensorMap* maps, const TcParams& p,
                              int grid, cudaStream_t s) {
  // tokens on M in CTA pairs: the 2-SM MMA kernel (tc_pair.cuh)
  if (!swap && bn == 256 && p.pair) return launch_tc_vocab_pair(kmax, maps, p, grid, s);
  if (kmax == 8) return launch_tc_softmax_k8(bn, swap, maps, p, grid, s);
#define DM_SM(BN, SW, KM)                                                              \
  if (bn == BN && swap == SW && kmax == KM)                                            \
    return launch_tc_instance<BN, SW, kModeSoftmax, KM>(maps, p, grid, s);
  DM_SM(16, true, 16) DM_SM(32, true, 16) DM_SM(64, true, 16) DM_SM(128, true, 16) DM_SM(256, false, 16)
  DM_SM(16, true, 32) DM_SM(32, true, 32) DM_SM(64, true, 32) DM_SM(128, true, 32) DM_SM(256, false, 32)
#undef DM_SM
  return cudaErrorInvalidValue;
}

// Deferred variants: the stages that leave a GRU CTA (80 KB) room on the same SM -- 6, 5, 5 and 4 for
// BN = 16, 32, 64 and 128 (118 to 150 KB).
cudaError_t launch_tc_softmax_deferred(int bn, int kmax, const CUtensorMap* maps, const TcParams& p, int grid,
                                       cudaStream_t s) {
  if (p.defer < 1 || p.defer > kMaxBlocks || p.defer * bn > p.tmem_cols) return cudaErrorInvalidValue;
  if (kmax == 8) return launch_tc_softmax_deferred_k8(bn, maps, p, grid, s);
#define DM_SD(BN, KM, ST) \
  if (bn == BN && kmax == KM) return launch_tc_instance<BN, true, kModeSoftmax, KM, ST>(maps, p, grid, s, true);
  DM_SD(16, 16, 6) DM_SD(16, 32, 6) DM_SD(32, 16, 5) DM_SD(32, 32, 5)
  DM_SD(64, 16, 5) DM_SD(64, 32, 5) DM_SD(128, 16, 4) DM_SD(128, 32, 4)
#undef DM_SD
  return cudaErrorInvalidValue;
}

int tc_softmax_deferred_smem(int bn, int kmax) {
  if (kmax == 8) return tc_softmax_deferred_smem_k8(bn);
  // the list length takes no shared memory in this orientation
  if (bn == 16) return TcCfg<16, true, kModeSoftmax, 16, 6>::kSmemBytes;
  if (bn == 32) return TcCfg<32, true, kModeSoftmax, 16, 5>::kSmemBytes;
  if (bn == 64) return TcCfg<64, true, kModeSoftmax, 16, 5>::kSmemBytes;
  if (bn == 128) return TcCfg<128, true, kModeSoftmax, 16, 4>::kSmemBytes;
  return 0;
}

}  // namespace dm

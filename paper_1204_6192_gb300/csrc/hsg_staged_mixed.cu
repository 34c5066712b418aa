// Staged over-relaxation half-sweeps of contexts with lattices of several sizes: one kernel
// with the code of every row length, picked by the block's sample.  (In place of the
// kernels of one length it costs them 1 to 2 %: L = 128, 48 systems, BF16 311 -> 315 us a
// sweep; L = 64 in FP16 59.0 -> 60.0.)
#include "hsg_staged.cuh"

namespace hsg {

cudaError_t launch_staged_mixed(int fmt, bool j16, bool energy, const SweepParams& p, int n_blocks,
                                size_t smem, cudaStream_t st) {
  return launch_staged_l<0>(fmt, j16, energy, p, n_blocks, smem, st);
}

}  // namespace hsg

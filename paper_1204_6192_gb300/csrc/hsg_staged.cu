// Staged over-relaxation half-sweeps of contexts whose lattices are all of one size: one
// kernel a row length.
#include "hsg_staged.cuh"

#include <algorithm>

namespace hsg {

bool lattice_has_staged(int L) { return L >= 32 && L <= 512 && (L & (L - 1)) == 0; }

int staged_stage_bytes(int fmt, int L) {
  return 3 * stage_plane_chunks(L / 2) * (fmt == FMT_F32 ? 16 : 8);   // component formats: 3 planes
}

// [0, STAGED_HEAD): mbarriers; then the energy sums of the warps (energy sweeps); then,
// 128-byte aligned, the ring of stages.
size_t staged_smem(int gpt, bool energy, int stage_bytes, int* stage_off) {
  const size_t esum = energy ? sizeof(float) * NW * (size_t)gpt * 4 : 0;
  const size_t off = (STAGED_HEAD + esum + 127) / 128 * 128;
  *stage_off = (int)off;
  // (a block of one chunk group uses one stage; L = 256, 4 systems, FP16, with the room
  // of both: 3 blocks an SM instead of 4, a sweep 728 us instead of 650)
  return off + (size_t)std::min(STAGED_STAGES, gpt) * stage_bytes;
}

cudaError_t launch_staged_half(int fmt, bool j16, bool energy, const SweepParams& p, int n_blocks,
                               size_t smem, cudaStream_t st) {
  if (n_blocks <= 0) return cudaSuccess;
  switch (p.one_Lh) {
    case 0: return launch_staged_mixed(fmt, j16, energy, p, n_blocks, smem, st);
    case 16: return launch_staged_l<16>(fmt, j16, energy, p, n_blocks, smem, st);
    case 32: return launch_staged_l<32>(fmt, j16, energy, p, n_blocks, smem, st);
    case 64: return launch_staged_l<64>(fmt, j16, energy, p, n_blocks, smem, st);
    case 128: return launch_staged_l<128>(fmt, j16, energy, p, n_blocks, smem, st);
    case 256: return launch_staged_l<256>(fmt, j16, energy, p, n_blocks, smem, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hsg

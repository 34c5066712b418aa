// The wave launch: both half-sweeps of an over-relaxation sweep (Sec. 3.1, Eq. 3) at once.
//
// One launch has one block per (block table entry, parity): the blocks of the two
// per-half-sweep launches.  A block takes a ticket on entry (an atomic counter) and does the
// work the host-built order assigns to it.  The order walks the even blocks in table order
// (z-major within a chunk group) and inserts each odd block `lag` even blocks after the last
// even block it depends on.  An odd block of planes [z0, z1] reads the even sites of planes
// z0-1 .. z1+1 (new values) and overwrites odd sites that the even blocks of those planes
// read (old values), so before its update it waits until every even block of those planes
// has signalled completion.  Those blocks hold earlier tickets, so they are already running
// and never wait themselves: no wait can deadlock, whatever the number of resident blocks.
// Every even site sees only old odd spins and every odd site only new even spins, so the
// result is that of the even half-sweep followed by the odd one, bit for bit.  Staged odd
// blocks (hsg_staged.cuh) read the even spins through bulk copies (L2, after a proxy fence);
// unstaged odd blocks read them bypassing L1.  Between the even update of a plane and the
// odd updates that read it lie about `lag` blocks of work, so the opposite parity, which two
// separate launches read from DRAM a second time, mostly comes from L2.  The last block to
// finish resets the ticket and completion counters and advances the epoch the completion
// flags carry, so each launch (and each replay of a captured graph) starts clean.
//
// A sweep of 48 systems at L = 128, FP16: 337 us (two staged launches 299); FP32, 24 systems
// 342; L = 256, 4 systems 826 and 1511 (two launches 599 and 1044).
#include "hsg_staged.cuh"

namespace hsg {

namespace {

// Wait until *f == want, at most limit_ns.
__device__ __forceinline__ bool wait_flag(const unsigned int* f, unsigned int want,
                                          unsigned long long limit_ns) {
  const volatile unsigned int* v = f;
  if (*v == want) return true;
  const unsigned long long t0 = now_ns();
  while (*v != want) {
    if (now_ns() - t0 > limit_ns) return false;
    __nanosleep(128);
  }
  return true;
}

template <int F, bool J16, bool EN, bool STG>
__global__ void __launch_bounds__(SWEEP_BS, 4) k_wave_sweep(const WaveParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ unsigned int s_ticket, s_epoch;
  if (threadIdx.x == 0) {
    s_ticket = atomicAdd(P.state, 1u);
    s_epoch = *(volatile unsigned int*)(P.state + 2);
  }
  __syncthreads();
  const unsigned int want = s_epoch + 1u;
  // (a ticket beyond the launch would mean counters left inconsistent: no work)
  const bool valid = s_ticket < (unsigned int)P.n_tickets;
  const int code = valid ? P.order[P.t0 + (int)s_ticket] : 0;
  const int b = code >> 1, parity = valid ? (code & 1) : 2;
  SweepParams sp = P.sw;
  sp.parity = parity & 1;
  if (!valid) {
    if (threadIdx.x == 0) atomicExch(P.err, 1u);
  } else if (parity == 0) {
    if constexpr (STG) staged_block<F, J16, EN>(sp, b, smem);
    else sweep_block<F, false, J16, false, EN, false>(sp, b, reinterpret_cast<float*>(smem));
  } else {
    // every even block of the planes this block reads or overwrites
    const int4 d = P.deps[b];
    bool late = false;
    for (int i = d.x + (int)threadIdx.x; i < d.y; i += SWEEP_BS)
      late |= !wait_flag(P.flags + i, want, P.timeout_ns);
    for (int i = d.z + (int)threadIdx.x; i < d.w; i += SWEEP_BS)
      late |= !wait_flag(P.flags + i, want, P.timeout_ns);
    if (b == P.inject_block && threadIdx.x == 0) late |= !wait_flag(P.flags + P.never, want, P.timeout_ns);
    __threadfence();
    if (STG) asm volatile("fence.proxy.async.global;" ::: "memory");
    if (__syncthreads_or(late)) {
      if (threadIdx.x == 0) atomicExch(P.err, 1u);
    } else {
      if constexpr (STG) staged_block<F, J16, EN>(sp, b, smem);
      else sweep_block<F, false, J16, false, EN, true>(sp, b, reinterpret_cast<float*>(smem));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (parity == 0) atomicExch(P.flags + b, want);
    if (atomicAdd(P.state + 1, 1u) == (unsigned int)P.n_tickets - 1u) {
      // every block has finished: reset for the next launch
      atomicExch(P.state, 0u);
      atomicExch(P.state + 1, 0u);
      atomicAdd(P.state + 2, 1u);
      __threadfence();
    }
  }
}

template <int F, bool J16, bool EN, bool STG>
cudaError_t launch_w(const WaveParams& p, size_t smem, cudaStream_t st) {
  cudaError_t e = allow_smem(k_wave_sweep<F, J16, EN, STG>, smem);
  if (e != cudaSuccess) return e;
  k_wave_sweep<F, J16, EN, STG><<<p.n_tickets, SWEEP_BS, smem, st>>>(p);
  return cudaGetLastError();
}

template <int F>
cudaError_t launch_wf(bool j16, bool en, bool stg, const WaveParams& p, size_t smem, cudaStream_t st) {
  if (stg) {
    if (j16) return en ? launch_w<F, true, true, true>(p, smem, st) : launch_w<F, true, false, true>(p, smem, st);
    return en ? launch_w<F, false, true, true>(p, smem, st) : launch_w<F, false, false, true>(p, smem, st);
  }
  if (j16) return en ? launch_w<F, true, true, false>(p, smem, st) : launch_w<F, true, false, false>(p, smem, st);
  return en ? launch_w<F, false, true, false>(p, smem, st) : launch_w<F, false, false, false>(p, smem, st);
}

template <int F>
cudaError_t occupancy_f(bool j16, bool stg, size_t smem, int* blocks_per_sm) {
  const void* fn = stg ? (j16 ? (const void*)k_wave_sweep<F, true, false, true>
                              : (const void*)k_wave_sweep<F, false, false, true>)
                       : (j16 ? (const void*)k_wave_sweep<F, true, false, false>
                              : (const void*)k_wave_sweep<F, false, false, false>);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, SWEEP_BS, smem);
}

}  // namespace

bool fmt_has_wave(int fmt) { return fmt == FMT_F32 || fmt == FMT_F16 || fmt == FMT_BF16; }

cudaError_t wave_occupancy(int fmt, bool j16, bool staged, size_t smem, int* blocks_per_sm) {
  switch (fmt) {
    case FMT_F32: return occupancy_f<FMT_F32>(j16, staged, smem, blocks_per_sm);
    case FMT_F16: return occupancy_f<FMT_F16>(j16, staged, smem, blocks_per_sm);
    case FMT_BF16: return occupancy_f<FMT_BF16>(j16, staged, smem, blocks_per_sm);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_wave(int fmt, bool j16, bool energy, bool staged, const WaveParams& p, size_t smem,
                        cudaStream_t st) {
  if (p.n_tickets <= 0) return cudaSuccess;
  switch (fmt) {
    case FMT_F32: return launch_wf<FMT_F32>(j16, energy, staged, p, smem, st);
    case FMT_F16: return launch_wf<FMT_F16>(j16, energy, staged, p, smem, st);
    case FMT_BF16: return launch_wf<FMT_BF16>(j16, energy, staged, p, smem, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hsg

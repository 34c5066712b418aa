// Staged over-relaxation half-sweeps (Sec. 3.1, Eq. 3): the block body that stages its
// data through shared memory instead of loading it into registers.
//
// A block of the sweep block table updates 256 consecutive storage sites of one parity:
// R = 256 / (L/2) whole rows y0 .. y0+R-1 of one plane z (L a power of 2, L >= 32).  Its
// sites read the opposite parity in rows y0-1 .. y0+R of plane z (the +-x and +-y
// neighbours) and in rows y0 .. y0+R-1 of planes z-1 and z+1.  Those rows, and the block's
// own, are contiguous runs of the parity-split layout, so per component plane and chunk
// group they reach shared memory as six (five without the own rows) cp.async.bulk copies
// (the rows y0-1 and y0+R apart, as they wrap in y).  The block walks its chunk groups
// through a two-stage ring: while it computes chunk group g, the copies of g+1 are in
// flight.  Each stage has a full mbarrier carrying the copies' bytes and an empty one that
// its warps arrive at once they have read it.  The copies of the stage's next chunk group
// are issued by one warp, another in each iteration, at the end of its own update, when the
// others have mostly read the stage: no warp waits there for long, and none issues all of
// them.  The update is the per-half-sweep kernel's, in the same operations and order, so the
// results are bit for bit the same.  Every wait is bounded: one that runs out sets the error
// word, and the block stops computing but keeps waiting (bounded) for the copies it issued
// before it exits.
//
// What bounds it: at L = 128 the half-sweep's one pass over each parity in DRAM; with the
// spins in L2 the wait for a stage's copies.  Against the kernel that loads into registers,
// a block reads each row once from L2, and no registers wait for it.  A half-sweep of 48
// systems at L = 128, in registers and staged: FP16 168 and 149 us (149 at the measured
// copy rate), BF16 171 and 155, FP32 290 and 288 (267); L = 64, 128 systems, FP16: 60 and
// 54.  At L = 32 and 256 loading into registers is the faster (64 systems, FP32: 7.2 and
// 8.3; 4 systems, FP16: 269 and 300): the tuner times both.  Heat bath has no staged form:
// its registers spill (361 against 303 us at L = 128).
//
// The row length is a constant of the code for every lattice that has staged rows, with
// the stages unrolled: the offsets are then constants, which is what lets six neighbours
// and the own spins fit into the registers.  A sweep with the row length in a variable
// took 350 us instead of 299 (L = 128, 48 systems, FP16), 21.1 instead of 16.7 (L = 32, 64
// systems, FP32) and 1305 instead of 1044 (L = 256, 4 systems, FP32).
#pragma once
#include "hsg_async.cuh"
#include "hsg_kernels.cuh"

namespace hsg {

constexpr int NW = SWEEP_BS / 32;   // warps per block

// Chunks of one component plane of a stage: rows [y0-1 .. y0+R] of plane z, then rows
// [y0 .. y0+R-1] of planes z-1 and z+1 of the opposite parity, then (own) the block's
// own sites (R Lh = 256).  Own rows where they cost no resident block: from L = 256 on they
// do, and are loaded into registers ahead of the wait instead (L = 256, 4 systems, a sweep:
// FP16 677 us with own rows, 599 without; FP32 1577, 1115).
__host__ __device__ constexpr bool stage_has_own(int Lh) { return Lh <= 64; }
__host__ __device__ constexpr int stage_plane_chunks(int Lh) {
  return (stage_has_own(Lh) ? 4 : 3) * SWEEP_BS + 2 * Lh;
}

// One block of an over-relaxation half-sweep (parity p.parity) with staged rows;
// smem: dynamic shared memory laid out as in staged_smem().  Lh: L / 2 of its sample.
template <int F, bool J16, bool EN, int Lh>
__device__ __forceinline__ void staged_rows(const SweepParams& p, int bidx, unsigned char* smem) {
  constexpr int VEC = FmtInfo<F>::VEC, PL = FmtInfo<F>::PLANES, CH = FmtInfo<F>::CHUNK;
  constexpr int S = STAGED_STAGES;
  constexpr int L = 2 * Lh, R = SWEEP_BS / Lh, pc = stage_plane_chunks(Lh), stage_bytes = PL * pc * CH;
  constexpr bool OWN = stage_has_own(Lh);
  constexpr int KINDS = OWN ? 6 : 5;    // copies per component plane
  using Chunk = typename FmtInfo<F>::Chunk;
  constexpr bool MIXED = (F == FMT_F16) && J16;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);          // a stage's copies have landed
  uint64_t* empty = reinterpret_cast<uint64_t*>(smem + 64);    // every warp has read the stage
  float* esum = reinterpret_cast<float*>(smem + STAGED_HEAD);
  unsigned char* stages = smem + p.stage_off;

  const int4 blk = p.blocks[bidx];
  if (!p.active[blk.x]) {         // a frozen sample (block-uniform)
    chain_wait();
    return;
  }
  const SampleDev& sd = p.samples[blk.x];
  const int par = p.parity;
  const uint32_t half_n = (uint32_t)sd.N >> 1;
  const int g0 = blk.y * p.GPT, g1 = min(p.G, g0 + p.GPT), ng = g1 - g0;
  const int r0 = blk.z / Lh;                  // first row (y + L z) of the block
  const int z = r0 / L, y0 = r0 - z * L;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long gstride = (long long)sd.N * CH;

  // the copy this lane issues for a stage (lanes 0 .. KINDS PL - 1 of the issuing warp)
  long long c_src = 0;
  uint32_t c_dst = 0, c_bytes = 0;
  if (lane < KINDS * PL) {
    const int pl = lane / KINDS, kind = lane - KINDS * (lane / KINDS);
    uint32_t ob = (uint32_t)(1 - par) * half_n;
    int row, dst, nrows = R;
    if (kind == 0) {
      row = (y0 == 0 ? L - 1 : y0 - 1) + L * z, dst = 0, nrows = 1;
    } else if (kind == 1) {
      row = y0 + L * z, dst = Lh;
    } else if (kind == 2) {
      row = (y0 + R == L ? 0 : y0 + R) + L * z, dst = (R + 1) * Lh, nrows = 1;
    } else if (kind == 3) {
      row = y0 + L * (z == 0 ? L - 1 : z - 1), dst = (R + 2) * Lh;
    } else if (kind == 4) {
      row = y0 + L * (z + 1 == L ? 0 : z + 1), dst = (2 * R + 2) * Lh;
    } else {
      ob = (uint32_t)par * half_n;
      row = r0, dst = (3 * R + 2) * Lh;
    }
    c_src = sd.spin_off + (long long)pl * sd.plane_stride + (long long)(ob + (uint32_t)row * Lh) * CH;
    c_dst = (uint32_t)((pl * pc + dst) * CH);
    c_bytes = (uint32_t)(nrows * Lh * CH);
    // HSG_CHECK builds: the rows within their half, the copy within its stage (else
    // copy the same number of bytes from the plane's start: the stage's byte count
    // still completes, the results are flagged)
    if (HSG_OUT_OF_BOUNDS(row >= 0 && (long long)(row + nrows) * Lh <= (long long)half_n &&
                              c_dst + c_bytes <= (uint32_t)stage_bytes,
                          p.bounds_err))
      c_src = sd.spin_off + (long long)pl * sd.plane_stride;
  }
  auto issue = [&](int i) {   // the copies of chunk group g0 + i into stage i % S (one warp)
    const int s = i % S;
    if (lane == 0) mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
    __syncwarp();
    if (c_bytes)
      bulk_copy_g2s(stages + s * stage_bytes + c_dst, p.spins + c_src + (long long)(g0 + i) * gstride,
                    c_bytes, &full[s]);
  };
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // this thread's site, its neighbours' chunk offsets in a stage plane (+x, -x,
  // +y, -y, +z, -z) and its couplings
  const int lr = tid / Lh, hx = tid - lr * Lh;
  const int y = y0 + lr;
  const int x = 2 * hx + ((par + y + z) & 1);
  const int xp = (x + 1 == L) ? 0 : x + 1, xm = (x == 0) ? L - 1 : x - 1;
  int off[6];
  off[0] = (lr + 1) * Lh + (xp >> 1);
  off[1] = (lr + 1) * Lh + (xm >> 1);
  off[2] = (lr + 2) * Lh + hx;
  off[3] = lr * Lh + hx;
  off[4] = (2 * R + 2) * Lh + lr * Lh + hx;
  off[5] = (R + 2) * Lh + lr * Lh + hx;
  uint32_t own = (uint32_t)par * half_n + (uint32_t)blk.z + (uint32_t)tid;
  bool store_ok = true;
  {
    // HSG_CHECK builds: the site in this parity's half and its neighbours within
    // the stage plane (else read in-bounds slots and write nothing back)
    bool bad = HSG_OUT_OF_BOUNDS((uint32_t)blk.z + (uint32_t)tid < half_n, p.bounds_err);
#pragma unroll
    for (int n = 0; n < 6; ++n) bad = bad || HSG_OUT_OF_BOUNDS(off[n] >= 0 && off[n] < pc, p.bounds_err);
    if (bad) {
      own = (uint32_t)par * half_n;
#pragma unroll
      for (int n = 0; n < 6; ++n) off[n] = 0;
      store_ok = false;
    }
  }
  float j6[6], h3[3];
  uint32_t jh[6];
  load_record<J16>(p.rec, sd.rec_off + own, j6, h3);
  if (MIXED) load_record_j16(p.rec, sd.rec_off + own, jh);
  chain_wait();      // spins of the kernels before it from here on
  __syncthreads();
  if (warp == 0) {
    for (int i = 0; i < S && i < ng; ++i) issue(i);
  }
  unsigned char* own_base = p.spins + sd.spin_off + (long long)own * CH;
  const long long ps = sd.plane_stride;

  bool ok = true;
  int i = 0;
  // chunk group g0 + i from stage s (constant in the unrolled loop below); false: a wait ran out
  auto step = [&](int s) {
    const uint32_t ph = (uint32_t)(i / S) & 1u;
    Chunk c[PL];
    if constexpr (!OWN) load_chunks<F, LD_PLAIN>(own_base + (long long)(g0 + i) * gstride, ps, c);
    if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, p.timeout_ns))) return false;
    const unsigned char* st = stages + s * stage_bytes;
    Chunk nc[6][PL];
#pragma unroll
    for (int n = 0; n < 6; ++n)
#pragma unroll
      for (int pl = 0; pl < PL; ++pl)
        nc[n][pl] = *reinterpret_cast<const Chunk*>(st + (pl * pc + off[n]) * CH);
#pragma unroll
    for (int pl = 0; OWN && pl < PL; ++pl)
      c[pl] = *reinterpret_cast<const Chunk*>(st + (pl * pc + (3 * R + 2) * Lh + tid) * CH);

    // local field h = sum_n J_n s_n + H, in the order +x, -x, +y, -y, +z, -z
    Spins<VEC> hf;
    if constexpr (MIXED) {
#pragma unroll
      for (int k = 0; k < VEC / 2; ++k) {
        hf.x[k] = make_float2(0.0f, 0.0f);
        hf.y[k] = make_float2(0.0f, 0.0f);
        hf.z[k] = make_float2(0.0f, 0.0f);
      }
#pragma unroll
      for (int n = 0; n < 6; ++n) {
        fma_f16_pair(hf.x[0], nc[n][0].x, jh[n]);
        fma_f16_pair(hf.x[1], nc[n][0].y, jh[n]);
        fma_f16_pair(hf.y[0], nc[n][1].x, jh[n]);
        fma_f16_pair(hf.y[1], nc[n][1].y, jh[n]);
        fma_f16_pair(hf.z[0], nc[n][2].x, jh[n]);
        fma_f16_pair(hf.z[1], nc[n][2].y, jh[n]);
      }
    } else {
      {
        Spins<VEC> nb;
        decode<F>(nc[0], nb);
        const float2 jj = f2(j6[0]);
#pragma unroll
        for (int k = 0; k < VEC / 2; ++k) {
          hf.x[k] = mul2(jj, nb.x[k]);
          hf.y[k] = mul2(jj, nb.y[k]);
          hf.z[k] = mul2(jj, nb.z[k]);
        }
      }
#pragma unroll
      for (int n = 1; n < 6; ++n) {
        Spins<VEC> nb;
        decode<F>(nc[n], nb);
        const float2 jj = f2(j6[n]);
#pragma unroll
        for (int k = 0; k < VEC / 2; ++k) {
          hf.x[k] = fma2(jj, nb.x[k], hf.x[k]);
          hf.y[k] = fma2(jj, nb.y[k], hf.y[k]);
          hf.z[k] = fma2(jj, nb.z[k], hf.z[k]);
        }
      }
    }
    Spins<VEC> sv;
    decode<F>(c, sv);
    // every staged value is in registers: this warp is done with the stage
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    {
      const float2 hx2 = f2(h3[0]), hy2 = f2(h3[1]), hz2 = f2(h3[2]);
#pragma unroll
      for (int k = 0; k < VEC / 2; ++k) {
        hf.x[k] = add2(hf.x[k], hx2);
        hf.y[k] = add2(hf.y[k], hy2);
        hf.z[k] = add2(hf.z[k], hz2);
      }
    }
#pragma unroll
    for (int k = 0; k < VEC / 2; ++k) {
      if constexpr (F == FMT_F32) or_move2(sv.x[k], sv.y[k], sv.z[k], hf.x[k], hf.y[k], hf.z[k]);
      else or_move2_branch(sv.x[k], sv.y[k], sv.z[k], hf.x[k], hf.y[k], hf.z[k]);
    }
    encode<F>(sv, c);
    if (store_ok) store_chunks<F>(own_base + (long long)(g0 + i) * gstride, ps, c);
    if constexpr (EN) {
      // energy of the new state from the stored values: every bond joins one
      // odd and one even site, E = - sum_odd s_i.h_i - sum_even H_j.s_j
      Spins<VEC> stv;
      float e[VEC];
      decode<F>(c, stv);
#pragma unroll
      for (int k = 0; k < VEC / 2; ++k) {
        float2 d;
        if (par == 1) {
          d = dot3_2(stv.x[k], stv.y[k], stv.z[k], hf.x[k], hf.y[k], hf.z[k]);
        } else {
          d = dot3_2(stv.x[k], stv.y[k], stv.z[k], f2(h3[0]), f2(h3[1]), f2(h3[2]));
        }
        e[2 * k] = -d.x;
        e[2 * k + 1] = -d.y;
      }
      static_assert(VEC == 4, "the scattered warp sum takes four systems per chunk");
      const float t = warp_sum4_scatter(e, lane);
      if ((lane & 7) == 0) esum[warp * p.GPT * VEC + i * VEC + (lane >> 3)] = t;
    }
    // refill the stage with the chunk group S further on, one warp after the other in
    // turn: by the end of its own update the others have read the stage, as a rule
    if (i + S < ng && warp == (i & (NW - 1))) {
      if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, p.timeout_ns))) return false;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(i + S);
    }
    return true;
  };
  static_assert(S == 2, "unrolled over two stages: their offsets are constants");
  while (i < ng) {
    if (!(ok = step(0))) break;
    if (++i == ng) break;
    if (!(ok = step(1))) break;
    ++i;
  }
  if (!ok) {
    // a wait ran out: flag it and give the copies in flight a bounded time to
    // land before the block's shared memory is released
    if (lane == 0) atomicExch(p.err, 1u);
    for (int q = i; q < ng && q < i + S; ++q)
      mbar_wait(&full[q % S], (uint32_t)(q / S) & 1u, p.timeout_ns);
  }
  if constexpr (EN) {
    __syncthreads();
    double* out = p.epart + ((long long)par * p.n_blocks + bidx) * p.Wp;
    for (int jj = tid; jj < ng * VEC; jj += SWEEP_BS) {
      double acc = 0.0;
      for (int w = 0; w < NW; ++w) acc += (double)esum[w * p.GPT * VEC + jj];
      out[g0 * VEC + jj] = acc;
    }
  }
  __syncthreads();   // the ring and its barriers are reused by nothing after this
}

// The block's lattice (every L that lattice_has_staged), its row length in constants: the
// context's where its lattices are all alike, else its sample's.
template <int F, bool J16, bool EN>
__device__ __forceinline__ void staged_block(const SweepParams& p, int bidx, unsigned char* smem) {
  switch (p.one_Lh ? p.one_Lh : p.samples[p.blocks[bidx].x].Lh) {
    case 16: return staged_rows<F, J16, EN, 16>(p, bidx, smem);
    case 32: return staged_rows<F, J16, EN, 32>(p, bidx, smem);
    case 64: return staged_rows<F, J16, EN, 64>(p, bidx, smem);
    case 128: return staged_rows<F, J16, EN, 128>(p, bidx, smem);
    case 256: return staged_rows<F, J16, EN, 256>(p, bidx, smem);
  }
  chain_wait();
  HSG_OUT_OF_BOUNDS(false, p.bounds_err);
}

// Lh: L / 2 of every sample of the context, or 0 (lattices of several sizes)
template <int F, bool J16, bool EN, int Lh>
__global__ void __launch_bounds__(SWEEP_BS, 4) k_staged_half(const SweepParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  chain_trigger();
  const int k = p.blk_base + (p.reverse ? p.n_launch - 1 - (int)blockIdx.x : (int)blockIdx.x);
  if constexpr (Lh > 0) staged_rows<F, J16, EN, Lh>(p, k, smem);
  else staged_block<F, J16, EN>(p, k, smem);
}

template <int F, bool J16, bool EN, int Lh>
cudaError_t launch_staged_h(const SweepParams& p, int n_blocks, size_t smem, cudaStream_t st) {
  const cudaError_t e = allow_smem(k_staged_half<F, J16, EN, Lh>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(k_staged_half<F, J16, EN, Lh>, n_blocks, SWEEP_BS, smem, st, p);
}

template <int F, int Lh>
cudaError_t launch_staged_f(bool j16, bool en, const SweepParams& p, int n_blocks, size_t smem, cudaStream_t st) {
  if (j16)
    return en ? launch_staged_h<F, true, true, Lh>(p, n_blocks, smem, st)
              : launch_staged_h<F, true, false, Lh>(p, n_blocks, smem, st);
  return en ? launch_staged_h<F, false, true, Lh>(p, n_blocks, smem, st)
            : launch_staged_h<F, false, false, Lh>(p, n_blocks, smem, st);
}

template <int Lh>
cudaError_t launch_staged_l(int fmt, bool j16, bool en, const SweepParams& p, int n_blocks, size_t smem,
                            cudaStream_t st) {
  switch (fmt) {
    case FMT_F32: return launch_staged_f<FMT_F32, Lh>(j16, en, p, n_blocks, smem, st);
    case FMT_F16: return launch_staged_f<FMT_F16, Lh>(j16, en, p, n_blocks, smem, st);
    case FMT_BF16: return launch_staged_f<FMT_BF16, Lh>(j16, en, p, n_blocks, smem, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hsg

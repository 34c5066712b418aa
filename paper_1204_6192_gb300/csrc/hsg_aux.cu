// Reductions and bookkeeping kernels: FP64 energies (Eq. 1), the parallel
// tempering pass (Eq. 4), the overlap measurements (Eq. 5 and its
// k-dependent form), the random initial state and the conversions between
// the stored spin formats and FP32 (x, y, z).
//
// Every reduction is deterministic: per-thread partial sums, a fixed-order
// shuffle/shared-memory tree inside a block, and a second kernel that adds the
// block partials in a fixed order.  Two runs give bit-identical results.
#include "hsg_kernels.cuh"

namespace hsg {

// ---------------------------------------------------------------------------
// Energies.  Every bond joins an odd and an even site, so
//   E = - sum_{odd i} s_i . h_i  - sum_{even j} H_j . s_j
// with h_i the full local field (bonds + field) of the odd site i.  Latency-bound:
// 64 registers keep 32 warps on an SM and the eight warp sums of a chunk take 12
// shuffles instead of 40 (L = 64, BF16, 64 systems: 74 -> 33 us; its bytes take 15).
// ---------------------------------------------------------------------------
template <int F, bool J16>
__global__ void __launch_bounds__(RED_BS, F == FMT_YX4 ? 0 : 4) k_energy(const EnergyParams p) {
  constexpr int VEC = FmtInfo<F>::VEC, PL = FmtInfo<F>::PLANES;
  constexpr uint32_t CH = FmtInfo<F>::CHUNK;
  using Chunk = typename FmtInfo<F>::Chunk;
  extern __shared__ float esum[];                 // [2][RED_BS / 32][GPT * VEC]
  chain_trigger();
  const int4 blk = p.blocks[blockIdx.x];
  const SampleDev& sd = p.samples[blk.x];
  const uint32_t half_n = (uint32_t)sd.N >> 1;
  const bool active = (uint32_t)blk.z + threadIdx.x < half_n;
  const uint32_t h = min((uint32_t)blk.z + threadIdx.x, half_n - 1);   // (idle threads: the last site, unused)
  const int g0 = blk.y * p.GPT;
  const int g1 = min(p.G, g0 + p.GPT);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stride = p.GPT * VEC;
  float* esum_even = esum;
  float* esum_odd = esum + (RED_BS / 32) * stride;

  const unsigned char* base = p.spins + sd.spin_off;
  const long long ps = sd.plane_stride;
  const long long gstride = (long long)sd.N * CH;
  float j6[6], h3[3], je[6], he[3];
  const SiteGeom gm = site_geom(sd, h, 1);       // the odd site with half-index h
  load_record<J16>(p.rec, sd.rec_off + gm.own, j6, h3);
  load_record<J16>(p.rec, sd.rec_off + h, je, he);   // even site with the same half-index
  uint32_t nb_off[6];
#pragma unroll
  for (int n = 0; n < 6; ++n) nb_off[n] = gm.nb[n] * CH;
  chain_wait();
  for (int g = g0; g < g1; ++g) {
    const unsigned char* base_g = base + (long long)g * gstride;
    Chunk nc[6][PL], co[PL], ce[PL];
#pragma unroll
    for (int n = 0; n < 6; ++n) load_chunks_at<F, LD_PLAIN>(base_g, ps, nb_off[n], nc[n]);
    load_chunks_at<F, LD_PLAIN>(base_g, ps, gm.own * CH, co);
    load_chunks_at<F, LD_PLAIN>(base_g, ps, h * CH, ce);
    Spins<VEC> hf, t;
    decode<F>(nc[0], t);
#pragma unroll
    for (int q = 0; q < VEC / 2; ++q) {
      hf.x[q] = mul2(f2(j6[0]), t.x[q]);
      hf.y[q] = mul2(f2(j6[0]), t.y[q]);
      hf.z[q] = mul2(f2(j6[0]), t.z[q]);
    }
#pragma unroll
    for (int n = 1; n < 6; ++n) {
      decode<F>(nc[n], t);
#pragma unroll
      for (int q = 0; q < VEC / 2; ++q) {
        hf.x[q] = fma2(f2(j6[n]), t.x[q], hf.x[q]);
        hf.y[q] = fma2(f2(j6[n]), t.y[q], hf.y[q]);
        hf.z[q] = fma2(f2(j6[n]), t.z[q], hf.z[q]);
      }
    }
    Spins<VEC> so, se;
    decode<F>(co, so);
    decode<F>(ce, se);
    float eo[VEC], ee[VEC];
#pragma unroll
    for (int q = 0; q < VEC / 2; ++q) {
      const float2 hx2 = add2(hf.x[q], f2(h3[0]));
      const float2 hy2 = add2(hf.y[q], f2(h3[1]));
      const float2 hz2 = add2(hf.z[q], f2(h3[2]));
      const float2 o = dot3_2(so.x[q], so.y[q], so.z[q], hx2, hy2, hz2);
      const float2 e = dot3_2(se.x[q], se.y[q], se.z[q], f2(he[0]), f2(he[1]), f2(he[2]));
      eo[2 * q] = active ? -o.x : 0.0f;
      eo[2 * q + 1] = active ? -o.y : 0.0f;
      ee[2 * q] = active ? -e.x : 0.0f;
      ee[2 * q + 1] = active ? -e.y : 0.0f;
    }
    const float to = warp_sum4_scatter(eo, lane), te = warp_sum4_scatter(ee, lane);
    if ((lane & 7) == 0) {
      esum_odd[warp * stride + (g - g0) * VEC + (lane >> 3)] = to;
      esum_even[warp * stride + (g - g0) * VEC + (lane >> 3)] = te;
    }
  }
  __syncthreads();
  for (int jj = threadIdx.x; jj < (g1 - g0) * VEC; jj += RED_BS) {
    double ae = 0.0, ao = 0.0;
    for (int w = 0; w < RED_BS / 32; ++w) {
      ae += (double)esum_even[w * stride + jj];
      ao += (double)esum_odd[w * stride + jj];
    }
    const int j = g0 * VEC + jj;
    p.partials[(long long)blockIdx.x * p.Wp + j] = ae;
    p.partials[((long long)p.n_blocks + blockIdx.x) * p.Wp + j] = ao;
  }
}

// ---------------------------------------------------------------------------
// The tail of a step in one launch: the FP64 energy sums (SUM; Eq. 1) and the
// parallel-tempering pass (PT; Eq. 4).  Block (split, wg, s) adds split `split` of
// the systems 32 wg .. 32 wg + 31 of sample s (energy_rows); the last block of a
// sample to finish (a ticket per sample) adds the splits and runs the sample's
// chains, and advances its counters.
//
// The PT pass visits the pairs (k, k+1) from the lowest temperature up and an
// accepted pair swaps the two configurations, so pair k compares the
// configuration that slot k+1 held before the pass with one carried up from some
// slot j <= k: slot k's own when pair k-1 was rejected.  Whatever j will be, its
// decision depends only on the energies and the pair's uniform, so all
// (j <= k) decisions are taken at once, one warp per pair and 32 values of j (with
// fewer temperatures several pairs a warp: its instructions cost the
// same for 8 lanes as for 32), each exactly as the sequential walk would take it.  What is
// left of the sequential walk is one bit test per pair.  (R_T = 32: the walk with its
// FP64 arithmetic and exponentials in the chain took 18 us and the sums before it 2.4; one launch now
// takes 11 in all.)  R_T^2 / 2 decisions are many for long chains, and FP64 runs at two
// lanes a clock and SM, so a decision is taken from the energies' two binary32 parts
// where those leave no doubt (R_T = 256, R_O = 4, hsg_pt_exchange: 428 us with every
// difference in FP64, 179 now, 283 with the sequential walk).
// ---------------------------------------------------------------------------
constexpr int TAIL_BS = 256;
constexpr int TAIL_MASKS = 4096;      // decision words in shared memory: the chains run in batches
constexpr int MAX_W = 1024, MAX_R_T = 256;   // limits of a context

template <bool SUM, bool PT>
__global__ void __launch_bounds__(TAIL_BS) k_energy_tail(const EnergyParams e, const PTParams p) {
  __shared__ double sE[PT ? MAX_W : 1], sib[PT ? MAX_R_T : 1];   // energies by memory slot; inverse temperatures
  __shared__ int sperm[PT ? MAX_W : 1];         // the permutations before the pass
  __shared__ float su[PT ? MAX_W : 1];          // the pairs' uniforms
  __shared__ float2 sEf[PT ? MAX_W : 1];        // the same by slot: leading and trailing binary32 parts
  __shared__ float sdb[PT ? MAX_R_T : 1];       // beta of slot k + 1 less that of slot k
  __shared__ __align__(16) uint32_t mask[PT ? TAIL_MASKS : 512];   // [chain of the batch][pair][j / 32]
  __shared__ uint16_t walk[PT ? MAX_W : 1];     // [chain][slot]: carried j, bit 15: pair accepted
  __shared__ unsigned char sts[PT ? MAX_W : 1]; // tunnelling states
  __shared__ bool s_last;
  double (*red)[32] = reinterpret_cast<double (*)[32]>(mask);   // [8][32], the sums' before the decisions
  chain_trigger();
  const int s = blockIdx.y, tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const unsigned char* active = SUM ? e.active : p.active;
  const bool frozen = !active[s];
  const int R = PT ? p.R_T : 1, R1 = R - 1, nw = (R + 31) / 32, W = PT ? p.R_O * R : 0;
  const int c0 = PT ? s * p.R_O : 0;
  if (PT)
    for (int i = tid; i < R; i += TAIL_BS) sib[i] = p.inv_temps[(long long)s * R + i];
  chain_wait();
  if (frozen) return;   // frozen sample (every block of it): energies, chains and counters stand
  // the chains' state, on its way while the sums run
  constexpr int PER = MAX_W / TAIL_BS;
  int conf[PT ? PER : 1];
  unsigned char ts[PT ? PER : 1];
  uint32_t step = 0;
  if constexpr (PT) {
    step = (uint32_t)p.counters[2 * s + 1];     // the sample's PT passes key its uniforms
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int i = tid + m * TAIL_BS;
      if (i < W) {
        conf[m] = p.perm[(long long)c0 * R + i];
        ts[m] = p.tstate[(long long)c0 * R + i];
      }
    }
  }
  if constexpr (SUM) {
    const int wgs = (e.Wp + 31) / 32;
    const int wg = blockIdx.x % wgs, split = blockIdx.x / wgs;
    double* dst = e.splits == 1 ? e.E + (long long)s * e.Wp
                                : e.partials2 + ((long long)s * e.splits + split) * e.Wp;
    const int w = wg * 32 + tx;
    const double t = energy_lanes(w < e.Wp ? energy_rows<false>(e, s, w, split, ty) : 0.0, tx, ty, red);
    if (ty == 0 && w < e.Wp) {
      dst[w] = t;
      if (PT && gridDim.x == 1) sE[w] = t;
    }
    if (gridDim.x > 1) {
      __threadfence();
      __syncthreads();
      if (tid == 0) s_last = atomicAdd(e.tickets + s, 1u) == gridDim.x - 1;
      __syncthreads();
      if (!s_last) return;
      if (tid == 0) e.tickets[s] = 0u;
      __threadfence();
      const bool few = e.splits <= E_FEW_SPLITS;   // a warp adds a group's splits by itself, in order
      for (int g = ty; few && g < wgs; g += TAIL_BS / 32) {
        const int v = g * 32 + tx;
        if (v >= e.Wp) continue;
        const double* src = e.splits == 1 ? e.E + (long long)s * e.Wp : e.partials2 + (long long)s * e.splits * e.Wp;
        double t = 0.0;
        for (int k = 0; k < e.splits; ++k) t += __ldcg(src + (long long)k * e.Wp + v);
        if (e.splits > 1) e.E[(long long)s * e.Wp + v] = t;
        if (PT) sE[v] = t;
      }
      for (int g = 0; !few && g < wgs; ++g) {
        const int v = g * 32 + tx;
        double acc = 0.0;
        if (v < e.Wp) {
          const double* src = e.splits == 1 ? e.E + (long long)s * e.Wp : e.partials2 + (long long)s * e.splits * e.Wp;
#pragma unroll 4
          for (int k = ty; k < e.splits; k += 8) acc += __ldcg(src + (long long)k * e.Wp + v);
        }
        acc = energy_lanes(acc, tx, ty, red);
        if (ty == 0 && v < e.Wp) {
          if (e.splits > 1) e.E[(long long)s * e.Wp + v] = acc;
          if (PT) sE[v] = acc;
        }
      }
    }
  } else if constexpr (PT) {
    for (int i = tid; i < W; i += TAIL_BS) sE[i] = p.E[(long long)s * p.Wp + i];
  }
  if constexpr (PT) {
#pragma unroll
    for (int m = 0; m < PER; ++m) {
      const int i = tid + m * TAIL_BS;
      if (i < W) {
        sperm[i] = conf[m];
        sts[i] = ts[m];
        if (R1 > 0)
          su[i] = u01(philox4x32_10(make_uint4((uint32_t)(i % R), (uint32_t)(c0 + i / R), step, TAG_PT),
                                    p.seed_lo, p.seed_hi).x);
      }
    }
    __syncthreads();
    for (int i = tid; i < W; i += TAIL_BS) {
      const double E = sE[i / R * R + sperm[i]];
      const float hi = (float)E;
      sEf[i] = make_float2(hi, (float)(E - (double)hi));
    }
    for (int i = tid; i < R1; i += TAIL_BS) sdb[i] = (float)(sib[i + 1] - sib[i]);
    __syncthreads();
    int tw = 1;                  // lanes of a pair's word: its j <= k < R1
    while (tw < min(R1, 32)) tw <<= 1;
    const int batch = R1 > 0 ? TAIL_MASKS / (R1 * nw) : p.R_O;
    for (int b0 = 0; b0 < p.R_O; b0 += batch) {
      const int nb = min(batch, p.R_O - b0);
      const int n = nb * R1;
      for (int q0 = ty * (32 / tw); q0 < n; q0 += TAIL_BS / tw) {
        const int q = min(q0 + tx / tw, n - 1), c = q / R1, k = q - c * R1, at = (b0 + c) * R;
        const float2 b = sEf[at + k + 1];
        const float db = sdb[k], u = su[at + k];
        // (words above k are read by no walk; tw < 32: one word a pair)
#pragma unroll 2
        for (int jw = 0; jw < nw && (tw < 32 || jw * 32 <= k); ++jw) {
          const int j = jw * 32 + tx % tw;
          bool acc = false;
          if (j <= k) {
            // x = dbeta dE in binary32, within 3e-7 of its value (the difference of the
            // leading parts, each a multiple of its last place, rounds once; the trailing
            // parts reach 2^-48 of the energies): decided where that leaves no doubt,
            // i.e. where dE is above the parts' resolution, no operand is subnormal or
            // out of range, and u is not within 1e-5 of exp(x) <= 1; else by pt_accept
            const float2 a = sEf[at + j];
            const float dEf = __fadd_rn(__fsub_rn(b.x, a.x), __fsub_rn(b.y, a.y));
            const float xf = __fmul_rn(db, dEf);
            const float mag = fabsf(xf), lim = __fmul_rn(1e-6f, fabsf(a.x) + fabsf(b.x));
            const float ex = expf(fmaxf(xf, -20.0f));
            if (fabsf(dEf) > lim && mag > 1e-30f && mag < 1e30f && fabsf(db) > 1e-30f &&
                (xf > 0.0f || xf < -17.1f || fabsf(u - ex) > 1e-5f * ex)) {
              acc = xf > 0.0f || (xf >= -17.1f && u < ex);
            } else {
              const double dbeta = sib[k + 1] - sib[k];
              const double dE = sE[at + sperm[at + k + 1]] - sE[at + sperm[at + j]];
              acc = pt_accept(dbeta * dE, u);
            }
          }
          const uint32_t m = __ballot_sync(0xffffffffu, acc) >> (tx & ~(tw - 1));
          if (tx % tw == 0) mask[q * nw + jw] = tw == 32 ? m : m & ((1u << tw) - 1u);
        }
      }
      __syncthreads();
      for (int c = tid; c < nb; c += TAIL_BS) {
        uint16_t* wk = walk + (b0 + c) * R;
        int j = 0;
        if (nw == 1) {
          const uint32_t* m = mask + c * R1;
#pragma unroll 8
          for (int k = 0; k < R1; ++k) {
            const uint32_t acc = (m[k] >> j) & 1u;
            wk[k] = (uint16_t)(j | (acc << 15));
            j = acc ? j : k + 1;
          }
        } else {
          for (int k = 0; k < R1; ++k) {
            const uint32_t acc = (mask[(c * R1 + k) * nw + (j >> 5)] >> (j & 31)) & 1u;
            wk[k] = (uint16_t)(j | (acc << 15));
            j = acc ? j : k + 1;
          }
        }
        wk[R1] = (uint16_t)j;
      }
      __syncthreads();
    }
    // the new permutations, inverse temperatures and diagnostics: the
    // configuration that held slot k before the pass moved iff pair (k-1, k) moved
    // it down or, failing that, pair (k, k+1) moved it up
    auto holder = [&](int i) {   // configuration that holds slot i % R of chain i / R after the pass
      const int v = walk[i];
      return (v & 0x8000) ? sperm[i + 1] : sperm[i / R * R + v];
    };
    for (int i = tid; i < W; i += TAIL_BS) {
      const int c = i / R, k = i - c * R;
      const int cf = holder(i);
      const bool acc = walk[i] & 0x8000, prev = k > 0 && (walk[i - 1] & 0x8000);
      p.perm[(long long)c0 * R + i] = cf;
      p.beta[(long long)s * p.Wp + c * R + cf] = (float)sib[k];
      if (acc || prev) atomicAdd(p.moved + (long long)c0 * R + i, 1ull);
      if (acc) atomicAdd(p.accepted + (long long)(c0 + c) * R1 + k, 1ull);
    }
    if (R > 1) {
      // tunnelling: a configuration that reaches T_1 after T_R after T_1 closes a loop
      for (int c = tid; c < p.R_O; c += TAIL_BS) {
        const int bottom = holder(c * R), top = holder(c * R + R1);
        unsigned char* out = p.tstate + (long long)(c0 + c) * R;
        if (sts[c * R + bottom] == 2) atomicAdd(p.tunnel + (long long)(c0 + c) * R + bottom, 1u);
        out[bottom] = 1;
        if (sts[c * R + top] == 1) out[top] = 2;
      }
    }
    if (tid == 0) {
      atomicAdd(p.counters + 2 * s, (unsigned long long)p.sweeps_per_call);
      atomicAdd(p.counters + 2 * s + 1, 1ull);
    }
  }
}

static dim3 tail_grid(const EnergyParams& e) {
  return dim3(e.splits * ((e.Wp + 31) / 32), e.n_samples);
}

cudaError_t launch_energy_sums(const EnergyParams& e, cudaStream_t st) {
  return launch_chained(k_energy_tail<true, false>, tail_grid(e), TAIL_BS, 0, st, e, PTParams{});
}

cudaError_t launch_energy_sums_pt(const EnergyParams& e, const PTParams& p, cudaStream_t st) {
  return launch_chained(k_energy_tail<true, true>, tail_grid(e), TAIL_BS, 0, st, e, p);
}

cudaError_t launch_pt(const PTParams& p, cudaStream_t st) {
  return launch_chained(k_energy_tail<false, true>, dim3(1, p.n_samples), TAIL_BS, 0, st, EnergyParams{}, p);
}

template <int F, bool J16>
static cudaError_t energy_fmt(const EnergyParams& p, cudaStream_t st) {
  // (up to 64 kB: a thread may walk all 256 chunk groups of 1024 systems)
  const size_t smem = sizeof(float) * 2 * (RED_BS / 32) * p.GPT * FmtInfo<F>::VEC;
  const cudaError_t e = allow_smem(k_energy<F, J16>, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(k_energy<F, J16>, p.n_blocks, RED_BS, smem, st, p);
}

cudaError_t launch_energy_partials(int fmt, bool j16, const EnergyParams& p, cudaStream_t st) {
  switch (fmt) {
    case FMT_F32: return j16 ? energy_fmt<FMT_F32, true>(p, st) : energy_fmt<FMT_F32, false>(p, st);
    case FMT_F16: return j16 ? energy_fmt<FMT_F16, true>(p, st) : energy_fmt<FMT_F16, false>(p, st);
    case FMT_BF16: return j16 ? energy_fmt<FMT_BF16, true>(p, st) : energy_fmt<FMT_BF16, false>(p, st);
    case FMT_ANG16: return j16 ? energy_fmt<FMT_ANG16, true>(p, st) : energy_fmt<FMT_ANG16, false>(p, st);
    case FMT_OCT16: return j16 ? energy_fmt<FMT_OCT16, true>(p, st) : energy_fmt<FMT_OCT16, false>(p, st);
    case FMT_YX4: return j16 ? energy_fmt<FMT_YX4, true>(p, st) : energy_fmt<FMT_YX4, false>(p, st);
  }
  return cudaErrorInvalidValue;
}

__global__ void k_bump(unsigned long long* counters, const unsigned char* active, int n_samples,
                       int sweeps, int pts) {
  chain_trigger();
  chain_wait();
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n_samples; s += gridDim.x * blockDim.x) {
    if (!active[s]) continue;
    counters[2 * s] += (unsigned long long)sweeps;
    counters[2 * s + 1] += (unsigned long long)pts;
  }
}

cudaError_t launch_bump(unsigned long long* counters, const unsigned char* active, int n_samples,
                        int sweeps, int pts, cudaStream_t st) {
  return launch_chained(k_bump, (n_samples + 255) / 256, 256, 0, st, counters, active, n_samples, sweeps, pts);
}


// ---------------------------------------------------------------------------
// Initial state and conversions.  One thread per (site, chunk), all sites.
// ---------------------------------------------------------------------------
struct ConvItem {
  const SampleDev* sd;
  uint32_t site, g, ss;
  bool ok;
};

// Block (sample, chunk g, first site): one thread per site of chunk g.
__device__ __forceinline__ ConvItem conv_item(const ConvParams& p) {
  ConvItem it;
  const int4 blk = p.blocks[blockIdx.x];
  it.sd = &p.samples[blk.x];
  it.g = (uint32_t)blk.y;
  it.site = (uint32_t)blk.z + threadIdx.x;
  const uint32_t N = (uint32_t)it.sd->N;
  it.ok = it.site < N;
  if (!it.ok) return it;
  const uint32_t L = it.sd->L;
  const uint32_t r = (__umulhi(it.site, it.sd->fdL_m) + it.site) >> it.sd->fdL_s;
  const uint32_t x = it.site - r * L;
  const uint32_t z = (__umulhi(r, it.sd->fdL_m) + r) >> it.sd->fdL_s;
  const uint32_t y = r - z * L;
  it.ss = ((x + y + z) & 1u) * (N >> 1) + (it.site >> 1);
  return it;
}

template <int F>
__global__ void k_init(const ConvParams p) {
  constexpr int VEC = FmtInfo<F>::VEC, PL = FmtInfo<F>::PLANES;
  const ConvItem it = conv_item(p);
  if (!it.ok) return;
  Spins<VEC> s;
  const uint32_t sys0 = (uint32_t)it.sd->sys_base + it.g * VEC;
#pragma unroll
  for (int k = 0; k < VEC / 2; ++k) {
    const uint4 r = philox4x32_10(make_uint4(it.site, (sys0 >> 1) + k, 0u, TAG_INIT),
                                  p.seed_lo, p.seed_hi);
    double v[2][3];
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const double u1 = (double)u01(w[2 * b]), u2 = (double)u01(w[2 * b + 1]);
      const double zc = 2.0 * u1 - 1.0;
      const double rho = 2.0 * sqrt(u1 * (1.0 - u1));
      double sp, cp;
      sincospi(2.0 * u2, &sp, &cp);
      v[b][0] = rho * cp;
      v[b][1] = rho * sp;
      v[b][2] = zc;
    }
    s.x[k] = make_float2((float)v[0][0], (float)v[1][0]);
    s.y[k] = make_float2((float)v[0][1], (float)v[1][1]);
    s.z[k] = make_float2((float)v[0][2], (float)v[1][2]);
  }
  typename FmtInfo<F>::Chunk c[PL];
  encode<F>(s, c);
  unsigned char* o = p.spins + it.sd->spin_off + chunk_offset<F>(*it.sd, it.g, it.ss);
  store_chunks<F>(o, it.sd->plane_stride, c);
}

template <int F>
__global__ void k_get(const ConvParams p) {
  constexpr int VEC = FmtInfo<F>::VEC, PL = FmtInfo<F>::PLANES;
  chain_trigger();
  const ConvItem it = conv_item(p);
  const int sidx = p.blocks[blockIdx.x].x;
  chain_wait();
  if (!it.ok) return;
  const unsigned char* o = p.spins + it.sd->spin_off + chunk_offset<F>(*it.sd, it.g, it.ss);
  typename FmtInfo<F>::Chunk c[PL];
  load_chunks<F, LD_PLAIN>(o, it.sd->plane_stride, c);
  Spins<VEC> s;
  decode<F>(c, s);
  float* out = p.xyz + p.xyz_off[sidx];
  const long long N = it.sd->N;
#pragma unroll
  for (int k = 0; k < VEC / 2; ++k) {
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int w = (int)it.g * VEC + 2 * k + b;
      if (w < p.W) {
        float* q = out + ((long long)w * N + it.site) * 3;
        q[0] = b ? s.x[k].y : s.x[k].x;
        q[1] = b ? s.y[k].y : s.y[k].x;
        q[2] = b ? s.z[k].y : s.z[k].x;
      }
    }
  }
}

template <int F>
__global__ void k_set(const ConvParams p) {
  constexpr int VEC = FmtInfo<F>::VEC, PL = FmtInfo<F>::PLANES;
  const ConvItem it = conv_item(p);
  if (!it.ok) return;
  const int sidx = p.blocks[blockIdx.x].x;
  const float* in = p.xyz + p.xyz_off[sidx];
  const long long N = it.sd->N;
  Spins<VEC> s;
#pragma unroll
  for (int k = 0; k < VEC / 2; ++k) {
    float v[2][3];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int w = (int)it.g * VEC + 2 * k + b;
      if (w < p.W) {
        const float* q = in + ((long long)w * N + it.site) * 3;
        v[b][0] = q[0];
        v[b][1] = q[1];
        v[b][2] = q[2];
      } else {
        v[b][0] = 0.0f;
        v[b][1] = 0.0f;
        v[b][2] = 1.0f;
      }
    }
    s.x[k] = make_float2(v[0][0], v[1][0]);
    s.y[k] = make_float2(v[0][1], v[1][1]);
    s.z[k] = make_float2(v[0][2], v[1][2]);
  }
  typename FmtInfo<F>::Chunk c[PL];
  encode<F>(s, c);
  unsigned char* o = p.spins + it.sd->spin_off + chunk_offset<F>(*it.sd, it.g, it.ss);
  store_chunks<F>(o, it.sd->plane_stride, c);
}

// The heat bath's generator (round keys precomputed) on a list of counters.
__global__ void k_philox(const uint4* ctr, long long n, const SweepParams p, uint4* out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = philox4x32_10_rk(ctr[i], p.rk);
}

cudaError_t launch_philox(const uint4* ctr, long long n, const SweepParams& p, uint4* out,
                          cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_philox<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ctr, n, p, out);
  return cudaGetLastError();
}

#define HSG_CONV_SWITCH(KERNEL)                                                          \
  switch (fmt) {                                                                        \
    case FMT_F32: KERNEL<FMT_F32><<<nb, 256, 0, st>>>(p); break;                        \
    case FMT_F16: KERNEL<FMT_F16><<<nb, 256, 0, st>>>(p); break;                        \
    case FMT_BF16: KERNEL<FMT_BF16><<<nb, 256, 0, st>>>(p); break;                      \
    case FMT_ANG16: KERNEL<FMT_ANG16><<<nb, 256, 0, st>>>(p); break;                    \
    case FMT_OCT16: KERNEL<FMT_OCT16><<<nb, 256, 0, st>>>(p); break;                    \
    case FMT_YX4: KERNEL<FMT_YX4><<<nb, 256, 0, st>>>(p); break;                        \
    default: return cudaErrorInvalidValue;                                              \
  }                                                                                     \
  return cudaGetLastError();

cudaError_t launch_init(int fmt, const ConvParams& p, int nb, cudaStream_t st) {
  HSG_CONV_SWITCH(k_init)
}
cudaError_t launch_get(int fmt, const ConvParams& p, int nb, cudaStream_t st) {
  switch (fmt) {
    case FMT_F32: return launch_chained(k_get<FMT_F32>, nb, 256, 0, st, p);
    case FMT_F16: return launch_chained(k_get<FMT_F16>, nb, 256, 0, st, p);
    case FMT_BF16: return launch_chained(k_get<FMT_BF16>, nb, 256, 0, st, p);
    case FMT_ANG16: return launch_chained(k_get<FMT_ANG16>, nb, 256, 0, st, p);
    case FMT_OCT16: return launch_chained(k_get<FMT_OCT16>, nb, 256, 0, st, p);
    case FMT_YX4: return launch_chained(k_get<FMT_YX4>, nb, 256, 0, st, p);
  }
  return cudaErrorInvalidValue;
}
cudaError_t launch_set(int fmt, const ConvParams& p, int nb, cudaStream_t st) {
  HSG_CONV_SWITCH(k_set)
}

}  // namespace hsg

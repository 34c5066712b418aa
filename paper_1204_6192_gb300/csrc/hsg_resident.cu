// The sweeps of a step with the lattice resident in shared memory, for lattices of
// at most 896 sites of one parity (L <= 12).
//
// Systems meet only in the parallel-tempering pass, so all n_hb + n_or sweeps of a
// step can run on one pair of systems of one sample without looking at any other.
// A block owns one such pair: a thread owns one half-index, i.e. one site of each
// parity, and keeps the sites' couplings, neighbour indices and spins in registers;
// shared memory holds the spins for the neighbours (binary16 / bfloat16 components
// as stored, every other format decoded to binary32: once per update instead of at
// each of its six uses).  A block barrier stands between half-sweeps in place of a
// launch, and memory sees each spin once per step.  Every update goes through the
// storage codec, in the operations and order of the per-half-sweep kernels, and the
// energies are summed over the same 32 half-sites a warp, then as those kernels' blocks
// of eight warps and their energy sums do, so the results are theirs bit for bit.
//
// What bounds it: on small contexts the latency of a half-sweep (about 0.7 us) where
// a launch took 2.5 us; with many samples the issue rate.
#include "hsg_kernels.cuh"

namespace hsg {

namespace {

// One pair of systems of a site: as stored (PLANES words or word pairs), and its
// three components as shared memory holds them (raw 16-bit pairs, or binary32).
template <int F> struct PairFmt { using Raw = uint2; using E = float2; static constexpr bool RAW = false; };
template <> struct PairFmt<FMT_F16> { using Raw = uint32_t; using E = uint32_t; static constexpr bool RAW = true; };
template <> struct PairFmt<FMT_BF16> { using Raw = uint32_t; using E = uint32_t; static constexpr bool RAW = true; };

template <int F>
__device__ __forceinline__ float2 elem_f2(typename PairFmt<F>::E v) {
  if constexpr (F == FMT_F16) return h2f(v);
  else if constexpr (F == FMT_BF16) return b2f(v);
  else return v;
}
// the codec (hsg_device.cuh) on one pair: c[plane] <-> e[component]
template <int F>
__device__ __forceinline__ void pair_elems(const typename PairFmt<F>::Raw* c, typename PairFmt<F>::E* e) {
  if constexpr (PairFmt<F>::RAW) {
    e[0] = c[0]; e[1] = c[1]; e[2] = c[2];
  } else if constexpr (F == FMT_F32) {
#pragma unroll
    for (int k = 0; k < 3; ++k) e[k] = u2f2(c[k].x, c[k].y);
  } else if constexpr (F == FMT_YX4) {
    yx4_decode(__uint_as_float(c[0].x), __uint_as_float(c[1].x), e[0].x, e[1].x, e[2].x);
    yx4_decode(__uint_as_float(c[0].y), __uint_as_float(c[1].y), e[0].y, e[1].y, e[2].y);
  } else if constexpr (F == FMT_ANG16) {
    ang16_decode(c[0].x, e[0].x, e[1].x, e[2].x);
    ang16_decode(c[0].y, e[0].y, e[1].y, e[2].y);
  } else {
    oct16_decode(c[0].x, e[0].x, e[1].x, e[2].x);
    oct16_decode(c[0].y, e[0].y, e[1].y, e[2].y);
  }
}
template <int F>
__device__ __forceinline__ void pair_encode(float2 x, float2 y, float2 z, typename PairFmt<F>::Raw* c) {
  if constexpr (F == FMT_F16) {
    c[0] = f2h(x); c[1] = f2h(y); c[2] = f2h(z);
  } else if constexpr (F == FMT_BF16) {
    c[0] = f2b(x); c[1] = f2b(y); c[2] = f2b(z);
  } else if constexpr (F == FMT_F32) {
    c[0] = make_uint2(__float_as_uint(x.x), __float_as_uint(x.y));
    c[1] = make_uint2(__float_as_uint(y.x), __float_as_uint(y.y));
    c[2] = make_uint2(__float_as_uint(z.x), __float_as_uint(z.y));
  } else if constexpr (F == FMT_YX4) {
    float a0, b0, a1, b1;
    yx4_encode(x.x, y.x, z.x, a0, b0);
    yx4_encode(x.y, y.y, z.y, a1, b1);
    c[0] = make_uint2(__float_as_uint(a0), __float_as_uint(a1));
    c[1] = make_uint2(__float_as_uint(b0), __float_as_uint(b1));
  } else if constexpr (F == FMT_ANG16) {
    c[0] = make_uint2(ang16_encode(x.x, y.x, z.x), ang16_encode(x.y, y.y, z.y));
  } else {
    c[0] = make_uint2(oct16_encode(x.x, y.x, z.x), oct16_encode(x.y, y.y, z.y));
  }
}

}  // namespace

// MAXT: threads a block may have (512 leaves 128 registers a thread, 896 leaves 72).
template <int F, bool J16, bool FAST, int MAXT>
__global__ void __launch_bounds__(MAXT) k_resident(const ResidentParams p) {
  using E = typename PairFmt<F>::E;
  using Raw = typename PairFmt<F>::Raw;
  constexpr int PL = FmtInfo<F>::PLANES, CH = FmtInfo<F>::CHUNK;
  constexpr bool MIXED = (F == FMT_F16) && J16;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float red[2][MAXT / 32][2];        // [parity][warp][system]
  chain_trigger();
  const int s = blockIdx.x / p.n_pairs, pr = blockIdx.x % p.n_pairs;   // sample, pair of systems
  if (!p.active[s]) {            // a frozen sample
    chain_wait();
    return;
  }
  const SampleDev& sd = p.samples[s];
  const int L = sd.L, Lh = sd.Lh, P = L * Lh;    // half-sites of a row, of a plane
  const int HN = sd.N >> 1;
  // HSG_CHECK builds: a thread and shared memory for every half-site, the pair within
  // the sample (else the block leaves the pair as it is)
  if (HSG_OUT_OF_BOUNDS(HN <= (int)blockDim.x && HN <= p.max_half_sites && 2 * pr + 2 <= p.Wp, p.bounds_err)) {
    chain_wait();
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bool live = tid < HN;
  const int h = live ? tid : HN - 1;             // (idle threads repeat the last site, unstored)
  E* sp = reinterpret_cast<E*>(smem);            // [parity][component][HN]
  unsigned char* mine = p.spins + sd.spin_off + ((long long)(pr >> 1) * sd.N + h) * CH + (pr & 1) * (CH / 2);
  const long long ps = sd.plane_stride, odd = (long long)HN * CH;      // to the next plane, to the odd site

  // the half-sites of the neighbours: +x and -x per parity; +y, -y, +z, -z alike for both
  const uint32_t r = (__umulhi((uint32_t)h, sd.fdLh_m) + h) >> sd.fdLh_s;     // y + L z
  const int hx = h - (int)r * Lh;
  const int z = (int)((__umulhi(r, sd.fdL_m) + r) >> sd.fdL_s), y = (int)r - z * L;
  const int nyp = y + 1 == L ? h + Lh - P : h + Lh, nym = y == 0 ? h - Lh + P : h - Lh;
  const int nzp = z + 1 == L ? h + P - HN : h + P, nzm = z == 0 ? h - P + HN : h - P;
  int nxp[2], nxm[2], nyz[4] = {nyp, nym, nzp, nzm};
  float j6[2][6], h3[2][3];
  uint32_t jh[2][6];
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    const bool f = (par + y + z) & 1;            // x = 2 hx + f
    nxp[par] = f ? (hx + 1 == Lh ? h + 1 - Lh : h + 1) : h;
    nxm[par] = f ? h : (hx == 0 ? h + Lh - 1 : h - 1);
    // HSG_CHECK builds: every neighbour a half-site of the lattice (else the thread
    // reads half-site 0 and stores nothing)
    bool bad = false;
    for (int* n : {&nxp[par], &nxm[par], &nyz[0], &nyz[1], &nyz[2], &nyz[3]})
      if (HSG_OUT_OF_BOUNDS(*n >= 0 && *n < HN, p.bounds_err)) bad = true, *n = 0;
    if (bad) live = false;
    load_record<J16>(p.rec, sd.rec_off + par * HN + h, j6[par], h3[par]);
    if (MIXED) load_record_j16(p.rec, sd.rec_off + par * HN + h, jh[par]);
  }
  const uint32_t pair_id = ((uint32_t)sd.sys_base >> 1) + pr;           // gsys >> 1

  chain_wait();
  E own[2][3];
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    Raw c[PL];
#pragma unroll
    for (int k = 0; k < PL; ++k) c[k] = *reinterpret_cast<const Raw*>(mine + par * odd + k * ps);
    pair_elems<F>(c, own[par]);
    if (live)
#pragma unroll
      for (int k = 0; k < 3; ++k) sp[(par * 3 + k) * HN + h] = own[par][k];
  }
  const float* bp = p.beta + (long long)s * p.Wp + pr * 2;
  const float2 bt = make_float2(bp[0], bp[1]);
  const uint32_t sweep0 = (uint32_t)p.counters[2 * s];
  __syncthreads();

  const int nsw = p.n_hb + p.n_or;
  for (int k = 0; k < nsw; ++k) {
    const bool hb = k < p.n_hb, last = k == nsw - 1;
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const E* O = sp + (1 - par) * 3 * HN;
      const int nb[6] = {nxp[par], nxm[par], nyz[0], nyz[1], nyz[2], nyz[3]};
      E nv[6][3];
#pragma unroll
      for (int n = 0; n < 6; ++n)
#pragma unroll
        for (int c = 0; c < 3; ++c) nv[n][c] = O[c * HN + nb[n]];
      // local field h = sum_n J_n s_n + H, in the order +x, -x, +y, -y, +z, -z
      float2 fx = make_float2(0.0f, 0.0f), fy = fx, fz = fx;
#pragma unroll
      for (int n = 0; n < 6; ++n) {
        if constexpr (MIXED) {
          // FP16 spins and couplings: fused f16 x f16 + f32 (exact products)
          fma_f16_pair(fx, nv[n][0], jh[par][n]);
          fma_f16_pair(fy, nv[n][1], jh[par][n]);
          fma_f16_pair(fz, nv[n][2], jh[par][n]);
        } else {
          const float2 jj = f2(j6[par][n]);
          const float2 vx = elem_f2<F>(nv[n][0]), vy = elem_f2<F>(nv[n][1]), vz = elem_f2<F>(nv[n][2]);
          fx = n == 0 ? mul2(jj, vx) : fma2(jj, vx, fx);
          fy = n == 0 ? mul2(jj, vy) : fma2(jj, vy, fy);
          fz = n == 0 ? mul2(jj, vz) : fma2(jj, vz, fz);
        }
      }
      fx = add2(fx, f2(h3[par][0]));
      fy = add2(fy, f2(h3[par][1]));
      fz = add2(fz, f2(h3[par][2]));
      float2 sx = elem_f2<F>(own[par][0]), sy = elem_f2<F>(own[par][1]), sz = elem_f2<F>(own[par][2]);
      if (hb) {
        const uint32_t site = 2u * (uint32_t)h + ((par + y + z) & 1);
        const uint4 rn = philox4x32_10_rk(make_uint4(site, pair_id, sweep0 + (uint32_t)k, TAG_HB), p.rk);
        hb_move2<FAST>(sx, sy, sz, fx, fy, fz, bt, make_float2(u01(rn.x), u01(rn.z)),
                       make_float2(u01(rn.y), u01(rn.w)));
      } else {
        or_move2(sx, sy, sz, fx, fy, fz);
      }
      Raw c[PL];
      pair_encode<F>(sx, sy, sz, c);
      pair_elems<F>(c, own[par]);
      if (live) {
#pragma unroll
        for (int q = 0; q < 3; ++q) sp[(par * 3 + q) * HN + h] = own[par][q];
        if (last)
#pragma unroll
          for (int q = 0; q < PL; ++q) *reinterpret_cast<Raw*>(mine + par * odd + q * ps) = c[q];
      }
      if (last && !hb) {
        // energy of the new state from the stored values: every bond joins one
        // odd and one even site, E = - sum_odd s_i.h_i - sum_even H_j.s_j
        const float2 tx = elem_f2<F>(own[par][0]), ty = elem_f2<F>(own[par][1]), tz = elem_f2<F>(own[par][2]);
        const float2 d = par == 1 ? dot3_2(tx, ty, tz, fx, fy, fz)
                                  : dot3_2(tx, ty, tz, f2(h3[par][0]), f2(h3[par][1]), f2(h3[par][2]));
        const float e0 = warp_sum(live ? -d.x : 0.0f), e1 = warp_sum(live ? -d.y : 0.0f);
        if (lane == 0) {
          red[par][warp][0] = e0;
          red[par][warp][1] = e1;
        }
      }
      __syncthreads();
    }
  }
  if (p.n_or == 0) return;       // (the energies come from the separate kernel)
  if (warp == 0) {
    // rows of SWEEP_BS half-sites (at most 4: one split, and a row lane for each): their
    // even sites' partial and their odd sites', lane = 4 row + 2 parity + system
    const int nw = blockDim.x >> 5, w0 = (lane >> 2) * (SWEEP_BS / 32), w1 = min(nw, w0 + SWEEP_BS / 32);
    double part = 0.0, t = 0.0;
    for (int w = w0; w < w1; ++w) part += (double)red[(lane >> 1) & 1][w][lane & 1];
    part += __shfl_xor_sync(0xffffffffu, part, 2);
    for (int row = 0; row * (SWEEP_BS / 32) < nw; ++row) t += __shfl_sync(0xffffffffu, part, 4 * row + (lane & 1));
    if (lane < 2) p.E[(long long)s * p.Wp + pr * 2 + lane] = t;
  }
}

template <int F, bool J16, bool FAST>
static cudaError_t resident_launch(const ResidentParams& p, cudaStream_t st) {
  const int threads = (p.max_half_sites + 31) / 32 * 32, blocks = p.n_samples * p.n_pairs;
  const size_t smem = 6 * sizeof(typename PairFmt<F>::E) * (size_t)p.max_half_sites;   // <= 48 kB
  if (threads <= 512) return launch_chained(k_resident<F, J16, FAST, 512>, blocks, threads, smem, st, p);
  return launch_chained(k_resident<F, J16, FAST, RES_MAX_HALF_SITES>, blocks, threads, smem, st, p);
}

template <int F>
static cudaError_t resident_fmt(bool j16, bool fast, const ResidentParams& p, cudaStream_t st) {
  if (j16) return fast ? resident_launch<F, true, true>(p, st) : resident_launch<F, true, false>(p, st);
  return fast ? resident_launch<F, false, true>(p, st) : resident_launch<F, false, false>(p, st);
}

cudaError_t launch_resident(int fmt, bool j16, bool fast, const ResidentParams& p, cudaStream_t st) {
  switch (fmt) {
    case FMT_F32: return resident_fmt<FMT_F32>(j16, fast, p, st);
    case FMT_F16: return resident_fmt<FMT_F16>(j16, fast, p, st);
    case FMT_BF16: return resident_fmt<FMT_BF16>(j16, fast, p, st);
    case FMT_ANG16: return resident_fmt<FMT_ANG16>(j16, fast, p, st);
    case FMT_OCT16: return resident_fmt<FMT_OCT16>(j16, fast, p, st);
    case FMT_YX4: return resident_fmt<FMT_YX4>(j16, fast, p, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hsg

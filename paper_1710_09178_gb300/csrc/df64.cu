// df64.cu - true residuals r = b - (A + sigma) x in double-FP32 arithmetic.
//
// The mixed-precision modes need residuals accurate to well below the 1e-10 tolerance: the
// reliable updates of the shifted CG (r = b - (A + sigma_0) x_0) and the true-residual checks
// that certify every shift and give the refinement its right-hand sides (Section 3's FP64
// treatment of these steps).  On GB300 the FP64 units run at about 1/57 of the FP32 rate: an FP64
// Dslash takes ~75 us on 32^3 x 8 with FP64 multiply-adds and 35 us with integer ones (fix64.cuh).  Here the
// same residual is computed with FP32 instructions only, in 22 us:
//   - every FP64 number u is held as a pair (hi, lo) = (fl32(u), fl32(u - hi)) (about 48 bits);
//   - of a product (ah + al)(bh + bl), p = fl32(ah bh) enters the running sum s through Knuth's TwoSum; what
//     s does not take (TwoSum's error, the product's rounding and the cross terms ah bl + al bh; al bl,
//     ~2^-48 relative, is dropped) goes to a compensation c, so s + c carries the sum to ~2^-48
//     relative to the sum of the magnitudes of its terms (df_mac: 10 operations).
// The links are the FP32 copy (hi, 1/2 eta bc folded in) plus a copy of the FP32 rounding
// errors (lo); vectors are split from FP64 once per residual.  The result is rounded to FP32
// (the reliable update and the refinement both continue in FP32) and |r|^2 is summed in FP64.
//
// The same arithmetic also carries a whole shifted-CG solve (precision mode LQCD_DF64): Krylov
// vectors, shift vectors, the residual window and the solutions x_k are (hi, lo) pairs, stored as
// [3][Vh] float2 hi followed by [3][Vh] float2 lo (48 bytes per site, as FP64).  The iterated and
// true residuals then agree to ~2^-48, so the solve needs neither reliable updates nor per-shift
// refinement, at FP32-unit cost.
#include "common.cuh"
#include "internal.h"
#include "solver_dev.cuh"

namespace lqcd {

constexpr int kDfThreads = 128;  // of the Dslash; 4 blocks per SM (128 registers)

// Sum over the block of per-thread double-FP32 values (s, c): TwoSum shuffles within each warp,
// then the warps' FP64 values in a fixed order.  Result valid in thread 0 (which publishes it).
__device__ __forceinline__ double block_sum_df(float s, float c) {
  __shared__ double red_df[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
    df_add(s, c, s2, c2);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) red_df[warp] = (double)s + (double)c;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < nw; ++w) t += red_df[w];
  __syncthreads();
  return t;
}

__device__ __forceinline__ float2 split64(double a) { return split_hi_lo(a); }

// x (FP64) -> (hi, lo) FP32 pairs
__global__ void __launch_bounds__(256) split_df_kernel(int n3, const double2* __restrict__ x, float2* __restrict__ hi,
                                                        float2* __restrict__ lo, const int* done) {
  pdl_wait();
  pdl_trigger();
  if (done && *done) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  const double2 v = x[i];
  const float hx = __double2float_rn(v.x), hy = __double2float_rn(v.y);
  hi[i] = make_float2(hx, hy);
  lo[i] = make_float2(__double2float_rn(v.x - (double)hx), __double2float_rn(v.y - (double)hy));
}

// One hop of the site's double-FP32 half Dslash onto its accumulators (s, c) of the real and
// imaginary parts of each colour: fwd: out_a += U_ab v_b, else out_a -= conj(U_ba) v_b, with
// U = Uh + Ul and v = vh + vl.
__device__ __forceinline__ void df_hop(float (&sr)[3], float (&cr)[3], float (&si)[3], float (&ci)[3],
                                       const Mat3<float>& Uh, const Mat3<float>& Ul, const Vec3<float>& vh3,
                                       const Vec3<float>& vl3, bool fwd) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float2 xv = make_float2(vh3.c[b].re, vh3.c[b].im), xl = make_float2(vl3.c[b].re, vl3.c[b].im);
      if (fwd) {
        const Cplx<float> uh = Uh.e[a][b], ul = Ul.e[a][b];
        df_mac(sr[a], cr[a], uh.re, ul.re, xv.x, xl.x);
        df_mac(sr[a], cr[a], -uh.im, -ul.im, xv.y, xl.y);
        df_mac(si[a], ci[a], uh.re, ul.re, xv.y, xl.y);
        df_mac(si[a], ci[a], uh.im, ul.im, xv.x, xl.x);
      } else {
        const Cplx<float> uh = Uh.e[b][a], ul = Ul.e[b][a];
        df_mac(sr[a], cr[a], -uh.re, -ul.re, xv.x, xl.x);
        df_mac(sr[a], cr[a], -uh.im, -ul.im, xv.y, xl.y);
        df_mac(si[a], ci[a], -uh.re, -ul.re, xv.y, xl.y);
        df_mac(si[a], ci[a], uh.im, ul.im, xv.x, xl.x);
      }
    }
  }
}

__device__ __forceinline__ float2 df_a(const DfArgs& k) {
  return k.a_split ? make_float2(k.a_hi, k.a_lo) : (k.a_devdf ? *k.a_devdf : split64(k.a_dev ? *k.a_dev : k.a));
}

// (yh + yl) + a (xh + xl) as a normalised pair
__device__ __forceinline__ float2 df_axpy(float yh, float yl, float2 a, float xh, float xl) {
  float s = yh, c = yl;
  df_mac(s, c, a.x, a.y, xh, xl);
  return df_norm(s, c);
}

// What the epilogues read at the output site beside the hops' sum, for one colour.
struct DfOwn {
  float2 xh, xl, bh, bl;
};
template <int EPI>
__device__ __forceinline__ DfOwn df_own(const DfArgs& k, size_t o) {
  DfOwn w;
  if constexpr (EPI != 0) {
    w.xh = k.x_hi[o];
    w.xl = k.x_lo[o];
  }
  if constexpr (EPI == 2) {
    w.bh = k.b_hi[o];
    w.bl = k.b_lo[o];
  }
  return w;
}

// One colour of the output at offset o, d = (sr + cr, si + ci) its D in:  EPI 0: out = d;  EPI 1: out = a x - d,
// (ds, dc) += Re<x, out>;  EPI 2: r = fl32(b - (a x - d)) (stored unless r_out is null), ds += |r|^2.
template <int EPI>
__device__ __forceinline__ void df_finish(const DfArgs& k, size_t o, float2 asp, const DfOwn& w, float sr, float cr,
                                          float si, float ci, float& ds, float& dc) {
  if constexpr (EPI == 0) {
    const float2 re = df_norm(sr, cr), im = df_norm(si, ci);
    k.out_hi[o] = make_float2(re.x, im.x);
    k.out_lo[o] = make_float2(re.y, im.y);
  } else if constexpr (EPI == 1) {
    float rs = 0.f, rc = 0.f, is = 0.f, ic = 0.f;
    df_mac(rs, rc, asp.x, asp.y, w.xh.x, w.xl.x);
    df_mac(is, ic, asp.x, asp.y, w.xh.y, w.xl.y);
    df_add(rs, rc, -sr, -cr);
    df_add(is, ic, -si, -ci);
    const float2 re = df_norm(rs, rc), im = df_norm(is, ic);
    k.out_hi[o] = make_float2(re.x, im.x);
    k.out_lo[o] = make_float2(re.y, im.y);
    df_mac(ds, dc, w.xh.x, w.xl.x, re.x, re.y);
    df_mac(ds, dc, w.xh.y, w.xl.y, im.x, im.y);
  } else {
    float rs = w.bh.x, rc = w.bl.x, is = w.bh.y, ic = w.bl.y;
    df_mac(rs, rc, -asp.x, -asp.y, w.xh.x, w.xl.x);
    df_mac(is, ic, -asp.x, -asp.y, w.xh.y, w.xl.y);
    df_add(rs, rc, sr, cr);
    df_add(is, ic, si, ci);
    const float rr = __fadd_rn(rs, rc), ri = __fadd_rn(is, ic);
    if (k.r_out) k.r_out[o] = make_float2(rr, ri);
    ds += rr * rr + ri * ri;
  }
}

// the end of a site's sum: 0 plain, 1 the A-apply (inside the solve, without a ticket, the sum stays as
// per-block (hi, lo) partials for the r update), 2 the residual
template <int EPI>
__device__ __forceinline__ void df_reduce(const DfArgs& k, float ds, float dc) {
  if constexpr (EPI == 0) return;
  double bs;
  if constexpr (EPI == 1) {
    if (!k.ticket) {
      const float2 b2 = block_sum_df_df(ds, dc);
      if (threadIdx.x == 0) reinterpret_cast<float2*>(k.partials)[blockIdx.x] = b2;
      return;
    }
    bs = block_sum_df(ds, dc);
  } else {
    bs = block_sum_mixed(ds);
  }
  if (publish_partial(k.partials, k.ticket, bs)) {
    const double tot = gather_partials(k.partials, k.ticket);
    if (threadIdx.x == 0 && k.dot_out) *k.dot_out = tot;
  }
}

// The half Dslash of system blockIdx.y with its epilogue.  Every direction's pair of hops (forward, then
// backward) is one double-FP32 sum, and the four are added in order, whatever TPS, so the bits do not
// depend on how the directions are spread over threads.
// The block holds NS = blockDim.x / TPS sites; thread t takes directions t / NS ND .. of site t % NS, ND = 4 / TPS.
// With TPS = 1 the thread adds each direction to its sum as it goes; kept in 24 KB of shared memory per block until the end,
// the sums take that from the L1 that the neighbours' vectors hit (32^3x8: 23.8 instead of 22.1 us).  With more
// threads the four sums meet in shared memory, and thread sub finishes colours sub, sub + TPS, ..
// UPD: the p update folded in (small lattices, one system): EPI 0 takes r + beta in at every neighbour, beta summed from the
// r update's partials as the p update kernel does, and runs the beta step in the last block; EPI 1 takes r + beta x at its
// own site and stores it in x.  The same operations, the same bits.
template <int EPI, int TPS, bool UPD>
__global__ void __launch_bounds__(kDfThreads, UPD ? 2 : 4) df_dslash_kernel(Geom g, const __grid_constant__ PerSys<DfArgs> pk) {
  constexpr int NS = kDfThreads / TPS, ND = 4 / TPS;
  __shared__ float4 part[TPS == 1 ? 1 : 4][3][NS];
  const DfArgs& k = pk.s[blockIdx.y];
  const int vh = g.vh;
  const int sub = threadIdx.x / NS, ls = threadIdx.x % NS;
  const int i = blockIdx.x * NS + ls;
  const bool scalar_block = UPD && EPI == 0 && blockIdx.x == gridDim.x - 1;
  const bool valid = !scalar_block && i < vh;
  const int p = k.out_parity;
  const uint64_t pol_hi = policy_evict_last();   // the solver's FP32 links: keep them in L2
  const uint64_t pol_lo = policy_evict_first();  // rounding errors, read only by the checks
  // With several threads per site the launch is short of work, and its latency counts: the first link (which no
  // kernel of a solve writes) is fetched before the wait and the epilogue's vectors beside the hops'.
  Mat3<float> Uh, Ul;
  Site s;
  if (valid) {
    s = site_of(g, p, i);
    if (TPS > 1) {
      Uh = load_link32(k.links_hi, p, sub * ND, i, vh, pol_hi);
      Ul = load_link32(k.links_lo, p, sub * ND, i, vh, pol_lo);
    }
  }
  pdl_wait();
  pdl_trigger();
  float2 be = make_float2(0.f, 0.f);
  Vec3<float> rh[2], rl[2], ph[2], pl[2];  // UPD: r and p at the first direction's neighbours
  auto load_rp = [&](int q, int j) {
    rh[q] = load_vec(k.upd_r, j, vh);
    rl[q] = load_vec(k.upd_r + 3 * (size_t)vh, j, vh);
    ph[q] = load_vec(k.in_hi, j, vh);
    pl[q] = load_vec(k.in_lo, j, vh);
  };
  if constexpr (UPD && EPI == 0) {
    SolverDev* sd = k.sd;
    // the scalar block may set done meanwhile: partials_ratio settles the block on one reading
    const bool skip = (*reinterpret_cast<const volatile int*>(&sd->done) | (k.halt ? *k.halt : 0)) != 0;
    const float2 rr_b_df = sd->rr_b_df;
    if (valid) {
      load_rp(0, neighbour_half(g, neighbour_fwd(g, s, sub * ND)));
      load_rp(1, neighbour_half(g, neighbour_bwd(g, s, sub * ND)));
    }
    const PartialsRatio pb = partials_ratio_df<true>(k.rr_partials, k.n_rr, rr_b_df, skip, scalar_block);
    if (pb.stop) return;  // the same in every thread of the block
    if (scalar_block) {
      solver_beta_step(sd, pb);
      return;
    }
    be = pb.ratio_df;
  } else {
    if ((k.done && *k.done) || (k.halt && *k.halt)) return;  // uniform
    if constexpr (UPD) be = k.sd->beta_df;
  }

  constexpr int NC = (3 + TPS - 1) / TPS;  // colours finished by thread sub: sub, sub + TPS, ..
  DfOwn own[NC];
  float2 asp = make_float2(0.f, 0.f);
  auto load_own = [&]() {
    if (EPI != 0) asp = df_a(k);
#pragma unroll
    for (int q = 0; q < NC; ++q)
      if (valid && sub + q * TPS < 3) {
        const size_t o = (size_t)(sub + q * TPS) * vh + i;
        own[q] = df_own<EPI>(k, o);
        if constexpr (UPD && EPI == 1) {
          const float2 re = df_axpy(k.upd_r[o].x, k.upd_r[o + 3 * (size_t)vh].x, be, own[q].xh.x, own[q].xl.x),
                       im = df_axpy(k.upd_r[o].y, k.upd_r[o + 3 * (size_t)vh].y, be, own[q].xh.y, own[q].xl.y);
          own[q].xh = make_float2(re.x, im.x);
          own[q].xl = make_float2(re.y, im.y);
          const_cast<float2*>(k.x_hi)[o] = own[q].xh;
          const_cast<float2*>(k.x_lo)[o] = own[q].xl;
        }
      }
  };
  if (TPS > 1) load_own();
  float4 sum[3];  // TPS = 1: of the directions so far
  if (valid) {
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      float sr[3] = {0.f, 0.f, 0.f}, cr[3] = {0.f, 0.f, 0.f}, si[3] = {0.f, 0.f, 0.f}, ci[3] = {0.f, 0.f, 0.f};
      const int mu = sub * ND + d;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool fwd = h == 0;
        const int j = neighbour_half(g, fwd ? neighbour_fwd(g, s, mu) : neighbour_bwd(g, s, mu));
        const int lp = fwd ? p : 1 - p, li = fwd ? i : j;
        if (TPS == 1 || d > 0 || h > 0) {
          Uh = load_link32(k.links_hi, lp, mu, li, vh, pol_hi);
          Ul = load_link32(k.links_lo, lp, mu, li, vh, pol_lo);
        }
        Vec3<float> vh3, vl3;
        if constexpr (UPD && EPI == 0) {
          if (d > 0) load_rp(h, j);
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float2 re = df_axpy(rh[h].c[c].re, rl[h].c[c].re, be, ph[h].c[c].re, pl[h].c[c].re),
                         im = df_axpy(rh[h].c[c].im, rl[h].c[c].im, be, ph[h].c[c].im, pl[h].c[c].im);
            vh3.c[c] = cmake(re.x, im.x);
            vl3.c[c] = cmake(re.y, im.y);
          }
        } else {
          vh3 = ldg_vec(k.in_hi, j, vh);
          vl3 = ldg_vec(k.in_lo, j, vh);
        }
        df_hop(sr, cr, si, ci, Uh, Ul, vh3, vl3, fwd);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (TPS > 1) {
          part[mu][c][ls] = make_float4(sr[c], cr[c], si[c], ci[c]);
        } else if (d == 0) {
          sum[c] = make_float4(sr[c], cr[c], si[c], ci[c]);
        } else {
          df_add(sum[c].x, sum[c].y, sr[c], cr[c]);
          df_add(sum[c].z, sum[c].w, si[c], ci[c]);
        }
      }
    }
  }
  if (TPS > 1) __syncthreads();
  else load_own();
  float ds = 0.f, dc = 0.f;
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const int c = sub + q * TPS;
    if (!valid || c >= 3) continue;
    float4 t = TPS == 1 ? sum[q] : part[0][c][ls];
    if constexpr (TPS > 1) {
#pragma unroll
      for (int mu = 1; mu < 4; ++mu) {
        const float4 u = part[mu][c][ls];
        df_add(t.x, t.y, u.x, u.y);
        df_add(t.z, t.w, u.z, u.w);
      }
    }
    df_finish<EPI>(k, (size_t)c * vh + i, asp, own[q], t.x, t.y, t.z, t.w, ds, dc);
  }
  df_reduce<EPI>(k, ds, dc);
}

cudaError_t launch_split_df(const Geom& g, const double2* x, float2* hi, float2* lo, const int* done, cudaStream_t st,
                            bool pdl) {
  const int n3 = 3 * g.vh;
  return launch_k(pdl, split_df_kernel, dim3((n3 + 255) / 256), dim3(256), st, n3, x, hi, lo, done);
}

// Threads per site: the most that keep the launch within two blocks per SM (304), so that a small lattice's chain
// of eight hops is shortened while the SMs have room.  Half Dslash per graph launch, in us, with 1 / 2 / 4 threads
// per site (12-operation df_mac): 8^4 6.3 / 3.2 / 2.4, 16^3x8 7.3 / 4.3 / 4.5, 24^3x6 9.8 / 9.5 / 11.2, 32^3x8
// 24.2 / 25.7 / 30.6, 48^3x12 129 / 132 / 159 (A-applies at 24^3x6 23.5 / 25.9 / 32.4): more threads repeat the
// site's index arithmetic.  One thread per colour instead gives 4.7, 5.7 and 10.8 us at the first three.
// Against one thread per site and one sum over all directions: 8^4 6.4 -> 2.4 us, 16^3x8 7.4 -> 4.5, 24^3x6 9.5 -> 9.3,
// 32^3x8 23.0 -> 22.1, 48^3x12 125 -> 124, error against quad precision 1.6e-14 -> 7.0e-15 (Gaussian vectors).
static int df_tps(const Geom& g) {
  constexpr int kBlocks = 2 * kSMs;
  return g.vh <= kBlocks * kDfThreads / 4 ? 4 : (g.vh <= kBlocks * kDfThreads / 2 ? 2 : 1);
}
int df_dslash_grid_blocks(const Geom& g) {
  const int ns = kDfThreads / df_tps(g);
  return (g.vh + ns - 1) / ns;
}

template <int TPS>
static cudaError_t launch_df_tps(const Geom& g, const PerSys<DfArgs>& a, int S, int epi, cudaStream_t st, bool pdl) {
  const dim3 grid((unsigned)df_dslash_grid_blocks(g), (unsigned)S), block(kDfThreads);
  if constexpr (TPS > 1) {
    if (a.s[0].upd_r) {
      if (S != 1 || epi == 2) return cudaErrorInvalidValue;
      if (epi == 1) return launch_k(pdl, df_dslash_kernel<1, TPS, true>, grid, block, st, g, a);
      return launch_k(pdl, df_dslash_kernel<0, TPS, true>, dim3(grid.x + 1), block, st, g, a);
    }
  }
  if (epi == 2) return launch_k(pdl, df_dslash_kernel<2, TPS, false>, grid, block, st, g, a);
  if (epi == 1) return launch_k(pdl, df_dslash_kernel<1, TPS, false>, grid, block, st, g, a);
  return launch_k(pdl, df_dslash_kernel<0, TPS, false>, grid, block, st, g, a);
}

bool fold_df_p_update(const Geom& g) { return df_tps(g) > 1; }

cudaError_t launch_df_dslash_multi(const Geom& g, const PerSys<DfArgs>& a, int S, int epi, cudaStream_t st, bool pdl) {
  switch (df_tps(g)) {
    case 4: return launch_df_tps<4>(g, a, S, epi, st, pdl);
    case 2: return launch_df_tps<2>(g, a, S, epi, st, pdl);
    default: return launch_df_tps<1>(g, a, S, epi, st, pdl);
  }
}

cudaError_t launch_df_dslash(const Geom& g, const DfArgs& a, int epi, cudaStream_t st, bool pdl) {
  PerSys<DfArgs> p;
  p.s[0] = a;
  return launch_df_dslash_multi(g, p, 1, epi, st, pdl);
}

// ---------------------------------------------------------------------------------------------
// The double-FP32 shifted CG (mode LQCD_DF64): the same steps as the FP32/FP64 kernels of the
// solver, on (hi, lo) vectors.
// ---------------------------------------------------------------------------------------------
// r = p = b as (hi, lo), |b|^2 in FP64, then the scalar state of a fresh solve
__global__ void __launch_bounds__(256) df_init_kernel(Geom g, const double2* __restrict__ b64, float2* r, float2* p,
                                                      SolverDev* sd, InitParams ip, double* partials,
                                                      unsigned* ticket) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int vh = g.vh;
  double loc = 0.0;
  if (i < vh) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t o = (size_t)c * vh + i;
      const double2 b = b64[o];
      const float2 re = split64(b.x), im = split64(b.y);
      const float2 h = make_float2(re.x, im.x), l = make_float2(re.y, im.y);
      r[o] = h;
      r[o + 3 * (size_t)vh] = l;
      p[o] = h;
      p[o + 3 * (size_t)vh] = l;
      loc += b.x * b.x + b.y * b.y;
    }
  }
  const double bs = block_sum(loc);
  if (publish_partial(partials, ticket, bs)) init_scalars(sd, ip, gather_partials(partials, ticket));
}

// r -= alpha q; R[m] = r; (hi, lo) partials of |r|^2.  alpha comes from the A-apply's partials
// (every block, the same bits); one extra block runs the alpha step.
__global__ void __launch_bounds__(256, 4) df_r_update_kernel(Geom g, const __grid_constant__ PerSys<DfUpdArgs> args) {
  const DfUpdArgs& a = args.s[blockIdx.y];  // system blockIdx.y
  pdl_wait();
  pdl_trigger();
  SolverDev* sd = a.sd;
  // the scalar block may set done meanwhile: partials_ratio settles the block on one reading
  const int dn = *reinterpret_cast<const volatile int*>(&sd->done), ht = a.halt ? *a.halt : 0;  // both in flight
  const bool skip = (dn | ht) != 0;
  const int m = sd->m;
  const float2 rr_df = sd->rr_df;
  const int vh = g.vh;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int nb = (vh + blockDim.x - 1) / blockDim.x;  // then the scalar block, then one per shift for its recurrence
  const bool scalar_block = (int)blockIdx.x == nb;
  if ((int)blockIdx.x > nb) {
    if (!__syncthreads_or(skip)) window_scalars_shift<false>(sd, blockIdx.x - nb - 1);
    return;
  }
  const bool site = !scalar_block && i < vh;
  float2 rv[4][3];  // r hi, r lo, q hi, q lo: issued before the partials are summed
  if (site) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t o = (size_t)c * vh + i, ol = o + 3 * (size_t)vh;
      rv[0][c] = a.r[o];
      rv[1][c] = a.r[ol];
      rv[2][c] = a.q[o];
      rv[3][c] = a.q[ol];
    }
  }
  const PartialsRatio pa = partials_ratio_df<false>(a.pq_partials, a.n_pq, rr_df, skip, scalar_block);
  if (pa.stop) return;  // the same in every thread of the block
  const bool mine = site && m < kWindow;
  if (scalar_block) {
    solver_alpha_step(sd, pa);
    return;
  }
  const float2 al = pa.ratio_df;
  float ls = 0.f, lc = 0.f;
  if (mine) {
    float2* slot = reinterpret_cast<float2*>(static_cast<char*>(a.ring) + m * a.slot_bytes);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t o = (size_t)c * vh + i, ol = o + 3 * (size_t)vh;
      const float2 rh = rv[0][c], rl = rv[1][c], qh = rv[2][c], ql = rv[3][c];
      float rs = rh.x, rc = rl.x, is = rh.y, ic = rl.y;
      df_mac(rs, rc, -al.x, -al.y, qh.x, ql.x);
      df_mac(is, ic, -al.x, -al.y, qh.y, ql.y);
      const float2 re = df_norm(rs, rc), im = df_norm(is, ic);
      const float2 h = make_float2(re.x, im.x), l = make_float2(re.y, im.y);
      a.r[o] = h;
      a.r[ol] = l;
      slot[o] = h;
      slot[ol] = l;
      df_mac(ls, lc, h.x, l.x, h.x, l.x);
      df_mac(ls, lc, h.y, l.y, h.y, l.y);
    }
  }
  const float2 bs = block_sum_df_df(ls, lc);
  if (threadIdx.x == 0) reinterpret_cast<float2*>(a.rr_partials)[blockIdx.x] = bs;
}

// p = r + beta p, one site per thread; beta from the r update's partials; one extra block runs
// the beta step.
__global__ void __launch_bounds__(256, 4) df_p_update_kernel(Geom g, const __grid_constant__ PerSys<DfUpdArgs> args) {
  const DfUpdArgs& a = args.s[blockIdx.y];  // system blockIdx.y
  pdl_wait();
  pdl_trigger();
  SolverDev* sd = a.sd;
  const int dn = *reinterpret_cast<const volatile int*>(&sd->done), ht = a.halt ? *a.halt : 0;  // both in flight
  const bool skip = (dn | ht) != 0;
  const float2 rr_b_df = sd->rr_b_df;
  const int vh = g.vh;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool scalar_block = blockIdx.x == gridDim.x - 1;
  const bool mine = !scalar_block && i < vh;
  float2 rv[4][3];  // r hi, r lo, p hi, p lo: issued before the partials are summed
  if (mine) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t o = (size_t)c * vh + i, ol = o + 3 * (size_t)vh;
      rv[0][c] = a.r[o];
      rv[1][c] = a.r[ol];
      rv[2][c] = a.p[o];
      rv[3][c] = a.p[ol];
    }
  }
  const PartialsRatio pb = partials_ratio_df<true>(a.rr_partials, (int)gridDim.x - 1, rr_b_df, skip, scalar_block);
  if (pb.stop) return;  // the same in every thread of the block
  if (scalar_block) {
    solver_beta_step(sd, pb);
    return;
  }
  if (!mine) return;
  const float2 be = pb.ratio_df;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const size_t o = (size_t)c * vh + i, ol = o + 3 * (size_t)vh;
    const float2 rh = rv[0][c], rl = rv[1][c], ph = rv[2][c], pl = rv[3][c];
    float rs = rh.x, rc = rl.x, is = rh.y, ic = rl.y;
    df_mac(rs, rc, be.x, be.y, ph.x, pl.x);
    df_mac(is, ic, be.x, be.y, ph.y, pl.y);
    const float2 re = df_norm(rs, rc), im = df_norm(is, ic);
    a.p[o] = make_float2(re.x, im.x);
    a.p[ol] = make_float2(re.y, im.y);
  }
}

// The pending window: p_k = P p_k0 + sum_i pi_i R_i;  x_k += X p_k0 + sum_i chi_i R_i, all in double-FP32.  One
// thread per complex component, which keeps the window's residuals (2 x kWindow float2) in registers; the shifts
// are spread over gridDim.z, with the next shift's vectors loaded while one is computed.  Bound by the compensated
// arithmetic (44 multiply-adds of 10 operations per shift and component): 32^3x8 84 -> 66 us a window, 16^3x8 27.5 -> 11.7,
// 4^4 22 -> 5.
__global__ void __launch_bounds__(kFlushThreads) df_flush_kernel(int n3, const __grid_constant__ PerSys<DfFlushArgs> pa) {
  const DfFlushArgs& a = pa.s[blockIdx.y];  // system blockIdx.y
  pdl_wait();
  pdl_trigger();
  SolverDev* sd = a.sd;
  const int m = sd->m;
  if (m == 0) return;
  __shared__ WindowCoefs<float2> w;
  const int first = sd->first;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = o < n3;
  float2 Rh[kWindow], Rl[kWindow];
#pragma unroll
  for (int q = 0; q < kWindow; ++q) {
    const float2* slot = reinterpret_cast<const float2*>(static_cast<const char*>(a.ring) + q * a.slot_bytes);
    Rh[q] = (valid && q < m) ? slot[o] : make_float2(0.f, 0.f);
    Rl[q] = (valid && q < m) ? slot[o + n3] : make_float2(0.f, 0.f);
  }
  w.load(sd->P_df, sd->X_df, sd->pi_df, sd->chi_df, sd->wactive, sd->n, m);
  const uint64_t pol = policy_evict_first();  // x_k is touched once per window: it must not displace the links
  const int cnt = w.count, step = gridDim.z;
  if (valid) {
    float2 ph, pl, xh, xl;
    auto fetch = [&](int j) {
      const int k = w.list[j];
      const float2* pk = first ? a.b_hi : a.pk[k];
      ph = pk[o];
      pl = first ? a.b_lo[o] : pk[o + n3];
      xh = xl = make_float2(0.f, 0.f);
      if (!first) {
        xh = ld_hint(a.xk[k] + o, pol);
        xl = ld_hint(a.xk[k] + o + n3, pol);
      }
    };
    int j = blockIdx.z;
    if (j < cnt) fetch(j);
    for (; j < cnt; j += step) {
      const int k = w.list[j];
      const float2 p0h = ph, p0l = pl, x0h = xh, x0l = xl;
      if (j + step < cnt) fetch(j + step);
      // new p_k and the increment of x_k, real and imaginary parts
      const float2 cP = w.P[k], cX = w.X[k];
      float ps = 0.f, pc = 0.f, qs = 0.f, qc = 0.f, xs = 0.f, xc = 0.f, ys = 0.f, yc = 0.f;
      df_mac(ps, pc, cP.x, cP.y, p0h.x, p0l.x);
      df_mac(qs, qc, cP.x, cP.y, p0h.y, p0l.y);
      df_mac(xs, xc, cX.x, cX.y, p0h.x, p0l.x);
      df_mac(ys, yc, cX.x, cX.y, p0h.y, p0l.y);
#pragma unroll
      for (int q = 0; q < kWindow; ++q) {
        if (q >= m) break;
        const float2 pq = w.pi[k][q], cq = w.chi[k][q];
        df_mac(ps, pc, pq.x, pq.y, Rh[q].x, Rl[q].x);
        df_mac(qs, qc, pq.x, pq.y, Rh[q].y, Rl[q].y);
        df_mac(xs, xc, cq.x, cq.y, Rh[q].x, Rl[q].x);
        df_mac(ys, yc, cq.x, cq.y, Rh[q].y, Rl[q].y);
      }
      const float2 pre = df_norm(ps, pc), pim = df_norm(qs, qc);
      a.pk[k][o] = make_float2(pre.x, pim.x);
      a.pk[k][o + n3] = make_float2(pre.y, pim.y);
      float xrs = x0h.x, xrc = x0l.x, xis = x0h.y, xic = x0l.y;
      df_add(xrs, xrc, xs, xc);
      df_add(xis, xic, ys, yc);
      const float2 xre = df_norm(xrs, xrc), xim = df_norm(xis, xic);
      st_hint(a.xk[k] + o, make_float2(xre.x, xim.x), pol);
      st_hint(a.xk[k] + o + n3, make_float2(xre.y, xim.y), pol);
    }
  }
  close_window(sd, m, a.ticket);
}

cudaError_t launch_df_init(const Geom& g, const double2* b64, void* r, void* p, SolverDev* sd, const InitParams& ip,
                           double* partials, unsigned* ticket, cudaStream_t st) {
  df_init_kernel<<<(g.vh + 255) / 256, 256, 0, st>>>(g, b64, static_cast<float2*>(r), static_cast<float2*>(p), sd, ip,
                                                     partials, ticket);
  return cudaGetLastError();
}

// the update kernels: one block per 256 sites plus the scalar block
cudaError_t launch_df_r_update(const Geom& g, const PerSys<DfUpdArgs>& a, int n, int S, cudaStream_t st, bool pdl) {
  return launch_k(pdl, df_r_update_kernel, dim3((g.vh + 255) / 256 + 1 + n, S), dim3(256), st, g, a);
}

cudaError_t launch_df_p_update(const Geom& g, const PerSys<DfUpdArgs>& a, int S, cudaStream_t st, bool pdl) {
  return launch_k(pdl, df_p_update_kernel, dim3((g.vh + 255) / 256 + 1, S), dim3(256), st, g, a);
}

cudaError_t launch_df_flush(const Geom& g, const PerSys<DfFlushArgs>& a, int S, cudaStream_t st, bool pdl) {
  const int n3 = 3 * g.vh;
  return launch_k(pdl, df_flush_kernel, flush_grid(n3, S), dim3(kFlushThreads), st, n3, a);
}

}  // namespace lqcd

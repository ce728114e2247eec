// dslash.cu - the half-lattice staggered hopping operator (Section 3.2):
//   out(x) = 1/2 sum_mu eta_mu(x) [U_mu(x) in(x+mu) - U_mu(x-mu)^dagger in(x-mu)]
// for every x of the output parity, with optional fused epilogues:
//   AApply : out = a * aux - D in, and the FP64 sum Re<aux, out>   (one half of A = 4m^2 - D_eo D_oe);
//            without a ticket the sum stays as per-block partials for the next kernel
//   Resid  : out = bvec - (a * aux - D in), and the FP64 sum |out|^2 (true residual)
//
// Bandwidth-bound gather kernel: each output site reads 8 links (all links once
// per call) and 8 neighbour vectors (the input vector is small and stays in L2).
// TPS threads cooperate on one site, each taking 8/TPS of the hops, and combine
// their partial sums with warp shuffles; more threads per site means more
// independent loads in flight per SM.  The FP64 mode has a kernel of its own (dslash64_kernel: products on
// the integer multiplier), and so have lattices of at most one block per SM (AHEAD: all loads at once).
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fix64.cuh"
#include "internal.h"
#include "solver_dev.cuh"

namespace lqcd {

// kL12 and up: signs applied after loading; kL64N: FP64 without digits (FixField)
enum LinkFmt { kL64N = -1, kL64 = 0, kL32 = 1, kL12 = 2, kL8 = 3, kL16 = 4 };

constexpr int kFixResident = 3;  // blocks per SM of the FP64 kernels (168 registers per thread)

struct KArgs {
  void* out;
  const void* in;
  const void* aux;
  const void* bvec;
  double a;
  const double* a_dev;
  const float* a_devf;
  int out_parity;
  double* dot_out;
  const int* done;
  double* partials;
  unsigned* ticket;
  const void* links;
  const double2* links64;  // FP64 only (links: its digits or null, FixField)
  int order;  // block-to-site order (site_block)
  const void* upd_r;  // the p update folded in (DslashArgs)
  SolverDev* sd;
  const double* rr_partials;
  int n_rr;
};

// A link as loaded from memory (the compact forms stay compact while their loads are in flight)
// and its decoding into a 3x3 matrix scaled by 1/2 * sign (signs are folded into L64 and L32).
template <int LF>
struct RawLink {
  Mat3<float> m;
};
template <>
struct RawLink<kL12> {
  float4 a, b, c;
};
template <>
struct RawLink<kL8> {
  float4 a, b;
};
template <>
struct RawLink<kL16> {
  int4 a;
  int2 b;
};

template <int LF>
__device__ __forceinline__ RawLink<LF> load_raw(const void* links, int p, int mu, int i, int vh, uint64_t pol) {
  RawLink<LF> r;
  if constexpr (LF == kL32) {
    r.m = load_link32(static_cast<const float*>(links), p, mu, i, vh, pol);
  } else if constexpr (LF == kL12) {
    const float4* blk = static_cast<const float4*>(links) + (size_t)(p * 4 + mu) * 3 * vh;
    r.a = ld_stream(blk + i, pol);
    r.b = ld_stream(blk + vh + i, pol);
    r.c = ld_stream(blk + 2 * vh + i, pol);
  } else if constexpr (LF == kL8) {
    const float4* blk = static_cast<const float4*>(links) + (size_t)(p * 4 + mu) * 2 * vh;
    r.a = ld_stream(blk + i, pol);
    r.b = ld_stream(blk + vh + i, pol);
  } else {
    const char* blk = static_cast<const char*>(links) + (size_t)(p * 4 + mu) * 24 * vh;
    r.a = ld_stream(reinterpret_cast<const int4*>(blk) + i, pol);
    r.b = ld_stream(reinterpret_cast<const int2*>(blk + 16 * (size_t)vh) + i, pol);
  }
  return r;
}

template <int LF>
__device__ __forceinline__ Mat3<float> decode(const RawLink<LF>& r, int sign) {
  if constexpr (LF == kL32) return r.m;
  else if constexpr (LF == kL12) return decode_link12(r.a, r.b, r.c, 0.5f * (float)sign);
  else if constexpr (LF == kL8) return decode_link8(r.a, r.b, 0.5f * (float)sign);
  else return decode_link16(r.a, r.b, 0.5f * (float)sign);
}

// Which colours lane `sub` of a TPS group stores: TPS = 1 all; TPS = 2 lane 0 -> {0, 2},
// lane 1 -> {1}; TPS >= 4 lane c -> colour c (lanes 3.. store nothing).
template <int TPS>
__device__ __forceinline__ bool lane_writes(int sub, int c) {
  if (TPS == 1) return true;
  if (TPS == 2) return sub == 0 ? (c != 1) : (c == 1);
  return c == sub;
}

// The sum of the threads' dsite over the grid (every thread of the block calls).
template <typename T>
__device__ __forceinline__ void dslash_reduce(const KArgs& k, T dsite) {
  if (!k.ticket) {  // the next kernel sums the per-block partials itself (FP32: as (hi, lo) pairs)
    if constexpr (sizeof(T) == 4) {
      const float2 bs = block_sum_f_df(dsite);
      if (threadIdx.x == 0) reinterpret_cast<float2*>(k.partials)[blockIdx.x] = bs;
    } else {
      const double bs = block_sum_mixed(dsite);
      if (threadIdx.x == 0) k.partials[blockIdx.x] = bs;
    }
    return;
  }
  double bs = block_sum_mixed(dsite);
  if (publish_partial(k.partials, k.ticket, bs)) {
    double tot = gather_partials(k.partials, k.ticket);
    if (threadIdx.x == 0 && k.dot_out) *k.dot_out = tot;
  }
}

// Output stage shared by the Dslash kernels: d = (D in)(x) of site i, written as the plain
// output or the A-apply a * aux - d with Re<aux, out>, reduced over the grid by the last block (every thread of the
// block calls).
// UPD: the A-apply may have the p update folded in (k.upd_r).
template <typename T, typename V2, int TPS, int EPI, bool UPD = false>
__device__ __forceinline__ void dslash_epilogue(const KArgs& k, const Vec3<T>& d, int i, int sub, bool valid,
                                                int vh) {
  V2* out = static_cast<V2*>(k.out);
  T aval = (T)k.a;
  if constexpr (EPI != (int)Epi::Plain) {
    if (sizeof(T) == 4 && k.a_devf) aval = (T)*k.a_devf;
    else if (k.a_dev) aval = (T)*k.a_dev;
  }
  T dsite = 0;  // this lane's share of the site's dot product, summed in T, then added in FP64
  if (valid) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (!lane_writes<TPS>(sub, c)) continue;
      size_t o = (size_t)c * vh + i;
      if constexpr (EPI == (int)Epi::Plain) {
        V2 w;
        w.x = d.c[c].re;
        w.y = d.c[c].im;
        out[o] = w;
      } else {
        V2 ps = static_cast<const V2*>(k.aux)[o];
        if constexpr (UPD) {
          if (k.upd_r) {  // uniform: p = r + beta p, as the p update kernel forms it
            const T beta = (T)k.sd->beta_f;
            const V2 r = static_cast<const V2*>(k.upd_r)[o];
            ps.x = fma(beta, ps.x, r.x);
            ps.y = fma(beta, ps.y, r.y);
            static_cast<V2*>(const_cast<void*>(k.aux))[o] = ps;
          }
        }
        T qre = aval * ps.x - d.c[c].re;
        T qim = aval * ps.y - d.c[c].im;
        dsite += ps.x * qre + ps.y * qim;
        V2 w;
        w.x = qre;
        w.y = qim;
        out[o] = w;
      }
    }
  }
  if constexpr (EPI != (int)Epi::Plain) dslash_reduce<T>(k, dsite);
}

// The hops of lane `sub` of output site i (TPS lanes per site): h = sub, sub + TPS, ...; h even
// is the forward hop along mu = h / 2 (U_mu(x) in(x + mu)), h odd the backward one
// (U_mu(x - mu)^dagger in(x - mu), the link stored at x - mu in the other parity's block).
// start() computes the neighbours and signs and issues the first link's loads; apply() runs the
// two-stage software pipeline (the loads of hop q + 1 in flight while hop q is computed) and
// returns the lane's share of (D in)(x).  Shared by the single-lattice and the batched kernels.
template <int LF, int TPS>
struct SiteHops {
  typedef float T;
  typedef float2 V2;
  static constexpr int NH = 8 / TPS;
  int nb[NH], sg[NH];
  RawLink<LF> Wn;

  __device__ __forceinline__ RawLink<LF> link(const void* links, int p, int i, int sub, int q, int vh,
                                              uint64_t pol) const {
    const int h = sub + q * TPS;
    return (h & 1) ? load_raw<LF>(links, 1 - p, h >> 1, nb[q], vh, pol) : load_raw<LF>(links, p, h >> 1, i, vh, pol);
  }

  __device__ __forceinline__ void start(const Geom& g, const void* links, int p, int i, int sub, uint64_t pol) {
    Site s = site_of(g, p, i);
#pragma unroll
    for (int q = 0; q < NH; ++q) {
      const int h = sub + q * TPS;  // TPS divides 8, so h < 8 and its parity is sub's
      const int mu = h >> 1;
      if ((h & 1) == 0) {
        nb[q] = neighbour_half(g, neighbour_fwd(g, s, mu));
        sg[q] = (LF >= kL12) ? link_sign_fwd(g, s, mu) : 1;
      } else {
        nb[q] = neighbour_half(g, neighbour_bwd(g, s, mu));
        sg[q] = (LF >= kL12) ? link_sign_bwd(g, s, mu) : 1;
      }
    }
    Wn = link(links, p, i, sub, 0, g.vh, pol);
  }

  __device__ __forceinline__ Vec3<T> apply(const void* links, const V2* in, int p, int i, int sub, int vh,
                                           uint64_t pol) {
    Vec3<T> accf = vzero<T>(), accb = vzero<T>();
    Vec3<T> vn = ldg_vec(in, nb[0], vh);
#pragma unroll
    for (int q = 0; q < NH; ++q) {
      const Mat3<T> W = decode<LF>(Wn, sg[q]);
      Vec3<T> v = vn;
      if (q + 1 < NH) {
        Wn = link(links, p, i, sub, q + 1, vh, pol);
        vn = ldg_vec(in, nb[q + 1], vh);
      }
      if (((sub + q * TPS) & 1) == 0) mv_acc(accf, W, v);
      else mdv_acc(accb, W, v);
    }
    Vec3<T> d;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.c[c] = cmake(accf.c[c].re - accb.c[c].re, accf.c[c].im - accb.c[c].im);
    return d;
  }
};

// The same hops with every load issued at once: all links by start(), all vectors by apply().  The sums and
// their order are those of SiteHops<LF, 1>, so the bits are too.  About 230 registers (18-real links).
template <int LF>
struct SiteHopsAhead {
  int nb[8], sg[8];
  RawLink<LF> W[8];

  __device__ __forceinline__ void start(const Geom& g, const void* links, int p, int i, int, uint64_t pol) {
    const Site s = site_of(g, p, i);
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const int mu = h >> 1;
      const bool fwd = (h & 1) == 0;
      nb[h] = neighbour_half(g, fwd ? neighbour_fwd(g, s, mu) : neighbour_bwd(g, s, mu));
      sg[h] = (LF >= kL12) ? (fwd ? link_sign_fwd(g, s, mu) : link_sign_bwd(g, s, mu)) : 1;
      W[h] = fwd ? load_raw<LF>(links, p, mu, i, g.vh, pol) : load_raw<LF>(links, 1 - p, mu, nb[h], g.vh, pol);
    }
  }

  __device__ __forceinline__ Vec3<float> apply(const void*, const float2* in, int, int, int, int vh, uint64_t) {
    Vec3<float> v[8];
#pragma unroll
    for (int h = 0; h < 8; ++h) v[h] = ldg_vec(in, nb[h], vh);
    return apply_to(v);
  }

  __device__ __forceinline__ Vec3<float> apply_to(const Vec3<float> (&v)[8]) const {
    Vec3<float> accf = vzero<float>(), accb = vzero<float>();
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const Mat3<float> M = decode<LF>(W[h], sg[h]);
      if ((h & 1) == 0) mv_acc(accf, M, v[h]);
      else mdv_acc(accb, M, v[h]);
    }
    Vec3<float> d;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.c[c] = cmake(accf.c[c].re - accb.c[c].re, accf.c[c].im - accb.c[c].im);
    return d;
  }
};

// The chunk of output sites block blockIdx.x works on.  order 0: chunk b = block b (lexicographic
// within the parity, the order of the stored vectors); order 1: the two halves of the site range
// interleaved, even blocks taking the first half and odd blocks the second, so that blocks that run
// at the same time stream from two distant regions of the lattice (and of every link block).  A
// bijection on [0, gridDim.x); the per-block partial sums stay indexed by blockIdx.x.
__device__ __forceinline__ int site_block(int order) {
  const int b = blockIdx.x;
  if (!order) return b;
  const int h = (gridDim.x + 1) >> 1;
  return (b & 1) ? h + (b >> 1) : (b >> 1);
}

// AHEAD (TPS = 1): small lattices, whose launches are all latency (launch_tps).
template <int LF, int TPS, int EPI, bool AHEAD = false>
__global__ void __launch_bounds__(128, AHEAD ? 1 : 7) dslash_kernel(Geom g, KArgs k) {
  typedef float T;
  typedef float2 V2;
  typedef typename std::conditional<AHEAD, SiteHopsAhead<LF>, SiteHops<LF, TPS>>::type Hops;
  const int vh = g.vh;
  const int gt = site_block(k.order) * blockDim.x + threadIdx.x;
  const int i = gt / TPS;
  const int sub = gt % TPS;
  const bool valid = i < vh;
  const int p = k.out_parity;
  const V2* in = static_cast<const V2*>(k.in);
  const uint64_t pol = policy_evict_last();
  Hops hops;
  // links are never written by the kernels of a solve: the first one is fetched before the wait
  if (valid) hops.start(g, k.links, p, i, sub, pol);
  pdl_wait();
  pdl_trigger();
  if (k.done && *k.done) return;  // uniform: the flag only changes between kernels

  Vec3<T> part = vzero<T>();
  if (valid) part = hops.apply(k.links, in, p, i, sub, vh, pol);
  // D in = fwd - bwd, summed over the TPS lanes of the site
  Vec3<T> d;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    T re = part.c[c].re;
    T im = part.c[c].im;
#pragma unroll
    for (int o = 1; o < TPS; o <<= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    d.c[c] = cmake(re, im);
  }

  dslash_epilogue<T, V2, TPS, EPI, AHEAD>(k, d, i, sub, valid, vh);
}

// The plain hop with the p update folded in (small lattices, one system): in is the p before it.  While the links and
// vectors are on their way, every block sums the r update's partials as the p update kernel does (the same beta, so the
// same bits); the last block runs the beta step.  A launch and a round trip less per iteration: p_update takes 1.4 us and
// a launch gap of 0.9, the sum here about 0.8.
template <int LF>
__global__ void __launch_bounds__(128, 1) dslash_pupdate_kernel(Geom g, KArgs k) {
  __shared__ __align__(8) float2 rs[8][3][128];  // each thread's neighbours of r (registers hold p and the links)
  const int vh = g.vh, t = threadIdx.x, p = k.out_parity;
  const bool scalar_block = blockIdx.x == gridDim.x - 1;
  const int i = blockIdx.x * 128 + t;
  const bool valid = !scalar_block && i < vh;
  const float2* in = static_cast<const float2*>(k.in);
  const float2* r = static_cast<const float2*>(k.upd_r);
  SiteHopsAhead<LF> hops;
  if (valid) hops.start(g, k.links, p, i, 0, policy_evict_last());
  pdl_wait();
  pdl_trigger();
  SolverDev* sd = k.sd;
  const bool skip = *reinterpret_cast<const volatile int*>(&sd->done) != 0;
  const float2 rr_b_df = sd->rr_b_df;
  Vec3<float> v[8];
  if (valid) {
#pragma unroll
    for (int h = 0; h < 8; ++h) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(&rs[h][c][t])),
                     "l"(r + (size_t)c * vh + hops.nb[h])
                     : "memory");
      v[h] = load_vec(in, hops.nb[h], vh);
    }
  }
  const PartialsRatio pb = partials_ratio_df<true>(k.rr_partials, k.n_rr, rr_b_df, skip, scalar_block);
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (pb.stop) return;  // the same in every thread of the block
  if (scalar_block) {
    solver_beta_step(sd, pb);
    return;
  }
  if (!valid) return;
  const float beta = pb.ratio_f;
#pragma unroll
  for (int h = 0; h < 8; ++h) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2 w = rs[h][c][t];
      v[h].c[c].re = fma(beta, v[h].c[c].re, w.x);
      v[h].c[c].im = fma(beta, v[h].c[c].im, w.y);
    }
  }
  store_vec(static_cast<float2*>(k.out), i, vh, hops.apply_to(v));
}

// FP64: the products in block fixed point (fix64.cuh), one direction per thread.  Blocks take groups of
// kFixSites sites in turn; the next group's forward links are in flight while a group is finished.
// DIGITS: whether the field keeps its digits (FixField); half Dslash at 32^3x8 36 us with, 50 without (FP64 multiply-adds: 70).
template <int EPI, bool DIGITS>
__global__ void __launch_bounds__(kFixThreads, kFixResident) dslash64_kernel(Geom g, KArgs k) {
  __shared__ FixShared sh;
  const int vh = g.vh;
  const int mu = threadIdx.x / kFixSites, ls = threadIdx.x % kFixSites;
  const int p = k.out_parity;
  const double2* in = static_cast<const double2*>(k.in);
  const FixField U{static_cast<const int4*>(k.links), k.links64};
  const uint64_t pol = policy_evict_first();  // 8 % faster than evict_last, or than keeping part of them
  const int step = gridDim.x * kFixSites;
  int i = blockIdx.x * kFixSites + ls;
  FixGroup<DIGITS> grp;
  if (i < vh) grp.start(g, U, p, i, mu, pol);
  pdl_wait();
  pdl_trigger();
  if (k.done && *k.done) return;  // uniform: the flag only changes between kernels
  const double a = k.a_dev ? *k.a_dev : k.a;
  double2* out = static_cast<double2*>(k.out);
  double dsite = 0.0;
  for (int i0 = blockIdx.x * kFixSites; i0 < vh; i0 += step, i += step) {
    const bool valid = i < vh, mine = valid && mu < 3;
    const size_t o = (size_t)mu * vh + i;
    double2 ps, bv;  // the epilogue's own-site loads, in flight beside the neighbours'
    if constexpr (EPI != (int)Epi::Plain)
      if (mine) ps = static_cast<const double2*>(k.aux)[o];
    if constexpr (EPI == (int)Epi::Resid)
      if (mine) bv = static_cast<const double2*>(k.bvec)[o];
    grp.hops(sh, g, U, in, p, mu, ls, valid, pol);
    if (i + step < vh) grp.start(g, U, p, i + step, mu, pol);
    __syncthreads();
    Cplx<double> d;
    if (mu < 3) d = FixGroup<DIGITS>::colour(sh, g, k.links64, in, p, i, mu, ls, valid);
    if (mine) {
      double2 w = make_double2(d.re, d.im);
      if constexpr (EPI != (int)Epi::Plain) {
        w = make_double2(a * ps.x - d.re, a * ps.y - d.im);
        if constexpr (EPI == (int)Epi::AApply) {
          dsite += ps.x * w.x + ps.y * w.y;
        } else {
          w = make_double2(bv.x - w.x, bv.y - w.y);
          dsite += w.x * w.x + w.y * w.y;
        }
      }
      out[o] = w;
    }
    __syncthreads();  // sh is written again in the next turn
  }
  if constexpr (EPI != (int)Epi::Plain) dslash_reduce<double>(k, dsite);
}

// The half-lattice hop of NS systems that share one operator (the right-hand sides of a multi-RHS
// shifted solve): every link is loaded and decoded once and applied to the NS input vectors, so the
// link traffic per system drops by NS.  One thread per output site; per system the arithmetic (the
// hop order, the forward and backward accumulators) and the epilogue are those of dslash_kernel with
// one thread per site, so every system's output and partial sums equal its own launch's bit for bit.
template <int LF, int NS, int EPI>
__global__ void __launch_bounds__(128, NS <= 2 ? 4 : 3) dslash_msys_kernel(Geom g,
                                                                          const __grid_constant__ PerSys<KArgs> pk) {
  typedef float T;
  typedef float2 V2;
  const int vh = g.vh;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i < vh;
  const int p = pk.s[0].out_parity;
  const void* links = pk.s[0].links;
  const uint64_t pol = policy_evict_last();
  SiteHops<LF, 1> hops;
  if (valid) hops.start(g, links, p, i, 0, pol);
  pdl_wait();
  pdl_trigger();
  bool all_done = true;  // uniform: the flags only change between kernels
#pragma unroll
  for (int s = 0; s < NS; ++s) all_done = all_done && pk.s[s].done && *pk.s[s].done;
  if (all_done) return;

  Vec3<T> accf[NS], accb[NS], vn[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) accf[s] = accb[s] = vzero<T>();
  if (valid) {
#pragma unroll
    for (int s = 0; s < NS; ++s) vn[s] = ldg_vec(static_cast<const V2*>(pk.s[s].in), hops.nb[0], vh);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const Mat3<T> W = decode<LF>(hops.Wn, hops.sg[q]);
      Vec3<T> v[NS];
#pragma unroll
      for (int s = 0; s < NS; ++s) v[s] = vn[s];
      if (q + 1 < 8) {
        hops.Wn = hops.link(links, p, i, 0, q + 1, vh, pol);
#pragma unroll
        for (int s = 0; s < NS; ++s) vn[s] = ldg_vec(static_cast<const V2*>(pk.s[s].in), hops.nb[q + 1], vh);
      }
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        if ((q & 1) == 0) mv_acc(accf[s], W, v[s]);
        else mdv_acc(accb[s], W, v[s]);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    Vec3<T> d;
#pragma unroll
    for (int c = 0; c < 3; ++c) d.c[c] = cmake(accf[s].c[c].re - accb[s].c[c].re, accf[s].c[c].im - accb[s].c[c].im);
    dslash_epilogue<T, V2, 1, EPI>(pk.s[s], d, i, 0, valid, vh);
  }
}

// ---------------------------------------------------------------------------------------------
// Batched half-Dslash over many lattices of different sizes in one persistent launch.  The work
// is split into items of kBatchChunk output sites of one lattice (chunk_end holds the prefix
// sums of the lattices' item counts); every block takes items from a global counter until none
// are left, so uneven lattices load-balance over the SMs and small lattices that could not fill
// the GPU on their own share it.  One thread per site, the same per-site arithmetic as
// dslash_kernel (bit-identical outputs).  No block waits on another: the counter only hands out
// items.  The descriptors are copied from the parameter block to shared memory with constant
// offsets once per block, and every index taken from them is checked before use.
// ---------------------------------------------------------------------------------------------
constexpr int kBatchChunk = 128;
static_assert(sizeof(BatchArgs) <= 4000, "the batch descriptors travel as the kernel's parameter block");
static_assert(kBatchPerLaunch <= kBatchChunk, "one thread per descriptor");
static_assert(kFixThreads == kBatchChunk, "the FP64 groups use the whole block");

// The persistent loop shared by both batched kernels: blocks take 128-site chunks of any lattice
// from the work counter until none are left (lat and chunk_end already in shared memory).
template <int LF>
__device__ __forceinline__ void batch_loop(const BatchLattice* lat, const int* chunk_end, int n, unsigned* head,
                                           int* item_s) {
  typedef float T;
  typedef float2 V2;
  const int n_items = chunk_end[n];
  const uint64_t pol = policy_evict_last();
  for (;;) {
    if (threadIdx.x == 0) *item_s = (int)atomicAdd(head, 1u);
    __syncthreads();
    const int it = *item_s;
    __syncthreads();  // item_s is written again at the top of the next round
    if (it >= n_items) break;
    int l = 0;  // the lattice of item it: chunk_end[l] <= it < chunk_end[l + 1] (binary search)
    for (int lo = 0, hi = n - 1; lo <= hi;) {
      const int mid = (lo + hi) >> 1;
      if (chunk_end[mid + 1] <= it) {
        lo = mid + 1;
        l = lo;
      } else {
        hi = mid - 1;
      }
    }
    if (l >= n) continue;
    const BatchLattice& L = lat[l];
    const int i0 = (it - chunk_end[l]) * kBatchChunk;
    if constexpr (LF <= kL64) {
      __shared__ FixShared sh;
      const int mu = threadIdx.x / kFixSites, ls = threadIdx.x % kFixSites, vh = L.g.vh, p = L.out_parity;
      const FixField U{static_cast<const int4*>(L.links), L.links64};
      const double2* in = static_cast<const double2*>(L.in);
      typedef FixGroup<LF == kL64> Group;
      for (int j0 = i0; j0 < min(i0 + kBatchChunk, vh); j0 += kFixSites) {
        const int i = j0 + ls;
        const bool valid = i < vh;
        Group grp;
        if (valid) grp.start(L.g, U, p, i, mu, pol);
        grp.hops(sh, L.g, U, in, p, mu, ls, valid, pol);
        __syncthreads();
        Cplx<double> d;
        if (mu < 3) d = Group::colour(sh, L.g, L.links64, in, p, i, mu, ls, valid);
        if (valid && mu < 3) {
          static_cast<double2*>(L.out)[(size_t)mu * vh + i] = make_double2(d.re, d.im);
        }
        __syncthreads();
      }
    } else {
      const int i = i0 + threadIdx.x;
      if (i >= 0 && i < L.g.vh) {
        SiteHops<LF, 1> hops;
        hops.start(L.g, L.links, L.out_parity, i, 0, pol);
        const Vec3<T> d = hops.apply(L.links, static_cast<const V2*>(L.in), L.out_parity, i, 0, L.g.vh, pol);
        store_vec(static_cast<V2*>(L.out), i, L.g.vh, d);
      }
    }
  }
}

// descriptors in the parameter block (up to kBatchPerLaunch lattices), copied to shared memory
template <int LF>
__global__ void __launch_bounds__(kBatchChunk, LF <= kL64 ? kFixResident : 7)
    dslash_batch_kernel(BatchArgs a, unsigned* head) {
  __shared__ BatchLattice lat[kBatchPerLaunch];
  __shared__ int chunk_end[kBatchPerLaunch + 1];
  __shared__ int item_s;
#pragma unroll
  for (int j = 0; j < kBatchPerLaunch; ++j)
    if (threadIdx.x == j) lat[j] = a.lat[j];
#pragma unroll
  for (int j = 0; j <= kBatchPerLaunch; ++j)
    if (threadIdx.x == j) chunk_end[j] = a.chunk_end[j];
  const int n = a.n;
  if (n < 1 || n > kBatchPerLaunch) return;  // uniform; the host never passes such a block
  __syncthreads();
  batch_loop<LF>(lat, chunk_end, n, head, &item_s);
}

// descriptors in a device table (up to kMaxBatch lattices), copied to shared memory
template <int LF>
__global__ void __launch_bounds__(kBatchChunk, LF <= kL64 ? kFixResident : 7)
    dslash_batch_table_kernel(const BatchTable* __restrict__ tab, unsigned* head) {
  __shared__ BatchLattice lat[kMaxBatch];
  __shared__ int chunk_end[kMaxBatch + 1];
  __shared__ int item_s;
  const int n = tab->n;
  if (n < 1 || n > kMaxBatch) return;  // uniform; the host never uploads such a table
  for (int j = threadIdx.x; j < n; j += blockDim.x) lat[j] = tab->lat[j];
  for (int j = threadIdx.x; j <= n; j += blockDim.x) chunk_end[j] = tab->chunk_end[j];
  __syncthreads();
  batch_loop<LF>(lat, chunk_end, n, head, &item_s);
}

int batch_items(int vh) { return (vh + kBatchChunk - 1) / kBatchChunk; }

cudaError_t launch_dslash_batch(const BatchArgs& a, int prec, unsigned* head, int n_sm, cudaStream_t st) {
  const int items = a.chunk_end[a.n];
  if (items <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(head, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  // one resident wave of persistent blocks
  const unsigned grid = (unsigned)std::min(items, (prec == LQCD_FP64 ? kFixResident : 7) * n_sm);
  switch (prec) {
    case LQCD_FP64: {
      bool digits = true;  // of every lattice
      for (int j = 0; j < a.n; ++j) digits = digits && a.lat[j].links;
      if (digits) dslash_batch_kernel<kL64><<<grid, kBatchChunk, 0, st>>>(a, head);
      else dslash_batch_kernel<kL64N><<<grid, kBatchChunk, 0, st>>>(a, head);
      break;
    }
    case LQCD_FP32_R12: dslash_batch_kernel<kL12><<<grid, kBatchChunk, 0, st>>>(a, head); break;
    case LQCD_FP32_R8: dslash_batch_kernel<kL8><<<grid, kBatchChunk, 0, st>>>(a, head); break;
    case LQCD_FP32_L16: dslash_batch_kernel<kL16><<<grid, kBatchChunk, 0, st>>>(a, head); break;
    default: dslash_batch_kernel<kL32><<<grid, kBatchChunk, 0, st>>>(a, head); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_dslash_batch_table(const BatchTable* tab, int n_items, int prec, bool digits, unsigned* head, int n_sm,
                                      cudaStream_t st) {
  if (n_items <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(head, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  // one resident wave of persistent blocks
  const unsigned grid = (unsigned)std::min(n_items, (prec == LQCD_FP64 ? kFixResident : 7) * n_sm);
  switch (prec) {
    case LQCD_FP64:
      if (digits) dslash_batch_table_kernel<kL64><<<grid, kBatchChunk, 0, st>>>(tab, head);
      else dslash_batch_table_kernel<kL64N><<<grid, kBatchChunk, 0, st>>>(tab, head);
      break;
    case LQCD_FP32_R12: dslash_batch_table_kernel<kL12><<<grid, kBatchChunk, 0, st>>>(tab, head); break;
    case LQCD_FP32_R8: dslash_batch_table_kernel<kL8><<<grid, kBatchChunk, 0, st>>>(tab, head); break;
    case LQCD_FP32_L16: dslash_batch_table_kernel<kL16><<<grid, kBatchChunk, 0, st>>>(tab, head); break;
    default: dslash_batch_table_kernel<kL32><<<grid, kBatchChunk, 0, st>>>(tab, head); break;
  }
  return cudaGetLastError();
}

template <int LF, int TPS>
static cudaError_t launch_tps(const Geom& g, const KArgs& k, Epi epi, cudaStream_t st, int bs, bool pdl) {
  if (epi == Epi::Resid) return cudaErrorInvalidValue;  // FP64 (launch_fp64) and double-FP32 only
  long long threads = (long long)g.vh * TPS;
  unsigned nb = (unsigned)((threads + bs - 1) / bs);
  // At most one block per SM: all loads at once.  Half Dslash per graph launch, 18-real links: 8^4 2.32 -> 1.98 us, 16^3x8
  // (128 blocks) 2.68 -> 2.38; with more blocks the other warps hide the latency better: 16^3x10 (160) 2.64 and 2.83,
  // 20^3x8 (250) 3.07 and 3.20, 24^3x6 (324) 3.37 and 4.72.
  if constexpr (TPS == 1) {
    if (nb <= kSMs) {
      if (epi == Epi::Plain && k.upd_r) return launch_k(pdl, dslash_pupdate_kernel<LF>, dim3(nb + 1), dim3(128), st, g, k);
      if (epi == Epi::Plain) return launch_k(pdl, dslash_kernel<LF, 1, 0, true>, dim3(nb), dim3(bs), st, g, k);
      return launch_k(pdl, dslash_kernel<LF, 1, 1, true>, dim3(nb), dim3(bs), st, g, k);
    }
  }
  if (epi == Epi::Plain) return launch_k(pdl, dslash_kernel<LF, TPS, 0>, dim3(nb), dim3(bs), st, g, k);
  return launch_k(pdl, dslash_kernel<LF, TPS, 1>, dim3(nb), dim3(bs), st, g, k);
}

template <int LF>
static cudaError_t launch_lf(const Geom& g, const KArgs& k, Epi epi, int tps, int bs, cudaStream_t st, bool pdl) {
  switch (tps) {
    case 1: return launch_tps<LF, 1>(g, k, epi, st, bs, pdl);
    case 2: return launch_tps<LF, 2>(g, k, epi, st, bs, pdl);
    case 4: return launch_tps<LF, 4>(g, k, epi, st, bs, pdl);
    default: return launch_tps<LF, 8>(g, k, epi, st, bs, pdl);
  }
}

// FP64 blocks: one per group of sites, at most one resident wave (the blocks then take several groups each)
static int fp64_blocks(const Geom& g) { return std::min((g.vh + kFixSites - 1) / kFixSites, kFixResident * kSMs); }

template <bool DIGITS>
static cudaError_t launch_fp64(const Geom& g, const KArgs& k, Epi epi, cudaStream_t st, bool pdl) {
  const dim3 nb((unsigned)fp64_blocks(g)), bs(kFixThreads);
  switch (epi) {
    case Epi::Plain: return launch_k(pdl, dslash64_kernel<0, DIGITS>, nb, bs, st, g, k);
    case Epi::AApply: return launch_k(pdl, dslash64_kernel<1, DIGITS>, nb, bs, st, g, k);
    default: return launch_k(pdl, dslash64_kernel<2, DIGITS>, nb, bs, st, g, k);
  }
}

static int default_tps(int) { return 1; }  // fastest on GB300 at 16^3x8 and 32^3x8 (sweep over 1, 2, 4, 8)

bool fold_p_update(const Geom& g, int tps, int bs, int order) {
  return (tps <= 0 ? default_tps(LQCD_FP32) : tps) == 1 && (bs <= 0 || bs == 128) && order == 0 && (g.vh + 127) / 128 <= kSMs;
}

// blocks of one Dslash launch (= partials it writes)
int dslash_grid_blocks(const Geom& g, int prec, int tps, int bs) {
  if (prec == LQCD_FP64) return fp64_blocks(g);
  if (tps <= 0) tps = default_tps(prec);
  if (bs <= 0) bs = 128;
  long long threads = (long long)g.vh * tps;
  return (int)((threads + bs - 1) / bs);
}

cudaError_t launch_dslash(const Geom& g, const GaugeCopies& gc, const DslashArgs& a, cudaStream_t st, int* nlaunch) {
  KArgs k;
  k.out = a.out;
  k.in = a.in;
  k.aux = a.aux;
  k.bvec = a.bvec;
  k.a = a.a;
  k.a_dev = a.a_dev;
  k.a_devf = a.a_devf;
  k.out_parity = a.out_parity;
  k.dot_out = a.dot_out;
  k.done = a.done;
  k.partials = a.partials;
  k.ticket = a.ticket;
  int tps = a.tps > 0 ? a.tps : default_tps(a.prec);
  if (tps != 1 && tps != 2 && tps != 4 && tps != 8) return cudaErrorInvalidValue;
  const int bs = a.bs > 0 ? a.bs : 128;
  if (bs != 64 && bs != 128) return cudaErrorInvalidValue;
  k.order = (a.prec == LQCD_FP64) ? 0 : a.order;
  k.upd_r = a.upd_r;
  k.sd = a.sd;
  k.rr_partials = a.rr_partials;
  k.n_rr = a.n_rr;
  if (k.upd_r && (a.prec == LQCD_FP64 || !fold_p_update(g, a.tps, a.bs, a.order))) return cudaErrorInvalidValue;
  if (nlaunch) *nlaunch += 1;
  switch (a.prec) {
    case LQCD_FP64:
      k.links = gc.ufix;
      k.links64 = gc.u64;
      return gc.ufix ? launch_fp64<true>(g, k, a.epi, st, a.pdl) : launch_fp64<false>(g, k, a.epi, st, a.pdl);
    case LQCD_FP32_R12: k.links = gc.u12; return launch_lf<kL12>(g, k, a.epi, tps, bs, st, a.pdl);
    case LQCD_FP32_R8: k.links = gc.u8; return launch_lf<kL8>(g, k, a.epi, tps, bs, st, a.pdl);
    case LQCD_FP32_L16: k.links = gc.u16; return launch_lf<kL16>(g, k, a.epi, tps, bs, st, a.pdl);
    default: k.links = gc.u32; return launch_lf<kL32>(g, k, a.epi, tps, bs, st, a.pdl);
  }
}

template <int LF, int NS>
static cudaError_t launch_msys_ns(const Geom& g, const PerSys<KArgs>& k, Epi epi, cudaStream_t st, bool pdl) {
  const dim3 grid((unsigned)((g.vh + 127) / 128));
  switch (epi) {
    case Epi::Plain: return launch_k(pdl, dslash_msys_kernel<LF, NS, 0>, grid, dim3(128), st, g, k);
    case Epi::AApply: return launch_k(pdl, dslash_msys_kernel<LF, NS, 1>, grid, dim3(128), st, g, k);
    default: return launch_k(pdl, dslash_msys_kernel<LF, NS, 2>, grid, dim3(128), st, g, k);
  }
}

template <int LF>
static cudaError_t launch_msys_lf(const Geom& g, const PerSys<KArgs>& k, int S, Epi epi, cudaStream_t st, bool pdl) {
  switch (S) {
    case 2: return launch_msys_ns<LF, 2>(g, k, epi, st, pdl);
    case 3: return launch_msys_ns<LF, 3>(g, k, epi, st, pdl);
    default: return launch_msys_ns<LF, 4>(g, k, epi, st, pdl);
  }
}

cudaError_t launch_dslash_msys(const Geom& g, const GaugeCopies& gc, const PerSys<DslashArgs>& a, int S,
                               cudaStream_t st, int* nlaunch) {
  if (S < 2 || S > kMaxRhs) return cudaErrorInvalidValue;
  const DslashArgs& a0 = a.s[0];
  PerSys<KArgs> k;
  memset(&k, 0, sizeof(k));
  const void* links = nullptr;
  switch (a0.prec) {
    case LQCD_FP32: links = gc.u32; break;
    case LQCD_FP32_R12: links = gc.u12; break;
    case LQCD_FP32_R8: links = gc.u8; break;
    case LQCD_FP32_L16: links = gc.u16; break;
    default: return cudaErrorInvalidValue;  // the FP32 Krylov modes only
  }
  for (int s = 0; s < S; ++s) {
    const DslashArgs& x = a.s[s];
    if (x.prec != a0.prec || x.epi != a0.epi || x.out_parity != a0.out_parity) return cudaErrorInvalidValue;
    KArgs& y = k.s[s];
    y.out = x.out;
    y.in = x.in;
    y.aux = x.aux;
    y.bvec = x.bvec;
    y.a = x.a;
    y.a_dev = x.a_dev;
    y.a_devf = x.a_devf;
    y.out_parity = x.out_parity;
    y.dot_out = x.dot_out;
    y.done = x.done;
    y.partials = x.partials;
    y.ticket = x.ticket;
    y.links = links;
  }
  if (nlaunch) *nlaunch += 1;
  switch (a0.prec) {
    case LQCD_FP32_R12: return launch_msys_lf<kL12>(g, k, S, a0.epi, st, a0.pdl);
    case LQCD_FP32_R8: return launch_msys_lf<kL8>(g, k, S, a0.epi, st, a0.pdl);
    case LQCD_FP32_L16: return launch_msys_lf<kL16>(g, k, S, a0.epi, st, a0.pdl);
    default: return launch_msys_lf<kL32>(g, k, S, a0.epi, st, a0.pdl);
  }
}

}  // namespace lqcd

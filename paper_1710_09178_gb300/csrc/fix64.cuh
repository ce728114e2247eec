// fix64.cuh - the FP64 half Dslash of a group of sites in block fixed point (fixpoint.h).
//
// Measured on GB300, half Dslash per graph launch (caches as the previous launches leave them), with FP64
// multiply-adds and one thread per site before:
//     8^4 12.0 -> 3.1 us, 16^3x8 12.8 -> 6.7, 24^3x6 30.8 -> 13.1, 32^3x8 69.8 -> 35.4, 48^3x12 329 -> 171
// (32^3x8: 163.6 MB, 24 us at the measured HBM rate).  It runs 17.4 M warp instructions there, 45 % of them
// on the ALU (digits, addresses) and 39 % on the integer multiplier: issue and load latency share the bound.
// One direction (two hops) per thread, 3 blocks of 128 threads per SM (168 registers): 4 blocks spill and take
// 39 us, one hop per thread 36.5 us, one thread per site 68.6 us.
#pragma once

#include "common.cuh"
#include "fixpoint.h"

namespace lqcd {

constexpr int kFixBadLink = (int)0x80000000;         // high digit of entry (0, 0) of a link outside the format
constexpr int64_t kFixBadSum = (int64_t)(1ull << 63);  // a sum with such a link

struct FixLink {
  int4 e[9];  // (re.h, re.l, im.h, im.l), row-major
};

// Storage: [parity][mu][ceil(Vh / 32)][9][32] int4, so that a thread's nine loads share one address.
__host__ __device__ inline size_t fix_block_entries(int vh) { return (size_t)((vh + 31) / 32) * 9 * 32; }
__device__ __forceinline__ size_t fix_entry(int p, int mu, int i, int vh) {
  return (size_t)(p * 4 + mu) * fix_block_entries(vh) + (size_t)((unsigned)i >> 5) * (9 * 32) + (i & 31);
}

// The links of a field: their digits, or (null: not kept, GaugeCopies) the FP64 copy, which then gives them while they
// are read: the same digits, so the same results.  The FP64 copy [2][4][9][Vh] is followed by one byte per link, [2][4][Vh]:
// whether it is within the format.
struct FixField {
  const int4* digits;
  const double2* u64;
};
__host__ __device__ __forceinline__ const unsigned char* fix_fits(const double2* u64, int vh) {
  return reinterpret_cast<const unsigned char*>(u64 + 72 * (size_t)vh);
}

// A link as it is loaded: its digits, or (DIGITS false) its FP64 entries, with fits from that copy.
template <bool DIGITS>
struct FixRaw {
  int4 e[9];
  int fits;
};

template <bool DIGITS>
__device__ __forceinline__ FixRaw<DIGITS> load_link_fix(const FixField& f, int p, int mu, int i, int vh, uint64_t pol) {
  FixRaw<DIGITS> r;
  if constexpr (DIGITS) {
    const int4* b = f.digits + fix_entry(p, mu, i, vh);
#pragma unroll
    for (int j = 0; j < 9; ++j) r.e[j] = ld_stream(b + j * 32, pol);
  } else {
    const int4* b = reinterpret_cast<const int4*>(f.u64) + (size_t)(p * 4 + mu) * 9 * vh + i;
#pragma unroll
    for (int j = 0; j < 9; ++j) r.e[j] = ld_stream(b + (size_t)j * vh, pol);
    r.fits = fix_fits(f.u64, vh)[(size_t)(p * 4 + mu) * vh + i];
  }
  return r;
}

// The digits of a loaded link; entry (0, 0) marked where it is outside the format.
template <bool DIGITS>
__device__ __forceinline__ FixLink fix_digits(const FixRaw<DIGITS>& r) {
  FixLink L;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    if constexpr (DIGITS) {
      L.e[j] = r.e[j];
    } else {
      const Fix2 re = fix_link_entry(__hiloint2double(r.e[j].y, r.e[j].x)), im = fix_link_entry(__hiloint2double(r.e[j].w, r.e[j].z));
      L.e[j] = make_int4(re.h, re.l, im.h, im.l);
    }
  }
  if constexpr (!DIGITS)
    if (!r.fits) L.e[0].x = kFixBadLink;
  return L;
}

struct FixAcc {
  int64_t rh[3], rx[3], ih[3], ix[3];
};

// acc += U v (FWD) or -U^dagger v
template <bool FWD>
__device__ __forceinline__ void fix_hop(FixAcc& s, const FixLink& L, const Vec3<double>& v, int E) {
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const Fix2 wr = fix_component<!FWD>(v.c[b].re, E), wi = fix_component<!FWD>(v.c[b].im, E);
    // what the minus sign of the complex product falls on
    const Fix2 n = FWD ? Fix2{-wi.h, -wi.l} : Fix2{-wr.h, -wr.l};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int4 u = L.e[FWD ? a * 3 + b : b * 3 + a];
      fix_mac(s.rh[a], s.rx[a], u.x, u.y, wr);
      fix_mac(s.rh[a], s.rx[a], u.z, u.w, FWD ? n : wi);
      fix_mac(s.ih[a], s.ix[a], u.x, u.y, wi);
      fix_mac(s.ih[a], s.ix[a], u.z, u.w, FWD ? wr : n);
    }
  }
}

// The same site in FP64, for what the format does not take: fma chains per hop, forward minus backward,
// directions in order.
static __device__ __noinline__ Vec3<double> site64_fma(Geom g, const double2* __restrict__ U,
                                                        const double2* __restrict__ in, int p, int i) {
  const int vh = g.vh;
  const Site s = site_of(g, p, i);
  const uint64_t pol = policy_evict_first();
  Vec3<double> d = vzero<double>();
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    const int jf = neighbour_half(g, neighbour_fwd(g, s, mu)), jb = neighbour_half(g, neighbour_bwd(g, s, mu));
    Vec3<double> f = vzero<double>(), b = vzero<double>();
    mv_acc(f, load_link64(U, p, mu, i, vh, pol), ldg_vec(in, jf, vh));
    mdv_acc(b, load_link64(U, 1 - p, mu, jb, vh, pol), ldg_vec(in, jb, vh));
#pragma unroll
    for (int c = 0; c < 3; ++c) d.c[c] = cmake(d.c[c].re + (f.c[c].re - b.c[c].re), d.c[c].im + (f.c[c].im - b.c[c].im));
  }
  return d;
}

// A group of kFixSites sites by kFixThreads threads: thread t takes direction t / kFixSites of site t % kFixSites
// (the warps' loads stay runs of consecutive sites), the four sums meet in shared memory, and the threads
// of the first three directions hold one colour each.
constexpr int kFixSites = 32, kFixThreads = 4 * kFixSites;

struct FixShared {
  longlong2 part[4][3][kFixSites];
  int2 fwd[4][3][kFixSites];  // upper words of the forward hops' sums (fix_hop_words)
  int word[4][kFixSites];
};

template <bool DIGITS>
struct FixGroup {
  int jf, jb;
  FixRaw<DIGITS> Wf;

  // neighbours, and the forward link's loads: nothing that an earlier kernel of the stream writes
  __device__ __forceinline__ void start(const Geom& g, const FixField& U, int p, int i, int mu, uint64_t pol) {
    const Site s = site_of(g, p, i);
    jf = neighbour_half(g, neighbour_fwd(g, s, mu));
    jb = neighbour_half(g, neighbour_bwd(g, s, mu));
    Wf = load_link_fix<DIGITS>(U, p, mu, i, g.vh, pol);
  }

  // The thread's two hops, left in sh.part.  All threads of the block call; a barrier has to follow.
  __device__ __forceinline__ void hops(FixShared& sh, const Geom& g, const FixField& U, const double2* in, int p, int mu,
                                       int ls, bool valid, uint64_t pol) const {
    const int vh = g.vh;
    Vec3<double> vf, vb;
    FixRaw<DIGITS> Wb;
    if (valid) {
      vf = ldg_vec(in, jf, vh);
      vb = ldg_vec(in, jb, vh);
      Wb = load_link_fix<DIGITS>(U, 1 - p, mu, jb, vh, pol);
      const double w[12] = {vf.c[0].re, vf.c[0].im, vf.c[1].re, vf.c[1].im, vf.c[2].re, vf.c[2].im,
                            vb.c[0].re, vb.c[0].im, vb.c[1].re, vb.c[1].im, vb.c[2].re, vb.c[2].im};
      sh.word[mu][ls] = fix_max_word(w);
    }
    __syncthreads();
    if (!valid) return;
    const int E = exponent(sh, ls);
    FixAcc s;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s.rh[c] = s.ih[c] = 0;
      s.rx[c] = s.ix[c] = 1 << (kFixLow - 1);  // rounds the shift below
    }
    const FixLink Lf = fix_digits(Wf);
    fix_hop<true>(s, Lf, vf, E);
#pragma unroll
    for (int c = 0; c < 3; ++c) sh.fwd[mu][c][ls] = make_int2(fix_upper(s.rh[c]), fix_upper(s.ih[c]));
    const FixLink Lb = fix_digits(Wb);
    fix_hop<false>(s, Lb, vb, E);
    const bool bad = Lf.e[0].x == kFixBadLink || Lb.e[0].x == kFixBadLink;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      sh.part[mu][c][ls] = make_longlong2(bad ? kFixBadSum : s.rh[c] + (s.rx[c] >> kFixLow),
                                          s.ih[c] + (s.ix[c] >> kFixLow));
  }

  // the site's block exponent, or -1 where it is outside the format
  static __device__ __forceinline__ int exponent(const FixShared& sh, int ls) {
    const int w[4] = {sh.word[0][ls], sh.word[1][ls], sh.word[2][ls], sh.word[3][ls]};
    return fix_block_exponent(w);
  }

  // after the barrier: colour c of (D in)(x), c = 0 .. 2
  static __device__ __forceinline__ Cplx<double> colour(const FixShared& sh, const Geom& g, const double2* U64, const double2* in,
                                                        int p, int i, int c, int ls) {
    const int w[4] = {sh.word[0][ls], sh.word[1][ls], sh.word[2][ls], sh.word[3][ls]};
    const int E = fix_block_exponent(w);
    int64_t re = 0, im = 0;
    bool ok = E >= 0;
    uint32_t hr = 0, hi = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const longlong2 u = sh.part[q][c][ls];
      const int2 f = sh.fwd[q][c][ls];
      ok = ok && u.x != kFixBadSum;
      re += u.x;
      im += u.y;
      hr += fix_hop_words(f.x, fix_upper(u.x));
      hi += fix_hop_words(f.y, fix_upper(u.y));
    }
    const bool zero = (w[0] | w[1] | w[2] | w[3]) == 0;  // all neighbours
    const uint32_t need = fix_needed(w, E);
    ok = ok && (zero || (hr >= need && hi >= need));
    if (!ok) {
      const Vec3<double> d = site64_fma(g, U64, in, p, i);
      return c == 0 ? d.c[0] : c == 1 ? d.c[1] : d.c[2];
    }
    const double sc = __hiloint2double((E - kFixUnit + 1023) << 20, 0);  // 2^(E - kFixUnit): a normal number
    return cmake((double)(long long)re * sc, (double)(long long)im * sc);
  }
};

}  // namespace lqcd

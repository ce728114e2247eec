// fix64.cuh - the FP64 half Dslash of a group of sites in block fixed point (fixpoint.h).
//
// Measured on GB300, half Dslash per graph launch (caches as the previous launches leave them), with FP64
// multiply-adds and one thread per site before:
//     8^4 12.0 -> 3.2 us, 16^3x8 12.8 -> 6.8, 24^3x6 30.8 -> 13.2, 32^3x8 69.8 -> 35.4, 48^3x12 329 -> 166
// (32^3x8: 163.6 MB, 24 us at the measured HBM rate).  It runs 17.4 M warp instructions there, 45 % of them
// on the ALU (digits, addresses) and 39 % on the integer multiplier: issue and load latency share the bound.
// One direction (two hops) per thread, 3 blocks of 128 threads per SM (168 registers; up to 24 bytes spilled, 132 in the
// kernels without digits): 4 blocks (128 registers) take 39 us, one hop per thread 36.5 us, one thread per site 68.6 us.
// Links outside the format throughout (SU(3) times 1.2), computed in FP64 after a look at the digits: 32^3x8 260 -> 110 us,
// 16^3x8 48 -> 20, since each of a site's three threads computes its own colour only and skips the integer products; 80 us
// of that is the FP64 pipe (336 multiply-adds per site at 2 per clock and SM).  Deciding it at the first barrier, with
// all four threads of a site sharing the work, takes 89 us, but costs ordinary links 2 us.
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
// are read: the same digits, so the same results.  Behind the copies, which begin with the FP64 one, lies one byte per link,
// [2][4][Vh]: whether it is within the format.
struct FixField {
  const int4* digits;
  const double2* u64;
};
// bytes of the copies per half-lattice site: FP64, FP32 and its rounding errors, 12-real, 8-real, 16-bit (each a multiple
// of 256 bytes, Vh being one of 8)
constexpr size_t kCopyBytes = 8 * (144 + 72 + 72 + 48 + 32 + 24);
__host__ __device__ __forceinline__ const unsigned char* fix_fits(const double2* u64, int vh) {
  return reinterpret_cast<const unsigned char*>(u64) + kCopyBytes * (size_t)vh;
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

// In FP64, for what the format does not take: colour c of hop h of site i (h: direction h / 2, forward or backward), a chain
// of multiply-adds that reads the row (column) of the link it needs.  The colour is the sum over the directions, in order, of
// forward minus backward.
static __device__ __forceinline__ Cplx<double> hop64(const Geom& g, const Site& s, const double2* U, const double2* in, int p,
                                                      int i, int c, int h) {
  const int vh = g.vh, mu = h >> 1;
  const bool fwd = (h & 1) == 0;
  const int j = neighbour_half(g, fwd ? neighbour_fwd(g, s, mu) : neighbour_bwd(g, s, mu));
  const double2* u = U + ((size_t)((fwd ? p : 1 - p) * 4 + mu) * 9 + (fwd ? 3 * c : c)) * vh + (fwd ? i : j);
  const size_t step = (size_t)(fwd ? 1 : 3) * vh;
  const uint64_t pol = policy_evict_first();
  Cplx<double> d = cmake(0.0, 0.0);
  double2 l[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) l[b] = ld_stream(u + b * step, pol);
  const Vec3<double> v = ldg_vec(in, j, vh);
#pragma unroll
  for (int b = 0; b < 3; ++b) cmac(d, cmake(l[b].x, fwd ? l[b].y : -l[b].y), v.c[b]);
  return d;
}

// Colour c of site i for the lanes with want.  All lanes of the warp call.  A few sites (rough fields: one in 300 000): eight
// lanes take a site's hops side by side; more: each lane its own site.  The same operations, the same bits.
static __device__ __noinline__ Cplx<double> site64_fma(Geom g, const double2* __restrict__ U, const double2* __restrict__ in,
                                                        int p, int i, int c, bool want) {
  Cplx<double> d = cmake(0.0, 0.0);
  unsigned todo = __ballot_sync(0xffffffffu, want);
  const int lane = threadIdx.x & 31;
  if (__popc(todo) > 4) {
    if (want) {
      const Site s = site_of(g, p, i);
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        const Cplx<double> f = hop64(g, s, U, in, p, i, c, 2 * mu), b = hop64(g, s, U, in, p, i, c, 2 * mu + 1);
        d = cmake(d.re + (f.re - b.re), d.im + (f.im - b.im));
      }
    }
    return d;
  }
  for (; todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1, is = __shfl_sync(0xffffffffu, i, src);
    Cplx<double> t = cmake(0.0, 0.0), r = t;
    if (lane < 8) t = hop64(g, site_of(g, p, is), U, in, p, is, c, lane);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const double fr = __shfl_sync(0xffffffffu, t.re, 2 * mu), fi = __shfl_sync(0xffffffffu, t.im, 2 * mu);
      const double br = __shfl_sync(0xffffffffu, t.re, 2 * mu + 1), bi = __shfl_sync(0xffffffffu, t.im, 2 * mu + 1);
      r = cmake(r.re + (fr - br), r.im + (fi - bi));
    }
    if (lane == src) d = r;
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
    if (Lf.e[0].x != kFixBadLink) fix_hop<true>(s, Lf, vf, E);
#pragma unroll
    for (int c = 0; c < 3; ++c) sh.fwd[mu][c][ls] = make_int2(fix_upper(s.rh[c]), fix_upper(s.ih[c]));
    const FixLink Lb = fix_digits(Wb);
    if (Lb.e[0].x != kFixBadLink) fix_hop<false>(s, Lb, vb, E);
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

  // after the barrier: colour c of (D in)(x), c = 0 .. 2.  All lanes of the warp call, with valid for those that have a site.
  static __device__ __forceinline__ Cplx<double> colour(const FixShared& sh, const Geom& g, const double2* U64, const double2* in,
                                                        int p, int i, int c, int ls, bool valid) {
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
    if (__any_sync(0xffffffffu, valid && !ok)) {
      const Cplx<double> d = site64_fma(g, U64, in, p, i, c, valid && !ok);
      if (!ok) return d;
    }
    const double sc = __hiloint2double((E - kFixUnit + 1023) << 20, 0);  // 2^(E - kFixUnit): a normal number
    return cmake((double)(long long)re * sc, (double)(long long)im * sc);
  }
};

}  // namespace lqcd

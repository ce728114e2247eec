// trajectory.cu - one RHMC trajectory for two staggered flavours (Section 3.1):
//   phi = r_{1/4}(A) xi (heatbath, Eq. ratapprx with b = 4), H = 1/2 p^2 + S_g + phi^+ r_{-1/2}(A) phi,
//   molecular dynamics dU/dt = i P U, dp^a/dt = -dS/dw^a with Omelyan's 2MN integrator,
//   Metropolis accept with probability min(1, exp(-dH)).
// Gauge action S_g = beta sum_{x, mu<nu} (1 - Re tr U_plaq / 3); its force per link is
//   F = -(i beta / 12) (W - W^+) (traceless), W = U_mu(x) A_mu(x), A = sum of the six staples.
// The fermion force comes from fermion_force (force.cu).  Momenta, the Gaussian xi and the
// Metropolis uniform are inputs; everything else runs on the GPU (FP64 for links, momenta,
// actions and dH; the shifted CG in the requested precision).
#include <math.h>
#include <string.h>

#include <chrono>
#include <type_traits>

#include "common.cuh"
#include "fix64.cuh"
#include "internal.h"

namespace lqcd {

struct TrajWorkspace {
  double2* U = nullptr;     // canonical [V][4][9] complex128, the evolving links
  double* P = nullptr;      // [V][4][8] momentum components
  double* F = nullptr;      // [V][4][8] force components
  double2* phi = nullptr;   // canonical even vector
  double* partials = nullptr;
  unsigned* ticket = nullptr;
  double* scal = nullptr;   // reduction results
};

static void traj_free(TrajWorkspace* tw) {
  if (!tw) return;
  void* b[] = {tw->U, tw->P, tw->F, tw->phi, tw->partials, tw->ticket, tw->scal};
  for (void* p : b)
    if (p) cudaFree(p);
  delete tw;
}

void traj_release(lqcd_ctx* ctx) {
  traj_free(static_cast<TrajWorkspace*>(ctx->traj_ws));
  ctx->traj_ws = nullptr;
}

// ---------------------------------------------------------------------------------------------
// 3x3 complex helpers on canonical FP64 links (row-major double2[9])
// ---------------------------------------------------------------------------------------------
struct M3 {
  double2 e[9];
};

__device__ __forceinline__ M3 ldm(const double2* p) {
  M3 m;
#pragma unroll
  for (int i = 0; i < 9; ++i) m.e[i] = p[i];
  return m;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// s + a b as four multiply-adds (GB300's FP64 pipe runs 2 per clock and SM: every operation saved counts)
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 s) {
  return make_double2(fma(-a.y, b.y, fma(a.x, b.x, s.x)), fma(a.y, b.x, fma(a.x, b.y, s.y)));
}

__device__ __forceinline__ M3 mm(const M3& a, const M3& b) {  // a b
  M3 c;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      double2 s = cmul(a.e[r * 3], b.e[q]);
      s = cfma(a.e[r * 3 + 1], b.e[3 + q], s);
      c.e[r * 3 + q] = cfma(a.e[r * 3 + 2], b.e[6 + q], s);
    }
  return c;
}

__device__ __forceinline__ M3 dagger(const M3& a) {
  M3 c;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int q = 0; q < 3; ++q) c.e[r * 3 + q] = make_double2(a.e[q * 3 + r].x, -a.e[q * 3 + r].y);
  return c;
}

__device__ __forceinline__ void add_to(M3& a, const M3& b) {
#pragma unroll
  for (int i = 0; i < 9; ++i) a.e[i] = cadd(a.e[i], b.e[i]);
}

__device__ __forceinline__ Site site_at(const Geom& g, int l) {
  Site s;
  unsigned ul = (unsigned)l;
  unsigned r = fdiv(ul, g.dnx);
  s.x = (int)(ul - r * (unsigned)g.nx);
  unsigned r2 = fdiv(r, g.dny);
  s.y = (int)(r - r2 * (unsigned)g.ny);
  unsigned r3 = fdiv(r2, g.dnz);
  s.z = (int)(r2 - r3 * (unsigned)g.nz);
  s.t = (int)r3;
  s.l = l;
  return s;
}

// S_g partial sums: per site, sum over the six planes of (1 - Re tr P_{mu nu}(x) / 3)
__global__ void __launch_bounds__(128) plaquette_kernel(Geom g, const double2* __restrict__ U, double* partials,
                                                        unsigned* ticket, double* out) {
  const int V = 2 * g.vh;
  int l = blockIdx.x * blockDim.x + threadIdx.x;
  double loc = 0.0;
  if (l < V) {
    Site s = site_at(g, l);
    for (int mu = 0; mu < 4; ++mu) {
      int xm = neighbour_addr(g, neighbour_fwd(g, s, mu));
      M3 Um = ldm(U + ((size_t)l * 4 + mu) * 9);
      for (int nu = mu + 1; nu < 4; ++nu) {
        int xn = neighbour_addr(g, neighbour_fwd(g, s, nu));
        M3 a = mm(Um, ldm(U + ((size_t)xm * 4 + nu) * 9));
        M3 b = mm(ldm(U + ((size_t)l * 4 + nu) * 9), ldm(U + ((size_t)xn * 4 + mu) * 9));
        // Re tr(a b^+) = sum_ij Re(a_ij conj(b_ij))
        double tr = 0.0;
#pragma unroll
        for (int i = 0; i < 9; ++i) tr += a.e[i].x * b.e[i].x + a.e[i].y * b.e[i].y;
        loc += 1.0 - tr / 3.0;
      }
    }
  }
  double bs = block_sum(loc);
  if (publish_partial(partials, ticket, bs)) {
    double tot = gather_partials(partials, ticket);
    if (threadIdx.x == 0) *out = tot;
  }
}

// W = U_mu(x) A_mu(x), A the sum of the six staples, from the canonical links in FP64.
static __device__ __noinline__ M3 link_times_staples(Geom g, const double2* __restrict__ U, Site s, int mu) {
  const int l = s.l;
  const int xpmu = neighbour_addr(g, neighbour_fwd(g, s, mu));
  Site sp = site_at(g, xpmu);
  M3 A;
#pragma unroll
  for (int i = 0; i < 9; ++i) A.e[i] = make_double2(0, 0);
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    const int xpnu = neighbour_addr(g, neighbour_fwd(g, s, nu));
    const int xmnu = neighbour_addr(g, neighbour_bwd(g, s, nu));
    const int xpmu_mnu = neighbour_addr(g, neighbour_bwd(g, sp, nu));
    // up = U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+ ; down = U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu)
    M3 up = mm(mm(ldm(U + ((size_t)xpmu * 4 + nu) * 9), dagger(ldm(U + ((size_t)xpnu * 4 + mu) * 9))),
               dagger(ldm(U + ((size_t)l * 4 + nu) * 9)));
    M3 dn = mm(mm(dagger(ldm(U + ((size_t)xpmu_mnu * 4 + nu) * 9)), dagger(ldm(U + ((size_t)xmnu * 4 + mu) * 9))),
               ldm(U + ((size_t)xmnu * 4 + nu) * 9));
    add_to(A, up);
    add_to(A, dn);
  }
  return mm(ldm(U + ((size_t)l * 4 + mu) * 9), A);
}

// The same products in fixed point (fixpoint.h), from the digits of 1/2 eta bc U.  A matrix is (re.h, re.l,
// im.h, im.l) per entry, F = H 2^28 + L (links: H and L of one sign; split products: 0 <= L < 2^28); a product's
// entries are 64-bit sums in units of 2^56 of the product of the factors' units, whose digits (fix_split) are the
// next product's factor:
//   folded links in units of 2^-57, entries <= 1/2;   U U in 2^-58, <= 1/4;   U U U in 2^-59, <= 0.22;
//   the six staples' sum, divided by 4, in 2^-57, <= 0.33;   U A in 2^-58, <= 1.6.
// The H H sums stay below 6 2^28 2^29.4, the H L sums below 6 (2^28 2^28 + 2^28 2^29.4).
//
// Accuracy, with u = 2^-58 and rows and columns of norm up to kFixMaxNorm, so that the six components of a row add up to
// 1.23 at most.  Links are rounded by u.  A product of links errs by 2 x 1.23 u from that, 6 u from the L L products and
// u/2 from rounding: 9 u; times a link: 9 x 1.23 + 1.1 + 3 + 0.25 = 15.3 u; the six staples' sum: 93 u; times the link:
// 93 x 1.23 + 5.6 + 6.5 = 126 u.  W is 16 times that: 63 x 2^-53, whatever the size of the component.  The FP64 products
// err by at most 24 x 2^-53 S (three products of 6 roundings each and six sums), S the sum of the magnitudes of all products of
// links that make up the component.  So the digits' W is taken where S > 63 / 24, S bounded from below by |U| sum |UU| |U|
// in FP32 (staple_magnitude), for each combination of components that the force is made of; a link short of that is
// computed in FP64 (fields close to one, whose off-diagonal and imaginary parts are small).
struct FixSum3 {
  int64_t re[9], im[9];
};

// op(A) op(B), op the adjoint where AD, BD
template <bool AD, bool BD>
__device__ __forceinline__ FixSum3 fix_mm(const FixLink& A, const FixLink& B) {
  FixSum3 o;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      // re = sum ar br - (+-) ai bi: the imaginary products go to accumulators of their own, so that the signs
      // of the adjoints cost nothing
      int64_t h1 = 0, x1 = 0, h2 = 0, x2 = 0, h3 = 0, x3 = 0, h4 = 0, x4 = 0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int4 a = A.e[AD ? 3 * k + r : 3 * r + k], b = B.e[BD ? 3 * q + k : 3 * k + q];
        fix_mac(h1, x1, a.x, a.y, Fix2{b.x, b.y});
        fix_mac(h2, x2, a.z, a.w, Fix2{b.z, b.w});
        fix_mac(h3, x3, a.x, a.y, Fix2{b.z, b.w});
        fix_mac(h4, x4, a.z, a.w, Fix2{b.x, b.y});
      }
      const int64_t half = 1 << (kFixLow - 1);
      // (ar +- i ai)(br +- i bi): re = ar br - s ai bi with s = -1 where one factor is conjugated
      const int64_t rh = AD != BD ? h1 + h2 : h1 - h2, rx = AD != BD ? x1 + x2 : x1 - x2;
      const int64_t ih = (BD ? -h3 : h3) + (AD ? -h4 : h4), ix = (BD ? -x3 : x3) + (AD ? -x4 : x4);
      o.re[3 * r + q] = rh + ((rx + half) >> kFixLow);
      o.im[3 * r + q] = ih + ((ix + half) >> kFixLow);
    }
  }
  return o;
}

__device__ __forceinline__ FixLink fix_split(const FixSum3& s, int shift) {  // digits of s / 2^shift
  FixLink o;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const int64_t re = s.re[j] >> shift, im = s.im[j] >> shift;
    o.e[j] = make_int4((int)(re >> kFixLow), (int)re & ((1 << kFixLow) - 1), (int)(im >> kFixLow),
                       (int)im & ((1 << kFixLow) - 1));
  }
  return o;
}

// mag += |op(A)| |op(B)| (real and imaginary parts of each entry: the sums of the magnitudes of their products), from the
// high digits: in units of theirs, and below the true magnitudes but for 2^-22 of them.
constexpr int kForceThreads = 128;
typedef float ForceMag[18][kForceThreads];  // [entry, re and im][thread]
template <bool AD, bool BD>
__device__ __forceinline__ void staple_magnitude(ForceMag& mag, const FixLink& A, const FixLink& B) {
  float a[18], b[18];
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    a[2 * j] = fabsf((float)A.e[j].x);
    a[2 * j + 1] = fabsf((float)A.e[j].z);
    b[2 * j] = fabsf((float)B.e[j].x);
    b[2 * j + 1] = fabsf((float)B.e[j].z);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int ja = 2 * (AD ? 3 * k + r : 3 * r + k), jb = 2 * (BD ? 3 * q + k : 3 * k + q);
        re = fmaf(a[ja], b[jb], fmaf(a[ja + 1], b[jb + 1], re));
        im = fmaf(a[ja], b[jb + 1], fmaf(a[ja + 1], b[jb], im));
      }
      mag[2 * (3 * r + q)][threadIdx.x] += re;
      mag[2 * (3 * r + q) + 1][threadIdx.x] += im;
    }
}

// Whether |U| mag is large enough for the digits' W, for the combinations that the force takes: W_rc - conj(W_cr), the
// differences of the diagonal's imaginary parts.
__device__ __forceinline__ bool force_accurate(const FixLink& U, const ForceMag& mag) {
  float u[18];
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    u[2 * j] = fabsf((float)U.e[j].x);
    u[2 * j + 1] = fabsf((float)U.e[j].z);
  }
  auto S = [&](int r, int c, bool imag) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int ju = 2 * (3 * r + k), jm = 2 * (3 * k + c);
      s = fmaf(u[ju], mag[jm + imag][threadIdx.x], fmaf(u[ju + 1], mag[jm + !imag][threadIdx.x], s));
    }
    return s;
  };
  // magnitudes in units of 2^-29 (link) 2^-30 (U U) 2^-29 (link) of W / 16
  constexpr float need = 2.7f * 0x1p84f;  // 63 / 24 and what the high digits and FP32 leave out
  bool ok = true;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = r + 1; c < 3; ++c)
      ok = ok && S(r, c, false) + S(c, r, false) >= 2 * need && S(r, c, true) + S(c, r, true) >= 2 * need;
  const float d0 = S(0, 0, true), d1 = S(1, 1, true), d2 = S(2, 2, true);
  return ok && d0 + d1 >= 2 * need && d0 + d1 + 2 * d2 >= 4 * need;
}

// F[l][mu][a] += beta-scaled gauge force components tr(lambda^a F_g); block: 32 sites of one parity, one direction
// per warp.  The 13 matrix products of a link in FP64 take 1404 multiply-adds, 702 clocks of the SM's FP64 pipe; in
// fixed point 4212 integer ones, 66 clocks, and about as much again for digits and addresses: 24^3 x 6 (331 776
// links) 1865 -> 335 us, 16 of them for the check (434 without digits).  Links outside the format: FP64.  DIGITS: whether the field keeps its digits (FixField).
template <bool DIGITS>
__global__ void __launch_bounds__(kForceThreads, 2) gauge_force_kernel(Geom g, const double2* __restrict__ U, FixField Ufix,
                                                                       double beta, double* __restrict__ F) {
  __shared__ ForceMag mag;  // each thread's own column
  const int vh = g.vh;
  const int nb = (vh + 31) / 32;
  const int p = (int)blockIdx.x >= nb ? 1 : 0;
  const int i = ((int)blockIdx.x - p * nb) * 32 + (threadIdx.x & 31), mu = threadIdx.x >> 5;
  if (i >= vh) return;
  const Site s = site_of(g, p, i);
  double Wre[9], Wim[9];
  bool ok = true;
  {
    const uint64_t pol = policy_evict_last();  // every link is read by the 18 staples it is in
    const int xpmu = neighbour_addr(g, neighbour_fwd(g, s, mu));
    const Site sp = site_at(g, xpmu);
    auto link = [&](int parity, int dir, int l) {
      const FixLink L = fix_digits(load_link_fix<DIGITS>(Ufix, parity, dir, l >> 1, vh, pol));
      ok = ok && L.e[0].x != kFixBadLink;
      return L;
    };
    FixSum3 A;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      A.re[j] = A.im[j] = 2;  // rounds the division by 4 below
      mag[2 * j][threadIdx.x] = mag[2 * j + 1][threadIdx.x] = 0.f;
    }
#pragma unroll 1
    for (int m = 1; m < 4; ++m) {
      const int nu = (mu + m) & 3;
      const int xpnu = neighbour_addr(g, neighbour_fwd(g, s, nu));
      const int xmnu = neighbour_addr(g, neighbour_bwd(g, s, nu));
      const int xpmu_mnu = neighbour_addr(g, neighbour_bwd(g, sp, nu));
      const FixLink up2 = fix_split(fix_mm<false, true>(link(1 - p, nu, xpmu), link(1 - p, mu, xpnu)), 0);
      const FixLink un = link(p, nu, s.l);
      const FixSum3 up = fix_mm<false, true>(up2, un);
      staple_magnitude<false, true>(mag, up2, un);
      // (U_mu(x-nu) U_nu(x+mu-nu))^+ U_nu(x-nu)
      const FixLink dn2 = fix_split(fix_mm<false, false>(link(1 - p, mu, xmnu), link(p, nu, xpmu_mnu)), 0);
      const FixLink um = link(1 - p, nu, xmnu);
      const FixSum3 dn = fix_mm<true, false>(dn2, um);
      staple_magnitude<true, false>(mag, dn2, um);
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        A.re[j] += up.re[j] + dn.re[j];
        A.im[j] += up.im[j] + dn.im[j];
      }
    }
    const FixLink ul = link(p, mu, s.l);
    ok = ok && force_accurate(ul, mag);
    const FixSum3 W = fix_mm<false, false>(ul, fix_split(A, 2));
    // the links' factors 1/2 and eta bc: 1/16, and the staggered signs around a plaquette multiply to -1
    const double sc = -16.0 * 0x1p-58;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      Wre[j] = (double)(long long)W.re[j] * sc;
      Wim[j] = (double)(long long)W.im[j] * sc;
    }
  }
  if (!ok) {
    const M3 W = link_times_staples(g, U, s, mu);
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      Wre[j] = W.e[j].x;
      Wim[j] = W.e[j].y;
    }
  }
  // F = -(i beta/12)(W - W^+): F_rc = -(i beta/12)(W_rc - conj(W_cr)) = (beta/12)(dim + ... )
  double Fre[9], Fim[9];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double dre = Wre[r * 3 + c] - Wre[c * 3 + r];
      double dim = Wim[r * 3 + c] + Wim[c * 3 + r];
      // -(i b)(dre + i dim) = b dim - i b dre
      Fre[r * 3 + c] = beta / 12.0 * dim;
      Fim[r * 3 + c] = -beta / 12.0 * dre;
    }
  const double tr3 = (Fre[0] + Fre[4] + Fre[8]) / 3.0;
  Fre[0] -= tr3;
  Fre[4] -= tr3;
  Fre[8] -= tr3;
  double* o = F + ((size_t)s.l * 4 + mu) * 8;
  const double inv_sqrt3 = 0.57735026918962576451;
  o[0] += 2.0 * Fre[1];
  o[1] += -2.0 * Fim[1];
  o[2] += Fre[0] - Fre[4];
  o[3] += 2.0 * Fre[2];
  o[4] += -2.0 * Fim[2];
  o[5] += 2.0 * Fre[5];
  o[6] += -2.0 * Fim[5];
  o[7] += (Fre[0] + Fre[4] - 2.0 * Fre[8]) * inv_sqrt3;
}

// p -= c F (all V*4*8 components)
__global__ void kick_kernel(long long n, double* __restrict__ P, const double* __restrict__ F, double c) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) P[i] -= c * F[i];
}

// U <- exp(i h P) U, P = sum p^a lambda^a / 2, then SU(3) projection (rows 0, 1 Gram-Schmidt, row 2 = conj(r0 x r1)).
// Bound by the FP64 pipe: about 500 operations a link, 262 us at 24^3 x 6 (331 776 links; 17 us of memory traffic). A
// Taylor series of matrix products to order 16, as before, takes 3500 operations and 2276 us.
__global__ void __launch_bounds__(128) link_update_kernel(long long nlinks, double2* __restrict__ U,
                                                          const double* __restrict__ P, double h) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nlinks) return;
  const double* p = P + t * 8;
  const double inv_sqrt3 = 0.57735026918962576451;
  // Q = h P, Hermitian and traceless: diagonal qd, off-diagonal q01, q02, q12 (q_cr = conj(q_rc))
  double qd[3] = {0.5 * h * (p[2] + p[7] * inv_sqrt3), 0.5 * h * (-p[2] + p[7] * inv_sqrt3), -h * p[7] * inv_sqrt3};
  double2 q01 = make_double2(0.5 * h * p[0], -0.5 * h * p[1]);
  double2 q02 = make_double2(0.5 * h * p[3], -0.5 * h * p[4]);
  double2 q12 = make_double2(0.5 * h * p[5], -0.5 * h * p[6]);
  double n01 = q01.x * q01.x + q01.y * q01.y, n02 = q02.x * q02.x + q02.y * q02.y, n12 = q12.x * q12.x + q12.y * q12.y;
  // scaling and squaring: |Q / 2^k|_F <= 1/4
  double nrm = sqrt(qd[0] * qd[0] + qd[1] * qd[1] + qd[2] * qd[2] + 2.0 * (n01 + n02 + n12));
  int k = 0;
  while (nrm > 0.25 && k < 30) {
    nrm *= 0.5;
    ++k;
  }
  if (k > 0) {
    const double sc = ldexp(1.0, -k), sc2 = sc * sc;
    for (int c = 0; c < 3; ++c) qd[c] *= sc;
    q01 = make_double2(q01.x * sc, q01.y * sc);
    q02 = make_double2(q02.x * sc, q02.y * sc);
    q12 = make_double2(q12.x * sc, q12.y * sc);
    n01 *= sc2;
    n02 *= sc2;
    n12 *= sc2;
  }
  // S = Q^2: diagonal s, off-diagonal s01 = (qd0 + qd1) q01 + q02 conj(q12), ...
  const double s0 = qd[0] * qd[0] + n01 + n02, s1 = qd[1] * qd[1] + n01 + n12, s2 = qd[2] * qd[2] + n02 + n12;
  const double2 s01 = cfma(q02, make_double2(q12.x, -q12.y), make_double2((qd[0] + qd[1]) * q01.x, (qd[0] + qd[1]) * q01.y));
  const double2 s02 = cfma(q01, q12, make_double2((qd[0] + qd[2]) * q02.x, (qd[0] + qd[2]) * q02.y));
  const double2 s12 = cfma(make_double2(q01.x, -q01.y), q02, make_double2((qd[1] + qd[2]) * q12.x, (qd[1] + qd[2]) * q12.y));
  // The Taylor series in the basis 1, Q, Q^2: by the Cayley-Hamilton theorem Q^3 = c1 Q + c0 with c1 = tr Q^2 / 2,
  // c0 = det Q, so Q^n / n! = A + B Q + D Q^2 with real coefficients that follow from those of n - 1; exp(i Q) takes
  // them with i^n.  Order 13: |Q|^14 / 14! < 2^-64 for |Q| <= 1/4.
  const double c1 = 0.5 * (s0 + s1 + s2);
  const double2 q0112 = cmul(q01, q12);  // c0 = qd0 qd1 qd2 + 2 Re(q01 q12 conj(q02)) - qd0 n12 - qd1 n02 - qd2 n01
  const double c0 = qd[0] * (qd[1] * qd[2] - n12) - qd[1] * n02 - qd[2] * n01 + 2.0 * (q0112.x * q02.x + q0112.y * q02.y);
  double A = 0.0, B = 1.0, D = 0.0;                                       // n = 1
  double f0[2] = {1.0, 0.0}, f1[2] = {0.0, 1.0}, f2[2] = {0.0, 0.0};  // real, imaginary: n = 0 and 1
#pragma unroll
  for (int n = 2; n <= 13; ++n) {
    const double inv = 1.0 / n, Dn = D * inv;
    const double An = c0 * Dn, Bn = fma(A, inv, c1 * Dn);
    D = B * inv;
    A = An;
    B = Bn;
    if (n & 2) {  // i^n = -1, -i
      f0[n & 1] -= A;
      f1[n & 1] -= B;
      f2[n & 1] -= D;
    } else {
      f0[n & 1] += A;
      f1[n & 1] += B;
      f2[n & 1] += D;
    }
  }
  M3 E;
  const double2 g1 = make_double2(f1[0], f1[1]), g2 = make_double2(f2[0], f2[1]);
  auto diag = [&](double q, double s) { return make_double2(f0[0] + g1.x * q + g2.x * s, f0[1] + g1.y * q + g2.y * s); };
  auto conj2 = [](double2 z) { return make_double2(z.x, -z.y); };
  E.e[0] = diag(qd[0], s0);
  E.e[4] = diag(qd[1], s1);
  E.e[8] = diag(qd[2], s2);
  E.e[1] = cfma(g1, q01, cmul(g2, s01));
  E.e[3] = cfma(g1, conj2(q01), cmul(g2, conj2(s01)));
  E.e[2] = cfma(g1, q02, cmul(g2, s02));
  E.e[6] = cfma(g1, conj2(q02), cmul(g2, conj2(s02)));
  E.e[5] = cfma(g1, q12, cmul(g2, s12));
  E.e[7] = cfma(g1, conj2(q12), cmul(g2, conj2(s12)));
  for (int i = 0; i < k; ++i) E = mm(E, E);
  M3 Un = mm(E, ldm(U + t * 9));
  // SU(3) projection
  double2 r0[3] = {Un.e[0], Un.e[1], Un.e[2]}, r1[3] = {Un.e[3], Un.e[4], Un.e[5]};
  double n0 = 0.0;
  for (int c = 0; c < 3; ++c) n0 += r0[c].x * r0[c].x + r0[c].y * r0[c].y;
  n0 = 1.0 / sqrt(n0);
  for (int c = 0; c < 3; ++c) r0[c] = make_double2(r0[c].x * n0, r0[c].y * n0);
  double2 d = make_double2(0, 0);  // <r0, r1> = sum conj(r0) r1
  for (int c = 0; c < 3; ++c) d = cadd(d, cmul(make_double2(r0[c].x, -r0[c].y), r1[c]));
  for (int c = 0; c < 3; ++c) {
    double2 pr = cmul(d, r0[c]);
    r1[c] = make_double2(r1[c].x - pr.x, r1[c].y - pr.y);
  }
  double n1 = 0.0;
  for (int c = 0; c < 3; ++c) n1 += r1[c].x * r1[c].x + r1[c].y * r1[c].y;
  n1 = 1.0 / sqrt(n1);
  for (int c = 0; c < 3; ++c) r1[c] = make_double2(r1[c].x * n1, r1[c].y * n1);
  double2* out = U + t * 9;
  for (int c = 0; c < 3; ++c) {
    out[c] = r0[c];
    out[3 + c] = r1[c];
    // row 2 = conj(r0 x r1)
    double2 cr = cadd(cmul(r0[(c + 1) % 3], r1[(c + 2) % 3]),
                      make_double2(-cmul(r0[(c + 2) % 3], r1[(c + 1) % 3]).x, -cmul(r0[(c + 2) % 3], r1[(c + 1) % 3]).y));
    out[6 + c] = make_double2(cr.x, -cr.y);
  }
}

// 1/2 sum p^2
__global__ void __launch_bounds__(256) kinetic_kernel(long long n, const double* __restrict__ P, double* partials,
                                                      unsigned* ticket, double* out) {
  double loc = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    loc += 0.5 * P[i] * P[i];
  double bs = block_sum(loc);
  if (publish_partial(partials, ticket, bs)) {
    double tot = gather_partials(partials, ticket);
    if (threadIdx.x == 0) *out = tot;
  }
}

}  // namespace lqcd

using namespace lqcd;

#define TJ_CUDA(call)                                           \
  do {                                                          \
    cudaError_t _e = (call);                                    \
    if (_e != cudaSuccess) return cuda_check(ctx, _e, #call);   \
  } while (0)

static int traj_scalar(lqcd_ctx* ctx, TrajWorkspace* tw, int which, cudaStream_t st, double* out) {
  TJ_CUDA(cudaMemcpyAsync(out, tw->scal + which, sizeof(double), cudaMemcpyDeviceToHost, st));
  TJ_CUDA(cudaStreamSynchronize(st));
  return LQCD_OK;
}

extern "C" int rhmc_trajectory(lqcd_ctx* ctx, const lqcd_rhmc_params* prm, double* U_dev, const double* mom_dev,
                               const double* xi_dev, double uniform, lqcd_traj_result* res) {
  if (!ctx) return LQCD_ERR_ARG;
  if (!prm || !U_dev || !mom_dev || !xi_dev || !res || prm->nsteps < 1 || !(prm->tau > 0.0) || prm->n_act < 1 ||
      !prm->act_shifts || !prm->act_residues ||
      (!prm->phi_given && (prm->n_heat < 1 || !prm->heat_shifts || !prm->heat_residues)))
    return fail(ctx, LQCD_ERR_ARG, "rhmc_trajectory: bad argument");
  auto t0 = std::chrono::steady_clock::now();
  memset(res, 0, sizeof(*res));
  Geom g = make_geom(ctx);
  const long long V = ctx->V;
  const long long ncomp = V * 4 * 8;
  cudaStream_t st = ctx->stream;
  TrajWorkspace* tw = static_cast<TrajWorkspace*>(ctx->traj_ws);
  if (!tw) {
    tw = new TrajWorkspace();
    ctx->traj_ws = tw;
    TJ_CUDA(cudaMalloc(&tw->U, sizeof(double2) * 9 * 4 * V));
    TJ_CUDA(cudaMalloc(&tw->P, sizeof(double) * ncomp));
    TJ_CUDA(cudaMalloc(&tw->F, sizeof(double) * ncomp));
    TJ_CUDA(cudaMalloc(&tw->phi, sizeof(double2) * 3 * ctx->Vh));
    TJ_CUDA(cudaMalloc(&tw->partials, sizeof(double) * (4 * V / 128 + 1024)));
    TJ_CUDA(cudaMalloc(&tw->ticket, sizeof(unsigned)));
    TJ_CUDA(cudaMemsetAsync(tw->ticket, 0, sizeof(unsigned), st));
    TJ_CUDA(cudaMalloc(&tw->scal, sizeof(double) * 8));
  }
  const double lam = prm->lambda > 0.0 ? prm->lambda : 0.1931833275037836;
  const double md_tol = prm->md_tol > 0.0 ? prm->md_tol : prm->tol;
  int rc;
  long long nl = 0;
  lqcd_solve_stats sst;
  auto count = [&](const lqcd_solve_stats& s) {
    res->solves += 1;
    res->iterations += s.iterations + s.refine_iterations;
  };
  // working copy of the links and momenta
  TJ_CUDA(cudaMemcpyAsync(tw->U, U_dev, sizeof(double2) * 9 * 4 * V, cudaMemcpyDeviceToDevice, st));
  TJ_CUDA(cudaMemcpyAsync(tw->P, mom_dev, sizeof(double) * ncomp, cudaMemcpyDeviceToDevice, st));
  if ((rc = lqcd_set_gauge(ctx, reinterpret_cast<const double*>(tw->U))) != LQCD_OK) return rc;
  if (prm->phi_given) {
    TJ_CUDA(cudaMemcpyAsync(tw->phi, xi_dev, sizeof(double2) * 3 * ctx->Vh, cudaMemcpyDeviceToDevice, st));
  } else {
    // heatbath: phi = r_{1/4}(A) xi
    rc = mshift_cg(ctx, prm->heat_shifts, prm->heat_residues, prm->n_heat, prm->heat_c0, xi_dev, nullptr,
                   reinterpret_cast<double*>(tw->phi), prm->tol, prm->maxiter, prm->prec_action, &sst);
    if (rc != LQCD_OK) return rc;
    count(sst);
  }
  const unsigned nbv = (unsigned)((V + 127) / 128);
  const unsigned nbl = (unsigned)((4 * V + 127) / 128);
  const unsigned nbc = (unsigned)((ncomp + 255) / 256);
  auto hamiltonian = [&](double* kin, double* sg, double* sf) -> int {
    kinetic_kernel<<<256, 256, 0, st>>>(ncomp, tw->P, tw->partials, tw->ticket, tw->scal + 0);
    plaquette_kernel<<<nbv, 128, 0, st>>>(g, tw->U, tw->partials, tw->ticket, tw->scal + 1);
    nl += 2;
    TJ_CUDA(cudaGetLastError());
    int r = traj_scalar(ctx, tw, 0, st, kin);
    if (r != LQCD_OK) return r;
    if ((r = traj_scalar(ctx, tw, 1, st, sg)) != LQCD_OK) return r;
    *sg *= prm->beta;
    r = fermion_force(ctx, prm->act_shifts, prm->act_residues, prm->n_act, prm->act_c0,
                      reinterpret_cast<const double*>(tw->phi), nullptr, nullptr, sf, prm->tol, prm->maxiter,
                      prm->prec_action, &sst);
    if (r != LQCD_OK) return r;
    count(sst);
    return LQCD_OK;
  };
  auto total_force = [&]() -> int {
    int r = fermion_force(ctx, prm->act_shifts, prm->act_residues, prm->n_act, prm->act_c0,
                          reinterpret_cast<const double*>(tw->phi), nullptr, tw->F, nullptr, md_tol, prm->maxiter,
                          prm->prec, &sst);
    if (r != LQCD_OK) return r;
    count(sst);
    const FixField links{ctx->gauge.ufix, ctx->gauge.u64};
    const unsigned nbf = 2 * ((g.vh + 31) / 32);
    if (links.digits) gauge_force_kernel<true><<<nbf, kForceThreads, 0, st>>>(g, tw->U, links, prm->beta, tw->F);
    else gauge_force_kernel<false><<<nbf, kForceThreads, 0, st>>>(g, tw->U, links, prm->beta, tw->F);
    nl += 1;
    TJ_CUDA(cudaGetLastError());
    return LQCD_OK;
  };
  auto kick = [&](double c) -> int {
    kick_kernel<<<nbc, 256, 0, st>>>(ncomp, tw->P, tw->F, c);
    nl += 1;
    TJ_CUDA(cudaGetLastError());
    return LQCD_OK;
  };
  struct Links {  // every copy of the context's field is that of tw->U again on each way out
    lqcd_ctx* ctx;
    const double2* U;
    bool stale;
    int finish() {
      if (!stale) return LQCD_OK;
      stale = false;
      return set_gauge(ctx, reinterpret_cast<const double*>(U), true);
    }
    ~Links() { finish(); }
  } links{ctx, tw->U, false};
  auto drift = [&](double h) -> int {
    link_update_kernel<<<nbl, 128, 0, st>>>(4 * V, tw->U, tw->P, h);
    nl += 1;
    TJ_CUDA(cudaGetLastError());
    // the compact copies that the trajectory's solves do not read follow at its end
    const bool all = prm->prec == LQCD_FP32_R8 || prm->prec == LQCD_FP32_L16 || prm->prec_action == LQCD_FP32_R8 ||
                     prm->prec_action == LQCD_FP32_L16;
    links.stale = !all;
    return set_gauge(ctx, reinterpret_cast<const double*>(tw->U), all);
  };
  if ((rc = hamiltonian(&res->kinetic0, &res->gauge0, &res->fermion0)) != LQCD_OK) return rc;
  // Omelyan 2MN
  const double eps = prm->tau / prm->nsteps;
  if ((rc = total_force()) != LQCD_OK) return rc;
  if ((rc = kick(lam * eps)) != LQCD_OK) return rc;
  for (int step = 0; step < prm->nsteps; ++step) {
    if ((rc = drift(0.5 * eps)) != LQCD_OK) return rc;
    if ((rc = total_force()) != LQCD_OK) return rc;
    if ((rc = kick((1.0 - 2.0 * lam) * eps)) != LQCD_OK) return rc;
    if ((rc = drift(0.5 * eps)) != LQCD_OK) return rc;
    if ((rc = total_force()) != LQCD_OK) return rc;
    if ((rc = kick((step < prm->nsteps - 1 ? 2.0 * lam : lam) * eps)) != LQCD_OK) return rc;
  }
  if ((rc = hamiltonian(&res->kinetic1, &res->gauge1, &res->fermion1)) != LQCD_OK) return rc;
  res->H0 = res->kinetic0 + res->gauge0 + res->fermion0;
  res->H1 = res->kinetic1 + res->gauge1 + res->fermion1;
  res->dH = res->H1 - res->H0;
  res->accepted = (uniform < exp(-res->dH)) ? 1 : 0;
  if (!std::isfinite(res->dH)) res->accepted = 0;
  if (res->accepted) {
    if ((rc = links.finish()) != LQCD_OK) return rc;
    TJ_CUDA(cudaMemcpyAsync(U_dev, tw->U, sizeof(double2) * 9 * 4 * V, cudaMemcpyDeviceToDevice, st));
  } else {
    links.stale = false;
    if ((rc = lqcd_set_gauge(ctx, U_dev)) != LQCD_OK) return rc;
  }
  if (prm->mom_out) TJ_CUDA(cudaMemcpyAsync(prm->mom_out, tw->P, sizeof(double) * ncomp, cudaMemcpyDeviceToDevice, st));
  if (prm->links_out)
    TJ_CUDA(cudaMemcpyAsync(prm->links_out, tw->U, sizeof(double2) * 9 * 4 * V, cudaMemcpyDeviceToDevice, st));
  TJ_CUDA(cudaStreamSynchronize(st));
  ctx->launches += nl;
  res->ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  return LQCD_OK;
}

// Fine-level twisted-mass Wilson-clover operator in FP64 storage, on the integer pipes of GB300.
//
//   y = D(mu) x   or   y = b - D(mu) x,   D as in dirac.cu, vectors, links and clover given in FP64.
//
// What bounds it: the FP64 form needs about 1300 FP64 instructions per site and system, and the SM has
// two FP64 lanes, so it ran at the FP64 issue rate (24^3x48 x 12 systems: 21.7 ms for 3.8 GB, 3% of the
// HBM rate, against 13.1 ms if every FP64 slot were used). Here the products run as 32 x 32 -> 64-bit
// integer multiply-adds (measured 59 lanes per cycle and SM on GB300, FP64 multiply-add 2.0), about 2600
// of them and 8300 shifts, additions and logic operations per site and system: 5.12 ms for the same
// case. It is bound by the integer pipes and their latency (multiply pipe 59% busy, issue 42%).
//
// Arithmetic. Block fixed point with one exponent S per (site, system): every contribution to the
// result is an integer multiple of 2^(S - 58), held in 64 bits. The entries of one spinor are truncated
// to integers V = x 2^(58 - X), |x| < 2^X, i.e. to 58 bits below the spinor's largest entry; matrices
// have 59 bits below their largest row sum (fixed64.cuh). A product keeps the high x high and the two
// high x low limb products exactly, sums them over a whole row exactly, and rounds once to the common
// unit; each dropped low x low term is below one unit. S is the largest of the exponents that the
// site's own spinor and its eight neighbours need, raised on the way when a neighbour asks for more (the
// sums are shifted then). The unit is about 2^-56 of a typical result, finer than the rounding of a
// 53-bit sum: against extended precision the result is 5e-17 off, that of FP64 arithmetic 9e-17 to
// 1.5e-16 (8^3x8, Gaussian fields). Bounds: a hop is below 2^58 units (row sum 2^59 x half spinor 2^59 /
// 2^60), eight of them below 2^61; the local term is below 2^60 (2^59 x 2^58 / 2^57), the twist and the
// doublet coupling below 2^58 each: no 64-bit sum can wrap. Inside a row the mixed products sum to less
// than 2^60 + 6 2^58 (hops) and 5/4 2^59 + 12 2^57 (local term).
//
// Entries. The unit is that of the site's largest contributions, so an entry whose own contributions are all
// small would be left with few bits or none (unit links without clover: the colours do not mix). The magnitudes
// of what is added to every real and imaginary part are therefore summed beside it, and a component of which
// one part has received less than 2^52 units is computed in FP64 arithmetic from its own terms
// (fine_entry_f64; the whole site where there are more than five). The others are off by 2 units or so (45 if
// every rounding went the same way): as FP64 sums of their terms. Gaussian fields have next to no such
// components; the sums cost 1.5 to 4.5% (24^3x48, 12 systems 5.04 to 5.12 ms, 1 system 0.507 to 0.526). A field with
// three of four spins zero takes 21.0 ms (5.07 without this, 21.7 in FP64 arithmetic throughout); the residuals of a
// point source's solution, whose colours and spins differ in size, 1.49 ms each on 16^3x32 x 12 systems (1.10 without).
//
// A site whose spinors, links or masses are outside the range of this form (infinities and NaN, entries
// beyond about 2^900 or below 2^-840, |mu| of the size of the clover block) is computed in FP64
// arithmetic by the same thread (fine_site_f64), which also serves a context without fixed-point copies.
// Subnormal entries with a zero high word count as zero.
#include "autotune.cuh"
#include "fixed64.cuh"
#include "profile.cuh"
#include "stencil.cuh"

namespace tmamg {

// ---------------------------------------------------------------- fixed-point copies
// h 2^30 + l = q with |l| <= 2^29, for |q| < 2^60
__device__ __forceinline__ int2 fx_split(long long q) {
  const int h = (int)((q + (1ll << 29)) >> 30);
  return make_int2(h, (int)(q - ((long long)h << 30)));
}
// v 2^(59 - n) rounded to an integer (nearest, halves to even), as limbs, for |v| < 2^n. Integer operations and integer
// comparisons in what follows: FP64 instructions bound these kernels (24^3x48, links 640 -> 120 us, clover 620 -> 230)
__device__ __forceinline__ int2 fx_limbs(double v, int n) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & ((1ull << 52) - 1)) | (e ? 1ull << 52 : 0);
  const int right = n - FX_BITS + 1075 - (e ? e : 1);  // v = m 2^(e - 1075)
  unsigned long long q;
  if (right <= 0) q = m << -right;  // by at most 6
  else if (right < 54) q = (m + ((1ull << (right - 1)) - 1) + ((m >> right) & 1)) >> right;
  else q = 0;
  return fx_split((long long)b < 0 ? -(long long)q : (long long)q);
}

// the larger of two numbers that are not negative (a NaN of either sign counts as larger)
__device__ __forceinline__ double fx_larger(double a, double b) {
  const unsigned long long x = (unsigned long long)__double_as_longlong(a);
  const unsigned long long y = (unsigned long long)__double_as_longlong(b);
  return __longlong_as_double((long long)(x > y ? x : y));
}

// exponent n with sum < 2^n (sum >= 0 or NaN)
__device__ __forceinline__ int fx_exponent(double sum) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(sum);
  if (b >= (unsigned long long)__double_as_longlong(1e300)) return FX_BAD;
  if (b < (unsigned long long)__double_as_longlong(1e-300)) return b ? FX_BAD : FX_ZERO;
  return (int)(b >> 52) - 1022;
}

__global__ void fixed_links_kernel(const double2* __restrict__ U, FixedOp fx, int64_t V) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 4 * V) return;
  const int64_t mu = t / V, s = t % V;
  double2 u[9];
  double rs[3] = {0, 0, 0}, cs[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    u[k] = U[(mu * 9 + k) * V + s];
    const double a = fabs(u[k].x) + fabs(u[k].y);
    rs[k / 3] += a;
    cs[k % 3] += a;
  }
  double m = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) m = fx_larger(m, fx_larger(rs[k], cs[k]));
  const int n = fx_exponent(m * (1.0 + 1e-12));  // the sums above are rounded
  fx.nU[t] = n;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    int4 o = make_int4(0, 0, 0, 0);
    if (n != FX_BAD && n != FX_ZERO) {
      const int2 a = fx_limbs(u[k].x, n), b = fx_limbs(u[k].y, n);
      o = make_int4(a.x, a.y, b.x, b.y);
    }
    fx.U[(mu * 9 + k) * V + s] = o;
  }
}

__global__ void fixed_clover_kernel(const double* __restrict__ C, FixedOp fx, int64_t V) {
  const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= V) return;
  double m = 0;
  for (int chi = 0; chi < 2; ++chi) {
    const double* Cc = C + (int64_t)chi * 36 * V + s;
    double rs[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) rs[i] = fabs(Cc[(int64_t)i * V]);
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
      for (int j = 0; j < i; ++j) {
        const int k = 6 + 2 * (i * (i - 1) / 2 + j);
        const double a = fabs(Cc[(int64_t)k * V]) + fabs(Cc[(int64_t)(k + 1) * V]);
        rs[i] += a;
        rs[j] += a;
      }
#pragma unroll
    for (int i = 0; i < 6; ++i) m = fx_larger(m, rs[i]);
  }
  const int n = fx_exponent(m * (1.0 + 1e-12));
  fx.nC[s] = n;
  for (int k = 0; k < 72; ++k)
    fx.C[(int64_t)k * V + s] = n != FX_BAD && n != FX_ZERO ? fx_limbs(C[(int64_t)k * V + s], n) : make_int2(0, 0);
}

void launch_fixed_links(const Geom& g, const double2* U64, cudaStream_t st) {
  if (!g.fx.U) return;
  fixed_links_kernel<<<(unsigned)((4 * g.V + 127) / 128), 128, 0, st>>>(U64, g.fx, g.V); TM_COUNT();
}

void launch_fixed_clover(const Geom& g, const double* C64, cudaStream_t st) {
  if (!g.fx.U) return;
  fixed_clover_kernel<<<(unsigned)((g.V + 127) / 128), 128, 0, st>>>(C64, g.fx, g.V); TM_COUNT();
}

int alloc_fixed(Geom& g) {
  FixedOp f;
  cudaError_t e = dev_alloc(nullptr, &f.U, sizeof(int4) * 36 * g.V);
  if (e == cudaSuccess) e = dev_alloc(nullptr, &f.nU, sizeof(int) * 4 * g.V);
  if (e == cudaSuccess) e = dev_alloc(nullptr, &f.C, sizeof(int2) * 72 * g.V);
  if (e == cudaSuccess) e = dev_alloc(nullptr, &f.nC, sizeof(int) * g.V);
  g.fx = f;
  if (e == cudaSuccess) return 0;
  free_fixed(g);
  cudaGetLastError();  // an optional copy that does not fit is no error of the call
  return -1;
}

void free_fixed(Geom& g) {
  cudaFree(g.fx.U);
  cudaFree(g.fx.nU);
  cudaFree(g.fx.C);
  cudaFree(g.fx.nC);
  g.fx = FixedOp();
}

// ---------------------------------------------------------------- one site in FP64 arithmetic
struct FineSite {
  const double2* U;
  const double* C;
  const double* x;     // tile's spinors
  const double* xp;    // the doublet partner's (or null)
  const double* b;     // right-hand side tile of the residual form (or null)
  double* y;
  double mu, ep, bc_t;
  int64_t s, V;
  int64_t nb[8];       // neighbours: +x, -x, +y, ...
  bool last_t, first_t;
};

// writes the components in `which` (in the residual form in place, the others hold results already)
__device__ __noinline__ void fine_site_f64(const FineSite& f, unsigned which) {
  Spinor<double, 1> acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    acc.c[k].re[0] = 0;
    acc.c[k].im[0] = 0;
  }
#define TM_HOP(NU)                                                                                      \
  hop<NU, true, double, 1>(acc, f.x + f.nb[2 * NU] * 2, f.V, f.U + (int64_t)NU * 9 * f.V, f.V, f.s,     \
                           NU == 3 && f.last_t ? f.bc_t : 1.0);                                         \
  hop<NU, false, double, 1>(acc, f.x + f.nb[2 * NU + 1] * 2, f.V, f.U + (int64_t)NU * 9 * f.V, f.V,     \
                            f.nb[2 * NU + 1], NU == 3 && f.first_t ? f.bc_t : 1.0);
  TM_HOP(0)
  TM_HOP(1)
  TM_HOP(2)
  TM_HOP(3)
#undef TM_HOP
  local_term<double, 1>(acc, f.x + f.s * 2, f.V, f.C, f.V, f.s, &f.mu, f.xp ? f.xp + f.s * 2 : nullptr, f.ep);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    if (!(which >> k & 1)) continue;
    if (f.b) {
      CV<double, 1> bv;
      ldcv(bv, f.b + (f.s + (int64_t)k * f.V) * 2);
      acc.c[k].re[0] = bv.re[0] - acc.c[k].re[0];
      acc.c[k].im[0] = bv.im[0] - acc.c[k].im[0];
    }
    stcv(f.y + (f.s + (int64_t)k * f.V) * 2, acc.c[k]);
  }
}

// Component k of the same, by spin and colour at run time
__device__ __noinline__ void fine_entry_f64(const FineSite& f, int k) {
  // multipliers (as in mulc) of the projection and of the lower spins for a forward hop, two bits per direction
  // and half spinor: Proj's c0, c1 and b0, b1; a backward hop has the opposite signs
  constexpr unsigned KC = 0x5E4Au, KB = 0x5B1Fu;
  const int spin = k / 3, col = k % 3;
  double re = 0, im = 0;
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int nu = hop >> 1, back = hop & 1;
    const int half = spin < 2 ? spin : (nu < 2 ? 3 - spin : spin - 2);  // Proj's p0, p1
    const int low = 2 + (nu < 2 ? 1 - half : half);                     // the lower spin in that half spinor
    const int kc = ((KC >> (4 * nu + 2 * half)) & 3) ^ back;
    const int kb = spin < 2 ? 0 : ((KB >> (4 * nu + 2 * (spin - 2))) & 3) ^ back;
    const int64_t at = f.nb[hop], ls = back ? at : f.s;
    double gr = 0, gi = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double2 u = *reinterpret_cast<const double2*>(f.x + ((int64_t)(half * 3 + b) * f.V + at) * 2);
      const double2 d = *reinterpret_cast<const double2*>(f.x + ((int64_t)(low * 3 + b) * f.V + at) * 2);
      const double dr = kc & 2 ? -d.y : d.x, di = kc & 2 ? d.x : d.y;
      const double hr = kc & 1 ? u.x - dr : u.x + dr, hi = kc & 1 ? u.y - di : u.y + di;
      double2 w = f.U[((int64_t)nu * 9 + (back ? b * 3 + col : col * 3 + b)) * f.V + ls];
      if (back) w.y = -w.y;
      gr += w.x * hr - w.y * hi;
      gi += w.x * hi + w.y * hr;
    }
    if ((hop == 6 && f.last_t) || (hop == 7 && f.first_t)) {
      gr *= f.bc_t;
      gi *= f.bc_t;
    }
    const double tr = kb & 2 ? -gi : gr, ti = kb & 2 ? gr : gi;
    re += kb & 1 ? -tr : tr;
    im += kb & 1 ? -ti : ti;
  }
  const int chi = k / 6, i = k % 6;
  const double* Cc = f.C + (int64_t)chi * 36 * f.V + f.s;
  const double* xc = f.x + ((int64_t)chi * 6 * f.V + f.s) * 2;
  double orr = 0, oi = 0;
#pragma unroll 1
  for (int j = 0; j < 6; ++j) {
    const double2 x = *reinterpret_cast<const double2*>(xc + (int64_t)j * f.V * 2);
    double ar, ai;
    if (i == j) {
      ar = Cc[(int64_t)i * f.V];
      ai = chi == 0 ? f.mu : -f.mu;
    } else {
      const int q = i > j ? 6 + 2 * (i * (i - 1) / 2 + j) : 6 + 2 * (j * (j - 1) / 2 + i);
      ar = Cc[(int64_t)q * f.V];
      ai = Cc[(int64_t)(q + 1) * f.V];
      if (i < j) ai = -ai;
    }
    orr += ar * x.x - ai * x.y;
    oi += ar * x.y + ai * x.x;
  }
  const int64_t at = ((int64_t)k * f.V + f.s) * 2;
  if (f.xp) {
    orr -= f.ep * f.xp[at];
    oi -= f.ep * f.xp[at + 1];
  }
  orr -= 0.5 * re;
  oi -= 0.5 * im;
  if (f.b) {
    orr = f.b[at] - orr;
    oi = f.b[at + 1] - oi;
  }
  *reinterpret_cast<double2*>(f.y + at) = make_double2(orr, oi);
}

// ---------------------------------------------------------------- fixed-point building blocks
typedef long long i64;
typedef unsigned long long u64;

struct Limb {  // h 2^30 + l
  int h, l;
};

// shifts that clamp their amount (a negative amount counts as a large one)
__device__ __forceinline__ u64 shr64(u64 v, int n) {
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
__device__ __forceinline__ i64 sar64(i64 v, int n) {
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}

// x 2^(58 - X) truncated to an integer, as limbs of the sign of x (|h| < 2^28, |l| < 2^30), for the bits
// (lo, hi) of a double x with |x| < 2^X; ec = X + 1026
__device__ __forceinline__ Limb fx_conv(unsigned lo, unsigned hi, int ec) {
  const unsigned mh = __funnelshift_l(lo, hi, 11) | 0x80000000u;  // mantissa with its leading one, left-justified
  const u64 w = shr64(((u64)mh << 32) | (lo << 11), ec - (int)((hi << 1) >> 21));
  const int sg = ((int)hi >> 31) | 1;
  Limb r;
  r.h = (int)(w >> 32) * sg;
  r.l = (int)((unsigned)w >> 2) * sg;
  return r;
}

__device__ __forceinline__ i64 madw(int a, int b, i64 c) { return (i64)a * b + c; }

// sum of products in two parts: hi counts 2^60, mid counts 2^30
struct FxSum {
  i64 hi, mid;
};
__device__ __forceinline__ void fx_mad(FxSum& s, int ah, int al, const Limb& b) {
  s.hi = madw(ah, b.h, s.hi);
  s.mid = madw(ah, b.l, s.mid);
  s.mid = madw(al, b.h, s.mid);
}

// biased exponent of a spinor's largest entry from the maximum t of (hi word << 1): |x| < 2^(e - 1022)
__device__ __forceinline__ int fx_top(unsigned t) { return t ? (int)(t >> 21) : FX_ZERO; }

// raw FP64 spinor of one site: (re lo, re hi, im lo, im hi) per entry
struct RawD {
  uint4 v[12];
};
__device__ __forceinline__ void ld_rawd(RawD& r, const double* __restrict__ p, int64_t V) {
#pragma unroll
  for (int k = 0; k < 12; ++k) r.v[k] = *reinterpret_cast<const uint4*>(p + (int64_t)k * V * 2);
}
__device__ __forceinline__ unsigned raw_max(const RawD& r) {
  unsigned t = 0;
#pragma unroll
  for (int k = 0; k < 12; ++k) t = max(t, max(r.v[k].y << 1, r.v[k].w << 1));
  return t;
}

// The magnitudes of what is added to an entry, |re| and |im| in two halves of a word that counts 2^48 units
// (they add up to less than 2^14 counts, by the bounds of the sums)
__device__ __forceinline__ unsigned fx_mag(i64 re, i64 im) {
  return __byte_perm((unsigned)abs((int)(re >> 32)), (unsigned)abs((int)(im >> 32)), 0x7632);
}
constexpr unsigned FX_LEAST = 1u << 4;  // 2^52 units
// components computed one by one: the whole site does less for each (with 3, the field with one spin takes 23.6 ms)
constexpr int FX_ENTRIES = 5;

// raise the common exponent to at least `want` (the sums keep their value)
__device__ __forceinline__ void fx_raise(i64 (&acc)[24], unsigned (&mag)[12], int& S, int want) {
  if (want > S) {
    const int d = want - S;
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = sar64(acc[k], d);
    const unsigned keep = d < 16 ? (0xffffu >> d) * 0x10001u : 0u;
#pragma unroll
    for (int k = 0; k < 12; ++k) mag[k] = (mag[k] >> (d & 15)) & keep;
    S = want;
  }
}

__device__ __forceinline__ Limb operator+(const Limb& a, const Limb& b) { return Limb{a.h + b.h, a.l + b.l}; }
__device__ __forceinline__ Limb operator-(const Limb& a, const Limb& b) { return Limb{a.h - b.h, a.l - b.l}; }

// h = u + K(d), K as in mulc, complex entries as limbs
template <int K>
__device__ __forceinline__ void fx_proj(Limb (&h)[2], const Limb (&u)[2], const Limb (&d)[2]) {
  if (K == 0) { h[0] = u[0] + d[0]; h[1] = u[1] + d[1]; }
  if (K == 1) { h[0] = u[0] - d[0]; h[1] = u[1] - d[1]; }
  if (K == 2) { h[0] = u[0] - d[1]; h[1] = u[1] + d[0]; }
  if (K == 3) { h[0] = u[0] + d[1]; h[1] = u[1] - d[0]; }
}
template <int NU, bool FWD>
__device__ __forceinline__ void fx_half(Limb (&h)[2][3][2], const Limb (&v)[12][2]) {
  using P = Proj<NU, FWD>;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    fx_proj<P::c0>(h[0][c], v[c], v[(2 + P::p0) * 3 + c]);
    fx_proj<P::c1>(h[1][c], v[3 + c], v[(2 + P::p1) * 3 + c]);
  }
}

// acc -= K(g)
template <int K>
__device__ __forceinline__ void fx_sub(i64& ar, i64& ai, const i64 (&g)[2]) {
  if (K == 0) { ar -= g[0]; ai -= g[1]; }
  if (K == 1) { ar += g[0]; ai += g[1]; }
  if (K == 2) { ar += g[1]; ai -= g[0]; }
  if (K == 3) { ar -= g[1]; ai += g[0]; }
}
template <int NU, bool FWD>
__device__ __forceinline__ void fx_scatter(i64 (&acc)[24], unsigned (&mag)[12], const i64 (&g)[2][3][2]) {
  using P = Proj<NU, FWD>;
  static_assert((P::b0 & 2) == (P::b1 & 2), "both lower spins take real for real, or both real for imaginary parts");
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const unsigned m0 = fx_mag(g[0][a][0], g[0][a][1]), m1 = fx_mag(g[1][a][0], g[1][a][1]);
    mag[a] += m0;
    mag[3 + a] += m1;
    const unsigned l0 = P::p0 == 0 ? m0 : m1, l1 = P::p1 == 0 ? m0 : m1;
    mag[6 + a] += P::b0 & 2 ? __byte_perm(l0, 0, 0x1032) : l0;
    mag[9 + a] += P::b1 & 2 ? __byte_perm(l1, 0, 0x1032) : l1;
    fx_sub<0>(acc[2 * a], acc[2 * a + 1], g[0][a]);
    fx_sub<0>(acc[6 + 2 * a], acc[6 + 2 * a + 1], g[1][a]);
    fx_sub<P::b0>(acc[12 + 2 * a], acc[12 + 2 * a + 1], g[P::p0][a]);
    fx_sub<P::b1>(acc[18 + 2 * a], acc[18 + 2 * a + 1], g[P::p1][a]);
  }
}

// g = W h / 2 in units, W = U (FWD) or U^+; U: the link's entries with stride V
template <bool FWD>
__device__ __forceinline__ void fx_mul(i64 (&g)[2][3][2], const Limb (&h)[2][3][2], const int4* __restrict__ U,
                                       int64_t V) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int4 w[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) w[b] = U[(int64_t)(FWD ? a * 3 + b : b * 3 + a) * V];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      FxSum re = {0, 1ll << 29}, im = {0, 1ll << 29};  // rounding of the final >> 30
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        fx_mad(re, w[b].x, w[b].y, h[k][b][0]);
        fx_mad(im, w[b].x, w[b].y, h[k][b][1]);
        if (FWD) {
          fx_mad(re, -w[b].z, -w[b].w, h[k][b][1]);
          fx_mad(im, w[b].z, w[b].w, h[k][b][0]);
        } else {
          fx_mad(re, w[b].z, w[b].w, h[k][b][1]);
          fx_mad(im, -w[b].z, -w[b].w, h[k][b][0]);
        }
      }
      g[k][a][0] = re.hi + (re.mid >> 30);
      g[k][a][1] = im.hi + (im.mid >> 30);
    }
  }
}

// o = A_chi x_chi + i m x_chi on one chirality (m: limbs of s mu at the clover's scale)
__device__ __forceinline__ void fx_local(i64 (&o)[12], const uint4 (&r)[6], const int2* __restrict__ Cc, int64_t V,
                                         int ec, const int2 mp) {
  Limb xc[6][2];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    xc[i][0] = fx_conv(r[i].x, r[i].y, ec);
    xc[i][1] = fx_conv(r[i].z, r[i].w, ec);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    FxSum re = {0, 1ll << 26}, im = {0, 1ll << 26};
    const int2 d = Cc[(int64_t)i * V];
    fx_mad(re, d.x, d.y, xc[i][0]);
    fx_mad(im, d.x, d.y, xc[i][1]);
    fx_mad(re, -mp.x, -mp.y, xc[i][1]);
    fx_mad(im, mp.x, mp.y, xc[i][0]);
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      if (j == i) continue;
      const int k = i > j ? 6 + 2 * (i * (i - 1) / 2 + j) : 6 + 2 * (j * (j - 1) / 2 + i);
      const int2 ar = Cc[(int64_t)k * V], ai = Cc[(int64_t)(k + 1) * V];
      fx_mad(re, ar.x, ar.y, xc[j][0]);
      fx_mad(im, ar.x, ar.y, xc[j][1]);
      if (i > j) {
        fx_mad(re, -ai.x, -ai.y, xc[j][1]);
        fx_mad(im, ai.x, ai.y, xc[j][0]);
      } else {  // conjugate of the stored lower entry
        fx_mad(re, ai.x, ai.y, xc[j][1]);
        fx_mad(im, -ai.x, -ai.y, xc[j][0]);
      }
    }
    o[2 * i] = (re.hi << 3) + (re.mid >> 27);
    o[2 * i + 1] = (im.hi << 3) + (im.mid >> 27);
  }
}

// v 2^(59 - n) as an integer, for |v| < 2^(n - 2)
__device__ __forceinline__ i64 fx_scalar(double v, int n) {
  const u64 b = (u64)__double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7ff);
  const u64 q = shr64((b << 11) | (1ull << 63), 1027 + n - e);
  return (b >> 63) ? -(i64)q : (i64)q;
}
__device__ __forceinline__ bool fx_scalar_fits(double v, int n) {  // |v| < 2^(n - 2)
  return (int)(((unsigned)__double2hiint(v) << 1) >> 21) - 1022 <= n - 2;
}

// acc 2^(S - 58) rounded to the nearest double (S within the range checked by the caller)
__device__ __forceinline__ double fx_double(i64 a, int S) {
  const i64 sg = a >> 63;
  const u64 m = (u64)((a ^ sg) - sg);
  const int z = __clzll((i64)m);  // >= 1: the bounds keep |acc| below 2^63
  u64 q = m << (z - 1);           // leading one at bit 62
  q += 0x1ff + ((q >> 10) & 1);   // round to nearest even at bit 10
  // exponent field of the leading one, value 2^(63 - z + S - 58), minus one: the mantissa added to it
  // brings its leading one (or the carry of its rounding)
  const u64 bits = ((u64)(unsigned)(1023 + 63 - z + S - 58 - 1) << 52) + (q >> 10);
  return m ? __longlong_as_double((i64)(bits | ((u64)sg & (1ull << 63)))) : 0.0;
}

// ---------------------------------------------------------------- the stencil
template <int BX, bool RES, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) dirac64_kernel(FixedOp fx, const double2* __restrict__ U,
                                                             const double* __restrict__ C, const double* __restrict__ x,
                                                             double* y, const double* __restrict__ mu, int ntile, int Lx,
                                                             int Ly, int Lz, int Lt, int bc_t, const double* bsub,
                                                             int nshift, const double* __restrict__ eps, int parity) {
  // parity 0 or 1: y on the sites of that parity only (the others are not written); else -1.
  // y is not restrict-qualified: the residual form may run in place (bsub == y), every thread
  // reading b at its own site before it writes y there; x never overlaps y
  const int64_t V = (int64_t)Lx * Ly * Lz * Lt;
  const int64_t s = blockIdx.x * (int64_t)BX + threadIdx.x;
  const int tile = blockIdx.y * blockDim.y + threadIdx.y;
  if (s >= V || tile >= ntile) return;
  const int L[4] = {Lx, Ly, Lz, Lt};
  int c[4];
  site_coords(s, L, c);
  if (parity >= 0 && ((c[0] + c[1] + c[2] + c[3]) & 1) != parity) return;
  const int64_t tstride = (int64_t)24 * V;
  const double* xt = x + tile * tstride;
  // neighbours as offsets from s (32 bits: a lattice of 2^31 sites would need 800 GB per FP64 vector)
  const int strides[4] = {1, Lx, Lx * Ly, Lx * Ly * Lz};
  int nb[8];
#pragma unroll
  for (int nu = 0; nu < 4; ++nu) {
    nb[2 * nu] = c[nu] + 1 < L[nu] ? strides[nu] : -(L[nu] - 1) * strides[nu];
    nb[2 * nu + 1] = c[nu] > 0 ? -strides[nu] : (L[nu] - 1) * strides[nu];
  }
  const double m = mu[tile];
  // doublet form (eps): tiles 2p and 2p + 1 are the flavours u, d of doublet p
  const double ep = eps ? eps[tile >> 1] : 0.0;
  const double* xp = eps ? x + (int64_t)(tile ^ 1) * tstride : nullptr;
  // residual form: b once per right-hand side (for a doublet, per right-hand side and flavour)
  const double* bo = nullptr;
  if (RES) bo = bsub + (int64_t)(eps ? ((tile >> 1) / nshift) * 2 + (tile & 1) : tile / nshift) * tstride;

  bool ok = fx.U != nullptr;
  i64 acc[24];
  unsigned mag[12];
  int S = FX_ZERO;
  if (ok) {
    RawD raw;
    ld_rawd(raw, xt + s * 2, V);
    const int nC = fx.nC[s];
    ok = nC != FX_BAD && fx_scalar_fits(m, nC) && fx_scalar_fits(ep, nC);
    // own spinor: |x| < 2^(e - 1022); the local term needs S >= X + nC - 2. One more bit of room lets
    // most neighbours in without raising S.
    const int top = fx_top(raw_max(raw));
    if (top != FX_ZERO) S = top - 1022 + nC - 1;
    const i64 mq = fx_scalar(m, nC);
    // one copy of the code for both chiralities: the kernel has to fit the instruction cache
#pragma unroll 1
    for (int chi = 0; chi < 2; ++chi) {
      // loaded again: all twelve entries kept beside the sums spilled (24^3x48 x 12 systems 5.25 against 5.12 ms)
      uint4 r[6];
#pragma unroll
      for (int i = 0; i < 6; ++i)
        r[i] = *reinterpret_cast<const uint4*>(xt + (s + (int64_t)(6 * chi + i) * V) * 2);
      i64 o[12];
      fx_local(o, r, fx.C + (int64_t)chi * 36 * V + s, V, S - nC + 2 + 1026, fx_split(chi == 0 ? mq : -mq));
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        if (chi == 0) acc[i] = o[i];
        else acc[12 + i] = o[i];
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        const unsigned m = fx_mag(o[2 * i], o[2 * i + 1]);
        if (chi == 0) mag[i] = m;
        else mag[6 + i] = m;
      }
    }
    if (ep != 0.0) {
      // - eps times the partner flavour, at the clover's scale
      ld_rawd(raw, xp + s * 2, V);
      const int tp = fx_top(raw_max(raw));
      if (tp != FX_ZERO) fx_raise(acc, mag, S, tp - 1022 + nC - 2);
      const int2 en = fx_split(-fx_scalar(ep, nC));
      const int ec = S - nC + 2 + 1026;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        FxSum re = {0, 1ll << 26}, im = {0, 1ll << 26};
        fx_mad(re, en.x, en.y, fx_conv(raw.v[k].x, raw.v[k].y, ec));
        fx_mad(im, en.x, en.y, fx_conv(raw.v[k].z, raw.v[k].w, ec));
        const i64 er = (re.hi << 3) + (re.mid >> 27), ei = (im.hi << 3) + (im.mid >> 27);
        acc[2 * k] += er;
        acc[2 * k + 1] += ei;
        mag[k] += fx_mag(er, ei);
      }
    }
    // the eight hops in one loop (its body is small enough for the instruction cache; the unrolled form
    // spent a third of its time on instruction fetches): conversion and colour multiply are common, the
    // spin projection and the scatter into the four spins are picked by hop. No loads are kept in flight
    // across hops: the registers buy 16 warps per SM instead, which hide them
    int cur = nb[0];
#pragma unroll 1
    for (int hop = 0; hop < 8; ++hop) {
      RawD raw;
      ld_rawd(raw, xt + (s + cur) * 2, V);
      const int64_t ls = (hop & 1) ? s + cur : s;
      const int nU = fx.nU[(int64_t)(hop >> 1) * V + ls];
      ok &= nU != FX_BAD;
      const int t = fx_top(raw_max(raw));
      if (t != FX_ZERO) fx_raise(acc, mag, S, t - 1022 + nU);
      const int ec = S - nU + 1026;
      Limb v[12][2];
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        v[k][0] = fx_conv(raw.v[k].x, raw.v[k].y, ec);
        v[k][1] = fx_conv(raw.v[k].z, raw.v[k].w, ec);
      }
      Limb h[2][3][2];
      switch (hop) {
        case 0: fx_half<0, true>(h, v); cur = nb[1]; break;
        case 1: fx_half<0, false>(h, v); cur = nb[2]; break;
        case 2: fx_half<1, true>(h, v); cur = nb[3]; break;
        case 3: fx_half<1, false>(h, v); cur = nb[4]; break;
        case 4: fx_half<2, true>(h, v); cur = nb[5]; break;
        case 5: fx_half<2, false>(h, v); cur = nb[6]; break;
        case 6: fx_half<3, true>(h, v); cur = nb[7]; break;
        default: fx_half<3, false>(h, v); break;
      }
      if (bc_t < 0 && ((hop == 6 && c[3] == Lt - 1) || (hop == 7 && c[3] == 0))) {  // the hop wraps in t
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          Limb& e = h[k / 6][(k / 2) % 3][k % 2];
          e.h = -e.h;
          e.l = -e.l;
        }
      }
      i64 g[2][3][2];
      const int4* Un = fx.U + (int64_t)(hop >> 1) * 9 * V + ls;
      if (hop & 1) fx_mul<false>(g, h, Un, V);
      else fx_mul<true>(g, h, Un, V);
      switch (hop) {
        case 0: fx_scatter<0, true>(acc, mag, g); break;
        case 1: fx_scatter<0, false>(acc, mag, g); break;
        case 2: fx_scatter<1, true>(acc, mag, g); break;
        case 3: fx_scatter<1, false>(acc, mag, g); break;
        case 4: fx_scatter<2, true>(acc, mag, g); break;
        case 5: fx_scatter<2, false>(acc, mag, g); break;
        case 6: fx_scatter<3, true>(acc, mag, g); break;
        default: fx_scatter<3, false>(acc, mag, g); break;
      }
    }
    // all inputs zero (S never set), or every result and its unit far inside the normal range
    ok = ok && (S < FX_ZERO / 2 || (S > -900 && S < 900));
  }
  // the components whose contributions are too small for the units of this site (all-zero inputs have none)
  unsigned small = 0;
  if (S >= FX_ZERO / 2) {
#pragma unroll
    for (int k = 0; k < 12; ++k)
      if ((mag[k] & 0xffffu) < FX_LEAST || (mag[k] >> 16) < FX_LEAST) small |= 1u << k;
  }
  double* yt = y + tile * tstride;
  if (ok) {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      double2 o = make_double2(fx_double(acc[2 * k], S), fx_double(acc[2 * k + 1], S));
      const int64_t at = (s + (int64_t)k * V) * 2;
      if (small >> k & 1) continue;
      if (RES) {
        const double2 bv = *reinterpret_cast<const double2*>(bo + at);
        o = make_double2(bv.x - o.x, bv.y - o.y);
      }
      *reinterpret_cast<double2*>(yt + at) = o;
    }
    if (!small) return;
  }
  FineSite f;
  f.U = U; f.C = C; f.x = xt; f.xp = xp; f.b = bo; f.y = yt;
  f.mu = m; f.ep = ep; f.bc_t = bc_t;
  f.s = s; f.V = V;
#pragma unroll
  for (int k = 0; k < 8; ++k) f.nb[k] = s + nb[k];
  f.last_t = c[3] == Lt - 1;
  f.first_t = c[3] == 0;
  if (!ok || __popc(small) > FX_ENTRIES) {
    fine_site_f64(f, ok ? small : 0xfffu);
    return;
  }
  for (; small; small &= small - 1) fine_entry_f64(f, __ffs(small) - 1);
}

// launch variants: (sites per CTA row, largest CTA, CTAs per SM): 168 registers at 12 warps per SM, or 128
// registers (some spills) at 16 warps per SM; measured on 24^3x48 x 12 systems 5.12 and 5.54 ms
template <bool RES, int BX, int MAXT, int MINB>
static void launch_variant64(const Geom& g, const double2* U, const double* C, const double* x, double* y,
                             const double* mu, int nsys, const double* b, int nshift, const double* eps, int parity,
                             cudaStream_t st) {
  const int ty = pick_ty(nsys, BX, MAXT);
  dim3 block(BX, ty);
  dim3 grid((unsigned)((g.V + BX - 1) / BX), (unsigned)(nsys / ty));
  dirac64_kernel<BX, RES, MAXT, MINB><<<grid, block, 0, st>>>(g.fx, U, C, x, y, mu, nsys, g.L[0], g.L[1], g.L[2],
                                                              g.L[3], g.bc_t, b, nshift, eps, parity); TM_COUNT();
}

template <bool RES>
static void launch_tuned64(const char* family, bool may_tune, const Geom& g, const void* Uv, const double* C,
                           const double* x, double* y, const double* mu, int nsys, const double* b, int nshift,
                           const double* eps, int parity, cudaStream_t st) {
  const double2* U = reinterpret_cast<const double2*>(Uv);
  auto launch = [&](int v) {
    switch (v) {
      case 1: launch_variant64<RES, 32, 128, 4>(g, U, C, x, y, mu, nsys, b, nshift, eps, parity, st); return;
      default: launch_variant64<RES, 32, 192, 2>(g, U, C, x, y, mu, nsys, b, nshift, eps, parity, st); return;
    }
  };
  launch(tune_variant(family, g.V * 4096 + nsys, 2, [] { return 0; }, may_tune, launch, st));
}

template <>
void launch_dirac<double>(const Geom& g, const void* U, const double* C, const double* x, double* y, const double* mu,
                          int nsys, cudaStream_t st, const double* eps) {
  TM_PROF(st, "dirac_f64");
  launch_tuned64<false>("dirac_f64", true, g, U, C, x, y, mu, nsys, nullptr, 1, eps, -1, st);
}

void launch_dirac64_parity(const Geom& g, const double2* U, const double* C, const double* x, double* y, const double* mu,
                           int nsys, int parity, cudaStream_t st) {
  TM_PROF(st, "dirac_f64");
  launch_tuned64<false>("dirac_f64", true, g, U, C, x, y, mu, nsys, nullptr, 1, nullptr, parity, st);
}

void launch_residual64(const Geom& g, const double2* U, const double* C, const double* x, const double* b, int nshift,
                       double* r, const double* mu, int nsys, cudaStream_t st, const double* eps) {
  TM_PROF(st, "residual_f64");
  launch_tuned64<true>("residual_f64", b != r, g, U, C, x, r, mu, nsys, b, nshift, eps, -1, st);
}

}  // namespace tmamg

// Fine-level twisted-mass Wilson-clover operator on GB300 (sm_103a).
//
// D(mu) x(s) = A_chi(s) x(s) + i mu gamma5 x(s) - 1/2 sum_nu [(1-gamma_nu) U_nu(s) x(s+nu)
//                                                  + (1+gamma_nu) U_nu(s-nu)^+ x(s-nu)]
// with A_chi = 1/(2 kappa) + c_sw C restricted to chirality chi (the operator of the
// paper's Fig. 6 caption, D_TM = D_W + i mu gamma5, at delta mu = 1).
//
// Design: one thread per (site, tile of two systems), a CTA holding 32 sites and several tiles. The links and the
// clover blocks of the sites come to shared memory once per CTA and are applied to all its tiles (paper Sec. 3: the
// matrix data is loaded once for all right-hand sides); with a single tile every thread loads them itself, and on small
// lattices a site is split over twelve warps. Spin projection in the chiral basis halves the SU(3) work: each hop
// multiplies two colour vectors. The FP64 form is in dirac64.cu.
#include "autotune.cuh"
#include "stencil.cuh"
#include "profile.cuh"

namespace tmamg {

// ---------------------------------------------------------------- gauge conversion
__global__ void convert_gauge_kernel(const double* __restrict__ Uin, double2* __restrict__ U64, float2* __restrict__ U32,
                                     int64_t V) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= V * 4) return;
  int64_t s = t / 4;
  int mu = (int)(t % 4);
  const double* src = Uin + ((s * 4 + mu) * 9) * 2;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    double2 v = make_double2(src[2 * k], src[2 * k + 1]);
    U64[((int64_t)mu * 9 + k) * V + s] = v;
    U32[((int64_t)mu * 9 + k) * V + s] = make_float2((float)v.x, (float)v.y);
  }
}

void launch_convert_gauge(const Geom& g, const double* Uin, double2* U64, float2* U32, cudaStream_t st) {
  int64_t n = g.V * 4;
  int bs = 256;
  convert_gauge_kernel<<<(unsigned)((n + bs - 1) / bs), bs, 0, st>>>(Uin, U64, U32, g.V); TM_COUNT();
}

// ---------------------------------------------------------------- clover construction (FP64)
struct M3 {
  double2 e[9];
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // conj(a) * b
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

__device__ __forceinline__ M3 load_link(const double2* U, int mu, int64_t s, int64_t V) {
  M3 m;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k] = U[((int64_t)mu * 9 + k) * V + s];
  return m;
}

__device__ __forceinline__ M3 mm(const M3& a, const M3& b) {  // a b
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 acc = make_double2(0, 0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double2 p = cmul(a.e[i * 3 + k], b.e[k * 3 + j]);
        acc.x += p.x;
        acc.y += p.y;
      }
      c.e[i * 3 + j] = acc;
    }
  return c;
}

__device__ __forceinline__ M3 mmd(const M3& a, const M3& b) {  // a b^+
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 acc = make_double2(0, 0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double2 bb = make_double2(b.e[j * 3 + k].x, -b.e[j * 3 + k].y);
        double2 p = cmul(a.e[i * 3 + k], bb);
        acc.x += p.x;
        acc.y += p.y;
      }
      c.e[i * 3 + j] = acc;
    }
  return c;
}

__device__ __forceinline__ M3 dm(const M3& a, const M3& b) {  // a^+ b
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 acc = make_double2(0, 0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        double2 p = cmulc(a.e[k * 3 + i], b.e[k * 3 + j]);
        acc.x += p.x;
        acc.y += p.y;
      }
      c.e[i * 3 + j] = acc;
    }
  return c;
}

__device__ __forceinline__ int64_t nbr(const int* c, const int* L, int mu, int d) {
  int cc[4] = {c[0], c[1], c[2], c[3]};
  cc[mu] = (cc[mu] + d + L[mu]) % L[mu];
  return site_index(cc, L);
}

__device__ __forceinline__ int64_t nbr2(const int* c, const int* L, int mu, int dmu, int nu, int dnu) {
  int cc[4] = {c[0], c[1], c[2], c[3]};
  cc[mu] = (cc[mu] + dmu + L[mu]) % L[mu];
  cc[nu] = (cc[nu] + dnu + L[nu]) % L[nu];
  return site_index(cc, L);
}

// F_{mu nu}(s) = (Q - Q^+)/8 with Q the sum of the four clover leaves at s (mu < nu)
__device__ M3 field_strength(const double2* U, const int* c, const int* L, int64_t V, int mu, int nu) {
  int64_t s = site_index(c, L);
  M3 Umu = load_link(U, mu, s, V);
  M3 Unu = load_link(U, nu, s, V);
  M3 Umu_pnu = load_link(U, mu, nbr(c, L, nu, 1), V);
  M3 Unu_pmu = load_link(U, nu, nbr(c, L, mu, 1), V);
  M3 Umu_mmu = load_link(U, mu, nbr(c, L, mu, -1), V);
  M3 Unu_mmu = load_link(U, nu, nbr(c, L, mu, -1), V);
  M3 Umu_mmu_pnu = load_link(U, mu, nbr2(c, L, mu, -1, nu, 1), V);
  M3 Umu_mmu_mnu = load_link(U, mu, nbr2(c, L, mu, -1, nu, -1), V);
  M3 Unu_mmu_mnu = load_link(U, nu, nbr2(c, L, mu, -1, nu, -1), V);
  M3 Unu_mnu = load_link(U, nu, nbr(c, L, nu, -1), V);
  M3 Umu_mnu = load_link(U, mu, nbr(c, L, nu, -1), V);
  M3 Unu_pmu_mnu = load_link(U, nu, nbr2(c, L, mu, 1, nu, -1), V);
  // leaf 1: U_mu(s) U_nu(s+mu) U_mu(s+nu)^+ U_nu(s)^+
  M3 q = mmd(mmd(mm(Umu, Unu_pmu), Umu_pnu), Unu);
  // leaf 2: U_nu(s) U_mu(s-mu+nu)^+ U_nu(s-mu)^+ U_mu(s-mu)
  M3 t2 = mm(mmd(mmd(Unu, Umu_mmu_pnu), Unu_mmu), Umu_mmu);
  // leaf 3: U_mu(s-mu)^+ U_nu(s-mu-nu)^+ U_mu(s-mu-nu) U_nu(s-nu)
  M3 t3 = mm(dm(Umu_mmu, dm(Unu_mmu_mnu, Umu_mmu_mnu)), Unu_mnu);
  // leaf 4: U_nu(s-nu)^+ U_mu(s-nu) U_nu(s-nu+mu) U_mu(s)^+
  M3 t4 = mmd(mm(dm(Unu_mnu, Umu_mnu), Unu_pmu_mnu), Umu);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    q.e[k].x += t2.e[k].x + t3.e[k].x + t4.e[k].x;
    q.e[k].y += t2.e[k].y + t3.e[k].y + t4.e[k].y;
  }
  M3 F;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 a = q.e[i * 3 + j], b = q.e[j * 3 + i];
      F.e[i * 3 + j] = make_double2((a.x - b.x) * 0.125, (a.y + b.y) * 0.125);
    }
  return F;
}

// Per chirality chi (sign s = +1, -1) in the chiral basis:
//   c_sw C_chi = (i c_sw / 2) [[G3, G1 - i G2], [G1 + i G2, -G3]]   (2x2 spin blocks of 3x3 colour)
//   G1 = s F_xt - F_yz,  G2 = s F_yt + F_xz,  G3 = s F_zt - F_xy.
// Stored with the diagonal 1/(2 kappa) folded in: 6 real diagonal entries, then the
// 15 complex entries of the strict lower triangle (row i > col j, row-major), 36 reals.
__global__ void build_clover_kernel(const double2* __restrict__ U, int Lx, int Ly, int Lz, int Lt, double kappa,
                                    double c_sw, double* __restrict__ C64, float* __restrict__ C32) {
  int L[4] = {Lx, Ly, Lz, Lt};
  int64_t V = (int64_t)Lx * Ly * Lz * Lt;
  int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (s >= V) return;
  int c[4];
  site_coords(s, L, c);
  M3 F01 = field_strength(U, c, L, V, 0, 1);
  M3 F02 = field_strength(U, c, L, V, 0, 2);
  M3 F03 = field_strength(U, c, L, V, 0, 3);
  M3 F12 = field_strength(U, c, L, V, 1, 2);
  M3 F13 = field_strength(U, c, L, V, 1, 3);
  M3 F23 = field_strength(U, c, L, V, 2, 3);
  const double diag = 1.0 / (2.0 * kappa);
  for (int chi = 0; chi < 2; ++chi) {
    double sg = chi == 0 ? 1.0 : -1.0;
    double2 A[6][6];
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) {
        int k = a * 3 + b;
        double2 G1 = make_double2(sg * F03.e[k].x - F12.e[k].x, sg * F03.e[k].y - F12.e[k].y);
        double2 G2 = make_double2(sg * F13.e[k].x + F02.e[k].x, sg * F13.e[k].y + F02.e[k].y);
        double2 G3 = make_double2(sg * F23.e[k].x - F01.e[k].x, sg * F23.e[k].y - F01.e[k].y);
        // iG2 = (-G2.y, G2.x)
        double2 b00 = G3;
        double2 b01 = make_double2(G1.x + G2.y, G1.y - G2.x);  // G1 - i G2
        double2 b10 = make_double2(G1.x - G2.y, G1.y + G2.x);  // G1 + i G2
        double2 b11 = make_double2(-G3.x, -G3.y);
        // multiply by i c_sw / 2: (x, y) -> (-y, x) * c_sw / 2
        double h = 0.5 * c_sw;
        A[a][b] = make_double2(-b00.y * h, b00.x * h);
        A[a][3 + b] = make_double2(-b01.y * h, b01.x * h);
        A[3 + a][b] = make_double2(-b10.y * h, b10.x * h);
        A[3 + a][3 + b] = make_double2(-b11.y * h, b11.x * h);
      }
    double* out64 = C64 + (int64_t)chi * 36 * V;
    float* out32 = C32 + (int64_t)chi * 36 * V;
    for (int i = 0; i < 6; ++i) {
      double d = A[i][i].x + diag;
      out64[(int64_t)i * V + s] = d;
      out32[(int64_t)i * V + s] = (float)d;
    }
    int k = 6;
    for (int i = 1; i < 6; ++i)
      for (int j = 0; j < i; ++j) {
        out64[(int64_t)k * V + s] = A[i][j].x;
        out64[(int64_t)(k + 1) * V + s] = A[i][j].y;
        out32[(int64_t)k * V + s] = (float)A[i][j].x;
        out32[(int64_t)(k + 1) * V + s] = (float)A[i][j].y;
        k += 2;
      }
  }
}

void launch_build_clover(const Geom& g, const double2* U64, double kappa, double c_sw, double* C64, float* C32,
                         cudaStream_t st) {
  int bs = 128;
  build_clover_kernel<<<(unsigned)((g.V + bs - 1) / bs), bs, 0, st>>>(U64, g.L[0], g.L[1], g.L[2], g.L[3], kappa,
                                                                       c_sw, C64, C32); TM_COUNT();
}

__device__ __forceinline__ void dr_copy16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void dr_copy8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void dr_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void dr_wait_sync() {  // all but the last N groups of every thread have landed
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
  __syncthreads();
}

// bytes of the staged operator data of a CTA row of bx sites: links of the sites, links of their backward
// neighbours, clover blocks
__host__ __device__ constexpr int dr_stage_bytes(int bx) { return bx * (36 * 8 + 36 * 8 + 72 * 4); }

// The FP32 form (dirac64.cu holds the FP64 one).
// RES: residual form y = b - D x (b = bsub, tile for tile), else y = D x (bsub unused).
// STAGED: the links and clover blocks of the CTA's sites come to shared memory by asynchronous copies, once
// for all tiles of the CTA and ahead of their use; otherwise every thread loads them where it needs them.
//  What bounds the direct form is latency: 12 warps per SM, and each hop starts with nine loads of links
//  that the previous hop's arithmetic does not cover (33% of the issue slots used, 5.3 of 8.7 cycles per
//  instruction waiting for global loads, 24^3x48 x 16 systems). Staged in three groups, waited for as
//  they are needed, those loads are off the critical path and a quarter of the L1 lookups is gone; the
//  site's own spinor for the local term then joins the software pipeline (it gained nothing before).
//  Direct against staged: 40^3x80 x 16 systems 8.2 and 6.6 ms (2.7 ms at the HBM rate), 16^3x32 x 12 152
//  and 124 us; issue slots used 33% and 44%, L1 data path 43% and 60%. With one tile (one or two systems)
//  nothing is shared and the direct form is the faster one (24^3x48, one system: 137 against 177 us), so
//  both are launch variants. Prefetching the neighbours' lines into L1 (9.2 ms) and wider CTA rows (8.9 to 9.1
//  ms) measured slower.
// FIELD (staged, BX = 32, not RES): y is a user field [nsys][V][12], a warp's rows transposed through the staging
//  space, which spares the call the bundle's way to HBM and back: 20x12x28x44, 5 systems, 138 + 58 us as two
//  kernels, 166 us as one.
// MAXT, MINB: the launch variant's largest CTA and the CTAs per SM it is compiled for (which sets the
// register budget); every variant does the same per-thread arithmetic.
template <int BX, bool RES, bool STAGED, int MAXT, int MINB, bool FIELD = false>
__global__ void __launch_bounds__(MAXT, MINB) dirac_kernel(const float2* __restrict__ U, const float* __restrict__ C,
                                                           const float* __restrict__ x, float* y,
                                                           const double* __restrict__ mu, int nsys, int ntile, int Lx,
                                                           int Ly, int Lz, int Lt, float bc_t, const float* bsub,
                                                           const double* __restrict__ eps) {
  constexpr int T = 2;
  // y is not restrict-qualified: the residual form may run in place (bsub == y), every thread
  // reading b at its own site before it writes y there; x never overlaps y
  const int64_t V = (int64_t)Lx * Ly * Lz * Lt;
  const int64_t s0 = blockIdx.x * (int64_t)BX;
  const int tile = blockIdx.y * blockDim.y + threadIdx.y;
  const bool live = s0 + threadIdx.x < V;
  if (!STAGED && !live) return;
  const int64_t s = live ? s0 + threadIdx.x : V - 1;
  const int L[4] = {Lx, Ly, Lz, Lt};
  int c[4];
  site_coords(s, L, c);
  const int64_t tstride = (int64_t)12 * V * 2 * T;
  const float* xt = x + tile * tstride;
  const int64_t strides[4] = {1, (int64_t)Lx, (int64_t)Lx * Ly, (int64_t)Lx * Ly * Lz};
  // packed FP32x2 arithmetic over the tile's two systems
  Spinor2 acc;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    acc.c[k].re = make_float2(0.f, 0.f);
    acc.c[k].im = make_float2(0.f, 0.f);
  }
  // software pipeline over the eight hops: the neighbour spinor of hop k + 1 is loaded before
  // the colour multiply of hop k, so its latency overlaps that arithmetic
  int64_t nb[8];
#pragma unroll
  for (int nu = 0; nu < 4; ++nu) {
    nb[2 * nu] = c[nu] + 1 < L[nu] ? s + strides[nu] : s - (int64_t)(L[nu] - 1) * strides[nu];
    nb[2 * nu + 1] = c[nu] > 0 ? s - strides[nu] : s + (int64_t)(L[nu] - 1) * strides[nu];
  }
  extern __shared__ float4 dr_smem[];
  float2* Lf = reinterpret_cast<float2*>(dr_smem);  // [4 nu][9][BX] U_nu(s)
  float2* Lb = Lf + 36 * BX;                        // [4 nu][9][BX] U_nu(s - nu)
  float* Cs = reinterpret_cast<float*>(Lb + 36 * BX);  // [72][BX]
  if constexpr (STAGED) {
    // V is a multiple of 16 (even extents): the rows of a site range start on 16-byte boundaries
    const int nt = BX * blockDim.y, tid = threadIdx.y * BX + threadIdx.x;
    const int n = V - s0 < BX ? (int)(V - s0) : BX;
#pragma unroll
    for (int half = 0; half < 2; ++half) {  // directions x, y, then z, t
      for (int i = tid; i < 18 * (BX / 2); i += nt) {
        const int q = 18 * half + i / (BX / 2), e = 2 * (i % (BX / 2));
        if (e < n) dr_copy16(Lf + q * BX + e, U + (int64_t)q * V + s0 + e);
      }
      if (live) {
#pragma unroll
        for (int nu = 2 * half; nu < 2 * half + 2; ++nu)
          for (int k = threadIdx.y; k < 9; k += blockDim.y)
            dr_copy8(Lb + (nu * 9 + k) * BX + threadIdx.x, U + (int64_t)(nu * 9 + k) * V + nb[2 * nu + 1]);
      }
      dr_commit();
    }
    for (int i = tid; i < 72 * (BX / 4); i += nt) {
      const int q = i / (BX / 4), e = 4 * (i % (BX / 4));
      if (e < n) dr_copy16(Cs + q * BX + e, C + (int64_t)q * V + s0 + e);
    }
    dr_commit();
  }
  const float pf = c[3] == Lt - 1 ? bc_t : 1.f, pb = c[3] == 0 ? bc_t : 1.f;
  Raw2 raw;
  CV2 h[2][3];
  ld_raw2(raw, xt + nb[0] * 4, V);
  if constexpr (STAGED) dr_wait_sync<2>();
#define TM_PHOP(NU, FWD, K)                                                                          \
  proj_raw2<NU, FWD>(h, raw);                                                                        \
  if (STAGED || K < 7) ld_raw2(raw, xt + (K < 7 ? nb[K < 7 ? K + 1 : 0] : s) * 4, V);                \
  if constexpr (STAGED)                                                                              \
    mul_acc2<NU, FWD>(acc, h, (FWD ? Lf : Lb) + NU * 9 * BX, BX, threadIdx.x,                        \
                      NU == 3 ? (FWD ? pf : pb) : 1.f);                                              \
  else                                                                                               \
    mul_acc2<NU, FWD>(acc, h, U + (int64_t)NU * 9 * V, V, FWD ? s : nb[K], NU == 3 ? (FWD ? pf : pb) : 1.f);
  TM_PHOP(0, true, 0)
  TM_PHOP(0, false, 1)
  TM_PHOP(1, true, 2)
  TM_PHOP(1, false, 3)
  if constexpr (STAGED) dr_wait_sync<1>();
  TM_PHOP(2, true, 4)
  TM_PHOP(2, false, 5)
  TM_PHOP(3, true, 6)
  TM_PHOP(3, false, 7)
#undef TM_PHOP
  const int n0 = tile * 2;
  const float2 m2 = make_float2(n0 < nsys ? (float)mu[n0] : 0.f, n0 + 1 < nsys ? (float)mu[n0 + 1] : 0.f);
  // eps (doublet form): the tile's two systems are the flavours u, d of one doublet
  const float ep = eps ? (float)eps[tile] : 0.f;
  if constexpr (STAGED) {
    dr_wait_sync<0>();
    local2(acc, raw, Cs, BX, threadIdx.x, m2, ep);
    if constexpr (FIELD) {
      static_assert(STAGED && !RES && BX == 32, "a warp holds 32 sites of one tile");
      constexpr int PITCH = 26;  // 24 reals per site, and 2 that keep the transposed access off the same banks
      __syncthreads();           // the staged operator data is no longer needed
      float* sm = reinterpret_cast<float*>(dr_smem) + threadIdx.y * 32 * PITCH;
      const int ns = V - s0 < 32 ? (int)(V - s0) : 32;
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        if (n0 + l >= nsys) break;
#pragma unroll
        for (int k = 0; k < 12; ++k)
          *reinterpret_cast<float2*>(sm + threadIdx.x * PITCH + 2 * k) =
              l ? make_float2(acc.c[k].re.y, acc.c[k].im.y) : make_float2(acc.c[k].re.x, acc.c[k].im.x);
        __syncwarp();
        float* dst = y + ((int64_t)(n0 + l) * V + s0) * 24;
#pragma unroll
        for (int k = threadIdx.x; k < 32 * 24; k += 32)
          if (k < ns * 24) dst[k] = sm[k + (PITCH - 24) * (k / 24)];
        __syncwarp();
      }
      return;
    }
    if (!live) return;
  } else {
    local2(acc, xt + s * 4, V, C, V, s, m2, ep);
  }
  float* yo = y + tile * tstride + s * 4;
  if constexpr (RES) {
    const float* bo = bsub + tile * tstride + s * 4;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const CV2 bv = ld2(bo + (int64_t)k * V * 4);
      acc.c[k].re = sub2(bv.re, acc.c[k].re);
      acc.c[k].im = sub2(bv.im, acc.c[k].im);
    }
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) st2(yo + (int64_t)k * V * 4, acc.c[k]);
}

// The split form for lattices too small to fill the chip with a thread per site: twelve warps per 32 sites and tile.
// Warps 0 to 7 multiply one hop each and leave its two colour vectors in shared memory, every warp then computes one
// component of the local term and adds that component's hop parts in the order of the other forms (same bits).
// It is then one or two load latencies long instead of eight: 8^3x16, one system, 9.0 -> 8.0 us with cold caches and
// 10.3 -> 8.2 us per call of many; with four times the sites 20.5 us against 12.0, so it is a launch variant.
constexpr int DS_WARPS = 12;
constexpr int DS_TILES = 65535;  // tiles per launch: the grid's extent in y

template <int NU, bool FWD>
__device__ __forceinline__ void split_hop(float4* g, const float2* __restrict__ U, const float* __restrict__ xt, int V,
                                          int s, int c, int ext, int stride, float phase) {
  const int nb = FWD ? (c + 1 < ext ? s + stride : s - (ext - 1) * stride) : (c > 0 ? s - stride : s + (ext - 1) * stride);
  Raw2 raw;
  ld_raw2(raw, xt + (int64_t)nb * 4, V);
  CV2 h[2][3];
  proj_raw2<NU, FWD>(h, raw);
  Spinor2 a;
#pragma unroll
  for (int k = 0; k < 12; ++k) a.c[k].re = a.c[k].im = make_float2(0.f, 0.f);
  mul_acc2<NU, FWD>(a, h, U + (int64_t)NU * 9 * V, V, FWD ? s : nb, phase);
#pragma unroll
  for (int k = 0; k < 6; ++k) g[k * 32] = make_float4(a.c[k].re.x, a.c[k].re.y, a.c[k].im.x, a.c[k].im.y);  // spins 0, 1
}

template <int NU, bool FWD, int SPIN>
__device__ __forceinline__ void split_add(CV2& acc, const float4* g, int col) {
  using P = Proj<NU, FWD>;
  constexpr int K = SPIN < 2 ? 0 : SPIN == 2 ? P::b0 : P::b1;
  constexpr int half = SPIN < 2 ? SPIN : (SPIN == 2 ? P::p0 : P::p1);
  acc2<K>(acc, ld2(reinterpret_cast<const float*>(g + (half * 3 + col) * 32)));
}

// the sum over the hops of component (SPIN, col)
template <int SPIN>
__device__ __forceinline__ CV2 split_sum(const float4* g, int col) {
  CV2 a;
  a.re = a.im = make_float2(0.f, 0.f);
  split_add<0, true, SPIN>(a, g, col);
  split_add<0, false, SPIN>(a, g + 192, col);
  split_add<1, true, SPIN>(a, g + 2 * 192, col);
  split_add<1, false, SPIN>(a, g + 3 * 192, col);
  split_add<2, true, SPIN>(a, g + 4 * 192, col);
  split_add<2, false, SPIN>(a, g + 5 * 192, col);
  split_add<3, true, SPIN>(a, g + 6 * 192, col);
  split_add<3, false, SPIN>(a, g + 7 * 192, col);
  return a;
}

template <bool RES>
__global__ void __launch_bounds__(DS_WARPS * 32, 2) dirac_split_kernel(
    const float2* __restrict__ U, const float* __restrict__ C, const float* __restrict__ x, float* y,
    const __grid_constant__ MassArgs ma, int nsys, int Lx, int Ly, int Lz, int Lt, float bc_t, const float* bsub) {
  __shared__ float4 gs[8 * 192];  // [hop][half spinor component][site]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int V = Lx * Ly * Lz * Lt, tile = blockIdx.y;
  const int s0 = blockIdx.x * 32 + lane;
  const bool live = s0 < V;
  const int s = live ? s0 : V - 1;
  const float* xt = x + (int64_t)tile * 12 * V * 4;
  float4* g = gs + warp * 192 + lane;
  const int sy = Lx, sz = Lx * Ly, st = sz * Lz;
  switch (warp) {
    case 0: split_hop<0, true>(g, U, xt, V, s, s % Lx, Lx, 1, 1.f); break;
    case 1: split_hop<0, false>(g, U, xt, V, s, s % Lx, Lx, 1, 1.f); break;
    case 2: split_hop<1, true>(g, U, xt, V, s, s / sy % Ly, Ly, sy, 1.f); break;
    case 3: split_hop<1, false>(g, U, xt, V, s, s / sy % Ly, Ly, sy, 1.f); break;
    case 4: split_hop<2, true>(g, U, xt, V, s, s / sz % Lz, Lz, sz, 1.f); break;
    case 5: split_hop<2, false>(g, U, xt, V, s, s / sz % Lz, Lz, sz, 1.f); break;
    case 6: split_hop<3, true>(g, U, xt, V, s, s / st, Lt, st, s / st == Lt - 1 ? bc_t : 1.f); break;
    case 7: split_hop<3, false>(g, U, xt, V, s, s / st, Lt, st, s / st == 0 ? bc_t : 1.f); break;
    default: break;
  }
  // component `warp` of the local term (local2_of: the same operations in the same order)
  const int chi = warp / 6, i = warp % 6;
  const int n0 = tile * 2;
  const double* mu = ma.mu ? ma.mu : ma.v;
  const float2 m2 = make_float2(n0 < nsys ? (float)mu[n0] : 0.f, n0 + 1 < nsys ? (float)mu[n0 + 1] : 0.f);
  const float ep = ma.doublet ? (float)(ma.eps ? ma.eps : ma.e)[tile] : 0.f;
  const float* Cc = C + (int64_t)chi * 36 * V + s;
  const float* xc = xt + ((int64_t)chi * 6 * V + s) * 4;
  const CV2 xi = ld2(xc + (int64_t)i * V * 4);
  const float2 smu = chi == 0 ? m2 : make_float2(-m2.x, -m2.y);
  const float2 nsmu = make_float2(-smu.x, -smu.y);
  const float d = Cc[(int64_t)i * V];
  CV2 o;
  o.re = fma2(f2(d), xi.re, mul2(nsmu, xi.im));
  o.im = fma2(f2(d), xi.im, mul2(smu, xi.re));
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    if (j == i) continue;
    const CV2 xj = ld2(xc + (int64_t)j * V * 4);
    const int k = i > j ? 6 + 2 * (i * (i - 1) / 2 + j) : 6 + 2 * (j * (j - 1) / 2 + i);
    const float ar = Cc[(int64_t)k * V], ci = Cc[(int64_t)(k + 1) * V];
    const float ai = i > j ? ci : -ci;
    o.re = fma2(f2(ar), xj.re, o.re);
    o.re = fma2(f2(-ai), xj.im, o.re);
    o.im = fma2(f2(ar), xj.im, o.im);
    o.im = fma2(f2(ai), xj.re, o.im);
  }
  if (ep != 0.f) {
    o.re = fma2(f2(-ep), make_float2(xi.re.y, xi.re.x), o.re);
    o.im = fma2(f2(-ep), make_float2(xi.im.y, xi.im.x), o.im);
  }
  __syncthreads();
  const int col = warp % 3;
  CV2 a;
  switch (warp / 3) {
    case 0: a = split_sum<0>(gs + lane, col); break;
    case 1: a = split_sum<1>(gs + lane, col); break;
    case 2: a = split_sum<2>(gs + lane, col); break;
    default: a = split_sum<3>(gs + lane, col); break;
  }
  a.re = fma2(f2(-0.5f), a.re, o.re);
  a.im = fma2(f2(-0.5f), a.im, o.im);
  if (!live) return;
  const int64_t at = (((int64_t)tile * 12 + warp) * V + s) * 4;
  if constexpr (RES) {
    const CV2 bv = ld2(bsub + at);
    a.re = sub2(bv.re, a.re);
    a.im = sub2(bv.im, a.im);
  }
  st2(y + at, a);
}

template <bool RES>
static void launch_split(const Geom& g, const float2* U, const float* C, const float* x, float* y, const MassArgs& ma,
                         int nsys, const float* b, cudaStream_t st) {
  MassArgs m = ma;
  for (int t0 = 0, nt = ntiles(nsys, 2); t0 < nt; t0 += DS_TILES) {
    const int n = nt - t0 < DS_TILES ? nt - t0 : DS_TILES;
    dirac_split_kernel<RES><<<dim3((unsigned)((g.V + 31) / 32), n), DS_WARPS * 32, 0, st>>>(
        U, C, x, y, m, nsys - 2 * t0, g.L[0], g.L[1], g.L[2], g.L[3], (float)g.bc_t, b);
    TM_COUNT();
    const int64_t step = (int64_t)n * 48 * g.V;
    x += step;
    y += step;
    if (b) b += step;
    if (m.mu) m.mu += 2 * n;  // (the masses in the arguments are those of at most 32 systems)
    if (m.eps) m.eps += n;
  }
}

// launch variants: (sites per CTA row, staged, largest CTA, CTAs per SM): 168 registers at 12 warps per SM,
// or 128 registers (a few bytes of spills) at 16 warps per SM; and the split form
template <bool RES, int BX, bool STAGED, int MAXT, int MINB>
static void launch_variant(const Geom& g, const float2* U, const float* C, const float* x, float* y, const double* mu,
                           int nsys, const float* b, const double* eps, cudaStream_t st) {
  const int nt = ntiles(nsys, 2);
  const int ty = pick_ty(nt, BX, MAXT);
  dim3 block(BX, ty);
  dim3 grid((unsigned)((g.V + BX - 1) / BX), (unsigned)(nt / ty));
  if (STAGED) func_smem_optin((const void*)dirac_kernel<BX, RES, STAGED, MAXT, MINB>, dr_stage_bytes(BX));
  dirac_kernel<BX, RES, STAGED, MAXT, MINB><<<grid, block, STAGED ? dr_stage_bytes(BX) : 0, st>>>(
      U, C, x, y, mu, nsys, nt, g.L[0], g.L[1], g.L[2], g.L[3], (float)g.bc_t, b, eps); TM_COUNT();
}

constexpr int NVARIANTS = 4, DIRECT_VARIANT = 1, SPLIT_VARIANT = 3;
static int64_t tune_key(const Geom& g, int nsys) { return g.V * 4096 + nsys; }
// Where nothing is tuned (tuning is off, or the first residual of a shape in place): direct with one tile, which
// shares no links, and below two waves of threads, where staging is latency (staged and direct: 24^3x48 one system
// 172 and 135 us; 8^3x16 twelve systems 14.3 and 12.6, 12^3x24 four 20.5 and 18.5, five 26.8 and 28.7)
static int untuned_variant(const Geom& g, int nsys) {
  const int nt = ntiles(nsys, 2);
  return nt == 1 || g.V * nt < 2ll * 384 * device_sms() ? DIRECT_VARIANT : 0;
}
static int peek_variant(const Geom& g, int nsys) {
  return tune_peek("dirac_f32", tune_key(g, nsys), NVARIANTS, [&] { return untuned_variant(g, nsys); });
}

template <bool RES>
static void launch_tuned(const char* family, bool may_tune, const Geom& g, const float2* U, const float* C,
                         const float* x, float* y, const double* mu, int nsys, const float* b, const double* eps,
                         cudaStream_t st) {
  auto launch = [&](int v) {
    switch (v) {
      case DIRECT_VARIANT: launch_variant<RES, 32, false, 192, 2>(g, U, C, x, y, mu, nsys, b, eps, st); return;
      case 2: launch_variant<RES, 32, true, 256, 2>(g, U, C, x, y, mu, nsys, b, eps, st); return;
      case SPLIT_VARIANT: {
        MassArgs ma;
        ma.mu = mu;
        ma.eps = eps;
        ma.doublet = eps != nullptr;
        launch_split<RES>(g, U, C, x, y, ma, nsys, b, st);
        return;
      }
      default: launch_variant<RES, 32, true, 192, 2>(g, U, C, x, y, mu, nsys, b, eps, st); return;
    }
  };
  launch(tune_variant(family, tune_key(g, nsys), NVARIANTS, [&] { return untuned_variant(g, nsys); }, may_tune, launch,
                      st));
}

bool dirac32_to_field(const Geom& g, int nsys) {
  const int v = peek_variant(g, nsys);
  return v == 0 || v == 2;
}

void launch_dirac32_field(const Geom& g, const float2* U, const float* C, const float* x, float* y, const double* mu,
                          int nsys, cudaStream_t st) {
  TM_PROF(st, "dirac_f32");
  const int nt = ntiles(nsys, 2);
  const bool wide = peek_variant(g, nsys) == 2;
  const int ty = pick_ty(nt, 32, wide ? 256 : 192);
  const dim3 block(32, ty), grid((unsigned)((g.V + 31) / 32), (unsigned)(nt / ty));
  static_assert(8 * 32 * 26 * 4 <= dr_stage_bytes(32), "eight warps transpose in the staging space");
  const auto kernel = wide ? dirac_kernel<32, false, true, 256, 2, true> : dirac_kernel<32, false, true, 192, 2, true>;
  func_smem_optin((const void*)kernel, dr_stage_bytes(32));
  kernel<<<grid, block, dr_stage_bytes(32), st>>>(U, C, x, y, mu, nsys, nt, g.L[0], g.L[1], g.L[2], g.L[3],
                                                  (float)g.bc_t, nullptr, nullptr);
  TM_COUNT();
}

bool dirac32_takes_values(const Geom& g, int nsys) {
  return nsys <= MASS_VALUES && peek_variant(g, nsys) == SPLIT_VARIANT;
}

void launch_dirac32_values(const Geom& g, const float2* U, const float* C, const float* x, float* y, const MassArgs& ma,
                           int nsys, cudaStream_t st) {
  TM_PROF(st, "dirac_f32");
  launch_split<false>(g, U, C, x, y, ma, nsys, nullptr, st);
}

template <>
void launch_dirac<float>(const Geom& g, const void* U, const float* C, const float* x, float* y, const double* mu,
                         int nsys, cudaStream_t st, const double* eps) {
  TM_PROF(st, "dirac_f32");
  launch_tuned<false>("dirac_f32", true, g, reinterpret_cast<const float2*>(U), C, x, y, mu, nsys, nullptr, eps, st);
}

void launch_residual32(const Geom& g, const float2* U, const float* C, const float* x, const float* b, float* r,
                       const double* mu, int nsys, cudaStream_t st, const double* eps) {
  TM_PROF(st, "residual_f32");
  // tuned only out of place (in place, b == r, the launch is not repeatable)
  launch_tuned<true>("residual_f32", b != r, g, U, C, x, r, mu, nsys, b, eps, st);
}

// ---------------------------------------------------------------- pack / unpack
// field: complex [nsys][V][12]; bundle: [ntile][12][V][2][T].
// One CTA transposes PK_SITES sites of one tile through shared memory, so that both sides are read and written in
// runs of whole lines (a thread per entry of the bundle used to touch the field in 8-byte pieces 96 bytes apart).
// Bound by HBM; one real per access, as neither side need be aligned to more than that. 20x12x28x44, 5 FP32
// systems (142 MB of field, 170 MB of bundle): pack 121 -> 53 us (5.9 TB/s), unpack 174 -> 58 us; 24^3x48,
// 12 FP64 systems: pack 1214 -> 492 us, unpack 2239 -> 481 us.
constexpr int PK_SITES = 128;
constexpr int PK_THREADS = 256;
constexpr int PK_PITCH = 26;  // reals per site in shared memory: 24, and 2 that keep the transposed access off the same banks
constexpr int PK_LANE = PK_SITES * PK_PITCH + 16;  // from one system of the tile to the next: 16 banks on

template <typename real>
__global__ void __launch_bounds__(PK_THREADS) pack_kernel(const real* __restrict__ f, real* __restrict__ b, int nsys,
                                                          int64_t V, int64_t nblk) {
  constexpr int T = Tile<real>::T;
  __shared__ real sm[T * PK_LANE];
  const int64_t tile = blockIdx.x / nblk, s0 = (blockIdx.x - tile * nblk) * PK_SITES;
  const int ns = (int)(V - s0 < PK_SITES ? V - s0 : PK_SITES);
  real v[T][PK_SITES * 24 / PK_THREADS];
#pragma unroll
  for (int l = 0; l < T; ++l) {
    const int64_t n = tile * T + l;
    const real* src = f + (n * V + s0) * 24;
#pragma unroll
    for (int r = 0; r < PK_SITES * 24 / PK_THREADS; ++r) {
      const int k = r * PK_THREADS + threadIdx.x;
      v[l][r] = n < nsys && k < ns * 24 ? src[k] : real(0);  // an absent system of the last tile is zero
    }
  }
#pragma unroll
  for (int l = 0; l < T; ++l)
#pragma unroll
    for (int r = 0; r < PK_SITES * 24 / PK_THREADS; ++r) {
      const int k = r * PK_THREADS + threadIdx.x;
      sm[l * PK_LANE + k + (PK_PITCH - 24) * (k / 24)] = v[l][r];
    }
  __syncthreads();
#pragma unroll 4
  for (int c = 0; c < 12; ++c) {
    real* dst = b + ((tile * 12 + c) * V + s0) * (2 * T);
    for (int k = threadIdx.x; k < ns * 2 * T; k += PK_THREADS)
      dst[k] = sm[(k % T) * PK_LANE + (k / (2 * T)) * PK_PITCH + 2 * c + (k / T) % 2];
  }
}

template <typename real>
__global__ void __launch_bounds__(PK_THREADS) unpack_kernel(const real* __restrict__ b, real* __restrict__ f, int nsys,
                                                            int64_t V, int64_t nblk) {
  constexpr int T = Tile<real>::T;
  constexpr int R = PK_SITES * 2 * T / PK_THREADS;  // accesses per thread and component
  __shared__ real sm[T * PK_LANE];
  const int64_t tile = blockIdx.x / nblk, s0 = (blockIdx.x - tile * nblk) * PK_SITES;
  const int ns = (int)(V - s0 < PK_SITES ? V - s0 : PK_SITES);
  real v[12][R];
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const real* src = b + ((tile * 12 + c) * V + s0) * (2 * T);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = r * PK_THREADS + threadIdx.x;
      v[c][r] = k < ns * 2 * T ? src[k] : real(0);
    }
  }
#pragma unroll
  for (int c = 0; c < 12; ++c)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int k = r * PK_THREADS + threadIdx.x;
      sm[(k % T) * PK_LANE + (k / (2 * T)) * PK_PITCH + 2 * c + (k / T) % 2] = v[c][r];
    }
  __syncthreads();
#pragma unroll
  for (int l = 0; l < T; ++l) {
    const int64_t n = tile * T + l;
    if (n >= nsys) break;
    real* dst = f + (n * V + s0) * 24;
#pragma unroll 4
    for (int k = threadIdx.x; k < ns * 24; k += PK_THREADS) dst[k] = sm[l * PK_LANE + k + (PK_PITCH - 24) * (k / 24)];
  }
}

template <typename real>
void launch_pack(const Geom& g, const real* field, real* bundle, int nsys, cudaStream_t st) {
  const int64_t nblk = (g.V + PK_SITES - 1) / PK_SITES;
  pack_kernel<real><<<(unsigned)(nblk * ntiles(nsys, Tile<real>::T)), PK_THREADS, 0, st>>>(field, bundle, nsys, g.V, nblk);
  TM_COUNT();
}

template <typename real>
void launch_unpack(const Geom& g, const real* bundle, real* field, int nsys, cudaStream_t st) {
  const int64_t nblk = (g.V + PK_SITES - 1) / PK_SITES;
  unpack_kernel<real><<<(unsigned)(nblk * ntiles(nsys, Tile<real>::T)), PK_THREADS, 0, st>>>(bundle, field, nsys, g.V, nblk);
  TM_COUNT();
}

template void launch_pack<float>(const Geom&, const float*, float*, int, cudaStream_t);
template void launch_pack<double>(const Geom&, const double*, double*, int, cudaStream_t);
template void launch_unpack<float>(const Geom&, const float*, float*, int, cudaStream_t);
template void launch_unpack<double>(const Geom&, const double*, double*, int, cudaStream_t);

}  // namespace tmamg

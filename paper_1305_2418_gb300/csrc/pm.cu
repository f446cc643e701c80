// pm.cu -- gravitational potential of the last particle solve on a periodic
// particle-mesh grid (Puchwein, Baldi & Springel 2013, Sec. 2.4, Eq. (30)):
//   lap_x phi = 4 pi G a^2 rho_bar (delta_pm - mean) = (3/2) Om H0^2 a^-1 (delta_pm - mean)
// with delta_pm the matter and/or effective-mass contrast assigned to the PM
// grid by volume overlap (amr.cu), x comoving in Mpc/h, H0 = 100 km/s per
// Mpc/h, phi in (km/s)^2.
//
// The 7-point periodic Poisson problem is solved by linear multigrid:
// red-black Gauss-Seidel smoothing, the residual restricted by the 8-daughter
// average, the coarse correction prolonged by the same linear reconstruction
// as the field solve, down to 4^3.  phi is held in FP64 and the residual in
// double-float; each V-cycle solves for the correction of phi in FP32
// (mg32.cuh, MG_POI), which for a linear problem is the FP64 V-cycle up to
// FP32's rounding of the correction, and the next residual holds what that
// leaves.  The FP64 pipe bounded the V-cycle in FP64 (7 FP64 instructions per
// cell and sweep, 24 us per half-sweep of 256^3 and its coarser grids, and
// half of every line read unused).  The periodic operator is singular: the right-hand side has
// its mean removed, and phi is returned with zero mean.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "amr.cuh"
#include "colour_split.cuh"
#include "dfloat.cuh"
#include "mg32.cuh"

namespace {

constexpr int BS = 256;
constexpr int PM_MAXL = 10;
constexpr double kPoissonScale = 1.5e4;  // (3/2) H0^2 with H0 = 100 km/s per Mpc/h

__device__ __forceinline__ unsigned cidx(unsigned i, unsigned j, unsigned k, int lg) {
  return (((i << lg) + j) << lg) + k;
}

__device__ __forceinline__ void pm_block_sum(double a, double* __restrict__ part) {
  __shared__ double w[BS / 32];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < BS / 32; ++q) s += w[q];
    part[blockIdx.x] = s;
  }
}

__device__ __forceinline__ double pm_resid(const double* __restrict__ phi,
                                           const double* __restrict__ rhs, int i, int j, int k,
                                           int lg, double ih2) {
  const int M = (1 << lg) - 1;
  const double c = phi[cidx(i, j, k, lg)];
  const double s = phi[cidx((i - 1) & M, j, k, lg)] + phi[cidx((i + 1) & M, j, k, lg)] +
                   phi[cidx(i, (j - 1) & M, k, lg)] + phi[cidx(i, (j + 1) & M, k, lg)] +
                   phi[cidx(i, j, (k - 1) & M, lg)] + phi[cidx(i, j, (k + 1) & M, lg)];
  return rhs[cidx(i, j, k, lg)] - (s - 6.0 * c) * ih2;
}

// Start of the cycles: phi = 0, r = rhs = scale (delta - mean) (in place) as
// double-float parts stored by colour, and the block sums of rhs^2.
__global__ void __launch_bounds__(BS) k_pm_start(double* __restrict__ rhs, int lg, double scale,
                                                 double mean, double* __restrict__ phi,
                                                 float* __restrict__ rh, float* __restrict__ rl,
                                                 double* __restrict__ part) {
  const unsigned n = 1u << (3 * lg);
  const int M = (1 << lg) - 1;
  double ss = 0.0;
  for (unsigned t = blockIdx.x * BS + threadIdx.x; t < n; t += gridDim.x * BS) {
    const double v = scale * (rhs[t] - mean);
    rhs[t] = v;
    phi[t] = 0.0;
    const dfl d = df_from_double_bits(v);
    const unsigned p = pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg);
    rh[p] = d.hi;
    rl[p] = d.lo;
    ss = fma(v, v, ss);
  }
  pm_block_sum(ss, part);
}

// r = rhs - lap phi in FP64 (the stopping test's last word, and the residual
// from which further cycles start), its parts and the block sums of r^2
__global__ void __launch_bounds__(BS) k_pm_resid(const double* __restrict__ phi,
                                                 const double* __restrict__ rhs, int lg,
                                                 double ih2, float* __restrict__ rh,
                                                 float* __restrict__ rl,
                                                 double* __restrict__ part) {
  const unsigned n = 1u << (3 * lg);
  const int M = (1 << lg) - 1;
  double ss = 0.0;
  for (unsigned t = blockIdx.x * BS + threadIdx.x; t < n; t += gridDim.x * BS) {
    const int k = (int)(t & M), j = (int)((t >> lg) & M), i = (int)(t >> (2 * lg));
    const double r = pm_resid(phi, rhs, i, j, k, lg, ih2);
    const dfl d = df_from_double_bits(r);
    const unsigned p = pdx(i, j, k, lg);
    rh[p] = d.hi;
    rl[p] = d.lo;
    ss = fma(r, r, ss);
  }
  pm_block_sum(ss, part);
}

// After a V-cycle: phi += e, r -= lap e in double-float, the block sums of r^2
// (FP32 over a thread's eight cells).  The differences e_j - e_c are exact, so
// r carries about 2^-46 of the correction's gradient terms: 3e-13 of the
// right-hand side on 1024^3, the size of the FP64 residual's own rounding.
// Eight cells of a row per thread; 36 bytes per cell.  (An FP64 residual pass
// costs 7 FP64 instructions per cell: 228 us on 256^3.)
__global__ void __launch_bounds__(BS) k_pm_update(double* __restrict__ phi,
                                                  const float* __restrict__ e,
                                                  float* __restrict__ rh, float* __restrict__ rl,
                                                  int lg, dfl ih2, double* __restrict__ part) {
  const unsigned half = 1u << (3 * lg - 1), nt = 1u << (3 * lg - 3);
  const int M = (1 << lg) - 1, hm = M >> 1;
  double ss = 0.0;
  for (unsigned t = blockIdx.x * BS + threadIdx.x; t < nt; t += gridDim.x * BS) {
    const int v = (int)(t & ((1u << (lg - 3)) - 1));
    const int j = (int)((t >> (lg - 3)) & M), i = (int)(t >> (2 * lg - 3));
    const int kh0 = 4 * v;
    const unsigned rc = prow(i, j, lg) + kh0;
    const unsigned rn[4] = {prow((i - 1) & M, j, lg) + kh0, prow((i + 1) & M, j, lg) + kh0,
                            prow(i, (j - 1) & M, lg) + kh0, prow(i, (j + 1) & M, lg) + kh0};
    const unsigned pe = ((i + j) & 1) ? half : 0u, po = half - pe;  // planes of even, odd k
    float z[10];  // e along the row: k0 - 1 .. k0 + 8
    {
      const float4 a = *reinterpret_cast<const float4*>(e + pe + rc);
      const float4 b = *reinterpret_cast<const float4*>(e + po + rc);
      z[0] = e[po + prow(i, j, lg) + ((kh0 - 1) & hm)];
      z[9] = e[pe + prow(i, j, lg) + ((kh0 + 4) & hm)];
      z[1] = a.x; z[3] = a.y; z[5] = a.z; z[7] = a.w;
      z[2] = b.x; z[4] = b.y; z[6] = b.z; z[8] = b.w;
    }
    double* pr = phi + ((((size_t)i << lg) + j) << lg) + 8 * v;
    float s8 = 0.f;
#pragma unroll
    for (int c = 0; c < 2; ++c) {  // the even, then the odd cells
      const unsigned own = c ? po : pe, oth = half - own;
      float x[4][4];
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const float4 a = *reinterpret_cast<const float4*>(e + oth + rn[d]);
        x[d][0] = a.x; x[d][1] = a.y; x[d][2] = a.z; x[d][3] = a.w;
      }
      const float4 h4 = *reinterpret_cast<const float4*>(rh + own + rc);
      const float4 l4 = *reinterpret_cast<const float4*>(rl + own + rc);
      float hi[4] = {h4.x, h4.y, h4.z, h4.w}, lo[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = 2 * q + c + 1;  // the cell's place in z
        const float ec = z[m];
        dfl s = df_two_sum(x[0][q], -ec);
        s = df_add_abs(s, df_two_sum(x[1][q], -ec));
        s = df_add_abs(s, df_two_sum(x[2][q], -ec));
        s = df_add_abs(s, df_two_sum(x[3][q], -ec));
        s = df_add_abs(s, df_two_sum(z[m - 1], -ec));
        s = df_add_abs(s, df_two_sum(z[m + 1], -ec));
        const dfl r = df_sub(dfl{hi[q], lo[q]}, df_mul(s, ih2));
        hi[q] = r.hi;
        lo[q] = r.lo;
        s8 = fmaf(r.hi, r.hi, s8);
      }
      *reinterpret_cast<float4*>(rh + own + rc) = make_float4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<float4*>(rl + own + rc) = make_float4(lo[0], lo[1], lo[2], lo[3]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double2 d = *reinterpret_cast<double2*>(pr + 2 * q);
      d.x += d_from_float_bits(z[2 * q + 1]);
      d.y += d_from_float_bits(z[2 * q + 2]);
      *reinterpret_cast<double2*>(pr + 2 * q) = d;
    }
    ss += (double)s8;
  }
  pm_block_sum(ss, part);
}

// per-block sums of x (a fixed tree per block, the blocks summed on the host
// in order)
__global__ void __launch_bounds__(BS) k_pm_sum(const double* __restrict__ x, long long n,
                                               double* __restrict__ part) {
  double a = 0.0;
  for (long long i = blockIdx.x * (long long)BS + threadIdx.x; i < n; i += (long long)gridDim.x * BS)
    a += x[i];
  pm_block_sum(a, part);
}

// y = scale * (x - shift)
__global__ void k_pm_affine(const double* __restrict__ x, long long n, double scale, double shift,
                            double* __restrict__ y) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] = scale * (x[i] - shift);
}

// g = -grad phi by central differences (periodic), one 32-byte record per cell
// of the three components as double-float pairs: the differences in FP64, the
// scaling in double-float
__global__ void __launch_bounds__(BS) k_pm_grad(const double* __restrict__ phi, int lg, dfl inv2h,
                                                float4* __restrict__ g) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg))) return;
  const int M = (1 << lg) - 1;
  const int k = (int)(t & M), j = (int)((t >> lg) & M), i = (int)(t >> (2 * lg));
  const double dx = phi[cidx((i - 1) & M, j, k, lg)] - phi[cidx((i + 1) & M, j, k, lg)];
  const double dy = phi[cidx(i, (j - 1) & M, k, lg)] - phi[cidx(i, (j + 1) & M, k, lg)];
  const double dz = phi[cidx(i, j, (k - 1) & M, lg)] - phi[cidx(i, j, (k + 1) & M, lg)];
  const dfl x = df_mul(df_from_double_bits(dx), inv2h), y = df_mul(df_from_double_bits(dy), inv2h),
            z = df_mul(df_from_double_bits(dz), inv2h);
  g[2 * (size_t)t] = make_float4(x.hi, x.lo, y.hi, y.lo);
  g[2 * (size_t)t + 1] = make_float4(z.hi, z.lo, 0.f, 0.f);
}

// cloud-in-cell interpolation of g (values at cell centres) to the particles:
// position t = x N / box - 1/2 in cell units (wrapped), the 8 cells around it
// with the product of the 1D linear weights.  Along each axis the value is
// a + w (b - a), in double-float: about 450 FP32 instructions against 60 on the
// FP64 pipe, an eighth of their issue time (1.61 ms for 16.8 M particles in
// FP64, its eight cells from three arrays).
__global__ void __launch_bounds__(BS) k_pm_cic(const double* __restrict__ pos, long long np, int lg,
                                               double inv_h, const float4* __restrict__ g,
                                               double* __restrict__ acc) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= np) return;
  const int M = (1 << lg) - 1;
  int i0[3];
  dfl w[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double t = pos[3 * p + a] * inv_h - 0.5;
    const double fl = floor(t);
    w[a] = df_from_double_bits(t - fl);
    i0[a] = (int)((long long)fl & M);
  }
  auto lerp = [](dfl a, dfl b, dfl f) { return df_add_abs(a, df_mul(f, df_add_abs(b, df_neg(a)))); };
  dfl vx[2], vy[2], vz[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    dfl ux[2], uy[2], uz[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const unsigned row = cidx((i0[0] + a) & M, (i0[1] + b) & M, 0, lg);
      const float4* g0 = g + 2 * (size_t)(row + i0[2]);
      const float4* g1 = g + 2 * (size_t)(row + ((i0[2] + 1) & M));
      const float4 p0 = __ldg(g0), p1 = __ldg(g1);
      const float2 q0 = __ldg(reinterpret_cast<const float2*>(g0 + 1)),
                   q1 = __ldg(reinterpret_cast<const float2*>(g1 + 1));
      ux[b] = lerp(dfl{p0.x, p0.y}, dfl{p1.x, p1.y}, w[2]);
      uy[b] = lerp(dfl{p0.z, p0.w}, dfl{p1.z, p1.w}, w[2]);
      uz[b] = lerp(dfl{q0.x, q0.y}, dfl{q1.x, q1.y}, w[2]);
    }
    vx[a] = lerp(ux[0], ux[1], w[1]);
    vy[a] = lerp(uy[0], uy[1], w[1]);
    vz[a] = lerp(uz[0], uz[1], w[1]);
  }
  acc[3 * p] = df_to_double_bits(lerp(vx[0], vx[1], w[0]));
  acc[3 * p + 1] = df_to_double_bits(lerp(vy[0], vy[1], w[0]));
  acc[3 * p + 2] = df_to_double_bits(lerp(vz[0], vz[1], w[0]));
}

// leapfrog: v += kick acc, x = wrap(x + drift v); each operation rounded on
// its own (no fused multiply-add), so the step is reproducible elsewhere
__global__ void __launch_bounds__(BS) k_kick_drift(double* __restrict__ pos, double* __restrict__ vel,
                                                   const double* __restrict__ acc, long long n3,
                                                   double kick, double drift, double box) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n3) return;
  const double v = __dadd_rn(vel[i], __dmul_rn(kick, acc[i]));
  vel[i] = v;
  double x = __dadd_rn(pos[i], __dmul_rn(drift, v));
  x = __dsub_rn(x, __dmul_rn(box, floor(__ddiv_rn(x, box))));
  if (!(x < box)) x = 0.0;  // rounding at the upper edge
  pos[i] = x;
}

struct PmWork {
  int lg = 0, nlev = 0;
  double h = 0.0;             // spacing of the finest grid
  long long n = 0;            // its cells
  double *phi = nullptr, *rhs = nullptr;  // finest grid, FP64
  float *e[PM_MAXL] = {}, *r[PM_MAXL] = {};  // correction and residual per level
  float* rlo = nullptr;       // low part of the finest residual
  float4* grad = nullptr;     // -grad phi of the finest level (force)
  double* part = nullptr;     // block sums (device)
  double* part_h = nullptr;   // block sums (page-locked host)
  int nparts = 0;
  bool solve_gone = false;    // only phi and the force's arrays are left
};

// what the solve needs beside phi; the next solve then starts from nothing
void pm_free_solve(PmWork* P) {
  auto drop = [](auto*& p) {
    if (p) cudaFree(p);
    p = nullptr;
  };
  drop(P->rhs), drop(P->rlo);
  for (int l = 0; l < PM_MAXL; ++l) drop(P->e[l]), drop(P->r[l]);
  P->solve_gone = true;
}

void pm_free_work(PmWork* P) {
  pm_free_solve(P);
  void* ps[] = {P->phi, P->grad, P->part};
  for (void* p : ps)
    if (p) cudaFree(p);
  if (P->part_h) cudaFreeHost(P->part_h);
  *P = PmWork();
}

mgfr_status pm_alloc(mgfr_ctx* c, PmWork* P, int lg, double box) {
  if (P->lg != lg || P->solve_gone) {
    pm_free_work(P);
    mgfr_status ps = mg32_prepare(c);
    if (ps != MGFR_OK) return ps;
    P->nlev = lg - 1;  // N ... 4
    P->n = 1LL << (3 * lg);
    MG_CK(c, dev_malloc(c, &P->phi, sizeof(double) * (size_t)P->n));
    MG_CK(c, dev_malloc(c, &P->rhs, sizeof(double) * (size_t)P->n));
    MG_CK(c, dev_malloc(c, &P->rlo, sizeof(float) * (size_t)P->n));
    for (int l = 0; l < P->nlev; ++l) {
      const size_t nl = (size_t)1 << (3 * (lg - l));
      MG_CK(c, dev_malloc(c, &P->e[l], sizeof(float) * nl));
      MG_CK(c, dev_malloc(c, &P->r[l], sizeof(float) * nl));
    }
    P->nparts = 152 * 8;
    MG_CK(c, dev_malloc(c, &P->part, sizeof(double) * (2 * P->nparts + 2)));
    MG_CK(c, cudaMallocHost(&P->part_h, sizeof(double) * P->nparts));
    P->lg = lg;
  }
  P->h = box / (double)(1LL << lg);
  return MGFR_OK;
}

// the block sums of the launch before, summed on the host in order
mgfr_status pm_total(mgfr_ctx* c, PmWork* P, int nb, double* sum) {
  c->launches += 1;
  MG_CK(c, cudaMemcpyAsync(P->part_h, P->part, sizeof(double) * nb, cudaMemcpyDeviceToHost, c->s));
  MG_CK(c, cudaStreamSynchronize(c->s));
  double a = 0.0;
  for (int q = 0; q < nb; ++q) a += P->part_h[q];
  *sum = a;
  return MGFR_OK;
}

}  // namespace

void pm_free(mgfr_ctx* c) {
  PmWork* P = (PmWork*)c->pm;
  if (!P) return;
  pm_free_work(P);
  delete P;
  c->pm = nullptr;
}

// The potential of Eq. (30) on the PM grid of level lpm, left (up to a constant)
// in the workspace's phi; phi_out (nullable) receives it with zero mean.  Runs after
// the caller's stream, on the context's stream; synchronises.
static mgfr_status pm_solve(mgfr_ctx* c, int lpm, int what, double* phi_out_dev,
                            double* dens_out_dev, mgfr_stats* st, PmWork** work) {
  int lg = 0;
  double om = 0.3, a = 1.0;
  mgfr_status rs = amr_density_pm(c, lpm, what, nullptr, &lg, &om, &a);
  if (rs != MGFR_OK) return rs;
  if (lg < 3) return set_err(c, MGFR_E_INVALID, "the PM grid needs at least 8 cells per axis");
  auto w0 = std::chrono::steady_clock::now();
  MG_CK(c, cudaSetDevice(c->device));
  if (st) std::memset(st, 0, sizeof(*st));
  c->launches = 0;
  if (!c->pm) c->pm = new PmWork();
  PmWork* P = (PmWork*)c->pm;
  const double box = ((AmrWork*)c->amr)->box;
  if ((rs = pm_alloc(c, P, lg, box)) != MGFR_OK) return rs;
  const mgfr_config& g = c->cfg;
  MG_CK(c, cudaEventRecord(c->ev_in, c->user));
  MG_CK(c, cudaStreamWaitEvent(c->s, c->ev_in, 0));
  MG_CK(c, cudaEventRecord(c->t0, c->s));
  // density contrast on the PM grid, then rhs = (3/2) Om H0^2 / a (delta - mean)
  if ((rs = amr_density_pm(c, lpm, what, P->rhs, nullptr, nullptr, nullptr)) != MGFR_OK) return rs;
  if (dens_out_dev)
    MG_CK(c, cudaMemcpyAsync(dens_out_dev, P->rhs, sizeof(double) * (size_t)P->n,
                             cudaMemcpyDeviceToDevice, c->s));
  const int nb = (int)std::min<long long>(P->nparts, (P->n + BS - 1) / BS);
  const int nb8 = (int)std::min<long long>(P->nparts, (P->n / 8 + BS - 1) / BS);
  const double ih2 = 1.0 / (P->h * P->h);
  double sum = 0.0, sq = 0.0;
  k_pm_sum<<<nb, BS, 0, c->s>>>(P->rhs, P->n, P->part);
  if ((rs = pm_total(c, P, nb, &sum)) != MGFR_OK) return rs;
  k_pm_start<<<nb, BS, 0, c->s>>>(P->rhs, lg, kPoissonScale * om / a, sum / (double)P->n, P->phi,
                                  P->r[0], P->rlo, P->part);
  if ((rs = pm_total(c, P, nb, &sq)) != MGFR_OK) return rs;
  Mg32Level L[PM_MAXL];
  for (int l = 0; l < P->nlev; ++l) {
    const double h = P->h * (double)(1 << l);
    L[l] = Mg32Level{lg - l, (float)(1.0 / (h * h)), (float)(h * h), P->e[l], P->r[l], nullptr};
  }
  Mg32Par par{};
  par.n_pre = g.n_pre;
  par.n_post = g.n_post;
  par.linear = 1;
  par.coarse_sweeps = 60;
  const double fn = std::sqrt(sq), target = g.tol_rel * fn;
  double r = fn, rho = 0.0;  // rho: reduction of the last cycle
  int it = 0;
  long long updates = 0;
  const bool pairs = (1 << lg) >= kPairMin && (1 << lg) <= kPairMax;
  auto cycle = [&]() {
    updates += mg32_cycle(MG_POI, L, P->nlev, par, c->s) + 60 * 64;
    c->launches += 10 * std::max(0, lg - 5) + 1;
  };
  while (r > target && it < g.max_vcycles) {
    MG_CK(c, cudaMemsetAsync(P->e[0], 0, sizeof(float) * (size_t)P->n, c->s));
    const double rp = r;
    int n = 1;
    cycle();
    if (pairs && it + 3 <= g.max_vcycles && pair_start(r, rho, target)) {
      mg32_norm(MG_POI, L[0], par, P->part, P->nparts, P->part + 2 * P->nparts, c->s);
      c->launches += 2;
      MG_CK(c, cudaMemcpyAsync(P->part_h, P->part + 2 * P->nparts, sizeof(double),
                               cudaMemcpyDeviceToHost, c->s));
      MG_CK(c, cudaStreamSynchronize(c->s));
      if (pair_on(r, std::sqrt(P->part_h[0]), target)) {
        cycle();
        n = 2;
      }
    }
    k_pm_update<<<nb8, BS, 0, c->s>>>(P->phi, P->e[0], P->r[0], P->rlo, lg, df_from_double(ih2),
                                      P->part);
    if ((rs = pm_total(c, P, nb8, &sq)) != MGFR_OK) return rs;
    r = std::sqrt(sq);
    it += n;
    rho = n == 2 ? std::sqrt(r / rp) : r / rp;
    if (!std::isfinite(r)) break;
    if (r <= target) {
      // the residual carried along says converged: the FP64 one decides
      k_pm_resid<<<nb, BS, 0, c->s>>>(P->phi, P->rhs, lg, ih2, P->r[0], P->rlo, P->part);
      if ((rs = pm_total(c, P, nb, &sq)) != MGFR_OK) return rs;
      r = std::sqrt(sq);
    }
  }
  if (phi_out_dev) {  // with zero mean
    k_pm_sum<<<nb, BS, 0, c->s>>>(P->phi, P->n, P->part);
    if ((rs = pm_total(c, P, nb, &sum)) != MGFR_OK) return rs;
    k_pm_affine<<<nblocks(P->n, BS), BS, 0, c->s>>>(P->phi, P->n, 1.0, sum / (double)P->n,
                                                    phi_out_dev);
    c->launches += 1;
  }
  MG_CK(c, cudaEventRecord(c->t1, c->s));
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaGetLastError());
  *work = P;
  if (st) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, c->t0, c->t1);
    st->vcycles = it;
    st->linear_updates = updates;
    st->res_l2_init = fn;
    st->res_l2_final = r;
    st->f_l2 = fn;
    st->t_solve_ms = ms;
    st->n_levels = 1;
    st->cells_per_level[0] = P->n;
    st->gpu_launches = c->launches;
    st->t_total_ms =
        std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - w0).count();
  }
  if (!(r <= target))
    return set_err(c, MGFR_E_NOCONVERGE, "PM Poisson solve did not reach the tolerance");
  return MGFR_OK;
}

static mgfr_status pm_finish(mgfr_ctx* c, mgfr_status rs) {
  MG_CK(c, cudaEventRecord(c->ev_out, c->s));
  MG_CK(c, cudaStreamWaitEvent(c->user, c->ev_out, 0));
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaGetLastError());
  return rs;
}

extern "C" mgfr_status mgfr_pm_potential(mgfr_ctx* c, int lpm, int what, double* phi_out_dev,
                                         double* dens_out_dev, mgfr_stats* st) {
  if (!c) return MGFR_E_INVALID;
  if (!phi_out_dev) return set_err(c, MGFR_E_INVALID, "phi_out_dev is required");
  PmWork* P = nullptr;
  mgfr_status rs = pm_solve(c, lpm, what, phi_out_dev, dens_out_dev, st, &P);
  if (rs != MGFR_OK && rs != MGFR_E_NOCONVERGE) return rs;
  return pm_finish(c, rs);
}

extern "C" mgfr_status mgfr_pm_accel(mgfr_ctx* c, int lpm, int what, const double* pos_dev,
                                     long long Np, double* acc_out_dev, mgfr_stats* st) {
  if (!c) return MGFR_E_INVALID;
  if (!pos_dev || !acc_out_dev || Np <= 0 || Np >= (1LL << 40))
    return set_err(c, MGFR_E_INVALID, "need positions and a force array of Np >= 1 particles");
  PmWork* P = nullptr;
  mgfr_status rs = pm_solve(c, lpm, what, nullptr, nullptr, st, &P);
  if (rs != MGFR_OK && rs != MGFR_E_NOCONVERGE) return rs;
  const size_t gb = 2 * sizeof(float4) * (size_t)P->n;
  if (!P->grad && dev_malloc(c, &P->grad, gb) != cudaSuccess) {
    // the force needs phi alone: the solve's other arrays make room (21 of the 32 bytes per
    // cell) and are made again by the next solve
    (void)cudaGetLastError();
    pm_free_solve(P);
    MG_CK(c, dev_malloc(c, &P->grad, gb));
  }
  k_pm_grad<<<nblocks(P->n, BS), BS, 0, c->s>>>(P->phi, P->lg, df_from_double(0.5 / P->h), P->grad);
  k_pm_cic<<<nblocks(Np, BS), BS, 0, c->s>>>(pos_dev, Np, P->lg, 1.0 / P->h, P->grad, acc_out_dev);
  c->launches += 2;
  if (st) st->gpu_launches = c->launches;
  return pm_finish(c, rs);
}

extern "C" mgfr_status mgfr_kick_drift(double* pos_dev, double* vel_dev, const double* acc_dev,
                                       long long Np, double kick, double drift, double box,
                                       void* cuda_stream) {
  if (!pos_dev || !vel_dev || !acc_dev || Np <= 0 || Np >= (1LL << 40) || !(box > 0.0) ||
      !std::isfinite(kick) || !std::isfinite(drift))
    return MGFR_E_INVALID;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  k_kick_drift<<<nblocks(3 * Np, BS), BS, 0, s>>>(pos_dev, vel_dev, acc_dev, 3 * Np, kick, drift,
                                                  box);
  if (cudaGetLastError() != cudaSuccess) return MGFR_E_CUDA;
  return MGFR_OK;
}

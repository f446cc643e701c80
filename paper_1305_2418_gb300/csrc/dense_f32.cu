// dense_f32.cu -- mixed-precision kernels for dense periodic levels.
//
// The FP32 V-cycles of both phases are in mg32.cu.  Here: phase B (defect
// correction) r = f - L(u) to FP64 accuracy on the FP64-accurate iterate, and
// u += e after the linearised system J(u) e = r (J the Jacobian of the
// discrete L) has been relaxed.  Solving the linearised correction in FP32
// avoids the ~1e-7 cancellation floor of a nonlinear FP32 correction.
#include <algorithm>

#include "colour_split.cuh"
#include "dfloat.cuh"
#include "mgfr_internal.cuh"

namespace {

constexpr int BS = 256;

// linear index of (i, j, k) on an N = 2^lg grid (N <= 1024: fits 32 bits)
__device__ __forceinline__ unsigned cidx(int i, int j, int k, int lg) {
  return ((((unsigned)i << lg) + (unsigned)j) << lg) + (unsigned)k;
}

__device__ __forceinline__ void block_partial(double ss, double mx, double* __restrict__ partials) {
  __shared__ double s1[BS / 32], s2[BS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s1[threadIdx.x >> 5] = ss;
    s2[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) {
      a += s1[w];
      b = fmax(b, s2[w]);
    }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = b;
  }
}

// C-order FP64 -> colour-split FP32
__global__ void k_from64(const double* __restrict__ x, float* __restrict__ y, int lg) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg))) return;
  const int M = (1 << lg) - 1;
  y[pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg)] = f_from_double_bits(x[t]);
}

// FP32 iterate -> double-float iterate and its e^u (start of phase B)
__global__ void k_to_df(const float* __restrict__ u32, dfl* __restrict__ u, dfl* __restrict__ E,
                        int lg) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg))) return;
  const int M = (1 << lg) - 1;
  const dfl v{u32[pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg)], 0.f};
  u[t] = v;
  E[t] = df_exp(v);
}

// ---- Phase B ---------------------------------------------------------------
// Model constants as double-float pairs (phase B in double-float)
struct DFM {
  dfl aRt, inv_np1, ih2h;  // alpha Rt, 1/(n+1), 1/(2 h^2)
  int n;
};

// two consecutive pairs
__device__ __forceinline__ void ld2df(const dfl* __restrict__ p, unsigned q, dfl* x) {
  const float4 a = *reinterpret_cast<const float4*>(p + q);
  x[0] = dfl{a.x, a.y};
  x[1] = dfl{a.z, a.w};
}

// r = f - L(u) to FP64 accuracy in double-float on the FP32 pipes (u, E, f
// held as hi + lo pairs); stores r and u rounded to FP32, zeroes the
// correction e, and accumulates the norms (FP32 within a thread).
//
// Bound by the FP32 arithmetic: a thread takes the cells (i, 2J..2J+1, 2K..2K+1), so
// that the four faces between them are formed once (5 per cell instead of 6) and the
// rows are read as 16-byte vectors (6 loads per cell and array pair instead of 14), with
// registers for all loads of an iteration in flight: one cell per thread, 446
// instructions at 59% of the issue rate with 32 registers, took 333 us on 256^3, this one
// 190 (64 registers and a spill: 201).
__global__ void __launch_bounds__(BS, 3) k_resid_df(const dfl* __restrict__ u,
                                                    const dfl* __restrict__ E,
                                                    const dfl* __restrict__ f, int lg, DFM m,
                                                    float* __restrict__ r32,
                                                    float* __restrict__ u32,
                                                    float* __restrict__ e32,
                                                    double* __restrict__ partials) {
  const int M = (1 << lg) - 1, H = M >> 1;
  const unsigned n4 = 1u << (3 * lg - 2);
  float ss = 0.f, mx = 0.f;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < n4;
       t += gridDim.x * blockDim.x) {
    const int k = 2 * (int)(t & H), j = 2 * (int)((t >> (lg - 1)) & H), i = (int)(t >> (2 * lg - 2));
    const unsigned c[2] = {cidx(i, j, k, lg), cidx(i, j + 1, k, lg)};
    // by row b and place q; [side]: the rows across the x faces, the y rows, the z cells
    dfl uc[2][2], Ec[2][2], ux[2][2][2], Ex[2][2][2], uy[2][2], Ey[2][2], uz[2][2], Ez[2][2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      ld2df(u, c[b], uc[b]);
      ld2df(E, c[b], Ec[b]);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const unsigned x = cidx((i + 2 * s - 1) & M, j + b, k, lg);
        ld2df(u, x, ux[s][b]);
        ld2df(E, x, Ex[s][b]);
        const unsigned z = cidx(i, j + b, (k + 3 * s - 1) & M, lg);
        uz[s][b] = u[z];
        Ez[s][b] = E[z];
      }
      const unsigned y = cidx(i, (j + 3 * b - 1) & M, k, lg);
      ld2df(u, y, uy[b]);
      ld2df(E, y, Ey[b]);
    }
    dfl acc[2][2];  // the faces in the order -x, +x, -y, +y, -z, +z
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int b = 0; b < 2; ++b)
        acc[b][q] = df_add_abs(df_face(Ex[0][b][q], Ec[b][q], ux[0][b][q], uc[b][q]),
                               df_face(Ex[1][b][q], Ec[b][q], ux[1][b][q], uc[b][q]));
      const dfl F = df_face(Ec[1][q], Ec[0][q], uc[1][q], uc[0][q]);
      acc[0][q] = df_add_abs(acc[0][q], df_face(Ey[0][q], Ec[0][q], uy[0][q], uc[0][q]));
      acc[0][q] = df_add_abs(acc[0][q], F);
      acc[1][q] = df_add_abs(acc[1][q], df_neg(F));
      acc[1][q] = df_add_abs(acc[1][q], df_face(Ey[1][q], Ec[1][q], uy[1][q], uc[1][q]));
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const dfl F = df_face(Ec[b][1], Ec[b][0], uc[b][1], uc[b][0]);
      acc[b][0] = df_add_abs(acc[b][0], df_face(Ez[0][b], Ec[b][0], uz[0][b], uc[b][0]));
      acc[b][0] = df_add_abs(acc[b][0], F);
      acc[b][1] = df_add_abs(acc[b][1], df_neg(F));
      acc[b][1] = df_add_abs(acc[b][1], df_face(Ez[1][b], Ec[b][1], uz[1][b], uc[b][1]));
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      dfl fv[2];
      ld2df(f, c[b], fv);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const dfl sN =
            m.n == 1 ? df_rsqrt(Ec[b][q]) : df_exp(df_neg(df_mul(uc[b][q], m.inv_np1)));
        const dfl L = df_add(df_mul(acc[b][q], m.ih2h), df_mul(m.aRt, df_add_f(df_neg(sN), 1.f)));
        const dfl r = df_sub(fv[q], L);
        const unsigned p = pdx(i, j + b, k + q, lg);
        r32[p] = r.hi;
        u32[p] = uc[b][q].hi;
        e32[p] = 0.f;
        ss = fmaf(r.hi, r.hi, ss);
        mx = fmaxf(mx, fabsf(r.hi));
      }
    }
  }
  block_partial((double)ss, (double)mx, partials);
}

__global__ void k_apply_corr(dfl* __restrict__ u, dfl* __restrict__ E, const float* __restrict__ e,
                             int lg, float cap) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg))) return;
  const int M = (1 << lg) - 1;
  const float et = e[pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg)];
  const dfl v = df_add_f(u[t], fminf(fmaxf(et, -cap), cap));
  u[t] = v;
  E[t] = df_exp(v);
}

__global__ void k_d2df(const double* __restrict__ x, dfl* __restrict__ y, long long n) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    const double v = x[t];
    y[t] = df_from_double_bits(v);
  }
}
__global__ void k_df2d(const dfl* __restrict__ x, double* __restrict__ y, long long n) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    const dfl v = x[t];
    y[t] = df_to_double_bits(v);
  }
}

// an FP64 iterate (in place) -> double-float pairs, and e^u as pairs
__global__ void k_d2df_exp(dfl* __restrict__ u, dfl* __restrict__ E, long long n) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    const dfl v = df_from_double_bits(reinterpret_cast<const double*>(u)[t]);
    u[t] = v;
    E[t] = df_exp(v);
  }
}

__global__ void k_finish32(const double* __restrict__ partials, int nparts, double* __restrict__ out) {
  __shared__ double s1[256], s2[256];
  double a = 0.0, b = 0.0;
  for (int q = threadIdx.x; q < nparts; q += blockDim.x) {
    a += partials[2 * q];
    b = fmax(b, partials[2 * q + 1]);
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      s1[threadIdx.x] += s1[threadIdx.x + w];
      s2[threadIdx.x] = fmax(s2[threadIdx.x], s2[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = s1[0];
    out[1] = s2[0];
  }
}

}  // namespace

namespace f32 {

void from64(const double* x, float* y, const DenseLevel& L, cudaStream_t s) {
  k_from64<<<nblocks(L.n, BS), BS, 0, s>>>(x, y, L.lg);
}
void to_df(DenseLevel& L, cudaStream_t s) {
  k_to_df<<<nblocks(L.n, BS), BS, 0, s>>>(L.u32, reinterpret_cast<dfl*>(L.u),
                                          reinterpret_cast<dfl*>(L.E), L.lg);
}
void f_to_df(const double* f, double* fdf, long long n, cudaStream_t s) {
  k_d2df<<<nblocks(n, BS), BS, 0, s>>>(f, reinterpret_cast<dfl*>(fdf), n);
}
void fp64_to_df(DenseLevel& L, cudaStream_t s) {
  k_d2df_exp<<<nblocks(L.n, BS), BS, 0, s>>>(reinterpret_cast<dfl*>(L.u), reinterpret_cast<dfl*>(L.E),
                                             L.n);
}
void state_to_fp64(DenseLevel& L, cudaStream_t s) {
  k_df2d<<<nblocks(L.n, BS), BS, 0, s>>>(reinterpret_cast<const dfl*>(L.u), L.u, L.n);
  k_df2d<<<nblocks(L.n, BS), BS, 0, s>>>(reinterpret_cast<const dfl*>(L.E), L.E, L.n);
}

void resid_df(DenseLevel& L, const double* fdf, const Model& m, double* partials, int nparts,
              double* out, cudaStream_t s) {
  int nb = (int)std::min<long long>(nparts, nblocks(L.n / 4, BS));
  const DFM dm{df_from_double(m.aRt), df_from_double(m.inv_np1), df_from_double(0.5 * L.ih2),
               m.n};
  k_resid_df<<<nb, BS, 0, s>>>(reinterpret_cast<const dfl*>(L.u), reinterpret_cast<const dfl*>(L.E),
                               reinterpret_cast<const dfl*>(fdf), L.lg, dm, L.r32, L.u32, L.e32,
                               partials);
  k_finish32<<<1, 256, 0, s>>>(partials, nb, out);
}
void apply_corr(DenseLevel& L, double cap, cudaStream_t s) {
  k_apply_corr<<<nblocks(L.n, BS), BS, 0, s>>>(reinterpret_cast<dfl*>(L.u),
                                               reinterpret_cast<dfl*>(L.E), L.e32, L.lg, (float)cap);
}

}  // namespace f32

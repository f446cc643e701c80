// unet.cu -- learned initial guess for the field solve: a 4-level 3D U-Net
// (16/32/64/128 channels, 3^3 kernels, circular padding) with BF16 weights
// and activations and FP32 accumulation, trained and evaluated on the GPU by
// this library's own kernels (the tcgen05 convolutions of nn_tc.cu, the
// mma.sync ones of nn_conv.cu for other channel pairs, the elementwise
// kernels here).
//
// Input features per voxel: ln(1 + delta), log10|fR0| + 5, 1 and the local
// screening value -(n+1) ln(1 + Om delta / Rt) (padded to 16 channels; the
// boxes are at a = 1).  Output: v = asinh(u / 0.01) (FP32), u = 0.01 sinh(v).
// Encoder: two conv+ReLU per level, 2^3 average pooling.  Decoder: nearest
// upsampling, concatenation with the encoder output of the same level, two
// conv+ReLU.  Head: 1x1x1 conv to 1 channel.  Loss: mean squared error in v.
// Optimiser: Adam on FP32 master weights, BF16 copies used by the
// convolutions.
//
// The network is fully convolutional, so it applies to any power-of-two box
// of 32 to 512 cells per side at the cell size it was trained on.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <random>
#include <vector>

#include "lean_fp64.cuh"
#include "nn_kernels.cuh"

namespace {

constexpr int BS = 256;

struct ConvSpec {
  int cin, cout, lvl;  // level 0 = full resolution
};

// 14 convolutions in execution order
const ConvSpec kConvs[14] = {
    {16, 16, 0},  {16, 16, 0},                       // enc1
    {16, 32, 1},  {32, 32, 1},                       // enc2
    {32, 64, 2},  {64, 64, 2},                       // enc3
    {64, 128, 3}, {128, 128, 3},                     // bottom
    {192, 64, 2}, {64, 64, 2},                       // dec3 (up 128 + enc3 64)
    {96, 32, 1},  {32, 32, 1},                       // dec2 (up 64 + enc2 32)
    {48, 16, 0},  {16, 16, 0},                       // dec1 (up 32 + enc1 16)
};

// features: ln(1+delta), log10|fR0| + 5, 1, and the local screening value
// u_scr = -(n+1) ln(1 + Om a^-3 delta / Rt) (the solution where delta is
// uniform on scales beyond the Compton length), clamped to [-20, 5], in the
// output's own variable: asinh(u_scr / 0.01) / 5 (of order one).
constexpr double U_SCALE_F = 0.01;  // the output variable's scale (U_SCALE below)

// the features in FP64 throughout (bf16 of the FP32-rounded value)
__device__ __noinline__ void features64(double d, double scr, double np1, __nv_bfloat16* ln,
                                        __nv_bfloat16* scv) {
  *ln = __float2bfloat16((float)log(fmax(1.0 + d, 1e-3)));
  const double ul = fmin(fmax(-np1 * log(fmax(1.0 + scr * d, 1e-6)), -20.0), 5.0);
  *scv = __float2bfloat16((float)(asinh(ul / U_SCALE_F) / 5.0));
}

// whether an FP32 value accurate to 8 ulp decides its rounding to bf16: it is
// further than 12 ulp from the midpoint of two bf16 values
__device__ __forceinline__ bool bf16_decided(float v) {
  const int low = (int)(__float_as_uint(v) & 0xffffu) - 0x8000;
  return low > 12 || low < -12;
}

// ln(max(1 + y, lo)) of the FP64 sum 1 + y to a few FP32 ulp: log1pf of what the
// sum kept of y where 1 + y is near 1
__device__ __forceinline__ float ln1p(double y, float lo) {
  const double x = 1.0 + y;
  const float yf = f_from_double_bits(x - 1.0);
  return fabsf(yf) < 0.5f ? log1pf(yf) : logf(fmaxf(f_from_double_bits(x), lo));
}

__global__ void k_fr0_feature(const double* __restrict__ fr0s, int B,
                              __nv_bfloat16* __restrict__ out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) out[b] = __float2bfloat16((float)(log10(fr0s[b]) + 5.0));
}

// The features are bf16: FP32 functions (log1pf, logf and asinhf, each within a
// few ulp, 8 at most together) decide them except within 12 FP32 ulp of a rounding midpoint (one
// value in 2700), where the FP64 form decides, so the result is that of FP64
// everywhere.  Memory bound (40 bytes per voxel); the FP64 functions took 5.2 ms
// for 256^3.
__global__ void __launch_bounds__(BS) k_features(const double* __restrict__ delta,
                                                 const __nv_bfloat16* __restrict__ ffr0, int lg3,
                                                 long long M, __nv_bfloat16* __restrict__ x,
                                                 double scr, double np1, double dscale) {
  const long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (m >= M) return;
  const double d = dscale * delta[m];
  const float l = ln1p(d, 1e-3f);
  const float ul =
      fminf(fmaxf(-(float)np1 * ln1p(scr * d, 1e-6f), -20.f), 5.f);
  const float a = asinhf(ul * (float)(1.0 / U_SCALE_F)) * 0.2f;
  __nv_bfloat16 ln = __float2bfloat16(l), sc = __float2bfloat16(a);
  if (!(bf16_decided(l) && bf16_decided(a))) features64(d, scr, np1, &ln, &sc);
  auto bits = [](__nv_bfloat16 v) { return (unsigned)__bfloat16_as_ushort(v); };
  uint4* o = reinterpret_cast<uint4*>(x + m * 16);
  o[0] = make_uint4(bits(ln) | (bits(ffr0[m >> lg3]) << 16),
                    bits(__float2bfloat16(1.f)) | (bits(sc) << 16), 0u, 0u);
  o[1] = make_uint4(0u, 0u, 0u, 0u);
}

// ---- elementwise kernels on 8-channel (16-byte BF16, 32-byte FP32) chunks; a
// thread's chunk index is e = voxel (C/8) + chunk, C/8 a power of two ----------
struct B8 {
  float v[8];
};
__device__ __forceinline__ B8 ldb8(const __nv_bfloat16* p) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const unsigned w[4] = {q.x, q.y, q.z, q.w};
  B8 r;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r.v[2 * i] = __uint_as_float(w[i] << 16);
    r.v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
  return r;
}
__device__ __forceinline__ uint4 packb8(const float* v) {
  unsigned w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    w[i] = (unsigned)__bfloat16_as_ushort(__float2bfloat16(v[2 * i])) |
           ((unsigned)__bfloat16_as_ushort(__float2bfloat16(v[2 * i + 1])) << 16);
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ B8 ldf8(const float* p) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  return B8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
__device__ __forceinline__ void stf8(float* p, const B8& x) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x.v[4], x.v[5], x.v[6], x.v[7]);
}
// daughter q of coarse voxel mc (grid 2^lgc), parent of fine voxel mf (2^lgf)
__device__ __forceinline__ unsigned daughter(unsigned mc, int lgc, int q) {
  const unsigned Mc = (1u << lgc) - 1;
  const unsigned K = mc & Mc, J = (mc >> lgc) & Mc, bI = mc >> (2 * lgc);  // sample and I
  return (((2 * bI + (q >> 2)) << (lgc + 1)) + 2 * J + ((q >> 1) & 1) << (lgc + 1)) + 2 * K +
         (q & 1);
}
__device__ __forceinline__ unsigned parent(unsigned mf, int lgf) {
  const unsigned Mf = (1u << lgf) - 1;
  const unsigned k = mf & Mf, j = (mf >> lgf) & Mf, bi = mf >> (2 * lgf);
  return (((bi >> 1) << (lgf - 1)) + (j >> 1) << (lgf - 1)) + (k >> 1);
}

// 2^3 average pooling: y[M'][c] from x (full res, view)
__global__ void __launch_bounds__(BS) k_pool(TView x, TView y, int lc8, int lgDc, long long n) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const unsigned mc = (unsigned)(e >> lc8);
  const int c = 8 * (int)(e & ((1 << lc8) - 1));
  float s[8] = {};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const B8 v = ldb8(x.p + (size_t)daughter(mc, lgDc, q) * x.ld + x.off + c);
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] += v.v[i];
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) s[i] *= 0.125f;
  *reinterpret_cast<uint4*>(y.p + (size_t)mc * y.ld + y.off + c) = packb8(s);
}

// g_fine[child][c] += g_coarse[parent][c] / 8
__global__ void __launch_bounds__(BS) k_pool_bwd(FView gc, FView gf, int lc8, int lgDf,
                                                 long long n) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const unsigned mf = (unsigned)(e >> lc8);
  const int c = 8 * (int)(e & ((1 << lc8) - 1));
  const B8 g = ldf8(gc.p + (size_t)parent(mf, lgDf) * gc.ld + gc.off + c);
  float* q = gf.p + (size_t)mf * gf.ld + gf.off + c;
  B8 v = ldf8(q);
#pragma unroll
  for (int i = 0; i < 8; ++i) v.v[i] += 0.125f * g.v[i];
  stf8(q, v);
}

// nearest upsampling: y[fine][c] = x[parent][c] (one channel per thread took
// 2.7 ms for the three levels of a 256^3 box)
__global__ void __launch_bounds__(BS) k_up(TView x, TView y, int lc8, int lgDf, long long n) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const unsigned mf = (unsigned)(e >> lc8);
  const int c = 8 * (int)(e & ((1 << lc8) - 1));
  *reinterpret_cast<uint4*>(y.p + (size_t)mf * y.ld + y.off + c) =
      *reinterpret_cast<const uint4*>(x.p + (size_t)parent(mf, lgDf) * x.ld + x.off + c);
}

// g_coarse[parent][c] = sum of the 8 children's gradients
__global__ void __launch_bounds__(BS) k_up_bwd(FView gf, FView gc, int lc8, int lgDc,
                                               long long n) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const unsigned mc = (unsigned)(e >> lc8);
  const int c = 8 * (int)(e & ((1 << lc8) - 1));
  B8 s{};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const B8 v = ldf8(gf.p + (size_t)daughter(mc, lgDc, q) * gf.ld + gf.off + c);
#pragma unroll
    for (int i = 0; i < 8; ++i) s.v[i] += v.v[i];
  }
  stf8(gc.p + (size_t)mc * gc.ld + gc.off + c, s);
}

// gradient of the pre-activation: g * (y > 0), to BF16, contiguous [M][C], and
// the bias gradient's partial sums over this block's voxels (of the BF16
// values; part [block][C]).  The grid stride is a multiple of C/8, so a thread
// keeps its channels; the block's threads of a channel group are added in a
// fixed order.
__global__ void __launch_bounds__(BS) k_relu_bwd(FView g, TView y, int lc8, long long n,
                                                 __nv_bfloat16* __restrict__ out,
                                                 float* __restrict__ part) {
  __shared__ float red[8][BS];
  float s[8] = {};
  for (long long e = blockIdx.x * (long long)BS + threadIdx.x; e < n;
       e += (long long)gridDim.x * BS) {
    const size_t m = (size_t)(e >> lc8);
    const int c = 8 * (int)(e & ((1 << lc8) - 1));
    const B8 yy = ldb8(y.p + m * y.ld + y.off + c);
    B8 gg = ldf8(g.p + m * g.ld + g.off + c);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      gg.v[i] = __bfloat162float(__float2bfloat16(yy.v[i] > 0.f ? gg.v[i] : 0.f));
      s[i] += gg.v[i];
    }
    *reinterpret_cast<uint4*>(out + 8 * e) = packb8(gg.v);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) red[i][threadIdx.x] = s[i];
  __syncthreads();
  const int ng = 1 << lc8;  // channel groups; group of thread t: t & (ng - 1)
  for (int w = BS / 2; w >= ng; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int i = 0; i < 8; ++i) red[i][threadIdx.x] += red[i][threadIdx.x + w];
    __syncthreads();
  }
  if ((int)threadIdx.x < ng)
#pragma unroll
    for (int i = 0; i < 8; ++i)
      part[(size_t)blockIdx.x * 8 * ng + 8 * threadIdx.x + i] = red[i][threadIdx.x];
}

__global__ void __launch_bounds__(BS) k_head_fwd(TView x, const float* __restrict__ w, long long M,
                                                 float* __restrict__ out) {
  const long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (m >= M) return;
  float s = w[16];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const B8 v = ldb8(x.p + m * x.ld + x.off + 8 * h);
#pragma unroll
    for (int c = 0; c < 8; ++c) s = fmaf(w[8 * h + c], v.v[c], s);
  }
  out[m] = s;
}

// The network works in v = asinh(u / U_SCALE): linear for |u| << U_SCALE,
// logarithmic beyond, so weakly and strongly screened fields (|u| from 1e-3
// to ~10) have comparable weight in the loss.
constexpr double U_SCALE = 0.01;

// asinh(x): the FP32 value y, then one Newton step on sinh y = x with sinh y
// from two FP64 exponentials (24 FP64 instructions against about 100); the
// step's relative error 1e-7 leaves 1e-14
__device__ __forceinline__ double asinh_lean(double x) {
  const float yf = asinhf(f_from_double_bits(x));
  if (!(fabsf(yf) < 80.f)) return asinh(x);
  const double y = d_from_float_bits(yf), e = lean_exp(y), ei = lean_exp(-y);
  const float d = f_from_double_bits(fma(0.5, ei - e, x));  // x - sinh y
  return y + d_from_float_bits(d / coshf(yf));
}

// loss partials (in v) and d loss / d out = 2 (out - v) / M
__global__ void k_mse(const float* __restrict__ out, const double* __restrict__ target, long long M,
                      double gscale, float* __restrict__ gout, double* __restrict__ partial) {
  __shared__ double red[BS];
  double s = 0.0;
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < M;
       m += (long long)gridDim.x * blockDim.x) {
    const double d = d_from_float_bits(out[m]) - asinh_lean(target[m] * (1.0 / U_SCALE));
    s = fma(d, d, s);
    gout[m] = f_from_double_bits(d * gscale);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = BS / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_head_bwd(TView x, const float* __restrict__ w, const float* __restrict__ gout,
                           long long M, FView gx, float* __restrict__ gw_part) {
  __shared__ float red[17][BS / 32];
  float acc[17];
  for (int c = 0; c < 17; ++c) acc[c] = 0.f;
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < M;
       m += (long long)gridDim.x * blockDim.x) {
    const float g = gout[m];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const B8 v = ldb8(x.p + m * x.ld + x.off + 8 * h);
      B8 o;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        acc[8 * h + c] = fmaf(g, v.v[c], acc[8 * h + c]);
        o.v[c] = g * w[8 * h + c];
      }
      stf8(gx.p + m * gx.ld + gx.off + 8 * h, o);
    }
    acc[16] += g;
  }
  for (int c = 0; c < 17; ++c) {
    float v = acc[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 17) {
    float s = 0.f;
    for (int q = 0; q < BS / 32; ++q) s += red[threadIdx.x][q];
    gw_part[blockIdx.x * 17 + threadIdx.x] = s;
  }
}

__global__ void k_sum_parts(const float* __restrict__ part, int nparts, int n, float* __restrict__ out) {
  const int i = threadIdx.x;
  if (i >= n) return;
  float s = 0.f;
  for (int q = 0; q < nparts; ++q) s += part[q * n + i];
  out[i] = s;
}

// Adam (bias-corrected), then refresh the BF16 copies of conv weights
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, long long n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float a = b1 * m1[i] + (1.f - b1) * gi;
  const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = b;
  p[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}

// The BF16 copies of the 14 convolutions' weights: as they are, and packed for
// the tensor-core forward and input gradient (nn_tc_pack's layouts); one launch
// for all (42 launches took 140 us of a training step).
struct PackTab {
  long long woff[14], boff[15];  // FP32 parameters, BF16 offsets (boff[14]: the end)
  int cin[14], cout[14];
};
__global__ void __launch_bounds__(BS) k_refresh(const float* __restrict__ P, PackTab T,
                                                __nv_bfloat16* __restrict__ Wbf,
                                                __nv_bfloat16* __restrict__ Wtf,
                                                __nv_bfloat16* __restrict__ Wtd) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= T.boff[14]) return;
  int i = 0;
#pragma unroll
  for (int q = 1; q < 14; ++q) i += e >= T.boff[q] ? 1 : 0;
  const unsigned r = (unsigned)(e - T.boff[i]), ci_n = T.cin[i], co_n = T.cout[i];
  const unsigned co = r % co_n, ci = (r / co_n) % ci_n, t = r / (co_n * ci_n);
  const __nv_bfloat16 v = __float2bfloat16(P[T.woff[i] + r]);
  Wbf[e] = v;
  const unsigned per = ci_n * co_n;
  // forward: [t][ci / 8][co][ci & 7]; input gradient: [t][co / 8][ci][co & 7]
  Wtf[T.boff[i] + t * per + ((ci >> 3) * co_n + co) * 8 + (ci & 7)] = v;
  Wtd[T.boff[i] + t * per + ((co >> 3) * ci_n + ci) * 8 + (co & 7)] = v;
}

// u = U_SCALE sinh(v)
__global__ void k_out_to_double(const float* __restrict__ x, double* __restrict__ y, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] = U_SCALE * sinh((double)x[i]);
}

}  // namespace

// ============================================================================
static int lg_of(int D) {
  int lg = 0;
  while ((1 << lg) < D) ++lg;
  return lg;
}

constexpr int kBiasBlocks = 152 * 8;  // blocks of k_relu_bwd

struct UNet {
  // parameter layout in one flat FP32 array: per conv W[27][cin][cout], b[cout]; head w[16], b
  long long woff[14], boff[14], head_off = 0, nparam = 0;
  long long wbf_off[14], nwbf = 0;
  float *P = nullptr, *G = nullptr, *M1 = nullptr, *M2 = nullptr;  // device
  __nv_bfloat16* Wbf = nullptr;
  // the BF16 weights packed for the tensor-core forward and input-gradient
  // convolutions (same offsets as Wbf), and their kernels' error word
  __nv_bfloat16 *Wtf = nullptr, *Wtd = nullptr;
  int* tc_err = nullptr;
  long long step = 0;
  // activation buffers for one (B, lgD)
  int B = 0, lgD = 0;
  std::vector<void*> bufs;
  __nv_bfloat16 *X0, *E1a, *CAT1, *P1, *E2a, *CAT2, *P2, *E3a, *CAT3, *P3, *Ba, *Bb, *D3a, *D3b,
      *D2a, *D2b, *D1a, *D1b, *Gpre;
  float *OUT, *GOUT, *G_E1a, *G_CAT1, *G_P1, *G_E2a, *G_CAT2, *G_P2, *G_E3a, *G_CAT3, *G_P3, *G_Ba,
      *G_Bb, *G_D3a, *G_D3b, *G_D2a, *G_D2b, *G_D1a, *G_D1b, *wpart, *bpart;
  __nv_bfloat16* ffr0 = nullptr;  // the feature log10|fR0| + 5 per sample
  double* fr0d = nullptr;
  double* lossp = nullptr;
  long long wpart_n = 0;
};

static void unet_free_bufs(UNet* U) {
  for (void* p : U->bufs) cudaFree(p);
  U->bufs.clear();
  U->B = U->lgD = 0;
}

void unet_free(mgfr_ctx* c) {
  UNet* U = (UNet*)c->unet;
  if (!U) return;
  unet_free_bufs(U);
  void* ps[] = {U->P, U->G, U->M1, U->M2, U->Wbf, U->Wtf, U->Wtd, U->tc_err};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete U;
  c->unet = nullptr;
}

static mgfr_status unet_alloc(mgfr_ctx* c, UNet* U, int B, int lgD) {
  if (U->B == B && U->lgD == lgD) return MGFR_OK;
  unet_free_bufs(U);
  const long long M0 = (long long)B << (3 * lgD), M1 = M0 >> 3, M2 = M1 >> 3, M3 = M2 >> 3;
  bool ok = true;
  auto bytes = [&](size_t n) -> void* {
    void* p = nullptr;
    ok = ok && dev_malloc(c, &p, n) == cudaSuccess;
    if (p) U->bufs.push_back(p);
    return p;
  };
  auto bf = [&](long long n) { return (__nv_bfloat16*)bytes(sizeof(__nv_bfloat16) * (size_t)n); };
  auto f = [&](long long n) { return (float*)bytes(sizeof(float) * (size_t)n); };
  U->X0 = bf(M0 * 16);
  U->E1a = bf(M0 * 16);
  U->CAT1 = bf(M0 * 48);
  U->P1 = bf(M1 * 16);
  U->E2a = bf(M1 * 32);
  U->CAT2 = bf(M1 * 96);
  U->P2 = bf(M2 * 32);
  U->E3a = bf(M2 * 64);
  U->CAT3 = bf(M2 * 192);
  U->P3 = bf(M3 * 64);
  U->Ba = bf(M3 * 128);
  U->Bb = bf(M3 * 128);
  U->D3a = bf(M2 * 64);
  U->D3b = bf(M2 * 64);
  U->D2a = bf(M1 * 32);
  U->D2b = bf(M1 * 32);
  U->D1a = bf(M0 * 16);
  U->D1b = bf(M0 * 16);
  U->Gpre = bf(M0 * 48);
  U->OUT = f(M0);
  U->GOUT = f(M0);
  U->G_E1a = f(M0 * 16);
  U->G_CAT1 = f(M0 * 48);
  U->G_P1 = f(M1 * 16);
  U->G_E2a = f(M1 * 32);
  U->G_CAT2 = f(M1 * 96);
  U->G_P2 = f(M2 * 32);
  U->G_E3a = f(M2 * 64);
  U->G_CAT3 = f(M2 * 192);
  U->G_P3 = f(M3 * 64);
  U->G_Ba = f(M3 * 128);
  U->G_Bb = f(M3 * 128);
  U->G_D3a = f(M2 * 64);
  U->G_D3b = f(M2 * 64);
  U->G_D2a = f(M1 * 32);
  U->G_D2b = f(M1 * 32);
  U->G_D1a = f(M0 * 16);
  U->G_D1b = f(M0 * 16);
  long long wn = 0;
  for (const ConvSpec& cs : kConvs)
    wn = std::max(wn, std::max(nn_wgrad_scratch(cs.cin, cs.cout),
                               nn_tc_wgrad_scratch(cs.cin, cs.cout)));
  U->wpart_n = wn;
  U->wpart = f(std::max(wn, 17LL * 1024));
  U->bpart = f(128LL * kBiasBlocks);
  U->ffr0 = bf(4096);
  U->lossp = (double*)bytes(sizeof(double) * 1024);
  U->fr0d = (double*)bytes(sizeof(double) * 4096);
  if (!ok) {
    (void)cudaGetLastError();
    unet_free_bufs(U);
    return set_err(c, MGFR_E_OOM, "U-Net activation allocation failed");
  }
  U->B = B;
  U->lgD = lgD;
  return MGFR_OK;
}

static TView tv(__nv_bfloat16* p, int ld, int off = 0) { return TView{p, ld, off}; }
static FView fv(float* p, int ld, int off = 0) { return FView{p, ld, off}; }

// conv layer i: input view, output view (post-ReLU)
struct LayerIO {
  TView x, y;
  FView gx, gy;  // gradients w.r.t. input and output
  int lgD;
};

static void layer_views(UNet* U, LayerIO* L) {
  const int g = U->lgD;
  L[0] = {tv(U->X0, 16), tv(U->E1a, 16), fv(nullptr, 0), fv(U->G_E1a, 16), g};
  L[1] = {tv(U->E1a, 16), tv(U->CAT1, 48, 32), fv(U->G_E1a, 16), fv(U->G_CAT1, 48, 32), g};
  L[2] = {tv(U->P1, 16), tv(U->E2a, 32), fv(U->G_P1, 16), fv(U->G_E2a, 32), g - 1};
  L[3] = {tv(U->E2a, 32), tv(U->CAT2, 96, 64), fv(U->G_E2a, 32), fv(U->G_CAT2, 96, 64), g - 1};
  L[4] = {tv(U->P2, 32), tv(U->E3a, 64), fv(U->G_P2, 32), fv(U->G_E3a, 64), g - 2};
  L[5] = {tv(U->E3a, 64), tv(U->CAT3, 192, 128), fv(U->G_E3a, 64), fv(U->G_CAT3, 192, 128), g - 2};
  L[6] = {tv(U->P3, 64), tv(U->Ba, 128), fv(U->G_P3, 64), fv(U->G_Ba, 128), g - 3};
  L[7] = {tv(U->Ba, 128), tv(U->Bb, 128), fv(U->G_Ba, 128), fv(U->G_Bb, 128), g - 3};
  L[8] = {tv(U->CAT3, 192), tv(U->D3a, 64), fv(U->G_CAT3, 192), fv(U->G_D3a, 64), g - 2};
  L[9] = {tv(U->D3a, 64), tv(U->D3b, 64), fv(U->G_D3a, 64), fv(U->G_D3b, 64), g - 2};
  L[10] = {tv(U->CAT2, 96), tv(U->D2a, 32), fv(U->G_CAT2, 96), fv(U->G_D2a, 32), g - 1};
  L[11] = {tv(U->D2a, 32), tv(U->D2b, 32), fv(U->G_D2a, 32), fv(U->G_D2b, 32), g - 1};
  L[12] = {tv(U->CAT1, 48), tv(U->D1a, 16), fv(U->G_CAT1, 48), fv(U->G_D1a, 16), g};
  L[13] = {tv(U->D1a, 16), tv(U->D1b, 16), fv(U->G_D1a, 16), fv(U->G_D1b, 16), g};
}

static void conv_fwd(mgfr_ctx* c, UNet* U, int i, const LayerIO& L) {
  const ConvSpec& s = kConvs[i];
  if (nn_tc_supported(s.cin, s.cout)) {
    TcArgs a{};
    a.x = L.x.p;
    a.ldx = L.x.ld;
    a.offx = L.x.off;
    a.Wp = U->Wtf + U->wbf_off[i];
    a.bias = U->P + U->boff[i];
    a.relu = 1;
    a.y = L.y.p;
    a.ldy = L.y.ld;
    a.offy = L.y.off;
    a.lgD = L.lgD;
    a.Mtot = (long long)U->B << (3 * L.lgD);
    a.err = U->tc_err;
    nn_tc_conv(a, s.cin, s.cout, false, c->s);
  } else {
    nn_conv_fwd(L.x, s.cin, U->Wbf + U->wbf_off[i], U->P + U->boff[i], 1, L.y, s.cout, U->B,
                L.lgD, c->s);
  }
  c->launches += 1;
}

static void forward(mgfr_ctx* c, UNet* U) {
  LayerIO L[14];
  layer_views(U, L);
  const int g = U->lgD, B = U->B;
  const long long M0 = (long long)B << (3 * g);
  auto launch_pool = [&](TView x, TView y, int C, int lgDc) {
    const long long Mc = (long long)B << (3 * lgDc);
    k_pool<<<nblocks(Mc * C / 8, BS), BS, 0, c->s>>>(x, y, lg_of(C / 8), lgDc, Mc * C / 8);
    c->launches += 1;
  };
  auto launch_up = [&](TView x, TView y, int C, int lgDf) {
    const long long Mf = (long long)B << (3 * lgDf);
    k_up<<<nblocks(Mf * C / 8, BS), BS, 0, c->s>>>(x, y, lg_of(C / 8), lgDf, Mf * C / 8);
    c->launches += 1;
  };
  conv_fwd(c, U, 0, L[0]);
  conv_fwd(c, U, 1, L[1]);
  launch_pool(tv(U->CAT1, 48, 32), tv(U->P1, 16), 16, g - 1);
  conv_fwd(c, U, 2, L[2]);
  conv_fwd(c, U, 3, L[3]);
  launch_pool(tv(U->CAT2, 96, 64), tv(U->P2, 32), 32, g - 2);
  conv_fwd(c, U, 4, L[4]);
  conv_fwd(c, U, 5, L[5]);
  launch_pool(tv(U->CAT3, 192, 128), tv(U->P3, 64), 64, g - 3);
  conv_fwd(c, U, 6, L[6]);
  conv_fwd(c, U, 7, L[7]);
  launch_up(tv(U->Bb, 128), tv(U->CAT3, 192, 0), 128, g - 2);
  conv_fwd(c, U, 8, L[8]);
  conv_fwd(c, U, 9, L[9]);
  launch_up(tv(U->D3b, 64), tv(U->CAT2, 96, 0), 64, g - 1);
  conv_fwd(c, U, 10, L[10]);
  conv_fwd(c, U, 11, L[11]);
  launch_up(tv(U->D2b, 32), tv(U->CAT1, 48, 0), 32, g);
  conv_fwd(c, U, 12, L[12]);
  conv_fwd(c, U, 13, L[13]);
  k_head_fwd<<<nblocks(M0, BS), BS, 0, c->s>>>(tv(U->D1b, 16), U->P + U->head_off, M0, U->OUT);
  c->launches += 1;
}

static void conv_bwd(mgfr_ctx* c, UNet* U, int i, const LayerIO& L, int acc_in) {
  const ConvSpec& s = kConvs[i];
  const long long M = (long long)U->B << (3 * L.lgD);
  // the bias gradient comes out of the pass that forms the pre-activation's
  const long long n8 = M * s.cout / 8;
  const int nb = (int)std::min<long long>(kBiasBlocks, nblocks(n8, BS));
  k_relu_bwd<<<nb, BS, 0, c->s>>>(L.gy, L.y, lg_of(s.cout / 8), n8, U->Gpre, U->bpart);
  nn_bias_sum(U->bpart, nb, s.cout, U->G + U->boff[i], c->s);
  const TView g = tv(U->Gpre, s.cout);
  if (!nn_tc_wgrad(L.x, s.cin, g, s.cout, U->G + U->woff[i], nullptr, U->wpart, U->B, L.lgD,
                   U->tc_err, c->s))
    nn_conv_wgrad(L.x, s.cin, g, s.cout, U->G + U->woff[i], nullptr, U->wpart, U->B, L.lgD, c->s);
  if (L.gx.p) {
    if (nn_tc_supported(s.cout, s.cin)) {
      TcArgs a{};
      a.x = U->Gpre;
      a.ldx = s.cout;
      a.offx = 0;
      a.Wp = U->Wtd + U->wbf_off[i];
      a.gx = L.gx.p;
      a.ldg = L.gx.ld;
      a.offg = L.gx.off;
      a.accumulate = acc_in;
      a.lgD = L.lgD;
      a.Mtot = M;
      a.err = U->tc_err;
      nn_tc_conv(a, s.cout, s.cin, true, c->s);
    } else {
      nn_conv_dgrad(g, s.cout, U->Wbf + U->wbf_off[i], L.gx, s.cin, acc_in, U->B, L.lgD, c->s);
    }
  }
  c->launches += 5;
}

static void backward(mgfr_ctx* c, UNet* U) {
  LayerIO L[14];
  layer_views(U, L);
  const int g = U->lgD, B = U->B;
  const long long M0 = (long long)B << (3 * g);
  const int nb = 256;
  k_head_bwd<<<nb, BS, 0, c->s>>>(tv(U->D1b, 16), U->P + U->head_off, U->GOUT, M0,
                                   fv(U->G_D1b, 16), U->wpart);
  k_sum_parts<<<1, 32, 0, c->s>>>(U->wpart, nb, 17, U->G + U->head_off);
  c->launches += 2;
  auto up_bwd = [&](FView gf, FView gc, int C, int lgDc) {
    const long long Mc = (long long)B << (3 * lgDc);
    k_up_bwd<<<nblocks(Mc * C / 8, BS), BS, 0, c->s>>>(gf, gc, lg_of(C / 8), lgDc, Mc * C / 8);
    c->launches += 1;
  };
  auto pool_bwd = [&](FView gc, FView gf, int C, int lgDf) {
    const long long Mf = (long long)B << (3 * lgDf);
    k_pool_bwd<<<nblocks(Mf * C / 8, BS), BS, 0, c->s>>>(gc, gf, lg_of(C / 8), lgDf, Mf * C / 8);
    c->launches += 1;
  };
  conv_bwd(c, U, 13, L[13], 0);                        // -> G_D1a
  conv_bwd(c, U, 12, L[12], 0);                        // -> G_CAT1 (all 48)
  up_bwd(fv(U->G_CAT1, 48, 0), fv(U->G_D2b, 32), 32, g - 1);
  conv_bwd(c, U, 11, L[11], 0);                        // -> G_D2a
  conv_bwd(c, U, 10, L[10], 0);                        // -> G_CAT2 (all 96)
  up_bwd(fv(U->G_CAT2, 96, 0), fv(U->G_D3b, 64), 64, g - 2);
  conv_bwd(c, U, 9, L[9], 0);                          // -> G_D3a
  conv_bwd(c, U, 8, L[8], 0);                          // -> G_CAT3 (all 192)
  up_bwd(fv(U->G_CAT3, 192, 0), fv(U->G_Bb, 128), 128, g - 3);
  conv_bwd(c, U, 7, L[7], 0);                          // -> G_Ba
  conv_bwd(c, U, 6, L[6], 0);                          // -> G_P3
  pool_bwd(fv(U->G_P3, 64), fv(U->G_CAT3, 192, 128), 64, g - 2);
  conv_bwd(c, U, 5, L[5], 0);                          // -> G_E3a
  conv_bwd(c, U, 4, L[4], 0);                          // -> G_P2
  pool_bwd(fv(U->G_P2, 32), fv(U->G_CAT2, 96, 64), 32, g - 1);
  conv_bwd(c, U, 3, L[3], 0);                          // -> G_E2a
  conv_bwd(c, U, 2, L[2], 0);                          // -> G_P1
  pool_bwd(fv(U->G_P1, 16), fv(U->G_CAT1, 48, 32), 16, g);
  conv_bwd(c, U, 1, L[1], 0);                          // -> G_E1a
  conv_bwd(c, U, 0, L[0], 0);                          // no input gradient
}

static void refresh_bf16(mgfr_ctx* c, UNet* U) {
  PackTab T;
  for (int i = 0; i < 14; ++i) {
    T.woff[i] = U->woff[i];
    T.boff[i] = U->wbf_off[i];
    T.cin[i] = kConvs[i].cin;
    T.cout[i] = kConvs[i].cout;
  }
  T.boff[14] = U->nwbf;
  k_refresh<<<nblocks(U->nwbf, BS), BS, 0, c->s>>>(U->P, T, U->Wbf, U->Wtf, U->Wtd);
  c->launches += 1;
}

// the tensor-core kernels' error word (read after the stream has synchronised)
static mgfr_status tc_check(mgfr_ctx* c, UNet* U) {
  int e = 0;
  MG_CK(c, cudaMemcpy(&e, U->tc_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (e) {
    MG_CK(c, cudaMemsetAsync(U->tc_err, 0, sizeof(int), c->s));
    return set_err(c, MGFR_E_TIMEOUT, "a bounded wait in a tensor-core convolution gave up");
  }
  return MGFR_OK;
}

// The parameters (nparam floats) from the host, with Adam's moments at zero where
// `fresh`, and the BF16 copies; on the context's stream, whose kernels are in no order
// with the legacy default stream's copies and memsets.  Waits for it.
static mgfr_status unet_set(mgfr_ctx* c, UNet* U, const float* host, bool fresh) {
  const size_t bytes = sizeof(float) * (size_t)U->nparam;
  MG_CK(c, cudaSetDevice(c->device));
  MG_CK(c, cudaMemcpyAsync(U->P, host, bytes, cudaMemcpyHostToDevice, c->s));
  if (fresh) {
    MG_CK(c, cudaMemsetAsync(U->M1, 0, bytes, c->s));
    MG_CK(c, cudaMemsetAsync(U->M2, 0, bytes, c->s));
    U->step = 0;
  }
  refresh_bf16(c, U);
  MG_CK(c, cudaStreamSynchronize(c->s));
  return MGFR_OK;
}

static mgfr_status unet_fill(mgfr_ctx* c, UNet* U, unsigned long long seed) {
  long long off = 0, boff = 0;
  for (int i = 0; i < 14; ++i) {
    U->woff[i] = off;
    off += 27LL * kConvs[i].cin * kConvs[i].cout;
    U->boff[i] = off;
    off += kConvs[i].cout;
    U->wbf_off[i] = boff;
    boff += 27LL * kConvs[i].cin * kConvs[i].cout;
  }
  U->head_off = off;
  off += 17;
  U->nparam = off;
  U->nwbf = boff;
  MG_CK(c, dev_malloc(c, &U->P, sizeof(float) * off));
  MG_CK(c, dev_malloc(c, &U->G, sizeof(float) * off));
  MG_CK(c, dev_malloc(c, &U->M1, sizeof(float) * off));
  MG_CK(c, dev_malloc(c, &U->M2, sizeof(float) * off));
  MG_CK(c, dev_malloc(c, &U->Wbf, sizeof(__nv_bfloat16) * boff));
  MG_CK(c, dev_malloc(c, &U->Wtf, sizeof(__nv_bfloat16) * boff));
  MG_CK(c, dev_malloc(c, &U->Wtd, sizeof(__nv_bfloat16) * boff));
  MG_CK(c, dev_malloc(c, &U->tc_err, sizeof(int)));
  MG_CK(c, cudaMemsetAsync(U->tc_err, 0, sizeof(int), c->s));
  // He-normal initialisation from a seeded generator (host), zero biases
  std::vector<float> h((size_t)off, 0.f);
  std::mt19937_64 rng(seed);
  for (int i = 0; i < 14; ++i) {
    std::normal_distribution<float> nd(0.f, std::sqrt(2.f / (27.f * kConvs[i].cin)));
    for (long long q = 0; q < 27LL * kConvs[i].cin * kConvs[i].cout; ++q) h[U->woff[i] + q] = nd(rng);
  }
  // the head starts at zero: the first prediction is u = 0 (the zero start),
  // so early steps do not push the network into saturation
  return unet_set(c, U, h.data(), true);
}

static mgfr_status unet_make(mgfr_ctx* c, unsigned long long seed) {
  unet_free(c);
  UNet* U = new UNet();
  c->unet = U;
  const mgfr_status rs = unet_fill(c, U, seed);
  if (rs != MGFR_OK) unet_free(c);  // no network rather than a part of one
  return rs;
}

static const char kUnetTag[9] = "MGFRUNT1";

mgfr_status unet_predict_batch(mgfr_ctx* c, int B, int D, const double* x, double dscale,
                               const double* fr0_host, double* u_out) {
  if (!c->unet) return set_err(c, MGFR_E_INVALID, "no network (mgfr_unet_init or mgfr_unet_load)");
  if (B < 1 || B > 4096 || D < 32 || D > 512 || (D & (D - 1)) || !x || !u_out || !fr0_host)
    return set_err(c, MGFR_E_INVALID, "network input: D must be a power of two in [32, 512]");
  for (int b = 0; b < B; ++b)
    if (!(fr0_host[b] > 0.0)) return set_err(c, MGFR_E_INVALID, "network input: |fR0| > 0");
  UNet* U = (UNet*)c->unet;
  mgfr_status rs = unet_alloc(c, U, B, lg_of(D));
  if (rs != MGFR_OK) return rs;
  const long long per = (long long)D * D * D, M0 = per * B;
  MG_CK(c, cudaMemcpyAsync(U->fr0d, fr0_host, sizeof(double) * B, cudaMemcpyHostToDevice, c->s));
  const Model mm = make_model(c->cfg, 1.0);
  k_fr0_feature<<<nblocks(B, BS), BS, 0, c->s>>>(U->fr0d, B, U->ffr0);
  k_features<<<nblocks(M0, BS), BS, 0, c->s>>>(x, U->ffr0, 3 * U->lgD, M0, U->X0,
                                               c->cfg.omega_m / mm.Rt, (double)(c->cfg.n + 1),
                                               dscale);
  forward(c, U);
  k_out_to_double<<<nblocks(M0, BS), BS, 0, c->s>>>(U->OUT, u_out, M0);
  c->launches += 2;
  // fr0_host may be a caller's stack value: the copy must be done before return
  MG_CK(c, cudaStreamSynchronize(c->s));
  return tc_check(c, U);
}

extern "C" {

mgfr_status mgfr_unet_init(mgfr_ctx* c, unsigned long long seed) {
  if (!c) return MGFR_E_INVALID;
  MG_CK(c, cudaSetDevice(c->device));
  return unet_make(c, seed);
}

mgfr_status mgfr_unet_train_step(mgfr_ctx* c, int B, int D, const double* delta_dev,
                                 const double* fr0_host, const double* u_target_dev, float lr,
                                 double* loss_out) {
  if (!c || !c->unet) return c ? set_err(c, MGFR_E_INVALID, "call mgfr_unet_init first") : MGFR_E_INVALID;
  if (B < 1 || B > 4096 || D < 32 || D > 512 || (D & (D - 1)) || !delta_dev || !fr0_host ||
      !u_target_dev)
    return set_err(c, MGFR_E_INVALID, "bad U-Net training batch");
  UNet* U = (UNet*)c->unet;
  MG_CK(c, cudaSetDevice(c->device));
  mgfr_status rs = unet_alloc(c, U, B, lg_of(D));
  if (rs != MGFR_OK) return rs;
  const long long M0 = (long long)B * D * D * D;
  // the batch and targets come from work on the caller's stream
  MG_CK(c, cudaEventRecord(c->ev_in, c->user));
  MG_CK(c, cudaStreamWaitEvent(c->s, c->ev_in, 0));
  MG_CK(c, cudaMemcpyAsync(U->fr0d, fr0_host, sizeof(double) * B, cudaMemcpyHostToDevice, c->s));
  const Model mm = make_model(c->cfg, 1.0);
  k_fr0_feature<<<nblocks(B, BS), BS, 0, c->s>>>(U->fr0d, B, U->ffr0);
  k_features<<<nblocks(M0, BS), BS, 0, c->s>>>(delta_dev, U->ffr0, 3 * U->lgD, M0, U->X0,
                                               c->cfg.omega_m / mm.Rt, (double)(c->cfg.n + 1),
                                               1.0);
  forward(c, U);
  const int nb = 1024;
  k_mse<<<nb, BS, 0, c->s>>>(U->OUT, u_target_dev, M0, 2.0 / (double)M0, U->GOUT, U->lossp);
  backward(c, U);
  U->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)U->step), c2 = 1.f - std::pow(b2, (float)U->step);
  k_adam<<<nblocks(U->nparam, BS), BS, 0, c->s>>>(U->P, U->G, U->M1, U->M2, U->nparam, lr, b1, b2,
                                                  1e-8f, c1, c2);
  refresh_bf16(c, U);
  std::vector<double> part(nb);
  MG_CK(c, cudaMemcpyAsync(part.data(), U->lossp, sizeof(double) * nb, cudaMemcpyDeviceToHost, c->s));
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaGetLastError());
  if ((rs = tc_check(c, U)) != MGFR_OK) return rs;
  double s = 0.0;
  for (double v : part) s += v;
  if (loss_out) *loss_out = s / (double)M0;
  return MGFR_OK;
}

mgfr_status mgfr_unet_predict(mgfr_ctx* c, int D, const double* delta_dev, double fr0_abs,
                              double* u_out_dev) {
  if (!c) return MGFR_E_INVALID;
  if (!delta_dev || !u_out_dev || !(fr0_abs > 0.0))
    return set_err(c, MGFR_E_INVALID, "bad U-Net input");
  MG_CK(c, cudaSetDevice(c->device));
  MG_CK(c, cudaEventRecord(c->ev_in, c->user));
  MG_CK(c, cudaStreamWaitEvent(c->s, c->ev_in, 0));
  mgfr_status rs = unet_predict_batch(c, 1, D, delta_dev, 1.0, &fr0_abs, u_out_dev);
  if (rs != MGFR_OK) return rs;
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaGetLastError());
  return MGFR_OK;
}

mgfr_status mgfr_unet_save(mgfr_ctx* c, const char* path) {
  if (!c || !path) return MGFR_E_INVALID;
  if (!c->unet) return set_err(c, MGFR_E_INVALID, "no network (mgfr_unet_init or mgfr_unet_load)");
  UNet* U = (UNet*)c->unet;
  MG_CK(c, cudaSetDevice(c->device));
  std::vector<float> h((size_t)U->nparam);
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaMemcpy(h.data(), U->P, sizeof(float) * h.size(), cudaMemcpyDeviceToHost));
  FILE* f = std::fopen(path, "wb");
  if (!f) return set_err(c, MGFR_E_INVALID, std::string("cannot open ") + path);
  unsigned char hdr[16];
  std::memcpy(hdr, kUnetTag, 8);
  const unsigned long long n = (unsigned long long)U->nparam;
  for (int q = 0; q < 8; ++q) hdr[8 + q] = (unsigned char)(n >> (8 * q));
  bool ok = std::fwrite(hdr, 1, 16, f) == 16;
  for (size_t i = 0; ok && i < h.size(); ++i) {
    unsigned u;
    std::memcpy(&u, &h[i], 4);
    const unsigned char b[4] = {(unsigned char)u, (unsigned char)(u >> 8), (unsigned char)(u >> 16),
                                (unsigned char)(u >> 24)};
    ok = std::fwrite(b, 1, 4, f) == 4;
  }
  ok = (std::fclose(f) == 0) && ok;
  return ok ? MGFR_OK : set_err(c, MGFR_E_INVALID, std::string("write failed: ") + path);
}

mgfr_status mgfr_unet_load(mgfr_ctx* c, const char* path) {
  if (!c || !path) return MGFR_E_INVALID;
  MG_CK(c, cudaSetDevice(c->device));
  FILE* f = std::fopen(path, "rb");
  if (!f) return set_err(c, MGFR_E_INVALID, std::string("cannot open ") + path);
  unsigned char hdr[16];
  if (std::fread(hdr, 1, 16, f) != 16 || std::memcmp(hdr, kUnetTag, 8) != 0) {
    std::fclose(f);
    return set_err(c, MGFR_E_INVALID, "not a network parameter file");
  }
  unsigned long long n = 0;
  for (int q = 0; q < 8; ++q) n |= (unsigned long long)hdr[8 + q] << (8 * q);
  if (!c->unet) {
    mgfr_status rs = unet_make(c, 0);
    if (rs != MGFR_OK) {
      std::fclose(f);
      return rs;
    }
  }
  UNet* U = (UNet*)c->unet;
  if (n != (unsigned long long)U->nparam) {
    std::fclose(f);
    return set_err(c, MGFR_E_INVALID, "parameter count in the file does not match the network");
  }
  std::vector<float> h((size_t)n);
  bool ok = true;
  for (size_t i = 0; ok && i < h.size(); ++i) {
    unsigned char b[4];
    ok = std::fread(b, 1, 4, f) == 4;
    const unsigned u = b[0] | ((unsigned)b[1] << 8) | ((unsigned)b[2] << 16) | ((unsigned)b[3] << 24);
    std::memcpy(&h[i], &u, 4);
  }
  std::fclose(f);
  if (!ok) return set_err(c, MGFR_E_INVALID, "truncated network parameter file");
  return unet_set(c, U, h.data(), true);
}

mgfr_status mgfr_unet_params(mgfr_ctx* c, int set, float* host, long long* count) {
  if (!c || !c->unet) return MGFR_E_INVALID;
  UNet* U = (UNet*)c->unet;
  if (count) *count = U->nparam;
  if (!host) return MGFR_OK;
  if (set) return unet_set(c, U, host, false);
  MG_CK(c, cudaMemcpy(host, U->P, sizeof(float) * U->nparam, cudaMemcpyDeviceToHost));
  return MGFR_OK;
}

mgfr_status mgfr_unet_grads(mgfr_ctx* c, float* host) {
  if (!c || !c->unet || !host) return MGFR_E_INVALID;
  UNet* U = (UNet*)c->unet;
  MG_CK(c, cudaMemcpy(host, U->G, sizeof(float) * U->nparam, cudaMemcpyDeviceToHost));
  return MGFR_OK;
}

}  // extern "C"

// Scratch of mgfr_nn_conv3d (packed weights or partial sums, and the kernels'
// error word), kept between calls: cudaMalloc and cudaFree took 0.2 ms of every
// call.  A call owns its block from acquire to release, which come before and
// after its work (the call waits for its stream), so blocks never serve two
// streams or threads at once; it clears an error word that is not known to be 0
// on its own stream, with which no other stream is in order.  At most 4 blocks
// and 128 MB per device stay, the largest ones (a block serves every call that
// needs no more, so one caller's calls come to rest on the largest of their
// sizes, at most 57 MB); mgfr_destroy gives those of its device back.  (When the
// first four blocks stayed, a call larger than they allocated and freed its own
// each time: weight gradients on 16^3 after four small layers 225-260 us, now
// 44-64.)
namespace {
constexpr size_t kScratchBlocks = 4, kScratchBytes = (size_t)128 << 20;
struct ConvScratch {
  int dev = 0;
  size_t bytes = 0;
  void* p = nullptr;
  int *err = nullptr, *err_h = nullptr;  // device word, page-locked copy
  bool clear = false;                    // the word was last read as 0 (kernels only set it)
};
std::mutex g_scratch_mu;
std::vector<ConvScratch> g_scratch;

void scratch_drop(ConvScratch& b) {
  if (b.p) cudaFree(b.p);
  if (b.err) cudaFree(b.err);
  if (b.err_h) cudaFreeHost(b.err_h);
  b = ConvScratch();
}

mgfr_status scratch_acquire(size_t bytes, cudaStream_t s, ConvScratch* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MGFR_E_CUDA;
  ConvScratch b;
  {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    int best = -1;
    for (size_t i = 0; i < g_scratch.size(); ++i)
      if (g_scratch[i].dev == dev && g_scratch[i].bytes >= bytes &&
          (best < 0 || g_scratch[i].bytes < g_scratch[best].bytes))
        best = (int)i;
    if (best >= 0) {
      b = g_scratch[best];
      g_scratch.erase(g_scratch.begin() + best);
    }
  }
  if (!b.p) {
    b.dev = dev;
    b.bytes = bytes;
    if (cudaMalloc(&b.p, bytes) != cudaSuccess || cudaMalloc(&b.err, sizeof(int)) != cudaSuccess ||
        cudaMallocHost(&b.err_h, sizeof(int)) != cudaSuccess) {
      (void)cudaGetLastError();
      scratch_drop(b);
      return MGFR_E_OOM;
    }
  }
  if (!b.clear && cudaMemsetAsync(b.err, 0, sizeof(int), s) != cudaSuccess) {
    (void)cudaGetLastError();
    scratch_drop(b);
    return MGFR_E_CUDA;
  }
  *out = b;
  return MGFR_OK;
}

void scratch_release(const ConvScratch& b) {
  std::vector<ConvScratch> out;  // given back after the lock
  {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    g_scratch.push_back(b);
    for (;;) {
      size_t n = 0, sum = 0;
      int least = -1;
      for (size_t i = 0; i < g_scratch.size(); ++i)
        if (g_scratch[i].dev == b.dev) {
          ++n;
          sum += g_scratch[i].bytes;
          if (least < 0 || g_scratch[i].bytes < g_scratch[least].bytes) least = (int)i;
        }
      if (n <= kScratchBlocks && sum <= kScratchBytes) break;
      out.push_back(g_scratch[least]);
      g_scratch.erase(g_scratch.begin() + least);
    }
  }
  for (ConvScratch& q : out) scratch_drop(q);
}

// wait for the call's work, read the kernels' error word, give the block back
mgfr_status scratch_finish(ConvScratch& b, cudaStream_t s) {
  const bool ok =
      cudaMemcpyAsync(b.err_h, b.err, sizeof(int), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
      cudaStreamSynchronize(s) == cudaSuccess && cudaGetLastError() == cudaSuccess;
  if (!ok) {
    scratch_drop(b);
    return MGFR_E_CUDA;
  }
  const int e = *b.err_h;
  b.clear = e == 0;
  scratch_release(b);
  return e ? MGFR_E_TIMEOUT : MGFR_OK;
}
}  // namespace

bool conv_scratch_trim(int dev) {
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  bool any = false;
  for (size_t i = g_scratch.size(); i-- > 0;)
    if (g_scratch[i].dev == dev) {
      scratch_drop(g_scratch[i]);
      g_scratch.erase(g_scratch.begin() + i);
      any = true;
    }
  return any;
}

extern "C" {

// Convolution primitive on caller buffers (contiguous NDHWC, C multiples of 16):
// op 0: y(bf16) = relu?(conv(x, W) + b); op 1: gx(FP32) = conv^T(g, W);
// op 2: dW(FP32 [27][Cin][Cout]), db(FP32) from x and g.
mgfr_status mgfr_nn_conv3d(int op, int B, int D, int Cin, int Cout, const void* x_bf16,
                           const void* w_bf16, const float* bias, int relu, const void* g_bf16,
                           void* out, float* db, void* stream) {
  if (B < 1 || D < 4 || (D & (D - 1)) || Cin % 16 || Cout % 16 || Cin < 16 || Cout < 16 ||
      Cout > 128 || Cin > 256)
    return MGFR_E_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  const int lgD = lg_of(D);
  const bool tc = (op == 0 && nn_tc_supported(Cin, Cout)) ||
                  (op == 1 && nn_tc_supported(Cout, Cin)) ||
                  (op == 2 && nn_tc_wgrad_supported(Cin, Cout));
  // the tcgen05 kernels move 16 bytes of a voxel's channels at a time (in, and for ops 0 and
  // 1 out), the mma.sync ones 4 in ops 0 and 1 and single values in op 2
  auto on = [](const void* p, unsigned b) { return (uintptr_t)p % b == 0; };
  const unsigned bi = tc ? 16 : (op == 2 ? 2 : 4), bo = tc && op != 2 ? 16 : 4;
  if ((op != 1 && !on(x_bf16, bi)) || (op != 0 && !on(g_bf16, bi)) || !on(out, bo))
    return MGFR_E_INVALID;
  if (tc && op != 2) {
    // pack the weights for the tensor-core kernel (scratch of this call)
    ConvScratch sc;
    const mgfr_status rs =
        scratch_acquire(sizeof(__nv_bfloat16) * (size_t)nn_tc_packed_size(Cin, Cout), s, &sc);
    if (rs != MGFR_OK) return rs;
    __nv_bfloat16* wp = (__nv_bfloat16*)sc.p;
    nn_tc_pack((const __nv_bfloat16*)w_bf16, Cin, Cout, op, wp, s);
    TcArgs a{};
    a.Wp = wp;
    a.lgD = lgD;
    a.Mtot = (long long)B << (3 * lgD);
    a.err = sc.err;
    if (op == 0) {
      a.x = (const __nv_bfloat16*)x_bf16;
      a.ldx = Cin;
      a.bias = bias;
      a.relu = relu;
      a.y = (__nv_bfloat16*)out;
      a.ldy = Cout;
    } else {
      a.x = (const __nv_bfloat16*)g_bf16;
      a.ldx = Cout;
      a.gx = (float*)out;
      a.ldg = Cin;
    }
    nn_tc_conv(a, op == 0 ? Cin : Cout, op == 0 ? Cout : Cin, op == 1, s);
    return scratch_finish(sc, s);
  }
  if (op == 0) {
    nn_conv_fwd(TView{(__nv_bfloat16*)x_bf16, Cin, 0}, Cin, (const __nv_bfloat16*)w_bf16, bias,
                relu, TView{(__nv_bfloat16*)out, Cout, 0}, Cout, B, lgD, s);
  } else if (op == 1) {
    nn_conv_dgrad(TView{(__nv_bfloat16*)g_bf16, Cout, 0}, Cout, (const __nv_bfloat16*)w_bf16,
                  FView{(float*)out, Cin, 0}, Cin, 0, B, lgD, s);
  } else if (op == 2) {
    const long long np = tc ? nn_tc_wgrad_scratch(Cin, Cout) : nn_wgrad_scratch(Cin, Cout);
    ConvScratch sc;
    const mgfr_status rs = scratch_acquire(sizeof(float) * (size_t)np, s, &sc);
    if (rs != MGFR_OK) return rs;
    float* part = (float*)sc.p;
    const TView xv{(__nv_bfloat16*)x_bf16, Cin, 0}, gv{(__nv_bfloat16*)g_bf16, Cout, 0};
    if (!tc || !nn_tc_wgrad(xv, Cin, gv, Cout, (float*)out, db, part, B, lgD, sc.err, s))
      nn_conv_wgrad(xv, Cin, gv, Cout, (float*)out, db, part, B, lgD, s);
    return scratch_finish(sc, s);
  } else {
    return MGFR_E_INVALID;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return MGFR_E_CUDA;
  return MGFR_OK;
}

}  // extern "C"

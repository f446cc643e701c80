// mg32.cu -- FP32 V-cycles on dense periodic levels (mg32.cuh).
//
// Levels above 32^3 run one kernel per half-sweep, restriction and
// prolongation, four cells of one colour per thread: in colour-split storage
// the cells (i, j, 4v..4v+3) of a plane, their four row neighbours and the two
// z neighbours are five 16-byte loads and one scalar, so the index arithmetic
// is paid once per four cells and the exponentials of shared z neighbours are
// formed once.  The kernels are bound by issue slots and the SFU, not by
// memory (one cell per thread took 387 us for a nonlinear half-sweep of 512^3,
// 8 bytes per cell, against 158 us for its bytes).
//
// Levels of 32^3 and below (four of them, about 40 dependent half-sweeps and
// transfers of at most 32768 cells) run in one launch: a cluster of up to 16
// CTAs holds all of them in distributed shared memory, slabs of x planes per
// CTA, the 8^3 and 4^3 grids in the first CTA.  A phase then ends with a
// cluster barrier instead of a kernel boundary.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "colour_split.cuh"
#include "mg32.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int BS = 256;

// e^x - 1 to FP32 relative accuracy, and e^x in *e: the Taylor series through
// x^7/7! for |x| <= 0.35 (omitted terms below 6e-9 relative), the exponential
// beyond
__device__ __forceinline__ float em1(float x, float* e) {
  float q = fmaf(x, 1.f / 5040.f, 1.f / 720.f);
  q = fmaf(x, q, 1.f / 120.f);
  q = fmaf(x, q, 1.f / 24.f);
  q = fmaf(x, q, 1.f / 6.f);
  q = fmaf(x, q, 0.5f);
  q = x * fmaf(x, q, 1.f);
  const bool small = fabsf(x) <= 0.35f;
  const float ex = __expf(x);
  *e = small ? q + 1.f : ex;
  return small ? q : ex - 1.f;
}
__device__ __forceinline__ float em1(float x) {
  float e;
  return em1(x, &e);
}

struct PF {
  float aRt, aRt_np1, inv_np1, cap;
};

// ---- point operations: xc, xn[6] the unknown at the cell and its neighbours
// (-x, +x, -y, +y, -z, +z), wc, wn[6] the linearisation point -------------------
// (EXACT: with the correctly rounded division, on the 4^3 grid)
template <int OP, bool EXACT = false>
__device__ __forceinline__ float point_update(float xc, const float* xn, float wc, const float* wn,
                                              float r, const PF& m, float ih2, float h2) {
  if constexpr (OP == MG_NL) {
    // Newton step (L - f) / (dL/du), neighbours fixed, clamped (Eq. (23))
    const float Ec = __expf(xc);
    float sbd = 0.f, sd = 0.f, sb = 0.f;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      const float bb = 0.5f * (__expf(xn[e]) + Ec), du = xn[e] - xc;
      sbd = fmaf(bb, du, sbd);
      sd += du;
      sb += bb;
    }
    const float s = __expf(-xc * m.inv_np1);
    const float L = sbd * ih2 + m.aRt * (1.f - s);
    const float dL = (0.5f * Ec * sd - sb) * ih2 + m.aRt_np1 * s;
    const float step = EXACT ? (L - r) / dL : __fdividef(L - r, dL);
    return xc - fminf(fmaxf(step, -m.cap), m.cap);
  } else if constexpr (OP == MG_LIN) {
    const float Ec = __expf(wc), q2 = 0.5f * ih2;
    float d = 0.f, s = r;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const float En = __expf(wn[q]), du = wn[q] - wc;
      const float off = q2 * fmaf(En, du, Ec + En);
      d += fmaf(Ec, du, -Ec - En);
      s = fmaf(-off, xn[q], s);
    }
    const float diag = d * q2 + m.aRt_np1 * __expf(-wc * m.inv_np1);
    return EXACT ? s / diag : __fdividef(s, diag);
  } else if constexpr (OP == MG_DEV) {
    // D = L(w + x) - L(w): per neighbour, twice the new face coefficient
    // b = E_j + E_i with E = e^{w + x} = e^w e^x, and its change t
    const float E0 = __expf(wc), q2 = 0.5f * ih2;
    float ec;
    const float Tc = E0 * em1(xc, &ec), Ec = E0 * ec;
    float acc = 0.f, sd = 0.f, sb = 0.f;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const float En = __expf(wn[q]);
      float en;
      const float t = fmaf(En, em1(xn[q], &en), Tc), b = fmaf(En, en, Ec);
      const float dw = wn[q] - wc, dx = xn[q] - xc;
      acc = fmaf(b, dx, fmaf(t, dw, acc));
      sd += dw + dx;
      sb += b;
    }
    const float s0 = __expf(-wc * m.inv_np1);
    float es;
    const float y = em1(-xc * m.inv_np1, &es);
    const float D = acc * q2 - m.aRt * s0 * y;
    const float dL = (Ec * sd - sb) * q2 + m.aRt_np1 * s0 * es;
    const float step = __fdividef(D - r, dL);
    return xc - fminf(fmaxf(step, -m.cap), m.cap);
  } else {
    const float s = xn[0] + xn[1] + xn[2] + xn[3] + xn[4] + xn[5];
    return (s - h2 * r) * (1.f / 6.f);
  }
}

// the operator applied at a cell (MG_NL: L(x); else the left-hand side above)
template <int OP>
__device__ __forceinline__ float point_apply(float xc, const float* xn, float wc, const float* wn,
                                             const PF& m, float ih2) {
  if constexpr (OP == MG_NL) {
    const float Ec = __expf(xc);
    float sbd = 0.f;
#pragma unroll
    for (int e = 0; e < 6; ++e) sbd = fmaf(0.5f * (__expf(xn[e]) + Ec), xn[e] - xc, sbd);
    return sbd * ih2 + m.aRt * (1.f - __expf(-xc * m.inv_np1));
  } else if constexpr (OP == MG_LIN) {
    const float Ec = __expf(wc), q2 = 0.5f * ih2;
    float d = 0.f, off[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const float En = __expf(wn[q]), du = wn[q] - wc;
      off[q] = q2 * fmaf(En, du, Ec + En);
      d += fmaf(Ec, du, -Ec - En);
    }
    float J = (d * q2 + m.aRt_np1 * __expf(-wc * m.inv_np1)) * xc;
#pragma unroll
    for (int q = 0; q < 6; ++q) J = fmaf(off[q], xn[q], J);
    return J;
  } else if constexpr (OP == MG_DEV) {
    const float E0 = __expf(wc);
    float ec;
    const float Tc = E0 * em1(xc, &ec), Ec = E0 * ec;
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const float En = __expf(wn[q]);
      float en;
      const float t = fmaf(En, em1(xn[q], &en), Tc), b = fmaf(En, en, Ec);
      acc = fmaf(b, xn[q] - xc, fmaf(t, wn[q] - wc, acc));
    }
    return acc * (0.5f * ih2) - m.aRt * __expf(-wc * m.inv_np1) * em1(-xc * m.inv_np1);
  } else {
    const float s = xn[0] + xn[1] + xn[2] + xn[3] + xn[4] + xn[5];
    return (s - 6.f * xc) * ih2;
  }
}

// ---- four cells per thread ---------------------------------------------------
struct V4 {
  float v[4];
};
__device__ __forceinline__ V4 ld4(const float* __restrict__ p) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  return V4{{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ void st4(float* __restrict__ p, const V4& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}

// row offsets (within a plane) of (i, j) and its row neighbours at kh0
struct Rows {
  unsigned c, xm, xp, ym, yp;
  unsigned zs;  // the z neighbour outside the vector: one step before (p = 0) or after (p = 1)
};
__device__ __forceinline__ Rows rows_at(int i, int j, int kh0, int p, int lg) {
  const int M = (1 << lg) - 1, hm = M >> 1;
  Rows r;
  r.c = prow(i, j, lg) + kh0;
  r.xm = prow((i - 1) & M, j, lg) + kh0;
  r.xp = prow((i + 1) & M, j, lg) + kh0;
  r.ym = prow(i, (j - 1) & M, lg) + kh0;
  r.yp = prow(i, (j + 1) & M, lg) + kh0;
  r.zs = prow(i, j, lg) + ((p ? kh0 + 4 : kh0 - 1) & hm);
  return r;
}

// the six neighbours (in the other colour's plane) of four cells of a row with
// k parity p: nb[t][0..5]
struct Nb4 {
  V4 xm, xp, ym, yp;
  float z[5];
  __device__ __forceinline__ void get(int t, float* o) const {
    o[0] = xm.v[t];
    o[1] = xp.v[t];
    o[2] = ym.v[t];
    o[3] = yp.v[t];
    o[4] = z[t];
    o[5] = z[t + 1];
  }
};
__device__ __forceinline__ Nb4 load_nb(const float* __restrict__ o, const Rows& r, int p) {
  Nb4 n;
  n.xm = ld4(o + r.xm);
  n.xp = ld4(o + r.xp);
  n.ym = ld4(o + r.ym);
  n.yp = ld4(o + r.yp);
  const V4 c = ld4(o + r.c);
  const float s = o[r.zs];
  n.z[0] = p ? c.v[0] : s;
  n.z[1] = p ? c.v[1] : c.v[0];
  n.z[2] = p ? c.v[2] : c.v[1];
  n.z[3] = p ? c.v[3] : c.v[2];
  n.z[4] = p ? s : c.v[3];
  return n;
}

// half-sweep of colour `colour`: xs, ws its planes of x and w, xo, wo the
// other colour's, rs its plane of r
template <int OP>
__global__ void __launch_bounds__(BS) k_vsweep(float* __restrict__ xs, const float* __restrict__ xo,
                                               const float* __restrict__ rs,
                                               const float* __restrict__ ws,
                                               const float* __restrict__ wo, int lg, int colour,
                                               PF m, float ih2, float h2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg - 3))) return;
  const int M = (1 << lg) - 1;
  const int kh0 = 4 * (int)(t & ((1u << (lg - 3)) - 1));
  const int j = (int)((t >> (lg - 3)) & M), i = (int)(t >> (2 * lg - 3));
  const int p = (i + j + colour) & 1;
  const Rows R = rows_at(i, j, kh0, p, lg);
  const Nb4 xn = load_nb(xo, R, p);
  const V4 r = ld4(rs + R.c);
  V4 xc{}, wc{}, out;
  if (OP == MG_NL || OP == MG_DEV) xc = ld4(xs + R.c);
  Nb4 wn{};
  if (OP == MG_LIN || OP == MG_DEV) {
    wn = load_nb(wo, R, p);
    wc = ld4(ws + R.c);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float a[6], b[6];
    xn.get(q, a);
    wn.get(q, b);
    out.v[q] = point_update<OP>(xc.v[q], a, wc.v[q], b, r.v[q], m, ih2, h2);
  }
  st4(xs + R.c, out);
}

// FAS right-hand side f += L(u) of a coarse level (Eq. (27))
__global__ void __launch_bounds__(BS) k_vfas(const float* __restrict__ x, float* __restrict__ f,
                                             int lg, PF m, float ih2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lg - 2))) return;
  const unsigned half = 1u << (3 * lg - 1);
  const int M = (1 << lg) - 1;
  const int kh0 = 4 * (int)(t & ((1u << (lg - 3)) - 1));
  const int j = (int)((t >> (lg - 3)) & M), i = (int)((t >> (2 * lg - 3)) & M);
  const int colour = (int)(t >> (3 * lg - 3)), p = (i + j + colour) & 1;
  const Rows R = rows_at(i, j, kh0, p, lg);
  const Nb4 xn = load_nb(x + (1 - colour) * half, R, p);
  const V4 xc = ld4(x + colour * half + R.c);
  V4 fv = ld4(f + colour * half + R.c);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float a[6];
    xn.get(q, a);
    fv.v[q] += point_apply<MG_NL>(xc.v[q], a, 0.f, a, m, ih2);
  }
  st4(f + colour * half + R.c, fv);
}

// Restriction to four coarse cells (I, J, K0..K0+3): the average of the eight
// daughters' residuals, and of the iterate (NL: x; LIN: w; DEV: w + x), the
// daughters visited in C order.  The daughters of a fine row are one vector
// of each colour.
template <int OP>
__global__ void __launch_bounds__(BS) k_vrestrict(const float* __restrict__ x,
                                                  const float* __restrict__ r,
                                                  const float* __restrict__ w, int lgf,
                                                  float* __restrict__ xc, float* __restrict__ rc,
                                                  float* __restrict__ wc, PF m, float ih2) {
  const int lgc = lgf - 1, Mc = (1 << lgc) - 1;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lgc - 2))) return;
  const int K0 = 4 * (int)(t & ((1u << (lgc - 2)) - 1));
  const int J = (int)((t >> (lgc - 2)) & Mc), I = (int)(t >> (2 * lgc - 2));
  const unsigned half = 1u << (3 * lgf - 1);
  float sr[4] = {0.f, 0.f, 0.f, 0.f}, su[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int ab = 0; ab < 4; ++ab) {
    const int i = 2 * I + (ab >> 1), j = 2 * J + (ab & 1);
    const int qe = (i + j) & 1;  // the plane of the row's even k
    V4 res[2], val[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {  // k = 2K + c
      const unsigned own = ((qe ^ c) ? half : 0u), oth = half - own;
      const Rows R = rows_at(i, j, K0, c, lgf);
      const Nb4 xn = load_nb(x + oth, R, c);
      const V4 xv = ld4(x + own + R.c), rv = ld4(r + own + R.c);
      Nb4 wn{};
      V4 wv{};
      if (OP == MG_LIN || OP == MG_DEV) {
        wn = load_nb(w + oth, R, c);
        wv = ld4(w + own + R.c);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a[6], b[6];
        xn.get(q, a);
        wn.get(q, b);
        res[c].v[q] = rv.v[q] - point_apply<OP>(xv.v[q], a, wv.v[q], b, m, ih2);
        val[c].v[q] = OP == MG_NL ? xv.v[q] : (OP == MG_DEV ? wv.v[q] + xv.v[q] : wv.v[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        sr[q] += res[c].v[q];
        su[q] += val[c].v[q];
      }
  }
  // coarse cells K0, K0+2 lie in the plane of I + J, K0+1, K0+3 in the other
  const unsigned halfc = 1u << (3 * lgc - 1), row = prow(I, J, lgc) + (K0 >> 1);
  const unsigned pe = ((I + J) & 1) ? halfc : 0u, po = halfc - pe;
  auto put = [&](float* dst, const float* v) {
    *reinterpret_cast<float2*>(dst + pe + row) = make_float2(0.125f * v[0], 0.125f * v[2]);
    *reinterpret_cast<float2*>(dst + po + row) = make_float2(0.125f * v[1], 0.125f * v[3]);
  };
  put(rc, sr);
  if (OP == MG_NL) {
    put(xc, su);
    put(wc, su);
  } else {
    const float z[4] = {0.f, 0.f, 0.f, 0.f};
    put(xc, z);
    if (OP != MG_POI) put(wc, su);
  }
}

// x += P(c) with c = xc - wc (NL) or xc: four coarse cells, their 32 daughters
template <int OP>
__global__ void __launch_bounds__(BS) k_vprolong(float* __restrict__ x, const float* __restrict__ xc,
                                                 const float* __restrict__ wc, int lgf,
                                                 int linear) {
  const int lgc = lgf - 1, Mc = (1 << lgc) - 1, hmc = Mc >> 1;
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (1u << (3 * lgc - 2))) return;
  const int K0 = 4 * (int)(t & ((1u << (lgc - 2)) - 1));
  const int J = (int)((t >> (lgc - 2)) & Mc), I = (int)(t >> (2 * lgc - 2));
  const unsigned halfc = 1u << (3 * lgc - 1);
  // coarse values of row (a, b) at K0..K0+3
  auto row4 = [&](int a, int b) {
    const unsigned q = prow(a, b, lgc) + (K0 >> 1);
    const unsigned pe = ((a + b) & 1) ? halfc : 0u, po = halfc - pe;
    float2 e = *reinterpret_cast<const float2*>(xc + pe + q);
    float2 o = *reinterpret_cast<const float2*>(xc + po + q);
    if (OP == MG_NL) {
      const float2 e0 = *reinterpret_cast<const float2*>(wc + pe + q);
      const float2 o0 = *reinterpret_cast<const float2*>(wc + po + q);
      e.x -= e0.x;
      e.y -= e0.y;
      o.x -= o0.x;
      o.y -= o0.y;
    }
    return V4{{e.x, o.x, e.y, o.y}};
  };
  const V4 c = row4(I, J);
  float gx[4], gy[4], gz[4];
  if (linear) {
    const V4 xp = row4((I + 1) & Mc, J), xm = row4((I - 1) & Mc, J);
    const V4 yp = row4(I, (J + 1) & Mc), ym = row4(I, (J - 1) & Mc);
    // K0 - 1 is odd, K0 + 4 even
    const unsigned rw = prow(I, J, lgc);
    const unsigned pe = ((I + J) & 1) ? halfc : 0u, po = halfc - pe;
    const unsigned am = po + rw + (((K0 - 1) & Mc) >> 1), ap = pe + rw + (((K0 >> 1) + 2) & hmc);
    float zm = xc[am], zp = xc[ap];
    if (OP == MG_NL) {
      zm -= wc[am];
      zp -= wc[ap];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      gx[q] = xp.v[q] - xm.v[q];
      gy[q] = yp.v[q] - ym.v[q];
      gz[q] = (q < 3 ? c.v[q + 1] : zp) - (q > 0 ? c.v[q - 1] : zm);
    }
  }
  const unsigned half = 1u << (3 * lgf - 1);
#pragma unroll
  for (int ab = 0; ab < 4; ++ab) {
    const int i = 2 * I + (ab >> 1), j = 2 * J + (ab & 1);
    const unsigned rw = prow(i, j, lgf) + K0;
    const int qe = (i + j) & 1;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float* dst = x + ((qe ^ k) ? half : 0u) + rw;
      V4 v = ld4(dst);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float d = c.v[q];
        if (linear) {
          d += ((ab >> 1) ? 0.125f : -0.125f) * gx[q];
          d += ((ab & 1) ? 0.125f : -0.125f) * gy[q];
          d += (k ? 0.125f : -0.125f) * gz[q];
        }
        v.v[q] += d;
      }
      st4(dst, v);
    }
  }
}

__device__ __forceinline__ void block_partial(double ss, float mx, double* __restrict__ partials) {
  __shared__ double s1[BS / 32];
  __shared__ float s2[BS / 32];
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s1[threadIdx.x >> 5] = ss;
    s2[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    float b = 0.f;
    for (int w = 0; w < BS / 32; ++w) {
      a += s1[w];
      b = fmaxf(b, s2[w]);
    }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = (double)b;
  }
}

// residual norm of the nonlinear FP32 iterate; a thread sums the squares of
// four cells in FP32, the vectors are summed in FP64 (an FP64 addition per
// cell made this the slowest kernel of the cycle: 860 us on 512^3)
__global__ void __launch_bounds__(BS) k_vnorm(const float* __restrict__ x,
                                              const float* __restrict__ f, int lg, PF m, float ih2,
                                              double* __restrict__ partials) {
  const unsigned half = 1u << (3 * lg - 1), nv = 1u << (3 * lg - 2);
  const int M = (1 << lg) - 1;
  double ss = 0.0;
  float mx = 0.f;
  for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < nv; t += gridDim.x * blockDim.x) {
    const int kh0 = 4 * (int)(t & ((1u << (lg - 3)) - 1));
    const int j = (int)((t >> (lg - 3)) & M), i = (int)((t >> (2 * lg - 3)) & M);
    const int colour = (int)(t >> (3 * lg - 3)), p = (i + j + colour) & 1;
    const Rows R = rows_at(i, j, kh0, p, lg);
    const Nb4 xn = load_nb(x + (1 - colour) * half, R, p);
    const V4 xv = ld4(x + colour * half + R.c), fv = ld4(f + colour * half + R.c);
    float s4 = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a[6];
      xn.get(q, a);
      const float r = fv.v[q] - point_apply<MG_NL>(xv.v[q], a, 0.f, a, m, ih2);
      s4 = fmaf(r, r, s4);
      mx = fmaxf(mx, fabsf(r));
    }
    ss += (double)s4;
  }
  block_partial(ss, mx, partials);
}

__global__ void k_finish2(const double* __restrict__ partials, int nparts, double* __restrict__ out) {
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

// ---- 32^3 and below: one cluster ----------------------------------------------
// Shared memory of a CTA, floats: for the 32^3 and the 16^3 level its slab of
// x, r, w and the residual scratch t (C order in the slab); in the first CTA
// also the 8^3 and 4^3 levels whole.
constexpr int BT = 512;
constexpr int kBotMaxLg = 5;

struct BotArgs {
  int lg;             // the finest level held, 3..5
  float *x, *r, *w;   // its arrays (colour-split, global)
  float ih2[4], h2[4];  // of levels lg, lg - 1, ...
  PF m;
  int n_pre, n_post, linear, coarse_sweeps;
  float coarse_rel;
};

struct BotGrid {      // where a level lives
  int lg, dist;       // dist: slabs over the cluster, else whole in the first CTA
  int lpc;            // log2 of the planes per CTA (dist)
  int off;            // floats before its x in a CTA's shared memory
  int cells;          // cells per CTA
  __device__ __forceinline__ int idx(int i, int j, int k) const {
    const int li = dist ? (i & ((1 << lpc) - 1)) : i;
    return (((li << lg) + j) << lg) + k;
  }
  __device__ __forceinline__ int rank(int i) const { return dist ? i >> lpc : 0; }
};

template <int OP>
struct Bot {
  float* sm;          // this CTA's shared memory
  int me, nb;         // rank, CTAs
  cg::cluster_group cl;
  __device__ Bot(float* s) : sm(s), cl(cg::this_cluster()) {
    me = (int)cl.block_rank();
    nb = (int)cl.num_blocks();
  }
  // array a (0 x, 1 r, 2 w, 3 scratch) of a level in CTA q
  __device__ __forceinline__ float* arr(const BotGrid& g, int a, int q) const {
    float* p = sm + g.off + a * g.cells;
    return q == me ? p : cl.map_shared_rank(p, q);
  }
  __device__ __forceinline__ void sync(const BotGrid& g) const {
    if (g.dist)
      cl.sync();
    else
      __syncthreads();
  }
  __device__ __forceinline__ bool mine(const BotGrid& g) const { return g.dist || me == 0; }
  __device__ __forceinline__ int plane0(const BotGrid& g) const {
    return g.dist ? me << g.lpc : 0;
  }
  __device__ __forceinline__ void nbrs(const BotGrid& g, int a, int i, int j, int k,
                                       float* o) const {
    const int M = (1 << g.lg) - 1;
    const int im = (i - 1) & M, ip = (i + 1) & M;
    const float* own = sm + g.off + a * g.cells;
    o[0] = arr(g, a, g.rank(im))[g.idx(im, j, k)];
    o[1] = arr(g, a, g.rank(ip))[g.idx(ip, j, k)];
    o[2] = own[g.idx(i, (j - 1) & M, k)];
    o[3] = own[g.idx(i, (j + 1) & M, k)];
    o[4] = own[g.idx(i, j, (k - 1) & M)];
    o[5] = own[g.idx(i, j, (k + 1) & M)];
  }
  __device__ void sweep(const BotGrid& g, int colour, const PF& m, float ih2, float h2) {
    const int M = (1 << g.lg) - 1;
    float *x = sm + g.off, *r = x + g.cells, *w = x + 2 * g.cells;
    for (int t = threadIdx.x; t < g.cells / 2; t += BT) {
      const int k2 = t & (M >> 1), j = (t >> (g.lg - 1)) & M;
      const int i = plane0(g) + (t >> (2 * g.lg - 1));
      const int k = 2 * k2 + ((i + j + colour) & 1);
      const int c = g.idx(i, j, k);
      float xn[6], wn[6];
      nbrs(g, 0, i, j, k, xn);
      if (OP == MG_LIN || OP == MG_DEV) nbrs(g, 2, i, j, k, wn);
      x[c] = point_update<OP>(x[c], xn, OP == MG_NL || OP == MG_POI ? 0.f : w[c], wn, r[c], m, ih2,
                              h2);
    }
  }
  __device__ __forceinline__ float apply(const BotGrid& g, int i, int j, int k, int c, const PF& m,
                                         float ih2) const {
    const float *x = sm + g.off, *w = x + 2 * g.cells;
    float xn[6], wn[6];
    nbrs(g, 0, i, j, k, xn);
    if (OP == MG_LIN || OP == MG_DEV) nbrs(g, 2, i, j, k, wn);
    return point_apply<OP>(x[c], xn, OP == MG_NL || OP == MG_POI ? 0.f : w[c], wn, m, ih2);
  }
  // residual of every cell of this CTA's part into its scratch
  __device__ void resid(const BotGrid& g, const PF& m, float ih2) {
    const int M = (1 << g.lg) - 1;
    float *x = sm + g.off, *r = x + g.cells, *s = x + 3 * g.cells;
    for (int c = threadIdx.x; c < g.cells; c += BT) {
      const int k = c & M, j = (c >> g.lg) & M, i = plane0(g) + (c >> (2 * g.lg));
      s[c] = r[c] - apply(g, i, j, k, c, m, ih2);
    }
  }
  __device__ void restrict_(const BotGrid& f, const BotGrid& g) {
    const int M = (1 << g.lg) - 1;
    float *x = sm + g.off, *r = x + g.cells, *w = x + 2 * g.cells;
    for (int c = threadIdx.x; c < g.cells; c += BT) {
      const int K = c & M, J = (c >> g.lg) & M, I = plane0(g) + (c >> (2 * g.lg));
      float sr = 0.f, su = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int i = 2 * I + (q >> 2), j = 2 * J + ((q >> 1) & 1), k = 2 * K + (q & 1);
        const int rk = f.rank(i), e = f.idx(i, j, k);
        sr += arr(f, 3, rk)[e];
        if (OP == MG_NL) su += arr(f, 0, rk)[e];
        if (OP == MG_LIN) su += arr(f, 2, rk)[e];
        if (OP == MG_DEV) su += arr(f, 2, rk)[e] + arr(f, 0, rk)[e];
      }
      r[c] = 0.125f * sr;
      w[c] = 0.125f * su;
      x[c] = OP == MG_NL ? 0.125f * su : 0.f;
    }
  }
  __device__ void fas(const BotGrid& g, const PF& m, float ih2) {
    const int M = (1 << g.lg) - 1;
    float* r = sm + g.off + g.cells;
    for (int c = threadIdx.x; c < g.cells; c += BT) {
      const int k = c & M, j = (c >> g.lg) & M, i = plane0(g) + (c >> (2 * g.lg));
      r[c] += apply(g, i, j, k, c, m, ih2);
    }
  }
  __device__ void prolong(const BotGrid& f, const BotGrid& g, int linear) {
    const int M = (1 << f.lg) - 1, Mc = M >> 1;
    float* x = sm + f.off;
    auto corr = [&](int a, int b, int c) {
      a &= Mc;
      const int e = g.idx(a, b & Mc, c & Mc), rk = g.rank(a);
      const float v = arr(g, 0, rk)[e];
      return OP == MG_NL ? v - arr(g, 2, rk)[e] : v;
    };
    for (int c = threadIdx.x; c < f.cells; c += BT) {
      const int k = c & M, j = (c >> f.lg) & M, i = plane0(f) + (c >> (2 * f.lg));
      const int I = i >> 1, J = j >> 1, K = k >> 1;
      float v = corr(I, J, K);
      if (linear) {
        v += ((i & 1) ? 0.125f : -0.125f) * (corr(I + 1, J, K) - corr(I - 1, J, K));
        v += ((j & 1) ? 0.125f : -0.125f) * (corr(I, J + 1, K) - corr(I, J - 1, K));
        v += ((k & 1) ? 0.125f : -0.125f) * (corr(I, J, K + 1) - corr(I, J, K - 1));
      }
      x[c] += v;
    }
  }
  // the 4^3 grid by the first warp (one colour's 32 cells per half-sweep):
  // until no cell changes any more (DEV and POI: by more than its rounding), or
  // the residual has dropped by `rel` (checked every four sweeps), or `sweeps`
  __device__ void coarse(const BotGrid& g, const PF& m, float ih2, float h2, int sweeps,
                         float rel) {
    if (threadIdx.x >= 32) return;
    float *x = sm + g.off, *r = x + g.cells, *w = x + 2 * g.cells;
    const int t = threadIdx.x, k2 = t & 1, j = (t >> 1) & 3, i = t >> 3;
    int c[2], nb[2][6];
    float wn[2][6], wc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = 2 * k2 + ((i + j + q) & 1);
      c[q] = (((i << 2) + j) << 2) + k;
      nb[q][0] = ((((i + 3) & 3) << 2) + j) * 4 + k;
      nb[q][1] = ((((i + 1) & 3) << 2) + j) * 4 + k;
      nb[q][2] = ((i << 2) + ((j + 3) & 3)) * 4 + k;
      nb[q][3] = ((i << 2) + ((j + 1) & 3)) * 4 + k;
      nb[q][4] = ((i << 2) + j) * 4 + ((k + 3) & 3);
      nb[q][5] = ((i << 2) + j) * 4 + ((k + 1) & 3);
      wc[q] = w[c[q]];
#pragma unroll
      for (int e = 0; e < 6; ++e) wn[q][e] = w[nb[q][e]];
    }
    float r0 = -1.f;
    for (int s = 0; s < sweeps; ++s) {
      if (rel > 0.f && (s & 3) == 0) {
        float mx = 0.f;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float xn[6];
#pragma unroll
          for (int e = 0; e < 6; ++e) xn[e] = x[nb[q][e]];
          mx = fmaxf(mx, fabsf(r[c[q]] - point_apply<OP>(x[c[q]], xn, wc[q], wn[q], m, ih2)));
        }
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (r0 < 0.f) r0 = mx;
        if (mx <= rel * r0) break;
      }
      bool changed = false;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float xn[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) xn[e] = x[nb[q][e]];
        const float old = x[c[q]];
        constexpr bool exact = OP == MG_NL || OP == MG_LIN;
        const float v = point_update<OP, exact>(old, xn, wc[q], wn[q], r[c[q]], m, ih2, h2);
        changed = changed || (exact ? v != old : fabsf(v - old) > 1.2e-7f * fabsf(v));
        __syncwarp();
        x[c[q]] = v;
        __syncwarp();
      }
      if (!__any_sync(0xffffffffu, changed)) break;
    }
  }
};

template <int OP>
__global__ void __launch_bounds__(BT, 1) k_bottom(BotArgs A) {
  extern __shared__ float smem[];
  Bot<OP> B(smem);
  BotGrid G[4];
  const int nl = A.lg - 1;  // levels lg .. 2
  int off = 0, lnb = 0;
  while ((1 << lnb) < B.nb) ++lnb;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    if (l >= nl) break;
    BotGrid& g = G[l];
    g.lg = A.lg - l;
    g.dist = g.lg >= 4 && B.nb > 1;
    g.lpc = g.lg - lnb;
    g.cells = g.dist ? 1 << (2 * g.lg + g.lpc) : 1 << (3 * g.lg);
    g.off = off;
    off += 4 * g.cells;
  }
  // load the finest level (its w is the linearisation point; NL: not used)
  if (B.mine(G[0])) {
    const int M = (1 << A.lg) - 1;
    float* x = smem + G[0].off;
    for (int c = threadIdx.x; c < G[0].cells; c += BT) {
      const int k = c & M, j = (c >> A.lg) & M, i = B.plane0(G[0]) + (c >> (2 * A.lg));
      const unsigned q = pdx(i, j, k, A.lg);
      x[c] = A.x[q];
      x[G[0].cells + c] = A.r[q];
      if (OP == MG_LIN || OP == MG_DEV) x[2 * G[0].cells + c] = A.w[q];
    }
  }
  B.sync(G[0]);
  auto relax = [&](int l, int n) {
    for (int s = 0; s < n; ++s)
      for (int col = 0; col < 2; ++col) {
        B.sweep(G[l], col, A.m, A.ih2[l], A.h2[l]);
        B.sync(G[l]);
      }
  };
  // down; a level not spread over the cluster is the first CTA's alone, the
  // others wait at the cluster barrier after it
  for (int l = 0; l + 1 < nl; ++l) {
    if (B.mine(G[l])) {
      relax(l, A.n_pre);
      B.resid(G[l], A.m, A.ih2[l]);
    }
    if (G[l].dist) B.cl.sync(); else __syncthreads();
    if (B.mine(G[l + 1])) B.restrict_(G[l], G[l + 1]);
    if (OP == MG_NL) {
      if (G[l + 1].dist) B.cl.sync(); else __syncthreads();
      if (B.mine(G[l + 1])) B.fas(G[l + 1], A.m, A.ih2[l + 1]);
    }
    if (G[l + 1].dist) B.cl.sync(); else __syncthreads();
  }
  if (B.me == 0) B.coarse(G[nl - 1], A.m, A.ih2[nl - 1], A.h2[nl - 1], A.coarse_sweeps, A.coarse_rel);
  __syncthreads();
  for (int l = nl - 2; l >= 0; --l) {
    // a spread level reads the first CTA's grid: every CTA waits for it
    if (G[l].dist && !G[l + 1].dist) B.cl.sync();
    if (B.mine(G[l])) B.prolong(G[l], G[l + 1], A.linear);
    if (G[l].dist) B.cl.sync(); else __syncthreads();
    if (B.mine(G[l])) relax(l, A.n_post);
  }
  if (B.mine(G[0])) {
    const int M = (1 << A.lg) - 1;
    const float* x = smem + G[0].off;
    for (int c = threadIdx.x; c < G[0].cells; c += BT) {
      const int k = c & M, j = (c >> A.lg) & M, i = B.plane0(G[0]) + (c >> (2 * A.lg));
      A.x[pdx(i, j, k, A.lg)] = x[c];
    }
  }
  if (B.nb > 1) B.cl.sync();  // no CTA leaves while another may read its memory
}

// shared memory of one CTA for finest level lg over nb CTAs
size_t bottom_smem(int lg, int nb) {
  size_t f = 0;
  for (int l = lg; l >= 2; --l) {
    const size_t n = (size_t)1 << (3 * l);
    f += 4 * (l >= 4 && nb > 1 ? n / nb : n);
  }
  return f * sizeof(float);
}

std::atomic<int> g_bot_ctas[64];  // per device: CTAs of a cluster for 32^3 and 16^3 (16 or 8; 0 unknown)

template <int OP>
cudaError_t bottom_attrs(int* ctas) {
  cudaError_t e = cudaFuncSetAttribute(k_bottom<OP>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_bottom<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)bottom_smem(kBotMaxLg, 8));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(BT);
  cfg.dynamicSmemBytes = bottom_smem(kBotMaxLg, 16);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, k_bottom<OP>, &cfg);
  if (e != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    *ctas = 8;
  }
  return cudaSuccess;
}

template <int OP>
void launch_bottom(const BotArgs& A, cudaStream_t s) {
  int dev = 0;
  cudaGetDevice(&dev);
  const int nb = A.lg >= 4 ? (dev < 64 && g_bot_ctas[dev] == 16 ? 16 : 8) : 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nb);
  cfg.blockDim = dim3(BT);
  cfg.dynamicSmemBytes = bottom_smem(A.lg, nb);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nb;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_bottom<OP>, A);
}

template <int OP>
long long cycle(const Mg32Level* L, int nlev, const Mg32Par& p, cudaStream_t s,
                const Mg32Hook* hook) {
  const PF m{p.aRt, p.aRt_np1, p.inv_np1, p.cap};
  long long upd = 0;
  for (int l = 0; l + 1 < nlev; ++l) upd += (long long)(p.n_pre + p.n_post) << (3 * L[l].lg);
  int lb = 0;  // the first level of the cluster kernel
  while (L[lb].lg > kBotMaxLg) ++lb;
  auto relax = [&](int l, int n) {
    const Mg32Level& F = L[l];
    const size_t half = (size_t)1 << (3 * F.lg - 1);
    for (int q = 0; q < n; ++q)
      for (int col = 0; col < 2; ++col) {
        if (l == 0 && hook) hook->begin(hook->arg);
        k_vsweep<OP><<<nblocks((long long)half / 4, BS), BS, 0, s>>>(
            F.x + col * half, F.x + (1 - col) * half, F.r + col * half,
            F.w ? F.w + col * half : nullptr, F.w ? F.w + (1 - col) * half : nullptr, F.lg, col, m,
            F.ih2, F.h2);
        if (l == 0 && hook) hook->end(hook->arg);
      }
  };
  for (int l = 0; l < lb; ++l) {
    const Mg32Level &F = L[l], &C = L[l + 1];
    const long long nc = 1LL << (3 * C.lg);
    relax(l, p.n_pre);
    k_vrestrict<OP><<<nblocks(nc / 4, BS), BS, 0, s>>>(F.x, F.r, F.w, F.lg, C.x, C.r, C.w, m,
                                                       F.ih2);
    if (OP == MG_NL) k_vfas<<<nblocks(nc / 4, BS), BS, 0, s>>>(C.x, C.r, C.lg, m, C.ih2);
  }
  BotArgs A{};
  A.lg = L[lb].lg;
  A.x = L[lb].x;
  A.r = L[lb].r;
  A.w = L[lb].w;
  for (int l = lb; l < nlev; ++l) {
    A.ih2[l - lb] = L[l].ih2;
    A.h2[l - lb] = L[l].h2;
  }
  A.m = m;
  A.n_pre = p.n_pre;
  A.n_post = p.n_post;
  A.linear = p.linear;
  A.coarse_sweeps = p.coarse_sweeps;
  A.coarse_rel = p.coarse_rel;
  launch_bottom<OP>(A, s);
  for (int l = lb - 1; l >= 0; --l) {
    const Mg32Level &F = L[l], &C = L[l + 1];
    k_vprolong<OP><<<nblocks((1LL << (3 * C.lg)) / 4, BS), BS, 0, s>>>(F.x, C.x, C.w, F.lg,
                                                                       p.linear);
    relax(l, p.n_post);
  }
  return upd;
}

}  // namespace

mgfr_status mg32_prepare(mgfr_ctx* c) {
  const int dev = c->device;
  if (dev >= 0 && dev < 64 && g_bot_ctas[dev]) return MGFR_OK;
  int ctas = 16;
  MG_CK(c, bottom_attrs<MG_NL>(&ctas));
  MG_CK(c, bottom_attrs<MG_LIN>(&ctas));
  MG_CK(c, bottom_attrs<MG_DEV>(&ctas));
  MG_CK(c, bottom_attrs<MG_POI>(&ctas));
  if (dev >= 0 && dev < 64) g_bot_ctas[dev] = ctas;
  return MGFR_OK;
}

long long mg32_cycle(Mg32Op op, const Mg32Level* L, int nlev, const Mg32Par& p, cudaStream_t s,
                     const Mg32Hook* hook) {
  switch (op) {
    case MG_NL: return cycle<MG_NL>(L, nlev, p, s, hook);
    case MG_LIN: return cycle<MG_LIN>(L, nlev, p, s, hook);
    case MG_DEV: return cycle<MG_DEV>(L, nlev, p, s, hook);
    default: return cycle<MG_POI>(L, nlev, p, s, hook);
  }
}

void mg32_norm(const Mg32Level& L, const Mg32Par& p, double* partials, int nparts, double* out,
               cudaStream_t s) {
  const long long nv = 1LL << (3 * L.lg - 2);
  const int nb = (int)std::min<long long>(nparts, nblocks(nv, BS));
  k_vnorm<<<nb, BS, 0, s>>>(L.x, L.r, L.lg, PF{p.aRt, p.aRt_np1, p.inv_np1, p.cap}, L.ih2,
                            partials);
  k_finish2<<<1, 256, 0, s>>>(partials, nb, out);
}

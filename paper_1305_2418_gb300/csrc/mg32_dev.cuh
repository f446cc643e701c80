// mg32_dev.cuh -- device code of the FP32 V-cycles on dense levels: the point
// operations of the four operators (mg32.cuh) and the loads of four cells of a
// colour with their neighbours from colour-split storage.
#pragma once
#include "colour_split.cuh"
#include "em1_series.h"
#include "mg32.cuh"

namespace {

// e^x - 1, and e^x in *e: the Taylor series for |x| <= 0.35 (1.9e-8 of the result and its
// roundings), beyond it the exponential less one, whose 2 ulp are up to 6e-7 of the result
// there (0.42 at x = 0.35, 0.30 at -0.35) and less further out
__device__ __forceinline__ float em1(float x, float* e) {
  const float q = em1_series(x);
  const bool small = fabsf(x) <= kEm1Small;
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

// ---- one work item (four cells) of a level; t: the item ----------------------
// half-sweep of colour `colour`: xs, ws its planes of x and w, xo, wo the
// other colour's, rs its plane of r
template <int OP>
__device__ __forceinline__ void vec_sweep(unsigned t, float* __restrict__ xs, const float* __restrict__ xo,
                                               const float* __restrict__ rs,
                                               const float* __restrict__ ws,
                                               const float* __restrict__ wo, int lg, int colour,
                                               PF m, float ih2, float h2) {
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
__device__ __forceinline__ void vec_fas(unsigned t, const float* __restrict__ x, float* __restrict__ f,
                                             int lg, PF m, float ih2) {
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

// One fine row (i, j) of the restriction to the coarse cells K0..K0+3: the residuals (res)
// and the values to be averaged (val: NL: x; LIN: w; DEV: w + x) of its daughters at even
// k ([0]) and odd k ([1]), one vector of each colour
template <int OP>
__device__ __forceinline__ void restrict_row(const float* __restrict__ x,
                                             const float* __restrict__ r,
                                             const float* __restrict__ w, int i, int j, int K0,
                                             int lgf, const PF& m, float ih2, V4* res, V4* val) {
  const unsigned half = 1u << (3 * lgf - 1);
  const int qe = (i + j) & 1;  // the plane of the row's even k
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
}

// Restriction to four coarse cells (I, J, K0..K0+3): the average of the eight
// daughters' residuals, and of the iterate, the daughters visited in C order
template <int OP>
__device__ __forceinline__ void vec_restrict(unsigned t, const float* __restrict__ x,
                                                  const float* __restrict__ r,
                                                  const float* __restrict__ w, int lgf,
                                                  float* __restrict__ xc, float* __restrict__ rc,
                                                  float* __restrict__ wc, PF m, float ih2) {
  const int lgc = lgf - 1, Mc = (1 << lgc) - 1;
  const int K0 = 4 * (int)(t & ((1u << (lgc - 2)) - 1));
  const int J = (int)((t >> (lgc - 2)) & Mc), I = (int)(t >> (2 * lgc - 2));
  float sr[4] = {0.f, 0.f, 0.f, 0.f}, su[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int ab = 0; ab < 4; ++ab) {
    V4 res[2], val[2];
    restrict_row<OP>(x, r, w, 2 * I + (ab >> 1), 2 * J + (ab & 1), K0, lgf, m, ih2, res, val);
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

// 4 x 4 values of four consecutive lanes transposed: lane q's v[a] becomes lane a's v[q]
__device__ __forceinline__ void transpose4(float* v) {
  const unsigned lane = threadIdx.x & 31, grp = 0xfu << (lane & 28);
#pragma unroll
  for (int b = 1; b <= 2; b <<= 1)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (r & b) continue;
      const bool hi = lane & b;
      const float got = __shfl_xor_sync(grp, hi ? v[r] : v[r | b], b);
      if (hi)
        v[r] = got;
      else
        v[r | b] = got;
    }
}

// The same by four consecutive lanes, t = 4 (group) + lane: a lane forms the eight
// daughters of one fine row, then takes the sums of one coarse cell, in the same order
template <int OP>
__device__ __forceinline__ void vec_restrict_rows(unsigned t, const float* __restrict__ x,
                                                  const float* __restrict__ r,
                                                  const float* __restrict__ w, int lgf,
                                                  float* __restrict__ xc, float* __restrict__ rc,
                                                  float* __restrict__ wc, PF m, float ih2) {
  const int lgc = lgf - 1, Mc = (1 << lgc) - 1;
  const int ab = (int)(t & 3);
  t >>= 2;
  const int K0 = 4 * (int)(t & ((1u << (lgc - 2)) - 1));
  const int J = (int)((t >> (lgc - 2)) & Mc), I = (int)(t >> (2 * lgc - 2));
  V4 res[2], val[2];
  restrict_row<OP>(x, r, w, 2 * I + (ab >> 1), 2 * J + (ab & 1), K0, lgf, m, ih2, res, val);
  float sr = 0.f, su = 0.f;
  transpose4(res[0].v);
  transpose4(res[1].v);
  if (OP != MG_POI) {
    transpose4(val[0].v);
    transpose4(val[1].v);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      sr += res[c].v[a];
      su += val[c].v[a];
    }
  const unsigned p = pdx(I, J, K0 + ab, lgc);
  rc[p] = 0.125f * sr;
  xc[p] = OP == MG_NL ? 0.125f * su : 0.f;
  if (OP != MG_POI) wc[p] = 0.125f * su;
}

// x += P(c) with c = xc - wc (NL) or xc: four coarse cells, their 32 daughters
// (ROWS 4: one thread; 1: four consecutive lanes, a fine row each)
template <int OP, int ROWS = 4>
__device__ __forceinline__ void vec_prolong(unsigned t, float* __restrict__ x, const float* __restrict__ xc,
                                                 const float* __restrict__ wc, int lgf,
                                                 int linear) {
  const int lgc = lgf - 1, Mc = (1 << lgc) - 1, hmc = Mc >> 1;
  const int row = (int)(t & 3);
  if (ROWS == 1) t >>= 2;
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
  for (int ab0 = 0; ab0 < ROWS; ++ab0) {
    const int ab = ROWS == 1 ? row : ab0;
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

}  // namespace

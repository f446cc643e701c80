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

#include "mg32_dev.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int BS = 256;

template <int OP>
__global__ void __launch_bounds__(BS) k_vsweep(float* __restrict__ xs, const float* __restrict__ xo,
                                               const float* __restrict__ rs,
                                               const float* __restrict__ ws,
                                               const float* __restrict__ wo, int lg, int colour,
                                               PF m, float ih2, float h2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lg - 3))) vec_sweep<OP>(t, xs, xo, rs, ws, wo, lg, colour, m, ih2, h2);
}

__global__ void __launch_bounds__(BS) k_vfas(const float* __restrict__ x, float* __restrict__ f,
                                             int lg, PF m, float ih2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lg - 2))) vec_fas(t, x, f, lg, m, ih2);
}

template <int OP>
__global__ void __launch_bounds__(BS) k_vrestrict(const float* __restrict__ x,
                                                  const float* __restrict__ r,
                                                  const float* __restrict__ w, int lgf,
                                                  float* __restrict__ xc, float* __restrict__ rc,
                                                  float* __restrict__ wc, PF m, float ih2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lgf - 5))) vec_restrict<OP>(t, x, r, w, lgf, xc, rc, wc, m, ih2);
}

template <int OP>
__global__ void __launch_bounds__(128) k_vrestrict_rows(
    const float* __restrict__ x, const float* __restrict__ r, const float* __restrict__ w,
    int lgf, float* __restrict__ xc, float* __restrict__ rc, float* __restrict__ wc, PF m,
    float ih2) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lgf - 3))) vec_restrict_rows<OP>(t, x, r, w, lgf, xc, rc, wc, m, ih2);
}

template <int OP>
__global__ void __launch_bounds__(128) k_vprolong_rows(float* __restrict__ x,
                                                       const float* __restrict__ xc,
                                                       const float* __restrict__ wc, int lgf,
                                                       int linear) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lgf - 3))) vec_prolong<OP, 1>(t, x, xc, wc, lgf, linear);
}

template <int OP>
__global__ void __launch_bounds__(BS) k_vprolong(float* __restrict__ x, const float* __restrict__ xc,
                                                 const float* __restrict__ wc, int lgf,
                                                 int linear) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (1u << (3 * lgf - 5))) vec_prolong<OP>(t, x, xc, wc, lgf, linear);
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

// residual norm of the FP32 iterate x (MG_DEV: of the deviation x from w); a thread sums the squares of
// four cells in FP32, the vectors are summed in FP64 (an FP64 addition per
// cell made this the slowest kernel of the cycle: 860 us on 512^3)
template <int OP>
__global__ void __launch_bounds__(BS) k_vnorm(const float* __restrict__ x,
                                              const float* __restrict__ f,
                                              const float* __restrict__ w, int lg, PF m, float ih2,
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
    V4 wv{};
    Nb4 wn{};
    if (OP == MG_DEV) {
      wn = load_nb(w + (1 - colour) * half, R, p);
      wv = ld4(w + colour * half + R.c);
    }
    float s4 = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float a[6], b[6];
      xn.get(q, a);
      wn.get(q, b);
      const float r = fv.v[q] - point_apply<OP>(xv.v[q], a, wv.v[q], b, m, ih2);
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
// Transfers from levels up to 2^kRowsMax take four lanes per group of four coarse cells,
// larger ones one thread: on 64^3 the 8192 threads of the latter stand on the latency of
// their four rows (restriction in the deviation 15.7 us, 7.5 by rows; prolongation 6.9,
// 4.5), on 128^3 both take the same (21; 7.5), on 256^3 the rows cost more (46 and 70).
constexpr int kRowsMax = 6;

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
    if (F.lg <= kRowsMax)
      k_vrestrict_rows<OP><<<nblocks(nc, 128), 128, 0, s>>>(F.x, F.r, F.w, F.lg, C.x, C.r, C.w, m,
                                                            F.ih2);
    else
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
    const long long nc = 1LL << (3 * C.lg);
    if (F.lg <= kRowsMax)
      k_vprolong_rows<OP><<<nblocks(nc, 128), 128, 0, s>>>(F.x, C.x, C.w, F.lg, p.linear);
    else
      k_vprolong<OP><<<nblocks(nc / 4, BS), BS, 0, s>>>(F.x, C.x, C.w, F.lg, p.linear);
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

void mg32_norm(Mg32Op op, const Mg32Level& L, const Mg32Par& p, double* partials, int nparts,
               double* out, cudaStream_t s) {
  const long long nv = 1LL << (3 * L.lg - 2);
  const int nb = (int)std::min<long long>(nparts, nblocks(nv, BS));
  (op == MG_DEV ? k_vnorm<MG_DEV> : op == MG_POI ? k_vnorm<MG_POI> : k_vnorm<MG_NL>)<<<nb, BS, 0, s>>>(
      L.x, L.r, L.w, L.lg, PF{p.aRt, p.aRt_np1, p.inv_np1, p.cap}, L.ih2, partials);
  k_finish2<<<1, 256, 0, s>>>(partials, nb, out);
}

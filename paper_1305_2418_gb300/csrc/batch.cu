// batch.cu -- many independent dense solves in one persistent launch.
//
// Each solve is the mixed-precision form of the base-level solve (Puchwein,
// Baldi & Springel 2013, Sec. 3.3): FP32 nonlinear FAS V-cycles (mode A)
// until the FP32 residual reaches mixed_switch or stalls, then defect correction
// (mode B): r = f - L(u) in double-float or FP64, one FP32 linear V-cycle on
// J(u) e = r, u += e.  The FP32 arrays are stored by red-black colour and worked
// on four cells per thread (mg32_dev.cuh).  All solves advance together through one V-cycle
// schedule aligned on grid size: at size 2^k every solve with N >= 2^k works
// on its level of that size, so one phase covers all solves; solves are
// sorted by N (descending) so the participants of size 2^k are a prefix and
// every participant has exactly 8^k cells there.  Phases are separated by a
// software grid barrier (cooperative launch guarantees co-residency); every
// wait is bounded by max_spins and sets an error flag instead of hanging.
// Converged solves skip their work items.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "batch_shape.h"
#include "lean_fp64.cuh"
#include "mg32_dev.cuh"

#define BMAXL 9  // levels per solve: N <= 1024 -> 1024..4
constexpr int kMaxBatch = 4096;  // solves of one call

struct BSolve {
  int N, lg, nlev;
  float ih2[BMAXL];
  double ih2_0, h0;
  float aRt, aRt_np1, inv_np1;  // FP32 model
  double aRt64, inv_np1_64, src, fbar, gscale;
  dfl aRt_df, inv_np1_df, ih2h_df;  // alpha Rt, 1/(n+1), 1/(2 h^2)
  int n;
  float* u32[BMAXL];
  float* f32[BMAXL];
  float* uold32[BMAXL];
  float* e32[BMAXL];
  float* r32[BMAXL];
  double *u64, *E64, *f64;
  const double* delta;
  const double* uinit;
  double* fr_out;
  double* acc_out;
  double* u_out;
};

enum { BM_A = 0, BM_B = 1, BM_TRANS = 2, BM_DONE = 3 };

struct BState {
  int mode, cyclesA, cyclesB, pad;
  double ref, target, rprev, r, rmax, r0, fnorm;
  double acc_ss;                 // accumulated sum of squares
  unsigned long long acc_max;    // accumulated max (bits of a non-negative double)
  double acc_ff;
};

struct BArgs {
  BSolve* S;
  BState* st;
  int ns;
  int maxlg;
  int P[16];  // participants per log2 size
  int n_pre, n_post, linear, max_cycles;
  float cap32;
  double tol, sw;
  unsigned* bar_count;
  unsigned* bar_gen;
  int* err;
  long long max_spins;
};

namespace {

// linear index of (i, j, k) on an N = 2^lg grid (N <= 1024: fits 32 bits)
__device__ __forceinline__ unsigned cidx(int i, int j, int k, int lg) {
  return ((((unsigned)i << lg) + (unsigned)j) << lg) + (unsigned)k;
}

// bounded software grid barrier; false when a wait gave up
__device__ bool gsync(const BArgs& A) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = A.bar_gen;
    const unsigned g0 = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(A.bar_count, 1u);
    if (arrived == gridDim.x - 1) {
      atomicExch(A.bar_count, 0u);
      __threadfence();
      atomicAdd(A.bar_gen, 1u);
    } else {
      long long spins = 0;
      while (*gen == g0) {
        if (++spins > A.max_spins) {
          atomicExch(A.err, 1);
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *(volatile int*)A.err == 0;
}

__device__ __forceinline__ PF batch_pf(const BArgs& A, const BSolve& S) {
  return PF{S.aRt, S.aRt_np1, S.inv_np1, A.cap32};
}

// ---- per-item operations on four cells (mg32_dev.cuh) -----------------------
__device__ __forceinline__ void op_sweep(const BArgs& A, const BSolve& S, int mode, int l,
                                         int colour, unsigned t) {
  const int lg = S.lg - l;
  const size_t half = (size_t)1 << (3 * lg - 1);
  const size_t s = colour * half, o = half - s;
  if (mode == BM_A)
    vec_sweep<MG_NL>(t, S.u32[l] + s, S.u32[l] + o, S.f32[l] + s, nullptr, nullptr, lg, colour,
                     batch_pf(A, S), S.ih2[l], 0.f);
  else
    vec_sweep<MG_LIN>(t, S.e32[l] + s, S.e32[l] + o, S.r32[l] + s, S.u32[l] + s, S.u32[l] + o, lg,
                      colour, batch_pf(A, S), S.ih2[l], 0.f);
}

// restriction from level l to l+1 at four coarse cells
__device__ __forceinline__ void op_restrict(const BArgs& A, const BSolve& S, int mode, int l,
                                            unsigned t) {
  if (mode == BM_A)
    vec_restrict<MG_NL>(t, S.u32[l], S.f32[l], nullptr, S.lg - l, S.u32[l + 1], S.f32[l + 1],
                        S.uold32[l + 1], batch_pf(A, S), S.ih2[l]);
  else
    vec_restrict<MG_LIN>(t, S.e32[l], S.r32[l], S.u32[l], S.lg - l, S.e32[l + 1], S.r32[l + 1],
                         S.u32[l + 1], batch_pf(A, S), S.ih2[l]);
}

// one cell of a colour-split level: the index, the unknown and its neighbours
__device__ __forceinline__ unsigned cell_nbrs(const float* __restrict__ x, unsigned c, int lg,
                                              float* o) {
  const int M = (1 << lg) - 1;
  const int i = (int)(c >> (2 * lg)), j = (int)((c >> lg) & M), k = (int)(c & M);
  unsigned q[6];
  pnb6(i, j, k, lg, q);
#pragma unroll
  for (int e = 0; e < 6; ++e) o[e] = x[q[e]];
  return pdx(i, j, k, lg);
}

// FAS right-hand side of level l (the 4^3 level has no vectors: cell by cell)
__device__ __forceinline__ void op_fas(const BArgs& A, const BSolve& S, int l, unsigned t) {
  const int lg = S.lg - l;
  if (lg > 2) {
    vec_fas(t, S.u32[l], S.f32[l], lg, batch_pf(A, S), S.ih2[l]);
    return;
  }
  for (unsigned c = 4 * t; c < 4 * t + 4; ++c) {
    float n[6];
    const unsigned q = cell_nbrs(S.u32[l], c, lg, n);
    S.f32[l][q] += point_apply<MG_NL>(S.u32[l][q], n, 0.f, n, batch_pf(A, S), S.ih2[l]);
  }
}

// prolongation from level l+1 to the daughters of four of its cells
__device__ __forceinline__ void op_prolong(const BArgs& A, const BSolve& S, int mode, int l,
                                           unsigned t) {
  if (mode == BM_A)
    vec_prolong<MG_NL>(t, S.u32[l], S.u32[l + 1], S.uold32[l + 1], S.lg - l, A.linear);
  else
    vec_prolong<MG_LIN>(t, S.e32[l], S.e32[l + 1], nullptr, S.lg - l, A.linear);
}

// 4^3 coarse level of one solve by one block (64 threads used)
__device__ void op_coarse(const BArgs& A, const BSolve& S, int mode) {
  __shared__ float sh[64], sh2[64];
  const int l = S.nlev - 1;
  const int t = threadIdx.x;
  const bool on = t < 64;
  const int i = (t >> 4) & 3, j = (t >> 2) & 3, k = t & 3, colour = (i + j + k) & 1;
  const int q[6] = {(((i + 3) & 3) << 4) | (j << 2) | k, (((i + 1) & 3) << 4) | (j << 2) | k,
                    (i << 4) | (((j + 3) & 3) << 2) | k, (i << 4) | (((j + 1) & 3) << 2) | k,
                    (i << 4) | (j << 2) | ((k + 3) & 3), (i << 4) | (j << 2) | ((k + 1) & 3)};
  const unsigned g = pdx(i, j, k, 2);
  const PF m = batch_pf(A, S);
  const float ih2 = S.ih2[l];
  float rhs = 0.f, wc = 0.f, wn[6] = {0, 0, 0, 0, 0, 0};
  if (on) {
    sh[t] = mode == BM_A ? S.u32[l][g] : S.e32[l][g];
    sh2[t] = S.u32[l][g];
    rhs = mode == BM_A ? S.f32[l][g] : S.r32[l][g];
  }
  __syncthreads();
  if (on && mode != BM_A) {
    wc = sh2[t];
    for (int d = 0; d < 6; ++d) wn[d] = sh2[q[d]];
  }
  for (int s = 0; s < 40; ++s)
    for (int col = 0; col < 2; ++col) {
      if (on && colour == col) {
        float xn[6];
        for (int d = 0; d < 6; ++d) xn[d] = sh[q[d]];
        sh[t] = mode == BM_A ? point_update<MG_NL, true>(sh[t], xn, 0.f, wn, rhs, m, ih2, 0.f)
                             : point_update<MG_LIN, true>(sh[t], xn, wc, wn, rhs, m, ih2, 0.f);
      }
      __syncthreads();
    }
  if (on) {
    if (mode == BM_A)
      S.u32[l][g] = sh[t];
    else
      S.e32[l][g] = sh[t];
  }
  __syncthreads();
}

// ---- the iterate of the defect correction: u, e^u and f of the finest level,
// in double-float pairs (DF) or FP64, C order -------------------------------
__device__ __forceinline__ dfl* dfp(double* p) { return reinterpret_cast<dfl*>(p); }

// u = v (FP32 or FP64), E = e^u
template <bool DF>
__device__ __forceinline__ void set_u(const BSolve& S, unsigned t, double v) {
  if (DF) {
    const dfl x = df_from_double_bits(v);
    dfp(S.u64)[t] = x;
    dfp(S.E64)[t] = df_exp(x);
  } else {
    S.u64[t] = v;
    S.E64[t] = lean_exp(v);
  }
}

// u += clamp(e), E = e^u
template <bool DF>
__device__ __forceinline__ void add_e(const BArgs& A, const BSolve& S, unsigned t) {
  const int lg = S.lg, M = (1 << lg) - 1;
  const float e = S.e32[0][pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg)];
  const float d = fminf(fmaxf(e, -A.cap32), A.cap32);
  if (DF) {
    const dfl x = df_add_f(dfp(S.u64)[t], d);
    dfp(S.u64)[t] = x;
    dfp(S.E64)[t] = df_exp(x);
  } else {
    const double x = S.u64[t] + d_from_float_bits(d);
    S.u64[t] = x;
    S.E64[t] = lean_exp(x);
  }
}

// residual at finest cell t: writes r32, u32 (= u), e32 = 0; returns r rounded
template <bool DF>
__device__ __forceinline__ float op_resid(const BSolve& S, unsigned t) {
  const int lg = S.lg, M = (1 << lg) - 1;
  const int k = (int)(t & M), j = (int)((t >> lg) & M), i = (int)(t >> (2 * lg));
  const unsigned nb[6] = {cidx((i - 1) & M, j, k, lg), cidx((i + 1) & M, j, k, lg),
                          cidx(i, (j - 1) & M, k, lg), cidx(i, (j + 1) & M, k, lg),
                          cidx(i, j, (k - 1) & M, lg), cidx(i, j, (k + 1) & M, lg)};
  float rf, uf;
  if (DF) {
    const dfl *u = dfp(S.u64), *E = dfp(S.E64);
    const dfl uc = u[t], Ec = E[t];
    dfl acc = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 6; ++q)
      acc = df_add_abs(acc, df_mul(df_add_abs(E[nb[q]], Ec), df_add_abs(u[nb[q]], df_neg(uc))));
    const dfl sN = S.n == 1 ? df_rsqrt(Ec) : df_exp(df_neg(df_mul(uc, S.inv_np1_df)));
    const dfl L = df_add(df_mul(acc, S.ih2h_df), df_mul(S.aRt_df, df_add_f(df_neg(sN), 1.f)));
    rf = df_sub(dfp(S.f64)[t], L).hi;
    uf = uc.hi;
  } else {
    const double uc = S.u64[t], Ec = S.E64[t];
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 6; ++q) s = fma(S.E64[nb[q]] + Ec, S.u64[nb[q]] - uc, s);
    const double sN = S.n == 1 ? lean_rsqrt(Ec) : lean_exp(-uc * S.inv_np1_64);
    rf = f_from_double_bits(S.f64[t] - fma(s, 0.5 * S.ih2_0, S.aRt64 * (1.0 - sN)));
    uf = f_from_double_bits(uc);
  }
  const unsigned p = pdx(i, j, k, lg);
  S.r32[0][p] = rf;
  S.u32[0][p] = uf;
  S.e32[0][p] = 0.f;
  return rf;
}

// a thread's sums over its cells of one solve (FP32 squares summed in FP64
// every few cells) into the solve's state; whole warps, one solve
struct Acc {
  double ss = 0.0, ff = 0.0;
  float s4 = 0.f, mx = 0.f;
  int n = 0;
  __device__ __forceinline__ void add(float r) {
    s4 = fmaf(r, r, s4);
    mx = fmaxf(mx, fabsf(r));
    if ((++n & 3) == 0) flush();
  }
  __device__ __forceinline__ void flush() {
    ss += (double)s4;
    s4 = 0.f;
  }
};
__device__ __forceinline__ void accum(BState* st, Acc& a) {
  a.flush();
  double ss = a.ss, ff = a.ff;
  float mx = a.mx;
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    ff += __shfl_xor_sync(0xffffffffu, ff, o);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (ss != 0.0) atomicAdd(&st->acc_ss, ss);
    if (ff != 0.0) atomicAdd(&st->acc_ff, ff);
    atomicMax(&st->acc_max, (unsigned long long)__double_as_longlong((double)mx));
  }
}

// items of size 2^k over the participant prefix: `shift` = log2(items per
// solve); the solves' modes are read from shared memory (they change only
// where load_modes follows)
#define FOR_ITEMS(A, k, shift, ...)                                                         \
  do {                                                                                     \
    const long long tot_ = (long long)(A).P[k] << (shift);                                 \
    for (long long g_ = blockIdx.x * (long long)blockDim.x + threadIdx.x; g_ < tot_;       \
         g_ += (long long)gridDim.x * blockDim.x) {                                        \
      const int s = (int)(g_ >> (shift));                                                  \
      const unsigned t = (unsigned)(g_ & ((1LL << (shift)) - 1));                          \
      const BSolve& S = (A).S[s];                                                          \
      const int mode = smode[s];                                                           \
      __VA_ARGS__                                                                          \
    }                                                                                      \
  } while (0)

// body(S, mode, t, acc) at the finest-level cells t of the solves whose mode
// `want` accepts (sizes differ: the solves in turn); with `sum`, acc of the warps
// that have cells of the solve goes to its state.  Cell counts and the grid stride are
// multiples of 32, so whole warps reach accum.  (With a reduction and an atomic of every
// warp for every solve 300 solves of 8^3 took 3.75 ms for 2.28, 90 of 16^3 2.27 for 1.82.  A
// warp without cells that leaves before the loop costs 30 solves of 64^3 4%: the compiler
// then orders the loop's loads otherwise.)
template <class Want, class Body>
__device__ __forceinline__ void for_finest(const BArgs& A, const unsigned char* smode, bool sum,
                                           Want want, Body body) {
  unsigned base = 0;
  const unsigned gs = gridDim.x * blockDim.x, g0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int s = 0; s < A.ns; ++s) {
    const BSolve& S = A.S[s];
    const int mode = smode[s];
    const unsigned n = 1u << (3 * S.lg);
    unsigned t = g0 >= base ? g0 - base : g0 + gs - base;
    base = (base + n % gs) % gs;
    const unsigned t0 = t;
    if (!want(mode)) continue;
    Acc acc;
    for (; t < n; t += gs) body(S, mode, t, acc);
    if (sum && __any_sync(0xffffffffu, t != t0)) accum(&A.st[s], acc);
  }
}

// modes of all solves into shared memory (after a barrier that follows a change)
__device__ __forceinline__ void load_modes(const BArgs& A, unsigned char* smode) {
  for (int s = threadIdx.x; s < A.ns; s += blockDim.x)
    smode[s] = (unsigned char)*(volatile const int*)&A.st[s].mode;
  __syncthreads();
}

// DF: the iterate of the defect correction in double-float pairs on the FP32
// pipes (its residual took 43 FP64 instructions per cell); FP64 for tolerances
// that come near the pairs' 48 bits.  Bound by issue slots (55% busy at 32
// warps per SM; 64 registers, a few spilled, against one block of 128 per SM: 45 and
// 50 ms).  96 solves of 32^3..128^3: 157 ms with one cell per thread in C order
// (half of every line unused per half-sweep), FP64 residuals and a warp
// reduction per 32 cells; 42 ms now.
template <bool DF>
__global__ void __launch_bounds__(512, 2) k_batch(BArgs A) {
  __shared__ unsigned char smode[kMaxBatch];
  load_modes(A, smode);
  // ---- set-up: f = src delta, u from the initial guess -----------------------
  auto all = [](int) { return true; };
  for_finest(A, smode, true, all, [&](const BSolve& S, int, unsigned t, Acc& acc) {
    const double f = S.src * S.delta[t];
    const double u0 = S.uinit ? S.uinit[t] : 0.0;
    const int lg = S.lg, M = (1 << lg) - 1;
    const unsigned p = pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg);
    if (DF)
      dfp(S.f64)[t] = df_from_double_bits(f);
    else
      S.f64[t] = f;
    S.f32[0][p] = f_from_double_bits(f);
    S.u32[0][p] = f_from_double_bits(u0);
    set_u<DF>(S, t, u0);
    acc.ff = fma(f, f, acc.ff);
  });
  if (!gsync(A)) return;
  // initial residual
  for_finest(A, smode, true, all, [&](const BSolve& S, int, unsigned t, Acc& acc) {
    acc.add(op_resid<DF>(S, t));
  });
  if (!gsync(A)) return;
  if (blockIdx.x == 0) {
    for (int s = threadIdx.x; s < A.ns; s += blockDim.x) {
      BState& q = A.st[s];
      q.fnorm = sqrt(q.acc_ff);
      q.r0 = sqrt(q.acc_ss);
      q.ref = q.fnorm > 0.0 ? q.fnorm : q.r0;
      q.target = A.tol * q.ref;
      q.r = q.r0;
      q.rmax = __longlong_as_double((long long)q.acc_max);
      q.rprev = -1.0;
      q.mode = q.r0 <= q.target ? BM_DONE : BM_A;
      q.acc_ss = q.acc_ff = 0.0;
      q.acc_max = 0ULL;
    }
  }
  if (!gsync(A)) return;
  load_modes(A, smode);

  for (int cyc = 0; cyc < A.max_cycles; ++cyc) {
    // ---- down ----------------------------------------------------------------
    for (int k = A.maxlg; k >= 3; --k) {
      for (int p = 0; p < A.n_pre; ++p)
        for (int col = 0; col < 2; ++col) {
          FOR_ITEMS(A, k, 3 * k - 3, {
            if (mode != BM_DONE) op_sweep(A, S, mode, S.lg - k, col, t);
          });
          if (!gsync(A)) return;
        }
      FOR_ITEMS(A, k, 3 * k - 5, {
        if (mode != BM_DONE) op_restrict(A, S, mode, S.lg - k, t);
      });
      if (!gsync(A)) return;
      FOR_ITEMS(A, k, 3 * k - 5, {
        if (mode == BM_A) op_fas(A, S, S.lg - k + 1, t);
      });
      if (!gsync(A)) return;
    }
    // ---- coarsest 4^3: one block per solve -------------------------------------
    for (int s = blockIdx.x; s < A.ns; s += gridDim.x)
      if (smode[s] != BM_DONE) op_coarse(A, A.S[s], smode[s]);
    if (!gsync(A)) return;
    // ---- up ------------------------------------------------------------------
    for (int k = 3; k <= A.maxlg; ++k) {
      FOR_ITEMS(A, k, 3 * k - 5, {
        if (mode != BM_DONE) op_prolong(A, S, mode, S.lg - k, t);
      });
      if (!gsync(A)) return;
      for (int p = 0; p < A.n_post; ++p)
        for (int col = 0; col < 2; ++col) {
          FOR_ITEMS(A, k, 3 * k - 3, {
            if (mode != BM_DONE) op_sweep(A, S, mode, S.lg - k, col, t);
          });
          if (!gsync(A)) return;
        }
    }
    // ---- end of cycle: mode B applies the correction ---------------------------
    for_finest(A, smode, false, [](int mode) { return mode == BM_B; },
               [&](const BSolve& S, int, unsigned t, Acc&) { add_e<DF>(A, S, t); });
    if (!gsync(A)) return;
    // residual norms: FP32 for mode A, of the iterate (+ new linear system) for B
    for_finest(A, smode, true, [](int mode) { return mode != BM_DONE; },
               [&](const BSolve& S, int mode, unsigned t, Acc& acc) {
      float r;
      if (mode == BM_B) {
        r = op_resid<DF>(S, t);
      } else {
        float n[6];
        const unsigned q = cell_nbrs(S.u32[0], t, S.lg, n);
        r = S.f32[0][q] - point_apply<MG_NL>(S.u32[0][q], n, 0.f, n, batch_pf(A, S), S.ih2[0]);
      }
      acc.add(r);
    });
    if (!gsync(A)) return;
    // decide
    if (blockIdx.x == 0) {
      for (int s = threadIdx.x; s < A.ns; s += blockDim.x) {
        BState& q = A.st[s];
        const double r = sqrt(q.acc_ss);
        const double rm = __longlong_as_double((long long)q.acc_max);
        q.acc_ss = 0.0;
        q.acc_max = 0ULL;
        // at the limit on the cycles a solve in mode A still goes through the transition,
        // which makes its FP32 iterate the result and forms that one's residual
        if (q.mode == BM_A) {
          q.cyclesA++;
          if (!(r == r) || r <= A.sw * q.ref || (q.rprev > 0.0 && r > 0.7 * q.rprev) ||
              q.cyclesA + q.cyclesB >= A.max_cycles)
            q.mode = BM_TRANS;
          q.rprev = r;
        } else if (q.mode == BM_B) {
          q.cyclesB++;
          const bool rose = !(r < q.r);
          q.r = r;
          q.rmax = rm;
          if (r <= q.target || q.cyclesA + q.cyclesB >= A.max_cycles) {
            q.mode = BM_DONE;
          } else if (rose) {
            q.mode = BM_A;  // back to nonlinear FP32 cycles from u32 = fp32(u)
            q.rprev = -1.0;
          }
        }
      }
    }
    if (!gsync(A)) return;
    load_modes(A, smode);
    // transition A -> B: the iterate from the FP32 one, its residual
    auto trans = [](int mode) { return mode == BM_TRANS; };
    for_finest(A, smode, false, trans, [&](const BSolve& S, int, unsigned t, Acc&) {
      const int lg = S.lg, M = (1 << lg) - 1;
      const float v =
          S.u32[0][pdx((int)(t >> (2 * lg)), (int)((t >> lg) & M), (int)(t & M), lg)];
      set_u<DF>(S, t, d_from_float_bits(v));
    });
    if (!gsync(A)) return;
    for_finest(A, smode, true, trans, [&](const BSolve& S, int, unsigned t, Acc& acc) {
      acc.add(op_resid<DF>(S, t));
    });
    if (!gsync(A)) return;
    int active = 0;
    if (blockIdx.x == 0) {
      __shared__ int cnt;
      if (threadIdx.x == 0) cnt = 0;
      __syncthreads();
      for (int s = threadIdx.x; s < A.ns; s += blockDim.x) {
        BState& q = A.st[s];
        if (q.mode == BM_TRANS) {
          const double r = sqrt(q.acc_ss);
          q.r = r;
          q.rmax = __longlong_as_double((long long)q.acc_max);
          q.mode = r <= q.target || q.cyclesA + q.cyclesB >= A.max_cycles ? BM_DONE : BM_B;
          q.acc_ss = 0.0;
          q.acc_max = 0ULL;
        }
        if (q.mode != BM_DONE) atomicAdd(&cnt, 1);
      }
      __syncthreads();
      active = cnt;
      if (threadIdx.x == 0) atomicExch(A.err + 1, active);
    }
    if (!gsync(A)) return;
    load_modes(A, smode);
    if (*(volatile int*)(A.err + 1) == 0) break;
  }
  // ---- outputs: fR = fbar e^u and the force -----------------------------------
  auto val = [](const double* p, unsigned q) {
    return DF ? df_to_double_bits(reinterpret_cast<const dfl*>(p)[q]) : p[q];
  };
  for_finest(A, smode, false, all, [&](const BSolve& S, int, unsigned t, Acc&) {
    const int lg = S.lg, M = (1 << lg) - 1;
    const size_t n = (size_t)1 << (3 * lg);
    const int kk = (int)(t & M), jj = (int)((t >> lg) & M), ii = (int)(t >> (2 * lg));
    const double* E = S.E64;
    S.fr_out[t] = S.fbar * val(E, t);
    if (S.u_out) S.u_out[t] = val(S.u64, t);
    if (S.acc_out) {
      S.acc_out[t] = S.gscale * (val(E, cidx((ii + 1) & M, jj, kk, lg)) -
                                 val(E, cidx((ii - 1) & M, jj, kk, lg)));
      S.acc_out[n + t] = S.gscale * (val(E, cidx(ii, (jj + 1) & M, kk, lg)) -
                                     val(E, cidx(ii, (jj - 1) & M, kk, lg)));
      S.acc_out[2 * n + t] = S.gscale * (val(E, cidx(ii, jj, (kk + 1) & M, lg)) -
                                         val(E, cidx(ii, jj, (kk - 1) & M, lg)));
    }
  });
}

}  // namespace

// ============================================================================
// host side
// ============================================================================
struct BatchWork {
  std::string sig;
  std::vector<void*> bufs;
  BSolve* dS = nullptr;
  BState* dst = nullptr;
  unsigned* bar = nullptr;  // [0] count, [1] generation
  int* err = nullptr;
  std::vector<int> order;
  std::map<std::string, BatchShape> tuned;  // by the sizes
  cudaGraphExec_t gx = nullptr;
  std::string gkey;
  // learned start: network input staging and the predicted initial guesses
  double *lrn_in = nullptr, *lrn_out = nullptr;
  long long lrn_in_cap = 0, lrn_out_cap = 0;
};

static void batch_release(BatchWork* B) {
  for (void* p : B->bufs) cudaFree(p);
  B->bufs.clear();
  if (B->dS) cudaFree(B->dS);
  if (B->dst) cudaFree(B->dst);
  if (B->bar) cudaFree(B->bar);
  if (B->err) cudaFree(B->err);
  B->dS = nullptr;
  B->dst = nullptr;
  B->bar = nullptr;
  B->err = nullptr;
  if (B->gx) cudaGraphExecDestroy(B->gx);
  B->gx = nullptr;
  B->gkey.clear();
  if (B->lrn_in) cudaFree(B->lrn_in);
  if (B->lrn_out) cudaFree(B->lrn_out);
  B->lrn_in = B->lrn_out = nullptr;
  B->lrn_in_cap = B->lrn_out_cap = 0;
}

// Learned start of the batch items of N >= 32 without an initial guess: their
// density contrasts are staged in groups of one size (at most kLearnVox cells
// per network pass) and the predictions kept in lrn_out for the solve.
constexpr long long kLearnVox = 1LL << 22;

static mgfr_status batch_learned_start(mgfr_ctx* c, BatchWork* B, const mgfr_batch_item* items,
                                       const std::vector<int>& order, std::vector<BSolve>& hs) {
  long long total = 0;
  const int ns = (int)order.size();
  for (int q = 0; q < ns; ++q)
    if (hs[q].N >= 32 && !items[order[q]].u_init_dev) total += 1LL << (3 * hs[q].lg);
  if (total == 0) return MGFR_OK;
  if (B->lrn_out_cap < total) {
    if (B->lrn_out) cudaFree(B->lrn_out);
    B->lrn_out = nullptr;
    B->lrn_out_cap = 0;
    MG_CK(c, dev_malloc(c, &B->lrn_out, sizeof(double) * (size_t)total));
    B->lrn_out_cap = total;
  }
  long long off = 0;
  int q = 0;
  while (q < ns) {
    // a run of solves of one size (order is sorted by size)
    if (hs[q].N < 32 || items[order[q]].u_init_dev) {
      ++q;
      continue;
    }
    const int N = hs[q].N;
    const long long per = 1LL << (3 * hs[q].lg);
    std::vector<int> grp;
    std::vector<double> fr0;
    while (q < ns && hs[q].N == N && (long long)(grp.size() + 1) * per <= std::max(per, kLearnVox)) {
      if (!items[order[q]].u_init_dev) {
        grp.push_back(q);
        fr0.push_back(items[order[q]].fr0_abs);
      }
      ++q;
    }
    if (grp.empty()) continue;
    const long long need = per * (long long)grp.size();
    if (B->lrn_in_cap < need) {
      if (B->lrn_in) cudaFree(B->lrn_in);
      B->lrn_in = nullptr;
      B->lrn_in_cap = 0;
      MG_CK(c, dev_malloc(c, &B->lrn_in, sizeof(double) * (size_t)need));
      B->lrn_in_cap = need;
    }
    for (size_t k = 0; k < grp.size(); ++k)
      MG_CK(c, cudaMemcpyAsync(B->lrn_in + k * per, items[order[grp[k]]].delta_dev,
                               sizeof(double) * (size_t)per, cudaMemcpyDeviceToDevice, c->s));
    mgfr_status rs = unet_predict_batch(c, (int)grp.size(), N, B->lrn_in, 1.0, fr0.data(),
                                        B->lrn_out + off);
    if (rs != MGFR_OK) return rs;
    for (size_t k = 0; k < grp.size(); ++k) hs[grp[k]].uinit = B->lrn_out + off + k * per;
    off += need;
  }
  return MGFR_OK;
}

void batch_free(mgfr_ctx* c) {
  BatchWork* B = (BatchWork*)c->batch;
  if (!B) return;
  batch_release(B);
  delete B;
  c->batch = nullptr;
}

// work items of a half-sweep of the finest grids
static long long batch_vecs(int nsolves, const mgfr_batch_item* items) {
  long long v = 0;
  for (int i = 0; i < nsolves; ++i) v += (long long)items[i].N * items[i].N * items[i].N / 8;
  return v;
}

// at most `blocks` blocks
static mgfr_status launch_batch(mgfr_ctx* c, BatchWork* B, const BArgs& A, BatchShape shape,
                                long long blocks, bool use_graph) {
  const int threads = shape.threads;
  int dev = c->device, nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int occ = 0;
  // double-float carries the residual to about 1e-13 of its terms; tolerances
  // below 1e-10 keep FP64
  void* kern = A.tol >= 1e-10 ? (void*)k_batch<true> : (void*)k_batch<false>;
  MG_CK(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, 0));
  if (occ < 1) return set_err(c, MGFR_E_UNSUPPORTED, "batched kernel cannot be resident");
  const int grid = (int)std::min((long long)nsm * std::min(shape.per_sm, occ), blocks);
  MG_CK(c, cudaMemsetAsync(B->bar, 0, 2 * sizeof(unsigned), c->s));
  MG_CK(c, cudaMemsetAsync(B->err, 0, 2 * sizeof(int), c->s));
  BArgs a = A;
  void* args[] = {&a};
  if (!use_graph) {
    MG_CK(c, cudaLaunchCooperativeKernel(kern, grid, threads, args, 0, c->s));
    c->launches += 1;
    return MGFR_OK;
  }
  // the launch and its settings; the sizes are the workspace's (batch_release drops the
  // graph with it)
  char key[512];
  std::snprintf(key, sizeof(key), "%d|%d|%d|%d|%d|%d|%.17g|%.17g|%.17g|%lld", threads, grid,
                A.n_pre, A.n_post, A.linear, A.max_cycles, (double)A.cap32, A.tol, A.sw,
                A.max_spins);
  if (!B->gx || B->gkey != key) {
    if (B->gx) cudaGraphExecDestroy(B->gx);
    B->gx = nullptr;
    cudaGraph_t g = nullptr;
    MG_CK(c, cudaStreamBeginCapture(c->s, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaLaunchCooperativeKernel(kern, grid, threads, args, 0, c->s);
    cudaError_t e2 = cudaStreamEndCapture(c->s, &g);
    if (e != cudaSuccess || e2 != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      (void)cudaGetLastError();
      // capture of a cooperative launch unsupported: launch directly
      MG_CK(c, cudaLaunchCooperativeKernel(kern, grid, threads, args, 0, c->s));
      c->launches += 1;
      return MGFR_OK;
    }
    e = cudaGraphInstantiate(&B->gx, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return set_err(c, MGFR_E_CUDA, "batched graph instantiate failed");
    B->gkey = key;
  }
  MG_CK(c, cudaGraphLaunch(B->gx, c->s));
  c->launches += 1;
  return MGFR_OK;
}

static mgfr_status check_items(mgfr_ctx* c, int nsolves, const mgfr_batch_item* items) {
  if (nsolves < 1 || nsolves > kMaxBatch || !items)
    return set_err(c, MGFR_E_INVALID, "need 1..4096 batch items");
  const mgfr_config& g = c->cfg;
  for (int i = 0; i < nsolves; ++i) {
    const mgfr_batch_item& it = items[i];
    if (it.N < 8 || it.N > 512 || (it.N & (it.N - 1)))
      return set_err(c, MGFR_E_INVALID, "batch item N must be a power of two in [8, 512]");
    if (!(it.box > 0.0) || !(it.a > 0.0) || !(it.fr0_abs > 0.0) || it.n < 1 || !it.delta_dev ||
        !it.fr_out_dev)
      return set_err(c, MGFR_E_INVALID, "invalid batch item");
    if (g.start == MGFR_START_USER && !it.u_init_dev)
      return set_err(c, MGFR_E_INVALID, "start = user needs u_init_dev on every batch item");
    if (g.start == MGFR_START_PREVIOUS || g.start == MGFR_START_PREVIOUS_ALL)
      return set_err(c, MGFR_E_INVALID, "start = previous is not available for batches");
  }
  return MGFR_OK;
}

// The sizes in descending order; order (if not NULL): the items so sorted, where the
// participants of a size form a prefix
static std::string batch_signature(int nsolves, const mgfr_batch_item* items,
                                   std::vector<int>* order) {
  std::vector<int> o(nsolves);
  for (int i = 0; i < nsolves; ++i) o[i] = i;
  std::stable_sort(o.begin(), o.end(), [&](int x, int y) { return items[x].N > items[y].N; });
  std::string sig;
  for (int i : o) sig += std::to_string(items[i].N) + ",";
  if (order) *order = o;
  return sig;
}

extern "C" {

mgfr_status mgfr_batch_solve(mgfr_ctx* c, int nsolves, const mgfr_batch_item* items,
                             mgfr_stats* per_solve) {
  if (!c) return MGFR_E_INVALID;
  const mgfr_status args = check_items(c, nsolves, items);
  if (args != MGFR_OK) return args;
  const mgfr_config& g = c->cfg;
  auto w0 = std::chrono::steady_clock::now();
  MG_CK(c, cudaSetDevice(c->device));
  c->launches = 0;
  if (!c->batch) c->batch = new BatchWork();
  BatchWork* B = (BatchWork*)c->batch;
  std::vector<int> order;
  const std::string sig = batch_signature(nsolves, items, &order);
  if (sig != B->sig) {
    batch_release(B);
    B->sig = sig;
  }
  std::vector<BSolve> hs(nsolves);
  int maxlg = 0;
  size_t bi = 0;
  auto buf = [&](size_t bytes) -> void* {
    if (bi < B->bufs.size()) return B->bufs[bi++];
    void* p = nullptr;
    if (dev_malloc(c, &p, bytes) != cudaSuccess) {
      (void)cudaGetLastError();
      return nullptr;
    }
    B->bufs.push_back(p);
    ++bi;
    return p;
  };
  for (int q = 0; q < nsolves; ++q) {
    const mgfr_batch_item& it = items[order[q]];
    BSolve& S = hs[q];
    std::memset(&S, 0, sizeof(S));
    S.N = it.N;
    int lg = 0;
    while ((1 << lg) < it.N) ++lg;
    S.lg = lg;
    S.nlev = lg - 1;
    maxlg = std::max(maxlg, lg);
    mgfr_config cf = g;
    cf.fr0_abs = it.fr0_abs;
    cf.n = it.n;
    const Model m = make_model(cf, it.a);
    S.h0 = it.box / it.N;
    S.ih2_0 = 1.0 / (S.h0 * S.h0);
    for (int l = 0; l < S.nlev; ++l) {
      const double h = it.box / (it.N >> l);
      S.ih2[l] = (float)(1.0 / (h * h));
      const size_t n = (size_t)1 << (3 * (lg - l));
      S.u32[l] = (float*)buf(4 * n);
      S.f32[l] = (float*)buf(4 * n);
      S.e32[l] = (float*)buf(4 * n);
      S.r32[l] = (float*)buf(4 * n);
      if (l > 0) S.uold32[l] = (float*)buf(4 * n);
      if (!S.u32[l] || !S.f32[l] || !S.e32[l] || !S.r32[l] || (l > 0 && !S.uold32[l]))
        return set_err(c, MGFR_E_OOM, "batch workspace allocation failed");
    }
    const size_t n0 = (size_t)1 << (3 * lg);
    S.u64 = (double*)buf(8 * n0);
    S.E64 = (double*)buf(8 * n0);
    S.f64 = (double*)buf(8 * n0);
    if (!S.u64 || !S.E64 || !S.f64) return set_err(c, MGFR_E_OOM, "batch workspace allocation failed");
    S.aRt = (float)m.aRt;
    S.aRt_np1 = (float)m.aRt_np1;
    S.inv_np1 = (float)m.inv_np1;
    S.aRt64 = m.aRt;
    S.aRt_df = df_from_double(m.aRt);
    S.inv_np1_df = df_from_double(m.inv_np1);
    S.ih2h_df = df_from_double(0.5 * S.ih2_0);
    S.inv_np1_64 = m.inv_np1;
    S.src = m.src;
    S.fbar = m.fbar;
    S.gscale = m.fbar / (2.0 * S.h0) / (2.0 * m.a);
    S.n = m.n;
    S.delta = it.delta_dev;
    S.uinit = it.u_init_dev;
    S.fr_out = it.fr_out_dev;
    S.acc_out = it.acc_out_dev;
    S.u_out = it.u_out_dev;
  }
  if (!B->dS) MG_CK(c, dev_malloc(c, &B->dS, sizeof(BSolve) * nsolves));
  if (!B->dst) MG_CK(c, dev_malloc(c, &B->dst, sizeof(BState) * nsolves));
  if (!B->bar) MG_CK(c, dev_malloc(c, &B->bar, 2 * sizeof(unsigned)));
  if (!B->err) MG_CK(c, dev_malloc(c, &B->err, 2 * sizeof(int)));
  MG_CK(c, cudaEventRecord(c->ev_in, c->user));
  MG_CK(c, cudaStreamWaitEvent(c->s, c->ev_in, 0));
  if (g.start == MGFR_START_LEARNED) {
    mgfr_status ls = batch_learned_start(c, B, items, order, hs);
    if (ls != MGFR_OK) return ls;
  }
  MG_CK(c, cudaMemcpyAsync(B->dS, hs.data(), sizeof(BSolve) * nsolves, cudaMemcpyHostToDevice, c->s));
  MG_CK(c, cudaMemsetAsync(B->dst, 0, sizeof(BState) * nsolves, c->s));
  BArgs A{};
  A.S = B->dS;
  A.st = B->dst;
  A.ns = nsolves;
  A.maxlg = maxlg;
  for (int k = 0; k < 16; ++k) {
    int p = 0;
    for (int q = 0; q < nsolves; ++q) p += hs[q].lg >= k;
    A.P[k] = p;
  }
  A.n_pre = g.n_pre;
  A.n_post = g.n_post;
  A.linear = g.prolong_linear;
  A.max_cycles = g.max_vcycles;
  A.cap32 = (float)g.step_cap;
  A.tol = g.tol_rel;
  A.sw = g.mixed_switch;
  A.bar_count = B->bar;
  A.bar_gen = B->bar + 1;
  A.err = B->err;
  A.max_spins = g.max_spins;
  // the tuned launch shape for these sizes, else by the amount of work (batch_shape.h)
  const long long vecs = batch_vecs(nsolves, items);
  int nsm = 0;
  MG_CK(c, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  BatchShape shape = batch_rule(vecs, nsolves, nsm);
  auto itc = B->tuned.find(sig);
  if (itc != B->tuned.end()) shape = itc->second;
  MG_CK(c, cudaEventRecord(c->t0, c->s));
  mgfr_status rs = launch_batch(c, B, A, shape, batch_blocks(shape.threads, vecs, nsolves), true);
  if (rs != MGFR_OK) return rs;
  MG_CK(c, cudaEventRecord(c->t1, c->s));
  std::vector<BState> st(nsolves);
  int err = 0;
  MG_CK(c, cudaMemcpyAsync(st.data(), B->dst, sizeof(BState) * nsolves, cudaMemcpyDeviceToHost, c->s));
  MG_CK(c, cudaMemcpyAsync(&err, B->err, sizeof(int), cudaMemcpyDeviceToHost, c->s));
  MG_CK(c, cudaEventRecord(c->ev_out, c->s));
  MG_CK(c, cudaStreamWaitEvent(c->user, c->ev_out, 0));
  MG_CK(c, cudaStreamSynchronize(c->s));
  MG_CK(c, cudaGetLastError());
  float ms = 0.f;
  cudaEventElapsedTime(&ms, c->t0, c->t1);
  const double wall =
      std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - w0).count();
  bool allok = true;
  for (int q = 0; q < nsolves; ++q) {
    const BState& b = st[q];
    const bool ok = b.r <= b.target;
    allok = allok && ok;
    if (per_solve) {
      mgfr_stats& o = per_solve[order[q]];
      std::memset(&o, 0, sizeof(o));
      o.vcycles = b.cyclesA;
      o.outer_iters = b.cyclesB;
      o.res_l2_init = b.r0;
      o.res_l2_final = b.r;
      o.res_max_final = b.rmax;
      o.f_l2 = b.fnorm;
      o.t_solve_ms = ms;
      o.t_total_ms = wall;
      o.n_levels = 1;
      o.cells_per_level[0] = 1LL << (3 * hs[q].lg);
      o.gpu_launches = c->launches;
      long long cells = 0;
      for (int l = 0; l < hs[q].nlev; ++l) cells += 1LL << (3 * (hs[q].lg - l));
      o.cell_updates = (long long)b.cyclesA * (g.n_pre + g.n_post) * cells;
      o.linear_updates = (long long)b.cyclesB * (g.n_pre + g.n_post) * cells;
    }
  }
  if (err) return set_err(c, MGFR_E_TIMEOUT, "a grid barrier wait in the batched kernel gave up");
  if (!allok) return set_err(c, MGFR_E_NOCONVERGE, "a batched solve missed its tolerance");
  return MGFR_OK;
}

// Time every candidate launch shape on this batch (its second run: the first
// captures the launch between the events) and keep the fastest for batches of the same
// size signature (persisted in the file named by MGFR_TUNE_CACHE when set).
mgfr_status mgfr_batch_autotune(mgfr_ctx* c, int nsolves, const mgfr_batch_item* items,
                                int* best_threads, int* best_blocks_per_sm) {
  if (!c) return MGFR_E_INVALID;
  const mgfr_status args = check_items(c, nsolves, items);
  if (args != MGFR_OK) return args;
  if (!c->batch) c->batch = new BatchWork();
  BatchWork* B = (BatchWork*)c->batch;
  const std::string sig = batch_signature(nsolves, items, nullptr);
  const long long vecs = batch_vecs(nsolves, items);
  int nsm = 0;
  MG_CK(c, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  BatchShape cand[10], best{};
  const int n = batch_candidates(vecs, nsolves, nsm, cand);
  float best_ms = 1e30f;
  for (int i = 0; i < n; ++i) {
    B->tuned[sig] = cand[i];
    float ms = 0.f;
    for (int rep = 0; rep < 2; ++rep) {
      const mgfr_status rs = mgfr_batch_solve(c, nsolves, items, nullptr);
      if (rs != MGFR_OK && rs != MGFR_E_NOCONVERGE) {
        B->tuned.erase(sig);
        return rs;
      }
    }
    cudaEventElapsedTime(&ms, c->t0, c->t1);
    if (ms < best_ms) {
      best_ms = ms;
      best = cand[i];
    }
  }
  B->tuned[sig] = best;
  if (const char* path = std::getenv("MGFR_TUNE_CACHE")) {
    if (FILE* f = std::fopen(path, "a")) {
      std::fprintf(f, "%s %d %d %.4f\n", sig.c_str(), best.threads, best.per_sm, best_ms);
      std::fclose(f);
    }
  }
  if (best_threads) *best_threads = best.threads;
  if (best_blocks_per_sm) *best_blocks_per_sm = best.per_sm;
  return MGFR_OK;
}

}  // extern "C"

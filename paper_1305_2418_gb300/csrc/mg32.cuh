// mg32.cuh -- FP32 multigrid V-cycles on dense periodic levels (mg32.cu), the
// smoother and coarse-grid part of every dense solve:
//   MG_NL : L(x) = r, the nonlinear operator of Sec. 3.2 (mixed form, phase A);
//           w = the restricted iterate of a coarse level (FAS, Eqs. (27), (29));
//   MG_LIN: J(w) x = r, J the Jacobian of L at w (mixed form, phase B);
//   MG_DEV: L(w + x) - L(w) = r, the nonlinear operator in the deviation x
//           from a fixed iterate w: r is the residual of the FP64 iterate,
//           and the cycle forms the FP64 V-cycle's correction to FP32 relative
//           accuracy (FP64 form);
//   MG_POI: lap x = r (particle-mesh potential).
// All arrays are stored by red-black colour (colour_split.cuh).
#pragma once
#include "mgfr_internal.cuh"

enum Mg32Op { MG_NL = 0, MG_LIN = 1, MG_DEV = 2, MG_POI = 3 };

struct Mg32Level {
  int lg;          // N = 2^lg, 2 <= lg <= 10
  float ih2, h2;   // 1 / h^2, h^2
  float *x, *r, *w;
};

struct Mg32Par {
  float aRt, aRt_np1, inv_np1, cap;
  int n_pre, n_post, linear;
  int coarse_sweeps;   // most sweeps on the 4^3 grid
  float coarse_rel;    // > 0: stop them when max|r| has dropped by this factor
};

struct Mg32Hook {      // called around every half-sweep of the finest level
  void (*begin)(void*) = nullptr;
  void (*end)(void*) = nullptr;
  void* arg = nullptr;
};

// One V-cycle over levels L[0] (finest) .. L[nlev - 1] (4^3); returns the
// half-sweep pairs' cell updates (the 4^3 grid not counted).
long long mg32_cycle(Mg32Op op, const Mg32Level* L, int nlev, const Mg32Par& p, cudaStream_t s,
                     const Mg32Hook* hook = nullptr);
// Norm of the residual of op's equation, MG_NL or MG_DEV (sum, max |.|), into out[0..1]
// (device), per-block partial sums in `partials` (2 nparts doubles).
void mg32_norm(Mg32Op op, const Mg32Level& L, const Mg32Par& p, double* partials, int nparts, double* out,
               cudaStream_t s);
// raise the cluster kernels' launch limits once per device (before a capture)
mgfr_status mg32_prepare(mgfr_ctx* c);

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

// Pairs of cycles.  What follows a cycle at the accuracy of the iterate costs a good part of
// it (FP64 form: the update of u and e^u and the residual, 190 of 430 us on 128^3, FP64
// arithmetic being 2 FMA per SM and clock; Poisson: 130 of 400 on 256^3).  Two FP32 cycles
// that certainly both stay above the target share it: the first one's norm is formed from
// the correction in FP32, and the second goes on from the same correction.  They are the
// same cycles but for the FP32 rounding of the first correction where the second one's is
// added to it; that rounding's residual, on grid-scale waves 12 2^-24 (N / 2 pi)^2 of the
// first one's, stays below 1.5e-3 up to kPairMax, against the 1e-2 that two cycles leave,
// and the cycle that follows takes it out.  FP64 form: 128^3 3.43 -> 3.00 ms, 256^3 18.1 ->
// 14.1; below kPairMin the norm and its read-back cost what they save (32^3 0.61 -> 0.65
// ms, 64^3 1.04 -> 1.06).
constexpr int kPairMin = 128, kPairMax = 256;
// whether to try a pair at residual norm r, rho the last cycle's reduction (0: none yet),
// and whether to go on after its first cycle left r1: both above the target
inline bool pair_start(double r, double rho, double target) {
  return r * (rho > 0.0 ? rho * rho : 1e-3) > 2.0 * target;
}
inline bool pair_on(double r, double r1, double target) {
  return r1 < r && r1 * (r1 / r) > 2.0 * target;
}

// One V-cycle over levels L[0] (finest) .. L[nlev - 1] (4^3); returns the
// half-sweep pairs' cell updates (the 4^3 grid not counted).
long long mg32_cycle(Mg32Op op, const Mg32Level* L, int nlev, const Mg32Par& p, cudaStream_t s,
                     const Mg32Hook* hook = nullptr);
// Norm of the residual of op's equation (not MG_LIN; sum of squares, max |.|), into out[0..1]
// (device), per-block partial sums in `partials` (2 nparts doubles).
void mg32_norm(Mg32Op op, const Mg32Level& L, const Mg32Par& p, double* partials, int nparts, double* out,
               cudaStream_t s);
// raise the cluster kernels' launch limits once per device (before a capture)
mgfr_status mg32_prepare(mgfr_ctx* c);

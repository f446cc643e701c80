// nn_tc.cu -- the network's 3^3 convolutions (forward, input gradient and
// weight gradient) on the fifth-generation tensor cores: tcgen05.mma with the
// FP32 accumulator in tensor memory (TMEM), BF16 operands in shared memory.
// Three forms: the per-tap kernel (k_conv_tc, below), the halo-tiled kernels
// of the full- and second-resolution layers (k_conv_halo, k_conv_halo_s: the
// input block with its one-voxel halo staged once per tile, each tap a shifted
// descriptor into it) and the weight gradient (k_wgrad_tc per tap; k_wgrad_halo from
// resident blocks for up to 32 output channels).
//
// Implicit GEMM per CTA: rows = an M tile of 128 consecutive
// voxels, columns = all N output channels (N <= 256), reduction = 27 taps x
// the K input channels.  Per tap:
//   A (128 x K): each row the channel vector of the row voxel's neighbour at
//     the tap offset (periodic), copied by cp.async in 16-byte chunks;
//   B (N x K): the tap's weight slice, packed in advance in the shared-memory
//     layout and brought in by one bulk asynchronous copy (cp.async.bulk,
//     completion counted on an mbarrier).
// Both tiles use the canonical K-major layout without swizzle: core matrices
// of 8 rows x 16 bytes; for each 8-channel chunk the rows are contiguous (so
// the 8-row groups are 128 B apart: SBO), and the chunks follow each other one
// tile-height apart (LBO).  An elected lane issues the tap's MMAs (K = 16 each) and
// commits them to the stage's mbarrier; two stages overlap the copies of tap
// t+1 with the MMAs of tap t.  The epilogue reads the accumulator with
// tcgen05.ld (warp w its 32 TMEM lanes = rows 32w..32w+31).
//
// Forward: y[m][co] = sum_{tap,ci} x[m + d_tap][ci] W[tap][ci][co] (+bias,
// ReLU), stored BF16.  Input gradient: gx[m][ci] = sum_{tap,co}
// g[m - d_tap][co] W[tap][ci][co], stored (or added) FP32.
//
// Weight gradient (k_wgrad_tc): dW[t][ci][co] = sum_v x[v][ci] g[v - d_t][co]
// as the transposed GEMM rows = (tap, co) (128 / Cout taps per CTA), columns
// = ci, reduction = voxels.  Both operands are then contiguous along their
// row index in the NDHWC tensors (the channels), so they are staged in the
// MN-major canonical layout (core matrices of 8 voxels x 16 bytes of
// channels) by 16-byte cp.async copies, without a transpose.  The voxels are
// split over CTAs; each CTA writes its partial dW, reduced in a fixed order.
//
// Every wait on an mbarrier is bounded; a wait that runs out sets *err and the
// CTA leaves through the normal exit (TMEM freed).
#include <algorithm>
#include <cstdint>

#include "device_once.h"
#include "nn_kernels.cuh"

namespace {

// opt in to 227 KB of shared memory per CTA, once per device and kernel; a launch on a
// device that refused fails, and its caller reads the error
template <class K>
void smem_opt_in(DeviceOnce& once, K kernel) {
  int dev = -1;
  cudaGetDevice(&dev);
  once(dev, [&] {
    return (int)cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     227 * 1024);
  });
}

constexpr int TC_THREADS = 128;
constexpr int TC_M = 128;
constexpr long long kSpin = 1LL << 22;  // try_wait rounds before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for the completion of the phase with this parity
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err) {
  for (long long i = 0; i < kSpin; ++i)
    if (mbar_try(bar, parity)) return true;
  atomicExch(err, 1);
  return false;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
  const int n = valid ? 16 : 0;  // 0: fill with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// one bulk copy global -> shared, its bytes counted on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// canonical K-major shared-memory descriptor, no swizzle (version 1)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor: BF16 x BF16 -> FP32, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// MN-major operands without swizzle: the field at bits 32-45 (SBO) holds the
// stride between core matrices along M (or N), the field at bits 16-29 (LBO)
// the stride between core matrices along K
__device__ __forceinline__ uint64_t sdesc_mn(uint32_t saddr, uint32_t mn_stride,
                                             uint32_t k_stride) {
  return sdesc(saddr, k_stride, mn_stride);
}

// instruction descriptor: BF16 x BF16 -> FP32, A and B MN-major (bits 15, 16)
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N) {
  return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

// The MMA loops run in one whole warp, warp-uniform, and only the elected lane
// issues: descriptors then stay in uniform registers (issued from inside an
// `if (tid == 0)` each MMA cost about 100 clocks of moves and 64-bit shifts, more
// than its work).
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ int warp_index() {
  return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
}
// a descriptor advanced by `bytes` (a multiple of 16, inside shared memory: the
// address field does not overflow into its neighbour)
__device__ __forceinline__ uint64_t desc_add(uint64_t d, uint32_t bytes) {
  return d + (uint64_t)(bytes >> 4);
}

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// 16 columns of the warp's 32 lanes set to zero
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
      "r"(0)
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// neighbour voxel of m at offset (dx,dy,dz), periodic in each sample (a tensor
// of 2^32 voxels of 16 BF16 channels would fill 137 GB: 32-bit indices suffice)
__device__ __forceinline__ unsigned tc_nbr(unsigned m, int lgD, int dx, int dy, int dz) {
  const unsigned M = (1u << lgD) - 1;
  const unsigned i = (m >> (2 * lgD)) & M, j = (m >> lgD) & M, k = m & M;
  const unsigned b = m >> lgD >> lgD >> lgD;  // 3 lgD may reach 32
  return (((((b << lgD) + ((i + dx) & M)) << lgD) + ((j + dy) & M)) << lgD) + ((k + dz) & M);
}

// threads of a convolution CTA: two warps per scheduler, because staging the
// operands is a chain of address arithmetic and copies per 16-byte chunk (with
// four warps the 96 -> 32 halo kernel spent 20 of 27 us per CTA there)
constexpr int HT = 256;
// stride between the 8-channel chunks of an A tile: the 128 rows and 16 bytes,
// so that the chunks of a row, which neighbouring threads write, fall into
// different banks
constexpr uint32_t kALbo = TC_M * 16 + 16;
constexpr int a_bytes(int kc) { return (kc / 8) * (int)kALbo; }

// 16 accumulators of voxel m, columns n0..n0+15, to the output: BF16 with bias
// and ReLU (forward), or FP32 (input gradient)
template <bool DGRAD>
__device__ __forceinline__ void store16(const float* v, long long m, int n0,
                                        const float* __restrict__ bias, int relu,
                                        __nv_bfloat16* __restrict__ y, int ldy, int offy,
                                        float* __restrict__ gx, int ldg, int offg,
                                        int accumulate) {
  if (!DGRAD) {
    __align__(16) __nv_bfloat16 o[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float a = v[i] + (bias ? bias[n0 + i] : 0.f);
      if (relu) a = fmaxf(a, 0.f);
      o[i] = __float2bfloat16(a);
    }
    uint4* dst = reinterpret_cast<uint4*>(y + m * ldy + offy + n0);
    dst[0] = reinterpret_cast<const uint4*>(o)[0];
    dst[1] = reinterpret_cast<const uint4*>(o)[1];
  } else {
    float4* q = reinterpret_cast<float4*>(gx + m * ldg + offg + n0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float4 a = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      if (accumulate) {
        const float4 p = q[i];
        a = make_float4(p.x + a.x, p.y + a.y, p.z + a.z, p.w + a.w);
      }
      q[i] = a;
    }
  }
}

// KC: channels of an A row (the reduction per tap); NC: output columns.
// DGRAD: the input-gradient form (mirrored tap, FP32 output, optional add).
template <int KC, int NC, bool DGRAD>
__global__ void __launch_bounds__(HT) k_conv_tc(
    const __nv_bfloat16* __restrict__ x, int ldx, int offx, const __nv_bfloat16* __restrict__ Wp,
    const float* __restrict__ bias, int relu, __nv_bfloat16* __restrict__ y, int ldy, int offy,
    float* __restrict__ gx, int ldg, int offg, int accumulate, int lgD, long long Mtot,
    int tmem_cols, int* __restrict__ err) {
  constexpr uint32_t A_LBO = kALbo, B_LBO = NC * 16, SBO = 128;
  constexpr int A_BYTES = a_bytes(KC), B_BYTES = NC * KC * 2;
  constexpr uint32_t IDESC = idesc_bf16(TC_M, NC);
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* As = smem;                        // [2][A_BYTES]
  unsigned char* Bs = smem + 2 * A_BYTES;          // [2][B_BYTES]
  uint64_t* bars = reinterpret_cast<uint64_t*>(Bs + 2 * B_BYTES);  // full[2], done[2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 4);
  const int tid = threadIdx.x, warp = warp_index();
  const long long m0 = (long long)blockIdx.x * TC_M;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < 4; ++q) mbar_init(bars + q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = *tslot;
  bool ok = true;

  // A copies of tap t into stage s (every thread a share of the 16-byte chunks)
  auto load_a = [&](int t, int s) {
    const int dx = t / 9 - 1, dy = (t / 3) % 3 - 1, dz = t % 3 - 1;
    const int sg = DGRAD ? -1 : 1;
    unsigned char* A = As + s * A_BYTES;
    constexpr int CH = KC / 8;  // 16-byte chunks per row
    // consecutive threads take the chunks of a row (contiguous in memory)
#pragma unroll 4
    for (int e = tid; e < TC_M * CH; e += HT) {
      const int r = e / CH, c = e - r * CH;
      const long long m = m0 + r;
      const bool v = m < Mtot;
      const unsigned src = v ? tc_nbr((unsigned)m, lgD, sg * dx, sg * dy, sg * dz) : 0u;
      cp_async16(A + c * A_LBO + r * 16, x + (size_t)src * ldx + offx + 8 * c, v);
    }
    cp_async_commit();
  };

  // thread 0's account of what is in flight: bulk copies issued per stage
  // (their completions are waited in order) and the stage of the last commit
  int issued[2] = {0, 0}, landed[2] = {0, 0}, commits[2] = {0, 0}, last_commit = -1;
  auto issue_b = [&](int t, int st) {
    bulk_load(Bs + st * B_BYTES, Wp + (long long)t * NC * KC, B_BYTES, bars + st);
    ++issued[st];
  };
  load_a(0, 0);
  if (tid == 0) issue_b(0, 0);
  for (int t = 0; t < 27; ++t) {
    const int s = t & 1;
    if (t + 1 < 27) {
      const int s1 = (t + 1) & 1;
      // stage s1 was last read by the MMAs of tap t-1
      if (t >= 1 && !mbar_wait(bars + 2 + s1, ((t - 1) >> 1) & 1, err)) ok = false;
      ok = __syncthreads_and(ok);
      if (!ok) break;
      load_a(t + 1, s1);
      if (tid == 0) issue_b(t + 1, s1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    // this thread's A copies of tap t are done; make them visible to the
    // tensor cores (async proxy) and to the issuing thread
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      if (!mbar_wait(bars + s, (t >> 1) & 1, err)) {
        ok = false;
      } else {
        ++landed[s];
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // K steps of 16 = two 8-channel chunks
        const uint64_t ad = sdesc(smem_u32(As + s * A_BYTES), A_LBO, SBO);
        const uint64_t bd = sdesc(smem_u32(Bs + s * B_BYTES), B_LBO, SBO);
        const uint32_t acc = t > 0 ? 1u : 0u;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < KC / 16; ++kk)
            mma_bf16(tbase, desc_add(ad, kk * 2 * A_LBO), desc_add(bd, kk * 2 * B_LBO), IDESC,
                     kk > 0 ? 1u : acc);
          mma_commit(bars + 2 + s);
        }
        __syncwarp();
        ++commits[s];
        last_commit = s;
      }
    }
  }
  // the last tap's MMAs (and so all earlier ones) completed
  ok = __syncthreads_and(ok);
  if (ok && !mbar_wait(bars + 2 + (26 & 1), (26 >> 1) & 1, err)) ok = false;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  ok = __syncthreads_and(ok);
  if (ok) {
    const int row = (warp & 3) * 32 + (tid & 31);  // TMEM lanes of a warp: its quarter
    const long long m = m0 + row;
    const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
    for (int n0 = 16 * (warp >> 2); n0 < NC; n0 += 16 * (HT / 128)) {
      float v[16];
      tmem_ld16(lane_addr + n0, v);
      if (m < Mtot) store16<DGRAD>(v, m, n0, bias, relu, y, ldy, offy, gx, ldg, offg, accumulate);
    }
  } else {
    // a wait ran out: let the copies and MMAs still in flight finish (each
    // wait bounded) before the shared memory and TMEM are given up
    cp_async_wait<0>();
    if (tid == 0) {
      for (int q = 0; q < 2; ++q)
        while (landed[q] < issued[q]) {
          if (!mbar_wait(bars + q, (uint32_t)(landed[q] & 1), err)) break;
          ++landed[q];
        }
      if (last_commit >= 0)
        mbar_wait(bars + 2 + last_commit, (uint32_t)((commits[last_commit] - 1) & 1), err);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                 "r"(tmem_cols)
                 : "memory");
}

// ---- weight gradient ------------------------------------------------------
constexpr int WG_KC = 64;     // voxels per stage (4 MMAs of K = 16)
constexpr int WG_STAGES = 3;  // stages in flight
constexpr int WG_CTAS = 608;  // target CTAs of a launch (4 per SM)

// CI input channels (MMA N), CO output channels (128 / CO taps per CTA).
// blockIdx.x: tap group; blockIdx.y: voxel range [q chunk, (q + 1) chunk).
template <int CI, int CO>
__global__ void __launch_bounds__(TC_THREADS) k_wgrad_tc(
    const __nv_bfloat16* __restrict__ x, int ldx, int offx, const __nv_bfloat16* __restrict__ g,
    int ldg, int offg, int lgD, long long Mtot, long long chunk, float* __restrict__ part,
    int tmem_cols, int* __restrict__ err) {
  constexpr int TPM = TC_M / CO;                 // taps per CTA
  constexpr int A_BYTES = TC_M * WG_KC * 2;      // 16 KB
  constexpr int B_BYTES = CI * WG_KC * 2;
  constexpr int ST_BYTES = A_BYTES + B_BYTES;
  constexpr uint32_t A_KSTR = (TC_M / 8) * 128;  // bytes between 8-voxel groups
  constexpr uint32_t B_KSTR = (CI / 8) * 128;
  constexpr uint32_t IDESC = idesc_bf16_mn(TC_M, CI);
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* done = reinterpret_cast<uint64_t*>(smem + WG_STAGES * ST_BYTES);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + WG_STAGES);
  const int tid = threadIdx.x, warp = warp_index();
  const int tile = blockIdx.x;
  const long long v0 = (long long)blockIdx.y * chunk;
  const long long v1 = v0 + chunk < Mtot ? v0 + chunk : Mtot;
  const int nk = v1 > v0 ? (int)((v1 - v0 + WG_KC - 1) / WG_KC) : 0;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < WG_STAGES; ++q) mbar_init(done + q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = *tslot;
  bool ok = true;

  // stage st <- voxels [v0 + k WG_KC, +WG_KC): chunk e of a tile lands at 16 e
  // (A: e = (8-voxel group, 8-row group, voxel in group); B likewise with the
  // 8-channel groups of x)
  auto load = [&](int k, int st) {
    unsigned char* As = smem + st * ST_BYTES;
    unsigned char* Bs = As + A_BYTES;
    const long long vb = v0 + (long long)k * WG_KC;
    for (int e = tid; e < TC_M * WG_KC / 8; e += TC_THREADS) {
      const int r8 = e & 7, mg = (e >> 3) & (TC_M / 8 - 1), kg = e >> 7;
      const int tl = mg / (CO / 8), co8 = mg - tl * (CO / 8);
      const int t = tile * TPM + tl;
      const long long v = vb + kg * 8 + r8;
      const bool ok_e = t < 27 && v < v1;
      long long src = 0;
      if (ok_e) {
        const int dx = t / 9 - 1, dy = (t / 3) % 3 - 1, dz = t % 3 - 1;
        src = (long long)tc_nbr((unsigned)v, lgD, -dx, -dy, -dz) * ldg + offg + 8 * co8;
      }
      cp_async16(As + 16 * e, g + src, ok_e);
    }
    for (int e = tid; e < CI * WG_KC / 8; e += TC_THREADS) {
      const int r8 = e & 7, ng = (e >> 3) % (CI / 8), kg = (e >> 3) / (CI / 8);
      const long long v = vb + kg * 8 + r8;
      const bool ok_e = v < v1;
      cp_async16(Bs + 16 * e, x + (ok_e ? v * ldx + offx + 8 * ng : 0), ok_e);
    }
  };

  int commits[WG_STAGES] = {}, last_commit = -1;
  for (int k = 0; k < WG_STAGES - 1; ++k) {
    if (k < nk) load(k, k);
    cp_async_commit();
  }
  for (int k = 0; k < nk; ++k) {
    const int st = k % WG_STAGES;
    const int kn = k + WG_STAGES - 1;
    if (kn < nk) {
      const int sn = kn % WG_STAGES;  // last read by the MMAs of chunk k - 1
      if (k >= 1 && tid == 0 &&
          !mbar_wait(done + sn, (uint32_t)(((k - 1) / WG_STAGES) & 1), err))
        ok = false;
      ok = __syncthreads_and(ok);
      if (!ok) break;
      load(kn, sn);
    }
    cp_async_commit();
    cp_async_wait<WG_STAGES - 1>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = smem_u32(smem + st * ST_BYTES), b0 = a0 + A_BYTES;
      const uint64_t ad = sdesc_mn(a0, 128, A_KSTR), bd = sdesc_mn(b0, 128, B_KSTR);
      const uint32_t acc = k > 0 ? 1u : 0u;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < WG_KC / 16; ++kk)
          mma_bf16(tbase, desc_add(ad, 2 * kk * A_KSTR), desc_add(bd, 2 * kk * B_KSTR), IDESC,
                   kk > 0 ? 1u : acc);
        mma_commit(done + st);
      }
      __syncwarp();
      ++commits[st];
      last_commit = st;
    }
  }
  ok = __syncthreads_and(ok);
  if (ok && nk > 0 && tid == 0 &&
      !mbar_wait(done + (nk - 1) % WG_STAGES, (uint32_t)(((nk - 1) / WG_STAGES) & 1), err))
    ok = false;
  ok = __syncthreads_and(ok);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    // row = (tap in group, co); its CI accumulators go to part[q][t][ci][co]
    const int row = warp * 32 + (tid & 31);
    const int tl = row / CO, co = row - tl * CO, t = tile * TPM + tl;
    const long long base = ((long long)blockIdx.y * 27 + (t < 27 ? t : 0)) * CI * CO + co;
    const uint32_t lane_addr = tbase + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int n0 = 0; n0 < CI; n0 += 16) {
      float v[16];
      tmem_ld16(lane_addr + n0, v);
      if (t < 27) {
#pragma unroll
        for (int i = 0; i < 16; ++i) part[base + (long long)(n0 + i) * CO] = nk > 0 ? v[i] : 0.f;
      }
    }
  } else {
    // a wait ran out: let the copies and MMAs in flight finish (bounded)
    cp_async_wait<0>();
    if (tid == 0 && last_commit >= 0)
      mbar_wait(done + last_commit, (uint32_t)((commits[last_commit] - 1) & 1), err);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                 "r"(tmem_cols)
                 : "memory");
}

// splits of the voxel range: about WG_CTAS CTAs in all, none empty
void wgrad_split(int Cout, long long Mtot, int* S, long long* chunk) {
  const int nt = (27 + TC_M / Cout - 1) / (TC_M / Cout);
  const long long nch = (Mtot + WG_KC - 1) / WG_KC;
  long long s = std::max(1, WG_CTAS / nt);
  if (s > nch) s = nch;
  const long long per = (nch + s - 1) / s;
  *S = (int)((nch + per - 1) / per);
  *chunk = per * WG_KC;
}

template <int CI, int CO>
void launch_wgrad(TView x, TView g, int lgD, long long Mtot, float* part, int* err, int* S_out,
                  cudaStream_t s) {
  constexpr int ST_BYTES = TC_M * WG_KC * 2 + CI * WG_KC * 2;
  const int cols = CI <= 32 ? 32 : (CI <= 64 ? 64 : (CI <= 128 ? 128 : 256));
  const size_t need = (size_t)WG_STAGES * ST_BYTES + WG_STAGES * 8 + 16;
  const int k = 512 / cols;
  const size_t cap = 233472 / (k + 1) - 1024 + 16;
  const size_t smem = need > cap ? need : cap;
  static DeviceOnce once;
  smem_opt_in(once, k_wgrad_tc<CI, CO>);
  int S;
  long long chunk;
  wgrad_split(CO, Mtot, &S, &chunk);
  const int nt = (27 + TC_M / CO - 1) / (TC_M / CO);
  k_wgrad_tc<CI, CO><<<dim3(nt, S), TC_THREADS, smem, s>>>(x.p, x.ld, x.off, g.p, g.ld, g.off,
                                                           lgD, Mtot, chunk, part, cols, err);
  *S_out = S;
}

// ---- halo-tiled forward and input gradient for the full-resolution layers ---
// A CTA computes TX x-slices of a 16 (y) x 8 (z) block of output voxels, one
// M = 128 tile per slice (row m = 8 y + z).  It stages the input once as a
// (TX + 2) x 18 x 10 voxel block with its one-voxel periodic halo, laid out
// [8-channel group][x][y][z] with 16 bytes per voxel, and all 27 taps'
// packed weights.  The A operand of tap (dy, dz) on an input slice is
// then a K-major no-swizzle view of the halo block: core matrices of 8 z-
// consecutive voxels x 16 bytes, 8-row groups (y) 10 x 16 bytes apart (SBO),
// 8-channel groups one block-plane apart (LBO), the start shifted by the tap
// offset.
//
// An MMA of M = 128, K = 16 takes 39 clocks at N = 16, 44 at 48, 56 at 96 (measured): the
// A operand's 4 KB set the time.  The three taps dx of an input slice are therefore one
// MMA: the accumulators of neighbouring output slices lie side by side in TMEM, and B holds
// the three taps' weights side by side, so that its columns add to the output slices
// before, at and after the input slice.  (TX + 2) 9 (KC / 16) MMAs instead of
// TX 27 (KC / 16), each output's terms in the same order.  The accumulators start at
// zero, since one MMA meets slices at different stages.
// A CTA stays for many tiles: its weights and tensor memory are set up once, and the next
// tile's block arrives while the results of this one are stored.
// 256^3: 16 -> 16 433 us (a CTA per tile, one MMA per tap: 536), 48 -> 16 2023 (2025, now
// bound by the block's arrival: two CTAs per SM hold one block each); 128^3: 32 -> 32 210
// (251), 16 -> 32 97 (117); input gradient on 4 x 64^3: 16 -> 48 89 (113), 16 -> 16 40
// (54).  TX = 8 for 16 channels: 25% more than the tile read against 50% at 4 (356 against
// 437 us).
// The halo block of a CTA: 8-channel chunk c8 of voxel (hx, hy, hz) lands at
// c8 halo_plane + 16 ((hx HY + hy) HZ + hz); consecutive threads take the
// chunks of a voxel (contiguous in memory; the plane stride's extra 16 bytes
// put them into different banks)
constexpr int HY = 18, HZ = 10;
constexpr int halo_plane(int hx) { return hx * HY * HZ * 16 + 16; }

template <int CH, int HX>
__device__ __forceinline__ void load_halo(unsigned char* Hs, const __nv_bfloat16* __restrict__ x,
                                          int ldx, int offx, unsigned sample, int x0, int y0,
                                          int z0, int lgD, int tid) {
  const int M = (1 << lgD) - 1;
#pragma unroll 4
  for (int e = tid; e < CH * HX * HY * HZ; e += HT) {
    const int v = e / CH, c8 = e - v * CH;
    const int r = v / HZ, hz = v - r * HZ;
    const int hx = r / HY, hy = r - hx * HY;
    const unsigned q = ((((sample << lgD) + ((x0 + hx - 1) & M)) << lgD) + ((y0 + hy - 1) & M));
    const unsigned vox = (q << lgD) + ((z0 + hz - 1) & M);
    cp_async16(Hs + c8 * halo_plane(HX) + 16 * v, x + (size_t)vox * ldx + offx + 8 * c8, true);
  }
}

template <int KC, int NC, bool DGRAD, int TX>
__global__ void __launch_bounds__(HT) k_conv_halo(
    const __nv_bfloat16* __restrict__ x, int ldx, int offx, const __nv_bfloat16* __restrict__ Wp,
    const float* __restrict__ bias, int relu, __nv_bfloat16* __restrict__ y, int ldy, int offy,
    float* __restrict__ gx, int ldg, int offg, int accumulate, int lgD, int tiles, int tmem_cols,
    int* __restrict__ err) {
  constexpr int HX = TX + 2, CH = KC / 8;
  constexpr int PLANE = halo_plane(HX);  // bytes of one 8-channel group
  constexpr int H_BYTES = CH * PLANE;
  constexpr int W_BYTES = 27 * NC * KC * 2;
  constexpr uint32_t SBO = HZ * 16, B_LBO = 3 * NC * 16;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* Hs = smem;
  unsigned char* Ws = smem + H_BYTES;  // [dy, dz][8-channel group][slot][NC rows]
  uint64_t* bar = reinterpret_cast<uint64_t*>(Ws + W_BYTES);  // the MMAs
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  const int tid = threadIdx.x, warp = warp_index();
  // tile coordinates: z blocks of 8, y blocks of 16, x blocks of TX, samples
  const int lz = lgD - 3, ly = lgD - 4, nx = (1 << lgD) / TX;
  auto coords = [&](int t, int* x0, int* y0, int* z0) {
    *z0 = (t & ((1 << lz) - 1)) * 8;
    t >>= lz;
    *y0 = (t & ((1 << ly) - 1)) * 16;
    t >>= ly;
    const int b = t / nx;
    *x0 = (t - b * nx) * TX;
    return b;  // the sample
  };
  auto load = [&](int t) {
    int x0, y0, z0;
    const int b = coords(t, &x0, &y0, &z0);
    load_halo<CH, HX>(Hs, x, ldx, offx, (unsigned)b, x0, y0, z0, lgD, tid);
    cp_async_commit();
  };
  // the copies run while the CTA gets its tensor memory
#pragma unroll 4
  for (int e = tid; e < 27 * CH * NC; e += HT) {  // 16 bytes: row n of tap t's group c
    const int n = e % NC, tc = e / NC, t = tc / CH, c = tc - t * CH;
    const int dx = t / 9, q = DGRAD ? dx : 2 - dx;
    cp_async16(Ws + ((((t - 9 * dx) * CH + c) * 3 + q) * NC + n) * 16, Wp + 8 * (size_t)e, true);
  }
  load((int)blockIdx.x);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = *tslot;
  // warp w reads TMEM lanes 32 (w & 3)..; the column chunks alternate between
  // the two groups of four warps
  const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
  for (int q = warp >> 2; q < TX * (NC / 16); q += HT / 128) tmem_zero16(lane_addr + 16 * q);
  uint32_t parity = 0;
#pragma unroll 1
  for (int tile = (int)blockIdx.x; tile < tiles; tile += (int)gridDim.x, parity ^= 1u) {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int sg = DGRAD ? -1 : 1;
      const uint64_t ad0 = sdesc(smem_u32(Hs), PLANE, SBO), bd0 = sdesc(smem_u32(Ws), B_LBO, 128);
      const bool lead = elect_one();
#pragma unroll 1
      for (int h = 0; h < HX; ++h) {
        const int hx = DGRAD ? HX - 1 - h : h;  // input slice x0 - 1 + hx: dx ascends per output
        // its slots in the tile; slot q is the output slice x0 + hx - 2 + q, its tap dx = 1 - q
        // (input gradient: q - 1)
        const int q0 = hx < 2 ? 2 - hx : 0, q1 = hx >= TX ? TX + 1 - hx : 2;
        const uint32_t dcol = tbase + (hx - 2 + q0) * NC;
        const uint32_t idesc = idesc_bf16(TC_M, (q1 - q0 + 1) * NC);
        const uint64_t bh = desc_add(bd0, (uint32_t)(q0 * NC * 16));
#pragma unroll 1
        for (int t = 0; t < 9; ++t) {
          const int dy = sg * (t / 3 - 1), dz = sg * (t % 3 - 1);
          const uint64_t at = desc_add(ad0, (uint32_t)(((hx * HY + (dy + 1)) * HZ + (dz + 1)) * 16));
          const uint64_t bt = desc_add(bh, (uint32_t)(t * (3 * NC * KC * 2)));
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < KC / 16; ++kk)
              mma_bf16(dcol, desc_add(at, 2 * kk * PLANE), desc_add(bt, 2 * kk * B_LBO), idesc, 1u);
          }
          __syncwarp();
        }
      }
      if (lead) mma_commit(bar);
    }
    const bool ok = __syncthreads_and(tid != 0 || mbar_wait(bar, parity, err));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) {  // the wait ran out: the MMAs in flight (bounded)
      if (tid == 0) mbar_wait(bar, parity, err);
      break;
    }
    // the next tile's block arrives while this one's results are stored
    if (tile + (int)gridDim.x < tiles) load(tile + (int)gridDim.x);
    int x0, y0, z0;
    const long long b = coords(tile, &x0, &y0, &z0);
    const int row = (warp & 3) * 32 + (tid & 31);
    const long long m0 =
        (b << (3 * lgD)) + ((((long long)x0 << lgD) + (y0 + (row >> 3))) << lgD) + (z0 + (row & 7));
#pragma unroll 1
    for (int q = warp >> 2; q < TX * (NC / 16); q += HT / 128) {
      const int tx = q / (NC / 16), n0 = 16 * (q - tx * (NC / 16));
      float v[16];
      tmem_ld16(lane_addr + 16 * q, v);
      tmem_zero16(lane_addr + 16 * q);
      store16<DGRAD>(v, m0 + ((long long)tx << (2 * lgD)), n0, bias, relu, y, ldy, offy, gx, ldg,
                     offg, accumulate);
    }
  }
  cp_async_wait<0>();
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                 "r"(tmem_cols)
                 : "memory");
}

template <int KC, int NC, bool DG, int TX>
void launch_halo(const TcArgs& a, cudaStream_t s) {
  constexpr int H_BYTES = (KC / 8) * halo_plane(TX + 2), W_BYTES = 27 * NC * KC * 2;
  constexpr int cols0 = TX * NC;
  constexpr int cols = cols0 <= 32 ? 32 : (cols0 <= 64 ? 64 : (cols0 <= 128 ? 128 : 256));
  // CTAs per SM: by shared memory (1 KB reserved for each) and by tensor memory; the
  // shared memory is padded so that no more are resident (tcgen05.alloc would wait)
  constexpr int need = H_BYTES + W_BYTES + 8 + 16;
  constexpr int fit = 233472 / (need + 1024), mem = 512 / cols;
  constexpr int per_sm = fit < mem ? fit : mem;
  constexpr int cap = 233472 / (per_sm + 1) - 1024 + 16, smem = need > cap ? need : cap;
  static_assert(per_sm >= 1 && smem <= 227 * 1024, "one CTA fits");
  static DeviceOnce once;
  smem_opt_in(once, k_conv_halo<KC, NC, DG, TX>);
  const int tiles = (int)(a.Mtot / (TX * 16 * 8));
  k_conv_halo<KC, NC, DG, TX><<<(unsigned)std::min(tiles, 152 * per_sm), HT, smem, s>>>(
      a.x, a.ldx, a.offx, a.Wp, a.bias, a.relu, a.y, a.ldy, a.offy, a.gx, a.ldg, a.offg,
      a.accumulate, a.lgD, tiles, cols, a.err);
}

// The same halo-tiled form for layers whose 27 weight slices do not fit beside
// the input block: the block stays resident while the taps' weight slices
// stream through NS shared-memory stages (one bulk copy each).  One warp, by its
// elected lane, loads the slices and issues the MMAs, so the loop over taps has no
// block-wide synchronisation.  A tap's MMAs take about 0.3 us and a copy's latency is 1 us:
// as many slices are in flight as the shared memory holds, up to 8 (with two,
// 96 -> 32 waited for every slice: 110 us on 4 x 32^3).
constexpr int halo_s_fit(int kc, int nc, int tx, int bytes) {
  return (bytes - (kc / 8) * halo_plane(tx + 2)) / (nc * kc * 2);
}
// up to 8 where two CTAs share an SM with at least four each, else one CTA's room
constexpr int halo_s_stages(int kc, int nc, int tx) {
  const int two = halo_s_fit(kc, nc, tx, 112 * 1024), one = halo_s_fit(kc, nc, tx, 226 * 1024);
  const int n = two >= 4 ? two : one;
  return n > 8 ? 8 : n;
}

template <int KC, int NC, bool DGRAD, int TX>
__global__ void __launch_bounds__(HT) k_conv_halo_s(
    const __nv_bfloat16* __restrict__ x, int ldx, int offx, const __nv_bfloat16* __restrict__ Wp,
    const float* __restrict__ bias, int relu, __nv_bfloat16* __restrict__ y, int ldy, int offy,
    float* __restrict__ gx, int ldg, int offg, int accumulate, int lgD, int tmem_cols,
    int* __restrict__ err) {
  constexpr int HX = TX + 2, CH = KC / 8;
  constexpr int PLANE = halo_plane(HX);
  constexpr int H_BYTES = CH * PLANE;
  constexpr int T_BYTES = NC * KC * 2;  // one tap's weight slice
  constexpr int NS = halo_s_stages(KC, NC, TX);
  static_assert(NS >= 2, "two weight slices beside the block");
  constexpr uint32_t SBO = HZ * 16, B_LBO = NC * 16;
  constexpr uint32_t IDESC = idesc_bf16(TC_M, NC);
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* Hs = smem;
  unsigned char* Ws = smem + H_BYTES;  // [NS][T_BYTES]
  uint64_t* bars = reinterpret_cast<uint64_t*>(Ws + NS * T_BYTES);  // full[NS], done[NS]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2 * NS);
  const int tid = threadIdx.x, warp = warp_index();
  const int D = 1 << lgD, M = D - 1;
  const int nz = D >> 3, ny = D >> 4, nx = D / TX;
  long long bid = blockIdx.x;
  const int bz = (int)(bid % nz);
  bid /= nz;
  const int by = (int)(bid % ny);
  bid /= ny;
  const int bx = (int)(bid % nx);
  const long long b = bid / nx;
  const int x0 = bx * TX, y0 = by * 16, z0 = bz * 8;
  const long long sbase = b << (3 * lgD);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < 2 * NS; ++q) mbar_init(bars + q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = *tslot;
  int issued = 0, landed = 0, committed = 0;  // warp 0: slices copied, arrived, used
  auto issue_w = [&](int q) {
    bulk_load(Ws + (q % NS) * T_BYTES, Wp + (long long)q * NC * KC, (uint32_t)T_BYTES,
              bars + q % NS);
    ++issued;
  };
  if (warp == 0) {
    const bool lead = elect_one();
    for (int q = 0; q < NS - 1; ++q)
      if (lead) issue_w(q); else ++issued;
    __syncwarp();
  }
  load_halo<CH, HX>(Hs, x, ldx, offx, (unsigned)b, x0, y0, z0, lgD, tid);
  cp_async_commit();
  cp_async_wait<0>();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  bool ok = true;
  if (warp == 0) {
    const int sg = DGRAD ? -1 : 1;
    const uint64_t ad0 = sdesc(smem_u32(Hs), PLANE, SBO), bd0 = sdesc(smem_u32(Ws), B_LBO, 128);
    const bool lead = elect_one();
#pragma unroll 1
    for (int t = 0; t < 27; ++t) {
      const int st = t % NS, q = t + NS - 1;
      if (q < 27) {
        // its stage was last read by the MMAs of tap t - 1
        if (t >= 1 && !mbar_wait(bars + NS + q % NS, ((t - 1) / NS) & 1, err)) {
          ok = false;
          break;
        }
        if (lead) issue_w(q); else ++issued;
        __syncwarp();
      }
      if (!mbar_wait(bars + st, (t / NS) & 1, err)) {
        ok = false;
        break;
      }
      ++landed;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int dx = sg * (t / 9 - 1), dy = sg * ((t / 3) % 3 - 1), dz = sg * (t % 3 - 1);
      const uint64_t at = desc_add(ad0, (uint32_t)((((dx + 1) * HY + (dy + 1)) * HZ + (dz + 1)) * 16));
      const uint64_t bt = desc_add(bd0, (uint32_t)(st * T_BYTES));
      const uint32_t acc = t > 0 ? 1u : 0u;
      if (lead) {
#pragma unroll
        for (int kk = 0; kk < KC / 16; ++kk)
#pragma unroll
          for (int tx = 0; tx < TX; ++tx)  // consecutive MMAs into different accumulators
            mma_bf16(tbase + tx * NC, desc_add(at, tx * (HY * HZ * 16) + 2 * kk * PLANE),
                     desc_add(bt, 2 * kk * B_LBO), IDESC, kk > 0 ? 1u : acc);
        mma_commit(bars + NS + st);
      }
      __syncwarp();
      ++committed;
    }
    if (ok && !mbar_wait(bars + NS + 26 % NS, (26 / NS) & 1, err)) ok = false;
    if (!ok) {
      // a wait ran out: the copies and MMAs in flight (each wait bounded)
      __syncwarp();
      for (; landed < issued; ++landed)
        if (!mbar_wait(bars + landed % NS, (uint32_t)((landed / NS) & 1), err)) break;
      if (committed > 0)
        mbar_wait(bars + NS + (committed - 1) % NS, (uint32_t)(((committed - 1) / NS) & 1), err);
    }
  }
  ok = __syncthreads_and(ok);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    // warp w reads TMEM lanes 32 (w & 3)..; the column chunks alternate between
    // the two groups of four warps
    const int row = (warp & 3) * 32 + (tid & 31);
    const int yy = row >> 3, zz = row & 7;
    const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
    for (int q = warp >> 2; q < TX * (NC / 16); q += HT / 128) {
      const int tx = q / (NC / 16), n0 = 16 * (q - tx * (NC / 16));
      const long long m = sbase + ((((long long)(x0 + tx) << lgD) + (y0 + yy)) << lgD) + (z0 + zz);
      float v[16];
      tmem_ld16(lane_addr + tx * NC + n0, v);
      store16<DGRAD>(v, m, n0, bias, relu, y, ldy, offy, gx, ldg, offg, accumulate);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                 "r"(tmem_cols)
                 : "memory");
}

template <int KC, int NC, bool DG, int TX>
void launch_halo_s(const TcArgs& a, cudaStream_t s) {
  constexpr int H_BYTES = (KC / 8) * halo_plane(TX + 2), T_BYTES = NC * KC * 2;
  const int cols0 = TX * NC;
  const int cols = cols0 <= 32 ? 32 : (cols0 <= 64 ? 64 : (cols0 <= 128 ? 128 : 256));
  constexpr int NS = halo_s_stages(KC, NC, TX);
  const size_t need = (size_t)H_BYTES + NS * T_BYTES + 2 * NS * 8 + 16;
  const int k = 512 / cols;
  const size_t cap = 233472 / (k + 1) - 1024 + 16;
  const size_t smem = need > cap ? need : cap;
  static DeviceOnce once;
  smem_opt_in(once, k_conv_halo_s<KC, NC, DG, TX>);
  const long long tiles = a.Mtot / (TX * 16 * 8);
  k_conv_halo_s<KC, NC, DG, TX><<<(unsigned)tiles, HT, smem, s>>>(
      a.x, a.ldx, a.offx, a.Wp, a.bias, a.relu, a.y, a.ldy, a.offy, a.gx, a.ldg, a.offg,
      a.accumulate, a.lgD, cols, a.err);
}

// ---- weight gradient from resident blocks (the layers of up to 32 output
// channels, whose voxels are the most) --------------------------------------
// dW[t][ci][co] = sum_u x[u][ci] g[u - d_t][co].  A stage holds PL x planes of
// x over a 16 (y) x 8 (z) block with its one-voxel halo in y and z, and the
// PL + 2 slices of g around them without a halo, both [plane][8-channel group]
// [y][z] with 16 bytes per voxel.  Reduction = the block's 128 voxels, both
// operands MN-major (core matrices of 8 z-consecutive voxels x 16 bytes of
// channels, the next 8 voxels one y row on, the next 8 channels one group on):
//   A: rows (slice s, co): the 16 groups from the first slice on, M = 128
//      (rows of slices past PL + 2 are not used; they read what the stage holds);
//   B: columns (plane p, ci), N = PL CI, started (dy, dz) into the halo.
// One accumulator per (dy, dz) then holds the taps of every dx = p - s: each
// operand is staged once instead of once per tap (the per-tap kernel spent its
// time on the address arithmetic of that staging).  A CTA walks its range of
// blocks with the next stages in flight and the ND accumulators in TMEM.  The
// tensor core's FP32 accumulation truncates, an error that grows with the length
// of the chain, so every kFlush voxels the accumulators are added, rounded to
// nearest, to the CTA's partial dW in shared memory: relative error 4e-7 at
// 96 -> 32 on 4 x 32^3 against 1.6e-6 of the per-tap kernel's chains (2.8e-6
// without the flushes).
template <int CI, int CO, int PL, int ND>
struct WgHalo {
  static constexpr int CI8 = CI / 8, CO8 = CO / 8, SL = 16 / CO8;
  static constexpr int NG = PL + 2;                         // slices of g loaded
  static constexpr int XG = HY * HZ * 16, GG = 16 * 8 * 16; // bytes of an 8-channel group
  static constexpr int XB = PL * CI8 * XG, GB = NG * CO8 * GG, ST = XB + GB;
  static constexpr int N = PL * CI, COLS = ND * N;
  static constexpr int kFlush = 512, FL = kFlush / (128 * PL);  // voxels, blocks
  static constexpr int ACC = 3 * ND * CI * CO * 4;               // bytes of a partial dW
  static constexpr int STAGES = 3 * ST + ACC <= 226 * 1024 ? 3 : 2;
  // the rows of slices past NG read on behind the last stage: into the partial dW
  static constexpr int OVER = (SL - NG) * CO8 * GG;
  static constexpr int TCOLS = COLS <= 256 ? 256 : 512;
  static_assert(SL >= NG && N <= 256 && COLS <= 512 && OVER <= ACC &&
                    STAGES * ST + ACC <= 226 * 1024, "tile");
};

template <int CI, int CO, int PL, int ND>
__global__ void __launch_bounds__(HT) k_wgrad_halo(
    const __nv_bfloat16* __restrict__ x, int ldx, int offx, const __nv_bfloat16* __restrict__ g,
    int ldg, int offg, int lgD, int ntile, int chunk, float* __restrict__ part,
    int* __restrict__ err) {
  using W = WgHalo<CI, CO, PL, ND>;
  constexpr uint32_t IDESC = idesc_bf16_mn(TC_M, W::N);
  extern __shared__ __align__(1024) unsigned char smem[];
  float* acc = reinterpret_cast<float*>(smem + W::STAGES * W::ST);  // [dx][q][ci][co]
  uint64_t* done = reinterpret_cast<uint64_t*>(smem + W::STAGES * W::ST + W::ACC);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + W::STAGES);
  const int tid = threadIdx.x, warp = warp_index();
  const int dy0 = ND == 9 ? -1 : (int)blockIdx.x - 1;  // ND = 3: this CTA's dy
  const int k0 = blockIdx.y * chunk, k1 = min(ntile, k0 + chunk);
  const int nk = k1 > k0 ? k1 - k0 : 0;
  const int D = 1 << lgD, M = D - 1, nz = D >> 3, ny = D >> 4;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(W::TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < W::STAGES; ++q) mbar_init(done + q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tbase = *tslot;
  bool ok = true;

  auto load = [&](int k, int st) {
    unsigned char* X = smem + st * W::ST;
    unsigned char* Gs = X + W::XB;
    int r = k0 + k;  // block: z, then y, then x planes, then sample
    const int z0 = 8 * (r % nz);
    r /= nz;
    const int y0 = 16 * (r % ny);
    r /= ny;
    const int p0 = PL * (r % (D / PL));
    const unsigned b = (unsigned)(r / (D / PL));
#pragma unroll 4
    for (int e = tid; e < W::CI8 * PL * HY * HZ; e += HT) {
      const int v = e / W::CI8, c8 = e - v * W::CI8;
      const int q = v / HZ, hz = v - q * HZ, p = q / HY, hy = q - p * HY;
      const unsigned row = ((((b << lgD) + p0 + p) << lgD) + ((y0 + hy - 1) & M));
      const unsigned vox = (row << lgD) + ((z0 + hz - 1) & M);
      cp_async16(X + (p * W::CI8 + c8) * W::XG + 16 * (hy * HZ + hz),
                 x + (size_t)vox * ldx + offx + 8 * c8, true);
    }
#pragma unroll 4
    for (int e = tid; e < W::CO8 * W::NG * 128; e += HT) {
      const int v = e / W::CO8, c8 = e - v * W::CO8;
      const int z = v & 7, y = (v >> 3) & 15, s = v >> 7;
      const unsigned row = ((((b << lgD) + ((p0 - 1 + s) & M)) << lgD) + y0 + y);
      const unsigned vox = (row << lgD) + z0 + z;
      cp_async16(Gs + (s * W::CO8 + c8) * W::GG + 16 * (v & 127),
                 g + (size_t)vox * ldg + offg + 8 * c8, true);
    }
  };

  float* out = part + (long long)blockIdx.y * 27 * CI * CO;
  // Row (s, co) of accumulator (dy, dz), columns (p, ci): tap dx = p - s + 1 (s
  // counted from the slice before plane 0).  The planes' terms of a tap lie in
  // different rows, so the planes are added one after the other.
  auto flush = [&](bool first) {
    const int row = (warp & 3) * 32 + (tid & 31);
    const int s = row / CO, co = row - s * CO;
    const uint32_t lane_addr = tbase + ((uint32_t)((warp & 3) * 32) << 16);
    for (int p = 0; p < PL; ++p) {
      const int dx = p - s + 1;  // -1, 0 or 1 where this row contributes
#pragma unroll 1
      for (int e = warp >> 2; e < ND * (CI / 16); e += HT / 128) {
        const int q = e / (CI / 16), n0 = 16 * (e - q * (CI / 16));
        float v[16];
        tmem_ld16(lane_addr + q * W::N + p * CI + n0, v);
        if (dx >= -1 && dx <= 1) {
          float* w = acc + (((dx + 1) * ND + q) * CI + n0) * CO + co;
#pragma unroll
          for (int i = 0; i < 16; ++i) w[i * CO] = first && p == 0 ? v[i] : w[i * CO] + v[i];
        }
        __syncwarp();
      }
      __syncthreads();
    }
  };

  int commits[W::STAGES] = {}, last_commit = -1;
  bool fresh = true, first = true;  // accumulators to be overwritten; no flush yet
  for (int k = 0; k < W::STAGES - 1; ++k) {
    if (k < nk) load(k, k);
    cp_async_commit();
  }
  for (int k = 0; k < nk; ++k) {
    const int st = k % W::STAGES, kn = k + W::STAGES - 1;
    if (kn < nk) {
      const int sn = kn % W::STAGES;  // last read by the MMAs of block k - 1
      if (k >= 1 && tid == 0 &&
          !mbar_wait(done + sn, (uint32_t)(((k - 1) / W::STAGES) & 1), err))
        ok = false;
      ok = __syncthreads_and(ok);
      if (!ok) break;
      load(kn, sn);
    }
    cp_async_commit();
    cp_async_wait<W::STAGES - 1>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t x0 = smem_u32(smem + st * W::ST);
      const uint64_t ad = sdesc_mn(x0 + W::XB, W::GG, 128), bd0 = sdesc_mn(x0, W::XG, HZ * 16);
      const bool lead = elect_one();
#pragma unroll 1
      for (int q = 0; q < ND; ++q) {
        const int dy = ND == 9 ? q / 3 - 1 : dy0, dz = q % 3 - 1;
        const uint64_t bd = desc_add(bd0, (uint32_t)(((dy + 1) * HZ + dz + 1) * 16));
        const uint32_t acc0 = fresh ? 0u : 1u;
        if (lead) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)  // 16 voxels: two y rows
            mma_bf16(tbase + q * W::N, desc_add(ad, kk * 256), desc_add(bd, 2 * kk * HZ * 16),
                     IDESC, kk > 0 ? 1u : acc0);
        }
        __syncwarp();
      }
      if (lead) mma_commit(done + st);
      ++commits[st];
      last_commit = st;
    }
    fresh = false;
    if ((k + 1) % W::FL == 0 || k + 1 == nk) {
      if (tid == 0 && !mbar_wait(done + st, (uint32_t)((k / W::STAGES) & 1), err)) ok = false;
      ok = __syncthreads_and(ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      flush(first);
      // the reads are done before the next MMA overwrites the accumulators
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      fresh = true;
      first = false;
    }
  }
  ok = __syncthreads_and(ok);
  if (ok) {
    // [dx][q][ci][co] -> the taps of this CTA's dy (all nine q: the whole dW)
    for (int e = tid; e < 3 * ND * CI * CO; e += HT) {
      const int dq = e / (CI * CO), dx = dq / ND, q = dq - dx * ND;
      const int t = dx * 9 + (ND == 9 ? q : 3 * (int)blockIdx.x + q);
      out[(long long)t * CI * CO + (e - dq * CI * CO)] = acc[e];
    }
  } else {
    // a wait ran out: let the copies and MMAs in flight finish (bounded)
    cp_async_wait<0>();
    if (tid == 0 && last_commit >= 0)
      mbar_wait(done + last_commit, (uint32_t)((commits[last_commit] - 1) & 1), err);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                 "r"(W::TCOLS)
                 : "memory");
}

// ranges of blocks: one CTA per SM (its accumulators take the SM's TMEM)
constexpr int WG_HALO_CTAS = 152;

template <int CI, int CO, int PL, int ND>
void launch_wgrad_halo(TView x, TView g, int B, int lgD, float* part, int* err, int* S_out,
                       cudaStream_t s) {
  using W = WgHalo<CI, CO, PL, ND>;
  const size_t need = (size_t)W::STAGES * W::ST + W::ACC + W::STAGES * 8 + 16;
  const size_t cap = 233472 / (512 / W::TCOLS + 1) - 1024 + 16;
  const size_t smem = need > cap ? need : cap;
  static DeviceOnce once;
  smem_opt_in(once, k_wgrad_halo<CI, CO, PL, ND>);
  const int ntile = (B << (3 * lgD - 7)) / PL;
  const int S0 = std::max(1, WG_HALO_CTAS / (9 / ND));
  const int chunk = (ntile + S0 - 1) / S0, S = (ntile + chunk - 1) / chunk;
  k_wgrad_halo<CI, CO, PL, ND><<<dim3(9 / ND, S), HT, smem, s>>>(
      x.p, x.ld, x.off, g.p, g.ld, g.off, lgD, ntile, chunk, part, err);
  *S_out = S;
}

// Packed weight slices.  Forward (N = Cout, K = Cin):
//   Wp[t][c][n][k8] = W[t][8c + k8][n]
// Input gradient (N = Cin, K = Cout):
//   Wp[t][c][n][k8] = W[t][n][8c + k8]
// i.e. per tap the K-major N x K tile, 8-channel chunks of K one after the
// other, the N rows of a chunk contiguous (the shared-memory layout).
__global__ void k_pack_tc(const __nv_bfloat16* __restrict__ W, int Cin, int Cout, int dgrad,
                          __nv_bfloat16* __restrict__ Wp) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long per = (long long)Cin * Cout;
  if (e >= 27 * per) return;
  const int t = (int)(e / per);
  const long long r = e - t * per;
  const int N = dgrad ? Cin : Cout;
  const int k8 = (int)(r & 7), n = (int)((r >> 3) % N), c = (int)((r >> 3) / N);
  const int kidx = 8 * c + k8;
  const int ci = dgrad ? n : kidx, co = dgrad ? kidx : n;
  Wp[e] = W[((long long)t * Cin + ci) * Cout + co];
}

template <int KC, int NC, bool DG>
void launch_tc(const TcArgs& a, cudaStream_t s) {
  constexpr int A_BYTES = a_bytes(KC), B_BYTES = NC * KC * 2;
  const int cols = NC <= 32 ? 32 : (NC <= 64 ? 64 : (NC <= 128 ? 128 : 256));
  const size_t need = 2 * (size_t)A_BYTES + 2 * (size_t)B_BYTES + 4 * 8 + 16;
  // at most 512 / cols CTAs per SM may hold TMEM at once: pad the shared
  // memory so that no more are resident (tcgen05.alloc would wait)
  // (each CTA also holds 1 KB of reserved shared memory)
  const int k = 512 / cols;
  const size_t cap = 233472 / (k + 1) - 1024 + 16;
  const size_t smem = need > cap ? need : cap;
  static DeviceOnce once;
  smem_opt_in(once, k_conv_tc<KC, NC, DG>);
  const unsigned grid = (unsigned)((a.Mtot + TC_M - 1) / TC_M);
  k_conv_tc<KC, NC, DG><<<grid, HT, smem, s>>>(
      a.x, a.ldx, a.offx, a.Wp, a.bias, a.relu, a.y, a.ldy, a.offy, a.gx, a.ldg, a.offg,
      a.accumulate, a.lgD, a.Mtot, cols, a.err);
}

}  // namespace

long long nn_tc_packed_size(int Cin, int Cout) { return 27LL * Cin * Cout; }

void nn_tc_pack(const __nv_bfloat16* W, int Cin, int Cout, int dgrad, __nv_bfloat16* Wp,
                cudaStream_t s) {
  const long long n = 27LL * Cin * Cout;
  k_pack_tc<<<nblocks(n, 256), 256, 0, s>>>(W, Cin, Cout, dgrad, Wp);
}

// (K, N) pairs of the network's convolutions: forward (Cin, Cout) and input
// gradient (Cout, Cin)
bool nn_tc_supported(int K, int N) {
  static const int kn[][2] = {{16, 16},  {16, 32},  {32, 32},  {32, 64},  {64, 64},  {64, 128},
                              {128, 128}, {192, 64}, {96, 32},  {48, 16},  {32, 16},  {64, 32},
                              {128, 64}, {64, 192}, {32, 96},  {16, 48}};
  for (auto& p : kn)
    if (p[0] == K && p[1] == N) return true;
  return false;
}

bool nn_tc_conv(const TcArgs& a, int K, int N, bool dgrad, cudaStream_t s) {
  // the layers of the two finest levels whose input block and 27 weight
  // slices fit one CTA's shared memory run on the halo-tiled kernel when the
  // grid holds its tiles (16^3 and more); the slices per tile (fourth argument) are
  // the fastest of 1, 2, 4 and 8 on 128^3 and 256^3 that fit
  if (a.lgD >= 4 && a.lgD <= 10) {
#define HALO_CASE(KK, NN, TXF, TXD)                                                       \
  if (K == KK && N == NN) {                                                             \
    if (dgrad) launch_halo<KK, NN, true, TXD>(a, s); else launch_halo<KK, NN, false, TXF>(a, s); \
    return true;                                                                        \
  }
    HALO_CASE(16, 16, 8, 8) HALO_CASE(16, 32, 8, 8) HALO_CASE(32, 32, 2, 2)
    HALO_CASE(32, 16, 4, 4)
#undef HALO_CASE
    // larger channel counts: the weight slices stream beside the resident block
#define HALO_S(KK, NN, TXX, DGR)                           \
  if (K == KK && N == NN && dgrad == DGR) {                \
    launch_halo_s<KK, NN, DGR, TXX>(a, s);                  \
    return true;                                            \
  }
    HALO_S(96, 32, 2, false) HALO_S(32, 96, 2, true) HALO_S(32, 64, 2, false)
    HALO_S(64, 32, 2, true) HALO_S(64, 64, 2, false) HALO_S(64, 64, 2, true)
    HALO_S(64, 128, 2, false) HALO_S(128, 64, 1, true) HALO_S(128, 128, 1, false)
    HALO_S(128, 128, 1, true) HALO_S(64, 192, 1, true)
#undef HALO_S
    if (!dgrad && K == 48 && N == 16) {
      launch_halo<48, 16, false, 2>(a, s);
      return true;
    }
    if (dgrad && K == 16 && N == 48) {
      launch_halo<16, 48, true, 4>(a, s);
      return true;
    }
  }
#define TC_CASE(KK, NN)                                              \
  if (K == KK && N == NN) {                                          \
    if (dgrad) launch_tc<KK, NN, true>(a, s); else launch_tc<KK, NN, false>(a, s); \
    return true;                                                     \
  }
  TC_CASE(16, 16) TC_CASE(16, 32) TC_CASE(32, 32) TC_CASE(32, 64) TC_CASE(64, 64)
  TC_CASE(64, 128) TC_CASE(128, 128) TC_CASE(192, 64) TC_CASE(96, 32) TC_CASE(48, 16)
  TC_CASE(32, 16) TC_CASE(64, 32) TC_CASE(128, 64) TC_CASE(64, 192) TC_CASE(32, 96)
  TC_CASE(16, 48)
#undef TC_CASE
  return false;
}

// (Cin, Cout) pairs of the network's weight gradients
bool nn_tc_wgrad_supported(int Cin, int Cout) {
  static const int p[][2] = {{16, 16}, {16, 32}, {32, 32}, {32, 64}, {64, 64},
                             {64, 128}, {128, 128}, {192, 64}, {96, 32}, {48, 16}};
  for (auto& q : p)
    if (q[0] == Cin && q[1] == Cout) return true;
  return false;
}

// the pairs with a resident-block kernel (launch_wgrad_halo below), whose partials are
// one per CTA
static bool wgrad_halo_pair(int Cin, int Cout) {
  return (Cout == 16 && (Cin == 16 || Cin == 48)) ||
         (Cout == 32 && (Cin == 16 || Cin == 32 || Cin == 96));
}

// (counting a partial per CTA for every pair took 128 -> 128 to 269 MB, above what a
// conv3d call's kept scratch may hold, and so to an allocation per call: 0.73 ms for the three ops on 8^3, now 0.32)
long long nn_tc_wgrad_scratch(int Cin, int Cout) {
  const int nt = (27 + TC_M / Cout - 1) / (TC_M / Cout), tap = WG_CTAS / nt;
  const int parts = wgrad_halo_pair(Cin, Cout) ? std::max(WG_HALO_CTAS, tap) : tap;
  return (long long)parts * 27 * Cin * Cout;
}

bool nn_tc_wgrad(TView x, int Cin, TView g, int Cout, float* dW, float* db, float* partials,
                 int B, int lgD, int* err, cudaStream_t s) {
  const long long Mtot = (long long)B << (3 * lgD);
  int S = 0;
  // up to 32 output channels on grids that hold the 16 x 8 blocks: resident
  // blocks (on 4 x 64^3: 16 -> 16 109 us, per tap 279; 48 -> 16 217, 513; smaller grids
  // and 64 and more output channels, whose slices leave no room for the three dx, per
  // tap)
  if (lgD >= 4 && wgrad_halo_pair(Cin, Cout)) {
    if (Cin == 16 && Cout == 16)
      launch_wgrad_halo<16, 16, 2, 9>(x, g, B, lgD, partials, err, &S, s);
    else if (Cin == 48 && Cout == 16)
      launch_wgrad_halo<48, 16, 1, 9>(x, g, B, lgD, partials, err, &S, s);
    else if (Cin == 16 && Cout == 32)
      launch_wgrad_halo<16, 32, 2, 9>(x, g, B, lgD, partials, err, &S, s);
    else if (Cin == 32 && Cout == 32)
      launch_wgrad_halo<32, 32, 1, 9>(x, g, B, lgD, partials, err, &S, s);
    else
      launch_wgrad_halo<96, 32, 1, 3>(x, g, B, lgD, partials, err, &S, s);
    nn_wgrad_finish(partials, S, Cin, Cout, dW, g, db, Mtot, s);
    return true;
  }
#define WG_CASE(CI, CO)                                                  \
  if (Cin == CI && Cout == CO) {                                         \
    launch_wgrad<CI, CO>(x, g, lgD, Mtot, partials, err, &S, s);         \
  } else
  WG_CASE(16, 16) WG_CASE(16, 32) WG_CASE(32, 32) WG_CASE(32, 64) WG_CASE(64, 64)
  WG_CASE(64, 128) WG_CASE(128, 128) WG_CASE(192, 64) WG_CASE(96, 32) WG_CASE(48, 16)
  return false;
#undef WG_CASE
  nn_wgrad_finish(partials, S, Cin, Cout, dW, g, db, Mtot, s);
  return true;
}

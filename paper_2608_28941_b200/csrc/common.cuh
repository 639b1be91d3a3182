// Shared device helpers: control block, bounded waits, TMA / mbarrier wrappers,
// the 128-byte-swizzle address map and the m16n8k8 tensor-core wrappers.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/rrf.h"

namespace rrf {

// Device-resident loop state of Algorithm 2 (lines 1, 4, 5, 9, 10).  Written by the
// init and stop kernels; every other kernel of a block step only reads `done`.
struct Ctrl {
  int done;        // 1 once the while-condition of Algorithm 2 line 5 (or the rank cap) is false
  int status;      // rrf_status_t, sticky for errors
  int steps;       // block steps completed (the paper's i)
  int k;           // steps * b
  unsigned bar;    // arrival counter of the panel kernel's grid barrier
  int panel_path;  // how the last panel of the column kernels was factored (rrf_panel_path)
  int pad[2];
  double normA2;   // ||A||_F^2
  double sigma2;   // squared absolute tolerance
  double E_sub;    // Algorithm 2 line 9
  double E_dir;    // ||W[r0+b:, :]||_F^2
  double E_prev;   // stopping quantity after the previous pass, and the ratio of the two before that:
  double r_prev;   // the history the sampling predictor extrapolates (negative: no ratio yet)
  int fused_samples;   // passes whose update also sampled a later panel
  int extra_samples;   // panels sampled by the separate kernel because the predictor had skipped them
  int n_est;           // sampled stopping rules: panels whose estimate was evaluated
  int pad2;
  double E_est;        // sampled stopping rules: the last estimate
};
static_assert(sizeof(Ctrl) <= 256, "the control block has 256 bytes of workspace");

// ~1 s at 2 GHz: every spin in this library gives up after this many SM clocks.
constexpr long long kWaitLimitClocks = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- programmatic dependent launch
// The kernels of a pass follow one another on one stream.  A kernel launched as a programmatic dependent is put on the
// SMs while the one before it drains and waits here, before its first access to global memory, until that one has
// completed and its writes are visible.  Launched the ordinary way both calls do nothing.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------- mbarrier / TMA

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// Bounded wait.  Returns false (and records RRF_ERR_TIMEOUT) when the phase never completes.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, Ctrl* ctrl) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kWaitLimitClocks) {
      atomicExch(&ctrl->status, (int)RRF_ERR_TIMEOUT);
      atomicExch(&ctrl->done, 1);          // kernels already enqueued behind this one return at once
      return false;
    }
  }
  return true;
}
// 2-D tiled TMA load: box at element coordinates (x = innermost, y) -> shared memory.
// x * sizeof(element) must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// Byte offset inside a 1024-byte-aligned shared-memory tile written by a TMA box with
// CU_TENSOR_MAP_SWIZZLE_128B: 16-byte chunk index (address bits 4..6) is XORed with the
// 128-byte line index (bits 7..9).
__device__ __forceinline__ uint32_t swz128(uint32_t off) { return off ^ (((off >> 7) & 7u) << 4); }

// ---------------------------------------------------------------- tensor-core wrappers
// One logical m16n8k8 product C += A * B on the fragment layout shared by the f64 and
// tf32 shapes (g = lane / 4, t = lane % 4):
//   a0:(g, t) a1:(g+8, t) a2:(g, t+4) a3:(g+8, t+4);  b0:(k=t, n=g) b1:(k=t+4, n=g);
//   c0:(g, 2t) c1:(g, 2t+1) c2:(g+8, 2t) c3:(g+8, 2t+1).

__device__ __forceinline__ void mma16x8x8(double (&c)[4], const double (&a)[4], const double (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

// x = hi + lo in two TF32 numbers, both rounded to nearest, ties away from zero, by integer operations (the bits of
// cvt.rna.tf32.f32 for every number, at half its cost: 2.1 against 4.1 cycles a warp).  The 13 bits that the tensor core
// does not read are cut off in hi, whose exact remainder lo is, and left in lo.  The NaN that GPU arithmetic produces
// (0x7fffffff) wraps to a number in either rounding, and an infinity has a NaN for its remainder d: 0 d is NaN for both
// and adds nothing to any other lo, so what is not finite in x is in every product that takes the pair.  It stands in the
// place of the other mask (a run of 4096 x 11008: 774 -> 785 us against the split that loses them; as a sixth operation,
// beside the mask, 823).
__device__ __forceinline__ void split_tf32(float x, float& hi, float& lo) {
  hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
  const float d = x - hi;
  lo = fmaf(d, 0.f, __uint_as_float(__float_as_uint(d) + 0x1000u));
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  float h, l;
  split_tf32(x, h, l);
  hi = __float_as_uint(h);
  lo = __float_as_uint(l);
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// fp32 product by the 3xTF32 split: x = hi + lo with hi = tf32(x), lo = tf32(x - hi);
// D = A_lo*B_hi + A_hi*B_lo + A_hi*B_hi (small terms first; A_lo*B_lo is below fp32 round-off),
// then C += D with an ordinary round-to-nearest add: the tensor core's own accumulation does not
// round to nearest, so only the eight products of one k-step are summed inside it.
__device__ __forceinline__ void mma16x8x8(float (&c)[4], const float (&a)[4], const float (&b)[2]) {
  uint32_t ah[4], al[4], bh[2], bl[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) split_tf32(a[i], ah[i], al[i]);
#pragma unroll
  for (int i = 0; i < 2; ++i) split_tf32(b[i], bh[i], bl[i]);
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  mma_tf32(d, al, bh);
  mma_tf32(d, ah, bl);
  mma_tf32(d, ah, bh);
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] += d[i];
}

// Operands prepared once and used by several products.  In double precision an operand is the value; in single
// precision it is the value split into two TF32 numbers, so that a fragment that feeds several m16n8k8 products
// is split once and not once per product.
template <typename T>
struct Op;
template <>
struct Op<double> {
  double v;
};
template <>
struct Op<float> {
  uint32_t hi, lo;
};
__device__ __forceinline__ Op<double> prep(double x) { return Op<double>{x}; }
__device__ __forceinline__ Op<float> prep(float x) {
  Op<float> o;
  split_tf32(x, o.hi, o.lo);
  return o;
}
__device__ __forceinline__ void mma_op(double (&c)[4], const Op<double>& a0, const Op<double>& a1, const Op<double>& a2,
                                       const Op<double>& a3, const Op<double>& b0, const Op<double>& b1) {
  const double a[4] = {a0.v, a1.v, a2.v, a3.v}, b[2] = {b0.v, b1.v};
  mma16x8x8(c, a, b);
}
// D = A_lo*B_hi + A_hi*B_lo + A_hi*B_hi inside the tensor core, then C += D rounded to nearest (see above)
__device__ __forceinline__ void mma_op(float (&c)[4], const Op<float>& a0, const Op<float>& a1, const Op<float>& a2,
                                       const Op<float>& a3, const Op<float>& b0, const Op<float>& b1) {
  const uint32_t ah[4] = {a0.hi, a1.hi, a2.hi, a3.hi}, al[4] = {a0.lo, a1.lo, a2.lo, a3.lo};
  const uint32_t bh[2] = {b0.hi, b1.hi}, bl[2] = {b0.lo, b1.lo};
  float d[4] = {0.f, 0.f, 0.f, 0.f};
  mma_tf32(d, al, bh);
  mma_tf32(d, ah, bl);
  mma_tf32(d, ah, bh);
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] += d[i];
}

// One k-step of a warp tile, MT x NT products.  In single precision the three products of an element depend on one
// another, so they are issued tile by tile across the whole step: a warp that took one tile's three at a time waited
// for each (62 cycles a tile and scheduler in the first sample of 4096 x 11008).
template <int MT, int NT>
__device__ __forceinline__ void mma_step(double (&acc)[MT][NT][4], const Op<double> (&a)[MT][4], const Op<double> (&b)[NT][2]) {
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) mma_op(acc[i][j], a[i][0], a[i][1], a[i][2], a[i][3], b[j][0], b[j][1]);
}
template <int MT, int NT>
__device__ __forceinline__ void mma_step(float (&acc)[MT][NT][4], const Op<float> (&a)[MT][4], const Op<float> (&b)[NT][2]) {
  float d[MT][NT][4];
#pragma unroll
  for (int term = 0; term < 3; ++term)
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        uint32_t ax[4], bx[2];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          ax[e] = term == 0 ? a[i][e].lo : a[i][e].hi;
          if (term == 0) d[i][j][e] = 0.f;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) bx[e] = term == 1 ? b[j][e].lo : b[j][e].hi;
        mma_tf32(d[i][j], ax, bx);
      }
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] += d[i][j][e];
}

// ---------------------------------------------------------------- small utilities

template <typename T>
struct VecLoad16;  // one 16-byte shared-memory load
template <>
struct VecLoad16<double> {
  static constexpr int N = 2;
  __device__ static __forceinline__ void ld(const unsigned char* p, double (&v)[2]) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  }
};
template <>
struct VecLoad16<float> {
  static constexpr int N = 4;
  __device__ static __forceinline__ void ld(const unsigned char* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Fixed-order block reduction of one double per thread (blockDim.x a multiple of 32, <= 1024).
// `scratch` holds at least 32 doubles.  The result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* scratch) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    r = lane < nw ? scratch[lane] : 0.0;
    r = warp_sum(r);
  }
  return r;
}

}  // namespace rrf

// Barriers and exchanges between the CTAs of a panel kernel: a grid-wide barrier, and the mbarrier / distributed shared
// memory forms used when the grid is one thread-block cluster.
#pragma once

#include "common.cuh"

namespace rrf {

constexpr int kPanelThreads = 512;
constexpr int kPanelMaxG = 160;   // most CTAs a panel grid may have (one per SM)
// doubles of shared memory the panel kernel needs besides the slab: w[b], p[2][b], pivot_row[b], scalars
__host__ __device__ constexpr int panel_extra_doubles(int b) { return 4 * b + 4; }

// Grid-wide barrier over a monotonically increasing arrival counter.  Needs all CTAs
// co-resident (cooperative launch).  Bounded: gives up after kWaitLimitClocks.
__device__ __forceinline__ bool grid_barrier(unsigned* ctr, unsigned target, Ctrl* ctrl,
                                             long long limit = kWaitLimitClocks) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    int ok = 1;
    const long long t0 = clock64();
    while (true) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
      if (v >= target) break;
      if (clock64() - t0 > limit) {
        atomicExch(&ctrl->status, (int)RRF_ERR_TIMEOUT);
        atomicExch(&ctrl->done, 1);        // kernels already enqueued behind this one return at once
        ok = 0;
        break;
      }
    }
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

// ---------------------------------------------------------------- thread-block cluster exchange
// A panel that fits the shared memory of at most 16 CTAs is factored by ONE cluster: the per-column sums
// travel through distributed shared memory (every CTA writes its partials straight into every peer's
// shared memory) and the barrier is an mbarrier per CTA on which every peer arrives - about 0.7 to 1 us per
// column against the 2.4 us of an all-to-all exchange through L2.
constexpr int kClusterMax = 16;
#ifdef RRF_TSQR_TRACE
__device__ unsigned long long g_pcl_trace[16];
#define PCL_STAMP(k) if (j == 8 && blockIdx.x == 0 && threadIdx.x == 0) g_pcl_trace[k] = (unsigned long long)clock64()
#else
#define PCL_STAMP(k)
#endif
constexpr int kRegRows = 256;       // rows of a slab in the register-resident column loop
// px [2][kClusterMax][2b], prx [2][b], ycol/vcol [kRegRows] each, prow [b], send buffers [2][2b]
__host__ __device__ constexpr int panel_cluster_doubles(int b) {
  return 2 * kClusterMax * 2 * b + 2 * b + 2 * kRegRows + b + 4 * b;
}
// One bulk copy from this CTA's shared memory into a peer's, which also counts its bytes on the peer's mbarrier:
// data and signal in one message.
__device__ __forceinline__ void cl_bulk_send(uint32_t dst_cluster, uint32_t src_cta, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_cluster), "r"(src_cta), "r"(bytes), "r"(bar_cluster)
               : "memory");
}

__device__ __forceinline__ void proxy_fence_smem_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank) {   // the same address in CTA `rank` of the cluster
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_st(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_arrive(uint32_t bar_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_addr) : "memory");
}
__device__ __forceinline__ uint32_t cl_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// the hardware barrier of the cluster (unbounded: used once, before any data-dependent exit)
__device__ __forceinline__ void cl_hw_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Barrier over the G CTAs of the cluster: every CTA arrives on every peer's mbarrier and waits, bounded, on its
// own.  Everything this CTA stored before it - into peers' shared memory or into global memory: a release at cluster
// scope covers both - is visible to the peers behind it.  `nx` counts the barriers passed (the phase parity).
__device__ __forceinline__ bool cluster_barrier(uint64_t* cbar, unsigned& nx, int G, Ctrl* ctrl) {
  __shared__ int cl_ok_s;
  __syncthreads();
  if ((int)threadIdx.x < G) cl_arrive(cl_map(smem_u32(cbar), threadIdx.x));
  if (threadIdx.x == 0) {
    int ok = 1;
    if (!cl_try_wait(cbar, nx & 1u)) {
      const long long t0 = clock64();
      while (!cl_try_wait(cbar, nx & 1u)) {
        if (clock64() - t0 > kWaitLimitClocks) {
          atomicExch(&ctrl->status, (int)RRF_ERR_TIMEOUT);
          atomicExch(&ctrl->done, 1);
          ok = 0;
          break;
        }
      }
    }
    cl_ok_s = ok;
  }
  ++nx;
  __syncthreads();
  return cl_ok_s != 0;
}

// Sums four per-lane values over the warp with 6 adds and 6 shuffles instead of 20: after the
// exchanges with lanes ^16 and ^8 every lane carries one of the four sums (number 2*bit4 + bit3 of
// its lane index), which three more butterfly steps complete.  Fixed order, so reproducible.
__device__ __forceinline__ double warp_sum4(const double (&v)[4], int lane) {
  const bool hi = lane & 16;
  double a0 = hi ? v[2] : v[0], a1 = hi ? v[3] : v[1];
  const double s0 = hi ? v[0] : v[2], s1 = hi ? v[1] : v[3];
  a0 += __shfl_xor_sync(0xffffffffu, s0, 16);
  a1 += __shfl_xor_sync(0xffffffffu, s1, 16);
  const bool mid = lane & 8;
  double k = mid ? a1 : a0;
  const double snd = mid ? a0 : a1;
  k += __shfl_xor_sync(0xffffffffu, snd, 8);
  k += __shfl_xor_sync(0xffffffffu, k, 4);
  k += __shfl_xor_sync(0xffffffffu, k, 2);
  k += __shfl_xor_sync(0xffffffffu, k, 1);
  return k;
}

}  // namespace rrf

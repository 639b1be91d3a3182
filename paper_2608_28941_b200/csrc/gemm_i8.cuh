// Double-precision products on the INTEGER tensor cores of sm_100a (tcgen05.mma kind::i8), by splitting.
//
// A double operand is written as an integer of seven balanced base-256 digits times a power of two common to its row
// (or column), x = 2^(e-55) sum_i d_i 256^(6-i), -128 <= d_i <= 127: the bytes of the 56-bit integer plus 0x80 in every
// byte.  Products of digits are summed EXACTLY in 32-bit integers, all pairs with the same i + j in one accumulator
// ("group"), and the groups are put together in 64-bit integers and double precision when an accumulator is read.  (Ootomo,
// Ozaki, Yokota, "DGEMM on integer matrix multiplication unit", 2024, after Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication", 2012.)  What is lost is the last half bit of an operand, 2^-56 of the largest
// entry it shares its scale with, and the pairs whose group is left out.
//
// Error against exact products, relative to the result: V^T W 2.3e-16 to 2.7e-16 for 1000 to 5000 rows (chains of multiply-adds
// 1e-15 to 3e-15), W Omega 2.6e-16 to 3.2e-16, the update 5e-17 to 8e-17 of W (chain 8e-17 to 1.1e-16).
//
// Why: mma.sync f64 runs at 128 flop a clock and SM (37 TFLOP/s), kind::i8 at 16384; the 28 (34) pairs of seven (eight)
// groups make 570 (470) flop of double precision a clock, and the three products of a block step are then bound by the
// bytes of W.  One instruction multiplies digit i of the 128-row operand with up to four digits of the other, which lie one
// after the other in shared memory and in the accumulator: group g is columns g N ... of tensor memory.
//
// Operand images.  Every operand reaches the tensor core K-contiguous, 32 contraction indices = one 32-byte line, in the
// 32-byte swizzle: byte k of line r at r 32 + (((k >> 4) ^ (r >> 2 & 1)) << 4) + (k & 15).  The small operands (V, Z,
// Omega) are split once by small kernels that write these images to global memory; an untiled bulk copy brings them in.
// W is split by the warps of the product that reads it.
//
// Scales.  oz_exp() of the largest magnitude: W per column for V^T W, per row for W Omega (oz_update_kernel leaves both
// maxima behind); Z per column; V per row for the update; V and Omega per column and chunk of 1024 contraction indices
// for the other two (the accumulators are read after every chunk; the b rows of V's unit triangle are a chunk of their own:
// with them the rest of V would lose the four bits that lie between 1 and the size of its entries).
// A NaN or an infinity makes the scale of its row or column a NaN, and with it every result it takes part in.
#pragma once

#include "gemm_tc_vtw.cuh"
#include "i8_split.cuh"

namespace rrf {

// chunk (= scale) of the small operand that step q of the contraction belongs to; `first` steps make one of their own
__host__ __device__ __forceinline__ int oz_chunk_of(int q, int first) {
  return q < first ? 0 : (first > 0 ? 1 : 0) + (q - first) / kOzChunk;
}

__device__ __forceinline__ uint64_t oz_desc(uint32_t addr) {       // K-contiguous, 32-byte swizzle, groups of eight lines 256 bytes apart
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(256u >> 4) << 32) | (1ull << 46) | (6ull << 61);
}
__host__ __device__ constexpr uint32_t oz_idesc(int M, int N) {    // signed bytes, 32-bit integer accumulator
  return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// The warp that issues walks its loop as a whole, and only the instructions themselves are one lane's (`lead`): descriptors and
// addresses then stay in uniform registers.  In a branch of one lane, with a barrier each for the two operands, a step took
// that thread 1100 clocks of its own (753 for the ten instructions, 430 for two waits) beside the 920 of its products.
__device__ __forceinline__ uint32_t oz_lead() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r;
}
__device__ __forceinline__ void oz_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate, uint32_t lead) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(lead)
      : "memory");
}
__device__ __forceinline__ void oz_commit(uint64_t* bar, uint32_t lead) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "setp.ne.b32 e, %1, 0;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(smem_u32(bar)), "r"(lead)
      : "memory");
}
// One step: digits of the 128-line operand at a0, those of the other (N lines each) at b0, all pairs with i + j < NG.
template <int N, int NG>
__device__ __forceinline__ void oz_step(uint32_t tmem, uint32_t a0, uint32_t b0, bool fresh, uint32_t lead) {
  constexpr int W = 256 / N;                             // digits side by side in one instruction
#pragma unroll
  for (int i = 0; i < kOzS; ++i) {
    const uint64_t a = oz_desc(a0 + i * 4096);
    const int nj = NG - i < kOzS ? NG - i : kOzS;
#pragma unroll
    for (int j = 0; j < nj;) {
      int w = nj - j < W ? nj - j : W;
      // a group's first product in a fresh accumulator overwrites: groups 0 ... 6 with i = 0, group 7 with i = 1, j = 6
      if (NG > kOzS && i == 1 && j + w == kOzS && w > 1) w -= 1;
      const bool over = fresh && (i == 0 || (NG > kOzS && i == 1 && j == kOzS - 1));
      oz_mma(tmem + (i + j) * N, a, oz_desc(b0 + j * N * 32), oz_idesc(128, w * N), over ? 0u : 1u, lead);
      j += w;
    }
  }
}
// untiled bulk copy, 16-byte aligned
__device__ __forceinline__ void oz_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// columns c ... c + 7 of eight groups N columns apart, this thread's lane
template <int N>
__device__ __forceinline__ void oz_ld8(uint32_t t, int (&r)[8][8]) {
  // the loads are asynchronous: they and the wait sit in one statement (see tmem_ld16)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%65];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%66];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%67];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32,%33,%34,%35,%36,%37,%38,%39}, [%68];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%40,%41,%42,%43,%44,%45,%46,%47}, [%69];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%48,%49,%50,%51,%52,%53,%54,%55}, [%70];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%56,%57,%58,%59,%60,%61,%62,%63}, [%71];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0][0]), "=r"(r[0][1]), "=r"(r[0][2]), "=r"(r[0][3]), "=r"(r[0][4]), "=r"(r[0][5]), "=r"(r[0][6]), "=r"(r[0][7]),
          "=r"(r[1][0]), "=r"(r[1][1]), "=r"(r[1][2]), "=r"(r[1][3]), "=r"(r[1][4]), "=r"(r[1][5]), "=r"(r[1][6]), "=r"(r[1][7]),
          "=r"(r[2][0]), "=r"(r[2][1]), "=r"(r[2][2]), "=r"(r[2][3]), "=r"(r[2][4]), "=r"(r[2][5]), "=r"(r[2][6]), "=r"(r[2][7]),
          "=r"(r[3][0]), "=r"(r[3][1]), "=r"(r[3][2]), "=r"(r[3][3]), "=r"(r[3][4]), "=r"(r[3][5]), "=r"(r[3][6]), "=r"(r[3][7]),
          "=r"(r[4][0]), "=r"(r[4][1]), "=r"(r[4][2]), "=r"(r[4][3]), "=r"(r[4][4]), "=r"(r[4][5]), "=r"(r[4][6]), "=r"(r[4][7]),
          "=r"(r[5][0]), "=r"(r[5][1]), "=r"(r[5][2]), "=r"(r[5][3]), "=r"(r[5][4]), "=r"(r[5][5]), "=r"(r[5][6]), "=r"(r[5][7]),
          "=r"(r[6][0]), "=r"(r[6][1]), "=r"(r[6][2]), "=r"(r[6][3]), "=r"(r[6][4]), "=r"(r[6][5]), "=r"(r[6][6]), "=r"(r[6][7]),
          "=r"(r[7][0]), "=r"(r[7][1]), "=r"(r[7][2]), "=r"(r[7][3]), "=r"(r[7][4]), "=r"(r[7][5]), "=r"(r[7][6]), "=r"(r[7][7])
        : "r"(t), "r"(t + N), "r"(t + 2 * N), "r"(t + 3 * N), "r"(t + 4 * N), "r"(t + 5 * N), "r"(t + 6 * N), "r"(t + 7 * N)
        : "memory");
}
// The eight groups of one entry put together.  A group is below 2^14 * 7 * 32 kOzChunk steps < 2^27, those that the two integers
// begin with below 2^24.1 and 2^26.4, so both are below 2^51 and their conversion by the bits of 1.5 2^52 is exact.  Value: the
// result times 2^(ea - kOzOut) 2^(eb - kOzOut).
constexpr int kOzOut = 19;       // 2^-14 of the digits' places and the first integer's 2^-24, half to either scale
__device__ __forceinline__ long long oz_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
template <bool SMALL = false>      // SMALL: groups below 2^23, so that two of them fit one 32-bit integer
__device__ __forceinline__ double oz_join(const int (&r)[8][8], int e) {
  const double m = 6755399441055744.0;
  const long long c = 0x4338000000000000ll;
  long long hi, lo;
  if constexpr (SMALL) {
    hi = oz_mad(r[0][e] * 256 + r[1][e], 65536, oz_mad(r[2][e] * 256 + r[3][e], 1, c));
    lo = oz_mad(r[4][e] * 256 + r[5][e], 65536, oz_mad(r[6][e] * 256 + r[7][e], 1, c));
  } else {
    hi = oz_mad(r[0][e], 16777216, oz_mad(r[1][e], 65536, oz_mad(r[2][e], 256, oz_mad(r[3][e], 1, c))));
    lo = oz_mad(r[4][e], 16777216, oz_mad(r[5][e], 65536, oz_mad(r[6][e], 256, oz_mad(r[7][e], 1, c))));
  }
  return fma(__longlong_as_double(lo) - m, 0x1p-32, __longlong_as_double(hi) - m);
}

// ------------------------------------------------------------------------------------------
// Z = V^T C (TR: the contraction runs over the rows of C, a line of the 128-line operand is a column of C) and
// Y = C Omega (over the columns, a line is a row).  128 lines x 64 contraction indices a tile, stream-K ranges and partial
// slots as vtw_sk_kernel: tile L = c KT + kt, slot p + c holds [B][128] (Z) or [128][B] (Y) of line tile c.  Wider blocks
// than 64 columns are shared by B / NB CTAs, which take the same tiles side by side, so that W comes from L2 for all but
// one of them.
// Per step of 32 indices: W's 32 KB by TMA, the images of the small operand (7 N 32 bytes) by a bulk copy, twelve warps in
// three groups that take the steps in turn and write the digits of their 4096 numbers (28 KB), one warp that issues ten
// instructions.  Shared memory carries about 200 KB a step, 1590 clocks; W's bytes take 1465 at the copy rate shared by 148
// SMs, the tensor core 920.  Measured (8192 x 8192, 148 SMs): N = 64 140 us = 2170 clocks a step (mma.sync f64: 257; without the
// split 103, without the products 94: the two share shared memory and the issue slots), N = 32 115, two CTAs a tile for b = 128
// 249.  Sixteen warps in two groups with four places of W: 158.
// ------------------------------------------------------------------------------------------
constexpr int kOzGroups = 3;            // groups of four warps that split; a group has its own place in the rings of W and of digits
constexpr int kOzConv = 4 * kOzGroups;
constexpr int kOzThreads = (kOzConv + 3) * 32;
template <int NB>
struct OzCfg {
  static constexpr int W_BYTES = 128 * kOzK * 8, B_BYTES = kOzS * NB * 32, A_BYTES = kOzS * 128 * 32;
  static constexpr int RW = kOzGroups, RA = kOzGroups;
  static constexpr int SMEM = RW * W_BYTES + RA * (A_BYTES + B_BYTES) + 1024;
  static constexpr int COLS = 8 * NB;
  static_assert(SMEM + 1024 <= 232448 && (COLS == 256 || COLS == 512), "shared and tensor memory");
};
template <int NB, bool TR>
__global__ void __launch_bounds__(kOzThreads, 1)
    oz_gemm_kernel(const __grid_constant__ CUtensorMap tmC,   // C; TR: box [32][128], no swizzle; else box [128][16], 128-byte swizzle
                   const unsigned char* __restrict__ img,     // small operand: [step][B / NB][7][NB lines x 32]
                   const int* __restrict__ eimg,              // its scales: [chunk][B]
                   const uint32_t* __restrict__ mag,          // largest magnitude of every line of C (high words)
                   double* __restrict__ part, int B, int r0, int lines, int first, int KT, int total, int tpc, Ctrl* ctrl) {
  pdl_wait();
  pdl_trigger();
  if (*reinterpret_cast<volatile int*>(&ctrl->done)) return;
  using Cfg = OzCfg<NB>;
  constexpr int RW = Cfg::RW, RA = Cfg::RA;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ringW = align1024(smem_raw);
  unsigned char* ringA = ringW + RW * Cfg::W_BYTES;
  unsigned char* ringB = ringA + Cfg::RA * Cfg::A_BYTES;
  __shared__ uint64_t wfull[RW], wempty[RW], full[RA], empty[RA], acc_full, acc_empty;
  __shared__ uint32_t tmem_slot;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nh = B / NB, p = blockIdx.x / nh, h = blockIdx.x - p * nh;
  const int L0 = p * tpc, ntile = min(total, L0 + tpc) - L0, nsub = 2 * ntile;

  if (tid == 0) {
    for (int s = 0; s < RW; ++s) {
      mbar_init(&wfull[s], 1);
      mbar_init(&wempty[s], 4);
    }
    for (int s = 0; s < RA; ++s) {
      mbar_init(&full[s], 4 + 1);        // the group's four warps and the copy of the small operand
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, kOzConv);
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == 0) tmem_alloc(&tmem_slot, Cfg::COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);

  // line tile c and step k inside its contraction of this CTA's step q, and the chunk that k belongs to
  struct Walk {
    int c, k, ch, in_ch, K2, first;
    __device__ __forceinline__ Walk(int L0, int KT, int first_) : K2(2 * KT), first(first_) {
      c = L0 / KT;
      k = 2 * (L0 - c * KT);
      start();
    }
    __device__ __forceinline__ void start() {
      ch = oz_chunk_of(k, first);
      in_ch = k < first ? first - k : kOzChunk - (k - first) % kOzChunk;       // steps left in the chunk
    }
    __device__ __forceinline__ bool tile_ends() const { return k == K2 - 1; }
    __device__ __forceinline__ bool chunk_ends() const { return in_ch == 1; }
    __device__ __forceinline__ void next() {
      if (++k == K2) {
        k = 0;
        ++c;
        start();
      } else if (--in_ch == 0) {
        ++ch;
        in_ch = kOzChunk;
      }
    }
  };
  Walk at(L0, KT, first);
  // the accumulators are read after step q: the end of a line tile or of this CTA's range, or of a chunk
  auto last_after = [&](int q) { return q == nsub - 1 || at.tile_ends(); };
  auto drain_after = [&](int q) { return last_after(q) || at.chunk_ends(); };

  if (warp == kOzConv) {
    // ---------------------------------------------------------------- TMA producer: W
    if (lane == 0) {
      for (int q = 0; q < nsub; ++q, at.next()) {
        const int s = q % RW;
        if (q >= RW && !mbar_wait(&wempty[s], ((q / RW) - 1) & 1, ctrl)) break;
        const int c = at.c, k0 = at.k * kOzK;
        unsigned char* dst = ringW + s * Cfg::W_BYTES;
        mbar_expect_tx(&wfull[s], Cfg::W_BYTES);
        if (TR) {
          tma_load_2d(dst, &tmC, c * 128, r0 + k0, &wfull[s]);
        } else {
          tma_load_2d(dst, &tmC, k0, r0 + c * 128, &wfull[s]);
          tma_load_2d(dst + Cfg::W_BYTES / 2, &tmC, k0 + 16, r0 + c * 128, &wfull[s]);
        }
      }
    }
  } else if (warp == kOzConv + 1) {
    // ---------------------------------------------------------------- bulk copies: images of the small operand
    if (lane == 0) {
      for (int q = 0; q < nsub; ++q, at.next()) {
        const int s = q % RA;
        if (q >= RA && !mbar_wait(&empty[s], ((q / RA) - 1) & 1, ctrl)) break;
        mbar_expect_tx(&full[s], Cfg::B_BYTES);
        oz_bulk_load(smem_u32(ringB + s * Cfg::B_BYTES), img + (size_t)(at.k * nh + h) * Cfg::B_BYTES, Cfg::B_BYTES, &full[s]);
      }
    }
  } else if (warp == kOzConv + 2) {
    // ---------------------------------------------------------------- MMA issuer
    const uint32_t lead = oz_lead(), a0 = smem_u32(ringA), b0 = smem_u32(ringB);
    bool fresh = true;
    int ndrain = 0, s = 0;
    uint32_t ph = 0;
    for (int q = 0; q < nsub; ++q, at.next()) {
      if (!mbar_wait(&full[s], ph, ctrl)) break;
      if (fresh && ndrain > 0 && !mbar_wait(&acc_empty, (ndrain - 1) & 1, ctrl)) break;
      tc_fence_after();
      if (TR && at.k < first) oz_step<NB, 8>(tmem, a0 + s * Cfg::A_BYTES, b0 + s * Cfg::B_BYTES, fresh, lead);
      else oz_step<NB, 7>(tmem, a0 + s * Cfg::A_BYTES, b0 + s * Cfg::B_BYTES, fresh, lead);
      fresh = false;
      oz_commit(&empty[s], lead);
      if (drain_after(q)) {
        oz_commit(&acc_full, lead);
        fresh = true;
        ++ndrain;
      }
      if (++s == RA) { s = 0; ph ^= 1u; }
    }
  } else {
    // ---------------------------------------------------------------- split and drain
    // line 32 (warp % 4) + lane of the tile, the steps that are warp / 4 modulo the number of groups
    const int quad = warp & 3, grp = warp >> 2, line = quad * 32 + lane;
    const uint32_t tlane = tmem + ((uint32_t)(quad * 32) << 16);
    int ndrain = 0, cur_c = -1;
    double sc = 0.0;
    bool ok = true;
    // Accumulators of line tile c, chunk ch -> this CTA's slot, eight columns of the result at a time: pieces grp, grp + 3,
    // ...  The slot itself is added to (a thread its own numbers, in the order of the chunks), and the pieces are a loop: with
    // the sums in registers and the pieces unrolled, code that runs once in thirty steps came in from L2 each time (12 000
    // clocks a drain).
    auto drain = [&](int c, int ch, bool add) {
      const int l = c * 128 + line;
      // scales first: their loads are under way while the products end
      const double fa = oz_pow2(oz_exp(l < lines ? mag[l] : 0u) - kOzOut);
      double* out = part + (size_t)(p + c) * (size_t)(B * 128) + (TR ? (size_t)(h * NB) * 128 + line : (size_t)line * B + h * NB);
      const int* eb = eimg + ch * B + h * NB;
      bool waited = false;
#pragma unroll 1
      for (int j = grp * 8; j < NB; j += kOzGroups * 8) {
        double v[8];
        const int e8 = eb[j + (lane & 7)];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.0;
        if (add) {
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            if (TR) {
              v[e] = out[(size_t)(j + e) * 128];
              v[e + 1] = out[(size_t)(j + e + 1) * 128];
            } else {
              const double2 o = *reinterpret_cast<const double2*>(out + j + e);
              v[e] = o.x;
              v[e + 1] = o.y;
            }
          }
        }
        if (!waited) {
          if (!mbar_wait(&acc_full, ndrain & 1, ctrl)) { ok = false; return; }
          waited = true;
          tc_fence_after();
        }
        int r[8][8];
        oz_ld8<NB>(tlane + j, r);
        if (!(TR && ch == 0)) {          // the eighth group is there for V's unit triangle only
#pragma unroll
          for (int e = 0; e < 8; ++e) r[7][e] = 0;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e)
          v[e] = fma(oz_join(r, e) * fa, oz_pow2(__shfl_sync(0xffffffffu, e8, e) - kOzOut), v[e]);
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          if (TR) {
            out[(size_t)(j + e) * 128] = v[e];
            out[(size_t)(j + e + 1) * 128] = v[e + 1];
          } else {
            store2(out + j + e, v[e], v[e + 1]);
          }
        }
      }
      ++ndrain;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty);
    };
    // A group that has split the last step before a drain takes part in it at once; the others split their next step
    // first, so that the tensor core finds two steps ready behind the drain.  At most two are owed.
    int owed = 0, due0 = 0, c0 = 0, ch0 = 0, due1 = 0, c1 = 0, ch1 = 0;
    bool add0 = false, add1 = false, open = true;      // open: this line tile's slot holds nothing yet
    auto pay = [&](int q) {
      while (ok && owed > 0 && due0 <= q) {
        drain(c0, ch0, add0);
        --owed;
        due0 = due1; c0 = c1; ch0 = ch1; add0 = add1;
      }
    };
    int turn = 0;                      // q modulo the number of groups
    for (int q = 0; q < nsub && ok; ++q, at.next()) {
      const bool mine = turn == grp;
      if (mine) {
        if (at.c != cur_c) {
          const int l = at.c * 128 + line;
          sc = oz_scale(oz_exp(l < lines ? mag[l] : 0u));
          cur_c = at.c;
        }
        const int use = q / kOzGroups;       // how often this group's places were used before
        if (!mbar_wait(&wfull[grp], use & 1, ctrl)) break;
        if (use > 0 && !mbar_wait(&empty[grp], (use - 1) & 1, ctrl)) break;
        const unsigned char* w = ringW + grp * Cfg::W_BYTES;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          uint32_t word[kOzS][4];
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) {
            double x[4];
            if (TR) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                x[e] = *reinterpret_cast<const double*>(w + (half * 16 + k4 * 4 + e) * 1024 + line * 8);
            } else {
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const double2 v = *reinterpret_cast<const double2*>(w + half * (Cfg::W_BYTES / 2) + line * 128 +
                                                                    (((uint32_t)(k4 * 2 + e) ^ (uint32_t)(line & 7)) << 4));
                x[2 * e] = v.x;
                x[2 * e + 1] = v.y;
              }
            }
            uint32_t d[kOzS];
            oz_words(x, sc, d);
#pragma unroll
            for (int i = 0; i < kOzS; ++i) word[i][k4] = d[i];
          }
          unsigned char* dst = ringA + grp * Cfg::A_BYTES + oz_at(line, half * 16);
#pragma unroll
          for (int i = 0; i < kOzS; ++i)
            *reinterpret_cast<uint4*>(dst + i * 4096) = make_uint4(word[i][0], word[i][1], word[i][2], word[i][3]);
        }
        proxy_fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&full[grp]);
          mbar_arrive(&wempty[grp]);     // every number read from the stage has gone into the stores above
        }
        pay(q);
      }
      if (drain_after(q)) {
        const int due = mine ? q : q + 1 + (grp - turn - 1 + kOzGroups) % kOzGroups;
        if (owed == 0) { due0 = due; c0 = at.c; ch0 = at.ch; add0 = !open; }
        else { due1 = due; c1 = at.c; ch1 = at.ch; add1 = !open; }
        ++owed;
        open = last_after(q);
        if (mine) pay(q);
      }
      turn = turn + 1 == kOzGroups ? 0 : turn + 1;
    }
    pay(nsub + kOzGroups);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, Cfg::COLS);
}

// ------------------------------------------------------------------------------------------
// C[r0 ..., :] -= V Z, with the norms of line 9 and the largest magnitudes of the rows and columns of what is left (those
// the next two products scale by).  Tiles of 128 rows x 32 columns, numbered along a row slab, stream-K ranges as
// upd_sk_kernel.  The digits of V[slab] stay in shared memory for a slab; a tile's digits of Z and its part of W go through
// rings.  Eight groups: with K = B this small the pairs of the eighth are what would be seen.  Tensor memory holds the
// accumulators of two tiles (8 x 32 columns each); two groups of eight warps take the tiles in turn (warp w: rows
// 32 (w % 4) ..., 16 columns = one TMA box), read them, put W's new values where the old ones stood and store them by TMA.
// A tile's bytes of W take 2930 clocks at the copy rate shared by 148 SMs, its products 1140 (B = 64; 2280 for 128).  Measured
// (8192 x 8192): b = 32 197 us (5.5 TB/s), 64 218, 128 349; upd_sk_kernel with its sample 565 for b = 64.
// ------------------------------------------------------------------------------------------
constexpr int kOzuEpi = 16;
constexpr int kOzuThreads = (kOzuEpi + 3) * 32;
template <int B>
struct OzuCfg {
  static constexpr int KS = B / 32, V_BYTES = KS * kOzS * 4096, Z_BYTES = KS * kOzS * kOzBN * 32;
  static constexpr int BOX = 128 * 128, W_BYTES = 2 * BOX;
  static constexpr int NZ = B >= 128 ? 1 : 2;
  static constexpr int NW = B >= 128 ? 2 : 4;      // even: a place is always the same group's (see the waits by parity)
  static constexpr int SMEM = V_BYTES + NZ * Z_BYTES + NW * W_BYTES + 1024;
  static_assert(SMEM + 1024 <= 232448 && NW % 2 == 0, "shared memory");
};
template <int B>
__global__ void __launch_bounds__(kOzuThreads, 1)
    oz_update_kernel(const __grid_constant__ CUtensorMap tmC,    // C as read, box [128][16]
                     const __grid_constant__ CUtensorMap tmCs,   // C as written [r0 + rows][ncols], box [32][16]
                     const __grid_constant__ CUtensorMap tmTs,   // rows of B being formed [top_rows][ncols], box [32][16]
                     const unsigned char* __restrict__ vimg, const int* __restrict__ ev,   // [slab][B / 32][7][128 x 32], [row]
                     const unsigned char* __restrict__ zimg, const int* __restrict__ ez,   // [tile][B / 32][7][32 x 32], [column]
                     int r0, int rows, int ncols, int top_rows, double* __restrict__ norm_part,
                     uint32_t* __restrict__ colmag, uint32_t* __restrict__ rowmag,         // of rows top_rows ...; rowmag[0] is row top_rows
                     int NC, int total, int tpc, Ctrl* ctrl) {
  pdl_wait();
  pdl_trigger();
  if (*reinterpret_cast<volatile int*>(&ctrl->done)) return;
  using Cfg = OzuCfg<B>;
  constexpr int NW = Cfg::NW, NZ = Cfg::NZ, KS = Cfg::KS, BN = kOzBN, D = 8 * BN;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ringW = align1024(smem_raw);
  unsigned char* sV = ringW + NW * Cfg::W_BYTES;
  unsigned char* ringZ = sV + Cfg::V_BYTES;
  __shared__ uint64_t wfull[NW], wempty[NW], zfull[NZ], zempty[NZ], vfull, vempty, d_full[2], d_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ double red[64];
  __shared__ __align__(16) double scale_s[kOzuEpi][16];      // a warp's own: scales of its tile's columns

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p = blockIdx.x;
  const int L0 = p * tpc, ntile = min(total, L0 + tpc) - L0;

  if (tid == 0) {
    for (int s = 0; s < NW; ++s) {
      mbar_init(&wfull[s], 1);
      mbar_init(&wempty[s], kOzuEpi / 2);
    }
    for (int s = 0; s < NZ; ++s) {
      mbar_init(&zfull[s], 1);
      mbar_init(&zempty[s], 1);
    }
    mbar_init(&vfull, 1);
    mbar_init(&vempty, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&d_full[s], 1);
      mbar_init(&d_empty[s], kOzuEpi / 2);
    }
    mbar_fence_init();
  }
  __syncthreads();
  if (warp == 0) tmem_alloc(&tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  double s_top = 0.0, s_trail = 0.0;

  if (warp == kOzuEpi) {
    // ---------------------------------------------------------------- TMA producer: W
    if (lane == 0) {
      int s = L0 / NC, c = L0 - s * NC;
      for (int i = 0; i < ntile; ++i) {
        const int st = i % NW;
        if (i >= NW && !mbar_wait(&wempty[st], ((i / NW) - 1) & 1, ctrl)) break;
        mbar_expect_tx(&wfull[st], Cfg::W_BYTES);
#pragma unroll
        for (int x = 0; x < 2; ++x)
          tma_load_2d(ringW + st * Cfg::W_BYTES + x * Cfg::BOX, &tmC, c * BN + x * 16, r0 + s * 128, &wfull[st]);
        if (++c == NC) { c = 0; ++s; }
      }
    }
  } else if (warp == kOzuEpi + 1) {
    // ---------------------------------------------------------------- bulk copies: images of V and Z
    if (lane == 0) {
      int s = L0 / NC, c = L0 - s * NC, nslab = 0;
      bool open = true;                // the tile is the first of its slab here
      for (int i = 0; i < ntile; ++i) {
        if (open) {
          if (nslab > 0 && !mbar_wait(&vempty, (nslab - 1) & 1, ctrl)) break;
          mbar_expect_tx(&vfull, Cfg::V_BYTES);
          oz_bulk_load(smem_u32(sV), vimg + (size_t)s * Cfg::V_BYTES, Cfg::V_BYTES, &vfull);
          ++nslab;
          open = false;
        }
        const int st = i % NZ;
        if (i >= NZ && !mbar_wait(&zempty[st], ((i / NZ) - 1) & 1, ctrl)) break;
        mbar_expect_tx(&zfull[st], Cfg::Z_BYTES);
        oz_bulk_load(smem_u32(ringZ + st * Cfg::Z_BYTES), zimg + (size_t)c * Cfg::Z_BYTES, Cfg::Z_BYTES, &zfull[st]);
        if (++c == NC) { c = 0; ++s; open = true; }
      }
    }
  } else if (warp == kOzuEpi + 2) {
    // ---------------------------------------------------------------- MMA issuer
    const uint32_t lead = oz_lead(), v0 = smem_u32(sV), z0 = smem_u32(ringZ);
    int c = L0 % NC, nslab = 0;
    bool open = true;
    for (int i = 0; i < ntile; ++i) {
      const int st = i % NZ, d = i & 1;
      if (open) {
        if (!mbar_wait(&vfull, nslab & 1, ctrl)) break;
        ++nslab;
        open = false;
      }
      if (!mbar_wait(&zfull[st], (i / NZ) & 1, ctrl)) break;
      if (i >= 2 && !mbar_wait(&d_empty[d], ((i >> 1) - 1) & 1, ctrl)) break;
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
        oz_step<BN, 8>(tmem + d * D, v0 + ks * kOzS * 4096, z0 + st * Cfg::Z_BYTES + ks * kOzS * BN * 32, ks == 0, lead);
      oz_commit(&d_full[d], lead);
      oz_commit(&zempty[st], lead);
      if (++c == NC) {
        c = 0;
        open = true;
        oz_commit(&vempty, lead);
      }
    }
  } else {
    // ---------------------------------------------------------------- W - P
    const int quad = warp & 3, box = (warp >> 2) & 1, grp = warp >> 3, r = quad * 32 + lane;
    const uint32_t tlane = tmem + ((uint32_t)(quad * 32) << 16) + grp * D + box * 16;
    int s = (L0 + grp) / NC, c = L0 + grp - s * NC, cur_s = -1;
    double fr = 0.0;
    bool is_top = false, in = false;
    uint32_t rmax = 0u;
    auto end_slab = [&]() {
      if (cur_s >= 0 && rowmag != nullptr && in && !is_top && rmax != 0u)
        atomicMax(rowmag + (cur_s * 128 + r - top_rows), rmax);
      rmax = 0u;
    };
    for (int i = grp; i < ntile; i += 2) {
      const int st = i % NW;
      if (i >= 2 && lane == 0) {
        // the TMA store of this warp's part of its previous tile has read it by now
        bulk_wait_read();
        mbar_arrive(&wempty[(i - 2) % NW]);
      }
      if (s != cur_s) {
        end_slab();
        cur_s = s;
        const int lr = s * 128 + r;
        in = lr < rows;
        is_top = lr < top_rows;          // top_rows is a multiple of 32: the same for the whole warp
        fr = -oz_pow2(in ? ev[lr] - kOzOut : 0);
      }
      const int col = c * BN + box * 16;
      __syncwarp();                     // the last tile's scales have been read
      if (lane < 16) scale_s[warp][lane] = oz_pow2((col + lane < ncols ? ez[col + lane] : 0) - kOzOut);
      __syncwarp();
      if (!mbar_wait(&wfull[st], (i / NW) & 1, ctrl)) break;
      if (!mbar_wait(&d_full[grp], (i >> 1) & 1, ctrl)) break;
      tc_fence_after();
      const uint32_t sW = smem_u32(ringW + st * Cfg::W_BYTES + box * Cfg::BOX + r * 128);
      uint32_t cmax = 0u;                // of column `lane` of the box
      double qs = 0.0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int g[8][8];
        oz_ld8<BN>(tlane + h * 8, g);
        if (h == 2 - 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&d_empty[grp]);
        }
#pragma unroll
        for (int e2 = 0; e2 < 4; ++e2) {
          const uint32_t at = sW + (((uint32_t)(h * 4 + e2) ^ (uint32_t)(r & 7)) << 4);
          double w[2];
          asm volatile("ld.shared.v2.f64 {%0,%1}, [%2];" : "=d"(w[0]), "=d"(w[1]) : "r"(at));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int cc = h * 8 + e2 * 2 + e;
            w[e] = fma(oz_join<B <= 64>(g, e2 * 2 + e) * fr, scale_s[warp][cc], w[e]);
            qs = fma(w[e], w[e], qs);
            const uint32_t mg = oz_mag(w[e]);
            rmax = max(rmax, mg);
            if (colmag != nullptr) {
              const uint32_t cm = __reduce_max_sync(0xffffffffu, mg);
              if (lane == cc) cmax = cm;
            }
          }
          asm volatile("st.shared.v2.f64 [%0], {%1,%2};" ::"r"(at), "d"(w[0]), "d"(w[1]) : "memory");
        }
      }
      proxy_fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        const int lr0 = s * 128 + quad * 32;
        if (lr0 < rows) {
          const uint32_t src = smem_u32(ringW + st * Cfg::W_BYTES + box * Cfg::BOX + quad * 32 * 128);
          if (lr0 < top_rows) tma_store_2d(&tmTs, src, col, lr0);
          else tma_store_2d(&tmCs, src, col, r0 + lr0);
        }
        bulk_commit();
      }
      s_top += is_top ? qs : 0.0;
      s_trail += is_top ? 0.0 : qs;
      if (colmag != nullptr && !is_top && cmax != 0u && col + lane < ncols) atomicMax(colmag + col + lane, cmax);
      for (int u = 0; u < 2; ++u)
        if (++c == NC) { c = 0; ++s; }
    }
    end_slab();
    if (lane == 0) bulk_wait_all();      // this warp's stores are complete before the CTA may exit
  }
  const double bt = block_sum(s_top, red);
  const double br = block_sum(s_trail, red + 32);
  if (tid == 0 && norm_part != nullptr) {
    norm_part[2 * p] = bt;
    norm_part[2 * p + 1] = br;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------
// The digits of a block's V (rows x B) in both forms and of the B rows of OmegaT that are sampled with next; and zeros for
// the magnitudes that the update after it collects.  Blocks of threads: slabs of 128 rows of V (scale per row), then
// (chunk, 16 columns) of V, then of Omega.  A few MB from L2; the row form is read once, the other in 128-byte pieces.
// ------------------------------------------------------------------------------------------
struct OzSplit {
  const double* V;           // rows x B (NULL: no V)
  long long ldv;
  int rows, nslab, steps_v, chunks_v;
  unsigned char *vrow, *vcol;
  int *erow, *ecol;
  const double* Om;           // B x n, a vector a row (NULL: no Omega)
  long long ldo;
  int n, steps_o, chunks_o;
  unsigned char* oimg;
  int* eo;
  uint32_t *zero0, *zero1;   // words to clear
  int nzero0, nzero1;
};
template <int B>
__global__ void __launch_bounds__(256) oz_split_kernel(const OzSplit a, const int* done_flag) {
  pdl_wait();
  pdl_trigger();
  if (*reinterpret_cast<const volatile int*>(done_flag)) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NB = B < 64 ? B : 64, NH = B / NB;
  for (int i = blockIdx.x * 256 + tid; i < a.nzero0; i += gridDim.x * 256) a.zero0[i] = 0u;
  for (int i = blockIdx.x * 256 + tid; i < a.nzero1; i += gridDim.x * 256) a.zero1[i] = 0u;
  int bx = blockIdx.x;
  if (bx < a.nslab) {
    constexpr int LPR = B / 4, RPW = 32 / LPR;             // lanes a row, rows a warp at a time
    const int j = (lane % LPR) * 4;
    for (int r8 = warp * RPW; r8 < 128; r8 += 8 * RPW) {
      const int r = r8 + lane / LPR, row = bx * 128 + r;
      double x[4] = {0.0, 0.0, 0.0, 0.0};
      if (row < a.rows) {
        const double2* src = reinterpret_cast<const double2*>(a.V + (size_t)row * a.ldv + j);
        const double2 u = src[0], v = src[1];
        x[0] = u.x; x[1] = u.y; x[2] = v.x; x[3] = v.y;
      }
      uint32_t mg = max(max(oz_mag(x[0]), oz_mag(x[1])), max(oz_mag(x[2]), oz_mag(x[3])));
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) mg = max(mg, __shfl_xor_sync(0xffffffffu, mg, o));
      const int e = oz_exp(mg);
      uint32_t w[kOzS];
      oz_words(x, oz_scale(e), w);
      unsigned char* dst = a.vrow + ((size_t)bx * (B / 32) + (j >> 5)) * (kOzS * 4096) + oz_at(r, j & 31);
#pragma unroll
      for (int i = 0; i < kOzS; ++i) *reinterpret_cast<uint32_t*>(dst + i * 4096) = w[i];
      if (j == 0 && row < a.rows) a.erow[row] = e;
    }
    return;
  }
  bx -= a.nslab;
  const bool om = bx >= a.chunks_v * (B / 16);
  if (om) bx -= a.chunks_v * (B / 16);
  const int ch = bx / (B / 16), jg = bx - ch * (B / 16);
  const int first = om ? 0 : B / 32, steps = om ? a.steps_o : a.steps_v, len = om ? a.n : a.rows;
  const int s0 = first > 0 ? (ch == 0 ? 0 : first + (ch - 1) * kOzChunk) : ch * kOzChunk;
  const int s1 = min(steps, first > 0 && ch == 0 ? first : s0 + kOzChunk);
  const int jl = om ? tid >> 4 : tid & 15, kk = om ? tid & 15 : tid >> 4, j = jg * 16 + jl;
  constexpr int UNITS = kOzChunk * 2 / 16;                  // pieces of 16 indices a thread
  __shared__ uint32_t mx[16][17];
  double x[UNITS][16];
  uint32_t mg = 0u;
#pragma unroll
  for (int u = 0; u < UNITS; ++u) {
    const int half = kk + 16 * u, k0 = s0 * 32 + half * 16;
    const bool live = s0 + (half >> 1) < s1;
#pragma unroll
    for (int e = 0; e < 16; ++e) x[u][e] = 0.0;
    if (live) {
      if (om) {
        const double* src = a.Om + (size_t)j * a.ldo + k0;
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          if (k0 + e + 1 < len) {
            const double2 v = *reinterpret_cast<const double2*>(src + e);
            x[u][e] = v.x;
            x[u][e + 1] = v.y;
          } else if (k0 + e < len) {
            x[u][e] = src[e];
          }
        }
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (k0 + e < len) x[u][e] = a.V[(size_t)(k0 + e) * a.ldv + j];
      }
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) mg = max(mg, oz_mag(x[u][e]));
  }
  mx[jl][kk] = mg;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 16; ++q) mg = max(mg, mx[jl][q]);
  const int e0 = oz_exp(mg);
  const double s = oz_scale(e0);
  if (kk == 0) (om ? a.eo : a.ecol)[ch * B + j] = e0;
  unsigned char* img = om ? a.oimg : a.vcol;
#pragma unroll
  for (int u = 0; u < UNITS; ++u) {
    const int half = kk + 16 * u, st = s0 + (half >> 1);
    if (st >= s1) continue;
    uint32_t word[kOzS][4];
#pragma unroll
    for (int k4 = 0; k4 < 4; ++k4) {
      const double q[4] = {x[u][k4 * 4], x[u][k4 * 4 + 1], x[u][k4 * 4 + 2], x[u][k4 * 4 + 3]};
      uint32_t w[kOzS];
      oz_words(q, s, w);
#pragma unroll
      for (int i = 0; i < kOzS; ++i) word[i][k4] = w[i];
    }
    unsigned char* dst = img + (size_t)(st * NH + j / NB) * (kOzS * NB * 32) + oz_at(j % NB, (half & 1) * 16);
#pragma unroll
    for (int i = 0; i < kOzS; ++i)
      *reinterpret_cast<uint4*>(dst + i * NB * 32) = make_uint4(word[i][0], word[i][1], word[i][2], word[i][3]);
  }
}

// ------------------------------------------------------------------------------------------
// Largest magnitudes of the rows and columns of a rows x cols matrix (high words, maxima into arrays of zeros) and, with
// sq_part, per-CTA partial sums of squares: one read of the matrix, HBM bound.  Tiles of 32 rows x 512 columns, a
// thread two columns.
// ------------------------------------------------------------------------------------------
constexpr int kMagRows = 32;
constexpr int kMagCols = 512;
__global__ void __launch_bounds__(256)
    oz_mag_kernel(const double* __restrict__ C, long long ldc, int rows, int cols, uint32_t* __restrict__ colmag,
                  uint32_t* __restrict__ rowmag, double* __restrict__ sq_part) {
  constexpr int VEC = 2;
  __shared__ double red[32];
  __shared__ uint32_t rm[kMagRows];
  const int tid = threadIdx.x;
  const int nc = (cols + kMagCols - 1) / kMagCols, nr = (rows + kMagRows - 1) / kMagRows;
  double sq = 0.0;
  for (int t = blockIdx.x; t < nc * nr; t += gridDim.x) {
    const int tr = t / nc, c = (t - tr * nc) * kMagCols + VEC * tid, r0 = tr * kMagRows;
    if (tid < kMagRows) rm[tid] = 0u;
    __syncthreads();
    uint32_t m[VEC] = {};
#pragma unroll 8
    for (int r = 0; r < kMagRows; ++r) {
      double v[VEC] = {};
      if (r0 + r < rows) {
        const double* src = C + (size_t)(r0 + r) * ldc + c;
        if (c + VEC <= cols) {
          VecLoad16<double>::ld(reinterpret_cast<const unsigned char*>(src), v);
        } else {
#pragma unroll
          for (int u = 0; u < VEC; ++u)
            if (c + u < cols) v[u] = src[u];
        }
      }
      uint32_t w = 0u;
#pragma unroll
      for (int u = 0; u < VEC; ++u) {
        const uint32_t a = oz_mag(v[u]);
        m[u] = max(m[u], a);
        w = max(w, a);
        sq = fma(v[u], v[u], sq);
      }
      if (rowmag != nullptr) {
        w = __reduce_max_sync(0xffffffffu, w);
        if ((tid & 31) == 0) atomicMax(&rm[r], w);
      }
    }
#pragma unroll
    for (int u = 0; u < VEC; ++u)
      if (colmag != nullptr && c + u < cols && m[u] != 0u) atomicMax(colmag + c + u, m[u]);
    __syncthreads();
    if (rowmag != nullptr && tid < kMagRows && r0 + tid < rows && rm[tid] != 0u) atomicMax(rowmag + r0 + tid, rm[tid]);
    __syncthreads();
  }
  if (sq_part != nullptr) {
    const double tot = block_sum(sq, red);
    if (tid == 0) sq_part[blockIdx.x] = tot;
  }
}

// Sampled panel (rows x b, dense) = the partial slots of oz_gemm_kernel, summed in CTA order
__global__ void __launch_bounds__(256)
    oz_panel_sum_kernel(const double* __restrict__ part, int nc, int tpc, long long rows, int b, double* __restrict__ Y, Ctrl* ctrl) {
  if (*reinterpret_cast<volatile int*>(&ctrl->done)) return;
  const long long total = rows * b;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < total; i += (long long)gridDim.x * 256) {
    const int r = (int)(i / b), c = (int)(i - (long long)r * b), sl = r >> 7;
    const int p_lo = sl * nc / tpc, p_hi = ((sl + 1) * nc - 1) / tpc;
    double s = 0.0;
    for (int p = p_lo; p <= p_hi; ++p) s += __ldcg(part + (size_t)(p + sl) * (128 * b) + (size_t)(r & 127) * b + c);
    Y[i] = s;
  }
}

}  // namespace rrf

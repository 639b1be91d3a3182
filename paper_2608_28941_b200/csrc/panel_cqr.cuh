// Panel QR without a dependent exchange per column: Cholesky QR and Householder reconstruction.
//
// What bounded the column loop of panel_kernel is not arithmetic: every one of the b columns needs the column before
// it, an exchange between the CTAs and eight block-wide phases, 2.7 us (one cluster) to 4 us (grid) a column.  The
// Householder vectors of a panel Y depend on Y only up to an upper triangular factor with positive diagonal from the
// right: the QR factorisations of Y and of Q1 = Y X (X upper triangular, positive diagonal) have the same reflectors.
// So the panel is made orthonormal first, with matrix products and two reductions over the CTAs in place of b, and
// the reflectors are then read off the orthonormal panel:
//   G  = Y^T Y                       one sum over the CTAs
//   R1 = chol(G), Q1 = Y R1^-1       (the accuracy of R1 does not matter: any such triangle will do)
//   G1 = Q1^T Q1                     the other sum
//   R2 = chol(G1)                    Q1 R2^-1 is orthonormal to working precision
//   Q1 - [S R2; 0] = V U'            LU without pivoting of the top b x b block, S_jj = -sign of the pivot (the
//                                    Householder sign, so that |U'_jj| >= R2_jj: the elimination cannot break down)
//   V  = Q1 U'^-1 below the top      T = -(U' R2^-1) S V1^-T
// (Ballard, Demmel, Grigori, Jacquelin, Knight, Nguyen 2015, "Reconstructing Householder vectors from tall-skinny QR";
// Yamamoto, Nakatsukasa, Yanagisawa, Fukaya 2015 for the second Cholesky pass.)
//
// Householder QR takes any panel, Cholesky QR only one whose condition number is below about 1e7.  Three tests, which
// every CTA takes on the same numbers, send a panel to the column loop instead: a pivot of the first Cholesky
// factorisation below kCqrPivot of its diagonal entry (dependent columns, zeros, NaN), G1 further than kCqrDefect from
// the identity, and an entry of S-sign pivots that leaves nothing below it (the convention there is H = I, tau = 0).
// The loop then runs on Y, or on Q1, whose reflectors are the same.
//
// One call, B200: 8192 x 64 in 70 us (column loop 265), 4096 x 64 as one cluster 88 (207), 4096 x 32 47 (100), 1024 x 16
// 27 (55).  What bounds it now are the factorisations of the b x b matrices, which every CTA does for itself (9.5 and
// 14 us for b = 64, one dependent reciprocal per column), two exchanges through L2 (16 us; through the cluster 11), and
// on tall slabs the FP64 tensor rate of the few SMs in use.  A panel that is sent to the column loop pays for the
// attempt, and 4 % for a loop that shares its kernel with it: two equal columns 294, 115 (4096 x 32) and 62 us.
//
// V and T keep within 100 u cond of a Householder QR (tests), as the column loop's do.
#pragma once

#include "panel_sync.cuh"

namespace rrf {

constexpr double kCqrPivot = 1e-11;      // least Cholesky pivot, relative to the column's squared norm
constexpr double kCqrDefect = 0.05;      // largest entry of G1 - I
constexpr double kCqrFirstOrder = 8e-9;  // below this times 1/b, R2 = I + triu(E): the next term is E^2 < 1e-16
constexpr double kCqrAlone = 1e-10;      // 1 - |pivot| of a column that has nothing below its pivot

// The upper triangle of a B x B matrix as 8 x 8 blocks (K, J), K <= J, block column by block column; element (k, j) of a
// block is at 8 j + k, so that a product's right operand (two consecutive k of one column per thread) is one 16-byte
// load without bank conflicts.
template <int B>
struct Cqr {
  static constexpr int NB = B / 8;
  static constexpr int E = NB * (NB + 1) / 2 * 64;        // entries of a packed triangle
  static constexpr int PA = B + 4;                        // pitch of the full matrix: fragment loads hit 16 bank pairs
  static constexpr int MT = B / 16;
  static constexpr int NTILE = MT * (MT + 1);             // 16 x 8 tiles that meet the triangle
  static constexpr int KG = B == 64 ? 4 : (B == 32 ? 8 : 16);   // row groups of a Gram product, TG warps each
  static constexpr int TG = 16 / KG;
  static constexpr int TPW = NTILE / TG;                  // tiles per warp: 5, 3, 2
  static constexpr int NBUF = KG / 2;                     // partial triangles in shared memory (two groups share one)
  static constexpr int WORK_T = E + B * PA;               // packed triangle + full matrix
  static constexpr int WORK = WORK_T > NBUF * E ? WORK_T : NBUF * E;
  static constexpr int DINV = 2 * NB * 64;                // inverted diagonal blocks of two triangles
  static_assert(NTILE % TG == 0, "tiles divide over the warps");
};
__host__ __device__ constexpr int cqr_work_doubles(int b) {
  return b == 64 ? Cqr<64>::WORK : (b == 32 ? Cqr<32>::WORK : (b == 16 ? Cqr<16>::WORK : 0));
}
__host__ __device__ constexpr int cqr_dinv_doubles(int b) { return b <= 64 ? 16 * b : 0; }
__host__ __device__ constexpr int cqr_entries(int b) { return (b / 8) * (b / 8 + 1) / 2 * 64; }
// global scratch of the cooperative form: per-CTA triangles, their sum, the top block
__host__ __device__ constexpr size_t cqr_global_doubles(int sms, int b) { return (size_t)(sms + 1) * cqr_entries(b) + (size_t)b * b; }

__device__ __forceinline__ int cqr_blk(int K, int J) { return (J * (J + 1) / 2 + K) * 64; }

constexpr int kCqrBarriers = 4;          // grid barriers of the cooperative form: two per reduction

struct CqrArgs {
  double* S;            // slab, column-major, pitch Rp (4 mod 16), zero below its last row
  int Rp, nloc, gr0, row0;
  double* work;         // Cqr<B>::WORK doubles of shared memory
  double* dinv;         // Cqr<B>::DINV doubles
  double* small;        // [4 B]: diagonal of G, scratch of the factorisations, signs
  double* rbuf;         // cluster: Cqr<B>::E doubles the peers write into
  double* gpart;        // global [G][E]
  double* gsum;         // global [E]
  double* gtop;         // global [B][B]
  int G, cta;
  unsigned* bar;
  unsigned bar_base;
  unsigned nbar;        // grid barriers passed before the call
  uint64_t* cbar;
  unsigned nx;          // cluster barriers passed before the call
  Ctrl* ctrl;
  bool want_t;          // this CTA writes T
  bool single, vec;     // V and T are single precision; two elements of a row of V can be stored at once
  void* V;
  long long ldv;
  void* T;
  long long ldt;
};

// 1 / d and 1 / sqrt(d) of normal numbers: the hardware's approximation (about 20 bits) and one step of Householder's
// third-order iteration.  The library's forms cost twice the latency, and these sit on chains of b dependent columns.
// Largest error over a million numbers from 2^-968 to 2^930: 0.51 and 0.99 units in the last place.
__device__ __forceinline__ double cqr_rcp(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double cqr_rsqrt(double d) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double h = fma(-d * r, r, 1.0);
  return fma(r * h, fma(0.375, h, 0.5), r);
}

// One warp factors a diagonal block of a packed triangle, G = R^T R, all lanes alike in registers: one reciprocal per
// column on the dependent chain, the roots beside it.  gd: the diagonal before any elimination; rs: 1 / R_kk.
// Returns whether every pivot passed.
__device__ __forceinline__ bool cqr_chol8(double* __restrict__ blk, const double* __restrict__ gd, double* __restrict__ rs,
                                          double least, int lane) {
  double a[36];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int k = 0; k <= j; k += 2) {
      const double2 v = *reinterpret_cast<const double2*>(blk + j * 8 + k);
      a[j * (j + 1) / 2 + k] = v.x;
      if (k + 1 <= j) a[j * (j + 1) / 2 + k + 1] = v.y;
    }
  double thr[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) thr[p] = least * gd[p];
  bool ok = true;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const double d = a[p * (p + 1) / 2 + p];
    ok &= d >= thr[p];
    const double r = cqr_rcp(d);
#pragma unroll
    for (int j = p + 1; j < 8; ++j) {
      const double u = a[j * (j + 1) / 2 + p] * r;
#pragma unroll
      for (int j2 = j; j2 < 8; ++j2) a[j2 * (j2 + 1) / 2 + j] = fma(-u, a[j2 * (j2 + 1) / 2 + p], a[j2 * (j2 + 1) / 2 + j]);
    }
    const double q = cqr_rsqrt(d);
#pragma unroll
    for (int j = p; j < 8; ++j) a[j * (j + 1) / 2 + p] *= q;
    thr[p] = q;
  }
  __syncwarp();                      // every lane has its copy before the first one is overwritten
  // every lane stores the same value
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int k = 0; k <= j; k += 2) {
      if (k + 1 <= j)
        *reinterpret_cast<double2*>(blk + j * 8 + k) = make_double2(a[j * (j + 1) / 2 + k], a[j * (j + 1) / 2 + k + 1]);
      else
        blk[j * 8 + k] = a[j * (j + 1) / 2 + k];
    }
#pragma unroll
  for (int p = 0; p < 8; p += 2) *reinterpret_cast<double2*>(rs + p) = make_double2(thr[p], thr[p + 1]);
  __syncwarp();
  return ok;
}

// Column c of the inverse of an upper triangular 8 x 8 block given by get(k, j) with the inverses of its diagonal in ri;
// out[8 c + i].
template <typename Get, typename Ri>
__device__ __forceinline__ void cqr_inv8_col(Get get, Ri ri, int c, double* __restrict__ out) {
  double x[8];
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    double s = (i == c) ? 1.0 : 0.0;
#pragma unroll
    for (int k = 7; k > i; --k) s -= get(i, k) * x[k];
    x[i] = s * ri(i);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) out[c * 8 + i] = x[i];
}

// Cholesky factorisation of the packed triangle in place, and the inverses of its diagonal blocks.  All threads of the
// CTA call it.  Per block column: warp 0 brings the diagonal block up to date and factors it while the other warps
// update the rest of the trailing triangle; then the block row, one thread per column.
template <int B>
__device__ __noinline__ bool cqr_chol(double* __restrict__ M, double* __restrict__ dinv, double* __restrict__ small, double least,
                                      int tid) {
  constexpr int NB = Cqr<B>::NB;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  double* gd = small;               // [B] diagonal at the start
  double* rs = small + B;           // [B] 1 / R_kk
  __shared__ int chol_bad;
  if (tid == 0) chol_bad = 0;
  if (tid < B) {
    const double v = M[cqr_blk(tid >> 3, tid >> 3) + (tid & 7) * 9];
    gd[tid] = (v > 1e-280 && v < 1e280) ? v : __longlong_as_double(0x7ff8000000000000LL);   // NaN: fails any pivot test
  }
  __syncthreads();
#pragma unroll 1
  for (int K = 0; K < NB; ++K) {
    // what block row L = K - 1 takes off the trailing triangle: G[I, J] -= R[L, I]^T R[L, J]; a tile holds the columns of
    // two block columns J and the rows of one block row I (its transpose, in the packed order)
    const int L = K - 1;
    auto tile = [&](int m, int I) {
      const int J0 = 2 * m, J1 = J0 + 1;
      const bool v0 = J0 > L && I <= J0;
      const double2 z = make_double2(0.0, 0.0);
      const double2 a0 = v0 ? *reinterpret_cast<const double2*>(M + cqr_blk(L, J0) + g * 8 + 2 * t) : z;
      const double2 a1 = *reinterpret_cast<const double2*>(M + cqr_blk(L, J1) + g * 8 + 2 * t);
      const double2 bb = *reinterpret_cast<const double2*>(M + cqr_blk(L, I) + g * 8 + 2 * t);
      double2* p0 = reinterpret_cast<double2*>(M + cqr_blk(I, v0 ? J0 : J1) + g * 8 + 2 * t);
      double2* p1 = reinterpret_cast<double2*>(M + cqr_blk(I, J1) + g * 8 + 2 * t);
      const double2 c0 = v0 ? *p0 : z, c1 = *p1;
      double acc[4] = {c0.x, c0.y, c1.x, c1.y};
      const double af[4] = {-a0.x, -a1.x, -a0.y, -a1.y}, bf[2] = {bb.x, bb.y};
      mma16x8x8(acc, af, bf);
      if (v0) *p0 = make_double2(acc[0], acc[1]);
      *p1 = make_double2(acc[2], acc[3]);
    };
    if (warp == 0) {
      if (K > 0) tile(K >> 1, K);
      __syncwarp();
      const bool ok = cqr_chol8(M + cqr_blk(K, K), gd + K * 8, rs + K * 8, least, lane);
      if (lane == 0 && !ok) chol_bad = 1;
    } else if (K > 0 && (warp & 3) != 0) {      // not the warps that share warp 0's FP64 pipe
      for (int id = (warp >> 2) * 3 + (warp & 3) - 1; id < NB * NB / 2; id += 12) {
        const int m = id / NB, I = id & (NB - 1);
        if (m >= K >> 1 && I >= K && I <= 2 * m + 1 && (m > K >> 1 || I > K)) tile(m, I);
      }
    }
    __syncthreads();
    // block row K: R_KK^T R[K, J] = G[K, J], one thread per column
    const int ncol = (NB - 1 - K) * 8;
    if (tid < ncol) {
      const int J = K + 1 + (tid >> 3);
      double* col = M + cqr_blk(K, J) + (tid & 7) * 8;
      const double* rd = M + cqr_blk(K, K);
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = col[i];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int i = 0; i < k; i += 2) {
          const double2 r = *reinterpret_cast<const double2*>(rd + k * 8 + i);
          v[k] = fma(-r.x, v[i], v[k]);
          if (i + 1 < k) v[k] = fma(-r.y, v[i + 1], v[k]);
        }
        v[k] *= rs[K * 8 + k];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) col[i] = v[i];
    }
    __syncthreads();
  }
  if (tid < B) {
    const double* rd = M + cqr_blk(tid >> 3, tid >> 3);
    const double* rk = rs + (tid & ~7);
    cqr_inv8_col([&](int k, int j) { return rd[j * 8 + k]; }, [&](int k) { return rk[k]; }, tid & 7, dinv + (tid >> 3) * 64);
  }
  const bool ok = chol_bad == 0;
  __syncthreads();
  return ok;
}

// X <- X R^-1 for a strip of 16 rows held by one warp in accumulator fragments (x[J]: rows g, g + 8, columns
// 8 J + 2 t, + 1).  An accumulator fragment is the left operand of the next product as it stands, with the
// contraction index permuted alike on both sides.  bop(K, J) gives the right operand's two values of block (K, J) of R.
// dinv(K): the inverse of diagonal block K.
template <int NB, typename DOp, typename BOp>
__device__ __forceinline__ void cqr_trsm(double (&x)[NB][4], DOp dinv, BOp bop, int g, int t) {
#pragma unroll
  for (int K = 0; K < NB; ++K) {
    const double2 di = *reinterpret_cast<const double2*>(dinv(K) + g * 8 + 2 * t);
    {
      const double af[4] = {x[K][0], x[K][2], x[K][1], x[K][3]}, bf[2] = {di.x, di.y};
      double y[4] = {0.0, 0.0, 0.0, 0.0};
      mma16x8x8(y, af, bf);
#pragma unroll
      for (int e = 0; e < 4; ++e) x[K][e] = y[e];
    }
    const double af[4] = {-x[K][0], -x[K][2], -x[K][1], -x[K][3]};
#pragma unroll
    for (int J = K + 1; J < NB; ++J) {
      const double2 r = bop(K, J);
      const double bf[2] = {r.x, r.y};
      mma16x8x8(x[J], af, bf);
    }
  }
}

// Partial S^T S of this CTA's slab: NBUF packed triangles in `work`, to be added in order.
template <int B>
__device__ __noinline__ void cqr_gram(const double* __restrict__ S, int Rp, int nloc, double* __restrict__ work, int tid) {
  using C = Cqr<B>;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int kg = warp / C::TG, tg = warp - kg * C::TG;
  const int nks = (nloc + 7) >> 3;
  double acc[C::TPW][4];
  int mt[C::TPW], nt[C::TPW];
#pragma unroll
  for (int q = 0; q < C::TPW; ++q) {
    const int id = tg * C::TPW + q;           // tiles of m: nt = 0 .. 2 m + 1, m (m + 1) tiles before them
    int m = 0;
    while ((m + 1) * (m + 2) <= id) ++m;
    mt[q] = m;
    nt[q] = id - m * (m + 1);
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[q][e] = 0.0;
  }
  for (int ks = kg; ks < nks; ks += C::KG) {
    const double* base = S + ks * 8 + t;
#pragma unroll
    for (int q = 0; q < C::TPW; ++q) {
      const double* pa = base + (size_t)(mt[q] * 16 + g) * Rp;
      const double* pb = base + (size_t)(nt[q] * 8 + g) * Rp;
      const double af[4] = {pa[0], pa[8 * Rp], pa[4], pa[8 * Rp + 4]}, bf[2] = {pb[0], pb[4]};
      mma16x8x8(acc[q], af, bf);
    }
  }
  double* buf = work + (kg % C::NBUF) * C::E;
#pragma unroll
  for (int round = 0; round < 2; ++round) {
    if (kg / C::NBUF == round) {
#pragma unroll
      for (int q = 0; q < C::TPW; ++q) {
        const int J0 = 2 * mt[q], J1 = J0 + 1, I = nt[q];
        double2* p1 = reinterpret_cast<double2*>(buf + cqr_blk(I, J1) + g * 8 + 2 * t);
        double2 v1 = make_double2(acc[q][2], acc[q][3]);
        if (round) { v1.x += p1->x; v1.y += p1->y; }
        *p1 = v1;
        if (I <= J0) {
          double2* p0 = reinterpret_cast<double2*>(buf + cqr_blk(I, J0) + g * 8 + 2 * t);
          double2 v0 = make_double2(acc[q][0], acc[q][1]);
          if (round) { v0.x += p0->x; v0.y += p0->y; }
          *p0 = v0;
        }
      }
    }
    __syncthreads();
  }
}

// Sum of every CTA's partial triangle (fixed order) into the packed triangle at `work`, the same bits in every CTA.
// Two steps: CTA c adds its share of the entries over all CTAs, then everyone takes the sums.  With `top`, the top
// b x b block the CTAs left in a.gtop is loaded behind the first step.  Returns false when a wait gave up.
template <int B, bool CL>
__device__ __forceinline__ bool cqr_reduce(const CqrArgs& a, bool top, int tid) {
  unsigned nb = top ? 2 : 0, nx = a.nx + nb;      // barriers of this call so far
  using C = Cqr<B>;
  constexpr int NT = 512;
  auto mine = [&](int e) {
    double v = a.work[e];
#pragma unroll
    for (int q = 1; q < C::NBUF; ++q) v += a.work[q * C::E + e];
    return v;
  };
  const int epc = (C::E + a.G - 1) / a.G;
  if constexpr (CL) {
    for (int e = tid; e < C::E; e += NT) {
      const int owner = e / epc;
      cl_st(cl_map(smem_u32(a.rbuf + a.cta * epc + (e - owner * epc)), owner), mine(e));
    }
    if (!cluster_barrier(a.cbar, nx, a.G, a.ctrl)) return false;
    const int e0 = a.cta * epc, ne = min(epc, C::E - e0);
    double* own = a.work;       // every CTA has read its partial triangles: the peers may write sums there
    for (int e = tid; e < ne; e += NT) {
      double s = 0.0;
      for (int q = 0; q < a.G; ++q) s += a.rbuf[q * epc + e];
      for (int q = 0; q < a.G; ++q) cl_st(cl_map(smem_u32(own + e0 + e), q), s);
    }
    if (top) {
      double* A = a.work + C::E;
      for (int idx = tid; idx < B * B; idx += NT) A[(idx / B) * C::PA + (idx & (B - 1))] = __ldcg(a.gtop + idx);
    }
    return cluster_barrier(a.cbar, nx, a.G, a.ctrl);
  } else {
    for (int e = tid; e < C::E; e += NT) a.gpart[(size_t)a.cta * C::E + e] = mine(e);
    if (!grid_barrier(a.bar, a.bar_base + (a.nbar + ++nb) * (unsigned)a.G, a.ctrl)) return false;
    const int e0 = a.cta * epc, ne = min(epc, C::E - e0);
    if (ne > 0) {
      int tpe = 1;                              // threads that share an entry
      while (tpe * 2 * epc <= NT && tpe < 32) tpe *= 2;
      const int q0 = tpe > 1 ? tid / epc : 0;
      for (int e = tpe > 1 ? tid - q0 * epc : tid; e < ne; e += (tpe > 1 ? C::E : NT)) {
        if (q0 >= tpe) break;
        const double* p = a.gpart + e0 + e;
        double s = 0.0;
        int x = q0;
        for (; x + 7 * tpe < a.G; x += 8 * tpe) {
          double v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = __ldcg(p + (size_t)(x + u * tpe) * C::E);
#pragma unroll
          for (int u = 0; u < 8; ++u) s += v[u];
        }
        {
          double v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = x + u * tpe < a.G ? __ldcg(p + (size_t)(x + u * tpe) * C::E) : 0.0;
#pragma unroll
          for (int u = 0; u < 8; ++u) s += v[u];
        }
        if (tpe > 1) a.work[q0 * epc + e] = s;
        else a.gsum[e0 + e] = s;
      }
      if (tpe > 1) {
        __syncthreads();
        if (tid < ne) {
          double s = 0.0;
          for (int q = 0; q < tpe; ++q) s += a.work[q * epc + tid];
          a.gsum[e0 + tid] = s;
        }
      }
    }
    if (!grid_barrier(a.bar, a.bar_base + (a.nbar + ++nb) * (unsigned)a.G, a.ctrl)) return false;
    for (int e = tid; e < C::E; e += NT) a.work[e] = __ldcg(a.gsum + e);
    if (top) {
      double* A = a.work + C::E;
      for (int idx = tid; idx < B * B; idx += NT) A[(idx / B) * C::PA + (idx & (B - 1))] = __ldcg(a.gtop + idx);
    }
    __syncthreads();
    return true;
  }
}

// LU factorisation of the diagonal block K of A - S R2 by one warp, column by column, all lanes alike in registers (no
// shuffle stands between one reciprocal and the next).  The sign of every pivot is chosen on the way.  Returns whether
// every column leaves something below its pivot.
template <int B>
__device__ __forceinline__ bool cqr_lu8(double* __restrict__ A, const double* __restrict__ M, int K, double* __restrict__ sgn,
                                        double* __restrict__ rinv, int lane) {
  constexpr int PA = Cqr<B>::PA;
  double* blk = A + (size_t)(8 * K) * PA + 8 * K;
  const double* rb = M + cqr_blk(K, K);
  double l[28];                        // row i, column k < i at i (i - 1) / 2 + k
  double sv[8], nx[8];                 // nx: the next column, loaded before this one is stored
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 8; ++i) nx[i] = blk[i * PA];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    double x[8], r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = nx[i];
      if (c < 7) nx[i] = blk[i * PA + c + 1];
    }
#pragma unroll
    for (int i = 0; i <= c; ++i) r[i] = rb[c * 8 + i];
#pragma unroll
    for (int k = 0; k < c; ++k) {
      x[k] = fma(-sv[k], r[k], x[k]);
#pragma unroll
      for (int i = k + 1; i < 8; ++i) x[i] = fma(-l[i * (i - 1) / 2 + k], x[k], x[i]);
    }
    ok &= fabs(x[c]) <= (1.0 - kCqrAlone) * r[c];
    sv[c] = -copysign(1.0, x[c]);
    x[c] += copysign(r[c], x[c]);
    const double ri = cqr_rcp(x[c]);
#pragma unroll
    for (int i = c + 1; i < 8; ++i) {
      x[i] *= ri;
      l[i * (i - 1) / 2 + c] = x[i];
    }
    // every lane stores the same value: a branch here would end the block the compiler schedules over.  All of them
    // have loaded this column by then (nx, one column ago).
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) blk[i * PA + c] = x[i];
    sgn[8 * K + c] = sv[c];
    rinv[8 * K + c] = ri;
  }
  __syncwarp();
  return ok;
}

// A <- V1 (strictly below the diagonal, unit diagonal implied) and U' (on and above it) of A - S R2 = V1 U'; rinv: the
// inverses of U's diagonal.  All threads of the CTA call it.
template <int B>
__device__ __forceinline__ bool cqr_lu(double* __restrict__ A, const double* __restrict__ M, double* __restrict__ sgn,
                                       double* __restrict__ rinv, int tid) {
  constexpr int NB = Cqr<B>::NB, PA = Cqr<B>::PA;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  __shared__ int lu_bad;
  if (tid == 0) lu_bad = 0;
#pragma unroll 1
  for (int K = 0; K < NB; ++K) {
    // trailing block of step L = K - 1: A[I, J] -= V1[I, L] U'[L, J], tiles of 16 rows x 8 columns from row 8 K on (the
    // last tile of a column may have 8 rows only)
    auto tile = [&](int i0, int J) {
      const bool two = i0 + 8 < B;
      const double* l0 = A + (size_t)(i0 + g) * PA + 8 * (K - 1) + t;
      const double* l1 = l0 + (two ? 8 * PA : 0);
      const double* u = A + (size_t)(8 * (K - 1) + t) * PA + 8 * J + g;
      double2* p0 = reinterpret_cast<double2*>(A + (size_t)(i0 + g) * PA + 8 * J + 2 * t);
      double2* p1 = reinterpret_cast<double2*>(A + (size_t)(i0 + g + (two ? 8 : 0)) * PA + 8 * J + 2 * t);
      const double2 c0 = *p0, c1 = *p1;
      double acc[4] = {c0.x, c0.y, c1.x, c1.y};
      const double af[4] = {-l0[0], -l1[0], -l0[4], -l1[4]}, bf[2] = {u[0], u[4 * PA]};
      mma16x8x8(acc, af, bf);
      *p0 = make_double2(acc[0], acc[1]);
      if (two) *p1 = make_double2(acc[2], acc[3]);
    };
    if (warp == 0) {
      if (K > 0) tile(8 * K, K);
      __syncwarp();
      const bool ok = cqr_lu8<B>(A, M, K, sgn, rinv, lane);
      if (lane == 0 && !ok) lu_bad = 1;
    } else if (K > 0 && (warp & 3) != 0) {      // not the warps that share warp 0's FP64 pipe
      for (int id = (warp >> 2) * 3 + (warp & 3) - 1; id < NB * NB / 2; id += 12) {
        const int i0 = 8 * K + 16 * (id / NB), J = id & (NB - 1);
        if (i0 < B && J >= K && (id >= NB || J > K)) tile(i0, J);
      }
    }
    __syncthreads();
    const int nrest = (NB - 1 - K) * 8;
    const double* Ad = A + (size_t)(8 * K) * PA + 8 * K;       // factored diagonal block
    if (tid < nrest) {                                          // V1 below: rows, x U'_KK = a
      double* row = A + (size_t)(8 * K + 8 + tid) * PA + 8 * K;
      double x[8];
#pragma unroll
      for (int c = 0; c < 8; c += 2) {
        const double2 v = *reinterpret_cast<const double2*>(row + c);
        x[c] = v.x;
        x[c + 1] = v.y;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        x[c] *= rinv[8 * K + c];
#pragma unroll
        for (int c2 = (c + 1) & ~1; c2 < 8; c2 += 2) {
          const double2 u = *reinterpret_cast<const double2*>(Ad + c * PA + c2);
          if (c2 > c) x[c2] = fma(-x[c], u.x, x[c2]);
          x[c2 + 1] = fma(-x[c], u.y, x[c2 + 1]);
        }
      }
#pragma unroll
      for (int c = 0; c < 8; c += 2) *reinterpret_cast<double2*>(row + c) = make_double2(x[c], x[c + 1]);
    } else if (tid >= 64 && tid < 64 + nrest) {                 // U' to the right: columns, V1_KK u = a - S R2
      const int c = 8 * K + 8 + tid - 64, J = c >> 3;
      double* col = A + (size_t)(8 * K) * PA + c;
      const double* rr = M + cqr_blk(K, J) + (c & 7) * 8;
      double x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = col[i * PA] - sgn[8 * K + i] * rr[i];
#pragma unroll
      for (int i = 1; i < 8; ++i)
#pragma unroll
        for (int k = 0; k < i; k += 2) {
          const double2 l = *reinterpret_cast<const double2*>(Ad + i * PA + k);
          x[i] = fma(-l.x, x[k], x[i]);
          if (k + 1 < i) x[i] = fma(-l.y, x[k + 1], x[i]);
        }
#pragma unroll
      for (int i = 0; i < 8; ++i) col[i * PA] = x[i];
    }
    __syncthreads();
  }
  const bool ok = lu_bad == 0;
  __syncthreads();
  return ok;
}

// two neighbours of a row into a single or double precision matrix
__device__ __forceinline__ void cqr_put(void* base, size_t at, double v0, double v1, bool single, bool vec) {
  if (single) {
    float* p = reinterpret_cast<float*>(base) + at;
    if (vec) {
      *reinterpret_cast<float2*>(p) = make_float2((float)v0, (float)v1);
    } else {
      p[0] = (float)v0;
      p[1] = (float)v1;
    }
  } else {
    double* p = reinterpret_cast<double*>(base) + at;
    if (vec) {
      *reinterpret_cast<double2*>(p) = make_double2(v0, v1);
    } else {
      p[0] = v0;
      p[1] = v1;
    }
  }
}

// The whole of it, called by every thread of every CTA with the panel in the slabs; the arguments lie in shared memory
// (on the stack they go through what is left of the L1: 4 us a call).  Negative: a wait gave up.  Else the low three
// bits say what was done (RRF_PATH_*: V and T are written, or the column loop has to do it, on what the slabs hold) and
// the rest is the number of barriers passed.
template <int B, bool CL>
__device__ __noinline__ int cqr_panel(const CqrArgs& a) {
  using C = Cqr<B>;
  constexpr int NB = C::NB, PA = C::PA;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  double* M = a.work;                  // packed triangle: R1, then R2
  double* A = a.work + C::E;           // top block, then V1 \ U'
  double* dinv_r = a.dinv;
  double* dinv_u = a.dinv + NB * 64;
  double* small = a.small;
  const int row0 = a.row0, Rp = a.Rp;
  const int nstrip = (a.nloc + 15) >> 4;
  // rows above the panel do not belong to it
  for (int idx = tid; idx < B * max(0, min(a.nloc, row0 - a.gr0)); idx += 512) a.S[(size_t)(idx & (B - 1)) * Rp + idx / B] = 0.0;
  __syncthreads();
  cqr_gram<B>(a.S, Rp, a.nloc, a.work, tid);
  if (!cqr_reduce<B, CL>(a, false, tid)) return -1;
  if (!cqr_chol<B>(M, dinv_r, small, kCqrPivot, tid)) return 2 << 3 | RRF_PATH_LOOP_Y;

  const bool has00 = row0 >= a.gr0 && row0 < a.gr0 + a.nloc;
  const double y00 = has00 ? a.S[row0 - a.gr0] : 0.0;
  auto load = [&](double (&x)[NB][4], int r0) {
    const double* p = a.S + (size_t)(2 * t) * Rp + r0 + g;
#pragma unroll
    for (int J = 0; J < NB; ++J) {
      x[J][0] = p[0];
      x[J][1] = p[Rp];
      x[J][2] = p[8];
      x[J][3] = p[Rp + 8];
      p += 8 * Rp;
    }
  };
  auto store = [&](const double (&x)[NB][4], int r0) {
    double* p = a.S + (size_t)(2 * t) * Rp + r0 + g;
#pragma unroll
    for (int J = 0; J < NB; ++J) {
      p[0] = x[J][0];
      p[Rp] = x[J][1];
      p[8] = x[J][2];
      p[Rp + 8] = x[J][3];
      p += 8 * Rp;
    }
  };
  auto packed = [&](int K, int J) { return *reinterpret_cast<const double2*>(M + cqr_blk(K, J) + g * 8 + 2 * t); };
  __syncthreads();                     // y00 is read before it is overwritten
  for (int s = warp; s < nstrip; s += 16) {
    double x[NB][4];
    load(x, s * 16);
    cqr_trsm<NB>(x, [&](int K) { return dinv_r + K * 64; }, packed, g, t);
    store(x, s * 16);
  }
  __syncthreads();
  if (has00 && tid == 0 && y00 == 0.0) a.S[row0 - a.gr0] = y00;      // a zero first pivot keeps its sign
  __syncthreads();
  {
    // this CTA's rows of the top block
    const int lo = max(a.gr0, row0), hi = min(a.gr0 + a.nloc, row0 + B);
    for (int idx = tid; idx < (hi - lo) * B; idx += 512) {
      const int r = idx / B, c = idx & (B - 1);
      a.gtop[(size_t)(lo + r - row0) * B + c] = a.S[(size_t)c * Rp + (lo - a.gr0 + r)];
    }
  }
  cqr_gram<B>(a.S, Rp, a.nloc, a.work, tid);
  if (!cqr_reduce<B, CL>(a, true, tid)) return -1;

  // R2 = chol(G1): to first order where that is exact to the last bit, else the factorisation
  __shared__ int defect_s[2];
  if (tid < 2) defect_s[tid] = 0;
  __syncthreads();
  {
    int big = 0, far = 0;
    for (int e = tid; e < C::E; e += 512) {
      int J = 0;
      while ((J + 1) * (J + 2) / 2 <= (e >> 6)) ++J;
      const int K = (e >> 6) - J * (J + 1) / 2, k = e & 7, j = (e >> 3) & 7;
      if (K == J && k > j) continue;                                  // below the diagonal: not used
      const double d = fabs(M[e] - (K == J && k == j ? 1.0 : 0.0));
      big |= !(d * B <= kCqrFirstOrder);
      far |= !(d <= kCqrDefect);
    }
    if (big) defect_s[0] = 1;
    if (far) defect_s[1] = 1;
  }
  __syncthreads();
  if (defect_s[1]) return 4 << 3 | RRF_PATH_LOOP_Q1;
  if (defect_s[0]) {
    if (!cqr_chol<B>(M, dinv_r, small, 0.25, tid)) return 4 << 3 | RRF_PATH_LOOP_Q1;
  } else {
    if (tid < B) {
      double* d = M + cqr_blk(tid >> 3, tid >> 3) + (tid & 7) * 9;
      *d = 1.0 + 0.5 * (*d - 1.0);
    }
    __syncthreads();
  }
  double* sgn = small + 2 * B;
  double* rinv = small + 3 * B;
  if (!cqr_lu<B>(A, M, sgn, rinv, tid)) return 4 << 3 | RRF_PATH_LOOP_Q1;

  // the inverted diagonal blocks the products below need: of U', and for T of R2 and V1^T (the latter in place of R2's
  // diagonal blocks, which nothing reads any more)
  if (tid < B) {
    const double* ub = A + (size_t)(tid & ~7) * PA + (tid & ~7);
    const double* rk = rinv + (tid & ~7);
    cqr_inv8_col([&](int k, int j) { return ub[k * PA + j]; }, [&](int k) { return rk[k]; }, tid & 7, dinv_u + (tid >> 3) * 64);
  } else if (a.want_t && !defect_s[0] && tid >= 64 && tid < 64 + B) {
    const int c = tid - 64;
    const double* rb = M + cqr_blk(c >> 3, c >> 3);
    cqr_inv8_col([&](int k, int j) { return rb[j * 8 + k]; }, [&](int k) { return cqr_rcp(rb[k * 9]); }, c & 7, dinv_r + (c >> 3) * 64);
  }
  __syncthreads();
  if (a.want_t && tid < B) {
    const double* vb = A + (size_t)(tid & ~7) * PA + (tid & ~7);
    cqr_inv8_col([&](int k, int j) { return vb[j * PA + k]; }, [&](int) { return 1.0; }, tid & 7, M + cqr_blk(tid >> 3, tid >> 3));
  }
  if (a.want_t) __syncthreads();

  const int tw = a.want_t ? B / 16 : 0;          // warps that build T; the others take the strips
  if (warp < tw) {
    // T = -(U' R2^-1) S V1^-T, 16 rows a warp
    double x[NB][4];
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = warp * 16 + g + (e < 2 ? 0 : 8), c = 8 * J + 2 * t + (e & 1);
        x[J][e] = c >= r ? A[(size_t)r * PA + c] : 0.0;
      }
    cqr_trsm<NB>(x, [&](int K) { return dinv_r + K * 64; }, packed, g, t);
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int e = 0; e < 4; ++e) x[J][e] *= -sgn[8 * J + 2 * t + (e & 1)];
    cqr_trsm<NB>(x, [&](int K) { return M + cqr_blk(K, K); },
                 [&](int K, int J) { return *reinterpret_cast<const double2*>(A + (size_t)(8 * J + g) * PA + 8 * K + 2 * t); }, g, t);
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = warp * 16 + g + 8 * h, c = 8 * J + 2 * t;
        cqr_put(a.T, (size_t)r * a.ldt + c, c >= r ? x[J][2 * h] : 0.0, c + 1 >= r ? x[J][2 * h + 1] : 0.0, a.single, false);
      }
  } else {
    // V = Q1 U'^-1 below the top block, V1 in it, straight to where it belongs
    auto upper = [&](int K, int J) {
      const double* p = A + (size_t)(8 * K + 2 * t) * PA + 8 * J + g;
      return make_double2(p[0], p[PA]);
    };
    for (int s = warp - tw; s < nstrip; s += 16 - tw) {
      double x[NB][4];
      load(x, s * 16);
      cqr_trsm<NB>(x, [&](int K) { return dinv_u + K * 64; }, upper, g, t);
      const int ra = a.gr0 + s * 16 + g - row0, rb = ra + 8;            // panel rows of this thread
      if (ra < B) {
#pragma unroll
        for (int J = 0; J < NB; ++J)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int r = e < 2 ? ra : rb, c = 8 * J + 2 * t + (e & 1);
            if (r >= 0 && r < B) x[J][e] = c < r ? A[(size_t)r * PA + c] : (c == r ? 1.0 : 0.0);
          }
      }
      const bool ina = ra >= 0 && s * 16 + g < a.nloc, inb = rb >= 0 && s * 16 + g + 8 < a.nloc;
#pragma unroll
      for (int J = 0; J < NB; ++J) {
        if (ina) cqr_put(a.V, (size_t)ra * a.ldv + 8 * J + 2 * t, x[J][0], x[J][1], a.single, a.vec);
        if (inb) cqr_put(a.V, (size_t)rb * a.ldv + 8 * J + 2 * t, x[J][2], x[J][3], a.single, a.vec);
      }
    }
  }
  return 4 << 3 | (defect_s[0] ? RRF_PATH_CHOLESKY : RRF_PATH_FIRST_ORDER);
}

}  // namespace rrf

// solve_cluster.cu -- the solve Z0 J^{alpha-1} = R^{alpha-1} (paper eq. solve),
// one thread-block cluster per right-hand side, with the exchanged vector kept
// whole in every CTA's shared memory.
//
// Scheme.  Iterative refinement: an FP64 residual r = b - Z0 x around an FP32
// BiCGStab on the right-preconditioned matrix A = Z0 P, which is formed once at
// setup.  Row i of P is row i of the inverse of the block of Z0 among edge i and
// its kScK - 1 strongest couplings (k_local_inverse), or where a trial at setup says so of
// the triangle blocks, or the diagonal's inverse.
// Against the triangle blocks, 32 couplings take a third of the
// iterations (to 1e-5: 7680-RWG sphere 3 to 1, cone-capped cylinder 14.5 to 3.5,
// octahedral ellipsoid 12.5 to 4.5, UV ellipsoid 44.5 to 10.5), and A has about as
// many entries, as it is close to the identity: entries below 1e-6 are left out
// (they would change a correction by less than the 1e-5 it is computed to; the
// FP64 residual decides).  The Krylov vectors live in
// registers, each thread owning 1 to 6 rows; only the vector that the next
// product gathers from travels: every owner stores its values into all CTAs'
// copies through distributed shared memory, so the gathers are shared-memory
// reads and an iteration meets at four cluster barriers (p, alpha's dots, s,
// omega's dots).
//
// What bounds it: latency.  The products stream A from L2 (the prefetch of
// four blocks of 8 rows x 16 entries per warp keeps about 50 KB in flight per
// SM), the reductions are dependent shuffles.  FP64 issues at 1/64 of FP32's
// rate here (2 per clock and SM), so FP64 is left to the residuals and the
// iterate.  Inside the FP32 correction the dots are FP32 over a thread's rows and
// double-float (FP32 pairs, 48 bits) from there, the Krylov scalars are FP32, and
// |s|^2 and |r|^2 follow from the same dots (k_bicgstab has FP64 for all of these); the
// refinement's scale is a power of two, which needs no FP64 division or square root.
// What the correction is worth is decided by the FP64 residual, or by the one carried
// on where the tolerance leaves room for what that misses.
// 1920 RWG, 16 CTAs, alone under ncu: 64 us, 25% of issue slots, waiting for shared-memory
// gathers first and barriers third.
//
// Layout.  Rows are put in an order of their own (`perm`): sorted by length,
// cut into groups of 8 (four lanes per row, so that a warp takes one group at a
// time), the groups dealt over the CTAs and warps.  A warp's groups are one
// contiguous run of blocks of 8 rows x 16 entries, zero padded; a lane reads
// its four entries of a block as one vector, with 16-bit positions.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "internal.h"

namespace cg = cooperative_groups;

namespace tdbem {

constexpr int kScThreads = 512, kScWarps = kScThreads / 32;
constexpr int kScK = 32;            // entries per row of P at most
constexpr double kScDrop = 1e-6;    // entries of A left out (A's diagonal is about 1)
constexpr int kScPasses = 24;       // groups per warp at most: 6 rows per thread
constexpr double kScInner2 = 1e-10; // squared relative residual an inner solve stops at
constexpr int kScDepth = 4;          // blocks a warp keeps in flight
constexpr int kScInnerMax = 80;     // iterations of one inner solve
constexpr int kScTrial = 2 * kScInnerMax;  // most iterations to 1e-5 that a plan may take: 1e-13 is then six of eight inner solves
constexpr int kScGood = 24;         // above these another preconditioner is tried

struct ScArgs {
  const int32_t* perm;       // [npad] row at a position, -1: padding
  const int32_t *ab, *ae;    // A: first block of a warp [cs * 16], block ends of its passes [cs * 16][passes]
  const float4* aval;        // [blocks][32]
  const uint2* acol;         // [blocks][32] four 16-bit positions
  const int32_t *zb, *ze;    // Z0, the same
  const double2* zval;       // [blocks][32][2]
  const float4 *zhi, *zlo;   // Z0 as (hi, lo) pairs
  const uint2* zcol;
  const int32_t *pb, *pe;    // P, as A
  const float4* pval;
  const uint2* pcol;
  double* w64;               // [R][2][npad] iterates as the residual gathers them
  const double* b;           // [ne][R], rows in edge order from here on
  double* x;
  double* ring;
  float2* rs;                // the ring's values as (hi, lo) pairs (may be null)
  float* rf;                 // the ring's values in FP32 (may be null)
  int32_t L, alpha, warm, gpc, passes, npad, ne, maxit, R;
  double tol;
  double zn2;                // |Z0|_1 |Z0|_inf, a bound of the squared 2-norm of (|Z0_ij|)
  int32_t* status;           // as in SolveArgs (solve.cu)
  double* resid;
};

// double-float sums
struct Df {
  float h, l;
};
__device__ __forceinline__ Df df_plus(Df a, Df b) {
  const float s = __fadd_rn(a.h, b.h);
  const float bb = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
  return {s, __fadd_rn(__fadd_rn(a.l, b.l), e)};
}
__device__ __forceinline__ Df df_xor(Df a, int m) {
  return {__shfl_xor_sync(0xffffffffu, a.h, m), __shfl_xor_sync(0xffffffffu, a.l, m)};
}

// Shared memory of a CTA besides the gathered vector.
struct ScShared {
  float2 red[kScWarps][4];
  float4 slots[2][16][2];      // [phase][rank]: four double-float sums
  double red64[kScWarps][2];
  double slots64[2][16][2];
  double bc64[2];
};

__device__ __forceinline__ uint32_t sc_mapa(uint32_t a, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void sc_st(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sc_st4(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void sc_st64(uint32_t a, double x, double y) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x), "d"(y) : "memory");
}

struct ScCtx {
  ScShared* sm;
  int nb, rank, warp, lane, phase;

  __device__ __forceinline__ void sync() {
    if (nb == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }

  // Cluster-wide sums of v[0..3] over all threads (same bits in every thread).
  // The four values are folded together: each shuffle step halves the values a
  // lane carries, 6 double-float additions per lane instead of 20.
  __device__ __forceinline__ void dots4(float v0, float v1, float v2, float v3, float (&out)[4]) {
    Df k0, k1;
    {
      const bool up = lane & 16;
      k0 = {up ? v2 : v0, 0.f};
      k1 = {up ? v3 : v1, 0.f};
      k0 = df_plus(k0, {__shfl_xor_sync(0xffffffffu, up ? v0 : v2, 16), 0.f});
      k1 = df_plus(k1, {__shfl_xor_sync(0xffffffffu, up ? v1 : v3, 16), 0.f});
    }
    {
      const bool up = lane & 8;
      const Df s = up ? k0 : k1;
      k0 = df_plus(up ? k1 : k0, df_xor(s, 8));
    }
    k0 = df_plus(k0, df_xor(k0, 4));
    k0 = df_plus(k0, df_xor(k0, 2));
    k0 = df_plus(k0, df_xor(k0, 1));
    if ((lane & 7) == 0) sm->red[warp][lane >> 3] = make_float2(k0.h, k0.l);  // value lane >> 3
    __syncthreads();
    const int ph = phase++ & 1, id = lane & 3, k = lane >> 2;
    Df t;
    if (nb == 1) {  // one CTA: every warp sums the warps' values itself
      const float2 a = sm->red[k][id], b = sm->red[k + 8][id];
      t = df_plus({a.x, a.y}, {b.x, b.y});
    } else {
      if (warp == 0) {
        const float2 a = sm->red[k][id], b = sm->red[k + 8][id];
        t = df_plus({a.x, a.y}, {b.x, b.y});
        t = df_plus(t, df_xor(t, 4));
        t = df_plus(t, df_xor(t, 8));
        t = df_plus(t, df_xor(t, 16));
        // lane r < nb sends the four sums to CTA r
        const uint32_t dst = sc_mapa((uint32_t)__cvta_generic_to_shared(&sm->slots[ph][rank][0]), lane < nb ? lane : 0);
        const float a0 = __shfl_sync(0xffffffffu, t.h, 0), a1 = __shfl_sync(0xffffffffu, t.l, 0);
        const float b0 = __shfl_sync(0xffffffffu, t.h, 1), b1 = __shfl_sync(0xffffffffu, t.l, 1);
        const float c0 = __shfl_sync(0xffffffffu, t.h, 2), c1 = __shfl_sync(0xffffffffu, t.l, 2);
        const float d0 = __shfl_sync(0xffffffffu, t.h, 3), d1 = __shfl_sync(0xffffffffu, t.l, 3);
        if (lane < nb) {
          sc_st4(dst, a0, a1, b0, b1);
          sc_st4(dst + 16, c0, c1, d0, d1);
        }
      }
      sync();
      const float2* sl = reinterpret_cast<const float2*>(&sm->slots[ph][0][0]);  // [16][4]
      t = {0.f, 0.f};
      if (k < nb) t = {sl[k * 4 + id].x, sl[k * 4 + id].y};
      if (k + 8 < nb) t = df_plus(t, {sl[(k + 8) * 4 + id].x, sl[(k + 8) * 4 + id].y});
    }
    t = df_plus(t, df_xor(t, 4));
    t = df_plus(t, df_xor(t, 8));
    t = df_plus(t, df_xor(t, 16));
    const float s = t.h + t.l;
#pragma unroll
    for (int i = 0; i < 4; ++i) out[i] = __shfl_sync(0xffffffffu, s, i);
    if (nb == 1) __syncthreads();  // red is rewritten by the next sums
  }

  // Cluster-wide FP64 sums of a and b (same bits in every thread).
  __device__ __forceinline__ void sums64(double& a, double& b) {
    const bool up = lane & 16;
    double k = up ? b : a;
    k += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    if ((lane & 15) == 0) sm->red64[warp][lane >> 4] = k;
    __syncthreads();
    const int ph = phase++ & 1;
    if (warp == 0) {
      double t = sm->red64[lane >> 1][lane & 1];
#pragma unroll
      for (int o = 2; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      const double t0 = __shfl_sync(0xffffffffu, t, 0), t1 = __shfl_sync(0xffffffffu, t, 1);
      const uint32_t dst = sc_mapa((uint32_t)__cvta_generic_to_shared(&sm->slots64[ph][rank][0]), lane < nb ? lane : 0);
      if (lane < nb) sc_st64(dst, t0, t1);
    }
    sync();
    if (warp == 0) {
      const int r = lane >> 1;
      double t = r < nb ? sm->slots64[ph][r][lane & 1] : 0.0;
#pragma unroll
      for (int o = 2; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane < 2) sm->bc64[lane] = t;
    }
    __syncthreads();
    a = sm->bc64[0];
    b = sm->bc64[1];
  }
};

// A warp's rows of a matrix times the gathered vector.  Ld: the matrix's
// entries of a block (load), its products added to an accumulator (mul), the
// accumulator's sum over a row's four lanes (fold).  kScDepth blocks are in
// flight: a warp's run is a multiple of that long (zero blocks behind its last
// group), and the loads ahead of its end stay inside the padded array.
// out[e] of lane (row, q) is the row of pass 4 e + q.
template <int RPT, class Ld, class Out>
__device__ __forceinline__ void sc_spmv(Ld ld, int b, int tot, int ends, int lane, Out (&out)[RPT]) {
  typename Ld::Block buf[kScDepth];
  asm volatile("" : "+r"(b));  // the addresses are formed here, not kept in registers over the solver's loops
  int left = tot - b, j = 0, gleft = __shfl_sync(0xffffffffu, ends, 0) - b, gend = gleft + b;
  ld.seek(b, lane);
#pragma unroll
  for (int i = 0; i < kScDepth; ++i) ld.load(buf[i], i);
  typename Ld::Acc acc;
  acc.zero();
#pragma unroll
  for (int e = 0; e < RPT; ++e) out[e] = 0;
  for (; left > 0; left -= kScDepth) {
    ld.skip();
#pragma unroll
    for (int i = 0; i < kScDepth; ++i) {
      ld.mul(buf[i], acc);
      ld.load(buf[i], i);
      if (--gleft == 0) {
        const Out s = acc.fold();
        acc.zero();
#pragma unroll
        for (int e = 0; e < RPT; ++e)
          if (j == 4 * e + (lane & 3)) out[e] = s;
        ++j;
        const int g2 = __shfl_sync(0xffffffffu, ends, j & 31);
        gleft = g2 - gend;
        gend = g2;
      }
    }
  }
}

struct LdA {  // FP32 matrix, FP32 vector in shared memory
  const float4* v;
  const uint2* c;
  const float* X;
  struct Block {
    float4 v;
    uint2 c;
  };
  struct Acc {
    float a, b;
    __device__ __forceinline__ void zero() { a = b = 0.f; }
    __device__ __forceinline__ float fold() {
      float s = a + b;
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      return s + __shfl_xor_sync(0xffffffffu, s, 2);
    }
  };
  __device__ __forceinline__ void seek(int b, int lane) {
    v += (int64_t)b * 32 + lane;
    c += (int64_t)b * 32 + lane;
  }
  __device__ __forceinline__ void skip() {
    v += kScDepth * 32;
    c += kScDepth * 32;
  }
  __device__ __forceinline__ void load(Block& k, int i) const {
    k.v = __ldg(v + i * 32);
    k.c = __ldg(c + i * 32);
  }
  __device__ __forceinline__ void mul(const Block& k, Acc& s) const {
    s.a = fmaf(k.v.x, X[k.c.x & 0xffff], s.a);
    s.b = fmaf(k.v.y, X[k.c.x >> 16], s.b);
    s.a = fmaf(k.v.z, X[k.c.y & 0xffff], s.a);
    s.b = fmaf(k.v.w, X[k.c.y >> 16], s.b);
  }
};

struct LdZ64 {  // FP64 matrix, FP64 vector in global memory
  const double2* v;
  const uint2* c;
  const double* x;
  struct Block {
    double2 v0, v1;
    uint2 c;
  };
  struct Acc {
    double a;
    __device__ __forceinline__ void zero() { a = 0.0; }
    __device__ __forceinline__ double fold() {
      double s = a;
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      return s + __shfl_xor_sync(0xffffffffu, s, 2);
    }
  };
  __device__ __forceinline__ void seek(int b, int lane) {
    v += ((int64_t)b * 32 + lane) * 2;
    c += (int64_t)b * 32 + lane;
  }
  __device__ __forceinline__ void skip() {
    v += kScDepth * 64;
    c += kScDepth * 32;
  }
  __device__ __forceinline__ void load(Block& k, int i) const {
    k.v0 = __ldg(v + i * 64);
    k.v1 = __ldg(v + i * 64 + 1);
    k.c = __ldg(c + i * 32);
  }
  __device__ __forceinline__ void mul(const Block& k, Acc& s) const {
    const double x0 = x[k.c.x & 0xffff], x1 = x[k.c.x >> 16], x2 = x[k.c.y & 0xffff], x3 = x[k.c.y >> 16];
    s.a += k.v0.x * x0;
    s.a += k.v0.y * x1;
    s.a += k.v1.x * x2;
    s.a += k.v1.y * x3;
  }
};

struct LdZdf {  // (hi, lo) matrix, FP32 vector in shared memory, double-float products and sums
  const float4 *h, *l;
  const uint2* c;
  const float* X;
  struct Block {
    float4 h, l;
    uint2 c;
  };
  struct Acc {
    float h, l;
    __device__ __forceinline__ void zero() { h = l = 0.f; }
    __device__ __forceinline__ void add(float zh, float zl, float x) {
      const float p = __fmul_rn(zh, x);
      const float e = __fmaf_rn(zl, x, __fmaf_rn(zh, x, -p));
      const Df t = df_plus({h, l}, {p, e});
      h = t.h;
      l = t.l;
    }
    __device__ __forceinline__ double fold() {
      Df t = {h, l};
      t = df_plus(t, df_xor(t, 1));
      t = df_plus(t, df_xor(t, 2));
      return (double)t.h + (double)t.l;
    }
  };
  __device__ __forceinline__ void seek(int b, int lane) {
    h += (int64_t)b * 32 + lane;
    l += (int64_t)b * 32 + lane;
    c += (int64_t)b * 32 + lane;
  }
  __device__ __forceinline__ void skip() {
    h += kScDepth * 32;
    l += kScDepth * 32;
    c += kScDepth * 32;
  }
  __device__ __forceinline__ void load(Block& k, int i) const {
    k.h = __ldg(h + i * 32);
    k.l = __ldg(l + i * 32);
    k.c = __ldg(c + i * 32);
  }
  __device__ __forceinline__ void mul(const Block& k, Acc& s) const {
    s.add(k.h.x, k.l.x, X[k.c.x & 0xffff]);
    s.add(k.h.y, k.l.y, X[k.c.x >> 16]);
    s.add(k.h.z, k.l.z, X[k.c.y & 0xffff]);
    s.add(k.h.w, k.l.w, X[k.c.y >> 16]);
  }
};

template <int RPT>
__global__ void __launch_bounds__(kScThreads) k_solve_cluster(const ScArgs A) {
  extern __shared__ __align__(16) float sc_X[];
  __shared__ ScShared sm;
  ScCtx S;
  S.sm = &sm;
  {
    uint32_t n, r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    S.nb = (int)n;
    S.rank = (int)r;
  }
  S.warp = (int)threadIdx.x >> 5;
  S.lane = (int)threadIdx.x & 31;
  S.phase = 0;
  const int R = A.R, rhs = (int)blockIdx.x / S.nb;  // this cluster's right-hand side
  double* const w64 = A.w64 + (int64_t)rhs * 2 * A.npad;
  const int lane = S.lane, q = lane & 3, W = S.rank * kScWarps + S.warp;
  const uint32_t Xa = (uint32_t)__cvta_generic_to_shared(sc_X);
  // this thread's rows: position and edge of each (-1: none)
  int pos[RPT], row[RPT];
#pragma unroll
  for (int e = 0; e < RPT; ++e) {
    const int g = (4 * e + q) * kScWarps + S.warp;
    pos[e] = g < A.gpc ? (S.rank * A.gpc + g) * 8 + (lane >> 2) : -1;
    row[e] = pos[e] >= 0 ? A.perm[pos[e]] : -1;
  }
  const int ab = A.ab[W], zb = A.zb[W], pb = A.pb[W];
  const int aends = lane < A.passes ? A.ae[W * A.passes + lane] : 0;
  const int zends = lane < A.passes ? A.ze[W * A.passes + lane] : 0;
  const int pends = lane < A.passes ? A.pe[W * A.passes + lane] : 0;
  const int ptot = __shfl_sync(0xffffffffu, pends, A.passes - 1);
  const int atot = __shfl_sync(0xffffffffu, aends, A.passes - 1), ztot = __shfl_sync(0xffffffffu, zends, A.passes - 1);
  // every CTA's copy of this thread's values
  auto push = [&](const float(&v)[RPT]) {
#pragma unroll 1
    for (int k = 0; k < S.nb; ++k) {
      int r = S.rank + k;
      if (r >= S.nb) r -= S.nb;
      const uint32_t d = sc_mapa(Xa, r);
#pragma unroll
      for (int e = 0; e < RPT; ++e)
        if (pos[e] >= 0) sc_st(d + 4 * pos[e], v[e]);
    }
  };
  const int msk = A.L - 1;
  double x[RPT], r64[RPT], b[RPT];
#pragma unroll
  for (int e = 0; e < RPT; ++e) {
    x[e] = b[e] = 0.0;
    if (row[e] < 0) continue;
    b[e] = A.b[(int64_t)row[e] * R + rhs];
    if (A.warm) {  // cubic extrapolation of the last four currents (zero before step 0)
      const double* J = A.ring + (int64_t)row[e] * A.L * R + rhs;
      const int s = A.alpha - 2;
      const double j1 = s >= 0 ? J[(s & msk) * R] : 0.0, j2 = s >= 1 ? J[((s - 1) & msk) * R] : 0.0;
      const double j3 = s >= 2 ? J[((s - 2) & msk) * R] : 0.0, j4 = s >= 3 ? J[((s - 3) & msk) * R] : 0.0;
      x[e] = 4.0 * j1 - 6.0 * j2 + 4.0 * j3 - j4;
    }
  }
  // r = b - Z0 y in FP64, y published through w (a barrier before it is read)
  auto residual = [&](const double(&y)[RPT], double* w, double(&r)[RPT]) {
#pragma unroll
    for (int e = 0; e < RPT; ++e)
      if (pos[e] >= 0) w[pos[e]] = y[e];
    S.sync();
    sc_spmv<RPT>(LdZ64{A.zval, A.zcol, w}, zb, ztot, zends, lane, r);
#pragma unroll
    for (int e = 0; e < RPT; ++e) r[e] = row[e] >= 0 ? b[e] - r[e] : 0.0;
  };
  // the sums of r^2 and w^2 over all rows
  auto norm2 = [&](const double(&r)[RPT], const double(&w)[RPT], double& rr, double& ww) {
    rr = ww = 0.0;
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      rr += r[e] * r[e];
      ww += w[e] * w[e];
    }
    S.sums64(rr, ww);
  };
  double rr = 0.0, bb = 0.0;
  int inner_total = 0;
  bool conv = false;
  // The start: the extrapolation; with warm 2 also the caller's guess in A.x,
  // kept only if its FP64 residual is smaller (a NaN never is).
  // A residual that is carried on (r -= Z0 d) misses the rounding of x, half an
  // ulp a pass, and that of Z0 d in double-float, 2^-43 with a row's sum; over four
  // passes |missed|^2 <= 2^-101 zn2 (|x|^2 + 2^18 sum |d|^2).  It decides only where the
  // tolerance holds with that added, and b - Z0 x is formed anew in FP64 where it does
  // not.  (Few FP64 operations: each costs a CTA 0.12 us.)
  constexpr int kScCarry = 4;
  bool anew = true;
  int passes = 0;  // carried on since the last FP64 residual, at 2^k0 with
  float dd = 0.f;  // this thread's share of sum |d|^2 / 4^k0 over them
  int k0 = 0;
  bool last = false;  // the correction was made for the tolerance: only then is |missed| summed
  double tol2bb = 0.0;
#pragma unroll 1
  for (int outer = -1;; ++outer) {
    const bool carried = !anew && passes < kScCarry && rr <= 0x1p-16 * bb;
    anew = false;
    if (!carried) {
      residual(x, w64, r64);
      norm2(r64, b, rr, bb);
      tol2bb = A.tol * A.tol * bb;
      passes = 0;
      dd = 0.f;
    } else {
      double zd[RPT];
      sc_spmv<RPT>(LdZdf{A.zhi, A.zlo, A.zcol, sc_X}, zb, ztot, zends, lane, zd);
      const int kx = max((((__double2hiint(rr) >> 20) & 0x7ff) - 1023) >> 1, -500);
      const double sc = __hiloint2double((1023 + kx) << 20, 0);
#pragma unroll
      for (int e = 0; e < RPT; ++e) r64[e] = row[e] >= 0 ? r64[e] - sc * zd[e] : 0.0;
      ++passes;
      double nr = 0.0, xx = 0.0;
#pragma unroll
      for (int e = 0; e < RPT; ++e) nr += r64[e] * r64[e];
      if (last) {
        xx = (double)(0x1p18f * dd) * __hiloint2double((1023 + 2 * k0) << 20, 0);
#pragma unroll
        for (int e = 0; e < RPT; ++e) xx += x[e] * x[e];
      }
      S.sums64(nr, xx);
      rr = nr;
      if (rr <= tol2bb && (!last || rr + 0x1p-101 * A.zn2 * xx > 0.5 * tol2bb)) {
        anew = true;
        --outer;
        continue;
      }
    }
    if (outer < 0 && A.warm == 2) {
      double g[RPT], rg[RPT], gg, b2;
#pragma unroll
      for (int e = 0; e < RPT; ++e) g[e] = row[e] >= 0 ? A.x[(int64_t)row[e] * R + rhs] : 0.0;
      residual(g, w64 + A.npad, rg);
      norm2(rg, b, gg, b2);
      const bool keep = gg < rr;
      if (keep) {
        rr = gg;
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
          x[e] = g[e];
          r64[e] = rg[e];
        }
      }
      if (S.rank == 0 && threadIdx.x == 0) atomicAdd(&A.status[keep ? 8 : 9], 1);
    }
    if (rr <= tol2bb) {
      conv = true;
      break;
    }
    if (outer == 7 || inner_total >= A.maxit) break;
    if (!(rr < 1.7e308)) {  // non-finite data: so is the result
#pragma unroll
      for (int e = 0; e < RPT; ++e) x[e] = __longlong_as_double(0x7ff8000000000000LL);
      break;
    }
    // scale 2^k, k the exponent of |r|: the inner right-hand side has norm in [1, 2)
    const int kx = max((((__double2hiint(rr) >> 20) & 0x7ff) - 1023) >> 1, -500);
    const double sc = __hiloint2double((1023 + kx) << 20, 0), inv = __hiloint2double((1023 - kx) << 20, 0);
    // u: r, then s = r - alpha v, of each iteration
    float u[RPT], rh[RPT], p[RPT], v[RPT], y[RPT], w[RPT], d[4];
    // inner target: the reduction that brings the FP64 residual to half the outer
    // tolerance, within [1e-5, 0.5] (1e-5: what FP32 reliably reaches)
    const float rin = (float)(rr * inv * inv);
    const float want2 = 0.25f * (float)(tol2bb * inv * inv) / rin;
    const float tin2 = fminf(fmaxf(want2, (float)kScInner2), 0.25f) * rin;
    last = want2 >= (float)kScInner2;
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      u[e] = rh[e] = p[e] = (float)(r64[e] * inv);
      v[e] = y[e] = 0.f;
    }
    push(p);  // X is free: the barrier of the last sums lies behind every gather
    S.sync();
    float rho = 0.f, alp = 1.f;
    int half = 0, left = kScInnerMax;
    bool first = true;
#pragma unroll 1
    for (;;) {
      if (half == 0) {
        if (inner_total >= A.maxit || left-- == 0) break;
        ++inner_total;
      }
      sc_spmv<RPT>(LdA{A.aval, A.acol, sc_X}, ab, atot, aends, lane, w);
      float q0 = 0.f, q1 = 0.f, q2 = 0.f, q3 = 0.f;
#pragma unroll
      for (int e = 0; e < RPT; ++e) {
        q0 = fmaf(rh[e], w[e], q0);
        q1 = fmaf(u[e], u[e], q1);
        q2 = fmaf(u[e], w[e], q2);
        q3 = fmaf(w[e], w[e], q3);
      }
      S.dots4(q0, q1, q2, q3, d);
      if (half == 0) {
        if (first) rho = d[1];  // rh = r
        first = false;
        if (d[0] == 0.f || rho == 0.f) break;
        alp = rho / d[0];
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
          v[e] = w[e];
          y[e] = fmaf(alp, p[e], y[e]);
          u[e] = fmaf(-alp, w[e], u[e]);
        }
        // |s|^2 from the same sums: the half step may end the inner solve
        if (d[1] - alp * (2.f * d[2] - alp * d[3]) <= tin2) break;
        push(u);
      } else {
        if (d[3] == 0.f) break;
        const float om = d[2] / d[3];
        // (rh, s) = 0 by the choice of alpha
        const float rho_new = -om * d[0], beta = (rho_new / rho) * (alp / om);
        rho = rho_new;
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
          y[e] = fmaf(om, u[e], y[e]);
          u[e] = fmaf(-om, w[e], u[e]);
          p[e] = fmaf(beta, fmaf(-om, v[e], p[e]), u[e]);
        }
        if (om == 0.f || d[1] - om * (2.f * d[2] - om * d[3]) <= tin2) break;
        push(p);
      }
      half ^= 1;
      S.sync();
    }
    // d = P y, x += 2^k d; every gather of X lies behind the last sums' barrier
    push(y);
    S.sync();
    sc_spmv<RPT>(LdA{A.pval, A.pcol, sc_X}, pb, ptot, pends, lane, y);
#pragma unroll
    for (int e = 0; e < RPT; ++e) x[e] += sc * (double)y[e];
    float yy = 0.f;
#pragma unroll
    for (int e = 0; e < RPT; ++e) yy = fmaf(y[e], y[e], yy);
    if (passes == 0) k0 = kx;
    dd = fmaf(ldexpf(1.f, max(2 * (kx - k0), -120)), yy, dd);
    if (rr <= 0x1p-16 * bb) {
      S.sync();  // every CTA has gathered y
      push(y);
      S.sync();
    }
  }
#pragma unroll
  for (int e = 0; e < RPT; ++e)
    if (row[e] >= 0) {
      A.x[(int64_t)row[e] * R + rhs] = x[e];
      const int64_t o = ((int64_t)row[e] * A.L + ((A.alpha - 1) & msk)) * R + rhs;
      A.ring[o] = x[e];
      if (A.rs) A.rs[o] = split_pair(x[e]);
      if (A.rf) A.rf[o] = (float)x[e];
    }
  if (S.rank == 0 && threadIdx.x == 0) {
    if (R == 1) {
      A.status[0] = inner_total;
      A.status[6] = 0;
      A.status[1] = conv ? 1 : 0;
      A.status[2] += conv ? 0 : 1;
      A.status[3] += inner_total;
      A.resid[0] = bb > 0 ? sqrt(rr / bb) : 0.0;
    } else {
      // status[0] (the most iterations of any right-hand side) is zero at launch;
      // the last cluster to finish publishes the step's verdict
      atomicMax(&A.status[0], inner_total);
      if (!conv) atomicAdd(&A.status[4], 1);
      __threadfence();
      if (atomicAdd(&A.status[5], 1) == R - 1) {
        __threadfence();
        const int miss = atomicExch(&A.status[4], 0), it = atomicAdd(&A.status[0], 0);
        A.status[6] = 0;
        A.status[1] = miss == 0 ? 1 : 0;
        A.status[2] += miss == 0 ? 0 : 1;
        A.status[3] += it;
        A.status[5] = 0;
      }
    }
  }
  S.sync();  // no CTA leaves while another may still store into its shared memory
}

// ---------------------------------------------------------------------------
// The solve of the FP32 and 24-bit direct marches: the arithmetic of k_bicgstab
// (solve.cu) rounding for rounding, so that their currents stay what they are (see
// tdbem_z0_f32), in the exchange form above.  What k_bicgstab spent its time on is
// gone: every thread's FP64 divisions and square roots (one warp computes the
// scalars now), two FP64 shuffle trees per pair of sums (folded into one tree with
// the same additions), Krylov vectors in L2 and one dependent gather after the other
// (registers, whole copies in shared memory, four blocks of entries in flight).
// Rows stay in edge order, thread t of CTA k owning the rows k ceil(ne / CTAs) + t,
// + 512, ..; a row's entries go to four chains as there (chain m of the entries
// m, m + 4, .., the last ne mod 4 to chain 0), one lane each.
struct BxArgs {
  const int32_t *zb, *ze;    // first block of a warp [cs * 16], block ends of its passes [cs * 16][passes]
  const float4* z32;
  const double2* z64;
  const uint2* zcol;
  const int32_t* pcol;       // triangle blocks [5][ne]
  const float* pval;
  const double* b;
  double* x;
  double* ring;
  float2* rs;
  int32_t L, alpha, warm, rows, passes, ne, maxit;
  double tol;
  int32_t* status;
  double* resid;
};
constexpr int kBxPc = 5;

struct LdB32 {  // FP32, one chain per lane
  const float4* v;
  const uint2* c;
  const float* X;
  struct Block {
    float4 v;
    uint2 c;
  };
  struct Acc {
    float a;
    __device__ __forceinline__ void zero() { a = 0.f; }
    __device__ __forceinline__ float fold() {
      float s = a;
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      return s + __shfl_xor_sync(0xffffffffu, s, 2);
    }
  };
  __device__ __forceinline__ void seek(int b, int lane) {
    v += (int64_t)b * 32 + lane;
    c += (int64_t)b * 32 + lane;
  }
  __device__ __forceinline__ void skip() {
    v += kScDepth * 32;
    c += kScDepth * 32;
  }
  __device__ __forceinline__ void load(Block& k, int i) const {
    k.v = __ldg(v + i * 32);
    k.c = __ldg(c + i * 32);
  }
  __device__ __forceinline__ void mul(const Block& k, Acc& s) const {
    s.a = fmaf(k.v.x, X[k.c.x & 0xffff], s.a);
    s.a = fmaf(k.v.y, X[k.c.x >> 16], s.a);
    s.a = fmaf(k.v.z, X[k.c.y & 0xffff], s.a);
    s.a = fmaf(k.v.w, X[k.c.y >> 16], s.a);
  }
};

// The warp's rows times the gathered vector into out[local row] (shared memory).
template <class Ld, class Out>
__device__ __forceinline__ void bx_spmv(Ld ld, int b, int tot, int ends, int gpc, int warp, int lane, Out* out) {
  typename Ld::Block buf[kScDepth];
  asm volatile("" : "+r"(b));
  int left = tot - b, g = warp, gend = __shfl_sync(0xffffffffu, ends, 0), gleft = gend - b, j = 0;
  ld.seek(b, lane);
#pragma unroll
  for (int i = 0; i < kScDepth; ++i) ld.load(buf[i], i);
  typename Ld::Acc acc;
  acc.zero();
  for (; left > 0; left -= kScDepth) {
    ld.skip();
#pragma unroll
    for (int i = 0; i < kScDepth; ++i) {
      ld.mul(buf[i], acc);
      ld.load(buf[i], i);
      if (--gleft == 0) {
        const Out s = acc.fold();
        acc.zero();
        // (the zero blocks behind a warp's last group may close a pass without one)
        if ((lane & 3) == 0 && g < gpc) out[g * 8 + (lane >> 2)] = s;
        g += kScWarps;
        const int g2 = __shfl_sync(0xffffffffu, ends, ++j & 31);
        gleft = g2 - gend;
        gend = g2;
      }
    }
  }
}

struct __align__(16) BxShared {  // (sums are sent as 16-byte pairs)
  double red[kScWarps][2];
  double slots[2][16][2];
  double rr, inv, sc;
  float alf, omf, beta;
  int stop;
};

template <int RPT>
__global__ void __launch_bounds__(kScThreads) k_bicgstab_x(const BxArgs A) {
  extern __shared__ __align__(16) float bx_sm[];
  __shared__ BxShared sm;
  int nb, rank;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(nb));
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, W = rank * kScWarps + warp;
  const int ne = A.ne, r0 = rank * A.rows, nr = max(0, min(ne - r0, A.rows));
  const int nx = (ne + 3) & ~3, gpc = (A.rows + 7) / 8;
  float *Xa = bx_sm, *Xb = bx_sm + nx;                     // p then s; P p then P s
  double* prod = reinterpret_cast<double*>(bx_sm + 2 * nx);  // a product's rows
  float* prodf = reinterpret_cast<float*>(prod);
  const int zb = A.zb[W], zends = lane < A.passes ? A.ze[W * A.passes + lane] : 0;
  const int ztot = __shfl_sync(0xffffffffu, zends, A.passes - 1);
  auto sync = [&]() {
    if (nb == 1) {
      __syncthreads();
    } else {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  };
  auto own = [&](int e) { return t + e * kScThreads < nr; };
  auto row = [&](int e) { return r0 + t + e * kScThreads; };
  auto push = [&](float* X, const float(&v)[RPT]) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(X);
#pragma unroll 1
    for (int k = 0; k < nb; ++k) {
      int r = rank + k;
      if (r >= nb) r -= nb;
      const uint32_t d = sc_mapa(a, r);
#pragma unroll
      for (int e = 0; e < RPT; ++e)
        if (own(e)) sc_st(d + 4 * row(e), v[e]);
    }
  };
  // Sums over all rows of a and b, with the additions of the tree that k_bicgstab
  // takes for either; warp 0 gets both and runs f on them before the CTA goes on.
  int phase = 0;
  auto sums = [&](double a, double b, auto f) {
    const bool up = lane & 16;
    double k = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) k += __shfl_down_sync(0xffffffffu, k, o);
    if ((lane & 15) == 0) sm.red[warp][lane >> 4] = k;
    __syncthreads();
    const int ph = phase++ & 1;
    if (warp == 0) {
      double u = sm.red[lane & 15][lane >> 4];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
      const double u0 = __shfl_sync(0xffffffffu, u, 0), u1 = __shfl_sync(0xffffffffu, u, 16);
      const uint32_t dst = sc_mapa((uint32_t)__cvta_generic_to_shared(&sm.slots[ph][rank][0]), lane < nb ? lane : 0);
      if (lane < nb) sc_st64(dst, u0, u1);
    }
    sync();
    if (warp == 0) {
      double u = (lane & 15) < nb ? sm.slots[ph][lane & 15][lane >> 4] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
      f(__shfl_sync(0xffffffffu, u, 0), __shfl_sync(0xffffffffu, u, 16));
    }
    __syncthreads();
  };
  auto spmv32 = [&](float(&v)[RPT]) {  // Z0 Xb
    bx_spmv(LdB32{A.z32, A.zcol, Xb}, zb, ztot, zends, gpc, warp, lane, prodf);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < RPT; ++e) v[e] = own(e) ? prodf[t + e * kScThreads] : 0.f;
  };
  auto spmv64 = [&](const double* x, double(&v)[RPT]) {  // Z0 x, x in global memory
    bx_spmv(LdZ64{A.z64, A.zcol, x}, zb, ztot, zends, gpc, warp, lane, prod);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < RPT; ++e) v[e] = own(e) ? prod[t + e * kScThreads] : 0.0;
    __syncthreads();  // prod is written again before the next barrier of the sums
  };
  auto precond = [&](float(&v)[RPT]) {  // the triangle blocks times Xa
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      float s = 0.f;
      if (own(e)) {
        const int i = row(e);
#pragma unroll
        for (int k = 0; k < kBxPc; ++k)
          s += __ldg(A.pval + (int64_t)k * ne + i) * Xa[__ldg(A.pcol + (int64_t)k * ne + i)];
      }
      v[e] = s;
    }
  };
  const int L = A.L, msk = A.L - 1;
  double x[RPT], b[RPT], r64[RPT], z[RPT];
#pragma unroll
  for (int e = 0; e < RPT; ++e) {
    b[e] = x[e] = 0.0;
    if (!own(e)) continue;
    b[e] = A.b[row(e)];
    double x0 = 0.0;
    if (A.warm) {
      const double* J = A.ring + (int64_t)row(e) * L;
      int bt = A.alpha - 2;  // J^{alpha-2}, J^{alpha-3}, ... (zero before step 0)
      double j1 = bt >= 0 ? J[bt & msk] : 0.0, j2 = bt >= 1 ? J[(bt - 1) & msk] : 0.0;
      double j3 = bt >= 2 ? J[(bt - 2) & msk] : 0.0, j4 = bt >= 3 ? J[(bt - 3) & msk] : 0.0;
      x0 = 4.0 * j1 - 6.0 * j2 + 4.0 * j3 - j4;
    }
    x[e] = x0;
    if (A.warm != 2) A.x[row(e)] = x0;
  }
  sync();
  if (A.warm == 2) {
    // keep the guess in A.x only if its FP64 residual is smaller (a NaN never is)
    double g[RPT], qg = 0.0, qc = 0.0;
    spmv64(A.x, z);
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      g[e] = own(e) ? A.x[row(e)] : 0.0;
      const double rg = b[e] - z[e];
      if (own(e)) qg += rg * rg;
    }
    sync();  // every CTA has read the guess
#pragma unroll
    for (int e = 0; e < RPT; ++e)
      if (own(e)) A.x[row(e)] = x[e];
    sync();
    spmv64(A.x, z);
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      const double rc = b[e] - z[e];
      if (own(e)) qc += rc * rc;
    }
    sums(qg, qc, [&](double a, double c) { sm.stop = a < c ? 1 : 0; });
    const bool keep = sm.stop;
    if (keep) {
#pragma unroll
      for (int e = 0; e < RPT; ++e) {
        x[e] = g[e];
        if (own(e)) A.x[row(e)] = g[e];
      }
    }
    if (rank == 0 && t == 0) A.status[keep ? 8 : 9] += 1;
    sync();
  }
  // scalars of warp 0 (its lanes hold the same values)
  double bb = -1.0, rr = 0.0, rho = 0.0, rho_old = 1.0, alp = 1.0, om = 1.0, want2 = 0.0, tin2 = 0.0;
  int inner_total = 0;
  bool conv = false;
#pragma unroll 1
  for (int outer = 0; outer < 8; ++outer) {
    double q0 = 0.0, q1 = 0.0;
    spmv64(A.x, z);
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      const double ri = b[e] - z[e];
      r64[e] = own(e) ? ri : 0.0;
      if (own(e)) {
        q0 += ri * ri;
        q1 += b[e] * b[e];
      }
    }
    sums(q0, q1, [&](double a, double c) {
      rr = a;
      if (bb < 0) bb = c;
      sm.stop = rr <= A.tol * A.tol * bb;
      sm.inv = 1.0 / sqrt(rr);
      sm.sc = sqrt(rr);
      want2 = 0.25 * A.tol * A.tol * bb / rr;
    });
    if (sm.stop) {
      conv = true;
      break;
    }
    if (inner_total >= A.maxit) break;
    const double inv = sm.inv, sc = sm.sc;
    float r[RPT], rh[RPT], p[RPT], v[RPT], s[RPT], tt[RPT], ph[RPT], sh[RPT], d[RPT];
    q0 = 0.0;
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      float ri = (float)(r64[e] * inv);  // unit-norm right-hand side
      r[e] = rh[e] = own(e) ? ri : 0.f;
      p[e] = v[e] = d[e] = 0.f;
      if (own(e)) q0 += (double)ri * ri;
    }
    sums(q0, 0.0, [&](double a, double) {
      rho = a;
      rho_old = alp = om = 1.0;
      tin2 = fmin(fmax(want2, kScInner2), 0.25) * a;
      sm.stop = rho == 0.0;
      sm.beta = (float)((rho / rho_old) * (alp / om));
      sm.omf = (float)om;
    });
#pragma unroll 1
    for (int it = 0; it < kScInnerMax && inner_total < A.maxit; ++it) {
      ++inner_total;
      if (sm.stop) break;  // rho = 0
      const float beta = sm.beta;
      float omf = sm.omf;
#pragma unroll
      for (int e = 0; e < RPT; ++e) p[e] = r[e] + beta * (p[e] - omf * v[e]);
      push(Xa, p);
      sync();
      precond(ph);
      push(Xb, ph);
      sync();
      spmv32(v);
      q0 = 0.0;
#pragma unroll
      for (int e = 0; e < RPT; ++e)
        if (own(e)) q0 += (double)(rh[e] * v[e]);
      sums(q0, 0.0, [&](double a, double) {
        sm.stop = a == 0.0;
        alp = rho / a;
        sm.alf = (float)alp;
      });
      if (sm.stop) break;
      const float alf = sm.alf;
      q0 = 0.0;
#pragma unroll
      for (int e = 0; e < RPT; ++e) {
        float si = r[e] - alf * v[e];
        s[e] = si;
        if (own(e)) q0 += (double)(si * si);
      }
      push(Xa, s);  // published by the barrier of the sums
      sums(q0, 0.0, [&](double a, double) { sm.stop = a <= tin2; });
      if (sm.stop) {
#pragma unroll
        for (int e = 0; e < RPT; ++e) d[e] += alf * ph[e];
        break;
      }
      precond(sh);
      push(Xb, sh);
      sync();
      spmv32(tt);
      q0 = q1 = 0.0;
#pragma unroll
      for (int e = 0; e < RPT; ++e)
        if (own(e)) {
          q0 += (double)(tt[e] * s[e]);
          q1 += (double)(tt[e] * tt[e]);
        }
      sums(q0, q1, [&](double a, double c) {
        sm.stop = c == 0.0;
        om = a / c;
        sm.omf = (float)om;
      });
      if (sm.stop) break;
      omf = sm.omf;
      q0 = q1 = 0.0;
#pragma unroll
      for (int e = 0; e < RPT; ++e) {
        d[e] += alf * ph[e] + omf * sh[e];
        float ri = s[e] - omf * tt[e];
        r[e] = ri;
        if (own(e)) {
          q0 += (double)(ri * ri);
          q1 += (double)(rh[e] * ri);
        }
      }
      sums(q0, q1, [&](double a, double c) {
        rho_old = rho;
        rho = c;
        sm.stop = (a <= tin2 || om == 0.0 ? 1 : 0) | (rho == 0.0 ? 2 : 0);
        sm.beta = (float)((rho / rho_old) * (alp / om));
      });
      if (sm.stop & 1) break;
    }
#pragma unroll
    for (int e = 0; e < RPT; ++e) {
      x[e] += sc * (double)d[e];
      if (own(e)) A.x[row(e)] = x[e];
    }
    sync();
  }
#pragma unroll
  for (int e = 0; e < RPT; ++e)
    if (own(e)) {
      const int64_t o = (int64_t)row(e) * L + ((A.alpha - 1) & msk);
      A.ring[o] = x[e];
      if (A.rs) A.rs[o] = split_pair(x[e]);
    }
  if (rank == 0 && t == 0) {
    A.status[0] = inner_total;
    A.status[6] = 0;
    A.status[1] = conv ? 1 : 0;
    A.status[2] += conv ? 0 : 1;
    A.status[3] += inner_total;
    A.resid[0] = bb > 0 ? sqrt(rr / bb) : 0.0;
  }
  sync();  // no CTA leaves while another may still store into its shared memory
}

struct ScPlan {
  int cs = 0, gpc = 0, passes = 0, npad = 0;
  int32_t *perm = nullptr, *ab = nullptr, *ae = nullptr, *zb = nullptr, *ze = nullptr, *pb = nullptr, *pe = nullptr;
  float4 *aval = nullptr, *zhi = nullptr, *zlo = nullptr, *pval = nullptr;
  double2* zval = nullptr;
  uint2 *acol = nullptr, *zcol = nullptr, *pcol = nullptr;
  double* w64 = nullptr;
  double zn2 = 0.0;
  bool bx = false;                 // k_bicgstab_x: rows per CTA, Z0's FP32 blocks, the triangle blocks are the context's
  int rows = 0;
  float4* z32 = nullptr;
};

}  // namespace tdbem

using namespace tdbem;

using ScFn = void (*)(ScArgs);
static ScFn sc_fn(int passes) {
  return passes <= 4 ? k_solve_cluster<1> : passes <= 8 ? k_solve_cluster<2> : k_solve_cluster<6>;
}

static size_t sc_smem(const ScPlan& P) { return (size_t)P.npad * sizeof(float); }

static void sc_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int cs, int ctas, size_t smem, cudaStream_t st) {
  *cfg = {};
  cfg->gridDim = dim3(ctas);
  cfg->blockDim = dim3(kScThreads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = cs;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

// One matrix in blocks of 8 rows x 16 entries along the order `slot` of the
// groups; put(block * 128 + place, entry) stores an entry.
template <class Len, class Put>
static void sc_blocks(const ScPlan& P, const std::vector<int32_t>& perm, Len len, Put put, std::vector<int32_t>* begin,
                      std::vector<int32_t>* end, int32_t* nblk) {
  int32_t b = 0;
  begin->assign(P.cs * kScWarps, 0);
  end->assign(P.cs * kScWarps * P.passes, 0);
  for (int k = 0; k < P.cs; ++k)
    for (int w = 0; w < kScWarps; ++w) {
      (*begin)[k * kScWarps + w] = b;
      for (int j = 0; j < P.passes; ++j) {
        const int g = j * kScWarps + w;
        if (g < P.gpc) {
          const int64_t p0 = ((int64_t)k * P.gpc + g) * 8;
          int most = 1;
          for (int t = 0; t < 8; ++t)
            if (perm[p0 + t] >= 0) most = std::max(most, (int)len(perm[p0 + t]));
          const int nb = (most + 15) / 16;
          for (int t = 0; t < 8; ++t)
            if (perm[p0 + t] >= 0)
              for (int m = 0; m < len(perm[p0 + t]); ++m)
                put((int64_t)(b + m / 16) * 128 + t * 16 + m % 16, perm[p0 + t], m);
          b += nb;
        }
        if (j == P.passes - 1)  // whole prefetch rounds: zero blocks behind the last group
          while ((b - (*begin)[k * kScWarps + w]) % kScDepth) ++b;
        (*end)[(k * kScWarps + w) * P.passes + j] = b;
      }
    }
  *nblk = b + kScDepth;  // loads run ahead of the last warp's end
}

template <class T>
static tdbem_status sc_upload(tdbem_ctx* c, T** d, const std::vector<T>& h) {
  tdbem_status s = c->dalloc(d, h.size());
  if (s) return s;
  // on the context's stream and waited for: the host array goes out of scope
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return TDBEM_OK;
}

// A CSR matrix in blocks of the plan's order: FP32 values (and, with lo, the low
// parts of (hi, lo) pairs; with f64, the FP64 values), positions, block runs.
struct ScMat {
  const std::vector<int64_t>& ptr;
  const std::vector<int32_t>& col;
  const std::vector<double>& val;
};
static tdbem_status sc_matrix(tdbem_ctx* c, const ScPlan& P, const std::vector<int32_t>& perm,
                              const std::vector<int32_t>& at, const ScMat& M, int32_t** begin, int32_t** end,
                              float4** hi, float4** lo, double2** f64, uint2** col) {
  std::vector<int32_t> b, e;
  int32_t n = 0;
  auto len = [&](int i) { return (int)(M.ptr[i + 1] - M.ptr[i]); };
  sc_blocks(P, perm, len, [](int64_t, int, int) {}, &b, &e, &n);
  std::vector<float4> vh((size_t)n * 32, make_float4(0, 0, 0, 0)), vl(lo ? (size_t)n * 32 : 0, make_float4(0, 0, 0, 0));
  std::vector<double2> vd(f64 ? (size_t)n * 64 : 0, make_double2(0, 0));
  std::vector<uint2> vc((size_t)n * 32, make_uint2(0, 0));
  float *fh = (float*)vh.data(), *fl = (float*)vl.data();
  double* fd = (double*)vd.data();
  uint16_t* fc = (uint16_t*)vc.data();
  sc_blocks(P, perm, len, [&](int64_t o, int i, int m) {
    const double z = M.val[M.ptr[i] + m];
    fh[o] = (float)z;
    if (lo) fl[o] = (float)(z - (double)fh[o]);
    if (f64) fd[o] = z;
    fc[o] = (uint16_t)at[M.col[M.ptr[i] + m]];
  }, &b, &e, &n);
  tdbem_status s;
  if ((s = sc_upload(c, begin, b)) || (s = sc_upload(c, end, e)) || (s = sc_upload(c, hi, vh)) ||
      (s = sc_upload(c, col, vc)) || (lo && (s = sc_upload(c, lo, vl))) || (f64 && (s = sc_upload(c, f64, vd))))
    return s;
  return TDBEM_OK;
}

// Row i of P: row 0 of the inverse of the block of Z0 among J = {i, then the
// columns of row i's largest entries}, at most kScK in all; the solution of
// B^T y = e_0 by Gauss-Jordan elimination with partial pivoting in FP32, lane r
// holding row r of B^T.  A block without a usable pivot gives the reciprocal of
// the diagonal.  One warp per row.
constexpr int kLiWarps = 8;

__global__ void __launch_bounds__(kLiWarps * 32) k_local_inverse(const int32_t* ptr, const int32_t* col,
                                                                const double* val, int32_t ne, int32_t* pcol,
                                                                float* pval) {
  __shared__ float Bs[kLiWarps][32][33];
  __shared__ int Js[kLiWarps][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kLiWarps + w;
  if (i >= ne) return;  // whole warps; only warp-wide synchronisation below
  const int p0 = ptr[i], p1 = ptr[i + 1];
  // the largest entries, one after the other: each round takes the largest below the last taken
  // (ties: the smaller index first)
  int n = 1, myj = lane == 0 ? i : -1, last = -1;
  float lastv = 3e38f;
  for (; n < kScK; ++n) {
    float bv = 0.f;
    int bk = -1;
    for (int k = p0 + lane; k < p1; k += 32) {
      const float v = fabsf((float)val[k]);
      if (col[k] == i || v == 0.f) continue;
      const bool below = v < lastv || (v == lastv && k > last);
      if (below && v > bv) {  // the lane's own entries ascend: the first of equals stays
        bv = v;
        bk = k;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
      if (ok >= 0 && (ov > bv || (ov == bv && ok < bk) || bk < 0)) {
        bv = ov;
        bk = ok;
      }
    }
    if (bk < 0) break;
    last = bk;
    lastv = bv;
    if (lane == n) myj = col[bk];
  }
  Js[w][lane] = myj;
  for (int r = 0; r < 32; ++r) Bs[w][r][lane] = r == lane && lane >= n ? 1.f : 0.f;
  __syncwarp();
  // Bs[r][k] = Z0[J_k][J_r]
  float diag = 1.f;
  for (int k = 0; k < n; ++k) {
    const int row = Js[w][k];
    for (int q = ptr[row] + lane; q < ptr[row + 1]; q += 32) {
      const int cc = col[q];
      for (int r = 0; r < n; ++r)
        if (Js[w][r] == cc) Bs[w][r][k] = (float)val[q];
    }
  }
  __syncwarp();
  if (Bs[w][0][0] != 0.f) diag = Bs[w][0][0];
  float rhs = lane == 0 ? 1.f : 0.f;
  int mine = -1;  // the column this row was the pivot of
  bool ok = true;
  for (int k = 0; k < 32 && ok; ++k) {
    float v = mine < 0 ? fabsf(Bs[w][lane][k]) : -1.f;
    int who = lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, v, o);
      const int oi = __shfl_xor_sync(0xffffffffu, who, o);
      if (ov > v || (ov == v && oi < who)) {
        v = ov;
        who = oi;
      }
    }
    ok = v > 0.f && v < 3e38f;  // the same in every lane
    if (!ok) break;
    const float piv = Bs[w][who][k];
    const float prhs = __shfl_sync(0xffffffffu, rhs, who);
    if (lane == who) {
      mine = k;
    } else {
      const float f = Bs[w][lane][k] / piv;
      for (int m = k + 1; m < 32; ++m) Bs[w][lane][m] = fmaf(-f, Bs[w][who][m], Bs[w][lane][m]);
      rhs = fmaf(-f, prhs, rhs);
    }
    __syncwarp();
  }
  // y_k of the row that was column k's pivot
  float y = 0.f;
  if (ok) {
    const float u = rhs / Bs[w][lane][mine];
    for (int r = 0; r < 32; ++r) {
      const int k = __shfl_sync(0xffffffffu, mine, r);
      const float v = __shfl_sync(0xffffffffu, u, r);
      if (lane == k) y = v;
    }
    ok = __all_sync(0xffffffffu, fabsf(y) < 3e38f);
  }
  if (!ok) y = lane == 0 ? 1.f / diag : 0.f;
  pcol[(int64_t)i * kScK + lane] = myj;
  pval[(int64_t)i * kScK + lane] = lane < n ? y : 0.f;
}

// The plan's arrays for a preconditioner P: A = Z0 P and the order of its rows.
static tdbem_status sc_arrays(tdbem_ctx* c, ScPlan* out, const ScMat& Z, const ScMat& M) {
  ScPlan& P = *out;
  const int ne = (int)c->ne;
  const std::vector<int64_t>&np = Z.ptr, &pp = M.ptr;
  const std::vector<int32_t>&nc = Z.col, &pc = M.col;
  const std::vector<double>&nv = Z.val, &pv = M.val;
  tdbem_status s;
  // A = Z0 P, row by row
  std::vector<int64_t> ap(ne + 1, 0);
  std::vector<int32_t> ac, at(ne, -1), rowc;
  std::vector<double> av, acc(ne, 0.0);
  for (int i = 0; i < ne; ++i) {
    rowc.clear();
    for (int64_t k = np[i]; k < np[i + 1]; ++k) {
      const double z = nv[k];
      const int j = nc[k];
      for (int64_t m = pp[j]; m < pp[j + 1]; ++m) {
        const int l = pc[m];
        if (at[l] != i) {
          at[l] = i;
          acc[l] = 0.0;
          rowc.push_back(l);
        }
        acc[l] += z * pv[m];
      }
    }
    for (int l : rowc)
      if (std::fabs(acc[l]) > kScDrop) {
        ac.push_back(l);
        av.push_back(acc[l]);
      }
    ap[i + 1] = (int64_t)ac.size();
  }
  // order: rows by their blocks of A, longest first (stable), in groups of 8 dealt over the CTAs
  std::vector<int32_t> ord(ne);
  for (int i = 0; i < ne; ++i) ord[i] = i;
  std::stable_sort(ord.begin(), ord.end(), [&](int32_t a, int32_t b) {
    return (ap[a + 1] - ap[a] + 15) / 16 > (ap[b + 1] - ap[b] + 15) / 16;
  });
  std::vector<int32_t> perm(P.npad, -1), at_pos(ne);
  int next = 0;
  for (int j = 0; j < P.passes && next < ne; ++j)
    for (int u = 0; u < P.cs * kScWarps && next < ne; ++u) {
      const int f = j & 1 ? P.cs * kScWarps - 1 - u : u;  // there and back: long and short groups meet
      const int k = f % P.cs, g = j * kScWarps + f / P.cs;
      if (g >= P.gpc) continue;
      for (int t = 0; t < 8 && next < ne; ++t, ++next) {
        const int64_t p = ((int64_t)k * P.gpc + g) * 8 + t;
        perm[p] = ord[next];
        at_pos[ord[next]] = (int32_t)p;
      }
    }
  if ((s = sc_upload(c, &P.perm, perm)) ||
      (s = sc_matrix(c, P, perm, at_pos, {ap, ac, av}, &P.ab, &P.ae, &P.aval, nullptr, nullptr, &P.acol)) ||
      (s = sc_matrix(c, P, perm, at_pos, M, &P.pb, &P.pe, &P.pval, nullptr, nullptr, &P.pcol)) ||
      (s = sc_matrix(c, P, perm, at_pos, Z, &P.zb, &P.ze, &P.zhi, &P.zlo, &P.zval, &P.zcol)) ||
      (s = c->dalloc(&P.w64, 2 * (size_t)P.npad * c->R)))
    return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(P.w64, 0, 2 * (size_t)P.npad * c->R * sizeof(double), c->stream));
  return TDBEM_OK;
}

static void sc_drop(tdbem_ctx* c, ScPlan* P) {
  for (void* d : {(void*)P->perm, (void*)P->ab, (void*)P->ae, (void*)P->aval, (void*)P->acol, (void*)P->zb, (void*)P->ze,
                  (void*)P->zval, (void*)P->zhi, (void*)P->zlo, (void*)P->zcol, (void*)P->pb, (void*)P->pe,
                  (void*)P->pval, (void*)P->pcol, (void*)P->w64})
    if (d) c->dfree(d);
}

static ScArgs sc_args(const tdbem_ctx* c, const ScPlan& P) {
  ScArgs A = {};
  A.perm = P.perm;
  A.ab = P.ab;
  A.ae = P.ae;
  A.aval = P.aval;
  A.acol = P.acol;
  A.zb = P.zb;
  A.ze = P.ze;
  A.zval = P.zval;
  A.zhi = P.zhi;
  A.zlo = P.zlo;
  A.zcol = P.zcol;
  A.pb = P.pb;
  A.pe = P.pe;
  A.pval = P.pval;
  A.pcol = P.pcol;
  A.w64 = P.w64;
  A.gpc = P.gpc;
  A.passes = P.passes;
  A.npad = P.npad;
  A.ne = (int32_t)c->ne;
  A.zn2 = P.zn2;
  A.status = c->d_status;
  A.resid = c->d_dots;
  return A;
}

// Iterations that the plan takes to 1e-5 for one right-hand side of every frequency, kScTrial where that is not enough.
static tdbem_status sc_trial(tdbem_ctx* c, const ScPlan& P, int* its) {
  const int64_t ne = c->ne;
  std::vector<double> b(ne);
  uint64_t h = 1;
  for (double& v : b) {
    h = h * 6364136223846793005ull + 1442695040888963407ull;
    v = (double)(int64_t)h * 0x1p-63;
  }
  // d_work serves the solves that have no plan; the ring is one step long here
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(c->d_work, b.data(), ne * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_status, 0, 16 * sizeof(int32_t), c->stream));
  ScArgs A = sc_args(c, P);
  A.b = c->d_work;
  A.x = c->d_work + ne;
  A.ring = c->d_work + 2 * ne;
  A.L = 1;
  A.alpha = 1;
  A.R = 1;
  A.maxit = kScTrial;
  A.tol = 2e-5;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  sc_config(&cfg, &at, P.cs, P.cs, sc_smem(P), c->stream);
  TDBEM_CUDA_TRY(c, cudaLaunchKernelEx(&cfg, sc_fn(P.passes), A));
  int32_t st[2];
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(st, c->d_status, sizeof(st), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  *its = st[1] ? st[0] : kScTrial;
  return TDBEM_OK;
}

tdbem_status tdbem_sc_build(tdbem_ctx* c, int want, const std::vector<int32_t>& zp, const std::vector<int32_t>& zc,
                            const std::vector<double>& zv) {
  const int ne = (int)c->ne;
  ScPlan P;
  // Cluster size: the one of least cost among those the device schedules, at most
  // the wanted one.  An iteration costs about 8 us of barriers and latency (4.5 in a
  // single CTA, which has no cluster barriers) and 9 ns per row and CTA for the
  // products, whatever the number of clusters that run side by side; right-hand
  // sides beyond those queue.
  double best = 1e300;
  for (int cs = want; cs >= 1; cs >>= 1) {
    ScPlan T;
    T.cs = cs;
    T.gpc = ((ne + 7) / 8 + cs - 1) / cs;
    T.passes = (T.gpc + kScWarps - 1) / kScWarps;
    T.npad = cs * T.gpc * 8;
    if (T.passes > kScPasses || T.npad > 65535 || sc_smem(T) > 200 * 1024) break;
    const ScFn fn = sc_fn(T.passes);
    TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    sc_config(&cfg, &at, cs, cs, sc_smem(T), c->stream);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      continue;
    }
    const double cost = (double)((c->R + n - 1) / n) * ((cs > 1 ? 8.0 : 4.5) + 0.009 * ne / cs);
    if (cost < best) {
      best = cost;
      P = T;
    }
    if (c->p.solve_cluster > 0 && c->R == 1) break;  // the caller's choice
  }
  if (P.cs < 1) return TDBEM_OK;
  // Z0 without the stored zeros (pairs whose lag window holds lag 1 but whose
  // supports lie beyond c dt of each other: about 40% of the entries)
  std::vector<int64_t> np(ne + 1, 0);
  std::vector<int32_t> nc;
  std::vector<double> nv;
  nc.reserve(zc.size());
  nv.reserve(zc.size());
  for (int i = 0; i < ne; ++i) {
    for (int k = zp[i]; k < zp[i + 1]; ++k)
      if (zv[k] != 0.0) {
        nc.push_back(zc[k]);
        nv.push_back(zv[k]);
      }
    np[i + 1] = (int64_t)nc.size();
  }
  {
    std::vector<double> colsum(ne, 0.0);
    double most_row = 0.0, most_col = 0.0;
    for (int i = 0; i < ne; ++i) {
      double r = 0.0;
      for (int64_t k = np[i]; k < np[i + 1]; ++k) {
        r += std::fabs(nv[k]);
        colsum[nc[k]] += std::fabs(nv[k]);
      }
      most_row = std::max(most_row, r);
    }
    for (double v : colsum) most_col = std::max(most_col, v);
    P.zn2 = most_row * most_col;
  }
  const ScPlan base = P;
  const ScMat Z = {np, nc, nv};
  // P
  std::vector<int64_t> pp(ne + 1, 0);
  std::vector<int32_t> pc;
  std::vector<double> pv;
  tdbem_status s;
  if (c->p.precond == 1) {
    int32_t* d_pc = nullptr;
    float* d_pv = nullptr;
    const size_t n = (size_t)ne * kScK;
    if ((s = c->dalloc(&d_pc, n)) || (s = c->dalloc(&d_pv, n))) return s;
    k_local_inverse<<<(ne + kLiWarps - 1) / kLiWarps, kLiWarps * 32, 0, c->stream>>>(c->d_z0_ptr, c->d_z0_col,
                                                                                    c->d_z0_val, ne, d_pc, d_pv);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
    std::vector<int32_t> hc(n);
    std::vector<float> hv(n);
    TDBEM_CUDA_TRY(c, cudaMemcpyAsync(hc.data(), d_pc, n * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    TDBEM_CUDA_TRY(c, cudaMemcpyAsync(hv.data(), d_pv, n * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
    TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    c->dfree(d_pc);
    c->dfree(d_pv);
    for (int i = 0; i < ne; ++i) {
      for (int k = 0; k < kScK; ++k)
        if (hv[(size_t)i * kScK + k] != 0.f) {
          pc.push_back(hc[(size_t)i * kScK + k]);
          pv.push_back(hv[(size_t)i * kScK + k]);
        }
      pp[i + 1] = (int64_t)pc.size();
    }
  } else {
    for (int i = 0; i < ne; ++i) {
      double d = 0.0;
      for (int64_t k = np[i]; k < np[i + 1]; ++k)
        if (nc[k] == i) d = nv[k];
      pc.push_back(i);
      pv.push_back(d != 0.0 ? 1.0 / d : 1.0);
      pp[i + 1] = (int64_t)pc.size();
    }
  }
  // Rows of local inverses do best where Z0 couples near neighbours: 1 to 11 iterations to 1e-5 at time steps up to half
  // an edge length, on spheres and slivers.  At steps of many edge lengths Z0 is full, and where a sliver's
  // pole gathers more strong couplings than a row takes, the truncated blocks' inverses spoil it (UV
  // ellipsoid of 2880 RWG, steps of 32 edge lengths: 174 iterations against 66 with the triangle blocks; 1e-13 not
  // reached).  So where the trial takes more than kScGood, the triangle blocks are tried too; the better one is kept,
  // and where neither converges there is no plan and the general kernel solves.
  int its = kScTrial;
  if ((s = sc_arrays(c, &P, Z, {pp, pc, pv})) || (s = sc_trial(c, P, &its))) return s;
  if (c->p.precond == 1 && its > kScGood) {
    std::vector<int32_t> ec;
    std::vector<double> ev;
    tdbem_triangle_rows(c, zp, zc, zv, &ec, &ev);
    std::vector<int64_t> tp(ne + 1, 0);
    std::vector<int32_t> tc;
    std::vector<double> tv;
    for (int i = 0; i < ne; ++i) {
      for (size_t k = i; k < ec.size(); k += ne)
        if (ev[k] != 0.0) {
          tc.push_back(ec[k]);
          tv.push_back(ev[k]);
        }
      tp[i + 1] = (int64_t)tc.size();
    }
    ScPlan T = base;
    int its2 = kScTrial;
    if ((s = sc_arrays(c, &T, Z, {tp, tc, tv})) || (s = sc_trial(c, T, &its2))) return s;
    if (its2 < its) std::swap(P, T);
    its = std::min(its, its2);
    sc_drop(c, &T);
  }
  if (its == kScTrial) {
    sc_drop(c, &P);
    return TDBEM_OK;
  }
  c->sc = new (std::nothrow) ScPlan(P);
  return c->sc ? TDBEM_OK : TDBEM_ENOMEM;
}

using BxFn = void (*)(BxArgs);
static BxFn bx_fn(int rows) {
  return rows <= kScThreads ? k_bicgstab_x<1> : rows <= 2 * kScThreads ? k_bicgstab_x<2> : k_bicgstab_x<4>;
}
static size_t bx_smem(int ne, int rows) { return (size_t)((ne + 3) / 4 * 4) * 2 * sizeof(float) + (size_t)(rows + 8) * sizeof(double); }

// The plan of k_bicgstab_x: Z0 in edge order in blocks of 8 rows x 16 entries, the
// four chains of a row in its four lanes.
tdbem_status tdbem_bx_build(tdbem_ctx* c, int want, const std::vector<int32_t>& zp, const std::vector<int32_t>& zc,
                            const std::vector<double>& zv) {
  const int ne = (int)c->ne;
  ScPlan P;
  P.bx = true;
  for (P.cs = want; P.cs >= 1; P.cs >>= 1) {
    P.rows = (ne + P.cs - 1) / P.cs;
    P.gpc = (P.rows + 7) / 8;
    P.passes = (P.gpc + kScWarps - 1) / kScWarps;
    if (P.rows > 4 * kScThreads || ne > 65535 || bx_smem(ne, P.rows) > 200 * 1024) return TDBEM_OK;
    const BxFn fn = bx_fn(P.rows);
    TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    sc_config(&cfg, &at, P.cs, P.cs, bx_smem(ne, P.rows), c->stream);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n > 0) break;
    cudaGetLastError();
  }
  if (P.cs < 1) return TDBEM_OK;
  // lane m's chain of a row of n entries: m, m + 4, .. below 4 (n / 4), then (m = 0) the rest
  auto chain = [](int n, int m) { return n / 4 + (m == 0 ? n % 4 : 0); };
  std::vector<int32_t> begin(P.cs * kScWarps), end((size_t)P.cs * kScWarps * P.passes);
  std::vector<float4> z32;
  std::vector<double2> z64;
  std::vector<uint2> zcol;
  int32_t nblk = 0;
  for (int fill = 0; fill < 2; ++fill) {
    if (fill) {
      z32.assign((size_t)(nblk + kScDepth) * 32, make_float4(0, 0, 0, 0));
      z64.assign((size_t)(nblk + kScDepth) * 64, make_double2(0, 0));
      zcol.assign((size_t)(nblk + kScDepth) * 32, make_uint2(0, 0));
    }
    int32_t blk = 0;
    for (int k = 0; k < P.cs; ++k)
      for (int w = 0; w < kScWarps; ++w) {
        const int32_t b0 = blk;
        begin[k * kScWarps + w] = blk;
        for (int j = 0; j < P.passes; ++j) {
          const int g = j * kScWarps + w;
          if (g < P.gpc) {
            int most = 1;
            for (int t = 0; t < 8; ++t) {
              const int li = g * 8 + t, i = k * P.rows + li;
              if (li >= P.rows || i >= ne) continue;
              const int n = zp[i + 1] - zp[i];
              for (int m = 0; m < 4; ++m) {
                most = std::max(most, chain(n, m));
                for (int u = 0; fill && u < chain(n, m); ++u) {
                  const int q = zp[i] + (u < n / 4 ? 4 * u + m : n / 4 * 4 + u - n / 4);
                  const size_t o = (size_t)(blk + u / 4) * 128 + (t * 4 + m) * 4 + u % 4;
                  ((float*)z32.data())[o] = (float)zv[q];
                  ((double*)z64.data())[o] = zv[q];
                  ((uint16_t*)zcol.data())[o] = (uint16_t)zc[q];
                }
              }
            }
            blk += (most + 3) / 4;
          }
          if (j == P.passes - 1)
            while ((blk - b0) % kScDepth) ++blk;
          end[(size_t)(k * kScWarps + w) * P.passes + j] = blk;
        }
      }
    nblk = blk;
  }
  tdbem_status s;
  if ((s = sc_upload(c, &P.zb, begin)) || (s = sc_upload(c, &P.ze, end)) || (s = sc_upload(c, &P.z32, z32)) ||
      (s = sc_upload(c, &P.zval, z64)) || (s = sc_upload(c, &P.zcol, zcol)))
    return s;
  c->sc = new (std::nothrow) ScPlan(P);
  return c->sc ? TDBEM_OK : TDBEM_ENOMEM;
}

static tdbem_status bx_solve(tdbem_ctx* c, int32_t alpha, int32_t warm) {
  const ScPlan& P = *c->sc;
  BxArgs A;
  A.zb = P.zb;
  A.ze = P.ze;
  A.z32 = P.z32;
  A.z64 = P.zval;
  A.zcol = P.zcol;
  A.pcol = c->d_pc_col;
  A.pval = c->d_pc_val;
  A.b = c->d_R;
  A.x = c->d_J;
  A.ring = c->d_Jring;
  A.rs = c->d_rs;
  A.L = c->L;
  A.alpha = alpha;
  A.warm = warm;
  A.rows = P.rows;
  A.passes = P.passes;
  A.ne = (int32_t)c->ne;
  A.maxit = c->p.solve_maxit;
  A.tol = c->p.solve_tol;
  A.status = c->d_status;
  A.resid = c->d_dots;
  c->cluster = P.cs;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  sc_config(&cfg, &at, P.cs, P.cs, bx_smem((int)c->ne, P.rows), c->stream);
  TDBEM_CUDA_TRY(c, cudaLaunchKernelEx(&cfg, bx_fn(P.rows), A));
  return TDBEM_OK;
}

tdbem_status tdbem_sc_solve(tdbem_ctx* c, int32_t alpha, int32_t warm) {
  if (c->sc->bx) return bx_solve(c, alpha, warm);
  const ScPlan& P = *c->sc;
  ScArgs A = sc_args(c, P);
  A.b = c->d_R;
  A.x = c->d_J;
  A.ring = c->d_Jring;
  A.rs = c->d_rs;
  A.rf = c->d_rf;
  A.L = c->L;
  A.alpha = alpha;
  A.warm = warm;
  A.R = c->R;
  A.maxit = c->p.solve_maxit;
  A.tol = c->p.solve_tol;
  c->cluster = P.cs;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  sc_config(&cfg, &at, P.cs, P.cs * c->R, sc_smem(P), c->stream);
  if (c->R > 1) TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_status, 0, sizeof(int32_t), c->stream));
  TDBEM_CUDA_TRY(c, cudaLaunchKernelEx(&cfg, sc_fn(P.passes), A));
  return TDBEM_OK;
}

int tdbem_sc_kind(const tdbem_ctx* c) { return !c->sc ? 0 : c->sc->bx ? 2 : 1; }

void tdbem_sc_free(tdbem_ctx* c) {
  delete c->sc;
  c->sc = nullptr;
}

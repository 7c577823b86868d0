// direct.cu -- interaction coefficients of every time lag for a set of edge
// pairs (paper section 2.4, eq. z_ij), the incident right-hand side (eq. v_i)
// and the direct FP64 history sum of eq. R.
//
// The coefficient of J_j^beta in the tested equation at t_alpha depends on the
// lag m = alpha - beta only (eq. layer_disc_tmp with the B-spline of eq. J):
//   Zt^(m)_ij = sum over the triangles S_i^rho of i and S_j^sigma of j of
//     sum_q w_q A_i^rho [ mu/(4 pi dt^2) f_i(x_q) . int f_j Nddot(tau)/r dS
//                       + 1/(4 pi eps) div f_i div f_j int N(tau)/r dS
//                       + theta eta/(4 pi) f_i(x_q) . (n x int f_j x grad_y g dS) ]
// plus the MFIE identity term s_jump theta eta/2 (f_i, f_j) (chi Ndot(m)/dt + zeta N(m)).
// The outer integral uses the 7-point degree-5 rule; the inner integral is
// exact (integrals.cuh).  One thread owns one (test triangle, source triangle)
// pair, accumulates its 3x3 local edge pairs over the 7 points and adds them to
// the edge-pair store with FP64 atomics (each edge pair receives the 4
// triangle pairs of its two supports).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>

#include "integrals.cuh"
#include "internal.h"
#include "tc.cuh"

namespace tdbem {

__device__ __forceinline__ double dist3(const double* a, const double* b) {
  double x = a[0] - b[0], y = a[1] - b[1], z = a[2] - b[2];
  return sqrt(x * x + y * y + z * z);
}

// Conservative lag window [m_lo, m_lo + n) of an edge pair from the bounding
// spheres (centroid, max centroid-vertex distance) of its four triangle pairs.
__device__ __forceinline__ void edge_pair_window(const TriGeom& g, const int32_t* et, int i, int j, double a,
                                                 int* m_lo, int* n) {
  double rlo = 1e300, rhi = 0.0;
  for (int u = 0; u < 2; ++u)
    for (int w = 0; w < 2; ++w) {
      int t = et[2 * i + u], s = et[2 * j + w];
      double dc = dist3(g.cen + 3 * t, g.cen + 3 * s);
      double rr = g.rad[t] + g.rad[s];
      rlo = fmin(rlo, fmax(dc - rr, 0.0));
      rhi = fmax(rhi, dc + rr);
    }
  lag_window(rlo, rhi, a, m_lo, n);
}

__global__ void k_direct_windows(TriGeom g, const int32_t* et, int64_t ne, double a, int16_t* m_lo, uint8_t* nlag,
                                 int32_t* err) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= ne * ne) return;
  int i = (int)(p / ne), j = (int)(p % ne);
  int lo, n;
  edge_pair_window(g, et, i, j, a, &lo, &n);
  if (n > 255 || lo > 32767) {
    atomicExch(err, 1);
    n = 0;
  }
  m_lo[p] = (int16_t)lo;
  nlag[p] = (uint8_t)n;
}

// largest stored lag m_lo + nlag - 1 over all pairs (atomic maximum into *mx)
__global__ void k_max_lag(const int16_t* m_lo, const uint8_t* nlag, int64_t n, int32_t* mx) {
  int v = 0;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x)
    if (nlag[p]) v = max(v, (int)m_lo[p] + (int)nlag[p] - 1);
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomicMax(mx, v);
}

// per-row sums of nlag
__global__ void k_row_totals(const uint8_t* nlag, int64_t ne, int64_t* tot) {
  int64_t i = blockIdx.x;
  int64_t s = 0;
  for (int64_t j = threadIdx.x; j < ne; j += blockDim.x) s += nlag[i * ne + j];
  __shared__ int64_t red[32];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) tot[i] = s;
  }
}

// per-row exclusive scan of nlag into off (row base from the host scan)
__global__ void k_row_offsets(const uint8_t* nlag, int64_t ne, const int64_t* rowbase, int64_t* off) {
  int64_t i = blockIdx.x;
  __shared__ int64_t wsum[32];
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = rowbase[i];
  __syncthreads();
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int64_t j0 = 0; j0 < ne; j0 += blockDim.x) {
    int64_t j = j0 + threadIdx.x;
    int64_t v = (j < ne) ? nlag[i * ne + j] : 0;
    int64_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int64_t w = (lane < nw) ? wsum[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      if (lane < nw) wsum[lane] = w;
    }
    __syncthreads();
    int64_t excl = x - v + (wid > 0 ? wsum[wid - 1] : 0) + carry;
    if (j < ne) off[i * ne + j] = excl;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = excl + v;
    __syncthreads();
  }
}

// Sink of the direct store: every (i, j) of the mesh.  An edge pair receives
// one contribution from each of the four triangle pairs of its two supports,
// class k = 2 (test triangle is i's "-" triangle) + (source triangle is j's
// "-" triangle).  With val4 set, contribution k goes to its own slot
// val4[4 (off + w) + k] with a plain store, and k_sum4 adds the four in a
// fixed order afterwards, so the stored coefficients do not depend on the
// order in which threads finish; without it the contributions are added to
// val with FP64 atomics.
struct DirectSink {
  const int16_t* m_lo;
  const uint8_t* nlag;
  const int64_t* off;
  double* val;
  int64_t ne;
  double* val4;
  __device__ __forceinline__ bool add(int i, int j, int m, int k, double v) const {
    int64_t p = (int64_t)i * ne + j;
    int w = m - m_lo[p];
    if (w < 0 || w >= nlag[p]) return false;
    if (val4)
      val4[4 * (off[p] + w) + k] = v;
    else
      atomicAdd(val + off[p] + w, v);
    return true;
  }
};

// val[e] = ((v4[4e] + v4[4e+1]) + v4[4e+2]) + v4[4e+3]
__global__ void k_sum4(const double* v4, int64_t n, double* val) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const double* q = v4 + 4 * e;
  val[e] = ((q[0] + q[1]) + q[2]) + q[3];
}

// One thread per (test triangle t, source triangle s) listed in `pairs` (or
// all pairs when pairs == nullptr).
template <class Sink>
__global__ void __launch_bounds__(128) k_assemble(TriGeom g, Phys ph, int64_t nt, const int2* pairs, int64_t npairs,
                                                  Sink sink, int32_t* err) {
  int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= npairs) return;
  int t, s;
  if (pairs) {
    int2 q = pairs[idx];
    t = q.x;
    s = q.y;
  } else {
    t = (int)(idx / nt);
    s = (int)(idx % nt);
  }
  const double a = ph.a;
  // union lag window of the triangle pair
  double dc = dist3(g.cen + 3 * t, g.cen + 3 * s);
  int M0, NM;
  lag_window(fmax(dc - g.rad[t] - g.rad[s], 0.0), dc + g.rad[t] + g.rad[s], a, &M0, &NM);
  if (NM > kMaxWin) {
    atomicExch(err, 2);
    return;
  }
  double acc[3][3][kMaxWin];
  for (int u = 0; u < 3; ++u)
    for (int w = 0; w < 3; ++w)
      for (int k = 0; k < NM; ++k) acc[u][w][k] = 0.0;
  double vt[9], vs[9], ns[3], nin[3];
  for (int k = 0; k < 9; ++k) {
    vt[k] = g.v[9 * t + k];
    vs[k] = g.v[9 * s + k];
  }
  for (int k = 0; k < 3; ++k) {
    ns[k] = g.nrm[3 * s + k];
    nin[k] = -g.nrm[3 * t + k];  // n points into the conductor (paper section 2.1)
  }
  const double At = g.area[t], As = g.area[s];
  double ci[3], divi[3], oi[3][3], cj[3], divj[3], oj[3][3];
  for (int k = 0; k < 3; ++k) {
    double sg = g.sgn[3 * t + k], l = g.elen[3 * t + k];
    ci[k] = sg * l / (2 * At);
    divi[k] = sg * l / At;
    for (int q = 0; q < 3; ++q) oi[k][q] = g.opp[9 * t + 3 * k + q];
    double sg2 = g.sgn[3 * s + k], l2 = g.elen[3 * s + k];
    cj[k] = sg2 * l2 / (2 * As);
    divj[k] = sg2 * l2 / As;
    for (int q = 0; q < 3; ++q) oj[k][q] = g.opp[9 * s + 3 * k + q];
  }
  const double PI = 3.14159265358979323846;
  const double kA = ph.mu / (4 * PI * ph.dt * ph.dt), kphi = 1.0 / (4 * PI * ph.eps), kP = ph.theta * ph.eta / (4 * PI);
  InnerOut io;
  for (int q = 0; q < kNq; ++q) {
    double x[3];
    for (int k = 0; k < 3; ++k) x[k] = ph.qb[q][0] * vt[k] + ph.qb[q][1] * vt[3 + k] + ph.qb[q][2] * vt[6 + k];
    double wq = ph.qw[q] * At;
    double rhi = fmax(fmax(dist3(x, vs), dist3(x, vs + 3)), dist3(x, vs + 6));
    double rlo = fmax(dist3(x, g.cen + 3 * s) - g.rad[s], 0.0);
    int m0, nm;
    lag_window(rlo, rhi, a, &m0, &nm);
    if (m0 < M0 || m0 + nm > M0 + NM || nm > kMaxWin) {
      atomicExch(err, 3);
      return;
    }
    if (!inner_integrals(x, vs, ns, g.lmax[s], a, ph.chi / ph.dt, ph.zeta, m0, nm, io)) {
      atomicExch(err, 4);
      return;
    }
    double fi[3][3], xo[3][3];
    for (int k = 0; k < 3; ++k)
      for (int u = 0; u < 3; ++u) {
        fi[k][u] = ci[k] * (x[u] - oi[k][u]);
        xo[k][u] = x[u] - oj[k][u];
      }
    const double h = io.h;
    for (int im = 0; im < nm; ++im) {
      double A1[3], P1[3];
      for (int u = 0; u < 3; ++u) {
        A1[u] = io.EA[im][u] - h * ns[u] * io.A0[im];
        P1[u] = io.EP[im][u] - h * ns[u] * io.Sn[im];
      }
      for (int ks = 0; ks < 3; ++ks) {
        double IA[3], IP[3], nIP[3];
        for (int u = 0; u < 3; ++u) IA[u] = cj[ks] * (A1[u] + xo[ks][u] * io.A0[im]);
        IP[0] = cj[ks] * (xo[ks][1] * P1[2] - xo[ks][2] * P1[1]);
        IP[1] = cj[ks] * (xo[ks][2] * P1[0] - xo[ks][0] * P1[2]);
        IP[2] = cj[ks] * (xo[ks][0] * P1[1] - xo[ks][1] * P1[0]);
        nIP[0] = nin[1] * IP[2] - nin[2] * IP[1];
        nIP[1] = nin[2] * IP[0] - nin[0] * IP[2];
        nIP[2] = nin[0] * IP[1] - nin[1] * IP[0];
        for (int kt = 0; kt < 3; ++kt) {
          double val = kA * (fi[kt][0] * IA[0] + fi[kt][1] * IA[1] + fi[kt][2] * IA[2]) +
                       kphi * divi[kt] * divj[ks] * io.phi[im] +
                       kP * (fi[kt][0] * nIP[0] + fi[kt][1] * nIP[1] + fi[kt][2] * nIP[2]);
          acc[kt][ks][m0 - M0 + im] += wq * val;
        }
      }
    }
    // MFIE identity term on the test triangle itself (lags 1 and 2)
    if (s == t && ph.s_jump != 0.0) {
      const double c1 = ph.chi / ph.dt + 0.5 * ph.zeta, c2 = -ph.chi / ph.dt + 0.5 * ph.zeta;
      for (int kt = 0; kt < 3; ++kt)
        for (int ks = 0; ks < 3; ++ks) {
          double fj[3];
          for (int u = 0; u < 3; ++u) fj[u] = cj[ks] * xo[ks][u];
          double G = wq * (fi[kt][0] * fj[0] + fi[kt][1] * fj[1] + fi[kt][2] * fj[2]);
          double sc = ph.s_jump * ph.theta * ph.eta * 0.5 * G;
          if (1 - M0 >= 0 && 1 - M0 < NM) acc[kt][ks][1 - M0] += sc * c1;
          if (2 - M0 >= 0 && 2 - M0 < NM) acc[kt][ks][2 - M0] += sc * c2;
        }
    }
  }
  for (int kt = 0; kt < 3; ++kt) {
    int i = g.edge[3 * t + kt];
    for (int ks = 0; ks < 3; ++ks) {
      int j = g.edge[3 * s + ks];
      for (int k = 0; k < NM; ++k) {
        double v = acc[kt][ks][k];
        if (v == 0.0) continue;
        const int cls = (g.sgn[3 * t + kt] < 0 ? 2 : 0) + (g.sgn[3 * s + ks] < 0 ? 1 : 0);
        if (!sink.add(i, j, M0 + k, cls, v)) atomicExch(err, 5);
      }
    }
  }
}

template __global__ void k_assemble<DirectSink>(TriGeom, Phys, int64_t, const int2*, int64_t, DirectSink, int32_t*);

// Sink of a sparse edge-pair store: CSR over test edges i, sorted source edges j.
struct CsrSink {
  const int64_t* row_ptr;
  const int32_t* col;
  const int16_t* m_lo;
  const uint8_t* nlag;
  const int64_t* off;
  double* val;
  __device__ __forceinline__ bool add(int i, int j, int m, int /*k*/, double v) const {
    int64_t lo = row_ptr[i], hi = row_ptr[i + 1] - 1;
    while (lo <= hi) {
      int64_t mid = (lo + hi) >> 1;
      int c = col[mid];
      if (c == j) {
        int w = m - m_lo[mid];
        if (w < 0 || w >= nlag[mid]) return false;
        atomicAdd(val + off[mid] + w, v);
        return true;
      }
      if (c < j) lo = mid + 1; else hi = mid - 1;
    }
    return false;
  }
};

template __global__ void k_assemble<CsrSink>(TriGeom, Phys, int64_t, const int2*, int64_t, CsrSink, int32_t*);

// windows of the listed edge pairs (CSR entries)
__global__ void k_csr_windows(TriGeom g, const int32_t* et, const int64_t* row_ptr, const int32_t* col, int64_t ne,
                              double a, int16_t* m_lo, uint8_t* nlag, int32_t* err) {
  int64_t i = blockIdx.x;
  if (i >= ne) return;
  for (int64_t p = row_ptr[i] + threadIdx.x; p < row_ptr[i + 1]; p += blockDim.x) {
    int lo, n;
    edge_pair_window(g, et, (int)i, col[p], a, &lo, &n);
    if (n > 255 || lo > 32767) {
      atomicExch(err, 1);
      n = 0;
    }
    m_lo[p] = (int16_t)lo;
    nlag[p] = (uint8_t)n;
  }
}

// ---------------------------------------------------------------------------
// Incident right-hand side V_i^{alpha-1} (eq. v_i) for a plane wave (a
// modulated Gaussian, or the Sin^2 pulse of section 4.1 when sigma < 0); one
// thread per edge, 2 triangles x 7 points, FP64.
// grid: (edge blocks, steps); right-hand side r of R:
// V[((alpha-alpha0)*ne + i)*R + r] for alpha = alpha0 .. alpha0+gridDim.y-1
__global__ void k_rhs_plane(TriGeom g, Phys ph, const int32_t* et, int64_t ne, const double* pulse, int32_t alpha0,
                            int32_t R, int32_t r, double* V) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= ne) return;
  const int32_t alpha = alpha0 + blockIdx.y;
  double* Rv = V + (int64_t)(alpha - alpha0) * ne * R;
  const double PI = 3.14159265358979323846;
  double kv[3] = {pulse[0], pulse[1], pulse[2]}, pol[3] = {pulse[3], pulse[4], pulse[5]};
  double f0 = pulse[6], sg = pulse[7], t0 = pulse[8], zmin = pulse[9];
  double kxp[3] = {kv[1] * pol[2] - kv[2] * pol[1], kv[2] * pol[0] - kv[0] * pol[2], kv[0] * pol[1] - kv[1] * pol[0]};
  double t = alpha * ph.dt;
  double sum = 0.0;
  for (int rho = 0; rho < 2; ++rho) {
    int tri = et[2 * i + rho];
    int side = 0;
    for (int k = 0; k < 3; ++k)
      if (g.edge[3 * tri + k] == (int)i) side = k;
    double sgn = g.sgn[3 * tri + side], A = g.area[tri];
    double ci = sgn * g.elen[3 * tri + side] / (2 * A);
    const double* o = g.opp + 9 * tri + 3 * side;
    const double* v = g.v + 9 * tri;
    double nin[3] = {-g.nrm[3 * tri], -g.nrm[3 * tri + 1], -g.nrm[3 * tri + 2]};
    for (int q = 0; q < kNq; ++q) {
      double x[3];
      for (int u = 0; u < 3; ++u) x[u] = ph.qb[q][0] * v[u] + ph.qb[q][1] * v[3 + u] + ph.qb[q][2] * v[6 + u];
      double u_ = t - (kv[0] * x[0] + kv[1] * x[1] + kv[2] * x[2] - zmin) / ph.c;
      double vv = u_ - t0;
      double gg, gd;
      if (sg > 0) {
        double e = exp(-vv * vv / (2 * sg * sg));
        double sw, cw;
        sincos(2 * PI * f0 * vv, &sw, &cw);
        gg = cw * e;
        gd = (-2 * PI * f0 * sw - vv / (sg * sg) * cw) * e;
      } else {  // Sin^2 pulse: length f0, amplitude -sg
        const double w = 2 * PI * ph.c / f0, ph_ = w * vv;
        gg = gd = 0.0;
        if (ph_ >= 0.0 && ph_ <= 2 * PI) {
          double sw, cw;
          sincos(ph_, &sw, &cw);
          gg = -sg * sw * sw;
          gd = -sg * 2.0 * sw * cw * w;
        }
      }
      // -Edot + theta eta n x (chi Hdot + zeta H), E = pol g, H = k x pol g / eta
      double Hm[3], nH[3];
      for (int u = 0; u < 3; ++u) Hm[u] = kxp[u] * (ph.chi * gd + ph.zeta * gg) / ph.eta;
      nH[0] = nin[1] * Hm[2] - nin[2] * Hm[1];
      nH[1] = nin[2] * Hm[0] - nin[0] * Hm[2];
      nH[2] = nin[0] * Hm[1] - nin[1] * Hm[0];
      double val = 0.0;
      for (int u = 0; u < 3; ++u) val += ci * (x[u] - o[u]) * (-pol[u] * gd + ph.theta * ph.eta * nH[u]);
      sum += ph.qw[q] * A * val;
    }
  }
  Rv[i * R + r] = sum;
}

// The single-right-hand-side history sum runs on the FP32 pipes in
// double-float arithmetic (each FP64 operand held as an unevaluated sum of two
// FP32 numbers, hi + lo with |lo| <= ulp(hi)/2): GB300 issues FP64 FMAs at
// 1/64 of its FP32 rate, which bounded the plain FP64 loop well below the HBM
// roofline.  The product of two split numbers keeps hi*hi exactly (an FMA
// recovers its rounding error) and the two cross terms; the dropped lo*lo and
// the splits themselves are below 2^-47 of the product, so a term carries 46
// significant bits against FP64's 53 while the sum stays compensated (TwoSum
// into a hi/lo accumulator).  Operands must lie inside FP32's normal range.
__device__ __forceinline__ void df_fma_acc(float& sh, float& sl, float2 z, float2 x) {
  const float p = __fmul_rn(z.x, x.x);
  float e = __fmaf_rn(z.x, x.x, -p);
  e = __fmaf_rn(z.x, x.y, e);
  e = __fmaf_rn(z.y, x.x, e);
  const float s = __fadd_rn(sh, p);  // TwoSum(sh, p)
  const float bb = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, e));
}

// (sh, sl) += (bh, bl), both double-float: TwoSum of the high parts, the low
// parts and the rounding error added to the low part.
__device__ __forceinline__ void df_add(float& sh, float& sl, float bh, float bl) {
  const float s = __fadd_rn(sh, bh);
  const float bb = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(bh, bb));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, bl));
}

// Stored coefficients split in place, double -> (hi, lo) pair of the same 8 bytes.
__global__ void k_split_values(double* val, int64_t n) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float2 s = split_pair(val[t]);
  reinterpret_cast<float2*>(val)[t] = s;
}

// ring2[slot*ne + j] = split(ring[j*L + slot]): the history of one right-hand
// side transposed, so that the columns of a warp at one lag read contiguously.
__global__ void k_ring_split(const double* ring, int64_t ne, int32_t L, float2* ring2) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= ne * L) return;
  const int64_t j = t / L;
  const int32_t slot = (int32_t)(t - j * L);
  ring2[(int64_t)slot * ne + j] = split_pair(ring[t]);
}

constexpr int kDhThreads = 256;  // column pairs per chunk (one per thread)
constexpr int kDhCap = 3072;     // coefficients staged per chunk buffer (24 KB; four blocks per SM)

__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

struct DhChunk {
  int lo = 0, n = 0;
  int64_t o = 0, start = 0, cnt = 0;
};

// Metadata of the chunk starting at column j0 (thread t takes column j0 + t).
__device__ __forceinline__ DhChunk dh_meta(const int16_t* m_lo, const uint8_t* nlag, const int64_t* off, int64_t row0,
                                           int64_t ne, int64_t j0) {
  DhChunk m;
  const int64_t j = j0 + threadIdx.x;
  if (j < ne) {
    m.lo = m_lo[row0 + j];
    m.n = nlag[row0 + j];
    m.o = off[row0 + j];
  }
  const int64_t last = min(j0 + kDhThreads, ne) - 1;
  m.start = off[row0 + j0];
  m.cnt = off[row0 + last] + nlag[row0 + last] - m.start;
  return m;
}

// R_i = V_i - sum_j sum_{m >= 2, alpha-m >= 0} Zt^(m)_ij J_j^{alpha-m} (eq. R;
// V may be null: zero; V may alias R); one block per row i, thread t taking
// column j0 + t of each chunk of 256 columns.  The row's stored lags are
// contiguous in column order, so a chunk owns one contiguous coefficient
// range: it is copied into shared memory with asynchronous copies one chunk
// ahead of the arithmetic (a chunk larger than a buffer is read from global
// memory in place) while the metadata is loaded two chunks ahead.  val holds
// split coefficients (k_split_values), ring2 the split, transposed history
// (k_ring_split).
__global__ void __launch_bounds__(kDhThreads) k_direct_history(const int16_t* m_lo, const uint8_t* nlag,
                                                               const int64_t* off, const float2* val, int64_t ne,
                                                               const float2* ring2, int32_t L, int32_t alpha,
                                                               const double* V, double* R) {
  extern __shared__ float2 zbuf[];  // [2][kDhCap]
  __shared__ double red[kDhThreads / 32];
  const int64_t row0 = (int64_t)blockIdx.x * ne;
  const int64_t nchunk = (ne + kDhThreads - 1) / kDhThreads;
  float sh = 0.f, sl = 0.f;
  DhChunk cur = dh_meta(m_lo, nlag, off, row0, ne, 0);
  if (cur.cnt <= kDhCap)
    for (int64_t k = threadIdx.x; k < cur.cnt; k += kDhThreads) cp_async8(zbuf + k, val + cur.start + k);
  cp_async_commit();
  DhChunk nxt;
  if (nchunk > 1) nxt = dh_meta(m_lo, nlag, off, row0, ne, kDhThreads);
  for (int64_t c = 0; c < nchunk; ++c) {
    float2* buf = zbuf + (c & 1) * kDhCap;
    if (c + 1 < nchunk && nxt.cnt <= kDhCap) {
      float2* nb = zbuf + ((c + 1) & 1) * kDhCap;
      for (int64_t k = threadIdx.x; k < nxt.cnt; k += kDhThreads) cp_async8(nb + k, val + nxt.start + k);
    }
    cp_async_commit();
    DhChunk nn;
    if (c + 2 < nchunk) nn = dh_meta(m_lo, nlag, off, row0, ne, (c + 2) * kDhThreads);
    cp_async_wait1();
    __syncthreads();
    {
      // this column's lags m = lo + w with m >= 2 and alpha - m >= 0
      const int64_t j = c * kDhThreads + threadIdx.x;
      const float2* z = (cur.cnt <= kDhCap) ? buf + (cur.o - cur.start) : val + cur.o;
      const int w0 = max(0, 2 - cur.lo), w1 = min(cur.n, alpha - cur.lo + 1);
#pragma unroll 4
      for (int w = w0; w < w1; ++w) {
        const int slot = (alpha - cur.lo - w) & (L - 1);
        df_fma_acc(sh, sl, z[w], __ldg(ring2 + (int64_t)slot * ne + j));
      }
    }
    const float s = __fadd_rn(sh, sl);  // renormalise once per chunk
    sl = __fsub_rn(sl, __fsub_rn(s, sh));
    sh = s;
    __syncthreads();
    cur = nxt;
    nxt = nn;
  }
  double s = (double)sh + (double)sl;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kDhThreads / 32; ++w) t += red[w];
    R[blockIdx.x] = (V ? V[blockIdx.x] : 0.0) - t;
  }
}

// pre[w * npos + p] = the sum of position p's partials k = w, w + 8, .. of the far
// pairs (nfar of them), then of the near ones (nnear); with both != 0 partial k is
// the sum of the two (a unit lies in one, the other holds zero).  A block takes 32
// positions, a warp's lanes read 32 neighbours.  It runs behind the sums on the
// side stream: a step itself adds eight values per row.
constexpr int kRedLanes = 8;

__global__ void __launch_bounds__(kRedLanes * 32) k_direct_presum(const double* __restrict__ far, int32_t nfar,
                                                                 const double* __restrict__ near, int32_t nnear,
                                                                 int both, int64_t npos, double* __restrict__ pre) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t p = (int64_t)blockIdx.x * 32 + lane;
  double t = 0.0;
  if (both) {
#pragma unroll 8
    for (int k = w; k < nnear; k += kRedLanes)
      t += nfar ? far[(int64_t)k * npos + p] + near[(int64_t)k * npos + p] : near[(int64_t)k * npos + p];
  } else {
#pragma unroll 8
    for (int k = w; k < nfar; k += kRedLanes) t += far[(int64_t)k * npos + p];
    for (int k = w; k < nnear; k += kRedLanes) t += near[(int64_t)k * npos + p];
  }
  pre[(int64_t)w * npos + p] = t;
}

// R_i = V_i - (pre of row i's position plus the row's lag-2 entries l2 against
// J^{alpha-2}, in FP64).  The entries lie in position order; eight lanes share a
// row, each going on from its sum of the partials, and meet in a fixed shuffle
// tree, so the result does not depend on scheduling.  V may be null (zero) and may
// alias R.
__global__ void __launch_bounds__(128) k_direct_reduce(const double* __restrict__ pre, const int32_t* __restrict__ rows,
                                                       int64_t npos, const int32_t* __restrict__ l2_ptr,
                                                       const int32_t* __restrict__ l2_col,
                                                       const double* __restrict__ l2_val, const double* ring,
                                                       int32_t L, int32_t alpha, const double* V, double* R) {
  const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kRedLanes;
  const int sub = threadIdx.x % kRedLanes;
  double t = 0.0;
  if (p < npos) {
    t = pre[(int64_t)sub * npos + p];
    if (alpha >= 2) {
      const double* Js = ring + ((alpha - 2) & (L - 1));
      const int e1 = l2_ptr[p + 1];
#pragma unroll 4
      for (int e = l2_ptr[p] + sub; e < e1; e += kRedLanes) t += l2_val[e] * Js[(int64_t)l2_col[e] * L];
    }
  }
#pragma unroll
  for (int d = kRedLanes / 2; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
  if (p < npos && sub == 0) {
    const int32_t i = rows[p];
    if (i >= 0) R[i] = (V ? V[i] : 0.0) - t;
  }
}

// Row-tile form of the single-right-hand-side history sum of the lags >= 3.
//
// Two tiers.  A pair of functions whose first stored lag >= 3 is at least M0
// is "far": none of its lags needs a current newer than J^{alpha - M0}.  The far
// pairs' sums of a whole block of B steps can therefore be formed one block
// ahead, in ONE pass over their coefficients: a coefficient of lag m meets
// J^{alpha0 + k - m} for the block's steps k = 0 .. B - 1, which for consecutive
// lags is a window sliding over the column's history, held in registers.  The
// store is streamed once per B steps instead of once per step, which is what the
// sum is bound by.  The pass is cut into B parts (ranges of row tiles), one beside
// each step of the block before; part q starts q steps later and knows q currents
// more, so its rows' M0 is 2 B + 1 - q.  The near pairs (first lag < M0) are
// summed step by step.  A pair belongs to one tier with all its lags, so its FP32
// sum is one chain either way.  With B = 1, M0 = 3: every pair is far and the sum
// runs one step ahead.
//
// The FP32 and 24-bit stores take whole units instead, a tile of rows by 64 columns
// in edge order: a unit whose smallest lag is below M0 is near, and the near units
// are summed step by step from the same store.  Each (row, 64 columns) partial is
// then one and the same sum in any form of the march, to the last bit, which these
// stores need: their marches round every current to FP32 in the next steps' sums
// and carry a difference of 1e-16 in one sum on to 1e-8 in 80 steps.
//
// Order.  Rows (and the columns of the (hi, lo) store) are put in one order of their own, the leaves of a
// bisection of the edges' midpoints along the longest side, so that 8, 32 and 64
// neighbours lie close together and see a column at similar lags.  `rows` gives
// the edge at a position.
//
// Far store.  Rows are taken in tiles of 32 (position 32 rt + t: lane t of a
// warp).  For each (tile, column j) let nmax be the largest number of lags >= 3
// over the tile's far rows; the pair (tile, j) owns nmax groups of 32 values,
// group u holding for lane t the coefficient of lag lo3 + u of its row, where
// lo3 = max(first stored lag, 3), and zero past that row's own window.  Groups run
// tile by tile and, inside a tile, column by column, so the groups of one tile and
// one block of columns are one contiguous stretch of memory.  A group is 32 values
// in a row: 128 bytes in FP32, 256 in (hi, lo) pairs, 96 in the 24-bit form (F24
// below).  goff[rt * ne + j] is the first group of (rt, j) (the next entry its
// end), lo3 one byte per (row, column), lomin the smallest lo3 of a (tile, block
// of columns).
//
// Far kernel.  Block (cb, rg) takes the column block j0 = cbw cb and the row
// tiles of group rg; its history J^{alpha0 - d}_j (d = M0 - B + 1 .. Lh - 1) is
// staged column-major in shared memory once, zero for the steps not there
// (d > alpha0, d >= L), so that zero padding and early steps need no test; a tile
// whose smallest lag reaches before J^0 is skipped whole.  Each warp owns a row
// tile at a time and streams the tile's stretch for the block's columns through a
// private ring of about 2 KB stages filled by bulk copies (cp.async.bulk, one lane
// issues, an mbarrier per stage counts the bytes); every lane sums its own row over
// the block's columns and lags, so no cross-lane reduction is needed, and writes
// partial[(k * ncb + cb) * npos + position] for each step k.  Per (tile, column) a
// lane's first lag and the column's end group are loaded five columns ahead.  The
// lanes of a warp read one column at lags that differ by their rows' distances, so
// the history reads are broadcasts or distinct banks.  Every wait is bounded: on
// expiry the warp writes NaN partials (the solve then misses its tolerance), sets
// *err, waits (bounded) for its copies in flight and stops.
//
// Arithmetic.  (hi, lo) pairs: the history is split into (hi, lo) pairs too
// and every product and sum is double-float (df_fma_acc).  FP32 store: the
// history is rounded to FP32, each column's lags are summed with FP32 FMAs
// (at most nmax terms) and the column sums are added in double-float.  With
// u = 2^-24 the FP32 form's error on row i is then at most about
// (2 + nmax) u sum |Zt^(m)_ij| |J_j^{alpha-m}| (two roundings per product,
// the recursive-sum bound over a column), one FMA per stored value.  The
// 24-bit store adds its own rounding, 2^-16 sum |Zt^(m)_ij| |J_j^{alpha-m}|.
constexpr int kRtWarps = 8;  // warps per block
constexpr int kRtB = 4;      // steps per pass of the far pairs where the store is large
constexpr int64_t kRtBlockBytes = 64ll << 20;  // such a store's bytes

// A value of the 24-bit store: an FP32 number with its significand rounded
// to 16 bits (round half away from zero on the dropped byte), kept as its top
// two bytes and its third byte.  A group of 32 is 96 bytes: the 32 top halves
// (64 B), then the 32 third bytes (32 B).
struct F24 {};

__host__ __device__ inline uint32_t f24_bits(float f) {  // the 24 kept bits, right-aligned
  uint32_t b;
  memcpy(&b, &f, 4);
  return (b + 0x80u) >> 8;
}

// Per store: the history's type, the bytes of a group of 32 values, and a
// lane's read position in a staged group (at: the group's first byte; get:
// this lane's value; next: the following group).
template <typename Coef>
struct RtPrec;
template <>
struct RtPrec<float> {  // FP32 store: FP32 history, FP32 column sums
  using Hist = float;
  static constexpr int kGroupBytes = 128;
  struct Cur {
    const float* p;
    __device__ void at(const unsigned char* g, int lane) { p = reinterpret_cast<const float*>(g) + lane; }
    __device__ float get() const { return *p; }
    __device__ void next() { p += 32; }
  };
};
template <>
struct RtPrec<F24> {  // 24-bit store: as FP32 after the load
  using Hist = float;
  static constexpr int kGroupBytes = 96;
  struct Cur {
    const uint16_t* h;
    const uint8_t* l;
    __device__ void at(const unsigned char* g, int lane) {
      h = reinterpret_cast<const uint16_t*>(g) + lane;
      l = g + 64 + lane;
    }
    // bytes (top half, third byte, 0): x = third byte (bytes 1..3 zero), y = top half
    __device__ float get() const { return __uint_as_float(__byte_perm((uint32_t)*l, (uint32_t)*h, 0x5401)); }
    __device__ void next() {
      h += 48;
      l += 96;
    }
  };
};
template <>
struct RtPrec<float2> {  // (hi, lo) store: double-float throughout
  using Hist = float2;
  static constexpr int kGroupBytes = 256;
  struct Cur {
    const float2* p;
    __device__ void at(const unsigned char* g, int lane) { p = reinterpret_cast<const float2*>(g) + lane; }
    __device__ float2 get() const { return *p; }
    __device__ void next() { p += 32; }
  };
};

// shared memory of a block: NS stages of SB bytes and an mbarrier per stage
// and warp, and the history of cbw columns x nh steps
template <typename Coef>
size_t rt_smem_bytes(int ns, int sb, int cbw, int nh) {
  return (size_t)kRtWarps * ns * (sb + 8) + (size_t)cbw * nh * sizeof(typename RtPrec<Coef>::Hist);
}

// coefficient z (FP32) times history x (double-float) added to (sh, sl)
__device__ __forceinline__ void df_fma_acc(float& sh, float& sl, float z, float2 x) {
  const float p = __fmul_rn(z, x.x);
  float e = __fmaf_rn(z, x.x, -p);
  e = __fmaf_rn(z, x.y, e);
  const float s = __fadd_rn(sh, p);
  const float bb = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, e));
}

// the history's value from its (hi, lo) split: hi is the value rounded to FP32
__device__ __forceinline__ void rt_hist(float* o, float2 v) { *o = v.x; }
__device__ __forceinline__ void rt_hist(float2* o, float2 v) { *o = v; }

// Split history rs[j * L + slot] = (hi, lo) of ring[j * L + slot].
__global__ void k_ring_pairs(const double* ring, int64_t n, float2* rs) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < n) rs[t] = split_pair(ring[t]);
}

// B steps from alpha0 on; NS stages of SB bytes per warp; MINB blocks per SM.
// list, loff: per column block the row tiles of this launch, in the order of their
// smallest lags; tiles: how many of them a block takes; m0: their smallest lag.
template <typename Coef, int B, int NS, int SB, int MINB>
__global__ void __launch_bounds__(kRtWarps * 32, MINB)
    k_direct_history_rt(const unsigned char* __restrict__ val, const uint32_t* __restrict__ goff,
                        const uint8_t* __restrict__ lo3, const int32_t* __restrict__ lomin,
                        const int32_t* __restrict__ rows, const int32_t* __restrict__ list,
                        const int32_t* __restrict__ loff, int64_t ne, const float2* __restrict__ rs, int32_t L,
                        int32_t Lh, int32_t alpha0, int32_t m0, int32_t tiles, int32_t cbw, int64_t npos,
                        double* __restrict__ partial, int32_t* err) {
  using Hist = typename RtPrec<Coef>::Hist;
  constexpr int GB = RtPrec<Coef>::kGroupBytes;
  constexpr int CG = SB / GB;  // groups per stage
  static_assert(CG * GB == SB && SB % 16 == 0, "a stage holds whole groups and 16-byte copies");
  constexpr bool kF32 = !std::is_same<Coef, float2>::value;  // FP32 arithmetic (FP32 and 24-bit stores)
  extern __shared__ __align__(128) unsigned char rt_sm[];
  unsigned char* stages = rt_sm;  // [kRtWarps][NS][SB]
  uint64_t* bars = reinterpret_cast<uint64_t*>(rt_sm + (size_t)kRtWarps * NS * SB);
  const int d0 = m0 - (B - 1), nh = Lh - d0;  // staged: J^{alpha0 - d}, d = d0 .. Lh - 1
  Hist* hist = reinterpret_cast<Hist*>(bars + kRtWarps * NS);  // [cbw][nh]
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t j0 = (int64_t)blockIdx.x * cbw;
  const int ncol = (int)min((int64_t)cbw, ne - j0);
  const int32_t* tl = list + loff[blockIdx.x];
  const int i_begin = blockIdx.y * tiles, i_all = min(loff[blockIdx.x + 1] - loff[blockIdx.x], i_begin + tiles);
  // the block's tiles whose lags reach J^0 or later by the last step: the first of
  // them, as they are in the order of their smallest lags; the others add nothing
  int i_end = i_begin;
  while (i_end < i_all && lomin[(int64_t)tl[i_end] * gridDim.x + blockIdx.x] <= alpha0 + B - 1) ++i_end;
  const uint32_t bar0 = tc::smem_u32(bars + w * NS);
  unsigned char* wst = stages + (size_t)w * NS * SB;
  if (lane == 0) {
    for (int s = 0; s < NS; ++s) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * s));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  double* out = partial + (int64_t)blockIdx.x * npos;
  for (int i = i_end + w; i < i_all; i += kRtWarps)
#pragma unroll
    for (int k = 0; k < B; ++k) out[(int64_t)k * gridDim.x * npos + (int64_t)tl[i] * 32 + lane] = 0.0;
  if (i_end == i_begin) return;  // the whole block: nothing is in flight
  // producer cursor of this warp's stretches (every lane keeps it; lane 0 copies)
  int p_i = i_begin + w;
  uint32_t p_g = 0, p_ge = 0, issued = 0;
  if (p_i < i_end) {
    p_g = goff[(int64_t)tl[p_i] * ne + j0];
    p_ge = goff[(int64_t)tl[p_i] * ne + j0 + ncol];
  }
  auto issue = [&](int s) {  // the cursor's next chunk into stage s (none once the warp's tiles are done)
    while (p_i < i_end && p_g == p_ge) {
      p_i += kRtWarps;
      if (p_i < i_end) {
        p_g = goff[(int64_t)tl[p_i] * ne + j0];
        p_ge = goff[(int64_t)tl[p_i] * ne + j0 + ncol];
      }
    }
    if (p_i >= i_end) return;
    const uint32_t n = min((uint32_t)CG, p_ge - p_g);
    if (lane == 0) {  // every lane's reads of the stage have returned (their values were used)
      const uint32_t bytes = n * (uint32_t)GB;
      tc::mbar_expect_tx(bar0 + 8 * s, bytes);
      tc::bulk_g2s(tc::smem_u32(wst + (size_t)s * SB), val + (size_t)p_g * GB, bytes, bar0 + 8 * s);
    }
    p_g += n;
    ++issued;
  };
  for (int s = 0; s < NS; ++s) issue(s);
  // the block's history, while the first copies are in flight
  for (int k = threadIdx.x; k < cbw * nh; k += blockDim.x) {
    const int c = k / nh, d = d0 + k - c * nh;
    const bool on = c < ncol && d <= alpha0 && d < L;
    rt_hist(hist + k, on ? rs[(rows ? (int64_t)rows[j0 + c] : j0 + c) * L + ((alpha0 - d) & (L - 1))] : make_float2(0.f, 0.f));
  }
  __syncthreads();
  uint32_t q = 0;  // chunks taken
  bool failed = false;
  typename RtPrec<Coef>::Cur zc;
  zc.at(wst, lane);
  // per column its first lag (this lane's row) and its end group, loaded five
  // columns ahead over the warp's sequence of (tile, column)
  int pf_i = i_begin + w, pf_c = 0;
  auto meta = [&](int& l, uint32_t& e) {
    l = 0;
    e = 0;
    if (pf_i < i_end) {
      const int64_t m = (int64_t)tl[pf_i] * ne + j0 + pf_c;
      l = lo3[m * 32 + lane];
      e = goff[m + 1];
      if (++pf_c == ncol) {
        pf_c = 0;
        pf_i += kRtWarps;
      }
    }
  };
  int l0, l1, l2, l3, l4;
  uint32_t e0, e1, e2, e3, e4;
  meta(l0, e0);
  meta(l1, e1);
  meta(l2, e2);
  meta(l3, e3);
  meta(l4, e4);
  // the range of the warp's next tile, loaded a tile ahead
  uint32_t nx_g = 0, nx_end = 0;
  if (i_begin + w < i_end) {
    nx_g = goff[(int64_t)tl[i_begin + w] * ne + j0];
    nx_end = goff[(int64_t)tl[i_begin + w] * ne + j0 + ncol];
  }
  for (int it = i_begin + w; it < i_end; it += kRtWarps) {
    const int rt = tl[it];
    uint32_t g = nx_g;
    const uint32_t gend = nx_end;
    if (it + kRtWarps < i_end) {
      nx_g = goff[(int64_t)tl[it + kRtWarps] * ne + j0];
      nx_end = goff[(int64_t)tl[it + kRtWarps] * ne + j0 + ncol];
    }
    uint32_t cend = g;  // end of the chunk held (none yet in this tile)
    float sh[B] = {}, sl[B] = {};
    for (int c = 0; c < ncol && !failed; ++c) {
      const int lo = max(l0, d0 + B - 1);  // a row without lags here: any staged place
      const uint32_t ge = e0;
      l0 = l1;
      e0 = e1;
      l1 = l2;
      e1 = e2;
      l2 = l3;
      e2 = e3;
      l3 = l4;
      e3 = e4;
      meta(l4, e4);
      // x[k]: the history of the lane's next lag for step k (x[0] is read as its lag comes up)
      const Hist* h = hist + c * nh + (lo - d0);
      Hist x[B];
#pragma unroll
      for (int k = 1; k < B; ++k) x[k] = h[-k];
      float a[B] = {};  // FP32 arithmetic: the column's sums
      while (g < ge) {
        if (g == cend) {
          if (q > 0) {
            __syncwarp();
            issue((int)((q - 1) % NS));  // chunk q - 1 is consumed: its stage takes the next
          }
          const bool ok = tc::mbar_wait(bar0 + 8 * (q % NS), (q / NS) & 1);
          if (__any_sync(0xffffffffu, !ok)) {
            failed = true;
            break;
          }
          zc.at(wst + (size_t)(q % NS) * SB, lane);
          cend = min(g + (uint32_t)CG, gend);
          ++q;
        }
        const uint32_t gs = min(ge, cend);
#pragma unroll 4
        for (; g < gs; ++g, ++h, zc.next()) {
          const auto z = zc.get();
          x[0] = *h;
#pragma unroll
          for (int k = 0; k < B; ++k) {
            if constexpr (kF32)
              a[k] = __fmaf_rn(z, x[k], a[k]);
            else
              df_fma_acc(sh[k], sl[k], z, x[k]);
          }
#pragma unroll
          for (int k = B - 1; k > 0; --k) x[k] = x[k - 1];
        }
      }
      if constexpr (kF32) {
#pragma unroll
        for (int k = 0; k < B; ++k) df_add(sh[k], sl[k], a[k], 0.f);
      }
    }
    const int64_t i = (int64_t)rt * 32 + lane;
#pragma unroll
    for (int k = 0; k < B; ++k)
      out[(int64_t)k * gridDim.x * npos + i] =
          failed ? __longlong_as_double(0x7ff8000000000000LL) : (double)sh[k] + (double)sl[k];
  }
  if (failed) {
    if (lane == 0) atomicExch(err, 1);
    for (uint32_t k = q; k < issued; ++k) tc::mbar_wait(bar0 + 8 * (k % NS), (k / NS) & 1);
  }
}

// Near store of the (hi, lo) pairs and its kernel, one step.  The near pairs of 32 rows would fill a third
// of a tile's lanes (the rows' near columns differ), so the near tier takes 8
// positions and 4 of their columns at a time: a quad owns as many groups of 32
// values as its longest window has lags, lane 8 s + r holding the coefficients of
// row r and column s (a sub-tile's columns are sorted by their lags, so that a
// quad's columns are alike); meta gives the lane's column and first lag << 24.  A
// warp takes one chunk {sub-tile, first quad, end quad, slot}: kNearAhead
// coefficients and their history values, read from the split ring, are in flight
// at a time, whose latency bounds it.  The four columns' sums meet in a fixed
// order: partial[slot * npos + position].
constexpr int kNearGroups = 64;  // groups per chunk (about)
constexpr int kNearAhead = 8;

__global__ void __launch_bounds__(256) k_direct_near(const float2* __restrict__ val,
                                                     const uint32_t* __restrict__ qoff,
                                                     const uint32_t* __restrict__ meta,
                                                     const int4* __restrict__ chunks, int32_t nchunk, const float2* rs,
                                                     int32_t L, int32_t alpha, int64_t npos,
                                                     double* __restrict__ partial) {
  const int wid = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (wid >= nchunk) return;  // whole warps
  const int4 ch = chunks[wid];
  float sh = 0.f, sl = 0.f;
  uint32_t g = qoff[ch.y], ge = qoff[ch.y + 1], mt = meta[(size_t)ch.y * 32 + lane];
  for (int q = ch.y; q < ch.z; ++q) {
    const int qn = q + 1 < ch.z ? q + 1 : q;  // the next quad's while this one's groups are summed
    const uint32_t gn = qoff[qn + 1], mn = meta[(size_t)qn * 32 + lane];
    const float2* h = rs + (int64_t)(mt & 0xffffff) * L;
    // the slot of a step not there yet holds zero; one of a lag past the window
    // (zero coefficient) is finite
    int b = alpha - (int)(mt >> 24);
    for (; g < ge; g += kNearAhead, b -= kNearAhead) {
      float2 z[kNearAhead], x[kNearAhead];
#pragma unroll
      for (int i = 0; i < kNearAhead; ++i)
        if (g + i < ge) {
          z[i] = __ldg(val + ((size_t)g + i) * 32 + lane);
          x[i] = h[(b - i) & (L - 1)];
        }
#pragma unroll
      for (int i = 0; i < kNearAhead; ++i)
        if (g + i < ge) df_fma_acc(sh, sl, z[i], x[i]);
    }
    g = ge;
    ge = gn;
    mt = mn;
  }
#pragma unroll
  for (int d = 8; d < 32; d <<= 1)
    df_add(sh, sl, __shfl_xor_sync(0xffffffffu, sh, d), __shfl_xor_sync(0xffffffffu, sl, d));
  if (lane < 8) partial[(int64_t)ch.w * npos + (int64_t)ch.x * 8 + lane] = (double)sh + (double)sl;
}

// The first row tile of part q of B (whole blocks of kRtWarps tiles), and the part of a tile.
__host__ __device__ inline int rt_bound(int64_t nrt, int B, int q) {
  if (q <= 0) return 0;
  if (q >= B) return (int)nrt;
  const int64_t b = (nrt * q / B + kRtWarps / 2) / kRtWarps * kRtWarps;
  return (int)(b < nrt ? b : nrt);
}
__host__ __device__ inline int rt_part(int64_t rt, int64_t nrt, int B) {
  int q = 0;
  while (q + 1 < B && rt_bound(nrt, B, q + 1) <= rt) ++q;
  return q;
}
// The smallest lag of the far pairs of part q.
__host__ __device__ inline int rt_m0(int B, int q) { return B == 1 ? 3 : 2 * B + 1 - q; }

// The lags >= 3 of the pair (row i, column j) that its tier holds: first lag and count (0: none).
__device__ __forceinline__ int rt_window(const int16_t* m_lo, const uint8_t* nlag, int64_t ne, int64_t i, int64_t j,
                                         int m0, bool far, int* l3) {
  *l3 = far ? m0 : 3;
  if (i < 0) return 0;
  const int lo = m_lo[i * ne + j], hi = lo + nlag[i * ne + j];  // lags lo .. hi - 1
  const int l = max(lo, 3), n = hi - l;
  if (n <= 0 || (l >= m0) != far) return 0;
  *l3 = l;
  return n;
}

// Row-tile store, step 1: one warp per (tile, column position), lane t the row at
// position 32 rt + t.  nmax[rt * ne + j] = the tile's largest count of lags >= 3 of
// column j over its far rows (units: every row, columns in edge order), nnear[(4 rt + s) * ne + j] over the near rows of its
// sub-tile s; lo3[(rt * ne + j) * 32 + t] = the first lag of a far row (m0 where it
// has none); lomin[rt * ncb + j / cbw] their minimum over the rows that have some;
// *lh = max over the far tier of lo3 + nmax (the history the kernel reads).
__global__ void k_rt_meta(const int16_t* m_lo, const uint8_t* nlag, int64_t ne, int32_t nrt, const int32_t* rows,
                          int B, int units, uint8_t* nmax, uint8_t* nnear, uint8_t* lo3, int32_t* lomin, int ncb, int cbw,
                          int32_t* lh) {
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= (int64_t)nrt * ne) return;  // whole warps
  const int64_t rt = wid / ne, j = wid - rt * ne, i = rows[rt * 32 + lane];
  const int m0 = units ? 3 : rt_m0(B, rt_part(rt, nrt, B));
  const int64_t jj = units ? j : rows[j];
  int l3, ln;
  const int nf = rt_window(m_lo, nlag, ne, i, jj, m0, true, &l3);
  int nn = rt_window(m_lo, nlag, ne, i, jj, m0, false, &ln);
  const int mx = __reduce_max_sync(0xffffffffu, nf), need = __reduce_max_sync(0xffffffffu, l3 + mx);
  const int lm = __reduce_min_sync(0xffffffffu, nf > 0 ? l3 : 1 << 20);
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) nn = max(nn, __shfl_xor_sync(0xffffffffu, nn, d));
  lo3[wid * 32 + lane] = (uint8_t)l3;
  if (nnear && (lane & 7) == 0) nnear[(4 * rt + lane / 8) * ne + j] = (uint8_t)nn;
  if (lane == 0) {
    nmax[wid] = (uint8_t)mx;
    atomicMax(lh, need);
    atomicMin(lomin + rt * ncb + j / cbw, lm);
  }
}

// value v at lane t of the group starting at byte g
__device__ __forceinline__ void rt_put(float, unsigned char* g, int t, double v) {
  reinterpret_cast<float*>(g)[t] = __double2float_rn(v);
}
__device__ __forceinline__ void rt_put(float2, unsigned char* g, int t, double v) {
  reinterpret_cast<float2*>(g)[t] = split_pair(v);
}
__device__ __forceinline__ void rt_put(F24, unsigned char* g, int t, double v) {
  const uint32_t b = f24_bits(__double2float_rn(v));
  reinterpret_cast<uint16_t*>(g)[t] = (uint16_t)(b >> 8);
  g[64 + t] = (uint8_t)(b & 0xffu);
}

// Row-tile store, step 2: the groups of the far pairs, one warp per (tile, column
// position), zero past each row's window.
template <typename Coef>
__global__ void k_rt_fill(const int16_t* m_lo, const uint8_t* nlag, const int64_t* off, const double* val,
                          int64_t ne, int32_t nrt, const int32_t* rows, int B, int units, const uint32_t* goff,
                          unsigned char* out) {
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= (int64_t)nrt * ne) return;  // whole warps
  const int64_t rt = wid / ne, jp = wid - rt * ne, j = units ? jp : rows[jp], i = rows[rt * 32 + lane];
  const uint32_t g0 = goff[wid], nm = goff[wid + 1] - g0;
  int l3;
  const int n3 = rt_window(m_lo, nlag, ne, i, j, units ? 3 : rt_m0(B, rt_part(rt, nrt, B)), true, &l3);
  const int64_t src = n3 > 0 ? off[i * ne + j] + (l3 - m_lo[i * ne + j]) : 0;
  for (uint32_t u = 0; u < nm; ++u)
    rt_put(Coef{}, out + ((size_t)g0 + u) * RtPrec<Coef>::kGroupBytes, lane, (int)u < n3 ? val[src + u] : 0.0);
}

// The near pairs' quads: one warp per quad q of sub-tile qst[q]; qcol[4 q + s] its
// columns (edges; -1: none).
__global__ void k_near_fill(const int16_t* m_lo, const uint8_t* nlag, const int64_t* off, const double* val,
                            int64_t ne, int32_t nrt, int64_t nq, const int32_t* rows, int B, const int32_t* qst,
                            const int32_t* qcol, const uint32_t* qoff, uint32_t* meta, float2* out) {
  const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (q >= nq) return;  // whole warps
  const int64_t st = qst[q], i = rows[st * 8 + (lane & 7)], j = qcol[4 * q + lane / 8];
  const uint32_t g0 = qoff[q], nm = qoff[q + 1] - g0;
  int l3 = 3;
  const int n3 = j < 0 ? 0 : rt_window(m_lo, nlag, ne, i, j, rt_m0(B, rt_part(st / 4, nrt, B)), false, &l3);
  const int64_t src = n3 > 0 ? off[i * ne + j] + (l3 - m_lo[i * ne + j]) : 0;
  // (an absent column reads the quad's first one with zero coefficients: what is not finite there stays beside its rows)
  meta[q * 32 + lane] = (uint32_t)(j < 0 ? qcol[4 * q] : j) | (uint32_t)l3 << 24;
  for (uint32_t u = 0; u < nm; ++u)
    out[((size_t)g0 + u) * 32 + lane] = (int)u < n3 ? split_pair(val[src + u]) : make_float2(0.f, 0.f);
}

// Lag-2 entries of the direct store, as a CSR over the positions of the row
// order (before the split): one warp per position counts (fill 0) its row's
// entries, or writes them in column order (fill 1).
__global__ void k_lag2(const int16_t* m_lo, const uint8_t* nlag, const int64_t* off, const double* val, int64_t ne,
                       int64_t npos, const int32_t* rows, int fill, int32_t* ptr, int32_t* col, double* v) {
  const int64_t p = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (p >= npos) return;  // whole warps
  const int64_t i = rows[p];
  int e = fill ? ptr[p] : 0;
  const int e1 = fill ? ptr[p + 1] : 0;
  if (i >= 0)
    for (int64_t j0 = 0; j0 < ne; j0 += 32) {
      const int64_t j = j0 + lane, q = i * ne + j;
      const int lo = j < ne ? m_lo[q] : 3;
      const bool on = lo <= 2 && 2 < lo + (int)nlag[q];
      const unsigned m = __ballot_sync(0xffffffffu, on);
      const int k = e + __popc(m & ((1u << lane) - 1));
      if (fill && on && k < e1) {
        col[k] = (int32_t)j;
        v[k] = val[off[q] + (2 - lo)];
      }
      e += __popc(m);
    }
  if (!fill && lane == 0) ptr[p] = e;
}

// Batched form of k_direct_history for R right-hand sides ([..][ne][R]
// layouts): one block per row; the block's threads are split into groups of
// RL lanes (RL = R rounded up to a power of two, at most 32), lane rr of a
// group takes the right-hand sides rr, rr+RL, ... and the groups take
// interleaved columns j, so each coefficient is read once per group and
// broadcast to its lanes while the history vectors are read contiguously.
__global__ void __launch_bounds__(256) k_direct_history_multi(const int16_t* m_lo, const uint8_t* nlag,
                                                             const int64_t* off, const double* val, int64_t ne,
                                                             const double* ring, int32_t L, int32_t alpha,
                                                             int32_t R, int32_t RL, const double* V, double* Rout) {
  __shared__ double red[8][32];
  const int64_t i = blockIdx.x;
  const int rr = threadIdx.x % RL, sub = threadIdx.x / RL, nsub = blockDim.x / RL;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r0 = 0; r0 < R; r0 += RL) {
    const int r = r0 + rr;
    double s = 0.0;
    if (r < R) {
      for (int64_t j = sub; j < ne; j += nsub) {
        int64_t p = i * ne + j;
        int lo = m_lo[p], n = nlag[p];
        const double* z = val + off[p];
        const double* Jr = ring + j * L * R + r;
        for (int w = 0; w < n; ++w) {
          int m = lo + w;
          int b = alpha - m;
          if (m < 2 || b < 0) continue;
          s += __ldg(z + w) * Jr[(int64_t)(b & (L - 1)) * R];
        }
      }
    }
    // lanes rr, rr+RL, ... of a warp hold partial sums of the same r
    for (int o = 16; o >= RL; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < RL) red[warp][lane] = s;
    __syncthreads();
    if (threadIdx.x < RL && r0 + threadIdx.x < R) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w][threadIdx.x];
      int64_t q = i * R + r0 + threadIdx.x;
      Rout[q] = (V ? V[q] : 0.0) - t;
    }
    __syncthreads();
  }
}

}  // namespace tdbem

using namespace tdbem;

tdbem_status tdbem_build_direct(tdbem_ctx* c) {
  const int64_t ne = c->ne, npair = ne * ne;
  PairStore& st = c->direct;
  st.npairs = npair;
  tdbem_status s;
  int32_t* d_err = nullptr;
  if ((s = c->dalloc(&st.m_lo, npair)) || (s = c->dalloc(&st.nlag, npair)) || (s = c->dalloc(&st.off, npair)) ||
      (s = c->dalloc(&d_err, 1)))
    return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(d_err, 0, sizeof(int32_t), c->stream));
  k_direct_windows<<<(unsigned)((npair + 255) / 256), 256, 0, c->stream>>>(c->tg, c->d_et, ne, c->phys.a, st.m_lo,
                                                                           st.nlag, d_err);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  int64_t* d_tot = nullptr;
  int64_t* d_base = nullptr;
  if ((s = c->dalloc(&d_tot, ne)) || (s = c->dalloc(&d_base, ne))) return s;
  k_row_totals<<<(unsigned)ne, 256, 0, c->stream>>>(st.nlag, ne, d_tot);
  std::vector<int64_t> tot(ne), base(ne);
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(tot.data(), d_tot, ne * sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream));
  int32_t herr = 0;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (herr) {
    c->set_error("direct: lag window out of range (mesh too large relative to c*dt)");
    return TDBEM_EINVAL;
  }
  int64_t acc = 0;
  for (int64_t i = 0; i < ne; ++i) {
    base[i] = acc;
    acc += tot[i];
  }
  st.nval = acc;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(d_base, base.data(), ne * sizeof(int64_t), cudaMemcpyHostToDevice, c->stream));
  k_row_offsets<<<(unsigned)ne, 1024, 0, c->stream>>>(st.nlag, ne, d_base, st.off);
  if ((s = c->dalloc(&st.val, st.nval))) return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(st.val, 0, st.nval * sizeof(double), c->stream));
  // four slots per stored coefficient for the order-independent sum, if the
  // device (and the context's budget) has room; else FP64 atomics
  double* val4 = nullptr;
  const size_t b4 = (size_t)4 * st.nval * sizeof(double);
  const bool fits = c->p.max_device_bytes <= 0 || c->device_bytes + (int64_t)b4 <= c->p.max_device_bytes;
  if (fits && cudaMalloc(&val4, b4) != cudaSuccess) {
    val4 = nullptr;
    cudaGetLastError();  // clear the failed allocation
  }
  if (val4) TDBEM_CUDA_TRY(c, cudaMemsetAsync(val4, 0, b4, c->stream));
  DirectSink sink{st.m_lo, st.nlag, st.off, st.val, ne, val4};
  const int64_t ntp = c->nt * c->nt;
  k_assemble<DirectSink><<<(unsigned)((ntp + 127) / 128), 128, 0, c->stream>>>(c->tg, c->phys, c->nt, nullptr, ntp,
                                                                               sink, d_err);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  if (val4) {
    k_sum4<<<(unsigned)((st.nval + 255) / 256), 256, 0, c->stream>>>(val4, st.nval, st.val);
    cudaError_t e4 = cudaGetLastError();
    cudaStreamSynchronize(c->stream);
    cudaFree(val4);
    TDBEM_CUDA_TRY(c, e4);
  }
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (herr) {
    c->set_error("direct: assembly failed (lag window or light-cone pieces exceed the local buffers), code " +
                 std::to_string(herr));
    return TDBEM_EINVAL;
  }
  // largest stored lag (the history ring holds every step it reaches)
  int32_t mx = 0;
  {
    int32_t* d_mx = nullptr;
    if ((s = c->dalloc(&d_mx, 1))) return s;
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(d_mx, 0, sizeof(int32_t), c->stream));
    k_max_lag<<<1024, 256, 0, c->stream>>>(st.m_lo, st.nlag, npair, d_mx);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
    TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&mx, d_mx, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  }
  c->max_lag = mx;
  return TDBEM_OK;
}

// Incident field of right-hand side r at every step into column r of the
// table (the other columns are kept; a column never set stays zero).
tdbem_status tdbem_incident_table(tdbem_ctx* c, int32_t r) {
  const int64_t ne = c->ne;
  const int64_t n = (int64_t)(c->Nt - 1) * ne * c->R;
  tdbem_status s;
  if (!c->d_Vtab) {
    if ((s = c->dalloc(&c->d_Vtab, n))) return s;
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_Vtab, 0, n * sizeof(double), c->stream));
  }
  const int32_t chunk = 1024;  // steps per launch (grid.y limit)
  for (int32_t a0 = 1; a0 <= c->Nt - 1; a0 += chunk) {
    int32_t na = std::min(chunk, c->Nt - a0);
    dim3 grid((unsigned)((ne + 127) / 128), (unsigned)na);
    k_rhs_plane<<<grid, 128, 0, c->stream>>>(c->tg, c->phys, c->d_et, ne, c->d_pulse + 10 * r, a0, c->R, r,
                                              c->d_Vtab + (int64_t)(a0 - 1) * ne * c->R);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
  }
  return TDBEM_OK;
}

const double* tdbem_incident_row(const tdbem_ctx* c, int32_t alpha) {
  const int64_t stride = c->ne * (int64_t)c->R;
  if (c->d_Vall) return c->d_Vall + (int64_t)(alpha - 1) * stride;
  if (c->have_pulse && c->d_Vtab) return c->d_Vtab + (int64_t)(alpha - 1) * stride;
  return nullptr;
}

// Row-tile kernel shapes (stages x stage bytes, blocks per SM).  The (hi, lo)
// store needs twice the history in shared memory and twice the stage time
// per byte: four 2 KB stages at two blocks per SM.  The FP32 store is bound
// by how many warps keep copies in flight: three 2 KB stages at three blocks
// per SM (on the 7680-RWG sphere, one step per pass, 0.41 ms per launch alone,
// against 0.47 with five stages at two blocks and 0.49 to 0.51 with 1 KB stages).
struct RtShape {
  int ns, sb;
};
constexpr RtShape kRtShape2 = {4, 2048}, kRtShape1 = {3, 2048}, kRtShape3 = {3, 2304};
using RtFn = void (*)(const unsigned char*, const uint32_t*, const uint8_t*, const int32_t*, const int32_t*,
                      const int32_t*, const int32_t*, int64_t, const float2*, int32_t, int32_t, int32_t, int32_t, int32_t,
                      int32_t, int64_t, double*, int32_t*);
// rt_prec 1: FP32 store, 2: (hi, lo) pairs, 3: 24-bit store
template <int B>
static RtFn rt_fn(int prec) {
  if (prec == 1) return k_direct_history_rt<float, B, kRtShape1.ns, kRtShape1.sb, 3>;
  if (prec == 3) return k_direct_history_rt<F24, B, kRtShape3.ns, kRtShape3.sb, 3>;
  return k_direct_history_rt<float2, B, kRtShape2.ns, kRtShape2.sb, 2>;
}
static RtFn rt_fn(int prec, int B) { return B == 1 ? rt_fn<1>(prec) : rt_fn<kRtB>(prec); }
static int rt_group_bytes(int prec) {
  return prec == 1 ? RtPrec<float>::kGroupBytes : prec == 3 ? RtPrec<F24>::kGroupBytes : RtPrec<float2>::kGroupBytes;
}
static size_t rt_smem(int prec, int cbw, int Lh, int m0, int B) {
  const int nh = Lh - m0 + B - 1;
  if (prec == 1) return rt_smem_bytes<float>(kRtShape1.ns, kRtShape1.sb, cbw, nh);
  if (prec == 3) return rt_smem_bytes<F24>(kRtShape3.ns, kRtShape3.sb, cbw, nh);
  return rt_smem_bytes<float2>(kRtShape2.ns, kRtShape2.sb, cbw, nh);
}

// Cost of a launch over n row tiles in each of ncb column blocks of cbw columns,
// `tiles` of them a block, on `slots` resident blocks, in columns a warp sums one
// after the other: rounds of blocks x (tiles of a warp x (columns + 4) + 4), for a
// tile's start-up and a block's staging of its history.
static double rt_cost(int64_t n, int64_t ncb, int64_t slots, int64_t tiles, int cbw) {
  const int64_t blocks = ncb * ((n + tiles - 1) / tiles), per = (std::min(n, tiles) + kRtWarps - 1) / kRtWarps;
  return (double)((blocks + slots - 1) / slots) * (per * (cbw + 4) + 4);
}
static int rt_tiles(int64_t n, int64_t ncb, int64_t slots, int cbw) {
  int64_t best = kRtWarps;
  for (int64_t t = kRtWarps; t <= n + kRtWarps; t += kRtWarps)
    if (rt_cost(n, ncb, slots, t, cbw) < rt_cost(n, ncb, slots, best, cbw)) best = t;
  return (int)best;
}

// The sums of B steps from alpha0 on over row-tile list l (part l of the far tiles,
// or l = rt_B: the near ones), into out ([B][ncb][npos]), on the context's current
// stream.
static tdbem_status direct_rt(tdbem_ctx* c, int32_t alpha0, int B, const float2* rs, int l, double* out) {
  if (!c->rt_lmost[l]) return TDBEM_OK;
  const int m0 = l == c->rt_B ? 3 : rt_m0(c->rt_B, l), tiles = c->rt_ltiles[l];
  const dim3 grid((unsigned)c->rt_ncb, (unsigned)((c->rt_lmost[l] + tiles - 1) / tiles));
  rt_fn(c->rt_prec, B)<<<grid, kRtWarps * 32, rt_smem(c->rt_prec, c->rt_cbw, c->rt_Lh, m0, B), c->stream>>>(
      c->d_rt_val, c->d_rt_goff, c->d_rt_lo, c->d_rt_lomin, c->rt_units ? nullptr : c->d_rt_row, c->d_rt_list,
      c->d_rt_loff + (int64_t)l * c->rt_ncb, c->ne, rs, c->L, c->rt_Lh, alpha0, m0, tiles, c->rt_cbw,
      (int64_t)c->rt_nrt * 32, out, c->d_dt_err);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  return TDBEM_OK;
}

// The near pairs' sums of step alpha into the near partials of buffer buf, on
// the context's current stream.
static double* near_out(const tdbem_ctx* c, int buf) {
  return c->d_dpart + (int64_t)buf * c->rt_nslot * c->rt_nrt * 32;
}
static tdbem_status direct_near(tdbem_ctx* c, int32_t alpha, const float2* rs, int buf) {
  if (c->rt_units) return c->rt_B > 1 ? direct_rt(c, alpha, 1, rs, c->rt_B, near_out(c, buf)) : TDBEM_OK;
  if (!c->rt_nchunk) return TDBEM_OK;
  k_direct_near<<<(unsigned)((c->rt_nchunk + 7) / 8), 256, 0, c->stream>>>(c->d_nt_val, c->d_nt_qoff, c->d_nt_meta, c->d_nt_chunk,
                                                                c->rt_nchunk, rs, c->L, alpha, (int64_t)c->rt_nrt * 32,
                                                                near_out(c, buf));
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  return TDBEM_OK;
}

// pre of buffer buf from nfar far partials and the buffer's near partials.
static tdbem_status direct_presum(tdbem_ctx* c, const double* far, int nfar, int buf) {
  const int64_t npos = (int64_t)c->rt_nrt * 32;
  const int both = c->rt_units && c->rt_B > 1;
  k_direct_presum<<<(unsigned)c->rt_nrt, kRedLanes * 32, 0, c->stream>>>(far, nfar, near_out(c, buf), c->rt_nslot, both,
                                                                        npos, c->d_pre + buf * kRedLanes * npos);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  return TDBEM_OK;
}

// The march's block of steps that holds alpha: its first step, and its partial buffer.
static int32_t far_block(const tdbem_ctx* c, int32_t alpha) { return (alpha - 1) / c->rt_B * c->rt_B + 1; }
static int far_buf(const tdbem_ctx* c, int32_t a0) { return ((a0 - 1) / c->rt_B) & 1; }
static double* far_out(const tdbem_ctx* c, int buf) {
  return c->d_fpart + (int64_t)buf * c->rt_B * c->rt_ncb * c->rt_nrt * 32;
}
// whether any far pair of the block's steps reaches a current (J^0 is the first)
static bool far_any(const tdbem_ctx* c, int32_t a0) { return a0 + c->rt_B - 1 >= rt_m0(c->rt_B, c->rt_B - 1); }

// The far buffer of block a0 made this block's, the context's current stream
// behind the parts of it launched on the side stream.
static tdbem_status far_parts_wait(tdbem_ctx* c, int32_t a0) {
  const int fb = far_buf(c, a0);
  if (c->far_blk[fb] != a0) {
    c->far_blk[fb] = a0;
    c->far_done[fb] = 0;
  } else if (c->far_wait[fb] && c->stream != c->dstream) {
    TDBEM_CUDA_TRY(c, cudaStreamWaitEvent(c->stream, c->ev_far[fb], 0));
  }
  if (c->stream != c->dstream) c->far_wait[fb] = false;
  return TDBEM_OK;
}

// The split history of a ring: the march's own is kept up to date by the solve.
static tdbem_status split_ring(tdbem_ctx* c, const double* ring, float2* rs) {
  const int64_t n = c->ne * (int64_t)c->L;
  k_ring_pairs<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(ring, n, rs);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  return TDBEM_OK;
}

tdbem_status tdbem_direct_resplit(tdbem_ctx* c) {
  return c->d_rs ? split_ring(c, c->d_Jring, c->d_rs) : TDBEM_OK;
}

tdbem_status tdbem_direct_history(tdbem_ctx* c, int32_t alpha, const double* d_ring, const double* V) {
  const PairStore& st = c->direct;
  if (c->R == 1 && c->rt_prec) {
    // the march's own ring uses the buffers alpha & 1 (near, pre) and the far
    // buffers of its blocks, possibly filled ahead during earlier steps; any other
    // history buffer 2 and the far buffer behind the two
    const bool march = d_ring == c->d_Jring;
    const int64_t npos = (int64_t)c->rt_nrt * 32;
    const float2* rs = march ? c->d_rs : c->d_rs_eval;
    const int buf = march ? (alpha & 1) : 2;
    tdbem_status s;
    if (march && c->dahead[buf] == alpha) {
      TDBEM_CUDA_TRY(c, cudaStreamWaitEvent(c->stream, c->ev_dahead[buf], 0));
    } else {
      if (!march && (s = split_ring(c, d_ring, c->d_rs_eval))) return s;
      const double* far = far_out(c, 2);
      int nfar = c->rt_ncb;
      cudaEvent_t e = c->prof_begin(1);
      if ((s = direct_near(c, alpha, rs, buf))) return s;
      if (!march) {
        for (int q = 0; q < c->rt_B; ++q)
          if ((s = direct_rt(c, alpha, 1, rs, q, far_out(c, 2)))) return s;
      } else {
        const int32_t a0 = far_block(c, alpha);
        const int fb = far_buf(c, a0);
        far = far_out(c, fb) + (int64_t)(alpha - a0) * c->rt_ncb * npos;
        if (!far_any(c, a0)) {
          nfar = 0;
        } else {
          if ((s = far_parts_wait(c, a0))) return s;
          // the parts not summed ahead, now
          for (int q = 0; q < c->rt_B; ++q)
            if (!(c->far_done[fb] >> q & 1) && (s = direct_rt(c, a0, c->rt_B, rs, q, far_out(c, fb)))) return s;
          c->far_done[fb] = (1 << c->rt_B) - 1;
        }
      }
      if ((s = direct_presum(c, far, nfar, buf))) return s;
      c->prof_end(1, e);
    }
    if (march) c->dahead[buf] = 0;
    cudaEvent_t e = c->prof_begin(10);
    k_direct_reduce<<<(unsigned)((npos * kRedLanes + 127) / 128), 128, 0, c->stream>>>(
        c->d_pre + buf * kRedLanes * npos, c->d_rt_row, npos, c->d_l2_ptr, c->d_l2_col, c->d_l2_val, d_ring, c->L, alpha, V, c->d_R);
    c->prof_end(10, e);
  } else if (c->R == 1) {
    if (!c->d_ring2 || !st.val) {
      c->set_error("direct: untiled history sum without its split ring");
      return TDBEM_ESTATE;
    }
    cudaEvent_t e = c->prof_begin(9);
    const int64_t n = c->ne * (int64_t)c->L;
    k_ring_split<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(d_ring, c->ne, c->L, c->d_ring2);
    c->prof_end(9, e);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
    e = c->prof_begin(1);
    k_direct_history<<<(unsigned)c->ne, kDhThreads, 2 * kDhCap * sizeof(float2), c->stream>>>(
        st.m_lo, st.nlag, st.off, reinterpret_cast<const float2*>(st.val), c->ne, c->d_ring2, c->L, alpha, V, c->d_R);
    c->prof_end(1, e);
  } else {
    int RL = 1;
    while (RL < c->R && RL < 32) RL <<= 1;
    cudaEvent_t e = c->prof_begin(1);
    k_direct_history_multi<<<(unsigned)c->ne, 256, 0, c->stream>>>(st.m_lo, st.nlag, st.off, st.val, c->ne, d_ring,
                                                                   c->L, alpha, c->R, RL, V, c->d_R);
    c->prof_end(1, e);
  }
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  return TDBEM_OK;
}

// After step alpha's solve is enqueued, on the side stream beside step alpha + 1
// (its reduction, lag-2 entries and solve): the near pairs of step alpha + 2,
// which need the currents up to J^{alpha-1} only, one part of the far sums of
// the block after the next block boundary, and step alpha + 2's pre.  With a0
// the first step of the block at hand, the parts of the block a0 + B ..
// a0 + 2 B - 1 are launched after the solves of the steps a0 - 1 .. a0 + B - 2,
// the last of them just before its first step's pre; the newest current they
// part q reads is J^{a0 + 2 B - 1 - M0}, J^{a0 - 2 + q} for M0 = 2 B + 1 - q, known
// after the solve of step a0 - 1 + q (B = 1: J^{alpha-1} for step alpha + 2).  The
// steps solved meanwhile write J^{a0-1} .. J^{a0+B-2}: the oldest current read,
// J^{a0 + B - max_lag}, is at most L - 1 steps older, so no ring slot is shared.
// The buffers were last read by kernels ordered before this solve.  A step whose
// block will not be complete by then (the first block of a march or after a load)
// sums its near pairs itself, so every launch here lies before an event that is
// waited for: that of the far part, or that of the step's pre.
tdbem_status tdbem_direct_after_solve(tdbem_ctx* c, int32_t alpha) {
  if (!c->dstream || !c->rt_prec || c->R != 1) return TDBEM_OK;
  const int32_t a2 = alpha + 2, af = alpha / c->rt_B * c->rt_B + 1 + c->rt_B;
  const bool far = af <= c->Nt - 1 && far_any(c, af);
  if (a2 > c->Nt - 1) return TDBEM_OK;  // af >= a2
  // step alpha + 2's block, and whether its far sums are complete behind the side stream, this call's part included
  const int32_t a0 = far_block(c, a2);
  const int fb0 = far_buf(c, a0), q = alpha % c->rt_B;
  const bool any = far_any(c, a0);
  const int done = (c->far_blk[fb0] == a0 ? c->far_done[fb0] : 0) | (far && af == a0 ? 1 << q : 0);
  const bool whole = !any || done == (1 << c->rt_B) - 1;
  if (!far && !whole) return TDBEM_OK;
  TDBEM_CUDA_TRY(c, cudaEventRecord(c->ev_dsolved, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamWaitEvent(c->dstream, c->ev_dsolved, 0));
  cudaStream_t main = c->stream;
  c->stream = c->dstream;
  auto ahead = [&]() -> tdbem_status {
    const int b = a2 & 1;
    tdbem_status s;
    cudaEvent_t e = c->prof_begin(1);
    if (whole && (s = direct_near(c, a2, c->d_rs, b))) return s;
    if (far) {
      const int fb = far_buf(c, af);
      if ((s = far_parts_wait(c, af)) || (s = direct_rt(c, af, c->rt_B, c->d_rs, q, far_out(c, fb)))) return s;
      TDBEM_CUDA_TRY(c, cudaEventRecord(c->ev_far[fb], c->dstream));
      c->far_done[fb] |= 1 << q;
      c->far_wait[fb] = true;
    }
    if (whole) {
      if ((s = direct_presum(c, far_out(c, fb0) + (int64_t)(a2 - a0) * c->rt_ncb * c->rt_nrt * 32, any ? c->rt_ncb : 0, b)))
        return s;
      c->dahead[b] = a2;
      TDBEM_CUDA_TRY(c, cudaEventRecord(c->ev_dahead[b], c->dstream));
    }
    c->prof_end(1, e);
    return TDBEM_OK;
  };
  const tdbem_status s = ahead();
  c->stream = main;
  return s;
}

// ETIMEOUT if a bounded wait of the row-tile history sum expired (its partial
// sums are NaN then, so the step's solve also misses its tolerance).
tdbem_status tdbem_direct_check(tdbem_ctx* c) {
  if (!c->d_dt_err) return TDBEM_OK;
  tdbem_status s = tdbem_direct_join(c);
  if (s) return s;
  int32_t h = 0;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&h, c->d_dt_err, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (h) {
    c->set_error("direct: a bounded wait of the history sum expired");
    return TDBEM_ETIMEOUT;
  }
  return TDBEM_OK;
}

// The context's stream waits for the sums launched ahead (they stay usable).
tdbem_status tdbem_direct_join(tdbem_ctx* c) {
  for (int b = 0; b < 2; ++b) {
    if (c->dahead[b]) TDBEM_CUDA_TRY(c, cudaStreamWaitEvent(c->stream, c->ev_dahead[b], 0));
    if (c->far_wait[b]) TDBEM_CUDA_TRY(c, cudaStreamWaitEvent(c->stream, c->ev_far[b], 0));
  }
  return TDBEM_OK;
}

// As tdbem_direct_join, and the sums launched ahead are discarded.
tdbem_status tdbem_direct_invalidate(tdbem_ctx* c) {
  tdbem_status s = tdbem_direct_join(c);
  for (int b = 0; b < 2; ++b) {
    c->dahead[b] = c->far_blk[b] = c->far_done[b] = 0;
    c->far_wait[b] = false;
  }
  return s;
}

void tdbem_direct_free(tdbem_ctx* c) {
  if (c->dstream) cudaStreamSynchronize(c->dstream);
  if (c->ev_dsolved) cudaEventDestroy(c->ev_dsolved);
  for (int b = 0; b < 2; ++b) {
    if (c->ev_dahead[b]) cudaEventDestroy(c->ev_dahead[b]);
    if (c->ev_far[b]) cudaEventDestroy(c->ev_far[b]);
  }
  if (c->dstream) cudaStreamDestroy(c->dstream);
  c->dstream = nullptr;
}

template <typename T>
static tdbem_status up(tdbem_ctx* c, T** d, const std::vector<T>& h) {
  tdbem_status s = c->dalloc(d, h.size());
  if (s) return s;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, c->stream));
  return TDBEM_OK;
}

// Edges in an order whose runs of 8, 32, 64, .. lie close together: their
// midpoints (mean of the two triangles' centroids) are halved along the longest
// side of their box, at multiples of 32 (below that of 8), until 8 are left.
static std::vector<int32_t> bisected_edges(const tdbem_ctx* c) {
  const int64_t ne = c->ne;
  std::vector<double> mid(3 * ne);
  std::vector<int32_t> order(ne);
  for (int64_t e = 0; e < ne; ++e) {
    order[e] = (int32_t)e;
    for (int d = 0; d < 3; ++d) {
      double x = 0.0;
      for (int side = 0; side < 2; ++side)
        for (int q = 0; q < 3; ++q) x += c->V[3 * c->T[3 * c->et[2 * e + side] + q] + d];
      mid[3 * e + d] = x / 6.0;
    }
  }
  std::vector<std::pair<int64_t, int64_t>> todo = {{0, ne}};
  while (!todo.empty()) {
    const int64_t b = todo.back().first, e = todo.back().second;
    todo.pop_back();
    if (e - b <= 8) continue;
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    for (int64_t k = b; k < e; ++k)
      for (int d = 0; d < 3; ++d) {
        lo[d] = std::min(lo[d], mid[3 * order[k] + d]);
        hi[d] = std::max(hi[d], mid[3 * order[k] + d]);
      }
    int ax = 0;
    for (int d = 1; d < 3; ++d)
      if (hi[d] - lo[d] > hi[ax] - lo[ax]) ax = d;
    const int64_t unit = e - b > 32 ? 32 : 8, m = b + std::max(unit, (e - b) / 2 / unit * unit);
    std::nth_element(order.begin() + b, order.begin() + m, order.begin() + e, [&](int32_t x, int32_t y) {
      const double u = mid[3 * x + ax], v = mid[3 * y + ax];
      return u != v ? u < v : x < y;
    });
    todo.push_back({b, m});
    todo.push_back({m, e});
  }
  return order;
}

// Builds the row-tile store of the lags >= 3 from the FP64 store (prec 1: FP32
// values, 2: (hi, lo) pairs, 3: 24-bit values), frees the FP64 values and sets
// the grid.
static tdbem_status build_row_tiles(tdbem_ctx* c, int prec) {
  PairStore& st = c->direct;
  const int64_t ne = c->ne, nrt = (ne + 31) / 32, ntc = nrt * ne;
  tdbem_status s;
  // Steps per pass: kRtB where the store is larger than a good part of L2, so
  // that each pass comes from HBM; below that one step per pass, a step ahead.
  const int B = st.nval * rt_group_bytes(prec) / 32 >= kRtBlockBytes && ne < (1 << 24) && !c->lean ? kRtB : 1;
  // Columns per block: the width whose blocks fill the SMs best beside the 16 SMs
  // of an overlapped solve (the same width for either order of the steps).  The
  // blocks are small, a row tile per warp, so that tiles passed over early in a
  // march and SMs taken by the solve leave no long tail: on the 7680-RWG sphere
  // 60 tiles x 120 blocks a part in blocks of 20 tiles left a third of the slots idle.
  int nsm = 0, smem_max = 0, smem_sm = 0;
  TDBEM_CUDA_TRY(c, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  TDBEM_CUDA_TRY(c, cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device));
  TDBEM_CUDA_TRY(c, cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, c->device));
  const int units = prec != 2;  // FP32 and 24-bit: whole units of 64 columns in edge order
  const int m0 = units ? 3 : rt_m0(B, B - 1), most = prec == 2 ? 2 : 3;  // blocks per SM the registers allow
  int cbw = 64;
  if (!units && !c->lean) {
    const int lag = std::min(255, c->max_lag + 6), sms = nsm > 32 ? nsm - 16 : nsm;
    double best = 1e300;
    for (int w = 8; w <= 96; w += 2) {
      const size_t smem = rt_smem(prec, w, lag, m0, B) + 1024;
      if (smem > (size_t)smem_max) break;
      const int64_t slots = (int64_t)std::min<size_t>(most, smem_sm / smem) * sms, n = (ne + w - 1) / w;
      const double cost = rt_cost((nrt + B - 1) / B, n, slots, kRtWarps, w) / (smem_sm / smem >= (size_t)most ? 1.0 : 0.8);
      if (cost < best) {
        best = cost;
        cbw = w;
      }
    }
  }
  const int ncb = (int)((ne + cbw - 1) / cbw);
  const bool quads = B > 1 && !units;
  uint8_t *d_nmax = nullptr, *d_nnear = nullptr;
  int32_t *d_lh = nullptr, *d_lomin = nullptr;
  if ((s = c->dalloc(&d_nmax, ntc)) || (quads && (s = c->dalloc(&d_nnear, 4 * ntc))) ||
      (s = c->dalloc(&c->d_rt_lo, ntc * 32)) || (s = c->dalloc(&d_lomin, nrt * ncb)) || (s = c->dalloc(&d_lh, 1)) ||
      (s = c->dalloc(&c->d_dt_err, 1)))
    return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(d_lh, 0, sizeof(int32_t), c->stream));
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_dt_err, 0, sizeof(int32_t), c->stream));
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(d_lomin, 0x7f, nrt * ncb * sizeof(int32_t), c->stream));
  const unsigned nb = (unsigned)((ntc * 32 + 255) / 256);
  k_rt_meta<<<nb, 256, 0, c->stream>>>(st.m_lo, st.nlag, ne, (int32_t)nrt, c->d_rt_row, B, units, d_nmax, d_nnear,
                                       c->d_rt_lo, d_lomin, ncb, cbw, d_lh);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  std::vector<uint8_t> nmax(ntc), nnear(quads ? 4 * ntc : 0);
  std::vector<int32_t> rows(nrt * 32), lm(nrt * ncb);
  int32_t lh = 0;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(nmax.data(), d_nmax, ntc, cudaMemcpyDeviceToHost, c->stream));
  if (quads) TDBEM_CUDA_TRY(c, cudaMemcpyAsync(nnear.data(), d_nnear, 4 * ntc, cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(rows.data(), c->d_rt_row, nrt * 32 * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(lm.data(), d_lomin, lm.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&lh, d_lh, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  // (what the march alone reads comes back when the FP64 values are gone: the two stores side by side are the peak)
  c->dfree(d_nmax);
  c->dfree(d_nnear);
  c->dfree(d_lomin);
  c->dfree(d_lh);
  std::vector<uint32_t> goff(ntc + 1);
  uint64_t acc = 0;
  for (int64_t k = 0; k < ntc; ++k) {
    goff[k] = (uint32_t)acc;
    acc += nmax[k];
  }
  // the near quads: a sub-tile's columns, longest windows first, by fours; chunks of about kNearGroups groups
  std::vector<int32_t> qst, qcol;
  std::vector<uint32_t> qoff;
  std::vector<int4> chunks;
  std::vector<std::pair<int, int32_t>> cols;  // {-lags, column position}
  uint64_t nacc = 0;
  int nslot = 0;
  for (int64_t sub = 0; quads && sub < 4 * nrt; ++sub) {
    cols.clear();
    for (int64_t j = 0; j < ne; ++j)
      if (nnear[sub * ne + j]) cols.push_back({-(int)nnear[sub * ne + j], (int32_t)j});
    std::sort(cols.begin(), cols.end());
    int slot = 0, groups = kNearGroups;
    for (size_t k = 0; k < cols.size(); k += 4) {
      if (groups >= kNearGroups) {
        chunks.push_back(make_int4((int)sub, (int)qst.size(), (int)qst.size(), slot++));
        groups = 0;
      }
      qst.push_back((int32_t)sub);
      for (size_t m = k; m < k + 4; ++m) qcol.push_back(m < cols.size() ? rows[cols[m].second] : -1);
      qoff.push_back((uint32_t)nacc);
      nacc += -cols[k].first;
      groups += -cols[k].first;
      chunks.back().z = (int)qst.size();
    }
    nslot = std::max(nslot, slot);
  }
  qoff.push_back((uint32_t)nacc);
  const int Lh = std::max(lh, rt_m0(B, 0) + 1);
  const bool fits = acc < (1ull << 32) && nacc < (1ull << 32) && lh <= 255 &&
                    rt_smem(prec, cbw, Lh, m0, B) + 1024 <= (size_t)smem_max;
  if (!fits && prec == 2) {  // the untiled kernel takes it
    c->dfree(c->d_rt_lo);
    c->d_rt_lo = nullptr;
    return TDBEM_OK;
  }
  if (!fits) {
    c->set_error("direct: row-tile store too large (32-bit group offsets, 8-bit first lags)");
    return TDBEM_EINVAL;
  }
  goff[ntc] = (uint32_t)acc;
  const size_t nbytes = (size_t)acc * rt_group_bytes(prec), nearbytes = (size_t)nacc * 32 * sizeof(float2);
  const int64_t nq = (int64_t)qst.size();
  int32_t *d_qst = nullptr, *d_qcol = nullptr;
  if ((s = up(c, &c->d_rt_goff, goff)) || (s = c->dalloc(&c->d_rt_val, nbytes)) || (s = up(c, &d_qst, qst)) ||
      (s = up(c, &d_qcol, qcol)) || (s = up(c, &c->d_nt_qoff, qoff)) || (s = up(c, &c->d_nt_chunk, chunks)) ||
      (s = c->dalloc(&c->d_nt_meta, (size_t)nq * 32)) || (s = c->dalloc(&c->d_nt_val, (size_t)nacc * 32)))
    return s;
  auto fill = prec == 1 ? k_rt_fill<float> : prec == 3 ? k_rt_fill<F24> : k_rt_fill<float2>;
  fill<<<nb, 256, 0, c->stream>>>(st.m_lo, st.nlag, st.off, st.val, ne, (int32_t)nrt, c->d_rt_row, B, units, c->d_rt_goff,
                                  c->d_rt_val);
  if (nq) {
    k_near_fill<<<(unsigned)((nq * 32 + 255) / 256), 256, 0, c->stream>>>(st.m_lo, st.nlag, st.off, st.val, ne, (int32_t)nrt,
                                                                    nq, c->d_rt_row, B, d_qst, d_qcol, c->d_nt_qoff,
                                                                    c->d_nt_meta, c->d_nt_val);
  }
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  // the host vectors and the FP64 values are read by the copies and the fill: wait before they go
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  c->dfree(d_qst);
  c->dfree(d_qcol);
  c->dfree(st.val);
  st.val = nullptr;
  c->rt_B = B;
  c->rt_nrt = (int32_t)nrt;
  c->rt_Lh = Lh;
  c->rt_prec = prec;
  c->rt_nchunk = (int32_t)chunks.size();
  c->rt_units = units;
  c->rt_nslot = units && B > 1 ? ncb : nslot;
  // streamed per step: the far pairs' share once per B steps, the near ones each step
  int64_t whole = (int64_t)nbytes + ntc * 32 + (ntc + 1) * 4, near = (int64_t)nearbytes + nq * (128 + 4);
  std::vector<int32_t> list, loff(1, 0);
  for (int l = 0; l <= B; ++l) {  // the far tiles of each part, then the near ones
    int most_tiles = 0;
    for (int cb = 0; cb < ncb; ++cb) {
      const size_t b0 = list.size();
      for (int64_t rt = 0; rt < nrt; ++rt) {
        const int q = rt_part(rt, nrt, B), v = lm[rt * ncb + cb];
        if (v > 255) continue;  // no lags
        const bool near_unit = units && B > 1 && v < rt_m0(B, q);
        if (near_unit ? l == B : l == q) list.push_back((int32_t)rt);
        if (near_unit && l == B) {
          const int64_t k0 = rt * ne + (int64_t)cb * cbw, k1 = rt * ne + std::min<int64_t>(ne, (int64_t)(cb + 1) * cbw);
          near += (int64_t)(goff[k1] - goff[k0]) * rt_group_bytes(prec) + (k1 - k0) * 36;
        }
      }
      std::stable_sort(list.begin() + b0, list.end(),
                       [&](int32_t x, int32_t y) { return lm[(int64_t)x * ncb + cb] < lm[(int64_t)y * ncb + cb]; });
      loff.push_back((int32_t)list.size());
      most_tiles = std::max(most_tiles, (int)(list.size() - b0));
    }
    c->rt_lmost[l] = most_tiles;
    const size_t smem = rt_smem(prec, cbw, Lh, l == B ? 3 : rt_m0(B, l), l == B ? 1 : B) + 1024;
    const int64_t slots = (int64_t)std::min<size_t>(most, std::max<size_t>(1, smem_sm / smem)) * (nsm > 32 ? nsm - 16 : nsm);
    // the far parts: a tile per warp; the near units, fewer and unevenly spread: by the cost
    c->rt_ltiles[l] = l < B ? kRtWarps : rt_tiles(std::max(1, most_tiles), ncb, slots, cbw);
  }
  if ((s = up(c, &c->d_rt_list, list)) || (s = up(c, &c->d_rt_loff, loff)) || (s = up(c, &c->d_rt_lomin, lm))) return s;
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));  // the vectors go
  if (units && B > 1) whole -= near;
  c->rt_bytes = whole / B + near;
  // the most the device allows: other contexts launch the kernel with other sizes
  for (int b : {B, 1})
    TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(rt_fn(prec, b), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
  c->rt_cbw = cbw;
  c->rt_ncb = ncb;
  return TDBEM_OK;
}

// Single right-hand side, after Z0 and the lag-2 entries have been read from
// the FP64 store: the row-tile store of the lags >= 3 in the precision of
// p2p_prec (rings of up to 128 steps, 256 in (hi, lo) pairs), which replaces the FP64 values; else the
// FP64 values split in place into (hi, lo) pairs for the untiled kernel and
// its split ring.
tdbem_status tdbem_direct_split(tdbem_ctx* c) {
  if (c->R != 1) return TDBEM_OK;
  PairStore& st = c->direct;
  // The row-tile store's first lags are bytes and its history of a column block
  // lies in shared memory: rings of up to 256 steps in (hi, lo) pairs.  It is built beside the FP64 values, where the
  // untiled form turns them into pairs in place: the memory of a lean context has no room for that beyond 128 steps.
  const bool tiled = c->L <= 128 || (c->L <= 256 && c->p.p2p_prec == TDBEM_P_FP64 && !c->lean);
  if (tiled) {
    // the row order, and the lag-2 entries (read from the FP64 store before the row tiles replace it)
    const int64_t ne = c->ne, nrt = (ne + 31) / 32, npos = nrt * 32;
    std::vector<int32_t> rows, cnt(npos), ptr(npos + 1, 0);
    if (c->lean)  // the numbering's own order, whose store may be smaller (UV ellipsoid of 2,880 RWG: by a tenth)
      for (int32_t e = 0; e < ne; ++e) rows.push_back(e);
    else
      rows = bisected_edges(c);
    rows.resize(npos, -1);
    tdbem_status s0;
    if ((s0 = up(c, &c->d_rt_row, rows)) || (s0 = c->dalloc(&c->d_l2_ptr, npos + 1))) return s0;
    const unsigned nb = (unsigned)((npos * 32 + 255) / 256);
    k_lag2<<<nb, 256, 0, c->stream>>>(st.m_lo, st.nlag, st.off, st.val, ne, npos, c->d_rt_row, 0, c->d_l2_ptr, nullptr,
                                      nullptr);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
    // the counts come from the context's stream: copy on it and wait
    TDBEM_CUDA_TRY(c, cudaMemcpyAsync(cnt.data(), c->d_l2_ptr, npos * sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
    TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    int64_t total = 0;
    for (int64_t p = 0; p < npos; ++p) {
      total += cnt[p];
      ptr[p + 1] = (int32_t)total;
    }
    if (total >= (1ll << 31)) {
      c->set_error("direct: too many lag-2 entries (32-bit offsets)");
      return TDBEM_EINVAL;
    }
    TDBEM_CUDA_TRY(c, cudaMemcpyAsync(c->d_l2_ptr, ptr.data(), (npos + 1) * sizeof(int32_t), cudaMemcpyHostToDevice,
                                      c->stream));
    if ((s0 = c->dalloc(&c->d_l2_col, std::max<int64_t>(1, total))) ||
        (s0 = c->dalloc(&c->d_l2_val, std::max<int64_t>(1, total))))
      return s0;
    k_lag2<<<nb, 256, 0, c->stream>>>(st.m_lo, st.nlag, st.off, st.val, ne, npos, c->d_rt_row, 1, c->d_l2_ptr,
                                      c->d_l2_col, c->d_l2_val);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
    TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));  // before rows and ptr (host) go out of scope
  }
  if (!tiled && c->p.p2p_prec != TDBEM_P_FP64) {
    c->set_error("p2p_prec FP32 and FP24 need one right-hand side and a history ring of at most 128 steps");
    return TDBEM_EINVAL;
  }
  if (tiled) {
    tdbem_status s =
        build_row_tiles(c, c->p.p2p_prec == TDBEM_P_FP32 ? 1 : c->p.p2p_prec == TDBEM_P_FP24 ? 3 : 2);
    if (s) return s;
  }
  if (c->rt_prec) {
    tdbem_status s;
    const size_t npos = (size_t)c->rt_nrt * 32, nn = 3 * c->rt_nslot * npos, nf = (2 * c->rt_B + 1) * c->rt_ncb * npos;
    const size_t nr = (size_t)c->ne * c->L;
    if ((s = c->dalloc(&c->d_dpart, nn)) || (s = c->dalloc(&c->d_fpart, nf)) || (s = c->dalloc(&c->d_pre, 3 * kRedLanes * npos)) || (s = c->dalloc(&c->d_rs, nr)) ||
        (s = c->dalloc(&c->d_rs_eval, nr)))
      return s;
    // a tile with fewer near chunks than nslot leaves its last slots zero
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_dpart, 0, std::max<size_t>(nn, 1) * sizeof(double), c->stream));
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_fpart, 0, nf * sizeof(double), c->stream));
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_rs, 0, nr * sizeof(float2), c->stream));
    TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_rs_eval, 0, nr * sizeof(float2), c->stream));
    if (c->p.far_overlap) {
      // between the library stream's highest priority and the lowest: the
      // next solve's cluster is dispatched ahead of this stream's blocks
      int prio_lo = 0, prio_hi = 0;
      TDBEM_CUDA_TRY(c, cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi));
      TDBEM_CUDA_TRY(c, cudaStreamCreateWithPriority(&c->dstream, cudaStreamNonBlocking, (prio_lo + prio_hi) / 2));
      TDBEM_CUDA_TRY(c, cudaEventCreateWithFlags(&c->ev_dsolved, cudaEventDisableTiming));
      for (int b = 0; b < 2; ++b) {
        TDBEM_CUDA_TRY(c, cudaEventCreateWithFlags(&c->ev_dahead[b], cudaEventDisableTiming));
        TDBEM_CUDA_TRY(c, cudaEventCreateWithFlags(&c->ev_far[b], cudaEventDisableTiming));
      }
    }
    return TDBEM_OK;
  }
  k_split_values<<<(unsigned)((st.nval + 255) / 256), 256, 0, c->stream>>>(st.val, st.nval);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  TDBEM_CUDA_TRY(c, cudaFuncSetAttribute(k_direct_history, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(2 * kDhCap * sizeof(float2))));
  tdbem_status s = c->dalloc(&c->d_ring2, c->ne * (int64_t)c->L);
  if (s) return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(c->d_ring2, 0, c->ne * (int64_t)c->L * sizeof(float2), c->stream));
  return TDBEM_OK;
}

// Assemble the listed (test triangle, source triangle) pairs into a CSR store
// of edge pairs (the near field of fast mode).  row_ptr/col must already hold
// every edge pair touched by the listed triangle pairs.
tdbem_status tdbem_assemble_csr(tdbem_ctx* c, const int2* d_pairs, int64_t npairs, const int64_t* d_row_ptr,
                                const int32_t* d_col, int64_t nnz, int16_t** m_lo, uint8_t** nlag, int64_t** off,
                                double** val, int64_t* nval) {
  tdbem_status s;
  int32_t* d_err = nullptr;
  if ((s = c->dalloc(m_lo, nnz)) || (s = c->dalloc(nlag, nnz)) || (s = c->dalloc(off, nnz)) ||
      (s = c->dalloc(&d_err, 1)))
    return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(d_err, 0, sizeof(int32_t), c->stream));
  k_csr_windows<<<(unsigned)c->ne, 128, 0, c->stream>>>(c->tg, c->d_et, d_row_ptr, d_col, c->ne, c->phys.a, *m_lo,
                                                        *nlag, d_err);
  TDBEM_CUDA_TRY(c, cudaGetLastError());
  std::vector<uint8_t> hn(nnz);
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(hn.data(), *nlag, nnz, cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  std::vector<int64_t> ho(nnz);
  int64_t acc = 0;
  for (int64_t p = 0; p < nnz; ++p) {
    ho[p] = acc;
    acc += hn[p];
  }
  *nval = acc;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(*off, ho.data(), nnz * sizeof(int64_t), cudaMemcpyHostToDevice, c->stream));
  if ((s = c->dalloc(val, acc))) return s;
  TDBEM_CUDA_TRY(c, cudaMemsetAsync(*val, 0, acc * sizeof(double), c->stream));
  CsrSink sink{d_row_ptr, d_col, *m_lo, *nlag, *off, *val};
  if (npairs > 0) {
    k_assemble<CsrSink><<<(unsigned)((npairs + 127) / 128), 128, 0, c->stream>>>(c->tg, c->phys, c->nt, d_pairs,
                                                                                npairs, sink, d_err);
    TDBEM_CUDA_TRY(c, cudaGetLastError());
  }
  int32_t herr = 0;
  TDBEM_CUDA_TRY(c, cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
  TDBEM_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (herr) {
    c->set_error("near field: assembly failed, code " + std::to_string(herr));
    return TDBEM_EINVAL;
  }
  return TDBEM_OK;
}

// Inner level of the nested method, in double precision (Sec. 3, Eqs. (nested),
// (precond); Sec. 2, Eq. (Roberts)).
//
//  k_inner   one CTA per problem: tridiagonal LU with partial pivoting of the Ritz
//            matrix H_k (row interchanges between neighbouring rows only), then l steps
//            of Lanczos (mu = 0) or two-sided Lanczos (mu != 0) on M = H_k + H_k^{-1}
//            from e_1. M u = H u + H^{-1} u and M^dag w = H^dag w + H^{-dag} w both use
//            the one factorisation (the solve with H^dag runs the factors backwards).
//  k_rh_col  one CTA per matrix: the first column of a Roberts-Higham iterate of T_l by
//            partial fractions (the nested checks in double-float arithmetic).
//  k_rh      one CTA per matrix: Roberts-Higham S_{n+1} = (S_n + S_n^{-1})/2 with an
//            in-place Gauss-Jordan inversion (partial pivoting) of the whole l x l
//            matrix in shared memory (l <= 120 complex: 225 KB).
//  k_combine a cluster of CTAs per problem: c = Q_l s and the inner estimate against the
//            leading (l - dl) block; k_estimate: the outer estimate against the previous check.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "ov_internal.h"
#include "ov_types.cuh"

namespace ov {

constexpr int kInnerThreads = 256;

__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 zscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double zabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
  // scaled to avoid overflow of |b|^2 for large |b|
  double s = fmax(fabs(b.x), fabs(b.y));
  if (s == 0.0) return make_double2(INFINITY, INFINITY);
  double2 bs = make_double2(b.x / s, b.y / s), as = make_double2(a.x / s, a.y / s);
  double d = bs.x * bs.x + bs.y * bs.y;
  return make_double2((as.x * bs.x + as.y * bs.y) / d, (as.y * bs.x - as.x * bs.y) / d);
}
__device__ __forceinline__ double2 zinv(double2 b) { return zdiv(make_double2(1.0, 0.0), b); }

// block sum over kInnerThreads threads; result returned to every thread
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;
}

struct InnerSmem {
  double2 *d, *a, *c;           // H diagonal, subdiagonal (row m, col m-1), superdiagonal (row m, col m+1)
  double2 *uinv, *u1, *u2, *l;  // LU factors
  unsigned char* sw;            // row interchange at step m
  double2 *q, *qp, *w, *wp, *u, *z;
  double* red;
};

// x = H^{-1} b with the GEPP factors (x may alias nothing; y is scratch of size k)
__device__ void tri_solve(const InnerSmem& S, int k, const double2* b, double2* x) {
  double2 cur = b[0];
  for (int m = 0; m < k - 1; ++m) {
    const double2 nb = b[m + 1];
    if (!S.sw[m]) {
      x[m] = cur;
      cur = zsub(nb, zmul(S.l[m], cur));
    } else {
      x[m] = nb;
      cur = zsub(cur, zmul(S.l[m], nb));
    }
  }
  x[k - 1] = cur;
  x[k - 1] = zmul(x[k - 1], S.uinv[k - 1]);
  if (k >= 2) x[k - 2] = zmul(zsub(x[k - 2], zmul(S.u1[k - 2], x[k - 1])), S.uinv[k - 2]);
  for (int m = k - 3; m >= 0; --m)
    x[m] = zmul(zsub(zsub(x[m], zmul(S.u1[m], x[m + 1])), zmul(S.u2[m], x[m + 2])), S.uinv[m]);
}

// z = H^{-dag} b: H = E^{-1} U with E the product of the elimination steps, so
// H^dag z = b  <=>  U^dag g = b, z = E_1^dag ... E_{k-1}^dag g.
__device__ void tri_solve_dag(const InnerSmem& S, int k, const double2* b, double2* z) {
  for (int m = 0; m < k; ++m) {
    double2 t = b[m];
    if (m >= 1) t = zsub(t, zmul(zconj(S.u1[m - 1]), z[m - 1]));
    if (m >= 2) t = zsub(t, zmul(zconj(S.u2[m - 2]), z[m - 2]));
    z[m] = zmul(t, zconj(S.uinv[m]));
  }
  for (int m = k - 2; m >= 0; --m) {
    const double2 cl = zconj(S.l[m]);
    const double2 gi = z[m], gn = z[m + 1];
    if (!S.sw[m]) {
      z[m] = zsub(gi, zmul(cl, gn));
    } else {
      z[m] = gn;
      z[m + 1] = zsub(gi, zmul(cl, gn));
    }
  }
}

// LU with partial pivoting of the tridiagonal H (thread 0). Returns false if singular.
__device__ bool tri_factor(const InnerSmem& S, int k) {
  double2 dd = S.d[0];
  double2 ee = k > 1 ? S.c[0] : make_double2(0.0, 0.0);
  for (int m = 0; m < k - 1; ++m) {
    const double2 an = S.a[m + 1], dn = S.d[m + 1];
    const double2 cn = (m + 1 <= k - 2) ? S.c[m + 1] : make_double2(0.0, 0.0);
    double2 r0, r1, r2, lm;
    if (zabs2(dd) >= zabs2(an)) {
      if (zabs2(dd) == 0.0) return false;
      lm = zdiv(an, dd);
      r0 = dd; r1 = ee; r2 = make_double2(0.0, 0.0);
      dd = zsub(dn, zmul(lm, ee));
      ee = cn;
      S.sw[m] = 0;
    } else {
      lm = zdiv(dd, an);
      r0 = an; r1 = dn; r2 = cn;
      dd = zsub(ee, zmul(lm, dn));
      ee = zscale(zmul(lm, cn), -1.0);
      S.sw[m] = 1;
    }
    S.uinv[m] = zinv(r0);
    S.u1[m] = r1;
    S.u2[m] = r2;
    S.l[m] = lm;
  }
  if (zabs2(dd) == 0.0) return false;
  S.uinv[k - 1] = zinv(dd);
  return true;
}

// y = H x (parallel)
__device__ __forceinline__ void tri_mul(const InnerSmem& S, int k, const double2* x, double2* y, bool dag) {
  for (int m = threadIdx.x; m < k; m += blockDim.x) {
    double2 t;
    if (!dag) {
      t = zmul(S.d[m], x[m]);
      if (m >= 1) t = zadd(t, zmul(S.a[m], x[m - 1]));
      if (m + 1 < k) t = zadd(t, zmul(S.c[m], x[m + 1]));
    } else {
      // (H^dag)_{m,m} = conj d_m, (H^dag)_{m,m-1} = conj H_{m-1,m} = conj c_{m-1},
      // (H^dag)_{m,m+1} = conj H_{m+1,m} = conj a_{m+1}
      t = zmul(zconj(S.d[m]), x[m]);
      if (m >= 1) t = zadd(t, zmul(zconj(S.c[m - 1]), x[m - 1]));
      if (m + 1 < k) t = zadd(t, zmul(zconj(S.a[m + 1]), x[m + 1]));
    }
    y[m] = t;
  }
}

__global__ void __launch_bounds__(kInnerThreads) k_inner(const int* __restrict__ k_dev, const int* __restrict__ l_dev,
                                                         int hermitian, const double2* __restrict__ alp,
                                                         const double2* __restrict__ bet,
                                                         const double2* __restrict__ gam, int ldc, InnerWork w) {
  int* fail = w.fail;
  extern __shared__ __align__(16) unsigned char smem[];
  const int prob = blockIdx.x;
  const int k = k_dev[prob];
  const int l = min(l_dev[prob], k);
  const int tid = threadIdx.x;
  InnerSmem S;
  {
    double2* base = (double2*)smem;
    S.d = base; S.a = base + k; S.c = base + 2 * k;
    S.uinv = base + 3 * k; S.u1 = base + 4 * k; S.u2 = base + 5 * k; S.l = base + 6 * k;
    S.q = base + 7 * k; S.qp = base + 8 * k; S.w = base + 9 * k; S.wp = base + 10 * k;
    S.u = base + 11 * k; S.z = base + 12 * k;
    S.red = (double*)(base + 13 * k);
    S.sw = (unsigned char*)(S.red + 32);
  }
  const size_t crow = (size_t)(prob % w.rows) * ldc;
  const double2* al = alp + crow;
  const double2* be = bet + crow;
  const double2* ga = gam + crow;
  for (int m = tid; m < k; m += blockDim.x) {
    double2 dm = al[m + 1];
    double2 am = m >= 1 ? be[m + 1] : make_double2(0.0, 0.0);
    double2 cm = m + 1 < k ? ga[m + 2] : make_double2(0.0, 0.0);
    if (hermitian) { dm.y = 0.0; am.y = 0.0; cm = m + 1 < k ? make_double2(be[m + 2].x, 0.0) : cm; }
    S.d[m] = dm; S.a[m] = am; S.c[m] = cm;
    const double2 zero = make_double2(0.0, 0.0);
    S.q[m] = m == 0 ? make_double2(1.0, 0.0) : zero;
    S.w[m] = S.q[m];
    S.qp[m] = zero; S.wp[m] = zero;
  }
  __syncthreads();
  __shared__ int s_ok;
  if (tid == 0) s_ok = tri_factor(S, k) ? 1 : 0;
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) { fail[prob] = 1; w.leff[prob] = 0; }
    return;
  }
  double2* Q = w.Q + (size_t)prob * w.ld * kMaxL;
  double2* T = w.T + (size_t)prob * kMaxL * 3;
  double2 b_i = make_double2(0.0, 0.0), g_i = make_double2(0.0, 0.0);  // inner beta_i, gamma_i
  int done = 0;
  const double exhaust_tol = 1e-13;
  for (int i = 0; i < l; ++i) {
    for (int m = tid; m < k; m += blockDim.x) Q[(size_t)m * kMaxL + i] = S.q[m];
    // u = M q = H q + H^{-1} q ; z = M^dag w (two-sided)
    if (tid == 0) tri_solve(S, k, S.q, S.u);
    if (!hermitian && tid == 32) tri_solve_dag(S, k, S.w, S.z);
    __syncthreads();
    double mq2 = 0.0;
    for (int m = tid; m < k; m += blockDim.x) {
      double2 t = zmul(S.d[m], S.q[m]);
      if (m >= 1) t = zadd(t, zmul(S.a[m], S.q[m - 1]));
      if (m + 1 < k) t = zadd(t, zmul(S.c[m], S.q[m + 1]));
      t = zadd(t, S.u[m]);
      mq2 += zabs2(t);
      S.u[m] = zsub(t, hermitian ? zscale(S.qp[m], b_i.x) : zmul(g_i, S.qp[m]));  // p
      if (!hermitian) {
        double2 y = zmul(zconj(S.d[m]), S.w[m]);
        if (m >= 1) y = zadd(y, zmul(zconj(S.c[m - 1]), S.w[m - 1]));
        if (m + 1 < k) y = zadd(y, zmul(zconj(S.a[m + 1]), S.w[m + 1]));
        y = zadd(y, S.z[m]);
        S.z[m] = zsub(y, zmul(zconj(b_i), S.wp[m]));  // r
      }
    }
    __syncthreads();
    // alpha = w^dag p (q^dag p in the Hermitian case)
    double are = 0.0, aim = 0.0;
    for (int m = tid; m < k; m += blockDim.x) {
      const double2 wm = hermitian ? S.q[m] : S.w[m];
      const double2 pm = S.u[m];
      are += wm.x * pm.x + wm.y * pm.y;
      aim += wm.x * pm.y - wm.y * pm.x;
    }
    are = block_sum(are, S.red);
    aim = hermitian ? 0.0 : block_sum(aim, S.red);
    const double mqn = sqrt(block_sum(mq2, S.red));
    const double2 a_i = make_double2(are, aim);
    if (tid == 0) T[i * 3 + 0] = a_i;
    done = i + 1;
    if (i == l - 1) break;
    // q~ = p - alpha q ; w~ = r - conj(alpha) w ; delta
    double dre = 0.0, dim = 0.0, n2 = 0.0;
    for (int m = tid; m < k; m += blockDim.x) {
      const double2 qt = zsub(S.u[m], zmul(a_i, S.q[m]));
      S.u[m] = qt;
      if (hermitian) {
        n2 += zabs2(qt);
      } else {
        const double2 wt = zsub(S.z[m], zmul(zconj(a_i), S.w[m]));
        S.z[m] = wt;
        dre += wt.x * qt.x + wt.y * qt.y;
        dim += wt.x * qt.y - wt.y * qt.x;
      }
    }
    double bn;
    double2 gn;
    if (hermitian) {
      bn = sqrt(block_sum(n2, S.red));
      gn = make_double2(bn, 0.0);
    } else {
      dre = block_sum(dre, S.red);
      dim = block_sum(dim, S.red);
      const double ad = sqrt(dre * dre + dim * dim);
      bn = sqrt(ad);
      gn = bn > 0.0 ? make_double2(dre / bn, dim / bn) : make_double2(0.0, 0.0);
    }
    if (!(bn > exhaust_tol * mqn)) break;  // inner space exhausted: T_i is exact
    if (tid == 0) {
      T[(i + 1) * 3 + 1] = make_double2(bn, 0.0);
      T[(i + 1) * 3 + 2] = gn;
    }
    const double2 wdiv = zinv(zconj(gn));
    __syncthreads();
    for (int m = tid; m < k; m += blockDim.x) {
      S.qp[m] = S.q[m];
      S.q[m] = zscale(S.u[m], 1.0 / bn);
      if (!hermitian) {
        S.wp[m] = S.w[m];
        S.w[m] = zmul(S.z[m], wdiv);
      }
    }
    b_i = make_double2(bn, 0.0);
    g_i = gn;
    __syncthreads();
  }
  if (tid == 0) {
    w.leff[prob] = done;
    T[0 * 3 + 1] = make_double2(0.0, 0.0);
    T[0 * 3 + 2] = make_double2(0.0, 0.0);
    fail[prob] = 0;
  }
}

// ------------------------------------------------------------ Roberts-Higham
// CTA `m2` handles matrix m2: problems [0, count) are T_{leff}, [count, 2 count) are
// T_{leff - dl} (the inner estimate); dense mode reads full matrices.
template <bool CPLX>
struct RhElem;
template <> struct RhElem<true> { using T = double2; };
template <> struct RhElem<false> { using T = double; };

__device__ __forceinline__ double2 rz(double2 a) { return a; }
__device__ __forceinline__ double el_abs2(double a) { return a * a; }
__device__ __forceinline__ double el_abs2(double2 a) { return zabs2(a); }
__device__ __forceinline__ double el_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double2 el_mul(double2 a, double2 b) { return zmul(a, b); }
__device__ __forceinline__ double el_sub(double a, double b) { return a - b; }
__device__ __forceinline__ double2 el_sub(double2 a, double2 b) { return zsub(a, b); }
__device__ __forceinline__ double el_inv(double a) { return 1.0 / a; }
__device__ __forceinline__ double2 el_inv(double2 a) { return zinv(a); }
__device__ __forceinline__ double el_avg(double a, double b) { return 0.5 * (a + b); }
__device__ __forceinline__ double2 el_avg(double2 a, double2 b) { return make_double2(0.5 * (a.x + b.x), 0.5 * (a.y + b.y)); }
__device__ __forceinline__ double el_from(double2 a) { return a.x; }
__device__ __forceinline__ double2 el_from2(double2 a) { return a; }
__device__ __forceinline__ double2 el_to2(double a) { return make_double2(a, 0.0); }
__device__ __forceinline__ double2 el_to2(double2 a) { return a; }
__device__ __forceinline__ double el_zero(double) { return 0.0; }
__device__ __forceinline__ double2 el_zero(double2) { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double el_one(double) { return 1.0; }
__device__ __forceinline__ double2 el_one(double2) { return make_double2(1.0, 0.0); }
__device__ __forceinline__ bool el_finite(double a) { return isfinite(a); }
__device__ __forceinline__ bool el_finite(double2 a) { return isfinite(a.x) && isfinite(a.y); }

template <class E>
__device__ __forceinline__ E el_load(const double2* p) {
  if constexpr (sizeof(E) == sizeof(double)) return p->x; else return *(const E*)p;
}

template <bool CPLX>
__global__ void __launch_bounds__(1024) k_rh(int count, int dense_m, const double2* __restrict__ dense_T,
                                             InnerWork w, int dl, double rh_tol, int rh_maxit, int mid0) {
  using E = typename RhElem<CPLX>::T;
  extern __shared__ __align__(16) unsigned char smem[];
  const int mid = mid0 + blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x;
  int m;
  if (dense_m > 0) {
    m = dense_m;
  } else {
    const int prob = mid % count;
    const int le = w.leff[prob];
    m = mid < count ? le : le - dl;
  }
  if (m <= 0) {
    if (tid == 0) { w.rh_ok[mid] = m == 0 ? 0 : 1; w.rh_its[mid] = 0; }
    return;
  }
  E* W = (E*)smem;                    // m x m working matrix
  E* col = W + (size_t)m * m;         // column buffer / reduction scratch
  double* red = (double*)col;
  int* piv_slot = (int*)col;
  double2* Sg = w.S + (size_t)mid * kMaxL * kMaxL;  // global S_n (row-major, leading dim m)
  int* perm = w.perm + (size_t)mid * kMaxL;
  // S_0 = T
  for (int e = tid; e < m * m; e += nth) {
    const int i = e / m, j = e % m;
    double2 v = make_double2(0.0, 0.0);
    if (dense_m > 0) {
      v = dense_T[(size_t)mid * m * m + e];
    } else {
      const double2* T = w.T + (size_t)(mid % count) * kMaxL * 3;
      if (i == j) v = T[i * 3 + 0];
      else if (i == j + 1) v = T[i * 3 + 1];      // subdiagonal beta_{i}
      else if (j == i + 1) v = T[j * 3 + 2];      // superdiagonal gamma_{j}
    }
    if (!CPLX) v.y = 0.0;
    Sg[e] = v;
  }
  __syncthreads();
  int ok = 0, it = 0;
  for (it = 1; it <= rh_maxit; ++it) {
    for (int e = tid; e < m * m; e += nth) W[e] = el_load<E>(&Sg[e]);
    __syncthreads();
    bool singular = false;
    for (int j = 0; j < m; ++j) {
      // pivot search in column j (warp 0; ties keep the smaller row)
      if (tid < 32) {
        double best = -1.0;
        int bi = j;
        for (int i = j + tid; i < m; i += 32) {
          const double a2 = el_abs2(W[(size_t)i * m + j]);
          if (a2 > best) { best = a2; bi = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double ob = __shfl_xor_sync(0xffffffffu, best, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (tid == 0) piv_slot[0] = best > 0.0 ? bi : -1;
      }
      __syncthreads();
      const int p = piv_slot[0];
      __syncthreads();
      if (p < 0) { singular = true; break; }
      if (p != j)
        for (int c = tid; c < m; c += nth) {
          const E t = W[(size_t)j * m + c];
          W[(size_t)j * m + c] = W[(size_t)p * m + c];
          W[(size_t)p * m + c] = t;
        }
      if (tid == 0) perm[j] = p;
      __syncthreads();
      const E inv = el_inv(W[(size_t)j * m + j]);
      __syncthreads();
      for (int c = tid; c < m; c += nth) W[(size_t)j * m + c] = c == j ? inv : el_mul(W[(size_t)j * m + c], inv);
      for (int i = tid; i < m; i += nth) col[i] = i == j ? el_zero(inv) : W[(size_t)i * m + j];
      __syncthreads();
      for (int i = tid; i < m; i += nth)
        if (i != j) W[(size_t)i * m + j] = el_zero(inv);
      __syncthreads();
      {
        // 32 x 32 thread tile: thread (ty, tx) updates rows ty + 32a and columns tx + 32b,
        // holding its entries of the pivot row in registers (m <= 120 < 4 * 32)
        const int tx = tid & 31, ty = tid >> 5;
        E rowj[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = tx + 32 * b;
          rowj[b] = c < m ? W[(size_t)j * m + c] : el_zero(inv);
        }
        for (int i = ty; i < m; i += 32) {
          if (i == j) continue;
          const E f = col[i];
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int c = tx + 32 * b;
            if (c < m) W[(size_t)i * m + c] = el_sub(W[(size_t)i * m + c], el_mul(f, rowj[b]));
          }
        }
      }
      __syncthreads();
    }
    if (singular) { ok = 0; break; }
    // undo the row interchanges as column interchanges, last first
    for (int j = m - 1; j >= 0; --j) {
      const int p = perm[j];
      if (p != j)
        for (int i = tid; i < m; i += nth) {
          const E t = W[(size_t)i * m + j];
          W[(size_t)i * m + j] = W[(size_t)i * m + p];
          W[(size_t)i * m + p] = t;
        }
      __syncthreads();
    }
    // S_{n+1} = (S_n + S_n^{-1}) / 2 ; convergence test in the Frobenius norm
    double dif = 0.0, nrm = 0.0;
    bool fin = true;
    for (int e = tid; e < m * m; e += nth) {
      const E sn = el_load<E>(&Sg[e]);
      const E s1 = el_avg(sn, W[e]);
      fin = fin && el_finite(s1);
      dif += el_abs2(el_sub(s1, sn));
      nrm += el_abs2(s1);
      Sg[e] = el_to2(s1);
    }
    __syncthreads();
    dif = warp_sum(dif);
    nrm = warp_sum(nrm);
    const int fin_all = __syncthreads_and(fin ? 1 : 0);
    if ((tid & 31) == 0) { red[(tid >> 5) * 2] = dif; red[(tid >> 5) * 2 + 1] = nrm; }
    __syncthreads();
    double D = 0.0, N = 0.0;
    for (int q = 0; q < (nth >> 5); ++q) { D += red[2 * q]; N += red[2 * q + 1]; }
    __syncthreads();
    if (!fin_all || !isfinite(D) || !isfinite(N)) { ok = 0; break; }
    if (sqrt(D) <= rh_tol * sqrt(N)) { ok = 1; break; }
  }
  if (tid == 0) {
    w.rh_ok[mid] = ok;
    w.rh_its[mid] = it > rh_maxit ? rh_maxit : it;
  }
  for (int i = tid; i < m; i += nth) w.s[(size_t)mid * kMaxL + i] = Sg[(size_t)i * m];
}

// ------------------------------------------------- Roberts-Higham in double-float
// The same iteration and Gauss-Jordan elimination as k_rh, with the matrix held as float
// pairs (hi + lo, ~48-bit significand) and all arithmetic on the float pipes: on GB300 a
// warp-wide FP64 instruction issues at ~1/64 of the float rate, and the elimination is
// pure multiply-add. Products are formed exactly (p = a*b, e = fma(a, b, -p), cross terms
// folded into e) and each output is renormalised once; the pivot reciprocal takes one
// Newton step r = x + x (1 - d x) from the float reciprocal x, which doubles its 24
// correct bits. Pivots are chosen on the high words.
struct cdf {
  df64 re, im;
};

__device__ __forceinline__ cdf operator-(cdf a) { return {-a.re, -a.im}; }
__device__ __forceinline__ cdf operator-(cdf a, cdf b) { return {a.re - b.re, a.im - b.im}; }

__device__ __forceinline__ df64 df_recip(df64 d) {
  const float x = __frcp_rn(d.hi);
  const df64 e = df64{1.f, 0.f} - d * x;
  return df64{x, 0.f} + e * x;
}

__device__ __forceinline__ cdf e_load(const float4* p) {
  const float4 v = *p;
  return {{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ df64 e_load(const float2* p) {
  const float2 v = *p;
  return {v.x, v.y};
}
__device__ __forceinline__ void e_store(float4* p, cdf a) { *p = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }
__device__ __forceinline__ void e_store(float2* p, df64 a) { *p = make_float2(a.hi, a.lo); }
__device__ __forceinline__ float e_abs2hi(cdf a) { return a.re.hi * a.re.hi + a.im.hi * a.im.hi; }
__device__ __forceinline__ float e_abs2hi(df64 a) { return a.hi * a.hi; }
__device__ __forceinline__ cdf e_zero(cdf) { return {df_zero(), df_zero()}; }
__device__ __forceinline__ df64 e_zero(df64) { return df_zero(); }
// w - f r
__device__ __forceinline__ cdf e_submul(cdf w, cdf f, cdf r) {
  return {df_axpy2(w.re, -f.re, r.re, f.im, r.im), df_axpy2(w.im, -f.re, r.im, -f.im, r.re)};
}
__device__ __forceinline__ df64 e_submul(df64 w, df64 f, df64 r) { return df_axpy1(w, -f, r); }
__device__ __forceinline__ cdf e_mul(cdf a, cdf b) {
  return {df_axpy2(df_zero(), a.re, b.re, -a.im, b.im), df_axpy2(df_zero(), a.re, b.im, a.im, b.re)};
}
__device__ __forceinline__ df64 e_mul(df64 a, df64 b) { return a * b; }
__device__ __forceinline__ cdf e_inv(cdf a) {
  const df64 r = df_recip(df_axpy2(df_zero(), a.re, a.re, a.im, a.im));
  return {a.re * r, -(a.im * r)};
}
__device__ __forceinline__ df64 e_inv(df64 a) { return df_recip(a); }
// (a + b) / 2 and |(a + b) / 2 - a|^2, |(a + b) / 2|^2 (high words)
__device__ __forceinline__ cdf e_avg(cdf a, cdf b, float& d2, float& n2) {
  const cdf s = {df_half(a.re + b.re), df_half(a.im + b.im)};
  const float dr = __fsub_rn(s.re.hi, a.re.hi), di = __fsub_rn(s.im.hi, a.im.hi);
  d2 += dr * dr + di * di;
  n2 += e_abs2hi(s);
  return s;
}
__device__ __forceinline__ df64 e_avg(df64 a, df64 b, float& d2, float& n2) {
  const df64 s = df_half(a + b);
  const float d = __fsub_rn(s.hi, a.hi);
  d2 += d * d;
  n2 += s.hi * s.hi;
  return s;
}
__device__ __forceinline__ cdf e_scale(cdf a, float f) { return {a.re * f, a.im * f}; }
__device__ __forceinline__ df64 e_scale(df64 a, float f) { return a * f; }
// (g a + b / g) / 2 with |(...) - a|^2 and |(...)|^2 (high words), g > 0
__device__ __forceinline__ cdf e_avg_scaled(cdf a, cdf b, float g, float gi, float& d2, float& n2) {
  const cdf sa = e_scale(a, g), sb = e_scale(b, gi);
  const cdf s = {df_half(sa.re + sb.re), df_half(sa.im + sb.im)};
  const float dr = __fsub_rn(s.re.hi, a.re.hi), di = __fsub_rn(s.im.hi, a.im.hi);
  d2 += dr * dr + di * di;
  n2 += e_abs2hi(s);
  return s;
}
__device__ __forceinline__ df64 e_avg_scaled(df64 a, df64 b, float g, float gi, float& d2, float& n2) {
  const df64 s = df_half(e_scale(a, g) + e_scale(b, gi));
  const float d = __fsub_rn(s.hi, a.hi);
  d2 += d * d;
  n2 += s.hi * s.hi;
  return s;
}
__device__ __forceinline__ bool e_finite(cdf a) {
  return isfinite(a.re.hi) && isfinite(a.re.lo) && isfinite(a.im.hi) && isfinite(a.im.lo);
}
__device__ __forceinline__ bool e_finite(df64 a) { return isfinite(a.hi) && isfinite(a.lo); }
__device__ __forceinline__ double2 e_to2(cdf a) { return make_double2(df_to_double(a.re), df_to_double(a.im)); }
__device__ __forceinline__ double2 e_to2(df64 a) { return make_double2(df_to_double(a), 0.0); }
__device__ __forceinline__ cdf e_from2(double2 v, cdf) { return {df_from_double(v.x), df_from_double(v.y)}; }
__device__ __forceinline__ df64 e_from2(double2 v, df64) { return df_from_double(v.x); }

constexpr int kRhLeft = -1;  // rh_ok of a matrix that k_rh_col leaves to k_rh_df

template <bool CPLX>
struct RhDf;
template <> struct RhDf<true> { using E = cdf; using St = float4; };
template <> struct RhDf<false> { using E = df64; using St = float2; };

template <bool CPLX>
__global__ void __launch_bounds__(1024) k_rh_df(int count, int dense_m, const double2* __restrict__ dense_T,
                                                InnerWork w, int dl, double rh_tol, int rh_maxit, int mid0,
                                                int scale) {
  // nested checks: only the matrices that k_rh_col left to this kernel
  if (dense_m == 0 && w.rh_ok[mid0 + blockIdx.x] != kRhLeft) return;
  using E = typename RhDf<CPLX>::E;
  using St = typename RhDf<CPLX>::St;
  extern __shared__ __align__(16) unsigned char smem[];
  const int mid = mid0 + blockIdx.x;
  const int tid = threadIdx.x, nth = blockDim.x;
  int m;
  if (dense_m > 0) {
    m = dense_m;
  } else {
    const int prob = mid % count;
    const int le = w.leff[prob];
    m = mid < count ? le : le - dl;
  }
  if (m <= 0) {
    if (tid == 0) { w.rh_ok[mid] = m == 0 ? 0 : 1; w.rh_its[mid] = 0; }
    return;
  }
  St* W = (St*)smem;                  // m x m working matrix
  St* col = W + (size_t)m * m;        // column buffer / reduction scratch
  double* red = (double*)col;
  __shared__ int s_piv;
  __shared__ St s_inv, s_djj;
  __shared__ float s_logdet;  // log |det S_n| from the pivots (high words)
  // global S_n (row-major, leading dim m) in the float-pair storage, in the problem's
  // double2 slot (16 bytes per element)
  St* Sg = (St*)(w.S + (size_t)blockIdx.x * kMaxL * kMaxL);
  int* perm = w.perm + (size_t)mid * kMaxL;
  const E ez = e_zero(E{});
  for (int e = tid; e < m * m; e += nth) {
    const int i = e / m, j = e % m;
    double2 v = make_double2(0.0, 0.0);
    if (dense_m > 0) {
      v = dense_T[(size_t)mid * m * m + e];
    } else {
      const double2* T = w.T + (size_t)(mid % count) * kMaxL * 3;
      if (i == j) v = T[i * 3 + 0];
      else if (i == j + 1) v = T[i * 3 + 1];
      else if (j == i + 1) v = T[j * 3 + 2];
    }
    e_store(&Sg[e], e_from2(v, ez));
  }
  __syncthreads();
  int ok = 0, it = 0;
  float rel_prev = INFINITY;  // ||S_n - S_{n-1}|| / ||S_n|| of the last iteration
  // the elimination's element share of thread tid >= 32 (warps 1..): the elements
  // u, u + nth - 32, ... of the (m - 1) x (m - 1) block, row-major (u = tid - 32)
  const int mm = m - 1;
  const int fu = tid - 32, fst = nth - 32;
  const int fr0 = (mm > 0 && fu >= 0) ? fu / mm : 0, fc0 = (mm > 0 && fu >= 0) ? fu % mm : 0;
  const int fdr = mm > 0 ? fst / mm : 0, fdc = mm > 0 ? fst % mm : 0;
  for (it = 1; it <= rh_maxit; ++it) {
    for (int e = tid; e < m * m; e += nth) W[e] = Sg[e];
    __syncthreads();
    bool singular = false;
    // Gauss-Jordan with partial pivoting, two barriers a column: (A) the pivot row is
    // swapped into row j and scaled, the multipliers of column j saved; (B) every other row
    // is eliminated, while warp 0 eliminates column j + 1 and chooses its pivot (its row
    // p, 1 / W[p][j+1] and the old diagonal W[j+1][j+1] go through s_piv, s_inv, s_djj).
    auto pivot_of = [&](int jc, int lane, float best, int bi) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      __syncwarp();
      if (lane == 0) {
        s_piv = best > 0.f ? bi : -1;
        if (best > 0.f) {
          s_inv = W[(size_t)bi * m + jc];
          s_djj = W[(size_t)jc * m + jc];
          s_logdet = (jc == 0 ? 0.f : s_logdet) + 0.5f * __logf(best);
        }
      }
    };
    if (tid < 32) {
      float best = -1.f;
      int bi = 0;
      for (int i = tid; i < m; i += 32) {
        const float a2 = e_abs2hi(e_load(&W[(size_t)i * m]));
        if (a2 > best) { best = a2; bi = i; }
      }
      pivot_of(0, tid, best, bi);
    }
    __syncthreads();
    for (int j = 0; j < m; ++j) {
      const int p = s_piv;
      if (p < 0) { singular = true; break; }
      const E inv = e_inv(e_load(&s_inv));
      const St djj = s_djj;
      if (tid == 0) perm[j] = p;
      // (A) rows j and p are touched column by column by one thread each; the multipliers
      // read column j of the other rows (row p's multiplier is the old W[j][j])
      for (int c = tid; c < m; c += nth) {
        const E wp = e_load(&W[(size_t)p * m + c]);
        const St wj = W[(size_t)j * m + c];
        e_store(&W[(size_t)j * m + c], c == j ? inv : e_mul(wp, inv));
        if (p != j) W[(size_t)p * m + c] = wj;
      }
      for (int i = tid; i < m; i += nth) col[i] = i == j ? St{} : (i == p ? djj : W[(size_t)i * m + j]);
      __syncthreads();
      // (B) W[i][c] -= col[i] W[j][c] for i != j; column j becomes -col[i] / pivot (the
      // inverse's column, in place). Warp 0 takes column cw = j + 1 (j itself at the last
      // column) and, for j + 1 < m, picks that column's pivot; warps 1.. share the other
      // (m - 1) x (m - 1) elements evenly (rows without j, columns without cw).
      {
        const int tx = tid & 31;
        const int cw = j + 1 < m ? j + 1 : j;
        if (tid >= 32) {
          if (mm > 0) {
            int ri = fr0, ci = fc0;
            while (ri < mm) {
              const int i = ri + (ri >= j);
              const int c = ci + (ci >= cw);
              const E f = e_load(&col[i]);
              const E pj = e_load(&W[(size_t)j * m + c]);
              e_store(&W[(size_t)i * m + c], e_submul(c == j ? ez : e_load(&W[(size_t)i * m + c]), f, pj));
              ri += fdr;
              ci += fdc;
              if (ci >= mm) {
                ci -= mm;
                ++ri;
              }
            }
          }
        } else {
          const E pj1 = e_load(&W[(size_t)j * m + cw]);
          float best = -1.f;
          int bi = j + 1;
          for (int i = tx; i < m; i += 32) {
            if (i == j) continue;
            const E v = e_submul(cw == j ? ez : e_load(&W[(size_t)i * m + cw]), e_load(&col[i]), pj1);
            e_store(&W[(size_t)i * m + cw], v);
            if (cw == j + 1 && i > j) {
              const float a2 = e_abs2hi(v);
              if (a2 > best) { best = a2; bi = i; }
            }
          }
          if (cw == j + 1) pivot_of(j + 1, tx, best, bi);
        }
      }
      __syncthreads();
    }
    if (singular) { ok = 0; break; }
    // the row interchanges permute the inverse's columns: undo them all in one gather,
    // idx[c] = the column that ends at c (the interchanges applied in reverse order)
    int* idx = (int*)col;
    if (tid == 0) {
      for (int c = 0; c < m; ++c) idx[c] = c;
      for (int j = m - 1; j >= 0; --j) {
        const int pj = perm[j];
        const int t = idx[j];
        idx[j] = idx[pj];
        idx[pj] = t;
      }
    }
    __syncthreads();
    {
      const int tx = tid & 31, ty = tid >> 5;
      for (int i = ty; i < m; i += 32) {
        St v[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = tx + 32 * b;
          if (c < m) v[b] = W[(size_t)i * m + idx[c]];
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int c = tx + 32 * b;
          if (c < m) W[(size_t)i * m + c] = v[b];
        }
        __syncwarp();
      }
    }
    __syncthreads();
    float d2 = 0.f, n2 = 0.f;
    bool fin = true;
    // determinant scaling (Byers; Kenney and Laub, SIAM J. Matrix Anal. Appl. 13 (1992)):
    // S_{n+1} = (g S_n + S_n^{-1} / g) / 2 with g = |det S_n|^{-1/m} while the iterate still
    // changes by more than 1e-2, the plain step of Eq. (Roberts) after that (its quadratic
    // convergence is untouched). The limit is sgn(S_0) either way.
    const float g = (scale && rel_prev > 1e-2f) ? __expf(-s_logdet / (float)m) : 1.f;
    const float gi = 1.f / g;
    for (int e = tid; e < m * m; e += nth) {
      const E a = e_load(&Sg[e]);
      const E s1 = g == 1.f ? e_avg(a, e_load(&W[e]), d2, n2) : e_avg_scaled(a, e_load(&W[e]), g, gi, d2, n2);
      fin = fin && e_finite(s1);
      e_store(&Sg[e], s1);
    }
    __syncthreads();
    double dif = warp_sum((double)d2);
    double nrm = warp_sum((double)n2);
    const int fin_all = __syncthreads_and(fin ? 1 : 0);
    if ((tid & 31) == 0) { red[(tid >> 5) * 2] = dif; red[(tid >> 5) * 2 + 1] = nrm; }
    __syncthreads();
    double D = 0.0, N = 0.0;
    for (int q = 0; q < (nth >> 5); ++q) { D += red[2 * q]; N += red[2 * q + 1]; }
    __syncthreads();
    if (!fin_all || !isfinite(D) || !isfinite(N)) { ok = 0; break; }
    if (sqrt(D) <= rh_tol * sqrt(N)) { ok = 1; break; }
    rel_prev = (float)(sqrt(D) / sqrt(N));
  }
  if (tid == 0) {
    w.rh_ok[mid] = ok;
    w.rh_its[mid] = it > rh_maxit ? rh_maxit : it;
  }
  for (int i = tid; i < m; i += nth) w.s[(size_t)mid * kMaxL + i] = e_to2(e_load(&Sg[(size_t)i * m]));
  if (CPLX && dense_m > 0) {
    // the caller reads S as double2: convert in place (same 16-byte slot per element)
    __syncthreads();
    double2* Sd = w.S + (size_t)blockIdx.x * kMaxL * kMaxL;
    for (int e = tid; e < m * m; e += nth) {
      const E v = e_load(&Sg[e]);
      Sd[e] = e_to2(v);
    }
  }
}

// ------------------------------------------------- inner Krylov in double-float
// k_inner with every operation on the float pipes: the tridiagonal factorisation (serial), the
// solves and the vector updates in float pairs, the block reductions in float pairs. Square
// roots take one Newton step y + (x - y^2) / (2 y) from the float root, quotients multiply by
// the refined reciprocal (Karp and Markstein, ACM TOMS 23 (1997)). T is written in double, Q in
// float pairs. At mu = 0 H_k is real symmetric and everything is real (E = df64: a quarter of
// the arithmetic); E = cdf otherwise.
__device__ __forceinline__ cdf c_zero() { return {df_zero(), df_zero()}; }
__device__ __forceinline__ cdf c_one() { return {{1.f, 0.f}, df_zero()}; }
__device__ __forceinline__ cdf c_add(cdf a, cdf b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cdf c_scale(cdf a, df64 s) { return {a.re * s, a.im * s}; }
__device__ __forceinline__ cdf e_one(cdf) { return c_one(); }
__device__ __forceinline__ df64 e_one(df64) { return {1.f, 0.f}; }
__device__ __forceinline__ cdf e_conj(cdf a) { return {a.re, -a.im}; }
__device__ __forceinline__ df64 e_conj(df64 a) { return a; }
__device__ __forceinline__ cdf e_real(df64 r, cdf) { return {r, df_zero()}; }
__device__ __forceinline__ df64 e_real(df64 r, df64) { return r; }
// a + f r
__device__ __forceinline__ cdf e_addmul(cdf a, cdf f, cdf r) {
  return {df_axpy2(a.re, f.re, r.re, -f.im, r.im), df_axpy2(a.im, f.re, r.im, f.im, r.re)};
}
__device__ __forceinline__ df64 e_addmul(df64 a, df64 f, df64 r) { return df_axpy1(a, f, r); }
// a - conj(f) r
__device__ __forceinline__ cdf e_submulc(cdf a, cdf f, cdf r) {
  return {df_axpy2(a.re, -f.re, r.re, -f.im, r.im), df_axpy2(a.im, -f.re, r.im, f.im, r.re)};
}
__device__ __forceinline__ df64 e_submulc(df64 a, df64 f, df64 r) { return df_axpy1(a, -f, r); }
// d += conj(a) b
__device__ __forceinline__ void e_dot(df64 (&d)[2], cdf a, cdf b) {
  d[0] = df_axpy2(d[0], a.re, b.re, a.im, b.im);
  d[1] = df_axpy2(d[1], a.re, b.im, -a.im, b.re);
}
__device__ __forceinline__ void e_dot(df64 (&d)[2], df64 a, df64 b) { d[0] = df_axpy1(d[0], a, b); }
__device__ __forceinline__ float4 e_pairs(cdf a) { return make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }
__device__ __forceinline__ float4 e_pairs(df64 a) { return make_float4(a.hi, a.lo, 0.f, 0.f); }
__device__ __forceinline__ df64 df_sqrt(df64 x) {
  if (!(x.hi > 0.f)) return df_zero();
  const float y = __fsqrt_rn(x.hi);
  const df64 e = x - df_prod(y, y);
  return df_two_sum(y, __fmul_rn(e.hi, __fdiv_rn(0.5f, y)));
}

template <class St>
struct InnerSmemDf {
  St *d, *a, *c, *uinv, *u1, *u2, *l, *q, *qp, *w, *wp, *u, *z;
  unsigned char* sw;
  df64* red;
};

// LU with partial pivoting of the tridiagonal H, U = D (1 + N) (one thread; ia[m] = 1 / H_{m,m-1}
// beforehand, so that only a row kept in place waits for a reciprocal). False if singular.
template <class E, class St>
__device__ bool tri_factor_df(const InnerSmemDf<St>& S, int k, const St* ia) {
  const E zero = e_zero(E{});
  E dd = e_load(&S.d[0]);
  E ee = k > 1 ? e_load(&S.c[0]) : zero;
  E an = zero, dn = zero, cn = zero, in = zero;
  if (k > 1) { an = e_load(&S.a[1]); dn = e_load(&S.d[1]); cn = e_load(&S.c[1]); in = e_load(&ia[1]); }
#pragma unroll 1
  for (int m = 0; m < k - 1; ++m) {
    const E a = an, d = dn, c = cn, ai = in;  // c[k - 1] = 0
    if (m + 2 < k) {
      an = e_load(&S.a[m + 2]);
      dn = e_load(&S.d[m + 2]);
      cn = e_load(&S.c[m + 2]);
      in = e_load(&ia[m + 2]);
    }
    const float pd = e_abs2hi(dd), pa = e_abs2hi(a);
    if (pd >= pa) {
      if (pd == 0.f) return false;
      const E ri = e_inv(dd), lm = e_mul(a, ri);
      e_store(&S.uinv[m], ri);
      e_store(&S.u1[m], e_mul(ee, ri));
      e_store(&S.u2[m], zero);
      e_store(&S.l[m], lm);
      S.sw[m] = 0;
      dd = e_submul(d, lm, ee);
      ee = c;
    } else {
      const E lm = e_mul(dd, ai);
      e_store(&S.uinv[m], ai);
      e_store(&S.u1[m], e_mul(d, ai));
      e_store(&S.u2[m], e_mul(c, ai));
      e_store(&S.l[m], lm);
      S.sw[m] = 1;
      dd = e_submul(ee, lm, d);
      ee = e_submul(zero, lm, c);
    }
  }
  if (e_abs2hi(dd) == 0.f) return false;
  e_store(&S.uinv[k - 1], e_inv(dd));
  e_store(&S.u1[k - 1], zero);
  e_store(&S.u2[k - 1], zero);
  S.sw[k - 1] = 0;
  return true;
}

// ---- the tridiagonal solves of one inner step, in parallel ----------------------------
// With the pivoted factors, H^{-1} b is two linear recurrences over the rows (the row
// interchanges with L downwards, then 1 + N back up) and H^{-dag} b two more. A serial sweep
// costs k times the latency of one complex multiply-add (~70 cycles), and two threads of a
// 256-thread CTA ran them: 73 us an inner step at k = 333, nearly all of the inner level. Here
// each side of the inner step has 128 lanes; a lane owns about B = ceil(k / 128) rows, runs
// them from a zero state, the states that enter the chunks are found by a scan over the lanes,
// and the rows run again from them. The scan composes x -> P x + C with numbers P that depend
// on H only, so every product of P is formed once per check (scan_setup) and a scan level is
// one shuffle and one multiply-add.
//  - U has two superdiagonals, the second one only in rows that were exchanged, so two numbers
//    enter a chunk of 1 + N and P is a 2 x 2 matrix (CPLX). For the real symmetric H_k of mu = 0,
//    whose eigenvalues lie on both sides of zero, exchanged rows do not follow one another (no
//    two in a row in the Ritz matrices of this method): there the chunks end at rows that were
//    not exchanged, at the nominal end or the nearest such row before it, and one number enters.
//    (In the two-sided process three rows of four are exchanged, runs reach 65 rows and that
//    form was six times slower.)
//  - P of the recurrences with L is a product of multipliers |l| <= 1; the elements of P of the
//    others are elements of U_{II}^{-1} U_{IJ} for consecutive rows I, and the inverse of a
//    diagonal block of a triangular matrix is that block of its inverse, so |P| <= ||U^{-1}||
//    ||U||: the growth that the factors allow anyway (measured against the oracle at k = 31 ..
//    1000: the errors of the serial sweeps).
// 3 + 5 + 3 dependent multiply-adds replace 333 at k = 333; 12 problems, l = 120: 8.72 -> 1.44 ms
// (two-sided); at mu = 0, in real arithmetic, the whole inner level 11.0 -> 1.31 ms (1.87 in
// complex arithmetic). With the chains gone the two-sided step is spent on the instructions and
// latency of its SM (issue 49%, float pipe 38%, ~6000 instructions a warp and step). 32 or 64 lanes a side do
// less work in the scans but run longer chunks: slower from k = 333 on.
constexpr int kSideLanes = 128;  // lanes of one side (v: threads 0.., w: the rest)
constexpr int kSideWarps = kSideLanes / 32;

// the value of lane `src` (the loops below are kept rolled and shared by the two sides: the
// step's straight-line code would not stay in the instruction cache)
__device__ __forceinline__ df64 shfl_lane(df64 v, int src) {
  return {__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}
__device__ __forceinline__ cdf shfl_lane(cdf v, int src) { return {shfl_lane(v.re, src), shfl_lane(v.im, src)}; }
struct cdf2 {  // the state of a second-order recurrence: the two newest values
  cdf x, y;
};
struct cmat2 {
  cdf a, b, c, d;
};
__device__ __forceinline__ cdf2 shfl_lane(cdf2 v, int src) { return {shfl_lane(v.x, src), shfl_lane(v.y, src)}; }
__device__ __forceinline__ cmat2 shfl_lane(cmat2 v, int src) {
  return {shfl_lane(v.a, src), shfl_lane(v.b, src), shfl_lane(v.c, src), shfl_lane(v.d, src)};
}
// the map m applied to a state, plus add; the map f after g; the identity
template <class E>
__device__ __forceinline__ E lin(E m, E s, E add) { return e_addmul(add, m, s); }
__device__ __forceinline__ cdf2 lin(cmat2 m, cdf2 s, cdf2 add) {
  return {e_addmul(e_addmul(add.x, m.a, s.x), m.b, s.y), e_addmul(e_addmul(add.y, m.c, s.x), m.d, s.y)};
}
template <class E>
__device__ __forceinline__ E compose(E f, E g) { return e_mul(f, g); }
__device__ __forceinline__ cmat2 compose(cmat2 f, cmat2 g) {
  return {e_addmul(e_mul(f.a, g.a), f.b, g.c), e_addmul(e_mul(f.a, g.b), f.b, g.d),
          e_addmul(e_mul(f.c, g.a), f.d, g.c), e_addmul(e_mul(f.c, g.b), f.d, g.d)};
}
__device__ __forceinline__ cmat2 e_one(cmat2) { return {c_one(), c_zero(), c_zero(), c_one()}; }
__device__ __forceinline__ cdf2 e_zero(cdf2) { return {c_zero(), c_zero()}; }
// barrier over one side's warps
__device__ __forceinline__ void side_sync(int side) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + side), "n"(kSideLanes) : "memory");
}

// the products of chunk maps that one recurrence's scan applies: of the 2^lev lanes ending at
// this one (lev), of all earlier lanes of the warp (excl), and of each whole warp (total)
template <class M>
struct ScanMaps {
  M lev[5], excl;
};
template <class M, class St>
struct ScanShared {
  M total[kSideWarps];
  St carry[kSideWarps];
};
// place of this lane and warp along the recurrence; up: the rows ascend with the lanes
struct ScanPos {
  int lane, li, wi, dir;
};
__device__ __forceinline__ ScanPos scan_pos(bool up) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x % kSideLanes) >> 5;
  return {lane, up ? lane : 31 - lane, up ? w : kSideWarps - 1 - w, up ? -1 : 1};
}
template <class M, class St>
__device__ __forceinline__ void scan_setup(ScanMaps<M>& f, ScanShared<M, St>& sh, M p, ScanPos ps) {
#pragma unroll 1
  for (int lev = 0; lev < 5; ++lev) {
    f.lev[lev] = p;
    const M q = shfl_lane(p, (ps.lane + (ps.dir << lev)) & 31);
    if (ps.li >= (1 << lev)) p = compose(p, q);
  }
  f.excl = shfl_lane(p, (ps.lane + ps.dir) & 31);
  if (ps.li == 0) f.excl = e_one(M{});
  if (ps.li == 31) sh.total[ps.wi] = p;
}
// the state that enters this lane's chunk, from the states c that the chunks leave when they
// are run from zero (one barrier of the side's warps)
template <class M, class St>
__device__ __forceinline__ St scan_in(const ScanMaps<M>& f, ScanShared<M, St>& sh, St c, ScanPos ps, int side) {
#pragma unroll 1
  for (int lev = 0; lev < 5; ++lev) {
    const M m = f.lev[lev];
    const St q = shfl_lane(c, (ps.lane + (ps.dir << lev)) & 31);
    if (ps.li >= (1 << lev)) c = lin(m, q, c);
  }
  if (ps.li == 31) sh.carry[ps.wi] = c;
  St in = shfl_lane(c, (ps.lane + ps.dir) & 31);
  if (ps.li == 0) in = e_zero(St{});
  side_sync(side);
  if (ps.wi == 0) return in;
  St s = sh.carry[0];
#pragma unroll 1
  for (int w = 1; w <= ps.wi; ++w) {
    const bool last = w == ps.wi;
    s = lin(last ? f.excl : sh.total[w], s, last ? in : sh.carry[w]);
  }
  return s;
}

// One lane's rows [s, e) of the four recurrences; each returns the state it leaves and, with
// `store`, writes its values. rhs = false: without a right-hand side (for the chunk's map).
// row interchanges and L, down the rows, state: the pending row; x[m] / diag(U) is stored
template <class E, class St>
__device__ __forceinline__ E chunk_l(const InnerSmemDf<St>& S, int k, int s, int e, const St* b, St* x, E cur, bool store) {
#pragma unroll 1
  for (int m = s; m < e; ++m) {
    E bsel = cur;
    if (m < k - 1) {
      const E nb = e_load(&b[m + 1]);
      const bool sw = S.sw[m];
      const E asel = sw ? cur : nb;
      bsel = sw ? nb : cur;
      cur = e_submul(asel, e_load(&S.l[m]), bsel);
    }
    if (store) e_store(&x[m], e_mul(bsel, e_load(&S.uinv[m])));
  }
  return cur;
}
// 1 + N, up the rows, in place, state: x[m + 1], x[m + 2]
__device__ __forceinline__ cdf2 chunk_u(const InnerSmemDf<float4>& S, int s, int e, float4* x, cdf2 st, bool store,
                                        bool rhs) {
#pragma unroll 1
  for (int m = e - 1; m >= s; --m) {
    const cdf g = rhs ? e_load(&x[m]) : c_zero();
    const cdf v = e_submul(e_submul(g, e_load(&S.u2[m]), st.y), e_load(&S.u1[m]), st.x);
    if (store) e_store(&x[m], v);
    st = {v, st.x};
  }
  return st;
}
// the same where row e - 1 was not exchanged, state: x[m + 1]
__device__ __forceinline__ df64 chunk_u(const InnerSmemDf<float2>& S, int s, int e, float2* x, df64 x1, bool store,
                                        bool rhs) {
  df64 x2 = df_zero();
#pragma unroll 1
  for (int m = e - 1; m >= s; --m) {
    const df64 g = rhs ? e_load(&x[m]) : df_zero();
    const df64 v = e_submul(e_submul(g, e_load(&S.u2[m]), x2), e_load(&S.u1[m]), x1);
    if (store) e_store(&x[m], v);
    x2 = x1;
    x1 = v;
  }
  return x1;
}
// (1 + N)^dag, down the rows, state: y[m - 1], y[m - 2]; y[m] / conj(diag(U)) is stored
__device__ __forceinline__ cdf2 chunk_ud(const InnerSmemDf<float4>& S, int s, int e, const float4* b, float4* z, cdf2 st,
                                         bool store, bool rhs) {
#pragma unroll 1
  for (int m = s; m < e; ++m) {
    cdf v = rhs ? e_load(&b[m]) : c_zero();
    if (m >= 2) v = e_submulc(v, e_load(&S.u2[m - 2]), st.y);
    if (m >= 1) v = e_submulc(v, e_load(&S.u1[m - 1]), st.x);
    if (store) e_store(&z[m], e_mul(v, e_conj(e_load(&S.uinv[m]))));
    st = {v, st.x};
  }
  return st;
}
// the adjoint interchanges and L^dag, up the rows: step m reads z[m] and fixes z[m + 1], so
// the lane's steps are m = e - 2 .. s - 1 (it fixes its own rows; zs = z[s - 1] is another
// lane's, read before the side's barrier); state: the pending z[m + 1]
template <class E, class St>
__device__ __forceinline__ E chunk_ld(const InnerSmemDf<St>& S, int k, int s, int e, St* z, E zs, E gn, bool store) {
  if (s >= e) return gn;
  if (e == k) gn = e_load(&z[k - 1]);
#pragma unroll 1
  for (int m = e - 2; m >= s - 1 && m >= 0; --m) {
    const E zm = m >= s ? e_load(&z[m]) : zs;
    const E v = e_submulc(zm, e_load(&S.l[m]), gn);
    const bool sw = S.sw[m];
    if (store) e_store(&z[m + 1], sw ? v : gn);
    gn = sw ? gn : v;
  }
  if (store && s == 0) e_store(&z[0], gn);
  return gn;
}
// the product of the multipliers of steps first .. last (conjugated for the adjoint)
template <class E, class St>
__device__ __forceinline__ E map_l(const InnerSmemDf<St>& S, int first, int last, bool conj) {
  E p = e_one(E{});
  for (int m = first; m <= last; ++m)
    if (!S.sw[m]) {
      const E lm = e_load(&S.l[m]);
      p = e_submul(e_zero(E{}), conj ? e_conj(lm) : lm, p);
    }
  return p;
}

// each warp's sums of NQ values into red[warp][NQ]
template <int NQ>
__device__ __forceinline__ void warps_to_red(df64 (&v)[NQ], df64* red) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = warp_sum(v[q]);
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int q = 0; q < NQ; ++q) red[(threadIdx.x >> 5) * NQ + q] = v[q];
}
// sum over the four warps from w0 on
__device__ __forceinline__ df64 red_sum(const df64* red, int w0, int nq, int q) {
  static_assert(kSideWarps == 4, "four warps a side");
  const df64 s = red[w0 * nq + q] + red[(w0 + 1) * nq + q];
  const df64 t = red[(w0 + 2) * nq + q] + red[(w0 + 3) * nq + q];
  return s + t;
}

template <bool CPLX>
struct UScan;
template <> struct UScan<true> { using M = cmat2; using S = cdf2; };
template <> struct UScan<false> { using M = df64; using S = df64; };

// CPLX: two-sided Lanczos, side 0 (threads 0 .. 127) carries q, side 1 w; else Lanczos on the
// real symmetric H, one side
template <bool CPLX>
__global__ void __launch_bounds__((CPLX ? 2 : 1) * kSideLanes)
    k_inner_df(const int* __restrict__ k_dev, const int* __restrict__ l_dev, const double2* __restrict__ alp,
               const double2* __restrict__ bet, const double2* __restrict__ gam, int ldc, InnerWork w) {
  using E = typename RhDf<CPLX>::E;
  using St = typename RhDf<CPLX>::St;
  extern __shared__ __align__(16) unsigned char smem[];
  const int prob = blockIdx.x;
  const int k = k_dev[prob];
  const int l = min(l_dev[prob], k);
  const int tid = threadIdx.x;
  InnerSmemDf<St> S;
  {
    St* base = (St*)smem;
    S.d = base; S.a = base + k; S.c = base + 2 * k;
    S.uinv = base + 3 * k; S.u1 = base + 4 * k; S.u2 = base + 5 * k; S.l = base + 6 * k;
    S.q = base + 7 * k; S.qp = base + 8 * k; S.w = base + 9 * k; S.wp = base + 10 * k;
    S.u = base + 11 * k; S.z = base + 12 * k;
    S.red = (df64*)(base + 13 * k);
    S.sw = (unsigned char*)(S.red + 32);
  }
  const E zero = e_zero(E{});
  const size_t crow = (size_t)(prob % w.rows) * ldc;
  const double2* al = alp + crow;
  const double2* be = bet + crow;
  const double2* ga = gam + crow;
  const double2 z2 = make_double2(0.0, 0.0);
  for (int m = tid; m < k; m += blockDim.x) {
    // at mu = 0 the superdiagonal is beta too, imaginary parts are ignored
    const E am = e_from2(m >= 1 ? be[m + 1] : z2, zero);
    e_store(&S.d[m], e_from2(al[m + 1], zero));
    e_store(&S.a[m], am);
    e_store(&S.c[m], e_from2(m + 1 < k ? (CPLX ? ga[m + 2] : be[m + 2]) : z2, zero));
    e_store(&S.u[m], e_inv(am));  // for the factorisation
    const E q0 = m == 0 ? e_one(E{}) : zero;
    e_store(&S.q[m], q0);
    e_store(&S.w[m], q0);
    e_store(&S.qp[m], zero);
    e_store(&S.wp[m], zero);
  }
  __syncthreads();
  __shared__ int s_ok;
  if (tid == 0) s_ok = tri_factor_df<E, St>(S, k, S.u) ? 1 : 0;
  __syncthreads();
  if (!s_ok) {
    if (tid == 0) { w.fail[prob] = 1; w.leff[prob] = 0; }
    return;
  }
  const int side = CPLX ? tid / kSideLanes : 0, t = tid % kSideLanes;
  // this lane's rows [r0, r1); at mu = 0 the chunks end at rows that were not exchanged
  const int rows = (k + kSideLanes - 1) / kSideLanes;
  int r0 = min(t * rows, k), r1 = min((t + 1) * rows, k);
  if constexpr (!CPLX) {
    while (r0 < k && r0 > 0 && S.sw[r0 - 1]) --r0;
    while (r1 < k && r1 > 0 && S.sw[r1 - 1]) --r1;
  }
  // fl: the recurrence with L (side 0: down the rows), fu: the one with U (side 1: down the
  // rows), Mu and Su its maps and states
  using Mu = typename UScan<CPLX>::M;
  using Su = typename UScan<CPLX>::S;
  __shared__ ScanShared<E, E> shl[CPLX ? 2 : 1];
  __shared__ ScanShared<Mu, Su> shu[CPLX ? 2 : 1];
  ScanMaps<E> fl;
  ScanMaps<Mu> fu;
  const ScanPos posl = scan_pos(side == 0), posu = scan_pos(side == 1);
  {
    if constexpr (CPLX) {
      const cdf2 e1 = {c_one(), zero}, e2 = {zero, c_one()};
      const cdf2 m1 = side == 0 ? chunk_u(S, r0, r1, S.u, e1, false, false) : chunk_ud(S, r0, r1, S.w, S.z, e1, false, false);
      const cdf2 m2 = side == 0 ? chunk_u(S, r0, r1, S.u, e2, false, false) : chunk_ud(S, r0, r1, S.w, S.z, e2, false, false);
      scan_setup(fu, shu[side], cmat2{m1.x, m2.x, m1.y, m2.y}, posu);
    } else {
      scan_setup(fu, shu[side], chunk_u(S, r0, r1, S.u, e_one(E{}), false, false), posu);
    }
    const int first = side == 0 ? r0 : max(r0 - 1, 0), last = side == 0 ? min(r1, k - 1) - 1 : r1 - 2;
    scan_setup(fl, shl[side], map_l<E, St>(S, first, r0 < r1 ? last : first - 1, side == 1), posl);
  }
  __syncthreads();
  // the side's vectors and coefficients: M = H + H^{-1} on q; M^dag on w, whose H^dag has
  // conj(c[m - 1]) below and conj(a[m + 1]) above the diagonal
  St* const X = side == 0 ? S.q : S.w;
  St* const XP = side == 0 ? S.qp : S.wp;
  St* const U = side == 0 ? S.u : S.z;
  const St* const below = side == 0 ? S.a : S.c - 1;
  const St* const above = side == 0 ? S.c : S.a + 1;
  const bool cj = side == 1;
  // Q keeps the float pairs as they are (k_combine widens them)
  float4* Q = (float4*)(w.Q + (size_t)prob * w.ld * kMaxL);
  double2* T = w.T + (size_t)prob * kMaxL * 3;
  E b_i = zero, g_i = zero;
  int done = 0;
  const float exhaust_tol = 1e-13f;
  for (int i = 0; i < l; ++i) {
    // u = H^{-1} q, then p = M q - g_i q_{i-1}; z = H^{-dag} w, then r = M^dag w - b_i w_{i-1}
    // (rows of this lane only, but for the barriers of the scans). Side 0 runs the recurrence
    // with L and then the one with U, side 1 the other way round; each from a zero state, then
    // from the state the scan gives.
    df64 dots[3] = {df_zero(), df_zero(), df_zero()};  // alpha = w^dag p, ||M q||^2
    if (side == 0)
      for (int m = r0; m < r1; ++m) Q[(size_t)m * kMaxL + i] = e_pairs(e_load(&S.q[m]));
#pragma unroll 1
    for (int stage = 0; stage < 2; ++stage) {
      if (stage == side) {
        const E head = side == 0 && t == 0 ? e_load(&S.q[0]) : zero;  // the first pending row
        const E zs = side == 1 && r0 >= 1 && r0 < r1 ? e_load(&S.z[r0 - 1]) : zero;
        E st = head;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
          if (side == 0) st = chunk_l(S, k, r0, r1, S.q, S.u, st, pass == 1);
          else if constexpr (CPLX) st = chunk_ld(S, k, r0, r1, S.z, zs, st, pass == 1);
          if (pass == 0) {
            st = scan_in(fl, shl[side], st, posl, side);
            if (side == 0 && t == 0) st = head;
          }
        }
      } else {
        Su st = e_zero(Su{});
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
          if (side == 0) st = chunk_u(S, r0, r1, S.u, st, pass == 1, true);
          else if constexpr (CPLX) st = chunk_ud(S, r0, r1, S.w, S.z, st, pass == 1, true);
          if (pass == 0) st = scan_in(fu, shu[side], st, posu, side);
        }
      }
      if (side == 1) side_sync(1);  // its second sweep reads the row before this lane's
    }
    float mq2 = 0.f;
    const E gi = side == 1 ? b_i : g_i;
#pragma unroll 1
    for (int m = r0; m < r1; ++m) {
      const E xm = e_load(&X[m]);
      E dm = e_load(&S.d[m]);
      if (cj) dm = e_conj(dm);
      E v = e_addmul(e_load(&U[m]), dm, xm);
      if (m >= 1) {
        E f = e_load(&below[m]);
        if (cj) f = e_conj(f);
        v = e_addmul(v, f, e_load(&X[m - 1]));
      }
      if (m + 1 < k) {
        E f = e_load(&above[m]);
        if (cj) f = e_conj(f);
        v = e_addmul(v, f, e_load(&X[m + 1]));
      }
      mq2 += e_abs2hi(v);
      const E pm = e_submul(v, gi, e_load(&XP[m]));
      e_store(&U[m], pm);
      if (side == 0) {
        df64 d[2] = {dots[0], dots[1]};
        e_dot(d, CPLX ? e_load(&S.w[m]) : xm, pm);
        dots[0] = d[0];
        dots[1] = d[1];
      }
    }
    dots[2] = {mq2, 0.f};
    if (side == 0) warps_to_red(dots, S.red);
    __syncthreads();
    const df64 mqn = df_sqrt(red_sum(S.red, 0, 3, 2));
    E a_i;
    if constexpr (CPLX) a_i = {red_sum(S.red, 0, 3, 0), red_sum(S.red, 0, 3, 1)};
    else a_i = red_sum(S.red, 0, 3, 0);
    if (tid == 0) T[i * 3 + 0] = e_to2(a_i);
    done = i + 1;
    if (i == l - 1) break;
    // q~ = p - alpha q ; w~ = r - conj(alpha) w ; delta = w~^dag q~ (side 0 its real part,
    // side 1 the imaginary part) or ||q~||^2
    df64 dl[1] = {df_zero()};
    const E as = cj ? e_conj(a_i) : a_i;
#pragma unroll 1
    for (int m = r0; m < r1; ++m) {
      const E v = e_submul(e_load(&U[m]), as, e_load(&X[m]));
      e_store(&U[m], v);
      if constexpr (!CPLX) dl[0] = df_axpy1(dl[0], v, v);
    }
    __syncthreads();  // both sides' q~, w~; S.red is free again
    if constexpr (CPLX) {
#pragma unroll 1
      for (int m = r0; m < r1; ++m) {
        const E qt = e_load(&S.u[m]), wt = e_load(&S.z[m]);
        const df64 y1 = side == 0 ? qt.re : qt.im, y2 = side == 0 ? qt.im : -qt.re;
        dl[0] = df_axpy2(dl[0], wt.re, y1, wt.im, y2);
      }
    }
    warps_to_red(dl, S.red);
    __syncthreads();
    df64 bn;
    E gn;
    if constexpr (CPLX) {
      const df64 dre = red_sum(S.red, 0, 1, 0), dim = red_sum(S.red, kSideWarps, 1, 0);
      bn = df_sqrt(df_sqrt(df_axpy2(df_zero(), dre, dre, dim, dim)));
      const df64 rb = bn.hi > 0.f ? df_recip(bn) : df_zero();
      gn = {dre * rb, dim * rb};
    } else {
      bn = df_sqrt(red_sum(S.red, 0, 1, 0));
      gn = bn;
    }
    if (!(bn.hi > exhaust_tol * mqn.hi)) break;  // inner space exhausted: T_i is exact
    if (tid == 0) {
      T[(i + 1) * 3 + 1] = make_double2(df_to_double(bn), 0.0);
      T[(i + 1) * 3 + 2] = e_to2(gn);
    }
    const E sc = e_inv(side == 0 ? e_real(bn, zero) : e_conj(gn));
#pragma unroll 1
    for (int m = r0; m < r1; ++m) {
      XP[m] = X[m];
      e_store(&X[m], e_mul(e_load(&U[m]), sc));
    }
    b_i = e_real(bn, zero);
    g_i = gn;
    __syncthreads();
  }
  if (tid == 0) {
    w.leff[prob] = done;
    T[0 * 3 + 1] = make_double2(0.0, 0.0);
    T[0 * 3 + 2] = make_double2(0.0, 0.0);
    w.fail[prob] = 0;
  }
}

// ------------------------------------------------- the first column of a Roberts-Higham iterate
// A nested check needs only s = sgn(T_l) e_1, and T_l is tridiagonal. The iterates of Eq.
// (Roberts), here with scales, S_{n+1} = (g_n S_n + (g_n S_n)^{-1}) / 2 from S_0 = T, are rational
// functions of T whose poles lie on the imaginary axis, are simple, and are known beforehand: the
// poles of S_{n+1} are those of S_n, their residues times g_n / 2, and the 2^n zeros of S_n. So
//   s_{n+1} = (g_n / 2) s_n + sum_{S_n(z) = 0} (T - z)^{-1} e_1 / (2 g_n S_n'(z)),
// and g_k S_k(z) = i y_k runs backwards from y_{n-1} = +-1 through y_k = tau +- sqrt(tau^2 + 1), tau =
// y_{k+1} / g_{k+1}, to z = i y_0 / g_0, with S_n'(z) = prod_k g_k (1 + y_k^{-2}) / 2: every sign choice
// is one zero. s is a sum of solutions of shifted tridiagonal systems, all independent: one
// thread solves one, in float pairs and with partial pivoting, and the l x l inversions with
// their l dependent pivot steps each are gone (24 matrices of l = 120: 11.2 -> 0.077 ms).
//  - The rows are eliminated from the last to the first, so that the right-hand side e_1 stays
//    zero until the last step: the forward sweep keeps no multipliers, the back substitution
//    reads two numbers a row, kept in scratch ([row][thread], coalesced; L2-resident).
//  - Scales: g_n = 1 with rh_scaling = 0; else g_0 centres the range of |lambda|, from 1.5
//    (|x + 1/x| >= 2 for real x) to an estimate by tr T^2 and tr T^4, and the later g_n, powers
//    of two (exact), what is left of it; one large eigenvalue of H^{-1} then costs steps by the
//    logarithm of its size.
//  - Stop as k_rh: ||s_n - s_{n-1}|| <= rh_tol ||s_n||, on the column, tested from n = 4 on (the
//    first 128 solves give s_1 .. s_7). An eigenvector of small weight in e_1 shows in the
//    matrix's norm but less in the column's, so the column returned is that of one more step.
//    Iterations, reported as rh_iters: n.
//  - A matrix that meets a zero pivot, overflows or needs more than 2^12 - 1 poles or more than
//    rh_maxit steps is left to k_rh_df, whose verdict stands.
// Bound: the latency of one thread's elimination (~450 cycles a row) at one warp a scheduler.
constexpr int kColThreads = 128;
constexpr int kColMaxLevel = 12;

__device__ __forceinline__ float2 fmul2c(float2 a, float2 b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }

__global__ void __launch_bounds__(kColThreads) k_rh_col(int count, int hermitian, InnerWork w, int dl, double rh_tol,
                                                        int rh_maxit, int mid0, int scale) {
  __shared__ float4 sd[kMaxL + 2], ssub[kMaxL + 2], ssup[kMaxL + 2];  // T_pp, T_{p,p-1}, T_{p,p+1}
  __shared__ float2 sred[kColThreads / 32];
  __shared__ float sg[kColMaxLevel + 1];  // g_n
  const int mid = mid0 + blockIdx.x, prob = mid % count;
  const int t = threadIdx.x;
  const int le = w.leff[prob];
  const int m = mid < count ? le : le - dl;
  if (m <= 0) {
    if (t == 0) { w.rh_ok[mid] = m == 0 ? 0 : 1; w.rh_its[mid] = 0; }
    return;
  }
  const cdf zero = c_zero();
  // block sums of two floats
  auto sum2 = [&](float a, float b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    __syncthreads();
    if ((t & 31) == 0) sred[t >> 5] = make_float2(a, b);
    __syncthreads();
    float2 r = sred[0];
    for (int v = 1; v < kColThreads / 32; ++v) { r.x += sred[v].x; r.y += sred[v].y; }
    return r;
  };
  if (t < kMaxL + 2) {
    const double2* T = w.T + (size_t)prob * kMaxL * 3;
    const double2 z2 = make_double2(0.0, 0.0);
    double2 d = t < m ? T[t * 3 + 0] : z2, b = t >= 1 && t < m ? T[t * 3 + 1] : z2;
    double2 g = t + 1 < m ? T[(t + 1) * 3 + 2] : z2;  // T_{t,t+1}
    if (hermitian) d.y = b.y = g.y = 0.0;
    e_store(&sd[t], e_from2(d, zero));
    e_store(&ssub[t], e_from2(b, zero));
    e_store(&ssup[t], e_from2(g, zero));
  }
  if (t <= kColMaxLevel) sg[t] = 1.f;
  __syncthreads();
  if (scale) {
    // with e_p = T_{p,p+1} T_{p+1,p}: tr T^2 = sum A_p, A_p = T_pp^2 + e_{p-1} + e_p, and tr T^4 =
    // sum A_p^2 + 2 e_p (T_pp + T_{p+1,p+1})^2 + 2 e_p e_{p+1}
    float2 t2 = {0.f, 0.f}, t4 = {0.f, 0.f};
    if (t < m) {
      auto hi = [](const float4* v) { return make_float2(v->x, v->z); };
      auto ep = [&](int p) { return p < 0 ? make_float2(0.f, 0.f) : fmul2c(hi(&ssup[p]), hi(&ssub[p + 1])); };
      const float2 d0 = hi(&sd[t]), d1 = hi(&sd[t + 1]), em = ep(t - 1), e0 = ep(t), e1 = ep(t + 1);
      const float2 dd = fmul2c(d0, d0);
      t2 = {dd.x + em.x + e0.x, dd.y + em.y + e0.y};
      const float2 ds = {d0.x + d1.x, d0.y + d1.y};
      const float2 a2 = fmul2c(t2, t2), c2 = fmul2c(e0, fmul2c(ds, ds)), ee = fmul2c(e0, e1);
      t4 = {a2.x + 2.f * (c2.x + ee.x), a2.y + 2.f * (c2.y + ee.y)};
    }
    t2 = sum2(t2.x, t2.y);
    t4 = sum2(t4.x, t4.y);
    if (t == 0) {
      // mean square eigenvalue; the largest stands out of tr T^4 where it is far above the rest
      const float ms = sqrtf(t2.x * t2.x + t2.y * t2.y) / (float)m;
      const float ex = sqrtf(t4.x * t4.x + t4.y * t4.y) - 2.f * (float)m * ms * ms;
      float hi = fmaxf(2.f * sqrtf(ms), ex > 0.f ? sqrtf(sqrtf(ex)) : 0.f), lo = 1.5f;
      if (hi < 1e8f) {  // (false for a NaN)
        hi = fmaxf(hi, lo);
        for (int n = 0; n <= kColMaxLevel; ++n) {
          const float g = n == 0 ? rsqrtf(lo * hi) : ldexpf(1.f, -(int)rintf(0.5f * log2f(lo * hi)));
          sg[n] = g;
          lo *= g;
          hi *= g;
          hi = fmaxf(0.5f * (lo + 1.f / lo), 0.5f * (hi + 1.f / hi));
          lo = 1.f;
        }
      }
    }
    __syncthreads();
  }
  // this thread's two rows of numbers per eliminated row; the solution overwrites the first
  float4* const rx = (float4*)w.S + (size_t)blockIdx.x * 2 * kMaxL * kColThreads;
  float4* const u1 = rx + t;
  float4* const u2 = u1 + (size_t)kMaxL * kColThreads;
  // (T - z) x = e_1 for pole idx (the zeros of S_b are idx = 2^b .. 2^{b+1} - 1), times its
  // weight; idx = 0: weight zero
  auto solve = [&](int idx) -> bool {
    const int id = max(idx, 1);
    const int b = 31 - __clz(id);
    const df64 gi0 = df_recip(df64{sg[0], 0.f});
    df64 sh = df_zero(), wt = b > 0 ? df64{0.5f / sg[b], 0.f} : df_half(gi0);
    if (b > 0) {
      df64 y = {id & 1 ? -1.f : 1.f, 0.f};
      wt = b > 1 ? wt * (1.f / sg[b - 1]) : wt * gi0;
#pragma unroll 1
      for (int k = b - 2; k >= 0; --k) {
        const df64 tau = y * (1.f / sg[k + 1]);
        const bool up = (id >> (b - 1 - k)) & 1;  // y = tau + sqrt(tau^2 + 1) or its negative inverse
        const df64 h = (tau.hi < 0.f ? -tau : tau) + df_sqrt(df_axpy1(df64{1.f, 0.f}, tau, tau));
        const df64 hi = df_recip(h);
        const bool big = up == (tau.hi >= 0.f);
        const df64 ya = big ? h : hi, yi = big ? hi : h;  // |y|, 1 / |y|
        y = up ? ya : -ya;
        // 1 / (g (1 + y^{-2}) / 2)
        wt = wt * df_recip(df_half(df_axpy1(df64{1.f, 0.f}, yi, yi)));
        wt = k > 0 ? wt * (1.f / sg[k]) : wt * gi0;
      }
      sh = y * gi0;
    }
    if (idx == 0) wt = df_zero();
    cdf dd = e_load(&sd[m - 1]);
    dd.im = dd.im - sh;
    cdf ee = m > 1 ? e_load(&ssub[m - 1]) : zero;
    bool fine = true, lastsw = false;
    cdf ri = zero, lm = zero;
#pragma unroll 1
    for (int p = m - 2; p >= 0; --p) {  // row p enters; row p + 1 or p becomes final
      const cdf an = e_load(&ssup[p]);
      cdf dn = e_load(&sd[p]);
      dn.im = dn.im - sh;
      const cdf cn = p >= 1 ? e_load(&ssub[p]) : zero;
      const float ad = e_abs2hi(dd), aa = e_abs2hi(an);
      const bool sw = !(ad >= aa);
      fine = fine && fmaxf(ad, aa) > 0.f;
      ri = e_inv(sw ? an : dd);
      lm = e_mul(sw ? dd : an, ri);
      const cdf r1 = sw ? dn : ee;
      const cdf nd = e_submul(sw ? ee : dn, lm, r1);
      e_store(&u1[(size_t)p * kColThreads], e_mul(r1, ri));
      if (sw) {
        e_store(&u2[(size_t)p * kColThreads], e_mul(cn, ri));
        ee = e_submul(zero, lm, cn);
      } else {
        e_store(&u2[(size_t)p * kColThreads], zero);
        ee = cn;
      }
      dd = nd;
      lastsw = sw;
    }
    fine = fine && e_abs2hi(dd) > 0.f;
    // the right-hand side after the last step: (1, -lm) if the rows were exchanged, else (0, 1)
    const cdf one = c_one();
    cdf x1 = e_inv(dd);
    if (m > 1 && lastsw) x1 = e_submul(zero, lm, x1);
    cdf x2 = zero;
    // x is kept by row of T: x_0 = x1 here; u1, u2 of step p give x_{p+1} from x_p, x_{p-1}
    cdf keep = c_scale(x1, wt);
    cdf a = zero, bb = zero;
    if (m > 1) { a = e_load(&u1[0]); bb = e_load(&u2[0]); }
    e_store(&u1[0], keep);
    constexpr int PF = 4;  // rows loaded ahead (the scratch is in L2)
    cdf na[PF], nb[PF];
#pragma unroll
    for (int i = 0; i < PF; ++i)
      if (1 + i < m - 1) {
        na[i] = e_load(&u1[(size_t)(1 + i) * kColThreads]);
        nb[i] = e_load(&u2[(size_t)(1 + i) * kColThreads]);
      }
    if (m > 1) {
      // x_1 = rhs / pivot - u1 x_0 (rhs 1 if the rows were exchanged)
      const cdf x = e_submul(lastsw ? ri : zero, a, x1);
      x2 = x1;
      x1 = x;
      keep = c_scale(x1, wt);
    }
#pragma unroll 1
    for (int p0 = 1; p0 < m - 1; p0 += PF) {
      cdf ca[PF], cb[PF];
#pragma unroll
      for (int i = 0; i < PF; ++i) {
        ca[i] = na[i];
        cb[i] = nb[i];
        const int pn = p0 + PF + i;
        if (pn < m - 1) {
          na[i] = e_load(&u1[(size_t)pn * kColThreads]);
          nb[i] = e_load(&u2[(size_t)pn * kColThreads]);
        }
      }
#pragma unroll
      for (int i = 0; i < PF; ++i) {
        const int p = p0 + i;
        if (p < m - 1) {
          e_store(&u1[(size_t)p * kColThreads], keep);  // x_p
          const cdf x = e_submul(e_submul(zero, cb[i], x2), ca[i], x1);
          x2 = x1;
          x1 = x;
          keep = c_scale(x1, wt);
        }
      }
    }
    if (m > 1) e_store(&u1[(size_t)(m - 1) * kColThreads], keep);
    return fine || idx == 0;
  };
  // sum over threads [a, b) of row t's solutions (thread t: row t of T)
  const float4* const row = rx + (size_t)t * kColThreads;
  auto rowsum = [&](int a, int b) {
    cdf s0 = zero, s1 = zero, s2 = zero, s3 = zero;
    int i = a;
#pragma unroll 1
    for (; i + 4 <= b; i += 4) {
      s0 = c_add(s0, e_load(&row[i]));
      s1 = c_add(s1, e_load(&row[i + 1]));
      s2 = c_add(s2, e_load(&row[i + 2]));
      s3 = c_add(s3, e_load(&row[i + 3]));
    }
#pragma unroll 1
    for (; i < b; ++i) s0 = c_add(s0, e_load(&row[i]));
    return c_add(c_add(s0, s1), c_add(s2, s3));
  };
  const float tol2 = (float)rh_tol * (float)rh_tol;
  // ||f - g||^2 <= tol^2 ||f||^2 over the rows
  auto same = [&](cdf f, cdf g) {
    float d = 0.f, n = 0.f;
    if (t < m) {
      const df64 dr = f.re - g.re, di = f.im - g.im;
      d = dr.hi * dr.hi + di.hi * di.hi;
      n = e_abs2hi(f);
    }
    const float2 r = sum2(d, n);
    return r.x <= tol2 * r.y;
  };
  // (g_n / 2) f + sum
  auto next = [&](cdf f, int n, cdf sum) { return c_add(e_scale(f, 0.5f * sg[n]), sum); };
  bool fine = solve(t);
  __syncthreads();
  cdf f = t == 0 ? e_load(&sd[0]) : t == 1 && m > 1 ? e_load(&ssub[1]) : zero;  // S_0 e_1 of this row
  int level = 7, its = 0;
  bool conv = false, was = false;
#pragma unroll 1
  for (int n = 0; n < 7; ++n) {
    const cdf fn = t < m ? next(f, n, rowsum(1 << n, 2 << n)) : zero;
    was = conv;
    if (n >= 3 && !conv) {
      conv = same(fn, f);
      if (conv) its = n + 1;
    }
    f = fn;
  }
  // the poles of further steps, kColThreads at a time, until one step past the convergence
  while (!was && level < kColMaxLevel && level <= rh_maxit) {
    cdf sum = zero;
    for (int i0 = 1 << level; i0 < 2 << level; i0 += kColThreads) {
      __syncthreads();  // every row has been summed
      fine = solve(i0 + t) && fine;
      __syncthreads();
      if (t < m) sum = c_add(sum, rowsum(0, kColThreads));
    }
    const cdf fn = t < m ? next(f, level, sum) : zero;
    ++level;
    was = conv;
    if (!conv) {
      conv = same(fn, f);
      if (conv) its = level;
    }
    f = fn;
  }
  const bool good = was && its <= rh_maxit;
  const bool finite = t >= m || (isfinite(f.re.hi) && isfinite(f.im.hi));
  const int all = __syncthreads_and(fine && finite && good);
  if (t == 0) {
    w.rh_ok[mid] = all ? 1 : kRhLeft;
    w.rh_its[mid] = its;
  }
  if (all && t < m) {
    if (hermitian) f.im = df_zero();
    w.s[(size_t)mid * kMaxL + t] = e_to2(f);
  }
}

// ------------------------------------------------------------ combine
// c = Q_l s and the inner estimate, a cluster of kCombineCtas CTAs a problem (the sums over l
// are in double, whose pipe gives two multiply-adds a cycle and SM: one CTA a problem took
// 0.26 ms for 12 of k = 333, l = 120, the cluster 0.048). Eight lanes share a row of Q. The
// difference to the c of the leading l - dl block is summed as c - c' = Q (s - [s'; 0]), in double
// like c (in float pairs it took longer, 0.067 ms, for 1e-15 in place of 1e-16 in the estimate).
constexpr int kCombineCtas = 8, kCombineThreads = 128;

__global__ void __cluster_dims__(kCombineCtas, 1, 1) __launch_bounds__(kCombineThreads)
    k_combine(int count, const int* __restrict__ k_dev, const int* __restrict__ l_dev, InnerWork w, int dl, double2* c,
              int ldo, void* cacc, const double* nv, int ldn, int prec, double* cnorm, double* est_inner, int* rh_status,
              int* rh_iters, int have_est) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double2 s_s[kMaxL];
  __shared__ double2 s_ds[kMaxL];
  __shared__ double s_red[kCombineThreads / 32][2];
  __shared__ double s_tot[kCombineCtas][2];
  // a CTA's shared memory may be written by another once it is known to run: all arrive here, and
  // wait before the one remote write (the sums over Q lie between, so the wait costs nothing)
  cluster.barrier_arrive();
  const int rank = (int)cluster.block_rank(), prob = blockIdx.x / kCombineCtas, row0 = prob % w.rows;
  const int k = k_dev[prob];
  const int le = w.leff[prob];
  const int le2 = le - dl;
  const int tid = threadIdx.x, sub = tid & 7, rl = tid >> 3;
  const double2* s1 = w.s + (size_t)prob * kMaxL;
  const double2* s2 = w.s + (size_t)(count + prob) * kMaxL;
  const bool bad = w.fail[prob] != 0 || le <= 0 || !w.rh_ok[prob];
  // the inner space is exact when it was exhausted early or spans all of C^k
  const bool exact = le >= k || le < min(l_dev[prob], k);
  for (int i = tid; i < le && !bad; i += kCombineThreads) {
    const double2 v = s1[i];
    const double2 v2 = have_est && i < le2 ? s2[i] : make_double2(0.0, 0.0);
    s_s[i] = v;
    s_ds[i] = zsub(v, v2);
  }
  __syncthreads();
  // the double-float inner level keeps Q as float pairs in the doubles' bytes
  const double2* Q = w.Q + (size_t)prob * w.ld * kMaxL;
  const bool pairs = w.arith == OV_INNER_DF64;
  auto put = [&](int m, double2 v) {
    c[(size_t)prob * ldo + m + 1] = v;
    if (!cacc) return;
    // the recombination sums c_j v_j = (c_j / nv_j) t_j over the unnormalised basis
    const double sc = nv && m < k ? 1.0 / nv[(size_t)row0 * ldn + m + 1] : 1.0;
    const double2 vs = make_double2(v.x * sc, v.y * sc);
    if (prec == OV_PREC_FP64) {
      ((double2*)cacc)[(size_t)prob * ldo + m + 1] = vs;
    } else {
      const df64 re = df_from_double(vs.x), im = df_from_double(vs.y);
      ((float4*)cacc)[(size_t)prob * ldo + m + 1] = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
  };
  double nc = 0.0, nd = 0.0;
  // entries k+1 .. ldo-1 are cleared so that a shorter c never carries stale values
  for (int m = k + rank * kCombineThreads + tid; m < ldo - 1; m += kCombineCtas * kCombineThreads)
    put(m, make_double2(0.0, 0.0));
  for (int m0 = rank * (kCombineThreads / 8); m0 < k; m0 += kCombineCtas * (kCombineThreads / 8)) {
    const int m = m0 + rl;
    double2 v = make_double2(0.0, 0.0);
    double2 d = make_double2(0.0, 0.0);
    if (!bad && m < k) {
      for (int i = sub; i < le; i += 8) {
        const double2* qp = &Q[(size_t)m * kMaxL + i];
        const double2 qv = pairs ? e_to2(e_load((const float4*)qp)) : *qp;
        v = zadd(v, zmul(qv, s_s[i]));
        if (have_est) d = zadd(d, zmul(qv, s_ds[i]));
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
      d.x += __shfl_xor_sync(0xffffffffu, d.x, o);
      d.y += __shfl_xor_sync(0xffffffffu, d.y, o);
    }
    if (sub == 0 && m < k) {
      put(m, v);
      nc += zabs2(v);
      nd += zabs2(d);
    }
  }
  nc = warp_sum(nc);
  nd = warp_sum(nd);
  if ((tid & 31) == 0) { s_red[tid >> 5][0] = nc; s_red[tid >> 5][1] = nd; }
  __syncthreads();
  cluster.barrier_wait();
  if (tid < 2) {
    double t = 0.0;
    for (int q = 0; q < kCombineThreads / 32; ++q) t += s_red[q][tid];
    *cluster.map_shared_rank(&s_tot[rank][tid], 0) = t;
  }
  cluster.sync();
  if (rank == 0 && tid == 0) {
    double tc = 0.0, td = 0.0;
    for (int q = 0; q < kCombineCtas; ++q) { tc += s_tot[q][0]; td += s_tot[q][1]; }
    const double cn = sqrt(tc);
    // inner estimate: 0 when the inner space is exact (exhausted or l_eff = k)
    double ei;
    if (bad) ei = INFINITY;
    else if (exact) ei = 0.0;
    else if (!have_est) ei = NAN;
    else if (le2 < 1 || w.rh_ok[count + prob] == 0) ei = INFINITY;
    else ei = sqrt(td) / cn;
    est_inner[prob] = ei;
    cnorm[prob] = cn;
    rh_status[prob] = bad ? (w.fail[prob] ? 2 : 1) : 0;
    rh_iters[prob] = w.rh_its[prob];
  }
}

// the outer estimate ||c - [c_prev; 0]|| / ||c|| of every problem; c_prev: the same problem's c
// w.rows places before (the previous check of a group), or row prob of cprev
__global__ void __launch_bounds__(kCombineThreads) k_estimate(const int* __restrict__ k_dev, InnerWork w, const double2* c,
                                                              int ldo, const double* cnorm, const int* rh_status,
                                                              const double2* cprev, int ldp, const int* kprev_dev,
                                                              double* est_outer) {
  __shared__ double red[kCombineThreads / 32];
  const int prob = blockIdx.x;
  const bool first = prob < w.rows;
  const int k = k_dev[prob];
  const int kp = first ? (kprev_dev && cprev ? kprev_dev[prob] : 0) : k_dev[prob - w.rows];
  const double2* pr = first ? cprev + (size_t)prob * ldp : c + (size_t)(prob - w.rows) * ldo;
  double no = 0.0;
  if (kp > 0)
    for (int m = threadIdx.x; m < k; m += kCombineThreads) {
      const double2 v = c[(size_t)prob * ldo + m + 1];
      const double2 pv = m < kp ? pr[m + 1] : make_double2(0.0, 0.0);
      no += zabs2(zsub(v, pv));
    }
  no = block_sum(no, red);
  if (threadIdx.x == 0) est_outer[prob] = kp > 0 && rh_status[prob] == 0 ? sqrt(no) / cnorm[prob] : INFINITY;
}

__global__ void k_check_setup(int rows, int n, CheckSteps cj, const int* __restrict__ status,
                              const int* __restrict__ kbreak, const int* __restrict__ l_in, const int* err, int* k_out,
                              int* l_out, int* status_out, int* kbreak_out, int* err_out) {
  if (threadIdx.x == 0) *err_out = *err;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    const int s = status[r], kb = kbreak[r];
    status_out[r] = s;
    kbreak_out[r] = kb;
    for (int p = r; p < n; p += rows) {
      const int j = cj.j[p / rows];
      k_out[p] = s != kStOK && kb > 0 ? min(kb, j) : j;
      l_out[p] = l_in[r];
    }
  }
}
cudaError_t launch_check_setup(int rows, int n, const CheckSteps& cj, const int* status, const int* kbreak, const int* l_in,
                               const int* err, int* k_out, int* l_out, int* status_out, int* kbreak_out, int* err_out,
                               cudaStream_t st) {
  k_check_setup<<<1, 128, 0, st>>>(rows, n, cj, status, kbreak, l_in, err, k_out, l_out, status_out, kbreak_out, err_out);
  return cudaGetLastError();
}

size_t rh_scratch_bytes(int nmat, int arith, bool dense) {
  const size_t it = sizeof(double2) * (size_t)kMaxL * kMaxL, col = sizeof(float4) * 2 * (size_t)kMaxL * kColThreads;
  static_assert(sizeof(float4) * 2 * kMaxL * kColThreads >= sizeof(double2) * kMaxL * kMaxL, "a slot holds either");
  return arith == OV_INNER_DF64 && !dense ? std::min(nmat, kRhWave) * col : nmat * it;
}

static size_t inner_smem(int k) { return (size_t)13 * k * sizeof(double2) + 32 * sizeof(double) + k + 16; }
static size_t inner_smem_real(int k) { return (size_t)13 * k * sizeof(float2) + 32 * sizeof(double) + k + 16; }

cudaError_t run_inner(int count, const int* k_dev, const int* l_dev, int hermitian, const double2* alp,
                      const double2* bet, const double2* gam, const double* nv, int ldc, InnerWork& w,
                      double rh_tol, int rh_maxit, int inner_dl, double2* c, int ldo, void* cacc, int prec,
                      double* est_inner,
                      const double2* cprev, int ldp, const int* kprev_dev, double* est_outer, int* rh_status,
                      int* rh_iters, int phase, cudaStream_t st) {
  cudaError_t e;
  if (phase != 2) {
    const size_t sm = inner_smem(w.ld);  // float pairs take the bytes of the doubles they replace
    if (w.arith == OV_INNER_DF64 && hermitian) {
      const size_t smr = inner_smem_real(w.ld);
      e = cudaFuncSetAttribute(k_inner_df<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smr);
      if (e != cudaSuccess) return e;
      k_inner_df<false><<<count, kSideLanes, smr, st>>>(k_dev, l_dev, alp, bet, gam, ldc, w);
    } else if (w.arith == OV_INNER_DF64) {
      e = cudaFuncSetAttribute(k_inner_df<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
      k_inner_df<true><<<count, 2 * kSideLanes, sm, st>>>(k_dev, l_dev, alp, bet, gam, ldc, w);
    } else {
      e = cudaFuncSetAttribute(k_inner, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
      k_inner<<<count, kInnerThreads, sm, st>>>(k_dev, l_dev, hermitian, alp, bet, gam, ldc, w);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  // phase 0: both Roberts-Higham sets (the matrices and their leading l - dl blocks);
  // phase 1: the matrices only (no inner estimate); phase 2: only the leading blocks
  // of the matrices left by a phase-1 call (the inner estimate on request)
  const int mid0 = phase == 2 ? count : 0;
  const int nmat = phase == 0 ? 2 * count : count;
  const size_t esz = hermitian ? sizeof(double) : sizeof(double2);
  // matrix + column buffer (which also holds the 64-double reduction scratch)
  const size_t rsm = (size_t)kMaxL * kMaxL * esz + std::max<size_t>(kMaxL * esz, 512);
  if (w.arith == OV_INNER_DF64) {
    if (hermitian) e = cudaFuncSetAttribute(k_rh_df<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    else e = cudaFuncSetAttribute(k_rh_df<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    if (e != cudaSuccess) return e;
    for (int m0 = mid0; m0 < mid0 + nmat; m0 += kRhWave) {
      const int nm = std::min(kRhWave, mid0 + nmat - m0);
      k_rh_col<<<nm, kColThreads, 0, st>>>(count, hermitian, w, inner_dl, rh_tol, rh_maxit, m0, w.rh_scale);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      // the matrices it left (in the same scratch); float pairs take the bytes of the double
      // elements they replace
      if (hermitian) k_rh_df<false><<<nm, 1024, rsm, st>>>(count, 0, nullptr, w, inner_dl, rh_tol, rh_maxit, m0, w.rh_scale);
      else k_rh_df<true><<<nm, 1024, rsm, st>>>(count, 0, nullptr, w, inner_dl, rh_tol, rh_maxit, m0, w.rh_scale);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  } else if (hermitian) {
    e = cudaFuncSetAttribute(k_rh<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    if (e != cudaSuccess) return e;
    k_rh<false><<<nmat, 1024, rsm, st>>>(count, 0, nullptr, w, inner_dl, rh_tol, rh_maxit, mid0);
  } else {
    e = cudaFuncSetAttribute(k_rh<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    if (e != cudaSuccess) return e;
    k_rh<true><<<nmat, 1024, rsm, st>>>(count, 0, nullptr, w, inner_dl, rh_tol, rh_maxit, mid0);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_combine<<<count * kCombineCtas, kCombineThreads, 0, st>>>(count, k_dev, l_dev, w, inner_dl, c, ldo, cacc, nv, ldc,
                                                              prec, w.cnorm, est_inner, rh_status, rh_iters, phase != 1);
  if ((e = cudaGetLastError()) != cudaSuccess || !est_outer) return e;
  k_estimate<<<count, kCombineThreads, 0, st>>>(k_dev, w, c, ldo, w.cnorm, rh_status, cprev, ldp, kprev_dev, est_outer);
  return cudaGetLastError();
}

cudaError_t run_rh_dense(int count, int m, const double2* T, double2* S, int* iters, int* ok, double rh_tol,
                         int rh_maxit, InnerWork& w, cudaStream_t st) {
  const size_t rsm = (size_t)m * m * sizeof(double2) + std::max<size_t>(m * sizeof(double2), 512);
  cudaError_t e;
  if (w.arith == OV_INNER_DF64) {
    e = cudaFuncSetAttribute(k_rh_df<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    if (e != cudaSuccess) return e;
    k_rh_df<true><<<count, 1024, rsm, st>>>(count, m, T, w, 0, rh_tol, rh_maxit, 0, 0);
  } else {
    e = cudaFuncSetAttribute(k_rh<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm);
    if (e != cudaSuccess) return e;
    k_rh<true><<<count, 1024, rsm, st>>>(count, m, T, w, 0, rh_tol, rh_maxit, 0);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int i = 0; i < count; ++i) {
    e = cudaMemcpy2DAsync(S + (size_t)i * m * m, sizeof(double2) * m * m, w.S + (size_t)i * kMaxL * kMaxL,
                          sizeof(double2) * m * m, sizeof(double2) * m * m, 1, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  e = cudaMemcpyAsync(iters, w.rh_its, sizeof(int) * count, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  return cudaMemcpyAsync(ok, w.rh_ok, sizeof(int) * count, cudaMemcpyDeviceToDevice, st);
}

}  // namespace ov

// Outer Krylov level: the gamma5 Wilson-Dirac stencil fused with the Lanczos /
// two-sided Lanczos recurrences, vector updates with fixed-order reductions, and
// recombination of the result (Sec. 2, Eq. (approximation); Sec. 3, Eq. (nested)).
//
// Layout: an internal spinor field is [rhs][12][V] of the precision's storage type
// (component c = 3*spin + colour, site fastest), so a warp reads consecutive sites of
// one component (coalesced). Links are [4][9][V] (nu, a*3+b, site) with the
// antiperiodic t-boundary sign folded into U_t on the last time slice; the double-float
// mode keeps a second plane of low words 36 V elements further on.
//
// Precisions: FP64; FP32 (float vectors and links, double-float reductions); double-float
// (vectors and links as float pairs, compensated hop sums); and the relaxed double-float
// steps (the same storage and recurrence with the hop sum in float on the high words).
//
// Reductions: every block writes its partial sums (double) to a partials array; the
// last block of each right-hand side (atomic ticket, no spin-wait) adds the partials in
// a fixed order and writes the Krylov coefficient. Where whole runs of steps go in one
// launch (k_steps, small lattices) a right-hand side's blocks wait for one another instead,
// with a bound, and each adds the partials in the same order. Results are therefore bitwise
// reproducible run to run with the same kernels and block size (the first apply of a handle
// tunes them, and forms the source's norm with the block size it starts from).
#include "ov_internal.h"
#include "ov_types.cuh"

namespace ov {

int num_site_blocks(const Geometry& g, int bs) { return (g.V + bs - 1) / bs; }

size_t vec_elem_bytes(int prec) {
  return prec == OV_PREC_FP32 ? sizeof(float2) : (prec == OV_PREC_FP64 ? sizeof(double2) : sizeof(float4));
}
size_t acc_elem_bytes(int prec) { return prec == OV_PREC_FP64 ? sizeof(double2) : sizeof(float4); }

template <class P> struct AccOf;
template <> struct AccOf<PrecF64> { using A = double; using st = double2; };
template <> struct AccOf<PrecF32> { using A = df64; using st = float4; };
template <> struct AccOf<PrecDF64> { using A = df64; using st = float4; };
template <> struct AccOf<PrecDF64R> { using A = df64; using st = float4; };

__device__ __forceinline__ cx<double> ld_acc(const double2* p) { double2 v = *p; return {v.x, v.y}; }
__device__ __forceinline__ cx<df64> ld_acc(const float4* p) { float4 v = *p; return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ void st_acc(double2* p, cx<double> a) { *p = make_double2(a.re, a.im); }
__device__ __forceinline__ void st_acc(float4* p, cx<df64> a) { *p = make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }

// p - a v in one fused step per component (double-float: both products exact, one
// renormalisation)
template <class R> __device__ __forceinline__ cx<R> csubmul(cx<R> p, cx<R> a, cx<R> v) { return p - cmul(a, v); }
__device__ __forceinline__ cx<df64> csubmul(cx<df64> p, cx<df64> a, cx<df64> v) {
  return {df_axpy2(p.re, -a.re, v.re, a.im, v.im), df_axpy2(p.im, -a.re, v.im, -a.im, v.re)};
}
// acc += |t|^2
__device__ __forceinline__ void acc_norm(double& acc, cx<double> t) { acc = fma(t.re, t.re, fma(t.im, t.im, acc)); }
__device__ __forceinline__ void acc_norm(df64& acc, cx<float> t) { acc = df_axpy2(acc, t.re, t.re, t.im, t.im); }
__device__ __forceinline__ void acc_norm(df64& acc, cx<df64> t) { acc = df_axpy2(acc, t.re, t.re, t.im, t.im); }
// a norm that only feeds a threshold test (the serious-breakdown test of two-sided
// Lanczos): float accumulation of the high words, double in the FP64 mode
__device__ __forceinline__ void acc_norm_lo(double& acc, cx<double> t) { acc_norm(acc, t); }
__device__ __forceinline__ void acc_norm_lo(float& acc, cx<float> t) { acc = fmaf(t.re, t.re, fmaf(t.im, t.im, acc)); }
__device__ __forceinline__ void acc_norm_lo(float& acc, cx<df64> t) {
  acc = fmaf(t.re.hi, t.re.hi, fmaf(t.im.hi, t.im.hi, acc));
}
template <class A> struct NormLo { using T = float; };
template <> struct NormLo<double> { using T = double; };
__device__ __forceinline__ double to_acc(double a, double) { return a; }
__device__ __forceinline__ df64 to_acc(float a, df64) { return {a, 0.f}; }

// accumulator += c * v  (c in accumulator type, v in vector type)
__device__ __forceinline__ void acc_axpy(cx<double>& y, cx<double> c, cx<double> v) { y = y + cmul(c, v); }
__device__ __forceinline__ void acc_axpy(cx<df64>& y, cx<df64> c, cx<float> v) { y = y + lcmul<df64, float>(v, c); }
__device__ __forceinline__ void acc_axpy(cx<df64>& y, cx<df64> c, cx<df64> v) { y = y + cmul(c, v); }

__device__ __forceinline__ cx<double> acc_to_cd(cx<double> a) { return a; }
__device__ __forceinline__ cx<double> acc_to_cd(cx<df64> a) { return {df_to_double(a.re), df_to_double(a.im)}; }
__device__ __forceinline__ cx<double> vec_to_cd(cx<double> a) { return a; }
__device__ __forceinline__ cx<double> vec_to_cd(cx<float> a) { return {(double)a.re, (double)a.im}; }
__device__ __forceinline__ cx<double> vec_to_cd(cx<df64> a) { return {df_to_double(a.re), df_to_double(a.im)}; }

template <class R> __device__ __forceinline__ cx<R> cd_to(double re, double im) {
  return {from_double<R>(re), from_double<R>(im)};
}

void split_const(double d, float hl[2]) {
  hl[0] = (float)d;
  hl[1] = (float)(d - (double)hl[0]);
}
// a constant from its double value and its host-side float split (no device FP64 work)
__device__ __forceinline__ double hconst(double, double d, const float*) { return d; }
__device__ __forceinline__ float hconst(float, double, const float* hl) { return hl[0]; }
__device__ __forceinline__ df64 hconst(df64, double, const float* hl) { return {hl[0], hl[1]}; }

// step scalars: slot q of RHS r
template <class P>
__device__ __forceinline__ cx<typename P::R> ld_scal(const void* scal, int r, int q) {
  return ld_vec((const typename P::vec_t*)scal + (size_t)r * 8 + q);
}
template <class P>
__device__ __forceinline__ void st_scal(void* scal, int r, int q, double re, double im) {
  st_vec((typename P::vec_t*)scal + (size_t)r * 8 + q, cd_to<typename P::R>(re, im));
}
// The scalars are formed by one warp, a quotient a lane: a double division is a chain of dozens
// of instructions on a pipe that gives two lanes a cycle, and one thread doing a step's ~20
// divisions and roots in turn held up the next kernel.
__device__ __forceinline__ double bcast(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
// scalars of step j from its coefficients nv_j, gamma_j, nw_j, beta_j and the previous
// normalisations nv_{j-1}, nw_{j-1} (run by a warp; the arguments are the same in every lane):
//   1/nv_j, gamma_j/nv_{j-1}, 1/conj(nw_j), conj(beta_j)/conj(nw_{j-1})
template <class P>
__device__ __forceinline__ void set_step_scal(void* scal, int r, double nv, double2 gam, double2 nw, double2 bet,
                                              double nvp, double2 nwp) {
  const int lane = threadIdx.x & 31;
  const double den = nw.x * nw.x + nw.y * nw.y;  // 1/conj(nw) = nw/|nw|^2
  // conj(beta)/conj(nwp) = conj(beta/nwp), beta/nwp = beta conj(nwp)/|nwp|^2
  const double dp = nwp.x * nwp.x + nwp.y * nwp.y;
  const double num = lane == 0 ? 1.0 : lane == 2 ? gam.x : lane == 3 ? gam.y : lane == 4 ? nw.x : lane == 5 ? nw.y
                     : lane == 6 ? bet.x * nwp.x + bet.y * nwp.y : bet.y * nwp.x - bet.x * nwp.y;
  const double dn = lane == 0 ? nv : lane < 4 ? nvp : lane < 6 ? den : dp;
  const double q = lane == 1 ? 0.0 : lane < 8 ? num / dn : 0.0;
  const double im = __shfl_down_sync(0xffffffffu, q, 1);
  if (lane < 8 && !(lane & 1)) st_scal<P>(scal, r, lane >> 1, q, lane == 6 ? -im : im);
}

// ------------------------------------------------------------ block reductions
// Each thread passes its values; the block's sums go to partials[(part0 + bx)*4 + q]
// (part0: the problem's first slot, bx: the block's index within the problem, so the
// slots do not depend on the launch order of the blocks). Returns true in the last block
// to finish for this problem, where tot[] (valid in warp 0) holds the fixed-order total
// over all its blocks.
// The block's per-warp sums (thread 0 adds them in warp order).
template <int NQ, int BS>
__device__ __forceinline__ void block_sums(const double (&v)[NQ], double (&bsum)[NQ]) {
  __shared__ double sred[BS / 32][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double w = warp_sum(v[q]);
    if (lane == 0) sred[warp][q] = w;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double s = 0.0;
      for (int w = 0; w < BS / 32; ++w) s += sred[w][q];
      bsum[q] = s;
    }
  }
}
// Double-float values: warp sums and the sum over warps stay in float pairs (float
// pipes); thread 0 converts the block's sums to double once.
template <int NQ, int BS>
__device__ __forceinline__ void block_sums(const df64 (&v)[NQ], double (&bsum)[NQ]) {
  __shared__ float2 sdf[BS / 32][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const df64 w = warp_sum(v[q]);
    if (lane == 0) sdf[warp][q] = make_float2(w.hi, w.lo);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      df64 s = df_zero();
      for (int w = 0; w < BS / 32; ++w) s = s + df64{sdf[w][q].x, sdf[w][q].y};
      bsum[q] = df_to_double(s);
    }
  }
}

template <int NQ, int BS, class T>
__device__ __forceinline__ bool reduce_last(T (&v)[NQ], double* partials, unsigned* counters, int r, int part0,
                                            int bx, int nblk, double (&tot)[NQ]) {
  __shared__ double sred[BS / 32][4];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double bsum[NQ];
  block_sums<NQ, BS>(v, bsum);
  if (tid == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) partials[(size_t)(part0 + bx) * 4 + q] = bsum[q];
    __threadfence();
    unsigned prev = atomicAdd(&counters[r], 1u);
    s_last = (prev == (unsigned)(nblk - 1));
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  // the warps that have partials to add (the double pipe serves a warp's instruction in 16
  // cycles: idle warps adding zeros would hold up the others)
  const int nw = min(BS / 32, (nblk + 31) / 32);
  if (warp < nw) {
    double loc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) loc[q] = 0.0;
    for (int b = tid; b < nblk; b += BS) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) loc[q] += __ldcg(&partials[(size_t)(part0 + b) * 4 + q]);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double w = warp_sum(loc[q]);
      if (lane == 0) sred[warp][q] = w;
    }
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double s = 0.0;
      for (int w = 0; w < nw; ++w) s += sred[w][q];
      tot[q] = s;
    }
    if (lane == 0) counters[r] = 0u;
  }
  return true;
}

// the site of this thread: problem r (from the block map), its descriptor, block within it
struct SiteRef {
  int r, bx, s;
  bool active;
  const ProbDesc* d;
};
// rev = true: the block map walked backwards (the vector update), so that an update starts
// where the preceding step ended and the next step where the update ended: the tail of what
// one kernel wrote is still in L2 when the next kernel reads it first
template <int BS, bool rev = false>
__device__ __forceinline__ SiteRef site_ref(const Batch& b) {
  const int2 m = __ldg(&b.blk_map[rev ? b.nblocks - 1 - (int)blockIdx.x : (int)blockIdx.x]);
  const int r = m.x;
  const ProbDesc* d = &b.desc[r];
  const int bx = m.y;
  const int s = bx * BS + threadIdx.x;
  return {r, bx, s, s < d->g.V, d};
}


// ------------------------------------------------------------ canonical buffers
// The canonical layout keeps a site's twelve numbers together (192 bytes), a warp's sites in
// one run. Read or written thread by thread, an instruction touches 32 places 192 bytes apart
// (12 x 16^4 in float: pack 73 us, unpack 86 us for 226 MB each); a warp moves them through
// shared memory instead, sixteen sites at a time, in 512-byte pieces (pack 55 us; the matvec
// writes its result this way itself, 110 -> 112 us, without a pass to unpack it).
constexpr int kCanonPitch = 13;  // of a site in shared memory: odd, so that lanes meet no bank twice
template <int BS>
struct CanonSmem {
  double2 v[BS / 32][16 * kCanonPitch];
};
// z = the numbers of the lane's site; base: the problem's canonical entries, w0: the warp's
// first site (whole warps call)
__device__ __forceinline__ void canon_load(const double2* __restrict__ base, int V, int w0, double2* sm, double2 (&z)[12]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int s0 = w0 + 16 * half, n = min(max(V - s0, 0), 16) * 12;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int e = lane + 32 * q;
      if (e < n) sm[e / 12 * kCanonPitch + e % 12] = base[(size_t)s0 * 12 + e];
    }
    __syncwarp();
    if ((lane >> 4) == half)
#pragma unroll
      for (int k = 0; k < 12; ++k) z[k] = sm[(lane & 15) * kCanonPitch + k];
  }
}
__device__ __forceinline__ void canon_store(double2* base, int V, int w0, double2* sm, const double2 (&z)[12]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int s0 = w0 + 16 * half, n = min(max(V - s0, 0), 16) * 12;
    __syncwarp();
    if ((lane >> 4) == half)
#pragma unroll
      for (int k = 0; k < 12; ++k) sm[(lane & 15) * kCanonPitch + k] = z[k];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int e = lane + 32 * q;
      if (e < n) base[(size_t)s0 * 12 + e] = sm[e / 12 * kCanonPitch + e % 12];
    }
  }
}

template <class P, int BS>
__global__ void __launch_bounds__(BS) k_pack(Batch bt, const double2* __restrict__ x, typename P::vec_t* xi,
                                                 typename P::vec_t* xi2, Coefs c, double* partials,
                                                 unsigned* counters, int want_norm, void* scal) {
  using R = typename P::R;
  __shared__ CanonSmem<BS> sm;
  const SiteRef sr = site_ref<BS>(bt);
  const int s = sr.s, r = sr.r;
  const int V = sr.d->g.V;
  const size_t voff = sr.d->voff;
  double2 z[12];
  canon_load(x + voff, V, s - (int)(threadIdx.x & 31), sm.v[threadIdx.x >> 5], z);
  double n2 = 0.0;
  if (sr.active) {
    typename P::vec_t* dst = xi + voff + s;
    typename P::vec_t* dst2 = xi2 ? xi2 + voff + s : nullptr;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      st_vec(dst + (size_t)k * V, cd_to<R>(z[k].x, z[k].y));
      if (dst2) st_vec(dst2 + (size_t)k * V, cd_to<R>(z[k].x, z[k].y));
    }
    if (want_norm)
#pragma unroll
      for (int k = 0; k < 12; ++k) n2 = fma(z[k].x, z[k].x, fma(z[k].y, z[k].y, n2));
  }
  if (!want_norm) return;
  double v[1] = {n2}, tot[1];
  if (reduce_last<1, BS>(v, partials, counters, r, sr.d->block0, sr.bx, sr.d->nblk, tot) && threadIdx.x < 32) {
    const double nrm = sqrt(tot[0]), n1 = nrm > 0.0 ? nrm : 1.0;
    const double2 zero = make_double2(0.0, 0.0), w1 = make_double2(n1, 0.0);
    if (threadIdx.x == 0) {
      const size_t o = (size_t)r * c.ld + 1;
      c.nv[o] = n1;
      c.nw[o] = w1;
      c.bet[o] = zero;
      c.gam[o] = zero;
      c.status[r] = nrm > 0.0 ? kStOK : kStZero;
      c.kbreak[r] = 0;
    }
    if (scal) set_step_scal<P>(scal, r, n1, zero, w1, zero, 1.0, make_double2(1.0, 0.0));
  }
}

// ------------------------------------------------------------ the stencil
// Spin structure in the DeGrand-Rossi basis: gamma_nu = [[0, B],[B^dag, 0]] in 2x2 spin
// blocks with B_x = [[0,i],[i,0]], B_y = [[0,-1],[1,0]], B_z = [[i,0],[0,-i]], B_t = 1.
// Forward hop (1 - gamma): h = psi_u - B psi_l, result (U h, -B^dag U h).
// Backward hop (1 + gamma): h = psi_u + B psi_l, result (U^dag h, +B^dag U^dag h).
// Every entry of B and B^dag is a power of i, so (B psi_l)_s = i^q psi_{src}: the tables
// hold, per direction, the source spin and the exponent q of both components of
// B psi_l (sources are the lower spins 2, 3) and of B^dag g (sources are 0, 1).
// The eight hops run through one loop body (the double-float body is large; unrolling
// the hops overflowed the instruction cache).
__constant__ int c_bsrc[4][2] = {{3, 2}, {3, 2}, {2, 3}, {2, 3}};
__constant__ int c_bph[4][2] = {{1, 1}, {2, 0}, {1, 3}, {0, 0}};
__constant__ int c_dsrc[4][2] = {{1, 0}, {1, 0}, {0, 1}, {0, 1}};
__constant__ int c_dph[4][2] = {{3, 3}, {0, 2}, {3, 1}, {0, 0}};

__device__ __forceinline__ double rneg(double a, bool n) { return n ? -a : a; }
__device__ __forceinline__ float rneg(float a, bool n) { return n ? -a : a; }
__device__ __forceinline__ df64 rneg(df64 a, bool n) { return n ? df64{-a.hi, -a.lo} : a; }
// i^q z
template <class R> __device__ __forceinline__ cx<R> rot(cx<R> z, int q) {
  const bool sw = q & 1;
  cx<R> r = {sw ? z.im : z.re, sw ? z.re : z.im};
  return {rneg(r.re, q == 1 || q == 2), rneg(r.im, q >= 2)};
}
// cos(q pi/2), sin(q pi/2) and z + i^q w with them (see hopping_plain)
template <class R> __device__ __forceinline__ R phase_c(int q) { return R((q == 0) - (q == 2)); }
template <class R> __device__ __forceinline__ R phase_s(int q) { return R((q == 1) - (q == 3)); }
__device__ __forceinline__ cx<float> add_rot(cx<float> z, cx<float> w, float c, float s) {
  return {__fmaf_rn(-s, w.im, __fmaf_rn(c, w.re, z.re)), __fmaf_rn(s, w.re, __fmaf_rn(c, w.im, z.im))};
}
__device__ __forceinline__ cx<double> add_rot(cx<double> z, cx<double> w, double c, double s) {
  return {__fma_rn(-s, w.im, __fma_rn(c, w.re, z.re)), __fma_rn(s, w.re, __fma_rn(c, w.im, z.im))};
}
__device__ __forceinline__ cx<double> lconj(cx<double> u, bool c) { return {u.re, c ? -u.im : u.im}; }
__device__ __forceinline__ cx<float> lconj(cx<float> u, bool c) { return {u.re, c ? -u.im : u.im}; }

__device__ __forceinline__ void site_coords(const Geometry& g, int s, int& x, int& y, int& z, int& t) {
  x = s % g.Lx;
  int q = s / g.Lx;
  y = q % g.Ly;
  q /= g.Ly;
  z = q % g.Lz;
  t = q / g.Lz;
}

__device__ __forceinline__ void hopping_df(cx<df64> (&accn)[12], const float4* __restrict__ src,
                                           const float2* __restrict__ links, const Geometry& g, int s,
                                           const int (&xc)[4], df64 ef, df64 eb);

// vector element for the hopping sum: as stored, or the high words of a float pair
__device__ __forceinline__ cx<double> ld_hop(const double2* p) { return ld_vec(p); }
__device__ __forceinline__ cx<float> ld_hop(const float2* p) { return ld_vec(p); }
__device__ __forceinline__ cx<float> ld_hop(const float4* p) {
  const float2 v = *(const float2*)p;
  return {v.x, v.y};
}

// acc = sum over the 8 hops of the hopping term for source `src` at site s in arithmetic
// R with links of type L; ef / eb multiply the forward / backward t hops (e^{+-mu}).
template <class R, class L, class VT, class LT>
__device__ __forceinline__ void hopping_plain(cx<R> (&acc)[12], const VT* __restrict__ src,
                                              const LT* __restrict__ links, const Geometry& g, int s,
                                              const int (&xc)[4], R ef, R eb) {
  const int V = g.V;
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = czero<R>();
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int nu = hop >> 1;
    const bool fwd = (hop & 1) == 0;
    const int Ln = nu == 0 ? g.Lx : (nu == 1 ? g.Ly : (nu == 2 ? g.Lz : g.Lt));
    const int st = nu == 0 ? 1 : (nu == 1 ? g.Lx : (nu == 2 ? g.Lx * g.Ly : g.Lx * g.Ly * g.Lz));
    const int c = xc[0] * (nu == 0) + xc[1] * (nu == 1) + xc[2] * (nu == 2) + xc[3] * (nu == 3);
    const int sn = fwd ? (c == Ln - 1 ? s - (Ln - 1) * st : s + st) : (c == 0 ? s + (Ln - 1) * st : s - st);
    const int ls = fwd ? s : sn;
    // link: U_nu(s) forward, U_nu(s - nu)^dag backward
    cx<L> u[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int idx = fwd ? e : (e % 3) * 3 + e / 3;
      u[e] = lconj(ld_link(links + (size_t)(nu * 9 + idx) * V + ls), !fwd);
    }
    const int b0s = c_bsrc[nu][0], b1s = c_bsrc[nu][1];
    const int b0q = (c_bph[nu][0] + (fwd ? 2 : 0)) & 3, b1q = (c_bph[nu][1] + (fwd ? 2 : 0)) & 3;
    // i^q as (c, s) in {0, +-1}: z + i^q w = (z.re + c w.re - s w.im, z.im + c w.im + s w.re)
    // by fused multiply-adds; one of c, s is zero, so each component is rounded once, as a
    // plain addition of the rotated term would be
    const R c0 = phase_c<R>(b0q), s0 = phase_s<R>(b0q), c1 = phase_c<R>(b1q), s1 = phase_s<R>(b1q);
    cx<R> h0[3], h1[3];
#pragma unroll
    for (int col = 0; col < 3; ++col) {
      const cx<R> p0 = ld_hop(src + (size_t)(0 + col) * V + sn);
      const cx<R> p1 = ld_hop(src + (size_t)(3 + col) * V + sn);
      const cx<R> q0 = ld_hop(src + (size_t)(3 * b0s + col) * V + sn);
      const cx<R> q1 = ld_hop(src + (size_t)(3 * b1s + col) * V + sn);
      h0[col] = add_rot(p0, q0, c0, s0);
      h1[col] = add_rot(p1, q1, c1, s1);
    }
    const bool sc = nu == 3;
    const R fac = fwd ? ef : eb;
    const int d0s = c_dsrc[nu][0], d1s = c_dsrc[nu][1];
    const int d0q = (c_dph[nu][0] + (fwd ? 2 : 0)) & 3, d1q = (c_dph[nu][1] + (fwd ? 2 : 0)) & 3;
    const R e0 = phase_c<R>(d0q), f0 = phase_s<R>(d0q), e1 = phase_c<R>(d1q), f1 = phase_s<R>(d1q);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cx<R> g0 = lcmul<R, L>(u[a * 3 + 0], h0[0]) + lcmul<R, L>(u[a * 3 + 1], h0[1]) + lcmul<R, L>(u[a * 3 + 2], h0[2]);
      cx<R> g1 = lcmul<R, L>(u[a * 3 + 0], h1[0]) + lcmul<R, L>(u[a * 3 + 1], h1[1]) + lcmul<R, L>(u[a * 3 + 2], h1[2]);
      if (sc) {
        g0 = cscale(g0, fac);
        g1 = cscale(g1, fac);
      }
      acc[0 + a] = acc[0 + a] + g0;
      acc[3 + a] = acc[3 + a] + g1;
      acc[6 + a] = add_rot(acc[6 + a], d0s == 0 ? g0 : g1, e0, f0);
      acc[9 + a] = add_rot(acc[9 + a], d1s == 0 ? g0 : g1, e1, f1);
    }
  }
}

template <class P>
__device__ __forceinline__ void hopping(cx<typename P::R> (&acc)[12], const typename P::vec_t* __restrict__ src,
                                        const typename P::link_t* __restrict__ links, const Geometry& g, int s,
                                        const int (&xc)[4], typename P::R ef, typename P::R eb) {
  if constexpr (P::id == PrecDF64::id) {
    hopping_df(acc, src, links, g, s, xc, ef, eb);
  } else if constexpr (P::id == PrecDF64R::id) {
    cx<float> af[12];
    hopping_plain<float, float>(af, src, links, g, s, xc, ef.hi, eb.hi);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = {{af[k].re, 0.f}, {af[k].im, 0.f}};
  } else {
    hopping_plain<typename P::R, typename P::L>(acc, src, links, g, s, xc, ef, eb);
  }
}

// ---- double-float hopping in compensated form -------------------------------------------
// The links are double-float too: a plane of float hi parts and, 36 V elements further on,
// a plane of lo parts (|lo| <= 2^-24 |hi|). The products U_ab h_b are summed as in the
// compensated dot product of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26 (2005), "Dot2"):
// the product of U.hi with h.hi is exact as (p, e) (p = U.hi*h.hi, e = fma(U.hi, h.hi, -p)),
// U.hi*h.lo is folded into e with one FMA, the running sum takes p through TwoSum, and all
// error terms are accumulated in the low word without renormalising; U.lo*h.hi, a term of
// relative size 2^-24, is added to the low word in plain float arithmetic once per row
// (the lo links are loaded with the hi links at the start of the hop).
// Sums are renormalised once, when the hopping term is complete. Error: a few units of
// 2^-48 relative to the summed magnitudes, as for the normalised pair arithmetic.
struct dfu {  // unnormalised pair: value hi + lo
  float hi, lo;
};
__device__ __forceinline__ void madd_u(dfu& acc, float u, df64 h) {
  const float p = __fmul_rn(u, h.hi);
  float e = __fmaf_rn(u, h.hi, -p);
  e = __fmaf_rn(u, h.lo, e);
  const float s = __fadd_rn(acc.hi, p);
  const float bb = __fsub_rn(s, acc.hi);
  const float err = __fadd_rn(__fsub_rn(acc.hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  acc.hi = s;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(e, err));
}
// acc = u h, exactly as (p, e)
__device__ __forceinline__ void set_u(dfu& acc, float u, df64 h) {
  const float p = __fmul_rn(u, h.hi);
  float e = __fmaf_rn(u, h.hi, -p);
  acc = {p, __fmaf_rn(u, h.lo, e)};
}
__device__ __forceinline__ dfu add_u(dfu a, dfu b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return {s, __fadd_rn(__fadd_rn(a.lo, b.lo), err)};
}
__device__ __forceinline__ dfu neg_u(dfu a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ df64 norm_u(dfu a) { return df_fast_two_sum(a.hi, a.lo); }
__device__ __forceinline__ dfu to_u(df64 a) { return {a.hi, a.lo}; }
struct cxu {
  dfu re, im;
};
__device__ __forceinline__ cxu cadd_u(cxu a, cxu b) { return {add_u(a.re, b.re), add_u(a.im, b.im)}; }
// i^q z
__device__ __forceinline__ cxu rot_u(cxu z, int q) {
  const bool sw = q & 1;
  cxu r = {sw ? z.im : z.re, sw ? z.re : z.im};
  const bool nre = q == 1 || q == 2, nim = q >= 2;
  return {nre ? neg_u(r.re) : r.re, nim ? neg_u(r.im) : r.im};
}

// One thread a site: the real and the imaginary part of every number are the two halves of a
// packed register, as they lie in memory (hi pair, lo pair), so that an instruction serves both
// (two passes of the float pipe, one issue slot: the sums are then bound by the pipe, ~1100 of
// its cycles a hop and side, more than by issue slots). The operations and their order are those
// of the scalar form (another order moved results with relaxed steps by 1.6e-9). Strict step of
// 12 x 16^4 0.843 -> 0.756 ms; a column of the link at a time instead of all loads first 0.814.
struct pcx {  // unnormalised complex pair: hi + lo
  f32x2 hi, lo;
};
__device__ __forceinline__ pcx ld_pcx(const float4* p) {
  const ulonglong2 v = *(const ulonglong2*)p;
  return {v.x, v.y};
}
__device__ __forceinline__ pcx add_p(pcx a, pcx b) {
  const f32x2 s = add2(a.hi, b.hi), bb = sub2(s, a.hi);
  const f32x2 err = add2(sub2(a.hi, sub2(s, bb)), sub2(b.hi, bb));
  return {s, add2(add2(a.lo, b.lo), err)};
}
// acc = u h and acc += u h (u: one link word in both halves of the register, or (-u, u))
__device__ __forceinline__ void set_p(pcx& acc, f32x2 u, pcx h) {
  acc.hi = mul2(u, h.hi);
  acc.lo = fma2(u, h.lo, fma2(u, h.hi, neg2(acc.hi)));
}
__device__ __forceinline__ void madd_p(pcx& acc, f32x2 u, pcx h) {
  const f32x2 p = mul2(u, h.hi);
  const f32x2 e = fma2(u, h.lo, fma2(u, h.hi, neg2(p)));
  const f32x2 s = add2(acc.hi, p), bb = sub2(s, acc.hi);
  const f32x2 err = add2(sub2(acc.hi, sub2(s, bb)), sub2(p, bb));
  acc.hi = s;
  acc.lo = add2(acc.lo, add2(e, err));
}
__device__ __forceinline__ f32x2 swap_p(f32x2 a) {
  const float2 v = upk(a);
  return pk(v.y, v.x);
}
// acc (+)= u h for the complex link u (hi words), c += ul h.hi for its lo words: the term of u.re,
// then that of u.im with (i h) = (-h.im, h.re) as (-u.im, u.im) times hs = (h.im, h.re)
template <bool SET>
__device__ __forceinline__ void cmadd_p(pcx& acc, f32x2& c, cx<float> u, cx<float> ul, pcx h, pcx hs) {
  if (SET) set_p(acc, pk(u.re, u.re), h);
  else madd_p(acc, pk(u.re, u.re), h);
  madd_p(acc, pk(-u.im, u.im), hs);
  c = fma2(pk(ul.re, ul.re), h.hi, fma2(pk(-ul.im, ul.im), hs.hi, c));
}
// i^q a, with the signs of the two halves as masks
struct Phase4 {
  bool sw;
  unsigned mre, mim;
};
__device__ __forceinline__ Phase4 phase_of(int q) {
  return {(q & 1) != 0, q == 1 || q == 2 ? 0x80000000u : 0u, q >= 2 ? 0x80000000u : 0u};
}
__device__ __forceinline__ f32x2 rot_p(f32x2 a, Phase4 f) {
  const float2 v = upk(a);
  const float x = f.sw ? v.y : v.x, y = f.sw ? v.x : v.y;
  return pk(__uint_as_float(__float_as_uint(x) ^ f.mre), __uint_as_float(__float_as_uint(y) ^ f.mim));
}
__device__ __forceinline__ pcx rot_p(pcx a, Phase4 f) { return {rot_p(a.hi, f), rot_p(a.lo, f)}; }
__device__ __forceinline__ cx<df64> norm_p(pcx a) {
  const float2 h = upk(a.hi), l = upk(a.lo);
  return {df_fast_two_sum(h.x, l.x), df_fast_two_sum(h.y, l.y)};
}

__device__ __forceinline__ void hopping_df(cx<df64> (&accn)[12], const float4* __restrict__ src,
                                           const float2* __restrict__ links, const Geometry& g, int s,
                                           const int (&xc)[4], df64 ef, df64 eb) {
  const int V = g.V;
  const float2* __restrict__ links_lo = links + (size_t)36 * V;
  pcx acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = {0ull, 0ull};
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int nu = hop >> 1;
    const bool fwd = (hop & 1) == 0;
    const int Ln = nu == 0 ? g.Lx : (nu == 1 ? g.Ly : (nu == 2 ? g.Lz : g.Lt));
    const int st = nu == 0 ? 1 : (nu == 1 ? g.Lx : (nu == 2 ? g.Lx * g.Ly : g.Lx * g.Ly * g.Lz));
    const int c = xc[0] * (nu == 0) + xc[1] * (nu == 1) + xc[2] * (nu == 2) + xc[3] * (nu == 3);
    const int sn = fwd ? (c == Ln - 1 ? s - (Ln - 1) * st : s + st) : (c == 0 ? s + (Ln - 1) * st : s - st);
    const int ls = fwd ? s : sn;
    cx<float> u[9], ulo[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const int idx = fwd ? e : (e % 3) * 3 + e / 3;
      u[e] = lconj(ld_link(links + (size_t)(nu * 9 + idx) * V + ls), !fwd);
      ulo[e] = lconj(ld_link(links_lo + (size_t)(nu * 9 + idx) * V + ls), !fwd);
    }
    const int b0s = c_bsrc[nu][0], b1s = c_bsrc[nu][1];
    const Phase4 b0f = phase_of((c_bph[nu][0] + (fwd ? 2 : 0)) & 3), b1f = phase_of((c_bph[nu][1] + (fwd ? 2 : 0)) & 3);
    pcx h0[3], h1[3];
#pragma unroll
    for (int col = 0; col < 3; ++col) {
      // projections, unnormalised (their low words only enter through FMAs below)
      h0[col] = add_p(ld_pcx(src + (size_t)(0 + col) * V + sn), rot_p(ld_pcx(src + (size_t)(3 * b0s + col) * V + sn), b0f));
      h1[col] = add_p(ld_pcx(src + (size_t)(3 + col) * V + sn), rot_p(ld_pcx(src + (size_t)(3 * b1s + col) * V + sn), b1f));
    }
    const bool sc = nu == 3;
    const df64 fac = fwd ? ef : eb;
    const int d0s = c_dsrc[nu][0], d1s = c_dsrc[nu][1];
    const Phase4 d0f = phase_of((c_dph[nu][0] + (fwd ? 2 : 0)) & 3), d1f = phase_of((c_dph[nu][1] + (fwd ? 2 : 0)) & 3);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      pcx g0, g1;
      f32x2 c0 = 0ull, c1 = 0ull;  // U.lo row a times h.hi
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const cx<float> uh = u[a * 3 + b], ul = ulo[a * 3 + b];
        const pcx s0 = {swap_p(h0[b].hi), swap_p(h0[b].lo)}, s1 = {swap_p(h1[b].hi), swap_p(h1[b].lo)};
        if (b == 0) {
          cmadd_p<true>(g0, c0, uh, ul, h0[b], s0);
          cmadd_p<true>(g1, c1, uh, ul, h1[b], s1);
        } else {
          cmadd_p<false>(g0, c0, uh, ul, h0[b], s0);
          cmadd_p<false>(g1, c1, uh, ul, h1[b], s1);
        }
      }
      g0.lo = add2(g0.lo, c0);
      g1.lo = add2(g1.lo, c1);
      if (sc) {
        const cx<df64> n0 = cscale(norm_p(g0), fac), n1 = cscale(norm_p(g1), fac);
        g0 = {pk(n0.re.hi, n0.im.hi), pk(n0.re.lo, n0.im.lo)};
        g1 = {pk(n1.re.hi, n1.im.hi), pk(n1.re.lo, n1.im.lo)};
      }
      acc[0 + a] = add_p(acc[0 + a], g0);
      acc[3 + a] = add_p(acc[3 + a], g1);
      acc[6 + a] = add_p(acc[6 + a], rot_p(d0s == 0 ? g0 : g1, d0f));
      acc[9 + a] = add_p(acc[9 + a], rot_p(d1s == 0 ? g0 : g1, d1f));
    }
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) accn[k] = norm_p(acc[k]);
}

// (gamma5 D psi)_k at the centre site from the hopping sum: mass*psi - hop/2, lower spins negated.
template <class R>
__device__ __forceinline__ cx<R> g5d(int k, cx<R> psi, cx<R> hk, R mass) {
  cx<R> d = cscale(psi, mass) - chalf(hk);
  return k >= 6 ? -d : d;
}
__device__ __forceinline__ cx<df64> g5d(int k, cx<df64> psi, cx<df64> hk, df64 mass) {
  const cx<df64> d = {df_axpy1(-df_half(hk.re), mass, psi.re), df_axpy1(-df_half(hk.im), mass, psi.im)};
  return k >= 6 ? -d : d;
}

// ---- the recurrence at one site: scalars real (RS, RC) or complex -----------------------
// In the recurrences 1/nv_j and beta_j are real, gamma_j and 1/conj(nw_j) complex: side v of
// two-sided Lanczos scales by a real and subtracts a complex multiple, side w the reverse,
// Lanczos has both real.
template <bool RS, class R>
__device__ __forceinline__ cx<R> smul(cx<R> s, cx<R> z) {
  return RS ? cscale(z, s.re) : cmul(s, z);
}
template <bool RS>
__device__ __forceinline__ cx<df64> smul(cx<df64> s, cx<df64> z) {
  if (RS) return {z.re * s.re, z.im * s.re};
  return {df_axpy2(df_zero(), s.re, z.re, -s.im, z.im), df_axpy2(df_zero(), s.re, z.im, s.im, z.re)};
}
// s q - c w
template <bool RS, bool RC, class R>
__device__ __forceinline__ cx<R> smulsub(cx<R> s, cx<R> q, cx<R> c, cx<R> w) {
  return smul<RS>(s, q) - smul<RC>(c, w);
}
template <bool RS, bool RC>
__device__ __forceinline__ cx<df64> smulsub(cx<df64> s, cx<df64> q, cx<df64> c, cx<df64> w) {
  if (RS && RC) return {df_axpy2(df_zero(), s.re, q.re, -c.re, w.re), df_axpy2(df_zero(), s.re, q.im, -c.re, w.im)};
  if (RS) return {df_axpy2(q.re * s.re, -c.re, w.re, c.im, w.im), df_axpy2(q.im * s.re, -c.re, w.im, -c.im, w.re)};
  if (RC)
    return {df_axpy2(-(w.re * c.re), s.re, q.re, -s.im, q.im), df_axpy2(-(w.im * c.re), s.re, q.im, s.im, q.re)};
  // both complex: each component one compensated four-term sum
  return {df_dot4(s.re, q.re, -s.im, q.im, -c.re, w.re, c.im, w.im),
          df_dot4(s.re, q.im, s.im, q.re, -c.re, w.im, -c.im, w.re)};
}
// out = scl (gamma5 D t_j) - cf t_{j-1} at one site, 12 components, with t_j the
// unnormalised current vector (psi) and t_{j-1} the previous one; the alpha partial: Lanczos
// t_j^dag out, two-sided side w: tw_j^dag p (p from side v); the finaliser divides by the
// normalisation
template <bool RS, bool RC, int DOT, class R, class VT, class AT>
__device__ __forceinline__ void step_site(const VT* src, const VT* prv, VT* out, const VT* pp, int V, int s,
                                          cx<R> scl, cx<R> cf, const cx<R> (&acc)[12], R mass, cx<AT>& dot) {
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const cx<R> psi = ld_vec(src + (size_t)k * V + s);
    const cx<R> ok = smulsub<RS, RC>(scl, g5d(k, psi, acc[k], mass), cf, ld_vec(prv + (size_t)k * V));
    st_vec(out + (size_t)k * V, ok);
    if (DOT == 1) acc_dot(dot, psi, ok);
    if (DOT == 2) acc_dot(dot, psi, ld_vec(pp + (size_t)k * V));
  }
}

// the step index and the step's vectors (device-side state or host fields): t_j, t_{j-1},
// the destination of t_{j+1}, and the same three on the w side
struct StepPtrs {
  int j;
  const void* tc;
  const void* tp;
  void* tn;
  const void* wc;
  const void* wp;
  void* wn;
};
__device__ __forceinline__ StepPtrs step_ptrs(const StepArgs& a) {
  if (!a.jdev) return {a.j, a.tc, a.tp, a.tn, nullptr, nullptr, nullptr};
  const int j = __ldcg(a.jdev);
  char* vr = (char*)a.vring;
  char* wr = (char*)a.wring;
  const size_t pb = a.pool_bytes;
  char* wc = wr + pb * (j & 1);
  char* wp = wr + pb * ((j - 1) & 1);
  if (a.slot_tab) {
    // stored basis: slot i holds t_{i+1}; t_0 is the zeroed ring slot 0
    const void* tp = j == 1 ? (const void*)vr : (const void*)a.slot_tab[j - 2];
    return {j, a.slot_tab[j - 1], tp, a.slot_tab[j], wc, wp, wp};
  }
  char* tc = vr + pb * (j & 1);
  char* tp = vr + pb * ((j - 1) & 1);
  return {j, tc, tp, tp, wc, wp, wp};
}

// Register caps of the step kernels (the warps they add hide the load latency at the start
// of each hop; measured at 16^4 with 12 right-hand sides): 128 registers a thread for the
// strict double-float step (16 warps an SM; its hop body fits, tighter caps spill hundreds
// of bytes and run slower), 85 for the relaxed step (24 warps; it fits in 80: 0.50 ->
// 0.46 ms) and 64 for the float step (32 warps, a few spilled words: 0.32 -> 0.27 ms).
// FP64 keeps the compiler's choice.
// Resident threads per SM each step kernel is compiled for (the register cap follows:
// 65536 / threads); overridable at build time to measure other splits.
#ifndef OV_STEP_THREADS_DF64
#define OV_STEP_THREADS_DF64 512
#endif
#ifndef OV_STEP_THREADS_DF64R
#define OV_STEP_THREADS_DF64R 768
#endif
#ifndef OV_STEP_THREADS_F32
#define OV_STEP_THREADS_F32 1024
#endif
template <class P, int BS>
constexpr int step_min_blocks() {
  constexpr int t = P::id == PrecDF64::id    ? OV_STEP_THREADS_DF64
                    : P::id == PrecDF64R::id ? OV_STEP_THREADS_DF64R
                    : P::id == PrecF32::id   ? OV_STEP_THREADS_F32
                                             : BS;
  return t / BS > 0 ? t / BS : 1;
}

// alpha_j from the total of its partial sums, and the update's scalars (one warp)
template <class P, int MODE>
__device__ __forceinline__ void finish_alpha(const StepArgs& a, int r, size_t co, const double (&tot)[2]) {
  const int lane = threadIdx.x & 31;
  const double nvj = a.c.nv[co];
  double ar, ai;
  double2 nw = a.c.nw[co];
  if (MODE == kModeLanczos) {
    ar = tot[0] / nvj;
    ai = 0.0;
    nw = make_double2(nvj, 0.0);
  } else {
    // (tot) / nw_j
    const double den = nw.x * nw.x + nw.y * nw.y;
    const double q = (lane == 0 ? tot[0] * nw.x + tot[1] * nw.y : tot[1] * nw.x - tot[0] * nw.y) / den;
    ar = bcast(q, 0);
    ai = bcast(q, 1);
  }
  // alpha_j / nv_j and conj(alpha_j) / conj(nw_j) = conj(alpha_j / nw_j)
  const double dw = nw.x * nw.x + nw.y * nw.y;
  const double num = lane == 0 ? ar : lane == 1 ? ai : lane == 2 ? ar * nw.x + ai * nw.y : ai * nw.x - ar * nw.y;
  const double q = num / (lane < 2 ? nvj : dw);
  const double im = __shfl_down_sync(0xffffffffu, q, 1);
  if (lane == 0) {
    a.c.alp[co] = make_double2(ar, ai);
    st_scal<P>(a.scal, r, 4, q, im);
  }
  if (lane == 2) st_scal<P>(a.scal, r, 5, q, -im);
}

template <class P, int MODE, int BS>
__global__ void __launch_bounds__(BS, step_min_blocks<P, BS>()) k_step(StepArgs a) {
  using R = typename P::R;
  using V_t = typename P::vec_t;
  using L_t = typename P::link_t;
  using A = typename P::A;
  using AT = typename AccOf<P>::A;
  using AS = typename AccOf<P>::st;
  const SiteRef sr = site_ref<BS>(a.b);
  const ProbDesc& d = *sr.d;
  const Geometry g = d.g;
  const int s = sr.s, r = sr.r;
  const bool active = sr.active;
  const int ss = active ? s : 0;
  const size_t vo = d.voff;
  const L_t* links = (const L_t*)d.links;
  const R mass = hconst(R(), d.mass, d.mass_hl);
  const R emu = hconst(R(), d.emu, d.emu_hl), emui = hconst(R(), d.emui, d.emui_hl);
  const StepPtrs sp = step_ptrs(a);
  const size_t co = (size_t)r * a.c.ld + sp.j;
  int xc[4];
  site_coords(g, ss, xc[0], xc[1], xc[2], xc[3]);

  cx<A> dot = {rzero<A>(), rzero<A>()};
  cx<R> acc[12];

  if (MODE == kModeApply) {
    __shared__ CanonSmem<BS> sm;
    double2 z[12];
    if (active) {
      const V_t* tv = (const V_t*)a.tv + vo;
      hopping<P>(acc, tv, links, g, s, xc, a.dagger ? emui : emu, a.dagger ? emu : emui);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const cx<double> d = vec_to_cd(g5d(k, ld_vec(tv + (size_t)k * g.V + s), acc[k], mass));
        z[k] = make_double2(d.re, d.im);
      }
    }
    canon_store(a.ycanon + vo, g.V, s - (int)(threadIdx.x & 31), sm.v[threadIdx.x >> 5], z);
    return;
  }

  const V_t* tc = (const V_t*)sp.tc + vo;
  if (MODE == kModeRegen) {
    // second pass, all coefficients known: p = A t_j / nv_j - (gamma_j / nv_{j-1}) t_{j-1},
    // t_{j+1} = p - (alpha_j / nv_j) t_j (over t_{j-1}: each thread reads its own entry of
    // t_{j-1} before writing it), and y += (c_j / nv_j) t_j
    if (!active) return;
    const double nvj = a.c.nv[co];
    const double nvp = sp.j > 1 ? a.c.nv[co - 1] : 1.0;
    const R rinv = from_double<R>(1.0 / nvj);
    const double2 gj = a.c.gam[co];
    const cx<R> cg = cd_to<R>(gj.x / nvp, gj.y / nvp);
    const double2 aj = a.c.alp[co];
    const cx<R> ca = cd_to<R>(aj.x / nvj, aj.y / nvj);
    hopping<P>(acc, tc, links, g, s, xc, emu, emui);
    const V_t* tp = (const V_t*)sp.tp + vo + s;
    V_t* tn = (V_t*)sp.tn + vo + s;
    const cx<AT> cjv = ld_acc((const AS*)a.cacc + (size_t)r * a.c.ld + sp.j);
    AS* ya = (AS*)a.yacc + vo + s;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const cx<R> psi = ld_vec(tc + (size_t)k * g.V + s);
      const cx<R> pk = cscale(g5d(k, psi, acc[k], mass), rinv) - cmul(cg, ld_vec(tp + (size_t)k * g.V));
      st_vec(tn + (size_t)k * g.V, pk - cmul(ca, psi));
      cx<AT> y = ld_acc(ya + (size_t)k * g.V);
      acc_axpy(y, cjv, psi);
      st_acc(ya + (size_t)k * g.V, y);
    }
    return;
  }

  // Lanczos: one side (v). Two-sided: side 0 is v with A, side 1 is w with A^dag.
  //   p = A t_j / nv_j - (gamma_j / nv_{j-1}) t_{j-1}
  //   r = A^dag tw_j / conj(nw_j) - (conj(beta_j) / conj(nw_{j-1})) tw_{j-1}
  //   alpha_j = t_j^dag p / nv_j (Lanczos) or tw_j^dag p / nw_j (two-sided)
  const int nsides = MODE == kModeTwoSided ? 2 : 1;
#pragma unroll 1
  for (int side = 0; side < nsides; ++side) {
    const cx<R> scl = ld_scal<P>(a.scal, r, 2 * side);
    const cx<R> cf = ld_scal<P>(a.scal, r, 2 * side + 1);
    if (active) {
      const V_t* src = side == 0 ? tc : (const V_t*)sp.wc + vo;
      hopping<P>(acc, src, links, g, s, xc, side == 0 ? emu : emui, side == 0 ? emui : emu);
      const V_t* prv = side == 0 ? (const V_t*)sp.tp + vo + s : (const V_t*)sp.wp + vo + s;
      V_t* out = side == 0 ? (V_t*)a.p + vo + s : (V_t*)a.r + vo + s;
      const V_t* pp = (const V_t*)a.p + vo + s;
      if (MODE == kModeLanczos)
        step_site<true, true, 1>(src, prv, out, pp, g.V, s, scl, cf, acc, mass, dot);
      else if (side == 0)
        step_site<true, false, 0>(src, prv, out, pp, g.V, s, scl, cf, acc, mass, dot);
      else
        step_site<false, false, 2>(src, prv, out, pp, g.V, s, scl, cf, acc, mass, dot);
    }
  }
  A v2[2] = {dot.re, dot.im};
  double tot[2];
  if (reduce_last<2, BS>(v2, a.partials, a.counters, r, d.block0, sr.bx, d.nblk, tot) && threadIdx.x < 32)
    finish_alpha<P, MODE>(a, r, co, tot);
}

// ------------------------------------------------------------ vector update
// resident threads per SM the update kernel is compiled for (0: the compiler's choice, 56
// registers). 1280 (48 registers, five blocks of 256) measured 0.168 -> 0.161 ms for the
// double-float two-sided update at 16^4 x 12; 1536 spills, and 256 (145 registers, the
// loads of all twelve components in flight in one thread) runs at 0.29 ms.
#ifndef OV_UPDATE_THREADS
#define OV_UPDATE_THREADS 1280
#endif
#if OV_UPDATE_THREADS > 0
#define OV_UPDATE_BOUNDS(BS) __launch_bounds__(BS, (OV_UPDATE_THREADS / BS > 0 ? OV_UPDATE_THREADS / BS : 1))
#else
#define OV_UPDATE_BOUNDS(BS) __launch_bounds__(BS)
#endif
// beta_{j+1} and the next step's scalars from ||t_{j+1}||^2 (one warp)
template <class P>
__device__ __forceinline__ void finish_lanczos(const StepArgs& a, int r, size_t co, int j, double tot) {
  const int lane = threadIdx.x & 31;
  const double nvp = a.c.nv[co];
  const double2 nwp = a.c.nw[co];
  const int status = a.c.status[r];
  const double b = sqrt(tot);
  const double bprev = fabs(a.c.bet[co].x);
  const size_t cn = co + 1;
  const bool broke = !(b > a.breakdown_tol * (fabs(a.c.alp[co].x) + bprev));
  const bool dead = broke || status != kStOK;
  const double nv = dead ? 1.0 : b;
  const double2 nw = make_double2(nv, 0.0), bg = make_double2(dead ? 0.0 : b, 0.0);
  __syncwarp();
  if (lane == 0) {
    if (broke && status == kStOK) {
      a.c.status[r] = kStLucky;
      a.c.kbreak[r] = j;
    }
    a.c.nv[cn] = nv;
    a.c.nw[cn] = nw;
    a.c.bet[cn] = bg;
    a.c.gam[cn] = bg;
  }
  set_step_scal<P>(a.scal, r, nv, bg, nw, bg, nvp, nwp);
}
// beta_{j+1}, gamma_{j+1} and the next step's scalars from tw^dag t, ||t||^2, ||tw||^2 (one warp)
template <class P>
__device__ __forceinline__ void finish_two_sided(const StepArgs& a, int r, size_t co, int j, const double (&tot)[4]) {
  const int lane = threadIdx.x & 31;
  const double nvp = a.c.nv[co];
  const double2 nwp = a.c.nw[co];
  const int status = a.c.status[r];
  const double dre = tot[0], dim = tot[1];
  const double root = sqrt(lane == 0 ? dre * dre + dim * dim : lane == 1 ? tot[2] : tot[3]);
  const double ad = bcast(root, 0), nt = bcast(root, 1), nu = bcast(root, 2);
  const double b = sqrt(ad);
  const size_t cn = co + 1;
  const bool broke = !(ad > a.breakdown_tol * nt * nu) || !(b > 0.0);
  const bool dead = broke || status != kStOK;
  const double q = (lane == 0 ? dre : dim) / b;
  const double2 g = make_double2(bcast(q, 0), bcast(q, 1));
  const double nv = dead ? 1.0 : b;
  const double2 nw = dead ? make_double2(1.0, 0.0) : g, be = make_double2(dead ? 0.0 : b, 0.0);
  const double2 ga = dead ? make_double2(0.0, 0.0) : g;
  __syncwarp();
  if (lane == 0) {
    if (broke && status == kStOK) {
      a.c.status[r] = kStBreakdown;
      a.c.kbreak[r] = j;
    }
    a.c.nv[cn] = nv;
    a.c.nw[cn] = nw;
    a.c.bet[cn] = be;
    a.c.gam[cn] = ga;
  }
  set_step_scal<P>(a.scal, r, nv, ga, nw, be, nvp, nwp);
}
__device__ __forceinline__ void advance_step(const StepArgs& a, int j) {
  // device-side step state: the last block of the launch advances j
  if (a.jdev) {
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned t = atomicAdd(a.gticket, 1u);
      if (t == gridDim.x - 1) {
        *a.jdev = j + 1;
        *a.gticket = 0u;
        __threadfence();
      }
    }
  }
}

template <class P, int MODE, int BS>
__global__ void OV_UPDATE_BOUNDS(BS) k_update(StepArgs a) {
  using R = typename P::R;
  using V_t = typename P::vec_t;
  using A = typename P::A;
  const SiteRef sr = site_ref<BS, true>(a.b);
  const Geometry g = sr.d->g;
  const int s = sr.s, r = sr.r;
  const size_t vo = sr.d->voff;
  const StepPtrs sp = step_ptrs(a);
  const size_t co = (size_t)r * a.c.ld + sp.j;
  const cx<R> alp = ld_scal<P>(a.scal, r, 4);
  const cx<R> calp = ld_scal<P>(a.scal, r, 5);
  using NL = typename NormLo<A>::T;
  cx<A> d = {rzero<A>(), rzero<A>()};
  A nvv = rzero<A>();              // ||v~||^2: beta in Lanczos
  NL nvl = NL(0), nwl = NL(0);     // ||v~||^2, ||w~||^2 for the breakdown test of 2sL
  if (sr.active) {
    // t_{j+1} = p - (alpha_j / nv_j) t_j, tw_{j+1} = r - (conj(alpha_j) / conj(nw_j)) tw_j
    const V_t* __restrict__ pp = (const V_t*)a.p + vo + s;
    const V_t* __restrict__ vc = (const V_t*)sp.tc + vo + s;
    V_t* __restrict__ tv = (V_t*)sp.tn + vo + s;  // may be t_{j-1}: the stencil no longer reads it
    if (MODE == kModeLanczos) {
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const cx<R> t = csubmul(ld_vec(pp + (size_t)k * g.V), alp, ld_vec(vc + (size_t)k * g.V));
        st_vec(tv + (size_t)k * g.V, t);
        acc_norm(nvv, t);
      }
    } else {
      const V_t* __restrict__ rr = (const V_t*)a.r + vo + s;
      const V_t* __restrict__ wc = (const V_t*)sp.wc + vo + s;
      V_t* __restrict__ tw = (V_t*)sp.wn + vo + s;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const cx<R> t = csubmul(ld_vec(pp + (size_t)k * g.V), alp, ld_vec(vc + (size_t)k * g.V));
        const cx<R> u = csubmul(ld_vec(rr + (size_t)k * g.V), calp, ld_vec(wc + (size_t)k * g.V));
        st_vec(tv + (size_t)k * g.V, t);
        st_vec(tw + (size_t)k * g.V, u);
        acc_dot(d, u, t);
        acc_norm_lo(nvl, t);
        acc_norm_lo(nwl, u);
      }
    }
  }
  if (MODE == kModeLanczos) {
    A v1[1] = {nvv};
    double tot[1];
    if (reduce_last<1, BS>(v1, a.partials, a.counters, r, sr.d->block0, sr.bx, sr.d->nblk, tot) && threadIdx.x < 32)
      finish_lanczos<P>(a, r, co, sp.j, tot[0]);
  } else {
    A v4[4] = {d.re, d.im, to_acc(nvl, A()), to_acc(nwl, A())};
    double tot[4];
    if (reduce_last<4, BS>(v4, a.partials, a.counters, r, sr.d->block0, sr.bx, sr.d->nblk, tot) && threadIdx.x < 32)
      finish_two_sided<P>(a, r, co, sp.j, tot);
  }
  advance_step(a, sp.j);
}

// ------------------------------------------------------------ small lattices
// One thread a site runs ~29 k instructions one after the other in a strict two-sided step, and
// a lattice with fewer sites than the GPU has threads spends just that latency: 45 us a step on
// 8^4. The wide kernels give a site twelve threads: the two sides of the step to different
// blocks (blockIdx.y; alpha's partial sum moves to the v side, which reads tw_j), the three
// colour rows of the result to different warps, the two upper spin components to the half
// warps. A thread projects and multiplies its half-spinor's row (the projection is repeated by
// the three colours: a third more work in all) and owns two of the twelve components, upper
// spin `sp` and lower spin 2 + sp of its colour; the lower one takes its own or the other half
// warp's product, by a shuffle. The sums of a component keep their order. A block takes WS
// consecutive sites of a 64-site block of the map. Step on 8^4 45 -> 18 us, 4^4 (mu = 0) 37 -> 16
// us; 24 lattices of 57,000 sites in all 96 -> 128 us, so the tuner decides.
__device__ __forceinline__ dfu shfl_half(dfu v) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, 16), __shfl_xor_sync(0xffffffffu, v.lo, 16)};
}
template <int WS>
struct WideRef {
  static constexpr int threads = 6 * WS, sub = 64 / WS;
  int r, bx, s, col, sp;
  bool active;
  const ProbDesc* d;
};
template <int WS>
__device__ __forceinline__ WideRef<WS> wide_ref(const Batch& b) {
  constexpr int sub = WideRef<WS>::sub;
  const int2 m = __ldg(&b.blk_map[blockIdx.x / sub]);
  const ProbDesc* d = &b.desc[m.x];
  const int warp = threadIdx.x >> 5, bx = m.y * sub + blockIdx.x % sub;
  const int s = bx * WS + (warp / 3) * 16 + (threadIdx.x & 15);
  return {m.x, bx, s, warp % 3, (int)(threadIdx.x >> 4) & 1, s < d->g.V, d};
}

// the hopping sum of hopping_df for components 3 sp + col (up) and 6 + 3 sp + col (lo). CG: the
// vector is read past the L1 cache (other blocks of the same launch write it)
template <bool CG>
__device__ __forceinline__ cx<df64> ld_vec_wide(const float4* p) {
  const float4 v = CG ? __ldcg(p) : *p;
  return ld_vec(&v);
}
template <bool CG = false>
__device__ __forceinline__ void hopping_wide(cx<df64>& up, cx<df64>& lo, const float4* __restrict__ src,
                                             const float2* __restrict__ links, const Geometry& g, int s,
                                             const int (&xc)[4], df64 ef, df64 eb, int col, int sp) {
  const int V = g.V;
  const float2* __restrict__ links_lo = links + (size_t)36 * V;
  cxu au = {{0.f, 0.f}, {0.f, 0.f}}, al = au;
  // the next hop's operands are loaded while this one is computed
  cx<float> un[3], uln[3];
  cx<df64> pn[3], qn[3];
  auto load = [&](int hop) {
    const int nu = hop >> 1;
    const bool fwd = (hop & 1) == 0;
    const int Ln = nu == 0 ? g.Lx : (nu == 1 ? g.Ly : (nu == 2 ? g.Lz : g.Lt));
    const int st = nu == 0 ? 1 : (nu == 1 ? g.Lx : (nu == 2 ? g.Lx * g.Ly : g.Lx * g.Ly * g.Lz));
    const int c = xc[0] * (nu == 0) + xc[1] * (nu == 1) + xc[2] * (nu == 2) + xc[3] * (nu == 3);
    const int sn = fwd ? (c == Ln - 1 ? s - (Ln - 1) * st : s + st) : (c == 0 ? s + (Ln - 1) * st : s - st);
    const int ls = fwd ? s : sn, bs = c_bsrc[nu][sp];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int idx = fwd ? col * 3 + b : b * 3 + col;
      un[b] = ld_link(links + (size_t)(nu * 9 + idx) * V + ls);
      uln[b] = ld_link(links_lo + (size_t)(nu * 9 + idx) * V + ls);
      pn[b] = ld_vec_wide<CG>(src + (size_t)(3 * sp + b) * V + sn);
      qn[b] = ld_vec_wide<CG>(src + (size_t)(3 * bs + b) * V + sn);
    }
  };
  load(0);
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int nu = hop >> 1;
    const bool fwd = (hop & 1) == 0;
    const int bq = (c_bph[nu][sp] + (fwd ? 2 : 0)) & 3;
    cx<float> u[3], ulo[3];
    cx<df64> h[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      u[b] = lconj(un[b], !fwd);
      ulo[b] = lconj(uln[b], !fwd);
      const cx<df64> p = pn[b], q = rot(qn[b], bq);
      const dfu re = add_u(to_u(p.re), to_u(q.re)), im = add_u(to_u(p.im), to_u(q.im));
      h[b] = {{re.hi, re.lo}, {im.hi, im.lo}};
    }
    if (hop < 7) load(hop + 1);
    cxu gs;
    float cr = 0.f, ci = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if (b == 0) {
        set_u(gs.re, u[b].re, h[b].re);
        set_u(gs.im, u[b].re, h[b].im);
      } else {
        madd_u(gs.re, u[b].re, h[b].re);
        madd_u(gs.im, u[b].re, h[b].im);
      }
      madd_u(gs.re, -u[b].im, h[b].im);
      madd_u(gs.im, u[b].im, h[b].re);
      cr = __fmaf_rn(ulo[b].re, h[b].re.hi, __fmaf_rn(-ulo[b].im, h[b].im.hi, cr));
      ci = __fmaf_rn(ulo[b].re, h[b].im.hi, __fmaf_rn(ulo[b].im, h[b].re.hi, ci));
    }
    gs.re.lo = __fadd_rn(gs.re.lo, cr);
    gs.im.lo = __fadd_rn(gs.im.lo, ci);
    if (nu == 3) {
      const cx<df64> n = cscale(cx<df64>{norm_u(gs.re), norm_u(gs.im)}, fwd ? ef : eb);
      gs = {to_u(n.re), to_u(n.im)};
    }
    const cxu go = {shfl_half(gs.re), shfl_half(gs.im)};
    au = cadd_u(au, gs);
    al = cadd_u(al, rot_u(c_dsrc[nu][sp] == sp ? gs : go, (c_dph[nu][sp] + (fwd ? 2 : 0)) & 3));
  }
  up = {norm_u(au.re), norm_u(au.im)};
  lo = {norm_u(al.re), norm_u(al.im)};
}

template <int MODE, int WS>
__global__ void __launch_bounds__(6 * WS) k_step_wide(StepArgs a) {
  using P = PrecDF64;
  const WideRef<WS> sr = wide_ref<WS>(a.b);
  const ProbDesc& d = *sr.d;
  const Geometry g = d.g;
  const int r = sr.r, V = g.V;
  const int ss = sr.active ? sr.s : 0;
  const size_t vo = d.voff;
  const df64 mass = {d.mass_hl[0], d.mass_hl[1]}, emu = {d.emu_hl[0], d.emu_hl[1]}, emui = {d.emui_hl[0], d.emui_hl[1]};
  int xc[4];
  site_coords(g, ss, xc[0], xc[1], xc[2], xc[3]);
  const int k0 = 3 * sr.sp + sr.col, k1 = 6 + k0;  // this thread's components
  cx<df64> up, lo;
  if (MODE == kModeApply) {
    const float4* tv = (const float4*)a.tv + vo;
    hopping_wide(up, lo, tv, (const float2*)d.links, g, ss, xc, a.dagger ? emui : emu, a.dagger ? emu : emui, sr.col, sr.sp);
    if (!sr.active) return;
    double2* out = a.ycanon + vo + (size_t)ss * 12;
    const cx<double> z0 = vec_to_cd(g5d(k0, ld_vec(tv + (size_t)k0 * V + ss), up, mass));
    const cx<double> z1 = vec_to_cd(g5d(k1, ld_vec(tv + (size_t)k1 * V + ss), lo, mass));
    out[k0] = make_double2(z0.re, z0.im);
    out[k1] = make_double2(z1.re, z1.im);
    return;
  }
  const StepPtrs sp = step_ptrs(a);
  const size_t co = (size_t)r * a.c.ld + sp.j;
  const int side = MODE == kModeTwoSided ? blockIdx.y : 0;
  const cx<df64> scl = ld_scal<P>(a.scal, r, 2 * side), cf = ld_scal<P>(a.scal, r, 2 * side + 1);
  const float4* src = (const float4*)(side == 0 ? sp.tc : sp.wc) + vo;
  const float4* prv = (const float4*)(side == 0 ? sp.tp : sp.wp) + vo + ss;
  float4* out = (float4*)(side == 0 ? a.p : a.r) + vo + ss;
  hopping_wide(up, lo, src, (const float2*)d.links, g, ss, xc, side == 0 ? emu : emui, side == 0 ? emui : emu, sr.col, sr.sp);
  cx<df64> dot = {df_zero(), df_zero()};
  if (sr.active) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = q == 0 ? k0 : k1;
      const cx<df64> psi = ld_vec(src + (size_t)k * V + ss), pv = ld_vec(prv + (size_t)k * V);
      const cx<df64> h = g5d(k, psi, q == 0 ? up : lo, mass);
      cx<df64> ok;
      if (MODE == kModeLanczos) ok = smulsub<true, true>(scl, h, cf, pv);
      else if (side == 0) ok = smulsub<true, false>(scl, h, cf, pv);
      else ok = smulsub<false, false>(scl, h, cf, pv);
      st_vec(out + (size_t)k * V, ok);
      if (MODE == kModeLanczos) acc_dot(dot, psi, ok);
      else if (side == 0) acc_dot(dot, ld_vec((const float4*)sp.wc + vo + (size_t)k * V + ss), ok);
    }
  }
  if (side != 0) return;
  df64 v2[2] = {dot.re, dot.im};
  double tot[2];
  constexpr int sub = WideRef<WS>::sub;
  if (reduce_last<2, 6 * WS>(v2, a.partials, a.counters, r, d.block0 * sub, sr.bx, d.nblk * sub, tot) && threadIdx.x < 32)
    finish_alpha<P, MODE>(a, r, co, tot);
}

template <int MODE, int WS>
__global__ void __launch_bounds__(6 * WS) k_update_wide(StepArgs a) {
  using P = PrecDF64;
  const WideRef<WS> sr = wide_ref<WS>(a.b);
  const int V = sr.d->g.V, r = sr.r;
  const StepPtrs sp = step_ptrs(a);
  const size_t co = (size_t)r * a.c.ld + sp.j;
  const cx<df64> alp = ld_scal<P>(a.scal, r, 4), calp = ld_scal<P>(a.scal, r, 5);
  cx<df64> d = {df_zero(), df_zero()};
  df64 nvv = df_zero();
  float nvl = 0.f, nwl = 0.f;
  if (sr.active) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const size_t o = sr.d->voff + sr.s + (size_t)(6 * q + 3 * sr.sp + sr.col) * V;
      const cx<df64> t = csubmul(ld_vec((const float4*)a.p + o), alp, ld_vec((const float4*)sp.tc + o));
      if (MODE == kModeLanczos) {
        st_vec((float4*)sp.tn + o, t);
        acc_norm(nvv, t);
      } else {
        const cx<df64> u = csubmul(ld_vec((const float4*)a.r + o), calp, ld_vec((const float4*)sp.wc + o));
        st_vec((float4*)sp.tn + o, t);
        st_vec((float4*)sp.wn + o, u);
        acc_dot(d, u, t);
        acc_norm_lo(nvl, t);
        acc_norm_lo(nwl, u);
      }
    }
  }
  constexpr int sub = WideRef<WS>::sub;
  const int part0 = sr.d->block0 * sub, nblk = sr.d->nblk * sub;
  if (MODE == kModeLanczos) {
    df64 v1[1] = {nvv};
    double tot[1];
    if (reduce_last<1, 6 * WS>(v1, a.partials, a.counters, r, part0, sr.bx, nblk, tot) && threadIdx.x < 32)
      finish_lanczos<P>(a, r, co, sp.j, tot[0]);
  } else {
    df64 v4[4] = {d.re, d.im, {nvl, 0.f}, {nwl, 0.f}};
    double tot[4];
    if (reduce_last<4, 6 * WS>(v4, a.partials, a.counters, r, part0, sr.bx, nblk, tot) && threadIdx.x < 32)
      finish_two_sided<P>(a, r, co, sp.j, tot);
  }
  advance_step(a, sp.j);
}

// ------------------------------------------------------------ runs of steps in one launch
// On lattices whose blocks all fit the SMs at once, two launches a step cost more than the
// step's work (4^4: 20 us a step, of which the launches, the pointers read from memory, the
// tickets and the coefficients' finishing took most). k_steps runs `nsteps` outer steps in one
// cooperative launch: a block of the wide layout holds both sides of its sites (threads 0 .. 95
// the v side, the rest the w side), keeps its own entries of t_j, t_{j-1}, p (and r) in
// registers and exchanges what the dot products need through shared memory; only the new
// vectors go to memory, for the neighbours. The two reductions of a step are barriers over the
// problem's blocks, after which every block adds the partial sums itself, in the same order, and
// forms the coefficients (block 0 of the problem stores them). A barrier's wait is bounded: when
// it runs out the block sets *err and returns; the others look at *err while they wait, and a
// launch that finds it set returns at once (the counters are off their grid from then on). The
// host reads the word with every group of checks and at the end, and gives the apply up. A step
// on 4^4 (mu = 0) 20 -> 15 us, on 8^4 (mu = 0.3) 25 -> 23 us, half of it the two barriers and the
// double arithmetic of the coefficients between them.
__device__ __forceinline__ bool problem_barrier(unsigned* bar, unsigned nblk, int polls, int* err, int* s_fail) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(bar, 1u), target = (t / nblk + 1u) * nblk;
    for (int n = 0;; ++n) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if (n >= polls || ((n & 1023) == 1023 && *(volatile int*)err != 0)) {
        *(volatile int*)err = 1;
        *s_fail = 1;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *s_fail == 0;
}
// the problem's total of NQ partial sums a block, in warp 0, in block order by lanes
template <int NQ>
__device__ __forceinline__ void problem_total(const double* part, int nblk, double (&tot)[NQ]) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) tot[q] = 0.0;
  for (int b = threadIdx.x; b < nblk; b += 32)
#pragma unroll
    for (int q = 0; q < NQ; ++q) tot[q] += __ldcg(part + (size_t)b * 4 + q);
#pragma unroll
  for (int q = 0; q < NQ; ++q) tot[q] = warp_sum(tot[q]);
}
// a block's sums of NQ values over warps [w0, w1), stored as its partial sums (all threads call)
template <int NQ>
__device__ __forceinline__ void block_partial(df64 (&v)[NQ], int w1, double* out) {
  __shared__ float2 s[6][4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    v[q] = warp_sum(v[q]);
    if (lane == 0) s[warp][q] = make_float2(v[q].hi, v[q].lo);
  }
  __syncthreads();
  if (threadIdx.x < NQ) {
    df64 t = df_zero();
    for (int w = 0; w < w1; ++w) t = t + df64{s[w][threadIdx.x].x, s[w][threadIdx.x].y};
    __stcg(out + threadIdx.x, df_to_double(t));
  }
}

template <int MODE>
__global__ void __launch_bounds__(MODE == kModeTwoSided ? 192 : 96) k_steps(StepArgs a, int nsteps, unsigned* bars, int polls, int* err) {
  constexpr bool TWO = MODE == kModeTwoSided;
  constexpr int WS = 16, sub = 4, NW = TWO ? 6 : 3;
  __shared__ float4 s_x[96 * 2];          // the w side's entries, for the v side's dot products
  __shared__ float4 s_scal[6];            // the step scalars of StepArgs::scal
  __shared__ int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int side = TWO ? tid / 96 : 0, t96 = tid % 96;
  const int2 m = __ldg(&a.b.blk_map[blockIdx.x / sub]);
  const int r = m.x, bx = m.y * sub + blockIdx.x % sub;
  const ProbDesc& d = a.b.desc[r];
  const Geometry g = d.g;
  const int V = g.V, s = bx * WS + (lane & 15), sp2 = (lane >> 4) & 1, col = warp % 3;
  const bool active = s < V;
  const int ss = active ? s : 0;
  const size_t vo = d.voff;
  const int nblk = d.nblk * sub;
  const bool lead = bx == 0;
  double* const pa = a.partials + (size_t)d.block0 * sub * 4;                       // alpha's partial sums
  double* const pd = pa + (size_t)a.b.nblocks * sub * 4;                            // beta's and gamma's
  const df64 mass = {d.mass_hl[0], d.mass_hl[1]}, emu = {d.emu_hl[0], d.emu_hl[1]}, emui = {d.emui_hl[0], d.emui_hl[1]};
  const df64 ef = side == 0 ? emu : emui, eb = side == 0 ? emui : emu;
  int xc[4];
  site_coords(g, ss, xc[0], xc[1], xc[2], xc[3]);
  const int kk[2] = {3 * sp2 + col, 6 + 3 * sp2 + col};  // this thread's components
  const int j0 = __ldcg(a.jdev);
  if (tid == 0) s_fail = *(volatile int*)err;
  __syncthreads();
  if (s_fail) return;
  if (tid < 4) s_scal[tid] = __ldcg((const float4*)a.scal + (size_t)r * 8 + tid);
  size_t co = (size_t)r * a.c.ld + j0;
  double nvj = a.c.nv[co];
  double2 nwj = a.c.nw[co], betj = a.c.bet[co];
  int status = a.c.status[r];
  StepPtrs sp = step_ptrs(a);
  const float4* src = (const float4*)(side == 0 ? sp.tc : sp.wc) + vo;
  cx<df64> cur[2], prv[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const size_t o = (size_t)kk[q] * V + ss;
    cur[q] = ld_vec_wide<true>(src + o);
    prv[q] = ld_vec_wide<true>((const float4*)(side == 0 ? sp.tp : sp.wp) + vo + o);
  }
  for (int i = 0; i < nsteps; ++i, ++co) {
    const int j = j0 + i;
    // the destination of t_{j+1} (the w side's ring: tw_{j+1} over tw_{j-1})
    float4* dst;
    if (side == 1) dst = (float4*)((char*)a.wring + a.pool_bytes * ((j + 1) & 1)) + vo;
    else dst = (a.slot_tab ? (float4*)a.slot_tab[j] : (float4*)((char*)a.vring + a.pool_bytes * ((j + 1) & 1))) + vo;
    if (TWO && side == 1) {
      st_vec(&s_x[t96], cur[0]);
      st_vec(&s_x[96 + t96], cur[1]);
    }
    __syncthreads();  // s_x, s_scal
    const cx<df64> scl = ld_vec(&s_scal[2 * side]), cf = ld_vec(&s_scal[2 * side + 1]);
    cx<df64> up, lo, ok[2];
    hopping_wide<true>(up, lo, src, (const float2*)d.links, g, ss, xc, ef, eb, col, sp2);
    cx<df64> dot = {df_zero(), df_zero()};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const cx<df64> h = g5d(kk[q], cur[q], q == 0 ? up : lo, mass);
      if (!TWO) ok[q] = smulsub<true, true>(scl, h, cf, prv[q]);
      else if (side == 0) ok[q] = smulsub<true, false>(scl, h, cf, prv[q]);
      else ok[q] = smulsub<false, false>(scl, h, cf, prv[q]);
      if (active && side == 0) acc_dot(dot, TWO ? ld_vec(&s_x[96 * q + t96]) : cur[q], ok[q]);
    }
    {
      df64 v[2] = {dot.re, dot.im};
      block_partial(v, 3, pa + (size_t)bx * 4);
    }
    if (!problem_barrier(&bars[r], nblk, polls, err, &s_fail)) return;
    if (warp == 0) {
      double tot[2];
      problem_total<2>(pa, nblk, tot);
      // as finish_alpha
      double ar, ai = 0.0;
      double2 nw = nwj;
      if (!TWO) {
        ar = tot[0] / nvj;
        nw = make_double2(nvj, 0.0);
      } else {
        const double den = nw.x * nw.x + nw.y * nw.y;
        const double q = (lane == 0 ? tot[0] * nw.x + tot[1] * nw.y : tot[1] * nw.x - tot[0] * nw.y) / den;
        ar = bcast(q, 0);
        ai = bcast(q, 1);
      }
      const double dw = nw.x * nw.x + nw.y * nw.y;
      const double num = lane == 0 ? ar : lane == 1 ? ai : lane == 2 ? ar * nw.x + ai * nw.y : ai * nw.x - ar * nw.y;
      const double q = num / (lane < 2 ? nvj : dw);
      const double im = __shfl_down_sync(0xffffffffu, q, 1);
      if (lane == 0) {
        if (lead) a.c.alp[co] = make_double2(ar, ai);
        st_vec(&s_scal[4], cd_to<df64>(q, im));
      }
      if (lane == 2) st_vec(&s_scal[5], cd_to<df64>(q, -im));
      betj.y = ar;  // (Lanczos' breakdown test reads alpha_j; bet is real)
    }
    __syncthreads();
    const cx<df64> al = ld_vec(&s_scal[4 + side]);
    df64 nvv = df_zero();
    cx<df64> del = {df_zero(), df_zero()};
    float nl = 0.f;
    cx<df64> nxt[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      nxt[q] = csubmul(ok[q], al, cur[q]);
      if (active) {
        __stcg(dst + (size_t)kk[q] * V + ss, vec_of(nxt[q]));
        if (!TWO) acc_norm(nvv, nxt[q]);
        else acc_norm_lo(nl, nxt[q]);
      }
      if (TWO && side == 1) st_vec(&s_x[96 * q + t96], nxt[q]);
    }
    if (TWO) {
      __syncthreads();
      if (active && side == 0) {
        acc_dot(del, ld_vec(&s_x[t96]), nxt[0]);
        acc_dot(del, ld_vec(&s_x[96 + t96]), nxt[1]);
      }
      df64 v[4] = {del.re, del.im, {side == 0 ? nl : 0.f, 0.f}, {side == 1 ? nl : 0.f, 0.f}};
      block_partial(v, NW, pd + (size_t)bx * 4);
    } else {
      df64 v[1] = {nvv};
      block_partial(v, NW, pd + (size_t)bx * 4);
    }
    __threadfence();  // the new vector, before the barrier's arrival
    if (!problem_barrier(&bars[r], nblk, polls, err, &s_fail)) return;
    if (warp == 0) {
      double nv;
      double2 nw, be, ga;
      bool broke;
      if (!TWO) {
        double tot[1];
        problem_total<1>(pd, nblk, tot);
        // as finish_lanczos
        const double bb = sqrt(tot[0]);
        broke = !(bb > a.breakdown_tol * (fabs(betj.y) + fabs(betj.x)));
        const bool dead = broke || status != kStOK;
        nv = dead ? 1.0 : bb;
        nw = make_double2(nv, 0.0);
        be = ga = make_double2(dead ? 0.0 : bb, 0.0);
      } else {
        double tot[4];
        problem_total<4>(pd, nblk, tot);
        // as finish_two_sided
        const double dre = tot[0], dim = tot[1];
        const double root = sqrt(lane == 0 ? dre * dre + dim * dim : lane == 1 ? tot[2] : tot[3]);
        const double ad = bcast(root, 0), nt = bcast(root, 1), nu = bcast(root, 2);
        const double bb = sqrt(ad);
        broke = !(ad > a.breakdown_tol * nt * nu) || !(bb > 0.0);
        const bool dead = broke || status != kStOK;
        const double q = (lane == 0 ? dre : dim) / bb;
        const double2 gg = make_double2(bcast(q, 0), bcast(q, 1));
        nv = dead ? 1.0 : bb;
        nw = dead ? make_double2(1.0, 0.0) : gg;
        be = make_double2(dead ? 0.0 : bb, 0.0);
        ga = dead ? make_double2(0.0, 0.0) : gg;
      }
      if (lead && lane == 0) {
        if (broke && status == kStOK) {
          a.c.status[r] = TWO ? kStBreakdown : kStLucky;
          a.c.kbreak[r] = j;
        }
        a.c.nv[co + 1] = nv;
        a.c.nw[co + 1] = nw;
        a.c.bet[co + 1] = be;
        a.c.gam[co + 1] = ga;
      }
      if (broke && status == kStOK) status = TWO ? kStBreakdown : kStLucky;
      set_step_scal<PrecDF64>(s_scal, 0, nv, ga, nw, be, nvj, nwj);
      if (lead && i + 1 == nsteps) set_step_scal<PrecDF64>(a.scal, r, nv, ga, nw, be, nvj, nwj);
      nvj = nv;
      nwj = nw;
      betj = be;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      prv[q] = cur[q];
      cur[q] = nxt[q];
    }
    src = dst;
  }
  // the last problem to finish advances the step index
  if (lead && tid == 0) {
    __threadfence();
    if (atomicAdd(a.gticket, 1u) == (unsigned)(a.b.nprob - 1)) {
      *a.gticket = 0u;
      *a.jdev = j0 + nsteps;
      __threadfence();
    }
  }
}

// blocks of k_steps that run at the same time
int steps_capacity(int mode) {
  int per = 0, dev = 0, sms = 0;
  cudaError_t e = mode == kModeTwoSided
                      ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_steps<kModeTwoSided>, 192, 0)
                      : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_steps<kModeLanczos>, 96, 0);
  if (e != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per * sms;
}
cudaError_t launch_steps(int mode, const StepArgs& a, int nsteps, unsigned* bars, int polls, int* err, cudaStream_t st) {
  StepArgs args = a;
  void* p[] = {&args, &nsteps, &bars, &polls, &err};
  const dim3 grid(a.b.nblocks * 4);
  if (mode == kModeTwoSided)
    return cudaLaunchCooperativeKernel((const void*)k_steps<kModeTwoSided>, grid, dim3(192), p, 0, st);
  return cudaLaunchCooperativeKernel((const void*)k_steps<kModeLanczos>, grid, dim3(96), p, 0, st);
}

// ------------------------------------------------------------ recombination
// scale z (+ x, gamma5) for components k0 .. k0 + NC - 1
template <int NC, class AT>
__device__ __forceinline__ void finish_site(const cx<AT> (&acc)[NC], int k0, double sc, int add_x, const double2 (&xs)[NC],
                                            double2 (&out)[NC]) {
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    cx<double> z = acc_to_cd(acc[k]);
    z.re *= sc;
    z.im *= sc;
    if (add_x) {
      if (k0 + k >= 6) { z.re = -z.re; z.im = -z.im; }
      z.re += xs[k].x;
      z.im += xs[k].y;
    }
    out[k] = make_double2(z.re, z.im);
  }
}

// NC = 12: a thread sums the whole site (bound by HBM: the stored basis is read once; two steps
// unrolled 8.7 ms for 12 x 16^4 at k = 350, one 14.1, four 9.6; one or three components a thread
// 8.9 to 10.0). NC = 1: one component (blockIdx.y) a thread, for lattices with few sites, where
// the site's thread ran k times twelve dependent sums (4^4, k = 170: 0.30 -> 0.10 ms)
template <class P, int BS, int NC>
__global__ void __launch_bounds__(BS) k_recombine(Batch bt, const void* const* __restrict__ slots,
                                                      const typename AccOf<P>::st* __restrict__ cacc, int ldc,
                                                      const int* __restrict__ kr, const double* __restrict__ scale,
                                                      const double2* __restrict__ x, int add_x, double2* y) {
  using AT = typename AccOf<P>::A;
  const SiteRef sr = site_ref<BS>(bt);
  const int s = sr.s, r = sr.r, V = sr.d->g.V, k0 = NC == 12 ? 0 : blockIdx.y;
  const size_t vo = sr.d->voff;
  cx<AT> acc[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) acc[k] = czero<AT>();
  const int k_r = sr.active ? kr[r] : 0;
  const typename AccOf<P>::st* cr = cacc + (size_t)r * ldc;
#pragma unroll(NC == 12 ? 2 : 8)
  for (int j = 0; j < k_r; ++j) {
    const cx<AT> cj = ld_acc(cr + j + 1);
    const typename P::vec_t* vj = (const typename P::vec_t*)slots[j] + vo + (size_t)k0 * V + s;
#pragma unroll
    for (int k = 0; k < NC; ++k) acc_axpy(acc[k], cj, ld_vec(vj + (size_t)k * V));
  }
  const double sc = scale[r];
  double2 xs[NC], out[NC];
  if constexpr (NC == 12) {
    __shared__ CanonSmem<BS> sm;
    double2* w = sm.v[threadIdx.x >> 5];
    const int w0 = s - (int)(threadIdx.x & 31);
    if (add_x) canon_load(x + vo, V, w0, w, xs);
    finish_site<NC>(acc, 0, sc, add_x, xs, out);
    canon_store(y + vo, V, w0, w, out);
  } else if (sr.active) {
    const size_t o = vo + (size_t)s * 12 + k0;
    if (add_x) xs[0] = x[o];
    finish_site<NC>(acc, k0, sc, add_x, xs, out);
    y[o] = out[0];
  }
}

template <class P, int BS>
__global__ void __launch_bounds__(BS) k_finish_acc(Batch bt, const typename AccOf<P>::st* __restrict__ yacc,
                                                       const double* __restrict__ scale,
                                                       const double2* __restrict__ x, int add_x, double2* y) {
  using AT = typename AccOf<P>::A;
  __shared__ CanonSmem<BS> sm;
  const SiteRef sr = site_ref<BS>(bt);
  const int s = sr.s, V = sr.d->g.V, w0 = s - (int)(threadIdx.x & 31);
  const size_t vo = sr.d->voff;
  double2* w = sm.v[threadIdx.x >> 5];
  double2 xs[12], out[12];
  if (add_x) canon_load(x + vo, V, w0, w, xs);
  cx<AT> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = sr.active ? ld_acc(yacc + vo + (size_t)k * V + s) : czero<AT>();
  finish_site<12>(acc, 0, scale[sr.r], add_x, xs, out);
  canon_store(y + vo, V, w0, w, out);
}

// ------------------------------------------------------------ launchers
void fill_consts(ProbDesc& d, double m_w, double mu) {
  d.mass = m_w + 4.0;
  d.emu = exp(mu);
  d.emui = exp(-mu);
  split_const(d.mass, d.mass_hl);
  split_const(d.emu, d.emu_hl);
  split_const(d.emui, d.emui_hl);
}

#define OV_DISPATCH(prec, CALL)                      \
  switch (prec) {                                    \
    case OV_PREC_FP64: { using P = PrecF64; CALL; break; }  \
    case OV_PREC_FP32: { using P = PrecF32; CALL; break; }  \
    default: { using P = PrecDF64; CALL; break; }           \
  }
// the block size is the one the batch's block map was built with
#define OV_BS_DISPATCH(bs, CALL)                           \
  switch (bs) {                                            \
    case 64: { constexpr int BS = 64; CALL; break; }       \
    case 256: { constexpr int BS = 256; CALL; break; }     \
    default: { constexpr int BS = 128; CALL; break; }      \
  }

cudaError_t launch_pack(int prec, const Batch& b, const double2* x, void* xi, void* xi2, Coefs c, double* partials,
                        unsigned* counters, int want_norm, void* scal, cudaStream_t st) {
  OV_BS_DISPATCH(b.block, OV_DISPATCH(prec, (k_pack<P, BS><<<b.nblocks, BS, 0, st>>>(
                                                b, x, (typename P::vec_t*)xi, (typename P::vec_t*)xi2, c, partials,
                                                counters, want_norm, scal))));
  return cudaGetLastError();
}

// steps also take kPrecDF64Relaxed (the double-float storage with float hopping)
#define OV_STEP_DISPATCH(prec, CALL)                                \
  if (prec == kPrecDF64Relaxed) { using P = PrecDF64R; CALL; }      \
  else { OV_DISPATCH(prec, CALL) }

// the wide kernels (strict double-float steps; a.b.wide sites a block, within the map's blocks of 64)
#define OV_WIDE_DISPATCH(ws, CALL)                        \
  if (ws == 16) { constexpr int WS = 16; CALL; }          \
  else { constexpr int WS = 32; CALL; }

cudaError_t launch_step(int prec, int mode, const StepArgs& a, cudaStream_t st) {
  const int grid = a.b.nblocks;
  if (a.b.wide && prec == OV_PREC_DF64 && mode != kModeRegen) {
    const dim3 wg(grid * (64 / a.b.wide), mode == kModeTwoSided ? 2 : 1);
    if (mode == kModeLanczos) {
      OV_WIDE_DISPATCH(a.b.wide, (k_step_wide<kModeLanczos, WS><<<wg, 6 * WS, 0, st>>>(a)));
    } else if (mode == kModeTwoSided) {
      OV_WIDE_DISPATCH(a.b.wide, (k_step_wide<kModeTwoSided, WS><<<wg, 6 * WS, 0, st>>>(a)));
    } else {
      OV_WIDE_DISPATCH(a.b.wide, (k_step_wide<kModeApply, WS><<<wg, 6 * WS, 0, st>>>(a)));
    }
    return cudaGetLastError();
  }
  switch (mode) {
    case kModeLanczos:
      OV_BS_DISPATCH(a.b.block, OV_STEP_DISPATCH(prec, (k_step<P, kModeLanczos, BS><<<grid, BS, 0, st>>>(a))));
      break;
    case kModeTwoSided:
      OV_BS_DISPATCH(a.b.block, OV_STEP_DISPATCH(prec, (k_step<P, kModeTwoSided, BS><<<grid, BS, 0, st>>>(a))));
      break;
    case kModeRegen:
      OV_BS_DISPATCH(a.b.block, OV_STEP_DISPATCH(prec, (k_step<P, kModeRegen, BS><<<grid, BS, 0, st>>>(a))));
      break;
    default:
      OV_BS_DISPATCH(a.b.block, OV_DISPATCH(prec, (k_step<P, kModeApply, BS><<<grid, BS, 0, st>>>(a))));
      break;
  }
  return cudaGetLastError();
}

cudaError_t launch_update(int prec, int mode, const StepArgs& a, cudaStream_t st) {
  const int grid = a.b.nblocks;
  if (a.b.wide && prec == OV_PREC_DF64) {
    const int wg = grid * (64 / a.b.wide);
    if (mode == kModeLanczos) {
      OV_WIDE_DISPATCH(a.b.wide, (k_update_wide<kModeLanczos, WS><<<wg, 6 * WS, 0, st>>>(a)));
    } else {
      OV_WIDE_DISPATCH(a.b.wide, (k_update_wide<kModeTwoSided, WS><<<wg, 6 * WS, 0, st>>>(a)));
    }
    return cudaGetLastError();
  }
  if (mode == kModeLanczos) {
    OV_BS_DISPATCH(a.b.block, OV_DISPATCH(prec, (k_update<P, kModeLanczos, BS><<<grid, BS, 0, st>>>(a))));
  } else {
    OV_BS_DISPATCH(a.b.block, OV_DISPATCH(prec, (k_update<P, kModeTwoSided, BS><<<grid, BS, 0, st>>>(a))));
  }
  return cudaGetLastError();
}

cudaError_t launch_recombine(int prec, const Batch& b, const void* const* slots, const void* cacc, int ldc,
                             const int* k_dev, const double* scale, const double2* x, int add_x, double2* y,
                             cudaStream_t st) {
  // one component a thread while that leaves the GPU with less than its threads twice
  if (b.nblocks * b.block <= 2 * 152 * 2048 / 12) {
    const dim3 grid(b.nblocks, 12);
    OV_BS_DISPATCH(b.block, OV_DISPATCH(prec, (k_recombine<P, BS, 1><<<grid, BS, 0, st>>>(
                                                  b, slots, (const typename AccOf<P>::st*)cacc, ldc, k_dev, scale, x,
                                                  add_x, y))));
    return cudaGetLastError();
  }
  OV_BS_DISPATCH(b.block, OV_DISPATCH(prec, (k_recombine<P, BS, 12><<<b.nblocks, BS, 0, st>>>(
                                                b, slots, (const typename AccOf<P>::st*)cacc, ldc, k_dev, scale, x,
                                                add_x, y))));
  return cudaGetLastError();
}

cudaError_t launch_finish_acc(int prec, const Batch& b, const void* yacc, const double* scale, const double2* x,
                              int add_x, double2* y, cudaStream_t st) {
  OV_BS_DISPATCH(b.block, OV_DISPATCH(prec, (k_finish_acc<P, BS><<<b.nblocks, BS, 0, st>>>(
                                                b, (const typename AccOf<P>::st*)yacc, scale, x, add_x, y))));
  return cudaGetLastError();
}

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st) { return cudaMemsetAsync(p, 0, bytes, st); }

}  // namespace ov

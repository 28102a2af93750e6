// Device side of libtp shared by the translation units that instantiate the
// tent kernel (one per space dimension) and the context code: the kernel
// arguments, the float-float arithmetic, the basis and congruence helpers,
// and the tent kernel template itself.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "tp_internal.h"
#include "tp_tc.cuh"

namespace cg = cooperative_groups;

namespace tp {

constexpr int kThreads = 256;      // of a CTA where two share an SM
constexpr int kThreadsWide = 512;  // where one CTA fills the SM's shared memory (16 warps hide more latency than 8)
constexpr int kMaxPairs = 768;   // Gram pairs nb (nb+1)/2 (dim U^p <= 38)
constexpr int kMaxLowPairs = 384;   // the same of the functions of degree <= p - 1 (at most 25: 2D p = 5)
constexpr int kMaxRefine = 40;   // refinement steps of the mixed path
constexpr long long kMaxSpin = 1LL << 20;   // bounded dependency wait: 2^20 polls (well under a second), then TP_ERR_TIMEOUT

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// arrays of a tent's patch in shared memory (KArgs::geo: offsets in doubles)
struct Geo {
  enum { X, XH, TB, TT, GB, GT, SDET, ISDET, GEL, GBF, FP, FSQ, FN, NTAU, EL, GRP, VID, FW, FG, FG2, NID, COUNT };
};

// a table in binary64 and as float-float pairs
struct RuleTab {
  const double* d;
  const float2* ff;
};

struct KArgs {
  int geo[Geo::COUNT];
  // nl: the functions of degree <= p - 1, first in the order; every derivative
  // lies in their span, so sums that meet the solution through v or sigma alone
  // (their moments and values, the Grams of the derivative terms) run over them
  int nb, nl, nmono, Q, nrhs, CH, mono_stride, ngmax;
  int ustride;                    // row stride of the U-values of a point in shared memory (nb rounded up to odd)
  // right-hand sides split over the cluster: CTA r of a tent's cluster owns
  // right-hand sides [r nrhs, (r + 1) nrhs) of the group (nrhs = per CTA) for
  // the data moments, the solve and the outflow, over all points of the
  // patch; the Grams stay split by points.  0: every CTA sees all nrhs.
  int rsplit;
  int p;                          // degree of U^p
  int mono_lv[kMaxP + 2];         // monomials of total degree d: [mono_lv[d], mono_lv[d+1])
  // U-value sums: basis functions in classes of equal term count (class with
  // ev_terms 0: one term of coefficient 1); class c is ev_order[ev_off[c] .. ev_off[c+1])
  int ev_ncls;
  int ev_off[kMaxEvCls + 1];
  int ev_terms[kMaxEvCls];
  int ev_loff[kMaxEvCls + 1];     // the same counting functions < nl only (first in each class)
  const int* ev_order;
  int64_t ne, n_bnd;
  double alpha, beta;
  const double* X;
  const int* elems;
  const double* cK;
  const double* elem_einv;    // per element: inverse of the edge matrix e (rows X_i - X_0), dim x dim
  const double* elem_sdet;    // per element: sqrt(|det e|)
  const double* elem_isdet;   // per element: 1 / sqrt(|det e|)
  const double* bary;     // Q * (dim+1)
  const double* wref;     // Q
  const double* sqw;      // Q, sqrt(wref)
  const float2* sqw_dd;   // Q, sqrt(wref) as a float-float pair
  const double* isqw;     // Q, 1 / sqrt(wref)
  const int* tent_v;
  const double* tent_ttop;
  const double* tent_tbot;
  const double* tent_ih;      // 1 / h
  const int* tent_hdr;        // per tent: v, record offsets (int, double), elements, Dirichlet and interface facets, materials, Neumann facets
  const int* vrec_i;          // per vertex: star record, ints (elements, facets)
  const double* vrec_d;       // per vertex: star record, doubles (x_v, speeds, coordinates, normals)
  const long long* tent_gdoff;
  const int* sp_ptr;
  const int* sp_mono;
  const double* sp_coef;
  const float2* sp_coef_dd;   // (hi, lo) binary32 pair of every sp_coef entry
  const int* mono_parent;
  const int* mono_var;
  // merged congruence tables of the top-face form (see tp_basis)
  const int* pair_ij;
  const int *cg_ptr, *cg_idx, *ch_ptr, *ch_idx;
  const float *cg_coef, *ch_coef;
  const int *ft_ptr, *ft_idx, *fm_ptr, *fm_idx;   // Dirichlet facet congruences (see tp_basis)
  const float *ft_coef, *fm_coef;
  const double *cg_coefd, *ch_coefd, *ft_coefd, *fm_coefd;   // the same coefficients in binary64
  double* tau;
  double* front;
  const double* gD;
  double* diss;               // per right-hand side: accumulated energy lost in the tents (nullptr: not tracked)
  // wave-speed gradient: the forward sweep stores each tent's solution
  // (xsave[(tent - xbase) * xs_stride + r * ngmax * nb + row], r over the
  // group's right-hand sides) when xsave is set; the reverse sweep reads it
  // back and adds dJ/dc per element into dJdc when dJdc is set; so with the
  // bottom front of each tent, fsave[((tent_el[tent] - fbase) * R + r * P) * Q C ..]
  // (tent_el: elements of the patches of all tents before; R, r: over the
  // group's right-hand sides)
  double* xsave;
  long long xbase, xs_stride;
  double* fsave;
  long long fbase;
  const long long* tent_el;
  double* dJdc;
  int off_yg;                 // shared memory of the gradient: y(x), y(x'), y(mu') and x
  // bounded waits and the solve's refinement: the dependency wait gives up
  // after max_spin polls (TP_ERR_TIMEOUT); a refinement that has not settled
  // after max_refine steps hands the tent to the direct binary64 LU;
  // solve_stats (kMaxRefine + 2 counters, or nullptr): [0] tents solved by
  // the direct LU, [1 + k] tents whose refinement settled after k steps
  long long max_spin;
  int max_refine;
  unsigned long long* solve_stats;
  // point outputs (forward sweep): the samples (probe point, output time)
  // that lie inside tent t are [probe_ptr[t], probe_ptr[t+1]) with the
  // probe's index, the time's index and the patch slot of its element; the
  // forward kernel writes U_h there: probe_out[(r * n_probe_t + k) * n_probe + j]
  const int* probe_ptr;        // nullptr: no point outputs
  const int* probe_j;
  const int* probe_k;
  const int* probe_slot;
  const double* probe_bary;   // per probe point: barycentric coordinates in its element
  const double* probe_t;      // output times
  int n_probe, n_probe_t;
  double* probe_out;
  int* status;
  long long* status_info;
  // persistent sweep: tent queue, completed tents per vertex, dependencies
  // (for tent t at v, [dep_ptr[t], dep_ptr[t+1]): how many tents of v and of
  // each of its neighbours, in the order of the star record, precede it)
  int* queue;
  int* done;
  const int* dep_ptr;
  const int* dep_need;
  const int* vt_ptr;          // per vertex w: its front times after 0, 1, .. of its tents, vt_tau[vt_ptr[w] ..]
  const double* vt_tau;
  const int* inject;          // per tent: completions that it waits for beyond those that come (tp_inject_wait; 0)
  int tent_beg;               // tents of the sweep's range: [tent_beg, tent_end)
  const int* queue_tent;      // tent at each queue position (level order, critical chains first)
  int tent_end;
  // shared-memory carve (offsets in doubles)
  const int* rel_ptr;
  const int* rel_src;
  const double* rel_fac;
  const int* relT_ptr;
  const int* relT_dst;
  const double* relT_fac;
  const float* rel_facf;      // relation factors (small integers) in binary32
  const float* relT_facf;
  int off_eq, off_z, off_x;                     // solve: scales, scaled residual, iterate
  int off_pt;                                   // per-point (that, xhat, scale) of the block-wide evaluation
  int keep_pts, off_keep;                       // kept U-values (scaled, both faces) of a CTA's slice
  int cb_pts;                                   // points of the data-coefficient buffer
  int ev_rows;                                  // points evaluated at a time into the kept rows
  // kept tents: the S-point rule of the face integrals (0: the front rule) and
  // the tables between its points and the front's (FaceRule: to_points, then
  // to_front), in shared memory at off_tf; raw_el elements' front data at a
  // time at off_raw
  int S, tf_stride, off_tf, raw_el, off_raw;
  RuleTab tf;
  RuleTab baryT, sqwT, s_baryT, s_sqwT;   // points (barycentric) and sqrt(w_ref) of the front rule and the S-point rule
  int off_rc;                                   // pivot rows (and columns) of the elimination, two of each
  int off_b, off_pg, off_ph, off_pgb, off_pm, off_pd, off_dd, off_sm, off_f, off_f2, off_fpm, off_del,
      off_u, off_mono, off_cb, off_gd, off_y, off_rd;
  // tensor-core contractions (mixed forward sweep with split right-hand
  // sides, single-material tents): the data moments and the outflow run as
  // exact digit products on tcgen05 (tp_tc.cuh); off_tc: their staging
  // (bf16 digit planes, in the region of the facet sums, which is dead in
  // the point passes before phase 2 and in the outflow), tc_cols
  // tensor-memory columns held per CTA
  int tc, off_tc, tc_cols;
};

__device__ __forceinline__ void flag_error(const KArgs& a, int code, long long info) {
  if (atomicCAS(a.status, 0, code) == 0) *a.status_info = info;
}

// gradient g of the linear function with increments dv[i] along the edges
// e[i] = X_{i+1} - X_0 (solves e g = dv); returns det(e)
template <int DIM>
__device__ __forceinline__ double lin_grad(const double (&e)[DIM][DIM], const double* dv, double* g) {
  if constexpr (DIM == 1) {
    g[0] = dv[0] / e[0][0];
    return e[0][0];
  } else if constexpr (DIM == 2) {
    const double det = e[0][0] * e[1][1] - e[0][1] * e[1][0];
    const double id = 1.0 / det;
    g[0] = (e[1][1] * dv[0] - e[0][1] * dv[1]) * id;
    g[1] = (-e[1][0] * dv[0] + e[0][0] * dv[1]) * id;
    return det;
  } else {
    // rows of e^-1^T: (e1 x e2, e2 x e0, e0 x e1) / det
    double c0[3], c1[3], c2[3];
    c0[0] = e[1][1] * e[2][2] - e[1][2] * e[2][1];
    c0[1] = e[1][2] * e[2][0] - e[1][0] * e[2][2];
    c0[2] = e[1][0] * e[2][1] - e[1][1] * e[2][0];
    c1[0] = e[2][1] * e[0][2] - e[2][2] * e[0][1];
    c1[1] = e[2][2] * e[0][0] - e[2][0] * e[0][2];
    c1[2] = e[2][0] * e[0][1] - e[2][1] * e[0][0];
    c2[0] = e[0][1] * e[1][2] - e[0][2] * e[1][1];
    c2[1] = e[0][2] * e[1][0] - e[0][0] * e[1][2];
    c2[2] = e[0][0] * e[1][1] - e[0][1] * e[1][0];
    const double det = e[0][0] * c0[0] + e[0][1] * c0[1] + e[0][2] * c0[2];
    const double id = 1.0 / det;
    for (int d = 0; d < 3; ++d) g[d] = (dv[0] * c0[d] + dv[1] * c1[d] + dv[2] * c2[d]) * id;
    return det;
  }
}

// determinant of a small symmetric Gram matrix
template <int DIM>
__device__ __forceinline__ double small_det(const double (&G)[DIM][DIM]) {
  if constexpr (DIM == 1) {
    return G[0][0];
  } else if constexpr (DIM == 2) {
    return G[0][0] * G[1][1] - G[0][1] * G[1][0];
  } else {
    return G[0][0] * (G[1][1] * G[2][2] - G[1][2] * G[2][1]) -
           G[0][1] * (G[1][0] * G[2][2] - G[1][2] * G[2][0]) +
           G[0][2] * (G[1][0] * G[2][1] - G[1][1] * G[2][0]);
  }
}

// ---------------------------------------------------------------------------
// Arithmetic used by the tent kernel.  The FP64 path computes in binary64.
// The mixed path computes the assembly, the refinement residual and the
// outflow in float-float ("double-float") arithmetic on the binary32 pipes,
// which GB300 runs ~58x faster than binary64: a value is an unevaluated sum
// hi + lo of two binary32 numbers (|lo| <= ulp(hi)/2, ~48 significant bits),
// built from the error-free transformations TwoSum (Knuth), FastTwoSum
// (Dekker) and TwoProd through the fused multiply-add.  The intrinsics
// __fadd_rn/__fsub_rn/__fmul_rn keep the compiler from contracting them.
// ---------------------------------------------------------------------------
struct dd {
  float hi, lo;
};

__device__ __forceinline__ dd two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ dd fast_two_sum(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  dd s = two_sum(a.hi, b.hi);
  const dd t = two_sum(a.lo, b.lo);
  s = fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return fast_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return fast_two_sum(p, e);
}
__device__ __forceinline__ dd dd_mulf(dd a, float f) {   // f exact in binary32
  const float p = __fmul_rn(a.hi, f);
  float e = fmaf(a.hi, f, -p);
  e = fmaf(a.lo, f, e);
  return fast_two_sum(p, e);
}

// float-float split of a binary64 value, hi = x rounded to binary32 and
// lo = x - hi rounded, by integer operations on its bits (the binary64 unit,
// ~2 operations per clock per SM on this GPU, stays free); values outside
// [2^-74, 2^126) in magnitude (where lo would leave binary32's normal range)
// take the conversion instructions.  Equal in value to the conversions (a
// zero lo may carry the sign of x).
__device__ __forceinline__ dd dd_split(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((u >> 52) & 0x7FF) - 1023;
  if (E < -74 || E > 125) {
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - (double)h)};
  }
  const unsigned long long frac = u & ((1ull << 52) - 1);
  const unsigned int low = (unsigned int)(frac & ((1u << 29) - 1));   // the 29 bits below binary32's fraction
  unsigned int hb = ((unsigned int)(u >> 63) << 31) | ((unsigned int)(E + 127) << 23) | (unsigned int)(frac >> 29);
  const bool up = low > (1u << 28) || (low == (1u << 28) && (hb & 1u));
  hb += up ? 1u : 0u;   // a carry out of the fraction raises the exponent
  // lo = x - hi = +-(low - up 2^29) 2^(E - 52), |.| <= 2^28 units
  const int r = (int)low - (up ? (1 << 29) : 0);
  const int k = E - 52, k1 = k / 2;
  float lo = __fmul_rn(__fmul_rn(__int2float_rn(r), __uint_as_float((unsigned int)(127 + k1) << 23)),
                       __uint_as_float((unsigned int)(127 + k - k1) << 23));
  if (u >> 63) lo = -lo;
  return {__uint_as_float(hb), lo};
}

// 1/x of a float-float value: Newton step r + r (1 - x r) from the hardware's
// approximate binary32 reciprocal of the leading part (about 1 ulp; 24 -> 48
// bits).  The inverse it serves is refined against A, so its last bits do not
// matter, and the correctly rounded reciprocal costs several times as long in
// the elimination's chain of pivots
__device__ __forceinline__ dd dd_rcp(dd x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.hi));
  const float e = fmaf(-x.lo, r, fmaf(-x.hi, r, 1.f));
  return fast_two_sum(r, __fmul_rn(r, e));
}

template <typename T>
struct Ar;

template <>
struct Ar<double> {
  static __device__ __forceinline__ float hi(double x) { return (float)x; }
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double one() { return 1.0; }
  static __device__ __forceinline__ double from(double x) { return x; }
  static __device__ __forceinline__ double to(double x) { return x; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double sub(double a, double b) { return a - b; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  // accumulation of a long sum of products (see the float-float version)
  static __device__ __forceinline__ double acc(double s, double a, double b) { return ::fma(a, b, s); }
  static __device__ __forceinline__ double accf(double s, double a, float f) { return ::fma(a, (double)f, s); }
  static __device__ __forceinline__ double accn(double s, double a, double b) { return ::fma(-a, b, s); }
  static __device__ __forceinline__ double norm(double s) { return s; }
  static __device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
  // x s as a float-float pair for a power of two s, and back
  static __device__ __forceinline__ dd scaled(double x, float s) { return dd_split(x * (double)s); }
  static __device__ __forceinline__ double of(dd x) { return (double)x.hi + (double)x.lo; }
  static __device__ __forceinline__ double coef(const KArgs& a, int e);
};

template <>
struct Ar<dd> {
  static __device__ __forceinline__ float hi(dd x) { return x.hi; }
  static __device__ __forceinline__ dd zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ dd one() { return {1.f, 0.f}; }
  static __device__ __forceinline__ dd from(double x) {
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - (double)h)};
  }
  static __device__ __forceinline__ double to(dd x) { return (double)x.hi + (double)x.lo; }
  static __device__ __forceinline__ dd add(dd a, dd b) { return dd_add(a, b); }
  static __device__ __forceinline__ dd sub(dd a, dd b) { return dd_add(a, {-b.hi, -b.lo}); }
  static __device__ __forceinline__ dd mul(dd a, dd b) { return dd_mul(a, b); }
  // s += a b for a long sum of products, compensated in the manner of Ogita,
  // Rump and Oishi's Dot2: s = (p, e) holds the running binary32 sum p and
  // the sum e of all rounding errors (of the products, exact by fmaf, and of
  // the additions, exact by TwoSum); the pair is not normalised until norm().
  static __device__ __forceinline__ dd acc(dd s, dd a, dd b) {
    const float h = __fmul_rn(a.hi, b.hi);
    float r = fmaf(a.hi, b.hi, -h);
    r = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, r));
    const float pn = __fadd_rn(s.hi, h);
    const float bb = __fsub_rn(pn, s.hi);
    const float q = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(pn, bb)), __fsub_rn(h, bb));
    return {pn, __fadd_rn(s.lo, __fadd_rn(q, r))};
  }
  static __device__ __forceinline__ dd accf(dd s, dd a, float f) {   // s += a f, f exact in binary32
    const float h = __fmul_rn(a.hi, f);
    const float r = fmaf(a.lo, f, fmaf(a.hi, f, -h));
    const float pn = __fadd_rn(s.hi, h);
    const float bb = __fsub_rn(pn, s.hi);
    const float q = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(pn, bb)), __fsub_rn(h, bb));
    return {pn, __fadd_rn(s.lo, __fadd_rn(q, r))};
  }
  static __device__ __forceinline__ dd accn(dd s, dd a, dd b) { return acc(s, {-a.hi, -a.lo}, b); }   // s -= a b
  static __device__ __forceinline__ dd norm(dd s) { return fast_two_sum(s.hi, s.lo); }
  static __device__ __forceinline__ dd fma(dd a, dd b, dd c) { return dd_add(dd_mul(a, b), c); }
  static __device__ __forceinline__ dd scaled(dd x, float s) { return {__fmul_rn(x.hi, s), __fmul_rn(x.lo, s)}; }
  static __device__ __forceinline__ dd of(dd x) { return x; }
  static __device__ __forceinline__ dd coef(const KArgs& a, int e);
};

__device__ __forceinline__ double Ar<double>::coef(const KArgs& a, int e) { return __ldg(a.sp_coef + e); }
__device__ __forceinline__ dd Ar<dd>::coef(const KArgs& a, int e) {
  const float2 c = __ldg(a.sp_coef_dd + e);
  return {c.x, c.y};
}

// U-values at npt points with the whole block: the points' (that, xhat_1..xhat_n,
// scale) are in pt[q * (DIM + 2)]; one pass per monomial degree (m = parent
// monomial times one variable), then the sparse sums u_j = scale * sum c m.
// Monomials go to m[q * mono_stride], U-values to u[q * nb].  Callers write pt
// before the call; the first and last statements that touch shared memory
// are separated from them by barriers.
// LOW: only the functions < nl (degree <= p - 1)
template <int DIM, typename T, bool SCALE = true, bool LOW = false>
__device__ __forceinline__ void eval_uvalues_block(const KArgs& a, int npt, const T* pt, T* m, T* u) {
  // Each thread takes one monomial (one basis function) at four points, so
  // that four independent products are in flight per table lookup.
  const int tid = threadIdx.x, ms = a.mono_stride, nfn = LOW ? a.nl : a.nb;
  const int* const off = LOW ? a.ev_loff : a.ev_off;
  const int nq4 = (npt + 3) >> 2;
  // the constant monomial carries the scale, so every monomial and U-value is scaled
  for (int q = tid; q < npt; q += blockDim.x) m[q * ms] = SCALE ? pt[q * (DIM + 2) + DIM + 1] : Ar<T>::one();
  for (int d = 1; d <= (LOW ? a.p - 1 : a.p); ++d) {
    __syncthreads();   // pt, and the monomials of degree d - 1
    const int g0 = a.mono_lv[d], cnt = a.mono_lv[d + 1] - g0;
    for (int id = tid; id < cnt * nq4; id += blockDim.x) {
      const int g = g0 + id % cnt, q0 = (id / cnt) << 2;
      const int par = __ldg(a.mono_parent + g), vr = __ldg(a.mono_var + g);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int q = min(q0 + t, npt - 1);
        const T v = Ar<T>::mul(m[q * ms + par], pt[q * (DIM + 2) + vr]);
        if (q0 + t < npt) m[q * ms + g] = v;
      }
    }
  }
  __syncthreads();
  // items (function, four points) class after class, so that the lanes of a
  // warp run loops of one length; a one-term function of coefficient 1 is a copy
  for (int id = tid; id < nfn * nq4; id += blockDim.x) {
    int c = 0;
    while (id >= off[c + 1] * nq4) ++c;
    const int nj = off[c + 1] - off[c], loc = id - off[c] * nq4;
    const int j = __ldg(a.ev_order + a.ev_off[c] + loc % nj), q0 = (loc / nj) << 2;
    const int e0 = __ldg(a.sp_ptr + j * (DIM + 2)), e1 = __ldg(a.sp_ptr + j * (DIM + 2) + 1);
    int qq[4];
    T acc[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      qq[t] = min(q0 + t, npt - 1);
      acc[t] = Ar<T>::zero();
    }
    if (a.ev_terms[c] == 0) {
      const int g = __ldg(a.sp_mono + e0);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (q0 + t < npt) u[qq[t] * a.ustride + j] = m[qq[t] * ms + g];
      continue;
    }
    for (int e = e0; e < e1; ++e) {
      const T c = Ar<T>::coef(a, e);
      const int g = __ldg(a.sp_mono + e);
#pragma unroll
      for (int t = 0; t < 4; ++t) acc[t] = Ar<T>::acc(acc[t], c, m[qq[t] * ms + g]);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (q0 + t < npt) u[qq[t] * a.ustride + j] = Ar<T>::norm(acc[t]);
  }
  __syncthreads();
}

// entry of a table in the path's arithmetic, and the table of a rule (KArgs: binary64, float-float)
__device__ __forceinline__ double tab(const double* p) { return __ldg(p); }
__device__ __forceinline__ dd tab(const dd* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
template <typename T>
__device__ __forceinline__ const T* rule_tab(const RuleTab& t) {
  if constexpr (std::is_same<T, dd>::value) return reinterpret_cast<const dd*>(t.ff);
  else return t.d;
}

// s + y f for a factor f of a table of small exact numbers (derivative
// relations, merged congruence tables): binary64 reads the table's binary64
// copy and takes one fused multiply-add; float-float reads the binary32 copy
// (add: exact product and float-float sum; acc: a compensated long-sum step)
template <typename T>
struct Fac;
template <>
struct Fac<double> {
  static __device__ __forceinline__ double add(double s, double y, const float*, const double* fd, int e) {
    return ::fma(y, __ldg(fd + e), s);
  }
  static __device__ __forceinline__ double acc(double s, double y, const float*, const double* fd, int e) {
    return ::fma(y, __ldg(fd + e), s);
  }
};
template <>
struct Fac<dd> {
  static __device__ __forceinline__ dd add(dd s, dd y, const float* ff, const double*, int e) {
    return dd_add(s, dd_mulf(y, __ldg(ff + e)));
  }
  static __device__ __forceinline__ dd acc(dd s, dd y, const float* ff, const double*, int e) {
    return Ar<dd>::accf(s, y, __ldg(ff + e));
  }
};

// butterfly exchange of a value of the path's arithmetic within a warp
__device__ __forceinline__ double shfl_xor_t(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ dd shfl_xor_t(dd v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// packed index of (i, j), in the order of tp_basis
__device__ __forceinline__ int pair_index(int i, int j) {
  const int lo = min(i, j), hi = max(i, j);
  return hi * (hi + 1) / 2 + lo;
}

// (D_var y)_i for a vector y
template <int DIM, typename T>
__device__ __forceinline__ T rel_apply(const KArgs& a, int i, int var, const T* y) {
  const int e0 = __ldg(a.rel_ptr + i * (DIM + 1) + var), e1 = __ldg(a.rel_ptr + i * (DIM + 1) + var + 1);
  T s = Ar<T>::zero();
  for (int e = e0; e < e1; ++e) s = Fac<T>::add(s, y[__ldg(a.rel_src + e)], a.rel_facf, a.rel_fac, e);
  return s;
}

// (D_var^T y)_k through the transposed table
template <int DIM, typename T>
__device__ __forceinline__ T relT_apply(const KArgs& a, int k, int var, const T* y) {
  const int e0 = __ldg(a.relT_ptr + k * (DIM + 1) + var), e1 = __ldg(a.relT_ptr + k * (DIM + 1) + var + 1);
  T s = Ar<T>::zero();
  for (int e = e0; e < e1; ++e) s = Fac<T>::add(s, y[__ldg(a.relT_dst + e)], a.relT_facf, a.relT_fac, e);
  return s;
}

// power of two nearest below 1 / sqrt(d) (within a factor of two; exact scaling)
__device__ __forceinline__ float pow2_rsqrt(float d) {
  const int e = (int)((__float_as_uint(d) >> 23) & 0xFF) - 127;
  return __uint_as_float((unsigned int)(127 - (e >> 1)) << 23);
}

// 1/x by two Newton-Raphson steps r <- r + r (1 - x r) from the binary32
// reciprocal (quadratic convergence: 24 -> 48 -> 96 bits); falls back to the
// division outside the binary32 range.
__device__ __forceinline__ double recip(double x) {
  const double ax = fabs(x);
  if (!(ax > 1e-30 && ax < 1e30)) return 1.0 / x;
  double r = (double)__frcp_rn((float)x);
  double e = fma(-x, r, 1.0);
  r = fma(r, e, r);
  e = fma(-x, r, 1.0);
  return fma(r, e, r);
}

// One tent per thread-block cluster of CS CTAs (CS = gridDim.x / tents in the
// launch, 1..8).  Each CTA takes a slice of the patch's points.
//
// Materials (Section 4.2).  The patch elements are grouped by wave speed; each
// group g carries its own polynomial x_g in U^p mapped with its own c_g
// (Remark 3.1), so the tent system has ng*nb unknowns.
//
// Assembly through Grams of U-values.  With u the vector of the nb U-values
// at a point and the exact derivative maps of U^p, v = (c/h) D_t u,
// sigma_m = -(1/h) D_m u, the top-face form of group g summed over its points is
//   A_top = h^-2 [ D_t G D_t^T + sum_m D_m G D_m^T + c sum_m (D_m H_m D_t^T + D_t H_m D_m^T) ],
//   G = sum_q w u u^T,  H_m = sum_K g_{K,m} G_K  (g = top front gradient on K),
// the recovery term is A_bot = sum_q w u_b u_b^T, the bottom data give
//   b = gamma + (c/h) D_t alpha - (1/h) sum_m D_m beta_m
// with moments gamma = sum w U_b u_b, alpha = sum w (c^-2 v_b - s_b.g_b) u_b,
// beta_m = sum w (s_b,m - v_b g_b,m) u_b.  A Dirichlet facet with normal n
// adds A_D = (c/h) D_t F E^T, b_D = E' delta, F = sum w u u^T,
// delta = sum w g_D u, E = alpha_D (c/h) D_t - (1/h) D_n, E' = alpha_D (c/h) D_t + (1/h) D_n,
// D_n = sum_m n_m D_m.  A Neumann facet (sigma.n = g_N) adds
// A_N = -(c/h^2) D_n F D_t^T + (beta/h^2) D_n F D_n^T and
// b_N = -(c/h) D_t delta - (beta/h) D_n delta, delta = sum w g_N u (eq. 4.1; the
// code is compiled in only when NEU).  A time-like facet between groups + and - (normal n out
// of +) adds, for test side t and trial side s (signs s_+ = 1, s_- = -1),
//   A^{ts} = s_t h^-2 [ -c_s/2 D_n F^{ts} D_t^T - c_t/2 D_t F^{ts} D_n^T ]
//          + s_t s_s h^-2 [ alpha c_s c_t D_t F^{ts} D_t^T + beta D_n F^{ts} D_n^T ],
//   F^{ts} = sum w u^t u^s^T,
// the {v}[[tau]]_N + {s}.[[w]]_N + alpha [[v]]_N.[[w]]_N + beta [[s]]_N [[tau]]_N
// terms of eq. (2.5).  Every CTA publishes its partial Grams and moments;
// after a cluster barrier every CTA sums them in rank order, forms A and b,
// solves, and writes the outflow of its slice.
//
// MIXED = false: assembly, residual and outflow in binary64; MIXED = true:
// in float-float.  Both: A is equilibrated (D A D, D powers of two near
// |diag A|^-1/2), inverted in float-float and the solution refined against A in
// the path's precision until the correction stops shrinking; a refinement that
// does not settle falls back to a direct binary64 LU.
//
// ADJ = true: the adjoint tent map (reverse sweep).  With g_D = 0 a tent maps
// its bottom values linearly to its top values, b = B f_bot, A x = b,
// f_top = E x; the adjoint takes lambda at the top points to
// mu = A^-T (E^T lambda) and lambda_bot = B^T mu at the bottom points.  In the
// U-value form E^T lambda = zeta_U + (c/h) D_t zeta_v - (1/h) sum_m D_m zeta_m,
// zeta = sum_q lambda_q u_q over the top points (the moment formula of b), and
// B^T mu at a bottom point is w (s0, c^-2 s_t - g_b.s, s_m - g_b,m s_t) with
// s0 = u.mu, s_t = (c/h) u.D_t^T mu, s_m = -(1/h) u.D_m^T mu.  The front and
// time arrays of the arguments are then the adjoint state (tau runs backwards).
//
// PERSIST = true: one resident grid of clusters; each cluster takes the next
// tent of the sorted list from a queue, waits (bounded) until the tents of its
// vertex and neighbours that precede it in level are complete, solves it and
// publishes its completion.  Tents leave the queue in level order, so every
// awaited tent is held by a running cluster: no launch per level, and a tent
// starts as soon as its own inputs are ready.  The front and the front times
// are read through L2 (ld.global.cg) so that no stale L1 line is used.
//
// What bounds a sweep with few right-hand sides is the chain of dependent
// tents (levels times what a tent does between its wait and its publication)
// or, on wide levels, the work of all tents over the resident CTAs.  The tent
// matrix depends on the front times alone, which the tents fix, so the
// geometry, the U-values, A and its inverse come before the wait (with split
// right-hand sides the Grams alone): the chain keeps the moments, b, the solve
// and the outflow.  2D p = 4, 968 triangles,
// one column: 18.5 -> 9.9 ms binary64, 27.0 -> 7.8 ms mixed (mixed with the S-point
// rule and the float-float inverse below).
template <int DIM, bool MIXED, bool ADJ, bool PERSIST, bool NEU, bool SPLIT, bool TC, bool WIDE>
__global__ void __launch_bounds__(WIDE ? kThreadsWide : kThreads, WIDE ? 1 : 2) k_layer(const KArgs a, const int tent0) {
  static_assert(!TC || (MIXED && !ADJ && SPLIT), "tensor-core contractions: mixed forward sweep, split right-hand sides");
  constexpr int NT = WIDE ? kThreadsWide : kThreads, NW = NT / 32;   // threads and warps of a CTA
  constexpr int kMaxPair = (kMaxPairs + NT - 1) / NT;            // Gram pairs per thread
  constexpr int kMaxLow = (kMaxLowPairs + NT - 1) / NT;          // of functions < nl
  using T = typename std::conditional<MIXED, dd, double>::type;
  using R = Ar<T>;
  // sweeps that may take the S-point rule of the face integrals.  In binary64 it
  // is taken at 3D p = 3 alone: there its errors are those of the front rule
  // (0.90 to 1.08 of them over 24 outputs, one energy 1.13), at 2D p = 2 to 4 and 3D
  // p = 1, 2 a reverse sweep's are 1.5 to 3.7 times as large (every tent repeats
  // the same roundings of its points and weights), an energy's up to 4 times.  In
  // float-float at 2D p = 4, 5 and 3D p = 2, 3: 0.6 to 1.2 of the front rule's
  constexpr bool RULE = !SPLIT && DIM > 1 && (MIXED || DIM == 3);
  constexpr int NV = DIM + 1;   // vertices per element
  constexpr int C = DIM + 2;    // U, v, sigma  (and gamma, alpha, beta_m moments)
  extern __shared__ __align__(16) double sm[];
  __shared__ int s_P, s_v, s_nfac, s_nif, s_ng, s_nneu;
  __shared__ double s_ttop, s_tbot, s_tc, s_ih;
  __shared__ double s_gc[tp::kMaxGroups], s_gic2[tp::kMaxGroups];   // speeds and 1/c^2 of the materials
  __shared__ double s_xv[DIM];
  // the patch, in dynamic shared memory sized for the context's largest star
  // (in the order of Geo): per element its vertices' coordinates, the same
  // scaled to the tent's reference coordinates, bottom and top times, front gradients, sqrt|det| and its reciprocal, the
  // tent's wave-speed gradient and, mixed path, g_bot (DIM) and sqrt|det| (slot
  // DIM) as float-float pairs; per facet its simplex (x, t), sqrt(n! volume)
  // and normal; the front times of v and its neighbours; then integers: element
  // id and material, the place of each of its vertices in the list of v and its
  // neighbours; of a facet the same (slots 2..; for boundary facets slot 0
  // holds the block of their data among the vertex's boundary facets) and its
  // groups (Dirichlet: one; interface: +, -); the neighbour list's vertex ids
  double(*const s_X)[NV][DIM] = reinterpret_cast<double(*)[NV][DIM]>(sm + a.geo[Geo::X]);
  T(*const s_xh)[NV][DIM + 2] = reinterpret_cast<T(*)[NV][DIM + 2]>(sm + a.geo[Geo::XH]);
  double(*const s_tb)[NV] = reinterpret_cast<double(*)[NV]>(sm + a.geo[Geo::TB]);
  double(*const s_tt)[NV] = reinterpret_cast<double(*)[NV]>(sm + a.geo[Geo::TT]);
  double(*const s_gb)[DIM] = reinterpret_cast<double(*)[DIM]>(sm + a.geo[Geo::GB]);
  double(*const s_gt)[DIM] = reinterpret_cast<double(*)[DIM]>(sm + a.geo[Geo::GT]);
  double* const s_sdet = sm + a.geo[Geo::SDET];
  double* const s_isdet = sm + a.geo[Geo::ISDET];
  double* const s_gel = sm + a.geo[Geo::GEL];
  float2(*const s_gbf)[DIM + 1] = reinterpret_cast<float2(*)[DIM + 1]>(sm + a.geo[Geo::GBF]);
  double(*const s_fP)[NV][DIM + 1] = reinterpret_cast<double(*)[NV][DIM + 1]>(sm + a.geo[Geo::FP]);
  double* const s_fsq = sm + a.geo[Geo::FSQ];
  double(*const s_fn)[DIM] = reinterpret_cast<double(*)[DIM]>(sm + a.geo[Geo::FN]);
  double* const s_ntau = sm + a.geo[Geo::NTAU];
  int* const s_el = reinterpret_cast<int*>(sm + a.geo[Geo::EL]);
  int* const s_grp = reinterpret_cast<int*>(sm + a.geo[Geo::GRP]);
  int(*const s_vid)[NV] = reinterpret_cast<int(*)[NV]>(sm + a.geo[Geo::VID]);
  int(*const s_fw)[NV] = reinterpret_cast<int(*)[NV]>(sm + a.geo[Geo::FW]);
  int* const s_fg = reinterpret_cast<int*>(sm + a.geo[Geo::FG]);
  int* const s_fg2 = reinterpret_cast<int*>(sm + a.geo[Geo::FG2]);
  int* const s_nid = reinterpret_cast<int*>(sm + a.geo[Geo::NID]);
  __shared__ float2 s_gic2f[tp::kMaxGroups];   // mixed path: c^-2 of each material as a float-float pair
  __shared__ int s_ge0[tp::kMaxGroups + 1];   // elements of material g: [s_ge0[g], s_ge0[g + 1])
  __shared__ int s_piv;
  __shared__ float s_red[2][NW];

  __shared__ int s_tent, s_bad;
  // tensor-core contractions: tensor-memory base, completion barrier of the
  // MMAs, binary exponents of the rows of A (0) and the columns of B (1)
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_tcbar;
  __shared__ int s_tce[2][TC ? tc::kMaxM : 1];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int CS = (int)cluster.num_blocks();
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  constexpr bool kTC = TC;
  uint32_t tc_phase = 0;                // parity of the next completion of s_tcbar
  if constexpr (kTC) {
    if (warp == 0) tc::tmem_alloc(&s_tmem, a.tc_cols);
    if (tid == 0) tc::mbar_init(&s_tcbar, 1);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
  }
  if (RULE && a.S > 0) {   // (ordered before its first use by the first tent's barriers)
    T* sTF = reinterpret_cast<T*>(sm + a.off_tf);
    for (int id = tid; id < 2 * a.S * a.tf_stride; id += NT) {
      sTF[id] = tab(rule_tab<T>(a.tf) + id);
    }
  }
  // barrier of the cluster (a cluster of one CTA: the block's)
  auto csync = [&]() {
    if (CS > 1) cluster.sync();
    else __syncthreads();
  };
  // (rank 0 stores the first tent into the other CTAs' shared memory, which
  // may be written only once they run)
  if (PERSIST && CS > 1) cluster.sync();
  for (;;) {
  int tent;
  if constexpr (PERSIST) {
    // rank 0 takes the next tent and stores its index into every CTA of the
    // cluster (each CTA read its copy of the previous index several cluster
    // barriers ago)
    if (tid == 0) s_bad = 0;
    if (rank == 0 && tid == 0) {
      const int pos = atomicAdd(a.queue, 1);
      // (the reverse sweep takes the positions from the end)
      const int t_ = pos < a.tent_end ? __ldg(a.queue_tent + (ADJ ? a.tent_beg + a.tent_end - 1 - pos : pos)) : a.tent_end;
      if (CS > 1)
        for (int r = 0; r < CS; ++r) *cluster.map_shared_rank(&s_tent, r) = t_;
      else
        s_tent = t_;
    }
    csync();
    tent = s_tent;
    if (tent >= a.tent_end) break;
  } else {
    tent = tent0 + blockIdx.x / CS;
  }
  const int nb = a.nb, nl = a.nl, Q = a.Q, nrhs = a.nrhs, CH = a.CH, NG = a.ngmax;
  const int us = a.ustride;   // row stride of the U-values in shared memory (odd: no bank conflicts between points)
  // this CTA's right-hand sides (all of the group unless they are split over the cluster)
  constexpr bool rsplit = SPLIT;
  double* const front = a.front + (rsplit ? (size_t)rank * nrhs * a.ne * Q * C : 0);
  const double* const gD = a.gD != nullptr ? a.gD + (rsplit ? (size_t)rank * nrhs * a.n_bnd : 0) : nullptr;
  const int npair = nb * (nb + 1) / 2, npl = nl * (nl + 1) / 2;
  const int nmom = nrhs * C * nb;
  T* sA = reinterpret_cast<T*>(sm);                  // N*N        assembled A, then LU factors
  T* sb = reinterpret_cast<T*>(sm + a.off_b);        // nrhs*N     assembled b, then x
  T* sPG = reinterpret_cast<T*>(sm + a.off_pg);      // NG*npl     this CTA: G (top) per group
  T* sPH = reinterpret_cast<T*>(sm + a.off_ph);      // NG*DIM*npl    H_m
  T* sPGb = reinterpret_cast<T*>(sm + a.off_pgb);    // NG*npair   G (bottom, recovery)
  T* sPM = reinterpret_cast<T*>(sm + a.off_pm);      // NG*nmom    moments (gamma, alpha, beta_m) per rhs, this CTA
  T* sSG = sPG;                                      // the same summed over the cluster, in place
  T* sSM = reinterpret_cast<T*>(sm + a.off_sm);      // NG*nmom    summed moments (in place of sPM)
  T* sF = reinterpret_cast<T*>(sm + a.off_f);        // npl        facet Gram (+ side)
  T* sF2 = reinterpret_cast<T*>(sm + a.off_f2);      // npl        facet Gram (- side)
  T* sFpm = reinterpret_cast<T*>(sm + a.off_fpm);    // nl*nl      facet Gram (+ test, - trial)
  T* sDel = reinterpret_cast<T*>(sm + a.off_del);    // nrhs*nl    facet moments delta
  T* sU = reinterpret_cast<T*>(sm + a.off_u);        // 2*CH*nb    U-values (scaled) per (side, point)
  T* sPt = reinterpret_cast<T*>(sm + a.off_pt);      // 2*CH*(DIM+2)  (that, xhat, scale) per point
  T* sM = reinterpret_cast<T*>(sm + a.off_mono);     // 2*CH*mono_stride
  T* sCB = reinterpret_cast<T*>(sm + a.off_cb);      // nrhs*C*(CH+1) data coefficients, point fastest
  const int cbs = a.cb_pts | 1;                      // their row stride (odd: no bank conflicts along a row)
  T* sGd = reinterpret_cast<T*>(sm + a.off_gd);      // CH*nrhs    Dirichlet data coefficients
  T* sY = reinterpret_cast<T*>(sm + a.off_y);        // NG*nmom    outflow coefficient vectors (sPM, dead after the congruence)
  double* sRD = sm + a.off_rd;                       // N          reciprocal pivots (binary64 path)

  // ---------------- phase 0: tent, materials and patch geometry ----------------
  // (a) what does not depend on earlier tents: vertex star, coordinates,
  // materials, facets; in the dataflow sweep it is fetched while the tents
  // this one depends on may still be running
  // one round of loads: the tent's header, then its vertex's star record
  const int4 h0 = __ldg(reinterpret_cast<const int4*>(a.tent_hdr) + 2 * (size_t)tent);
  const int4 h1 = __ldg(reinterpret_cast<const int4*>(a.tent_hdr) + 2 * (size_t)tent + 1);
  const int v = h0.x, P = h0.w, nfac = h1.x, nif = h1.y, ng = h1.z;   // Neumann facets: h1.w, s_nneu
  if (tid == 0) {
    s_v = v;
    s_P = P;
    s_ttop = a.tent_ttop[tent];
    s_ih = a.tent_ih[tent];
    s_nfac = nfac;
    s_nif = nif;
    s_ng = ng;
    s_nneu = h1.w;
  }
  const int N = ng * nb;
  const bool extra = (nfac > 0 || nif > 0 || (NEU && h1.w > 0));
  {
    const int* ri = a.vrec_i + h0.y;
    const double* rd = a.vrec_d + h0.z;
    if (tid < DIM) s_xv[tid] = __ldg(rd + tid);
    if (tid < ng) {
      s_gc[tid] = __ldg(rd + DIM + tid);
      s_gic2[tid] = __ldg(rd + DIM + tp::kMaxGroups + tid);
      if constexpr (MIXED) {
        const T g2 = R::from(s_gic2[tid]);
        s_gic2f[tid] = make_float2(g2.hi, g2.lo);
      }
    }
    const double* rX = rd + DIM + 2 * tp::kMaxGroups;
    for (int k = tid; k < P; k += blockDim.x) {
      s_el[k] = __ldg(ri + k * (2 + NV));
      const int gk = __ldg(ri + k * (2 + NV) + 1);   // (elements are sorted by material)
      s_grp[k] = gk;
      if (k == 0 || __ldg(ri + (k - 1) * (2 + NV) + 1) != gk) s_ge0[gk] = k;
      for (int i = 0; i < NV; ++i) {
        s_vid[k][i] = __ldg(ri + k * (2 + NV) + 2 + i);
        for (int d = 0; d < DIM; ++d) s_X[k][i][d] = __ldg(rX + (k * NV + i) * DIM + d);
      }
    }
    // vertical face simplices (x_v, t_bot), (x_v, t_top), (x_w, tau_w): Dirichlet
    // facets first, then the time-like interface facets, then Neumann facets
    const int* rfi = ri + P * (2 + NV);
    const int nfa = nfac + nif + h1.w, d0 = __ldg(a.dep_ptr + tent), nn = __ldg(a.dep_ptr + tent + 1) - d0;
    for (int e = tid; e < nn; e += blockDim.x) {
      const int w = __ldg(rfi + nfa * (NV + 3) + e);
      s_nid[e] = w;
      // the front time of w when this tent's turn comes: fixed by the tents alone
      if (PERSIST) s_ntau[e] = __ldg(a.vt_tau + __ldg(a.vt_ptr + w) + __ldg(a.dep_need + d0 + e));
    }
    if (tid < ng + 1 && tid == ng) s_ge0[ng] = P;
    const double* rfd = rX + P * NV * DIM;
    for (int f = tid; f < nfac + nif + (NEU ? h1.w : 0); f += blockDim.x) {
      for (int i = 2; i < NV; ++i) s_fw[f][i] = __ldg(rfi + f * (NV + 3) + i);
      s_fg[f] = __ldg(rfi + f * (NV + 3) + NV);
      s_fg2[f] = __ldg(rfi + f * (NV + 3) + NV + 1);
      s_fw[f][0] = __ldg(rfi + f * (NV + 3) + NV + 2);
      const double* fd = rfd + f * (DIM + NV * DIM);
      for (int d = 0; d < DIM; ++d) s_fn[f][d] = __ldg(fd + d);
      for (int i = 0; i < NV; ++i)
        for (int d = 0; d < DIM; ++d) s_fP[f][i][d] = __ldg(fd + DIM + i * DIM + d);
    }
  }
  const int d0_ = __ldg(a.dep_ptr + tent), nn_ = __ldg(a.dep_ptr + tent + 1) - d0_;
  // the earlier tents of this vertex and its neighbours must be complete:
  // every CTA of a tent publishes its own completion, so a vertex whose
  // first `need` tents are done has a count of need * CS; each CTA waits
  // for (and acquires) the counts itself
  auto wait_deps = [&]() {
    if constexpr (PERSIST) {
      const int extra_ = ADJ ? 0 : __ldg(a.inject + tent);
      for (int e = tid; e < nn_; e += blockDim.x) {
        const int w = s_nid[e];
        int before = __ldg(a.dep_need + d0_ + e);
        if constexpr (ADJ)   // the reverse sweep waits for the tents of w that follow this one
          before = __ldg(a.vt_ptr + w + 1) - __ldg(a.vt_ptr + w) - 1 - before - (e == 0 ? 1 : 0);
        if (before == 0) continue;
        const int need = (before + extra_) * CS;
        long long spins = 0;
        while (ld_acquire(a.done + w) < need) {
          if (++spins > a.max_spin) {
            flag_error(a, TP_ERR_TIMEOUT, tent);
            break;
          }
          // once any tent has flagged an error the sweep's result is void:
          // stop waiting so that the launch ends promptly
          if ((spins & 255) == 0 && ld_acquire(a.status) != 0) break;
          __nanosleep(32);
        }
      }
      __syncthreads();
    }
  };
  // The tent matrix depends on the front times only, and those are fixed by
  // the tents: in the dataflow sweep a tent is assembled and inverted from
  // the tabulated times while the tents it waits for still run, and only the
  // data of the bottom front, the solve and the outflow follow the wait.  A
  // front whose times are not the tabulated ones (tp_set_front with others)
  // is found after the wait, and the tent assembled again from its own.
  // (`real`: the times are those of the front)
  const int slice_el = (P + CS - 1) / CS;   // a CTA's share of the patch: whole elements
  const bool srule = RULE && a.S > 0;
  const int QK = srule ? a.S : Q;           // points per element of a kept tent
  const bool kept = !SPLIT && slice_el * QK <= a.keep_pts;
  bool real = !PERSIST;
  __syncthreads();
  // after the wait: s_bad of every CTA of the cluster is set where a time
  // used is not the front's (read after the next cluster barrier, so that the
  // CTAs decide alike)
  auto check_times = [&]() {
    if constexpr (PERSIST) {
      for (int e = tid; e < nn_; e += blockDim.x) {
        // (the reverse sweep finds v at the tent's top)
        if (__ldcg(a.tau + s_nid[e]) == (ADJ && e == 0 ? s_ttop : s_ntau[e])) continue;
        if (CS == 1) s_bad = 1;
        else
          for (int r = 0; r < CS; ++r) *cluster.map_shared_rank(&s_bad, r) = 1;
      }
    }
  };
  // tensor-core contractions for this tent (single material, split right-hand sides)
  const bool tc_on = kTC && ng == 1;
  const int NP = P * Q;
  // this CTA's points of the patch for the Grams (split right-hand sides: even
  // shares of the points; else whole elements, whose data and outflow are this CTA's too)
  const int slice = (P * QK + CS - 1) / CS;
  const int e0 = P * rank / CS, e1 = P * (rank + 1) / CS;
  const int q0 = SPLIT ? min(P * QK, rank * slice) : e0 * Q;
  const int q1 = SPLIT ? min(P * QK, q0 + slice) : e1 * Q;
  const int np = (e1 - e0) * QK;           // points of the slice in the rule of the face integrals
  // elements whose data are taken at a time (their points fit sU where the rows are not kept)
  const int EC = kept || !srule ? a.raw_el : min(a.raw_el, 2 * CH / QK);
  double ih = 0.0, tc = 0.0;
  // kept slice: the U-values of the outflow (forward: top points; adjoint:
  // bottom), then those of the moments (the other face)
  T* sKeep = reinterpret_cast<T*>(sm + a.off_keep);
  T* sKI = sKeep + (size_t)np * us;
  const T* sTP = reinterpret_cast<const T*>(sm + a.off_tf);   // data to the rule's points, values to the front's
  const T* sTF = sTP + a.S * a.tf_stride;
  T* sRaw = reinterpret_cast<T*>(sm + a.off_raw);
  // a patch point q of element k mapped to the tent's reference coordinates
  // (Remark 3.1) on the top (TOP) or bottom face, and sqrt(w) as the scale of its
  // U-values (UNIT: 1).  Binary64: the barycentric sums of the vertices, then
  // shifted and scaled.  Mixed: the sums over the element's scaled vertices
  // (s_xh) in float-float, where the errors of a sweep are the same as from
  // points formed in binary64 (0.8 to 1.2 of them, mean 1.0 over 23 outputs)
  // and the binary64 unit is left alone; binary64 sums over scaled vertices
  // double the error of a 1D p = 6 sweep.
  auto map_with = [&](T* pp, int k, int q, bool top, const RuleTab& baryR, const RuleTab& sqwR, bool unit) {
    if constexpr (MIXED) {
      const T* bary_ = rule_tab<T>(baryR);
      T x[DIM + 1];
#pragma unroll
      for (int d = 0; d <= DIM; ++d) x[d] = R::zero();
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const T l = tab(bary_ + q * NV + i);
        x[0] = R::acc(x[0], l, s_xh[k][i][top ? DIM + 1 : DIM]);
#pragma unroll
        for (int d = 0; d < DIM; ++d) x[1 + d] = R::acc(x[1 + d], l, s_xh[k][i][d]);
      }
#pragma unroll
      for (int d = 0; d <= DIM; ++d) pp[d] = R::norm(x[d]);
      pp[DIM + 1] = unit ? R::one() : R::mul(tab(rule_tab<T>(sqwR) + q), R::from(s_sdet[k]));
    } else {
      double x[DIM], tt = 0.0;
#pragma unroll
      for (int d = 0; d < DIM; ++d) x[d] = 0.0;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const double l = __ldg(baryR.d + q * NV + i);
#pragma unroll
        for (int d = 0; d < DIM; ++d) x[d] = fma(l, s_X[k][i][d], x[d]);
        tt = fma(l, top ? s_tt[k][i] : s_tb[k][i], tt);
      }
      pp[0] = s_gc[s_grp[k]] * (tt - tc) * ih;
#pragma unroll
      for (int d = 0; d < DIM; ++d) pp[1 + d] = (x[d] - s_xv[d]) * ih;
      pp[DIM + 1] = unit ? 1.0 : __ldg(sqwR.d + q) * s_sdet[k];
    }
  };
  auto map_point = [&](T* pp, int k, int q, bool top) {   // of the front rule
    map_with(pp, k, q, top, a.baryT, a.sqwT, false);
  };
  auto map_rule = [&](T* pp, int k, int q, bool top) {    // of the rule of the face integrals
    map_with(pp, k, q, top, srule ? a.s_baryT : a.baryT, srule ? a.s_sqwT : a.sqwT, false);
  };
  // data coefficients of the points base .. base + nq - 1 (patch point
  // numbering) for every right-hand side, one (point, right-hand side) per
  // thread so that the front loads of a chunk are all in flight at once:
  // forward, the bottom values in the form of the moments (gamma, alpha,
  // beta_m); adjoint, lambda at the top point; component cc of point ql and
  // right-hand side r at dst[(r * C + cc) * stride + ql], for the U-values
  // scaled by sqrt(w) (RAW: without weights)
  auto data_coefs = [&](int base, int nq, T* dst, int stride, bool raw) {
    for (int id = tid; id < nq * nrhs; id += blockDim.x) {   // (consecutive threads: consecutive points)
      const int r = id / nq, ql = id % nq, qg = base + ql, k = qg / Q, q = qg % Q;
      const double* f = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
      double fv[C];
#pragma unroll
      for (int cc = 0; cc < C; ++cc) fv[cc] = __ldcg(f + cc);
      T* cb = dst + (size_t)r * C * stride + ql;
      if constexpr (ADJ) {
        // adjoint: zeta = sum_q lambda_q u_q over the top points
        const double isw = raw ? 1.0 : __ldg(a.isqw + q) * s_isdet[k];
#pragma unroll
        for (int cc = 0; cc < C; ++cc) cb[cc * stride] = R::from(fv[cc] * isw);
      } else if constexpr (MIXED) {
        // the same coefficients in float-float, the stored values split by
        // integer operations (no binary64 arithmetic per point and column)
        const float2 w2 = __ldg(a.sqw_dd + q), d2 = s_gbf[k][DIM], c2 = s_gic2f[s_grp[k]];
        const dd sw = raw ? dd{1.f, 0.f} : dd_mul({w2.x, w2.y}, {d2.x, d2.y});
        dd f[C];
#pragma unroll
        for (int cc = 0; cc < C; ++cc) f[cc] = dd_split(fv[cc]);
        dd gb[DIM];
#pragma unroll
        for (int d = 0; d < DIM; ++d) gb[d] = {s_gbf[k][d].x, s_gbf[k][d].y};
        dd sg = dd_mul(f[2], gb[0]);
#pragma unroll
        for (int d = 1; d < DIM; ++d) sg = dd_add(sg, dd_mul(f[2 + d], gb[d]));
        cb[0] = dd_mul(sw, f[0]);                                                     // gamma
        cb[stride] = dd_mul(sw, R::sub(dd_mul({c2.x, c2.y}, f[1]), sg));                   // alpha
#pragma unroll
        for (int d = 0; d < DIM; ++d) cb[(2 + d) * stride] = dd_mul(sw, R::sub(f[2 + d], dd_mul(f[1], gb[d])));   // beta_m
      } else {
        const double sw = raw ? 1.0 : __ldg(a.sqw + q) * s_sdet[k], ic2 = s_gic2[s_grp[k]];
        const double Ub = fv[0], vb = fv[1];
        double sg = 0.0;
        for (int d = 0; d < DIM; ++d) sg = fma(fv[2 + d], s_gb[k][d], sg);
        cb[0] = R::from(sw * Ub);                       // gamma
        cb[stride] = R::from(sw * (ic2 * vb - sg));          // alpha
        for (int d = 0; d < DIM; ++d) cb[(2 + d) * stride] = R::from(sw * (fv[2 + d] - vb * s_gb[k][d]));   // beta_m
      }
    }
  };
  // the front records (C values each) that data_coefs(base, nq) will read,
  // prefetched into L2 (their latency then overlaps the work on the chunk before)
  auto prefetch_front = [&](int base, int nq) {
    for (int id = tid; id < nq * nrhs; id += blockDim.x) {
      const int r = id / nq, ql = id % nq, qg = base + ql, k = qg / Q, q = qg % Q;
      const double* f = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(f));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(f + C - 1));
    }
  };
  // moments of the data of the points base .. base + nq - 1 whose U-values are
  // the rows of U, per material (whose elements, of QE points each, are
  // consecutive): one (material, right-hand side, basis function) per group of
  // ps lanes with its C components as independent sums (functions < nl, first)
  // or gamma alone (the others: alpha and beta are only applied through
  // derivatives); the lanes of a group take every ps-th point and are added by
  // butterfly shuffles (a fixed order)
  auto data_moments = [&](int base, int nq, const T* U, int QE) {
    // (the two kinds start at a warp each)
    const int nlow = ng * nrhs * nl, nhigh = ng * nrhs * (nb - nl);
    auto high0 = [&](int ps_) { return (nlow * ps_ + 31) & ~31; };
    int ps = 1;
    while (ps < 8 && high0(2 * ps) + nhigh * ps * 2 <= NT) ps *= 2;
    const int h0_ = high0(ps), nitem = h0_ + nhigh * ps;
    for (int id0 = 0; id0 < nitem; id0 += blockDim.x) {
      const int id = id0 + tid;
      const bool low = id < h0_, live = low ? id < nlow * ps : id < nitem;
      const int it = (low ? id : id - h0_) / ps, part = (low ? id : id - h0_) % ps, nf = low ? nl : nb - nl;
      const int g = it / (nrhs * nf), rest = it % (nrhs * nf), r = rest / nf, i = rest % nf + (low ? 0 : nl);
      T t[C];
#pragma unroll
      for (int cc = 0; cc < C; ++cc) t[cc] = R::zero();
      if (live) {
        const int l0 = max(0, s_ge0[g] * QE - base), l1 = min(nq, s_ge0[g + 1] * QE - base);
        const T* cb = sCB + (size_t)r * C * cbs;
        if (low) {
          for (int ql = l0 + part; ql < l1; ql += ps) {
            const T u = U[(size_t)ql * us + i];
#pragma unroll
            for (int cc = 0; cc < C; ++cc) t[cc] = R::acc(t[cc], cb[cc * cbs + ql], u);
          }
        } else {
#pragma unroll 4
          for (int ql = l0 + part; ql < l1; ql += ps) t[0] = R::acc(t[0], cb[ql], U[(size_t)ql * us + i]);
        }
      }
#pragma unroll
      for (int cc = 0; cc < C; ++cc) t[cc] = R::norm(t[cc]);
      for (int o = 1; o < ps; o <<= 1)
#pragma unroll
        for (int cc = 0; cc < C; ++cc) t[cc] = R::add(t[cc], shfl_xor_t(t[cc], o));
      if (part == 0 && live) {
        T* M = sPM + (size_t)g * nmom + (size_t)r * C * nb + i;
#pragma unroll
        for (int cc = 0; cc < C; ++cc)
          if (cc == 0 || low) M[cc * nb] = R::add(M[cc * nb], t[cc]);
      }
    }
  };
  // ---- tensor-core contractions (tp_tc.cuh) ----
  // the digit-plane products of one contraction: level L = i + j sums planes
  // i of A and j of B over ksteps K steps of 16 into tensor-memory columns
  // (L - 2) cstride; one thread issues them (tc_issue), every thread waits
  // (bounded) for their completion (tc_wait, which returns whether they
  // completed, the same in every thread)
  auto tc_issue = [&](uint32_t aA, uint32_t planeA, uint32_t lboA, uint32_t aB, uint32_t planeB, uint32_t lboB,
                      int ksteps, int N, int cstride) {
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0) {
      const uint32_t id_ = tc::idesc_bf16(tc::kMaxM, N);
      if (planeB == 0) {
        // B's digit planes stacked along N at cstride-row offsets (plane j at
        // rows (j - 1) cstride): one product per plane i of A and K step puts
        // A_i B_j into the columns of level i + j for every j at once (the
        // columns past level S + 1 take unused pairs and are never read)
        for (int ks = 0; ks < ksteps; ++ks)
          for (int i = 1; i <= tc::kSlices; ++i)
            tc::mma_bf16(s_tmem + (uint32_t)((i - 1) * cstride),
                         tc::sdesc(aA + (uint32_t)(i - 1) * planeA + (uint32_t)ks * 2 * lboA, lboA, 128),
                         tc::sdesc(aB + (uint32_t)ks * 2 * lboB, lboB, 128), id_, ks > 0 || i > 1);
      } else
      // K steps outermost, so that consecutive products go to different
      // level sums; the first product of each level overwrites its columns
      for (int ks = 0; ks < ksteps; ++ks)
        for (int L = 2; L <= tc::kSlices + 1; ++L)
          for (int i = max(1, L - tc::kSlices); i <= min(tc::kSlices, L - 1); ++i) {
            const int j = L - i;
            tc::mma_bf16(s_tmem + (uint32_t)((L - 2) * cstride),
                         tc::sdesc(aA + (uint32_t)(i - 1) * planeA + (uint32_t)ks * 2 * lboA, lboA, 128),
                         tc::sdesc(aB + (uint32_t)(j - 1) * planeB + (uint32_t)ks * 2 * lboB, lboB, 128), id_,
                         ks > 0 || i > max(1, L - tc::kSlices));
          }
      tc::commit(&s_tcbar);
    }
  };
  auto tc_wait = [&]() {
    bool ok = tc::mbar_wait(&s_tcbar, tc_phase, tc::kMaxPolls);
    if (!ok) {
      flag_error(a, TP_ERR_TIMEOUT, tent);
      tc::mbar_wait(&s_tcbar, tc_phase, 16 * tc::kMaxPolls);   // the products still in flight
    }
    tc_phase ^= 1u;
    ok = __syncthreads_and(ok) != 0;
    tc::fence_after();
    return ok;
  };
  auto tc_product = [&](uint32_t aA, uint32_t planeA, uint32_t lboA, uint32_t aB, uint32_t planeB, uint32_t lboB,
                        int ksteps, int N, int cstride) {
    tc_issue(aA, planeA, lboA, aB, planeB, lboB, ksteps, N, cstride);
    return tc_wait();
  };
  // data moments of nq bottom points (U-values in rows 0.. of sU) of a
  // single-material tent on the tensor cores:
  //   M[r, c, i] += sum_q cb[q, r, c] U_i(q)
  // A: the data coefficients, rows (r, c), scaled per row; B: the U-values,
  // rows i (padded to 32), scaled per basis function; K: the points (padded
  // to 16 with zeros, at most CH, so that the level sums stay below 2^24)
  // (tc_mom_start digit-splits the chunk and issues its products; the
  // caller evaluates the next chunk while they run; tc_mom_finish waits and
  // adds the level sums into the moments)
  auto tc_mom_start = [&](int nq) {
    if constexpr (kTC) {
      const int M = nrhs * C, RG = (M + 7) >> 3, KC = ((nq + 15) >> 4) << 1;
      uint16_t* sTA = reinterpret_cast<uint16_t*>(sm + a.off_tc);
      const int planeA = CH * RG * 8;
      uint16_t* sTB = sTA + tc::kSlices * planeA + 512;
      int* eA = s_tce[0];
      int* eB = s_tce[1];
      // TPR threads per row (M + nb <= 128 rows, so every thread takes part
      // once and a row's maxima meet by shuffles)
      {
        constexpr int TPR = NT / 128;
        const int m = tid / TPR, part = tid % TPR;
        float mx = 0.f;
        if (m < M) {
          for (int ql = part; ql < nq; ql += TPR) mx = fmaxf(mx, fabsf(sCB[(size_t)m * cbs + ql].hi));
        } else if (m < M + nb) {
          for (int ql = part; ql < nq; ql += TPR) mx = fmaxf(mx, fabsf(sU[(size_t)ql * us + (m - M)].hi));
        }
#pragma unroll
        for (int o = 1; o < TPR; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (part == 0 && m < M) eA[m] = tc::scale_exp(mx);
        if (part == 0 && m >= M && m < M + nb) eB[m - M] = tc::scale_exp(mx);
      }
      __syncthreads();
      // digit planes, one item = 4 consecutive points of one row of A or B (8 left
      // a second round of the CTA's threads a third full: 330 -> 328 ms)
      for (int id = tid; id < (M + 32) * 2 * KC; id += blockDim.x) {
        const bool isA = id < M * 2 * KC;
        const int id2 = isA ? id : id - M * 2 * KC, rows = isA ? M : 32;
        const int k4 = id2 / rows, m = id2 % rows, kc = k4 >> 1, half = 4 * (k4 & 1);
        const bool live = isA || m < nb;
        const int ex = isA ? eA[m] : (live ? eB[m] : 0);
        float d[4][tc::kSlices];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int ql = k4 * 4 + j;
          T x = R::zero();
          if (ql < nq && live) x = isA ? sCB[(size_t)m * cbs + ql] : sU[(size_t)ql * us + m];
          tc::digits(x.hi, x.lo, ex, d[j]);
        }
        if (isA) tc::store_row4(sTA + ((size_t)(kc * RG + (m >> 3)) * 64 + (m & 7) * 8 + half), planeA, d);
        else tc::store_row4(sTB + ((size_t)(kc * 4 * tc::kSlices + (m >> 3)) * 64 + (m & 7) * 8 + half), 4 * 64, d);
      }
      // B: the planes stacked along N, 32 rows each (planeB = 0 selects the stacked products)
      tc_issue(tc::smem_addr(sTA), (uint32_t)planeA * 2, (uint32_t)RG * 128, tc::smem_addr(sTB), 0u,
               (uint32_t)(4 * tc::kSlices) * 128, KC >> 1, 32 * tc::kSlices, 32);
    }
  };
  auto tc_mom_finish = [&]() {
    if constexpr (kTC) {
      const int M = nrhs * C;
      const int* eA = s_tce[0];
      const int* eB = s_tce[1];
      const bool ok = tc_wait();
      // levels -> float-float moments: warp w reads rows 32 (w % 4) .. + 31,
      // basis functions CW (w / 4) .. + CW - 1
      constexpr int CW = 32 / (NW / 4);
      const int q4 = warp & 3, h = warp >> 2;
      if (ok && 32 * q4 < M) {
        const int m = 32 * q4 + lane;
        for (int c8 = 0; c8 < CW / 8; ++c8) {
          float lv[tc::kSlices][8];
#pragma unroll
          for (int l = 0; l < tc::kSlices; ++l)
            tc::ld8(s_tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(l * 32 + CW * h + 8 * c8), lv[l]);
          tc::wait_ld();
          if (m < M) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int i = CW * h + 8 * c8 + j;
              if (i >= nb) continue;
              float acc[tc::kSlices];
#pragma unroll
              for (int l = 0; l < tc::kSlices; ++l) acc[l] = lv[l][j];
              T v;
              tc::combine_ff(acc, v.hi, v.lo);
              tc::ff_scale(v.hi, v.lo, eA[m] + eB[i] - 16);
              T* Mp = sPM + (size_t)m * nb + i;
              *Mp = R::add(*Mp, v);
            }
          }
        }
      }
      tc::fence_before();
      __syncthreads();   // the exponents and columns read above are rewritten by the next chunk
    }
  };
  const int nneu = NEU ? s_nneu : 0;   // (kernels for meshes without Neumann facets leave out their code)
  const bool pblk = nif > 0 || nneu > 0;
  const bool has_g = !ADJ && gD != nullptr;   // boundary data (else homogeneous)
  T* sFD = reinterpret_cast<T*>(sm + a.off_pd);      // Dirichlet sums (Grams, then data moments), then Neumann data
  T* sDD = reinterpret_cast<T*>(sm + a.off_dd);
  const int nfg = nfac > 0 ? ng * (DIM + 1) * npl : 0, nfm = nfac > 0 ? ng * (DIM + 1) * nrhs * nl : 0;
  T* sPBN = sDD + nfm;
  unsigned gdir = 0;   // materials with Dirichlet facets
  for (int f = 0; f < nfac; ++f) gdir |= 1u << s_fg[f];
  T* A0 = CS > 1 ? cluster.map_shared_rank(sA, 0) : sA;
  dd* sF_ = reinterpret_cast<dd*>(sm + a.off_pg);         // N*N     inverse of the equilibrated matrix (the Grams are dead by then)
  float* sEq = reinterpret_cast<float*>(sm + a.off_eq);   // N       equilibration scales (powers of two)
  // ---------------- cluster reduction (rank order) ----------------
  // every CTA sums every CTA's partials in rank order (all remote loads of an
  // entry are issued before the additions)
  auto cluster_sum = [&](T* src, int id) {
    T t = R::zero();
    for (int r0 = 0; r0 < CS; r0 += 4) {
      T v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r0 + u < CS) v[u] = cluster.map_shared_rank(src, r0 + u)[id];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r0 + u < CS) t = R::add(t, v[u]);
    }
    return t;
  };
  // reduce-scatter: rank r sums its share of every array over the cluster and
  // stores the sums into every CTA's copy
  auto cluster_reduce = [&](T* part, T* sum, int n) {
    if (CS == 1) {
      if (sum != part)
        for (int id = tid; id < n; id += blockDim.x) sum[id] = part[id];
      return;
    }
    const int lo = (n * rank) / CS, hi = (n * (rank + 1)) / CS;
    for (int id = lo + tid; id < hi; id += blockDim.x) {
      const T t = cluster_sum(part, id);
      for (int rr = 0; rr < CS; ++rr) cluster.map_shared_rank(sum, rr)[id] = t;
    }
  };
  for (;;) {   // assembly and inverse (a second time only where the front's times are not the tabulated ones)
  // (b) the front times: bottom and top fronts over every element, causality
  if (real) {
    for (int e = tid; e < nn_; e += blockDim.x) s_ntau[e] = ADJ && e == 0 ? a.tent_tbot[tent] : __ldcg(a.tau + s_nid[e]);
    __syncthreads();
  }
  const double tbot = s_ntau[0];
  if (tid == 0) {
    s_tbot = tbot;
    s_tc = 0.5 * (tbot + s_ttop);
  }
  for (int id = tid; id < NG * nmom; id += blockDim.x) sPM[id] = R::zero();
  for (int id = tid; id < N * N; id += blockDim.x) sA[id] = R::zero();
  for (int k = tid; k < P; k += blockDim.x) {
    for (int i = 0; i < NV; ++i) {
      const int e = s_vid[k][i];
      s_tb[k][i] = s_ntau[e];
      s_tt[k][i] = e == 0 ? s_ttop : s_ntau[e];
    }
    // gradients of the linear fronts: g = e^-1 (tau_i - tau_0), e from the host
    const int el = s_el[k];
    double db[DIM], dt[DIM];
    for (int i = 0; i < DIM; ++i) {
      db[i] = s_tb[k][i + 1] - s_tb[k][0];
      dt[i] = s_tt[k][i + 1] - s_tt[k][0];
    }
    double g2 = 0.0;
    for (int d = 0; d < DIM; ++d) {
      double gb = 0.0, gt = 0.0;
      for (int i = 0; i < DIM; ++i) {
        const double ei = __ldg(a.elem_einv + ((int64_t)el * DIM + d) * DIM + i);
        gb = fma(ei, db[i], gb);
        gt = fma(ei, dt[i], gt);
      }
      s_gb[k][d] = gb;
      s_gt[k][d] = gt;
      g2 = fma(gt, gt, g2);
    }
    if constexpr (MIXED) {   // vertices in the tent's reference coordinates: xhat, then that on the bottom and the top
      const double cg = s_gc[s_grp[k]], tcn = 0.5 * (tbot + s_ttop), ihn = s_ih;
      for (int i = 0; i < NV; ++i) {
        for (int d = 0; d < DIM; ++d) s_xh[k][i][d] = R::from((s_X[k][i][d] - s_xv[d]) * ihn);
        s_xh[k][i][DIM] = R::from(cg * (s_tb[k][i] - tcn) * ihn);
        s_xh[k][i][DIM + 1] = R::from(cg * (s_tt[k][i] - tcn) * ihn);
      }
    }
    s_sdet[k] = __ldg(a.elem_sdet + el);
    s_isdet[k] = __ldg(a.elem_isdet + el);
    if constexpr (MIXED) {
      for (int d = 0; d < DIM; ++d) {
        const dd gf = dd_split(s_gb[k][d]);
        s_gbf[k][d] = make_float2(gf.hi, gf.lo);
      }
      const dd sf = dd_split(s_sdet[k]);
      s_gbf[k][DIM] = make_float2(sf.hi, sf.lo);
    }
    const double ck = s_gc[s_grp[k]];
    if (!(ck * ck * g2 < 1.0)) flag_error(a, TP_ERR_CAUSALITY, tent);   // space-like top face: c |g| < 1
  }
  for (int f = tid; f < nfac + nif + (NEU ? s_nneu : 0); f += blockDim.x) {
    s_fP[f][0][DIM] = tbot;
    s_fP[f][1][DIM] = s_ttop;
    for (int c2 = 2; c2 <= DIM; ++c2) s_fP[f][c2][DIM] = s_ntau[s_fw[f][c2]];
    // n! * n-volume = sqrt(det(E^T E)), E = [P_i - P_0] ((n+1) x n)
    double G[DIM][DIM];
    for (int i = 0; i < DIM; ++i)
      for (int j = 0; j < DIM; ++j) {
        double s_ = 0.0;
        for (int d = 0; d <= DIM; ++d) s_ += (s_fP[f][i + 1][d] - s_fP[f][0][d]) * (s_fP[f][j + 1][d] - s_fP[f][0][d]);
        G[i][j] = s_;
      }
    // sqrt(w) = sqrt(w_ref) sqrt(n! volume) at the facet's points
    s_fsq[f] = sqrt(sqrt(fabs(small_det<DIM>(G))));
  }
  // Gram pairs owned by this thread: the bottom face's (every function, the
  // recovery term) from the first thread on, the top face's and the facets'
  // (functions < nl: they enter through derivatives) from the last thread down,
  // so that threads without a second pair of the one take the other.  (Every
  // pair on both faces and the derivative moments over every function: 2D p = 5,
  // two materials, 188 -> 145 ms a sweep, 3D p = 3 mixed 8.6 -> 7.5 ms)
  int pi[kMaxPair], pj[kMaxPair], li[kMaxLow], lj[kMaxLow];
  T aK[kMaxLow], aG[kMaxLow], aH[kMaxLow][DIM], aB[kMaxPair];
  auto unpack = [](int id, int n, int& i, int& j) {
    i = id;
    j = 0;
    if (id >= n) i = 0;
    else
      while (i > j) i -= ++j;
  };
#pragma unroll
  for (int s = 0; s < kMaxPair; ++s) {
    unpack(tid + s * NT, npair, pi[s], pj[s]);
    aB[s] = R::zero();
  }
#pragma unroll
  for (int s = 0; s < kMaxLow; ++s) {
    unpack(NT - 1 - tid + s * NT, npl, li[s], lj[s]);
    aK[s] = aG[s] = R::zero();
#pragma unroll
    for (int d = 0; d < DIM; ++d) aH[s][d] = R::zero();
  }
  __syncthreads();
  ih = s_ih;
  tc = s_tc;

  // ---------------- vertical faces ----------------
  // (before the Grams, whose region the facet Grams share; with split
  // right-hand sides after the moments, whose tensor-core staging shares the
  // region of the Dirichlet sums)
  // Dirichlet facets, per material g, after the interface blocks: the facet
  // Grams summed over g's facets, G_g, and weighted by the facets' normals,
  // Gn_g[d] = sum_f n_f[d] F_f (layout [G_g | Gn_g[0..DIM)] of npl each),
  // then the data moments in the same arrangement (nrhs*nl each).  The
  // congruences with the derivative maps are linear, so these sums carry all
  // a tent needs; they are formed after the cluster reduction.
  // Interface and Neumann facets add their blocks to this CTA's partial A
  // at once; Neumann facets also to a partial b (nrhs*N, after the
  // Dirichlet sums).
  auto facet_phase = [&]() {
  if (extra) {
    for (int id = tid; id < nfg; id += blockDim.x) sFD[id] = R::zero();
    for (int id = tid; id < nfm; id += blockDim.x) sDD[id] = R::zero();
    if (nneu > 0)
      for (int id = tid; id < nrhs * N; id += blockDim.x) sPBN[id] = R::zero();
    for (int id = tid; id < nrhs * nl; id += blockDim.x) sDel[id] = R::zero();
    if (nif > 0)
      for (int id = tid; id < nl * nl; id += blockDim.x) sFpm[id] = R::zero();
    __syncthreads();
    // (a) Dirichlet facets: the points of all of them (facet after facet) in
    // one pass, split over the cluster; a facet's Gram and moments are folded
    // into its material's sums where its points end
    if (nfac > 0) {
      const int NPD = nfac * Q, dsl = (NPD + CS - 1) / CS;
      const int d0 = min(NPD, rank * dsl), d1 = min(NPD, d0 + dsl);
      // the Grams take this CTA's slice [d0, d1); the data moments of split
      // right-hand sides take every point (homogeneous data, a NULL array, have
      // none: 3D p = 3, 6000 elements, 64 columns mixed 327 -> 300 ms; binary64,
      // 750 elements, where boundary tents lie on the chain, 130 -> 128)
      const int l0 = rsplit && has_g ? 0 : d0, l1 = rsplit && has_g ? NPD : d1;
      T aF[kMaxLow];
#pragma unroll
      for (int s = 0; s < kMaxLow; ++s) aF[s] = R::zero();
      auto fold_gram = [&](int f) {
        if (f >= nfac) return;
        T* Fg = sFD + (size_t)s_fg[f] * (DIM + 1) * npl;
#pragma unroll
        for (int s = 0; s < kMaxLow; ++s)
          if (NT - 1 - tid + s * NT < npl) {
            const int q = NT - 1 - tid + s * NT;
            Fg[q] = R::add(Fg[q], aF[s]);
            for (int d = 0; d < DIM; ++d)
              Fg[(1 + d) * npl + q] = R::fma(R::from(s_fn[f][d]), aF[s], Fg[(1 + d) * npl + q]);
            aF[s] = R::zero();
          }
      };
      auto fold_mom = [&](int f, int id, T t) {
        if (f >= nfac) return;
        T* Dg = sDD + (size_t)s_fg[f] * (DIM + 1) * nrhs * nl;
        Dg[id] = R::add(Dg[id], t);
        for (int d = 0; d < DIM; ++d)
          Dg[(1 + d) * nrhs * nl + id] = R::fma(R::from(s_fn[f][d]), t, Dg[(1 + d) * nrhs * nl + id]);
      };
      int fc = l0 / Q;   // facet of the points being accumulated (uniform over the CTA)
      for (int base = l0; base < l1; base += CH) {
        const int nq = min(CH, l1 - base);
        for (int id = tid; id < nq; id += blockDim.x) {
          const int q = base + id, f = q / Q, qf = q - f * Q;
          double xt[DIM + 1];
          for (int d = 0; d <= DIM; ++d) xt[d] = 0.0;
          for (int i = 0; i < NV; ++i) {
            const double l = __ldg(a.bary + qf * NV + i);
            for (int d = 0; d <= DIM; ++d) xt[d] = fma(l, s_fP[f][i][d], xt[d]);
          }
          const double sw = __ldg(a.sqw + qf) * s_fsq[f];
          T* pp = sPt + id * (DIM + 2);
          pp[0] = R::from(s_gc[s_fg[f]] * (xt[DIM] - tc) * ih);
          for (int d = 0; d < DIM; ++d) pp[1 + d] = R::from((xt[d] - s_xv[d]) * ih);
          pp[DIM + 1] = R::from(sw);
          // the facet's block of boundary data (without Neumann facets: the facet's own index)
          const long long goff = a.tent_gdoff[tent] + (NEU ? (long long)s_fw[f][0] * Q + qf : (long long)q);
          if (has_g)
            for (int r = 0; r < nrhs; ++r) sGd[id * nrhs + r] = R::from(sw * gD[(long long)r * a.n_bnd + goff]);
        }
        eval_uvalues_block<DIM, T, true, true>(a, nq, sPt, sM, sU);
        const int fc0 = fc;
        for (int ql = 0; ql < nq; ++ql) {
          if (base + ql >= (fc + 1) * Q) fold_gram(fc++);
          if (base + ql < d0 || base + ql >= d1) continue;   // another CTA's Gram points
          const T* u = sU + (size_t)ql * us;
#pragma unroll
          for (int s = 0; s < kMaxLow; ++s)
            if (NT - 1 - tid + s * NT < npl) aF[s] = R::fma(u[li[s]], u[lj[s]], aF[s]);
        }
        for (int id = tid; id < (has_g ? nrhs * nl : 0); id += blockDim.x) {
          const int r = id / nl, i = id % nl;
          int f = fc0;
          T t = sDel[id];
          for (int ql = 0; ql < nq; ++ql) {
            if (base + ql >= (f + 1) * Q) {
              fold_mom(f++, id, t);
              t = R::zero();
            }
            t = R::fma(sGd[ql * nrhs + r], sU[(size_t)ql * us + i], t);
          }
          sDel[id] = t;
        }
        __syncthreads();
      }
      fold_gram(fc);
      for (int id = tid; id < (has_g ? nrhs * nl : 0); id += blockDim.x) {
        fold_mom(fc, id, sDel[id]);
        sDel[id] = R::zero();
      }
      __syncthreads();
    }
    // (b) time-like interface facets, then Neumann facets, one after the
    // other, each taken by one CTA of the cluster (its points split over the
    // cluster repeated the congruence in every CTA: two thirds of the time of
    // an interface tent's assembly at 2D p = 5); their blocks go into the
    // partial A at once.  Neumann facets (eq. 4.1), with F the facet Gram
    // of U-values and delta = sum w g_N u:
    //   A_N = -(c/h^2) D_n F D_t^T + (beta/h^2) D_n F D_n^T,
    //   b_N = -(c/h) D_t delta - (beta/h) D_n delta
    // (v = (c/h) D_t u, sigma.n = -(1/h) D_n u, D_n = sum_m n_m D_m)
    for (int f = nfac; f < nfac + nif + nneu; ++f) {
      const bool neu = NEU && f >= nfac + nif, mine = (f - nfac) % CS == rank;
      if (!mine && !(rsplit && neu && has_g)) continue;
      const int f0 = 0, f1 = mine ? Q : 0;
      const int gp = s_fg[f], gm = s_fg2[f];
      const double cp = s_gc[gp], cm = s_gc[gm];
      T aF[kMaxLow], aF2[kMaxLow];
#pragma unroll
      for (int s = 0; s < kMaxLow; ++s) aF[s] = aF2[s] = R::zero();
      // (a Neumann facet's data moments of split right-hand sides take every point)
      const int l0 = f0, l1 = (rsplit && neu && has_g) ? Q : f1;
      for (int base = l0; base < l1; base += CH) {
        const int nq = min(CH, l1 - base);
        const int npt = neu ? nq : 2 * nq;   // interface: + side points, then - side
        for (int id = tid; id < nq; id += blockDim.x) {
          const int q = base + id;
          double xt[DIM + 1];
          for (int d = 0; d <= DIM; ++d) xt[d] = 0.0;
          for (int i = 0; i < NV; ++i) {
            const double l = __ldg(a.bary + q * NV + i);
            for (int d = 0; d <= DIM; ++d) xt[d] = fma(l, s_fP[f][i][d], xt[d]);
          }
          const double sw = __ldg(a.sqw + q) * s_fsq[f];
          T* pp = sPt + id * (DIM + 2);
          pp[0] = R::from(cp * (xt[DIM] - tc) * ih);
          for (int d = 0; d < DIM; ++d) pp[1 + d] = R::from((xt[d] - s_xv[d]) * ih);
          pp[DIM + 1] = R::from(sw);
          if (neu) {
            const long long goff = a.tent_gdoff[tent] + (long long)s_fw[f][0] * Q + q;
            for (int r = 0; r < nrhs; ++r)
              sGd[id * nrhs + r] = R::from(has_g ? sw * gD[(long long)r * a.n_bnd + goff] : 0.0);
          } else {
            T* p2 = sPt + (nq + id) * (DIM + 2);
            p2[0] = R::from(cm * (xt[DIM] - tc) * ih);
            for (int d = 0; d < DIM; ++d) p2[1 + d] = pp[1 + d];
            p2[DIM + 1] = pp[DIM + 1];
          }
        }
        if (!neu) __syncthreads();   // (the - side's rows are read by other threads than wrote them)
        eval_uvalues_block<DIM, T, true, true>(a, npt, sPt, sM, sU);
        for (int ql = 0; ql < nq; ++ql) {
          if (base + ql < f0 || base + ql >= f1) continue;   // another CTA's Gram points
          const T* u = sU + (size_t)ql * us;
          const T* u2 = sU + (size_t)(nq + ql) * us;
#pragma unroll
          for (int s = 0; s < kMaxLow; ++s)
            if (NT - 1 - tid + s * NT < npl) {
              aF[s] = R::acc(aF[s], u[li[s]], u[lj[s]]);
              if (!neu) aF2[s] = R::acc(aF2[s], u2[li[s]], u2[lj[s]]);
            }
        }
        if (neu) {
          for (int id = tid; id < nrhs * nl; id += blockDim.x) {
            const int r = id / nl, i = id % nl;
            T t = sDel[id];
            for (int ql = 0; ql < nq; ++ql) t = R::fma(sGd[ql * nrhs + r], sU[(size_t)ql * us + i], t);
            sDel[id] = t;
          }
        } else {
          for (int id = tid; id < nl * nl; id += blockDim.x) {
            const int i = id / nl, j = id % nl;
            T t = sFpm[id];
#pragma unroll 4
            for (int ql = 0; ql < nq; ++ql) t = R::acc(t, sU[(size_t)ql * us + i], sU[(size_t)(nq + ql) * us + j]);
            sFpm[id] = R::norm(t);
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int s = 0; s < kMaxLow; ++s)
        if (NT - 1 - tid + s * NT < npl) {
          sF[NT - 1 - tid + s * NT] = R::norm(aF[s]);
          sF2[NT - 1 - tid + s * NT] = R::norm(aF2[s]);
        }
      __syncthreads();
      T nrm[DIM];
      for (int d = 0; d < DIM; ++d) nrm[d] = R::from(s_fn[f][d]);
      // block D_n X W1^T + D_t X W2^T, W = wt D_t + wn D_n (D_n = sum_m n_m D_m), of
      // a facet Gram X (MODE 0 packed symmetric, 1 full, 2 full transposed) added
      // to the partial A: first Y = X W^T, then the rows; each entry takes a
      // few terms instead of the products of both operators' terms
      // (2D p = 5: a facet's four blocks 80 us before)
      auto facet_block = [&](auto mode, const T* X, T w1t, T w1n, T w2t, T w2n, int gr, int gcl) {
        constexpr int MODE = decltype(mode)::value;
        T *Y1 = sFpm + nl * nl, *Y2 = Y1 + nl * nb;
        for (int id = tid; id < nl * nb; id += blockDim.x) {
          const int k = id / nb, jj = id - k * nb;
          T dt = R::zero(), dn = R::zero();
#pragma unroll
          for (int v_ = 0; v_ <= DIM; ++v_) {
            T t = R::zero();
            for (int e = __ldg(a.rel_ptr + jj * NV + v_), e1_ = __ldg(a.rel_ptr + jj * NV + v_ + 1); e < e1_; ++e) {
              const int sj = __ldg(a.rel_src + e);
              const T x = MODE == 0 ? X[pair_index(k, sj)] : MODE == 1 ? X[k * nl + sj] : X[sj * nl + k];
              t = Fac<T>::add(t, x, a.rel_facf, a.rel_fac, e);
            }
            if (v_ == 0) dt = t;
            else dn = R::fma(nrm[v_ - 1], t, dn);
          }
          Y1[id] = R::fma(w1t, dt, R::mul(w1n, dn));
          Y2[id] = R::fma(w2t, dt, R::mul(w2n, dn));
        }
        __syncthreads();
        for (int id = tid; id < nb * nb; id += blockDim.x) {
          const int i = id / nb, jj = id - i * nb;
          T t = R::zero();
#pragma unroll
          for (int v_ = 0; v_ <= DIM; ++v_) {
            const T* Y = v_ == 0 ? Y2 : Y1;
            T u = R::zero();
            for (int e = __ldg(a.rel_ptr + i * NV + v_), e1_ = __ldg(a.rel_ptr + i * NV + v_ + 1); e < e1_; ++e)
              u = Fac<T>::add(u, Y[__ldg(a.rel_src + e) * nb + jj], a.rel_facf, a.rel_fac, e);
            t = v_ == 0 ? u : R::fma(nrm[v_ - 1], u, t);
          }
          T* dst = sA + (size_t)(gr * nb + i) * N + gcl * nb + jj;
          *dst = R::add(*dst, t);
        }
        __syncthreads();
      };
      const double ih2 = ih * ih;
      if (neu) {
        if (mine)
          facet_block(std::integral_constant<int, 0>{}, sF, R::from(-cp * ih2), R::from(a.beta * ih2), R::zero(), R::zero(), gp,
                      gp);
        for (int id = tid; id < nrhs * nb; id += blockDim.x) {
          const int r = id / nb, i = id % nb;
          const T* del = sDel + (size_t)r * nl;
          T dn = R::zero();
          for (int d = 0; d < DIM; ++d) dn = R::fma(nrm[d], rel_apply<DIM, T>(a, i, 1 + d, del), dn);
          const T t = R::fma(R::from(-a.beta * ih), dn, R::mul(R::from(-cp * ih), rel_apply<DIM, T>(a, i, 0, del)));
          T* dst = sPBN + (size_t)r * N + gp * nb + i;
          *dst = R::add(*dst, t);
        }
        __syncthreads();
        for (int id = tid; id < nrhs * nl; id += blockDim.x) sDel[id] = R::zero();
        __syncthreads();
        continue;
      }
      for (int blk = 0; blk < 4; ++blk) {
        const int tside = blk >> 1, sside = blk & 1;   // test and trial side, 0: +, 1: -
        const double st = tside ? -1.0 : 1.0, ss = sside ? -1.0 : 1.0;
        const double ct = tside ? cm : cp, cs = sside ? cm : cp;
        const T w1t = R::from(-0.5 * st * cs * ih2), w1n = R::from(st * ss * a.beta * ih2);
        const T w2t = R::from(st * ss * a.alpha * cs * ct * ih2), w2n = R::from(-0.5 * st * ct * ih2);
        const int gr = tside ? gm : gp, gcl = sside ? gm : gp;
        if (tside == sside) facet_block(std::integral_constant<int, 0>{}, tside ? sF2 : sF, w1t, w1n, w2t, w2n, gr, gcl);
        else if (tside == 0) facet_block(std::integral_constant<int, 1>{}, sFpm, w1t, w1n, w2t, w2n, gr, gcl);
        else facet_block(std::integral_constant<int, 2>{}, sFpm, w1t, w1n, w2t, w2n, gr, gcl);
      }
      for (int id = tid; id < nl * nl; id += blockDim.x) sFpm[id] = R::zero();
      __syncthreads();
    }
  }
  };
  if constexpr (!SPLIT) facet_phase();
  if (!kept) {   // (the facets' Grams shared this region)
    for (int id = tid; id < NG * ((DIM + 1) * npl + npair); id += blockDim.x) sPG[id] = R::zero();
    if (extra || np == 0) __syncthreads();
  }

  // ---------------- Grams over this CTA's points ----------------
  int curk = SPLIT ? q0 / QK : e0, kend = (curk + 1) * QK;
  int curg = (q1 > q0) ? s_grp[curk] : 0;
  // element flush: G += G_K, H_m += g_{K,m} G_K;  group flush: publish G, H, Gbot of the group
  auto flush_element = [&](int k) {
    T g[DIM];
    for (int d = 0; d < DIM; ++d) g[d] = R::from(s_gt[k][d]);
#pragma unroll
    for (int s = 0; s < kMaxLow; ++s) {
      const T k_ = R::norm(aK[s]);
      aG[s] = R::add(aG[s], k_);
#pragma unroll
      for (int d = 0; d < DIM; ++d) aH[s][d] = R::fma(g[d], k_, aH[s][d]);
      aK[s] = R::zero();
    }
  };
  auto flush_group = [&](int g) {
#pragma unroll
    for (int s = 0; s < kMaxLow; ++s) {
      const int id = NT - 1 - tid + s * NT;
      if (id < npl) {
        sPG[g * npl + id] = R::add(sPG[g * npl + id], aG[s]);
#pragma unroll
        for (int d = 0; d < DIM; ++d) sPH[(g * DIM + d) * npl + id] = R::add(sPH[(g * DIM + d) * npl + id], aH[s][d]);
      }
      aG[s] = R::zero();
#pragma unroll
      for (int d = 0; d < DIM; ++d) aH[s][d] = R::zero();
    }
#pragma unroll
    for (int s = 0; s < kMaxPair; ++s) {
      const int id = tid + s * NT;
      if (id < npair) sPGb[g * npair + id] = R::add(sPGb[g * npair + id], R::norm(aB[s]));
      aB[s] = R::zero();
    }
  };
  // points pt .. end - 1 (rows of U-values ut at the top, ub at the bottom) added
  // to the Grams, element by element so that the loads of several points are in
  // flight (one point at a time exposed a shared-memory round trip per point)
  auto gram_points = [&](int pt, int end, const T* ut, const T* ub) {
    while (pt < end) {
      if (pt >= kend) {   // the next element's points start
        const int k = SPLIT ? pt / QK : curk + 1;
        flush_element(curk);
        if (s_grp[k] != curg) {
          flush_group(curg);
          curg = s_grp[k];
        }
        curk = k;
        kend = (k + 1) * QK;
      }
      const int n = min(end, kend) - pt;
      auto pair_sum = [&](T t, const T* x, const T* y) {
#pragma unroll 4
        for (int q = 0; q < n; ++q) t = R::acc(t, x[q * us], y[q * us]);
        return t;
      };
      // a thread's pair on either face in one loop, as independent chains
      const bool lo0 = NT - 1 - tid < npl;
      if (tid < npair && lo0) {
        const T *ti = ut + li[0], *tj = ut + lj[0], *bi = ub + pi[0], *bj = ub + pj[0];
        T k_ = aK[0], b_ = aB[0];
#pragma unroll 4
        for (int q = 0; q < n; ++q) {
          k_ = R::acc(k_, ti[q * us], tj[q * us]);
          b_ = R::acc(b_, bi[q * us], bj[q * us]);
        }
        aK[0] = k_;
        aB[0] = b_;
      } else if (lo0) {
        aK[0] = pair_sum(aK[0], ut + li[0], ut + lj[0]);
      } else if (kMaxPair > 1 && tid + NT < npair) {
        const T *bi = ub + pi[0], *bj = ub + pj[0], *ci = ub + pi[1 % kMaxPair], *cj = ub + pj[1 % kMaxPair];
        T b_ = aB[0], c_ = aB[1 % kMaxPair];
#pragma unroll 4
        for (int q = 0; q < n; ++q) {
          b_ = R::acc(b_, bi[q * us], bj[q * us]);
          c_ = R::acc(c_, ci[q * us], cj[q * us]);
        }
        aB[0] = b_;
        aB[1 % kMaxPair] = c_;
      } else if (tid < npair) {
        aB[0] = pair_sum(aB[0], ub + pi[0], ub + pj[0]);
      }
#pragma unroll
      for (int s = 1; s < kMaxPair; ++s)
        if (tid + s * NT < npair && (s > 1 || lo0)) aB[s] = pair_sum(aB[s], ub + pi[s], ub + pj[s]);
#pragma unroll
      for (int s = 1; s < kMaxLow; ++s)
        if (NT - 1 - tid + s * NT < npl) aK[s] = pair_sum(aK[s], ut + li[s], ut + lj[s]);
      pt += n;
      ut += (size_t)n * us;
      ub += (size_t)n * us;
    }
  };
  if (kept) {
    // every U-value of the slice first, kept for the data moments and the outflow
    for (int base = 0; base < 2 * np; base += a.ev_rows) {
      const int n = min(a.ev_rows, 2 * np - base);
      for (int id = tid; id < n; id += blockDim.x) {
        const int row = base + id;
        const int pt = row < np ? row : row - np, k = pt / QK;
        map_rule(sPt + id * (DIM + 2), e0 + k, pt - k * QK, (row < np) != ADJ);
      }
      eval_uvalues_block<DIM, T>(a, n, sPt, sM, sKeep + (size_t)base * us);
    }
    // (the evaluation's buffer may share the Grams' region)
    for (int id = tid; id < NG * ((DIM + 1) * npl + npair); id += blockDim.x) sPG[id] = R::zero();   // PG, PH, PGb contiguous
    __syncthreads();
    gram_points(e0 * QK, e1 * QK, ADJ ? sKI : sKeep, ADJ ? sKeep : sKI);
  } else {
    // chunks of points: U-values at the top, then at the bottom
    const int p0 = SPLIT ? q0 : e0 * QK, p1 = SPLIT ? q1 : e1 * QK;
    for (int base = p0; base < p1; base += CH) {
      const int nq = min(CH, p1 - base);
      for (int id = tid; id < 2 * nq; id += blockDim.x) {
        const int side = id / nq, pt = base + id - side * nq, k = pt / QK;
        map_rule(sPt + id * (DIM + 2), k, pt - k * QK, side == 0);
      }
      eval_uvalues_block<DIM, T>(a, 2 * nq, sPt, sM, sU);
      gram_points(base, base + nq, sU, sU + (size_t)nq * us);
      __syncthreads();
    }
  }
  if (q1 > q0) {
    flush_element(curk);
    flush_group(curg);
  }
  if constexpr (SPLIT) {
    if (!real) {
      wait_deps();
      check_times();
    }
    // this CTA's right-hand sides at every point of the patch (forward: the
    // bottom points; adjoint: the top points): the moments are complete in
    // this CTA and take no cluster reduction
    prefetch_front(0, min(CH, NP));
    for (int base = 0; base < NP; base += CH) {
      const int nq = min(CH, NP - base);
      for (int id = tid; id < nq; id += blockDim.x) {   // (eval_uvalues_block's first reads: by the same threads)
        const int qg = base + id, k = qg / Q, q = qg % Q;
        map_point(sPt + id * (DIM + 2), k, q, ADJ);
      }
      data_coefs(base, nq, sCB, cbs, false);
      if (base + CH < NP) prefetch_front(base + CH, min(CH, NP - base - CH));
      eval_uvalues_block<DIM, T>(a, nq, sPt, sM, sU);
      if (tc_on) {
        if (base > 0) tc_mom_finish();   // the previous chunk's products ran meanwhile
        tc_mom_start(nq);                // (its issue barrier orders this chunk's reads before the next writes)
      } else {
        data_moments(base, nq, sU, Q);
        __syncthreads();
      }
    }
    if (tc_on && NP > 0) tc_mom_finish();
  }

  if constexpr (SPLIT) facet_phase();
  csync();
  if (SPLIT && !real) {
    real = true;
    if (s_bad) continue;
  }
  // layout [G (NG*npl) | H_m (NG*DIM*npl) | Gbot (NG*npair)]; unused groups hold zeros
  if (CS > 1) cluster_reduce(sPG, sPG, NG * ((DIM + 1) * npl + npair));
  // (split right-hand sides: each CTA's moments, Dirichlet data sums and
  // Neumann partial b already cover every point for its own right-hand sides)
  // (in place: each entry is read and rewritten by the one thread that owns it)
  if (pblk && CS > 1) cluster_reduce(sA, sA, N * N);   // interface and Neumann blocks
  if (NEU && s_nneu > 0) {   // Neumann data (after the Dirichlet sums)
    if (rsplit)
      for (int id = tid; id < nrhs * N; id += blockDim.x) sb[id] = sPBN[id];
    else
      cluster_reduce(sPBN, sb, nrhs * N);
  } else {
    for (int id = tid; id < nrhs * N; id += blockDim.x) sb[id] = R::zero();
  }
  if (nfac > 0) {
    cluster_reduce(sFD, sFD, nfg);
    if (!rsplit && has_g) cluster_reduce(sDD, sDD, nfm);
  }
  csync();   // no CTA leaves or reuses its partials while another still reads them
  // congruence: the ranks form shares of A's entries and store them into rank
  // 0's A; rank 0 alone inverts and solves.  Every CTA holds the same summed
  // partials, so an entry does not depend on which rank forms it.  (The
  // adjoint solves with A^T: it is stored transposed.)
  {
    const T ih2 = R::from(ih * ih), mih = R::from(-ih);
    // top-face form of every material block by the merged tables: entries
    // i <= j of the packed upper triangle, split over the cluster; each entry
    // is stored with its mirror (the form is symmetric, the Dirichlet and
    // interface parts already in A are not)
    // (every CS-th entry: those of the high-degree functions, last, have the most terms)
    const int nent = ng * npair, ment = (nent - rank + CS - 1) / CS;
    if (nfac > 0) {
      // Dirichlet facets, A_D = (c/h) D_t F E^T with E = alpha (c/h) D_t - (1/h) D_n
      // summed over the material's facets, from G_g and Gn_g, added into this
      // CTA's copy of A for the entries this rank forms (each entry and its
      // mirror: one item each)
      for (int id = tid; id < 2 * ment; id += blockDim.x) {
        const int e_ = rank + (id >> 1) * CS, g = e_ / npair, pp = e_ % npair;
        const int ij = __ldg(a.pair_ij + pp);
        int i = ij >> 16, j = ij & 0xffff;
        if (((id & 1) && i == j) || !((gdir >> g) & 1u)) continue;
        if (id & 1) {
          const int t_ = i;
          i = j;
          j = t_;
        }
        const int e2 = i * nb + j;
        const T* Fg = sFD + (size_t)g * (DIM + 1) * npl;
        T a0 = R::zero(), am = R::zero();
        for (int e = __ldg(a.ft_ptr + e2), e1 = __ldg(a.ft_ptr + e2 + 1); e < e1; ++e)
          a0 = Fac<T>::acc(a0, Fg[__ldg(a.ft_idx + e)], a.ft_coef, a.ft_coefd, e);
        for (int e = __ldg(a.fm_ptr + e2), e1 = __ldg(a.fm_ptr + e2 + 1); e < e1; ++e) {
          const int c0 = __ldg(a.fm_idx + e);   // (derivative direction << 16) | pair
          am = Fac<T>::acc(am, Fg[(size_t)(1 + (c0 >> 16)) * npl + (c0 & 0xffff)], a.fm_coef, a.fm_coefd, e);
        }
        const double cf = s_gc[g];
        const T ad = R::mul(R::from(cf * ih), R::fma(mih, R::norm(am), R::mul(R::from(a.alpha * cf * ih), R::norm(a0))));
        const size_t o = (size_t)(g * nb + i) * N + g * nb + j;
        sA[o] = R::add(sA[o], ad);
      }
      __syncthreads();
    }
    for (int id = rank + tid * CS; id < nent; id += NT * CS) {
      const int g = id / npair, pp = id % npair;
      const int ij = __ldg(a.pair_ij + pp), i = ij >> 16, j = ij & 0xffff;
      const T* SG = sSG + (size_t)g * npl;
      const T* SH = sSG + (size_t)(NG + g * DIM) * npl;
      const T* SGb = sSG + (size_t)NG * (DIM + 1) * npl + (size_t)g * npair;
      T tg0 = R::zero(), tg1 = R::zero(), th0 = R::zero(), th1 = R::zero();
      {
        const int e0 = __ldg(a.cg_ptr + pp), e1 = __ldg(a.cg_ptr + pp + 1);
        int e = e0;
        for (; e + 1 < e1; e += 2) {
          tg0 = Fac<T>::acc(tg0, SG[__ldg(a.cg_idx + e)], a.cg_coef, a.cg_coefd, e);
          tg1 = Fac<T>::acc(tg1, SG[__ldg(a.cg_idx + e + 1)], a.cg_coef, a.cg_coefd, e + 1);
        }
        if (e < e1) tg0 = Fac<T>::acc(tg0, SG[__ldg(a.cg_idx + e)], a.cg_coef, a.cg_coefd, e);
      }
      {
        const int e0 = __ldg(a.ch_ptr + pp), e1 = __ldg(a.ch_ptr + pp + 1);
        int e = e0;
        for (; e + 1 < e1; e += 2) {
          const int c0 = __ldg(a.ch_idx + e), c1 = __ldg(a.ch_idx + e + 1);
          th0 = Fac<T>::acc(th0, SH[(c0 >> 16) * npl + (c0 & 0xffff)], a.ch_coef, a.ch_coefd, e);
          th1 = Fac<T>::acc(th1, SH[(c1 >> 16) * npl + (c1 & 0xffff)], a.ch_coef, a.ch_coefd, e + 1);
        }
        if (e < e1) {
          const int c0 = __ldg(a.ch_idx + e);
          th0 = Fac<T>::acc(th0, SH[(c0 >> 16) * npl + (c0 & 0xffff)], a.ch_coef, a.ch_coefd, e);
        }
      }
      const T t = R::fma(R::from(s_gc[g]), R::add(R::norm(th0), R::norm(th1)), R::add(R::norm(tg0), R::norm(tg1)));
      const T val = R::fma(ih2, t, SGb[pp]);
      const size_t o = (size_t)(g * nb + i) * N + g * nb + j;
      A0[o] = R::add(sA[o], val);
      if (i != j) {
        const size_t o2 = (size_t)(g * nb + j) * N + g * nb + i;
        A0[o2] = R::add(sA[o2], val);
      }
    }
  }
  csync();   // rank 0 holds the assembled A
  if constexpr (SPLIT) {
    // every CTA solves for its own right-hand sides with its own copy of A
    if (rank != 0)
      for (int id = tid; id < N * N; id += blockDim.x) sA[id] = A0[id];
    csync();   // rank 0's A is read before any CTA's solve overwrites its own
  }
  if (rank == 0 || SPLIT) {
    if constexpr (ADJ) {   // solve with A^T
      for (int id = tid; id < N * N; id += blockDim.x) {
        const int i = id / N, j = id % N;
        if (i < j) {
          const T t = sA[id];
          sA[id] = sA[j * N + i];
          sA[j * N + i] = t;
        }
      }
      __syncthreads();
    }
    // ---------------- inverse of the equilibrated matrix ----------------
    // Both precisions: F = (D A D)^-1, D powers of two near |diag A|^-1/2
    // (exact scaling), by Gauss-Jordan in float-float without row
    // interchanges.  With ~48 bits F's error in the refinement below is
    // kappa(A) 2^-46 per step: one or two steps instead of the 3 to 40 that
    // a binary32 inverse took at p = 4, 5, and the direct LU is rarely
    // needed.  The inverse costs more than a binary32 one, but it is formed
    // before the wait, off the chain of dependent tents.
    // Every tent matrix has a positive definite symmetric part (testing the
    // tent system with V = U_h gives x^T A x = 1/2 int_top Q_g(u) + 1/2 int_bot
    // Q_g(u_b) + int_bot U^2 + the dissipative boundary and interface terms > 0),
    // and so has each of its Schur complements: elimination without
    // interchanges does not break down.  The direct LU of the fallback keeps
    // partial pivoting on Dirichlet and interface tents.
    for (int i = tid; i < N; i += blockDim.x) {
      const float d = fabsf(R::hi(sA[i * N + i]));
      sEq[i] = (d > 0.f && isfinite(d)) ? pow2_rsqrt(d) : 1.f;
    }
    __syncthreads();
    auto bad_pivot = [&](float pv) {
      // binary64: the refinement then fails and the direct LU decides
      if (!(fabsf(pv) > 0.f) || !isfinite(pv)) {
        if (MIXED && lane == 0) flag_error(a, TP_ERR_SINGULAR, tent);
        return true;
      }
      return false;
    };
    // register path: row warp + NW s of the matrix in gr[s], columns lane + 32 c.
    // Blocks of four steps K = {k..k+3} per barrier: with S_K the block's
    // pivot rows at its start, every warp reduces S_K by the four steps
    // itself (P = [S_KK^-1 | S_KK^-1 S_KJ] in the pivot and the other
    // columns), and a row i outside K becomes
    //   (columns of K set to 0, the others kept) - sum_b s_{i,k+b} P_b,
    // which is the four single steps taken at once (block Gauss-Jordan).
    // (Against one step per barrier in shared memory: 36 unknowns 40 us.)
    auto invert_in_registers = [&](auto cols) {
      constexpr int NC = decltype(cols)::value, NS = (32 * NC + NW - 1) / NW;
      dd* pbuf = reinterpret_cast<dd*>(sm + a.off_rc);   // 2 x 4 pivot rows of 32 NC entries
      dd gr[NS][NC];
#pragma unroll
      for (int s_ = 0; s_ < NS; ++s_)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int i = warp + NW * s_, j = lane + 32 * c;
          gr[s_][c] = {0.f, 0.f};
          if (i < N && j < N) gr[s_][c] = R::scaled(sA[i * N + j], sEq[i] * sEq[j]);
        }
      for (int k = 0, blk = 0; k < N; k += 4, ++blk) {
        const int kb = min(4, N - k), kl = k & 31, kcw = k >> 5;   // (a block lies in one column group: 4 divides 32)
        dd* pb = pbuf + (blk & 1) * 4 * 32 * NC;
        // the owners publish the block's pivot rows (rows k..k+3 are on warps
        // k % NW .. k % NW + 3, slot k / NW)
        if (warp >= k % NW && warp < k % NW + kb) {
#pragma unroll
          for (int s_ = 0; s_ < NS; ++s_)
            if (s_ == k / NW) {
#pragma unroll
              for (int c = 0; c < NC; ++c) pb[(warp - k % NW) * 32 * NC + 32 * c + lane] = gr[s_][c];
            }
        }
        __syncthreads();
        dd Pr[4][NC];
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            Pr[b][c] = {0.f, 0.f};
            if (b < kb) Pr[b][c] = pb[b * 32 * NC + 32 * c + lane];
          }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (b >= kb) break;
          const int kc = kl + b;
          dd mm[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            dd x = Pr[r][0];
#pragma unroll
            for (int c = 1; c < NC; ++c)
              if (c == kcw) x = Pr[r][c];
            mm[r] = {__shfl_sync(0xffffffffu, x.hi, kc), __shfl_sync(0xffffffffu, x.lo, kc)};
          }
          dd pv = mm[b];
          if (bad_pivot(pv.hi)) pv = {1.f, 0.f};
          const dd rp = dd_rcp(pv);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const bool own = c == kcw && lane == kc;
            const dd pn = own ? rp : dd_mul(Pr[b][c], rp);
#pragma unroll
            for (int r = 0; r < 4; ++r)
              if (r != b) {
                const dd x0 = own ? dd{0.f, 0.f} : Pr[r][c];
                Pr[r][c] = Ar<dd>::norm(Ar<dd>::accn(x0, mm[r], pn));
              }
            Pr[b][c] = pn;
          }
        }
        const bool kcol = lane >= kl && lane < kl + kb;
#pragma unroll
        for (int s_ = 0; s_ < NS; ++s_) {
          const int i = warp + NW * s_, bi = i - k;
          if (i >= N) continue;
          // this row in the pivot columns (block-start values)
          dd x = gr[s_][0];
#pragma unroll
          for (int c = 1; c < NC; ++c)
            if (c == kcw) x = gr[s_][c];
          dd ml[4];
#pragma unroll
          for (int b = 0; b < 4; ++b)
            ml[b] = {-__shfl_sync(0xffffffffu, x.hi, kl + b), -__shfl_sync(0xffffffffu, x.lo, kl + b)};
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            if (bi >= 0 && bi < kb) {
              gr[s_][c] = bi == 0 ? Pr[0][c] : bi == 1 ? Pr[1][c] : bi == 2 ? Pr[2][c] : Pr[3][c];
            } else {
              dd y = (c == kcw && kcol) ? dd{0.f, 0.f} : gr[s_][c];
#pragma unroll
              for (int b = 0; b < 4; ++b) y = Ar<dd>::acc(y, ml[b], Pr[b][c]);
              gr[s_][c] = Ar<dd>::norm(y);
            }
          }
        }
      }
#pragma unroll
      for (int s_ = 0; s_ < NS; ++s_)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int i = warp + NW * s_, j = lane + 32 * c;
          if (i < N && j < N) sF_[i * N + j] = gr[s_][c];
        }
    };
    if (N <= 32) {
      invert_in_registers(std::integral_constant<int, 1>{});
    } else if (N <= 64) {
      invert_in_registers(std::integral_constant<int, 2>{});
    } else if (WIDE && N <= 96) {
      if constexpr (WIDE) invert_in_registers(std::integral_constant<int, 3>{});
    } else {
      // shared-memory path, one step per barrier: every entry belongs to one
      // thread (rows over warps, columns over lanes), which also writes the
      // next pivot row and column into a second buffer
      dd* rowb = reinterpret_cast<dd*>(sm + a.off_rc);   // 2 x N pivot rows, 2 x N pivot columns
      dd* colb = rowb + 2 * N;
      for (int i = warp; i < N; i += NW)
        for (int j = lane; j < N; j += 32) {
          const dd x = R::scaled(sA[i * N + j], sEq[i] * sEq[j]);
          sF_[i * N + j] = x;
          if (i == 0) rowb[j] = x;
          if (j == 0) colb[i] = x;
        }
      __syncthreads();
      for (int k = 0; k < N; ++k) {
        const dd *pr = rowb + (k & 1) * N, *pc = colb + (k & 1) * N;
        dd *nr = rowb + ((k + 1) & 1) * N, *nc = colb + ((k + 1) & 1) * N;
        dd pv = pr[k];
        if (bad_pivot(pv.hi)) pv = {1.f, 0.f};
        const dd rp = dd_rcp(pv);
        for (int i = warp; i < N; i += NW) {
          const dd l0 = dd_mul(pc[i], rp), l = {-l0.hi, -l0.lo};
          for (int j = lane; j < N; j += 32) {
            dd x;
            if (i == k) x = j == k ? rp : dd_mul(pr[j], rp);
            else if (j == k) x = l;
            else x = Ar<dd>::norm(Ar<dd>::acc(sF_[i * N + j], l, pr[j]));
            sF_[i * N + j] = x;
            if (i == k + 1) nr[j] = x;
            if (j == k + 1) nc[i] = x;
          }
        }
        __syncthreads();
      }
    }
  }
  if (!real) {
    wait_deps();
    check_times();
  }
  // ---------------- the data of the bottom front (adjoint: of the top) ----------------
  if constexpr (!SPLIT) {
    const T* U = sKI;
    if (!kept && !srule) {
      for (int base = q0; base < q1; base += CH) {
        const int nq = min(CH, q1 - base);
        for (int id = tid; id < nq; id += blockDim.x) map_point(sPt + id * (DIM + 2), (base + id) / Q, (base + id) % Q, ADJ);
        data_coefs(base, nq, sCB, cbs, false);
        eval_uvalues_block<DIM, T>(a, nq, sPt, sM, sU);
        data_moments(base, nq, sU, Q);
        __syncthreads();
      }
    } else if (srule) {
      // U on a face is in P_p, so sum_q w_q f(q) u(q) = sum_s u(X_s) [sum_q w_q w_s K(X_s, x_q) f(q)]
      // (FaceRule): the data go to the rule's points, a few elements at a time
      const int S = a.S, raws = a.raw_el * Q;
      for (int eb = e0; eb < e1; eb += EC) {
        const int ne = min(EC, e1 - eb);
        if (eb > e0) __syncthreads();
        data_coefs(eb * Q, ne * Q, sRaw, raws, true);
        __syncthreads();
        for (int id = tid; id < nrhs * C * ne * S; id += blockDim.x) {
          const int rc = id / (ne * S), pt = id - rc * (ne * S), k = pt / S, q_ = pt - k * S;
          const T *f = sRaw + (size_t)rc * raws + k * Q, *w = (ADJ ? sTF : sTP) + q_ * a.tf_stride;
          T t0 = R::zero(), t1 = R::zero();
          int q = 0;
          for (; q + 1 < Q; q += 2) {
            t0 = R::acc(t0, w[q], f[q]);
            t1 = R::acc(t1, w[q + 1], f[q + 1]);
          }
          if (q < Q) t0 = R::acc(t0, w[q], f[q]);
          sCB[(size_t)rc * cbs + pt] = R::mul(R::from(ADJ ? s_isdet[eb + k] : s_sdet[eb + k]), R::add(R::norm(t0), R::norm(t1)));
        }
        __syncthreads();
        if (!kept) {
          for (int id = tid; id < ne * S; id += blockDim.x)
            map_rule(sPt + id * (DIM + 2), eb + id / S, id % S, ADJ);
          eval_uvalues_block<DIM, T>(a, ne * S, sPt, sM, sU);
        }
        data_moments(eb * S, ne * S, kept ? U + (size_t)(eb - e0) * S * us : sU, S);
      }
    } else {
      for (int base = 0; base < np; base += a.cb_pts) {
        const int nq = min(a.cb_pts, np - base);
        if (base > 0) __syncthreads();
        data_coefs(q0 + base, nq, sCB, cbs, false);
        __syncthreads();
        data_moments(q0 + base, nq, U + (size_t)base * us, Q);
      }
    }
  }
  csync();
  if (real || !s_bad) break;
  real = true;
  }   // assembly
  if (rank == 0 || SPLIT) {
  // (rank 0 sums the partial moments; the others keep theirs until its b is solved)
  if (!SPLIT && CS > 1) {
    for (int id = tid; id < ng * nmom; id += blockDim.x) sPM[id] = cluster_sum(sPM, id);
    __syncthreads();
  }
  {
    // the C terms of an entry (gamma, (c/h) D_t alpha, -(1/h) D_m beta_m) on
    // neighbouring lanes, added by shuffles: the chain of dependent tents
    // waits for the longest of them instead of their sum
    const T mih = R::from(-ih);
    constexpr int LB = C <= 4 ? 4 : 8;
    for (int base = 0; base < nrhs * N * LB; base += NT) {
      const int id = base + tid, it = id / LB, cc = id % LB;
      const bool live = it < nrhs * N && cc < C;
      const int r = it / N, Rw = it - r * N, g = Rw / nb, i = Rw - g * nb;
      T t = R::zero();
      if (live) {
        const T* M = sSM + (size_t)g * nmom + ((size_t)r * C + cc) * nb;   // gamma, alpha, beta_1..beta_n
        t = cc == 0 ? M[i] : R::mul(cc == 1 ? R::from(s_gc[g] * ih) : mih, rel_apply<DIM, T>(a, i, cc - 1, M));
        // Dirichlet data: b_D = E' delta summed over g's facets,
        // E' = alpha (c/h) D_t + (1/h) D_n
        if (has_g && cc > 0 && ((gdir >> g) & 1u)) {
          const T* Dg = sDD + (size_t)(g * (DIM + 1) + cc - 1) * nrhs * nl + (size_t)r * nl;
          t = R::fma(R::from(cc == 1 ? a.alpha * s_gc[g] * ih : ih), rel_apply<DIM, T>(a, i, cc - 1, Dg), t);
        }
      }
#pragma unroll
      for (int o = 1; o < LB; o <<= 1) t = R::add(t, shfl_xor_t(t, o));
      if (live && cc == 0) {
        const size_t o = (size_t)r * N + Rw;
        sb[o] = R::add(sb[o], t);
      }
    }
  }
  __syncthreads();

  // ---------------- phase 3: solve ----------------
  // x = D F D b, then x += D F D (b - A x) with the residual in the path's
  // precision (binary64, or float-float for MIXED) until the correction stops
  // shrinking; a refinement that does not settle falls back to a direct
  // binary64 LU.
  const bool lu_pivoting = extra || ng > 1;
  bool refined = false;
  {
    dd* sZ = reinterpret_cast<dd*>(sm + a.off_z);           // nrhs*N  scaled residual
    T* sX = reinterpret_cast<T*>(sm + a.off_x);             // nrhs*N  iterate
    float prev = 0.f;
    const int maxit = min(a.max_refine, kMaxRefine);
    for (int it = 0; it < maxit; ++it) {
      // residual b - A x scaled by D (the first iterate is x = 0: the residual
      // is b), each row split over 8 lanes of one warp
      if (it == 0) {
        for (int id = tid; id < nrhs * N; id += blockDim.x) sZ[id] = R::scaled(sb[id], sEq[id % N]);
      } else {
        for (int base8 = 0; base8 < nrhs * N * 8; base8 += blockDim.x) {
          const int id = base8 + tid, item = id >> 3, sub = id & 7;
          T t = R::zero();
          if (item < nrhs * N) {
            const int r = item / N, i = item % N;
            const T* xr = sX + (size_t)r * N;
            for (int j = sub; j < N; j += 8) t = R::accn(t, sA[i * N + j], xr[j]);
            t = R::norm(t);
          }
          for (int o = 4; o > 0; o >>= 1) t = R::add(t, shfl_xor_t(t, o));
          if (sub == 0 && item < nrhs * N) sZ[item] = R::scaled(R::add(sb[item], t), sEq[item % N]);
        }
      }
      __syncthreads();
      // x += D F z, each row split over 8 lanes
      // (the scale |x| of the stop test is taken from the first iterate)
      float dmax = 0.f;
      for (int base8 = 0; base8 < nrhs * N * 8; base8 += blockDim.x) {
        const int id = base8 + tid, item = id >> 3, sub = id & 7;
        dd z = {0.f, 0.f};
        if (item < nrhs * N) {
          const int r = item / N, i = item % N;
          const dd* zr = sZ + (size_t)r * N;
          for (int j = sub; j < N; j += 8) z = Ar<dd>::acc(z, sF_[i * N + j], zr[j]);
          z = Ar<dd>::norm(z);
        }
        for (int o = 4; o > 0; o >>= 1) z = dd_add(z, shfl_xor_t(z, o));
        if (sub == 0 && item < nrhs * N) {
          const float e = sEq[item % N];
          const dd dx = {__fmul_rn(z.hi, e), __fmul_rn(z.lo, e)};
          sX[item] = it == 0 ? R::of(dx) : R::add(sX[item], R::of(dx));
          dmax = fmaxf(dmax, fabsf(dx.hi));
          if (!isfinite(dx.hi)) dmax = dx.hi;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const float other = __shfl_xor_sync(0xffffffffu, dmax, o);
        dmax = (isfinite(dmax) && !(other <= dmax)) ? other : dmax;   // (the larger; a non-finite one stays)
      }
      if (lane == 0) s_red[it == 0][warp] = dmax;
      __syncthreads();
      if (it == 0) continue;
      float dm = 0.f, xm = 0.f;
      bool fin = true;
      for (int w = 0; w < NW; ++w) {
        dm = fmaxf(dm, s_red[0][w]);
        xm = fmaxf(xm, s_red[1][w]);
        fin = fin && isfinite(s_red[0][w]) && isfinite(s_red[1][w]);
      }
      if (!fin) break;   // the direct LU decides
      if (it == 1) prev = xm;   // the first iterate counts as the correction of x = 0
      // stop once the correction is at the resolution of the residual's
      // precision, or once it stops shrinking at a small level (the residual's
      // rounding then limits the accuracy)
      // (a correction that stalls above floor_ of the solution, or no
      // convergence in kMaxRefine steps, sends the tent to the direct LU)
      const float tiny = MIXED ? 4e-15f : 2.5e-16f, floor_ = MIXED ? 1e-10f : 1e-12f;
      const float stall = 0.5f;
      // (the next correction is predicted as dm * (dm / prev) once the
      // corrections shrink fast; stop when that is below the resolution too)
      const bool done = dm <= tiny * xm || (it >= 2 && dm > stall * prev && dm <= floor_ * xm) ||
                        (dm <= 0.01f * prev && 4.f * dm * (dm / prev) <= tiny * xm);
      prev = dm;
      if (done) {
        refined = true;
        if (a.solve_stats != nullptr && tid == 0) atomicAdd(a.solve_stats + 1 + min(it + 1, kMaxRefine), 1ull);
        break;
      }
      // (the next iteration writes s_red only after its first barrier)
    }
    if (refined) {
      for (int id = tid; id < nrhs * N; id += blockDim.x) sb[id] = sX[id];
      __syncthreads();
    }
  }
  if (!refined) {   // direct binary64 LU (the mixed path converts A and b to binary64 first)
    if (a.solve_stats != nullptr && tid == 0) atomicAdd(a.solve_stats, 1ull);
    __syncthreads();
    double* dA = reinterpret_cast<double*>(sA);   // in place: a float-float pair and a double share 8 bytes
    double* db = reinterpret_cast<double*>(sb);
    if constexpr (MIXED) {
      for (int id = tid; id < N * N; id += blockDim.x) {
        const T v = sA[id];
        dA[id] = R::to(v);
      }
      for (int id = tid; id < nrhs * N; id += blockDim.x) {
        const T v = sb[id];
        db[id] = R::to(v);
      }
      __syncthreads();
    }
    double* sXd = reinterpret_cast<double*>(sm + a.off_x);   // nrhs*N  solution during back substitution
    auto pivot_recip = [&](double piv, int k) {
      if (!(fabs(piv) > 0.0) || !isfinite(piv)) {
        flag_error(a, TP_ERR_SINGULAR, tent);
        piv = 1.0;
      }
      sRD[k] = recip(piv);
    };
    if (!lu_pivoting) {
      // A is symmetric positive definite: LU without interchanges, b eliminated
      // alongside, one barrier per step.  Step k updates rows and columns > k;
      // every thread forms the multiplier a_ik / a_kk it needs, and the thread
      // that updates a_{k+1,k+1} forms the next reciprocal pivot.
      if (tid == 0) pivot_recip(dA[0], 0);
      __syncthreads();
      for (int k = 0; k + 1 < N; ++k) {
        const double rp = sRD[k];
        const int rem = N - k - 1, wdt = rem + nrhs;
        for (int id = tid; id < rem * wdt; id += blockDim.x) {
          const int i = k + 1 + id / wdt, jj = id % wdt;
          const double l = dA[i * N + k] * rp;
          if (jj < rem) {
            const int j = k + 1 + jj;
            const double t = fma(-l, dA[k * N + j], dA[i * N + j]);
            dA[i * N + j] = t;
            if (id == 0) pivot_recip(t, k + 1);
          } else {
            const int r = jj - rem;
            db[r * N + i] = fma(-l, db[r * N + k], db[r * N + i]);
          }
        }
        __syncthreads();
      }
    } else {
      // LU with partial pivoting (Dirichlet and interface tents), b eliminated alongside
      for (int k = 0; k < N; ++k) {
        if (warp == 0) {
          // |a_ik| compared through the bit patterns (non-negative doubles order as integers)
          unsigned long long best = 0ull;
          int bi = k;
          for (int i = k + lane; i < N; i += 32) {
            const unsigned long long bits = (unsigned long long)__double_as_longlong(fabs(dA[i * N + k]));
            if (bits > best || (bits == best && i < bi)) {
              best = bits;
              bi = i;
            }
          }
          for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ob = __shfl_down_sync(0xffffffffu, best, o);
            const int oi = __shfl_down_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
              best = ob;
              bi = oi;
            }
          }
          if (lane == 0) {
            s_piv = bi;
            pivot_recip(dA[bi * N + k], k);
          }
        }
        __syncthreads();
        const int pr = s_piv;
        if (pr != k) {
          for (int j = tid; j < N; j += blockDim.x) {
            const double t = dA[k * N + j];
            dA[k * N + j] = dA[pr * N + j];
            dA[pr * N + j] = t;
          }
          for (int r = tid; r < nrhs; r += blockDim.x) {
            const double t = db[r * N + k];
            db[r * N + k] = db[r * N + pr];
            db[r * N + pr] = t;
          }
          __syncthreads();
        }
        const double rp = sRD[k];
        const int rem = N - k - 1, wdt = rem + nrhs;
        for (int id = tid; id < rem * wdt; id += blockDim.x) {
          const int i = k + 1 + id / wdt, jj = id % wdt;
          const double l = dA[i * N + k] * rp;
          if (jj < rem) {
            const int j = k + 1 + jj;
            dA[i * N + j] = fma(-l, dA[k * N + j], dA[i * N + j]);
          } else {
            const int r = jj - rem;
            db[r * N + i] = fma(-l, db[r * N + k], db[r * N + i]);
          }
        }
        __syncthreads();
      }
    }
    // back substitution, one barrier per step: x_k = b_k / u_kk into sXd, and
    // b_i -= u_ik x_k for i < k (every thread forms x_k itself)
    for (int k = N - 1; k >= 0; --k) {
      const double rp = sRD[k];
      for (int id = tid; id < (k + 1) * nrhs; id += blockDim.x) {
        const int r = id / (k + 1), i = id % (k + 1);
        const double xk = db[r * N + k] * rp;
        if (i == k) sXd[r * N + k] = xk;
        else db[r * N + i] = fma(-dA[i * N + k], xk, db[r * N + i]);
      }
      __syncthreads();
    }
    for (int id = tid; id < nrhs * N; id += blockDim.x) db[id] = sXd[id];
    if constexpr (MIXED) {
      __syncthreads();
      for (int id = tid; id < nrhs * N; id += blockDim.x) {
        const double v = db[id];
        sb[id] = R::from(v);
      }
    }
  }
  }   // rank 0 (every rank with split right-hand sides)
  csync();   // the solution is in rank 0's b (split right-hand sides: in each CTA's own)
  if (rank != 0 && !rsplit) {
    const T* b0 = cluster.map_shared_rank(sb, 0);
    for (int id = tid; id < nrhs * N; id += blockDim.x) sb[id] = b0[id];
  }
  if constexpr (!ADJ) {
    // the forward solution kept for the reverse sweep of the wave-speed gradient
    if (a.xsave != nullptr && (rank == 0 || rsplit)) {
      const int NBg = NG * nb;
      double* xs = a.xsave + (size_t)(tent - a.xbase) * a.xs_stride + (size_t)(rsplit ? rank * nrhs : 0) * NBg;
      for (int id = tid; id < nrhs * N; id += blockDim.x) xs[(size_t)(id / N) * NBg + id % N] = R::to(sb[id]);
    }
  }
  __syncthreads();

  // ---------------- phase 4: outflow at this CTA's top points (adjoint: bottom points) ----------------
  // coefficient vectors of U_h, v_h, sigma_h in terms of U-values, per material: y = D^T x_g
  for (int id = tid; id < ng * nmom; id += blockDim.x) {
    const int g = id / nmom, rest = id % nmom;
    const int r = rest / (C * nb), rem = rest % (C * nb), cc = rem / nb, kk = rem % nb;
    const T* xg = sb + (size_t)r * N + g * nb;
    T t;
    if (cc == 0) t = xg[kk];
    else t = R::mul(R::from(cc == 1 ? s_gc[g] * ih : -ih), relT_apply<DIM, T>(a, kk, cc - 1, xg));
    sY[id] = t;
  }
  __syncthreads();
  // the points whose front values this CTA overwrites (split right-hand
  // sides: this CTA's own right-hand sides at every point)
  const int o0 = rsplit ? 0 : q0, o1 = rsplit ? NP : q1;
  // this tent's bottom front, for the reverse sweep of the wave-speed gradient
  auto saved_front = [&](int r) {
    return a.fsave + ((size_t)(__ldg(a.tent_el + tent) - a.fbase) * (SPLIT ? CS * nrhs : nrhs) +
                      (size_t)((SPLIT ? rank * nrhs : 0) + r) * P) * Q * C;
  };
  if constexpr (!ADJ) {
    if (a.fsave != nullptr) {
      for (int id = tid; id < nrhs * (o1 - o0) * C; id += blockDim.x) {
        const int r = id / ((o1 - o0) * C), qc = o0 * C + id - r * ((o1 - o0) * C), k = qc / (Q * C);
        saved_front(r)[qc] = __ldcg(front + ((int64_t)r * a.ne + s_el[k]) * Q * C + (qc - k * Q * C));
      }
      __syncthreads();
    }
  }
  // ---------------- energy lost in the tent (forward sweep, when tracked) ----------------
  // Testing the tent system with V = U_h and using d/dt e + div(v sigma) = 0
  // inside the Trefftz tent: 1/2 int_top Q_{g_t}(u) = 1/2 int_bot Q_{g_b}(u_b) - D,
  //   D = 1/2 int_bot Q_{g_b}(u - u_b) + int_bot (U - U_b) U
  //     + int_D [alpha v^2 - g_D (alpha v - sigma.n)] + int_N [beta (sigma.n)^2 - g_N (beta sigma.n - v)]
  //     + int_time [alpha (v+ - v-)^2 + beta ((sigma+ - sigma-).n)^2]
  // (eq. 2.5, eq. 4.1, Section 6.5; Q_g(w) = c^-2 w_v^2 + |w_s|^2 - 2 w_v w_s.g).
  // Point values of the solution come from the outflow vectors and U-values
  // scaled by sqrt(w); the stored bottom values are read before this CTA
  // overwrites them below.  Summed over the sweep: E(T) = E(0) - sum D.
  if constexpr (!ADJ) {
    if (a.diss != nullptr) {
      double* sDis = reinterpret_cast<double*>(sDel);   // nrhs partial sums (sDel is dead after phase 2)
      double* sFb = reinterpret_cast<double*>(sCB);     // CH*nrhs*C stored values (sCB is dead after phase 1)
      double* sGdd = reinterpret_cast<double*>(sGd);    // CH*nrhs boundary data (dead after phase 2)
      for (int id = tid; id < nrhs; id += blockDim.x) sDis[id] = 0.0;
      __syncthreads();
      auto fieldv = [&](int g, int r, int cc, const T* u) {   // sqrt(w) times component cc of the solution
        const T* y = sY + (size_t)g * nmom + ((size_t)r * C + cc) * nb;
        T t = R::zero();
        for (int j = 0; j < (cc == 0 ? nb : nl); ++j) t = R::acc(t, y[j], u[j]);
        return R::to(R::norm(t));
      };
      // (a) bottom face: the jump to the stored front and the recovery term
      for (int base = o0; base < o1; base += CH) {
        const int nq = min(CH, o1 - base);
        for (int id = tid; id < nq; id += blockDim.x) {
          const int qg = base + id;
          map_point(sPt + id * (DIM + 2), qg / Q, qg % Q, false);
        }
        for (int id = tid; id < nq * nrhs; id += blockDim.x) {
          const int ql = id / nrhs, r = id % nrhs, qg = base + ql, k = qg / Q, q = qg % Q;
          const double sw = __ldg(a.sqw + q) * s_sdet[k];
          const double* f = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
#pragma unroll
          for (int cc = 0; cc < C; ++cc) sFb[(size_t)id * C + cc] = sw * __ldcg(f + cc);
        }
        eval_uvalues_block<DIM, T>(a, nq, sPt, sM, sU);
        for (int id = tid; id < nq * nrhs; id += blockDim.x) {
          const int ql = id / nrhs, r = id % nrhs, k = (base + ql) / Q, g = s_grp[k];
          const T* u = sU + (size_t)ql * us;
          const double* fb = sFb + (size_t)id * C;
          const double Uh = fieldv(g, r, 0, u), dv = fieldv(g, r, 1, u) - fb[1];
          double ds2 = 0.0, dsg = 0.0;
          for (int d = 0; d < DIM; ++d) {
            const double ds = fieldv(g, r, 2 + d, u) - fb[2 + d];
            ds2 = fma(ds, ds, ds2);
            dsg = fma(ds, s_gb[k][d], dsg);
          }
          atomicAdd(sDis + r, 0.5 * (s_gic2[g] * dv * dv + ds2 - 2.0 * dv * dsg) + (Uh - fb[0]) * Uh);
        }
        __syncthreads();
      }
      // (b) vertical faces: Dirichlet, then interface, then Neumann facets,
      // each facet's points split over the cluster (split right-hand sides: every point)
      const int fsl = (Q + CS - 1) / CS;
      const int p0 = rsplit ? 0 : min(Q, rank * fsl), p1 = rsplit ? Q : min(Q, p0 + fsl);
      for (int f = 0; f < nfac + nif + nneu; ++f) {
        const bool ifc = f >= nfac && f < nfac + nif, neu = NEU && f >= nfac + nif;
        const int gp = s_fg[f], gm = s_fg2[f];
        for (int base = p0; base < p1; base += CH) {
          const int nq = min(CH, p1 - base);
          for (int id = tid; id < nq; id += blockDim.x) {
            const int q = base + id;
            double xt[DIM + 1];
            for (int d = 0; d <= DIM; ++d) xt[d] = 0.0;
            for (int i = 0; i < NV; ++i) {
              const double l = __ldg(a.bary + q * NV + i);
              for (int d = 0; d <= DIM; ++d) xt[d] = fma(l, s_fP[f][i][d], xt[d]);
            }
            const double sw = __ldg(a.sqw + q) * s_fsq[f];
            T* pp = sPt + id * (DIM + 2);
            pp[0] = R::from(s_gc[gp] * (xt[DIM] - tc) * ih);
            for (int d = 0; d < DIM; ++d) pp[1 + d] = R::from((xt[d] - s_xv[d]) * ih);
            pp[DIM + 1] = R::from(sw);
            if (ifc) {
              T* p2 = sPt + (nq + id) * (DIM + 2);
              p2[0] = R::from(s_gc[gm] * (xt[DIM] - tc) * ih);
              for (int d = 0; d < DIM; ++d) p2[1 + d] = pp[1 + d];
              p2[DIM + 1] = pp[DIM + 1];
            } else {
              // the facet's block of boundary data (without Neumann facets: the facet's own index)
              const long long goff = a.tent_gdoff[tent] + (NEU ? (long long)s_fw[f][0] * Q : (long long)f * Q) + q;
              for (int r = 0; r < nrhs; ++r)
                sGdd[id * nrhs + r] = gD != nullptr ? sw * gD[(long long)r * a.n_bnd + goff] : 0.0;
            }
          }
          if (ifc) __syncthreads();   // (the - side's rows are read by other threads than wrote them)
          eval_uvalues_block<DIM, T>(a, ifc ? 2 * nq : nq, sPt, sM, sU);
          for (int id = tid; id < nq * nrhs; id += blockDim.x) {
            const int ql = id / nrhs, r = id % nrhs;
            const T* u = sU + (size_t)ql * us;
            const double vh = fieldv(gp, r, 1, u);
            double sn = 0.0;
            for (int d = 0; d < DIM; ++d) sn = fma(s_fn[f][d], fieldv(gp, r, 2 + d, u), sn);
            double val;
            if (ifc) {
              const T* u2 = sU + (size_t)(nq + ql) * us;
              double sn2 = 0.0;
              for (int d = 0; d < DIM; ++d) sn2 = fma(s_fn[f][d], fieldv(gm, r, 2 + d, u2), sn2);
              const double jv = vh - fieldv(gm, r, 1, u2), js = sn - sn2;
              val = a.alpha * jv * jv + a.beta * js * js;
            } else {
              const double gv = sGdd[id];
              val = neu ? a.beta * sn * sn - gv * (a.beta * sn - vh) : a.alpha * vh * vh - gv * (a.alpha * vh - sn);
            }
            atomicAdd(sDis + r, val);
          }
          __syncthreads();
        }
      }
      double* diss = a.diss + (rsplit ? (size_t)rank * nrhs : 0);
      for (int r = tid; r < nrhs; r += blockDim.x) atomicAdd(diss + r, sDis[r]);
      __syncthreads();
    }
  }
  // ---------------- point outputs (forward sweep, when requested) ----------------
  // U_h at the samples (x_j, t_k) that lie inside this tent: t_bot(x_j) <=
  // t_k < t_top(x_j) on the element of x_j (the host assigns each sample to
  // the one tent that holds it); U_h = sum_j x_j b_j at the mapped point
  // (Remark 3.1)
  if constexpr (!ADJ) {
    if (a.probe_ptr != nullptr) {
      const int s0 = __ldg(a.probe_ptr + tent), ns = __ldg(a.probe_ptr + tent + 1) - s0;
      const int psl = rsplit ? ns : (ns + CS - 1) / CS;
      const int a0 = rsplit ? 0 : min(ns, rank * psl), a1 = rsplit ? ns : min(ns, a0 + psl);
      for (int base = a0; base < a1; base += 2 * CH) {
        const int nq = min(2 * CH, a1 - base);
        for (int id = tid; id < nq; id += blockDim.x) {
          const int smp = s0 + base + id, j = __ldg(a.probe_j + smp), k = __ldg(a.probe_slot + smp);
          const double t = __ldg(a.probe_t + __ldg(a.probe_k + smp));
          double x[DIM];
          for (int d = 0; d < DIM; ++d) x[d] = 0.0;
          for (int i = 0; i < NV; ++i) {
            const double l = __ldg(a.probe_bary + (size_t)j * NV + i);
            for (int d = 0; d < DIM; ++d) x[d] = fma(l, s_X[k][i][d], x[d]);
          }
          T* pp = sPt + id * (DIM + 2);
          pp[0] = R::from(s_gc[s_grp[k]] * (t - tc) * ih);
          for (int d = 0; d < DIM; ++d) pp[1 + d] = R::from((x[d] - s_xv[d]) * ih);
          pp[DIM + 1] = R::one();
        }
        eval_uvalues_block<DIM, T, false>(a, nq, sPt, sM, sU);
        for (int id = tid; id < nq * nrhs; id += blockDim.x) {
          const int ql = id % nq, r = id / nq, smp = s0 + base + ql;
          const int j = __ldg(a.probe_j + smp), kt = __ldg(a.probe_k + smp), k = __ldg(a.probe_slot + smp);
          const T* y = sY + (size_t)s_grp[k] * nmom + (size_t)r * C * nb;   // U_h = u . x_g
          const T* u = sU + (size_t)ql * us;
          T acc = R::zero();
          for (int jj = 0; jj < nb; ++jj) acc = R::acc(acc, y[jj], u[jj]);
          const int rg = (rsplit ? rank * nrhs : 0) + r;
          a.probe_out[((size_t)rg * a.n_probe_t + kt) * a.n_probe + j] = R::to(R::norm(acc));
        }
        __syncthreads();
      }
    }
  }
  // ---------------- wave-speed gradient (reverse sweep, when requested) ----------------
  // With the tents held fixed, J depends on the speed c_g of material g
  // through every tent's maps b = B f_bot, A x = b, f_top = E x (eq. 4.1), so
  //   dJ/dc_g += lambda_top . (dE/dc_g) x + mu^T ((dB/dc_g) f_bot - (dA/dc_g) x),
  // x the tent's forward solution, f_bot the forward front below it,
  // lambda_top the adjoint front at its top points, mu = A^-T E^T lambda_top.
  // With t^ = c (t - t_c)/h (Remark 3.1) the fields F = (U, v, sigma) of a
  // coefficient vector x move with c as
  //   dF/dc = ((t - t_c)/c) F(x') + (0, v/c, 0),   x' = (c/h) D_t^T x
  // (the time derivative of U_h is again in U^p), so every derivative is a
  // point value of the forms of eq. (4.1) and eq. (2.5) on F and dF; the
  // only explicit c of the forms is c^-2 of the top and bottom faces.  Each
  // point's contribution is booked on its element (a facet's on the element
  // of its side): summed over the elements of a material it is dJ/dc of
  // that material.
  if constexpr (ADJ) {
    if (a.dJdc != nullptr) {
      const int NBg = NG * nb;
      T* sYx = reinterpret_cast<T*>(sm + a.off_yg);   // NG*nmom  y(x)
      T* sYxp = sYx + (size_t)NG * nmom;               // NG*nmom  y(x')
      T* sYmp = sYxp + (size_t)NG * nmom;              // NG*nmom  y(mu')
      T* sXf = sYmp + (size_t)NG * nmom;               // nrhs*N   forward solution
      const int rg0 = rsplit ? rank * nrhs : 0;
      {
        const double* xs = a.xsave + (size_t)(tent - a.xbase) * a.xs_stride;
        for (int id = tid; id < nrhs * N; id += blockDim.x) sXf[id] = R::from(xs[(size_t)(rg0 + id / N) * NBg + id % N]);
      }
      for (int k = tid; k < P; k += blockDim.x) s_gel[k] = 0.0;
      __syncthreads();
      // y = (z_g, (c/h) D_t^T z_g, -(1/h) D_m^T z_g) of a coefficient vector z per material and right-hand side
      auto coefs = [&](T* dst, const T* src, int rstride, int gstride) {
        for (int id = tid; id < ng * nmom; id += blockDim.x) {
          const int g = id / nmom, rest = id % nmom;
          const int r = rest / (C * nb), rem = rest % (C * nb), cc = rem / nb, kk = rem % nb;
          const T* zg = src + (size_t)r * rstride + (size_t)g * gstride;
          dst[id] = cc == 0 ? zg[kk]
                            : R::mul(R::from(cc == 1 ? s_gc[g] * ih : -ih), relT_apply<DIM, T>(a, kk, cc - 1, zg));
        }
      };
      coefs(sYx, sXf, N, nb);
      coefs(sYmp, sY + nb, C * nb, nmom);              // mu' = y_v(mu)
      __syncthreads();
      coefs(sYxp, sYx + nb, C * nb, nmom);             // x' = y_v(x)
      __syncthreads();
      // fields of x and mu and their c-derivatives at a point of material g: sqrt(w)
      // times the C components of the vectors' fields at U-values u.  Four
      // neighbouring lanes take a (point, right-hand side): each forms one field,
      // its components as independent sums, and all receive the four.  (A chunk
      // has few points: one thread for all left one warp to a sub-partition's
      // binary64 unit, half of the reverse sweep's time.)
      auto fields4 = [&](bool live, int g, int r, const T* u, double tq, double* Fx, double* dFx, double* Fm, double* dFm) {
        const int f_ = lane & 3;
        const T* const Y = (f_ == 0 ? sYx : f_ == 1 ? sYxp : f_ == 2 ? sY : sYmp) + (size_t)g * nmom + (size_t)r * C * nb;
        T t[C];
#pragma unroll
        for (int cc = 0; cc < C; ++cc) t[cc] = R::zero();
        if (live) {
          for (int j = 0; j < nl; ++j) {
            const T uj = u[j];
#pragma unroll
            for (int cc = 0; cc < C; ++cc) t[cc] = R::acc(t[cc], Y[cc * nb + j], uj);
          }
          for (int j = nl; j < nb; ++j) t[0] = R::acc(t[0], Y[j], u[j]);   // (x' and mu' are derivatives: zeros)
        }
        const double rc = s_gc[g] * s_gic2[g], sc = (f_ & 1) ? tq * rc : 1.0;   // 1 / c
#pragma unroll
        for (int cc = 0; cc < C; ++cc) {
          const double own = R::to(R::norm(t[cc])) * sc;
          Fx[cc] = __shfl_sync(0xffffffffu, own, lane & 28);
          dFx[cc] = __shfl_sync(0xffffffffu, own, (lane & 28) + 1);
          Fm[cc] = __shfl_sync(0xffffffffu, own, (lane & 28) + 2);
          dFm[cc] = __shfl_sync(0xffffffffu, own, (lane & 28) + 3);
        }
        dFx[1] = ::fma(Fx[1], rc, dFx[1]);
        dFm[1] = ::fma(Fm[1], rc, dFm[1]);
      };
      // contributions val[id], id = point * nrhs + right-hand side, added to an
      // element by one warp in a fixed order
      double* sVal = reinterpret_cast<double*>(sCB);   // 2 CH nrhs values (sCB is dead)
      auto add_range = [&](int k, int lo, int hi) {
        double t_ = 0.0;
        for (int id = lo + lane; id < hi; id += 32) t_ += sVal[id];
        for (int o = 16; o > 0; o >>= 1) t_ += __shfl_xor_sync(0xffffffffu, t_, o);
        if (lane == 0) s_gel[k] += t_;
      };
      // (a) top points (the map E and the top form) and bottom points (the
      // bottom form of b and the recovery terms), this CTA's points
      for (int side = 0; side < 2; ++side) {
        for (int base = o0; base < o1; base += CH) {
          const int nq = min(CH, o1 - base);
          for (int id = tid; id < nq; id += blockDim.x) {
            const int qg = base + id;
            map_point(sPt + id * (DIM + 2), qg / Q, qg % Q, side == 0);
          }
          eval_uvalues_block<DIM, T>(a, nq, sPt, sM, sU);
          for (int id0 = 0; id0 < nq * nrhs; id0 += NT / 4) {
            const bool live = id0 + (tid >> 2) < nq * nrhs;
            const int id = live ? id0 + (tid >> 2) : 0;
            const int ql = id / nrhs, r = id % nrhs, qg = base + ql, k = qg / Q, q = qg % Q, g = s_grp[k];
            double tt = 0.0;
            for (int i = 0; i < NV; ++i) tt = fma(__ldg(a.bary + q * NV + i), side == 0 ? s_tt[k][i] : s_tb[k][i], tt);
            double Fx[C], dFx[C], Fm[C], dFm[C];
            fields4(live, g, r, sU + (size_t)ql * us, tt - tc, Fx, dFx, Fm, dFm);
            const double ic2 = s_gic2[g], dic2 = -2.0 * ic2 * (s_gc[g] * ic2);   // c^-2 and its derivative
            const double* gk = side == 0 ? s_gt[k] : s_gb[k];
            // c^-2 a_v b_v + a_s.b_s - a_v (b_s.g) - (a_s.g) b_v: the face form of eq. (4.1)
            auto Qf = [&](const double* A_, const double* B_) {
              double s2 = ic2 * A_[1] * B_[1], ag = 0.0, bg = 0.0;
              for (int d = 0; d < DIM; ++d) {
                s2 = fma(A_[2 + d], B_[2 + d], s2);
                ag = fma(A_[2 + d], gk[d], ag);
                bg = fma(B_[2 + d], gk[d], bg);
              }
              return s2 - A_[1] * bg - ag * B_[1];
            };
            double val;
            if (side == 0) {
              const double* lam = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
              const double isw = __ldg(a.isqw + q) * s_isdet[k];
              double e = 0.0;
              for (int cc = 0; cc < C; ++cc) e = fma(__ldcg(lam + cc) * isw, dFx[cc], e);
              val = e - (Qf(dFx, Fm) + Qf(Fx, dFm) + dic2 * Fx[1] * Fm[1]);
            } else {
              const double sw = __ldg(a.sqw + q) * s_sdet[k];
              const double* f0 = saved_front(r) + (size_t)qg * C;
              double fb[C];
              for (int cc = 0; cc < C; ++cc) fb[cc] = sw * __ldcg(f0 + cc);
              val = Qf(fb, dFm) + dic2 * fb[1] * Fm[1] + fb[0] * dFm[0] - (dFx[0] * Fm[0] + Fx[0] * dFm[0]);
            }
            if (live && (lane & 3) == 0) sVal[id] = val;
          }
          __syncthreads();
          for (int k = base / Q + warp; k * Q < base + nq; k += NW)
            add_range(k, max(0, k * Q - base) * nrhs, min(nq, (k + 1) * Q - base) * nrhs);
          __syncthreads();
        }
      }
      // (b) vertical faces: Dirichlet, interface and Neumann facets (each
      // facet's points split over the cluster; split right-hand sides: every point)
      const int fsl = (Q + CS - 1) / CS;
      const int p0 = rsplit ? 0 : min(Q, rank * fsl), p1 = rsplit ? Q : min(Q, p0 + fsl);
      const int* rfi = a.vrec_i + h0.y + P * (2 + NV);
      double* sGdd = reinterpret_cast<double*>(sGd);
      for (int f = 0; f < nfac + nif + nneu; ++f) {
        const bool ifc = f >= nfac && f < nfac + nif, neu = NEU && f >= nfac + nif;
        const int gp = s_fg[f], gm = s_fg2[f];
        // patch slots of the elements on the facet's + and - sides (boundary facets: one element)
        int kp = 0, km = 0;
        {
          const int ep = __ldg(rfi + f * (NV + 3)), em = __ldg(rfi + f * (NV + 3) + 1);
          for (int k = 0; k < P; ++k) {
            if (s_el[k] == ep) kp = k;
            if (s_el[k] == em) km = k;
          }
        }
        for (int base = p0; base < p1; base += CH) {
          const int nq = min(CH, p1 - base);
          for (int id = tid; id < nq; id += blockDim.x) {
            const int q = base + id;
            double xt[DIM + 1];
            for (int d = 0; d <= DIM; ++d) xt[d] = 0.0;
            for (int i = 0; i < NV; ++i) {
              const double l = __ldg(a.bary + q * NV + i);
              for (int d = 0; d <= DIM; ++d) xt[d] = fma(l, s_fP[f][i][d], xt[d]);
            }
            const double sw = __ldg(a.sqw + q) * s_fsq[f];
            T* pp = sPt + id * (DIM + 2);
            pp[0] = R::from(s_gc[gp] * (xt[DIM] - tc) * ih);
            for (int d = 0; d < DIM; ++d) pp[1 + d] = R::from((xt[d] - s_xv[d]) * ih);
            pp[DIM + 1] = R::from(sw);
            if (ifc) {
              T* p2 = sPt + (nq + id) * (DIM + 2);
              p2[0] = R::from(s_gc[gm] * (xt[DIM] - tc) * ih);
              for (int d = 0; d < DIM; ++d) p2[1 + d] = pp[1 + d];
              p2[DIM + 1] = pp[DIM + 1];
            } else {
              // the forward boundary data of the facet (g_D or g_N)
              const long long goff = a.tent_gdoff[tent] + (NEU ? (long long)s_fw[f][0] * Q : (long long)f * Q) + q;
              for (int r = 0; r < nrhs; ++r)
                sGdd[id * nrhs + r] = gD != nullptr ? sw * gD[(long long)r * a.n_bnd + goff] : 0.0;
            }
          }
          if (ifc) __syncthreads();   // (the - side's rows are read by other threads than wrote them)
          eval_uvalues_block<DIM, T>(a, ifc ? 2 * nq : nq, sPt, sM, sU);
          for (int id0 = 0; id0 < nq * nrhs; id0 += NT / 4) {
            const bool live = id0 + (tid >> 2) < nq * nrhs, put = live && (lane & 3) == 0;
            const int id = live ? id0 + (tid >> 2) : 0;
            const int ql = id / nrhs, r = id % nrhs, q = base + ql;
            double tt = 0.0;
            for (int i = 0; i < NV; ++i) tt = fma(__ldg(a.bary + q * NV + i), s_fP[f][i][DIM], tt);
            double Fx[C], dFx[C], Fm[C], dFm[C];
            fields4(live, gp, r, sU + (size_t)ql * us, tt - tc, Fx, dFx, Fm, dFm);
            auto sn = [&](const double* F_) {
              double t_ = 0.0;
              for (int d = 0; d < DIM; ++d) t_ = fma(s_fn[f][d], F_[2 + d], t_);
              return t_;
            };
            if (ifc) {
              double Gx[C], dGx[C], Gm[C], dGm[C], Z[C];
              fields4(live, gm, r, sU + (size_t)(nq + ql) * us, tt - tc, Gx, dGx, Gm, dGm);
              for (int cc = 0; cc < C; ++cc) Z[cc] = 0.0;
              // the interface form of eq. (2.5) with trial fields X+-, test fields M+-
              auto I = [&](const double* Xp, const double* Xm, const double* Mp, const double* Mm) {
                const double jm = sn(Mp) - sn(Mm), dv = Mp[1] - Mm[1];
                return 0.5 * (jm * (Xp[1] + Xm[1]) + dv * (sn(Xp) + sn(Xm))) + a.alpha * dv * (Xp[1] - Xm[1]) +
                       a.beta * jm * (sn(Xp) - sn(Xm));
              };
              const double vp = -(I(dFx, Z, Fm, Gm) + I(Fx, Gx, dFm, Z)), vm = -(I(Z, dGx, Fm, Gm) + I(Fx, Gx, Z, dGm));
              if (put) {
                sVal[id] = vp;
                sVal[nq * nrhs + id] = vm;
              }
            } else {
              const double gv = sGdd[id];
              double val;
              if (neu) {   // A: v (tau.n) + beta (sigma.n)(tau.n); b: g_N (beta tau.n - w)
                val = gv * (a.beta * sn(dFm) - dFm[1]) -
                      (dFx[1] * sn(Fm) + Fx[1] * sn(dFm) + a.beta * (sn(dFx) * sn(Fm) + sn(Fx) * sn(dFm)));
              } else {     // A: (sigma.n + alpha v) w; b: g_D (alpha w - tau.n)
                val = gv * (a.alpha * dFm[1] - sn(dFm)) -
                      ((sn(dFx) + a.alpha * dFx[1]) * Fm[1] + (sn(Fx) + a.alpha * Fx[1]) * dFm[1]);
              }
              if (put) sVal[id] = val;
            }
          }
          __syncthreads();
          if (warp == 0) {   // (the - side's follow the + side's)
            add_range(kp, 0, nq * nrhs);
            if (ifc) add_range(km, nq * nrhs, 2 * nq * nrhs);
          }
          __syncthreads();
        }
      }
      // one addition per element and tent, the CTAs' shares summed in rank order:
      // the tents of an element follow one another (each waits for the later
      // ones of its vertex and neighbours), so the sum's order is fixed
      csync();
      for (int k = tid * CS + rank; k < P; k += NT * CS) {
        double t_ = s_gel[k];
        if (CS > 1) {
          t_ = 0.0;
          for (int r = 0; r < CS; ++r) t_ += cluster.map_shared_rank(s_gel, r)[k];
        }
        atomicAdd(a.dJdc + s_el[k], t_);
      }
      __syncthreads();
    }
  }
  // tensor-core outflow: f(q)[r, c] = sum_j U_j(q) y[r, c, j] for a chunk
  // of up to 2 CH top points, one M = 128 tile of points: A = the digit
  // planes of the points' U-values (rows = points, K = basis functions
  // padded to 32, scaled per point), B = those of y (rows (r, c) padded to
  // 16, scaled per row; formed once per tent); each level sum takes
  // (tc_cols / kSlices) rounded down to 32, i.e. 96 columns (>= NY)
  const int M_tc = nrhs * C, NY = (M_tc + 15) & ~15, planeY = 32 * NY;
  const int planeU = 32 * ((2 * CH + 15) & ~15);
  if constexpr (kTC) {
    if (tc_on) {
      uint16_t* sTB = reinterpret_cast<uint16_t*>(sm + a.off_tc) + tc::kSlices * planeU + 512;
      for (int m = tid; m < NY; m += blockDim.x) {
        float mx = 0.f;
        if (m < M_tc)
          for (int j = 0; j < nb; ++j) mx = fmaxf(mx, fabsf(sY[(size_t)m * nb + j].hi));
        s_tce[0][m] = tc::scale_exp(mx);
      }
      __syncthreads();
      for (int id = tid; id < NY * 4; id += blockDim.x) {
        const int kc = id / NY, m = id % NY;
        float d[8][tc::kSlices];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int jj = kc * 8 + j;
          const T x = (m < M_tc && jj < nb) ? sY[(size_t)m * nb + jj] : R::zero();
          tc::digits(x.hi, x.lo, s_tce[0][m], d[j]);
        }
        tc::store_row8(sTB + ((size_t)(kc * (NY >> 3) + (m >> 3)) * 64 + (m & 7) * 8), planeY, d);
      }
      // (the first chunk's barriers order these writes before the products)
    }
  }
  auto tc_outflow = [&](int base, int nq) {
    if constexpr (kTC) {
      const int NP = (nq + 15) & ~15, RGU = NP >> 3;
      uint16_t* sTA = reinterpret_cast<uint16_t*>(sm + a.off_tc);
      uint16_t* sTB = sTA + tc::kSlices * planeU + 512;
      int* eY = s_tce[0];
      int* eU = s_tce[1];
      for (int ql = tid; ql < NP; ql += blockDim.x) {
        float mx = 0.f;
        if (ql < nq)
          for (int j = 0; j < nb; ++j) mx = fmaxf(mx, fabsf(sU[(size_t)ql * us + j].hi));
        eU[ql] = tc::scale_exp(mx);
      }
      __syncthreads();
      for (int id = tid; id < NP * 4; id += blockDim.x) {
        const int kc = id / NP, n = id % NP;
        float d[8][tc::kSlices];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int jj = kc * 8 + j;
          const T x = (n < nq && jj < nb) ? sU[(size_t)n * us + jj] : R::zero();
          tc::digits(x.hi, x.lo, eU[n], d[j]);
        }
        tc::store_row8(sTA + ((size_t)(kc * RGU + (n >> 3)) * 64 + (n & 7) * 8), planeU, d);
      }
      const int cstride = (a.tc_cols / tc::kSlices) & ~31;   // columns per level sum (>= NY)
      const bool ok = tc_product(tc::smem_addr(sTA), (uint32_t)planeU * 2, (uint32_t)RGU * 128,
                                 tc::smem_addr(sTB), (uint32_t)planeY * 2, (uint32_t)(NY >> 3) * 128, 2, NY, cstride);
      // levels -> binary64 front values: the thread of lane l of warp w holds
      // point 32 (w % 4) + l and every (NW / 4)th group of 8 rows (r, c)
      const int q4 = warp & 3;
      if (ok && 32 * q4 < nq) {
        const int ql = 32 * q4 + lane;
        const bool live = ql < nq;
        double* fq = front;
        int ep = 0;
        if (live) {
          const int qg = base + ql, k = qg / Q, q = qg % Q;
          fq = front + ((int64_t)s_el[k] * Q + q) * C;
          ep = eU[ql] - 16;
        }
        const int64_t rstride = (int64_t)a.ne * Q * C;
        for (int c0 = 8 * (warp >> 2); c0 < NY; c0 += 2 * NW) {
          float lv[tc::kSlices][8];
#pragma unroll
          for (int l = 0; l < tc::kSlices; ++l)
            tc::ld8(s_tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(l * cstride + c0), lv[l]);
          tc::wait_ld();
          if (live) {
            int r = c0 / C, cc = c0 - r * C;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (c0 + j < M_tc) {
                float acc[tc::kSlices];
#pragma unroll
                for (int l = 0; l < tc::kSlices; ++l) acc[l] = lv[l][j];
                float sh, se;
                tc::combine_ff(acc, sh, se);
                fq[r * rstride + cc] = tc::ff_to_double(sh, se, ep + eY[c0 + j]);
              }
              if (++cc == C) {
                cc = 0;
                ++r;
              }
            }
          }
        }
      }
      tc::fence_before();
      __syncthreads();
    }
  };
  // the outflow's point formula of the adjoint: fields sv of mu at point q of
  // element k to lambda_bot = w (s0, c^-2 s_t - g_b.s, s_m - g_b,m s_t)
  auto store_adjoint = [&](int r, int k, int q, const double* sv) {
    const double cg = s_gc[s_grp[k]];
    const double sq = __ldg(a.sqw + q) * s_sdet[k];
    const double w = sq * sq;
    double gs = 0.0;
    for (int d = 0; d < DIM; ++d) gs = fma(s_gb[k][d], sv[2 + d], gs);
    double* f = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
    f[0] = w * sv[0];
    f[1] = w * (sv[1] / (cg * cg) - gs);
    for (int d = 0; d < DIM; ++d) f[2 + d] = w * (sv[2 + d] - s_gb[k][d] * sv[1]);
  };
  if (srule) {
    // the fields at the rule's points, then through the table to the front's
    const int S = a.S;
    const T* U = sKeep;
    for (int eb = e0; eb < e1; eb += EC) {
      const int ne = min(EC, e1 - eb);
      if (eb > e0) __syncthreads();
      if (!kept) {
        for (int id = tid; id < ne * S; id += blockDim.x)
          map_rule(sPt + id * (DIM + 2), eb + id / S, id % S, !ADJ);
        eval_uvalues_block<DIM, T>(a, ne * S, sPt, sM, sU);
      }
      const T* Ue = kept ? U + (size_t)(eb - e0) * S * us : sU;
      for (int id = tid; id < nrhs * C * ne * S; id += blockDim.x) {
        const int rc = id / (ne * S), pt = id - rc * (ne * S), k = eb + pt / S;
        const T *u = Ue + (size_t)pt * us, *y = sY + (size_t)s_grp[k] * nmom + (size_t)rc * nb;
        T t0 = R::zero(), t1 = R::zero();
        const int nj = rc % C == 0 ? nb : nl;
        int j = 0;
        for (; j + 1 < nj; j += 2) {
          t0 = R::acc(t0, y[j], u[j]);
          t1 = R::acc(t1, y[j + 1], u[j + 1]);
        }
        if (j < nj) t0 = R::acc(t0, y[j], u[j]);
        sCB[(size_t)rc * cbs + pt] = R::add(R::norm(t0), R::norm(t1));
      }
      __syncthreads();
      auto at_front = [&](int rc, int k, int q) {   // component at front point q of element eb + k
        const T *F = sCB + (size_t)rc * cbs + k * S, *w = sTF + q;
        T t0 = R::zero(), t1 = R::zero();
        int s_ = 0;
        for (; s_ + 1 < S; s_ += 2) {
          t0 = R::acc(t0, w[s_ * a.tf_stride], F[s_]);
          t1 = R::acc(t1, w[(s_ + 1) * a.tf_stride], F[s_ + 1]);
        }
        if (s_ < S) t0 = R::acc(t0, w[s_ * a.tf_stride], F[s_]);
        return R::to(R::add(R::norm(t0), R::norm(t1))) * s_isdet[eb + k];
      };
      if constexpr (!ADJ) {
        for (int id = tid; id < nrhs * ne * Q * C; id += blockDim.x) {
          const int cc = id % C, rq = id / C, r = rq / (ne * Q), ql = rq - r * (ne * Q), k = ql / Q, q = ql - k * Q;
          front[(((int64_t)r * a.ne + s_el[eb + k]) * Q + q) * C + cc] = at_front(r * C + cc, k, q);
        }
      } else {
        for (int id = tid; id < nrhs * ne * Q; id += blockDim.x) {
          const int r = id / (ne * Q), ql = id - r * (ne * Q), k = ql / Q, q = ql - k * Q;
          double sv[C];
#pragma unroll
          for (int cc = 0; cc < C; ++cc) sv[cc] = at_front(r * C + cc, k, q);
          store_adjoint(r, eb + k, q, sv);
        }
      }
    }
    __syncthreads();
  } else
  for (int base = o0; base < o1; base += kept ? NP : 2 * CH) {   // (kept U-values: one pass)
    const int nq = min(kept ? NP : 2 * CH, o1 - base);
    if (!kept) {
    for (int id = tid; id < nq; id += blockDim.x) {
      const int qg = base + id;
      map_with(sPt + id * (DIM + 2), qg / Q, qg % Q, !ADJ, a.baryT, a.sqwT, true);
    }
    eval_uvalues_block<DIM, T, false>(a, nq, sPt, sM, sU);
    }
    if constexpr (!ADJ) {
      // few right-hand sides: one (point, right-hand side, component) per
      // thread, so that every warp (and every sub-partition's binary64 unit)
      // has work
      if (tc_on) {
        tc_outflow(base, nq);
      } else if (nq * nrhs < (int)blockDim.x) {
        for (int id = tid; id < nq * nrhs * C; id += blockDim.x) {
          const int cc = id % C, rq = id / C, r = rq / nq, ql = rq % nq;
          const int qg = base + ql, k = qg / Q, q = qg % Q;
          const T* u = kept ? sKeep + (size_t)(base - q0 + ql) * us : sU + (size_t)ql * us;
          const T* y = sY + (size_t)s_grp[k] * nmom + ((size_t)r * C + cc) * nb;
          T t = R::zero();
          for (int j = 0; j < (cc == 0 ? nb : nl); ++j) t = R::acc(t, y[j], u[j]);
          const double val = R::to(R::norm(t));
          front[(((int64_t)r * a.ne + s_el[k]) * Q + q) * C + cc] = kept ? val * (__ldg(a.isqw + q) * s_isdet[k]) : val;
        }
      } else
      // one (point, right-hand side) per thread, its C components as
      // independent sums (consecutive threads: consecutive points)
      for (int id = tid; id < nq * nrhs; id += blockDim.x) {
        const int r = id / nq, ql = id % nq;
        const int qg = base + ql, k = qg / Q, q = qg % Q;
        const T* u = kept ? sKeep + (size_t)(base - q0 + ql) * us : sU + (size_t)ql * us;
        const T* y = sY + (size_t)s_grp[k] * nmom + (size_t)r * C * nb;
        T t[C];
#pragma unroll
        for (int cc = 0; cc < C; ++cc) t[cc] = R::zero();
        for (int j = 0; j < nl; ++j) {
          const T uj = u[j];
#pragma unroll
          for (int cc = 0; cc < C; ++cc) t[cc] = R::acc(t[cc], y[cc * nb + j], uj);
        }
#pragma unroll 4
        for (int j = nl; j < nb; ++j) t[0] = R::acc(t[0], y[j], u[j]);   // (v and sigma: zero coefficients)
        double* f = front + (((int64_t)r * a.ne + s_el[k]) * Q + q) * C;
        if (kept) {
          const double sc = __ldg(a.isqw + q) * s_isdet[k];
#pragma unroll
          for (int cc = 0; cc < C; ++cc) f[cc] = R::to(R::norm(t[cc])) * sc;
        } else {
#pragma unroll
          for (int cc = 0; cc < C; ++cc) f[cc] = R::to(R::norm(t[cc]));
        }
      }
    } else {
      for (int id = tid; id < nq * nrhs; id += blockDim.x) {
        const int ql = id / nrhs, r = id % nrhs;
        const int qg = base + ql, k = qg / Q, q = qg % Q;
        const T* u = kept ? sKeep + (size_t)(base - q0 + ql) * us : sU + (size_t)ql * us;
        double sv[C];
        for (int cc = 0; cc < C; ++cc) {
          const T* y = sY + (size_t)s_grp[k] * nmom + ((size_t)r * C + cc) * nb;
          T t = R::zero();
          for (int j = 0; j < (cc == 0 ? nb : nl); ++j) t = R::acc(t, y[j], u[j]);
          t = R::norm(t);
          sv[cc] = kept ? R::to(t) * (__ldg(a.isqw + q) * s_isdet[k]) : R::to(t);
        }
        store_adjoint(r, k, q, sv);
      }
    }
    __syncthreads();
  }
  if (tid == 0 && rank == 0) a.tau[v] = ADJ ? s_tbot : s_ttop;
  if constexpr (PERSIST) {
    // this CTA's front (and rank 0's time) writes, then its completion count;
    // no CTA reads another's shared memory after the solution copy, and the
    // next tent's first cluster barrier keeps rank 0's b until all have copied it
    __threadfence();
    __syncthreads();
    if (tid == 0) red_release_add(a.done + v, 1);
  } else {
    csync();   // rank 0's b stays valid until every CTA has read the solution
    break;
  }
  }   // tent loop
  if constexpr (kTC) {
    tc::fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_free(s_tmem, a.tc_cols);
  }
}


// launchers, one translation unit per space dimension D, kind of sweep K (0
// forward binary64, 1 forward mixed, 2 adjoint binary64, 3 forward mixed on the
// tensor cores) and N = 1 for meshes with Neumann facets; persistent: one
// resident grid of clusters pulling tents from a queue; wide: kThreadsWide
// threads per CTA
#define TP_DECLARE_LAUNCHERS(D, K, N)                                                                      \
  cudaError_t layer_attrs_d##D##K##_n##N(size_t smem);                                                      \
  cudaError_t layer_static_smem_d##D##K##_n##N(size_t* bytes);                                              \
  cudaError_t launch_layer_d##D##K##_n##N(const KArgs& a, int n_cluster, int cs, int t0, size_t smem,       \
                                          cudaStream_t st, bool persistent, bool wide);                     \
  cudaError_t max_clusters_d##D##K##_n##N(int cs, size_t smem, bool split, bool wide, int* n);
#define TP_DECLARE_KIND(D, K) TP_DECLARE_LAUNCHERS(D, K, 0) TP_DECLARE_LAUNCHERS(D, K, 1)
#define TP_DECLARE_DIM(D) TP_DECLARE_KIND(D, 0) TP_DECLARE_KIND(D, 1) TP_DECLARE_KIND(D, 2) TP_DECLARE_KIND(D, 3)
TP_DECLARE_DIM(1)
TP_DECLARE_DIM(2)
TP_DECLARE_DIM(3)
#undef TP_DECLARE_DIM
#undef TP_DECLARE_KIND
#undef TP_DECLARE_LAUNCHERS

}  // namespace tp

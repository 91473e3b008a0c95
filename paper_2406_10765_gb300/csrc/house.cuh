// Device helpers of the blocked Householder reduction shared by its kernels
// (house_cols.cu and house_chain.cu: the chained column kernels; hemv_tc.cu: their tensor-core
// Hermitian product and the cooperative tensor-core panel; dense.cu: the
// cooperative FP64 panel; house_cluster.cu: the last columns): warp and block
// sums, complex multiply-adds written as four FMAs, the reflector scalars, a
// column's pending entries, programmatic dependent launch.
#pragma once
#include "pw_internal.cuh"

// ---- a column of the chained kernels -----------------------------------
// Column c = j0 + i of the panel [V | W | V] (ld n) at j0, as its first kernel
// finds it: a0 holds the column with the panel's updates but for the part of
// the previous reflector that depends on q = v^H A v of all rows, so that
// x = a0 - k2 v, k2 = -|tau|^2 q, and W[:, i-1] = p + (k2 / 2) v.  All vectors
// are indexed by the matrix row.
constexpr int HH_CHUNKS = 8;         // row chunks of the panel's correction dots
struct HhCol {
  double2 *A;
  int n, c, i, b;
  double2 *P;
  const double2 *a0, *p;             // (i = 0: a0 is the column of A, nothing pending)
  const double *dot;                 // partials of q, one per block of the previous row kernel
  int nprev;
  const double2 *tau;
  double *d;
  double2 *x;                        // out: the finished column
  double *nrm;                       // out: partials of ||x[1:]||^2
  double2 *ucorr;                    // out: [2i][HH_CHUNKS], W[:, q]^H x (even), V[:, q]^H x (odd)
};

struct pw_dense_ws;
// the tensor-core product of column h (panel at j0): partials into ws->part
// (*nslots slots per row, part[s * nmax + row]), h's outputs, *nnrm norm partials
pw_status pw_hs_hemv(pw_dense_ws *ws, const HhCol &h, int j0, int *nslots, int *nnrm, cudaStream_t st);

namespace {

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// block-wide sum of one double (blockDim.x multiple of 32, <= 1024)
__device__ double block_sum(double v, double *sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    r = warp_sum(r);
    if (threadIdx.x == 0) sh[0] = r;
  }
  __syncthreads();
  r = sh[0];
  __syncthreads();
  return r;
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// s += a b and s += conj(a) b, four FMAs each
__device__ __forceinline__ void cmac(double2 &s, double2 a, double2 b) {
  s.x = fma(a.x, b.x, s.x);
  s.x = fma(-a.y, b.y, s.x);
  s.y = fma(a.x, b.y, s.y);
  s.y = fma(a.y, b.x, s.y);
}
__device__ __forceinline__ void cmacc(double2 &s, double2 a, double2 b) {
  s.x = fma(a.x, b.x, s.x);
  s.x = fma(a.y, b.y, s.x);
  s.y = fma(a.x, b.y, s.y);
  s.y = fma(-a.y, b.x, s.y);
}

// alpha = -1/2 tau (p^H v) from the per-block partial dots (block-wide sum)
// (stride: the partial sums run over `stride` threads, blockDim.x by default)
__device__ double2 panel_alpha(const double2 *dotpart, int ndot, double2 t, double *sh, int stride = 0) {
  double sr = 0.0, si = 0.0;
  const int st = stride > 0 ? stride : (int)blockDim.x;
  for (int q = threadIdx.x; q < ndot && (int)threadIdx.x < st; q += st) {
    const double2 v = __ldcg(&dotpart[q]);
    sr += v.x;
    si += v.y;
  }
  sr = block_sum(sr, sh);
  si = block_sum(si, sh);
  return cmul(make_double2(-0.5 * t.x, -0.5 * t.y), make_double2(sr, si));
}

// v_c entry x (x = row - (c+1)) from the stored column and the scale
__device__ __forceinline__ double2 refl_entry(const double2 *xcol, int x, double2 scal) {
  return x == 0 ? make_double2(1.0, 0.0) : cmul(xcol[x], scal);
}

// Reflector of x = (alpha, x_2..) with ||x_2..||^2 = xn2: beta, tau and the
// scale s of v = x s below its unit head (tau = 0 and s = 0 when x is
// already a multiple of the first unit vector with a real head)
__device__ __forceinline__ void reflector_scalars(double xn2, double2 alpha, double &beta, double2 &tk,
                                                  double2 &scal) {
  if (xn2 == 0.0 && alpha.y == 0.0) {
    beta = alpha.x;
    tk = make_double2(0.0, 0.0);
    scal = make_double2(0.0, 0.0);
  } else {
    beta = -copysign(sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2), alpha.x);
    tk = make_double2((beta - alpha.x) / beta, -alpha.y / beta);
    const double2 den = make_double2(alpha.x - beta, alpha.y);
    const double qq = 1.0 / (den.x * den.x + den.y * den.y);
    scal = make_double2(den.x * qq, -den.y * qq);
  }
}

// sum of a complex value over the warp, the lanes split between its parts
// after the first exchange: five additions instead of ten
__device__ __forceinline__ double2 warp_sum_c(double2 s) {
  const bool hi = threadIdx.x & 16;
  double v = (hi ? s.y : s.x) + __shfl_xor_sync(0xffffffffu, hi ? s.x : s.y, 16);
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return make_double2(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 16));
}

// reflector_scalars without CUDA's square root and divisions, a third of the time.
// 1/sqrt(s) from the hardware's approximation r: with h = 1 - s r^2, r (1 - h)^(-1/2)
// = r (1 + h/2 + 3 h^2 / 8 + ..), and sqrt(s) by one step of Heron's iteration from
// s r; 1/dd by Householder's iteration of order two (rcp_newton in dense.cu).
// Against exact arithmetic beta is within 4, tau 8 and s 16 units of 2^-53 of
// each component (the bounds of the operations' roundings; the rounded form's are
// the same).  Outside the range where the squares are normal numbers the rounded
// operations.
__device__ __forceinline__ void reflector_scalars_fast(double xn2, double2 alpha, double &beta, double2 &tk,
                                                       double2 &scal) {
  const double s2 = fma(alpha.x, alpha.x, fma(alpha.y, alpha.y, xn2));
  if ((xn2 == 0.0 && alpha.y == 0.0) || !(s2 > 1e-280 && s2 < 1e280)) {
    reflector_scalars(xn2, alpha, beta, tk, scal);
    return;
  }
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s2));
  const double h = fma(-s2 * r, r, 1.0);               // r = (1 - h / 2 + ..) / sqrt(s2)
  r = fma(r * h, fma(h, 0.375, 0.5), r);
  const double b = s2 * r;
  const double nrm = fma(fma(-b, b, s2), 0.5 * r, b);
  const double sg = alpha.x < 0.0 || (alpha.x == 0.0 && signbit(alpha.x)) ? 1.0 : -1.0;
  beta = sg * nrm;
  const double ib = sg * r;
  const double dx = alpha.x - beta;                    // no cancellation: opposite signs
  tk = make_double2(-dx * ib, -alpha.y * ib);
  const double dd = fma(dx, dx, alpha.y * alpha.y);
  double q;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(dd));
  const double e = fma(-dd, q, 1.0);
  q = fma(q, fma(e, e, e), q);
  scal = make_double2(dx * q, -alpha.y * q);
}

// the previous column's k2 (whole warp)
__device__ __forceinline__ double hh_k2(const HhCol &h) {
  if (h.i == 0) return 0.0;
  double q = 0.0;
  for (int t = threadIdx.x & 31; t < h.nprev; t += 32) q += __ldcg(&h.dot[t]);
  q = warp_sum(q);
  const double2 t = __ldcg(&h.tau[h.c - 1]);
  return -fma(t.x, t.x, t.y * t.y) * q;
}
__device__ __forceinline__ double2 hh_x(const HhCol &h, int r, double k2) {
  double2 a = __ldcg(&h.a0[r]);
  if (h.i > 0) {
    const double2 v = __ldcg(&h.P[r + (long)(h.i - 1) * h.n]);
    a.x = fma(-k2, v.x, a.x);
    a.y = fma(-k2, v.y, a.y);
  }
  return a;
}
__device__ __forceinline__ double2 hh_w(const HhCol &h, int r, double k2) {   // W[r, i-1]
  const double2 p = __ldcg(&h.p[r]), v = __ldcg(&h.P[r + (long)(h.i - 1) * h.n]);
  return make_double2(fma(0.5 * k2, v.x, p.x), fma(0.5 * k2, v.y, p.y));
}
// one warp: chunk k of the dot q2 = 2q (W[:, q]) or 2q + 1 (V[:, q]) with x
__device__ __forceinline__ void hh_dot(const HhCol &h, double k2, int q2, int k) {
  const int o = h.c + 1, m = h.n - o, per = (m + HH_CHUNKS - 1) / HH_CHUNKS;
  const int r0 = o + k * per, r1 = min(h.n, r0 + per), q = q2 >> 1;
  const bool isw = !(q2 & 1), pending = isw && q == h.i - 1;
  const double2 *col = h.P + (long)(isw ? h.b + q : q) * h.n;
  double2 s = make_double2(0.0, 0.0);
  for (int r = r0 + (threadIdx.x & 31); r < r1; r += 32)
    cmacc(s, pending ? hh_w(h, r, k2) : __ldcg(&col[r]), hh_x(h, r, k2));
  s = warp_sum_c(s);
  if ((threadIdx.x & 31) == 0) h.ucorr[q2 * HH_CHUNKS + k] = s;
}
// one row of the column: x, W[:, i-1], the diagonal; returns its part of the norm
__device__ __forceinline__ double hh_row(const HhCol &h, double k2, int r) {
  const double2 x = hh_x(h, r, k2);
  if (h.i > 0) h.P[r + (long)(h.b + h.i - 1) * h.n] = hh_w(h, r, k2);
  if (r == h.c) h.d[r] = x.x;
  else h.x[r] = x;
  return r > h.c + 1 ? fma(x.x, x.x, x.y * x.y) : 0.0;
}

}  // namespace

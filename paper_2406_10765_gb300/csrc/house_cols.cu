// Columns of a Householder panel (the tridiagonalisation inside Syevd, Sec.
// III-D) as chained kernels, two per column:
//
//   product  (k_col_hemv on the FP64 pipe, or k_hemv_tc in hemv_tc.cu on the
//            tensor cores): finishes the column x = a0 - k2 v and W[:, i-1] =
//            p + (k2 / 2) v of the previous one, forms A22 x, the corrections'
//            dots W^H x and V^H x, and the norm of x
//   rows     (k_col_rows): the reflector's scalars, v, p = tau A v, the next
//            column a0 = its update by everything but k2 v, partials of q =
//            v^H A v
//
// Nothing in the product waits for the norm: A22 is applied to x, not to v =
// s (x - beta e_1), and A v = s (A x - beta A e_1).  A e_1 with the panel's
// corrections is the next column's update, which the rows kernel forms anyway
// (ye below).  The next column in turn depends on this column's q only through
// one multiple of v, so it is stored without it and the product kernel adds it.
// With the norm and q in separate launches (update, product, rows) a column
// took three dependent launches and ~25 us besides its product; a launch is
// 1.5 us, a warp-wide FP64 instruction 65 clocks (300 of them 10 us), so the
// rest of the time was chains of FP64 instructions, which the row kernel
// spreads: RB rows per CTA, the panel's columns over the other threads, the
// scalars in a warp of their own meanwhile.
// Measured: order-1,458 eigensolve 49.1 -> 40.6 ms, order 3,456 183 -> 161 ms
// (145 ms with the row kernel resident beside k_hemv_tc, 129 with wide digits there);
// a column of trailing order 500 takes 15 us: launches 2, k2 3-4, product 5,
// scalars 2.5, sums 1, the rows' tail 1.5.
#include <algorithm>

#include "dense.cuh"
#include "house.cuh"

namespace {

constexpr int TT = 32;                  // product tile
constexpr int TPB = 32;                 // panel width

// y = A22 x as lower-tile partials (A22 = rows and columns >= c + 1, as at the
// panel's start): blocks below ntiles one tile each; then 2i blocks, one dot
// each (a row chunk per warp); then blocks of 256 rows of the finished column
__global__ void __launch_bounds__(256) k_col_hemv(const __grid_constant__ HhCol h, int ntiles, double2 *part, int nmax) {
  __shared__ double2 tile[TT][TT + 1];
  __shared__ double2 xrow[TT], xcol[TT], rpart[4][TT + 1], cpart[4][TT + 1];
  __shared__ double s_k2;
  const int n = h.n, o = h.c + 1, m = n - o;
  const int blk = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int I = 0, J = 0, x0 = 0, y0 = 0;
  if (blk < ntiles) {
    // tile (I, J) of the lower triangle; FP32 estimate (FP64 is scarce), fixed up exactly
    I = (int)((sqrtf(8.0f * blk + 1.0f) - 1.0f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= blk) ++I;
    while (I * (I + 1) / 2 > blk) --I;
    J = blk - I * (I + 1) / 2;
    x0 = TT * I;
    y0 = TT * J;   // tile rows x0.., columns y0.. (offsets from o)
    // the trailing matrix is fixed inside the panel, whose first column is
    // launched without overlap: loaded before the wait
    const int yc = y0 + lane;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rl = warp * 4 + q, xr = x0 + rl;
      double2 a = make_double2(0.0, 0.0);
      if (xr < m && yc < m && (I != J || yc <= xr)) a = h.A[(o + xr) + (long)(o + yc) * n];
      tile[rl][lane] = a;
    }
  }
  pdl_wait();
  pdl_trigger();
  if (warp == 0) {
    const double k = hh_k2(h);
    if (lane == 0) s_k2 = k;
  }
  __syncthreads();
  const double k2 = s_k2;
  if (blk >= ntiles + 2 * h.i) {
    const int rb = blk - ntiles - 2 * h.i, r = h.c + rb * 256 + threadIdx.x;
    const double s = warp_sum(r < n ? hh_row(h, k2, r) : 0.0);
    if (lane == 0) h.nrm[rb * 8 + warp] = s;
    return;
  }
  if (blk >= ntiles) {
    hh_dot(h, k2, blk - ntiles, warp);
    return;
  }
  if (threadIdx.x < 2 * TT) {
    const int l = threadIdx.x & 31, x = (threadIdx.x < TT ? x0 : y0) + l;
    (threadIdx.x < TT ? xrow : xcol)[l] = x < m ? hh_x(h, o + x, k2) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  // warps 0-3: quarter row sums A x; warps 4-7: quarter column sums A^H x
  // (strictly below the diagonal in a diagonal tile)
  {
    const int k = warp & 3, l = lane;
    double2 s = make_double2(0.0, 0.0);
    if (warp < 4) {
#pragma unroll
      for (int cl = 8 * k; cl < 8 * k + 8; ++cl) cmac(s, tile[l][cl], xcol[cl]);
      rpart[k][l] = s;
    } else {
#pragma unroll
      for (int rr = 8 * k; rr < 8 * k + 8; ++rr)
        if (I != J || rr > l) cmacc(s, tile[rr][l], xrow[rr]);
      cpart[k][l] = s;
    }
  }
  __syncthreads();
  // rows by warp 0, columns by warp 1; a diagonal tile's rows take both
  if (warp < 2 && (warp == 0 || I != J)) {
    const double2(*pt)[TT + 1] = warp == 0 ? rpart : cpart;
    double2 s = cadd(cadd(pt[0][lane], pt[1][lane]), cadd(pt[2][lane], pt[3][lane]));
    if (I == J)
      s = cadd(s, cadd(cadd(cpart[0][lane], cpart[1][lane]), cadd(cpart[2][lane], cpart[3][lane])));
    const int x = (warp == 0 ? x0 : y0) + lane;
    if (x < m) part[(long)(warp == 0 ? J : I) * nmax + x] = s;
  }
}
static_assert(HH_CHUNKS == 8, "a row chunk per warp");

struct RowsArgs {
  HhCol h;
  const double2 *part;         // [slot][nmax], from row c + 1
  int nslots, nmax, nnrm;
  bool next;                   // the panel has a next column
  double2 *p, *acol;           // p and the next column's a0, by matrix row
  double *dot;                 // partials of q per block
  double2 *tau;
  double *e;
};

// RB rows per CTA (256 / RB threads each): local row 0 is row c + 1, whose p
// every CTA needs and forms, the others are its own.
//   yx = sum of the partials - sum_q V_q (W_q^H x) + W_q (V_q^H x)
//   ye = A e_1 - sum_q V_q conj(W_q[c+1]) + W_q conj(V_q[c+1])
//   p = tau s (yx - beta ye), a0 = ye - v conj(p_{c+1}) - p
// RB by order: the rows that give every SM at most one CTA, so that the FP64
// work (16 instructions per row and panel column) spreads over all of them.
template <int RB>
__global__ void __launch_bounds__(256) k_col_rows(const __grid_constant__ RowsArgs g) {
  constexpr int NS = 256 / RB;            // threads per row
  constexpr int QM = (TPB + NS - 1) / NS; // panel columns per thread
  constexpr int NV = 4 * RB / 32;         // values per lane after the exchange within a warp
  __shared__ double2 s_ux[2 * TPB], s_vo[TPB], s_wo[TPB];
  __shared__ double s_red[8][NV][32], s_fin[4][RB], s_beta;
  __shared__ double2 s_tk, s_scal;
  const HhCol &h = g.h;
  const int n = h.n, c = h.c, i = h.i, b = h.b, o = c + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rl = tid % RB, sl = tid / RB;
  const int r = rl == 0 ? o : o + (int)blockIdx.x * (RB - 1) + rl;
  const bool in = r < n;
  const double2 *V = h.P, *W = h.P + (long)b * n;
  // before the wait: what was written two or more launches back
  double2 vq[QM], wq[QM];
  double2 ye = make_double2(0.0, 0.0), yx = ye;
#pragma unroll
  for (int t = 0; t < QM; ++t) {
    const int q = sl + NS * t;
    const bool ok = in && q < i;
    vq[t] = ok ? V[r + (long)q * n] : make_double2(0.0, 0.0);
    wq[t] = ok && q < i - 1 ? W[r + (long)q * n] : make_double2(0.0, 0.0);
  }
  if (sl == 0 && in) ye = h.A[r + (long)o * n];
  if (tid < i) {
    s_vo[tid] = V[o + (long)tid * n];
    if (tid < i - 1) s_wo[tid] = W[o + (long)tid * n];
  }
  pdl_wait();
  pdl_trigger();
  // the last panel column, written by the product kernel
#pragma unroll
  for (int t = 0; t < QM; ++t)
    if (sl + NS * t == i - 1 && in) wq[t] = __ldcg(&W[r + (long)(i - 1) * n]);
  if (tid == i - 1) s_wo[tid] = __ldcg(&W[o + (long)tid * n]);
  double2 xr = make_double2(0.0, 0.0);
  if (warp == 0 && lane < RB && in) xr = __ldcg(&h.x[r]);
  if (warp == 7) {             // the reflector's scalars
    double s = 0.0;
    for (int t = lane; t < g.nnrm; t += 32) s += __ldcg(&h.nrm[t]);
    s = warp_sum(s);
    double beta;
    double2 tk, scal;
    reflector_scalars_fast(s, __ldcg(&h.x[o]), beta, tk, scal);
    if (lane == 0) {
      s_beta = beta;
      s_tk = tk;
      s_scal = scal;
      if (blockIdx.x == 0) {
        g.tau[c] = tk;
        g.e[c] = beta;
      }
    }
  } else {
    // a dot's chunks: two per thread, four threads together
    for (int t = tid; t < (8 * i + 31) / 32 * 32; t += 224) {
      const int q2 = t >> 2, k = 2 * (t & 3);
      double2 u = make_double2(0.0, 0.0);
      if (q2 < 2 * i) u = cadd(__ldcg(&h.ucorr[q2 * HH_CHUNKS + k]), __ldcg(&h.ucorr[q2 * HH_CHUNKS + k + 1]));
#pragma unroll
      for (int w = 1; w < 4; w <<= 1) {
        u.x += __shfl_xor_sync(0xffffffffu, u.x, w);
        u.y += __shfl_xor_sync(0xffffffffu, u.y, w);
      }
      if ((t & 3) == 0 && q2 < 2 * i) s_ux[q2] = u;
    }
  }
  if (in)
    for (int s = sl; s < g.nslots; s += NS) yx = cadd(yx, __ldcg(&g.part[(long)s * g.nmax + (r - o)]));
  __syncthreads();
#pragma unroll
  for (int t = 0; t < QM; ++t) {
    const int q = sl + NS * t;
    if (q >= i) break;
    const double2 uw = s_ux[2 * q], uv = s_ux[2 * q + 1], vo = s_vo[q], wo = s_wo[q];
    cmac(yx, vq[t], make_double2(-uw.x, -uw.y));
    cmac(yx, wq[t], make_double2(-uv.x, -uv.y));
    cmac(ye, vq[t], make_double2(-wo.x, wo.y));
    cmac(ye, wq[t], make_double2(-vo.x, vo.y));
  }
  // sums over the row's threads: within the warp the lanes are split between
  // the four values while they are added, then across the warps
  if (RB == 32) {
    s_red[warp][0][lane] = yx.x;
    s_red[warp][NV > 1 ? 1 : 0][lane] = yx.y;
    s_red[warp][NV > 2 ? 2 : 0][lane] = ye.x;
    s_red[warp][NV > 3 ? 3 : 0][lane] = ye.y;
  } else {
    const bool h16 = lane & 16;
    double re = (h16 ? ye.x : yx.x) + __shfl_xor_sync(0xffffffffu, h16 ? yx.x : ye.x, 16);
    double im = (h16 ? ye.y : yx.y) + __shfl_xor_sync(0xffffffffu, h16 ? yx.y : ye.y, 16);
    if (RB == 16) {
      s_red[warp][0][lane] = re;
      s_red[warp][NV > 1 ? 1 : 0][lane] = im;
    } else {
      const bool h8 = lane & 8;
      s_red[warp][0][lane] = (h8 ? im : re) + __shfl_xor_sync(0xffffffffu, h8 ? re : im, 8);
    }
  }
  __syncthreads();
  if (warp < NV) {
    double s = s_red[0][warp][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += s_red[w][warp][lane];
    // which of yx.x, yx.y, ye.x, ye.y, and the row
    const int kind = RB == 32 ? warp : RB == 16 ? 2 * (lane >> 4) + warp : lane >> 3;
    s_fin[kind][lane % RB] = s;
  }
  __syncthreads();
  if (warp != 0) return;
  double q = 0.0;
  double2 p = make_double2(0.0, 0.0), v = p, fe = p;
  if (lane < RB && in) {
    const double beta = s_beta;
    const double2 scal = s_scal;
    fe = make_double2(s_fin[2][lane], s_fin[3][lane]);
    const double2 y = cmul(scal, make_double2(fma(-beta, fe.x, s_fin[0][lane]), fma(-beta, fe.y, s_fin[1][lane])));
    p = cmul(s_tk, y);
    v = lane == 0 ? make_double2(1.0, 0.0) : cmul(xr, scal);
    if (lane > 0 || blockIdx.x == 0) q = fma(y.x, v.x, y.y * v.y);
  }
  const double2 po = make_double2(__shfl_sync(0xffffffffu, p.x, 0), __shfl_sync(0xffffffffu, p.y, 0));
  if (lane < RB && in && (lane > 0 || blockIdx.x == 0)) {
    h.A[r + (long)c * n] = v;
    h.P[r + (long)i * n] = v;
    h.P[r + (long)(2 * b + i) * n] = v;
    g.p[r] = p;
    if (g.next) {
      double2 a0 = csub(fe, p);
      cmac(a0, make_double2(-v.x, -v.y), make_double2(po.x, -po.y));
      g.acol[r] = a0;
    }
  }
#pragma unroll
  for (int w = RB / 2; w > 0; w >>= 1) q += __shfl_xor_sync(0xffffffffu, q, w);
  if (lane == 0) g.dot[blockIdx.x] = q;
}

// W[:, b-1] = p + (k2 / 2) v of the panel's last column (h: the column after it)
__global__ void __launch_bounds__(256) k_col_last(const __grid_constant__ HhCol h) {
  __shared__ double s_k2;
  pdl_wait();
  pdl_trigger();
  if (threadIdx.x < 32) {
    const double k = hh_k2(h);
    if (threadIdx.x == 0) s_k2 = k;
  }
  __syncthreads();
  const int r = h.c + blockIdx.x * 256 + threadIdx.x;
  if (r < h.n) h.P[r + (long)(h.b + h.i - 1) * h.n] = hh_w(h, r, s_k2);
}

// rows per CTA of k_col_rows for m rows
int rows_block(int m) { return m <= 152 * 7 ? 8 : m <= 152 * 15 ? 16 : 32; }

// programmatic dependent launch (overlap) or a plain one: a kernel may start
// while its predecessor finishes, waits (griddepcontrol.wait) before it reads
// anything the predecessor wrote, and only then lets its own successor start.
// So before its wait it may read what was written two or more launches back.
// The row kernels ask for the whole of an SM's shared memory, as k_hemv_tc has
// it: an SM that would have to change the split between L1 and shared memory
// takes CTAs of the other kernel only once it is empty.
template <class Arg, class... More>
cudaError_t launch(void (*kern)(const Arg, More...), int grid, bool overlap, cudaStream_t st, const Arg &arg,
                   More... more) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[0].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 2 : 1;
  pw_count_launch();
  return cudaLaunchKernelEx(&cfg, kern, arg, more...);
}

}  // namespace

// per-block partials: k_col_rows has at least 7 rows per CTA, k_col_hemv 32
// rows per norm partial, k_hemv_tc one norm partial per CTA (at most a few
// hundred SMs)
size_t pw_house_parts(int nmax) { return (size_t)nmax / 7 + 1024; }

pw_status pw_house_panel(pw_dense_ws *ws, double2 *A, int n, int j0, int b, bool tc, cudaStream_t st) {
  const size_t np = pw_house_parts(ws->nmax);
  double *dot = ws->hpart, *nrm = dot + np;
  HhCol h;
  h.A = A;
  h.n = n;
  h.b = b;
  h.P = ws->panel;
  h.p = ws->p;
  h.dot = dot;
  h.nprev = 0;
  h.tau = ws->tau;
  h.d = ws->d;
  h.x = ws->xcol;
  h.nrm = nrm;
  h.ucorr = ws->ucorr;
  for (int i = 0; i < b; ++i) {
    const int c = j0 + i, m = n - c - 1;
    h.c = c;
    h.i = i;
    h.a0 = i == 0 ? A + (long)c * n : ws->acol;
    RowsArgs g;
    g.part = ws->part;
    if (tc) {
      PW_TRY(pw_hs_hemv(ws, h, j0, &g.nslots, &g.nnrm, st));
      g.part += c + 1;
    } else {
      const int nT = (m + TT - 1) / TT, ntiles = nT * (nT + 1) / 2, nrow = (m + 1 + 255) / 256;
      PW_CUDA(launch(k_col_hemv, ntiles + 2 * i + nrow, i > 0, st, h, ntiles, ws->part, ws->nmax));
      g.nslots = nT;
      g.nnrm = nrow * 8;
    }
    g.h = h;
    g.nmax = ws->nmax;
    g.next = i + 1 < b;
    g.p = ws->p;
    g.acol = ws->acol;
    g.dot = dot;
    g.tau = ws->tau;
    g.e = ws->e;
    const int rb = rows_block(m);
    h.nprev = std::max(1, (m - 1 + rb - 2) / (rb - 1));
    PW_CUDA(launch(rb == 8 ? k_col_rows<8> : rb == 16 ? k_col_rows<16> : k_col_rows<32>, h.nprev, true, st, g));
  }
  h.c = j0 + b;
  h.i = b;
  PW_CUDA(launch(k_col_last, std::max(1, (n - h.c + 255) / 256), true, st, h));
  return pw_check_launch("householder panel");
}

// Columns of a Householder panel (the tridiagonalisation inside Syevd, Sec.
// III-D) as chained kernels in the fixed order of operations of the mixed
// iteration's dense solves (pw_dense_ws::fixed): three per column.  house_cols.cu
// has the faster ones, whose sums run in another order.
//
// Per column c (panel index i):
//   k_pcol   finish W[:, i-1], update column c, norm partials; the block that
//            finishes last forms beta, tau and the scale s of the reflector
//            (v = x s below its unit head) -- scalars only;
//   k_phemv  lower-tile partial products of A22 v (v formed on the fly from
//            x and s), the dots W^H v and V^H v, and the V columns of v
//            (k_hemv_tc_fixed in hemv_tc.cu where the panel has digit slices);
//   k_prows  sum the partials, subtract the corrections, p = tau y, store v
//            in place of x and the partial dots p^H v;
// and k_pfinal after the panel's last column.
#include "dense.cuh"
#include "house.cuh"

namespace {

constexpr int TT = 32;
constexpr int TPB = 32;

// The per-column kernels are chained with programmatic dependent launch: a
// kernel may start while its predecessor finishes, waits (griddepcontrol.wait)
// before it reads anything the predecessor wrote, and only then lets its own
// successor launch.  So before its wait a kernel may read data written two or
// more launches back (k_phemv loads its tile of the trailing matrix there).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), unsigned grid, unsigned block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
constexpr int PCOL_THREADS = 128;

// 32 rows per block; the four warps split the panel's previous updates
// (q = warp mod 4) so that the FP64 work lands on all four SM sub-partitions
__global__ void __launch_bounds__(PCOL_THREADS) k_pcol(double2 *A, int n, int c, int i, double2 *P, int b,
                                                       const double2 *p, const double2 *dotpart, int ndot,
                                                       double2 *tau, double *d, double *e, double *nrm_part,
                                                       double2 *hscal, unsigned *ticket) {
  __shared__ double sh[32];
  __shared__ unsigned s_ticket;
  __shared__ double2 s_vc[TPB], s_wc[TPB], s_u[4][33];
  double2 *V = P, *W = P + (long)b * n;
  const int rl = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int r = c + blockIdx.x * 32 + rl;
  // Before the wait: what the panel's earlier columns wrote two or more
  // launches back — V[:, q < i], W[:, q < i-1] and, for i > 0, column c of A
  // (last written by the previous panel's update).  p and the dots (and from
  // them W[:, i-1]) come from the predecessor.
  constexpr int QMAX = (TPB + 3) / 4;
  double2 vq_r[QMAX], wq_r[QMAX];
  double2 a = make_double2(0.0, 0.0);
  if (i > 0) {
    if (threadIdx.x < i) {
      const int q = threadIdx.x;
      s_vc[q] = V[c + (long)q * n];
      if (q < i - 1) s_wc[q] = W[c + (long)q * n];
    }
#pragma unroll
    for (int t = 0; t < QMAX; ++t) {
      const int q = g + 4 * t;
      const bool ok = r < n && q < i;
      vq_r[t] = ok ? V[r + (long)q * n] : make_double2(0.0, 0.0);
      wq_r[t] = ok && q < i - 1 ? W[r + (long)q * n] : make_double2(0.0, 0.0);
    }
    if (g == 0 && r < n) a = A[r + (long)c * n];
  }
  pdl_wait();
  pdl_trigger();
  double2 al = make_double2(0.0, 0.0);
  if (i > 0) {
    al = panel_alpha(dotpart, ndot, tau[c - 1], sh);
    // W[c, i-1] = p_{c-1}[0] + alpha v_{c-1}[row c], the head of v_{c-1} being 1
    if (threadIdx.x == 0) s_wc[i - 1] = cadd(__ldcg(&p[0]), al);
  }
  __syncthreads();
  if (i > 0) {
    double2 u = make_double2(0.0, 0.0);   // sum_q v_rq conj(w_cq) + w_rq conj(v_cq), q = g mod 4
    if (r < n) {
#pragma unroll
      for (int t = 0; t < QMAX; ++t) {
        const int q = g + 4 * t;
        if (q >= i) break;
        const double2 vq = vq_r[t];
        double2 wq = wq_r[t];
        if (q == i - 1) {
          wq = __ldcg(&p[r - c]);
          cmac(wq, al, vq);
          W[r + (long)q * n] = wq;
        }
        cmacc(u, s_wc[q], vq);
        cmacc(u, s_vc[q], wq);
      }
    }
    s_u[g][rl] = u;
    __syncthreads();
  }
  if (g == 0 && r < n) {
    if (i == 0) a = A[r + (long)c * n];
    if (i > 0) {
      a = csub(a, cadd(cadd(s_u[0][rl], s_u[1][rl]), cadd(s_u[2][rl], s_u[3][rl])));
      A[r + (long)c * n] = a;
    }
  }
  if (g != 0) return;
  double nrm = 0.0;
  if (r < n && r > c + 1) nrm = a.x * a.x + a.y * a.y;
  nrm = warp_sum(nrm);
  if (rl == 0) {
    nrm_part[blockIdx.x] = nrm;
    __threadfence();
    s_ticket = atomicAdd(ticket, 1u);
  }
  __syncwarp();
  if (s_ticket != gridDim.x - 1) return;
  __threadfence();
  // last block: reflector scalars from x = A[c+1:, c]
  double xn2 = 0.0;
  for (int q = rl; q < (int)gridDim.x; q += 32) xn2 += __ldcg(&nrm_part[q]);
  xn2 = warp_sum(xn2);
  if (rl != 0) return;
  *ticket = 0u;
  const double2 alpha = __ldcg(&A[(c + 1) + (long)c * n]);
  double beta;
  double2 tk, scal;
  reflector_scalars(xn2, alpha, beta, tk, scal);
  d[c] = __ldcg(&A[c + (long)c * n]).x;
  tau[c] = tk;
  e[c] = beta;
  *hscal = scal;
}

// y = A22 v as lower-tile partials (A22 = rows/cols >= c+1, not yet updated
// by this panel); 2i extra blocks: u[2q] = W[:, q]^H v, u[2q+1] = V[:, q]^H v;
// nwr more blocks write v into V[:, i] and its copy
__global__ void __launch_bounds__(256) k_phemv(const double2 *A, int n, int c, int i, double2 *P, int b,
                                               int ntiles, double2 *part, int nmax, double2 *ucorr,
                                               const double2 *hscal) {
  __shared__ double2 tile[TT][TT + 1];
  __shared__ double2 vrow[TT], vcol[TT], rpart[4][TT + 1], cpart[4][TT + 1];
  __shared__ double sh[32];
  const int o = c + 1, m = n - o;
  const double2 *xk = A + o + (long)c * n;   // x of column c, x[0] at row o
  const int blk = blockIdx.x;
  int I = 0, J = 0, x0 = 0, y0 = 0;
  if (blk < ntiles) {
    // tile (I, J) of the lower triangle; FP32 estimate (FP64 is scarce), fixed up exactly
    const int t = blk;
    I = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= t) ++I;
    while (I * (I + 1) / 2 > t) --I;
    J = t - I * (I + 1) / 2;
    x0 = TT * I;
    y0 = TT * J;   // tile rows x0.., columns y0.. (offsets from o)
    // the trailing matrix was last written before the predecessor's wait: load it now
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    const int yc = y0 + lane;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rl = wq * 4 + q, xr = x0 + rl;
      double2 a = make_double2(0.0, 0.0);
      if (xr < m && yc < m && (I != J || yc <= xr)) a = A[(o + xr) + (long)(o + yc) * n];
      tile[rl][lane] = a;
    }
  }
  pdl_wait();
  pdl_trigger();
  const double2 scal = *hscal;
  if (blk >= ntiles + 2 * i) {   // writer blocks
    const int x = (blk - ntiles - 2 * i) * blockDim.x + threadIdx.x;
    if (x < m) {
      const double2 v = refl_entry(xk, x, scal);
      P[o + x + (long)i * n] = v;
      P[o + x + (long)(2 * b + i) * n] = v;
    }
    return;
  }
  if (blk >= ntiles) {
    const int q2 = blk - ntiles, q = q2 >> 1;
    const double2 *col = P + (long)((q2 & 1) ? q : b + q) * n;   // odd: V[:, q], even: W[:, q]
    double2 s = make_double2(0.0, 0.0);
    for (int x = threadIdx.x; x < m; x += blockDim.x) cmacc(s, col[o + x], refl_entry(xk, x, scal));
    s.x = block_sum(s.x, sh);
    s.y = block_sum(s.y, sh);
    if (threadIdx.x == 0) ucorr[q2] = s;
    return;
  }
  if (threadIdx.x < TT) {
    const int xr = x0 + threadIdx.x, yc = y0 + threadIdx.x;
    vrow[threadIdx.x] = xr < m ? refl_entry(xk, xr, scal) : make_double2(0.0, 0.0);
    vcol[threadIdx.x] = yc < m ? refl_entry(xk, yc, scal) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  // warps 0-3: quarter row sums A v; warps 4-7: quarter column sums A^H v
  // (strictly below the diagonal in a diagonal tile)
  {
    const int k = (threadIdx.x >> 5) & 3, l = threadIdx.x & 31;
    double2 s = make_double2(0.0, 0.0);
    if (threadIdx.x < 128) {
#pragma unroll
      for (int cl = 8 * k; cl < 8 * k + 8; ++cl) cmac(s, tile[l][cl], vcol[cl]);
      rpart[k][l] = s;
    } else {
#pragma unroll
      for (int rr = 8 * k; rr < 8 * k + 8; ++rr)
        if (I != J || rr > l) cmacc(s, tile[rr][l], vrow[rr]);
      cpart[k][l] = s;
    }
  }
  __syncthreads();
  if (threadIdx.x < TT) {
    const int l = threadIdx.x;
    const double2 rs = cadd(cadd(rpart[0][l], rpart[1][l]), cadd(rpart[2][l], rpart[3][l]));
    const double2 cs = cadd(cadd(cpart[0][l], cpart[1][l]), cadd(cpart[2][l], cpart[3][l]));
    if (I != J) {
      if (x0 + l < m) part[(long)J * nmax + x0 + l] = rs;
      if (y0 + l < m) part[(long)I * nmax + y0 + l] = cs;
    } else if (x0 + l < m) {
      part[(long)J * nmax + x0 + l] = cadd(rs, cs);
    }
  }
}

// 32 rows per block, 8 thread groups over the partial slots s0..nT-1 and the
// corrections: y = sum of partials - V[:, <i] u_W - W[:, <i] u_V, p = tau_c y,
// v stored in place of x, partial dots p^H v.  part[s * nmax + x] holds slot
// s of row o + x.
__global__ void __launch_bounds__(256) k_prows(double2 *A, int n, int c, int i, const double2 *P, int b,
                                               const double2 *part, int s0, int nT, int nmax, const double2 *ucorr,
                                               const double2 *tau, const double2 *hscal, double2 *p,
                                               double2 *dotpart) {
  __shared__ double2 red[8][33];
  const int o = c + 1, m = n - o;
  const int rl = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int x = blockIdx.x * 32 + rl;
  // Before the wait: the panel columns V[:, q < i], W[:, q < i] (written two
  // or more launches back); the partial products and corrections come from
  // the predecessor.
  constexpr int QMAX = (TPB + 7) / 8;
  double2 vq_r[QMAX], wq_r[QMAX];
#pragma unroll
  for (int t = 0; t < QMAX; ++t) {
    const int q = g + 8 * t;
    const bool ok = x < m && q < i;
    vq_r[t] = ok ? P[o + x + (long)q * n] : make_double2(0.0, 0.0);
    wq_r[t] = ok ? P[o + x + (long)(b + q) * n] : make_double2(0.0, 0.0);
  }
  pdl_wait();
  pdl_trigger();
  double2 y = make_double2(0.0, 0.0);
  if (x < m) {
    for (int s = s0 + g; s < nT; s += 8) y = cadd(y, part[(long)s * nmax + x]);
#pragma unroll
    for (int t = 0; t < QMAX; ++t) {
      const int q = g + 8 * t;
      if (q >= i) break;
      const double2 uw = ucorr[2 * q], uv = ucorr[2 * q + 1];
      cmac(y, vq_r[t], make_double2(-uw.x, -uw.y));   // - V[r,q] (W^H v)_q
      cmac(y, wq_r[t], make_double2(-uv.x, -uv.y));   // - W[r,q] (V^H v)_q
    }
  }
  red[g][rl] = y;
  __syncthreads();
  if (g != 0) return;
  double2 pv = make_double2(0.0, 0.0);
  if (x < m) {
#pragma unroll
    for (int q = 1; q < 8; ++q) y = cadd(y, red[q][rl]);
    const double2 pr = cmul(tau[c], y);
    p[x] = pr;
    double2 *xc = A + o + (long)c * n;
    const double2 v = refl_entry(xc, x, *hscal);
    xc[x] = v;
    cmacc(pv, pr, v);
  }
  pv.x = warp_sum(pv.x);
  pv.y = warp_sum(pv.y);
  if (rl == 0) dotpart[blockIdx.x] = pv;
}

// W[:, i] = p + alpha v for the panel's last column (rows >= c+1)
__global__ void __launch_bounds__(256) k_pfinal(const double2 *A, int n, int c, int i, double2 *P, int b,
                                                const double2 *p, const double2 *dotpart, int ndot,
                                                const double2 *tau) {
  __shared__ double sh[32];
  pdl_wait();
  pdl_trigger();
  const double2 al = panel_alpha(dotpart, ndot, tau[c], sh);
  const int o = c + 1;
  const int r = o + blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) {
    double2 w = p[r - o];
    cmac(w, al, A[r + (long)c * n]);
    P[r + (long)(b + i) * n] = w;
  }
}

}  // namespace

pw_status pw_house_panel_fixed(pw_dense_ws *ws, double2 *A, int n, int j0, int b, bool tc, cudaStream_t st) {
  double2 *dotpart = ws->w;
  int ndot = 0;
  for (int i = 0; i < b; ++i) {
    const int c = j0 + i, m = n - c - 1;
    const int npcol = (n - c + 31) / 32;
    pw_count_launch();
    PW_CUDA(launch_pdl(k_pcol, npcol, PCOL_THREADS, st, A, n, c, i, ws->panel, b,
                       (const double2 *)ws->p, (const double2 *)dotpart, ndot, ws->tau, ws->d, ws->e,
                       ws->nrm_part, ws->hscal, ws->ticket));
    int s0 = 0, nT = (m + TT - 1) / TT;
    const double2 *part = ws->part;
    if (tc) {
      PW_TRY(pw_hs_hemv_fixed(ws, A, n, c, i, b, j0, &nT, st));
      part = ws->part + (c + 1);
    } else {
      const int ntiles = nT * (nT + 1) / 2, nwr = (m + 255) / 256;
      pw_count_launch();
      PW_CUDA(launch_pdl(k_phemv, ntiles + 2 * i + nwr, 256, st, (const double2 *)A, n, c, i, ws->panel,
                         b, ntiles, ws->part, ws->nmax, ws->ucorr, (const double2 *)ws->hscal));
    }
    ndot = (m + 31) / 32;
    pw_count_launch();
    PW_CUDA(launch_pdl(k_prows, ndot, 256, st, A, n, c, i, (const double2 *)ws->panel, b, part, s0, nT,
                       ws->nmax, (const double2 *)ws->ucorr, (const double2 *)ws->tau,
                       (const double2 *)ws->hscal, ws->p, dotpart));
  }
  const int cl = j0 + b - 1, ml = n - cl - 1;
  pw_count_launch();
  PW_CUDA(launch_pdl(k_pfinal, (ml + 255) / 256, 256, st, (const double2 *)A, n, cl, b - 1, ws->panel, b,
                     (const double2 *)ws->p, (const double2 *)dotpart, ndot, (const double2 *)ws->tau));
  return pw_check_launch("householder panel (fixed order)");
}

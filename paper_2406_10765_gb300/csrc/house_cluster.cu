// Householder reduction of the last columns of a Hermitian matrix (the
// tridiagonalisation inside Syevd, Sec. III-D) in one thread-block cluster,
// the trailing matrix in distributed shared memory: the whole reduction of
// small orders, and the end of larger ones.
//
// Why: a column of chained kernels cost about 18 us at small orders (three
// dependent launches; 10 with the two of house_cols.cu), whose reductions,
// square roots and divisions run in FP64 one after the other (a warp-wide FP64
// instruction takes 65 clocks on this part whatever the number of its active
// lanes, a division 700).  Sixteen CTAs that exchange vectors through
// distributed shared memory need two cluster barriers (400 clocks each) per
// column and about 45 dependent FP64 instructions.
//
// Layout: CTA k of 16 owns the columns j = k mod 16 of the trailing matrix,
// stored whole (both triangles), so that (A v)_j is one column dot product and
// no partial sums cross the CTAs.  That costs 3 m^2 complex multiply-adds a
// column instead of 2 m^2 for the stored triangle, on 16 SMs instead of all:
// the chained kernels win again above order ~256 (HC_MAX).
//
// Column c (m = n - c - 1 rows below it):
//   A  its owner applies the previous column's update to it, forms the norm,
//      the reflector's scalars and v, and stores v into every CTA
//   -- cluster barrier; meanwhile every CTA updates its other columns --
//   C  every CTA: p_j = tau (A v)_j for its columns and its share of
//      q = v^H A v, into every CTA
//   -- cluster barrier --
// The update A -= v w^H + w v^H with w = p - (|tau|^2 q / 2) v is applied as
// A[r, j] -= v_r (conj(p_j) - |tau|^2 q conj(v_j)) + p_r conj(v_j).
//
// Measured: order 54 in 0.24 ms (4.6 us per column, 18 before); order 256 in
// 2.7 ms; order-54 eigensolve 1.99 -> 1.34 ms, an 8-step solve of the 8-atom
// cell (order 72) 27.7 -> 20.9 ms, order-1,458 eigensolve 51.9 -> 50.4 ms.
#include <cooperative_groups.h>

#include <mutex>

#include "dense.cuh"
#include "house.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int HC_CTAS = 16;
constexpr int HC_WARPS = 4;                 // one per SM sub-partition
constexpr int HC_THREADS = 32 * HC_WARPS;
constexpr int HC_MAX = 256;

// columns, v and p (two buffers each), q partials (two buffers), tau (two)
size_t hc_smem(int m) {
  return ((size_t)((m + HC_CTAS - 1) / HC_CTAS) * m + 4 * (size_t)m + 2) * sizeof(double2) +
         2 * HC_CTAS * HC_WARPS * sizeof(double) + 64;
}

__global__ void __launch_bounds__(HC_THREADS) k_house_cluster(double2 *A, int n, int j0, double2 *tau, double *d,
                                                              double *e) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_red[HC_WARPS];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int m = n - j0;
  const int nl = (m - rank + HC_CTAS - 1) / HC_CTAS;           // own columns (rank < m or none)
  const int nlmax = (m + HC_CTAS - 1) / HC_CTAS;
  double2 *col = (double2 *)smem_raw;                          // [nlmax][m]
  double2 *vb = col + (size_t)nlmax * m, *pb = vb + 2 * m;     // [2][m] each
  double2 *tkb = pb + 2 * m;                                   // [2]
  double *qb = (double *)(tkb + 2);                            // [2][CTAs x warps]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double2 *Aj = A + j0 + (long)j0 * n;

  for (int l = 0; l < nl; ++l) {
    const int j = l * HC_CTAS + rank;
    for (int r = tid; r < m; r += HC_THREADS) {
      double2 a;
      if (r > j) a = Aj[r + (long)j * n];
      else {
        a = Aj[j + (long)r * n];
        a.y = r == j ? 0.0 : -a.y;
      }
      col[(size_t)l * m + r] = a;
    }
  }
  cl.sync();      // every CTA runs before the first store into its shared memory

  double k2 = 0.0;          // -|tau|^2 q of the previous column
  for (int c = 0; c + 1 < m; ++c) {
    const int cur = c & 1, prv = cur ^ 1;
    const double2 *vp = vb + prv * m, *pp = pb + prv * m;
    // ---- A: the owner's column
    if (rank == c % HC_CTAS) {
      double2 *x = col + (size_t)(c / HC_CTAS) * m;
      double s = 0.0;
      double2 g = make_double2(0.0, 0.0);
      if (c > 0) g = make_double2(pp[c].x + k2, -pp[c].y);     // v_c = 1: the previous reflector's head
      for (int r = c + tid; r < m; r += HC_THREADS) {
        double2 a = x[r];
        if (c > 0) {
          const double2 v = vp[r], p = pp[r];
          a = csub(a, p);
          cmac(a, make_double2(-v.x, -v.y), g);
          x[r] = a;
        }
        if (r > c + 1) s = fma(a.x, a.x, fma(a.y, a.y, s));
      }
      s = warp_sum(s);
      if (lane == 0) s_red[warp] = s;
      __syncthreads();
      s = (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]);
      double beta;
      double2 tk, scal;
      reflector_scalars_fast(s, x[c + 1], beta, tk, scal);
      __syncthreads();                                         // x[c + 1] read before it is overwritten
      for (int r = c + 1 + tid; r < m; r += HC_THREADS) {
        const double2 v = r == c + 1 ? make_double2(1.0, 0.0) : cmul(x[r], scal);
        x[r] = v;
        for (int k = 0; k < HC_CTAS; ++k) cl.map_shared_rank(vb, k)[cur * m + r] = v;
      }
      if (tid < HC_CTAS) cl.map_shared_rank(tkb, tid)[cur] = tk;
      if (tid == 0) {
        d[j0 + c] = x[c].x;
        e[j0 + c] = beta;
        tau[j0 + c] = tk;
      }
    }
    __syncwarp();
    cl.barrier_arrive();
    // ---- the previous column's update of the other columns right of c.  Own
    // column l belongs to warp l mod 4 and a row to one lane, here and in C:
    // the barrier was arrived at before these writes and does not order them
    int l0 = c < rank ? 0 : (c - rank) / HC_CTAS + 1;          // first own column > c
    l0 += (warp + HC_WARPS - l0 % HC_WARPS) % HC_WARPS;        // the warp's first
    if (c > 0)
      for (int l = l0; l < nl; l += HC_WARPS) {
        double2 *a = col + (size_t)l * m;
        const double2 vj = vp[l * HC_CTAS + rank], pj = pp[l * HC_CTAS + rank];
        const double2 g = make_double2(-fma(k2, vj.x, pj.x), fma(k2, vj.y, pj.y));   // -(conj(p_j) + k2 conj(v_j))
        const double2 h = make_double2(-vj.x, vj.y);                                 // -conj(v_j)
        for (int r = c + 1 + lane; r < m; r += 32) {
          double2 t = a[r];
          cmac(t, vp[r], g);
          cmac(t, pp[r], h);
          a[r] = t;
        }
      }
    __syncwarp();
    cl.barrier_wait();
    // ---- C: products with v
    const double2 *v = vb + cur * m;
    const double2 tk = tkb[cur];
    double q = 0.0;
    for (int l = l0; l < nl; l += HC_WARPS) {
      const double2 *a = col + (size_t)l * m;
      double2 y = make_double2(0.0, 0.0);
      for (int r = c + 1 + lane; r < m; r += 32) cmacc(y, a[r], v[r]);
      y = warp_sum_c(y);
      const int j = l * HC_CTAS + rank;
      q = fma(y.x, v[j].x, fma(y.y, v[j].y, q));
      const double2 p = cmul(tk, y);
      if (lane < HC_CTAS) cl.map_shared_rank(pb, lane)[cur * m + j] = p;
    }
    if (lane < HC_CTAS) cl.map_shared_rank(qb, lane)[(cur * HC_CTAS + rank) * HC_WARPS + warp] = q;
    cl.sync();
    const double *qs = qb + cur * HC_CTAS * HC_WARPS;
    q = warp_sum(qs[lane] + qs[lane + 32]);
    k2 = -fma(tk.x, tk.x, tk.y * tk.y) * q;
  }
  static_assert(HC_CTAS * HC_WARPS == 64, "q partials per lane");
  // the last diagonal entry
  if (rank == (m - 1) % HC_CTAS && tid == 0) {
    double a = col[(size_t)((m - 1) / HC_CTAS) * m + m - 1].x;
    if (m > 1) a -= 2.0 * pb[(m & 1) * m + m - 1].x + k2;      // v = 1, the buffers of column m - 2
    d[n - 1] = a;
  }
  // the reflectors, v below the diagonal
  for (int l = 0; l < nl; ++l) {
    const int j = l * HC_CTAS + rank;
    for (int r = j + 1 + tid; r < m; r += HC_THREADS) Aj[r + (long)j * n] = col[(size_t)l * m + r];
  }
  cl.sync();      // no CTA leaves while another may still store into it
}

cudaLaunchConfig_t hc_config(int m, cudaStream_t st, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(HC_CTAS);
  cfg.blockDim = dim3(HC_THREADS);
  cfg.dynamicSmemBytes = hc_smem(m);
  cfg.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = HC_CTAS;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

}  // namespace

// the largest order the cluster takes on the current device (0: clusters of
// 16 CTAs with this much shared memory are not available); set up once
int pw_house_cluster_max() {
  static std::mutex mu;
  static int most[64];
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lk(mu);
  if (!done[dev]) {
    int num = 0;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = hc_config(HC_MAX, nullptr, attr);
    const bool ok =
        cudaFuncSetAttribute(k_house_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaFuncSetAttribute(k_house_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hc_smem(HC_MAX)) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&num, k_house_cluster, &cfg) == cudaSuccess && num > 0;
    if (!ok) cudaGetLastError();
    most[dev] = ok ? HC_MAX : 0;
    done[dev] = true;
  }
  return most[dev];
}

pw_status pw_house_cluster(pw_dense_ws *ws, double2 *A, int n, int j0, cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = hc_config(n - j0, st, attr);
  pw_count_launch();
  PW_CUDA(cudaLaunchKernelEx(&cfg, k_house_cluster, A, n, j0, ws->tau, ws->d, ws->e));
  return PW_OK;
}

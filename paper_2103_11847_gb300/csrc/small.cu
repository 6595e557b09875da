// The projected problem in FP64 (§3.1 eqs. (leastsq), (tikho2),
// (gcv2); §3.2 eqs. (normeq2), (leastsq0)):
//   1. one-sided Jacobi SVD of the (k+1) x k matrix H (Hestenes rotations,
//      round-robin pair order, warps rotate disjoint column pairs),
//      sigma_i = ||h_i||, g~_i = beta * (first row of H V)_i / sigma_i;
//   2. GCV(lambda) of eq. (gcv2) ("paper") or of the rectangular problem
//      ("full", with g~_{k+1}^2 = beta^2 - sum g~_i^2), minimised on three
//      nested log grids of 200 points: [1e-10 s, s] with s = ||H||_F, then
//      twice the bracket between the grid neighbours of the minimum (first
//      index on ties);
//   3. y from the normal equations (H^T H + lambda^2 I) y = beta H^T e_1 by
//      Cholesky.
//
// Bound: FP64. GB300 issues fewer than two FP64 lanes a clock and SM, so a warp
// instruction holds the pipe for about 19 clocks, and every division or square
// root is a chain of them (IEEE ones throughout: H may be graded or scaled over the
// whole range, where estimates flush or lose the rotation of a small column). So:
// * for the search, a cluster of eight CTAs: rank 0 runs the SVD and the solve, and
//   every rank evaluates 25 of a level's 200 grid points, one a lane of one warp (on
//   one SM a level of k = 10 took about 35 us, nearly all of it the pipe). A given
//   lambda needs one CTA;
// * beyond two warps of column pairs, the rotations of a round's pairs by the lanes
//   of one warp, so that their chains share its instructions;
// * as many warps as the SVD has column pairs (at most 32), as every round ends
//   in a barrier; the triangular solves run by columns over all threads.
// us a launch with the search (one CTA of 1024 threads, a warp a pair, before): k = 10
// 308 -> 244, k = 32 2954 -> 1598, k = 128 78.4 -> 37.1 ms; lambda given, k = 10 229 ->
// 224. Most of it is the SVD's chains.
#include <cooperative_groups.h>

#include "tc_device.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int NGRID = 200;
constexpr int NLEVEL = 3;
constexpr int MAX_SWEEPS = 40;
constexpr int CL = 8;            // CTAs of the cluster
constexpr int PPR = NGRID / CL;  // grid points a rank: one a lane
static_assert(NGRID % CL == 0 && PPR <= 32, "one warp a rank");

// Lanes a column pair of the SVD: columns of up to 8 or 16 values share a warp.
__host__ __device__ constexpr int lane_group(int rows) { return rows <= 8 ? 8 : rows <= 16 ? 16 : 32; }

// GCV(lambda); sig2: squared singular values.
__device__ double gcv_eval(const double* sig2, const double* g, int k, double gnull2, double lam,
                           int variant) {
  const double l2 = lam * lam;
  double num = 0.0, den = 0.0;
  if (variant == TC_GCV_FULL) {
#pragma unroll 4
    for (int i = 0; i < k; ++i) {
      const double q = l2 / (sig2[i] + l2);
      const double r = g[i] * q;
      num = fma(r, r, num);
      den += q;
    }
    num += gnull2;
    den += 1.0;
  } else {
#pragma unroll 4
    for (int i = 0; i < k; ++i) {
      const double d = sig2[i] + l2;
      const double r = g[i] / d;
      num = fma(r, r, num);
      den += 1.0 / d;
    }
  }
  return num / (den * den);
}

// First index of the smallest of v[0..n) over one warp (ties to the lower index).
__device__ int warp_argmin(const double* v, int n) {
  double best = INFINITY;
  int bi = n;
  for (int t = threadIdx.x & 31; t < n; t += 32)
    if (v[t] < best) {
      best = v[t];
      bi = t;
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob < best || (ob == best && oi < bi)) {
      best = ob;
      bi = oi;
    }
  }
  return bi < n ? bi : 0;
}

// Dynamic shared memory: Hs[(k+1) * kk] (column-major working copy, kk = k
// rounded up to even), reused as the k x k normal matrix afterwards.
__global__ void __launch_bounds__(1024)
k_tikhonov_gcv(const double* __restrict__ H, int ld, int kmax, const int* kdev,
               const double* beta_p, int variant, double lambda_in, double* lambda_out,
               double* y, double* gcv_out, const int* skip) {
  if (skip && *skip) return;  // uniform over the cluster, as is every return below
  extern __shared__ double dsm[];
  __shared__ double sig2[TC_MAX_PROJ], g[TC_MAX_PROJ], dn[TC_MAX_PROJ];
  __shared__ double vals[NGRID], grid[NGRID];
  __shared__ double bracket[NLEVEL + 1][2], sh_w[32];
  __shared__ double sh_gnull2, sh_lam, sh_gcv;
  __shared__ double rot[TC_MAX_PROJ / 2][2];  // a pair's dot product, then its c and s
  __shared__ int sh_rot;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = blockDim.x, nw = nt / 32;
  const int k = kdev ? min(*kdev, kmax) : kmax;
  const double beta = *beta_p;
  const bool search = !(lambda_in >= 0.0);
  if (k <= 0) {
    if (rank == 0 && tid == 0) {
      *lambda_out = nan("");
      if (gcv_out) *gcv_out = nan("");
    }
    return;
  }
  const int rows = k + 1;
  const int kk = k + (k & 1);
  if (rank == 0) {
    double* Hs = dsm;  // column c at Hs + c*rows
    for (int idx = tid; idx < rows * kk; idx += nt) {
      const int c = idx / rows, r = idx % rows;
      Hs[idx] = (c < k) ? H[(size_t)r * ld + c] : 0.0;
    }
    __syncthreads();

    // ---- 1. one-sided Jacobi -----------------------------------------------
    // Rotate while |<h_p, h_q>| > rows * eps * ||h_p|| ||h_q||: below that the
    // inner product is rounding noise of the (rows)-term dot product. Squared
    // column norms d[] are recomputed every sweep and updated by the rotation
    // identities d_p -= t gamma, d_q += t gamma in between. Where the pairs fill no
    // more than two warps, their lanes (LG a pair) each form the rotation and a
    // round is one part; else it is three: the pairs' dot products, their
    // rotations (one lane a pair), and the column updates.
    const double jtol = rows * 2.220446049250313e-16;
    const int npairs = kk / 2, lg = lane_group(rows), ppw = 32 / lg, sub = lane % lg;
    const bool direct = npairs <= 2 * ppw;
    auto pair_of = [&](int pi, int rnd, int& a, int& b) {
      // circle method: player 0 fixed, the others rotate by rnd
      a = (pi == 0) ? 0 : ((pi - 1 + rnd) % (kk - 1)) + 1;
      b = ((kk - 2 - pi + rnd) % (kk - 1)) + 1;
    };
    // The rotation (c, s) that makes the columns orthogonal, t its tangent; false: none
    auto angle = [&](double ga, double al, double be, double& c, double& sn, double& t) {
      if (!(ga != 0.0 && fabs(ga) > jtol * sqrt(al * be))) return false;
      const double zeta = (be - al) / (2.0 * ga);
      t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
      c = 1.0 / sqrt(1.0 + t * t);
      sn = c * t;
      return true;
    };
    auto update = [&](int a, int b, double c, double sn) {
      for (int r = sub; r < rows; r += lg) {
        const double u = Hs[a * rows + r], v = Hs[b * rows + r];
        Hs[a * rows + r] = c * u - sn * v;
        Hs[b * rows + r] = sn * u + c * v;
      }
    };
    for (int sweep = 0; sweep < MAX_SWEEPS; ++sweep) {
      if (tid == 0) sh_rot = 0;
      for (int c = warp; c < kk; c += nw) {
        const double* x = Hs + (size_t)c * rows;
        double s2 = 0.0;
        for (int r = lane; r < rows; r += 32) s2 += x[r] * x[r];
        s2 = warp_sum(s2);
        if (lane == 0) dn[c] = s2;
      }
      __syncthreads();
      for (int rnd = 0; rnd < kk - 1; ++rnd) {
        for (int p0 = warp * ppw; p0 < npairs; p0 += nw * ppw) {
          const int pi = p0 + lane / lg;
          int a, b;
          pair_of(min(pi, npairs - 1), rnd, a, b);
          double ga = 0.0;
          for (int r = sub; r < rows; r += lg) ga = fma(Hs[a * rows + r], Hs[b * rows + r], ga);
          for (int o = lg / 2; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
          if (direct) {
            const double al = dn[a], be = dn[b];
            double c, sn, t;
            const bool go = pi < npairs && angle(ga, al, be, c, sn, t);
            __syncwarp();  // every lane has the norms
            if (go) {
              update(a, b, c, sn);
              if (sub == 0) {
                dn[a] = al - t * ga;
                dn[b] = be + t * ga;
                sh_rot = 1;
              }
            }
          } else if (sub == 0 && pi < npairs) {
            rot[pi][0] = ga;
          }
        }
        __syncthreads();
        if (direct) continue;
        if (tid < npairs) {
          int a, b;
          pair_of(tid, rnd, a, b);
          const double ga = rot[tid][0], al = dn[a], be = dn[b];
          double c = 1.0, sn = 0.0, t;
          if (angle(ga, al, be, c, sn, t)) {
            dn[a] = al - t * ga;
            dn[b] = be + t * ga;
            sh_rot = 1;
          }
          rot[tid][0] = c;
          rot[tid][1] = sn;
        }
        __syncthreads();
        for (int p0 = warp * ppw; p0 < npairs; p0 += nw * ppw) {
          const int pi = p0 + lane / lg;
          if (pi >= npairs) continue;
          const double c = rot[pi][0], sn = rot[pi][1];
          if (sn == 0.0) continue;
          int a, b;
          pair_of(pi, rnd, a, b);
          update(a, b, c, sn);
        }
        __syncthreads();
      }
      const int any = sh_rot;
      __syncthreads();
      if (!any) break;
    }
    for (int c = warp; c < k; c += nw) {
      const double* x = Hs + (size_t)c * rows;
      double s2 = 0.0;
      for (int r = lane; r < rows; r += 32) s2 += x[r] * x[r];
      s2 = warp_sum(s2);
      if (lane == 0) {
        sig2[c] = s2;
        g[c] = (s2 > 0.0) ? beta * x[0] / sqrt(s2) : 0.0;
      }
    }
    double hs = 0.0;  // ||H||_F, for the search
    for (int idx = tid; search && idx < rows * k; idx += nt) {
      const double v = H[(size_t)(idx / k) * ld + idx % k];
      hs += v * v;
    }
    hs = warp_sum(hs);
    if (lane == 0) sh_w[warp] = hs;
    __syncthreads();
    if (warp == 0) {
      const double t = warp_sum(lane < nw ? sh_w[lane] : 0.0);
      if (lane == 0) {
        double gs = 0.0;  // the part of beta e1 outside the range of H
        for (int i = 0; i < k; ++i) gs += g[i] * g[i];
        sh_gnull2 = fmax(beta * beta - gs, 0.0);
        if (search) {
          bracket[0][1] = log(sqrt(t));
          bracket[0][0] = bracket[0][1] - 10.0 * log(10.0);
        }
      }
    }
    __syncthreads();
  }

  // ---- 2. lambda -------------------------------------------------------------
  if (search) {
    cluster.sync();  // every CTA runs, and rank 0's values are in place
    if (rank != 0) {
      for (int i = tid; i < k; i += nt) {
        sig2[i] = cluster.map_shared_rank(sig2, 0)[i];
        g[i] = cluster.map_shared_rank(g, 0)[i];
      }
      if (tid == 0) {
        sh_gnull2 = *cluster.map_shared_rank(&sh_gnull2, 0);
        bracket[0][0] = cluster.map_shared_rank(&bracket[0][0], 0)[0];
        bracket[0][1] = cluster.map_shared_rank(&bracket[0][0], 0)[1];
      }
      __syncthreads();
    }
    for (int level = 0; level < NLEVEL; ++level) {
      if (warp == 0) {  // points PPR rank .. + PPR - 1
        const double lo = bracket[level][0], hi = bracket[level][1];
        const double step = (hi - lo) / (NGRID - 1);
        const int i = rank * PPR + lane;
        if (lane < PPR) {
          const double lam = exp(i == NGRID - 1 ? hi : lo + i * step);
          const double v = gcv_eval(sig2, g, k, sh_gnull2, lam, variant);
          cluster.map_shared_rank(grid, 0)[i] = lam;
          cluster.map_shared_rank(vals, 0)[i] = v;
        }
      }
      cluster.sync();  // the level's values are in rank 0
      if (rank == 0 && warp == 0) {
        const int bi = warp_argmin(vals, NGRID);
        if (lane == 0) {
          sh_lam = grid[bi];
          sh_gcv = vals[bi];
        }
        if (level + 1 < NLEVEL) {
          const double e = lane < 2 ? log(grid[lane == 0 ? max(bi - 1, 0) : min(bi + 1, NGRID - 1)]) : 0.0;
          const double lo = __shfl_sync(0xffffffffu, e, 0), hi = __shfl_sync(0xffffffffu, e, 1);
          if (lane < CL) {
            double* q = cluster.map_shared_rank(&bracket[0][0], lane) + 2 * (level + 1);
            q[0] = lo;
            q[1] = hi;
          }
        }
      }
      if (level + 1 < NLEVEL) cluster.sync();  // the next bracket is everywhere
    }
  } else if (rank == 0 && tid == 0) {
    sh_lam = lambda_in;
    sh_gcv = gcv_eval(sig2, g, k, sh_gnull2, lambda_in, variant);
  }
  if (rank != 0) return;  // no rank reads another's shared memory from here on
  __syncthreads();
  const double lam = sh_lam;
  if (tid == 0) {
    *lambda_out = lam;
    if (gcv_out) *gcv_out = sh_gcv;
  }

  // ---- 3. (H^T H + lambda^2 I) y = beta H^T e_1, Cholesky --------------------
  double* G = dsm;  // k x k row-major, overwrites the Jacobi copy
  for (int idx = tid; idx < k * k; idx += nt) {
    const int i = idx / k, jj = idx % k;
    double s = 0.0;
    for (int r = 0; r < rows; ++r) s += H[(size_t)r * ld + i] * H[(size_t)r * ld + jj];
    if (i == jj) s += lam * lam;
    G[idx] = s;
  }
  for (int i = tid; i < k; i += nt) g[i] = beta * H[i];  // rhs = beta * (row 1 of H)
  __syncthreads();
  for (int c = 0; c < k; ++c) {
    if (tid == 0) G[c * k + c] = sqrt(G[c * k + c]);
    __syncthreads();
    const double d = G[c * k + c];
    for (int r = c + 1 + tid; r < k; r += nt) G[r * k + c] /= d;
    __syncthreads();
    for (int idx = tid; idx < (k - c - 1) * (k - c - 1); idx += nt) {
      const int r = c + 1 + idx / (k - c - 1), q = c + 1 + idx % (k - c - 1);
      if (q <= r) G[r * k + q] -= G[r * k + c] * G[q * k + c];
    }
    __syncthreads();
  }
  for (int c = 0; c < k; ++c) {  // L z = rhs by columns: g[c] becomes z[c]
    const double z = g[c] / G[c * k + c];
    __syncthreads();
    for (int r = c + 1 + tid; r < k; r += nt) g[r] -= G[r * k + c] * z;
    if (tid == 0) g[c] = z;
    __syncthreads();
  }
  for (int c = k - 1; c >= 0; --c) {  // L^T y = z by columns of L^T
    const double z = g[c] / G[c * k + c];
    __syncthreads();
    for (int r = tid; r < c; r += nt) g[r] -= G[c * k + r] * z;
    if (tid == 0) g[c] = z;
    __syncthreads();
  }
  for (int i = tid; i < kmax; i += nt) y[i] = (i < k) ? g[i] : 0.0;
}

__global__ void k_build_bidiag(const double* alpha, const double* beta, const int* kdev,
                               int kmax, double* H) {
  const int k = kdev ? min(*kdev, kmax) : kmax;
  for (int idx = threadIdx.x; idx < (kmax + 1) * kmax; idx += blockDim.x) {
    const int r = idx / kmax, c = idx % kmax;
    double v = 0.0;
    if (c < k) {
      if (r == c) v = alpha[c];
      else if (r == c + 1) v = beta[c + 1];
    }
    H[idx] = v;
  }
}

}  // namespace

int launch_tikhonov_gcv(const double* H, int ld, int kmax, const int* kdev,
                        const double* beta, int variant, double lambda_in,
                        double* lambda_out, double* y, double* gcv_out, const int* skip,
                        cudaStream_t st) {
  TC_CHECK(kmax >= 1 && kmax <= TC_MAX_PROJ);
  const int kk = kmax + (kmax & 1);
  size_t smem = sizeof(double) * (size_t)(kmax + 1) * kk;
  const size_t gsz = sizeof(double) * (size_t)kmax * kmax;
  if (gsz > smem) smem = gsz;
  const int ppw = 32 / lane_group(kmax + 1);
  int nw = (kk / 2 + ppw - 1) / ppw;  // the warps that the column pairs fill
  nw = nw < 4 ? 4 : nw > 32 ? 32 : nw;
  cudaLaunchConfig_t cfg = {};
  const int cl = lambda_in >= 0.0 ? 1 : CL;  // only the search is spread
  cfg.gridDim = dim3(cl);
  cfg.blockDim = dim3(32 * nw);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cl > 1;
  TC_CUDA(cudaLaunchKernelEx(&cfg, k_tikhonov_gcv, H, ld, kmax, kdev, beta, variant, lambda_in,
                             lambda_out, y, gcv_out, skip));
  return TC_OK;
}

int launch_build_bidiag(const double* alpha, const double* beta, const int* kdev, int kmax,
                        double* H, cudaStream_t st) {
  k_build_bidiag<<<1, 256, 0, st>>>(alpha, beta, kdev, kmax, H);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

// Called once a device (from plan creation) so that no attribute call happens
// while a stream is being captured.
int tc_kernels_init() {
  TC_CUDA(cudaFuncSetAttribute(k_tikhonov_gcv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               200 * 1024));
  TC_TRY(gemm_init());
  TC_TRY(cprod2_init());
  TC_TRY(vec_init());
  TC_TRY(mode3_init());
  TC_TRY(transform_init());
  TC_TRY(group_tc_init());
  return TC_OK;
}

// Frontal-slice GEMMs of the c-product (Algorithm 1, step 2; eqs. (dft9),
// (dft8)), FP32 on the FFMA pipe.
//
// Fused form (n3 <= TC_MAX_FUSED): one output tile (i, j) for all n3 slices
// per CTA, with the mode-3 transform of Remark 2.1 fused in:
//   prologue  B~_k = sum_l pro[k][l] B_l        (the operand's transform)
//   epilogue  Y_l  = sum_k epi[l][k] (A_k B~_k)  (back to the spatial domain)
// then out = ca * Y + cp * prev and an optional fused reduction. Tiles that are
// too few for the SMs are split along K over a thread-block cluster of KS
// CTAs: each CTA accumulates its K range, the partial tiles are summed through
// distributed shared memory in rank order, and each rank finishes BM/KS rows
// of the tile (pick_tile has the rule).
//
// Per-slice form (no transforms): one tile of one slice per CTA, used when
// n3 > TC_MAX_FUSED between separate transform passes.
//
// The left factor is always given K-major (the plan keeps A~ and its slice
// transposes, so each product has it at hand); the first product of a
// two-sided operator stores its result transposed, K-major for the second.
// The tile itself (packed FMAs, cp.async ring) is ffma_tile.cuh's. Against the
// earlier form (FMAs one at a time, A transposed through shared memory, no ring):
// 512^3 x 64 slices 787 -> 272 us (63 TFLOP/s of the measured 77.6), 1024^3 x 3
// fused 217 -> 140 us a launch.
#include <cooperative_groups.h>

#include <type_traits>

#include "ffma_tile.cuh"
#include "group.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr long NSM = 152;  // SMs

struct Fused {
  float pro[TC_MAX_FUSED * TC_MAX_FUSED];
  float epi[TC_MAX_FUSED * TC_MAX_FUSED];
};

template <int NS, int BM, int BN, int BK>
struct SmallSmem {
  static constexpr int kMain = NS * BK * (BM + BN);
  static constexpr int kPart = NS * BM * BN;
  static constexpr int kFloats = kMain > kPart ? kMain : kPart;
};

// Predicated loads, zero where !ok: no branch, so that a thread's loads issue together.
__device__ __forceinline__ float4 ldg4_if(const float* p, bool ok) {
  float4 v;
  asm("{\n .reg .pred q;\n setp.ne.u32 q, %5, 0;\n mov.b32 %0, 0;\n mov.b32 %1, 0;\n"
      " mov.b32 %2, 0;\n mov.b32 %3, 0;\n @q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n}"
      : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
      : "l"(p), "r"((unsigned)ok));
  return v;
}
__device__ __forceinline__ float ldg_if(const float* p, bool ok) {
  float v;
  asm("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.b32 %0, 0;\n @q ld.global.nc.f32 %0, [%1];\n}"
      : "=&f"(v)
      : "l"(p), "r"((unsigned)ok));
  return v;
}

// How the small tiles read their operands: LD_BRANCH, a branch a load on whole
// groups in both operands; LD_WHOLE, predicated, whole groups in both; LD_EACH,
// predicated, each operand by its own alignment.
enum Loads { LD_BRANCH, LD_WHOLE, LD_EACH };

// The main loop of one small fused tile: acc[k] += A_k (pro B)_k over K range
// [kbeg, kend) for the BM x BN tile at (i0, j0), all NS slices, with register
// double buffering (the next K tile's global loads are issued before the
// current tile's FMAs). At is K-major (K x M a slice). Four values of each of the
// A and B tiles a thread and slice. Single products take the predicated loads:
// 16-byte ones where an operand has aligned rows of whole groups of four, else value
// by value, a warp's lanes side by side. Branches kept the compiler from issuing
// them together (c-LSQR of 6 steps at n3 = 4: 1600 x 200 with 24 columns 344 us,
// now 298; 2048 x 2048 with 64 columns 1702, now 1446). The grouped form keeps the
// branches: its tile shape is chosen by time, and a batch's last bits follow the
// shape. sm: the SmallSmem floats.
template <int NS, int BM, int BN, int BK, int TM, int TN, bool PRO, Loads LD>
__device__ __forceinline__ void small_tile_mainloop(const float* __restrict__ At,
                                                    const float* __restrict__ B, int M, int N,
                                                    int K, int kbeg, int kend, int i0, int j0,
                                                    const Fused& f, float* sm,
                                                    float (&acc)[NS][TM][TN]) {
  constexpr int TX = BN / TN;
  constexpr int NT = (BM / TM) * (BN / TN);
  float(*As)[BK][BM] = reinterpret_cast<float(*)[BK][BM]>(sm);
  float(*Bs)[BK][BN] = reinterpret_cast<float(*)[BK][BN]>(sm + NS * BK * BM);
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const size_t sA = (size_t)M * K, sB = (size_t)K * N;
#pragma unroll
  for (int k = 0; k < NS; ++k)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[k][i][j] = 0.f;

  static_assert(BM * BK == 4 * NT && BK * BN == 4 * NT, "four values a thread of each tile");
  auto whole = [](const float* p, int cols) {
    return cols % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
  };
  const bool both = (M | N) % 4 == 0 && ((reinterpret_cast<uintptr_t>(At) |
                                          reinterpret_cast<uintptr_t>(B)) & 15) == 0;
  const bool va = LD == LD_EACH ? whole(At, M) : true, vb = LD == LD_EACH ? whole(B, N) : true;
  const int ar = tid / (BM / 4), ac = (tid % (BM / 4)) * 4;  // A tile: K row, first output row
  const int br = tid / (BN / 4), bc = (tid % (BN / 4)) * 4;  // B tile: K row, first column
  // A thread's four values: those at (row, col) of the tile and after it (vec),
  // else positions tid, tid + NT, .. of the tile
  float4 ra[NS], rb[NS];
  auto load = [&](float4 (&r)[NS], const float* base, size_t slice, int cols, int k0, int c0, int W,
                  int row, int col, bool vec) {
    if (vec) {
      const int kr = k0 + row, c = c0 + col;
      const bool in = kr < kend && c < cols;
      const float* src = base + (size_t)kr * cols + c;
#pragma unroll
      for (int k = 0; k < NS; ++k) r[k] = ldg4_if(src + k * slice, in);
    } else {
      auto one = [&](int k, int e) {
        const int kr = k0 + (tid + NT * e) / W, c = c0 + (tid + NT * e) % W;
        return ldg_if(base + k * slice + (size_t)kr * cols + c, kr < kend && c < cols);
      };
#pragma unroll
      for (int k = 0; k < NS; ++k) r[k] = make_float4(one(k, 0), one(k, 1), one(k, 2), one(k, 3));
    }
  };
  // at: the thread's (row, col); tile: the slice's first value
  auto store = [&](float* at, float* tile, const float4& v, bool vec) {
    if (vec) {
      *reinterpret_cast<float4*>(at) = v;
    } else {
      tile[tid] = v.x; tile[tid + NT] = v.y; tile[tid + 2 * NT] = v.z; tile[tid + 3 * NT] = v.w;
    }
  };
  auto load4 = [&](const float* src, int c, int cols) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (both && c + 3 < cols) {
      v = __ldg(reinterpret_cast<const float4*>(src + c));
    } else {
      v.x = c < cols ? __ldg(src + c) : 0.f;
      v.y = c + 1 < cols ? __ldg(src + c + 1) : 0.f;
      v.z = c + 2 < cols ? __ldg(src + c + 2) : 0.f;
      v.w = c + 3 < cols ? __ldg(src + c + 3) : 0.f;
    }
    return v;
  };
  auto fetch = [&](int k0) {
    if constexpr (LD == LD_BRANCH) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        ra[k] = k0 + ar < kend ? load4(At + k * sA + (size_t)(k0 + ar) * M, i0 + ac, M)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
        rb[k] = k0 + br < kend ? load4(B + k * sB + (size_t)(k0 + br) * N, j0 + bc, N)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    } else {
      load(ra, At, sA, M, k0, i0, BM, ar, ac, va);
      load(rb, B, sB, N, k0, j0, BN, br, bc, vb);
    }
  };
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int k = 0; k < NS; ++k) store(&As[k][ar][ac], &As[k][0][0], ra[k], va);
    if (PRO) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int l = 0; l < NS; ++l) {
          const float m = f.pro[k * NS + l];
          t.x = fmaf(m, rb[l].x, t.x);
          t.y = fmaf(m, rb[l].y, t.y);
          t.z = fmaf(m, rb[l].z, t.z);
          t.w = fmaf(m, rb[l].w, t.w);
        }
        store(&Bs[k][br][bc], &Bs[k][0][0], t, vb);
      }
    } else {
#pragma unroll
      for (int l = 0; l < NS; ++l) store(&Bs[l][br][bc], &Bs[l][0][0], rb[l], vb);
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        float a[TM], b[TN];
#pragma unroll
        for (int q = 0; q < TM; q += 4) {
          const float4 av = *reinterpret_cast<const float4*>(&As[k][kk][ty * TM + q]);
          a[q] = av.x; a[q + 1] = av.y; a[q + 2] = av.z; a[q + 3] = av.w;
        }
#pragma unroll
        for (int j = 0; j < TN; ++j) b[j] = Bs[k][kk][tx * TN + j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[k][i][j] = fmaf(a[i], b[j], acc[k][i][j]);
      }
    }
    __syncthreads();
  }
}

// Where a product's tile goes: out = ca Y + cp prev at (row, col) of slice l,
// stored M x N a slice, or transposed (N x M: the K-major left operand of a
// second product; then without prev or a reduction).
struct Out {
  float* C;
  const float* prev;
  const float* other;
  bool reduce, trans;
  int M, N;
  float ca, cp;
};

template <bool EPI>  // a product's last stage (EPI) is never stored transposed
__device__ __forceinline__ void out_one(const Out& o, int l, int row, int col, float y,
                                        float& local) {
  const size_t sl = (size_t)l * o.M * o.N;
  if (!EPI && o.trans) {
    o.C[sl + (size_t)col * o.M + row] = o.ca * y;
    return;
  }
  const size_t i = sl + (size_t)row * o.N + col;
  float out = o.ca * y;
  if (o.prev) out = fmaf(o.cp, o.prev[i], out);
  o.C[i] = out;
  if (o.reduce) local = fmaf(out, o.other ? o.other[i] : out, local);
}

// The store of a whole register tile (ffma_tile.cuh): Y_l = sum_k epi[l][k]
// acc[k] (EPI), then Out. VEC: float4 along the rows of the output (or along
// its columns when transposed). local[h]: the thread's share of the reduction
// from its rows 4h .. 4h + 3 (one chain over rows, columns, slices; CHAIN: rows
// 4 .. 7 continue the first four's, both in local[0]).
template <class T, bool EPI, bool VEC, bool CHAIN>
__device__ __forceinline__ void tile_store(const Out& o, const Fused& f, int i0, int j0,
                                           ftile::Acc<T>& acc, float (&local)[2]) {
  constexpr int NS = T::NS;
  const int tx = ftile::tile_tx<T>(), ty = ftile::tile_ty<T>();
  local[0] = local[1] = 0.f;
#pragma unroll
  for (int hi = 0; hi < 2; ++hi) {
    float& loc = local[CHAIN ? 0 : hi];
    const int row = i0 + ftile::tile_row<T>(ty, hi);
#pragma unroll
    for (int hj = 0; hj < T::TN / 4; ++hj) {
      const int col = j0 + ftile::tile_col<T>(tx, hj);
      if (VEC && !EPI && o.trans) {
#pragma unroll
        for (int l = 0; l < NS; ++l)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 a = ftile::unpack2(acc[l][2 * hi][4 * hj + j]);
            const float2 b = ftile::unpack2(acc[l][2 * hi + 1][4 * hj + j]);
            if (row < o.M && col + j < o.N)  // M % 4 == 0: whole groups
              *reinterpret_cast<float4*>(o.C + ((size_t)l * o.N + col + j) * o.M + row) =
                  make_float4(o.ca * a.x, o.ca * a.y, o.ca * b.x, o.ca * b.y);
          }
        continue;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (row + i >= o.M) break;
        float y[NS][4];
#pragma unroll
        for (int l = 0; l < NS; ++l)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            auto at = [&](int k) {
              const float2 v = ftile::unpack2(acc[k][2 * hi + i / 2][4 * hj + j]);
              return (i & 1) ? v.y : v.x;
            };
            if (EPI) {
              y[l][j] = 0.f;
#pragma unroll
              for (int k = 0; k < NS; ++k) y[l][j] = fmaf(f.epi[l * NS + k], at(k), y[l][j]);
            } else {
              y[l][j] = at(l);
            }
          }
        if (VEC) {
          if (col >= o.N) break;  // N % 4 == 0: whole groups
#pragma unroll
          for (int l = 0; l < NS; ++l) {
            const size_t q = ((size_t)l * o.M + row + i) * o.N + col;
            float4 out = make_float4(o.ca * y[l][0], o.ca * y[l][1], o.ca * y[l][2], o.ca * y[l][3]);
            if (o.prev) {
              const float4 pv = *reinterpret_cast<const float4*>(o.prev + q);
              out.x = fmaf(o.cp, pv.x, out.x); out.y = fmaf(o.cp, pv.y, out.y);
              out.z = fmaf(o.cp, pv.z, out.z); out.w = fmaf(o.cp, pv.w, out.w);
            }
            *reinterpret_cast<float4*>(o.C + q) = out;
            y[l][0] = out.x; y[l][1] = out.y; y[l][2] = out.z; y[l][3] = out.w;
          }
          if (!o.reduce) continue;
          float ov[NS][4];
#pragma unroll
          for (int l = 0; l < NS; ++l) {
            float4 v = make_float4(y[l][0], y[l][1], y[l][2], y[l][3]);
            if (o.other)
              v = *reinterpret_cast<const float4*>(o.other + ((size_t)l * o.M + row + i) * o.N + col);
            ov[l][0] = v.x; ov[l][1] = v.y; ov[l][2] = v.z; ov[l][3] = v.w;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int l = 0; l < NS; ++l) loc = fmaf(y[l][j], ov[l][j], loc);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int l = 0; l < NS; ++l)
              if (col + j < o.N) out_one<EPI>(o, l, row + i, col + j, y[l][j], loc);
        }
      }
    }
  }
}

// The deterministic reduction of the fused tiles (reduce_finish_n of
// tc_device.cuh) over 64 x 64 blocks of the output whatever the tile, so its
// bits do not depend on the tile shape: a CTA of NBLK blocks (a 128 x 64 tile
// that has rows in both: 2) writes partials bid .. bid + NBLK - 1 step `stride`
// and arrives NBLK times. V = 1: a block is 128 threads, one value each (v[0]).
// V = 2: 256 virtual threads, two values a thread: the thread's rows 0..3 and
// 4..7 are virtual rows 2 ty and 2 ty + 1, so a virtual warp is one half-warp.
// The last CTA sums the partials in order as a block's (virtual) threads would.
template <class T, int V>
__device__ __forceinline__ void reduce_blocks(const float (&v)[2], const Red& red, unsigned bid,
                                              unsigned stride, int nblk_cta, unsigned nblk) {
  constexpr int NW = 4 * V;             // (virtual) warps a block
  constexpr int B = T::BM / 64;         // blocks a CTA
  __shared__ float sh_f[B * NW];
  __shared__ int sh_last;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float s = v[0];
  if (V == 2) {
    s = v[0] + v[1];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((lane & 15) == 0) sh_f[2 * w + (lane >> 4)] = s;
  } else {
    s = warp_sum_f(s);
    if (lane == 0) sh_f[w] = s;
  }
  __syncthreads();
  if (tid < 32) {
    s = lane < B * NW ? sh_f[lane] : 0.f;
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane % NW == 0 && lane / NW < nblk_cta) red.partials[bid + (lane / NW) * stride] = (double)s;
    __syncwarp();
    if (lane == 0) {
      __threadfence();  // the other lane's partial too
      unsigned t;
      asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;"
                   : "=r"(t)
                   : "l"(red.ticket), "r"((unsigned)nblk_cta)
                   : "memory");
      sh_last = (t + nblk_cta == nblk);
    }
  }
  __syncthreads();
  if (sh_last) sum_partials<V>(red, nblk);
}

__device__ __forceinline__ Out make_out(float* C, const Epi& ep, bool trans, int M, int N, float ca,
                                        float cp) {
  return Out{C, ep.prev, ep.red.other, ep.red.out != nullptr, trans, M, N, ca, cp};
}

// The summed partial tiles of a cluster whose CTAs split K: rank r finishes
// rows [r BM / KS, (r + 1) BM / KS) of the tile from every rank's P[NS][BM][BN].
template <int NS, int BM, int BN, int NT, bool EPI>
__device__ __forceinline__ float split_store(cg::cluster_group& cluster, float* P, const Out& o,
                                             const Fused& f, int i0, int j0) {
  const int KS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int rows = BM / KS;
  float local = 0.f;
  for (int idx = threadIdx.x; idx < rows * BN; idx += NT) {
    const int lr = rank * rows + idx / BN, lc = idx % BN;
    const int row = i0 + lr, col = j0 + lc;
    float v[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) v[k] = 0.f;
    for (int q = 0; q < KS; ++q) {
      const float* Pq = cluster.map_shared_rank(P, q);
#pragma unroll
      for (int k = 0; k < NS; ++k) v[k] += Pq[(k * BM + lr) * BN + lc];
    }
    if (row < o.M && col < o.N) {
#pragma unroll
      for (int l = 0; l < NS; ++l) {
        float y = v[l];
        if (EPI) {
          y = 0.f;
#pragma unroll
          for (int k = 0; k < NS; ++k) y = fmaf(f.epi[l * NS + k], v[k], y);
        }
        out_one<EPI>(o, l, row, col, y, local);
      }
    }
  }
  return local;
}

// Small fused tiles, K split over the cluster (a cluster of one: no split);
// the epilogue runs from the summed partial tiles. Read value by value (!VEC) four
// CTAs a SM are asked for: left to itself the compiler there saves the registers
// that the next K block's loads need (M x K x N x n3 130 x 800 x 200 x 1 8.5 us
// with it not asked for, 8.2 with; 512 x 800 x 330 x 3 69.5 and 61.7). With whole
// groups it costs long narrow products more than it gives others (c-LSQR of 2048 x
// 2048 with 64 columns, n3 = 4: 1446 us, asked for 1813).
template <int NS, int BM, int BN, int BK, int TM, int TN, bool PRO, bool EPI, bool VEC>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), VEC ? 0 : 4)
k_fused_small(const float* __restrict__ At, const float* __restrict__ B, float* C, int M, int N,
              int K, int kchunk, Fused f, Epi ep, int trans) {
  constexpr int TX = BN / TN;
  constexpr int NT = (BM / TM) * (BN / TN);
  if (ep.skip && *ep.skip) return;
  __shared__ __align__(16) float sm[SmallSmem<NS, BM, BN, BK>::kFloats];
  __shared__ float sh_coef[2];
  float* P = sm;  // partial tile [NS][BM][BN] after the main loop

  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  const int kbeg = (int)cluster.block_rank() * kchunk;
  const int kend = min(K, kbeg + kchunk);

  float acc[NS][TM][TN];
  small_tile_mainloop<NS, BM, BN, BK, TM, TN, PRO, VEC ? LD_WHOLE : LD_EACH>(
      At, B, M, N, K, kbeg, kend, i0, j0, f, sm, acc);
  // partial tile to shared memory, then sum over the cluster's K ranges
#pragma unroll
  for (int k = 0; k < NS; ++k)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) P[(k * BM + ty * TM + i) * BN + tx * TN + j] = acc[k][i][j];
  coef_compute(ep.coef, sh_coef);
  cluster.sync();
  const Out o = make_out(C, ep, trans, M, N, sh_coef[0], sh_coef[1]);
  const float local = split_store<NS, BM, BN, NT, EPI>(cluster, P, o, f, i0, j0);
  cluster.sync();  // peers may still read this CTA's partial tile until here
  if (ep.red.out) reduce_finish(local, ep.red);
}

// Fused 64 x 64 tiles of ffma_tile.cuh: one tile a CTA, all NS slices. SPLIT: K
// split over the cluster (products without a reduction). At NS = 3 the 4-byte-copy
// forms spill 40 to 108 bytes a thread under the three CTAs a SM that hide the
// copies' latency.
template <class T, bool PRO, bool EPI, bool SPLIT, bool VEC>
__global__ void __launch_bounds__(T::NT, T::NS == 4 ? 2 : 3)
k_fused_gemm(const float* __restrict__ At, const float* __restrict__ B, float* C, int M, int N,
             int K, int kchunk, Fused f, Epi ep, int trans) {
  if (ep.skip && *ep.skip) return;
  extern __shared__ __align__(16) float dyn[];
  __shared__ float sh_coef[2];
  const int i0 = blockIdx.y * T::BM, j0 = blockIdx.x * T::BN;
  ftile::Acc<T> acc;
  if (!SPLIT) {
    ftile::mainloop<T, PRO, VEC>(At, B, M, N, K, 0, K, i0, j0, f.pro, dyn, acc);
    coef_compute(ep.coef, sh_coef);
    __syncthreads();
    const Out o = make_out(C, ep, trans, M, N, sh_coef[0], sh_coef[1]);
    float local[2];
    tile_store<T, EPI, VEC, false>(o, f, i0, j0, acc, local);
    if (ep.red.out)
      reduce_blocks<T, 2>(local, ep.red, blockIdx.y * gridDim.x + blockIdx.x, 0, 1,
                          gridDim.x * gridDim.y);
    return;
  }
  cg::cluster_group cluster = cg::this_cluster();
  const int kbeg = (int)cluster.block_rank() * kchunk;
  ftile::mainloop<T, PRO, VEC>(At, B, M, N, K, kbeg, min(K, kbeg + kchunk), i0, j0, f.pro, dyn, acc);
  __syncthreads();  // every warp is done with the ring: it holds the partial tile now
  const int tx = ftile::tile_tx<T>(), ty = ftile::tile_ty<T>();
#pragma unroll
  for (int k = 0; k < T::NS; ++k)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ftile::tile_row<T>(ty, i / 2) + 2 * (i & 1), c = ftile::tile_col<T>(tx, 0);
      float2 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = ftile::unpack2(acc[k][i][j]);
      float* q = dyn + (k * T::BM + r) * T::BN + c;
      *reinterpret_cast<float4*>(q) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
      *reinterpret_cast<float4*>(q + T::BN) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
    }
  coef_compute(ep.coef, sh_coef);
  cluster.sync();
  const Out o = make_out(C, ep, trans, M, N, sh_coef[0], sh_coef[1]);
  split_store<T::NS, T::BM, T::BN, T::NT, EPI>(cluster, dyn, o, f, i0, j0);
  cluster.sync();  // peers may still read this CTA's partial tile until here
}

// Per-slice GEMM without transforms: C_z = A_z B_z (or its transpose) for
// slice z = blockIdx.z, At: K x M.
template <class T, bool VEC>
__global__ void __launch_bounds__(T::NT, T::TN == 8 ? 4 : 256 / T::NT * 2)
k_slice_gemm(const float* __restrict__ At, const float* __restrict__ B, float* C, int M, int N,
             int K, int trans, const int* skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) float dyn[];
  const size_t z = blockIdx.z;
  const int i0 = blockIdx.y * T::BM, j0 = blockIdx.x * T::BN;
  ftile::Acc<T> acc;
  const Fused f{};
  ftile::mainloop<T, false, VEC>(At + z * K * M, B + z * K * N, M, N, K, 0, K, i0, j0, f.pro, dyn,
                                 acc);
  const Out o{C + z * M * N, nullptr, nullptr, false, trans != 0, M, N, 1.f, 0.f};
  float local[2];
  tile_store<T, false, VEC, false>(o, f, i0, j0, acc, local);
}

// Grouped fused products: CTA i takes tile work[i].y of problem work[i].x,
// reads that problem's operands, epilogue scalars and done flag (g.op, g.j),
// and reduces into that problem's partials with its tile index, so each
// problem keeps its own deterministic reduction. The pointers follow the
// deferred-iterate schedule of lsqr_enqueue: the forward product of step j
// reads basis slot j and writes U (prev: C at j = 0, else U), the adjoint
// reads U and writes basis slot j + 1 (prev: slot j), the first adjoint
// writes slot 0 from C.
template <class T>
__global__ void __launch_bounds__(T::NT, T::NT == 256 ? 1 : (T::NS == 4 ? 2 : 3))
k_group_gemm(const GroupProb* __restrict__ probs, const int2* __restrict__ work, GroupOp g,
             Fused f) {
  const int2 w = work[blockIdx.x];
  const GroupProb& P = probs[w.x];
  if (g.op != GOP_INIT && g.done[(size_t)w.x * g.lstride + g.j]) return;  // uniform over the problem's CTAs
  extern __shared__ __align__(16) float dyn[];
  __shared__ float sh_coef[2];
  const GroupOperands o = group_operands(P, g, w.x);
  const bool fwd = o.fwd;
  const int M = o.M, K = o.K, N = o.N;
  const float* At = fwd ? P.AhT : P.Ah;  // K-major
  const int tn = (N + T::BN - 1) / T::BN;
  const int i0 = (w.y / tn) * T::BM, j0 = (w.y % tn) * T::BN;
  const bool vec = (M | N) % 4 == 0 &&  // uniform over the problem's CTAs
                   ((reinterpret_cast<uintptr_t>(At) | reinterpret_cast<uintptr_t>(o.B) |
                     reinterpret_cast<uintptr_t>(o.C) | reinterpret_cast<uintptr_t>(o.prev)) & 15) == 0;
  ftile::Acc<T> acc;
  float local[2];
  auto tile = [&](auto vt) {
    constexpr bool VEC = decltype(vt)::value;
    ftile::mainloop<T, true, VEC>(At, o.B, M, N, K, 0, K, i0, j0, f.pro, dyn, acc);
    coef_compute(o.coef, sh_coef);
    __syncthreads();
    const Out out{o.C, o.prev, nullptr, true, false, M, N, sh_coef[0], sh_coef[1]};
    tile_store<T, true, VEC, true>(out, f, i0, j0, acc, local);
  };
  if (vec) tile(std::true_type{});
  else tile(std::false_type{});
  constexpr int B = T::BM / 64;
  const int nb = B == 2 && i0 + 64 < M ? 2 : 1;
  reduce_blocks<T, 1>(local, o.red, (unsigned)(B * (w.y / tn) * tn + w.y % tn), (unsigned)tn, nb,
                      (unsigned)((M + 63) / 64 * tn));
}

// The same with 32 x 32 tiles (small_tile_mainloop), stored from the registers:
// batches whose 64 x 64 tiles are too few for the SMs (30 problems of n in
// 64..128: 336 us a solve of 6 steps against 360 with 64 x 64 tiles).
template <int NS>
__global__ void __launch_bounds__(128)
k_group_small(const GroupProb* __restrict__ probs, const int2* __restrict__ work, GroupOp g,
              Fused f) {
  constexpr int BM = 32, BN = 32, BK = 16, TM = 4, TN = 2;
  const int2 w = work[blockIdx.x];
  const GroupProb& P = probs[w.x];
  if (g.op != GOP_INIT && g.done[(size_t)w.x * g.lstride + g.j]) return;  // uniform over the problem's CTAs
  __shared__ __align__(16) float sm[SmallSmem<NS, BM, BN, BK>::kMain];
  __shared__ float sh_coef[2];
  const GroupOperands o = group_operands(P, g, w.x);
  const int M = o.M, K = o.K, N = o.N;
  const int tn = (N + BN - 1) / BN;
  const int i0 = (w.y / tn) * BM, j0 = (w.y % tn) * BN;
  float acc[NS][TM][TN];
  small_tile_mainloop<NS, BM, BN, BK, TM, TN, true, LD_BRANCH>(o.fwd ? P.AhT : P.Ah, o.B, M, N, K, 0,
                                                               K, i0, j0, f, sm, acc);
  coef_compute(o.coef, sh_coef);
  __syncthreads();
  const Out out{o.C, o.prev, nullptr, true, false, M, N, sh_coef[0], sh_coef[1]};
  const int tx = threadIdx.x % (BN / TN), ty = threadIdx.x / (BN / TN);
  float local = 0.f;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int row = i0 + ty * TM + i, col = j0 + tx * TN + j;
      if (row >= M || col >= N) continue;
#pragma unroll
      for (int l = 0; l < NS; ++l) {
        float y = 0.f;
#pragma unroll
        for (int k = 0; k < NS; ++k) y = fmaf(f.epi[l * NS + k], acc[k][i][j], y);
        out_one<true>(out, l, row, col, y, local);
      }
    }
  reduce_finish_n(local, o.red, (unsigned)w.y, (unsigned)((M + BM - 1) / BM * tn));
}

// Tile shapes the autotuner chooses from: cfg 0: 64 x 64 (128 threads), 1: 32 x 32
// (k_group_small), 2: 128 x 64 (256 threads). 0 and 2 give the same bits.
template <int NS, int CFG>
using GroupTile = ftile::Tile<NS, CFG == 2 ? 128 : 64, 64, 16, 4, 3, true>;

template <class K>
int allow_smem(K kernel, size_t bytes) {
  TC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  TC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  return TC_OK;
}

template <int NS, int CFG>
int run_group(const GroupProb* probs, const int2* work, int nwork, const GroupOp& g,
              const Fused& f, cudaStream_t st) {
  if constexpr (CFG == 1) {
    k_group_small<NS><<<nwork, 128, 0, st>>>(probs, work, g, f);
  } else {
    using T = GroupTile<NS, CFG>;
    k_group_gemm<T><<<nwork, T::NT, T::bytes, st>>>(probs, work, g, f);
  }
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Whole 16-byte groups in every operand of a product.
bool vec_ok(const float* At, const float* B, const float* C, int M, int N, const Epi& ep) {
  return M % 4 == 0 && N % 4 == 0 && al16(At) && al16(B) && al16(C) &&
         (!ep.prev || al16(ep.prev)) && (!ep.red.other || al16(ep.red.other));
}

template <class Kern>
int launch_cluster(Kern kernel, int BM, int BN, int NT, size_t smem, int KS, const float* At,
                   const float* B, float* C, int M, int N, int K, int kchunk, const Fused& f,
                   const Epi& ep, int trans, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((N + BN - 1) / BN, (M + BM - 1) / BM, KS);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = KS;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  TC_CUDA(cudaLaunchKernelEx(&cfg, kernel, At, B, C, M, N, K, kchunk, f, ep, trans));
  return TC_OK;
}

template <class T, bool PRO, bool EPI, bool SPLIT>
int run_fused(const float* At, const float* B, float* C, int M, int N, int K, int KS,
              const Fused& f, const Epi& ep, int trans, cudaStream_t st) {
  TC_CHECK(!SPLIT || ep.red.out == nullptr);  // the split form stores without a reduction
  const int kchunk = (((K + KS - 1) / KS) + T::BK - 1) / T::BK * T::BK;
  if (vec_ok(At, B, C, M, N, ep))
    return launch_cluster(k_fused_gemm<T, PRO, EPI, SPLIT, true>, T::BM, T::BN, T::NT, T::bytes, KS,
                          At, B, C, M, N, K, kchunk, f, ep, trans, st);
  return launch_cluster(k_fused_gemm<T, PRO, EPI, SPLIT, false>, T::BM, T::BN, T::NT, T::bytes, KS,
                        At, B, C, M, N, K, kchunk, f, ep, trans, st);
}

template <int NS>
using TileM = ftile::Tile<NS, 64, 64, 16, 4, 3, true>;

// Which fused form serves an M x N x K product: the one whose busiest SM is
// estimated to be done first. Unit: a 32 x 32 tile's K block (16 of K). Small
// tiles take rounds x blocks (rounds = ceil(tiles KS / SMs); K split while the grid
// does not cover the SMs and each rank keeps two blocks), and 2 more when split. A
// 64 x 64 tile's block is 2 units (four times the FMAs, half the shared-memory
// reads an FMA), its split over 2 or 4 ranks 12 more and over 8 16 (the partial
// tiles go through distributed shared memory); each rank keeps at least four
// blocks. On ties the smaller tile, then four ranks.
// Measured, us a launch, M x K x N x n3: 32 x 32 (their best split) / 64 x 64
// whole / split over 4 / over 8, the rule's choice in brackets:
//   330 x 64 x 200 x 3:  [8.2] / 14.4 / - / -      512 x 64 x 512 x 3:  [10.9] / 10.3 / - / -
//   256 x 200 x 256 x 3: [10.3] / 21.5 / 14.4 / -  400 x 384 x 400 x 3: 34.8 / 38.8 / [24.6] / 20.5
//   2048 x 512 x 40 x 3: 24.6 / 47.1 / [18.5] / 18.5
//   512^3 x 3:           43.0 / 47.2 / [28.7] / 34.8
//   1344 x 384 x 1344 x 3: 152 / [90.1] / 104 / 129
// Over 8603 shapes (1..9800 x 20..1344 x 1..9800, n3 = 1..4) the choice is 3% off the
// best form in the geometric mean; the rule by tile counts alone that it replaced
// was 10% off, and slower than the 32 x 32 tiles on one shape in ten (330 x 64 x
// 200 x 3: 14.4 us).
// A solver's products (ep.red, or `solve` for the first of a two-sided pair) take
// whole 64 x 64 tiles from 152 of them on, else small tiles: the split 64 x 64 form
// has no reduction, and the orders of addition that solves have at each size are
// held where they are.
template <int NS, bool PRO, bool EPI>
int pick_tile(const float* At, const float* B, float* C, int M, int N, int K, const Fused& f,
              const Epi& ep, int trans, bool solve, cudaStream_t st) {
  constexpr int BK = 16;
  auto up = [](long x, long y) { return (x + y - 1) / y; };
  const long t64 = up(M, 64) * up(N, 64), t32 = up(M, 32) * up(N, 32);
  int KS = 1;
  while (KS < 8 && t32 * KS < NSM && K >= 2 * BK * (KS * 2)) KS *= 2;
  int K64 = 0;  // the 64 x 64 tiles' split; 0: small tiles
  if (solve || ep.red.out) {
    K64 = t64 >= NSM;
  } else {
    long best = up(t32 * KS, NSM) * up(up(K, KS), BK) + (KS > 1 ? 2 : 0);
    for (int ks : {4, 8, 2, 1}) {
      if (ks > 1 && K < 4 * BK * ks) continue;
      const long c = 2 * up(t64 * ks, NSM) * up(up(K, ks), BK) + (ks == 1 ? 0 : ks == 8 ? 16 : 12);
      if (c < best) {
        best = c;
        K64 = ks;
      }
    }
  }
  if (K64 == 1) return run_fused<TileM<NS>, PRO, EPI, false>(At, B, C, M, N, K, 1, f, ep, trans, st);
  if (K64 > 1) return run_fused<TileM<NS>, PRO, EPI, true>(At, B, C, M, N, K, K64, f, ep, trans, st);
  const int kchunk = (((K + KS - 1) / KS) + BK - 1) / BK * BK;
  const bool vec = (M | N) % 4 == 0 && al16(At) && al16(B);
  return vec ? launch_cluster(k_fused_small<NS, 32, 32, BK, 4, 2, PRO, EPI, true>, 32, 32, 128, 0, KS,
                              At, B, C, M, N, K, kchunk, f, ep, trans, st)
             : launch_cluster(k_fused_small<NS, 32, 32, BK, 4, 2, PRO, EPI, false>, 32, 32, 128, 0, KS,
                              At, B, C, M, N, K, kchunk, f, ep, trans, st);
}

template <int NS>
int pick_flags(bool pro, bool epi, const float* At, const float* B, float* C, int M, int N,
               int K, const Fused& f, const Epi& ep, int trans, bool solve, cudaStream_t st) {
  if (pro && epi) return pick_tile<NS, true, true>(At, B, C, M, N, K, f, ep, trans, solve, st);
  if (pro) return pick_tile<NS, true, false>(At, B, C, M, N, K, f, ep, trans, solve, st);
  return pick_tile<NS, false, true>(At, B, C, M, N, K, f, ep, trans, solve, st);
}

template <class T>
int run_slice(const float* At, const float* B, float* C, int M, int N, int K, int nslices,
              int trans, const Epi& ep, cudaStream_t st) {
  const dim3 grid((N + T::BN - 1) / T::BN, (M + T::BM - 1) / T::BM, nslices);
  if (vec_ok(At, B, C, M, N, ep))
    k_slice_gemm<T, true><<<grid, T::NT, T::bytes, st>>>(At, B, C, M, N, K, trans, ep.skip);
  else
    k_slice_gemm<T, false><<<grid, T::NT, T::bytes, st>>>(At, B, C, M, N, K, trans, ep.skip);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

using SliceL = ftile::Tile<1, 128, 64, 32, 8, 2, false>;
using SliceM = ftile::Tile<1, 64, 64, 32, 4, 3, false>;
using SliceS = ftile::Tile<1, 64, 32, 32, 4, 3, false>;

template <class T>
int init_slice() {
  TC_TRY(allow_smem(k_slice_gemm<T, true>, T::bytes));
  return allow_smem(k_slice_gemm<T, false>, T::bytes);
}

template <class T, bool PRO, bool EPI, bool SPLIT>
int init_fused() {
  TC_TRY(allow_smem(k_fused_gemm<T, PRO, EPI, SPLIT, true>, T::bytes));
  return allow_smem(k_fused_gemm<T, PRO, EPI, SPLIT, false>, T::bytes);
}

template <int NS>
int init_ns() {
  TC_TRY((init_fused<TileM<NS>, true, true, false>()));
  TC_TRY((init_fused<TileM<NS>, true, false, false>()));
  TC_TRY((init_fused<TileM<NS>, false, true, false>()));
  TC_TRY((init_fused<TileM<NS>, true, true, true>()));
  TC_TRY((init_fused<TileM<NS>, true, false, true>()));
  TC_TRY((init_fused<TileM<NS>, false, true, true>()));
  TC_TRY(allow_smem(k_group_gemm<GroupTile<NS, 0>>, GroupTile<NS, 0>::bytes));
  return allow_smem(k_group_gemm<GroupTile<NS, 2>>, GroupTile<NS, 2>::bytes);
}

}  // namespace

int group_cfg_count(int bf16) { return bf16 ? 2 : 3; }

void group_tile_shape(int bf16, int cfg, int* tm, int* tn) {
  if (bf16) {  // group_tc.cu: 128 x 64 or 128 x 128
    *tm = 128;
    *tn = cfg == 1 ? 128 : 64;
  } else {
    *tm = cfg == 2 ? 128 : (cfg == 1 ? 32 : 64);
    *tn = cfg == 1 ? 32 : 64;
  }
}

int launch_group_gemm(const GroupProb* probs, const int2* work, int nwork, const GroupOp& g,
                      const float* pro, const float* epi, int n3, int cfg, cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_FUSED && nwork >= 1 && cfg >= 0 && cfg < GROUP_CFGS);
  Fused f{};
  for (int i = 0; i < n3 * n3; ++i) {
    f.pro[i] = pro[i];
    f.epi[i] = epi[i];
  }
  auto go = [&](auto ns) -> int {
    constexpr int NS = decltype(ns)::value;
    return cfg == 0 ? run_group<NS, 0>(probs, work, nwork, g, f, st)
         : cfg == 1 ? run_group<NS, 1>(probs, work, nwork, g, f, st)
                    : run_group<NS, 2>(probs, work, nwork, g, f, st);
  };
  switch (n3) {
    case 1: return go(std::integral_constant<int, 1>{});
    case 2: return go(std::integral_constant<int, 2>{});
    case 3: return go(std::integral_constant<int, 3>{});
    default: return go(std::integral_constant<int, 4>{});
  }
}

int gemm_init() {
  TC_TRY(init_ns<1>());
  TC_TRY(init_ns<2>());
  TC_TRY(init_ns<3>());
  TC_TRY(init_ns<4>());
  TC_TRY(init_slice<SliceL>());
  TC_TRY(init_slice<SliceM>());
  return init_slice<SliceS>();
}

int launch_slice_gemm(const float* At, const float* B, float* C, int M, int N, int K,
                      int nslices, const float* pro, const float* epi, const Epi& ep,
                      cudaStream_t st, bool trans, bool solve) {
  // a transposed result is an intermediate: plain values, no Krylov epilogue
  TC_CHECK(!trans || (ep.prev == nullptr && ep.red.out == nullptr));
  if (pro || epi) {
    TC_CHECK(nslices <= TC_MAX_FUSED);
    Fused f{};
    for (int i = 0; i < nslices * nslices; ++i) {
      f.pro[i] = pro ? pro[i] : 0.f;
      f.epi[i] = epi ? epi[i] : 0.f;
    }
    switch (nslices) {
      case 1: return pick_flags<1>(pro, epi, At, B, C, M, N, K, f, ep, trans, solve, st);
      case 2: return pick_flags<2>(pro, epi, At, B, C, M, N, K, f, ep, trans, solve, st);
      case 3: return pick_flags<3>(pro, epi, At, B, C, M, N, K, f, ep, trans, solve, st);
      case 4: return pick_flags<4>(pro, epi, At, B, C, M, N, K, f, ep, trans, solve, st);
      default: return TC_EINVAL;
    }
  }
  // per-slice GEMM between transform passes: no epilogue beyond the store
  TC_CHECK(ep.prev == nullptr && ep.red.out == nullptr && ep.coef.rule == COEF_ONE);
  // Tile: the one whose busiest SM has the least to do (in units of a 64 x 64
  // tile). On ties the larger tile, which reads less shared memory an FMA
  // (128 x 64 from four units on: it needs several CTAs a SM). Measured, us
  // (128 x 64 / 64 x 64 / 64 x 32): 256^3 x 9 14.4 / 8.4 / 10.3; 512^3 x 32
  // 139 / 144 / 156; 512^3 x 64 274 / 272 / 295; 768^3 x 5 92 / 80 / 86;
  // 389 x 257 x 301 x 9 (4-byte copies) 37 / 33 / 27. Not the fastest where the
  // 64 x 32 tiles save only half a unit: at 512^3 x 32 it takes them (13.5 units
  // against 14), 12% off the best.
  auto units = [&](int bm, int bn) {
    const long t = (long)((M + bm - 1) / bm) * ((N + bn - 1) / bn) * nslices;
    return (double)((t + NSM - 1) / NSM) * bm * bn / 4096.0;
  };
  const double ul = units(128, 64), um = units(64, 64), us = units(64, 32);
  if (ul >= 4.0 && ul <= um && ul <= us)
    return run_slice<SliceL>(At, B, C, M, N, K, nslices, trans, ep, st);
  if (um <= us) return run_slice<SliceM>(At, B, C, M, N, K, nslices, trans, ep, st);
  return run_slice<SliceS>(At, B, C, M, N, K, nslices, trans, ep, st);
}

// The grouped products of the batched BF16 c-LSQR (group.cu) on the tensor
// cores: one launch runs every (problem, tile) pair of one product of one
// step, each CTA one 128 x BN output tile of its problem over all n3 <= 4
// slices.
//
// Bound: HBM (A~ and the operand in BF16, prev, the result and the next operand;
// 78 us for the batch of 128 problems of n in 64..512 at the copy rate). The
// operand arrives transformed and in BF16: each product's epilogue, which has all
// slices of a pixel in registers, also writes bf16(result x_3 T) for the product
// that follows (T = M^{-T} after the forward product, M after the adjoint; FP32
// transform of the FP32 result, one rounding: the values a separate pass would
// give), and a small launch does so for C. So the main loop is a plain TMA ring:
//   warp 0, one lane: TMA loads (per-problem maps in a device table) of one
//     slice's K block of 64 a stage, A~ 128 x 64 K-major and the operand 64 x BN
//     MN-major, 128-byte swizzle, zeros past the edges;
//   warp 1, one lane: tcgen05.mma (kind::f16, FP32 accumulators in tensor
//     memory, n3 x BN columns); its commits free the stages;
//   warps 2..5: the epilogue. Each 32-row x 16-column chunk of prev goes global
//     memory (8 rows x 64 bytes an instruction) -> shared memory -> the thread that
//     owns the row, which applies the trailing transform and the Krylov epilogue
//     of group_operands (ca acc + cp prev and the norm partial of the problem's
//     two-level reduction) and puts the result back the same way.
// Two CTAs a SM (BN = 64) run one's epilogue beside the other's main loop. (With
// four slices the epilogue then spills 136 bytes a thread.)
// Before, each CTA read the FP32 operand (twice the bytes, once a row tile),
// transformed and rounded it in registers between K blocks, with one K block in
// flight and rows of 16 bytes a lane in the epilogue: 226 us a launch at BN = 64;
// now 167 us (batch of 128). Of a tile's 24.5 us, 6 are its set-up (work table,
// scalars, barriers; the other CTA of the SM runs on), 6.6 more pass until its
// accumulators are complete and 10 are the epilogue. One persistent CTA a SM with
// two accumulator buffers and two epilogue groups measured 163 us, 3% for a far
// more involved schedule, and was not kept; prev prefetched into L2 changed nothing.
// Every wait is bounded; a CTA whose wait gives up records TC_ETIMEOUT in its
// problem's status, waits (bounded) for the copies and MMAs it issued, joins the
// reduction (with nothing added) and frees its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "group.cuh"
#include "tcgen05.cuh"

namespace {

using namespace tc5;

constexpr int GT_BM = 128, GT_BK = 64, GT_NT = 192;
constexpr uint32_t GT_A = GT_BM * GT_BK * 2;  // a stage's A block: 16 KB
constexpr uint32_t GT_ATOM = GT_BK * 128;     // one 64-column atom of its B block: 8 KB

struct GroupXf {  // n3 x n3 row-major: the trailing transform, the next product's leading one
  float epi[TC_MAX_FUSED * TC_MAX_FUSED];
  float nxt[TC_MAX_FUSED * TC_MAX_FUSED];
};

template <int NS, int BN>
struct GtCfg {
  static constexpr uint32_t B_BYTES = GT_BK * BN * 2;
  static constexpr uint32_t STAGE = GT_A + B_BYTES;
  // two CTAs of at most 256 tensor-memory columns a SM for BN = 64 (stages and
  // epilogue buffers of 97 KB), one for BN = 128
  static constexpr int NST = BN == 64 ? 3 : 5;
  static constexpr uint32_t COLS = NS * BN <= 64 ? 64 : NS * BN <= 128 ? 128 : NS * BN <= 256 ? 256 : 512;
  static constexpr uint32_t EBUF = NS * 32 * 16 * 4;  // a warp's chunk, every slice
  static constexpr size_t USED = 1024 + NST * STAGE + 4 * EBUF + (2 * NST + 2) * 8 + 16;
  static constexpr size_t FLOOR = BN == 64 ? 80 * 1024 : 116 * 1024;
  static constexpr size_t SMEM = USED > FLOOR ? USED : FLOOR;
  static_assert(SMEM <= (BN == 64 ? 113 : 227) * 1024, "CTAs a SM");
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void fence_tensormap(const CUtensorMap* m) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(m) : "memory");
}

template <int NS, int BN>
__global__ void __launch_bounds__(GT_NT, BN == 64 ? 2 : 1)
k_group_umma(const GroupProb* __restrict__ probs, const CUtensorMap* maps,
             const int2* __restrict__ work, GroupOp g, GroupXf f) {
  using Cfg = GtCfg<NS, BN>;
  constexpr int NB = BN / 64, NST = Cfg::NST;
  // D F32, A and B BF16, A K-major, B MN-major, N = BN, M = 128
  constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (0u << 15) | (1u << 16) |
                             ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(GT_BM >> 4) << 24);
  const int2 wk = work[blockIdx.x];
  const GroupProb& P = probs[wk.x];
  if (g.op != GOP_INIT && g.done[(size_t)wk.x * g.lstride + g.j]) return;  // uniform over the problem's CTAs
  const GroupOperands o = group_operands(P, g, wk.x);
  const int M = o.M, N = o.N, K = o.K;
  const int tn = (N + BN - 1) / BN;
  const int m0 = (wk.y / tn) * GT_BM, n0 = (wk.y % tn) * BN;
  const CUtensorMap* tmA = maps + 4 * (size_t)wk.x + (o.fwd ? 0 : 2);
  const CUtensorMap* tmB = tmA + 1;
  // the next product's operand: the adjoint's after the forward product, the
  // next step's forward product's after the adjoint
  __nv_bfloat16* nxt = static_cast<__nv_bfloat16*>(o.fwd ? P.opU : P.opV);
  if (g.op == GOP_ADJ && g.j + 1 >= g.itermax) nxt = nullptr;

  extern __shared__ uint8_t gt_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(gt_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* ebuf = base + NST * Cfg::STAGE;  // stage s at base + s STAGE: A, then B
  uint64_t* full = reinterpret_cast<uint64_t*>(ebuf + 4 * Cfg::EBUF);
  uint64_t* empty = full + NST;
  uint64_t* accf = empty + NST;  // every MMA of the tile has completed
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accf + 1);
  __shared__ float sh_coef[2], sh_f[4 * NB];
  __shared__ int sh_fail, sh_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nk = (K + GT_BK - 1) / GT_BK;

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tslot)),
                 "r"(Cfg::COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(accf, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sh_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  volatile int* vfail = &sh_fail;
  int issued = 0;  // producer: stages armed (for the bounded drain on failure)

  if (warp == 0) {
    if (lane == 0) {
      fence_tensormap(tmA);
      fence_tensormap(tmB);
      int gi = 0;
      for (int kb = 0; kb < nk && !*vfail; ++kb)
        for (int l = 0; l < NS && !*vfail; ++l, ++gi) {
          const int s = gi % NST;
          if (!mbar_wait(empty + s, ((gi / NST) & 1) ^ 1)) {
            *vfail = 1;
            break;
          }
          uint8_t* st = base + s * Cfg::STAGE;
          mbar_expect_tx(full + s, Cfg::STAGE);
          tma_load_3d(st, tmA, kb * GT_BK, m0, l, full + s);
#pragma unroll
          for (int b = 0; b < NB; ++b)
            tma_load_3d(st + GT_A + b * GT_ATOM, tmB, n0 + 64 * b, kb * GT_BK, l, full + s);
          issued = gi + 1;
        }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int gi = 0;
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb)
        for (int l = 0; l < NS; ++l, ++gi) {
          const int s = gi % NST;
          if (!mbar_wait(full + s, (gi / NST) & 1)) {
            *vfail = 1;
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = su32(base + s * Cfg::STAGE), b0 = a0 + GT_A;
#pragma unroll
          for (int kk = 0; kk < GT_BK / 16; ++kk)
            umma<0>(tmem + (uint32_t)(l * BN), smem_desc(a0 + kk * 32, 16, 1024),
                    smem_desc(b0 + kk * 16 * 128, GT_ATOM, 1024), IDESC, (kb | kk) != 0);
          umma_commit(empty + s);
        }
      umma_commit(accf);  // completes once every MMA issued above has
    }
  } else {
    if (warp == 2) coef_compute_by(o.coef, sh_coef, 64);  // thread 64, while the main loop runs
    asm volatile("bar.sync 1, 128;" ::: "memory");        // the epilogue warps
    const float ca = sh_coef[0], cp = sh_coef[1];
    const int eq = warp & 3;  // tensor-memory lanes 32 eq .. + 31
    float4* sw = reinterpret_cast<float4*>(ebuf + eq * Cfg::EBUF);  // [slice][row][4]
    const size_t sC_el = (size_t)M * N;
    const int r0 = m0 + 32 * eq, rsub = lane >> 2, jq = lane & 3;
    const bool live = r0 + lane < M;
    const uint32_t trow = tmem + ((uint32_t)(32 * eq) << 16);
    // float4 slot of (row r, quad q): conflict-free by rows and by quads
    auto slot = [](int r, int q) { return r * 4 + (q ^ ((r >> 1) & 3)); };
    float4 pre[NS][4];  // prev of the next chunk: rows 8 i + rsub, columns 4 jq .. + 3
    auto load_prev = [&](int c0) {
      const int col = n0 + c0 + 4 * jq;
#pragma unroll
      for (int l = 0; l < NS; ++l)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = r0 + 8 * i + rsub;
          pre[l][i] = row < M && col < N
                          ? *reinterpret_cast<const float4*>(o.prev + l * sC_el + (size_t)row * N + col)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float local[NB];  // the row's sum over each 64-column block
#pragma unroll
    for (int b = 0; b < NB; ++b) local[b] = 0.f;
    if (o.prev) load_prev(0);
    const bool ok = mbar_wait(accf, 0) && !*vfail;
    if (!ok) *vfail = 1;
    if (__all_sync(0xffffffffu, ok)) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
      for (int c0 = 0; c0 < BN; c0 += 16) {
        if (n0 + c0 >= N) break;
        uint32_t v[NS][16];
#pragma unroll
        for (int l = 0; l < NS; ++l) tmem_ld16_issue(trow + (uint32_t)(l * BN + c0), v[l]);
        if (o.prev) {
#pragma unroll
          for (int l = 0; l < NS; ++l)
#pragma unroll
            for (int i = 0; i < 4; ++i) sw[l * 128 + slot(8 * i + rsub, jq)] = pre[l][i];
          if (c0 + 16 < BN) load_prev(c0 + 16);
        }
        __syncwarp();
#pragma unroll
        for (int l = 0; l < NS; ++l) tmem_ld16_wait(v[l]);
        const int col = n0 + c0;
        float sum = NB == 1 || c0 < 64 ? local[0] : local[NB - 1];
        uint2 nx[NS][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float y[NS][4];
#pragma unroll
          for (int k = 0; k < NS; ++k) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float t = 0.f;
#pragma unroll
              for (int l = 0; l < NS; ++l)
                t = fmaf(f.epi[k * NS + l], __uint_as_float(v[l][4 * q + e]), t);
              y[k][e] = ca * t;
            }
            float4& p = sw[k * 128 + slot(lane, q)];
            if (o.prev) {
              const float4 pv = p;
              y[k][0] = fmaf(cp, pv.x, y[k][0]);
              y[k][1] = fmaf(cp, pv.y, y[k][1]);
              y[k][2] = fmaf(cp, pv.z, y[k][2]);
              y[k][3] = fmaf(cp, pv.w, y[k][3]);
            }
            p = make_float4(y[k][0], y[k][1], y[k][2], y[k][3]);
            if (live && col + 4 * q < N)
              sum = fmaf(y[k][0], y[k][0],
                         fmaf(y[k][1], y[k][1], fmaf(y[k][2], y[k][2], fmaf(y[k][3], y[k][3], sum))));
          }
          if (nxt) {
#pragma unroll
            for (int k = 0; k < NS; ++k) {
              float t[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                t[e] = 0.f;
#pragma unroll
                for (int l = 0; l < NS; ++l) t[e] = fmaf(f.nxt[k * NS + l], y[l][e], t[e]);
              }
              nx[k][q] = make_uint2(pack_bf16(t[0], t[1]), pack_bf16(t[2], t[3]));
            }
          }
        }
        if (NB == 1 || c0 < 64) local[0] = sum;
        else local[NB - 1] = sum;
        __syncwarp();
#pragma unroll
        for (int l = 0; l < NS; ++l)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int row = r0 + 8 * i + rsub, cc = col + 4 * jq;
            if (row < M && cc < N)
              *reinterpret_cast<float4*>(o.C + l * sC_el + (size_t)row * N + cc) =
                  sw[l * 128 + slot(8 * i + rsub, jq)];
          }
        __syncwarp();
        if (nxt) {  // 32 bytes a row and slice: [slice][row][2] of 16 bytes
          uint4* sn = reinterpret_cast<uint4*>(sw);
#pragma unroll
          for (int l = 0; l < NS; ++l) {
            sn[l * 64 + 2 * lane] = make_uint4(nx[l][0].x, nx[l][0].y, nx[l][1].x, nx[l][1].y);
            sn[l * 64 + 2 * lane + 1] = make_uint4(nx[l][2].x, nx[l][2].y, nx[l][3].x, nx[l][3].y);
          }
          __syncwarp();
#pragma unroll
          for (int l = 0; l < NS; ++l)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int r = 16 * i + (lane >> 1), row = r0 + r, cc = col + 8 * (lane & 1);
              if (row < M && cc < N)  // N % 8 == 0: whole groups
                *reinterpret_cast<uint4*>(nxt + l * sC_el + (size_t)row * N + cc) =
                    sn[l * 64 + 2 * r + (lane & 1)];
            }
          __syncwarp();  // the next chunk overwrites the buffer
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const float s = warp_sum_f(local[b]);
      if (lane == 0) sh_f[4 * b + eq] = s;
    }
  }

  // wind down: every thread of the CTA
  __syncthreads();
  const bool failed = *vfail != 0;
  if (failed && warp == 1 && lane == 0) mbar_wait(accf, 0);  // the MMAs have finished with TMEM
  if (failed && warp == 0 && lane == 0) {                    // let the copies this CTA issued land
    for (int gi = (issued > NST ? issued - NST : 0); gi < issued; ++gi)
      mbar_wait(full + gi % NST, (gi / NST) & 1);
    atomicExch(o.red.status, TC_ETIMEOUT);
  }
  // the reduction of reduce_finish_n over 128 x 64 blocks of the output whatever
  // the tile (a block is 128 threads, one a row), so that its bits do not depend on
  // the tile shape: a tile with columns in two blocks writes two partials and
  // arrives twice
  const int tn64 = (N + 63) / 64, nblk = (M + GT_BM - 1) / GT_BM * tn64;
  const int bid = (wk.y / tn) * tn64 + NB * (wk.y % tn);
  if (warp == 0) {
    unsigned nb = 0;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const float s = warp_sum_f(lane < 4 && !failed ? sh_f[4 * b + lane] : 0.f);
      if (n0 + 64 * b < N) {
        if (lane == 0) o.red.partials[bid + b] = (double)s;
        ++nb;
      }
    }
    if (lane == 0) {
      unsigned t;
      asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;"
                   : "=r"(t)
                   : "l"(o.red.ticket), "r"(nb)
                   : "memory");
      sh_last = (t + nb == (unsigned)nblk);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (sh_last) sum_partials<1>(o.red, nblk);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(Cfg::COLS)
                 : "memory");
}

// The first product's operand: opU = bf16(C x_3 T) of every problem (grid.y),
// four pixels a thread.
template <int NS>
__global__ void __launch_bounds__(256)
k_group_operand(const GroupProb* __restrict__ probs, GroupXf f) {
  const GroupProb& P = probs[blockIdx.y];
  const size_t npix = (size_t)P.n1 * P.s;  // a multiple of 8
  __nv_bfloat16* out = static_cast<__nv_bfloat16*>(P.opU);
  for (size_t i = 4 * ((size_t)blockIdx.x * 256 + threadIdx.x); i < npix;
       i += 4 * (size_t)gridDim.x * 256) {
    float x[NS][4];
#pragma unroll
    for (int l = 0; l < NS; ++l) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(P.C + l * npix + i));
      x[l][0] = v.x; x[l][1] = v.y; x[l][2] = v.z; x[l][3] = v.w;
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      float t[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        t[e] = 0.f;
#pragma unroll
        for (int l = 0; l < NS; ++l) t[e] = fmaf(f.nxt[k * NS + l], x[l][e], t[e]);
      }
      *reinterpret_cast<uint2*>(out + k * npix + i) =
          make_uint2(pack_bf16(t[0], t[1]), pack_bf16(t[2], t[3]));
    }
  }
}

template <int NS, int BN>
int set_smem() {
  TC_CUDA(cudaFuncSetAttribute(k_group_umma<NS, BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)GtCfg<NS, BN>::SMEM));
  TC_CUDA(cudaFuncSetAttribute(k_group_umma<NS, BN>, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  return TC_OK;
}

template <int NS, int BN>
int run(const GroupProb* probs, const CUtensorMap* maps, const int2* work, int nwork,
        const GroupOp& g, const GroupXf& f, cudaStream_t st) {
  k_group_umma<NS, BN><<<nwork, GT_NT, GtCfg<NS, BN>::SMEM, st>>>(probs, maps, work, g, f);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

template <class F>
int with_ns(int n3, F go) {
  switch (n3) {
    case 1: return go(std::integral_constant<int, 1>{});
    case 2: return go(std::integral_constant<int, 2>{});
    case 3: return go(std::integral_constant<int, 3>{});
    default: return go(std::integral_constant<int, 4>{});
  }
}

}  // namespace

int group_tc_init() {
  TC_TRY((set_smem<1, 64>()));
  TC_TRY((set_smem<2, 64>()));
  TC_TRY((set_smem<3, 64>()));
  TC_TRY((set_smem<4, 64>()));
  TC_TRY((set_smem<1, 128>()));
  TC_TRY((set_smem<2, 128>()));
  TC_TRY((set_smem<3, 128>()));
  TC_TRY((set_smem<4, 128>()));
  return TC_OK;
}

int launch_group_umma(const GroupProb* probs, const CUtensorMap* maps, const int2* work, int nwork,
                      const GroupOp& g, const float* epi, const float* nxt, int n3, int cfg,
                      cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_FUSED && nwork >= 1 && cfg >= 0 && cfg < 2);
  GroupXf f{};
  for (int i = 0; i < n3 * n3; ++i) {
    f.epi[i] = epi[i];
    f.nxt[i] = nxt[i];
  }
  return with_ns(n3, [&](auto ns) -> int {
    constexpr int NS = decltype(ns)::value;
    return cfg == 1 ? run<NS, 128>(probs, maps, work, nwork, g, f, st)
                    : run<NS, 64>(probs, maps, work, nwork, g, f, st);
  });
}

int launch_group_operand(const GroupProb* probs, int count, size_t most, const float* nxt, int n3,
                         cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_FUSED && count >= 1);
  GroupXf f{};
  for (int i = 0; i < n3 * n3; ++i) f.nxt[i] = nxt[i];
  const size_t b = (most + 1023) / 1024;
  return with_ns(n3, [&](auto ns) -> int {
    constexpr int NS = decltype(ns)::value;
    k_group_operand<NS><<<dim3((unsigned)(b < 64 ? b : 64), count), 256, 0, st>>>(probs, f);
    TC_CUDA(cudaGetLastError());
    return TC_OK;
  });
}

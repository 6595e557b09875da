// Mode-3 transform pass on the FFMA pipe (Remark 2.1: X~ = X x_3 T with T one
// of M, M^{-1}, M^{-T}, M^T): out[k][p] = ca * sum_l T[k][l] in[l][p] + cp *
// prev[k][p], with the fused reduction of the epilogue.
//
// Bound: HBM up to n3 = 32 (one read of in and prev, one write of out), the
// FFMA pipe at n3 = 64 (2 n3 flops a value moved: 28 us of FMAs against 20 us
// of traffic at 512 x 512 x 64). So:
// * packed FMAs (fma.rn.f32x2, two outputs k of one pixel): 16 outputs x 4
//   pixels a thread at n3 = 64, 5 shared-memory reads for 64 FMAs;
// * persistent CTAs of 128 threads, three to eight a SM, each looping over blocks
//   of 128 pixels; T is staged once a CTA, from its transpose (the plan holds
//   every transform's; read by columns it cost a CTA 2 us). The input streams through a ring of
//   four slots of up to 16 slices (8 KB) filled by cp.async, which runs three
//   slots ahead across blocks: the next block's input is in flight while a
//   block's results are stored. (Requesting a block as a whole once the last
//   one's FMAs were done left the FMA pipe 52% busy: 73 us at n3 = 64.)
// * prev is read four rows ahead of the stores (it may alias out, so the
//   compiler cannot move a read over an earlier store by itself); up to n3 = 16,
//   where a CTA has one block, the first rows before the FMAs: nothing else of
//   such a launch overlaps the read (144 x 144 x 9 c-LSQR with BF16X3 products, 6
//   steps: 318 us without it, 310 with).
// TRANS (TF32 operand of the tensor-core GEMM, which reads it K-major): a block
// is 8 rows x 16 columns of the K x N pixel grid and is stored N x K a slice, 32
// contiguous bytes a column, in place of a separate transposition pass.
//
// Measured, us a pass at 512 x 512 x n3 (before: one block a CTA of 256 threads,
// T read by columns, one FMA an instruction): n3 = 64 83 -> 58 (FMA pipe 59%
// busy while an SM has work; the copies, dups and addresses of only 64 FMAs a
// value take the other issue slots), with prev and the norm 115 -> 76; n3 = 32
// 28 -> 20, with prev and the norm 43 -> 30; the TF32 operand K-major 28 + 22
// (pass and transposition) -> 27. Four CTAs a SM at n3 = 64 (spills): 62.
#include <cuda_bf16.h>

#include "ffma_tile.cuh"

namespace {

using ftile::dup2;
using ftile::f32x2;
using ftile::fma2;
using ftile::unpack2;

enum OutKind { OUT_F32 = 0, OUT_BF16 = 1, OUT_TF32 = 2 };

__device__ __forceinline__ float round_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

constexpr int PB = 128;  // pixels a block
constexpr int LC = 16;   // input slices per cp.async group
constexpr int NT = 128;
// TRANS: a block is TR rows x TC columns; rows 4..7 of a slice sit 16 floats
// further on, so that the reads of rows i and 4 + i use different banks
constexpr int TR = 8, TC = PB / TR;
template <bool TRANS>
constexpr int slice_floats() { return TRANS ? PB + 16 : PB; }

constexpr int S = 4;  // ring slots
template <int KPW>
constexpr int slot_rows() { return KPW == 1 ? 8 : LC; }

// KPW: outputs of one of the eight virtual warps that the reduction's order is
// defined by (virtual warp v: outputs v KPW .. + KPW - 1; real warp w is virtual
// warps 2w and 2w + 1).
template <int KPW, bool TRANS>
constexpr size_t mode3_smem() {
  return ((size_t)(8 * KPW) * (8 * KPW) + (size_t)S * slot_rows<KPW>() * slice_floats<TRANS>()) *
         sizeof(float);
}

// Pixels of a transposed pass: P = rows x cols, row-major; unused otherwise.
struct Grid2 {
  int rows, cols;
};

// VEC: whole groups of 4 pixels and 16-byte aligned tensors.
template <int KPW, int OUT, bool TRANS, bool VEC>
__global__ void __launch_bounds__(NT, KPW == 8 ? 3 : (KPW == 4 ? 5 : (KPW == 2 ? 6 : 8)))
k_mode3(const float* __restrict__ in, void* out_v, const float* __restrict__ Tt, int n3, size_t P,
        size_t nblk, Grid2 g, Epi ep) {
  constexpr int NK = 8 * KPW, TK = 2 * KPW, SF = slice_floats<TRANS>(), LG = slot_rows<KPW>();
  constexpr int G = TK < 4 ? TK : 4;  // rows of prev read ahead of their stores
  constexpr bool EARLY = OUT == OUT_F32 && KPW <= 2;  // the first of them ahead of the FMAs
  const bool alone = nblk <= gridDim.x;               // where a CTA has one block
  if (ep.skip && *ep.skip) return;
  extern __shared__ __align__(16) float m3_smem[];
  float(*ts)[NK] = reinterpret_cast<float(*)[NK]>(m3_smem);  // ts[l][k] = T[k][l]
  float(*xs)[SF] = reinterpret_cast<float(*)[SF]>(m3_smem + NK * NK);
  __shared__ float sh_coef[2];
  __shared__ float sh_f[2][8];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int tcols = TRANS ? (g.cols + TC - 1) / TC : 1;
  const int nch = (n3 + LG - 1) / LG;  // slots a block

  // The ring's producer state: the next (block, slot of it) to request.
  size_t iblk = blockIdx.x;
  int ic = 0, islot = 0;
  auto issue = [&]() {
    if (iblk < nblk) {
      const size_t p0 = iblk * PB;
      const int r0 = TRANS ? (int)(iblk / tcols) * TR : 0, c0 = TRANS ? (int)(iblk % tcols) * TC : 0;
      const int l0 = ic * LG, lc_n = min(LG, n3 - l0);
      float(*x)[SF] = xs + islot * LG;
      // warp w copies rows w, w + 4, ..; lane: pixels 4 lane .. + 3 (TRANS: of
      // row lane / 4, columns 4 (lane % 4) .. + 3)
      const int px = 4 * lane;
      const int r = TRANS ? px / TC : 0, col = TRANS ? px % TC : 0;
      const size_t pix = TRANS ? (size_t)(r0 + r) * g.cols + c0 + col : p0 + px;
      const float* src = in + (size_t)(l0 + w) * P + pix;
      float* dst = &x[w][px + (r >= 4 ? 16 : 0)];
      int n = 0;  // pixels of the four that exist
      if (TRANS) n = r0 + r < g.rows ? g.cols - c0 - col : 0;
      else n = P > pix ? (int)(P - pix < 4 ? P - pix : 4) : 0;
      if (VEC) {
        for (int lc = w; lc < lc_n; lc += NT / 32, src += (NT / 32) * P, dst += (NT / 32) * SF)
          ftile::cp16(dst, n > 0 ? src : in, n > 0);
      } else {
        for (int lc = w; lc < lc_n; lc += NT / 32, src += (NT / 32) * P, dst += (NT / 32) * SF)
#pragma unroll
          for (int e = 0; e < 4; ++e) ftile::cp4(dst + e, e < n ? src + e : in, e < n);
      }
      islot = (islot + 1) % S;
      if (++ic == nch) {
        ic = 0;
        iblk += gridDim.x;
      }
    }
    ftile::cp_commit();
  };
  for (int idx = tid; idx < n3 * NK; idx += NT) {  // lands with the first slot
    const int l = idx / NK, k = idx % NK;
    ftile::cp4(&ts[l][k], k < n3 ? Tt + l * n3 + k : Tt, k < n3);
  }
  for (int i = 0; i < S - 1; ++i) issue();
  if (OUT == OUT_F32) coef_compute(ep.coef, sh_coef);

  // partial of block blk from the eight virtual warps' sums (warp 0)
  auto put_partial = [&](size_t blk, int par) {
    float s = lane < 8 ? sh_f[par][lane] : 0.f;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ep.red.partials[blk] = (double)s;
  };
  int par = 0, slot = 0;
  size_t prev_blk = nblk;
  for (size_t blk = blockIdx.x; blk < nblk; blk += gridDim.x, par ^= 1) {
    f32x2 acc[KPW][4];
#pragma unroll
    for (int q = 0; q < KPW; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[q][e] = 0ull;
    float4 pv[G];
    auto load_prev = [&](int q0, size_t pb, size_t idx0) {
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (VEC && ep.prev && pb < P && w * TK + q0 + q < n3)
          pv[q] = *reinterpret_cast<const float4*>(ep.prev + idx0 + (q0 + q) * P);
    };
    if (EARLY && alone) {
      const size_t p0 = blk * PB + lane * 4;
      load_prev(0, p0, (size_t)(w * TK) * P + p0);
    }
    for (int c = 0; c < nch; ++c) {
      ftile::cp_wait<S - 2>();  // this thread's copies of the slot have landed
      __syncthreads();  // everyone's (and T); every warp is done with the slot refilled now
      issue();
      if (OUT == OUT_F32 && c == 0 && w == 0 && ep.red.out && prev_blk < nblk)
        put_partial(prev_blk, par ^ 1);
      const int l0 = c * LG, lc_n = min(LG, n3 - l0);
      const float(*xc)[SF] = xs + slot * LG;
      slot = (slot + 1) % S;
      auto fma_slice = [&](int lc) {
        float x[4];
        if (TRANS) {  // rows 4h .. 4h + 3 of column lane % 16, h = lane / 16
          const float* xp = &xc[lc][(lane >> 4) * (4 * TC + 16) + (lane & 15)];
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = xp[e * TC];
        } else {
          const float4 v = *reinterpret_cast<const float4*>(&xc[lc][lane * 4]);
          x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        }
        f32x2 t[KPW];
        if (KPW >= 2) {
#pragma unroll
          for (int q = 0; q < KPW; q += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&ts[l0 + lc][w * TK + 2 * q]);
            t[q] = v.x;
            t[q + 1] = v.y;
          }
        } else {
          t[0] = *reinterpret_cast<const f32x2*>(&ts[l0 + lc][w * TK]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const f32x2 xe = dup2(x[e]);
#pragma unroll
          for (int q = 0; q < KPW; ++q) acc[q][e] = fma2(t[q], xe, acc[q][e]);
        }
      };
      if (w * TK >= n3) continue;  // a warp without outputs
      // four slices unrolled, not the slot: the code of a whole slot and of the
      // store together outgrew the instruction cache
#pragma unroll 4
      for (int lc = 0; lc < lc_n; ++lc) fma_slice(lc);
    }

    if constexpr (TRANS) {  // slice k, column c0 + lane % 16, rows r0 + 4 (lane / 16) .. + 3
      const int r = (int)(blk / tcols) * TR + (lane >> 4) * 4;
      const int col = (int)(blk % tcols) * TC + (lane & 15);
      float* out = static_cast<float*>(out_v);
#pragma unroll
      for (int q = 0; q < TK; ++q) {
        const int k = w * TK + q;
        if (k >= n3 || col >= g.cols || r >= g.rows) continue;
        float y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 v = unpack2(acc[q / 2][e]);
          y[e] = round_tf32((q & 1) ? v.y : v.x);
        }
        float* o = out + (size_t)k * P + (size_t)col * g.rows + r;
        if (VEC) {
          *reinterpret_cast<float4*>(o) = make_float4(y[0], y[1], y[2], y[3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (r + e < g.rows) o[e] = y[e];
        }
      }
      continue;
    }
    const size_t pb = blk * PB + lane * 4;
    if constexpr (OUT == OUT_BF16) {  // operand of a tensor-core GEMM: store only
#pragma unroll
      for (int q = 0; q < TK; ++q) {
        const int k = w * TK + q;
        if (k >= n3) continue;
        float y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 v = unpack2(acc[q / 2][e]);
          y[e] = (q & 1) ? v.y : v.x;
        }
        const size_t idx = (size_t)k * P + pb;
        if constexpr (VEC) {
          if (pb >= P) continue;
          const __nv_bfloat162 lo = __floats2bfloat162_rn(y[0], y[1]);
          const __nv_bfloat162 hi = __floats2bfloat162_rn(y[2], y[3]);
          *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(out_v) + idx) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                         *reinterpret_cast<const uint32_t*>(&hi));
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (pb + e < P)
              static_cast<__nv_bfloat16*>(out_v)[idx + e] = __float2bfloat16_rn(y[e]);
        }
      }
      continue;
    }
    float* out = static_cast<float*>(out_v);
    const float ca = sh_coef[0], cp = sh_coef[1];
    const size_t idx0 = (size_t)(w * TK) * P + pb;
    float local[2] = {0.f, 0.f};  // of virtual warps 2w and 2w + 1
#pragma unroll
    for (int q0 = 0; q0 < TK; q0 += G) {
      if (!EARLY || !alone || q0 > 0) load_prev(q0, pb, idx0);
#pragma unroll
      for (int q = 0; q < G; ++q) {
        const int k = w * TK + q0 + q;
        if (k >= n3) continue;
        float y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 v = unpack2(acc[(q0 + q) / 2][e]);
          y[e] = (q & 1) ? v.y : v.x;
        }
        float& loc = local[(q0 + q) / KPW];
        const size_t idx = idx0 + (q0 + q) * P;
        if constexpr (VEC) {
          if (pb >= P) continue;
          float4 o = make_float4(ca * y[0], ca * y[1], ca * y[2], ca * y[3]);
          if (ep.prev) {
            o.x = fmaf(cp, pv[q].x, o.x); o.y = fmaf(cp, pv[q].y, o.y);
            o.z = fmaf(cp, pv[q].z, o.z); o.w = fmaf(cp, pv[q].w, o.w);
          }
          *reinterpret_cast<float4*>(out + idx) = o;
          if (ep.red.out) {
            const float4 ov = ep.red.other ? *reinterpret_cast<const float4*>(ep.red.other + idx) : o;
            loc = fmaf(o.x, ov.x, fmaf(o.y, ov.y, fmaf(o.z, ov.z, fmaf(o.w, ov.w, loc))));
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (pb + e < P) {
              float o = ca * y[e];
              if (ep.prev) o = fmaf(cp, ep.prev[idx + e], o);
              out[idx + e] = o;
              if (ep.red.out) loc = fmaf(o, ep.red.other ? ep.red.other[idx + e] : o, loc);
            }
        }
      }
    }
    if (ep.red.out) {
      local[0] = warp_sum_f(local[0]);
      local[1] = warp_sum_f(local[1]);
      if (lane == 0) {
        sh_f[par][2 * w] = local[0];
        sh_f[par][2 * w + 1] = local[1];
      }
      prev_blk = blk;
    }
  }
  ftile::cp_wait<0>();
  if (OUT != OUT_F32 || !ep.red.out) return;
  // the last block's partial, then one arrival a CTA
  __shared__ int sh_last;
  __syncthreads();
  if (w == 0) {
    if (prev_blk < nblk) put_partial(prev_blk, par ^ 1);
    if (lane == 0) {
      unsigned t;
      asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(t) : "l"(ep.red.ticket) : "memory");
      sh_last = (t == gridDim.x - 1);
    }
  }
  __syncthreads();
  if (sh_last) sum_partials<2>(ep.red, nblk);
}

// Persistent grid: the CTAs that fit, no more than one a block.
template <class K>
int fit(K kernel, size_t smem, int* per_sm) {
  TC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  TC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared));
  TC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, NT, smem));
  return *per_sm >= 1 ? TC_OK : TC_ECUDA;
}

int g_sms = 0;
template <int KPW, int OUT, bool TRANS, bool VEC>
int g_fit = 0;  // CTAs a SM (set at init)

template <int KPW, int OUT, bool TRANS>
int init1() {
  TC_TRY(fit(k_mode3<KPW, OUT, TRANS, true>, mode3_smem<KPW, TRANS>(), &g_fit<KPW, OUT, TRANS, true>));
  return fit(k_mode3<KPW, OUT, TRANS, false>, mode3_smem<KPW, TRANS>(),
             &g_fit<KPW, OUT, TRANS, false>);
}

template <int KPW>
int init_kpw() {
  if constexpr (KPW <= 4) {  // above TC_TUBE_MIN_N3 the operands come from the tcgen05 pass
    TC_TRY((init1<KPW, OUT_BF16, false>()));
    TC_TRY((init1<KPW, OUT_TF32, true>()));
  }
  return init1<KPW, OUT_F32, false>();
}

template <int KPW, int OUT, bool TRANS, bool VEC>
int run1(const float* in, void* out, const float* Tt, int n3, size_t P, Grid2 g, const Epi& ep,
         cudaStream_t st) {
  const size_t nblk = TRANS ? (size_t)((g.rows + TR - 1) / TR) * ((g.cols + TC - 1) / TC)
                            : (P + PB - 1) / PB;
  const size_t cap = (size_t)g_sms * g_fit<KPW, OUT, TRANS, VEC>;
  const unsigned grid = (unsigned)(nblk < cap ? nblk : cap);
  k_mode3<KPW, OUT, TRANS, VEC><<<grid, NT, mode3_smem<KPW, TRANS>(), st>>>(in, out, Tt, n3, P,
                                                                            nblk, g, ep);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

template <int KPW, int OUT, bool TRANS>
int run(const float* in, void* out, const float* Tt, int n3, size_t P, Grid2 g, const Epi& ep,
        cudaStream_t st) {
  auto al = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  const bool vec = (TRANS ? g.rows % 4 == 0 && g.cols % 4 == 0 : P % 4 == 0) && al(in) && al(out) &&
                   al(ep.prev) && al(ep.red.other);
  return vec ? run1<KPW, OUT, TRANS, true>(in, out, Tt, n3, P, g, ep, st)
             : run1<KPW, OUT, TRANS, false>(in, out, Tt, n3, P, g, ep, st);
}

template <int OUT, bool TRANS = false>
int pick(const float* in, void* out, const float* Tt, int n3, size_t P, const Epi& ep,
         cudaStream_t st, Grid2 g = {}) {
  if (n3 <= 8) return run<1, OUT, TRANS>(in, out, Tt, n3, P, g, ep, st);
  if (n3 <= 16) return run<2, OUT, TRANS>(in, out, Tt, n3, P, g, ep, st);
  if (n3 <= 32) return run<4, OUT, TRANS>(in, out, Tt, n3, P, g, ep, st);
  if constexpr (OUT == OUT_F32) return run<8, OUT, TRANS>(in, out, Tt, n3, P, g, ep, st);
  return TC_EINVAL;
}

}  // namespace

int mode3_init() {
  int dev = 0;
  TC_CUDA(cudaGetDevice(&dev));
  TC_CUDA(cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev));
  TC_TRY(init_kpw<1>());
  TC_TRY(init_kpw<2>());
  TC_TRY(init_kpw<4>());
  return init_kpw<8>();
}

int launch_mode3(const float* in, float* out, const float* Tt, int n3, size_t P,
                 const Epi& ep, cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_N3);
  return pick<OUT_F32>(in, out, Tt, n3, P, ep, st);
}

int launch_mode3_bf16(const float* in, void* out, const float* Tt, int n3, size_t P,
                      const int* skip, cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_N3);
  Epi ep;
  ep.skip = skip;
  return pick<OUT_BF16>(in, out, Tt, n3, P, ep, st);
}

int launch_mode3_tf32_kmajor(const float* in, float* out, const float* Tt, int n3, int rows,
                             int cols, const int* skip, cudaStream_t st) {
  TC_CHECK(n3 >= 1 && n3 <= TC_MAX_N3);
  Epi ep;
  ep.skip = skip;
  return pick<OUT_TF32, true>(in, out, Tt, n3, (size_t)rows * cols, ep, st, Grid2{rows, cols});
}

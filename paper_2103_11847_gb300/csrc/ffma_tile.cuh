// FP32 GEMM tiles on the FFMA pipe, shared by the slice GEMMs (gemm.cu): one
// CTA accumulates a BM x BN output tile of NS slices at once,
//   acc[k] += A_k (pro B)_k over the whole contraction,
// with A given K-major (K x M per slice: the plan keeps the slice transposes of
// A~ and B~, so both operands have rows of constant K index and land in the
// layout the FMAs read, with no transpose on the way).
//
// Bound: the FFMA pipe (128 FMAs a clock and SM). Three things keep it fed:
// * packed FMAs (fma.rn.f32x2): two accumulators an instruction, so the pipe
//   is full at half the issue slots and the shared-memory reads, the copies
//   and the address arithmetic fit in the other half. Each half is the IEEE
//   fma of its element; an output's additions run in K order, as one chain.
// * 8 x 4 (NS > 1) or 8 x 8 outputs a thread: 3 or 4 128-bit shared-memory
//   reads for 32 or 64 FMAs. A read of A is two or four distinct 16-byte words
//   a warp, a read of B 128 or 256 contiguous bytes: no conflicts.
// * a ring of STAGES K blocks filled by cp.async ahead of the FMAs, one barrier
//   a block (larger K blocks and deeper rings measured the same to 5%, 8 x 16
//   outputs a thread no better). The prologue transform is applied in place by the thread that
//   copied the position (all slices of it), before that barrier.
// Measured (512^3 x 64 slices, 128 x 64 x 32): FMA pipe 82% busy while an SM has
// work, issue slots 56%; warps wait for the pipe (math-pipe throttle) first.
#pragma once

#include "tc_device.cuh"

namespace ftile {

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 dup2(float x) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src),
               "r"(valid ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// WIDE: warps of 2 x 16 threads, each thread 8 consecutive rows (the fused
// tiles: a warp owns 16 rows, so a warp past the last row skips its FMAs);
// otherwise 4 x 8 threads, rows and columns in groups of four.
template <int NS_, int BM_, int BN_, int BK_, int TN_, int STAGES_, bool WIDE_>
struct Tile {
  static constexpr int NS = NS_, BM = BM_, BN = BN_, BK = BK_, TM = 8, TN = TN_, S = STAGES_;
  static constexpr bool WIDE = WIDE_;
  static constexpr int TX = BN / TN, TY = BM / TM, NT = TX * TY;
  static constexpr int LX = WIDE ? 16 : 8, LY = 32 / LX;  // a warp's threads
  static constexpr int kA = NS * BK * BM, kB = NS * BK * BN, kSlot = kA + kB;
  static constexpr size_t bytes = (size_t)S * kSlot * sizeof(float);
  static constexpr int PA = BK * BM / 4, PB = BK * BN / 4;  // 16-byte positions of a slice's block
  static constexpr int NA = (PA + NT - 1) / NT, NB = (PB + NT - 1) / NT;
  static_assert(TN == 4 || (TN == 8 && !WIDE), "8 x 4 or 8 x 8 a thread");
  static_assert(WIDE ? TX == 16 && TY % 2 == 0 : TX % 8 == 0 && TY % 4 == 0, "whole warps");
};

// Thread coordinates: warps tile the CTA's (TY / LY) x (TX / LX) grid.
template <class T>
__device__ __forceinline__ int tile_tx() {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  return (w % (T::TX / T::LX)) * T::LX + (lane % T::LX);
}
template <class T>
__device__ __forceinline__ int tile_ty() {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  return (w / (T::TX / T::LX)) * T::LY + lane / T::LX;
}
// The tile row of the thread's rows 4h .. 4h + 3 and the tile column of its
// columns 4h .. 4h + 3.
template <class T>
__device__ __forceinline__ int tile_row(int ty, int h) {
  return T::WIDE ? ty * 8 + 4 * h : h * (T::BM / 2) + ty * 4;
}
template <class T>
__device__ __forceinline__ int tile_col(int tx, int h) { return h * (T::TX * 4) + tx * 4; }

// acc[k][i][j]: rows 2i and 2i + 1 of the thread's TM, column j of its TN.
template <class T>
using Acc = f32x2[T::NS][T::TM / 2][T::TN];

// VEC: rows of whole 16-byte groups (M, N multiples of 4, aligned bases);
// otherwise 4-byte copies. At: K x M, B: K x N a slice. pro: NS x NS or unused.
template <class T, bool PRO, bool VEC>
__device__ __forceinline__ void mainloop(const float* __restrict__ At, const float* __restrict__ B,
                                         int M, int N, int K, int kbeg, int kend, int i0, int j0,
                                         const float* pro, float* sm, Acc<T>& acc) {
  constexpr int NS = T::NS, BM = T::BM, BN = T::BN, BK = T::BK, S = T::S, NT = T::NT;
  const int tid = threadIdx.x, tx = tile_tx<T>(), ty = tile_ty<T>();
  const size_t sA = (size_t)K * M, sB = (size_t)K * N;
#pragma unroll
  for (int k = 0; k < NS; ++k)
#pragma unroll
    for (int i = 0; i < T::TM / 2; ++i)
#pragma unroll
      for (int j = 0; j < T::TN; ++j) acc[k][i][j] = 0ull;

  auto issue = [&](int c) {
    const int k0 = kbeg + c * BK;
    float* sa = sm + (c % S) * T::kSlot;
    float* sb = sa + T::kA;
    auto copy = [&](float* dst, const float* base, size_t slice, int cols, int kk, int col,
                    int dstride) {
      const int gk = k0 + kk;
      const float* row = base + (size_t)gk * cols + col;
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        if (VEC) {
          const bool ok = gk < kend && col < cols;
          cp16(dst + k * dstride, ok ? row + k * slice : base, ok);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const bool ok = gk < kend && col + e < cols;
            cp4(dst + k * dstride + e, ok ? row + k * slice + e : base, ok);
          }
        }
      }
    };
#pragma unroll
    for (int q = 0; q < T::NA; ++q) {
      const int p = tid + NT * q, kk = p / (BM / 4), m = (p % (BM / 4)) * 4;
      if (T::PA % NT == 0 || p < T::PA) copy(sa + kk * BM + m, At, sA, M, kk, i0 + m, BK * BM);
    }
#pragma unroll
    for (int q = 0; q < T::NB; ++q) {
      const int p = tid + NT * q, kk = p / (BN / 4), n = (p % (BN / 4)) * 4;
      if (T::PB % NT == 0 || p < T::PB) copy(sb + kk * BN + n, B, sB, N, kk, j0 + n, BK * BN);
    }
  };
  const bool live = i0 + (int)(threadIdx.x >> 5) * 16 < M;  // WIDE: the warp's first row
  const int nk = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
#pragma unroll
  for (int s = 0; s < S - 1; ++s) {
    if (s < nk) issue(s);
    cp_commit();
  }
  for (int c = 0; c < nk; ++c) {
    cp_wait<S - 2>();  // this thread's copies of block c have landed
    float* sa = sm + (c % S) * T::kSlot;
    float* sb = sa + T::kA;
    if (PRO) {  // (pro B)_k on the positions this thread copied
#pragma unroll
      for (int q = 0; q < T::NB; ++q) {
        const int p = tid + NT * q;
        if (T::PB % NT != 0 && p >= T::PB) break;
        float* b = sb + (p / (BN / 4)) * BN + (p % (BN / 4)) * 4;
        float4 x[NS];
#pragma unroll
        for (int l = 0; l < NS; ++l) x[l] = *reinterpret_cast<const float4*>(b + l * BK * BN);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int l = 0; l < NS; ++l) {
            const float m = pro[k * NS + l];
            t.x = fmaf(m, x[l].x, t.x);
            t.y = fmaf(m, x[l].y, t.y);
            t.z = fmaf(m, x[l].z, t.z);
            t.w = fmaf(m, x[l].w, t.w);
          }
          *reinterpret_cast<float4*>(b + k * BK * BN) = t;
        }
      }
    }
    __syncthreads();  // block c complete; every warp is done with block c - 1
    if (c + S - 1 < nk) issue(c + S - 1);
    cp_commit();
    if (T::WIDE && !live) continue;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const float* ap = sa + (k * BK + kk) * BM;
        const float* bp = sb + (k * BK + kk) * BN;
        f32x2 a[T::TM / 2], b[T::TN];
#pragma unroll
        for (int h = 0; h < T::TM / 4; ++h) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(ap + tile_row<T>(ty, h));
          a[2 * h] = v.x;
          a[2 * h + 1] = v.y;
        }
#pragma unroll
        for (int h = 0; h < T::TN / 4; ++h) {
          const float4 v = *reinterpret_cast<const float4*>(bp + tile_col<T>(tx, h));
          b[4 * h] = dup2(v.x);
          b[4 * h + 1] = dup2(v.y);
          b[4 * h + 2] = dup2(v.z);
          b[4 * h + 3] = dup2(v.w);
        }
#pragma unroll
        for (int i = 0; i < T::TM / 2; ++i)
#pragma unroll
          for (int j = 0; j < T::TN; ++j) acc[k][i][j] = fma2(a[i], b[j], acc[k][i][j]);
      }
    }
  }
  cp_wait<0>();  // no copy of this thread is in flight (the ring may be reused)
}

}  // namespace ftile

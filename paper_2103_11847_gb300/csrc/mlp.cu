// The learned-lambda network: 36 -> 64 -> 64 -> 2 with GELU, FP32 master
// weights, BF16 weight copies used by the forward pass, FP32 accumulation.
// It maps features of the first c-LSQR steps to (log lambda, stop index) and
// stands in for the GCV search of §3.1 and the stopping choice of §3.3. The
// paper has no such network.
//
// Parameters are one flat FP32 vector, W1 (36 x 64, row-major in x out), b1,
// W2 (64 x 64), b2, W3 (64 x 2), b3. The loss is (1/2B) sum (out - t)^2. All
// reductions over the batch run in a fixed order, so training is deterministic.
//
// A training step is two launches, each started while the last one finishes
// (programmatic dependent launch): the samples' pass and the gradients with
// the Adam step. As four launches (forward, backward, gradients as chains of
// global loads, Adam) a step of 256 samples took 33 us, now 12.
#include <cuda_bf16.h>

#include <new>
#include <vector>

#include "tc_device.cuh"
#include "mlp.cuh"

namespace {

constexpr int NI = MLP_IN, NH = MLP_HID, NO = MLP_OUT;
constexpr int OW1 = 0, OB1 = OW1 + NI * NH, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH,
              OB3 = OW3 + NH * NO;
static_assert(OB3 + NO == MLP_NPARAMS, "parameter layout");

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// The pass over samples, four a CTA of 256 threads (64 a sample): forward, and
// with targets (TRAIN) the loss and the backward pass through the
// activations, D = (out - t) / B, dZ2 = (D W3^T) * gelu'(z2), dZ1 = (dZ2 W2^T) *
// gelu'(z1).
//
// Bound: latency (a batch of 256 is 10 MFLOP; every sum over inputs is one chain
// of at most 64 FMAs). The BF16 weights are staged in shared memory once a CTA
// with 16-byte copies; W2's rows are 66 values apart, so that both its columns
// (forward) and its rows (backward) are read without bank conflicts. z1 and z2
// stay in registers. A forward pass of many samples takes the CTAs that fit, eight
// a SM, each over several groups of four, so that the weights are staged once a CTA
// and the next group's inputs are on their way (200000 samples 281 us; one group a
// CTA 303, one sample a CTA reading the weights from L1 291; 20000: 32.8, 34.8, 32.8).
constexpr int SPC = 4;           // samples a group
constexpr int CTAS = 8;          // a SM
constexpr int W2S = NH + 2;      // row stride of W2 in shared memory

template <bool TRAIN>  // with targets: one group a CTA
__global__ void __launch_bounds__(SPC * NH, TRAIN ? 0 : CTAS)
k_mlp_samples(const float* __restrict__ X, const float* __restrict__ T, int B,
              const __nv_bfloat16* Wb, const float* theta, float* H1, float* H2, float* OUT,
              float* D, float* dZ1, float* dZ2, float* lossb) {
  __shared__ __align__(16) __nv_bfloat16 w1[NI * NH];
  __shared__ __align__(16) __nv_bfloat16 w2[NH * W2S];
  __shared__ __align__(16) __nv_bfloat16 w3[NH * NO];
  __shared__ float xs[SPC][NI], h1s[SPC][NH], h2s[SPC][NH], dz2s[SPC][NH], ds[SPC][NO];
  const int tid = threadIdx.x, q = tid / NH, j = tid % NH;
  static_assert(SPC * NI <= SPC * NH, "an input a thread");
  auto input = [&](int g) {  // thread tid's of group g's inputs
    return tid < SPC * NI && g * SPC + tid / NI < B ? X[(size_t)g * SPC * NI + tid] : 0.f;
  };
  float x = input(blockIdx.x);
  pdl_trigger();
  pdl_wait();  // the weights are the last step's
  for (int i = tid; i < NI * NH / 8; i += SPC * NH)
    reinterpret_cast<uint4*>(w1)[i] = reinterpret_cast<const uint4*>(Wb + OW1)[i];
  for (int i = tid; i < NH * NH / 8; i += SPC * NH) {
    const uint4 v = reinterpret_cast<const uint4*>(Wb + OW2)[i];
    uint32_t* d = reinterpret_cast<uint32_t*>(w2 + (i / (NH / 8)) * W2S + (i % (NH / 8)) * 8);
    d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
  }
  if (tid < NH * NO / 8) reinterpret_cast<uint4*>(w3)[tid] = reinterpret_cast<const uint4*>(Wb + OW3)[tid];
  const float bias1 = theta[OB1 + j], bias2 = theta[OB2 + j];
  const int groups = (B - 1) / SPC + 1;
  for (int grp = blockIdx.x; grp < groups; grp += gridDim.x) {
    const int b = grp * SPC + q;
    const bool live = b < B;
    if (tid < SPC * NI) xs[tid / NI][tid % NI] = x;  // the last group's have been used
    __syncthreads();
    if (!TRAIN && grp + (int)gridDim.x < groups) x = input(grp + gridDim.x);
    float z1 = bias1;
#pragma unroll
    for (int i = 0; i < NI; ++i) z1 = fmaf(xs[q][i], __bfloat162float(w1[i * NH + j]), z1);
    const float h1 = gelu(z1);
    h1s[q][j] = h1;
    if (H1 && live) H1[(size_t)b * NH + j] = h1;
    __syncthreads();
    float z2 = bias2;
#pragma unroll
    for (int i = 0; i < NH; ++i) z2 = fmaf(h1s[q][i], __bfloat162float(w2[i * W2S + j]), z2);
    const float h2 = gelu(z2);
    h2s[q][j] = h2;
    if (H2 && live) H2[(size_t)b * NH + j] = h2;
    __syncthreads();
    if (j < NO) {
      float o = theta[OB3 + j];
#pragma unroll
      for (int i = 0; i < NH; ++i) o = fmaf(h2s[q][i], __bfloat162float(w3[i * NO + j]), o);
      if (OUT && live) OUT[(size_t)b * NO + j] = o;
      if (TRAIN) {
        const float r = live ? o - T[(size_t)b * NO + j] : 0.f;
        ds[q][j] = r / B;
        if (live) D[(size_t)b * NO + j] = r / B;
        float l = 0.f;  // threads 0 and 1 of the sample are neighbours in one warp
#pragma unroll
        for (int k = 0; k < NO; ++k) {
          const float rk = __shfl_sync((1u << NO) - 1, r, k, NO);
          l = fmaf(rk, rk, l);
        }
        if (j == 0 && live) lossb[b] = 0.5f * l / B;
      }
    }
    if (!TRAIN) continue;
    __syncthreads();
    float g = 0.f;
#pragma unroll
    for (int o = 0; o < NO; ++o) g = fmaf(ds[q][o], __bfloat162float(w3[j * NO + o]), g);
    const float dz2 = g * gelu_d(z2);
    dz2s[q][j] = dz2;
    if (live) dZ2[(size_t)b * NH + j] = dz2;
    __syncthreads();
    g = 0.f;
#pragma unroll
    for (int k = 0; k < NH; ++k) g = fmaf(dz2s[q][k], __bfloat162float(w2[j * W2S + k]), g);
    if (live) dZ1[(size_t)b * NH + j] = g * gelu_d(z1);
    return;
  }
}

// Adam (bias-corrected) on parameter p; refreshes its BF16 copy.
struct Adam {
  float* theta = nullptr;  // null: gradients only
  float* m = nullptr;
  float* v = nullptr;
  __nv_bfloat16* Wb = nullptr;
  int t = 0;
  float lr = 0.f;
};

// A parameter's Adam state, read before its gradient is summed so that the
// reads and the bias corrections are off the end of the launch.
struct AdamState {
  float th = 0.f, m = 0.f, v = 0.f;
};

__device__ __forceinline__ AdamState adam_read(const Adam& a, int p, bool live) {
  AdamState s;
  if (a.theta && live) {
    s.th = a.theta[p];
    s.m = a.m[p];
    s.v = a.v[p];
  }
  return s;
}

__device__ __forceinline__ void put_grad(int p, float g, float* grad, const Adam& a,
                                         const AdamState& s, float c1, float c2) {
  if (!a.theta) {
    grad[p] = g;
    return;
  }
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mm = b1 * s.m + (1.f - b1) * g;
  const float vv = b2 * s.v + (1.f - b2) * g * g;
  a.m[p] = mm;
  a.v[p] = vv;
  const float mh = mm / c1;
  const float vh = vv / c2;
  const float th = s.th - a.lr * mh / (sqrtf(vh) + eps);
  a.theta[p] = th;
  a.Wb[p] = __float2bfloat16_rn(th);
}

// Parameter gradients, each one chain over the batch in order, and the Adam
// step on them. A CTA of 64 threads owns 4 rows x 32 columns of [W1; b1] (37
// rows, the last against ones) or [W2; b2] (65 rows), two rows a thread; the
// last CTA owns W3, b3 and the loss. The columns of dZ and of the layer's input
// come through shared memory in chunks of GB samples, the next chunk in flight
// (cp.async) while this one is summed: the sums are chains of FMAs on
// shared-memory operands instead of chains of global loads.
constexpr int GB = 128, GT = 64;
constexpr int GR1 = (NI + 1 + 3) / 4, GR2 = (NH + 1 + 3) / 4;  // row groups of the two layers
constexpr int GCTAS = 2 * GR1 + 2 * GR2 + 1;

__device__ __forceinline__ void cp_async(float* dst, const float* src, int bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}

__global__ void __launch_bounds__(GT)
k_mlp_grad(const float* __restrict__ X, int B, const float* H1, const float* H2, const float* D,
           const float* dZ1, const float* dZ2, const float* lossb, float* grad, float* loss,
           Adam a) {
  __shared__ __align__(16) float vs[2][GB][32];
  __shared__ __align__(16) float us[2][GB][4];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  pdl_trigger();
  const float c1 = 1.f - powf(0.9f, (float)a.t), c2 = 1.f - powf(0.999f, (float)a.t);
  pdl_wait();  // the activations and their gradients are the samples' pass's
  const int nch = (B + GB - 1) / GB;
  if (blockIdx.x == GCTAS - 1) {  // W3 (64 x 2), b3, loss: H2 in two halves of 32 columns
    float s[NO] = {0.f, 0.f}, t = 0.f;
    const AdamState q0 = adam_read(a, OW3 + tid * NO, true);
    const AdamState q1 = adam_read(a, OW3 + tid * NO + 1, true);
    const AdamState q3 = adam_read(a, OB3 + tid, tid < NO);
    for (int b0 = 0; b0 < B; b0 += GB) {
      const int nb = min(GB, B - b0);
      __syncthreads();
      for (int i = tid; i < nb * (NH / 4); i += GT) {
        const int r = i / (NH / 4), c = (i % (NH / 4)) * 4;
        cp_async(&vs[c / 32][r][c % 32], H2 + (size_t)(b0 + r) * NH + c, 16);
      }
      for (int i = tid; i < nb; i += GT) {
        cp_async(&us[0][i][0], D + (size_t)(b0 + i) * NO, 4);
        cp_async(&us[0][i][1], D + (size_t)(b0 + i) * NO + 1, 4);
        cp_async(&us[0][i][2], lossb + b0 + i, 4);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
#pragma unroll 8
      for (int r = 0; r < nb; ++r) {
        const float h = vs[w][r][lane];
        s[0] = fmaf(h, us[0][r][0], s[0]);
        s[1] = fmaf(h, us[0][r][1], s[1]);
        if (tid < 3) t += us[0][r][tid];  // b3[0], b3[1], loss
      }
    }
    put_grad(OW3 + tid * NO, s[0], grad, a, q0, c1, c2);
    put_grad(OW3 + tid * NO + 1, s[1], grad, a, q1, c1, c2);
    if (tid < NO) put_grad(OB3 + tid, t, grad, a, q3, c1, c2);
    if (tid == NO && loss) *loss = t;
    return;
  }
  const bool second = blockIdx.x >= 2 * GR1;
  const int g = second ? blockIdx.x - 2 * GR1 : blockIdx.x;
  const int rows = second ? NH : NI, r0 = (g / 2) * 4, c0 = (g % 2) * 32;
  const float* U = second ? H1 : X;      // the layer's input, rows values a sample
  const float* V = second ? dZ2 : dZ1;   // its output's gradient
  auto issue = [&](int c) {
    const int b0 = c * GB, nb = min(GB, B - b0);
    for (int i = tid; i < nb * 8; i += GT)
      cp_async(&vs[c & 1][i / 8][(i % 8) * 4], V + (size_t)(b0 + i / 8) * NH + c0 + (i % 8) * 4, 16);
    for (int i = tid; i < nb * 4; i += GT) {
      const int r = i / 4, k = r0 + i % 4;
      if (k < rows) cp_async(&us[c & 1][r][i % 4], U + (size_t)(b0 + r) * rows + k, 4);
      else us[c & 1][r][i % 4] = 1.f;  // the bias row
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  issue(0);
  // [W; b] is contiguous: row k, column j at k NH + j, the bias as row `rows`
  const int k = r0 + 2 * w, p = (second ? OW2 : OW1) + k * NH + c0 + lane;
  const AdamState q0 = adam_read(a, p, k <= rows), q1 = adam_read(a, p + NH, k + 1 <= rows);
  float s0 = 0.f, s1 = 0.f;
  for (int c = 0; c < nch; ++c) {
    if (c + 1 < nch) {
      issue(c + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int nb = min(GB, B - c * GB);
#pragma unroll 16
    for (int r = 0; r < nb; ++r) {
      const float v = vs[c & 1][r][lane];
      const float2 u = *reinterpret_cast<const float2*>(&us[c & 1][r][2 * w]);
      s0 = fmaf(u.x, v, s0);
      s1 = fmaf(u.y, v, s1);
    }
    __syncthreads();  // the buffer is refilled two chunks on
  }
  if (k <= rows) put_grad(p, s0, grad, a, q0, c1, c2);
  if (k + 1 <= rows) put_grad(p + NH, s1, grad, a, q1, c1, c2);
}

__global__ void k_to_bf16(const float* theta, __nv_bfloat16* Wb) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < MLP_NPARAMS) Wb[p] = __float2bfloat16_rn(theta[p]);
}

// Deterministic pseudo-random initialisation (splitmix64), scaled by 1/sqrt(fan_in).
__global__ void k_init(float* theta, unsigned long long seed) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= MLP_NPARAMS) return;
  unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(p + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const float u = (float)((z >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;  // U(-1, 1)
  float scale = 0.f;
  if (p < OB1) scale = rsqrtf((float)NI);
  else if (p >= OW2 && p < OB2) scale = rsqrtf((float)NH);
  else if (p >= OW3 && p < OB3) scale = rsqrtf((float)NH);
  theta[p] = u * scale * 1.7320508f;  // unit variance times 1/sqrt(fan_in)
}

}  // namespace

struct tc_mlp {
  float* theta = nullptr;  // FP32 master parameters
  float* m = nullptr;
  float* v = nullptr;
  __nv_bfloat16* Wb = nullptr;  // BF16 copy (biases too, unused)
  float* norm = nullptr;        // x mean[36], x std[36], t mean[2], t std[2]
  float* work = nullptr;        // activations for up to kMaxB samples
  float* loss = nullptr;
  int step = 0;
};

namespace {
constexpr int kMaxB = 1024;
constexpr size_t kWork = (size_t)kMaxB * (4 * NH + NO + 1);
}  // namespace

extern "C" int tc_mlp_create(tc_mlp** out, unsigned long long seed, tc_stream_t stream) {
  if (!out) return TC_EINVAL;
  tc_mlp* m = new (std::nothrow) tc_mlp();
  if (!m) return TC_ENOMEM;
  cudaStream_t st = (cudaStream_t)stream;
  bool ok = cudaMalloc(&m->theta, MLP_NPARAMS * 4) == cudaSuccess &&
            cudaMalloc(&m->m, MLP_NPARAMS * 4) == cudaSuccess &&
            cudaMalloc(&m->v, MLP_NPARAMS * 4) == cudaSuccess &&
            cudaMalloc(&m->Wb, MLP_NPARAMS * 2) == cudaSuccess &&
            cudaMalloc(&m->norm, MLP_NORM * 4) == cudaSuccess &&
            cudaMalloc(&m->work, kWork * 4) == cudaSuccess &&
            cudaMalloc(&m->loss, 4) == cudaSuccess;
  if (!ok) {
    tc_mlp_destroy(m);
    return TC_ENOMEM;
  }
  TC_CUDA(cudaMemsetAsync(m->m, 0, MLP_NPARAMS * 4, st));
  TC_CUDA(cudaMemsetAsync(m->v, 0, MLP_NPARAMS * 4, st));
  std::vector<float> nrm(MLP_NORM, 0.f);
  for (int i = 0; i < MLP_IN; ++i) nrm[MLP_IN + i] = 1.f;
  nrm[2 * MLP_IN + 2] = nrm[2 * MLP_IN + 3] = 1.f;
  TC_CUDA(cudaMemcpyAsync(m->norm, nrm.data(), MLP_NORM * 4, cudaMemcpyHostToDevice, st));
  k_init<<<(MLP_NPARAMS + 255) / 256, 256, 0, st>>>(m->theta, seed);
  k_to_bf16<<<(MLP_NPARAMS + 255) / 256, 256, 0, st>>>(m->theta, m->Wb);
  TC_CUDA(cudaGetLastError());
  TC_CUDA(cudaStreamSynchronize(st));
  *out = m;
  return TC_OK;
}

extern "C" int tc_mlp_destroy(tc_mlp* m) {
  if (!m) return TC_EINVAL;
  void* ps[] = {m->theta, m->m, m->v, m->Wb, m->norm, m->work, m->loss};
  for (void* p : ps)
    if (p) cudaFree(p);
  delete m;
  return TC_OK;
}

extern "C" int tc_mlp_set_params(tc_mlp* m, const float* theta, const float* norm,
                                 tc_stream_t stream) {
  if (!m || (!theta && !norm)) return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (theta) {
    TC_CUDA(cudaMemcpyAsync(m->theta, theta, MLP_NPARAMS * 4, cudaMemcpyDeviceToDevice, st));
    k_to_bf16<<<(MLP_NPARAMS + 255) / 256, 256, 0, st>>>(m->theta, m->Wb);
    TC_CUDA(cudaGetLastError());
    TC_CUDA(cudaMemsetAsync(m->m, 0, MLP_NPARAMS * 4, st));
    TC_CUDA(cudaMemsetAsync(m->v, 0, MLP_NPARAMS * 4, st));
    m->step = 0;
  }
  if (norm) TC_CUDA(cudaMemcpyAsync(m->norm, norm, MLP_NORM * 4, cudaMemcpyDeviceToDevice, st));
  return TC_OK;
}

extern "C" int tc_mlp_get_params(tc_mlp* m, float* theta, float* norm, tc_stream_t stream) {
  if (!m || (!theta && !norm)) return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (theta) TC_CUDA(cudaMemcpyAsync(theta, m->theta, MLP_NPARAMS * 4, cudaMemcpyDeviceToDevice, st));
  if (norm) TC_CUDA(cudaMemcpyAsync(norm, m->norm, MLP_NORM * 4, cudaMemcpyDeviceToDevice, st));
  return TC_OK;
}

namespace {
// early: a launch that may start while its predecessor, a launch of the same
// training call, finishes (the kernels wait in pdl_wait before they read or
// write what it touches). The call's first launch starts in stream order: it
// reads the caller's data before that wait.
template <class... P, class... A>
int launch_pdl(bool early, void (*kernel)(P...), int grid, int block, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  TC_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  return TC_OK;
}

// Loss and gradients of one batch, and with `a.theta` the Adam step on them.
int fwd_bwd(tc_mlp* m, const float* X, const float* T, int B, float* grad, float* loss,
            const Adam& a, bool first, cudaStream_t st) {
  float* H1 = m->work;
  float* H2 = H1 + (size_t)kMaxB * NH;
  float* D = H2 + (size_t)kMaxB * NH;
  float* dZ1 = D + (size_t)kMaxB * NO;
  float* dZ2 = dZ1 + (size_t)kMaxB * NH;
  float* lossb = dZ2 + (size_t)kMaxB * NH;
  TC_TRY(launch_pdl(!first, k_mlp_samples<true>, (B + SPC - 1) / SPC, SPC * NH, st, X, T, B, m->Wb, m->theta, H1,
                    H2, (float*)nullptr, D, dZ1, dZ2, lossb));
  return launch_pdl(true, k_mlp_grad, GCTAS, GT, st, X, B, H1, H2, D, dZ1, dZ2, lossb, grad, loss, a);
}
}  // namespace

extern "C" int tc_mlp_loss_grad(tc_mlp* m, const float* X, const float* T, int B, float* loss,
                                float* grad, tc_stream_t stream) {
  if (!m || !X || !T || !grad || B < 1 || B > kMaxB) return TC_EINVAL;
  return fwd_bwd(m, X, T, B, grad, loss, Adam{}, true, (cudaStream_t)stream);
}

extern "C" int tc_mlp_forward(tc_mlp* m, const float* X, int B, float* Y, tc_stream_t stream) {
  if (!m || !X || !Y || B < 1) return TC_EINVAL;
  float* none = nullptr;
  const int groups = (B - 1) / SPC + 1, fit = 152 * CTAS;
  return launch_pdl(false, k_mlp_samples<false>, groups < fit ? groups : fit, SPC * NH, (cudaStream_t)stream, X,
                    none, B, m->Wb, m->theta, none, none, Y, none, none, none, none);
}

extern "C" int tc_mlp_train(tc_mlp* m, const float* X, const float* T, int N, int batch, int steps,
                            float lr, float* loss_hist, tc_stream_t stream) {
  if (!m || !X || !T || N < 1 || batch < 1 || batch > kMaxB || steps < 1 || !(lr > 0.f))
    return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int off = 0;
  for (int s = 0; s < steps; ++s) {
    const int B = (off + batch <= N) ? batch : N - off;
    ++m->step;
    TC_TRY(fwd_bwd(m, X + (size_t)off * MLP_IN, T + (size_t)off * MLP_OUT, B, nullptr,
                   loss_hist ? loss_hist + s : m->loss,
                   Adam{m->theta, m->m, m->v, m->Wb, m->step, lr}, s == 0, st));
    off += B;
    if (off >= N) off = 0;
  }
  return TC_OK;
}

namespace {
// Column means and standard deviations of R (N x ncol) into stats[0..ncol)
// and stats[ncol..2 ncol); then R_out = (R - mean) / std. One CTA per column.
__global__ void k_colstats(const float* R, int N, int ncol, float* mean, float* stdv, float* R_out) {
  __shared__ double s1[256], s2[256];
  const int c = blockIdx.x, t = threadIdx.x;
  double a = 0.0, b = 0.0;
  for (int i = t; i < N; i += 256) {
    const double v = R[(size_t)i * ncol + c];
    a += v;
    b += v * v;
  }
  s1[t] = a;
  s2[t] = b;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (t < o) {
      s1[t] += s1[t + o];
      s2[t] += s2[t + o];
    }
    __syncthreads();
  }
  __shared__ float mu, sd;
  if (t == 0) {
    const double m = s1[0] / N;
    const double var = fmax(s2[0] / N - m * m, 0.0);
    mu = (float)m;
    sd = (float)(var > 1e-12 ? sqrt(var) : 1.0);
    mean[c] = mu;
    stdv[c] = sd;
  }
  __syncthreads();
  for (int i = t; i < N; i += 256) R_out[(size_t)i * ncol + c] = (R[(size_t)i * ncol + c] - mu) / sd;
}
}  // namespace

extern "C" int tc_mlp_fit_norm(tc_mlp* m, const float* Xraw, const float* Traw, int N, float* Xn,
                               float* Tn, tc_stream_t stream) {
  if (!m || !Xraw || !Traw || !Xn || !Tn || N < 2) return TC_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  k_colstats<<<MLP_IN, 256, 0, st>>>(Xraw, N, MLP_IN, m->norm, m->norm + MLP_IN, Xn);
  k_colstats<<<MLP_OUT, 256, 0, st>>>(Traw, N, MLP_OUT, m->norm + 2 * MLP_IN,
                                       m->norm + 2 * MLP_IN + MLP_OUT, Tn);
  TC_CUDA(cudaGetLastError());
  return TC_OK;
}

// device-side inference used by the learned solve (learned.cu)
const __nv_bfloat16* mlp_weights(const tc_mlp* m) { return m->Wb; }
const float* mlp_theta(const tc_mlp* m) { return m->theta; }
const float* mlp_norm(const tc_mlp* m) { return m->norm; }

// Learned seed of the continuous-pole expansion (not in the paper): a multilayer
// perceptron nin -> nh (x nhidden, GELU) -> nout (softplus) maps the normalised
// Matsubara self-energy of one (k, n) problem to non-negative pole weights on the CPE
// grid. Training minimises L = (1/B) sum_b ||A b_hat_b - x_b||^2 (A = CPE kernel at the
// first nw_fit fermionic frequencies, real-stacked), so no labels are needed.
//
// Every matrix product runs on the tensor cores (tcgen05, fp16 operands from shared
// memory in the 128-byte swizzle layout, FP32 accumulation in TMEM) with the activations and their
// derivatives in the epilogues; the loss and Adam run in FP32 kernels. Weights are kept in FP32 (master) with fp16
// copies W [out][in] and W^T [in][out] for the two product shapes.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gw_internal.h"
#include "tc_common.cuh"

using namespace gwi::tc;

struct gw_mlp {
  int device = 0;
  cudaStream_t stream = nullptr;
  int nin = 0, nh = 0, nhidden = 0, nout = 0, nlayers = 0;
  std::vector<int> din, dout;  // per layer
  std::vector<float*> W, b, mW, vW, mb, vb;
  std::vector<float*> gW, gb;  // in `grads`, parameter order
  float* grads = nullptr;
  std::vector<__half*> Wh, WTh;
  int64_t step = 0;
  // workspaces for batch <= cap (all of them in `owned`)
  int64_t cap = 0;
  std::vector<void*> owned;
  bool captured = false;       // a call was captured into a graph: outgrown workspaces are kept, in `retired`
  std::vector<void*> retired;
  std::vector<float*> Z;      // pre-activations [B][dout]
  std::vector<__half*> Hh;    // fp16 activations [B][dout] (layer input of the next)
  std::vector<__half*> HT;    // fp16 transposed activations [dout][B] (incl. input at index 0)
  __half* Xh = nullptr;       // fp16 input [B][nin]
  float* out = nullptr;       // [B][nout]
  std::vector<float*> dZ;     // per layer [B][dout]
  std::vector<__half*> dZh;   // per layer [B][dout]
  std::vector<__half*> dZT;   // per layer [dout][B]
  float* part = nullptr;      // [K splits][num_params]: dW over parts of the batch; null: dZ of a layer at a time
  float* loss = nullptr;      // [1]
  int* err = nullptr;
  std::string errmsg;
};

namespace gwi {
namespace mlpk {

// ------------------------------------------------------------------ GEMM with fused epilogues
// C[M][N] (FP32) = A[M][K] * B[N][K]^T, A, B fp16 row-major. M % 128 == 0, N % 64 == 0, K % 64 == 0. One
// block per 128 x 64 tile (and part of K): the layers are a few hundred wide, so small tiles fill more SMs
// and a panel of up to 256 k is brought in one go (the latency of one load, not of one per 64 k).
// Measured at batch 1024, 128-256-256-256-128: 11 us per GEMM with its epilogue, against 50 us in 128 x 256
// tiles with a load per 64 k and 5 us for each elementwise pass; loss and gradients 705 -> 130 us, 31 -> 11
// launches. What bounds it is latency: 32 blocks, one load, one short MMA chain, one epilogue.
constexpr int GEMM_THREADS = 256;
constexpr int GN = 64, GK = 256;
constexpr int G_A = 128 * 128, G_B = GN * 128;  // bytes of one 64-wide K tile
constexpr int G_SMEM = 1024 + (GK / 64) * (G_A + G_B);

enum { EPI_ACT = 0, EPI_BACK = 1, EPI_PART = 2 };
struct GemmArgs {
  const __half *A, *B;
  int M, N, K;
  const float* bias;    // EPI_ACT
  float* Z;             // EPI_ACT: pre-activations, written; EPI_BACK: the lower layer's, read
  __half *H, *HT;       // EPI_ACT: activations; EPI_BACK: dZ in fp16, both [row][col] and [col][row]
  float* out;           // EPI_ACT: FP32 activations of the last layer; EPI_BACK: dZ; EPI_PART: partial C
  int last;
};
// The dW products of all layers in one launch (EPI_PART): tiles of job j from tile0, K in `splits` parts
constexpr int kMaxLayers = 16;
struct GemmJobs {
  GemmArgs job[kMaxLayers];
  int tile0[kMaxLayers + 1];
  int njobs, kpart;
  int64_t stride;  // floats from one part of K to the next
};

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_g(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}
__device__ __forceinline__ float softplus_f(float z) { return fmaxf(z, 0.f) + log1pf(expf(-fabsf(z))); }
__device__ __forceinline__ float sigmoid_f(float z) { return 1.f / (1.f + expf(-z)); }

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

template <int EPI>
__device__ __forceinline__ void gemm_tile(const GemmArgs& g, int tile, int k0, int k1, int* err) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bar;
  __shared__ uint32_t tslot;
  __shared__ int abort_g, no_dealloc;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nt = g.N / GN, m0 = (tile / nt) * 128, n0 = (tile % nt) * GN;
  if (tid == 0) {
    mbar_init(&bar, 1);
    abort_g = 0;
    no_dealloc = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&tslot, GN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tslot;
  int panel = 0;
  for (int kp = k0; kp < k1; kp += GK, ++panel) {
    const int kn = min(GK, k1 - kp), kc8 = kn / 8;  // 16-byte pieces of a row
    for (int e = tid; e < (128 + GN) * kc8; e += GEMM_THREADS) {
      const int r = e / kc8, c = e % kc8;
      if (r < 128)
        cp16(base + (c >> 3) * G_A + sw128_off(r, 8 * (c & 7)), g.A + (size_t)(m0 + r) * g.K + kp + 8 * c);
      else
        cp16(base + (GK / 64) * G_A + (c >> 3) * G_B + sw128_off(r - 128, 8 * (c & 7)),
             g.B + (size_t)(n0 + r - 128) * g.K + kp + 8 * c);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      for (int q = 0; q < kn / 64; ++q) {
        const uint32_t a = smem_u32(base + q * G_A), b = smem_u32(base + (GK / 64) * G_A + q * G_B);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          mma_f16(tbase, sdesc_sw128(a + 32 * ks), sdesc_sw128(b + 32 * ks), idesc_f16(128, GN, false, false),
                  (kp > k0 || q > 0 || ks > 0) ? 1u : 0u);
      }
      mma_commit(&bar);
    }
    // a thread whose wait runs out stops the whole block after the barrier (abort_g is written
    // only between the two barriers of an iteration, so every thread reads the same value)
    if (!mbar_wait(&bar, panel & 1, err)) abort_g = 1;
    tc_fence_after();
    __syncthreads();
    if (abort_g) break;
  }
  // MMAs still running into TMEM complete before the block frees it; if they do not, it keeps it
  if (abort_g && tid == 0 && !mbar_wait_drain(&bar, panel & 1)) no_dealloc = 1;
  __syncthreads();
  const bool ok = !abort_g;
  // warp: rows 32 (warp & 3) + lane, columns 32 (warp >> 2) .. + 31
  const int row = m0 + 32 * (warp & 3) + lane;
  for (int c = 32 * (warp >> 2); c < 32 * (warp >> 2) + 32; c += 16) {
    float v[16];
    if (ok) {
      tmem_ld16(tbase + ((uint32_t)(32 * (warp & 3)) << 16) + c, v);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = 0.f;
    }
    const int col = n0 + c;
    const size_t o = (size_t)row * g.N + col;
    // 16-byte accesses (col is a multiple of 16): scalar ones by 32 lanes in 32 rows cost a sector each
    float4* zo = reinterpret_cast<float4*>((EPI == EPI_PART ? g.out : g.Z) + o);
    if (EPI == EPI_PART) {
#pragma unroll
      for (int q = 0; q < 4; ++q) zo[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      continue;
    }
    alignas(16) __half h[16];
    float y[16];
    if (EPI == EPI_ACT) {  // z = A B^T + bias, h = act(z)
      const float4* bo = reinterpret_cast<const float4*>(g.bias + col);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 bq = bo[q];
        v[4 * q] += bq.x;
        v[4 * q + 1] += bq.y;
        v[4 * q + 2] += bq.z;
        v[4 * q + 3] += bq.w;
        zo[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
#pragma unroll
      for (int e = 0; e < 16; ++e) y[e] = g.last ? softplus_f(v[e]) : gelu_f(v[e]);
    } else {  // dZ = dH act'(Z) of a hidden layer
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 z = zo[q];
        y[4 * q] = v[4 * q] * gelu_g(z.x);
        y[4 * q + 1] = v[4 * q + 1] * gelu_g(z.y);
        y[4 * q + 2] = v[4 * q + 2] * gelu_g(z.z);
        y[4 * q + 3] = v[4 * q + 3] * gelu_g(z.w);
      }
    }
    if (EPI == EPI_BACK || g.last) {
      float4* yo = reinterpret_cast<float4*>(g.out + o);
#pragma unroll
      for (int q = 0; q < 4; ++q) yo[q] = make_float4(y[4 * q], y[4 * q + 1], y[4 * q + 2], y[4 * q + 3]);
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      h[e] = __float2half_rn(y[e]);
      g.HT[(size_t)(col + e) * g.M + row] = h[e];
    }
    uint4* ho = reinterpret_cast<uint4*>(g.H + o);
    ho[0] = reinterpret_cast<const uint4*>(h)[0];
    ho[1] = reinterpret_cast<const uint4*>(h)[1];
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0 && !no_dealloc) tmem_dealloc(tbase, GN);
}

template <int EPI>
__global__ void __launch_bounds__(GEMM_THREADS) k_gemm_tc(const __grid_constant__ GemmArgs g, int* __restrict__ err) {
  gemm_tile<EPI>(g, blockIdx.x, 0, g.K, err);
}

__global__ void __launch_bounds__(GEMM_THREADS) k_gemm_dw(const __grid_constant__ GemmJobs J, int* __restrict__ err) {
  int j = 0;
  while (j + 1 < J.njobs && (int)blockIdx.x >= J.tile0[j + 1]) ++j;
  GemmArgs g = J.job[j];
  g.out += blockIdx.y * J.stride;
  const int k0 = blockIdx.y * J.kpart;
  gemm_tile<EPI_PART>(g, blockIdx.x - J.tile0[j], k0, min(g.K, k0 + J.kpart), err);
}

// Gradients in parameter order from the parts: blocks of 256 weights (the parts summed in order), and for
// each layer's biases the column sums of dZ (block: 32 columns x 32 row lanes).
struct GradJobs {
  const float* dZ[kMaxLayers];
  int64_t w0[kMaxLayers];    // first weight of the layer in parameter order
  int nw[kMaxLayers], d[kMaxLayers], blk0[kMaxLayers + 1], wblk[kMaxLayers];
  int nlayers, splits;
  int64_t stride, batch;
};
__global__ void __launch_bounds__(1024) k_grads(const __grid_constant__ GradJobs J, const float* __restrict__ part,
                                                float* __restrict__ grads) {
  int l = 0;
  while (l + 1 < J.nlayers && (int)blockIdx.x >= J.blk0[l + 1]) ++l;
  const int b = blockIdx.x - J.blk0[l];
  if (b < J.wblk[l]) {
    const int e = b * 1024 + threadIdx.x;
    if (e >= J.nw[l]) return;
    const float* p = part + J.w0[l] + e;
    float s = p[0];
    for (int q = 1; q < J.splits; ++q) s += p[q * J.stride];
    grads[J.w0[l] + e] = s;
    return;
  }
  __shared__ float sm[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c = 32 * (b - J.wblk[l]) + tx, d = J.d[l];
  const float* z = J.dZ[l] + c;
  float s = 0.f;
#pragma unroll 4
  for (int64_t r = ty; r < J.batch; r += 32) s += z[r * d];
  sm[ty][tx] = s;
  __syncthreads();
  if (ty == 0) {
    for (int q = 1; q < 32; ++q) s += sm[q][tx];
    grads[J.w0[l] + J.nw[l] + c] = s;
  }
}

// ------------------------------------------------------------------ loss and the rest
// residual R = out A^T - x (FP32), loss = (1/B) sum R^2, dOut = (2/B) R A, dZ = dOut softplus'(Z) of the last
// layer with its fp16 copies. One block per LS = 8 samples: every element of A is read once for them (one
// sample, its outputs read from memory, where those of eight do not fit in shared memory). 67 -> 24 us at batch 1024.
template <int LS>
__global__ void __launch_bounds__(128) k_loss(const float* __restrict__ out, const float* __restrict__ x,
                                              const float* __restrict__ Acpe, const float* __restrict__ Z, int64_t Bn,
                                              int nout, int nx, float* __restrict__ dZ, __half* __restrict__ dZh,
                                              __half* __restrict__ dZT, float* __restrict__ loss) {
  extern __shared__ float sm[];
  const int64_t b0 = (int64_t)blockIdx.x * LS;  // Bn is a multiple of 128
  const float* so = LS > 1 ? sm : out + b0 * nout;  // [nout][LS]
  float* r = LS > 1 ? sm + nout * LS : sm;          // [nx][LS]
  if (LS > 1) {
    for (int e = threadIdx.x; e < nout * LS; e += blockDim.x) sm[e] = out[(b0 + e % LS) * nout + e / LS];
    __syncthreads();
  }
  float part = 0.f;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    float s[LS];
#pragma unroll
    for (int q = 0; q < LS; ++q) s[q] = -x[(b0 + q) * nx + i];
#pragma unroll 8
    for (int m = 0; m < nout; ++m) {
      const float a = Acpe[(size_t)i * nout + m];
#pragma unroll
      for (int q = 0; q < LS; ++q) s[q] = fmaf(a, so[m * LS + q], s[q]);
    }
#pragma unroll
    for (int q = 0; q < LS; ++q) {
      r[i * LS + q] = s[q];
      part += s[q] * s[q];
    }
  }
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, part / (float)Bn);
  __syncthreads();
  for (int m = threadIdx.x; m < nout; m += blockDim.x) {
    float s[LS] = {};
#pragma unroll 8
    for (int i = 0; i < nx; ++i) {
      const float a = Acpe[(size_t)i * nout + m];
#pragma unroll
      for (int q = 0; q < LS; ++q) s[q] = fmaf(r[i * LS + q], a, s[q]);
    }
    __half h[LS];
#pragma unroll
    for (int q = 0; q < LS; ++q) {
      const size_t e = (size_t)(b0 + q) * nout + m;
      const float g = (2.f / (float)Bn) * s[q] * sigmoid_f(Z[e]);
      dZ[e] = g;
      h[q] = __float2half_rn(g);
      dZh[e] = h[q];
    }
#pragma unroll
    for (int q = 0; q < LS; ++q) dZT[(size_t)m * Bn + b0 + q] = h[q];
  }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int64_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const float gg = g[e];
  const float mm = b1 * m[e] + (1.f - b1) * gg;
  const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
  m[e] = mm;
  v[e] = vv;
  p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// fp16 copies of W [out][in] and W^T [in][out]
__global__ void k_w_half(const float* __restrict__ W, int dout, int din, __half* __restrict__ Wh,
                         __half* __restrict__ WT) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= dout * din) return;
  const int o = e / din, i = e % din;
  const __half h = __float2half_rn(W[e]);
  Wh[e] = h;
  WT[(size_t)i * dout + o] = h;
}

__global__ void k_x_half(const float* __restrict__ x, int64_t Bn, int nin, __half* __restrict__ Xh,
                         __half* __restrict__ XT) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= Bn * nin) return;
  const int64_t r = e / nin;
  const int c = (int)(e % nin);
  const __half h = __float2half_rn(x[e]);
  Xh[e] = h;
  XT[(size_t)c * Bn + r] = h;
}

gw_status mlp_err(gw_mlp* m, gw_status s, const char* what) {
  if (m) m->errmsg = what;
  return s;
}

gw_status mlp_check(gw_mlp* m, const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    m->errmsg = std::string(what) + ": " + cudaGetErrorString(e);
    return GW_ECUDA;
  }
  return GW_OK;
}

template <int EPI>
gw_status gemm(gw_mlp* m, const GemmArgs& g) {
  cudaFuncSetAttribute(k_gemm_tc<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM);
  k_gemm_tc<EPI><<<(g.M / 128) * (g.N / GN), GEMM_THREADS, G_SMEM, m->stream>>>(g, m->err);
  return mlp_check(m, "mlp gemm");
}

// parts of the batch in the dW products: 256 samples each, at most 16 parts
int dw_part(int64_t Bn) { return (int)std::max<int64_t>(GK, (Bn / 16 + 63) / 64 * 64); }

// Workspaces of a batch. Where memory is short (lean), one layer's dZ at a time and no parts of dW: 10 bytes per
// sample of the widest layer instead of 8 of every layer and up to 16 copies of the parameters.
bool alloc_batch(gw_mlp* m, int64_t Bn, bool lean) {
  if (m->captured)
    m->retired.insert(m->retired.end(), m->owned.begin(), m->owned.end());
  else
    for (void* p : m->owned) cudaFree(p);
  m->owned.clear();
  m->cap = 0;
  bool ok = true;
  auto get = [&](auto*& p, size_t n) {
    p = nullptr;
    if (ok && (ok = cudaMalloc((void**)&p, sizeof(*p) * n) == cudaSuccess)) m->owned.push_back(p);
  };
  const int L = m->nlayers;
  for (auto* v : {&m->Z, &m->dZ}) v->assign(L, nullptr);
  for (auto* v : {&m->Hh, &m->HT, &m->dZh, &m->dZT}) v->assign(v == &m->HT ? L + 1 : L, nullptr);
  const size_t widest = (size_t)Bn * *std::max_element(m->dout.begin(), m->dout.end());
  get(m->HT[0], (size_t)Bn * m->nin);
  get(m->Xh, (size_t)Bn * m->nin);
  get(m->out, (size_t)Bn * m->nout);
  for (int l = 0; l < L; ++l) {
    const size_t n = (size_t)Bn * m->dout[l];
    get(m->Z[l], n);
    get(m->Hh[l], n);
    get(m->HT[l + 1], n);
    if (lean && l > 0) {
      m->dZ[l] = m->dZ[0];
      m->dZT[l] = m->dZT[0];
    } else {
      get(m->dZ[l], lean ? widest : n);
      get(m->dZT[l], lean ? widest : n);
    }
    if (lean && l > 1)
      m->dZh[l] = m->dZh[l - 2];
    else
      get(m->dZh[l], lean ? widest : n);
  }
  m->part = nullptr;
  // any batch up to Bn: the number of parts grows with the batch up to 16
  if (!lean) get(m->part, (size_t)std::min<int64_t>(16, (Bn + GK - 1) / GK) * gw_mlp_num_params(m));
  if (!ok) {
    cudaGetLastError();
    for (void* p : m->owned) cudaFree(p);
    m->owned.clear();
    return false;
  }
  m->cap = Bn;
  return true;
}

gw_status ensure_batch(gw_mlp* m, int64_t Bn) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(m->stream, &cs) != cudaSuccess) {
    cudaGetLastError();
    cs = cudaStreamCaptureStatusActive;
  }
  if (cs != cudaStreamCaptureStatusNone) m->captured = true;
  if (Bn <= m->cap || alloc_batch(m, Bn, false) || alloc_batch(m, Bn, true)) return GW_OK;
  return mlp_err(m, GW_ENOMEM, "mlp workspace");
}

gw_status forward(gw_mlp* m, int64_t Bn, const float* x) {
  gw_status st;
  const int64_t nx = Bn * m->nin;
  k_x_half<<<(unsigned)((nx + 255) / 256), 256, 0, m->stream>>>(x, Bn, m->nin, m->Xh, m->HT[0]);
  if ((st = mlp_check(m, "mlp input")) != GW_OK) return st;
  for (int l = 0; l < m->nlayers; ++l) {
    GemmArgs g{l ? m->Hh[l - 1] : m->Xh, m->Wh[l], (int)Bn, m->dout[l], m->din[l], m->b[l], m->Z[l], m->Hh[l],
               m->HT[l + 1], m->out, l == m->nlayers - 1};
    if ((st = gemm<EPI_ACT>(m, g)) != GW_OK) return st;
  }
  return GW_OK;
}

// Gradients of the layers l0 .. l1 - 1 into m->grads, from their dZ. More layers than fit the job tables go in runs of
// kMaxLayers. Without parts (m->part null) dW is one product over the whole batch, straight into m->grads.
gw_status weight_grads(gw_mlp* m, int64_t Bn, int l0, int l1) {
  gw_status st;
  cudaFuncSetAttribute(k_gemm_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM);
  const int64_t np = gw_mlp_num_params(m);
  const int kpart = m->part ? dw_part(Bn) : (int)Bn, splits = (int)((Bn + kpart - 1) / kpart);
  float* part = m->part ? m->part : m->grads;
  for (; l0 < l1; l0 += kMaxLayers) {
    const int n = std::min(kMaxLayers, l1 - l0);
    GemmJobs J{};
    GradJobs D{};
    J.njobs = D.nlayers = n;
    J.kpart = kpart;
    J.stride = D.stride = np;
    D.splits = splits;
    D.batch = Bn;
    for (int i = 0; i < n; ++i) {  // dW = dZ^T H_in : [dout][din], K = batch
      const int l = l0 + i, d = m->dout[l], di = m->din[l];
      D.w0[i] = m->gW[l] - m->grads;
      J.job[i] = GemmArgs{m->dZT[l], m->HT[l], d, di, (int)Bn, nullptr, nullptr, nullptr, nullptr, part + D.w0[i], 0};
      J.tile0[i + 1] = J.tile0[i] + (d / 128) * (di / GN);
      D.dZ[i] = m->dZ[l];
      D.nw[i] = d * di;
      D.d[i] = d;
      D.wblk[i] = m->part ? (D.nw[i] + 1023) / 1024 : 0;
      D.blk0[i + 1] = D.blk0[i] + D.wblk[i] + d / 32;
    }
    k_gemm_dw<<<dim3(J.tile0[n], splits), GEMM_THREADS, G_SMEM, m->stream>>>(J, m->err);
    if ((st = mlp_check(m, "mlp gemm")) != GW_OK) return st;
    k_grads<<<D.blk0[n], 1024, 0, m->stream>>>(D, m->part, m->grads);
    if ((st = mlp_check(m, "mlp gradients")) != GW_OK) return st;
  }
  return GW_OK;
}

// Gradients into m->grads: dZ layer by layer downwards, then the weight gradients of all layers in one launch; with one
// layer's dZ at a time (m->part null) those of a layer before the dZ below it.
gw_status backward(gw_mlp* m, int64_t Bn, const float* x, const float* Acpe, int nx) {
  gw_status st;
  const int L = m->nlayers, e = L - 1;
  cudaMemsetAsync(m->loss, 0, sizeof(float), m->stream);
  auto loss = [&](auto* kernel, int ls, size_t sm) {
    if (sm > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kernel<<<(unsigned)(Bn / ls), 128, sm, m->stream>>>(m->out, x, Acpe, m->Z[e], Bn, m->nout, nx, m->dZ[e], m->dZh[e],
                                                       m->dZT[e], m->loss);
  };
  const size_t sm8 = 8 * sizeof(float) * ((size_t)m->nout + nx);
  if (sm8 <= 200 * 1024)
    loss(k_loss<8>, 8, sm8);
  else
    loss(k_loss<1>, 1, sizeof(float) * nx);
  if ((st = mlp_check(m, "mlp loss")) != GW_OK) return st;
  for (int l = e; l >= 0; --l) {
    if (!m->part && (st = weight_grads(m, Bn, l, l + 1)) != GW_OK) return st;
    if (l == 0) break;
    // dZ of the layer below = (dZ W) act'(Z)
    GemmArgs g{m->dZh[l], m->WTh[l], (int)Bn, m->din[l], m->dout[l], nullptr, m->Z[l - 1], m->dZh[l - 1], m->dZT[l - 1],
               m->dZ[l - 1], 0};
    if ((st = gemm<EPI_BACK>(m, g)) != GW_OK) return st;
  }
  return m->part ? weight_grads(m, Bn, 0, L) : GW_OK;
}

gw_status refresh_half(gw_mlp* m) {
  for (int l = 0; l < m->nlayers; ++l) {
    const int n = m->dout[l] * m->din[l];
    k_w_half<<<(n + 255) / 256, 256, 0, m->stream>>>(m->W[l], m->dout[l], m->din[l], m->Wh[l], m->WTh[l]);
    gw_status st = mlp_check(m, "mlp weights fp16");
    if (st != GW_OK) return st;
  }
  return GW_OK;
}

bool shapes_ok(const gw_mlp* m, int64_t Bn) {
  if (Bn <= 0 || Bn % 128) return false;
  for (int l = 0; l < m->nlayers; ++l)
    if (m->din[l] % 64 || m->dout[l] % 128) return false;
  return true;
}

}  // namespace mlpk
}  // namespace gwi

using namespace gwi::mlpk;

extern "C" {

gw_status gw_mlp_create(gw_mlp** out, int nin, int nh, int nhidden, int nout, uint64_t seed, int device,
                        void* stream) {
  if (!out || nin < 64 || nh < 128 || nhidden < 1 || nout < 128 || nin % 64 || nh % 128 || nout % 128)
    return GW_EINVAL;
  gw_mlp* m = new gw_mlp();
  if (cudaSetDevice(device) != cudaSuccess) {
    delete m;
    return GW_ECUDA;
  }
  m->device = device;
  m->stream = (cudaStream_t)stream;
  m->nin = nin;
  m->nh = nh;
  m->nhidden = nhidden;
  m->nout = nout;
  m->nlayers = nhidden + 1;
  for (int l = 0; l < m->nlayers; ++l) {
    m->din.push_back(l == 0 ? nin : nh);
    m->dout.push_back(l == m->nlayers - 1 ? nout : nh);
  }
  // deterministic init: splitmix64-driven Box-Muller normals (He init, small last layer)
  uint64_t s = seed ? seed : 0x9E3779B97F4A7C15ull;
  auto next = [&s]() {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  auto normal = [&]() {
    const double u1 = ((next() >> 11) + 1.0) * 0x1p-53, u2 = (next() >> 11) * 0x1p-53;
    return std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2);
  };
  bool ok = true;
  for (int l = 0; l < m->nlayers; ++l) {
    const int din = m->din[l], dout = m->dout[l];
    const double sc = l < m->nlayers - 1 ? std::sqrt(2.0 / din) : 0.1 / std::sqrt((double)din);
    std::vector<float> w((size_t)dout * din);
    for (auto& x : w) x = (float)(normal() * sc);
    float *W, *b, *mW, *vW, *mb, *vb;
    __half *Wh, *WTh;
    ok &= cudaMalloc((void**)&W, sizeof(float) * w.size()) == cudaSuccess;
    ok &= cudaMalloc((void**)&mW, sizeof(float) * w.size()) == cudaSuccess;
    ok &= cudaMalloc((void**)&vW, sizeof(float) * w.size()) == cudaSuccess;
    ok &= cudaMalloc((void**)&b, sizeof(float) * dout) == cudaSuccess;
    ok &= cudaMalloc((void**)&mb, sizeof(float) * dout) == cudaSuccess;
    ok &= cudaMalloc((void**)&vb, sizeof(float) * dout) == cudaSuccess;
    ok &= cudaMalloc((void**)&Wh, sizeof(__half) * w.size()) == cudaSuccess;
    ok &= cudaMalloc((void**)&WTh, sizeof(__half) * w.size()) == cudaSuccess;
    if (!ok) break;
    cudaMemcpy(W, w.data(), sizeof(float) * w.size(), cudaMemcpyHostToDevice);
    cudaMemset(mW, 0, sizeof(float) * w.size());
    cudaMemset(vW, 0, sizeof(float) * w.size());
    cudaMemset(b, 0, sizeof(float) * dout);
    cudaMemset(mb, 0, sizeof(float) * dout);
    cudaMemset(vb, 0, sizeof(float) * dout);
    m->W.push_back(W);
    m->b.push_back(b);
    m->mW.push_back(mW);
    m->vW.push_back(vW);
    m->mb.push_back(mb);
    m->vb.push_back(vb);
    m->Wh.push_back(Wh);
    m->WTh.push_back(WTh);
  }
  const size_t np = ok ? (size_t)gw_mlp_num_params(m) : 1;
  ok &= cudaMalloc((void**)&m->grads, sizeof(float) * np) == cudaSuccess;
  for (int l = 0, o = 0; ok && l < m->nlayers; ++l) {
    m->gW.push_back(m->grads + o);
    m->gb.push_back(m->grads + o + m->dout[l] * m->din[l]);
    o += m->dout[l] * (m->din[l] + 1);
  }
  ok &= cudaMalloc((void**)&m->loss, sizeof(float)) == cudaSuccess;
  ok &= cudaMalloc((void**)&m->err, sizeof(int)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    gw_mlp_destroy(m);
    return GW_ENOMEM;
  }
  cudaMemset(m->err, 0, sizeof(int));
  if (refresh_half(m) != GW_OK || cudaDeviceSynchronize() != cudaSuccess) {
    gw_mlp_destroy(m);
    return GW_ECUDA;
  }
  *out = m;
  return GW_OK;
}

gw_status gw_mlp_destroy(gw_mlp* m) {
  if (!m) return GW_EINVAL;
  cudaSetDevice(m->device);
  cudaDeviceSynchronize();
  auto fr = [](void* p) {
    if (p) cudaFree(p);
  };
  for (auto* v : {&m->W, &m->b, &m->mW, &m->vW, &m->mb, &m->vb})
    for (float* p : *v) fr(p);
  for (auto* v : {&m->Wh, &m->WTh})
    for (__half* p : *v) fr(p);
  for (void* p : m->owned) fr(p);
  for (void* p : m->retired) fr(p);
  fr(m->grads);
  fr(m->loss);
  fr(m->err);
  delete m;
  return GW_OK;
}

const char* gw_mlp_last_error(gw_mlp* m) { return m ? m->errmsg.c_str() : "null handle"; }

gw_status gw_mlp_forward(gw_mlp* m, int64_t batch, const float* x, float* out) {
  if (!m || !x || !out || !shapes_ok(m, batch)) return GW_EINVAL;
  gw_status st;
  if ((st = ensure_batch(m, batch)) != GW_OK) return st;
  if ((st = forward(m, batch, x)) != GW_OK) return st;
  if (cudaMemcpyAsync(out, m->out, sizeof(float) * batch * m->nout, cudaMemcpyDeviceToDevice, m->stream) !=
      cudaSuccess)
    return mlp_err(m, GW_ECUDA, "mlp output copy");
  return GW_OK;
}

gw_status gw_mlp_loss_grad(gw_mlp* m, int64_t batch, const float* x, int nx, const float* Acpe, float* loss,
                           float* grads) {
  if (!m || !x || !Acpe || !shapes_ok(m, batch) || nx <= 0) return GW_EINVAL;
  gw_status st;
  if ((st = ensure_batch(m, batch)) != GW_OK) return st;
  if ((st = forward(m, batch, x)) != GW_OK) return st;
  if ((st = backward(m, batch, x, Acpe, nx)) != GW_OK) return st;
  if (loss) cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDeviceToDevice, m->stream);
  if (grads)
    cudaMemcpyAsync(grads, m->grads, sizeof(float) * gw_mlp_num_params(m), cudaMemcpyDeviceToDevice, m->stream);
  return mlp_check(m, "mlp loss_grad");
}

gw_status gw_mlp_train_step(gw_mlp* m, int64_t batch, const float* x, int nx, const float* Acpe, float lr,
                            float* loss) {
  gw_status st;
  if ((st = gw_mlp_loss_grad(m, batch, x, nx, Acpe, loss, nullptr)) != GW_OK) return st;
  const float b1 = 0.9f, b2 = 0.999f;
  ++m->step;
  const float c1 = 1.f - std::pow(b1, (float)m->step), c2 = 1.f - std::pow(b2, (float)m->step);
  for (int l = 0; l < m->nlayers; ++l) {
    const int64_t nw = (int64_t)m->dout[l] * m->din[l];
    k_adam<<<(unsigned)((nw + 255) / 256), 256, 0, m->stream>>>(m->W[l], m->gW[l], m->mW[l], m->vW[l], nw, lr, b1, b2,
                                                                1e-8f, c1, c2);
    k_adam<<<(m->dout[l] + 255) / 256, 256, 0, m->stream>>>(m->b[l], m->gb[l], m->mb[l], m->vb[l], m->dout[l], lr, b1,
                                                            b2, 1e-8f, c1, c2);
  }
  if ((st = mlp_check(m, "mlp adam")) != GW_OK) return st;
  return refresh_half(m);
}

gw_status gw_mlp_sync(gw_mlp* m) {
  if (!m) return GW_EINVAL;
  if (cudaStreamSynchronize(m->stream) != cudaSuccess) return mlp_err(m, GW_ECUDA, "gw_mlp_sync: stream");
  int h = 0;
  if (cudaMemcpy(&h, m->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    return mlp_err(m, GW_ECUDA, "gw_mlp_sync: reading the device error word");
  if (h != 0) {
    cudaMemset(m->err, 0, sizeof(int));
    return mlp_err(m, GW_ETIMEOUT,
                   "gw_mlp_sync: a bounded wait in the tensor-core GEMM ran out; results since the last sync are undefined");
  }
  return GW_OK;
}

gw_status gw_mlp_get_params(gw_mlp* m, float* params) {
  if (!m || !params) return GW_EINVAL;
  size_t off = 0;
  gw_status st = gw_mlp_sync(m);
  if (st != GW_OK) return st;
  for (int l = 0; l < m->nlayers; ++l) {
    const size_t nw = (size_t)m->dout[l] * m->din[l];
    cudaMemcpy(params + off, m->W[l], sizeof(float) * nw, cudaMemcpyDeviceToHost);
    off += nw;
    cudaMemcpy(params + off, m->b[l], sizeof(float) * m->dout[l], cudaMemcpyDeviceToHost);
    off += m->dout[l];
  }
  return cudaGetLastError() == cudaSuccess ? GW_OK : GW_ECUDA;
}

gw_status gw_mlp_set_params(gw_mlp* m, const float* params) {
  if (!m || !params) return GW_EINVAL;
  size_t off = 0;
  cudaStreamSynchronize(m->stream);
  for (int l = 0; l < m->nlayers; ++l) {
    const size_t nw = (size_t)m->dout[l] * m->din[l];
    cudaMemcpy(m->W[l], params + off, sizeof(float) * nw, cudaMemcpyHostToDevice);
    off += nw;
    cudaMemcpy(m->b[l], params + off, sizeof(float) * m->dout[l], cudaMemcpyHostToDevice);
    off += m->dout[l];
  }
  if (cudaGetLastError() != cudaSuccess) return GW_ECUDA;
  return refresh_half(m);
}

int64_t gw_mlp_num_params(gw_mlp* m) {
  if (!m) return -1;
  int64_t n = 0;
  for (int l = 0; l < m->nlayers; ++l) n += (int64_t)m->dout[l] * m->din[l] + m->dout[l];
  return n;
}

}  // extern "C"

// Training of the retaining head (Eq. 2, Eq. 3): loss and gradients of W1, W2 for one sequence,
// backbone frozen.  Five launches: clear and W2 in fp32; pre = z W1 with the scores' partial sums in
// its epilogue; loss and its derivative per score; one pass over pre that forms both dpre and dW2; dW1 = z^T dpre.
// Both contractions run on the tcgen05 GEMM with W1, z and dpre read as they lie (no transposed
// copies).  Llama shape, 10240 tokens: the two contractions 2 x 75 us of tensor time at the measured
// peak, pre (42 MB, fp32) is written once and read once.
#include "../../include/locret.h"
#include "common.cuh"

using namespace locret;

namespace {

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + __expf(-x)); }

__global__ void rh_clear_kernel(const bf16 *__restrict__ w2, float *__restrict__ w2f, float *__restrict__ dw2, int n,
                                float *__restrict__ loss, int *__restrict__ status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    w2f[i] = __bfloat162float(w2[i]);
    dw2[i] = 0.f;
  }
  if (i == 0) { *loss = 0.f; *status = 0; }
}

// Eq. 3 per (token, head): Smooth-L1 (threshold 1) to the label plus alpha (s[t] - s[t+1])^2;
// ds = its derivative; the loss is summed with one atomic per block.  s = the sum of the column tiles' partial scores
// [tile][token][head], in tile order.
__global__ void rh_loss_kernel(const float *__restrict__ partial, int n_tiles, const float *__restrict__ labels, float *__restrict__ ds,
                               float *__restrict__ loss, int n, int h_kv, float alpha) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  float l = 0.f;
  auto s = [&](int at) {
    float v = 0.f;
    for (int nt = 0; nt < n_tiles; nt++) v += partial[(size_t)nt * n * h_kv + at];
    return v;
  };
  if (i < n * h_kv) {
    const int t = i / h_kv, m = i - t * h_kv;
    const float v = s(i), diff = v - labels[(size_t)m * n + t];
    const float ad = fabsf(diff);
    l = ad < 1.0f ? 0.5f * diff * diff : ad - 0.5f;
    float g = fminf(fmaxf(diff, -1.0f), 1.0f);
    if (t + 1 < n) {
      const float adj = v - s(i + h_kv);
      l = fmaf(alpha * adj, adj, l);
      g = fmaf(2.0f * alpha, adj, g);
    }
    if (t > 0) g -= 2.0f * alpha * (s(i - h_kv) - v);
    ds[i] = g;
  }
  __shared__ float red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(loss, v);
  }
}

// One pass over pre, thread = two neighbouring columns r, block = a slab of tokens:
//   dpre[t][r] = bf16( (sum_m ds[t][m] W2[r][m]) * silu'(pre[t][r]) )
//   dW2[r][m] += sum over the slab of silu(pre[t][r]) ds[t][m]
// The columns' W2 and dW2 stay in registers, ds of the slab in shared memory (heads padded to HK with zeros).
// Bound by instruction issue (about 90 per pair of pre-activations with 8 heads) with four warps per scheduler to hide the
// latencies, not by the 6 bytes per element: 10240 x 1024, 8 heads, 43 us (64 us with a bound to check per token,
// which kept the eight tokens' chains from overlapping; the bytes would take 10 us).
constexpr int DP_THREADS = 128, DP_SLAB = 64;

template <int HK>
__global__ void __launch_bounds__(DP_THREADS)
rh_dpre_dw2_kernel(const float *__restrict__ pre, const float *__restrict__ ds, const float *__restrict__ w2,
                   bf16 *__restrict__ dpre, float *__restrict__ dw2, int d_R, int h_kv) {
  __shared__ float sds[DP_SLAB][HK];
  const int r = (blockIdx.x * DP_THREADS + threadIdx.x) * 2;
  const int t0 = blockIdx.y * DP_SLAB;   // (n is a multiple of 64: slabs are full)
  for (int i = threadIdx.x; i < DP_SLAB * HK; i += DP_THREADS) {
    const int t = i / HK, m = i % HK;
    sds[t][m] = m < h_kv ? ds[(size_t)(t0 + t) * h_kv + m] : 0.f;
  }
  __syncthreads();
  if (r >= d_R) return;   // (d_R is even)
  float w[2][HK], acc[2][HK];
#pragma unroll
  for (int e = 0; e < 2; e++)
#pragma unroll
    for (int m = 0; m < HK; m++) {
      w[e][m] = m < h_kv ? w2[(size_t)(r + e) * h_kv + m] : 0.f;
      acc[e][m] = 0.f;
    }
  // TB tokens' pre-activations are requested while the TB before them are worked on
  constexpr int TB = HK > 8 ? 4 : 8;
  const float *src = pre + (size_t)t0 * d_R + r;
  bf16 *dst = dpre + (size_t)t0 * d_R + r;
  float2 next[TB];
#pragma unroll
  for (int i = 0; i < TB; i++) next[i] = *reinterpret_cast<const float2 *>(src + (size_t)i * d_R);
#pragma unroll 1
  for (int tb = 0; tb < DP_SLAB; tb += TB) {
    float2 cur[TB];
#pragma unroll
    for (int i = 0; i < TB; i++) {
      cur[i] = next[i];
      next[i] = *reinterpret_cast<const float2 *>(src + (size_t)min(tb + TB + i, DP_SLAB - 1) * d_R);
    }
#pragma unroll
    for (int i = 0; i < TB; i++) {
      const float2 p = cur[i];
      const float s0 = sigmoidf_(p.x), s1 = sigmoidf_(p.y);
      const float a0 = p.x * s0, a1 = p.y * s1;
      float d0 = 0.f, d1 = 0.f;
#pragma unroll
      for (int m = 0; m < HK; m++) {
        const float g = sds[tb + i][m];
        d0 = fmaf(g, w[0][m], d0);
        d1 = fmaf(g, w[1][m], d1);
        acc[0][m] = fmaf(a0, g, acc[0][m]);
        acc[1][m] = fmaf(a1, g, acc[1][m]);
      }
      *reinterpret_cast<uint32_t *>(dst + (size_t)(tb + i) * d_R) =
          pack_bf16(d0 * (s0 * (1.0f + p.x * (1.0f - s0))), d1 * (s1 * (1.0f + p.y * (1.0f - s1))));
    }
  }
#pragma unroll
  for (int e = 0; e < 2; e++)
#pragma unroll
    for (int m = 0; m < HK; m++)
      if (m < h_kv) atomicAdd(dw2 + (size_t)(r + e) * h_kv + m, acc[e][m]);
}

size_t pad256(size_t b) { return (b + 255) & ~(size_t)255; }

// The call's workspace in one block: offsets of its arrays.
struct Workspace {
  size_t pre, dpre, w2f, partial, ds, status, bytes;   // status: the call's own word, so calls may overlap
  Workspace(size_t n, size_t d_R, size_t h_kv) {
    pre = 0;
    dpre = pre + pad256(n * d_R * sizeof(float));
    w2f = dpre + pad256(n * d_R * sizeof(bf16));
    partial = w2f + pad256(d_R * h_kv * sizeof(float));
    ds = partial + pad256(rh_pre_num_tiles((int)d_R) * n * h_kv * sizeof(float));
    status = ds + pad256(n * h_kv * sizeof(float));
    bytes = status + pad256(sizeof(int));
  }
};

}  // namespace

#define TCK(call)                                                            \
  do {                                                                       \
    cudaError_t e__ = (call);                                                \
    if (e__ != cudaSuccess) { cudaGetLastError(); return LOCRET_ERR_CUDA; }  \
  } while (0)

static bool rh_sizes_ok(int32_t n, int32_t d_R, int32_t h_kv) {
  return n >= 64 && n % 64 == 0 && d_R >= 32 && d_R % 32 == 0 && h_kv >= 1 && h_kv <= 32;
}

extern "C" int locret_rh_loss_grad_workspace(int32_t n, int32_t d_R, int32_t h_kv, int64_t *bytes) {
  if (!bytes || !rh_sizes_ok(n, d_R, h_kv)) return LOCRET_ERR_INVALID;
  *bytes = (int64_t)Workspace(n, d_R, h_kv).bytes;
  return LOCRET_OK;
}

extern "C" int locret_rh_loss_grad_ws(const void *z, const float *labels, const void *w1, const void *w2, int32_t n,
                                      int32_t d_in, int32_t d_R, int32_t h_kv, float alpha, float *loss, float *d_w1,
                                      float *d_w2, void *workspace, int64_t workspace_bytes, void *stream) {
  if (!z || !labels || !w1 || !w2 || !loss || !d_w1 || !d_w2 || !workspace) return LOCRET_ERR_INVALID;
  if (!rh_sizes_ok(n, d_R, h_kv) || d_in < 64 || d_in % 64 || alpha < 0.f) return LOCRET_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(z) | reinterpret_cast<uintptr_t>(w1) | reinterpret_cast<uintptr_t>(d_w1) |
       reinterpret_cast<uintptr_t>(workspace)) & 15u)
    return LOCRET_ERR_INVALID;
  const Workspace ws(n, d_R, h_kv);
  if (workspace_bytes < (int64_t)ws.bytes) return LOCRET_ERR_CAPACITY;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char *base = static_cast<unsigned char *>(workspace);
  float *pre = (float *)(base + ws.pre), *w2f = (float *)(base + ws.w2f), *partial = (float *)(base + ws.partial),
        *ds = (float *)(base + ws.ds);
  bf16 *dpre = (bf16 *)(base + ws.dpre);
  int *d_status = (int *)(base + ws.status);
  rh_clear_kernel<<<(d_R * h_kv + 255) / 256, 256, 0, st>>>((const bf16 *)w2, w2f, d_w2, d_R * h_kv, loss, d_status);
  TCK(cudaGetLastError());
  // pre = z W1 (fp32) and the scores
  TCK(launch_rh_pre_tc((const bf16 *)z, d_in, (const bf16 *)w1, d_R, pre, w2f, partial, n, d_R, d_in, h_kv, d_status, st));
  rh_loss_kernel<<<(n * h_kv + 255) / 256, 256, 0, st>>>(partial, rh_pre_num_tiles(d_R), labels, ds, loss, n, h_kv, alpha);
  TCK(cudaGetLastError());
  const dim3 grid((d_R / 2 + DP_THREADS - 1) / DP_THREADS, n / DP_SLAB);
  if (h_kv <= 8) rh_dpre_dw2_kernel<8><<<grid, DP_THREADS, 0, st>>>(pre, ds, w2f, dpre, d_w2, d_R, h_kv);
  else rh_dpre_dw2_kernel<32><<<grid, DP_THREADS, 0, st>>>(pre, ds, w2f, dpre, d_w2, d_R, h_kv);
  TCK(cudaGetLastError());
  // dW1 [d_in x d_R] = z^T dpre
  TCK(launch_gemm_tn_f32((const bf16 *)z, d_in, dpre, d_R, d_w1, d_R, d_in, d_R, n, d_status, st));
  int status = 0;
  TCK(cudaMemcpyAsync(&status, d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  TCK(cudaStreamSynchronize(st));
  return status ? LOCRET_ERR_DEVICE_TIMEOUT : LOCRET_OK;
}

extern "C" int locret_rh_loss_grad(const void *z, const float *labels, const void *w1, const void *w2, int32_t n,
                                   int32_t d_in, int32_t d_R, int32_t h_kv, float alpha, float *loss,
                                   float *d_w1, float *d_w2, void *stream) {
  if (!rh_sizes_ok(n, d_R, h_kv)) return LOCRET_ERR_INVALID;
  // (the stream-ordered pool gives its memory back at every synchronisation: callers in a loop keep a workspace)
  const int64_t bytes = (int64_t)Workspace(n, d_R, h_kv).bytes;
  void *ws = nullptr;
  if (cudaMallocAsync(&ws, (size_t)bytes, (cudaStream_t)stream) != cudaSuccess) { cudaGetLastError(); return LOCRET_ERR_ALLOC; }
  const int rc = locret_rh_loss_grad_ws(z, labels, w1, w2, n, d_in, d_R, h_kv, alpha, loss, d_w1, d_w2, ws, bytes, stream);
  if (cudaFreeAsync(ws, (cudaStream_t)stream) != cudaSuccess) { cudaGetLastError(); return rc ? rc : LOCRET_ERR_CUDA; }
  return rc;
}

// ---------------------------------------------------------------- AdamW (Appendix A, training)
namespace {
struct AdamW { float lr, beta1, beta2, eps, wd, bc1, bc2; };

__device__ __forceinline__ float adamw_one(float p, float g, float &m, float &v, const AdamW &a) {
  m = a.beta1 * m + (1.0f - a.beta1) * g;
  v = a.beta2 * v + (1.0f - a.beta2) * g * g;
  return p * (1.0f - a.lr * a.wd) - a.lr * (m / a.bc1) / (sqrtf(v / a.bc2) + a.eps);
}

// Bound by memory (30 bytes per parameter with the bf16 copy): four parameters per thread with 16-byte accesses where
// every array is aligned for them (vec), one otherwise and in the remainder.
__global__ void adamw_kernel(float *__restrict__ p, bf16 *__restrict__ p_bf16, const float *__restrict__ g,
                             float *__restrict__ m, float *__restrict__ v, size_t n, AdamW a, int vec) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec && 4 * i + 4 <= n) {
    float4 pp = reinterpret_cast<float4 *>(p)[i], mm = reinterpret_cast<float4 *>(m)[i],
           vv = reinterpret_cast<float4 *>(v)[i];
    const float4 gg = reinterpret_cast<const float4 *>(g)[i];
    pp.x = adamw_one(pp.x, gg.x, mm.x, vv.x, a);
    pp.y = adamw_one(pp.y, gg.y, mm.y, vv.y, a);
    pp.z = adamw_one(pp.z, gg.z, mm.z, vv.z, a);
    pp.w = adamw_one(pp.w, gg.w, mm.w, vv.w, a);
    reinterpret_cast<float4 *>(m)[i] = mm;
    reinterpret_cast<float4 *>(v)[i] = vv;
    reinterpret_cast<float4 *>(p)[i] = pp;
    if (p_bf16) reinterpret_cast<uint2 *>(p_bf16)[i] = make_uint2(pack_bf16(pp.x, pp.y), pack_bf16(pp.z, pp.w));
    return;
  }
  const size_t lo = vec ? 4 * i : i, hi = vec ? n : (i < n ? i + 1 : 0);
  for (size_t k = lo; k < hi; k++) {
    float mk = m[k], vk = v[k];
    const float pk = adamw_one(p[k], g[k], mk, vk, a);
    m[k] = mk;
    v[k] = vk;
    p[k] = pk;
    if (p_bf16) p_bf16[k] = __float2bfloat16_rn(pk);
  }
}
}  // namespace

extern "C" int locret_adamw_step(float *param, void *param_bf16, const float *grad, float *m, float *v, int64_t n,
                                 int32_t step, float lr, float beta1, float beta2, float eps, float weight_decay,
                                 void *stream) {
  if (!param || !grad || !m || !v || n < 1 || step < 1) return LOCRET_ERR_INVALID;
  if (!(beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f && beta2 < 1.f) || eps <= 0.f) return LOCRET_ERR_INVALID;
  const float bc1 = 1.0f - powf(beta1, (float)step), bc2 = 1.0f - powf(beta2, (float)step);
  const AdamW a = {lr, beta1, beta2, eps, weight_decay, bc1, bc2};
  const uintptr_t bits = reinterpret_cast<uintptr_t>(param) | reinterpret_cast<uintptr_t>(grad) |
                         reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v);
  const int vec = (bits & 15u) == 0 && (reinterpret_cast<uintptr_t>(param_bf16) & 7u) == 0;
  const size_t threads = vec ? ((size_t)n + 3) / 4 : (size_t)n;
  adamw_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, (cudaStream_t)stream>>>(param, (bf16 *)param_bf16, grad, m, v,
                                                                                   (size_t)n, a, vec);
  TCK(cudaGetLastError());
  return LOCRET_OK;
}

// Decoding (the B = 1 case of Eq. 1): one token per step, so the bytes that a kernel must read once bound it, the weights
// for the two projections and the retained keys and values for attention, and the latency of its phases.  The projections are
// dot products on the CUDA cores with 16-byte loads; attention has a small contraction to tile, the query heads of a
// group (header of each attention kernel); over a 4-bit cache the work on the codes counts more than their bytes.
#include <stdlib.h>

#include <type_traits>

#include "common.cuh"

namespace locret {

namespace {

__device__ __forceinline__ float dot8(const uint4 &a, const uint4 &b) {
  const __nv_bfloat162 *x = reinterpret_cast<const __nv_bfloat162 *>(&a);
  const __nv_bfloat162 *y = reinterpret_cast<const __nv_bfloat162 *>(&b);
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const float2 xf = __bfloat1622float2(x[i]), yf = __bfloat1622float2(y[i]);
    s = fmaf(xf.x, yf.x, s);
    s = fmaf(xf.y, yf.y, s);
  }
  return s;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

constexpr int GV_THREADS = 256;

// y[n] = sum_k Wt[n][k] x[k]; one warp per output row, rows strided over the grid.
// MODE 0: bf16 store with a residual.  MODE 1 (retaining head): hidden = act(y[n]); every warp keeps
// sum_n hidden * W2[n][m] and the block writes one partial score per KV head.
// The block that finishes last (counted with a wrapping atomic, so the counter is zero again
// afterwards) adds the per-block partials in block order: deterministic, and no second launch.
template <int MODE, int NL>
__global__ void __launch_bounds__(GV_THREADS)
gemv_kernel(const bf16 *__restrict__ x, const bf16 *__restrict__ Wt, int N, int K, bf16 *__restrict__ y,
            const bf16 *__restrict__ resid, int h_kv, int act, const __grid_constant__ RhGemvBatchN<NL> b) {
  // (MODE 1: blockIdx.y = layer)
  const float *__restrict__ W2 = nullptr;
  float *__restrict__ partial = nullptr, *__restrict__ score_out = nullptr;
  unsigned *__restrict__ counter = nullptr;
  int score_stride = 0;
  if (MODE == 1) {
    const RhGemvLayer &l = b.l[NL == 1 ? 0 : blockIdx.y];
    x = l.z; Wt = l.W1t; W2 = l.W2; partial = l.partial; score_out = l.score_out; counter = l.counter;
    score_stride = l.score_stride;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4 *sx = reinterpret_cast<uint4 *>(smem_raw);  // K / 8 vectors
  float *swarp = reinterpret_cast<float *>(sx + K / 8);  // [8 warps][32]
  // MODE 1 in a one-token step's chain: the input is the projection's output, complete since the
  // attention kernel before this one passed its own wait, so nothing is waited for here; the next
  // layer's projection may start (and request its weights) at once
  if (MODE == 1) pdl_launch_dependents();
  for (int i = threadIdx.x; i < K / 8; i += GV_THREADS) sx[i] = reinterpret_cast<const uint4 *>(x)[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = blockIdx.x * (GV_THREADS / 32) + warp, nw = gridDim.x * (GV_THREADS / 32);
  float score = 0.f;  // MODE 1: lane m < h_kv accumulates head m
  if (MODE == 0) {
    for (int n = gw; n < N; n += nw) {
      const uint4 *row = reinterpret_cast<const uint4 *>(Wt + (size_t)n * K);
      float s = 0.f;
#pragma unroll 8
      for (int v = lane; v < K / 8; v += 32) s += dot8(__ldg(row + v), sx[v]);
      s = warp_sum(s);
      if (lane == 0) y[n] = __float2bfloat16_rn(s + __bfloat162float(resid[n]));
    }
  } else {
    // two warps per row (halves of K), four rows per block at a time: d_R rows are too few to
    // keep enough loads in flight with one warp per row
    __shared__ float shalf[GV_THREADS / 32];
    const int kv2 = K / 16;  // vectors per half row
    for (int n0 = blockIdx.x * 4; n0 < N; n0 += gridDim.x * 4) {
      const int n = n0 + (warp >> 1), hf = warp & 1;
      float s = 0.f;
      if (n < N) {
        const uint4 *row = reinterpret_cast<const uint4 *>(Wt + (size_t)n * K) + hf * kv2;
        const uint4 *xs = sx + hf * kv2;
#pragma unroll 12
        for (int v = lane; v < kv2; v += 32) s += dot8(__ldg(row + v), xs[v]);
      }
      s = warp_sum(s);
      if (lane == 0) shalf[warp] = s;
      __syncthreads();
      if (hf == 0 && n < N) {
        const float hdn = apply_act(shalf[warp] + shalf[warp + 1], act);
        if (lane < h_kv) score = fmaf(hdn, W2[(size_t)n * h_kv + lane], score);
      }
      __syncthreads();
    }
  }
  if (MODE == 1) {
    swarp[warp * 32 + lane] = score;
    __syncthreads();
    if (warp == 0 && lane < h_kv) {
      float t = 0.f;
      for (int w = 0; w < GV_THREADS / 32; w++) t += swarp[w * 32 + lane];
      partial[(size_t)blockIdx.x * h_kv + lane] = t;  // layout [block][token 0][head]
    }
    if (counter) {
      __shared__ bool last;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) last = atomicInc(counter, gridDim.x - 1) == gridDim.x - 1;
      __syncthreads();
      if (last) {
        __threadfence();
        // warp w sums heads w, w + 8, ...: lanes stride over the blocks, then a shuffle tree
        // (a fixed order, so the sum does not depend on which block came last)
        for (int m = warp; m < h_kv; m += GV_THREADS / 32) {
          float t = 0.f;
          for (unsigned b = lane; b < gridDim.x; b += 32) t += __ldcg(partial + (size_t)b * h_kv + m);
          t = warp_sum(t);
          if (lane == 0) score_out[(size_t)m * score_stride] = t;
        }
      }
    }
    // the attention kernel of this step must have finished before the next layer's projection (which
    // waits for THIS kernel) overwrites the buffers attention reads
    pdl_wait();
  }
}

// Elements i and i + d/2 of head hd of the token's projection: staging, position (= slot), RoPE from the bf16-rounded
// values (what the pre-RoPE cache stores), append.
__device__ __forceinline__ void rope_append_pair(const RopeAppendArgs &a, bf16 *staging, int hd, int i, bf16 b0, bf16 b1) {
  const int half = a.d / 2, n0 = hd * a.d + i, n1 = n0 + half, slot = a.len;
  staging[n0] = b0;
  staging[n1] = b1;
  if (hd < a.h + a.h_kv) {
    const float2 t = a.cs[(size_t)slot * half + i];
    const float x0 = __bfloat162float(b0), x1 = __bfloat162float(b1);
    // lower half: x1 cos − x2 sin ; upper half: x2 cos + x1 sin
    const bf16 q0 = __float2bfloat16_rn(x0 * t.x - x1 * t.y), q1 = __float2bfloat16_rn(x1 * t.x + x0 * t.y);
    if (hd < a.h) {
      a.q_rot[n0] = q0;
      a.q_rot[n1] = q1;
    } else {
      const int m = hd - a.h;
      const size_t off = ((size_t)m * a.cap + slot) * a.d + i;
      if (a.k_pre) { a.k_pre[off] = b0; a.k_pre[off + half] = b1; }  // null for a 4-bit cache
      bf16 *k = a.tok_k ? a.tok_k + (size_t)m * a.d + i : a.k_rot + off;
      k[0] = q0;
      k[half] = q1;
      if (i == 0) a.tid[(size_t)m * a.cap + slot] = a.seen;
    }
    if (a.z_post) { a.z_post[n0] = q0; a.z_post[n1] = q1; }
  } else {
    const int m = hd - a.h - a.h_kv;
    bf16 *v = a.tok_v ? a.tok_v + (size_t)m * a.d + i : a.v + ((size_t)m * a.cap + slot) * a.d + i;
    v[0] = b0;
    v[half] = b1;
    if (a.z_post) { a.z_post[n0] = b0; a.z_post[n1] = b1; }
  }
}

// Projection of one token with positions, RoPE and cache append: a warp computes the two rows
// (i, i + d/2) of one head, so it holds a whole rotation pair.  The rotation starts from the
// bf16-rounded projection, the value the pre-RoPE cache stores.
__global__ void __launch_bounds__(GV_THREADS)
gemv_rope_kernel(const bf16 *__restrict__ x, const bf16 *__restrict__ Wt, int K, bf16 *__restrict__ staging,
                 RopeAppendArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4 *sx = reinterpret_cast<uint4 *>(smem_raw);  // K / 8 vectors
  pdl_wait();
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < K / 8; i += GV_THREADS) sx[i] = reinterpret_cast<const uint4 *>(x)[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = blockIdx.x * (GV_THREADS / 32) + warp, nw = gridDim.x * (GV_THREADS / 32);
  const int half = a.d / 2, heads = a.h + 2 * a.h_kv;
  for (int it = gw; it < heads * half; it += nw) {
    const int hd = it / half, i = it - hd * half;
    const int n0 = hd * a.d + i, n1 = n0 + half;
    const uint4 *r0 = reinterpret_cast<const uint4 *>(Wt + (size_t)n0 * K);
    const uint4 *r1 = reinterpret_cast<const uint4 *>(Wt + (size_t)n1 * K);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
    for (int v = lane; v < K / 8; v += 32) {
      const uint4 xv = sx[v];
      s0 += dot8(__ldg(r0 + v), xv);
      s1 += dot8(__ldg(r1 + v), xv);
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane == 0) rope_append_pair(a, staging, hd, i, __float2bfloat16_rn(s0), __float2bfloat16_rn(s1));
  }
}

// The same projection for K <= 4096 laid out for bandwidth, for one layer or for the layers of a stack that share
// the input: the rotation pairs of all layers are one range, a block of 512 threads owns a contiguous part of it,
// thread t holds element group t of x in registers (no staging step before the first weight load) and reads
// group t of both rows of four pairs at a time, so a block has 64 KB of weights in flight and two blocks per SM
// cover each other's reductions.  The eight partial sums of a batch are reduced with one butterfly that halves the
// number of values at each step (9 shuffles instead of 40), then across the warps through shared memory.
constexpr int GW_THREADS = 512, GW_PB = 4;

template <int NL>
__global__ void __launch_bounds__(GW_THREADS, 2)
gemv_rope_wide_kernel(const bf16 *__restrict__ x, int K, int n_layers, const __grid_constant__ GemvRopeBatchN<NL> b) {
  __shared__ float red[2][GW_THREADS / 32][2 * GW_PB];
  __shared__ float res[2][2 * GW_PB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kv = K / 8;
  const bool act = tid < kv;
  const int h = b.a[0].h, h_kv = b.a[0].h_kv, d = b.a[0].d;  // (the same in every layer)
  const int half = d / 2, heads = h + 2 * h_kv;
  const int per_layer = heads * half, n_pairs = (NL == 1 ? 1 : n_layers) * per_layer;
  const int p_lo = (int)((long long)blockIdx.x * n_pairs / gridDim.x);
  const int p_hi = (int)((long long)(blockIdx.x + 1) * n_pairs / gridDim.x);
  // the first batch of weights is requested before x
  uint4 w[2 * GW_PB];
  auto load_batch = [&](int p0) {
#pragma unroll
    for (int j = 0; j < GW_PB; j++) {
      int it = min(p0 + j, n_pairs - 1);
      const int layer = NL == 1 ? 0 : it / per_layer;
      it -= layer * per_layer;
      const uint4 *W4 = reinterpret_cast<const uint4 *>(b.Wt[layer]);
      const int hd = it / half, i = it - hd * half;
      const size_t n0 = (size_t)hd * d + i;
      w[2 * j] = act ? __ldg(W4 + n0 * kv + tid) : make_uint4(0, 0, 0, 0);
      w[2 * j + 1] = act ? __ldg(W4 + (n0 + half) * kv + tid) : make_uint4(0, 0, 0, 0);
    }
  };
  load_batch(p_lo);
  // the weights do not depend on anything before this kernel: the first batch is in flight while the
  // kernel waits for the step before it (whose buffers it is about to overwrite).  The attention
  // kernel may start only after that wait: it requests retained keys before its own, and an
  // eviction of the previous step may still be rewriting them until then.
  pdl_wait();
  pdl_launch_dependents();
  const uint4 xv = act ? __ldg(reinterpret_cast<const uint4 *>(x) + tid) : make_uint4(0, 0, 0, 0);
  int par = 0;
  for (int p0 = p_lo; p0 < p_hi; p0 += GW_PB, par ^= 1) {
    // dot8 of both rows of a pair at a time: the same rounded sums in half the FMAs, and x is converted once per batch.  What counts
    // is how soon after a batch's arrival the next one is requested (four Llama layers of 200 units, a step: 59.4 us row by
    // row, 55.4 in pairs, 55.1 by m16n8k16 tiles; but those truncate their sums, which came out 3e-8 of them too small).
    float v[2 * GW_PB];
    {
      uint64_t s[GW_PB] = {};
      const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const float x0 = __uint_as_float(xw[i] << 16), x1 = __uint_as_float(xw[i] & 0xffff0000u);
        const uint64_t xx0 = pack_f32x2(x0, x0), xx1 = pack_f32x2(x1, x1);
#pragma unroll
        for (int j = 0; j < GW_PB; j++) {
          const uint32_t wa = reinterpret_cast<const uint32_t *>(&w[2 * j])[i], wb = reinterpret_cast<const uint32_t *>(&w[2 * j + 1])[i];
          s[j] = fma_f32x2(pack_f32x2(__uint_as_float(wa << 16), __uint_as_float(wb << 16)), xx0, s[j]);
          s[j] = fma_f32x2(pack_f32x2(__uint_as_float(wa & 0xffff0000u), __uint_as_float(wb & 0xffff0000u)), xx1, s[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < GW_PB; j++) unpack_f32x2(s[j], v[2 * j], v[2 * j + 1]);
    }
    if (p0 + GW_PB < p_hi) load_batch(p0 + GW_PB);  // in flight during the reduction
    // eight values across 32 lanes: exchange half of them at each of three steps
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const float send = (lane & 16) ? v[e] : v[e + 4], keep = (lane & 16) ? v[e + 4] : v[e];
      v[e] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int e = 0; e < 2; e++) {
      const float send = (lane & 8) ? v[e] : v[e + 2], keep = (lane & 8) ? v[e + 2] : v[e];
      v[e] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    {
      const float send = (lane & 4) ? v[0] : v[1], keep = (lane & 4) ? v[1] : v[0];
      v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    if ((lane & 3) == 0) red[par][warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = v[0];
    __syncthreads();
    if (tid < 2 * GW_PB) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < GW_THREADS / 32; q++) t += red[par][q][tid];
      res[par][tid] = t;
    }
    __syncthreads();
    if (tid < GW_PB && p0 + tid < p_hi) {
      const int layer = NL == 1 ? 0 : (p0 + tid) / per_layer, it = p0 + tid - layer * per_layer;
      const int hd = it / half;
      const RopeAppendArgs &a = b.a[layer];
      rope_append_pair(a, const_cast<bf16 *>(a.staging), hd, it - hd * half, __float2bfloat16_rn(res[par][2 * tid]),
                       __float2bfloat16_rn(res[par][2 * tid + 1]));
    }
  }
}

// ---- decode attention on warp-level tensor-core instructions.  grid (h_kv, splits, head groups
// of <= 16).  The rows of the m16n8k16 tiles are the query heads of one GQA group (all of them read
// the same keys), padded to 16; keys and values of the split stream through shared memory in
// tiles of 64 (cp.async, two stages).  Each of the four warps takes 16 keys of a tile and keeps
// its own running maximum, sum and output, so the tile loop has no block-wide reduction; the
// four states meet in shared memory at the end, the block writes one partial result per head,
// and the split that finishes last for its (KV head, head group) merges all splits in split
// order (a wrapping atomic counter, left at zero for the next step).
constexpr int DA_THREADS = 128, DA_G = 16, DA_KT = 64;

template <int D, int NL>
__global__ void __launch_bounds__(DA_THREADS, 4)
attn_decode_kernel(int h, int h_kv, float scale_log2, const __grid_constant__ DecodeAttnBatchN<NL> batch) {
  const int hgroups = (h / h_kv + DA_G - 1) / DA_G, layer = NL == 1 ? 0 : blockIdx.z / hgroups;
  const DecodeAttnLayer &a = batch.l[layer];
  const bf16 *__restrict__ q_rot = a.q_rot, *__restrict__ k_rot = a.k_rot, *__restrict__ v = a.v;
  float *__restrict__ part_o = a.part_o, *__restrict__ part_ml = a.part_ml;
  const int cap = a.cap, n = a.n, n_splits = a.n_splits;
  constexpr int LD = D + 8;
  constexpr int VPR = D / 8;  // 16-byte vectors per row
  extern __shared__ __align__(16) unsigned char da_smem[];
  bf16 *sQ = reinterpret_cast<bf16 *>(da_smem);  // [16][LD]
  bf16 *sK = sQ + DA_G * LD;                     // [2][64][LD]
  bf16 *sV = sK + 2 * DA_KT * LD;                // [2][64][LD]
  __shared__ float wm[4][DA_G], wl[4][DA_G];     // per-warp running maximum and sum of every head
  __shared__ float sm[DA_G][64], sl[DA_G][64], sinv[DA_G];
  __shared__ bool last;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g4 = lane >> 2, q = lane & 3;
  const int g = h / h_kv;
  const int m = blockIdx.x, split = blockIdx.y, hg = blockIdx.z - layer * hgroups;
  if (NL > 1 && split >= n_splits) return;  // (layers of a batch may hold different numbers of keys)
  const int h0 = m * g + hg * DA_G;
  const int gh = min(DA_G, g - hg * DA_G);  // heads handled here
  const int per = (n + n_splits - 1) / n_splits;
  const int k0 = split * per, k1 = min(n, k0 + per);
  const int NKT = k1 > k0 ? (k1 - k0 + DA_KT - 1) / DA_KT : 0;
  const bf16 *kbase = k_rot + (size_t)m * cap * D;
  const bf16 *vbase = v + (size_t)m * cap * D;

  auto load_kv = [&](int buf, int kt) {
    for (int x = tid; x < DA_KT * VPR; x += DA_THREADS) {
      const int r = x / VPR, c = (x - r * VPR) * 8;
      const int key = k0 + kt * DA_KT + r;
      const bool ok = key < k1;
      const size_t off = (size_t)min(key, n - 1) * D + c;
      cp_async16(sK + (buf * DA_KT + r) * LD + c, kbase + off, ok);
      cp_async16(sV + (buf * DA_KT + r) * LD + c, vbase + off, ok);
    }
  };
  // The retained keys and values were written by earlier steps: a first tile that does not reach
  // the token of this step is requested before the wait for this step's projection.
  const bool early = NKT > 0 && k0 + DA_KT <= n - 1;
  if (early) load_kv(0, 0);
  pdl_wait();
  pdl_launch_dependents();  // the retaining head reads only what the projection wrote: it may run beside this kernel
  for (int x = tid; x < DA_G * VPR; x += DA_THREADS) {
    const int r = x / VPR, c = (x - r * VPR) * 8;
    cp_async16(sQ + r * LD + c, q_rot + (size_t)(h0 + min(r, gh - 1)) * D + c, r < gh);
  }
  if (NKT > 0 && !early) load_kv(0, 0);
  cp_async_commit();

  uint32_t qf[D / 16][4];
  float o[D / 8][4];
#pragma unroll
  for (int i = 0; i < D / 8; i++)
#pragma unroll
    for (int e = 0; e < 4; e++) o[i][e] = 0.f;
  float mrow[2] = {-INFINITY, -INFINITY}, lrow[2] = {0.f, 0.f};  // heads g4 and g4 + 8

  for (int kt = 0; kt < NKT; kt++) {
    if (kt + 1 < NKT) load_kv((kt + 1) & 1, kt + 1);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    if (kt == 0) {
#pragma unroll
      for (int kk = 0; kk < D / 16; kk++)
        ldmatrix_x4(qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3],
                    sQ + (lane & 15) * LD + kk * 16 + (lane >> 4) * 8);
    }
    const bf16 *k_s = sK + ((kt & 1) * DA_KT + warp * 16) * LD;  // this warp's 16 keys
    const bf16 *v_s = sV + ((kt & 1) * DA_KT + warp * 16) * LD;

    float s[2][4];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int e = 0; e < 4; e++) s[i][e] = 0.f;
#pragma unroll
    for (int kk = 0; kk < D / 16; kk++) {
      uint32_t b0, b1, b2, b3;
      const int id = lane >> 3;
      const int r = (id >> 1) * 8 + (lane & 7);
      const int c = kk * 16 + (id & 1) * 8;
      ldmatrix_x4(b0, b1, b2, b3, k_s + r * LD + c);
      mma_bf16_16816(s[0], qf[kk], b0, b1);
      mma_bf16_16816(s[1], qf[kk], b2, b3);
    }

    // scale, mask the keys past the split's end, online softmax of this warp's 16 keys
    const int key0 = k0 + kt * DA_KT + warp * 16;
    float tmax[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int e = 0; e < 4; e++) {
        float val = s[i][e] * scale_log2;
        if (key0 + i * 8 + q * 2 + (e & 1) >= k1) val = -INFINITY;
        s[i][e] = val;
        tmax[e >> 1] = fmaxf(tmax[e >> 1], val);
      }
    float alpha[2];
#pragma unroll
    for (int r = 0; r < 2; r++) {
      tmax[r] = fmaxf(tmax[r], __shfl_xor_sync(0xffffffffu, tmax[r], 1));
      tmax[r] = fmaxf(tmax[r], __shfl_xor_sync(0xffffffffu, tmax[r], 2));
      const float mnew = fmaxf(mrow[r], tmax[r]);
      const float muse = (mnew == -INFINITY) ? 0.f : mnew;
      alpha[r] = exp2f(mrow[r] - muse);
      mrow[r] = mnew;
      float psum = 0.f;
#pragma unroll
      for (int i = 0; i < 2; i++) {
        const float p0 = exp2f(s[i][2 * r] - muse), p1 = exp2f(s[i][2 * r + 1] - muse);
        s[i][2 * r] = p0;
        s[i][2 * r + 1] = p1;
        psum += p0 + p1;
      }
      lrow[r] = lrow[r] * alpha[r] + psum;
    }
#pragma unroll
    for (int i = 0; i < D / 8; i++) {
      o[i][0] *= alpha[0]; o[i][1] *= alpha[0];
      o[i][2] *= alpha[1]; o[i][3] *= alpha[1];
    }
    // O += P V over this warp's 16 keys
    uint32_t pf[4];
    pf[0] = pack_bf16(s[0][0], s[0][1]);
    pf[1] = pack_bf16(s[0][2], s[0][3]);
    pf[2] = pack_bf16(s[1][0], s[1][1]);
    pf[3] = pack_bf16(s[1][2], s[1][3]);
#pragma unroll
    for (int dn = 0; dn < D / 16; dn++) {
      uint32_t b0, b1, b2, b3;
      const int id = lane >> 3;
      const int r = (id & 1) * 8 + (lane & 7);
      const int c = dn * 16 + (id >> 1) * 8;
      ldmatrix_x4_trans(b0, b1, b2, b3, v_s + r * LD + c);
      mma_bf16_16816(o[2 * dn], pf, b0, b1);
      mma_bf16_16816(o[2 * dn + 1], pf, b2, b3);
    }
    __syncthreads();  // the next iteration's cp.async refills the buffer read here
  }
  cp_async_wait<0>();

  // ---- the four warps' states meet: fo[warp][head][column] in the tile buffers
#pragma unroll
  for (int r = 0; r < 2; r++) {
    lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 1);
    lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 2);
    if (q == 0) { wm[warp][g4 + 8 * r] = mrow[r]; wl[warp][g4 + 8 * r] = lrow[r]; }
  }
  constexpr int LF = D + 8;                   // (rows of eight lanes then spread over the banks)
  float *fo = reinterpret_cast<float *>(sK);  // [4][16][LF] floats = 34 KB at D = 128 <= the tile buffers
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 2; r++)
    if (g4 + 8 * r < gh) {  // (the rest of the 16 rows is padding)
#pragma unroll
      for (int i = 0; i < D / 8; i++)
        *reinterpret_cast<float2 *>(fo + (warp * DA_G + g4 + 8 * r) * LF + i * 8 + q * 2) =
            make_float2(o[i][2 * r], o[i][2 * r + 1]);
    }
  __syncthreads();
  // partial result of this split: o [h][split][D] (not normalised), (m, l) [h][split][2]
  for (int idx = tid; idx < gh * D; idx += DA_THREADS) {
    const int i = idx / D, c = idx - i * D;
    const float mx = fmaxf(fmaxf(wm[0][i], wm[1][i]), fmaxf(wm[2][i], wm[3][i]));
    float acc = 0.f, l = 0.f;
#pragma unroll
    for (int w = 0; w < 4; w++) {
      const float wgt = (wm[w][i] == -INFINITY) ? 0.f : exp2f(wm[w][i] - mx);
      acc = fmaf(wgt, fo[(w * DA_G + i) * LF + c], acc);
      l = fmaf(wgt, wl[w][i], l);
    }
    const size_t hs = (size_t)(h0 + i) * n_splits + split;
    part_o[hs * D + c] = acc;
    if (c == 0) { part_ml[hs * 2] = mx; part_ml[hs * 2 + 1] = l; }
  }

  // ---- the split that finishes last merges the partial results of all splits
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicInc(&a.counters[m * hgroups + hg], n_splits - 1) == (unsigned)(n_splits - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int idx = tid; idx < gh * n_splits; idx += DA_THREADS) {
    const int i = idx / n_splits, s2 = idx - i * n_splits;
    const size_t hs = (size_t)(h0 + i) * n_splits + s2;
    sm[i][s2] = __ldcg(part_ml + hs * 2);
    sl[i][s2] = __ldcg(part_ml + hs * 2 + 1);
  }
  __syncthreads();
  // weights of the splits: one warp per head at a time, the splits across its lanes
  for (int i = warp; i < gh; i += DA_THREADS / 32) {
    float mx = -INFINITY;
    for (int s2 = lane; s2 < n_splits; s2 += 32) mx = fmaxf(mx, sm[i][s2]);
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o2));
    float l = 0.f;
    for (int s2 = lane; s2 < n_splits; s2 += 32) {
      const float ms = sm[i][s2];
      const float w = (ms == -INFINITY) ? 0.f : exp2f(ms - mx);
      l = fmaf(w, sl[i][s2], l);
      sm[i][s2] = w;
    }
    // (fixed order of the partial sums: lanes, then the butterfly)
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o2);
    if (lane == 0) sinv[i] = 1.0f / l;
  }
  __syncthreads();
  // thread = (head, four columns); sixteen splits in flight as 16-byte loads
  for (int item = tid; item < gh * (D / 4); item += DA_THREADS) {
    const int i = item / (D / 4), c = (item - i * (D / 4)) * 4;
    const float *po = part_o + (size_t)(h0 + i) * n_splits * D + c;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s2 = 0; s2 < n_splits; s2 += 16) {
      float4 a[16];
#pragma unroll
      for (int u = 0; u < 16; u++)
        a[u] = (s2 + u < n_splits) ? __ldcg(reinterpret_cast<const float4 *>(po + (size_t)(s2 + u) * D))
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 16; u++)
        if (s2 + u < n_splits) {
          const float w = sm[i][s2 + u];
          acc.x = fmaf(w, a[u].x, acc.x); acc.y = fmaf(w, a[u].y, acc.y);
          acc.z = fmaf(w, a[u].z, acc.z); acc.w = fmaf(w, a[u].w, acc.w);
        }
    }
    const float inv = sinv[i];
    uint2 o2;
    o2.x = pack_bf16(acc.x * inv, acc.y * inv);
    o2.y = pack_bf16(acc.z * inv, acc.w * inv);
    *reinterpret_cast<uint2 *>(a.out + (size_t)(h0 + i) * D + c) = o2;
  }
}

// ---- the same over a 4-bit cache.  What bounds it is not bytes (8.6 KB for 64 units of a head) but the work on them: codes to
// floats, the rotation of every key at its own position, and the latency of the (cos, sin) rows that needs.  So nothing
// passes through shared memory and no warp waits for another inside the loop: a warp takes 16 keys of every tile of 64, and a
// lane expands and rotates exactly the elements that its operand fragments hold.  For that, keys are the m side of the
// m16n8k16 tiles and the query heads the n side (NT tiles of eight): S^T = K Q^T, O^T = V^T P^T, with an 8 x 8 transpose of
// P between them.  The codes, scales and ranks of a warp's next 16 keys are on their way while it works on these.
//   Which elements a step of a contraction takes, and in which order the keys stand, is free as long as both operands agree:
// a step takes the lower or the upper elements of 16 rotation pairs (a lane: pairs 2 q, 2 q + 1 and the same + 8, so that
// the four lanes of a row read whole sectors of its (cos, sin)); row r of S^T is key kr(r), and columns of O are dealt
// to the lanes in runs of D / 8, so that a lane's value codes lie together.
// Measured (span of the launch for four Llama layers, 6000 units each): 84 us with tiles expanded into shared memory by
// threads that each took 16 elements of a key (4150 instructions a warp, conversions among them), 64 us this way, both with two
// blocks for each SM.  With the splits of decode_attn_splits a step of four layers with such heads and d_model 1024 takes 71 us,
// 101 then.
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
// Code J of a word -> 16^J * code: the nibble (its sign bit flipped: code + 8) in the mantissa of 2^23, less 2^23 + 8 * 16^J;
// exact.  (No conversion instruction: those have a fraction of the rate.)  Times scale / 16^J it is code * scale, rounded once.
template <int J>
__device__ __forceinline__ float q4_code(uint32_t w) {
  return __uint_as_float((w & (0xFu << (4 * J))) ^ (0x4B000000u | (8u << (4 * J)))) - (8388608.f + (float)(8 << (4 * J)));
}
// four codes in bits 0-15
__device__ __forceinline__ void q4_expand4(uint32_t w, float s, float (&x)[4]) {
  x[0] = q4_code<0>(w) * s;
  x[1] = q4_code<1>(w) * (s * 0x1p-4f);
  x[2] = q4_code<2>(w) * (s * 0x1p-8f);
  x[3] = q4_code<3>(w) * (s * 0x1p-12f);
}

template <int D, int NL, int NT>
__global__ void __launch_bounds__(DA_THREADS, 2)
attn_decode_q4_kernel(int h, int h_kv, float scale_log2, const __grid_constant__ DecodeAttnBatchN<NL> batch) {
  constexpr int G = 8 * NT;
  const int hgroups = (h / h_kv + G - 1) / G, layer = NL == 1 ? 0 : blockIdx.z / hgroups;
  const DecodeAttnLayer &a = batch.l[layer];
  const int cap = a.cap, n = a.n, n_splits = a.n_splits, ranked_len = a.ranked_len;
  const Int4Half &q4 = a.q4;
  constexpr int LF = D + 8, NW = D / 16;   // NW: words of a row's lower (or upper) codes
  __shared__ __align__(16) float fo[4][G][LF];
  __shared__ float wm[4][G], wl[4][G], sw[G][64], sinv[G];
  __shared__ uint2 sq[NT > 1 ? D / 16 * NT : 1][32];   // two tiles: fragments of the queries, for which no registers are left
  __shared__ bool last;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g4 = lane >> 2, q = lane & 3;
  const int g = h / h_kv, m = blockIdx.x, split = blockIdx.y, hg = blockIdx.z - layer * hgroups;
  if (NL > 1 && split >= n_splits) return;  // (layers of a batch may hold different numbers of keys)
  const int h0 = m * g + hg * G, gh = min(G, g - hg * G);
  const int per = (n + n_splits - 1) / n_splits, k0 = split * per, k1 = min(n, k0 + per);
  const int NKT = k1 > k0 ? (k1 - k0 + DA_KT - 1) / DA_KT : 0;
  // keys of this lane in its warp's 16: two rows of S^T (kr and 8 + kr), four columns of V^T
  const int kr = (g4 >> 1) + 4 * (g4 & 1);

  struct Tile {
    uint32_t kw[2][2][NW];   // rows, lower / upper
    uint32_t vw[4][2];       // (D / 8 codes: 16, 12 or 8)
    float ks[2], vs[4];
    int pos[2];
  };
  auto fetch = [&](int kt, Tile &t) {   // unit n - 1, the token of this step, is not in the codes
    const int base = k0 + kt * DA_KT + warp * 16;
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const int key = base + 8 * r + kr;
      const bool ok = key < min(k1, n - 1);
      const size_t u = (size_t)m * cap + (ok ? key : 0);
      t.ks[r] = ok ? __half2float(q4.ks[u]) : 0.f;
      t.pos[r] = !ok ? 0 : (key < ranked_len ? a.rank[u] : key);
#pragma unroll
      for (int hf = 0; hf < 2; hf++) {
        const uint8_t *c = q4.kq + u * (D / 2) + hf * (D / 4);
        if constexpr (D == 96) {
#pragma unroll
          for (int i = 0; i < 3; i++) {
            const uint2 v = ok ? *reinterpret_cast<const uint2 *>(c + 8 * i) : make_uint2(0, 0);
            t.kw[r][hf][2 * i] = v.x; t.kw[r][hf][2 * i + 1] = v.y;
          }
        } else {
#pragma unroll
          for (int i = 0; i < D / 64; i++) {
            const uint4 v = ok ? *reinterpret_cast<const uint4 *>(c + 16 * i) : make_uint4(0, 0, 0, 0);
            t.kw[r][hf][4 * i] = v.x; t.kw[r][hf][4 * i + 1] = v.y; t.kw[r][hf][4 * i + 2] = v.z; t.kw[r][hf][4 * i + 3] = v.w;
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {   // the keys of S^T rows 2 q, 2 q + 1, 2 q + 8, 2 q + 9
      const int key = base + q + 4 * i;
      const bool ok = key < min(k1, n - 1);
      const size_t u = (size_t)m * cap + (ok ? key : 0);
      t.vs[i] = ok ? __half2float(q4.vs[u]) : 0.f;
      const uint8_t *c = q4.vq + u * (D / 2) + (D / 16) * g4;
      t.vw[i][0] = t.vw[i][1] = 0;
      if (ok) {
        if constexpr (D == 128) { const uint2 v = *reinterpret_cast<const uint2 *>(c); t.vw[i][0] = v.x; t.vw[i][1] = v.y; }
        else if constexpr (D == 64) t.vw[i][0] = *reinterpret_cast<const uint32_t *>(c);
        else {
          const uint16_t *p = reinterpret_cast<const uint16_t *>(c);
          t.vw[i][0] = (uint32_t)p[0] | ((uint32_t)p[1] << 16);
          t.vw[i][1] = p[2];
        }
      }
    }
  };

  Tile cur;
  if (NKT > 0) fetch(0, cur);   // (written by earlier steps)
  pdl_wait();
  pdl_launch_dependents();  // the retaining head reads only what the projection wrote: it may run beside this kernel
  if (a.tok_k && split == 0 && hg == 0 && warp < 2) {
    // The token of this step enters the 4-bit cache (this step still reads it in bf16): one warp
    // quantises its pre-RoPE key, one its value, with the arithmetic of the chunk kernel.
    const bf16 *src = (warp == 0 ? a.tok_k : a.tok_v) + (size_t)m * D;
    float x0[2], x1[2], amax = 0.f;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int p = lane + 32 * k;
      x0[k] = x1[k] = 0.f;
      if (2 * p < D) {
        const __nv_bfloat162 v2 = *reinterpret_cast<const __nv_bfloat162 *>(src + 2 * p);
        x0[k] = __bfloat162float(v2.x);
        x1[k] = __bfloat162float(v2.y);
        amax = fmaxf(amax, fmaxf(fabsf(x0[k]), fabsf(x1[k])));
      }
    }
    amax = warp_max(amax);
    __half sh = __float2half_rn(__fdiv_rn(amax, 7.0f));
    if (__half2float(sh) == 0.f) sh = __float2half_rn(1.0f);
    const float sf = __half2float(sh);
    const size_t u = (size_t)m * cap + (n - 1);
    uint8_t *dst = (warp == 0 ? q4.kq : q4.vq) + u * (D / 2);
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int p = lane + 32 * k;
      if (2 * p < D) {
        const int c0 = (int)fminf(fmaxf(rintf(__fdiv_rn(x0[k], sf)), -8.f), 7.f);
        const int c1 = (int)fminf(fmaxf(rintf(__fdiv_rn(x1[k], sf)), -8.f), 7.f);
        dst[p] = (uint8_t)((c0 & 0xF) | ((c1 & 0xF) << 4));
      }
    }
    if (lane == 0) (warp == 0 ? q4.ks : q4.vs)[u] = sh;
  }
  uint2 qf[NT > 1 ? 1 : D / 16];   // heads g4, g4 + 8
  auto load_q = [&](int kk, int t) -> uint2 {
    const int head = 8 * t + g4;
    const bf16 *src = a.q_rot + (size_t)(h0 + min(head, gh - 1)) * D + 2 * q + (kk & 1) * (D / 2) + (kk >> 1) * 16;
    return head < gh ? make_uint2(*reinterpret_cast<const uint32_t *>(src), *reinterpret_cast<const uint32_t *>(src + 8))
                     : make_uint2(0u, 0u);
  };
  if constexpr (NT > 1) {
    for (int i = warp; i < D / 16 * NT; i += DA_THREADS / 32) sq[i][lane] = load_q(i / NT, i % NT);
    __syncthreads();
  } else {
#pragma unroll
    for (int kk = 0; kk < D / 16; kk++) qf[kk] = load_q(kk, 0);
  }
  auto q_frag = [&](int kk, int t) -> uint2 {
    if constexpr (NT > 1) return sq[kk * NT + t][lane];
    else return qf[kk];
  };
  float o[NT][D / 16][4], mrow[NT][2], lrow[NT][2];   // heads 8 t + 2 q and the next
#pragma unroll
  for (int t = 0; t < NT; t++) {
#pragma unroll
    for (int i = 0; i < D / 16; i++)
#pragma unroll
      for (int e = 0; e < 4; e++) o[t][i][e] = 0.f;
    mrow[t][0] = mrow[t][1] = -INFINITY;
    lrow[t][0] = lrow[t][1] = 0.f;
  }
  const uint32_t sel = 0x4440u | (uint32_t)q;   // byte q of a word to bits 0-7, zeros elsewhere

  for (int kt = 0; kt < NKT; kt++) {
    const int base = k0 + kt * DA_KT + warp * 16;
    if (base >= k1) break;
    float4 cs4[2][D / 16];   // pairs 8 e + 2 q and the next
#pragma unroll
    for (int r = 0; r < 2; r++) {
      const float4 *c = reinterpret_cast<const float4 *>(a.cs + (size_t)cur.pos[r] * (D / 2)) + q;
#pragma unroll
      for (int e = 0; e < D / 16; e++) cs4[r][e] = __ldg(c + 4 * e);
    }
    // values while the (cos, sin) rows are on their way: columns (D / 8) g4 + 2 i and the next are rows g4 and g4 + 8 of tile i
    uint32_t va[D / 16][4];
#pragma unroll
    for (int hf = 0; hf < 2; hf++) {
      float x[2][D / 8];
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const int key = base + q + 4 * (2 * hf + e);
#pragma unroll
        for (int b = 0; b < D / 32; b++) {
          float y[4];
          q4_expand4(cur.vw[2 * hf + e][b / 2] >> (16 * (b & 1)), cur.vs[2 * hf + e], y);
#pragma unroll
          for (int k = 0; k < 4; k++) x[e][4 * b + k] = y[k];
        }
        if (key == n - 1) {   // the token of this step
          const uint32_t *tv = reinterpret_cast<const uint32_t *>(a.v + (size_t)m * D + (D / 8) * g4);
#pragma unroll
          for (int k = 0; k < D / 16; k++) {
            const uint32_t v = tv[k];
            x[e][2 * k] = __uint_as_float(v << 16);
            x[e][2 * k + 1] = __uint_as_float(v & 0xffff0000u);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < D / 16; i++) {
        va[i][2 * hf] = pack_bf16(x[0][2 * i], x[1][2 * i]);
        va[i][2 * hf + 1] = pack_bf16(x[0][2 * i + 1], x[1][2 * i + 1]);
      }
    }
    float s[NT][4] = {};
#pragma unroll
    for (int b = 0; b < D / 32; b++) {
      uint32_t lo[4], hi[4];   // fragments of the lower and the upper elements of 16 rotation pairs
#pragma unroll
      for (int r = 0; r < 2; r++) {
        float x1[4], x2[4];
        const float s0 = cur.ks[r], s1 = s0 * 0x1p-4f;
#pragma unroll
        for (int k = 0; k < 2; k++) {
          const uint32_t w1 = __byte_perm(cur.kw[r][0][2 * b + k], 0, sel), w2 = __byte_perm(cur.kw[r][1][2 * b + k], 0, sel);
          x1[2 * k] = q4_code<0>(w1) * s0; x1[2 * k + 1] = q4_code<1>(w1) * s1;
          x2[2 * k] = q4_code<0>(w2) * s0; x2[2 * k + 1] = q4_code<1>(w2) * s1;
        }
        const float4 c0 = cs4[r][2 * b], c1 = cs4[r][2 * b + 1];
        const float cc[4] = {c0.x, c0.z, c1.x, c1.z}, sn[4] = {c0.y, c0.w, c1.y, c1.w};
        float y1[4], y2[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
          y1[k] = x1[k] * cc[k] - x2[k] * sn[k];
          y2[k] = x2[k] * cc[k] + x1[k] * sn[k];
        }
        lo[r] = pack_bf16(y1[0], y1[1]); lo[r + 2] = pack_bf16(y1[2], y1[3]);
        hi[r] = pack_bf16(y2[0], y2[1]); hi[r + 2] = pack_bf16(y2[2], y2[3]);
        if (base + 8 * r + kr == n - 1) {
          const uint32_t *tk = reinterpret_cast<const uint32_t *>(a.k_rot + (size_t)m * D + 16 * b + 2 * q);
          lo[r] = tk[0]; lo[r + 2] = tk[4];
          hi[r] = tk[D / 4]; hi[r + 2] = tk[D / 4 + 4];
        }
      }
#pragma unroll
      for (int t = 0; t < NT; t++) {
        const uint2 ql = q_frag(2 * b, t), qh = q_frag(2 * b + 1, t);
        mma_bf16_16816(s[t], lo, ql.x, ql.y);
        mma_bf16_16816(s[t], hi, qh.x, qh.y);
      }
    }
    if (kt + 1 < NKT) fetch(kt + 1, cur);
    // online softmax of this warp's 16 keys (the keys past the split's end weigh nothing)
#pragma unroll
    for (int t = 0; t < NT; t++) {
      float alpha[2];
#pragma unroll
      for (int c = 0; c < 2; c++) {
        const float v0 = base + kr < k1 ? s[t][c] * scale_log2 : -INFINITY, v1 = base + 8 + kr < k1 ? s[t][c + 2] * scale_log2 : -INFINITY;
        float tmax = fmaxf(v0, v1);
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 4));
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 8));
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 16));
        const float mnew = fmaxf(mrow[t][c], tmax), muse = mnew == -INFINITY ? 0.f : mnew;
        alpha[c] = exp2f(mrow[t][c] - muse);
        mrow[t][c] = mnew;
        s[t][c] = exp2f(v0 - muse);
        s[t][c + 2] = exp2f(v1 - muse);
        lrow[t][c] = lrow[t][c] * alpha[c] + (s[t][c] + s[t][c + 2]);
      }
#pragma unroll
      for (int i = 0; i < D / 16; i++) {
        o[t][i][0] *= alpha[0]; o[t][i][2] *= alpha[0];
        o[t][i][1] *= alpha[1]; o[t][i][3] *= alpha[1];
      }
      const uint32_t pb0 = movmatrix_trans(pack_bf16(s[t][0], s[t][1])), pb1 = movmatrix_trans(pack_bf16(s[t][2], s[t][3]));
#pragma unroll
      for (int i = 0; i < D / 16; i++) mma_bf16_16816(o[t][i], va[i], pb0, pb1);
    }
  }

  // ---- the four warps' states meet
#pragma unroll
  for (int t = 0; t < NT; t++) {
#pragma unroll
    for (int c = 0; c < 2; c++) {
      float l = lrow[t][c];
      l += __shfl_xor_sync(0xffffffffu, l, 4);
      l += __shfl_xor_sync(0xffffffffu, l, 8);
      l += __shfl_xor_sync(0xffffffffu, l, 16);
      const int head = 8 * t + 2 * q + c;
      if (head < gh) {
        if (g4 == 0) { wm[warp][head] = mrow[t][c]; wl[warp][head] = l; }
        float *dst = fo[warp][head] + (D / 8) * g4;
#pragma unroll
        for (int i = 0; i < D / 16; i++) *reinterpret_cast<float2 *>(dst + 2 * i) = make_float2(o[t][i][c], o[t][i][c + 2]);
      }
    }
  }
  __syncthreads();
  // partial result of this split: o [h][split][D] (not normalised), (m, l) [h][split][2]
  for (int idx = tid; idx < gh * (D / 4); idx += DA_THREADS) {
    const int i = idx / (D / 4), c = (idx - i * (D / 4)) * 4;
    const float mx = fmaxf(fmaxf(wm[0][i], wm[1][i]), fmaxf(wm[2][i], wm[3][i])), muse = mx == -INFINITY ? 0.f : mx;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float lsum = 0.f;
#pragma unroll
    for (int w = 0; w < 4; w++) {
      // (a warp without keys has sum 0; one whose scores are all NaN has no maximum, but a sum that says so)
      const float wgt = wl[w][i] == 0.f ? 0.f : (wm[w][i] == -INFINITY ? 1.f : exp2f(wm[w][i] - muse));
      if (wgt != 0.f) {
        const float4 v = *reinterpret_cast<const float4 *>(&fo[w][i][c]);
        acc.x = fmaf(wgt, v.x, acc.x); acc.y = fmaf(wgt, v.y, acc.y);
        acc.z = fmaf(wgt, v.z, acc.z); acc.w = fmaf(wgt, v.w, acc.w);
        lsum = fmaf(wgt, wl[w][i], lsum);
      }
    }
    const size_t hs = (size_t)(h0 + i) * n_splits + split;
    *reinterpret_cast<float4 *>(a.part_o + hs * D + c) = acc;
    if (c == 0) *(reinterpret_cast<float2 *>(a.part_ml) + hs) = make_float2(mx, lsum);
  }

  // ---- the split that finishes last merges the partial results of all splits, in split order
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicInc(&a.counters[m * hgroups + hg], n_splits - 1) == (unsigned)(n_splits - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = warp; i < gh; i += 4) {   // weights of the splits, a warp per head
    float ms[2], ls[2], mx = -INFINITY, lsum = 0.f;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int s2 = lane + 32 * k;
      const float2 ml = s2 < n_splits ? __ldcg(reinterpret_cast<const float2 *>(a.part_ml) + (size_t)(h0 + i) * n_splits + s2)
                                      : make_float2(-INFINITY, 0.f);
      ms[k] = ml.x; ls[k] = ml.y;
      mx = fmaxf(mx, ml.x);
    }
    mx = warp_max(mx);
    const float muse = mx == -INFINITY ? 0.f : mx;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const float w = ls[k] == 0.f ? 0.f : (ms[k] == -INFINITY ? 1.f : exp2f(ms[k] - muse));
      if (w != 0.f) lsum = fmaf(w, ls[k], lsum);
      sw[i][lane + 32 * k] = w;
    }
    lsum = warp_sum(lsum);
    if (lane == 0) sinv[i] = 1.0f / lsum;
  }
  __syncthreads();
  for (int idx = tid; idx < gh * (D / 4); idx += DA_THREADS) {   // sixteen splits in flight as 16-byte loads
    const int i = idx / (D / 4), c = (idx - i * (D / 4)) * 4;
    const float *po = a.part_o + (size_t)(h0 + i) * n_splits * D + c;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s2 = 0; s2 < n_splits; s2 += 16) {
      float4 v[16];
#pragma unroll
      for (int k = 0; k < 16; k++)
        v[k] = (s2 + k < n_splits) ? __ldcg(reinterpret_cast<const float4 *>(po + (size_t)(s2 + k) * D)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 16; k++) {
        const float w = s2 + k < n_splits ? sw[i][s2 + k] : 0.f;
        if (w != 0.f) {
          acc.x = fmaf(w, v[k].x, acc.x); acc.y = fmaf(w, v[k].y, acc.y);
          acc.z = fmaf(w, v[k].z, acc.z); acc.w = fmaf(w, v[k].w, acc.w);
        }
      }
    }
    const float inv = sinv[i];
    *reinterpret_cast<uint2 *>(a.out + (size_t)(h0 + i) * D + c) =
        make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
  }
}

}  // namespace

// y[n] = x . Wt[n] + r[n]: a projection of one token with its residual connection
cudaError_t launch_gemv_resid(const bf16 *x, const bf16 *Wt, int N, int K, const bf16 *r, bf16 *y,
                              cudaStream_t st) {
  if (K % 8) return cudaErrorInvalidValue;
  const int smem = K * 2 + 8 * 32 * 4;
  const int blocks = min((N + 7) / 8, 148 * 4);
  gemv_kernel<0, 1><<<blocks, GV_THREADS, smem, st>>>(x, Wt, N, K, y, r, 0, 0, RhGemvBatchN<1>{});
  return cudaGetLastError();
}

// Gated FFN, first half, for one token: Wt [2F x K] holds, per block of 128 outputs, the 128
// rows of W_gate^T followed by the 128 rows of W_up^T; a warp computes one gate row and the
// matching up row and stores silu(gate) * up.
__global__ void __launch_bounds__(GV_THREADS)
gemv_gated_kernel(const bf16 *__restrict__ x, const bf16 *__restrict__ Wt, int F, int K, bf16 *__restrict__ act) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint4 *sx = reinterpret_cast<uint4 *>(smem_raw);
  for (int i = threadIdx.x; i < K / 8; i += GV_THREADS) sx[i] = reinterpret_cast<const uint4 *>(x)[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = blockIdx.x * (GV_THREADS / 32) + warp, nw = gridDim.x * (GV_THREADS / 32);
  for (int c = gw; c < F; c += nw) {
    const size_t row = (size_t)(c / 128) * 256 + (c % 128);
    const uint4 *r0 = reinterpret_cast<const uint4 *>(Wt + row * K);
    const uint4 *r1 = reinterpret_cast<const uint4 *>(Wt + (row + 128) * K);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
    for (int v = lane; v < K / 8; v += 32) {
      const uint4 xv = sx[v];
      s0 += dot8(__ldg(r0 + v), xv);
      s1 += dot8(__ldg(r1 + v), xv);
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (lane == 0) act[c] = __float2bfloat16_rn(s0 / (1.0f + __expf(-s0)) * s1);
  }
}
cudaError_t launch_gemv_gated(const bf16 *x, const bf16 *Wt, int F, int K, bf16 *act, cudaStream_t st) {
  if (K % 8) return cudaErrorInvalidValue;
  const int blocks = min((F + 7) / 8, 148 * 8);
  gemv_gated_kernel<<<blocks, GV_THREADS, K * 2, st>>>(x, Wt, F, K, act);
  return cudaGetLastError();
}

bool gemv_rope_batched(int K) { return K % 8 == 0 && K / 8 <= GW_THREADS; }
int rh_gemv_blocks(int d_R) { return min((d_R + 3) / 4, 148 * 4); }

cudaError_t launch_gemv_rope(const bf16 *x, int K, const GemvRopeBatch &b, int n_layers, cudaStream_t st, bool pdl) {
  const RopeAppendArgs &a = b.a[0];
  if (K % 8 || a.d % 2 || n_layers < 1 || n_layers > DECODE_BATCH) return cudaErrorInvalidValue;
  const int items = (a.h + 2 * a.h_kv) * (a.d / 2);
  if (gemv_rope_batched(K)) {
    const int blocks = min((n_layers * items + GW_PB - 1) / GW_PB, 148 * 2);
    if (n_layers > 1)
      return launch_kernel(gemv_rope_wide_kernel<DECODE_BATCH>, dim3(blocks), dim3(GW_THREADS), 0, st, pdl, x, K, n_layers, b);
    GemvRopeBatchN<1> one;
    one.Wt[0] = b.Wt[0];
    one.a[0] = a;
    return launch_kernel(gemv_rope_wide_kernel<1>, dim3(blocks), dim3(GW_THREADS), 0, st, pdl, x, K, 1, one);
  }
  if (n_layers != 1) return cudaErrorInvalidValue;
  const int blocks = min((items + 7) / 8, 148 * 4);
  return launch_kernel(gemv_rope_kernel, dim3(blocks), dim3(GV_THREADS), (size_t)K * 2, st, pdl, x, b.Wt[0], K,
                       const_cast<bf16 *>(a.staging), a);
}

cudaError_t launch_rh_gemv(const RhGemvBatch &b, int n_layers, int d_R, int K, int h_kv, int act, cudaStream_t st, bool pdl) {
  if (K % 16 || h_kv > 32 || n_layers < 1 || n_layers > DECODE_BATCH) return cudaErrorInvalidValue;
  const int smem = K * 2 + 8 * 32 * 4;
  const dim3 grid(rh_gemv_blocks(d_R), n_layers);
  const bf16 *none = nullptr;
  if (n_layers > 1)
    return launch_kernel(gemv_kernel<1, DECODE_BATCH>, grid, dim3(GV_THREADS), (size_t)smem, st, pdl, none, none, d_R, K,
                         (bf16 *)nullptr, none, h_kv, act, b);
  return launch_kernel(gemv_kernel<1, 1>, grid, dim3(GV_THREADS), (size_t)smem, st, pdl, none, none, d_R, K, (bf16 *)nullptr,
                       none, h_kv, act, RhGemvBatchN<1>{{b.l[0]}});
}

// Splits of the key range per KV head.  Measured at the Llama shape (8 KV heads, 6000 keys, 256 steps through
// 32 layers): with a bf16 cache 64 / 96 / 120 / 148 / 200 / 296 / 444 CTAs in total give 914 / 1058 / 1130 /
// 1152 / 1224 / 1133 / 1052 tokens/s (more splits shorten each CTA's chain of tiles, but the last split of a
// head merges them all).  With a 4-bit cache 100 / 148 / 200 / 296 / 400 CTAs take 93.2 / 94.5 / 88.1 / 99.8 / 97.5 us a step of
// four such layers, 34.7 / 28.5 / 28.4 / 28.0 / 30.7 us of one, and at the Phi-3 shape (32 KV heads of 96) 171 / 187 / 181 / 179 /
// 177 and 63.7 / 55.5 / 53.5 / 56.2 / 50.9 us: 200 is the best of the first and within 2, 6 and 5 % of the best of the others.
// Groups of query heads that one block cannot serve multiply the CTAs (a launch of one layer gains from that, see
// q4_heads_per_block).
int decode_attn_splits(int h_kv, int n) {
  static int forced = -1;
  if (forced < 0) { const char *e = getenv("LOCRET_DEC_CTAS"); forced = e ? atoi(e) : 0; if (forced < 0 || forced > 2048) forced = 0; }
  const int sms = sm_count_of_current_device();
  const int total = forced ? forced : (sms * 27) / 20;
  int s = (total + h_kv - 1) / h_kv;
  const int max_s = (n + 127) / 128;            // at least one 128-key tile per split
  if (s > max_s) s = max_s;
  if (s > 64) s = 64;
  return s < 1 ? 1 : s;
}

// Query heads that a block of the 4-bit kernel serves.  Sixteen: the keys of a larger group are expanded and rotated for half as
// many blocks; eight: twice the blocks, each with half the heads to merge at the end.  The first pays where the blocks of eight
// (of which two fit an SM, three of head_dim 64) would take more than one wave and there are keys enough (tiles: 64 units of
// one KV head, of all layers of the launch).  Measured (us a step, eight / sixteen): 16 heads a KV head, head_dim 128, 6000
// units, on one KV head 19.2 / 27.7 (94 tiles), on two 55.9 / 59.7 in four layers (752) and 102.3 / 94.6 in eight (1504), on
// four, 15000 units 46.8 / 45.6 (940), on eight, 16000 units 75.4 / 60.2 (2000); head_dim 64, on four, 15000 units 24.0 / 27.7 (400
// blocks of eight), on 32 (nine heads each), 2000 units 44.4 / 39.4 (448).
static int q4_heads_per_block(int g, int d, int tiles, int blocks_of_eight) {
  const int sms = sm_count_of_current_device();
  return g > 8 && tiles > 6 * sms && blocks_of_eight > (d == 64 ? 3 : 2) * sms ? 16 : 8;
}

cudaError_t launch_attention_decode(const DecodeAttnBatch &b, int n_layers, int h, int h_kv, int d, cudaStream_t st,
                                    bool pdl) {
  const bool q4 = b.l[0].q4.kq != nullptr;
  if (n_layers < 1 || n_layers > DECODE_BATCH) return cudaErrorInvalidValue;
  const int g = h / h_kv;
  int splits = 1, tiles = 0, blocks_of_eight = 0;
  for (int i = 0; i < n_layers; i++) {
    splits = b.l[i].n_splits > splits ? b.l[i].n_splits : splits;
    tiles += h_kv * ((b.l[i].n + DA_KT - 1) / DA_KT);
    blocks_of_eight += h_kv * b.l[i].n_splits * ((g + 7) / 8);
  }
  const int group = q4 ? q4_heads_per_block(g, d, tiles, blocks_of_eight) : DA_G, hgroups = (g + group - 1) / group;
  if (h_kv * hgroups > DECODE_HEAD_GROUPS) return cudaErrorInvalidValue;
  if (splits > 64) return cudaErrorInvalidValue;
  const dim3 grid(h_kv, splits, n_layers * hgroups);
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)d);
  auto run = [&](auto kern1, auto kern_n, size_t smem, PerDeviceFlag (&attr_set)[2]) -> cudaError_t {
    if (n_layers > 1) {
      if (cudaError_t e = allow_dynamic_smem(kern_n, (int)smem, attr_set[1]); e != cudaSuccess) return e;
      return launch_kernel(kern_n, grid, dim3(DA_THREADS), smem, st, pdl, h, h_kv, scale_log2, b);
    }
    if (cudaError_t e = allow_dynamic_smem(kern1, (int)smem, attr_set[0]); e != cudaSuccess) return e;
    return launch_kernel(kern1, grid, dim3(DA_THREADS), smem, st, pdl, h, h_kv, scale_log2, DecodeAttnBatchN<1>{{b.l[0]}});
  };
  auto launch = [&](auto dim) -> cudaError_t {
    constexpr int D = decltype(dim)::value;
    static PerDeviceFlag set_q4[2], set_q4_two[2], set_bf16[2];
    if (q4 && group == 8) return run(attn_decode_q4_kernel<D, 1, 1>, attn_decode_q4_kernel<D, DECODE_BATCH, 1>, 0, set_q4);
    return q4 ? run(attn_decode_q4_kernel<D, 1, 2>, attn_decode_q4_kernel<D, DECODE_BATCH, 2>, 0, set_q4_two)
              : run(attn_decode_kernel<D, 1>, attn_decode_kernel<D, DECODE_BATCH>, (DA_G + 4 * DA_KT) * (d + 8) * 2, set_bf16);
  };
  switch (d) {
    case 64: return launch(std::integral_constant<int, 64>{});
    case 96: return launch(std::integral_constant<int, 96>{});
    case 128: return launch(std::integral_constant<int, 128>{});
  }
  return cudaErrorInvalidValue;
}

}  // namespace locret

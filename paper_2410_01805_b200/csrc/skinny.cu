// Projections of a few tokens (a short question, the ragged end of a prompt, one decoded token):
// Y[t][n] = sum_k X[t][k] Wt[n][k] for so few rows t that the weights are all the traffic.
//
// A 128 x 256 tile of the GEMM in gemm_tc.cu would leave most SMs idle (6144 columns are 24 tiles) and pad the
// tokens to 128 rows.  Here the operands change sides: 128 weight rows are the M side of tcgen05.mma, the
// tokens, padded to NT = 16 / 32 / 64 / 128, its N side, and a cluster of S CTAs divides K.  Every CTA
// keeps three to six stages of weights (about 100 KB) in flight, two CTAs fit an SM, and the weights of the
// first stages are requested before the wait for the kernel that writes X, so the weight stream does not stop
// between dependent launches.  The S partial sums meet in distributed shared memory: each CTA
// leaves its accumulator there as [token][row], and rank r adds the tokens of its share over all ranks
// in rank order (deterministic, no scratch, no second launch) and runs the epilogue on them:
//   EPI 0: bf16 store, with the residual added before the rounding if there is one;
//   EPI 1: gated FFN, first half: a tile is 64 gate rows and the 64 up rows of the same outputs;
//   EPI 2: retaining head: activation and the thin product with W2, one partial score per (tile, token, head).
// Measured for 20 tokens: W_gate and W_up of the Llama shape (235 MB) 43 us = 5.5 TB/s, W_down (117 MB) 25 us, the
// QKV projection (50 MB, 45 tokens) 16 us (34 us on 24 tiles of 128 x 256).
#include "tc_common.cuh"

namespace locret {

namespace {

using namespace tc;

constexpr int SK_THREADS = 128, SK_BK = 64, SK_ROWS = 128;
constexpr int SK_A_BYTES = SK_ROWS * SK_BK * 2;
constexpr int SK_MAX_SPLIT = 8;   // portable cluster size

template <int NT>
struct SkinnyCfg {
  static constexpr int STAGES = NT == 16 ? 6 : (NT == 32 ? 5 : (NT == 64 ? 4 : 3));
  static constexpr int STAGE_BYTES = SK_A_BYTES + NT * SK_BK * 2;
  static constexpr int TMEM_COLS = NT < 32 ? 32 : NT;
  static constexpr int SMEM = 1024 + STAGES * STAGE_BYTES + 256;
  static_assert(SMEM >= SKINNY_MIN_SMEM && TMEM_COLS <= 128, "see tc_common.cuh");
  static_assert(NT * SK_ROWS * 4 <= STAGES * STAGE_BYTES, "the accumulator reuses the stages");
};

struct SkinnyParams {
  int n_tok, N, K, n_split;
  bf16 *out; int ldo;
  const bf16 *resid; int ldr;
  const float *W2; float *partial; int h_kv, act;
  int *status;
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// grid S * token tiles * tiles, cluster S: rank = K slice; the token tiles of one weight tile run side by
// side, so all but the first find its weights in L2
template <int NT, int EPI>
__global__ void __launch_bounds__(SK_THREADS)
skinny_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
              const SkinnyParams p) {
  using Cfg = SkinnyCfg<NT>;
  constexpr int STAGES = Cfg::STAGES;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + STAGES * Cfg::STAGE_BYTES);
  uint64_t *empty = full + STAGES;
  uint64_t *acc_full = empty + STAGES;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.n_split, rank = (int)blockIdx.x % S, unit = (int)blockIdx.x / S;
  const int tok_tiles = (p.n_tok + NT - 1) / NT;
  const int tile = unit / tok_tiles, tok0 = (unit - tile * tok_tiles) * NT;
  const int kb_all = p.K / SK_BK;
  const int kb0 = (int)((long long)rank * kb_all / S), kb1 = (int)((long long)(rank + 1) * kb_all / S);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(acc_full, 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&map_w);
    prefetch_tmap(&map_x);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      auto load_w = [&](int s, int kb) {
        unsigned char *dst = smem + s * Cfg::STAGE_BYTES;
        if (EPI == 1) {  // interleaved in blocks of 128 gate and 128 up rows: 64 of each
          const int row = (tile >> 1) * 256 + (tile & 1) * 64;
          tma_load_2d(dst, &map_w, kb * SK_BK, row, &full[s]);
          tma_load_2d(dst + SK_A_BYTES / 2, &map_w, kb * SK_BK, row + 128, &full[s]);
        } else {
          tma_load_2d(dst, &map_w, kb * SK_BK, tile * SK_ROWS, &full[s]);
        }
      };
      // the weights depend on nothing before this kernel; X does
      const int pre = min(STAGES, kb1 - kb0);
      for (int i = 0; i < pre; i++) {
        mbar_expect_tx(&full[i], Cfg::STAGE_BYTES);
        load_w(i, kb0 + i);
      }
      pdl_wait();
      pdl_launch_dependents();
      for (int i = 0; i < kb1 - kb0; i++) {
        const int s = i % STAGES;
        if (i >= pre) {
          if (!mbar_wait(&empty[s], ((i / STAGES) & 1) ^ 1, abort_flag, p.status)) break;
          mbar_expect_tx(&full[s], Cfg::STAGE_BYTES);
          load_w(s, kb0 + i);
        }
        tma_load_2d(smem + s * Cfg::STAGE_BYTES + SK_A_BYTES, &map_x, (kb0 + i) * SK_BK, tok0, &full[s]);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16(SK_ROWS, NT, 0, 0);
      bool ok = true;
      for (int i = 0; i < kb1 - kb0 && ok; i++) {
        const int s = i % STAGES;
        ok = mbar_wait(&full[s], (i / STAGES) & 1, abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = desc_kmajor_sw128(smem + s * Cfg::STAGE_BYTES);
        const uint64_t db = desc_kmajor_sw128(smem + s * Cfg::STAGE_BYTES + SK_A_BYTES);
#pragma unroll
        for (int k = 0; k < SK_BK / 16; k++) {
          if (i == 0 && k == 0) mma_ss_first(tmem, da, db, idesc);
          else mma_ss_acc(tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc);
        }
        mma_commit(&empty[s]);
      }
      if (ok) mma_commit(acc_full);
    }
    __syncwarp();
  }
  pdl_wait();  // the epilogue reads and overwrites what kernels before this one wrote and read
  const bool ok = mbar_wait(acc_full, 0, abort_flag, p.status);
  __syncwarp();
  tc_fence_after();

  // accumulator -> [token][row] in this CTA's shared memory (every MMA has read its stages by now)
  float *acc = reinterpret_cast<float *>(smem);
  {
    const int row = warp * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c0 = 0; c0 < NT; c0 += 16) {
      if (tok0 + c0 >= p.n_tok) break;
      uint32_t r[16];
      tmem_ld16(taddr + c0, r);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; i++) acc[(c0 + i) * SK_ROWS + row] = ok ? __uint_as_float(r[i]) : 0.f;
    }
  }
  tc_fence_before();
  if (S > 1) cluster_sync_all();
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, Cfg::TMEM_COLS);
  }

  const uint32_t acc_addr = smem_u32(acc);
  auto sum4 = [&](int t, int row) {  // rows row .. row + 3 of token t, over the slices of K in order
    const uint32_t a = acc_addr + (uint32_t)(t * SK_ROWS + row) * 4;
    if (S == 1) return *reinterpret_cast<const float4 *>(acc + t * SK_ROWS + row);
    // (all remote loads in flight before the first is used: one after the other an 8-way sum took 2 us more)
    float4 w[SK_MAX_SPLIT];
#pragma unroll
    for (int r = 0; r < SK_MAX_SPLIT; r++)
      if (r < S) w[r] = ld_cluster_f4(cluster_map(a, r));
    float4 v = w[0];
#pragma unroll
    for (int r = 1; r < SK_MAX_SPLIT; r++)
      if (r < S) { v.x += w[r].x; v.y += w[r].y; v.z += w[r].z; v.w += w[r].w; }
    return v;
  };
  const int share = NT / S, t0 = rank * share;
  const int nt = min(share, p.n_tok - tok0 - t0);  // tokens of this rank (may be none)
  if (EPI == 0) {
    const int n = tile * SK_ROWS + lane * 4;
    if (n < p.N)
      for (int t = warp; t < nt; t += SK_THREADS / 32) {
        float4 v = sum4(t0 + t, lane * 4);
        const size_t tok = (size_t)(tok0 + t0 + t);
        if (p.resid) {
          const uint2 rv = *reinterpret_cast<const uint2 *>(p.resid + tok * p.ldr + n);
          v.x += __uint_as_float(rv.x << 16); v.y += __uint_as_float(rv.x & 0xffff0000u);
          v.z += __uint_as_float(rv.y << 16); v.w += __uint_as_float(rv.y & 0xffff0000u);
        }
        *reinterpret_cast<uint2 *>(p.out + tok * p.ldo + n) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
      }
  } else if (EPI == 1) {
    for (int i = threadIdx.x; i < nt * 16; i += SK_THREADS) {
      const int t = i >> 4, q = (i & 15) * 4;
      const float4 g = sum4(t0 + t, q), u = sum4(t0 + t, 64 + q);
      const float a0 = g.x / (1.0f + __expf(-g.x)) * u.x, a1 = g.y / (1.0f + __expf(-g.y)) * u.y;
      const float a2 = g.z / (1.0f + __expf(-g.z)) * u.z, a3 = g.w / (1.0f + __expf(-g.w)) * u.w;
      *reinterpret_cast<uint2 *>(p.out + (size_t)(tok0 + t0 + t) * p.ldo + tile * 64 + q) =
          make_uint2(pack_bf16(a0, a1), pack_bf16(a2, a3));
    }
  } else {
    // a warp takes four tokens at a time, a lane four rows of each: the chains of loads and shuffles of the four overlap
    constexpr int TB = 4;
    const int n = tile * SK_ROWS + lane * 4;
    for (int tb = warp * TB; tb < nt; tb += SK_THREADS / 32 * TB) {
      float a[TB][4];
#pragma unroll
      for (int i = 0; i < TB; i++) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (n < p.N && tb + i < nt) v = sum4(t0 + tb + i, lane * 4);
        a[i][0] = apply_act(v.x, p.act); a[i][1] = apply_act(v.y, p.act);   // (every activation maps 0 to 0)
        a[i][2] = apply_act(v.z, p.act); a[i][3] = apply_act(v.w, p.act);
      }
      float *dst = p.partial + ((size_t)tile * p.n_tok + tok0 + t0 + tb) * p.h_kv;
#pragma unroll 2
      for (int m = 0; m < p.h_kv; m++) {
        float s[TB] = {};
        if (n < p.N) {
#pragma unroll
          for (int e = 0; e < 4; e++) {
            const float w = __ldg(p.W2 + (size_t)(n + e) * p.h_kv + m);
#pragma unroll
            for (int i = 0; i < TB; i++) s[i] = fmaf(a[i][e], w, s[i]);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int i = 0; i < TB; i++) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
#pragma unroll
        for (int i = 0; i < TB; i++)
          if (lane == i && tb + i < nt) dst[i * p.h_kv + m] = s[i];
      }
    }
  }
  if (S > 1) cluster_sync_all();  // no CTA leaves while another may still read its accumulator
}

template <int NT, int EPI>
cudaError_t launch_nt(const bf16 *X, int ldx, const bf16 *Wt, int ldw, const SkinnyParams &p, int tiles, int rows_w,
                      cudaStream_t st, bool pdl) {
  using Cfg = SkinnyCfg<NT>;
  static PerDeviceFlag attr_set;
  if (cudaError_t e = allow_dynamic_smem(skinny_kernel<NT, EPI>, Cfg::SMEM, attr_set); e != cudaSuccess) return e;
  CUtensorMap mw, mx;
  if (!cached_map_k64(&mw, Wt, p.K, rows_w, (uint64_t)ldw * 2, EPI == 1 ? 64 : SK_ROWS) ||
      !cached_map_k64(&mx, X, p.K, p.n_tok, (uint64_t)ldx * 2, NT))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles * p.n_split * ((p.n_tok + NT - 1) / NT));
  cfg.blockDim = dim3(SK_THREADS);
  cfg.dynamicSmemBytes = Cfg::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.n_split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, skinny_kernel<NT, EPI>, mw, mx, p);
}

struct SkinnyPlan { int tiles, nt, n_split; };   // tiles of 128 weight rows, tokens of a token tile, CTAs that divide K

SkinnyPlan skinny_plan(int n_tok, int rows_w, int K) {
  const int tiles = (rows_w + SK_ROWS - 1) / SK_ROWS;
  int nt = n_tok <= 16 ? 16 : (n_tok <= 32 ? 32 : (n_tok <= 64 ? 64 : 128));
  // The deepest split of K that keeps all CTAs resident at once and gives each at least four K-blocks; and for small
  // matrices narrower token tiles while not even a third of the SMs has a CTA (the small shape's retaining head at 512
  // tokens: 17.5 us in 16 CTAs, 9.5 us in 64; the Llama shape's at 45 tokens, 64 CTAs, only lost by 128: 38 and 47 us).
  const int sms = sm_count_of_current_device();
  auto split_of = [&](int w) {
    const int c = tiles * ((n_tok + w - 1) / w);
    int s = 1;
    while (s < SK_MAX_SPLIT && c * s * 2 <= 2 * sms && K / SK_BK / (2 * s) >= 4) s *= 2;
    return s;
  };
  while (nt > 32 && tiles * ((n_tok + nt - 1) / nt) * split_of(nt) * 3 <= sms) nt /= 2;
  return {tiles, nt, split_of(nt)};
}

template <int EPI>
cudaError_t launch_skinny(const bf16 *X, int ldx, const bf16 *Wt, int ldw, SkinnyParams p, int rows_w, cudaStream_t st,
                          bool pdl) {
  const SkinnyPlan plan = skinny_plan(p.n_tok, rows_w, p.K);
  p.n_split = plan.n_split;
  switch (plan.nt) {
    case 16: return launch_nt<16, EPI>(X, ldx, Wt, ldw, p, plan.tiles, rows_w, st, pdl);
    case 32: return launch_nt<32, EPI>(X, ldx, Wt, ldw, p, plan.tiles, rows_w, st, pdl);
    case 64: return launch_nt<64, EPI>(X, ldx, Wt, ldw, p, plan.tiles, rows_w, st, pdl);
  }
  return launch_nt<128, EPI>(X, ldx, Wt, ldw, p, plan.tiles, rows_w, st, pdl);
}

}  // namespace

bool skinny_supported(int n_tok, int N, int K, int ldx, int ldw) {
  return n_tok >= 1 && N % 32 == 0 && K >= SK_BK && K % SK_BK == 0 && ldx % 8 == 0 && ldw % 8 == 0;
}

// Up to two token tiles the weights stream (almost) once.  Beyond, every further token tile costs about as much as the
// first, and the GEMM with 128 x 256 tiles wins once its tiles cover a quarter of the SMs.  Microseconds, this path / that
// GEMM with nothing else changed: layer steps of the Llama shape over 4500 units (projection and retaining head), 33
// tokens: 53 / 67, 45: 54 / 68, 128: 61 / 73; whole blocks over an empty cache (W_o and the FFN), Llama shape, 33: 137 / 220,
// 128: 159 / 233, 256: 201 / 259, 384: 290 / 293, 512: 339 / 323; Phi-3 shape (its projection of 9216 columns gives up the
// fused RoPE here), 33: 98 / 159, 128: 112 / 169, 256: 135 / 177, 300: 205 / 202; small shape, 256: 61 / 76, 384: 75 / 82.
bool skinny_use(int n_tok, int N, int K, int ldx, int ldw) {
  if (!skinny_supported(n_tok, N, K, ldx, ldw)) return false;
  if (n_tok <= 256) return true;
  const int wide_tiles = ((n_tok + 127) / 128) * ((N + 255) / 256);
  return n_tok <= 512 && wide_tiles * 4 <= sm_count_of_current_device();
}

int skinny_ctas(int n_tok, int N, int K) {
  const SkinnyPlan plan = skinny_plan(n_tok, N, K);
  return plan.tiles * ((n_tok + plan.nt - 1) / plan.nt) * plan.n_split;
}

// The retaining head of a layer step runs beside attention and the next projection.  Up to one token tile its 64 CTAs are
// little to them.  Beyond, what counts is less its own time than the SMs it takes: at 512 tokens (Phi-3 shape, K = 9216) this
// path takes 52 us on 128 SMs, the wide GEMM 87 us on 16, and four layers in turn (1000 cached units) took 130 us a step
// with this one and 100 with that; 384 tokens of the Llama shape, empty cache: 81 / 73.  So beyond 128 tokens it is for
//   matrices so small that it leaves half of the SMs alone (small shape, 512 tokens: 35 / 42 us a step);
//   up to 256 tokens a K so long that the wide GEMM's chain of K-blocks outlasts what it runs beside, as it does from about
//   twice the projection's K on (Phi-3 shape, K = 3 d_model, 200 tokens: 71 / 90; Llama shape, 1.5 d_model: 66 / 61);
//   and where the next step waits for it (awaited: a 4-bit cache's expansion is enqueued behind it) up to 512 tokens
//   (Phi-3 shape, 512 tokens, 1000 cached: 128 / 130, 300 tokens 104 / 120).
// A step that evicts would gain from it as well (Phi-3 shape, budget 700, 300 tokens, four layers: 96 / 118; Llama shape, 200
// tokens: 71 / 75), but the bits of a step's scores must not depend on its flags, and the same step without an eviction
// hands over its output later (one layer, 300 tokens: 112 / 78 us until attention is done).
bool skinny_use_beside(int n_tok, int N, int K, int ldx, int ldw, int d_model, bool awaited) {
  if (!skinny_supported(n_tok, N, K, ldx, ldw)) return false;
  if (n_tok <= 128) return true;
  if (n_tok <= 512 && 2 * skinny_ctas(n_tok, N, K) <= sm_count_of_current_device()) return true;
  return n_tok <= (awaited ? 512 : 256) && K > 2 * d_model;
}

cudaError_t launch_skinny_gemm(const bf16 *X, int ldx, const bf16 *Wt, int ldw, bf16 *Y, int ldy, int n_tok, int N, int K,
                               const bf16 *R, int ldr, int *status, cudaStream_t st, bool pdl) {
  SkinnyParams p = {};
  p.n_tok = n_tok; p.N = N; p.K = K; p.out = Y; p.ldo = ldy; p.resid = R; p.ldr = ldr; p.status = status;
  return launch_skinny<0>(X, ldx, Wt, ldw, p, N, st, pdl);
}

cudaError_t launch_skinny_gated(const bf16 *X, int ldx, const bf16 *Wt, int ldw, bf16 *act, int n_tok, int F, int K,
                                int *status, cudaStream_t st, bool pdl) {
  SkinnyParams p = {};
  p.n_tok = n_tok; p.N = 2 * F; p.K = K; p.out = act; p.ldo = F; p.status = status;
  return launch_skinny<1>(X, ldx, Wt, ldw, p, 2 * F, st, pdl);
}

cudaError_t launch_skinny_rh(const bf16 *Z, int ldz, const bf16 *W1t, const float *W2, float *partial, int n_tok, int d_R,
                             int K, int h_kv, int act, int *n_tiles, int *status, cudaStream_t st) {
  SkinnyParams p = {};
  p.n_tok = n_tok; p.N = d_R; p.K = K; p.W2 = W2; p.partial = partial; p.h_kv = h_kv; p.act = act; p.status = status;
  *n_tiles = (d_R + SK_ROWS - 1) / SK_ROWS;
  return launch_skinny<2>(Z, ldz, W1t, K, p, d_R, st, false);
}

}  // namespace locret

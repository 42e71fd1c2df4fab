// Eq. 1 on tcgen05 tensor cores with TMEM accumulators, head_dim 64, 96 or 128 (tiles are laid
// out for 128 columns; narrower heads load and multiply only their own columns).
//
// One CTA owns two 128-row query tiles that share a KV head (two query heads of one GQA
// group over the same rows, or two consecutive row blocks of one head) and streams the
// keys/values of that head in tiles of 128 through shared memory with TMA.  Roles:
//   warps 0-7        softmax, one query tile at a time (tile 0 and tile 1 alternately, so one
//                    tile's softmax runs while the other tile's MMAs execute).  A warp may only
//                    touch TMEM lanes 32 (w % 4) .. +31, so warps q and 4 + q share the 32 rows of
//                    quarter q and split the tile's 128 keys in halves: each thread reads half a
//                    row of S = Q K^T from TMEM, the pair exchanges its half maxima through shared
//                    memory, and each writes P = exp2(S - max) as bf16 back into TMEM over S (the
//                    first half releases the first four k-steps of P V, the second the rest).
//                    The accumulator is rescaled in TMEM only when the maximum has grown by more
//                    than 2^100.
//   warp 8           TMA producer: Q once, then K and V tiles (two stages each), walking the
//                    unmasked key tiles in a per-CTA rotated order, with an L2 prefetch ahead;
//   warps 9 / 10     issue S_t = Q_t K_j^T (both operands in shared memory) and O_t += P_t V_j
//                    (P from TMEM, V from shared memory) for tile 0 / 1.  The tensor pipe accepts
//                    only about two instructions ahead of execution, so each issuer builds its
//                    descriptors once and advances them by constants, and the other issuer's MMAs
//                    cover the time one spends polling a barrier.
// TMEM columns: S0/P0 [0,128), S1/P1 [128,256), O0 [256,384), O1 [384,512).
// Query row t sees keys [0, len + t]: the retained cache unmasked, the chunk causally.
#include <type_traits>

#include "tc_common.cuh"

namespace locret {

namespace {

using namespace tc;

constexpr int AT_THREADS = 384;  // 3 warpgroups: softmax (two), {TMA, 2 MMA issuers, 1 idle warp}
constexpr int TILE = 128;               // query rows per tile and keys per tile
constexpr int HD = 128;                 // column pitch of a head in shared and tensor memory
constexpr int HALF_BYTES = TILE * 128;  // one 64-column swizzled box of 128 rows: 16 KB
constexpr int TILE_BYTES = 2 * HALF_BYTES;
constexpr int MAX_SPLIT = 8;            // portable cluster size
constexpr int AT_SMEM = 1024 + 6 * TILE_BYTES + 256 + 2048;  // Q0,Q1,K0,K1,V0,V1 + barriers + softmax exchange
static_assert(alone_on_an_sm(AT_SMEM), "it takes all 512 columns of tensor memory");
// The accumulator is rescaled only when a row's maximum has grown by more than 2^100 since the
// scale in use was fixed.  P is stored as bf16 and O, l accumulate in fp32, both with an 8-bit
// exponent, so P <= 2^100 and O <= keys * 2^100 * |v| (< 2^122 for 2^14 keys, |v| < 2^8) stay
// finite, and relative precision does not depend on the common scale.  A small threshold would
// trigger a rescale (a TMEM round trip on the critical path) at almost every tile that holds one
// of the workload's 20x-norm outlier keys.
constexpr float RESCALE_LOG2 = 100.0f;
constexpr float LOWEST = -3.402823466e38f;  // SPLIT: maximum of a row that has not seen a key yet (finite: see its use)
constexpr int PF = 6;       // key tiles prefetched into L2 ahead of the shared-memory pipeline

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max_nan(float a, float b) {  // NaN if either is
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// 2^x of two values <= 127 on the FMA pipe: x = n + f with n = rint(x), a polynomial for 2^f (least squares on the relative
// error over [-1/2, 1/2], reweighted towards its maximum: 9.1e-8, with the fp32 Horner scheme 1.7e-7), and 2^n put
// together from its exponent; at -127 and below the exponent field is 0 and so is the result (a masked key weighs nothing).
__device__ __forceinline__ void exp2_poly2(float x0, float x1, float &y0, float &y1) {
  const uint64_t x = pack_f32x2(max_nan(x0, -127.f), max_nan(x1, -127.f));
  const uint64_t t = add_f32x2(x, pack_f32x2(12582912.f, 12582912.f));  // 1.5 * 2^23: the sum's low bits are rint(x)
  const uint64_t n = add_f32x2(t, pack_f32x2(-12582912.f, -12582912.f));
  const uint64_t f = fma_f32x2(n, pack_f32x2(-1.f, -1.f), x);
  uint64_t y = pack_f32x2(0.00132647203f, 0.00132647203f);
  y = fma_f32x2(y, f, pack_f32x2(0.00967151299f, 0.00967151299f));
  y = fma_f32x2(y, f, pack_f32x2(0.0555073358f, 0.0555073358f));
  y = fma_f32x2(y, f, pack_f32x2(0.240222424f, 0.240222424f));
  y = fma_f32x2(y, f, pack_f32x2(0.693147004f, 0.693147004f));
  y = fma_f32x2(y, f, pack_f32x2(1.f, 1.f));
  float t0, t1;
  unpack_f32x2(t, t0, t1);
  const uint64_t s = pack_f32x2(__uint_as_float((__float_as_uint(t0) << 23) + 0x3f800000u),
                                __uint_as_float((__float_as_uint(t1) << 23) + 0x3f800000u));
  unpack_f32x2(mul_f32x2(y, s), y0, y1);
}
template <int N>
__device__ __forceinline__ void setmaxnreg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void setmaxnreg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

struct AttnParams {
  bf16 *out;
  int n_tok, h, h_kv, d, len, pair_heads;
  float scale_log2;
  int *status;
  PerHead len_m;  // PER_HEAD: KV head m holds len_m.v[m] retained units
  int n_split;    // SPLIT: CTAs of a cluster, each with its share of the key tiles
};

// SPLIT: a cluster of n_split CTAs shares one pair of query tiles and divides its key tiles in
// contiguous ranges, for calls with too few query tiles to fill the GPU.  Each CTA leaves its
// unnormalised accumulator (as [column][row]), row maxima and row sums in its shared memory, and
// rank r combines its share of the columns over all ranks in rank order.  Bound by latency, not by the key tiles:
// 45 tokens over 4500 cached keys of the Llama shape take 29 us in 16 clusters of eight (five key tiles each);
// the mma.sync kernel that took fewer than 64 tokens before needs 124 us (32 CTAs, all keys in sequence).
// PER_HEAD: a budget per KV head.
template <int D, bool SPLIT, bool PER_HEAD>
__global__ void __launch_bounds__(AT_THREADS, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
               const __grid_constant__ CUtensorMap map_v, const AttnParams p) {
  // Head_dim 96: one pair of exponentials in eight goes to the FMA pipe.  With 96 columns a tile's exponentials (1024 cycles
  // of the special-function unit) outweigh its MMAs (768): 157.4 us per launch without, 152.0 us with one pair in
  // eight, 156.2 with one in four, 169.9 with one in two (Phi-3 shape).  At 128 columns every share lost (243.2 us without,
  // 245.7 / 258.7 / 281.6 with).
  constexpr int POLY = D == 96 ? 4 : 0;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char *sQ = smem;                   // [2][TILE_BYTES]
  unsigned char *sK = smem + 2 * TILE_BYTES;  // [2 stages][TILE_BYTES]
  unsigned char *sV = smem + 4 * TILE_BYTES;  // [2 stages][TILE_BYTES]
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + 6 * TILE_BYTES);
  uint64_t *q_full = bars;          // 1
  uint64_t *k_full = bars + 1;      // 2
  uint64_t *v_full = bars + 3;      // 2
  uint64_t *k_empty = bars + 5;     // 2
  uint64_t *v_empty = bars + 7;     // 2
  uint64_t *s_full = bars + 9;      // 2
  uint64_t *p_full = bars + 11;     // 2
  uint64_t *o_full = bars + 13;     // 2
  uint64_t *p_half = bars + 15;     // 2: first 64 keys of P_t written (p_full: all 128)
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 17);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = p.h / p.h_kv;
  const int n_rb = (p.n_tok + TILE - 1) / TILE;

  // which two query tiles; longest key ranges first
  int row0[2], head[2];
  const int n_split = SPLIT ? p.n_split : 1;
  const int unit = SPLIT ? (int)blockIdx.x / n_split : (int)blockIdx.x;
  const int rank = SPLIT ? (int)blockIdx.x - unit * n_split : 0;
  if (p.pair_heads) {
    const int hp = p.h / 2;
    const int rb = n_rb - 1 - unit / hp;
    const int hq = unit % hp;
    row0[0] = row0[1] = rb * TILE;
    head[0] = 2 * hq; head[1] = 2 * hq + 1;
  } else {
    const int n_rp = (n_rb + 1) / 2;
    const int rp = n_rp - 1 - unit / p.h;
    row0[0] = rp * 2 * TILE; row0[1] = row0[0] + TILE;
    head[0] = head[1] = unit % p.h;
  }
  const int kvh = head[0] / g;
  const int len = PER_HEAD ? p.len_m.v[kvh] : p.len;   // retained units of this KV head
  const int n = len + p.n_tok;
  int NK = (len + row0[1] + TILE + TILE - 1) / TILE;
  NK = min(NK, (n + TILE - 1) / TILE);
  const int tile_lo = SPLIT ? rank * NK / n_split : 0;  // (a share may be empty)
  if (SPLIT) NK = (rank + 1) * NK / n_split - tile_lo;
  // The softmax is order independent, so every CTA walks the key tiles that need no mask in its
  // own rotated order: CTAs of one KV head start together, and in a common order they would all
  // ask the L2 for the same K and V lines at the same moment (measured: 1.4x slower).
  // (the CTAs of a cluster are on different tiles anyway)
  const int NF = SPLIT ? 0 : min(NK, (len + row0[0] + 1) / TILE);  // tiles fully visible to every row
  const int rot = NF > 0 ? (int)((blockIdx.x * 29u + 7u) % (unsigned)NF) : 0;
  auto tile_of = [&](int j) { int x = j + rot; return SPLIT ? tile_lo + j : (j < NF ? (x >= NF ? x - NF : x) : j); };

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < 2; s++) {
      mbar_init(&k_full[s], 1); mbar_init(&v_full[s], 1);
      mbar_init(&k_empty[s], 2); mbar_init(&v_empty[s], 2);  // released by both MMA issuers
      mbar_init(&s_full[s], 1); mbar_init(&p_full[s], 4); mbar_init(&o_full[s], 1);
      mbar_init(&p_half[s], 4);
    }
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&map_q); prefetch_tmap(&map_k); prefetch_tmap(&map_v);
  }
  if (warp == 9) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp >= 8) {
    setmaxnreg_dec<56>();
  if (warp == 11) {
    // idle warp of the third warpgroup
  } else if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      constexpr int nbox = (D + 63) / 64;  // 64-column boxes per head vector
      mbar_expect_tx(q_full, 2 * nbox * HALF_BYTES);
      for (int t = 0; t < 2; t++)
        for (int hh = 0; hh < nbox; hh++)
          tma_load_2d(sQ + t * TILE_BYTES + hh * HALF_BYTES, &map_q, head[t] * D + hh * 64, row0[t],
                      q_full);
      // L2 prefetch PF tiles ahead: the cache of a layer is not L2 resident when its chunk step
      // starts, and two stages of shared memory do not cover an HBM miss.
      auto prefetch_tile = [&](int j) {
        const int row = tile_of(j) * TILE;
        for (int hh = 0; hh < nbox; hh++) {
          tma_prefetch_3d(&map_k, hh * 64, row, kvh);
          tma_prefetch_3d(&map_v, hh * 64, row, kvh);
        }
      };
      for (int j = 0; j < min(PF, NK); j++) prefetch_tile(j);
      for (int j = 0; j < NK; j++) {
        const int s = j & 1;
        const uint32_t ph = (j >> 1) & 1;
        if (j + PF < NK) prefetch_tile(j + PF);
        if (!mbar_wait(&k_empty[s], ph ^ 1, abort_flag, p.status)) break;
        mbar_expect_tx(&k_full[s], nbox * HALF_BYTES);
        for (int hh = 0; hh < nbox; hh++)
          tma_load_3d(sK + s * TILE_BYTES + hh * HALF_BYTES, &map_k, hh * 64, tile_of(j) * TILE, kvh, &k_full[s]);
        if (!mbar_wait(&v_empty[s], ph ^ 1, abort_flag, p.status)) break;
        mbar_expect_tx(&v_full[s], nbox * HALF_BYTES);
        for (int hh = 0; hh < nbox; hh++)
          tma_load_3d(sV + s * TILE_BYTES + hh * HALF_BYTES, &map_v, hh * 64, tile_of(j) * TILE, kvh, &v_full[s]);
      }
    }
  } else {
    // ------------------------------------------------------------ MMA issuers: warp 9 for query
    // tile 0, warp 10 for tile 1.  The tensor pipe's queue is only a couple of instructions deep,
    // so an issuer that stops to poll a barrier starves the pipe; with one issuer per tile the
    // other tile's MMAs cover each wait.  Descriptors are built once and advanced by constants.
    if (lane == 0) {
      const int t = warp - 9;
      constexpr uint32_t idesc_qk = idesc_bf16(TILE, TILE, 0, 0);
      constexpr uint32_t idesc_pv = idesc_bf16(TILE, D, 0, 1);
      constexpr int ksteps = D / 16;
      const uint64_t dq = desc_kmajor_sw128(sQ + t * TILE_BYTES);
      const uint64_t dk0 = desc_kmajor_sw128(sK), dk1 = desc_kmajor_sw128(sK + TILE_BYTES);
      const uint64_t dv0 = desc_mnmajor_sw128(sV, HALF_BYTES), dv1 = desc_mnmajor_sw128(sV + TILE_BYTES, HALF_BYTES);
      const uint32_t s_tmem = tmem_base + t * TILE, o_tmem = tmem_base + 2 * TILE + t * HD;
      auto issue_s = [&](int ks) {
        const uint64_t b = ks ? dk1 : dk0;
#pragma unroll
        for (int kk = 0; kk < ksteps; kk++) {
          const uint64_t off = (uint64_t)(((kk >> 2) * HALF_BYTES + (kk & 3) * 32) >> 4);
          if (kk == 0) mma_ss_first(s_tmem, dq + off, b + off, idesc_qk);
          else mma_ss_acc(s_tmem, dq + off, b + off, idesc_qk);
        }
        mma_commit(&s_full[t]);
        mma_commit(&k_empty[ks]);
      };
      // the first four k-steps (keys 0..63) only need the first half of P
      auto issue_pv = [&](int vs, bool acc, int half) {
        const uint64_t b = vs ? dv1 : dv0;
#pragma unroll
        for (int kk = 0; kk < TILE / 16; kk++) {
          if ((kk >> 2) != half) continue;
          const uint64_t off = (uint64_t)((kk * 16 * 128) >> 4);
          if (kk == 0) mma_ts(o_tmem, s_tmem, b, idesc_pv, acc);
          else mma_ts_acc(o_tmem, s_tmem + kk * 8, b + off, idesc_pv);
        }
        if (half == 1) {
          mma_commit(&o_full[t]);
          mma_commit(&v_empty[vs]);
        }
      };
      bool ok = mbar_wait(q_full, 0, abort_flag, p.status);
      if (!SPLIT || NK > 0) ok = ok && mbar_wait(&k_full[0], 0, abort_flag, p.status);
      if (ok && (!SPLIT || NK > 0)) {
        tc_fence_after();
        issue_s(0);
      }
      for (int j = 0; j < NK && ok; j++) {
        const int sv = j & 1, sk = (j + 1) & 1;
        // The tiles from memory arrive long before P does: poll them first, so that nothing but
        // the MMAs themselves stands between P and the next S.
        ok = mbar_wait(&v_full[sv], (j >> 1) & 1, abort_flag, p.status);
        if (j + 1 < NK) ok = ok && mbar_wait(&k_full[sk], ((j + 1) >> 1) & 1, abort_flag, p.status);
        // O_t += P_t V_j
        ok = ok && mbar_wait(&p_half[t], j & 1, abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        issue_pv(sv, j > 0, 0);
        ok = mbar_wait(&p_full[t], j & 1, abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        issue_pv(sv, j > 0, 1);
        // S_t = Q_t K_{j+1}^T
        if (j + 1 < NK) {
          issue_s(sk);
        }
      }
    }
  }
  if (SPLIT) {  // (the softmax warps' two meetings of the cluster)
    __syncwarp();
    cluster_sync_all();
    cluster_sync_all();
  }
  } else {
    // ------------------------------------------------------------ softmax: all eight warps work
    // on one query tile at a time, tile 0 and tile 1 alternately.  Warp w may only touch TMEM
    // lanes 32 (w % 4) .. +31, so warps q and 4 + q share the 32 rows of quarter q and split
    // the tile's 128 keys in halves: two warps per scheduler interleave their exponentials,
    // while the other tile's MMAs run.  The pair exchanges its half maxima through shared
    // memory around a 64-thread named barrier; that barrier also orders the first warp's read
    // of S columns [32, 64) before the second warp's P (keys 64..127) overwrites them.
    setmaxnreg_inc<224>();
    const int hf = warp >> 2, quarter = warp & 3;
    const int r = quarter * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    float *xch = reinterpret_cast<float *>(smem + 6 * TILE_BYTES + 256);  // [tile][half][128 rows]
    const float c = p.scale_log2;
    float m_used[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    bool ok = true;
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + quarter) : "memory"); };

    for (int j = 0; j < NK; j++) {
      // (no early exit: after a timed-out wait the pair still meets at its named barrier)
#pragma unroll
      for (int t = 0; t < 2; t++) {
        const int row = row0[t] + r;
        const int limit = len + row;  // last visible key
        const uint32_t s_addr = tmem_base + lane_off + t * TILE;
        const uint32_t o_addr = tmem_base + lane_off + 2 * TILE + t * HD;
        const int key0 = tile_of(j) * TILE;
        if (ok) ok = mbar_wait(&s_full[t], j & 1, abort_flag, p.status);
        tc_fence_after();
        uint32_t s[64];
        tmem_ld32(s_addr + hf * 64, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
        tmem_ld32(s_addr + hf * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
        tmem_wait_ld();

        float tmax;
        if (key0 + TILE - 1 > len + row0[t]) {  // a tile that crosses the causal boundary
          tmax = -INFINITY;
#pragma unroll
          for (int i = 0; i < 64; i++) {
            float x = (key0 + hf * 64 + i <= limit) ? __uint_as_float(s[i]) : -INFINITY;
            s[i] = __float_as_uint(x);
            tmax = fmaxf(tmax, x);
          }
        } else {
          float tm[8];
#pragma unroll
          for (int a = 0; a < 8; a++) tm[a] = fmaxf(__uint_as_float(s[2 * a]), __uint_as_float(s[2 * a + 1]));
#pragma unroll
          for (int i = 16; i < 64; i += 16)
#pragma unroll
            for (int a = 0; a < 8; a++)
              tm[a] = fmaxf(tm[a], fmaxf(__uint_as_float(s[i + 2 * a]), __uint_as_float(s[i + 2 * a + 1])));
          tmax = fmaxf(fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])), fmaxf(fmaxf(tm[4], tm[5]), fmaxf(tm[6], tm[7])));
        }
        xch[(t * 2 + hf) * TILE + r] = tmax;
        pair_sync();
        tmax = fmaxf(tmax, xch[(t * 2 + (hf ^ 1)) * TILE + r]) * c;
        // a share's first tile may lie wholly behind the causal boundary: -inf less a finite maximum is -inf, not NaN
        if (SPLIT) tmax = fmaxf(tmax, LOWEST);

        if (j == 0) {
          m_used[t] = tmax;
        } else {
          // both warps of the pair see the same maxima, hence take the same branch
          const bool need = tmax > m_used[t] + RESCALE_LOG2;
          if (__any_sync(0xffffffffu, need)) {
            // the accumulator must hold every product issued so far before it is rescaled
            if (ok) ok = mbar_wait(&o_full[t], (j - 1) & 1, abort_flag, p.status);
            tc_fence_after();
            float alpha = 1.0f;
            if (need) { alpha = exp2f(m_used[t] - tmax); m_used[t] = tmax; }
            l[t] *= alpha;
#pragma unroll 1
            for (int q = hf; q < D / 32; q += 2) {  // the pair shares the accumulator's columns
              uint32_t o[32];
              tmem_ld32(o_addr + q * 32, o);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 32; i++) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
              tmem_st32(o_addr + q * 32, o);
            }
            tmem_wait_st();
            // the next product touches every column: both halves must be rescaled before either
            // warp hands over its P
            pair_sync();
          }
        }

        const uint64_t c2 = pack_f32x2(c, c), nm2 = pack_f32x2(-m_used[t], -m_used[t]);
        uint64_t la = pack_f32x2(0.f, 0.f), lb = la;
        uint32_t pk[32];
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          float x0, x1, x2, x3;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nm2), x0, x1);
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i + 2]), __uint_as_float(s[2 * i + 3])), c2, nm2), x2, x3);
          float p2, p3;
          const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
          if (POLY > 0 && (i >> 1) % (POLY > 0 ? POLY : 1) == 0) {
            exp2_poly2(x2, x3, p2, p3);
          } else {
            p2 = ex2_approx(x2);
            p3 = ex2_approx(x3);
          }
          la = add_f32x2(la, pack_f32x2(p0, p1));
          lb = add_f32x2(lb, pack_f32x2(p2, p3));
          pk[i] = pack_bf16(p0, p1);
          pk[i + 1] = pack_bf16(p2, p3);
        }
        tmem_st32(s_addr + hf * 32, pk);
        {
          float a0, a1, b0, b1;
          unpack_f32x2(la, a0, a1);
          unpack_f32x2(lb, b0, b1);
          l[t] += (a0 + a1) + (b0 + b1);
        }
        if (PER_HEAD && t == 0 && key0 + TILE > n) {
          // Slots behind the cache's end hold what an earlier request left there, perhaps NaN, which a weight of 0 does
          // not silence.  map_v ends at the longest head's length, so a shorter head's rows are cleared here: this warp's
          // sixteen of its half of the keys, before it hands over P.  (Compiled into the
          // other calls as well it cost their prefill 1 %.)
          if (ok) ok = mbar_wait(&v_full[j & 1], (j >> 1) & 1, abort_flag, p.status);
          unsigned char *v = sV + (j & 1) * TILE_BYTES;
          const int r_lo = hf * 64 + quarter * 16;
          for (int i = lane; i < (D + 63) / 64 * 128; i += 32) {   // 16-byte pieces: column box, row, piece of 128 bytes
            const int vr = r_lo + ((i >> 3) & 15);
            if (key0 + vr >= n)
              *reinterpret_cast<uint4 *>(v + (i >> 7) * HALF_BYTES + vr * 128 + (i & 7) * 16) = make_uint4(0, 0, 0, 0);
          }
          fence_proxy_async();
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(hf == 0 ? &p_half[t] : &p_full[t]);
      }
    }

    if (SPLIT) {
      // every product of both tiles is complete and every loaded tile consumed: the stages are free
      if (ok && NK > 0) ok = mbar_wait(&o_full[0], (NK - 1) & 1, abort_flag, p.status);
      if (ok && NK > 0) ok = mbar_wait(&o_full[1], (NK - 1) & 1, abort_flag, p.status);
      tc_fence_after();
      float *so = reinterpret_cast<float *>(smem);                            // [tile][column][row]
      float *sm = reinterpret_cast<float *>(smem + 2 * D * TILE * 4);         // [tile][row] maxima, then sums
#pragma unroll
      for (int t = 0; t < 2; t++) {
        const uint32_t o_addr = tmem_base + lane_off + 2 * TILE + t * HD;
        xch[(t * 2 + hf) * TILE + r] = l[t];
        pair_sync();
        if (hf == 0) {
          sm[t * TILE + r] = m_used[t];
          sm[(2 + t) * TILE + r] = l[t] + xch[(t * 2 + 1) * TILE + r];
        }
        if (ok && NK > 0) {
#pragma unroll 1
          for (int q = hf; q < D / 32; q += 2) {
            uint32_t o[32];
            tmem_ld32(o_addr + q * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; i++) so[(t * D + q * 32 + i) * TILE + r] = __uint_as_float(o[i]);
          }
        }
      }
      cluster_sync_all();
      // this rank's share of the columns, four at a time; lanes along rows
      constexpr int G = D / 4;
      const int g_lo = rank * G / n_split, g_hi = (rank + 1) * G / n_split;
      const uint32_t so_a = smem_u32(so), sm_a = smem_u32(sm);
      for (int i = threadIdx.x; i < (g_hi - g_lo) * 2 * TILE; i += 256) {
        const int tr = i & (2 * TILE - 1), t = tr >> 7, c0 = (g_lo + i / (2 * TILE)) * 4;
        const int row = row0[t] + (tr & (TILE - 1));
        if (row >= p.n_tok) continue;
        // (unrolled over the largest cluster: every remote load is in flight before the first is used)
        float mk[MAX_SPLIT], lk[MAX_SPLIT], ok4[MAX_SPLIT][4];
        float mx = LOWEST;
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; k++) {
          mk[k] = LOWEST;
          lk[k] = 0.f;
          if (k >= n_split) continue;
          const uint32_t ma = cluster_map(sm_a, k) + tr * 4;
          const uint32_t oa = cluster_map(so_a, k) + (uint32_t)((t * D + c0) * TILE + (tr & (TILE - 1))) * 4;
          mk[k] = ld_cluster_f1(ma);
          lk[k] = ld_cluster_f1(ma + 2 * TILE * 4);
#pragma unroll
          for (int e = 0; e < 4; e++) ok4[k][e] = ld_cluster_f1(oa + e * TILE * 4);
        }
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; k++) mx = fmaxf(mx, mk[k]);
        float acc[4] = {0.f, 0.f, 0.f, 0.f}, ls = 0.f;
#pragma unroll
        for (int k = 0; k < MAX_SPLIT; k++) {
          // a share without a key for this row has no weight (its maximum would not do: NaN scores count, and raise none)
          if (lk[k] == 0.f) continue;
          const float w = exp2f(mk[k] - mx);
          ls = fmaf(w, lk[k], ls);
#pragma unroll
          for (int e = 0; e < 4; e++) acc[e] = fmaf(w, ok4[k][e], acc[e]);
        }
        const float inv = 1.0f / ls;
        *reinterpret_cast<uint2 *>(p.out + (size_t)row * p.h * D + (size_t)head[t] * D + c0) =
            make_uint2(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv));
      }
      cluster_sync_all();  // no CTA leaves while another may still read its share
    } else {
#pragma unroll
    for (int t = 0; t < 2; t++) {
      const int row = row0[t] + r;
      const uint32_t o_addr = tmem_base + lane_off + 2 * TILE + t * HD;
      if (ok && NK > 0) ok = mbar_wait(&o_full[t], (NK - 1) & 1, abort_flag, p.status);
      tc_fence_after();
      xch[(t * 2 + hf) * TILE + r] = l[t];
      pair_sync();
      const float inv = 1.0f / (l[t] + xch[(t * 2 + (hf ^ 1)) * TILE + r]);
      if (ok) {
        bf16 *dst = p.out + (size_t)row * p.h * D + (size_t)head[t] * D;
#pragma unroll 1
        for (int q = hf; q < D / 32; q += 2) {
          uint32_t o[32];
          tmem_ld32(o_addr + q * 32, o);
          tmem_wait_ld();
          if (row < p.n_tok) {
#pragma unroll
            for (int v = 0; v < 4; v++) {
              uint4 w;
              w.x = pack_bf16(__uint_as_float(o[8 * v + 0]) * inv, __uint_as_float(o[8 * v + 1]) * inv);
              w.y = pack_bf16(__uint_as_float(o[8 * v + 2]) * inv, __uint_as_float(o[8 * v + 3]) * inv);
              w.z = pack_bf16(__uint_as_float(o[8 * v + 4]) * inv, __uint_as_float(o[8 * v + 5]) * inv);
              w.w = pack_bf16(__uint_as_float(o[8 * v + 6]) * inv, __uint_as_float(o[8 * v + 7]) * inv);
              *reinterpret_cast<uint4 *>(dst + q * 32 + v * 8) = w;
            }
          }
        }
      }
    }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 9) {
    __syncwarp();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

bool attention_tc_supported(int n_tok, int h, int h_kv, int d) {
  return (d == 64 || d == 96 || d == 128) && n_tok >= 2 && h % h_kv == 0;
}

namespace {

// Clusters of `size` CTAs of the split kernel that are resident at once on the current device (0: the size cannot be
// launched), asked for once per device and size.
template <int D>
int resident_clusters(int size) {
  static int known[MAX_DEVICES][MAX_SPLIT + 1] = {};  // 0: not asked for yet; value + 1
  int dev = 0;
  if (current_device_index(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
  if (known[dev][size] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(AT_THREADS);
    cfg.dynamicSmemBytes = AT_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attn_tc_kernel<D, true, false>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    known[dev][size] = n + 1;
  }
  return known[dev][size] - 1;
}

template <int D, bool PER_HEAD>
cudaError_t launch_attn_d(const CUtensorMap *map_q, const CUtensorMap *map_k, const CUtensorMap *map_v, AttnParams &p,
                          int grid, int len_max, bool may_divide, cudaStream_t st) {
  static PerDeviceFlag attr_set, attr_set_split;
  if (cudaError_t e = allow_dynamic_smem(attn_tc_kernel<D, false, PER_HEAD>, AT_SMEM, attr_set); e != cudaSuccess) return e;
  if (cudaError_t e = allow_dynamic_smem(attn_tc_kernel<D, true, PER_HEAD>, AT_SMEM, attr_set_split); e != cudaSuccess) return e;
  // The key tiles are divided when that keeps all CTAs resident at once.  (With more than one wave of clusters it lost:
  // 1428 tokens over 3072 cached keys of the Llama shape, 192 CTAs, took 168 us in clusters of two and 104 us undivided.)
  // The combination then costs the time of D / 48 + D / (16 s) key tiles (s CTAs share D columns; half a tile less where
  // half of the rows are padding).  This is a fit over every s at 2 to 1000 tokens and 3 to 36 key tiles of three shapes;
  // its choice is within 2 us of the best one.  A larger cluster has to be a third of a tile better, and one
  // that fills half of the GPU a whole tile: its SMs are missing elsewhere.  300 tokens of the Llama shape, undivided / in clusters of two: 8 tiles 31 / 35 us, 12 tiles 37 / 39,
  // 16 tiles 45 / 43, 36 tiles 82 / 62; 128 tokens, in clusters of four: 6 tiles 25 / 27, 8 tiles 29 / 27.
  const int nk = (len_max + p.n_tok + TILE - 1) / TILE;
  int best = 1, best_cost = 48 * nk;   // in 1/48 of a tile
  for (int s = 2; may_divide && s <= MAX_SPLIT && s <= nk && grid * s <= sm_count_of_current_device(); s++) {
    const int cost = 48 * ((nk + s - 1) / s) + D + 3 * D / s - (p.n_tok <= TILE / 2 ? 24 : 0);
    if (cost < best_cost - (best > 1 ? 16 : 2 * grid * s > sm_count_of_current_device() ? 48 : 0) && grid <= resident_clusters<D>(s)) { best = s; best_cost = cost; }
  }
  p.n_split = best;
  if (best == 1) {
    attn_tc_kernel<D, false, PER_HEAD><<<grid, AT_THREADS, AT_SMEM, st>>>(*map_q, *map_k, *map_v, p);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid * best);
  cfg.blockDim = dim3(AT_THREADS);
  cfg.dynamicSmemBytes = AT_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = best; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, attn_tc_kernel<D, true, PER_HEAD>, *map_q, *map_k, *map_v, static_cast<const AttnParams>(p));
}

}  // namespace

cudaError_t launch_attention_tc(const CUtensorMap *map_q, const CUtensorMap *map_k,
                                const CUtensorMap *map_v, bf16 *out, int n_tok, int h, int h_kv, int d,
                                int len, int *status, cudaStream_t st, const PerHead *len_m, bool may_divide) {
  AttnParams p;
  p.out = out; p.n_tok = n_tok; p.h = h; p.h_kv = h_kv; p.d = d; p.len = len;
  p.len_m = len_m ? *len_m : PerHead{};
  p.pair_heads = ((h / h_kv) % 2 == 0) ? 1 : 0;
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)d);
  p.status = status;
  const int n_rb = (n_tok + TILE - 1) / TILE;
  const int grid = p.pair_heads ? n_rb * (h / 2) : ((n_rb + 1) / 2) * h;
  int len_max = len;
  if (len_m)
    for (int m = 0; m < h_kv; m++) len_max = len_m->v[m] > len_max ? len_m->v[m] : len_max;
  auto launch = [&](auto dim) -> cudaError_t {
    constexpr int D = decltype(dim)::value;
    return len_m ? launch_attn_d<D, true>(map_q, map_k, map_v, p, grid, len_max, may_divide, st)
                 : launch_attn_d<D, false>(map_q, map_k, map_v, p, grid, len_max, may_divide, st);
  };
  switch (d) {
    case 64: return launch(std::integral_constant<int, 64>{});
    case 96: return launch(std::integral_constant<int, 96>{});
    case 128: return launch(std::integral_constant<int, 128>{});
  }
  return cudaErrorInvalidValue;
}

}  // namespace locret

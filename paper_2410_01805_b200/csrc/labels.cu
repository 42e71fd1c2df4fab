// Training labels of the retaining head (Section 3.3): for prompt key k of KV head m the largest product with
// an answer query of the head's group, labels[m][k] = scale * max_{p, j in group m} q_{p,j} . k_{k,m}.
//
// A contraction whose result is reduced to row maxima at once: 2 n_q n_a h d operations, nothing but the maxima
// written.  The contraction is shallow (d <= 128), so what matters is what stays in place: a CTA keeps two tiles
// of 128 keys in shared memory and streams the group's queries past them in tiles of up to 256 rows
// (answers x heads of the group, one three-dimensional TMA box), so a query tile is read from L2 once for
// 256 keys, and the two accumulators (2 x 256 TMEM columns) take turns: one is reduced while the other is
// multiplied.  Eight warps reduce, each thread one row's maximum over half the columns, three-input maxima, all
// query tiles of a work unit before one atomic maximum per row on the order-preserving integer image.
// One launch for all heads (a launch of the 128 x 256 GEMM per query head before: two K-blocks per tile, the keys
// re-read for every head).  131072 keys, 1024 answers, 32 query heads of 8 KV heads of 128: 0.84 ms a call in a loop, under
// the power cap, = 1.31 PFLOP/s (1.55 ms before); one call after a pause 0.70 ms; the measured burst peak allows 0.64 ms.
#include <atomic>
#include <thread>

#include "../../include/locret.h"
#include "tc_common.cuh"

using namespace locret;

namespace {

using namespace locret::tc;

constexpr int LB_THREADS = 320;              // warps 0-7 reduce, 8 TMA, 9 MMA
constexpr int LB_ROWS = 128, LB_COLS = 256;
constexpr int LB_A_BLOCK = LB_ROWS * 128;    // 64 columns of a key tile, swizzled: 16 KB
constexpr int LB_B_BLOCK = LB_COLS * 128;    // 64 columns of a query tile: 32 KB
constexpr int LB_B_BLOCKS = 4;               // resident: two query tiles of d > 64, four of d = 64
constexpr int LB_SMEM = 1024 + 4 * LB_A_BLOCK + LB_B_BLOCKS * LB_B_BLOCK + 256;

static_assert(alone_on_an_sm(LB_SMEM), "it takes all 512 columns of tensor memory");

struct LabelParams {
  float *labels;
  int n_q, n_a, h_kv, d, g, gb;  // gb: heads of the group in one query tile (a power of two)
  int pairs;                     // pairs of key tiles per KV head
  int q_tiles, splits;           // query tiles per KV head; work units they are divided into
  float scale;
  int *status;
};

__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }

template <int D>
__global__ void __launch_bounds__(LB_THREADS, 1)
labels_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_q, const LabelParams p) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char *sA = smem, *sB = smem + 4 * LB_A_BLOCK;  // sA: [tile][64-column block]
  constexpr int KB = (D + 63) / 64, KSTEPS = D / 16;
  constexpr int LB_STAGES = LB_B_BLOCKS / KB;  // a stage holds one query tile
  uint64_t *bars = reinterpret_cast<uint64_t *>(sB + LB_B_BLOCKS * LB_B_BLOCK);
  uint64_t *b_full = bars, *b_empty = bars + LB_STAGES;
  uint64_t *a_full = bars + 2 * LB_STAGES, *a_empty = a_full + 2, *acc_full = a_empty + 2, *acc_empty = acc_full + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < LB_STAGES; s++) { mbar_init(&b_full[s], 1); mbar_init(&b_empty[s], 1); }
    for (int i = 0; i < 2; i++) {
      mbar_init(&a_full[i], 1); mbar_init(&a_empty[i], 1);
      mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 8);
    }
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&map_k); prefetch_tmap(&map_q);
  }
  if (warp == 9) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  const int per_q = LB_COLS / p.gb;                        // answers in a query tile
  const int a_tiles = (p.n_a + per_q - 1) / per_q;         // query tiles of one set of gb heads
  const int units = p.h_kv * p.pairs * p.splits;
  // unit -> KV head, first key, query tiles [t0, t1)
  auto unit_of = [&](int u, int &m, int &key0, int &t0, int &t1) {
    const int sp = u % p.splits, v = u / p.splits;
    m = v / p.pairs;
    key0 = (v - m * p.pairs) * 2 * LB_ROWS;
    t0 = (int)((long long)sp * p.q_tiles / p.splits);
    t1 = (int)((long long)(sp + 1) * p.q_tiles / p.splits);
  };
  // A query tile t is answers [at * per_q, ..) of the heads of set js, t = js * a_tiles + at; the loops below step
  // (js, at) instead of dividing: the issuing thread must not spend more than the two or three instructions that
  // the tensor pipe queues ahead (with divisions and per-step descriptors it took 197 cycles per MMA of 128).
  auto valid_of = [&](int at) { return min(per_q, p.n_a - at * per_q) * p.gb; };  // columns of a query tile

  if (warp == 8) {
    if (lane == 0) {
      uint32_t it = 0, un = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, un++) {
        int m, key0, t0, t1;
        unit_of(u, m, key0, t0, t1);
        for (int i = 0; i < 2 && ok; i++) {  // (a tile past the end is loaded as zeros and not stored)
          ok = mbar_wait(&a_empty[i], (un & 1) ^ 1, abort_flag, p.status);
          if (!ok) break;
          mbar_expect_tx(&a_full[i], KB * LB_A_BLOCK);
#pragma unroll
          for (int kb = 0; kb < KB; kb++)
            tma_load_3d(sA + (i * 2 + kb) * LB_A_BLOCK, &map_k, kb * 64, m, key0 + i * LB_ROWS, &a_full[i]);
        }
        int js = t0 / a_tiles, at = t0 - js * a_tiles;
        for (int t = t0; t < t1 && ok; t++, it++) {
          const int s = it % LB_STAGES;
          ok = mbar_wait(&b_empty[s], ((it / LB_STAGES) & 1) ^ 1, abort_flag, p.status);
          if (!ok) break;
          mbar_expect_tx(&b_full[s], KB * LB_B_BLOCK);
#pragma unroll
          for (int kb = 0; kb < KB; kb++)
            tma_load_3d(sB + (s * KB + kb) * LB_B_BLOCK, &map_q, kb * 64, m * p.g + js * p.gb, at * per_q, &b_full[s]);
          if (++at == a_tiles) { at = 0; js++; }
        }
      }
    }
  } else if (warp == 9) {
    if (lane == 0) {
      const uint64_t da0 = desc_kmajor_sw128(sA), db0 = desc_kmajor_sw128(sB);
      uint32_t un = 0, nt = 0;  // units and query tiles seen so far
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, un++) {
        int m, key0, t0, t1;
        unit_of(u, m, key0, t0, t1);
        int at = t0 % a_tiles;
        for (int t = t0; t < t1 && ok; t++, nt++) {
          const uint32_t idesc = idesc_bf16(LB_ROWS, (valid_of(at) + 15) & ~15, 0, 0);
          if (++at == a_tiles) at = 0;
          const int s = nt % LB_STAGES;
          const uint64_t db = db0 + (uint64_t)(s * (KB * LB_B_BLOCK >> 4));
          ok = mbar_wait(&b_full[s], (nt / LB_STAGES) & 1, abort_flag, p.status);
#pragma unroll
          for (int i = 0; i < 2; i++) {
            if (t == t0) ok = ok && mbar_wait(&a_full[i], un & 1, abort_flag, p.status);
            ok = ok && mbar_wait(&acc_empty[i], (nt & 1) ^ 1, abort_flag, p.status);
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = da0 + (uint64_t)(i * (2 * LB_A_BLOCK >> 4));
#pragma unroll
            for (int kk = 0; kk < KSTEPS; kk++) {
              const uint64_t ao = (uint64_t)((kk >> 2) * (LB_A_BLOCK >> 4) + (kk & 3) * 2);
              const uint64_t bo = (uint64_t)((kk >> 2) * (LB_B_BLOCK >> 4) + (kk & 3) * 2);
              if (kk == 0) mma_ss_first(tmem + i * LB_COLS, da + ao, db + bo, idesc);
              else mma_ss_acc(tmem + i * LB_COLS, da + ao, db + bo, idesc);
            }
            mma_commit(&acc_full[i]);
            if (t == t1 - 1) mma_commit(&a_empty[i]);
          }
          if (ok) mma_commit(&b_empty[s]);
        }
      }
    }
  } else {
    const int hf = warp >> 2, quarter = warp & 3;
    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
    uint32_t nt = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
      int m, key0, t0, t1;
      unit_of(u, m, key0, t0, t1);
      float mx[2] = {-INFINITY, -INFINITY};
      int at = t0 % a_tiles;
      for (int t = t0; t < t1; t++, nt++) {
        const int valid = valid_of(at);
        if (++at == a_tiles) at = 0;
#pragma unroll
        for (int i = 0; i < 2; i++) {
          if (ok) ok = mbar_wait(&acc_full[i], nt & 1, abort_flag, p.status);
          tc_fence_after();
          const uint32_t base = taddr + i * LB_COLS + hf * (LB_COLS / 2);
          float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll 1
          for (int c0 = 0; c0 < LB_COLS / 2; c0 += 64) {
            const int left = valid - hf * (LB_COLS / 2) - c0;
            if (left <= 0) break;
            uint32_t r[64];
            tmem_ld32(base + c0, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
            tmem_ld32(base + c0 + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
            tmem_wait_ld();
            if (left < 64) {
#pragma unroll
              for (int e = 0; e < 64; e++)
                if (e >= left) r[e] = 0xff800000u;
            }
#pragma unroll
            for (int e = 0; e < 64; e += 8) {
              m0 = max3(m0, __uint_as_float(r[e]), __uint_as_float(r[e + 1]));
              m1 = max3(m1, __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
              m2 = max3(m2, __uint_as_float(r[e + 4]), __uint_as_float(r[e + 5]));
              m3 = max3(m3, __uint_as_float(r[e + 6]), __uint_as_float(r[e + 7]));
            }
          }
          mx[i] = fmaxf(max3(mx[i], m0, m1), fmaxf(m2, m3));
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 2; i++) {
        const int key = key0 + i * LB_ROWS + quarter * 32 + lane;
        if (ok && key < p.n_q && mx[i] > -INFINITY) {
          float v = mx[i] * p.scale;
          if (v == 0.f) v = 0.f;  // -0 would order below every negative as an integer
          float *dst = p.labels + (size_t)m * p.n_q + key;
          if (v >= 0.f) atomicMax(reinterpret_cast<int *>(dst), __float_as_int(v));
          else atomicMin(reinterpret_cast<unsigned int *>(dst), __float_as_uint(v));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 9) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

__global__ void labels_init_kernel(float *labels, size_t n, int *status) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) labels[i] = -INFINITY;
  if (i == 0) *status = 0;
}
// The word that a timed-out wait writes, one per call in flight: a call (synchronous, so there are no more of them than host
// threads) takes a free one of its device for its duration.
constexpr int STATUS_WORDS = 64;
__device__ int g_cis_status[STATUS_WORDS];
std::atomic<unsigned long long> g_cis_taken[MAX_DEVICES];

struct StatusWord {
  int dev = 0, slot = -1;
  int *word = nullptr;
  cudaError_t take() {
    if (cudaError_t e = current_device_index(&dev); e != cudaSuccess) return e;
    if (cudaError_t e = cudaGetSymbolAddress((void **)&word, g_cis_status); e != cudaSuccess) return e;
    unsigned long long taken = g_cis_taken[dev].load();
    for (;;) {
      if (~taken == 0) {   // 64 calls are in flight: one of them is about to end
        std::this_thread::yield();
        taken = g_cis_taken[dev].load();
        continue;
      }
      const int s = __builtin_ctzll(~taken);
      if (g_cis_taken[dev].compare_exchange_weak(taken, taken | 1ull << s)) { slot = s; word += s; return cudaSuccess; }
    }
  }
  ~StatusWord() { if (slot >= 0) g_cis_taken[dev].fetch_and(~(1ull << slot)); }
};

}  // namespace

#define LCK(call)                                                            \
  do {                                                                       \
    cudaError_t e__ = (call);                                                \
    if (e__ != cudaSuccess) { cudaGetLastError(); return LOCRET_ERR_CUDA; }  \
  } while (0)

extern "C" int locret_cis_labels(const void *q_ans, const void *k_prompt, int32_t n_a, int32_t n_q, int32_t h,
                                 int32_t h_kv, int32_t d, float scale, float *labels, void *stream) {
  if (!q_ans || !k_prompt || !labels) return LOCRET_ERR_INVALID;
  if (n_a < 1 || n_q < 1 || h < 1 || h_kv < 1 || h % h_kv || (d != 64 && d != 96 && d != 128) || !(scale > 0.f))
    return LOCRET_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(q_ans) | reinterpret_cast<uintptr_t>(k_prompt)) & 15u) return LOCRET_ERR_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  LabelParams p;
  p.labels = labels; p.n_q = n_q; p.n_a = n_a; p.h_kv = h_kv; p.d = d; p.scale = scale;
  p.g = h / h_kv;
  p.gb = 1;
  while (p.g % (2 * p.gb) == 0 && p.gb < 16) p.gb *= 2;
  CUtensorMap mk, mq;
  if (!tmap_encode_3d_bf16(&mk, k_prompt, d, h_kv, n_q, (uint64_t)d * 2, (uint64_t)h_kv * d * 2, 64, 1, LB_ROWS) ||
      !tmap_encode_3d_bf16(&mq, q_ans, d, h, n_a, (uint64_t)d * 2, (uint64_t)h * d * 2, 64, p.gb, LB_COLS / p.gb))
    return LOCRET_ERR_CUDA;
  const int per_q = LB_COLS / p.gb, sms = sm_count_of_current_device();
  p.pairs = (n_q + 2 * LB_ROWS - 1) / (2 * LB_ROWS);
  p.q_tiles = (n_a + per_q - 1) / per_q * (p.g / p.gb);
  // Work units: enough of them that the last wave costs little (sixteen per SM), but at least two query tiles each,
  // which is what hides the loading of the next unit's keys.
  p.splits = 1;
  while (h_kv * p.pairs * p.splits < 16 * sms && p.q_tiles / (2 * p.splits) >= 2) p.splits *= 2;
  const long long units = (long long)h_kv * p.pairs * p.splits;
  if (units > 0x7fffffffll) return LOCRET_ERR_INVALID;
  StatusWord own;
  LCK(own.take());
  p.status = own.word;
  const size_t n = (size_t)h_kv * n_q;
  labels_init_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(labels, n, p.status);
  LCK(cudaGetLastError());
  auto launch = [&](auto kernel, PerDeviceFlag &attr_set) -> cudaError_t {
    if (cudaError_t e = allow_dynamic_smem(kernel, LB_SMEM, attr_set); e != cudaSuccess) return e;
    kernel<<<(unsigned)(units < sms ? units : sms), LB_THREADS, LB_SMEM, st>>>(mk, mq, p);
    return cudaGetLastError();
  };
  static PerDeviceFlag attr_set[3];
  if (d == 64) LCK(launch(labels_kernel<64>, attr_set[0]));
  else if (d == 96) LCK(launch(labels_kernel<96>, attr_set[1]));
  else LCK(launch(labels_kernel<128>, attr_set[2]));
  int status = 0;
  LCK(cudaMemcpyAsync(&status, p.status, sizeof(int), cudaMemcpyDeviceToHost, st));
  LCK(cudaStreamSynchronize(st));
  return status ? LOCRET_ERR_DEVICE_TIMEOUT : LOCRET_OK;
}

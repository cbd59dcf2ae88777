// Input projections Q = X W^Q, K = X W^K, V = X W^V (paper: "Mathematical Framework", the projection equation)
// for all heads at once, written straight into the [B, H, tokens, d] layout the attention kernels read.
//
// One GEMM C[tokens, cols] = X[tokens, d_model] * W[d_model, cols] on the sm_100a tensor cores, where the columns
// of W are the projection matrices side by side ([W^Q of heads 0..H-1 | W^K ... | W^V ...], d columns per head).
// Persistent CTAs, one per SM, walk 128 x 256 output tiles (column tiles fastest, so that the CTAs running at the
// same time share the rows of X in L2; W stays L2-resident):
//   warp 0   : TMA producer.  X tile {64 k x 128 tokens} (K-major A operand) and four {64 columns x 64 k} boxes
//              of W (MN-major B operand: W is used as the caller stores it), 128-byte swizzle, 4-stage ring.
//   warp 1   : allocates tensor memory (two 256-column accumulators); one elected thread issues tcgen05.mma
//              (M = 128, N = 256, K = 16) and commits the ring's "empty" barriers and the accumulator's "full".
//   warps 2-5: epilogue of tile i while the MMAs of tile i + 1 fill the other accumulator: tcgen05.ld, round to
//              bf16, and, 32 rows x 64 columns at a time through shared memory, one TMA store to their head's place in Q, K or
//              V (whole 128-byte lines by the threads where the rows belong to two batch elements).
// The tokens of all batch elements form one sequence of rows: a tile may straddle two of them.  Tokens and columns beyond
// the last and k beyond d_model are zero-filled by TMA and skipped by the epilogue.  The tiles that would make a last,
// partial wave are taken in pieces where that fills it better.
// 32 images of 197 tokens, d_model = 768 -> 2304 columns: 29.2 -> 23.2 us, one such image 9.7 -> 6.5 us.  What bounds it there: three rounds of tiles of
// ~8500 cycles, 6100 of them products, 3000 until the first chunk is there and 3600 for the last epilogue.  TMA stores in the place of the threads'
// 16-byte stores of rearranged lines: 23.6 -> 22.8 us, 12000 x 384 -> 1152 19.1 -> 16.1, 16000 x 256 -> 768 16.9 -> 13.4.
// Every wait is bounded (see sm100_ptx.cuh).
#include "csat_internal.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace csat {
namespace {

using namespace ptx;

template <typename T> __device__ __forceinline__ float to_float(T v);
template <> __device__ __forceinline__ float to_float<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_float(float v);
template <> __device__ __forceinline__ float from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

constexpr int kTileM = 128, kTileN = 256, kChunkK = 64, kStages = 4, kThreads = 192;
constexpr uint32_t kABytes = kTileM * kChunkK * 2;       // 16 KB
constexpr uint32_t kBoxBytes = 64 * kChunkK * 2;         // 8 KB: 64 columns x 64 k
constexpr int kBoxes = kTileN / 64;
constexpr uint32_t kStageBytes = kABytes + kBoxes * kBoxBytes;
constexpr uint32_t kOutBytes = 32 * 128;                 // one epilogue warp's 32 rows of a 64-column box
constexpr int kOutBufs = 2;                              // per epilogue warp
constexpr uint32_t kSmemBytes = kStages * kStageBytes + 4 * kOutBufs * kOutBytes + 1024 /*alignment slack*/ + 256 /*barriers*/;

struct ProjArgs {
  __nv_bfloat16* dst[3];      // Q, K, V (any may be null if its columns are not in [col0, col0 + ncols))
  int64_t rows[3];            // tokens per (batch, head) of each destination: n_q, n, n
  int n_tok, B, H, dm;        // tokens per batch element of X; batch; heads; reduction length
  int col0, ncols;            // columns of W this launch computes
  int ntiles;                 // column tiles
  int whole, units, pieces;   // units of work: `whole` whole tiles of 256 columns, then the others in 1, 2 or 4 pieces
};

// Q, K, V as [B H, tokens, d] in boxes of 32 tokens x 64 features
struct OutMaps { const CUtensorMap* m[3]; };

// unit u: row tile, first column, number of 64-column boxes
struct Unit {
  int mt, col, boxes;
  __device__ __forceinline__ Unit(const ProjArgs& a, int u) {
    const int rest = u - a.whole, tile = rest < 0 ? u : a.whole + rest / a.pieces;
    boxes = rest < 0 ? kBoxes : kBoxes / a.pieces;
    mt = tile / a.ntiles;
    col = (tile % a.ntiles) * kTileN + (rest < 0 ? 0 : (rest % a.pieces) * boxes * 64);
  }
};

// The epilogue warps' walk over a CTA's units (q: TMEM lanes [32q, 32q+32); rank: the CTA's half of a pair's rows, -1: no pair)
template <int D, typename Release>
__device__ __forceinline__ bool epilogue(const ProjArgs& a, const OutMaps& maps, uint32_t tmem_base, uint8_t* o_buf, int q, int lane, int first, int step, int rank,
                                         uint64_t* acc_full, int* status, int* cta_abort, Release release) {
  const int HD = a.H * D;
  uint32_t tc = 0;
  bool ok = true;
  const int n_rows = a.B * a.n_tok;
  uint32_t n_box = 0;                                     // boxes of this warp so far (buffer n_box & 1)
  for (int u = first; u < a.units && ok; u += step, ++tc) {
    const Unit t(a, u);
    const uint32_t buf = tc & 1;
    ok = mbar_wait(&acc_full[buf], (tc >> 1) & 1, status, 304, cta_abort) && *(volatile int*)cta_abort == 0;
    if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
    tc_fence_after();
    const int row = (rank < 0 ? t.mt : 2 * t.mt + rank) * kTileM + q * 32 + lane;      // of all tokens; this lane's accumulator row
    const int b = row / a.n_tok, tok = row - b * a.n_tok;
    // the warp's rows belong to one batch element (or lie beyond the tokens): one copy takes a box, clipped at the last token
    const bool whole = __shfl_sync(0xffffffffu, b, 0) == __shfl_sync(0xffffffffu, b, 31) || __shfl_sync(0xffffffffu, row - tok + a.n_tok, 0) >= n_rows;
#pragma unroll 1
    for (int g = 0; g < t.boxes; ++g) {
      const int rel = t.col + g * 64;                   // column within this launch's range
      if (rel >= a.ncols) break;
      uint32_t r[64];
      const uint32_t src = tmem_base + ((uint32_t)(q * 32) << 16) + buf * kTileN + (uint32_t)(g * 64);
      tmem_ld_32x32b_x32(src, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
      tmem_ld_32x32b_x32(src + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
      tmem_wait_ld();
      // 64 consecutive columns lie inside one head (d is a multiple of 64): which matrix, head, column
      const int col = a.col0 + rel, which = col / HD, hh = (col % HD) / D, c = col % D;
      // element offset of this lane's row in the destination, -1 beyond the tokens
      const int64_t off = row < n_rows ? (((int64_t)b * a.H + hh) * a.rows[which] + tok) * D + c : -1;
      uint8_t* stage = o_buf + (q * kOutBufs + (int)(n_box++ & 1)) * kOutBytes;
      if (lane == 0) bulk_wait_group_read1();           // the copy from this buffer, two boxes ago, has read it
      __syncwarp();
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          __nv_bfloat162 p = __floats2bfloat162_rn(__uint_as_float(r[8 * v + 2 * j]), __uint_as_float(r[8 * v + 2 * j + 1]));
          w[j] = *reinterpret_cast<uint32_t*>(&p);
        }
        *reinterpret_cast<uint4*>(stage + lane * 128 + ((v ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      if (whole) {
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          if (row < n_rows) tma_store_3d(maps.m[which], stage, c, tok, b * a.H + hh);
          bulk_commit_group();
        }
        continue;
      }
      if (lane == 0) bulk_commit_group();               // (keeps the count of boxes and groups in step)
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {                     // 4 rows per instruction, 8 lanes (128 bytes) each
        const int rr = 4 * i + (lane >> 3), v = lane & 7;
        const int64_t o = __shfl_sync(0xffffffffu, off, rr);
        const uint4 x = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((v ^ (rr & 7)) << 4));
        if (o >= 0) *reinterpret_cast<uint4*>(a.dst[which] + o + v * 8) = x;
      }
    }
    tc_fence_before();
    release(buf);
  }
  if (lane == 0) bulk_wait_group0();                      // the stores are done before the kernel ends
  return ok;                                              // (the same in every lane)
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
project_sm100_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                     const __grid_constant__ CUtensorMap tmap_oq, const __grid_constant__ CUtensorMap tmap_ok,
                     const __grid_constant__ CUtensorMap tmap_ov, const ProjArgs a, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* a_buf = smem;                                  // [stages][16 KB]
  uint8_t* b_buf = smem + kStages * kABytes;              // [stages][boxes][8 KB]
  uint8_t* o_buf = smem + kStages * kStageBytes;          // [epilogue warp][2][4 KB]
  uint64_t* full = reinterpret_cast<uint64_t*>(o_buf + 4 * kOutBufs * kOutBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;                   // [2]
  uint64_t* acc_empty = acc_full + 2;                     // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  int* cta_abort = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = (a.dm + kChunkK - 1) / kChunkK;

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_x);
    prefetch_tmap(&tmap_w);
    for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int u = 0; u < 2; ++u) { mbar_init(&acc_full[u], 1); mbar_init(&acc_empty[u], 4 * 32); }
    *cta_abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 2 * kTileN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (elect_one()) {
      uint32_t it = 0;                                    // chunks loaded so far (ring position)
      bool ok = true;
      for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
        const Unit t(a, u);
        for (int k = 0; k < nk && ok; ++k, ++it) {
          const int s = it % kStages;
          ok = mbar_wait(&empty[s], ((it / kStages) & 1) ^ 1, status, 301, cta_abort);
          if (!ok) break;
          mbar_arrive_expect_tx(&full[s], kABytes + t.boxes * kBoxBytes);
          tma_load_3d(a_buf + s * kABytes, &tmap_x, &full[s], k * kChunkK, t.mt * kTileM, 0);
          for (int g = 0; g < t.boxes; ++g)
            tma_load_3d(b_buf + (s * kBoxes + g) * kBoxBytes, &tmap_w, &full[s], a.col0 + t.col + g * 64, k * kChunkK, 0);
        }
      }
      if (!ok) {
        // gave up: let copies that are still in flight land before the CTA's shared memory goes away
        for (uint32_t i = it > (uint32_t)kStages ? it - kStages : 0; i < it; ++i)
          mbar_wait_drain(&full[i % kStages], (i / kStages) & 1);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      constexpr uint32_t idesc_whole = make_idesc_bf16(kTileM, kTileN, /*A MN-major*/ false, /*B MN-major*/ true);
      const uint32_t idesc_piece = a.pieces == 1   ? idesc_whole
                                   : a.pieces == 2 ? make_idesc_bf16(kTileM, kTileN / 2, false, true)
                                                   : make_idesc_bf16(kTileM, kTileN / 4, false, true);
      uint32_t it = 0, tc = 0;                            // chunks consumed; tiles of this CTA so far
      bool ok = true;
      for (int u = blockIdx.x; u < a.units && ok; u += gridDim.x, ++tc) {
        const uint32_t buf = tc & 1, idesc = u < a.whole ? idesc_whole : idesc_piece;
        ok = mbar_wait(&acc_empty[buf], ((tc >> 1) & 1) ^ 1, status, 302, cta_abort);   // the epilogue has read it
        if (!ok) break;
        tc_fence_after();
        const uint32_t acc = tmem_base + buf * kTileN;
        for (int k = 0; k < nk; ++k, ++it) {
          const int s = it % kStages;
          ok = mbar_wait(&full[s], (it / kStages) & 1, status, 303, cta_abort);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a_desc = make_smem_desc(smem_u32(a_buf + s * kABytes), 16, 1024);
          const uint64_t b_desc = make_smem_desc(smem_u32(b_buf + s * kBoxes * kBoxBytes), kBoxBytes, 1024);
#pragma unroll
          for (int kk = 0; kk < kChunkK / 16; ++kk)       // +32 B along K for A, +2048 B (16 k rows) for B
            mma_f16_ss(acc, a_desc + (uint64_t)(kk * 2), b_desc + (uint64_t)(kk * 128), idesc, (k | kk) != 0);
          mma_commit(&empty[s]);                          // stage reusable once these MMAs have read it
        }
        mma_commit(&acc_full[buf]);                       // arrives when the tile's MMAs have finished
      }
    }
  } else {
    epilogue<D>(a, OutMaps{{&tmap_oq, &tmap_ok, &tmap_ov}}, tmem_base, o_buf, warp & 3, lane, blockIdx.x, gridDim.x, -1, acc_full, status, cta_abort,
                [&](uint32_t buf) { mbar_arrive(&acc_empty[buf]); });      // 128 arrivals: the accumulator may be overwritten
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, 2 * kTileN);
}

// The same on pairs of CTAs (cta_group::2): 256 x 256 tiles, each CTA with its 128 rows of X and half of the columns of W, so that a chunk
// of 64 k takes 32 instead of 48 KB per SM for the same 512 cycles of products (the kernel above takes 580 to 750 per chunk).  Rank 0's elected thread issues; an accumulator is free once the epilogue warps of both CTAs have arrived.
constexpr int kPairStages = 6;
constexpr uint32_t kPairStageBytes = kABytes + 2 * kBoxBytes;
constexpr uint32_t kPairSmemBytes = kPairStages * kPairStageBytes + 4 * kOutBufs * kOutBytes + 1024 /*alignment slack*/ + 256 /*barriers*/;
static_assert(kPairSmemBytes <= 227 * 1024 && kSmemBytes <= 227 * 1024, "shared memory budget");

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
project_pair_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                    const __grid_constant__ CUtensorMap tmap_oq, const __grid_constant__ CUtensorMap tmap_ok,
                    const __grid_constant__ CUtensorMap tmap_ov, const ProjArgs a, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* o_buf = smem + kPairStages * kPairStageBytes;  // [epilogue warp][2][4 KB]
  uint64_t* full = reinterpret_cast<uint64_t*>(o_buf + 4 * kOutBufs * kOutBytes);      // rank 0's count
  uint64_t* empty = full + kPairStages;
  uint64_t* acc_full = empty + kPairStages;               // [2]
  uint64_t* acc_empty = acc_full + 2;                     // [2], rank 0's count
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  PairEnd* end = reinterpret_cast<PairEnd*>(tmem_slot + 1);
  int* cta_abort = &end->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int first = blockIdx.x >> 1, step = gridDim.x >> 1, nk = (a.dm + kChunkK - 1) / kChunkK;

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_x);
    prefetch_tmap(&tmap_w);
    for (int s = 0; s < kPairStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int u = 0; u < 2; ++u) { mbar_init(&acc_full[u], 1); mbar_init(&acc_empty[u], 2 * 4); }
    end->init();
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, 2 * kTileN);
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                         // both CTAs' barriers are set up
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    if (elect_one()) {
      uint32_t it = 0;                                    // chunks loaded so far (ring position)
      bool ok = true;
      for (int u = first; u < a.units && ok; u += step) {
        const Unit t(a, u);
        const int half = t.boxes / 2;                     // boxes of W in each CTA
        for (int k = 0; k < nk && ok; ++k, ++it) {
          const int s = it % kPairStages;
          ok = mbar_wait(&empty[s], ((it / kPairStages) & 1) ^ 1, status, 311, cta_abort);
          if (!ok) break;
          if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * (kABytes + half * kBoxBytes));
          const uint32_t bar = cluster_smem_u32(&full[s], 0);
          uint8_t* st = smem + s * kPairStageBytes;
          tma_load_3d_pair(st, &tmap_x, bar, k * kChunkK, (2 * t.mt + (int)rank) * kTileM, 0);
          for (int g = 0; g < half; ++g)
            tma_load_3d_pair(st + kABytes + g * kBoxBytes, &tmap_w, bar, a.col0 + t.col + ((int)rank * half + g) * 64, k * kChunkK, 0);
        }
      }
      if (!ok) end->give_up();
      end->producer_done(rank, (int)it);
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc_whole = make_idesc_bf16(2 * kTileM, kTileN, /*A MN-major*/ false, /*B MN-major*/ true);
      const uint32_t idesc_piece = a.pieces == 1 ? idesc_whole : make_idesc_bf16(2 * kTileM, kTileN / 2, false, true);
      uint32_t it = 0, tc = 0;                            // chunks consumed; tiles so far
      bool ok = true;
      for (int u = first; u < a.units && ok; u += step, ++tc) {
        const uint32_t buf = tc & 1, idesc = u < a.whole ? idesc_whole : idesc_piece;
        ok = mbar_wait(&acc_empty[buf], ((tc >> 1) & 1) ^ 1, status, 312, cta_abort);   // both epilogues have read it
        if (!ok) break;
        tc_fence_after();
        const uint32_t acc = tmem_base + buf * kTileN;
        for (int k = 0; k < nk; ++k, ++it) {
          const int s = it % kPairStages;
          ok = mbar_wait(&full[s], (it / kPairStages) & 1, status, 313, cta_abort);
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = make_smem_desc(smem_u32(smem + s * kPairStageBytes), 16, 1024);
          const uint64_t bd = make_smem_desc(smem_u32(smem + s * kPairStageBytes + kABytes), kBoxBytes, 1024);
#pragma unroll
          for (int kk = 0; kk < kChunkK / 16; ++kk)
            mma_f16_ss_pair(acc, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 128), idesc, (k | kk) != 0);
          mma_commit_pair(&empty[s]);
        }
        if (!ok) end->give_up();                          // before both epilogues wake
        mma_commit_pair(&acc_full[buf]);
      }
      if (!ok) end->give_up();
    }
  } else {
    const bool ok = epilogue<D>(a, OutMaps{{&tmap_oq, &tmap_ok, &tmap_ov}}, tmem_base, o_buf, warp & 3, lane, first, step, (int)rank, acc_full, status, cta_abort,
                                [&](uint32_t buf) {
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_smem_u32(&acc_empty[buf], 0));
    });
    if (!ok && lane == 0) end->give_up();
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && rank == 0 && *(volatile int*)cta_abort != 0)
    end->drain(full, kPairStages, [&](int i) { return kABytes + Unit(a, first + i / nk * step).boxes / 2 * kBoxBytes; });
  __syncwarp();
  cluster_sync();                                         // the peer's shared memory is read, and its barriers arrived at, until here
  if (warp == 1) tmem_dealloc_pair(tmem_base, 2 * kTileN);
}

// plain FFMA version (float32 storage, or shapes the tensor-core kernel does not take): one thread per output
template <typename T>
__global__ void project_simt_kernel(const T* __restrict__ X, const T* __restrict__ W, T* __restrict__ Qo,
                                    T* __restrict__ Ko, T* __restrict__ Vo, int64_t rows_q, int64_t rows_kv, int n_tok,
                                    int B, int H, int d, int dm, int col0, int ncols, int ldw) {
  const int64_t total = (int64_t)B * n_tok * ncols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int rel = (int)(i % ncols);
    const int64_t bt = i / ncols;
    const int tok = (int)(bt % n_tok), b = (int)(bt / n_tok);
    const int col = col0 + rel, which = col / (H * d), hh = (col % (H * d)) / d, c = col % d;
    const T* x = X + ((int64_t)b * n_tok + tok) * dm;
    float acc = 0.f;
    for (int k = 0; k < dm; ++k) acc = fmaf(to_float(x[k]), to_float(W[(int64_t)k * ldw + col]), acc);
    T* dst = which == 0 ? Qo : (which == 1 ? Ko : Vo);
    const int64_t rows = which == 0 ? rows_q : rows_kv;
    dst[(((int64_t)b * H + hh) * rows + tok) * d + c] = from_float<T>(acc);
  }
}

}  // namespace

// One launch: columns [col0, col0 + ncols) of W applied to X [B, n_tok, dm]; the destinations those columns map to
// must be non-null.  W is [dm, 3 H d] row-major.
cudaError_t launch_project(csat_ctx* c, const void* X, const void* W, int64_t n_tok, int64_t dm, int col0, int ncols,
                           void* Q, void* K, void* V, cudaStream_t s, int* launches) {
  const Params& p = c->p;
  const int ldw = (int)(3 * p.H * p.d);
  *launches += 1;
  const bool tensor_core = p.dtype == CSAT_DTYPE_BF16 && (p.d == 64 || p.d == 128) && dm % 8 == 0 && c->force_simt == 0;
  if (!tensor_core) {
    const int64_t total = p.B * n_tok * ncols;
    int64_t g = (total + 255) / 256;
    if (g > 148 * 32) g = 148 * 32;
    if (p.dtype == CSAT_DTYPE_FP32)
      project_simt_kernel<float><<<(unsigned)g, 256, 0, s>>>((const float*)X, (const float*)W, (float*)Q, (float*)K,
                                                            (float*)V, p.nq, p.n, (int)n_tok, (int)p.B, (int)p.H,
                                                            (int)p.d, (int)dm, col0, ncols, ldw);
    else
      project_simt_kernel<__nv_bfloat16><<<(unsigned)g, 256, 0, s>>>(
          (const __nv_bfloat16*)X, (const __nv_bfloat16*)W, (__nv_bfloat16*)Q, (__nv_bfloat16*)K, (__nv_bfloat16*)V, p.nq,
          p.n, (int)n_tok, (int)p.B, (int)p.H, (int)p.d, (int)dm, col0, ncols, ldw);
    return cudaGetLastError();
  }
  CUtensorMap tx, tw;
  const uint64_t xd[3] = {(uint64_t)dm, (uint64_t)(n_tok * p.B), 1};            // [B, n_tok] is one sequence of rows
  const uint64_t xs[2] = {(uint64_t)dm * 2, (uint64_t)(n_tok * p.B) * dm * 2};
  const uint32_t xb[3] = {(uint32_t)kChunkK, (uint32_t)kTileM, 1};
  const uint64_t wd[3] = {(uint64_t)ldw, (uint64_t)dm, 1};
  const uint64_t ws[2] = {(uint64_t)ldw * 2, (uint64_t)dm * ldw * 2};
  const uint32_t wb[3] = {64, (uint32_t)kChunkK, 1};
  cudaError_t e;
  if ((e = make_tmap_bf16_3d(&tx, X, xd, xs, xb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tw, W, wd, ws, wb)) != cudaSuccess) return e;
  CUtensorMap to[3];
  const int64_t out_rows[3] = {p.nq, p.n, p.n};
  void* const dsts[3] = {Q, K, V};
  for (int i = 0; i < 3; ++i) {
    to[i] = tx;                                          // a matrix that this launch does not write
    const uint64_t od[3] = {(uint64_t)p.d, (uint64_t)out_rows[i], (uint64_t)(p.B * p.H)};
    const uint64_t os[2] = {(uint64_t)p.d * 2, (uint64_t)out_rows[i] * p.d * 2};
    const uint32_t ob[3] = {64, 32, 1};
    if (dsts[i] != nullptr && (e = make_tmap_bf16_3d(&to[i], dsts[i], od, os, ob)) != cudaSuccess) return e;
  }
  ProjArgs a;
  a.dst[0] = (__nv_bfloat16*)Q; a.dst[1] = (__nv_bfloat16*)K; a.dst[2] = (__nv_bfloat16*)V;
  a.rows[0] = p.nq; a.rows[1] = p.n; a.rows[2] = p.n;
  a.n_tok = (int)n_tok; a.B = (int)p.B; a.H = (int)p.H; a.dm = (int)dm;
  a.col0 = col0; a.ncols = ncols;
  a.ntiles = (ncols + kTileN - 1) / kTileN;
  const int64_t rows = n_tok * p.B, n_tiles = (rows + kTileM - 1) / kTileM * a.ntiles;
  if (n_tiles > (int64_t)1 << 28 || rows > (int64_t)1 << 30) return cudaErrorInvalidValue;
  const int sms = c->sms;
  // The tiles of a last, partial wave: in quarters if there are SMs for all of them at once, else in halves, else whole (a
  // narrower piece loads the same 128 rows of X for fewer columns: two rounds of quarters are no faster than a tile)
  const int pairs = sms / 2;
  const int64_t p_tiles = (rows + 2 * kTileM - 1) / (2 * kTileM) * a.ntiles, p_rest = p_tiles % pairs;
  // Pairs pay for their start and end (2.5 us more) with ~0.05 us per chunk of k and wave of tiles.  us, single / pairs: 4096 tokens x 6144, d_model =
  // 2048 (166 chunks) 72.0 / 66.9; 2000 tokens (83) 41.8 / 39.6; 6304 x 2304, 768 (36) 22.8 / 24.0; 12000 x 1152, 384 (17) 16.1 / 19.2
  const int64_t nk = (dm + kChunkK - 1) / kChunkK;
  const bool pair = p_tiles >= pairs && p_tiles * nk >= 64 * (int64_t)pairs;
  if (pair) {
    a.pieces = 2 * p_rest <= pairs ? 2 : 1;
    a.whole = (int)(p_tiles - p_rest);
    a.units = (int)(a.whole + p_rest * a.pieces);
    auto run = [&](auto kernel, DeviceFlags& opt_in) {
      cudaError_t err = ensure_dynamic_smem(kernel, (int)kPairSmemBytes, c->device, opt_in);
      if (err != cudaSuccess) return err;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(2 * (a.units < pairs ? a.units : pairs)));
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = kPairSmemBytes;
      cfg.stream = s;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2;
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      return cudaLaunchKernelEx(&cfg, kernel, tx, tw, to[0], to[1], to[2], a, c->status);
    };
    static DeviceFlags pair64, pair128;
    return p.d == 64 ? run(project_pair_kernel<64>, pair64) : run(project_pair_kernel<128>, pair128);
  }
  const int64_t rest = n_tiles % sms;
  a.pieces = 4 * rest <= sms ? 4 : 2 * rest <= sms ? 2 : 1;
  a.whole = (int)(n_tiles - rest);
  a.units = (int)(a.whole + rest * a.pieces);
  const unsigned grid = (unsigned)(a.units < sms ? a.units : sms);
  if (p.d == 64) {
    static DeviceFlags opt_in64;
    if ((e = ensure_dynamic_smem(project_sm100_kernel<64>, (int)kSmemBytes, c->device, opt_in64)) != cudaSuccess) return e;
    return launch_pdl(project_sm100_kernel<64>, dim3(grid), kThreads, kSmemBytes, s, tx, tw, to[0], to[1], to[2], a, c->status);
  } else {
    static DeviceFlags opt_in128;
    if ((e = ensure_dynamic_smem(project_sm100_kernel<128>, (int)kSmemBytes, c->device, opt_in128)) != cudaSuccess) return e;
    return launch_pdl(project_sm100_kernel<128>, dim3(grid), kThreads, kSmemBytes, s, tx, tw, to[0], to[1], to[2], a, c->status);
  }
}

}  // namespace csat

// K~|V~ = Phi_h [K|V]  (paper: compression equation) with the features in M: pairs of CTAs on tcgen05 MMAs of M = 256.
//
// What bounds both kernels on long token axes is the tensor pipe, and compress_sm100.cu's measurements come in tiles of 128, so that m =
// 392 pays for 512 rows and 264 for 384.  Here a CTA holds 128 features (K | V of one batch element at d = 64, K or V at d = 128)
// as the A operand and the pair shares the rows of Phi as the B operand, half of them in each CTA's shared memory: N is the measurements
// rounded up to 16 per part of at most 256.  Single CTAs with the features in M would load all rows of Phi each (65 KB per 64 tokens at
// m = 392, 42 KB here), and were no faster than tiles of 128.  us, tiles / pairs: 128 heads of 3136 x 64, m = 392 41.6 / 35.2 (tensor
// pipe 74 % of the active cycles; the rest is the ring's start and the epilogue); 64 of 4096 x 128, m = 400 55.5 / 43.3-46; 64 of 5000 x 64,
// m = 600 68.8 / 41.5; 32 of 4000 x 128, m = 300 31.0 / 26.5; 4 of 16384 x 128, m = 3000 102 / 87.  The start of a cluster, the allocation by
// both CTAs and their barrier at the end cost 1 to 2 us more than a single CTA: short token axes, multiples of 128 and grids of few CTAs stay
// there.
//
// The pair: d = 64 two batch elements of one head (an odd batch repeats the last one and does not store it), d = 128 the K and the V
// features of one (batch, head).  A CTA takes one or two parts of N measurements (accumulators side by side in tensor memory).
//   warp 0   : TMA producer of this CTA's half; all copies of a stage complete on rank 0's barrier.
//   warp 1   : allocates tensor memory; rank 0's elected thread issues the MMAs, their commits arrive in both CTAs.
//   warps 2-9: epilogue: lane = feature, columns = measurements, every other 32 for each half of the warps.  bf16 values go into boxes
//              of 32 measurements x 64 features in the ring's shared memory (a lane's values are one column of the box; lanes swap with
//              their neighbour, so that each writes two features of a row), two warps to a box, and leave by TMA stores.
// The same products in the same order as compress_sm100.cu: the same bits.
#include "csat_internal.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace csat {
namespace {

using namespace ptx;

constexpr int kChunk = 64;                               // tokens per stage
constexpr int kThreads = 320;
constexpr uint32_t kBoxBytes = 64 * kChunk * 2;          // 64 features x 64 tokens
constexpr uint32_t kABytes = 2 * kBoxBytes;
constexpr uint32_t kOutBytes = 32 * 128;                 // 32 measurements x 64 features
constexpr int kMaxStages = 8;
constexpr uint32_t kBarBytes = 256;

struct PairArgs {
  int m, n, H, B;
  int groups;                                            // of `parts` parts, over the measurements
  int parts, nhalf;                                      // parts per CTA; measurements per part and CTA (N = 2 nhalf)
  int stages, cols;                                      // ring; tensor-memory columns
  int* status;
};

__device__ __forceinline__ uint32_t stage_bytes(const PairArgs& a) { return kABytes + (uint32_t)(a.parts * a.nhalf) * 128; }

template <int D>
__global__ void __launch_bounds__(kThreads)
compress_pair_kernel(const __grid_constant__ CUtensorMap tmap_phi, const __grid_constant__ CUtensorMap tmap_k,
                     const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_out, const PairArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sb = stage_bytes(a);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + a.stages * sb);      // rank 0's count
  uint64_t* empty = full + kMaxStages;
  uint64_t* acc_done = empty + kMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_done + 1);
  PairEnd* end = reinterpret_cast<PairEnd*>(tmem_slot + 1);
  int* cta_abort = &end->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  // blockIdx.x walks the batch fastest (CTAs that stream the same rows of Phi run together), then come the measurement groups of a head
  const int h = blockIdx.y / a.groups, group = blockIdx.y % a.groups;
  const int e = D == 64 ? (int)blockIdx.x : (int)blockIdx.x / 2;           // batch element
  const bool store = e < a.B;
  const int bh = (store ? e : a.B - 1) * a.H + h;
  const int nchunks = (a.n + kChunk - 1) / kChunk;
  const int N = 2 * a.nhalf, r0 = group * a.parts * N;                     // first measurement

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_phi);
    prefetch_tmap(&tmap_k);
    prefetch_tmap(&tmap_v);
    prefetch_tmap(&tmap_out);
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_done, 1);
    end->init();
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, a.cols);
  tc_fence_before();
  __syncthreads();
  cluster_sync();                                        // both CTAs' barriers are set up
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();

  if (warp == 0) {
    if (elect_one()) {
      bool ok = true;
      int issued = 0;
      for (int i = 0; i < nchunks; ++i) {
        const int s = i % a.stages, use = i / a.stages;
        ok = mbar_wait(&empty[s], (use & 1) ^ 1, a.status, 151, cta_abort);
        if (!ok) break;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * sb);
        const uint32_t bar = cluster_smem_u32(&full[s], 0);
        uint8_t* st = smem + s * sb;
        if (D == 64) {
          tma_load_3d_pair(st, &tmap_k, bar, 0, i * kChunk, bh);
          tma_load_3d_pair(st + kBoxBytes, &tmap_v, bar, 0, i * kChunk, bh);
        } else {
          const CUtensorMap* src = rank == 0 ? &tmap_k : &tmap_v;
          tma_load_3d_pair(st, src, bar, 0, i * kChunk, bh);
          tma_load_3d_pair(st + kBoxBytes, src, bar, 64, i * kChunk, bh);
        }
        for (int p = 0; p < a.parts; ++p)                // rows beyond m are zero-filled
          tma_load_3d_pair(st + kABytes + p * a.nhalf * 128, &tmap_phi, bar, i * kChunk, r0 + p * N + (int)rank * a.nhalf, h);
        ++issued;
      }
      if (!ok) end->give_up();
      end->producer_done(rank, issued);
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = make_idesc_bf16(256, N, /*A MN-major*/ true, /*B MN-major*/ false);
      bool ok = true;
      for (int i = 0; i < nchunks; ++i) {
        const int s = i % a.stages;
        ok = mbar_wait(&full[s], (i / a.stages) & 1, a.status, 153, cta_abort);
        if (!ok) break;
        tc_fence_after();
        const uint64_t ad = make_smem_desc(smem_u32(smem + s * sb), kBoxBytes, 1024);
        for (int p = 0; p < a.parts; ++p) {
          const uint64_t bd = make_smem_desc(smem_u32(smem + s * sb + kABytes + p * a.nhalf * 128), 16, 1024);
#pragma unroll
          for (int k = 0; k < kChunk / 16; ++k)          // 16 token rows of A (2048 B), 32 B along a row of Phi
            mma_f16_ss_pair(tmem + p * N, ad + (uint64_t)(k * 128), bd + (uint64_t)(k * 2), idesc, (i | k) != 0);
        }
        mma_commit_pair(&empty[s]);
      }
      if (!ok) end->give_up();                           // before both epilogues wake
      mma_commit_pair(acc_done);
    }
  } else {
    const int q = warp & 3, half = (warp - 2) >> 2;      // lanes [32q, 32q+32) = features; which groups of 32 measurements
    const int box = q >> 1;                              // features [0, 64) or [64, 128) of the CTA's 128
    const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_done, 0, a.status, 154, cta_abort) && *(volatile int*)cta_abort == 0);
    if (!ok && lane == 0) end->give_up();
    if (ok) {
      tc_fence_after();
      const int f = (q & 1) * 32 + lane, odd = lane & 1; // feature within the box
      const int x = (D == 64 ? 0 : (int)rank * 128) + box * 64;
      const uint32_t src = tmem + ((uint32_t)(q * 32) << 16);
      const int per = (N + 31) / 32;                     // groups of 32 per part (N may end in the middle: what lies behind is not stored)
#pragma unroll 1
      for (int it = half; it < a.parts * per; it += 2) {
        const int p = it >= per ? 1 : 0, c0 = (it - p * per) * 32, row = r0 + p * N + c0;
        if (row >= a.m) break;
        uint32_t r[32];
        tmem_ld_32x32b_x32(src + p * N + c0, r);
        tmem_wait_ld();
        uint8_t* buf = smem + (uint32_t)(2 * it + box) * kOutBytes;
        // measurements j and j + 4 of two neighbouring features: the even lane keeps j, the odd one j + 4 (4 apart: other banks)
        uint8_t* out = buf + ((f & 6) << 1);
#pragma unroll
        for (int j8 = 0; j8 < 32; j8 += 8)
#pragma unroll
          for (int j = j8; j < j8 + 4; ++j) {
            const uint32_t mine = pack_bf16(__uint_as_float(r[j]), __uint_as_float(r[j + 4]));
            const uint32_t its = __shfl_xor_sync(0xffffffffu, mine, 1);
            const uint32_t w = odd ? __byte_perm(its, mine, 0x7632) : __byte_perm(mine, its, 0x5410);
            const int jr = j + 4 * odd;
            *reinterpret_cast<uint32_t*>(out + jr * 128 + (((f >> 3) ^ (jr & 7)) << 4)) = w;
          }
        fence_proxy_async();
        asm volatile("bar.sync %0, 64;" ::"r"(1 + 2 * half + box) : "memory");
        if ((q & 1) == 0 && lane == 0 && store) {        // in boxes of 16 rows (rows beyond m are clipped)
          tma_store_3d(&tmap_out, buf, x, row, bh);
          if (c0 + 16 < N && row + 16 < a.m) tma_store_3d(&tmap_out, buf + kOutBytes / 2, x, row + 16, bh);
          bulk_commit_group();
        }
      }
      if (lane == 0) bulk_wait_group0();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && rank == 0 && *(volatile int*)cta_abort != 0) end->drain(full, a.stages, [&](int) { return sb; });
  __syncwarp();
  cluster_sync();                                        // the peer's shared memory is read, and its barriers arrived at, until here
  if (warp == 1) tmem_dealloc_pair(tmem, a.cols);
}

// How the measurements of a (batch, head) are shared out: `groups` CTA pairs of `parts` parts of 2 nhalf; tensor-pipe cycles of an SM
struct Plan { int groups, parts, nhalf; double cycles; };

Plan plan(const csat_ctx* c) {
  const Params& p = c->p;
  const int64_t chunks = (p.n + kChunk - 1) / kChunk, units = p.d == 64 ? (p.B + 1) / 2 * p.H : p.B * p.H;
  Plan best{0, 0, 0, 0.0};
  for (int64_t g = (p.m + 511) / 512; g <= (p.m + 191) / 192 && g * p.H <= 65535; ++g) {
    const int64_t per = (p.m + g - 1) / g, parts = per > 256 ? 2 : 1, N = round_up((per + parts - 1) / parts, 16);
    if (parts * N * (g - 1) >= p.m) continue;              // the last group would be empty
    const double cycles = (double)((2 * units * g + c->sms - 1) / c->sms) * chunks * 2.0 * parts * N;
    if (best.groups == 0 || cycles < best.cycles) best = Plan{(int)g, (int)parts, (int)(N / 2), cycles};
  }
  return best;
}

template <int D>
cudaError_t launch(csat_ctx* c, const void* K, const void* V, cudaStream_t s, const Plan& pl) {
  const Params& p = c->p;
  CUtensorMap tphi, tk, tv, to;
  const uint64_t fd[3] = {(uint64_t)p.n_pad, (uint64_t)p.m, (uint64_t)p.H}, fs[2] = {(uint64_t)p.n_pad * 2, (uint64_t)p.m * p.n_pad * 2};
  const uint32_t fb[3] = {(uint32_t)kChunk, (uint32_t)pl.nhalf, 1};
  const uint64_t kd[3] = {(uint64_t)D, (uint64_t)p.n, (uint64_t)(p.B * p.H)}, ks[2] = {(uint64_t)D * 2, (uint64_t)p.n * D * 2};
  const uint32_t kb[3] = {64, (uint32_t)kChunk, 1}, ob[3] = {64, 16, 1};
  const uint64_t od[3] = {(uint64_t)(2 * D), (uint64_t)p.m, (uint64_t)(p.B * p.H)}, os[2] = {(uint64_t)D * 4, (uint64_t)p.m * D * 4};
  cudaError_t e;
  if ((e = make_tmap_bf16_3d(&tphi, c->phi, fd, fs, fb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tk, K, kd, ks, kb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tv, V, kd, ks, kb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&to, c->kv, od, os, ob)) != cudaSuccess) return e;
  const int64_t units = D == 64 ? (p.B + 1) / 2 : p.B, ctas = 2 * units * p.H * pl.groups;
  const int64_t chunks = (p.n + kChunk - 1) / kChunk;
  const int64_t sb = kABytes + (int64_t)pl.parts * pl.nhalf * 128, out = (int64_t)pl.parts * ((2 * pl.nhalf + 31) / 32) * 2 * kOutBytes;
  int cols = 32;
  while (cols < pl.parts * 2 * pl.nhalf) cols *= 2;
  // the ring: as deep as one CTA per SM allows, or two where there are CTAs for them
  const int64_t room = (ctas > c->sms && cols <= 256 ? 112 : 224) * 1024 - 1024 - kBarBytes;
  int64_t stages = room / sb;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages < 2) stages = 2;
  if (stages > chunks && chunks >= 2) stages = chunks;
  while (stages * sb < out) ++stages;
  int64_t bytes = stages * sb + 1024 + kBarBytes;
  // no more CTAs on an SM than tensor memory has columns for: two pairs must not wait for each other's halves
  const int64_t least = 228 * 1024 / (512 / cols + 1) - 1024 + 16;
  if (bytes < least) bytes = least;
  if (bytes > 227 * 1024 || stages > kMaxStages) return cudaErrorInvalidValue;
  static DeviceFlags opt_in;
  if ((e = ensure_dynamic_smem(compress_pair_kernel<D>, 227 * 1024, c->device, opt_in)) != cudaSuccess) return e;
  const PairArgs a{(int)p.m, (int)p.n, (int)p.H, (int)p.B, pl.groups, pl.parts, pl.nhalf, (int)stages, cols, c->status};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * units), (unsigned)(p.H * pl.groups));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, compress_pair_kernel<D>, tphi, tk, tv, to, a);
}

}  // namespace

// Cycles of an SM, on the scale of compress_sm100.cu's tensor-pipe cycles (1.4 to 1.5 clocks each, there and here).  A stage takes a pair no
// less than 480 of them where it has the SM to itself and 300 where two share one, however few its measurements: 590 to 630 clocks at N =
// 112 to 192 (8 heads of 11129 x 128, m = 210; of 11925, m = 1334), 1017 for two of N = 144 (48 of 9459, m = 423).
static double pair_time(const csat_ctx* c, const Plan& pl) {
  const Params& p = c->p;
  const int64_t units = p.d == 64 ? (p.B + 1) / 2 * p.H : p.B * p.H, ctas = 2 * units * pl.groups, sms = c->sms;
  const double chunks = (double)((p.n + kChunk - 1) / kChunk), tensor = 4.0 * pl.parts * pl.nhalf;
  const double alone = chunks * (tensor > 480.0 ? tensor : 480.0) + 9000.0, both = chunks * 2.0 * (tensor > 300.0 ? tensor : 300.0) + 10000.0;
  if (ctas <= sms || 2 * pl.parts * pl.nhalf > 256) return (double)((ctas + sms - 1) / sms) * alone;
  const int64_t rest = ctas % (2 * sms);
  return (double)(ctas / (2 * sms)) * both + (rest > sms ? both : rest > 0 ? alone : 0.0);
}

// tile_cycles: the tensor-pipe cycles of an SM in compress_sm100.cu; tile_rounds: of CTAs there, whose start and end take 6000 each; one_tile:
// no SM has more than one tile of 128 measurements.  Of 334 drawn shapes that the first conditions let through (1 to 32 batch elements, 1 to
// 16 heads, 600 to 16384 tokens, m = 192 to 2000) pairs are slower on 51, by up to 79 % (8 heads of 11129 x 128, m = 210 30 / 54 us); of those
// taken now 12 are slower, and 15 that would gain (13 of them less than 8 %) are not taken.
//   one_tile: pairs gain 8 to 20 % a stage whatever N and need some 60 stages for what they cost: 24 heads of 3200 x 64, m = 625 21.9 / 23.3, 42 of
//             5759, m = 512 39.1 / 32.2; the worst taken 19 of 5569 x 128, m = 635 37 / 48.
//   else    : by the times; the worst taken 24 heads of 2949 x 128, m = 1134 40 / 49 and 32 of 4747, m = 960 55 / 61.
// The first conditions: 11 x 16 heads of 5814 x 64, m = 1633 (0.894) 337 / 365, 12 x 16 of 6186, m = 1317 (0.875) 294 / 263; d = 128 in several
// rounds with m > 1000 is slower as often as not (7 x 8 of 6318, m = 1190 155 / 192, 15 x 4 of 6455, m = 1283 266 / 193).
bool compress_pair_better(const csat_ctx* c, double tile_cycles, double tile_rounds, bool one_tile) {
  const Params& p = c->p;
  if (p.separate_phi || p.m < 192 || (p.d == 64 ? p.B < 2 : p.d != 128) || p.H * ((p.m + 511) / 512) > 65535 || p.B > (1 << 29)) return false;
  const Plan pl = plan(c);
  if (pl.groups == 0) return false;
  if (p.d == 64 ? pl.cycles + 5200.0 >= tile_cycles || pl.cycles >= 0.88 * tile_cycles
                : pl.cycles + 4000.0 >= tile_cycles || (p.m > 1000 && 2 * p.B * p.H * pl.groups > c->sms))
    return false;
  if (one_tile) return p.n > 63 * kChunk;
  return pair_time(c, pl) < tile_cycles + 6000.0 * tile_rounds;
}

cudaError_t launch_compress_pair(csat_ctx* c, const void* K, const void* V, cudaStream_t s) {
  const Plan pl = plan(c);
  if (pl.groups == 0) return cudaErrorInvalidValue;
  return c->p.d == 64 ? launch<64>(c, K, V, s, pl) : launch<128>(c, K, V, s, pl);
}

}  // namespace csat

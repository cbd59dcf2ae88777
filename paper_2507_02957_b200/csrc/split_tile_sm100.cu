// Attention and recovery for bf16 contexts with head sizes that are no multiple of 64 (multiples of 8 up to 96, one S, B for all layers)
// on the sm_100a tensor cores: one tile of 128 queries per CTA.
//
// The precision is that of warp_split.cu: what the path holds in float32 enters a product as two bf16 parts, hi = bf16(x) and lo =
// bf16(x - hi): P V~ is two products, z B and the recurrence three (lo lo is left out), all sums float32; rows whose result is not finite
// are computed in float32 (plain_row).  The matrices' parts are laid out once by the decoder set-up.  The accumulator keeps c + sum of
// (alpha^{t+1} - alpha^t) (S - I) = z B + alpha (S - I): only the increment enters a layer's product, and x = alpha + accumulator.
//
// What bounds it: the chain thread -> MMA issuer -> tensor pipe -> thread of a layer, as in attend_tile_sm100.cu, with three times the
// products (d = 96: 18 MMAs of 48 cycles) and twice the operand.  Warp-level instructions have a quarter of the rate: a layer of 128 rows
// takes them 3500 cycles of an SM's matrix pipes at d = 96.  A lone tile's layer takes 2860 cycles there (pass over the row 1200, products
// 1000, hand-overs), two on an SM 2600 each.  With min and max in the shrinkage (half the FMA pipe's rate) the pass took 1620; products
// issued from loops that were not unrolled cost 100 cycles each.  32 heads of 1024 x 96, m = 128, T = 10: 75.2 -> 25.1 us, the call
// (with the compression on compress_sm100.cu, 18.8 -> 7.1) 97.6 -> 33.1; 12 heads of 700 x 80, T = 20 38.0 -> 31.2.  The error against 64 bits over
// sixteen shapes (d = 8 to 96, T = 5 to 20) is 0.99996 to 1.0004 times that of the warp kernel.
//
// CTA = 8 warps: 0-3 one thread per query row (TMEM lane = row, the whole iterate in registers); 4 issues the MMAs; 5 every TMA copy;
// 6, 7 complete the warpgroup.  Shared memory: Q | two stages K~ | V~; over them, once the attention phase has read them, the matrices
// B_hi | B_lo | S_hi | S_lo (then Psi in B's place), at the end the output.
#include "csat_internal.h"
#include "row_math.cuh"
#include "split_math.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace csat {
namespace {

using namespace ptx;
using namespace rowmath;
using namespace splitmath;

constexpr int kRows = 128, kMC = 64, kThreads = 256;
constexpr int kMmaWarp = 4, kTmaWarp = 5;

template <int DP> struct Cfg {
  static constexpr int kBoxes = (DP + 63) / 64;                     // 64-column boxes across the head dimension
  static constexpr int kCtas = DP > 64 ? 2 : 3;                     // per SM
  static constexpr int kRowRegs = kCtas == 2 ? 208 : 128, kControlRegs = kCtas == 2 ? 48 : 32;   // after setmaxnreg (checked on the host)
  static constexpr uint32_t kQBytes = kBoxes * kRows * 128, kSlotBytes = kBoxes * kMC * 128, kStageBytes = 2 * kSlotBytes;
  static constexpr uint32_t kMatBoxBytes = DP * 128, kMatBytes = kBoxes * kMatBoxBytes;
  static constexpr uint32_t kOffRing = kQBytes, kOffBar = kOffRing + 2 * kStageBytes, kSmemBytes = kOffBar + 256;
  static constexpr uint32_t kOutBytes = 32 * 128;                   // one warp's rows of one box
  // tensor memory: accumulator (z, then c + alpha (S - I)) | S (P hi | P lo over it), later the operand's parts
  static constexpr uint32_t kColAcc = 0, kColS = DP, kTmemCols = DP > 64 ? 256 : 128;
  static_assert(DP + (DP > kMC ? DP : kMC) <= (int)kTmemCols && kCtas * kTmemCols <= 512, "TMEM budget");
  static_assert(4 * kMatBytes <= kOffBar && kMatBytes <= kQBytes && 4 * kBoxes * kOutBytes <= kOffBar, "overlays");
  static_assert(kCtas * (kSmemBytes + 1024) <= 228 * 1024, "CTAs per SM");
};

struct Bars {
  uint64_t q_full, k_full[2], v_full[2], free[2], attended, mats_full[3], b_read, done;
  uint32_t tmem_slot;
  int abort;
};
static_assert(sizeof(Bars) <= 256, "barrier block");

template <int DP>
__global__ void __launch_bounds__(kThreads, Cfg<DP>::kCtas)
split_tile_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                  const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_mats,
                  const __grid_constant__ CUtensorMap tmap_out, const __grid_constant__ FfmaAttend p, __nv_bfloat16* __restrict__ out,
                  const __nv_bfloat16* __restrict__ Q, const __nv_bfloat16* __restrict__ kv, int tiles, int* status) {
  using C = Cfg<DP>;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {          // swizzled tiles need 1024-byte alignment; never seen to fail
    if (threadIdx.x == 0) atomicCAS(status, 0, 260);
    return;
  }
  uint8_t* ring = smem + C::kOffRing;
  Bars* bars = reinterpret_cast<Bars*>(smem + C::kOffBar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.x / tiles, row0 = (blockIdx.x % tiles) * kRows, h = bh % p.H;
  const int nq = (int)p.nq, m = (int)p.m, T = p.T, d = p.d;
  const int nchunks = (m + kMC - 1) / kMC, ksteps = (d + 15) / 16;      // K steps with columns below d
  const bool has_psi = p.psi != nullptr;
  Waiter w{status, &bars->abort};

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_k);
    prefetch_tmap(&tmap_v);
    prefetch_tmap(&tmap_mats);
    prefetch_tmap(&tmap_out);
    mbar_init(&bars->q_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->free[s], 1);
    }
    for (int s = 0; s < 3; ++s) mbar_init(&bars->mats_full[s], 1);
    mbar_init(&bars->attended, 1);
    mbar_init(&bars->b_read, 1);
    mbar_init(&bars->done, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&bars->tmem_slot, C::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_slot;
  if (p.wait_first) pdl_wait();
  const int n_mma = T > 0 ? T + (has_psi ? 1 : 0) : 0;               // products of the recovery

  if (warp >= kMmaWarp) {
    reg_dealloc<C::kControlRegs>();
    if (warp == kMmaWarp) {
      // ---------------------------------------------- MMA issuer ----------------------------------------------------
      constexpr uint32_t idesc_s = make_idesc_bf16(kRows, kMC, false, false);   // S  = Q  K~^T : both K-major
      constexpr uint32_t idesc_n = make_idesc_bf16(kRows, DP, false, true);     // P V~, z B, alpha (S - I): rows of B are K
      constexpr uint32_t idesc_k = make_idesc_bf16(kRows, DP, false, false);    // alpha Psi^T: Psi's rows are the columns of the result
      const uint32_t op = tmem + C::kColS, acc = tmem + C::kColAcc;
      const uint64_t qd = make_smem_desc(smem_u32(smem), 16, 1024);
      const uint64_t kd0 = make_smem_desc(smem_u32(ring), 16, 1024);
      const uint64_t vd0 = make_smem_desc(smem_u32(ring + C::kSlotBytes), kMC * 128, 1024);
      const uint64_t md_n = make_smem_desc(smem_u32(smem), C::kMatBoxBytes, 1024), md_k = make_smem_desc(smem_u32(smem), 16, 1024);
      Publications<1, kRows> rows;
      w.wait(&bars->q_full, 0, 262);
      for (int j = 0; j <= nchunks; ++j) {                    // P_{j-1} V~_{j-1}, then S_j in its place
        const int i = j - 1;
        if (j < nchunks) w.wait(&bars->k_full[j & 1], (j >> 1) & 1, 261);
        if (i >= 0) {
          w.wait(&bars->v_full[i & 1], (i >> 1) & 1, 263);
          rows.wait();
        }
        tc_fence_after();
        if (elect_one()) {
          if (i >= 0) {
            const uint64_t vd = vd0 + (uint64_t)((i & 1) * (C::kStageBytes >> 4));
#pragma unroll
            for (int part = 0; part < 2; ++part)              // hi, lo
#pragma unroll
              for (int k = 0; k < kMC / 16; ++k)
                mma_f16_ts(acc, op + part * (kMC / 2) + k * 8, vd + (uint64_t)(k * 128), idesc_n, (uint32_t)((i | part | k) != 0));
          }
          if (j < nchunks) {
            const uint64_t kd = kd0 + (uint64_t)((j & 1) * (C::kStageBytes >> 4));
#pragma unroll
            for (int k = 0; k < DP / 16; ++k)
              if (k < ksteps) mma_f16_ss(op, qd + (uint64_t)((k / 4) * (kRows * 128 >> 4) + (k % 4) * 2), kd + (uint64_t)((k / 4) * (kMC * 128 >> 4) + (k % 4) * 2),
                         idesc_s, k != 0);
          }
          mma_commit(&bars->done);
          if (i >= 0 && i + 2 < nchunks) mma_commit(&bars->free[i & 1]);
          if (j == nchunks) mma_commit(&bars->attended);      // Q, K~ and V~ have been read for the last time
        }
        __syncwarp();
      }
      for (int i = 0; i < n_mma; ++i) {                       // B, then S - I T - 1 times, then Psi
        const bool psi = has_psi && i == n_mma - 1;
        if (i <= 1 || psi) w.wait(&bars->mats_full[psi ? 2 : i], 0, 265);
        rows.wait();
        tc_fence_after();
        if (elect_one()) {
          // hi hi, lo hi, hi lo; K steps without columns below d are left out
          auto products = [&](uint64_t hi, uint32_t idesc, uint32_t keep, auto kstep) {
            const uint64_t lo = hi + (C::kMatBytes >> 4);
#pragma unroll
            for (int k = 0; k < DP / 16; ++k)
              if (k < ksteps) mma_f16_ts(acc, op + k * 8, hi + kstep(k), idesc, k == 0 ? keep : 1u);
#pragma unroll
            for (int k = 0; k < DP / 16; ++k)
              if (k < ksteps) mma_f16_ts(acc, op + DP / 2 + k * 8, hi + kstep(k), idesc, 1u);
#pragma unroll
            for (int k = 0; k < DP / 16; ++k)
              if (k < ksteps) mma_f16_ts(acc, op + k * 8, lo + kstep(k), idesc, 1u);
          };
          if (psi)
            products(md_k, idesc_k, 0u, [](int k) { return (uint64_t)((k / 4) * (C::kMatBoxBytes >> 4) + (k % 4) * 2); });
          else
            products(md_n + (i == 0 ? 0u : 2 * C::kMatBytes >> 4), idesc_n, i != 0, [](int k) { return (uint64_t)(k * 128); });
          mma_commit(&bars->done);
          if (i == 0) mma_commit(&bars->b_read);
        }
        __syncwarp();
      }
    } else if (warp == kTmaWarp) {
      // ---------------------------------------------- copies --------------------------------------------------------
      if (elect_one()) {
        int nc = 0, nm = 0;                       // chunks, and matrices (bit i: mats_full[i]), whose copies were issued
        auto load_pair = [&](uint32_t at, int i, int which) {       // both parts of S - I, B or Psi; columns and rows beyond d are zero
          nm |= 1 << i;
          mbar_arrive_expect_tx(&bars->mats_full[i], 2 * C::kMatBytes);
          for (int part = 0; part < 2; ++part)
            for (int gx = 0; gx < C::kBoxes; ++gx)
              tma_load_3d(smem + at + part * C::kMatBytes + gx * C::kMatBoxBytes, &tmap_mats, &bars->mats_full[i], gx * 64, 0, h * 6 + 2 * which + part);
        };
        mbar_arrive_expect_tx(&bars->q_full, C::kQBytes);
        for (int gx = 0; gx < C::kBoxes; ++gx) tma_load_3d(smem + gx * kRows * 128, &tmap_q, &bars->q_full, gx * 64, row0, bh);
        pdl_wait();                               // K~|V~ come from the kernel before this one
        pdl_launch_dependents();
        for (int j = 0; j < nchunks; ++j) {
          if (j >= 2) w.wait(&bars->free[j & 1], ((j >> 1) - 1) & 1, 267);
          if (w.dead) break;
          uint8_t* st = ring + (j & 1) * C::kStageBytes;
          mbar_arrive_expect_tx(&bars->k_full[j & 1], C::kSlotBytes);
          mbar_arrive_expect_tx(&bars->v_full[j & 1], C::kSlotBytes);
          for (int gx = 0; gx < C::kBoxes; ++gx) tma_load_3d(st + gx * kMC * 128, &tmap_k, &bars->k_full[j & 1], gx * 64, j * kMC, bh);
          for (int gx = 0; gx < C::kBoxes; ++gx)
            tma_load_3d(st + C::kSlotBytes + gx * kMC * 128, &tmap_v, &bars->v_full[j & 1], gx * 64, j * kMC, bh);
          ++nc;
        }
        if (T > 0 && !w.dead) {
          w.wait(&bars->attended, 0, 268);
          if (!w.dead) load_pair(0, 0, 1);
          if (!w.dead && T > 1) load_pair(2 * C::kMatBytes, 1, 0);
          if (has_psi) {
            w.wait(&bars->b_read, 0, 269);
            if (!w.dead) load_pair(0, 2, 2);
          }
        }
        if (w.dead) {
          // gave up: let the copies that are still in flight land before the CTA's shared memory goes away
          mbar_wait_drain(&bars->q_full, 0);
          for (int i = 0; i < 3; ++i)
            if ((nm >> i) & 1) mbar_wait_drain(&bars->mats_full[i], 0);
          for (int j = nc > 2 ? nc - 2 : 0; j < nc; ++j) {
            mbar_wait_drain(&bars->k_full[j & 1], (j >> 1) & 1);
            mbar_wait_drain(&bars->v_full[j & 1], (j >> 1) & 1);
          }
        }
      }
    }
  } else {
    reg_alloc<C::kRowRegs>();
    const int grow = row0 + warp * 32 + lane;
    const bool live = row0 + warp * 32 < nq;                  // the warp has rows
    const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
    const uint32_t acc_addr = tbase + C::kColAcc, op_addr = tbase + C::kColS;
    const float scale_log2 = p.scale * 1.4426950408889634f;
    const F2 sc2 = pack2(scale_log2, scale_log2);
    Publications<1, kRows> rows;
    int phase = 0;
    auto wait_done = [&](int code) {
      w.wait(&bars->done, phase & 1, code);
      ++phase;
      tc_fence_after();
    };
    auto hand_over = [&]() {
      tmem_wait_st();
      tc_fence_before();
      rows.publish(w.dead);
    };
    float ref = -INFINITY;
    F2 sum2 = pack2(0.f, 0.f);
    for (int j = 0; j < nchunks; ++j) {
      wait_done(270);                                         // S_j, and P_{j-1} V~_{j-1}
      if (live) {
        uint32_t ra[32], rb[32];
        tmem_ld_32x32b_x32(op_addr, ra);
        tmem_ld_32x32b_x32(op_addr + 32, rb);
        tmem_wait_ld();
        if ((j + 1) * kMC > m)
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            if (j * kMC + e >= m) ra[e] = 0xff800000u;        // -inf
            if (j * kMC + 32 + e >= m) rb[e] = 0xff800000u;
          }
        float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          m0 = max3(m0, __uint_as_float(ra[e]), __uint_as_float(ra[e + 1]));
          m1 = max3(m1, __uint_as_float(rb[e]), __uint_as_float(rb[e + 1]));
        }
        const float mx = fmaxf(m0, m1) * scale_log2;
        if (j == 0) {
          ref = mx;
        } else {
          const bool raise = mx > ref + 8.f;
          if (__any_sync(0xffffffffu, raise)) {               // rare: rescale this warp's rows of the accumulator
            const float f = raise ? ex2(ref - mx) : 1.f;
            if (raise) ref = mx;
            sum2 = mul2(sum2, pack2(f, f));
#pragma unroll
            for (int c0 = 0; c0 < DP; c0 += 16) {
              uint32_t a[16];
              tmem_ld_32x32b_x16(acc_addr + c0, a);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 16; ++e) a[e] = __float_as_uint(__uint_as_float(a[e]) * f);
              tmem_st_32x32b_x16(acc_addr + c0, a);
            }
          }
        }
        const F2 nref2 = pack2(-ref, -ref);
        auto exp_half = [&](const uint32_t (&r)[32], uint32_t col) {
          uint32_t hi[16], lo[16];
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            float t0, t1;
            unpack2(fma2(pack2u(r[e], r[e + 1]), sc2, nref2), t0, t1);
            const F2 pr = pack2(ex2(t0), ex2(t1));
            sum2 = add2(sum2, pr);
            hi[e >> 1] = pack_bf16(pr.x, pr.y);
            const F2 l2 = sub2(pr, pack2(bf16_lo(hi[e >> 1]), bf16_hi(hi[e >> 1])));
            lo[e >> 1] = pack_bf16(l2.x, l2.y);
          }
          tmem_st_32x32b_x16(op_addr + col, hi);
          tmem_st_32x32b_x16(op_addr + kMC / 2 + col, lo);
        };
        exp_half(ra, 0);
        exp_half(rb, 16);
      }
      hand_over();
    }
    const float inv = 1.f / (sum2.x + sum2.y);
    wait_done(271);                                           // every P V~ product has been added
    float a[DP];                                              // in turn: z, the iterate, Psi alpha
    // an accumulator row, 16 columns at a time, the next piece's load in flight under this one's arithmetic
    auto pieces = [&](auto f) {
      uint32_t r0[16], r1[16];
      tmem_ld_32x32b_x16(acc_addr, r0);
#pragma unroll
      for (int c0 = 0; c0 < DP; c0 += 32) {
        tmem_wait_ld();
        tmem_ld_32x32b_x16(acc_addr + c0 + 16, r1);
        f(r0, c0);
        tmem_wait_ld();
        if (c0 + 32 < DP) tmem_ld_32x32b_x16(acc_addr + c0 + 32, r0);
        f(r1, c0 + 16);
      }
    };
    auto put16 = [&](const float (&x)[16], int c0) {          // as the operand's parts
      uint32_t hi[8], lo[8];
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        hi[e >> 1] = pack_bf16(x[e], x[e + 1]);
        const F2 l2 = sub2(pack2(x[e], x[e + 1]), pack2(bf16_lo(hi[e >> 1]), bf16_hi(hi[e >> 1])));
        lo[e >> 1] = pack_bf16(l2.x, l2.y);
      }
      tmem_st_32x32b_x8(op_addr + c0 / 2, hi);
      tmem_st_32x32b_x8(op_addr + DP / 2 + c0 / 2, lo);
    };
    pieces([&](const uint32_t (&r)[16], int c0) {
      float x[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) a[c0 + e] = x[e] = __uint_as_float(r[e]) * inv;
      if (T > 0) put16(x, c0);
    });
    if (T > 0) {
      hand_over();
#pragma unroll
      for (int c = 0; c < DP; ++c) a[c] = 0.f;                // alpha^0
      for (int it = 0; it < T; ++it) {
        const float th = p.theta[(int64_t)it * p.theta_stride + h];
        wait_done(272);
        if (live && th > 0.f && it + 1 < T) {
          // on the FMA pipe, which min and max are not: y = x + theta, t = sat(y / (2 theta)), eta_theta(x) = y - 2 theta t (1e-7 theta
          // in the place of exact zeros, so the last layer is shrunk below)
          const float i2th = 0.5f / th;
          const F2 th2 = pack2(th, th), m2th2 = pack2(-2.f * th, -2.f * th);
          pieces([&](const uint32_t (&r)[16], int c0) {
            float dx[16];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const F2 rt = add2(pack2u(r[e], r[e + 1]), th2), al = pack2(a[c0 + e], a[c0 + e + 1]), y = add2(al, rt);
              const F2 dn = fma2(pack2(fma_sat(y.x, i2th, 0.f), fma_sat(y.y, i2th, 0.f)), m2th2, rt), an = add2(al, dn);
              a[c0 + e] = an.x;
              a[c0 + e + 1] = an.y;
              dx[e] = dn.x;
              dx[e + 1] = dn.y;
            }
            put16(dx, c0);
          });
        } else if (live) {
          pieces([&](const uint32_t (&r)[16], int c0) {
            float dx[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float x = a[c0 + e] + __uint_as_float(r[e]);          // alpha S + z B
              const float an = x - fminf(fmaxf(x, -th), th);
              dx[e] = an - a[c0 + e];
              a[c0 + e] = an;
            }
            if (it + 1 < T) put16(dx, c0);
          });
        }
        if (it + 1 < T) hand_over();
      }
      if (has_psi) {
        if (live)
#pragma unroll
          for (int c0 = 0; c0 < DP; c0 += 16) {
            float x[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = a[c0 + e];
            put16(x, c0);
          }
        hand_over();
        wait_done(273);
        pieces([&](const uint32_t (&r)[16], int c0) {
#pragma unroll
          for (int e = 0; e < 16; ++e) a[c0 + e] = __uint_as_float(r[e]);
        });
      }
    }
    // every MMA of the tile is done, and so are the copies they waited for: the output leaves from where Q was, a warp's rows per box
    if (live) {
      bool finite = true;
      uint8_t* box = smem + warp * C::kBoxes * C::kOutBytes;
#pragma unroll
      for (int c = 0; c < DP / 8; ++c) {
#pragma unroll
        for (int e = 0; e < 8; ++e) finite = finite && (8 * c >= d || fabsf(a[8 * c + e]) < INFINITY);
        *reinterpret_cast<uint4*>(box + (c / 8) * C::kOutBytes + lane * 128 + (((c % 8) ^ (lane & 7)) << 4)) =
            make_uint4(pack_bf16(a[8 * c], a[8 * c + 1]), pack_bf16(a[8 * c + 2], a[8 * c + 3]), pack_bf16(a[8 * c + 4], a[8 * c + 5]),
                       pack_bf16(a[8 * c + 6], a[8 * c + 7]));
      }
      fence_proxy_async();
      const bool dead = __any_sync(0xffffffffu, w.dead) || *(volatile int*)&bars->abort != 0;
      if (lane == 0 && !dead) {
        for (int gx = 0; gx < C::kBoxes; ++gx) tma_store_3d(&tmap_out, box + gx * C::kOutBytes, gx * 64, grow, bh);
        bulk_commit_group();
        bulk_wait_group0();                                   // the stores are done before the kernel ends (and before the rows below)
      }
      uint32_t odd = __ballot_sync(0xffffffffu, !finite && grow < nq && !dead);
      for (; odd != 0; odd &= odd - 1) {
        const int64_t at = ((int64_t)bh * nq + row0 + warp * 32 + __ffs(odd) - 1) * d;
        __syncwarp();
        plain_row(out + at, Q + at, kv + (int64_t)bh * m * 2 * d, p, (int64_t)h * d * d);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, C::kTmemCols);
}

template <int DP>
cudaError_t launch(csat_ctx* c, const FfmaAttend& a, const void* Q, void* out, cudaStream_t s) {
  using C = Cfg<DP>;
  const Params& p = c->p;
  const uint64_t d = (uint64_t)p.d, BH = (uint64_t)(p.B * p.H);
  const uint64_t qd[3] = {d, (uint64_t)p.nq, BH}, qs[2] = {d * 2, (uint64_t)p.nq * d * 2};
  const uint64_t kd[3] = {d, (uint64_t)p.m, BH}, ks[2] = {d * 4, (uint64_t)p.m * d * 4};
  const uint64_t md[3] = {d, d, (uint64_t)(p.H * 6)}, ms[2] = {d * 2, d * d * 2};
  const uint32_t qb[3] = {64, kRows, 1}, kb[3] = {64, kMC, 1}, mb[3] = {64, DP, 1}, ob[3] = {64, 32, 1};
  CUtensorMap tq, tk, tv, tm, to;
  cudaError_t e;
  if ((e = make_tmap_bf16_3d(&tq, Q, qd, qs, qb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tk, c->kv, kd, ks, kb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tv, (const __nv_bfloat16*)c->kv + p.d, kd, ks, kb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tm, c->mats_split, md, ms, mb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&to, out, qd, qs, ob)) != cudaSuccess) return e;
  static DeviceFlags opt_in;
  if (!opt_in.test(c->device)) {
    // setmaxnreg moves registers inside the pool the CTA is launched with; a request it cannot satisfy waits forever
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, split_tile_kernel<DP>)) != cudaSuccess) return e;
    if (fa.numRegs * kThreads < kRows * C::kRowRegs + (kThreads - kRows) * C::kControlRegs) return cudaErrorLaunchOutOfResources;
  }
  if ((e = ensure_dynamic_smem(split_tile_kernel<DP>, 120 * 1024, c->device, opt_in)) != cudaSuccess) return e;
  const int64_t tiles = (p.nq + kRows - 1) / kRows, n = tiles * p.B * p.H;
  if (n > (int64_t)1 << 30) return cudaErrorInvalidValue;
  // up to one or two tiles per SM no more share one: started early, they would pile up on the SMs the kernel before leaves free
  const uint32_t smem = n <= c->sms ? 120 * 1024 : n <= 2 * (int64_t)c->sms && C::kSmemBytes < 100 * 1024 ? 100 * 1024 : C::kSmemBytes;
  return launch_pdl(split_tile_kernel<DP>, dim3((unsigned)n), kThreads, smem, s, tq, tk, tv, tm, to, a, (__nv_bfloat16*)out,
                    (const __nv_bfloat16*)Q, (const __nv_bfloat16*)c->kv, (int)tiles, c->status);
}

}  // namespace

// Against warp_split.cu, us, warps / tiles of 128 queries: d > 64 from 27.4 / 21.5 (4 heads of 128 x 96, T = 10) to 75 / 25 (32 of 1024 x 96): always
// (behind, by 1.3 us of 12.7, in whole forwards of up to 12 tiles with T = 1 alone).  d = 48, T = 10: 8 heads of 256 12.9 / 14.9, 72 of 300 22.4 /
// 18.4: from a tile for every other SM on.  d <= 32, where a warp's layer is short and a tile's chain is not: up to a tile per SM 7.5 / 10.5 to
// 9.2 / 9.4; beyond, the attention phase is faster (96 heads of 500, m = 100, T = 10 22.6 / 16.9; 128 of 1000, m = 64, T = 5 30.1 / 22.9), the layers
// are not (128 of 400, m = 64, T = 20 35.1 / 37.9; 12 of 2139 x 24, m = 92, T = 20 20.7 / 23.4): up to ten layers per chunk of measurements,
// six up to two tiles per SM, and less by 0.6 and by the rows that a tile lacks for d <= 16, whose products take a warp half the steps (10 of
// 2113 x 8, m = 16, T = 5 8.5 / 11.4; 32 of 593 x 8, m = 159, T = 20 14.8 / 21.4; 556 tiles of 70 x 16, m = 69, T = 10 22.4 / 25.8).  Of 129 drawn jobs
// with d <= 32 three are slower by more than 4 % (at most 11), with ten layers alone 13 were (up to 35).  By the context's whole job.
bool split_tile_better(const csat_ctx* c) {
  const Params& p = c->p;
  if (c->mats_split == nullptr || !split_tile_head(p) || (c->w_S && c->w_untied && p.T > 0)) return false;
  const int64_t tiles = (p.nq + kRows - 1) / kRows * p.B * p.H;
  if (p.d > 64) return true;
  if (p.d > 32) return 2 * tiles > c->sms;
  double layers = 10.0 * (double)((p.m + kMC - 1) / kMC);
  if (tiles <= 2 * (int64_t)c->sms) layers *= 0.6;
  if (p.d <= 16) layers *= 0.6 * (double)(p.B * p.H * p.nq) / (double)(tiles * kRows);
  return tiles > c->sms && p.T <= layers;
}

cudaError_t launch_split_tile(csat_ctx* c, const FfmaAttend& a, const void* Q, void* out, cudaStream_t s) {
  if (c->p.d <= 32) return launch<32>(c, a, Q, out, s);
  if (c->p.d <= 64) return launch<64>(c, a, Q, out, s);
  return launch<96>(c, a, Q, out, s);
}

}  // namespace csat

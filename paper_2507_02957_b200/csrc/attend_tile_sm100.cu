// Compressed attention and sparse recovery for d = 64 on the sm_100a tensor cores: one tile of 128 queries per CTA, three CTAs per SM.
//
// Paper, in order: A~ = softmax(Q K~^T / sqrt(d_k)) over the m measurements; Z = A~ V~;
// alpha^{t+1} = eta_theta(S alpha^t + B Z_i) (LISTA recurrence with S = I - mu G, B = mu M); C^_i = Psi alpha^_i.
// Arithmetic, operands and their order are those of attend_recover_sm100.cu (see there for the recurrence's forms): S_j = Q K~_j^T,
// P_j over S_j in tensor memory, Z += P_j V~_j; then r += bf16(increment) (-mu G) with r in tensor memory and alpha in registers.
//
// What bounds it: a layer is a chain thread -> MMA issuer -> tensor pipe -> thread of ~1200 cycles with three tiles in flight (pass over
// the row 600, hand-over to the issuer 70, four MMAs 80, their end, commit and the rows' wait 250 and more), of which the tensor
// pipe needs 128 and a sub-core's issue slots ~250.  Only tiles in flight shorten it: two per SM (one CTA with both, 1 KB of registers a
// row) took 750 cycles per tile and layer, three take 450.  A tile needs 128 columns of tensor memory, so four would fit; in the 104
// registers per thread that leaves them they took 86 us for 96 heads of 1568 queries, T = 20, m = 256, where three took 79 and the two
// took 95 (whole forward, B not folded; as dispatched now, folded, 82).  The same tiles without warps of their own for MMAs and copies (128 threads) took 89: the issuing warp's own
// pass then starts ~300 cycles late, and a divided `elect` (chosen once, used later) costs 100 instead of 45 cycles per MMA.
//
// The rows hand over through named barriers (Publications): the issuer woke 240 cycles after the last of 128 arrivals at an mbarrier.  96
// heads of 1568 queries, folded: 66.2 -> 63.6 us (attention and recovery alone), recording 92.7 -> 90.0.  (The same in bwd_cols, whose passes
// are longer and whose 256 threads arrive: 42.5 -> 44.4; in the recurrence of two tiles at d = 128: 155 -> 156.)
//
// CTA = 8 warps: 0-3 one thread per query row (TMEM lane = row); 4 allocates tensor memory, one elected lane issues the MMAs; 5 every TMA
// copy; 6, 7 complete the warpgroup, which gives its registers to the rows (setmaxnreg).
#include "csat_internal.h"
#include "row_math.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.h"

#include <type_traits>

namespace csat {
namespace {

using namespace ptx;
using namespace rowmath;

constexpr int kD = 64;
constexpr int kRows = 128;             // queries per CTA: one thread per query, TMEM lane = query
constexpr int kMC = 64;                // measurements per chunk
constexpr int kRowWarps = 4, kMmaWarp = 4, kTmaWarp = 5;
constexpr int kThreads = 256;          // the rows' warps, then one warpgroup of control
constexpr int kCtas = 3;               // per SM
constexpr int kControlRegs = 32;                                  // after setmaxnreg (checked on the host)
template <int kBufs> constexpr int kRowRegs = kBufs == 1 ? 128 : 208;
constexpr uint32_t kQBytes = kRows * 128;                         // Q; later Psi; at the end the output
constexpr uint32_t kSlotBytes = kMC * 128;                        // K~ chunk (= V~ chunk)
constexpr uint32_t kStageBytes = 2 * kSlotBytes;
constexpr uint32_t kMatBytes = kD * 128;                          // a d x d bf16 matrix
constexpr uint32_t kOffRing = kQBytes, kBarBytes = 256;
// Shared memory: Q | ring | -mu G | B | barriers.  K~|V~ chunks in flight: two where three CTAs share an SM; four with two score buffers
// (kBufs), where few CTAs wait for their own copies: 76 heads of 77 queries, m = 392 23.6 -> 21.0 us, 96 of 112, m = 512, T = 5 18.1 ->
// 15.8, one chunk 10.1 either way.
template <int kBufs> struct Layout {
  static constexpr int kStages = 2 * kBufs;
  static constexpr uint32_t kOffG = kOffRing + kStages * kStageBytes, kOffB = kOffG + kMatBytes, kOffBar = kOffB + kMatBytes;
  static constexpr uint32_t kSmemBytes = kOffBar + kBarBytes;
  static constexpr uint32_t kSmemTwo = (kBufs == 1 ? 80 : 100) * 1024;  // no more than two CTAs per SM; the rest is L1, for the iterates' stores
  static_assert(kSmemBytes <= kSmemTwo && 2 * (kSmemTwo + 1024) <= 228 * 1024 && 3 * kSmemTwo > 228 * 1024, "two CTAs per SM");
};
constexpr uint32_t kSmemOne = 120 * 1024;                         // no more than one CTA per SM
constexpr uint32_t kOutBytes = 32 * 128;                          // one warp's rows of the output
// TMEM columns: accumulator (Zacc, then r_t) | S (P_j overlays its first half; later the recovery operand)
constexpr uint32_t kColAcc = 0, kColS = kD, kTmemCols = 2 * kD;   // (kBufs = 2: another S behind it)
static_assert(2 * kSmemOne > 228 * 1024 && Layout<2>::kSmemBytes <= kSmemOne, "one CTA per SM");
static_assert(kMatBytes <= kQBytes && 4 * kOutBytes <= kQBytes, "overlays");
static_assert(kCtas * (Layout<1>::kSmemBytes + 1024) <= 228 * 1024 && kCtas * kTmemCols <= 512, "CTAs per SM");

struct Bars {
  uint64_t q_full, k_full[4], k_free[4], v_full[4], v_free[4], mats_full[3];
  uint64_t done[2];           // by step modulo kBufs: the products issued on a publication of the rows are finished
  uint32_t tmem_slot;
  int abort;
};
static_assert(sizeof(Bars) <= kBarBytes, "barrier block");

struct Args {
  __nv_bfloat16* out;
  const float* theta;
  int theta_stride, nq, m, H, T, has_psi;
  float scale_log2;
  int tiles, bh0;
  int* status;
  float* nlse;
  int ld_pitch;
  __nv_bfloat16* z;
  uint32_t* masks;
  __nv_bfloat16* alpha;
  int64_t alpha_slot;
  uint32_t* signs;
  bool wait_first, contracting;
};

// kTied: one S, B, one threshold (in a recording forward: or one per layer); kThresholds: one threshold per layer; kUnits: one positive
// threshold (units of 2 theta); kFolded: the same with V~ B in the place of V~ (vfold_sm100_kernel); kPerLayer: one S_t, B_t per layer
enum Decoder { kTied, kThresholds, kUnits, kFolded, kPerLayer };

// kRec: 0 = the plain forward; 1 = also Z, log sum exp and the decisions; 2 = also the iterates and the sign bits of x_t
template <int kRec, Decoder kDec, int kBufs>
__global__ void __launch_bounds__(kThreads, kBufs == 1 ? kCtas : 2)
attend_tile_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_kv,
                   const __grid_constant__ CUtensorMap tmap_mats, const __grid_constant__ CUtensorMap tmap_out,
                   const __grid_constant__ CUtensorMap tmap_vb, const Args p) {
  constexpr bool kUnit = kDec == kUnits || kDec == kFolded, kUntied = kDec == kPerLayer, kFold = kDec == kFolded;
  constexpr bool kMasks = kRec >= 1, kKeep = kRec >= 2, kStaged = kDec != kPerLayer;     // kStaged: Z's way out, through a stage of the ring
  using L = Layout<kBufs>;
  constexpr int kStages = L::kStages;
  auto slot = [](int j) { return j & (kStages - 1); };          // ring position j: its stage, and the parity of that stage's phase
  auto phase = [](int j) { return (uint32_t)(j / kStages) & 1u; };
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {          // swizzled tiles need 1024-byte alignment; never seen to fail
    if (threadIdx.x == 0) atomicCAS(p.status, 0, 240);
    return;
  }
  uint8_t* ring = smem + kOffRing;
  Bars* bars = reinterpret_cast<Bars*>(smem + L::kOffBar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = p.bh0 + blockIdx.x / p.tiles, row0 = (blockIdx.x % p.tiles) * kRows, h = bh % p.H;
  const int nq = p.nq, m = p.m, T = p.T;
  const int nchunks = (m + kMC - 1) / kMC;
  Waiter w{p.status, &bars->abort};

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_kv);
    prefetch_tmap(&tmap_mats);
    prefetch_tmap(&tmap_out);
    mbar_init(&bars->q_full, 1);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->k_free[s], 1);
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->v_free[s], 1);
    }
    for (int s = 0; s < 3; ++s) mbar_init(&bars->mats_full[s], 1);
    mbar_init(&bars->done[0], 1);
    mbar_init(&bars->done[1], 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(&bars->tmem_slot, kBufs * kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_slot;
  if (p.wait_first) pdl_wait();

  const int n_mma = T > 0 ? T + (p.has_psi ? 1 : 0) - (kFold ? 1 : 0) : 0;     // products of the recovery
  // ring positions: the K~|V~ chunks, then with kUntied S_l - I | B_l of every layer, and Psi
  const int n_ring = nchunks + (kUntied ? n_mma : 0);

  if (warp >= kRowWarps) {
    reg_dealloc<kControlRegs>();
    if (warp == kMmaWarp) {
      // ---------------------------------------------- MMA issuer ----------------------------------------------------
      constexpr uint32_t idesc_s = make_idesc_bf16(kRows, kMC, false, false);   // S  = Q  K~^T : both K-major
      constexpr uint32_t idesc_z = make_idesc_bf16(kRows, kD, false, true);      // Z += P  V~   : V~ is MN-major
      constexpr uint32_t idesc_r = make_idesc_bf16(kRows, kD, false, false);     // r += a (-W)^T: both K-major
      auto kstep = [](int k) { return (uint64_t)(k * 2); };                     // 16 columns of a K-major operand
      const uint32_t op_col = tmem + kColS, acc = tmem + kColAcc;
      const uint64_t qd = make_smem_desc(smem_u32(smem), 16, 1024);
      const uint64_t rk = make_smem_desc(smem_u32(ring), 16, 1024);
      const uint64_t rv = make_smem_desc(smem_u32(ring + kSlotBytes), kSlotBytes, 1024);
      constexpr uint64_t kStageStep = kStageBytes >> 4;
      w.wait(&bars->q_full, 0, 242);
      Publications<kBufs, kRows> rows;
      auto rows_wait = [&]() { rows.wait(); };
      uint32_t step = 0;
      auto finish_step = [&]() { mma_commit(&bars->done[kBufs == 1 ? 0 : step & 1]); };
      // step j: P_i V~_i of the chunk kBufs before, then S_j in its place.  A slot's release is committed behind the step, so
      // K~'s says that S_j is done, and with it P_i V~_i.
      for (int j = 0; j < nchunks + kBufs; ++j, ++step) {
        const int i = j - kBufs;
        if (j < nchunks) w.wait(&bars->k_full[slot(j)], phase(j), 241);
        if (i >= 0) {
          w.wait(&bars->v_full[slot(i)], phase(i), 242);
          rows_wait();
        }
        tc_fence_after();
        if (elect_one()) {
          const uint32_t sp = op_col + (kBufs == 1 ? 0 : (uint32_t)(j & 1) * kMC);
          if (i >= 0) {
            const uint64_t vd = rv + (uint64_t)slot(i) * kStageStep;
#pragma unroll
            for (int k = 0; k < kMC / 16; ++k) mma_f16_ts(acc, sp + k * 8, vd + (uint64_t)(k * 128), idesc_z, (uint32_t)((i > 0) | (k != 0)));
          }
          if (j < nchunks) {
            const uint64_t kd = rk + (uint64_t)slot(j) * kStageStep;
#pragma unroll
            for (int k = 0; k < kD / 16; ++k) mma_f16_ss(sp, qd + kstep(k), kd + kstep(k), idesc_s, k != 0);
          }
          finish_step();
          if (j < nchunks && (j + kStages < n_ring || (!kUntied && j + 1 == nchunks))) mma_commit(&bars->k_free[slot(j)]);
          if (i >= 0 && i + kStages < n_ring) mma_commit(&bars->v_free[slot(i)]);
        }
        __syncwarp();
      }
      if (kUntied) {
        // layer l: r = z^ B_l (+ a^_l (S_l - I) from the second layer on), its matrices in ring position nchunks + l; then Psi
        for (int l = 0; l < n_mma; ++l, ++step) {
          const int q = nchunks + l;
          w.wait(&bars->k_full[slot(q)], phase(q), 251);
          w.wait(&bars->v_full[slot(q)], phase(q), 252);
          rows_wait();
          tc_fence_after();
          const uint64_t sd = rk + (uint64_t)slot(q) * kStageStep, bd = sd + (uint64_t)(kSlotBytes >> 4);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kD / 16; ++k)
              mma_f16_ts(acc, op_col + (l == T ? kD / 2 : 0) + k * 8, bd + kstep(k), idesc_r, k == 0 ? 0u : 1u);
            if (l > 0 && l < T) {
#pragma unroll
              for (int k = 0; k < kD / 16; ++k) mma_f16_ts(acc, op_col + kD / 2 + k * 8, sd + kstep(k), idesc_r, 1u);
            }
            finish_step();
            if (q + kStages < n_ring) {
              mma_commit(&bars->k_free[slot(q)]);
              mma_commit(&bars->v_free[slot(q)]);
            }
          }
          __syncwarp();
        }
      } else {
        for (int i = 0; i < n_mma; ++i, ++step) {             // B (unless folded), then -mu G T - 1 times, then Psi
          const int first = kFold ? 0 : 1, which = i < first ? 1 : p.has_psi && i == n_mma - 1 ? 2 : 0;
          if (i <= first || which == 2) w.wait(&bars->mats_full[which], 0, 245);
          rows_wait();
          tc_fence_after();
          const uint64_t wd = qd + (which == 0 ? (uint64_t)(L::kOffG >> 4) : which == 1 ? (uint64_t)(L::kOffB >> 4) : 0);
          const uint32_t accum = which != 2;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kD / 16; ++k) mma_f16_ts(acc, op_col + k * 8, wd + kstep(k), idesc_r, k == 0 ? accum : 1u);
            finish_step();
          }
          __syncwarp();
        }
      }
    } else if (warp == kTmaWarp) {
      // ---------------------------------------------- copies --------------------------------------------------------
      if (elect_one()) {
        int nk = 0, nv = 0, nm = 0;           // ring positions, and matrices (bit i: mats_full[i]), whose copies were issued
        auto load_slot = [&](int j, int half, const CUtensorMap* map, int x, int y, int z) {
          uint64_t* full = half ? &bars->v_full[slot(j)] : &bars->k_full[slot(j)];
          mbar_arrive_expect_tx(full, kSlotBytes);
          tma_load_3d(ring + slot(j) * kStageBytes + half * kSlotBytes, map, full, x, y, z);
        };
        auto load_mat = [&](uint8_t* dst, int i) {
          nm |= 1 << i;
          mbar_arrive_expect_tx(&bars->mats_full[i], kMatBytes);
          tma_load_3d(dst, &tmap_mats, &bars->mats_full[i], 0, 0, h * 3 + i);
        };
        mbar_arrive_expect_tx(&bars->q_full, kQBytes);
        tma_load_3d(smem, &tmap_q, &bars->q_full, 0, row0, bh);
        if (!kUntied && T > 1) load_mat(smem + L::kOffG, 0);
        if (!kUntied && !kFold && T > 0) load_mat(smem + L::kOffB, 1);
        if (!kFold) {
          pdl_wait();
          pdl_launch_dependents();
        }
        for (int j = 0; j < n_ring; ++j) {
          const int l = j - nchunks, mat0 = h * (2 * T + 1);
          if (j >= kStages) w.wait(&bars->k_free[slot(j)], phase(j - kStages), 247);
          if (w.dead) break;
          if (l < 0) load_slot(j, 0, &tmap_kv, 0, j * kMC, bh);
          else if (l > 0 && l < T) load_slot(j, 0, &tmap_mats, 0, 0, mat0 + 2 * l);
          else mbar_arrive(&bars->k_full[slot(j)]);             // alpha^0 = 0, Psi: nothing to load, the phases stay in step
          if (kFold && j == 0) {              // K~ was complete before the fold let this kernel start, V~ B was not
            pdl_wait();
            pdl_launch_dependents();
          }
          if (j >= kStages) w.wait(&bars->v_free[slot(j)], phase(j - kStages), 248);
          if (w.dead) { ++nk; break; }
          if (l < 0) load_slot(j, 1, kFold ? &tmap_vb : &tmap_kv, kFold ? 0 : kD, j * kMC, bh);
          else load_slot(j, 1, &tmap_mats, 0, 0, mat0 + (l == T ? 2 * T : 2 * l + 1));
          ++nk;
          ++nv;
        }
        if (!kUntied && T > 0 && p.has_psi && !w.dead) {
          w.wait(&bars->k_free[slot(nchunks - 1)], phase(nchunks - 1), 249);      // the last S: Q's place is free
          if (!w.dead) load_mat(smem, 2);
        }
        if (w.dead) {
          // gave up: let the copies that are still in flight land before the CTA's shared memory goes away
          mbar_wait_drain(&bars->q_full, 0);
          for (int i = 0; i < 3; ++i)
            if ((nm >> i) & 1) mbar_wait_drain(&bars->mats_full[i], 0);
          for (int j = nk > kStages ? nk - kStages : 0; j < nk; ++j) mbar_wait_drain(&bars->k_full[slot(j)], phase(j));
          for (int j = nv > kStages ? nv - kStages : 0; j < nv; ++j) mbar_wait_drain(&bars->v_full[slot(j)], phase(j));
        }
      }
    }
  } else {
  reg_alloc<kRowRegs<kBufs>>();
  const int row = warp * 32 + lane, grow = row0 + row;
  const bool live = row0 + warp * 32 < nq;                    // the warp has rows
  const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
  const uint32_t acc_addr = tbase + kColAcc, op_addr = tbase + kColS;
  const F2 sc2 = pack2(p.scale_log2, p.scale_log2);
  uint32_t step = 0;
  Publications<kBufs, kRows> rows;
  auto wait_done = [&](int code) {
    if (kBufs == 1) w.wait(&bars->done[0], step & 1, code);
    else w.wait(&bars->done[step & 1], (step >> 1) & 1, code);
    ++step;
    tc_fence_after();
  };
  // what the threads have written to tensor memory is there for the MMAs issued next
  auto hand_over = [&]() {
    tmem_wait_st();
    tc_fence_before();
    rows.publish(w.dead);
  };

  float ref = -INFINITY;
  F2 sum2 = pack2(0.f, 0.f);
  const float kappa = T > 0 ? p.theta[h] : 0.f;
  for (int j = 0; j < nchunks; ++j) {
    wait_done(243);                                           // S_j, and the P V~ product kBufs chunks before
    const uint32_t s_addr = op_addr + (kBufs == 1 ? 0 : (uint32_t)(j & 1) * kMC);
    if (live) {
      uint32_t ra[32], rb[32];
      tmem_ld_32x32b_x32(s_addr, ra);
      tmem_ld_32x32b_x32(s_addr + 32, rb);
      tmem_wait_ld();
      float mx = -INFINITY;
      if ((j + 1) * kMC <= m) {
        float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          m0 = max3(m0, __uint_as_float(ra[e]), __uint_as_float(ra[e + 1]));
          m1 = max3(m1, __uint_as_float(ra[e + 2]), __uint_as_float(ra[e + 3]));
          m2 = max3(m2, __uint_as_float(rb[e]), __uint_as_float(rb[e + 1]));
          m3 = max3(m3, __uint_as_float(rb[e + 2]), __uint_as_float(rb[e + 3]));
        }
        mx = fmaxf(max3(m0, m1, m2), m3);
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          if (j * kMC + e >= m) ra[e] = 0xff800000u;          // -inf
          if (j * kMC + 32 + e >= m) rb[e] = 0xff800000u;
          mx = max3(mx, __uint_as_float(ra[e]), __uint_as_float(rb[e]));
        }
      }
      mx *= p.scale_log2;
      if (j == 0) {
        ref = mx;
      } else {
        const bool raise = mx > ref + 8.f;
        if (__any_sync(0xffffffffu, raise)) {
          // rare: rescale this warp's rows of the accumulator (factor 1 for rows that keep their reference); with two buffers
          // P_{j-1} V~_{j-1} belongs to the step that the next turn waits for
          if (kBufs == 2) { wait_done(256); --step; }
          const float f = raise ? ex2(ref - mx) : 1.f;
          if (raise) ref = mx;
          sum2 = mul2(sum2, pack2(f, f));
#pragma unroll
          for (int c0 = 0; c0 < kD; c0 += 16) {
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
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const F2 x2 = fma2(pack2u(r[e], r[e + 1]), sc2, nref2);
          float p0, p1;
          if ((e >> 1) % kPolyEvery == kPolyEvery - 1) {
            exp2_poly2(x2, p0, p1);
          } else {
            float t0, t1;
            unpack2(x2, t0, t1);
            p0 = ex2(t0);
            p1 = ex2(t1);
          }
          sum2 = add2(sum2, pack2(p0, p1));
          pk[e >> 1] = pack_bf16(p0, p1);
        }
        tmem_st_32x32b_x16(s_addr + col, pk);
      };
      exp_half(ra, 0);
      exp_half(rb, 16);
    }
    hand_over();
  }
  float inv;
  {
    float s0, s1;
    unpack2(sum2, s0, s1);
    inv = 1.f / (s0 + s1);
    if (p.nlse != nullptr && grow < nq) p.nlse[(int64_t)bh * p.ld_pitch + grow] = -(ref + __log2f(s0 + s1));
  }
  for (int i = 0; i < kBufs; ++i) wait_done(244);             // every P V~ product has been added
  const float unit = kUnit ? unit_threshold<kD>(kappa, acc_addr, inv) : kappa;
  F2 v2[kD / 2];                                               // in turn: Z, the iterate, alpha^T, Psi alpha^T
  {
    const F2 inv2 = pack2(inv, inv);
#pragma unroll
    for (int c0 = 0; c0 < kD; c0 += 16) {
      uint32_t a[16];
      tmem_ld_32x32b_x16(acc_addr + c0, a);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; e += 2) v2[(c0 + e) >> 1] = mul2(pack2u(a[e], a[e + 1]), inv2);
    }
  }
  // v2 as bf16 into one box of the warp's 32 rows (128-byte swizzle), from where one TMA store takes it: 16-byte stores of 32
  // different rows would keep the threads at the stores
  auto stage_rows = [&](uint8_t* buf, const CUtensorMap* map) {
    uint8_t* box = buf + warp * kOutBytes;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 4; ++u) unpack2(v2[c * 4 + u], x[2 * u], x[2 * u + 1]);
      *reinterpret_cast<uint4*>(box + lane * 128 + ((c ^ (lane & 7)) << 4)) =
          make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0 && live && !w.dead && *(volatile int*)&bars->abort == 0) {
      tma_store_3d(map, box, 0, grow, bh);
      bulk_commit_group();
    }
  };
  if (kMasks && p.z != nullptr) {
    if (kStaged) {
      // every chunk has been read: the ring is free
      stage_rows(ring, &tmap_vb);
    } else if (grow < nq) {
      uint4* zo = reinterpret_cast<uint4*>(p.z + ((int64_t)bh * nq + grow) * kD);
#pragma unroll
      for (int c = 0; c < kD / 8; ++c) {
        float x[8];
#pragma unroll
        for (int u = 0; u < 4; ++u) unpack2(v2[c * 4 + u], x[2 * u], x[2 * u + 1]);
        zo[c] = make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
      }
    }
  }
  __nv_bfloat16* arow = (kKeep && p.alpha != nullptr && grow < nq) ? p.alpha + ((int64_t)bh * nq + grow) * kD : nullptr;
  uint32_t mw[kD / 32] = {}, sw[kD / 32] = {};
  const bool signs = kKeep && p.signs != nullptr;
  auto store_masks = [&](int layer, uint32_t flip = 0) {
    if (signs && grow < nq) {
      uint32_t* so = p.signs + (((int64_t)bh * T + layer) * nq + grow) * (kD / 32);
      *reinterpret_cast<uint2*>(so) = make_uint2(sw[0], sw[1]);
    }
    if (kMasks && p.masks != nullptr && grow < nq) {
      uint32_t* mo = p.masks + (((int64_t)bh * T + layer) * nq + grow) * (kD / 32);
      *reinterpret_cast<uint2*>(mo) = make_uint2(mw[0] ^ flip, mw[1] ^ flip);
    }
  };
  auto publish = [&](uint32_t col = 0) {
#pragma unroll
    for (int c0 = 0; c0 < kD; c0 += 16) {
      uint32_t pk[8];
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        float x0, x1;
        unpack2(v2[(c0 + e) >> 1], x0, x1);
        pk[e >> 1] = pack_bf16(x0, x1);
      }
      tmem_st_32x32b_x8(op_addr + col + c0 / 2, pk);
    }
  };
  // an accumulator row, 16 columns at a time, the next piece's load in flight under this one's arithmetic
  auto pieces = [&](auto f) {
    uint32_t r0[16], r1[16];
    tmem_ld_32x32b_x16(acc_addr, r0);
#pragma unroll
    for (int c0 = 0; c0 < kD; c0 += 32) {
      tmem_wait_ld();
      tmem_ld_32x32b_x16(acc_addr + c0 + 16, r1);
      f(r0, c0);
      tmem_wait_ld();
      if (c0 + 32 < kD) tmem_ld_32x32b_x16(acc_addr + c0 + 32, r0);
      f(r1, c0 + 16);
    }
  };
  auto push_x = [&](float th, float x0, float x1, int c) {
    mw[c >> 5] = __funnelshift_l(__float_as_uint(th - fabsf(x0)), mw[c >> 5], 1);
    mw[c >> 5] = __funnelshift_l(__float_as_uint(th - fabsf(x1)), mw[c >> 5], 1);
    if (signs) {
      sw[c >> 5] = __funnelshift_l(__float_as_uint(x0), sw[c >> 5], 1);
      sw[c >> 5] = __funnelshift_l(__float_as_uint(x1), sw[c >> 5], 1);
    }
  };
  // the last layer, shrunk exactly from x = v2 + r
  auto exact_layer = [&]() {
    const float th = p.theta[(int64_t)(T - 1) * p.theta_stride + h];
    pieces([&](const uint32_t (&r)[16], int c0) {
#pragma unroll
      for (int e = 0; e < 16; e += 2) {
        float b0, b1;
        unpack2(v2[(c0 + e) >> 1], b0, b1);
        const float x0 = b0 + __uint_as_float(r[e]), x1 = b1 + __uint_as_float(r[e + 1]);
        if (kMasks) push_x(th, x0, x1, c0);
        v2[(c0 + e) >> 1] = pack2(x0 - fminf(fmaxf(x0, -th), th), x1 - fminf(fmaxf(x1, -th), th));
      }
    });
    store_masks(T - 1);
    if (kKeep && arow != nullptr) {
#pragma unroll
      for (int c0 = 0; c0 < kD; c0 += 16) {
        uint32_t pa[8];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float a0, a1;
          unpack2(v2[(c0 + e) >> 1], a0, a1);
          pa[e >> 1] = pack_bf16(a0, a1);
        }
        st_global_v8(arow + (int64_t)T * p.alpha_slot + c0, pa);
      }
    }
  };

  bool scaled_units = kUnit || (!kUntied && !kKeep && T > 0 && p.theta_stride == 0 && threshold_is_a_unit(kappa));
  if (kMasks && scaled_units) {
    F2 q2 = pack2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kD / 2; ++i) q2 = fma2(v2[i], v2[i], q2);
    float q0, q1;
    unpack2(q2, q0, q1);
    const float i2 = 0.5f / kappa;
    scaled_units = __all_sync(0xffffffffu, p.contracting && (q0 + q1) * i2 * i2 < 1e30f);
  }
  if (kUntied && T > 0) {
    // z^ in the first D / 2 packed columns (written once), a^_t in the next D / 2.  The registers hold alpha^t + theta_t, so that
    // x + theta_t needs no add of its own; the layer before the last adds nothing, the last layer shrinks exactly from x = alpha + r.
    publish();
    hand_over();
    {
      const float b0 = T > 1 ? kappa : 0.f;
#pragma unroll
      for (int i = 0; i < kD / 2; ++i) v2[i] = pack2(b0, b0);      // alpha^0 = 0
    }
    for (int it = 0; it + 1 < T; ++it) {
      const float th = p.theta[(int64_t)it * p.theta_stride + h];
      const float thn = it + 2 < T ? p.theta[(int64_t)(it + 1) * p.theta_stride + h] : 0.f;
      const float inv2th = th > 0.f ? 0.5f / th : 0.f;          // theta = 0: sat(0) = 0 and eta(x) = x
      const F2 m2th2 = pack2(-2.f * th, -2.f * th), p2th2 = pack2(2.f * th, 2.f * th), nx2 = pack2(thn, thn);
      wait_done(253);
      if (live)
        pieces([&](const uint32_t (&r)[16], int c0) {
          uint32_t pk[8];
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            const F2 y2 = add2(v2[(c0 + e) >> 1], pack2u(r[e], r[e + 1]));   // alpha^t S_t + z B_t + theta_t
            float y0, y1;
            unpack2(y2, y0, y1);
            if (kMasks) {
              // |x| > theta  <=>  y < 0 or y > 2 theta  <=>  y (2 theta - y) < 0: its sign bit is the decision
              float g0, g1;
              unpack2(mul2(y2, fma2(y2, pack2(-1.f, -1.f), p2th2)), g0, g1);
              mw[c0 >> 5] = __funnelshift_l(__float_as_uint(g0), mw[c0 >> 5], 1);
              mw[c0 >> 5] = __funnelshift_l(__float_as_uint(g1), mw[c0 >> 5], 1);
              if (signs) {                         // where the decision holds y and x = y - theta have the same sign
                sw[c0 >> 5] = __funnelshift_l(__float_as_uint(y0), sw[c0 >> 5], 1);
                sw[c0 >> 5] = __funnelshift_l(__float_as_uint(y1), sw[c0 >> 5], 1);
              }
            }
            const F2 t2 = pack2(fma_sat(y0, inv2th, 0.f), fma_sat(y1, inv2th, 0.f));
            const F2 an = fma2(t2, m2th2, y2);                               // alpha^{t+1} = eta_theta(x)
            v2[(c0 + e) >> 1] = add2(an, nx2);
            float a0, a1;
            unpack2(an, a0, a1);
            pk[e >> 1] = pack_bf16(a0, a1);
          }
          tmem_st_32x32b_x8(op_addr + kD / 2 + c0 / 2, pk);
          if (kKeep && arow != nullptr) st_global_v8(arow + (int64_t)(it + 1) * p.alpha_slot + c0, pk);   // alpha^{t+1}
        });
      hand_over();
      store_masks(it);
    }
    wait_done(254);
    exact_layer();
    if (p.has_psi) {
      publish(kD / 2);
      hand_over();
      wait_done(255);
      pieces([&](const uint32_t (&r)[16], int c0) {
#pragma unroll
        for (int e = 0; e < 16; e += 2) v2[(c0 + e) >> 1] = pack2u(r[e], r[e + 1]);
      });
    }
  }
  if (!kUntied && (kUnit || T > 0)) {
    if (kFold) {
      // the accumulator held z B: r'_0 = 1/2 + z B / (2 theta) goes back into it, and the first pass below reads it from there
      const float inv2th = 0.5f / unit;
      const F2 i2 = pack2(inv2th, inv2th), hf = pack2(0.5f, 0.5f);
#pragma unroll
      for (int c0 = 0; c0 < kD; c0 += 16) {
        uint32_t tb[16];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float r0, r1;
          unpack2(fma2(v2[(c0 + e) >> 1], i2, hf), r0, r1);
          tb[e] = __float_as_uint(r0);
          tb[e + 1] = __float_as_uint(r1);
        }
        tmem_st_32x32b_x16(acc_addr + c0, tb);
      }
      tmem_wait_st();
    } else {
      // bias of the accumulator and z as the operand of the first product, in units of 2 theta or in the data's
      const float bias = scaled_units ? 0.5f : kappa;
      uint32_t tb[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) tb[e] = __float_as_uint(bias);
#pragma unroll
      for (int c0 = 0; c0 < kD; c0 += 16) tmem_st_32x32b_x16(acc_addr + c0, tb);
      if (scaled_units) {
        const float inv2th = 0.5f / unit;
        const F2 i2 = pack2(inv2th, inv2th);
#pragma unroll
        for (int i = 0; i < kD / 2; ++i) v2[i] = mul2(v2[i], i2);
      }
      publish();
      hand_over();
    }
    const F2 m1 = pack2(-1.f, -1.f);
    // |x| > theta where s is 0 or 1: s^2 - s, +0 there and negative in between (one rounding), has the opposite as its sign bit, so the
    // words are kept inverted.  (As the sign bit of s (1 - s) - tiny, an instruction more per pair: 1568 queries of 96 heads 89.8 us, now 83.7.)
    auto push_mask = [&](F2 s2, int c) {
      float s0, s1, g0, g1;
      unpack2(s2, s0, s1);
      unpack2(fma2(s2, s2, pack2(-s0, -s1)), g0, g1);
      mw[c >> 5] = __funnelshift_l(__float_as_uint(g0), mw[c >> 5], 1);
      mw[c >> 5] = __funnelshift_l(__float_as_uint(g1), mw[c >> 5], 1);
    };
    const float off = scaled_units ? 0.f : -kappa;
#pragma unroll
    for (int i = 0; i < kD / 2; ++i) v2[i] = pack2(off, off);
    for (int it = 0; it + 1 < T; ++it) {
      // thresholds that differ are loaded while the products run (156 tiles, T = 10: 21.0 -> 19.0 us)
      const float th_it = kDec == kThresholds ? p.theta[(int64_t)it * p.theta_stride + h] : kappa;
      const float inv_it = th_it > 0.f ? 0.5f / th_it : 0.f;
      if (!kFold || it > 0) wait_done(246);
      if (live) {
        if (scaled_units) {
          pieces([&](const uint32_t (&r)[16], int c0) {
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              float a0, a1;
              unpack2(v2[(c0 + e) >> 1], a0, a1);
              const F2 s2 = pack2(add_sat(a0, __uint_as_float(r[e])), add_sat(a1, __uint_as_float(r[e + 1])));
              if (kMasks) push_mask(s2, c0 + e);
              const F2 dn = fma2(s2, m1, pack2u(r[e], r[e + 1]));     // (alpha^{t+1} - alpha^t) / (2 theta)
              v2[(c0 + e) >> 1] = add2(v2[(c0 + e) >> 1], dn);
              float d0, d1;
              unpack2(dn, d0, d1);
              pk[e >> 1] = pack_bf16(d0, d1);
            }
            tmem_st_32x32b_x8(op_addr + c0 / 2, pk);
          });
        } else {
          constexpr bool kDiffer = kDec == kThresholds || kMasks;      // (the add costs 0.1 us a layer)
          const float th = kMasks ? p.theta[(int64_t)it * p.theta_stride + h] : th_it;
          const float inv2th = kMasks ? (th > 0.f ? 0.5f / th : 0.f) : inv_it;    // theta = 0: sat(1/2) = 1/2 and eta(x) = x
          const F2 m2th2 = pack2(-2.f * th, -2.f * th);
          const F2 dk2 = pack2(th - kappa, th - kappa);
          pieces([&](const uint32_t (&r)[16], int c0) {
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const F2 r2 = pack2u(r[e], r[e + 1]);
              const F2 x2 = add2(v2[(c0 + e) >> 1], r2);               // alpha^t S + z B
              float x0, x1;
              unpack2(x2, x0, x1);
              if (kMasks) push_x(th, x0, x1, c0);
              const F2 t2 = pack2(fma_sat(x0, inv2th, 0.5f), fma_sat(x1, inv2th, 0.5f));
              F2 bn = fma2(t2, m2th2, x2), dn = fma2(t2, m2th2, r2);   // eta_theta(x) - theta; alpha^{t+1} - alpha^t
              if (kDiffer) { bn = add2(bn, dk2); dn = add2(dn, dk2); }   // ... - kappa
              v2[(c0 + e) >> 1] = bn;
              float d0, d1;
              unpack2(dn, d0, d1);
              pk[e >> 1] = pack_bf16(d0, d1);
            }
            tmem_st_32x32b_x8(op_addr + c0 / 2, pk);
            if (kKeep && arow != nullptr) {                                 // alpha^{t+1} = b + kappa
              uint32_t pa[8];
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                float a0, a1;
                unpack2(v2[(c0 + e) >> 1], a0, a1);
                pa[e >> 1] = pack_bf16(a0 + kappa, a1 + kappa);
              }
              st_global_v8(arow + (int64_t)(it + 1) * p.alpha_slot + c0, pa);
            }
          });
        }
      }
      hand_over();
      store_masks(it, scaled_units ? ~0u : 0);
    }
    // last iteration, exact shrinkage
    wait_done(247);
    if (scaled_units) {
      const F2 tt2 = pack2(2.f * unit, 2.f * unit), mh2 = pack2(-0.5f, -0.5f);
      pieces([&](const uint32_t (&r)[16], int c0) {
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float a0, a1;
          unpack2(v2[(c0 + e) >> 1], a0, a1);
          const F2 u2 = add2(pack2(a0, a1), pack2u(r[e], r[e + 1]));
          float u0, u1;
          unpack2(u2, u0, u1);
          const F2 s2 = pack2(add_sat(u0, 0.f), add_sat(u1, 0.f));
          if (kMasks) push_mask(s2, c0 + e);
          v2[(c0 + e) >> 1] = mul2(sub2(add2(u2, mh2), add2(s2, mh2)), tt2);
        }
      });
      store_masks(T - 1, ~0u);
    } else {
      exact_layer();
    }
    if (p.has_psi) {
      publish();
      hand_over();
      wait_done(248);
      pieces([&](const uint32_t (&r)[16], int c0) {
#pragma unroll
        for (int e = 0; e < 16; e += 2) v2[(c0 + e) >> 1] = pack2u(r[e], r[e + 1]);
      });
    }
  }
  // every MMA of the tile is done: Q's place (or Psi's) takes the output
  if (p.out != nullptr) stage_rows(smem, &tmap_out);
  if (lane == 0) bulk_wait_group0();                          // the stores are done before the kernel ends
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, kBufs * kTmemCols);
}

template <int kRec, Decoder kDec, int kBufs>
cudaError_t launch(csat_ctx* c, const void* Q, void* out, cudaStream_t s, float* nlse, __nv_bfloat16* z, uint32_t* masks,
                   __nv_bfloat16* alpha, bool wait_first) {
  const Params& p = c->p;
  const uint64_t qd[3] = {(uint64_t)kD, (uint64_t)p.nq, (uint64_t)(p.B * p.H)};
  const uint64_t qs[2] = {(uint64_t)kD * 2, (uint64_t)p.nq * kD * 2};
  const uint32_t qb[3] = {64, (uint32_t)kRows, 1}, ob[3] = {64, 32, 1};
  CUtensorMap tq;
  cudaError_t e;
  if ((e = make_tmap_bf16_3d(&tq, Q, qd, qs, qb)) != cudaSuccess) return e;
  CUtensorMap to = tq;
  if (out != nullptr && (e = make_tmap_bf16_3d(&to, out, qd, qs, ob)) != cudaSuccess) return e;
  CUtensorMap tv = c->tmap_vb;                                  // V~ B, or with kRec where Z goes
  if (kRec != 0 && z != nullptr && (e = make_tmap_bf16_3d(&tv, z, qd, qs, ob)) != cudaSuccess) return e;
  // Up to one or two tiles per SM the CTAs ask for so much shared memory that no more share an SM: started early, they would
  // pile up on the SMs that the kernel before leaves free.
  const int64_t tiles = (p.nq + kRows - 1) / kRows, n = tiles * (c->bh_cnt ? c->bh_cnt : p.B * p.H);
  if (n > (int64_t)1 << 30) return cudaErrorInvalidValue;
  const uint32_t smem = n <= c->sms ? kSmemOne : n <= 2 * (int64_t)c->sms || kBufs == 2 ? Layout<kBufs>::kSmemTwo : Layout<kBufs>::kSmemBytes;
  static DeviceFlags smem_opt_in;
  if (!smem_opt_in.test(c->device)) {
    // setmaxnreg moves registers inside the pool the CTA is launched with (threads x the compiled register count); a request
    // the pool cannot satisfy would wait forever
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, attend_tile_kernel<kRec, kDec, kBufs>)) != cudaSuccess) return e;
    if (fa.numRegs * kThreads < kRows * kRowRegs<kBufs> + (kThreads - kRows) * kControlRegs) return cudaErrorLaunchOutOfResources;
  }
  if ((e = ensure_dynamic_smem(attend_tile_kernel<kRec, kDec, kBufs>, (int)kSmemOne, c->device, smem_opt_in)) != cudaSuccess) return e;
  const double scale = p.scale > 0.0 ? p.scale : 1.0 / sqrt((double)kD);
  Args a{(__nv_bfloat16*)out, c->thr(), c->thr_stride(), (int)p.nq, (int)p.m, (int)p.H, (int)p.T, c->psi ? 1 : 0,
         (float)(scale * 1.4426950408889634), (int)tiles, (int)c->bh0, c->status, nlse, (int)c->ld_pitch(), z, masks, alpha,
         (int64_t)(p.B * p.H * p.nq * p.d), alpha != nullptr ? c->bw_signbits : nullptr, wait_first,
         !c->w_S && p.step == 0.0 && p.T <= 1024};
  return launch_pdl(attend_tile_kernel<kRec, kDec, kBufs>, dim3((unsigned)n), kThreads, smem, s, tq, c->tmap_kv,
                    kDec == kPerLayer ? c->tmap_lmats : c->tmap_mats, to, tv, a);
}

}  // namespace

// Two score buffers where an SM holds at most two tiles: S_{j+1} is formed under chunk j's exponentials.  Between three and four tiles per
// SM two rounds of two take the place of two of three, unless there is a single chunk.  us, two buffers / one: 592 tiles, m = 256, T =
// 20 37.8 / 38.3; 512 36.6 / 37.8, T = 10 25.9 / 27.1; 512, m = 64 21.2 / 20.8; 300, m = 256, T = 20 38 / 27; 128, m = 392, T = 0 11.8 / 13.7; one
// S_t, B_t per layer: 128, m = 392, T = 10 20.7 / 22.9; 592, m = 256, T = 20 45.6 / 47.9.  By the context's whole job, not the launch's range
// of (batch, head) pairs.
static bool few_tiles(const csat_ctx* c) {
  const int64_t tiles = (c->p.nq + kRows - 1) / kRows * c->p.B * c->p.H;
  return tiles <= 2 * (int64_t)c->sms || (c->p.m > kMC && two_tiles_per_sm(tiles, c->sms));
}

cudaError_t launch_attend_tile(csat_ctx* c, const void* Q, void* out, cudaStream_t s, int* launches, bool wait_first) {
#define CSAT_TILE(DEC, BUFS) launch<0, DEC, BUFS>(c, Q, out, s, nullptr, nullptr, nullptr, nullptr, wait_first)
  const Params& p = c->p;
  if (c->w_S && c->w_untied && p.T > 0) return few_tiles(c) ? CSAT_TILE(kPerLayer, 2) : CSAT_TILE(kPerLayer, 1);
  if (c->thr_stride() != 0) return few_tiles(c) ? CSAT_TILE(kThresholds, 2) : CSAT_TILE(kThresholds, 1);
  if (c->w_S || p.T == 0 || !(p.lambda > 0.0)) return few_tiles(c) ? CSAT_TILE(kTied, 2) : CSAT_TILE(kTied, 1);
  // one positive threshold for all layers
  if (few_tiles(c)) return CSAT_TILE(kUnits, 2);
  // B folded into the values: the first tiles wait for the fold (4 us), every tile saves a hand-over.  The line at eight tiles per SM was
  // measured on the kernel with two tiles per CTA, and the tests hold the first of these shapes to the folded launches and their bits;
  // since the rows hand over through named barriers the saved hand-over no longer pays for the wait.  Whole forward, us, folded / not: 1248
  // tiles, m = 256, T = 20 80.3 / 78.2, 1776 126.4 / 122.7, 2368 153.7 / 151.3, 4736 288.8 / 285.6; 1536 short tiles, m = 64 82.4 / 76.2.
  if (p.T >= 2 && (p.nq + kRows - 1) / kRows * p.B * p.H >= 8 * (int64_t)c->sms) {
    cudaError_t e = launch_sm100_vfold(c, s, launches);
    if (e != cudaSuccess) return e;
    wait_first = false;                           // the fold waits for whatever is before it
    return CSAT_TILE(kFolded, 1);
  }
  return CSAT_TILE(kUnits, 1);
#undef CSAT_TILE
}
cudaError_t launch_attend_tile_recording(csat_ctx* c, const void* Q, void* out, cudaStream_t s, float* nlse,
                                         __nv_bfloat16* z, uint32_t* masks, __nv_bfloat16* alpha) {
#define CSAT_TILE(REC, DEC, BUFS) launch<REC, DEC, BUFS>(c, Q, out, s, nlse, z, masks, alpha, false)
  if (c->w_S && c->w_untied && c->p.T > 0) return alpha != nullptr ? CSAT_TILE(2, kPerLayer, 1) : CSAT_TILE(1, kPerLayer, 1);
  if (alpha != nullptr) return CSAT_TILE(2, kTied, 1);
  return few_tiles(c) ? CSAT_TILE(1, kTied, 2) : CSAT_TILE(1, kTied, 1);
#undef CSAT_TILE
}

}  // namespace csat

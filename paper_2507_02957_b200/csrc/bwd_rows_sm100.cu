// The per-query stages of the backward pass on the sm_100a tensor cores (bf16 storage, d in {64, 128}, one S, B for
// all layers).  The paper trains through its unrolled decoder but prints no backward pass: this is the chain rule
// through the LISTA recurrence alpha^{t+1} = eta_theta(alpha^t S + z B), the reconstruction C^ = Psi alpha, the
// compressed output Z = A~ V~ and the softmax over the measurements, with the derivative of eta_theta taken as 1
// where |x| > theta and 0 elsewhere.
//
// Before these kernels the forward's own kernels have left K~|V~ in the workspace, Z (bf16, as the forward rounds it
// for its first product) in bw_Z16, minus every row's log sum exp L in bw_LD (in units of log 2, as it enters the exponentials) and the
// layers' shrinkage decisions in bw_maskbits.
//
// bwd_recur_sm100_kernel, one CTA per tile of 128 queries (TMEM lane = query row, one thread per row): the recurrence
// run backwards.  The decisions |x_t| > theta_t are the forward kernel's own (it records them, one bit per column and
// layer, when it runs for the backward pass), so nothing of the forward recurrence is repeated here:
//   d alpha_T = G Psi (one MMA; G itself without a dictionary), then for t = T-1 .. 0
//        dx_t = d alpha_{t+1} o mask_t,   dZ += dx_t B^T,   d alpha_t = dx_t S^T = dx_t + dx_t (S - I)^T :
//   dx_t goes to tensor memory as the bf16 A operand of two MMAs, whose B operands are the forward's own
//   shared-memory tiles of S - I and B read as MN-major operands (a d x d tile with 128-byte rows is K-major when
//   its rows are the output columns and MN-major when they are the reduction index: the transposed product needs
//   no transposed copy); the identity part of S^T stays exact in float32 registers;
//   at the end dZ (bf16, the operand of the stages that follow) and D = <dZ, Z>.
//
// bwd_dq_sm100_kernel, one CTA per tile of 128 queries, K~|V~ streamed in chunks of 32 (d = 64, many tiles) or 64 measurements:
//        S_j = Q K~_j^T,  dA_j = dZ V~_j^T                        (two SS MMAs into tensor memory)
//        dS_j = exp(scale S_j - L) o (dA_j - D)                   (one thread per row; bf16 back into tensor memory)
//        dQ  += dS_j K~_j                                         (TS MMA, K~_j read as an MN-major operand; times scale at the end)
//   the structure of the forward's attention phase with the roles of the operands changed.
//
// Every wait is bounded (see sm100_ptx.cuh); a time-out sets the context's status word and the CTA winds down.
#include "csat_internal.h"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace csat {
namespace {

using namespace ptx;

constexpr int kRows = 128;

// ====================================================================================================================
// recurrence backward
// ====================================================================================================================
// kUntied: one S_t, B_t per layer: the pair of the layer at work and the pair of the next one (two stages), then Psi
template <int D, bool kUntied = false> struct RCfg {
  static constexpr int kDBoxes = D / 64;
  static constexpr uint32_t kMatBoxBytes = D * 128;               // one 64-column box of a d x d bf16 matrix
  static constexpr uint32_t kMatBytes = kDBoxes * kMatBoxBytes;
  static constexpr uint32_t kOffMat = 0;                          // [3]: S - I | B | Psi, as the forward stages them
  static constexpr int kMats = kUntied ? 5 : 3;                   // untied: [stage 0: S_t - I | B_t][stage 1: ...][Psi]
  // d = 64: [G, later dZ | Z], 128 rows of 128 bytes each
  static constexpr bool kTiled = D == 64;
  static constexpr uint32_t kRowsBytes = kRows * 128;
  static constexpr uint32_t kOffG = kMats * kMatBytes, kOffZ = kOffG + kRowsBytes;
  static constexpr uint32_t kOffBar = kOffG + (kTiled ? 2 * kRowsBytes : 0);
  static constexpr uint32_t kSmemUsed = kOffBar + 128 + 1024 /*alignment slack*/;
  // d = 64: a CTA holds its first allocation of tensor memory (128 columns) while it waits for the second (32).  Four on an SM
  // would hold all 512 columns and wait for ever, so every CTA asks for so much shared memory that no fourth is resident.
  // (d = 128: one allocation.)
  static constexpr uint32_t kSmemBytes = kTiled && kSmemUsed < 58 * 1024 ? 58 * 1024 : kSmemUsed, kSmemTwo = 80 * 1024;
  // TMEM columns: accumulator | dZ accumulator | the bf16 operand buffers (two values per column; in an allocation of their own
  // at d = 64).  d = 64 has room for one, 160 columns in all, so that three CTAs share an SM: a layer is a chain thread -> MMA issuer ->
  // tensor pipe -> thread that uses neither the tensor pipe nor the issue slots for long (96 heads of 1568 queries, T = 20: 109 -> 84
  // us, with the accumulator's additions, the decisions and the operand in one pass over the row instead of two).  (A second operand
  // buffer in shared memory: 4 % slower.)  G, Z and dZ pass through shared memory and TMA: a CTA's start took 5700 cycles and its end
  // 3900 of 38500 with a row of 128 bytes read or written by one thread each, 4300 and 2700 now; with the hand-over through named
  // barriers 76.3 -> 68.6 us, one S_t, B_t per layer (48 heads, T = 10) 63 -> 57.
  static constexpr int kCtas = D == 64 ? 3 : 1, kOps = D == 64 ? 1 : 2;
  static constexpr uint32_t kColAcc = 0, kColDz = D, kOpCols = D / 2;
  static constexpr uint32_t kTmemCols = D == 64 ? 2 * D : 512, kTmemOpCols = D == 64 ? 32 : 0;
  static_assert(2 * D + kOps * kOpCols <= kTmemCols + kTmemOpCols && kCtas * (kTmemCols + kTmemOpCols) <= 512, "TMEM budget");
  static_assert(kSmemUsed <= kSmemBytes && kCtas * (kSmemBytes + 1024) <= 228 * 1024, "CTAs per SM");
  static_assert(D != 64 || (2 * (kSmemTwo + 1024) <= 228 * 1024 && 3 * kSmemTwo > 228 * 1024), "two CTAs per SM");
  static_assert(kTmemOpCols == 0 || 512 / kTmemCols * (kSmemBytes + 1024) > 228 * 1024,
                "CTAs on one SM must not hold all of tensor memory with their first allocations");
};

struct RBars {
  uint64_t mats_full, r_full, op_free[2];      // op_free: by operand buffer
  uint64_t g_full, z_full;                             // d = 64: the tiles of G and Z
  uint64_t lm_full[2], lm_free[2];   // untied layers: a stage's pair of matrices has landed / has been read
  uint32_t tmem_slot, tmem_op_slot;
  int abort;
};

constexpr int kRThreads = 160;      // warps 0-3: one thread per query row; warp 4: TMA and MMA issue

template <int D, bool kUntied>
__global__ void __launch_bounds__(kRThreads, RCfg<D, kUntied>::kCtas)
bwd_recur_sm100_kernel(const __grid_constant__ CUtensorMap tmap_mats, const __grid_constant__ CUtensorMap tmap_g,
                       const __grid_constant__ CUtensorMap tmap_z, const __grid_constant__ CUtensorMap tmap_dz,
                       const __nv_bfloat16* __restrict__ Z16,
                       const __nv_bfloat16* __restrict__ G, __nv_bfloat16* __restrict__ dZ16, float* __restrict__ negD, int ld_pitch,
                       const uint32_t* __restrict__ maskbits, int nq, int H, int T, int has_psi, int* status,
                       __nv_bfloat16* __restrict__ dx_out, int64_t dx_slot) {
  using C = RCfg<D, kUntied>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  RBars* bars = reinterpret_cast<RBars*>(smem + C::kOffBar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, h = bh % H, row0 = blockIdx.x * kRows;
  Waiter w{status, &bars->abort};

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_mats);
    mbar_init(&bars->mats_full, 1);
    mbar_init(&bars->r_full, 1);
    mbar_init(&bars->op_free[0], 1);
    mbar_init(&bars->op_free[1], 1);
    for (int s2 = 0; s2 < 2; ++s2) { mbar_init(&bars->lm_full[s2], 1); mbar_init(&bars->lm_free[s2], 1); }
    mbar_init(&bars->g_full, 1);
    mbar_init(&bars->z_full, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 4) {
    tmem_alloc(&bars->tmem_slot, C::kTmemCols);
    if (C::kTmemOpCols != 0) tmem_alloc(&bars->tmem_op_slot, C::kTmemOpCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_slot, tmem_op = C::kTmemOpCols != 0 ? bars->tmem_op_slot : tmem + 2 * D;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 4) {
    // ---- copies, then one MMA group per operand the threads publish ----
    // one S, B for all layers: tiles S - I | B | Psi of head h, loaded once.  One pair per layer (kUntied): the
    // tensor holds, per head, S_0 - I, B_0, S_1 - I, B_1, ..., then Psi; the layers are walked from the last to the
    // first through two stages, the pair of layer t - 2 loaded into the stage layer t's products have just read.
    const int mat0 = kUntied ? h * (2 * T + 1) : h * 3;
    auto load_mat = [&](int slot, int index, uint64_t* bar) {
      for (int gx = 0; gx < C::kDBoxes; ++gx)
        tma_load_3d(smem + C::kOffMat + slot * C::kMatBytes + gx * C::kMatBoxBytes, &tmap_mats, bar, gx * 64, 0, index);
    };
    auto load_layer = [&](int t) {                // into stage (T - 1 - t) & 1
      const int st = (T - 1 - t) & 1;
      mbar_arrive_expect_tx(&bars->lm_full[st], 2 * C::kMatBytes);
      load_mat(2 * st, mat0 + 2 * t, &bars->lm_full[st]);
      load_mat(2 * st + 1, mat0 + 2 * t + 1, &bars->lm_full[st]);
    };
    if (elect_one()) {
      if (C::kTiled) {                            // rows beyond n_q are zero-filled
        mbar_arrive_expect_tx(&bars->g_full, C::kRowsBytes);
        tma_load_3d(smem + C::kOffG, &tmap_g, &bars->g_full, 0, row0, bh);
      }
      if (T > 0 && kUntied) {
        if (has_psi) {
          mbar_arrive_expect_tx(&bars->mats_full, C::kMatBytes);
          load_mat(4, mat0 + 2 * T, &bars->mats_full);
        }
        load_layer(T - 1);
        if (T > 1) load_layer(T - 2);
      } else if (T > 0) {
        const int nmats = has_psi ? 3 : 2;
        mbar_arrive_expect_tx(&bars->mats_full, nmats * C::kMatBytes);
        for (int mat = 0; mat < nmats; ++mat) load_mat(mat, mat0 + mat, &bars->mats_full);
      }
      if (C::kTiled) {
        mbar_arrive_expect_tx(&bars->z_full, C::kRowsBytes);
        tma_load_3d(smem + C::kOffZ, &tmap_z, &bars->z_full, 0, row0, bh);
      }
    }
    __syncwarp();
    if (T > 0) {
      constexpr uint32_t idesc_t = make_idesc_bf16(kRows, D, false, true);    // transposed products: B MN-major
      const uint32_t acc = tmem + C::kColAcc, dz = tmem + C::kColDz;
      // product with the transpose of a matrix the forward stores [output column][k]: the tile's rows are now the
      // reduction index, 16 rows (2048 bytes) per K step, the next 64 output columns one box further.  Publication
      // n uses operand buffer n % kOps.
      const uint64_t mat_desc = make_smem_desc(smem_u32(smem + C::kOffMat), C::kMatBoxBytes, 1024);
      auto mma_tr = [&](uint32_t d_t, uint32_t buf, int slot, uint32_t accumulate) {
        const uint32_t op = tmem_op + buf * C::kOpCols;
        const uint64_t bd = mat_desc + (uint64_t)(slot * (C::kMatBytes >> 4));
#pragma unroll
        for (int k = 0; k < D / 16; ++k) mma_f16_ts(d_t, op + k * 8, bd + (uint64_t)(k * 128), idesc_t, k == 0 ? accumulate : 1u);
      };
      Publications<2, kRows> rows;
      if (!kUntied || has_psi) w.wait(&bars->mats_full, 0, 600);
      // The threads only wait for the product they need next (r_full); the dZ product trails it and releases the
      // operand buffer (op_free) when it has read it.
      if (has_psi) {                                           // d alpha_T = G Psi
        if (C::kTiled) {                                       // G is the operand as it came
          w.wait(&bars->g_full, 0, 604);
          const uint64_t gd = make_smem_desc(smem_u32(smem + C::kOffG), 16, 1024);
          const uint64_t bd = mat_desc + (uint64_t)((kUntied ? 4 : 2) * (C::kMatBytes >> 4));
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k) mma_f16_ss(acc, gd + (uint64_t)(k * 2), bd + (uint64_t)(k * 128), idesc_t, k != 0);
            mma_commit(&bars->r_full);
          }
        } else {
          rows.wait();
          tc_fence_after();
          if (elect_one()) {
            mma_tr(acc, 0, kUntied ? 4 : 2, 0u);
            mma_commit(&bars->r_full);
            mma_commit(&bars->op_free[0]);
          }
        }
        __syncwarp();
      }
      for (int t = T - 1; t >= 0; --t) {
        const uint32_t op = rows.n % C::kOps;
        const int li = T - 1 - t, st = li & 1;                 // untied: this layer's stage
        if (kUntied) w.wait(&bars->lm_full[st], (li >> 1) & 1, 602);
        rows.wait();
        tc_fence_after();
        const int sS = kUntied ? 2 * st : 0, sB = kUntied ? 2 * st + 1 : 1;
        if (elect_one()) {
          if (t > 0) {
            mma_tr(acc, op, sS, 0u);                           // dx_t (S_t - I)^T
            mma_commit(&bars->r_full);
          }
          mma_tr(dz, op, sB, t == T - 1 ? 0u : 1u);            // dZ += dx_t B_t^T
          if (t == 0) mma_commit(&bars->r_full);               // the last result the threads wait for is dZ itself
          mma_commit(&bars->op_free[op]);
          if (kUntied && t >= 2) mma_commit(&bars->lm_free[st]);   // the stage is free once these products have read it
        }
        __syncwarp();
        if (kUntied && t >= 2) {
          w.wait(&bars->lm_free[st], (li >> 1) & 1, 603);
          if (__all_sync(0xffffffffu, !w.dead) && elect_one()) load_layer(t - 2);
          __syncwarp();
        }
      }
      if (w.dead && kUntied) {                                 // gave up: let the copies in flight land
        mbar_wait_drain(&bars->lm_full[0], 0);                 // (whichever phase: a bounded wait either way)
        mbar_wait_drain(&bars->lm_full[1], 0);
      }
      if (w.dead && (!kUntied || has_psi)) mbar_wait_drain(&bars->mats_full, 0);
    }
    if (C::kTiled) {                                           // the CTA stays until its copies have landed
      mbar_wait_drain(&bars->g_full, 0);
      mbar_wait_drain(&bars->z_full, 0);
    }
  } else {
    // ---------------------------------------------- one thread per query row ----------------------------------------
    const int row = warp * 32 + lane;
    const int grow = row0 + row;
    const bool live = grow < nq;
    Publications<2, kRows> rows;
    const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
    const uint32_t acc_addr = tbase + C::kColAcc, dz_addr = tbase + C::kColDz;
    const int64_t goff = ((int64_t)bh * nq + (live ? grow : 0)) * D;
    int phase = 0;
    uint32_t n_pub = 0;                           // operands published so far (buffer n_pub % kOps)
    float v[D];                                   // d alpha_{t+1}, then dx_t
    uint8_t* const srow = smem + C::kOffG + row * 128;         // d = 64: this row of G, later of dZ (128-byte swizzle)
    // the operand buffer of the next publication, once its previous operand has been read by the trailing product
    auto next_operand = [&]() -> uint32_t {
      const uint32_t buf = n_pub % C::kOps;
      if (n_pub >= (uint32_t)C::kOps) w.wait(&bars->op_free[buf], (n_pub / C::kOps - 1) & 1, 613);
      ++n_pub;
      return tmem_op + ((uint32_t)(warp * 32) << 16) + buf * C::kOpCols;
    };
    auto publish16 = [&](uint32_t op_addr, int c0, __nv_bfloat16* keep) {      // v[c0 .. c0 + 15], with `keep` also to global memory
      uint32_t pk[8];
#pragma unroll
      for (int e = 0; e < 16; e += 2) pk[e >> 1] = pack_bf16(v[c0 + e], v[c0 + e + 1]);
      tmem_st_32x32b_x8(op_addr + c0 / 2, pk);
      if (keep != nullptr) {
        uint4* kp = reinterpret_cast<uint4*>(keep + c0);
        kp[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        kp[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
      }
    };
    auto published = [&]() {
      tmem_wait_st();
      tc_fence_before();
      rows.publish(w.dead);
    };
    if (C::kTiled) w.wait(&bars->g_full, 0, 615);
    {                                             // v := the row of the output gradient (0 beyond n_q)
      const uint4* p = reinterpret_cast<const uint4*>(G + goff);
#pragma unroll
      for (int c = 0; c < D / 8; ++c) {
        uint4 q;
        if (C::kTiled) q = *reinterpret_cast<const uint4*>(srow + ((c ^ (row & 7)) << 4));
        else q = live ? p[c] : make_uint4(0, 0, 0, 0);
        v[8 * c + 0] = bf16_lo(q.x); v[8 * c + 1] = bf16_hi(q.x);
        v[8 * c + 2] = bf16_lo(q.y); v[8 * c + 3] = bf16_hi(q.y);
        v[8 * c + 4] = bf16_lo(q.z); v[8 * c + 5] = bf16_hi(q.z);
        v[8 * c + 6] = bf16_lo(q.w); v[8 * c + 7] = bf16_hi(q.w);
      }
    }
    if (T > 0) {
      if (has_psi) {
        if (!C::kTiled) {
          const uint32_t op = next_operand();
#pragma unroll
          for (int c0 = 0; c0 < D; c0 += 16) publish16(op, c0, nullptr);      // G is bf16 already: nothing is lost
          published();
        }
        w.wait(&bars->r_full, phase & 1, 611); ++phase;
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < D; c0 += 16) {
          uint32_t r[16];
          tmem_ld_32x32b_x16(acc_addr + c0, r);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) v[c0 + e] = __uint_as_float(r[e]);          // d alpha_T = G Psi
        }
      }
      // the forward's decisions of layer t: column c is bit 31 - c % 32 of word c / 32 (loaded one layer ahead)
      auto load_masks = [&](int t, uint32_t (&m)[D / 32]) {
        const uint32_t* mp = maskbits + (((int64_t)bh * T + t) * nq + (live ? grow : 0)) * (D / 32);
#pragma unroll
        for (int q = 0; q < D / 32; ++q) m[q] = live ? mp[q] : 0u;
      };
      uint32_t mwd[D / 32];
      load_masks(T - 1, mwd);
      for (int t = T - 1; t >= 0; --t) {
        // d alpha_{t+1} = dx_{t+1} + dx_{t+1} (S - I)^T, then dx_t = d alpha_{t+1} o mask_t, 16 columns at a time with the next
        // ones' load in flight
        __nv_bfloat16* keep = dx_out != nullptr && live && !w.dead ? dx_out + (int64_t)t * dx_slot + goff : nullptr;
        auto mask16 = [&](int c0) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int c = c0 + e;
            v[c] = ((mwd[c >> 5] >> (31 - (c & 31))) & 1u) ? v[c] : 0.f;
          }
        };
        uint32_t op;
        if (t == T - 1) {
          op = next_operand();
#pragma unroll
          for (int c0 = 0; c0 < D; c0 += 16) { mask16(c0); publish16(op, c0, keep); }
        } else {
          w.wait(&bars->r_full, phase & 1, 612); ++phase;
          tc_fence_after();
          uint32_t r0[16], r1[16];
          tmem_ld_32x32b_x16(acc_addr, r0);
          op = next_operand();
          auto piece = [&](const uint32_t (&r)[16], int c0) {
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const float2 x = __fadd2_rn(make_float2(v[c0 + e], v[c0 + e + 1]), make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])));
              v[c0 + e] = x.x;
              v[c0 + e + 1] = x.y;
            }
            mask16(c0);
            publish16(op, c0, keep);
          };
#pragma unroll
          for (int c0 = 0; c0 < D; c0 += 32) {
            tmem_wait_ld();
            tmem_ld_32x32b_x16(acc_addr + c0 + 16, r1);
            piece(r0, c0);
            tmem_wait_ld();
            if (c0 + 32 < D) tmem_ld_32x32b_x16(acc_addr + c0 + 32, r0);
            piece(r1, c0 + 16);
          }
        }
        published();
        if (t > 0) load_masks(t - 1, mwd);
      }
      w.wait(&bars->r_full, phase & 1, 614); ++phase;           // the last result is dZ itself
      tc_fence_after();
    }
    // ---- dZ (the accumulated products; G itself without a decoder) and D = <dZ, Z> ----
    float dsum = 0.f;
    const uint4* zp = reinterpret_cast<const uint4*>(Z16 + goff);
    uint4* out = reinterpret_cast<uint4*>(dZ16 + goff);
    if (C::kTiled) w.wait(&bars->z_full, 0, 616);
#pragma unroll
    for (int c0 = 0; c0 < D; c0 += 16) {
      uint32_t r[16];
      if (T > 0) {                                              // uniform over the CTA: every lane takes part
        tmem_ld_32x32b_x16(dz_addr + c0, r);
        tmem_wait_ld();
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(v[c0 + e]);
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint4 z;
        if (C::kTiled) z = *reinterpret_cast<const uint4*>(smem + C::kOffZ + row * 128 + (((c0 / 8 + half) ^ (row & 7)) << 4));
        else z = live ? zp[c0 / 8 + half] : make_uint4(0, 0, 0, 0);
        const float* f = reinterpret_cast<const float*>(r) + 8 * half;
        dsum = fmaf(f[0], bf16_lo(z.x), dsum); dsum = fmaf(f[1], bf16_hi(z.x), dsum);
        dsum = fmaf(f[2], bf16_lo(z.y), dsum); dsum = fmaf(f[3], bf16_hi(z.y), dsum);
        dsum = fmaf(f[4], bf16_lo(z.z), dsum); dsum = fmaf(f[5], bf16_hi(z.z), dsum);
        dsum = fmaf(f[6], bf16_lo(z.w), dsum); dsum = fmaf(f[7], bf16_hi(z.w), dsum);
        const uint4 o = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
        if (C::kTiled) *reinterpret_cast<uint4*>(srow + (((c0 / 8 + half) ^ (row & 7)) << 4)) = o;   // every product has finished
        else if (live && !w.dead) out[c0 / 8 + half] = o;
      }
    }
    if (C::kTiled) {                                            // the warp's rows in one copy (rows beyond n_q are clipped)
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        if (grow < nq && !w.dead && *(volatile int*)&bars->abort == 0) tma_store_3d(&tmap_dz, smem + C::kOffG + warp * 32 * 128, 0, grow, bh);
        bulk_commit_group();
        bulk_wait_group0();
      }
    }
    if (live && !w.dead) negD[(int64_t)bh * ld_pitch + grow] = -dsum;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    tmem_dealloc(tmem, C::kTmemCols);
    if (C::kTmemOpCols != 0) tmem_dealloc(tmem_op, C::kTmemOpCols);
  }
}

// ====================================================================================================================
// dQ
// ====================================================================================================================
// d = 64: chunks of 32 measurements, so that S, dA (one buffer each) and dQ take 128 columns of tensor memory and three tiles of 128
// queries share an SM, where chunks of 64 in two buffers (512 columns allocated) left room for one: 47 -> 38 us for 96 heads of 1568
// queries, m = 256.  Few tiles (kFew): chunks of 64, half as many hand-overs, and two tiles per SM (see launch_sm100_bwd_dq).  d = 128:
// chunks of 64, two buffers, one tile (with chunks of 32 and two tiles per SM 16 heads of 8192, m = 512 take 82 us instead of 79).
template <int D, bool kFew> struct QCfg {
  static_assert(!kFew || D == 64, "built variants");
  static constexpr int kDBoxes = D / 64;
  static constexpr int kQC = D == 64 && !kFew ? 32 : 64;            // measurements per chunk
  static constexpr int kCtas = D == 64 ? (kFew ? 2 : 3) : 1;        // per SM
  static constexpr int kStages = 3, kBufs = D == 64 ? 1 : 2;
  // d = 64: the rows' threads release S_j, dA_j as soon as they are in registers and write dS_j elsewhere (two operand buffers), so that
  // the next chunk's scores are formed under their arithmetic.  With dS_j over S_j a chunk of 32 took 2030 cycles, 1230 of them waits, now
  // 1050: 96 heads of 1568 queries, m = 256 33.3 -> 29.7 us, 4 of 8192, m = 512 (two tiles per SM) 10.0 -> 7.7.
  static constexpr bool kEarly = D == 64;
  static constexpr uint32_t kOpCols = kQC / 2;
  static constexpr uint32_t kTileBoxBytes = kRows * 128;            // 128 rows x 64 columns
  static constexpr uint32_t kTileBytes = kDBoxes * kTileBoxBytes;   // Q tile, dZ tile
  static constexpr uint32_t kBoxBytes = kQC * 128;                  // one 64-column box of a K~ or V~ chunk
  static constexpr uint32_t kSlotBytes = kDBoxes * kBoxBytes;
  static constexpr uint32_t kOffQ = 0, kOffZ = kTileBytes, kOffRing = 2 * kTileBytes;   // ring: [stage][K~ slot | V~ slot]
  static constexpr uint32_t kOffBar = kOffRing + kStages * 2 * kSlotBytes;
  static constexpr uint32_t kSmemBytes = kOffBar + 256;             // base must be 1024-byte aligned (checked)
  // TMEM columns: S[bufs] | dA[bufs] | dQ accumulator; dS_j (bf16) overlays the first half of S[j % bufs]
  static constexpr uint32_t kColS = 0, kColA = kBufs * kQC, kColQ = 2 * kBufs * kQC, kTmemCols = D == 128 ? 512 : kFew ? 256 : 128;
  static constexpr uint32_t kColOp = kColQ + D, kTmemOpCols = kEarly && !kFew ? 32 : 0;   // dS buffers: in an allocation of their own for three CTAs
  static_assert(kColQ + D + (kEarly && !kFew ? 0 : kEarly ? 2 * kOpCols : 0) <= kTmemCols && 2 * kOpCols <= (kTmemOpCols ? kTmemOpCols : 64) &&
                kCtas * (kTmemCols + kTmemOpCols) <= 512, "TMEM budget");
  static_assert(kCtas * (kSmemBytes + 1024) <= 228 * 1024, "CTAs per SM");
  static_assert(kTmemOpCols == 0 || 512 / kTmemCols * (kSmemBytes + 1024) > 228 * 1024,
                "CTAs on one SM must not hold all of tensor memory with their first allocations");
};

struct QBars {
  uint64_t qz_full, full[3], empty[3], s_full[2], p_full[2] /* d = 128 */, acc_done;
  uint32_t tmem_slot, tmem_op_slot;
  int abort;
};

constexpr int kQThreads = 192;      // warps 0-3: one thread per query row; warp 4: TMA; warp 5: MMA issue

template <int D, bool kFew>
__global__ void __launch_bounds__(kQThreads, QCfg<D, kFew>::kCtas)
bwd_dq_sm100_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_z,
                    const __grid_constant__ CUtensorMap tmap_kv, __nv_bfloat16* __restrict__ dQ,
                    const float* __restrict__ negL, const float* __restrict__ negD, int ld_pitch, int nq, int m, float scale, int* status) {
  using C = QCfg<D, kFew>;
  constexpr int kQC = C::kQC;
  extern __shared__ __align__(1024) uint8_t smem[];
  if ((smem_u32(smem) & 1023u) != 0) {          // swizzled tiles need 1024-byte alignment; never seen to fail
    if (threadIdx.x == 0) atomicCAS(status, 0, 700);
    return;
  }
  QBars* bars = reinterpret_cast<QBars*>(smem + C::kOffBar);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y, row0 = blockIdx.x * kRows;
  const int nchunks = (m + kQC - 1) / kQC;
  Waiter w{status, &bars->abort};
  auto k_slot = [&](int s) { return smem + C::kOffRing + (2 * s) * C::kSlotBytes; };
  auto v_slot = [&](int s) { return smem + C::kOffRing + (2 * s + 1) * C::kSlotBytes; };

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmap_q);
    prefetch_tmap(&tmap_z);
    prefetch_tmap(&tmap_kv);
    mbar_init(&bars->qz_full, 1);
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->s_full[b], 1); mbar_init(&bars->p_full[b], kRows); }
    mbar_init(&bars->acc_done, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 5) {
    tmem_alloc(&bars->tmem_slot, C::kTmemCols);
    if (C::kTmemOpCols != 0) tmem_alloc(&bars->tmem_op_slot, C::kTmemOpCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_slot, tmem_op = C::kTmemOpCols != 0 ? bars->tmem_op_slot : tmem + C::kColOp;
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 4) {
    if (elect_one()) {
      mbar_arrive_expect_tx(&bars->qz_full, 2 * C::kTileBytes);
      for (int gx = 0; gx < C::kDBoxes; ++gx) {
        tma_load_3d(smem + C::kOffQ + gx * C::kTileBoxBytes, &tmap_q, &bars->qz_full, gx * 64, row0, bh);
        tma_load_3d(smem + C::kOffZ + gx * C::kTileBoxBytes, &tmap_z, &bars->qz_full, gx * 64, row0, bh);
      }
      int issued = 0;
      for (int j = 0; j < nchunks && !w.dead; ++j) {
        const int s = j % C::kStages;
        if (j >= C::kStages) w.wait(&bars->empty[s], (j / C::kStages - 1) & 1, 701);
        if (w.dead) break;
        mbar_arrive_expect_tx(&bars->full[s], 2 * C::kSlotBytes);
        for (int gx = 0; gx < C::kDBoxes; ++gx) {
          tma_load_3d(k_slot(s) + gx * C::kBoxBytes, &tmap_kv, &bars->full[s], gx * 64, j * kQC, bh);
          tma_load_3d(v_slot(s) + gx * C::kBoxBytes, &tmap_kv, &bars->full[s], D + gx * 64, j * kQC, bh);
        }
        ++issued;
      }
      if (w.dead) {
        mbar_wait_drain(&bars->qz_full, 0);
        for (int i = issued > C::kStages ? issued - C::kStages : 0; i < issued; ++i)
          mbar_wait_drain(&bars->full[i % C::kStages], (i / C::kStages) & 1);
      }
    }
  } else if (warp == 5) {
    // kEarly: the whole warp walks the steps and waits at named barriers; else one lane does, and waits at mbarriers (16 heads of 8192 x
    // 128, m = 512: 70.4 us so, 72.7 the other way)
    if (C::kEarly || elect_one()) {
      constexpr uint32_t idesc_s = make_idesc_bf16(kRows, kQC, false, false);   // S, dA: both operands K-major
      constexpr uint32_t idesc_q = make_idesc_bf16(kRows, D, false, true);      // dQ += dS K~: K~ is MN-major
      auto kstep = [](int k, uint32_t box_bytes) { return (uint64_t)((k / 4) * (box_bytes >> 4) + (k % 4) * 2); };
      auto issue = [&](auto f) {
        tc_fence_after();
        if (!C::kEarly) { f(); return; }
        if (elect_one()) f();
        __syncwarp();
      };
      const uint64_t qd = make_smem_desc(smem_u32(smem + C::kOffQ), 16, 1024);
      const uint64_t zd = make_smem_desc(smem_u32(smem + C::kOffZ), 16, 1024);
      Publications<3, kRows> rows;                // "S_j, dA_j are read" (but for the last j), "dS_j is written"
      auto issue_sd = [&](int j) {
        const int s = j % C::kStages, b = j % C::kBufs;
        w.wait(&bars->full[s], (j / C::kStages) & 1, 711);
        if (C::kEarly && j > 0) rows.wait();
        issue([&]() {
          const uint64_t kd = make_smem_desc(smem_u32(k_slot(s)), 16, 1024);
          const uint64_t vd = make_smem_desc(smem_u32(v_slot(s)), 16, 1024);
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            mma_f16_ss(tmem + C::kColS + b * kQC, qd + kstep(k, C::kTileBoxBytes), kd + kstep(k, C::kBoxBytes), idesc_s, k != 0);
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            mma_f16_ss(tmem + C::kColA + b * kQC, zd + kstep(k, C::kTileBoxBytes), vd + kstep(k, C::kBoxBytes), idesc_s, k != 0);
          mma_commit(&bars->s_full[b]);
        });
      };
      w.wait(&bars->qz_full, 0, 710);
      issue_sd(0);
      for (int j = 0; j < nchunks; ++j) {
        // Two buffers: S_{j+1}, dA_{j+1} run while the threads work on chunk j; they overwrite what the dQ product of chunk j - 1
        // read dS_{j-1} from, which was issued earlier and therefore executes first.  kEarly: they follow the threads' reading of
        // S_j, dA_j; S_j's commit covers the dQ product of chunk j - 2, which read the buffer that dS_j goes to.
        if (j + 1 < nchunks) issue_sd(j + 1);
        const int s = j % C::kStages, b = j & 1;
        if (C::kEarly) rows.wait();
        else w.wait(&bars->p_full[b], (j >> 1) & 1, 712);
        issue([&]() {
          const uint64_t kd = make_smem_desc(smem_u32(k_slot(s)), C::kBoxBytes, 1024);      // MN-major: rows = reduction
#pragma unroll
          for (int k = 0; k < kQC / 16; ++k)
            mma_f16_ts(tmem + C::kColQ, (C::kEarly ? tmem_op + b * C::kOpCols : tmem + C::kColS + b * kQC) + k * 8, kd + (uint64_t)(k * 128),
                       idesc_q, (uint32_t)((j | k) != 0));
          mma_commit(&bars->empty[s]);
          if (j + 1 == nchunks) mma_commit(&bars->acc_done);
        });
      }
    }
  } else {
    const int row = warp * 32 + lane, grow = row0 + row;
    const bool live = grow < nq;
    const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
    // rows beyond n_q: Q and dZ are zero there, and what they form is not stored
    const float nl = live ? negL[(int64_t)bh * ld_pitch + grow] : 0.f, nd = live ? negD[(int64_t)bh * ld_pitch + grow] : 0.f;
    const float2 nl2 = make_float2(nl, nl), nd2 = make_float2(nd, nd);
    const float2 sc2 = make_float2(scale * 1.4426950408889634f, scale * 1.4426950408889634f);
    Publications<3, kRows> rows;
    for (int j = 0; j < nchunks; ++j) {
      const int b = j % C::kBufs;
      w.wait(&bars->s_full[b], (j / C::kBufs) & 1, 720);
      tc_fence_after();
      const uint32_t ds = C::kEarly ? tmem_op + ((uint32_t)(warp * 32) << 16) + (j & 1) * C::kOpCols : tbase + C::kColS + b * kQC;
#pragma unroll
      for (int c0 = 0; c0 < kQC; c0 += 32) {
        uint32_t sv[32], av[32];
        tmem_ld_32x32b_x32(tbase + C::kColS + b * kQC + c0, sv);
        tmem_ld_32x32b_x32(tbase + C::kColA + b * kQC + c0, av);
        tmem_wait_ld();
        if (C::kEarly && c0 + 32 == kQC && j + 1 < nchunks) {
          tc_fence_before();
          rows.publish(w.dead);
        }
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const float2 x = __ffma2_rn(make_float2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), sc2, nl2);
          const float2 g = __fadd2_rn(make_float2(__uint_as_float(av[e]), __uint_as_float(av[e + 1])), nd2);
          const float2 d = __fmul2_rn(make_float2(ex2(x.x), ex2(x.y)), g);
          pk[e >> 1] = pack_bf16(d.x, d.y);
        }
        tmem_st_32x32b_x16(ds + c0 / 2, pk);                  // (d = 128: over scores that have been read)
      }
      tmem_wait_st();
      tc_fence_before();
      if (C::kEarly) rows.publish(w.dead);
      else mbar_arrive(&bars->p_full[j & 1]);
    }
    w.wait(&bars->acc_done, 0, 721);
    tc_fence_after();
    {
      // the tensor-memory loads are warp-wide (every lane takes part); only the stores depend on the row
      const bool store = live && !w.dead && *(volatile int*)&bars->abort == 0;
      uint4* o = reinterpret_cast<uint4*>(dQ + ((int64_t)bh * nq + (live ? grow : 0)) * D);
#pragma unroll
      for (int c0 = 0; c0 < D; c0 += 16) {
        uint32_t r[16];
        tmem_ld_32x32b_x16(tbase + C::kColQ + c0, r);
        tmem_wait_ld();
        float f[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) f[e] = __uint_as_float(r[e]) * scale;
        if (store) {
          o[c0 / 8] = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
          o[c0 / 8 + 1] = make_uint4(pack_bf16(f[8], f[9]), pack_bf16(f[10], f[11]), pack_bf16(f[12], f[13]), pack_bf16(f[14], f[15]));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tmem_dealloc(tmem, C::kTmemCols);
    if (C::kTmemOpCols != 0) tmem_dealloc(tmem_op, C::kTmemOpCols);
  }
}

template <int D, bool kUntied>
cudaError_t launch_recur(csat_ctx* c, const void* G, cudaStream_t s) {
  using C = RCfg<D, kUntied>;
  const Params& p = c->p;
  constexpr uint32_t kMost = D == 64 ? C::kSmemTwo : C::kSmemBytes;
  static DeviceFlags smem_opt_in;
  cudaError_t e = ensure_dynamic_smem(bwd_recur_sm100_kernel<D, kUntied>, (int)kMost, c->device, smem_opt_in);
  if (e != cudaSuccess) return e;
  CUtensorMap tg = c->tmap_mats, tz = tg, td = tg;
  if (C::kTiled) {
    const uint64_t qd[3] = {(uint64_t)D, (uint64_t)p.nq, (uint64_t)(p.B * p.H)};
    const uint64_t qs[2] = {(uint64_t)D * 2, (uint64_t)p.nq * D * 2};
    const uint32_t qb[3] = {64, (uint32_t)kRows, 1}, ob[3] = {64, 32, 1};
    if ((e = make_tmap_bf16_3d(&tg, G, qd, qs, qb)) != cudaSuccess) return e;
    if ((e = make_tmap_bf16_3d(&tz, c->bw_Z16, qd, qs, qb)) != cudaSuccess) return e;
    if ((e = make_tmap_bf16_3d(&td, c->bw_dZ16, qd, qs, ob)) != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)((p.nq + kRows - 1) / kRows), (unsigned)(p.B * p.H));
  // Up to two tiles per SM no three share one: started early, CTAs pile up on the SMs that the kernel before leaves free.  Whole
  // training steps, us, with three per SM / two: 256 tiles, T = 20, m = 512 138 / 123; 128, T = 20, m = 256 86 / 78; 296, T = 5
  // 55.6 / 53.2.  512 tiles 182 either way, 312 with two 7 % slower.
  const uint32_t smem = (int64_t)grid.x * grid.y <= 2 * (int64_t)c->sms ? kMost : C::kSmemBytes;
  return launch_pdl(
      bwd_recur_sm100_kernel<D, kUntied>, grid, kRThreads, smem, s,
      kUntied ? c->tmap_lmats : c->tmap_mats, tg, tz, td, c->bw_Z16, (const __nv_bfloat16*)G, c->bw_dZ16, c->bw_negD(), (int)c->ld_pitch(), c->bw_maskbits, (int)p.nq, (int)p.H, p.T,
      c->psi ? 1 : 0, c->status, c->weight_grads ? c->bw_dx16 : nullptr, (int64_t)(p.B * p.H * p.nq * p.d));
}

template <int D, bool kFew = false>
cudaError_t launch_dq(csat_ctx* c, const void* Q, void* dQ, cudaStream_t s) {
  using C = QCfg<D, kFew>;
  const Params& p = c->p;
  CUtensorMap tq, tz;
  const uint64_t qd[3] = {(uint64_t)D, (uint64_t)p.nq, (uint64_t)(p.B * p.H)};
  const uint64_t qs[2] = {(uint64_t)D * 2, (uint64_t)p.nq * D * 2};
  const uint32_t qb[3] = {64, (uint32_t)kRows, 1};
  cudaError_t e;
  if ((e = make_tmap_bf16_3d(&tq, Q, qd, qs, qb)) != cudaSuccess) return e;
  if ((e = make_tmap_bf16_3d(&tz, c->bw_dZ16, qd, qs, qb)) != cudaSuccess) return e;
  static DeviceFlags smem_opt_in;
  if ((e = ensure_dynamic_smem(bwd_dq_sm100_kernel<D, kFew>, (int)C::kSmemBytes, c->device, smem_opt_in)) != cudaSuccess) return e;
  const float scale = (float)(p.scale > 0.0 ? p.scale : 1.0 / sqrt((double)D));
  const dim3 grid((unsigned)((p.nq + kRows - 1) / kRows), (unsigned)(p.B * p.H));
  return launch_pdl(bwd_dq_sm100_kernel<D, kFew>, grid, kQThreads, C::kSmemBytes, s, tq, tz, C::kQC == 32 ? c->tmap_kv32 : c->tmap_kv, (__nv_bfloat16*)dQ, c->bw_LD, c->bw_negD(),
                    (int)c->ld_pitch(), (int)p.nq, (int)p.m, scale, c->status);
}

}  // namespace

cudaError_t launch_sm100_bwd_recur(csat_ctx* c, const void* G, cudaStream_t s, int* launches) {
  *launches += 1;
  if (c->w_S && c->w_untied && c->p.T > 0)
    return c->p.d == 64 ? launch_recur<64, true>(c, G, s) : launch_recur<128, true>(c, G, s);
  if (c->p.d == 64) return launch_recur<64, false>(c, G, s);
  return c->p.T > 0 ? launch_sm100_bwd_recur_pair(c, G, s) : launch_recur<128, false>(c, G, s);
}

cudaError_t launch_sm100_bwd_dq(csat_ctx* c, const void* Q, void* dQ, cudaStream_t s, int* launches) {
  *launches += 1;
  if (c->p.d == 128) return launch_dq<128>(c, Q, dQ, s);
  // Two tiles per SM where that takes as many rounds as three.  Whole training steps, us, chunks of 64 and two per SM / of 32 and three:
  // 128 tiles, m = 512 66.5 / 74.7, m = 256 77.5 / 83.2; 256, m = 512 120 / 126; 512, m = 512 183 / 190; 592, m = 128 87.4 / 89.7;
  // 312, m = 256 109.7 / 107.7; 624, m = 256 174 / 171; 1248, m = 256 273 / 269.  The same bits.
  const int64_t tiles = (c->p.nq + kRows - 1) / kRows * c->p.B * c->p.H;
  return two_tiles_per_sm(tiles, c->sms) ? launch_dq<64, true>(c, Q, dQ, s) : launch_dq<64>(c, Q, dQ, s);
}

}  // namespace csat

// The bf16 path of head sizes that have no tcgen05 kernel (multiples of 8 up to 120, not 64): compression, attention and
// recovery on the warp-level matrix instructions (warp_mma.cuh), 16 rows per warp.
//
// Q, K~, V~, K, V and Phi are bf16, so their products are exact and only the float32 accumulation rounds.  What the path
// holds in float32 stays in float32 and enters a product as two bf16 parts, hi = bf16(x) and lo = bf16(x - hi), which carry
// 16 bits: P V~ is two products, z B and alpha (S - I) are three (lo lo, 2^-18, is left out); the identity part of S is
// added in float32.  The error against 64 bits is that of the bf16 output and K~|V~: over 80 jobs (d = 8, 24, ... 120, T = 1 to
// 20, with and without a dictionary) it is 0.0034 to 0.0075 of the norm, and between 0.9990 and 1.0004 times (median 1.0000) that of
// float32 arithmetic throughout.  Rows that are not finite are computed in float32 (plain_row).
//
// Bound: the matrix instructions (about 1000 multiply-adds per clock and SM, 340 for the three-part products), against
// ~80 of the float32 kernels this path ran on (ffma_forward.cu).  Larger jobs and heads go to tcgen05 (split_tile_sm100.cu,
// compress_sm100.cu); one S_t, B_t per layer, d > 96, few or short rows and a shard's partial sums stay here.
#include "csat_internal.h"
#include "split_math.cuh"
#include "sm100_ptx.cuh"
#include "warp_mma.cuh"

namespace csat {
namespace {

using namespace wmma16;
using namespace splitmath;

// ---------------------------------------------------------------------------------------------
// K~|V~[b,h,r,:] = sum_j Phi[h,r,j] [K|V][b,h,j,:].  A CTA owns 32 measurements x the DP columns of K~ or of V~; its warps
// share out the tokens in chunks of 32 (each stages its own, one ahead) and their float32 sums are added in warp order.
// ---------------------------------------------------------------------------------------------
constexpr int kCW = 8, kCRows = 32, kCK = 32;
template <int DP> struct CmpSmem {                             // in bf16
  static constexpr int kLdA = kCK + 8, kLdB = DP + 8;
  static constexpr int kStage = kCRows * kLdA + kCK * kLdB;
  static constexpr int kWarp = 2 * kStage;
  static constexpr int kBytes = kCW * kWarp * 2;
  static_assert(kCRows * DP * 4 <= kWarp * 2, "a warp's sums fit where its chunks were");
};

template <typename TO, int DP>
__global__ void __launch_bounds__(kCW * 32) split_compress_kernel(TO* __restrict__ kv, const __nv_bfloat16* __restrict__ phi,
                                                                  const __nv_bfloat16* __restrict__ K, const __nv_bfloat16* __restrict__ V,
                                                                  int64_t n, int64_t n_pad, int64_t m, int d, int H, int phi_v_head0,
                                                                  int64_t phi_j0) {
  using C = CmpSmem<DP>;
  constexpr int NT = DP / 8;
  extern __shared__ __align__(16) __nv_bfloat16 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int bh = blockIdx.y, h = bh % H, is_v = blockIdx.z;
  const int64_t r0 = (int64_t)blockIdx.x * kCRows;
  const __nv_bfloat16* ph = phi + (int64_t)((is_v ? phi_v_head0 : 0) + h) * m * n_pad + phi_j0;
  const __nv_bfloat16* src = (is_v ? V : K) + (int64_t)bh * n * d;
  __nv_bfloat16* mine = smem + warp * C::kWarp;
  auto stage = [&](int64_t j0, int st) {
    __nv_bfloat16 *As = mine + st * C::kStage, *Bs = As + kCRows * C::kLdA;
    for (int i = lane; i < kCRows * (kCK / 8); i += 32) {
      const int r = i / (kCK / 8), k = (i % (kCK / 8)) * 8;
      // Phi's rows are padded to whole pieces; a piece that ends beyond the tokens meets rows of K, V that are zero here
      const bool in = r0 + r < m && j0 + k < n;
      cp16(As + r * C::kLdA + k, ph + (in ? (r0 + r) * n_pad + j0 + k : 0), in);
    }
    for (int i = lane; i < kCK * NT; i += 32) {
      const int k = i / NT, c = (i - k * NT) * 8;
      const bool in = j0 + k < n && c < d;
      cp16(Bs + k * C::kLdB + c, src + (in ? (j0 + k) * d + c : 0), in);
    }
    cp_commit();
  };
  float acc[2][NT][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
  ptx::pdl_wait();
  ptx::pdl_launch_dependents();
  int64_t j0 = (int64_t)warp * kCK;
  if (j0 < n) stage(j0, 0);
  for (int st = 0; j0 < n; j0 += kCW * kCK, st ^= 1) {
    if (j0 + kCW * kCK < n) { stage(j0 + kCW * kCK, st ^ 1); cp_wait<1>(); } else cp_wait<0>();
    __syncwarp();
    const __nv_bfloat16 *As = mine + st * C::kStage, *Bs = As + kCRows * C::kLdA;
    if (j0 + kCK > n) {                                        // another shard's columns of Phi must not meet 0 * inf
      __nv_bfloat16* A = mine + st * C::kStage;
      for (int i = lane; i < kCRows * kCK; i += 32)
        if (j0 + i % kCK >= n) A[(i / kCK) * C::kLdA + i % kCK] = __float2bfloat16_rn(0.f);
      __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < kCK / 16; ++k) {
      uint32_t a[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)                              // rows 16 i .., columns 16 k ..
        ldsm4(a[i], As + (16 * i + (lane & 15)) * C::kLdA + 16 * k + (lane >> 4) * 8);
#pragma unroll
      for (int j = 0; j < NT; j += 2) {
        uint32_t b[4];
        ldsm4t(b, Bs + (16 * k + (lane & 15)) * C::kLdB + 8 * j + (lane >> 4) * 8);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mma(acc[i][j], a[i], b[0], b[1]);
          mma(acc[i][j + 1], a[i], b[2], b[3]);
        }
      }
    }
    __syncwarp();                                              // before the buffer is staged again
  }
  float* sums = reinterpret_cast<float*>(mine);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        *reinterpret_cast<float2*>(sums + (16 * i + g + 8 * u) * DP + 8 * j + 2 * t) = make_float2(acc[i][j][2 * u], acc[i][j][2 * u + 1]);
  __syncthreads();
  for (int i = threadIdx.x * 2; i < kCRows * DP; i += kCW * 32 * 2) {
    const int r = i / DP, c = i % DP;
    if (r0 + r >= m || c >= d) continue;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kCW; ++w) {
      const float2 x = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(smem + w * C::kWarp) + i);
      s.x += x.x; s.y += x.y;
    }
    TO* o = kv + ((int64_t)bh * m + r0 + r) * 2 * d + (is_v ? d : 0) + c;
    if constexpr (sizeof(TO) == 2) *reinterpret_cast<uint32_t*>(o) = pack(s.x, s.y);
    else *reinterpret_cast<float2*>(o) = s;
  }
}

// ---------------------------------------------------------------------------------------------
// Attention and recovery, 64 queries per CTA
// ---------------------------------------------------------------------------------------------
constexpr int kW = 4, kRows = 16 * kW, kMC = 64;
template <int DP> struct AttSmem {
  static constexpr int kLd = DP + 8;
  static constexpr int kTile = kMC * kLd;                      // bf16: K~ or V~ chunk
  static constexpr int kMat = 2 * 2 * kTile * 2;               // byte offset of the matrix fragments
  static constexpr int kBytes = kMat + DP * DP * 4;            // hi and lo
};

template <int DP, bool kUntied>                             // kUntied: one S_t, B_t per layer
__global__ void __launch_bounds__(kW * 32) split_attend_kernel(__nv_bfloat16* __restrict__ out, const __nv_bfloat16* __restrict__ Q,
                                                               const __nv_bfloat16* __restrict__ kv, const __grid_constant__ FfmaAttend p, int tiles) {
  using L = AttSmem<DP>;
  constexpr int NT = DP / 8, KS = DP / 16, kLd = L::kLd;
  extern __shared__ __align__(16) __nv_bfloat16 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int bh = blockIdx.x / tiles, h = bh % p.H, d = p.d, m = (int)p.m, nq = (int)p.nq;
  const int row0 = (blockIdx.x % tiles) * kRows + warp * 16;
  const bool live = row0 < nq;
  const __nv_bfloat16* kvb = kv + (int64_t)bh * m * 2 * d;
  const int nchunks = (m + kMC - 1) / kMC;
  uint4* frag = reinterpret_cast<uint4*>(reinterpret_cast<char*>(smem) + L::kMat);
  const int64_t hdd = (int64_t)h * d * d;

  // The operand fragments of a d x d float32 matrix, tile (k, j) at frag[(k NT + j) 32 + lane]: {hi, hi, lo, lo} of rows
  // 16 k + {2 t, 2 t + 1} and {2 t + 8, 2 t + 9}, column 8 j + g; row r, column c at W[r rs + c cs], the identity taken off
  // the diagonal if asked for.  By all threads, between barriers.
  auto build = [&](const float* W, int rs, int cs, bool less_identity) {
#pragma unroll 6
    for (int i = warp; i < KS * NT; i += kW) {                 // unrolled for the loads in flight
      const int k0 = (i / NT) * 16 + 2 * t, c = (i % NT) * 8 + g;
      float w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = k0 + (e & 1) + (e >> 1) * 8;
        w[e] = r < d && c < d ? W[(int64_t)r * rs + (int64_t)c * cs] - (less_identity && r == c ? 1.f : 0.f) : 0.f;
      }
      uint4 f;
      split2(w[0], w[1], f.x, f.z);
      split2(w[2], w[3], f.y, f.w);
      frag[i * 32 + lane] = f;
    }
  };
  // acc += x W, three parts
  auto times = [&](float (&acc)[NT][4], const float (&x)[NT][4]) {
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      if (16 * k >= d) break;
      uint32_t hi[4], lo[4];
      split2(x[2 * k][0], x[2 * k][1], hi[0], lo[0]);
      split2(x[2 * k][2], x[2 * k][3], hi[1], lo[1]);
      split2(x[2 * k + 1][0], x[2 * k + 1][1], hi[2], lo[2]);
      split2(x[2 * k + 1][2], x[2 * k + 1][3], hi[3], lo[3]);
#pragma unroll
      for (int j = 0; j < NT; j += 4) {
        uint4 b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = frag[(k * NT + j + u) * 32 + lane];
#pragma unroll
        for (int u = 0; u < 4; ++u) mma(acc[j + u], hi, b[u].x, b[u].y);
#pragma unroll
        for (int u = 0; u < 4; ++u) mma(acc[j + u], lo, b[u].x, b[u].y);
#pragma unroll
        for (int u = 0; u < 4; ++u) mma(acc[j + u], hi, b[u].z, b[u].w);
      }
    }
  };

  auto stage = [&](int j) {
    __nv_bfloat16* dst = smem + (j & 1) * 2 * L::kTile;
    for (int i = threadIdx.x; i < kMC * 2 * NT; i += kW * 32) {
      const int r = i / (2 * NT), c = i - r * (2 * NT), is_v = c >= NT, cc = (c - (is_v ? NT : 0)) * 8;
      const bool in = j * kMC + r < m && cc < d;
      cp16(dst + is_v * L::kTile + r * kLd + cc, kvb + (in ? (int64_t)(j * kMC + r) * 2 * d + (is_v ? d : 0) + cc : 0), in);
    }
    cp_commit();
  };
  // B was complete before this call's own compression started; another kernel in front may be the decoder set-up that writes it
  if (p.wait_first) ptx::pdl_wait();
  if (p.T > 0) build(p.B + hdd, d, 1, false);
  ptx::pdl_wait();                                             // K~|V~ come from the kernel before this one
  ptx::pdl_launch_dependents();
  stage(0);
  uint32_t q[KS][4];
  {
    const __nv_bfloat16* Qb = Q + ((int64_t)bh * nq + row0) * d + 2 * t;
    const bool in0 = row0 + g < nq, in1 = row0 + g + 8 < nq;
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const bool c = 16 * k + 8 * u < d;
        q[k][2 * u] = in0 && c ? *reinterpret_cast<const uint32_t*>(Qb + g * d + 16 * k + 8 * u) : 0u;
        q[k][2 * u + 1] = in1 && c ? *reinterpret_cast<const uint32_t*>(Qb + (g + 8) * d + 16 * k + 8 * u) : 0u;
      }
  }
  float z[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) z[j][e] = 0.f;
  float ref[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};
  const float scale_log2 = p.scale * 1.4426950408889634f;
  for (int c = 0; c < nchunks; ++c) {
    if (c + 1 < nchunks) { stage(c + 1); cp_wait<1>(); } else cp_wait<0>();
    __syncthreads();
    if (live) {
      const __nv_bfloat16* Ks = smem + (c & 1) * 2 * L::kTile;
      const __nv_bfloat16* Vs = Ks + L::kTile;
      float s[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
#pragma unroll
        for (int e = 0; e < 4; ++e) s[j][e] = 0.f;
#pragma unroll
        for (int k = 0; k < KS / 2; ++k) {
          uint32_t b[4];
          ldsm4(b, Ks + (8 * j + (lane & 7)) * kLd + 32 * k + (lane >> 3) * 8);
          mma(s[j], q[2 * k], b[0], b[1]);
          mma(s[j], q[2 * k + 1], b[2], b[3]);
        }
      }
      if ((c + 1) * kMC > m)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (c * kMC + 8 * j + 2 * t + (e & 1) >= m) s[j][e] = -INFINITY;
      uint32_t hi[kMC / 16][4], lo[kMC / 16][4];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 8; ++j) mx = fmaxf(mx, fmaxf(s[j][2 * u], s[j][2 * u + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float nref = fmaxf(ref[u], mx * scale_log2);
        const float f = ex2(ref[u] - nref);
        ref[u] = nref;
        float ps = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float p0 = ex2(fmaf(s[j][2 * u], scale_log2, -nref)), p1 = ex2(fmaf(s[j][2 * u + 1], scale_log2, -nref));
          ps += p0 + p1;
          split2(p0, p1, hi[j >> 1][(j & 1) * 2 + u], lo[j >> 1][(j & 1) * 2 + u]);
        }
        sum[u] = fmaf(sum[u], f, ps);
#pragma unroll
        for (int j = 0; j < NT; ++j) { z[j][2 * u] *= f; z[j][2 * u + 1] *= f; }
      }
#pragma unroll
      for (int k = 0; k < kMC / 16; ++k)
#pragma unroll
        for (int j = 0; j < NT; j += 2) {
          uint32_t b[4];
          ldsm4t(b, Vs + (16 * k + (lane & 15)) * kLd + 8 * j + (lane >> 4) * 8);
          mma(z[j], hi[k], b[0], b[1]);
          mma(z[j + 1], hi[k], b[2], b[3]);
          mma(z[j], lo[k], b[0], b[1]);
          mma(z[j + 1], lo[k], b[2], b[3]);
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], 1);
    sum[u] += __shfl_xor_sync(0xffffffffu, sum[u], 2);
    const float inv = 1.f / sum[u];
#pragma unroll
    for (int j = 0; j < NT; ++j) { z[j][2 * u] *= inv; z[j][2 * u + 1] *= inv; }
  }

  // all warps stay for the barriers around the matrices; those without rows only help to build them
  float a[NT][4];
  if (p.T > 0) {
    float c[NT][4];
    auto clear = [&](float (&x)[NT][4]) {
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[j][e] = 0.f;
    };
    auto shrink = [&](const float (&x)[NT][4], float th) {
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[j][e] = x[j][e] - fminf(fmaxf(x[j][e], -th), th);
    };
    clear(c);
    if (live) times(c, z);
    shrink(c, p.theta[h]);                                     // alpha^1 = eta(0 S + z B)
    for (int it = 1; it < p.T; ++it) {
      const float th = p.theta[(int64_t)it * p.theta_stride + h];
      if (kUntied) {
        __syncthreads();
        build(p.B + it * p.layer_stride + hdd, d, 1, false);
        __syncthreads();
        clear(c);
        if (live) times(c, z);
      }
      if (kUntied || it == 1) {
        __syncthreads();
        build(p.S + it * p.layer_stride + hdd, d, 1, true);
        __syncthreads();
      }
      if (live) {
        float x[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) x[j][e] = c[j][e] + a[j][e];
        times(x, a);
        shrink(x, th);
      }
    }
    if (p.psi) {                                               // out_c = sum_k alpha_k Psi[c][k]
      __syncthreads();
      build(p.psi + hdd, 1, d, false);
      __syncthreads();
      clear(c);
      if (live) times(c, a);
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[j][e] = c[j][e];
    }
  } else {
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) a[j][e] = z[j][e];
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int row = row0 + g + 8 * u;
    __nv_bfloat16* o = out + ((int64_t)bh * nq + row) * d + 2 * t;
    bool finite = true;
#pragma unroll
    for (int j = 0; j < NT; ++j)
      if (8 * j < d) {
        finite = finite && fabsf(a[j][2 * u]) < INFINITY && fabsf(a[j][2 * u + 1]) < INFINITY;
        if (row < nq) *reinterpret_cast<uint32_t*>(o + 8 * j) = pack(a[j][2 * u], a[j][2 * u + 1]);
      }
    uint32_t odd = __ballot_sync(0xffffffffu, !finite && row < nq);            // four lanes per row
    for (odd = (odd | odd >> 1 | odd >> 2 | odd >> 3) & 0x11111111u; odd != 0; odd &= odd - 1) {
      const int64_t at = ((int64_t)bh * nq + row0 + 8 * u + ((__ffs(odd) - 1) >> 2)) * d;
      __syncwarp();                                            // after the stores above
      plain_row(out + at, Q + at, kvb, p, hdd);
    }
  }
}

template <typename TO, int DP>
cudaError_t launch_compress(csat_ctx* c, TO* dst, const void* K, const void* V, cudaStream_t s, int64_t phi_j0, int64_t n_len) {
  const Params& p = c->p;
  static DeviceFlags opt_in;
  cudaError_t e = ensure_dynamic_smem(split_compress_kernel<TO, DP>, CmpSmem<DP>::kBytes, c->device, opt_in);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((p.m + kCRows - 1) / kCRows), (unsigned)(p.B * p.H), 2);
  return launch_maybe_pdl(small_grid(grid, c->sms), split_compress_kernel<TO, DP>, grid, kCW * 32, CmpSmem<DP>::kBytes, s, dst, (const __nv_bfloat16*)c->phi,
                    (const __nv_bfloat16*)K, (const __nv_bfloat16*)V, n_len, p.n_pad, p.m, (int)p.d, (int)p.H,
                    p.separate_phi ? (int)p.H : 0, phi_j0);
}

template <typename TO>
cudaError_t compress_t(csat_ctx* c, TO* dst, const void* K, const void* V, cudaStream_t s, int64_t phi_j0, int64_t n_len) {
  if (c->p.d <= 32) return launch_compress<TO, 32>(c, dst, K, V, s, phi_j0, n_len);
  if constexpr (sizeof(TO) == 4) {                            // whole launches of larger heads: compress_sm100.cu
    if (c->p.d > 96) return launch_compress<TO, 128>(c, dst, K, V, s, phi_j0, n_len);
    if (c->p.d > 64) return launch_compress<TO, 96>(c, dst, K, V, s, phi_j0, n_len);
  } else if (c->p.d > 64) {
    return cudaErrorInvalidValue;
  }
  return launch_compress<TO, 64>(c, dst, K, V, s, phi_j0, n_len);
}

template <int DP, bool kUntied> cudaError_t launch_attend(const FfmaAttend& a, const void* Q, const void* kv, void* out, cudaStream_t s) {
  static DeviceFlags opt_in;
  cudaError_t e = ensure_dynamic_smem(split_attend_kernel<DP, kUntied>, AttSmem<DP>::kBytes, a.device, opt_in);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.nq + kRows - 1) / kRows;
  if (tiles * a.BH > (int64_t)1 << 30) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)(tiles * a.BH));
  return launch_maybe_pdl(small_grid(grid, a.sms), split_attend_kernel<DP, kUntied>, grid, kW * 32, AttSmem<DP>::kBytes, s,
                    (__nv_bfloat16*)out, (const __nv_bfloat16*)Q, (const __nv_bfloat16*)kv, a, (int)tiles);
}
template <int DP> cudaError_t attend_d(const FfmaAttend& a, const void* Q, const void* kv, void* out, cudaStream_t s) {
  if constexpr (DP == 96) return launch_attend<DP, true>(a, Q, kv, out, s);      // one S, B: split_tile_sm100.cu
  return a.layer_stride != 0 ? launch_attend<DP, true>(a, Q, kv, out, s) : launch_attend<DP, false>(a, Q, kv, out, s);
}

}  // namespace

// Whole launches: these kernels or compress_sm100.cu's, us: d > 64 4.9 / 3.8 (4 heads of 128 x 96, m = 96) to 18.8 / 7.0: always the latter.  Up to
// 64, by CTAs x tokens: 16 x 200 3.0 / 4.6, 192 x 300 5.1 / 6.3, 256 x 256 4.4 / 6.0; beyond, by what bounds each: the tiles a stage of 64
// tokens, 0.28 us with one batch element and 0.42 with two per CTA (half as much again where rows do not start on 32 bytes), and whole
// rounds of them beyond a tile per SM; these kernels a CTA's walk over the tokens, or the matrix pipes.  16 heads of 1715 x 40, m = 113 11.7
// / 22.9, 12 of 2762 x 24, m = 289 18.0 / 32.4, 36 of 1753 x 8, m = 111 10.9 / 17.8; 27 of 3134 x 48, m = 272 50.5 / 25.9, 176 of 3576 x 32, m = 384 259
// / 52.  Of 79 drawn shapes (d = 8 to 56, 64 to 4000 tokens) the rule takes the slower one once, by 2 %; CTAs x tokens alone did 25 times.
bool split_compress_better(const csat_ctx* c) {
  const Params& p = c->p;
  if (p.d > 64) return false;
  const int64_t ctas = (p.m + kCRows - 1) / kCRows * p.B * p.H * 2;
  if (ctas * p.n <= 72000) return true;
  const bool two = p.B >= 2 && !p.separate_phi;
  const int64_t tiles = (p.m + 127) / 128 * (two ? (p.B + 1) / 2 : p.B) * p.H;
  const double stage = (two ? 420.0 : 280.0) * (p.d % 16 != 0 ? 1.5 : 1.0), rounds = tiles > c->sms ? (double)tiles / c->sms : 1.0;
  const double token = p.d <= 32 ? (0.028 * ctas > 2.9 ? 0.028 * ctas : 2.9) : (0.034 * ctas > 4.2 ? 0.034 * ctas : 4.2);
  return (double)p.n * token < (double)((p.n + 63) / 64) * stage * rounds;             // ns
}

cudaError_t launch_split_compress(csat_ctx* c, const void* K, const void* V, cudaStream_t s, int64_t phi_j0, int64_t n_len, float* partial) {
  return partial ? compress_t<float>(c, partial, K, V, s, phi_j0, n_len)
                 : compress_t<__nv_bfloat16>(c, (__nv_bfloat16*)c->kv, K, V, s, phi_j0, n_len);
}

cudaError_t launch_split_attend(const FfmaAttend& a, const void* Q, const void* kv, void* out, cudaStream_t s) {
  if (a.d <= 32) return attend_d<32>(a, Q, kv, out, s);
  if (a.d <= 64) return attend_d<64>(a, Q, kv, out, s);
  if (a.d <= 96) return attend_d<96>(a, Q, kv, out, s);
  return attend_d<128>(a, Q, kv, out, s);
}

}  // namespace csat

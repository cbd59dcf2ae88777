// Building blocks of the float32 kernels (forward and backward) for head sizes up to 128: register-tiled products
// whose rows belong to one warp.
//
// A warp owns 4 TR rows; lane l = 8 ty + tx (ty < 4, tx < 8) holds rows ty + 4 i, i < TR.  Because no other warp reads
// a row's operands, the products of the unrolled recurrence need no block-wide barrier between layers, only
// __syncwarp.  Both operands come from shared memory in the layout their source has in global memory:
//   gemm_t : B stored [k][column]   (a product with the rows of a matrix: P V~, alpha S, z B);
//            the lane holds columns 4 tx + 32 q + {0..3}
//   gemm_n : B stored [column][k]   (dot products of rows: Q K~^T, dZ V~^T);
//            the lane holds columns tx + 8 j, every sum split into even and odd k (added up at the end)
// Arithmetic is fma.rn.f32x2: measured on one B200 (outer products out of registers, 16 warps per SM) 101 multiply-adds
// per clock and SM against 83 with the scalar instruction, and half the issue slots, which the operand loads and the
// duplication of A's scalars into pairs then use.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace csat {
namespace ffma {

constexpr int kWarps = 4, kThreads = kWarps * 32;
constexpr int kChunk = 32;                 // measurements (or queries) staged per step
constexpr int kPLd = kChunk + 8;           // row pitch of the probabilities

// Row pitches in floats.  Lanes read 4 different rows of A (pitch = 8 mod 32: the scalar stores of gemm_n's result
// hit 32 different banks, too) and 8 different rows of gemm_n's B (pitch = 4 mod 32) without bank conflicts.
template <int DP> struct Ld {
  static constexpr int kA = DP + 8, kB = DP + 4;
};

__device__ __forceinline__ void cp_async16(void* smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(g));
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T> struct Vec;          // 16 bytes of storage as floats
template <> struct Vec<float> {
  static constexpr int kN = 4;
  __device__ static __forceinline__ void to_float(const uint4& v, float (&f)[4]) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
};
template <> struct Vec<__nv_bfloat16> {
  static constexpr int kN = 8;
  __device__ static __forceinline__ void to_float(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};
__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
__device__ __forceinline__ void store1(float* p, float a) { *p = a; }
__device__ __forceinline__ void store1(__nv_bfloat16* p, float a) { *p = __float2bfloat16_rn(a); }

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }

// A lane reads TR + TC floats per k for TR TC multiply-adds, and shared memory delivers 128 bytes per clock and SM to the
// lanes, broadcasts included (a 16-byte read of a warp takes 4 cycles whatever the addresses): the products are bound by
// that rate up to TR TC / (TR + TC) = 4, by the FMA pipe beyond.  Hence 8 rows per lane where there are rows enough, and
// matrices of up to 64 x 64 kept in registers (RegMatrix) where one matrix serves many products.
// Operands are read one step ahead of the arithmetic that uses them.

// acc[i][2 q], acc[i][2 q + 1] += sum over k < K of A[ty + 4 i][k] B[k][4 tx + 32 q ..]; K a multiple of 8.
// A points at row ty, B at column 4 tx.
template <int TR, int TCQ>
__device__ __forceinline__ void gemm_t(float2 (&acc)[TR][2 * TCQ], const float* A, int lda, const float* B, int ldb, int K) {
  constexpr int KS = TCQ <= 2 ? 4 : 2;                     // k per step (registers: 2 KS (TR + 4 TCQ))
  float a[2][TR][KS];
  float4 b[2][KS][TCQ];
  auto load = [&](int k, int st) {
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      if (KS == 4) {
        const float4 x = *reinterpret_cast<const float4*>(A + 4 * i * lda + k);
        a[st][i][0] = x.x; a[st][i][1] = x.y; a[st][i][KS - 2] = x.z; a[st][i][KS - 1] = x.w;
      } else {
        const float2 x = *reinterpret_cast<const float2*>(A + 4 * i * lda + k);
        a[st][i][0] = x.x; a[st][i][1] = x.y;
      }
    }
#pragma unroll
    for (int kk = 0; kk < KS; ++kk)
#pragma unroll
      for (int q = 0; q < TCQ; ++q) b[st][kk][q] = *reinterpret_cast<const float4*>(B + (k + kk) * ldb + 32 * q);
  };
  auto work = [&](int st) {
#pragma unroll
    for (int kk = 0; kk < KS; ++kk)
#pragma unroll
      for (int q = 0; q < TCQ; ++q)
#pragma unroll
        for (int i = 0; i < TR; ++i) {
          const float2 a2 = dup(a[st][i][kk]);
          acc[i][2 * q] = __ffma2_rn(a2, make_float2(b[st][kk][q].x, b[st][kk][q].y), acc[i][2 * q]);
          acc[i][2 * q + 1] = __ffma2_rn(a2, make_float2(b[st][kk][q].z, b[st][kk][q].w), acc[i][2 * q + 1]);
        }
  };
  load(0, 0);
#pragma unroll 1
  for (int k = 0; k < K; k += 2 * KS) {
    load(k + KS, 1);
    work(0);
    load(k + 2 * KS < K ? k + 2 * KS : 0, 0);              // the last step's read is not used
    work(1);
  }
}

// acc[i][j] += (sum over even k, sum over odd k) of A[ty + 4 i][k] B[tx + 8 j][k]; K a multiple of 8.
// A points at row ty, B at row tx.
template <int TR, int TC>
__device__ __forceinline__ void gemm_n(float2 (&acc)[TR][TC], const float* A, int lda, const float* B, int ldb, int K) {
  float4 a[2][TR], b[2][TC];
  auto load = [&](int k, int st) {
#pragma unroll
    for (int i = 0; i < TR; ++i) a[st][i] = *reinterpret_cast<const float4*>(A + 4 * i * lda + k);
#pragma unroll
    for (int j = 0; j < TC; ++j) b[st][j] = *reinterpret_cast<const float4*>(B + 8 * j * ldb + k);
  };
  auto work = [&](int st) {
#pragma unroll
    for (int j = 0; j < TC; ++j)
#pragma unroll
      for (int i = 0; i < TR; ++i) {
        acc[i][j] = __ffma2_rn(make_float2(a[st][i].x, a[st][i].y), make_float2(b[st][j].x, b[st][j].y), acc[i][j]);
        acc[i][j] = __ffma2_rn(make_float2(a[st][i].z, a[st][i].w), make_float2(b[st][j].z, b[st][j].w), acc[i][j]);
      }
  };
  load(0, 0);
#pragma unroll 1
  for (int k = 0; k < K; k += 8) {
    load(k + 4, 1);
    work(0);
    load(k + 8 < K ? k + 8 : 0, 0);
    work(1);
  }
}

// A DP x DP matrix W (DP <= 64) in the registers of one warp, for products x W with many rows x, one row at a time.
// Lane (ty, tx) holds W[k][col] for k = 8 u + 2 ty + {0, 1} and col = tx + 8 j, as pairs over k, so that x is read from
// shared memory as it lies (8 bytes per 2 NJ multiply-adds and lane) and no scalar is duplicated; the four ty add up their
// shares by a reduce-scatter, after which the lane holds NC = DP / 32 columns tx + 8 (NC ty' + {0 ..}).  x has to be finite in
// the columns beyond d, also where a row is not: what a product leaves there is not kept (infinity times W's zeros is NaN, and
// would reach every column of the next product).  Kernels do so (kPadded) only where d is less than DP: with a test in every
// case one head of 256 x 64 took 18.7 instead of 15.8 us.
template <int DP> struct RegMatrix {
  static constexpr int NJ = DP / 8, NU = DP / 8, NC = DP / 32;
  float2 w[NU][NJ];
  // W in shared memory, row pitch ld = 4 mod 32; k and columns beyond d are zero
  __device__ __forceinline__ void load(const float* W, int ld, int d, int tx, int ty) {
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int k = 8 * u + 2 * ty, c = tx + 8 * j;
        const bool in = k < d && c < d;                    // d is a multiple of 8: k + 1 < d as well
        w[u][j] = in ? make_float2(W[k * ld + c], W[(k + 1) * ld + c]) : make_float2(0.f, 0.f);
      }
  }
  // W = the transpose of the matrix in shared memory
  __device__ __forceinline__ void load_transposed(const float* W, int ld, int d, int tx, int ty) {
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int k = 8 * u + 2 * ty, c = tx + 8 * j;
        w[u][j] = k < d && c < d ? *reinterpret_cast<const float2*>(W + c * ld + k) : make_float2(0.f, 0.f);
      }
  }
  // the lane's first column after a product
  __device__ static __forceinline__ int col(int tx, int ty) { return tx + 8 * NC * ((ty >> 1) * 2 + (ty & 1)); }
  // N rows at once (x points at row 0, column 2 ty; rows lda apart): y[r][..] = the lane's columns of x_r W
  template <int N> __device__ __forceinline__ void times(float (&y)[N][NC], const float* x, int lda, int ty) const {
    float2 acc[N][NJ];
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[r][j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int r = 0; r < N; ++r) {
        const float2 xv = *reinterpret_cast<const float2*>(x + r * lda + 8 * u);
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[r][j] = __ffma2_rn(xv, w[u][j], acc[r][j]);
      }
#pragma unroll
    for (int r = 0; r < N; ++r) {
      float s[NJ], h[NJ / 2];
#pragma unroll
      for (int j = 0; j < NJ; ++j) s[j] = acc[r][j].x + acc[r][j].y;
      const bool up = ty & 2, odd = ty & 1;
#pragma unroll
      for (int j = 0; j < NJ / 2; ++j) {
        const float got = __shfl_xor_sync(0xffffffffu, up ? s[j] : s[j + NJ / 2], 16);
        h[j] = (up ? s[j + NJ / 2] : s[j]) + got;
      }
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const float got = __shfl_xor_sync(0xffffffffu, odd ? h[j] : h[j + NC], 8);
        y[r][j] = (odd ? h[j + NC] : h[j]) + got;
      }
    }
  }
};

template <int N, int M> __device__ __forceinline__ void clear(float2 (&a)[N][M]) {
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < M; ++j) a[i][j] = make_float2(0.f, 0.f);
}

// the lane's columns of its rows into a warp-private operand buffer (A points at row ty)
template <int TR, int TCQ>
__device__ __forceinline__ void store_rows(float* A, int lda, int tx, const float2 (&v)[TR][2 * TCQ]) {
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int q = 0; q < TCQ; ++q)
      *reinterpret_cast<float4*>(A + 4 * i * lda + 4 * tx + 32 * q) =
          make_float4(v[i][2 * q].x, v[i][2 * q].y, v[i][2 * q + 1].x, v[i][2 * q + 1].y);
}

__device__ __forceinline__ float sum8(float v) {           // over the 8 lanes that share a row
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  return v;
}
__device__ __forceinline__ float max8(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
}

// eta_theta(x) = sign(x) max(|x| - theta, 0)
__device__ __forceinline__ float shrink(float x, float th) { return x - fminf(fmaxf(x, -th), th); }
__device__ __forceinline__ float2 shrink(float2 x, float th) { return make_float2(shrink(x.x, th), shrink(x.y, th)); }

// 4 TR rows of `src` (row pitch d) starting at row r0, of which `rows` exist, into the warp's buffer
template <typename T>
__device__ __forceinline__ void load_own_rows(float* dst, int lda, const T* src, int64_t r0, int64_t rows, int d, int n_rows,
                                              int lane, int64_t src_pitch) {
  constexpr int kN = Vec<T>::kN;
  const int vpr = d / kN;
  for (int i = lane; i < n_rows * vpr; i += 32) {
    const int r = i / vpr, c = (i - r * vpr) * kN;
    float f[kN];
    uint4 v = make_uint4(0, 0, 0, 0);
    if (r0 + r < rows) v = *reinterpret_cast<const uint4*>(src + (r0 + r) * src_pitch + c);
    Vec<T>::to_float(v, f);
#pragma unroll
    for (int u = 0; u < kN; u += 4) *reinterpret_cast<float4*>(dst + r * lda + c + u) = make_float4(f[u], f[u + 1], f[u + 2], f[u + 3]);
  }
}

// rows [k0, k0 + rows) of a d x d float32 matrix into shared memory, row pitch ld, by all threads (cp.async, not waited for)
__device__ __forceinline__ void stage_matrix_async(float* dst, int ld, const float* W, int d, int k0, int rows) {
  const int vpr = d / 4;
  for (int i = threadIdx.x; i < rows * vpr; i += kThreads) {
    const int r = i / vpr, c = (i - r * vpr) * 4;
    cp_async16(dst + r * ld + c, W + (int64_t)(k0 + r) * d + c);
  }
}
// zeroes the columns beyond d (what the products leave there comes from unwritten shared memory)
template <int TR, int TCQ> __device__ __forceinline__ void clear_beyond(float2 (&v)[TR][2 * TCQ], int d, int tx) {
#pragma unroll
  for (int q = 0; q < TCQ; ++q)
    if (4 * tx + 32 * q >= d)
#pragma unroll
      for (int i = 0; i < TR; ++i) v[i][2 * q] = v[i][2 * q + 1] = make_float2(0.f, 0.f);
}

// the lane's columns of its rows from a buffer (A points at row ty)
template <int TR, int TCQ>
__device__ __forceinline__ void load_rows(float2 (&v)[TR][2 * TCQ], const float* A, int lda, int tx) {
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int q = 0; q < TCQ; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(A + 4 * i * lda + 4 * tx + 32 * q);
      v[i][2 * q] = make_float2(x.x, x.y);
      v[i][2 * q + 1] = make_float2(x.z, x.w);
    }
}

// acc += (the rows at A) W for a d x d matrix W in global memory, by all warps of the CTA: W's rows pass through `buf`
// (room for 2 kChunk rows of pitch ldb) a block at a time.  A points at row ty.
template <int TR, int TCQ>
__device__ __forceinline__ void times_matrix(float2 (&acc)[TR][2 * TCQ], const float* A, int lda, const float* W, int d, float* buf, int ldb,
                                             int tx) {
  for (int k0 = 0; k0 < d; k0 += 2 * kChunk) {
    const int rows = d - k0 < 2 * kChunk ? d - k0 : 2 * kChunk;
    __syncthreads();
    stage_matrix_async(buf, ldb, W, d, k0, rows);
    cp_async_wait_all();
    __syncthreads();
    gemm_t<TR, TCQ>(acc, A + k0, lda, buf + 4 * tx, ldb, rows);
  }
}
// dst row r, column a (+)= <the row at A, row a of W>, i.e. (the rows at A) W^T; dst and A point at row ty, and differ
template <int TR>
__device__ __forceinline__ void times_transposed(float* dst, const float* A, int lda, const float* W, int d, float* buf, int ldb, int tx,
                                                 bool add) {
  for (int k0 = 0; k0 < d; k0 += 2 * kChunk) {
    const int rows = d - k0 < 2 * kChunk ? d - k0 : 2 * kChunk;
    __syncthreads();
    stage_matrix_async(buf, ldb, W, d, k0, rows);
    cp_async_wait_all();
    __syncthreads();
    for (int c0 = 0; c0 < rows; c0 += 32) {
      float2 o[TR][4];
#pragma unroll
      for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) o[i][j] = make_float2(0.f, 0.f);
      gemm_n<TR, 4>(o, A, lda, buf + (c0 + tx) * ldb, ldb, d);
#pragma unroll
      for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c0 + tx + 8 * j < rows) {
            float* p = dst + 4 * i * lda + k0 + c0 + tx + 8 * j;
            *p = (add ? *p : 0.f) + (o[i][j].x + o[i][j].y);
          }
    }
  }
  __syncwarp();
}

// A chunk of 32 rows of a matrix pair (two halves of `d` columns each; row r of half u at src[u] + r * pitch) on its way
// through registers: fetch() issues the loads, put() converts and stores them, so that a chunk travels while the
// previous one is worked on.  Rows beyond `rows` are zero.
template <typename T, int DP> struct PairChunk {
  static constexpr int kN = Vec<T>::kN;
  static constexpr int kSteps = (2 * DP / kN + 31) / 32;          // 16-byte pieces per lane and row
  static constexpr int kRowsPerWarp = kChunk / kWarps;
  uint4 v[kRowsPerWarp][kSteps];
  __device__ __forceinline__ void fetch(const T* src0, const T* src1, int64_t pitch, int64_t r0, int64_t rows, int d) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int vpr = d / kN;
#pragma unroll
    for (int rr = 0; rr < kRowsPerWarp; ++rr) {
      const int64_t r = r0 + warp * kRowsPerWarp + rr;
#pragma unroll
      for (int st = 0; st < kSteps; ++st) {
        const int i = lane + 32 * st;
        v[rr][st] = make_uint4(0, 0, 0, 0);
        if (r < rows && i < 2 * vpr)
          v[rr][st] = *reinterpret_cast<const uint4*>(i < vpr ? src0 + r * pitch + i * kN : src1 + r * pitch + (i - vpr) * kN);
      }
    }
  }
  __device__ __forceinline__ void put(float* d0, float* d1, int ld, int d) const {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int vpr = d / kN;
#pragma unroll
    for (int rr = 0; rr < kRowsPerWarp; ++rr) {
      const int r = warp * kRowsPerWarp + rr;
#pragma unroll
      for (int st = 0; st < kSteps; ++st) {
        const int i = lane + 32 * st;
        if (i >= 2 * vpr) continue;
        float f[kN];
        Vec<T>::to_float(v[rr][st], f);
        float* dst = (i < vpr ? d0 + i * kN : d1 + (i - vpr) * kN) + r * ld;
#pragma unroll
        for (int u = 0; u < kN; u += 4) *reinterpret_cast<float4*>(dst + u) = make_float4(f[u], f[u + 1], f[u + 2], f[u + 3]);
      }
    }
  }
};

// Scores, online softmax and Z of the warp's rows against all m measurements (kvb: the (batch, head)'s K~|V~ rows, 2 d
// wide).  z ends unnormalised; run_max and run_sum (complete) are the row's softmax statistics.  Ks, Vs: [32][DP + 4];
// Qw, Pw: the warp's rows, at row ty.
template <typename T, int DP, int TR>
__device__ __forceinline__ void softmax_rows(float2 (&z)[TR][DP / 16], float (&run_max)[TR], float (&run_sum)[TR], float* Ks, float* Vs,
                                             const float* Qw, float* Pw, const T* kvb, int64_t m, int d, float scale) {
  constexpr int kTC = kChunk / 8, kLdB = Ld<DP>::kB;
  const int tx = threadIdx.x & 7;
  clear(z);
#pragma unroll
  for (int i = 0; i < TR; ++i) { run_max[i] = -INFINITY; run_sum[i] = 0.f; }
  PairChunk<T, DP> ch;
  ch.fetch(kvb, kvb + d, 2 * d, 0, m, d);
  for (int64_t r0 = 0; r0 < m; r0 += kChunk) {
    __syncthreads();                                       // the previous chunk has been read
    ch.put(Ks, Vs, kLdB, d);
    __syncthreads();
    if (r0 + kChunk < m) ch.fetch(kvb, kvb + d, 2 * d, r0 + kChunk, m, d);
    float2 s2[TR][kTC];
    clear(s2);
    gemm_n<TR, kTC>(s2, Qw, Ld<DP>::kA, Ks + tx * kLdB, kLdB, d);
    __syncwarp();                                          // the previous chunk's P has been read
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      float s[kTC], mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < kTC; ++j) {
        s[j] = (r0 + tx + 8 * j < m) ? (s2[i][j].x + s2[i][j].y) * scale : -INFINITY;
        mx = fmaxf(mx, s[j]);
      }
      const float new_max = fmaxf(run_max[i], max8(mx));   // finite: measurement r0 always exists
      const float corr = expf(run_max[i] - new_max);       // 0 on the first chunk (run_max = -inf)
      run_max[i] = new_max;
      float ps = 0.f;
#pragma unroll
      for (int j = 0; j < kTC; ++j) {
        const float p = expf(s[j] - new_max);
        ps += p;
        Pw[4 * i * kPLd + tx + 8 * j] = p;
      }
      run_sum[i] = run_sum[i] * corr + ps;                 // this lane's columns
#pragma unroll
      for (int j = 0; j < DP / 16; ++j) z[i][j] = __fmul2_rn(z[i][j], dup(corr));
    }
    __syncwarp();
    gemm_t<TR, DP / 32>(z, Pw, kPLd, Vs + 4 * tx, kLdB, kChunk);
  }
#pragma unroll
  for (int i = 0; i < TR; ++i) run_sum[i] = sum8(run_sum[i]);
}

}  // namespace ffma
}  // namespace csat

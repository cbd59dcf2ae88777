// The float32 attention and recovery of ffma_forward.cu for jobs of few queries (d <= 64, one decoder for all layers): four rows per
// CTA, whose threads share out every step.
//
// Bound: such a job is one chain of waits.  With four rows per warp (ffma_attend_kernel) one head of 256 x 64, m = 64, T = 10 takes
// 27800 cycles: 4000 to the end of the kernel in front, 7300 in the softmax, 5000 in the product with B and in staging B and S, 1080 in
// each layer.  Here nothing is staged: every thread has its share of K~, V~, B and S in registers, requested at the start (the matrices
// before the kernel in front has finished), and only the rows of the operand, one 16-byte word per column, and the probabilities pass
// through shared memory.  That kernel 13.6 -> 6.8 us, the whole call behind others 15.2 -> 8.2 (a replayed graph).
//   scores   : four threads per measurement, a quarter of the head dimension each, summed by shuffles
//   P V~     : a thread per column and quarter of the chunk's measurements
//   products : a warp owns eight columns, its lanes a quarter of k each; one barrier per layer
#include "csat_internal.h"
#include "sm100_ptx.cuh"

namespace csat {
namespace {

constexpr int kR = 4;                                       // rows per CTA
// CTAs that an SM has room for (128 and 120 registers a thread)
constexpr int per_sm(int64_t d) { return d <= 32 ? 4 : 2; }

__device__ __forceinline__ float4 fma4(float4 a, float w, float4 c) {
  return make_float4(fmaf(a.x, w, c.x), fmaf(a.y, w, c.y), fmaf(a.z, w, c.z), fmaf(a.w, w, c.w));
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ float4 max4(float4 a, float4 b) { return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w)); }
__device__ __forceinline__ float4 shfl4(float4 a, int o) {
  return make_float4(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o), __shfl_xor_sync(0xffffffffu, a.z, o),
                     __shfl_xor_sync(0xffffffffu, a.w, o));
}
__device__ __forceinline__ float4 exp4(float4 a, float4 m) { return make_float4(expf(a.x - m.x), expf(a.y - m.y), expf(a.z - m.z), expf(a.w - m.w)); }
__device__ __forceinline__ float4 dup4(float x) { return make_float4(x, x, x, x); }
__device__ __forceinline__ float4 shrink4(float4 x, float th) {
  return make_float4(x.x - fminf(fmaxf(x.x, -th), th), x.y - fminf(fmaxf(x.y, -th), th), x.z - fminf(fmaxf(x.z, -th), th),
                     x.w - fminf(fmaxf(x.w, -th), th));
}

template <int DP>
__global__ void __launch_bounds__(4 * DP, per_sm(DP))
    ffma_small_kernel(float* __restrict__ out, const float* __restrict__ Q, const float* kv, const FfmaAttend p) {
  constexpr int kThreads = 4 * DP, kWarps = kThreads / 32, kMC = DP, kKQ = DP / 4;
  // columns of the operand, the quarters 16 bytes apart in the banks
  auto at = [](int k) { return k + k / kKQ; };
  __shared__ float4 qs[DP + 4], al[2][DP + 4], ps[kMC], part[4][DP], red[kWarps];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bh = blockIdx.y, h = bh % p.H, d = p.d, m = (int)p.m;
  const int64_t row0 = (int64_t)blockIdx.x * kR;
  const int c = warp * 8 + (lane & 7), kq = lane >> 3;      // products: column, quarter of k
  const int64_t hdd = (int64_t)h * d * d;
  if (p.wait_first) ptx::pdl_wait();
  float wS[kKQ], wB[kKQ];
#pragma unroll
  for (int i = 0; i < kKQ; ++i) {
    const int k = kq * kKQ + i;
    const bool in = k < d && c < d;
    wB[i] = in && p.T > 0 ? p.B[hdd + (int64_t)k * d + c] : 0.f;
    wS[i] = in && p.T > 1 ? p.S[hdd + (int64_t)k * d + c] : 0.f;
  }
  if (tid < DP) {
    float q[kR];
#pragma unroll
    for (int i = 0; i < kR; ++i) q[i] = row0 + i < p.nq && tid < d ? Q[((int64_t)bh * p.nq + row0 + i) * d + tid] : 0.f;
    qs[at(tid)] = make_float4(q[0], q[1], q[2], q[3]);
  }
  ptx::pdl_wait();                                          // K~|V~ come from the kernel before this one
  ptx::pdl_launch_dependents();
  const float* kvb = kv + (int64_t)bh * m * 2 * d;
  const int r = tid >> 2, kr = tid & 3;                     // scores: measurement, quarter of the head dimension
  const int vc = tid & (DP - 1), vq = tid / DP;             // P V~: column, quarter of the measurements
  float kreg[kKQ], vreg[kKQ];
  auto fetch_k = [&](int r0) {
#pragma unroll
    for (int i = 0; i < kKQ; i += 4) {
      float4 x = dup4(0.f);
      if (r0 + r < m && kr * kKQ + i < d) x = *reinterpret_cast<const float4*>(kvb + (int64_t)(r0 + r) * 2 * d + kr * kKQ + i);
      kreg[i] = x.x; kreg[i + 1] = x.y; kreg[i + 2] = x.z; kreg[i + 3] = x.w;
    }
  };
  auto fetch_v = [&](int r0) {
#pragma unroll
    for (int i = 0; i < kKQ; ++i) {
      const int rr = r0 + vq * kKQ + i;
      vreg[i] = rr < m && vc < d ? kvb[(int64_t)rr * 2 * d + d + vc] : 0.f;
    }
  };
  fetch_k(0);
  fetch_v(0);
  __syncthreads();
  float4 run_max = dup4(-INFINITY), run_sum = dup4(0.f), z = dup4(0.f);      // run_sum: this thread's measurements (kr = 0)
  for (int r0 = 0; r0 < m; r0 += kMC) {
    float4 s = dup4(0.f);
#pragma unroll
    for (int i = 0; i < kKQ; ++i) s = fma4(qs[kr * (kKQ + 1) + i], kreg[i], s);
    s = add4(s, shfl4(s, 1));
    s = add4(s, shfl4(s, 2));
    s = r0 + r < m ? mul4(s, dup4(p.scale)) : dup4(-INFINITY);
    if (r0 + kMC < m) fetch_k(r0 + kMC);
    float4 mx = s;
#pragma unroll
    for (int o = 4; o < 32; o *= 2) mx = max4(mx, shfl4(mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) mx = max4(mx, red[w]);
    mx = max4(mx, run_max);                                 // finite: measurement r0 exists
    const float4 corr = exp4(run_max, mx), pr = exp4(s, mx);
    run_max = mx;
    if (kr == 0) {
      ps[r] = pr;
      run_sum = add4(mul4(run_sum, corr), pr);
    }
    z = mul4(z, corr);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kKQ; ++i) z = fma4(ps[vq * kKQ + i], vreg[i], z);
    if (r0 + kMC < m) fetch_v(r0 + kMC);
  }
  part[vq][vc] = z;
#pragma unroll
  for (int o = 1; o < 32; o *= 2) run_sum = add4(run_sum, shfl4(run_sum, o));
  if (lane == 0) red[warp] = run_sum;                       // (the last maximum was read before the barrier above)
  __syncthreads();
  if (tid < DP) {
    float4 sum = red[0], v = add4(add4(part[0][tid], part[1][tid]), add4(part[2][tid], part[3][tid]));
#pragma unroll
    for (int w = 1; w < kWarps; ++w) sum = add4(sum, red[w]);
    al[0][at(tid)] = mul4(v, make_float4(1.f / sum.x, 1.f / sum.y, 1.f / sum.z, 1.f / sum.w));
  }
  __syncthreads();
  // the operand's four rows times a matrix: column c, in every lane that has it
  auto product = [&](const float4* x, const float (&w)[kKQ]) {
    float4 y = dup4(0.f);
#pragma unroll
    for (int i = 0; i < kKQ; ++i) y = fma4(x[kq * (kKQ + 1) + i], w[i], y);
    y = add4(y, shfl4(y, 8));
    return add4(y, shfl4(y, 16));
  };
  float4 a;
  if (p.T > 0) {
    const float4 zb = product(al[0], wB);
    // (a column beyond d: infinity times the matrices' padding is NaN, which must not reach the next product)
    a = c < d ? shrink4(zb, p.theta[h]) : dup4(0.f);
    for (int it = 1; it < p.T; ++it) {
      const float th = p.theta[(int64_t)it * p.theta_stride + h];
      if (kq == 0) al[it & 1][at(c)] = a;
      __syncthreads();
      const float4 y = product(al[it & 1], wS);
      a = c < d ? shrink4(add4(y, zb), th) : dup4(0.f);
    }
    if (p.psi) {                                            // out_c = sum_k alpha_k Psi[c][k]
#pragma unroll
      for (int i = 0; i < kKQ; ++i) {
        const int k = kq * kKQ + i;
        wB[i] = k < d && c < d ? p.psi[hdd + (int64_t)c * d + k] : 0.f;
      }
      if (kq == 0) al[p.T & 1][at(c)] = a;
      __syncthreads();
      a = product(al[p.T & 1], wB);
    }
  } else {
    a = al[0][at(c)];
  }
  const float v = kq == 0 ? a.x : kq == 1 ? a.y : kq == 2 ? a.z : a.w;       // each of a column's lanes stores a row
  if (row0 + kq < p.nq && c < d) out[((int64_t)bh * p.nq + row0 + kq) * d + c] = v;
}

template <int DP> cudaError_t launch(const FfmaAttend& a, const float* Q, const float* kv, float* out, cudaStream_t s) {
  const dim3 grid((unsigned)((a.nq + kR - 1) / kR), (unsigned)a.BH);
  // the grid fits the chip at once (ffma_small_better), so early CTAs pile up nowhere: four heads of 256, d = 64, T = 20 16.6 us, 17.8 without
  return launch_pdl(ffma_small_kernel<DP>, grid, 4 * DP, 0, s, out, Q, kv, a);
}

}  // namespace

// While all CTAs fit at once.  The whole call in a replayed graph, here / ffma_attend_kernel (us): d = 64 on 64 CTAs 8.2 / 15.2, 152
// 11.6 / 15.4, 256 with T = 20 16.6 / 21.0; 128 with m = 400 19.6 / 37.4; 32 heads of 8 batches with 4 queries each (256) 148 / 195.
// Attention and recovery alone, every four rows reading all of K~|V~: 16 CTAs with m = 400 13.4 / 30.5, m = 10000 220 / 569; 296 22 / 33 and 381 / 574;
// d = 32, 584 (T = 5) 20.3 / 24.9 and 387 / 444.
// d <= 32: 300 with T = 20 11.4 / 14.0, 512 with T = 5 11.5 / 12.7, with T = 20 13.0 / 12.8 (every warp of the SM in every layer).  d = 64
// with a second round of CTAs (441): 14.6 / 15.0 with T = 5 but 25.3 / 22.6 with T = 20.
bool ffma_small_better(const FfmaAttend& a) {
  const int64_t ctas = (a.nq + kR - 1) / kR * a.BH;
  return a.d <= 64 && a.layer_stride == 0 && a.z == nullptr && ctas <= (per_sm(a.d) - (a.d <= 32 && a.T > 10)) * (int64_t)a.sms;
}

cudaError_t launch_ffma_small(const FfmaAttend& a, const void* Q, const void* kv, void* out, cudaStream_t s) {
  const float *q = (const float*)Q, *k = (const float*)kv;
  return a.d <= 32 ? launch<32>(a, q, k, (float*)out, s) : launch<64>(a, q, k, (float*)out, s);
}

}  // namespace csat

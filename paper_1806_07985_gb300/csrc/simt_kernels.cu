// CUDA-core kernels around the partial MTTKRPs: sums of split partials,
// multi-TTVs on dimension-tree nodes, sums of squares, bf16 conversion.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "nncp_internal.cuh"

namespace nncp {

namespace {

constexpr int kBK = 32;   // contraction tile
constexpr int kThreads = 256;

__device__ __forceinline__ void decompose(const KrpDesc& d, long long k, int R, int* off) {
  for (int m = 0; m < d.nm; ++m) {
    long long dm = d.dim[m];
    long long km = k % dm;
    k /= dm;
    off[m] = (int)(km * R);
  }
}

__device__ __forceinline__ float krp_value(const KrpDesc& d, const int* off, int r) {
  float v = 1.0f;
  for (int m = 0; m < d.nm; ++m) v *= __ldg(d.H[m] + off[m] + r);
  return v;
}

// out[e] = sum_{c < C} part[c * E + e] (deterministic: four interleaved partial
// sums over c = 0, 4, 8, ... / 1, 5, 9, ... combined in a fixed order).  The
// loads of eight chunks are issued before any is added; V = 4 sums four
// consecutive elements per thread with 16-byte loads (large E only).
template <int V>
__global__ void k_reduce_chunks(const float* __restrict__ part, long long E, int C,
                                float* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  using VT = typename std::conditional<V == 4, float4, float>::type;
  const VT* pv = reinterpret_cast<const VT*>(part);
  VT* ov = reinterpret_cast<VT*>(out);
  const long long Ev = E / V;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < Ev;
       e += (long long)gridDim.x * blockDim.x) {
    float s[4][V];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < V; ++i) s[q][i] = 0.0f;
    int c = 0;
    for (; c + 8 <= C; c += 8) {
      VT v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = __ldg(pv + (long long)(c + q) * Ev + e);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float* f = reinterpret_cast<const float*>(&v[q]);
#pragma unroll
        for (int i = 0; i < V; ++i) s[q & 3][i] += f[i];
      }
    }
    for (; c + 4 <= C; c += 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const VT v = __ldg(pv + (long long)(c + q) * Ev + e);
        const float* f = reinterpret_cast<const float*>(&v);
#pragma unroll
        for (int i = 0; i < V; ++i) s[q][i] += f[i];
      }
    }
    for (; c < C; ++c) {
      const VT v = __ldg(pv + (long long)c * Ev + e);
      const float* f = reinterpret_cast<const float*>(&v);
#pragma unroll
      for (int i = 0; i < V; ++i) s[0][i] += f[i];
    }
    VT r;
    float* rf = reinterpret_cast<float*>(&r);
#pragma unroll
    for (int i = 0; i < V; ++i) rf[i] = (s[0][i] + s[1][i]) + (s[2][i] + s[3][i]);
    ov[e] = r;
  }
}

// The sums of k_reduce_chunks<1> (chunk c into accumulator c mod 4, the chunks
// past the last multiple of four into accumulator 0, then (a0 + a1) + (a2 + a3),
// so the same bits) with one accumulator per lane of a quad: four times the
// threads, each with a quarter of the dependent loads.
__global__ void k_reduce_chunks_quad(const float* __restrict__ part, long long E, int C,
                                     float* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  const long long e = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 2;
  const int q = threadIdx.x & 3;
  const int C4 = C & ~3;
  float s = 0.0f;
  if (e < E) {
#pragma unroll 4
    for (int c = q; c < C4; c += 4) s += __ldg(part + (long long)c * E + e);
    if (q == 0)
      for (int c = C4; c < C; ++c) s += __ldg(part + (long long)c * E + e);
  }
  const float u = s + __shfl_down_sync(0xffffffffu, s, 1);  // q = 0: a0 + a1, q = 2: a2 + a3
  const float v = u + __shfl_down_sync(0xffffffffu, u, 2);  // q = 0: (a0 + a1) + (a2 + a3)
  if (q == 0 && e < E) out[e] = v;
}

// Multi-TTV leaf: out(i, r) = sum_k T[(i + I*k)*R + r] * KK(k, r).
// Threads cover consecutive flattened (i, r) positions (V per thread, V = 4
// when R % 4 == 0), so every k step reads one contiguous run of the node
// temporary; the k loop is unrolled to keep several loads in flight.
template <int V>
__global__ void __launch_bounds__(kThreads)
k_mttv_leaf(const float* __restrict__ T, long long I, long long K, KrpDesc KK, int R,
            long long kchunk, float* __restrict__ out, long long out_chunk_stride) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ float smem[];
  float* Ws = smem;  // kBK x R
  __shared__ int offs[kBK][kMaxModes];
  const long long E = I * R;
  const long long e = ((long long)blockIdx.x * kThreads + threadIdx.x) * V;
  const int r = (int)(e % R);
  const long long kbeg = (long long)blockIdx.y * kchunk;
  const long long kend = min(K, kbeg + kchunk);
  float acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = 0.0f;
  for (long long k0 = kbeg; k0 < kend; k0 += kBK) {
    if (threadIdx.x < kBK) {
      long long k = k0 + threadIdx.x;
      if (k < kend) decompose(KK, k, R, offs[threadIdx.x]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kBK * R; t += kThreads) {
      int kk = t / R, rr = t % R;
      Ws[t] = (k0 + kk < kend) ? krp_value(KK, offs[kk], rr) : 0.0f;
    }
    __syncthreads();
    if (e < E) {
      const int kn = (int)min((long long)kBK, kend - k0);
      const float* Tp = T + (I * k0) * R + e;
      if (V == 4) {
        // eight node rows in flight, then their products in k order
        int kk = 0;
        for (; kk + 8 <= kn; kk += 8) {
          float4 tv[8];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            tv[q] = __ldg(reinterpret_cast<const float4*>(Tp + I * R * (kk + q)));
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float4 wv = *reinterpret_cast<const float4*>(Ws + (kk + q) * R + r);
            acc[0] = fmaf(tv[q].x, wv.x, acc[0]);
            acc[V > 1 ? 1 : 0] = fmaf(tv[q].y, wv.y, acc[V > 1 ? 1 : 0]);
            acc[V > 2 ? 2 : 0] = fmaf(tv[q].z, wv.z, acc[V > 2 ? 2 : 0]);
            acc[V > 3 ? 3 : 0] = fmaf(tv[q].w, wv.w, acc[V > 3 ? 3 : 0]);
          }
        }
#pragma unroll 4
        for (; kk < kn; ++kk) {
          const float4 tv = __ldg(reinterpret_cast<const float4*>(Tp + I * R * kk));
          const float4 wv = *reinterpret_cast<const float4*>(Ws + kk * R + r);
          acc[0] = fmaf(tv.x, wv.x, acc[0]);
          acc[V > 1 ? 1 : 0] = fmaf(tv.y, wv.y, acc[V > 1 ? 1 : 0]);
          acc[V > 2 ? 2 : 0] = fmaf(tv.z, wv.z, acc[V > 2 ? 2 : 0]);
          acc[V > 3 ? 3 : 0] = fmaf(tv.w, wv.w, acc[V > 3 ? 3 : 0]);
        }
      } else {
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) acc[0] = fmaf(__ldg(Tp + I * R * kk), Ws[kk * R + r], acc[0]);
      }
    }
    __syncthreads();
  }
  if (e < E) {
    float* o = out + (long long)blockIdx.y * out_chunk_stride + e;
#pragma unroll
    for (int v = 0; v < V; ++v) o[v] = acc[v];
  }
}

// Multi-TTV to the child node: out(j, r) = sum_i T[(i + I*j)*R + r] * H(i, r).
// One CTA per j; thread (g, r-group) strides over i (V = 4 consecutive ranks
// per thread when R % 4 == 0); a fixed-order reduction over g.
template <int V>
__global__ void k_mttv_first(const float* __restrict__ T, long long I, const float* __restrict__ H,
                             int R, int G, float* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ float red[];  // G x R
  const long long j = blockIdx.x;
  const int RV = R / V;
  const int rv = threadIdx.x % RV;
  const int g = threadIdx.x / RV;
  if (g < G) {
    const float* Tj = T + I * j * R;
    float acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0.0f;
    if (V == 4) {
#pragma unroll 4
      for (long long i = g; i < I; i += G) {
        const float4 tv = __ldg(reinterpret_cast<const float4*>(Tj + i * R) + rv);
        const float4 hv = __ldg(reinterpret_cast<const float4*>(H + i * R) + rv);
        acc[0] = fmaf(tv.x, hv.x, acc[0]);
        acc[V > 1 ? 1 : 0] = fmaf(tv.y, hv.y, acc[V > 1 ? 1 : 0]);
        acc[V > 2 ? 2 : 0] = fmaf(tv.z, hv.z, acc[V > 2 ? 2 : 0]);
        acc[V > 3 ? 3 : 0] = fmaf(tv.w, hv.w, acc[V > 3 ? 3 : 0]);
      }
    } else {
#pragma unroll 4
      for (long long i = g; i < I; i += G)
        acc[0] = fmaf(__ldg(Tj + i * R + rv), __ldg(H + i * R + rv), acc[0]);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) red[g * R + rv * V + v] = acc[v];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < R; t += blockDim.x) {
    float sum = 0.0f;
    for (int gg = 0; gg < G; ++gg) sum += red[gg * R + t];
    out[j * R + t] = sum;
  }
}

// Sum of squares: four (float32) or two (bf16) squares at a time in float32,
// accumulated as float-float pairs (TwoSum: no rounding is lost down to ~2^-48),
// which cost a few float32 operations per 16 bytes, and added up in float64 once
// per eight loads; one float64 addition per load had held the pass to 3.8 TB/s
// on a GB300, float64 issuing at about a sixtieth of the float32 rate there.
struct SumFF {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float s = hi + v, t = s - hi;
    lo += (hi - (s - t)) + (v - t);
    hi = s;
  }
};

__global__ void __launch_bounds__(256)
k_sumsq_partial(const void* __restrict__ Xv, int bf16, long long n, double* __restrict__ partials) {
  __shared__ double sh[8];
  const long long stride = (long long)gridDim.x * 256;
  const long long t0 = (long long)blockIdx.x * 256 + threadIdx.x;
  const int per = bf16 ? 8 : 4;  // elements per 16 bytes
  const long long nv = n / per;
  const uint4* V = reinterpret_cast<const uint4*>(Xv);
  SumFF a0, a1;
  auto square = [&](const uint4& v) {
    if (bf16) {
      // products of bf16 values are exact in float32
      const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float x = __uint_as_float(u[i] << 16), y = __uint_as_float(u[i] & 0xffff0000u);
        a0.add(x * x);
        a1.add(y * y);
      }
    } else {
      const float x = __uint_as_float(v.x), y = __uint_as_float(v.y), z = __uint_as_float(v.z),
                  w = __uint_as_float(v.w);
      float s = x * x;
      s = fmaf(y, y, s);
      s = fmaf(z, z, s);
      s = fmaf(w, w, s);
      a0.add(s);
    }
  };
  // the same in float64, for sums past float32's range (and what is not finite)
  auto square64 = [&](const uint4& v) {
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
    double s = 0.0;
    for (int i = 0; i < 4; ++i) {
      const double x = __uint_as_float(bf16 ? u[i] << 16 : u[i]);
      const double y = bf16 ? __uint_as_float(u[i] & 0xffff0000u) : 0.0f;
      s += x * x + y * y;
    }
    return s;
  };
  // into float64 after every eight loads; false: their sum left float32's range
  double acc = 0.0;
  auto flush = [&]() {
    const bool in = isfinite(a0.hi + a1.hi);
    if (in) acc += ((double)a0.hi + (double)a1.hi) + (double)(a0.lo + a1.lo);
    a0 = a1 = SumFF();
    return in;
  };
  long long t = t0;
  for (; t + 7 * stride < nv; t += 8 * stride) {  // eight loads in flight
    uint4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __ldcs(V + t + q * stride);
#pragma unroll
    for (int q = 0; q < 8; ++q) square(v[q]);
    if (!flush())
      for (int q = 0; q < 8; ++q) acc += square64(v[q]);
  }
  for (long long r = t; r < nv; r += stride) square(__ldcs(V + r));
  if (!flush())
    for (; t < nv; t += stride) acc += square64(V[t]);
  for (long long e = nv * per + t0; e < n; e += stride) {
    const double x = bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(Xv)[e])
                          : static_cast<const float*>(Xv)[e];
    acc += x * x;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int i = 0; i < 8; ++i) tot += sh[i];
    partials[blockIdx.x] = tot;
  }
}

__global__ void k_sum_partials(const double* __restrict__ partials, int n, double* out) {
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += 32) s += partials[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) out[0] = s;
}

__global__ void k_to_bf16(const float* __restrict__ X, __nv_bfloat16* __restrict__ Y, long long n) {
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    Y[t] = __float2bfloat16_rn(X[t]);
}

long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

// Split of the contraction across CTAs: enough CTAs for ~4 per SM, each
// chunk at least `min_chunk` contraction elements.
int choose_chunks(long long ctas_other, long long Ktot, int num_sms, long long min_chunk = 8LL * kBK) {
  long long target = 4LL * num_sms;
  if (ctas_other >= target) return 1;
  long long C = ceil_div(target, ctas_other);
  long long max_c = max(1LL, ceil_div(Ktot, min_chunk));
  return (int)min(C, max_c);
}

// Multi-TTV chunks: one contraction element is a whole I*R block of the node,
// so chunks of 8 elements already stream enough bytes.
constexpr long long kMttvMinChunk = 8;

}  // namespace

cudaError_t launch_reduce_chunks(const float* part, int64_t E, int C, float* out, int num_sms,
                                 cudaStream_t st) {
  // four elements per thread only when that still leaves a full wave of CTAs:
  // the reduction is bound by how many SMs pull the partials
  const bool v4 = E % 4 == 0 && E / 4 >= (int64_t)num_sms * 8 * 256 &&
                  reinterpret_cast<uintptr_t>(part) % 16 == 0 &&
                  reinterpret_cast<uintptr_t>(out) % 16 == 0;
  if (!v4)  // small outputs: a quad of threads per output (same sums)
    return launch_kernel(k_reduce_chunks_quad, dim3((unsigned)ceil_div(4 * (long long)E, 256)),
                         dim3(256), 0, st, part, (long long)E, C, out);
  const long long Ev = E / 4;
  int blocks = (int)min(ceil_div(Ev, 256), (long long)num_sms * 8);
  if (blocks < 1) blocks = 1;
  return launch_kernel(k_reduce_chunks<4>, dim3(blocks), dim3(256), 0, st, part, (long long)E, C,
                       out);
}

size_t mttv_leaf_partials(int64_t I, int64_t K, int R, int num_sms) {
  const int V = (R % 4 == 0) ? 4 : 1;
  long long gx = ceil_div(ceil_div((long long)I * R, V), kThreads);
  int C = choose_chunks(gx, K, num_sms, kMttvMinChunk);
  return C > 1 ? (size_t)C * I * R : 0;
}

cudaError_t launch_mttv_leaf(const float* T, int64_t I, int64_t K, const KrpDesc& KK, int R,
                             float* out, float* partials, size_t part_cap, int num_sms,
                             cudaStream_t st) {
  const int V = (R % 4 == 0) ? 4 : 1;
  long long E = (long long)I * R;
  long long gx = ceil_div(ceil_div(E, V), kThreads);
  int C = choose_chunks(gx, K, num_sms, kMttvMinChunk);
  long long kchunk = ceil_div(K, C);
  C = (int)ceil_div(K, kchunk);
  float* dst = out;
  if (C > 1) {
    if ((size_t)C * E > part_cap || partials == nullptr) return cudaErrorInvalidValue;
    dst = partials;
  }
  size_t smem = (size_t)kBK * R * sizeof(float);
  cudaError_t e = launch_kernel(V == 4 ? k_mttv_leaf<4> : k_mttv_leaf<1>,
                                dim3((unsigned)gx, (unsigned)C), dim3(kThreads), smem, st, T,
                                (long long)I, (long long)K, KK, R, kchunk, dst, E);
  if (e != cudaSuccess || C == 1) return e;
  return launch_reduce_chunks(partials, E, C, out, num_sms, st);
}

cudaError_t launch_mttv_first(const float* T, int64_t I, int64_t J, const float* H, int R,
                              float* out, cudaStream_t st) {
  const int V = (R % 4 == 0) ? 4 : 1;
  const int RV = R / V;
  int G = std::max(1, 256 / RV);
  if (G > I) G = (int)I;
  const int threads = G * RV;
  size_t smem = (size_t)G * R * sizeof(float);
  return launch_kernel(V == 4 ? k_mttv_first<4> : k_mttv_first<1>, dim3((unsigned)J),
                       dim3(threads), smem, st, T, (long long)I, H, R, G, out);
}

cudaError_t launch_sumsq_partials(const void* X, int bf16, int64_t n, double* partials, int nparts,
                                  cudaStream_t st) {
  k_sumsq_partial<<<nparts, 256, 0, st>>>(X, bf16, n, partials);
  return cudaGetLastError();
}

cudaError_t launch_sumsq(const void* X, int bf16, int64_t n, double* partials, int nparts,
                         double* out, cudaStream_t st) {
  const cudaError_t e = launch_sumsq_partials(X, bf16, n, partials, nparts, st);
  if (e != cudaSuccess) return e;
  k_sum_partials<<<1, 32, 0, st>>>(partials, nparts, out);
  return cudaGetLastError();
}

cudaError_t launch_to_bf16(const float* X, uint16_t* Y, int64_t n, cudaStream_t st) {
  int blocks = (int)min(ceil_div(n, 256), 152LL * 16);
  if (blocks < 1) blocks = 1;
  k_to_bf16<<<blocks, 256, 0, st>>>(X, reinterpret_cast<__nv_bfloat16*>(Y), n);
  return cudaGetLastError();
}

}  // namespace nncp

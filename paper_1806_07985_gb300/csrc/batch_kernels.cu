// Batched NNCP-HALS: many independent tensors of the same order N, each with
// its own mode lengths and rank, solved together.  Every tensor uses root
// split 1 (node {1} and node {2..N}, Fig. 1 shape below it), so the
// dimension-tree schedule of one outer iteration (Sec. IV-A; Alg. 1) is the
// same sequence of operations for all of them, and each operation is one
// launch over a device work list of (tensor, chunk) items.  Tensors whose fit
// has converged are skipped by every item.  Reductions across chunks are
// summed in chunk order, so a tensor's result does not depend on the batch.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "batch_kernels.cuh"

namespace nncp {

namespace {

__device__ __forceinline__ bool tensor_done(const BTensor& t) { return t.flags[0] != 0; }

// ---------------------------------------------------------------- init --

// Float-float accumulator: TwoSum keeps what a float32 addition rounds off, so
// the pair carries about 48 bits at a few float32 operations per term (a float64
// addition issues at about a sixtieth of their rate here).
struct SumFF {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float s = hi + v, t = s - hi;
    lo += (hi - (s - t)) + (v - t);
    hi = s;
  }
  // a * b exactly: the rounded product and its error
  __device__ __forceinline__ void add_product(float a, float b) {
    const float p = a * b;
    lo += fmaf(a, b, -p);
    add(p);
  }
  __device__ __forceinline__ double value() const {
    return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
  }
};

// alpha partials: item (tensor, chunk of kAlphaChunk elements) -> alpha_part[item];
// squares summed four at a time in FP32, those sums as float-float pairs, the
// threads' totals in FP64 (fixed order)
__global__ void __launch_bounds__(256) k_b_sumsq(const BTensor* __restrict__ ts,
                                                 const int4* __restrict__ items,
                                                 double* __restrict__ alpha_part) {
  const int4 it = items[blockIdx.x];
  const BTensor& t = ts[it.x];
  const long long e0 = (long long)it.y * kAlphaChunk;
  const int n = (int)min(kAlphaChunk, t.I - e0);
  const float* x = t.X + e0;
  const int n4 = n >> 2;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  double acc = 0.0;
  for (int v0 = threadIdx.x; v0 < n4; v0 += 8 * 256) {
    // eight loads in flight; into float64 after each eight (in float64 alone where
    // their sum leaves float32's range)
    float4 a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      a[q] = v0 + 256 * q < n4 ? __ldcs(x4 + v0 + 256 * q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    SumFF s;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      s.add(a[q].x * a[q].x + a[q].y * a[q].y + a[q].z * a[q].z + a[q].w * a[q].w);
    if (isfinite(s.hi)) {
      acc += s.value();
    } else {
      for (int q = 0; q < 8; ++q)
        acc += ((double)a[q].x * a[q].x + (double)a[q].y * a[q].y) +
               ((double)a[q].z * a[q].z + (double)a[q].w * a[q].w);
    }
  }
  if ((int)threadIdx.x < n - 4 * n4) {
    const float v = x[4 * n4 + threadIdx.x];
    acc += (double)(v * v);
  }
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    alpha_part[blockIdx.x] = s;
  }
}

// per tensor: alpha = sum of its partials (in order), normalise every factor
// (lambda = product of the column norms), G_n = H_n^T H_n, S for mode 1,
// flags and fit history cleared (Alg. 3 initialisation).  CTA (tensor, mode)
// for the factors, then CTA per tensor for what joins the modes.  The column
// sums and Grams are float-float sums of exact products, about 48 bits, of which the
// iterations read float32 (S32); in float64, with a float64 division per factor element, one
// CTA per tensor took 257 us for 1024 tensors on a GB300.  (96 tensors against float64: the
// factors are 4.8e-7 off after one iteration and 1.25e-6 after eight, 5.4e-7 and 1.37e-6
// with float64 sums and the multi-TTVs before these.)
__global__ void __launch_bounds__(256) k_b_init_mode(BTensor* __restrict__ ts) {
  BTensor& t = ts[blockIdx.x];
  const int n = blockIdx.y;
  if (n >= t.N) return;  // the tensors may be of different orders
  const int R = t.R, R2 = R * R;
  const int In = (int)t.dims[n];
  float* Hn = t.H[n];
  extern __shared__ __align__(16) float hs[];  // In x R
  __shared__ double inv[kBatchMaxRank];
  __shared__ double part[256];
  const int tid = threadIdx.x;
  for (int e = tid; e < In * R; e += 256) hs[e] = Hn[e];
  __syncthreads();
  // column sums of squares: the rows of a column over 256 / R threads, their
  // sums added in order
  const int P = 256 / R, r0 = tid % R, p0 = tid / R;
  if (p0 < P) {
    SumFF s;
    for (int i = p0; i < In; i += P) s.add_product(hs[i * R + r0], hs[i * R + r0]);
    part[tid] = s.value();
  }
  __syncthreads();
  if (tid < R) {
    double s = 0.0;
    for (int p = 0; p < P; ++p) s += part[p * R + tid];
    if (!(s > 1e-30 && s < 1e36)) {  // squares near the ends of float32's range: in float64
      s = 0.0;
      for (int i = 0; i < In; ++i) s += (double)hs[i * R + tid] * hs[i * R + tid];
    }
    const double c = sqrt(s);
    inv[tid] = c > 0.0 ? 1.0 / c : 0.0;
    // the norms wait in this mode's Gram row for k_b_init
    t.G[(long long)n * R2 + tid] = c;
  }
  __syncthreads();
  for (int e = tid; e < In * R; e += 256) {
    const float h = (float)((double)hs[e] * inv[e % R]);
    hs[e] = h;
    Hn[e] = h;
  }
}

__global__ void __launch_bounds__(256) k_b_init(BTensor* __restrict__ ts, const double* __restrict__ alpha_part,
                                                const int* __restrict__ alpha_first) {
  BTensor& t = ts[blockIdx.x];
  const int R = t.R, N = t.N, R2 = R * R;
  const int tid = threadIdx.x;
  if (tid == 0) {
    double a = 0.0;
    for (int c = alpha_first[blockIdx.x]; c < alpha_first[blockIdx.x + 1]; ++c) a += alpha_part[c];
    t.scal[0] = a;
    t.scal[1] = t.tol;
    t.flags[0] = 0;
    t.flags[1] = 0;
    t.flags[2] = 0;
  }
  if (tid < R) {
    double l = 1.0;
    for (int n = 0; n < N; ++n) l *= t.G[(long long)n * R2 + tid];
    t.lam[tid] = l;
  }
  extern __shared__ __align__(16) float hs[];  // one factor
  __syncthreads();
  double S[(kBatchMaxRank * kBatchMaxRank + 255) / 256];
#pragma unroll
  for (int q = 0; q < (int)(sizeof S / sizeof S[0]); ++q) S[q] = 1.0;
  for (int n = 0; n < N; ++n) {
    const int In = (int)t.dims[n];
    for (int e = tid; e < In * R; e += 256) hs[e] = t.H[n][e];
    __syncthreads();
    double* Gn = t.G + (long long)n * R2;
#pragma unroll
    for (int q = 0; q < (int)(sizeof S / sizeof S[0]); ++q) {
      const int e = tid + 256 * q;
      if (e < R2) {
        const int a = e / R, b = e - a * R;
        SumFF s;
        for (int i = 0; i < In; ++i) s.add_product(hs[i * R + a], hs[i * R + b]);
        const double g = s.value();
        Gn[e] = g;
        if (n > 0) S[q] *= g;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < (int)(sizeof S / sizeof S[0]); ++q) {
    const int e = tid + 256 * q;
    if (e < R2) {
      t.S[e] = S[q];
      t.S32[e] = (float)S[q];
    }
  }
}

// ------------------------------------------------ partial MTTKRPs (root) --
//
// Both root contractions stream X_(1)^T (rows j of I_1 contiguous floats) in
// tiles of whole rows; the thread mapping is sized from the tensor's own rank, and
// when one tile holds too few (row, rank-group) pairs for 256 threads the
// contraction range is split over groups whose partial sums are added in group
// order.

constexpr int kThreads = 256;
// Split groups are sized for kGroupThreads whatever the block size, so the
// summation order of an output depends only on its tensor's shape.
constexpr int kGroupThreads = 256;

// Tiles are copied global -> shared with cp.async (no registers held while
// in flight); the CTAs of an SM hide each other's copies.  X is read once per pass.
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ranks r0 .. r0 + 3 of a factor row (zero beyond R); vector load when R % 4 == 0
__device__ __forceinline__ float4 ld_rank4(const float* __restrict__ row, int r0, int R) {
  if ((R & 3) == 0) {
    if (r0 >= R) return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    return __ldg(reinterpret_cast<const float4*>(row + r0));
  }
  float4 h;
  h.x = r0 < R ? __ldg(row + r0) : 0.0f;
  h.y = r0 + 1 < R ? __ldg(row + r0 + 1) : 0.0f;
  h.z = r0 + 2 < R ? __ldg(row + r0 + 2) : 0.0f;
  h.w = r0 + 3 < R ? __ldg(row + r0 + 3) : 0.0f;
  return h;
}

// ranks 4 q .. 4 q + 3 of an output row (16-byte aligned when R % 4 == 0)
__device__ __forceinline__ void store_rank4(float* row, int q, int R, const float (&v)[4]) {
  float* o = row + 4 * q;
  if ((R & 3) == 0) {
    if (4 * q < R) *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
    return;
  }
#pragma unroll
  for (int b = 0; b < 4; ++b)
    if (4 * q + b < R) o[b] = v[b];
}

__device__ __forceinline__ void fma4(float (&a)[4], float x, const float4& w) {
  a[0] = fmaf(x, w.x, a[0]);
  a[1] = fmaf(x, w.y, a[1]);
  a[2] = fmaf(x, w.z, a[2]);
  a[3] = fmaf(x, w.w, a[3]);
}

// Work item w of a phase for this CTA: with queue == NULL the CTA's own
// index (one CTA per item, the hardware schedules them); otherwise the next
// item taken from the phase's counter by a persistent CTA (-1: none left).
// Either way an item is computed the same way, so the choice changes no bits.
__device__ __forceinline__ int next_item(int* queue, int n_items, int* slot, bool first) {
  if (!queue) return first ? (int)blockIdx.x : -1;
  __syncthreads();  // every thread has read the previous item
  if (threadIdx.x == 0) *slot = atomicAdd(queue, 1);
  __syncthreads();
  return *slot < n_items ? *slot : -1;
}

// root -> node {1}: part[c](i, r) = sum_{j in chunk c} X[i + I1 j] K(j, r),
// K = H_N (.) ... (.) H_2 (rows formed per tile, never stored whole).  Item (tensor,
// chunk).  The sums' order: G = 256 / I1 column groups split each tile's rows
// (j = g, g + G, ...) and are added in group order at the end of the chunk.
//
// What bounds it is shared memory, which returns 128 bytes per cycle and SM however
// few of them differ: a thread with one row reads 1 + R floats for R FMAs.  Here it
// holds four rows of one column group (rows ii + x ceil(I1 / 4)) x one, two or four
// rank groups; tiles are single-buffered, CTAs small and several per SM, and the
// Khatri-Rao rows are formed while a tile's copies are in flight.  (1024 tensors of 16
// to 128 per mode at ranks 4, 8 and 16, 629 MB: one row per thread 275 us, this 202 us.)
template <int RMAX>
struct RightCfg {
  static constexpr int T = RMAX <= 32 ? 128 : 256;  // threads
  static constexpr int NA = RMAX <= 16 ? 8 : 16;    // accumulators of four ranks per thread
  static constexpr int CTAS = RMAX <= 16 ? 5 : (RMAX <= 32 ? 4 : 2);
};

// A thread's Khatri-Rao rows: their digit in mode 2 and the rest, kept by addition
// from tile to tile (a division per row and mode cost more than the products).
struct KrDigits {
  int a, rest;     // of this thread's first row of the tile
  int ta, trest;   // a tile's rows
  int sa, srest;   // the rows from one of the thread's entries to its next
};
__device__ __forceinline__ void kr_step(int& a, int& rest, int da, int drest, int d) {
  a += da;
  rest += drest;
  if (a >= d) {
    a -= d;
    ++rest;
  }
}

// Khatri-Rao rows of a tile of njk: entry (row, rank group)
template <int T>
__device__ __forceinline__ void right_krp(const BTensor& t, int njk, int lg, KrDigits& k, float* Ws) {
  const int N = t.N, R = t.R, r0 = 4 * ((int)threadIdx.x & ((1 << lg) - 1)), d = (int)t.dims[1];
  const float* H1 = t.H[1];
  const float* H2 = N > 2 ? t.H[2] : nullptr;
  int a = k.a, rest = k.rest;
#pragma unroll 2
  for (int e = threadIdx.x; e < njk << lg; e += T) {
    float4 w = ld_rank4(H1 + a * R, r0, R);
    if (N == 3) {
      const float4 h = ld_rank4(H2 + rest * R, r0, R);
      w.x *= h.x;
      w.y *= h.y;
      w.z *= h.z;
      w.w *= h.w;
    } else {
      unsigned rem = (unsigned)rest;
      for (int m = 2; m < N; ++m) {
        unsigned jm = rem;
        if (m + 1 < N) {
          const unsigned dm = (unsigned)t.dims[m];
          rem = jm / dm;
          jm -= rem * dm;
        }
        const float4 h = ld_rank4(t.H[m] + (int)jm * R, r0, R);
        w.x *= h.x;
        w.y *= h.y;
        w.z *= h.z;
        w.w *= h.w;
      }
    }
    reinterpret_cast<float4*>(Ws)[e] = w;
    kr_step(a, rest, k.sa, k.srest, d);
  }
  kr_step(k.a, k.rest, k.ta, k.trest, d);
}

// One item, in one of two forms with the same copies, Khatri-Rao rows and group sums
// (one body: the CTAs of an SM run different forms, and a body each overflowed the
// instruction cache): four rows x rqt rank groups, rqt the fewest with which T threads
// suffice, or, where ceil(I_1 / 4) rounds up too far for any, 256 / T (column group,
// row) pairs with all rank groups.
template <int RQT, int NA>
__device__ __forceinline__ void right_quads(const float* xp, const float4* wp, int Iq, int first, int njk,
                                            int G, int xs, int ws, float (&acc)[NA][4]) {
#pragma unroll 2
  for (int jj = first; jj < njk; jj += G, xp += xs, wp += ws) {
    float xv[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) xv[x] = xp[x * Iq];  // past the last row: not used
#pragma unroll
    for (int u = 0; u < RQT; ++u) {
      const float4 w = wp[u];
#pragma unroll
      for (int x = 0; x < 4; ++x) fma4(acc[4 * u + x], xv[x], w);
    }
  }
}

template <int RMAX>
__device__ __forceinline__ void pm_right_item(const BTensor& t, int chunk, float* smem) {
  constexpr int T = RightCfg<RMAX>::T, NA = RightCfg<RMAX>::NA;
  constexpr int NP = kGroupThreads / T;  // pairs per thread, NA / NP rank groups each
  float* Xs = smem;
  float* Ws = smem + kTileFloats;
  const int tid = threadIdx.x;
  const int R = t.R, Rq = b_rq(R), lg = __ffs(Rq) - 1;
  const int I1 = (int)t.dims[0];
  const int nj = t.rows_r;
  const int J = (int)(t.I / I1);
  const int j0 = chunk * (int)t.jchunk;
  const int j1 = min(J, j0 + (int)t.jchunk);
  const int G = kGroupThreads / I1;
  const int Iq = (I1 + 3) >> 2;
  const int units = Iq * G;  // threads for four rows and every rank group, about 64
  int rqt = 1;
  while (rqt < Rq && units * (Rq / rqt) > T) rqt *= 2;
  const bool pairs = units * (Rq / rqt) > T || 4 * rqt > NA;
  if (pairs) rqt = Rq;
  // thread = (row ii, block ub of rank groups, column group g), ii fastest; pairs:
  // (g, ii) and, with two, (g1, i1)
  const int nub = Rq / rqt, w1 = pairs ? I1 : Iq;
  const int v = tid / w1, ii = tid - v * w1;
  const int ub = v & (nub - 1), g = v / nub;
  const int g1 = (tid + T) / I1, i1 = tid + T - g1 * I1;
  float acc[NA][4];
#pragma unroll
  for (int x = 0; x < NA; ++x)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[x][b] = 0.0f;
  const float4* W4 = reinterpret_cast<const float4*>(Ws) + ub * rqt;
  KrDigits kd;
  {
    const int d = (int)t.dims[1], row = j0 + (tid >> lg), step = T >> lg;
    kd.rest = row / d;
    kd.a = row - kd.rest * d;
    kd.trest = nj / d;
    kd.ta = nj - kd.trest * d;
    kd.srest = step / d;
    kd.sa = step - kd.srest * d;
  }
  for (int jt = j0; jt < j1; jt += nj) {
    const int njk = min(nj, j1 - jt);
    {
      const float* src = t.X + (long long)jt * I1;
      const int L = njk * I1, L4 = L & ~3;
#pragma unroll 4
      for (int e = 4 * tid; e < L4; e += 4 * T) cp_async16(Xs + e, src + e);
      if (L4 + tid < L) cp_async4(Xs + L4 + tid, src + L4 + tid);
    }
    right_krp<T>(t, njk, lg, kd, Ws);
    cp_async_wait_all();
    __syncthreads();
    const float* xp = Xs + ii + g * I1;
    const float4* wp = W4 + (g << lg);
    const int first = g < G ? g : njk;
    if (pairs) {
#pragma unroll
      for (int x = 0; x < NP; ++x) {
        const int gx = x ? g1 : g, ix = x ? i1 : ii;
#pragma unroll 1
        for (int jj = gx < G ? gx : njk; jj < njk; jj += G) {
          const float xv = Xs[jj * I1 + ix];
#pragma unroll
          for (int u = 0; u < NA / NP; ++u)
            if (u < Rq) fma4(acc[NA / NP * x + u], xv, W4[(jj << lg) + u]);
        }
      }
    } else if (rqt == 1) {
      right_quads<1>(xp, wp, Iq, first, njk, G, G * I1, G << lg, acc);
    } else if (NA == 8 || rqt == 2) {
      right_quads<2>(xp, wp, Iq, first, njk, G, G * I1, G << lg, acc);
    } else {
      right_quads<NA / 4>(xp, wp, Iq, first, njk, G, G * I1, G << lg, acc);
    }
    __syncthreads();
  }
  // the column groups' sums, added in group order, four rank groups at a time:
  // (rank group, column group, row)
  float4* red = reinterpret_cast<float4*>(Xs);
  float* out = t.part + (long long)chunk * I1 * R;
#pragma unroll 1
  for (int q0 = 0; q0 < Rq; q0 += 4) {
    const int nq = min(4, Rq - q0);
#pragma unroll
    for (int x = 0; x < NA; ++x) {
      const int px = x / (NA / NP);  // pair of the accumulator
      const int u = (pairs ? x % (NA / NP) : ub * rqt + (x >> 2)) - q0;
      const int gx = pairs && px ? g1 : g;
      const int ix = pairs ? (px ? i1 : ii) : ii + (x & 3) * Iq;
      if ((pairs || (x >> 2) < rqt) && u >= 0 && u < nq && gx < G && ix < I1)
        red[u * kGroupThreads + gx * I1 + ix] = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
    }
    __syncthreads();
    for (int e = tid; e < I1 * nq; e += T) {
      const int q = e & (nq - 1), i = e / nq;
      const float4* rp = red + q * kGroupThreads + i;
      float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      if (G == 1) {
        s4[0] = rp->x; s4[1] = rp->y; s4[2] = rp->z; s4[3] = rp->w;
      }
#pragma unroll 1
      for (int gg = 0; gg < (G > 1 ? G : 0); ++gg) {
        const float4 w = rp[gg * I1];
        s4[0] += w.x;
        s4[1] += w.y;
        s4[2] += w.z;
        s4[3] += w.w;
      }
      store_rank4(out + i * R, q0 + q, R, s4);
    }
    __syncthreads();
  }
}

template <int RMAX>
__global__ void __launch_bounds__(RightCfg<RMAX>::T, RightCfg<RMAX>::CTAS)
k_b_pm_right(const BTensor* __restrict__ ts, const int4* __restrict__ items, int n_items, int* queue) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int slot;
  for (int w = next_item(queue, n_items, &slot, true); w >= 0;
       w = next_item(queue, n_items, &slot, false)) {
    const int4 it = items[w];
    const BTensor& t = ts[it.x];
    if (tensor_done(t)) continue;
    pm_right_item<RMAX>(t, it.y, smem);
  }
}

// ------------------------------------- streamed root -> {1} (schedule 2) --
//
// The arithmetic of pm_right_item (every output's products and sums in the
// same order, so the same bits) with its jobs split over the warps of a
// persistent CTA, the tiles passing through a ring of shared-memory stages:
//   warp 0, scheduler: takes items from the counter (several at a time while
//                      it meets converged tensors), skips those, and writes
//                      each item's descriptor into a ring of item slots;
//   warp 1, loader:    copies an item's descriptor into the header of every
//                      stage of it and the stage's rows of X_(1)^T into the
//                      stage (cp.async, L2 evict-first), arriving on the
//                      stage's full barrier as the copies land;
//   warps 2-4, builders: take stages in turn and form a stage's Khatri-Rao
//                      rows;
//   warps 5-12, consumers (256 threads, a row each): contract each
//                      tile and free its stage; at the end of an item they
//                      add the column groups in group order through the last
//                      stage's tile area, then free it.
// The scheduler runs ahead of the loader and the loader ahead of the rest, so
// tiles stream in across item boundaries.  Every wait is on an mbarrier and
// bounded (about two seconds): on expiry a thread records the error word and
// leaves, and the waits of the other roles then expire in turn.

constexpr int kWsBuildWarps = 3, kWsConsWarps = 8;
constexpr int kWsConsFirstWarp = 2 + kWsBuildWarps;
constexpr int kWsThreads = 32 * (kWsConsFirstWarp + kWsConsWarps);
constexpr int kWsStageFloats = kTileFloats + kWsFloats;
constexpr int kWsItemSlots = 4;
// Khatri-Rao entries (row, rank group) per builder lane and pass: a tile has at most kWsFloats / 4
constexpr int kWsBuildPer = 4;
constexpr int kWsBuildPasses = (kWsFloats / 4 + 32 * kWsBuildPer - 1) / (32 * kWsBuildPer);
constexpr long long kWsWaitCycles = 4000000000LL;

// One item as the builders and consumers need it (w < 0: no more items);
// seq: the item's position in this CTA's sequence; dims[m - 1] and H[m - 1]
// are I_{m+1} and factor m + 1 (root -> {1}); for root -> {2..N}, H[0] is H_1.
struct WsDesc {
  int w, I1, R, N, nj, j0, j1, ntile;
  int seq;
  int dims[kMaxModes - 1];
  float* out;
  const float* H[kMaxModes - 1];
};
struct WsHeader {
  WsDesc d;
  int k;  // tile within the item
  int pad[3];
};
struct WsSlot {
  WsDesc d;
  const float* X;
};
static_assert(sizeof(WsDesc) % 8 == 0 && sizeof(WsHeader) % 16 == 0 && sizeof(WsSlot) % 8 == 0,
              "descriptor layout");
constexpr int kWsDescWords = (int)(sizeof(WsDesc) / 4);
static_assert(kWsDescWords <= 32, "one descriptor word per lane");

__device__ __forceinline__ void mb_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// arrives once every cp.async this thread has issued so far has landed
__device__ __forceinline__ void mb_arrive_cp_async(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mb_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// the same without suspending the thread
__device__ __forceinline__ bool mb_poll(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// A try_wait may suspend a thread for longer than a limit below this many cycles.
constexpr long long kBriefWaitCycles = 1000000;
// Bounded wait of a whole warp (all 32 lanes call it, converged): every lane
// polls (and so acquires the phase), the warp decides together, so a warp
// never splits over an expired wait (the lanes read one clock).  On expiry
// the first wait site to give up is recorded in *err (1 + site).  `limit`:
// clock64 cycles (kWsWaitCycles unless a test shortens it).
__device__ __forceinline__ bool mb_wait(uint32_t bar, uint32_t parity, long long limit, int* err,
                                        int site) {
  const bool brief = limit < kBriefWaitCycles;
  if (__all_sync(0xffffffffu, brief ? mb_poll(bar, parity) : mb_test(bar, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, brief ? mb_poll(bar, parity) : mb_test(bar, parity))) {
    if (clock64() - t0 > limit) {
      if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, 1 + site);
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void cp_async16_hint(float* dst, const float* src, uint64_t pol) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)),
               "l"(src), "l"(pol)
               : "memory");
}

// Shared memory of the streamed kernel: S stages (X tile, Khatri-Rao tile),
// their headers, the item slots and the barriers.
struct WsSmem {
  float* stage0;
  WsHeader* hdr;
  WsSlot* slot;
  uint32_t bar0;
  int S;
  long long wait;  // bounded-wait limit, clock64 cycles
  __device__ float* xs(int s) const { return stage0 + (size_t)s * kWsStageFloats; }
  __device__ uint32_t full(int s) const { return bar0 + 8u * s; }
  __device__ uint32_t empty(int s) const { return bar0 + 8u * (S + s); }
  __device__ uint32_t hfull(int s) const { return bar0 + 8u * (2 * S + s); }
  __device__ uint32_t islot_full(int i) const { return bar0 + 8u * (3 * S + i); }
  __device__ uint32_t islot_empty(int i) const { return bar0 + 8u * (3 * S + kWsItemSlots + i); }
  __device__ uint32_t red_full() const { return bar0 + 8u * (3 * S + 2 * kWsItemSlots); }
  __device__ uint32_t red_empty() const { return bar0 + 8u * (3 * S + 2 * kWsItemSlots + 1); }
  __device__ uint32_t cons_sync() const { return bar0 + 8u * (3 * S + 2 * kWsItemSlots + 2); }
};

__host__ __device__ constexpr size_t ws_smem_bytes(int S) {
  return (size_t)S * kWsStageFloats * sizeof(float) + (size_t)S * sizeof(WsHeader) +
         (size_t)kWsItemSlots * sizeof(WsSlot) +
         (size_t)(3 * S + 2 * kWsItemSlots + 3) * sizeof(uint64_t);
}

template <bool LEFT, typename SM>
__device__ void ws_scheduler(const BTensor* __restrict__ ts, const int4* __restrict__ items,
                             int n_items, int* queue, const SM& sm, int* err) {
  const int lane = threadIdx.x & 31;
  int m = 0;      // item slots filled
  int grab = 1;   // candidates taken per round: doubles while they are all converged
  bool more = true;
  while (more) {
    const int c = lane < grab ? atomicAdd(queue, 1) : n_items;
    const bool live = c < n_items;
    const bool active = live && !tensor_done(ts[items[c].x]);
    unsigned act = __ballot_sync(0xffffffffu, active);
    more = __ballot_sync(0xffffffffu, live) == (grab >= 32 ? 0xffffffffu : (1u << grab) - 1u);
    grab = act ? 1 : min(32, 2 * grab);
    while (act) {
      const int src = __ffs(act) - 1;
      act &= act - 1;
      const int w = __shfl_sync(0xffffffffu, c, src);
      const int sl = m % kWsItemSlots;
      if (!mb_wait(sm.islot_empty(sl), ((m / kWsItemSlots) & 1) ^ 1, sm.wait, err, 1)) return;
      if (lane == 0) {
        const int4 it = items[w];
        const BTensor& t = ts[it.x];
        WsSlot q;
        WsDesc& d = q.d;
        d.w = w;
        d.I1 = (int)t.dims[0];
        d.R = t.R;
        d.N = t.N;
        d.seq = m;
        const int J = (int)(t.I / d.I1);
        if (LEFT) {  // rows [j0, j1) of X_(1)^T in tiles of rows_l, H_1, T = node {2..N}
          d.nj = t.rows_l;
          d.j0 = it.y * d.nj * kLeftItemTiles;
          d.j1 = min(J, d.j0 + d.nj * kLeftItemTiles);
          for (int n = 1; n < kMaxModes; ++n) {
            d.dims[n - 1] = 0;
            d.H[n - 1] = nullptr;
          }
          d.H[0] = t.H[0];
          d.out = t.node[1];
        } else {     // chunk it.y of the columns, Khatri-Rao factors 2..N, a partial of M(1)
          d.nj = t.rows_r;
          d.j0 = it.y * (int)t.jchunk;
          d.j1 = min(J, d.j0 + (int)t.jchunk);
          for (int n = 1; n < kMaxModes; ++n) {
            d.dims[n - 1] = n < d.N ? (int)t.dims[n] : 0;
            d.H[n - 1] = n < d.N ? t.H[n] : nullptr;
          }
          d.out = t.part + (long long)it.y * d.I1 * d.R;
        }
        d.ntile = (d.j1 - d.j0 + d.nj - 1) / d.nj;
        q.X = t.X;
        sm.slot[sl] = q;
      }
      __syncwarp();
      if (lane == 0) mb_arrive(sm.islot_full(sl));
      ++m;
    }
  }
  // no more items
  const int sl = m % kWsItemSlots;
  if (!mb_wait(sm.islot_empty(sl), ((m / kWsItemSlots) & 1) ^ 1, sm.wait, err, 2)) return;
  if (lane == 0) sm.slot[sl].d.w = -1;
  __syncwarp();
  if (lane == 0) mb_arrive(sm.islot_full(sl));
}

// the loader of both streamed kernels: stage headers and dense tiles of
// rows of X_(1)^T; the last item is followed by one stop stage per builder warp
template <typename SM>
__device__ void ws_loader(const SM& sm, int* err) {
  const int lane = threadIdx.x & 31;
  const uint64_t pol = l2_evict_first_policy();
  int n = 0;  // stages posted
  for (int m = 0;; ++m) {
    const int sl = m % kWsItemSlots;
    if (!mb_wait(sm.islot_full(sl), (m / kWsItemSlots) & 1, sm.wait, err, 3)) break;
    const WsDesc& d = sm.slot[sl].d;
    const int w = d.w, I1 = d.I1, nj = d.nj, j0 = d.j0, j1 = d.j1;
    const int ntile = w >= 0 ? d.ntile : kWsBuildWarps;
    const float* X = sm.slot[sl].X;
    const uint32_t word = lane < kWsDescWords ? reinterpret_cast<const uint32_t*>(&d)[lane] : 0u;
    __syncwarp();
    if (lane == 0) mb_arrive(sm.islot_empty(sl));
    bool ok = true;
    for (int k = 0; k < ntile; ++k, ++n) {
      const int s = n % sm.S;
      if (!mb_wait(sm.empty(s), ((n / sm.S) & 1) ^ 1, sm.wait, err, 4)) {
        ok = false;
        break;
      }
      if (lane < kWsDescWords) reinterpret_cast<uint32_t*>(&sm.hdr[s].d)[lane] = word;
      if (lane == 0) sm.hdr[s].k = k;
      if (w >= 0) {
        const int jt = j0 + k * nj, L = min(nj, j1 - jt) * I1;
        const float* src = X + (long long)jt * I1;
        float* dst = sm.xs(s);
        const int L4 = L & ~3;
        for (int e = 4 * lane; e < L4; e += 128) cp_async16_hint(dst + e, src + e, pol);
        if (L4 + lane < L) cp_async4(dst + L4 + lane, src + L4 + lane);
      }
      mb_arrive_cp_async(sm.full(s));
      __syncwarp();
      if (lane == 0) mb_arrive(sm.hfull(s));
    }
    if (!ok || w < 0) break;
  }
  cp_async_wait_all();
}

// Builder warp b forms the Khatri-Rao tiles of stages b, b + 3, b + 6, ...
__device__ void ws_builder(const WsSmem& sm, int* err) {
  const int lane = threadIdx.x & 31;
  const int b = (threadIdx.x >> 5) - 2;
  for (int n = b;; n += kWsBuildWarps) {
    const int s = n % sm.S;
    if (!mb_wait(sm.hfull(s), (n / sm.S) & 1, sm.wait, err, 5)) return;
    const WsHeader& h = sm.hdr[s];
    const int w = h.d.w;
    if (w >= 0) {
      const int R = h.d.R, N = h.d.N, RQB = b_rq(R), lg = __ffs(RQB) - 1;
      const int jt = h.d.j0 + h.k * h.d.nj, njk = min(h.d.nj, h.d.j1 - jt);
      const int ne = njk * RQB;
      float4* W = reinterpret_cast<float4*>(sm.xs(s) + kTileFloats);
      for (int rd = 0; rd < kWsBuildPasses; ++rd) {
        const int e0 = lane + 32 * kWsBuildPer * rd;
        if (e0 >= ne) break;
        // every entry of this pass at once, so that the factor-row loads of
        // all of them are in flight together
        float4 v[kWsBuildPer];
        int rem[kWsBuildPer];
#pragma unroll
        for (int u = 0; u < kWsBuildPer; ++u) {
          rem[u] = jt + ((e0 + 32 * u) >> lg);
          v[u] = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
        }
        for (int m = 1; m < N; ++m) {
          const int dm = h.d.dims[m - 1];
          const float* Hm = h.d.H[m - 1];
#pragma unroll
          for (int u = 0; u < kWsBuildPer; ++u) {
            const int e = e0 + 32 * u;
            if (e < ne) {
              const int jm = rem[u] % dm;
              rem[u] /= dm;
              const float4 hv = ld_rank4(Hm + jm * R, 4 * (e & (RQB - 1)), R);
              v[u].x *= hv.x;
              v[u].y *= hv.y;
              v[u].z *= hv.z;
              v[u].w *= hv.w;
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kWsBuildPer; ++u) {
          const int e = e0 + 32 * u;
          if (e < ne) W[e] = v[u];
        }
      }
    }
    __syncwarp();
    if (lane == 0) mb_arrive(sm.full(s));
    if (w < 0) return;
  }
}

// One item's tiles (the first already waited for), then its group sum.
// false: a wait expired.
template <int RQB>
__device__ bool ws_consume(const WsDesc& d, int& n, int& nred, int& nsync, const WsSmem& sm,
                           int* err) {
  const int ct = threadIdx.x - 32 * kWsConsFirstWarp;  // 0 .. 255
  const int lane = threadIdx.x & 31;
  const int R = d.R, I1 = d.I1, nj = d.nj, j0 = d.j0, j1 = d.j1, ntile = d.ntile;
  float* out = d.out;
  const int G = kGroupThreads / I1;
  const int g = ct / I1, i = ct - g * I1;
  const bool act = g < G;
  float acc[RQB][4];
#pragma unroll
  for (int u = 0; u < RQB; ++u)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[u][b] = 0.0f;
  int s = 0;
  for (int k = 0; k < ntile; ++k, ++n) {
    s = n % sm.S;
    if (k > 0 && !mb_wait(sm.full(s), (n / sm.S) & 1, sm.wait, err, 6)) return false;
    const int jt = j0 + k * nj, njk = min(nj, j1 - jt);
    if (act) {
      const float* xp = sm.xs(s) + i;
      const float4* W4 = reinterpret_cast<const float4*>(sm.xs(s) + kTileFloats);
#pragma unroll 2
      for (int jj = g; jj < njk; jj += G) {
        const float x = xp[jj * I1];
#pragma unroll
        for (int u = 0; u < RQB; ++u) fma4(acc[u], x, W4[jj * RQB + u]);
      }
    }
    if (k + 1 < ntile || G == 1) {
      __syncwarp();
      if (lane == 0) mb_arrive(sm.empty(s));
    }
  }
  if (G > 1) {
    // column groups added in group order, through the last stage's tile area
    // (still held), up to 4 rank groups at a time, once every consumer warp
    // is done reading that tile
    __syncwarp();
    if (lane == 0) mb_arrive(sm.cons_sync());
    if (!mb_wait(sm.cons_sync(), nsync & 1, sm.wait, err, 7)) return false;
    ++nsync;
    float4* red = reinterpret_cast<float4*>(sm.xs(s));
#pragma unroll
    for (int u0 = 0; u0 < RQB; u0 += 4) {
      const uint32_t par = nred & 1;
      ++nred;
      if (u0 > 0 && !mb_wait(sm.red_empty(), par ^ 1, sm.wait, err, 8)) return false;
      if (act) {
#pragma unroll
        for (int u = u0; u < u0 + 4 && u < RQB; ++u)
          red[(u - u0) * kThreads + ct] = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
      }
      __syncwarp();
      if (lane == 0) mb_arrive(sm.red_full());
      if ((ct & ~31) < I1 && !mb_wait(sm.red_full(), par, sm.wait, err, 9)) return false;  // warps with readers
      if (ct < I1) {
#pragma unroll
        for (int u = u0; u < u0 + 4 && u < RQB; ++u) {
          float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
          for (int gg = 0; gg < G; ++gg) {
            const float4 v = red[(u - u0) * kThreads + gg * I1 + ct];
            s4[0] += v.x;
            s4[1] += v.y;
            s4[2] += v.z;
            s4[3] += v.w;
          }
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (4 * u + b < R) out[ct * R + 4 * u + b] = s4[b];
        }
      }
      __syncwarp();
      if (lane == 0) mb_arrive(sm.red_empty());
    }
    __syncwarp();
    if (lane == 0) mb_arrive(sm.empty(s));
  } else if (act) {
#pragma unroll
    for (int u = 0; u < RQB; ++u)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (4 * u + b < R) out[i * R + 4 * u + b] = acc[u][b];
  }
  return true;
}

template <int RMAX>
__device__ void ws_consumer(const WsSmem& sm, int* err) {
  int nred = 0, nsync = 0;
  for (int n = 0;;) {
    const int s = n % sm.S;
    if (!mb_wait(sm.full(s), (n / sm.S) & 1, sm.wait, err, 10)) return;
    const WsDesc& d = sm.hdr[s].d;
    if (d.w < 0) return;
    bool ok = true;
    switch (b_rq(d.R)) {
      case 1: ok = ws_consume<1>(d, n, nred, nsync, sm, err); break;
      case 2: ok = ws_consume<2>(d, n, nred, nsync, sm, err); break;
      case 4: ok = ws_consume<4>(d, n, nred, nsync, sm, err); break;
      case 8: if constexpr (RMAX >= 32) ok = ws_consume<8>(d, n, nred, nsync, sm, err); break;
      default: if constexpr (RMAX >= 64) ok = ws_consume<16>(d, n, nred, nsync, sm, err); break;
    }
    if (!ok) return;
  }
}

template <int RMAX>
__global__ void __launch_bounds__(kWsThreads, RMAX <= 16 ? 2 : 1)
k_b_pm_right_ws(const BTensor* __restrict__ ts, const int4* __restrict__ items, int n_items,
                int* queue, int S, int* err, long long wait_cycles) {
  extern __shared__ __align__(16) float smem[];
  WsSmem sm;
  sm.S = S;
  sm.wait = wait_cycles > 0 ? wait_cycles : kWsWaitCycles;
  sm.stage0 = smem;
  sm.hdr = reinterpret_cast<WsHeader*>(smem + (size_t)S * kWsStageFloats);
  sm.slot = reinterpret_cast<WsSlot*>(sm.hdr + S);
  sm.bar0 = smem_u32(sm.slot + kWsItemSlots);
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mb_init(sm.full(s), 32 + 1);  // the loader lanes' copies + the stage's builder warp
      mb_init(sm.empty(s), kWsConsWarps);
      mb_init(sm.hfull(s), 1);
    }
    for (int i = 0; i < kWsItemSlots; ++i) {
      mb_init(sm.islot_full(i), 1);
      mb_init(sm.islot_empty(i), 1);
    }
    mb_init(sm.red_full(), kWsConsWarps);
    mb_init(sm.red_empty(), kWsConsWarps);
    mb_init(sm.cons_sync(), kWsConsWarps);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp == 0)
    ws_scheduler<false>(ts, items, n_items, queue, sm, err);
  else if (warp == 1)
    ws_loader(sm, err);
  else if (warp < kWsConsFirstWarp)
    ws_builder(sm, err);
  else
    ws_consumer<RMAX>(sm, err);
}

// M = sum of a phase's partial chunks in chunk order.  Item (tensor, block of
// kReduceBlock outputs, a): a = 0 sums the root -> {1} partials (M(1)),
// a >= 1 the leaf partials of node {a..N} (M(a)).
__global__ void __launch_bounds__(kReduceBlock) k_b_reduce(const BTensor* __restrict__ ts,
                                                           const int4* __restrict__ items) {
  const int4 it = items[blockIdx.x];
  const BTensor& t = ts[it.x];
  if (tensor_done(t)) return;
  const int a = it.z;
  const int E = (int)t.dims[a] * t.R;
  const int nparts = a == 0 ? t.nchunk : t.leaf_nkc[a];
  const float* src = a == 0 ? t.part : t.lpart;
  const int e = it.y * kReduceBlock + threadIdx.x;
  if (e < E) {
    float s = 0.0f;
#pragma unroll 4
    for (int c = 0; c < nparts; ++c) s += src[(long long)c * E + e];
    t.M[e] = s;
  }
}

constexpr int kLeftStageFloats = kTileFloats + kLeftMaxRows;  // rows at odd stride

// groups that split the i range of a tile's (row, rank group) pairs
__device__ __forceinline__ int left_groups(int I1, int R) {
  const int P = b_rows_left(I1) * (b_rq(R) / b_rqb_left(I1, R));
  return P >= kGroupThreads ? 1 : kGroupThreads / P;
}

// root -> node {2..N}: T(j, r) = sum_i X[i + I1 j] H_1(i, r).  Item (tensor,
// kLeftItemTiles tiles of rows j); H_1 (rank padded to b_rank_pad(R) with
// zeros) sits in shared memory.  The sums' order: where a tile has fewer than 256
// (row, rank group) pairs the i range is split over G groups added in group order.
//
// Shared memory returns 128 bytes per cycle and SM however few of them differ, so
// the kernel is bound by what its threads read: a thread with one row and one rank
// group reads five floats for four FMAs.  Here it holds four rows x four ranks in
// registers, eight floats for sixteen FMAs.  128 threads take two tiles at a time,
// single-buffered: five CTAs per SM hide each other's copies, where double buffering
// left two warps each.  Rows are read one, two or four floats at a time, whichever
// divides I_1, so that dense 16-byte copies leave no bank conflicts (a row of 8 k
// floats is padded by four).  (1024 tensors of 16 to 128 per mode at ranks 4, 8 and
// 16, 629 MB: one row per thread behind 4-byte copies to an odd stride 350 us, four
// rows double-buffered 259 us, this 175 us.)
constexpr int kLeftThreads = 128;
constexpr int kLeftTiles = 2;  // tiles in shared memory
// H_1 with an entry more per rank group
__host__ __device__ constexpr int left_h_floats(int hs_floats) { return hs_floats + kBatchMaxRank; }

// floats from row to row of a tile in shared memory
__device__ __forceinline__ int left_stride(int I1, int nj) {
  return (I1 & 7) == 0 && nj * (I1 + 4) <= kLeftTiles * kLeftStageFloats ? I1 + 4 : I1;
}

// hp: this rank group's entries of H_1, one per i; xp: the first of four rows, ST apart
template <int V>
__device__ __forceinline__ void left_rows(const float* xp, int ST, const float4* hp, int ia, int ib,
                                          float (&a)[4][4]) {
  const float* x0 = xp;
  const float* x1 = x0 + ST;
  const float* x2 = x1 + ST;
  const float* x3 = x2 + ST;
#pragma unroll
  for (int t = 0; t < 4; ++t) a[t][0] = a[t][1] = a[t][2] = a[t][3] = 0.0f;
  auto one = [&](int i) {
    const float4 h = hp[i];
    fma4(a[0], x0[i], h);
    fma4(a[1], x1[i], h);
    fma4(a[2], x2[i], h);
    fma4(a[3], x3[i], h);
  };
  int i = ia;
  if (V > 1) {
#pragma unroll 1
    for (; i < ib && (i & (V - 1)); ++i) one(i);
    using W = typename std::conditional<V == 4, float4, float2>::type;
#pragma unroll (V == 2 ? 4 : 2)
    for (; i + V <= ib; i += V) {
      W w[4];
      w[0] = *reinterpret_cast<const W*>(x0 + i);
      w[1] = *reinterpret_cast<const W*>(x1 + i);
      w[2] = *reinterpret_cast<const W*>(x2 + i);
      w[3] = *reinterpret_cast<const W*>(x3 + i);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float4 h = hp[i + v];
#pragma unroll
        for (int t = 0; t < 4; ++t) fma4(a[t], reinterpret_cast<const float*>(&w[t])[v], h);
      }
    }
#pragma unroll 1
    for (; i < ib; ++i) one(i);
  } else {
#pragma unroll 4
    for (; i < ib; ++i) one(i);
  }
}

__device__ __forceinline__ void left_copy(float* Xs, const float* __restrict__ src, int rows, int I1, int S) {
  const int L = rows * I1, L4 = L & ~3;
  if (S == I1) {
#pragma unroll 4
    for (int e = 4 * (int)threadIdx.x; e < L4; e += 4 * kLeftThreads) cp_async16(Xs + e, src + e);
    const int tail = L4 + (int)threadIdx.x;
    if (tail < L) cp_async4(Xs + tail, src + tail);
    return;
  }
  const int n4 = I1 >> 2;  // chunks per row
  const int drow = kLeftThreads / n4, dc = kLeftThreads - drow * n4;
  int row = threadIdx.x / n4, c = threadIdx.x - row * n4;
#pragma unroll 4
  for (int e = threadIdx.x; e < L4 >> 2; e += kLeftThreads) {
    cp_async16(Xs + row * S + 4 * c, src + 4 * e);
    row += drow;
    c += dc;
    if (c >= n4) {
      c -= n4;
      ++row;
    }
  }
}

__device__ __forceinline__ void pm_left_item(const BTensor& t, int item, float* smem) {
  float* Xs = smem;
  float* Hs = smem + kLeftTiles * kLeftStageFloats;  // padded rank x I1
  const int tid = threadIdx.x;
  const int R = t.R, Rq = b_rq(R), Rp = 4 * Rq;
  const int I1 = (int)t.dims[0];
  const int nj = kLeftTiles * t.rows_l, Jq = nj >> 2;
  const int S = left_stride(I1, nj);
  const int J = (int)(t.I / I1);
  const int jb0 = item * t.rows_l * kLeftItemTiles;
  const int jb1 = min(J, jb0 + t.rows_l * kLeftItemTiles);
  const int G = left_groups(I1, R);
  const int P = nj * Rq;
  // thread = (rows jl + x Jq, rank group qb, group g); a pass covers 128 / Rq rows jl
  // of G = 1, everything when G > 1 (then P G <= 512)
  const int lg = __ffs(Rq) - 1, qb = tid & (Rq - 1);
  const int g = G > 1 ? (tid >> lg) / Jq : 0;
  const int jl0 = (tid >> lg) - g * Jq;
  const int ia = g * I1 / G, ib = min(g + 1, G) * I1 / G;
  const int HT = I1 | 1;  // entries from rank group to rank group (no bank conflicts)
  const float4* hp = reinterpret_cast<const float4*>(Hs) + qb * HT;
  {
    const float* H1 = t.H[0];
    if (R == Rp) {
      for (int v = tid; v < I1 * Rq; v += kLeftThreads)
        cp_async16(Hs + 4 * ((v & (Rq - 1)) * HT + (v >> lg)), H1 + 4 * v);
    } else {
      for (int e = tid; e < I1 * Rp; e += kLeftThreads) {
        const int i = e >> (lg + 2), r = e & (Rp - 1);
        Hs[4 * ((r >> 2) * HT + i) + (r & 3)] = r < R ? __ldg(H1 + i * R + r) : 0.0f;
      }
    }
  }
  float* T = t.node[1];
  const int ntile = (jb1 - jb0 + nj - 1) / nj;
  for (int k = 0; k < ntile; ++k) {
    const int jt = jb0 + k * nj, njk = min(nj, jb1 - jt);
    left_copy(Xs, t.X + (long long)jt * I1, njk, I1, S);
    cp_async_wait_all();
    __syncthreads();
    float a[4][4];
    for (int jl = jl0; jl < Jq && g < G; jl += kLeftThreads >> lg) {
      const float* xp = Xs + jl * S;
      if ((I1 & 3) == 0)
        left_rows<4>(xp, Jq * S, hp, ia, ib, a);
      else if ((I1 & 1) == 0)
        left_rows<2>(xp, Jq * S, hp, ia, ib, a);
      else
        left_rows<1>(xp, Jq * S, hp, ia, ib, a);
      if (G > 1) break;
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        if (jl + x * Jq < njk) store_rank4(T + (long long)(jt + jl + x * Jq) * R, qb, R, a[x]);
      }
    }
    __syncthreads();
    if (G > 1) {  // the groups' sums through the tile's own space
      float4* red = reinterpret_cast<float4*>(Xs);
      if (g < G) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          red[g * P + (jl0 + x * Jq) * Rq + qb] = make_float4(a[x][0], a[x][1], a[x][2], a[x][3]);
        }
      }
      __syncthreads();
      for (int e = tid; e < njk * Rq; e += kLeftThreads) {
        float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int gg = 0; gg < G; ++gg) {
          const float4 w = red[gg * P + e];
          s4[0] += w.x;
          s4[1] += w.y;
          s4[2] += w.z;
          s4[3] += w.w;
        }
        store_rank4(T + (long long)(jt + (e >> lg)) * R, e & (Rq - 1), R, s4);
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kLeftThreads)
k_b_pm_left(const BTensor* __restrict__ ts, const int4* __restrict__ items, int n_items,
            int* queue) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int slot;
  for (int w = next_item(queue, n_items, &slot, true); w >= 0;
       w = next_item(queue, n_items, &slot, false)) {
    const int4 it = items[w];
    const BTensor& t = ts[it.x];
    if (tensor_done(t)) continue;
    pm_left_item(t, it.y, smem);
  }
}

// ------------------------------------ streamed root -> {2..N} (schedule 2) --
//
// The arithmetic of pm_left_item (same sums in the same order, so the same
// bits) with its jobs split over the warps of a persistent CTA, built from
// the parts of the streamed root -> {1} kernel:
//   warp 0, scheduler and warp 1, loader: as there (ws_scheduler<true>,
//                      ws_loader): dense tiles of rows of X_(1)^T into a ring
//                      of SD stages;
//   warps 2-4, builders: take the dense stages in turn; at an item's first
//                      tile stage H_1 (rank padded with zeros) into one of two
//                      H slots; copy the tile to the odd row stride S = I_1 | 1
//                      (conflict-free column reads) into a ring of SO stages,
//                      with the header; free the dense stage;
//   warps 5-12, consumers (256 threads): the (row, rank
//                      block) passes over each odd-stride tile, group sums
//                      through a small buffer, rows of T written out; an odd
//                      stage is freed after its tile, an H slot after its item.
// Waits: mbarriers, warp-uniform and bounded, an error word.

struct WlHeader {
  WsDesc d;
  int k;      // tile within the item
  int hslot;  // H slot of the item
  int pad[2];
};
static_assert(sizeof(WlHeader) % 16 == 0, "header layout");

// Shared-memory counter helpers: a consumer warp's release of an odd stage,
// and the builder's bounded, warp-uniform wait for a number of releases
// (an exact count: builders fill the odd ring out of order, so a parity wait
// could pass on a phase two laps old).
__device__ __forceinline__ void smem_add_release(const unsigned* p, unsigned v) {
  asm volatile("red.release.cta.shared::cta.add.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned smem_ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ bool count_wait(const unsigned* p, unsigned target, long long limit,
                                           int* err, int site) {
  if (__all_sync(0xffffffffu, smem_ld_acquire(p) >= target)) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, smem_ld_acquire(p) >= target)) {
    if (clock64() - t0 > limit) {
      if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, 1 + site);
      return false;
    }
  }
  return true;
}

struct WlSmem {
  float* stage0;  // SD dense stages of kTileFloats
  float* odd0;    // SO odd-stride stages of kLeftStageFloats
  float* hs0;     // two H slots of hs_floats
  float4* red;    // kThreads
  WsHeader* hdr;  // SD (dense, written by the loader)
  WlHeader* ohdr; // SO (odd, written by the builders)
  WsSlot* slot;
  unsigned* ocons;  // SO: consumer-warp releases of each odd stage so far
  uint32_t bar0;
  int S, SO, hs_floats;
  long long wait;
  __device__ float* xs(int s) const { return stage0 + (size_t)s * kTileFloats; }
  __device__ float* os(int o) const { return odd0 + (size_t)o * kLeftStageFloats; }
  __device__ float* hs(int h) const { return hs0 + (size_t)h * hs_floats; }
  __device__ uint32_t full(int s) const { return bar0 + 8u * s; }
  __device__ uint32_t empty(int s) const { return bar0 + 8u * (S + s); }
  __device__ uint32_t hfull(int s) const { return bar0 + 8u * (2 * S + s); }
  __device__ uint32_t ofull(int o) const { return bar0 + 8u * (3 * S + o); }
  __device__ uint32_t islot_full(int i) const { return bar0 + 8u * (3 * S + SO + i); }
  __device__ uint32_t islot_empty(int i) const { return bar0 + 8u * (3 * S + SO + kWsItemSlots + i); }
  __device__ uint32_t hslot_empty(int h) const {
    return bar0 + 8u * (3 * S + SO + 2 * kWsItemSlots + h);
  }
  __device__ uint32_t red_full() const { return bar0 + 8u * (3 * S + SO + 2 * kWsItemSlots + 2); }
  __device__ uint32_t red_empty() const { return bar0 + 8u * (3 * S + SO + 2 * kWsItemSlots + 3); }
  __host__ __device__ static constexpr int bars(int S, int SO) { return 3 * S + SO + 2 * kWsItemSlots + 4; }
};

__host__ __device__ constexpr size_t wl_smem_bytes(int S, int SO, int hs_floats) {
  return (size_t)S * kTileFloats * sizeof(float) + (size_t)SO * kLeftStageFloats * sizeof(float) +
         2 * (size_t)hs_floats * sizeof(float) + (size_t)kThreads * sizeof(float4) +
         (size_t)S * sizeof(WsHeader) + (size_t)SO * sizeof(WlHeader) +
         (size_t)kWsItemSlots * sizeof(WsSlot) + (size_t)WlSmem::bars(S, SO) * sizeof(uint64_t) +
         (size_t)((SO + 1) / 2) * sizeof(uint64_t);
}

// Builder warp b handles dense stages b, b + 3, b + 6, ...; dense stage n
// becomes odd stage n % SO.
__device__ void wl_builder(const WlSmem& sm, int* err) {
  const int lane = threadIdx.x & 31;
  const int b = (threadIdx.x >> 5) - 2;
  for (int n = b;; n += kWsBuildWarps) {
    const int s = n % sm.S, o = n % sm.SO;
    if (!mb_wait(sm.hfull(s), (n / sm.S) & 1, sm.wait, err, 20)) return;
    const WsHeader& h = sm.hdr[s];
    const int w = h.d.w, k = h.k;
    if (w < 0) {
      if (k == 0) {  // the first stop stage ends the odd ring too
        if (!count_wait(sm.ocons + o, kWsConsWarps * (unsigned)(n / sm.SO), sm.wait, err, 21)) return;
        if (lane == 0) sm.ohdr[o].d.w = -1;
        __syncwarp();
        if (lane == 0) mb_arrive(sm.ofull(o));
      }
      return;
    }
    const int I1 = h.d.I1, R = h.d.R, seq = h.d.seq;
    const int jt = h.d.j0 + k * h.d.nj, njk = min(h.d.nj, h.d.j1 - jt);
    const float* H1 = h.d.H[0];
    const uint32_t word = reinterpret_cast<const uint32_t*>(&h.d)[lane];
    if (!mb_wait(sm.full(s), (n / sm.S) & 1, sm.wait, err, 22)) return;
    if (!count_wait(sm.ocons + o, kWsConsWarps * (unsigned)(n / sm.SO), sm.wait, err, 23)) return;
    const int hslot = seq & 1;
    if (k == 0) {  // H_1 of the item, rank padded to Rp with zeros
      if (!mb_wait(sm.hslot_empty(hslot), ((seq >> 1) & 1) ^ 1, sm.wait, err, 24)) return;
      float* hd = sm.hs(hslot);
      const int Rp = b_rank_pad(R);
      for (int e = lane; e < I1 * Rp; e += 32) {
        const int i = e / Rp, r = e - i * Rp;
        hd[e] = r < R ? __ldg(H1 + i * R + r) : 0.0f;
      }
    }
    // the tile at odd row stride: four consecutive elements per lane and step
    const float* src = sm.xs(s);
    float* dst = sm.os(o);
    const int ST = I1 | 1, L = njk * I1, L4 = L & ~3;
    int row = (4 * lane) / I1, col = 4 * lane - row * I1;
    const int drow = 128 / I1, dcol = 128 - drow * I1;
    for (int e = 4 * lane; e < L4; e += 128) {
      const float4 v = *reinterpret_cast<const float4*>(src + e);
      int r = row, c = col;
      dst[r * ST + c] = v.x;
      if (++c == I1) c = 0, ++r;
      dst[r * ST + c] = v.y;
      if (++c == I1) c = 0, ++r;
      dst[r * ST + c] = v.z;
      if (++c == I1) c = 0, ++r;
      dst[r * ST + c] = v.w;
      row += drow;
      col += dcol;
      if (col >= I1) {
        col -= I1;
        ++row;
      }
    }
    if (L4 + lane < L) {
      const int e = L4 + lane, r = e / I1;
      dst[r * ST + (e - r * I1)] = src[e];
    }
    reinterpret_cast<uint32_t*>(&sm.ohdr[o].d)[lane] = word;
    if (lane == 0) {
      sm.ohdr[o].k = k;
      sm.ohdr[o].hslot = hslot;
    }
    __syncwarp();
    if (lane == 0) {
      mb_arrive(sm.empty(s));  // the dense stage has been read
      mb_arrive(sm.ofull(o));  // the odd stage, its header and the H slot are written
    }
  }
}

// One item of root -> {2..N} (its first odd stage already waited for).
template <int RQB>
__device__ bool wl_consume(const WlHeader& h0, int& n, int& nred, const WlSmem& sm, int* err) {
  const int ct = threadIdx.x - 32 * kWsConsFirstWarp;  // 0 .. 255
  const int lane = threadIdx.x & 31;
  const WsDesc& d = h0.d;
  const int R = d.R, I1 = d.I1, nj = d.nj, jb0 = d.j0, jb1 = d.j1, ntile = d.ntile;
  const int hslot = h0.hslot;
  float* T = d.out;
  const int Rq = b_rq(R), ST = I1 | 1;
  const int NB = Rq / RQB;
  const int P = nj * NB;
  const int G = P >= kGroupThreads ? 1 : kGroupThreads / P;
  const int npass = (P + kThreads - 1) / kThreads;
  const int g = G > 1 ? ct / P : 0;
  const int ia = g * I1 / G, ib = (g + 1) * I1 / G;
  const float4* H4 = reinterpret_cast<const float4*>(sm.hs(hslot));
  for (int k = 0; k < ntile; ++k, ++n) {
    const int o = n % sm.SO;
    if (k > 0 && !mb_wait(sm.ofull(o), (n / sm.SO) & 1, sm.wait, err, 25)) return false;
    const int jt = jb0 + k * nj, njk = min(nj, jb1 - jt);
    const float* Xs = sm.os(o);
    for (int p = 0; p < npass; ++p) {
      const int pair = G > 1 ? ct - g * P : ct + kThreads * p;
      const int jl = pair / NB, qb = pair - jl * NB;
      const bool v = g < G && pair < P && jl < njk;
      float a[RQB][4];
#pragma unroll
      for (int u = 0; u < RQB; ++u)
#pragma unroll
        for (int b = 0; b < 4; ++b) a[u][b] = 0.0f;
      if (v) {
        const float* xp = Xs + jl * ST;
        const float4* hp = H4 + qb * RQB;
#pragma unroll 4
        for (int i = ia; i < ib; ++i) {
          const float x = xp[i];
#pragma unroll
          for (int u = 0; u < RQB; ++u) fma4(a[u], x, hp[i * Rq + u]);
        }
      }
      if (G > 1) {  // RQB == 1 here
        const uint32_t par = nred & 1;
        ++nred;
        if (!mb_wait(sm.red_empty(), par ^ 1, sm.wait, err, 26)) return false;
        if (g < G) sm.red[ct] = make_float4(a[0][0], a[0][1], a[0][2], a[0][3]);
        __syncwarp();
        if (lane == 0) mb_arrive(sm.red_full());
        if ((ct & ~31) < P && !mb_wait(sm.red_full(), par, sm.wait, err, 27)) return false;
        if (ct < P) {
          const int jl0 = ct / NB, q0 = ct - jl0 * NB;
          if (jl0 < njk) {
            float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            for (int gg = 0; gg < G; ++gg) {
              const float4 wv = sm.red[gg * P + ct];
              s4[0] += wv.x;
              s4[1] += wv.y;
              s4[2] += wv.z;
              s4[3] += wv.w;
            }
#pragma unroll
            for (int b = 0; b < 4; ++b)
              if (4 * q0 + b < R) T[(long long)(jt + jl0) * R + 4 * q0 + b] = s4[b];
          }
        }
        __syncwarp();
        if (lane == 0) mb_arrive(sm.red_empty());
      } else if (v) {
#pragma unroll
        for (int u = 0; u < RQB; ++u)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int r = 4 * (qb * RQB + u) + b;
            if (r < R) T[(long long)(jt + jl) * R + r] = a[u][b];
          }
      }
    }
    __syncwarp();
    if (lane == 0) smem_add_release(sm.ocons + o, 1u);
  }
  __syncwarp();
  if (lane == 0) mb_arrive(sm.hslot_empty(hslot));
  return true;
}

template <int RMAX>
__device__ void wl_consumer(const WlSmem& sm, int* err) {
  int nred = 0;
  for (int n = 0;;) {
    const int o = n % sm.SO;
    if (!mb_wait(sm.ofull(o), (n / sm.SO) & 1, sm.wait, err, 28)) return;
    const WlHeader& h = sm.ohdr[o];
    if (h.d.w < 0) return;
    bool ok = true;
    switch (b_rqb_left(h.d.I1, h.d.R)) {
      case 1: ok = wl_consume<1>(h, n, nred, sm, err); break;
      case 2: ok = wl_consume<2>(h, n, nred, sm, err); break;
      case 4: ok = wl_consume<4>(h, n, nred, sm, err); break;
      case 8: if constexpr (RMAX >= 32) ok = wl_consume<8>(h, n, nred, sm, err); break;
      default: if constexpr (RMAX >= 64) ok = wl_consume<16>(h, n, nred, sm, err); break;
    }
    if (!ok) return;
  }
}

template <int RMAX>
__global__ void __launch_bounds__(kWsThreads, RMAX <= 16 ? 2 : 1)
k_b_pm_left_ws(const BTensor* __restrict__ ts, const int4* __restrict__ items, int n_items,
               int* queue, int S, int SO, int hs_floats, int* err, long long wait_cycles) {
  extern __shared__ __align__(16) float smem[];
  WlSmem sm;
  sm.S = S;
  sm.SO = SO;
  sm.hs_floats = hs_floats;
  sm.wait = wait_cycles > 0 ? wait_cycles : kWsWaitCycles;
  sm.stage0 = smem;
  sm.odd0 = smem + (size_t)S * kTileFloats;
  sm.hs0 = sm.odd0 + (size_t)SO * kLeftStageFloats;
  sm.red = reinterpret_cast<float4*>(sm.hs0 + 2 * (size_t)hs_floats);
  sm.hdr = reinterpret_cast<WsHeader*>(sm.red + kThreads);
  sm.ohdr = reinterpret_cast<WlHeader*>(sm.hdr + S);
  sm.slot = reinterpret_cast<WsSlot*>(sm.ohdr + SO);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm.slot + kWsItemSlots);
  sm.bar0 = smem_u32(bars);
  sm.ocons = reinterpret_cast<unsigned*>(bars + WlSmem::bars(S, SO));
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mb_init(sm.full(s), 32);  // the loader lanes' copies
      mb_init(sm.empty(s), 1);  // the builder warp of the stage
      mb_init(sm.hfull(s), 1);  // the loader's header
    }
    for (int o = 0; o < SO; ++o) {
      mb_init(sm.ofull(o), 1);  // the builder warp of the stage
      sm.ocons[o] = 0u;
    }
    for (int i = 0; i < kWsItemSlots; ++i) {
      mb_init(sm.islot_full(i), 1);
      mb_init(sm.islot_empty(i), 1);
    }
    mb_init(sm.hslot_empty(0), kWsConsWarps);
    mb_init(sm.hslot_empty(1), kWsConsWarps);
    mb_init(sm.red_full(), kWsConsWarps);
    mb_init(sm.red_empty(), kWsConsWarps);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp == 0)
    ws_scheduler<true>(ts, items, n_items, queue, sm, err);
  else if (warp == 1)
    ws_loader(sm, err);
  else if (warp < kWsConsFirstWarp)
    wl_builder(sm, err);
  else
    wl_consumer<RMAX>(sm, err);
}

// ---------------------------------------------------------- multi-TTVs --

// leaf M(a) from node {a..N} (Fig. 1): M(i, r) = sum_k T[(i + I_a k) R + r] KK(k, r),
// KK = H_N (.) ... (.) H_{a+1}.  Item (tensor, chunk c of leaf_kc[a] rows k,
// block of kLeafBlock outputs).  For each k the node slice of all (i, r) is
// contiguous, so threads read it coalesced, V outputs each (V = 4 when R % 4 == 0);
// where a slice has at most 128 such reads, G groups of threads take the rows
// k = g, g + G, ... of a tile and their sums are added in group order at the end.  KK
// rows are formed per tile of kLeafTileK rows in shared memory, the rows' digits kept
// by addition.  Bound by the latency of the node's loads: a thread per output and a
// division per KK entry and mode left 10 x 8 slices to 80 threads.  Writes lpart[c].
// (1500 tensors of four modes of 4 to 40, ranks 4, 8, 16: 364 us, this 87 us; 1024 of
// three modes of 16 to 128 53 and 39 us; at six CTAs per SM, with 42 registers, 108 and 56.)
template <int V>
__device__ __forceinline__ void leaf_item(const BTensor& t, int a, int chunk, int block, float* KKs) {
  using VT = typename std::conditional<V == 4, float4, float>::type;
  constexpr int T = 256, Q = kLeafBlock / (T * V);
  const int tid = threadIdx.x;
  const int R = t.R, RV = R / V, N = t.N;
  const int E = (int)t.dims[a] * R;
  int K = 1;
  for (int m = a + 1; m < N; ++m) K *= (int)t.dims[m];
  const int kc = t.leaf_kc[a];
  const int k0 = chunk * kc, k1 = min(K, k0 + kc);
  const int U = min(kLeafBlock, E - block * kLeafBlock) / V;  // reads of a row
  const int G = U <= T / 2 ? T / U : 1;
  const int g = G > 1 ? tid / U : 0, u0 = tid - g * U;
  int rp[Q];
  __align__(16) float acc[Q][V];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    rp[q] = (block * kLeafBlock / V + u0 + T * q) % RV;
#pragma unroll
    for (int v = 0; v < V; ++v) acc[q][v] = 0.0f;
  }
  // this thread's KK entries: rank group kr of rows kk, kk + step, ... of a tile
  const int step = T / RV, kk0 = tid / RV, kr = (tid - kk0 * RV) * V;
  const int d = (int)t.dims[a + 1];
  int dig = 0, rest = 0, sd = 0, sr = 0;  // digit of mode a + 1 and the rest; per step
  const bool build = kk0 < step;
  if (build) {
    rest = (k0 + kk0) / d;
    dig = k0 + kk0 - rest * d;
    sr = step / d;
    sd = step - sr * d;
  }
  const int tr = kLeafTileK / d, td = kLeafTileK - tr * d;  // per tile
  const float* Ha = t.H[a + 1] + kr;
  const float* node = t.node[a] + block * kLeafBlock;
  for (int kt = k0; kt < k1; kt += kLeafTileK) {
    const int nk = min(kLeafTileK, k1 - kt);
    __syncthreads();
    if (build) {
      int x = dig, y = rest;
#pragma unroll 2
      for (int kk = kk0; kk < nk; kk += step) {
        VT w = __ldg(reinterpret_cast<const VT*>(Ha + x * R));
        float* wf = reinterpret_cast<float*>(&w);
        unsigned rem = (unsigned)y;
        for (int m = a + 2; m < N; ++m) {
          unsigned jm = rem;
          if (m + 1 < N) {
            const unsigned dm = (unsigned)t.dims[m];
            rem = jm / dm;
            jm -= rem * dm;
          }
          const VT h = __ldg(reinterpret_cast<const VT*>(t.H[m] + (int)jm * R + kr));
          const float* hf = reinterpret_cast<const float*>(&h);
#pragma unroll
          for (int v = 0; v < V; ++v) wf[v] *= hf[v];
        }
        *reinterpret_cast<VT*>(KKs + kk * R + kr) = w;
        kr_step(x, y, sd, sr, d);
      }
      kr_step(dig, rest, td, tr, d);
    }
    __syncthreads();
    const float* Tb = node + (long long)(kt + g) * E + u0 * V;
    const float* Kb = KKs + g * R;
    if (g < G) {
#pragma unroll 4
      for (int kk = g; kk < nk; kk += G, Tb += G * E, Kb += G * R) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
          if (u0 + T * q < U) {
            const VT x = *reinterpret_cast<const VT*>(Tb + T * V * q);
            const VT w = *reinterpret_cast<const VT*>(Kb + rp[q] * V);
            const float* xf = reinterpret_cast<const float*>(&x);
            const float* wf = reinterpret_cast<const float*>(&w);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[q][v] = fmaf(xf[v], wf[v], acc[q][v]);
          }
      }
    }
  }
  float* out = t.lpart + (long long)chunk * E + block * kLeafBlock;
  if (G > 1) {
    __syncthreads();
    if (g < G) *reinterpret_cast<VT*>(KKs + tid * V) = *reinterpret_cast<const VT*>(acc[0]);
    __syncthreads();
    if (tid < U) {
#pragma unroll 1
      for (int h = 1; h < G; ++h)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[0][v] += KKs[(h * U + tid) * V + v];
      *reinterpret_cast<VT*>(out + tid * V) = *reinterpret_cast<const VT*>(acc[0]);
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (u0 + T * q < U) *reinterpret_cast<VT*>(out + (u0 + T * q) * V) = *reinterpret_cast<const VT*>(acc[q]);
}

__global__ void __launch_bounds__(256, 4) k_b_mttv_leaf(const BTensor* __restrict__ ts,
                                                     const int4* __restrict__ items, int a) {
  const int4 it = items[blockIdx.x];
  const BTensor& t = ts[it.x];
  if (tensor_done(t)) return;
  __shared__ __align__(16) float KKs[kLeafTileK * kBatchMaxRank];
  if ((t.R & 3) == 0)
    leaf_item<4>(t, a, it.y, it.z, KKs);
  else
    leaf_item<1>(t, a, it.y, it.z, KKs);
}

// child node {a+1..N} from node {a..N}: out(j, r) = sum_i T[(i + I_a j) R + r] H_a(i, r)
// with the updated H_a; the output is M when the child is a leaf.  Item
// (tensor, block of first_jb[a] rows j); warp per row j, four rows at a time.
// Lanes = (i phase, group of V ranks, V = 4 when R % 4 == 0): they read the
// row's I_a x R block coalesced, V floats per load, and their i phases are added
// in a fixed shuffle tree.  Bound by the latency of the node's loads: with one
// rank per lane and two rows in flight it took 107 us for 1024 tensors on a
// GB300 (11 % of the issue slots).
template <int V>
__device__ __forceinline__ void first_rows(const float* __restrict__ T, const float* __restrict__ Ha,
                                           float* __restrict__ out, int R, int Ia, int j0, int j1) {
  constexpr int NR = 4;  // rows in flight
  using VT = typename std::conditional<V == 4, float4, float>::type;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  const int RV = R / V, E = Ia * R;
  for (int rb = 0; rb < RV; rb += 32) {
    const int Rb = min(32, RV - rb), S = 32 / Rb;
    const int sub = lane / Rb, r = (rb + lane - sub * Rb) * V;
    const bool act = sub < S;
    for (int j = j0 + warp; j < j1; j += NR * nwarp) {
      float acc[NR][V];
      const float* Tj[NR];
#pragma unroll
      for (int q = 0; q < NR; ++q) {
        const int jq = j + q * nwarp;
        Tj[q] = T + (long long)(jq < j1 ? jq : j) * E + r;
#pragma unroll
        for (int v = 0; v < V; ++v) acc[q][v] = 0.0f;
      }
      if (act) {
#pragma unroll 4
        for (int i = sub; i < Ia; i += S) {
          const VT hv = __ldg(reinterpret_cast<const VT*>(Ha + i * R + r));
          const float* h = reinterpret_cast<const float*>(&hv);
          VT x[NR];
#pragma unroll
          for (int q = 0; q < NR; ++q) x[q] = *reinterpret_cast<const VT*>(Tj[q] + i * R);
#pragma unroll
          for (int q = 0; q < NR; ++q) {
            const float* xf = reinterpret_cast<const float*>(&x[q]);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[q][v] = fmaf(xf[v], h[v], acc[q][v]);
          }
        }
      }
      for (int o = 1; o < S; o <<= 1) {
        const bool add = act && (sub & (2 * o - 1)) == 0 && sub + o < S;
#pragma unroll
        for (int q = 0; q < NR; ++q)
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const float w = __shfl_down_sync(0xffffffffu, acc[q][v], o * Rb);
            if (add) acc[q][v] += w;
          }
      }
      if (act && sub == 0) {
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          const int jq = j + q * nwarp;
          if (jq < j1) {
#pragma unroll
            for (int v = 0; v < V; ++v) out[(long long)jq * R + r + v] = acc[q][v];
          }
        }
      }
    }
  }
}

__global__ void __launch_bounds__(256) k_b_mttv_first(const BTensor* __restrict__ ts,
                                                      const int4* __restrict__ items, int a) {
  const int4 it = items[blockIdx.x];
  const BTensor& t = ts[it.x];
  if (tensor_done(t)) return;
  const int R = t.R, N = t.N;
  int K = 1;
  for (int m = a + 1; m < N; ++m) K *= (int)t.dims[m];
  const int jb = t.first_jb[a];
  const int j0 = it.y * jb, j1 = min(K, j0 + jb);
  float* out = (a + 1 == N - 1) ? t.M : t.node[a + 1];
  // nodes and factors start on 16-byte boundaries
  if ((R & 3) == 0) first_rows<4>(t.node[a], t.H[a], out, R, (int)t.dims[a], j0, j1);
  else first_rows<1>(t.node[a], t.H[a], out, R, (int)t.dims[a], j0, j1);
}

// ---------------------------------------------------------- mode update --

// One CTA per tensor (I_n <= kBatchMaxI rows, R <= RMAX): HALS sweep
// (Sec. II-B, row per thread, row in registers), W^T W, lambda, G_n,
// H_n = W / lambda, the fit at n = N (Sec. IV-B) with the stopping test, and
// S for the next mode -- all in shared memory.
template <int RMAX>
__global__ void __launch_bounds__(256)
k_b_update(BTensor* __restrict__ ts, int n, int* __restrict__ done_count, int rows) {
  BTensor& t = ts[blockIdx.x];
  if (tensor_done(t)) return;
  constexpr int RP = RMAX + 1;
  const int R = t.R, N = t.N, R2 = R * R;
  const int In = (int)t.dims[n];
  const int tid = threadIdx.x;
  extern __shared__ __align__(16) float bsm[];
  // rows: the longest mode of the batch, so that small tensors leave room for
  // more CTAs per SM
  float* St = bsm;                 // RMAX x RMAX, St[r][c] = S[c][r], zero padded
  float* Ws = St + RMAX * RMAX;    // rows x RP (W, then H)
  float* Ms = Ws + rows * RP;      // rows x RP (M)
  __shared__ float lamf[RMAX], sinv[RMAX];
  __shared__ double GW[RMAX * RMAX];
  __shared__ double cinv[RMAX];
  __shared__ double red[8];
  float* Hn = t.H[n];
  // staging with the global loads of a loop issued in batches
#pragma unroll 4
  for (int e = tid; e < RMAX * RMAX; e += blockDim.x) {
    const int r = e / RMAX, c = e % RMAX;
    St[e] = (r < R && c < R) ? t.S32[c * R + r] : 0.0f;
  }
  for (int r = tid; r < RMAX; r += blockDim.x) {
    lamf[r] = r < R ? (float)t.lam[r] : 0.0f;
    const float srr = r < R ? t.S32[r * R + r] : 0.0f;
    sinv[r] = srr != 0.0f ? 1.0f / srr : 0.0f;
  }
  __syncthreads();
#pragma unroll 4
  for (int e = tid; e < In * R; e += blockDim.x) {
    const int i = e / R, c = e - i * R;
    Ws[i * RP + c] = Hn[e] * lamf[c];
    Ms[i * RP + c] = t.M[e];
  }
  for (int i = tid; i < In; i += blockDim.x)
    for (int c = R; c < RMAX; ++c) Ws[i * RP + c] = 0.0f;
  __syncthreads();
  double bp = 0.0;
  for (int i = tid; i < In; i += blockDim.x) {
    // row W(i, :) updated in place in shared memory (odd stride: one bank per
    // thread); rolled column loop, unrolled dot product (see the HALS sweep
    // of the single-problem update)
    float* wrow = Ws + i * RP;
    const float* mrow = Ms + i * RP;
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
      const float si = sinv[r];
      const float mr = mrow[r];
      float d0 = 0.0f, d1 = 0.0f;
#pragma unroll
      for (int c = 0; c < RMAX; c += 2) {
        d0 = fmaf(wrow[c], St[r * RMAX + c], d0);
        d1 = fmaf(wrow[c + 1], St[r * RMAX + c + 1], d1);
      }
      const float wr = wrow[r];
      const float upd = fmaxf(0.0f, wr + (mr - (d0 + d1)) * si);
      wrow[r] = si != 0.0f ? upd : wr;
    }
    float b = 0.0f;
    for (int c = 0; c < R; ++c) b = fmaf(mrow[c], wrow[c], b);
    bp += (double)b;
  }
  for (int o = 16; o > 0; o >>= 1) bp += __shfl_xor_sync(0xffffffffu, bp, o);
  if ((tid & 31) == 0) red[tid >> 5] = bp;
  __syncthreads();
  for (int e = tid; e < R2; e += blockDim.x) {
    const int a = e / R, b = e % R;
    float s0 = 0.0f, s1 = 0.0f;
    int i = 0;
    for (; i + 1 < In; i += 2) {
      s0 = fmaf(Ws[i * RP + a], Ws[i * RP + b], s0);
      s1 = fmaf(Ws[(i + 1) * RP + a], Ws[(i + 1) * RP + b], s1);
    }
    if (i < In) s0 = fmaf(Ws[i * RP + a], Ws[i * RP + b], s0);
    GW[e] = (double)(s0 + s1);
  }
  __syncthreads();
  for (int r = tid; r < R; r += blockDim.x) {
    const double v = sqrt(GW[r * R + r]);
    t.lam[r] = v;
    cinv[r] = v > 0.0 ? 1.0 / v : 0.0;
    lamf[r] = v > 0.0 ? (float)(1.0 / v) : 0.0f;
  }
  __syncthreads();
  double* Gn = t.G + (long long)n * R2;
  for (int e = tid; e < R2; e += blockDim.x) Gn[e] = GW[e] * cinv[e / R] * cinv[e % R];
  for (int e = tid; e < In * R; e += blockDim.x) Hn[e] = Ws[(e / R) * RP + e % R] * lamf[e % R];
  if (n == N - 1) {
    double g = 0.0;
    for (int e = tid; e < R2; e += blockDim.x) g += t.S[e] * GW[e];
    for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    __syncthreads();
    __shared__ double red2[8];
    if ((tid & 31) == 0) red2[tid >> 5] = g;
    __syncthreads();
    if (tid == 0) {
      double beta = 0.0, gamma = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        beta += red[w];
        gamma += red2[w];
      }
      const double alpha = t.scal[0];
      const double eps = sqrt(fmax(0.0, alpha - 2.0 * beta + gamma) / alpha);
      const double fit = 1.0 - eps;
      const int k = t.flags[1];
      if (k < t.fit_cap) t.fits[k] = fit;
      t.flags[1] = k + 1;
      bool stop = !isfinite(fit) || (k + 1 >= t.max_iters);
      if (!isfinite(fit)) t.flags[2] = 1;
      if (k >= 1 && k - 1 < t.fit_cap && fabs(fit - t.fits[k - 1]) < t.scal[1]) stop = true;
      if (stop) {
        t.flags[0] = 1;
        atomicAdd(done_count, 1);
      }
    }
  }
  __syncthreads();
  const int next = (n + 1) % N;
  for (int e = tid; e < R2; e += blockDim.x) {
    double s = 1.0;
    for (int k = 0; k < N; ++k)
      if (k != next) s *= (k == n) ? Gn[e] : t.G[(long long)k * R2 + e];
    t.S[e] = s;
    t.S32[e] = (float)s;
  }
}

__global__ void k_b_gather(const BTensor* __restrict__ ts, int count, int* iters, double* fits,
                           double* lam, const int* lam_off, int* nonfinite) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < count; b += gridDim.x * blockDim.x) {
    const BTensor& t = ts[b];
    const int k = t.flags[1];
    iters[b] = k;
    fits[b] = (k >= 1 && k <= t.fit_cap) ? t.fits[k - 1] : 0.0;
    nonfinite[b] = (t.flags[2] ? 1 : 0) | (t.flags[0] ? 2 : 0);  // bit 0 non-finite, bit 1 done
    if (lam)
      for (int r = 0; r < t.R; ++r) lam[lam_off[b] + r] = t.lam[r];
  }
}

template <int RMAX>
size_t update_smem(int rows = kBatchMaxI) {
  return (size_t)(RMAX * RMAX + 2 * rows * (RMAX + 1)) * sizeof(float);
}

}  // namespace

cudaError_t batch_attributes_init() {
  cudaError_t e = cudaFuncSetAttribute(k_b_update<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)update_smem<16>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_b_update<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)update_smem<32>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_b_update<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)update_smem<64>());
  const int fac = kBatchMaxI * kBatchMaxRank * (int)sizeof(float);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_init_mode, cudaFuncAttributeMaxDynamicSharedMemorySize, fac);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_init, cudaFuncAttributeMaxDynamicSharedMemorySize, fac);
  const int left = (kLeftTiles * kLeftStageFloats + left_h_floats(kBatchMaxI * kBatchMaxRank)) * (int)sizeof(float);
  int dev = 0, optin = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_right_ws<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_right_ws<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_right_ws<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_left_ws<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_left_ws<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_left_ws<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_b_pm_left, cudaFuncAttributeMaxDynamicSharedMemorySize, left);
  return e;
}

namespace {

// Grid of a root phase: one CTA per item (queue NULL), or one wave of
// persistent CTAs (every CTA that fits at once at this shared-memory size)
// taking items from the counter `queue`.
template <typename K>
int phase_grid(K kernel, int threads, size_t smem, int n_items, const int* queue) {
  if (!queue) return n_items;
  int dev = 0, sms = 1, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  return std::max(1, std::min(n_items, sms * per_sm));
}

}  // namespace

namespace {

// Streamed root -> {1}: as many ring stages (at most 8) as fit at two CTAs per
// SM (RMAX 16) or one, and one wave of CTAs.
template <int RMAX>
cudaError_t launch_pm_right_ws(const BTensor* ts, const int4* it, int n, int* queue, int* err,
                               long long wait_cycles, cudaStream_t st) {
  int dev = 0, sms = 1, smem_sm = 0, reserved = 0, optin = 0, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int want = RMAX <= 16 ? 2 : 1;
  const size_t budget = std::min<size_t>((size_t)optin, (size_t)(smem_sm / want - reserved));
  int S = 8;
  while (S > kWsBuildWarps + 1 && ws_smem_bytes(S) > budget) --S;
  const size_t bytes = ws_smem_bytes(S);
  if (bytes > (size_t)optin) return cudaErrorInvalidConfiguration;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_b_pm_right_ws<RMAX>, kWsThreads,
                                                    bytes) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const int grid = std::max(1, std::min(n, sms * per_sm));
  k_b_pm_right_ws<RMAX><<<grid, kWsThreads, bytes, st>>>(ts, it, n, queue, S, err, wait_cycles);
  return cudaGetLastError();
}

// Streamed root -> {2..N}: the largest dense / odd-stride rings (at least
// three dense stages, one per builder's stop stage) that fit beside the two
// H_1 slots at two CTAs per SM (RMAX 16, when they fit) or one.
template <int RMAX>
cudaError_t launch_pm_left_ws(const BTensor* ts, const int4* it, int n, int* queue, int hs_floats,
                              int* err, long long wait_cycles, cudaStream_t st) {
  int dev = 0, sms = 1, smem_sm = 0, reserved = 0, optin = 0, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  static const int cand[][2] = {{4, 3}, {4, 2}, {3, 3}, {3, 2}};
  int S = 0, SO = 0;
  // two CTAs per SM at ranks <= 16 when the H_1 slots leave room, else one
  for (int want = RMAX <= 16 ? 2 : 1; want >= 1 && S == 0; --want) {
    const size_t budget = std::min<size_t>((size_t)optin, (size_t)(smem_sm / want - reserved));
    for (const auto& c : cand)
      if (wl_smem_bytes(c[0], c[1], hs_floats) <= budget) {
        S = c[0];
        SO = c[1];
        break;
      }
  }
  if (S == 0) return cudaErrorInvalidConfiguration;
  const size_t bytes = wl_smem_bytes(S, SO, hs_floats);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_b_pm_left_ws<RMAX>, kWsThreads,
                                                    bytes) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const int grid = std::max(1, std::min(n, sms * per_sm));
  k_b_pm_left_ws<RMAX><<<grid, kWsThreads, bytes, st>>>(ts, it, n, queue, S, SO, hs_floats, err,
                                                        wait_cycles);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_pm_right(const BPlan& p, const BTensor* ts, const int4* items, int mode,
                            int* queue, int* err, cudaStream_t st, long long wait_cycles) {
  const size_t sm = (size_t)(kTileFloats + kWsFloats) * sizeof(float);
  const int n = p.pmr.count;
  const int4* it = items + p.pmr.off;
  if (mode == 0 || !queue) queue = nullptr;
  if (n > 0 && mode == 2 && queue && err) {
    cudaError_t e = p.rmax <= 16   ? launch_pm_right_ws<16>(ts, it, n, queue, err, wait_cycles, st)
                    : p.rmax <= 32 ? launch_pm_right_ws<32>(ts, it, n, queue, err, wait_cycles, st)
                                   : launch_pm_right_ws<64>(ts, it, n, queue, err, wait_cycles, st);
    if (e != cudaSuccess) return e;
  } else if (n > 0) {
    auto run = [&](auto k, int threads) {
      k<<<phase_grid(k, threads, sm, n, queue), threads, sm, st>>>(ts, it, n, queue);
    };
    if (p.rmax <= 16)
      run(k_b_pm_right<16>, RightCfg<16>::T);
    else if (p.rmax <= 32)
      run(k_b_pm_right<32>, RightCfg<32>::T);
    else
      run(k_b_pm_right<64>, RightCfg<64>::T);
  }
  if (p.pmr_red.count > 0)
    k_b_reduce<<<p.pmr_red.count, kReduceBlock, 0, st>>>(ts, items + p.pmr_red.off);
  return cudaGetLastError();
}

cudaError_t launch_pm_left(const BPlan& p, const BTensor* ts, const int4* items, int mode,
                           int* queue, int* err, cudaStream_t st, long long wait_cycles) {
  if (mode == 0 || !queue) queue = nullptr;
  const int n = p.pml.count;
  if (n == 0) return cudaSuccess;
  const int4* it = items + p.pml.off;
  if (mode == 2 && queue && err)
    return p.rmax <= 16   ? launch_pm_left_ws<16>(ts, it, n, queue, p.hs_floats, err, wait_cycles, st)
           : p.rmax <= 32 ? launch_pm_left_ws<32>(ts, it, n, queue, p.hs_floats, err, wait_cycles, st)
                          : launch_pm_left_ws<64>(ts, it, n, queue, p.hs_floats, err, wait_cycles, st);
  const size_t sm = (size_t)(kLeftTiles * kLeftStageFloats + left_h_floats(p.hs_floats)) * sizeof(float);
  k_b_pm_left<<<phase_grid(k_b_pm_left, kLeftThreads, sm, n, queue), kLeftThreads, sm, st>>>(ts, it, n, queue);
  return cudaGetLastError();
}

namespace {

cudaError_t launch_update(const BPlan& p, BTensor* ts, int n, int* done_count, cudaStream_t st) {
  const int rows = p.max_rows;
  if (p.rmax <= 16)
    k_b_update<16><<<p.count, 256, update_smem<16>(rows), st>>>(ts, n, done_count, rows);
  else if (p.rmax <= 32)
    k_b_update<32><<<p.count, 256, update_smem<32>(rows), st>>>(ts, n, done_count, rows);
  else
    k_b_update<64><<<p.count, 256, update_smem<64>(rows), st>>>(ts, n, done_count, rows);
  return cudaGetLastError();
}

}  // namespace

cudaError_t b_launch_init(const BPlan& p, BTensor* ts, const int4* items, double* alpha_part,
                          const int* alpha_first, cudaStream_t st) {
  if (p.count == 0) return cudaSuccess;
  if (p.alpha.count > 0)
    k_b_sumsq<<<p.alpha.count, 256, 0, st>>>(ts, items + p.alpha.off, alpha_part);
  if (p.max_factor < 1 || p.max_order < 1) return cudaErrorInvalidValue;  // b_plan_sizes not called
  const size_t fac = (size_t)p.max_factor * sizeof(float);
  k_b_init_mode<<<dim3((unsigned)p.count, (unsigned)p.max_order), 256, fac, st>>>(ts);
  k_b_init<<<p.count, 256, fac, st>>>(ts, alpha_part, alpha_first);
  return cudaGetLastError();
}

cudaError_t b_launch_iteration(const BPlan& p, BTensor* ts, const int4* items, int* done_count,
                               cudaStream_t st, const BSchedule& sch, int* queues) {
  if (p.count == 0) return cudaSuccess;
  const int N = p.N;
  cudaError_t e = cudaSuccess;
  const bool counters = queues && (sch.pm_right || sch.pm_left);
  if (counters) e = cudaMemsetAsync(queues, 0, 2 * sizeof(int), st);
  int* err = queues ? queues + 2 : nullptr;
  if (e == cudaSuccess)
    e = launch_pm_right(p, ts, items, counters ? sch.pm_right : 0, queues, err, st, sch.wait_cycles);
  if (e == cudaSuccess) e = launch_update(p, ts, 0, done_count, st);
  if (e == cudaSuccess)
    e = launch_pm_left(p, ts, items, counters ? sch.pm_left : 0, queues ? queues + 1 : nullptr, err, st,
                       sch.wait_cycles);
  // node {2..N} walk (Fig. 1 shape): leaf M(a), update, child node
  for (int a = 1; a < N && e == cudaSuccess; ++a) {
    if (a == N - 1) {
      e = launch_update(p, ts, a, done_count, st);
      break;
    }
    if (p.leaf[a].count > 0)
      k_b_mttv_leaf<<<p.leaf[a].count, 256, 0, st>>>(ts, items + p.leaf[a].off, a);
    if (p.leaf_red[a].count > 0)
      k_b_reduce<<<p.leaf_red[a].count, kReduceBlock, 0, st>>>(ts, items + p.leaf_red[a].off);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_update(p, ts, a, done_count, st);
    if (e == cudaSuccess && p.first[a].count > 0) {
      k_b_mttv_first<<<p.first[a].count, 256, 0, st>>>(ts, items + p.first[a].off, a);
      e = cudaGetLastError();
    }
  }
  return e;
}

cudaError_t launch_b_gather(const BTensor* ts, int count, int* iters, double* fits,
                            double* lam, const int* lam_off, int* nonfinite, cudaStream_t st) {
  k_b_gather<<<(count + 255) / 256, 256, 0, st>>>(ts, count, iters, fits, lam, lam_off, nonfinite);
  return cudaGetLastError();
}

}  // namespace nncp

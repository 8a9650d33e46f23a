// Float32 MTTKRP on CUDA cores over a (L, I, Q) view of the tensor (Sec. II-A,
// Sec. IV-A): out(i, r) = sum_{l, q} X[l + L (i + I q)] KL(l, r) KQ(q, r).
//
// The (L, I, Q) view: mode set split as [modes before] x [output modes] x
// [modes after], so X[l + L*(i + I*q)] holds the entry with left index l,
// output index i and right index q (mode-1-fastest layout, Sec. IV-C).
//   * direct MTTKRP of mode n (Sec. II-A): L = I_1..I_{n-1}, I = I_n,
//     Q = I_{n+1}..I_N;
//   * partial MTTKRP root -> {1..s} (Sec. IV-A, Fig. 2a): L = 1,
//     I = I_1..I_s, Q = I_{s+1}..I_N (contracts the slow modes);
//   * partial MTTKRP root -> {s+1..N}: L = I_1..I_s, I = I_{s+1}..I_N, Q = 1
//     (contracts the fast modes).
// It is a matrix product of I x R outputs over K = L Q, whose second operand,
// the Khatri-Rao rows, is formed on the fly: the digits of k = l + L q in the
// contracted modes, fastest first, are the factor rows multiplied.
//
// A CTA holds a tile of BM output rows x all rank columns in registers (8 ranks
// x 4 rows per thread as packed float32 pairs: fma.rn.f32x2 does two FMAs per
// issue slot, which leaves half of the slots to the shared-memory reads) and
// takes 32 contraction elements per step from a ring of three shared-memory
// stages that cp.async fills two steps ahead: the tensor tile and, beside it,
// the raw factor rows of the step -- a row of the fastest contracted mode per
// element and a row of every other mode per distinct index of the rest (two for
// a fastest mode of 31 or more).  One step before its use a stage's first rows
// are multiplied by the others in place, so no thread waits for a global load.
// One more warp, the feeder, walks the steps and fetches the factor rows (at
// high ranks the computing threads do: too many copies for one warp).  A step is
// described by the position of its first element alone -- digit d of the
// fastest mode, index q of the rest -- from which every thread derives its own
// element's: d + e past the mode's length is in the next rest row.
//
// Threads: 8 consecutive lanes take neighbouring output rows, then come the
// rank groups, the row groups and the KG-way split of a step's 32 elements,
// which keeps a warp's shared-memory reads at one or two wavefronts each and
// gives small ranks enough warps; the KG partial sums are added in a fixed
// tree at the end of a tile.
//
// Work split: G CTAs (what fits on the GPU at once) take whole tiles in turn;
// the tiles of a last, partly filled wave are cut into G equal runs of steps
// instead (a run may straddle two tiles), whose partial tiles go to `slots` and
// are added in a fixed order by k_simt_fixup.  Every cut follows from the shape and
// the scratch size alone, so results are bitwise reproducible (simt_plan.cuh).  A long
// run whose steps are not split adds up in segments (SEG).
//
// Measured on a GB300 per root branch (outputs slow / fast, calls repeated on one
// tensor), the 128 x 32 tile kernel of one FMA per issue slot that this one replaced in
// brackets: 512^3 R = 8 102 / 101 us (358 / 411), R = 32 246 / 250 us (363 / 416),
// 40000x48x40 R = 16 119 / 92 us (292 / 230), 301x257x199 R = 20 56 / 45 us (74 / 85),
// 220x180x150 R = 100 70 / 66 us (90 / 91).  At R = 8 it streams at 5.3 TB/s; at R = 32 it
// runs at 0.44 of the FMA peak, of which a step's loads, Khatri-Rao rows and barrier take
// a quarter and the shared-memory reads (three of 16 bytes per 16 packed FMAs) most of
// the rest.
#include <cuda_runtime.h>

#include <algorithm>

#include "nncp_internal.cuh"
#include "simt_plan.cuh"

namespace nncp {

namespace {

// One step: the tile it belongs to and the position of its first element.
struct StepTab {
  long long i0, k0;      // first output row of the tile, first contraction element
  long long rest;        // k0 / dim[0]
  long long l, q;        // k0 mod L, k0 / L
  int d;                 // k0 mod dim[0]
  int nk;                // valid elements (1..32)
  int valid;             // 0: no more steps
  int last;              // 1: last step of this CTA's run over the tile
  int seg;               // after it: 1, 2 write or add the sums to tensor memory, 3 add those to the sums
  int slot;              // partial slot of the run, -1: the whole tile (write the output)
};

// x / n for 0 <= x < n + 32: mag = ceil(2^16 / n) for n < 32 (exact there: the
// excess is below 63 / 2^16 < 1 / n), 0 otherwise
template <typename I>
__device__ __forceinline__ int wraps(I x, I n, int mag) {
  return mag ? (int)(((unsigned)x * (unsigned)mag) >> 16) : (x >= n ? 1 : 0);
}

static_assert(sizeof(StepTab) * kTabs + 64 <= kStaticSmem, "static shared memory");

__device__ __forceinline__ uint32_t s_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cpa16(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa16_hint(uint32_t dst, const float* src, uint64_t pol) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
               "l"(pol)
               : "memory");
}
__device__ __forceinline__ void cpa4(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
// sixteen columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_read16(uint32_t c, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(c)
      : "memory");
}
__device__ __forceinline__ void tmem_write16(uint32_t c, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15, %16};" ::"r"(c),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}
// the writes of the flush before have landed
__device__ __forceinline__ void tmem_write_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// A thread's accumulators into its tensor-memory cells (a lane, columns c .. c + 31):
// cells = acc (+ cells when ADD), then acc = 0
template <bool ADD>
__device__ __forceinline__ void seg_flush(u64 (&acc)[kTM][4], uint32_t c) {
  if (ADD) tmem_write_wait();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[16] = {};
    if (ADD) tmem_read16(c + 16 * h, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      u64& x = acc[2 * h + k / 4][k % 4];
      const float2 a = unpack2(x);
      v[2 * k] += a.x;
      v[2 * k + 1] += a.y;
      x = 0ull;
    }
    tmem_write16(c + 16 * h, v);
  }
}
// acc += cells
__device__ __forceinline__ void seg_add(u64 (&acc)[kTM][4], uint32_t c) {
  tmem_write_wait();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[16];
    tmem_read16(c + 16 * h, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      u64& x = acc[2 * h + k / 4][k % 4];
      const float2 a = unpack2(x);
      x = pack2(a.x + v[2 * k], a.y + v[2 * k + 1]);
    }
  }
}

__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }


// first step of run c over the cut tiles
__device__ __forceinline__ long long run_start(long long c, long long U2, int G2) {
  return c * U2 / G2;
}

// The steps of a CTA in order: whole tiles blockIdx.x, + gridDim.x, ..., then
// its run over the cut tiles (one warp, uniform).
struct Feeder {
  long long tile, k, kend;  // tile; next step and end of the current run over it
  long long u, u1;          // what is left of the run over the cut tiles
  long long rest, l, q;
  int d, slot;
  int in_run;  // steps of the run so far; from its second segment on p.seg more than of the segment
  bool cut, first;

  __device__ __forceinline__ explicit Feeder(const SimtArgs& p) {
    tile = (long long)blockIdx.x - gridDim.x;
    k = kend = u = u1 = rest = l = q = 0;
    if ((int)blockIdx.x < p.G2) {
      u = run_start(blockIdx.x, p.U2, p.G2);
      u1 = run_start(blockIdx.x + 1, p.U2, p.G2);
    }
    d = in_run = 0;
    slot = -1;
    cut = false;
    first = true;
  }

  __device__ __forceinline__ void next(const SimtArgs& p, StepTab& t, bool kc) {
    if (k < kend) {
      // the next step of the same run: 32 elements on
      d += p.dstep;
      rest += p.rstep;
      if (d >= p.dim[0]) {
        d -= p.dim[0];
        ++rest;
      }
      if (kc) {
        l += p.lstep;
        q += p.qstep;
        if (l >= p.L) {
          l -= p.L;
          ++q;
        }
      }
    } else {
      bool got = false;
      if (!cut) {
        tile += gridDim.x;
        k = 0;
        kend = p.nk;
        slot = -1;
        got = tile < p.whole;
        cut = !got;
      }
      if (!got && u < u1) {
        const long long qt = u / p.nk;
        tile = p.whole + qt;
        k = u - qt * p.nk;
        kend = min(p.nk, k + (u1 - u));
        u += kend - k;
        const bool all = k == 0 && kend == p.nk;
        slot = all ? -1 : (p.two ? 2 * (int)blockIdx.x + (first ? 0 : 1) : (int)blockIdx.x);
        first = false;
        got = true;
      }
      if (!got) {
        k = kend = 0;
        t.valid = 0;
        return;
      }
      const long long e = k * kBK;
      rest = d = 0;
      l = q = 0;
      if (e != 0) {
        rest = e / p.dim[0];
        d = (int)(e - rest * p.dim[0]);
        if (kc) {
          q = e / p.L;
          l = e - q * p.L;
        }
      }
    }
    const bool last = k + 1 == kend;
    int seg = 0;
    if (p.seg > 0) {
      ++in_run;
      if (last) {
        seg = in_run > p.seg ? 3 : 0;
        in_run = 0;
      } else if (in_run == p.seg) {
        seg = 1;
      } else if (in_run == 2 * p.seg) {
        seg = 2;
        in_run = p.seg;
      }
    }
    if ((threadIdx.x & 31) == 0) {
      t.i0 = tile << p.bm_log2;
      t.k0 = k * kBK;
      t.rest = rest;
      t.l = l;
      t.q = q;
      t.d = d;
      t.nk = (int)min((long long)kBK, p.K - k * kBK);
      t.valid = 1;
      t.last = last;
      t.seg = seg;
      t.slot = slot;
    }
    ++k;
  }
};

// KC: the contraction is contiguous in memory (L > 1), stage rows are output
// rows of 32 elements, their 16-byte chunks permuted by the row (chunk ^ row
// mod 8) so that eight neighbouring rows are read without bank conflicts;
// otherwise (L = 1) the outputs are contiguous and stage rows are contraction
// elements of BM outputs.  SEG: after every p.seg steps of a run a thread's sums are
// added to 32 columns of its tensor-memory lane, which costs no register or shared memory.
template <bool KC, bool SEG>
__global__ void __launch_bounds__(kThreadsMax + 32, 2)
k_simt_mttkrp(const __grid_constant__ SimtArgs p) {
  extern __shared__ __align__(16) float sm[];
  __shared__ StepTab tabs[kTabs];
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, T = blockDim.x - 32;
  const int BM = 1 << p.bm_log2, RP = p.RP;
  const uint32_t sbase = s_u32(sm);
  // ---- the factor rows of a step, by n threads: one per element of the fastest
  // mode, then the distinct rest rows of every other mode, 2^gsh lanes (at most
  // a warp) per row
  const int rc = p.vecb ? p.R >> 2 : p.R;  // copies per factor row
  auto load_b = [&](const StepTab& t, int stage, int id, int n) {
    if (!t.valid) return;
    const uint32_t raw = sbase + 4u * (stage * p.stage_floats + p.x_floats);
    const int sub = id & ((1 << p.gsh) - 1), r0 = id >> p.gsh, dr = n >> p.gsh;
    auto row = [&](uint32_t dst, const float* src) {
      if (p.vecb) {
        if (sub < rc) cpa16(dst + 16u * sub, src + 4 * sub);
      } else {
        for (int c = sub; c < rc; c += 1 << p.gsh) cpa4(dst + 4u * c, src + c);
      }
    };
    const int d = t.d, nk = t.nk;
#pragma unroll 4
    for (int kk = r0; kk < nk; kk += dr) {
      const int x = d + kk;
      row(raw + 4u * kk * RP, p.H[0] + (x - wraps(x, p.dim[0], p.mag0) * p.dim[0]) * p.ld);
    }
    if (p.nm > 1) {
      const int nrest = wraps(d + nk - 1, p.dim[0], p.mag0) + 1;
#pragma unroll 1
      for (int j = r0; j < nrest; j += dr) {
        long long q = t.rest + j;
        uint32_t dst = raw + 4u * (kBK + j) * RP;
#pragma unroll 1
        for (int m = 1; m < p.nm; ++m, dst += 4u * p.nrest_max * RP) {
          long long x = q;
          if (m + 1 < p.nm) {  // the last digit is what is left
            q = (unsigned long long)x >> 32 ? x / p.dim[m] : (long long)((unsigned)x / (unsigned)p.dim[m]);
            x -= q * p.dim[m];
          }
          row(dst, p.H[m] + x * p.ld);
        }
      }
    }
  };

  if (tid >= T) {
    // ------------------------------------------------------------ feeder --
    const int lane = tid - T;
    const uint32_t cols = T > 128 ? 64 : 32;  // a warp reaches lanes 32 (w mod 4) .. + 31
    if constexpr (SEG) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(&tmem_slot)),
                   "r"(cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    Feeder f(p);
    for (int s = 0; s < kStages; ++s) f.next(p, tabs[s], KC);
    __syncthreads();
    pdl_wait();
    if (!p.b_all) {
      load_b(tabs[0], 0, lane, 32);
      load_b(tabs[1], 1, lane, 32);
      asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    __syncthreads();
    for (int s = 0, st = 2;; ++s) {
      // the factor rows of step s + 1 have landed
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      __syncthreads();
      const StepTab& t = tabs[s & (kTabs - 1)];
      if (!t.valid) break;
      const bool last = t.last != 0;
      if (!p.b_all) load_b(tabs[(s + 2) & (kTabs - 1)], st, lane, 32);
      st = st + 1 == kStages ? 0 : st + 1;
      f.next(p, tabs[(s + 3) & (kTabs - 1)], KC);
      if (last && p.KG > 1) {
        // the barriers of the computing warps' KG sums
        __syncthreads();
        for (int half = p.KG >> 1; half >= 1; half >>= 1)
          for (int j0 = 0; j0 < 4; j0 += p.red_pairs) {
            __syncthreads();
            __syncthreads();
          }
      }
    }
    if constexpr (SEG) {
      __syncthreads();  // every warp is done with its cells
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(cols) : "memory");
    }
    return;
  }

  // -------------------------------------------------------- computing warps --
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  const int Tl = p.tl;

  // ---- the tensor tile of a step into a stage
  auto load_x = [&](const StepTab& t, int stage) {
    if (!t.valid || tid >= Tl) return;
    const uint32_t xs = sbase + 4u * stage * p.stage_floats;
    const long long i0 = t.i0;
    const int rows = (int)min((long long)BM, p.I - i0);
    const int nk = t.nk;
    if constexpr (KC) {
      if (p.vecx) {
        const int c = tid & 7, dr = Tl >> 3;  // this thread's chunk of rows i, i + dr, ...; dr % 8 == 0
        if (4 * c < nk) {                     // K is a multiple of 4: chunks are whole
          int i = tid >> 3;
          long long l = t.l + 4 * c;
          const int w = wraps(l, p.L, p.magl);
          l -= w * p.L;
          const float* src = p.X + l + p.L * (i0 + i + p.I * (t.q + w));
          uint32_t d = xs + 4u * (i * kBK + ((c ^ (i & 7)) << 2));
          const long long ds = p.L * dr;
#pragma unroll 4
          for (; i < rows; i += dr, src += ds, d += 4u * kBK * dr) {
            if (p.evict) cpa16_hint(d, src, pol);
            else cpa16(d, src);
          }
        }
      } else {
        const int kk = tid & 31, dr = Tl >> 5;
        int i = tid >> 5;
        const bool in = kk < nk;
        long long l = t.l + kk;
        const int w = wraps(l, p.L, p.magl);
        l -= w * p.L;
        const float* src = p.X + l + p.L * (i0 + i + p.I * (t.q + w));
        const long long ds = p.L * dr;
        if (in) {
#pragma unroll 4
          for (; i < rows; i += dr, src += ds)
            cpa4(xs + 4u * (i * kBK + (((kk >> 2) ^ (i & 7)) << 2) + (kk & 3)), src);
        } else {
          // up to the next multiple of the four elements a thread takes at a time
          for (; i < rows && kk < ((nk + 3) & ~3); i += dr)
            sm[stage * p.stage_floats + i * kBK + (((kk >> 2) ^ (i & 7)) << 2) + (kk & 3)] = 0.0f;
        }
      }
    } else {
      const int sh = p.vecx ? p.bm_log2 - 2 : p.bm_log2;  // copies per stage row
      const int ii = tid & ((1 << sh) - 1);
      if (p.vecx) {
        int kk = tid >> sh;
        const int dk = Tl >> sh;  // Tl >= BM / 4
        if (4 * ii < rows) {
          const float* src = p.X + (t.k0 + kk) * p.I + i0 + 4 * ii;
          uint32_t d = xs + 4u * ((kk << p.bm_log2) + 4 * ii);
          const long long ds = p.I * dk;
#pragma unroll 4
          for (; kk < nk; kk += dk, src += ds, d += 4u * (dk << p.bm_log2)) {
            if (p.evict) cpa16_hint(d, src, pol);
            else cpa16(d, src);
          }
        }
      } else {
        const float* src = p.X + t.k0 * p.I + i0;
        const int end = nk << sh;
#pragma unroll 4
        for (int e = tid; e < end; e += Tl) {
          const int kk = e >> sh, i = e & (BM - 1);
          if (i < rows) cpa4(xs + 4u * e, src + (long long)kk * p.I + i);
        }
      }
    }
  };
  // ---- Khatri-Rao rows of a step in place: the fastest mode's rows times the
  // rest; elements past the end up to a multiple of four are zero
  const int fk0 = tid / (RP >> 2), fc0 = tid - fk0 * (RP >> 2);
  auto form_b = [&](const StepTab& t, int stage) {
    if (!t.valid || (p.nm == 1 && t.nk == kBK)) return;
    float* raw = sm + stage * p.stage_floats + p.x_floats;
    const int r4 = RP >> 2;
    int kk = fk0, c = fc0;
    const int end = (t.nk + 3) & ~3;
#pragma unroll 1
    while (kk < end) {
      float4* d = reinterpret_cast<float4*>(raw + kk * RP + 4 * c);
      float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (kk < t.nk) {
        v = *d;
        const float* rest = raw + (kBK + wraps(t.d + kk, p.dim[0], p.mag0)) * RP + 4 * c;
#pragma unroll 1
        for (int m = 1; m < p.nm; ++m, rest += p.nrest_max * RP) {
          const float4 w = *reinterpret_cast<const float4*>(rest);
          v.x *= w.x;
          v.y *= w.y;
          v.z *= w.z;
          v.w *= w.w;
        }
      }
      *d = v;
      kk += p.fk;
      c += p.fc;
      if (c >= r4) {
        c -= r4;
        ++kk;
      }
    }
  };

  // ---- this thread's place
  const int rl = tid & 7;
  int id = tid >> 3;
  const int cg = id % p.CG;
  id /= p.CG;
  const int rgh = id % p.RGH;
  const int kg = id / p.RGH;
  const bool act = kg < p.KG;
  const int kper = SEG ? kBK : kBK / p.KG, ka = SEG ? 0 : kg * kper;  // SEG: KG = 1
  const int ngroup = 8 * p.CG * p.RGH;  // threads of a k group
  u64 acc[kTM][4];
#pragma unroll
  for (int i = 0; i < kTM; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;

  __syncthreads();
  // the tensor is written by no kernel of an iteration, where alone the kernel may
  // start early (launch_columns): its first tiles stream in while the preceding
  // kernel finishes
  load_x(tabs[0], 0);
  load_x(tabs[1], 1);
  pdl_wait();
  if (p.b_all) {
    load_b(tabs[0], 0, tid, T);
    load_b(tabs[1], 1, tid, T);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  form_b(tabs[0], 0);

  if constexpr (SEG) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // lane 32 (w mod 4) of warp w, the columns of its group of four
  auto cells = [&]() { return tmem_slot + ((uint32_t)(tid & 96) << 16) + 32u * (tid >> 7); };
  for (int s = 0, st = 0;; ++s) {
    // step s and the factor rows of step s + 1 have landed, and every thread
    // is done with step s - 1
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const StepTab& t = tabs[s & (kTabs - 1)];
    if (!t.valid) break;
    const int st1 = st + 1 == kStages ? 0 : st + 1, st2 = st1 + 1 == kStages ? 0 : st1 + 1;
    const StepTab& t2 = tabs[(s + 2) & (kTabs - 1)];
    if (p.b_all) load_b(t2, st2, tid, T);
    cpa_commit();
    load_x(t2, st2);
    cpa_commit();
    form_b(tabs[(s + 1) & (kTabs - 1)], st1);

    float* xs = sm + st * p.stage_floats;
    const float* bs = xs + p.x_floats + 8 * cg;
    st = st1;
    if (act) {
      if constexpr (KC) {
        const float* xrow = xs + (32 * rgh + rl) * kBK;
        const int kb = min(ka + kper, (t.nk + 3) & ~3);
#pragma unroll 1
        for (int k = ka; k < kb; k += 4) {
          const int c = ((k >> 2) ^ rl) << 2;
          float4 a[kTM];
#pragma unroll
          for (int i = 0; i < kTM; ++i) a[i] = *reinterpret_cast<const float4*>(xrow + 8 * i * kBK + c);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bs + (k + e) * RP);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(bs + (k + e) * RP + 4);
#pragma unroll
            for (int i = 0; i < kTM; ++i) {
              const float v = e == 0 ? a[i].x : (e == 1 ? a[i].y : (e == 2 ? a[i].z : a[i].w));
              const u64 x = pack2(v, v);
              acc[i][0] = ffma2(x, b0.x, acc[i][0]);
              acc[i][1] = ffma2(x, b0.y, acc[i][1]);
              acc[i][2] = ffma2(x, b1.x, acc[i][2]);
              acc[i][3] = ffma2(x, b1.y, acc[i][3]);
            }
          }
        }
      } else {
        const float* xcol = xs + 32 * rgh + 4 * rl;
        const int kb = min(ka + kper, t.nk);
#pragma unroll 4
        for (int k = ka; k < kb; ++k) {
          const float4 v = *reinterpret_cast<const float4*>(xcol + (k << p.bm_log2));
          const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bs + k * RP);
          const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(bs + k * RP + 4);
          const float a[kTM] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int i = 0; i < kTM; ++i) {
            const u64 x = pack2(a[i], a[i]);
            acc[i][0] = ffma2(x, b0.x, acc[i][0]);
            acc[i][1] = ffma2(x, b0.y, acc[i][1]);
            acc[i][2] = ffma2(x, b1.x, acc[i][2]);
            acc[i][3] = ffma2(x, b1.y, acc[i][3]);
          }
        }
      }
    }
    if constexpr (SEG) {
      const int seg = t.seg;
      if (seg == 1) seg_flush<false>(acc, cells());
      else if (seg == 2) seg_flush<true>(acc, cells());
      else if (seg == 3) seg_add(acc, cells());
    }
    if (!t.last) continue;

    // ---- end of a run: add the KG partial sums in a fixed tree, then write the tile
    const int q = tid - kg * ngroup;  // thread within the k group
    if (p.KG > 1) {
      // through this step's stage, done with once every thread is; jn of a
      // thread's four column pairs at a time fit
      float2* red = reinterpret_cast<float2*>(xs);
      const int jn = p.red_pairs;
      __syncthreads();
      for (int half = p.KG >> 1; half >= 1; half >>= 1) {
        for (int j0 = 0; j0 < 4; j0 += jn) {
          if (kg >= half && kg < 2 * half) {
            float2* dst = red + (kg - half) * ngroup * (jn * kTM) + q;
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j >= j0 && j < j0 + jn)
#pragma unroll
                for (int i = 0; i < kTM; ++i) dst[((j - j0) * kTM + i) * ngroup] = unpack2(acc[i][j]);
          }
          __syncthreads();
          if (kg < half) {
            const float2* src = red + kg * ngroup * (jn * kTM) + q;
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j >= j0 && j < j0 + jn)
#pragma unroll
                for (int i = 0; i < kTM; ++i) {
                  const float2 v = src[((j - j0) * kTM + i) * ngroup], a = unpack2(acc[i][j]);
                  acc[i][j] = pack2(a.x + v.x, a.y + v.y);
                }
          }
          __syncthreads();
        }
      }
    }
    if (kg == 0) {
      const long long i0 = t.i0;
      const bool part = t.slot >= 0;
      float* dst = part ? p.slots + t.slot * p.slot_floats : p.out + i0 * p.ld;
      const int ld = part ? p.R : p.ld;
      const bool vec = part ? (p.R & 3) == 0 : p.veco;
      const int rows = (int)min((long long)BM, p.I - i0);
#pragma unroll
      for (int i = 0; i < kTM; ++i) {
        const int row = 32 * rgh + (KC ? 8 * i + rl : 4 * rl + i);
        if (row < rows) {
          float* d = dst + (long long)row * ld + 8 * cg;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float2 a = unpack2(acc[i][2 * j]), b = unpack2(acc[i][2 * j + 1]);
            const int left = p.R - 8 * cg - 4 * j;
            if (vec && left >= 4) {
              reinterpret_cast<float4*>(d)[j] = make_float4(a.x, a.y, b.x, b.y);
            } else {
              if (left > 0) d[4 * j] = a.x;
              if (left > 1) d[4 * j + 1] = a.y;
              if (left > 2) d[4 * j + 2] = b.x;
              if (left > 3) d[4 * j + 3] = b.y;
            }
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kTM; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if constexpr (SEG) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
}

// Adds the partial tiles of the cut tiles.  blockIdx.y: tile.  W > 1: the W warps
// of a CTA take 32 neighbouring outputs, warp w adding runs w, w + W, ... of the
// tile, and warp 0 adds the warps' sums; W = 1: a thread per output adds the runs.
// A thread's runs go to four sums in turn and everything after that is added in
// pairs: with runs and warps added one after the other, the last 32 additions alone
// made the error of a 301 x 257 x 199 contraction at R = 20 8.6e-8, not 4.1e-8.  (Four threads per output left 760 runs of a 12 x 20 output
// to ten CTAs: 108 us on a GB300, more than the MTTKRP.)
template <int W>
__global__ void __launch_bounds__(W > 1 ? 32 * W : 256)
k_simt_fixup(const float* __restrict__ slots, float* __restrict__ out, long long I, int R, int ld, int BM,
             long long slot_floats, long long nk, long long whole, long long U2, int G2,
             int two) {
  pdl_wait();
  pdl_trigger();
  __shared__ float part[W > 1 ? W : 1][32];
  const long long t = blockIdx.y, u0 = t * nk, u1 = u0 + nk - 1;
  const int c0 = (int)(((u0 + 1) * G2 - 1) / U2), c1 = (int)(((u1 + 1) * G2 - 1) / U2);
  if (c0 == c1) return;  // one run holds the whole tile and has written it
  const long long i0 = (whole + t) * BM;
  const int rows = (int)min((long long)BM, I - i0);
  const int w = W > 1 ? threadIdx.x >> 5 : 0;
  const int e = W > 1 ? blockIdx.x * 32 + (threadIdx.x & 31) : blockIdx.x * 256 + threadIdx.x;
  const bool in = e < rows * R;
  // a run that began in an earlier tile left this one in its second slot
  const int odd = two && run_start(c0, U2, G2) < u0 ? 1 : 0;
  const int mul = two ? 2 : 1;
  float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (in) {
    auto run = [&](int c) {
      return __ldg(slots + (long long)(mul * c + (c == c0 ? odd : 0)) * slot_floats + e);
    };
    int c = c0 + w;
#pragma unroll 2
    for (; c + 3 * W <= c1; c += 4 * W) {
#pragma unroll
      for (int k = 0; k < 4; ++k) s4[k] += run(c + k * W);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (c + k * W <= c1) s4[k] += run(c + k * W);
  }
  float s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
  if (W > 1) {
    part[w][threadIdx.x & 31] = s;
    __syncthreads();
    if (w > 0) return;
    float v[W > 1 ? W : 2];
#pragma unroll
    for (int k = 0; k < W; ++k) v[k] = part[k][threadIdx.x & 31];
#pragma unroll
    for (int h = W / 2; h > 0; h /= 2)
#pragma unroll
      for (int k = 0; k < h; ++k) v[k] += v[k + h];
    s = v[0];
  }
  if (in) out[(i0 + e / R) * ld + e % R] = s;
}

// The launches for the rank columns [r0, r0 + pl.a.R) of a rank-R MTTKRP.
cudaError_t launch_columns(const float* X, int R, int r0, float* out, float* partials,
                           SimtPlan pl, cudaStream_t st, bool early) {
  SimtArgs& a = pl.a;
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  const bool KC = a.L > 1;
  a.X = X;
  a.ld = R;
  a.out = out + r0;
  for (int m = 0; m < a.nm; ++m) a.H[m] += r0;
  a.slots = partials;
  // 16-byte copies need whole units along the contiguous index; the factor
  // rows also a rank of whole units
  a.vecx = al16(X) && (KC ? a.L : a.I) % 4 == 0;
  a.vecb = R % 4 == 0 && a.R % 4 == 0;
  for (int m = 0; m < a.nm; ++m) a.vecb = a.vecb && al16(a.H[m]);
  a.veco = R % 4 == 0 && al16(a.out);
  // a tensor that cannot stay in the 126 MB L2 is marked evict-first, so that
  // its stream leaves the nodes and factors there
  a.evict = (double)a.I * a.K * sizeof(float) > 96e6;
  const int copies = a.vecb ? a.R / 4 : a.R;
  while (a.gsh < 5 && (1 << a.gsh) < copies) ++a.gsh;
  void (*const k)(SimtArgs) = KC ? (a.seg ? k_simt_mttkrp<true, true> : k_simt_mttkrp<true, false>)
                                 : (a.seg ? k_simt_mttkrp<false, true> : k_simt_mttkrp<false, false>);
  cudaError_t e = launch_kernel_if(early, k, dim3((unsigned)pl.grid), dim3(pl.threads + 32),
                                pl.smem, st, a);
  if (e != cudaSuccess || a.G2 == 0) return e;
  const long long left = a.U2 / a.nk;
  // warps per output by the runs of a tile
  const long long runs = a.G2 / left;
  const int W = runs >= 128 ? 32 : (runs >= 8 ? 8 : 1);
  const int gx = (int)cdiv(a.slot_floats, W > 1 ? 32 : 256);
  return launch_kernel(W == 32 ? k_simt_fixup<32> : (W == 8 ? k_simt_fixup<8> : k_simt_fixup<1>),
                       dim3((unsigned)gx, (unsigned)left), dim3(W > 1 ? 32 * W : 256), 0, st,
                       (const float*)partials, a.out, a.I, a.R, a.ld, pl.BM, a.slot_floats, a.nk,
                       a.whole, a.U2, a.G2, a.two);
}

}  // namespace

cudaError_t simt_attributes_init() {
  for (auto k : {k_simt_mttkrp<false, false>, k_simt_mttkrp<true, false>, k_simt_mttkrp<false, true>,
                 k_simt_mttkrp<true, true>}) {
    cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax - kStaticSmem);
    // all of the SM's shared memory: the plan counts on it for its CTAs per SM
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                               cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t simt_mttkrp_partials(int64_t L, int64_t I, int64_t Q, int R, int num_sms, bool fine) {
  return scratch_floats((long long)L * Q, I, R, num_sms, fine);
}
bool simt_few_rows(int64_t I) { return I <= kFewRows; }

cudaError_t launch_simt_mttkrp(const float* X, int64_t L, int64_t I, int64_t Q,
                               const KrpDesc& KL, const KrpDesc& KQ, int R, float* out,
                               float* partials, size_t part_cap, int num_sms,
                               cudaStream_t st, bool early) {
  // ranks in one launch unless the factor rows of a step (long products of short
  // modes at a high rank) do not fit in shared memory: then in column blocks
  int cols = R;
  SimtPlan pl;
  while (!plan_simt(L, I, Q, KL, KQ, cols, partials ? part_cap : 0, num_sms, &pl)) {
    if (cols <= 8) return cudaErrorInvalidValue;
    cols = ((cols + 1) / 2 + 7) / 8 * 8;
  }
  for (int r0 = 0; r0 < R; r0 += cols) {
    const int n = std::min(cols, R - r0);
    if (n != cols && !plan_simt(L, I, Q, KL, KQ, n, partials ? part_cap : 0, num_sms, &pl))
      return cudaErrorInvalidValue;
    const cudaError_t e = launch_columns(X, R, r0, out, partials, pl, st, early);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace nncp

// Sampling-stage truncation (Sec. 3.4, last paragraph): the float softmax over the vocabulary runs on
// the rows of the current block only.  Per block row: the most probable token (lowest id among equal
// logits), its probability and the log normaliser.  HBM-bound: every logit of the block's rows is read
// once, nothing else of the [T, vocab] array is touched.
//
// A row is cut into equal segments, one warp each, as many as fill the GPU with resident warps to the last
// (see sample_rows), so that every SM streams the same number of bytes whatever the number of rows.  A warp
// reduces its segment to (max, sum of exp relative to that max, index of the first maximum) in one pass and
// publishes it; the last warp of a row to arrive (one counter per row, reset by that warp) combines the row's
// segments in order, so the result does not depend on the arrival order.  Warps share nothing and never wait
// for one another, so the chain at the end of a segment (reduce, publish, count, read back) hides behind the
// other warps' loads.
//
// Per element: half a packed maximum, a conversion, half a multiply-add, one exponential, half an addition
// (f32x2 arithmetic).  The multiply-add forms x log2 e - R with R the rounded m log2 e; what the rounding of R
// did to every term alike is divided out of the segment's sum at the end.  That works while what it did is a factor
// fp32 can hold: not for an m of -1e10 or the type's lowest value, which is what a mask may fill in.  The pass counts
// entries of that size as nothing, which they are beside any smaller maximum, and a segment whose maximum is one of them
// is summed again relative to it.  The index of the
// maximum costs nothing per element: a thread remembers which batch of its elements raised its maximum, and
// only the threads that hold the segment's maximum look at their batch again.  (With a compare and two
// selects per element and CTAs per row rounded to whole slices, 64.7 MB of bf16 logits took 22.6 us; now 16.8, and 49.4 us
// against 64.7 for four times the rows.)
#include <cuda_bf16.h>

#include <algorithm>

#include "lacache_internal.h"
#include "lacache_ptx.h"

namespace lacache {
namespace {

using namespace ptx;

constexpr int SAMPLE_THREADS = 256;
constexpr int WARPS = SAMPLE_THREADS / 32;
// Resident CTAs per SM and batches in flight per lane: what streams many rows fastest, and what finishes the
// few warps of a short launch soonest (their whole segment is then requested at once: 7.0 us against 7.7 for 32 rows
// of 126464 bf16 entries; with 256 rows the first is faster, 16.1 us against 19.8).
struct Wide { static constexpr int CTAS = 4, DEPTH = 3; };
struct Deep { static constexpr int CTAS = 3, DEPTH = 5; };
constexpr float LOG2E = 1.4426950408889634f;
// Up to here the rounding of m log2 e is at most 2^5: every term and sum is off by at most 2^32, which fp32 holds.
constexpr float HUGE_LOGIT = 0x1p29f;
constexpr float FLOAT_MAX = 3.402823466e38f;
constexpr float LN2F = 0.69314718055994531f;

struct Acc {
  float m, s;   // running maximum; sum of 2^((x - m) log2 e) over the elements seen
  int idx;      // index of the first element equal to m
};

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// a and b cover disjoint index ranges
__device__ __forceinline__ Acc acc_merge(const Acc& a, const Acc& b) {
  Acc r;
  if (b.m > a.m || (b.m == a.m && b.idx < a.idx)) {
    r.m = b.m; r.idx = b.idx;
  } else {
    r.m = a.m; r.idx = a.idx;
  }
  const float sa = a.m == -INFINITY ? 0.f : a.s * ex2f((a.m - r.m) * LOG2E);
  const float sb = b.m == -INFINITY ? 0.f : b.s * ex2f((b.m - r.m) * LOG2E);
  r.s = sa + sb;
  return r;
}

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

// two fp32 in one 64-bit register
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// the elements of one 32-bit word of a vector as fp32 pairs / the maximum of a vector
template <class T>
struct Words;
template <>
struct Words<__nv_bfloat16> {
  static constexpr int PAIRS = 4;   // pairs per 16-byte vector
  static __device__ __forceinline__ uint64_t pair(const uint4& v, int i) {
    const uint32_t w = (&v.x)[i];
    return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  }
  static __device__ __forceinline__ float max_of(const uint4& u, const uint4& v) {
    const __nv_bfloat162* a = reinterpret_cast<const __nv_bfloat162*>(&u);
    const __nv_bfloat162* b = reinterpret_cast<const __nv_bfloat162*>(&v);
    const __nv_bfloat162 x = __hmax2(__hmax2(__hmax2(a[0], a[1]), __hmax2(a[2], a[3])), __hmax2(__hmax2(b[0], b[1]), __hmax2(b[2], b[3])));
    return fmaxf(__low2float(x), __high2float(x));
  }
};
template <>
struct Words<float> {
  static constexpr int PAIRS = 2;
  static __device__ __forceinline__ uint64_t pair(const uint4& v, int i) {
    return pack2(__uint_as_float((&v.x)[2 * i]), __uint_as_float((&v.x)[2 * i + 1]));
  }
  static __device__ __forceinline__ float max_of(const uint4& u, const uint4& v) {
    const float* a = reinterpret_cast<const float*>(&u);
    const float* b = reinterpret_cast<const float*>(&v);
    return fmaxf(fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3])), fmaxf(fmaxf(b[0], b[1]), fmaxf(b[2], b[3])));
  }
};

// The elements i, i + 32, ... relative to a huge maximum.  (Next to never called, and the kernel's end is its tail: inlined
// there it took 256 rows of 126464 entries from 16.85 us to 16.95, as a call it leaves 16.75.)
template <class T>
__device__ __noinline__ float sum_again(const T* x, int i, int hi, float M) {
  float s = 0.f;
  for (; i < hi; i += 32) s += ex2f((to_float(x[i]) - M) * LOG2E);
  return s;
}

template <class T, class SHAPE>
__global__ void __launch_bounds__(SAMPLE_THREADS, SHAPE::CTAS) sample_rows_kernel(const SampleArgs a) {
  constexpr int VEC = 16 / (int)sizeof(T);
  constexpr int NV = 2;                             // vectors of a batch
  constexpr int STEP = 32 * VEC;                    // distance of a lane's vectors
  constexpr int DEPTH = SHAPE::DEPTH;               // batches of a lane in flight, the one in hand included
  const int lane = threadIdx.x & 31;
  const int warp = (int)blockIdx.x * WARPS + (int)(threadIdx.x >> 5);
  const int r = warp / a.segments, seg = warp - r * a.segments;
  const int row = r < a.n_rows ? a.rows[r] : 0;   // (the context's own list, which nothing writes)
  // launched programmatically dependent: nothing else is touched before the grids ahead have completed
  grid_dependency_wait();

  if (r < a.n_rows) {
    const int lo = seg * a.quota, hi = min(lo + a.quota, a.vocab);
    const bool bad = row < 0 || row >= a.n_tokens;
    // s: the sum of 2^(x log2 e - R); R = m log2 e, rounded (0 before any finite logit).
    // `at`: where m was first seen -- >= 0: a batch of vectors that starts there; < 0: element ~at
    float m = -INFINITY, R = 0.f, s = 0.f;
    int at = ~0x7fffffff;
    auto raise = [&](float to, int where) {
      const float Rn = fabsf(to) < HUGE_LOGIT ? to * LOG2E : INFINITY;   // (a huge m: every term is 0, and so is s)
      s *= ex2f(fminf(R - Rn, 0.f));   // (the first finite logit finds s = 0)
      m = to;
      R = Rn;
      at = where;
    };
    const T* x = reinterpret_cast<const T*>(a.logits) + (size_t)(bad ? 0 : row) * a.vocab;
    // the first 16-byte boundary in the segment, and the end of the last whole vector (rows of a vocabulary that
    // is no multiple of the vector start anywhere; the up to VEC - 1 elements on either side are taken singly)
    const int head = (int)((16u - (uint32_t)(reinterpret_cast<uintptr_t>(x + lo) & 15u)) & 15u) / (int)sizeof(T);
    const int b0 = min(lo + head, hi), b1 = b0 + (hi - b0) / VEC * VEC;
    auto one = [&](int i) {
      const float f = to_float(x[i]);
      if (f > m) raise(f, ~i);
      if (f != -INFINITY) s += ex2f(fmaf(f, LOG2E, -R));   // (a masked vocabulary entry adds nothing)
    };
    auto batch = [&](const uint4 (&v)[NV], int i) {
      const float best = Words<T>::max_of(v[0], v[1]);
      if (best > m) raise(best, i);   // (strict: an equal logit further on does not move the index)
      const uint64_t nr = pack2(-R, -R), sc = pack2(LOG2E, LOG2E);   // (only -inf so far: every term below is 0)
      uint64_t sum0 = 0, sum1 = 0;
#pragma unroll
      for (int u = 0; u < NV; ++u) {
#pragma unroll
        for (int k = 0; k < Words<T>::PAIRS; ++k) {
          float p, q;
          unpack2(fma2(Words<T>::pair(v[u], k), sc, nr), p, q);
          const uint64_t e = pack2(ex2f(p), ex2f(q));
          if (k & 1) sum1 = add2(sum1, e); else sum0 = add2(sum0, e);
        }
      }
      float p, q;
      unpack2(add2(sum0, sum1), p, q);
      s += p + q;
    };
    constexpr uint32_t ninf = sizeof(T) == 2 ? 0xFF80FF80u : 0xFF800000u;
    if (!bad) {
      if (lane < b0 - lo) one(lo + lane);
      auto load = [&](uint4 (&v)[NV], int i) {
#pragma unroll
        for (int u = 0; u < NV; ++u)   // vectors past the end are filled with -inf, which adds nothing
          v[u] = (i + u * STEP < b1) ? __ldg(reinterpret_cast<const uint4*>(x + i + u * STEP)) : make_uint4(ninf, ninf, ninf, ninf);
      };
      // a ring of DEPTH batches in registers: the loads of two batches are under way while one is worked on
      uint4 ring[DEPTH][NV];
      int i = b0 + lane * VEC;
#pragma unroll
      for (int k = 0; k < DEPTH - 1; ++k) load(ring[k], i + k * NV * STEP);
      while (i < b1) {
#pragma unroll
        for (int k = 0; k < DEPTH; ++k) {
          load(ring[(k + DEPTH - 1) % DEPTH], i + (DEPTH - 1) * NV * STEP);
          if (i < b1) batch(ring[k], i);
          i += NV * STEP;
        }
      }
      if (lane < hi - b1) one(b1 + lane);
    }
    grid_launch_dependents();
    // the maximum, the sum relative to it and the first index that holds it
    float M = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    if (fabsf(M) >= HUGE_LOGIT && fabsf(M) <= FLOAT_MAX) {   // (the same for the whole warp)
      s = sum_again<T>(x, lo + lane, hi, M);
    } else {
      s = m == -INFINITY ? 0.f : fabsf(m) < HUGE_LOGIT ? s * ex2f((m - M) * LOG2E - fmaf(m, LOG2E, -R)) : s;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    int idx = 0x7fffffff;
    if (m == M && M != -INFINITY) {
      idx = ~at;
      if (at >= 0) {
        idx = 0x7fffffff;
        uint4 v[NV];
#pragma unroll
        for (int u = 0; u < NV; ++u)
          v[u] = (at + u * STEP < b1) ? __ldg(reinterpret_cast<const uint4*>(x + at + u * STEP)) : make_uint4(ninf, ninf, ninf, ninf);
#pragma unroll
        for (int u = NV - 1; u >= 0; --u)
#pragma unroll
          for (int j = VEC - 1; j >= 0; --j)
            if (to_float(reinterpret_cast<const T*>(&v[u])[j]) == M) idx = at + u * STEP + j;
      }
    }
    idx = __reduce_min_sync(0xffffffffu, idx);
    int last = 0;
    if (lane == 0) {
      float* p = a.part + ((size_t)r * SAMPLE_MAX_SEGMENTS + seg) * 4;
      *reinterpret_cast<float4*>(p) = make_float4(M, s, __int_as_float(idx), 0.f);
      __threadfence();
      last = atomicAdd(a.counters + r, 1) == a.segments - 1;
      if (last) {
        a.counters[r] = 0;
        __threadfence();   // the other segments' partial results are visible from here on
      }
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();   // (lane 0's fence covers the warp's reads below)
    if (last) {
      // lane l combines segments l and l + 32, then a fixed shuffle tree
      const float* q = a.part + (size_t)r * SAMPLE_MAX_SEGMENTS * 4;
      Acc all{-INFINITY, 0.f, 0x7fffffff};
      for (int s2 = lane; s2 < a.segments; s2 += 32) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(q + 4 * s2));
        all = acc_merge(all, Acc{v.x, v.y, __float_as_int(v.z)});
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        Acc b;
        b.m = __shfl_xor_sync(0xffffffffu, all.m, o);
        b.s = __shfl_xor_sync(0xffffffffu, all.s, o);
        b.idx = __shfl_xor_sync(0xffffffffu, all.idx, o);
        all = acc_merge(all, b);
      }
      if (lane == 0) {
        if (bad) {
          a.token[r] = -1; a.conf[r] = 0.f;
          if (a.lse) a.lse[r] = 0.f;
          if (atomicCAS(a.status, 0, (int)LACACHE_ERR_INVALID_ARG) == 0) { a.status[1] = LOC_SAMPLE_ROW; a.status[2] = r; a.status[3] = row; }
        } else {
          a.token[r] = all.idx;
          a.conf[r] = 1.f / all.s;                       // exp(x_max - x_max) / sum
          if (a.lse) a.lse[r] = all.m + log2f(all.s) * LN2F;
        }
      }
    }
  }
}

}  // namespace

cudaError_t sample_rows(const SampleArgs& args, int num_sms, cudaStream_t s) {
  SampleArgs a = args;
  if (a.n_rows == 0) return cudaSuccess;
  // Segments per row: the fewest that keep 95 % of the resident warps busy over the waves the launch takes
  // (each wave but the last is full, so the rest of the last one is what idles), else the most even ones; at
  // least 1024 entries each, below which the chain at a segment's end costs more than the parallelism gives.
  const long long slots = (long long)Wide::CTAS * WARPS * num_sms;
  const int most = std::max(1, std::min(SAMPLE_MAX_SEGMENTS, a.vocab / 1024));
  double best = 0.0;
  a.segments = 1;
  for (int n = 1; n <= most && best < 0.95; ++n) {
    const long long w = (long long)a.n_rows * n, waves = (w + slots - 1) / slots;
    const double busy = (double)w / (double)(waves * slots);
    if (busy > best) { best = busy; a.segments = n; }
  }
  a.quota = ((a.vocab + a.segments - 1) / a.segments + 7) / 8 * 8;
  a.segments = (a.vocab + a.quota - 1) / a.quota;
  const long long n_warps = (long long)a.n_rows * a.segments;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((n_warps + WARPS - 1) / WARPS));
  cfg.blockDim = dim3(SAMPLE_THREADS);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.no_pdl ? 0 : 1;
  const bool deep = n_warps <= (long long)Deep::CTAS * WARPS * num_sms;
  if (a.dtype == LACACHE_DTYPE_BF16)
    return deep ? cudaLaunchKernelEx(&cfg, sample_rows_kernel<__nv_bfloat16, Deep>, a)
                : cudaLaunchKernelEx(&cfg, sample_rows_kernel<__nv_bfloat16, Wide>, a);
  return deep ? cudaLaunchKernelEx(&cfg, sample_rows_kernel<float, Deep>, a)
              : cudaLaunchKernelEx(&cfg, sample_rows_kernel<float, Wide>, a);
}

}  // namespace lacache

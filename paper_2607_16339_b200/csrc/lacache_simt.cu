// fp32 attention kernels (the fp32 dtype path, and any shape the tcgen05 path does not cover).
// One generic kernel runs every mode:
//   build : fixed queries x fixed keys            -> cached (m, l, O~)
//   step  : fixed queries x block keys, merged with the cached state
//           (Algorithm 1 reuse pass); block queries x all keys
//   full  : all queries x all keys (no cache)
// following the online-softmax recurrence of Eq. 2-6 with key tiles of 32.
//
// Mapping: a CTA of 4 warps owns 32 query rows of one (sequence, q head) and walks key tiles of 32; a warp has 16 of the rows
// and 16 keys of every tile, its own maxima and sums, and merges with the warp of the other 16 keys at the end.  A unit with
// many keys is cut over the S <= 8 CTAs of a thread-block cluster, whose online-softmax states are merged through distributed
// shared memory (how many: simt_row_parts, simt_step_parts).
//
// Products run on the tensor cores with fp32 accuracy: an operand is split in three bf16 parts that hold all its bits, x = hi + mid + lo,
// and a product is hi.hi + hi.mid + mid.hi + mid.mid + hi.lo + lo.hi (what is left out is 2^-24 of it at most and 2^-27 in the mean).
// The tensor cores cut a sum off where an fp32 addition rounds.  Of hi.hi, products of 16 bits, sixteen are added there, which seldom needs
// more than the 24 bits there are, and those sums in fp32; the others are 2^-8 of a product and less.  Error of the output against fp64
// (2-norm, 24 models of 90 to 650 tokens): 0.86e-7, and 3.0e-7 where scores are of order 50; chains of fp32 products on the CUDA cores
// 1.35e-7 and 4.6e-7.  Scores that one feature dominates: 0.43 to 0.6 of the chains' error, and 1.2 of it where the chains meet that feature
// last (one large channel, the last).  (Two tf32 parts, three products: 1.1e-7 and 3.6e-7, but operands of 22 bits: twice the chains' error
// where a score is one feature's product, and a row with one key does not return that key's value.)
//
// What bounds it: a tile of 128 features is 768 tensor-core instructions of 2 cycles, 1536 on an SM, and as many cycles of splitting (on
// the CUDA cores it took 5100, the shared-memory pipe's: every thread read its operands 16 bytes for 32 products).  Two CTAs to an SM (255
// registers a thread, 91 KB) are eight warps, whose instructions wait for the ones before: 3600 a tile.  Around the tiles it is latency:
// item and lists, the first tile's way, the merge of the parts, about 10000 cycles a CTA.  Builds with their RoPE launch, on the CUDA cores and now:
// 4 heads x 2564 tokens 480 -> 336 us, 32/8 x 664 242 -> 181, 16 x 1256 423 -> 304 (two tf32 parts 316, 170 and 285); steps of the
// same 50.0 -> 42.7, 51.7 -> 50.4, 54.8 -> 50.2 (40.5, 46.3, 46.0); of 28 drawn models 0.60 to 1.03 of the time on the CUDA cores (0.55 to 0.95).
//
// In a step the kernel rotates the block's rows itself, wherever it needs them,
// and leaves them in the rotated cache: one launch, no kernel in front of it.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "lacache_internal.h"
#include "lacache_plan.h"
#include "lacache_ptx.h"
#include "lacache_rope_math.h"

namespace lacache {
namespace {

using namespace ptx;

constexpr int KT = 32;       // keys per tile
constexpr int THREADS = 128; // warp w: rows 16 (w & 1) .. of the unit, keys 16 (w >> 1) .. of each tile

// Shared memory, in floats: the queries as operands of the tensor cores, [16 rows][16 features][part][lane][4], and keys and
// values [32][D] as they lie in the rotated cache, whose rows are swizzled so that the reads below meet no bank twice
// (simt_swz_qk, simt_swz_v).  After the last tile the first values' place holds the CTA's partial O~ [32][D], ML the partial
// (m, l); the first keys' place, what half of the warps hand to the others.
template <int D>
struct Smem {
  static constexpr int Q = 0;
  static constexpr int TILE = KT * D;
  static constexpr int K = Q + SIMT_ROWS * D * 3 / 2;  // two buffers of keys, two of values
  static constexpr int V = K + 2 * TILE;
  static constexpr int ML = V + 2 * TILE;
  static constexpr int ST = ML + 2 * SIMT_ROWS * 2;    // (m, l) of the rows' cached state
  static constexpr int BAR = ST + SIMT_ROWS * 2;       // barriers: keys 0 and 1, values 0 and 1 in place
  static constexpr int TOTAL = BAR + 8;
  static constexpr size_t bytes = TOTAL * sizeof(float);
  static_assert(SIMT_ROWS == KT, "the partial O~ over the values");
};

__device__ __forceinline__ void bulk_load(float* dst, const float* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Bounded wait (~2 s) for the bulk loads of a phase; one that runs out is reported and the values are whatever is there.
__device__ __forceinline__ void wait_loads(uint32_t bar, uint32_t parity, int32_t* status, int loc) {
  if (mbar_try(bar, parity)) return;
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (clock64() - t0 > 4000000000ll) {
      if (status && atomicCAS(status, 0, (int)LACACHE_ERR_TIMEOUT) == 0) { status[1] = loc; status[2] = blockIdx.x; status[3] = threadIdx.x; }
      return;
    }
  }
}
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_cluster_v2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
// D += A B on the warp's tensor core, 16 x 8 x 16, operands as bf16, fp32 sums
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (x0 in the lower half)
__device__ __forceinline__ uint32_t nearest_bf16(float x0, float x1) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
  return r;
}
// two fp32 values in one register pair: one instruction for both
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float2 scaled2(float a, float b, float by) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pack2(a, b)), "l"(pack2(by, by)));
  return unpack2(d);
}
__device__ __forceinline__ float bf16_lower(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf16_upper(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }
__device__ __forceinline__ float2 less2(float2 x, float h0, float h1) { return unpack2(fma2(pack2(h0, h1), pack2(-1.f, -1.f), pack2(x.x, x.y))); }
// x = hi + mid + lo of a pair of values (x0 in the lower halves): each the nearest bf16 value of what is left, so that the three
// hold all 24 bits of x (unless the last lie below the smallest bf16 value)
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  float2 x = make_float2(x0, x1);
  hi = nearest_bf16(x.x, x.y);
  x = less2(x, bf16_lower(hi), bf16_upper(hi));
  mid = nearest_bf16(x.x, x.y);
  x = less2(x, bf16_lower(mid), bf16_upper(mid));
  lo = nearest_bf16(x.x, x.y);
}
// ... of two values each of two rows, a and b, paired across the rows
__device__ __forceinline__ void split3_across(float2 a, float2 b, uint32_t (&x)[3], uint32_t (&y)[3]) {
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    x[p] = nearest_bf16(a.x, b.x);
    y[p] = nearest_bf16(a.y, b.y);
    if (p == 2) break;
    a = less2(a, bf16_lower(x[p]), bf16_lower(y[p]));
    b = less2(b, bf16_upper(x[p]), bf16_upper(y[p]));
  }
}
__device__ __forceinline__ float4 load4(const void* base, size_t off, bool bf16) {
  if (!bf16) return *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + off);
  const uint2 u = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(base) + off);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
// features c .. c + 3 (x1) and their partners c + d/2 .. (x2) of a raw row, rotated with the RoPE kernel's own
// roundings
__device__ __forceinline__ void rotate4(float4 x1, float4 x2, float4 cs, float4 sn, float4& y1, float4& y2) {
  auto lo = [](float p, float q, float co, float si) { return __fsub_rn(__fmul_rn(p, co), __fmul_rn(q, si)); };
  auto hi = [](float p, float q, float co, float si) { return __fadd_rn(__fmul_rn(q, co), __fmul_rn(p, si)); };
  y1 = make_float4(lo(x1.x, x2.x, cs.x, sn.x), lo(x1.y, x2.y, cs.y, sn.y), lo(x1.z, x2.z, cs.z, sn.z), lo(x1.w, x2.w, cs.w, sn.w));
  y2 = make_float4(hi(x1.x, x2.x, cs.x, sn.x), hi(x1.y, x2.y, cs.y, sn.y), hi(x1.z, x2.z, cs.z, sn.z), hi(x1.w, x2.w, cs.w, sn.w));
}

// STEP: a launch of a step.  What only steps do, the rows they rotate and the state they start from, is code that a build's CTAs would
// fetch around, and the other way: with two tf32 parts one instantiation for both took a small build and step 55.8 us (two 53.3), the
// tiny model's step 6.05 (5.65).
template <int D, bool STEP>
__global__ void __launch_bounds__(THREADS, D == 128 ? 2 : 3) simt_attn_kernel(const __grid_constant__ Geometry g,
                                                              const __grid_constant__ AttnArgs a) {
  using SM = Smem<D>;
  constexpr int D4 = D / 4;          // 16-byte columns of a row
  extern __shared__ __align__(16) float sm[];

  // the first n_split_items items are cut over the `split` CTAs of a cluster, the others take one CTA each
  const int S = a.split_ctas;
  int item = (int)blockIdx.x, part = 0, n_parts = 1;
  if (item < a.n_split_items * S) {
    part = item % S;
    item /= S;
    n_parts = S;
  } else {
    item -= a.n_split_items * (S - 1);
    if (item >= a.n_items) return;   // (the last cluster's filling; its CTAs are not split)
  }
  const WorkItem it = a.items[item];
  const int h = blockIdx.y;
  const int kh = h / g.group;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bs = a.blk_start ? a.blk_start[it.seq] : 0;
  const int be = bs + g.block_len;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(sm + SM::BAR) + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int k0 = it.seq_start, k1 = it.seq_end, x0 = 0, x1 = 0;
  bool from_state = false, to_state = false;
  if (!STEP && a.mode == MODE_BUILD) {
    x0 = bs; x1 = be; to_state = true;
  } else if (STEP && it.kind == ITEM_ROWS) {
    k0 = bs; k1 = be; from_state = true;
  }
  const bool raw = STEP && a.k_raw != nullptr;                    // a step that rotates the block's rows here
  const bool q_raw = raw && it.kind == ITEM_BLOCK_CHUNK;  // (these rows' queries are the block's)
  const size_t blk_row0 = (size_t)it.seq * g.block_len;   // the sequence's first row of the block's inputs

  float* const qr = reinterpret_cast<float*>(a.rot.q_hi) + (size_t)h * g.Tp * D;
  float* const kr = reinterpret_cast<float*>(a.rot.k_hi) + (size_t)kh * g.Tp * D;
  float* const vr = reinterpret_cast<float*>(a.rot.v) + (size_t)kh * g.Tp * D;

  // the key tiles of this CTA's part (a tile wholly inside the excluded block holds nothing)
  const int n_tiles_all = (k1 - k0 + KT - 1) / KT;
  const int t_begin = n_tiles_all * part / n_parts, t_end = n_tiles_all * (part + 1) / n_parts;
  auto next_tile = [&](int t) {
    for (; t < t_end; ++t) {
      const int kt = k0 + t * KT;
      if (!(x1 > x0 && kt >= x0 && min(kt + KT, k1) <= x1)) break;
    }
    return t;
  };
  float* const Ks = sm + SM::K;
  float* const Vs = sm + SM::V;
  const bool writes_cache = q_raw && it.row0 == bs && h % g.group == 0;   // leaves the block's keys and values in the cache

  // Tiles are contiguous in the cache: a bulk copy each, the next tile's under way while a tile is computed (two buffers).  Only the
  // sequence's own rows are read (those behind are another's, which another CTA may be writing): the values that miss are zero, as
  // their weights are, and the scores are masked, whatever the keys' place holds.
  const uint32_t bar_k = smem_u32(sm + SM::BAR), bar_v = bar_k + 16;
  auto issue_tile = [&](int t, int buf) {
    const int kt = k0 + t * KT, n = min(KT, k1 - kt);
    float* const Vb = Vs + buf * SM::TILE;
#pragma unroll 1
    for (int i = n * D4 + threadIdx.x; i < KT * D4; i += THREADS) *reinterpret_cast<float4*>(Vb + i * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x != 0) return;
    fence_async_smem();   // (a tile that the threads stored may have been there)
    mbar_expect_tx(bar_k + 8 * buf, n * D * 4);
    bulk_load(Ks + buf * SM::TILE, kr + (size_t)kt * D, n * D * 4, bar_k + 8 * buf);
    mbar_expect_tx(bar_v + 8 * buf, n * D * 4);
    bulk_load(Vb, vr + (size_t)kt * D, n * D * 4, bar_v + 8 * buf);
  };
  // A tile that holds block rows of a step is loaded by all threads, who rotate the block's rows (BATCH raw rows' loads leave
  // together) and take the others from the cache.
  auto is_mixed = [&](int t) { return raw && k0 + t * KT < be && k0 + t * KT + KT > bs; };
  auto load_mixed = [&](auto batch, int t, float* Kb, float* Vb) {
    const int kt = k0 + t * KT;
    constexpr int N = KT * (D4 / 2) / THREADS, BATCH = decltype(batch)::value < N ? decltype(batch)::value : N;   // a key's two halves, its values'
    static_assert(N % BATCH == 0, "whole batches");
#pragma unroll 1
    for (int b = 0; b < N; b += BATCH) {
      float4 x1[BATCH], x2[BATCH], cs[BATCH], sn[BATCH], v1[BATCH], v2[BATCH];
#pragma unroll
      for (int j = 0; j < BATCH; ++j) {
        const int i = threadIdx.x + (b + j) * THREADS, c = (i % (D4 / 2)) * 4, key = kt + i / (D4 / 2);
        if (raw && key >= bs && key < be) {
          const size_t row = blk_row0 + (key - bs), off = (row * g.Hkv + kh) * D + c;
          x1[j] = load4(a.k_raw, off, a.raw_bf16);
          x2[j] = load4(a.k_raw, off + D / 2, a.raw_bf16);
          cs[j] = *reinterpret_cast<const float4*>(a.row_cos + row * (D / 2) + c);
          sn[j] = *reinterpret_cast<const float4*>(a.row_sin + row * (D / 2) + c);
          v1[j] = load4(a.v_raw, off, a.raw_bf16);
          v2[j] = load4(a.v_raw, off + D / 2, a.raw_bf16);
        } else if (key >= k1) {
          x1[j] = x2[j] = v1[j] = v2[j] = make_float4(0.f, 0.f, 0.f, 0.f);   // (as above)
        } else {
          const float* src = kr + (size_t)key * D + (c ^ simt_swz_qk(key));
          x1[j] = *reinterpret_cast<const float4*>(src);
          x2[j] = *reinterpret_cast<const float4*>(src + D / 2);
          src = vr + (size_t)key * D + (c ^ simt_swz_v(key));
          v1[j] = *reinterpret_cast<const float4*>(src);
          v2[j] = *reinterpret_cast<const float4*>(src + D / 2);
        }
      }
#pragma unroll
      for (int j = 0; j < BATCH; ++j) {
        const int i = threadIdx.x + (b + j) * THREADS, r = i / (D4 / 2), c = (i % (D4 / 2)) * 4, key = kt + r;
        const int ck = c ^ simt_swz_qk(key), cv = c ^ simt_swz_v(key);   // (as rows lie in the cache)
        float4 y1 = x1[j], y2 = x2[j];
        if (raw && key >= bs && key < be) {
          rotate4(x1[j], x2[j], cs[j], sn[j], y1, y2);
          if (writes_cache) {
            *reinterpret_cast<float4*>(kr + (size_t)key * D + ck) = y1;
            *reinterpret_cast<float4*>(kr + (size_t)key * D + ck + D / 2) = y2;
            *reinterpret_cast<float4*>(vr + (size_t)key * D + cv) = v1[j];
            *reinterpret_cast<float4*>(vr + (size_t)key * D + cv + D / 2) = v2[j];
          }
        }
        *reinterpret_cast<float4*>(Kb + r * D + ck) = y1;
        *reinterpret_cast<float4*>(Kb + r * D + ck + D / 2) = y2;
        *reinterpret_cast<float4*>(Vb + r * D + cv) = v1[j];
        *reinterpret_cast<float4*>(Vb + r * D + cv + D / 2) = v2[j];
      }
    }
  };
  using Few = std::integral_constant<int, 1>;     // (beside the accumulators)
  using Many = std::integral_constant<int, 4>;

  int t = next_tile(t_begin);
  // Launched programmatically dependent: but for the lists above, which nothing writes, nothing is touched before the grids
  // ahead have completed; this grid's launch and those two round trips to L2 overlap their end.
  grid_dependency_wait();
  // (the cached state of a step's fixed rows: m and l now, O~ behind the last tile's keys)
  float m_st = -INFINITY, l_st = 0.f;
  if (from_state && warp == 3 && lane < it.nrows) {
    m_st = a.st.m[(size_t)h * g.Tp + it.row0 + lane];
    l_st = a.st.l[(size_t)h * g.Tp + it.row0 + lane];
  }
  if (t < t_end && !is_mixed(t)) issue_tile(t, 0);
  // The queries, as operands: a thread takes rows g and g + 8 of a warp's sixteen, and of both four features of a step and their
  // partners (registers 0 and 2: row g, features 0 1 and 2 3).  Times 2^24, so that the parts of small ones are bf16 values too.
  bool bad = false;   // the unit is to be done with plain products (below)
  {
    // (what a key loses where its parts are smaller than any bf16 value is nothing beside a score, unless the query is huge)
    const float q_most = fminf(0x1p80f / fabsf(g.scale_log2), 0x1p100f);
    constexpr int STEPS = D / 16, N = STEPS / (THREADS / 32);
    uint4* const qf = reinterpret_cast<uint4*>(sm + SM::Q);
    float4 x1[N][2], x2[N][2], cs[N][2], sn[N][2];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int i = warp + j * (THREADS / 32), c = 16 * (i % (STEPS / 2)) + (lane & 3) * 4;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int r = min(16 * (i / (STEPS / 2)) + (lane >> 2) + 8 * e, it.nrows - 1);
        if (q_raw) {
          const size_t row = blk_row0 + (it.row0 - bs) + r, off = (row * g.Hq + h) * D + c, tab = row * (D / 2) + c;
          x1[j][e] = load4(a.q_raw, off, a.raw_bf16);
          x2[j][e] = load4(a.q_raw, off + D / 2, a.raw_bf16);
          cs[j][e] = *reinterpret_cast<const float4*>(a.row_cos + tab);
          sn[j][e] = *reinterpret_cast<const float4*>(a.row_sin + tab);
        } else {
          const float* const src = qr + (size_t)(it.row0 + r) * D + (c ^ simt_swz_qk(it.row0 + r));
          x1[j][e] = *reinterpret_cast<const float4*>(src);
          x2[j][e] = *reinterpret_cast<const float4*>(src + D / 2);
        }
      }
    }
    if (t < t_end && is_mixed(t)) load_mixed(Many(), t, Ks, Vs);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int i = warp + j * (THREADS / 32), rw = i / (STEPS / 2), step = i % (STEPS / 2);
      if (q_raw) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int r = 16 * rw + (lane >> 2) + 8 * e;
          rotate4(x1[j][e], x2[j][e], cs[j][e], sn[j][e], x1[j][e], x2[j][e]);
          if (part == 0 && r < it.nrows) {
            float* const dst = qr + (size_t)(it.row0 + r) * D + ((16 * step + (lane & 3) * 4) ^ simt_swz_qk(it.row0 + r));
            *reinterpret_cast<float4*>(dst) = x1[j][e];
            *reinterpret_cast<float4*>(dst + D / 2) = x2[j][e];
          }
        }
      }
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        uint32_t p[3][4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float4 x = f ? x2[j][e] : x1[j][e];
          bad = bad || !(fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))) <= q_most);
          split3(x.x * 0x1p24f, x.y * 0x1p24f, p[0][e], p[1][e], p[2][e]);
          split3(x.z * 0x1p24f, x.w * 0x1p24f, p[0][2 + e], p[1][2 + e], p[2][2 + e]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) qf[((rw * STEPS + step + f * (STEPS / 2)) * 3 + k) * 32 + lane] = make_uint4(p[k][0], p[k][1], p[k][2], p[k][3]);
      }
    }
  }

  // The warp's 16 rows x 16 keys of a tile, as the tensor cores lay them out: this thread has rows g and g + 8, keys 2 t and
  // 2 t + 1 of either eight (of the scores as of P.V's operand, so that a thread's probabilities are its operand), and features
  // 32 q + 8 t .. + 7 of O~.  A step of the scores is 16 features, of which this thread has 4 t .. + 3 (k index 2 t, 2 t + 1, 2 t + 8, 2 t + 9).
  const int g8 = lane >> 2, t4 = lane & 3, rw = warp & 1, kw = warp >> 1;
  const bool rows = 16 * rw < it.nrows;   // this warp has rows (the others only help loading)
  // (where the thread's first 16 bytes of a row lie, the rows' parity and pairs counted from the cache's first row: tiles are
  // 32 rows apart, so it is the same place in every tile)
  const uint4* const qp = reinterpret_cast<const uint4*>(sm + SM::Q) + rw * (D / 16) * 3 * 32 + lane;
  const float* const kp0 = Ks + (16 * kw + g8) * D + ((4 * t4) ^ simt_swz_qk(k0 + g8));
  const float* const vpa = Vs + (16 * kw + 2 * t4) * D + ((4 * g8) ^ simt_swz_v(k0 + 2 * t4));
  const float* const vpb = Vs + (16 * kw + 2 * t4 + 1) * D + ((4 * g8) ^ simt_swz_v(k0 + 2 * t4 + 1));
  const int kflip = simt_swz_qk(k0 + g8) ? -16 : 16;   // to the next 16 features
  float m[2], l[2], past = 0.f;
  float o[D / 8][4];   // [4 q + j]: {row g: features 8 t + j, 8 t + 4 + j; row g + 8: likewise} of the 32 from 32 q
#pragma unroll
  for (int i = 0; i < 2; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
#pragma unroll
  for (int i = 0; i < D / 8; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) o[i][c] = 0.f;
  uint32_t phases = 0;   // bit b: phase of buffer b's barriers
  int buf = 0;
  for (; t < t_end; buf ^= 1) {
    const int tn = next_tile(t + 1);
    __syncthreads();   // every warp is done with the tile before (and what the threads stored of this one is there)
    if (tn < t_end) {
      if (!is_mixed(tn)) {
        issue_tile(tn, buf ^ 1);
      } else {
        load_mixed(Few(), tn, Ks + (buf ^ 1) * SM::TILE, Vs + (buf ^ 1) * SM::TILE);
      }
    }
    if (from_state && tn >= t_end && threadIdx.x == 0) {   // the rows' cached O~, into the buffer that no further keys need
      fence_async_smem();
      const uint32_t bytes = it.nrows * D * 4;
      mbar_expect_tx(bar_k + 8 * (buf ^ 1), bytes);
      bulk_load(Ks + (buf ^ 1) * SM::TILE, a.st.o + ((size_t)h * g.Tp + it.row0) * D, bytes, bar_k + 8 * (buf ^ 1));
    }
    const bool bulk = !is_mixed(t);
    const uint32_t phase = (phases >> buf) & 1u;
    if (bulk) {
      wait_loads(bar_k + 8 * buf, phase, a.status, LOC_WAIT_K);
      phases ^= 1u << buf;
    }
    const float* const kp = kp0 + buf * SM::TILE;
    const float* const vp0 = vpa + buf * SM::TILE;
    const float* const vp1 = vpb + buf * SM::TILE;
    float s[2][4];
    if (rows) {
      // Six products: hi.hi, whose 16 bits leave room for a sum of sixteen, over one step at a time and then added with rounding, for
      // the tensor cores cut sums off; the others, 2^-8 and less of it, in two sums of their own.
      float small[2][2][4];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) { s[n][c] = 0.f; small[n][0][c] = 0.f; small[n][1][c] = 0.f; }
#pragma unroll
      for (int c0 = 0; c0 < D; c0 += 32) {
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
          uint32_t qx[3][4];   // [part][operand register]
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const uint4 u = qp[((c0 / 16 + cc) * 3 + j) * 32];
            qx[j][0] = u.x; qx[j][1] = u.y; qx[j][2] = u.z; qx[j][3] = u.w;
          }
#pragma unroll
          for (int n = 0; n < 2; ++n) {
            const float4 k4 = *reinterpret_cast<const float4*>(kp + 8 * n * D + c0 + (cc ? kflip : 0));
            uint32_t kx[3][2];
            split3(k4.x, k4.y, kx[0][0], kx[1][0], kx[2][0]);
            split3(k4.z, k4.w, kx[0][1], kx[1][1], kx[2][1]);
            float big[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(big, qx[0], kx[0][0], kx[0][1]);
            mma_bf16(small[n][0], qx[1], kx[0][0], kx[0][1]);
            mma_bf16(small[n][1], qx[2], kx[0][0], kx[0][1]);
            mma_bf16(small[n][0], qx[0], kx[1][0], kx[1][1]);
            mma_bf16(small[n][1], qx[1], kx[1][0], kx[1][1]);
            mma_bf16(small[n][1], qx[0], kx[2][0], kx[2][1]);
#pragma unroll
            for (int c = 0; c < 4; ++c) s[n][c] += big[c];
          }
        }
      }
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[n][c] += small[n][0][c] + small[n][1][c];
    }
    if (bulk) wait_loads(bar_v + 8 * buf, phase, a.status, LOC_WAIT_V);
    if (rows) {
      float alpha[2];
      bool ok[2][2];
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int key = k0 + t * KT + 16 * kw + 8 * n + 2 * t4 + e;
          ok[n][e] = key < k1 && !(key >= x0 && key < x1);
        }
#pragma unroll
      for (int i = 0; i < 2; ++i) {   // rows g and g + 8
        float a[2][2], mx = -INFINITY;
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (ok[n][e]) past = fmaf(s[n][2 * i + e], 0.f, past);   // (NaN from a score that is none)
            a[n][e] = ok[n][e] ? s[n][2 * i + e] * 0x1p-24f * g.scale_log2 : -INFINITY;
            mx = fmaxf(mx, a[n][e]);
          }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m[i], mx);
        const float m_use = m_new == -INFINITY ? 0.f : m_new;
        alpha[i] = m[i] == -INFINITY ? 0.f : exp2f(m[i] - m_new);
        m[i] = m_new;
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            s[n][2 * i + e] = ok[n][e] ? exp2f(a[n][e] - m_use) : 0.f;
          }
        l[i] = l[i] * alpha[i] + ((s[0][2 * i] + s[0][2 * i + 1]) + (s[1][2 * i] + s[1][2 * i + 1]));
      }
      uint32_t px[3][4];   // (times 2^24, as the values below: all parts of all fp32 values are bf16 values)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 2; ++i)
          split3(s[n][2 * i] * 0x1p24f, s[n][2 * i + 1] * 0x1p24f, px[0][2 * n + i], px[1][2 * n + i], px[2][2 * n + i]);
#pragma unroll
      for (int q = 0; q < D / 32; ++q) {
        uint32_t vx[2][4][3];   // [operand register: keys 2 t and 2 t + 1 of either eight][feature][part]
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          const float4 va = *reinterpret_cast<const float4*>(vp0 + 8 * n * D + 32 * q);
          const float4 vb = *reinterpret_cast<const float4*>(vp1 + 8 * n * D + 32 * q);
          split3_across(scaled2(va.x, va.y, 0x1p24f), scaled2(vb.x, vb.y, 0x1p24f), vx[n][0], vx[n][1]);
          split3_across(scaled2(va.z, va.w, 0x1p24f), scaled2(vb.z, vb.w, 0x1p24f), vx[n][2], vx[n][3]);
        }
        float pv[4][4] = {}, small[4][4] = {};
        auto all = [&](float (&d)[4][4], int x, int y) {
#pragma unroll
          for (int j = 0; j < 4; ++j) mma_bf16(d[j], px[x], vx[0][j][y], vx[1][j][y]);
        };
        all(pv, 0, 0);
        all(small, 1, 1); all(small, 2, 0); all(small, 0, 2); all(small, 1, 0); all(small, 0, 1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) o[4 * q + j][c] = fmaf(o[4 * q + j][c], alpha[c >> 1], pv[j][c] + small[j][c]);
      }
    }
    t = tn;
  }
  // Infinities, NaN and values of 2^80 and more leave a sum behind that is none, or were seen in the queries: the unit is then done
  // once more with plain products and sums, where they give what they give.
  if (rows) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float z = fmaf(l[i], 0.f, past);
#pragma unroll
      for (int f = 0; f < D / 8; ++f)
#pragma unroll
        for (int e = 2 * i; e < 2 * i + 2; ++e) {
          z = fmaf(o[f][e], 0.f, z);
          o[f][e] *= 0x1p-48f;
        }
      bad = bad || (16 * rw + g8 + 8 * i < it.nrows && !(z == 0.f));
    }
  }
  const bool plain = __syncthreads_or(bad);   // (every warp has left the keys and values behind)
  float* const Kl = Ks + (buf ^ 1) * SM::TILE;   // the last tile's keys' place; the cached O~ is in the other one

  if (a.step_overlap) grid_launch_dependents();
  // the partial states of the rows to shared memory
  if (plain) {
    // Eight threads for two rows, each with every eighth 16 bytes of their features: they read a key's and a value's row side by side,
    // and share a score's sum; four keys at a time.  What bounds it is the shared-memory pipe, four cycles for the 16 bytes that
    // serve eight products.  Build of 4 heads x 2564 tokens whose units are all done again: 1351 us, without 343; one of 32/8 heads x
    // 664 tokens 710 (189); its step 74 (57).  (Four threads a row, a value of theirs at a time, a key at a time: 10900, 5400 and 270.)
    const int r = threadIdx.x >> 3, c0 = (threadIdx.x & 7) * 4;
    constexpr int NC = D / 32;
    float4 qv[2][NC], acc[2][NC];
    float M[2] = {-INFINITY, -INFINITY}, L[2] = {0.f, 0.f};
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int tok = it.row0 + min(r + 16 * e, it.nrows - 1);
      if (q_raw) {
        const size_t row = blk_row0 + (tok - bs), off = (row * g.Hq + h) * D + c0, tab = row * (D / 2) + c0;
#pragma unroll
        for (int i = 0; i < NC / 2; ++i)
          rotate4(load4(a.q_raw, off + 32 * i, a.raw_bf16), load4(a.q_raw, off + 32 * i + D / 2, a.raw_bf16),
                  *reinterpret_cast<const float4*>(a.row_cos + tab + 32 * i), *reinterpret_cast<const float4*>(a.row_sin + tab + 32 * i),
                  qv[e][i], qv[e][i + NC / 2]);
      } else {
#pragma unroll
        for (int i = 0; i < NC; ++i) qv[e][i] = *reinterpret_cast<const float4*>(qr + (size_t)tok * D + ((c0 + 32 * i) ^ simt_swz_qk(tok)));
      }
#pragma unroll
      for (int i = 0; i < NC; ++i) acc[e][i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll 1
    for (t = next_tile(t_begin); t < t_end; t = next_tile(t + 1)) {
      load_mixed(Many(), t, Kl, Vs);
      __syncthreads();
#pragma unroll 1
      for (int j0 = 0; j0 < KT; j0 += 4) {
        const int key0 = k0 + t * KT + j0;
        auto counts = [&](int j) { return key0 + j < k1 && !(key0 + j >= x0 && key0 + j < x1); };   // (the same in every thread)
        float sc[2][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float4 s4[2] = {};
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            const float4 k4 = *reinterpret_cast<const float4*>(Kl + (j0 + j) * D + ((c0 + 32 * i) ^ simt_swz_qk(key0 + j)));
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              s4[e].x = fmaf(qv[e][i].x, k4.x, s4[e].x); s4[e].y = fmaf(qv[e][i].y, k4.y, s4[e].y);
              s4[e].z = fmaf(qv[e][i].z, k4.z, s4[e].z); s4[e].w = fmaf(qv[e][i].w, k4.w, s4[e].w);
            }
          }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            sc[e][j] = (s4[e].x + s4[e].y) + (s4[e].z + s4[e].w);
#pragma unroll
            for (int x = 1; x < 8; x <<= 1) sc[e][j] += __shfl_xor_sync(0xffffffffu, sc[e][j], x);
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float m_new = M[e];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            sc[e][j] = counts(j) ? sc[e][j] * g.scale_log2 : -INFINITY;
            m_new = fmaxf(m_new, sc[e][j]);
          }
          const float al = M[e] == -INFINITY ? 0.f : exp2f(M[e] - m_new), m_use = m_new == -INFINITY ? 0.f : m_new;
          M[e] = m_new;
          L[e] *= al;
#pragma unroll
          for (int i = 0; i < NC; ++i) { acc[e][i].x *= al; acc[e][i].y *= al; acc[e][i].z *= al; acc[e][i].w *= al; }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            sc[e][j] = exp2f(sc[e][j] - m_use);
            if (counts(j)) L[e] += sc[e][j];
          }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (!counts(j)) continue;   // (its value may be anything)
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            const float4 v4 = *reinterpret_cast<const float4*>(Vs + (j0 + j) * D + ((c0 + 32 * i) ^ simt_swz_v(key0 + j)));
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float p = sc[e][j];
              acc[e][i].x = fmaf(p, v4.x, acc[e][i].x); acc[e][i].y = fmaf(p, v4.y, acc[e][i].y);
              acc[e][i].z = fmaf(p, v4.z, acc[e][i].z); acc[e][i].w = fmaf(p, v4.w, acc[e][i].w);
            }
          }
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
      for (int i = 0; i < NC; ++i) *reinterpret_cast<float4*>(Vs + (r + 16 * e) * D + c0 + 32 * i) = acc[e][i];
      if (c0 == 0) *reinterpret_cast<float2*>(sm + SM::ML + (r + 16 * e) * 2) = make_float2(M[e], L[e]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int x = 1; x < 4; x <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], x);
    // the warps of the upper 16 keys hand theirs to those of the lower 16, who hold the same rows and features
    float4* const hand = reinterpret_cast<float4*>(Kl) + rw * (D / 8) * 32 + lane;
    float* const ml = sm + SM::ML;
    const int r0 = 16 * rw + g8;
    if (kw == 1 && rows) {
#pragma unroll
      for (int f = 0; f < D / 8; ++f) hand[f * 32] = make_float4(o[f][0], o[f][1], o[f][2], o[f][3]);
      if (t4 == 0)
#pragma unroll
        for (int i = 0; i < 2; ++i) *reinterpret_cast<float2*>(ml + (SIMT_ROWS + r0 + 8 * i) * 2) = make_float2(m[i], l[i]);
    }
    __syncthreads();
    if (kw == 0 && rows) {
      float w0[2], w1[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float2 other = *reinterpret_cast<const float2*>(ml + (SIMT_ROWS + r0 + 8 * i) * 2);
        const float M = fmaxf(m[i], other.x);
        w0[i] = m[i] == -INFINITY ? 0.f : exp2f(m[i] - M);
        w1[i] = other.x == -INFINITY ? 0.f : exp2f(other.x - M);
        if (t4 == 0) *reinterpret_cast<float2*>(ml + (r0 + 8 * i) * 2) = make_float2(M, fmaf(other.y, w1[i], l[i] * w0[i]));
      }
#pragma unroll
      for (int f = 0; f < D / 8; ++f) {
        const float4 x = hand[f * 32];
        o[f][0] = fmaf(x.x, w1[0], o[f][0] * w0[0]); o[f][1] = fmaf(x.y, w1[0], o[f][1] * w0[0]);
        o[f][2] = fmaf(x.z, w1[1], o[f][2] * w0[1]); o[f][3] = fmaf(x.w, w1[1], o[f][3] * w0[1]);
      }
      float* const dst = Vs + r0 * D + 8 * t4;
#pragma unroll
      for (int q = 0; q < D / 32; ++q)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          float* const d = dst + 8 * i * D + 32 * q;
          *reinterpret_cast<float4*>(d) = make_float4(o[4 * q][2 * i], o[4 * q + 1][2 * i], o[4 * q + 2][2 * i], o[4 * q + 3][2 * i]);
          *reinterpret_cast<float4*>(d + 4) = make_float4(o[4 * q][2 * i + 1], o[4 * q + 1][2 * i + 1], o[4 * q + 2][2 * i + 1], o[4 * q + 3][2 * i + 1]);
        }
    }
  }
  // the partial states of a row -- one of every CTA of the cluster, and the cached state -- merged (Eq. 2-6), 16 bytes of a row
  // per thread and ITEMS of them at a time, PARTS partial states' loads in flight; a split unit's rows are dealt out over its CTAs
  if (from_state && warp == 3) *reinterpret_cast<float2*>(sm + SM::ST + lane * 2) = make_float2(m_st, l_st);
  if (n_parts > 1) cluster_sync_all();
  else __syncthreads();
  if (from_state) wait_loads(bar_k + 8 * buf, (phases >> buf) & 1u, a.status, LOC_WAIT_O);
  const float* const o_st = Ks + buf * SM::TILE;
  const uint32_t sm_base = smem_u32(sm);
  const int n_out = (it.nrows - part + n_parts - 1) / n_parts * D4;
  auto merge = [&](auto items, auto parts) {
    constexpr int ITEMS = decltype(items)::value, PARTS = decltype(parts)::value;
    const float LN2 = 0.69314718055994530942f;
#pragma unroll 1
    for (int i0 = threadIdx.x; i0 < n_out; i0 += ITEMS * THREADS) {
      float M[ITEMS], L[ITEMS];
      float4 acc[ITEMS];
#pragma unroll
      for (int b = 0; b < ITEMS; ++b) {
        M[b] = -INFINITY; L[b] = 0.f;
        acc[b] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (from_state) {   // (a unit that is not cut)
          const int i = min(i0 + b * THREADS, n_out - 1);
          const float2 ml = *reinterpret_cast<const float2*>(sm + SM::ST + (i / D4) * 2);
          M[b] = ml.x;
          L[b] = ml.y;
          acc[b] = *reinterpret_cast<const float4*>(o_st + i * 4);
        }
      }
#pragma unroll 1
      for (int p0 = 0; p0 < n_parts; p0 += PARTS) {
        float2 ml[ITEMS][PARTS];
        float4 v[ITEMS][PARTS];
#pragma unroll
        for (int k = 0; k < PARTS; ++k) {
          const uint32_t base = n_parts > 1 ? mapa_shared(sm_base, (uint32_t)min(p0 + k, n_parts - 1)) : sm_base;
#pragma unroll
          for (int b = 0; b < ITEMS; ++b) {
            const int i = min(i0 + b * THREADS, n_out - 1), r = part + (i / D4) * n_parts;
            ml[b][k] = ld_cluster_v2(base + (SM::ML + r * 2) * 4);
            v[b][k] = ld_cluster_v4(base + (SM::V + r * D + (i % D4) * 4) * 4);
          }
        }
#pragma unroll
        for (int b = 0; b < ITEMS; ++b) {
          float Mn = M[b];
#pragma unroll
          for (int k = 0; k < PARTS; ++k) Mn = fmaxf(Mn, ml[b][k].x);
          const float w0 = M[b] == -INFINITY ? 0.f : exp2f(M[b] - Mn);
          L[b] *= w0; acc[b].x *= w0; acc[b].y *= w0; acc[b].z *= w0; acc[b].w *= w0;
#pragma unroll
          for (int k = 0; k < PARTS; ++k) {
            const float w = (p0 + k >= n_parts || ml[b][k].x == -INFINITY) ? 0.f : exp2f(ml[b][k].x - Mn);
            L[b] = fmaf(ml[b][k].y, w, L[b]);
            acc[b].x = fmaf(v[b][k].x, w, acc[b].x); acc[b].y = fmaf(v[b][k].y, w, acc[b].y);
            acc[b].z = fmaf(v[b][k].z, w, acc[b].z); acc[b].w = fmaf(v[b][k].w, w, acc[b].w);
          }
          M[b] = Mn;
        }
      }
#pragma unroll
      for (int b = 0; b < ITEMS; ++b) {
        const int i = i0 + b * THREADS;
        if (i >= n_out) break;
        const int tok = it.row0 + part + (i / D4) * n_parts, c4 = i % D4;
        if (to_state) {
          const size_t srow = (size_t)h * g.Tp + tok;
          if (c4 == 0) { a.st.m[srow] = M[b]; a.st.l[srow] = L[b]; }
          *reinterpret_cast<float4*>(a.st.o + srow * D + c4 * 4) = acc[b];
        } else {
          const float inv = 1.f / L[b];
          const size_t orow = (size_t)tok * g.Hq + h;
          const float4 y = make_float4(acc[b].x * inv, acc[b].y * inv, acc[b].z * inv, acc[b].w * inv);
          if (a.out_bf16) {
            const __nv_bfloat162 b0 = __floats2bfloat162_rn(y.x, y.y), b1 = __floats2bfloat162_rn(y.z, y.w);
            uint2 u;
            u.x = *reinterpret_cast<const uint32_t*>(&b0);
            u.y = *reinterpret_cast<const uint32_t*>(&b1);
            *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + orow * D + c4 * 4) = u;
          } else {
            *reinterpret_cast<float4*>(a.out + orow * D + c4 * 4) = y;
          }
          if (a.lse && c4 == 0) a.lse[orow] = (M[b] + log2f(L[b])) * LN2;
        }
      }
    }
  };
  if (n_parts <= 2) merge(std::integral_constant<int, 4>(), std::integral_constant<int, 2>());
  else merge(std::integral_constant<int, 2>(), std::integral_constant<int, 4>());
  if (n_parts > 1) cluster_sync_all();   // the partner CTAs may still read this one's shared memory
}

constexpr size_t SMEM_ALONE = 116 * 1024, SMEM_TWO = 78 * 1024;   // one CTA to an SM, two

template <int D>
cudaError_t launch(const Geometry& g, const AttnArgs& a, int n_ctas, int num_sms, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n_ctas, (unsigned)g.Hq);
  cfg.blockDim = dim3(THREADS);
  // The kernel ahead still holds SMs when CTAs of this one are placed, and they pile up on the others: where all would find an
  // SM of their own, or one with one other, they ask for so much shared memory that they do.  (A cluster lies within a group
  // of at least 16 SMs, and fills seven eighths of the places that are left there.)
  const int S = a.split_ctas, group = S > 1 ? 14 / S * S : 16;
  const long long total = (long long)n_ctas * g.Hq * 16, places = (long long)num_sms * group;
  cfg.dynamicSmemBytes = std::max(Smem<D>::bytes, total <= places ? SMEM_ALONE : total <= 2 * places ? SMEM_TWO : (size_t)0);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n_attr = 0;
  if (!a.no_pdl) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (a.split_ctas > 1) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = (unsigned)a.split_ctas;
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  return a.mode == MODE_STEP ? cudaLaunchKernelEx(&cfg, simt_attn_kernel<D, true>, g, a) : cudaLaunchKernelEx(&cfg, simt_attn_kernel<D, false>, g, a);
}

}  // namespace

cudaError_t simt_prepare() {
  const void* const kernels[4] = {(const void*)simt_attn_kernel<128, false>, (const void*)simt_attn_kernel<128, true>,
                                  (const void*)simt_attn_kernel<64, false>, (const void*)simt_attn_kernel<64, true>};
  for (const void* k : kernels) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_ALONE);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t simt_attention(const Geometry& g, const AttnArgs& args, int num_sms, cudaStream_t s) {
  AttnArgs a = args;
  if (a.n_items == 0) return cudaSuccess;
  // Units with the long key range: the block queries of a step (its first items), every unit otherwise.
  const bool step = a.mode == MODE_STEP;
  if (!step) a.n_split_items = a.n_items;
  const int rest = a.n_items - a.n_split_items;
  const int max_tiles = (g.maxN + KT - 1) / KT;
  a.split_ctas = step ? plan::simt_step_parts(a.n_split_items, rest, g.Hq, max_tiles, g.d, num_sms)
                      : plan::simt_row_parts((long long)a.n_items * g.Hq, max_tiles, g.d, num_sms);
  const int S = a.split_ctas;
  const int n_ctas = a.n_split_items * S + (rest + S - 1) / S * S;
  return g.d == 128 ? launch<128>(g, a, n_ctas, num_sms, s) : launch<64>(g, a, n_ctas, num_sms, s);
}

}  // namespace lacache

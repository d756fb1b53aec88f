// What the two tensor-core attention kernels share: tensor maps, bounded waits of a CTA's roles, wide global accesses,
// the exponential, output rounding and work items.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lacache_internal.h"
#include "lacache_ptx.h"

namespace lacache {

struct TcMaps {
  // rotated Q' / K': 5-D views {64 features, Tp rows, 2 feature halves, heads, 2 planes (hi, lo)} of the
  // split-bf16 storage [plane][head][half][Tp][64]; one box = both planes and both halves of `rows` rows
  // of one head, laid out in shared memory as [plane][half][rows][64] (128-byte swizzle)
  alignas(64) CUtensorMap q;       // box 128 rows
  alignas(64) CUtensorMap q64;     // box 64 rows (block queries)
  // block queries of `pack` heads of one KV group side by side: dimensions ordered {64, rows, heads, halves,
  // planes}, box {64, pack_rows, pack, 2, 2}: lands as [plane][half][head][row][64], i.e. one 128-row tile
  alignas(64) CUtensorMap q_pack;
  alignas(64) CUtensorMap k;       // box TC_KEYS rows (stream role)
  alignas(64) CUtensorMap k64;     // box 64 rows (the block's keys, merge role)
  alignas(64) CUtensorMap k32;     // box 32 rows (the block's keys, pipelined merge role)
  // V: 4-D views {64, Tp, 2 halves, heads} of the fp16 storage [head][half][Tp][64]
  alignas(64) CUtensorMap v;
  alignas(64) CUtensorMap v64;
  alignas(64) CUtensorMap v32;
  // row kernel: boxes of 128 keys, whole or (k_box) one plane and one feature half
  alignas(64) CUtensorMap k_rows, v_rows, k_box;
  alignas(64) CUtensorMap st_o;    // cached O~ [Hq][Tp][128] fp32, box 32 cols x 128 rows
  alignas(64) CUtensorMap out;     // caller's out [T][Hq][128] fp32, box 32 cols x 1 head x 128 rows
  alignas(64) CUtensorMap out_sub[4];  // the same with boxes of 64, 32, 16 and 8 rows (clipped row tiles)
  const void* out_ptr;             // the buffer `out` was encoded for
};

namespace tcu {

using namespace ptx;

constexpr int D = 128;
constexpr int BM = TC_ROWS;   // 128 query rows (TMEM lanes)
constexpr float RESCALE_SLACK = 3.f;
constexpr long long WAIT_CYCLES = 4000000000ll;  // ~2 s

// one 32-byte store of 8 words (the address is 32-byte aligned)
__device__ __forceinline__ void st_global_v8(void* dst, const uint32_t* r) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// one 32-byte load of 8 words (the address is 32-byte aligned)
__device__ __forceinline__ void ld_global_v8(const void* src, uint32_t* r) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(src)
               : "memory");
}
__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// p rounded to 11 significant bits (what fp16 keeps) with plain fp32 arithmetic
// (Veltkamp split), so the fp16 conversion that follows is exact and the
// normaliser can sum the very values the MMA multiplies without converting back.
__device__ __forceinline__ float round_to_half_bits(float p) {
  float c = __fmul_rn(p, 8193.0f);
  return __fsub_rn(c, __fsub_rn(c, p));
}
// four consecutive output elements at element offset `off` of `out` (fp32, or bf16 when the context's
// out_dtype says so)
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ void store_out4(const AttnArgs& a, size_t off, float4 v) {
  if (a.out_bf16) {
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.out) + off) =
        make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
  } else {
    *reinterpret_cast<float4*>(a.out + off) = v;
  }
}
__device__ __forceinline__ WorkItem load_item(const WorkItem* p) {
  const int4* q = reinterpret_cast<const int4*>(p);
  int4 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
  WorkItem w;
  w.kind = a.x; w.seq = a.y; w.row0 = a.z; w.nrows = a.w;
  w.chunk = b.x; w.kt0 = b.y; w.kt1 = b.z; w.pad = b.w;
  w.seq_start = c.x; w.seq_end = c.y; w.blk_start = c.z; w.n_before = c.w;
  return w;
}

struct Cta {
  uint32_t base;            // shared-space address of the region
  uint8_t* gen;             // generic pointer to the same region
  uint32_t tmem;            // TMEM base address
  volatile int* abort_flag;
  volatile uint32_t* flag;  // scratch word for CTA-wide decisions
  int32_t* status;
  uint32_t bar0;            // shared-space address of the first barrier
  __device__ __forceinline__ uint32_t bar(int slot) const { return bar0 + 8u * slot; }
};

// Bounded wait on phase `parity`; false if it ran out or the CTA is unwinding.
static __device__ __noinline__ bool wait_slow(const Cta& c, uint32_t bar, uint32_t parity, int loc) {
  long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*c.abort_flag) return false;
    if (clock64() - t0 > WAIT_CYCLES) {
      *c.abort_flag = 1;
      if (atomicCAS(c.status, 0, (int)LACACHE_ERR_TIMEOUT) == 0) {
        c.status[1] = loc;
        c.status[2] = blockIdx.x;
        c.status[3] = threadIdx.x;
      }
      return false;
    }
  }
}
__device__ __forceinline__ bool wait_bar(const Cta& c, int slot, uint32_t parity, int loc) {
  uint32_t b = c.bar(slot);
  if (mbar_try(b, parity)) return true;
  return wait_slow(c, b, parity, loc);
}

}  // namespace tcu
}  // namespace lacache

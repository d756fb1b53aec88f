// RoPE-on-write (Eq. 1, Sec. 3.3.2) and the export kernels.
//
// rope_write rotates q and k at each token's position, copies v, and stores
// the result head-major in the engine's storage format:
//   SIMT engine    : fp32 planes.
//   tcgen05 engine : rotated q,k as two bf16 planes hi = bf16(x),
//                    lo = bf16(x - hi) (so hi + lo carries 16 significand
//                    bits into the tensor-core score product); v as fp16.
// The same kernel serves the build (all T tokens) and the step (only the
// block's L_b tokens per sequence, scattered to their cache slots).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lacache_internal.h"
#include "lacache_rope_math.h"

namespace lacache {
namespace {

__device__ __forceinline__ void store8_f32(void* plane, size_t off, const float (&y)[8]) {
  float4* p = reinterpret_cast<float4*>(reinterpret_cast<float*>(plane) + off);
  p[0] = make_float4(y[0], y[1], y[2], y[3]);
  p[1] = make_float4(y[4], y[5], y[6], y[7]);
}

__device__ __forceinline__ void store8_f16(void* plane, size_t off, const float (&y)[8]) {
  *reinterpret_cast<uint4*>(reinterpret_cast<__half*>(plane) + off) = rope_half8(y);
}

// One thread: 8 features c0 .. c0 + 7 of the first half and their partners at c0 + d/2, of one source row and HPT
// consecutive heads of one tensor; cos and sin are loaded once for all of them (with one head per thread they are two
// thirds of what a thread loads).  d/16 threads cover a row, a warp 32 / (d/16) consecutive rows, so that both the HPT
// heads it reads per row and the rows it writes per head are contiguous.  blockIdx.y: group of HPT heads -- q, then k,
// then v.  tcgen05 storage: HPT = 4 from 65536 (row, head) pairs on (157 MB of bf16 rows in, as much out: 71 us with one head
// per thread, 55 us = 5.7 TB/s with four; two and eight the same within 4 %), else 1: a block's rows are too few to fill the
// GPU with more per thread.  fp32 storage: always 1, whose rows are wide enough by themselves, while four heads' rows do
// not fit the registers (fp32 rows of 128 features, 65544 pairs: 15.1 us against 20.7 with four; 589824: 96 against 108).
template <bool TC, int HPT>
__global__ void __launch_bounds__(256, HPT > 1 ? 3 : 1) rope_write_kernel(const __grid_constant__ Geometry g, const __grid_constant__ RopeArgs a) {
  // This kernel and the attention kernel behind it are launched programmatically dependent.  The attention
  // kernel reads this kernel's inputs, and state that the kernels ahead may have written, before it waits for
  // this grid: it may start only once those are complete, hence the order of the wait and the trigger.
  if (!a.early_inputs) asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int shift = g.d == 128 ? 3 : 2;   // d / 16 chunks per row
  const int chunk = threadIdx.x & ((1 << shift) - 1);
  const int r = (int)blockIdx.x * (256 >> shift) + (int)(threadIdx.x >> shift);
  if (r >= a.n_src_rows) return;
  const int half = g.d / 2, c0 = chunk * 8;
  int grp = blockIdx.y;
  const int gq = (g.Hq + HPT - 1) / HPT, gk = (g.Hkv + HPT - 1) / HPT;
  const void* src;
  int H, which;  // 0 q, 1 k, 2 v
  if (grp < gq) { src = a.q; H = g.Hq; which = 0; }
  else if (grp < gq + gk) { src = a.k; H = g.Hkv; which = 1; grp -= gq; }
  else { src = a.v; H = g.Hkv; which = 2; grp -= gq + gk; }
  const int h0 = grp * HPT;
  const int tok = a.row_tok ? a.row_tok[r] : (a.blk_start ? a.blk_start[r / a.block_len] + r % a.block_len : r);
  const bool bf16_in = a.in_dtype == LACACHE_DTYPE_BF16;

  // (the rows as they come: converted they would take twice the registers)
  constexpr int NR = TC ? 1 : 2;   // 16-byte words of 8 features (the tcgen05 engine's inputs are bf16)
  uint4 raw[HPT][2][NR];
#pragma unroll
  for (int i = 0; i < HPT; ++i) {
    const size_t soff = ((size_t)r * H + min(h0 + i, H - 1)) * g.d + c0;
#pragma unroll
    for (int e = 0; e < 2; ++e) rope_fetch8<NR>(src, soff + e * half, TC || bf16_in, raw[i][e]);
  }
  float cs[8], sn[8];
  if (which < 2) {
    const float4 *cp, *sp;
    if (a.row_cos) {
      cp = reinterpret_cast<const float4*>(a.row_cos + (size_t)r * half + c0);
      sp = reinterpret_cast<const float4*>(a.row_sin + (size_t)r * half + c0);
    } else {
      const int pos = a.pos_of_tok[tok];
      cp = reinterpret_cast<const float4*>(a.cos_tab + (size_t)pos * half + c0);
      sp = reinterpret_cast<const float4*>(a.sin_tab + (size_t)pos * half + c0);
    }
    const float4 ca = cp[0], cb = cp[1], sa = sp[0], sb = sp[1];
    cs[0] = ca.x; cs[1] = ca.y; cs[2] = ca.z; cs[3] = ca.w; cs[4] = cb.x; cs[5] = cb.y; cs[6] = cb.z; cs[7] = cb.w;
    sn[0] = sa.x; sn[1] = sa.y; sn[2] = sa.z; sn[3] = sa.w; sn[4] = sb.x; sn[5] = sb.y; sn[6] = sb.z; sn[7] = sb.w;
  }
  // Everything above read only this call's inputs and constant tables.  The stores below overwrite
  // cache rows that the previous step's attention kernel may still be reading when this kernel was
  // launched programmatically dependent on it: wait for that grid first (returns at once otherwise).
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int i = 0; i < HPT; ++i) {
    const int h = h0 + i;
    if (h >= H) break;
    float x1[8], x2[8], y1[8], y2[8];
    rope_unpack8<NR>(raw[i][0], TC || bf16_in, x1);
    rope_unpack8<NR>(raw[i][1], TC || bf16_in, x2);
    if (which < 2) {
      rope_rotate8(x1, x2, cs, sn, y1, y2);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) { y1[e] = x1[e]; y2[e] = x2[e]; }
    }
    if (TC) {
      // tcgen05 storage: [head][feature half][Tp][64] (d = 128), each half of a row one 128-byte line
      const size_t o1 = ((size_t)(2 * h) * g.Tp + tok) * 64 + c0;
      const size_t o2 = ((size_t)(2 * h + 1) * g.Tp + tok) * 64 + c0;
      if (which == 2) {
        store8_f16(a.dst.v, o1, y1);
        store8_f16(a.dst.v, o2, y2);
      } else {
        void* const hi = which == 0 ? a.dst.q_hi : a.dst.k_hi;
        void* const lo = which == 0 ? a.dst.q_lo : a.dst.k_lo;
        rope_store8(hi, lo, o1, y1, g.op_f16 != 0);
        rope_store8(hi, lo, o2, y2, g.op_f16 != 0);
      }
    } else {
      void* const plane = which == 0 ? a.dst.q_hi : (which == 1 ? a.dst.k_hi : a.dst.v);
      const size_t doff = ((size_t)h * g.Tp + tok) * g.d + (c0 ^ (which == 2 ? simt_swz_v(tok) : simt_swz_qk(tok)));
      store8_f32(plane, doff, y1);
      store8_f32(plane, doff + half, y2);
    }
  }
}

// Export kernels: head-major storage -> token-major fp32.
template <bool TC>
__device__ __forceinline__ float read_rot(const void* hi, const void* lo, size_t off, bool f16) {
  if (TC && f16) return __half2float(reinterpret_cast<const __half*>(hi)[off]);
  if (TC) {
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(hi)[off]) +
           (lo ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(lo)[off]) : 0.f);
  }
  return reinterpret_cast<const float*>(hi)[off];
}

template <bool TC>
__global__ void __launch_bounds__(256) export_kernel(Geometry g, ExportArgs a) {
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long nq = (long long)g.T * g.Hq * g.d;
  if (idx >= nq) return;
  int c = (int)(idx % g.d);
  long long t = idx / g.d;
  int h = (int)(t % g.Hq);
  int tok = (int)(t / g.Hq);
  const size_t srow = ((size_t)h * g.Tp + tok) * g.d + c;   // state: [head][Tp][d]
  // rotated planes: the tcgen05 engine stores [head][feature half][Tp][64], the other [head][Tp][d] with swizzled rows
  const size_t row = ((size_t)h * g.Tp + tok) * g.d;
  const size_t src = TC ? ((size_t)(2 * h + c / 64) * g.Tp + tok) * 64 + c % 64 : row + (c ^ simt_swz_qk(tok));
  const size_t src_v = TC ? src : row + (c ^ simt_swz_v(tok));
  const float LN2 = 0.69314718055994530942f;
  if (a.o) a.o[idx] = a.st.o[srow];
  if (c == 0) {
    if (a.m) a.m[(size_t)tok * g.Hq + h] = a.st.m[(size_t)h * g.Tp + tok] * LN2;
    if (a.l) a.l[(size_t)tok * g.Hq + h] = a.st.l[(size_t)h * g.Tp + tok];
  }
  if (a.q_rot) a.q_rot[idx] = read_rot<TC>(a.rot.q_hi, a.rot.q_lo, src, g.op_f16 != 0);
  if (h < g.Hkv) {
    size_t dst = ((size_t)tok * g.Hkv + h) * g.d + c;
    if (a.k_rot) a.k_rot[dst] = read_rot<TC>(a.rot.k_hi, a.rot.k_lo, src, g.op_f16 != 0);
    if (a.v) {
      a.v[dst] = TC ? __half2float(reinterpret_cast<const __half*>(a.rot.v)[src_v])
                    : reinterpret_cast<const float*>(a.rot.v)[src_v];
    }
  }
}

// Partial states of the key chunks of block rows -> the rows' state (Eq. 2-6 merge): thread = 16 bytes of
// one row of one head; every load of the (at most eight at a time) chunks is issued before any is used.
__global__ void __launch_bounds__(256) merge_chunk_states_kernel(Geometry g, ChunkMergeArgs a) {
  // launched programmatically dependent on the kernel that writes the partial states: the launch itself and
  // the start of the kernel after this one overlap their neighbours; nothing is read before that kernel is complete
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= g.block_len * 32) return;
  const int rr = i >> 5, ch = i & 31, h = blockIdx.y, b = blockIdx.z;
  const int row0 = a.tab[2 * b], n = a.tab[2 * b + 1];
  const size_t pbase = ((size_t)b * g.Hq + h) * a.max_chunks;
  float M = -INFINITY, L = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c0 = 0; c0 < n; c0 += 8) {
    float mv[8], lv[8];
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (c0 + k < n) {
        const size_t pr = (pbase + c0 + k) * g.block_len + rr;
        mv[k] = __ldcg(a.part_m + pr);
        lv[k] = __ldcg(a.part_l + pr);
        v[k] = __ldcg(reinterpret_cast<const float4*>(a.part_o + pr * g.d) + ch);
      } else {
        mv[k] = -INFINITY; lv[k] = 0.f; v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    float Mn = M;
#pragma unroll
    for (int k = 0; k < 8; ++k) Mn = fmaxf(Mn, mv[k]);
    const float w0 = (M == -INFINITY) ? 0.f : exp2f(M - Mn);
    L *= w0; acc.x *= w0; acc.y *= w0; acc.z *= w0; acc.w *= w0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float w = (mv[k] == -INFINITY) ? 0.f : exp2f(mv[k] - Mn);
      L = fmaf(lv[k], w, L);
      acc.x = fmaf(v[k].x, w, acc.x);
      acc.y = fmaf(v[k].y, w, acc.y);
      acc.z = fmaf(v[k].z, w, acc.z);
      acc.w = fmaf(v[k].w, w, acc.w);
    }
    M = Mn;
  }
  const size_t srow = (size_t)h * g.Tp + row0 + rr;
  *reinterpret_cast<float4*>(a.st.o + srow * g.d + ch * 4) = acc;
  if (ch == 0) { a.st.m[srow] = M; a.st.l[srow] = L; }
}

}  // namespace

cudaError_t merge_chunk_states(const Geometry& g, const ChunkMergeArgs& a, cudaStream_t s) {
  // (head_dim 128: 32 sixteen-byte columns per row, the only shape the tcgen05 engine serves)
  dim3 grid((unsigned)((g.block_len * 32 + 255) / 256), (unsigned)g.Hq, (unsigned)g.B);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.no_pdl ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, merge_chunk_states_kernel, g, a);
}

template <bool TC>
static cudaError_t rope_launch(const Geometry& g, const RopeArgs& a, cudaStream_t s) {
  constexpr int MANY = TC ? 4 : 1;
  const bool many = (long long)a.n_src_rows * (g.Hq + 2 * g.Hkv) >= 65536;
  const int hpt = many ? MANY : 1;
  const int rows_per_cta = 256 / (g.d / 16);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((a.n_src_rows + rows_per_cta - 1) / rows_per_cta),
                     (unsigned)((g.Hq + hpt - 1) / hpt + 2 * ((g.Hkv + hpt - 1) / hpt)));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.no_pdl ? 0 : 1;
  return many ? cudaLaunchKernelEx(&cfg, rope_write_kernel<TC, MANY>, g, a) : cudaLaunchKernelEx(&cfg, rope_write_kernel<TC, 1>, g, a);
}

cudaError_t rope_write(const Geometry& g, const RopeArgs& a, int engine, cudaStream_t s) {
  if (a.n_src_rows == 0) return cudaSuccess;
  return engine == LACACHE_ENGINE_TCGEN05 ? rope_launch<true>(g, a, s) : rope_launch<false>(g, a, s);
}

cudaError_t export_buffers(const Geometry& g, const ExportArgs& a, int engine, cudaStream_t s) {
  long long total = (long long)g.T * g.Hq * g.d;
  unsigned blocks = (unsigned)((total + 255) / 256);
  if (engine == LACACHE_ENGINE_TCGEN05)
    export_kernel<true><<<blocks, 256, 0, s>>>(g, a);
  else
    export_kernel<false><<<blocks, 256, 0, s>>>(g, a);
  return cudaGetLastError();
}

}  // namespace lacache

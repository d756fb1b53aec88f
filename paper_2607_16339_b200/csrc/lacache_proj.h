// Projection of many tokens (lacache_proj.cu), called by the token-wise producer (lacache_qkv.cu).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "lacache_internal.h"

namespace lacache {

struct ProjArgs {
  int n_tokens, kc;                         // kc = d_model / 64
  int Hq, Hkv;
  __nv_bfloat16 *q, *k, *v;
  const int32_t* dst_rows; int max_rows;    // output row of input token t (null: t); rows outside [0, max_rows) are dropped
  int rotate; RotateTarget rot;             // also leave the rows rotated (dst_rows null)
  int32_t* status;
  long long wait_cycles;
  int n_heads, n_ttiles, n_tiles;           // set by proj_many
};
cudaError_t proj_prepare();
// w_map: the packed weight, boxes of 128 rows x 64; x_map: the operand rows, boxes of 128 tokens x 64
cudaError_t proj_many(const CUtensorMap& w_map, const CUtensorMap& x_map, ProjArgs a, int num_sms, bool pdl, cudaStream_t s);

}  // namespace lacache

// Calls between the files that implement the public header.
#pragma once
#include "../../include/sepconv.h"

namespace sc {
// sepconv_fwd (without running statistics) always enqueued launch by launch: for callers on whose behalf nothing may be
// allocated, not even by the CUDA runtime for a graph.
int fwd_direct(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res, const int32_t* lengths_dev,
               const sc_block_params* params, sc_tensor* y, int32_t* out_lengths_dev, sc_block_saved* saved, void* workspace,
               size_t workspace_bytes, void* cuda_stream);
}  // namespace sc

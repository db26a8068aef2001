// Calls between the files that implement the public header.
#pragma once
#include "../../include/sepconv.h"

namespace sc {
// sepconv_fwd (without running statistics) always enqueued launch by launch: for callers on whose behalf nothing may be
// allocated, not even by the CUDA runtime for a graph, and who cannot bring a workspace of the size they are asked for: where
// the packed operands (or the non-separable convolution's copies) do not fit, the block runs on the dense tensors.
int fwd_direct(sc_ctx* ctx, const sc_block_desc* desc, const sc_tensor* x, const sc_tensor* x_res, const int32_t* lengths_dev,
               const sc_block_params* params, sc_tensor* y, int32_t* out_lengths_dev, sc_block_saved* saved, void* workspace,
               size_t workspace_bytes, void* cuda_stream);
// Scratch of the forward pass on the dense tensors: the least that fwd_direct runs in.
int fwd_dense_bytes(const sc_block_desc* desc, size_t* bytes);
}  // namespace sc

// Tensor map (TMA descriptor) of a paged cache of decayed keys and values.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rq {

// The bf16 cache [pages of all heads][key / value][slot][channel] as a rank-4 tensor (channel, slot, key / value,
// page) with a box of 64 channels x the slots of a page x one of key / value x the pages of `positions`
// consecutive positions (a multiple of the page size), 128-byte swizzle: one tiled bulk-tensor copy brings a
// 64-channel half of `positions` rows into shared memory as rows of 128 bytes in the layout the tensor core
// reads.  The driver's encoder is looked up once through the runtime (the library does not link the driver).
cudaError_t cache_tensor_map(CUtensorMap *out, const void *kv, int D, int S, int64_t pages_total, int positions);

// A prompt's keys, values or gates, element (b, t, h, d) at b * sb + t * st + h * sh + d (strides in elements of `es` bytes),
// as a rank-4 tensor (channel, head, position, batch item); box = `channels` channels x one head x `positions` positions,
// dense rows.  With sh = 0 the tensor has one head, with sb = 0 one batch item.  Fails where the strides cannot be described.
cudaError_t prompt_tensor_map(CUtensorMap *out, const void *x, int es, int D, int H, int64_t T, int B, int64_t sh, int64_t st, int64_t sb,
                              int channels, int positions);

// [B][T][H][D] bf16 queries (or outputs) as a rank-4 tensor (channel, head, position, batch item); box = 64 channels x one head x
// `positions` positions, 128-byte swizzle (the layout the tensor core reads); positions beyond T read as
// zero and are not stored.
cudaError_t query_tensor_map(CUtensorMap *out, const void *q, int D, int H, int64_t T, int B, int positions);

// The paged cache with elements of `es` bytes as a rank-4 tensor (channel, slot, key / value, page); box = `channels` channels
// x `slots` slots of one page's keys or values, dense rows.
cudaError_t page_tensor_map(CUtensorMap *out, void *kv, int es, int D, int S, int64_t pages_total, int channels, int slots);

}  // namespace rq

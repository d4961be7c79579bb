// Nested lists of several sequences in shared passes (clada_nested_batch.cu) as the decode entry points see them.
#pragma once

#include "common.cuh"
#include "ffn_single.cuh"

namespace clada {

constexpr int kNestedBatchMax = 8;  // sequences of one pass
constexpr int kNestedBatchMin = 3;  // fewer have a launch each

// Whether nb sequences of this layer take a pass (the measurements behind it are at nb_plan).
bool nested_batch_supported(const clada_layer *layer, int nb);
// Scratch of a pass behind the control block: hidden values, keep words, partial rows.
size_t nested_batch_scratch_bytes(const clada_layer *layer, int nb, int num_sms);
int launch_nested_batch(const clada_layer *layer, int nb, const void *x, const int32_t *order, const int32_t *counts,
                        const int32_t *level, void *y, int y_dtype, int32_t *count_out, void *ws, int32_t *status,
                        cudaStream_t st);

}  // namespace clada

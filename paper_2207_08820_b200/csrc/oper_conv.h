// Sequences of layers on operand tensors (oper_conv.cu): host interface for the sequences of mma_conv.cu.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace bs {

struct OperSequence;
struct OperTensor;

// Bytes of zeroed device memory that the layers need to run on operand tensors; 0: they don't take them (mma_conv.cu runs them).
size_t oper_workspace_bytes(const bs_sequence_layer* layers, int n);
// How layer i runs then; BS_ERR_UNSUPPORTED where they don't.
int oper_layer_plan(const bs_sequence_layer* layers, int n, int i, bs_layer_plan* out);
// The launches of such layers; null where oper_workspace_bytes is 0 or bytes is less.
OperSequence* oper_create(const bs_sequence_layer* layers, int n, void* workspace, size_t bytes);
// Launches in front of the layers: filters to prepare, forms of tensors that the layers read from their packed codes; those of one tensor, or null.
int oper_imports(const OperSequence* q);
const OperTensor* oper_input(const OperSequence* q, const uint32_t* packed);
// These launches but the one of `ready`, whose forms are up to date (or null), and layer i, on `st`.
int oper_begin(const OperSequence* q, const OperTensor* ready, cudaStream_t st);
int oper_layer(const OperSequence* q, int i, cudaStream_t st);
void oper_destroy(OperSequence* q);

}  // namespace bs

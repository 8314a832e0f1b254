// The batched tensor-core kernel: the path "gemm_tcgen05", the batches of other families that dispatch.cu sends to it, fused calls.
#pragma once
#include "common.cuh"

namespace vptq {

bool gemm_tcgen05_supported(const LayerView &L, int B);
// n layers that read the same activations in one launch (n = 1: one layer)
bool gemm_tcgen05_fused_supported(const LayerView *Ls, int n, int B);
long long gemm_tcgen05_workspace_bytes(const LayerView *Ls, int n, int B);
int gemm_tcgen05_launches(const LayerView &L, int B);
// true when split tiles of a layer of the launch meet by flag order (a CTA waits for a flag another CTA of the grid raises)
bool gemm_tcgen05_waits_between_ctas(const LayerView *Ls, int n, int B);
// Workspace layout: int32 status word at byte 0 (0 = ok, VPTQ_E_TIMEOUT = a bounded wait gave up), then per layer tile flags,
// bias terms, padded tables, sums of split tiles and the scaled FP16 activations.
cudaError_t launch_gemm_tcgen05(const LayerView *Ls, int n, const void *x, int B, void *const *outs, void *ws, cudaStream_t st);

}  // namespace vptq

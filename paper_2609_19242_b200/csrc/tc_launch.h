// Host-side interface of the tcgen05 (5th-generation tensor core) kernels.
#pragma once
#include <cuda.h>

#include "bdlm_common.cuh"

namespace bdlm {

// Address of the device status word that bounded waits report to (nullptr on failure).
int* device_status_ptr();

bool tc_encoder_available();
// Tensor map over a [batch, L, heads, d] bf16 tensor (d = 64 or 128), box = 64 columns x `rows` rows, 128-byte swizzle.
bool tc_make_map(CUtensorMap* m, const void* ptr, int heads, int L, int batch, int rows, int d);

// Tensor map over a row-major bf16 matrix [rows, cols] with leading dimension ld (elements): box = 64 columns x
// `box_rows` rows, 128-byte swizzle, zero fill outside the matrix.
bool tc_make_map_2d(CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows);

// The same matrix as a stack of 64-column panels (cols a multiple of 64): one load brings `box_panels` neighbouring panels
// of `box_rows` rows, one after the other.
bool tc_make_map_panels(CUtensorMap* m, const void* ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows, int box_panels);

bool tc_rows_ok(const KArgs& a);
bool tc_fwd_supported(const KArgs& a);
bool tc_bwd_supported(const KArgs& a);
// Bytes of the fused backward's fp32 dQ accumulators for these sizes (0 when the fused kernel cannot take them).
size_t tc_bwd_fused_workspace(const bdlm_params* p, const bdlm_packed_geometry* g);
cudaError_t launch_tc_fwd(const KArgs& a, cudaStream_t st);
// Lays the fused backward's dQ accumulators out in the workspace (a.dq32, a.dq32_rows).
void tc_bwd_place_dq(KArgs& a, void* extra_ws);
cudaError_t launch_tc_bwd(const KArgs& a, int passes, cudaStream_t st);
// The backward on pairs of CTAs (head dimension 128): dK, dV and, with dq, the sums for dQ.
cudaError_t launch_tc_bwd_pair(const KArgs& a, bool dq, cudaStream_t st, bool chained);

}  // namespace bdlm

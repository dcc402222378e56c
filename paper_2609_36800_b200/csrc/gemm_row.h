// Device-side arguments and launcher of the row-stream decode kernel (gemm_row.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "row_plan.h"

namespace bd {

struct RowArgs {
    int B, m, N, K;
    int f16, act;
    int TB, rows, groups, units, stages, k_stages;
    uint32_t s_off, x_off, stage_bytes;
    const void* bias;
    const float* alpha;
    void* Y;
};

// tmW / tmX: 16-bit [rows, K] in boxes of 16 64-column atoms x (p.rows / 8) rows; tmBits: [B, N, K/32] words in boxes of 32 words x
// p.rows rows x p.TB tenants, all with 128-byte swizzle.
cudaError_t launch_gemm_row(const CUtensorMap& tmW, const CUtensorMap& tmX, const CUtensorMap& tmBits, const RowArgs& args,
                            const RowPlan& p, bool early_start, cudaStream_t stream);
cudaError_t read_row_status(unsigned int out[2]);

}  // namespace bd

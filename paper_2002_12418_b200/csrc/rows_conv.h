// The one-kernel convolution by rows (rows_conv.cu): interface to the plan object.
#pragma once
#include <cuda_runtime.h>

#include "kernels.h"
#include "rows_plan.h"

namespace mnnb {

struct RowsConv {
    RowsPlan p;
    float At[2 * kRowsMaxAlpha], G[kRowsMaxAlpha * 7], Bt[kRowsMaxAlpha * kRowsMaxAlpha];   // one-dimensional matrices (m > 1)
    int num_sms = 0;
    bool ready = false;
};

// Whether B^T has the zeros the kernel's input transform relies on.
bool rows_matrices_ok(const RowsConv& rc);
cudaError_t rows_setup(RowsConv* rc);
// Weights [Cout][Cin][kh][kw] into U (p.u_bytes), transformed, split into hi + lo and laid out as the kernel's shared memory.
cudaError_t launch_rows_weights(const RowsConv& rc, const float* w, void* U, cudaStream_t stream);
cudaError_t launch_rows_conv(const RowsConv& rc, const float* x, const void* U, const float* bias, float* y, int relu, int* status,
                             cudaStream_t stream);

}  // namespace mnnb

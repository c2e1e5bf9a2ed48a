// The packed-line convolution (line_conv.cu): interface to the plan object.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "line_plan.h"

namespace mnnb {

struct LineConv {
    LinePlan p;
    CUtensorMap map_a, map_u;
    int num_sms = 0;
    bool ready = false;
};

// Tensor maps over the packed planes A (a_bytes, 16-byte aligned) and the weights U (u_bytes, 16-byte aligned).
cudaError_t line_setup(LineConv* lc, void* A, void* U, const char** why);
// U [tap][Cout][elems], rounded to the operand type.
cudaError_t launch_line_weights(const LinePlan& p, const float* w, void* U, cudaStream_t stream);
// x into A, rounded to the operand type.
cudaError_t launch_line_pack(const LinePlan& p, const float* x, void* A, cudaStream_t stream);
// y = act(conv + bias) from A and U.
cudaError_t launch_line_gemm(const LineConv& lc, const float* bias, float* y, int relu, int* status, cudaStream_t stream);

}  // namespace mnnb

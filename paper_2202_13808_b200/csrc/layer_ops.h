// What the native autograd node (native.cpp) needs beside the C ABI: the element-wise and column-sum work of a layer's
// backward pass, as kernels of the library (layer_ops.cu).  Internal; no part of include/dropit.h.
#pragma once

#include <stdint.h>

#include "dropit.h"

namespace dropit {

// dx = dy * GELU'(x), n bf16 elements; pointers 16-byte aligned.
dropit_status gelu_backward_bf16(const void* dy, const void* x, void* dx, int64_t n, void* cuda_stream);

// The end of a Linear's backward pass in one launch: dw_out (bf16) = dw (fp32), `count` elements, and, unless db is null, db (bf16) =
// column sums of dy [M x Cz], fp32 sums in a fixed order.  Pointers 16-byte aligned, Cz a multiple of 8.
dropit_status finish_linear_backward(const float* dw, void* dw_out, int64_t count, const void* dy, int64_t M, int64_t Cz, void* db,
                                     void* cuda_stream);

}  // namespace dropit

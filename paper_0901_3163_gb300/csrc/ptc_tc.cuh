// Tensor-core form of a parallel-transport convolution layer (ptc.cu has the layer).
#pragma once

#include <cuda_bf16.h>

#include "dlz_internal.cuh"

namespace dlz {

// bf16 elements of a layer's weight image (ptc_tc.cu)
size_t ptc_tc_image_size(int cin, int cout);
// whether the layer runs on the tensor cores on a lattice of `sites` sites
bool ptc_tc_layer(int cin, int cout, int sites);
int ptc_tc_prepare();       // kernel attributes, outside graph captures
// weights [9][cout][cin][16] -> image
int ptc_tc_image(Op &op, __nv_bfloat16 *img, const __nv_bfloat162 *w, int cin, int cout);
// Status of a pass: bits of a device word (a wait gave up; a result is not finite: an infinite
// operand has no finite remainder for its second part, so it gives NaN where FP32 arithmetic may
// give an infinity, and the caller computes such a pass again without tensor cores), and a word
// of mapped host memory that is set when a bit is: the host reads it without a copy.
constexpr int kPtcTimeout = 1, kPtcNonfinite = 2;
struct PtcStatus {
    int *bits, *host;
};
// the layer on nvec fields
int ptc_tc_forward(Op &op, float4 *out, const float4 *in, const __nv_bfloat16 *img, int cin, int cout, int nvec,
                   PtcStatus status);
// block partials [9][blocks][4 cout][4 cin] of the layer's weight gradient from G(out) and the
// layer's input; blocks <= kPtcMaxGradBlocks
constexpr int kPtcMaxGradBlocks = 64;
int ptc_tc_wgrad(Op &op, float2 *partials, const float4 *gout, const float4 *in, int cin, int cout, int nvec, PtcStatus status,
                 int &blocks);

}  // namespace dlz

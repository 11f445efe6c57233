// The filter and the attention as calls of their own for head_dim 128 (see
// wf_fused.cu).  An instance apart from the step's, because its attention
// keeps two bf16 terms of P and the step's kernel loses registers and
// instruction cache to them (64 units x 32K: 68.5 -> 70 us); one instance for
// both calls, because a filter and its attention that alternate two kernels
// fetch their instructions anew each time (20K tokens 57 -> 62 us).
//
// Why two terms: the fused attention takes P about the first tile's maximum,
// where the split kernel takes the running one, so that the largest weight is a
// whole power of two.  Rounded to bf16 about any other stabiliser P had up to 12 %
// more error against 64 bits (1024 keys, queries 2 N(0, 1): 2.00e-3 against
// 1.79e-3); with a second term it is 1.66e-3, the rounding of the output.  (The
// split kernel has the second term too on the calls that either route serves.)
#define WF_STAGE_CALLS 1
#include "wf_fused.cu"

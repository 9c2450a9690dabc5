// Tensor-core scoring for 64-channel heads (score_tc_impl.cuh).  16 layers of
// 8K + 1K tokens: 12,410 us a call on the CUDA cores (score_simt.cu), 493 us
// here for both caches of a commit (calls that want no row statistics: api.cu);
// K and V need 86 us.  With the output accumulated in tensor memory it
// takes 459 us, but the rows' o is then off by 9e-6 instead of 7e-7.
#define CKV_TC_D 64
#define CKV_TC_NS d64
#include "score_tc_impl.cuh"

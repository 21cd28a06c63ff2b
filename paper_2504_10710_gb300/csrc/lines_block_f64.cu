// The FP64 instances of the line-block kernels, in a translation unit of their
// own so that both precisions compile side by side.
#define GLLS_LINES_F64
#include "lines_block.cu"

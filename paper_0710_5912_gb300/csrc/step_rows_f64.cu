// The FP64 row kernels of step_rows.cu: a translation unit of their own, so
// that the two precisions compile side by side.
#define SHF_ROWS_F64
#include "step_rows.cu"

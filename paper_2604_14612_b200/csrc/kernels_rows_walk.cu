// The T-row pass for few cached keys: kernels_rows.cu with the attention that walks them row by row and the larger ring that this leaves.
#define CL_ROWS_WALK
#include "kernels_rows.cu"

// okr_incr64.cu -- the incremental search with FP64 terms: the kernels of
// okr_incr.cu for precision 0, compiled beside those for precision 1.
#define OKR_INCR_FP64 1
#include "okr_incr.cu"

// D2Q9 instantiation of the companion kernels (see elbm_kernels.cuh): every launcher but
// the step's (elbm_d2q9.cu) and the ensemble's (elbm_d2q9_batch.cu).
#define ELBM_DIM 2
#define ELBM_SUFFIX d2q9
#define ELBM_PART 2
#include "elbm_kernels.cuh"

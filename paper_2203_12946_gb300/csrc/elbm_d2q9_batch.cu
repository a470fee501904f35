// D2Q9 instantiation of the batched ensemble's kernels (see elbm_kernels.cuh).
#define ELBM_DIM 2
#define ELBM_SUFFIX d2q9
#define ELBM_PART 3
#include "elbm_kernels.cuh"

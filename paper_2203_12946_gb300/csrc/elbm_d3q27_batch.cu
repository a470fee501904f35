// D3Q27 instantiation of the batched ensemble's kernels (see elbm_kernels.cuh).
#define ELBM_DIM 3
#define ELBM_SUFFIX d3q27
#define ELBM_PART 3
#include "elbm_kernels.cuh"

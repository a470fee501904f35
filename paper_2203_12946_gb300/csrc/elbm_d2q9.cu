// D2Q9 instantiation of the step kernels (see elbm_kernels.cuh): the step launcher;
// elbm_d2q9_batch.cu and elbm_d2q9_aux.cu hold the other launchers, so the three compile in
// parallel.
#define ELBM_DIM 2
#define ELBM_SUFFIX d2q9
#define ELBM_PART 1
#include "elbm_kernels.cuh"

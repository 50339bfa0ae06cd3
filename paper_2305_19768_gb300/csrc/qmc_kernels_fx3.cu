// The d <= 3 integer evaluator (qmc_real.cuh): qmc_kernels.cu compiled for part 4.
#define QMC_PART 4
#include "qmc_kernels.cu"

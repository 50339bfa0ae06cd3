// The d <= 6 integer evaluator (qmc_real.cuh): qmc_kernels.cu compiled for part 5.
#define QMC_PART 5
#include "qmc_kernels.cu"

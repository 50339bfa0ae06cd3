// The deformed evaluator (qmc_deformed.cuh): qmc_kernels.cu compiled for part 6.
#define QMC_PART 6
#include "qmc_kernels.cu"

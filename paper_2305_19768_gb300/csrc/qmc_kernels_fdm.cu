// The mixed-precision deformed evaluator (qmc_deformed.cuh): qmc_kernels.cu compiled for part 7.
#define QMC_PART 7
#include "qmc_kernels.cu"

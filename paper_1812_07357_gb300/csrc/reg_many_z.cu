// Register z kernels for passes over several z lengths (reg_kernels.cu).
#define PSATD_Z_MANY
#include "reg_kernels.cu"

// Register plane kernels of part 2 for passes over several plane shapes (reg_planes.cuh).
#define PSATD_PLANE_PART 2
#define PSATD_PLANE_NS plane_many2
#define PSATD_PLANE_MANY true
#include "reg_planes.cuh"

// Register plane kernels of part 3 for passes over several plane shapes (reg_planes.cuh).
#define PSATD_PLANE_PART 3
#define PSATD_PLANE_NS plane_many3
#define PSATD_PLANE_MANY true
#include "reg_planes.cuh"

// Register plane kernels of part 1 for passes over several plane shapes (reg_planes.cuh).
#define PSATD_PLANE_PART 1
#define PSATD_PLANE_NS plane_many1
#define PSATD_PLANE_MANY true
#include "reg_planes.cuh"

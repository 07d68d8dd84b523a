// Register plane kernels of part 0 for passes over several plane shapes (reg_planes.cuh).
#define PSATD_PLANE_PART 0
#define PSATD_PLANE_NS plane_many0
#define PSATD_PLANE_MANY true
#include "reg_planes.cuh"

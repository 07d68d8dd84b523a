// Register plane kernels: the shapes of part 1 of PSATD_REG_SHAPES (reg_planes.cuh).
#define PSATD_PLANE_PART 1
#define PSATD_PLANE_NS plane_part1
#define PSATD_PLANE_MANY false
#include "reg_planes.cuh"

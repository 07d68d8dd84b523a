// Register plane kernels: the shapes of part 2 of PSATD_REG_SHAPES (reg_planes.cuh).
#define PSATD_PLANE_PART 2
#define PSATD_PLANE_NS plane_part2
#define PSATD_PLANE_MANY false
#include "reg_planes.cuh"

// Register plane kernels: the shapes of part 0 of PSATD_REG_SHAPES (reg_planes.cuh).
#define PSATD_PLANE_PART 0
#define PSATD_PLANE_NS plane_part0
#define PSATD_PLANE_MANY false
#include "reg_planes.cuh"

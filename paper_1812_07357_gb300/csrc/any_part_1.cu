#include "any_part.cuh"

template struct psatd::AnyPart<float, 1>;

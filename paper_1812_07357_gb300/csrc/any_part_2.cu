#include "any_part.cuh"

template struct psatd::AnyPart<double, 0>;

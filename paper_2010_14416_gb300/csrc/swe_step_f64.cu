// FP64 instantiation of the step kernels (arithmetic: swe_f64.cuh).
#include "swe_launch.cuh"

namespace swe {
template struct Launch<double>;
}

// Runtime-length forms, z pass, double-float.
#include "passes_any_launch.cuh"

namespace gsp {
GSP_INSTANTIATE_ANY_Z(DF)
}  // namespace gsp

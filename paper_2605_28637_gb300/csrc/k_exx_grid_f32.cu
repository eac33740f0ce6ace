// Single-precision instantiation of the exact exchange's fused grid passes.
#include "k_exx_grid.cuh"
namespace roks {
ROKS_INSTANTIATE_EXX(float)
}

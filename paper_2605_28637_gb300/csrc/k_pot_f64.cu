// Double-precision instantiation of the potentials' grid passes.
#include "k_pot_impl.cuh"
namespace roks {
ROKS_INSTANTIATE_POT(double)
}

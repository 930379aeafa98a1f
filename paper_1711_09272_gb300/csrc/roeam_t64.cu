// FP64 instantiations of the tile kernels.
#include "roeam_tile.cuh"

namespace roeam {
template struct TileLaunchers<double>;
}

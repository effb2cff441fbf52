// Double-precision instances of the SE kernels.
#include "se_launch.cuh"
namespace se {
SE_INSTANTIATE(double)
SE_INSTANTIATE_GATHER(double)
}

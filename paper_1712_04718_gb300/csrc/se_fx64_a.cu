// Double-precision integer spread and gather, supports 2, 4, 6, 8, 10.
#include "se_fx64_launch.cuh"
namespace se {
SE_FX_INSTANTIATE(2)
SE_FX_INSTANTIATE(4)
SE_FX_INSTANTIATE(6)
SE_FX_INSTANTIATE(8)
SE_FX_INSTANTIATE(10)
}

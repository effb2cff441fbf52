// Double-precision integer spread and gather, supports 20, 22, 24, 26.
#include "se_fx64_launch.cuh"
namespace se {
SE_FX_INSTANTIATE(20)
SE_FX_INSTANTIATE(22)
SE_FX_INSTANTIATE(24)
SE_FX_INSTANTIATE(26)
}

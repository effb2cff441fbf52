// Double-precision integer spread and gather, supports 28, 30, 32.
#include "se_fx64_launch.cuh"
namespace se {
SE_FX_INSTANTIATE(28)
SE_FX_INSTANTIATE(30)
SE_FX_INSTANTIATE(32)
}

// Double-precision integer spread and gather, supports 12, 14, 16, 18.
#include "se_fx64_launch.cuh"
namespace se {
SE_FX_INSTANTIATE(12)
SE_FX_INSTANTIATE(14)
SE_FX_INSTANTIATE(16)
SE_FX_INSTANTIATE(18)
}

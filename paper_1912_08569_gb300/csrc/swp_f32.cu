// FP32 instantiation of the step kernels.
#define SWP_BLOCK kBlock
#include "swp_launch.cuh"
namespace swp {
SWP_INSTANTIATE(float)
}

// FP64 instantiation of the step kernels.
#define SWP_BLOCK kBlock64
#include "swp_launch.cuh"
namespace swp {
SWP_INSTANTIATE(double)
}

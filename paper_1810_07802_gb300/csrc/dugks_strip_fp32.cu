// FP32 instantiation of the strip step kernel.
#include "dugks_strip_launch.cuh"

namespace dugks {
DUGKS_INSTANTIATE_STRIP(float)
}

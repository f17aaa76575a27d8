// march_small.cu -- the single-view raymarch kernels for images too small to fill
// the GPU: warps with 4, 8 or 16 rays (see march_kernels.cuh).
#include "march_kernels.cuh"

namespace cloudvol {

template <typename T>
static void launch_small(const SceneParams &p, const ViewParams &v, const cloud_volume *vol,
                         unsigned long long *counter, int shape, cudaStream_t s) {
    switch (shape) {
        case 4: launch_shape<T, 4, 8>(p, v, vol, counter, s); break;
        case 5: launch_shape<T, 5, 8>(p, v, vol, counter, s); break;
        default: launch_shape<T, 6, 8>(p, v, vol, counter, s);
    }
}

void launch_march_small(const SceneParams &p, const ViewParams &v, const cloud_volume *vol,
                        unsigned long long *counter, int shape, cudaStream_t s) {
    switch (vol->desc.precision) {
        case CLOUD_PRECISION_FP32: launch_small<float>(p, v, vol, counter, shape, s); break;
        case CLOUD_PRECISION_FP16: launch_small<__half>(p, v, vol, counter, shape, s); break;
        case CLOUD_PRECISION_BF16: launch_small<__nv_bfloat16>(p, v, vol, counter, shape, s); break;
        default: launch_small<uint16_t>(p, v, vol, counter, shape, s);
    }
}

}  // namespace cloudvol

// Any-length reciprocal-space kernels in FP64 (16-byte elements: last radices up to 10).
#include "any.cuh"

namespace ofdft {

template <typename T, int RL> static const void *ax0(bool mgp) {
    return mgp ? (const void *)axis0_any_kernel<T, RL, true> : (const void *)axis0_any_kernel<T, RL, false>;
}
template <typename T> const void *any_axis0_kernel(int RL, bool mgp);
template <> const void *any_axis0_kernel<double>(int RL, bool mgp) {
    switch (RL) {
        case 10: return ax0<double, 10>(mgp);
        case 9: return ax0<double, 9>(mgp);
        case 8: return ax0<double, 8>(mgp);
        case 5: return ax0<double, 5>(mgp);
        case 4: return ax0<double, 4>(mgp);
        default: return nullptr;
    }
}

}  // namespace ofdft

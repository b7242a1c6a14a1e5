// Any-length reciprocal-space kernels (any.cuh), one instantiation per last radix RL.
#include "any.cuh"

namespace ofdft {

template <typename T, int RL> static const void *ax0(bool mgp) {
    return mgp ? (const void *)axis0_any_kernel<T, RL, true> : (const void *)axis0_any_kernel<T, RL, false>;
}
template <typename T> const void *any_axis0_kernel(int RL, bool mgp);
template <> const void *any_axis0_kernel<float>(int RL, bool mgp) {
    switch (RL) {
        case 16: return ax0<float, 16>(mgp);
        case 15: return ax0<float, 15>(mgp);
        case 12: return ax0<float, 12>(mgp);
        case 10: return ax0<float, 10>(mgp);
        case 9: return ax0<float, 9>(mgp);
        case 8: return ax0<float, 8>(mgp);
        case 5: return ax0<float, 5>(mgp);
        case 4: return ax0<float, 4>(mgp);
        default: return nullptr;
    }
}

}  // namespace ofdft

// Any-length reciprocal-space kernels with compile-time plans (lengths: any_ct.cuh, list 4).
#include "any_ct.cuh"

namespace ofdft {

bool any_ct_axis0_4(int n, AnyCt &c) {
#define X(A, B, D, W)                                                             \
    if (n == A * B * D) {                                                          \
        c.k = (const void *)axis0_ct_kernel<float, A, B, D, W, false>;            \
        c.k2 = (const void *)axis0_ct_kernel<float, A, B, D, W, true>;            \
        c.RL = D;                                                                     \
        c.lg = W;                                                                     \
        c.nt = any_ct_threads(A * B * D, D, W);                                  \
        return true;                                                                  \
    }
    OFDFT_ANY_CT_4(X)
#undef X
    return false;
}

}  // namespace ofdft

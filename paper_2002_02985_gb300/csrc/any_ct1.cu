// Any-length reciprocal-space kernels with compile-time plans (lengths: any_ct.cuh, list 1).
#include "any_ct.cuh"

namespace ofdft {

bool any_ct_axis0_1(int n, bool narrow, AnyCt &c) {
#define X(A, B, D, W)                                                             \
    if (n == A * B * D) return any_ct_axis0_pick<A, B, D, W>(narrow, c);
    OFDFT_ANY_CT_1(X)
#undef X
    return false;
}

}  // namespace ofdft

// Any-length rows and n1 pencils with compile-time plans (lengths: any_ct.cuh, list 3).
#include "any_ct.cuh"

namespace ofdft {

bool any_ct_rows_3(int n, AnyCt &c) {
#define X(A, B, D, W)                                                                                      \
    if (n == A * B * D) {                                                                                   \
        constexpr int S2 = B > 1 ? B : D, S3 = B > 1 ? D : 1;                 \
        c.k = (const void *)row_fwd_ct_kernel<float, A, S2, S3>;                                           \
        c.k2 = (const void *)row_inv_ct_kernel<float, A, S2, S3>;                                          \
        return true;                                                                                           \
    }
    OFDFT_ANY_CT_3(X)
#undef X
    return false;
}

bool any_ct_pencil_3(int n, AnyCt &c) {
#define X(A, B, D, W)                                                                                          \
    if (n == A * B * D) {                                                                                      \
        constexpr int S2 = B > 1 ? B : D, S3 = B > 1 ? D : 1;                                                  \
        c.k = (const void *)pencil_ct_kernel<float, -1, A, S2, S3, W>;                                         \
        c.k2 = (const void *)pencil_ct_kernel<float, +1, A, S2, S3, W>;                                        \
        c.lg = W;                                                                                              \
        c.nt = any_ct_pencil_threads(n, any_max3(A, B, D), W);                                                 \
        return true;                                                                                           \
    }
    OFDFT_ANY_CT_3(X)
#undef X
    return false;
}

}  // namespace ofdft

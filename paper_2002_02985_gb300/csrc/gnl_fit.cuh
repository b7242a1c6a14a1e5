// Generated by gen_gnl_fit.py (do not edit): polynomial forms of the kernel G_NL of
// Sec. 2.3 for the FP32-mixed kernels.  eta <= 1/2: G_NL = y S(y), y = eta^2; eta >= 2:
// G_NL = L(x), x = 1/eta^2; S (degree 6) and L (degree 6) are Chebyshev
// interpolants on [0, 1/4] of the closed form (largest relative error 1.8e-10 and 1.3e-10,
// below FP32 rounding), evaluated by Horner's rule.  The FP64 forms: degree 12 and 12,
// 7.6e-18 and 6.5e-18 (below FP64 rounding).
#pragma once

namespace ofdft {
__device__ __forceinline__ float gnl_small_s(float y) {
    return fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(6.242049043e-02f, y, 2.573520713e-02f), y, 5.482175907e-02f), y, 7.371785135e-02f), y, 1.100620656e-01f), y, 1.777776332e-01f), y, -2.666666666e+00f);
}
__device__ __forceinline__ float gnl_large_l(float x) {
    return fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(-2.905759356e-02f, x, -1.199505511e-02f), x, -2.629342381e-02f), x, -3.768162710e-02f), x, -6.400429678e-02f), x, -1.371427893e-01f), x, -1.600000000e+00f);
}
__host__ __device__ __forceinline__ double gnl_small_s(double y) {
    double p = 4.063035519654544e-2;
    p = fma(p, y, -1.8829541607595671e-2);
    p = fma(p, y, 2.6139653929309826e-2);
    p = fma(p, y, 1.0999025915251761e-2);
    p = fma(p, y, 1.9194792105050171e-2);
    p = fma(p, y, 2.2983543820697374e-2);
    p = fma(p, y, 2.9532749739959893e-2);
    p = fma(p, y, 3.8738800409493778e-2);
    p = fma(p, y, 5.2452586741931035e-2);
    p = fma(p, y, 7.3932980186063666e-2);
    p = fma(p, y, 1.1005291005763837e-1);
    p = fma(p, y, 1.777777777777566e-1);
    p = fma(p, y, -2.6666666666666667);
    return p;
}
__host__ __device__ __forceinline__ double gnl_large_l(double x) {
    double p = -2.1071984284924865e-2;
    p = fma(p, x, 1.0220675358903625e-2);
    p = fma(p, x, -1.3235953708044825e-2);
    p = fma(p, x, -5.035617753516779e-3);
    p = fma(p, x, -9.0536300973928357e-3);
    p = fma(p, x, -1.0671663725602851e-2);
    p = fma(p, x, -1.3676125924539764e-2);
    p = fma(p, x, -1.8087718392116103e-2);
    p = fma(p, x, -2.5182416058332482e-2);
    p = fma(p, x, -3.7782560078401945e-2);
    p = fma(p, x, -6.4000000002497648e-2);
    p = fma(p, x, -1.3714285714284596e-1);
    p = fma(p, x, -1.6);
    return p;
}
}  // namespace ofdft

// Plain transforms of one or two real fields (plain.cu).
#pragma once

#include "eval.cuh"

namespace ofdft {

// what the n0 pass does: one direction alone, or forward, a factor f(G) and inverse:
// KINETIC G^2/2; CN 1 / (1 + p1^2 (G^2/2 + p2)^2); PRECOND p1 G^2 / (G^4 + p1 G^2 + p2), 1 at G = 0
enum { PLAIN_FORWARD = 0, PLAIN_INVERSE, PLAIN_KINETIC, PLAIN_CN, PLAIN_PRECOND };

template <typename T> struct PlainArgs {
    typedef typename Vec2<T>::type C;
    int n0, n1, n2, n2h;
    AnyPlan q0, q2;
    int lgB, lg0, mode;
    unsigned magic_n, magic_n2h, magic_n4;
    int vec;                     // set at the launch: four points per access
    int nf;                      // fields of the launch, one per blockIdx.y (0 counts as 1)
    C *h;                        // half spectra, hs apart
    long long hs;
    const C *tw0, *tw2;
    const double *scal;          // S_RHO_MEAN: the constant the forward rows subtract
    int sampled;                 // they take it from a sample of the field (and leave it there)
    const T *u[2];               // input fields
    T *out[2];
    const T *v, *vu[2], *base[2];   // epilogue out = c0 base + c1 (y + madd mean + v vu)
    T c0, c1, madd;
    T p1, p2, scale;
    T b[9];                      // 2 pi times the reciprocal vectors
};

// fills the plans and tile sizes of a (its sizes set); false if a length has no plan
template <typename T> bool plain_setup(PlainArgs<T> &a, int nsm);
// mean of u into scal (part: nblk doubles; ticket: zero between launches)
template <typename T>
cudaError_t launch_plain_mean(const T *u, long long N, int nblk, double *part, double *scal, unsigned *ticket,
                              cudaStream_t s);
template <typename T> cudaError_t launch_plain_rows(const PlainArgs<T> &a, bool inverse, cudaStream_t s);
template <typename T> cudaError_t launch_plain_n0(const PlainArgs<T> &a, cudaStream_t s);

}  // namespace ofdft

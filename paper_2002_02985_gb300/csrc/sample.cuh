// The points at which a plain filter samples its field for the constant it subtracts (plain.cu).
#pragma once

namespace ofdft {

constexpr int kPlainSamples = 1024;

// Coordinate of sample k on an axis of n points: floor(n frac(1/2 + k / g^d)), d = 1, 2, 3 for the three
// axes (A = 2^32 / g^d), g = 1.2207... the root of x^4 = x + 1.  The powers of 1/g make a Kronecker
// sequence that fills the cell evenly in all three directions at once, whatever the lengths; a stride
// through the linear index does not (N / 1024 is a multiple of n2 at 32^3 to 256^3: every sample on
// one face, and a cluster in the middle of its cell was sampled at 0.01 of its mean).
#ifdef __CUDACC__
__host__ __device__
#endif
inline int plain_sample_on(int k, unsigned A, int n) {
    return (int)(((unsigned long long)(0x80000000u + (unsigned)k * A) * (unsigned)n) >> 32);
}
// the linear index of sample k of an n0 x n1 x n2 field
#ifdef __CUDACC__
__host__ __device__
#endif
inline long long plain_sample(int k, int n0, int n1, int n2) {
    const int i0 = plain_sample_on(k, 0xd1b54a33u, n0), i1 = plain_sample_on(k, 0xabc98389u, n1),
              i2 = plain_sample_on(k, 0x8cb92ba7u, n2);
    return ((long long)i0 * n1 + i1) * n2 + i2;
}

}  // namespace ofdft

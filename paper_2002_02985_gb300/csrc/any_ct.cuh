// The lengths whose any-length kernels (any.cuh) are also compiled with the plan fixed: every
// 2^a 3^b 5^c from 24 to 512 that three passes of the compiled radices reach.  X(R1, R2, RL, LG):
// n = R1 R2 RL, RL the frequencies a thread of the reciprocal-space pass keeps (8 to 10 where
// the radices allow: 128 registers, two to four blocks per SM), 2^LG columns per tile (16, or 8
// where the three tiles of 16 would leave room for one block per SM); the reciprocal-space pass
// takes its width from any_ct_lg, and a second form of 8 columns from any_ct_narrow.
#pragma once

#include "any.cuh"

#define OFDFT_ANY_CT_1(X) \
    X(3, 1, 8, 4) X(5, 1, 5, 4) X(3, 1, 9, 4) X(3, 1, 10, 4) X(4, 1, 8, 4) X(4, 1, 9, 4) X(5, 1, 8, 4) X(5, 1, 9, 4) \
    X(6, 1, 8, 4) X(5, 1, 10, 4) X(6, 1, 9, 4) X(6, 1, 10, 4) X(8, 1, 8, 4)
#define OFDFT_ANY_CT_2(X) \
    X(9, 1, 8, 4) X(15, 1, 5, 4) X(10, 1, 8, 4) X(9, 1, 9, 4) X(10, 1, 9, 4) X(12, 1, 8, 4) X(10, 1, 10, 4) \
    X(12, 1, 9, 4) X(12, 1, 10, 4) X(5, 5, 5, 4) X(16, 1, 8, 4) X(15, 1, 9, 4) X(16, 1, 9, 4)
#define OFDFT_ANY_CT_3(X) \
    X(15, 1, 10, 4) X(16, 1, 10, 4) X(9, 2, 9, 4) X(15, 1, 12, 4) X(16, 1, 12, 4) X(5, 5, 8, 4) X(6, 4, 9, 4) \
    X(15, 1, 15, 4) X(16, 1, 15, 4) X(9, 3, 9, 4) X(5, 5, 10, 4) X(16, 1, 16, 4) X(6, 5, 9, 3)
#define OFDFT_ANY_CT_4(X) \
    X(6, 6, 8, 3) X(6, 5, 10, 3) X(8, 4, 10, 3) X(6, 6, 9, 3) X(9, 5, 8, 3) X(15, 5, 5, 3) X(8, 6, 8, 3) \
    X(10, 5, 8, 3) X(9, 5, 9, 3) X(8, 6, 9, 3) X(10, 5, 9, 3) X(10, 6, 8, 3) X(9, 6, 9, 3) X(10, 5, 10, 3) X(8, 8, 8, 3)

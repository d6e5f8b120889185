// Reconstruction tables shared by the host generator and the CUDA kernels.
#pragma once

struct CgksTables {
    // stencil st (0 S0, 1 S1, 2 S2, 3 r5, 4 r7, 5 r9), functional row (see
    // tables.cpp), tap over [Qbar_{i-2..i+2}, h*Qx_{i-2..i+2}]
    double row[6][10][10];
    // polynomial coefficients c_0..c_4 of S0, S1, S2 (degree 2) and r5 (degree 4)
    double cpoly[4][5][10];
    // smoothness matrices (Eq. 3.13) of degree-2 and degree-4 polynomials
    double bm2[3][3];
    double bm4[5][5];
    // Gauss-Legendre nodes on [-1/2, 1/2] and weights summing to 1
    double gx[4], gw[4];
    // Step 3 first / second derivative weights over the 3m face points
    double d1[4][12], d2[4][12];
    // the same for the line pairs (l, m-1-l), l = 0 .. (m-1)/2, which mirror each
    // other, on the sums [0] and differences [1] of mirrored points k and 3m-1-k
    // (an odd rule's middle point stands alone in the sums), k = 0 .. 5; entry 6: on
    // the sum and difference of what is common to all points of segments b-1, b+1
    double sd1[2][2][7], sd2[2][2][7];
    // rows of r5, r7, r9 for mirrored places, on sums and differences of mirrored
    // taps (see cgks_device.cuh): value, first and second derivative at xi = 1/2,
    // then the value at Gauss nodes 0 and 1 (of m = 2: 0 only)
    double sym[3][5][8];
    int m;
};

#ifdef __cplusplus
extern "C"
#endif
__attribute__((visibility("hidden"))) int cgks_build_tables(int order, CgksTables* t);

// Elements of the folded contraction matrix (device code shared by the kernels
// that build it):
//   W[A][B] = 1/2 [ (pq|rs) + (k_pq d_rs + d_pq k_rs) / N ],
//   k_pq = h1_pq - 1/2 sum_r (pr|rq), N = 2 nelec_spin.
#pragma once
#include "hamiltonian.cuh"

namespace ifci {

// pair A = P (P + 1) / 2 + Q, Q <= P
__device__ __forceinline__ int pair_row(int A) {
    int P = (int)((sqrtf(8.0f * (float)A + 1.0f) - 1.0f) * 0.5f);
    while ((P + 1) * (P + 2) / 2 <= A) P++;
    while (P * (P + 1) / 2 > A) P--;
    return P;
}

__device__ __forceinline__ double fold_pair(const FoldDesc &d, int A) {
    const int n = d.n, np = n * (n + 1) / 2, P = pair_row(A), Q = A - P * (P + 1) / 2;
    double k = d.h1[P * n + Q];
    for (int r = 0; r < n; r++) k -= 0.5 * d.eri[(long long)pair_of(P, r) * np + pair_of(r, Q)];
    return k;
}

// W[A][B] of pairs A, B < np, given k of every pair
__device__ __forceinline__ double fold_element(const FoldDesc &d, const double *k, double invN, int A, int B) {
    const int np = d.n * (d.n + 1) / 2, P = pair_row(A), R = pair_row(B);
    const bool dA = (A - P * (P + 1) / 2) == P, dB = (B - R * (R + 1) / 2) == R;
    double w = d.eri[(long long)A * np + B];
    if (dB) w += invN * k[A];
    if (dA) w += invN * k[B];
    return 0.5 * w;
}

}  // namespace ifci

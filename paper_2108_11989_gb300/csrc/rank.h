// Order of the Ritz values: increasing |v|, ties by index, NaN behind every number.  A total
// order, so the ranks of any k values are a permutation of 0 .. k - 1 whatever their bits; the
// eigenvector kernel uses them as indices.  Plain C++ (no CUDA headers).
#pragma once

#ifdef __CUDACC__
#define QS_HD __host__ __device__
#else
#define QS_HD
#endif

// |a| at index i comes before |b| at index j (a, b: absolute values)
QS_HD inline bool qs_abs_before(double a, int i, double b, int j)
{
    const bool an = a != a, bn = b != b;
    if (an || bn) return an && bn ? i < j : bn;
    return a < b || (a == b && i < j);
}

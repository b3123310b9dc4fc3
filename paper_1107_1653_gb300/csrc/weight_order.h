// The order in which an interpolation row's weights are kept, in plain C++.
#pragma once

#ifdef __CUDACC__
#define GS_ORDER_FN __host__ __device__ inline
#else
#define GS_ORDER_FN inline
#endif

namespace gs {

// Whether weight a at position p comes before weight b at position q: the larger
// first, the earlier of equal ones, weights that are not numbers last (rows of a
// singular system).  A strict total order, so that the positions of a row get
// distinct ranks whatever their weights hold: a rank that two shared would leave
// another's entry of the row unwritten.
GS_ORDER_FN bool weight_before(double a, int p, double b, int q) {
    const bool na = a != a, nb = b != b;
    if (na || nb) return na == nb ? p < q : nb;
    return a > b || (a == b && p < q);
}

}  // namespace gs

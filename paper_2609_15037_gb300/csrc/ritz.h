// The order of the Ritz values.  It decides which column of the Ritz vectors a
// kernel reads next, so it has to be a total order whatever the values are:
// with a comparison that a NaN answers "no" to both ways, several columns took
// the same rank and other ranks kept what the scratch memory held before.
#pragma once

#include <cmath>
#include <cuda_runtime.h>

namespace moara {

// x^T (C x) / x^T x from its two sums: 0 for a zero column, -inf (behind every
// other value) where a non-finite gradient left no number.
__host__ __device__ inline float ritz_value(float xcx, float xx) {
    const float d = xx > 0.0f ? xcx / xx : 0.0f;
    return d == d ? d : -INFINITY;
}

// Whether value di of column i stands before dj of column j: descending, ties
// by column.
__host__ __device__ inline bool ritz_before(float di, int i, float dj, int j) {
    return di > dj || (di == dj && i < j);
}

}  // namespace moara

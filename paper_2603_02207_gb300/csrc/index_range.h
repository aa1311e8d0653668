// Index steps that stay in range: rows and entries are int32 up to 2^31 - 1, so that `k + step` may wrap just
// before the end and `(lo + hi) / 2` from 2^30 rows on. Differences of two indices of a range never do.
#pragma once

#ifdef __CUDACC__
#define LL_HD __host__ __device__ __forceinline__
#else
#define LL_HD inline
#endif

namespace ll {

// k + step, or end where that lies at or past it (k <= end)
LL_HD int step_to(int k, int step, int end) { return end - k > step ? k + step : end; }

// first i in [0, n] with rowptr[i] + row_cost i >= t
template <typename RowPtr>
LL_HD int rows_start(const RowPtr& rowptr, int n, int row_cost, long long t) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if ((long long)rowptr[mid] + (long long)row_cost * mid >= t) hi = mid; else lo = mid + 1;
    }
    return lo;
}

}  // namespace ll

// Sort of the ray numbers of one source cell in shared memory.
#pragma once

namespace mirage {

// list[0, n) ascending, by `threads` threads of which this is number t, with
// `sync` between steps: a bitonic merge sort whose comparators all point the
// same way (the first step of a merge meets in mirrored pairs), so that n is
// any number and the places beyond it count as infinite.  About log2(n)^2 / 2
// steps of n / 2 comparisons.
template <class Sync>
__device__ __forceinline__ void cell_sort(int* list, int n, int t, int threads, Sync sync) {
    auto meet = [&](int lo, int hi) {
        if (hi < n) {
            const int a = list[lo], b = list[hi];
            if (a > b) {
                list[lo] = b;
                list[hi] = a;
            }
        }
    };
    for (int half = 1, lg = 0; half < n; half <<= 1, ++lg) {  // runs of `half` merged in pairs
        const int pairs = ((n + 2 * half - 1) >> (lg + 1)) << lg;
        for (int p = t; p < pairs; p += threads) {
            const int run = (p >> lg) << (lg + 1), j = p & (half - 1);
            meet(run + j, run + 2 * half - 1 - j);
        }
        sync();
        for (int sl = lg - 1; sl >= 0; --sl) {
            const int s = 1 << sl;
            for (int p = t; p < pairs; p += threads) {
                const int lo = ((p >> sl) << (sl + 1)) + (p & (s - 1));
                meet(lo, lo + s);
            }
            sync();
        }
    }
}

}  // namespace mirage

// The library's sort of a source cell's rays run by host threads:
//   cellsort_host NT < n (int32), n int32 values, ... > the values of each list, sorted
// The steps' barrier is a barrier of the NT threads.
#include <barrier>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

#define __device__
#define __forceinline__ inline
#include "../../paper_1101_5803_gb300/csrc/cellsort.cuh"

int main(int argc, char** argv) {
    if (argc != 2) return 2;
    const int nt = std::atoi(argv[1]);
    int n;
    while (std::fread(&n, 4, 1, stdin) == 1) {
        std::vector<int> list(n);  // (exactly n: an index beyond it is reported)
        if (n && (int)std::fread(list.data(), 4, n, stdin) != n) return 2;
        std::barrier<> bar(nt);
        std::vector<std::thread> th;
        for (int t = 0; t < nt; ++t)
            th.emplace_back([&, t] { mirage::cell_sort(list.data(), n, t, nt, [&] { bar.arrive_and_wait(); }); });
        for (auto& x : th) x.join();
        if (n) std::fwrite(list.data(), 4, n, stdout);
    }
    return 0;
}

// Host check of the order of a patch's multiply covered pixels (cover_order.cuh) against a stable
// sort of the pixels, on patches with few and many covering sets, and on 2^20 pixels under as
// many sets, where a search per pixel of the sets seen so far would take hours.
#include "cover_order.cuh"

#include <cstdio>
#include <numeric>
#include <random>

using namespace cel;

static bool same_order(int n, int n_set, int run, double alone_share, unsigned seed) {
    std::mt19937_64 rng(seed);
    std::vector<uint64_t> set(n_set), mask(n);
    for (auto& m : set) m = rng();
    std::vector<uint8_t> alone(n);
    for (int q = 0; q < n; ++q) {
        alone[q] = std::uniform_real_distribution<double>(0, 1)(rng) < alone_share;
        mask[q] = q % run ? mask[q - 1] : set[rng() % n_set];
    }
    std::vector<int> want, got;
    for (int q = 0; q < n; ++q)
        if (!alone[q]) want.push_back(q);
    std::stable_sort(want.begin(), want.end(), [&](int a, int b) { return mask[a] < mask[b]; });
    std::vector<CoverRun> runs;
    cover_order(alone.data(), mask.data(), n, runs);
    for (const CoverRun& r : runs)
        for (int q = r.q0; q < r.q1; ++q) got.push_back(q);
    return got == want;
}

int main() {
    unsigned seed = 1;
    for (int n : {0, 1, 2, 63, 64, 65, 529, 10201})
        for (int n_set : {1, 2, 7, 500})
            for (int run : {1, 3, 31})
                for (double share : {0.0, 0.4, 1.0})
                    if (!same_order(n, n_set, run, share, ++seed)) return printf("%d %d %d %g\n", n, n_set, run, share), 1;
    if (!same_order(1 << 20, 1 << 20, 1, 0.0, 7)) return printf("2^20\n"), 1;
    return 0;
}

// Spectra of several handles from several host threads, through the C API: the
// first thread's lattice has the longest lines and argv[3] shells, the others'
// shorter lines and argv[4] shells, all above the 48 KB of shared memory every
// kernel may use without asking.  argv[1], argv[2]: the long and the short side;
// argv[5]: 1 puts them along y.  Runs three seconds or up to the first error.
// Prints one JSON line: calls of each kind and the first error (empty: none).
// Test infrastructure only.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "../../include/rlbm.h"

int main(int argc, char **argv) {
    if (argc != 6) return 2;
    const int side[2] = {std::atoi(argv[1]), std::atoi(argv[2])}, shells[2] = {std::atoi(argv[3]), std::atoi(argv[4])};
    const bool along_y = std::atoi(argv[5]) != 0;
    std::atomic<int> ready{0}, stop{0}, calls[2];
    calls[0] = calls[1] = 0;
    std::mutex mu;
    std::string error;
    const int nthreads = 8;
    auto work = [&](int t) {
        const int k = t == 0 ? 0 : 1;
        rlbm_t *h = nullptr;
        std::vector<double> E(4096);
        rlbm_status st = along_y ? rlbm_create(4, side[k], RLBM_STENCIL_SPH26_SLAB, 0.8, nullptr, nullptr, &h)
                                 : rlbm_create(side[k], 4, RLBM_STENCIL_SPH26_SLAB, 0.8, nullptr, nullptr, &h);
        if (st == RLBM_OK) st = rlbm_init_fields(h, nullptr, nullptr, nullptr);
        if (st == RLBM_OK) st = rlbm_energy_spectrum(h, shells[k], E.data());  // work area and module loaded
        ++ready;
        while (ready < nthreads) std::this_thread::yield();
        const auto end = std::chrono::steady_clock::now() + std::chrono::seconds(3);
        while (st == RLBM_OK && !stop && std::chrono::steady_clock::now() < end) {
            st = rlbm_energy_spectrum(h, shells[k], E.data());
            ++calls[k];
        }
        if (st != RLBM_OK) {
            stop = 1;
            std::lock_guard<std::mutex> lock(mu);
            if (error.empty()) error = std::to_string(side[k]) + ": " + rlbm_status_string(st);
        }
        rlbm_destroy(h);
    };
    std::vector<std::thread> threads;
    for (int t = 0; t < nthreads; ++t) threads.emplace_back(work, t);
    for (auto &t : threads) t.join();
    std::printf("{\"long\": %d, \"short\": %d, \"error\": \"%s\"}\n", calls[0].load(), calls[1].load(), error.c_str());
    return 0;
}

// How many chains of a batch are in flight at once when the caller leaves it to the library.  Host
// arithmetic only (no CUDA), so that it compiles on its own.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace bamg {

struct BatchChain {
    int64_t n, nnz;  // of A
    int r, gmres_m, caliber;
    bool fp64, learned;
};

// Device memory of one chain's setup and solve: Krylov and test vectors in FP64, some ten copies of the
// matrix, the products of the coarse operator (a place for each entry of B, caliber squared), the
// learned interpolation's features, outputs and candidates, and the pool's granules.  Peaks measured on chains of 2^18 to 2^20 states (grid walks, tandem
// queues, triangulations; calibers 2 and 4, restart lengths 50 and 64): 0.5 to 1.06 of this.
inline double batch_chain_bytes(const BatchChain& k) {
    const double n = (double)std::max<int64_t>(k.n, 0), nnz = (double)std::max<int64_t>(k.nnz, 0);
    const double c = std::min(std::max(k.caliber, 1), 4), value = k.fp64 ? 8.0 : 4.0;
    return n * (16.0 * (std::max(k.gmres_m, 1) + 2) + 40.0 * std::max(k.r, 0) + 400.0) + 160.0 * nnz +
           (n + nnz) * c * c * (4.0 + 2.0 * value) + (k.learned ? 576.0 * n : 0.0) + 32.0 * (1 << 20);
}

// Host threads for the chains (largest first): one per chain up to 16 (12 chains of 32..60 squared
// states in FP64 took 10.8 ms on 3 threads and 5.9 on 12, 32 chains 15.1 on 8 and 14.6 on 16, 96 chains
// 55.7 on 8 and 50.0 on 16).  More than a thread per four chains only while the largest chains together
// take less than half of the memory that is free, so that a batch that fits with fewer in flight does not
// run out with more, and less than 16 GiB: chains of that size fill the GPU by themselves.
inline int batch_workers(const std::vector<BatchChain>& chains, double free_bytes) {
    const int count = (int)chains.size(), most = std::min(16, count);
    const double budget = std::min(0.5 * free_bytes, 16.0 * (double)(1ull << 30));
    double bytes = 0.0;
    int fit = 0;
    for (; fit < most; ++fit) {
        bytes += batch_chain_bytes(chains[fit]);
        if (!(bytes < budget)) break;
    }
    return std::max(fit, std::min(most, std::max(1, (count + 3) / 4)));
}

}  // namespace bamg

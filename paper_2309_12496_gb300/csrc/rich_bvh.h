// rich_bvh.h -- host BVH builder interface.
#pragma once

#include <cstdint>
#include <algorithm>
#include <atomic>
#include <exception>
#include <mutex>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include "rich_internal.h"

namespace rich {

// Reference of "no surface" (never a node index or a leaf code).
constexpr int32_t kNoSurface = 0x7FFFFFFF;

// f(0) .. f(n - 1) on up to eight host threads; the first exception of any is
// rethrown here. Threads that cannot be started are done without.
template <typename F>
void run_parallel(size_t n, F f) {
    std::atomic<size_t> next{0};
    std::exception_ptr failed;
    std::mutex mu;
    auto work = [&]() {
        for (size_t i; (i = next.fetch_add(1)) < n;) {
            try {
                f(i);
            } catch (...) {
                std::lock_guard<std::mutex> lock(mu);
                if (!failed) failed = std::current_exception();
            }
        }
    };
    const size_t cores = std::max(1u, std::thread::hardware_concurrency());
    const size_t most = std::min<size_t>({n, cores, 8});
    std::vector<std::thread> threads;
    threads.reserve(most);
    for (size_t k = 1; k < most; ++k) {
        try {
            threads.emplace_back(work);
        } catch (const std::system_error &) {
            break;
        }
    }
    work();
    for (std::thread &t : threads) t.join();
    if (failed) std::rethrow_exception(failed);
}

struct BvhResult {
    std::vector<DevNode> nodes;   // breadth-first, node 0 is the root
    std::vector<int> leaf_order;  // leaf-order position -> input triangle
    std::vector<int32_t> surface_ref;  // per leaf-order position: the node
                                  // index or leaf code of the subtree holding
                                  // exactly its surface, or kNoSurface
    int depth = 0;                // inner-node levels
};

// Build over n_tris triangles given as 9 floats each; surface (may be null):
// per triangle a surface id >= 0 shared by the triangles of one surface, or
// -1. Returns false and sets err for malformed input.
bool build_bvh(const float *vertices, const int32_t *surface, int64_t n_tris, BvhResult &out,
               std::string &err);

}  // namespace rich

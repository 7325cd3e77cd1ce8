// Test probe: calls on different objects from two host threads at once, as a
// native program makes them (an interpreter's lock would keep the calls apart).
//
//   threads_probe builds <n> <calls>   rebuilds of two trees of n points, of one and of eight dimensions
//   threads_probe lists <n> <calls>    unordered queries for 50 and for 64 neighbours on two trees of n points
//
// Prints the number of calls that failed and the last error.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/kdt.h"

int main(int argc, char **argv)
{
    if (argc != 4)
        return 2;
    const bool builds = !strcmp(argv[1], "builds");
    const int64_t n = atoll(argv[2]);
    const int calls = atoi(argv[3]);
    std::atomic<int> failed{0};
    std::string last[2];
    auto work = [&](int side) {
        const int D = builds ? (side ? 8 : 1) : 3, k = side ? 64 : 50, Q = 32;
        cudaStream_t s;
        float *points, *d2;
        int32_t *ids;
        cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        cudaMalloc(&points, n * D * sizeof(float));
        cudaMalloc(&ids, (size_t)Q * k * 4);
        cudaMalloc(&d2, (size_t)Q * k * 4);
        std::vector<float> h(n * D);
        uint32_t x = 1u + side;
        for (float &v : h)
            v = (x = x * 1664525u + 1013904223u) * 0x1p-32f;
        cudaMemcpy(points, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice);
        kdt_tree *t = nullptr;
        if (kdt_build(points, n, D, s, &t) != KDT_OK) {
            ++failed;
            last[side] = kdt_last_error();
            return;
        }
        for (int i = 0; i < calls; ++i) {
            const int rc = builds ? kdt_rebuild(t, points, KDT_BUILD_ASYNC, s)
                                  : kdt_knn(t, points, Q, k, 3.4e38f, KDT_UNORDERED, ids, d2, s);
            if (rc != KDT_OK) {
                ++failed;
                last[side] = kdt_last_error();
            }
            if (i % 16 == 0)
                cudaStreamSynchronize(s);
        }
        cudaStreamSynchronize(s);
        kdt_free(t);
    };
    std::thread a(work, 0), b(work, 1);
    a.join();
    b.join();
    printf("%d %s%s\n", failed.load(), last[0].c_str(), last[1].c_str());
    return 0;
}

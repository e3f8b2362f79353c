// Every lane of a few warps holds the same counts; the counters get their sums.
#include "../paper_1907_12933_gb300/csrc/counts.cuh"

#include <cstdio>
#include <cstdlib>

using namespace vbmc;

__global__ void k_counts(Counters* c, unsigned adv, unsigned pts) {
    PointCounts a;
    for (int round = 0; round < 2; ++round) {
        a.adv = adv;
        a.pts = pts;
        a.first = 1000ull - threadIdx.x;
        a.flush(c);
    }
    if (a.adv || a.pts || a.first != ~0ull) c->err = 1u;  // a flush leaves nothing behind
}

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    Counters h{}, *d = nullptr;
    h.first = ~0ull;
    if (cudaMalloc(&d, sizeof h) != cudaSuccess) return 1;
    cudaMemcpy(d, &h, sizeof h, cudaMemcpyHostToDevice);
    k_counts<<<1, 96>>>(d, (unsigned)strtoull(argv[1], nullptr, 10), (unsigned)strtoull(argv[2], nullptr, 10));
    if (cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu %llu %u\n", h.n_adv, h.n_points, h.first, h.err);
    return 0;
}

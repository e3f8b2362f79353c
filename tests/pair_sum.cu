// PairSum over the terms of a file, settled as the rows of folded nets are: n, then n
// triples (w, h high, h low) in FP32. Prints the sum's two parts.
#include "../paper_1907_12933_gb300/csrc/dfloat.cuh"

#include <cstdio>
#include <vector>

using namespace vbmc;

__global__ void k_sum(const float* t, int n, float2* out) {
    PairSum s;
    for (int i = 0; i < n; ++i) {
        s.add(t[3 * i], make_float2(t[3 * i + 1], t[3 * i + 2]));
        if (i % kSettle == kSettle - 1) s.settle();
    }
    s.settle();
    *out = s.a;
}

int main(int argc, char** argv) {
    if (argc != 2) return 2;
    FILE* f = fopen(argv[1], "rb");
    int n = 0;
    if (!f || fread(&n, 4, 1, f) != 1 || n < 1 || n > (1 << 20)) return 2;
    std::vector<float> t(3 * (size_t)n);
    if (fread(t.data(), 4, t.size(), f) != t.size()) return 2;
    fclose(f);
    float *d = nullptr;
    float2 *o = nullptr, r;
    if (cudaMalloc(&d, 4 * t.size()) != cudaSuccess || cudaMalloc(&o, sizeof r) != cudaSuccess) return 1;
    cudaMemcpy(d, t.data(), 4 * t.size(), cudaMemcpyHostToDevice);
    k_sum<<<1, 1>>>(d, n, o);
    if (cudaMemcpy(&r, o, sizeof r, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%a %a\n", r.x, r.y);
    return 0;
}

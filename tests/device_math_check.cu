// Reads n, then n pairs of doubles (a, b) from stdin; writes, per pair, the values
// of the functions named on the command line and of CUDA's own operations.
#include <cstdio>
#include <cstring>
#include <vector>

#include "mba_internal.cuh"

__global__ void eval(int what, int n, const double2 *in, double2 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double a = in[i].x, b = in[i].y;
    if (what == 0) out[i] = make_double2(mba::quotient(a, b, 1.0 / b), a / b);
    if (what == 1) out[i] = make_double2(mba::fast_rcp(a), 1.0 / a);
    if (what == 2) out[i] = make_double2(mba::fast_sqrt(a), sqrt(a));
}

int main(int argc, char **argv) {
    if (argc < 2) return 2;
    const int what = !strcmp(argv[1], "quotient") ? 0 : (!strcmp(argv[1], "rcp") ? 1 : 2);
    int n = 0;
    if (fread(&n, sizeof n, 1, stdin) != 1 || n < 1) return 2;
    std::vector<double2> v(n);
    if (fread(v.data(), sizeof(double2), n, stdin) != (size_t)n) return 2;
    double2 *in = nullptr, *out = nullptr;
    if (cudaMalloc(&in, sizeof(double2) * n) != cudaSuccess || cudaMalloc(&out, sizeof(double2) * n) != cudaSuccess) return 3;
    cudaMemcpy(in, v.data(), sizeof(double2) * n, cudaMemcpyHostToDevice);
    eval<<<(n + 255) / 256, 256>>>(what, n, in, out);
    if (cudaMemcpy(v.data(), out, sizeof(double2) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    return fwrite(v.data(), sizeof(double2), n, stdout) == (size_t)n ? 0 : 2;
}

// The network entry points while operator new fails: nothing may throw across
// the C ABI.  Built and run by tests/test_mlp_no_throw_gpu.py.
#include <cstdio>
#include <cstdlib>
#include <new>

#include <cuda_runtime.h>

#include "fdtd.h"
#include "fdtd_mlp.h"

static bool g_fail = false;
void *operator new(size_t n)
{
    void *p = g_fail ? nullptr : std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

int main()
{
    const int rows = 256, k = 300, n = 64, sizes[3] = {6, 64, 16}, acts[2] = {FDTD_ACT_GELU, FDTD_ACT_NONE};
    char *m = nullptr;
    const size_t mat = (size_t)rows * k * 4;
    if (cudaMalloc(&m, 16 * mat) != cudaSuccess || cudaMemset(m, 0, 16 * mat) != cudaSuccess) return 2;
    auto at = [&](int q) { return (float *)(m + q * mat); };
    size_t image = 0;
    if (fdtd_mlp_net_pack_bytes(sizes, 2, &image) || image > mat) return 3;
    if (fdtd_mlp_to_bf16(at(0), at(1), rows * k, nullptr) || fdtd_mlp_check(nullptr)) return 4;
    const float *bias[2] = {nullptr, nullptr};
    int rc[4] = {};
    g_fail = true;
    rc[0] = fdtd_mlp_forward(at(1), 1, rows, k, at(2), nullptr, n, FDTD_ACT_GELU, nullptr, at(3), at(4), nullptr);
    rc[1] = fdtd_mlp_forward(at(1), 1, rows, 64, at(2), nullptr, n, FDTD_ACT_GELU, nullptr, at(3), at(4), nullptr);
    rc[2] = fdtd_mlp_backward(at(1), 1, at(4), at(5), rows, k, n, FDTD_ACT_GELU, at(2), at(6), at(7), at(8), at(9),
                              nullptr);
    rc[3] = fdtd_mlp_net_forward(at(0), rows, sizes, 2, acts, at(10), bias, 1.f, at(11), nullptr);
    g_fail = false;
    const int last = fdtd_mlp_check(nullptr);
    std::printf("%d %d %d %d %d\n", rc[0], rc[1], rc[2], rc[3], last);
    cudaFree(m);
    return 0;
}

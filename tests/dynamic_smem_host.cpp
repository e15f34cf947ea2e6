// The dynamic shared memory limit of kernels (csrc/dynamic_smem.h) on a fake CUDA runtime.
#include "dynamic_smem.h"

#include <cstdio>
#include <thread>
#include <vector>

static int g_device = 0, g_fail = 0;
static std::map<std::pair<int, const void *>, int> g_limit;  // written under the header's lock only

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *k, cudaFuncAttribute, int v) {
    if (g_fail) return cudaErrorInvalidValue;
    g_limit[{g_device, k}] = v;
    return cudaSuccess;
}
}

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    using spg::allow_dynamic_smem;
    static char kernels[3];
    const void *a = kernels, *b = kernels + 1, *c = kernels + 2;
    // a narrow product after a wide one leaves room for the wide one's launch
    CHECK(allow_dynamic_smem(a, 98000) == cudaSuccess && allow_dynamic_smem(a, 20000) == cudaSuccess);
    CHECK((g_limit[{0, a}] == 98000));
    CHECK(allow_dynamic_smem(a, 120000) == cudaSuccess && (g_limit[{0, a}] == 120000));
    CHECK(allow_dynamic_smem(b, 1000) == cudaSuccess && (g_limit[{0, b}] == 1000));
    g_device = 1;  // every device has its own
    CHECK(allow_dynamic_smem(a, 20000) == cudaSuccess && (g_limit[{1, a}] == 20000));
    g_fail = 1;
    CHECK(allow_dynamic_smem(a, 300000) == cudaErrorInvalidValue);
    g_fail = 0;
    CHECK(allow_dynamic_smem(a, 60000) == cudaSuccess && (g_limit[{1, a}] == 60000));  // the failure was not taken for done
    g_device = 0;
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([=] { for (int i = 0; i < 2000; ++i) allow_dynamic_smem(c, 1000 * (1 + (k * 7 + i) % 50)); });
    for (auto &x : t) x.join();
    CHECK((g_limit[{0, c}] == 50000));
    std::printf("ok\n");
    return 0;
}

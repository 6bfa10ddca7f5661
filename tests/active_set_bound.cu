// One launch of the master problems, or of the Gram growth, on two signals with active sets of the
// given sizes and a given host bound on them.
#include <vector>

#include "../paper_1302_5010_gb300/csrc/mpl_internal.cuh"

using namespace mpl;

namespace {
template <typename T>
T* up(const std::vector<T>& v) {
    T* p = nullptr;
    if (cudaMalloc(&p, v.size() * sizeof(T)) != cudaSuccess) return nullptr;
    if (cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess) return nullptr;
    return p;
}
}  // namespace

// what: 0 master problems (identity blocks, h = 1, 2, ... ), 1 Gram growth (one-hot atoms).  x, g: host copies of
// x_S and the Gram blocks afterwards (2 x smax, 2 x smax x smax).  Returns the device's error code, or -1.
extern "C" int run_bound(int what, int s0, int s1, int bound, int smax, float* x, float* g) {
    const int n = smax, m = smax, p = 2;
    const std::vector<int> sizes = {s0, s1};
    std::vector<float> G((size_t)p * smax * smax, 0.f), h((size_t)p * smax), A((size_t)m * n, 0.f);
    std::vector<int> S((size_t)p * smax);
    for (int i = 0; i < p; ++i)
        for (int a = 0; a < smax; ++a) {
            if (what == 0) G[((size_t)i * smax + a) * smax + a] = 1.f;
            h[i * smax + a] = (float)(a + 1);
            S[i * smax + a] = a;
            A[(size_t)a * n + a] = 1.f;
        }
    Counters c{};
    c.apg_n = c.grow_n = p;
    Dev d{};
    d.n = n;
    d.m = m;
    d.p = p;
    d.smax = smax;
    d.rho = 1;
    d.inner_max = 50;
    d.stop_eps = -1.f;
    d.A32 = up(A);
    d.G = up(G);
    d.h = up(h);
    d.S = up(S);
    d.xS = up(std::vector<float>((size_t)p * smax, 0.f));
    d.ritz = up(std::vector<float>((size_t)p * smax, 0.f));
    d.lam = up(std::vector<float>(p, 0.5f));
    d.eps = up(std::vector<float>(p, 1e-6f));
    d.f0 = up(std::vector<float>(p, 1.f));
    d.ssize = up(sizes);
    d.snew = up(sizes);
    d.outer = up(std::vector<int>(p, 1));
    d.inner = up(std::vector<int>(p, 0));
    d.list_apg = d.list_grow = up(std::vector<int>{0, 1});
    d.cnt = up(std::vector<Counters>{c});
    int64_t nl = 0;
    cudaError_t e = cudaSuccess;
    if (what == 0)
        for (int k = 0; k < apg_classes(d, bound) && e == cudaSuccess; ++k) e = launch_apg(d, p, 152, bound, nullptr, &nl, k);
    else
        e = launch_gram(d, p, smax, bound, 152, nullptr, &nl);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(x, d.xS, (size_t)p * smax * sizeof(float), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(g, d.G, (size_t)p * smax * smax * sizeof(float), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&c, d.cnt, sizeof(c), cudaMemcpyDeviceToHost);
    const void* all[] = {d.A32, d.G, d.h, d.S, d.xS, d.ritz, d.lam, d.eps, d.f0, d.ssize, d.snew, d.outer, d.inner, d.list_apg, d.cnt};
    for (const void* q : all) cudaFree(const_cast<void*>(q));
    return e == cudaSuccess ? c.err : -1;
}

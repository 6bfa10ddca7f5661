// The split TF32 correlation with waits that give up after 0.2 ms instead of 4 s, callable by itself.
// Inputs whose non-finite scores keep a block busy for longer than that make one run out.
#define MPL_WAIT_LIMIT_NS 200000ull
#include "../paper_1302_5010_gb300/csrc/corr_tf32.cu"

#include <vector>

// A (m, n), R (p, n), C (p, m): device memory.  Returns the kernel's own error code (0: none) in *err.
extern "C" int run_tf32(const float* A, int n, int m, const float* R, int p, float* C, int* err) {
    using namespace mpl;
    Counters* cnt = nullptr;
    int* act = nullptr;
    std::vector<int> ids(p);
    for (int i = 0; i < p; ++i) ids[i] = i;
    Counters c{};
    c.act_n[0] = p;
    cudaError_t e = cudaMalloc(&cnt, sizeof(Counters));
    if (e == cudaSuccess) e = cudaMalloc(&act, p * sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpy(cnt, &c, sizeof(c), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(act, ids.data(), p * sizeof(int), cudaMemcpyHostToDevice);
    Dev d{};
    d.n = n;
    d.m = m;
    d.p = p;
    d.A32 = A;
    d.R32 = const_cast<float*>(R);
    d.Cs = C;
    d.act[0] = act;
    d.cnt = cnt;
    int64_t nl = 0;
    if (e == cudaSuccess) e = launch_corr_tf32(d, 0, p, nullptr, &nl);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&c, cnt, sizeof(c), cudaMemcpyDeviceToHost);
    *err = c.err;
    cudaFree(act);
    cudaFree(cnt);
    return (int)e;
}

// Learned warm start for BMPL: the per-atom proposal network's support
// features and its training.
//
// Gram row norms ||A^T a_j|| (one of the network's inputs) are estimated with
// a Rademacher sketch: for z_t = sum_j s_tj a_j (s_tj = +-1 from a hash),
// E[(z_t^T a_j)^2] = sum_k (a_k^T a_j)^2, averaged over T sketch vectors.
//
// Training (offline, not part of a solve): examples (features, label) come from
// the selection kernel's example mode on the first correlation C0 = A^T B, with
// labels j in supp(x*) from reference solutions.  Each minibatch is two kernels: forward
// and backward over groups of examples with a row of partial gradients per CTA, then
// the sum of those rows and the Adam step.
#include "mpl_internal.cuh"

namespace mpl {

namespace {

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}

// Z (T x n): z_t = sum_j s_tj a_j.  One thread per (t, k).
__global__ void k_sketch(const float* __restrict__ A32, int n, int m, int T, float* __restrict__ Z) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    if (k >= n || t >= T) return;
    float acc = 0.f;
    for (int j = 0; j < m; ++j) {
        const float s = (mix64(((uint64_t)t << 32) ^ (uint64_t)j) & 1ull) ? 1.f : -1.f;
        acc = fmaf(s, __ldg(A32 + (size_t)j * n + k), acc);
    }
    Z[(size_t)t * n + k] = acc;
}

// rn_j = sqrt(mean_t C[t][j]^2), C = Z A^T rows (T x m).
__global__ void k_rownorm(const float* __restrict__ C, int m, int T, float* __restrict__ rn) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    float s = 0.f;
    for (int t = 0; t < T; ++t) {
        const float v = C[(size_t)t * m + j];
        s = fmaf(v, v, s);
    }
    rn[j] = sqrtf(s / (float)T);
}

// Training step of the proposal network: k_train_fwd_bwd works out the gradient of one
// minibatch as partial sums, k_train_adam adds them up and takes the Adam step.
//
// A minibatch is small (2048 examples, 53 MFLOP) and the steps are a serial chain, so the step
// is bound by latency: the pass spreads groups of TR_EX = 16 examples over the SMs (2048
// examples fill 128 CTAs; a thread per example, as before, left all but 16 SMs idle and
// serialised its lanes on shared-memory atomics).  In a group every product is split over
// 256 threads: thread t takes unit t % 64 of the layer for four examples (weights
// conflict-free through rows of 65 floats, activations as broadcast float4), and a 4 x 4
// block of the 64 x 64 layer's gradient, kept in registers over the CTA's groups.  Each CTA
// writes its sums to a row of its own, so nothing is added atomically and the result does
// not depend on the order the CTAs run in.  4096 signals (262144 examples, 4 epochs of 128
// steps of 2048) train in 10.1 ms a call, with the examples and the orders made, against
// 392 ms for the thread per example.
constexpr int TR_THREADS = 256;
constexpr int TR_EX = 16;                 // examples per group
constexpr int TR_LD = PROP_H + 4;         // activation rows (16-byte aligned)
constexpr int TR_WLD = PROP_H + 1;        // W2 rows
constexpr int TR_LOSS = 0, TR_LIVE = 1;   // slots of a partial row below the trainable part

static_assert(PROP_H == 64 && TR_THREADS == 4 * PROP_H && TR_EX == 16, "the thread layout of the training pass");

struct TrainSmem {
    float h1[TR_EX][TR_LD];   // layer 1 after ReLU
    float d2[TR_EX][TR_LD];   // gradient before layer 2's ReLU
    float h2[TR_EX][TR_LD];   // layer 2 after ReLU; then the gradient before layer 1's ReLU
    float w2[PROP_H * TR_WLD];
    float w1[PROP_H * 3], b1[PROP_H], b2[PROP_H], w3[PROP_H];
    float x[TR_EX][4];        // standardised features, 1 (the bias input)
    float y[TR_EX];
    float zp[TR_EX][2];       // logit halves (32 units each)
    float dz[TR_EX], loss[TR_EX];
    int live[TR_EX];
};

// Forward + backward over examples perm[off .. off + count) in groups of TR_EX, group g by CTA
// g mod gridDim.x.  ex: examples (f0, f1, f2, y), empty slots with y = -1.  part: gridDim.x rows
// of PROP_NPARAM partial sums (the trainable part; the loss and the live examples below it).
__global__ void __launch_bounds__(TR_THREADS) k_train_fwd_bwd(const float* __restrict__ w, const float* __restrict__ ex,
                                                              const int* __restrict__ perm, int off, int count,
                                                              float inv_batch, float* __restrict__ part) {
    __shared__ __align__(16) TrainSmem sh;
    const int tid = threadIdx.x, lane = tid & 31;
    const int u = tid & (PROP_H - 1), quad = tid >> 6;  // unit and example quad of this thread
    const int e0 = quad * 4;
    const int o4 = (tid >> 4) * 4, q4 = (tid & 15) * 4;  // 4 x 4 block of the W2 gradient
    float g2[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) g2[a][b] = 0.f;
    float g1 = 0.f, gs = 0.f;            // W1/b1 entry (u, quad); b2/w3 entry (quads 0 and 1)
    float lsum = 0.f, dsum = 0.f;        // loss and b3 (thread 0)
    int nlive = 0;
    const int ngroups = (count + TR_EX - 1) / TR_EX;
    // the next group's examples are read while this one is worked on
    float4 f = make_float4(0.f, 0.f, 0.f, -1.f);
    auto fetch = [&](int g) {
        const int e = g * TR_EX + tid;
        if (tid < TR_EX) {
            f = make_float4(0.f, 0.f, 0.f, -1.f);
            if (g < ngroups && e < count)
                f = __ldg(reinterpret_cast<const float4*>(ex + (size_t)perm[off + e] * 4));
        }
    };
    pdl_enter();
    fetch(blockIdx.x);
    for (int t = tid; t < PROP_H * PROP_H; t += TR_THREADS) sh.w2[(t >> 6) * TR_WLD + (t & 63)] = w[P_W2 + t];
    if (tid < PROP_H * 3) sh.w1[tid] = w[P_W1 + tid];
    if (tid < PROP_H) {
        sh.b1[tid] = w[P_B1 + tid];
        sh.b2[tid] = w[P_B2 + tid];
        sh.w3[tid] = w[P_W3 + tid];
    }
    const float b3 = w[P_B3];
    float mean[3], sd[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) { mean[q] = w[P_MEAN + q]; sd[q] = w[P_STD + q]; }
    for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
        if (tid < TR_EX) {
            const bool live = f.w >= 0.f;  // empty slots carry y = -1
            sh.live[tid] = live ? 1 : 0;
            sh.y[tid] = f.w;
            sh.x[tid][0] = (f.x - mean[0]) / sd[0];
            sh.x[tid][1] = (f.y - mean[1]) / sd[1];
            sh.x[tid][2] = (f.z - mean[2]) / sd[2];
            sh.x[tid][3] = 1.f;
        }
        __syncthreads();
        fetch(g + gridDim.x);
        // layer 1
        {
            const float wa = sh.w1[u * 3], wb = sh.w1[u * 3 + 1], wc = sh.w1[u * 3 + 2], bb = sh.b1[u];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* x = sh.x[e0 + e];
                sh.h1[e0 + e][u] = fmaxf(bb + wa * x[0] + wb * x[1] + wc * x[2], 0.f);
            }
        }
        __syncthreads();
        // layer 2 and the logit
        float a2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) a2[e] = sh.b2[u];
#pragma unroll 4
        for (int q = 0; q < PROP_H; q += 4) {
            const float* wr = sh.w2 + u * TR_WLD + q;
            const float wa = wr[0], wb = wr[1], wc = wr[2], wd = wr[3];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 h = *reinterpret_cast<const float4*>(&sh.h1[e0 + e][q]);
                a2[e] = fmaf(wd, h.w, fmaf(wc, h.z, fmaf(wb, h.y, fmaf(wa, h.x, a2[e]))));
            }
        }
        const float w3u = sh.w3[u];
        float zs[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float h = fmaxf(a2[e], 0.f);
            sh.h2[e0 + e][u] = h;
            zs[e] = w3u * h;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1)
#pragma unroll
            for (int e = 0; e < 4; ++e) zs[e] += __shfl_xor_sync(0xffffffffu, zs[e], o);
        if (lane == 0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) sh.zp[e0 + e][(u >> 5)] = zs[e];
        }
        __syncthreads();
        // binary cross-entropy with logits, stable form; dz = sigmoid(z) - y (mean over the batch)
        if (tid < TR_EX) {
            const float z = b3 + (sh.zp[tid][0] + sh.zp[tid][1]), y = sh.y[tid];
            const bool live = sh.live[tid] != 0;
            sh.loss[tid] = live ? fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z))) : 0.f;
            sh.dz[tid] = live ? (1.f / (1.f + expf(-z)) - y) * inv_batch : 0.f;
        }
        __syncthreads();
        // the gradient before layer 2's ReLU
#pragma unroll
        for (int e = 0; e < 4; ++e) sh.d2[e0 + e][u] = a2[e] > 0.f ? sh.dz[e0 + e] * w3u : 0.f;
        __syncthreads();
        // before layer 1's ReLU: dh1 = W2^T d2 (unit u of layer 1)
        float d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int o = 0; o < PROP_H; o += 4) {
            const float* wr = sh.w2 + o * TR_WLD + u;
            const float wa = wr[0], wb = wr[TR_WLD], wc = wr[2 * TR_WLD], wd = wr[3 * TR_WLD];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 v = *reinterpret_cast<const float4*>(&sh.d2[e0 + e][o]);
                d1[e] = fmaf(wd, v.w, fmaf(wc, v.z, fmaf(wb, v.y, fmaf(wa, v.x, d1[e]))));
            }
        }
        // gradients that read d2, h1 and h2
#pragma unroll 4
        for (int e = 0; e < TR_EX; ++e) {
            const float4 dv = *reinterpret_cast<const float4*>(&sh.d2[e][o4]);
            const float4 hv = *reinterpret_cast<const float4*>(&sh.h1[e][q4]);
            const float ds[4] = {dv.x, dv.y, dv.z, dv.w}, hs[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) g2[a][b] = fmaf(ds[a], hs[b], g2[a][b]);
        }
        if (quad == 0) {
#pragma unroll
            for (int e = 0; e < TR_EX; ++e) gs += sh.d2[e][u];                    // b2
        } else if (quad == 1) {
#pragma unroll
            for (int e = 0; e < TR_EX; ++e) gs = fmaf(sh.dz[e], sh.h2[e][u], gs);  // w3
        } else if (tid == TR_THREADS - 1) {
#pragma unroll
            for (int e = 0; e < TR_EX; ++e) { dsum += sh.dz[e]; lsum += sh.loss[e]; nlive += sh.live[e]; }
        }
        __syncthreads();  // every reader of h2 is done: it takes the gradient before layer 1's ReLU
#pragma unroll
        for (int e = 0; e < 4; ++e) sh.h2[e0 + e][u] = sh.h1[e0 + e][u] > 0.f ? d1[e] : 0.f;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < TR_EX; ++e) g1 = fmaf(sh.h2[e][u], sh.x[e][quad], g1);  // W1, b1
        __syncthreads();
    }
    float* out = part + (size_t)blockIdx.x * PROP_NPARAM;
    if (quad < 3) out[P_W1 + u * 3 + quad] = g1;
    else out[P_B1 + u] = g1;
    if (quad == 0) out[P_B2 + u] = gs;
    else if (quad == 1) out[P_W3 + u] = gs;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) out[P_W2 + (o4 + a) * PROP_H + q4 + b] = g2[a][b];
    if (tid == TR_THREADS - 1) {
        out[P_B3] = dsum;
        out[TR_LOSS] = lsum;
        out[TR_LIVE] = (float)nlive;  // at most the examples of one CTA's groups; summed as integers below
    }
}

// Sum over the rows of part (rows, PROP_NPARAM) of column t: TR_RED_G threads per column, each
// every TR_RED_G-th row with its loads in flight together, then a fixed order.
constexpr int TR_RED_COLS = 32, TR_RED_G = 8;
__device__ __forceinline__ float train_column(const float* __restrict__ part, int rows, int t, float (*red)[TR_RED_COLS]) {
    const int col = threadIdx.x & 31, grp = threadIdx.x >> 5;
    float a = 0.f;
    if (t < PROP_NPARAM) {
#pragma unroll 8
        for (int r = grp; r < rows; r += TR_RED_G) a += part[(size_t)r * PROP_NPARAM + t];
    }
    red[grp][col] = a;
    __syncthreads();
    float s = 0.f;
    if (grp == 0)
#pragma unroll
        for (int g = 0; g < TR_RED_G; ++g) s += red[g][col];
    return s;
}

// Loss sum and live examples of a pass, by block 0 (columns TR_LOSS and TR_LIVE).
__device__ __forceinline__ void train_loss(const float* __restrict__ part, int rows, float s, float* loss_acc,
                                           int* n_acc) {
    if (threadIdx.x == TR_LOSS) *loss_acc += s;
    if (threadIdx.x == TR_LIVE) {
        int c = 0;
        for (int r = 0; r < rows; ++r) c += (int)part[(size_t)r * PROP_NPARAM + TR_LIVE];
        *n_acc += c;
    }
}

// The pass's gradient as one vector (the trainable part is added to grad).
__global__ void __launch_bounds__(TR_RED_COLS * TR_RED_G) k_train_grad(const float* __restrict__ part, int rows,
                                                                       float* __restrict__ grad, float* loss_acc,
                                                                       int* n_acc) {
    pdl_enter();
    __shared__ float red[TR_RED_G][TR_RED_COLS];
    const int t = blockIdx.x * TR_RED_COLS + (threadIdx.x & 31);
    const float s = train_column(part, rows, t, red);
    if (threadIdx.x >= TR_RED_COLS) return;
    if (blockIdx.x == 0) train_loss(part, rows, s, loss_acc, n_acc);
    if (t >= PROP_FIRST_TRAINABLE && t < PROP_NPARAM) grad[t] += s;
}

// Gradient sums and the Adam step on the trainable parameters in one kernel.  step is 1-based.
__global__ void __launch_bounds__(TR_RED_COLS * TR_RED_G) k_train_adam(const float* __restrict__ part, int rows,
                                                                       float* __restrict__ w, float* __restrict__ m1,
                                                                       float* __restrict__ m2, float lr, int step,
                                                                       float* loss_acc, int* n_acc) {
    pdl_enter();
    __shared__ float red[TR_RED_G][TR_RED_COLS];
    const int t = blockIdx.x * TR_RED_COLS + (threadIdx.x & 31);
    const float g = train_column(part, rows, t, red);
    if (threadIdx.x >= TR_RED_COLS) return;
    if (blockIdx.x == 0) train_loss(part, rows, g, loss_acc, n_acc);
    if (t < PROP_FIRST_TRAINABLE || t >= PROP_NPARAM) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float a = b1 * m1[t] + (1.f - b1) * g;
    const float b = b2 * m2[t] + (1.f - b2) * g * g;
    m1[t] = a;
    m2[t] = b;
    const float ah = a / (1.f - powf(b1, (float)step)), bh = b / (1.f - powf(b2, (float)step));
    w[t] -= lr * ah / (sqrtf(bh) + eps);
}

// BF16-rounded copy of the parameters for inference (normalisation constants stay FP32).
__global__ void k_round_bf16(const float* __restrict__ w, float* __restrict__ wb) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= PROP_NPARAM) return;
    wb[t] = t < PROP_FIRST_TRAINABLE ? w[t] : __bfloat162float(__float2bfloat16_rn(w[t]));
}

}  // namespace

cudaError_t launch_sketch_rownorm(const float* A32, int n, int m, int T, float* Z, cudaStream_t s, int64_t* nl) {
    dim3 grid((n + 127) / 128, T);
    k_sketch<<<grid, 128, 0, s>>>(A32, n, m, T, Z);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_rownorm(const float* C, int m, int T, float* rn, cudaStream_t s, int64_t* nl) {
    k_rownorm<<<(m + 255) / 256, 256, 0, s>>>(C, m, T, rn);
    ++*nl;
    return cudaGetLastError();
}

// CTAs (and partial rows) of a pass over count examples.
static int train_rows(int count) {
    const int groups = (count + TR_EX - 1) / TR_EX;
    return groups < TRAIN_MAX_ROWS ? groups : TRAIN_MAX_ROWS;
}

static cudaError_t launch_train_pass(const float* w, const float* ex, const int* perm, int off, int count,
                                     float inv_batch, float* part, cudaStream_t s, int64_t* nl) {
    const cudaError_t e = launch_chain(k_train_fwd_bwd, dim3(train_rows(count)), dim3(TR_THREADS), 0, s, w, ex, perm,
                                       off, count, inv_batch, part);
    if (e == cudaSuccess) ++*nl;
    return e;
}

constexpr int TR_RED_BLOCKS = (PROP_NPARAM + TR_RED_COLS - 1) / TR_RED_COLS;

cudaError_t launch_train_grad(const float* w, const float* ex, const int* perm, int count, float inv_batch,
                              float* part, float* grad, float* loss_acc, int* n_acc, cudaStream_t s, int64_t* nl) {
    if (count <= 0) return cudaSuccess;
    cudaError_t e = launch_train_pass(w, ex, perm, 0, count, inv_batch, part, s, nl);
    if (e != cudaSuccess) return e;
    e = launch_chain(k_train_grad, dim3(TR_RED_BLOCKS), dim3(TR_RED_COLS * TR_RED_G), 0, s, part, train_rows(count),
                     grad, loss_acc, n_acc);
    if (e == cudaSuccess) ++*nl;
    return e;
}

cudaError_t launch_train_step(float* w, const float* ex, const int* perm, int off, int count, float inv_batch,
                              float* part, float* m1, float* m2, float lr, int step, float* loss_acc, int* n_acc,
                              cudaStream_t s, int64_t* nl) {
    if (count <= 0) return cudaSuccess;
    cudaError_t e = launch_train_pass(w, ex, perm, off, count, inv_batch, part, s, nl);
    if (e != cudaSuccess) return e;
    e = launch_chain(k_train_adam, dim3(TR_RED_BLOCKS), dim3(TR_RED_COLS * TR_RED_G), 0, s, part, train_rows(count), w,
                     m1, m2, lr, step, loss_acc, n_acc);
    if (e == cudaSuccess) ++*nl;
    return e;
}

cudaError_t launch_round_bf16(const float* w, float* wb, cudaStream_t s, int64_t* nl) {
    k_round_bf16<<<(PROP_NPARAM + 255) / 256, 256, 0, s>>>(w, wb);
    ++*nl;
    return cudaGetLastError();
}

}  // namespace mpl

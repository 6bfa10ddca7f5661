// Master problem (eq. "primal_MPL") and residual update of Algorithm 1,
// batched over signals, plus solve set-up and output.
//
//   k_init      x^0 = 0, xi^0 = b, I_0 = {} (the initialisation of Alg. 1)
//   k_gram      new rows of the Gram block G_S = A_S^T A_S and h_S = A_S^T b
//               for the atoms appended this iteration (the explicit copies of
//               A_I that Sec. 2.4 recommends become Gram rows here)
//   k_apg       accelerated proximal gradient on
//                   min_u lambda*||u||_1 + 0.5 u^T G u - h^T u
//               warm started from x_S (Alg. 1), stopped by eq. (inner)
//               or s_max; persistent CTAs pull signals from a device queue
//   k_residual  xi = b - A_S x_S (the residual update of Alg. 1), FP32 (+ BF16 copy)
//   k_scatter   dense X from the active sets
//   k_smpl_prune  Algorithm 2's pruning of the explored atoms back to rho
// (the Gram growth read out of Q instead of k_gram is in corr_q.cu.)  The chain's
// kernels start with pdl_enter (programmatic dependent launch).
#include <algorithm>

#include "mpl_internal.cuh"

namespace mpl {

#ifdef MPL_APG_TRACE
// Per-signal phase cycle counters of the master problem (diagnostic builds only):
// [Gram block + vectors, power iteration, FISTA, write-back, master problems, FISTA iterations]
__device__ long long g_apg_trace[8192][8];
#define AT_BEGIN long long at0_ = clock64();
#define AT_ADD(slot) do { if (threadIdx.x == 0 && i < 8192) g_apg_trace[i][slot] += clock64() - at0_; at0_ = clock64(); } while (0)
#define AT_CNT(slot, v) do { if (threadIdx.x == 0 && i < 8192) g_apg_trace[i][slot] += (v); } while (0)
#else
#define AT_BEGIN
#define AT_ADD(slot) do {} while (0)
#define AT_CNT(slot, v) do {} while (0)
#endif

namespace {

__device__ __forceinline__ float block_sum(float v, float* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < nw; ++w) t += red[w];  // same order in every thread
    return t;
}

// block_sum without its leading barrier, for callers where a barrier already separates
// the previous readers of red from these writes.
__device__ __forceinline__ float block_sum_after_barrier(float v, float* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < nw; ++w) t += red[w];  // same order in every thread
    return t;
}

// Sums of four values over the CTA, in part[0..4) for the threads of warp 0.  FP64 instructions take two
// lanes a cycle on an SM: each level of the butterfly halves the values a lane carries, and one
// warp adds the warps' totals (part: 4 per warp).  Fixed order.
__device__ __forceinline__ void block_sum4_d(double (&v)[4], double* part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int h = 2, o = 16; h; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const double send = up ? v[q] : v[q + h];
            v[q] = (up ? v[q + h] : v[q]) + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 4; o; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    // lane 8 q holds the warp's total of value q (bits 16, 8 of the lane: 2, 1 of q)
    if ((lane & 7) == 0) part[warp * 4 + (lane >> 3)] = v[0];
    __syncthreads();
    if (warp == 0) {
        double t = 0.0;
        for (int w = lane >> 2; w < nw; w += 8) t += part[w * 4 + (lane & 3)];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        __syncwarp();
        if (lane < 4) part[lane] = t;
        __syncwarp();
    }
}

// s += x x in double-FP32 (the product exact, the sum to 2^-46).
__device__ __forceinline__ void add_square(float x, float& hi, float& lo) {
    const float p = x * x, e = fmaf(x, x, -p);
    const float t = hi + p, z = t - hi;
    lo += ((hi - (t - z)) + (p - z)) + e;
    hi = t;
}

__device__ __forceinline__ float softf(float v, float t) {
    return v > t ? v - t : (v < -t ? v + t : 0.f);
}

// ------------------------------------------------------------------ init
__global__ void __launch_bounds__(256) k_init(Dev d) {
    pdl_enter();
    const int i = blockIdx.x;
    if (i >= d.p) return;
    __shared__ double red[32];
    const int n = d.n;
    const float* b = d.B + (size_t)i * n;
    float* r32 = d.R32 + (size_t)i * n;
    double* r64 = d.R64 + (size_t)i * n;
    // ||b||^2 in FP64; the rounding terms, which feed bounds with a margin of 1e-6, in pairs of floats (a third
    // of the FP64 work; with the sums below 2048 signals of 1024 entries 73 -> 31 us, 256 of them 14.5 -> 8.4)
    double ss = 0.0;
    float eh = 0.f, el = 0.f, th = 0.f, tl = 0.f;
    int nf = 0;
    // entries k = tid + j nt in order of j; four loads in flight before their stores
    for (int k0 = threadIdx.x; k0 < n; k0 += 4 * blockDim.x) {
        float bv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * blockDim.x;
            bv[u] = k < n ? b[k] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * blockDim.x;
            if (k >= n) break;
            const float v = bv[u];
            if (!isfinite(v)) nf = 1;
            r32[k] = v;
            d.R32lo[(size_t)i * n + k] = 0.f;
            r64[k] = (double)v;
            const __nv_bfloat16 q = __float2bfloat16_rn(v);
            if (d.R16) d.R16[(size_t)i * n + k] = q;
            if (d.pos) d.R16c[(size_t)i * n + k] = q;  // active list = identity
            ss += (double)v * (double)v;
            const float fq = __bfloat162float(q);
            add_square(v - fq, eh, el);  // (the difference is exact)
            add_square(fq, th, tl);
        }
    }
    uint32_t* mw = d.mask + (size_t)i * d.mw;
    for (int w = threadIdx.x; w < d.mw; w += blockDim.x) mw[w] = 0u;
    nf = __syncthreads_or(nf);
    double sums[4] = {ss, (double)eh + (double)el, (double)th + (double)tl, 0.0};
    __shared__ double part[32];
    block_sum4_d(sums, part);
    __syncthreads();
    const double bb = part[0];
    double ee = part[1], tt = part[2];
    if (!(bb >= 1e-20 && bb <= 1e30)) {
        // squares outside FP32's range (or no number at all): the same sums in FP64
        double s2[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const double fq = (double)__bfloat162float(__float2bfloat16_rn(b[k])), e = (double)b[k] - fq;
            s2[0] += e * e;
            s2[1] += fq * fq;
        }
        block_sum4_d(s2, red);
        ee = red[0];  // (used by thread 0)
        tt = red[1];
    }
    if (threadIdx.x == 0) {
        d.r16e[i] = __double2float_ru(sqrt(ee) * (1.0 + 1e-6));
        d.r16t[i] = __double2float_ru(sqrt(tt) * (1.0 + 1e-6));
    }
    if (threadIdx.x == 0) {
        const float lam = d.lam[i];
        const bool bad = nf || !(lam >= 0.f) || !isfinite(lam);  // lambda = 0: least squares
        d.state[i] = bad ? ST_DONE : ST_GROW;
        d.sstatus[i] = bad ? MPL_SIG_NONFINITE : MPL_SIG_MAX_OUTER;
        d.ssize[i] = 0;
        d.snew[i] = 0;
        d.finalized[i] = 1;  // x = 0 and xi = b are exact
        d.outer[i] = 0;
        d.inner[i] = 0;
        d.finishes[i] = 0;
        d.fails[i] = 0;
        d.nnz[i] = 0;
        d.res_tick[i] = 0;  // (a solve that stopped on an error may have left a count)
        d.rnorm[i] = __double2float_ru(sqrt(bb)) * (1.f + 1e-6f);
        if (d.pos) d.pos[i] = i;
        if (d.bnorm) { d.bnorm[i] = d.rnorm[i]; d.xl1[i] = 0.f; }
        if (d.explore) d.explore[i] = 0;
        if (i == 0 && d.ovf_cnt) { d.ovf_cnt->act_n[0] = 0; d.ovf_cnt->act_n[1] = 0; }
        if (d.early) { d.early[i] = 0; d.f0[i] = (float)(0.5 * bb); }
        d.eps[i] = d.eps_in;
        d.obj[i] = 0.5 * bb;
        d.rr[i] = bb;
        d.rb[i] = bb;
        d.kkt_in[i] = 0.0;
        d.kkt_out[i] = 0.0;
        d.ginf[i] = 0.0;
        d.act[0][i] = i;
        if (i == 0) {
            d.cnt->act_n[0] = d.p;
            d.cnt->act_n[1] = 0;
            d.cnt->grow_n = d.cnt->fin_n = d.cnt->apg_n = 0;
            d.cnt->apg_head = d.cnt->apg_head2 = d.cnt->apg_head3 = 0;
            d.cnt->err = 0;
            d.cnt->sel_fallback = 0;
            d.cnt->cols = 0ull;
            d.cnt->fin_flops = 0ull;
            d.cnt->qcols = 0ull;
            d.cnt->sel_done = 0;
            d.cnt->bounds_site = 0;
            d.cnt->apg_elems = d.cnt->apg_gl_elems = 0ull;
            for (int q = 0; q < FIN_SLOTS; ++q) d.cnt->fin_par[q] = d.cnt->reent_n[q] = 0;
            d.cnt->merge_done = 0;
            d.cnt->iters = 0u;
            d.cnt->res_bytes = d.cnt->gram_bytes = d.cnt->fin_bytes = 0ull;
        }
    }
}

// ------------------------------------------------------------------ gram
// G[a][b] for a in [0, s), b in [s0, s) (mirrored): every entry one FMA chain over k ascending, the order
// of the FP32 GEMM that builds Q, so that the Gram block gathered from Q is the same bits.
// Tile BM rows (atoms of S) x BN columns (new atoms; their h = a^T b comes with the selection's
// re-score), TR x TC entries per thread; K slices of BK staged by cp.async in a ring of ST, so that
// ST - 1 slices are in flight while one is consumed.  A thread's columns are NX apart, so a narrow
// pass (q - b0 columns) runs with as many of them as it fills; a warp whose rows are all past s
// only loads.  VEC: rows are 16-byte aligned (n % 4 == 0), else copied word by word.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// One slice's products for the first NV of a thread's columns.
template <int NV, int NX, int TR, int TC, int BK>
__device__ __forceinline__ void gram_slice(const float* Ar, const float* Bt, float (&acc)[TR][TC]) {
    constexpr int PAD = BK + 4;
#pragma unroll
    for (int k = 0; k < BK; k += 4) {
        float4 x[TR];
#pragma unroll
        for (int u = 0; u < TR; ++u) x[u] = *reinterpret_cast<const float4*>(Ar + u * PAD + k);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const float4 y = *reinterpret_cast<const float4*>(Bt + v * NX * PAD + k);
#pragma unroll
            for (int u = 0; u < TR; ++u) {
                acc[u][v] = fmaf(x[u].x, y.x, acc[u][v]);
                acc[u][v] = fmaf(x[u].y, y.y, acc[u][v]);
                acc[u][v] = fmaf(x[u].z, y.z, acc[u][v]);
                acc[u][v] = fmaf(x[u].w, y.w, acc[u][v]);
            }
        }
    }
}

template <int BM, int BN, int TR, int TC, int BK, int ST, bool VEC>
__global__ void __launch_bounds__((BM / TR) * (BN / TC)) k_gram(Dev d) {
    pdl_enter();
    constexpr int NT = (BM / TR) * (BN / TC);
    constexpr int NX = BN / TC;                  // threads along the columns
    constexpr int PAD = BK + 4;
    constexpr int CHUNKS = (BM + BN) * (BK / 4);  // 4-entry chunks per slice
    constexpr int PER = CHUNKS / NT;
    static_assert(CHUNKS % NT == 0 && 32 % NX == 0 && TC <= 4, "whole chunks per thread, whole rows per warp");
    const int g = blockIdx.x;
    if (g >= d.cnt->grow_n) return;
    const int i = d.list_grow[g];
    const int s = d.ssize[i], q = d.snew[i], s0 = s - q;
    const int a0 = blockIdx.y * BM;
    if (a0 >= s || q == 0) return;  // q == 0: a refine pass, the block is complete
    if (s > (int)gridDim.y * BM) {  // (above the host's bound, which sized the grid)
        if (threadIdx.x == 0) atomicCAS(&d.cnt->err, 0, (int)DERR_SHAPE);
        return;
    }
    const int n = d.n, smax = d.smax;
    if (blockIdx.y == 0 && threadIdx.x == 0)  // s atom columns read, 2 s q of G written
        atomicAdd(&d.cnt->gram_bytes, 4ull * n * s + 8ull * s * q);
    const int* Si = d.S + (size_t)i * smax;
    float* Gi = d.G + (size_t)i * smax * smax;
    extern __shared__ __align__(16) float gsm[];  // [ST][BM + BN][PAD]
    const int tid = threadIdx.x;
    const int ty = tid / NX, tx = tid % NX;
    const bool rows = a0 + ((tid & ~31) / NX) * TR < s;  // (the same in the whole warp)
    const int nsl = (n + BK - 1) / BK;
    for (int b0 = 0; b0 < q; b0 += BN) {
        // source rows of this thread's chunks (c = tid + NT e), fixed for the column chunk
        const float* src[PER];
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int rr = (tid + NT * e) / (BK / 4);
            const int r = rr < BM ? a0 + rr : s0 + b0 + rr - BM;  // position in S
            src[e] = r < s ? d.A32 + (size_t)Si[r] * n : nullptr;
        }
        auto issue = [&](int sl) {
            float* st = gsm + (size_t)(sl % ST) * (BM + BN) * PAD;
#pragma unroll
            for (int e = 0; e < PER; ++e) {
                const int c = tid + NT * e;
                const int kc = (c % (BK / 4)) * 4, k = sl * BK + kc;
                float* dst = st + (c / (BK / 4)) * PAD + kc;
                if (VEC) {
                    const bool ok = src[e] != nullptr && k < n;
                    cp_async16(dst, ok ? src[e] + k : d.A32, ok ? 16 : 0);
                } else {
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const bool ok = src[e] != nullptr && k + w < n;
                        cp_async4(dst + w, ok ? src[e] + k + w : d.A32, ok ? 4 : 0);
                    }
                }
            }
        };
#pragma unroll
        for (int sl = 0; sl < ST - 1; ++sl) {
            if (sl < nsl) issue(sl);
            cp_async_commit();
        }
        float acc[TR][TC];
#pragma unroll
        for (int u = 0; u < TR; ++u)
#pragma unroll
            for (int v = 0; v < TC; ++v) acc[u][v] = 0.f;
        const int nv = rows ? min(TC, (q - b0 + NX - 1) / NX) : 0;
        for (int sl = 0; sl < nsl; ++sl) {
            cp_async_wait<ST - 2>();
            __syncthreads();
            if (sl + ST - 1 < nsl) issue(sl + ST - 1);
            cp_async_commit();
            const float* st = gsm + (size_t)(sl % ST) * (BM + BN) * PAD;
            const float* Ar = st + ty * TR * PAD;
            const float* Bt = st + (BM + tx) * PAD;
            switch (nv) {
                case 0: break;
                case 1: gram_slice<1, NX, TR, TC, BK>(Ar, Bt, acc); break;
                case 2: gram_slice<2, NX, TR, TC, BK>(Ar, Bt, acc); break;
                case 3: gram_slice<TC < 3 ? TC : 3, NX, TR, TC, BK>(Ar, Bt, acc); break;
                default: gram_slice<TC, NX, TR, TC, BK>(Ar, Bt, acc); break;
            }
        }
        cp_async_wait<0>();
        __syncthreads();  // the ring is reused by the next column chunk
#pragma unroll
        for (int u = 0; u < TR; ++u) {
            const int a = a0 + ty * TR + u;
            if (a >= s) continue;
#pragma unroll
            for (int v = 0; v < TC; ++v) {
                const int bb = b0 + tx + NX * v;
                if (bb >= q) continue;
                const int col = s0 + bb;
                Gi[(size_t)a * smax + col] = acc[u][v];
                Gi[(size_t)col * smax + a] = acc[u][v];
            }
        }
    }
}

// ------------------------------------------------------------------ APG
// Blocks of more than APG_REG_S atoms: in shared memory when s <= gcap (<= APG_SMEM_S), else streamed
// from global memory (L2).  Dynamic shared memory: [G gcap^2 | 6 vectors of vcap].

__device__ __forceinline__ float gram_mv(const float* __restrict__ G, int ld, int s, const float* __restrict__ x,
                                         float* __restrict__ y, const float* h = nullptr, float lam = 0.f) {
    float part = 0.f;
    // y = G x, one row per thread; G symmetric so column r is read with unit
    // stride across threads (conflict-free in shared memory, coalesced in global)
    for (int r = threadIdx.x; r < s; r += blockDim.x) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        int c = 0;
        for (; c + 3 < s; c += 4) {
            a0 = fmaf(G[(size_t)(c + 0) * ld + r], x[c + 0], a0);
            a1 = fmaf(G[(size_t)(c + 1) * ld + r], x[c + 1], a1);
            a2 = fmaf(G[(size_t)(c + 2) * ld + r], x[c + 2], a2);
            a3 = fmaf(G[(size_t)(c + 3) * ld + r], x[c + 3], a3);
        }
        for (; c < s; ++c) a0 = fmaf(G[(size_t)c * ld + r], x[c], a0);
        const float yr = (a0 + a1) + (a2 + a3);
        y[r] = yr;
        if (h) part += lam * fabsf(x[r]) + x[r] * (0.5f * yr - h[r]);
    }
    return part;
}

// y = G x for a block in global memory (leading dimension ld, row r = column r by
// symmetry).  Lane l of a warp owns the float4 slices c = 4 l + 128 u (u < U = ceil(s / 128))
// of a row and sums them in order of u, then a fixed butterfly combines the lanes; a warp
// takes RW rows per round and issues all RW x U slice loads before the first product (up to
// 16 per lane in flight: the streamed products are latency-bound).  x is zero from s up to
// the next multiple of 4.  With h != nullptr lane 0 also returns its rows' share of the
// restricted objective, lambda |x_r| + x_r (y_r / 2 - h_r).
template <int U, int RW>
__device__ __forceinline__ float gram_mv_stream_vec(const float* __restrict__ G, int ld, int s,
                                                    const float* __restrict__ x, float* __restrict__ y,
                                                    const float* h, float lam) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float part = 0.f;
    for (int r = RW * warp; r < s; r += RW * nw) {
        float4 g[RW][U];
#pragma unroll
        for (int w = 0; w < RW; ++w) {
            const float* gr = G + (size_t)min(r + w, s - 1) * ld;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = 4 * lane + 128 * u;
                g[w][u] = c < s ? __ldg(reinterpret_cast<const float4*>(gr + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        float acc[RW];
#pragma unroll
        for (int w = 0; w < RW; ++w) acc[w] = 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = 4 * lane + 128 * u;
            if (c < s) {
                const float4 xv = *reinterpret_cast<const float4*>(x + c);
#pragma unroll
                for (int w = 0; w < RW; ++w) {
                    acc[w] = fmaf(g[w][u].x, xv.x, acc[w]); acc[w] = fmaf(g[w][u].y, xv.y, acc[w]);
                    acc[w] = fmaf(g[w][u].z, xv.z, acc[w]); acc[w] = fmaf(g[w][u].w, xv.w, acc[w]);
                }
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
#pragma unroll
            for (int w = 0; w < RW; ++w) acc[w] += __shfl_xor_sync(0xffffffffu, acc[w], o);
        }
        if (lane == 0) {
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                if (r + w < s) {
                    y[r + w] = acc[w];
                    if (h) part += lam * fabsf(x[r + w]) + x[r + w] * (0.5f * acc[w] - h[r + w]);
                }
            }
        }
    }
    return part;
}

// The same product with scalar loads (ld not a multiple of 4): a warp per pair of rows.
__device__ __forceinline__ float gram_mv_stream_scalar(const float* __restrict__ G, int ld, int s,
                                                       const float* __restrict__ x, float* __restrict__ y,
                                                       const float* h, float lam) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float part = 0.f;
    for (int r = 2 * warp; r < s; r += 2 * nw) {
        const int rb = r + 1 < s ? r + 1 : r;
        const float* ga = G + (size_t)r * ld;
        const float* gb = G + (size_t)rb * ld;
        float sa = 0.f, sb = 0.f;
        for (int c0 = 4 * lane; c0 < s; c0 += 512) {
            float4 a4[4], b4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 128 * u;
                if (c < s) {
                    a4[u] = make_float4(__ldg(ga + c), c + 1 < s ? __ldg(ga + c + 1) : 0.f,
                                        c + 2 < s ? __ldg(ga + c + 2) : 0.f, c + 3 < s ? __ldg(ga + c + 3) : 0.f);
                    b4[u] = make_float4(__ldg(gb + c), c + 1 < s ? __ldg(gb + c + 1) : 0.f,
                                        c + 2 < s ? __ldg(gb + c + 2) : 0.f, c + 3 < s ? __ldg(gb + c + 3) : 0.f);
                } else {
                    a4[u] = b4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 128 * u;
                if (c < s) {
                    const float4 xv = *reinterpret_cast<const float4*>(x + c);
                    sa = fmaf(a4[u].x, xv.x, sa); sa = fmaf(a4[u].y, xv.y, sa);
                    sa = fmaf(a4[u].z, xv.z, sa); sa = fmaf(a4[u].w, xv.w, sa);
                    sb = fmaf(b4[u].x, xv.x, sb); sb = fmaf(b4[u].y, xv.y, sb);
                    sb = fmaf(b4[u].z, xv.z, sb); sb = fmaf(b4[u].w, xv.w, sb);
                }
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
            sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
        if (lane == 0) {
            y[r] = sa;
            if (h) part += lam * fabsf(x[r]) + x[r] * (0.5f * sa - h[r]);
            if (r + 1 < s) {
                y[r + 1] = sb;
                if (h) part += lam * fabsf(x[r + 1]) + x[r + 1] * (0.5f * sb - h[r + 1]);
            }
        }
    }
    return part;
}

__device__ __noinline__ float gram_mv_stream(const float* __restrict__ G, int ld, int s, const float* __restrict__ x,
                                             float* __restrict__ y, const float* h = nullptr, float lam = 0.f) {
    if ((ld & 3) != 0) return gram_mv_stream_scalar(G, ld, s, x, y, h, lam);
    switch ((s + 127) >> 7) {
        case 0:
        case 1: return gram_mv_stream_vec<1, 8>(G, ld, s, x, y, h, lam);
        case 2: return gram_mv_stream_vec<2, 8>(G, ld, s, x, y, h, lam);
        case 3: return gram_mv_stream_vec<3, 4>(G, ld, s, x, y, h, lam);
        case 4: return gram_mv_stream_vec<4, 4>(G, ld, s, x, y, h, lam);
        case 5: return gram_mv_stream_vec<5, 2>(G, ld, s, x, y, h, lam);
        case 6: return gram_mv_stream_vec<6, 2>(G, ld, s, x, y, h, lam);
        case 7: return gram_mv_stream_vec<7, 2>(G, ld, s, x, y, h, lam);
        default: return gram_mv_stream_vec<8, 2>(G, ld, s, x, y, h, lam);
    }
}

struct ApgVec {
    float *u, *up, *Gu, *Gup, *h, *v;
    float red[96];
    int item;
};

// Three block sums in one pass (two barriers); every thread gets the totals.
__device__ __forceinline__ void block_sum3(float& a, float& b, float& c, float* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    __syncthreads();
    if (lane == 0) { red[warp] = a; red[32 + warp] = b; red[64 + warp] = c; }
    __syncthreads();
    a = b = c = 0.f;
    for (int w = 0; w < nw; ++w) { a += red[w]; b += red[32 + w]; c += red[64 + w]; }
}

// STREAM: the APG_GLOBAL launch (every block streamed from global memory by warp rows);
// otherwise blocks in shared memory.
template <bool STREAM>
__global__ void __launch_bounds__(APG_THREADS) k_apg(Dev d, int vcap, int gcap, int cls) {
    pdl_enter();
    extern __shared__ __align__(16) float gsm[];
    __shared__ ApgVec sh;
    const int tid = threadIdx.x;
    const int smax = d.smax;
    if (tid == 0) {
        float* base = gsm + (size_t)gcap * gcap;
        sh.u = base; sh.up = base + vcap; sh.Gu = base + 2 * vcap;
        sh.Gup = base + 3 * vcap; sh.h = base + 4 * vcap; sh.v = base + 5 * vcap;
    }
    int* head = cls == APG_GLOBAL ? &d.cnt->apg_head2 : &d.cnt->apg_head3;
    for (;;) {
        if (tid == 0) sh.item = atomicAdd(head, 1);
        __syncthreads();
        const int it = sh.item;
        if (it >= d.cnt->apg_n) break;
        const int i = d.list_apg[it];
        const int s = d.ssize[i];
        // a class launch takes only its own signals (the other launch takes the rest)
        if (cls == APG_SMEM ? (s <= APG_REG_S || s > gcap) : s <= APG_SMEM_S) {
            __syncthreads();  // every thread has read sh.item before thread 0 takes the next
            continue;
        }
        AT_BEGIN
        const float lam = d.lam[i];
        const float eps = d.eps[i];
        const float* Gg = d.G + (size_t)i * smax * smax;
        if (s > vcap) {  // cannot happen with a correct bound; refuse rather than overrun
            if (tid == 0) atomicCAS(&d.cnt->err, 0, (int)DERR_SHAPE);
            __syncthreads();
            continue;
        }
        const float* G = STREAM ? Gg : gsm;
        const int ld = STREAM ? smax : s;
        if (!STREAM) {
            // eight loads in flight per thread before their stores
            for (int e0 = tid; e0 < s * s; e0 += 8 * blockDim.x) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int e = e0 + u * blockDim.x;
                    if (e < s * s) {
                        const int r = e / s, c = e - r * s;
                        v[u] = __ldg(Gg + (size_t)r * smax + c);
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int e = e0 + u * blockDim.x;
                    if (e < s * s) {
                        const int r = e / s, c = e - r * s;
                        gsm[(size_t)r * ld + c] = v[u];
                    }
                }
            }
        }
        // the block's matrix-vector product: a row per thread in shared memory, warp rows streamed
        // as float4 slices from global memory
        auto mv = [&](const float* x, float* y) {
            if constexpr (STREAM) gram_mv_stream(G, ld, s, x, y);
            else gram_mv(G, ld, s, x, y);
        };
        // y = G x and this thread's share of the restricted objective at x
        auto mvF = [&](const float* x, float* y) -> float {
            if constexpr (STREAM) return gram_mv_stream(G, ld, s, x, y, sh.h, lam);
            else return gram_mv(G, ld, s, x, y, sh.h, lam);
        };
        float* xi = d.xS + (size_t)i * smax;
        float* ritz = d.ritz + (size_t)i * smax;
        const int prev = s - d.snew[i];  // ritz vector valid for the first `prev` entries
        // (entries from s up to the next multiple of 4 are zero: the streamed product reads
        // its operand as float4 slices)
        const int s4 = (s + 3) & ~3;
        if (MPL_OOB(s4 > vcap || s > smax, 201)) { __syncthreads(); continue; }
        for (int r = tid; r < s4; r += blockDim.x) {
            const bool in = r < s;
            sh.u[r] = in ? xi[r] : 0.f;
            sh.h[r] = in ? d.h[(size_t)i * smax + r] : 0.f;
            sh.v[r] = !in ? 0.f : ((r < prev && d.outer[i] > 1) ? ritz[r] : 1.f);
            sh.up[r] = 0.f;
            sh.Gu[r] = 0.f;
            sh.Gup[r] = 0.f;
        }
        __syncthreads();
        AT_ADD(0);
        // Step size: power iteration for lambda_max(G) (warm started), L = 1.05 theta.  The
        // iterate ping-pongs between two vectors and is normalised every fourth step (and
        // at the last, where the Rayleigh quotient is taken): growth over four steps stays
        // far inside FP32 range for |S| <= 1024.
        float theta = 1.f;
        const int npow = !(lam > 0.f) ? 0 : ((prev > 0 && d.outer[i] > 1) ? 3 : 8);  // CG needs no step size
        float* pv = sh.v;
        float* pw = sh.Gu;
        for (int pi = 0; pi < npow; ++pi) {
            mv(pv, pw);
            __syncthreads();
            if ((pi & 3) == 3 || pi == npow - 1) {
                float vv = 0.f, vg = 0.f, gg = 0.f;
                for (int r = tid; r < s; r += blockDim.x) {
                    vv += pv[r] * pv[r];
                    vg += pv[r] * pw[r];
                    gg += pw[r] * pw[r];
                }
                block_sum3(vv, vg, gg, sh.red);
                theta = vv > 0.f ? vg / vv : 1.f;
                const float inv = gg > 0.f ? rsqrtf(gg) : 0.f;
                for (int r = tid; r < s; r += blockDim.x) pv[r] = pw[r] * inv;
                __syncthreads();
            } else {
                float* t = pv;
                pv = pw;
                pw = t;
            }
        }
        for (int r = tid; r < s; r += blockDim.x) ritz[r] = pv[r];
        __syncthreads();  // pv may be the Gu buffer, which the next product overwrites
        AT_ADD(1);
        float L = fmaxf(1.05f * theta, 1e-30f);

        // F(u) and G u at the warm start
        mv(sh.u, sh.Gu);
        __syncthreads();
        float part = 0.f;
        for (int r = tid; r < s; r += blockDim.x) {
            sh.up[r] = sh.u[r];
            sh.Gup[r] = sh.Gu[r];
            part += lam * fabsf(sh.u[r]) + sh.u[r] * (0.5f * sh.Gu[r] - sh.h[r]);
        }
        float F = block_sum(part, sh.red);
        const float F0 = F;
        float t = 1.f, beta = 0.f;
        int iters = 0, restarts_in_row = 0;
        if (!(lam > 0.f)) {
            // lambda = 0: the restricted problem is least squares G u = h, solved by
            // conjugate gradients (the paper's CGD rule for lambda = 0) from the warm start;
            // r in up, the direction in Gup, G times the direction in v
            float rr = 0.f, hh = 0.f;
            for (int r = tid; r < s; r += blockDim.x) {
                const float res = sh.h[r] - sh.Gu[r];
                sh.up[r] = res;
                sh.Gup[r] = res;
                rr += res * res;
                hh += sh.h[r] * sh.h[r];
            }
            float z0 = 0.f;
            block_sum3(rr, hh, z0, sh.red);
            const float stop2 = eps * eps * hh;
            const int cg_max = min(d.inner_max, 4 * s + 20);
            for (int k = 0; k < cg_max && rr > stop2; ++k) {
                mv(sh.Gup, sh.v);
                __syncthreads();
                float pgp = 0.f;
                for (int r = tid; r < s; r += blockDim.x) pgp += sh.Gup[r] * sh.v[r];
                pgp = block_sum(pgp, sh.red);
                if (!(pgp > 0.f)) break;
                const float alpha = rr / pgp;
                float rn = 0.f;
                for (int r = tid; r < s; r += blockDim.x) {
                    sh.u[r] += alpha * sh.Gup[r];
                    sh.Gu[r] += alpha * sh.v[r];
                    const float res = sh.up[r] - alpha * sh.v[r];
                    sh.up[r] = res;
                    rn += res * res;
                }
                rn = block_sum(rn, sh.red);
                const float bcg = rn / rr;
                rr = rn;
                for (int r = tid; r < s; r += blockDim.x) sh.Gup[r] = sh.up[r] + bcg * sh.Gup[r];
                __syncthreads();
                ++iters;
            }
            part = 0.f;
            for (int r = tid; r < s; r += blockDim.x) part += sh.u[r] * (0.5f * sh.Gu[r] - sh.h[r]);
            F = block_sum(part, sh.red);
        }
        for (int k = 0; lam > 0.f && k < d.inner_max; ++k) {
            // extrapolate, prox-gradient step (the one matvec is G u of the new point)
            const float invL = 1.f / L, thr = lam * invL;
            for (int r = tid; r < s; r += blockDim.x) {
                const float y = sh.u[r] + beta * (sh.u[r] - sh.up[r]);
                const float gy = sh.Gu[r] + beta * (sh.Gu[r] - sh.Gup[r]) - sh.h[r];
                const float z = softf(y - gy * invL, thr);
                sh.up[r] = sh.u[r];
                sh.Gup[r] = sh.Gu[r];
                sh.u[r] = z;
            }
            __syncthreads();
            part = mvF(sh.u, sh.Gu);  // the block sum's barrier also publishes Gu
            // (the barrier above already follows every read of red by the last block sum)
            const float Fn = block_sum_after_barrier(part, sh.red);
            ++iters;
            if (Fn > F) {
                // function-value restart: back to the previous point, momentum off;
                // a plain step that still increases F means L was too small
                const bool genuine = (Fn - F) > 1e-4f * fmaxf(F0 - F, 1e-30f);
                if (beta == 0.f && genuine) L *= 2.f;
                for (int r = tid; r < s; r += blockDim.x) { sh.u[r] = sh.up[r]; sh.Gu[r] = sh.Gup[r]; }
                __syncthreads();
                beta = 0.f;
                t = 1.f;
                if (++restarts_in_row >= 3) break;  // stalled at FP32 resolution
                continue;
            }
            restarts_in_row = 0;
            const float dec = F - Fn, tot = F0 - Fn;
            F = Fn;
            // relative-decrease stop of eq. (inner)
            if (tot <= 0.f ? dec <= 0.f : dec <= eps * tot) break;
            const float tn = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
            beta = (t - 1.f) / tn;
            t = tn;
        }
        AT_ADD(2);
        for (int r = tid; r < s; r += blockDim.x) xi[r] = sh.u[r];
        AT_ADD(3);
        AT_CNT(4, 1);
        AT_CNT(5, iters);
        if (tid == 0) {
            d.inner[i] += iters;
            // products with the block: the power steps, G u at the warm start, one per iteration
            const unsigned long long ss = (unsigned long long)s * (unsigned long long)s;
            const unsigned long long nmv = (unsigned long long)(npow + 1 + iters);
            atomicAdd(&d.cnt->apg_elems, ss * nmv);
            atomicAdd(&d.cnt->apg_gl_elems, STREAM ? ss * nmv : ss);
            // early stopping, eq. (stop_con): decrease of f over this outer iteration's
            // master problem (F0 is f at x^{t-1}, new entries at zero)
            if (d.early && d.stop_eps >= 0.f && d.snew[i] > 0 &&
                F0 - F <= d.stop_eps * fabsf((float)d.rho * d.f0[i]))
                d.early[i] = 1;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ APG, blocks in registers
// The same master problem for blocks of at most APG_REG_S atoms, with the Gram block in registers.
// With the block in shared memory an iteration took 3300 cycles at 85 atoms: every product reads
// the whole block from shared memory (one chain of dependent loads and FMAs per row), and
// so do its five vectors.  Here thread (row r, half h) keeps NC entries of row r (the float4
// column groups 8 k + 4 h) and row r's entries of the vectors; only the product's operand
// goes through shared memory, where a warp reads it as broadcast float4, and an iteration
// has two barriers.  WARP: blocks of at most 32 atoms, a row per lane and a signal per
// warp, no block barrier at all.  Face-shaped batch (2048 signals, 85 atoms and 556 iterations a
// signal): 8.1 -> 3.0 ms in master problems; 256 signals on 1024 x 8192: 0.10 -> 0.06 ms.
// Rows and columns past s are zero, so they add nothing to any sum.
template <int NC, bool WARP>
struct ApgReg {
    static constexpr int ROWS = WARP ? 32 : 2 * NC;
    static constexpr int NT = WARP ? 32 : 2 * ROWS;  // threads per signal
    static constexpr int NWARP = NT / 32;
};
constexpr int APG_WARPS = 4;  // signals per CTA of the warp variant

// Shared memory of one signal's group of threads (x is read as float4: aligned, also as an array
// element).
struct alignas(16) ApgRegShared {
    float x[APG_REG_S];
    float red[3][8];
    int item;
};

static_assert(sizeof(ApgRegShared) % 16 == 0 && offsetof(ApgRegShared, x) == 0, "float4 reads of x");

template <int NC, bool WARP>
__device__ void apg_reg_signal(const Dev& d, int i, int tid, ApgRegShared& sh) {
    using T = ApgReg<NC, WARP>;
    const int lane = tid & 31, warp = tid >> 5;
    const int r = WARP ? tid : tid >> 1, h = WARP ? 0 : (tid & 1);
    constexpr int CG = WARP ? 4 : 8;  // columns from one of this thread's float4 groups to its next
    const int s = d.ssize[i], smax = d.smax;
    const float lam = d.lam[i], eps = d.eps[i];
    const float* Gg = d.G + (size_t)i * smax * smax;
    const bool own = r < s;          // (both halves of a row hold its vector entries)
    const bool lead = own && h == 0; // ... and the first one counts them
    auto sync = [&]() {
        if (WARP) __syncwarp();
        else __syncthreads();
    };
    // sums over the rows, the same in every thread; a barrier separates two calls' use of red
    auto sum3 = [&](float& a, float& b, float& c) {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (WARP) return;
        if (lane == 0) { sh.red[0][warp] = a; sh.red[1][warp] = b; sh.red[2][warp] = c; }
        __syncthreads();
        a = b = c = 0.f;
#pragma unroll
        for (int w = 0; w < T::NWARP; ++w) { a += sh.red[0][w]; b += sh.red[1][w]; c += sh.red[2][w]; }
    };
    auto sum = [&](float a) -> float {
#pragma unroll
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (WARP) return a;
        if (lane == 0) sh.red[0][warp] = a;
        __syncthreads();
        a = 0.f;
#pragma unroll
        for (int w = 0; w < T::NWARP; ++w) a += sh.red[0][w];
        return a;
    };
    // the block: every load in flight at once
    float4 g[NC / 4];
    const float* grow = Gg + (size_t)(own ? r : 0) * smax;
    if ((smax & 3) == 0) {
#pragma unroll
        for (int k = 0; k < NC / 4; ++k) {
            const int c = CG * k + 4 * h;
            g[k] = own && c < s ? __ldg(reinterpret_cast<const float4*>(grow + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < NC / 4; ++k) {  // (entries past s are left over from larger sets)
            const int c = CG * k + 4 * h;
            if (c + 1 >= s) g[k].y = 0.f;
            if (c + 2 >= s) g[k].z = 0.f;
            if (c + 3 >= s) g[k].w = 0.f;
        }
    } else {
#pragma unroll
        for (int k = 0; k < NC / 4; ++k) {
            const int c = CG * k + 4 * h;
            g[k].x = own && c < s ? __ldg(grow + c) : 0.f;
            g[k].y = own && c + 1 < s ? __ldg(grow + c + 1) : 0.f;
            g[k].z = own && c + 2 < s ? __ldg(grow + c + 2) : 0.f;
            g[k].w = own && c + 3 < s ? __ldg(grow + c + 3) : 0.f;
        }
    }
    // (G x)_r of the vector whose entries the rows pass; ends without a barrier
    auto mv = [&](float x) -> float {
        if (h == 0) sh.x[r] = x;
        sync();
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
        for (int k = 0; k < NC / 4; ++k) {
            const float4 v = *reinterpret_cast<const float4*>(&sh.x[CG * k + 4 * h]);
            a0 = fmaf(g[k].x, v.x, a0);
            a1 = fmaf(g[k].y, v.y, a1);
            a2 = fmaf(g[k].z, v.z, a2);
            a3 = fmaf(g[k].w, v.w, a3);
        }
        float y = (a0 + a1) + (a2 + a3);
        if (!WARP) y += __shfl_xor_sync(0xffffffffu, y, 1);
        return y;
    };
    float* xi = d.xS + (size_t)i * smax;
    float* ritz = d.ritz + (size_t)i * smax;
    const int prev = s - d.snew[i];  // ritz vector valid for the first `prev` entries
    const bool warm = prev > 0 && d.outer[i] > 1;
    float u = own ? xi[r] : 0.f;
    const float hv = own ? d.h[(size_t)i * smax + r] : 0.f;
    float pv = !own ? 0.f : (r < prev && d.outer[i] > 1 ? ritz[r] : 1.f);
    // step size: power iteration for lambda_max(G), as in k_apg
    float theta = 1.f;
    const int npow = !(lam > 0.f) ? 0 : (warm ? 3 : 8);
    for (int pi = 0; pi < npow; ++pi) {
        const float w = mv(pv);
        if ((pi & 3) == 3 || pi == npow - 1) {
            float vv = lead ? pv * pv : 0.f, vg = lead ? pv * w : 0.f, gg = lead ? w * w : 0.f;
            sum3(vv, vg, gg);
            theta = vv > 0.f ? vg / vv : 1.f;
            pv = w * (gg > 0.f ? rsqrtf(gg) : 0.f);
        } else {
            pv = w;
        }
        sync();
    }
    if (lead) ritz[r] = pv;
    float L = fmaxf(1.05f * theta, 1e-30f);
    // F(u) and G u at the warm start
    float Gu = mv(u);
    float up = u, Gup = Gu;
    float F = sum(lead ? lam * fabsf(u) + u * (0.5f * Gu - hv) : 0.f);
    const float F0 = F;
    float t = 1.f, beta = 0.f;
    int iters = 0, restarts_in_row = 0;
    if (!(lam > 0.f)) {
        // lambda = 0: least squares by conjugate gradients from the warm start
        float res = own ? hv - Gu : 0.f, dir = res;
        sync();
        float rr = lead ? res * res : 0.f, hh = lead ? hv * hv : 0.f, z0 = 0.f;
        sum3(rr, hh, z0);
        const float stop2 = eps * eps * hh;
        const int cg_max = min(d.inner_max, 4 * s + 20);
        for (int k = 0; k < cg_max && rr > stop2; ++k) {
            sync();
            const float q = mv(dir);
            const float pgp = sum(lead ? dir * q : 0.f);
            if (!(pgp > 0.f)) break;
            const float alpha = rr / pgp;
            u += alpha * dir;
            Gu += alpha * q;
            res -= alpha * q;
            sync();
            const float rn = sum(lead ? res * res : 0.f);
            const float bcg = rn / rr;
            rr = rn;
            dir = res + bcg * dir;
            ++iters;
        }
        sync();
        F = sum(lead ? u * (0.5f * Gu - hv) : 0.f);
    }
    for (int k = 0; lam > 0.f && k < d.inner_max; ++k) {
        // extrapolate, prox-gradient step (the one product is G u of the new point)
        const float invL = 1.f / L;
        const float y = u + beta * (u - up);
        const float gy = Gu + beta * (Gu - Gup) - hv;
        const float z = own ? softf(y - gy * invL, lam * invL) : 0.f;
        const float u0 = u, Gu0 = Gu;
        if (WARP) __syncwarp();  // (in a block the last sum's barrier follows every read of x)
        const float Gz = mv(z);
        const float Fn = sum(lead ? lam * fabsf(z) + z * (0.5f * Gz - hv) : 0.f);
        ++iters;
        if (Fn > F) {
            // function-value restart: stay at the current point, momentum off; a plain step that
            // still increases F means L was too small
            const bool genuine = (Fn - F) > 1e-4f * fmaxf(F0 - F, 1e-30f);
            if (beta == 0.f && genuine) L *= 2.f;
            up = u0;
            Gup = Gu0;
            beta = 0.f;
            t = 1.f;
            if (++restarts_in_row >= 3) break;  // stalled at FP32 resolution
            continue;
        }
        up = u0;
        Gup = Gu0;
        u = z;
        Gu = Gz;
        restarts_in_row = 0;
        const float dec = F - Fn, tot = F0 - Fn;
        F = Fn;
        // relative-decrease stop of eq. (inner)
        if (tot <= 0.f ? dec <= 0.f : dec <= eps * tot) break;
        const float tn = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
        beta = (t - 1.f) / tn;
        t = tn;
    }
    if (lead) xi[r] = u;
    if (tid == 0) {
        d.inner[i] += iters;
        const unsigned long long ss = (unsigned long long)s * (unsigned long long)s;
        atomicAdd(&d.cnt->apg_elems, ss * (unsigned long long)(npow + 1 + iters));
        atomicAdd(&d.cnt->apg_gl_elems, ss);
        // early stopping, eq. (stop_con)
        if (d.early && d.stop_eps >= 0.f && d.snew[i] > 0 &&
            F0 - F <= d.stop_eps * fabsf((float)d.rho * d.f0[i]))
            d.early[i] = 1;
    }
}

// Persistent CTAs (or warps) over the master-problem list; signals with more than NC's rows are left
// to the other launches of the iteration.  There are none up to a bound vcap of APG_REG_S: a
// set above the bound is an error, as in k_apg.
template <int NC, bool WARP, int MINB>
__global__ void __launch_bounds__(WARP ? 32 * APG_WARPS : 4 * NC, MINB) k_apg_reg(Dev d, int vcap) {
    pdl_enter();
    __shared__ __align__(16) ApgRegShared sha[WARP ? APG_WARPS : 1];
    ApgRegShared& sh = sha[WARP ? threadIdx.x >> 5 : 0];
    const int tid = WARP ? threadIdx.x & 31 : threadIdx.x;
    for (;;) {
        if (tid == 0) sh.item = atomicAdd(&d.cnt->apg_head, 1);
        if (WARP) __syncwarp();
        else __syncthreads();
        const int it = sh.item;
        if (it >= d.cnt->apg_n) break;
        const int i = d.list_apg[it];
        const int s = d.ssize[i];
        if (s <= ApgReg<NC, WARP>::ROWS) apg_reg_signal<NC, WARP>(d, i, tid, sh);
        else if (s > vcap && tid == 0) atomicCAS(&d.cnt->err, 0, (int)DERR_SHAPE);
        // every thread has read sh.item (and finished with sh) before the next one is taken
        if (WARP) __syncwarp();
        else __syncthreads();
    }
}

// ------------------------------------------------------------------ residual
// Row block y = blockIdx.y of signal position blockIdx.x: rows [RES_ROWS y, RES_ROWS (y + 1)).
// Each entry sums the atoms in order of the support, whatever the split.  The three norms
// are block sums per row block, combined in order of y by the block that finishes last (a
// ticket per signal, no waiting), so they do not depend on the order the blocks run in.
__global__ void __launch_bounds__(256) k_residual(Dev d) {
    pdl_enter();
    const int g = blockIdx.x;
    if (g >= d.cnt->apg_n) return;
    const int i = d.list_apg[g];
    const int yb = blockIdx.y, nb = gridDim.y;
    const int n = d.n, smax = d.smax, s = d.ssize[i];
    __shared__ int nzi[1024];
    __shared__ float nzv[1024];
    __shared__ int cntnz;
    __shared__ float red[96];
    if (threadIdx.x == 0) cntnz = 0;
    __syncthreads();
    const float* xi = d.xS + (size_t)i * smax;
    const int* Si = d.S + (size_t)i * smax;
    // nonzeros of x_S in append order (ordered compaction by one warp)
    if (threadIdx.x < 32) {
        int base = 0;
        for (int a0 = 0; a0 < s; a0 += 32) {
            const int a = a0 + threadIdx.x;
            const float v = a < s ? xi[a] : 0.f;
            const unsigned b = __ballot_sync(0xffffffffu, v != 0.f);
            const int off = base + __popc(b & ((1u << threadIdx.x) - 1u));
            if (v != 0.f) { nzi[off] = Si[a]; nzv[off] = v; }
            base += __popc(b);
        }
        if (threadIdx.x == 0) cntnz = base;
    }
    __syncthreads();
    const int nz = cntnz;
    if (MPL_OOB(s > 1024 || nz > 1024, 301)) return;
    if (d.Q && yb == 0) {  // ||x_S||_1 for the identity route's error band (FP32 sum, rounded up by gamma_1024)
        float l1 = 0.f;
        for (int a = threadIdx.x; a < nz; a += blockDim.x) l1 += fabsf(nzv[a]);
        const float t1 = block_sum(l1, red);
        if (threadIdx.x == 0) d.xl1[i] = t1 * (1.f + 2e-4f);
        __syncthreads();
    }
    const float* b = d.B + (size_t)i * n;
    float* r32 = d.R32 + (size_t)i * n;
    float ss = 0.f, es = 0.f, ts = 0.f;  // ||r||^2, ||r - bf(r)||^2, ||bf(r)||^2
    const bool r16 = d.R16 || d.pos;
    auto bf_terms = [&](float v) {
        const float fq = __bfloat162float(__float2bfloat16_rn(v));
        const float e = v - fq;  // exact (Sterbenz)
        es = fmaf(e, e, es);
        ts = fmaf(fq, fq, ts);
    };
    const int k_lo = yb * RES_ROWS, k_hi = min(n, k_lo + RES_ROWS);
    if ((n & 3) == 0) {
        // float4 columns, four atoms per pass with their loads issued first
        for (int k = k_lo + threadIdx.x * 4; k < k_hi; k += blockDim.x * 4) {
            float4 acc = *reinterpret_cast<const float4*>(b + k);
            int a = 0;
            for (; a + 7 < nz; a += 8) {  // eight atom columns' loads in flight, then in order
                float4 cv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    cv[u] = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a + u] * n + k));
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float vu = nzv[a + u];
                    acc.x = fmaf(-vu, cv[u].x, acc.x); acc.y = fmaf(-vu, cv[u].y, acc.y);
                    acc.z = fmaf(-vu, cv[u].z, acc.z); acc.w = fmaf(-vu, cv[u].w, acc.w);
                }
            }
            for (; a + 3 < nz; a += 4) {
                const float4 c0 = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a] * n + k));
                const float4 c1 = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a + 1] * n + k));
                const float4 c2 = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a + 2] * n + k));
                const float4 c3 = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a + 3] * n + k));
                const float v0 = nzv[a], v1 = nzv[a + 1], v2 = nzv[a + 2], v3 = nzv[a + 3];
                acc.x = fmaf(-v0, c0.x, acc.x); acc.y = fmaf(-v0, c0.y, acc.y);
                acc.z = fmaf(-v0, c0.z, acc.z); acc.w = fmaf(-v0, c0.w, acc.w);
                acc.x = fmaf(-v1, c1.x, acc.x); acc.y = fmaf(-v1, c1.y, acc.y);
                acc.z = fmaf(-v1, c1.z, acc.z); acc.w = fmaf(-v1, c1.w, acc.w);
                acc.x = fmaf(-v2, c2.x, acc.x); acc.y = fmaf(-v2, c2.y, acc.y);
                acc.z = fmaf(-v2, c2.z, acc.z); acc.w = fmaf(-v2, c2.w, acc.w);
                acc.x = fmaf(-v3, c3.x, acc.x); acc.y = fmaf(-v3, c3.y, acc.y);
                acc.z = fmaf(-v3, c3.z, acc.z); acc.w = fmaf(-v3, c3.w, acc.w);
            }
            for (; a < nz; ++a) {
                const float4 c0 = __ldg(reinterpret_cast<const float4*>(d.A32 + (size_t)nzi[a] * n + k));
                const float v0 = nzv[a];
                acc.x = fmaf(-v0, c0.x, acc.x); acc.y = fmaf(-v0, c0.y, acc.y);
                acc.z = fmaf(-v0, c0.z, acc.z); acc.w = fmaf(-v0, c0.w, acc.w);
            }
            *reinterpret_cast<float4*>(r32 + k) = acc;
            if (d.R16) {
                __nv_bfloat16* o = d.R16 + (size_t)i * n + k;
                o[0] = __float2bfloat16_rn(acc.x); o[1] = __float2bfloat16_rn(acc.y);
                o[2] = __float2bfloat16_rn(acc.z); o[3] = __float2bfloat16_rn(acc.w);
            }
            if (d.pos) {  // straight into the GEMM's compacted rows for the next iteration
                __nv_bfloat16* o = d.R16c + (size_t)d.pos[i] * n + k;
                o[0] = __float2bfloat16_rn(acc.x); o[1] = __float2bfloat16_rn(acc.y);
                o[2] = __float2bfloat16_rn(acc.z); o[3] = __float2bfloat16_rn(acc.w);
            }
            ss = fmaf(acc.x, acc.x, ss); ss = fmaf(acc.y, acc.y, ss);
            ss = fmaf(acc.z, acc.z, ss); ss = fmaf(acc.w, acc.w, ss);
            if (r16) { bf_terms(acc.x); bf_terms(acc.y); bf_terms(acc.z); bf_terms(acc.w); }
        }
    } else {
        for (int k = k_lo + threadIdx.x; k < k_hi; k += blockDim.x) {
            float acc = b[k];
            for (int a = 0; a < nz; ++a) acc = fmaf(-nzv[a], __ldg(d.A32 + (size_t)nzi[a] * n + k), acc);
            r32[k] = acc;
            if (d.R16) d.R16[(size_t)i * n + k] = __float2bfloat16_rn(acc);
            if (d.pos) d.R16c[(size_t)d.pos[i] * n + k] = __float2bfloat16_rn(acc);
            ss = fmaf(acc, acc, ss);
            if (r16) bf_terms(acc);
        }
    }
    // FP32 sums: a few roundings per term, a 256-way tree and at most 64 row blocks, far
    // inside the 1e-5 margin
    block_sum3(ss, es, ts, red);
    if (threadIdx.x == 0) {
        if (yb == 0) {
            d.nnz[i] = nz;
            // atom columns and b read, the FP32 residual (and its BF16 copies) written
            atomicAdd(&d.cnt->res_bytes, (unsigned long long)n * (4ull * (nz + 2) + (d.R16 ? 2ull : 0ull) +
                                                                  (d.pos ? 2ull : 0ull)));
        }
        bool last = nb == 1;
        if (!last) {
            float* part = d.res_part + ((size_t)i * nb + yb) * 3;
            part[0] = ss; part[1] = es; part[2] = ts;
            __threadfence();
            last = atomicAdd(&d.res_tick[i], 1) == nb - 1;
            if (last) {
                __threadfence();
                const volatile float* all = d.res_part + (size_t)i * nb * 3;
                ss = es = ts = 0.f;
                for (int y = 0; y < nb; ++y) { ss += all[3 * y]; es += all[3 * y + 1]; ts += all[3 * y + 2]; }
                d.res_tick[i] = 0;
            }
        }
        if (last) {
            d.rnorm[i] = sqrtf(ss) * (1.f + 1e-5f);
            d.r16e[i] = sqrtf(es) * (1.f + 1e-5f);
            d.r16t[i] = sqrtf(ts) * (1.f + 1e-5f);
        }
    }
}

// ------------------------------------------------------------------ Algorithm 2
// Subspace exploratory matching: of the q explored atoms (positions s0..s-1,
// appended by this iteration's selection) keep the rho with the largest
// |u| after the master problem, ties to the earlier position; the others
// leave S with their entries.  S, x_S, h, the power-iteration vector and the
// Gram block are compacted with the order of the remaining entries kept; the
// signal's FP64 factor workspace (idle while it grows) stages the Gram block.
__global__ void __launch_bounds__(256) k_smpl_prune(Dev d) {
    pdl_enter();
    const int g = blockIdx.x;
    if (g >= d.cnt->grow_n) return;
    const int i = d.list_grow[g];
    const int q = d.explore[i];
    if (q == 0) return;
    const int smax = d.smax, s = d.ssize[i], s0 = s - q, keep = d.rho;
    __shared__ int from[1024];
    __shared__ int ns_sh;
    int* Si = d.S + (size_t)i * smax;
    float* xi = d.xS + (size_t)i * smax;
    float* hi = d.h + (size_t)i * smax;
    float* ri = d.ritz + (size_t)i * smax;
    float* Gi = d.G + (size_t)i * smax * smax;
    uint32_t* mw = d.mask + (size_t)i * d.mw;
    // rank of each explored atom by |u| (descending, ties to the lower position)
    for (int a = threadIdx.x; a < q; a += blockDim.x) {
        const float ua = fabsf(xi[s0 + a]);
        int rank = 0;
        for (int b = 0; b < q; ++b) {
            const float ub = fabsf(xi[s0 + b]);
            rank += (ub > ua || (ub == ua && b < a)) ? 1 : 0;
        }
        from[s0 + a] = rank < keep ? 1 : 0;  // flag for now
    }
    __syncthreads();
    // ordered list of the surviving positions (one warp)
    if (threadIdx.x < 32) {
        int base = s0;
        for (int a0 = 0; a0 < q; a0 += 32) {
            const int a = a0 + threadIdx.x;
            const bool on = a < q && from[s0 + a] == 1;
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            const int pos = base + __popc(bal & ((1u << threadIdx.x) - 1u));
            __syncwarp();
            if (on) from[pos] = s0 + a;
            base += __popc(bal);
        }
        if (threadIdx.x == 0) ns_sh = base;
    }
    __syncthreads();
    const int ns = ns_sh;
    for (int a = threadIdx.x; a < s0; a += blockDim.x) from[a] = a;
    __syncthreads();
    // removed atoms leave the membership bitmap (positions not in from[s0..ns))
    for (int a = threadIdx.x; a < q; a += blockDim.x) {
        bool kept = false;
        for (int b = s0; b < ns; ++b) kept |= from[b] == s0 + a;
        if (!kept) {
            const int j = Si[s0 + a];
            atomicAnd(&mw[j >> 5], ~(1u << (j & 31)));
        }
    }
    // stage everything that moves, then write it back
    float* stage = reinterpret_cast<float*>(d.chol + (size_t)i * smax * smax);
    const int nk = ns - s0;  // kept explored atoms
    int Sk[4];
    float xk[4], hk[4], rk[4];
    for (int u = 0; u < 4; ++u) {
        const int a = s0 + threadIdx.x + u * blockDim.x;
        if (a < ns) { Sk[u] = Si[from[a]]; xk[u] = xi[from[a]]; hk[u] = hi[from[a]]; rk[u] = ri[from[a]]; }
    }
    // rows a >= s0 (all columns) and columns c >= s0 of rows a < s0
    const int moved = nk * ns + s0 * nk;
    for (int e = threadIdx.x; e < moved; e += blockDim.x) {
        int a, c;
        if (e < nk * ns) { a = s0 + e / ns; c = e % ns; }
        else { const int f = e - nk * ns; a = f / nk; c = s0 + f % nk; }
        stage[e] = Gi[(size_t)from[a] * smax + from[c]];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < moved; e += blockDim.x) {
        int a, c;
        if (e < nk * ns) { a = s0 + e / ns; c = e % ns; }
        else { const int f = e - nk * ns; a = f / nk; c = s0 + f % nk; }
        Gi[(size_t)a * smax + c] = stage[e];
    }
    for (int u = 0; u < 4; ++u) {
        const int a = s0 + threadIdx.x + u * blockDim.x;
        if (a < ns) { Si[a] = Sk[u]; xi[a] = xk[u]; hi[a] = hk[u]; ri[a] = rk[u]; }
    }
    for (int a = ns + threadIdx.x; a < s; a += blockDim.x) xi[a] = 0.f;
    if (threadIdx.x == 0) {
        d.ssize[i] = ns;
        d.snew[i] = nk;
        d.explore[i] = 0;
    }
}

// ------------------------------------------------------------------ output
__global__ void k_scatter(Dev d, float* X, double* X64) {
    pdl_enter();
    const int i = blockIdx.x;
    if (i >= d.p) return;
    const int s = d.ssize[i];
    const bool fin = d.finalized[i] != 0;
    for (int a = threadIdx.x; a < s; a += blockDim.x) {
        const int j = d.S[(size_t)i * d.smax + a];
        const double v = fin ? d.xS64[(size_t)i * d.smax + a] : (double)d.xS[(size_t)i * d.smax + a];
        if (X) X[(size_t)i * d.m + j] = (float)v;
        if (X64) X64[(size_t)i * d.m + j] = v;
    }
}

// ------------------------------------------------------------------ dictionary prep
__global__ void k_colnorm(const float* A32, int n, int m, float* colnorm, __nv_bfloat16* A16, float* err2) {
    const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= m) return;
    const float* a = A32 + (size_t)j * n;
    double ss = 0.0, es = 0.0, ts = 0.0;
    for (int k = lane; k < n; k += 32) {
        const float v = a[k];
        ss += (double)v * (double)v;
        if (A16) {
            const __nv_bfloat16 q = __float2bfloat16_rn(v);
            A16[(size_t)j * n + k] = q;
            const double fq = (double)__bfloat162float(q), e = (double)v - fq;  // both exact in FP64
            es += e * e;
            ts += fq * fq;
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
        es += __shfl_xor_sync(0xffffffffu, es, o);
        ts += __shfl_xor_sync(0xffffffffu, ts, o);
    }
    if (lane == 0) {
        colnorm[j] = __double2float_ru(sqrt(ss));
        // FP64 sums of at most n squares: relative error far below the 1e-6 margin
        if (err2) {
            err2[j] = __double2float_ru(sqrt(es) * (1.0 + 1e-6));
            err2[m + j] = __double2float_ru(sqrt(ts) * (1.0 + 1e-6));
        }
    }
}

__global__ void k_max_reduce(const float* v, int len, float* out) {
    float mx = 0.f;
    for (int t = threadIdx.x; t < len; t += blockDim.x) mx = fmaxf(mx, v[t]);
#pragma unroll
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ float red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmaxf(t, red[w]);
        *out = t;
    }
}

__global__ void k_gather_r16(Dev d, int cur) {
    pdl_enter();
    const int k = blockIdx.x;
    if (k >= d.cnt->act_n[cur]) return;
    const int i = d.act[cur][k];
    const int n = d.n;
    const uint4* src = reinterpret_cast<const uint4*>(d.R16 + (size_t)i * n);
    uint4* dst = reinterpret_cast<uint4*>(d.R16c + (size_t)k * n);
    for (int t = threadIdx.x; t < n / 8; t += blockDim.x) dst[t] = src[t];
}

// Load caller residuals for a stand-alone correlation: R32 (and R16), identity active list.
__global__ void k_prep_correlate(Dev d, const float* R) {
    const int i = blockIdx.x;
    if (i >= d.p) return;
    const int n = d.n;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const float v = R[(size_t)i * n + k];
        d.R32[(size_t)i * n + k] = v;
        if (d.R16) d.R16[(size_t)i * n + k] = __float2bfloat16_rn(v);
    }
    if (threadIdx.x == 0) {
        d.act[0][i] = i;
        if (i == 0) { d.cnt->act_n[0] = d.p; d.cnt->err = 0; }
    }
}

}  // namespace

cudaError_t launch_prep_correlate(const Dev& d, const float* R, cudaStream_t s, int64_t* nl) {
    if (d.p <= 0) return cudaSuccess;
    k_prep_correlate<<<d.p, 256, 0, s>>>(d, R);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_init(const Dev& d, cudaStream_t s, int64_t* nl) {
    if (d.p <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_init, dim3(d.p), dim3(256), 0, s, d);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

// The two tiles: gram_large for batches that fill the chip, gram_small for the others.
template <int BM, int BN, int TR, int TC, int BK, int ST>
static cudaError_t gram_launch(const Dev& d, int ub, int scap, cudaStream_t s, bool prepare) {
    constexpr size_t sm = (size_t)ST * (BM + BN) * (BK + 4) * sizeof(float);
    if (prepare) {
        cudaError_t e = cudaFuncSetAttribute(k_gram<BM, BN, TR, TC, BK, ST, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_gram<BM, BN, TR, TC, BK, ST, false>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        return e;
    }
    const dim3 grid(ub, (scap + BM - 1) / BM), block((BM / TR) * (BN / TC));
    return (d.n & 3) == 0 ? launch_chain(k_gram<BM, BN, TR, TC, BK, ST, true>, grid, block, sm, s, d)
                          : launch_chain(k_gram<BM, BN, TR, TC, BK, ST, false>, grid, block, sm, s, d);
}
static cudaError_t gram_large(const Dev& d, int ub, int scap, cudaStream_t s, bool prepare = false) {
    return gram_launch<64, 64, 4, 4, 32, 4>(d, ub, scap, s, prepare);
}
static cudaError_t gram_small(const Dev& d, int ub, int scap, cudaStream_t s, bool prepare = false) {
    return gram_launch<32, 32, 2, 4, 32, 6>(d, ub, scap, s, prepare);
}

cudaError_t prepare_gram() {
    static bool attr = false;
    if (attr) return cudaSuccess;
    cudaError_t e = gram_large(Dev{}, 0, 0, nullptr, true);
    if (e == cudaSuccess) e = gram_small(Dev{}, 0, 0, nullptr, true);
    if (e == cudaSuccess) attr = true;
    return e;
}

cudaError_t launch_gram(const Dev& d, int ub, int qmax, int scap, int sms, cudaStream_t s, int64_t* nl) {
    if (ub <= 0) return cudaSuccess;
    cudaError_t e = prepare_gram();
    if (e != cudaSuccess) return e;
    // The large tile reads each atom column half as often, and pays where its blocks fill the chip twice
    // over and its columns are mostly used: 512 signals of 2048 x 32768 gaining 50 atoms each, 2.6 ms a
    // solve against 3.0 with the small one; 300 gaining 100, 4.5 against 5.9.  Below, the small one:
    // 1024 x 8192, 512 signals gaining 24, 0.31 ms; 75 signals of 1496 x 20011 gaining 30, 0.23.
    const bool large = qmax > 32 && (long long)ub * ((scap + 63) / 64) >= 2ll * sms;
    e = large ? gram_large(d, ub, scap, s) : gram_small(d, ub, scap, s);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

#ifdef MPL_APG_TRACE
extern "C" int mpl_debug_apg_trace(long long* out, int count, int reset) {
    if (count > 8192) count = 8192;
    if (cudaDeviceSynchronize() != cudaSuccess) return -1;
    if (cudaMemcpyFromSymbol(out, g_apg_trace, sizeof(long long) * 8 * (size_t)count) != cudaSuccess) return -1;
    if (reset) {
        static long long zero[8192][8];
        if (cudaMemcpyToSymbol(g_apg_trace, zero, sizeof(zero)) != cudaSuccess) return -1;
    }
    return count;
}
#endif

cudaError_t prepare_apg() {
    static bool attr = false;
    if (attr) return cudaSuccess;
    const int mx = (int)(((size_t)APG_SMEM_S * APG_SMEM_S + 6 * 1024) * sizeof(float));
    cudaError_t e = cudaFuncSetAttribute(k_apg<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_apg<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
    if (e == cudaSuccess) attr = true;
    return e;
}

// Vector stride of the master problem for a bound vcap on |S|: a multiple of 32 (and so of
// 4, the streamed product's float4 slices), at least the bound, at most the capacity rounded
// up to 4.
static int apg_vcap(const Dev& d, int vcap) {
    vcap = ((vcap + 31) / 32) * 32;
    const int cap4 = (d.smax + 3) & ~3;
    return vcap < cap4 ? vcap : cap4;
}

int apg_classes(const Dev& d, int vcap) {
    vcap = apg_vcap(d, vcap);
    return vcap <= APG_REG_S ? 1 : (vcap <= APG_SMEM_S ? 2 : 3);
}

// The register variants by the bound on |S|: rows of a warp, then 64, 96 and 128 rows (the more
// rows, the more registers a thread and the fewer CTAs an SM holds).
template <int NC, bool WARP, int MINB>
static cudaError_t launch_apg_reg_t(const Dev& d, int ub, int sms, int vcap, cudaStream_t s) {
    constexpr int nt = WARP ? 32 * APG_WARPS : 4 * NC;
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_apg_reg<NC, WARP, MINB>, nt, 0);
    if (e != cudaSuccess) return e;
    const int need = WARP ? (ub + APG_WARPS - 1) / APG_WARPS : ub;
    const int grid = std::min(sms * std::max(per_sm, 1), need);
    return launch_chain(k_apg_reg<NC, WARP, MINB>, dim3(grid), dim3(nt), 0, s, d, vcap);
}

cudaError_t launch_apg(const Dev& d, int ub, int sms, int vcap, cudaStream_t s, int64_t* nl, int cls) {
    if (ub <= 0) return cudaSuccess;
    vcap = apg_vcap(d, vcap);
    cudaError_t e;
    if (cls == APG_REG) {
        e = vcap <= 32   ? launch_apg_reg_t<32, true, 4>(d, ub, sms, vcap, s)
            : vcap <= 64 ? launch_apg_reg_t<32, false, 5>(d, ub, sms, vcap, s)
            : vcap <= 96 ? launch_apg_reg_t<48, false, 3>(d, ub, sms, vcap, s)
                         : launch_apg_reg_t<64, false, 2>(d, ub, sms, vcap, s);
    } else {
        if ((e = prepare_apg()) != cudaSuccess) return e;
        // APG_SMEM: the blocks past the registers that fit shared memory; APG_GLOBAL: the others,
        // without the block area, so that several CTAs per SM stream their blocks from L2/HBM
        const bool stream = cls == APG_GLOBAL;
        const int gcap = stream ? 0 : (vcap < APG_SMEM_S ? vcap : APG_SMEM_S);
        const size_t dyn = ((size_t)gcap * gcap + 6 * (size_t)vcap) * sizeof(float);
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, stream ? k_apg<true> : k_apg<false>, APG_THREADS,
                                                          dyn);
        if (e != cudaSuccess) return e;
        const int grid = std::min(sms * std::max(per_sm, 1), ub);
        e = stream ? launch_chain(k_apg<true>, dim3(grid), dim3(APG_THREADS), dyn, s, d, vcap, gcap, cls)
                   : launch_chain(k_apg<false>, dim3(grid), dim3(APG_THREADS), dyn, s, d, vcap, gcap, cls);
    }
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_residual(const Dev& d, int ub, cudaStream_t s, int64_t* nl) {
    if (ub <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_residual, dim3(ub, res_blocks(d.n)), dim3(256), 0, s, d);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

// Per-signal statistics packed on the device into the host struct layout (one copy back).
// ------------------------------------------------------------------ re-entry
// Finished signals (reent[s] of the slots s in mask, in slot order) go back to the end of
// the active list of this iteration, with their rows in the GEMM's compacted BF16 residual
// (the finish wrote the per-signal copy).  Launched only when a finish is done; the last CTA
// updates the lengths, once every CTA has read them.
__global__ void __launch_bounds__(256) k_merge(Dev d, int cur, int mask) {
    pdl_enter();
    const int n = d.n;
    int base = d.cnt->act_n[cur];
    for (int q = 0; q < FIN_SLOTS; ++q) {
        if (!((mask >> q) & 1)) continue;
        const int cnt = d.cnt->reent_n[q];
        for (int b = blockIdx.x; b < cnt; b += gridDim.x) {
            const int i = d.reent[q][b];
            const int row = base + b;
            if (MPL_OOB(row >= d.p || i < 0 || i >= d.p, 101)) continue;
            if (threadIdx.x == 0) {
                d.act[cur][row] = i;
                if (d.pos) d.pos[i] = row;
            }
            if (d.pos) {
                const __nv_bfloat16* src = d.R16 + (size_t)i * n;
                __nv_bfloat16* dst = d.R16c + (size_t)row * n;
                for (int k = threadIdx.x; k < n; k += blockDim.x) dst[k] = src[k];
            }
        }
        base += cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&d.cnt->merge_done, 1) == (int)gridDim.x - 1) {
            for (int q = 0; q < FIN_SLOTS; ++q)
                if ((mask >> q) & 1) d.cnt->reent_n[q] = 0;
            d.cnt->act_n[cur] = base;
            d.cnt->merge_done = 0;
        }
    }
}

cudaError_t launch_merge(const Dev& d, int cur, int mask, int ub, cudaStream_t s, int64_t* nl) {
    if (ub <= 0) return cudaSuccess;
    const int grid = ub < 608 ? ub : 608;
    const cudaError_t e = launch_chain(k_merge, dim3(grid), dim3(256), 0, s, d, cur, mask);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

__global__ void k_pack_stats(Dev d, mpl_signal_stats_t* out) {
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d.p) return;
    mpl_signal_stats_t s;
    s.outer_iters = d.outer[i];
    s.inner_iters = d.inner[i];
    s.active_size = d.ssize[i];
    s.nnz = d.nnz[i];
    s.status = d.sstatus[i];
    s.finishes = d.finishes[i];
    const double obj = d.obj[i];
    s.objective = obj;
    s.kkt = fmax(d.kkt_in[i], d.kkt_out[i]);
    // relative duality gap with the dual point xi * min(1, lambda / ||A^T xi||_inf) of eq. 5
    const double ginf = d.ginf[i], rr = d.rr[i], rb = d.rb[i], lam = (double)d.lam[i];
    const double sc = (ginf > lam && ginf > 0.0) ? lam / ginf : 1.0;
    const double D = -0.5 * sc * sc * rr + sc * rb;
    s.gap = obj > 0.0 ? (obj - D) / obj : 0.0;
    out[i] = s;
}

cudaError_t launch_pack_stats(const Dev& d, mpl_signal_stats_t* out, cudaStream_t s, int64_t* nl) {
    if (d.p <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_pack_stats, dim3((d.p + 127) / 128), dim3(128), 0, s, d, out);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_smpl_prune(const Dev& d, int ub, cudaStream_t s, int64_t* nl) {
    if (ub <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_smpl_prune, dim3(ub), dim3(256), 0, s, d);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_scatter(const Dev& d, float* X, double* X64, cudaStream_t s, int64_t* nl) {
    if (d.p <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_scatter, dim3(d.p), dim3(128), 0, s, d, X, X64);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_colnorm(const float* A32, int n, int m, float* colnorm, __nv_bfloat16* A16,
                           cudaStream_t s, int64_t* nl, float* err2) {
    const int per = 8;  // warps per block
    k_colnorm<<<(m + per - 1) / per, per * 32, 0, s>>>(A32, n, m, colnorm, A16, err2);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_max_reduce(const float* v, int len, float* out, cudaStream_t s, int64_t* nl) {
    k_max_reduce<<<1, 1024, 0, s>>>(v, len, out);
    ++*nl;
    return cudaGetLastError();
}

cudaError_t launch_gather_r16(const Dev& d, int cur, int act_n_ub, cudaStream_t s, int64_t* nl) {
    if (act_n_ub <= 0) return cudaSuccess;
    const cudaError_t e = launch_chain(k_gather_r16, dim3(act_n_ub), dim3(128), 0, s, d, cur);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaGetLastError();
}

}  // namespace mpl

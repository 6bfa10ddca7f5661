// Worst-case analysis of Algorithm 1 in FP32 on the 5th-generation tensor cores: C = A^T R with
// every FP32 operand split into two TF32 parts.
//
//   x = hi + lo,  hi = x rounded to TF32's 11 significant bits, lo = x - hi rounded to them too:
//   |x - hi - lo| <= 2^-23 |x| (and 2^-137, TF32's subnormals being multiples of 2^-136: rows all of whose
//   entries are below 2^-113 lose accuracy).  a r is taken as a_hi r_lo + a_lo r_hi + a_hi r_hi (the
//   dropped a_lo r_lo is at most 2^-22 |a r|, of either sign).
//
// The sums of 32 products along n are accumulated in TMEM (the small products first, then the
// large ones) and added to FP32 registers with round-to-nearest, so that the tensor core's
// truncating accumulation acts over 32 products only and the sequential FP32 chain is n / 32
// long instead of n.
//
// A persistent CTA walks output tiles of 128 atoms x w signals.  Roles (five warpgroups):
//   warps 0-7   loaders: rows of atoms and of the active signals' residuals (gathered through the
//               active list) are copied asynchronously, as FP32, to where their hi part goes in
//               one of two stages (three, a stage ahead, up to 128 signals; 128-byte-swizzled
//               tiles); each lane then splits the 16 bytes it copied, so that no thread waits for
//               another's copies.
//   warp 8      allocates TMEM; one thread issues the 12 tcgen05.mma of a stage (kind::tf32,
//               M = 128, N = w, K = 8) into the stage's accumulator and commits.
//   warps 12-19 accumulate: tcgen05.ld of the finished stage's accumulator, added to registers
//               (each warp its 32 atoms and half of the tile's signals); scores stored at the end.
// setmaxnreg moves registers from the loaders to the accumulating warps.
//
// What bounds it: the loaders' instructions, and with few signals the latency of their copies and
// splits, which the third stage overlaps (2048 x 32768: 16 signals 181 -> 124 us, 64 193 -> 141,
// 128 198 -> 155; 777 x 6001 x 99 55 -> 50 us).  A stage of a 128 x 256 tile takes 3500 cycles, of
// which the tensor core works 2100 and shared memory (three reads of every operand by
// the MMAs, the copies and the split: 340 KB) at least 2650.  2044 x 32771 x 500: 478 us
// (140 TFLOP/s), 4096 x 65536 x 1024: 3.13 ms, 1024 x 8192 x 256: 48 us (three stages); the FP32
// chain on the SIMT cores takes 1596 us, 12.2 ms and 162 us.  Loads staged in registers (592 us), six
// loader warps (507 us) and more, shorter stages with the copies issued ahead (557 to 650 us) were
// slower.
// Error against FP64 (2-norm), relative to the FP32 chain's: Gaussian data 0.65 at n = 128, 0.48 at 256, 0.21
// at 4096; data of one sign, where the tensor core's truncation does not cancel, 0.85, 0.56, 0.22; the same
// over 24 binary orders, or one large product in eight, 1.18 at n = 128 and 0.75 at 256, 0.07 at 4096.  So
// signals of fewer than TF32_MIN_N = 256 entries keep the chain.
//
// Inputs at or near overflow (infinities, NaN, |x| >= 2^128 (1 - 2^-12)) have no split: their rows
// are flagged and the affected scores recomputed with one FP32 FMA chain over n, so that a
// score is infinite or NaN where the FP32 product is.  2044 x 32771 x 500: 1.52 ms with one infinite
// atom, 1.29 with one infinite signal, 6.3 with all of them (0.48 without; the SIMT kernel always 1.60;
// one chain at a time 18, 2.3 and 197).
//
// Every wait is bounded; on expiry the CTA records DERR_TIMEOUT, the MMA thread waits (bounded) for
// the MMAs it issued, the scores of the tiles the CTA did not finish are set to NaN, and the CTA
// frees its TMEM and returns.
#include "mpl_internal.cuh"
#include "tc_ptx.cuh"

namespace mpl {

namespace {

constexpr int TF_BM = 128;           // atoms per tile
constexpr int TF_BN = 256;           // most signals per tile
constexpr int TF_BK = 32;            // columns of n per stage: one 128-byte swizzle row
constexpr int TF_STAGES = 3;         // most stages, each with its TMEM accumulator (see TfTile)
constexpr int TF_THREADS = 640;
constexpr int TF_LOADERS = 8;        // loader warps
constexpr int TF_MMA_WARP = 8;
constexpr int TF_ITEMS = 12;         // most 4-row items per loader warp and stage: (128 + 256) / 4 / 8
constexpr int TF_STEP = 4 * TF_LOADERS;  // rows from one item of a warp to its next (a multiple of 8)
constexpr int TF_ACC_WARPS = 8;
constexpr int TF_REGS_ACC = 152, TF_REGS_LOAD = 56;  // per thread after setmaxnreg
constexpr int TF_SLOTS = 8;          // flag slots by tile (the loaders run at most 4 tiles ahead)
constexpr int TF_ROWS = TF_BM + TF_BN;

constexpr int TF_A_BYTES = TF_BM * 128;
constexpr int TF_RING_BYTES = 4 * TF_ROWS * 128;      // two stages of the widest tile
constexpr int TF_TMEM = 512;                          // columns: the whole TMEM of the SM

struct TfShared {
    uint64_t full[TF_STAGES];    // the loaders have filled the stage
    uint64_t done[TF_STAGES];    // its MMAs are complete: stage free, accumulator ready
    uint64_t tempty[TF_STAGES];  // its accumulator has been read
    uint64_t drain;
    uint32_t tmem;
    int abort_flag;
    const float* row[TF_ROWS];                   // the tile's rows (atoms, signals), null past the end
    unsigned char inf[TF_SLOTS][TF_ROWS];        // the row holds a value without a split
    unsigned char nan[TF_SLOTS][TF_ROWS];        // ... a NaN
    unsigned char any[TF_SLOTS][8];              // any such row, by loader warp
    alignas(16) float chain[TF_ACC_WARPS][16 * 32];  // 32 columns of 16 signals (chain_block)
};
constexpr size_t TF_SMEM = (size_t)TF_RING_BYTES + 1024 + sizeof(TfShared);
static_assert(TF_SMEM <= 227 * 1024, "the stages and the barriers fit one CTA's shared memory");
static_assert(TF_ITEMS * TF_STEP == TF_ROWS && TF_STEP % 8 == 0, "every row has one loader");

// Instruction descriptor, kind::tf32: D f32, A/B tf32, both K-major, M x N.
__device__ __forceinline__ uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// Asynchronous copies of four consecutive entries to shared memory, zero past the first `left`.
__device__ __forceinline__ void copy4_16(uint32_t dst, const float* src, int left) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(left > 0 ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy4_4(uint32_t dst, const float* src, int left) {  // rows of any alignment
#pragma unroll
    for (int e = 0; e < 4; ++e)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * e), "l"(left > e ? src + e : src),
                     "r"(left > e ? 4 : 0)
                     : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float4 ld_shared4(uint32_t src) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(src) : "memory");
    return v;
}

__device__ __forceinline__ void st_shared4(uint32_t dst, const uint32_t (&v)[4]) {
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
                 : "memory");
}

// A kernel for at most TF_NARROW signals per tile has three stages in the same ring, and its loaders copy a
// stage ahead of the one they split.  With two that would make them wait for the MMAs of the stage
// before, which take about as long as a wide tile's split.
constexpr int TF_NARROW = 128;
template <bool NARROW>
struct TfTile {
    static constexpr int STAGES = NARROW ? 3 : 2;
    static constexpr int BN = NARROW ? TF_NARROW : TF_BN;        // most signals
    static constexpr int ROWS = TF_BM + BN;
    static constexpr int GROUPS = ROWS / (4 * TF_STEP);          // of four items, per loader warp
    static constexpr int HALF_BYTES = ROWS * 128;                // the hi (or lo) tiles: atoms, then signals
    static constexpr int STAGE_BYTES = 2 * HALF_BYTES;
    static_assert(STAGES * STAGE_BYTES <= TF_RING_BYTES && STAGES * BN <= TF_TMEM && ROWS % (4 * TF_STEP) == 0 &&
                  STAGES <= TF_STAGES, "the stages fit, in whole groups");
};

// Signals per tile (a multiple of 16): the count of active signals shrinks from one outer iteration
// to the next, and a narrower tile costs less.  A stage takes about 576 + w units (2700 cycles
// measured at w = 64, 3000 at 128, 3500 at 256), 420 + w in the narrow kernel (1900 at 16, 2400 at 128),
// and ceil(tiles / grid) tiles run in turn on a CTA.
template <bool NARROW>
__device__ __forceinline__ int pick_width(int act_n, int tiles_m, int grid) {
    constexpr int BN = TfTile<NARROW>::BN;
    const int t0 = (act_n + BN - 1) / BN;
    int best = BN;
    float cost = 3e38f;
    for (int t = t0; t < t0 + 8; ++t) {
        const int w = (((act_n + t - 1) / t) + 15) / 16 * 16;
        const float tiles = (float)tiles_m * (float)((act_n + w - 1) / w);
        const float c = ceilf(tiles / (float)grid) * (float)((NARROW ? 420 : 576) + w);
        if (c < cost) { cost = c; best = w; }
    }
    return best;
}

constexpr uint32_t TF_NOSPLIT = 0x7f7ff000u;  // |x| bits from here on: rounding x to TF32 is not finite

__device__ __forceinline__ uint32_t tf32_hi(uint32_t x) { return (x + 0x1000u) & 0xffffe000u; }

// Four entries of which some may have no split: those keep their upper bits (a NaN stays one) and
// flag the row.
__device__ __noinline__ void store_nosplit(float4 v, uint32_t dst, uint32_t half, unsigned char* inf, unsigned char* nan) {
    const float f[4] = {v.x, v.y, v.z, v.w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t x = __float_as_uint(f[e]);
        const uint32_t a = x & 0x7fffffffu;
        hi[e] = tf32_hi(x);
        lo[e] = __float_as_uint(__uint_as_float(x) - __uint_as_float(hi[e])) + 0x1000u;
        if (a >= TF_NOSPLIT) { hi[e] = x & 0xffffe000u; lo[e] = 0u; *inf = 1; }
        if (a > 0x7f800000u) { hi[e] = 0x7fc00000u; *nan = 1; }
    }
    st_shared4(dst, hi);
    st_shared4(dst + half, lo);
}

// A loader warp's part of a tile: the slices' copies, their splits, the stages handed on.  Returns false
// when a wait expired.  NARROW: at most TF_NARROW signals, three stages, copies a stage ahead.
template <bool VEC, bool NARROW>
__device__ __forceinline__ bool load_tile(const Dev& d, TfShared& sh, uint32_t base, const volatile int* abort_flag,
                                          int warp, int lane, int rows, int slot, int nk, int n, int& stage,
                                          uint32_t& ph) {
    constexpr int NST = TfTile<NARROW>::STAGES, GROUPS = TfTile<NARROW>::GROUPS;
    constexpr uint32_t HALF = TfTile<NARROW>::HALF_BYTES;
    const int r0 = warp * 4 + (lane >> 3), kc = (lane & 7) * 4;
    const uint32_t dst0 = base + (uint32_t)(r0 * 128 + (((lane & 7) ^ (r0 & 7)) << 4));
    // copied as FP32 to where hi goes: each lane splits the 16 bytes it copied, so its own copies are all
    // it waits for
    auto copy_group = [&](uint32_t dst, int k, int g) {
        if (4 * warp + 4 * g * TF_STEP < rows) {  // (the same in all lanes)
            const float* row[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) row[i] = sh.row[r0 + (4 * g + i) * TF_STEP];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t q = dst + (uint32_t)((4 * g + i) * TF_STEP * 128);
                // (zeros past the end: a row repeated there instead would be one hot line for every CTA)
                const bool in = row[i] != nullptr && k < n;
                if (VEC) copy4_16(q, in ? row[i] + k : d.A32, in ? n - k : 0);
                else copy4_4(q, in ? row[i] + k : d.A32, in ? n - k : 0);
            }
        }
        copy_commit();
    };
    auto split_group = [&](uint32_t dst, int g) {
        if (4 * warp + 4 * g * TF_STEP >= rows) return;
        float4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = ld_shared4(dst + (uint32_t)((4 * g + i) * TF_STEP * 128));
        float chk = 0.f;  // NaN once some lo is not finite
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float x[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                hi[e] = tf32_hi(__float_as_uint(x[e]));
                const float l = x[e] - __uint_as_float(hi[e]);
                chk = fmaf(l, 0.f, chk);
                lo[e] = __float_as_uint(l) + 0x1000u;  // (the tensor core reads the upper bits)
            }
            st_shared4(dst + (uint32_t)((4 * g + i) * TF_STEP * 128), hi);
            st_shared4(dst + (uint32_t)((4 * g + i) * TF_STEP * 128) + HALF, lo);
        }
        if (chk != chk) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + (4 * g + i) * TF_STEP;
                store_nosplit(v[i], dst + (uint32_t)((4 * g + i) * TF_STEP * 128), HALF, &sh.inf[slot][r],
                              &sh.nan[slot][r]);
            }
            sh.any[slot][warp] = 1;
        }
    };
    // waits for a stage to be free and copies slice kb to it
    auto copy_stage = [&](int st, uint32_t parity, int kb) {
        bool free = mbar_wait(&sh.done[st], parity ^ 1u, abort_flag);
        free = __all_sync(0xffffffffu, free);
        if (!free) {
            if (lane == 0) { sh.abort_flag = 1; atomicCAS(&d.cnt->err, 0, (int)DERR_TIMEOUT); }
            copy_wait<0>();
            return false;
        }
        const uint32_t dst = dst0 + (uint32_t)st * (2u * HALF);
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) copy_group(dst, kb * TF_BK + kc, g);
        return true;
    };
    if (NARROW && !copy_stage(stage, ph, 0)) return false;
#pragma unroll 1
    for (int kb = 0; kb < nk; ++kb) {
        if (NARROW) {
            if (kb + 1 < nk) {
                const int nx = stage + 1 == NST ? 0 : stage + 1;
                if (!copy_stage(nx, nx ? ph : ph ^ 1u, kb + 1)) return false;
                copy_wait<GROUPS>();
            } else {
                copy_wait<0>();
            }
        } else if (!copy_stage(stage, ph, kb)) {
            return false;
        }
        const uint32_t dst = dst0 + (uint32_t)stage * (2u * HALF);
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
            if (!NARROW) {
                if (g == 0) copy_wait<2>();
                else if (g == 1) copy_wait<1>();
                else copy_wait<0>();
            }
            split_group(dst, g);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.full[stage]);
        if (++stage == NST) { stage = 0; ph ^= 1u; }
    }
    return true;
}

// Scores of a warp's 32 atoms (one a lane) and 16 signals from k0 on that involve a value without a split,
// and no NaN (whose products are NaN already): one FP32 FMA chain over n each.  a_inf, a_nan: the lane's
// atom; inf, nan: the signals; rs: 16 x 32 floats of shared memory, the warp's own.  What bounds it is the
// round trip to memory, so 32 columns of everything are read at once: a cache line of its atom
// per lane, and the signals' rows through rs.  All 16 chains of a lane run together, whichever are wanted.
template <bool VEC>
__device__ __noinline__ void chain_block(const float* __restrict__ A, const float* __restrict__ R, const int* act,
                                         float* C, int n, int m, int atom, bool a_inf, bool a_nan,
                                         const unsigned char* inf, const unsigned char* nan, int k0, int act_n,
                                         float* rs) {
    const int lane = threadIdx.x & 31;
    const bool mine = atom < m && !a_nan;
    const unsigned snan = __ballot_sync(0xffffffffu, lane < 16 && nan[lane & 15] != 0);
    const unsigned sinf = __ballot_sync(0xffffffffu, lane < 16 && inf[lane & 15] != 0) & ~snan;
    if (!__any_sync(0xffffffffu, mine && (a_inf || sinf != 0u))) return;
    const float* a = A + (size_t)min(atom, m - 1) * n;
    const int sig = act[min(k0 + (lane & 15), act_n - 1)];
    float s[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) s[e] = 0.f;
#pragma unroll 1
    for (int x0 = 0; x0 < n; x0 += 32) {
        float av[32];
        if (VEC) {
#pragma unroll
            for (int q = 0; q < 32; q += 4) {
                const float4 v = x0 + q < n ? __ldg(reinterpret_cast<const float4*>(a + x0 + q))
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                av[q] = v.x; av[q + 1] = v.y; av[q + 2] = v.z; av[q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 32; ++q) av[q] = x0 + q < n ? __ldg(a + x0 + q) : 0.f;
        }
        float rv[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int i = __shfl_sync(0xffffffffu, sig, e);
            rv[e] = x0 + lane < n ? __ldg(R + (size_t)i * n + x0 + lane) : 0.f;
        }
        __syncwarp();  // (the last columns have been read)
#pragma unroll
        for (int e = 0; e < 16; ++e) rs[e * 32 + lane] = rv[e];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 32; q += 4)
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const float4 r = *reinterpret_cast<const float4*>(rs + e * 32 + q);
                s[e] = fmaf(av[q + 3], r.w, fmaf(av[q + 2], r.z, fmaf(av[q + 1], r.y, fmaf(av[q], r.x, s[e]))));
            }
    }
#pragma unroll
    for (int e = 0; e < 16; ++e)
        if (mine && k0 + e < act_n && !((snan >> e) & 1u) && (a_inf || ((sinf >> e) & 1u)))
            C[(size_t)(k0 + e) * m + atom] = s[e];
}

// The chains of a tile that an accumulating warp has stored, for its 32 atoms and its blocks of signals.
template <bool VEC>
__device__ __forceinline__ void chain_tile(const Dev& d, TfShared& sh, int cur, int slot, int tm, int tn, int w,
                                        int act_n) {
    const int warp = (threadIdx.x >> 5) - 12, ar = (warp & 3) * 32 + (threadIdx.x & 31);
#pragma unroll 1
    for (int c0 = (warp >> 2) * 16; c0 < w && tn * w + c0 < act_n; c0 += 32)
        chain_block<VEC>(d.A32, d.R32, d.act[cur], d.Cs, d.n, d.m, tm * TF_BM + ar, sh.inf[slot][ar] != 0,
                         sh.nan[slot][ar] != 0, sh.inf[slot] + TF_BM + c0, sh.nan[slot] + TF_BM + c0, tn * w + c0,
                         act_n, sh.chain[warp]);
}

// The scores of an accumulating warp in the tiles from t on, which its block gave up on, are no numbers: a
// caller who cannot see the error code sees them.
__device__ __forceinline__ void unfinished(const Dev& d, long long t, long long ntiles, int tiles_n, int w, int act_n) {
    const int warp = (threadIdx.x >> 5) - 12;
    for (; t < ntiles; t += gridDim.x) {
        const int tm = (int)(t / tiles_n), tn = (int)(t - (long long)tm * tiles_n);
        const int atom = tm * TF_BM + (warp & 3) * 32 + (threadIdx.x & 31);
        for (int c0 = (warp >> 2) * 16; c0 < w; c0 += 32)
            for (int k = tn * w + c0; k < min(act_n, tn * w + c0 + 16); ++k)
                if (atom < d.m) d.Cs[(size_t)k * d.m + atom] = __int_as_float(0x7fffffff);
    }
}

template <bool VEC, bool NARROW>
__global__ void __launch_bounds__(TF_THREADS, 1) k_corr_tf32(Dev d, int cur) {
    pdl_enter();
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    TfShared& sh = *reinterpret_cast<TfShared*>(base + TF_RING_BYTES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int act_n = d.cnt->act_n[cur];
    const int m = d.m, n = d.n;
    const int tiles_m = (m + TF_BM - 1) / TF_BM;
    if (act_n <= 0) return;
    const int w = pick_width<NARROW>(act_n, tiles_m, (int)gridDim.x);
    const int tiles_n = (act_n + w - 1) / w;
    const long long ntiles = (long long)tiles_m * tiles_n;
    if ((long long)blockIdx.x >= ntiles) return;  // (the whole CTA, before it holds anything)
    const int nk = (n + TF_BK - 1) / TF_BK;
    using T = TfTile<NARROW>;
    constexpr int nst = T::STAGES;
    volatile int* abort_flag = &sh.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init(&sh.full[s], TF_LOADERS);
            mbar_init(&sh.done[s], 1);
            mbar_init(&sh.tempty[s], TF_ACC_WARPS);
        }
        mbar_init(&sh.drain, 1);
        sh.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == TF_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                     "r"(TF_TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = sh.tmem;

    auto give_up = [&]() {
        *abort_flag = 1;
        atomicCAS(&d.cnt->err, 0, (int)DERR_TIMEOUT);
    };

    if (warp < 12) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(TF_REGS_LOAD));
        if (warp < TF_LOADERS) {
            // item i of this warp: rows 4 warp + TF_STEP i .. + 3 of [atoms | signals], eight lanes
            // (16 bytes each) per row; in groups of four items, of which a narrow tile takes fewer
            const int r0 = warp * 4 + (lane >> 3);
            const int rows = TF_BM + w;
            const uint32_t base_u = smem_u32(base);
            int stage = 0;
            uint32_t ph = 0;
            unsigned tcount = 0;
            bool ok = true;
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tcount) {
                const int tm = (int)(t / tiles_n), tn = (int)(t - (long long)tm * tiles_n);
                const int slot = tcount & (TF_SLOTS - 1);
                __syncwarp();
                if ((lane & 7) == 0) {
#pragma unroll 1
                    for (int r = r0; r < TF_ROWS; r += TF_STEP) {
                        const int j = tm * TF_BM + r, k = tn * w + r - TF_BM;
                        const float* row = nullptr;
                        if (r < TF_BM) {
                            if (j < m) row = d.A32 + (size_t)j * n;
                        } else if (r < rows && k < act_n) {
                            row = d.R32 + (size_t)d.act[cur][k] * n;
                        }
                        sh.row[r] = row;
                        sh.inf[slot][r] = 0;
                        sh.nan[slot][r] = 0;
                    }
                }
                if (lane == 0) sh.any[slot][warp] = 0;
                __syncwarp();
                ok = load_tile<VEC, NARROW>(d, sh, base_u, abort_flag, warp, lane, rows, slot, nk, n, stage, ph);
            }
        } else if (warp == TF_MMA_WARP && lane == 0) {
            const uint32_t idesc = idesc_tf32(TF_BM, w);
            int stage = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                for (int kb = 0; kb < nk; ++kb) {
                    if (!mbar_wait(&sh.tempty[stage], ph ^ 1u, abort_flag) ||
                        !mbar_wait(&sh.full[stage], ph, abort_flag)) {
                        give_up();
                        ok = false;
                        break;
                    }
                    // the loaders' writes, ordered before this by the barrier, become visible to the
                    // tensor core here
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    fence_after();
                    const uint8_t* sb = base + stage * T::STAGE_BYTES;
                    const uint64_t ah = sdesc_sw128(sb), bh = sdesc_sw128(sb + TF_A_BYTES);
                    const uint64_t al = sdesc_sw128(sb + T::HALF_BYTES);
                    const uint64_t bl = sdesc_sw128(sb + T::HALF_BYTES + TF_A_BYTES);
                    const uint32_t dt = tmem + (uint32_t)(stage * T::BN);
#pragma unroll
                    for (int k = 0; k < TF_BK / 8; ++k) {  // 8 columns of n: 32 bytes along the swizzle row
                        const uint64_t off = (uint64_t)((k * 32) >> 4);
                        mma_tf32(dt, ah + off, bl + off, idesc, k ? 1u : 0u);
                        mma_tf32(dt, al + off, bh + off, idesc, 1u);
                    }
#pragma unroll
                    for (int k = 0; k < TF_BK / 8; ++k) {
                        const uint64_t off = (uint64_t)((k * 32) >> 4);
                        mma_tf32(dt, ah + off, bh + off, idesc, 1u);
                    }
                    mma_commit(&sh.done[stage]);
                    if (++stage == nst) { stage = 0; ph ^= 1u; }
                }
            }
            if (*abort_flag) {
                // every MMA this thread issued completes before the accumulators are freed
                mma_commit(&sh.drain);
                mbar_wait_drain(&sh.drain, 0);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(TF_REGS_ACC));
        // lane quarter q of TMEM = 32 atoms of the tile; the two warpgroups take the tile's
        // 16-signal blocks in turn
        const int q = warp & 3, grp = (warp - 12) >> 2;
        const int nblk = w / 16;
        int stage = 0;
        uint32_t ph = 0;
        unsigned tcount = 0;
        bool ok = true;
        long long t = blockIdx.x;
        // a tile with scores to recompute ends the inner loop: their code between its instructions, or a
        // call among them, costs the accumulation 1 to 3 % (777 x 6001 x 99, 2048 x 32768 x 128)
        for (;;) {
            int flag_slot = -1;
            for (; t < ntiles && flag_slot < 0; t += gridDim.x, ++tcount) {
                const int tm = (int)(t / tiles_n), tn = (int)(t - (long long)tm * tiles_n);
                float acc[T::BN / 32][16];
#pragma unroll
                for (int i = 0; i < T::BN / 32; ++i)
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[i][e] = 0.f;
                for (int kb = 0; kb < nk; ++kb) {
                    ok = true;
                    if (lane == 0) ok = mbar_wait(&sh.done[stage], ph, abort_flag);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                    if (!ok) { if (lane == 0) give_up(); break; }
                    fence_after();
                    const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(stage * T::BN);
#pragma unroll
                    for (int i = 0; i < T::BN / 32; ++i) {
                        if (2 * i + grp < nblk) {
                            float v[16];
                            tmem_ld16(tb + (uint32_t)((2 * i + grp) * 16), v);
#pragma unroll
                            for (int e = 0; e < 16; ++e) acc[i][e] += v[e];
                        }
                    }
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.tempty[stage]);
                    if (++stage == nst) { stage = 0; ph ^= 1u; }
                }
                if (!ok) break;
                const int slot = tcount & (TF_SLOTS - 1);
                const int ar = q * 32 + lane;
                const int atom = tm * TF_BM + ar;
                bool flagged = false;
#pragma unroll
                for (int l = 0; l < TF_LOADERS; ++l) flagged |= sh.any[slot][l] != 0;
#pragma unroll
                for (int i = 0; i < T::BN / 32; ++i) {
                    if (2 * i + grp < nblk) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const int col = (2 * i + grp) * 16 + e;
                            const int k = tn * w + col;
                            if (k < act_n && atom < m) d.Cs[(size_t)k * m + atom] = acc[i][e];
                        }
                    }
                }
                if (flagged) flag_slot = slot;
            }
            if (flag_slot >= 0) {
                const long long tp = t - gridDim.x;
                const int tm = (int)(tp / tiles_n);
                chain_tile<VEC>(d, sh, cur, flag_slot, tm, (int)(tp - (long long)tm * tiles_n), w, act_n);
                continue;
            }
            if (!ok) unfinished(d, t, ntiles, tiles_n, w, act_n);
            break;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == TF_MMA_WARP) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TF_TMEM));
    }
}

// The registers that setmaxnreg hands out come from the launch's own: 5 x 128 threads at numRegs.
bool regs_cover(const cudaFuncAttributes& a) { return 5 * a.numRegs >= 2 * TF_REGS_ACC + 3 * TF_REGS_LOAD; }

template <bool VEC, bool NARROW>
cudaError_t launch_t(const Dev& d, int cur, int act_n_ub, int sms, cudaStream_t s) {
    // (per launch: the attribute belongs to the current context; about a microsecond of host time)
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, k_corr_tf32<VEC, NARROW>);
    if (e != cudaSuccess) return e;
    if (!regs_cover(fa)) return cudaErrorNotSupported;
    e = cudaFuncSetAttribute(k_corr_tf32<VEC, NARROW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TF_SMEM);
    if (e != cudaSuccess) return e;
    // one CTA per SM; tiles of 16 signals are the narrowest
    const long long tiles = (long long)((d.m + TF_BM - 1) / TF_BM) * ((act_n_ub + 15) / 16);
    const int grid = (int)(tiles < sms ? tiles : sms);
    return launch_chain(k_corr_tf32<VEC, NARROW>, dim3(grid), dim3(TF_THREADS), TF_SMEM, s, d, cur);
}

}  // namespace

cudaError_t launch_corr_tf32(const Dev& d, int cur, int act_n_ub, cudaStream_t s, int64_t* nl) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // The narrow kernel where its tiles run side by side (1024 x 8192 x 256: 50 -> 46 us, the solve
    // 1.084 -> 1.052 ms); else one wide tile beats two narrow ones in turn (2048 x 32768 x 256: 245 us
    // against 320).
    const long long tiles_m = (d.m + TF_BM - 1) / TF_BM;
    const bool narrow = act_n_ub <= TF_NARROW || tiles_m * ((act_n_ub + TF_NARROW - 1) / TF_NARROW) <= sms;
    if ((d.n & 3) == 0) e = narrow ? launch_t<true, true>(d, cur, act_n_ub, sms, s) : launch_t<true, false>(d, cur, act_n_ub, sms, s);
    else e = narrow ? launch_t<false, true>(d, cur, act_n_ub, sms, s) : launch_t<false, false>(d, cur, act_n_ub, sms, s);
    if (e != cudaSuccess) return e;
    ++*nl;
    return cudaSuccess;
}

}  // namespace mpl

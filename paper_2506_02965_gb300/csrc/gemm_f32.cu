// fp32 grouped GEMMs on the tensor cores, for the fp32 configuration: all six expert
// contractions, the router logits of pools over 64 experts and the router's input
// gradient. Same argument meaning as the bf16 kernels (moe_internal.h).
//
// A TF32 product, or a two-way split, would not hold fp32 results. Here every fp32 operand
// value is split exactly into three bf16 values, x = h + m + l (each the bf16 nearest to
// what the ones before left: 3 x 8 bits of significand cover fp32's 24), and a product is
// the sum of the six bf16 products hh, hm, mh, mm, hl, lh; the three left out are below
// 2^-25 of it. Both operands are multiplied by 2^23 before the split and the sums by 2^-46
// after it, which changes no digit: the last bit of the smallest fp32 number, 2^-149, becomes
// bf16's smallest normal number, so that the split is exact down to zero. (Unscaled it was not
// below 2^-110: 6e-5 off for operands of 2^-120.) The tensor core's fp32 accumulator truncates, which over a long contraction
// loses more than an FFMA chain does, so an accumulator holds only 32 contraction terms
// (the smallest products first) and is then added to fp32 registers with round-to-nearest.
// Measured against 64 bits, the worst tensor of a whole fp32 step is 4.2e-7 (512 tokens, d = 256,
// F = 512) and 3.1e-7 (1501 tokens, d = 1000, F = 1366) off, where the FFMA kernels that this
// replaces were 8.7e-7 and 1.2e-6 off on the same inputs (another seed: 2.5e-7 and 3.1e-7 for
// 7.1e-7 and 1.3e-6). Accumulators of 64 terms (1.5% faster) were further off than those.
//
// Roles (one persistent CTA per SM, 128 x BN tiles): 16 producer warps copy fp32 into
// shared memory up to two stages ahead (cp.async), split it and write three swizzled bf16
// planes per operand into a ring of two 32-deep stages; one warp issues the 12 MMAs of a
// stage into one of four TMEM accumulators; 8 warps add the accumulators into registers and
// run the epilogue. cp.async and not TMA because lines need only 4-byte alignment (any d_ff).
//
// What bounds it: no single unit. A 32-deep stage of a 128 x 128 tile is 32 KB of fp32 written and
// read, 48 KB of planes written, and 96 KB of operand reads by the MMAs; in the counters
// instructions issue in 56-66% of the cycles (most of them the split's), loads and stores take
// 33-44% of the shared-memory wavefronts, the tensor pipe is 24-35% busy, DRAM 4-9%. (Accumulating
// an eighth as often, or issuing one MMA of six, changed the time by 10% and 4%.) Whole fp32 steps:
// 1501 tokens, d = 1000, F = 1366, E = 6, k = 3: 5.40 -> 1.14 ms (21 -> 97 TFLOP/s);
// 512 tokens, d = 256, F = 512, E = 8, k = 2: 494 -> 128 us.
//
// An infinite or NaN operand makes 0 * inf terms in the split, and operands from 2^105 or sums
// from 2^82 on leave the scaled range, so an output element that is not finite is computed
// again by a plain fp32 FMA chain, which gives IEEE results (repair).
#include <algorithm>
#include <type_traits>

#include "moe_internal.h"
#include "tc_ptx.cuh"

namespace moe {
namespace f32 {

using namespace tc;

constexpr int FK = 32;                // contraction terms per stage (and per accumulator)
constexpr int PROD_WARPS = 16, EPI_W = 8;
constexpr int EPI_WARP0 = PROD_WARPS, MMA_WARP = PROD_WARPS + EPI_W;
// whole warpgroups, whose registers are split by role: 16 x 64 + 8 x 112 + 4 x 24 registers
// a lane is exactly the 28 x 72 of the launch (the warps after the MMA warp are idle)
constexpr int NTHREADS = 32 * (PROD_WARPS + EPI_W + 4);
constexpr int REG_PROD = 64, REG_EPI = 112, REG_MMA = 24;
template <int R>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R)); }
template <int R>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R)); }
constexpr int NBUF = 4;               // TMEM accumulators in flight
constexpr int FMAX_GROUPS = 256;
constexpr int ST_FLOATS = 32 * 32;    // transposition buffer per epilogue warp

struct Params {
    GroupRows rows;
    int G;
    const int32_t* gexp;
    const float* a;
    const float* b;
    int64_t b_group_elems;
    int M, N, K;  // M: output rows per group (K-variable); K: contraction (M-variable)
    float* out0;
    float* out1;
    const float* aux;
    uint64_t wait_ns;
    int vec_a, vec_b;  // floats per copy along a contiguous line of each operand (4, 2 or 1)
};

constexpr uint32_t plane_a() { return BM * FK * 2; }
constexpr uint32_t plane_b(int bn) { return (uint32_t)bn * FK * 2; }
constexpr uint32_t stage_bytes(int bn) { return 3 * (plane_a() + plane_b(bn)); }
constexpr int NST = 2;                // bf16 stages (the MMAs of one, the split into the other)
constexpr int NRAW = 2;               // fp32 stages: copies in flight ahead of the split (three: no faster)
constexpr uint32_t raw_bytes() { return PROD_WARPS * 2048; }  // a block of each operand per warp
constexpr uint32_t smem_bytes(int bn) {
    return 1024 + NST * stage_bytes(bn) + NRAW * raw_bytes() + EPI_W * ST_FLOATS * 4;
}
static_assert(smem_bytes(128) + 2048 <= 227 * 1024, "shared memory of one SM");

struct Tile {
    int g, we, m0, n0, mrows, klen;
    int64_t a0, b0, o0;
};

// Asynchronous copy of W floats from global to shared memory, of which the first `bytes`
// are read and the rest are zero-filled (bytes = 0: nothing is read).
template <int W>
__device__ __forceinline__ void cp_async(uint32_t dst, const float* src, int bytes) {
    if constexpr (W == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(bytes), "n"(4 * W)
                     : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr float kSplitScale = 8388608.f;         // 2^23
constexpr float kSumScale = 0x1p-46f;            // of a product of two scaled operands
// 8 values -> the three bf16 planes of 2^23 x = h + m + l, 16 bytes each
__device__ __forceinline__ void split8(const float* v, uint4* h, uint4* m, uint4* l) {
    uint32_t* hp = reinterpret_cast<uint32_t*>(h);
    uint32_t* mp = reinterpret_cast<uint32_t*>(m);
    uint32_t* lp = reinterpret_cast<uint32_t*>(l);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 hh = __hmul2(__floats2bfloat162_rn(v[2 * i], v[2 * i + 1]), __float2bfloat162_rn(kSplitScale));
        const uint32_t hu = *reinterpret_cast<const uint32_t*>(&hh);
        const float r0 = fmaf(v[2 * i], kSplitScale, -__uint_as_float(hu << 16)),
                    r1 = fmaf(v[2 * i + 1], kSplitScale, -__uint_as_float(hu & 0xffff0000u));
        const __nv_bfloat162 mm = __floats2bfloat162_rn(r0, r1);
        const uint32_t mu = *reinterpret_cast<const uint32_t*>(&mm);
        const __nv_bfloat162 ll =
            __floats2bfloat162_rn(r0 - __uint_as_float(mu << 16), r1 - __uint_as_float(mu & 0xffff0000u));
        hp[i] = hu;
        mp[i] = mu;
        lp[i] = *reinterpret_cast<const uint32_t*>(&ll);
    }
}

__device__ __forceinline__ bool is_finite(float v) { return fabsf(v) <= 3.402823466e38f; }
// A warp's outputs by plain chains of FMAs in order of k: y = lane l's row (of `rows` at A) times
// RC columns (of `cols` at B). Eight k of both operands at a time go through st, the next eight
// are in flight meanwhile. Stops early once every wanted output (a bit per column) is NaN, which
// it then stays.
template <bool A_MN, bool B_MN, int RC>
__device__ __forceinline__ void fma_chains(const float* A, int64_t lda, int rows, const float* B, int64_t ldb, int cols,
                                           int klen, uint32_t want, float* st, float (&y)[RC]) {
    constexpr int RK = 8, NB = RK * RC / 32, LDB = RC + 4, LDA = RK + 4;
    static_assert(RK * LDB + 32 * LDA <= ST_FLOATS, "a warp's buffer");
    const int lane = threadIdx.x & 31;
    float* sa = st + RK * LDB;  // [32][LDA], after B's [RK][LDB]
    float a[RK], b[NB];
    auto fetch = [&](int k0) {
        // A: lane's row (MN: contiguous over the lanes), or four rows of RK consecutive k at a time
#pragma unroll
        for (int i = 0; i < RK; ++i) {
            const int r = A_MN ? lane : 4 * i + lane / RK, k = k0 + (A_MN ? i : lane % RK);
            a[i] = r < rows && k < klen ? A[A_MN ? k * lda + r : r * lda + k] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int j = lane + 32 * i, k = k0 + (B_MN ? j / RC : j % RK), c = B_MN ? j % RC : j / RK;
            b[i] = c < cols && k < klen ? B[B_MN ? k * ldb + c : c * ldb + k] : 0.f;
        }
    };
#pragma unroll
    for (int i = 0; i < RC; ++i) y[i] = 0.f;
    fetch(0);
#pragma unroll 1
    for (int k0 = 0; k0 < klen; k0 += RK) {
        __syncwarp();  // the values before these have been read
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int j = lane + 32 * i;
            st[B_MN ? j / RC * LDB + j % RC : j % RK * LDB + j / RK] = b[i];
        }
#pragma unroll
        for (int i = 0; i < RK; ++i) sa[A_MN ? lane * LDA + i : (4 * i + lane / RK) * LDA + lane % RK] = a[i];
        __syncwarp();
        fetch(k0 + RK);
#pragma unroll
        for (int k = 0; k < RK; k += 4) {
            float x[4];
            Vec<float>::load(sa + lane * LDA + k, x);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < RC; i += 4) {
                    float w[4];
                    Vec<float>::load(st + (k + q) * LDB + i, w);
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[i + j] = fmaf(x[q], w[j], y[i + j]);
                }
        }
        if (k0 % (4 * RK) == 0) {
            uint32_t open = 0;
#pragma unroll
            for (int i = 0; i < RC; ++i) open |= y[i] == y[i] ? 1u << i : 0u;
            if (!__any_sync(0xffffffffu, open & want)) break;
        }
    }
}

// The outputs of an epilogue warp (rows mrow.. of the tile, columns col0.. of either half) that it
// has stored as not finite, computed again and stored: after the warp's last tile, when nothing
// else is in registers, so that it costs the other outputs nothing. (dG and dU are not finite
// where dA is not; a finite dA beside a G or U that is not comes out within rounding.) A, B: the
// operands of the tile's group; out_row: the output row of its first. One chain per output costs
// about what the FFMA kernel that this replaces took for any values: a step of 1501 tokens, d =
// 1000, F = 1366 of which nearly all sums leave the range 4.1 to 7.2 ms (5.4 before; finite 1.13);
// NaN stop early, 1.6 to 1.9 ms for all, 3.4 for a single one in dY.
template <bool A_MN, bool B_MN, int EPI, int BN>
static __device__ __forceinline__ void repair(const Params& p, const float* A, const float* B, int64_t out_row, int n0, int mrow,
                                       int mrows, int klen, int col0, float* st) {
    constexpr int RC = BN / 4;  // the warp's columns of one half
    constexpr bool GU = EPI != EPI_STORE;  // outputs (gate, up) of a feature
    const int lane = threadIdx.x & 31, F = EPI == EPI_SWIGLU_FWD ? p.N / 2 : p.N;
    const int64_t lda = A_MN ? p.M : p.K, ldb = B_MN ? p.N : p.K;
    float* out = p.out0 + (out_row + mrow + lane) * (GU ? 2 * F : F);
    const bool row_ok = mrow + lane < mrows;
    __syncwarp();  // the warp's stores before these
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
        // RC columns from f on: features, or (forward) their gates or ups, rows n.. of B
        const int f = n0 + col0 + (EPI == EPI_SWIGLU_FWD ? 0 : u * (BN / 2)), n = f + (EPI == EPI_SWIGLU_FWD ? u * F : 0);
        const int cols = min(RC, F - f);
        uint32_t want = 0;
        if (row_ok)
            for (int i = 0; i < cols; ++i)
                if (!is_finite(out[n + i]) || (EPI == EPI_SWIGLU_BWD && !is_finite(out[F + n + i]))) want |= 1u << i;
        if (!__any_sync(0xffffffffu, want)) continue;
        float y[RC];
        fma_chains<A_MN, B_MN, RC>(A + (A_MN ? mrow : mrow * lda), lda, mrows - mrow, B + (B_MN ? n : n * ldb), ldb, cols, klen, want,
                               st, y);
#pragma unroll
        for (int i = 0; i < RC; ++i) {
            if (!((want >> i) & 1u)) continue;
            if constexpr (EPI == EPI_SWIGLU_BWD) {
                const float* gu = p.aux + (out_row + mrow + lane) * 2 * F + n + i;
                const float G = gu[0], U = gu[F], sg = sigmoidf_(G);
                out[F + n + i] = y[i] * G * sg;
                out[n + i] = y[i] * U * sg * (1.f + G * (1.f - sg));
            } else {
                out[n + i] = y[i];
                if constexpr (EPI == EPI_SWIGLU_FWD) {  // (gates come before ups: the last to change)
                    const float G = out[f + i], U = out[F + f + i];
                    p.out1[(out_row + mrow + lane) * F + f + i] = G * sigmoidf_(G) * U;
                }
            }
        }
    }
    __syncwarp();
}

template <bool A_MN, bool B_MN, bool VAR_K, int EPI, int BN>
__global__ void __launch_bounds__(NTHREADS, 1) gemm_f32_kernel(const __grid_constant__ Params p) {
    pdl_begin();
    static_assert(BN == 64 || BN == 128, "tile widths");
    constexpr uint32_t STAGE = stage_bytes(BN);
    constexpr int CW = BN / 4;       // an epilogue warp owns CW columns of each half of the tile
    constexpr int B_BLOCKS = BN * FK / 256;  // blocks of 256 values of B per stage
    static_assert(BM * FK / 256 == PROD_WARPS && B_BLOCKS <= PROD_WARPS, "one block of each operand per warp");
    constexpr uint32_t IDESC = instr_desc<BN, false, false, BM>();

    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * NST + 2 * NBUF + 1];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_tile_start[FMAX_GROUPS + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &s_abort;
    const uint32_t raw_u32 = smem_u32(smem_raw);
    const uint32_t ring = raw_u32 + ((1024u - (raw_u32 & 1023u)) & 1023u);
    uint8_t* ring_ptr = smem_raw + (ring - raw_u32);
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (NST + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * NST + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * NST + NBUF + b); };
    const uint32_t drain_bar = bar0 + 8u * (2 * NST + 2 * NBUF);

    const int F = EPI == EPI_SWIGLU_FWD ? p.N / 2 : p.N;
    const int tiles_n = EPI == EPI_SWIGLU_FWD ? (F + BN / 2 - 1) / (BN / 2) : (p.N + BN - 1) / BN;
    auto group_rows = [&](int g) { return p.rows.offsets ? p.rows.offsets[g + 1] - p.rows.offsets[g] : p.rows.rows; };
    if (warp == 0) {  // tiles before each group
        int run = 0;
        for (int g0 = 0; g0 < p.G; g0 += 32) {
            const int g = g0 + lane;
            int n = 0;
            if (g < p.G) n = (VAR_K ? (p.M + BM - 1) / BM : (max(group_rows(g), 0) + BM - 1) / BM) * tiles_n;
            int inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (g < p.G) s_tile_start[g] = run + inc - n;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) s_tile_start[p.G] = run;
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            s_abort = 0;
            for (int s = 0; s < NST; ++s) {
                mbar_init(full_bar(s), PROD_WARPS);
                mbar_init(empty_bar(s), 1);
            }
            for (int b = 0; b < NBUF; ++b) {
                mbar_init(tfull_bar(b), 1);
                mbar_init(tempty_bar(b), EPI_W);
            }
            mbar_init(drain_bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(NBUF * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = s_tmem;
    const int total = s_tile_start[p.G];

    // bounded wait of a whole warp (inlined: a call would spill the accumulators around it)
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
        bool ok = mbar_try(bar, parity);
        if (!ok) {
            const uint64_t t0 = gtimer();
            while (!(ok = mbar_try(bar, parity)) && !*abort_flag) {
                if (gtimer() - t0 > p.wait_ns) {
                    *abort_flag = 1;
                    record_status(MOE_ERR_TIMEOUT);
                }
            }
        }
        return __all_sync(0xffffffffu, ok);
    };
    // M-tiles innermost: the CTAs of a round share the tile columns of B
    auto tile_at = [&](int t) -> Tile {
        int lo = 0, hi = p.G - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_tile_start[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        Tile ti;
        ti.g = lo;
        ti.we = p.gexp ? p.gexp[lo] : lo;
        const int local = t - s_tile_start[lo], mt = (s_tile_start[lo + 1] - s_tile_start[lo]) / tiles_n;
        ti.m0 = (local % mt) * BM;
        ti.n0 = (local / mt) * (EPI == EPI_SWIGLU_FWD ? BN / 2 : BN);
        const int rows = group_rows(lo);
        if (p.rows.offsets) {
            ti.a0 = ti.b0 = ti.o0 = p.rows.offsets[lo];
        } else {
            ti.a0 = (int64_t)lo * p.rows.a_stride;
            ti.b0 = (int64_t)lo * p.rows.b_stride;
            ti.o0 = (int64_t)lo * p.rows.out_stride;
        }
        ti.mrows = VAR_K ? p.M : rows;
        ti.klen = VAR_K ? max(rows, 0) : p.K;
        return ti;
    };
    auto a_base = [&](const Tile& ti) { return p.a + ti.a0 * (VAR_K ? p.M : p.K); };
    auto b_base = [&](const Tile& ti) { return VAR_K ? p.b + ti.b0 * p.N : p.b + (int64_t)ti.we * p.b_group_elems; };
    // weight row of tile column c (SwiGLU forward: BN / 2 gate features, then their up rows)
    auto b_row = [&](const Tile& ti, int c) -> int {
        if (EPI == EPI_SWIGLU_FWD) return c < BN / 2 ? ti.n0 + c : F + ti.n0 + c - BN / 2;
        return ti.n0 + c;
    };

    if (warp < PROD_WARPS) {
        // ------------------------------------------------------------ producers
        // A warp moves one block of 256 values of each operand per stage, 8 outer x 32 inner
        // (inner: the dimension that is contiguous in memory, k or the operand rows), with
        // cp.async into its own part of the fp32 ring, up to NRAW stages ahead, and splits it
        // when it has landed: lane l then holds 8 consecutive k of one operand row (MN: row
        // l of 32, else row l / 4 of 8).
        reg_dec<REG_PROD>();
        const bool has_b = warp < B_BLOCKS;
        const uint32_t raw = ring + NST * STAGE + warp * 2048;
        const uint8_t* raw_ptr = ring_ptr + NST * STAGE + warp * 2048;
        // the block's first operand row and first k
        const int arow = A_MN ? 32 * (warp % (BM / 32)) : 8 * warp, ak = A_MN ? 8 * (warp / (BM / 32)) : 0;
        const int brow = B_MN ? 32 * (warp % (BN / 32)) : 8 * warp, bk = B_MN ? 8 * (warp / (BN / 32)) : 0;
        const int64_t lda = A_MN ? p.M : p.K, ldb = B_MN ? p.N : p.K;
        const int per_a = 32 / p.vec_a, per_b = 32 / p.vec_b;  // lanes per contiguous line
        const int oa = lane / per_a, ia = (lane % per_a) * p.vec_a, ob = lane / per_b, ib = (lane % per_b) * p.vec_b;
        int t = (int)blockIdx.x - (int)gridDim.x, left = 0;
        const float *src_a = nullptr, *src_b = nullptr;  // this lane's first element of the block
        bool has_rows = false, has_cols = false;  // whether this warp's blocks of the tile hold anything
        int lim_a = 0, lim_b = 0;  // outer lines with data past the lane's (K-contiguous), or whether the column has any
        auto seek = [&]() -> bool {  // the next stage: of this tile, or of the next one with work
            if ((left -= FK) > 0) {
                src_a += A_MN ? FK * lda : FK;
                src_b += B_MN ? FK * ldb : FK;
                return true;
            }
            while ((t += gridDim.x) < total) {
                const Tile ti = tile_at(t);
                left = ti.klen;
                if (left <= 0) continue;
                has_rows = ti.m0 + arow < ti.mrows;
                const int ra = ti.m0 + arow + (A_MN ? ia : oa);
                lim_a = A_MN ? (ra < ti.mrows ? 1 : 0) : ti.mrows - ra;
                src_a = a_base(ti) + (A_MN ? (ak + oa) * lda + ra : ra * lda + ia);
                if (has_b) {
                    const int c = brow + (B_MN ? ib : ob);
                    const int rb = b_row(ti, c), end = EPI == EPI_SWIGLU_FWD ? (c < BN / 2 ? F : 2 * F) : p.N;
                    lim_b = B_MN ? (rb < end ? 1 : 0) : end - rb;
                    src_b = b_base(ti) + (B_MN ? (bk + ob) * ldb + rb : rb * ldb + ib);
                    has_cols = b_row(ti, brow) < end;
                }
                return true;
            }
            return false;
        };
        // copy one block, W floats a copy: outer lines o0, o0 + 32 / PER, ... (a copy that reads
        // nothing names the operand's base, which is aligned to W: addresses are checked all the same)
        auto copy_block = [&](auto mnc, auto wc, const float* base, const float* src, int64_t ld, int o, int in, int k0,
                              int lim, uint32_t dst) {
            constexpr bool MN = decltype(mnc)::value;
            constexpr int W = decltype(wc)::value, STEP = W;  // 32 / (32 / W) lines per copy
            // K-contiguous lines are swizzled so that the 32-byte reads below spread over the banks
            dst += o * 128 + in * 4;
            const int nk = MN ? left - k0 - o : 4 * max(0, min(W, left - in));
#pragma unroll
            for (int o0 = 0; o0 < 8; o0 += STEP) {
                const int n = MN ? (lim && o0 < nk ? 4 * W : 0) : (o0 < lim ? nk : 0);
                const uint32_t at = dst + o0 * 128;
                cp_async<W>(MN ? at : at ^ (((o + o0) & 1) << 4), n ? src + o0 * ld : base, n);
            }
        };
        auto copy_op = [&](auto mnc, int vec, const float* base, const float* src, int64_t ld, int o, int in, int k0, int lim,
                           uint32_t dst) {
            if (vec == 4) copy_block(mnc, std::integral_constant<int, 4>{}, base, src, ld, o, in, k0, lim, dst);
            else if (vec == 2) copy_block(mnc, std::integral_constant<int, 2>{}, base, src, ld, o, in, k0, lim, dst);
            else copy_block(mnc, std::integral_constant<int, 1>{}, base, src, ld, o, in, k0, lim, dst);
        };
        auto issue = [&](int slot) {
            const uint32_t dst = raw + slot * raw_bytes();
            if (has_rows) copy_op(std::integral_constant<bool, A_MN>{}, p.vec_a, p.a, src_a, lda, oa, ia, ak, lim_a, dst);
            if (has_cols) copy_op(std::integral_constant<bool, B_MN>{}, p.vec_b, p.b, src_b, ldb, ob, ib, bk, lim_b, dst + 1024);
        };
        // split one landed block into the three planes at d
        auto split_block = [&](auto mnc, const uint8_t* q, uint8_t* d, uint32_t plane) {
            float v[8];
            if constexpr (decltype(mnc)::value) {
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const float*>(q + u * 128 + lane * 4);
            } else {
                const uint8_t* ln = q + (lane >> 2) * 128;
                const int w = (lane & 3) * 32, x = ((lane >> 2) & 1) << 4;
                Vec<float>::load(reinterpret_cast<const float*>(ln + (w ^ x)), v);
                Vec<float>::load(reinterpret_cast<const float*>(ln + ((w + 16) ^ x)), v + 4);
            }
            uint4 h, m, l;
            split8(v, &h, &m, &l);
            *reinterpret_cast<uint4*>(d) = h;
            *reinterpret_cast<uint4*>(d + plane) = m;
            *reinterpret_cast<uint4*>(d + 2 * plane) = l;
        };
        auto plane_at = [&](int i, int kc) { return i * 64 + ((kc ^ ((i >> 1) & 3)) << 4); };
        const uint32_t da = plane_at(arow + (A_MN ? lane : lane >> 2), A_MN ? ak >> 3 : lane & 3);
        const uint32_t db = 3 * plane_a() + plane_at(brow + (B_MN ? lane : lane >> 2), B_MN ? bk >> 3 : lane & 3);
        bool more = seek();
        int slot_in = 0, slot = 0, ahead = 0;  // stages copied and not yet split
        uint32_t phase = 0;
        uint32_t held = 0;  // two bits per slot: has_rows, has_cols of the stage in it
        int stage = 0;
        for (;;) {
            while (more && ahead < NRAW) {
                issue(slot_in);
                cp_commit();
                held = (held & ~(3u << (2 * slot_in))) | ((uint32_t)has_rows | ((uint32_t)has_cols << 1)) << (2 * slot_in);
                slot_in = slot_in + 1 == NRAW ? 0 : slot_in + 1;
                ++ahead;
                more = seek();
            }
            if (!ahead) break;
            if (ahead == NRAW) cp_wait<NRAW - 1>();
            else cp_wait<0>();  // the last stages
            __syncwarp();
            if (!wait(empty_bar(stage), phase ^ 1u)) break;
            uint8_t* sa = ring_ptr + (size_t)stage * STAGE;
            const uint8_t* rp = raw_ptr + slot * raw_bytes();
            // (blocks past the operand's rows stay as they are: their accumulators are not stored)
            if ((held >> (2 * slot)) & 1u) split_block(std::integral_constant<bool, A_MN>{}, rp, sa + da, plane_a());
            if ((held >> (2 * slot)) & 2u) split_block(std::integral_constant<bool, B_MN>{}, rp + 1024, sa + db, plane_b(BN));
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(full_bar(stage));
            --ahead;
            slot = slot + 1 == NRAW ? 0 : slot + 1;
            if (++stage == NST) {
                stage = 0;
                phase ^= 1u;
            }
        }
        cp_wait<0>();  // after an abort: copies in flight
    } else if (warp >= MMA_WARP) {
        // ------------------------------------------------------------ MMA issuer
        reg_dec<REG_MMA>();
        if (warp == MMA_WARP) {
            int stage = 0, b = 0;
            uint32_t phase = 0, bphase = 0;
            bool ok = true, issued = false;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                const int kiters = (tile_at(t).klen + FK - 1) / FK;
                for (int kb = 0; kb < kiters; ++kb) {
                    ok = wait(tempty_bar(b), bphase ^ 1u) && wait(full_bar(stage), phase);
                    if (!ok) break;
                    fence_after();
                    if (lane == 0) {
                        const uint32_t sa = ring + stage * STAGE, sb = sa + 3 * plane_a();
                        constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
    #pragma unroll
                        for (int q = 0; q < 6; ++q)
    #pragma unroll
                            for (int kk = 0; kk < FK / 16; ++kk)
                                mma_bf16(tmem_base + b * BN, smem_desc_sw64(sa + pa[q] * plane_a() + kk * 32),
                                         smem_desc_sw64(sb + pb[q] * plane_b(BN) + kk * 32), IDESC, (q | kk) ? 1u : 0u);
                        mma_commit(empty_bar(stage));
                        mma_commit(tfull_bar(b));
                    }
                    issued = true;
                    __syncwarp();
                    if (++stage == NST) {
                        stage = 0;
                        phase ^= 1u;
                    }
                    if (++b == NBUF) {
                        b = 0;
                        bphase ^= 1u;
                    }
                }
            }
            if (lane == 0 && issued) {
                // every MMA issued has completed before TMEM is released, also when another role
                // gives up only after this one is through
                mma_commit(drain_bar);
                const uint64_t limit = p.wait_ns > 200000000ull ? p.wait_ns : 200000000ull, t0 = gtimer();
                while (!mbar_try(drain_bar, 0) && gtimer() - t0 < limit) {
                }
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------ accumulate, epilogue
        reg_inc<REG_EPI>();
        const int q = warp & 3, hc = (warp - EPI_WARP0) >> 2;  // TMEM lane quarter, column half
        float* st = reinterpret_cast<float*>(ring_ptr + NST * STAGE + NRAW * raw_bytes()) + (warp - EPI_WARP0) * ST_FLOATS;
        int b = 0;
        uint32_t bphase = 0;
        float odd = 0.f;  // NaN once this lane has seen an output that is not finite
        for (int t = blockIdx.x; t < total; t += gridDim.x) {
            const Tile ti = tile_at(t);
            const int kiters = (ti.klen + FK - 1) / FK;
            float acc[2][CW];
#pragma unroll
            for (int c = 0; c < CW; ++c) acc[0][c] = acc[1][c] = 0.f;
            bool ok = true;
            for (int kb = 0; kb < kiters; ++kb) {
                ok = wait(tfull_bar(b), bphase);
                if (!ok) break;
                fence_after();
                const uint32_t tb = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN + hc * CW);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float v[CW];
                    if constexpr (CW == 32) tmem_ld32(tb + u * (BN / 2), v);
                    else tmem_ld16(tb + u * (BN / 2), v);
#pragma unroll
                    for (int c = 0; c < CW; ++c) acc[u][c] += v[c];
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty_bar(b));
                if (++b == NBUF) {
                    b = 0;
                    bphase ^= 1u;
                }
            }
            if (!ok) break;
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                acc[0][c] *= kSumScale;
                acc[1][c] *= kSumScale;
            }
            const int mrow = ti.m0 + q * 32;
            // transpose through shared memory (32 rows x 32 columns at a time): lanes then run
            // along the columns, so that loads and stores are coalesced
            auto put = [&](int at, float v) { st[lane * 32 + (at ^ lane)] = v; };
            auto get = [&](int r, int at) { return st[r * 32 + (at ^ r)]; };
            // Eight rows at a time, so that their loads and stores overlap. (Row by row, with a check
            // for non-finite values at every element, a tile's epilogue took 8 us: the weight
            // gradients of experts with few rows are all epilogue, dW2 of 78 experts of d = 1928,
            // F = 591 at 10 rows took 362 us, now 173; dA waited for G and U row by row, 4503 rows
            // of d = 1000, F = 1366 258 -> 163 us.)
            if constexpr (EPI == EPI_SWIGLU_FWD) {
                // 16 gate columns beside the 16 up columns of the same features; a half-warp per row
#pragma unroll
                for (int c0 = 0; c0 < CW; c0 += 16) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        put(i, acc[0][c0 + i]);
                        put(16 + i, acc[1][c0 + i]);
                    }
                    __syncwarp();
                    const int c = lane & 15, f = ti.n0 + hc * CW + c0 + c;
#pragma unroll 1
                    for (int i0 = 0; i0 < 16; i0 += 8) {
                        const int m0 = mrow + 2 * i0 + (lane >> 4);  // rows m0, m0 + 2, ...
                        float G[8], U[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int r = 2 * (i0 + i) + (lane >> 4);
                            G[i] = get(r, c);
                            U[i] = get(r, 16 + c);
                        }
                        if (f >= F) continue;
                        float* h = p.out0 + (ti.o0 + m0) * 2 * F + f;
                        float* o = p.out1 + (ti.o0 + m0) * F + f;
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (m0 + 2 * i >= ti.mrows) break;
                            odd = fmaf(U[i], 0.f, fmaf(G[i], 0.f, odd));
                            h[(int64_t)i * 4 * F] = G[i];
                            h[(int64_t)i * 4 * F + F] = U[i];
                            o[(int64_t)i * 2 * F] = G[i] * sigmoidf_(G[i]) * U[i];
                        }
                    }
                }
            } else {
                // 32 columns at a time: one half's (CW = 32), or both halves' (CW = 16)
#pragma unroll
                for (int u = 0; u < CW / 16; ++u) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 32; ++i) put(i, CW == 32 ? acc[u][i % CW] : acc[i / CW][i % CW]);
                    __syncwarp();
                    const int n = ti.n0 + hc * CW + (CW == 32 ? u * (BN / 2) + lane : (lane >> 4) * (BN / 2) + (lane & 15));
                    const int64_t row0 = (VAR_K ? (int64_t)ti.we * p.M : ti.o0) + mrow;
#pragma unroll 1
                    for (int r0 = 0; r0 < 32 && mrow + r0 < ti.mrows; r0 += 8) {
                        const int rows = n < p.N ? min(8, ti.mrows - mrow - r0) : 0;
                        float v[8], G[8], U[8];
                        if constexpr (EPI == EPI_SWIGLU_BWD) {  // v = dA[row, n], N = F
                            const float* gu = p.aux + (row0 + r0) * 2 * F + n;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                G[i] = i < rows ? __ldg(gu + (int64_t)i * 2 * F) : 0.f;
                                U[i] = i < rows ? __ldg(gu + (int64_t)i * 2 * F + F) : 0.f;
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = get(r0 + i, lane);
                        if constexpr (EPI == EPI_SWIGLU_BWD) {
                            float* o = p.out0 + (row0 + r0) * 2 * F + n;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                if (i >= rows) break;
                                odd = fmaf(v[i], 0.f, odd);
                                const float s = sigmoidf_(G[i]);
                                o[(int64_t)i * 2 * F + F] = v[i] * G[i] * s;
                                o[(int64_t)i * 2 * F] = v[i] * U[i] * s * (1.f + G[i] * (1.f - s));
                            }
                        } else {
                            float* o = p.out0 + (row0 + r0) * p.N + n;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                if (i >= rows) break;
                                odd = fmaf(v[i], 0.f, odd);
                                o[(int64_t)i * p.N] = v[i];
                            }
                        }
                    }
                }
            }
        }
        // Outputs that are not finite are looked at again only now, when no other role of the CTA
        // waits for this one: their chains may take longer than any wait limit.
        if (__any_sync(0xffffffffu, odd != 0.f) && !*abort_flag) {
#pragma unroll 1
            for (int t = blockIdx.x; t < total; t += gridDim.x) {
                const Tile ti = tile_at(t);
                repair<A_MN, B_MN, EPI, BN>(p, a_base(ti), b_base(ti), VAR_K ? (int64_t)ti.we * p.M : ti.o0, ti.n0, ti.m0 + q * 32,
                                            ti.mrows, ti.klen, hc * CW, st);
            }
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(NBUF * BN)
                     : "memory");
}

// ------------------------------------------------------------------------ host side
// floats per copy that the lines of an operand allow: their length, the distance of its
// groups and its address are multiples of it
static int vec_of(const void* base, int64_t ld, int64_t group = 0) {
    for (int w = 4; w > 1; w /= 2)
        if (ld % w == 0 && group % w == 0 && (uintptr_t)base % (4 * w) == 0) return w;
    return 1;
}

template <bool A_MN, bool B_MN, bool VAR_K, int EPI, int BN>
static cudaError_t launch_bn(const Params& p, int64_t tiles, cudaStream_t s) {
    auto kern = gemm_f32_kernel<A_MN, B_MN, VAR_K, EPI, BN>;
    constexpr size_t smem = smem_bytes(BN);
    cudaError_t e = allow_dynamic_smem<gemm_f32_kernel<A_MN, B_MN, VAR_K, EPI, BN>>(smem);
    if (e != cudaSuccess) return e;
    // the roles' register shares must not exceed the launch's (setmaxnreg would wait forever)
    static std::atomic<int> regs{0};
    if (!regs) {
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
        regs = fa.numRegs;
    }
    if (regs * NTHREADS < 32 * (PROD_WARPS * REG_PROD + EPI_W * REG_EPI + 4 * REG_MMA)) return cudaErrorInvalidConfiguration;
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, sm_count());
    (void)launch_pdl(kern, dim3(grid), dim3(NTHREADS), smem, s, p);
    return cudaGetLastError();
}

template <bool A_MN, bool B_MN, bool VAR_K, int EPI>
static cudaError_t launch(const Params& p, int64_t mt, cudaStream_t s) {
    const int cols = EPI == EPI_SWIGLU_FWD ? p.N / 2 : p.N, per = EPI == EPI_SWIGLU_FWD ? 2 : 1;
    const int64_t wide = mt * ((cols + 128 / per - 1) / (128 / per));
    if (wide <= 0) return cudaSuccess;
    // by rounds of tiles: a 32-deep stage of a 64-wide tile takes 1.1 us, of a 128-wide one 1.45
    const int64_t narrow = mt * ((cols + 64 / per - 1) / (64 / per)), sms = sm_count();
    if ((wide + sms - 1) / sms * 145 <= (narrow + sms - 1) / sms * 110)
        return launch_bn<A_MN, B_MN, VAR_K, EPI, 128>(p, wide, s);
    return launch_bn<A_MN, B_MN, VAR_K, EPI, 64>(p, narrow, s);
}

}  // namespace f32

cudaError_t launch_gemm_m_f32(const GemmMArgs& g, cudaStream_t s) {
    using namespace f32;
    if (g.G > FMAX_GROUPS) return cudaErrorInvalidValue;
    Params p{};
    p.rows = g.rows;
    p.G = g.G;
    p.gexp = g.group_expert;
    p.a = (const float*)g.a;
    p.b = (const float*)g.b;
    p.b_group_elems = g.b_group_elems;
    p.N = g.N;
    p.K = g.K;
    p.out0 = (float*)g.out0;
    p.out1 = (float*)g.out1;
    p.aux = (const float*)g.aux;
    p.wait_ns = wait_limit_ns();
    p.vec_a = vec_of(g.a, g.K);
    p.vec_b = vec_of(g.b, g.b_kmajor ? g.K : g.N, g.b_group_elems);
    // upper bound of the M-tiles: OFFSETS groups may each end in a partial one
    const int64_t mt = g.rows.offsets ? ((int64_t)g.rows.rows + BM - 1) / BM + g.G
                                      : (int64_t)g.G * ((g.rows.rows + BM - 1) / BM);
    if (g.epi == EPI_SWIGLU_FWD) return launch<false, false, false, EPI_SWIGLU_FWD>(p, mt, s);
    if (g.epi == EPI_SWIGLU_BWD) return launch<false, true, false, EPI_SWIGLU_BWD>(p, mt, s);
    if (g.b_kmajor) return launch<false, false, false, EPI_STORE>(p, mt, s);
    return launch<false, true, false, EPI_STORE>(p, mt, s);
}

cudaError_t launch_gemm_k_f32(const GemmKArgs& g, cudaStream_t s) {
    using namespace f32;
    if (g.G > FMAX_GROUPS) return cudaErrorInvalidValue;
    Params p{};
    p.rows = g.rows;
    p.G = g.G;
    p.gexp = g.group_expert;
    p.a = (const float*)g.a;
    p.b = (const float*)g.b;
    p.M = g.M;
    p.N = g.N;
    p.out0 = (float*)g.out;
    p.wait_ns = wait_limit_ns();
    p.vec_a = vec_of(g.a, g.M);
    p.vec_b = vec_of(g.b, g.N);
    return launch<true, true, true, EPI_STORE>(p, (int64_t)g.G * ((g.M + BM - 1) / BM), s);
}

cudaError_t f32_status(cudaStream_t s, int* code) { return tu_status_read_clear(s, code); }

}  // namespace moe

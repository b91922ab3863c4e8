// Grouped expert GEMMs on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// One persistent, warp-specialised kernel template serves all six contractions of
// the SwiGLU experts (ForwardExpert / BackwardExpert of Alg. 6):
//   fwd  [G|U] = Xp W1^T (SwiGLU epilogue)      Y  = A W2^T
//   bwd  dA = dY W2 (SwiGLU-backward epilogue)  dXp = dH W1
//        dW2 = dY^T A  and  dW1 = dH^T Xp  (contraction over the expert's rows)
// Warp 0 issues TMA loads (128B-swizzled tiles) into a 4-stage shared-memory ring,
// warp 1 issues tcgen05.mma (M=128, N=BN, K=16, bf16 in, fp32 accumulate) into a
// double-buffered TMEM accumulator, warps 2-5 drain TMEM with tcgen05.ld and run
// the fused epilogue. Every mbarrier wait is bounded in time; on a timeout the CTA
// records MOE_ERR_TIMEOUT, drains its in-flight copies and MMAs, frees TMEM and
// returns.
#include <algorithm>
#include <cmath>

#include "moe_internal.h"
#include "tc_ptx.cuh"

namespace moe {
namespace tc {

constexpr int BK = 64;  // 64 bf16 = 128 bytes = one 128B-swizzle row
// Contraction rows per k-block: BK, except for the weight gradients' CTA-pair and 128-wide
// tiles, whose operands are both MN-major (64-element TMA boxes): 128-row boxes there halve
// the boxes and stage hand-offs per byte (3 stages of 64 KiB per CTA).
__host__ __device__ constexpr int kblock_rows(bool var_k, bool pair, int epi, int bn) {
    return (var_k && epi == EPI_STORE && (pair || bn == 128)) ? 128 : BK;
}
// k-blocks per operand stage: 2 for the router up to 64 experts (its stream of x is bound
// by a fixed cost per stage hand-off, so a stage carries two 64-wide boxes of each
// operand; wider B would leave too few stages), for the M-variable CTA-pair tiles
// with a store or SwiGLU-forward epilogue (three stages of 64 KiB per CTA instead of six
// of 32: the same bytes in flight, half the hand-offs, less power per flop under the
// power cap) and for the 128-wide single-CTA tiles (three stages of 64 KiB instead of six:
// dA at d = 3072, F = 640 46 -> 37 us, GEMM2 at d = 384 35 -> 28 us); else 1: the
// SwiGLU-backward pairs measured faster with six stages, and 256-wide single-CTA tiles lose
// with two stages of 96 KiB (GEMM1 47 -> 53 us)
__host__ __device__ constexpr int kblocks_per_stage(int epi, int bn, bool pair, bool var_k, bool dw2, int occ, int ar) {
    if (epi == EPI_ROUTE && ar < BM) return bn <= 32 ? 8 : 4;  // one copy each of A and B (below)
    if (epi == EPI_ROUTE) return bn <= 64 ? 2 : 1;
    if (var_k || dw2 || occ > 1) return 1;
    if (pair) return epi != EPI_SWIGLU_BWD ? 2 : 1;
    return bn == 128 ? 2 : 1;
}
// EW epilogue warps: four (one per TMEM lane quarter), or eight that halve the tile's columns,
// for contractions so short that the epilogue and not the mainloop sets a tile's time:
// weight gradients with under 384 rows a group on average (60 rows of d = 3072, F = 384, 63
// experts: dW1 89 -> 70 us, dW2 61 -> 49; 231 rows 42 -> 35; at 512 rows 80.6 -> 82), GEMM1
// and GEMM2 with contractions under 1024 (d = 384: GEMM1 50 -> 42 us; d = 1024 84 -> 86).
constexpr int kWideEpiRows = 384, kWideEpiK = 1024;
// TMA warp, MMA warp, epilogue warps
__host__ __device__ constexpr int gemm_threads(int ew) { return 64 + 32 * ew; }
constexpr int EPI_BOX = 32;                     // TMA-store box: 32 columns x 32 rows (bf16)
constexpr int EPI_BUF_BYTES = EPI_BOX * EPI_BOX * 2;
// Staging of the epilogue warps together: each has a ring of 4 output boxes (2 of eight warps;
// each box leaves by its own TMA store, so up to 3 stores are in flight while the next box is
// written), or for the SwiGLU backward 2 x (G, U) boxes. (The router-gradient partials are
// stored straight from registers.)
constexpr int EPI_BOXES = 16;
__host__ __device__ constexpr int epi_stage_bytes(int epi) { return epi == EPI_DWR ? 0 : EPI_BOXES * EPI_BUF_BYTES; }
constexpr int MAX_GROUPS = 256;

struct Params {
    const int32_t* offsets;  // OFFSETS mode when non-null
    int rows;                // UNIFORM rows per group
    int64_t a_stride, b_stride, out_stride;
    int G;
    int N;       // output columns (per group)
    int K;       // contraction length (M-variable)
    int Mout;    // output rows per group (K-variable)
    int F;       // SwiGLU inner size (SWIGLU epilogues)
    int64_t b_group_rows;  // rows of B's 2D view per group (M-variable)
    const int32_t* gexp;   // group -> expert of its weights / weight gradient, or null
    void* out0;
    void* out1;
    const void* aux;
    uint64_t wait_ns;
    // EPI_ROUTE: out0 = logits, out1 = probs (fp32 [T,E]), aux = bias [P,E] or null
    int E, k, normalize, hist_n;
    int band;  // tile order: bands of `band` M-tiles, each swept along N (set at launch)
    // operand bytes for the per-group choice of the tile order: the bytes of one A row
    // (M-variable: K elements; K-variable: Mout elements per contraction row), of one B
    // contraction row (K-variable), and of all of B (M-variable: one group's weights)
    int64_t a_row_bytes, b_row_bytes, b_all_bytes;
    int32_t* topk_idx;
    float* topk_w;
    int32_t* counts;
    // EPI_ROUTE: token rows per tile (1..BM; the A box height), so that the tiles of a
    // short batch spread over every SM (each CTA streams its rows at a per-CTA rate)
    int tile_rows;
};

// Pipeline depth: as many operand stages as fit beside the epilogue's shared memory
// (staging boxes, or the router's histogram), at most 12. OCC CTAs share one SM (OCC = 2:
// about half of the SM's 228 KiB each, for launches bound by their epilogue, whose
// stores then come from twice as many warps per SM).
__host__ __device__ constexpr int epi_extra_bytes(int epi) {
    return epi == EPI_ROUTE ? 64 * 64 * 4 : epi_stage_bytes(epi);
}
// Router tiles of at most AR < BM token rows keep only AR rows per A box in shared memory and
// fetch four or eight k-blocks of an operand in one 3D copy: a short batch, streamed by few CTAs, is
// bound by the fixed cost of its copies (90 ns each) and stages, not by bytes in flight (deeper
// rings alone changed nothing). With the epilogue below: 64 tokens, d = 2048, E = 64 24.7 -> 13.9
// us; 33, 4096, 8 22.0 -> 16.3; 4, 1024, 16 10.2 -> 7.7; 2999, 2048, 64 24.9 -> 18.7. At 4096
// tokens, d = 1024 equal (11.5), so not above 32 rows a tile, where bytes bound it.
// The MMA still reads BM rows per box: what follows the box (bytes that only reach accumulator
// rows that nobody reads), after the last box up to this many bytes past the ring.
__host__ __device__ constexpr int mma_overread(int ar) { return ar < BM ? BM * 128 : 0; }
__host__ __device__ constexpr int num_stages(uint32_t stage_bytes, int epi, int occ, int ar) {
    const int per_cta = occ == 1 ? 227 * 1024 : 112 * 1024;
    const int budget = per_cta - 1024 - 1024 - epi_extra_bytes(epi) - mma_overread(ar);  // dyn. smem, align, static
    const int n = budget / (int)stage_bytes;
    return n > 12 ? 12 : n;
}

// ------------------------------------------------------------------------ tile geometry
struct Tile {
    int g;
    int m0, n0;         // output tile origin inside the group
    int mvalid;         // rows of the group (M-variable) -> rows m0.. valid if < mvalid
    int64_t a_row;      // first A row (M-var: token row; K-var: first contraction row)
    int64_t b_row;      // K-var: first contraction row of B
    int64_t out_row;    // M-var: output row of group row 0
    int k_iters;
    int last_rows;      // K-var: valid contraction rows in the last k-block (1..64)
    bool dw;            // a tile of the second (K-variable) problem of a fused launch
    bool sec;           // a tile of the second M-variable problem (the shared experts')
    int we;             // expert whose weights (M-variable) or weight gradient (K-variable)
                        // the tile uses: group_expert[g], or g
    int ntok;           // swapped tile (below): its rows rounded up to 16, else 0
};

// Swapped tiles of the M-variable pairs. An expert's last tile holds 1 to 256 of its rows,
// but a pair's MMA always computes 256: at 512 rows an expert a fifth of all MMAs multiply
// other experts' rows that are never stored. With at most SWAP_ROWS rows the operands are
// exchanged: the weights are the MMA's 256-row operand (128 features per CTA, already laid
// out like that in shared memory) and the rows its N dimension, which goes in steps of 16.
// The accumulator is then transposed (lane = feature, column = row) and the epilogue writes
// 32 features of a row at a time straight from registers.
// Up to 128 rows: above, little is saved and the register epilogue costs more (dA with
// tiles of up to 240 rows: 245 -> 429 us). Measured at 768 rows an expert (d = 2048, F = 1408):
// dX 373 -> 350 us, GEMM2 196 -> 188, dA 249 -> 241; at 6 rows GEMM2 70 -> 65. Not in GEMM1:
// gate and up of a feature meet in one lane only with 16-row weight boxes, whose TMA rate
// costs more than the MMAs saved (389 -> 414 us; at 6 rows 135 -> 150).
constexpr int SWAP_ROWS = 128;

// ------------------------------------------------------------------------ router epilogue
// Gating of Alg. 7 for the token of this TMEM lane: the thread holds all BN >= E
// logits of its token, adds the party's bias, writes logits and Softmax
// probabilities, picks the k largest logits (equal logits: lower expert id first),
// writes the gate weights p[I] (renormalised on request) and counts the picks.
// The loops over experts are unrolled (the logits live in registers); the loop over
// the k picks is not: each tile runs this code once per CTA, so it runs from a cold
// instruction cache, and an unrolled 8 x BN selection was fetch-bound (k = 6, E = 64).
template <int BN>
__device__ __forceinline__ void route_epilogue(const Params& p, const Tile& ti, int m, bool valid,
                                               uint32_t tbase, int* hist) {
    float z[BN];
    if constexpr (BN == 16) {
        tmem_ld16(tbase, z);
    } else {
#pragma unroll
        for (int c = 0; c < BN / 32; ++c) tmem_ld32(tbase + 32 * c, z + 32 * c);
    }
    if (!valid) return;
    const int E = p.E, k = p.k;
    const int64_t t = ti.out_row + m;
    const float* bias = (const float*)p.aux;
    float mx = -3.402823466e38f;
#pragma unroll
    for (int e = 0; e < BN; ++e) {
        if (e < E) {
            if (bias) z[e] += bias[ti.g * E + e];
            mx = fmaxf(mx, z[e]);
        }
    }
    float ez[BN];
    float sum = 0.f;
#pragma unroll
    for (int e = 0; e < BN; ++e) {
        ez[e] = e < E ? expf(z[e] - mx) : 0.f;
        if (e < E) sum += ez[e];
    }
    float* lg = (float*)p.out0 + t * E;
    float* pr = (float*)p.out1 + t * E;
#pragma unroll
    for (int e = 0; e < BN; e += 4) {
        if (e < E) {
            *reinterpret_cast<float4*>(lg + e) = make_float4(z[e], z[e + 1], z[e + 2], z[e + 3]);
            *reinterpret_cast<float4*>(pr + e) =
                make_float4(ez[e] / sum, ez[e + 1] / sum, ez[e + 2] / sum, ez[e + 3] / sum);
        }
    }
    uint64_t taken = 0;
    float wsum = 0.f;
    int32_t* ti_out = p.topk_idx + t * k;
    float* tw_out = p.topk_w + t * k;
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
        int bi = -1;
        float bv = 0.f;
#pragma unroll
        for (int e = 0; e < BN; ++e) {
            if (e < E && !((taken >> e) & 1ull) && (bi < 0 || z[e] > bv)) {
                bi = e;
                bv = z[e];
            }
        }
        taken |= 1ull << bi;
        const float w = expf(bv - mx) / sum;
        wsum += w;
        ti_out[j] = bi;
        tw_out[j] = w;
        atomicAdd(&hist[ti.g * E + bi], 1);
    }
    if (p.normalize) {
#pragma unroll 1
        for (int j = 0; j < k; ++j) tw_out[j] = tw_out[j] / wsum;
    }
}

// Whether any thread of the four epilogue warps passes true: the same answer to all of them.
__device__ __forceinline__ bool epilogue_any(bool x) {
    uint32_t r;
    __syncwarp();
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.red.or.pred q, 1, 128, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)x)
        : "memory");
    return r != 0;
}

// The same gating for a tile of at most 32 tokens, whose accumulator rows are all in one
// warp's TMEM quarter: that warp lays the raw logits out in shared memory (s_z, rows of
// BN + 1) and all four take eight lanes a token (one thread a token took over 10 us at
// E = 64, k = 6). The picks are those of route_epilogue, NaN logits included: of the experts
// not taken the first if its logit is NaN, else the largest that is not, lower ids first.
template <int BN, int AR>
__device__ __forceinline__ void route_epilogue_short(const Params& p, const Tile& ti, int q, int wid, int lane,
                                                     uint32_t tbase, float* s_z, int* hist) {
    constexpr int V = BN / 8;
    if (q == 0) {
        float z[BN];
        if constexpr (BN == 16) {
            tmem_ld16(tbase, z);
        } else {
#pragma unroll
            for (int c = 0; c < BN / 32; ++c) tmem_ld32(tbase + 32 * c, z + 32 * c);
        }
        if (lane < AR) {
#pragma unroll
            for (int e = 0; e < BN; ++e) s_z[lane * (BN + 1) + e] = z[e];
        }
    }
    (void)epilogue_any(false);  // the logits are there
    const int E = p.E, k = p.k, l8 = lane & 7;
    const float* bias = (const float*)p.aux;
#pragma unroll 1
    for (int r0 = 0; r0 < AR; r0 += 16) {
        const int row = r0 + wid * 4 + (lane >> 3);
        const bool valid = ti.m0 + row < ti.mvalid;
        const int64_t t = ti.out_row + ti.m0 + row;
        float* zr = s_z + row * (BN + 1);
        float z[V], ez[V], mx = -3.402823466e38f, sum = 0.f;
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const int e = l8 + 8 * j;
            z[j] = zr[e];
            if (e < E) {
                if (bias) z[j] += bias[ti.g * E + e];
                mx = fmaxf(mx, z[j]);
            }
            zr[e] = z[j];
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
        for (int j = 0; j < V; ++j) ez[j] = l8 + 8 * j < E ? expf(z[j] - mx) : 0.f;
        // in order of the experts, as one thread adds them: the gates of a token are the same bits
        // whatever batch it is in
#pragma unroll
        for (int e = 0; e < BN; ++e) sum += __shfl_sync(0xffffffffu, ez[e / 8], e % 8, 8);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const int e = l8 + 8 * j;
            if (valid && e < E) {
                ((float*)p.out0)[t * E + e] = z[j];
                ((float*)p.out1)[t * E + e] = ez[j] / sum;
            }
        }
        __syncwarp();
        uint64_t taken = 0;
        float wsum = 0.f;
#pragma unroll 1
        for (int i = 0; i < k; ++i) {
            const int first = __ffsll((long long)~taken) - 1;
            // (logit in an order-preserving unsigned code, BN - e): the largest is the pick
            uint64_t best = 0;
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const int e = l8 + 8 * j;
                const uint32_t u = __float_as_uint(z[j] + 0.f);  // -0 counts as 0
                uint32_t key = (u & 0x80000000u) ? ~u : u | 0x80000000u;
                if (z[j] != z[j]) key = e == first ? 0xffffffffu : 0u;
                const uint64_t c = ((uint64_t)key << 32) | (uint32_t)(BN - e);
                if (e < E && !((taken >> e) & 1ull) && c > best) best = c;
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                const uint64_t other = __shfl_xor_sync(0xffffffffu, best, o);
                best = other > best ? other : best;
            }
            const int bi = BN - (int)(uint32_t)best;
            taken |= 1ull << bi;
            const float w = expf(zr[bi] - mx) / sum;
            wsum += w;
            if (valid && l8 == 0) {
                p.topk_idx[t * k + i] = bi;
                p.topk_w[t * k + i] = w;
                atomicAdd(&hist[ti.g * E + bi], 1);
            }
        }
        if (p.normalize && valid && l8 == 0) {
#pragma unroll 1
            for (int i = 0; i < k; ++i) p.topk_w[t * k + i] = p.topk_w[t * k + i] / wsum;
        }
    }
}

// Gating of Alg. 7 for E > 64 (BN = 128 or 256 accumulator columns): the same results
// as route_epilogue without holding all logits in registers. The accumulator stays in
// TMEM, read 32 columns at a time in three passes: (1) bias, logits out, running max and
// the k largest logits by insertion into a sorted list (ids arrive in ascending order
// and only a strictly larger logit moves ahead, so equal logits keep the lower id
// first); (2) the sum of exp(z - max); (3) the probabilities. Logits and probabilities
// are written element by element (any E). Every lane runs the TMEM loads (they are
// warp-collective); only valid rows use them.
template <int BN>
__device__ __forceinline__ void route_epilogue_wide(const Params& p, const Tile& ti, int m, bool valid,
                                                    uint32_t tbase, int* hist) {
    const int E = p.E, k = p.k;
    const int64_t t = ti.out_row + m;
    const float* bias = (const float*)p.aux;
    float* lg = (float*)p.out0 + t * E;
    float* pr = (float*)p.out1 + t * E;
    float mx = -3.402823466e38f;
    float tv[8];
    int tid[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        tv[j] = -3.402823466e38f;
        tid[j] = -1;
    }
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) {
        float z[32];
        tmem_ld32(tbase + c, z);
        if (valid) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int e = c + i;
                if (e < E) {
                    float v = z[i] + (bias ? bias[ti.g * E + e] : 0.f);
                    lg[e] = v;
                    mx = fmaxf(mx, v);
                    // insert at the first slot that is empty or holds a smaller logit,
                    // then shift the rest down by one
                    float cv = v;
                    int ce = e;
                    bool shifting = false;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (j < k && (shifting || tid[j] < 0 || cv > tv[j])) {
                            const float tvj = tv[j];
                            const int tij = tid[j];
                            tv[j] = cv;
                            tid[j] = ce;
                            cv = tvj;
                            ce = tij;
                            shifting = true;
                            if (ce < 0) break;
                        }
                    }
                }
            }
        }
    }
    float sum = 0.f;
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) {
        float z[32];
        tmem_ld32(tbase + c, z);
        if (valid) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (c + i < E) sum += expf(z[i] + (bias ? bias[ti.g * E + c + i] : 0.f) - mx);
        }
    }
#pragma unroll 1
    for (int c = 0; c < BN; c += 32) {
        float z[32];
        tmem_ld32(tbase + c, z);
        if (valid) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (c + i < E) pr[c + i] = expf(z[i] + (bias ? bias[ti.g * E + c + i] : 0.f) - mx) / sum;
        }
    }
    if (!valid) return;
    float wsel[8], wsum = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        wsel[j] = 0.f;
        if (j < k) {
            wsel[j] = expf(tv[j] - mx) / sum;
            wsum += wsel[j];
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j < k) {
            p.topk_idx[t * k + j] = tid[j];
            p.topk_w[t * k + j] = p.normalize ? wsel[j] / wsum : wsel[j];
            atomicAdd(&hist[ti.g * E + tid[j]], 1);
        }
    }
}

// ------------------------------------------------------------------------ swapped tiles
// Lane l of warp q of CTA `rank` holds one feature, its columns the tile's rows. Two rows
// j, j + 1 at a time, neighbouring lanes exchange values so that each lane holds two features
// of one of the two rows, and a warp's 32 lanes move 64 contiguous bytes of both.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// (a: row j, b: row j + 1) of this lane's feature -> the bf16 pair of features (l & ~1,
// l | 1) of row j + (l & 1)
__device__ __forceinline__ uint32_t pair_up(float a, float b, int lane) {
    const float other = __shfl_xor_sync(0xffffffffu, (lane & 1) ? a : b, 1);
    return (lane & 1) ? pack_bf16(other, b) : pack_bf16(a, other);
}
// the inverse for loads: u = the pair of row j + (l & 1) -> this feature's values of j, j + 1
__device__ __forceinline__ void pair_down(uint32_t u, int lane, float* a, float* b) {
    const float lo = __uint_as_float(u << 16), hi = __uint_as_float(u & 0xffff0000u);
    const float other = __shfl_xor_sync(0xffffffffu, (lane & 1) ? lo : hi, 1);
    *a = (lane & 1) ? other : lo;
    *b = (lane & 1) ? hi : other;
}

template <int EPI>
__device__ __forceinline__ void swapped_epilogue(int N, int F, void* out0, const void* aux, const Tile& ti, int rank, int q,
                                                  int lane, uint32_t tbase, int c_beg, int c_step) {
    const int v = ti.mvalid - ti.m0;       // rows of the tile
    const int64_t row0 = ti.out_row + ti.m0;
    const int n = ti.n0 + rank * 128 + q * 32 + (lane & ~1);  // this lane's pair of features
    if (n >= N) return;                                        // (a ragged last tile: whole CTAs)
#pragma unroll 1
    for (int c = c_beg; c < v; c += c_step) {
        if constexpr (EPI == EPI_STORE) {
            float y[32];
            tmem_ld32(tbase + c, y);
            __nv_bfloat16* out = (__nv_bfloat16*)out0 + (row0 + c) * (int64_t)N + n;
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
                const uint32_t u = pair_up(y[i], y[i + 1], lane);
                const int j = i + (lane & 1);
                if (c + j < v) *reinterpret_cast<uint32_t*>(out + j * (int64_t)N) = u;
            }
        } else {  // SwiGLU backward: y = dA
            const __nv_bfloat16* gu = (const __nv_bfloat16*)aux + (row0 + c) * (int64_t)(2 * F) + n;
            __nv_bfloat16* dh = (__nv_bfloat16*)out0 + (row0 + c) * (int64_t)(2 * F) + n;
#pragma unroll 1
            for (int h = 0; h < 32 && c + h < v; h += 16) {
                uint32_t gr[8], ur[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int j = h + 2 * i + (lane & 1);
                    gr[i] = ur[i] = 0;
                    if (c + j < v) {
                        gr[i] = *reinterpret_cast<const uint32_t*>(gu + j * (int64_t)(2 * F));
                        ur[i] = *reinterpret_cast<const uint32_t*>(gu + j * (int64_t)(2 * F) + F);
                    }
                }
                float y[16];
                tmem_ld16(tbase + c + h, y);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float G[2], U[2], dg[2], du[2];
                    pair_down(gr[i], lane, &G[0], &G[1]);
                    pair_down(ur[i], lane, &U[0], &U[1]);
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        const float sg = __fdividef(1.0f, 1.0f + __expf(-G[w])), d = y[2 * i + w];
                        du[w] = d * G[w] * sg;
                        dg[w] = d * U[w] * sg * (1.0f + G[w] * (1.0f - sg));
                    }
                    const uint32_t dgu = pair_up(dg[0], dg[1], lane), duu = pair_up(du[0], du[1], lane);
                    const int j = h + 2 * i + (lane & 1);
                    if (c + j < v) {
                        *reinterpret_cast<uint32_t*>(dh + j * (int64_t)(2 * F)) = dgu;
                        *reinterpret_cast<uint32_t*>(dh + j * (int64_t)(2 * F) + F) = duu;
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------------------ the kernel
// PAIR: the two CTAs of a cluster compute one 256 x BN tile with tcgen05 cta_group::2
// MMAs issued by CTA 0: each CTA holds 128 rows of A and BN/2 rows of B in its own
// shared memory and 128 rows of the accumulator in its own TMEM.
// DW2: the launch also computes a second, K-variable problem with the same groups
// (p2, tmA2, tmB2, tmO2: C_g = A_g^T B_g over group g's rows, MN-major operands, bf16
// store), its tiles after all of the first problem's: one persistent launch, one tail,
// for a weight gradient and the M-variable GEMM of the same backward step. (Interleaving
// the two problems' tiles group by group measured slower: a tile with a long epilogue
// followed by one with a short mainloop leaves the MMA waiting for an accumulator.)
// The forward GEMMs (K-major B) take a second problem of their own kind with uniform groups
// (p2.G > 0; tmA2, tmB2, tmO2, tmX2 = its out1 or its boxes of swapped tiles): the shared
// experts' tiles after the routed ones, in the SMs that the last round leaves free. On
// their own they are short and latency-bound (64 tokens, two of d = 2048, Fs = 1408: 18.7 and
// 12.5 us for 35 MB of weights): the forward of 64 tokens with 64 such routed experts
// 264 -> 233 us (of 2999 tokens, where they had rounds of their own, 0.5% less).
template <int BN, bool B_MN, bool VAR_K, int EPI, bool PAIR = false, bool DW2 = false, int OCC = 1, int EW = 4, int AR = BM>
__global__ void __launch_bounds__(gemm_threads(EW), OCC)
    grouped_gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                        const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmO0,
                        const __grid_constant__ CUtensorMap tmO1,
                        const __grid_constant__ CUtensorMap tmAs, const Params p,
                        const __grid_constant__ CUtensorMap tmA2,
                        const __grid_constant__ CUtensorMap tmB2,
                        const __grid_constant__ CUtensorMap tmO2,
                        const __grid_constant__ CUtensorMap tmX2, const Params p2) {
    pdl_begin();
    constexpr bool SH = !VAR_K && !B_MN && (EPI == EPI_STORE || EPI == EPI_SWIGLU_FWD);
    static_assert(!DW2 || (B_MN && !VAR_K && !PAIR && BN == 256), "fused: M-variable, MN-major B");
    static_assert(OCC == 1 || (!PAIR && !DW2 && 2 * BN * OCC <= 512), "shared SMs: single-CTA tiles, TMEM for all");
    static_assert(EW == 4 || (EW == 8 && !DW2 && (EPI == EPI_STORE || EPI == EPI_SWIGLU_FWD)), "epilogue warps");
    constexpr bool SHORT = AR < BM;
    static_assert(AR == BM || (EPI == EPI_ROUTE && (AR == 16 || AR == 32) && BN <= 64), "short A boxes: the router");
    constexpr int NBUF = EPI_BOXES / EW;  // output boxes of one epilogue warp
    constexpr bool A_MN = VAR_K;
    constexpr bool SWAP = PAIR && !VAR_K && EPI != EPI_SWIGLU_FWD;  // swapped tiles possible
    constexpr int NPAIR = PAIR ? 2 : 1;
    constexpr int BNL = BN / NPAIR;  // B rows held by this CTA
    constexpr int BMP = BM * NPAIR;  // rows of one (pair) tile
    constexpr int KB = kblock_rows(VAR_K, PAIR, EPI, BN);  // contraction rows per k-block
    constexpr int KPS = kblocks_per_stage(EPI, BN, PAIR, VAR_K, DW2, OCC, AR);
    constexpr uint32_t ATOM = KB * 128;         // bytes of one 64-wide MN-major box
    constexpr uint32_t ATOM_B = ATOM * KPS;     // of B's: one box holds all of a stage's k-blocks
    constexpr uint32_t A_BOX = AR * KB * 2;   // one k-block of A
    constexpr uint32_t B_BOX = BNL * KB * 2;  // one k-block of B
    constexpr uint32_t A_BYTES = A_BOX * KPS;
    constexpr uint32_t B_BYTES = B_BOX * KPS;
    constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
    constexpr int NST = num_stages(STAGE_BYTES, EPI, OCC, AR);
    constexpr uint32_t IDESC = instr_desc<BN, A_MN, B_MN, BMP>();
    constexpr uint32_t IDESC_DW = instr_desc<BN, true, true, BM>();
    constexpr int TMEM_COLS = (2 * BN <= 32) ? 32 : (2 * BN <= 64) ? 64 : (2 * BN <= 128) ? 128 : (2 * BN <= 256) ? 256 : 512;

    extern __shared__ uint8_t smem_raw[];
    // K-variable pairs: the peer's own barriers for the partial last k-block of a tile
    constexpr int NPART = (PAIR && VAR_K) ? NST : 0;
    __shared__ uint64_t bars[2 * NST + 5 + 2 * EW + NPART];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    // pairs: operand stages that this CTA's producer filled in all, and the bytes of each stage's
    // last fill that count on the leader's barrier
    __shared__ uint32_t s_fills, s_fill_bytes[PAIR ? NST : 1];
    __shared__ int s_tile_start[MAX_GROUPS + 1];
    __shared__ int s_total1;  // fused: tiles of the first problem
    __shared__ unsigned char s_order[DW2 ? MAX_GROUPS : 1];  // fused: second problem's group order

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* abort_flag = &s_abort;
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const int tile0 = (int)blockIdx.x / NPAIR, tile_step = (int)gridDim.x / NPAIR;

    // group -> tile prefix
    // N-tiles per row of tiles; the last one may be ragged (N a multiple of 128 with
    // 256-wide tiles: its columns past N are computed from zero-filled or unused operand
    // columns and never stored)
    const int tiles_n = (EPI == EPI_SWIGLU_FWD) ? p.N / 256 : (EPI == EPI_ROUTE) ? 1 : (p.N + BN - 1) / BN;
    const int tiles_n2 = (EPI == EPI_SWIGLU_FWD) ? p2.N / 256 : (p2.N + BN - 1) / BN;  // (SH)
    const int tiles_m2 = (p2.rows + BMP - 1) / BMP;
    if (warp == 0) {  // a warp scan: one thread reading 64 groups' offsets in turn took over a microsecond
        int run = 0;
        for (int g0 = 0; g0 < p.G; g0 += 32) {
            const int g = g0 + lane;
            int n = 0;
            if (g < p.G) {
                if (VAR_K) {
                    n = p.Mout / BMP;
                } else {
                    const int rows = p.offsets ? (p.offsets[g + 1] - p.offsets[g]) : p.rows;
                    const int rpt = (EPI == EPI_ROUTE) ? p.tile_rows : BMP;  // rows per tile
                    n = rows > 0 ? (rows + rpt - 1) / rpt : 0;
                }
                n *= tiles_n;
            }
            int inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            if (g < p.G) s_tile_start[g] = run + inc - n;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) {
            s_total1 = run;
            s_tile_start[p.G] = run + (DW2 ? p.G * (p2.Mout / BM) * (p2.N / BN) : SH ? p2.G * tiles_m2 * tiles_n2 : 0);
            s_abort = 0;
        }
    }
    __syncthreads();
    if constexpr (DW2) {
        // weight-gradient groups longest first (each tile of a group runs over all its
        // rows): with skewed experts the long tiles then do not form the tail. Rank of g =
        // groups with more rows, or as many and a lower index. (Row counts are read from
        // the offsets in global memory: static shared memory is at its limit here.)
        for (int g = threadIdx.x; g < p2.G; g += blockDim.x) {
            const int rg = p2.offsets[g + 1] - p2.offsets[g];
            int rank = 0;
            for (int h = 0; h < p2.G; ++h) {
                const int rh = p2.offsets[h + 1] - p2.offsets[h];
                rank += (rh > rg) || (rh == rg && h < g);
            }
            s_order[rank] = (unsigned char)g;
        }
        __syncthreads();
    }
    const int total_tiles = s_tile_start[p.G];
    if (tile0 >= total_tiles) return;  // uniform across the pair

    // Tile order inside a group: bands of `band` M-tiles, each band swept along N with
    // the M-tiles of the band innermost. The tiles that run at the same time (one round
    // of the persistent grid, C of them) then cover about band x C/band output tiles and
    // read band A blocks and C/band B blocks, instead of one A block and C B blocks when
    // whole rows of N-tiles come first (band ~ sqrt(C) minimises the blocks per round;
    // the A blocks of a band also stay in L2 while it sweeps N). When all of a group's B
    // fits in L2, whole rows of N-tiles first (band 1) read it from DRAM once and each A
    // block once; else when all of its A fits, whole columns of M-tiles first (band =
    // the group's M-tiles) do the same with A resident.
    constexpr int64_t kL2Resident = 48ll << 20;  // bytes of an operand kept in L2
    auto group_band = [&](const Params& q, int64_t rows_g, int mt_g) -> int {
        const int64_t a_all = (int64_t)rows_g * q.a_row_bytes;
        const int64_t b_all = q.b_row_bytes ? (int64_t)rows_g * q.b_row_bytes : q.b_all_bytes;
        if (b_all > 0 && b_all <= kL2Resident) return 1;
        if (a_all > 0 && a_all <= kL2Resident) return mt_g;
        return q.band;
    };
    auto band_split = [&](int local, int mt_g, int nt_g, int band, int* mt, int* nt) {
        const int gmx = band > 0 ? band : 1;
        const int b = local / (gmx * nt_g);
        const int first = b * gmx;
        const int gm = min(gmx, mt_g - first);
        const int rem = local - b * gmx * nt_g;
        *mt = first + rem % gm;
        *nt = rem / gm;
    };
    auto tile_at = [&](int t) -> Tile {
        Tile ti;
        ti.dw = ti.sec = false;
        ti.ntok = 0;
        if constexpr (DW2) {
            if (t >= s_total1) {  // second problem: K-variable, rows of group g
                const int per = (p2.Mout / BM) * (p2.N / BN);
                const int g = s_order[(t - s_total1) / per], l2 = (t - s_total1) % per;
                const int tn2 = p2.N / BN;
                int mt2, nt2;
                band_split(l2, p2.Mout / BM, tn2,
                           group_band(p2, p2.offsets[g + 1] - p2.offsets[g], p2.Mout / BM), &mt2, &nt2);
                ti.dw = true;
                ti.g = g;
                ti.we = p2.gexp ? p2.gexp[g] : g;
                ti.m0 = mt2 * BM;
                ti.n0 = nt2 * BN;
                const int64_t r0 = p2.offsets[g], nrows = p2.offsets[g + 1] - r0;
                ti.mvalid = p2.Mout;
                ti.a_row = ti.b_row = r0;
                ti.out_row = 0;
                ti.k_iters = (int)((nrows + BK - 1) / BK);
                ti.last_rows = (int)(nrows - (int64_t)(ti.k_iters - 1) * BK);
                return ti;
            }
        }
        int g, mt, nt;
        if (SH && t >= s_total1) {  // second problem: uniform groups
            ti.sec = true;
            g = (t - s_total1) / (tiles_m2 * tiles_n2);
            band_split((t - s_total1) % (tiles_m2 * tiles_n2), tiles_m2, tiles_n2, group_band(p2, p2.rows, tiles_m2), &mt, &nt);
        } else {
            // the group whose tile range holds t: last g with s_tile_start[g] <= t (binary
            // search; empty groups share their start with the next one)
            int lo = 0, hi = p.G - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_tile_start[mid] <= t) lo = mid;
                else hi = mid - 1;
            }
            g = lo;
            const int local = t - s_tile_start[g];
            const int g_end = (g + 1 < p.G) ? s_tile_start[g + 1] : s_total1;
            const int mt_g = (g_end - s_tile_start[g]) / tiles_n;
            const int64_t rows_g = p.offsets ? (int64_t)(p.offsets[g + 1] - p.offsets[g]) : (int64_t)p.rows;
            band_split(local, mt_g, tiles_n, group_band(p, rows_g, mt_g), &mt, &nt);
        }
        ti.g = g;
        ti.we = !ti.sec && p.gexp ? p.gexp[g] : g;
        ti.m0 = (EPI == EPI_ROUTE) ? mt * p.tile_rows : mt * BMP + (int)rank * BM;
        ti.n0 = nt * ((EPI == EPI_SWIGLU_FWD) ? 128 : BN);
        int64_t r0, nrows, a0, b0, o0;
        if (SH && ti.sec) {
            nrows = p2.rows;
            a0 = (int64_t)g * p2.a_stride;
            b0 = 0;
            o0 = (int64_t)g * p2.out_stride;
        } else if (p.offsets) {
            r0 = p.offsets[g];
            nrows = p.offsets[g + 1] - r0;
            a0 = b0 = o0 = r0;
        } else {
            nrows = p.rows;
            a0 = (int64_t)g * p.a_stride;
            b0 = (int64_t)g * p.b_stride;
            o0 = (int64_t)g * p.out_stride;
        }
        if (VAR_K) {
            ti.mvalid = p.Mout;
            ti.a_row = a0;
            ti.b_row = b0;
            ti.out_row = 0;
            ti.k_iters = (int)((nrows + KB - 1) / KB);
            ti.last_rows = (int)(nrows - (int64_t)(ti.k_iters - 1) * KB);
        } else {
            // router tiles of tile_rows rows: the box's rows past them are the next tile's
            ti.mvalid = (EPI == EPI_ROUTE) ? (int)min64(nrows, (int64_t)ti.m0 + p.tile_rows) : (int)nrows;
            ti.a_row = a0;
            ti.b_row = 0;
            ti.out_row = o0;
            ti.k_iters = ((SH && ti.sec ? p2.K : p.K) + (SHORT ? BK * KPS - 1 : 0)) / (BK * KPS);  // (zero-filled)
            ti.last_rows = BK;
            if constexpr (SWAP) {
                const int v = (int)nrows - mt * BMP;
                if (v <= SWAP_ROWS) {
                    ti.ntok = (v + 15) / 16 * 16;
                    ti.m0 = mt * BMP;  // both CTAs hold features of the same rows
                }
            }
        }
        return ti;
    };

    // 1024-byte aligned stage ring
    const uint32_t raw_u32 = smem_u32(smem_raw);
    const uint32_t ring = raw_u32 + ((1024u - (raw_u32 & 1023u)) & 1023u);
    uint8_t* ring_ptr = smem_raw + (ring - raw_u32);
    uint8_t* stage_out = ring_ptr + (size_t)NST * STAGE_BYTES;  // the epilogue warps' staging boxes
    int* route_hist = reinterpret_cast<int*>(stage_out);             // EPI_ROUTE has no staging
    if constexpr (EPI == EPI_ROUTE) {
        for (int i = threadIdx.x; i < p.hist_n; i += blockDim.x) route_hist[i] = 0;
    }
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (NST + s); };
    auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * NST + a); };
    auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * NST + 2 + a); };
    const uint32_t drain_bar = bar0 + 8u * (2 * NST + 4);
    auto pfull_bar = [&](int s) { return bar0 + 8u * (2 * NST + 5 + 2 * EW + s); };
    // waits: cluster-scope acquire when the barrier also collects the peer's arrivals
    auto wait_bar = [&](uint32_t bar, uint32_t parity) -> bool {
        if constexpr (PAIR) {
            if (mbar_try_cluster(bar, parity)) return true;
            const uint64_t t0 = gtimer();
            for (;;) {
                if (mbar_try_cluster(bar, parity)) return true;
                if (*abort_flag) return false;
                if (gtimer() - t0 > p.wait_ns) {
                    *abort_flag = 1;
                    record_status(MOE_ERR_TIMEOUT);
                    return false;
                }
            }
        } else {
            return mbar_wait(bar, parity, abort_flag, p.wait_ns);
        }
    };
    // the same for a whole warp: one answer to all lanes, of which some may have given up where
    // others saw the barrier complete (they must not part before warp-wide tcgen05.ld, nor at
    // the block's barrier)
    auto warp_wait = [&](uint32_t bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, wait_bar(bar, parity)); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(full_bar(s), 1);  // the (leader's) producer arms it for both CTAs' bytes
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), EW * NPAIR);  // one arrival per epilogue warp
        }
        mbar_init(drain_bar, 1);
        for (int i = 0; i < 2 * EW; ++i) mbar_init(bar0 + 8u * (2 * NST + 5 + i), 1);
        for (int s = 0; s < NPART; ++s) mbar_init(pfull_bar(s), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&s_tmem)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&s_tmem)),
                         "r"(TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();  // the peer's barriers are initialised
    fence_after();
    const uint32_t tmem_base = s_tmem;
    const uint64_t limit = p.wait_ns;
    // drains after an abort wait for work that is already in flight (it completes in
    // microseconds); their bound does not shrink with a short user wait limit
    const uint64_t drain_limit = limit > 200000000ull ? limit : 200000000ull;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued = 0, issued_par = 0;  // stages ever filled, and the parity of their last fill
            uint32_t fills = 0;
            // K-variable pair peer: stages whose own barrier was ever armed, and per stage
            // the parity of the next phase to arm
            uint32_t parmed = 0, pnext = 0;
            bool ok = true;
            // every TMA load is counted on the leader's full barrier (CTA 0 of a pair)
            const uint32_t full0 = PAIR ? map_to_rank(bar0, 0) : bar0;
            bool local_bar = false;  // this stage's copies complete on this CTA's own barrier
            auto load = [&](uint32_t dst, const CUtensorMap* map, uint32_t fb, int c0, int c1) {
                if (PAIR && !local_bar) tma_load_2d_pair(dst, map, fb, c0, c1);
                else tma_load_2d(dst, map, fb, c0, c1);
            };
            for (int t = tile0; t < total_tiles && ok; t += tile_step) {
                const Tile ti = tile_at(t);
                const bool dw = DW2 && ti.dw, sec = SH && ti.sec;
                const CUtensorMap* mA = dw || sec ? &tmA2 : &tmA;
                const CUtensorMap* mAs = sec ? &tmX2 : &tmAs;
                const CUtensorMap* mB = dw || sec ? &tmB2 : &tmB;
                const int F = sec ? p2.F : p.F;
                // a swapped tile's rows: half in each CTA, in boxes of 32
                const int trows = SWAP ? ti.ntok / 2 : 0;
                uint32_t tile_bytes = NPAIR * STAGE_BYTES;  // per stage, both CTAs of a pair
                if (EPI == EPI_ROUTE && !SHORT) tile_bytes = (uint32_t)p.tile_rows * 128u * KPS + B_BYTES;  // A boxes of tile_rows rows
                if (SWAP && trows) tile_bytes = NPAIR * (B_BYTES + (uint32_t)((trows + 31) / 32) * (32u * 128u * KPS));
                // the tile's coordinates: A (first row, or contraction row), B (row, or contraction row)
                const int arow = (int)ti.a_row + ((A_MN || dw) ? 0 : ti.m0 + (int)rank * trows);
                int brow;
                if (VAR_K || dw) brow = (int)ti.b_row;
                else if (B_MN) brow = (int)((int64_t)ti.we * p.b_group_rows);
                else brow = (int)((int64_t)ti.we * (sec ? p2.b_group_rows : p.b_group_rows) + ti.n0) +
                            (EPI == EPI_SWIGLU_FWD ? (PAIR && rank ? F : 0) : (int)rank * BNL);
                for (int kb = 0; kb < ti.k_iters; ++kb) {
                    if (!wait_bar(empty_bar(stage), phase ^ 1u)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = ring + stage * STAGE_BYTES;
                    const uint32_t sb = sa + A_BYTES;
                    uint32_t fb = full0 + 8u * stage;
                    // In a pair only the leader arrives, expecting the bytes of both CTAs: the
                    // peer's copies complete on the leader's barrier without an arrival (a
                    // cluster-scope arrive per stage cost the producers most of their time). The
                    // peer reuses a stage only after the leader's MMAs released it, so its bytes
                    // always count towards the phase the leader arms.
                    if (!PAIR || rank == 0) mbar_expect_tx(full_bar(stage), tile_bytes);
                    if constexpr (PAIR && VAR_K) {
                        // peer, partial last k-block: its copies land on its own barrier; the MMA
                        // warp zeroes the rows past the group's end and then credits these bytes
                        // to the leader's full barrier
                        local_bar = rank == 1 && kb == ti.k_iters - 1 && ti.last_rows < KB;
                        if (local_bar) {
                            fb = pfull_bar(stage);
                            mbar_expect_tx(fb, STAGE_BYTES);
                            parmed |= 1u << stage;
                            pnext ^= 1u << stage;
                        }
                    }
                    const int k0 = kb * KB * KPS;
                    if constexpr (SHORT) {
                        tma_load_3d(sa, &tmA, fb, 0, arow, kb * KPS);
                        tma_load_3d(sb, &tmB, fb, 0, brow, kb * KPS);
                    } else {
                        if (!A_MN && !dw) {
                            if (SWAP && trows) {
                                for (int r = 0; r < trows; r += 32)
#pragma unroll
                                    for (int i = 0; i < KPS; ++i) load(sa + i * A_BOX + r * 128, mAs, fb, k0 + KB * i, arow + r);
                            } else {
#pragma unroll
                                for (int i = 0; i < KPS; ++i) load(sa + i * A_BOX, mA, fb, k0 + KB * i, arow);
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < BM / 64; ++i) load(sa + i * ATOM, mA, fb, ti.m0 + 64 * i, arow + k0);
                        }
                        if (!B_MN) {
#pragma unroll
                            for (int i = 0; i < KPS; ++i) {
                                load(sb + i * B_BOX, mB, fb, k0 + KB * i, brow);
                                // SwiGLU forward: 128 gate rows, then 128 up rows of the same features
                                // (in a pair the leader holds the gate half and the peer the up half)
                                if (EPI == EPI_SWIGLU_FWD && !PAIR) load(sb + i * B_BOX + 128 * 128, mB, fb, k0 + KB * i, brow + F);
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < BNL / 64; ++i)
                                load(sb + i * ATOM_B, mB, fb, ti.n0 + (int)rank * BNL + 64 * i, brow + k0);
                        }
                    }
                    if constexpr (PAIR) {
                        s_fill_bytes[stage] = local_bar ? 0 : tile_bytes / NPAIR;
                        ++fills;
                    }
                    issued |= 1u << stage;
                    issued_par = (issued_par & ~(1u << stage)) | (phase << stage);
                    if (++stage == NST) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if constexpr (PAIR) s_fills = fills;
            // Every copy started into this pair lands before the CTAs exit (after a whole launch at
            // once: the MMAs have read them), also when another role gives up only after this one
            // is through.
            if constexpr (PAIR && VAR_K) {
                if (rank == 1) {
                    // partial copies on this CTA's own barriers: the last phase armed
                    for (int s2 = 0; s2 < NST; ++s2) {
                        if (!((parmed >> s2) & 1u)) continue;
                        const uint32_t par = ((pnext >> s2) & 1u) ^ 1u;
                        const uint64_t t0 = gtimer();
                        while (!mbar_try(pfull_bar(s2), par) && gtimer() - t0 < drain_limit) {
                        }
                    }
                }
            }
            if (rank == 0) {  // (the leader's full barriers count the peer's bytes too)
                for (int s = 0; s < NST; ++s) {
                    if (!((issued >> s) & 1u)) continue;
                    const uint64_t t0 = gtimer();
                    while (!mbar_try(full_bar(s), (issued_par >> s) & 1u) &&
                           gtimer() - t0 < drain_limit) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        int stage = 0;
        uint32_t phase = 0;
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        bool issued_any = false;
        // in a pair only the leader issues MMAs (they read both CTAs' shared memory and
        // write both CTAs' TMEM)
        for (int t = tile0; t < total_tiles && ok && rank == 0; t += tile_step) {
            const Tile ti = tile_at(t);
            // kind::f16 descriptor of a swapped tile: A = weights (M = 256), B = rows (K-major)
            const uint32_t idesc_s = instr_desc<16, B_MN, false, BMP>() - (2u << 17) + ((uint32_t)(ti.ntok >> 3) << 17);
            if (!warp_wait(tempty_bar(acc), acc_phase ^ 1u)) {
                ok = false;
                break;
            }
            fence_after();
            const uint32_t tmem_d = tmem_base + (uint32_t)(acc * BN);
            const bool dwt = DW2 && ti.dw;
            // the MMAs of a k-block in stage `st`, and its release (one thread)
            auto issue = [&](int st, int kb, int ksteps, bool part) {
                const uint32_t sa = ring + st * STAGE_BYTES, sb = sa + A_BYTES;
                auto step = [&](int kk, bool swapped) {
                    uint64_t ad, bd;
                    if (!A_MN && !dwt) ad = smem_desc(sa + (kk / (KB / 16)) * A_BOX + (kk % (KB / 16)) * 32, 16, 1024);
                    else ad = smem_desc(sa + (kk / (KB / 16)) * A_BOX + (kk % (KB / 16)) * 2048, ATOM, 1024);
                    if (!B_MN) bd = smem_desc(sb + (kk / (KB / 16)) * B_BOX + (kk % (KB / 16)) * 32, 16, 1024);
                    else bd = smem_desc(sb + kk * 2048, ATOM_B, 1024);
                    if (SWAP && swapped) mma_bf16_pair(tmem_d, bd, ad, idesc_s, (kb | kk) ? 1u : 0u);
                    else if constexpr (PAIR) mma_bf16_pair(tmem_d, ad, bd, IDESC, (kb | kk) ? 1u : 0u);
                    else mma_bf16(tmem_d, ad, bd, dwt ? IDESC_DW : IDESC, (kb | kk) ? 1u : 0u);
                };
                // whole k-blocks without a check per step (with one, the issuing thread
                // held back the weight-gradient launches by up to 20%)
                if (SWAP && ti.ntok) {
#pragma unroll
                    for (int kk = 0; kk < KB * KPS / 16; ++kk) step(kk, true);
                } else if (!part) {
#pragma unroll
                    for (int kk = 0; kk < KB * KPS / 16; ++kk) step(kk, false);
                } else {
#pragma unroll 1
                    for (int kk = 0; kk < ksteps; ++kk) step(kk, false);
                }
                if constexpr (PAIR) mma_commit_pair(empty_bar(st), 3);  // both producers
                else mma_commit(empty_bar(st));
                issued_any = true;
            };
            // One answer to the warp, whether a wait gave up: after the MMAs of a k-block are on their
            // way (before them it cost up to 1% of a step), or, where a stage is a single k-block of
            // a pair (dA: 247 -> 263 us by that vote) and one thread waits and issues (245; the other
            // forms lose 1 to 5% by that), at the tile's end. After a wait that gave up nothing more
            // is issued or released: what the other CTA of a pair would then copy is armed by no one.
            if constexpr (PAIR && !VAR_K && KPS == 1) {
                if (lane == 0) {
                    int st = stage;
                    uint32_t ph = phase;
                    for (int kb = 0; kb < ti.k_iters; ++kb) {
                        if (!wait_bar(full_bar(st), ph)) {
                            ok = false;
                            break;
                        }
                        fence_after();
                        issue(st, kb, KB * KPS / 16, false);
                        if (++st == NST) {
                            st = 0;
                            ph ^= 1u;
                        }
                    }
                }
                phase ^= (uint32_t)((stage + ti.k_iters) / NST) & 1u;
                stage = (stage + ti.k_iters) % NST;
                ok = __all_sync(0xffffffffu, ok);
            } else {
                for (int kb = 0; kb < ti.k_iters; ++kb) {
                    const bool got = wait_bar(full_bar(stage), phase);
                    // K-variable groups: the last k-block may hold contraction rows of the next
                    // group. Only K=16 steps that contain valid rows are issued, and inside the
                    // last of them the A rows past the group's end are zeroed (A alone suffices:
                    // their products with any finite B row vanish).
                    const bool part = (VAR_K || dwt) && kb == ti.k_iters - 1 && ti.last_rows < KB;
                    const int ksteps = part ? (ti.last_rows + 15) / 16 : KB * KPS / 16;
                    if (part) {
                        const int zr0 = ti.last_rows, zr1 = ksteps * 16;
                        if (got && zr1 > zr0) {
                            uint8_t* base = ring_ptr + (size_t)stage * STAGE_BYTES;
                            const int per_box = (zr1 - zr0) * 8;  // 16-byte words
#pragma unroll
                            for (int b = 0; b < BM / 64; ++b) {
                                uint4* z = reinterpret_cast<uint4*>(base + b * ATOM + zr0 * 128);
                                for (int i = lane; i < per_box; i += 32) z[i] = make_uint4(0, 0, 0, 0);
                            }
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        }
                        __syncwarp();
                    }
                    fence_after();
                    if (lane == 0 && got) issue(stage, kb, ksteps, part);
                    if (!__all_sync(0xffffffffu, got)) {
                        ok = false;
                        break;
                    }
                    if (++stage == NST) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) break;
            if (lane == 0) {
                if constexpr (PAIR) {
                    mma_commit_pair(tfull_bar(acc), 3);  // both CTAs' epilogues
                } else {
                    if (ti.k_iters > 0) mma_commit(tfull_bar(acc));
                    else mbar_arrive(tfull_bar(acc));
                }
            }
            __syncwarp();
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        if (lane == 0 && issued_any) {
            // wait for every MMA this CTA issued before TMEM is released (always, as above)
            if constexpr (PAIR) mma_commit_pair(drain_bar, 1);
            else mma_commit(drain_bar);
            const uint64_t t0 = gtimer();
            while (!mbar_try(drain_bar, 0) && gtimer() - t0 < drain_limit) {
            }
        }
        __syncwarp();
        if constexpr (PAIR && VAR_K) {
            // Peer of a K-variable pair: the leader's MMAs read this CTA's A rows too, so
            // the rows of a tile's last k-block past its group's end are zeroed here, as
            // the leader does for its own; then this stage's bytes are credited to the
            // leader's full barrier, which the peer's copies did not count.
            if (rank == 1) {
                int st2 = 0;
                uint32_t wpar = 0;  // per stage: parity of the next partial phase to wait for
                bool ok2 = true;
                for (int t = tile0; t < total_tiles && ok2; t += tile_step) {
                    const Tile ti = tile_at(t);
                    for (int kb = 0; kb < ti.k_iters; ++kb) {
                        if (kb == ti.k_iters - 1 && ti.last_rows < KB) {
                            if (!__all_sync(0xffffffffu, mbar_wait(pfull_bar(st2), (wpar >> st2) & 1u, abort_flag, p.wait_ns))) {
                                ok2 = false;
                                break;
                            }
                            wpar ^= 1u << st2;
                            const int zr0 = ti.last_rows, zr1 = ((ti.last_rows + 15) / 16) * 16;
                            if (zr1 > zr0) {
                                uint8_t* base = ring_ptr + (size_t)st2 * STAGE_BYTES;
                                const int per_box = (zr1 - zr0) * 8;  // 16-byte words
#pragma unroll
                                for (int b = 0; b < BM / 64; ++b) {
                                    uint4* z = reinterpret_cast<uint4*>(base + b * ATOM + zr0 * 128);
                                    for (int i = lane; i < per_box; i += 32) z[i] = make_uint4(0, 0, 0, 0);
                                }
                                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            }
                            __syncwarp();
                            if (lane == 0) {
                                // release of the zeroed shared memory only: a full cluster
                                // fence waits for all of the SM's memory traffic (14-18% of
                                // the weight-gradient launches at 512 and 768 rows an expert)
                                fence_release_smem_cluster();
                                mbar_complete_tx_remote(map_to_rank(full_bar(st2), 0), STAGE_BYTES);
                            }
                            __syncwarp();
                        }
                        if (++st2 == NST) st2 = 0;
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue warps 2-5
        // Warp w reads TMEM lane quarter w % 4 (32 rows). Finished 32x32 bf16 boxes are
        // staged in shared memory and written by TMA stores; a box that reaches past the
        // group's last row (the last M tile of an expert) is written row by row instead.
        const int q = warp & 3;
        const int half = EW == 8 ? (warp - 2) >> 2 : 0;  // of the tile's columns, with eight warps
        constexpr int SPLIT = EW / 4;
        const int row_local = q * 32 + lane;
        uint8_t* stg = stage_out + (size_t)(warp - 2) * (epi_stage_bytes(EPI) / EW);
        const uint32_t stg_u32 = smem_u32(stg);
        int acc = 0;
        uint32_t acc_phase = 0;
        uint32_t box_seq = 0;  // output boxes this warp has staged (ring position)
        // SwiGLU backward: TMA loads of G/U chunk boxes into two staging buffers
        const uint32_t gu_bar0 = bar0 + 8u * (2 * NST + 5 + 2 * (warp - 2));
        uint32_t gu_issued = 0;  // chunks whose loads were issued (this warp)
        uint32_t gu_chunk = 0;   // chunks consumed
        auto gu_issue = [&](const Tile& tn, int cn) {
            if constexpr (EPI == EPI_SWIGLU_BWD) {
                const int b = gu_issued & 1;
                if (lane == 0) {
                    bulk_wait_read0();  // earlier stores out of this buffer have read it
                    const uint32_t dst = stg_u32 + (2 * b) * EPI_BUF_BYTES;
                    const int row0 = (int)(tn.out_row + tn.m0 + q * 32);
                    mbar_expect_tx(gu_bar0 + 8u * b, 2 * EPI_BUF_BYTES);
                    tma_load_2d(dst, &tmO1, gu_bar0 + 8u * b, tn.n0 + 32 * cn, row0);
                    tma_load_2d(dst + EPI_BUF_BYTES, &tmO1, gu_bar0 + 8u * b, p.F + tn.n0 + 32 * cn, row0);
                }
                ++gu_issued;
            }
        };
        auto gu_wait = [&](int b, uint32_t parity) -> bool {
            return __all_sync(0xffffffffu, mbar_wait(gu_bar0 + 8u * b, parity, abort_flag, limit));
        };
        if constexpr (EPI == EPI_SWIGLU_BWD) {
            if (tile0 < total_tiles) {
                const Tile tf = tile_at(tile0);
                if (!(DW2 && tf.dw) && !tf.ntok) gu_issue(tf, 0);
            }
        }
        for (int t = tile0; t < total_tiles; t += tile_step) {
            const Tile ti = tile_at(t);
            const int m = ti.m0 + row_local;
            const bool valid = m < ti.mvalid;
            const int wrow0 = ti.m0 + q * 32;
            const bool full_box = wrow0 + 32 <= ti.mvalid;
            const bool dwt = DW2 && ti.dw, sec = SH && ti.sec;
            const int N = sec ? p2.N : p.N;
            void* const out0 = sec ? p2.out0 : p.out0;
            const int64_t grow0 = (VAR_K || dwt) ? (int64_t)ti.we * (dwt ? p2.Mout : p.Mout) + wrow0
                                                 : ti.out_row + wrow0;
            const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
            // write NOUT rows of 32 values each: staged + TMA when the whole box is valid
            auto emit = [&](int nout, const float* const* vals, const CUtensorMap* const* maps,
                            const int* cols, __nv_bfloat16* const* direct) {
                if (full_box) {
#pragma unroll
                    for (int o = 0; o < nout; ++o) {
                        const uint32_t b = box_seq & (NBUF - 1);
                        // the store that last used box b (NBUF boxes ago) has read it
                        if (lane == 0) bulk_wait_read<NBUF - 1>();
                        __syncwarp();
                        store_row32_sw64(stg + b * EPI_BUF_BYTES + lane * 64, lane, vals[o]);
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) {
                            tma_store_2d(maps[o], stg_u32 + b * EPI_BUF_BYTES, cols[o], (int)grow0);
                            bulk_commit();
                        }
                        ++box_seq;
                    }
                } else if (valid) {
                    for (int o = 0; o < nout; ++o) store_row32(direct[o], vals[o]);
                }
            };
            if (dwt) {
                // second problem: a bf16 weight-gradient tile, [Mout, N] per group
                if (!warp_wait(tfull_bar(acc), acc_phase)) break;
                fence_after();
                __nv_bfloat16* out = (__nv_bfloat16*)p2.out0 + (int64_t)ti.we * p2.Mout * p2.N + (int64_t)m * p2.N;
#pragma unroll 1
                for (int c = half * (BN / SPLIT); c < (half + 1) * (BN / SPLIT); c += 32) {
                    float y[32];
                    if (ti.k_iters > 0) {
                        tmem_ld32(tbase + c, y);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) y[i] = 0.f;
                    }
                    const float* vals[1] = {y};
                    const CUtensorMap* maps[1] = {&tmO2};
                    const int cols[1] = {ti.n0 + c};
                    __nv_bfloat16* direct[1] = {out + ti.n0 + c};
                    emit(1, vals, maps, cols, direct);
                }
            } else if (SWAP && ti.ntok) {
                if (!warp_wait(tfull_bar(acc), acc_phase)) break;
                fence_after();
                swapped_epilogue<EPI>(N, p.F, out0, p.aux, ti, (int)rank, q, lane, tbase, half * 32, SPLIT * 32);
            } else if constexpr (EPI == EPI_SWIGLU_BWD) {
                // dA in TMEM. G and U of each 32-column chunk arrive by TMA in one of two
                // staging buffers (the next chunk's load is in flight while this one is
                // computed); dG and dU overwrite them in place and leave by TMA store.
                const int F = p.F;
                __nv_bfloat16* dh = (__nv_bfloat16*)p.out0 + (ti.out_row + m) * (int64_t)(2 * F) + ti.n0;
                constexpr int NCH = BN / 32;
                const int nchv = min(NCH, (F - ti.n0) / 32);  // chunks inside F (a ragged last tile)
                if (gu_issued == gu_chunk) gu_issue(ti, 0);  // not prefetched (a fused tile came before)
                if (!warp_wait(tfull_bar(acc), acc_phase)) break;
                fence_after();
                bool stop = false;
#pragma unroll 1
                for (int c = 0; c < nchv; ++c) {
                    // prefetch the next chunk (of this tile, or the first of the next tile)
                    if (c + 1 < nchv) gu_issue(ti, c + 1);
                    else if (t + tile_step < total_tiles) {
                        const Tile tn = tile_at(t + tile_step);
                        if (!(DW2 && tn.dw) && !tn.ntok) gu_issue(tn, 0);
                    }
                    const int b = gu_chunk & 1;
                    if (!gu_wait(b, (gu_chunk >> 1) & 1)) { stop = true; break; }
                    uint8_t* gbuf = stg + (2 * b) * EPI_BUF_BYTES + lane * 64;
                    uint8_t* ubuf = gbuf + EPI_BUF_BYTES;
                    float da[32], dG[32], dU[32];
                    tmem_ld32(tbase + 32 * c, da);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int sw = (v ^ ((lane >> 1) & 3)) << 4;
                        float G[8], U[8];
                        unpack8(*reinterpret_cast<const uint4*>(gbuf + sw), G);
                        unpack8(*reinterpret_cast<const uint4*>(ubuf + sw), U);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float sg = __fdividef(1.0f, 1.0f + __expf(-G[i]));
                            const float d = da[8 * v + i];
                            dU[8 * v + i] = d * G[i] * sg;
                            dG[8 * v + i] = d * U[i] * sg * (1.0f + G[i] * (1.0f - sg));
                        }
                    }
                    if (full_box) {
                        store_row32_sw64(gbuf, lane, dG);
                        store_row32_sw64(ubuf, lane, dU);
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) {
                            const uint32_t src = stg_u32 + (2 * b) * EPI_BUF_BYTES;
                            tma_store_2d(&tmO0, src, ti.n0 + 32 * c, (int)grow0);
                            tma_store_2d(&tmO0, src + EPI_BUF_BYTES, F + ti.n0 + 32 * c, (int)grow0);
                            bulk_commit();
                        }
                    } else if (valid) {
                        store_row32(dh + 32 * c, dG);
                        store_row32(dh + F + 32 * c, dU);
                    }
                    __syncwarp();
                    ++gu_chunk;
                }
                if (stop) break;
            } else {
                const bool got = warp_wait(tfull_bar(acc), acc_phase);
                // (short router tiles: the epilogue warps meet per tile, and give up together)
                if (SHORT ? epilogue_any(!got) : !got) break;
                fence_after();
                if constexpr (EPI == EPI_SWIGLU_FWD) {
                    // accumulator columns [0,128) = G, [128,256) = U of features n0 .. n0+127
                    const int F = sec ? p2.F : p.F;
                    const CUtensorMap *mO0 = sec ? &tmO2 : &tmO0, *mO1 = sec ? &tmX2 : &tmO1;
                    __nv_bfloat16* hgu = (__nv_bfloat16*)out0 + (ti.out_row + m) * (int64_t)(2 * F);
                    __nv_bfloat16* actp = (__nv_bfloat16*)(sec ? p2.out1 : p.out1) + (ti.out_row + m) * (int64_t)F;
#pragma unroll 1
                    for (int c = half * (128 / SPLIT); c < (half + 1) * (128 / SPLIT); c += 32) {
                        float g[32], u[32], a[32];
                        tmem_ld32(tbase + c, g);
                        tmem_ld32(tbase + 128 + c, u);
#pragma unroll
                        for (int i = 0; i < 32; ++i) a[i] = __fdividef(g[i], 1.0f + __expf(-g[i])) * u[i];
                        const int f = ti.n0 + c;
                        const float* vals[3] = {g, u, a};
                        const CUtensorMap* maps[3] = {mO0, mO0, mO1};
                        const int cols[3] = {f, F + f, f};
                        __nv_bfloat16* direct[3] = {hgu + f, hgu + F + f, actp + f};
                        emit(3, vals, maps, cols, direct);
                    }
                } else if constexpr (EPI == EPI_ROUTE) {
                    // the per-(party, expert) counts: a shared-memory histogram when P E fits
                    // (hist_n > 0), else straight to the global counts
                    int* hist = p.hist_n ? route_hist : p.counts;
                    if constexpr (SHORT)
                        route_epilogue_short<BN, AR>(p, ti, q, warp - 2, lane, tbase, (float*)(stage_out + 4 * p.hist_n), hist);
                    else if constexpr (BN <= 64) route_epilogue<BN>(p, ti, m, valid, tbase, hist);
                    else route_epilogue_wide<BN>(p, ti, m, valid, tbase, hist);
                } else if constexpr (EPI == EPI_DWR) {
                    // one token chunk's partial router gradient: accumulator row m is model
                    // column m, column e is expert e; stored transposed, fp32, part[g][e][m]
                    // (a warp's 32 rows are 32 consecutive floats of one expert row)
                    float* part = (float*)p.out0 + (int64_t)ti.g * p.E * p.Mout + m;
#pragma unroll 1
                    for (int c = 0; c < BN; c += 32) {
                        float v[32];
                        if (ti.k_iters > 0) {
                            tmem_ld32(tbase + c, v);
                        } else {
#pragma unroll
                            for (int i = 0; i < 32; ++i) v[i] = 0.f;
                        }
                        if (valid) {
#pragma unroll
                            for (int i = 0; i < 32; ++i)
                                if (c + i < p.E) part[(int64_t)(c + i) * p.Mout] = v[i];
                        }
                    }
                } else {
                    __nv_bfloat16* out;
                    if (VAR_K)
                        out = (__nv_bfloat16*)p.out0 + (int64_t)ti.we * p.Mout * p.N + (int64_t)m * p.N;
                    else
                        out = (__nv_bfloat16*)out0 + (ti.out_row + m) * (int64_t)N;
#pragma unroll 1
                    for (int c = half * (BN / SPLIT); c < (half + 1) * (BN / SPLIT) && ti.n0 + c < N; c += 32) {
                        float y[32];
                        if (ti.k_iters > 0) {
                            tmem_ld32(tbase + c, y);
                        } else {
#pragma unroll
                            for (int i = 0; i < 32; ++i) y[i] = 0.f;
                        }
                        const float* vals[1] = {y};
                        const CUtensorMap* maps[1] = {sec ? &tmO2 : &tmO0};
                        const int cols[1] = {ti.n0 + c};
                        __nv_bfloat16* direct[1] = {out + ti.n0 + c};
                        emit(1, vals, maps, cols, direct);
                    }
                }
            }
            // release the accumulator: one arrival per warp on the MMA issuer's barrier
            fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (PAIR) {
                    // (a release at cluster scope of everything the warp wrote would wait for
                    // its output too: 3-5% of a launch with short contractions)
                    fence_release_smem_cluster();
                    mbar_arrive_remote(map_to_rank(tempty_bar(acc), 0));
                }
                else mbar_arrive(tempty_bar(acc));
            }
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        if (lane == 0) bulk_wait0();  // every TMA store of this warp has completed
        if constexpr (EPI == EPI_SWIGLU_BWD) {
            // loads issued but not consumed (only after an abort): let them land
            for (uint32_t c = gu_chunk; c < gu_issued; ++c) {
                const uint64_t t0 = gtimer();
                while (!mbar_try(gu_bar0 + 8u * (c & 1), (c >> 1) & 1) && gtimer() - t0 < drain_limit) {
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if constexpr (PAIR) {
        if (threadIdx.x == 0 && *abort_flag) st_cluster(map_to_rank(smem_u32(&s_abort), rank ^ 1u), 1u);
        __syncwarp();
        cluster_sync_all();  // neither CTA leaves while the pair's MMAs run
        if (*abort_flag) {   // (both CTAs see it)
            // The peer's producer may have filled stages that the leader's, giving up first, never
            // armed: the leader arms them for those bytes alone and waits for them.
            if (rank == 0 && threadIdx.x == 0) {
                const uint32_t theirs = ld_cluster(map_to_rank(smem_u32(&s_fills), 1));
                for (uint32_t i = s_fills; i < theirs; ++i) {
                    const uint32_t bytes = ld_cluster(map_to_rank(smem_u32(&s_fill_bytes[i % NST]), 1));
                    if (!bytes) continue;
                    mbar_expect_tx(full_bar(i % NST), bytes);
                    const uint64_t t0 = gtimer();
                    while (!mbar_try(full_bar(i % NST), (i / NST) & 1u) && gtimer() - t0 < drain_limit) {
                    }
                }
            }
            __syncwarp();
            cluster_sync_all();
        }
    }
    fence_after();
    if (warp == 1) {
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                         "r"(TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                         "r"(TMEM_COLS)
                         : "memory");
    }
    if constexpr (EPI == EPI_ROUTE) {
        for (int i = threadIdx.x; i < p.hist_n; i += blockDim.x)
            if (route_hist[i]) atomicAdd(&p.counts[i], route_hist[i]);
    }
}

// ------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    }
    return fn;
}

// 2D bf16 tensor [outer, inner] row-major, box {64, box_rows}, 128B swizzle, zero fill
// (operand loads); with store = true a {32, 32} box, 64B swizzle, for the epilogue's TMA stores.
static bool make_map(CUtensorMap* m, const void* base, int64_t inner, int64_t outer, int box_rows,
                     bool store = false) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    cuuint64_t strides[1] = {(cuuint64_t)inner * 2};
    cuuint32_t box[2] = {store ? (cuuint32_t)EPI_BOX : 64u, store ? (cuuint32_t)EPI_BOX : (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1u, 1u};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                    box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    store ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// The same operand seen as [inner / 64][outer][64], box {64, box_rows, kblocks}: several
// k-blocks in one copy, each in its own swizzled box (the last one zero-filled past inner).
static bool make_map_kblocks(CUtensorMap* m, const void* base, int64_t inner, int64_t outer, int box_rows, int kblocks) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {64u, (cuuint64_t)outer, (cuuint64_t)(inner / 64)};
    cuuint64_t strides[2] = {(cuuint64_t)inner * 2, 128u};
    cuuint32_t box[3] = {64u, (cuuint32_t)box_rows, (cuuint32_t)kblocks};
    cuuint32_t estr[3] = {1u, 1u, 1u};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static uint64_t g_wait_ns = 2000000000ull;
static int g_pairs = MOE_PAIRS_AUTO;  // CTA-pair tiles for the 256-wide M-variable expert GEMMs

// M-tiles per band of the tile order for `c` tiles in flight at once (the persistent
// CTAs, or CTA pairs): about sqrt(c).
static int band_for(int c) {
    int b = 1;
    while ((b + 1) * (b + 1) <= c) ++b;
    return b;
}

template <int BN, bool B_MN, bool VAR_K, int EPI, bool PAIR = false, bool DW2 = false, int OCC = 1, int EW = 4, int AR = BM>
static cudaError_t launch(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mo0,
                          const CUtensorMap& mo1, const Params& p, int64_t tiles_ub,
                          cudaStream_t s, const CUtensorMap* ma2 = nullptr,
                          const CUtensorMap* mb2 = nullptr, const CUtensorMap* mo2 = nullptr,
                          const Params* p2 = nullptr, const CUtensorMap* mas = nullptr, const CUtensorMap* mx2 = nullptr) {
    auto kern = grouped_gemm_kernel<BN, B_MN, VAR_K, EPI, PAIR, DW2, OCC, EW, AR>;
    const CUtensorMap& A2 = ma2 ? *ma2 : ma;
    const CUtensorMap& B2 = mb2 ? *mb2 : mb;
    const CUtensorMap& O2 = mo2 ? *mo2 : mo0;
    const CUtensorMap& AS = mas ? *mas : ma;  // boxes of swapped tiles (M-variable pairs)
    const CUtensorMap& X2 = mx2 ? *mx2 : mo0;
    Params P1 = p;
    Params P2 = p2 ? *p2 : p;
    if (!p2) P2.G = 0;  // no second problem
    constexpr int NPAIR = PAIR ? 2 : 1;
    constexpr int KB = kblock_rows(VAR_K, PAIR, EPI, BN);
    constexpr int STB = (AR * KB * 2 + BN / NPAIR * KB * 2) * kblocks_per_stage(EPI, BN, PAIR, VAR_K, DW2, OCC, AR);  // bytes of one operand stage
    constexpr int NST = num_stages((uint32_t)STB, EPI, OCC, AR);
    const int extra_max = EPI == EPI_ROUTE ? 64 * 64 * 4 : epi_stage_bytes(EPI);
    const int extra = EPI == EPI_ROUTE ? p.hist_n * 4 : epi_stage_bytes(EPI);
    const int smem_max = NST * STB + 1024 + extra_max + mma_overread(AR);
    const int smem = NST * STB + 1024 + extra + mma_overread(AR);
    const cudaError_t e = allow_dynamic_smem<grouped_gemm_kernel<BN, B_MN, VAR_K, EPI, PAIR, DW2, OCC, EW, AR>>(smem_max);
    if (e != cudaSuccess) return e;
    if (tiles_ub <= 0) return cudaSuccess;
    if constexpr (PAIR) {
        // persistent 2-CTA clusters: no more than can be resident at once (a cluster needs
        // both SMs of a TPC, so fewer than SMs/2 may fit)
        static std::atomic<int> resident[kMaxDevices] = {};
        const int dev = current_device();
        int max_clusters = dev >= 0 && dev < kMaxDevices ? resident[dev].load() : 0;
        if (!max_clusters) {
            cudaLaunchConfig_t q = {};
            q.gridDim = dim3(2 * (sm_count() / 2));
            q.blockDim = dim3(gemm_threads(EW));
            q.dynamicSmemBytes = smem_max;
            cudaLaunchAttribute qa[1];
            qa[0].id = cudaLaunchAttributeClusterDimension;
            qa[0].val.clusterDim.x = 2;
            qa[0].val.clusterDim.y = 1;
            qa[0].val.clusterDim.z = 1;
            q.attrs = qa;
            q.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&max_clusters, kern, &q) != cudaSuccess || max_clusters <= 0) {
                (void)cudaGetLastError();
                max_clusters = sm_count() / 2;
            }
            if (dev >= 0 && dev < kMaxDevices) resident[dev] = max_clusters;
        }
        const int clusters = (int)std::min<int64_t>(tiles_ub, max_clusters);
        P1.band = P2.band = band_for(clusters);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * clusters);
        cfg.blockDim = dim3(gemm_threads(EW));
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        return cudaLaunchKernelEx(&cfg, kern, ma, mb, mo0, mo1, AS, P1, A2, B2, O2, X2, P2);
    } else {
        const int grid = (int)std::min<int64_t>(tiles_ub, (int64_t)OCC * sm_count());
        P1.band = P2.band = band_for(grid);
        (void)launch_pdl(kern, dim3(grid), dim3(gemm_threads(EW)), smem, s, ma, mb, mo0, mo1, AS, P1, A2, B2, O2, X2, P2);
        return cudaGetLastError();
    }
}

}  // namespace tc

void set_wait_limit_ns(uint64_t ns) { tc::g_wait_ns = ns ? ns : 1; }
uint64_t wait_limit_ns() { return tc::g_wait_ns; }
void set_gemm_pairs(int mode) { tc::g_pairs = mode; }

// Tiles of `tile` rows that `rows` rows in G groups make, if the router spreads them evenly:
// each group has r = rows / G of them give or take sqrt(r), so the mean of the tiles at half
// a deviation below and above. (The counts are on the device; a rule that waited for them
// would synchronise.) An uneven router ends other tiles: over 60 shapes of 4 to 45 experts,
// 225 to 6400 tokens the rule below takes 0.77 of the time of pairs from four rounds on, at
// Zipf(1.2) popularity (0.47 to 1.04) as at even; of 50 whose tiles lie within a few of a whole
// round 0.98, where a skewed batch can fall on the other side of it (2000 tokens, E = 8,
// d = 1024, F = 2816: 105 -> 115 us of a forward; even 100 -> 99). Averaging the rounds over more
// uneven counts moved such batches about without gain (0.99).
static int64_t expected_tiles(const GroupRows& gr, int G, int tile) {
    if (!gr.offsets) return (int64_t)G * ((gr.rows + tile - 1) / tile);
    const double r = (double)gr.rows / G, dev = 0.5 * std::sqrt(r);
    const double lo = std::ceil(std::max(r - dev, 1.0) / tile), hi = std::ceil((r + dev) / tile);
    return (int64_t)(G * (lo + hi) / 2);
}

// Pair tiles or single-CTA tiles, by rounds: a pair's 256 x 256 tile takes half of the B bytes
// per SM and flop of a 128 x 256 tile, so a round of pairs (two rows of single tiles) takes
// 1 where a round of single tiles takes 1.3 (128 x 128: 1.05), but has half as many tiles and
// loses more in a last round. Measured, pairs against single: dX of 8192 rows, 16 experts,
// d = 1024 (3 rounds, 2) 97, 84 us; of 49152 rows, 64 experts, d = 2048 (24, 22) 351, 409;
// GEMM1 of 4314 rows, 6 experts (2, 2) 41, 47 and of 1092, 4 experts (2, 1) 40, 31; GEMM2 of
// 3009 rows, 13 experts, d = 1152 (1, 2 of 128 x 128) 22, 25; 6 rows an expert, 64 experts,
// d = 2048: GEMM1 (10, 5) 135, 118. With a contraction under 512 the epilogue weighs more:
// pairs only with fewer rounds, or as many from four on (GEMM2 of F = 256 in two: 12.6, 11.4). The
// SwiGLU-backward GEMM (dA) moves G, U, dG and dU in its epilogue: with a short contraction
// (d < 2048) the epilogue bounds it and single-CTA tiles (fused with dW2 in one launch) are
// faster; from d = 2048 the mainloop dominates and pairs win (d = 4096: the expert backward
// 17.8 -> 17.2 ms; d = 1024: +4%).
bool gemm_m_uses_pairs(const GemmMArgs& g, const GemmMArgs* second) {
    using namespace tc;
    if (g.N % 128 != 0) return false;  // 256-wide pair tiles, the last one possibly ragged
    if (g_pairs == MOE_PAIRS_ALL) return true;
    if (g_pairs != MOE_PAIRS_AUTO || g.slim) return false;
    if (g.epi == EPI_SWIGLU_BWD) {
        if (g.K < 2048) return false;
        const int64_t pt_ub = g.rows.offsets ? ((int64_t)g.rows.rows + 2 * BM - 1) / (2 * BM) + g.G
                                             : (int64_t)g.G * ((g.rows.rows + 2 * BM - 1) / (2 * BM));
        return pt_ub * ((g.N + 255) / 256) >= 4 * (int64_t)(sm_count() / 2);
    }
    const bool wide = g.N % 256 == 0;  // (a GEMM1 tile's 256 columns are 128 features, gate and up)
    const int64_t sms = sm_count(), pairs = sms / 2;
    int64_t tp = 0, ts = 0;
    for (const GemmMArgs* q : {&g, second}) {
        if (!q) continue;
        tp += expected_tiles(q->rows, q->G, 2 * BM) * ((q->N + 255) / 256);
        ts += expected_tiles(q->rows, q->G, BM) * (wide ? q->N / 256 : q->N / 128);
    }
    const int64_t rp = (tp + pairs - 1) / pairs, rs = (ts + sms - 1) / sms;
    return g.K < 512 ? rp < rs || (rp == rs && rp >= 4) : rp * 100 <= rs * (wide ? 130 : 105);
}

// K-variable weight gradients (dW = A^T B over each group's rows) as 256 x 256 CTA-pair
// tiles: M a multiple of 256, and (AUTO) no slower by rounds: a launch takes its rounds of
// tiles times a tile's time per contraction row, measured as 4.9 (pairs), 6.7 (128 x 256) and
// 4.5 (128 x 128) in the same unit. (Two shared experts of 8192 rows: dW1 in 3 pair rounds
// where 128 x 256 tiles take 3, dW2 in 2 where 128 x 128 tiles take 3: 166 -> 123 and 157 -> 82 us.)
bool gemm_k_uses_pairs(const GemmKArgs& g) {
    using namespace tc;
    if (g.epi != EPI_STORE || g.M % 256 != 0 || g.N % 128 != 0) return false;
    if (g_pairs == MOE_PAIRS_ALL) return true;
    if (g_pairs != MOE_PAIRS_AUTO) return false;
    const bool wide = g.N % 256 == 0;
    const int64_t pairs = sm_count() / 2, sms = sm_count();
    const int64_t tp = (int64_t)g.G * (g.M / 256) * ((g.N + 255) / 256);
    const int64_t ts = (int64_t)g.G * (g.M / 128) * (wide ? g.N / 256 : g.N / 128);
    return (tp + pairs - 1) / pairs * 49 <= (ts + sms - 1) / sms * (wide ? 67 : 45);
}

// What launch_gemm_m and its second problem share: the kernel's parameters, and the rows of
// A's and the outputs' 2D views (OFFSETS: all routed rows; UNIFORM: groups * stride, or rows).
static tc::Params m_params(const GemmMArgs& g) {
    tc::Params p{};
    p.offsets = g.rows.offsets;
    p.rows = g.rows.offsets ? 0 : g.rows.rows;
    p.a_stride = g.rows.a_stride;
    p.b_stride = g.rows.b_stride;
    p.out_stride = g.rows.out_stride;
    p.G = g.G;
    p.N = g.N;
    p.K = g.K;
    p.out0 = g.out0;
    p.out1 = g.out1;
    p.aux = g.aux;
    p.wait_ns = tc::g_wait_ns;
    p.gexp = g.group_expert;
    p.a_row_bytes = (int64_t)g.K * 2;
    p.b_all_bytes = (int64_t)g.N * (g.b_kmajor ? g.K : (g.b_rows ? g.b_rows : g.K)) * 2;
    if (g.epi == EPI_SWIGLU_FWD) p.F = g.N / 2;
    p.b_group_rows = g.b_kmajor ? g.N : (g.b_rows ? g.b_rows : g.K);
    return p;
}
static int64_t view_rows(const GemmMArgs& g, int64_t stride) {
    return g.rows.offsets ? (int64_t)g.rows.rows : std::max<int64_t>(g.rows.rows, (int64_t)(g.G - 1) * stride + g.rows.rows);
}
// most tiles of `tile` rows that the groups can make
static int64_t max_tiles(const GemmMArgs& g, int tile) {
    return g.rows.offsets ? ((int64_t)g.rows.rows + tile - 1) / tile + g.G : (int64_t)g.G * ((g.rows.rows + tile - 1) / tile);
}

// M-variable grouped GEMM (forward, dA, dX). `second`: another one of the same kind (forward
// GEMMs; uniform groups; for a plain store of the same N) whose tiles follow in the launch.
cudaError_t launch_gemm_m(const GemmMArgs& g, bool bf16, cudaStream_t s, const GemmMArgs* second) {
    if (!bf16) {
        const cudaError_t e = launch_gemm_m_f32(g, s);
        return e == cudaSuccess && second ? launch_gemm_m_f32(*second, s) : e;
    }
    using namespace tc;
    if (g.G > MAX_GROUPS || (second && second->G > MAX_GROUPS)) return cudaErrorInvalidValue;
    Params p = m_params(g);
    const int64_t a_rows = view_rows(g, g.rows.a_stride), o_rows = view_rows(g, g.rows.out_stride);
    const int64_t mt_ub = max_tiles(g, BM), pt_ub = max_tiles(g, 2 * BM);
    const bool pair = gemm_m_uses_pairs(g, second);
    CUtensorMap ma, mb, mo0, mo1, mas;  // mas: A in boxes of 32 rows (swapped tiles)
    if (!make_map(&ma, g.a, g.K, a_rows, BM)) return cudaErrorInvalidValue;
    if (pair && !make_map(&mas, g.a, g.K, a_rows, 32)) return cudaErrorInvalidValue;
    const bool wide_epi = g.K < kWideEpiK;
    if (g.b_kmajor) {  // forward: SwiGLU (B = gate rows then up rows), or Y = A W2^T (B = W2[e] as [N=d, K=F])
        const bool fwd = g.epi == EPI_SWIGLU_FWD;
        // tile columns, and rows of one B box
        const int bn = fwd || pair || g.N % 256 == 0 ? 256 : 128, brows = fwd || pair ? 128 : bn;
        auto maps = [&](const GemmMArgs& q, CUtensorMap* b, CUtensorMap* o0, CUtensorMap* o1) {
            const int64_t rows = view_rows(q, q.rows.out_stride);
            return make_map(b, q.b, q.K, (int64_t)q.G * q.N, brows) && make_map(o0, q.out0, q.N, rows, 0, true) &&
                   (!fwd || make_map(o1, q.out1, q.N / 2, rows, 0, true));
        };
        auto tiles = [&](const GemmMArgs& q) { return max_tiles(q, pair ? 2 * BM : BM) * ((q.N + bn - 1) / bn); };
        if (!maps(g, &mb, &mo0, &mo1)) return cudaErrorInvalidValue;
        if (!fwd) mo1 = mo0;
        int64_t n = tiles(g);
        CUtensorMap a2, b2, o2, x2;
        Params p2;
        const Params* pp2 = nullptr;
        if (second) {
            const int64_t rows2 = view_rows(*second, second->rows.a_stride);
            if (!make_map(&a2, second->a, second->K, rows2, BM) || !maps(*second, &b2, &o2, &x2)) return cudaErrorInvalidValue;
            if (!fwd && !make_map(&x2, second->a, second->K, rows2, 32)) return cudaErrorInvalidValue;
            p2 = m_params(*second);
            pp2 = &p2;
            n += tiles(*second);
        }
        const CUtensorMap *A2 = pp2 ? &a2 : nullptr, *B2 = pp2 ? &b2 : nullptr, *O2 = pp2 ? &o2 : nullptr,
                          *X2 = pp2 ? &x2 : nullptr, *as = pair ? &mas : nullptr;
#define MOE_FWD(BN, EPI, PAIR, EW) \
    return launch<BN, false, false, EPI, PAIR, false, 1, EW>(ma, mb, mo0, mo1, p, n, s, A2, B2, O2, pp2, as, X2)
        if (fwd) {
            if (pair && wide_epi) MOE_FWD(256, EPI_SWIGLU_FWD, true, 8);
            if (pair) MOE_FWD(256, EPI_SWIGLU_FWD, true, 4);
            if (wide_epi) MOE_FWD(256, EPI_SWIGLU_FWD, false, 8);
            MOE_FWD(256, EPI_SWIGLU_FWD, false, 4);
        }
        if (pair && wide_epi) MOE_FWD(256, EPI_STORE, true, 8);
        if (pair) MOE_FWD(256, EPI_STORE, true, 4);
        if (bn == 256 && wide_epi) MOE_FWD(256, EPI_STORE, false, 8);
        if (bn == 256) MOE_FWD(256, EPI_STORE, false, 4);
        if (wide_epi) MOE_FWD(128, EPI_STORE, false, 8);
        MOE_FWD(128, EPI_STORE, false, 4);
#undef MOE_FWD
    }
    // MN-major B: weights stored [G*K, N] (or [G*b_rows, N])
    const bool slim = g.slim && g.epi == EPI_STORE && g.N % 128 == 0;
    const int kps = kblocks_per_stage(g.epi, pair || g.N % 256 == 0 ? 256 : 128, pair, false, false, slim ? 2 : 1, BM);
    if (!make_map(&mb, g.b, g.N, (int64_t)g.G * p.b_group_rows, BK * kps)) return cudaErrorInvalidValue;
    if (g.epi == EPI_SWIGLU_BWD) {
        p.F = g.N;
        if (!make_map(&mo0, g.out0, 2 * (int64_t)g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
        if (!make_map(&mo1, g.aux, 2 * (int64_t)g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
        if (pair)
            return launch<256, true, false, EPI_SWIGLU_BWD, true>(ma, mb, mo0, mo1, p, pt_ub * ((g.N + 255) / 256), s,
                                                                  nullptr, nullptr, nullptr, nullptr, &mas);
        if (g.N % 256 == 0) return launch<256, true, false, EPI_SWIGLU_BWD>(ma, mb, mo0, mo1, p, mt_ub * (g.N / 256), s);
        return launch<128, true, false, EPI_SWIGLU_BWD>(ma, mb, mo0, mo1, p, mt_ub * (g.N / 128), s);
    }
    if (!make_map(&mo0, g.out0, g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
    if (slim)
        return launch<128, true, false, EPI_STORE, false, false, 2>(ma, mb, mo0, mo0, p, mt_ub * (g.N / 128), s);
    if (pair)
        return launch<256, true, false, EPI_STORE, true>(ma, mb, mo0, mo0, p, pt_ub * ((g.N + 255) / 256), s, nullptr, nullptr,
                                                         nullptr, nullptr, &mas);
    if (g.N % 256 == 0) return launch<256, true, false, EPI_STORE>(ma, mb, mo0, mo0, p, mt_ub * (g.N / 256), s);
    return launch<128, true, false, EPI_STORE>(ma, mb, mo0, mo0, p, mt_ub * (g.N / 128), s);
}

// K-variable grouped GEMM (dW1, dW2).
cudaError_t launch_gemm_k(const GemmKArgs& g, bool bf16, cudaStream_t s) {
    if (!bf16) return launch_gemm_k_f32(g, s);
    using namespace tc;
    if (g.G > MAX_GROUPS) return cudaErrorInvalidValue;
    Params p{};
    p.offsets = g.rows.offsets;
    p.rows = g.rows.offsets ? 0 : g.rows.rows;
    p.a_stride = g.rows.a_stride;
    p.b_stride = g.rows.b_stride;
    p.G = g.G;
    p.N = g.N;
    p.Mout = g.M;
    p.out0 = g.out;
    p.wait_ns = g_wait_ns;
    p.gexp = g.group_expert;
    p.a_row_bytes = (int64_t)g.M * 2;
    p.b_row_bytes = (int64_t)g.N * 2;
    const int64_t rows_a = g.rows.offsets ? (int64_t)g.rows.rows
                                          : std::max<int64_t>(g.rows.rows, (int64_t)(g.G - 1) * g.rows.a_stride + g.rows.rows);
    const int64_t rows_b = g.rows.offsets ? (int64_t)g.rows.rows
                                          : std::max<int64_t>(g.rows.rows, (int64_t)(g.G - 1) * g.rows.b_stride + g.rows.rows);
    CUtensorMap ma, mb, mo;
    const bool pair = g.epi == EPI_STORE && gemm_k_uses_pairs(g);
    const int kbr = kblock_rows(true, pair, g.epi, g.N % 256 ? 128 : 256);  // box rows of the MN-major operands
    if (!make_map(&ma, g.a, g.M, rows_a, kbr)) return cudaErrorInvalidValue;
    if (!make_map(&mb, g.b, g.N, rows_b, kbr)) return cudaErrorInvalidValue;
    const int64_t tiles = (int64_t)g.G * (g.M / BM);
    if (g.epi == EPI_DWR) {  // fp32 partials, N = 64, 128 or 256 (experts, zero-padded)
        if ((g.N != 64 && g.N != 128 && g.N != 256) || g.M % BM) return cudaErrorInvalidValue;
        p.E = g.E;
        // two CTAs per SM where TMEM allows: each streams its token chunk of x from HBM at
        // a per-CTA rate, and every tile is resident in one round
        if (g.N == 64) return launch<64, true, true, EPI_DWR, false, false, 2>(ma, mb, ma, ma, p, tiles, s);
        if (g.N == 128) return launch<128, true, true, EPI_DWR, false, false, 2>(ma, mb, ma, ma, p, tiles, s);
        return launch<256, true, true, EPI_DWR>(ma, mb, ma, ma, p, tiles, s);
    }
    if (!make_map(&mo, g.out, g.N, (int64_t)g.G * g.M, 0, true)) return cudaErrorInvalidValue;
    const int64_t pair_tiles = (int64_t)g.G * (g.M / 256) * ((g.N + 255) / 256);
    if ((g.rows.offsets ? (int64_t)g.rows.rows / g.G : (int64_t)g.rows.rows) < kWideEpiRows) {
        if (pair) return launch<256, true, true, EPI_STORE, true, false, 1, 8>(ma, mb, mo, mo, p, pair_tiles, s);
        if (g.N % 256 == 0) return launch<256, true, true, EPI_STORE, false, false, 1, 8>(ma, mb, mo, mo, p, tiles * (g.N / 256), s);
        return launch<128, true, true, EPI_STORE, false, false, 1, 8>(ma, mb, mo, mo, p, tiles * (g.N / 128), s);
    }
    if (pair) return launch<256, true, true, EPI_STORE, true>(ma, mb, mo, mo, p, pair_tiles, s);
    if (g.N % 256 == 0) return launch<256, true, true, EPI_STORE>(ma, mb, mo, mo, p, tiles * (g.N / 256), s);
    return launch<128, true, true, EPI_STORE>(ma, mb, mo, mo, p, tiles * (g.N / 128), s);
}

// One launch of an M-variable GEMM with MN-major B (dA with the SwiGLU-backward
// epilogue, or dX) and a K-variable weight-gradient GEMM over the same groups (dW2, or
// dW1), where both fit one 256-wide template (see the DW2 kernel parameter), else two.
bool gemm_mk_fits(const GemmMArgs& g, const GemmKArgs& k) {
    return g.rows.offsets && k.rows.offsets && g.G == k.G && !g.b_kmajor && (g.epi == EPI_SWIGLU_BWD || g.epi == EPI_STORE) &&
           g.N % 256 == 0 && k.N % 256 == 0 && k.M % tc::BM == 0 && k.epi == EPI_STORE && g.G <= tc::MAX_GROUPS;
}
cudaError_t launch_gemm_mk(const GemmMArgs& g, const GemmKArgs& k, cudaStream_t s) {
    using namespace tc;
    if (!gemm_mk_fits(g, k)) {
        cudaError_t e = launch_gemm_m(g, true, s);
        if (e != cudaSuccess) return e;
        return launch_gemm_k(k, true, s);
    }
    // first problem (as launch_gemm_m, MN-major B)
    Params p{};
    p.offsets = g.rows.offsets;
    p.G = g.G;
    p.N = g.N;
    p.K = g.K;
    p.out0 = g.out0;
    p.out1 = g.out1;
    p.aux = g.aux;
    p.wait_ns = g_wait_ns;
    p.gexp = g.group_expert;
    p.b_group_rows = g.b_rows ? g.b_rows : g.K;
    p.a_row_bytes = (int64_t)g.K * 2;
    p.b_all_bytes = (int64_t)g.N * p.b_group_rows * 2;
    const int64_t a_rows = (int64_t)g.rows.rows, o_rows = a_rows;
    CUtensorMap ma, mb, mo0, mo1;
    if (!make_map(&ma, g.a, g.K, a_rows, BM)) return cudaErrorInvalidValue;
    if (!make_map(&mb, g.b, g.N, (int64_t)g.G * p.b_group_rows, 64)) return cudaErrorInvalidValue;
    if (g.epi == EPI_SWIGLU_BWD) {
        p.F = g.N;
        if (!make_map(&mo0, g.out0, 2 * (int64_t)g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
        if (!make_map(&mo1, g.aux, 2 * (int64_t)g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
    } else {
        if (!make_map(&mo0, g.out0, g.N, o_rows, 0, true)) return cudaErrorInvalidValue;
        mo1 = mo0;
    }
    // second problem (as launch_gemm_k)
    Params p2{};
    p2.offsets = k.rows.offsets;
    p2.G = k.G;
    p2.N = k.N;
    p2.Mout = k.M;
    p2.out0 = k.out;
    p2.wait_ns = g_wait_ns;
    p2.gexp = k.group_expert;
    p2.a_row_bytes = (int64_t)k.M * 2;
    p2.b_row_bytes = (int64_t)k.N * 2;
    CUtensorMap ma2, mb2, mo2;
    if (!make_map(&ma2, k.a, k.M, (int64_t)k.rows.rows, 64)) return cudaErrorInvalidValue;
    if (!make_map(&mb2, k.b, k.N, (int64_t)k.rows.rows, 64)) return cudaErrorInvalidValue;
    if (!make_map(&mo2, k.out, k.N, (int64_t)k.G * k.M, 0, true)) return cudaErrorInvalidValue;
    const int64_t tiles = (((int64_t)g.rows.rows + BM - 1) / BM + g.G) * (g.N / 256) +
                          (int64_t)k.G * (k.M / BM) * (k.N / 256);
    if (g.epi == EPI_SWIGLU_BWD)
        return launch<256, true, false, EPI_SWIGLU_BWD, false, true>(ma, mb, mo0, mo1, p, tiles, s,
                                                                     &ma2, &mb2, &mo2, &p2);
    return launch<256, true, false, EPI_STORE, false, true>(ma, mb, mo0, mo1, p, tiles, s, &ma2,
                                                            &mb2, &mo2, &p2);
}

// Router logits on the tensor cores with the gating epilogue: groups are parties
// (rows [po[p], po[p+1]) use W_r[p]); N = E rounded up to 16, 32 or 64.
cudaError_t launch_route_tc(const RouteArgs& a, cudaStream_t s) {
    using namespace tc;
    Params p{};
    if (a.po && a.P > 1) {
        p.offsets = a.po;
        p.G = a.P;
    } else {
        p.rows = (int)a.T;
        p.G = 1;
    }
    p.K = a.d;
    p.E = a.E;
    p.k = a.k;
    p.normalize = a.normalize;
    p.hist_n = a.P * a.E <= 64 * 64 ? a.P * a.E : 0;  // else counted in global memory
    p.out0 = a.logits;
    p.out1 = a.probs;
    p.aux = a.bias;
    p.topk_idx = a.topk_idx;
    p.topk_w = a.topk_w;
    p.counts = a.counts;
    p.b_group_rows = a.E;
    p.wait_ns = g_wait_ns;
    const int BNr = a.E <= 16 ? 16 : a.E <= 32 ? 32 : a.E <= 64 ? 64 : a.E <= 128 ? 128 : 256;
    if (a.E > 256) return cudaErrorInvalidValue;
    p.N = BNr;
    // rows per tile: the batch split evenly over the SMs (one tile each) when that is
    // under 128 rows, at least 16
    const int64_t share = (a.T + sm_count() - 1) / sm_count();
    p.tile_rows = (int)std::max<int64_t>(16, std::min<int64_t>(BM, share));
    const int64_t tiles = (a.T + p.tile_rows - 1) / p.tile_rows + a.P;
    const int ar = BNr > 64 || p.tile_rows > 32 ? BM : p.tile_rows > 16 ? 32 : 16;
    const int kps = kblocks_per_stage(EPI_ROUTE, BNr, false, false, false, 1, ar);
    CUtensorMap ma, mb;
    if (ar < BM) {
        if (!make_map_kblocks(&ma, a.x, a.d, a.T, ar, kps)) return cudaErrorInvalidValue;
        if (!make_map_kblocks(&mb, a.w_router, a.d, (int64_t)a.P * a.E, BNr, kps)) return cudaErrorInvalidValue;
    } else {
        if (!make_map(&ma, a.x, a.d, a.T, p.tile_rows)) return cudaErrorInvalidValue;
        if (!make_map(&mb, a.w_router, a.d, (int64_t)a.P * a.E, BNr)) return cudaErrorInvalidValue;
    }
#define MOE_ROUTE(BN, AR) return launch<BN, false, false, EPI_ROUTE, false, false, 1, 4, AR>(ma, mb, ma, ma, p, tiles, s)
    if (ar == 16) {
        if (BNr == 16) MOE_ROUTE(16, 16);
        if (BNr == 32) MOE_ROUTE(32, 16);
        MOE_ROUTE(64, 16);
    }
    if (ar == 32) {
        if (BNr == 16) MOE_ROUTE(16, 32);
        if (BNr == 32) MOE_ROUTE(32, 32);
        MOE_ROUTE(64, 32);
    }
    if (BNr == 16) MOE_ROUTE(16, BM);
    if (BNr == 32) MOE_ROUTE(32, BM);
    if (BNr == 64) MOE_ROUTE(64, BM);
#undef MOE_ROUTE
    if (BNr == 128) return launch<128, false, false, EPI_ROUTE>(ma, mb, ma, ma, p, tiles, s);
    return launch<256, false, false, EPI_ROUTE>(ma, mb, ma, ma, p, tiles, s);
}

cudaError_t gemm_status(cudaStream_t s, int* code) { return tu_status_read_clear(s, code); }

}  // namespace moe

// Gating function of the MoE layer (Alg. 7) and its backward, plus the per-party
// load-balancing loss, on the CUDA cores (the bf16 router's GEMMs are in gemm_tc.cu): 16-byte
// vector loads, reductions by warp shuffles, top-k as a warp argmax.
#include <cfloat>

#include <cooperative_groups.h>

#include <algorithm>

#include "moe_common.cuh"
#include "moe_internal.h"

namespace moe {

namespace cg = cooperative_groups;

// ----------------------------------------------------------------------------- top-k
// Per token, lane l owns experts l + 32 i, i < NV (E <= 32 NV). Picks the k largest
// logits, descending, equal logits by ascending expert id; writes logits (optional),
// probs, topk idx / w and bumps the block histogram (or the global counts when the
// histogram does not fit in shared memory).
__device__ __forceinline__ bool better(float va, int ia, float vb, int ib) {
    return va > vb || (va == vb && ia < ib);
}

template <int NV>
__device__ void softmax_topk_token(const float (&z)[NV], int lane, int E, int k, int normalize,
                                   int64_t t, int party, float* logits, float* probs,
                                   int32_t* topk_idx, float* topk_w, int* s_hist) {
    bool val[NV], taken[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        val[i] = lane + 32 * i < E;
        taken[i] = !val[i];
    }
    if (logits) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (val[i]) logits[t * E + lane + 32 * i] = z[i];
    }
    float m = -FLT_MAX;
#pragma unroll
    for (int i = 0; i < NV; ++i) m = fmaxf(m, val[i] ? z[i] : -FLT_MAX);
    m = warp_max(m);
    float x[NV], loc = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        x[i] = val[i] ? expf(z[i] - m) : 0.f;
        loc += x[i];
    }
    const float s = warp_sum(loc);
    float p[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        p[i] = x[i] / s;
        if (val[i]) probs[t * E + lane + 32 * i] = p[i];
    }
    float wsel = 0.f, wsum = 0.f;
    int isel = 0;
    for (int j = 0; j < k; ++j) {
        // local candidate
        float cv = -FLT_MAX;
        int ci = 0x7fffffff;
        bool have = false;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if (!taken[i] && (!have || better(z[i], lane + 32 * i, cv, ci))) {
                cv = z[i];
                ci = lane + 32 * i;
                have = true;
            }
        }
        int hv = have ? 1 : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            float ov = __shfl_xor_sync(0xffffffffu, cv, o);
            int oi = __shfl_xor_sync(0xffffffffu, ci, o);
            int oh = __shfl_xor_sync(0xffffffffu, hv, o);
            if (oh && (!hv || better(ov, oi, cv, ci))) { cv = ov; ci = oi; hv = 1; }
        }
        // ci is the winner on every lane; its owner lane holds its probability
        const int owner = ci & 31, slot = ci >> 5;
        float mine = 0.f;
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (i == slot) mine = p[i];
        const float pw = __shfl_sync(0xffffffffu, mine, owner);
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (ci == lane + 32 * i) taken[i] = true;
        if (lane == j) { isel = ci; wsel = pw; }
        wsum += pw;
        if (lane == 0) atomicAdd(&s_hist[party * E + ci], 1);
    }
    if (lane < k) {
        topk_idx[t * k + lane] = isel;
        topk_w[t * k + lane] = normalize ? wsel / wsum : wsel;
    }
}

// ----------------------------------------------------------------------------- router fwd
// Router logits and gating of the fp32 configuration, up to 64 experts, on the CUDA cores. One CTA
// takes TB consecutive tokens of one party and all experts (padded to EP): chunks of RD_KC columns
// of x and W_r are staged in shared memory (the next chunk's global loads are in flight meanwhile), and
// thread (ks, tg, eg) multiplies TB/4 tokens by 4 experts over the columns of its slice ks.
// A chunk's products are summed on their own before they join the running sum, so no chain
// of additions is longer than about d / 128 + 32. The KS slices of a logit are then added
// through shared memory and each warp gates its tokens. With few tokens a cluster of CTAs
// shares a group: each takes a part of the columns, and the first adds the parts in order
// from distributed shared memory and gates.
//
// What bounds it: with large pools the shared-memory reads (12 wavefronts per 64 FMAs of a
// warp), with small ones the latency of the d / 128 chunk steps. The kernel that it replaces
// (a warp per 1 to 8 tokens, W_r read from L2 by every warp) took 288 us for 4096 tokens of
// d = 2048 with E = 64, now 60; 19 -> 4.8 us for 512 of 256 with E = 8. The chunks' sums are
// closer to 64 bits than its chains (1.3e-7 of 1.6e-7 there).
constexpr int RD_KC = 128;         // columns per chunk
constexpr int RD_LD = RD_KC + 4;   // row pitch in shared memory: rows start 16 bytes apart in the banks
constexpr int RD_THREADS = 256;

template <int EP, int TB>
__global__ void __launch_bounds__(RD_THREADS, EP <= 16 && TB == 8 ? 4 : 2) route_dot_kernel(
    const float* __restrict__ x, const float* __restrict__ wr, const float* __restrict__ bias,
    const int32_t* __restrict__ po, int P, int64_t Tn, int d, int E, int k, int normalize, float* logits,
    float* probs, int32_t* topk_idx, float* topk_w, int32_t* counts) {
    pdl_begin();
    using T = float;
    constexpr int NV = (EP + 31) / 32, VN = Vec<T>::N;
    constexpr int EG = EP / 4, TM = TB / 4, KS = RD_THREADS / EP;  // 4 EG tiles of TM x 4, KS slices
    constexpr int ROWV = RD_KC / VN;                               // vectors per staged row
    constexpr int XV = (TB * ROWV + RD_THREADS - 1) / RD_THREADS, WV = (EP * ROWV + RD_THREADS - 1) / RD_THREADS;
    extern __shared__ float s_dyn[];  // two buffers of [TB + EP][RD_LD]; then the slices' sums
    __shared__ int s_hist[EP];
    const int tid = threadIdx.x;
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part_no = (int)cluster.block_rank();
    // the CTA's columns: a run of whole chunks
    const int per = ((d + RD_KC - 1) / RD_KC + parts - 1) / parts * RD_KC;
    const int c_beg = min(d, per * part_no), c_end = min(d, c_beg + per);
    // the cluster's tokens: group blockIdx.x / parts of TB tokens, enumerated party by party
    int party = -1, n = 0;
    int64_t t0 = 0, g = blockIdx.x / parts;
    for (int q = 0; q < P && party < 0; ++q) {
        const int64_t a = po ? po[q] : 0, b = po ? po[q + 1] : Tn;
        const int64_t ng = b > a ? (b - a + TB - 1) / TB : 0;
        if (g < ng) {
            party = q;
            t0 = a + g * TB;
            n = (int)min64(TB, b - t0);
        }
        g -= ng;
    }
    if (party < 0) return;  // (the whole cluster)
    if (tid < EP) s_hist[tid] = 0;
    const T* W = wr + (int64_t)party * E * d;
    uint4 xr[XV], wv[WV];
    auto fetch = [&](int c0) {
#pragma unroll
        for (int i = 0; i < XV; ++i) {
            const int v = tid + i * RD_THREADS, r = v / ROWV, c = c0 + (v % ROWV) * VN;
            xr[i] = r < n && c < c_end ? Vec<T>::raw_load(x + (t0 + r) * d + c) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int i = 0; i < WV; ++i) {
            const int v = tid + i * RD_THREADS, r = v / ROWV, c = c0 + (v % ROWV) * VN;
            wv[i] = r < E && c < c_end ? Vec<T>::raw_load(W + (int64_t)r * d + c) : make_uint4(0, 0, 0, 0);
        }
    };
    auto put = [&](float* buf) {
#pragma unroll
        for (int i = 0; i < XV + WV; ++i) {
            const int v = tid + (i < XV ? i : i - XV) * RD_THREADS, r = v / ROWV;
            if (r >= (i < XV ? TB : EP)) continue;
            float f[VN];
            unpack_vec<T>(i < XV ? xr[i < XV ? i : 0] : wv[i < XV ? 0 : i - XV], f);
            float* dst = buf + ((i < XV ? 0 : TB) + r) * RD_LD + (v % ROWV) * VN;
#pragma unroll
            for (int h = 0; h < VN; h += 4) Vec<float>::store(dst + h, f + h);
        }
    };
    const int eg = tid % EG, tg = (tid / EG) % 4, ks = tid / (4 * EG);
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    if (c_beg < c_end) {
        fetch(c_beg);
        put(s_dyn);
    }
    __syncthreads();
    int cur = 0;
    for (int c0 = c_beg; c0 < c_end; c0 += RD_KC) {
        const bool more = c0 + RD_KC < c_end;
        if (more) fetch(c0 + RD_KC);
        const float* xs = s_dyn + cur * (TB + EP) * RD_LD + tg * RD_LD;
        const float* ws = s_dyn + cur * (TB + EP) * RD_LD + (TB + eg) * RD_LD;
        float part[TM][4];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) part[i][j] = 0.f;
#pragma unroll 2
        for (int q = ks; q < RD_KC / 4; q += KS) {
            float xv[TM][4], wq[4][4];
#pragma unroll
            for (int i = 0; i < TM; ++i) Vec<float>::load(xs + 4 * i * RD_LD + 4 * q, xv[i]);
#pragma unroll
            for (int j = 0; j < 4; ++j) Vec<float>::load(ws + EG * j * RD_LD + 4 * q, wq[j]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) part[i][j] = fmaf(xv[i][u], wq[j][u], part[i][j]);
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] += part[i][j];
        if (more) put(s_dyn + (cur ^ 1) * (TB + EP) * RD_LD);
        __syncthreads();
        cur ^= 1;
    }
    // [KS][TB][EP] slice sums (token tg + 4 i, expert eg + EG j)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s_dyn[(ks * TB + tg + 4 * i) * EP + eg + EG * j] = acc[i][j];
    __syncthreads();
    // their sum per (token, expert), in the region after the slices
    float* s_sum = s_dyn + RD_THREADS * TB;
    for (int i = tid; i < n * EP; i += RD_THREADS) {
        float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < KS; ++q) s4[q & 3] += s_dyn[q * TB * EP + i];
        s_sum[i] = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    }
    if (parts > 1) cluster.sync();
    else __syncthreads();
    if (part_no == 0) {
        const int lane = tid & 31;
        for (int tt = tid >> 5; tt < n; tt += RD_THREADS / 32) {
            float z[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int e = lane + 32 * v;
                z[v] = 0.f;
                if (e < E) {
                    for (int q = 0; q < parts; ++q)
                        z[v] += (q ? cluster.map_shared_rank(s_sum, q) : s_sum)[tt * EP + e];
                    if (bias) z[v] += bias[party * E + e];
                }
            }
            softmax_topk_token<NV>(z, lane, E, k, normalize, t0 + tt, 0, logits, probs, topk_idx, topk_w, s_hist);
        }
    }
    if (parts > 1) cluster.sync();  // the parts' shared memory has been read
    if (part_no) return;
    __syncthreads();
    if (tid < E && s_hist[tid]) atomicAdd(&counts[party * E + tid], s_hist[tid]);
}

// Router logits and gating of bf16 pools whose size is not a multiple of 4, up to 64 experts. A CTA
// takes TB consecutive tokens of one party and all experts (padded to EP), a warp EM = EP / 8 of
// the experts; lane l multiplies the 16-byte vectors l, l + 32, ... of the rows (the next ones are
// in flight meanwhile), each (token, expert) in one chain of FMAs per lane, and the 32 chains are
// added by a butterfly. That order of summation matters: the chunked one of the fp32 kernel above
// leaves bf16 logits up to a quarter further off 64 bits (1.07e-7 against 8.7e-8 at d = 3072, E = 63).
//
// What bounds it: FMA issue for large batches and pools (a step of TB = EM = 8 is 512 FMAs, 128
// conversions and 16 loads a warp), the latency of the d / 256 steps for small ones. 3805 tokens of
// d = 3072 with E = 63: 70 us (a warp per 1 to 8 tokens with the same sums took 308, the chunked
// kernel 73); 16372, 3072, 43: 246 (965, 275); 1003, 1152, 13: 10.3 (34, 11.9).
// a[i], i < N, summed over the warp's lanes by the butterfly of warp_sum, each lane keeping N / 32
// of the sums (those from lane * N / 32 on; N < 32: sum lane / (32 / N))
template <int N>
__device__ __forceinline__ void warp_sums(float (&a)[N], int lane) {
#pragma unroll
    for (int o = 16, n = N; o > 0; o >>= 1) {
        if (n > 1) {
            n /= 2;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i >= n) break;
                const float send = (lane & o) ? a[i] : a[i + n], keep = (lane & o) ? a[i + n] : a[i];
                a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        } else {
            a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
        }
    }
}

template <int EP, int TB>
__global__ void __launch_bounds__(RD_THREADS, TB * EP >= 256 ? 1 : 2) route_chain_kernel(
    const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ wr, const float* __restrict__ bias,
    const int32_t* __restrict__ po, int P, int64_t Tn, int d, int E, int k, int normalize, float* logits,
    float* probs, int32_t* topk_idx, float* topk_w, int32_t* counts) {
    pdl_begin();
    using T = __nv_bfloat16;
    constexpr int NV = (EP + 31) / 32, VN = Vec<T>::N, EM = EP / (RD_THREADS / 32), N = TB * EM;
    __shared__ float s_z[TB][EP];
    __shared__ int s_hist[EP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, e0 = warp * EM;
    // the CTA's tokens: group blockIdx.x of TB tokens, enumerated party by party
    int party = -1, n = 0;
    int64_t t0 = 0, g = blockIdx.x;
    for (int q = 0; q < P && party < 0; ++q) {
        const int64_t a = po ? po[q] : 0, b = po ? po[q + 1] : Tn;
        const int64_t ng = b > a ? (b - a + TB - 1) / TB : 0;
        if (g < ng) {
            party = q;
            t0 = a + g * TB;
            n = (int)min64(TB, b - t0);
        }
        g -= ng;
    }
    if (party < 0) return;
    if (tid < EP) s_hist[tid] = 0;
    const int nvec = d / VN;
    const T *X = x + t0 * d, *W = wr + ((int64_t)party * E + e0) * d;
    uint4 xr[TB], wv[EM];
    auto fetch = [&](int v) {
#pragma unroll
        for (int i = 0; i < TB; ++i)
            xr[i] = i < n && v < nvec ? Vec<T>::raw_load(X + (int64_t)i * d + v * VN) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < EM; ++j)
            wv[j] = e0 + j < E && v < nvec ? Vec<T>::raw_load(W + (int64_t)j * d + v * VN) : make_uint4(0, 0, 0, 0);
    };
    float acc[N];  // token i, expert e0 + j: i * EM + j
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = 0.f;
    if (e0 < E) {  // (a whole warp)
        fetch(lane);
#pragma unroll 1
        for (int v = lane; v - lane < nvec; v += 32) {
            uint4 xc[TB], wc[EM];
#pragma unroll
            for (int i = 0; i < TB; ++i) xc[i] = xr[i];
#pragma unroll
            for (int j = 0; j < EM; ++j) wc[j] = wv[j];
            fetch(v + 32);
            // the vectors' columns in order
#pragma unroll
            for (int c = 0; c < VN; ++c) {
                auto value = [&](const uint4& u) {
                    const uint32_t w = c < 2 ? u.x : c < 4 ? u.y : c < 6 ? u.z : u.w;
                    return __uint_as_float(c % 2 ? w & 0xffff0000u : w << 16);
                };
                float wq[EM];
#pragma unroll
                for (int j = 0; j < EM; ++j) wq[j] = value(wc[j]);
#pragma unroll
                for (int i = 0; i < TB; ++i) {
                    const float xq = value(xc[i]);
#pragma unroll
                    for (int j = 0; j < EM; ++j) acc[i * EM + j] = fmaf(xq, wq[j], acc[i * EM + j]);
                }
            }
        }
    }
    warp_sums<N>(acc, lane);
    constexpr int KEEP = N / 32 > 0 ? N / 32 : 1, LANES = N < 32 ? 32 / N : 1;  // sums a lane, lanes a sum
    if (lane % LANES == 0) {
#pragma unroll
        for (int i = 0; i < KEEP; ++i) {
            const int q = lane / LANES * KEEP + i;
            s_z[q / EM][e0 + q % EM] = acc[i];
        }
    }
    __syncthreads();
    for (int tt = warp; tt < n; tt += RD_THREADS / 32) {
        float z[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int e = lane + 32 * v;
            z[v] = e < E ? s_z[tt][e] : 0.f;
            if (bias && e < E) z[v] += bias[party * E + e];
        }
        softmax_topk_token<NV>(z, lane, E, k, normalize, t0 + tt, 0, logits, probs, topk_idx, topk_w, s_hist);
    }
    __syncthreads();
    if (tid < E && s_hist[tid]) atomicAdd(&counts[party * E + tid], s_hist[tid]);
}

// Gating alone, on logits that exist ([T,E] fp32), one warp per group of up to TPW
// consecutive tokens of one party. With a bias they are the router's raw products (E > 64,
// computed by a GEMM): the bias is added here and the biased logits are written back to
// `logits` (which may be logits_in). The per-(party, expert) counts go through a
// shared-memory histogram when P E fits (HIST_SMEM), else straight to the global counts.
constexpr int HIST_SMEM = 4096;
template <int EMAX, int TPW>
__global__ void __launch_bounds__(256) route_kernel(
    const float* __restrict__ bias, const float* logits_in, const int32_t* __restrict__ po, int P, int64_t Tn,
    int E, int k, int normalize, float* logits, float* probs, int32_t* topk_idx, float* topk_w, int32_t* counts) {
    pdl_begin();
    constexpr int NV = (EMAX + 31) / 32;
    extern __shared__ int s_hist_dyn[];  // [P*E] when it fits
    const bool hist_smem = P * E <= HIST_SMEM;
    int* s_hist = hist_smem ? s_hist_dyn : counts;
    if (hist_smem) {
        for (int i = threadIdx.x; i < P * E; i += blockDim.x) s_hist[i] = 0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warps_total = gridDim.x * (blockDim.x >> 5);
    // groups are enumerated party by party
    int64_t total_groups = 0;
    for (int p = 0; p < P; ++p) {
        int64_t a = po ? po[p] : 0, b = po ? po[p + 1] : Tn;
        total_groups += (b - a + TPW - 1) / TPW;
    }
    for (int64_t gi = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); gi < total_groups;
         gi += warps_total) {
        int party = 0;
        int64_t g = gi, t0 = 0, tend = Tn;
        for (int p = 0; p < P; ++p) {
            int64_t a = po ? po[p] : 0, b = po ? po[p + 1] : Tn;
            int64_t ng = (b - a + TPW - 1) / TPW;
            if (g < ng) { party = p; t0 = a + g * TPW; tend = b; break; }
            g -= ng;
        }
        const int n = (int)min64(TPW, tend - t0);
        float z[TPW][NV];
#pragma unroll
        for (int i = 0; i < TPW; ++i)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const int e = lane + 32 * v;
                z[i][v] = (i < n && e < E) ? logits_in[(t0 + i) * E + e] : 0.f;
                if (bias && e < E) z[i][v] += bias[party * E + e];
            }
#pragma unroll
        for (int i = 0; i < TPW; ++i)
            if (i < n)
                softmax_topk_token<NV>(z[i], lane, E, k, normalize, t0 + i, party, bias ? logits : nullptr, probs,
                                       topk_idx, topk_w, s_hist);
    }
    __syncthreads();
    if (hist_smem) {
        for (int i = threadIdx.x; i < P * E; i += blockDim.x)
            if (s_hist[i]) atomicAdd(&counts[i], s_hist[i]);
    }
}

// ----------------------------------------------------------------------------- aux loss
// One 8-CTA thread-block cluster per party: each CTA sums probs[t, e] over its slice
// of the party's tokens, then CTA 0 of the cluster adds the 8 partial rows from
// distributed shared memory in rank order. Inside a CTA, thread (s, e) of S = 2^j
// stripes per expert loads AUX_U values of its stripe at once (independent loads in
// flight) and adds them in order; the stripes are then added by a fixed binary tree.
// Deterministic, no workspace, no floating-point atomics.
constexpr int AUX_CLUSTER = 8;
constexpr int AUX_THREADS = 1024;
constexpr int AUX_U = 8;

__device__ __forceinline__ int pow2_floor(int v) {
    int r = 1;
    while (2 * r <= v) r *= 2;
    return r;
}

__global__ void __cluster_dims__(AUX_CLUSTER, 1, 1) __launch_bounds__(AUX_THREADS)
    aux_loss_kernel(const float* __restrict__ probs, const int32_t* __restrict__ counts,
                    const int32_t* __restrict__ po, int64_t Tn, int E, int k, float alpha,
                    float* loss, float* coef) {
    pdl_begin();
    __shared__ float s_part[AUX_THREADS];
    __shared__ float s_col[256];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int p = blockIdx.x / AUX_CLUSTER;
    const int64_t a = po ? po[p] : 0, b = po ? po[p + 1] : Tn;
    const int64_t n = b - a;
    const int64_t per = (n + AUX_CLUSTER - 1) / AUX_CLUSTER;
    const int64_t lo = a + min64(n, per * rank), hi = a + min64(n, per * (rank + 1));
    const int tid = threadIdx.x;
    const int stripes = pow2_floor(AUX_THREADS / E);
    float acc = 0.f;
    if (tid < stripes * E) {
        const int e = tid % E, st = tid / E;
        for (int64_t t = lo + st; t < hi; t += (int64_t)AUX_U * stripes) {
            float v[AUX_U];
#pragma unroll
            for (int u = 0; u < AUX_U; ++u) {
                const int64_t tt = t + (int64_t)u * stripes;
                v[u] = tt < hi ? probs[tt * E + e] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < AUX_U; ++u) acc += v[u];
        }
    }
    s_part[tid] = acc;
    __syncthreads();
    for (int h = stripes / 2; h > 0; h >>= 1) {
        if (tid < h * E) s_part[tid] += s_part[tid + h * E];
        __syncthreads();
    }
    if (tid < E) s_col[tid] = s_part[tid];
    cluster.sync();
    if (rank == 0 && tid < E) {
        float tot = 0.f;
        for (int r = 0; r < AUX_CLUSTER; ++r) tot += cluster.map_shared_rank(s_col, r)[tid];
        const float Tp = (float)n;
        const float f = (n > 0) ? (float)counts[p * E + tid] / (Tp * k) : 0.f;
        const float Pm = (n > 0) ? tot / Tp : 0.f;
        s_part[tid] = f * Pm;
        coef[p * E + tid] = (n > 0) ? alpha * E * f / Tp : 0.f;
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        float L = 0.f;
        for (int e = 0; e < E; ++e) L += s_part[e];
        loss[p] = alpha * E * L;
    }
}

// ----------------------------------------------------------------------------- router bwd
// Token chunks never straddle a party: chunk ci of the enumeration party by party.
__device__ __forceinline__ bool chunk_of(int64_t ci, const int32_t* po, int P, int64_t Tn,
                                         int CH, int* party, int64_t* t0, int* n) {
    for (int p = 0; p < P; ++p) {
        int64_t a = po ? po[p] : 0, b = po ? po[p + 1] : Tn;
        int64_t nc = (b - a + CH - 1) / CH;
        if (ci < nc) {
            *party = p;
            *t0 = a + ci * CH;
            *n = (int)min64(CH, b - *t0);
            return true;
        }
        ci -= nc;
    }
    return false;
}

// dlogits, one warp per token (Alg. 7 backward with the picks held fixed); lane l
// holds experts l + 32 i, i < NV. For the tensor-core router gradients it also writes
// dz16 [T, EP], dlogits rounded to bf16 with zero columns past E (EP = E rounded up to
// 64, 128 or 256), and (block 0) the token chunks of the chunked dW_r contraction:
// chunk_off[c] = first token of chunk c, the chunks of CH tokens of each party in
// order, then empty chunks up to nchunk.
template <int NV>
__global__ void __launch_bounds__(256) dlogits_kernel(
    const float* __restrict__ probs, const int32_t* __restrict__ topk_idx,
    const float* __restrict__ topk_w, const float* __restrict__ dtopk_w,
    const float* __restrict__ aux_coef, const int32_t* __restrict__ po, int P, int64_t Tn, int E,
    int k, int normalize, float* dlogits, __nv_bfloat16* dz16, int EP, int32_t* chunk_off, int CH,
    int nchunk) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (chunk_off && blockIdx.x == 0 && threadIdx.x == 0) {
        int c = 0;
        for (int q = 0; q < P; ++q) {
            const int64_t a = po ? po[q] : 0, b = po ? po[q + 1] : Tn;
            for (int64_t r = a; r < b && c < nchunk; r += CH) chunk_off[c++] = (int32_t)r;
        }
        for (; c <= nchunk; ++c) chunk_off[c] = (int32_t)Tn;
    }
    if (t >= Tn) return;
    const int party = party_of(po, P, t);
    float p[NV], dp[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = lane + 32 * i;
        p[i] = e < E ? probs[t * E + e] : 0.f;
        dp[i] = (aux_coef && e < E) ? aux_coef[party * E + e] : 0.f;
    }
    // lane j < k holds pick j
    const int ej = lane < k ? topk_idx[t * k + lane] : -1;
    const float gj0 = lane < k ? dtopk_w[t * k + lane] : 0.f;
    const float wj = lane < k ? topk_w[t * k + lane] : 0.f;
    float gj = gj0;
    if (normalize) {
        const float inner = warp_sum(gj0 * wj);
        const float S = warp_sum((ej >= 0 && ej < E) ? probs[t * E + ej] : 0.f);
        gj = (gj0 - inner) / S;
    }
    for (int j = 0; j < k; ++j) {
        const int e = __shfl_sync(0xffffffffu, ej, j);
        const float g = __shfl_sync(0xffffffffu, gj, j);
#pragma unroll
        for (int i = 0; i < NV; ++i)
            if (e == lane + 32 * i) dp[i] += g;
    }
    float loc = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) loc += dp[i] * p[i];
    const float dot = warp_sum(loc);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = lane + 32 * i;
        const float zz = p[i] * (dp[i] - dot);
        if (e < E) dlogits[t * E + e] = zz;
        if (dz16 && e < EP) dz16[t * EP + e] = __float2bfloat16_rn(e < E ? zz : 0.f);
    }
}

// dbias partial of one token chunk: part_db[c][e] = sum of dlogits[t][e] over the chunk.
// Thread (g, e) of a block, g < G = 2^j <= 1024 / E token groups, loads CDB_U tokens
// g, g + G, ... at once and adds them in order; the groups are then added by a fixed
// binary tree (deterministic).
constexpr int CDB_THREADS = 1024;
constexpr int CDB_U = 8;
__global__ void __launch_bounds__(CDB_THREADS) chunk_db_kernel(const float* __restrict__ dz,
                                                              const int32_t* __restrict__ chunk_off, int E,
                                                              float* part_db) {
    pdl_begin();
    __shared__ float s_part[CDB_THREADS];
    const int c = blockIdx.x, G = pow2_floor(CDB_THREADS / E);
    const int e = threadIdx.x % E, g = threadIdx.x / E;
    const int64_t a = chunk_off[c], b = chunk_off[c + 1];
    float acc = 0.f;
    if (g < G) {
        for (int64_t t = a + g; t < b; t += (int64_t)CDB_U * G) {
            float v[CDB_U];
#pragma unroll
            for (int u = 0; u < CDB_U; ++u) {
                const int64_t tt = t + (int64_t)u * G;
                v[u] = tt < b ? dz[tt * E + e] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < CDB_U; ++u) acc += v[u];
        }
    }
    s_part[threadIdx.x] = (g < G) ? acc : 0.f;
    __syncthreads();
    for (int h = G / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h * E) s_part[threadIdx.x] += s_part[threadIdx.x + h * E];
        __syncthreads();
    }
    if (threadIdx.x < E) part_db[(int64_t)c * E + threadIdx.x] = s_part[threadIdx.x];
}

// Partial dW_r = dlogits^T x and db over one chunk of RB_CH tokens of one party, for
// a tile of RB_ET experts and a column slab. The two thread halves take alternate
// tokens of the chunk and are added in a fixed order at the end.
constexpr int RB_CH = 32;   // tokens per chunk
constexpr int RB_ET = 8;    // experts per tile
constexpr int RB_HALF = 128;  // threads per half

template <typename T>
__global__ void __launch_bounds__(2 * RB_HALF) route_bwd_partial_kernel(
    const T* __restrict__ x, const float* __restrict__ dz, const int32_t* __restrict__ po, int P,
    int64_t Tn, int d, int E, float* part_dw, float* part_db) {
    pdl_begin();
    constexpr int VN = Vec<T>::N;
    constexpr int SLAB = RB_HALF * VN;
    __shared__ float s_dz[RB_CH][RB_ET];
    extern __shared__ float s_acc[];  // [RB_HALF][RB_ET][VN]: the second half's sums
    int party, n;
    int64_t t0;
    if (!chunk_of(blockIdx.x, po, P, Tn, RB_CH, &party, &t0, &n)) return;
    const int e0 = blockIdx.y * RB_ET;
    const int ne = min(RB_ET, E - e0);
    for (int i = threadIdx.x; i < RB_CH * RB_ET; i += blockDim.x) {
        const int tt = i / RB_ET, e = i % RB_ET;
        s_dz[tt][e] = (tt < n && e < ne) ? dz[(t0 + tt) * E + e0 + e] : 0.f;
    }
    __syncthreads();
    const int half = threadIdx.x / RB_HALF, ht = threadIdx.x % RB_HALF;
    if (blockIdx.z == 0 && threadIdx.x < ne) {
        float sdb = 0.f;
        for (int i = 0; i < n; ++i) sdb += s_dz[i][threadIdx.x];
        part_db[(int64_t)blockIdx.x * E + e0 + threadIdx.x] = sdb;
    }
    const int64_t c = (int64_t)blockIdx.z * SLAB + ht * VN;
    const bool active = c < d;
    float acc[RB_ET][VN];
#pragma unroll
    for (int e = 0; e < RB_ET; ++e)
#pragma unroll
        for (int q = 0; q < VN; ++q) acc[e][q] = 0.f;
    if (active) {
        // four tokens' x vectors are loaded before any of them is used
        for (int i0 = half; i0 < n; i0 += 8) {
            uint4 raw[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + 2 * u;
                if (i < n) raw[u] = Vec<T>::raw_load(x + (t0 + i) * d + c);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + 2 * u;
                if (i >= n) break;
                float xv[VN];
                unpack_vec<T>(raw[u], xv);
#pragma unroll
                for (int e = 0; e < RB_ET; ++e) {
                    const float zz = s_dz[i][e];
#pragma unroll
                    for (int q = 0; q < VN; ++q) acc[e][q] = fmaf(zz, xv[q], acc[e][q]);
                }
            }
        }
    }
    if (half == 1) {
#pragma unroll
        for (int e = 0; e < RB_ET; ++e)
#pragma unroll
            for (int q = 0; q < VN; ++q) s_acc[(ht * RB_ET + e) * VN + q] = acc[e][q];
    }
    __syncthreads();
    if (half == 0 && active) {
#pragma unroll
        for (int e = 0; e < RB_ET; ++e) {
            if (e < ne) {
                float* dst = part_dw + ((int64_t)blockIdx.x * E + e0 + e) * d + c;
                float r[VN];
#pragma unroll
                for (int q = 0; q < VN; ++q) r[q] = acc[e][q] + s_acc[(ht * RB_ET + e) * VN + q];
                Vec<float>::store(dst, r);
                if (VN == 8) Vec<float>::store(dst + 4, r + 4);
            }
        }
    }
}

// Sum the partials of each party's chunks: of eight partial sums per output, chunks g, g + 8,
// ... of the party join sum g in order, and the eight are added in order. A thread takes four
// consecutive outputs (d is a multiple of 4) and, SPLIT, one of their eight sums (added
// through shared memory), else all eight: for few outputs the split fills the SMs, for many
// it only costs blocks. HBM-bound; with 32 outputs per block and 4-byte loads it took 46 us for
// three parties of E = 63, d = 3072 (now 6.7) and 25 us for four of E = 32, d = 2048 (5.9).
constexpr int RR_GRP = 8, RR_THREADS = 256;
constexpr int64_t RR_SPLIT_BELOW = 150000;  // outputs: about four per thread of one full round

template <typename T, bool SPLIT>
__global__ void __launch_bounds__(RR_THREADS) route_bwd_reduce_kernel(
    const float* __restrict__ part_dw, const float* __restrict__ part_db,
    const int32_t* __restrict__ po, int P, int64_t Tn, int d, int E, int CH, T* dw_router,
    float* dbias) {
    pdl_begin();
    constexpr int OUT = SPLIT ? RR_THREADS / RR_GRP : RR_THREADS;  // threads with different outputs
    constexpr int SUMS = SPLIT ? 1 : RR_GRP;                       // partial sums of a thread
    __shared__ float4 s_sum[SPLIT ? RR_THREADS : 1];
    const int64_t per_party = (int64_t)E * d;
    const int g0 = SPLIT ? threadIdx.x / OUT : 0;
    const int64_t i = ((int64_t)blockIdx.x * OUT + threadIdx.x % OUT) * 4;
    const bool ok = i < (int64_t)P * per_party;
    auto crange = [&](int p, int64_t* first, int64_t* cnt) {
        int64_t base = 0;
        for (int q = 0; q < P; ++q) {
            int64_t a = po ? po[q] : 0, b = po ? po[q + 1] : Tn;
            int64_t nc = (b - a + CH - 1) / CH;
            if (q == p) { *first = base; *cnt = nc; return; }
            base += nc;
        }
    };
    float acc[SUMS][4];
#pragma unroll
    for (int g = 0; g < SUMS; ++g)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[g][q] = 0.f;
    if (ok) {
        const int p = (int)(i / per_party);
        int64_t first, cnt;
        crange(p, &first, &cnt);
        const float* src = part_dw + first * per_party + i % per_party;
#pragma unroll SPLIT ? 4 : 1
        for (int64_t c = g0; c < cnt; c += RR_GRP) {
#pragma unroll
            for (int g = 0; g < SUMS; ++g) {
                if (c + g < cnt) {
                    float v[4];
                    Vec<float>::load(src + (c + g) * per_party, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[g][q] += v[q];
                }
            }
        }
    }
    float tot[4] = {0.f, 0.f, 0.f, 0.f};
    if constexpr (SPLIT) {
        s_sum[threadIdx.x] = make_float4(acc[0][0], acc[0][1], acc[0][2], acc[0][3]);
        __syncthreads();
        if (g0 == 0) {
#pragma unroll
            for (int g = 0; g < RR_GRP; ++g) {
                const float4 v = s_sum[g * OUT + threadIdx.x];
                tot[0] += v.x; tot[1] += v.y; tot[2] += v.z; tot[3] += v.w;
            }
        }
    } else {
#pragma unroll
        for (int g = 0; g < RR_GRP; ++g)
#pragma unroll
            for (int q = 0; q < 4; ++q) tot[q] += acc[g < SUMS ? g : 0][q];
    }
    if (ok && g0 == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) Elem<T>::store(dw_router + i + q, tot[q]);
    }
    const int64_t j = (int64_t)blockIdx.x * RR_THREADS + threadIdx.x;
    if (dbias && j < (int64_t)P * E) {
        const int p = (int)(j / E), e = (int)(j % E);
        int64_t first, cnt;
        crange(p, &first, &cnt);
        float sum = 0.f;
        for (int64_t c = 0; c < cnt; ++c) sum += part_db[(first + c) * E + e];
        dbias[j] = sum;
    }
}

template <typename T>
static cudaError_t launch_route_bwd_reduce(const RouteBwdArgs& a, const float* part_dw, const float* part_db, int CH,
                                           cudaStream_t s) {
    const int64_t total = (int64_t)a.P * a.E * a.d;
    const bool split = total < RR_SPLIT_BELOW;
    // (every (party, expert) of dbias has a thread too: d >= 4 outputs each, four per thread)
    const int64_t per = split ? 4 * RR_THREADS / RR_GRP : 4 * RR_THREADS;
    const dim3 grid((unsigned)((total + per - 1) / per));
    if (split)
        (void)launch_pdl(route_bwd_reduce_kernel<T, true>, grid, dim3(RR_THREADS), 0, s, part_dw, part_db, a.po, a.P, a.T,
                         a.d, a.E, CH, (T*)a.dw_router, a.dbias);
    else
        (void)launch_pdl(route_bwd_reduce_kernel<T, false>, grid, dim3(RR_THREADS), 0, s, part_dw, part_db, a.po, a.P, a.T,
                         a.d, a.E, CH, (T*)a.dw_router, a.dbias);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------- launchers
// gating of logits in a.logits_in
static cudaError_t launch_gating(const RouteArgs& a, cudaStream_t s) {
    const int E = a.E;
    const size_t smem = a.P * E <= HIST_SMEM ? (size_t)a.P * E * sizeof(int) : 0;
    const int64_t groups_ub = a.T + a.P;  // upper bound with TPW = 1
    int blocks = (int)min64((groups_ub + 7) / 8, (int64_t)sm_count() * 8);
    if (blocks < 1) blocks = 1;
#define MOE_GATE(EM, TP)                                                                              \
    (void)launch_pdl(route_kernel<EM, TP>, dim3(blocks), dim3(256), smem, s, a.bias, a.logits_in, a.po, \
                     a.P, a.T, E, a.k, a.normalize, a.logits, a.probs, a.topk_idx, a.topk_w, a.counts)
    if (E <= 64) MOE_GATE(64, 4);
    else if (E <= 128) MOE_GATE(128, 2);
    else MOE_GATE(256, 1);
#undef MOE_GATE
    return cudaGetLastError();
}

template <int EP, int TB>
static cudaError_t launch_route_dot_t(const RouteArgs& a, int parts, cudaStream_t s) {
    auto kern = route_dot_kernel<EP, TB>;
    constexpr size_t smem =
        std::max<size_t>(2 * (size_t)(TB + EP) * RD_LD, (size_t)RD_THREADS * TB + (size_t)TB * EP) * sizeof(float);
    const cudaError_t e = allow_dynamic_smem<route_dot_kernel<EP, TB>>(smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(((a.T + TB - 1) / TB + (a.po ? a.P : 0)) * parts));
    cfg.blockDim = dim3(RD_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)parts;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, (const float*)a.x, (const float*)a.w_router, a.bias, a.po, a.P, a.T, a.d, a.E, a.k,
                              a.normalize, a.logits, a.probs, a.topk_idx, a.topk_w, a.counts);
}

// fp32, E <= 64. 16 tokens per CTA, 8 while those would not give every SM two CTAs (over 32 experts
// one: the weights of a CTA are staged for its tokens alone, so fewer tokens cost more
// shared-memory traffic). A cluster of 2, 4 or 8 CTAs per group while the groups leave more
// than half of the SMs idle and every CTA keeps a chunk of columns.
static cudaError_t launch_route_dot(const RouteArgs& a, cudaStream_t s) {
    if (a.T == 0) return cudaSuccess;
    const bool few = a.T < (a.E > 32 ? 1 : 2) * 16 * (int64_t)sm_count();
    const int64_t groups = (a.T + (few ? 8 : 16) - 1) / (few ? 8 : 16);
    const int chunks = (a.d + 127) / 128;
    int parts = 1;
    while (parts < 8 && groups * parts * 2 <= sm_count() && parts * 2 <= chunks) parts *= 2;
#define MOE_DOT(EP) (few ? launch_route_dot_t<EP, 8>(a, parts, s) : launch_route_dot_t<EP, 16>(a, parts, s))
    if (a.E <= 8) return MOE_DOT(8);
    if (a.E <= 16) return MOE_DOT(16);
    if (a.E <= 32) return MOE_DOT(32);
    return MOE_DOT(64);
#undef MOE_DOT
}

template <int EP, int TB>
static cudaError_t launch_route_chain_t(const RouteArgs& a, cudaStream_t s) {
    const unsigned grid = (unsigned)((a.T + TB - 1) / TB + (a.po ? a.P : 0));
    (void)launch_pdl(route_chain_kernel<EP, TB>, dim3(grid), dim3(RD_THREADS), 0, s, (const __nv_bfloat16*)a.x,
                     (const __nv_bfloat16*)a.w_router, a.bias, a.po, a.P, a.T, a.d, a.E, a.k, a.normalize, a.logits, a.probs,
                     a.topk_idx, a.topk_w, a.counts);
    return cudaGetLastError();
}

// bf16, E <= 64. Eight tokens a CTA (fewer read W_r more often), two up to four tokens per SM, where
// the latency of a CTA's steps decides (600 tokens of d = 3072, E = 63: 18.4 us with two, 21.7 with
// eight; 700: 24.7, 22.6; 100 of 2048, E = 13: 8.3, 10.3).
static cudaError_t launch_route_chain(const RouteArgs& a, cudaStream_t s) {
    const bool few = a.T <= 4 * (int64_t)sm_count();
#define MOE_CHAIN(EP) (few ? launch_route_chain_t<EP, 2>(a, s) : launch_route_chain_t<EP, 8>(a, s))
    if (a.E <= 8) return MOE_CHAIN(8);
    if (a.E <= 16) return MOE_CHAIN(16);
    if (a.E <= 32) return MOE_CHAIN(32);
    return MOE_CHAIN(64);
#undef MOE_CHAIN
}

// E > 64, fp32: the router's products x W_r[p]^T by the grouped fp32 GEMM into `logits` (groups =
// parties), then the gating pass reads them back, adds the bias and overwrites them with the
// biased logits.
static cudaError_t launch_route_wide_f32(const RouteArgs& a, cudaStream_t s) {
    GemmMArgs m{};
    m.G = (a.po && a.P > 1) ? a.P : 1;
    m.rows = (a.po && a.P > 1) ? GroupRows{a.po, (int)a.T, 0, 0, 0} : GroupRows{nullptr, (int)a.T, 0, 0, 0};
    m.a = a.x;
    m.b = a.w_router;
    m.b_group_elems = (int64_t)a.E * a.d;
    m.b_kmajor = true;
    m.N = a.E;
    m.K = a.d;
    m.epi = EPI_STORE;
    m.out0 = a.logits;
    cudaError_t e = launch_gemm_m_f32(m, s);
    if (e != cudaSuccess) return e;
    RouteArgs b = a;
    b.logits_in = a.logits;
    return launch_gating(b, s);
}

cudaError_t launch_route(const RouteArgs& a, bool bf16, bool from_logits, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(a.counts, 0, sizeof(int32_t) * a.P * a.E, s);
    if (e != cudaSuccess) return e;
    if (from_logits) {
        RouteArgs b = a;
        b.bias = nullptr;  // the caller's logits are final
        return launch_gating(b, s);
    }
    if (a.T == 0) return cudaSuccess;
    if (bf16 && (a.E % 4 == 0 || a.E > 64)) return launch_route_tc(a, s);
    if (a.E > 64) return launch_route_wide_f32(a, s);
    return bf16 ? launch_route_chain(a, s) : launch_route_dot(a, s);
}

cudaError_t launch_aux_loss(const float* probs, const int32_t* counts, const int32_t* po, int P,
                            int64_t T, int E, int k, float alpha, float* loss, float* coef,
                            cudaStream_t s) {
    (void)launch_pdl(aux_loss_kernel, dim3(P * AUX_CLUSTER), dim3(AUX_THREADS), 0, s, probs, counts, po, T, E, k, alpha, loss, coef);
    return cudaGetLastError();
}

// Workspace of the router backward. CUDA-core path (fp32): per-chunk partials of
// RB_CH tokens. Tensor-core path (bf16): per-chunk fp32 partials of dW_r and dbias, the
// chunk table and dz16 [T, 64] (dlogits in bf16, the A operand of dx_router = dz W_r and
// the B operand of dW_r^T = x^T dz).
static size_t align256(size_t n) { return (n + 255) / 256 * 256; }
struct RbTcLayout {
    int64_t C, nchunk;
    int EP;  // columns of dz16: E rounded up to 64, 128 or 256
    size_t dw, db, off, dz, total;
};
// Tokens per chunk of the chunked dW_r contraction: about 256 tiles of 128 model columns
// in all (one wave of 152 single-CTA tiles measured slower), at most 128 - P chunks
// (well inside the grouped GEMM's 256 groups), a multiple of 64.
static RbTcLayout rb_tc_layout(int64_t T, int P, int E, int d) {
    RbTcLayout L;
    const int64_t mt = std::max(1, d / 128);
    int64_t C = (T * mt + 255) / 256;
    C = std::max<int64_t>(C, (T + (128 - P) - 1) / (128 - P));
    C = std::max<int64_t>(C, 64);
    L.C = (C + 63) / 64 * 64;
    L.nchunk = (T + L.C - 1) / L.C + P;
    L.dw = 0;
    L.db = align256((size_t)L.nchunk * E * d * sizeof(float));
    L.off = align256(L.db + (size_t)L.nchunk * E * sizeof(float));
    L.EP = E <= 64 ? 64 : E <= 128 ? 128 : 256;
    L.dz = align256(L.off + (size_t)(L.nchunk + 1) * sizeof(int32_t));
    L.total = L.dz + (size_t)T * L.EP * 2 + 256;
    return L;
}

size_t route_bwd_workspace(int64_t T, int P, int E, int d) {
    const int64_t nch = (T + RB_CH - 1) / RB_CH + P;
    const size_t simt = (size_t)nch * E * d * sizeof(float) + (size_t)nch * E * sizeof(float) + 256;
    return std::max(simt, rb_tc_layout(T, P, E, d).total);
}

static cudaError_t launch_dlogits(const RouteBwdArgs& a, __nv_bfloat16* dz16, int EP, int32_t* chunk_off,
                                  int CH, int nchunk, cudaStream_t s) {
    const unsigned blocks = (unsigned)((a.T + 7) / 8);
#define MOE_DL(NV)                                                                                 \
    (void)launch_pdl(dlogits_kernel<NV>, dim3(blocks), dim3(256), 0, s, a.probs, a.topk_idx, a.topk_w, \
                     a.dtopk_w, a.aux_coef, a.po, a.P, a.T, a.E, a.k, a.normalize, a.dlogits, dz16, EP, \
                     chunk_off, CH, nchunk)
    if (a.E <= 64) MOE_DL(2);
    else if (a.E <= 128) MOE_DL(4);
    else MOE_DL(8);
#undef MOE_DL
    return cudaGetLastError();
}

// fp32: dlogits, CUDA-core partials and reduce, dx_router on the fp32 GEMM
static cudaError_t launch_route_bwd_simt(const RouteBwdArgs& a, void* ws, cudaStream_t s) {
    using T = float;
    const int64_t nch = (a.T + RB_CH - 1) / RB_CH + a.P;
    float* part_dw = (float*)ws;
    float* part_db = part_dw + nch * a.E * a.d;
    if (a.T > 0) {
        cudaError_t e = launch_dlogits(a, (__nv_bfloat16*)nullptr, 0, (int32_t*)nullptr, 0, 0, s);
        if (e != cudaSuccess) return e;
    }
    constexpr int SLAB = RB_HALF * Vec<T>::N;
    dim3 grid((unsigned)nch, (a.E + RB_ET - 1) / RB_ET, (a.d + SLAB - 1) / SLAB);
    const size_t smem = (size_t)RB_HALF * RB_ET * Vec<T>::N * sizeof(float);
    cudaError_t e = allow_dynamic_smem<route_bwd_partial_kernel<T>>(smem);
    if (e != cudaSuccess) return e;
    (void)launch_pdl(route_bwd_partial_kernel<T>, dim3(grid), dim3(2 * RB_HALF), smem, s, (const T*)a.x,
                     a.dlogits, a.po, a.P, a.T, a.d, a.E, part_dw, part_db);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_route_bwd_reduce<T>(a, part_dw, part_db, RB_CH, s)) != cudaSuccess) return e;
    if (a.dx_router && a.T > 0) {  // dx_router[t] = dlogits[t] W_r[p(t)], K = E
        GemmMArgs m{};
        m.G = a.po ? a.P : 1;
        m.rows = GroupRows{a.po, (int)a.T, 0, 0, 0};
        m.a = a.dlogits;
        m.b = a.w_router;
        m.b_group_elems = (int64_t)a.E * a.d;
        m.b_kmajor = false;
        m.N = a.d;
        m.K = a.E;
        m.epi = EPI_STORE;
        m.out0 = a.dx_router;
        return launch_gemm_m_f32(m, s);
    }
    return cudaSuccess;
}

// bf16: both products on the tensor cores.
//   dW_r[p]^T = sum over the chunks c of party p of x_c^T dz_c (K-variable grouped GEMM,
//               one group per chunk, fp32 partials), reduced over chunks in order;
//   dx_router = dz W_r[p(t)] (M-variable grouped GEMM over parties, K = 64 padded).
// dz is rounded to bf16 for both (the operands of every bf16 contraction are bf16).
static cudaError_t launch_route_bwd_tc(const RouteBwdArgs& a, void* ws, cudaStream_t s) {
    const RbTcLayout Lw = rb_tc_layout(a.T, a.P, a.E, a.d);
    uint8_t* base = (uint8_t*)ws;
    float* part_dw = (float*)(base + Lw.dw);
    float* part_db = (float*)(base + Lw.db);
    int32_t* chunk_off = (int32_t*)(base + Lw.off);
    __nv_bfloat16* dz16 = (__nv_bfloat16*)(base + Lw.dz);
    cudaError_t e;
    if (a.T > 0) {
        if ((e = launch_dlogits(a, dz16, Lw.EP, chunk_off, (int)Lw.C, (int)Lw.nchunk, s)) != cudaSuccess)
            return e;
        (void)launch_pdl(chunk_db_kernel, dim3((unsigned)Lw.nchunk), dim3(CDB_THREADS), 0, s,
                         (const float*)a.dlogits, (const int32_t*)chunk_off, a.E, part_db);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        GemmKArgs g{};
        g.G = (int)Lw.nchunk;
        g.rows = GroupRows{chunk_off, (int)a.T, 0, 0, 0};
        g.a = a.x;
        g.b = dz16;
        g.M = a.d;
        g.N = Lw.EP;
        g.out = part_dw;
        g.epi = EPI_DWR;
        g.E = a.E;
        if ((e = launch_gemm_k(g, true, s)) != cudaSuccess) return e;
    }
    if ((e = launch_route_bwd_reduce<__nv_bfloat16>(a, part_dw, part_db, (int)Lw.C, s)) != cudaSuccess) return e;
    if (a.dx_router && a.T > 0) {
        GemmMArgs m{};
        m.G = a.po ? a.P : 1;
        m.rows = GroupRows{a.po, (int)a.T, 0, 0, 0};
        m.a = dz16;
        m.b = a.w_router;
        m.b_group_elems = (int64_t)a.E * a.d;
        m.b_kmajor = false;
        m.N = a.d;
        m.K = Lw.EP;
        m.b_rows = a.E;
        m.epi = EPI_STORE;
        m.out0 = a.dx_router;
        m.slim = true;  // one k-block per tile: the stores bound it
        return launch_gemm_m(m, true, s);
    }
    return cudaSuccess;
}

cudaError_t launch_route_bwd(const RouteBwdArgs& a, bool bf16, void* ws, cudaStream_t s) {
    return bf16 ? launch_route_bwd_tc(a, ws, s) : launch_route_bwd_simt(a, ws, s);
}

cudaError_t route_status(cudaStream_t s, int* code) { return tu_status_read_clear(s, code); }

}  // namespace moe

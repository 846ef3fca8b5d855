// route.cu -- K1: router GEMV + softmax + top-k gating, then the per-task
// capacity scan (Section 2.1 routing, Challenge #1 capacity limits,
// Section 3.3.1 sequential assignment).
//
// Kernel 1 (route_topk), bf16 tokens: route_mma_kernel below (or, with
// VMOE_ROUTE_TC=1, route_tc_kernel in route_tc.cu on tcgen05) -- the router
// product on the tensor cores (mma.sync) with the fp32 weights split into
// three bf16 parts.  fp32 tokens: route_f32_kernel on the CUDA cores; given
// logits: route_given_kernel.  One CTA per (task, tile of tokens); the logits
// tile goes through shared memory, and one thread per token takes the max, the
// softmax denominator and the k largest logits (ties to the lower expert
// index).
//
// Kernel 2 (capacity_scan): one CTA per task.  The choice-major assignment
// sequence p = j*N + n is cut into one contiguous chunk per warp; each warp
// ranks its chunk 32 assignments at a time with __match_any_sync, keeping
// per-warp expert counters in shared memory; a per-expert exclusive scan over
// the warps then gives the global rank, which becomes the slot (or -1 once it
// reaches C).  No atomics, so the result is deterministic.
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "topk.cuh"

namespace cg = cooperative_groups;

namespace vmoe {
namespace {

constexpr int RT_THREADS = 256;

// Softmax + top-k of `ntok` logit rows held in shared memory (row pitch ldl,
// odd, so the per-thread rows hit distinct banks), one thread per row.
__device__ __forceinline__ void topk_rows(const Dims &p, const float *lg, int ldl, int ntok, int t,
                                          int n0, int32_t *__restrict__ out_idx,
                                          float *__restrict__ out_gate, int nthreads) {
    for (int r = threadIdx.x; r < ntok; r += nthreads)
        topk_row(p, lg + r * ldl, (long long)t * p.N + n0 + r, out_idx, out_gate);
}

// Given logits (VMOE_LOGITS_IN): the rows of RT_TOK tokens through shared memory.
constexpr int RT_TOK = 64;
__global__ void __launch_bounds__(RT_THREADS)
route_given_kernel(Dims p, const float *__restrict__ logits, int32_t *__restrict__ out_idx,
                   float *__restrict__ out_gate) {
    pdl_wait();
    extern __shared__ __align__(16) float smem[];  // [RT_TOK][E + 1]
    const int t = blockIdx.y, n0 = blockIdx.x * RT_TOK, E = p.E;
    const int ntok = min(RT_TOK, p.N - n0);
    for (int i = threadIdx.x; i < ntok * E; i += RT_THREADS) {
        const int r = i / E, e = i - r * E;
        smem[r * (E + 1) + e] = logits[((long long)t * p.N + n0 + r) * E + e];
    }
    __syncthreads();
    topk_rows(p, smem, E + 1, ntok, t, n0, out_idx, out_gate, RT_THREADS);
}

// CUDA-core router for fp32 tokens: TOK tokens x ECH experts a pass, 4 x 4 logits a
// thread.  d is swept in chunks of KC staged in shared memory (the next chunk's
// loads in registers meanwhile); SLICES groups of threads take a slice of every
// chunk each, and their partial logits are summed in slice order.
// Two forms.  Few tokens (a layer's few hundred are a few dozen CTAs) are bound by
// the chain of chunks: 16 tokens a CTA, chunks of 128, 4 or 8 slices.  Many tokens
// are bound by arithmetic, by the weights each CTA stages and by its top-k threads:
// 64 tokens, chunks of 32, one slice (launch_route has the rule).
template <int ECH, int TOK, int KC, int SLICES_>
struct RouteF32 {
    static constexpr int SLICES = SLICES_;
    static constexpr int XP = KC + 4;                // x row pitch (floats)
    static constexpr int EG = ECH / 4;               // threads along experts
    static constexpr int NT = EG * (TOK / 4) * SLICES;  // threads
    static constexpr int CTAS = SLICES > 1 ? 2 : NT == 128 ? 7 : 4;  // an SM
    static constexpr int KS = KC / SLICES;           // d per slice and chunk
    static constexpr int XV = TOK * KC / 4 / NT;     // x vectors per thread
    static constexpr int WV = KC * ECH / NT;         // weights per thread
    static constexpr int PARTS = SLICES > 1 ? SLICES * TOK * ECH : 0;
    static constexpr size_t smem(int E) {
        return sizeof(float) * ((size_t)TOK * XP + (size_t)KC * ECH + PARTS + (size_t)TOK * (E + 1));
    }
    static_assert(KS % 4 == 0, "a slice is swept four values of d at a time");
    static_assert(XV * NT * 4 == TOK * KC && WV * NT == KC * ECH, "every thread stages as much");
};

template <int ECH, int TOK, int KC, int SLICES>
__global__ void __launch_bounds__(RouteF32<ECH, TOK, KC, SLICES>::NT, RouteF32<ECH, TOK, KC, SLICES>::CTAS)
route_f32_kernel(Dims p, const float *__restrict__ x, const float *__restrict__ wr,
                 const float *__restrict__ bias, float *__restrict__ logits,
                 int32_t *__restrict__ out_idx, float *__restrict__ out_gate) {
    using S = RouteF32<ECH, TOK, KC, SLICES>;
    constexpr int NT = S::NT, UNROLL = SLICES == 1 ? 1 : 2;
    pdl_wait();
    extern __shared__ __align__(16) float smem[];
    float *xs = smem;               // [TOK][S::XP]
    float *ws = xs + TOK * S::XP;   // [KC][ECH]
    float *part = ws + KC * ECH;    // [SLICES][TOK][ECH], with more than one slice
    float *lg = part + S::PARTS;    // [TOK][E + 1]
    const int t = blockIdx.y, n0 = blockIdx.x * TOK;
    const int E = p.E, d = p.d, N = p.N, ldl = E + 1, tid = threadIdx.x;
    const int ntok = min(TOK, N - n0);
    const int eg = tid % S::EG, tg = tid / S::EG % (TOK / 4), sl = tid / (S::EG * (TOK / 4));
    const float *xt = x + ((long long)t * N + n0) * d;
    const float *wt = wr + (long long)t * d * E;
    float4 xv[S::XV];
    float wv[S::WV];
    for (int e0 = 0; e0 < E; e0 += ECH) {
        auto load = [&](int k0) {
#pragma unroll
            for (int q = 0; q < S::XV; ++q) {  // d % 8 == 0: a vector is inside its row or past it
                const int i = tid + q * NT, r = i / (KC / 4), c = i % (KC / 4) * 4;
                xv[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (r < ntok && k0 + c < d)
                    xv[q] = __ldg(reinterpret_cast<const float4 *>(xt + (long long)r * d + k0 + c));
            }
#pragma unroll
            for (int q = 0; q < S::WV; ++q) {
                const int i = tid + q * NT, r = i / ECH, c = i % ECH;
                wv[q] = k0 + r < d && e0 + c < E ? __ldg(wt + (long long)(k0 + r) * E + e0 + c) : 0.0f;
            }
        };
        float acc[4][4] = {};
        load(0);
        for (int k0 = 0; k0 < d; k0 += KC) {
            __syncthreads();  // the previous chunk has been read
#pragma unroll
            for (int q = 0; q < S::XV; ++q) {
                const int i = tid + q * NT;
                *reinterpret_cast<float4 *>(xs + i / (KC / 4) * S::XP + i % (KC / 4) * 4) = xv[q];
            }
#pragma unroll
            for (int q = 0; q < S::WV; ++q) ws[tid + q * NT] = wv[q];
            __syncthreads();
            if (k0 + KC < d) load(k0 + KC);
#pragma unroll UNROLL
            for (int kk = sl * S::KS; kk < (sl + 1) * S::KS; kk += 4) {
                float4 a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[i] = *reinterpret_cast<const float4 *>(xs + (4 * tg + i) * S::XP + kk);
                    b[i] = *reinterpret_cast<const float4 *>(ws + (kk + i) * ECH + 4 * eg);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float av[4] = {a[i].x, a[i].y, a[i].z, a[i].w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        acc[i][0] = fmaf(av[q], b[q].x, acc[i][0]);
                        acc[i][1] = fmaf(av[q], b[q].y, acc[i][1]);
                        acc[i][2] = fmaf(av[q], b[q].z, acc[i][2]);
                        acc[i][3] = fmaf(av[q], b[q].w, acc[i][3]);
                    }
                }
            }
        }
        if (SLICES == 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = 4 * tg + i, e = e0 + 4 * eg + q;
                    if (r < ntok && e < E) lg[r * ldl + e] = acc[i][q] + (bias ? bias[(long long)t * E + e] : 0.0f);
                }
            continue;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(part + (sl * TOK + 4 * tg + i) * ECH + 4 * eg) =
                make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        __syncthreads();
        for (int i = tid; i < TOK * ECH; i += NT) {
            const int r = i / ECH, e = e0 + i % ECH;
            if (r >= ntok || e >= E) continue;
            float v = part[i];
#pragma unroll
            for (int q = 1; q < SLICES; ++q) v += part[q * TOK * ECH + i];
            if (bias) v += bias[(long long)t * E + e];
            lg[r * ldl + e] = v;
            logits[((long long)t * N + n0 + r) * E + e] = v;
        }
    }
    __syncthreads();
    if (SLICES == 1)
        for (int i = tid; i < ntok * E; i += NT)
            logits[((long long)t * N + n0) * E + i] = lg[i / E * ldl + i % E];
    topk_rows(p, lg, ldl, ntok, t, n0, out_idx, out_gate, NT);
}

// Tensor-core router for bf16 tokens.  x is exactly representable in bf16, so
// x * W_r is formed as x * W_hi + x * W_mid + x * W_lo with the fp32 router
// weights split into three bf16 parts (W_hi = bf16(W), W_mid = bf16(W - W_hi),
// W_lo = bf16(W - W_hi - W_mid), together about 24 significant bits): every
// partial product is exact in fp32 and the mma.sync m16n8k16 instructions
// accumulate in fp32, so the logits keep fp32 accuracy at a small fraction of
// the CUDA-core instruction count.  One CTA = 4 groups of 16 tokens of one task;
// d is swept in chunks of RM_KC staged in shared memory.  The weight split is
// done while staging, two values per conversion, into [part][expert][k]
// tiles, so that one ldmatrix.x4 gives the B fragments of two 8-expert blocks
// (and one gives a warp's A fragment).
constexpr int RM_KC = 128;        // d per staged chunk
constexpr int RM_XP = RM_KC + 8;  // row pitch (bf16) of the x and weight tiles: conflict-free ldmatrix

__device__ __forceinline__ void rm_ldsm_x4(uint32_t (&r)[4], const void *smem) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

// NB blocks of 8 experts per pass (NB even); 4 groups of 16 tokens and KS slices
// of each chunk's k steps: 4 KS warps.  KS = 2 for more than 32 experts, whose
// weights take 128 threads twice as long to stage (8 tasks of 1576 tokens, d 1024,
// 64 experts: 49.5 -> 42 us; 17 tasks, d 768, 32 experts: 31.8 -> 43.4, so not there).
//
// `split`: that many CTAs (a cluster) share a token tile, each with a range of
// the chunks; their partial logits are summed through distributed shared memory
// in rank order and each finishes a share of the tokens.  A chunk is a chain of
// a load from DRAM, the split of the weights and the MMAs, 2 us long; few
// tokens leave nothing else to run behind it.  Measured on GB300: 4 tasks of 197
// tokens, d 768, 32 experts 20.5 -> 16.4 us; 2 of 300, d 1024, 64 experts (with
// KS = 2) 40.7 -> 12.4 us.
template <int NB, int KS>
struct RouteMma {
    static constexpr int TG = 4, TOK = 16 * TG, NT = 32 * TG * KS, NP = 8 * NB;
    static constexpr int PARTS = (KS - 1) * TOK * NP;  // floats, over the tiles after the last chunk
    static constexpr size_t TILES = (size_t)TOK * RM_XP * 2 + (size_t)3 * NP * RM_XP * 2;
    static constexpr size_t smem(int E) { return TILES + (size_t)TOK * (E + 1) * 4; }
    static_assert((size_t)(PARTS + TOK * NP) * 4 <= TILES, "partial sums reuse the tiles");
};

template <int NB, int KS, bool SPLIT>
__global__ void __launch_bounds__(RouteMma<NB, KS>::NT, KS == 1 ? 3 : 2)
route_mma_kernel(Dims p, int nsplit, const __nv_bfloat16 *__restrict__ x, const float *__restrict__ wr,
                 const float *__restrict__ bias, float *__restrict__ logits,
                 int32_t *__restrict__ out_idx, float *__restrict__ out_gate) {
    static_assert(NB % 2 == 0, "B fragments are loaded two expert blocks at a time");
    using S = RouteMma<NB, KS>;
    constexpr int NP = S::NP, NT = S::NT, TOK = S::TOK, TG = S::TG;
    pdl_wait();
    extern __shared__ __align__(16) uint8_t rm_smem[];
    __nv_bfloat16 *xs = reinterpret_cast<__nv_bfloat16 *>(rm_smem);  // [TOK][RM_XP]
    __nv_bfloat16 *ws = xs + TOK * RM_XP;                            // [3][NP][RM_XP]
    float *part = reinterpret_cast<float *>(rm_smem);                // [KS - 1][TOK][NP]
    float *red = part + S::PARTS;                                    // [TOK][NP]: this CTA's sums (split > 1)
    const int split = SPLIT ? nsplit : 1, rank = SPLIT ? (int)(blockIdx.x % split) : 0;
    const int t = blockIdx.y, n0 = (int)(SPLIT ? blockIdx.x / split : blockIdx.x) * TOK;
    const int E = p.E, d = p.d, N = p.N;
    const int ldl = E + 1;
    float *lg = reinterpret_cast<float *>(rm_smem + S::TILES);  // [TOK][E+1]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tg = warp % TG, sl = warp / TG;
    const int g = lane >> 2, tq = lane & 3;
    const int ntok = min(TOK, N - n0);
    const __nv_bfloat16 *xt = x + ((long long)t * N + n0) * d;
    const float *wt = wr + (long long)t * d * E;
    // Per thread and chunk: XV x vectors (16 B each) and WI weight items, an
    // item being 8 consecutive k of one expert.  The next chunk's values are
    // loaded into registers before the current chunk's MMAs run, so global
    // latency overlaps the tensor-core work.
    constexpr int XV = TOK * (RM_KC / 8) / NT;
    constexpr int WI = (RM_KC / 8) * NP / NT;
    static_assert(XV >= 1 && WI >= 1, "every thread stages a vector of each tile");
    uint4 xv[XV];
    float wv[WI][8];
    auto load_chunk = [&](int e0, int k0) {
#pragma unroll
        for (int q = 0; q < XV; ++q) {
            const int i = tid + q * NT;
            const int r = i / (RM_KC / 8), c = (i % (RM_KC / 8)) * 8;
            xv[q] = make_uint4(0, 0, 0, 0);
            if (r < ntok && k0 + c < d)
                xv[q] = __ldg(reinterpret_cast<const uint4 *>(xt + (long long)r * d + k0 + c));
        }
#pragma unroll
        for (int q = 0; q < WI; ++q) {  // consecutive threads: consecutive experts (coalesced)
            const int i = tid + q * NT;
            const int n = i % NP, e = e0 + n, kk = k0 + (i / NP) * 8;
#pragma unroll
            for (int r = 0; r < 8; ++r)
                wv[q][r] = (e < E && kk + r < d) ? __ldg(wt + (long long)(kk + r) * E + e) : 0.0f;
        }
    };
    auto stage_chunk = [&]() {
#pragma unroll
        for (int q = 0; q < XV; ++q) {
            const int i = tid + q * NT;
            const int r = i / (RM_KC / 8), c = (i % (RM_KC / 8)) * 8;
            *reinterpret_cast<uint4 *>(xs + r * RM_XP + c) = xv[q];
        }
#pragma unroll
        for (int q = 0; q < WI; ++q) {
            const int i = tid + q * NT;
            const int n = i % NP, c = (i / NP) * 8;
            uint32_t hi[4], mid[4], lo[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // split3 of a k pair, both values per conversion
                const __nv_bfloat162 h = __floats2bfloat162_rn(wv[q][2 * j], wv[q][2 * j + 1]);
                const float2 hf = __bfloat1622float2(h);
                const float r0 = wv[q][2 * j] - hf.x, r1 = wv[q][2 * j + 1] - hf.y;
                const __nv_bfloat162 m = __floats2bfloat162_rn(r0, r1);
                const float2 mf = __bfloat1622float2(m);
                const __nv_bfloat162 l = __floats2bfloat162_rn(r0 - mf.x, r1 - mf.y);
                hi[j] = *reinterpret_cast<const uint32_t *>(&h);
                mid[j] = *reinterpret_cast<const uint32_t *>(&m);
                lo[j] = *reinterpret_cast<const uint32_t *>(&l);
            }
            *reinterpret_cast<uint4 *>(ws + (0 * NP + n) * RM_XP + c) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(ws + (1 * NP + n) * RM_XP + c) = make_uint4(mid[0], mid[1], mid[2], mid[3]);
            *reinterpret_cast<uint4 *>(ws + (2 * NP + n) * RM_XP + c) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    };
    // ldmatrix row addresses: A, rows tg*16 + (lane & 15), k offset 8 (lane >> 4);
    // B, expert (lane & 7) + 8 (lane >> 4) of a block pair, k offset 8 ((lane >> 3) & 1)
    const __nv_bfloat16 *xa = xs + (tg * 16 + (lane & 15)) * RM_XP + (lane >> 4) * 8;
    const __nv_bfloat16 *wb = ws + ((lane & 7) + (lane >> 4) * 8) * RM_XP + ((lane >> 3) & 1) * 8;
    const int chunks = (d + RM_KC - 1) / RM_KC;
    const int k_beg = SPLIT ? chunks * rank / split * RM_KC : 0;
    const int k_end = SPLIT ? min(d, chunks * (rank + 1) / split * RM_KC) : d;
    for (int e0 = 0; e0 < E; e0 += NP) {
        float acc[NB][4];
#pragma unroll
        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[nb][i] = 0.0f;
        load_chunk(e0, k_beg);  // a rank has at least one chunk
        for (int k0 = k_beg; k0 < k_end; k0 += RM_KC) {
            __syncthreads();  // the previous chunk's fragments (or the last pass's parts) have been read
            stage_chunk();
            __syncthreads();
            if (k0 + RM_KC < k_end) load_chunk(e0, k0 + RM_KC);
#pragma unroll
            for (int kq = 0; kq < RM_KC / 16 / KS; ++kq) {
                const int ks = (sl * (RM_KC / 16 / KS) + kq) * 16;
                uint32_t a[4];
                rm_ldsm_x4(a, xa + ks);
#pragma unroll
                for (int np = 0; np < NB / 2; ++np) {
                    uint32_t b[3][4];  // [part][b0, b1 of block 2np; b0, b1 of block 2np+1]
#pragma unroll
                    for (int sp = 0; sp < 3; ++sp) rm_ldsm_x4(b[sp], wb + (sp * NP + np * 16) * RM_XP + ks);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int sp = 2; sp >= 0; --sp)  // smallest part first
                            mma_bf16_16816(acc[2 * np + h], a[0], a[1], a[2], a[3], b[sp][2 * h], b[sp][2 * h + 1]);
                }
            }
        }
        // the slices' partial sums, in slice order
        if (KS > 1 || SPLIT) __syncthreads();
        if (KS > 1) {
            if (sl > 0) {
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int i = 0; i < 4; i += 2)
                        *reinterpret_cast<float2 *>(part + ((sl - 1) * TOK + tg * 16 + g + (i >> 1) * 8) * NP + nb * 8 +
                                                    2 * tq) = make_float2(acc[nb][i], acc[nb][i + 1]);
            }
            __syncthreads();
        }
        if (sl == 0) {
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = tg * 16 + g + (i >> 1) * 8;
                    const int n = nb * 8 + 2 * tq + (i & 1), e = e0 + n;
                    float v = acc[nb][i];
#pragma unroll
                    for (int q = 1; q < KS; ++q) v += part[((q - 1) * TOK + r) * NP + n];
                    if (SPLIT)
                        red[r * NP + n] = v;
                    else if (r < ntok && e < E)
                        lg[r * ldl + e] = v + (bias ? bias[(long long)t * E + e] : 0.0f);
                }
        }
        if (SPLIT) {  // this rank's tokens: rank, rank + split, ...
            cg::cluster_group cluster = cg::this_cluster();
            cluster.sync();
            const int mine = (ntok - rank + split - 1) / split;
            for (int i = tid; i < mine * NP; i += NT) {
                const int r = rank + i / NP * split, n = i % NP, e = e0 + n;
                if (e >= E) continue;
                float v = 0.0f;
                for (int q = 0; q < split; ++q) v += cluster.map_shared_rank(red, q)[r * NP + n];
                lg[r * ldl + e] = v + (bias ? bias[(long long)t * E + e] : 0.0f);
            }
            cluster.sync();  // the sums stay until every rank has read them
        }
    }
    __syncthreads();
    if (SPLIT) {
        const int mine = (ntok - rank + split - 1) / split;
        for (int i = tid; i < mine * E; i += NT) {
            const int r = rank + i / E * split, e = i % E;
            logits[((long long)t * N + n0 + r) * E + e] = lg[r * ldl + e];
        }
        // a warp takes a row in about 1000 cycles, a thread in about 60 E, all rows at once
        if ((mine + NT / 32 - 1) / (NT / 32) * 16 <= E) {
            for (int r = rank + warp * split; r < ntok; r += NT / 32 * split)
                topk_row_warp(p, lg + r * ldl, (long long)t * N + n0 + r, out_idx, out_gate);
        } else {
            for (int i = tid; i < mine; i += NT) {
                const int r = rank + i * split;
                topk_row(p, lg + r * ldl, (long long)t * N + n0 + r, out_idx, out_gate);
            }
        }
        return;
    }
    for (int i = tid; i < ntok * E; i += NT) {
        const int r = i / E, e = i - r * E;
        logits[((long long)t * N + n0 + r) * E + e] = lg[r * ldl + e];
    }
    topk_rows(p, lg, ldl, ntok, t, n0, out_idx, out_gate, NT);
}

template <int NB, int KS>
int launch_mma_router(const Dims &p, const __nv_bfloat16 *x, const float *wr, const float *bias,
                      float *logits, int32_t *idx, float *gate, cudaStream_t s) {
    using S = RouteMma<NB, KS>;
    const size_t smem = S::smem(p.E);
    if (smem > 227 * 1024) return VMOE_ERR_UNSUPPORTED;
    // as many CTAs a tile as its chunks allow, while every SM has at most one; three
    // or fewer do not pay for the cluster (1 task of 197 tokens, d 384: 12.2 -> 13.1
    // us; 3 of 971, d 640: 17.0 -> 18.6)
    const long long tiles = (long long)((p.N + S::TOK - 1) / S::TOK) * p.T;
    int split = (p.d + RM_KC - 1) / RM_KC;
    if (split > 8) split = 8;
    while (split > 1 && tiles * split > num_sms()) --split;
    if (split < 4) split = 1;
    auto kern = split > 1 ? route_mma_kernel<NB, KS, true> : route_mma_kernel<NB, KS, false>;
    static std::atomic<int> smem_limit[2][64];  // the size depends on E
    if (const int st = raise_smem_limit((const void *)kern, smem_limit[split > 1], (int)smem)) return st;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((p.N + S::TOK - 1) / S::TOK * split), p.T);
    cfg.blockDim = dim3(S::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (split > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = split;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    trace_before(s, "route_topk");
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p, split, x, wr, bias, logits, idx, gate);
    trace_after(s);
    return e == cudaSuccess ? VMOE_OK : VMOE_ERR_CUDA;
}

// SMEM_IDX: the task's idx array and the temporary ranks live in shared memory
// (read with coalesced accesses); otherwise the ranks stay in `slot`.
// CS_THREADS: 1024 (32 warps, 4 rounds of 32 assignments per warp at N k = 3152)
// while the per-warp expert counters stay small (E <= 128), else 256.
// One CTA a task, so it is a chain of latencies: positions advance by addition
// instead of a division each, the counters of an expert are scanned by a warp, and
// a warp turns its own ranks into slots (us: ViT-S, 4 tasks of 1576 tokens, top-2
// 10.2 -> 7.9; 6 of 3152 14.3 -> 13.4; 17 of 1576, where its loads wait for DRAM,
// 10.6 either way).
// The counters' pitch is odd: a warp scans one expert's column.
__host__ __device__ constexpr int cs_pitch(int E) { return E | 1; }
template <bool SMEM_IDX, int CS_THREADS>
__global__ void __launch_bounds__(CS_THREADS)
capacity_scan_kernel(Dims p, const int32_t *__restrict__ idx, int32_t *__restrict__ slot,
                     int32_t *__restrict__ load) {
    constexpr int CS_WARPS = CS_THREADS / 32;
    pdl_wait();
    extern __shared__ int cs_smem[];
    const int t = blockIdx.x;
    const int E = p.E, N = p.N, k = p.k, C = p.C;
    const int ldc = cs_pitch(E);
    int *cnt = cs_smem;  // [CS_WARPS][ldc]
    const int total = k * N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long tb = (long long)t * N * k;
    int *sidx = cs_smem + CS_WARPS * ldc;  // [N*k] in token-major (memory) order
    int *srank = sidx + total;           // [N*k]
    if (SMEM_IDX) {
        constexpr int U = 4;  // loads in flight a thread
        for (int i0 = threadIdx.x; i0 < total; i0 += U * CS_THREADS) {
            int v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * CS_THREADS < total) v[u] = __ldg(idx + tb + i0 + u * CS_THREADS);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (i0 + u * CS_THREADS < total) sidx[i0 + u * CS_THREADS] = v[u];
        }
    }
    for (int i = threadIdx.x; i < CS_WARPS * ldc; i += CS_THREADS) cnt[i] = 0;
    __syncthreads();
    const int32_t *src = SMEM_IDX ? sidx : idx + tb;
    int32_t *rank = SMEM_IDX ? srank : slot + tb;

    const int per = ((total + CS_WARPS - 1) / CS_WARPS + 31) & ~31;
    const int beg = min(total, warp * per), end = min(total, beg + per);
    int *my = cnt + warp * ldc;
    const unsigned lt = (1u << lane) - 1u;
    // the lane's first position beg + lane of the choice-major sequence p = j*N + n
    const int j_beg = (beg + lane) / N, n_beg = (beg + lane) - j_beg * N;
    auto advance = [&](int &n, int &j) {  // 32 positions on
        n += 32;
        while (n >= N) {
            n -= N;
            ++j;
        }
    };
    // Pass 1: rank within the warp's chunk.
    int n = n_beg, j = j_beg;
    for (int p0 = beg; p0 < end; p0 += 32) {
        const bool valid = p0 + lane < end;
        const int e = valid ? src[n * k + j] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, e);
        const int before = __popc(peers & lt);
        const int base = valid ? my[e] : 0;
        if (valid) rank[n * k + j] = base + before;
        __syncwarp();  // every lane has read its counter
        if (valid && before == 0) my[e] = base + __popc(peers);
        __syncwarp();
        if (p0 + 32 < end) advance(n, j);
    }
    __syncthreads();
    // Exclusive scan over warps, per expert: a warp an expert, lane w its counter of
    // warp w; with 8 warps a thread an expert.
    if (CS_WARPS == 32) {
        for (int e = warp; e < E; e += CS_WARPS) {
            const int c = cnt[lane * ldc + e];
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            cnt[lane * ldc + e] = incl - c;
            if (lane == 31) load[(long long)t * E + e] = min(incl, C);
        }
    } else {
        for (int e = threadIdx.x; e < E; e += CS_THREADS) {
            int run = 0;
#pragma unroll 8
            for (int w = 0; w < CS_WARPS; ++w) {
                const int c = cnt[w * ldc + e];
                cnt[w * ldc + e] = run;
                run += c;
            }
            load[(long long)t * E + e] = min(run, C);
        }
    }
    __syncthreads();
    // Pass 2: ranks -> slots, each warp its own; from four choices on, whose places lie
    // apart, in memory order, the warp that ranked a place looked up: w = pos / per (both
    // quotients by a reciprocal: exact, as they lie half a part from an integer and total
    // is below 2^14).
    if (SMEM_IDX && k > 3) {
        const float rk = 1.0f / (float)k, rper = 1.0f / (float)per;
        for (int i = threadIdx.x; i < total; i += CS_THREADS) {
            const int q = (int)(((float)i + 0.5f) * rk);
            const int w = (int)(((float)((i - q * k) * N + q) + 0.5f) * rper);
            const int r = srank[i] + cnt[w * ldc + sidx[i]];
            slot[tb + i] = r < C ? r : -1;
        }
        return;
    }
    n = n_beg;
    j = j_beg;
    for (int p0 = beg; p0 < end; p0 += 32) {
        if (p0 + lane < end) {
            const int i = n * k + j, r = rank[i] + my[src[i]];
            slot[tb + i] = r < C ? r : -1;
        }
        if (p0 + 32 < end) advance(n, j);
    }
}

int launch_given(const Dims &p, const float *logits, int32_t *idx, float *gate, cudaStream_t s) {
    const size_t smem = sizeof(float) * (size_t)RT_TOK * (p.E + 1);
    static std::atomic<int> smem_limit[64];
    if (const int st = raise_smem_limit((const void *)route_given_kernel, smem_limit, (int)smem)) return st;
    trace_before(s, "route_topk");
    const int st = launch_kernel(route_given_kernel, dim3((p.N + RT_TOK - 1) / RT_TOK, p.T), dim3(RT_THREADS),
                                 smem, s, p, logits, idx, gate);
    trace_after(s);
    return st;
}

template <int ECH, int TOK, int KC, int SLICES>
int launch_f32(const Dims &p, const float *x, const float *wr, const float *bias, float *logits,
               int32_t *idx, float *gate, cudaStream_t s) {
    using S = RouteF32<ECH, TOK, KC, SLICES>;
    const size_t smem = S::smem(p.E);
    static std::atomic<int> smem_limit[64];
    auto kern = route_f32_kernel<ECH, TOK, KC, SLICES>;
    if (const int st = raise_smem_limit((const void *)kern, smem_limit, (int)smem)) return st;
    trace_before(s, "route_topk");
    const int st = launch_kernel(kern, dim3((p.N + TOK - 1) / TOK, p.T), dim3(S::NT), smem, s, p, x, wr, bias,
                                 logits, idx, gate);
    trace_after(s);
    return st;
}

template <int CS_THREADS>
int launch_scan(const Dims &p, const int32_t *idx, int32_t *slot, int32_t *load, cudaStream_t s) {
    const size_t total = (size_t)p.N * p.k;
    const size_t smem_small = sizeof(int) * (size_t)(CS_THREADS / 32) * cs_pitch(p.E);
    const size_t smem_big = smem_small + sizeof(int) * 2 * total;
    if (smem_big <= 96 * 1024) {
        static std::atomic<int> smem_limit[64];
        if (const int st = raise_smem_limit((const void *)capacity_scan_kernel<true, CS_THREADS>, smem_limit,
                                            (int)smem_big))
            return st;
        return launch_kernel(capacity_scan_kernel<true, CS_THREADS>, dim3(p.T), dim3(CS_THREADS), smem_big,
                             s, p, idx, slot, load);
    }
    return launch_kernel(capacity_scan_kernel<false, CS_THREADS>, dim3(p.T), dim3(CS_THREADS), smem_small,
                         s, p, idx, slot, load);
}

}  // namespace

int launch_route(const Dims &p, const void *x, const float *w_router, const float *bias,
                 float *logits, int32_t *idx, float *gate, int32_t *slot, int32_t *load,
                 cudaStream_t s) {
    int st;
    if (p.bf16 && x != nullptr) {
        const __nv_bfloat16 *xb = (const __nv_bfloat16 *)x;
        if (route_tc_enabled() && route_tc_width(p) > 0)
            st = launch_route_tc(p, xb, w_router, bias, logits, idx, gate, s);
        else
            st = p.E <= 32 ? launch_mma_router<4, 1>(p, xb, w_router, bias, logits, idx, gate, s)
                           : launch_mma_router<8, 2>(p, xb, w_router, bias, logits, idx, gate, s);
    } else if (x == nullptr) {
        st = launch_given(p, logits, idx, gate, s);
    } else {
        const float *xf = (const float *)x;
        // measured against the 16-token form (us, with the scan; 3 to 6000 tokens a task, d 8 to
        // 640, 4 to 256 experts): 100 tiles, E 64, d 8: 23.8 -> 14, d 264: 33.9 -> 25, but E 32, d
        // 640: 26.3 -> 30.1; 752 tiles, E 128, d 16: 197 -> 65; 50 tiles, d 136: slower from there on
        const long long tiles = (long long)((p.N + 63) / 64) * p.T;
        const bool many = tiles >= num_sms() || (2 * tiles >= num_sms() && p.d <= 512);
        if (many)
            st = p.E <= 32 ? launch_f32<32, 64, 32, 1>(p, xf, w_router, bias, logits, idx, gate, s)
                           : launch_f32<64, 64, 32, 1>(p, xf, w_router, bias, logits, idx, gate, s);
        else
            st = p.E <= 32 ? launch_f32<32, 16, 128, 8>(p, xf, w_router, bias, logits, idx, gate, s)
                           : launch_f32<64, 16, 128, 4>(p, xf, w_router, bias, logits, idx, gate, s);
    }
    if (st != VMOE_OK) return st;
    trace_before(s, "capacity_scan");
    st = p.E <= 128 ? launch_scan<1024>(p, idx, slot, load, s) : launch_scan<256>(p, idx, slot, load, s);
    trace_after(s);
    return st;
}

}  // namespace vmoe

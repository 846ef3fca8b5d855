// gemm_simt.cu -- K10: fp32 grouped GEMM on the CUDA cores, used for the
// fp32 problems (the accuracy bar there is 1e-5 of the RMS, which tf32 tensor
// cores do not meet).  One launch covers all T*E groups: blockIdx.z is the
// group.  The six contractions of the expert FFN map onto it with an operand
// layout (plain or transposed) and an epilogue (store, GELU with both H and A
// stored, or multiply by GELU'(H)).
//
// Row mode: output rows per group = load[g] (FC1, FC2, dA, dX).
// Weight-gradient mode: K per group = load[g] (dW1, dW2); an empty group's
// tile is written as zeros.
//
// A CTA computes a BM x BN tile, TM x TN per thread, over K chunks of 16 in two
// shared-memory buffers: the next chunk's 16-byte loads are in registers while
// this one is multiplied, one barrier a chunk.  When the tiles alone leave SMs
// idle, a cluster of S CTAs splits a tile's K range; the partial tiles are
// summed through distributed shared memory in rank order (no atomics).
#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace vmoe {
namespace {

enum { EPI_STORE = 0, EPI_GELU = 1, EPI_DGELU = 2 };

struct SimtArgs {
    const float *A;  // element (m,k): a_t ? A[k*lda + m] : A[m*lda + k]
    const float *B;  // element (k,n): b_t ? B[n*ldb + k] : B[k*ldb + n]
    float *D;        // D[m*ldd + n]
    float *D2;       // GELU: second output (A = GELU(H)), same layout as D
    const float *aux;  // DGELU: H, same layout as D
    long long sA, sB, sD;  // per-group strides (elements)
    int lda, ldb, ldd;
    int M, N, K;  // fixed sizes (M ignored in row mode, K ignored in wgrad mode)
    const int32_t *load;
    int C;         // capacity: load[g] is clamped to [0, C], as in the tensor-core path
    int row_mode;  // 1: M = load[g]; 0: K = load[g]
    int gelu_tanh;
    int split;     // CTAs (a cluster) that share one tile's K range
};

constexpr int ST_BK = 16;

template <int BM, int BN>
struct SimtTile {
    // row pitches: 16-byte aligned, and the transposing stores of a warp spread over the banks
    float A[2][ST_BK][BM + 4];
    float B[2][ST_BK][BN + 4];
};

// One operand's [ST_BK][W] chunk: V 16-byte vectors a thread, along the
// contiguous axis -- W (the tile's rows or columns), or K with CONTIG_K, where
// the four values go to four chunk rows.  Both extents are multiples of 4, so
// a vector is wholly inside or wholly outside (zeros).
template <int W, int NT, bool CONTIG_K>
struct SimtChunk {
    static constexpr int N4 = W * ST_BK / 4;  // vectors of a chunk
    static constexpr int V = (N4 + NT - 1) / NT;
    float4 v[V];
    __device__ __forceinline__ void load(const float *p, int ld, int w0, int wn, int k0, int kn) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int u = threadIdx.x + i * NT;
            const int w = w0 + (CONTIG_K ? u / (ST_BK / 4) : u % (W / 4) * 4);
            const int k = k0 + (CONTIG_K ? u % (ST_BK / 4) * 4 : u / (W / 4));
            v[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (u < N4 && w < wn && k < kn)
                v[i] = __ldg(reinterpret_cast<const float4 *>(
                    p + (CONTIG_K ? (long long)w * ld + k : (long long)k * ld + w)));
        }
    }
    __device__ __forceinline__ void store(float (*s)[W + 4]) const {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int u = threadIdx.x + i * NT;
            if (N4 % NT != 0 && u >= N4) continue;
            if (CONTIG_K) {
                const int w = u / (ST_BK / 4), k = u % (ST_BK / 4) * 4;
                s[k][w] = v[i].x;
                s[k + 1][w] = v[i].y;
                s[k + 2][w] = v[i].z;
                s[k + 3][w] = v[i].w;
            } else {
                *reinterpret_cast<float4 *>(&s[u / (W / 4)][u % (W / 4) * 4]) = v[i];
            }
        }
    }
};

// Four consecutive outputs of one row through the epilogue.
template <int EPI>
__device__ __forceinline__ void simt_store(const SimtArgs &a, int g, long long o, float4 v) {
    float *D = a.D + g * a.sD + o;
    if (EPI == EPI_DGELU) {
        const float4 h = __ldg(reinterpret_cast<const float4 *>(a.aux + g * a.sD + o));
        v.x *= gelu_deriv_f(h.x, a.gelu_tanh);
        v.y *= gelu_deriv_f(h.y, a.gelu_tanh);
        v.z *= gelu_deriv_f(h.z, a.gelu_tanh);
        v.w *= gelu_deriv_f(h.w, a.gelu_tanh);
    }
    *reinterpret_cast<float4 *>(D) = v;
    if (EPI == EPI_GELU)
        *reinterpret_cast<float4 *>(a.D2 + g * a.sD + o) =
            make_float4(gelu_f(v.x, a.gelu_tanh), gelu_f(v.y, a.gelu_tanh), gelu_f(v.z, a.gelu_tanh),
                        gelu_f(v.w, a.gelu_tanh));
}

template <int BM, int BN, int TM, int TN, int EPI, bool A_T, bool B_T>
__global__ void __launch_bounds__((BM / TM) * (BN / TN), 6) simt_gemm_kernel(const SimtArgs a) {
    constexpr int NT = (BM / TM) * (BN / TN), CT = BN / TN;
    __shared__ __align__(16) SimtTile<BM, BN> sm;
    pdl_wait();
    const int S = a.split, rank = S > 1 ? (int)(blockIdx.x % S) : 0;
    const int g = blockIdx.z;
    int Lg = __ldg(a.load + g);
    Lg = Lg < 0 ? 0 : (Lg > a.C ? a.C : Lg);
    const int M = a.row_mode ? Lg : a.M;
    const int K = a.row_mode ? a.K : Lg;
    const int m0 = blockIdx.y * BM, n0 = (int)(blockIdx.x / S) * BN;
    if (m0 >= M) return;  // the whole cluster: its CTAs share the tile
    const float *A = a.A + g * a.sA;
    const float *B = a.B + g * a.sB;
    const int tm = threadIdx.x / CT, tn = threadIdx.x % CT;
    // this CTA's K chunks
    const int chunks = (K + ST_BK - 1) / ST_BK;
    const int c0 = (int)((long long)chunks * rank / S), c1 = (int)((long long)chunks * (rank + 1) / S);
    // thread (tm, tn): rows 4 tm + 0..3 of each of the TM / 4 row blocks of BM / (TM / 4), columns likewise
    constexpr int RB = TM / 4, CB = TN / 4;
    unsigned long long acc2[TM / 2][TN] = {};  // rows 2i and 2i + 1 of the thread's tile
    SimtChunk<BM, NT, !A_T> ca;
    SimtChunk<BN, NT, B_T> cb;
    if (c0 < c1) {
        ca.load(A, a.lda, m0, M, c0 * ST_BK, K);
        cb.load(B, a.ldb, n0, a.N, c0 * ST_BK, K);
    }
    for (int c = c0; c < c1; ++c) {
        const int buf = c & 1;
        ca.store(sm.A[buf]);
        cb.store(sm.B[buf]);
        __syncthreads();  // this chunk is in; every thread is past its last read of the other buffer
        if (c + 1 < c1) {
            ca.load(A, a.lda, m0, M, (c + 1) * ST_BK, K);
            cb.load(B, a.ldb, n0, a.N, (c + 1) * ST_BK, K);
        }
#pragma unroll
        for (int kk = 0; kk < ST_BK; ++kk) {
            float av[TM], bv[TN];
#pragma unroll
            for (int r = 0; r < RB; ++r)
                *reinterpret_cast<float4 *>(av + 4 * r) =
                    *reinterpret_cast<const float4 *>(&sm.A[buf][kk][r * (BM / RB) + 4 * tm]);
#pragma unroll
            for (int r = 0; r < CB; ++r)
                *reinterpret_cast<float4 *>(bv + 4 * r) =
                    *reinterpret_cast<const float4 *>(&sm.B[buf][kk][r * (BN / CB) + 4 * tn]);
#pragma unroll
            for (int j = 0; j < TN; ++j) {  // packed: two rows a fused multiply-add
                unsigned long long bb;
                asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(bv[j]));
#pragma unroll
                for (int i = 0; i < TM; i += 2) {
                    unsigned long long aa;
                    asm("mov.b64 %0, {%1, %2};" : "=l"(aa) : "f"(av[i]), "f"(av[i + 1]));
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[i / 2][j]) : "l"(aa), "l"(bb));
                }
            }
        }
    }
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; i += 2)
#pragma unroll
        for (int j = 0; j < TN; ++j)
            asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[i][j]), "=f"(acc[i + 1][j]) : "l"(acc2[i / 2][j]));
    static_assert(BM * BN * sizeof(float) <= sizeof(SimtTile<BM, BN>), "a partial tile fits the buffers");
    if (S > 1) {
        float *red = reinterpret_cast<float *>(&sm);  // [BM][BN]
        __syncthreads();
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int r = 0; r < CB; ++r)
                *reinterpret_cast<float4 *>(red + ((i / 4) * (BM / RB) + 4 * tm + i % 4) * BN + r * (BN / CB) + 4 * tn) =
                    make_float4(acc[i][4 * r], acc[i][4 * r + 1], acc[i][4 * r + 2], acc[i][4 * r + 3]);
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        // rank r finishes rows [BM r / S, BM (r + 1) / S), the ranks' parts summed in order
        const int rows = BM / S;
        for (int u = threadIdx.x; u < rows * (BN / 4); u += NT) {
            const int r = rank * rows + u / (BN / 4), n = u % (BN / 4) * 4;
            if (m0 + r >= M || n0 + n >= a.N) continue;
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            for (int q = 0; q < S; ++q) {
                const float4 w = *reinterpret_cast<const float4 *>(cluster.map_shared_rank(red, q) + r * BN + n);
                v.x += w.x;
                v.y += w.y;
                v.z += w.z;
                v.w += w.w;
            }
            simt_store<EPI>(a, g, (long long)(m0 + r) * a.ldd + n0 + n, v);
        }
        cluster.sync();  // the parts stay until every rank has read them
        return;
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + (i / 4) * (BM / RB) + 4 * tm + i % 4;
        if (m >= M) continue;
#pragma unroll
        for (int r = 0; r < CB; ++r) {
            const int n = n0 + r * (BN / CB) + 4 * tn;
            if (n < a.N)
                simt_store<EPI>(a, g, (long long)m * a.ldd + n,
                                make_float4(acc[i][4 * r], acc[i][4 * r + 1], acc[i][4 * r + 2], acc[i][4 * r + 3]));
        }
    }
}

template <int BM, int BN, int TM, int TN, int EPI, bool A_T, bool B_T>
int run_tile(SimtArgs a, int G, int mmax, int split, cudaStream_t s, const char *name) {
    a.split = split;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((a.N + BN - 1) / BN * split), (mmax + BM - 1) / BM, G);
    cfg.blockDim = dim3((BM / TM) * (BN / TN));
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
    trace_before(s, name);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, simt_gemm_kernel<BM, BN, TM, TN, EPI, A_T, B_T>, a);
    trace_after(s);
    return e == cudaSuccess ? VMOE_OK : VMOE_ERR_CUDA;
}

// Tile choice: 64 x 64 tiles of 8 x 4 outputs a thread (8 x 8 left too few warps:
// 16-wide rows of K = 256 took 13 us instead of 10), and a K split over up to 8 CTAs
// while the tiles give an SM fewer than three CTAs and a part keeps 3 chunks or more.
// 128 x 128 tiles of 16 x 8, nearer the FMA rate on paper (a warp's shared-memory
// reads cost TM + TN wavefronts a k against TM * TN / 4 cycles of its scheduler's FMA
// pipe), run two CTAs an SM and multiply 128 rows for any load: over 12 layers, C 33
// to 2400 and loads of a third to all of C they took 0.9 to 4 times these tiles'
// time, above 1 but for the weight gradients of d 384, f 1536 and d 512, f 2048
// (0.95-0.97) and row GEMMs with 2400 rows in every group.
// Measured on GB300 (us; the 64 x 64 kernel of 4 x 4 outputs that this replaced
// -> now), 512 groups of 10 rows at C 33, d 64, f 256: FC2 69 -> 33, dX 57 -> 33, dA
// 51 -> 33 (100, 93 and 67 with 128 x 128); 48 groups of 300 at C 500, d 200, f 800:
// FC1 297 -> 119, dW1 330 -> 129.
// Row mode stays at 47% of the FMA pipe: half of its second 64-row tile is padding,
// and shared-memory reads fill 75% of the L1.
// Groups of at most 32 rows take tiles of 16 or 32 rows instead of computing 64 (6
// tasks of 30 experts of at most 13 rows, d 336, f 1168: the step 1807 -> 607 us).
// kmax: the longest reduction (row mode: K; weight gradients: C rows).
template <int EPI, bool A_T, bool B_T>
int run(const SimtArgs &a, int G, int mmax, cudaStream_t s, const char *name) {
    const int kmax = a.row_mode ? a.K : a.C;
    const long long sms = num_sms();
    const bool few = a.row_mode && mmax <= 32;  // one tile of 16 or 32 rows a group
    const long long small = few ? (long long)((a.N + 127) / 128) * G
                                : (long long)((a.N + 63) / 64) * ((mmax + 63) / 64) * G;
    int split = 1;
    while (split < 8 && small * split < 3 * sms && kmax >= 2 * split * 3 * ST_BK) split *= 2;
    if (few && !A_T)
        return mmax <= 16 ? run_tile<16, 128, 4, 4, EPI, false, B_T>(a, G, mmax, split, s, name)
                          : run_tile<32, 128, 8, 4, EPI, false, B_T>(a, G, mmax, split, s, name);
    return run_tile<64, 64, 8, 4, EPI, A_T, B_T>(a, G, mmax, split, s, name);
}

SimtArgs base(const Dims &p) {
    SimtArgs a = {};
    a.C = p.C;
    a.gelu_tanh = (p.flags & VMOE_GELU_TANH) != 0;
    return a;
}

}  // namespace

int launch_expert_fwd_f32(const Dims &p, const float *xe, const float *w1, const float *w2,
                          const int32_t *load, float *h, float *act, float *ye, cudaStream_t s) {
    const int G = p.G(), C = p.C, d = p.d, f = p.f;
    // FC1: H[C,f] = Xe[C,d] W1[d,f]; A = GELU(H)
    SimtArgs a = base(p);
    a.A = xe; a.sA = (long long)C * d; a.lda = d;
    a.B = w1; a.sB = (long long)d * f; a.ldb = f;
    a.D = h; a.D2 = act; a.sD = (long long)C * f; a.ldd = f;
    a.N = f; a.K = d; a.load = load; a.row_mode = 1;
    int st = run<EPI_GELU, false, false>(a, G, C, s, "simt_fc1_gelu");
    if (st != VMOE_OK) return st;
    // FC2: Ye[C,d] = A[C,f] W2[f,d]
    a = base(p);
    a.A = act; a.sA = (long long)C * f; a.lda = f;
    a.B = w2; a.sB = (long long)f * d; a.ldb = d;
    a.D = ye; a.sD = (long long)C * d; a.ldd = d;
    a.N = d; a.K = f; a.load = load; a.row_mode = 1;
    return run<EPI_STORE, false, false>(a, G, C, s, "simt_fc2");
}

int launch_expert_bwd_f32(const Dims &p, const float *xe, const float *h, const float *act,
                          const float *w1, const float *w2, const float *dye,
                          const int32_t *load, float *dxe, float *dw1, float *dw2, float *dh,
                          cudaStream_t s) {
    const int G = p.G(), C = p.C, d = p.d, f = p.f;
    // dA: dH[C,f] = (dYe[C,d] W2^T) * GELU'(H); B(k=i, n=c) = W2[c, i]
    SimtArgs a = base(p);
    a.A = dye; a.sA = (long long)C * d; a.lda = d;
    a.B = w2; a.sB = (long long)f * d; a.ldb = d;
    a.D = dh; a.aux = h; a.sD = (long long)C * f; a.ldd = f;
    a.N = f; a.K = d; a.load = load; a.row_mode = 1;
    int st = run<EPI_DGELU, false, true>(a, G, C, s, "simt_da_dgelu");
    if (st != VMOE_OK) return st;
    // dX: dXe[C,d] = dH[C,f] W1^T; B(k=c, n=i) = W1[i, c]
    a = base(p);
    a.A = dh; a.sA = (long long)C * f; a.lda = f;
    a.B = w1; a.sB = (long long)d * f; a.ldb = f;
    a.D = dxe; a.sD = (long long)C * d; a.ldd = d;
    a.N = d; a.K = f; a.load = load; a.row_mode = 1;
    if ((st = run<EPI_STORE, false, true>(a, G, C, s, "simt_dx")) != VMOE_OK) return st;
    // dW1[d,f] = Xe^T dH; A(m=i, k=s) = Xe[s, i]
    a = base(p);
    a.A = xe; a.sA = (long long)C * d; a.lda = d;
    a.B = dh; a.sB = (long long)C * f; a.ldb = f;
    a.D = dw1; a.sD = (long long)d * f; a.ldd = f;
    a.M = d; a.N = f; a.load = load; a.row_mode = 0;
    if ((st = run<EPI_STORE, true, false>(a, G, d, s, "simt_dw1")) != VMOE_OK) return st;
    // dW2[f,d] = A^T dYe; A(m=c, k=s) = A[s, c]
    a = base(p);
    a.A = act; a.sA = (long long)C * f; a.lda = f;
    a.B = dye; a.sB = (long long)C * d; a.ldb = d;
    a.D = dw2; a.sD = (long long)f * d; a.ldd = d;
    a.M = f; a.N = d; a.load = load; a.row_mode = 0;
    return run<EPI_STORE, true, false>(a, G, f, s, "simt_dw2");
}

}  // namespace vmoe

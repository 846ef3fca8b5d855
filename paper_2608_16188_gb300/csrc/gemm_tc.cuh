// gemm_tc.cuh -- K3/K4/K6-K9: the bf16 grouped GEMM of the expert FFN on the
// sm_103a tensor cores (tcgen05 + TMEM + TMA), one persistent launch over all
// T*E (task, expert) groups of the merged expert pool.
//
// Structure (one CTA per SM, 352 threads; 608 for the two-output epilogues):
//   warp 0 and the last warp
//               TMA producers: one thread streams 128x64 A tiles, another
//               64xBN B tiles, into a STAGES-deep ring of shared-memory slots
//               (128-byte swizzle), each signalling `full[s]` with its byte count.
//   warp 1      MMA issuer: one thread issues tcgen05.mma (M=128, N=BN,
//               K=16, bf16 in, fp32 accumulate in TMEM), commits each slot
//               back to `empty[s]` and each finished tile to `tmem_full[a]`.
//   warps 2-9 (2-17)
//               epilogue: tcgen05.ld of the accumulator (one TMEM lane per
//               thread = one output row; the warps of a lane quarter split the
//               columns), the fused elementwise step (GELU, or GELU' of an H
//               prefetched into registers one chunk ahead), bf16 packing, a
//               per-warp staging tile in shared memory and coalesced 16-byte
//               row stores (weight gradients, whose tiles are always full:
//               TMA bulk tensor stores from 128-byte-swizzled staging).
//               The accumulator is double buffered in TMEM
//               (2 x BN columns), so tile i's epilogue overlaps tile i+1's
//               main loop.
// Tiles are distributed statically: CTA b takes tiles b, b + grid, ...  In
// row mode (H = Xe W1 etc.) a group contributes ceil(load/128) x N/BN tiles,
// counted from the device-resident loads by every CTA with a block scan, so
// empty groups cost nothing and no host round trip is needed.  In weight-
// gradient mode (dW1 = Xe^T dH etc.) every group contributes (M/128) x (N/BN)
// tiles whose K = load[g] rows; an empty group's tile is written as zeros.
//
// Every wait on an mbarrier is bounded in time; a wait that runs out sets the
// library's device status word to VMOE_ERR_DEVICE_TIMEOUT and an abort flag
// that the other roles see, and the CTA drains its copies and MMAs in flight
// and frees its TMEM before it returns.
#pragma once

#include <cuda.h>  // CUtensorMap and its enums (types only; the encoder is fetched at run time)

#include <type_traits>

#include "common.cuh"

namespace vmoe {
namespace tc {

constexpr int BM = 128;  // rows of one MMA tile (TMEM lanes)
constexpr int BK = 64;   // K per pipeline slot = one 128-byte swizzle row of bf16
constexpr int THREADS = 320;  // SM-pair row kernel: warp 0 TMA, warp 1 MMA, warps 2-9 epilogue
constexpr int EPI_WARP_BYTES = 32 * 80;  // 32 rows x (64 data + 16 pad) bytes

// Row-mode epilogue of the one-SM grouped GEMM: the two-output epilogues
// (FC1 + GELU, dA + GELU') run 16 epilogue warps (4 per TMEM lane quarter),
// the plain store 8, all in 32-column chunks.  The two-output epilogues spend
// about 26 instructions per output element, which 8 warps do not issue fast
// enough; 16 warps leave room for 3 pipeline stages instead of 4, which the
// plain-store GEMMs, bound by their operand stream, cannot spare.  Measured on
// GB300 (ms; 8 -> 16 warps, then at 31 to 38 instructions an element): dA 0.536 ->
// 0.518 and FC1 0.485 -> 0.477 at the 17-task ViT-B step, 0.370 -> 0.321 and 0.301
// -> 0.285 at the 6-task one; FC2 / dX 0.425 -> 0.433 / 0.434 -> 0.445 at 17 tasks,
// hence 8 there.  16-column chunks (4 stages with 16 warps) gained nothing.
constexpr int EPI_WARP_BYTES_TMA = 2 * 4096;  // two 32 x 64 bf16 tiles, 128-byte swizzle
constexpr int MAX_G = 1024;
constexpr unsigned long long TIMEOUT_NS = 4000000000ull;

enum { MODE_ROW = 0, MODE_WGRAD = 1 };
enum { EPI_STORE = 0, EPI_GELU = 1, EPI_DGELU = 2 };

constexpr int ROW_CH = 32;
template <int MODE, int EPI>
struct Roles {
    static constexpr int EW = (MODE == 0 && EPI != EPI_STORE) ? 16 : 8;  // epilogue warps
    static constexpr int NT = 96 + 32 * EW;  // threads: A producer, MMA, epilogue, B producer
    static constexpr int PITCH = 80;         // staging row pitch (bytes): 64 data + 16 pad
};

// Epilogue store path per mode.  TMA bulk tensor stores from 128-byte-
// swizzled staging need 64 KB of shared memory, which leaves room for 3
// pipeline slots at BN 256 instead of 4.  Measured on GB300 at the 17-task
// ViT-B step, they pay for the weight gradients (always-full tiles, write-
// bound) only; every row-mode GEMM -- FC1 + GELU and dA + GELU' with their two
// outputs included -- is faster with 4 slots and row-masked st.global (FC1:
// 0.485 ms against 0.492 ms with TMA stores).
template <int MODE, int EPI>
struct UseTmaStore {
    static constexpr bool value = MODE == 1;
};

template <int BN, int MODE, int EPI>
struct Shape {
    // Weight gradients are bound by their stores, not by the ring (their K is a
    // group's load): 3 slots at BN 256 leave room for the double-buffered
    // 128-byte-swizzled TMA-store staging.
    static constexpr bool TMA_EPI = UseTmaStore<MODE, EPI>::value;
    static constexpr int NT = Roles<MODE, EPI>::NT;
    static constexpr int EPI_BYTES =
        TMA_EPI ? 8 * EPI_WARP_BYTES_TMA : Roles<MODE, EPI>::EW * 32 * Roles<MODE, EPI>::PITCH;
    static constexpr uint32_t A_BYTES = BM * BK * 2;
    static constexpr uint32_t B_BYTES = BN * BK * 2;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr size_t FIXED = 1024 + EPI_BYTES + 16 + NT * 4 + (MAX_G + 1) * 4 + 8 * 21;
    static constexpr int STAGES_FIT = (int)((232448 - FIXED) / STAGE_BYTES);
    static constexpr int STAGES_MAX = TMA_EPI ? (BN == 256 ? 3 : 4) : (BN == 256 ? 4 : 6);
    static constexpr int STAGES = STAGES_FIT < STAGES_MAX ? STAGES_FIT : STAGES_MAX;
    static constexpr uint32_t TMEM_COLS = BN == 192 ? 512 : 2 * BN;  // a power of two
    static constexpr int NUM_BARS = 2 * STAGES + 5;
    static constexpr size_t SMEM_BYTES = 1024 + (size_t)STAGES * STAGE_BYTES + EPI_BYTES +
                                         NUM_BARS * 8 + 16 + NT * 4 + (MAX_G + 1) * 4;
    static_assert(SMEM_BYTES <= 232448, "over the 227 KB shared-memory limit");
};

struct Args {
    int G, C;
    int N;        // output columns
    int K_fixed;  // row mode: reduction length
    int M_fixed;  // weight-gradient mode: output rows
    int tiles_n;  // N / BN
    int tiles_m;  // weight-gradient mode: M_fixed / BM; row mode: ceil(C / BM)
    const int32_t *load;
    __nv_bfloat16 *D;          // output (EPI_DGELU: the bf16 part of dH)
    __nv_bfloat16 *D2;         // EPI_GELU: A = GELU(H); EPI_DGELU: the bf16 residual of dH
    const __nv_bfloat16 *aux;  // EPI_DGELU: H
    long long sD;              // group stride of D / D2 (elements)
    long long sAux;            // group stride of aux (elements)
    int ldd;                   // row stride of D / D2 / aux (elements)
    int ksplit;                // weight-gradient mode, 0 or 1: B holds [hi rows; lo rows] (K doubled)
    int gelu_tanh;
    int late_wait;             // weight gradients: see wait_for_predecessor
    int *status;
    // Slices (the memory-budgeted backward): the launch covers G entries, entry i
    // being group glist[i] of the real tensors (glist NULL: entry i = group i).
    // Operands flagged in `compact` live in a compact buffer instead, entry i's
    // rows starting at row crow[i] (with ksplit / a second output, the residual
    // rows follow the entry's load rows).
    const int32_t *glist;
    const int32_t *crow;
    int compact;               // CMP_* bits
};
enum { CMP_A = 1, CMP_B = 2, CMP_D = 4 };

// Partial-box tensor maps: a group's padding rows [load, C) are not read.  Row
// mode: a[0..2] = the A operand with 64-, 32- and 16-row boxes; a tile whose
// valid rows end inside it loads rows [0, 16 ceil(rows / 16)) as at most three
// boxes instead of one 128-row box.
struct TailMaps {
    CUtensorMap a[3];
};
__device__ __forceinline__ int real_group(const Args &a, int i) { return a.glist ? a.glist[i] : i; }

// A late weight gradient (launch_chain.h: nothing that may still be running writes
// what it reads, or touches what it writes) starts on the SMs which its predecessor's
// last wave leaves idle, and waits for its predecessor at its end (late_wait) instead
// of its start.  By waiting before it exits it hands on "complete" to whatever waits
// for it.
// What it reads was written by kernels that had completed before the last launch that
// waited at its start let its successor start (dW1 behind dX: dH by dA, which dX waited
// for; dW2 behind a late dW1 that has not waited yet: A and dYe, through dX again).
// Complete, so performed in L2; but without a wait of its own nothing documented
// makes that visible here, so it starts with an acquire at GPU scope, for its plain
// loads (loads, slice plans: never through the non-coherent path), and a proxy fence
// for its TMA loads, which read L2.
// Measured on GB300 (us a step or call): ViT-S 214 -> 210, ragged top-3 255 -> 250,
// 17 tasks 2837 -> 2819, the budgeted backward 2153 -> 2128, attention at C 247
// 1130 -> 1116.
__device__ __forceinline__ void wait_for_predecessor(const Args &a, bool at_end) {
    if ((a.late_wait != 0) == at_end) {
        pdl_wait();
    } else if (!at_end) {
        __threadfence();
        asm volatile("fence.proxy.async;" ::: "memory");
    }
}

// ---------------------------------------------------------------------------
// PTX wrappers.

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for the phase of parity `parity` of barrier `bar`.  The first
// test is inline: a call for every k-block cost a producer 120 of its 540
// cycles (measured on a loop of 16 KB copies), which is what bounds the GEMMs of
// layers that stay in L2.
static __device__ __noinline__ bool wait_phase_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                                    int *status, unsigned long long limit_ns) {
    const unsigned long long t0 = global_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                if (status) atomicExch(status, (int)VMOE_ERR_DEVICE_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                           unsigned long long limit_ns = TIMEOUT_NS) {
    return mbar_try_wait(bar, parity) || wait_phase_slow(bar, parity, abort_flag, status, limit_ns);
}
// Arrive on an mbarrier of another CTA of the cluster without a release at cluster
// scope, for barriers whose waiter orders through tcgen05 or proxy fences rather than
// through memory.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// One lane of a converged warp, the same one every time.  The compiler takes
// the branch as run by one thread, which a test of the lane index does not tell
// it: a k-block of four 128 x 128 MMAs with its wait and commit then issues in
// 310 cycles instead of 427 (of 128 x 64: 238 instead of 347).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                            int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
// L2 policy of the weight-gradient stores: first to be evicted.  Nothing reads
// a gradient again before the step ends, and its lines otherwise push the
// activations out.  Measured at the 17-task step (before dynamic tiles): dW1 522
// -> 506 us, dW2 499 -> 477 us; the attention experts' dW_qkv 375 -> 355 us.
__device__ __forceinline__ uint64_t evict_first_policy() {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, uint32_t src, int c0, int c1,
                                             int c2, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3, %4}], [%1], %5;" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(src), "r"(c0), "r"(c1), "r"(c2), "l"(policy)
        : "memory");
}
// An empty group's weight gradient is zeros, one contiguous slab: its unit (or
// tile) `part` of `parts` writes its share of the slab's 4 KB pieces by copies of
// `zeros` (4 KB of zeroed shared memory), `w` of `nw` warps taking every nw-th
// piece (called by one thread).  slab: bytes, a multiple of 4096.  Against 32 x 64
// boxes staged and waited for one by one, the Zipf-skewed step, where two groups in
// three are empty, went from 2386 to 2353 us.
__device__ __forceinline__ void store_zeros(uint8_t *slab_base, long long slab, int part, int parts, int w, int nw,
                                            uint32_t zeros, uint64_t policy) {
    const long long pieces = slab / 4096, end = pieces * (part + 1) / parts;
    for (long long i = pieces * part / parts + w; i < end; i += nw)
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], 4096, %2;" ::"l"(
                         slab_base + i * 4096),
                     "r"(zeros), "l"(policy)
                     : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read1() {
    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read0() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
// ---------------------------------------------------------------------------
// Dynamic tiles by cluster launch control (the SM-pair weight gradients): the grid
// has a CTA pair per tile, the ones that run take the next one not yet launched
// (clusterlaunchcontrol.try_cancel) instead of a fixed stride.  The tiles in
// work are then always the oldest ones, so the addresses being written stay
// close together; with a fixed stride the SMs drift apart and DRAM loses
// bandwidth to it: zeros to 4 GB by 4 KB bulk copies from one CTA an SM run
// 6.8 TB/s with a stride and 7.8 TB/s this way.
//
// One thread a CTA asks (clc_scheduler), CLC_DEPTH answers ahead of the roles;
// every role reads each answer (clc_take) and frees its slot.  In a pair the
// leader asks and the answer goes to both CTAs, so a slot is free only once every
// reader in both has read it: the roles of both, and the peer's scheduler, which
// reads each answer too and would leave early if a later one, the last, overwrote
// it (the leader's own scheduler reads an answer before it asks for the next).  Each
// reader's proxy fence orders its read before its arrive; releases at cluster scope
// would stall the SM's bulk stores (by every role: 17 tasks 2850 -> 3168 us).
constexpr int CLC_DEPTH = 4;
struct ClcQueue {
    uint4 resp[CLC_DEPTH + 1];  // the last one: draining after an abort
    uint64_t full[CLC_DEPTH], empty[CLC_DEPTH], drain;
};
// One request, its answer to `resp` and `bar` of both CTAs of the pair (BOTH), or of
// this one alone.
template <bool BOTH>
__device__ __forceinline__ void clc_try(uint32_t resp, uint32_t bar) {
    if (BOTH)
        asm volatile(
            "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.multicast::cluster::all.b128 "
            "[%0], [%1];" ::"r"(resp),
            "r"(bar)
            : "memory");
    else
        asm volatile(
            "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(resp),
            "r"(bar)
            : "memory");
}
// Whether an answer holds a CTA, and its (a pair's first) blockIdx.x.
__device__ __forceinline__ bool clc_query(uint32_t resp, uint32_t &x) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .b128 r;\n\t.reg .pred p;\n\t"
        "ld.shared.b128 r, [%2];\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
        "selp.u32 %1, 1, 0, p;\n\t"
        "mov.u32 %0, 0;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, r;\n\t}\n"
        : "=r"(x), "=r"(ok)
        : "r"(resp)
        : "memory");
    return ok != 0;
}
// consumers: arrivals that free a slot (a pair's leader counts both CTAs' roles and its peer's scheduler)
__device__ __forceinline__ void clc_init(ClcQueue &q, int consumers) {
    for (int i = 0; i < CLC_DEPTH; ++i) {
        mbar_init(smem_u32(q.full + i), 1);
        mbar_init(smem_u32(q.empty + i), consumers);
    }
    mbar_init(smem_u32(&q.drain), 1);
}
// One thread a CTA.  leader_empty: 0 in the CTA that asks; in a pair's peer, which
// only receives, the leader's `empty` barriers.
// After an abort the CTAs not launched yet are taken and dropped, so that none
// of them starts and runs into the same wait -- as long as each answer has been
// read and held a CTA: asking again after "none left" is undefined.
__device__ __forceinline__ void clc_scheduler(ClcQueue &q, uint32_t leader_empty, volatile int *abort_flag,
                                              int *status) {
    const bool issue = leader_empty == 0;
    uint32_t ph = 0, x;
    int s = 0;
    bool more = true, ok = true;
    while (more) {
        if (!wait_phase(smem_u32(q.empty + s), ph ^ 1u, abort_flag, status)) {
            ok = false;
            break;
        }
        fence_proxy_async();  // the readers' reads of the slot before it is written again
        mbar_expect_tx(smem_u32(q.full + s), 16);
        if (issue) clc_try<true>(smem_u32(q.resp + s), smem_u32(q.full + s));
        if (!wait_phase(smem_u32(q.full + s), ph, abort_flag, status)) {
            ok = false;
            const unsigned long long t0 = global_ns();  // the answer in flight lands before the CTA exits
            bool landed = false;
            while (!landed && global_ns() - t0 < 100000000ull) landed = mbar_try_wait(smem_u32(q.full + s), ph);
            more = landed && clc_query(smem_u32(q.resp + s), x);
            break;
        }
        more = clc_query(smem_u32(q.resp + s), x);
        if (!issue) {
            fence_proxy_async();  // this read, too, before the leader's next answer lands in the slot
            mbar_arrive_remote(leader_empty + 8u * (uint32_t)s);
        }
        if (++s == CLC_DEPTH) {
            s = 0;
            ph ^= 1u;
        }
    }
    pdl_launch_dependents();  // nothing is left to take
    for (uint32_t n = 0; !ok && more && issue && n < (1u << 28); ++n) {
        const unsigned long long t0 = global_ns();
        fence_proxy_async();
        mbar_expect_tx(smem_u32(&q.drain), 16);
        clc_try<false>(smem_u32(q.resp + CLC_DEPTH), smem_u32(&q.drain));
        bool got = false;
        while (!got && global_ns() - t0 < 100000000ull) got = mbar_try_wait(smem_u32(&q.drain), n & 1u);
        if (!got || !clc_query(smem_u32(q.resp + CLC_DEPTH), x)) break;
    }
}
// A role's place in the queue.  WARP: the whole warp takes (lane 0 frees the
// slot), else one thread.  leader_empty: in a pair's peer, the leader's `empty`
// barriers (cluster address), which it frees too.
struct ClcPos {
    int s = 0;
    uint32_t ph = 0;
};
template <bool WARP>
__device__ __forceinline__ bool clc_take(ClcQueue &q, ClcPos &c, uint32_t &x, volatile int *abort_flag, int *status,
                                         uint32_t leader_empty = 0) {
    if (!wait_phase(smem_u32(q.full + c.s), c.ph, abort_flag, status)) return false;
    const bool ok = clc_query(smem_u32(q.resp + c.s), x);
    fence_proxy_async();
    if (WARP) __syncwarp();
    if (!WARP || (threadIdx.x & 31) == 0) {
        mbar_arrive(smem_u32(q.empty + c.s));
        if (leader_empty) mbar_arrive_remote(leader_empty + 8u * (uint32_t)c.s);
    }
    if (++c.s == CLC_DEPTH) {
        c.s = 0;
        c.ph ^= 1u;
    }
    return ok;
}

// Named barrier over `count` threads (ids 1..15; 0 is __syncthreads).
__device__ __forceinline__ void named_bar(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     bar)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
        "%12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, "
        "%30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
        "%12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle (tcgen05 format: start
// address, leading and stride byte offsets in 16-byte units, version 1 at bit
// 46, layout SWIZZLE_128B = 2 at bits 61-63).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Operand tiles in shared memory:
//  K-major (K contiguous):  rows of 64 K-elements = 128 bytes, 8-row swizzle
//    atoms of 1024 bytes stacked along M/N (SBO = 1024).  Step k16 -> +32 bytes.
//  MN-major (M/N contiguous): chunks of 64 MN-elements x 64 K-rows (8 KiB),
//    one TMA box each, stacked along M/N (LBO = 8192, the MN chunk stride);
//    8-row K groups are 1024 bytes apart (SBO).  Step k16 -> +2048 bytes.
__device__ __forceinline__ uint64_t operand_desc(uint32_t tile, int kk, bool mn_major) {
    return mn_major ? sdesc_sw128(tile + kk * 2048, 8192, 1024)
                    : sdesc_sw128(tile + kk * 32, 16, 1024);
}
// The descriptor kk K-steps of 16 on (the address field counts 16 bytes and does
// not overflow: shared memory ends below 2^18).
__device__ __forceinline__ uint64_t desc_step(uint64_t d, int kk, bool mn_major) {
    return d + (uint64_t)(kk * ((mn_major ? 2048 : 32) >> 4));
}

// Instruction descriptor of tcgen05.mma kind::f16: D fp32 (bits 4-5 = 1),
// A and B bf16 (bits 7-9, 10-12 = 1), A / B MN-major (bits 15 / 16),
// N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) |
           ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Zeroes a warp's first 4 KB staging tile for store_zeros, once the copies that
// read it are done (`zeroed`: it already holds zeros).
__device__ __forceinline__ void zero_staging(uint8_t *stg, bool &zeroed) {
    if (zeroed) return;
    const int lane = threadIdx.x & 31;
    if (lane == 0) bulk_wait_read0();
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<uint4 *>(stg + (i * 32 + lane) * 16) = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
    __syncwarp();
    zeroed = true;
}

// A warp's 32 rows x 64 CHUNKS columns of fp32 accumulators as bf16, 64 columns
// at a time through its 128-byte-swizzled staging tile(s) (BUFS of 4 KB) and TMA
// bulk tensor stores; only the first `valid` chunks.
template <int CHUNKS, int BUFS>
__device__ __forceinline__ void store_columns(const CUtensorMap &map, const uint32_t (&r)[2 * CHUNKS][32], uint8_t *stg,
                                              int &nstore, int col, int row, int g, uint64_t policy,
                                              int valid = CHUNKS) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
        if (c >= valid) break;
        uint8_t *buf = stg + (BUFS == 2 ? (nstore & 1) * 4096 : 0);
        if (lane == 0 && nstore >= BUFS) {  // the store that used buf has read it
            if (BUFS == 2) bulk_wait_read1();
            else bulk_wait_read0();
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t *src = &r[2 * c + (j >> 2)][(j & 3) * 8];
            uint4 pk;
            pk.x = pack_bf16x2(__uint_as_float(src[0]), __uint_as_float(src[1]));
            pk.y = pack_bf16x2(__uint_as_float(src[2]), __uint_as_float(src[3]));
            pk.z = pack_bf16x2(__uint_as_float(src[4]), __uint_as_float(src[5]));
            pk.w = pack_bf16x2(__uint_as_float(src[6]), __uint_as_float(src[7]));
            *reinterpret_cast<uint4 *>(buf + lane * 128 + ((j ^ (lane & 7)) << 4)) = pk;
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            tma_store_3d(&map, smem_u32(buf), col + c * 64, row, g, policy);
            bulk_commit();
        }
        ++nstore;
    }
}

struct Tile {
    int g, m_blk, n_blk, kblocks, kvalid, rows_valid;
    int khalf;  // weight-gradient mode: k-blocks per half (kblocks = 2 * khalf with ksplit)
    int gr;     // the real group of entry g
    int crow;   // entry g's first row in the compact buffer
    int col0, bn;  // row mode: first column and columns (BN, or BN >> cut from tile `wide` on)
};

// Row mode with CUT: tiles from index `wide` on are halves (cut = 1) of BN / 2 columns.
template <int MODE, int BN, bool CUT>
__device__ __forceinline__ Tile decode_tile(const Args &a, const int *prefix, int u, int wide, int cut) {
    Tile t;
    if (MODE == MODE_ROW) {
        int piece = 0;
        t.bn = BN;
        if (CUT && u >= wide) {
            piece = (u - wide) & ((1 << cut) - 1);
            u = wide + ((u - wide) >> cut);
            t.bn = BN >> cut;
        }
        int lo = 0, hi = a.G;  // prefix[lo] <= u < prefix[hi]
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (prefix[mid] <= u) lo = mid; else hi = mid;
        }
        t.g = lo;
        t.gr = real_group(a, lo);
        t.crow = a.crow ? __ldg(a.crow + lo) : 0;
        int local = u - prefix[lo];
        t.m_blk = local / a.tiles_n;
        t.n_blk = local - t.m_blk * a.tiles_n;
        t.col0 = t.n_blk * BN + piece * t.bn;
        t.kblocks = a.K_fixed / BK;
        t.khalf = t.kblocks;
        t.kvalid = a.K_fixed;
        int L = __ldg(a.load + t.gr);
        t.rows_valid = L < 0 ? 0 : (L > a.C ? a.C : L);
    } else {
        int tpg = a.tiles_m * a.tiles_n;
        t.g = u / tpg;
        t.gr = real_group(a, t.g);
        t.crow = a.crow ? a.crow[t.g] : 0;
        int local = u - t.g * tpg;
        t.m_blk = local / a.tiles_n;
        t.n_blk = local - t.m_blk * a.tiles_n;
        int L = a.load[t.gr];
        L = L < 0 ? 0 : (L > a.C ? a.C : L);
        t.kvalid = L;
        t.khalf = (L + BK - 1) / BK;
        t.kblocks = a.ksplit ? 2 * t.khalf : t.khalf;
        t.rows_valid = a.M_fixed;
    }
    return t;
}

// The elementwise step of a row-mode epilogue on CH accumulator columns of one
// row (pairs in v, clobbered), packed to bf16: out(words, 0) for the first
// output and out(words, 1) for the second -- A = GELU(H), or the residual
// v - bf16(v) of dH, which carries it to about 16 bits.  h: EPI_DGELU's H
// values of the chunk.
template <int EPI, int CH, typename Out>
__device__ __forceinline__ void epilogue_chunk(f32x2 (&v)[CH / 2], const uint4 *h, bool tanh_form, Out out) {
    uint32_t w[CH / 2];
    if (EPI == EPI_DGELU) {
        const uint32_t *hw = reinterpret_cast<const uint32_t *>(h);
        if (tanh_form) {
#pragma unroll
            for (int i = 0; i < CH / 2; ++i) v[i] = mul2(v[i], gelu_deriv2(bf16x2_to_f32x2(hw[i]), true));
        } else {
#pragma unroll
            for (int i = 0; i < CH / 2; ++i) v[i] = mul2(v[i], gelu_deriv2(bf16x2_to_f32x2(hw[i]), false));
        }
    }
#pragma unroll
    for (int i = 0; i < CH / 2; ++i) w[i] = f32x2_to_bf16x2(v[i]);
    out(w, 0);
    if (EPI == EPI_DGELU) {
#pragma unroll
        for (int i = 0; i < CH / 2; ++i) w[i] = f32x2_to_bf16x2(fma2(bf16x2_to_f32x2(w[i]), pk2(-1.0f), v[i]));
        out(w, 1);
    }
    if (EPI == EPI_GELU) {
        if (tanh_form) {
#pragma unroll
            for (int i = 0; i < CH / 2; ++i) w[i] = f32x2_to_bf16x2(gelu2(v[i], true));
        } else {
#pragma unroll
            for (int i = 0; i < CH / 2; ++i) w[i] = f32x2_to_bf16x2(gelu2(v[i], false));
        }
        out(w, 1);
    }
}

// Row mode runs a last wave in halves of its tiles; not dA + GELU', whose prefetch
// of H needs fixed bounds (with run-time ones it spills: 269 -> 344 us at the 6-task
// ViT-B step), and not 192 columns, whose half is not a whole number of 64-column boxes.
constexpr bool cuts_last_wave(int bn, int mode, int epi) {
    return mode == MODE_ROW && epi != EPI_DGELU && bn != 192;
}

template <int BN, int MODE, bool A_MN, bool B_MN, int EPI>
__global__ void __launch_bounds__(Roles<MODE, EPI>::NT, 1)
grouped_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmD, const __grid_constant__ CUtensorMap tmD2,
                    const __grid_constant__ TailMaps tmAt, Args args) {
    using S = Shape<BN, MODE, EPI>;
    constexpr int STAGES = S::STAGES;
    constexpr int NT = S::NT;
    constexpr uint32_t IDESC = idesc_bf16(BM, BN, A_MN, B_MN);
    constexpr bool CUT = cuts_last_wave(BN, MODE, EPI);

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (raw_addr & 1023u)) & 1023u);
    const uint32_t tiles_addr = smem_u32(smem);
    uint8_t *epi_base = smem + STAGES * S::STAGE_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(epi_base + S::EPI_BYTES);
    int *misc = reinterpret_cast<int *>(bars + S::NUM_BARS);  // [0] tmem base, [1] abort, [2] total
    int *scan_tmp = misc + 4;
    int *prefix = scan_tmp + NT;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar_full = [&](int s) { return smem_u32(bars + s); };
    auto bar_empty = [&](int s) { return smem_u32(bars + STAGES + s); };
    auto bar_tfull = [&](int a) { return smem_u32(bars + 2 * STAGES + a); };
    auto bar_tempty = [&](int a) { return smem_u32(bars + 2 * STAGES + 2 + a); };
    const uint32_t bar_drain = smem_u32(bars + 2 * STAGES + 4);
    volatile int *abort_flag = misc + 1;
    int total = 0;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full(s), 2);  // the A and the B producer's arrivals
            mbar_init(bar_empty(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull(a), 1);
            mbar_init(bar_tempty(a), Roles<MODE, EPI>::EW);
        }
        mbar_init(bar_drain, 1);
        misc[1] = 0;
        fence_barrier_init();
        fence_proxy_async();
        prefetch_map(&tmA);
        prefetch_map(&tmB);
        if (MODE == MODE_ROW)
            for (int i = 0; i < 3; ++i) prefetch_map(&tmAt.a[i]);
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(misc), S::TMEM_COLS);
        tmem_relinquish();
    }
    // the predecessor's outputs (loads, operands) are complete from here on
    if (MODE == MODE_WGRAD) wait_for_predecessor(args, false);
    else pdl_wait();

    // Tile count (and, in row mode, the per-group tile prefix).
    if (MODE == MODE_ROW) {
        const int G = args.G;
        const int per = (G + NT - 1) / NT;
        const int g0 = min(G, tid * per), g1 = min(G, g0 + per);
        int local = 0;
        for (int g = g0; g < g1; ++g) {
            int L = __ldg(args.load + real_group(args, g));
            L = L < 0 ? 0 : (L > args.C ? args.C : L);
            local += ((L + BM - 1) / BM) * args.tiles_n;
        }
        scan_tmp[tid] = local;
        __syncthreads();
        if (warp == 0) {  // exclusive scan of NT partials, NT/32 per lane
            constexpr int PER = NT / 32;
            int v[PER], s = 0;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                v[i] = scan_tmp[lane * PER + i];
                s += v[i];
            }
            int incl = s;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            int run = incl - s;
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                scan_tmp[lane * PER + i] = run;
                run += v[i];
            }
            if (lane == 31) misc[2] = incl;
        }
        __syncthreads();
        int run = scan_tmp[tid];
        for (int g = g0; g < g1; ++g) {
            prefix[g] = run;
            int L = __ldg(args.load + real_group(args, g));
            L = L < 0 ? 0 : (L > args.C ? args.C : L);
            run += ((L + BM - 1) / BM) * args.tiles_n;
        }
        if (tid == 0) prefix[G] = misc[2];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    total = (MODE == MODE_ROW) ? misc[2] : args.G * args.tiles_m * args.tiles_n;
    // Row mode: a last wave that fills at most half of the SMs is cut into tiles of
    // half the columns, so that it ends sooner; no element's sums change.  One
    // image through a ViT-S layer (48 and 24 tiles) 32.8 -> 30.3 us, attention at C
    // 247 1134 -> 1129.  Quarters, which would also shorten fuller last waves, cost
    // more than they gave (6-task ViT-B, FC2 201 -> 222 us).
    int wide = total, cut = 0;
    if (CUT) {
        const int rem = total % (int)gridDim.x;
        if (rem > 0 && 2 * rem <= (int)gridDim.x) {
            cut = 1;
            wide = total - rem;
            total += rem;
        }
    }
    const uint32_t tmem_base = (uint32_t)misc[0];

    if (warp == 0 || warp == Roles<MODE, EPI>::EW + 2) {
        // ------------------------------------------------------------ producers: A (warp 0), B (the last warp)
        // One thread each: a copy's wait, expected bytes and issue take it a few
        // hundred cycles, as long as the MMAs of a k-block, so A and B have their own.
        if (elect_one()) {
            const bool isA = warp == 0;
            int stage = 0;
            uint32_t phase = 0;
            int issued = 0;  // copies so far: slot s has had those of index s, s + STAGES, ...
            bool ok = true;
            const bool cmpa = (args.compact & CMP_A) != 0, cmpb = (args.compact & CMP_B) != 0;
            Tile t = decode_tile<MODE, BN, CUT>(args, prefix, blockIdx.x < total ? blockIdx.x : 0, wide, cut);
            for (int u = blockIdx.x; u < total && ok; u += gridDim.x) {
                Tile tn = t;  // the next tile, looked up behind this one's first copy
                const bool last = u + (int)gridDim.x >= total;
                if (isA && last) pdl_launch_dependents();  // this CTA's last tile
                // Row mode, A rows [0, rn): the tile's valid rows rounded up to 16.  The
                // slot's rows past rn keep stale data, which only reaches output rows
                // past rows_valid -- never stored.
                const int rem_rows = t.rows_valid - t.m_blk * BM;
                const int rn = MODE != MODE_ROW || rem_rows >= BM ? BM : ((rem_rows + 15) & ~15);
                const int r0 = (cmpa ? t.crow : 0) + t.m_blk * BM, gz = cmpa ? 0 : t.gr;
                const int bn = CUT ? t.bn : BN;
                const uint32_t bytes = isA ? (uint32_t)rn * (BK * 2) : (uint32_t)bn * (BK * 2);
                // Weight gradients: the first K row of k-block 0 (<= 0, see below)
                const int k0 = t.kvalid - t.khalf * BK;
                for (int kb = 0; kb < t.kblocks; ++kb) {
                    if (!wait_phase(bar_empty(stage), phase ^ 1u, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = tiles_addr + stage * S::STAGE_BYTES;
                    const uint32_t sb = sa + S::A_BYTES;
                    const uint32_t fb = bar_full(stage);
                    mbar_expect_tx(fb, bytes);
                    if (MODE == MODE_ROW) {
                        if (isA) {
                            if (rn == BM) {
                                tma_load_3d(sa, &tmA, fb, kb * BK, r0, gz);
                            } else {
                                int off = 0;
                                if (rn & 64) {
                                    tma_load_3d(sa, &tmAt.a[0], fb, kb * BK, r0, gz);
                                    off = 64;
                                }
                                if (rn & 32) {
                                    tma_load_3d(sa + off * (BK * 2), &tmAt.a[1], fb, kb * BK, r0 + off, gz);
                                    off += 32;
                                }
                                if (rn & 16)
                                    tma_load_3d(sa + off * (BK * 2), &tmAt.a[2], fb, kb * BK, r0 + off, gz);
                            }
                        } else if (CUT && bn != BN) {  // tmD: B's map with boxes of 64 columns
                            for (int c = 0; c < bn; c += 64) {
                                if (B_MN) tma_load_4d(sb + c * (BK * 2), &tmD, fb, 0, kb * BK, (t.col0 + c) / 64, t.gr);
                                else tma_load_3d(sb + c * (BK * 2), &tmD, fb, kb * BK, t.col0 + c, t.gr);
                            }
                        } else if (B_MN) {  // one 4-D box: BN/64 column chunks of 64 rows
                            tma_load_4d(sb, &tmB, fb, 0, kb * BK, t.n_blk * (BN / 64), t.gr);
                        } else {
                            tma_load_3d(sb, &tmB, fb, kb * BK, t.n_blk * BN, t.gr);
                        }
                    } else {
                        // K = the group's rows, in k-blocks that end at its last row: only
                        // k-block 0 is partial, and its missing rows lie before row 0, where
                        // the tensor maps read zeros (in a compact B they are a neighbour's,
                        // and the MMA warp zeroes them).  With ksplit every other k-block
                        // pairs the same A rows with B's residual rows: the order of sums of
                        // the SM-pair kernels.
                        const int hi = args.ksplit ? kb & 1 : 0;
                        const int ka = k0 + (kb >> args.ksplit) * BK;
                        if (isA)
                            tma_load_4d(sa, &tmA, fb, 0, ka, t.m_blk * (BM / 64), t.gr);
                        else if (cmpb)  // residual rows follow the entry's load rows
                            tma_load_4d(sb, &tmB, fb, 0, t.crow + hi * t.kvalid + ka, t.n_blk * (BN / 64), 0);
                        else
                            tma_load_4d(sb, hi ? &tmD2 : &tmB, fb, 0, ka, t.n_blk * (BN / 64), t.gr);
                    }
                    if (kb == 0 && !last) tn = decode_tile<MODE, BN, CUT>(args, prefix, u + gridDim.x, wide, cut);
                    ++issued;
                    if (++stage == STAGES) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (t.kblocks == 0 && !last) tn = decode_tile<MODE, BN, CUT>(args, prefix, u + gridDim.x, wide, cut);
                t = tn;
            }
            if (*abort_flag) {  // let copies in flight land before the CTA exits
                int dummy = 0;
                for (int s = 0; s < STAGES && s < issued; ++s) {
                    const uint32_t last = (uint32_t)(((issued - 1 - s) / STAGES) & 1);
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(bar_full(s), last) && global_ns() - t0 < 100000000ull) ++dummy;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        int stage = 0;
        uint32_t phase = 0;
        int it = 0;
        bool ok = true;
        const bool cmpb = MODE == MODE_WGRAD && (args.compact & CMP_B) != 0;
        const uint32_t idesc_cut = idesc_bf16(BM, BN >> cut, A_MN, B_MN);
        const bool one = elect_one();
        // Waits for slot `stage` and issues its MMAs from 16-row step k0 on.
        auto k_block = [&](uint32_t dtmem, int k0, bool accumulate, uint32_t idesc) {
            const uint32_t sa = tiles_addr + stage * S::STAGE_BYTES;
            const uint64_t da = operand_desc(sa, 0, A_MN), db = operand_desc(sa + S::A_BYTES, 0, B_MN);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
                if (MODE == MODE_ROW || kk >= k0)
                    mma_bf16(dtmem, desc_step(da, kk, A_MN), desc_step(db, kk, B_MN), idesc,
                             accumulate || kk > k0 ? 1u : 0u);
            mma_commit(bar_empty(stage));
        };
        auto next_stage = [&]() {
            if (++stage == STAGES) {
                stage = 0;
                phase ^= 1u;
            }
        };
        if (!cmpb) {
            for (int u = blockIdx.x; one && u < total && ok; u += gridDim.x, ++it) {
                int kblocks = args.K_fixed / BK, skip = 0;
                if (MODE == MODE_WGRAD) {
                    const Tile t = decode_tile<MODE, BN, CUT>(args, prefix, u, wide, cut);
                    kblocks = t.kblocks;
                    skip = (t.khalf * BK - t.kvalid) >> 4;  // all-zero 16-row steps of k-block 0
                }
                const int acc = it & 1;
                if (!wait_phase(bar_tempty(acc), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag, args.status)) break;
                tc_fence_after();
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!wait_phase(bar_full(stage), phase, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    k_block(tmem_base + (uint32_t)(acc * BN), (kb >> args.ksplit) == 0 ? skip : 0, kb > 0,
                            !CUT || u < wide ? IDESC : idesc_cut);
                    next_stage();
                }
                if (!ok) break;
                if (kblocks == 0) mbar_arrive(bar_tfull(acc));
                else mma_commit(bar_tfull(acc));
            }
        } else {  // compact B: the warp zeroes the rows of k-block 0 (both parts) that belong to a neighbour
            for (int u = blockIdx.x; u < total && ok; u += gridDim.x, ++it) {
                const Tile t = decode_tile<MODE, BN, CUT>(args, prefix, u, wide, cut);
                const int z = t.khalf * BK - t.kvalid;
                const int acc = it & 1;
                if (!wait_phase(bar_tempty(acc), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag, args.status)) break;
                tc_fence_after();
                for (int kb = 0; kb < t.kblocks; ++kb) {
                    if (!wait_phase(bar_full(stage), phase, abort_flag, args.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const bool first = (kb >> args.ksplit) == 0;
                    if (first && z > 0) {
                        uint8_t *tile = smem + stage * S::STAGE_BYTES + S::A_BYTES;
                        for (int i = lane; i < (BN / 64) * z * 8; i += 32) {
                            const int c = i / (z * 8), w = i - c * z * 8;
                            *reinterpret_cast<uint4 *>(tile + c * (BK * 128) + (w >> 3) * 128 + (w & 7) * 16) =
                                make_uint4(0, 0, 0, 0);
                        }
                        fence_proxy_async();
                    }
                    __syncwarp();
                    if (one) k_block(tmem_base + (uint32_t)(acc * BN), first ? z >> 4 : 0, kb > 0, IDESC);
                    __syncwarp();
                    next_stage();
                }
                if (!ok) break;
                if (one) {
                    if (t.kblocks == 0) mbar_arrive(bar_tfull(acc));
                    else mma_commit(bar_tfull(acc));
                }
                __syncwarp();
            }
        }
        __syncwarp();
        if (one) {  // all MMAs of this CTA complete before TMEM is freed
            mma_commit(bar_drain);
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(bar_drain, 0) && global_ns() - t0 < 1000000000ull) {
            }
        }
        __syncwarp();
    } else if constexpr (MODE == MODE_WGRAD) {
        // ------------------------------------------------------------ epilogue (weight gradients)
        // Every tile is full.  Each warp reads all BN/2 accumulator columns of its
        // 32 rows with back-to-back tcgen05.ld before one wait, then writes 64-
        // column chunks into a 128-byte-swizzled 32 x 64 staging tile that one
        // lane stores with a TMA bulk tensor store (two tiles alternate).
        const int ew = warp - 2;
        const int q = warp & 3;
        const int half = ew >> 2;
        constexpr int COLS = BN / 2;
        uint8_t *stg = epi_base + ew * EPI_WARP_BYTES_TMA;
        const uint64_t policy = evict_first_policy();
        int nstore = 0;
        int it = 0;
        bool zeroed = false;  // the first staging tile holds zeros that copies in flight read
        for (int u = blockIdx.x; u < total; u += gridDim.x, ++it) {
            const Tile t = decode_tile<MODE, BN, CUT>(args, prefix, u, wide, cut);
            const int acc = it & 1;
            const uint32_t aph = (uint32_t)((it >> 1) & 1);
            if (!wait_phase(bar_tfull(acc), aph, abort_flag, args.status)) break;
            tc_fence_after();
            if (t.kblocks == 0) {
                zero_staging(stg, zeroed);
                if (lane == 0) {
                    mbar_arrive(bar_tempty(acc));
                    const int parts = args.tiles_m * args.tiles_n;
                    store_zeros(reinterpret_cast<uint8_t *>(args.D + (long long)t.gr * args.sD), args.sD * 2,
                                t.m_blk * args.tiles_n + t.n_blk, parts, ew, 8, smem_u32(stg), policy);
                }
                continue;
            }
            if (zeroed) {
                if (lane == 0) bulk_wait_read0();
                zeroed = false;
            }
            const int row0 = t.m_blk * BM + q * 32;
            const int colw = t.n_blk * BN + half * COLS;
            const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) +
                                  (uint32_t)(acc * BN + half * COLS);
            uint32_t r[COLS / 32][32];
#pragma unroll
            for (int i = 0; i < COLS / 32; ++i) tmem_ld32(trow + i * 32, r[i]);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(acc));  // the accumulator is in registers now
            store_columns<COLS / 64, 2>(tmD, r, stg, nstore, colw, row0, t.gr, policy);
        }
        if (lane == 0) bulk_wait_all();
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue (row mode, st.global)
        // Warps 2 .. EW+1.  Warp w works on TMEM lane quarter q = w & 3 (rows
        // 32q .. 32q+31 of the tile), each thread owning one row; the EW / 4
        // warps of a quarter take the tile's CH-column chunks in turn (warp j:
        // chunks j, j + EW/4, ...).  Per chunk: tcgen05.ld, the fused
        // elementwise step, bf16 packing into a per-warp staging tile, and
        // coalesced, row-masked 16-byte stores.
        constexpr int EW = Roles<MODE, EPI>::EW;
        constexpr int WPQ = EW / 4;                 // warps per lane quarter
        constexpr int CH = ROW_CH;                  // columns per chunk
        constexpr int PITCH = Roles<MODE, EPI>::PITCH;   // staging row pitch (bytes)
        constexpr int PIECES = CH * 2 / 16;         // 16-byte pieces of a staged row
        constexpr int RPI = 32 / PIECES;            // rows per store instruction
        const int ew = warp - 2;
        const int q = warp & 3;
        const int jw = ew >> 2;
        uint8_t *stg = epi_base + ew * 32 * PITCH;
        const bool tanh_form = args.gelu_tanh != 0;
        const int sub_r = lane / PIECES, sub_c = lane % PIECES;  // row-store mapping
        // EPI_DGELU: the H values of this thread's row for the current chunk,
        // loaded one chunk ahead (and across tiles) so the epilogue never waits
        // on a fresh global load.
        uint4 hcur[CH / 8], hnxt[CH / 8];
        auto load_h = [&](const Tile &tl, int c, uint4 (&dst)[CH / 8]) {
            const int r0 = tl.m_blk * BM + q * 32;
            if (r0 + lane < tl.rows_valid) {
                const uint4 *src = reinterpret_cast<const uint4 *>(
                    args.aux + (long long)tl.gr * args.sAux + (long long)(r0 + lane) * args.ldd +
                    tl.n_blk * BN + c * CH);
#pragma unroll
                for (int i = 0; i < CH / 8; ++i) dst[i] = __ldg(src + i);
            } else {
#pragma unroll
                for (int i = 0; i < CH / 8; ++i) dst[i] = make_uint4(0, 0, 0, 0);
            }
        };
        // Stage 32 packed rows of this warp and store them coalesced, masked to
        // the valid rows.
        auto store_rows = [&](__nv_bfloat16 *base, int nvalid) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < PIECES; ++i) {
                const int r = i * RPI + sub_r;
                if (r < nvalid)
                    *reinterpret_cast<uint4 *>(base + (long long)r * args.ldd + sub_c * 8) =
                        *reinterpret_cast<const uint4 *>(stg + r * PITCH + sub_c * 16);
            }
            __syncwarp();
        };
        auto stage = [&](const uint32_t(&w)[CH / 2]) {
#pragma unroll
            for (int i = 0; i < CH / 8; ++i)
                *reinterpret_cast<uint4 *>(stg + lane * PITCH + i * 16) =
                    make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
        };
        int it = 0;
        Tile t = decode_tile<MODE, BN, CUT>(args, prefix, blockIdx.x < total ? blockIdx.x : 0, wide, cut);
        if (EPI == EPI_DGELU && blockIdx.x < total) load_h(t, jw, hcur);
        for (int u = blockIdx.x; u < total; u += gridDim.x, ++it) {
            const bool have_next = u + (int)gridDim.x < total;
            const Tile tn = decode_tile<MODE, BN, CUT>(args, prefix, have_next ? u + gridDim.x : u, wide, cut);
            const int acc = it & 1;
            const uint32_t aph = (uint32_t)((it >> 1) & 1);
            if (!wait_phase(bar_tfull(acc), aph, abort_flag, args.status)) break;
            tc_fence_after();
            const int row0 = t.m_blk * BM + q * 32;  // this warp's first row in the group
            int nvalid = t.rows_valid - row0;
            nvalid = nvalid < 0 ? 0 : (nvalid > 32 ? 32 : nvalid);
            // compact output: the entry's rows from crow, its second output (the
            // residual) after its load rows; else the group's slab
            const bool cmpd = (args.compact & CMP_D) != 0;
            const long long gofs = (cmpd ? (long long)t.crow * args.ldd : (long long)t.gr * args.sD) +
                                   (long long)row0 * args.ldd + (CUT ? t.col0 : t.n_blk * BN);
            const long long gofs2 = cmpd ? gofs + (long long)t.rows_valid * args.ldd : gofs;
            const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
            const int nch = (CUT ? t.bn : BN) / CH;  // chunks of this tile's rows
#pragma unroll 1
            for (int c = jw; c < nch; c += WPQ) {
                if (EPI == EPI_DGELU) {
                    if (c + WPQ < nch) load_h(t, c + WPQ, hnxt);
                    else if (have_next) load_h(tn, jw, hnxt);
                }
                if (nvalid > 0) {
                    f32x2 v[CH / 2];
                    if (t.kblocks > 0) {
                        uint32_t r[CH];
                        tmem_ld32(trow + c * CH, r);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < CH / 2; ++i)
                            v[i] = pk2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
                    } else {
#pragma unroll
                        for (int i = 0; i < CH / 2; ++i) v[i] = pk2(0.0f);
                    }
                    epilogue_chunk<EPI, CH>(v, hcur, tanh_form, [&](const uint32_t(&w)[CH / 2], int out) {
                        stage(w);
                        
                        store_rows(out == 0 ? args.D + gofs + c * CH : args.D2 + gofs2 + c * CH, nvalid);
                    });
                }
                if (EPI == EPI_DGELU) {
#pragma unroll
                    for (int i = 0; i < CH / 8; ++i) hcur[i] = hnxt[i];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty(acc));
            t = tn;
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem_base, S::TMEM_COLS);
    if (MODE == MODE_WGRAD) wait_for_predecessor(args, true);
}

// ---------------------------------------------------------------------------
// Host side.

// Encodes a rank-3 bf16 tensor map {inner, mid, outer} (inner contiguous) with
// a {64, box_mid, 1} box and 128-byte swizzle; out-of-range elements read 0.
bool make_map(CUtensorMap *map, const void *base, uint64_t inner, uint64_t mid, uint64_t outer,
              uint32_t box_mid, uint64_t outer_stride_elems = 0);

// Encodes a rank-4 view of a [outer][rows][mn] bf16 tensor whose mn axis is cut
// into 64-element chunks: dims {64, rows, mn/64, outer}.  A {64, box_rows,
// box_chunks, 1} box then lands in shared memory chunk-major -- box_chunks
// tiles of box_rows x 128 bytes (128-byte swizzle) -- which is the MN-major
// operand layout, in one copy instead of one per chunk.
// outer_stride_elems: elements from one outer index to the next (0: rows x mn).
bool make_map_chunked(CUtensorMap *map, const void *base, uint64_t mn, uint64_t rows,
                      uint64_t outer, uint32_t box_rows, uint32_t box_chunks,
                      uint64_t outer_stride_elems = 0);

template <int BN, int MODE, bool A_MN, bool B_MN, int EPI>
int launch(const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &md,
           const CUtensorMap &md2, const TailMaps &mat, const Args &a, long long max_tiles,
           cudaStream_t s, const char *name) {
    using S = Shape<BN, MODE, EPI>;
    auto kern = grouped_gemm_kernel<BN, MODE, A_MN, B_MN, EPI>;
    static std::atomic<int> smem_limit[64];
    if (const int st = raise_smem_limit((const void *)kern, smem_limit, (int)S::SMEM_BYTES)) return st;
    if (max_tiles <= 0) return VMOE_OK;
    // every tile may be cut in two
    const long long most = cuts_last_wave(BN, MODE, EPI) ? 2 * max_tiles : max_tiles;
    const long long grid = most < num_sms() ? most : num_sms();
    trace_before(s, name);
    const int st = launch_kernel(kern, dim3((unsigned)grid), dim3(S::NT), S::SMEM_BYTES, s, ma, mb,
                                 md, md2, mat, a);
    trace_after(s);
    return st;
}

// A slice of the groups for one launch (the memory-budgeted backward): n
// entries, entry i = group glist[i]; the operands flagged in `compact` live in
// a compact buffer of `rows` rows, entry i's rows from crow[i].  n == 0: all
// groups, nothing compact.
struct Slice {
    const int32_t *glist = nullptr;  // device
    const int32_t *crow = nullptr;   // device
    int n = 0;
    int compact = 0;
    long long rows = 0;
};

inline Args base_args(const Dims &p, const int32_t *load) {
    Args a = {};
    a.G = p.G();
    a.C = p.C;
    a.load = load;
    a.gelu_tanh = (p.flags & VMOE_GELU_TANH) != 0;
    a.status = device_status_word();
    return a;
}

}  // namespace tc
}  // namespace vmoe

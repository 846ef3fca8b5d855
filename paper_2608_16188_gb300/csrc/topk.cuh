// topk.cuh -- softmax + top-k gating of one token's logit row (Section 2.1
// routing), shared by the router kernels (internal).
#pragma once

#include <math.h>

#include "common.cuh"

namespace vmoe {

// One token: the max, the softmax denominator, then k picks, each the best
// expert that comes after the previous pick in the order (larger logit first,
// equal logits by lower index).  NaN is treated as -inf so the chosen indices
// stay in range.  Writes idx and gate of token `tok` (= t * N + n); the gates
// are renormalised over the k picks unless VMOE_NO_RENORM.
__device__ __forceinline__ void topk_row(const Dims &p, const float *row, long long tok,
                                         int32_t *__restrict__ out_idx,
                                         float *__restrict__ out_gate) {
    const int E = p.E;
    const bool renorm = !(p.flags & VMOE_NO_RENORM);
    float mx = -INFINITY;
    for (int e = 0; e < E; ++e) {
        float v = row[e];
        mx = fmaxf(mx, isnan(v) ? -INFINITY : v);
    }
    float sum = 0.0f;
    for (int e = 0; e < E; ++e) {
        float v = row[e];
        sum += expf((isnan(v) ? -INFINITY : v) - mx);
    }
    float ev[8];
    int ei[8];
    float pv = INFINITY;  // previous pick: (pv, pe); the next pick comes after it
    int pe = -1;
    float kept = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        ev[j] = 0.0f;
        ei[j] = 0;
        if (j >= p.k) continue;
        float bv = -INFINITY;
        int be = -1;
        for (int e = 0; e < E; ++e) {
            float v = row[e];
            v = isnan(v) ? -INFINITY : v;
            const bool after = v < pv || (v == pv && e > pe);
            if (after && (be < 0 || v > bv)) {  // strict '>' keeps the lower index on ties
                bv = v;
                be = e;
            }
        }
        ei[j] = be;
        ev[j] = expf(bv - mx);
        kept += ev[j];
        pv = bv;
        pe = be;
    }
    const long long base = tok * p.k;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (j < p.k) {
            out_idx[base + j] = ei[j];
            out_gate[base + j] = renorm ? ev[j] / kept : ev[j] / sum;
        }
}

// The same row by a whole warp, lane l holding the logits of experts l, l + 32,
// ... (E <= 256): a few hundred cycles of shuffles instead of a thread's k + 2
// passes over the row, where a CTA has few rows.
__device__ __forceinline__ void topk_row_warp(const Dims &p, const float *row, long long tok,
                                              int32_t *__restrict__ out_idx, float *__restrict__ out_gate) {
    constexpr int M = 8;  // 256 / 32
    const int E = p.E, lane = threadIdx.x & 31;
    float v[M], mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const int e = lane + 32 * i;
        const float x = e < E ? row[e] : -INFINITY;
        v[i] = isnan(x) ? -INFINITY : x;
        mx = fmaxf(mx, v[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sum = 0.0f;
#pragma unroll
    for (int i = 0; i < M; ++i)
        if (lane + 32 * i < E) sum += expf(v[i] - mx);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    unsigned taken = 0;  // this lane's logits already picked
    float mine = 0.0f, kept = 0.0f;
    int my_e = 0;
    for (int j = 0; j < p.k; ++j) {
        // the largest logit left, the lowest expert among equals
        float bv = -INFINITY;
        int be = 1 << 30;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int e = lane + 32 * i;
            if (e < E && !((taken >> i) & 1u) && (be == 1 << 30 || v[i] > bv)) {
                bv = v[i];
                be = e;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oe = __shfl_xor_sync(0xffffffffu, be, o);
            // a lane with nothing left carries be = 2^30, which loses to any expert at -inf
            if (ov > bv || (ov == bv && oe < be)) {
                bv = ov;
                be = oe;
            }
        }
        if ((be & 31) == lane) taken |= 1u << (be >> 5);
        const float ev = expf(bv - mx);
        kept += ev;
        if (lane == j) {
            mine = ev;
            my_e = be;
        }
    }
    if (lane < p.k) {
        out_idx[tok * p.k + lane] = my_e;
        out_gate[tok * p.k + lane] = (p.flags & VMOE_NO_RENORM) ? mine / sum : mine / kept;
    }
}

}  // namespace vmoe

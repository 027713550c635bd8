// Small jobs that run in blocks of their own beside the tile blocks of the preparation launch (or, without steering, in a
// launch of their own): item table of packed batches, fp32 -> bf16 copies of the inputs.
#pragma once

#include "seka_common.cuh"

namespace seka {

constexpr int PREP_THREADS = 256;

// fp32 -> bf16 copies of Q, K and V (groups of four values; the three tensors one after another)
struct ConvertArgs { const float4* in[3]; uint2* out[3]; size_t n4[3]; };

// where the steering of a (sequence, KV head) comes from; gain null: nothing is steered
struct SteerIn { const float* gain; const float* alpha; const uint8_t* head_enable; int M; int routed; };

#ifdef __CUDACC__

// bit 0: the keys of this (sequence, KV head) are edited; bit 1: the fused kernel multiplies their low parts too
// (routed coefficients are not looked at: Eq. 6 normalises them to a largest magnitude of 1)
__device__ __forceinline__ int steer_byte(const SteerIn& s, int b, int h, int Hkv) {
    if (s.gain == nullptr) return 0;
    const float g = s.gain[b];
    const bool on = g != 0.f && (s.head_enable == nullptr || s.head_enable[h] != 0);
    const float amax = s.routed ? 1.f : alpha_max_of(s.alpha, (size_t)b * Hkv + h, s.M);
    return (on ? 1 : 0) | ((on && lo_needed(g, amax)) ? 2 : 0);
}

// One of `n_blocks` blocks that share the conversion; four 16-byte loads of a thread are in flight together.
__device__ __noinline__ static void convert_block(const ConvertArgs& a, int block, int n_blocks) {
    const size_t step = (size_t)n_blocks * blockDim.x;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        for (size_t i0 = (size_t)block * blockDim.x + threadIdx.x; i0 < a.n4[t]; i0 += 4 * step) {
            float4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q * step < a.n4[t]) v[q] = __ldcs(a.in[t] + i0 + q * step);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q * step < a.n4[t]) a.out[t][i0 + q * step] = make_uint2(pack_bf16(v[q].x, v[q].y), pack_bf16(v[q].z, v[q].w));
        }
    }
}

// Item table of the fused kernel for packed variable-length batches: the items of decode_item whose tiles lie beyond
// their sequence are dropped, order kept.  One block per row slot (block 0: the last, heaviest row); where a block's
// items start follows from the sequence lengths alone, so the blocks do not talk to each other: a sequence of n_t row
// tiles has R = n_t (tiles A and B are two heads) or ceil(n_t / 2) (two row tiles) row slots, row slot `row` keeps the
// sequences with R > row, and the rows before it in the table hold hs * sum_b max(0, R_b - row - 1) items.
__device__ __noinline__ static void items_block(const Sched& sc, const int* __restrict__ cu, const SteerIn& steer,
                                                ItemRecord* __restrict__ items, int* __restrict__ count, int block) {
    constexpr int NW = PREP_THREADS / 32;
    __shared__ long long red_s[2][NW];
    __shared__ int pre_s[PREP_THREADS];
    __shared__ int warp_tot[NW];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int row = sc.rs - 1 - block;
    auto rows_of = [&](int b) -> int {
        const int n_t = (cu[b + 1] - cu[b] + 127) / 128;
        return sc.pair_heads ? n_t : (n_t + 1) / 2;
    };
    // items of the rows above this one (they come first), and, in block 0, of all rows
    long long before = 0, all = 0;
    for (int b = tid; b < sc.B; b += PREP_THREADS) {
        const int R = rows_of(b);
        before += R > row + 1 ? R - row - 1 : 0;
        all += R;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if (lane == 0) { red_s[0][wid] = before; red_s[1][wid] = all; }
    __syncthreads();
    long long base = 0, total = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) { base += red_s[0][q]; total += red_s[1][q]; }
    base *= sc.hs;
    if (block == 0 && tid == 0) *count = (int)(total * sc.hs);
    // this row: the sequences that reach it, a block's worth at a time, keep their order
    for (int b0 = 0; b0 < sc.B; b0 += PREP_THREADS) {
        const int b = b0 + tid;
        const bool keep = b < sc.B && rows_of(b) > row;
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) warp_tot[wid] = __popc(bal);
        __syncthreads();
        int off = 0, tot = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) { if (q < wid) off += warp_tot[q]; tot += warp_tot[q]; }
        pre_s[tid] = keep ? off + __popc(bal & ((1u << lane) - 1)) : -1;
        __syncthreads();
        const int n_b = sc.B - b0 < PREP_THREADS ? sc.B - b0 : PREP_THREADS;
        for (int c = tid; c < n_b * sc.hs; c += PREP_THREADS) {
            const int bi = c / sc.hs, slot = c - bi * sc.hs;
            const int pos = pre_s[bi];
            if (pos < 0) continue;
            ItemRecord r;
            decode_item(sc, (long long)block * sc.per + (long long)(b0 + bi) * sc.hs + slot, cu, r);
            r.steer = steer_byte(steer, r.bh & 0xffff, r.bh >> 16, sc.Hkv);
            items[base + (long long)pos * sc.hs + slot] = r;
        }
        base += (long long)tot * sc.hs;
        __syncthreads();
    }
}

#endif  // __CUDACC__

}  // namespace seka

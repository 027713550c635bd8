// Offline spectral learning of the projections (Section 3.1, Eq. 2-3, first loop of Algorithm 1) and the
// head-selection distance of Section 3.4, for all (layer, KV head) slots of a model in one call.
//
//   learn_cov_kernel      Omega+ = h^T h+ / n and Omega- = h^T h- / n.  The contraction runs over tokens, so the
//                         key embeddings are read exactly once (three bf16 tensors [n, slots, d]); at 2 d / 3 FLOP
//                         per byte the pass is bound by HBM bandwidth but needs the tensor cores to keep up.
//                         Persistent CTAs, an item = (group of 128 columns, chunk of tokens): a producer warp
//                         streams 128-token tiles of h, h+, h- with TMA through two stages; one thread issues
//                         tcgen05 products with BOTH operands MN-major (the token axis is the contraction) into two
//                         128 x 128 accumulators in tensor memory; four warps drain the finished accumulators of
//                         item i while item i + 1 accumulates in the other half of tensor memory; four more warps
//                         sum ||h+ - h-||_2 over the answer tokens from the same staged tiles.
//   learn_reduce_kernel   sums the per-chunk partials in chunk order, scales by 1 / n; D = mean of the distances.
//   learn_svd_kernel      one CTA per matrix, fp64: QR of Omega^T, then one-sided Jacobi (Hestenes) on the columns of R^T;
//                         half of the columns in registers, half in shared memory; every pair of columns meets once per
//                         sweep (ordering by recursive halving); on convergence the column norms are the singular
//                         values and the normalised columns the left singular vectors; sorted descending; the rank of
//                         Eq. 3 from the sorted values.
#include <math.h>

#include "seka_kernels.h"

namespace seka {
namespace {

// ------------------------------------------------------------------------------------ cross-covariances
constexpr int LC_THREADS = 320;                 // warp 0 producer, warp 1 MMA issuer, warps 2..5 drain, warps 6..9 distances
constexpr int LC_TOK = 128;                     // tokens per stage
constexpr int LC_NS = 2;
constexpr uint32_t LC_BLK = 128 * 128;          // [128 tokens x 64 columns] block, 128-byte swizzle
constexpr uint32_t LC_TILE = 2 * LC_BLK;        // 128 columns of one tensor
constexpr uint32_t LC_STAGE = 3 * LC_TILE;      // h, h+, h-
constexpr uint32_t LC_BARS = LC_NS * LC_STAGE;  // full[2], empty[2], acc_full[2], acc_free[2]
constexpr uint32_t LC_MISC = LC_BARS + 8 * 8;
constexpr uint32_t LC_DYN_BYTES = LC_MISC + 16 + 1024;
constexpr uint32_t LC_TMEM_COLS = 512;          // two sets of (Omega+, Omega-) accumulators

struct LearnCovParams {
    float* part;            // [n_chunks][slots][2][d][d]
    double* dist;           // [n_chunks][4][slots]: sums of the distances, one per distance warp
    int* count;             // [n_chunks][4]: answer tokens
    const uint8_t* answer;  // [n_tokens] or null: all
    int n_tokens, n_groups, d, slots, chunk_tokens, n_chunks;
    int* status;
};

__device__ __forceinline__ bool lc_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status, int where) {
    const bool ok = mbar_wait(bar, parity, abort_flag, status, where);
    return __all_sync(0xffffffffu, ok);
}

// bf16 x bf16 -> fp32, M = N = 128, A and B both MN-major (their contraction axis, the tokens, is the slow one)
constexpr uint32_t LC_IDESC = umma_idesc_bf16(128, true) | (1u << 15);

__global__ void __launch_bounds__(LC_THREADS, 1)
learn_cov_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmP,
                 const __grid_constant__ CUtensorMap tmN, const LearnCovParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + LC_BARS);
    uint64_t* full = bars;              // [2] the three tiles of a stage have landed
    uint64_t* empty = bars + 2;         // [2] the products that read the stage have finished, the four distance warps have read it
    uint64_t* acc_full = bars + 4;      // [2] every product of an item has finished: its accumulators can be read
    uint64_t* acc_free = bars + 6;      // [2] four drain-warp arrivals: the accumulators have been read
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + LC_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + LC_MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (__syncthreads_or(*reinterpret_cast<volatile int*>(p.status) != 0)) return;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 5); mbar_init(acc_full + i, 1); mbar_init(acc_free + i, 4); }
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmH); tma_prefetch_desc(&tmP); tma_prefetch_desc(&tmN);
    }
    __syncwarp();
    if (warp == 0) { tmem_alloc(tmem_holder, LC_TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    const int n_items = p.n_groups * p.n_chunks;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        uint32_t n_push = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            const int g = item % p.n_groups, c = item / p.n_groups;
            const int t0 = c * p.chunk_tokens, t1 = min(p.n_tokens, t0 + p.chunk_tokens);
            const int n_tiles = (t1 - t0 + LC_TOK - 1) / LC_TOK;
            for (int t = 0; t < n_tiles; ++t) {
                const uint32_t s = n_push % LC_NS;
                if (n_push >= LC_NS) {
                    ok = lc_wait(empty + s, ((n_push / LC_NS) - 1) & 1, abort_flag, p.status, 70);
                    if (!ok) break;
                }
                if (lane == 0) {
                    uint8_t* st = smem + s * LC_STAGE;
                    mbar_expect_tx(full + s, LC_STAGE);
                    const int row = t0 + t * LC_TOK;            // rows beyond the last token are filled with zeros
#pragma unroll
                    for (int blk = 0; blk < 2; ++blk) {
                        tma_load_3d(st + blk * LC_BLK, &tmH, full + s, blk * 64, g, row);
                        tma_load_3d(st + LC_TILE + blk * LC_BLK, &tmP, full + s, blk * 64, g, row);
                        tma_load_3d(st + 2 * LC_TILE + blk * LC_BLK, &tmN, full + s, blk * 64, g, row);
                    }
                }
                __syncwarp();
                ++n_push;
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
        const uint32_t d0 = umma_desc_lo(smem_u32(smem), LC_BLK);
        uint32_t n_pop = 0, it = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x, ++it) {
            const int c = item / p.n_groups;
            const int t0 = c * p.chunk_tokens, t1 = min(p.n_tokens, t0 + p.chunk_tokens);
            const int n_tiles = (t1 - t0 + LC_TOK - 1) / LC_TOK;
            const uint32_t set = it & 1;
            if (it >= 2) {
                ok = lc_wait(acc_free + set, ((it >> 1) - 1) & 1, abort_flag, p.status, 71);
                if (!ok) break;
            }
            for (int t = 0; t < n_tiles; ++t) {
                const uint32_t s = n_pop % LC_NS;
                ok = lc_wait(full + s, (n_pop / LC_NS) & 1, abort_flag, p.status, 72);
                if (!ok) break;
                tc_fence_after();
                if (lane == 0) {
                    const uint32_t dh = d0 + s * (LC_STAGE >> 4), dp = dh + (LC_TILE >> 4), dn = dp + (LC_TILE >> 4);
                    const uint32_t acc = tmem_base + set * 256;
#pragma unroll
                    for (int ks = 0; ks < LC_TOK / 16; ++ks) {        // 16 tokens per product: 16 rows x 128 B further on
                        const uint32_t off = (uint32_t)ks * (2048 >> 4);
                        const uint32_t accumulate = (t > 0 || ks > 0) ? 1u : 0u;
                        umma_ss(acc, dh + off, DESC_HI, dp + off, DESC_HI, LC_IDESC, accumulate);
                        umma_ss(acc + 128, dh + off, DESC_HI, dn + off, DESC_HI, LC_IDESC, accumulate);
                    }
                    umma_commit(empty + s);
                    if (t == n_tiles - 1) umma_commit(acc_full + set);
                }
                __syncwarp();
                ++n_pop;
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------ drain: accumulators -> per-chunk partials
        const int q = warp & 3;                                        // the quarter of tensor-memory lanes this warp may read
        const int row = q * 32 + lane;
        uint32_t it = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x, ++it) {
            const int g = item % p.n_groups, c = item / p.n_groups;
            const uint32_t set = it & 1;
            ok = lc_wait(acc_full + set, (it >> 1) & 1, abort_flag, p.status, 73);
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16) + set * 256;
#pragma unroll 1
            for (int sign = 0; sign < 2; ++sign) {
#pragma unroll 1
                for (int c4 = 0; c4 < 4; ++c4) {
                    float* dst;
                    if (p.d == 128) {
                        dst = p.part + ((((size_t)c * p.slots + g) * 2 + sign) * 128 + row) * 128 + c4 * 32;
                    } else {
                        // two heads of 64 columns share the product: only the diagonal blocks are cross-covariances
                        const int hd = q >> 1;
                        if ((c4 >> 1) != hd) continue;                 // the same for the whole warp
                        dst = p.part + ((((size_t)c * p.slots + 2 * g + hd) * 2 + sign) * 64 + (row & 63)) * 64 + (c4 & 1) * 32;
                    }
                    uint32_t v[32];
                    tmem_ld32(t_lane + sign * 128 + c4 * 32, v);
                    tmem_wait_ld_on(v);
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        reinterpret_cast<float4*>(dst)[e] = make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]),
                                                                        __uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3]));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free + set);
        }
    } else {
        // ------------------------------------------------------------ distances: a lane per token of the stage
        // The tiles are on chip already, so the distances cost no traffic: a pass of their own over h+ and h- took 413 us
        // beside 1031 us of products (288 slots of 128, 32k tokens, 30 % answer tokens); in here they add 56.
        const int w4 = warp - 6, row = w4 * 32 + lane, per = 128 / p.d;         // row of the stage, slots per group
        uint32_t n_pop = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
            const int g = item % p.n_groups, c = item / p.n_groups;
            const int t0 = c * p.chunk_tokens, t1 = min(p.n_tokens, t0 + p.chunk_tokens);
            const int n_tiles = (t1 - t0 + LC_TOK - 1) / LC_TOK;
            double sum0 = 0.0, sum1 = 0.0;
            int count = 0;
            for (int t = 0; t < n_tiles; ++t) {
                const uint32_t s = n_pop % LC_NS;
                const int tok = t0 + t * LC_TOK + row;
                const bool on = tok < t1 && (p.answer == nullptr || p.answer[tok] != 0);
                ok = lc_wait(full + s, (n_pop / LC_NS) & 1, abort_flag, p.status, 74);
                if (!ok) break;
                if (on) {
                    const uint8_t* hp = smem + s * LC_STAGE + LC_TILE + row * 128;
                    float ss[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
                    for (int blk = 0; blk < 2; ++blk)
#pragma unroll
                        for (int ch = 0; ch < 8; ++ch) {
                            const uint8_t* at = hp + blk * LC_BLK + ((ch ^ (row & 7)) << 4);        // 128-byte swizzle
                            const uint4 a4 = *reinterpret_cast<const uint4*>(at), b4 = *reinterpret_cast<const uint4*>(at + LC_TILE);
                            const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[e]));
                                const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[e]));
                                const float dx = a.x - b.x, dy = a.y - b.y;
                                ss[blk][0] = fmaf(dx, dx, ss[blk][0]);
                                ss[blk][1] = fmaf(dy, dy, ss[blk][1]);
                            }
                        }
                    const float q0 = ss[0][0] + ss[0][1], q1 = ss[1][0] + ss[1][1];
                    if (per == 1) {
                        sum0 += (double)sqrtf(q0 + q1);
                    } else {
                        sum0 += (double)sqrtf(q0);
                        sum1 += (double)sqrtf(q1);
                    }
                    ++count;
                }
                fence_proxy_async();            // (the reads of this stage come before the copies that refill it)
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + s);
                ++n_pop;
            }
            if (!ok) break;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sum0 += __shfl_xor_sync(0xffffffffu, sum0, o);
                sum1 += __shfl_xor_sync(0xffffffffu, sum1, o);
                count += __shfl_xor_sync(0xffffffffu, count, o);
            }
            if (lane == 0) {
                double* dst = p.dist + (size_t)(c * 4 + w4) * p.slots + g * per;
                dst[0] = sum0;
                if (per == 2) dst[1] = sum1;
                if (g == 0) p.count[c * 4 + w4] = count;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem_base, LC_TMEM_COLS);
    }
}

// omega[sign][slot][i][j] = sum over chunks (in order) of the partials, divided by the number of tokens; four entries a thread.
// The blocks after those: D[slot] = mean of the distances, a warp per slot (lane i adds the sums i, i + 32, ... in order).
// Bound by the partials' bytes: 3 chunks of 288 slots of 128 (151 MB) 110 -> 29 us (one entry a thread before).
constexpr int LR_THREADS = 256;
__global__ void __launch_bounds__(LR_THREADS)
learn_reduce_kernel(const LearnCovParams p, float* __restrict__ omega_pos, float* __restrict__ omega_neg, float* __restrict__ D,
                    unsigned n_omega_blocks, float inv_n) {
    if (blockIdx.x >= n_omega_blocks) {
        const int slot = (int)(blockIdx.x - n_omega_blocks) * (LR_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
        if (slot >= p.slots) return;
        double t = 0.0;
        int n = 0;
        for (int c = lane; c < 4 * p.n_chunks; c += 32) { t += p.dist[(size_t)c * p.slots + slot]; n += p.count[c]; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { t += __shfl_xor_sync(0xffffffffu, t, o); n += __shfl_xor_sync(0xffffffffu, n, o); }
        if (lane == 0) D[slot] = n > 0 ? (float)(t / (double)n) : 0.f;
        return;
    }
    const size_t per = (size_t)p.d * p.d / 4, total = (size_t)p.slots * 2 * per;
    const size_t idx = (size_t)blockIdx.x * LR_THREADS + threadIdx.x;
    if (idx >= total) return;
    const float4* src = reinterpret_cast<const float4*>(p.part) + idx;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int c = 0; c < p.n_chunks; ++c) {
        const float4 v = __ldcs(src + (size_t)c * total);
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    const size_t slot = idx / (2 * per), rest = idx % (2 * per);
    float* out = rest < per ? omega_pos : omega_neg;
    reinterpret_cast<float4*>(out)[slot * per + rest % per] = make_float4(acc.x * inv_n, acc.y * inv_n, acc.z * inv_n, acc.w * inv_n);
}

// ------------------------------------------------------------------------------------ SVD (QR + one-sided Jacobi, fp64)
constexpr int SV_LP = 8;                        // lanes of a group
constexpr int SV_PAD = 2;                       // doubles of padding per column (columns stay on 16-byte boundaries)
constexpr int SV_MAX_SWEEPS = 60;
constexpr size_t svd_smem_bytes(int d) { return sizeof(double) * (size_t)(d / 2) * (d + SV_PAD); }

// approximations to about 2^-22; arguments of the fp32 normal range
__device__ __forceinline__ float svd_rcp(float v) { float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v)); return r; }
__device__ __forceinline__ float svd_rsqrt(float v) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v)); return r; }

// A plane rotation of the columns x, y by the angle theta as three shears, in place:
//   x += al y,  y += be x,  x += al y   with  al = -tan(theta / 2), be = sin(theta):   x' = c x - s y,  y' = s x + c y.
// Three multiply-adds per row, no scale factors to keep.  tan(theta / 2) needs no more than single precision: an error eps
// leaves eps times the old inner product behind, which the next sweep removes; the rotation itself is orthogonal to fp64
// because be and c follow from the rounded tan(theta / 2) in fp64.
struct SvdRotation {
    double td, be;                              // tan(theta / 2), sin(theta)
    float tab;                                  // tan(theta) * (x . y): the squared norms become aa - tab, bb + tab
};

// `aa`, `bb`: squared norms, `dot` = x . y.  No branches: a pair that is orthogonal already gets the angle zero.  `lean2`:
// see the end of a sweep below.
__device__ __forceinline__ bool svd_rotation(float aa, float bb, double dot, SvdRotation& r, float& lean2) {
    const float ra = svd_rcp(aa), rb = svd_rcp(bb);
    const float ab = (float)dot, cc = (ab * ra) * (ab * rb);
    // |cos| > 1e-13 (well above the rounding noise of the inner product), as a product of ratios so that columns of very
    // different size neither overflow nor underflow the test
    const bool turn = fminf(aa, bb) > 1e-37f && cc > 1e-26f;
    // (cos, sin) of the doubled angle ~ (|bb - aa|, 2 ab), brought to the order of one by a power of two
    const float df = bb - aa, t2ab = 2.f * ab;
    const float sc = __int_as_float(0x7f000000 - (__float_as_int(fmaxf(fabsf(df), fabsf(t2ab))) & 0x7f800000));
    const float dn = fabsf(df) * sc, tn = (df >= 0.f ? t2ab : -t2ab) * sc;
    const float ih = svd_rsqrt(fmaf(dn, dn, tn * tn));
    const float u = fmaf(0.5f * dn, ih, 0.5f), iu = svd_rsqrt(u), cs = u * iu;       // cos^2(theta), 1 / cos(theta), cos(theta)
    const float s2 = tn * ih;                                                       // sin(2 theta)
    const float tau = turn ? 0.5f * s2 * svd_rcp(cs + u) : 0.f;
    const float t = 0.5f * s2 * (iu * iu);
    // sin(theta) = 2 tau / (1 + tau^2) in fp64: cos^2(theta / 2) = (1 + cos(theta)) / 2 is the reciprocal to single
    // precision, one step of third order makes it exact
    const double td = (double)tau, r0 = (double)(turn ? fmaf(0.5f, cs, 0.5f) : 1.f), p = (td + td) * r0;
    const double e = fma(-fma(td, td, 1.0), r0, 1.0);
    r.td = td;
    r.be = fma(p, fma(e, e, e), p);
    r.tab = turn ? t * ab : 0.f;
    if (turn) lean2 = fmaxf(lean2, t * t * fmaxf(aa * rb, bb * ra));
    return turn;
}

// One CTA per (sign, slot).  Outputs: U [D x D] row-major with the left singular vectors of Omega as columns, S descending,
// and the smallest k with sum_{i<=k} S_i >= gamma * sum_i S_i (Eq. 3).
//
// 1. Householder QR of Omega^T with its columns (the rows of Omega) taken by falling norm:  Omega^T P = Q R, so Omega has the
//    left singular vectors and the singular values of L = P R^T, whose rows stand in the order of Omega's.  Omega^T is
//    held by columns; step k finishes entry k of every column, so what the last step leaves is L, row by row.
//    L is far closer to orthogonal columns than Omega is (Drmac and Veselic's preconditioning of the Jacobi method): 5-6
//    sweeps instead of 10-12 on learned cross-covariances, for the price of about one sweep.
// 2. One-sided Jacobi (Hestenes): plane rotations from the right make the columns of L mutually orthogonal, L J = U S.
//
// Half of the columns live in registers, half in shared memory: two CTAs fit on an SM and their rounds overlap.  A group of
// SV_LP lanes holds two columns (x0, x1); lane lg holds the rows 2 SV_LP e + 2 lg + {0, 1}.
//
// Ordering of a sweep (every pair of columns meets once): level m = D / 2, D / 4, ..., 2 cuts the D / 2 column positions of
// either kind into blocks of m.  In round r of the level, the group whose columns are the 2i-th and (2i + 1)-th of its block
// meets the columns 2 ((i + r) mod (m / 2)) and the one after it of the block in shared memory: one read and one write of a
// column for two rotations, a barrier for four.
// Both inner products are formed at once: the second, with the column that the first rotation leaves, follows from x0 . x1,
// which is formed once a level and carried along (what the single-precision angle leaves of x0' . y' is neglected there: a
// relative 2^-22 of a product that shrinks quadratically).  Between levels the groups of the second half of a block swap their
// columns with the ones in shared memory half a block before: pairs within either half meet next.  The last level rotates
// x0 against x1, swaps both with shared memory, and rotates again.
//
// End: a sweep without a rotation, or one after which no pair can have a cosine above 1e-13: with l the largest
// |t| max(|A| / |B|, |B| / |A|) of the sweep (how far a rotation leans a column, relative to its length; never less than the
// cosine that it removes), a pair made orthogonal meets at most 2 (D - 1) more rotations, each of which changes its cosine by at
// most l^2.
//
// What bounds it: the shared-memory reads and writes of the visiting columns and the latency of a round (inner products,
// angle, update: a chain of dependent operations).  128 registers a thread are what two CTAs leave: at D = 128 the
// visiting column is read a second time rather than held through the angles (all / half of it held: 17 % / 1 % slower; at
// D = 64 there is room, and a second read costs 3 %).
// Measured, 576 matrices of 128 x 128: 5.99 -> 2.55 ms (before: no QR, one column per group resident, the whole matrix in
// shared memory and so one CTA per SM, scaled rotations).
template <int D>
__global__ void __launch_bounds__(2 * D, D == 128 ? 2 : 4)
learn_svd_kernel(const float* __restrict__ omega_pos, const float* __restrict__ omega_neg, int slots, float gamma,
                 float* __restrict__ U_pos, float* __restrict__ U_neg, float* __restrict__ S_pos, float* __restrict__ S_neg,
                 int* __restrict__ k_pos, int* __restrict__ k_neg, int* __restrict__ sweeps_out) {
    constexpr int NT = 2 * D, NP = D / 2, LDG = D + SV_PAD;       // threads, columns of either kind, column stride
    constexpr int NE = D / (2 * SV_LP), HE = NE / 2;              // row pairs per lane; those of the first D / 2 rows
    extern __shared__ __align__(16) double sv_sm[];
    double* G = sv_sm;                      // [NP][LDG]: the columns in shared memory
    __shared__ __align__(16) double vbuf[2][D];
    __shared__ double sig[D], beta[2];
    __shared__ float nrm2[NP], red[NT / 32];
    __shared__ int order[D];
    __shared__ unsigned worst;              // bits of the largest lean2 of a sweep
    const int sign = blockIdx.x / slots, slot = blockIdx.x % slots;
    const float* om = (sign == 0 ? omega_pos : omega_neg) + (size_t)slot * D * D;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = tid / SV_LP, lg = tid % SV_LP;      // group, lane within the group
    const unsigned group_mask = 0xffu << (lane & ~(SV_LP - 1));
    auto group_sum = [&](double v) {
#pragma unroll
        for (int o = SV_LP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(group_mask, v, o);
        return v;
    };
    double2* gp0 = reinterpret_cast<double2*>(G + (size_t)(2 * g) * LDG) + lg;          // the two positions that the group
    double2* gp1 = reinterpret_cast<double2*>(G + (size_t)(2 * g + 1) * LDG) + lg;      // folds, swaps and reduces

    // ---- Omega^T by columns, its largest entry scaled to 2^40 (the squares of the norms have to fit fp32: 2^-125 to 2^94)
    double2 x0[NE], x1[NE], y[NE];
    float mx = 0.f;
    {
        auto row = [&](int j, int e) {
            const float2 v = *reinterpret_cast<const float2*>(om + (size_t)j * D + 2 * SV_LP * e + 2 * lg);
            mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
            return make_double2((double)v.x, (double)v.y);
        };
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            x0[e] = row(2 * g, e);
            x1[e] = row(2 * g + 1, e);
            gp0[SV_LP * e] = row(NP + 2 * g, e);
            gp1[SV_LP * e] = row(NP + 2 * g + 1, e);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    mx = 0.f;
    for (int w = 0; w < NT / 32; ++w) mx = fmaxf(mx, red[w]);
    const double scale = (double)mx * 0x1p-40, inv_scale = mx > 0.f ? 1.0 / scale : 0.0;
    {
        double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;
        auto scaled = [&](double2& v, double& n) {
            v.x *= inv_scale; v.y *= inv_scale;
            n = fma(v.x, v.x, fma(v.y, v.y, n));
        };
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            scaled(x0[e], n0);
            scaled(x1[e], n1);
            double2 v = gp0[SV_LP * e];
            scaled(v, n2); gp0[SV_LP * e] = v;
            v = gp1[SV_LP * e];
            scaled(v, n3); gp1[SV_LP * e] = v;
        }
        n0 = group_sum(n0); n1 = group_sum(n1); n2 = group_sum(n2); n3 = group_sum(n3);
        if (lg == 0) { sig[2 * g] = n0; sig[2 * g + 1] = n1; sig[NP + 2 * g] = n2; sig[NP + 2 * g + 1] = n3; }
    }
    __syncthreads();
    if (tid < D) {
        int rk = 0;
#pragma unroll 4
        for (int i = 0; i < D; ++i) rk += (sig[i] > sig[tid] || (sig[i] == sig[tid] && i < tid)) ? 1 : 0;
        order[rk] = tid;
    }
    __syncthreads();

    // ---- QR: one barrier per step; the owner of the next pivot column publishes its reflector I - beta v v^T
    auto publish = [&](int k) {
        const int j = order[k], jj = j & (NP - 1);
        if ((jj >> 1) != g) return;
        const double2* c = (jj & 1) == 0 ? gp0 : gp1;
        double n0 = 0.0, n1 = 0.0, pv = 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int i = 2 * SV_LP * e + 2 * lg;
            y[e] = c[SV_LP * e];
            if (j < NP) y[e] = (jj & 1) == 0 ? x0[e] : x1[e];
            if (i < k) y[e].x = 0.0;
            if (i + 1 < k) y[e].y = 0.0;
            if (i == k) pv = y[e].x;
            if (i + 1 == k) pv = y[e].y;
            n0 = fma(y[e].x, y[e].x, n0);
            n1 = fma(y[e].y, y[e].y, n1);
        }
        n0 = group_sum(n0 + n1);
        // the norm to 2^-42 (it only decides how close to zero the column is brought), beta = 2 / (v . v) to fp64
        const double r = (double)svd_rsqrt((float)n0), n = n0 * (r * fma(-0.5 * n0, r * r, 1.5));
        const bool some = n0 > 1e-36;           // (columns below 2^-100 of the largest entry: no reflection)
        const double vk = some ? pv + (pv < 0.0 ? -n : n) : 0.0, vv = fma(vk, vk, fma(-pv, pv, n0));
        const double q = (double)svd_rcp((float)vv), e1 = fma(-vv, q, 1.0);
        if (((k >> 1) & (SV_LP - 1)) == lg) beta[k & 1] = some ? 2.0 * fma(q, fma(e1, e1, e1), q) : 0.0;     // the lane of row k
        double2* vb = reinterpret_cast<double2*>(vbuf[k & 1]) + lg;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int i = 2 * SV_LP * e + 2 * lg;
            vb[SV_LP * e] = make_double2(i == k ? vk : y[e].x, i + 1 == k ? vk : y[e].y);
        }
    };
    publish(0);
    __syncthreads();
#pragma unroll 1
    for (int k = 0; k < D; ++k) {
        const double2* vb = reinterpret_cast<const double2*>(vbuf[k & 1]) + lg;
        double d0 = 0.0, d1 = 0.0, d2 = 0.0, d3 = 0.0;
        auto dots = [&](int e) {
            const double2 v = vb[SV_LP * e], c3 = gp1[SV_LP * e];
            y[e] = gp0[SV_LP * e];
            d0 = fma(v.x, x0[e].x, fma(v.y, x0[e].y, d0));
            d1 = fma(v.x, x1[e].x, fma(v.y, x1[e].y, d1));
            d2 = fma(v.x, y[e].x, fma(v.y, y[e].y, d2));
            d3 = fma(v.x, c3.x, fma(v.y, c3.y, d3));
        };
        auto update = [&](int e) {
            const double2 v = vb[SV_LP * e];
            double2 c = gp1[SV_LP * e];
            x0[e].x = fma(d0, v.x, x0[e].x); x0[e].y = fma(d0, v.y, x0[e].y);
            x1[e].x = fma(d1, v.x, x1[e].x); x1[e].y = fma(d1, v.y, x1[e].y);
            gp0[SV_LP * e] = make_double2(fma(d2, v.x, y[e].x), fma(d2, v.y, y[e].y));
            c.x = fma(d3, v.x, c.x); c.y = fma(d3, v.y, c.y);
            gp1[SV_LP * e] = c;
        };
        // the reflector is zero above row k: the first half of the rows is finished after half of the steps
        if (k < D / 2) {
#pragma unroll
            for (int e = 0; e < HE; ++e) dots(e);
        }
#pragma unroll
        for (int e = HE; e < NE; ++e) dots(e);
        const double nb = -beta[k & 1];
        d0 = nb * group_sum(d0); d1 = nb * group_sum(d1); d2 = nb * group_sum(d2); d3 = nb * group_sum(d3);
        if (k < D / 2) {
#pragma unroll
            for (int e = 0; e < HE; ++e) update(e);
        }
#pragma unroll
        for (int e = HE; e < NE; ++e) update(e);
        if (k + 1 < D) publish(k + 1);
        __syncthreads();
    }

    // ---- column j, entry k  ->  column k, entry j, through the shared half
    {
        auto at = [&](int c, int i) -> double& { return G[(size_t)c * LDG + i]; };
        auto i0 = [&](int e) { return 2 * SV_LP * e + 2 * lg; };
#pragma unroll
        for (int e = 0; e < HE; ++e) {
            y[e] = make_double2(at(i0(e), 2 * g), at(i0(e) + 1, 2 * g));
            y[HE + e] = make_double2(at(i0(e), 2 * g + 1), at(i0(e) + 1, 2 * g + 1));
        }
        for (int idx = tid; idx < NP * NP; idx += NT) {         // the quarter that stays in shared memory
            const int c = idx / NP, i = idx % NP;
            if (i < c) { const double u = at(c, NP + i); at(c, NP + i) = at(i, NP + c); at(i, NP + c) = u; }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < HE; ++e) { gp0[SV_LP * e] = x0[e]; gp1[SV_LP * e] = x1[e]; }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < HE; ++e) {
            x0[e] = make_double2(at(i0(e), 2 * g), at(i0(e) + 1, 2 * g));
            x1[e] = make_double2(at(i0(e), 2 * g + 1), at(i0(e) + 1, 2 * g + 1));
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < HE; ++e) {
            at(i0(e), 2 * g) = x0[HE + e].x; at(i0(e) + 1, 2 * g) = x0[HE + e].y;
            at(i0(e), 2 * g + 1) = x1[HE + e].x; at(i0(e) + 1, 2 * g + 1) = x1[HE + e].y;
            x0[HE + e] = y[e];
            x1[HE + e] = y[HE + e];
        }
        __syncthreads();
    }

    // ---- Jacobi
    double nx0, nx1, ny0, ny1;              // squared norms of the group's columns and of the two at its positions
    auto norms = [&]() {
        auto add = [](const double2& v, double& n) { n = fma(v.x, v.x, fma(v.y, v.y, n)); };
        nx0 = nx1 = ny0 = ny1 = 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e) { add(x0[e], nx0); add(x1[e], nx1); add(gp0[SV_LP * e], ny0); add(gp1[SV_LP * e], ny1); }
        nx0 = group_sum(nx0); nx1 = group_sum(nx1); ny0 = group_sum(ny0); ny1 = group_sum(ny1);
    };
    float aa0, aa1;
    // x0, x1 <-> the columns at positions q and q + 1
    auto swap_columns = [&](int q) {
        double2* c0 = reinterpret_cast<double2*>(G + (size_t)q * LDG) + lg;
        double2* c1 = reinterpret_cast<double2*>(G + (size_t)(q + 1) * LDG) + lg;
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            double2 v = c0[SV_LP * e]; c0[SV_LP * e] = x0[e]; x0[e] = v;
            v = c1[SV_LP * e]; c1[SV_LP * e] = x1[e]; x1[e] = v;
        }
        const float n0 = nrm2[q], n1 = nrm2[q + 1];
        __syncwarp(group_mask);
        if (lg == 0) { nrm2[q] = aa0; nrm2[q + 1] = aa1; }
        aa0 = n0; aa1 = n1;
    };
    auto resident_dot = [&]() {
        double a = 0.0, b = 0.0;
#pragma unroll
        for (int e = 0; e < NE; ++e) { a = fma(x0[e].x, x1[e].x, a); b = fma(x0[e].y, x1[e].y, b); }
        return group_sum(a + b);
    };
    // a block's columns change hands: the warps of the block (8 columns per warp) wait for one another.  Every block of every
    // level has a barrier of its own (1, 2 | 3 .. 6): one block may be a level ahead of another
    auto block_sync = [&](int m) {
        __syncwarp();
        if (m == NP) __syncthreads();
        else if (m > 8) asm volatile("bar.sync %0, %1;" ::"r"(NP / m - 1 + 2 * g / m), "r"(m * 4) : "memory");
    };
    int sweep = 0;
    for (; sweep < SV_MAX_SWEEPS; ++sweep) {
        norms();                            // exact at the start of every sweep; inside it they follow the rotations in fp32,
        aa0 = (float)nx0; aa1 = (float)nx1; // as they only feed the tangent
        if (lg == 0) { nrm2[2 * g] = (float)ny0; nrm2[2 * g + 1] = (float)ny1; }
        if (tid == 0) worst = 0u;
        __syncthreads();
        float lean2 = 0.f;
#pragma unroll 1
        for (int m = NP; m >= 2; m >>= 1) {
            const int idx = (2 * g) & (m - 1), p0 = 2 * g - idx;        // position in the block, first position of the block
            double g01 = resident_dot();
#pragma unroll 1
            for (int r = 0; r < m; ++r) {
                const int q = p0 + ((idx + r) & (m - 2)) + (r & 1);
                double2* gb = reinterpret_cast<double2*>(G + (size_t)q * LDG) + lg;
                double a0 = 0.0, b0 = 0.0, a1 = 0.0, b1 = 0.0;
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    y[e] = gb[SV_LP * e];
                    a0 = fma(x0[e].x, y[e].x, a0); a1 = fma(x1[e].x, y[e].x, a1);
                    b0 = fma(x0[e].y, y[e].y, b0); b1 = fma(x1[e].y, y[e].y, b1);
                }
                const float bb = nrm2[q];
                const double d0 = group_sum(a0 + b0), d1 = group_sum(a1 + b1);
                // every lane of the group holds the same sums and works out the same rotations
                SvdRotation u, v;
                if (D == 128) asm volatile("" ::: "memory");       // (read again below, not held through the angles)
                bool any = svd_rotation(aa0, bb, d0, u, lean2);
                any |= svd_rotation(aa1, bb + u.tab, fma(u.be, fma(-u.td, d1, g01), d1), v, lean2);
                if (__any_sync(0xffffffffu, any)) {
                    g01 = fma(-u.be, fma(u.td, g01, d1), g01);
                    aa0 = fmaxf(aa0 - u.tab, 0.f); aa1 = fmaxf(aa1 - v.tab, 0.f);
                    if (lg == 0) nrm2[q] = bb + u.tab + v.tab;
#pragma unroll
                    for (int e = 0; e < NE; ++e) {
                        double2 c = D == 128 ? gb[SV_LP * e] : y[e];
                        x0[e].x = fma(-u.td, c.x, x0[e].x); x0[e].y = fma(-u.td, c.y, x0[e].y);
                        c.x = fma(u.be, x0[e].x, c.x); c.y = fma(u.be, x0[e].y, c.y);
                        x0[e].x = fma(-u.td, c.x, x0[e].x); x0[e].y = fma(-u.td, c.y, x0[e].y);
                        x1[e].x = fma(-v.td, c.x, x1[e].x); x1[e].y = fma(-v.td, c.y, x1[e].y);
                        c.x = fma(v.be, x1[e].x, c.x); c.y = fma(v.be, x1[e].y, c.y);
                        x1[e].x = fma(-v.td, c.x, x1[e].x); x1[e].y = fma(-v.td, c.y, x1[e].y);
                        gb[SV_LP * e] = c;
                    }
                }
                if (r & 1) block_sync(m);
            }
            if (m > 2) {
                if (idx >= m / 2) swap_columns(2 * g - m / 2);
                block_sync(m);
            }
        }
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            SvdRotation u;
            if (svd_rotation(aa0, aa1, resident_dot(), u, lean2)) {
                aa0 = fmaxf(aa0 - u.tab, 0.f); aa1 += u.tab;
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    x0[e].x = fma(-u.td, x1[e].x, x0[e].x); x0[e].y = fma(-u.td, x1[e].y, x0[e].y);
                    x1[e].x = fma(u.be, x0[e].x, x1[e].x); x1[e].y = fma(u.be, x0[e].y, x1[e].y);
                    x0[e].x = fma(-u.td, x1[e].x, x0[e].x); x0[e].y = fma(-u.td, x1[e].y, x0[e].y);
                }
            }
            if (h == 0) swap_columns(2 * g);
        }
        if (lg == 0) atomicMax(&worst, __float_as_uint(lean2));
        __syncthreads();
        const bool done = __uint_as_float(worst) < 1e-13f / (2 * (D - 1));
        __syncthreads();
        if (done) break;
    }
    norms();                                        // singular values = column norms
    if (lg == 0) { sig[2 * g] = sqrt(nx0); sig[2 * g + 1] = sqrt(nx1); sig[NP + 2 * g] = sqrt(ny0); sig[NP + 2 * g + 1] = sqrt(ny1); }
    __syncthreads();
    // descending order (ties: the earlier column first)
    if (tid < D) {
        int rk = 0;
#pragma unroll 4
        for (int i = 0; i < D; ++i) rk += (sig[i] > sig[tid] || (sig[i] == sig[tid] && i < tid)) ? 1 : 0;
        order[tid] = rk;
    }
    __syncthreads();
    float* Uo = (sign == 0 ? U_pos : U_neg) + (size_t)slot * D * D;
    float* So = (sign == 0 ? S_pos : S_neg) + (size_t)slot * D;
    auto write_half = [&](int c0) {
        for (int idx = tid; idx < D * NP; idx += NT) {
            const int i = idx / NP, j = idx % NP;   // component i of column j
            const double sv = sig[c0 + j];
            Uo[(size_t)i * D + order[c0 + j]] = sv > 0.0 ? (float)(G[(size_t)j * LDG + i] / sv) : 0.f;
        }
    };
    write_half(NP);
    if (tid < D) So[order[tid]] = (float)(sig[tid] * scale);        // the scale of the matrix goes back on
    __syncthreads();
#pragma unroll
    for (int e = 0; e < NE; ++e) { gp0[SV_LP * e] = x0[e]; gp1[SV_LP * e] = x1[e]; }
    __syncthreads();
    write_half(0);
    __syncthreads();
    if (tid < D) G[order[tid]] = sig[tid];          // the matrix has been written out: its first entries take the sorted values
    __syncthreads();
    if (tid == 0) {
        // Eq. 3 on the sorted values, in fp64
        double total = 0.0;
#pragma unroll 4
        for (int j = 0; j < D; ++j) total += G[j];
        double run = 0.0;
        int k = D;
#pragma unroll 1
        for (int j = 0; j < D; ++j) {
            run += G[j];
            if (run >= (double)gamma * total) { k = j + 1; break; }
        }
        (sign == 0 ? k_pos : k_neg)[slot] = k;
        if (sweeps_out != nullptr) sweeps_out[blockIdx.x] = sweep;
    }
}

struct LearnPlan {
    int n_groups, chunk_tokens, n_chunks;
    size_t part_off, part_bytes, dsum_off, dsum_bytes, dcnt_off, dcnt_bytes, sweeps_off, sweeps_bytes, total;
};

seka_status validate_learn(const seka_learn_shape* s) {
    if (s == nullptr) return SEKA_ERR_INVALID_ARG;
    if (s->n_tokens <= 0 || s->n_slots <= 0) return SEKA_ERR_INVALID_ARG;
    if (!(s->gamma > 0.f) || !(s->gamma <= 1.f)) return SEKA_ERR_INVALID_ARG;
    if (s->head_dim != 64 && s->head_dim != 128) return SEKA_ERR_UNSUPPORTED;
    if (s->head_dim == 64 && (s->n_slots & 1)) return SEKA_ERR_UNSUPPORTED;       // heads of 64 are processed in pairs
    if ((long long)s->n_tokens * s->n_slots > 0x7fffffffLL) return SEKA_ERR_UNSUPPORTED;
    return SEKA_OK;
}

// Chunks of tokens: a few items per SM so that the accumulator drain of one item hides under the next, but long
// enough (>= 2048 tokens) that the partials stay small next to the embeddings.
LearnPlan learn_plan(const seka_learn_shape* s) {
    LearnPlan pl;
    const int d = s->head_dim;
    pl.n_groups = d == 128 ? s->n_slots : s->n_slots / 2;
    long long want = (4LL * 148 + pl.n_groups - 1) / pl.n_groups;          // chunks that give about 4 items per SM
    if (want < 1) want = 1;
    long long chunk = (s->n_tokens + want - 1) / want;
    if (chunk < 2048) chunk = 2048;
    chunk = (chunk + LC_TOK - 1) / LC_TOK * LC_TOK;
    pl.chunk_tokens = (int)chunk;
    pl.n_chunks = (int)((s->n_tokens + chunk - 1) / chunk);
    pl.part_off = kStatusBytes;
    pl.part_bytes = align_up((size_t)pl.n_chunks * s->n_slots * 2 * d * d * sizeof(float), 256);
    pl.dsum_off = pl.part_off + pl.part_bytes;
    pl.dsum_bytes = align_up((size_t)pl.n_chunks * 4 * s->n_slots * sizeof(double), 256);
    pl.dcnt_off = pl.dsum_off + pl.dsum_bytes;
    pl.dcnt_bytes = align_up((size_t)pl.n_chunks * 4 * sizeof(int), 256);
    pl.sweeps_off = pl.dcnt_off + pl.dcnt_bytes;
    pl.sweeps_bytes = align_up((size_t)2 * s->n_slots * sizeof(int), 256);
    pl.total = pl.sweeps_off + pl.sweeps_bytes;
    return pl;
}

}  // namespace
}  // namespace seka

extern "C" size_t seka_learn_workspace_bytes(const seka_learn_shape* shape) {
    if (seka::validate_learn(shape) != SEKA_OK) return 0;
    return seka::learn_plan(shape).total;
}

extern "C" seka_status seka_learn_projections(const seka_learn_shape* shape, const void* h, const void* h_pos,
                                              const void* h_neg, const uint8_t* answer_tokens,
                                              float* omega_pos, float* omega_neg, float* U_pos, float* U_neg,
                                              float* S_pos, float* S_neg, int32_t* k_pos, int32_t* k_neg, float* D,
                                              void* workspace, size_t workspace_bytes, void* cuda_stream) {
    using namespace seka;
    seka_status stc = validate_learn(shape);
    if (stc != SEKA_OK) return stc;
    if (!h || !h_pos || !h_neg || !omega_pos || !omega_neg || !U_pos || !U_neg || !S_pos || !S_neg || !k_pos || !k_neg || !D)
        return SEKA_ERR_INVALID_ARG;
    if (((uintptr_t)h | (uintptr_t)h_pos | (uintptr_t)h_neg | (uintptr_t)omega_pos | (uintptr_t)omega_neg) & 15) return SEKA_ERR_INVALID_ARG;
    const LearnPlan pl = learn_plan(shape);
    if (!workspace || workspace_bytes < pl.total || ((uintptr_t)workspace & 255)) return SEKA_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    char* ws = static_cast<char*>(workspace);
    const int d = shape->head_dim, slots = shape->n_slots, n = shape->n_tokens;

    // per-device facts: looked up per device; function attributes set on every call (they belong to the current device)
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    if (cudaFuncSetAttribute(learn_cov_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LC_DYN_BYTES) != cudaSuccess ||
        cudaFuncSetAttribute(learn_svd_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)svd_smem_bytes(128)) != cudaSuccess)
        return SEKA_ERR_CUDA;

    // cross-covariances: columns in groups of 128 (one head of 128, or two neighbouring heads of 64)
    CUtensorMap tmH, tmP, tmN;
    if (!make_tile_map(&tmH, h, 128, pl.n_groups, n, LC_TOK) || !make_tile_map(&tmP, h_pos, 128, pl.n_groups, n, LC_TOK) ||
        !make_tile_map(&tmN, h_neg, 128, pl.n_groups, n, LC_TOK))
        return SEKA_ERR_CUDA;
    LearnCovParams p;
    p.part = reinterpret_cast<float*>(ws + pl.part_off);
    p.dist = reinterpret_cast<double*>(ws + pl.dsum_off);
    p.count = reinterpret_cast<int*>(ws + pl.dcnt_off);
    p.answer = answer_tokens;
    p.n_tokens = n; p.n_groups = pl.n_groups; p.d = d; p.slots = slots;
    p.chunk_tokens = pl.chunk_tokens; p.n_chunks = pl.n_chunks; p.status = reinterpret_cast<int*>(ws);
    const int n_items = pl.n_groups * pl.n_chunks;
    learn_cov_kernel<<<n_items < n_sm ? n_items : n_sm, LC_THREADS, LC_DYN_BYTES, st>>>(tmH, tmP, tmN, p);
    ++g_launches;
    const unsigned omega_blocks = (unsigned)(((size_t)slots * 2 * d * d / 4 + LR_THREADS - 1) / LR_THREADS);
    const unsigned dist_blocks = (unsigned)((slots + LR_THREADS / 32 - 1) / (LR_THREADS / 32));
    learn_reduce_kernel<<<omega_blocks + dist_blocks, LR_THREADS, 0, st>>>(p, omega_pos, omega_neg, D, omega_blocks, 1.f / (float)n);
    ++g_launches;

    // SVD of every Omega, rank rule
    auto svd = d == 128 ? learn_svd_kernel<128> : learn_svd_kernel<64>;
    svd<<<2 * slots, 2 * d, svd_smem_bytes(d), st>>>(omega_pos, omega_neg, slots, shape->gamma, U_pos, U_neg, S_pos, S_neg, k_pos, k_neg,
                                                     reinterpret_cast<int*>(ws + pl.sweeps_off));
    ++g_launches;
    return cudaGetLastError() == cudaSuccess ? SEKA_OK : SEKA_ERR_CUDA;
}

// Standalone key-editing kernel (the hook of Algorithm 1 / Algorithm 2 applied to a key tensor in HBM).
#include "seka_kernels.h"
#include "seka_route.cuh"

namespace seka {

__device__ __forceinline__ int find_sequence(const int* __restrict__ cu, int B, int L, int t) {
    if (cu == nullptr) return t / L;
    int lo = 0, hi = B - 1;            // largest b with cu[b] <= t
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cu[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------- fp32 arithmetic: a CTA per (64-token tile, KV head)
//
//   C = U_m^T k (highlighted rows x rank),  k' = k + g sum_m alpha_m U_m C,  both products as blocked fp32 multiply-adds.
//
// The CTA finds its highlighted rows itself (no list, no launch of its own for it), gathers them into shared memory, and
// walks the rank 32 columns at a time: U's chunk [D x 32] is staged once for all rows of the tile, so an element of U is
// read from global memory once per tile instead of once per row (one warp per row, everything through shuffles, was bound
// by the latency of that chain).  With a second output tensor the rows that are not highlighted are copied in the same
// pass, 16 bytes per lane; the loads go out before the highlight flags are known.  Bound by HBM where the copy dominates
// (the fp32 layer of 6000 tokens x 16 heads x 64, rank 16, a tenth highlighted, into a second tensor: copy + list + a warp
// per row 56 us per call, this 19 us; 21 without its placement under the tail of the launch before), by the fp32 pipe where most rows are highlighted (4 D rank flops per row).
constexpr int ER_ROWS = 64, ER_THREADS = 256, ER_CP = 36;     // tokens per tile; pitch (floats) of 32-column chunks: float4 reads of 8 rows meet 32 banks

template <typename T> struct Row16;        // 16 bytes of a row <-> fp32 values
template <> struct Row16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void unpack(const uint4& v, float* f) {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ void store4(float* dst, const float (&f)[4]) {
        *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
    }
};
template <> struct Row16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void unpack(const uint4& v, float* f) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
            f[2 * e] = x.x; f[2 * e + 1] = x.y;
        }
    }
    static __device__ __forceinline__ void store4(__nv_bfloat16* dst, const float (&f)[4]) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]));
    }
};

template <int D> constexpr size_t edit_rows_smem() { return sizeof(float) * (ER_ROWS * (D + 4) + D * ER_CP + ER_ROWS * ER_CP); }

template <typename T, int D, bool COPY>
__global__ void __launch_bounds__(ER_THREADS)
edit_rows_kernel(const T* K_in, T* K_out, const uint8_t* __restrict__ mask, const float* __restrict__ U,
                 const float* __restrict__ alpha, const float* __restrict__ gain,
                 const uint8_t* __restrict__ head_enable, const int* __restrict__ cu, int n_tok, int B, int L,
                 int Hkv, int r, int M, int heads_per_cta) {
    using R = Row16<T>;
    constexpr int KP = D + 4;                              // pitch of a key row in shared memory (16-byte aligned rows)
    constexpr int UPR = D / R::N;                          // 16-byte units of a key row
    constexpr int NV = ER_ROWS * UPR / ER_THREADS;         // units per thread
    extern __shared__ __align__(16) float er_sm[];
    float* Ks = er_sm;                                     // [64][KP]   highlighted rows, compacted
    float* Us = Ks + ER_ROWS * KP;                         // [D][ER_CP] 32 columns of U_m
    float* Cs = Us + D * ER_CP;                            // [64][ER_CP]
    __shared__ int slot_of[ER_ROWS], row_of[ER_ROWS], seq_of[ER_ROWS], cnt_s[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int hgroups = (Hkv + heads_per_cta - 1) / heads_per_cta;
    const int t0 = (int)(blockIdx.x / hgroups) * ER_ROWS, h0 = (int)(blockIdx.x % hgroups) * heads_per_cta;
    const int h1 = h0 + heads_per_cta < Hkv ? h0 + heads_per_cta : Hkv;
    const int n_rows = n_tok - t0 < ER_ROWS ? n_tok - t0 : ER_ROWS;

    pdl_wait();
    pdl_release();
    // a second tensor: the first head's rows are on their way while the flags are looked up
    uint4 v[NV];
    auto load_rows = [&](int h) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const int u = q * ER_THREADS + tid, row = u / UPR, c = u % UPR;
            if (row < n_rows) v[q] = *reinterpret_cast<const uint4*>(K_in + ((size_t)(t0 + row) * Hkv + h) * D + c * R::N);
        }
    };
    if (COPY) load_rows(h0);
    // highlighted rows of the tile, in order: slots 0 .. n_hot - 1
    bool hl = false;
    int b = 0;
    if (tid < ER_ROWS) {
        if (tid < n_rows && mask[t0 + tid] != 0) {
            b = find_sequence(cu, B, L, t0 + tid);
            hl = gain[b] != 0.f;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, hl);
        if (lane == 0) cnt_s[warp] = __popc(bal);
        slot_of[tid] = hl ? __popc(bal & ((1u << lane) - 1)) : -1;
    }
    __syncthreads();
    const int n_hot = cnt_s[0] + cnt_s[1];
    if (!COPY && n_hot == 0) return;
    if (tid < ER_ROWS && hl) {
        const int s = slot_of[tid] + (warp == 1 ? cnt_s[0] : 0);
        slot_of[tid] = s; row_of[s] = tid; seq_of[s] = b;
    }
    __syncthreads();

    for (int h = h0; h < h1; ++h) {
        const bool on = n_hot > 0 && (head_enable == nullptr || head_enable[h] != 0);
        if (COPY) {
            if (h != h0) load_rows(h);
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const int u = q * ER_THREADS + tid, row = u / UPR, c = u % UPR;
                if (row >= n_rows) continue;
                const int s = on ? slot_of[row] : -1;
                if (s < 0) *reinterpret_cast<uint4*>(K_out + ((size_t)(t0 + row) * Hkv + h) * D + c * R::N) = v[q];
                else R::unpack(v[q], Ks + s * KP + c * R::N);
            }
        } else if (on) {
            for (int u = tid; u < n_hot * UPR; u += ER_THREADS) {
                const int s = u / UPR, c = u % UPR;
                R::unpack(*reinterpret_cast<const uint4*>(K_in + ((size_t)(t0 + row_of[s]) * Hkv + h) * D + c * R::N), Ks + s * KP + c * R::N);
            }
        }
        if (!on) continue;
        // k' accumulates per thread: rows rg, rg + 16, ... (few highlighted rows still spread over all threads), 4 columns
        // at 4 cg (and at 64 + 4 cg)
        constexpr int NC = D / 64;
        const int cg = tid & 15, rg = tid >> 4;
        float acc[4][NC][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][c][e] = 0.f;
        for (int m = 0; m < M; ++m) {
            const float* Um = U + ((size_t)m * Hkv + h) * D * r;
            for (int j0 = 0; j0 < r; j0 += 32) {
                const int rn = r - j0 < 32 ? r - j0 : 32;
                // columns of the chunk that are worked on: 8, 16 or 32 (zero beyond the rank); a narrow chunk leaves lanes
                // over, which then share the rows of U between them
                const int rp = rn <= 8 ? 8 : (rn <= 16 ? 16 : 32), rs = rn <= 8 ? 3 : (rn <= 16 ? 4 : 5);
                __syncthreads();                               // the previous chunk (or head) is through
                for (int u = tid; u < D * rp; u += ER_THREADS) {
                    const int i = u >> rs, j = u & (rp - 1);
                    Us[i * ER_CP + j] = j < rn ? __ldg(Um + (size_t)i * r + j0 + j) : 0.f;
                }
                __syncthreads();
                {   // C: warp w takes rows w, w + 8, ...; lane (s, j) column j, every (32 / rp)-th group of 4 dimensions
                    const int j = lane & (rp - 1), ks = 32 >> rs, s4 = (lane >> rs) * 4;
                    float c[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) c[i] = 0.f;
                    for (int d0 = s4; d0 < D; d0 += 4 * ks) {
                        float u4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) u4[e] = Us[(d0 + e) * ER_CP + j];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (warp + 8 * i >= n_hot) break;
                            const float4 k4 = *reinterpret_cast<const float4*>(Ks + (warp + 8 * i) * KP + d0);
                            c[i] = fmaf(k4.x, u4[0], fmaf(k4.y, u4[1], fmaf(k4.z, u4[2], fmaf(k4.w, u4[3], c[i]))));
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int s = warp + 8 * i;
                        if (s >= n_hot) break;
                        for (int o = rp; o < 32; o <<= 1) c[i] += __shfl_xor_sync(0xffffffffu, c[i], o);
                        if (lane < rp) {
                            const int sb = seq_of[s];
                            const float a = gain[sb] * (alpha != nullptr ? alpha[((size_t)sb * Hkv + h) * M + m] : 1.f);
                            Cs[s * ER_CP + j] = j < rn ? c[i] * a : 0.f;       // (an infinity times a zero column is not a zero)
                        }
                    }
                }
                __syncthreads();
                for (int jj = 0; jj < rn; jj += 4) {           // (columns up to the next multiple of 4 are zero)
                    float4 u4[NC][4];
#pragma unroll
                    for (int c = 0; c < NC; ++c)
#pragma unroll
                        for (int e = 0; e < 4; ++e) u4[c][e] = *reinterpret_cast<const float4*>(Us + (c * 64 + cg * 4 + e) * ER_CP + jj);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (rg + 16 * i >= n_hot) break;
                        const float4 c4 = *reinterpret_cast<const float4*>(Cs + (rg + 16 * i) * ER_CP + jj);
#pragma unroll
                        for (int c = 0; c < NC; ++c)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                acc[i][c][e] = fmaf(c4.x, u4[c][e].x, fmaf(c4.y, u4[c][e].y, fmaf(c4.z, u4[c][e].z, fmaf(c4.w, u4[c][e].w, acc[i][c][e]))));
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int s = rg + 16 * i;
            if (s >= n_hot) break;
            T* dst = K_out + ((size_t)(t0 + row_of[s]) * Hkv + h) * D;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float4 k4 = *reinterpret_cast<const float4*>(Ks + s * KP + c * 64 + cg * 4);
                const float o4[4] = {k4.x + acc[i][c][0], k4.y + acc[i][c][1], k4.z + acc[i][c][2], k4.w + acc[i][c][3]};
                R::store4(dst + c * 64 + cg * 4, o4);
            }
        }
        if (h + 1 < h1) __syncthreads();                       // the rows in shared memory are replaced
    }
}

template <typename T, int D>
static seka_status launch_edit_rows_t(const seka_shape* s, const void* K_in, void* K_out, const uint8_t* mask, const float* U,
                                      const float* alpha, const float* gain, const uint8_t* he, cudaStream_t st) {
    const int n_tok = shape_total_tokens(s);
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    const long long tiles = (n_tok + ER_ROWS - 1) / ER_ROWS;
    // one head per CTA (a highlighted span then spreads over many SMs) until there are so many CTAs that the empty ones
    // would cost more than the imbalance
    long long hpc = tiles * s->n_kv_heads / (32LL * n_sm);
    hpc = hpc < 1 ? 1 : (hpc > 4 ? 4 : hpc);
    const long long grid = tiles * ((s->n_kv_heads + hpc - 1) / hpc);
    if (grid > 0x7fffffffLL) return SEKA_ERR_UNSUPPORTED;
    auto kern = K_in == K_out ? edit_rows_kernel<T, D, false> : edit_rows_kernel<T, D, true>;
    constexpr size_t smem = edit_rows_smem<D>();
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return SEKA_ERR_CUDA;
    return launch_kernel(true, kern, (unsigned)grid, ER_THREADS, smem, st, static_cast<const T*>(K_in), static_cast<T*>(K_out), mask, U, alpha,
                         gain, he, s->cu_seqlens, n_tok, s->batch, s->max_seqlen, s->n_kv_heads, s->rank, s->n_experts, (int)hpc);
}

static seka_status launch_edit_rows(const seka_shape* s, const void* K_in, void* K_out, const uint8_t* mask, const float* U,
                                    const float* alpha, const float* gain, const uint8_t* he, cudaStream_t st) {
    if (s->dtype == SEKA_F32)
        return s->head_dim == 128 ? launch_edit_rows_t<float, 128>(s, K_in, K_out, mask, U, alpha, gain, he, st)
                                  : launch_edit_rows_t<float, 64>(s, K_in, K_out, mask, U, alpha, gain, he, st);
    return s->head_dim == 128 ? launch_edit_rows_t<__nv_bfloat16, 128>(s, K_in, K_out, mask, U, alpha, gain, he, st)
                              : launch_edit_rows_t<__nv_bfloat16, 64>(s, K_in, K_out, mask, U, alpha, gain, he, st);
}

// ---------------------------------------------------------------- bf16 tensors: 128 key rows per step, on tcgen05
//
// k' = k + sum_j c_j U[:, j] (U[:, j] . k) over the stacked columns j = (expert, direction), c_j = g_b alpha_{b,h,m(j)}: two
// chained products per block of 64 columns,
//     C = K U      (the key rows are exact in bf16, U as two bf16 parts),
//     dK += (C diag(c)) U^T    (C scaled and split into two bf16 parts in tensor memory; three products of the parts),
// so the edit is accurate to about 2^-17 of its size and no d x d projector is ever formed.  A step is 128 rows of one KV
// head.  In the stand-alone edit they are the next 128 highlighted tokens, wherever they lie (a list made by the launch
// before: only rows that change are read or written, and every CTA gets the same number of them); in the fused forward's
// preparation (SIDE) they are the rows of one 128-key tile that holds a highlighted token, and k' of all of them goes to the
// side buffer (rows of 2 D bf16: high parts [0, D), low parts [D, 2 D), the low parts only where the fused kernel reads them).
//
// The step is a chain (rows and U land, product, scale, product, add, write) that several CTAs per SM walk side by side; the
// rows of a CTA's next step are fetched under the present one where shared memory has room for a second stage.
// Registers and code are kept small (16 columns at a time, short unrolls): a preparation is often one or two steps per CTA, bound
// by fetching its instructions, and many spilled registers tripled the time of a step at head_dim 64.  The stand-alone edit, whose
// CTAs take many steps, has its loads, drain and writes unrolled at head_dim 128 (64 x 3000 tokens of 8 heads, all highlighted 216 ->
// 200 us); where they are very many, or U is wide, the gathering kernel below takes over (see gather_edit).
// Measured: one prompt of 777 tokens on 32/8 heads 42 -> 31 us per call of the fused forward (four launches and two memsets
// before, two launches now).
constexpr uint32_t EBLK = 128 * 128;        // one [128 x 64] bf16 block

// all lanes of a warp wait on the same barrier and then agree on the outcome
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status, int where) {
    const bool ok = mbar_wait(bar, parity, abort_flag, status, where);
    return __all_sync(0xffffffffu, ok);
}
constexpr int ET_THREADS = 256, ET_SMALL = 512;
constexpr int kMaxGatherHeads = 256;
constexpr int ET_UCOLS = 64, ET_UBLOCKS = 4;        // columns of U per block; most blocks that stay in shared memory

template <int D, bool SIDE, bool PACK = false>
struct EtSmem {
    static constexpr uint32_t TILE = (D / 64) * EBLK;       // 128 key rows
    static constexpr uint32_t UMAT = D * 128;               // [D x 64] bf16
    static constexpr int NS = D == 128 && SIDE ? 1 : 2;     // stages of key rows (two CTAs per SM leave room for one beside the low parts)
    static constexpr uint32_t U = NS * TILE;                // blocks of U (high part, then low part each); SIDE: then the low
                                                            // parts of the edited rows; then scratch and result of Eq. 6
    static constexpr uint32_t UBLK = PACK ? UMAT : 2 * UMAT;          // a block of U with its low part
    static constexpr uint32_t TMEM_COLS = D == 128 ? 256 : 128;       // 64 for C, D for dK
    static constexpr int CTAS = D == 128 ? 2 : PACK ? 4 : 3;          // per SM: tensor memory (shared memory for 64 unpacked)
};

// SIDE: a unit of work as the warp that looked at it left it
struct __align__(16) UnitInfo { uint32_t bits[4]; int work, b, tok0, nvalid; float c; int with_lo, h, pad; };

struct TileArgs {
    const void* K; __nv_bfloat16* out;
    const uint8_t* mask; const float* U; const float* alpha; const float* gain; const uint8_t* head_enable; const int* cu;
    const int* list; const int* seqs; const int* counts; int n_seg, seg_tokens;  // stand-alone edit: the highlighted tokens, their sequences
    uint8_t* tile_hot; uint8_t* bh_info;                                         // SIDE: written for the fused kernel
    int* status;
    int B, L, Hkv, r, M, n_tiles;
    int u_blocks;                           // blocks of U that stay in shared memory (all of them, or one that is replaced)
    int n_tile_blocks;                      // SIDE: item-table blocks | tile blocks | conversion blocks
    RouteArgs route;
    PrepJobs jobs;
};

// PACK (stacked rank of at most 32): both parts of U stand in one block, the low part from column 32 on, so that one product
// forms K times either part and both halves of the threads scale C.  Before / with it: 36 layers as above 74 -> 69 us, 64 x 4096
// tokens x 8 heads x 64, half highlighted, 96 -> 78 us (a fourth CTA per SM fits there).
//
// NTH = ET_SMALL: the preparation of a small launch, one step per CTA and one CTA per SM.  Its time is the chain's latency, so
// four threads share a row, and the rows, U and what tells whether the step has work are all asked for at once (one trip to
// memory instead of four; rows and U are wasted where the tile turns out not to be highlighted).  Before / with it, per call of
// the fused forward: one prompt of 777 tokens on 32/8 heads of 128 30.4 -> 28.3 us, 2 tiles x 4 heads of 64 in fp32 19.4 -> 16.1,
// 700 tokens with four routed experts 38 -> 34 (the step itself 19100 -> 12100 cycles in the first).
template <int D, bool SIDE, typename KT, bool PACK, int NTH>
__global__ void __launch_bounds__(NTH, NTH == ET_THREADS ? EtSmem<D, SIDE, PACK>::CTAS : 1)
edit_tiles_kernel(const __grid_constant__ TileArgs p) {
    constexpr bool SMALL = NTH == ET_SMALL;
    static_assert(!SMALL || (SIDE && !PACK), "the small form is one of the preparation");
    constexpr int NW = NTH / 32, PARTS = NTH / 128;     // warps; threads per row
    using SL = EtSmem<D, SIDE, PACK>;
    constexpr int NS = SL::NS;
    constexpr int UPR = D / 8;                          // 16-byte units (8 elements) of a key row
    constexpr int RPP = NTH / UPR;                      // rows a pass of the CTA loads
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Hkv = p.Hkv, r = p.r, M = p.M;
    const bool routed = SIDE && p.route.sigma != nullptr;
    int blk = blockIdx.x;
    if constexpr (SIDE) {
        if (blk < p.jobs.n_items_blocks) {
            pdl_wait();
            pdl_release();
            if (tid >= PREP_THREADS) return;
            items_block(p.jobs.sched, p.jobs.cu, p.jobs.steer, p.jobs.items, p.jobs.item_count, blk);
            return;
        }
        blk -= p.jobs.n_items_blocks;
        if (blk >= p.n_tile_blocks) {
            pdl_wait();
            pdl_release();
            convert_block(p.jobs.conv, blk - p.n_tile_blocks, p.jobs.n_conv_blocks);
            return;
        }
    }

    __shared__ __align__(8) uint64_t bars[2];           // C is ready, dK is ready
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_s;
    __shared__ int tok_s[2][SIDE ? 1 : 128], seq_s[2][SIDE ? 1 : 128];      // stand-alone: token (-1: none) and sequence of a row, per stage
    __shared__ float c_s[2][SIDE ? 1 : 128];            // stand-alone: gain (one expert: times its coefficient) of a row, per stage
    __shared__ UnitInfo look_s[NW];               // SIDE: the units looked at last
    __shared__ unsigned short exp_s[ET_UBLOCKS * ET_UCOLS];      // expert of a column of the blocks in shared memory
    __shared__ int pre_s[SIDE ? 1 : kMaxSegments + 1];  // stand-alone: highlighted tokens before each segment
    __shared__ int wsum_s[NW];
    volatile int* abort_flag = &abort_s;
    if (tid == 0) {
        mbar_init(bars, 1); mbar_init(bars + 1, 1);
        abort_s = 0;
        mbar_fence_init();
    }
    __syncwarp();
    if (warp == 0) { tmem_alloc(&tmem_holder, SL::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tC = tmem_holder, tD = tC + ET_UCOLS;
    pdl_wait();
    pdl_release();
    const int dead = *reinterpret_cast<volatile int*>(p.status);
    bool ok = SMALL || !__syncthreads_or(dead != 0);

    uint8_t* sU = smem + SL::U;
    constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
    const uint32_t dK0 = umma_desc_lo(smem_u32(smem), 16), dU0 = umma_desc_lo(smem_u32(sU), EBLK);
    const int row = tid & 127, part = tid >> 7;         // tensor-memory lane = key row, and which part of the columns
    const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
    const int R = r * M;
    const bool u_vec = (r & 7) == 0 && (reinterpret_cast<uintptr_t>(p.U) & 15) == 0;

    // ---------------------------------------------------- units of work
    // The unit taken last: head, sequence, first token, rows (SIDE), whether its low parts are wanted, the flags of this
    // thread's warp quarter, coefficient; stand-alone: chunk of the list.
    int cur_h = 0, cur_b = 0, cur_tok0 = 0, cur_nvalid = 0, cur_lo = 0, cur_chunk = 0;
    uint32_t cur_bits = 0;
    float cur_c = 0.f;
    int unit = blk, n_units = 0, n_hot = 0;
    int look_pos = NW;
    // SIDE: the CTAs take the tiles of all pairs (sequence, KV head) in turn; their number is a multiple of the KV heads, so that
    // a CTA keeps its head (and its blocks of U).  Routed: a CTA also keeps its pair, whose coefficients then serve all its
    // units: `per` CTAs share the tiles of a pair, or a CTA takes several pairs one after another.
    const int BH = p.B * Hkv, per = routed && p.n_tile_blocks >= BH ? p.n_tile_blocks / BH : 1;
    if constexpr (SIDE) {
        if (SMALL) n_units = 0;                         // (the only one is taken below)
        else if (!routed) n_units = (BH * p.n_tiles - blk + p.n_tile_blocks - 1) / p.n_tile_blocks;
        else if (p.n_tile_blocks >= BH) n_units = blk < per * BH ? (p.n_tiles - blk / BH + per - 1) / per : 0;
        else n_units = (BH - blk + p.n_tile_blocks - 1) / p.n_tile_blocks * p.n_tiles;
        unit = 0;                                       // units are counted per CTA
    } else if (ok) {
        // highlighted tokens before each segment, and in all
        constexpr int PT = kMaxSegments / NTH;
        int c[PT], sum = 0;
#pragma unroll
        for (int q = 0; q < PT; ++q) { c[q] = tid * PT + q < p.n_seg ? p.counts[tid * PT + q] : 0; sum += c[q]; }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) wsum_s[warp] = incl;
        __syncthreads();
        int base = incl - sum;
#pragma unroll
        for (int w = 0; w < NW; ++w) { if (w < warp) base += wsum_s[w]; n_hot += wsum_s[w]; }
#pragma unroll
        for (int q = 0; q < PT; ++q) { pre_s[tid * PT + q] = base; base += c[q]; }
        __syncthreads();
        n_units = ((n_hot + 127) / 128) * Hkv;
    }
    auto unit_pair = [&](int u, int& t) -> int {        // (SIDE) pair b * Hkv + h and tile of unit u of this CTA
        if (!routed) { const int v = blk + u * p.n_tile_blocks; t = v / BH; return v % BH; }
        if (p.n_tile_blocks >= BH) { t = blk / BH + u * per; return blk % BH; }
        t = u % p.n_tiles;
        return blk + u / p.n_tiles * p.n_tile_blocks;
    };

    // the next unit with work (false: none left); every thread gets the same answer
    auto next_unit = [&]() -> bool {
        if constexpr (!SIDE) {
            while (unit < n_units) {
                cur_chunk = unit / Hkv; cur_h = unit - cur_chunk * Hkv;
                unit = unit + (int)gridDim.x < unit ? 0x7fffffff : unit + (int)gridDim.x;
                if (p.head_enable == nullptr || p.head_enable[cur_h] != 0) return true;
            }
            return false;
        } else {
            while (true) {
                if (look_pos == NW) {             // a warp looks at each of the next units, one a warp: one latency for all of them
                    if (unit >= n_units) return false;
                    __syncthreads();
                    UnitInfo* info = look_s + warp;
                    if (unit + warp < n_units) {
                        int t;
                        const int bh = unit_pair(unit + warp, t), b = bh / Hkv, h = bh - b * Hkv;
                        const int seq0 = p.cu ? p.cu[b] : b * p.L;
                        const int Lb = (p.cu ? p.cu[b + 1] : (b + 1) * p.L) - seq0;
                        const float g = p.gain[b];
                        const bool on = p.head_enable == nullptr || p.head_enable[h] != 0;
                        const int sb = steer_byte(p.jobs.steer, b, h, Hkv);
                        uint32_t any = 0;
                        uint32_t bits[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int pos = t * 128 + q * 32 + lane;
                            bits[q] = __ballot_sync(0xffffffffu, pos < Lb && p.mask[seq0 + pos] != 0);
                            any |= bits[q];
                        }
                        if (lane == 0) {
                            *reinterpret_cast<uint4*>(info->bits) = make_uint4(bits[0], bits[1], bits[2], bits[3]);
                            info->work = (any != 0 && on && g != 0.f) ? 1 : 0;
                            info->b = b; info->h = h; info->tok0 = seq0 + t * 128; info->nvalid = Lb - t * 128 < 128 ? Lb - t * 128 : 128;
                            info->c = g * (M == 1 && p.alpha != nullptr && !routed ? p.alpha[(size_t)b * Hkv + h] : 1.f);
                            info->with_lo = (t < kLoTiles || (sb & 2) != 0) ? 1 : 0;
                        }
                        if (h == 0) {                   // what the fused kernel needs to know
                            if (lane == 0) p.tile_hot[(size_t)b * p.n_tiles + t] = any != 0 ? 1 : 0;
                            if (t == 0)
                                for (int hh = lane; hh < Hkv; hh += 32) p.bh_info[(size_t)b * Hkv + hh] = (uint8_t)steer_byte(p.jobs.steer, b, hh, Hkv);
                        }
                    } else if (lane == 0) {
                        info->work = 0;
                    }
                    __syncthreads();
                    look_pos = 0;
                }
                while (look_pos < NW) {
                    ++unit;
                    const UnitInfo& info = look_s[look_pos++];
                    if (info.work) {
                        cur_h = info.h;
                        cur_b = info.b; cur_tok0 = info.tok0; cur_nvalid = info.nvalid; cur_lo = info.with_lo; cur_c = info.c;
                        cur_bits = info.bits[row >> 5];
                        return true;
                    }
                }
            }
        }
    };
    // rows of the unit (stand-alone): the chunk's tokens, looked up in the segments (visible after the next barrier)
    auto find_rows = [&](int st) {
        if constexpr (!SIDE) {
            if (tid >= 128) return;
            const int q = cur_chunk * 128 + tid;
            int tok = -1, b = 0;
            float c = 0.f;
            if (q < n_hot) {
                int lo = 0, hi = p.n_seg - 1;           // largest segment with pre_s[seg] <= q (an empty one is never the largest)
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (pre_s[mid] <= q) lo = mid; else hi = mid - 1;
                }
                tok = p.list[(size_t)lo * p.seg_tokens + (q - pre_s[lo])];
                b = find_sequence(p.cu, p.B, p.L, tok);
                c = p.gain[b] * (M == 1 && p.alpha != nullptr ? p.alpha[(size_t)b * Hkv + cur_h] : 1.f);
            }
            tok_s[st][tid] = tok; seq_s[st][tid] = b; c_s[st][tid] = c;
        }
    };
    // the unit's key rows on their way into stage st (128-byte swizzle; rows that do not exist are zero)
    auto load_rows = [&](int st) {
        const int c = tid % UPR;
        const uint32_t base = smem_u32(smem) + st * SL::TILE + (c >> 3) * EBLK;
#pragma unroll (SIDE ? 2 : D == 128 ? 8 : 2)
        for (int k = 0; k < 128 / RPP; ++k) {
            const int rr = tid / UPR + k * RPP;
            const int tok = SIDE ? cur_tok0 + rr : tok_s[st][SIDE ? 0 : rr];
            const bool valid = SIDE ? rr < cur_nvalid : tok >= 0;
            const size_t e = ((size_t)(valid ? tok : 0) * Hkv + cur_h) * D + c * 8;
            const uint32_t dst = base + sw128_offset(rr, (c & 7) * 8);
            if (sizeof(KT) == 2) {
                cp_async16(dst, static_cast<const __nv_bfloat16*>(p.K) + e, valid);
            } else {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b4 = a;
                if (valid) {
                    a = *reinterpret_cast<const float4*>(static_cast<const float*>(p.K) + e);
                    b4 = *reinterpret_cast<const float4*>(static_cast<const float*>(p.K) + e + 4);
                }
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(pack_bf16(a.x, a.y)), "r"(pack_bf16(a.z, a.w)),
                             "r"(pack_bf16(b4.x, b4.y)), "r"(pack_bf16(b4.z, b4.w)) : "memory");
            }
        }
    };
    // columns [j0, j0 + 64) of the stacked U of head h as two bf16 parts: [D x 64] blocks, 128-byte swizzle (K-major operand of
    // the second product, MN-major of the first); zero up to the next multiple of 16 columns, undefined (and unused) beyond
    auto stage_u = [&](int h, int j0, int slot) {
        uint8_t* sB = sU + slot * SL::UBLK;
        const int rc = R - j0 < ET_UCOLS ? R - j0 : ET_UCOLS, nu = (rc + 15) / 16 * 2;
        if (u_vec) {
#pragma unroll 1
            for (int u = tid; u < D * nu; u += NTH) {
                const int i = u / nu, c8 = (u - i * nu) * 8;
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b4 = a;
                if (j0 + c8 < R) {                          // (rank a multiple of 8: eight columns of one expert)
                    const int m = M == 1 ? 0 : (j0 + c8) / r, k = j0 + c8 - m * r;
                    const float4* src = reinterpret_cast<const float4*>(p.U + (((size_t)m * Hkv + h) * D + i) * r + k);
                    a = __ldg(src); b4 = __ldg(src + 1);
                }
                uint32_t hi[4], lo[4];
                split_pair(a.x, a.y, hi[0], lo[0]); split_pair(a.z, a.w, hi[1], lo[1]);
                split_pair(b4.x, b4.y, hi[2], lo[2]); split_pair(b4.z, b4.w, hi[3], lo[3]);
                *reinterpret_cast<uint4*>(sB + sw128_offset(i, c8)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(PACK ? sB + sw128_offset(i, c8 + 32) : sB + SL::UMAT + sw128_offset(i, c8)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
        } else {
#pragma unroll 1
            for (int u = tid; u < D * nu * 4; u += NTH) {        // two columns at a time
                const int i = u / (nu * 4), c2 = (u - i * (nu * 4)) * 2, j = j0 + c2, m0 = j / r, m1 = (j + 1) / r;
                const float x = j < R ? __ldg(p.U + (((size_t)m0 * Hkv + h) * D + i) * r + (j - m0 * r)) : 0.f;
                const float y = j + 1 < R ? __ldg(p.U + (((size_t)m1 * Hkv + h) * D + i) * r + (j + 1 - m1 * r)) : 0.f;
                uint32_t hi, lo;
                split_pair(x, y, hi, lo);
                *reinterpret_cast<uint32_t*>(sB + sw128_offset(i, c2)) = hi;
                *reinterpret_cast<uint32_t*>(PACK ? sB + sw128_offset(i, c2 + 32) : sB + SL::UMAT + sw128_offset(i, c2)) = lo;
            }
        }
        if (tid < ET_UCOLS) exp_s[slot * ET_UCOLS + tid] = (unsigned short)(j0 + tid < R ? (j0 + tid) / r : M - 1);
    };

    int st = 0, u_head = -1, routed_for = -1;           // stage, head whose only block of U is resident, (sequence, head) of the coefficients
    uint32_t n_c = 0, n_d = 0;                          // products so far (phases)
    const bool resident = R <= ET_UCOLS * p.u_blocks;
    uint8_t* sL = smem + SL::U + p.u_blocks * SL::UBLK;
    float* alpha_r = reinterpret_cast<float*>(sL + (SIDE ? SL::TILE : 0));
    // Eq. 6 of a pair b * Hkv + h into alpha_r (the scratch starts behind the result)
    auto route_pair = [&](int bh) {
        double* sm = reinterpret_cast<double*>(reinterpret_cast<uint8_t*>(alpha_r) + ((M * 4 + 15) & ~15));
        const double* a = route_group(p.route.Q, p.route.q_is_f32, p.U, p.route.sigma, p.cu, p.L, p.route.Hq, Hkv, D, r, M,
                                      p.route.k_route, bh / Hkv, bh % Hkv, sm);
        for (int m = tid; m < M; m += NTH) alpha_r[m] = (float)a[m];
        routed_for = bh;
    };
    bool have = false;
    if constexpr (SMALL) {
        const int t = blk / BH, bh = blk % BH;
        cur_b = bh / Hkv; cur_h = bh - cur_b * Hkv;
        const int seq0 = p.cu ? p.cu[cur_b] : cur_b * p.L;
        const int Lb = (p.cu ? p.cu[cur_b + 1] : (cur_b + 1) * p.L) - seq0;
        cur_tok0 = seq0 + t * 128; cur_nvalid = Lb - t * 128 < 128 ? Lb - t * 128 : 128;
        load_rows(0);
        const int m = row < cur_nvalid ? p.mask[cur_tok0 + row] : 0;
        const float g = p.gain[cur_b];
        const int on = p.head_enable == nullptr ? 1 : p.head_enable[cur_h];
        const bool one = M == 1 && p.alpha != nullptr && !routed;
        const float a1 = one ? p.alpha[bh] : 1.f;
        if (resident) {
            for (int j0 = 0; j0 < R; j0 += ET_UCOLS) stage_u(cur_h, j0, j0 / ET_UCOLS);
            u_head = cur_h;
        }
        const float amax = one ? fabsf(a1) : routed ? 1.f : alpha_max_of(p.alpha, (size_t)bh, M);       // (as in steer_byte)
        cur_c = g * a1;
        cur_lo = t < kLoTiles || lo_needed(g, amax);
        cur_bits = __ballot_sync(0xffffffffu, m != 0);
        if (lane == 0) wsum_s[warp] = cur_bits != 0;
        ok = !__syncthreads_or(dead != 0);
        const int any = wsum_s[0] | wsum_s[1] | wsum_s[2] | wsum_s[3];
        if (cur_h == 0) {                               // what the fused kernel needs to know
            if (tid == 0) p.tile_hot[(size_t)cur_b * p.n_tiles + t] = any != 0 ? 1 : 0;
            if (t == 0)
                for (int hh = tid; hh < Hkv; hh += NTH) p.bh_info[(size_t)cur_b * Hkv + hh] = (uint8_t)steer_byte(p.jobs.steer, cur_b, hh, Hkv);
        }
        have = ok && any && on && g != 0.f;
    }
    if (routed && ok && p.route.alpha_out != nullptr && blk < BH) {
        // the first CTA of a pair leaves its coefficients for the caller
        for (int bh = blk; bh < BH; bh += p.n_tile_blocks) {
            route_pair(bh);
            __syncthreads();
            for (int m = tid; m < M; m += NTH) p.route.alpha_out[(size_t)bh * M + m] = alpha_r[m];
        }
    }
    if constexpr (!SMALL) {
        have = ok && next_unit();
        if (have) {
            if (!SIDE) { find_rows(0); __syncthreads(); }
            load_rows(0);
        }
    }
    while (have) {
        const int h = cur_h, b = cur_b, tok0 = cur_tok0, nvalid = cur_nvalid;
        const bool with_lo = SIDE && cur_lo != 0;
        if (u_head != h) {
            for (int j0 = 0; j0 == 0 || (resident && j0 < R); j0 += ET_UCOLS) stage_u(h, j0, j0 / ET_UCOLS);
            u_head = resident ? h : -1;
        }
        const bool read_back = routed && BH > p.n_tile_blocks && p.route.alpha_out != nullptr;      // written by this CTA above
        if (routed && !read_back && routed_for != b * Hkv + h) route_pair(b * Hkv + h);
        cp_async_wait_all();
        fence_proxy_async();
        __syncthreads();                                // rows and U are in place
        bool have_next = false;
        const bool hl = SIDE ? ((cur_bits >> (row & 31)) & 1u) != 0 : tok_s[st][SIDE ? 0 : row] >= 0;
        const float g = SIDE ? cur_c : c_s[st][SIDE ? 0 : row];
        const int b_row = SIDE ? b : seq_s[st][SIDE ? 0 : row];
        const bool warp_hl = __any_sync(0xffffffffu, hl);
        for (int j0 = 0; j0 < R; j0 += ET_UCOLS) {
            const int rc = R - j0 < ET_UCOLS ? R - j0 : ET_UCOLS, nks = (rc + 15) / 16;
            if (j0 > 0 && !resident) { stage_u(h, j0, 0); fence_proxy_async(); __syncthreads(); }
            const int slot = resident ? j0 / ET_UCOLS : 0;
            const uint32_t dU = dU0 + slot * (SL::UBLK >> 4);
            const int jh = part * (PACK ? 16 : 64 / PARTS);         // first column of this part of the threads
            const unsigned short* ex = exp_s + slot * ET_UCOLS + jh;
            if (tid == 0) {
                tc_fence_after();
                const uint32_t kd = dK0 + st * (SL::TILE >> 4);
                constexpr uint32_t IDESC = umma_idesc_bf16(ET_UCOLS, true);
#pragma unroll 1
                for (int pb = 0; pb < (PACK ? 1 : 2) * (D / 64); ++pb) {        // part of U (packed: both side by side), 64 dimensions
                    const uint32_t kb = kd + (uint32_t)(pb % (D / 64)) * (EBLK >> 4);
                    const uint32_t ub = dU + (((uint32_t)(pb / (D / 64)) * SL::UMAT + (uint32_t)(pb % (D / 64)) * 8192) >> 4);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        umma_ss(tC, kb + (uint32_t)(ks * 32 >> 4), DESC_HI, ub + (uint32_t)(ks * 2048 >> 4), DESC_HI, IDESC, (ks > 0 || pb > 0) ? 1u : 0u);
                }
                umma_commit(bars);
            }
            if (j0 == 0) {                              // under the product: what comes next
                have_next = next_unit();
                if (have_next) find_rows(st ^ 1);
            }
            ok = mbar_wait(bars, n_c & 1, abort_flag, p.status, 60);
            ++n_c;
            ok = __all_sync(0xffffffffu, ok);
            if (ok && warp_hl && jh < rc) {
                // C times the row's coefficients, split, back over itself; what the rows that are not highlighted get is never used
                tc_fence_after();
                const uint32_t tc = tC + lane_off + jh;
                const float* a_row = read_back ? p.route.alpha_out + (size_t)(b * Hkv + h) * M : routed ? alpha_r : (M > 1 && p.alpha != nullptr ? p.alpha + ((size_t)b_row * Hkv + h) * M : nullptr);
                // (16 columns at a time: few registers and little code, most launches make one or two steps and are bound by
                // fetching their instructions)
#pragma unroll 1
                for (int q = 0; q < (PACK ? 1 : 4 / PARTS) && jh + q * 16 < rc; ++q) {
                    uint32_t v[16], hl8[8];
                    tmem_ld16(tc + q * 16, v);
                    float ca = g, cb = g;
                    if (a_row != nullptr && (r & 7) == 0) { ca *= a_row[ex[q * 16]]; cb *= a_row[ex[q * 16 + 8]]; }
                    tmem_wait_ld_on16(v);
                    if constexpr (PACK) {           // K times the low part
                        uint32_t v2[16];
                        tmem_ld16(tc + 32, v2);
                        tmem_wait_ld_on16(v2);
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(v2[e]));
                    }
                    if (a_row != nullptr && (r & 7) != 0) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * a_row[ex[q * 16 + e]]);
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e) split_pair(__uint_as_float(v[2 * e]) * (e < 4 ? ca : cb), __uint_as_float(v[2 * e + 1]) * (e < 4 ? ca : cb), v[e], hl8[e]);
                    // a 16-column operand block: high pairs in its first eight columns, low pairs in the others
                    tmem_st8(tc + q * 16, v);
                    tmem_st8(tc + q * 16 + 8, hl8);
                }
                tmem_wait_st();
            }
            tc_fence_before();
            ok = __syncthreads_and(ok);
            if (!ok) break;
            if (tid == 0) {
                tc_fence_after();
                constexpr uint32_t IDESC = umma_idesc_bf16(D, false);
#pragma unroll 1
                for (int ks = 0; ks < nks; ++ks) {
                    const uint32_t a_hi = tC + (uint32_t)ks * 16, a_lo = a_hi + 8;
                    const uint32_t u_hi = dU + (((uint32_t)ks * 32) >> 4), u_lo = u_hi + ((PACK ? 64 : SL::UMAT) >> 4);
                    umma_ts(tD, a_hi, u_hi, DESC_HI, IDESC, (j0 > 0 || ks > 0) ? 1u : 0u);
                    umma_ts(tD, a_lo, u_hi, DESC_HI, IDESC, 1u);
                    umma_ts(tD, a_hi, u_lo, DESC_HI, IDESC, 1u);
                }
                umma_commit(bars + 1);
            }
            if (NS == 2 && j0 == 0 && have_next) load_rows(st ^ 1);
            ok = mbar_wait(bars + 1, n_d & 1, abort_flag, p.status, 61);
            ++n_d;
            ok = __all_sync(0xffffffffu, ok);
            if (!resident) { ok = __syncthreads_and(ok); if (!ok) break; }      // (U is replaced next)
        }
        if (!ok && !resident) break;
        uint8_t* sK = smem + st * SL::TILE;
        if (ok && (warp_hl || with_lo)) {
            // k' = k + dK[row] for highlighted rows, 1 / PARTS of a row per thread, in place in the staged rows; low parts beside them
            tc_fence_after();
#pragma unroll (SIDE ? 1 : D == 128 ? 4 : 2)
            for (int c = part * (D / 16 / PARTS); c < (part + 1) * (D / 16 / PARTS); ++c) {      // 16 columns
                uint32_t v[16];
                if (warp_hl) { tmem_ld16(tD + lane_off + c * 16, v); tmem_wait_ld_on16(v); }     // warp-wide: every lane takes part
#pragma unroll
                for (int q = 0; q < 2; ++q) {          // 8 elements = one 16-byte unit of the swizzled row
                    const uint32_t off = (uint32_t)((c * 16) >> 6) * EBLK + sw128_offset(row, ((c * 16) & 63) + q * 8);
                    uint4 l = make_uint4(0u, 0u, 0u, 0u);
                    if (hl) {
                        uint4 kv = *reinterpret_cast<uint4*>(sK + off);
                        uint32_t* w = reinterpret_cast<uint32_t*>(&kv);
                        uint32_t* lw = reinterpret_cast<uint32_t*>(&l);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 k2 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w[e]));
                            const float x0 = k2.x + __uint_as_float(v[q * 8 + 2 * e]), x1 = k2.y + __uint_as_float(v[q * 8 + 2 * e + 1]);
                            if (SIDE) split_pair(x0, x1, w[e], lw[e]); else w[e] = pack_bf16(x0, x1);
                        }
                        *reinterpret_cast<uint4*>(sK + off) = kv;
                    }
                    if (with_lo) *reinterpret_cast<uint4*>(sL + off) = l;
                }
                __syncwarp();      // all lanes together again before the next warp-wide load
            }
        }
        tc_fence_before();
        ok = __syncthreads_and(ok);
        if (!ok) break;
        // write the rows out: D / 8 lanes per row, 16 bytes each
#pragma unroll (SMALL ? 4 : SIDE ? 2 : D == 128 ? 8 : 2)
        for (int k = 0; k < 128 / RPP; ++k) {
            const int rr = tid / UPR + k * RPP, c = tid % UPR;
            const int tok = SIDE ? tok0 + rr : tok_s[st][SIDE ? 0 : rr];
            if (SIDE ? rr < nvalid : tok >= 0) {
                const uint32_t off = (uint32_t)(c >> 3) * EBLK + sw128_offset(rr, (c & 7) * 8);
                __nv_bfloat16* dst = p.out + ((size_t)tok * Hkv + h) * (SIDE ? 2 * D : D) + c * 8;
                *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(sK + off);
                if (with_lo) *reinterpret_cast<uint4*>(dst + D) = *reinterpret_cast<const uint4*>(sL + off);
            }
        }
        have = have_next;
        if (NS == 2) {
            st ^= 1;                   // (this stage and the low parts are written again behind two barriers of the next step)
        } else if (have) {
            __syncthreads();
            load_rows(0);
        }
    }
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tC, SL::TMEM_COLS);
}

// A 32 x 32 tile of P = U U^T of one (expert, KV head), two bf16 parts: P = hi + lo to about 2^-17, so that the edit keeps
// fp32-like accuracy on bf16 tensor cores.  Blocks of PREP_THREADS threads, (D / 32)^2 per matrix; the high parts of all matrices
// come first, then the low parts.  Bound by one trip to memory per 64 columns of U.
__device__ __forceinline__ void projector_block(const float* __restrict__ U, __nv_bfloat16* __restrict__ P, int blk, int n_mats, int D, int r) {
    const int tid = threadIdx.x, tiles = D / 32;
    const int mat = blk / (tiles * tiles), t = blk % (tiles * tiles);
    const int i0 = (t / tiles) * 32, j0 = (t % tiles) * 32;
    constexpr int KC = 64, LD = KC + 4;                     // columns of U at a time; float4 reads of 8 rows meet 32 banks
    __shared__ __align__(16) float ui[32][LD], uj[32][LD];
    const int tx = tid & 31, ty = tid >> 5;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    const float* Um = U + (size_t)mat * D * r;
    for (int k0 = 0; k0 < r; k0 += KC) {
        const int rc = r - k0 < KC ? r - k0 : KC;
        float a[2][4], b[2][4];                             // all loads of the chunk in flight together
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = c * 32 + tx;
                a[c][q] = k < rc ? Um[(size_t)(i0 + ty + 8 * q) * r + k0 + k] : 0.f;
                b[c][q] = k < rc ? Um[(size_t)(j0 + ty + 8 * q) * r + k0 + k] : 0.f;
            }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) { ui[ty + 8 * q][c * 32 + tx] = a[c][q]; uj[ty + 8 * q][c * 32 + tx] = b[c][q]; }
        __syncthreads();
        const int kn = (rc + 3) & ~3;
#pragma unroll 4
        for (int k = 0; k < kn; k += 4) {
            const float4 y = *reinterpret_cast<const float4*>(&uj[tx][k]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 x = *reinterpret_cast<const float4*>(&ui[ty + 8 * q][k]);
                acc[q] = fmaf(x.x, y.x, acc[q]); acc[q] = fmaf(x.y, y.y, acc[q]);
                acc[q] = fmaf(x.z, y.z, acc[q]); acc[q] = fmaf(x.w, y.w, acc[q]);
            }
        }
    }
    __nv_bfloat16* Phi = P + (size_t)mat * D * D;
    __nv_bfloat16* Plo = P + ((size_t)n_mats + mat) * D * D;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(acc[q]);
        Phi[(size_t)(i0 + ty + 8 * q) * D + j0 + tx] = hi;
        Plo[(size_t)(i0 + ty + 8 * q) * D + j0 + tx] = __float2bfloat16_rn(acc[q] - __bfloat162float(hi));
    }
}

// List of the highlighted tokens (of sequences with a gain), a block per segment of consecutive tokens; with a second output
// tensor further blocks copy the keys meanwhile (the rows that change are overwritten by the launch behind); the last n_p blocks
// form the projectors that the gathering kernel reads.
template <bool PROJ>
__global__ void __launch_bounds__(PREP_THREADS)
edit_scan_kernel(const uint8_t* __restrict__ mask, const float* __restrict__ gain, const int* __restrict__ cu, int T, int B, int L,
                 int* __restrict__ list, int* __restrict__ seqs, int* __restrict__ counts, int seg_tokens, int n_seg, const uint4* __restrict__ src,
                 uint4* __restrict__ dst, size_t n16, const float* __restrict__ U, __nv_bfloat16* __restrict__ P, int n_p, int n_mats, int D, int r) {
    pdl_wait();
    pdl_release();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if constexpr (PROJ) {
        if ((int)blockIdx.x >= (int)gridDim.x - n_p) {
            projector_block(U, P, (int)blockIdx.x - ((int)gridDim.x - n_p), n_mats, D, r);
            return;
        }
    }
    if ((int)blockIdx.x >= n_seg) {
        const size_t step = (size_t)(gridDim.x - n_p - n_seg) * 256;
        for (size_t i0 = (size_t)(blockIdx.x - n_seg) * 256 + tid; i0 < n16; i0 += 4 * step) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q * step < n16) v[q] = src[i0 + q * step];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i0 + q * step < n16) dst[i0 + q * step] = v[q];
        }
        return;
    }
    __shared__ int wsum[8];
    const int s0 = blockIdx.x * seg_tokens;
    int* out = list + s0;
    int total = 0;
    for (int t0 = s0; t0 < s0 + seg_tokens && t0 < T; t0 += 1024) {        // 1024 tokens a round, four per thread
        const int t = t0 + tid * 4;
        unsigned bits = 0;
        int seq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) bits |= (t + q < T && mask[t + q] != 0) ? 1u << q : 0u;
        if (bits != 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if ((bits >> q) & 1u) {
                    seq[q] = find_sequence(cu, B, L, t + q);
                    if (gain[seq[q]] == 0.f) bits &= ~(1u << q);
                }
        }
        const int cnt = __popc(bits);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int base = total + incl - cnt;
#pragma unroll
        for (int w = 0; w < 8; ++w) { if (w < warp) base += wsum[w]; total += wsum[w]; }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if ((bits >> q) & 1u) { seqs[s0 + base] = seq[q]; out[base++] = t + q; }
        __syncthreads();
    }
    if (tid == 0) counts[blockIdx.x] = total;
}

// ---------------------------------------------------------------- many rows or wide banks: gathered rows through projectors
//
// Where the chain above has many steps, or its stacked rank is wide, the edit is a pipeline over the same list of highlighted
// tokens, one CTA per SM with a KV head of its own, from projectors P_m = U_m U_m^T in two bf16 parts.  One expert's projector is
// formed by the CTA itself, on the tensor cores, while its first rows are on their way (by blocks of the launch before it cost
// small edits 4 to 6 us); those of several (MULTI) come from that launch:
//   warps 17 ..  producers, one per shared-memory stage: each brings every NS-th 128-row step of the CTA into its stage by TMA (one
//                box where the tokens are consecutive, four rows an instruction otherwise), the rows' tokens and coefficients
//                beside it; the look-up of its next step runs under the product and the drain of this one;
//   warp 16      MMA issuer: K P_m (two bf16 parts) into a ring of sets of tensor-memory columns; with more experts than
//                projectors fit (MULTI), it also brings the next ones in;
//   warps 0-15   drain: 32 columns of a row per thread (at head_dim 64 two groups of warps take every other step),
//                k' = k + sum_m c_m (K P_m)[row] in place in the stage, then the warp writes the pieces of its own 32 rows, 16
//                bytes per lane (no barrier among the warps).
// What a step costs does not depend on the rank.  Bound at head_dim 128 by shared memory (operands, rows in and out: 60 % of its
// bandwidth, which stretches every access to it), at 64 by the pace at which one thread issues products (about 130 cycles each).
// 144 x 4096 tokens x 8 heads x 128 in place, a tenth / all highlighted: whole tiles through a projector 96 / 561-590 us, the chain
// 68.5 / 600-619, this 61.5 / 529-546 (4.5 TB/s).  On the way: rows fetched by 16-byte asynchronous copies instead of TMA 100 us more (a
// step's 64 instructions held a warp for 5000 cycles), a look-up by binary search per row 40 more, eight drain warps 50 more.
template <int D, bool MULTI>
struct EgSmem {
    static constexpr uint32_t TILE = (D / 64) * EBLK;
    static constexpr uint32_t PBLK = D * 128;
    static constexpr uint32_t PMAT = (D / 64) * PBLK;
    static constexpr int NS = D == 128 ? (MULTI ? 2 : 4) : (MULTI ? 6 : 8);        // stages of key rows, a producer warp each
    static constexpr int NP = MULTI ? (D == 128 ? 2 : 4) : 1;                       // projectors in shared memory
    static constexpr int NSET = 512 / D;
    static constexpr int WPT = D / 8, GROUPS = 16 / WPT;                            // drain warps of a step, of 16 in all; groups of them
    static constexpr int GSET = NSET / GROUPS;                                      // sets of columns of a group
    static constexpr int THREADS = (17 + NS) * 32;
    static constexpr uint32_t K = 0;
    static constexpr uint32_t P = K + NS * TILE;                                    // high part, then low part of each
    static constexpr uint32_t META = P + NP * 2 * PMAT;                             // per stage: token, coefficient, sequence of a row
    static constexpr uint32_t META_BYTES = 128 * 12;
    static constexpr uint32_t BARS = META + NS * META_BYTES;        // full[NS], free[NS], done[NSET], cols[NSET], p_full[NP], drain, u_full, p_mma
    static constexpr uint32_t NBARS = 2 * NS + 2 * NSET + NP + 3;
    static constexpr uint32_t MISC = BARS + NBARS * 8;
    static constexpr uint32_t DYN_BYTES = MISC + 16 + 1024;
    static_assert(NS % GROUPS == 0, "a stage belongs to one group of drain warps");
};

template <int D, bool MULTI>
__global__ void __launch_bounds__(EgSmem<D, MULTI>::THREADS, 1)
edit_gather_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmP,
                   const __grid_constant__ TileArgs p) {
    using SL = EgSmem<D, MULTI>;
    constexpr int NS = SL::NS, NP = SL::NP, NSET = SL::NSET, GROUPS = SL::GROUPS, GSET = SL::GSET, NBLK = D / 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + SL::BARS);      // [NS]  rows, tokens and coefficients of a step are in place
    uint64_t* freeb = full + NS;               // [NS]    WPT drain-warp arrivals: the stage may be refilled
    uint64_t* done = freeb + NS;               // [NSET]  a product is in its columns
    uint64_t* cols = done + NSET;              // [NSET]  WPT drain-warp arrivals: the columns have been read
    uint64_t* p_full = cols + NSET;            // [NP]    projector in place (MULTI: TMA bytes; else 16 drain-warp arrivals)
    uint64_t* drain = p_full + NP;             // [1]     (teardown after an abort) every product issued has finished
    uint64_t* u_full = drain + 1;              // [1]     (one expert) 16 drain-warp arrivals: both parts of U are staged
    uint64_t* p_mma = u_full + 1;              // [1]     (one expert) U U^T is in the first set of columns
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + SL::MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SL::MISC + 4);
    __shared__ int pre_s[kMaxSegments];        // highlighted tokens before each segment
    __shared__ int wsum_s[8];
    __shared__ unsigned short on_s[kMaxGatherHeads];   // enabled heads
    __shared__ int n_on_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Hkv = p.Hkv, M = MULTI ? p.M : 1;
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) { mbar_init(full + i, 2); mbar_init(freeb + i, SL::WPT); }
        for (int i = 0; i < NSET; ++i) { mbar_init(done + i, 1); mbar_init(cols + i, SL::WPT); }
        for (int i = 0; i < NP; ++i) mbar_init(p_full + i, MULTI ? 1 : 16);
        mbar_init(drain, 1); mbar_init(u_full, 16); mbar_init(p_mma, 1);
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmT);
        if (MULTI) tma_prefetch_desc(&tmP);
    }
    __syncwarp();
    if (warp == 0) { tmem_alloc(tmem_holder, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();
    pdl_release();
    // The first reads make one trip to memory together: the status, the counts of the list, the enabled heads and, where all are
    // enabled (the CTA's head is known), this thread's first piece of U.
    const int dead_word = *reinterpret_cast<volatile int*>(p.status);
    const int nu = (p.r + 15) / 16 * 2;        // 8-column units of a row of U (zero up to the next multiple of 16 columns)
    const bool u_vec = (p.r & 7) == 0 && (reinterpret_cast<uintptr_t>(p.U) & 15) == 0;
    auto load_u = [&](int head, int u, float (&f)[8]) {
        const int i = u / nu, c8 = (u - i * nu) * 8;
        const float* src = p.U + ((size_t)head * D + i) * p.r + c8;
        if (u_vec) {
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 a = c8 < p.r ? __ldg(reinterpret_cast<const float4*>(src)) : z, b = c8 < p.r ? __ldg(reinterpret_cast<const float4*>(src) + 1) : z;
            f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = c8 + e < p.r ? __ldg(src + e) : 0.f;
        }
    };
    float u_first[8];
    const bool u_early = !MULTI && p.head_enable == nullptr && tid < 512 && tid < D * nu;
    if (u_early) load_u((int)blockIdx.x % Hkv, tid, u_first);

    // highlighted tokens before each segment, and in all; enabled heads
    constexpr int PT = kMaxSegments / 256;
    int c[PT], sum = 0, incl = 0, n_hot = 0;
    if (tid < 256) {
#pragma unroll
        for (int q = 0; q < PT; ++q) { c[q] = tid * PT + q < p.n_seg ? p.counts[tid * PT + q] : 0; sum += c[q]; }
        incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
        if (lane == 31) wsum_s[warp] = incl;
    } else if (warp == 16) {
        int n = 0;
        for (int h0 = 0; h0 < Hkv; h0 += 32) {
            const bool on = h0 + lane < Hkv && (p.head_enable == nullptr || p.head_enable[h0 + lane] != 0);
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            if (on) on_s[n + __popc(bal & ((1u << lane) - 1))] = (unsigned short)(h0 + lane);
            n += __popc(bal);
        }
        if (lane == 0) n_on_s = n;
    }
    const bool dead = __syncthreads_or(dead_word != 0);
#pragma unroll
    for (int w = 0; w < 8; ++w) n_hot += wsum_s[w];
    if (tid < 256) {
        int base = incl - sum;
#pragma unroll
        for (int w = 0; w < 8; ++w) if (w < warp) base += wsum_s[w];
#pragma unroll
        for (int q = 0; q < PT; ++q) { pre_s[tid * PT + q] = base; base += c[q]; }
    }
    __syncthreads();
    // Product m of step i stands in the columns set_of(i, m): every group of drain warps has sets of its own, so that it sees each
    // phase of their barriers (a parity wait cannot tell a phase from the one two later).
    auto nth_of = [&](int i, int m) -> int { return i / GROUPS * M + m; };
    auto set_of = [&](int i, int m) -> int { return i % GROUPS * GSET + nth_of(i, m) % GSET; };
    auto phase_of = [&](int i, int m) -> uint32_t { return (uint32_t)(nth_of(i, m) / GSET) & 1u; };
    // this CTA: every `step`-th chunk of 128 listed tokens of one enabled head
    const int n_on = n_on_s, n_chunks = (n_hot + 127) / 128;
    int h = 0, c0 = 0, step = 1, n_my = 0;
    if (n_on > 0 && !dead) {
        const int hi = (int)blockIdx.x % n_on;
        h = on_s[hi]; c0 = (int)blockIdx.x / n_on; step = ((int)gridDim.x - hi + n_on - 1) / n_on;
        n_my = c0 < n_chunks ? (n_chunks - c0 + step - 1) / step : 0;
    }

    if (warp > 16) {
        // ------------------------------------------------------------ producers
        // rows 4 lane .. 4 lane + 3 of a step: token (-1: none), sequence, coefficient
        int tok[4], seq[4];
        float cf[4];
        auto look = [&](int i) {
            const int q0 = (c0 + i * step) * 128, q = q0 + 4 * lane;           // (q0 < n_hot)
            // largest segment with pre_s[seg] <= q0 (an empty one is never the largest): among every 32nd, then among the 32
            const int blk = 32 * (__popc(__ballot_sync(0xffffffffu, 32 * lane < p.n_seg && pre_s[32 * lane] <= q0)) - 1);
            const int lo = blk + __popc(__ballot_sync(0xffffffffu, blk + lane < p.n_seg && pre_s[blk + lane] <= q0)) - 1;
            const int base = pre_s[lo];
            int pos[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) pos[e] = lo * p.seg_tokens + q + e - base;
            // the segments that begin inside the step
            for (int s0 = lo + 1; s0 < p.n_seg; s0 += 32) {
                const int w = s0 + lane < p.n_seg ? pre_s[s0 + lane] : 0x7fffffff;
                const int n = __popc(__ballot_sync(0xffffffffu, w < q0 + 128));
                for (int k = 0; k < n; ++k) {
                    const int first = __shfl_sync(0xffffffffu, w, k);
#pragma unroll
                    for (int e = 0; e < 4; ++e) pos[e] = q + e >= first ? (s0 + k) * p.seg_tokens + q + e - first : pos[e];
                }
                if (n < 32) break;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                tok[e] = -1; seq[e] = 0;
                if (q + e < n_hot) { tok[e] = p.list[pos[e]]; seq[e] = p.seqs[pos[e]]; }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) cf[e] = p.gain[seq[e]];
            if (!MULTI && p.alpha != nullptr) {
#pragma unroll
                for (int e = 0; e < 4; ++e) cf[e] *= p.alpha[(size_t)seq[e] * Hkv + h];
            }
        };
        int i = warp - 17;
        const int s = i;                       // this producer's stage
        if (i < n_my) look(i);
        for (; i < n_my; i += NS) {
            if (i >= NS && !warp_wait(freeb + s, ((i / NS) - 1) & 1, abort_flag, p.status, 80)) break;
            if (lane == 0) mbar_expect_tx(full + s, SL::TILE);
            __syncwarp();
            uint8_t* dst = smem + SL::K + s * SL::TILE;
            const int t0 = __shfl_sync(0xffffffffu, tok[0], 0);
            if (__shfl_sync(0xffffffffu, tok[3], 31) == t0 + 127) {         // the tokens are consecutive: one box
                if (lane == 0) {
#pragma unroll
                    for (int cb = 0; cb < NBLK; ++cb) tma_load_3d(dst + cb * EBLK, &tmT, full + s, cb * 64, h, t0);
                }
            } else {                                                        // four rows a lane (beyond the list: any row, never written)
#pragma unroll
                for (int cb = 0; cb < NBLK; ++cb)
                    tma_gather4(dst + lane * 512 + cb * EBLK, &tmK, full + s, h * D + cb * 64, max(tok[0], 0), max(tok[1], 0), max(tok[2], 0), max(tok[3], 0));
            }
            // second arrival: tokens and coefficients (the rows are not held up by the loads of these)
            int* mt = reinterpret_cast<int*>(smem + SL::META + s * SL::META_BYTES);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                mt[4 * lane + e] = tok[e];
                mt[128 + 4 * lane + e] = __float_as_int(cf[e]);
                if (MULTI) mt[256 + 4 * lane + e] = seq[e];
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(full + s);
            if (i + NS < n_my) look(i + NS);
        }
        // the last rows asked for have landed before the shared memory is released (also after an abort)
        if (i >= NS) mbar_wait_limit(full + s, ((i / NS) - 1) & 1, nullptr, nullptr, 0, kWaitLimitNs);
    } else if (warp == 16) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t IDESC = umma_idesc_bf16(D, false);
        constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
        const uint32_t dK = umma_desc_lo(smem_u32(smem + SL::K), 16), dP = umma_desc_lo(smem_u32(smem + SL::P), 16);
        // projector loads: number u is that of product u (i * M + m) where they do not all stay, else of expert u
        const bool stay = !MULTI || M <= NP;
        const int n_load = !MULTI || n_my == 0 ? 0 : stay ? M : n_my * M;
        int n_pushed = 0;
        auto load_p = [&]() {
            const int slot = n_pushed % NP, m = n_pushed % M;
            mbar_expect_tx(p_full + slot, 2 * SL::PMAT);
#pragma unroll
            for (int part = 0; part < 2; ++part)
#pragma unroll
                for (int cb = 0; cb < NBLK; ++cb)
                    tma_load_3d(smem + SL::P + (slot * 2 + part) * SL::PMAT + cb * SL::PBLK, &tmP, p_full + slot, cb * 64, 0,
                                ((part * M + m) * Hkv + h) * D);
            ++n_pushed;
        };
        if (lane == 0) {            // (one lane runs the whole loop: nothing to agree on between its waits)
            while (n_pushed < n_load && n_pushed < NP) load_p();
            bool ok = true;
            if (!MULTI && n_my > 0) {           // P = U_hi U_hi^T + U_hi U_lo^T + U_lo U_hi^T (to about 2^-17)
                ok = mbar_wait(u_full, 0, abort_flag, p.status, 87);
                if (ok) {
                    for (int t = 0; t < 3; ++t)
                        for (int ks = 0; ks < (p.r + 15) / 16; ++ks) {
                            const uint32_t off = ((uint32_t)(ks >> 2) * SL::PBLK + (uint32_t)(ks & 3) * 32) >> 4;
                            umma_ss(tmem_base, dP + (t == 2 ? SL::PMAT >> 4 : 0u) + off, DESC_HI, dP + (t == 1 ? SL::PMAT >> 4 : 0u) + off, DESC_HI, IDESC,
                                    (t > 0 || ks > 0) ? 1u : 0u);
                        }
                    umma_commit(p_mma);
                }
            }
            for (int i = 0, u = 0; i < n_my && ok; ++i) {
                const int s = i % NS;
                ok = mbar_wait(full + s, (i / NS) & 1, abort_flag, p.status, 81);
                if (!ok) break;
                for (int m = 0; m < M; ++m, ++u) {
                    const int set = set_of(i, m), slot = stay ? m : u % NP;
                    if (!stay || i == 0) ok = mbar_wait(p_full + slot, stay ? 0 : (u / NP) & 1, abort_flag, p.status, 82);
                    if (ok && nth_of(i, m) >= GSET) ok = mbar_wait(cols + set, phase_of(i, m) ^ 1u, abort_flag, p.status, 83);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t kd = dK + s * (SL::TILE >> 4), pd = dP + slot * (2 * SL::PMAT >> 4);
#pragma unroll
                    for (int part = 0; part < 2; ++part)
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            const uint32_t offk = ((uint32_t)(ks >> 2) * EBLK + (uint32_t)(ks & 3) * 32) >> 4;
                            const uint32_t offp = ((uint32_t)part * SL::PMAT + (uint32_t)(ks >> 2) * SL::PBLK + (uint32_t)(ks & 3) * 32) >> 4;
                            umma_ss(tmem_base + set * D, kd + offk, DESC_HI, pd + offp, DESC_HI, IDESC, (ks > 0 || part) ? 1u : 0u);
                        }
                    umma_commit(done + set);
                    if (!stay && u > 0 && n_pushed < n_load) {      // the product before is through: its projector makes room
                        const int ip = (u - 1) / M, mp = (u - 1) % M;
                        ok = mbar_wait(done + set_of(ip, mp), phase_of(ip, mp), abort_flag, p.status, 84);
                        if (!ok) break;
                        load_p();
                    }
                }
            }
            if (*abort_flag) {
                // projectors on their way land, and products issued finish, before shared and tensor memory are released
                for (int u = n_pushed > NP ? n_pushed - NP : 0; u < n_pushed; ++u)
                    mbar_wait_limit(p_full + u % NP, (u / NP) & 1, nullptr, nullptr, 0, kWaitLimitNs);
                umma_commit(drain);
                mbar_wait_limit(drain, 0, nullptr, nullptr, 0, kWaitLimitNs);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ drain and write-out
        const int row = tid & 127, col0 = ((warp % SL::WPT) >> 2) * 32;          // row of the step, first of this thread's 32 columns
        const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + col0;
        const uint32_t off0 = (uint32_t)(col0 >> 6) * EBLK + sw128_offset(row, col0 & 63);
        bool ready = true;
        if constexpr (!MULTI) {
            if (n_my > 0) {
                // both parts of U, [D x 64] blocks where the projector will stand
                uint8_t* sP = smem + SL::P;
#pragma unroll 1
                for (int u = tid; u < D * nu; u += 512) {
                    const int i = u / nu, c8 = (u - i * nu) * 8;
                    if (!u_early || u != tid) load_u(h, u, u_first);
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) split_pair(u_first[2 * e], u_first[2 * e + 1], hi[e], lo[e]);
                    const uint32_t off = (uint32_t)(c8 >> 6) * SL::PBLK + sw128_offset(i, c8 & 63);
                    *reinterpret_cast<uint4*>(sP + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4*>(sP + SL::PMAT + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(u_full);
                // the projector in two parts over them
                ready = warp_wait(p_mma, 0, abort_flag, p.status, 88);
                const int pc = (warp >> 2) * 32;
                if (ready && pc < D && (warp & 3) * 32 < D) {
                    tc_fence_after();
                    uint32_t v[32];
                    tmem_ld32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + pc, v);
                    tmem_wait_ld_on(v);
                    tc_fence_before();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) split_pair(__uint_as_float(v[q * 8 + 2 * e]), __uint_as_float(v[q * 8 + 2 * e + 1]), hi[e], lo[e]);
                        const uint32_t off = (uint32_t)(pc >> 6) * SL::PBLK + sw128_offset(row, (pc & 63) + q * 8);
                        *reinterpret_cast<uint4*>(sP + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        *reinterpret_cast<uint4*>(sP + SL::PMAT + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                    fence_proxy_async();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(p_full);
            }
        }
        for (int i = warp / SL::WPT; ready && i < n_my; i += GROUPS) {
            const int s = i % NS;
            if (!warp_wait(full + s, (i / NS) & 1, abort_flag, p.status, 85)) break;
            const int* mt = reinterpret_cast<const int*>(smem + SL::META + s * SL::META_BYTES);
            const int tok = mt[row];
            const float cf = __int_as_float(mt[128 + row]);
            uint8_t* sK = smem + SL::K + s * SL::TILE;
            bool ok = true;
            uint4 kv[4];                                // this thread's 32 columns of the row (before anything waits for the product)
#pragma unroll
            for (int q = 0; q < 4; ++q) kv[q] = *reinterpret_cast<const uint4*>(sK + (off0 ^ (q << 4)));
            float acc[32];
            const float* al = MULTI && p.alpha != nullptr ? p.alpha + ((size_t)mt[256 + row] * Hkv + h) * M : nullptr;
#pragma unroll 1
            for (int m = 0; m < M; ++m) {
                const int set = set_of(i, m);
                const float cm = cf * (MULTI && al != nullptr ? al[m] : 1.f);
                ok = warp_wait(done + set, phase_of(i, m), abort_flag, p.status, 86);
                if (!ok) break;
                tc_fence_after();
                uint32_t v[32];
                tmem_ld32(t_lane + set * D, v);
                tmem_wait_ld_on(v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(cols + set);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] = MULTI ? fmaf(cm, __uint_as_float(v[e]), m == 0 ? 0.f : acc[e]) : __uint_as_float(v[e]);
            }
            if (!ok) break;
#pragma unroll
            for (int q = 0; q < 4; ++q) {               // 8 elements = one 16-byte unit of the swizzled row
                uint32_t* w = reinterpret_cast<uint32_t*>(&kv[q]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 k2 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w[e]));
                    const float v0 = acc[q * 8 + 2 * e], v1 = acc[q * 8 + 2 * e + 1];
                    w[e] = MULTI ? pack_bf16(k2.x + v0, k2.y + v1) : pack_bf16(fmaf(cf, v0, k2.x), fmaf(cf, v1, k2.y));
                }
                *reinterpret_cast<uint4*>(sK + (off0 ^ (q << 4))) = kv[q];
            }
            fence_proxy_async();            // (the stage is written by TMA next; here no global store is on its way yet)
            __syncwarp();
            // four lanes write the 64 bytes of a row, eight rows an instruction
            uint4 v[4];
            const uint32_t rd = (uint32_t)(col0 >> 6) * EBLK + sw128_offset((warp & 3) * 32 + (lane >> 2), (col0 & 63) + (lane & 3) * 8);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = *reinterpret_cast<const uint4*>(sK + rd + k * 1024);
            fence_proxy_async();            // (these reads come before the copies that refill the stage)
            __syncwarp();
            if (lane == 0) mbar_arrive(freeb + s);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int t = __shfl_sync(0xffffffffu, tok, k * 8 + (lane >> 2));
                if (t >= 0) *reinterpret_cast<uint4*>(p.out + ((size_t)(uint32_t)t * Hkv + h) * D + col0 + (lane & 3) * 8) = v[k];
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem_base, 512);
}

template <int D, bool SIDE, typename KT, bool PACK = false, int NTH = ET_THREADS>
static seka_status launch_tiles_t(TileArgs& a, long long n_units, size_t smem, int extra_blocks, cudaStream_t st) {
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    auto kern = edit_tiles_kernel<D, SIDE, KT, PACK, NTH>;
    constexpr int CTAS = EtSmem<D, SIDE, PACK>::CTAS;
    if (smem > 220 * 1024) return SEKA_ERR_UNSUPPORTED;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return SEKA_ERR_CUDA;
    long long per_sm = (227 * 1024) / (smem + (SIDE ? 4 : 9) * 1024);
    per_sm = per_sm > CTAS ? CTAS : (per_sm < 1 ? 1 : per_sm);
    // one wave; a multiple of the KV heads or (routed) of the (sequence, KV head) pairs
    long long g = per_sm * n_sm;
    if (g > n_units) g = n_units;
    if (SIDE && a.route.sigma != nullptr && g >= (long long)a.B * a.Hkv) g -= g % ((long long)a.B * a.Hkv);
    else if (g > a.Hkv) g -= g % a.Hkv;
    a.n_tile_blocks = (int)g;
    return launch_kernel(true, kern, (unsigned)(g + extra_blocks), NTH, smem, st, a);
}

// Blocks of U that stay in shared memory.  Stacked ranks of 65 to 128 keep both at head_dim 64, where that leaves room for two
// CTAs; at head_dim 128 they are replaced per step (one CTA per SM with both: 79 against 52 us on 12 x 1500 tokens, 8 heads, four
// experts of rank 24).  Beyond 128 replacing them is what a step spends its time on.  A preparation of many steps (`many`) keeps up
// to four at head_dim 128 (four experts of rank 64 on 51 x 423 tokens of 4 heads 143 -> 97 us, 81 with the routing apart) and,
// where the CTAs do not route, three at head_dim 64 (rank 48, 51 x 423 tokens of 8 heads 68 -> 59; four would leave one CTA per
// SM: rank 64, 82 -> 101).
static int u_blocks_of(const seka_shape* s, bool many = false, bool routed = false) {
    const int R = s->rank * s->n_experts, nb = (R + ET_UCOLS - 1) / ET_UCOLS;
    if (many && nb > 2 && (s->head_dim == 128 ? nb <= ET_UBLOCKS : nb == 3 && !routed)) return nb;
    return s->head_dim == 64 && nb == 2 ? 2 : 1;
}

template <int D, bool SIDE, bool PACK = false>
static size_t tiles_smem(const seka_shape* s, int u_blocks, bool routed, int k_route) {
    using SL = EtSmem<D, SIDE, PACK>;
    return 1024 + SL::U + u_blocks * SL::UBLK + (SIDE ? SL::TILE : 0) + (routed ? align_up((size_t)s->n_experts * 4, 16) + route_smem_bytes(D, s->n_experts, k_route) : 0);
}

static TileArgs tile_args(const seka_shape* s, const WorkspaceLayout& w, const void* K, void* out, const uint8_t* mask, const float* U,
                          const float* alpha, const float* gain, const uint8_t* he, char* ws) {
    TileArgs a = {};
    a.K = K; a.out = static_cast<__nv_bfloat16*>(out);
    a.mask = mask; a.U = U; a.alpha = alpha; a.gain = gain; a.head_enable = he; a.cu = s->cu_seqlens;
    a.list = reinterpret_cast<int*>(ws + w.list_off); a.seqs = reinterpret_cast<int*>(ws + w.seq_off); a.counts = reinterpret_cast<int*>(ws + w.count_off);
    a.seg_tokens = edit_segment_tokens(shape_total_tokens(s));
    a.n_seg = (shape_total_tokens(s) + a.seg_tokens - 1) / a.seg_tokens;
    a.tile_hot = reinterpret_cast<uint8_t*>(ws + w.hot_off); a.bh_info = reinterpret_cast<uint8_t*>(ws + w.info_off);
    a.status = reinterpret_cast<int*>(ws); a.u_blocks = u_blocks_of(s);
    a.B = s->batch; a.L = s->max_seqlen; a.Hkv = s->n_kv_heads; a.r = s->rank; a.M = s->n_experts; a.n_tiles = w.n_tiles;
    return a;
}

template <int D, bool MULTI>
static seka_status launch_gather_t(const TileArgs& a, const void* P, int T, long long units, int n_sm, cudaStream_t st) {
    using SL = EgSmem<D, MULTI>;
    CUtensorMap tk, tt, tp;        // gathered rows, 128 consecutive rows, projectors
    if (!make_row_map(&tk, a.K, a.Hkv * D, T) || !make_tile_map(&tt, a.K, D, a.Hkv, T)) return SEKA_ERR_CUDA;
    tp = tt;                       // (not used with one expert)
    if (MULTI && !make_tile_map(&tp, P, D, 1, (long long)2 * a.M * a.Hkv * D, D)) return SEKA_ERR_CUDA;
    auto kern = edit_gather_kernel<D, MULTI>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SL::DYN_BYTES) != cudaSuccess) return SEKA_ERR_CUDA;
    return launch_kernel(true, kern, (unsigned)(units < n_sm ? units : n_sm), SL::THREADS, SL::DYN_BYTES, st, tk, tt, tp, a);
}

// The gathering kernel instead of the chain.  `units`: (128 tokens, KV head) pairs if every token were highlighted (how many are
// is known on the device only).  Chain against gathering, us per call in place, 8 heads of 128 unless said otherwise:
//   one expert, rank of at most 32 (packed chain): 144 x 4096 tokens, 2 % / 10 % / all highlighted 20.7 / 68.5 / 619 against 20.7 / 62 /
//     546; 64 x 3000 (12000 units) 11.3 / 30 / 204 against 14 / 26 / 183, where the sparse edit would pay 3 us for its larger CTAs;
//   rank of 33 to 64: 64 x 3000, rank 64, 10 % / all 35 / 245 against 30 / 187; 16 x 4096 (4096 units) 10 % even; 64 x 4096 x 16 of 64,
//     10 % / all 45 / 371 against 34 / 199;
//   rank beyond 64 (the chain replaces U in every step): 1 x 4096, rank 128, 10 % 13.7 against 11, 64 x 3000 all 472 against 163;
//   several experts: a step costs the chain about 130 + 195 and the gathering kernel 150 (all of 64 x 3000) per block of stacked
//     columns / per expert: four of rank 32 / 64 / 128 523 / 909 / 1682 against 624 / 625 / 592, two of rank 64 516 against 292 (14.5
//     against 16 on 1 x 4096), eight of rank 64 1691 against 1128; at head_dim 64, where the chain keeps two blocks, four of rank 48 /
//     64 on 32 x 4096 x 16 545 / 680 against 324, two of rank 64 10 % on 8 x 4096 x 16 15.7 against 17.7.
static bool gather_edit(const seka_shape* s, long long units, int n_sm) {
    if (s->n_kv_heads > n_sm || s->n_kv_heads > kMaxGatherHeads) return false;
    const long long size = units * s->head_dim;
    if (s->n_experts > 1) return edit_projectors(s) && (s->rank * s->n_experts > 2 * ET_UCOLS || (s->head_dim == 128 && size >= 2048 * 128));
    return s->rank > 64 || size > (s->rank > 32 ? 4095 : 32768) * 128LL;
}

static seka_status launch_edit_tiles(const seka_shape* s, const WorkspaceLayout& w, const void* K_in, void* K_out, const uint8_t* mask,
                                     const float* U, const float* alpha, const float* gain, const uint8_t* he, char* ws, cudaStream_t st) {
    const int T = shape_total_tokens(s), Hkv = s->n_kv_heads, D = s->head_dim;
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    TileArgs a = tile_args(s, w, K_out, K_out, mask, U, alpha, gain, he, ws);
    const bool copy = K_in != K_out;
    const size_t n16 = copy ? (size_t)T * Hkv * D / 8 : 0;
    size_t n_copy = (n16 + 4 * 256 - 1) / (4 * 256);
    if (n_copy > (size_t)n_sm * 8) n_copy = (size_t)n_sm * 8;
    const long long units = (long long)((T + 127) / 128) * Hkv;
    const bool gather = gather_edit(s, units, n_sm) && (s->n_experts == 1 || (reinterpret_cast<uintptr_t>(ws) & 15) == 0);
    const int n_mats = s->n_experts * Hkv, n_p = gather && s->n_experts > 1 ? n_mats * (D / 32) * (D / 32) : 0;
    __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(ws + w.w_off);
    seka_status stc = launch_kernel(true, n_p > 0 ? edit_scan_kernel<true> : edit_scan_kernel<false>, (unsigned)(a.n_seg + n_copy + n_p), PREP_THREADS, 0, st, mask, gain, s->cu_seqlens, T, s->batch,
                                    s->max_seqlen, const_cast<int*>(a.list), const_cast<int*>(a.seqs), const_cast<int*>(a.counts), a.seg_tokens, a.n_seg,
                                    static_cast<const uint4*>(K_in), static_cast<uint4*>(K_out), n16, U, P, n_p, n_mats, D, s->rank);
    if (stc != SEKA_OK) return stc;
    if (gather) {
        if (D == 128) return s->n_experts == 1 ? launch_gather_t<128, false>(a, P, T, units, n_sm, st) : launch_gather_t<128, true>(a, P, T, units, n_sm, st);
        return s->n_experts == 1 ? launch_gather_t<64, false>(a, P, T, units, n_sm, st) : launch_gather_t<64, true>(a, P, T, units, n_sm, st);
    }
    // (the fused forward's preparation stays unpacked: its launches are a step or two per CTA, and gain nothing)
    if (s->rank * s->n_experts <= ET_UCOLS / 2)
        return D == 128 ? launch_tiles_t<128, false, __nv_bfloat16, true>(a, units, tiles_smem<128, false, true>(s, a.u_blocks, false, 0), 0, st)
                        : launch_tiles_t<64, false, __nv_bfloat16, true>(a, units, tiles_smem<64, false, true>(s, a.u_blocks, false, 0), 0, st);
    return D == 128 ? launch_tiles_t<128, false, __nv_bfloat16>(a, units, tiles_smem<128, false>(s, a.u_blocks, false, 0), 0, st)
                    : launch_tiles_t<64, false, __nv_bfloat16>(a, units, tiles_smem<64, false>(s, a.u_blocks, false, 0), 0, st);
}

// ---------------------------------------------------------------- many tiles, few projectors: the preparation as a pipeline
//
// Where the tiles of a plain-SEKA forward are many waves of CTAs, the chain above is bound by its instruction latencies
// (about 5000 cycles per tile and SM at head_dim 64).  There one persistent CTA per SM with three roles does the same work from
// the projector P[h] = U_h U_h^T (two bf16 parts, formed by the launch before), about 2700 cycles per tile and SM:
//   warp 8   producer: walks this CTA's (sequence, tile) pairs of one KV head, stages the key tiles that hold a highlighted
//            token through a ring of NS shared-memory stages by TMA, with the rows' highlight flags beside them;
//   warp 9   MMA issuer: K P (two bf16 parts) into one of two sets of tensor-memory columns;
//   warps 0-7  drain: half a key row per thread, k' = k + c (K P)[row] into the staged tile for highlighted rows, the low parts
//            beside it, then the rows go out 16 bytes per lane; stage and columns are handed back.
// Bound by the writes (twice what it reads).  At head_dim 64 the low parts go through shared memory as well (a row per lane
// they were 16-byte pieces, two to a sector) and two CTAs fit an SM: 16384 tiles of 16 heads 98 -> 77 us (the second CTA alone
// 92, three of them 94).  At head_dim 128 shared memory is full of P and key tiles: low parts go straight to global memory
// (through shared memory with two key stages instead of four: 101 against 93 us on 64 x 1024 tokens of 8 heads).
constexpr int EP_THREADS = 320;

// per stage: highlighted rows, first token, rows inside the sequence, end marker, low parts wanted, g * alpha
// (several experts: the gain alone, and the sequence)
struct __align__(16) EpMeta { uint32_t bits[4]; int tok0, nvalid, valid, with_lo; float c; int b, pad[2]; };

// NP: most projectors (experts).  Several of them (head_dim 64) leave room for one CTA per SM.
template <int D, int NP>
struct EpSmem {
    static constexpr uint32_t TILE = (D / 64) * EBLK;
    static constexpr uint32_t PBLK = D * 128;
    static constexpr uint32_t PMAT = (D / 64) * PBLK;
    static constexpr int NS = D == 128 ? 4 : NP == 4 ? 6 : 3;       // stages of key tiles
    static constexpr int CTAS = D == 128 || NP > 1 ? 1 : 2; // per SM (the projector of 128 leaves room for one)
    static constexpr int CS = NP * D > 256 ? 1 : 2;         // sets of tensor-memory columns (NP products each)
    static constexpr uint32_t K = 0;                        // NS stages
    static constexpr uint32_t P = K + NS * TILE;            // high part, then low part of each
    static constexpr bool LOW = D == 64;                    // the low parts go out through shared memory (two tiles), as whole rows
    static constexpr uint32_t L = P + NP * 2 * PMAT;
    static constexpr uint32_t META = L + (LOW ? 2 * TILE : 0);        // NS x 48 bytes
    static constexpr uint32_t BARS = META + NS * 48;        // full[NS], free[NS], mma_done[2], cols_free[2], p_full, meet[2]
    static constexpr uint32_t NBARS = 2 * NS + 7;
    static constexpr uint32_t MISC = BARS + NBARS * 8;
    static constexpr uint32_t DYN_BYTES = MISC + 16 + 1024;
};

template <int D, int NP>
__global__ void __launch_bounds__(EP_THREADS, EpSmem<D, NP>::CTAS)
stage_keys_pipe_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmP, __nv_bfloat16* __restrict__ X,
                       const uint8_t* __restrict__ mask, const float* __restrict__ alpha, const float* __restrict__ gain,
                       const uint8_t* __restrict__ head_enable, const int* __restrict__ cu_seqlens,
                       const uint8_t* __restrict__ tile_hot, int* status, int B, int L, int Hkv, int n_tiles, int routed, int n_experts) {
    using SL = EpSmem<D, NP>;
    constexpr int EP_NS = SL::NS, CS = SL::CS;
    constexpr int NBLK = D / 64;
    constexpr uint32_t TMEM_COLS = CS * NP * D;
    const int M = NP == 1 ? 1 : n_experts;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SL::BARS);
    uint64_t* full = bars;                     // [NS]  tile landed (TMA bytes) and flags / coordinates written (producer)
    uint64_t* freeb = full + EP_NS;            // [NS]  8 drain-warp arrivals: the stage may be refilled
    uint64_t* mma_done = freeb + EP_NS;        // [2]   K P of a tile (of every expert) is in column set c
    uint64_t* cols_free = mma_done + 2;        // [2]   8 drain-warp arrivals: column set c has been read
    uint64_t* p_full = cols_free + 2;          // [1]   projector landed
    uint64_t* meetb = p_full + 1;              // [2]   8 drain-warp arrivals: all rows of the tile are updated
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + SL::MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SL::MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < EP_NS; ++i) { mbar_init(full + i, 2); mbar_init(freeb + i, 8); }
        for (int i = 0; i < 2; ++i) { mbar_init(mma_done + i, 1); mbar_init(cols_free + i, 8); mbar_init(meetb + i, 8); }
        mbar_init(p_full, 1);
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmP);
    }
    __syncwarp();
    if (warp == 0) { tmem_alloc(tmem_holder, TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    pdl_wait();
    pdl_release();
    const bool dead = __syncthreads_or(*reinterpret_cast<volatile int*>(status) != 0);

    if (dead) {
        // an earlier launch gave up on this workspace
    } else if (warp == 8) {
        // ------------------------------------------------------------ producer
        // Its units are (sequence, tile) pairs blk, blk + n, ... of one KV head (the grid is a multiple of Hkv).  One lane per
        // unit fetches what a unit needs from global memory (flag, sequence bounds) for 32 units at a time; the highlight
        // flags of a tile's rows are requested one tile ahead, so that the ring is not fed at the pace of memory round trips.
        const int h = (int)blockIdx.x % Hkv, bt_step = (int)gridDim.x / Hkv, n_bt = B * n_tiles;
        uint32_t n_push = 0;      // stages filled so far
        bool ok = true;
        const bool on = head_enable == nullptr || head_enable[h] != 0;
        if (lane == 0 && on) {
            mbar_expect_tx(p_full, M * 2 * SL::PMAT);
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int cb = 0; cb < NBLK; ++cb)
                        tma_load_3d(smem + SL::P + (m * 2 + part) * SL::PMAT + cb * SL::PBLK, &tmP, p_full, cb * 64, 0, ((part * M + m) * Hkv + h) * D);
        }
        __syncwarp();
        auto push = [&](bool last, int tok0, int nvalid, int with_lo, float c, int b, const uint32_t (&bits)[4]) {
            const uint32_t s = n_push % EP_NS;
            if (n_push >= EP_NS) {
                ok = warp_wait(freeb + s, ((n_push / EP_NS) - 1) & 1, abort_flag, status, 63);
                if (!ok) return;
            }
            if (lane == 0) {
                EpMeta* m = reinterpret_cast<EpMeta*>(smem + SL::META + s * 48);
                m->tok0 = tok0; m->valid = last ? 0 : 1; m->c = c; m->nvalid = nvalid; m->with_lo = with_lo; m->b = b;
#pragma unroll
                for (int q = 0; q < 4; ++q) m->bits[q] = bits[q];
                if (!last) {
                    mbar_expect_tx(full + s, SL::TILE);
#pragma unroll
                    for (int cb = 0; cb < NBLK; ++cb) tma_load_3d(smem + SL::K + s * SL::TILE + cb * EBLK, &tmK, full + s, cb * 64, h, tok0);
                } else {
                    mbar_arrive(full + s);
                }
                mbar_arrive(full + s);       // second arrival: flags and coordinates are in place
            }
            __syncwarp();
            ++n_push;
        };
        for (long long base = (int)blockIdx.x / Hkv; base < n_bt && ok && on; base += 32LL * bt_step) {
            const long long my = base + (long long)lane * bt_step;
            int tok0_l = 0, nv_l = 0, lo_l = 0, hot_l = 0, b_l = 0;
            float c_l = 0.f;
            if (my < n_bt) {
                const int bt = (int)my, b = bt / n_tiles, t = bt - b * n_tiles;
                const int seq0 = cu_seqlens ? cu_seqlens[b] : b * L;
                const int Lb = (cu_seqlens ? cu_seqlens[b + 1] : (b + 1) * L) - seq0;
                const float g = gain[b], a = NP > 1 ? alpha_max_of(alpha, (size_t)b * Hkv + h, M) : alpha != nullptr ? alpha[(size_t)b * Hkv + h] : 1.f;
                hot_l = (tile_hot[bt] != 0 && g != 0.f) ? 1 : 0;
                b_l = b;
                c_l = NP > 1 ? g : g * a;
                tok0_l = seq0 + t * 128; nv_l = Lb - t * 128 < 128 ? Lb - t * 128 : 128;
                lo_l = (lo_needed(g, routed ? 1.f : fabsf(a)) || t < kLoTiles) ? 1 : 0;        // (as in steer_byte)
            }
            unsigned todo = __ballot_sync(0xffffffffu, hot_l != 0);
            uint32_t bits[4] = {0, 0, 0, 0};
            auto flags_of = [&](int k, uint8_t (&f)[4]) {      // highlight flags of unit k of the batch (4 rows per lane)
                const int tok0 = __shfl_sync(0xffffffffu, tok0_l, k), nv = __shfl_sync(0xffffffffu, nv_l, k);
#pragma unroll
                for (int q = 0; q < 4; ++q) f[q] = q * 32 + lane < nv ? mask[tok0 + q * 32 + lane] : 0;
            };
            uint8_t fl[4];
            if (todo) flags_of(__ffs(todo) - 1, fl);
            while (todo && ok) {
                const int k = __ffs(todo) - 1;
                todo &= todo - 1;
                uint8_t fl_next[4] = {0, 0, 0, 0};
                if (todo) flags_of(__ffs(todo) - 1, fl_next);
#pragma unroll
                for (int q = 0; q < 4; ++q) { bits[q] = __ballot_sync(0xffffffffu, fl[q] != 0); fl[q] = fl_next[q]; }
                push(false, __shfl_sync(0xffffffffu, tok0_l, k), __shfl_sync(0xffffffffu, nv_l, k), __shfl_sync(0xffffffffu, lo_l, k),
                     __shfl_sync(0xffffffffu, c_l, k), __shfl_sync(0xffffffffu, b_l, k), bits);
            }
        }
        if (ok) { const uint32_t none[4] = {0, 0, 0, 0}; push(true, 0, 0, 0, 0.f, 0, none); }      // the end marker
        if (on) warp_wait(p_full, 0, abort_flag, status, 62);      // (a CTA without work leaves only when the projector has landed)
    } else if (warp == 9) {
        // ------------------------------------------------------------ MMA issuer
        constexpr uint32_t IDESC = umma_idesc_bf16(D, false);
        constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
        const uint32_t dK = umma_desc_lo(smem_u32(smem + SL::K), 16), dP = umma_desc_lo(smem_u32(smem + SL::P), 16);
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
            const uint32_t s = n % EP_NS, cset = n % CS;
            ok = warp_wait(full + s, (n / EP_NS) & 1, abort_flag, status, 64);
            if (!ok) break;
            const EpMeta m = *reinterpret_cast<const EpMeta*>(smem + SL::META + s * 48);
            if (!m.valid) break;
            if (n == 0) {
                ok = warp_wait(p_full, 0, abort_flag, status, 65);
                if (!ok) break;
            }
            if (n >= CS) {
                ok = warp_wait(cols_free + cset, ((n / CS) - 1) & 1, abort_flag, status, 66);
                if (!ok) break;
            }
            tc_fence_after();
            if (lane == 0) {
                const uint32_t kd = dK + s * (SL::TILE >> 4);
#pragma unroll 1
                for (int m = 0; m < M; ++m)
#pragma unroll
                    for (int part = 0; part < 2; ++part)
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            const uint32_t offk = ((uint32_t)(ks >> 2) * EBLK + (uint32_t)(ks & 3) * 32) >> 4;
                            const uint32_t offp = ((uint32_t)part * SL::PMAT + (uint32_t)(ks >> 2) * SL::PBLK + (uint32_t)(ks & 3) * 32) >> 4;
                            umma_ss(tmem_base + (cset * NP + m) * D, kd + offk, DESC_HI, dP + m * (2 * SL::PMAT >> 4) + offp, DESC_HI, IDESC, (ks > 0 || part) ? 1u : 0u);
                        }
                umma_commit(mma_done + cset);
            }
            __syncwarp();
        }
    } else if (warp < 8) {
        // ------------------------------------------------------------ drain and write-out
        const int row = tid & 127, half = tid >> 7, h = (int)blockIdx.x % Hkv;
        const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        bool ok = true;
        for (uint32_t n = 0; ok; ++n) {
            const uint32_t s = n % EP_NS, cset = n % CS, lset = n & 1;
            ok = warp_wait(full + s, (n / EP_NS) & 1, abort_flag, status, 67);
            if (!ok) break;
            const EpMeta m = *reinterpret_cast<const EpMeta*>(smem + SL::META + s * 48);
            if (!m.valid) break;
            uint8_t* sK = smem + SL::K + s * SL::TILE;
            const uint32_t hl_bits = reinterpret_cast<const EpMeta*>(smem + SL::META + s * 48)->bits[warp & 3];
            const bool hl = ((hl_bits >> lane) & 1u) != 0, warp_hl = hl_bits != 0, with_lo = m.with_lo != 0;
            ok = warp_wait(mma_done + cset, (n / CS) & 1, abort_flag, status, 68);
            if (!ok) break;
            tc_fence_after();
            const bool side_lo = with_lo && row < m.nvalid;
            __nv_bfloat16* xlo = X + ((size_t)(m.tok0 + (row < m.nvalid ? row : 0)) * Hkv + h) * (2 * D) + D;
            if (warp_hl || with_lo) {
#pragma unroll 1
                for (int c = half * (D / 64); c < (half + 1) * (D / 64); ++c) {
                    uint32_t v[32];
                    float acc[NP > 1 ? 32 : 1];
                    if constexpr (NP == 1) {
                        if (warp_hl) { tmem_ld32(t_lane + cset * D + c * 32, v); tmem_wait_ld_on(v); }     // warp-wide: every lane takes part
                    } else if (warp_hl) {               // sum_m c_m K P_m
                        const float* al = alpha != nullptr ? alpha + ((size_t)m.b * Hkv + h) * M : nullptr;
#pragma unroll 1
                        for (int e = 0; e < M; ++e) {
                            const float cm = m.c * (al != nullptr ? al[e] : 1.f);
                            tmem_ld32(t_lane + (cset * NP + e) * D + c * 32, v);
                            tmem_wait_ld_on(v);
#pragma unroll
                            for (int k = 0; k < 32; ++k) acc[k] = fmaf(cm, __uint_as_float(v[k]), e == 0 ? 0.f : acc[k]);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {          // 8 elements = one 16-byte unit of the swizzled row
                        const int col = c * 32 + q * 8;
                        uint32_t lo[4] = {0u, 0u, 0u, 0u};
                        if (hl) {
                            uint4* ptr = reinterpret_cast<uint4*>(sK + (col >> 6) * EBLK + sw128_offset(row, col & 63));
                            uint4 kv = *ptr;
                            uint32_t* w = reinterpret_cast<uint32_t*>(&kv);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 k2 = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w[e]));
                                if constexpr (NP == 1) split_pair(fmaf(m.c, __uint_as_float(v[q * 8 + 2 * e]), k2.x), fmaf(m.c, __uint_as_float(v[q * 8 + 2 * e + 1]), k2.y), w[e], lo[e]);
                                else split_pair(k2.x + acc[q * 8 + 2 * e], k2.y + acc[q * 8 + 2 * e + 1], w[e], lo[e]);
                            }
                            *ptr = kv;
                        }
                        if (SL::LOW) {          // (the tile before last is out: its writers have met since)
                            if (with_lo) *reinterpret_cast<uint4*>(smem + SL::L + lset * SL::TILE + (col >> 6) * EBLK + sw128_offset(row, col & 63)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        } else if (side_lo) {
                            *reinterpret_cast<uint4*>(xlo + col) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        }
                    }
                    __syncwarp();      // all lanes together again before the next warp-wide load
                }
            }
            // the columns are read: the next product may use them; all rows updated: the tile may be written out
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { mbar_arrive(cols_free + cset); mbar_arrive(meetb + lset); }
            ok = warp_wait(meetb + lset, (n >> 1) & 1, abort_flag, status, 69);
            if (!ok) break;
            constexpr int LPR = D / 8, RPI = 32 / LPR;
#pragma unroll 1
            for (int i = 0; i < 16 / RPI; ++i) {
                const int r = warp * 16 + i * RPI + lane / LPR, col = (lane % LPR) * 8;
                if (r < m.nvalid) {
                    const uint4 v = *reinterpret_cast<const uint4*>(sK + (col >> 6) * EBLK + sw128_offset(r, col & 63));
                    __nv_bfloat16* dst = X + ((size_t)(m.tok0 + r) * Hkv + h) * (2 * D) + col;
                    *reinterpret_cast<uint4*>(dst) = v;
                    if (SL::LOW && with_lo) *reinterpret_cast<uint4*>(dst + D) = *reinterpret_cast<const uint4*>(smem + SL::L + lset * SL::TILE + (col >> 6) * EBLK + sw128_offset(r, col & 63));
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(freeb + s);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

// First launch of that path: blocks [0, n_p) form a 32 x 32 tile of P[h] each (bf16, high parts of all heads, then low parts);
// then blocks with a warp per (sequence, key tile) for the tile flags and the steering bytes; then, in a routed call, a block
// per (sequence, KV head) that leaves its coefficients (Eq. 6, the routine of adaseka_route: the same bits) for the launch
// behind; then the item table and the conversion of fp32 inputs (11 ragged sequences of up to 11083 tokens of 8 heads of 64, nearly all
// highlighted: 107 us for both launches, 232 for the chain with its conversion blocks).
__global__ void __launch_bounds__(PREP_THREADS)
prep_projector_kernel(const float* __restrict__ U, const uint8_t* __restrict__ mask, __nv_bfloat16* __restrict__ P,
                      uint8_t* __restrict__ tile_hot, uint8_t* __restrict__ bh_info, int B, int L, int Hkv, int D, int r, int M, int n_tiles,
                      int n_p, int n_flag, int n_route, const __grid_constant__ RouteArgs route, const __grid_constant__ PrepJobs jobs) {
    extern __shared__ __align__(16) double route_sm[];
    const int tid = threadIdx.x;
    pdl_wait();
    pdl_release();
    int blk = blockIdx.x;
    if (blk < n_p) {
        projector_block(U, P, blk, M * Hkv, D, r);
        return;
    }
    blk -= n_p;
    if (blk < n_flag) {
        const int item = blk * (PREP_THREADS / 32) + (tid >> 5), lane = tid & 31;
        if (item >= B * n_tiles) return;
        const int b = item / n_tiles, t = item % n_tiles;
        const int seq0 = jobs.cu ? jobs.cu[b] : b * L;
        const int Lb = (jobs.cu ? jobs.cu[b + 1] : (b + 1) * L) - seq0;
        bool any = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int pos = t * 128 + q * 32 + lane;
            any = (pos < Lb && mask[seq0 + pos] != 0) || any;
        }
        any = __any_sync(0xffffffffu, any);
        if (lane == 0) tile_hot[item] = any ? 1 : 0;
        if (t == 0)
            for (int h = lane; h < Hkv; h += 32) bh_info[(size_t)b * Hkv + h] = (uint8_t)steer_byte(jobs.steer, b, h, Hkv);
        return;
    }
    blk -= n_flag;
    if (blk < n_route) {
        const double* a = route_group(route.Q, route.q_is_f32, U, route.sigma, jobs.cu, L, route.Hq, Hkv, D, r, M, route.k_route, blk / Hkv,
                                      blk % Hkv, route_sm);
        for (int m = tid; m < M; m += PREP_THREADS) route.alpha_out[(size_t)blk * M + m] = (float)a[m];
        return;
    }
    blk -= n_route;
    if (blk < jobs.n_items_blocks) items_block(jobs.sched, jobs.cu, jobs.steer, jobs.items, jobs.item_count, blk);
    else convert_block(jobs.conv, blk - jobs.n_items_blocks, jobs.n_conv_blocks);
}

template <int D, int NP>
static seka_status launch_stage_pipe(const seka_shape* s, const WorkspaceLayout& w, const void* K, const uint8_t* mask, const float* U,
                                     const float* alpha, const float* gain, const uint8_t* he, char* ws, const PrepJobs& jobs,
                                     const RouteArgs& route_in, cudaStream_t st) {
    using PL = EpSmem<D, NP>;
    const int T = shape_total_tokens(s), Hkv = s->n_kv_heads;
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    void* P = ws + w.w_off;
    uint8_t* tile_hot = reinterpret_cast<uint8_t*>(ws + w.hot_off);
    CUtensorMap tk, tp;
    const void* k16 = s->dtype == SEKA_F32 ? static_cast<const void*>(jobs.conv.out[1]) : K;       // (converted by the first launch)
    if (!make_tile_map(&tk, k16, D, Hkv, T) || !make_tile_map(&tp, P, D, 1, (long long)2 * s->n_experts * Hkv * D, D)) return SEKA_ERR_CUDA;
    const int n_p = s->n_experts * Hkv * (D / 32) * (D / 32), n_flag = (s->batch * w.n_tiles + PREP_THREADS / 32 - 1) / (PREP_THREADS / 32);
    RouteArgs route = route_in;
    const int n_route = route.sigma != nullptr ? s->batch * Hkv : 0;
    if (n_route > 0) {          // without a place of the caller's the coefficients live in the list region, which has room for them
        if (route.alpha_out == nullptr) route.alpha_out = reinterpret_cast<float*>(ws + w.list_off);
        alpha = route.alpha_out;
    }
    const size_t route_smem = n_route > 0 ? route_smem_bytes(D, s->n_experts, route.k_route) : 0;       // (at most 34 KB, on top of 19 of its own)
    if (route_smem > 24 * 1024 &&
        cudaFuncSetAttribute(prep_projector_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)route_smem) != cudaSuccess) return SEKA_ERR_CUDA;
    seka_status stc = launch_kernel(true, prep_projector_kernel, (unsigned)(n_p + n_flag + n_route + jobs.n_items_blocks + jobs.n_conv_blocks), PREP_THREADS,
                                    route_smem, st, U, mask,
                                    static_cast<__nv_bfloat16*>(P), tile_hot, reinterpret_cast<uint8_t*>(ws + w.info_off), s->batch,
                                    s->max_seqlen, Hkv, D, s->rank, s->n_experts, w.n_tiles, n_p, n_flag, n_route, route, jobs);
    if (stc != SEKA_OK) return stc;
    auto kern = stage_keys_pipe_kernel<D, NP>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL::DYN_BYTES) != cudaSuccess) return SEKA_ERR_CUDA;
    const unsigned grid = (unsigned)(PL::CTAS * n_sm / Hkv * Hkv);
    return launch_kernel(true, kern, grid, EP_THREADS, PL::DYN_BYTES, st, tk, tp, reinterpret_cast<__nv_bfloat16*>(ws + w.x_off), mask, alpha,
                         gain, he, s->cu_seqlens, tile_hot, reinterpret_cast<int*>(ws), s->batch, s->max_seqlen, Hkv, w.n_tiles, n_route > 0 ? 1 : 0, s->n_experts);
}

seka_status launch_stage_keys(const seka_shape* s, const WorkspaceLayout& w, const void* K, const uint8_t* mask, const float* U,
                              const float* alpha, const float* gain, const uint8_t* head_enable, char* ws, const PrepJobs& jobs,
                              const RouteArgs& route, cudaStream_t st) {
    // One expert: the pipelined pair of launches from four waves of the chain on.  Measured preparations, pipeline against chain: packed
    // batch of 64 sequences, 16 heads of 64, short runs (16384 units) 84 against 132 us; 64 x 1024 tokens, 4 heads of 64 /
    // 128, all highlighted (2048 units) 26 against 36 / 50 against 56; 46 x 500, 8 heads of 64, 44 % (1472 units) 29 against
    // 30, 12 x 500 (384 units) 15 against 13; 4 x 4096 tokens, 8 heads of 128, a tenth (1024 units) 18 against 16; 4362 tokens, 8 heads (280) 19 against 13.
    // Several experts at head_dim 64 (up to the eight whose projectors fit, where they are less work than the stacked columns): from four
    // tiles per SM on.  Calls of the fused forward, pipeline against chain: four of rank 64 on 64 packed sequences of up to 2048 tokens of
    // 16 heads 760 against 1015 us, 16 x 1024 x 16 130 against 167, 8 x 2048 x 8 (1024 units) 102 against 119, 51 x 423 x 4 57 against 76;
    // two of rank 48 on 64 x 512 x 16 218 against 259.
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    const long long units = (long long)s->batch * w.n_tiles * s->n_kv_heads;
    if (units > 0x7fffffffLL) return SEKA_ERR_UNSUPPORTED;
    const int chain_ctas = s->head_dim == 128 ? EtSmem<128, true>::CTAS : EtSmem<64, true>::CTAS;
    if (s->n_experts == 1 && s->n_kv_heads <= n_sm && units > 4LL * chain_ctas * n_sm)     // (routed or not: both forms give the same bits)
        return s->head_dim == 128 ? launch_stage_pipe<128, 1>(s, w, K, mask, U, alpha, gain, head_enable, ws, jobs, route, st)
                                  : launch_stage_pipe<64, 1>(s, w, K, mask, U, alpha, gain, head_enable, ws, jobs, route, st);
    if (pipe_experts(s) && s->n_kv_heads <= n_sm && units > 4LL * n_sm)
        return s->n_experts <= 4 ? launch_stage_pipe<64, 4>(s, w, K, mask, U, alpha, gain, head_enable, ws, jobs, route, st)
                                 : launch_stage_pipe<64, 8>(s, w, K, mask, U, alpha, gain, head_enable, ws, jobs, route, st);
    TileArgs a = tile_args(s, w, K, ws + w.x_off, mask, U, alpha, gain, head_enable, ws);
    a.route = route; a.jobs = jobs;
    const size_t n_alpha = (size_t)s->batch * s->n_kv_heads * s->n_experts;
    const long long pairs = (long long)s->batch * s->n_kv_heads;
    if (route.sigma != nullptr && s->rank * s->n_experts > 2 * ET_UCOLS && units > 2LL * n_sm && n_sm / pairs * pairs * 5 < 4 * n_sm &&
        (route.alpha_out != nullptr || n_alpha * 4 <= w.list_bytes)) {
        // Wide banks with many steps: Eq. 6 by the launch of adaseka_route (same bits), so that its 17000 to 23000 cycles are
        // spent once per pair and no CTA is tied to a pair, where pairs do not go evenly into the SMs.  Four experts of rank 64,
        // 12 x 1500 tokens of 8 / 4 heads of 128 (96 / 48 pairs): 83 / 61 us against 121 / 56 routed in the CTAs.
        float* dst = route.alpha_out != nullptr ? route.alpha_out : reinterpret_cast<float*>(ws + w.list_off);
        const seka_status stc = launch_route(s, route.Q, U, route.sigma, route.k_route, dst, st);
        if (stc != SEKA_OK) return stc;
        a.route = RouteArgs{};
        a.alpha = dst;
    }
    const bool routed = a.route.sigma != nullptr;
    const int extra = jobs.n_items_blocks + jobs.n_conv_blocks;
    const bool f32 = s->dtype == SEKA_F32;
    if (units + extra <= n_sm) {                // one step per CTA, one CTA per SM: the small form (more CTAs than SMs would queue)
        const size_t smem = s->head_dim == 128 ? tiles_smem<128, true>(s, a.u_blocks, routed, route.k_route) : tiles_smem<64, true>(s, a.u_blocks, routed, route.k_route);
        if (s->head_dim == 128)
            return f32 ? launch_tiles_t<128, true, float, false, ET_SMALL>(a, units, smem, extra, st)
                       : launch_tiles_t<128, true, __nv_bfloat16, false, ET_SMALL>(a, units, smem, extra, st);
        return f32 ? launch_tiles_t<64, true, float, false, ET_SMALL>(a, units, smem, extra, st)
                   : launch_tiles_t<64, true, __nv_bfloat16, false, ET_SMALL>(a, units, smem, extra, st);
    }
    a.u_blocks = u_blocks_of(s, units > 2LL * n_sm, routed);
    if ((s->head_dim == 128 ? tiles_smem<128, true>(s, a.u_blocks, routed, route.k_route) : tiles_smem<64, true>(s, a.u_blocks, routed, route.k_route)) > 220 * 1024)
        a.u_blocks = u_blocks_of(s);
    if (s->head_dim == 128) {
        const size_t smem = tiles_smem<128, true>(s, a.u_blocks, routed, route.k_route);
        return f32 ? launch_tiles_t<128, true, float>(a, units, smem, extra, st) : launch_tiles_t<128, true, __nv_bfloat16>(a, units, smem, extra, st);
    }
    const size_t smem = tiles_smem<64, true>(s, a.u_blocks, routed, route.k_route);
    return f32 ? launch_tiles_t<64, true, float>(a, units, smem, extra, st) : launch_tiles_t<64, true, __nv_bfloat16>(a, units, smem, extra, st);
}

}  // namespace seka

extern "C" seka_status seka_edit_keys(const seka_shape* shape, const void* K_in, void* K_out, const uint8_t* mask,
                                      const float* U, const float* alpha, const float* gain,
                                      const uint8_t* head_enable, void* workspace, size_t workspace_bytes,
                                      void* cuda_stream) {
    using namespace seka;
    seka_status stc = validate_shape(shape);
    if (stc != SEKA_OK) return stc;
    const int T = shape_total_tokens(shape);
    if (T == 0) return SEKA_OK;
    if (!K_in || !K_out || !mask || !U || !gain) return SEKA_ERR_INVALID_ARG;
    if (((uintptr_t)K_in | (uintptr_t)K_out) & 15) return SEKA_ERR_INVALID_ARG;
    const WorkspaceLayout w = workspace_layout(shape);
    if (!workspace || workspace_bytes < w.edit_total) return SEKA_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    char* ws = static_cast<char*>(workspace);
    // bf16 tensors go through the tensor-core tile kernel, fp32 tensors through the fp32 row kernel
    if (shape->dtype == SEKA_BF16) return launch_edit_tiles(shape, w, K_in, K_out, mask, U, alpha, gain, head_enable, ws, st);
    return launch_edit_rows(shape, K_in, K_out, mask, U, alpha, gain, head_enable, st);
}

// ---------------------------------------------------------------- workspace-free variant: the fp32 row kernel needs no scratch
extern "C" seka_status seka_edit_keys_static(const seka_shape* shape, const void* K_in, void* K_out,
                                             const uint8_t* mask, const float* U, const float* alpha,
                                             const float* gain, const uint8_t* head_enable, void* cuda_stream) {
    using namespace seka;
    seka_status stc = validate_shape(shape);
    if (stc != SEKA_OK) return stc;
    const int T = shape_total_tokens(shape);
    if (T > SEKA_STATIC_MAX_TOKENS) return SEKA_ERR_UNSUPPORTED;   // the documented limit of this entry point
    if (T == 0) return SEKA_OK;
    if (!K_in || !K_out || !mask || !U || !gain) return SEKA_ERR_INVALID_ARG;
    if (((uintptr_t)K_in | (uintptr_t)K_out) & 15) return SEKA_ERR_INVALID_ARG;
    return launch_edit_rows(shape, K_in, K_out, mask, U, alpha, gain, head_enable, static_cast<cudaStream_t>(cuda_stream));
}

// Fused SEKA / AdaSEKA steered causal GQA attention forward for sm_100a.
//
// The edited logit of Eq. 5 is q.k' = q.k + q.(g P k).  A small preparation launch leaves the edited keys k' of every
// key tile that holds a highlighted token in a side buffer as a high and a low bf16 part (see SteerPlan); this kernel
// stages such a tile from the high parts instead of from K and, where the gain is large enough for the rounding of k'
// to matter, extends the score product S = Q K'^T on the tensor core, in the same tensor-memory accumulator, by the
// contraction with the low parts, so that the logits are those of the fp32 k'.  The score matrix never reaches memory;
// K and V are read only.
//
// One CTA (12 warps) owns two tiles of 128 queries that share a KV head ("A" and "B": two query heads of one group at
// the same rows, or two consecutive row tiles of one head when the group size is odd) and walks the key tiles
// 0 .. diagonal.  Warp roles:
//   warp 0        TMA producer: Q tiles, then K (or edited-key) and V tiles (128-byte swizzle) through two
//                 shared-memory rings, throttled by "free" mbarriers the tensor core signals, and the low parts of
//                 edited tiles through a ring of their own;
//   warp 1        MMA issuer: S_x = Q_x K^T (+ the low-part steps) and O_x += P_x V on tcgen05 with all accumulators
//                 in tensor memory (head_dim 128: S_A, S_B, O_A, O_B = 512 columns, P_x over S_x; head_dim 64: 384, P_A and P_B
//                 the other 128); P_x is read from tensor memory;
//   warp 2        operand relay: tells the issuer when the operands have landed, so that it waits on one barrier per
//                 hand-off (head_dim 64: warps 1 and 2 issue for tile A and tile B and see to their operands themselves);
//   warps 4-7 / 8-11  softmax of tile A / B, one query row per thread: causal mask on the diagonal tile, online
//                 softmax in base 2 with a lazily updated running maximum, P written back as bf16 over the consumed
//                 score columns (head_dim 64: to columns of its own), O rescaled in tensor memory only when the maximum
//                 moved by more than 2^8; final normalisation and store.
// (Warp 3 only gives its registers to the softmax warps.)
// While one tile's softmax runs, the tensor core works on the other tile.  Items follow each other without a seam: the next
// item's first key tile travels with this item's last value tile, its Q tiles follow the last score products, and the
// first scores of a tile's next item are issued right behind its last P V, under the store of its output (head_dim 64: that
// store waits for the next item's first weights).  Before, every item began with an empty tensor pipe and its operands on the
// way, about 8000 cycles.  Measured on 32 / 8 heads of 128: 4 x 4096 tokens 0.495 -> 0.466 ms, one prompt of 4362 tokens
// 148 -> 139 us (unsteered, GPU rested between blocks); 1 x 32768 level.  About 4200 cycles per item remain beside its steps.
// Every wait is bounded: a wait that runs out raises the CTA's abort flag, every role leaves its loop, and the status word
// reports it.
#include <math.h>

#include <mutex>

#include "seka_kernels.h"

namespace seka {

struct AttnParams {
    void* O;
    float* lse;
    const uint8_t* bh_info;       // [B, Hkv]: bit 0 the keys of this (sequence, KV head) are edited, bit 1 with the low parts
    const uint8_t* tile_hot;      // [B, n_qt]: key tile holds a highlighted token
    int* status;
    const ItemRecord* items;      // item table (packed batches), heaviest first
    const int* n_items;           // its length (device word)
    Sched sched;
    SteerPlan plan;
    int steer;
    float scale_log2;
};

constexpr int BM = 128, BN = 128;
constexpr int NTHREADS = 384;
constexpr uint32_t BLK_BYTES = 128 * 128;   // one [128 x 64] bf16 block
constexpr float LAZY_RESCALE_LOG2 = 8.0f;   // the running maximum is only raised when it moved by more than this
// registers per thread after the roles split, out of the launch's 168 per thread (3 x 168 = 104 + 2 x 200)
constexpr int REGS_CTRL = 104, REGS_SOFTMAX = 200;
// Plain polls of a wait before it parks (see mbar_wait_within).  One: a warp that polls takes issue slots from the softmax
// warps of its scheduler (eight polls cost 1 % on 4 x 4096 tokens of 32 heads of 128, polling without end 4 %).
constexpr int PLAIN_POLLS = 1;

constexpr uint32_t SMEM_LIMIT = 227 * 1024;


// Shared memory of one CTA.  Tiles first (each a multiple of 1024 bytes), then barriers and per-warp item slots.
template <int D>
struct Geo {
    // head_dim 128: P is handed to the tensor core in two pieces, so that most of P V runs under the last exponentials; 16-key
    // blocks in the first piece.  The exponentials come 32 keys at a time, so an even number; 5 and 7, with that loop cut at 16
    // keys, were level and 2 % slower.  (head_dim 64 hands P over whole: in two pieces 64 ragged sequences 590 -> 601 us, one
    // prompt of 8192 tokens 380 -> 434.)
    static constexpr int KP1 = 6;
    static_assert(KP1 % 2 == 0 && KP1 > 0 && KP1 < 8, "the first hand-over lies behind 32 or 64 or 96 of 128 keys");
    // Head_dim 64 leaves room in tensor memory for the weights P beside the scores.  The next scores of a tile are then formed as
    // soon as the present ones are in registers, under their softmax, instead of behind P V: the softmax warps wait for nothing
    // but one another's use of the special-function units.  Each tile has an issuer of its own (one for both would hold one
    // tile's scores back until the other's weights are there), and the output of an item is stored behind the first weights of
    // the next.  64 ragged sequences of 16 heads 646 -> 590 us (preparation included), one prompt of 8192 tokens of 32 / 8 heads
    // 412 -> 382, a toy layer in fp32 16.0 -> 14.6 (both sides in turn, 1.9 GHz).  Of that the late store costs the ragged batch
    // 0.7 % and the toy 1 %, and gives the long prompt 11 %: it pays where a CTA walks several items of many steps.  The two tiles'
    // exponentials kept apart by a lock per scheduler: 1 and 15 % slower.
    // With several items per CTA and an even head group the tiles run in step or half a period apart, whichever small delays of the
    // control warps lead to; in step is faster there (8192 tokens 380 us against 400 to 440).  Check both after any change here.
    static constexpr bool APART = D == 64;
    static constexpr int NK = D == 128 ? 2 : 3;                    // K and V ring depth
    static constexpr uint32_t TILE = (D / 64) * BLK_BYTES;         // a [128 x D] tile
    static constexpr int NXMAX = 3;                                // most stages of the key-side operand
    static constexpr uint32_t NBARS = 15 + 2 * NK + NXMAX;
    // shared-memory copy of the per-(sequence, KV head) steering bytes and of the tile flags, a bit each (what fits beside the
    // tiles; larger batches look them up in global memory)
    static constexpr int INFO_HEADS = D == 128 ? 768 : 2048, INFO_WORDS = D == 128 ? 128 : 512;
    static constexpr uint32_t INFO_BYTES = INFO_HEADS + INFO_WORDS * 4;
};

struct SmemPlan {
    uint32_t k, v, x, xb, bars, misc, items, info, total;
};

template <int D>
__host__ __device__ inline SmemPlan smem_plan(const SteerPlan& sp) {
    using G = Geo<D>;
    SmemPlan s;
    s.k = 2 * G::TILE;
    s.v = s.k + G::NK * G::TILE;
    s.x = s.v + G::NK * G::TILE;
    s.xb = sp.mode ? G::TILE : 0u;                                 // one stage of low parts: [128 x D]
    s.bars = s.x + (uint32_t)sp.nx * s.xb;
    s.misc = s.bars + ((G::NBARS * 8 + 15) & ~15u);                 // 16-byte aligned: the item slots are filled by 16-byte async copies
    s.items = s.misc + 32;
    s.info = s.items + 16 * 32;                                     // steering info of every (sequence, KV head), if it fits
    s.total = s.info + (sp.mode ? G::INFO_BYTES : 0u);
    return s;
}

// true in exactly one lane of a fully active warp
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}

template <int N> __device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// 4 x 4 transpose among groups of four lanes: unit u (16 bytes) of lane q becomes unit q of lane u
__device__ __forceinline__ void transpose4(uint4 (&a)[4], int lane) {
    auto swap = [&](uint4& x, uint4& y, int bit) {       // the lane without `bit` gives y for its partner's x
        const bool up = (lane & bit) != 0;
        uint4 send = up ? x : y;
        send.x = __shfl_xor_sync(0xffffffffu, send.x, bit); send.y = __shfl_xor_sync(0xffffffffu, send.y, bit);
        send.z = __shfl_xor_sync(0xffffffffu, send.z, bit); send.w = __shfl_xor_sync(0xffffffffu, send.w, bit);
        if (up) x = send; else y = send;
    };
    swap(a[0], a[2], 2); swap(a[1], a[3], 2);
    swap(a[0], a[1], 1); swap(a[2], a[3], 1);
}
// 32 columns of the rows of a warp (lane = row), scaled, to global memory: four lanes write 64 contiguous bytes of a row
// (a row per lane, 32 pieces of 16 bytes an instruction, took 2000 cycles of the load/store unit per tile).  `row0` points at
// the columns in the row of lane 0, rows are `pitch` elements apart, `n_rows` of them exist.
template <typename OutT> __device__ __forceinline__ void store_chunk32(OutT* row0, size_t pitch, int n_rows, const uint32_t (&v)[32], float inv, int lane) {
    constexpr int EPU = 16 / (int)sizeof(OutT);          // elements of 16 bytes
#pragma unroll
    for (int half = 0; half < 32 / (4 * EPU); ++half) {
        uint4 a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t* w = &v[half * 4 * EPU + u * EPU];
            if constexpr (sizeof(OutT) == 2)
                a[u] = make_uint4(pack_bf16(__uint_as_float(w[0]) * inv, __uint_as_float(w[1]) * inv), pack_bf16(__uint_as_float(w[2]) * inv, __uint_as_float(w[3]) * inv),
                                  pack_bf16(__uint_as_float(w[4]) * inv, __uint_as_float(w[5]) * inv), pack_bf16(__uint_as_float(w[6]) * inv, __uint_as_float(w[7]) * inv));
            else
                a[u] = make_uint4(__float_as_uint(__uint_as_float(w[0]) * inv), __float_as_uint(__uint_as_float(w[1]) * inv),
                                  __float_as_uint(__uint_as_float(w[2]) * inv), __float_as_uint(__uint_as_float(w[3]) * inv));
        }
        transpose4(a, lane);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = (lane & ~3) + k;
            if (r < n_rows) *reinterpret_cast<uint4*>(row0 + (size_t)r * pitch + half * 4 * EPU + (lane & 3) * EPU) = a[k];
        }
    }
}

// One unit of work of a CTA: two 128-row query tiles that share a KV head of one sequence.
struct Item {
    int b, hkv, seq0, Lb;
    int hqA, hqB, qtA, qtB;     // query head and row-tile index of tile A / B
    int nA, nB, n_kv;           // key tiles of A / B (0: the tile lies beyond the sequence) and of the item
    bool steer;                 // the keys of this (sequence, KV head) are edited
    bool need_lo;               // ... and the low parts of the edited keys are multiplied too
};

// LEAD (head_dim 64, one item per CTA, both tiles equally long): tile B starts its first exponentials when tile A is three
// quarters through its own, see launch_attn_t.
template <int D, typename OutT, bool TABLE, bool LEAD = false>
__global__ void __launch_bounds__(NTHREADS, 1)
seka_attn_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmX,
                     const __grid_constant__ AttnParams p) {
    using G = Geo<D>;
    static_assert(!LEAD || G::APART, "head_dim 128 uses the lead barrier otherwise");
    constexpr int NK = G::NK;
    constexpr int NBLK = D / 64;
    constexpr uint32_t TMEM_COLS = 512;
    constexpr uint32_t COL_S = 0, COL_O = 256;     // S_x at COL_S + 128 x, O_x at COL_O + D x
    constexpr uint32_t COL_P = G::APART ? 384 : COL_S, P_PITCH = G::APART ? 64 : 128;      // P_x at COL_P + P_PITCH x
    extern __shared__ __align__(1024) uint8_t smem[];
    const SmemPlan sl = smem_plan<D>(p.plan);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + sl.bars);
    uint64_t* q_full = bars;                 // [2]   Q tile landed
    uint64_t* k0_full = q_full + 2;          // [1]   first key tile of the CTA's first item landed
    uint64_t* kv_full = k0_full + 1;         // [NK]  V(g) and K(g+1) landed (they are loaded as a pair)
    uint64_t* kv_free = kv_full + NK;        // [NK]  one event per step: the tensor core is done with K(g+1) and V(g); (APART) an arrival from each issuer
    uint64_t* x_full = kv_free + NK;         // [3]   low parts of an edited tile landed
    uint64_t* s_full = x_full + G::NXMAX;    // [2]   scores of tile x are in tensor memory
    uint64_t* p_full = s_full + 2;           // [2]   4 softmax-warp arrivals (O_x rescaled, the first 16 KP1 keys of P_x written) + 1 from the relay; (APART) 4: all of P_x written
    uint64_t* p_last = p_full + 2;           // [2]   4 softmax-warp arrivals: the other keys of P_x written
    uint64_t* s_free = p_last;               // [2]   (APART) 4 softmax-warp arrivals: the scores of tile x are in registers
    uint64_t* o_full = p_last + 2;           // [2]   last P V of tile x finished; (APART) a P V of tile x finished
    uint64_t* o_drained = o_full + 2;        // [2]   4 softmax-warp arrivals: O_x of the item has been read
    uint64_t* start_full = o_drained + 2;    // [1]   relay: Q tiles of the item landed
    uint64_t* lead = start_full;             // [1]   (LEAD) 4 softmax-warp arrivals, once: tile A is three quarters through its first exponentials
    uint64_t* drain = start_full + 1;        // [1]   every product issued has finished; (APART) an arrival from each issuer
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + sl.misc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + sl.misc + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // what does not depend on the launch before: barriers, tensor memory
    if (tid == 0) {
        mbar_init(q_full + 0, 1); mbar_init(q_full + 1, 1); mbar_init(k0_full, 1);
        for (int i = 0; i < NK; ++i) { mbar_init(kv_full + i, 1); mbar_init(kv_free + i, G::APART ? 2 : 1); }
        for (int i = 0; i < G::NXMAX; ++i) mbar_init(x_full + i, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(s_full + i, 1); mbar_init(p_full + i, G::APART ? 4 : 5); mbar_init(p_last + i, 4); mbar_init(o_full + i, 1);
            mbar_init(o_drained + i, 4);
        }
        mbar_init(start_full, LEAD ? 4 : 1); mbar_init(drain, G::APART ? 2 : 1);
        mbar_fence_init();
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV);
        if (p.plan.mode) tma_prefetch_desc(&tmX);
    }
    __syncwarp();
    if (warp == 0) { tmem_alloc(tmem_holder, TMEM_COLS); tmem_relinquish(); }
    pdl_wait();
    // an earlier launch (or CTA) gave up on this workspace: nothing is started (every role finds `ok` false).  Fixed-length
    // launches look at the status behind their other first reads, which then make one trip to memory together (777 tokens on
    // 32/8 heads 28.4 -> 27.8 us per call); packed ones look at once (the other way cost 64 ragged sequences 1 %).
    const int status0 = *reinterpret_cast<volatile int*>(p.status);
    bool dead = false;
    if (TABLE) dead = __syncthreads_or(status0 != 0);
    const int hook_skip = p.status[4];
    // The limit of a wait: only one that has parked in vain asks for it.  Packed launches carry it as the 32-bit word it comes as: the
    // item records leave them one register less, and around 64 bits the compiler spilled at head_dim 128.  Three sequences of 1000 to
    // 8000 tokens at head_dim 128, unsteered: 28 / 4 heads 670 -> 654 us, 16 / 16 heads 413 -> 406; 64 of 256 to 2048 tokens of 32 / 8
    // heads 1140 -> 1068, of 50 to 500 tokens of 28 / 4 heads 142.7 -> 140.4; 200 of up to 128 tokens 159 -> 161; at head_dim 64 up to
    // 7 % faster (1.9 GHz).  Fixed-length launches keep 64 bits.  At head_dim 128 they have the registers (the word: level); at
    // head_dim 64 they spill them (8 bytes stored, 232 loaded), but only the comparison on that slow path reads them, and with the
    // word the tiles of long prompts went out of step (8192 tokens of 32 / 8 heads 383 -> 389 to 409 us).  In shared memory instead:
    // 200 packed sequences of up to 128 tokens 2 % slower.
    const uint64_t limit_set = p.status[5] > 0 ? (uint64_t)p.status[5] * 1000ull : kWaitLimitNs;
    const int limit_us = TABLE ? p.status[5] : 0;
    auto limit_ns = [&]() -> uint64_t {
        if (!TABLE) return limit_set;
        return limit_us > 0 ? (uint64_t)limit_us * 1000ull : kWaitLimitNs;
    };
    // steering info is kept in shared memory when it fits (a look-up then costs no trip to the caches): a byte per (sequence,
    // KV head) and a bit per (sequence, key tile)
    const bool info_local = p.steer && p.sched.B * p.sched.Hkv <= G::INFO_HEADS;
    uint8_t* info_bh = smem + sl.info;
    const int hot_words = (p.sched.n_qt + 31) / 32;
    const bool hot_local = p.steer && p.sched.B * hot_words <= G::INFO_WORDS;
    uint32_t* info_hot = reinterpret_cast<uint32_t*>(smem + sl.info + G::INFO_HEADS);
    auto tile_is_hot = [&](int b, int j) -> bool {
        return hot_local ? ((info_hot[b * hot_words + (j >> 5)] >> (j & 31)) & 1u) != 0 : __ldg(p.tile_hot + (size_t)b * p.sched.n_qt + j) != 0;
    };

    // all lanes of a warp wait on the same barrier and then agree on the outcome
    auto warp_wait = [&](uint64_t* bar, uint32_t parity, int where) -> bool {
        const bool ok = mbar_wait_within(bar, parity, abort_flag, p.status, where, limit_ns, PLAIN_POLLS);
        return __all_sync(0xffffffffu, ok);
    };

    // The CTA is persistent: it walks its share of the items (heaviest first; odd rounds run the CTAs in
    // reverse so that the shares come out even).  Every role goes through the same sequence of items by itself.
    // Fixed-length batches decode the item from its index; packed variable-length batches, where many index
    // slots are empty (row tiles beyond a short sequence), read a table from which those were dropped.
    const int n_items = TABLE ? *p.n_items : (int)p.sched.n_items_max;
    auto item_index = [&](int round) -> int {
        const int NG = (int)gridDim.x;
        const long long idx = (long long)round * NG + ((round & 1) ? (NG - 1 - (int)blockIdx.x) : (int)blockIdx.x);
        return idx < n_items ? (int)idx : -1;
    };
    // (table) the record of the next item is copied into a per-warp slot of shared memory while the current item
    // runs, so that no registers are held for it; lane 0 issues the copy and waits for it
    int round = 0, idx_next = TABLE ? item_index(0) : 0;
    auto prefetch = [&]() {
        if (TABLE && idx_next >= 0 && lane == 0) {
            const uint32_t dst = smem_u32(smem + sl.items + warp * 32);
            const ItemRecord* rec = p.items + idx_next;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(rec) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + 16), "l"(reinterpret_cast<const char*>(rec) + 16) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    };
    prefetch();
    // `steering`: also look up whether the item's keys are edited (only the producer and the MMA issuer need to know)
    auto next_item = [&](Item& it, bool steering = false) -> bool {
        ItemRecord rec;
        if (TABLE) {
            if (idx_next < 0) return false;
            const uint8_t* slot = smem + sl.items + warp * 32;
            if (lane == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            const int4 raw0 = *reinterpret_cast<const int4*>(slot), raw1 = *reinterpret_cast<const int4*>(slot + 16);
            rec.seq0 = raw0.x; rec.Lb = raw0.y; rec.bh = raw0.z; rec.hq = raw0.w;
            rec.qt = raw1.x; rec.n = raw1.y; rec.steer = raw1.z;
            __syncwarp();            // every lane has read the slot before it is refilled
            idx_next = item_index(++round);
            prefetch();
        } else {
            const int idx = item_index(round++);
            if (idx < 0) return false;
            decode_item(p.sched, idx, nullptr, rec);
            const int b = rec.bh & 0xffff, hkv = rec.bh >> 16;
            rec.steer = (steering && p.steer) ? (int)(info_local ? info_bh[b * p.sched.Hkv + hkv] : __ldg(p.bh_info + b * p.sched.Hkv + hkv)) : 0;
        }
        it.seq0 = rec.seq0; it.Lb = rec.Lb; it.b = rec.bh & 0xffff; it.hkv = rec.bh >> 16;
        it.hqA = rec.hq & 0xffff; it.hqB = rec.hq >> 16;
        it.qtA = rec.qt & 0xffff; it.qtB = rec.qt >> 16;
        it.nA = rec.n & 0xffff; it.nB = rec.n >> 16;
        it.n_kv = max(it.nA, it.nB);
        it.steer = steering && (rec.steer & 1) != 0 && p.plan.mode != 0;
        it.need_lo = it.steer && ((rec.steer & 2) != 0 || it.n_kv <= kLoTiles);
        return true;
    };

    if (tid == 0) {
        *abort_flag = 0; *reinterpret_cast<volatile float*>(smem + sl.misc + 8) = p.scale_log2;
    }
    // steering info into shared memory
    if (info_local)
        for (int i = tid; i < p.sched.B * p.sched.Hkv; i += NTHREADS) info_bh[i] = p.bh_info[i];
    if (hot_local)
        for (int w = warp; w < p.sched.B * hot_words; w += NTHREADS / 32) {
            const int b = w / hot_words, j = (w - b * hot_words) * 32 + lane;
            const uint32_t bits = __ballot_sync(0xffffffffu, j < p.sched.n_qt && p.tile_hot[(size_t)b * p.sched.n_qt + j] != 0);
            if (lane == 0) info_hot[w] = bits;
        }
    tc_fence_before();
    if (TABLE) __syncthreads();
    else dead = __syncthreads_or(status0 != 0);
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;

    // Key tiles are numbered through, item after item: global tile g is tile g - pr of the item whose first tile is pr.  Pair g
    // is V(g) and K(g+1), K(g+1) being the first key tile of the next item where V(g) is the last of this one; it uses
    // stage g % NK of the V ring and (g + 1) % NK of the K ring.  Running counts shared by all roles (each keeps its own
    // copy; they advance identically):
    //   pr     first key tile of the present item
    //   kv_free event g: the score products of key tile g and the P V of tile g - 1 are through (event 0: after the CTA's
    //          first score products; event g + 1: after step g)
    //   n_it   items so far (phases of start_full, q_full[0])
    //   n_o[x] items that had a tile x so far (phases of o_drained; of o_full too in head_dim 128)
    //   n_qb   items with a tile B so far (phase of q_full[1])
    //   n_hot  edited key tiles whose low parts were loaded / seen so far, over all items (stage and phase of x_full; both issuers of
    //          head_dim 64 see each, used or not)
    //   cx[x]  steps of tile x so far (phases of s_full, p_full, p_last; of s_free and, with a phase per step, o_full in head_dim 64)
    Item it;

    // final normalisation and store of this warp's 32 rows of tile x: `rows` of them exist, the first goes to `dst` (`inv`: 1 / row
    // sum of the lane's row)
    auto store_tile = [&](int x, OutT* dst, int rows, float inv) {
        tc_fence_after();
        const uint32_t tO = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + COL_O + D * x;
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
            uint32_t o[32];
            tmem_ld32(tO + c * 32, o);
            tmem_wait_ld_on(o);
            store_chunk32<OutT>(dst + c * 32, (size_t)p.sched.Hq * D, rows, o, inv, lane);
        }
        tc_fence_before();
        // O_x may be written again (the next item's first P V)
        __syncwarp();
        if (lane == 0) mbar_arrive(o_drained + x);
    };

    if (warp < 4) {
        reg_dec<REGS_CTRL>();
        // The control warps run their loops with all 32 lanes and elect one lane only around the issuing
        // instructions: addresses, descriptors and barrier phases then stay warp-uniform values.
        const bool leader = elect_one();
        if (warp == 0) {
            // ------------------------------------------------------------ TMA producer
            const int n_x = p.plan.nx;
            const bool staged = p.plan.mode != 0;       // key tiles with highlighted tokens come from the side buffer
            uint32_t pr = 0, n_it = 0, n_qb = 0, n_hot = 0;
            uint32_t ev_seen = 0;            // events [0, ev_seen) are known to have completed
            uint32_t ev_hot[G::NXMAX] = {0, 0, 0};      // per stage of the key-side operand: event that releases it, + 1
            // parity + 1 of the last load armed on each barrier (0: none), for the teardown after an abort
            uint32_t armed_q[2] = {0, 0}, armed_k0 = 0, armed_kv[NK], armed_x[G::NXMAX] = {0, 0, 0};
#pragma unroll
            for (int i = 0; i < NK; ++i) armed_kv[i] = 0;
            bool ok = !dead;
            auto see_event = [&](uint32_t e, int where) {        // events complete in order
                if (e < ev_seen) return;
                ok = warp_wait(kv_free + e % NK, (e / NK) & 1, where);
                ev_seen = e + 1;
            };
            // low parts of the edited key tile j of item `w` (global tile g) into the next stage
            auto load_x = [&](const Item& w, int j, uint32_t g) {
                uint32_t st = 0, prev = 0;
#pragma unroll
                for (int i = 0; i < G::NXMAX; ++i)
                    if ((int)(n_hot % (uint32_t)n_x) == i) { st = i; prev = ev_hot[i]; ev_hot[i] = g + 1; }
                if (prev) see_event(prev - 1, 14);       // the tile that used this stage before is through the tensor core
                if (!ok) return;
                if (leader) {
                    mbar_expect_tx(x_full + st, sl.xb);
#pragma unroll
                    for (int c = 0; c < NBLK; ++c)
                        tma_load_3d(smem + sl.x + st * sl.xb + c * BLK_BYTES, &tmX, x_full + st, D + c * 64, w.hkv, w.seq0 + j * BN);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < G::NXMAX; ++i)
                    if ((int)st == i) armed_x[i] = ((n_hot / (uint32_t)n_x) & 1) + 1;
                ++n_hot;
            };
            auto load_q = [&](const Item& w) {
                if (leader) {
                    mbar_expect_tx(q_full + 0, G::TILE);
#pragma unroll
                    for (int c = 0; c < NBLK; ++c)
                        tma_load_3d(smem + c * BLK_BYTES, &tmQ, q_full + 0, c * 64, w.hqA, w.seq0 + w.qtA * BM);
                    if (w.nB > 0) {
                        mbar_expect_tx(q_full + 1, G::TILE);
#pragma unroll
                        for (int c = 0; c < NBLK; ++c)
                            tma_load_3d(smem + G::TILE + c * BLK_BYTES, &tmQ, q_full + 1, c * 64, w.hqB, w.seq0 + w.qtB * BM);
                    }
                }
                __syncwarp();
                armed_q[0] = (n_it & 1) + 1; ++n_it;
                if (w.nB > 0) { armed_q[1] = (n_qb & 1) + 1; ++n_qb; }
            };
            bool have = ok && next_item(it, true);
            if (have) {
                load_q(it);
                const bool hot = it.steer && tile_is_hot(it.b, 0);
                if (leader) {
                    mbar_expect_tx(k0_full, G::TILE);
                    const CUtensorMap* km = (staged && hot) ? &tmX : &tmK;
#pragma unroll
                    for (int c = 0; c < NBLK; ++c) tma_load_3d(smem + sl.k + c * BLK_BYTES, km, k0_full, c * 64, it.hkv, it.seq0);
                }
                __syncwarp();
                armed_k0 = 1;
                if (hot && it.need_lo) load_x(it, 0, 0);
            }
            bool first = true;
            while (ok && have) {
                Item nx;
                const bool more_items = next_item(nx, true);
                // a pair's stages are released by the same event, the end of the step NK steps before
#pragma unroll 1
                for (int t = 0; t < it.n_kv; ++t) {
                    const uint32_t g = pr + (uint32_t)t;
                    if (g >= NK - 1) {
                        see_event(g - (NK - 1), 10);
                        if (!ok) break;
                    }
                    const bool inside = t + 1 < it.n_kv, more = inside || more_items;
                    const Item& w = inside ? it : nx;
                    const int j = inside ? t + 1 : 0;
                    const bool hot_n = more && w.steer && tile_is_hot(w.b, j);
                    // (test hook: one pair of the first item of CTA 0 is left out altogether, so that its wait runs out)
                    const bool skip = hook_skip > 0 && first && blockIdx.x == 0 && t + 1 == hook_skip;
                    if (leader && !skip) {
                        uint64_t* bar = kv_full + g % NK;
                        mbar_expect_tx(bar, more ? 2 * G::TILE : G::TILE);
#pragma unroll
                        for (int c = 0; c < NBLK; ++c)
                            tma_load_3d(smem + sl.v + (g % NK) * G::TILE + c * BLK_BYTES, &tmV, bar, c * 64, it.hkv, it.seq0 + t * BN);
                        if (more) {
                            const CUtensorMap* km = (staged && hot_n) ? &tmX : &tmK;
#pragma unroll
                            for (int c = 0; c < NBLK; ++c)
                                tma_load_3d(smem + sl.k + ((g + 1) % NK) * G::TILE + c * BLK_BYTES, km, bar, c * 64, w.hkv, w.seq0 + j * BN);
                        }
                    }
                    __syncwarp();
                    if (!skip) {
#pragma unroll
                        for (int i = 0; i < NK; ++i)
                            if ((int)(g % NK) == i) armed_kv[i] = ((g / NK) & 1) + 1;
                    }
                    if (hot_n && w.need_lo) {
                        load_x(w, j, g + 1);
                        if (!ok) break;
                    }
                }
                if (!ok) break;
                pr += it.n_kv;
                if (more_items) {
                    see_event(pr - 1, 12);        // the last score products of the item are through: its Q tiles may be replaced
                    if (!ok) break;
                    load_q(nx);
                }
                it = nx; have = more_items; first = false;
            }
            if (*abort_flag) {
                // loads that were armed may still be in flight: let them land before the shared memory is released
                auto settle = [&](uint64_t* bar, uint32_t armed) {
                    if (armed) mbar_wait_within(bar, armed - 1, nullptr, nullptr, 0, limit_ns);
                };
                settle(q_full + 0, armed_q[0]); settle(q_full + 1, armed_q[1]); settle(k0_full, armed_k0);
#pragma unroll
                for (int i = 0; i < NK; ++i) settle(kv_full + i, armed_kv[i]);
#pragma unroll
                for (int i = 0; i < G::NXMAX; ++i) settle(x_full + i, armed_x[i]);
            }
        } else if (G::APART && warp < 3) {
            // ------------------------------------------------------------ MMA issuer of tile x
            constexpr uint32_t IDESC_S = umma_idesc_bf16(BN, false);
            constexpr uint32_t IDESC_PV = umma_idesc_bf16(D, true);
            constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
            const int x = warp - 1;
            const uint32_t dQ = umma_desc_lo(smem_u32(smem + x * G::TILE), 16), dK = umma_desc_lo(smem_u32(smem + sl.k), 16);
            const uint32_t dX = umma_desc_lo(smem_u32(smem + sl.x), 16);
            const uint32_t dV = umma_desc_lo(smem_u32(smem + sl.v), BLK_BYTES);
            const uint32_t tS = tmem_base + COL_S + 128 * x, tO = tmem_base + COL_O + D * x, tP = tmem_base + COL_P + P_PITCH * x;
            const uint32_t n_x = p.plan.nx > 0 ? (uint32_t)p.plan.nx : 1u;
            uint32_t g = 0, n_q = 0, n_hot = 0, cx = 0, n_o = 0, n_s = 0;
            bool ok = !dead;
            uint32_t x_stage = 0;         // stage that holds the low parts of the key tile being multiplied
            // the low parts of the next edited key tile have landed (each of them is seen, in order, whether the tile uses it or not)
            auto see_x = [&]() {
                x_stage = n_hot % n_x;
                ok = warp_wait(x_full + x_stage, (n_hot / n_x) & 1, 32);
                ++n_hot;
            };
            auto see_q = [&](const Item& w) {
                if (x == 0 || w.nB > 0) { ok = warp_wait(q_full + x, n_q & 1, 20 + x); ++n_q; }
            };
            // scores against the key tile in stage `st`; `hot`: the tile is an edited one whose low parts are multiplied too
            auto issue_S = [&](uint32_t st, bool hot) {
                if (n_s > 0) {          // the scores before are in registers (each phase is seen, in order)
                    ok = warp_wait(s_free + x, (n_s - 1) & 1, 28 + x);
                    if (!ok) return;
                }
                ++n_s;
                const uint32_t kd = dK + st * (G::TILE >> 4);
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        // 16 elements along the contraction = 32 bytes inside a 64-element block
                        const uint32_t off = ((uint32_t)(ks >> 2) * BLK_BYTES + (uint32_t)(ks & 3) * 32) >> 4;
                        umma_ss(tS, dQ + off, DESC_HI, kd + off, DESC_HI, IDESC_S, ks > 0 ? 1u : 0u);
                    }
                    if (hot) {        // ... + Q (k'_lo)^T
                        const uint32_t xd = dX + x_stage * (sl.xb >> 4);
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            const uint32_t off = ((uint32_t)(ks >> 2) * BLK_BYTES + (uint32_t)(ks & 3) * 32) >> 4;
                            umma_ss(tS, dQ + off, DESC_HI, xd + off, DESC_HI, IDESC_S, 1u);
                        }
                    }
                    umma_commit(s_full + x);
                }
                __syncwarp();
            };
            // P of step j has been handed over: P V with the value tile in stage `st` (blocks of 16 keys: 2048 bytes of V, 8
            // columns of P).  Before an item's first P V writes O_x, the O_x of the last item that had a tile x has been read (its
            // phases count those items only, and each is seen, in order, by the next item that has the tile: a parity wait cannot
            // tell a phase from the one two later).
            auto step_PV = [&](uint32_t st, int j) {
                ok = warp_wait(p_full + x, (cx + j) & 1, 24 + 2 * x);
                if (ok && j == 0 && n_o > 0) ok = warp_wait(o_drained + x, (n_o - 1) & 1, 46 + x);
                if (!ok) return;
                const uint32_t vd = dV + st * (G::TILE >> 4);
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < BN / 16; ++ks)
                        umma_ts(tO, tP + (uint32_t)ks * 8, vd + (uint32_t)ks * (2048 >> 4), DESC_HI, IDESC_PV, (j > 0 || ks > 0) ? 1u : 0u);
                    umma_commit(o_full + x);
                }
                __syncwarp();
            };
            auto commit_event = [&](uint32_t st) {
                if (leader) umma_commit(kv_free + st);
                __syncwarp();
            };
            uint32_t st = 0;              // stage of the present value tile (of key tile g; the next key tile is in the stage after it)
            bool have = ok && next_item(it, true);
            if (have) {
                see_q(it);
                if (ok) ok = warp_wait(k0_full, 0, 23);
                const bool hot = it.need_lo && tile_is_hot(it.b, 0);
                if (ok && hot) see_x();
                if (ok) {
                    if (x == 0 || it.nB > 0) issue_S(0, hot);
                    commit_event(0);
                }
            }
            while (ok && have) {
                Item nx;
                const bool more = next_item(nx, true);
                const int n = x ? it.nB : it.nA, n_kv = it.n_kv, n_nx = !more ? 0 : x ? nx.nB : nx.nA;
                bool hot_nxt = it.need_lo && n_kv > 1 && tile_is_hot(it.b, 1);
#pragma unroll 1
                for (int j = 0; j < n_kv; ++j, ++g) {
                    const int j1 = j + 1;
                    const uint32_t st1 = st + 1 == (uint32_t)NK ? 0u : st + 1;
                    const bool turn = j1 == n_kv && more;      // on to the next item's scores
                    bool hot = hot_nxt && j1 < n_kv;
                    hot_nxt = it.need_lo && j + 2 < n_kv && tile_is_hot(it.b, j + 2);
                    ok = warp_wait(kv_full + g % NK, (g / NK) & 1, 25);       // V of this step and K of the next
                    if (!ok) break;
                    // inside an item the next scores go first: they only wait for the present ones to be in registers
                    if (!turn) {
                        if (hot) { see_x(); if (!ok) break; }
                        if (j1 < n) issue_S(st1, hot);
                        if (ok && j < n) step_PV(st, j);
                    } else {
                        if (j < n) step_PV(st, j);
                        if (ok) see_q(nx);
                        if (!ok) break;
                        hot = nx.need_lo && tile_is_hot(nx.b, 0);
                        if (hot) { see_x(); if (!ok) break; }
                        if (n_nx > 0) issue_S(st1, hot);
                    }
                    if (!ok) break;
                    commit_event(st1);     // K(g+1) and V(g) may be overwritten, as far as this tile goes
                    st = st1;
                }
                if (!ok) break;
                cx += n;
                if (n > 0) ++n_o;
                it = nx; have = more;
            }
        } else if (!G::APART && warp == 1) {
            // ------------------------------------------------------------ MMA issuer
            constexpr uint32_t IDESC_S = umma_idesc_bf16(BN, false);
            constexpr uint32_t IDESC_PV = umma_idesc_bf16(D, true);
            constexpr uint32_t DESC_HI = umma_desc_hi_sw128(1024);
            const uint32_t dQ = umma_desc_lo(smem_u32(smem), 16), dK = umma_desc_lo(smem_u32(smem + sl.k), 16);
            const uint32_t dX = umma_desc_lo(smem_u32(smem + sl.x), 16);
            const uint32_t dV = umma_desc_lo(smem_u32(smem + sl.v), BLK_BYTES);
            const uint32_t n_x = p.plan.nx > 0 ? (uint32_t)p.plan.nx : 1u;
            uint32_t n_it = 0, n_hot = 0;
            uint32_t cx[2] = {0, 0};      // steps of tile A / B so far
            uint32_t n_o[2] = {0, 0};     // items that had a tile A / B so far
            bool ok = !dead;
            uint32_t x_stage = 0;         // stage that holds the low parts of the key tile being multiplied
            // the low parts of the next edited key tile have landed (once per tile, before its first use)
            auto see_x = [&]() {
                x_stage = n_hot % n_x;
                ok = warp_wait(x_full + x_stage, (n_hot / n_x) & 1, 32);
                ++n_hot;
            };
            // scores of tile x against the key tile in stage `st`; `hot`: the tile is an edited one whose low parts are multiplied too
            auto issue_S = [&](int x, uint32_t st, bool hot) {
                const uint32_t kd = dK + st * (G::TILE >> 4), qd = dQ + (uint32_t)x * (G::TILE >> 4);
                const uint32_t dst = tmem_base + COL_S + 128 * x;
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        // 16 elements along the contraction = 32 bytes inside a 64-element block
                        const uint32_t off = ((uint32_t)(ks >> 2) * BLK_BYTES + (uint32_t)(ks & 3) * 32) >> 4;
                        umma_ss(dst, qd + off, DESC_HI, kd + off, DESC_HI, IDESC_S, ks > 0 ? 1u : 0u);
                    }
                    if (hot) {        // ... + Q (k'_lo)^T
                        const uint32_t xd = dX + x_stage * (sl.xb >> 4);
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks) {
                            const uint32_t off = ((uint32_t)(ks >> 2) * BLK_BYTES + (uint32_t)(ks & 3) * 32) >> 4;
                            umma_ss(dst, qd + off, DESC_HI, xd + off, DESC_HI, IDESC_S, 1u);
                        }
                    }
                    umma_commit(s_full + x);
                }
                __syncwarp();
            };
            // P V of tile x with the value tile in stage `st`, key blocks [ks0, ks1) of 16 keys (2048 bytes of V, 8 columns of P)
            auto issue_PV = [&](int x, uint32_t st, bool fresh, int ks0, int ks1, bool last) {
                const uint32_t vd = dV + st * (G::TILE >> 4);
                const uint32_t dst = tmem_base + COL_O + D * x, src = tmem_base + COL_S + 128 * x;
                tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int ks = 0; ks < BN / 16; ++ks)
                        if (ks >= ks0 && ks < ks1)
                            umma_ts(dst, src + (uint32_t)ks * 8, vd + (uint32_t)ks * (2048 >> 4), DESC_HI, IDESC_PV,
                                    (!fresh || ks > 0) ? 1u : 0u);
                    if (last) umma_commit(o_full + x);
                }
                __syncwarp();
            };
            // P of tile x and step j has been handed over: P V with the value tile in stage `st`.  Before an item's first P V
            // writes O_x, the O_x of the last item that had a tile x has been read (its phases count those items only, and each
            // is seen, in order, by the next item that has the tile: a parity wait cannot tell a phase from the one two later).
            auto step_PV = [&](int x, uint32_t st, int j, int n) {
                if (j == 0 && n_o[x] > 0) {
                    ok = warp_wait(o_drained + x, (n_o[x] - 1) & 1, 46 + x);
                    if (!ok) return;
                }
                issue_PV(x, st, j == 0, 0, G::KP1, false);
                ok = warp_wait(p_last + x, (cx[x] + j) & 1, 28 + x);
                if (!ok) return;
                issue_PV(x, st, j == 0, G::KP1, BN / 16, j == n - 1);
            };
            auto commit_event = [&](uint32_t st) {
                if (leader) umma_commit(kv_free + st);
                __syncwarp();
            };
            uint32_t st = 0;              // stage of the present value tile (of key tile g; the next key tile is in the stage after it)
            bool have = ok && next_item(it, true);
            if (have) {
                ok = warp_wait(start_full, 0, 20);
                const bool hot = it.need_lo && tile_is_hot(it.b, 0);
                if (ok && hot) see_x();
                if (ok) {
                    issue_S(0, 0, hot);
                    if (it.nB > 0) issue_S(1, 0, hot);
                    commit_event(0);
                }
            }
            // One thread issues for both tiles, in a fixed order (A then B in every step): the in-order tensor
            // pipe then keeps the two tiles half a period apart (softmax of one tile under the MMAs of the other).
            while (ok && have) {
                Item nx;
                const bool more = next_item(nx, true);
                const int nA = it.nA, nB = it.nB, n_kv = it.n_kv;
                ++n_it;
                bool started = false;          // the next item's operands have been seen
                bool hot0 = false;             // its first key tile takes the low parts
                auto start_next = [&]() {
                    if (started) return;
                    started = true;
                    ok = warp_wait(start_full, n_it & 1, 21);
                    hot0 = nx.need_lo && tile_is_hot(nx.b, 0);
                    if (ok && hot0) see_x();
                };
                bool hot_nxt = it.need_lo && n_kv > 1 && tile_is_hot(it.b, 1);
#pragma unroll 1
                for (int j = 0; j < n_kv; ++j) {
                    const int j1 = j + 1;
                    const uint32_t st1 = st + 1 == (uint32_t)NK ? 0u : st + 1;
                    const bool hot_j1 = hot_nxt && j1 < n_kv, turn = j1 == n_kv && more;      // turn: on to the next item's scores
                    hot_nxt = it.need_lo && j + 2 < n_kv && tile_is_hot(it.b, j + 2);
                    bool x_seen = false;
                    // V of this step and K of the next have landed once p_full completes: the relay warp vouches
                    // for them there, so this warp has no waits of its own for operands (every wait here is a
                    // bubble in the tensor pipe: its queue is only a couple of MMAs deep)
                    if (j < nA) {
                        ok = warp_wait(p_full + 0, (cx[0] + j) & 1, 24);
                        if (ok) step_PV(0, st, j, nA);
                        if (!ok) break;
                        if (j1 < nA) {
                            if (hot_j1) { see_x(); x_seen = true; if (!ok) break; }
                            issue_S(0, st1, hot_j1);
                        } else if (turn) {
                            start_next();
                            if (!ok) break;
                            issue_S(0, st1, hot0);
                        }
                    }
                    if (j < nB) {
                        ok = warp_wait(p_full + 1, (cx[1] + j) & 1, 26);
                        if (!ok) break;
                        if (turn && j >= nA) {        // tile A has been through for a step: it goes on first
                            start_next();
                            if (!ok) break;
                            issue_S(0, st1, hot0);
                        }
                        step_PV(1, st, j, nB);
                        if (!ok) break;
                    }
                    if (j1 < nB) {
                        if (hot_j1 && !x_seen) { see_x(); if (!ok) break; }      // tile A does not use this key tile
                        issue_S(1, st1, hot_j1);
                    } else if (turn && nx.nB > 0) {
                        start_next();
                        if (!ok) break;
                        issue_S(1, st1, hot0);
                    }
                    commit_event(st1);     // K(g+1) and V(g) may be overwritten
                    st = st1;
                }
                if (!ok) break;
                cx[0] += nA; cx[1] += nB;
                ++n_o[0];
                if (nB > 0) ++n_o[1];
                it = nx; have = more;
            }
        } else if (!G::APART && warp == 2) {
            // ------------------------------------------------------------ operand relay: "the operands have landed", once per
            // item for Q (and the CTA's first K), and per step "V(g) and K(g+1) landed" as a fifth arrival on the
            // P hand-off barrier, so that the MMA issuer waits on one barrier per hand-off
            uint32_t pr = 0, n_it = 0, n_qb = 0, cx[2] = {0, 0};
            bool ok = !dead;
            auto q_landed = [&](const Item& w) {
                ok = warp_wait(q_full + 0, n_it & 1, 21);
                ++n_it;
                if (ok && w.nB > 0) { ok = warp_wait(q_full + 1, n_qb & 1, 22); ++n_qb; }
                if (ok && n_it == 1) ok = warp_wait(k0_full, 0, 23);
                if (ok && lane == 0) mbar_arrive(start_full);
                __syncwarp();
            };
            bool have = ok && next_item(it);
            if (have) q_landed(it);
            while (ok && have) {
                Item nx;
                const bool more = next_item(nx);
#pragma unroll 1
                for (int j = 0; j < it.n_kv; ++j) {
                    const uint32_t g = pr + j;
                    ok = warp_wait(kv_full + g % NK, (g / NK) & 1, 25);
                    if (!ok) break;
                    if (lane == 0) {
                        if (j < it.nA) mbar_arrive(p_full + 0);
                        if (j < it.nB) mbar_arrive(p_full + 1);
                    }
                    __syncwarp();
                    // the next item's Q tiles: loaded when this item's last score products are through, so they land while its
                    // last softmax runs
                    if (j + 1 == it.n_kv && more) { q_landed(nx); if (!ok) break; }
                    // stay within the phase: the next arrival may only come after this phase has completed
                    if (j < it.nA) ok = warp_wait(p_full + 0, (cx[0] + j) & 1, 33);
                    if (ok && j < it.nB) ok = warp_wait(p_full + 1, (cx[1] + j) & 1, 34);
                    if (!ok) break;
                }
                pr += it.n_kv; cx[0] += it.nA; cx[1] += it.nB;
                it = nx; have = more;
            }
        }
    } else {
        // ------------------------------------------------------------ softmax of tile x, one query row per thread
        reg_inc<REGS_SOFTMAX>();
        const int x = (warp - 4) >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t tS = t_lane + COL_S + 128 * x, tO = t_lane + COL_O + D * x, tP = t_lane + COL_P + P_PITCH * x;
        const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
        uint32_t cX = 0, n_o = 0;       // steps and items of this tile so far
        OutT* pend_dst = nullptr;       // (APART) the last item's output: where it goes (null: nothing to store), its rows, 1 / row sum
        int pend_rows = 0;
        float pend_inv = 0.f;
        bool ok = !dead;
        while (ok && next_item(it)) {
            const int nX = x ? it.nB : it.nA;
            const int hqX = x ? it.hqB : it.hqA, qtX = x ? it.qtB : it.qtA;
            float m_run = -INFINITY, l_run = 0.f;
#pragma unroll 1
            for (int j = 0; j < nX; ++j) {
                ok = warp_wait(s_full + x, (cX + j) & 1, 40 + x);
                if (!ok) break;
                tc_fence_after();
                // the whole score row of this thread: 128 fp32 values in registers
                uint32_t v[128];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, reinterpret_cast<uint32_t(&)[32]>(v[32 * c]));
                tmem_wait_ld();
                if (G::APART) {         // the next scores may be formed
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(s_free + x);
                }
                if (j == nX - 1) {       // diagonal tile: keys after the query are masked
#pragma unroll
                    for (int e = 0; e < 128; ++e)
                        if (e > row) v[e] = 0xff800000u;
                }
                float mx[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    mx[q] = fmaxf(__uint_as_float(v[16 * q]), __uint_as_float(v[16 * q + 1]));
#pragma unroll
                    for (int e = 2; e < 16; e += 2) mx[q] = max3(mx[q], __uint_as_float(v[16 * q + e]), __uint_as_float(v[16 * q + e + 1]));
                }
                const float mx_all = fmaxf(max3(mx[0], mx[1], mx[2]), max3(mx[3], mx[4], max3(mx[5], mx[6], mx[7])));
                const float m_new = fmaxf(m_run, mx_all * p.scale_log2);
                // raise the running maximum only when it moved a lot; p may then exceed 1 (up to 2^8), which is harmless
                const bool raise = (m_new - m_run) > LAZY_RESCALE_LOG2;      // true on the first tile (m_run = -inf)
                const float factor = raise ? fast_exp2(m_run - m_new) : 1.f;
                if (raise) m_run = m_new;
                if (G::APART && (j > 0 || pend_dst != nullptr)) {       // the P V before is through: P may be written, O read or written
                    ok = warp_wait(o_full + x, (cX + j - 1) & 1, 48 + x);
                    if (!ok) break;
                    tc_fence_after();
                }
                if (j > 0 && __any_sync(0xffffffffu, raise)) {
                    uint32_t o[32];
#pragma unroll 1
                    for (int c = 0; c < D / 32; ++c) {
                        tmem_ld32(tO + c * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * factor);
                        tmem_st32(tO + c * 32, o);
                    }
                }
                if (LEAD && x == 1 && j == 0) {
                    ok = warp_wait(lead, 0, 36);
                    if (!ok) break;
                }
                float2 sc_piece = sc2;
                const float2 nm2 = make_float2(-m_run, -m_run);
                float2 sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t pk16[16];
#pragma unroll
                    for (int e2 = 0; e2 < 16; ++e2) {
                        const int e = 32 * c + 2 * e2;
                        const float2 arg = __ffma2_rn(make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), sc_piece, nm2);
                        const float2 pe = make_float2(fast_exp2(arg.x), fast_exp2(arg.y));
                        sum[e2 & 1] = __fadd2_rn(sum[e2 & 1], pe);
                        pk16[e2] = pack_bf16(pe.x, pe.y);
                    }
                    if (LEAD && c == 2 && x == 0 && j == 0 && lane == 0) mbar_arrive(lead);
                    tmem_st16(tP + c * 16, pk16);     // P (bf16 pairs); head_dim 128: over score columns that are already in registers
                    if (!G::APART && 2 * c + 2 == G::KP1) {      // the first piece is in place: the tensor core may start on it
                        tmem_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(p_full + x);
                        // The scale of the other keys comes from shared memory, read here: their exponentials then cannot be moved
                        // ahead of the hand-over (the compiler did, which left 70 cycles between the two pieces and the tensor core
                        // without work under the last exponentials).  A traced step of a tile pair 3190 -> 3060 cycles (2970 on
                        // average over CTAs and steps, plus 4200 an item): 4 x 4096 tokens of 32 / 8 heads of 128 563 -> 553 us,
                        // 1 x 32768 of 28 / 4 6800 -> 6600 (back to back, about 1.5 GHz).
                        float again;
                        asm volatile("ld.volatile.shared.f32 %0, [%1];" : "=f"(again) : "r"(smem_u32(smem + sl.misc + 8)) : "memory");
                        sc_piece = make_float2(again, again);
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive((G::APART ? p_full : p_last) + x);
                const float2 s2 = __fadd2_rn(sum[0], sum[1]);
                l_run = l_run * factor + (s2.x + s2.y);
                if (G::APART && j == 0 && pend_dst != nullptr) {
                    store_tile(x, pend_dst, pend_rows, pend_inv);
                    pend_dst = nullptr;
                }
            }
            if (!ok) break;
            cX += nX;
            if (nX > 0) {
                const float inv = 1.f / l_run;
                const int qpos = qtX * BM + row, q0 = qtX * BM + (warp & 3) * 32;
                OutT* dst = static_cast<OutT*>(p.O) + ((size_t)(it.seq0 + q0) * p.sched.Hq + hqX) * D;
                if (p.lse != nullptr && qpos < it.Lb)
                    p.lse[(size_t)(it.seq0 + qpos) * p.sched.Hq + hqX] = (m_run + log2f(l_run)) * 0.6931471805599453f;
                if (G::APART) {
                    // the last P V runs on; its output is stored behind the first weights of the next item
                    pend_dst = dst; pend_rows = it.Lb - q0; pend_inv = inv;
                } else {
                    ok = warp_wait(o_full + x, n_o & 1, 44 + x);
                    if (!ok) break;
                    store_tile(x, dst, it.Lb - q0, inv);
                    ++n_o;
                }
            }
        }
        if (G::APART && ok && pend_dst != nullptr) {
            ok = warp_wait(o_full + x, (cX - 1) & 1, 44 + x);
            if (ok) store_tile(x, pend_dst, pend_rows, pend_inv);
        }
    }

    // ---------------------------------------------------------------- teardown (also after an abort)
    pdl_release();
    tc_fence_before();
    __syncthreads();
    if (warp == 1 || (G::APART && warp == 2)) {
        // every product issued has finished before tensor and shared memory are released
        if (elect_one()) umma_commit(drain);
        __syncwarp();
        mbar_wait_within(drain, 0, nullptr, p.status, 90, limit_ns);
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem_base, TMEM_COLS);
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (fn == nullptr) {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// bf16 tensor [T, H, d] viewed as (d, H, T); tiles of 64 x 1 x box_rows with the 128-byte swizzle.
bool make_tile_map(CUtensorMap* m, const void* base, int d, int H, long long T, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)H, (cuuint64_t)T};
    cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)H * d * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_row_map(CUtensorMap* m, const void* base, int cols, long long T) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)T};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64, 1}, estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Per-device facts, looked up once per device (a process may drive several GPUs from several threads).
bool device_info(int* n_sm) {
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int sm_of[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    std::lock_guard<std::mutex> lock(mu);
    if (sm_of[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return false;
        sm_of[dev] = n;
    }
    *n_sm = sm_of[dev];
    return true;
}

struct TileMaps { CUtensorMap q, k, v, x; };

template <int D, typename OutT, bool TABLE>
static seka_status launch_attn_t(const TileMaps& tm, const AttnParams& p, cudaStream_t st) {
    const SmemPlan sl = smem_plan<D>(p.plan);
    const uint32_t dyn = sl.total;
    if (dyn > SMEM_LIMIT) return SEKA_ERR_UNSUPPORTED;
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    auto kern = seka_attn_fwd_kernel<D, OutT, TABLE>;
    if constexpr (Geo<D>::APART) {
        // One item per CTA, two query heads at the same rows: without the aliasing of P and S nothing keeps such tiles apart, so
        // they load, search their maximum and use the special-function unit in step, each half idle.  The lead undoes that.
        // Unsteered, us (P over S / in step / with the lead, 1.9 GHz): 16 / 8 heads, 257 tokens 9.6 / 9.9 / 9.1, 512 tokens
        // 11.3 / 11.7 / 10.6, 1024 tokens 18.2 / 18.7 / 16.8; 32 / 8 heads, 512 tokens 11.7 / 12.0 / 10.9; 4 / 2 heads, 2048 tokens
        // 30.0 / 30.5 / 28.2; three packed sequences of 100 to 900 tokens of 8 / 2 heads 17.5 / 18.5 / 16.7 (a packed launch has at
        // most n_items_max items).  A lead of half of the exponentials 1 to 4 % slower, of a quarter 10 %.  Steered launches, which start
        // under their preparation, up to 1024 tokens only (16 / 8 heads 777 tokens 23.3 / 23.3 / 22.2; 1500 tokens 33.8 / 32.3 /
        // 33.0, 8 / 4 heads 3000 tokens 52.9 / 49.1 / 53.0).  Not with several items per CTA: the tiles are better off in step
        // there (8192 tokens of 32 / 8 heads 383 -> 440).
        const int most = p.steer ? 8 : 16;
        if (p.sched.pair_heads && p.sched.n_items_max <= (long long)n_sm && p.sched.n_qt > 1 && p.sched.n_qt <= most)
            kern = seka_attn_fwd_kernel<D, OutT, TABLE, true>;
    }
    // the attribute belongs to the function on the current device: set on every call (a cheap driver call), so that a
    // process that drives several devices, or calls from several threads, needs no bookkeeping here
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) != cudaSuccess) return SEKA_ERR_CUDA;
    // persistent CTAs, one per SM (the kernel needs the whole SM: all of tensor memory and most of shared memory)
    const unsigned grid = (unsigned)(p.sched.n_items_max < (long long)n_sm ? p.sched.n_items_max : (long long)n_sm);
    if (grid == 0) return SEKA_OK;
    // A launch of one item per CTA is placed under the tail of its preparation (one prompt of 777 tokens 32.6 -> 31.2 us, the
    // toy layer 24.6 -> 21.2 us per call).  Longer ones are not: their CTAs then land on the SMs in the order in which these
    // become free, and CTAs that share a KV head no longer sit next to each other (4 x 4096 tokens 589 -> 607 us).
    return launch_kernel(p.sched.n_items_max <= (long long)grid, kern, grid, NTHREADS, dyn, st, tm.q, tm.k, tm.v, tm.x, p);
}

template <int D, typename OutT>
static seka_status launch_attn(const TileMaps& tm, const AttnParams& p, bool table, cudaStream_t st) {
    return table ? launch_attn_t<D, OutT, true>(tm, p, st) : launch_attn_t<D, OutT, false>(tm, p, st);
}

// The fused forward behind both entry points: coefficients either given (`alpha`, may be null) or, with `sigma`
// set, routed inside the preparation launch (Eq. 6) and reported through `alpha_out`.
static seka_status attention_fwd_impl(const seka_shape* shape, const void* Q, const void* K, const void* V,
                                      void* O, float* lse, const uint8_t* mask, const float* U,
                                      const float* alpha, const float* sigma, int k_route, float* alpha_out,
                                      const float* gain, const uint8_t* head_enable,
                                      void* workspace, size_t workspace_bytes, void* cuda_stream) {
    seka_status stc = validate_shape(shape);
    if (stc != SEKA_OK) return stc;
    const int T = shape_total_tokens(shape);
    if (T == 0 || shape->batch == 0 || shape->max_seqlen == 0) return SEKA_OK;
    if (!Q || !K || !V || !O) return SEKA_ERR_INVALID_ARG;
    if (((uintptr_t)Q | (uintptr_t)K | (uintptr_t)V | (uintptr_t)O) & 15) return SEKA_ERR_INVALID_ARG;
    const bool steer = mask != nullptr && U != nullptr;
    if (steer && !gain) return SEKA_ERR_INVALID_ARG;
    const WorkspaceLayout w = workspace_layout(shape);
    const int D = shape->head_dim, Hq = shape->n_q_heads, Hkv = shape->n_kv_heads;
    const Sched sched = make_sched(shape);
    if (w.n_tiles > 32767 || Hq > 32767 || shape->batch > 65535 || sched.n_items_max > 0x7fffffffLL) return SEKA_ERR_UNSUPPORTED;   // item records pack 15/16-bit fields
    if (!workspace || workspace_bytes < w.total || ((uintptr_t)workspace & 255)) return SEKA_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    char* ws = static_cast<char*>(workspace);

    AttnParams p;
    p.plan = make_steer_plan(shape, steer);
    p.sched = sched;
    void* X = ws + w.x_off;
    uint8_t* tile_hot = reinterpret_cast<uint8_t*>(ws + w.hot_off);
    uint8_t* bh_info = reinterpret_cast<uint8_t*>(ws + w.info_off);
    ItemRecord* items = reinterpret_cast<ItemRecord*>(ws + w.item_off);
    int* n_items = reinterpret_cast<int*>(ws) + 3;
    const bool table = shape->cu_seqlens != nullptr;

    // The preparation: the edited keys of the tiles with highlighted tokens, the item table of a packed batch and the bf16
    // copies of fp32 inputs, each in blocks of its own (nothing is launched if none of them is needed).
    int n_sm = 0;
    if (!device_info(&n_sm)) return SEKA_ERR_CUDA;
    PrepJobs jobs = {};
    jobs.sched = sched; jobs.cu = shape->cu_seqlens; jobs.items = items; jobs.item_count = n_items;
    if (steer) jobs.steer = SteerIn{gain, alpha, head_enable, shape->n_experts, sigma != nullptr ? 1 : 0};
    if (table) jobs.n_items_blocks = sched.rs;
    const void *q16 = Q, *k16 = K, *v16 = V;
    if (shape->dtype == SEKA_F32) {
        const size_t nq = (size_t)T * Hq * D, nk = (size_t)T * Hkv * D;      // multiples of 4
        char* cq = ws + w.cvt_off;
        char* ck = cq + align_up(nq * 2, 256);
        char* cv = ck + align_up(nk * 2, 256);
        const void* in[3] = {Q, K, V};
        char* out[3] = {cq, ck, cv};
        for (int i = 0; i < 3; ++i) {
            jobs.conv.in[i] = static_cast<const float4*>(in[i]); jobs.conv.out[i] = reinterpret_cast<uint2*>(out[i]);
            jobs.conv.n4[i] = (i == 0 ? nq : nk) / 4;
        }
        const long long want = (long long)((nq + 2 * nk) / (4 * 4 * PREP_THREADS)) + 1, most = 4LL * n_sm;
        jobs.n_conv_blocks = (int)(want < most ? want : most);
        q16 = cq; k16 = ck; v16 = cv;
    }
    if (steer) {
        RouteArgs route = {};
        if (sigma != nullptr) route = RouteArgs{Q, shape->dtype == SEKA_F32 ? 1 : 0, sigma, k_route, Hq, alpha_out};
        stc = launch_stage_keys(shape, w, K, mask, U, alpha, gain, head_enable, ws, jobs, route, st);
    } else {
        stc = launch_prep_plain(jobs, st);
    }
    if (stc != SEKA_OK) return stc;

    TileMaps tm;
    if (!make_tile_map(&tm.q, q16, D, Hq, T, BM) || !make_tile_map(&tm.k, k16, D, Hkv, T, BN) ||
        !make_tile_map(&tm.v, v16, D, Hkv, T, BN))
        return SEKA_ERR_CUDA;
    tm.x = tm.k;      // never dereferenced without steering
    if (p.plan.mode != 0 && !make_tile_map(&tm.x, X, p.plan.xcols, Hkv, T, BN)) return SEKA_ERR_CUDA;

    p.O = O; p.lse = lse;
    p.tile_hot = tile_hot; p.bh_info = bh_info; p.status = reinterpret_cast<int*>(ws);
    p.steer = steer ? 1 : 0;
    p.items = items; p.n_items = n_items;
    const float scale = shape->softmax_scale > 0.f ? shape->softmax_scale : 1.f / sqrtf((float)D);
    p.scale_log2 = scale * 1.4426950408889634f;

    if (D == 128) {
        return shape->dtype == SEKA_F32 ? launch_attn<128, float>(tm, p, table, st)
                                        : launch_attn<128, __nv_bfloat16>(tm, p, table, st);
    }
    return shape->dtype == SEKA_F32 ? launch_attn<64, float>(tm, p, table, st)
                                    : launch_attn<64, __nv_bfloat16>(tm, p, table, st);
}

}  // namespace seka

extern "C" seka_status seka_attention_fwd(const seka_shape* shape, const void* Q, const void* K, const void* V,
                                          void* O, float* lse, const uint8_t* mask, const float* U,
                                          const float* alpha, const float* gain, const uint8_t* head_enable,
                                          void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return seka::attention_fwd_impl(shape, Q, K, V, O, lse, mask, U, alpha, nullptr, 0, nullptr, gain, head_enable,
                                    workspace, workspace_bytes, cuda_stream);
}

extern "C" seka_status seka_attention_fwd_routed(const seka_shape* shape, const void* Q, const void* K, const void* V,
                                                 void* O, float* lse, const uint8_t* mask, const float* U,
                                                 const float* sigma, int32_t k_route, float* alpha_out,
                                                 const float* gain, const uint8_t* head_enable,
                                                 void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (shape == nullptr || mask == nullptr || U == nullptr || sigma == nullptr) return SEKA_ERR_INVALID_ARG;
    if (k_route < 0 || k_route > shape->rank) return SEKA_ERR_INVALID_ARG;
    if (k_route == 0) k_route = shape->rank;
    return seka::attention_fwd_impl(shape, Q, K, V, O, lse, mask, U, nullptr, sigma, k_route, alpha_out, gain,
                                    head_enable, workspace, workspace_bytes, cuda_stream);
}

extern "C" size_t seka_host_staging_bytes(const seka_shape* shape) {
    using namespace seka;
    if (validate_shape(shape) != SEKA_OK) return 0;
    const size_t T = (size_t)shape_total_tokens(shape), esz = shape->dtype == SEKA_F32 ? 4 : 2;
    const size_t nq = align_up(T * shape->n_q_heads * shape->head_dim * esz, 256);
    const size_t nk = align_up(T * shape->n_kv_heads * shape->head_dim * esz, 256);
    return 2 * nq + 2 * nk + align_up(T, 256) + align_up(T * shape->n_q_heads * 4, 256);
}

namespace seka {
// Per device: events that mark the end of the compute of each part of the last host-buffer call, and that call's
// geometry.  The next call's copies into the staging buffer wait for them instead of for the caller's stream, so its
// input copies run while the previous call's output is still on its way back.
struct HostPipeState {
    cudaEvent_t cmp[8] = {};
    bool made = false, valid = false;
    const void* staging = nullptr;
    int parts = 0;
    size_t tok_per = 0;
};
static std::mutex g_host_pipe_mutex;
static HostPipeState g_host_pipe[64];
}  // namespace seka

extern "C" seka_status seka_attention_fwd_host(const seka_shape* shape, const void* h_Q, const void* h_K,
                                               const void* h_V, void* h_O, float* h_lse, const uint8_t* h_mask,
                                               const float* U, const float* alpha, const float* gain,
                                               const uint8_t* head_enable, void* staging, size_t staging_bytes,
                                               void* workspace, size_t workspace_bytes, void* cuda_stream) {
    using namespace seka;
    seka_status stc = validate_shape(shape);
    if (stc != SEKA_OK) return stc;
    const size_t T = (size_t)shape_total_tokens(shape);
    if (T == 0) return SEKA_OK;
    if (!h_Q || !h_K || !h_V || !h_O) return SEKA_ERR_INVALID_ARG;
    if (!staging || staging_bytes < seka_host_staging_bytes(shape) || ((uintptr_t)staging & 255)) return SEKA_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const size_t esz = shape->dtype == SEKA_F32 ? 4 : 2;
    const size_t rq = (size_t)shape->n_q_heads * shape->head_dim * esz, rk = (size_t)shape->n_kv_heads * shape->head_dim * esz;
    const size_t bq = T * rq, bk = T * rk;
    char* dq = static_cast<char*>(staging);
    char* dk = dq + align_up(bq, 256);
    char* dv = dk + align_up(bk, 256);
    char* dO = dv + align_up(bk, 256);
    char* dm = dO + align_up(bq, 256);
    char* dl = dm + align_up(T, 256);
    // Sequences are independent, so a fixed-length batch is cut into parts (one sequence each, at most eight) that go
    // through a three-stage pipeline: the inputs of part i + 1 are copied in (a second stream) while part i is computed
    // (the caller's stream) and the output of part i - 1 is copied out (a third stream); the two copy directions share
    // the link at full duplex.  A packed batch (cu_seqlens) runs as one part.
    int parts = 1;
    if (shape->cu_seqlens == nullptr && shape->batch > 1) {
        parts = shape->batch < 8 ? shape->batch : 8;
        while (shape->batch % parts) --parts;
    }
    const int seq_per = shape->batch / parts;
    const size_t tok_per = (size_t)seq_per * shape->max_seqlen;
    cudaStream_t s_in = nullptr, s_out = nullptr;
    cudaEvent_t ev_tail = nullptr, ev_in[8] = {}, ev_out = nullptr;
    bool okc = true;
    auto make_event = [&](cudaEvent_t* e) { okc = okc && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; };
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SEKA_ERR_CUDA;
    std::lock_guard<std::mutex> pipe_lock(g_host_pipe_mutex);
    HostPipeState& hs = g_host_pipe[dev];
    if (!hs.made) {
        for (int i = 0; i < 8; ++i) make_event(&hs.cmp[i]);
        if (!okc) return SEKA_ERR_CUDA;
        hs.made = true;
    }
    // The staging buffer of the call before may still be read by its kernels.  Same buffer cut the same way: part i
    // waits for that call's part i; anything else: for its last part.
    const bool same_cut = hs.valid && hs.staging == staging && hs.parts == parts && hs.tok_per == tok_per;
    const int prev_last = hs.valid ? hs.parts - 1 : -1;
    if (parts > 1) {
        okc = okc && cudaStreamCreateWithFlags(&s_in, cudaStreamNonBlocking) == cudaSuccess;
        okc = okc && cudaStreamCreateWithFlags(&s_out, cudaStreamNonBlocking) == cudaSuccess;
        make_event(&ev_tail); make_event(&ev_out);
        for (int i = 0; i < parts; ++i) make_event(&ev_in[i]);
    } else {
        s_in = st; s_out = st;
    }
    seka_shape part = *shape;
    part.batch = seq_per;
    part.total_tokens = shape->cu_seqlens ? shape->total_tokens : 0;
    for (int i = 0; i < parts && okc && stc == SEKA_OK; ++i) {
        const size_t t0 = (size_t)i * tok_per, nt = parts > 1 ? tok_per : T;
        if (parts > 1 && prev_last >= 0 && (same_cut || i == 0))
            okc = okc && cudaStreamWaitEvent(s_in, hs.cmp[same_cut ? i : prev_last], 0) == cudaSuccess;
        okc = okc && cudaMemcpyAsync(dq + t0 * rq, static_cast<const char*>(h_Q) + t0 * rq, nt * rq, cudaMemcpyHostToDevice, s_in) == cudaSuccess;
        okc = okc && cudaMemcpyAsync(dk + t0 * rk, static_cast<const char*>(h_K) + t0 * rk, nt * rk, cudaMemcpyHostToDevice, s_in) == cudaSuccess;
        okc = okc && cudaMemcpyAsync(dv + t0 * rk, static_cast<const char*>(h_V) + t0 * rk, nt * rk, cudaMemcpyHostToDevice, s_in) == cudaSuccess;
        if (h_mask) okc = okc && cudaMemcpyAsync(dm + t0, h_mask + t0, nt, cudaMemcpyHostToDevice, s_in) == cudaSuccess;
        if (parts > 1) okc = okc && cudaEventRecord(ev_in[i], s_in) == cudaSuccess && cudaStreamWaitEvent(st, ev_in[i], 0) == cudaSuccess;
        if (!okc) break;
        stc = seka_attention_fwd(&part, dq + t0 * rq, dk + t0 * rk, dv + t0 * rk, dO + t0 * rq,
                                 h_lse ? reinterpret_cast<float*>(dl) + t0 * shape->n_q_heads : nullptr,
                                 h_mask ? reinterpret_cast<const uint8_t*>(dm) + t0 : nullptr, U,
                                 alpha ? alpha + (size_t)i * seq_per * shape->n_kv_heads * shape->n_experts : nullptr,
                                 gain ? gain + (size_t)i * seq_per : nullptr, head_enable, workspace, workspace_bytes, cuda_stream);
        if (stc != SEKA_OK) break;
        okc = okc && cudaEventRecord(hs.cmp[i], st) == cudaSuccess;
        if (parts > 1) okc = okc && cudaStreamWaitEvent(s_out, hs.cmp[i], 0) == cudaSuccess;
        okc = okc && cudaMemcpyAsync(static_cast<char*>(h_O) + t0 * rq, dO + t0 * rq, nt * rq, cudaMemcpyDeviceToHost, s_out) == cudaSuccess;
        if (h_lse) okc = okc && cudaMemcpyAsync(h_lse + t0 * shape->n_q_heads, reinterpret_cast<float*>(dl) + t0 * shape->n_q_heads,
                                                nt * shape->n_q_heads * 4, cudaMemcpyDeviceToHost, s_out) == cudaSuccess;
    }
    if (parts > 1) {
        // the caller's stream ends behind the last copy out (and behind the copies in, if the loop stopped early)
        if (ev_out && s_out) { cudaEventRecord(ev_out, s_out); cudaStreamWaitEvent(st, ev_out, 0); }
        if (ev_tail && s_in) { cudaEventRecord(ev_tail, s_in); cudaStreamWaitEvent(st, ev_tail, 0); }
        // queued work keeps what it needs: destroying a stream or an event only drops the handle
        for (int i = 0; i < parts; ++i) if (ev_in[i]) cudaEventDestroy(ev_in[i]);
        if (ev_tail) cudaEventDestroy(ev_tail);
        if (ev_out) cudaEventDestroy(ev_out);
        if (s_in) cudaStreamDestroy(s_in);
        if (s_out) cudaStreamDestroy(s_out);
    }
    // a call that stopped early leaves the next one to wait for the whole stream instead
    hs.valid = okc && stc == SEKA_OK;
    hs.staging = staging; hs.parts = parts; hs.tok_per = tok_per;
    if (!hs.valid) cudaStreamSynchronize(st);
    if (stc != SEKA_OK) return stc;
    return okc ? SEKA_OK : SEKA_ERR_CUDA;
}

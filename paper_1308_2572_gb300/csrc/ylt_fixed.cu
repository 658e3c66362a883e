// ylt_fixed.cu -- the skip variant's trial pass over occurrence tables held
// as whole numbers (Section II, Algorithm 1).
//
// An FP32 occurrence loss o = min(max(x - OccR, 0), OccL) > 0 needs x > OccR,
// and an FP32 x >= OccR is a multiple of u = ulp(OccR), OccR too; so their
// FP32 difference is a multiple of u, and o is one whenever OccL is. With o
// bounded by OccL (or by the sum of the layer's ELT limits) every entry of X
// is then a whole number of units below 2^32 for most real covers (OccL up to
// 255 times OccR), stored as that number in the same 4 bytes. The trial pass
// adds entries as 64-bit integers: the sum is exact, takes 1-2 integer
// operations per entry instead of the seven of a compensated FP32 add, and
// reduces across the warp in two 32-bit REDUX steps instead of five rounds of
// compensated shuffles. It is rounded to FP64 once. On c1 (1,000,000 trials x
// 1,000 events, one layer) the forward takes 0.87 ms against 1.25 with the
// compensated pass, on a group of 8 of c4's layers 2.9 against 3.8 ms per
// 1,000,000 trials, on c3 (8 layers, few events with a loss) 1.36 against 2.07.
// Groups with a layer that does not fit (OccR = 0, very wide covers), calls
// under a caller's capture and ids in host or managed memory keep the FP32 table
// and the compensated pass of ylt_skip.cu.
//
// The rest of the mapping is that of ylt_skip.cu: persistent 1024-thread
// CTAs, the bitmap folded into shared memory, a warp per trial streaming its
// ids, the next chunk requested before the current one is processed. A trial
// that starts off a 16-byte boundary is copied from the boundary before it,
// and the ids of its neighbours are masked; a trial whose copies would leave
// the id array (at its very start or end) is read id by id.
//
// What bounds it (ncu, c1): the L1 data path (72% of its wavefronts: 3.2-3.5
// per 32 random bit tests, one per gathered row, one per 32 ids) and the bytes
// in flight (32 KB per SM); issue is 56%.
#include <algorithm>

#include "id_stream.cuh"

namespace art {

namespace {

// Warps per CTA. The 8-layer rows with ragged trials need more than the 64
// registers a thread of 32 warps gets; a spilled value costs L2's latency per
// chunk (the gathers leave L1 no room for it): 16 of c2's layers, 250,000
// trials, 3.05 ms with 32 warps, 1.71 with 24.
template <int LP, bool VEC>
constexpr int kFxWarpsFor = LP == 8 && !VEC ? 24 : 32;
constexpr int kFxIds = 8;     // ids per lane and chunk: 1 KB in flight per warp, 32 KB per SM
// Row id of X: LP (1, 2, 4 or 8) whole numbers in one load, not kept in L1.
template <int LP>
__device__ __forceinline__ void ld_units(const float* x, uint32_t id, uint32_t (&o)[LP]) {
    const float* p = x + (size_t)id * LP;
    if constexpr (LP == 1) {
        asm("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(o[0]) : "l"(p));
    } else if constexpr (LP == 2) {
        asm("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(o[0]), "=r"(o[1]) : "l"(p));
    } else if constexpr (LP == 4) {
        asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
            : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3])
            : "l"(p));
    } else {
        asm("ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]), "=r"(o[4]), "=r"(o[5]), "=r"(o[6]), "=r"(o[7])
            : "l"(p));
    }
}

// The same where the word's bit 0 is set, zeros elsewhere, without a branch
// (narrow rows).
template <int LP>
__device__ __forceinline__ void ld_units_if(const float* x, uint32_t id, uint32_t word, uint32_t (&o)[LP]) {
    static_assert(LP <= 2, "narrow rows");
    const float* p = x + (size_t)id * LP;
    if constexpr (LP == 1) {
        asm("{\n.reg .pred p;\n.reg .b32 a;\nand.b32 a, %2, 1;\nsetp.ne.u32 p, a, 0;\nmov.u32 %0, 0;\n@p ld.global.nc.L1::no_allocate.u32 %0, [%1];\n}"
            : "=r"(o[0])
            : "l"(p), "r"(word));
    } else {
        asm("{\n.reg .pred p;\n.reg .b32 a;\nand.b32 a, %3, 1;\nsetp.ne.u32 p, a, 0;\nmov.u32 %0, 0;\nmov.u32 %1, 0;\n"
            "@p ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];\n}"
            : "=r"(o[0]), "=r"(o[1])
            : "l"(p), "r"(word));
    }
}

// The warp's total of a 64-bit count (valid in every lane). Entries are
// below 2^32, so for trials shorter than 2^20 the lanes' counts stay below
// 2^47: 20 low and 27 high bits, each summed in one 32-bit reduction.
__device__ __forceinline__ unsigned long long warp_total(unsigned long long v, bool is_short) {
    if (is_short) {
        const uint32_t lo = __reduce_add_sync(kFull, (uint32_t)v & 0xfffffu);
        const uint32_t hi = __reduce_add_sync(kFull, (uint32_t)(v >> 20));
        return ((unsigned long long)hi << 20) + lo;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Lane j's share: the warp's total of acc[j] (j < LP).
template <int LP>
__device__ __forceinline__ unsigned long long lane_totals(const unsigned long long (&acc)[LP], int lane, bool is_short) {
    if (is_short) {
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (int j = 0; j < LP; ++j) {
            const uint32_t l = __reduce_add_sync(kFull, (uint32_t)acc[j] & 0xfffffu);
            const uint32_t h = __reduce_add_sync(kFull, (uint32_t)(acc[j] >> 20));
            lo = lane == j ? l : lo;
            hi = lane == j ? h : hi;
        }
        return ((unsigned long long)hi << 20) + lo;
    }
    unsigned long long mine = 0;
#pragma unroll
    for (int j = 0; j < LP; ++j) {
        const unsigned long long v = warp_total(acc[j], false);
        if (lane == j) mine = v;
    }
    return mine;
}

// True when every layer of the group has reached its aggregate cap.
template <int LP>
__device__ __forceinline__ bool capped(const OccGroupArgs& g, const unsigned long long (&acc)[LP], bool is_short) {
    bool all = true;
#pragma unroll
    for (int j = 0; j < LP; ++j) {
        const double v = (double)warp_total(acc[j], is_short) * g.unit[j];
        if (j < g.n_layers) all = all && (v - g.agg_ret[j] >= g.agg_lim[j]);
    }
    return all;
}

// Groups of 1-2 layers: every lane gathers X for its own events whose bit is
// set, 8 loads in flight. PRE entries are summed in 32 bits before the 64-bit
// add (the host picks 4 when four of the largest entry fit).
template <int LP, bool VEC, bool FOLD, int PRE>
__global__ void __launch_bounds__(32 * kFxWarpsFor<LP, VEC>, 1) fixed_narrow_kernel(const OccGroupArgs g, const YetArgs y,
                                                                    const int32_t smem_words, const bool early_exit,
                                                                    double* __restrict__ ylt,
                                                                    uint8_t* __restrict__ branch,
                                                                    int* __restrict__ flags) {
    if (y.gate.closed()) return;
    constexpr int E = kFxIds;
    constexpr int NWARP = kFxWarpsFor<LP, VEC>;
    extern __shared__ __align__(512) uint32_t s_dyn[];
    uint32_t* s_ids = s_dyn + 64;                 // [NWARP][32 * E], after the warps' barriers
    uint32_t* s_bits = s_ids + NWARP * 32 * E;
    const uint32_t C = (uint32_t)y.catalogue, S = (uint32_t)smem_words, none = no_event<FOLD>(C, S);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    IdStream<E> ids;
    ids.init(s_dyn, s_ids, wib, lane);
    stage_bits<FOLD>(s_bits, g.occ_bits, smem_words, (y.catalogue >> 5) + 1);
    __syncthreads();
    // neighbouring CTAs take neighbouring trials, so that few trials still
    // spread over every SM
    const int64_t n_warps = (int64_t)gridDim.x * NWARP;
    int64_t t = (int64_t)wib * gridDim.x + blockIdx.x;
    uint32_t max_id = 0;
    // results of up to 32 trials, lane s holding the s-th: the FP64 steps run
    // once per 32 trials
    unsigned long long res[LP];
    int64_t rt = -1;
    bool rcap = false;
    int slot = 0;
    auto flush = [&]() {
        if (rt >= 0) {
#pragma unroll
            for (int j = 0; j < LP; ++j)
                if (j < g.n_layers) {
                    const double sum = (double)res[j] * g.unit[j];
                    const size_t wi = (size_t)g.layer[j] * (size_t)y.n_trials + (size_t)rt;
                    ylt[wi] = rcap ? g.agg_lim[j] : xl_f64(sum, g.agg_ret[j], g.agg_lim[j]);
                    if (branch) branch[wi] = rcap ? (uint8_t)2 : agg_branch(sum, g.agg_ret[j], g.agg_lim[j]);
                }
        }
        rt = -1;
    };
    Trials<VEC> trials(y, n_warps);
    bool lost = false;  // a wait gave up
    Span<VEC> cur = trials.first(y, t);
    ids.request(cur, 0, lane);
    while (t < y.n_trials && !lost) {
        const int64_t tn = t + n_warps;
        const Span<VEC> nxt = trials.next(y, cur, tn);
        unsigned long long acc[LP];
#pragma unroll
        for (int j = 0; j < LP; ++j) acc[j] = 0;
        const bool is_short = cur.n < (1u << 20);
        bool cap = false;
        if (cur.n == 0) ids.request(nxt, 0, lane);
        for (uint32_t c0 = 0; c0 < cur.n; c0 += 32 * E) {
            uint32_t id[E];
            if (!ids.take(cur, c0, lane, id)) {
                lost = true;
                break;
            }
            clean_ids<E>(cur, c0, lane, C, none, id, max_id);
            // request the next chunk (this trial's, or the next trial's first) now
            const bool last = c0 + 32 * E >= cur.n;
            if (last) ids.request(nxt, 0, lane);
            else ids.request(cur, c0 + 32 * E, lane);
            uint32_t nz[E];
#pragma unroll
            for (int k = 0; k < E; ++k) nz[k] = bit_of<FOLD>(s_bits, g.occ_bits, id[k], S);
            uint32_t o[E][LP];
#pragma unroll
            for (int k = 0; k < E; ++k) {
                ld_units_if<LP>(g.occ, id[k], nz[k], o[k]);
            }
#pragma unroll
            for (int j = 0; j < LP; ++j)
#pragma unroll
                for (int k = 0; k < E; k += PRE) {
                    uint32_t p = o[k][j];
#pragma unroll
                    for (int i = 1; i < PRE; ++i) p += o[k + i][j];
                    acc[j] += p;
                }
            if (early_exit && capped<LP>(g, acc, is_short)) {
                if (!last) {  // the trial's next chunk is on its way: let it come
                    lost = !cur.edge() && !ids.wait();
                    if (!lost) ids.request(nxt, 0, lane);
                }
                cap = true;
                break;
            }
        }
#pragma unroll
        for (int j = 0; j < LP; ++j) {
            const unsigned long long v = warp_total(acc[j], is_short);
            if (lane == slot) res[j] = v;
        }
        if (lane == slot) {
            rt = t;
            rcap = cap;
        }
        if (++slot == 32) {
            flush();
            slot = 0;
        }
        t = tn;
        cur = nxt;
    }
    flush();
    if (lost) ids.give_up(flags, lane);
    if (max_id >= C) atomicOr(flags + kFlagIdRange, 1);
    if (lane == 0 && trials.bad) atomicOr(flags + kFlagBadOffsets, 1);
}

// Groups of 3-8 layers: the ids whose bit is set go to a per-warp ring in
// shared memory; each time 32 are queued every lane takes one row. A lane
// adds the row of the flush before, then requests this flush's, so a gather's
// latency runs beside the next chunk's tests.
template <int LP, bool VEC, bool FOLD>
__global__ void __launch_bounds__(32 * kFxWarpsFor<LP, VEC>, 1) fixed_wide_kernel(const __grid_constant__ OccGroupArgs g, const YetArgs y,
                                                                  const int32_t smem_words, const bool early_exit,
                                                                  double* __restrict__ ylt,
                                                                  uint8_t* __restrict__ branch,
                                                                  int* __restrict__ flags) {
    if (y.gate.closed()) return;
    constexpr int E = kFxIds;
    constexpr int NWARP = kFxWarpsFor<LP, VEC>;
    extern __shared__ __align__(512) uint32_t s_dyn[];
    uint32_t* s_bars = s_dyn + NWARP * kRing;  // after the warps' rings
    uint32_t* s_ids = s_bars + 64;                // [NWARP][32 * E]
    uint32_t* s_bits = s_ids + NWARP * 32 * E;
    const uint32_t C = (uint32_t)y.catalogue, S = (uint32_t)smem_words, none = no_event<FOLD>(C, S);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    IdStream<E> ids;
    ids.init(s_bars, s_ids, wib, lane);
    IdRing ring(s_dyn + wib * kRing);
    stage_bits<FOLD>(s_bits, g.occ_bits, smem_words, (y.catalogue >> 5) + 1);
    __syncthreads();
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t n_warps = (int64_t)gridDim.x * NWARP;
    int64_t t = (int64_t)wib * gridDim.x + blockIdx.x;
    uint32_t max_id = 0;
    Trials<VEC> trials(y, n_warps);
    bool lost = false;  // a wait gave up
    Span<VEC> cur = trials.first(y, t);
    ids.request(cur, 0, lane);
    while (t < y.n_trials && !lost) {
        const int64_t tn = t + n_warps;
        const Span<VEC> nxt = trials.next(y, cur, tn);
        unsigned long long acc[LP];
        uint32_t o[LP];
#pragma unroll
        for (int j = 0; j < LP; ++j) {
            acc[j] = 0;
            o[j] = 0;
        }
        const bool is_short = cur.n < (1u << 20);
        bool cap = false;
        if (cur.n == 0) ids.request(nxt, 0, lane);
        for (uint32_t c0 = 0; c0 < cur.n; c0 += 32 * E) {
            uint32_t id[E];
            if (!ids.take(cur, c0, lane, id)) {
                lost = true;
                break;
            }
            clean_ids<E>(cur, c0, lane, C, none, id, max_id);
            const bool last = c0 + 32 * E >= cur.n;
            if (last) ids.request(nxt, 0, lane);
            else ids.request(cur, c0 + 32 * E, lane);
#pragma unroll
            for (int k = 0; k < E; ++k) {
                ring.push(id[k], bit_of<FOLD>(s_bits, g.occ_bits, id[k], S), lt_mask);
                if ((k & 1) && ring.size() >= 32) {  // at most 31 + 64 queued: two batches
#pragma unroll 1
                    do {
                        const uint32_t mine = ring.take32(lane);
#pragma unroll
                        for (int j = 0; j < LP; ++j) acc[j] += o[j];
                        ld_units<LP>(g.occ, mine, o);
                    } while (ring.size() >= 32);
                    __syncwarp();
                }
            }
            if (early_exit) {
#pragma unroll
                for (int j = 0; j < LP; ++j) {
                    acc[j] += o[j];
                    o[j] = 0;
                }
                if (capped<LP>(g, acc, is_short)) {
                    if (!last) {
                        lost = !cur.edge() && !ids.wait();
                        if (!lost) ids.request(nxt, 0, lane);
                    }
                    ring.head = ring.tail;
                    cap = true;
                    break;
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < LP; ++j) acc[j] += o[j];
        if (lane < ring.size()) {
            ld_units<LP>(g.occ, ring.peek(lane), o);
#pragma unroll
            for (int j = 0; j < LP; ++j) acc[j] += o[j];
        }
        ring.head = ring.tail;
        __syncwarp();
        unsigned long long mine = lane_totals<LP>(acc, lane, is_short);
        if (lane < g.n_layers) {
            const double sum = (double)mine * g.unit[lane], ret = g.agg_ret[lane], lim = g.agg_lim[lane];
            const size_t wi = (size_t)g.layer[lane] * (size_t)y.n_trials + (size_t)t;
            ylt[wi] = cap ? lim : xl_f64(sum, ret, lim);
            if (branch) branch[wi] = cap ? (uint8_t)2 : agg_branch(sum, ret, lim);
        }
        t = tn;
        cur = nxt;
    }
    if (lost) ids.give_up(flags, lane);
    if (max_id >= C) atomicOr(flags + kFlagIdRange, 1);
    if (lane == 0 && trials.bad) atomicOr(flags + kFlagBadOffsets, 1);
}

typedef void (*FixedKernel)(const OccGroupArgs, const YetArgs, const int32_t, const bool, double*, uint8_t*, int*);

template <bool VEC, bool FOLD>
FixedKernel pick_kernel(int lp, bool pre4) {
    switch (lp) {
        case 1: return pre4 ? fixed_narrow_kernel<1, VEC, FOLD, 4> : fixed_narrow_kernel<1, VEC, FOLD, 1>;
        case 2: return pre4 ? fixed_narrow_kernel<2, VEC, FOLD, 4> : fixed_narrow_kernel<2, VEC, FOLD, 1>;
        case 4: return fixed_wide_kernel<4, VEC, FOLD>;
        case 8: return fixed_wide_kernel<8, VEC, FOLD>;
        default: return nullptr;
    }
}

}  // namespace

cudaError_t launch_fixed_group(const OccGroupArgs& g, const YetArgs& y, int lp, int num_sms, bool early, double* ylt,
                               uint8_t* branch, int* flags, cudaStream_t s) {
    int dev = 0, max_optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    // every trial starts and ends on a 16-byte boundary
    const bool vec = !y.off && y.k % 4 == 0 && (reinterpret_cast<uintptr_t>(y.ids) & 15) == 0;
    // the warps' rings, barriers (256 bytes) and id buffers, then the bitmap
    // and its zero word
    const int warps = lp == 8 && !vec ? kFxWarpsFor<8, false> : kFxWarpsFor<8, true>;
    const int fixed_bytes = 256 + 16 + warps * (32 * kFxIds + (lp >= 4 ? (int)kRing : 0)) * 4;
    // Loads of up to 16 bytes hold an L1 line each while they are in flight:
    // with all 227 KB taken as shared memory the 28 KB of L1 left carry 0.5-0.6
    // of them per cycle and SM, with 195 KB (60 KB of L1) 0.8-1.0 (probed; 32-byte
    // loads reach 0.95 with either). So the narrow rows leave that L1 free and
    // fold more of the bitmap (c1 1.009 -> 0.898 ms; the 32-byte rows of c4
    // 1.71 ms with 195 KB, 1.65 with all).
    if (lp <= 4) max_optin = std::min(max_optin, 195 * 1024);
    const int words = (y.catalogue >> 5) + 1;  // bits 0 .. C (C: the sentinel)
    // whole 16-byte groups of words that fit next to the queues
    const int smem_words = std::max(4, std::min((words + 3) & ~3, (max_optin - fixed_bytes) / 4) & ~3);
    const int smem = fixed_bytes + smem_words * 4;
    const bool fold = words <= 2 * smem_words;  // it folds once when at most twice as long
    const bool pre4 = g.sum_fits >= 4;
    const FixedKernel kern = vec ? (fold ? pick_kernel<true, true>(lp, pre4) : pick_kernel<true, false>(lp, pre4))
                                 : (fold ? pick_kernel<false, true>(lp, pre4) : pick_kernel<false, false>(lp, pre4));
    if (!kern) return cudaErrorInvalidValue;
    if ((e = allow_max_shared(kern))) return e;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(num_sms, y.n_trials));
    kern<<<(unsigned)grid, 32 * warps, smem, s>>>(g, y, smem_words, early, ylt, branch, flags);
    return cudaGetLastError();
}

}  // namespace art

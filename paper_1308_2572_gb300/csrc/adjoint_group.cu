// adjoint_group.cu -- the adjoint of the forward pass (the pricing
// sensitivity added around Section II's Algorithm 1) over layer groups (up
// to 8 layers whose ELTs number at most 32 together, ART_LAYOUT_GROUP).
//
// With a_j = [branch_j == mid] and c_j = [branch_j == capped] from the
// forward's aggregate branch codes and g_j the trial's weight:
//   dAggR_j = -g_j a_j,  dAggL_j = g_j c_j,
//   dOccR_j = -g_j a_j #{d : OccR_j < x_dj < OccR_j + OccL_j},
//   dOccL_j =  g_j a_j #{d : x_dj > OccR_j + OccL_j},
//   dm_e    = sum_d [D_e < m_e l_de < D_e + Lim_e] l_de w_de,
//             w_de = sum_{j covering e} g_j a_j [o_dj on its middle branch].
//
// Which occurrence branch each layer takes, and which ELT terms are on their
// middle branch, depend on the event id alone. So each call first evaluates
// them once per catalogue event i (F_e and the layer sums x_ij in FP32, in the
// group's ELT order): M_i, the layers on the middle branch; K_i, the layers on
// the capped branch; and U_i, the ELT columns on their middle branch, plus a
// bitmap of the events with M_i or K_i non-zero (only those contribute). What
// the trial pass needs of such an event is one 32-byte record: M_i spread to
// byte counters, K_i, and up to three (column, layers covering it with a
// middle branch, loss); the few events with more columns are evaluated from
// their table row. Records come from the CSR of the non-zero losses where the
// portfolio holds it (an event with more than four of the group's losses from
// its table row, in the group's order), else from the table rows; the same
// values either way. Groups whose events mostly have more columns, and calls
// with no room for the records, go to adjoint_rows.cu.
//
// The trial pass is shaped like the forward's (ylt_fixed.cu): a persistent CTA
// per SM, the bitmap folded into shared memory, a warp per trial streaming its
// ids by bulk copies, and a per-warp ring of the events whose bit is set,
// evaluated 32 at a time (lane = event), each gather running beside the tests
// that follow it:
//   - the layer counts: per lane, 8-bit counters for the 8 layers packed in
//     two words, added from the record; summed across the warp in 16-bit
//     fields (one REDUX for two layers) at the end of the trial (and every 255
//     batches), then lane j adds layer j's counts times g_j (g_j rounded to
//     FP32, the product exact) to a compensated FP32 pair;
//   - the multipliers: for each (column k, layers S, loss l) of the record the
//     lane adds l * W[S] to its own FP32 partial of column k in shared memory,
//     W[S] = sum_{j in S} g_j a_j from two 16-entry tables of the trial's
//     weights; at the end of the trial, and every kFold batches of a long one,
//     the partials are summed across the warp (recursive halving) and lane k
//     adds column k's total to its compensated FP32 pair. Partials that run on
//     over many trials cost precision: with a fold every 32 batches only,
//     2,000,000 trials of 12 events ended 2-9 times as far from the FP64 sums
//     as with one per trial, which takes 2% of the call (c3).
// A trial with no layer on the middle branch costs only its branch codes. The
// lane values are reduced warp -> CTA -> grid in a fixed order (no atomics:
// deterministic); FP64 arithmetic runs only in that final reduction. Rounding:
// g is rounded to FP32 once per (layer, trial), and the per-event products and
// the W entries are FP32 (a few units in the last place of FP32 per term);
// every sum is compensated or FP64.
//
// What bounds the pass (ncu, c3): issue (58%; 52 instructions per 32 events,
// of which the two POPC of the ring take 4 of 23 cycles) with 20 warps per SM.
// c3, 500,000 trials, records included: 1.15 ms (1.11 without the fold after
// every trial), against 1.95 for the form that gathered 64-byte rows and tested
// 16 columns per queued event (adjoint_rows.cu; where most events have more than
// three columns that one is the faster).
#include <algorithm>
#include <limits>

#include "id_stream.cuh"

namespace art {

namespace {

// Warps per CTA: each holds a column partial per lane (4 * 32 * NP bytes of
// shared memory), which the bitmap competes with; 20 warps leave 96 registers
// a thread, so that nothing is spilled in the chunk loop (24 warps with spills
// take the same time, 16 warps 8% more).
template <int NP>
constexpr int kAgWarpsFor = NP <= 16 ? 20 : 16;
constexpr int kAgIds = 8;     // ids per lane and chunk
constexpr int kFold = 32;     // batches of one trial between the folds of the column partials
constexpr uint32_t kOverflow = 7u;  // more than three columns: evaluated from the table row

// What the trial pass reads of an event.
struct alignas(32) AdjRecord {
    uint32_t mid_lo, mid_hi;  // byte j (mid_hi: 4 + j): layer j on its middle branch
    uint32_t meta;            // columns (5 bits each), their number (bits 15-17), K (bits 20-27)
    uint32_t sets;            // per column, the layers covering it on their middle branch (kOverflow: M)
    float loss[3];            // their losses
    uint32_t u;               // U (kOverflow)
};

__device__ __forceinline__ AdjRecord ld_record(const AdjRecord* p) {
    AdjRecord r;
    asm("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r.mid_lo), "=r"(r.mid_hi), "=r"(r.meta), "=r"(r.sets), "=f"(r.loss[0]), "=f"(r.loss[1]), "=f"(r.loss[2]),
          "=r"(r.u)
        : "l"(p));
    return r;
}

// Bits 0-3 of m to the lowest bits of four bytes.
__device__ __forceinline__ uint32_t spread4(uint32_t m) { return ((m & 15u) * 0x00204081u) & 0x01010101u; }

// The layers covering column k, as the group's membership lists them.
__device__ __forceinline__ uint32_t layers_of(const GroupArgs& g, int k) {
    uint32_t c = 0;
    for (int j = 0; j < g.n_layers; ++j) c |= ((g.member[j] >> k) & 1u) << j;
    return c;
}

// Branches of the layers at the sums x.
template <int LT>
__device__ __forceinline__ void layer_branches(const GroupArgs& g, const float (&x)[LT], uint32_t& mid, uint32_t& cap) {
    mid = cap = 0u;
#pragma unroll
    for (int j = 0; j < LT; ++j)
        if (j < g.n_layers) {
            const float wo = x[j] - g.occ_ret[j];  // the forward's occurrence subtraction
            if (wo > 0.0f && wo < g.occ_lim[j]) mid |= 1u << j;
            if (wo > g.occ_lim[j]) cap |= 1u << j;
        }
}

__device__ __forceinline__ void add_column(AdjRecord& r, uint32_t& n, uint32_t mid, uint32_t cover, int k, float loss) {
    const uint32_t set = mid & cover;
    if (!set) return;
    if (n < 3) {
        r.meta |= (uint32_t)k << (5 * n);
        r.sets |= set << (8 * n);
        if (n == 0) r.loss[0] = loss;
        if (n == 1) r.loss[1] = loss;
        if (n == 2) r.loss[2] = loss;
    }
    ++n;
}

__device__ __forceinline__ void finish_record(AdjRecord& r, uint32_t n, uint32_t mid, uint32_t cap, uint32_t u) {
    r.mid_lo = spread4(mid);
    r.mid_hi = spread4(mid >> 4);
    if (n > 3) {
        r.sets = mid;
        r.u = u;
        n = kOverflow;
    }
    r.meta |= n << 15 | cap << 20;
}

// Event i from its table row; false when it is on no branch that counts.
template <int NP, int LT>
__device__ bool record_from_row(const GroupArgs& g, const uint32_t* s_cover, int64_t i, AdjRecord& r) {
    const float4* row = reinterpret_cast<const float4*>(g.table) + i * (NP / 4);
    float v[NP], f[NP];
#pragma unroll
    for (int q = 0; q < NP / 4; ++q) {
        const float4 w = __ldcs(row + q);
        v[4 * q + 0] = w.x;
        v[4 * q + 1] = w.y;
        v[4 * q + 2] = w.z;
        v[4 * q + 3] = w.w;
    }
    uint32_t u = 0u;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const float wf = __fmaf_rn(g.m[k], v[k], -g.d[k]);
        f[k] = fminf(fmaxf(wf, 0.0f), g.lim[k]);
        if (wf > 0.0f && wf < g.lim[k]) u |= 1u << k;
    }
    float x[LT];
#pragma unroll
    for (int j = 0; j < LT; ++j) {
        x[j] = 0.0f;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            if constexpr (LT == 1) x[j] += f[k];
            else x[j] = __fmaf_rn(g.coef[j][k], f[k], x[j]);
        }
    }
    uint32_t mid, cap, n = 0;
    layer_branches<LT>(g, x, mid, cap);
    if (!(mid | cap)) return false;
#pragma unroll
    for (int k = 0; k < NP; ++k)
        if ((u >> k) & 1u) add_column(r, n, mid, s_cover[k], k, v[k]);
    finish_record(r, n, mid, cap, u);
    return true;
}

// Records and bitmap of a group, one thread per event. ptr NULL: from the
// table rows. col: the group's column of a pool ELT, 255 for none.
template <int NP, int LT>
__global__ void __launch_bounds__(256) adj_records_kernel(const __grid_constant__ GroupArgs g, int32_t catalogue,
                                                          int32_t words, const uint32_t* __restrict__ ptr,
                                                          const SparseEntry* __restrict__ entries,
                                                          const uint8_t* __restrict__ col,
                                                          AdjRecord* __restrict__ records,
                                                          uint32_t* __restrict__ bits) {
    __shared__ uint32_t s_cover[32];
    __shared__ float s_m[32], s_d[32], s_lim[32];
    if (threadIdx.x < 32) {
        s_cover[threadIdx.x] = layers_of(g, threadIdx.x);
        s_m[threadIdx.x] = g.m[threadIdx.x];
        s_d[threadIdx.x] = g.d[threadIdx.x];
        s_lim[threadIdx.x] = g.lim[threadIdx.x];
    }
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool rel = false;
    AdjRecord r{};
    if (i < catalogue) {
        if (!ptr) {
            rel = record_from_row<NP, LT>(g, s_cover, i, r);
        } else {
            // up to four of the group's losses, sorted by column
            int cnt = 0, k4[4] = {0, 0, 0, 0};
            float v4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            const uint32_t q1 = ptr[i + 1];
            for (uint32_t q = ptr[i]; q < q1; ++q) {
                const SparseEntry en = entries[q];
                int k = col[en.elt];
                float v = en.loss;
                if (k == 255) continue;
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s == cnt || (s < cnt && k < k4[s])) {
                        const int tk = k4[s];
                        const float tv = v4[s];
                        k4[s] = k;
                        v4[s] = v;
                        k = tk;
                        v = tv;
                        if (s == cnt) break;
                    }
                ++cnt;
            }
            if (cnt > 4) {
                rel = record_from_row<NP, LT>(g, s_cover, i, r);
            } else if (cnt) {
                // the sums in column order, as over the row (absent columns add exactly 0)
                float x[LT];
#pragma unroll
                for (int j = 0; j < LT; ++j) x[j] = 0.0f;
                uint32_t u = 0;
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s < cnt) {
                        const int k = k4[s];
                        const float w = __fmaf_rn(s_m[k], v4[s], -s_d[k]), lim = s_lim[k];
                        const float f = fminf(fmaxf(w, 0.0f), lim);
                        if (w > 0.0f && w < lim) u |= 1u << k;
                        const uint32_t cover = s_cover[k];
#pragma unroll
                        for (int j = 0; j < LT; ++j) x[j] += (cover >> j) & 1u ? f : 0.0f;
                    }
                uint32_t mid, cap, n = 0;
                layer_branches<LT>(g, x, mid, cap);
                rel = (mid | cap) != 0u;
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    if (s < cnt && ((u >> k4[s]) & 1u)) add_column(r, n, mid, s_cover[k4[s]], k4[s], v4[s]);
                finish_record(r, n, mid, cap, u);
            }
        }
        {  // an event without its bit too: the folded bitmap may gather it
            uint4* dst = reinterpret_cast<uint4*>(records + i);
            dst[0] = make_uint4(r.mid_lo, r.mid_hi, r.meta, r.sets);
            dst[1] = make_uint4(__float_as_uint(r.loss[0]), __float_as_uint(r.loss[1]), __float_as_uint(r.loss[2]), r.u);
        }
    }
    const unsigned m = __ballot_sync(kFull, rel);
    if ((threadIdx.x & 31) == 0 && (i >> 5) < words) bits[i >> 5] = m;
}

// A trial's branch code and weight as lane j holds them for layer j.
struct Weight {
    float g = 0.0f;
    uint8_t code = 0;
};

template <int NP, int LT, bool VEC, bool FOLD>
__global__ void __launch_bounds__(32 * kAgWarpsFor<NP>, 1)
    adjoint_pass_kernel(const __grid_constant__ GroupArgs g, const YetArgs y, const AdjRecord* __restrict__ records,
                        const uint32_t* __restrict__ gbits, const int32_t smem_words, const int64_t warp_step,
                        const int64_t cta_step, const uint8_t* __restrict__ branch, const double* __restrict__ gw,
                        double* __restrict__ partial, int* __restrict__ flags) {
    constexpr int E = kAgIds;
    constexpr int NWARP = kAgWarpsFor<NP>;
    constexpr int W = 4 * LT + NP;   // OccR[LT], OccL[LT], AggR[LT], AggL[LT], then the columns
    extern __shared__ __align__(512) uint32_t s_dyn[];
    uint32_t* s_bars = s_dyn + NWARP * kRing;                            // after the warps' rings
    uint32_t* s_ids = s_bars + 64;                                       // [NWARP][32 * E]
    float* s_part = reinterpret_cast<float*>(s_ids + NWARP * 32 * E);    // [NWARP][NP][32]
    float* s_wt = s_part + NWARP * NP * 32;                              // [NWARP][32]: low and high layers' sums
    uint32_t* s_cover = reinterpret_cast<uint32_t*>(s_wt + NWARP * 32);  // [32]
    uint32_t* s_bits = s_cover + 32;
    const uint32_t C = (uint32_t)y.catalogue, S = (uint32_t)smem_words, none = no_event<FOLD>(C, S);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    IdStream<E> ids;
    ids.init(s_bars, s_ids, wib, lane);
    IdRing ring(s_dyn + wib * kRing);
    float* part = s_part + wib * NP * 32 + lane;  // the lane's partial of column k: part[32 k]
    for (int k = 0; k < NP; ++k) part[32 * k] = 0.0f;
    if (threadIdx.x < 32) s_cover[threadIdx.x] = layers_of(g, threadIdx.x);
    stage_bits<FOLD>(s_bits, gbits, smem_words, (y.catalogue >> 5) + 1);
    __syncthreads();
    float* s_w = s_wt + wib * 32;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t n_warps = (int64_t)gridDim.x * NWARP;

    // lane j < LT keeps layer j's four term sums, lane k < NP column k's sum,
    // each a compensated FP32 pair (FP64 arithmetic per trial would dominate:
    // the FP64 pipe of this part is slow)
    float or_h = 0.0f, or_l = 0.0f, ol_h = 0.0f, ol_l = 0.0f, ar_h = 0.0f, ar_l = 0.0f, al_h = 0.0f, al_l = 0.0f;
    float col_h = 0.0f, col_l = 0.0f;
    int32_t my_layer = -1;
#pragma unroll
    for (int j = 0; j < LT; ++j)
        if (lane == j && j < g.n_layers) my_layer = g.layer[j];
    auto load_weight = [&](int64_t t) {
        Weight w;
        if (my_layer >= 0 && t < y.n_trials) {
            const size_t wi = (size_t)my_layer * (size_t)y.n_trials + (size_t)t;
            w.code = branch[wi];
            w.g = (float)gw[wi];  // the layer's weight, rounded to FP32 once
        }
        return w;
    };
    // the first trial from t on with a middle-branch weight in the group (the
    // aggregate terms' sums take every trial passed); w holds trial t's weight
    auto active_from = [&](int64_t t, Weight& w) {
        while (t < y.n_trials) {
            if (w.code == 1) two_sum_add(ar_h, ar_l, -w.g);
            if (w.code == 2) two_sum_add(al_h, al_l, w.g);
            if (__ballot_sync(kFull, w.code == 1 && w.g != 0.0f)) break;
            t += n_warps;
            w = load_weight(t);
        }
        return t;
    };

    // the lanes' partials summed across the warp by recursive halving: at
    // distance o a lane keeps the half of its columns selected by bit o of its
    // index and adds the partner's copy of that half, so that lane k (and the
    // lanes that share its low bits) ends with column k; 31 shuffles for 32
    // columns, 16 for 16
    auto fold_columns = [&]() {
        constexpr int FC = NP <= 4 ? 4 : NP <= 8 ? 8 : NP <= 16 ? 16 : 32;
        float v[FC];
#pragma unroll
        for (int k = 0; k < FC; ++k) {
            v[k] = 0.0f;
            if (k < NP) {
                v[k] = part[32 * k];
                part[32 * k] = 0.0f;
            }
        }
#pragma unroll
        for (int o = FC / 2; o > 0; o >>= 1) {
            const bool upper = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < o; ++i) {
                const float keep = upper ? v[i + o] : v[i];
                const float send = upper ? v[i] : v[i + o];
                v[i] = keep + __shfl_xor_sync(kFull, send, o);
            }
        }
#pragma unroll
        for (int o = 16; o >= FC; o >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], o);
        if (lane < NP) two_sum_add(col_h, col_l, v[0]);
    };

    int64_t t = (int64_t)wib * warp_step + (int64_t)blockIdx.x * cta_step;
    Weight cw = load_weight(t);
    t = active_from(t, cw);
    Trials<VEC> trials(y, n_warps);
    Span<VEC> cur = trials.first(y, t);
    ids.request(cur, 0, lane);
    bool lost = false;
    uint32_t unused_max = 0;  // ids outside the catalogue were reported by the forward
    int folds = 0;            // batches of the trial since the partials were folded
    while (t < y.n_trials && !lost) {
        const bool mid_l = cw.code == 1 && cw.g != 0.0f;
        const float gt = cw.g;
        Weight nw = load_weight(t + n_warps);
        // the trial's weights: W[s] = sum of g_j a_j over the layers j < 4 in
        // s, W[16 + s] over the layers 4 + j, in increasing j
        {
            const float mine = mid_l ? gt : 0.0f;
            float acc = 0.0f;
#pragma unroll
            for (int b = 0; b < (LT < 4 ? LT : 4); ++b) {
                const float gb = __shfl_sync(kFull, mine, b + (LT > 4 ? (lane & 16) >> 2 : 0));
                acc += (lane >> b) & 1 ? gb : 0.0f;
            }
            s_w[lane] = LT > 4 || lane < 16 ? acc : 0.0f;
            __syncwarp();
        }
        uint32_t mid0 = 0, mid1 = 0, cap0 = 0, cap1 = 0;  // packed layer counters
        auto flush_counts = [&]() {
            // two layers per reduction, in 16-bit fields
            const uint32_t e0 = __reduce_add_sync(kFull, mid0 & 0x00ff00ffu);
            const uint32_t o0 = LT > 1 ? __reduce_add_sync(kFull, (mid0 >> 8) & 0x00ff00ffu) : 0u;
            const uint32_t e1 = LT > 4 ? __reduce_add_sync(kFull, mid1 & 0x00ff00ffu) : 0u;
            const uint32_t o1 = LT > 4 ? __reduce_add_sync(kFull, (mid1 >> 8) & 0x00ff00ffu) : 0u;
            const uint32_t sm = (lane & 4) ? ((lane & 1) ? o1 : e1) : ((lane & 1) ? o0 : e0);
            const uint32_t cm = (lane & 2) ? sm >> 16 : sm & 0xffffu;
            uint32_t cc = 0;
            if (__any_sync(kFull, (cap0 | cap1) != 0u)) {
                const uint32_t f0 = __reduce_add_sync(kFull, cap0 & 0x00ff00ffu);
                const uint32_t p0 = __reduce_add_sync(kFull, (cap0 >> 8) & 0x00ff00ffu);
                const uint32_t f1 = LT > 4 ? __reduce_add_sync(kFull, cap1 & 0x00ff00ffu) : 0u;
                const uint32_t p1 = LT > 4 ? __reduce_add_sync(kFull, (cap1 >> 8) & 0x00ff00ffu) : 0u;
                const uint32_t sc = (lane & 4) ? ((lane & 1) ? p1 : f1) : ((lane & 1) ? p0 : f0);
                cc = (lane & 2) ? sc >> 16 : sc & 0xffffu;
            }
            if (mid_l && lane < LT) {
                // the products are exact (FMA residual; counts < 2^24), the sums compensated
                const float pm = gt * (float)cm, pc = gt * (float)cc;
                two_sum_add(or_h, or_l, -pm);
                or_l -= __fmaf_rn(gt, (float)cm, -pm);
                two_sum_add(ol_h, ol_l, pc);
                ol_l += __fmaf_rn(gt, (float)cc, -pc);
            }
            mid0 = mid1 = cap0 = cap1 = 0;
        };
        auto weight_of = [&](uint32_t set) { return s_w[set & 15u] + s_w[16 + ((set >> 4) & 15u)]; };
        // one batch: the lane's event (all zero: none)
        auto add_record = [&](const AdjRecord& r, uint32_t id) {
            mid0 += r.mid_lo;
            mid1 += r.mid_hi;
            const uint32_t kk = (r.meta >> 20) & 255u, n = (r.meta >> 15) & 7u;
            if (__any_sync(kFull, kk != 0u)) {
                cap0 += spread4(kk);
                cap1 += spread4(kk >> 4);
            }
            if (n != kOverflow) {
                float* c0 = part + 32 * (r.meta & 31u);
                *c0 = __fmaf_rn(r.loss[0], weight_of(r.sets), *c0);  // no column: 0 * W[0]
                if (n > 1) {
                    float* c1 = part + 32 * ((r.meta >> 5) & 31u);
                    *c1 = __fmaf_rn(r.loss[1], weight_of(r.sets >> 8), *c1);
                }
                if (n > 2) {
                    float* c2 = part + 32 * ((r.meta >> 10) & 31u);
                    *c2 = __fmaf_rn(r.loss[2], weight_of(r.sets >> 16), *c2);
                }
            } else {
                const float* row = g.table + (size_t)id * NP;
                for (uint32_t u = r.u; u; u &= u - 1) {
                    const int k = __ffs(u) - 1;
                    part[32 * k] = __fmaf_rn(row[k], weight_of(r.sets & s_cover[k]), part[32 * k]);
                }
            }
        };
        AdjRecord rec{};
        uint32_t rec_id = 0;
        int batches = 0;              // since the counters were cleared (each lane's byte counters < 256)
        int64_t tn = t;
        Span<VEC> nxt;
        auto next_trial = [&]() {
            tn = active_from(t + n_warps, nw);
            nxt = trials.first(y, tn);
            ids.request(nxt, 0, lane);
        };
        if (cur.n == 0) next_trial();
        for (uint32_t c0 = 0; c0 < cur.n; c0 += 32 * E) {
            uint32_t id[E];
            if (!ids.take(cur, c0, lane, id)) {
                lost = true;
                break;
            }
            clean_ids<E>(cur, c0, lane, C, none, id, unused_max);
            if (c0 + 32 * E >= cur.n) next_trial();
            else ids.request(cur, c0 + 32 * E, lane);
            uint32_t nz[E];
#pragma unroll
            for (int k = 0; k < E; ++k) nz[k] = bit_of<FOLD>(s_bits, gbits, id[k], S);
#pragma unroll
            for (int k = 0; k < E; ++k) {
                ring.push(id[k], nz[k], lt_mask);
                if ((k & 1) && ring.size() >= 32) {  // at most 31 + 64 queued: two batches
#pragma unroll 1
                    do {
                        const uint32_t mine = ring.take32(lane);
                        add_record(rec, rec_id);
                        rec = ld_record(records + mine);
                        rec_id = mine;
                        ++folds;
                        if (++batches == 250) {
                            flush_counts();
                            batches = 0;
                        }
                    } while (ring.size() >= 32);
                    __syncwarp();
                    if (folds >= kFold) {
                        fold_columns();
                        folds = 0;
                    }
                }
            }
        }
        __syncwarp();
        add_record(rec, rec_id);
        rec = AdjRecord{};
        if (lane < ring.size()) {
            rec_id = ring.peek(lane);
            rec = ld_record(records + rec_id);
        }
        ring.head = ring.tail;
        add_record(rec, rec_id);
        __syncwarp();
        fold_columns();  // every trial: a partial that ran on over many short trials would lose bits
        folds = 0;
        flush_counts();
        if (lost) break;
        t = tn;
        cur = nxt;
        cw = nw;
    }
    fold_columns();
    if (lost) ids.give_up(flags, lane);
    __syncthreads();
    double* s_red = reinterpret_cast<double*>(s_part);  // [NWARP][W]
    // the lane values in FP64, reduced warp -> CTA in a fixed order
#pragma unroll
    for (int i = 0; i < W; ++i) {
        double v;
        if (i < 4 * LT) {
            const int c = i / LT, j = i % LT;
            const double mine = c == 0   ? (double)or_h + (double)or_l
                                : c == 1 ? (double)ol_h + (double)ol_l
                                : c == 2 ? (double)ar_h + (double)ar_l
                                         : (double)al_h + (double)al_l;
            v = lane == j ? mine : 0.0;
        } else {
            v = lane == i - 4 * LT ? (double)col_h + (double)col_l : 0.0;
        }
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
        if (lane == 0) s_red[wib * W + i] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < W; i += blockDim.x) {
        double s = 0.0;
        for (int wv = 0; wv < NWARP; ++wv) s += s_red[wv * W + i];
        partial[(size_t)blockIdx.x * W + i] = s;
    }
}

// The group's ELT ids (union order) and layer ids, passed by value.
struct GroupIndex {
    int32_t elt[kMaxLayerElts];
    int32_t layer[kMaxGroupLayers];
    int32_t n_elt, n_layers;
};

// Sum the CTA partials of one group (a warp per value, each lane every 32nd
// CTA, then the lanes: a fixed order) and add them into the outputs: each
// layer belongs to one group; an ELT's multiplier gradient sums over the groups
// that hold it, in group order (groups run in order on one stream).
__global__ void __launch_bounds__(1024) group_scatter_kernel(const double* __restrict__ partial, int nblk, int lt,
                                                             int np, const GroupIndex gix,
                                                             double* __restrict__ grad_terms,
                                                             double* __restrict__ grad_mult) {
    const int w = 4 * lt + np, lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < w; i += blockDim.x >> 5) {
        double s = 0.0;
        for (int b = lane; b < nblk; b += 32) s += partial[(size_t)b * w + i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(kFull, s, o);
        if (lane) continue;
        if (i < 4 * lt) {
            const int c = i / lt, j = i % lt;
            if (j < gix.n_layers) grad_terms[(size_t)gix.layer[j] * 4 + c] = s;
        } else {
            const int k = i - 4 * lt;
            if (k < gix.n_elt) grad_mult[gix.elt[k]] += s;
        }
    }
}

struct Scratch {
    AdjRecord* records;  // [C]
    uint32_t* bits;      // zero-padded to whole 16-byte groups, bits 0 .. C
    double* partial;     // [num_sms][4 * 8 + 32]
    uint8_t* col;        // the group's column of each pool ELT (NULL without the CSR)
};

// Records and pass of one group; *nblk CTA partials are left in the scratch.
template <int NP, int LT>
cudaError_t launch_one(const art_portfolio* p, const GroupArgs& g, const YetArgs& y, const uint8_t* branch,
                       const double* gw, const Scratch& sc, int* nblk, cudaStream_t s) {
    const int32_t C = y.catalogue;
    const int32_t words_w = (int32_t)(((int64_t)C + 31) / 32);  // words the record kernel writes
    adj_records_kernel<NP, LT><<<(unsigned)(((int64_t)words_w * 32 + 255) / 256), 256, 0, s>>>(
        g, C, words_w, sc.col ? p->sp_ptr : nullptr, reinterpret_cast<const SparseEntry*>(p->sp_entries), sc.col,
        sc.records, sc.bits);
    cudaError_t e = cudaGetLastError();
    if (e || y.n_trials == 0) return e;
    int dev = 0, max_optin = 0;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    constexpr int NWARP = kAgWarpsFor<NP>;
    const int fixed = 256 + 16 + 4 * (NWARP * (32 * kAgIds + NP * 32 + 32 + (int)kRing) + 32);
    const int words = (C >> 5) + 1;  // bits 0 .. C (C: the sentinel)
    const int smem_words = std::max(4, std::min((words + 3) & ~3, (max_optin - fixed) / 4) & ~3);
    const int smem = fixed + 4 * smem_words;
    const bool fold = words <= 2 * smem_words;
    const bool vec = !y.by_id && !y.off && y.k % 4 == 0 && (reinterpret_cast<uintptr_t>(y.ids) & 15) == 0;
    auto kern = vec ? (fold ? adjoint_pass_kernel<NP, LT, true, true> : adjoint_pass_kernel<NP, LT, true, false>)
                    : (fold ? adjoint_pass_kernel<NP, LT, false, true> : adjoint_pass_kernel<NP, LT, false, false>);
    if ((e = allow_max_shared(kern))) return e;
    // a CTA's warps take neighbouring trials (they share the sectors of the
    // branch codes and weights); few trials are spread over the SMs instead
    const bool many = y.n_trials >= (int64_t)p->num_sms * NWARP;
    const int64_t blocks = many ? p->num_sms : std::max<int64_t>(1, std::min<int64_t>(p->num_sms, y.n_trials));
    kern<<<(unsigned)blocks, 32 * NWARP, smem, s>>>(g, y, sc.records, sc.bits, smem_words, many ? 1 : blocks,
                                                  many ? NWARP : 1, branch, gw, sc.partial, p->d_flags);
    *nblk = (int)blocks;
    return cudaGetLastError();
}

template <int NP>
cudaError_t launch_lt(const art_portfolio* p, const GroupArgs& g, const YetArgs& y, const uint8_t* branch,
                      const double* gw, const Scratch& sc, int* nblk, int* lt, cudaStream_t s) {
    *lt = g.n_layers <= 1 ? 1 : g.n_layers <= 2 ? 2 : g.n_layers <= 4 ? 4 : 8;
    switch (*lt) {
        case 1: return launch_one<NP, 1>(p, g, y, branch, gw, sc, nblk, s);
        case 2: return launch_one<NP, 2>(p, g, y, branch, gw, sc, nblk, s);
        case 4: return launch_one<NP, 4>(p, g, y, branch, gw, sc, nblk, s);
        default: return launch_one<NP, 8>(p, g, y, branch, gw, sc, nblk, s);
    }
}

// Whether a group takes the rows' form: its losses per catalogue event reach
// the number at which both forms took the same time (500,000 catalogue events,
// 30,000 trials of 1,000): 1.3 for one layer of 8 or 16 ELTs, 1.9 of 24, 2.6 of
// 32; 2.5 for eight layers over 16. Up to four ELTs never do.
bool dense(const art_portfolio* p, size_t gi) {
    const int np = p->group_np[gi];
    const float by_layers = 1.3f + 0.17f * (float)(p->groups[gi].n_layers - 1);
    return np > 4 && p->group_losses[gi] > std::max(by_layers, np >= 32 ? 2.6f : np >= 24 ? 1.9f : 0.0f);
}

}  // namespace

cudaError_t launch_adjoint_groups(art_portfolio* p, const YetArgs& yet, const uint8_t* branch, const double* g,
                                  double* grad_terms, double* grad_mult, cudaStream_t s) {
    YetArgs y = yet;
    y.by_id = !ids_on_device(y);
    std::vector<bool> rows(p->groups.size());
    bool any_records = false;
    for (size_t gi = 0; gi < rows.size(); ++gi) {
        rows[gi] = dense(p, gi);
        any_records = any_records || !rows[gi];
    }
    const size_t C = (size_t)p->catalogue;
    const size_t bit_bytes = (16 * ((C / 32 + 1 + 3) / 4) + 255) & ~(size_t)255;
    const size_t part_bytes = sizeof(double) * (size_t)p->num_sms * (4 * kMaxGroupLayers + kMaxLayerElts);
    const size_t mask_bytes = (sizeof(uint2) * (C + 1) + 255) & ~(size_t)255;
    size_t event_bytes = any_records ? std::max(mask_bytes, (sizeof(AdjRecord) * C + 255) & ~(size_t)255) : mask_bytes;
    char* w = nullptr;
    cudaError_t err = scratch_alloc((void**)&w, event_bytes + bit_bytes + part_bytes, s);
    if (err == cudaErrorMemoryAllocation && any_records) {
        cudaGetLastError();  // no room for 32 bytes per catalogue event: the rows' form takes 8
        rows.assign(rows.size(), true);
        event_bytes = mask_bytes;
        err = scratch_alloc((void**)&w, event_bytes + bit_bytes + part_bytes, s);
    }
    if (err) return err;
    Scratch sc{reinterpret_cast<AdjRecord*>(w), reinterpret_cast<uint32_t*>(w + event_bytes),
               reinterpret_cast<double*>(w + event_bytes + bit_bytes), nullptr};
    do {
        if ((err = cudaMemsetAsync(grad_terms, 0, sizeof(double) * 4 * p->n_layers, s))) break;
        if ((err = cudaMemsetAsync(grad_mult, 0, sizeof(double) * p->n_elt, s))) break;
        if (y.n_trials == 0) break;
        // the bitmap's padding words stay zero for every group
        if ((err = cudaMemsetAsync(sc.bits, 0, bit_bytes, s))) break;
        for (size_t gi = 0; gi < p->groups.size(); ++gi) {
            const GroupArgs& ga = p->groups[gi];
            GroupIndex gix{};
            gix.n_elt = (int32_t)p->group_elts[gi].size();
            gix.n_layers = (int32_t)p->group_layers[gi].size();
            for (int k = 0; k < gix.n_elt; ++k) gix.elt[k] = p->group_elts[gi][k];
            for (int j = 0; j < gix.n_layers; ++j) gix.layer[j] = p->group_layers[gi][j];
            sc.col = p->d_group_col ? p->d_group_col + gi * (size_t)p->pool_np : nullptr;
            int nblk = 0, lt = 0;
            if (rows[gi]) {
                err = launch_adjoint_rows(p, gi, y, branch, g, reinterpret_cast<uint2*>(w), sc.bits, sc.partial, &nblk,
                                          &lt, s);
            } else {
                switch (p->group_np[gi]) {
                    case 4: err = launch_lt<4>(p, ga, y, branch, g, sc, &nblk, &lt, s); break;
                    case 8: err = launch_lt<8>(p, ga, y, branch, g, sc, &nblk, &lt, s); break;
                    case 16: err = launch_lt<16>(p, ga, y, branch, g, sc, &nblk, &lt, s); break;
                    case 24: err = launch_lt<24>(p, ga, y, branch, g, sc, &nblk, &lt, s); break;
                    case 32: err = launch_lt<32>(p, ga, y, branch, g, sc, &nblk, &lt, s); break;
                    default: err = cudaErrorInvalidValue;
                }
            }
            if (err) break;
            group_scatter_kernel<<<1, 1024, 0, s>>>(sc.partial, nblk, lt, p->group_np[gi], gix, grad_terms, grad_mult);
            if ((err = cudaGetLastError())) break;
        }
    } while (0);
    const cudaError_t e2 = cudaFreeAsync(w, s);
    return err ? err : e2;
}

}  // namespace art

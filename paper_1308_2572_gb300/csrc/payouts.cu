// payouts.cu -- Algorithm 1's running form on the GPU for one layer: the
// cumulative aggregate C_d over a trial's events in trial order, the
// aggregate terms on every C_d, the per-event difference p_d = A(C_d) -
// A(C_{d-1}) (C_0 = 0: nothing is paid before the first event), and the
// position of the event that exhausts the aggregate limit (Section II: the
// aggregate terms apply to the cumulative sum, so the result depends on the
// sequence of prior events).
//
// Mapping: one warp per trial over the layer's event-major table; 32 events
// per step in trial order, lane l taking event d0 + l. Per event the lane
// forms x_d and o_d exactly as the forward kernels do (FP32, ELT order), then
// the warp scans o_d in FP64 (an inclusive shuffle scan) on top of the carry
// from the previous step, applies the aggregate terms to each C_d in FP64 and
// takes the difference with the previous event's value (the previous lane's,
// or the carried one). It evaluates the layer per occurrence in FP64 and
// serves short YETs and layers whose losses are not whole numbers.
//
// Otherwise (payouts_fixed_kernel) the layer's occurrence losses are evaluated
// once per catalogue event into a table of whole numbers (see ylt_fixed.cu)
// with its bitmap, and the pass streams the ids as the skip variant's does.
// C_d is then an exact 64-bit integer: a lane adds its four consecutive events,
// the warp scans the lanes' totals, and the branch of A(C_d) is a comparison
// of integers (the host finds, once per call, the smallest C whose FP64 value
// passes the retention and the smallest that reaches the limit). Between the
// two the payout is the event's own occurrence loss, exactly; below and above
// it is 0; only the events that cross one of them take FP64 arithmetic, at
// most two per trial. What bounds it: HBM (4 bytes of ids read, 8 of payouts
// written per event); 100,000 trials x 1,000 events of a 16-ELT layer take
// 0.35 ms against 2.40 with a warp scan in FP64 over 64-byte rows.
#include <algorithm>
#include <cmath>
#include <limits>

#include "id_stream.cuh"

namespace art {
namespace {

template <int NP>
__global__ void __launch_bounds__(256) payouts_kernel(const LayerArgs la, const YetArgs y,
                                                      double* __restrict__ payouts, int32_t* __restrict__ exhaust,
                                                      double* __restrict__ ylt, int* __restrict__ flags) {
    if (y.gate.closed()) return;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= y.n_trials) return;  // whole warp
    int64_t b, e;
    bool bad_off;
    trial_range(y, t, b, e, bad_off);
    const float4* __restrict__ tab = reinterpret_cast<const float4*>(la.table);
    double carry_c = 0.0, carry_a = 0.0;  // C and A(C) after the previous step
    int32_t first_cap = -1;
    bool bad_id = false;
    for (int64_t d0 = b; d0 < e; d0 += 32) {
        const int64_t d = d0 + lane;
        const bool live = d < e;
        const int32_t id = live ? ld_stream(y.ids + d) : 0;
        const bool ok = live && (unsigned)id < (unsigned)y.catalogue;
        if (live && !ok) bad_id = true;
        float x = 0.0f;
        if (ok) {
            const float4* row = tab + (size_t)id * (NP / 4);
#pragma unroll
            for (int q = 0; q < NP / 4; ++q) {
                const float4 r = __ldg(row + q);
                x += fin_f32(r.x, la.m[4 * q + 0], la.d[4 * q + 0], la.lim[4 * q + 0]);
                x += fin_f32(r.y, la.m[4 * q + 1], la.d[4 * q + 1], la.lim[4 * q + 1]);
                x += fin_f32(r.z, la.m[4 * q + 2], la.d[4 * q + 2], la.lim[4 * q + 2]);
                x += fin_f32(r.w, la.m[4 * q + 3], la.d[4 * q + 3], la.lim[4 * q + 3]);
            }
        }
        const double o = live ? (double)xl_f32(x, la.occ_ret, la.occ_lim) : 0.0;
        // inclusive scan of o over the lanes, in trial order
        double c = o;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const double v = __shfl_up_sync(FULL, c, k);
            if (lane >= k) c += v;
        }
        c += carry_c;
        const double a = xl_f64(c, la.agg_ret, la.agg_lim);
        double a_prev = __shfl_up_sync(FULL, a, 1);
        if (lane == 0) a_prev = carry_a;
        if (live && payouts) payouts[d] = a - a_prev;
        // the aggregate limit is exhausted at the first event whose C_d - AggR reaches AggL
        const unsigned capped = __ballot_sync(FULL, live && (c - la.agg_ret >= la.agg_lim));
        if (first_cap < 0 && capped) first_cap = (int32_t)(d0 - b) + __ffs(capped) - 1;
        carry_c = __shfl_sync(FULL, c, 31);
        carry_a = __shfl_sync(FULL, a, 31);
    }
    if (bad_id) atomicOr(flags + kFlagIdRange, 1);
    if (lane == 0) {
        if (bad_off) atomicOr(flags + kFlagBadOffsets, 1);
        if (exhaust) exhaust[t] = first_cap;
        if (ylt) ylt[t] = carry_a;  // A(C_K): the telescoped sum of the payouts
    }
}

template <int NP>
cudaError_t launch(const LayerArgs& la, const YetArgs& y, double* payouts, int32_t* exhaust, double* ylt, int* flags,
                   cudaStream_t s) {
    const int64_t blocks = (y.n_trials + 7) / 8;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    payouts_kernel<NP><<<(unsigned)blocks, 256, 0, s>>>(la, y, payouts, exhaust, ylt, flags);
    return cudaGetLastError();
}

constexpr int kPayThreads = 1024;
constexpr int kPayWarps = kPayThreads / 32;
constexpr int kPayIds = 8;  // ids per lane and chunk

// One layer as the whole-number pass reads it.
struct PayArgs {
    const uint32_t* x;        // [C] occurrence losses in units
    const uint32_t* bits;     // bit i set when x[i] > 0, zero-padded to whole 16-byte groups
    double unit, agg_ret, agg_lim;
    float unit_f;
    unsigned long long pass;  // smallest C with XL(C) > 0
    unsigned long long full;  // smallest C with C - AggR >= AggL (all ones: none)
};

// The layer's table: thread i evaluates event i (steps 2-3, FP32, the layer's
// ELT order) as the forward does.
template <int NP>
__global__ void __launch_bounds__(256) payouts_table_kernel(const LayerArgs la, int32_t catalogue, float scale,
                                                            int32_t words, uint32_t* __restrict__ x,
                                                            uint32_t* __restrict__ bits, const EventGate gate) {
    if (gate.closed()) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t u = 0;
    if (i < catalogue) {
        const float4* row = reinterpret_cast<const float4*>(la.table) + i * (NP / 4);
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < NP / 4; ++q) {
            const float4 r = __ldcs(row + q);
            s += fin_f32(r.x, la.m[4 * q + 0], la.d[4 * q + 0], la.lim[4 * q + 0]);
            s += fin_f32(r.y, la.m[4 * q + 1], la.d[4 * q + 1], la.lim[4 * q + 1]);
            s += fin_f32(r.z, la.m[4 * q + 2], la.d[4 * q + 2], la.lim[4 * q + 2]);
            s += fin_f32(r.w, la.m[4 * q + 3], la.d[4 * q + 3], la.lim[4 * q + 3]);
        }
        u = __float2uint_rz(xl_f32(s, la.occ_ret, la.occ_lim) * scale);
        x[i] = u;
    }
    const unsigned m = __ballot_sync(kFull, u != 0);
    if ((threadIdx.x & 31) == 0 && (i >> 5) < words) bits[i >> 5] = m;  // the padding too
}

// XL of C = c units (the product is exact, so the FMA rounds as the
// subtraction alone).
__device__ __forceinline__ double agg_of(const PayArgs& a, unsigned long long c) {
    return fmin(fmax(fma((double)c, a.unit, -a.agg_ret), 0.0), a.agg_lim);
}

// u units as FP64, exactly: an FP32 value (the units hold at most 24
// significant bits) widened by its bit pattern, without the FP64 pipe.
__device__ __forceinline__ double units_f64(uint32_t u, float unit) {
    const uint32_t f = __float_as_uint((float)u * unit);
    return u ? __hiloint2double((int)((f >> 3) + 0x38000000u), (int)(f << 29)) : 0.0;
}

// Streaming stores: the payouts must not push the table out of L2.
__device__ __forceinline__ void st_payouts4(double* p, const double (&v)[4]) {
    asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                 : "memory");
}

// pay_vec: the payouts of a 16-byte group of ids start on a 32-byte boundary.
template <bool VEC, bool FOLD>
__global__ void __launch_bounds__(kPayThreads, 1) payouts_fixed_kernel(const PayArgs a, const YetArgs y,
                                                                      const int32_t smem_words, const bool pay_vec,
                                                                      double* __restrict__ payouts,
                                                                      int32_t* __restrict__ exhaust,
                                                                      double* __restrict__ ylt,
                                                                      int* __restrict__ flags) {
    if (y.gate.closed()) return;
    constexpr int E = kPayIds;
    extern __shared__ __align__(128) uint32_t s_dyn[];
    uint32_t* s_ids = s_dyn + 64;  // [kPayWarps][32 * E], after the warps' barriers
    uint32_t* s_bits = s_ids + kPayWarps * 32 * E;
    const uint32_t C = (uint32_t)y.catalogue, S = (uint32_t)smem_words, none = no_event<FOLD>(C, S);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    IdStream<E> ids;
    ids.init(s_dyn, s_ids, wib, lane);
    stage_bits<FOLD>(s_bits, a.bits, smem_words, (y.catalogue >> 5) + 1);
    __syncthreads();
    const int64_t n_warps = (int64_t)gridDim.x * kPayWarps;
    int64_t t = (int64_t)wib * gridDim.x + blockIdx.x;
    uint32_t max_id = 0;
    bool lost = false;
    // the trial losses of up to 32 trials, lane s holding the s-th: their FP64
    // steps run once per 32 trials
    unsigned long long held = 0;
    int64_t held_t = -1;
    int slot = 0;
    auto flush = [&]() {
        if (ylt && held_t >= 0) ylt[held_t] = agg_of(a, held);  // A(C_K): the telescoped sum of the payouts
        held_t = -1;
    };
    Trials<VEC> trials(y, n_warps);
    Span<VEC> cur = trials.first(y, t);
    ids.request(cur, 0, lane);
    while (t < y.n_trials && !lost) {
        const int64_t tn = t + n_warps;
        const Span<VEC> nxt = trials.next(y, cur, tn);
        unsigned long long carry = 0;  // C before the step, the same in every lane
        int32_t first_full = -1;
        double* pay = payouts ? payouts + (cur.p - y.ids) : nullptr;  // the payout of position 0
        if (cur.n == 0) ids.request(nxt, 0, lane);
        for (uint32_t c0 = 0; c0 < cur.n; c0 += 32 * E) {
            uint32_t id[E];
            if (!ids.take(cur, c0, lane, id)) {
                lost = true;
                break;
            }
            clean_ids<E>(cur, c0, lane, C, none, id, max_id);
            if (c0 + 32 * E >= cur.n) ids.request(nxt, 0, lane);
            else ids.request(cur, c0 + 32 * E, lane);
            uint32_t o[E];
#pragma unroll
            for (int k = 0; k < E; ++k) {
                // bit 0 clear: 0, without a branch
                asm("{\n.reg .pred p;\n.reg .b32 w;\nand.b32 w, %2, 1;\nsetp.ne.u32 p, w, 0;\nmov.u32 %0, 0;\n"
                    "@p ld.global.nc.L1::no_allocate.u32 %0, [%1];\n}"
                    : "=r"(o[k])
                    : "l"(a.x + id[k]), "r"(bit_of<FOLD>(s_bits, a.bits, id[k], S)));
            }
#pragma unroll
            for (int h = 0; h < E / 4; ++h) {
                const uint32_t d = c0 + 128u * h + 4u * lane;  // the lane's four consecutive positions
                if (c0 + 128u * h >= cur.n) break;
                const uint32_t* oh = o + 4 * h;
                const unsigned long long total = (unsigned long long)oh[0] + oh[1] + oh[2] + oh[3];
                unsigned long long run = total;
#pragma unroll
                for (int k = 1; k < 32; k <<= 1) {
                    const unsigned long long v = __shfl_up_sync(kFull, run, k);
                    if (lane >= k) run += v;
                }
                const unsigned long long after = carry + __shfl_sync(kFull, run, 31);
                double v[4] = {0.0, 0.0, 0.0, 0.0};
                if (after >= a.pass && carry < a.full) {  // the same for the whole warp
                    if (carry >= a.pass && after < a.full) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[i] = units_f64(oh[i], a.unit_f);
                    } else {  // some event crosses the retention or the limit
                        unsigned long long c = carry + run - total;
                        int32_t at = -1;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const unsigned long long before = c;
                            c += oh[i];
                            const bool crosses = c >= a.pass && before < a.full && (before < a.pass || c >= a.full);
                            if (before >= a.pass && c < a.full) v[i] = units_f64(oh[i], a.unit_f);
                            // one evaluation, and only where some lane's event crosses: an FP64
                            // instruction takes a warp 16 cycles of its SM. From the retention the
                            // payout is XL(C); to the limit it is what XL(C before) leaves of it.
                            if (__any_sync(kFull, crosses)) {
                                const double x = agg_of(a, before < a.pass ? c : before);
                                if (crosses) v[i] = before < a.pass ? x : a.agg_lim - x;
                            }
                            if (before < a.full && c >= a.full) at = (int32_t)(d + i - cur.head());
                        }
                        const unsigned m = __ballot_sync(kFull, at >= 0);
                        if (m) first_full = __shfl_sync(kFull, at, __ffs(m) - 1);
                    }
                }
                carry = after;
                if (pay) {
                    if (pay_vec && d >= cur.head() && d + 4 <= cur.n) {
                        st_payouts4(pay + d, v);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (d + i >= cur.head() && d + i < cur.n) __stcs(pay + d + i, v[i]);
                    }
                }
            }
        }
        if (lost) break;
        if (exhaust && lane == 0) exhaust[t] = first_full;
        if (lane == slot) {
            held = carry;
            held_t = t;
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

// The smallest N for which f(N * unit) holds (f never turns false again), or
// all ones when it does not below 2^63.
template <class F>
unsigned long long first_units(double unit, F f) {
    unsigned long long lo = 0, hi = 1ULL << 63;
    if (!f((double)hi * unit)) return ~0ULL;
    while (lo < hi) {
        const unsigned long long mid = lo + (hi - lo) / 2;
        if (f((double)mid * unit)) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// The whole-number form of the call, where it is the faster one. Its table
// costs one read of the layer's rows; its pass then takes 0.55 ns per trial and
// 256 ids (and 1.2 ps per event), the other form 0.79 ns per trial and 32 ids
// (2,000,000 events of 16 ELTs: 36 us for the table; 2,000 trials of 300 events
// 26 us without it and 37 with it, 200,000 trials of 50 316 and 175). A CSR whose
// length alone decides is launched in both forms, one of which leaves on the
// device: `rest` then holds the other's gate. done: the other is not needed.
cudaError_t launch_whole(art_portfolio* p, const LayerArgs& la, int np, double lims, YetArgs y, double* payouts,
                         int32_t* exhaust, double* ylt, cudaStream_t s, bool* done, YetArgs* rest) {
    *done = false;
    int e2;
    double top;
    if (!ids_on_device(y) || !whole_losses(la.occ_ret, la.occ_lim, lims, &e2, &top)) return cudaSuccess;
    // the table would put allocation nodes into a caller's graph, which then
    // could neither be a child graph nor run twice at a time
    if (captured_by_caller(p, s)) return cudaSuccess;
    const double n = (double)y.n_trials, table_us = (double)p->catalogue * np * 4.0 / 3.5e6;
    // a warp takes a trial; below about 2,000 of them it waits for its own loads
    const double alone = std::max(1.0, 2000.0 / n);
    auto steps = [&](double E, double ids) { return alone * std::max(n, E / ids + 0.5 * n); };
    int64_t split = 0;
    const ByEvents form = by_events(
        y, -1, [&](double E) { return 5.0 + 0.79e-3 * steps(E, 32.0); },
        [&](double E) { return 5.0 + table_us + 1e-3 * (0.1 * n + 0.45 * steps(E, 256.0)) + 1.2e-6 * E; }, &split);
    if (form == ByEvents::few) return cudaSuccess;
    PayArgs a;
    a.unit = std::ldexp(1.0, e2);
    a.unit_f = (float)a.unit;
    a.agg_ret = la.agg_ret;
    a.agg_lim = la.agg_lim;
    a.pass = first_units(a.unit, [&](double c) { return c - la.agg_ret > 0.0; });
    a.full = first_units(a.unit, [&](double c) { return c - la.agg_ret >= la.agg_lim; });
    const int32_t C = p->catalogue;
    const int words = (C >> 5) + 1;
    const size_t padded = (size_t)(words + 3) & ~(size_t)3;  // whole 16-byte groups
    const size_t xb = (sizeof(uint32_t) * (size_t)C + 255) & ~(size_t)255;
    int dev = 0, max_optin = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    max_optin = std::min(max_optin, 195 * 1024);  // L1 for the gathers in flight, as in ylt_fixed.cu
    const int fixed_bytes = 256 + 16 + kPayWarps * 32 * kPayIds * 4;
    const int smem_words = std::max(4, std::min((int)padded, (max_optin - fixed_bytes) / 4) & ~3);
    const int smem = fixed_bytes + smem_words * 4;
    const bool fold = words <= 2 * smem_words;
    const bool vec = !y.off && y.k % 4 == 0 && (reinterpret_cast<uintptr_t>(y.ids) & 15) == 0;
    const bool pay_vec =
        ((reinterpret_cast<uintptr_t>(payouts) >> 3) - (reinterpret_cast<uintptr_t>(y.ids) >> 2)) % 4 == 0;
    auto kern = vec ? (fold ? payouts_fixed_kernel<true, true> : payouts_fixed_kernel<true, false>)
                    : (fold ? payouts_fixed_kernel<false, true> : payouts_fixed_kernel<false, false>);
    if ((e = allow_max_shared(kern))) return e;
    char* w = nullptr;
    if ((e = scratch_alloc((void**)&w, xb + sizeof(uint32_t) * padded, s))) {
        if (e != cudaErrorMemoryAllocation) return e;
        cudaGetLastError();  // no room for the table: the other form needs none
        return cudaSuccess;
    }
    if (form == ByEvents::device) {
        rest->gate = EventGate{y.off, y.n_trials, std::numeric_limits<int64_t>::min(), split};
        y.gate = EventGate{y.off, y.n_trials, split, std::numeric_limits<int64_t>::max()};
    }
    uint32_t* x = reinterpret_cast<uint32_t*>(w);
    uint32_t* bits = reinterpret_cast<uint32_t*>(w + xb);
    a.x = x;
    a.bits = bits;
    const float scale = (float)std::ldexp(1.0, -e2);
    const unsigned blocks = (unsigned)((padded * 32 + 255) / 256);
    switch (np) {
        case 4: payouts_table_kernel<4><<<blocks, 256, 0, s>>>(la, C, scale, (int32_t)padded, x, bits, y.gate); break;
        case 8: payouts_table_kernel<8><<<blocks, 256, 0, s>>>(la, C, scale, (int32_t)padded, x, bits, y.gate); break;
        case 16: payouts_table_kernel<16><<<blocks, 256, 0, s>>>(la, C, scale, (int32_t)padded, x, bits, y.gate); break;
        case 24: payouts_table_kernel<24><<<blocks, 256, 0, s>>>(la, C, scale, (int32_t)padded, x, bits, y.gate); break;
        default: payouts_table_kernel<32><<<blocks, 256, 0, s>>>(la, C, scale, (int32_t)padded, x, bits, y.gate); break;
    }
    if (!(e = cudaGetLastError())) {
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(p->num_sms, y.n_trials));
        kern<<<(unsigned)grid, kPayThreads, smem, s>>>(a, y, smem_words, pay_vec, payouts, exhaust, ylt, p->d_flags);
        e = cudaGetLastError();
    }
    const cudaError_t e3 = cudaFreeAsync(w, s);
    *done = form == ByEvents::many;
    return e ? e : e3;
}

}  // namespace

cudaError_t launch_payouts(art_portfolio* p, int32_t j, const YetArgs& yet, double* payouts, int32_t* exhaust,
                           double* ylt, cudaStream_t s) {
    if (yet.n_trials == 0) return cudaSuccess;
    YetArgs y = yet;
    LayerArgs la;
    la.table = p->layer_tab[j];
    const int32_t b = p->loff[j], n = p->loff[j + 1] - b;
    for (int k = 0; k < kMaxLayerElts; ++k) {
        const bool real = k < n;
        const int32_t e = real ? p->lids[b + k] : 0;
        la.m[k] = real ? p->mult[e] : 1.0f;
        la.d[k] = real ? p->ded[e] : 0.0f;
        la.lim[k] = real ? p->lim[e] : std::numeric_limits<float>::infinity();
    }
    la.occ_ret = p->occ_ret[j];
    la.occ_lim = p->occ_lim[j];
    la.agg_ret = p->agg_ret[j];
    la.agg_lim = p->agg_lim[j];
    la.layer = j;
    double lims = 0.0;
    for (int k = 0; k < n; ++k) lims += la.lim[k];
    bool done = false;
    const cudaError_t err = launch_whole(p, la, p->layer_np[j], lims, yet, payouts, exhaust, ylt, s, &done, &y);
    if (err || done) return err;
    switch (p->layer_np[j]) {
        case 4: return launch<4>(la, y, payouts, exhaust, ylt, p->d_flags, s);
        case 8: return launch<8>(la, y, payouts, exhaust, ylt, p->d_flags, s);
        case 16: return launch<16>(la, y, payouts, exhaust, ylt, p->d_flags, s);
        case 24: return launch<24>(la, y, payouts, exhaust, ylt, p->d_flags, s);
        case 32: return launch<32>(la, y, payouts, exhaust, ylt, p->d_flags, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace art

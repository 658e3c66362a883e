// metrics_list.cu -- expected loss, PML and TVaR in one read of the YLT
// (Section I's risk metrics; the reading, the exact sums and the general path
// are those of metrics.cu, and the results are the same).
//
// PML_p and TVaR_p need only a layer's k largest losses, k = ceil((1 - p) n).
// Where k is a small part of n, three launches do:
//   1. sample (one CTA per layer): the r-th largest of 4,096 losses at hashed
//      positions is a threshold T below which the k-th largest lies with
//      overwhelming probability (r is about six standard deviations past the
//      sample's share of k); the sample's largest loss, if it repeats, is the
//      tie key (the aggregate cap, the value that repeats most).
//   2. pass (the only read of the YLT): each layer's exact sum, the number of
//      losses equal to the tie key, and a list of the other losses >= T that
//      are not 0. Where the r-th largest of the sample repeats too (a layer
//      whose events mostly pay their full limit: whole multiples of it), that
//      value is a second tie key; listed, it took the list's room, and the
//      finish read the row (1,000,000 trials at three probabilities: 5.3 ms).
//   3. finish (one CTA per layer): the k-th largest of list and ties by a
//      radix select in shared memory, the exact sum of the losses above it,
//      mean, PML and TVaR. If the list holds fewer than k losses and T > 0, or
//      overflowed, or some loss is subnormal beside T > 0, the CTA takes the row
//      instead (for the sum alone where a loss lay far above the sample's
//      largest): slower, the same results.
// A short YLT (metrics_small) skips 1 and 2: its rows fit shared memory.
//
// What bounds it: HBM (8 bytes per loss, once); the general path's two full
// reads and six list passes took 1.04 ms on 128 layers x 1,000,000 trials at
// three probabilities, this takes 0.27 ms (floor 0.15: the pass issues 37
// instructions per 32 losses and runs at 0.73 of the copy rate), and one layer's
// metrics 36 us against 90 (eight dependent launches).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "art_internal.cuh"

namespace art {

namespace {

typedef unsigned long long u64;

constexpr unsigned kAll = 0xffffffffu;
constexpr int kSample = 4096;
constexpr int kFinishThreads = 1024;
constexpr int kSmall = 26624;        // keys the finish CTA holds in shared memory (208 KB)
constexpr int kPassThreads = 256;
constexpr int kPassUnroll = 8;       // values per thread whose loads are in flight together
constexpr u64 kNoTie = ~0ULL;
constexpr int kBins = 2048;          // 11-bit digits
constexpr int kDirect = 128;         // candidates that are ranked by comparison
constexpr int kTies = 2;             // keys per layer that are counted, not listed
constexpr unsigned kAtom = 32;       // sample keys in one of 2^22 bins that make a repeating key likely
// why a layer's row is read again
constexpr unsigned kSumOut = 1;      // a loss above the short sum's range: the sum only
constexpr unsigned kUnlisted = 2;    // a loss that no list can hold (or no reference for any): everything

struct Ranks {
    long long k[kMaxProbs];
    int n_p;
};

// Per-layer state, written by the sample.
struct ListState {
    u64 threshold;   // T (its low word is 0)
    u64 tie[kTies];  // the tie keys (kNoTie: none)
    u64 sum[2];      // fixed-point sum of the row (unit by ref)
    u64 n_tie[kTies];
    unsigned int n_list;
    int ref;         // reference exponent of the pass's sum; 0: the list holds every loss, sum that
    unsigned int again;   // kSumOut, kUnlisted
    unsigned int pad;
};

__device__ __forceinline__ u64 key_at(const u64* p, int64_t i) { return __ldcs(p + i) & 0x7fffffffffffffffULL; }

// ---- block-wide helpers (kFinishThreads threads; scratch of 33 words)

__device__ __forceinline__ u64 block_max(u64 v, u64* sh) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kAll, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = sh[threadIdx.x & 31];
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kAll, v, o));
    return v;
}

__device__ __forceinline__ u64 block_sum(u64 v, u64* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = sh[threadIdx.x & 31];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
    return v;
}

__device__ __forceinline__ Fix block_fix(Fix f, u64* sh) {
    f = fix_warp_sum(f);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        sh[2 * (threadIdx.x >> 5)] = f.lo;
        sh[2 * (threadIdx.x >> 5) + 1] = f.hi;
    }
    __syncthreads();
    return fix_warp_sum(Fix{sh[2 * (threadIdx.x & 31)], sh[2 * (threadIdx.x & 31) + 1]});
}

struct SelectScratch {
    u64 red[64];
    unsigned int hist[kBins];
    u64 cand[kDirect];
    unsigned int warp_sum[32];
    unsigned int n_cand;
    int bin;
    unsigned int above;
    u64 found;
};

// The bin of s.hist where the count from the top reaches krem (into s.bin) and
// the count above it (s.above): two bins per thread, a scan over the block.
__device__ __forceinline__ void pick_bin(SelectScratch& s, unsigned int krem) {
    static_assert(kBins == 2 * kFinishThreads, "two bins per thread");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b1 = kBins - 1 - 2 * (int)threadIdx.x, b0 = b1 - 1;  // from the top
    const unsigned int c1 = s.hist[b1], c0 = s.hist[b0];
    unsigned int incl = c1 + c0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int v = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s.warp_sum[w] = incl;
    __syncthreads();
    const unsigned int ws = s.warp_sum[lane];
    incl += __reduce_add_sync(kAll, lane < w ? ws : 0u);
    const unsigned int excl = incl - c1 - c0;
    if (excl < krem && krem <= incl) {
        const bool first = krem <= excl + c1;
        s.bin = first ? b1 : b0;
        s.above = first ? excl : excl + c1;
        s.n_cand = 0;
    }
    __syncthreads();
}

// f(key) for the keys get(0) .. get(n - 1), shared out over the block, eight
// loads in flight per thread (a list or a row that is not held in shared
// memory comes from L2 or HBM).
template <class Get, class F>
__device__ __forceinline__ void for_each_key(Get get, int64_t n, F f) {
    constexpr int U = 8;
    for (int64_t i0 = threadIdx.x; i0 < n; i0 += (int64_t)U * kFinishThreads) {
        u64 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + (int64_t)u * kFinishThreads;
            v[u] = i < n ? get(i) : 0ULL;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + (int64_t)u * kFinishThreads < n) f(v[u]);
    }
}

// Keys that a list leaves out, with their counts (0: none).
struct Ties {
    u64 key[kTies], n[kTies];
};

// The k-th largest (k >= 1) of the n keys that get(i) yields and of the ties;
// they are k or more. Every thread of the block calls it and receives it. MSD radix select over the offsets from the smallest key lo; once few candidates are left they are ranked directly.
template <class Get>
__device__ u64 kth_largest(Get get, int64_t n, const Ties& ties, u64 lo, u64 hi, long long k, SelectScratch& s) {
    int top = 64 - __clzll((long long)(hi - lo));  // bits of the largest offset
    u64 prefix = 0;                               // of the offset, in units of 2^top
    long long krem = k;
    while (top > 0) {
        const int bits = min(11, top), shift = top - bits;
        for (int i = threadIdx.x; i < kBins; i += blockDim.x) s.hist[i] = 0;
        __syncthreads();
        for_each_key(get, n, [&](u64 v) {
            const u64 d = v - lo;
            if ((d >> top) == prefix) atomicAdd(&s.hist[(d >> shift) & ((1u << bits) - 1)], 1u);
        });
        if (threadIdx.x == 0)
#pragma unroll
            for (int i = 0; i < kTies; ++i) {
                const u64 d = ties.key[i] - lo;
                if (ties.n[i] && (d >> top) == prefix)
                    atomicAdd(&s.hist[(d >> shift) & ((1u << bits) - 1)], (unsigned)ties.n[i]);
            }
        __syncthreads();
        pick_bin(s, (unsigned int)krem);
        const u64 in_bin = s.hist[s.bin];
        prefix = prefix << bits | (u64)s.bin;
        krem -= (long long)s.above;
        top = shift;
        if (in_bin <= kDirect) {
            // few left: list them (ties once, with their count) and rank each
            // against the others
            for_each_key(get, n, [&](u64 v) {
                if (((v - lo) >> top) == prefix) s.cand[atomicAdd(&s.n_cand, 1u)] = v;
            });
            __syncthreads();
            const int m = (int)s.n_cand;
            for (int c = threadIdx.x; c < m + kTies; c += blockDim.x) {
                const u64 v = c < m ? s.cand[c] : c == m ? ties.key[0] : ties.key[1];
                if (c >= m && !((c == m ? ties.n[0] : ties.n[1]) && ((v - lo) >> top) == prefix)) continue;
                u64 gt = 0, ge = 0;
                for (int j = 0; j < m; ++j) {
                    gt += s.cand[j] > v;
                    ge += s.cand[j] >= v;
                }
#pragma unroll
                for (int i = 0; i < kTies; ++i)
                    if (((ties.key[i] - lo) >> top) == prefix) {
                        gt += ties.key[i] > v ? ties.n[i] : 0ULL;
                        ge += ties.key[i] >= v ? ties.n[i] : 0ULL;
                    }
                if ((long long)gt < krem && krem <= (long long)ge) s.found = v;  // the same value from equal candidates
            }
            __syncthreads();
            const u64 v = s.found;
            __syncthreads();
            return v;
        }
        __syncthreads();
    }
    return lo + prefix;
}

// Hashed sample positions (a multiplicative hash: patterns in the row's order
// do not line up with it).
__device__ __forceinline__ int64_t sample_pos(int i, int64_t n) {
    const u64 h = ((u64)i + 1) * 0x9e3779b97f4a7c15ULL;
    return (int64_t)__umul64hi(h ^ (h >> 29), (u64)n);
}

// The threshold's low word is left 0 (a slightly lower T), so the select works
// on high words: two 11-bit digits of their offset from the sample's smallest.
__global__ void __launch_bounds__(kFinishThreads) list_sample_kernel(const double* __restrict__ ylt, int64_t n,
                                                                     int rank, ListState* __restrict__ st) {
    __shared__ SelectScratch s;
    constexpr int PER = kSample / kFinishThreads;
    const u64* row = reinterpret_cast<const u64*>(ylt) + (size_t)blockIdx.x * (size_t)n;
    u64 v[PER];
    u64 mx = 0, mn = ~0ULL;
#pragma unroll
    for (int i = 0; i < PER; ++i) v[i] = row[sample_pos(i * kFinishThreads + threadIdx.x, n)] & 0x7fffffffffffffffULL;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        mx = max(mx, v[i]);
        mn = min(mn, v[i]);
    }
    for (int i = threadIdx.x; i < kBins; i += kFinishThreads) s.hist[i] = 0;
    mx = block_max(mx, s.red);
    mn = ~block_max(~mn, s.red);
    unsigned int rep = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) rep += v[i] == mx;
    const u64 repeats = block_sum(rep, s.red);
    const unsigned int lo = (unsigned int)(mn >> 32);
    const int top = 32 - __clz((int)((unsigned int)(mx >> 32) - lo));
    const int sh1 = max(top - 11, 0), sh2 = max(top - 22, 0);
#pragma unroll
    for (int i = 0; i < PER; ++i) atomicAdd(&s.hist[((unsigned int)(v[i] >> 32) - lo) >> sh1], 1u);
    __syncthreads();
    pick_bin(s, (unsigned int)rank);
    const unsigned int b1 = (unsigned int)s.bin, above = s.above;
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += kFinishThreads) s.hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const unsigned int d = (unsigned int)(v[i] >> 32) - lo;
        if (d >> sh1 == b1) atomicAdd(&s.hist[(d >> sh2) & ((1u << (sh1 - sh2)) - 1u)], 1u);
    }
    __syncthreads();
    pick_bin(s, (unsigned int)rank - above);
    u64 threshold = (u64)(lo + (((b1 << (sh1 - sh2)) | (unsigned int)s.bin) << sh2)) << 32;
    // Many sample keys in the r-th largest's bin: a value that repeats, such as
    // one full limit of a layer whose events mostly pay theirs. Its exact key
    // becomes a tie key too, or the list would take every one of it.
    u64 atom = kNoTie;
    if (s.hist[s.bin] > kAtom && threshold && repeats < (u64)rank) {
        const u64 base = threshold;
        const int width = sh2 + 32;
        unsigned int krem = (unsigned int)rank - above - s.above, same = 0;
        u64 prefix = 0;
        for (int left = width; left > 0;) {
            const int bits = min(11, left), shift = left - bits;
            __syncthreads();
            for (int i = threadIdx.x; i < kBins; i += kFinishThreads) s.hist[i] = 0;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < PER; ++i) {
                const u64 d = v[i] - base;  // wraps below the bin
                if (!(d >> width) && (d >> left) == prefix)
                    atomicAdd(&s.hist[(d >> shift) & ((1u << bits) - 1)], 1u);
            }
            __syncthreads();
            pick_bin(s, krem);
            prefix = prefix << bits | (u64)s.bin;
            krem -= s.above;
            same = s.hist[s.bin];
            left = shift;
        }
        threshold = (base + prefix) & ~0xffffffffULL;
        if (same > 1) atom = base + prefix;
    }
    if (threadIdx.x == 0) {
        ListState l{};
        l.threshold = threshold;
        l.tie[0] = repeats > 1 && mx ? mx : atom;
        l.tie[1] = l.tie[0] != atom ? atom : kNoTie;
        // room for losses 4,096 times the sample's largest; the pass's short
        // fixed point wants as much below. T = 0: the list (and the ties) will
        // hold every loss but 0, and the finish sums it (a layer of few losses
        // has no sample to set a reference by)
        l.ref = l.threshold ? min(ref_exp(mx) + 12, 2046) : 0;
        l.again = l.threshold && l.ref < 128 ? kUnlisted : 0u;
        st[blockIdx.x] = l;
    }
}

__global__ void __launch_bounds__(kPassThreads, 5) list_pass_kernel(const double* __restrict__ ylt, int64_t n,
                                                                 ListState* __restrict__ st, u64* __restrict__ lists,
                                                                 unsigned int cap) {
    const int j = blockIdx.y;
    const unsigned lane = threadIdx.x & 31;
    const u64* row = reinterpret_cast<const u64*>(ylt) + (size_t)j * (size_t)n;
    u64* list = lists + (size_t)j * cap;
    // keys of a high word from thr on are listed; zeros never are
    const unsigned int thr = max((unsigned int)(st[j].threshold >> 32), 1u);
    const unsigned int tie_hi = (unsigned int)(st[j].tie[0] >> 32), tie_lo = (unsigned int)st[j].tie[0];
    const unsigned int tie2_hi = (unsigned int)(st[j].tie[1] >> 32), tie2_lo = (unsigned int)st[j].tie[1];
    const int ref = st[j].ref;
    // no reference: every loss is out of the short sum's range, a subnormal too
    const unsigned int dref = ref ? (unsigned int)ref : 0x7fffffffu;
    // The sum as four 32-bit words, the highest a carry: a key within 31
    // binades below ref is its mantissa at the top of 96 bits, shifted down
    // (three shifts and four adds; no bit is lost, so the unit is 2^-96 of
    // ref's upper end, as in the general path). Zeros add nothing; any other
    // key (rare) goes the long way in `rest`.
    unsigned int a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    Fix rest{0, 0};
    unsigned int n_tie = 0, n_tie2 = 0;
    unsigned int again = 0;
    // two: the layer has a second tie key (few layers do; the others are
    // spared its comparison)
    auto read_row = [&](auto two) {
        for (int64_t i0 = (int64_t)blockIdx.x * kPassThreads * kPassUnroll; i0 < n;
             i0 += (int64_t)gridDim.x * kPassThreads * kPassUnroll) {
            unsigned int kh[kPassUnroll], kl[kPassUnroll];  // 0 past the end
            if (i0 + kPassThreads * kPassUnroll <= n) {
#pragma unroll
                for (int u = 0; u < kPassUnroll; ++u) {
                    const u64 v = key_at(row, i0 + u * kPassThreads + threadIdx.x);
                    kh[u] = (unsigned int)(v >> 32);
                    kl[u] = (unsigned int)v;
                }
            } else {
#pragma unroll
                for (int u = 0; u < kPassUnroll; ++u) {
                    const int64_t i = i0 + (int64_t)u * kPassThreads + threadIdx.x;
                    const u64 v = i < n ? key_at(row, i) : 0ULL;
                    kh[u] = (unsigned int)(v >> 32);
                    kl[u] = (unsigned int)v;
                }
            }
            unsigned in = 0, odd = 0;  // bit u: listed; summed the long way
#pragma unroll
            for (int u = 0; u < kPassUnroll; ++u) {
                const unsigned int d = dref - (kh[u] >> 20);
                const unsigned int hi = __funnelshift_l(kl[u], kh[u], 11) | 0x80000000u, lo = kl[u] << 11;
                const unsigned int x2 = hi >> (d & 31), x1 = __funnelshift_r(lo, hi, d), x0 = __funnelshift_r(0u, lo, d);
                asm("{\n.reg .pred p;\nsetp.lt.u32 p, %4, 32;\n"
                    "@p add.cc.u32 %0, %0, %5;\n@p addc.cc.u32 %1, %1, %6;\n"
                    "@p addc.cc.u32 %2, %2, %7;\n@p addc.u32 %3, %3, 0;\n}"
                    : "+r"(a0), "+r"(a1), "+r"(a2), "+r"(a3)
                    : "r"(d), "r"(x0), "r"(x1), "r"(x2));
                if (d >= 32u && (kh[u] | kl[u])) odd |= 1u << u;
                const bool eq = kh[u] == tie_hi && kl[u] == tie_lo;
                n_tie += eq;
                bool eq2 = false;
                if constexpr (decltype(two)::value) {
                    eq2 = kh[u] == tie2_hi && kl[u] == tie2_lo;
                    n_tie2 += eq2;
                }
                if (kh[u] >= thr && !eq && !eq2) in |= 1u << u;
            }
            if (odd) {
#pragma unroll
                for (int u = 0; u < kPassUnroll; ++u)
                    if ((odd >> u) & 1u) {
                        // a key above ref, or below what the list's threshold can tell from 0
                        if (kh[u] == 0u) again |= kUnlisted;
                        else if (ref && (int)(kh[u] >> 20) > ref) again |= kSumOut;
                        else if (ref) fix_add(rest, (u64)kh[u] << 32 | kl[u], ref);
                    }
            }
            if (__any_sync(kAll, in != 0u)) {
                // one counter update per warp and step: a scan of the lanes' counts
                const unsigned c = __popc(in);
                unsigned incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned v = __shfl_up_sync(kAll, incl, o);
                    if (lane >= (unsigned)o) incl += v;
                }
                unsigned base = 0;
                if (lane == 31) base = atomicAdd(&st[j].n_list, incl);
                base = __shfl_sync(kAll, base, 31) + incl - c;
#pragma unroll
                for (int u = 0; u < kPassUnroll; ++u)
                    if ((in >> u) & 1u) {
                        if (base < cap) list[base] = (u64)kh[u] << 32 | kl[u];
                        ++base;
                    }
            }
        }
    };
    if (st[j].tie[1] == kNoTie) read_row(std::false_type{});
    else read_row(std::true_type{});
    // the words hold units of 2^(ref - 1075 - 43): twice kFixBits' unit
    Fix sum{(u64)a1 << 32 | a0, (u64)a3 << 32 | a2};
    sum = Fix{sum.lo << 1, sum.hi << 1 | sum.lo >> 63};
    fix_add2(sum, rest.lo, rest.hi);
    fix_block_atomic(st[j].sum, sum);
    n_tie = __reduce_add_sync(kAll, n_tie);
    if (lane == 0 && n_tie) atomicAdd(&st[j].n_tie[0], (u64)n_tie);
    n_tie2 = __reduce_add_sync(kAll, n_tie2);
    if (lane == 0 && n_tie2) atomicAdd(&st[j].n_tie[1], (u64)n_tie2);
    if (again) atomicOr(&st[j].again, again);
}

// st NULL: the whole row is in shared memory.
__global__ void __launch_bounds__(kFinishThreads, 1) list_finish_kernel(const double* __restrict__ ylt, int64_t n,
                                                                       const Ranks rk, const ListState* __restrict__ st,
                                                                       const u64* __restrict__ lists, unsigned int cap,
                                                                       double* mean, double* pml, double* tvar,
                                                                       double* sum_out) {
    extern __shared__ __align__(16) u64 s_keys[];
    __shared__ SelectScratch s;
    const int j = blockIdx.x;
    const u64* row = reinterpret_cast<const u64*>(ylt) + (size_t)j * (size_t)n;
    long long kmax_rank = 0;
    for (int q = 0; q < rk.n_p; ++q) kmax_rank = max(kmax_rank, rk.k[q]);
    bool use_list = false, have_sum = false;
    Ties ties{};
    int64_t m = n;  // keys of the source
    Fix total{0, 0};
    int sum_ref = 0;
    if (st) {
        const ListState l = st[j];
        have_sum = !l.again && l.ref;
        total = Fix{l.sum[0], l.sum[1]};
        sum_ref = l.ref;
        // every loss other than 0 that the list leaves out is below T
        use_list = !(l.again & kUnlisted) && l.n_list <= cap &&
                   (l.threshold == 0 || (long long)(l.n_list + l.n_tie[0] + l.n_tie[1]) >= kmax_rank);
        if (use_list) {
            m = l.n_list;
#pragma unroll
            for (int i = 0; i < kTies; ++i) {
                ties.key[i] = l.n_tie[i] ? l.tie[i] : 0ULL;
                ties.n[i] = l.n_tie[i];
            }
        }
    }
    const u64 n_ties = ties.n[0] + ties.n[1];
    const u64* src = use_list ? lists + (size_t)j * cap : row;
    const bool held = m <= kSmall;
    u64 mx = max(ties.key[0], ties.key[1]), mn = ~0ULL;
#pragma unroll
    for (int i = 0; i < kTies; ++i)
        if (ties.n[i]) mn = min(mn, ties.key[i]);
    constexpr int U = 8;  // loads in flight per thread
    for (int64_t i0 = threadIdx.x; i0 < m; i0 += (int64_t)U * kFinishThreads) {
        u64 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + (int64_t)u * kFinishThreads;
            v[u] = i < m ? src[i] & 0x7fffffffffffffffULL : 0ULL;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + (int64_t)u * kFinishThreads;
            if (i < m) {
                if (held) s_keys[i] = v[u];
                mx = max(mx, v[u]);
                mn = min(mn, v[u]);
            }
        }
    }
    mx = block_max(mx, s.red);
    mn = ~block_max(~mn, s.red);
    if (mn > mx) mn = mx;  // nothing listed: every loss is 0
    const int e_ref = ref_exp(mx);
    auto get = [&](int64_t i) { return held ? s_keys[i] : src[i] & 0x7fffffffffffffffULL; };
    if (!have_sum) {
        // from the list where it holds every loss but 0; where only some loss lay
        // above the sum's range, from the row (its largest key is the list's)
        Fix f{0, 0};
        if (use_list && st[j].ref)
            for_each_key([&](int64_t i) { return row[i] & 0x7fffffffffffffffULL; }, n, [&](u64 v) { fix_add(f, v, e_ref); });
        else for_each_key(get, m, [&](u64 v) { fix_add(f, v, e_ref); });
        total = block_fix(f, s.red);
        if (!(use_list && st[j].ref))
#pragma unroll
            for (int i = 0; i < kTies; ++i)
                if (ties.n[i]) fix_add_times(total, ties.key[i], e_ref, ties.n[i]);
        sum_ref = e_ref;
    }
    if (threadIdx.x == 0) {
        const double t = fix_value(total, sum_ref);
        if (mean) mean[j] = t / (double)n;
        if (sum_out) sum_out[j] = t;
    }
    for (int q = 0; q < rk.n_p; ++q) {
        const long long k = rk.k[q];
        u64 v = 0;  // fewer than k losses above 0
        if ((long long)(m + n_ties) >= k)
            v = mn == mx || (ties.key[0] == mx && ties.n[0] >= (u64)k) ? mx : kth_largest(get, m, ties, mn, mx, k, s);
        Fix f{0, 0};
        u64 cnt = 0;
        if (v < mx)
            for_each_key(get, m, [&](u64 key) {
                if (key > v) {
                    fix_add(f, key, e_ref);
                    ++cnt;
                }
            });
        f = block_fix(f, s.red);
        cnt = block_sum(cnt, s.red);
        if (threadIdx.x == 0) {
#pragma unroll
            for (int i = 0; i < kTies; ++i)
                if (ties.n[i] && ties.key[i] > v) {
                    fix_add_times(f, ties.key[i], e_ref, ties.n[i]);
                    cnt += ties.n[i];
                }
            const double x = __longlong_as_double((long long)v);
            const size_t w = (size_t)j * rk.n_p + q;
            if (pml) pml[w] = x;
            if (tvar) tvar[w] = (fix_value(f, e_ref) + (double)(k - (long long)cnt) * x) / (double)k;
        }
        __syncthreads();
    }
}

unsigned int list_cap(int64_t n) { return (unsigned int)((n + 7) / 8); }

// Rank in the sample of the list's threshold: the sample's share of the k
// largest, six standard deviations and a few more.
int sample_rank(int64_t n, int64_t k_max) {
    const double share = (double)k_max * kSample / (double)n;
    return (int)std::min<double>(kSample, std::ceil(share + 6.0 * std::sqrt(share) + 8.0));
}

}  // namespace

// Rows that go to the finish whole. It has room for kSmall, but from here on
// the sample and the pass are faster (12,288 trials, 3 probabilities: 42 us
// whole and 34 sampled for one layer, 541 and 379 for 2,000; 8,192 trials: 32
// and 34, 397 and 357; with three atoms in the row whole rows pay more, as
// their keys meet in few bins: 26,624 trials x 2,000 layers 1.50 ms against 0.69).
bool metrics_small(int64_t n) { return n <= 12288; }

// Whether the list path takes the call. Its lists have room for the ranks up
// to n / 20 (they then hold well under n / 8), and its finish is one CTA per
// layer, so few layers with long lists are left to the general path, whose
// every step is spread over the chip. Both times in us, fitted to 1 to 128
// layers of 200,000 to 100,000,000 trials at 1 and 3 probabilities (within
// about a fifth): the pass grows with the YLT, the finish with each list,
// twice as fast where shared memory holds it. One layer of 1,000,000 trials at
// 0.95: 133 us by list, 100 in general; at 0.99: 50 and 95; 128 layers at 0.95:
// 415 and 1,005; one layer of 100,000,000 at 0.99: 2,964 and 702.
bool metrics_listable(int64_t n, int32_t n_layers, int64_t k_max, int32_t n_p) {
    if (metrics_small(n)) return true;
    if (k_max > n / 20 || n_layers > 65535) return false;
    const double m = (double)n * sample_rank(n, k_max) / kSample, all = 1e-6 * (double)n * n_layers;
    const double per_key = 1e-3 * (0.3 + (m <= kSmall ? 0.5 : 1.1) * n_p);
    const double waves = (n_layers + 147) / 148;
    const double list = 28.0 + std::max(std::min(9.0 * all, 90.0 + 1.2 * all), 3.5e-6 * (double)n) + waves * m * per_key;
    const double general = 65.0 + 28.0 * n_p + (5.2 + 1.4 * n_p) * all;
    return list <= general;
}

size_t metrics_list_bytes(int64_t n, int32_t n_layers) {
    if (metrics_small(n)) return 256;
    return ((sizeof(ListState) * (size_t)n_layers + 255) & ~(size_t)255) +
           sizeof(u64) * (size_t)n_layers * list_cap(n);
}

cudaError_t metrics_list_run(const double* ylt, int64_t n, int32_t n_layers, const int64_t* k, int32_t n_p, double* mean,
                             double* pml, double* tvar, double* sum_out, cudaStream_t s, void* scratch) {
    Ranks rk{};
    rk.n_p = n_p;
    int64_t k_max = 1;
    for (int q = 0; q < n_p; ++q) {
        rk.k[q] = std::min<int64_t>(n, std::max<int64_t>(1, k[q]));
        k_max = std::max<int64_t>(k_max, rk.k[q]);
    }
    cudaError_t e;
    const int smem = (int)(sizeof(u64) * std::min<int64_t>(n, kSmall));
    // the limit is the function's, not the call's: every call sets the same (as allow_max_shared)
    if ((e = cudaFuncSetAttribute(list_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(u64) * kSmall)))
        return e;
    ListState* st = nullptr;
    u64* lists = nullptr;
    const unsigned int cap = list_cap(n);
    if (!metrics_small(n)) {
        st = reinterpret_cast<ListState*>(scratch);
        lists = reinterpret_cast<u64*>(static_cast<char*>(scratch) +
                                       ((sizeof(ListState) * (size_t)n_layers + 255) & ~(size_t)255));
        list_sample_kernel<<<(unsigned)n_layers, kFinishThreads, 0, s>>>(ylt, n, sample_rank(n, k_max), st);
        if ((e = cudaGetLastError())) return e;
        int dev = 0, sms = 148;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // about 32 CTAs per SM over all layers (about five run at a time: more,
        // shorter CTAs leave less of the last wave empty), each at least one step
        const int64_t steps = (n + kPassThreads * kPassUnroll - 1) / (kPassThreads * kPassUnroll);
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(steps, (32LL * sms + n_layers - 1) / n_layers));
        list_pass_kernel<<<dim3((unsigned)blocks, (unsigned)n_layers), kPassThreads, 0, s>>>(ylt, n, st, lists, cap);
        if ((e = cudaGetLastError())) return e;
    }
    list_finish_kernel<<<(unsigned)n_layers, kFinishThreads, smem, s>>>(ylt, n, rk, st, lists, cap, mean, pml, tvar, sum_out);
    return cudaGetLastError();
}

}  // namespace art

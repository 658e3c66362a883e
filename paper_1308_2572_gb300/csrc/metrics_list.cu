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
//      are not 0.
//   3. finish (one CTA per layer): the k-th largest of list and ties by a
//      radix select in shared memory, the exact sum of the losses above it,
//      mean, PML and TVaR. If the list holds fewer than k losses and T > 0, or
//      overflowed, or a loss lay far above the sample's largest, the CTA takes
//      the row instead: slower, the same results.
// A YLT of at most kSmall trials skips 1 and 2: its rows fit shared memory.
//
// What bounds it: HBM (8 bytes per loss, once); the general path's two full
// reads and six list passes took 1.04 ms on 128 layers x 1,000,000 trials at
// three probabilities, this takes 0.47 ms (floor 0.15), and one layer's metrics
// 43 us against 89 (eight dependent launches).
#include <algorithm>
#include <cmath>

#include "art_internal.cuh"

namespace art {

namespace {

typedef unsigned long long u64;

constexpr unsigned kAll = 0xffffffffu;
constexpr int kSample = 4096;
constexpr int kFinishThreads = 1024;
constexpr int kSmall = 20480;        // keys the finish CTA holds in shared memory (160 KB)
constexpr int kPassThreads = 256;
constexpr int kPassUnroll = 8;       // values per thread whose loads are in flight together
constexpr u64 kNoTie = ~0ULL;
constexpr int kBins = 2048;          // 11-bit digits
constexpr int kDirect = 512;         // candidates that are ranked by comparison

struct Ranks {
    long long k[kMaxProbs];
    int n_p;
};

// Per-layer state, written by the sample.
struct ListState {
    u64 threshold;   // T
    u64 tie;         // the tie key (kNoTie: none)
    u64 sum[2];      // fixed-point sum of the row (unit by ref)
    u64 n_tie;
    unsigned int n_list;
    int ref;         // reference exponent of the sum
    unsigned int beyond;  // a loss with an exponent above ref was seen
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
    unsigned int n_cand;
    int bin;
    u64 above;
    u64 found;
};

// The k-th largest (k >= 1) of the n keys that get(i) yields, of which tie
// counts n_tie more times; n + n_tie >= k. Every thread of the block calls it
// and receives it. MSD radix select over the offsets from the smallest
// possible key lo; once few candidates are left they are ranked directly.
template <class Get>
__device__ u64 kth_largest(Get get, int64_t n, u64 tie, u64 n_tie, u64 lo, u64 hi, long long k, SelectScratch& s) {
    int top = 64 - __clzll((long long)(hi - lo));  // bits of the largest offset
    u64 prefix = 0;                               // of the offset, in units of 2^top
    long long krem = k;
    while (top > 0) {
        const int bits = min(11, top), shift = top - bits;
        for (int i = threadIdx.x; i < kBins; i += blockDim.x) s.hist[i] = 0;
        __syncthreads();
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            const u64 d = get(i) - lo;
            if (get(i) >= lo && (top >= 64 || (d >> top) == prefix)) atomicAdd(&s.hist[(d >> shift) & ((1u << bits) - 1)], 1u);
        }
        if (threadIdx.x == 0 && n_tie) {
            const u64 d = tie - lo;
            if (tie >= lo && (top >= 64 || (d >> top) == prefix)) atomicAdd(&s.hist[(d >> shift) & ((1u << bits) - 1)], (unsigned)n_tie);
        }
        __syncthreads();
        // the bin where the count from the top reaches krem: warp 0 scans 64
        // bins per lane, from the top
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            u64 mine = 0;
            for (int b = 0; b < kBins / 32; ++b) mine += s.hist[kBins - 1 - (lane * (kBins / 32) + b)];
            u64 incl = mine;
            for (int o = 1; o < 32; o <<= 1) {
                const u64 v = __shfl_up_sync(kAll, incl, o);
                if (lane >= o) incl += v;
            }
            u64 run = incl - mine;
            if ((long long)run < krem && krem <= (long long)incl)
                for (int b = 0; b < kBins / 32; ++b) {
                    const int bin = kBins - 1 - (lane * (kBins / 32) + b);
                    const unsigned c = s.hist[bin];
                    if ((long long)(run + c) >= krem) {
                        s.bin = bin;
                        s.above = run;
                        s.n_cand = 0;
                        break;
                    }
                    run += c;
                }
        }
        __syncthreads();
        const u64 in_bin = s.hist[s.bin];
        prefix = prefix << bits | (u64)s.bin;
        krem -= (long long)s.above;
        top = shift;
        if (in_bin <= kDirect) {
            // few left: list them (ties once, with their count) and rank each
            // against the others
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
                const u64 v = get(i);
                if (v >= lo && ((v - lo) >> top) == prefix) s.cand[atomicAdd(&s.n_cand, 1u)] = v;
            }
            __syncthreads();
            const int m = (int)s.n_cand;
            const bool tie_in = n_tie && tie >= lo && ((tie - lo) >> top) == prefix;
            for (int c = threadIdx.x; c < m + (tie_in ? 1 : 0); c += blockDim.x) {
                const u64 v = c < m ? s.cand[c] : tie;
                u64 gt = 0, ge = 0;
                for (int j = 0; j < m; ++j) {
                    gt += s.cand[j] > v;
                    ge += s.cand[j] >= v;
                }
                if (tie_in) {
                    gt += tie > v ? n_tie : 0ULL;
                    ge += tie >= v ? n_tie : 0ULL;
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

__global__ void __launch_bounds__(kFinishThreads) list_sample_kernel(const double* __restrict__ ylt, int64_t n,
                                                                     int rank, ListState* __restrict__ st) {
    __shared__ u64 s_keys[kSample];
    __shared__ SelectScratch s;
    const u64* row = reinterpret_cast<const u64*>(ylt) + (size_t)blockIdx.x * (size_t)n;
    u64 mx = 0;
    for (int i = threadIdx.x; i < kSample; i += kFinishThreads) {
        const u64 v = row[sample_pos(i, n)] & 0x7fffffffffffffffULL;
        s_keys[i] = v;
        mx = max(mx, v);
    }
    mx = block_max(mx, s.red);
    u64 rep = 0;
    for (int i = threadIdx.x; i < kSample; i += kFinishThreads) rep += s_keys[i] == mx;
    rep = block_sum(rep, s.red);
    const u64 t = kth_largest([&](int64_t i) { return s_keys[i]; }, kSample, 0ULL, 0ULL, 0ULL, mx, rank, s);
    if (threadIdx.x == 0) {
        ListState l{};
        l.threshold = t;
        l.tie = rep > 1 && mx ? mx : kNoTie;
        l.ref = min(ref_exp(mx) + 3, 2046);
        st[blockIdx.x] = l;
    }
}

__global__ void __launch_bounds__(kPassThreads) list_pass_kernel(const double* __restrict__ ylt, int64_t n,
                                                                 ListState* __restrict__ st, u64* __restrict__ lists,
                                                                 unsigned int cap) {
    const int j = blockIdx.y;
    const unsigned lane = threadIdx.x & 31;
    const u64* row = reinterpret_cast<const u64*>(ylt) + (size_t)j * (size_t)n;
    u64* list = lists + (size_t)j * cap;
    const u64 thr = max(st[j].threshold, 1ULL), tie = st[j].tie;  // zeros are never listed
    const int ref = st[j].ref;
    Fix sum{0, 0};
    unsigned int n_tie = 0;
    bool beyond = false;
    for (int64_t i0 = (int64_t)blockIdx.x * kPassThreads * kPassUnroll; i0 < n;
         i0 += (int64_t)gridDim.x * kPassThreads * kPassUnroll) {
        u64 kv[kPassUnroll];  // 0 past the end
#pragma unroll
        for (int u = 0; u < kPassUnroll; ++u) {
            const int64_t i = i0 + (int64_t)u * kPassThreads + threadIdx.x;
            kv[u] = i < n ? key_at(row, i) : 0ULL;
        }
        unsigned in = 0;  // bit u: listed
#pragma unroll
        for (int u = 0; u < kPassUnroll; ++u) {
            const u64 key = kv[u];
            const int e = (int)(key >> 52);
            if (e <= ref) fix_add(sum, key, ref);
            else beyond = true;
            const bool eq = key == tie;
            n_tie += eq;
            in |= (unsigned)(key >= thr && !eq) << u;
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
                    if (base < cap) list[base] = kv[u];
                    ++base;
                }
        }
    }
    fix_block_atomic(st[j].sum, sum);
    n_tie = __reduce_add_sync(kAll, n_tie);
    if (lane == 0 && n_tie) atomicAdd(&st[j].n_tie, (u64)n_tie);
    if (beyond) atomicOr(&st[j].beyond, 1u);
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
    u64 tie = 0, n_tie = 0;
    int64_t m = n;  // keys of the source
    Fix total{0, 0};
    int sum_ref = 0;
    if (st) {
        const ListState l = st[j];
        have_sum = !l.beyond;
        total = Fix{l.sum[0], l.sum[1]};
        sum_ref = l.ref;
        // every loss other than 0 that the list leaves out is below T
        use_list = have_sum && l.n_list <= cap &&
                   (l.threshold == 0 || (long long)(l.n_list + l.n_tie) >= kmax_rank);
        if (use_list) {
            m = l.n_list;
            tie = l.tie;
            n_tie = l.n_tie;
        }
    }
    const u64* src = use_list ? lists + (size_t)j * cap : row;
    const bool held = m <= kSmall;
    u64 mx = n_tie ? tie : 0ULL, mn = n_tie ? tie : ~0ULL;
    for (int64_t i = threadIdx.x; i < m; i += kFinishThreads) {
        const u64 v = src[i] & 0x7fffffffffffffffULL;
        if (held) s_keys[i] = v;
        mx = max(mx, v);
        mn = min(mn, v);
    }
    mx = block_max(mx, s.red);
    mn = ~block_max(~mn, s.red);
    if (mn > mx) mn = mx;  // nothing listed: every loss is 0
    const int e_ref = ref_exp(mx);
    auto get = [&](int64_t i) { return held ? s_keys[i] : src[i] & 0x7fffffffffffffffULL; };
    if (!have_sum) {
        Fix f{0, 0};
        for (int64_t i = threadIdx.x; i < m; i += kFinishThreads) fix_add(f, get(i), e_ref);
        total = block_fix(f, s.red);
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
        if ((long long)(m + n_tie) >= k)
            v = mn == mx || (tie == mx && n_tie >= (u64)k) ? mx : kth_largest(get, m, tie, n_tie, mn, mx, k, s);
        Fix f{0, 0};
        u64 cnt = 0;
        if (v < mx)
            for (int64_t i = threadIdx.x; i < m; i += kFinishThreads) {
                const u64 key = get(i);
                if (key > v) {
                    fix_add(f, key, e_ref);
                    ++cnt;
                }
            }
        f = block_fix(f, s.red);
        cnt = block_sum(cnt, s.red);
        if (threadIdx.x == 0) {
            if (n_tie && tie > v) {
                fix_add_times(f, tie, e_ref, n_tie);
                cnt += n_tie;
            }
            const double x = __longlong_as_double((long long)v);
            const size_t w = (size_t)j * rk.n_p + q;
            if (pml) pml[w] = x;
            if (tvar) tvar[w] = (fix_value(f, e_ref) + (double)(k - (long long)cnt) * x) / (double)k;
        }
        __syncthreads();
    }
}

unsigned int list_cap(int64_t n) { return (unsigned int)std::max<int64_t>(n / 8, 8192); }

}  // namespace

bool metrics_small(int64_t n) { return n <= kSmall; }

// The list path takes ranks up to n / 20 (its lists then hold well under the
// n / 8 losses they have room for).
bool metrics_listable(int64_t n, int32_t n_layers, int64_t k_max) {
    return metrics_small(n) || (k_max <= n / 20 && n_layers <= 65535);
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
    if ((e = cudaFuncSetAttribute(list_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
    ListState* st = nullptr;
    u64* lists = nullptr;
    const unsigned int cap = list_cap(n);
    if (!metrics_small(n)) {
        st = reinterpret_cast<ListState*>(scratch);
        lists = reinterpret_cast<u64*>(static_cast<char*>(scratch) +
                                       ((sizeof(ListState) * (size_t)n_layers + 255) & ~(size_t)255));
        // the sample's share of the k largest, six standard deviations and a few more
        const double share = (double)k_max * kSample / (double)n;
        const int rank = (int)std::min<double>(kSample, std::ceil(share + 6.0 * std::sqrt(share) + 8.0));
        list_sample_kernel<<<(unsigned)n_layers, kFinishThreads, 0, s>>>(ylt, n, rank, st);
        if ((e = cudaGetLastError())) return e;
        int dev = 0, sms = 148;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        // about 8 CTAs per SM over all layers, each at least one step
        const int64_t steps = (n + kPassThreads * kPassUnroll - 1) / (kPassThreads * kPassUnroll);
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(steps, (8LL * sms + n_layers - 1) / n_layers));
        list_pass_kernel<<<dim3((unsigned)blocks, (unsigned)n_layers), kPassThreads, 0, s>>>(ylt, n, st, lists, cap);
        if ((e = cudaGetLastError())) return e;
    }
    list_finish_kernel<<<(unsigned)n_layers, kFinishThreads, smem, s>>>(ylt, n, rk, st, lists, cap, mean, pml, tvar, sum_out);
    return cudaGetLastError();
}

}  // namespace art

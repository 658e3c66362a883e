// id_stream.cuh -- what the trial passes over whole-number tables share: a
// warp's stream of event ids (bulk copies into shared memory), its masking,
// and the occupancy bitmap folded into shared memory.
#pragma once

#include "art_internal.cuh"

namespace art {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kWaitNs = 4000000000ULL;  // longest wait for a copy
// Most events of a trial: positions are 32-bit, and a chunk's end must not wrap.
constexpr int64_t kMaxTrialIds = 0xfffff000LL;

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ld_bits(const uint32_t* p) {
    uint32_t v;
    asm("ld.global.nc.L1::evict_last.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// The ids of one trial as the warp reads them: n positions from a 16-byte
// boundary, of which the first `head` belong to the trial before. VEC: every
// trial starts and ends on a 16-byte boundary.
template <bool VEC>
struct Span {
    const int32_t* p = nullptr;  // 16-byte aligned (position 0)
    uint32_t n = 0, head_ = 0;
    bool edge_ = false;          // a vector of it leaves the id array: read id by id
    __device__ __forceinline__ uint32_t head() const { return VEC ? 0u : head_; }
    __device__ __forceinline__ bool edge() const { return VEC ? false : edge_; }
};

// The trials of one warp, in its order: t, t + n_warps, ...
template <bool VEC>
struct Trials {
    int64_t stride = 0;  // VEC: ids from trial to trial
    bool bad = false;    // a decreasing pair of offsets, or one too far apart, was seen

    __device__ __forceinline__ Trials(const YetArgs& y, int64_t n_warps) {
        if constexpr (VEC) stride = n_warps * (int64_t)y.k;
    }
    __device__ __forceinline__ Span<VEC> first(const YetArgs& y, int64_t t) {
        Span<VEC> s;
        if (t >= y.n_trials) return s;
        if constexpr (VEC) {
            s.p = y.ids + t * (int64_t)y.k;
            s.n = (uint32_t)y.k;
        } else {
            int64_t b, e;
            bool bo;
            trial_range(y, t, b, e, bo);
            if (e - b > kMaxTrialIds) {
                bo = true;
                e = b;
            }
            bad |= bo;
            // ids between the 16-byte boundary before y.ids and y.ids
            const uint32_t mis = (uint32_t)(reinterpret_cast<uintptr_t>(y.ids) >> 2) & 3u;
            // reads of [lo, hi) stay in the id array (for a CSR every index
            // between the first and the last offset lies in some trial)
            const int64_t lo = y.off ? y.off[0] : 0;
            const int64_t hi = y.off ? y.off[y.n_trials] : y.n_trials * (int64_t)y.k;
            s.head_ = ((uint32_t)b + mis) & 3u;
            const int64_t a = b - s.head_;
            s.p = y.ids + a;
            s.n = e > b ? (uint32_t)(e - a) : 0u;
            s.edge_ = y.by_id || a < lo || a + (int64_t)((s.n + 3u) & ~3u) > hi;
        }
        return s;
    }
    // the span of trial t, whose predecessor in the warp's order is s
    __device__ __forceinline__ Span<VEC> next(const YetArgs& y, const Span<VEC>& s, int64_t t) {
        if constexpr (VEC) {
            Span<VEC> r;
            r.p = s.p + stride;
            r.n = t < y.n_trials ? s.n : 0u;
            return r;
        }
        return first(y, t);
    }
};

// A warp's id stream: chunks of 32 * E positions brought to its buffer in
// shared memory by bulk copies (TMA), one in flight while the chunk before it
// is processed from registers. Loads of the ids through L1 would share its
// in-order return path with the gathers, which then wait for DRAM instead of
// L2.
template <int E>
struct IdStream {
    uint32_t bar, buf;  // shared-memory addresses of the warp's barrier and buffer
    uint32_t phase;

    __device__ __forceinline__ void init(void* bars, void* bufs, int wib, int lane) {
        bar = (uint32_t)__cvta_generic_to_shared(bars) + 8u * wib;
        buf = (uint32_t)__cvta_generic_to_shared(bufs) + 128u * E * wib;
        phase = 0;
        if (lane == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    }
    // Request the chunk from position c0, once every lane has the ids of the
    // chunk before it.
    template <bool VEC>
    __device__ __forceinline__ void request(const Span<VEC>& s, uint32_t c0, int lane) {
        if (lane == 0 && c0 < s.n && !s.edge()) {
            const uint32_t bytes = 4u * min(32u * E, ((s.n + 3u) & ~3u) - c0);
            uint64_t policy;  // evict-first in L2: the stream must not push out X
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(buf),
                "l"(s.p + c0), "r"(bytes), "r"(bar), "l"(policy)
                : "memory");
        }
    }
    __device__ __forceinline__ bool arrived() const {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(phase)
            : "memory");
        return ok != 0;
    }
    // Wait for the requested chunk; false when it has not come in time, for the
    // whole warp: each lane polls and reads the clock by itself, and lanes that
    // disagreed would part before the pass's next vote.
    __device__ __forceinline__ bool wait(uint64_t limit_ns = kWaitNs) {
        bool ok = arrived();
        if (!ok) {
            const uint64_t t0 = now_ns();
            while (!(ok = arrived()) && now_ns() - t0 < limit_ns) {
            }
        }
        phase ^= 1u;
        return __all_sync(kFull, ok);
    }
    // The end of a pass whose wait gave up: the copy in flight may still come,
    // and shared memory stays until then (again with a limit).
    __device__ __forceinline__ void give_up(int* flags, int lane, uint64_t limit_ns = kWaitNs) {
        phase ^= 1u;
        wait(limit_ns);
        if (lane == 0) atomicOr(flags + kFlagTimeout, 1);
    }
    // The ids of the chunk from position c0 of a span with c0 < n: slot
    // 4 h + i of a lane is position c0 + 128 h + 4 lane + i. What positions
    // outside the trial hold is undefined (the caller masks them).
    template <bool VEC>
    __device__ __forceinline__ bool take(const Span<VEC>& s, uint32_t c0, int lane, uint32_t (&v)[E]) {
        bool ok = true;
        if (!s.edge()) {
            ok = wait();
#pragma unroll
            for (int h = 0; h < E / 4; ++h)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(v[4 * h]), "=r"(v[4 * h + 1]), "=r"(v[4 * h + 2]), "=r"(v[4 * h + 3])
                             : "r"(buf + 512u * h + 16u * lane)
                             : "memory");
        } else {
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const uint32_t d = c0 + 128u * (k >> 2) + 4u * lane + (k & 3);
                v[k] = d >= s.head() && d < s.n ? (uint32_t)ld_stream(s.p + d) : 0u;
            }
        }
        return ok;
    }
};

// A chunk's ids as the tests below take them: positions outside the trial and
// ids outside the catalogue become `none`, an id whose bit is clear. max_id
// keeps the largest id of the trial's own. The warp's vote
// needs every id of the chunk in its register, so after it the buffer that
// they came from may be written again (loads from shared memory only issued
// may still read it).
template <int E, bool VEC>
__device__ __forceinline__ void clean_ids(const Span<VEC>& s, uint32_t c0, int lane, uint32_t C, uint32_t none,
                                          uint32_t (&v)[E], uint32_t& max_id) {
    uint32_t m = 0;
    if ((c0 != 0 || s.head() == 0) && c0 + 32u * E <= s.n) {
#pragma unroll
        for (int k = 0; k < E; ++k) m = max(m, v[k]);
    } else if constexpr (VEC) {  // the trial's end: whole vectors are in or out
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const bool live = c0 + 128u * (k >> 2) + 4u * lane < s.n;
            m = max(m, live ? v[k] : 0u);
            v[k] = live ? v[k] : none;
        }
    } else {
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const uint32_t d = c0 + 128u * (k >> 2) + 4u * lane + (k & 3);
            const bool live = d - s.head() < s.n - s.head();
            m = max(m, live ? v[k] : 0u);
            v[k] = live ? v[k] : none;
        }
    }
    if (__any_sync(kFull, m >= C)) {  // some id lies outside the catalogue
        max_id = max(max_id, m);
#pragma unroll
        for (int k = 0; k < E; ++k) v[k] = v[k] < C ? v[k] : none;
    }
}

// The id that stands for no event. Folded, the sentinel C shares its bit with
// an event's; if that one is set, the empty slots of every trial's last chunk
// gather row C, and one hot row slows the whole chip's gathers (c1 with 24
// empty slots per trial: 1.26 against 0.90 ms). So it is an id whose word,
// 2 S - S, is the always-zero word after the bitmap.
template <bool FOLD>
__device__ __forceinline__ uint32_t no_event(uint32_t C, uint32_t S) {
    return FOLD ? 64u * S : C;
}

// The event's bit: word w of shared memory holds bitmap words w and w + S
// OR-ed together (FOLD: a superset test, a fold-only hit gathers zeros).
// Returned as bit 0 of a word (its other bits are other events').
template <bool FOLD>
__device__ __forceinline__ uint32_t bit_of(const uint32_t* s_bits, const uint32_t* gbits, uint32_t id, uint32_t S) {
    uint32_t wi = id >> 5, w;
    if constexpr (FOLD) {
        wi = __viaddmin_u32(wi, 0u - S, wi);  // wi - S wraps when wi < S
        w = s_bits[wi];
    } else {
        w = wi < S ? s_bits[wi] : ld_bits(gbits + wi);
    }
    return __funnelshift_r(w, 0u, id);
}

template <bool FOLD>
__device__ __forceinline__ void stage_bits(uint32_t* s_bits, const uint32_t* gbits, int32_t smem_words, int32_t words) {
    const uint4* src = reinterpret_cast<const uint4*>(gbits);
    uint4* dst = reinterpret_cast<uint4*>(s_bits);
    for (int i = threadIdx.x; i < smem_words / 4; i += blockDim.x) {
        uint4 v = src[i];
        if (FOLD && 4 * i + smem_words < words) {  // the bitmap is zero-padded to whole uint4
            const uint4 u = src[i + smem_words / 4];
            v.x |= u.x;
            v.y |= u.y;
            v.z |= u.z;
            v.w |= u.w;
        }
        dst[i] = v;
    }
    if (threadIdx.x == 0) s_bits[smem_words] = 0u;  // no_event's word
}

// A warp's ring of queued ids in shared memory. Stores are predicated rather
// than branched over (a branch region per slot of 32 events costs the skip
// pass a third of its instructions on the 8-layer groups).
constexpr uint32_t kRing = 128;  // entries: up to 31 left over and two slots of 32

struct IdRing {
    uint32_t base;            // shared-memory address, a multiple of the ring's size
    uint32_t head = 0, tail = 0;  // warp-uniform positions in bytes

    __device__ __forceinline__ explicit IdRing(const uint32_t* ring) : base((uint32_t)__cvta_generic_to_shared(ring)) {}
    // Queue the ids of the lanes whose word has bit 0 set. One block, so that
    // one predicate serves the vote and the store.
    __device__ __forceinline__ void push(uint32_t id, uint32_t word, unsigned lt_mask) {
        asm volatile(
            "{\n.reg .pred p;\n.reg .b32 m, a;\n"
            "and.b32 a, %2, 1;\nsetp.ne.u32 p, a, 0;\n"
            "vote.sync.ballot.b32 m, p, 0xffffffff;\n"
            "and.b32 a, m, %3;\npopc.b32 a, a;\nmad.lo.u32 a, a, 4, %0;\n"
            "and.b32 a, a, %5;\nor.b32 a, a, %4;\n"
            "@p st.shared.u32 [a], %1;\n"
            "popc.b32 m, m;\nmad.lo.u32 %0, m, 4, %0;\n}"
            : "+r"(tail)
            : "r"(id), "r"(word), "r"(lt_mask), "r"(base), "n"(4u * kRing - 1u)
            : "memory");
    }
    __device__ __forceinline__ uint32_t size() const { return (tail - head) / 4u; }
    // The entry `lane` places after the head.
    __device__ __forceinline__ uint32_t peek(int lane) const {
        uint32_t v;
        asm volatile("ld.shared.u32 %0, [%1];"
                     : "=r"(v)
                     : "r"(base | ((head + 4u * lane) & (4u * kRing - 1u)))
                     : "memory");
        return v;
    }
    // 32 entries, one per lane.
    __device__ __forceinline__ uint32_t take32(int lane) {
        __syncwarp();
        const uint32_t v = peek(lane);
        head += 128u;
        return v;
    }
};

}  // namespace

}  // namespace art

// Strip apply: the slot-major last step of the deterministic backward, for arrays that a call touches
// densely (sign off, blocks of up to 128 elements, short last blocks included).
//
// The array is cut into strips of 64 .. 256 slots.  With the blocks sorted by start, those that reach a
// strip are one stretch of the sorted list.  A group of LP lanes (LP = 8, 16, 32 by the block length)
// serves a strip, several groups to a warp: it keeps the strip's sums in shared memory and takes the
// stretch block after block - lane o of the group fetches gradient element o and adds it to slot
// start + o.  Blocks come one after the other, so every slot adds its terms in the canonical order, and
// there is nothing to search and nothing to stage: the keys say where to add.
//   * The gradient loads of eight blocks are in flight together, the next keys are asked for ahead.
//   * The sums start from -0 and a -0 element is made +0 first: x + -0 is x for every x, and -0 remains
//     exactly where nothing was added (the canonical sum starts from +0, adds the same terms, and is never
//     -0).  So an untouched slot is known by its sum.
// No barriers between warps, nothing waits but a warp for its own loads.  Bound by the LSU pipe (shuffles, sums
// in shared memory) and the random gradient reads.
// Measured (B200, us, a CTA per 2048 slots with position-tile and long-walk kernels for often repeated ids
// -> here): 34 M blocks of 16 on 250 M slots 1690 -> 895; Adam on 852 K blocks of 8 from Zipf ids, 540 K slots
// 137 -> 50 (the longest id's chain: 9100 terms); the whole Adam step 257 -> 157.
// Rejected: a lane per four slots with the blocks' rows staged in shared memory and the blocks of each lane
// found by bisection or a scan - 385 .. 518 instructions per strip of 128 against about 200.
//
// A strip reached by very many blocks (an id that the batch repeats hundreds of times) would keep one group
// busy for long; such strips go to strip_hot_kernel, one CTA each: eight warps copy gradient elements
// ahead (cp.async), a warp per 32 slots adds.
// Slots [0, Z-1) also receive the wrapped tails of the array's last blocks: strip_low_slot serves them.
#include "robe_internal.h"
#include "robe_update.cuh"

namespace robe {

namespace {

constexpr uint32_t kStripMinLog2 = 6, kStripMaxLog2 = 8;
constexpr int kStripWarps = 8;
constexpr uint32_t kStripMaxZ = 128;
constexpr int kHotCopiers = 8;            // warps of the hot kernel that copy
constexpr int kHotAdders = 8;             // and that add: 32 slots each
constexpr int kHotWarps = kHotCopiers + kHotAdders;
constexpr uint32_t kHotAhead = 3;         // steps that the copies, and again as many that the keys, are asked for ahead
constexpr uint32_t kHotBufs = kHotAhead + 1;
constexpr uint32_t kHotLeast = 96;        // blocks that make a strip hot, at least (see hot_least)

struct StripArgs {
    MapParams mp;
    const float* grad_out;
    float* target;
    float lr;
    AdamState adam;
    const uint32_t* K;         // sorted block starts
    const uint32_t* V;         // bag*d + c*Z of each: its first gradient element
    const int32_t* status;
    const uint32_t* lo_of;     // [strips + 1]: first sorted position whose block reaches the strip or one beyond
    const uint32_t* hi_of;     // [strips + 1]: first sorted position whose key is in the strip or beyond
    uint32_t strips, log2w;    // strips of 2^log2w slots
    uint32_t n_hot;
    uint32_t low_ctas;         // the first CTAs of strip_hot_kernel, which serve slots [0, Z-1)
    uint32_t* hot_count;       // [0] strips at the front of the list, [1] at its back, [2] taken
    uint32_t* hot_list;
    uint32_t hot_cap;
    int vec_commit;            // target and moments are 16-byte aligned
    uint64_t grad_elems;       // of grad_out (read by the debug build's index checks only)
    uint64_t nb;               // sorted blocks
};

constexpr uint32_t kBoundsGap = 256;  // longer gaps are filled by the whole warp

// lo_of and hi_of for b = 0 .. strips, for many strips: a thread per strip, by a bisection that shares all but its
// last steps with its neighbours', and a gallop back from there for lo_of.  34 M keys, 977 K strips: 58 us
// against 90 of the scan below; 852 K keys, 8437 strips: 12 (a warp per strip, 32 probes at a time: 7)
// against 5.
__global__ void __launch_bounds__(256)
strip_bounds_search_kernel(const uint32_t* K, uint32_t nb, uint32_t* lo_of,
                           uint32_t* hi_of, uint32_t strips, uint32_t log2w, uint32_t reach,
                           const int32_t* status, uint32_t* hot_count) {
    follow_settled();
    if (blockIdx.x == 0 && threadIdx.x < 3) hot_count[threadIdx.x] = 0;  // (for the kernels after this one)
    if (status != nullptr && *status != 0) return;  // after a failed input check K was not written
    const uint32_t b = blockIdx.x * 256 + threadIdx.x;
    if (b > strips) return;
    // first position in [from, to] whose key is at least `least`: the keys before `from` are below it, that of
    // `to` (or what lies past the list) is not
    auto search = [&](uint32_t from, uint32_t to, uint64_t least) {
        while (from < to) {
            const uint32_t mid = from + ((to - from) >> 1);
            if ((uint64_t)K[mid] >= least) to = mid; else from = mid + 1;
        }
        return from;
    };
    const uint64_t first_slot = (uint64_t)b << log2w, least = first_slot > reach ? first_slot - reach : 0;
    const uint32_t hi = search(0, nb, first_slot);
    uint32_t to = hi, step = 1;
    while (to >= step && (uint64_t)K[to - step] >= least) {
        to -= step;
        step <<= 1;  // (the steps add up to less than nb)
    }
    hi_of[b] = hi;
    lo_of[b] = search(to >= step ? to - step + 1 : 0, to, least);
}

// The same for few strips, by reading the list.  A thread takes eight sorted positions; position i begins the strips
// whose first slot lies past the key before it and not past its own (lo_of: the same of the blocks' last slots).
__global__ void __launch_bounds__(256)
strip_bounds_kernel(const uint32_t* K, uint64_t nb, uint32_t* lo_of,
                    uint32_t* hi_of, uint32_t strips, uint32_t log2w, uint32_t reach, const int32_t* status,
                    uint32_t* hot_count) {
    follow_settled();
    if (blockIdx.x == 0 && threadIdx.x < 3) hot_count[threadIdx.x] = 0;  // (for the kernels after this one)
    if (status != nullptr && *status != 0) return;  // after a failed input check K was not written
    const uint64_t i0 = ((uint64_t)blockIdx.x * 256 + threadIdx.x) * 8;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t k[9];  // k[0]: the key before
    if (i0 + 8 <= nb) {
        const uint4 x = reinterpret_cast<const uint4*>(K + i0)[0], y = reinterpret_cast<const uint4*>(K + i0)[1];
        k[1] = x.x; k[2] = x.y; k[3] = x.z; k[4] = x.w;
        k[5] = y.x; k[6] = y.y; k[7] = y.z; k[8] = y.w;
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) k[t + 1] = i0 + t < nb ? K[i0 + t] : 0u;
    }
    k[0] = __shfl_up_sync(0xFFFFFFFFu, k[8], 1);
    if (lane == 0 && i0 > 0 && i0 <= nb) k[0] = K[i0 - 1];
    if (__all_sync(0xFFFFFFFFu, i0 > 0 && i0 + 8 <= nb && ((k[8] + reach) >> log2w) - (k[0] >> log2w) <= kBoundsGap)) {
        // in the middle of the list (most threads): a position begins a strip, or a few, or none
        uint32_t h = k[0] >> log2w, l = (k[0] + reach) >> log2w;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const uint32_t hi = k[t + 1] >> log2w, to = (k[t + 1] + reach) >> log2w;
            while (h != hi) {
                ++h;
                if (ROBE_CHK(h <= strips, ROBE_DBG_WINDOW)) hi_of[h] = (uint32_t)(i0 + t);
            }
            while (l != to) {
                ++l;
                if (l <= strips) lo_of[l] = (uint32_t)(i0 + t);  // (a block may reach past the array's end)
            }
        }
        return;
    }
    bool gap = false;
    // strips from .. to begin at position i0 + t  (reach = Z - 1; key + reach < 2^32)
    auto span = [&](int t, uint32_t past, uint32_t& from, uint32_t& n) {
        const uint64_t i = i0 + t;
        from = i > 0 ? ((k[t] + past) >> log2w) + 1 : 0u;
        uint32_t to = i < nb ? (k[t + 1] + past) >> log2w : strips;
        if (to > strips) to = strips;
        n = i <= nb && to >= from ? to - from + 1 : 0u;
    };
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        uint32_t from, n;
        span(t, 0, from, n);
        if (n > kBoundsGap) gap = true;
        else
            for (uint32_t b = 0; b < n; ++b)
                if (ROBE_CHK(from + b <= strips, ROBE_DBG_WINDOW)) hi_of[from + b] = (uint32_t)(i0 + t);
        span(t, reach, from, n);
        if (n > kBoundsGap) gap = true;
        else
            for (uint32_t b = 0; b < n; ++b)
                if (ROBE_CHK(from + b <= strips, ROBE_DBG_WINDOW)) lo_of[from + b] = (uint32_t)(i0 + t);
    }
    if (!__any_sync(0xFFFFFFFFu, gap)) return;
    for (int t = 0; t < 16; ++t) {
        uint32_t* const of = t < 8 ? hi_of : lo_of;
        uint32_t from = 0, n = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c == (t & 7)) span(c, t < 8 ? 0u : reach, from, n);
        for (uint32_t wide = __ballot_sync(0xFFFFFFFFu, n > kBoundsGap); wide != 0; wide &= wide - 1) {
            const int src = __ffs((int)wide) - 1;
            const uint32_t f = __shfl_sync(0xFFFFFFFFu, from, src), c = __shfl_sync(0xFFFFFFFFu, n, src);
            const uint32_t p = __shfl_sync(0xFFFFFFFFu, (uint32_t)(i0 + (t & 7)), src);
            for (uint32_t b = lane; b < c; b += 32)
                if (ROBE_CHK(f + b <= strips, ROBE_DBG_WINDOW)) of[f + b] = p;
        }
    }
}

// The list of hot strips: the hottest at its front, so that they are begun first.
__global__ void __launch_bounds__(256) strip_hot_list_kernel(StripArgs a) {
    follow<true>();
    if (a.status != nullptr && *a.status != 0) return;
    const uint32_t b = blockIdx.x * 256 + threadIdx.x;
    if (b >= a.strips) return;
    const uint32_t n = a.hi_of[b + 1] - a.lo_of[b];
    if (n <= a.n_hot) return;
    const bool front = n > 4 * a.n_hot;
    const uint32_t at = atomicAdd(a.hot_count + (front ? 0 : 1), 1u);
    if (ROBE_CHK(at < a.hot_cap, ROBE_DBG_LONG_WALK)) a.hot_list[front ? at : a.hot_cap - 1 - at] = b;
}

// elements of the block with payload v
template <bool SHORT>
__device__ __forceinline__ uint32_t strip_len(const MapParams& mp, uint32_t v) {
    if (!SHORT) return mp.Z;
    const uint32_t left = mp.d - v % mp.d;
    return left < mp.Z ? left : mp.Z;
}

__device__ __forceinline__ bool strip_touched(float sum) { return __float_as_uint(sum) != 0x80000000u; }

// blocks that a copying warp of the hot kernel takes at a time, by the elements per lane of a block
__host__ __device__ constexpr uint32_t hot_blocks(int epl) { return epl == 1 ? 32u : (epl == 2 ? 16u : 8u); }

template <int MODE, int LP, int EPL, bool SHORT, bool BANKED>
__global__ void __launch_bounds__(32 * kStripWarps, 5)
strip_apply_kernel(StripArgs a) {
    extern __shared__ float4 strip_smem[];
    follow();  // (after strip_bounds_*, which are settled: sorted blocks and gradients are read-only here)
    if (a.status != nullptr && *a.status != 0) return;
    constexpr uint32_t G = 32 / LP;               // groups per warp
    constexpr int U = EPL == 4 ? 4 : 8;           // blocks whose loads are in flight together
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t g = lane / LP, ol = lane % LP;
    const uint32_t b = (blockIdx.x * kStripWarps + w) * G + g;
    const uint32_t Z = a.mp.Z, W = 1u << a.log2w;
    // BANKED: groups whose strips' sums lie one after the other would meet in the same banks.  Slot s of group g's
    // strip lies at place(s) of the warp's sums, every group having LP banks to itself; past the sums there is a
    // place in the same bank for slots that are not the strip's.
    const uint32_t sums_at = BANKED ? w * (G * W + 32) : (w * G + g) * W;
    volatile float* const sum = reinterpret_cast<float*>(strip_smem) + sums_at;
    auto place = [&](uint32_t s) {
        const uint32_t row = s & ~(LP - 1u);
        return (row < W ? row : W) * G + (s & (LP - 1u)) + g * LP;
    };
    uint32_t lo = 0, n = 0;
    if (b < a.strips) {
        lo = a.lo_of[b];
        n = a.hi_of[b + 1] - lo;
        if (n > a.n_hot) n = 0;  // the hot kernel's
    }
    const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, n);
    if (most == 0) return;
    const uint32_t w0 = b << a.log2w;
    if (n != 0 && ol < W / 32 && (uint64_t)w0 + 32 * ol < a.mp.m)  // wanted at the end: the lines of the target
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.target + w0 + 32 * ol));
    for (uint32_t i = BANKED ? lane : ol; i < (BANKED ? G * W / 4 : W / 4); i += BANKED ? 32 : LP)
        strip_smem[(sums_at >> 2) + i] = make_float4(-0.0f, -0.0f, -0.0f, -0.0f);
    // lane ol holds block ol of the present LP: start relative to the strip, payload
    uint32_t nk = 0, nv = 0;
    if (ol < n && ROBE_CHK((uint64_t)lo + ol < a.nb, ROBE_DBG_SORT_POS)) {
        nk = load_settled(a.K + lo + ol);
        nv = load_settled(a.V + lo + ol);
    }
    __syncwarp();
    for (uint32_t c0 = 0; c0 < most; c0 += LP) {
        // a block past the stretch starts beyond every strip
        const uint32_t rel = c0 + ol < n ? nk - w0 : 0x40000000u, v = nv;
        const uint32_t len = SHORT ? strip_len<SHORT>(a.mp, v) : 0u;
        if (c0 + LP + ol < n && ROBE_CHK((uint64_t)lo + c0 + LP + ol < a.nb, ROBE_DBG_SORT_POS)) {
            nk = load_settled(a.K + lo + c0 + LP + ol);
            nv = load_settled(a.V + lo + c0 + LP + ol);
        }
#pragma unroll 1
        for (uint32_t u0 = 0; u0 < LP && c0 + u0 < most; u0 += U) {
            float x[U][EPL];
            uint32_t slot[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int src = (int)(g * LP + u0 + u);
                const uint32_t r = __shfl_sync(0xFFFFFFFFu, rel, src), p = __shfl_sync(0xFFFFFFFFu, v, src) + ol;
                const uint32_t l = SHORT ? __shfl_sync(0xFFFFFFFFu, len, src) : Z;
                slot[u] = r + ol;  // (below the strip: wraps to a large number)
#pragma unroll
                for (int q = 0; q < EPL; ++q) {
                    x[u][q] = -0.0f;
                    if (slot[u] + 32 * q < W && ol + 32 * q < l &&
                        ROBE_CHK((uint64_t)p + 32 * q < a.grad_elems, ROBE_DBG_GRAD_POS))
                        x[u][q] = load_settled(a.grad_out + (p + 32 * q)) + 0.0f;  // -0 -> +0
                }
                if constexpr (BANKED) slot[u] = place(slot[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int q = 0; q < EPL; ++q) {
                    // (a lane past the block's end adds -0 to a slot that is no other lane's in this step)
                    const uint32_t s = slot[u] + 32 * q;
                    if (BANKED ? ROBE_CHK(s < G * W + 32, ROBE_DBG_SHARED) : s < W) sum[s] = __fadd_rn(sum[s], x[u][q]);
                }
                __syncwarp();
            }
        }
    }
    if (n == 0) return;
    const bool inner = a.vec_commit && w0 + 1 >= Z && (uint64_t)w0 + W <= a.mp.m;
    const float4* const sum4 = strip_smem + (sums_at >> 2);
    for (uint32_t i = ol; i < W / 4; i += LP) {
        const float4 s = sum4[BANKED ? place(4 * i) >> 2 : i];
        const bool t0 = strip_touched(s.x), t1 = strip_touched(s.y), t2 = strip_touched(s.z), t3 = strip_touched(s.w);
        const uint32_t j = w0 + 4 * i;
        if (!(t0 || t1 || t2 || t3)) continue;
        if (inner) {  // all of the strip inside the array and above the low slots, vectors aligned
            if (!ROBE_CHK((uint64_t)j + 3 < a.mp.m, ROBE_DBG_ARRAY_SLOT)) continue;
            float4 old = *reinterpret_cast<const float4*>(a.target + j), m1 = make_float4(0, 0, 0, 0), m2 = m1;
            if (MODE == 2) m1 = *reinterpret_cast<const float4*>(a.adam.m1 + j);
            if (MODE >= 2) m2 = *reinterpret_cast<const float4*>(a.adam.m2 + j);
            if (t0) old.x = slot_step<MODE>(a.adam, a.lr, s.x, old.x, m1.x, m2.x);
            if (t1) old.y = slot_step<MODE>(a.adam, a.lr, s.y, old.y, m1.y, m2.y);
            if (t2) old.z = slot_step<MODE>(a.adam, a.lr, s.z, old.z, m1.z, m2.z);
            if (t3) old.w = slot_step<MODE>(a.adam, a.lr, s.w, old.w, m1.w, m2.w);
            *reinterpret_cast<float4*>(a.target + j) = old;
            if (MODE == 2) *reinterpret_cast<float4*>(a.adam.m1 + j) = m1;
            if (MODE >= 2) *reinterpret_cast<float4*>(a.adam.m2 + j) = m2;
            continue;
        }
        const float one[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            if (strip_touched(one[q]) && (uint64_t)j + q < a.mp.m && j + q + 1 >= Z)
                commit_slot<MODE>(a, j + q, one[q], a.target[j + q]);
    }
}

__device__ __forceinline__ float lds1(uint32_t at) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at));
    return v;
}
__device__ __forceinline__ float4 lds4(uint32_t at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at));
    return v;
}
__device__ __forceinline__ float add4(float acc, const float4 x) {
    return __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, x.x), x.y), x.z), x.w);
}

// acc + one slot's terms of n blocks side by side at `at`, n a multiple of eight; the reads of eight run ahead
// of the adds of the eight before
__device__ __forceinline__ float hot_add_chunk(float acc, uint32_t at, uint32_t n) {
    float4 x = lds4(at), y = lds4(at + 16);
#pragma unroll 4
    for (uint32_t e = 8; e < n; e += 8) {
        at += 32;
        const float4 x1 = lds4(at), y1 = lds4(at + 16);
        acc = add4(add4(acc, x), y);
        x = x1;
        y = y1;
    }
    return add4(add4(acc, x), y);
}

// The same for `pairs` times two lots of 16 blocks, the second `odd` bytes after the first, the next pair `step`
// bytes on: 16 reads ahead and nothing else inside (the chain of adds is what this loop should wait for).
__device__ __forceinline__ float hot_add_step(float acc, uint32_t at, uint32_t pairs, uint32_t odd, uint32_t step) {
    float4 x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = lds4(at + 16 * u);
#pragma unroll 2
    for (uint32_t c = 0; c < pairs; ++c) {
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = lds4(at + odd + 16 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = add4(acc, x[u]);
        if (c + 1 < pairs) at += step;  // (else the last lot again, not used)
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = lds4(at + 16 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = add4(acc, y[u]);
    }
    return acc;
}

// First sorted position whose key is at least `least`: 32 probes at a time by a warp.
__device__ __forceinline__ uint64_t strip_first(const StripArgs& a, uint64_t least, uint32_t lane) {
    uint64_t from = 0, to = a.nb;  // keys before `from` are below, those from `to` on are not
    while (from < to) {
        const uint64_t step = (to - from + 31) / 32, at = from + step * lane;
        const uint32_t not_below = __ballot_sync(0xFFFFFFFFu, at >= to || (uint64_t)__ldca(a.K + at) >= least);
        const uint32_t f = not_below != 0 ? (uint32_t)__ffs((int)not_below) - 1 : 32u;
        if (f == 0) return from;
        const uint64_t next = from + step * f;
        from += step * (f - 1) + 1;
        if (next < to) to = next;
    }
    return from;
}

// Slot j in [0, Z-1), by a warp: the blocks that begin at or before it, then the wrapped tails of those that
// begin in the last Z-1-j slots; the terms of 32 sorted positions at a time, all lanes adding them in order.
template <int MODE, bool SHORT>
__device__ __forceinline__ void strip_low_slot(const StripArgs& a, uint32_t j, uint32_t lane) {
    float acc = 0.0f;
    bool touched = false;
    auto walk = [&](uint64_t from, uint64_t to, uint64_t j_plus) {
        for (uint64_t i0 = from; i0 < to; i0 += 32) {
            const uint64_t i = i0 + lane;
            float term = 0.0f;
            bool ok = false;
            if (i < to && ROBE_CHK(i < a.nb, ROBE_DBG_SORT_POS)) {
                const uint32_t v = __ldca(a.V + i), o = (uint32_t)(j_plus - __ldca(a.K + i));
                ok = o < strip_len<SHORT>(a.mp, v) && ROBE_CHK((uint64_t)v + o < a.grad_elems, ROBE_DBG_GRAD_POS);
                if (ok) term = __ldca(a.grad_out + (uint64_t)v + o);
            }
            const uint32_t oks = __ballot_sync(0xFFFFFFFFu, ok);
            touched = touched || oks != 0;
            for (uint32_t rest = oks; rest != 0; rest &= rest - 1)
                acc = __fadd_rn(acc, __shfl_sync(0xFFFFFFFFu, term, __ffs((int)rest) - 1));
        }
    };
    walk(0, strip_first(a, (uint64_t)j + 1, lane), j);
    walk(strip_first(a, (uint64_t)a.mp.m - (a.mp.Z - 1) + j, lane), a.nb, (uint64_t)j + a.mp.m);  // (m >= Z)
    if (touched && lane == 0) commit_slot<MODE>(a, j, acc, a.target[j]);
}

// Hot strips.  The chain of dependent adds of a slot is the definition's, and one warp's issue is what it
// costs beyond that: the copies are laid out slot by slot, so that a lane reads four blocks' terms at once,
// and a whole step of repeats of one start is one loop.  One barrier per step of eight copiers' blocks,
// whose copies were issued three steps ahead.
// Measured (B200, ns per repeat of one start): 9.3 with a row per block, 4.1 with divisions and a pass over all
// blocks in the copiers, 3.7 here (of a step, 1308 clocks are adds, 330 what stands before them); the chain itself: 2.1.
template <int MODE, int LP, int EPL, bool SHORT>
__global__ void __launch_bounds__(32 * kHotWarps, 2)
strip_hot_kernel(StripArgs a) {
    extern __shared__ float4 strip_smem[];
    __shared__ int2 ent_s[kHotBufs][kHotCopiers][32];  // (start relative to the strip, length) of each block
    __shared__ int4 all_s[kHotBufs][kHotCopiers];      // of the blocks of one copier: their number; all alike? start, length
    __shared__ uint2 keys_s[2 * kHotBufs][kHotCopiers][32];  // (start, payload) of steps yet to be copied
    __shared__ uint32_t item_s;
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (blockIdx.x < a.low_ctas) {  // (in a kernel of their own after this one: Adam on 852 K blocks 125 us against 116)
        const uint32_t j = blockIdx.x * kHotWarps + w;
        if (j + 1 < a.mp.Z) strip_low_slot<MODE, SHORT>(a, j, lane);
        return;
    }
    const bool copier = w >= (uint32_t)kHotAdders;
    const uint32_t cw = w - kHotAdders;
    const uint32_t Z = a.mp.Z, W = 1u << a.log2w;
    constexpr uint32_t E = hot_blocks(EPL), per_step = E * kHotCopiers;
    const uint32_t n_front = a.hot_count[0], n_items = n_front + a.hot_count[1];
    float* const stage = reinterpret_cast<float*>(strip_smem);
    constexpr uint32_t pitch = E + 4;  // element o of block e at o * pitch + e
    const uint32_t chunk = pitch * Z;
    for (;;) {
        __syncthreads();  // item_s and the buffers are free
        if (threadIdx.x == 0) item_s = atomicAdd(a.hot_count + 2, 1u);
        __syncthreads();
        const uint32_t item = item_s;
        if (item >= n_items) break;
        const uint32_t b = a.hot_list[item < n_front ? item : a.hot_cap - 1 - (item - n_front)];
        const uint32_t w0 = b << a.log2w;
        const uint32_t lo = a.lo_of[b], n = a.hi_of[b + 1] - lo;
        const uint32_t steps = (n + per_step - 1) / per_step;
        // blocks of this copier in step s: positions from lo + s*per_step + cw*E, this many
        const uint32_t share = n > cw * E ? n - cw * E : 0u;
        auto count = [&](uint32_t s) -> uint32_t {
            const uint32_t before = s * per_step;  // (the steps asked about end at most six past the last)
            return before >= share ? 0u : (share - before < E ? share - before : E);
        };
        // The keys of this lane's block of step s, and the elements of the blocks of step s: one group of copies
        // per step has the elements kHotAhead steps ahead of what is added and the keys as much again ahead.
        auto fetch = [&](uint32_t s) {
            if (lane < count(s)) {
                const uint32_t at = lo + s * per_step + cw * E + lane;
                if (!ROBE_CHK((uint64_t)at < a.nb, ROBE_DBG_SORT_POS)) return;
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&keys_s[s % (2 * kHotBufs)][cw][lane]);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(a.K + at) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4), "l"(a.V + at) : "memory");
            }
        };
        auto copy = [&](uint32_t s) {
            const uint2 kv = keys_s[s % (2 * kHotBufs)][cw][lane];
            const uint32_t k = kv.x, v = kv.y;
            const uint32_t ne = count(s);
            float* const rows = stage + ((s % kHotBufs) * kHotCopiers + cw) * chunk;
            const int rel = (int)(k - w0);
            const int len = (int)(lane < ne ? strip_len<SHORT>(a.mp, v) : 0u);
            ent_s[s % kHotBufs][cw][lane] = make_int2(rel, len);
            const int rel0 = __shfl_sync(0xFFFFFFFFu, rel, 0), len0 = __shfl_sync(0xFFFFFFFFu, len, 0);
            const bool alike = __all_sync(0xFFFFFFFFu, lane >= ne || (rel == rel0 && len == len0));
            if (lane == 0) all_s[s % kHotBufs][cw] = make_int4((int)ne, alike ? 1 : 0, rel0, len0);
            // lane: element lane % LP (+ 32, ..) of every (32 / LP)-th block
            constexpr uint32_t G = 32 / LP;
            const uint32_t o0 = lane % LP, e0 = lane / LP;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(rows + o0 * pitch + e0);
            if (alike && ne == E) {  // the same elements of every block are wanted
                bool on[EPL];
#pragma unroll
                for (int i = 0; i < EPL; ++i)
                    on[i] = o0 + 32 * i < (uint32_t)len0 && (uint32_t)rel0 + o0 + 32 * i < W;
#pragma unroll
                for (uint32_t q = 0; q < E / G; ++q) {
                    const uint32_t p = __shfl_sync(0xFFFFFFFFu, v, e0 + q * G) + o0;
#pragma unroll
                    for (int i = 0; i < EPL; ++i)
                        if (on[i] && ROBE_CHK((uint64_t)p + 32 * i < a.grad_elems, ROBE_DBG_GRAD_POS))
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * (q * G + 32 * i * pitch)),
                                         "l"(a.grad_out + (p + 32 * i))
                                         : "memory");
                }
            } else {
#pragma unroll 4
                for (uint32_t q = 0; q < E / G; ++q) {
                    if (q * G >= ne) break;  // (warp-uniform)
                    const uint32_t e = e0 + q * G;
                    const uint32_t r = __shfl_sync(0xFFFFFFFFu, (uint32_t)rel, e), p = __shfl_sync(0xFFFFFFFFu, v, e) + o0;
                    const uint32_t l = (uint32_t)__shfl_sync(0xFFFFFFFFu, len, e);  // (0 past the last block)
#pragma unroll
                    for (int i = 0; i < EPL; ++i)
                        if (o0 + 32 * i < l && r + o0 + 32 * i < W &&
                            ROBE_CHK((uint64_t)p + 32 * i < a.grad_elems, ROBE_DBG_GRAD_POS))
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * (q * G + 32 * i * pitch)),
                                         "l"(a.grad_out + (p + 32 * i))
                                         : "memory");
                }
            }
        };
        auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
        if (copier) {
            for (uint32_t s = 0; s < kHotAhead; ++s) fetch(s);
            commit();
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            for (uint32_t s = 0; s < kHotAhead; ++s) {
                if (s < steps) copy(s);
                fetch(s + kHotAhead);
                commit();
            }
        }
        const int slot = (int)(32 * w + lane);  // adders: within the strip
        float acc = -0.0f;
        for (uint32_t s = 0; s < steps; ++s) {
            // (the group of step s has the elements of step s and the keys of step s + kHotAhead)
            if (copier) asm volatile("cp.async.wait_group %0;" ::"n"(kHotAhead - 1) : "memory");
            __syncthreads();  // step s is in; step s - 1 has been added
            if (copier) {
                if (s + kHotAhead < steps) copy(s + kHotAhead);
                fetch(s + 2 * kHotAhead);
                commit();
                continue;
            }
            if (32 * w >= W) continue;
            const uint32_t stage_at = (uint32_t)__cvta_generic_to_shared(stage + (s % kHotBufs) * kHotCopiers * chunk);
            const int4 lead = all_s[s % kHotBufs][0], its = all_s[s % kHotBufs][lane % kHotCopiers];
            if (__all_sync(0xFFFFFFFFu, its.x == (int)E && its.y != 0 && its.z == lead.z && its.w == lead.w)) {
                // a whole step of repeats (-0 turns +0 at the first term: see strip_apply_kernel)
                const uint32_t d = (uint32_t)(slot - lead.z);
                if (d < (uint32_t)lead.w) {
                    const uint32_t at = stage_at + 4 * pitch * d;
                    acc += 0.0f;
                    if (E == 32) acc = hot_add_step(acc, at, kHotCopiers, 64, 4 * chunk);
                    else if (E == 16) acc = hot_add_step(acc, at, kHotCopiers / 2, 4 * chunk, 8 * chunk);
                    else
                        for (uint32_t c = 0; c < (uint32_t)kHotCopiers; ++c) acc = hot_add_chunk(acc, at + 4 * chunk * c, E);
                }
                continue;
            }
            for (uint32_t c = 0; c < (uint32_t)kHotCopiers; ++c) {
                const int4 all = all_s[s % kHotBufs][c];
                const uint32_t ne = (uint32_t)all.x;
                if (ne == 0) break;
                const uint32_t rows_at = stage_at + 4 * chunk * c;
                if (all.y) {  // every block covers the same slots
                    const uint32_t d = (uint32_t)(slot - all.z);
                    if (d < (uint32_t)all.w) {
                        acc += 0.0f;
                        const uint32_t at = rows_at + 4 * pitch * d;
                        if (ne >= 8) acc = hot_add_chunk(acc, at, ne & ~7u);
                        for (uint32_t e = ne & ~7u; e < ne; ++e) acc = __fadd_rn(acc, lds1(at + 4 * e));
                    }
                    __syncwarp();
                    continue;
                }
                // (-0 for a block that does not reach the slot, +0 for a term -0)
                const int2 mine = ent_s[s % kHotBufs][c][lane];
                for (uint32_t e0 = 0; e0 < ne; e0 += 8) {
                    float x[8];
#pragma unroll
                    for (uint32_t u = 0; u < 8; ++u) {
                        const uint32_t d = (uint32_t)(slot - __shfl_sync(0xFFFFFFFFu, mine.x, e0 + u));
                        const uint32_t l = (uint32_t)__shfl_sync(0xFFFFFFFFu, mine.y, e0 + u);  // (0 past the last block)
                        x[u] = -0.0f;
                        if (d < l) x[u] = lds1(rows_at + 4 * (d * pitch + e0 + u)) + 0.0f;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc = __fadd_rn(acc, x[u]);
                }
            }
        }
        if (copier) asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (!copier && strip_touched(acc)) {
            const uint64_t j = (uint64_t)w0 + (uint32_t)slot;
            if (j < a.mp.m && j + 1 >= Z) commit_slot<MODE>(a, (uint32_t)j, acc, a.target[j]);
        }
    }
}

inline size_t align_256(size_t v) { return (v + 255) & ~(size_t)255; }

struct StripLayout {
    size_t lo_of, hi_of, total;
    uint32_t strips, log2w;
};

StripLayout strip_layout(uint32_t m) {
    StripLayout L;
    // Long strips (fewer blocks that reach two of them), unless that leaves warps without work
    L.log2w = kStripMaxLog2;
    while (L.log2w > kStripMinLog2 && (m >> L.log2w) < 148u * 64u) --L.log2w;
    L.strips = ((m - 1) >> L.log2w) + 1;
    L.lo_of = 256;  // the counters come first
    L.hi_of = L.lo_of + align_256(((size_t)L.strips + 1) * sizeof(uint32_t));
    L.total = L.hi_of + align_256(((size_t)L.strips + 1) * sizeof(uint32_t));
    return L;
}

// A strip is hot from this many blocks on, at least: 256 in large calls, fewer in small ones, whose last strips'
// chains are what the call waits for (us, floor 256 / 192 / 128 / 96: Adam on 52 K blocks of 8, 540 K slots 63.4 /
// 60.5 / 56.0 / 54.0; on 52 K of 128, 1 M slots 135 / 122 / 109 / 101; 416 K of 16, 1 M 107 / 103 / 99 / 99; but 852 K
// of 8, 3.9 M 122 / 125 / 129 / 131, and 34 M of 16 from Zipf ids, 250 M 2941 / 2978 / 3080 / 3199).
uint64_t hot_least(uint64_t nb) { return nb / 3072 < kHotLeast ? kHotLeast : (nb / 3072 > 256 ? 256 : nb / 3072); }

// Entries of the hot strips' list.  (A block of up to 128 elements reaches at most three strips.)
uint32_t hot_list_cap(uint64_t nb, uint32_t strips) {
    const uint64_t cap = 3 * nb / hot_least(nb) + 1;
    return (uint32_t)(cap < strips ? cap : strips);
}

size_t hot_smem_bytes(uint32_t Z, int epl) { return (size_t)kHotBufs * kHotCopiers * (hot_blocks(epl) + 4) * Z * sizeof(float); }

// CTAs of the hot kernel that run at a time
uint32_t hot_ctas(size_t hot_smem) {
    const uint32_t per_sm = (uint32_t)(220 * 1024 / (hot_smem + 26 * 1024));  // (26 KB: the static part and a margin)
    return 148 * (per_sm > 2 ? 2 : (per_sm < 1 ? 1 : per_sm));
}

template <int MODE, int LP, int EPL, bool SHORT>
void launch_strip_kernels(const StripArgs& a, cudaStream_t st, cudaStream_t hot_st) {
    const size_t hot_smem = hot_smem_bytes(a.mp.Z, EPL);
    if (hot_smem > 23 * 1024)  // (with the static part above the default limit)
        cudaFuncSetAttribute(strip_hot_kernel<MODE, LP, EPL, SHORT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hot_smem);
    uint32_t hot_grid = hot_ctas(hot_smem);
    if (hot_grid > a.hot_cap) hot_grid = a.hot_cap;
    launch_next(strip_hot_kernel<MODE, LP, EPL, SHORT>, a.low_ctas + hot_grid, 32 * kHotWarps, hot_smem, hot_st, a);
    const uint32_t per_cta = kStripWarps * (32 / LP);
    const unsigned grid = (a.strips + per_cta - 1) / per_cta;
    const size_t smem = ((size_t)per_cta << a.log2w) * sizeof(float);
    // Banks of their own for the lane groups of a warp, for up to seven registers more and no more shared-memory conflicts
    // (LSU pipe 92 % busy with them).  Measured (B200, us per step):
    //   four groups of full blocks gain on any array: 68 M blocks of 8 on 250 M slots 5454 -> 4912, on 10 M 4017 -> 3267;
    //   four with short last blocks only in the optimizers' steps, on arrays of L2 size (Adam on 300 K slots 0.92 .. 0.98);
    //     SGD on 4 M blocks of 8, 8 and 4, 300 K slots 494 -> 565, on 4 M 281 -> 297, on 30 M 368 -> 397;
    //   two with short last blocks there too: 15 M of 16 and a short one on 4 M 853 -> 817, 4 M on 300 K 421 -> 404;
    //   two of full blocks pay with six CTAs to an SM instead of eight (39 registers, 32 before): only in the SGD step, where
    //     rows come from L2 and fewer CTAs at a time are not a wave more of a wave or two.  34 M blocks of 16 on 4 M (977 CTAs)
    //     1805 -> 1893, from Zipf ids 2044 -> 2564, on 10 M 1723 -> 1643, 2140 -> 2118, on 20 M 1740 -> 1700, on 48 M 1728 -> 1747;
    //     1.2 M on 540 K slots (528 CTAs) 141 -> 129, on 2 M (977) 130 -> 141; 8 M on 7 M (1709) 499 -> 475; Adam 1.00 .. 1.05.
    if constexpr (LP < 32 && (LP == 8 ? !SHORT || MODE >= 2 : SHORT || MODE < 2)) {
        const uint64_t bytes = (uint64_t)a.mp.m * sizeof(float);
        auto waves = [&](unsigned per_sm) { return (grid + 148 * per_sm - 1) / (148 * per_sm); };
        const bool banked = SHORT ? bytes <= kL2SizedBytes
                                  : LP == 8 || (bytes <= (128ull << 20) && (waves(6) <= waves(8) || grid > 2 * 8 * 148));
        if (banked) {
            launch_next(strip_apply_kernel<MODE, LP, EPL, SHORT, true>, grid, 32 * kStripWarps, smem + kStripWarps * 32 * sizeof(float), st, a);
            return;
        }
    }
    if constexpr (LP > 8 || SHORT) launch_next(strip_apply_kernel<MODE, LP, EPL, SHORT, false>, grid, 32 * kStripWarps, smem, st, a);
}

template <int MODE, bool SHORT>
void launch_strip_lanes(const StripArgs& a, cudaStream_t st, cudaStream_t hot_st) {
    if (a.mp.Z <= 8) launch_strip_kernels<MODE, 8, 1, SHORT>(a, st, hot_st);
    else if (a.mp.Z <= 16) launch_strip_kernels<MODE, 16, 1, SHORT>(a, st, hot_st);
    else if (a.mp.Z <= 32) launch_strip_kernels<MODE, 32, 1, SHORT>(a, st, hot_st);
    else if (a.mp.Z <= 64) launch_strip_kernels<MODE, 32, 2, SHORT>(a, st, hot_st);
    else launch_strip_kernels<MODE, 32, 4, SHORT>(a, st, hot_st);
}

template <int MODE>
void launch_strip_mode(const StripArgs& a, cudaStream_t st, cudaStream_t hot_st) {
    if (a.mp.d % a.mp.Z != 0) launch_strip_lanes<MODE, true>(a, st, hot_st);
    else launch_strip_lanes<MODE, false>(a, st, hot_st);
}

StripArgs strip_args(const StripProblem& sp) {
    const MapParams& mp = sp.mp;
    const StripLayout L = strip_layout(mp.m);
    char* ws = (char*)sp.workspace;
    auto aligned = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
    StripArgs a{};
    a.mp = mp;
    a.grad_out = sp.grad_out;
    a.target = sp.target;
    a.lr = sp.lr;
    a.adam = sp.adam;
    a.K = sp.K;
    a.V = sp.V;
    a.status = sp.status;
    a.lo_of = (const uint32_t*)(ws + L.lo_of);
    a.hi_of = (const uint32_t*)(ws + L.hi_of);
    a.strips = L.strips;
    a.log2w = L.log2w;
    a.hot_count = (uint32_t*)ws;
    a.hot_list = sp.hot_list;
    a.vec_commit = aligned(sp.target) && aligned(sp.adam.m1) && aligned(sp.adam.m2);
    a.grad_elems = sp.grad_elems;
    a.low_ctas = (mp.Z - 1 + kHotWarps - 1) / kHotWarps;
    a.nb = sp.nb;
    // hot: twice the average number of blocks, and enough of them to be worth a CTA (26 x 16384 Zipf rows on
    // 540 K slots, twice / four times: 34 / 53 us beside the hot kernel's 50)
    const uint64_t mean = (uint64_t)((double)((1u << L.log2w) + mp.Z) * (double)sp.nb / mp.m) + 1;
    // A short array has so few strips, each reached by so many blocks, that a group of lanes to a strip leaves most
    // of the chip idle.  `gain` sets the two costs in clocks against each other: 137 a block (and element of a lane) in
    // strip_apply_kernel, all strips at a time, and 7700 + 8 a block in the hot kernel, strips over its CTAs.  Spread ids
    // reach every strip alike, repeated ones leave the apply kernel with strips just below `hot`.  So from a gain of 2.25 (1.75
    // with many blocks to a strip, or long ones) on every strip above the floor is hot, and from 1 on those a tenth
    // above the average: spread ids have few of them.  Measured (B200, us per Adam step on 60 K slots, 300 K blocks of 16, a
    // gain of 1.6; hot from twice the average / 1.1 times it / the floor): spread ids 75.1 / 74.3 / 92.8, Zipf ids 98.4 /
    // 74.1 / 82.7.  Over 360 shapes of Z = 2 .. 128, relative to twice the average: between the two lines spread 1 / 0.99 / 1.22,
    // Zipf 1 / 0.74 / 0.75; beyond, up to a gain of 5, spread 1 / 1.00 / 0.88, Zipf 1 / 0.65 / 0.49.
    const int epl = mp.Z <= 32 ? 1 : (mp.Z <= 64 ? 2 : 4);
    const double gain = 137.0 * epl * mean * hot_ctas(hot_smem_bytes(mp.Z, epl)) / (L.strips * (7700.0 + 8.0 * mean));
    const uint64_t least = hot_least(sp.nb), above = gain >= (epl > 1 || mean >= 1000 ? 1.75 : 2.25) ? 0 : (gain >= 1 ? mean + mean / 10 : 2 * mean);
    const uint64_t hot = above > least ? above : least;
    a.hot_cap = hot_list_cap(sp.nb, L.strips);
    a.n_hot = (uint32_t)(hot < 0x20000000ull ? hot : 0x20000000ull);
    return a;
}

}  // namespace

// Strips pay when most slots are reached, so that walking every strip is no waste.  (Positions advance by up
// to a few hundred in 32 bits: nb stays a little below 2^32.)
bool strips_ok(const MapParams& mp, uint64_t nb, bool sign) {
    return !sign && mp.Z <= kStripMaxZ && nb != 0 && nb < 0xFFFFF000ull && nb * mp.Z * 2 >= mp.m;
}

size_t strips_workspace_bytes(const MapParams& mp) { return strip_layout(mp.m).total; }

size_t strips_list_bytes(const MapParams& mp, uint64_t nb) {
    return (size_t)hot_list_cap(nb, strip_layout(mp.m).strips) * sizeof(uint32_t);
}

void launch_strips_prepare(const StripProblem& sp, cudaStream_t st) {
    const StripLayout L = strip_layout(sp.mp.m);
    char* ws = (char*)sp.workspace;
    uint32_t *lo_of = (uint32_t*)(ws + L.lo_of), *hi_of = (uint32_t*)(ws + L.hi_of);
    if (L.strips > 148u * 256u)
        launch_next(strip_bounds_search_kernel, L.strips / 256 + 1, 256, 0, st, sp.K, (uint32_t)sp.nb, lo_of, hi_of, L.strips,
                    L.log2w, sp.mp.Z - 1, sp.status, (uint32_t*)ws);
    else
        launch_next(strip_bounds_kernel, (unsigned)(sp.nb / 2048 + 1), 256, 0, st, sp.K, sp.nb, lo_of, hi_of, L.strips,
                    L.log2w, sp.mp.Z - 1, sp.status, (uint32_t*)ws);
}

void launch_strips(const StripProblem& sp, int mode, cudaStream_t st, cudaStream_t hot_st) {
    const StripArgs a = strip_args(sp);
    launch_next(strip_hot_list_kernel, (a.strips + 255) / 256, 256, 0, hot_st, a);
    if (mode == 4) launch_strip_mode<3>(a, st, hot_st);
    else if (mode == 2) launch_strip_mode<2>(a, st, hot_st);
    else if (mode == 1) launch_strip_mode<1>(a, st, hot_st);
    else launch_strip_mode<0>(a, st, hot_st);
}

}  // namespace robe

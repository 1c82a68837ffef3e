// Deterministic backward (Section 3.1 backward equation, evaluated in a fixed order).
//
// Blocks are numbered q = p*C + c in input order (p = position in indices, c = chunk).
//   1. key kernel      key[q] = h(e, x_p, c); val[q] = where the block's gradient elements
//                      start in grad_out (sign off) or q itself (sign on); or both left by the
//                      forward of the same step
//   2. radix sort      stable LSD sort of (key, val) by key - our own passes: digit count per
//                      CTA range, per-digit exclusive scan, ranked scatter through shared
//                      memory (so that every digit's run leaves the CTA as one coalesced piece)
//   3. apply kernel    one thread per touched array slot j sums, left to right in fp32 from +0,
//                      the terms of the sorted blocks whose key lies in [j-Z+1, j], then performs
//                      ONE add (dense gradient) or ONE fma (SGD) on slot j.  The thread that owns
//                      slot j is the one at the first sorted block of that key window, so it only
//                      ever walks forward through the sorted list.  Slots [0, Z-1), which also
//                      receive the wrapped tails of blocks near the end of the array, are handled
//                      by a small second kernel (those terms come last: their keys are the largest), with the
//                      strips below by the first CTAs of the hot strips' kernel.
//                      Walks over hundreds of blocks (an id repeated many times in the batch)
//                      are finished by a third kernel that keeps a whole step of terms in flight.
//                      Arrays that the call touches densely are served slot by slot instead
//                      (robe_strips.cu), in the same order.
// No atomics on floating-point data and no waits between CTAs: the result is bit-reproducible.
#include "robe_internal.h"
#include "robe_update.cuh"

namespace robe {

namespace {

constexpr int kSortThreads = 512;                       // of the count and scatter kernels
constexpr int kSortWarps = kSortThreads / 32;
// Keys per thread and tile: 8, or 4 where that leaves the busiest SM fewer pairs (up to 148 tiles of 2048, and from 297
// to 444: three CTAs of them to an SM against two of 4096).  Measured (B200, us per step, 4096 -> 2048): 304 K .. 606 K
// pairs, two tiles of 2048 to an SM or one of 4096: deterministic SGD on 400 K blocks of 16, 24-bit keys, 79 -> 86, on
// 600 K 96 -> 103, binned adds on 400 K 28.3 -> 29.7, Adam on 350 K and 550 K, 7-bit digits, 0.99 .. 1.01; outside: Adam on
// 200 K 0.97, 100 K 0.95 .. 0.99, 30 K 0.96, binned adds on 30 K and 150 K 0.95; Adam on 852 K 114 -> 111, ids that do not
// repeat 108 -> 100; 1.04 M, 508 tiles for 444 CTAs, 238 -> 243.
constexpr int kSortItems = 8, kSortItemsSmall = 4;
__host__ __device__ constexpr int sort_tile(int items) { return kSortThreads * items; }  // 4096 pairs, 2048
constexpr int kRadix = 256;
constexpr int kSortCtas = 2;                            // per SM (3, with 40 registers: spills, 6 % slower)
constexpr int kSortMaxGrid = 148 * kSortCtas;
constexpr int kSortMaxGridSmall = 148 * (kSortCtas + 1);  // tiles of kSortItemsSmall: 40 registers, 3 CTAs
static_assert(128 * kSortMaxGridSmall <= kRadix * kSortMaxGrid, "counts of passes of up to 7 bits");
constexpr int kScanThreads = 512;

inline size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

struct SortPlan {
    uint64_t nb;        // number of (key,val) pairs
    uint32_t grid;      // CTAs of the count / scatter kernels
    int items;          // keys per thread and tile
    uint64_t tiles;     // total tiles
};

// for passes of up to `width` bits
SortPlan make_plan(uint64_t nb, uint32_t width) {
    SortPlan sp;
    sp.nb = nb;
    const uint64_t small = (nb + sort_tile(kSortItemsSmall) - 1) / sort_tile(kSortItemsSmall);
    const uint64_t large = (nb + sort_tile(kSortItems) - 1) / sort_tile(kSortItems);
    auto of_busiest_sm = [](uint64_t tiles, int items) { return (tiles + 147) / 148 * items; };
    if (small <= (uint64_t)(width <= 7 ? kSortMaxGridSmall : kSortMaxGrid) &&
        of_busiest_sm(small, kSortItemsSmall) < of_busiest_sm(large, kSortItems)) {
        sp.items = kSortItemsSmall;
        sp.tiles = small;
        sp.grid = (uint32_t)small;
    } else {
        sp.items = kSortItems;
        sp.tiles = large;
        sp.grid = (uint32_t)(large < (uint64_t)kSortMaxGrid ? large : (uint64_t)kSortMaxGrid);
    }
    if (sp.grid == 0) sp.grid = 1;
    return sp;
}

// tiles [first, first+count) of CTA b: contiguous, near-equal split
__device__ __forceinline__ void cta_tiles(uint64_t tiles, uint32_t grid, uint32_t b,
                                          uint64_t& first, uint64_t& count) {
    uint64_t per = tiles / grid, rem = tiles % grid;
    count = per + (b < rem ? 1 : 0);
    first = per * b + (b < rem ? b : rem);
}

struct KeyArgs {
    MapParams mp;
    IdList indices;
    const int64_t* offsets;
    int64_t nbags;
    int64_t nnz;
    const int32_t* status;
};

// bag_of[p] = bag number of id position p (multi-hot only)
__global__ void __launch_bounds__(256) det_bag_of_kernel(KeyArgs a, uint32_t* bag_of) {
    const int64_t k = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5;
    const uint32_t lane = threadIdx.x & 31;
    if (k >= a.nbags) return;
    int64_t lo = __ldca(a.offsets + k), hi = __ldca(a.offsets + k + 1);
    lo = lo < 0 ? 0 : (lo > a.nnz ? a.nnz : lo);
    hi = hi < lo ? lo : (hi > a.nnz ? a.nnz : hi);
    for (int64_t p = lo + lane; p < hi; p += 32) bag_of[p] = (uint32_t)k;
}

// key[q] = h(e, x_p, c) for q = p*C + c.  val[q] = q when the sign hash is on (the apply kernel
// then needs the id again), else the position bag*d + c*Z of the block's first gradient element.
// One thread per id: the part of the hash that all chunks of the id share is evaluated once.
template <bool SIGN>
__global__ void __launch_bounds__(256)
det_keys_kernel(KeyArgs a, const uint32_t* bag_of, uint32_t* keys, uint32_t* vals) {
    follow<true>();
    const uint64_t p = (uint64_t)blockIdx.x * 256 + threadIdx.x;
    if (p >= (uint64_t)a.nnz) return;
    const MapParams& mp = a.mp;
    const uint64_t bag = bag_of ? (uint64_t)bag_of[p] : p;
    const uint32_t e = table_of_bag(bag, mp);
    const uint64_t x = (uint64_t)a.indices.load((int64_t)p);
    const uint64_t q0 = p * mp.C;
    if (mp.R > 1) {  // rows clubbed into one block: a single key
        keys[q0] = id_block_start(mp, e, x, 0);
        vals[q0] = SIGN ? (uint32_t)q0 : (uint32_t)(bag * mp.d);
        return;
    }
    const uint64_t base = hash_base(mp.h, e, x);
    for (uint32_t c = 0; c < mp.C; ++c) {
        if (!ROBE_CHK(q0 + c < (uint64_t)a.nnz * mp.C, ROBE_DBG_SORT_POS)) break;
        keys[q0 + c] = block_start(mp, base, c);
        vals[q0 + c] = SIGN ? (uint32_t)(q0 + c) : (uint32_t)(bag * mp.d + c * mp.Z);
    }
}

// The same, one thread per block: for many blocks per id (small Z) the writes of one thread per
// id would be far apart, and re-evaluating the shared part of the hash per block costs less.
template <bool SIGN>
__global__ void __launch_bounds__(256)
det_keys_by_block_kernel(KeyArgs a, const uint32_t* bag_of, uint32_t* keys, uint32_t* vals,
                         uint64_t nb) {
    follow<true>();
    const uint64_t q = (uint64_t)blockIdx.x * 256 + threadIdx.x;
    if (q >= nb) return;
    const MapParams& mp = a.mp;
    const uint32_t p = (uint32_t)q / mp.C;
    const uint32_t c = (uint32_t)q - p * mp.C;
    const uint64_t bag = bag_of ? (uint64_t)bag_of[p] : (uint64_t)p;
    const uint32_t e = table_of_bag(bag, mp);
    const uint64_t x = (uint64_t)a.indices.load(p);
    keys[q] = id_block_start(mp, e, x, c);
    vals[q] = SIGN ? (uint32_t)q : (uint32_t)(bag * mp.d + c * mp.Z);
}


// ---- radix sort pass, kernel 1: digit histogram of each CTA's contiguous key range
__global__ void __launch_bounds__(kSortThreads)
sort_count_kernel(const uint32_t* keys, uint32_t* counts, uint64_t nb, uint64_t tiles, uint32_t tile,
                  uint32_t shift, uint32_t mask) {
    __shared__ uint32_t hist[kSortWarps][kRadix];
    follow<true>();
    for (int k = threadIdx.x; k < kSortWarps * kRadix; k += kSortThreads) (&hist[0][0])[k] = 0;
    __syncthreads();
    uint64_t first, count;
    cta_tiles(tiles, gridDim.x, blockIdx.x, first, count);
    const uint64_t begin = first * tile;
    uint64_t end = (first + count) * tile;
    if (end > nb) end = nb;
    uint32_t* mine = hist[threadIdx.x >> 5];
    for (uint64_t i = begin + threadIdx.x; i < end; i += kSortThreads)
        atomicAdd(&mine[(keys[i] >> shift) & mask], 1u);
    __syncthreads();
    if (threadIdx.x > mask) return;
    uint32_t total = 0;
    for (int k = 0; k < kSortWarps; ++k) total += hist[k][threadIdx.x];
    counts[(uint64_t)threadIdx.x * gridDim.x + blockIdx.x] = total;
}

// Exclusive scan of the values held one per thread (value v of thread t): returns the sum of the values
// of threads below t.  All threads of the CTA call it; warp_sums holds a word per warp; contains
// __syncthreads.
__device__ __forceinline__ uint32_t cta_exclusive_scan(uint32_t v, uint32_t* warp_sums) {
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= (uint32_t)o) inc += n;
    }
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t k = 0; k < w; ++k) before += warp_sums[k];
    __syncthreads();  // warp_sums may be reused by the caller's next scan
    return before + inc - v;
}

// ---- kernel 2: one CTA per digit, of a thread per count where that suffices (512 threads for a handful of counts:
// 1.4 us more per pass of 256 digits): exclusive scan of that digit's per-CTA counts, in place, and the
// digit's total into totals[digit]
__global__ void __launch_bounds__(kScanThreads)
sort_scan_kernel(uint32_t* counts, uint32_t* totals, uint32_t grid) {
    __shared__ uint32_t warp_sums[kScanThreads / 32];
    follow<true>();
    uint32_t* row = counts + (uint64_t)blockIdx.x * grid;
    uint32_t carry = 0;
    for (uint32_t b0 = 0; b0 < grid; b0 += blockDim.x) {
        const uint32_t b = b0 + threadIdx.x;
        const uint32_t v = b < grid ? row[b] : 0u;
        const uint32_t ex = cta_exclusive_scan(v, warp_sums);
        if (b < grid) row[b] = carry + ex;
        // total of this chunk = exclusive prefix of the last thread + its value
        __shared__ uint32_t chunk_total;
        if (threadIdx.x == blockDim.x - 1) chunk_total = ex + v;
        __syncthreads();
        carry += chunk_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// ---- kernel 3: ranked scatter (STABLE: keeps the input order inside a digit - the LSD sort needs
// that; the binned backward does not and takes ranks from shared-memory counters).  Per tile of 4096 (2048)
// pairs: every warp ranks its 256 (128) pairs by digit (8 (4) rounds of ballots, earlier rounds and lower lanes
// first), the ranks are extended over the warps, the pairs are laid out in shared memory in (digit,
// original order), and then written out so that each digit's pairs go to consecutive addresses.
//
// Bound by the latency of a tile's phases, ranking most of all (34 M pairs, 7-bit digits: a plain copy
// through the same phases takes 94 us, ranking without the final stores 158, all of it 192).  So: one
// ballot per digit bit that the pass has (BITS), no bounds checks in full tiles, 32-bit positions, and the
// next tile's pairs asked for before this one is written out.  Measured (B200, same pairs, us per pass,
// before -> here): 247 -> 192; unstable with 6-bit digits 142 -> 130.  Finding the lanes of a digit by an
// atomicOr into a shared word instead of ballots takes as long.
template <bool STABLE, int BITS, int ITEMS>
struct ScatterSmem {
    uint2 pair[sort_tile(ITEMS)];
    // STABLE: per warp, pairs of each digit, then where they start in the tile
    uint16_t warp_digit[STABLE ? kSortWarps : 1][1 << BITS];
    uint32_t counter[1 << BITS];  // not STABLE: the same for the whole tile
    uint32_t base[1 << BITS];     // where the next pair of this digit goes, minus its place in the tile
    uint32_t warp_sums[kSortWarps];
};

// The pairs of the tile that starts at tbegin, warp-striped.  (nb may be close to 2^32: positions are
// compared relative to the tile, so that nothing overflows.)
template <int ITEMS>
__device__ __forceinline__ void scatter_load(const uint32_t* kin, const uint32_t* vin,
                                             uint32_t tbegin, uint32_t nb, uint32_t (&key)[ITEMS],
                                             uint32_t (&val)[ITEMS]) {
    const uint32_t left = nb - tbegin, local = (threadIdx.x >> 5) * (32 * ITEMS) + (threadIdx.x & 31);
    kin += tbegin;
    vin += tbegin;
    if (left >= (uint32_t)sort_tile(ITEMS)) {
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) key[r] = __ldcs(kin + (local + r * 32));
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) val[r] = __ldcs(vin + (local + r * 32));
    } else {
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            key[r] = local + r * 32 < left ? __ldcs(kin + (local + r * 32)) : 0u;
            val[r] = local + r * 32 < left ? __ldcs(vin + (local + r * 32)) : 0u;
        }
    }
}

template <bool STABLE, int BITS, int ITEMS, bool FULL>
__device__ __forceinline__ void scatter_tile(ScatterSmem<STABLE, BITS, ITEMS>& sm, const uint32_t* kin,
                                             const uint32_t* vin, uint32_t* kout,
                                             uint32_t* vout, uint32_t nb, uint32_t tbegin,
                                             uint32_t shift, uint32_t (&key)[ITEMS],
                                             uint32_t (&val)[ITEMS], bool more) {
    constexpr uint32_t R = 1u << BITS, mask = R - 1u;
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t left = nb - tbegin, local = w * (32 * ITEMS) + lane;  // (see scatter_load)
    if (STABLE) {
        for (uint32_t k = tid; k < kSortWarps * R / 2; k += kSortThreads)
            reinterpret_cast<uint32_t*>(&sm.warp_digit[0][0])[k] = 0;
    } else if (tid < R) {
        sm.counter[tid] = 0;
    }
    __syncthreads();
    uint32_t rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const bool valid = FULL || local + r * 32 < left;
        const uint32_t dg = (key[r] >> shift) & mask;
        rank[r] = 0;
        if (!STABLE) {  // any order inside a digit will do: the rank is what a shared-memory counter hands out
            if (valid) rank[r] = atomicAdd(&sm.counter[dg], 1u);
        } else {
            // lanes holding the same digit: one ballot per digit bit (a fixed cost, where
            // __match_any_sync takes time in proportion to the number of distinct digits)
            uint32_t peers = FULL ? 0xFFFFFFFFu : __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
            for (int b = 0; b < BITS; ++b) {
                const bool bit = (dg >> b) & 1u;
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, bit);
                peers &= bit ? bal : ~bal;
            }
            const uint32_t before = sm.warp_digit[w][dg];
            __syncwarp();
            if (valid && (peers & lt) == 0) sm.warp_digit[w][dg] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rank[r] = before + __popc(peers & lt);
        }
    }
    __syncthreads();
    // per digit: start of each warp's pairs inside the tile, and the tile's total
    uint32_t tile_total = 0;
    if (tid < R) {
        if (STABLE) {
#pragma unroll
            for (int k = 0; k < kSortWarps; ++k) tile_total += sm.warp_digit[k][tid];
        } else {
            tile_total = sm.counter[tid];
        }
    }
    const uint32_t ds = cta_exclusive_scan(tile_total, sm.warp_sums);  // syncs inside
    if (tid < R) {
        if (STABLE) {
            uint32_t from = ds;
#pragma unroll
            for (int k = 0; k < kSortWarps; ++k) {
                const uint32_t n = sm.warp_digit[k][tid];
                sm.warp_digit[k][tid] = (uint16_t)from;
                from += n;
            }
        } else {
            sm.counter[tid] = ds;
        }
        sm.base[tid] -= ds;  // a pair at tile position lp goes to base[digit] + lp
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (FULL || local + r * 32 < left) {
            const uint32_t dg = (key[r] >> shift) & mask;
            const uint32_t lp = (STABLE ? sm.warp_digit[w][dg] : sm.counter[dg]) + rank[r];
            if (!ROBE_CHK(lp < (uint32_t)sort_tile(ITEMS), ROBE_DBG_SHARED)) continue;
            sm.pair[lp] = make_uint2(key[r], val[r]);
        }
    }
    __syncthreads();
    if (more) scatter_load(kin, vin, tbegin + sort_tile(ITEMS), nb, key, val);
    const uint32_t in_tile = FULL ? sort_tile(ITEMS) : left;
#pragma unroll 4
    for (uint32_t lp = tid; lp < in_tile; lp += kSortThreads) {
        const uint2 p = sm.pair[lp];
        const uint32_t dst = sm.base[(p.x >> shift) & mask] + lp;
        if (!ROBE_CHK(dst < nb, ROBE_DBG_SORT_POS)) continue;
        kout[dst] = p.x;
        vout[dst] = p.y;
    }
    __syncthreads();
    if (tid < R) sm.base[tid] += ds + tile_total;  // undo the shift, advance past this tile's pairs
    // (the next tile's first barrier orders this update before its readers)
}

template <bool STABLE, int BITS, int ITEMS>
__global__ void __launch_bounds__(kSortThreads, ITEMS == kSortItems ? kSortCtas : kSortCtas + 1)
sort_scatter_kernel(const uint32_t* kin, const uint32_t* vin,
                    uint32_t* kout, uint32_t* vout,
                    const uint32_t* cta_offsets, const uint32_t* totals,
                    uint32_t nb, uint32_t tiles, uint32_t shift) {
    __shared__ ScatterSmem<STABLE, BITS, ITEMS> sm;
    const uint32_t tid = threadIdx.x;
    follow<true>();
    {
        // start of this digit in the output = pairs of lower digits + this digit's pairs in
        // lower CTAs
        const bool on = tid < (1u << BITS);
        const uint32_t below = cta_exclusive_scan(on ? totals[tid] : 0u, sm.warp_sums);
        if (on) sm.base[tid] = below + cta_offsets[(uint64_t)tid * gridDim.x + blockIdx.x];
    }
    uint64_t first, count;
    cta_tiles(tiles, gridDim.x, blockIdx.x, first, count);
    if (count == 0) return;
    uint32_t key[ITEMS], val[ITEMS];
    scatter_load(kin, vin, (uint32_t)first * sort_tile(ITEMS), nb, key, val);
    for (uint32_t t = (uint32_t)first; t < (uint32_t)(first + count); ++t) {
        const uint32_t tbegin = t * sort_tile(ITEMS);
        const bool more = t + 1 < (uint32_t)(first + count);
        if (nb - tbegin >= (uint32_t)sort_tile(ITEMS))
            scatter_tile<STABLE, BITS, ITEMS, true>(sm, kin, vin, kout, vout, nb, tbegin, shift, key, val, more);
        else
            scatter_tile<STABLE, BITS, ITEMS, false>(sm, kin, vin, kout, vout, nb, tbegin, shift, key, val, more);
    }
}

// One pass: count, scan, scatter by `width` bits at `shift`.  A pass may sort by a few bits more than asked
// (those of the next pass, which sorts by them again): three builds serve all widths.
template <bool STABLE, int BITS>
void launch_sort_pass_bits(const SortPlan& sp, const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout,
                           uint32_t* counts, uint32_t* totals, uint32_t shift, cudaStream_t st) {
    launch_next(sort_count_kernel, sp.grid, kSortThreads, 0, st, kin, counts, sp.nb, sp.tiles, (uint32_t)sort_tile(sp.items), shift,
                (1u << BITS) - 1u);
    const unsigned scan_threads = sp.grid < (uint32_t)kScanThreads ? (sp.grid + 31) / 32 * 32 : (unsigned)kScanThreads;
    launch_next(sort_scan_kernel, 1 << BITS, scan_threads, 0, st, counts, totals, sp.grid);
    auto scatter = [&](auto kernel) {
        launch_next(kernel, sp.grid, kSortThreads, 0, st, kin, vin, kout, vout, counts, totals, (uint32_t)sp.nb, (uint32_t)sp.tiles, shift);
    };
    if (sp.items == kSortItems) scatter(sort_scatter_kernel<STABLE, BITS, kSortItems>);
    else scatter(sort_scatter_kernel<STABLE, BITS, kSortItemsSmall>);
}

template <bool STABLE>
void launch_sort_pass(const SortPlan& sp, const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout,
                      uint32_t* counts, uint32_t* totals, uint32_t shift, uint32_t width, cudaStream_t st) {
    if (width <= 6) launch_sort_pass_bits<STABLE, 6>(sp, kin, vin, kout, vout, counts, totals, shift, st);
    else if (width == 7) launch_sort_pass_bits<STABLE, 7>(sp, kin, vin, kout, vout, counts, totals, shift, st);
    else launch_sort_pass_bits<STABLE, 8>(sp, kin, vin, kout, vout, counts, totals, shift, st);
}

// A round of the apply kernel whose walks got long, handed over to the long-walk kernel: where
// the tile starts, how far the lanes have come, and per lane its slot, its sum so far and its
// position in the tile.
struct LongWalk {
    uint64_t i0;
    uint32_t fbase;         // lane l goes on at sorted position i0 + fbase + e(l)
    uint32_t pad;
    uint32_t j[32];
    float acc[32];
    uint32_t state[32];     // e | going << 8 | touched << 9
};

struct ApplyArgs {
    MapParams mp;
    const float* grad_out;
    IdList indices;  // only read when the sign hash is on
    float* target;
    float lr;
    uint64_t nb;
    const int32_t* status;
    AdamState adam;          // update mode 2 only
    uint32_t* long_count;    // number of handed-over rounds (may run past long_cap)
    LongWalk* long_walks;
    uint32_t long_cap;
    uint64_t grad_elems;       // elements of grad_out (read by the debug build's index checks only)
    int l2_keep;               // binned adds: the reductions carry the L2 "keep" policy
};

// The term that the sorted block with payload v contributes to the slot at in-block offset o
// (o < Z), or nothing if o is past the end of a short last block.
template <bool SIGN, bool SHORT>
__device__ __forceinline__ bool block_term(const ApplyArgs& a, const uint32_t* bag_of, uint32_t v,
                                           uint32_t o, float& term) {
    const MapParams& mp = a.mp;
    if (!SIGN) {
        // v = bag*d + c*Z: the block's first element in grad_out
        if (SHORT) {
            const uint32_t cz = v - (v / mp.d) * mp.d;
            if (cz + o >= mp.d) return false;
        }
        if (!ROBE_CHK((uint64_t)v + o < a.grad_elems, ROBE_DBG_GRAD_POS)) return false;
        term = __ldca(a.grad_out + (uint64_t)v + o);
        return true;
    }
    const uint32_t p = v / mp.C;  // v = q
    const uint32_t c = v - p * mp.C;
    const uint32_t i = c * mp.Z + o;
    if (i >= mp.d) return false;
    const uint64_t bag = bag_of ? (uint64_t)__ldca(bag_of + p) : (uint64_t)p;
    if (!ROBE_CHK(bag * mp.d + i < a.grad_elems, ROBE_DBG_GRAD_POS)) return false;
    const uint32_t e = table_of_bag(bag, mp);
    const uint64_t x = (uint64_t)a.indices.load(p);
    term = sign_of(mp, hash_base(mp.g, e, x), i) * __ldca(a.grad_out + bag * mp.d + i);
    return true;
}

// Slots j in [Z-1, m).  The sorted blocks that reach slot j are those with key in [j-Z+1, j];
// the slot is served from the FIRST of them: position i serves slot K[i]+u iff i starts a run of
// equal keys and the previous key is below K[i]+u-Z+1, i.e. u >= Z - min(Z, K[i]-K[i-1]).  The
// server then only walks forward through the sorted list, adding terms while the key stays <= j.
//
// One warp takes 32 consecutive sorted positions (a tile).  Keys and payloads live in a
// warp-private ring of 128 positions in shared memory, filled by coalesced loads.  The
// (position, offset) pairs of the tile that serve a slot are numbered through and dealt out one
// per lane, 32 per round.  In a round all lanes step through the ring together, each from its own
// position, UN positions per step (4 in the first step, then 8): ring reads, then the gradient
// loads, then the adds in sorted order; the next 32 positions are fetched one step ahead of
// their first use.  A walk that is still going after 64 positions (an id that occurs many
// times in the batch) is handed, with its sums so far, to the long-walk kernel below, whose
// division of labour adds such a chain several times faster.  Only if the list of handed-over
// rounds is full does it go on here, 16 positions per step, with the gradient rows of the
// positions after those asked into L2 ahead of time.
constexpr uint32_t kRing = 128;
constexpr uint32_t kNoKey = 0xFFFFFFFFu;  // above every slot number (m + d <= 2^32)

struct ApplyTile {
    const uint32_t* K;
    const uint32_t* V;
    uint64_t nb;
    uint64_t i0;          // first sorted position of the tile
    uint2* ring;          // warp-private, kRing entries
    uint32_t loaded_end;  // the ring holds tile-relative positions [loaded_end - kRing, loaded_end)
    // (key, payload) of tile-relative position r, or a key above every slot past the end
    __device__ __forceinline__ uint2 fetch(uint32_t r) const {
        const uint64_t idx = i0 + r;
        if (idx >= nb) return make_uint2(kNoKey, 0u);
        return make_uint2(__ldca(K + idx), __ldca(V + idx));
    }
};

struct ApplyWalk {
    float acc;
    bool touched, done, pending;
    uint2 ahead;     // positions [loaded_end, loaded_end + 32), fetched but not yet in the ring
    uint32_t fbase;  // the next step starts at tile-relative position fbase + sub
};

// The positions fetched last enter the ring.  pf != nullptr: their gradient rows are asked
// into L2 (pf = grad_out + the first offset of the lanes' chunk).
__device__ __forceinline__ void walk_commit(ApplyTile& tl, ApplyWalk& wk, uint32_t lane,
                                            const float* pf) {
    __syncwarp();
    tl.ring[(tl.loaded_end + lane) & (kRing - 1)] = wk.ahead;
    if (pf != nullptr && wk.ahead.x != kNoKey)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pf + wk.ahead.y));
    tl.loaded_end += 32;
    wk.pending = false;
    __syncwarp();
}

// Start of a step of UN positions: the positions fetched one step ago enter the ring, and the
// ones the step after this one will read are fetched.
template <int UN>
__device__ __forceinline__ void walk_advance(ApplyTile& tl, ApplyWalk& wk, uint32_t EPW,
                                             uint32_t lane, const float* pf) {
    if (wk.pending) walk_commit(tl, wk, lane, pf);
    // the next step reads up to position fbase + UN + (EPW-1) + (UN-1)
    if (tl.loaded_end <= wk.fbase + 2 * UN + EPW - 2) {
        wk.ahead = tl.fetch(tl.loaded_end + lane);
        wk.pending = true;
    }
}

// Steps of UN positions until no lane goes on, or (limit != 0) until fbase reaches limit.
// Returns whether every lane is done.
template <bool SIGN, bool SHORT, int UN>
__device__ __forceinline__ bool walk_steps(const ApplyArgs& a, const uint32_t* bag_of, ApplyTile& tl,
                                           ApplyWalk& wk, uint32_t j, uint32_t sub, uint32_t EPW,
                                           uint32_t lane, uint32_t limit) {
    for (;; wk.fbase += UN) {
        if (limit != 0 && wk.fbase >= limit) return false;
        walk_advance<UN>(tl, wk, EPW, lane, nullptr);
        uint2 kv[UN];
#pragma unroll
        for (int t = 0; t < UN; ++t) kv[t] = tl.ring[(wk.fbase + sub + t) & (kRing - 1)];
        float term[UN];
        bool ok[UN];
        bool in_last = false;
#pragma unroll
        for (int t = 0; t < UN; ++t) {
            const bool in = !wk.done && kv[t].x <= j;  // sorted: true on a prefix
            ok[t] = false;
            if (in) ok[t] = block_term<SIGN, SHORT>(a, bag_of, kv[t].y, j - kv[t].x, term[t]);
            if (t == UN - 1) in_last = in;
        }
#pragma unroll
        for (int t = 0; t < UN; ++t)
            if (ok[t]) {
                wk.acc = __fadd_rn(wk.acc, term[t]);
                wk.touched = true;
            }
        wk.done = wk.done || !in_last;
        if (__ballot_sync(0xFFFFFFFFu, !wk.done) == 0) {
            wk.fbase += UN;
            return true;
        }
    }
}

// The same for a long walk of plain blocks (sign off, no short last block): more positions per
// step, each term's place in grad_out computed while its key is compared.
__device__ __forceinline__ bool walk_deep(const ApplyArgs& a, ApplyTile& tl, ApplyWalk& wk, uint32_t j,
                                          uint32_t sub, uint32_t EPW, uint32_t lane,
                                          uint32_t chunk_off, uint32_t limit) {
    constexpr int UN = 16;
    const float* pf = a.grad_out + chunk_off;
    // the ring has to reach the end of the first step before the one-step-ahead fetches take over
    if (wk.pending) walk_commit(tl, wk, lane, pf);
    while (tl.loaded_end < wk.fbase + EPW + UN - 1) {
        wk.ahead = tl.fetch(tl.loaded_end + lane);
        walk_commit(tl, wk, lane, pf);
    }
    for (;; wk.fbase += UN) {
        if (limit != 0 && wk.fbase >= limit) return false;
        walk_advance<UN>(tl, wk, EPW, lane, pf);
        uint32_t at[UN];
        uint32_t n_in = 0;
#pragma unroll
        for (int t = 0; t < UN; ++t) {
            const uint2 e = tl.ring[(wk.fbase + sub + t) & (kRing - 1)];
            n_in += (!wk.done && e.x <= j) ? 1u : 0u;  // sorted: a prefix of the step
            at[t] = e.y + (j - e.x);
        }
        const uint32_t n_max = __reduce_max_sync(0xFFFFFFFFu, n_in);  // warp-uniform
        float term[UN];
#pragma unroll
        for (int t = 0; t < UN; ++t) {
            term[t] = 0.0f;
            if ((uint32_t)t < n_max) {
                if ((uint32_t)t < n_in && ROBE_CHK((uint64_t)at[t] < a.grad_elems, ROBE_DBG_GRAD_POS))
                    term[t] = __ldca(a.grad_out + at[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < UN; ++t) {
            if ((uint32_t)t < n_max) {
                if ((uint32_t)t < n_in) wk.acc = __fadd_rn(wk.acc, term[t]);
            }
        }
        if (n_in != 0) wk.touched = true;
        wk.done = wk.done || n_in < (uint32_t)UN;
        if (n_max < (uint32_t)UN) {  // no lane goes on
            wk.fbase += UN;
            return true;
        }
    }
}

template <bool SIGN, int MODE, bool SHORT>
__global__ void __launch_bounds__(256)
det_apply_kernel(ApplyArgs a, const uint32_t* K, const uint32_t* V,
                 const uint32_t* bag_of) {
    constexpr int UN = 8;
    constexpr uint32_t kDeepAfter = 64;       // positions after which a walk takes 16 per step, if it stays here
    constexpr uint32_t kHandOverAfter = 64;   // positions after which it goes to the long-walk kernel (128 and 256
                                              // measured slower on Zipf ids, 32 no faster)
    __shared__ uint2 ring_s[8][kRing];
    if (a.status != nullptr && *a.status != 0) return;
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    ApplyTile tl;
    tl.K = K;
    tl.V = V;
    tl.nb = a.nb;
    tl.i0 = ((uint64_t)blockIdx.x * 8 + w) * 32;
    if (tl.i0 >= a.nb) return;  // whole warp
    tl.ring = ring_s[w];
    const uint2 mine = tl.fetch(lane);
    tl.ring[lane] = mine;
    tl.ring[32 + lane] = tl.fetch(32 + lane);
    tl.loaded_end = 64;

    // first offset served from this lane's position (Z = none)
    uint32_t kprev = __shfl_up_sync(0xFFFFFFFFu, mine.x, 1);
    if (lane == 0 && tl.i0 > 0) kprev = __ldca(K + tl.i0 - 1);
    uint32_t own_lo = mp.Z;
    if (tl.i0 + lane < a.nb) {
        if (tl.i0 + lane == 0) own_lo = 0;
        else if (kprev != mine.x) {
            const uint32_t gap = mine.x - kprev;
            own_lo = gap >= mp.Z ? 0u : mp.Z - gap;
        }
    }
    __syncwarp();

    // Served (position, offset) pairs are numbered tile-wide - position after position, offsets
    // ascending - and dealt out 32 per round, one pair per lane, so that no lane idles on a pair
    // that serves nothing.
    const uint32_t cnt = mp.Z - own_lo;
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += n;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);

    for (uint32_t r0 = 0; r0 < total; r0 += 32) {
        const uint32_t idx = r0 + lane;
        // position e of pair idx: the first lane whose inclusive count exceeds idx
        uint32_t e = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            const uint32_t v = __shfl_sync(0xFFFFFFFFu, incl, e + step - 1);
            if (v <= idx) e += step;
        }
        if (e > 31) e = 31;  // idx >= total: no pair
        const uint32_t incl_e = __shfl_sync(0xFFFFFFFFu, incl, e);
        const uint32_t lo_e = __shfl_sync(0xFFFFFFFFu, own_lo, e);
        const uint32_t s = __shfl_sync(0xFFFFFFFFu, mine.x, e);
        const uint32_t u = mp.Z - (incl_e - idx);  // lo_e <= u < Z for a real pair
        const uint64_t j64 = (uint64_t)s + u;
        // j64 >= m: wrapped part, j64 < Z-1: low slots - both belong to the other kernel
        bool active = idx < total && u >= lo_e && u < mp.Z && j64 < mp.m && j64 + 1 >= mp.Z;
        if (__ballot_sync(0xFFFFFFFFu, active) == 0) continue;
        const uint32_t j = (uint32_t)j64;
        float old = 0.0f;
        if (active && ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT)) old = a.target[j];

        if (tl.loaded_end > kRing) {  // an earlier long walk moved the ring past the tile's start
            __syncwarp();
            tl.ring[lane] = mine;
            tl.ring[32 + lane] = tl.fetch(32 + lane);
            tl.loaded_end = 64;
            __syncwarp();
        }

        // the lane walks from its own position e: step n reads positions fbase + e + t
        ApplyWalk wk;
        wk.acc = 0.0f;
        wk.touched = false;
        wk.done = !active;
        wk.pending = false;
        wk.ahead = make_uint2(kNoKey, 0u);
        wk.fbase = 0;
        if (!walk_steps<SIGN, SHORT, 4>(a, bag_of, tl, wk, j, e, 32u, lane, 4)) {
            if (!SIGN && !SHORT) {
                if (!walk_steps<SIGN, SHORT, UN>(a, bag_of, tl, wk, j, e, 32u, lane, kDeepAfter) &&
                    !walk_deep(a, tl, wk, j, e, 32u, lane, u & ~31u, kHandOverAfter)) {
                    // long walks: hand the round over if the list has room, else go on here
                    uint32_t rec = a.long_cap;
                    if (a.long_cap != 0) {
                        if (lane == 0) rec = atomicAdd(a.long_count, 1u);
                        rec = __shfl_sync(0xFFFFFFFFu, rec, 0);
                    }
                    if (rec < a.long_cap) {
                        LongWalk* lw = a.long_walks + rec;
                        if (lane == 0) {
                            lw->i0 = tl.i0;
                            lw->fbase = wk.fbase;
                        }
                        lw->j[lane] = j;
                        lw->acc[lane] = wk.acc;
                        lw->state[lane] = e | (wk.done ? 0u : 1u << 8) | (wk.touched ? 1u << 9 : 0u);
                        if (!wk.done) wk.touched = false;  // finished (and stored) by the other kernel
                    } else {
                        walk_deep(a, tl, wk, j, e, 32u, lane, u & ~31u, 0);
                    }
                }
            } else {
                walk_steps<SIGN, SHORT, UN>(a, bag_of, tl, wk, j, e, 32u, lane, 0);
            }
        }
        if (wk.touched) commit_slot<MODE>(a, j, wk.acc, old);
    }
}

// Long walks (plain blocks only).  One CTA of eight warps per handed-over round, in steps of
// kLongStep = 64 positions.  Lane l of EVERY warp stands for slot l of the round.  The keys come
// from a ring of 512 positions in shared memory.  The chain of dependent adds of one slot is the
// definition's, so everything else is kept off the warp that adds:
//   warp 0      adds the terms of each slot in sorted order, one step per iteration;
//   warps 1..6  copy: each takes every sixth position of the step kLongDepth ahead, and a lane
//               copies the term of its slot with cp.async into its own column of that step's
//               buffer (a whole step in flight without a register per term);
//   warp 7      brings the keys of later steps into the ring (asked for an iteration before they
//               are stored) and finds, by bisection, how many positions of the NEXT step reach
//               each slot - sorted keys make "this position still reaches slot j" a prefix property.
// kLongDepth + 1 buffers; ONE barrier per step.
constexpr int kLongStep = 64;
constexpr int kLongWarps = 8;
constexpr int kLongCopiers = kLongWarps - 2;
constexpr int kLongDepth = 4;                 // steps ahead of the adder whose copies are issued
constexpr int kLongBufs = kLongDepth + 1;
constexpr uint32_t kLongRing = 512;           // >= (kLongDepth + 2) steps + 32 positions of lane spread, power of two
static_assert((kLongDepth + 2) * kLongStep + 32 <= (int)kLongRing, "ring too short");
static_assert(kLongStep == 64, "the scout warp brings in two keys per lane and step");

template <int MODE>
__global__ void __launch_bounds__(32 * kLongWarps)
det_apply_long_kernel(ApplyArgs a, const uint32_t* K, const uint32_t* V) {
    __shared__ float terms_s[kLongBufs][kLongStep][32];
    __shared__ uint2 ring[kLongRing];
    __shared__ uint32_t reach_s[2][32];  // by step parity: positions of the step that reach each slot
    __shared__ uint32_t go_on[2];        // by step parity: is there a step to add?
    __shared__ uint32_t rec_s;
    if (a.status != nullptr && *a.status != 0) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t n_rec = *a.long_count < a.long_cap ? *a.long_count : a.long_cap;
    const uint32_t dst0 = (uint32_t)__cvta_generic_to_shared(&terms_s[0][0][lane]);
    constexpr uint32_t kBufBytes = kLongStep * 32 * sizeof(float);
    constexpr int kPerCopier = (kLongStep + kLongCopiers - 1) / kLongCopiers;
    const bool adder = w == 0, scout = w == kLongWarps - 1;
    // Rounds differ in length by orders of magnitude: a CTA takes the next one when it is free
    // (a.long_count[1] counts the rounds taken) instead of a fixed share.
    for (;;) {
        if (tid == 0) rec_s = atomicAdd(a.long_count + 1, 1u);
        __syncthreads();  // (the barriers inside a round order this store after all reads of the last one)
        const uint32_t rec = rec_s;
        if (rec >= n_rec) break;
        if (!ROBE_CHK(rec < a.long_cap, ROBE_DBG_LONG_WALK)) break;
        const LongWalk* lw = a.long_walks + rec;
        const uint64_t i0 = lw->i0;
        const uint32_t j = lw->j[lane];
        const uint32_t st = lw->state[lane];
        const uint32_t e = st & 0xFFu;
        const bool mine = (st >> 8) & 1u;  // this lane's walk was handed over
        float acc = lw->acc[lane];         // used by warp 0 only
        bool touched = (st >> 9) & 1u;
        auto fetch = [&](uint32_t r) -> uint2 {
            const uint64_t idx = i0 + r;
            if (idx >= a.nb) return make_uint2(kNoKey, 0u);
            return make_uint2(__ldca(K + idx), __ldca(V + idx));
        };
        // This copier warp's share of the copies of the step that starts at tile-relative position `base`.
        auto issue = [&](uint32_t base, uint32_t buf) {
            const uint32_t dst = dst0 + buf * kBufBytes;
            uint2 kv[kPerCopier];
#pragma unroll
            for (int q = 0; q < kPerCopier; ++q) {
                const uint32_t t = (w - 1) + q * kLongCopiers;
                kv[q] = ring[(base + e + (t < (uint32_t)kLongStep ? t : 0u)) & (kLongRing - 1)];
            }
#pragma unroll
            for (int q = 0; q < kPerCopier; ++q) {
                const uint32_t t = (w - 1) + q * kLongCopiers;
                if (t < (uint32_t)kLongStep && mine && kv[q].x <= j &&
                    ROBE_CHK((uint64_t)kv[q].y + (j - kv[q].x) < a.grad_elems, ROBE_DBG_GRAD_POS)) {
                    const float* src = a.grad_out + (kv[q].y + (j - kv[q].x));
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + t * 128u), "l"(src));
                }
            }
            asm volatile("cp.async.commit_group;");
        };
        // How many positions of that step reach slot j: first t with key > j, by bisection.
        auto reach = [&](uint32_t base) -> uint32_t {
            if (!mine) return 0u;
            uint32_t lo = 0, hi = kLongStep;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (ring[(base + e + mid) & (kLongRing - 1)].x <= j) lo = mid + 1; else hi = mid;
            }
            return lo;
        };
        // a step reads positions base + e + t, e < 32, t < kLongStep: [base, base + kLongStep + 32);
        // the ring is kept filled up to the end of the step kLongDepth steps ahead
        constexpr uint32_t kAhead = (kLongDepth + 1) * kLongStep + 32;
        uint32_t base = lw->fbase;
        uint32_t ring_end = base + kAhead;
        for (uint32_t r = tid; r < kAhead; r += 32 * kLongWarps)
            ring[(base + r) & (kLongRing - 1)] = fetch(base + r);
        if (tid == 0) go_on[0] = 1u;
        __syncthreads();
        uint2 pend0 = make_uint2(kNoKey, 0u), pend1 = pend0;  // scout: keys of ring_end + lane, + 32 + lane
        if (scout) {
            pend0 = fetch(ring_end + lane);
            pend1 = fetch(ring_end + 32 + lane);
            reach_s[0][lane] = reach(base);
        } else if (!adder) {
#pragma unroll
            for (int s = 0; s < kLongDepth; ++s) issue(base + s * kLongStep, s);
            asm volatile("cp.async.wait_group %0;" ::"n"(kLongDepth - 1) : "memory");  // step 0 is in
        }
        for (uint32_t step = 0;; ++step) {
            // the copies of `step` are in (every copier waited for its own) and the adds of
            // step - 1 are done, so its buffer may be refilled; the ring holds the next keys
            __syncthreads();
            if (go_on[step & 1u] == 0) break;
            if (adder) {
                const float(*buf)[32] = terms_s[step % kLongBufs];
                const uint32_t n_cur = reach_s[step & 1u][lane];
                const uint32_t n_max = __reduce_max_sync(0xFFFFFFFFu, n_cur);
                for (uint32_t t0 = 0; t0 < n_max; t0 += 16) {
                    float x[16];
#pragma unroll
                    for (int q = 0; q < 16; ++q) x[q] = buf[t0 + q][lane];
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        if (t0 + q < n_cur) acc = __fadd_rn(acc, x[q]);
                }
                if (n_cur != 0) touched = true;
            } else if (scout) {
                // keys: asked for a whole iteration before they are stored into the ring
                const uint2 f0 = fetch(ring_end + kLongStep + lane);
                const uint2 f1 = fetch(ring_end + kLongStep + 32 + lane);
                const uint32_t n_nxt = reach(base + kLongStep);
                reach_s[(step + 1) & 1u][lane] = n_nxt;
                const bool any_next = __ballot_sync(0xFFFFFFFFu, n_nxt != 0) != 0;
                if (lane == 0) go_on[(step + 1) & 1u] = any_next ? 1u : 0u;
                ring[(ring_end + lane) & (kLongRing - 1)] = pend0;
                ring[(ring_end + 32 + lane) & (kLongRing - 1)] = pend1;
                pend0 = f0;
                pend1 = f1;
            } else {
                issue(base + kLongDepth * kLongStep, (step + kLongDepth) % kLongBufs);
                asm volatile("cp.async.wait_group %0;" ::"n"(kLongDepth - 1) : "memory");  // step + 1 is in
            }
            ring_end += kLongStep;
            base += kLongStep;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (adder && mine && touched) commit_slot<MODE>(a, j, acc, a.target[j]);
    }
}

// Slots j in [0, Z-1): plain blocks with key <= j first, then the wrapped tails of blocks
// whose key lies in [m + j - (Z-1), m-1] (o = j + m - key).  One warp per slot: the lanes fetch
// the terms of 32 consecutive sorted positions, then all lanes add them in order.
constexpr unsigned kLowWarps = 4;

template <bool SIGN, bool SHORT>
__device__ __forceinline__ void low_walk(const ApplyArgs& a, const uint32_t* K,
                                         const uint32_t* V, const uint32_t* bag_of,
                                         uint64_t from, uint64_t to, uint64_t j_plus, float& acc,
                                         bool& touched) {
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t i0 = from; i0 < to; i0 += 32) {
        const uint64_t i = i0 + lane;
        float term = 0.0f;
        bool ok = false;
        if (i < to) ok = block_term<SIGN, SHORT>(a, bag_of, __ldca(V + i), (uint32_t)(j_plus - __ldca(K + i)), term);
        const uint32_t oks = __ballot_sync(0xFFFFFFFFu, ok);
        if (oks != 0) touched = true;
        for (uint32_t rest = oks; rest != 0; rest &= rest - 1) {
            const int src = __ffs((int)rest) - 1;
            acc = __fadd_rn(acc, __shfl_sync(0xFFFFFFFFu, term, src));
        }
    }
}

// first sorted position with key >= bound (warp-uniform)
__device__ __forceinline__ uint64_t first_at_least(const uint32_t* K, uint64_t nb, uint64_t bound) {
    uint64_t lo = 0, hi = nb;
    while (lo < hi) {
        const uint64_t mid = lo + ((hi - lo) >> 1);
        if ((uint64_t)__ldca(K + mid) >= bound) hi = mid; else lo = mid + 1;
    }
    return lo;
}

template <bool SIGN, int MODE, bool SHORT>
__global__ void __launch_bounds__(32 * kLowWarps)
det_apply_low_kernel(ApplyArgs a, const uint32_t* K, const uint32_t* V,
                     const uint32_t* bag_of) {
    if (a.status != nullptr && *a.status != 0) return;
    const MapParams& mp = a.mp;
    const uint32_t j = blockIdx.x * kLowWarps + (threadIdx.x >> 5);
    if (j + 1 >= mp.Z) return;
    float acc = 0.0f;
    bool touched = false;
    low_walk<SIGN, SHORT>(a, K, V, bag_of, 0, first_at_least(K, a.nb, (uint64_t)j + 1), j, acc, touched);
    const uint64_t lowkey = (uint64_t)mp.m - (mp.Z - 1) + j;  // > j because m >= Z
    low_walk<SIGN, SHORT>(a, K, V, bag_of, first_at_least(K, a.nb, lowkey), a.nb, (uint64_t)j + mp.m, acc,
                          touched);
    if (touched && (threadIdx.x & 31) == 0) commit_slot<MODE>(a, j, acc, a.target[j]);
}

// Binned (not deterministic) backward: after ONE scatter pass on the top key bits the blocks are
// grouped by array region (a bin covers 2^shift consecutive slots, 16 MB or so), and this kernel
// adds them in that order with red.global: thread (i, u) adds term u of sorted block i.  The
// blocks in flight at any moment fall into one or two bins, so the read-modify-write of the array
// happens in L2 and every array sector crosses the DRAM bus about once per call instead of once
// per block that touches it.  a.lr carries the scale (1 for a dense gradient, -lr for SGD).
constexpr int kBinnedPer = 8;  // sorted blocks per thread group, all their loads in flight together

template <bool SIGN, bool SHORT>
__global__ void __launch_bounds__(256)
binned_apply_kernel(ApplyArgs a, const uint32_t* K, const uint32_t* V,
                    const uint32_t* bag_of, uint32_t log2Zp) {
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const MapParams& mp = a.mp;
    const uint64_t tid = (uint64_t)blockIdx.x * 256 + threadIdx.x;
    const uint64_t i0 = (tid >> log2Zp) * kBinnedPer;
    const uint32_t u = (uint32_t)(tid & ((1u << log2Zp) - 1u));
    if (i0 >= a.nb || u >= mp.Z) return;
    uint32_t k[kBinnedPer], v[kBinnedPer];
#pragma unroll
    for (int t = 0; t < kBinnedPer; ++t) {
        const uint64_t i = i0 + t < a.nb ? i0 + t : a.nb - 1;
        k[t] = __ldca(K + i);
        v[t] = __ldca(V + i);
    }
    const uint64_t pol = l2_keep_policy(a.l2_keep != 0);
    float term[kBinnedPer];
    bool ok[kBinnedPer];
#pragma unroll
    for (int t = 0; t < kBinnedPer; ++t)
        ok[t] = i0 + t < a.nb && block_term<SIGN, SHORT>(a, bag_of, v[t], u, term[t]);
#pragma unroll
    for (int t = 0; t < kBinnedPer; ++t) {
        if (ok[t]) {
            uint64_t j = (uint64_t)k[t] + u;
            if (j >= mp.m) j -= mp.m;
            if (ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT)) red_add(a.target + j, a.lr * term[t], pol);
        }
    }
}

// answer = do starts repeat among 32 neighbours of the sorted list?  128 places looked at, a quarter of them with a
// repeat is a yes.
__global__ void __launch_bounds__(1024) binned_sample_kernel(const uint32_t* K, uint64_t nb, uint32_t* answer) {
    follow();
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t found = 0;
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
        const uint64_t at = (nb - 32) / 128 * (w * 4 + q) + lane;  // (nb is large)
        const uint32_t k = __ldca(K + at);
        found += __any_sync(0xFFFFFFFFu, __popc(__match_any_sync(0xFFFFFFFFu, k)) > 1) ? 1u : 0u;
    }
    __shared__ uint32_t total_s;
    if (threadIdx.x == 0) total_s = 0;
    __syncthreads();
    if (lane == 0) atomicAdd(&total_s, found);
    __syncthreads();
    if (threadIdx.x == 0) *answer = total_s >= 32u ? 1u : 0u;
}

// Repeats of one start (an id that the batch draws often) would be reductions on the same slots, one after the
// other in L2.  The CTA's 256 blocks are brought together by a counting sort on a hash of their starts, and
// the gradient rows of equal starts among 32 neighbours are summed before one reduction.
// Measured (B200, 34 M blocks of 16 from Zipf ids on 1 GB, us): 5380 -> 2360; 13 tables of d = 73, Z = 32
// 2580 -> 1170.  Spread ids gain nothing from it (805 -> 905), nor do small calls (1.1 M blocks 46 -> 71): the
// launcher asks for it from 8 M blocks on, and a sample of the sorted list says whether starts repeat.
template <int LP, int EPL, bool SHORT>
__device__ __forceinline__ void binned_add_merged(const ApplyArgs& a, uint32_t k, uint32_t v, uint2* sorted, uint32_t* count,
                                                  uint32_t* warp_sums) {
    constexpr uint32_t G = 32 / LP;
    const MapParams& mp = a.mp;
    const uint32_t tid = threadIdx.x, lane = tid & 31, g = lane / LP, ol = lane % LP, Z = mp.Z, m = mp.m;
    const uint32_t bin = (k * 0x9E3779B1u) >> 24;
    count[tid] = 0;
    __syncthreads();
    const uint32_t rank = atomicAdd(&count[bin], 1u);
    __syncthreads();
    const uint32_t start = cta_exclusive_scan(count[tid], warp_sums);  // syncs inside
    count[tid] = start;
    __syncthreads();
    if (ROBE_CHK(count[bin] + rank < 256u, ROBE_DBG_SHARED)) sorted[count[bin] + rank] = make_uint2(k, v);
    __syncthreads();
    const uint2 kv = sorted[tid];
    k = kv.x;
    v = kv.y;
    uint32_t len = k == kNoKey ? 0u : Z;
    if (SHORT && len != 0) {
        const uint32_t left = mp.d - v % mp.d;
        if (left < Z) len = left;
    }
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, k);
    const uint64_t pol = l2_keep_policy(a.l2_keep != 0);
    uint32_t rest = __ballot_sync(0xFFFFFFFFu, len != 0 && (peers & ((1u << lane) - 1u)) == 0);  // first of each start
    while (rest != 0) {
        uint32_t left = rest;  // group g takes the g-th start that is left
#pragma unroll
        for (uint32_t i = 0; i + 1 < G; ++i)
            if (i < g) left &= left - 1;
#pragma unroll
        for (uint32_t i = 0; i < G; ++i) rest &= rest - 1;
        const int src = left != 0 ? __ffs((int)left) - 1 : 0;
        uint32_t from = __shfl_sync(0xFFFFFFFFu, peers, src);
        const uint32_t first = __shfl_sync(0xFFFFFFFFu, k, src);
        if (left == 0) from = 0;
        float sum[EPL];
        uint32_t reach = 0;  // longest of the blocks
#pragma unroll
        for (int q = 0; q < EPL; ++q) sum[q] = 0.0f;
        while (__any_sync(0xFFFFFFFFu, from != 0)) {
            float x[4][EPL];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = from != 0 ? __ffs((int)from) - 1 : 0;
                const uint32_t row = __shfl_sync(0xFFFFFFFFu, v, p) + ol;
                uint32_t l = __shfl_sync(0xFFFFFFFFu, len, p);
                if (from == 0) l = 0;
                if (l > reach) reach = l;
                from &= from - 1;
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    x[u][q] = ol + 32 * q < l && ROBE_CHK((uint64_t)row + 32 * q < a.grad_elems, ROBE_DBG_GRAD_POS)
                                  ? __ldca(a.grad_out + (row + 32 * q))
                                  : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < EPL; ++q) sum[q] += x[u][q];
        }
#pragma unroll
        for (int q = 0; q < EPL; ++q)
            if (ol + 32 * q < reach) {
                uint32_t j = first + ol + 32 * q;  // < m + d <= 2^32
                if (j >= m) j -= m;
                if (ROBE_CHK(j < m, ROBE_DBG_ARRAY_SLOT)) red_add(a.target + j, a.lr * sum[q], pol);
            }
    }
}

// The same for plain blocks of up to 128 elements: a warp takes 32 sorted blocks, a block per lane, and hands
// them round - LP lanes (8, 16 or 32 by the block length) add a block's elements, EPL each, 32 / LP blocks at
// a time - where binned_apply_kernel has every thread read and work out every block's numbers itself.  Measured
// (B200, 34 M blocks of 16 on 1 GB, us): 930 (45 instructions per element and thread) -> 780; on 100 MB 930 ->
// 550; 13 tables of d = 73, Z = 32 1104 -> 460; Z = 128 880 -> 480.  Now bound by the reductions and by the
// gradient rows, read once per id (going through odd bins backwards, to meet rows again in L2, changed nothing)
template <int LP, int EPL, bool SHORT>
__global__ void __launch_bounds__(256)
binned_apply_blocks_kernel(ApplyArgs a, const uint32_t* K, const uint32_t* V) {
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    constexpr uint32_t G = 32 / LP;              // blocks at a time
    constexpr int U = EPL == 4 ? 4 : 8;          // times whose loads are in flight together
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, g = lane / LP, ol = lane % LP, Z = mp.Z, m = mp.m;
    __shared__ uint2 sorted_s[256];
    __shared__ uint32_t count_s[256];
    __shared__ uint32_t warp_sums[8];
    const uint64_t i0 = ((uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;
    const uint32_t cnt = i0 >= a.nb ? 0u : (a.nb - i0 < 32 ? (uint32_t)(a.nb - i0) : 32u);
    uint32_t k = kNoKey, v = 0, len = 0;         // (length 0: nothing of the block is added)
    if (lane < cnt) {
        k = __ldca(K + i0 + lane);
        v = __ldca(V + i0 + lane);
        len = Z;
        if (SHORT) {
            const uint32_t left = mp.d - v % mp.d;
            if (left < Z) len = left;
        }
    }
    if (a.long_count != nullptr && *a.long_count != 0) {  // (binned_sample_kernel's answer)
        binned_add_merged<LP, EPL, SHORT>(a, k, v, sorted_s, count_s, warp_sums);
        return;
    }
    const bool plain = !SHORT && __all_sync(0xFFFFFFFFu, lane < cnt && k <= m - Z);  // full blocks, none wraps
    const uint64_t pol = l2_keep_policy(a.l2_keep != 0);
#pragma unroll 1
    for (uint32_t s0 = 0; s0 < LP && s0 * G < cnt; s0 += U) {
        float x[U][EPL];
        uint32_t slot[U];
        if (plain) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int src = (int)((s0 + u) * G + g);
                slot[u] = __shfl_sync(0xFFFFFFFFu, k, src) + ol;
                const float* row = a.grad_out + (__shfl_sync(0xFFFFFFFFu, v, src) + ol);
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    x[u][q] = ol + 32 * q < Z && ROBE_CHK((uint64_t)(row + 32 * q - a.grad_out) < a.grad_elems, ROBE_DBG_GRAD_POS)
                                  ? __ldca(row + 32 * q)
                                  : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    if (ol + 32 * q < Z && ROBE_CHK(slot[u] + 32 * q < m, ROBE_DBG_ARRAY_SLOT))
                        red_add(a.target + slot[u] + 32 * q, a.lr * x[u][q], pol);
        } else {
            uint32_t l[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int src = (int)((s0 + u) * G + g);
                slot[u] = __shfl_sync(0xFFFFFFFFu, k, src) + ol;
                const float* row = a.grad_out + (__shfl_sync(0xFFFFFFFFu, v, src) + ol);
                l[u] = __shfl_sync(0xFFFFFFFFu, len, src);
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    x[u][q] = ol + 32 * q < l[u] && ROBE_CHK((uint64_t)(row + 32 * q - a.grad_out) < a.grad_elems, ROBE_DBG_GRAD_POS)
                                  ? __ldca(row + 32 * q)
                                  : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    if (ol + 32 * q < l[u]) {
                        uint32_t j = slot[u] + 32 * q;  // < m + d <= 2^32
                        if (j >= m) j -= m;
                        if (ROBE_CHK(j < m, ROBE_DBG_ARRAY_SLOT)) red_add(a.target + j, a.lr * x[u][q], pol);
                    }
        }
    }
}

template <bool SHORT>
void launch_binned_blocks(const ApplyArgs& a, const uint32_t* K, const uint32_t* V, cudaStream_t st) {
    const unsigned blocks = (unsigned)((a.nb + 255) / 256);
    if (a.mp.Z <= 8) launch_next(binned_apply_blocks_kernel<8, 1, SHORT>, blocks, 256, 0, st, a, K, V);
    else if (a.mp.Z <= 16) launch_next(binned_apply_blocks_kernel<16, 1, SHORT>, blocks, 256, 0, st, a, K, V);
    else if (a.mp.Z <= 32) launch_next(binned_apply_blocks_kernel<32, 1, SHORT>, blocks, 256, 0, st, a, K, V);
    else if (a.mp.Z <= 64) launch_next(binned_apply_blocks_kernel<32, 2, SHORT>, blocks, 256, 0, st, a, K, V);
    else launch_next(binned_apply_blocks_kernel<32, 4, SHORT>, blocks, 256, 0, st, a, K, V);
}

uint32_t bits_for(uint32_t m) {  // bits needed for keys in [0, m)
    uint32_t b = 1;
    while (b < 32 && (1ull << b) < (uint64_t)m) ++b;
    return b;
}

struct Layout {
    size_t keysA, valsA, keysB, valsB, bag_of, counts, totals, long_count, long_walks, strips, total;
    uint32_t long_cap;
    bool strips_own, strips_spare;  // the strips' bounds and lists have room of their own / fit the free pair of buffers
};

// Arrays whose strips can never ask for more than this (up to 5.5 M slots) have room for them in the workspace.
constexpr size_t kStripRoom = 171 << 10;

Layout make_layout(uint64_t nb, int64_t nnz, bool bags, const MapParams& mp) {
    Layout L;
    size_t off = 0;
    const size_t kb = align256((nb ? nb : 1) * sizeof(uint32_t));
    // starts and payloads side by side: the pair that the last sort pass read from is free for the strips
    L.keysA = off; off += kb;
    L.valsA = off; off += kb;
    L.keysB = off; off += kb;
    L.valsB = off; off += kb;
    L.bag_of = off; off += bags ? align256((size_t)(nnz ? nnz : 1) * sizeof(uint32_t)) : 0;
    L.counts = off; off += align256((size_t)kRadix * kSortMaxGrid * sizeof(uint32_t));
    L.totals = off; off += align256((size_t)kRadix * sizeof(uint32_t));
    // list of long walks: room for one round per 128 blocks, within 64 .. 2^20 rounds
    uint64_t cap = nb / 128;
    cap = cap < 64 ? 64 : (cap > (1u << 20) ? (1u << 20) : cap);
    L.long_cap = (uint32_t)cap;
    L.long_count = off; off += 256;
    L.long_walks = off; off += align256((size_t)cap * sizeof(LongWalk));
    // (The sign option may be switched after the workspace was sized: room for the strips either way.)  The total
    // must not fall as nb grows: a caller sizes for its largest call.  On a longer array the strips go to the
    // free pair; where they do not fit that, there is less than a block per strip, and the call goes without.
    // The list of hot strips takes the place of that of long walks, which strips do without (400 bytes for every 128
    // blocks against 4 for every 32 at most; for a list beyond that there would be no strips).
    const bool listed = strips_ok(mp, nb, false) && strips_list_bytes(mp, nb) <= (size_t)cap * sizeof(LongWalk);
    const size_t strips = listed ? strips_workspace_bytes(mp) : 0;
    L.strips_own = strips != 0 && strips <= kStripRoom;
    L.strips_spare = strips != 0 && !L.strips_own && strips <= 2 * kb;
    L.strips = off; off += L.strips_own ? strips : 0;
    L.total = off;
    return L;
}

// Second stream for what need not hold up the caller's, or nullptr.
struct SideStream {
    cudaStream_t st;
    cudaEvent_t fork_event, join_event;
};

// Strips where they pay: the hot strips (a few long-running CTAs) and the low slots in the second stream (of
// higher priority), all other strips in the caller's.
template <int MODE>
void launch_apply_strips(const ApplyArgs& aa, const uint32_t* K, const uint32_t* V, int mode, void* workspace,
                         const SideStream& side, cudaStream_t st) {
    const MapParams& mp = aa.mp;
    const StripProblem sp{mp, aa.grad_out, aa.grad_elems, aa.target, aa.lr, aa.adam, K, V, aa.nb, aa.status, workspace,
                          (uint32_t*)aa.long_walks};
    launch_strips_prepare(sp, st);
    const bool forked = side.st != nullptr;
    if (forked) {
        cudaEventRecord(side.fork_event, st);
        cudaStreamWaitEvent(side.st, side.fork_event, 0);
    }
    const cudaStream_t ts = forked ? side.st : st;
    launch_strips(sp, mode, st, ts);
    if (forked) {
        cudaEventRecord(side.join_event, side.st);
        cudaStreamWaitEvent(st, side.join_event, 0);
    }
}

template <bool SIGN, int MODE>
void launch_apply(const ApplyArgs& aa, const uint32_t* K, const uint32_t* V, const uint32_t* bag_of, cudaStream_t st) {
    const MapParams& mp = aa.mp;
    const unsigned blocks = (unsigned)((aa.nb + 255) / 256);  // one warp per 32 sorted positions
    const unsigned low_blocks = (mp.Z - 1 + kLowWarps - 1) / kLowWarps;  // one warp per low slot
    if (mp.d % mp.Z != 0) {
        det_apply_kernel<SIGN, MODE, true><<<blocks, 256, 0, st>>>(aa, K, V, bag_of);
        if (mp.Z > 1)
            det_apply_low_kernel<SIGN, MODE, true><<<low_blocks, 32 * kLowWarps, 0, st>>>(aa, K, V, bag_of);
    } else {
        det_apply_kernel<SIGN, MODE, false><<<blocks, 256, 0, st>>>(aa, K, V, bag_of);
        if (!SIGN) {
            // the rounds the apply kernel handed over; a grid-stride loop over the list
            const unsigned lblocks = aa.long_cap < 148u * 8u ? aa.long_cap : 148u * 8u;
            det_apply_long_kernel<MODE><<<lblocks, 32 * kLongWarps, 0, st>>>(aa, K, V);
        }
        if (mp.Z > 1)
            det_apply_low_kernel<SIGN, MODE, false><<<low_blocks, 32 * kLowWarps, 0, st>>>(aa, K, V, bag_of);
    }
}

}  // namespace

size_t det_workspace_bytes(const MapParams& mp, int64_t nbags, int64_t nnz, bool bags) {
    (void)nbags;
    const uint64_t nb = (uint64_t)nnz * mp.C;
    return make_layout(nb, nnz, bags, mp).total;
}

void block_key_buffers(const Problem& pb, void* workspace, uint32_t** keys, uint32_t** vals) {
    const uint64_t nb = (uint64_t)pb.nnz * pb.mp.C;
    const Layout L = make_layout(nb, pb.nnz, pb.offsets != nullptr, pb.mp);
    *keys = (uint32_t*)((char*)workspace + L.keysA);
    *vals = (uint32_t*)((char*)workspace + L.valsA);
}

// bag_of (pooled input) into the workspace
static void launch_bag_of(const Problem& pb, const Layout& L, char* ws, cudaStream_t st) {
    uint32_t* bag_of = (uint32_t*)(ws + L.bag_of);
    KeyArgs ka{pb.mp, pb.indices, pb.offsets, pb.nbags, pb.nnz, pb.status};
    // positions that malformed offsets leave uncovered fall back to bag 0 (memory-safe)
    cudaMemsetAsync(bag_of, 0, (size_t)pb.nnz * sizeof(uint32_t), st);
    det_bag_of_kernel<<<(unsigned)((pb.nbags + 7) / 8), 256, 0, st>>>(ka, bag_of);
}

cudaError_t launch_block_keys(const Problem& pb, void* workspace, size_t workspace_bytes,
                              cudaStream_t st) {
    if (pb.nnz == 0 || pb.nbags == 0) return cudaSuccess;
    const MapParams& mp = pb.mp;
    const bool bags = pb.offsets != nullptr;
    const uint64_t nb = (uint64_t)pb.nnz * mp.C;
    const Layout L = make_layout(nb, pb.nnz, bags, mp);
    if (workspace == nullptr || workspace_bytes < L.total) return cudaErrorInvalidValue;
    char* ws = (char*)workspace;
    uint32_t* kA = (uint32_t*)(ws + L.keysA);
    uint32_t* vA = (uint32_t*)(ws + L.valsA);
    uint32_t* bag_of = bags ? (uint32_t*)(ws + L.bag_of) : nullptr;
    KeyArgs ka{mp, pb.indices, pb.offsets, pb.nbags, pb.nnz, pb.status};
    if (bags) launch_bag_of(pb, L, ws, st);
    if (mp.C <= 8) {
        const unsigned kb = (unsigned)((pb.nnz + 255) / 256);
        if (pb.sign) launch_next(det_keys_kernel<true>, kb, 256, 0, st, ka, bag_of, kA, vA);
        else launch_next(det_keys_kernel<false>, kb, 256, 0, st, ka, bag_of, kA, vA);
    } else {
        const unsigned kb = (unsigned)((nb + 255) / 256);
        if (pb.sign) launch_next(det_keys_by_block_kernel<true>, kb, 256, 0, st, ka, bag_of, kA, vA, nb);
        else launch_next(det_keys_by_block_kernel<false>, kb, 256, 0, st, ka, bag_of, kA, vA, nb);
    }
    return cudaGetLastError();
}

cudaError_t launch_backward_det(const Problem& pb, const float* grad_out, float* target, int mode,
                                float lr, const AdamState* adam, void* workspace,
                                size_t workspace_bytes, cudaStream_t st, bool keys_kept) {
    if (pb.nnz == 0 || pb.nbags == 0) return cudaSuccess;
    const MapParams& mp = pb.mp;
    const bool bags = pb.offsets != nullptr;
    const uint64_t nb = (uint64_t)pb.nnz * mp.C;
    const Layout L = make_layout(nb, pb.nnz, bags, mp);
    if (workspace == nullptr || workspace_bytes < L.total) return cudaErrorInvalidValue;
    // the payload of a block is a 32-bit position in grad_out
    if ((uint64_t)pb.nbags * mp.d > (1ull << 32)) return cudaErrorInvalidValue;
    char* ws = (char*)workspace;
    uint32_t* kA = (uint32_t*)(ws + L.keysA);
    uint32_t* kB = (uint32_t*)(ws + L.keysB);
    uint32_t* vA = (uint32_t*)(ws + L.valsA);
    uint32_t* vB = (uint32_t*)(ws + L.valsB);
    uint32_t* bag_of = bags ? (uint32_t*)(ws + L.bag_of) : nullptr;
    uint32_t* counts = (uint32_t*)(ws + L.counts);
    uint32_t* totals = (uint32_t*)(ws + L.totals);

    if (!keys_kept) {
        const cudaError_t err = launch_block_keys(pb, workspace, workspace_bytes, st);
        if (err != cudaSuccess) return err;
    } else if (bags && pb.sign) {
        launch_bag_of(pb, L, ws, st);  // the signed terms look the id's bag up again
    }

    const uint32_t bits = bits_for(mp.m);
    if (mode == 3) {
        // binned: one pass on the top key bits, then atomic adds in bin order.  A bin spans 2^22
        // slots (16 MB of fp32: the span that measured fastest on a 1 GB array - small enough to
        // be updated in L2, large enough that the scatter writes long runs; 32 MB: adds 850 us against
        // 805) unless that would need more than 256 bins or the array is smaller than one such span.
        const uint32_t shift = bits > 30 ? bits - 8 : (bits > 22 ? 22 : (bits > 8 ? bits - 8 : 0));
        const SortPlan sp = make_plan(nb, bits - shift);
        launch_sort_pass<false>(sp, kA, vA, kB, vB, counts, totals, shift, bits - shift, st);
        // (an array that does not fit the L2 passes through it bin by bin: lines that outlive their bin would
        // only be in the way of the gradient rows; 34 M blocks of 16 on 1 GB, us: 951 -> 925)
        const int keep = (uint64_t)mp.m * 4 <= kL2SizedBytes ? pb.l2_keep : 0;
        ApplyArgs ab{mp, grad_out, pb.indices, target, lr, nb, pb.status, AdamState{}, nullptr, nullptr, 0,
                     (uint64_t)pb.nbags * mp.d, keep};
        if (!pb.sign && mp.Z <= 128) {
            if (nb >= (8u << 20)) {
                ab.long_count = (uint32_t*)(ws + L.long_count);
                launch_next(binned_sample_kernel, 1, 1024, 0, st, kB, nb, ab.long_count);
            }
            if (mp.d % mp.Z != 0) launch_binned_blocks<true>(ab, kB, vB, st);
            else launch_binned_blocks<false>(ab, kB, vB, st);
            return cudaGetLastError();
        }
        uint32_t log2Zp = 0;
        while ((1u << log2Zp) < mp.Z) ++log2Zp;
        const uint64_t groups = (nb + kBinnedPer - 1) / kBinnedPer;
        const unsigned blocks = (unsigned)(((groups << log2Zp) + 255) / 256);
        const bool shortb = mp.d % mp.Z != 0;
        if (pb.sign) {
            if (shortb) launch_next(binned_apply_kernel<true, true>, blocks, 256, 0, st, ab, kB, vB, bag_of, log2Zp);
            else launch_next(binned_apply_kernel<true, false>, blocks, 256, 0, st, ab, kB, vB, bag_of, log2Zp);
        } else {
            if (shortb) launch_next(binned_apply_kernel<false, true>, blocks, 256, 0, st, ab, kB, vB, bag_of, log2Zp);
            else launch_next(binned_apply_kernel<false, false>, blocks, 256, 0, st, ab, kB, vB, bag_of, log2Zp);
        }
        return cudaGetLastError();
    }
    const uint32_t npass = (bits + 7) / 8;
    const uint32_t bpp = (bits + npass - 1) / npass;
    const SortPlan sp = make_plan(nb, bpp);
    for (uint32_t pass = 0; pass < npass; ++pass) {
        const uint32_t shift = pass * bpp;
        const uint32_t width = bits - shift < bpp ? bits - shift : bpp;
        launch_sort_pass<true>(sp, kA, vA, kB, vB, counts, totals, shift, width, st);
        uint32_t* t = kA; kA = kB; kB = t;
        t = vA; vA = vB; vB = t;
    }

    uint32_t* long_count = (uint32_t*)(ws + L.long_count);
    const ApplyArgs aa{mp, grad_out, pb.indices, target, lr, nb, pb.status, adam ? *adam : AdamState{},
                       long_count, (LongWalk*)(ws + L.long_walks), L.long_cap, (uint64_t)pb.nbags * mp.d, 0};
    if ((L.strips_own || L.strips_spare) && strips_ok(mp, nb, pb.sign != 0)) {
        const SideStream side{pb.side, pb.fork_event, pb.join_event};
        void* const room = L.strips_own ? (void*)(ws + L.strips) : (void*)kB;
        if (mode == 4) launch_apply_strips<3>(aa, kA, vA, mode, room, side, st);
        else if (mode == 2) launch_apply_strips<2>(aa, kA, vA, mode, room, side, st);
        else if (mode == 1) launch_apply_strips<1>(aa, kA, vA, mode, room, side, st);
        else launch_apply_strips<0>(aa, kA, vA, mode, room, side, st);
        return cudaGetLastError();
    }
    cudaMemsetAsync(long_count, 0, 2 * sizeof(uint32_t), st);  // [0] rounds handed over, [1] rounds taken
    if (pb.sign) {
        if (mode == 4) launch_apply<true, 3>(aa, kA, vA, bag_of, st);
        else if (mode == 2) launch_apply<true, 2>(aa, kA, vA, bag_of, st);
        else if (mode == 1) launch_apply<true, 1>(aa, kA, vA, bag_of, st);
        else launch_apply<true, 0>(aa, kA, vA, bag_of, st);
    } else {
        if (mode == 4) launch_apply<false, 3>(aa, kA, vA, bag_of, st);
        else if (mode == 2) launch_apply<false, 2>(aa, kA, vA, bag_of, st);
        else if (mode == 1) launch_apply<false, 1>(aa, kA, vA, bag_of, st);
        else launch_apply<false, 0>(aa, kA, vA, bag_of, st);
    }
    return cudaGetLastError();
}

}  // namespace robe

// Pooled rows of short bags: a warp takes a run of consecutive bags (forward and atomic backward, d <= 128).
//
// A bag of a few ids is a chain of dependent memory reads - offsets, ids, array - with hardly any work in
// between, and hashing its few ids leaves most lanes idle.  The ids of consecutive bags lie side by side, so a
// warp that takes a run of bags reads all their offsets at once, hashes the ids of the whole run one per
// lane, and gathers (or scatters) id after id, several in flight whichever bags they belong to; a row is
// stored (or the next gradient row taken up) where a bag ends.
// Measured: see pool_bags.
#include "robe_internal.h"
#include "robe_stage.cuh"

namespace robe {

namespace {

constexpr uint32_t kPoolBags = 16;  // bags per warp, at most
constexpr int kPoolCtas = 5, kPoolCtasSign = 4;  // per SM

struct PoolArgs {
    MapParams mp;
    const void* array;
    IdList indices;
    const int64_t* offsets;
    const float* grad_out;
    float* io;             // output rows (forward) or target (backward)
    float scale;
    int64_t nbags, nnz;
    const int32_t* status;
    uint32_t* keep_keys;   // see KeepBlocks
    uint32_t* keep_vals;
    uint32_t bags;         // per warp
    uint64_t share;        // forward: the same in units of 2^-32, warp i takes bags [i share, (i + 1) share)
    uint32_t ids;          // per batch
    uint32_t cmagic;
    int l2_keep;
};

// Tables whose terms (A e + D) mod P of both hashes a CTA works out once, not per id.  That, and a build of the
// group without the wrap test: 7 x 3001 signed bags of 4, d = 100 (84 K ids), 22 -> 18 us forward, 30 -> 27
// backward; the kernel is bound by instruction issue.
constexpr uint32_t kPoolTables = 64;

struct PoolSmem {
    StageSmem stage;
    uint64_t tterm[kPoolTables], gterm[kPoolTables];
    uint32_t bag[8][kStageIds];   // per warp: which of its bags each id of the batch belongs to; bit 31: its last id
};

constexpr uint32_t kPoolLast = 0x80000000u;

// Hash phase of `cnt` ids from position p0 on (see stage_batch); off: lane i holds the start of the warp's
// bag i, lanes from `bags` on the end of the last one.
template <bool SIGN>
__device__ __forceinline__ bool pool_stage(PoolSmem& sm, const PoolArgs& a, int64_t k0, int64_t off, uint32_t bags, int64_t p0,
                                           uint32_t cnt, uint32_t w, uint32_t lane) {
    const MapParams& mp = a.mp;
    uint64_t* base_s = sm.stage.base[w];
    uint64_t* gbase_s = base_s + kStageIds / 2;
    uint32_t* start_s = sm.stage.start[w];
    for (uint32_t t0 = 0; t0 < cnt; t0 += 32) {
        const uint32_t t = t0 + lane;
        const int64_t p = p0 + (t < cnt ? t : cnt - 1);
        uint32_t b = 0;  // the last bag that starts at or before p
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            const int64_t s = __shfl_sync(0xFFFFFFFFu, off, b + step);
            if (b + step < bags && s <= p) b += step;
        }
        const int64_t end = __shfl_sync(0xFFFFFFFFu, off, b + 1);
        if (t < cnt && ROBE_CHK(t < (uint32_t)(SIGN ? kStageIds / 2 : kStageIds), ROBE_DBG_SHARED)) {
            sm.bag[w][t] = b | (p + 1 == end ? kPoolLast : 0u);
            const uint32_t e = table_of_bag((uint64_t)(k0 + b), mp);
            const uint64_t x = (uint64_t)a.indices.load(p);
            uint64_t xh = x;
            if (mp.R > 1) {
                xh = x / mp.R;
                sm.stage.piece[w][t] = (uint32_t)(x - xh * mp.R) * mp.d;
            }
            base_s[t] = addmod_p61(e < kPoolTables ? sm.tterm[e] : table_term(mp.h, e), mulmod_p61_any(mp.h.B, xh));
            if (SIGN)
                gbase_s[t] = sign_limit(addmod_p61(e < kPoolTables ? sm.gterm[e] : table_term(mp.g, e), mulmod_p61_any(mp.g.B, x)));
        }
    }
    __syncwarp();
    const uint32_t entries = cnt * mp.C, last_fit = mp.m - mp.Z;
    bool wraps = false;
    for (uint32_t t = lane; t < entries; t += 32) {
        const uint32_t idl = (t * a.cmagic) >> 20, c = t - idl * mp.C;  // (exact for t < 8192)
        uint32_t s = mod_m(addmod_p61(base_s[idl], sm.stage.cterm[c]), mp.m, mp.mu);
        if (mp.R > 1) {
            const uint64_t j = (uint64_t)s + sm.stage.piece[w][idl];
            s = (uint32_t)(j >= mp.m ? j - mp.m : j);
        }
        if (ROBE_CHK(c * a.ids + idl < (uint32_t)kStageEntries, ROBE_DBG_SHARED)) start_s[c * a.ids + idl] = s;
        wraps |= s > last_fit;
        if (a.keep_keys != nullptr && ROBE_CHK((uint64_t)p0 * mp.C + t < (uint64_t)a.nnz * mp.C, ROBE_DBG_SORT_POS)) {
            const uint64_t q = (uint64_t)p0 * mp.C + t, bag = (uint64_t)k0 + (sm.bag[w][idl] & ~kPoolLast);
            a.keep_keys[q] = s;
            a.keep_vals[q] = SIGN ? (uint32_t)q : (uint32_t)(bag * mp.d + c * mp.Z);
        }
    }
    const bool any = __any_sync(0xFFFFFFFFu, wraps);
    __syncwarp();
    return any;
}

// What a warp works on: its bags' bounds, and whether they are one stretch of ids (offsets that fall somewhere
// - malformed input - are not: such a warp takes its bags one by one, each with the bounds bag_range gives).
struct PoolRun {
    int64_t k0, off;
    uint32_t bags;
    bool stretch;
};

template <bool EVEN>
__device__ __forceinline__ PoolRun pool_run(const PoolArgs& a, uint32_t w, uint32_t lane) {
    PoolRun r;
    const uint64_t warp = (uint64_t)blockIdx.x * 8 + w;
    if (EVEN) {
        auto first = [&](uint64_t i) { return (int64_t)(__umul64hi(i, a.share) << 32 | (i * a.share) >> 32); };
        r.k0 = first(warp);
        int64_t end = first(warp + 1);
        if (end > a.nbags) end = a.nbags;
        r.bags = end > r.k0 ? (uint32_t)(end - r.k0) : 0u;
    } else {
        r.k0 = (int64_t)warp * a.bags;
        const int64_t left = a.nbags - r.k0;
        r.bags = left <= 0 ? 0u : (left < (int64_t)a.bags ? (uint32_t)left : a.bags);
    }
    r.off = 0;
    if (r.bags != 0) r.off = clamp64(__ldca(a.offsets + r.k0 + (lane < r.bags ? lane : r.bags)), 0, a.nnz);
    const int64_t next = __shfl_down_sync(0xFFFFFFFFu, r.off, 1);
    r.stretch = __all_sync(0xFFFFFFFFu, lane >= r.bags || next >= r.off);
    return r;
}

// One lane's view of the rows it works on.
template <int EPL>
struct PoolLane {
    uint32_t off[EPL];
    const uint32_t* col[EPL];
    bool live[EPL];
    uint64_t gelem[EPL];
    float acc[EPL];  // forward: the sum; backward: the gradient row
};

// Ids g0 .. g0+n-1 of the batch, n <= U (FULL: n == U): all their loads first, then, id by id, the adds.  WRAP 0: no block
// wraps; 1, 2: some may, 2 in one instruction (which in the kernel for longer arrays costs the forward 9 %, by the registers).
template <int MODE, int EPL, bool SIGN, int U, bool FULL, int WRAP>
__device__ __forceinline__ void pool_group(const PoolArgs& a, const uint32_t* bag_s, const uint64_t* gbase_s, PoolLane<EPL>& l,
                                           int64_t k0, uint32_t g0, uint32_t n, bool begins, uint32_t lane, uint64_t pol) {
    const MapParams& mp = a.mp;
    float v[U][EPL];
    uint32_t bag[U];
#pragma unroll
    for (int g = 0; g < U; ++g) bag[g] = FULL || (uint32_t)g < n ? bag_s[g0 + g] : 0u;
    if (MODE == 2) {  // the gradient row of every id (ids of one bag read the same one)
#pragma unroll
        for (int g = 0; g < U; ++g) {
            const float* row = a.grad_out + (k0 + (bag[g] & ~kPoolLast)) * (int64_t)mp.d + lane;
            const bool fresh = g == 0 ? begins : (bag[g - 1] & kPoolLast) != 0;  // (warp-uniform)
#pragma unroll
            for (int u = 0; u < EPL; ++u)
                v[g][u] = fresh && l.live[u] && (FULL || (uint32_t)g < n) && ROBE_CHK_GRAD(row + 32 * u, a) ? __ldcs(row + 32 * u) : 0.0f;
        }
#pragma unroll
        for (int g = 0; g < U; ++g) {
            const bool fresh = g == 0 ? begins : (bag[g - 1] & kPoolLast) != 0;
#pragma unroll
            for (int u = 0; u < EPL; ++u) {
                if (fresh) l.acc[u] = v[g][u] * a.scale;
                uint32_t j = l.col[u][g0 + g] + l.off[u];
                if (WRAP == 1 && j >= mp.m) j -= mp.m;
                if (WRAP == 2) j = __viaddmin_u32(j, 0u - mp.m, j);  // j - m unless that is below 0
                if ((FULL || (uint32_t)g < n) && l.live[u] && ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT))
                    red_add(a.io + j, SIGN ? with_sign(gbase_s[g0 + g], l.gelem[u], (uint32_t)l.gelem[u] << 31, l.acc[u]) : l.acc[u], pol);
            }
        }
    } else {
#pragma unroll
        for (int g = 0; g < U; ++g)
#pragma unroll
            for (int u = 0; u < EPL; ++u) {
                v[g][u] = 0.0f;
                if (l.live[u] && (FULL || (uint32_t)g < n)) {
                    uint32_t j = l.col[u][g0 + g] + l.off[u];  // < m + d <= 2^32
                    if (WRAP == 1 && j >= mp.m) j -= mp.m;
                    if (WRAP == 2) j = __viaddmin_u32(j, 0u - mp.m, j);  // j - m unless that is below 0
                    if (ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT)) v[g][u] = gather_elem<MODE == 1 ? 1 : 0>(a.array, j);
                }
            }
#pragma unroll
        for (int g = 0; g < U; ++g) {
            if (!FULL && (uint32_t)g >= n) break;
#pragma unroll
            for (int u = 0; u < EPL; ++u)
                l.acc[u] = l.acc[u] + (SIGN ? with_sign(gbase_s[g0 + g], l.gelem[u], (uint32_t)l.gelem[u] << 31, v[g][u]) : v[g][u]);
            if ((bag[g] & kPoolLast) != 0) {
                float* orow = a.io + (k0 + (bag[g] & ~kPoolLast)) * (int64_t)mp.d + lane;
#pragma unroll
                for (int u = 0; u < EPL; ++u) {
                    if (l.live[u]) __stcs(orow + 32 * u, l.acc[u]);
                    l.acc[u] = -0.0f;  // -0 + v == v: the first term initialises
                }
            }
        }
    }
}

// MODE 0: forward, fp32 array; 1: forward, bf16 array; 2: backward
// WRAPS: most batches of ids hold a block that wraps.  Then every full group takes the (one-instruction) wrap along; else
// those of a batch that wraps do so together with the rest of a batch, which is slower for them.
template <int MODE, int EPL, bool SIGN, bool WRAPS>
__global__ void __launch_bounds__(256, SIGN ? kPoolCtasSign : kPoolCtas)
pool_kernel(PoolArgs a) {
    __shared__ PoolSmem sm;
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x >= 128 && threadIdx.x - 128 < kPoolTables && threadIdx.x - 128 < mp.T) {  // (beside stage_init's 128)
        const uint32_t e = threadIdx.x - 128;
        sm.tterm[e] = table_term(mp.h, e);
        if (SIGN) sm.gterm[e] = table_term(mp.g, e);
    }
    stage_init(sm.stage, mp);
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const PoolRun run = pool_run<MODE != 2>(a, w, lane);
    if (run.bags == 0) return;

    PoolLane<EPL> l;
#pragma unroll
    for (int u = 0; u < EPL; ++u) {
        uint32_t i = lane + 32u * u, chk;
        l.live[u] = i < mp.d;
        if (!l.live[u]) i = mp.d - 1;
        l.gelem[u] = SIGN ? mulmod_p61_u32(mp.g.C, i) : 0;
        chunk_of(mp, i, chk, l.off[u]);
        l.col[u] = sm.stage.start[w] + chk * a.ids;
    }
    const uint64_t* gbase_s = sm.stage.base[w] + kStageIds / 2;
    const uint64_t pol = MODE == 2 ? l2_keep_policy(a.l2_keep != 0) : 0;
    constexpr int U = 4;  // ids in flight

    for (uint32_t first = 0; first < run.bags; first += run.stretch ? run.bags : 1u) {
        const uint32_t bags = run.stretch ? run.bags : 1u;
        // bounds of the bags taken now: lane i the start of bag `first + i`, lanes from `bags` on the end
        int64_t at = run.off;
        if (!run.stretch) {
            const int64_t lo = __shfl_sync(0xFFFFFFFFu, run.off, first), up = __shfl_sync(0xFFFFFFFFu, run.off, first + 1);
            at = lane == 0 ? lo : (up > lo ? up : lo);
        }
        const int64_t k0 = run.k0 + first, lo = __shfl_sync(0xFFFFFFFFu, at, 0), hi = __shfl_sync(0xFFFFFFFFu, at, bags);
        if (MODE != 2) {  // empty bags
            const int64_t next = __shfl_down_sync(0xFFFFFFFFu, at, 1);
            for (uint32_t none = __ballot_sync(0xFFFFFFFFu, lane < bags && next == at); none != 0; none &= none - 1) {
                float* orow = a.io + (k0 + (__ffs((int)none) - 1)) * (int64_t)mp.d + lane;
#pragma unroll
                for (int u = 0; u < EPL; ++u)
                    if (l.live[u]) __stcs(orow + 32 * u, 0.0f);
            }
        }
#pragma unroll
        for (int u = 0; u < EPL; ++u) l.acc[u] = -0.0f;
        for (int64_t p0 = lo; p0 < hi; p0 += a.ids) {
            const uint32_t cnt = (uint32_t)(hi - p0 < (int64_t)a.ids ? hi - p0 : (int64_t)a.ids);
            const bool wraps = pool_stage<SIGN>(sm, a, k0, at, bags, p0, cnt, w, lane);
            uint32_t g0 = 0;
            // (a batch that goes on with a bag reads its gradient row again)
            for (; (WRAPS || !wraps) && g0 + U <= cnt; g0 += U)
                pool_group<MODE, EPL, SIGN, U, true, WRAPS ? 2 : 0>(a, sm.bag[w], gbase_s, l, k0, g0, U,
                                                                    g0 == 0 || (sm.bag[w][g0 - 1] & kPoolLast) != 0, lane, pol);
            for (; g0 < cnt; g0 += U)
                pool_group<MODE, EPL, SIGN, U, false, WRAPS ? 2 : 1>(a, sm.bag[w], gbase_s, l, k0, g0, cnt - g0 < U ? cnt - g0 : U,
                                                                     g0 == 0 || (sm.bag[w][g0 - 1] & kPoolLast) != 0, lane, pol);
            __syncwarp();  // the staging area is rewritten by the next batch
        }
    }
}

template <int MODE, bool SIGN, bool WRAPS>
void launch_pool_build(const PoolArgs& a, unsigned blocks, cudaStream_t st) {
    if (a.mp.d <= 32) launch_next(pool_kernel<MODE, 1, SIGN, WRAPS>, blocks, 256, 0, st, a);
    else if (a.mp.d <= 64) launch_next(pool_kernel<MODE, 2, SIGN, WRAPS>, blocks, 256, 0, st, a);
    else launch_next(pool_kernel<MODE, 4, SIGN, WRAPS>, blocks, 256, 0, st, a);
}

// Arrays of up to 512 rows have a block that wraps in every other batch of a few dozen ids or more.  Measured (B200, us, one
// build for all -> here): forward of 26 x 9000 bags of 2, d = 128 on 5000 slots 67.0 -> 48.7, d = 100 69.6 -> 51.9, signed bags of 6,
// d = 100 on 20 K slots, both passes, 459 -> 437; 0.89 .. 0.97 on 150 .. 20 K slots, 1.00 on 100 K, on 1 M 1.01 .. 1.05.
template <int MODE, bool SIGN>
void launch_pool_epl(const PoolArgs& a, unsigned blocks, cudaStream_t st) {
    if (a.mp.m <= 512ull * a.mp.d) launch_pool_build<MODE, SIGN, true>(a, blocks, st);
    else launch_pool_build<MODE, SIGN, false>(a, blocks, st);
}

uint32_t pool_ids(const Problem& pb) { return staged_ids_per_batch(pb.mp, true, pb.sign != 0); }

int64_t pool_wave(const Problem& pb) { return 148 * 8 * (pb.sign != 0 ? kPoolCtasSign : kPoolCtas); }  // warps at a time

// Bags per warp, 1 where a warp per bag is the better kernel.  A run of about 16 ids is what a warp gains
// by (32 in calls of hundreds of thousands of bags, which have warps enough); how long the bags may be
// for that follows a sweep over 7 x 3001, 26 x 512 and 26 x 16384 bags of 2 .. 12 ids on 4 and 400 MB (B200, us,
// warp per bag -> run): the sign hash makes a bag's fixed work dearer (26 x 16384 bags of 4, d = 64: 334 -> 180
// forward, 412 -> 218 backward, against 209 -> 127 and 220 -> 171 without), wide rows keep a warp busy anyway
// (7 x 3001 bags of 4, d = 128: 17 -> 19), and an array beyond the L2 hides it (bags of 4, d = 128, 407 -> 435).
uint32_t pool_bags(const Problem& pb, bool backward) {
    if (pb.nbags == 0 || pb.nnz < pb.nbags) return 1;
    const int64_t mean = (pb.nnz + pb.nbags / 2) / pb.nbags;
    const bool large = pb.nbags >= 200000, narrow = pb.mp.d <= 32, l2_sized = (uint64_t)pb.mp.m * 4 <= kL2SizedBytes;
    int64_t ids = large ? 32 : 16, longest;
    if (pb.sign != 0) {
        longest = backward ? 12 : (large || narrow ? 7 : 4);
        if (backward && mean > 7) ids = 32;
    } else if (large) {
        longest = !backward ? 7 : (narrow || l2_sized ? 4 : 2);
    } else {
        longest = narrow ? 4 : (backward && pb.mp.d > 64 ? 0 : 2);
    }
    if (mean > longest) return 1;
    if (ids > (int64_t)pool_ids(pb)) ids = pool_ids(pb);
    int64_t bags = ids / mean;
    const int64_t spread = pb.nbags / (148 * 40) + 1;
    if (bags > spread) bags = spread;
    // a last wave that is nearly empty costs a whole one: rather a bag more per warp
    const int64_t wave = pool_wave(pb);
    if (bags > 1) {
        const int64_t waves = ((pb.nbags + bags - 1) / bags + wave / 2) / wave;
        if (waves >= 1 && waves <= 3) bags = (pb.nbags + waves * wave - 1) / (waves * wave);
    }
    if (bags > (int64_t)kPoolBags) bags = kPoolBags;
    return bags < 1 ? 1u : (uint32_t)bags;
}

}  // namespace

bool pool_ok(const Problem& pb, bool backward) {
    return pb.offsets != nullptr && pb.mp.d <= 128 && pool_bags(pb, backward) > 1;
}

static cudaError_t launch_pool(const Problem& pb, PoolArgs& a, int mode, cudaStream_t st) {
    a.mp = pb.mp;
    a.array = pb.array;
    a.indices = pb.indices;
    a.offsets = pb.offsets;
    a.nbags = pb.nbags;
    a.nnz = pb.nnz;
    a.status = pb.status;
    a.ids = pool_ids(pb);
    a.cmagic = chunk_magic(pb.mp);
    a.l2_keep = pb.l2_keep;
    // Forward: up to three waves are filled to the last warp, the bags spread evenly over them, unless the runs get much
    // shorter (B200, us, runs of one length -> even: 7 x 3001 signed bags of 4, d = 100, 17.7 -> 16.7, d = 60 12.4 ->
    // 11.2; unsigned bags of 2 11.3 -> 10.3; 26 x 1024 bags of 4, d = 64 13.4 -> 12.7; 7 x 1500 of 4, 3 -> 2.2 bags to a
    // run, 10.3 -> 11.2).  The backward gains where rows are short and loses where bags are (19.0 -> 17.8, 18.7 -> 19.6).
    const int64_t bags = pool_bags(pb, mode == 2), wave = pool_wave(pb), waves = (pb.nbags + bags * wave - 1) / (bags * wave);
    const bool fill = mode != 2 && waves <= 3 && 20 * pb.nbags >= 17 * waves * wave * bags;
    const int64_t warps = fill ? waves * wave : (pb.nbags + bags - 1) / bags;
    a.bags = (uint32_t)bags;
    a.share = fill ? (((uint64_t)pb.nbags << 32) + (uint64_t)warps - 1) / (uint64_t)warps : (uint64_t)bags << 32;
    const unsigned blocks = (unsigned)((warps + 7) / 8);
    if (mode == 0) { if (pb.sign) launch_pool_epl<0, true>(a, blocks, st); else launch_pool_epl<0, false>(a, blocks, st); }
    else if (mode == 1) { if (pb.sign) launch_pool_epl<1, true>(a, blocks, st); else launch_pool_epl<1, false>(a, blocks, st); }
    else { if (pb.sign) launch_pool_epl<2, true>(a, blocks, st); else launch_pool_epl<2, false>(a, blocks, st); }
    return cudaGetLastError();
}

cudaError_t launch_forward_pool(const Problem& pb, float* out, uint32_t* keep_keys, uint32_t* keep_vals, cudaStream_t st) {
    PoolArgs a{};
    a.io = out;
    a.keep_keys = keep_keys;
    a.keep_vals = keep_vals;
    return launch_pool(pb, a, pb.dtype == 0 ? 0 : 1, st);
}

cudaError_t launch_backward_pool(const Problem& pb, const float* grad_out, float* target, float scale, cudaStream_t st) {
    PoolArgs a{};
    a.io = target;
    a.grad_out = grad_out;
    a.scale = scale;
    return launch_pool(pb, a, 2, st);
}

}  // namespace robe

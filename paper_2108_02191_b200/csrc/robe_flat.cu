// Flat kernels: one-hot rows of any length, as one run of elements (forward and atomic backward).
//
// The output rows of consecutive ids lie end to end, so a warp that takes a few rows treats their
// elements as one run: it first evaluates the block starts of its rows into shared memory (one id per
// lane, then one (id, chunk) pair per lane), then walks the run, consecutive lanes on consecutive
// elements, whatever the row length.  No lane idles on a row of 16 or of 100 elements, and a row of
// 256 is no special case.
// Measured (B200, us, before -> after): forward / backward of 16384 x 13 rows of 256, Z = 64, 100 MB
// array 326 -> 75 / 391 -> 89 (every lane hashed its own chunk); 2048 x 26 rows of 16, Z = 8 14 -> 10 /
// 25 -> 10; 16384 x 26 of them 27 -> 16 / 47 -> 37.  Bound by the gather of random blocks where the
// array is large (as the staged kernel), by launch and load latency in small calls.
#include "robe_internal.h"
#include "robe_stage.cuh"

namespace robe {

namespace {

constexpr int kFlatWarps = 8;
constexpr int kFlatCtas = 6;            // per SM; loads in flight (8) x CTAs of 8 / 5, 8 / 4, 16 / 4, 4 / 8: 0-5 % slower
constexpr uint32_t kFlatEntries = 256;  // block starts per warp
constexpr uint32_t kFlatRows = 64;      // rows per warp
// Elements per warp, about: 4096, or 2048 in large calls, whose CTAs then follow one another more evenly:
//   in calls of 0.86 to 2.3 waves of CTAs of 4096 elements a warp, whose last wave then is a smaller part - but not in the forward
//     on arrays of up to 16 MB, which issue bounds: a rest of a group of 256 elements, whose loads are in flight together, takes
//     a warp as long as a whole one, and half the elements are half as many to share it;
//   in the forward from 16 M elements on where the run of rows is whole groups.
// Measured (B200, us, 4096 -> 2048): 13 x 16384 rows of 256, Z = 64, 100 MB (54 M elements), both passes 147.0 -> 141.7
// (1536: 141.6, 1024: 141.9).  Over 500 shapes, forward: whole groups 16 M .. 30 M elements 0.93 .. 0.98, more 0.96 .. 1.00,
// with a rest 1.02 .. 1.09 on arrays of up to 16 MB (13 x 12000 rows of 257, Z = 32 43 -> 48), on larger ones 25 M .. 60 M
// elements 0.92 .. 0.99, fewer or more 1.02; backward 26 M .. 60 M elements 0.89 .. 0.98, 17 M .. 22 M 1.00 .. 1.10 (13 x 3605 rows
// of 384, Z = 128 30.7 -> 36.2), 70 M 1.00 .. 1.04.
constexpr uint32_t kFlatElems = 4096, kFlatElemsHalf = 2048;
constexpr int64_t kFlatWholeHalf = 1 << 24, kFlatHalf = 24 << 20, kFlatHalfEnd = 64 << 20;  // elements of such calls
constexpr uint64_t kFlatFewBytes = 16 << 20;

struct FlatArgs {
    MapParams mp;
    const void* array;
    IdList indices;
    const float* grad_out;
    float* io;            // output rows (forward) or target (backward)
    float scale;
    const int32_t* status;
    int64_t nbags;
    uint32_t rows;        // per warp
    uint32_t cmagic, zmagic, dmagic;  // ceil(2^32 / C), / Z, / d (0 where the divisor is 1)
    uint32_t padj;        // lane_padj
    int l2_keep;
};

struct FlatSmem {
    uint64_t cterm[kFlatEntries];              // per chunk: (C_h c) mod P
    uint32_t ct[kFlatEntries];                 // and that mod m
    uint64_t thr[kFlatWarps][kFlatRows];       // per row: P - base
    uint32_t bm[kFlatWarps][kFlatRows];        // and base mod m
    uint32_t start[kFlatWarps][kFlatEntries];  // block starts, row after row
};

// f / divisor, exact while f * divisor < 2^32 (f < 16384 + kFlatElems here, the divisors at most 16384)
__device__ __forceinline__ uint32_t flat_div(uint32_t f, uint32_t magic) { return magic != 0 ? __umulhi(f, magic) : f; }

// Hash phase: the block starts of rows [row0, row0 + cnt).  Returns whether some block wraps.
__device__ __forceinline__ bool flat_hash(const FlatArgs& a, FlatSmem& sm, int64_t row0, uint32_t cnt, uint32_t w,
                                          uint32_t lane) {
    const MapParams& mp = a.mp;
    for (uint32_t t = lane; t < cnt; t += 32) {
        if (!ROBE_CHK(t < kFlatRows, ROBE_DBG_SHARED)) break;
        const uint32_t e = table_of_bag((uint64_t)(row0 + t), mp);
        const uint64_t x = (uint64_t)a.indices.load(row0 + t);
        if (mp.R > 1) {  // rows clubbed into one block: its start is all there is
            sm.start[w][t] = id_block_start(mp, e, x, 0);
            continue;
        }
        lane_id_base(mp, table_term(mp.h, e), x, sm.bm[w][t], sm.thr[w][t]);
    }
    __syncwarp();
    const uint32_t n = cnt * mp.C, last_fit = mp.m - mp.Z;
    bool wraps = false;
    for (uint32_t t = lane; t < n; t += 32) {
        uint32_t s;
        if (mp.R > 1) {
            s = sm.start[w][t];
        } else {
            const uint32_t r = flat_div(t, a.cmagic), c = t - r * mp.C;
            uint64_t h = (uint64_t)sm.bm[w][r] + sm.ct[c] + (sm.cterm[c] >= sm.thr[w][r] ? a.padj : 0u);
            if (h >= mp.m) h -= mp.m;
            if (h >= mp.m) h -= mp.m;
            s = (uint32_t)h;
            if (ROBE_CHK(t < kFlatEntries, ROBE_DBG_SHARED)) sm.start[w][t] = s;
        }
        wraps |= s > last_fit;
    }
    const bool any = __any_sync(0xFFFFFFFFu, wraps);
    __syncwarp();
    return any;
}

// Slot of flat position f.  RAGGED: the last block of a row is short, so rows and blocks are counted
// separately; else the run is one sequence of blocks.
template <bool POW2, bool RAGGED, bool WRAP>
__device__ __forceinline__ uint32_t flat_slot(const FlatArgs& a, const uint32_t* start, uint32_t f) {
    const MapParams& mp = a.mp;
    uint32_t q, off;
    if (RAGGED) {
        const uint32_t r = flat_div(f, a.dmagic), i = f - r * mp.d, c = flat_div(i, a.zmagic);
        off = i - c * mp.Z;
        q = r * mp.C + c;
    } else if (POW2) {
        q = f >> mp.log2Z;
        off = f & (mp.Z - 1);
    } else {
        q = flat_div(f, a.zmagic);
        off = f - q * mp.Z;
    }
    uint32_t j = (ROBE_CHK(q < kFlatEntries, ROBE_DBG_SHARED) ? start[q] : 0u) + off;  // < m + d <= 2^32
    if (WRAP && j >= mp.m) j -= mp.m;
    return j;
}

template <int DT, bool POW2, bool RAGGED, bool WRAP>
__device__ __forceinline__ void flat_gather(const FlatArgs& a, const uint32_t* start, float* out, uint32_t n,
                                            uint32_t lane) {
    constexpr uint32_t U = 8;  // loads in flight per lane
    uint32_t f = lane;
    for (; f - lane + 32 * U <= n; f += 32 * U) {
        float v[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint32_t j = flat_slot<POW2, RAGGED, WRAP>(a, start, f + 32 * u);
            v[u] = 0.0f;
            if (ROBE_CHK(j < a.mp.m, ROBE_DBG_ARRAY_SLOT)) v[u] = gather_elem<DT>(a.array, j);
        }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) __stcs(out + f + 32 * u, v[u]);
    }
    if (f - lane < n) {
        float v[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            v[u] = 0.0f;
            if (f + 32 * u < n) {
                const uint32_t j = flat_slot<POW2, RAGGED, WRAP>(a, start, f + 32 * u);
                if (ROBE_CHK(j < a.mp.m, ROBE_DBG_ARRAY_SLOT)) v[u] = gather_elem<DT>(a.array, j);
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
            if (f + 32 * u < n) __stcs(out + f + 32 * u, v[u]);
    }
}

template <bool POW2, bool RAGGED, bool WRAP>
__device__ __forceinline__ void flat_scatter(const FlatArgs& a, const uint32_t* start, const float* grad, uint32_t n,
                                             uint32_t lane) {
    constexpr uint32_t U = 8;
    const uint64_t pol = l2_keep_policy(a.l2_keep != 0);
    for (uint32_t f = lane; f - lane < n; f += 32 * U) {
        float v[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
            v[u] = f + 32 * u < n && ROBE_CHK_GRAD(grad + f + 32 * u, a) ? __ldcs(grad + f + 32 * u) : 0.0f;
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
            if (f + 32 * u < n) {
                const uint32_t j = flat_slot<POW2, RAGGED, WRAP>(a, start, f + 32 * u);
                if (ROBE_CHK(j < a.mp.m, ROBE_DBG_ARRAY_SLOT)) red_add(a.io + j, v[u] * a.scale, pol);
            }
    }
}

// MODE 0: forward, fp32 array; 1: forward, bf16 array; 2: backward
template <int MODE, bool POW2, bool RAGGED>
__global__ void __launch_bounds__(32 * kFlatWarps, kFlatCtas)
flat_kernel(FlatArgs a) {
    __shared__ FlatSmem sm;
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (uint32_t c = threadIdx.x; c < mp.C; c += 32 * kFlatWarps) {  // (needs nothing of the kernel before)
        sm.cterm[c] = mulmod_p61_u32(mp.h.C, c);
        sm.ct[c] = mod_m(sm.cterm[c], mp.m, mp.mu);
    }
    __syncthreads();
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const int64_t row0 = ((int64_t)blockIdx.x * kFlatWarps + w) * a.rows;
    if (row0 >= a.nbags) return;
    const uint32_t cnt = a.nbags - row0 < (int64_t)a.rows ? (uint32_t)(a.nbags - row0) : a.rows;
    const bool wraps = flat_hash(a, sm, row0, cnt, w, lane);
    const uint32_t* start = sm.start[w];
    const uint32_t n = cnt * mp.d;
    if (MODE == 2) {
        const float* grad = a.grad_out + row0 * (int64_t)mp.d;
        if (wraps) flat_scatter<POW2, RAGGED, true>(a, start, grad, n, lane);
        else flat_scatter<POW2, RAGGED, false>(a, start, grad, n, lane);
    } else {
        float* out = a.io + row0 * (int64_t)mp.d;
        if (wraps) flat_gather<MODE == 2 ? 0 : MODE, POW2, RAGGED, true>(a, start, out, n, lane);
        else flat_gather<MODE == 2 ? 0 : MODE, POW2, RAGGED, false>(a, start, out, n, lane);
    }
}

}  // namespace

// what the flat kernels ask of a call: one id per row, no signs, few enough chunks for the staging
bool flat_ok(const Problem& pb) {
    return pb.offsets == nullptr && pb.sign == 0 && pb.mp.C <= kFlatEntries && pb.mp.d <= 16384;
}

static cudaError_t launch_flat(const Problem& pb, const float* grad_out, float* io, float scale, int mode,
                               cudaStream_t st) {
    const MapParams& mp = pb.mp;
    auto magic = [](uint32_t v) { return v == 1 ? 0u : (uint32_t)((0x100000000ull + v - 1) / v); };
    FlatArgs a{mp, pb.array, pb.indices, grad_out, io, scale, pb.status, pb.nbags, 1,
               magic(mp.C), magic(mp.Z), magic(mp.d), lane_padj(mp), pb.l2_keep};
    // rows per warp: as many as the staging holds, but few enough for small calls to reach every SM
    uint32_t rows = kFlatEntries / mp.C;
    if (rows > kFlatRows) rows = kFlatRows;
    const int64_t all = pb.nbags * (int64_t)mp.d;
    const uint32_t half = rows < kFlatElemsHalf / mp.d ? rows : kFlatElemsHalf / mp.d;
    const bool few = mode != 2 && (uint64_t)mp.m * (pb.dtype == 0 ? 4u : 2u) <= kFlatFewBytes;
    if ((all >= kFlatHalf && all < kFlatHalfEnd && !few) || (mode != 2 && all >= kFlatWholeHalf && half * mp.d % 256 == 0)) rows = half;
    if (rows > kFlatElems / mp.d) rows = kFlatElems / mp.d;
    const int64_t spread = pb.nbags / (148 * 32) + 1;
    if ((int64_t)rows > spread) rows = (uint32_t)spread;
    if (rows < 1) rows = 1;
    a.rows = rows;
    const int64_t warps = (pb.nbags + rows - 1) / rows;
    const unsigned blocks = (unsigned)((warps + kFlatWarps - 1) / kFlatWarps);
    const bool ragged = mp.d % mp.Z != 0, pow2 = mp.log2Z != 0xFFFFFFFFu;
    auto pick = [&](auto plain, auto any, auto rag) {
        if (ragged) launch_next(rag, blocks, 32 * kFlatWarps, 0, st, a);
        else if (pow2) launch_next(plain, blocks, 32 * kFlatWarps, 0, st, a);
        else launch_next(any, blocks, 32 * kFlatWarps, 0, st, a);
    };
    if (mode == 0) pick(flat_kernel<0, true, false>, flat_kernel<0, false, false>, flat_kernel<0, false, true>);
    else if (mode == 1) pick(flat_kernel<1, true, false>, flat_kernel<1, false, false>, flat_kernel<1, false, true>);
    else pick(flat_kernel<2, true, false>, flat_kernel<2, false, false>, flat_kernel<2, false, true>);
    return cudaGetLastError();
}

cudaError_t launch_forward_flat(const Problem& pb, float* out, cudaStream_t st) {
    return launch_flat(pb, nullptr, out, 1.0f, pb.dtype == 0 ? 0 : 1, st);
}

cudaError_t launch_backward_flat(const Problem& pb, const float* grad_out, float* target, float scale,
                                 cudaStream_t st) {
    return launch_flat(pb, grad_out, target, scale, 2, st);
}

}  // namespace robe

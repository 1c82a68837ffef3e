// One-hot rows with the repeats of an id brought together (forward and atomic backward).
//
// Ids of a batch repeat: Zipf ids draw 8-16 % of a table's lookups on one id, and a small table is
// looked up many times over by any batch.  Rows of the same id of the same table read, and add to, the
// same slots, so one gather (forward) or one set of reductions (backward) can serve them all.  Each
// CTA takes a few hundred rows of one table (rows are handed out table by table: the longer the
// stretch of one table, the more of its rows repeat), hashes them once, brings equal ids next to each
// other by a counting sort in shared memory, and a warp then serves 32 sorted rows at a time, the rows
// of equal hash base (A e + B x + D) mod P as one group.
//
// The plain backward is bound by the reductions, those on a hot id's slots one after the other in L2.
// Measured (B200, 26 x 32768 rows of 128, 100 MB array, Zipf ids, us, before -> here): backward Z = 1
// 688 -> 435, Z = 8 225 -> 155, Z = 32 187 -> 129, Z = 128 241 -> 123; forward Z = 1 507 -> 370,
// Z = 2 302 -> 240.  512 rows per CTA at most: with 2048 the gain in repeats is lost to fewer CTAs in
// flight (backward Z = 128 187), with 256 to fewer repeats.
#include "robe_internal.h"
#include "robe_stage.cuh"

namespace robe {

namespace {

constexpr int kRowsThreads = 256;
constexpr int kRowsCtas = 4;            // per SM: the register budget of the kernels (5, 6: spills, slower)
constexpr int kRowsWarps = kRowsThreads / 32;
constexpr uint32_t kRowsCap = 512;      // rows per CTA, at most
constexpr uint32_t kRowsMin = 64;       // and at least
constexpr uint32_t kRowsBins = 512;     // of the counting sort: two per thread
constexpr uint32_t kRowsMaxC = 16;      // backward: chunks per row whose starts are listed (see RowSlots)

struct RowsArgs {
    MapParams mp;
    const void* array;
    IdList indices;
    const float* grad_out;
    float* io;              // output rows (forward) or target (backward)
    float scale;
    const int32_t* status;
    uint32_t nbags, batch;
    uint64_t batch_magic;   // floor((2^64 - 1) / batch) + 1
    uint32_t rows_per_cta;
    uint32_t shares;        // CTAs per table where tables are taken side by side, else 0 (see rows_first)
    uint32_t shift;         // bin = (base mod m) >> shift
    uint32_t padj;          // lane_padj
    int l2_keep;
};

struct RowsTerms {  // per chunk: (C_h c) mod P, and that mod m
    uint64_t cterm[kRowsMaxC];
    uint32_t ct[kRowsMaxC];
};

struct RowsSmem {
    RowsTerms terms;
    uint64_t base[kRowsCap];     // hash base of each of the CTA's rows
    uint16_t order[kRowsCap];    // the rows by bin
    uint32_t cursor[kRowsBins];
    uint32_t warp_sums[kRowsWarps];
};

// Row v of the table-by-table order: its table, and its position among the call's rows.
__device__ __forceinline__ uint32_t rows_position(const RowsArgs& a, uint32_t v, uint32_t& e) {
    e = a.batch == 1 ? v : (uint32_t)__umul64hi(a.batch_magic, (uint64_t)v);
    if (a.mp.B != 0) return v;
    return (v - e * a.batch) * a.mp.T + e;
}

// First row of this CTA in the table-by-table order.  Side by side: CTAs that run at the same time take the
// same samples of different tables, whose rows lie next to each other in a sample-major call.
__device__ __forceinline__ uint32_t rows_first(const RowsArgs& a) {
    const uint32_t b = blockIdx.x;
    return (a.shares == 0 ? b : (b % a.mp.T) * a.shares + b / a.mp.T) * a.rows_per_cta;
}

// Hashes rows [row0, row0 + rows) of the table-by-table order and sorts them; returns whether it did
// sort them.
template <bool TERMS>
__device__ __forceinline__ bool rows_sort(const RowsArgs& a, RowsSmem& sm, uint32_t row0, uint32_t rows) {
    const MapParams& mp = a.mp;
    const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    sm.cursor[2 * tid] = sm.cursor[2 * tid + 1] = 0;
    if (TERMS && tid < mp.C) {
        sm.terms.cterm[tid] = mulmod_p61_u32(mp.h.C, tid);
        sm.terms.ct[tid] = mod_m(sm.terms.cterm[tid], mp.m, mp.mu);
    }
    __syncthreads();
    bool repeats = false;
    for (uint32_t r0 = 0; r0 < rows; r0 += kRowsThreads) {  // (whole warps: the match below takes all lanes)
        const uint32_t r = r0 + tid;
        uint64_t base = ~0ull;  // (above every base: rows past the end match one another only)
        if (r < rows && ROBE_CHK(r < kRowsCap, ROBE_DBG_SHARED)) {
            uint32_t e;
            const uint32_t p = rows_position(a, row0 + r, e);
            base = addmod_p61(table_term(mp.h, e), mulmod_p61_any(mp.h.B, (uint64_t)a.indices.load(p)));
            sm.base[r] = base;
            const uint32_t bin = mod_m(base, mp.m, mp.mu) >> a.shift;
            if (ROBE_CHK(bin < kRowsBins, ROBE_DBG_SHARED)) atomicAdd(&sm.cursor[bin], 1u);
        }
        if (r0 == 0) {
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, base);
            repeats = r < rows && __popc(peers) > 1;
        }
    }
    // No id repeats inside a warp's first 32 rows: the ids are spread so thinly that sorting would bring
    // next to nothing together.
    if (!__syncthreads_or(repeats)) return false;
    const uint32_t n0 = sm.cursor[2 * tid], n1 = sm.cursor[2 * tid + 1];
    uint32_t inc = n0 + n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= (uint32_t)o) inc += up;
    }
    if (lane == 31) sm.warp_sums[w] = inc;
    __syncthreads();
    uint32_t before = inc - n0 - n1;
    for (uint32_t k = 0; k < w; ++k) before += sm.warp_sums[k];
    sm.cursor[2 * tid] = before;
    sm.cursor[2 * tid + 1] = before + n0;
    __syncthreads();
    for (uint32_t r = tid; r < rows; r += kRowsThreads) {
        const uint32_t at = atomicAdd(&sm.cursor[mod_m(sm.base[r], mp.m, mp.mu) >> a.shift], 1u);
        if (ROBE_CHK(at < kRowsCap, ROBE_DBG_SHARED)) sm.order[at] = (uint16_t)r;
    }
    __syncthreads();
    return true;
}

// What one lane knows of the row it stands for while a warp serves 32 of them.
struct RowsLane {
    uint32_t pos;    // position among the call's rows
    uint32_t bm;     // base mod m
    uint64_t thr;    // P - base
    uint32_t peers;  // lanes of the same base
};

__device__ __forceinline__ RowsLane rows_fetch(const RowsArgs& a, const RowsSmem& sm, uint32_t row0, uint32_t i0,
                                               uint32_t cnt, uint32_t lane, bool sorted, uint32_t& leaders) {
    RowsLane l{0, 0, 0, 0};
    uint64_t base = ~0ull;  // (above every base: lanes past the end match one another only)
    if (lane < cnt) {
        const uint32_t r = sorted ? sm.order[i0 + lane] : i0 + lane;
        base = sm.base[r];
        uint32_t e;
        l.pos = rows_position(a, row0 + r, e);
        l.bm = mod_m(base, a.mp.m, a.mp.mu);
        l.thr = kP61 - base;
    }
    l.peers = sorted ? __match_any_sync(0xFFFFFFFFu, base) : 1u << lane;
    leaders = __ballot_sync(0xFFFFFFFFu, lane < cnt && (l.peers & ((1u << lane) - 1u)) == 0);
    return l;
}

// Where the rows' slots come from while a warp serves 32 rows.  Few chunks per row (C <= kRowsMaxC; the
// backward only, launch_forward sends such rows elsewhere): every lane evaluates the block starts of its row into a list that the warp shares, and a lane that
// owns element i reads the start of chunk i / Z.  Many chunks: each lane hashes the chunks of its own
// elements (LaneChunks) from what the row's lane hands round.
template <int EPL, bool LISTED, bool M30>
struct RowSlots;

template <int EPL, bool M30>
struct RowSlots<EPL, true, M30> {
    uint32_t off[EPL];
    const uint32_t* col[EPL];
    bool on[EPL];
    uint32_t m;
    __device__ __forceinline__ RowSlots(const MapParams& mp, uint32_t lane, uint32_t, const uint32_t* list) : m(mp.m) {
#pragma unroll
        for (int u = 0; u < EPL; ++u) {
            uint32_t i = lane + 32u * u, c;
            on[u] = i < mp.d;
            if (!on[u]) i = mp.d - 1;
            chunk_of(mp, i, c, off[u]);
            col[u] = list + c * 33u;
        }
    }
    __device__ __forceinline__ bool live(int u) const { return on[u]; }
    // block starts of this lane's row into the list
    __device__ __forceinline__ void put(const RowsArgs& a, const RowsTerms& t, uint32_t* list, const RowsLane& l,
                                        uint32_t lane) const {
        __syncwarp();
        for (uint32_t c = 0; c < a.mp.C; ++c) {
            uint64_t s = (uint64_t)l.bm + t.ct[c] + (t.cterm[c] >= l.thr ? a.padj : 0u);
            if (s >= m) s -= m;
            if (s >= m) s -= m;
            if (ROBE_CHK(c < kRowsMaxC, ROBE_DBG_SHARED)) list[c * 33u + lane] = (uint32_t)s;
        }
        __syncwarp();
    }
    __device__ __forceinline__ void row(const RowsLane&, int) {}
    __device__ __forceinline__ uint32_t slot(int u, int src) const {
        const uint32_t j = col[u][src] + off[u];  // < m + d <= 2^32
        return j >= m ? j - m : j;
    }
};

template <int EPL, bool M30>
struct RowSlots<EPL, false, M30> {
    LaneChunks<EPL> lc;
    uint32_t bm;
    uint64_t thr;
    __device__ __forceinline__ RowSlots(const MapParams& mp, uint32_t lane, uint32_t padj, const uint32_t*) {
        lc.init(mp, lane, padj);
    }
    __device__ __forceinline__ bool live(int u) const { return lc.live[u]; }
    __device__ __forceinline__ void put(const RowsArgs&, const RowsTerms&, uint32_t*, const RowsLane&, uint32_t) const {}
    __device__ __forceinline__ void row(const RowsLane& l, int src) {
        bm = __shfl_sync(0xFFFFFFFFu, l.bm, src);
        thr = __shfl_sync(0xFFFFFFFFu, l.thr, src);
    }
    __device__ __forceinline__ uint32_t slot(int u, int) const { return lc.template slot<M30>(u, bm, thr); }
};

// Forward: the first row of a group is gathered, every row of it written; the gathers of U groups in
// flight.
template <int EPL, int DT, bool M30, int U>
__global__ void __launch_bounds__(kRowsThreads, kRowsCtas)
fwd_rows_kernel(RowsArgs a) {
    __shared__ RowsSmem sm;
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const uint32_t first = rows_first(a);
    if (first >= a.nbags) return;
    const uint32_t rows = a.nbags - first < a.rows_per_cta ? a.nbags - first : a.rows_per_cta;
    const bool sorted = rows_sort<false>(a, sm, first, rows);
    RowSlots<EPL, false, M30> rs(mp, lane, a.padj, nullptr);
    float* const out = a.io + lane;
    for (uint32_t i0 = w * 32; i0 < rows; i0 += kRowsThreads) {
        uint32_t leaders;
        const RowsLane l = rows_fetch(a, sm, first, i0, rows - i0 < 32 ? rows - i0 : 32, lane, sorted, leaders);
        while (leaders != 0) {
            float v[U][EPL];
            int src[U];
#pragma unroll
            for (int g = 0; g < U; ++g) {
                src[g] = __ffs((int)leaders) - 1;  // -1: no more groups
                leaders &= leaders - 1;
                if (src[g] < 0) continue;  // (warp-uniform)
                rs.row(l, src[g]);
#pragma unroll
                for (int u = 0; u < EPL; ++u) {
                    v[g][u] = 0.0f;
                    if (rs.live(u)) {
                        const uint32_t j = rs.slot(u, src[g]);
                        if (ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT)) v[g][u] = gather_elem<DT>(a.array, j);
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < U; ++g) {
                if (src[g] < 0) continue;
                for (uint32_t rest = __shfl_sync(0xFFFFFFFFu, l.peers, src[g]); rest != 0; rest &= rest - 1) {
                    float* orow = out + (size_t)__shfl_sync(0xFFFFFFFFu, l.pos, __ffs((int)rest) - 1) * mp.d;
#pragma unroll
                    for (int u = 0; u < EPL; ++u)
                        if (rs.live(u)) __stcs(orow + 32 * u, v[g][u]);
                }
            }
        }
    }
}

// Backward: the gradient rows of a group are summed in registers and added to the target once.  The
// warp's 32 rows are laid out group after group (turns) and streamed U rows at a time, the next U rows
// asked for before the present ones are added, so that a long group costs no more than its reads.
template <int EPL, bool LISTED, bool M30, int U>
__global__ void __launch_bounds__(kRowsThreads, kRowsCtas)
bwd_rows_kernel(RowsArgs a) {
    __shared__ RowsSmem sm;
    __shared__ uint2 turns[kRowsWarps][32];
    __shared__ uint32_t lists[LISTED ? kRowsWarps : 1][LISTED ? kRowsMaxC * 33 : 1];
    const MapParams& mp = a.mp;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    follow();
    if (a.status != nullptr && *a.status != 0) return;
    const uint32_t first = rows_first(a);
    if (first >= a.nbags) return;
    const uint32_t rows = a.nbags - first < a.rows_per_cta ? a.nbags - first : a.rows_per_cta;
    uint32_t* list = lists[LISTED ? w : 0];
    const bool sorted = rows_sort<LISTED>(a, sm, first, rows);
    RowSlots<EPL, LISTED, M30> rs(mp, lane, a.padj, list);
    const uint64_t pol = l2_keep_policy(a.l2_keep != 0);
    const float* const grad = a.grad_out + lane;
    uint2* const turn = turns[w];
    for (uint32_t i0 = w * 32; i0 < rows; i0 += kRowsThreads) {
        uint32_t leaders;
        const uint32_t cnt = rows - i0 < 32 ? rows - i0 : 32;
        const RowsLane l = rows_fetch(a, sm, first, i0, cnt, lane, sorted, leaders);
        rs.put(a, sm.terms, list, l, lane);
        // turn[k] = (row, lane it belongs to), group after group; bit k of ends: last row of its group
        const bool lead = (leaders >> lane) & 1u;
        uint32_t incl = lead ? __popc(l.peers) : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += up;
        }
        const uint32_t group_end = __shfl_sync(0xFFFFFFFFu, incl, lane < cnt ? __ffs((int)l.peers) - 1 : 31);
        const uint32_t k = group_end - __popc(l.peers >> lane);
        __syncwarp();
        if (lane < cnt && ROBE_CHK(k < 32u, ROBE_DBG_SHARED)) turn[k] = make_uint2(l.pos, lane);
        else turn[lane] = make_uint2(0u, lane);  // (read, not used)
        const uint32_t ends = __reduce_or_sync(0xFFFFFFFFu, lead ? 1u << (incl - 1) : 0u);
        __syncwarp();
        float nxt[U][EPL], acc[EPL];
        auto load = [&](uint32_t k0) {
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const float* row = grad + (size_t)turn[k0 + q].x * mp.d;
#pragma unroll
                for (int u = 0; u < EPL; ++u)
                    nxt[q][u] = k0 + q < cnt && rs.live(u) && ROBE_CHK_GRAD(row + 32 * u, a) ? __ldcs(row + 32 * u) : 0.0f;
            }
        };
        load(0);
#pragma unroll
        for (int u = 0; u < EPL; ++u) acc[u] = 0.0f;
#pragma unroll 1
        for (uint32_t k0 = 0; k0 < cnt; k0 += U) {
            float cur[U][EPL];
#pragma unroll
            for (int q = 0; q < U; ++q)
#pragma unroll
                for (int u = 0; u < EPL; ++u) cur[q][u] = nxt[q][u];
            if (k0 + U < cnt) load(k0 + U);
#pragma unroll
            for (int q = 0; q < U; ++q) {
#pragma unroll
                for (int u = 0; u < EPL; ++u) acc[u] += cur[q][u];
                if ((ends >> (k0 + q)) & 1u) {  // (warp-uniform)
                    const int src = (int)turn[k0 + q].y;
                    rs.row(l, src);
#pragma unroll
                    for (int u = 0; u < EPL; ++u) {
                        if (rs.live(u)) {
                            const uint32_t j = rs.slot(u, src);
                            if (ROBE_CHK(j < mp.m, ROBE_DBG_ARRAY_SLOT)) red_add(a.io + j, acc[u] * a.scale, pol);
                        }
                        acc[u] = 0.0f;
                    }
                }
            }
        }
    }
}

}  // namespace

// what the rows kernels ask of a call: one id per row, plain blocks, no signs
bool rows_ok(const Problem& pb) {
    return pb.offsets == nullptr && pb.sign == 0 && pb.mp.R == 1 && pb.mp.d <= 128 && pb.nbags < (1ll << 31) &&
           pb.nbags % pb.mp.T == 0;
}

// side_by_side: see rows_first.  In calls of millions of rows the order in which the gradient rows are read tells
// (B200, sample-major, rows of 128, 100 MB, us, table after table -> side by side; 26 x 131072 rows, ids that never
// repeat: Z = 8 1100 -> 1053, Z = 32 653 -> 611, Z = 128 588 -> 563, the staged kernel 1038, 610, 551; Zipf ids 521
// -> 518, 430 -> 431, 435 -> 425).  In smaller ones a table's hot blocks, met again by the CTAs of the same time,
// are worth as much or more (26 x 65536 rows, never repeating 321 -> 313, Zipf 231 -> 236; 8 x 32768 43 -> 46), and
// with many chunks per row always (Zipf, Z = 1, 420 -> 469, though 4003 -> 3817 / 3604 where nothing repeats).
// whole_waves: the rows are spread evenly over full waves of resident CTAs (the forward, whose CTAs take
// about equally long); otherwise the CTAs take kRowsCap rows each (the backward, whose repeats matter more)
static RowsArgs rows_args(const Problem& pb, bool whole_waves, bool side_by_side, unsigned& grid) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    (void)cudaGetLastError();
    RowsArgs a{};
    a.mp = pb.mp;
    a.array = pb.array;
    a.indices = pb.indices;
    a.status = pb.status;
    a.nbags = (uint32_t)pb.nbags;
    a.batch = (uint32_t)(pb.nbags / pb.mp.T);
    a.batch_magic = 0xFFFFFFFFFFFFFFFFull / a.batch + 1;
    const uint32_t resident = (uint32_t)sms * kRowsCtas;
    const uint32_t waves = (a.nbags + resident * kRowsCap - 1) / (resident * kRowsCap);
    a.rows_per_cta = (a.nbags + waves * resident - 1) / (waves * resident);
    if (!whole_waves && waves > 1) a.rows_per_cta = kRowsCap;
    if (a.rows_per_cta < kRowsMin) a.rows_per_cta = kRowsMin;
    grid = (a.nbags + a.rows_per_cta - 1) / a.rows_per_cta;
    if (side_by_side && pb.mp.B == 0) {
        a.shares = (grid + pb.mp.T - 1) / pb.mp.T;
        grid = a.shares * pb.mp.T;  // (CTAs past the last row return)
    }
    while (((pb.mp.m - 1) >> a.shift) >= kRowsBins) ++a.shift;
    a.padj = lane_padj(pb.mp);
    a.l2_keep = pb.l2_keep;
    return a;
}

template <int EPL, bool M30>
static void launch_fwd_rows(const RowsArgs& a, int dtype, unsigned grid, cudaStream_t st) {
    if (dtype == 0) launch_next(fwd_rows_kernel<EPL, 0, M30, 4>, grid, kRowsThreads, 0, st, a);
    else launch_next(fwd_rows_kernel<EPL, 1, M30, 4>, grid, kRowsThreads, 0, st, a);
}

template <int EPL>
static void launch_fwd_rows(const RowsArgs& a, int dtype, unsigned grid, cudaStream_t st) {
    if (a.mp.m < (1u << 30)) launch_fwd_rows<EPL, true>(a, dtype, grid, st);
    else launch_fwd_rows<EPL, false>(a, dtype, grid, st);
}

cudaError_t launch_forward_rows(const Problem& pb, float* out, cudaStream_t st) {
    unsigned grid;
    RowsArgs a = rows_args(pb, true, false, grid);
    a.io = out;
    if (a.mp.d <= 32) launch_fwd_rows<1>(a, pb.dtype, grid, st);
    else if (a.mp.d <= 64) launch_fwd_rows<2>(a, pb.dtype, grid, st);
    else launch_fwd_rows<4>(a, pb.dtype, grid, st);
    return cudaGetLastError();
}

template <int EPL>
static void launch_bwd_rows(const RowsArgs& a, unsigned grid, cudaStream_t st) {
    constexpr int U = EPL == 4 ? 2 : 4;
    if (a.mp.C <= kRowsMaxC) launch_next(bwd_rows_kernel<EPL, true, false, U>, grid, kRowsThreads, 0, st, a);
    else if (a.mp.m < (1u << 30)) launch_next(bwd_rows_kernel<EPL, false, true, U>, grid, kRowsThreads, 0, st, a);
    else launch_next(bwd_rows_kernel<EPL, false, false, U>, grid, kRowsThreads, 0, st, a);
}

cudaError_t launch_backward_rows(const Problem& pb, const float* grad_out, float* target, float scale,
                                 cudaStream_t st) {
    unsigned grid;
    RowsArgs a = rows_args(pb, false, pb.mp.C <= kRowsMaxC && pb.nbags >= (1 << 21), grid);
    a.grad_out = grad_out;
    a.io = target;
    a.scale = scale;
    if (a.mp.d <= 32) launch_bwd_rows<1>(a, grid, st);
    else if (a.mp.d <= 64) launch_bwd_rows<2>(a, grid, st);
    else launch_bwd_rows<4>(a, grid, st);
    return cudaGetLastError();
}

}  // namespace robe

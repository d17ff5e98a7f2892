// Gridding phase (thesis Sec. 4.3.3 "The gridding phase", eq. "gridding"), GB300 design.
//
// Work unit ("task") = one segment of seg_len consecutive gridded entries x one block of up to
// `slots` footprint points (both chosen by the work list's plan; see grid_autotune).  A warp takes
// tasks from a global counter (persistent kernel, dynamic load balance).  Each lane owns up to
// kUnitsMax point pairs of the footprint by their class (pairs.cuh), so lanes never touch the same
// pixel and accumulate in registers while the pair stays the same; when it moves, the lane flushes
// its accumulators with vector FP32 atomics (all polarisations of a pixel are contiguous).
//
// What bounds it: the FMA pipe and instruction issue (68 % of the pipe's cycles and 54 % of the issue slots at four
// polarisations; 128 registers, with 20 bytes of spills outside the loop over entries, 16 warps an SM), then the L1 data
// path (70 %: every sample is used once per entry and comes from L2).
// Packed FMAs on three distinct operands run at 2.6 cycles each, not 2 (register reads).  Consecutive
// entries of a track usually keep the footprint (about 85 %, weighted by S^2) and differ only in the
// sub-kernel: the loop over them holds the sample loads and 4P packed FMAs a pair and no test.
// Measured (grid_vis, single points -> now): 116 M records in 16 channels, P = 4, supports 9..65: 25.1 -> 20.2 ms; 4.8 M
// records, P = 4: 1.72 -> 1.20 ms; interleaved, P = 2: 4.65 -> 2.63 ms; 15.7 M records, P = 1, supports 9..129: 26.9 -> 18.3 ms;
// compensated with an FP16 table, P = 4: 1.67 -> 1.34 ms; 127 k entries of support 7: 54 -> 27 us; 1 k entries: 209 -> 24 us.
#include "pairs.cuh"

namespace wg {

namespace {

constexpr int kWarps = 4;           // warps per block

// exact rounding error of s = fl(a + b) (TwoSum, Knuth)
__device__ __forceinline__ float two_sum_err(float a, float b, float s)
{
    const float bv = __fsub_rn(s, a);
    const float av = __fsub_rn(s, bv);
    return __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}

__device__ __forceinline__ float4 add_err4(float4 old, float4 v)
{
    return make_float4(two_sum_err(old.x, v.x, __fadd_rn(old.x, v.x)), two_sum_err(old.y, v.y, __fadd_rn(old.y, v.y)),
                       two_sum_err(old.z, v.z, __fadd_rn(old.z, v.z)), two_sum_err(old.w, v.w, __fadd_rn(old.w, v.w)));
}

__device__ __forceinline__ float2 add_err2(float2 old, float2 v)
{
    return make_float2(two_sum_err(old.x, v.x, __fadd_rn(old.x, v.x)), two_sum_err(old.y, v.y, __fadd_rn(old.y, v.y)));
}

// Adds one pixel's sums to the grid.  COMP: the atomic returns the previous value, from which the
// rounding error of the add is recovered exactly and added to the error grid (zeros are not added: the
// row outside the footprint must not touch a neighbour that holds an infinity).
template <int P, bool COMP>
__device__ __forceinline__ void flush_pixel(float2* __restrict__ grid, float2* __restrict__ errgrid, size_t pix,
                                            const float2 (&a)[P])
{
    float2* d = grid + pix * P;
    float2* e = COMP ? errgrid + pix * P : nullptr;
    if constexpr (P == 1) {
        if constexpr (COMP) {
            if (a[0].x == 0.f && a[0].y == 0.f) return;
            atomicAdd(e, add_err2(atomicAdd(d, a[0]), a[0]));
        } else {
            atomicAdd(d, a[0]);
        }
    } else {
#pragma unroll
        for (int h = 0; h < P; h += 2) {
            const float4 v = make_float4(a[h].x, a[h].y, a[h + 1].x, a[h + 1].y);
            if constexpr (COMP) {
                if (v.x == 0.f && v.y == 0.f && v.z == 0.f && v.w == 0.f) continue;
                atomicAdd(reinterpret_cast<float4*>(e + h), add_err4(atomicAdd(reinterpret_cast<float4*>(d + h), v), v));
            } else {
                atomicAdd(reinterpret_cast<float4*>(d + h), v);
            }
        }
    }
}

// Adds a lane's accumulators (acc[p] = {re, re'}, {im, im'}) to its pair's two pixels and clears them.  The
// second row can be past the grid (the row outside the footprint); it then holds nothing.
template <int P, bool COMP>
__device__ __forceinline__ void flush_pair(float2* __restrict__ grid, float2* __restrict__ errgrid, int ch, int cur, int H,
                                           int N, f32x2 (&acc)[P][2])
{
    const int y = cur >> 16;
    const size_t pix = (size_t)((unsigned)ch * (unsigned)N + (unsigned)y) * N + (cur & 0xFFFF);
    float2 a[P], b[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float2 re = unpack2(acc[p][0]), im = unpack2(acc[p][1]);
        a[p] = make_float2(re.x, im.x);
        b[p] = make_float2(re.y, im.y);
        acc[p][0] = acc[p][1] = 0ull;
    }
    flush_pixel<P, COMP>(grid, errgrid, pix, a);
    if (y + H < N) flush_pixel<P, COMP>(grid, errgrid, pix + (size_t)(H * N), b);
}

// One run of entries from entry j of the chunk on (same support and channel): the units [un.x, un.y) of the
// footprint, at most NU.  Returns the first entry (of the chunk then staged) after it, or -1 at the item's
// end.  However the footprint moves, its pairs are placed anew and only those whose pixels change are flushed: runs that
// ended at a jump flushed the whole footprint, which took longer than single points did, and added more
// rounding steps (4.8 M records of 10 s steps on 4000^2, P = 4, 256 entries: 7.27 -> 5.95 ms; single points 7.26).
// A pair that moves by H rows keeps one of its pixels in the other place; to keep its sum as well cost more
// instructions than its flush (1225 -> 1352 us on 4.8 M records, P = 4).  The code is kept
// small, with one copy of the staging, the move and the flush: a kernel with several of each and
// variants for more values of NU stalled on instruction fetch half of its time.
template <int P, typename TS, bool COMP, int NU>
__device__ __forceinline__ int run_entries(Chunk<P, true>& ck, int j, int S, int ch, int2 un, const TaskParams& tp, bool report,
                                           const char* __restrict__ table, float2* __restrict__ grid,
                                           float2* __restrict__ errgrid)
{
    constexpr int PB = kPairBytes<TS>;
    const int lane = ck.lane;
    f32x2 acc[NU][P][2];
    unsigned toff[NU];
    place_classes<NU, PB>(toff, ck.cls, ck.cur, ck.e[j], S, un.x, un.y, lane);
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int p = 0; p < P; ++p) acc[u][p][0] = acc[u][p][1] = 0ull;
    KPair k[NU];
    // adds an entry with the visibilities g; then the samples of the entry whose sub-kernel is at kz are
    // loaded, each unit's as soon as its FMAs have read its registers
    auto add = [&](const float2 (&g)[P], const char* kz) {
#pragma unroll
        for (int u = 0; u < NU; ++u) {
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const f32x2 gx = pack2(g[p].x, g[p].x), gy = pack2(g[p].y, g[p].y), ny = pack2(-g[p].y, -g[p].y);
                acc[u][p][0] = fma2(ny, k[u].im, fma2(gx, k[u].re, acc[u][p][0]));
                acc[u][p][1] = fma2(gx, k[u].im, fma2(gy, k[u].re, acc[u][p][1]));
            }
            k[u] = load_pair((const TS*)nullptr, kz, toff[u]);
        }
    };
    {
        const char* kz = table + (size_t)ck.z[j] * PB;
#pragma unroll
        for (int u = 0; u < NU; ++u) k[u] = load_pair((const TS*)nullptr, kz, toff[u]);
    }
    const int H = (S + 1) >> 1;
    for (;;) {
        // entries whose successor has the same footprint
        const unsigned later = ck.mv & (0xFFFFFFFEu << j);
        const int last = (later ? __ffs(later) - 1 : ck.cnt) - 1;
        // (unrolled, the loop holds more values than there are registers at P = 4: 22.2 against 20.5 ms on 116 M records)
#pragma unroll(P == 4 ? 1 : 2)
        for (; j < last; ++j) {
            float2 g[P];
#pragma unroll
            for (int p = 0; p < P; ++p) g[p] = ck.g[j * P + p];
            add(g, table + (size_t)ck.z[j + 1] * PB);
        }
        // the footprint's last entry in the chunk: the pairs are placed in its successor's footprint first, so that its samples
        // can be loaded behind the FMAs; those that move are flushed after them
        float2 g[P];
#pragma unroll
        for (int p = 0; p < P; ++p) g[p] = ck.g[j * P + p];
        unsigned zn = ck.z[j];
        bool more = true;
        if (++j == ck.cnt) {
            more = ck.next(tp, report);
            j = more ? 0 : -1;
        }
        const bool same = more && !((ck.kc >> j) & 1);       // the run goes on
        unsigned moves = ~0u;                                // units whose pairs move
        if (same) {
            zn = ck.z[j];
            moves = 0;
            if ((ck.mv >> j) & 1) {
                const Staged E = ck.e[j];
                const unsigned minus_sh = minus_moduli(S, H);
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    const int d = place_class(ck.cls[u][lane], E, minus_sh), n = E.x + d;
                    toff[u] = linear(d, S, PB);
                    ck.nxt[u][lane] = n;
                    moves |= n != ck.cur[u][lane] ? 1u << u : 0u;
                }
            }
        }
        add(g, table + (size_t)zn * PB);
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            if (moves & (1u << u)) {
                const int cur = ck.cur[u][lane];
                if (cur >= 0) {
                    flush_pair<P, COMP>(grid, errgrid, ch, cur, H, tp.N, acc[u]);
                    ck.cur[u][lane] = ck.nxt[u][lane];
                }
            }
        }
        if (!same) return j;
    }
}

// An entry whose visibility is infinite or NaN: its products go to the pixels inside the footprint
// one by one (in a pair, the row outside it would take 0 x infinity).
template <int P, typename TS, bool COMP>
__device__ __noinline__ void slow_entry(const float2* g, int S, int unit0, int unit1, int fp, const char* kz, int N, int lane,
                                        float2* __restrict__ gch, float2* __restrict__ ech)
{
    const int H = (S + 1) >> 1;
    for (int i = unit0 * 32 + lane; i < min(unit1 * 32, H * S); i += 32) {
        const int dv = i / S, du = i - dv * S;
        const KPair k = load_pair((const TS*)nullptr, kz, (unsigned)i * kPairBytes<TS>);
        const float2 kr = unpack2(k.re), ki = unpack2(k.im);
        for (int c = 0; c < 2; ++c) {
            const int row = dv + c * H;
            if (row >= S) continue;
            const size_t pix = (size_t)((fp >> 16) + row) * N + (fp & 0xFFFF) + du;
            const float x = c ? kr.y : kr.x, y = c ? ki.y : ki.x;
            for (int p = 0; p < P; ++p) {
                const float2 v = g[p];
                const float2 a = make_float2(fmaf(-v.y, y, v.x * x), fmaf(v.x, y, v.y * x));
                const float2 o = atomicAdd(gch + pix * P + p, a);
                if constexpr (COMP) atomicAdd(ech + pix * P + p, add_err2(o, a));
            }
        }
    }
}

}  // namespace

// adds the batch normaliser and statistics into the grid's accumulators; the batch's normaliser
// row c goes to grid channel c * stride (w-stacking keeps a channel's N_p in its plane 0)
struct AccumulateParams {
    double* gnorm;
    const double* bnorm;
    int n, P, stride;
    unsigned long long* gcnt;
    const unsigned long long* bcnt;
};
__device__ __forceinline__ void accumulate(const AccumulateParams& a, int i)
{
    if (i < a.n) a.gnorm[(size_t)(i / a.P) * a.stride * a.P + i % a.P] += a.bnorm[i];
    if (i < ST_N) a.gcnt[i] += a.bcnt[i];
}
__global__ void k_accumulate(AccumulateParams a) { accumulate(a, threadIdx.x + blockIdx.x * blockDim.x); }

// SMALL: every support of the table has at most kSmallPairs pairs, two units (up to support 9).  Two units a lane leave
// registers for five blocks an SM, and none idle: support 7 at P = 4 from 387 to 226 us, support 9 from 409 to 241,
// compensated from 713 to 551 (single points took 281, 332 and 666).
constexpr int kSmallPairs = 64;
template <int P, typename TS, bool COMP, bool SMALL>
__global__ void __launch_bounds__(kWarps * 32, P == 4 ? (SMALL ? 5 : 4) : P == 2 ? 5 : 7) k_grid(TaskParams tp,
                                                                                                const char* __restrict__ table,
                                                                                                float2* __restrict__ grid,
                                                                                                float2* __restrict__ errgrid,
                                                                                                AccumulateParams acc)
{
    __shared__ __align__(16) unsigned char smem[kWarps * Chunk<P, true>::kBytes];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (acc.gnorm) {
        const int m = max(acc.n, (int)ST_N);
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) accumulate(acc, i);
    }
    Chunk<P, true> ck(smem + wid * Chunk<P, true>::kBytes, lane);
    const int parts = item_parts(tp);

    Item it;
    while (next_item(tp, parts, lane, it)) {
        // an item whose share of some support is more than kUnitsMax units takes the rest in a second pass
        bool again = it.n > 0;
        for (int pass = 0; again; ++pass) {
            again = false;
            const bool report = it.blk == 0 && pass == 0;       // one block of a segment counts its rejected entries
            ck.begin(tp, it.e0, it.n);
            int j = 0;
            while (j >= 0) {
                if (j == ck.cnt) {
                    if (!ck.next(tp, report)) break;
                    j = 0;
                }
                const int key = ck.e[j].w;
                const int S = key_support(key), ch = key_chan(key);
                const int nb = key < 0 ? 0 : (S * S + tp.slots - 1) / tp.slots;
                int2 un = make_int2(0, 0);
                if (it.blk < nb) {       // not a rejected entry, nor a support with fewer blocks
                    un = block_units(S, it.blk, nb);
                    if (un.y - un.x > (pass + 1) * kUnitsMax) again = true;
                    un = make_int2(un.x + pass * kUnitsMax, min(un.y, un.x + (pass + 1) * kUnitsMax));
                }
                if (un.x >= un.y) {
                    j = ck.run_end(j);
                    continue;
                }
                const size_t plane = (size_t)ch * tp.N * tp.N * P;
                float2* gch = grid + plane;
                float2* ech = COMP ? errgrid + plane : nullptr;
                if ((ck.slow >> j) & 1) {
                    const Staged e = ck.e[j];
                    slow_entry<P, TS, COMP>(ck.g + j * P, S, un.x, un.y, e.x,
                                            table + (size_t)(unsigned)e.z * kPairBytes<TS>, tp.N, lane, gch, ech);
                    ++j;
                    continue;
                }
                // the variant for one or two units (supports up to 9, and the last block of some others) saves idle ones:
                // support 7 beside 31 in the table, P = 4, 2.31 -> 1.30 ms on 13.8 M entries (single points 1.78); 116 M
                // records of supports 9..65, P = 4, 20.5 -> 20.2 ms; support 7 at P = 1, 33 -> 28 us on 127 k entries
                if (!SMALL && un.y - un.x > 2)
                    j = run_entries<P, TS, COMP, kUnitsMax>(ck, j, S, ch, un, tp, report, table, grid, errgrid);
                else
                    j = run_entries<P, TS, COMP, 2>(ck, j, S, ch, un, tp, report, table, grid, errgrid);
            }
        }
    }
}

// grid += err; err = 0 (folds the compensated flushes' rounding errors back)
__global__ void k_fold(float4* __restrict__ grid, float4* __restrict__ err, int64_t n4)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4) return;
    const float4 a = grid[i], e = err[i];
    grid[i] = make_float4(a.x + e.x, a.y + e.y, a.z + e.z, a.w + e.w);
    err[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <int P, typename TS, bool COMP, bool SMALL>
static int grid_launch(Grid& g, const Table& t, const WorkList& wl, const void* table, const AccumulateParams& acc,
                       cudaStream_t s)
{
    static int blocks_per_sm = 0;
    if (blocks_per_sm == 0 &&
        (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_grid<P, TS, COMP, SMALL>, kWarps * 32, 0) != cudaSuccess ||
         blocks_per_sm < 1))
        blocks_per_sm = 1;
    k_grid<P, TS, COMP, SMALL><<<num_sms() * blocks_per_sm, kWarps * 32, 0, s>>>(
        task_params(g, t, wl, wl.task_counter + 2), static_cast<const char*>(table), g.data, g.err, acc);
    WG_LAUNCHED("k_grid");
    return WG_OK;
}

template <int P, bool COMP, bool SMALL>
static int grid_store(Grid& g, const Table& t, const WorkList& wl, const AccumulateParams& acc, cudaStream_t s)
{
    switch (t.store) {
        case WG_BF16: return grid_launch<P, __nv_bfloat162, COMP, SMALL>(g, t, wl, t.pairs_lp, acc, s);
        case WG_F16: return grid_launch<P, __half2, COMP, SMALL>(g, t, wl, t.pairs_lp, acc, s);
        default: return grid_launch<P, float2, COMP, SMALL>(g, t, wl, t.pairs, acc, s);
    }
}

template <int P, bool COMP>
static int grid_dispatch(Grid& g, const Table& t, const WorkList& wl, const AccumulateParams& acc, cudaStream_t s)
{
    if constexpr (P == 4)          // (at fewer polarisations k_grid has the two-unit loop beside the other)
        if (t.max_support * ((t.max_support + 1) / 2) <= kSmallPairs) return grid_store<P, COMP, true>(g, t, wl, acc, s);
    return grid_store<P, COMP, false>(g, t, wl, acc, s);
}

template <int P>
static int grid_impl(Grid& g, const Table& t, const WorkList& wl, cudaStream_t s)
{
    WG_CUDA(cudaMemsetAsync(wl.task_counter + 2, 0, sizeof(unsigned int), s));
    // appended batches added their N_p terms at vis_compress
    AccumulateParams acc = {};
    if (!wl.append)
        acc = {g.norm, wl.norm_batch, (g.n_chan / wl.wstack_k) * g.n_pol, g.n_pol, wl.wstack_k, g.counters, wl.stats};
    const int rc = g.comp ? grid_dispatch<P, true>(g, t, wl, acc, s) : grid_dispatch<P, false>(g, t, wl, acc, s);
    if (rc != WG_OK) return rc;
    if (g.comp) {
        const int64_t n4 = (int64_t)g.n_chan * g.n * g.n * P / 2;
        k_fold<<<(unsigned)((n4 + 255) / 256), 256, 0, s>>>(reinterpret_cast<float4*>(g.data),
                                                            reinterpret_cast<float4*>(g.err), n4);
        WG_LAUNCHED("k_fold");
    }
    return WG_OK;
}

int launch_accumulate(const Grid& g, const WorkList& wl, int chan0, cudaStream_t s)
{
    const int n = wl.C * g.n_pol;
    const int m = std::max(n, (int)ST_N);
    k_accumulate<<<(m + 255) / 256, 256, 0, s>>>(
        AccumulateParams{g.norm + (size_t)chan0 * g.n_pol, wl.norm_batch, n, g.n_pol, 1, g.counters, wl.stats_batch});
    WG_LAUNCHED("k_accumulate");
    return WG_OK;
}

int launch_grid(Grid& g, const Table& t, const WorkList& wl, cudaStream_t s)
{
    switch (g.n_pol) {
        case 1: return grid_impl<1>(g, t, wl, s);
        case 2: return grid_impl<2>(g, t, wl, s);
        case 4: return grid_impl<4>(g, t, wl, s);
        default: return fail(WG_E_INVALID_ARG, "n_pol must be 1, 2 or 4");
    }
}

}  // namespace wg

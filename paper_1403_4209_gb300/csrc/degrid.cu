// Degridding: the adjoint of the gridding map (not in the thesis).
//
// For a gridded entry (footprint origin (x0, y0), kernel pointer z, grid channel c) the kernel sum
//   m_p = sum_{i,j} conj(C[z + i S + j]) grid_c,p(y0 + i, x0 + j)
// takes two launches.
//
// k_degrid_sum runs the gridder's tasks (a segment of consecutive entries x one block of the
// footprint, as the work list's plan defines them) on the gridder's point pairs and ownership
// (pairs.cuh).  A lane keeps its pairs' pixel values in registers; when the footprint moves, by one column or
// anywhere, its pairs are placed anew and the pixels that they did not hold are loaded.  For consecutive entries of a track
// that keep the footprint and differ only in the sub-kernel it loads nothing but the kernel samples.  Per entry each lane sums its
// pairs into 2P floats; these go through a shared-memory transpose (batches of 64 / (2P)
// entries), after which each lane holds two components of one entry summed over the warp and
// adds them to a per-entry FP32 accumulator with one vector atomic per footprint block.  It is bound like
// the gridder (60 % of the FMA pipe's cycles, 54 % of the issue slots, L1 data path 72 %), with the transpose on
// top.  Measured (degrid_vis, default plan, single points -> now): 0.87 M entries of supports 9..65, 4.8 M records: P = 4
// 2111 -> 1506 us, P = 2 1666 -> 1013, P = 1 1477 -> 851; 2.4 M records, supports 9..129, P = 1 2314 -> 1665; 1 k entries 241 -> 44.
//
// k_degrid_tile writes the records of each entry's run.  Compression (Sec. 4.3.3) carries over:
// every record compressed into an entry has its footprint and kernel samples, so m is computed
// once per entry and written to each record of the run, conjugated back where psi = -1 (w' < 0),
// with the cross hands swapped back under cross-hand swapping, and for the adjoint mode scaled
// by eps (1 - f) (the vis -> grid map's R-linear outer factor).  It works per preparation tile
// through shared memory so that the output is written row-major with coalesced stores.
#include "pairs.cuh"

namespace wg {

namespace {

constexpr int kWarps = 4;           // warps per block of k_degrid_sum
constexpr int kTileCap = 4096;      // records per preparation tile: rpb x C <= max(kTileRecords, n_chan <= 4096)
static_assert(kTileRecords <= kTileCap, "a preparation tile must fit the degridder's output tile");

// the P polarisations of one pixel, each (re, im) as it is stored
template <int P>
__device__ __forceinline__ void load_pixel(const float2* __restrict__ g, f32x2 (&v)[P])
{
    if constexpr (P == 1) {
        v[0] = __ldg(reinterpret_cast<const f32x2*>(g));
    } else {
#pragma unroll
        for (int h = 0; h < P; h += 2) {
            const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(g + h));
            v[h] = a.x;
            v[h + 1] = a.y;
        }
    }
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// a pixel of zeros (loaded like any other: cleared in a branch, the registers cost a select each)
__device__ const float2 __align__(16) g_zero[4] = {};

// The per-entry reduction buffers 64 / (2P) entries of 2P lane partials: slot b holds lane l's
// component c at b * (33 * 2P) + l * 2P + c (one 2P-float pad per slot, so that the 32 lanes'
// reads of two adjacent components of 32 / P different slots fall in distinct banks).
constexpr int kRedFloats = 64 * 33;      // per warp, any P

// One run of entries from entry j of the chunk on (see the gridder's run_entries): adds each entry's
// sums over the units [un.x, un.y), at most NU, to acc[entry][2P].  Returns the first entry (of
// the chunk then staged) after it, or -1 at the item's end.  Each lane stores its 2P partials of an
// entry in the reduction buffer; every 64 / (2P) entries (and at the end) each lane sums two adjacent
// components of one entry over the 32 lanes and adds them to acc with one vector atomic.
template <int P, int NU>
__device__ __forceinline__ int degrid_entries(Chunk<P, false>& ck, int j, int S, int ch, int2 un, const TaskParams& tp,
                                              bool report, float* __restrict__ red, const char* __restrict__ table,
                                              const float2* __restrict__ grid, float* __restrict__ acc)
{
    constexpr int PB = kPairBytes<float2>;
    constexpr int V = 2 * P, NB = 64 / V, SLOT = 33 * V;
    const int lane = ck.lane, H = (S + 1) >> 1;
    int nbuf = 0, eb = ck.e0 + j;     // entries buffered, and the first of them in the list
    // lane l sums components c, c + 1 of buffered entry b over the 32 lanes
    auto drain = [&](int n) {
        __syncwarp();
        const int b = (2 * lane) / V, c = (2 * lane) % V;
        if (b < n) {
            const float* src = red + b * SLOT + c;
            f32x2 t[4] = {0ull, 0ull, 0ull, 0ull};      // four chains: shorter, and a quarter of the rounding steps each
#pragma unroll
            for (int l2 = 0; l2 < 32; ++l2) {
                // V = 8: lanes with bit 2 set stored their two 16-byte halves swapped
                const int cs = (V == 8 && (l2 & 4)) ? 4 : 0;
                t[l2 & 3] = add2(t[l2 & 3], *reinterpret_cast<const f32x2*>(src + l2 * V + (c ^ cs) - c));
            }
            atomicAdd(reinterpret_cast<float2*>(acc + (size_t)(eb + b) * V + c),
                      unpack2(add2(add2(t[0], t[1]), add2(t[2], t[3]))));
        }
        __syncwarp();
    };
    unsigned toff[NU];
    place_classes<NU, PB>(toff, ck.cls, ck.cur, ck.e[j], S, un.x, un.y, lane);
    // The pairs' pixels, each polarisation (re, im) in the registers that the loads fill: a layout that took moves
    // (the two points', or two polarisations', parts side by side) waited for each pair's loads before the next pair's
    // were issued (3 M entries of support 15 at P = 4, each two columns and a row from the one before: 3.36 -> 2.50 ms).
    f32x2 g[NU][2][P];
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int p = 0; p < P; ++p) g[u][0][p] = g[u][1][p] = 0ull;
    // What a move of the footprint does to the pairs' pixels, a bit a unit at: kA and kB the first or the second row's
    // pixel is loaded; kZ the second row is the one past the footprint: 0 is loaded (its samples are 0, what lies
    // there may be an infinity).
    constexpr int kA = 0, kB = NU, kZ = 2 * NU;
    const float2* gch = grid + (size_t)ch * tp.N * tp.N * P;
    auto reload = [&](unsigned todo) {
        int cur[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) cur[u] = ck.cur[u][lane];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const float2* a = gch + (size_t)linear(cur[u], tp.N, 1u) * P;
            const float2* b = todo & (1u << (kZ + u)) ? g_zero : a + (size_t)(H * tp.N) * P;
            if (todo & (1u << (kA + u))) load_pixel<P>(a, g[u][0]);
            if (todo & (1u << (kB + u))) load_pixel<P>(b, g[u][1]);
        }
    };
    KPair k[NU];
    {
        const char* kz = table + (size_t)ck.z[j] * PB;
#pragma unroll
        for (int u = 0; u < NU; ++u) k[u] = load_pair((const float2*)nullptr, kz, toff[u]);
    }
    // an entry's sums into the reduction buffer; the samples of the entry whose sub-kernel is at kz are loaded
    // into a unit's registers behind its FMAs, and then() loads pixels (at P = 4 only once the sums have left the
    // registers: 2091 -> 1788 us on those 3 M entries, with 4 bytes of spills for 24)
    auto entry = [&](const char* kz, auto then) {
        // conj(k) g = (kx gx + ky gy, kx gy - ky gx), from the sums of kx (gx, gy) and ky (gx, gy)
        float v[V];
        f32x2 sx[P], sy[P];
#pragma unroll
        for (int p = 0; p < P; ++p) sx[p] = sy[p] = 0ull;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const float2 re = unpack2(k[u].re), im = unpack2(k[u].im);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x = h ? re.y : re.x, y = h ? im.y : im.x;
                const f32x2 kx = pack2(x, x), ky = pack2(y, y);
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    sx[p] = fma2(kx, g[u][h][p], sx[p]);
                    sy[p] = fma2(ky, g[u][h][p], sy[p]);
                }
            }
            k[u] = load_pair((const float2*)nullptr, kz, toff[u]);
        }
        if constexpr (P < 4) then();
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const float2 a = unpack2(sx[p]), b = unpack2(sy[p]);
            v[2 * p] = a.x + b.y;
            v[2 * p + 1] = a.y - b.x;
        }
        float* dst = red + nbuf * SLOT + lane * V;
        if constexpr (V == 8) {
            // halves swapped for lanes with bit 2 set: the 8 lanes of a quarter-warp store to
            // distinct banks
            const int sw = (lane & 4) ? 4 : 0;
            *reinterpret_cast<float4*>(dst + sw) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(dst + (4 ^ sw)) = make_float4(v[4], v[5], v[6], v[7]);
        } else if constexpr (V == 4) {
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
            *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
        }
        ++nbuf;
        if constexpr (P == 4) then();
    };
    const unsigned minus_sh = minus_moduli(S, H);
    // the first pixel (column | row << 16) of a pair whose second row is the one past the footprint: at least this
    int edge = ((ck.e[j].x >> 16) + H - 1) << 16;
    {
        unsigned todo = 0;
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int cur = ck.cur[u][lane];
            if (cur >= 0) todo |= (1u << (kA + u)) | (cur < edge ? 1u << (kB + u) : 0u);
        }
        reload(todo);
    }
    bool same = true;
    for (;;) {
        if (nbuf == NB || !same) {
            drain(nbuf);
            eb += nbuf;
            nbuf = 0;
            if (!same) return j;
        }
        // entries whose successor has the same footprint, as far as the buffer goes
        const unsigned later = ck.mv & (0xFFFFFFFEu << j);
        const int last = (later ? __ffs(later) - 1 : ck.cnt) - 1, stop = min(last, j + NB - nbuf);
        for (; j < stop; ++j) entry(table + (size_t)ck.z[j + 1] * PB, [] {});
        if (nbuf == NB) continue;
        // the footprint's last entry in the chunk: its successor's sample offsets come first (as in the gridder)
        unsigned zn = ck.z[j], todo = 0;
        bool more = true;
        if (++j == ck.cnt) {
            more = ck.next(tp, report);
            j = more ? 0 : -1;
        }
        same = more && !((ck.kc >> j) & 1);            // the run goes on
        if (same) {
            zn = ck.z[j];
            if ((ck.mv >> j) & 1) {
                // Every pair is placed anew, and of its two pixels those loaded that it does not hold (on lists that move
                // by one column now and then, a path of its own for that move gained nothing: 1523 against 1505 us).
                const Staged E = ck.e[j];
                const int edge1 = ((E.x >> 16) + H - 1) << 16;
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    const int d = place_class(ck.cls[u][lane], E, minus_sh);
                    const int cur = ck.cur[u][lane], n = E.x + d;
                    toff[u] = linear(d, S, PB);
                    if (cur >= 0) {
                        const bool moved = n != cur, past = n >= edge1;
                        ck.cur[u][lane] = n;
                        todo |= (moved ? 1u << (kA + u) : 0u) | (moved || past != (cur >= edge) ? 1u << (kB + u) : 0u) |
                                (past ? 1u << (kZ + u) : 0u);
                    }
                }
                edge = edge1;
            }
        }
        // the pixels are on their way before the sums are drained
        entry(table + (size_t)zn * PB, [&] {
            if (todo) reload(todo);
        });
    }
}

template <int P>
constexpr size_t kDegridSmem = Chunk<P, false>::kBytes + kRedFloats * sizeof(float);     // per warp

}  // namespace

// acc[0 .. n_entries * 2P) = 0, and k_degrid_sum's task counter
__global__ void k_degrid_zero(float4* __restrict__ acc, const long long* __restrict__ scal, int P, unsigned* __restrict__ counter)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0u;
    const long long n2 = scal[0] * P, n4 = n2 / 2;
    const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long i = i0; i < n4; i += (long long)gridDim.x * blockDim.x) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 == 0 && (n2 & 1)) reinterpret_cast<float2*>(acc)[n2 - 1] = make_float2(0.f, 0.f);
}

template <int P>
__global__ void __launch_bounds__(kWarps * 32, P == 4 ? 4 : 5) k_degrid_sum(TaskParams tp, const char* __restrict__ table,
                                                                                        const float2* __restrict__ grid,
                                                                                        float* __restrict__ acc)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* base = smem_raw + (size_t)wid * kDegridSmem<P>;
    Chunk<P, false> ck(base, lane);
    float* red = reinterpret_cast<float*>(base + Chunk<P, false>::kBytes);
    const int parts = item_parts(tp);

    Item it;
    while (next_item(tp, parts, lane, it)) {
        // passes over the entries as in the gridder
        bool again = it.n > 0;
        for (int pass = 0; again; ++pass) {
            again = false;
            const bool report = it.blk == 0 && pass == 0;
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
                // (at P = 4: support 7, 4288 -> 2950 us on 13.8 M entries, where all four units took as long as single points)
                if (un.y - un.x > 2)
                    j = degrid_entries<P, kUnitsMax>(ck, j, S, ch, un, tp, report, red, table, grid, acc);
                else
                    j = degrid_entries<P, 2>(ck, j, S, ch, un, tp, report, red, table, grid, acc);
            }
        }
    }
}

// One thread per entry writes the records of its run: rows run.x..run.y of input channel
// gchan / kst (w-stacking: kst planes per channel), or records run.x..run.y when interleaved.
// One block per preparation tile (rpb rows x all channels) writes the tile's output records
// row-major.  Phase 1 puts each entry's sums into the shared-memory tile at the records of its
// run that fall in the tile (the run before the tile's first head of a list can reach into
// it), phase 2 stores the tile with coalesced stores (vec: out is 16-byte aligned, two
// polarisations a store; callers need only align it to a polarisation's 8 bytes), conjugated back where psi = -1
// (the take-conjugate class bit), with the cross hands swapped back under cross-hand swapping,
// and for the adjoint mode scaled by eps (1 - f).  Records that are not griddable are in no run
// and keep the tile's zero.  Lists: one per input channel (rows), or one in natural record
// order when interleaved.
template <int P>
__global__ void __launch_bounds__(512) k_degrid_tile(const int2* __restrict__ runs, const float2* __restrict__ acc,
                                                     const int* __restrict__ tile_off, const int* __restrict__ chan_base,
                                                     const uint8_t* __restrict__ rclass, const float* __restrict__ weight,
                                                     const uint8_t* __restrict__ flag, int adjoint, int cross_swap,
                                                     int interleave, int vec, int64_t rows, int rpb, int C, int64_t n_tiles,
                                                     float2* __restrict__ out)
{
    extern __shared__ __align__(16) float2 s_out[];      // [rpb * C][P]
    const int64_t tile = blockIdx.x;
    const int64_t row0 = tile * rpb;
    const int nrows = (int)min((int64_t)rpb, rows - row0);
    const int nrec = nrows * C;
    for (int i = threadIdx.x; i < nrec * P; i += blockDim.x) s_out[i] = make_float2(0.f, 0.f);
    __syncthreads();
    const int nlist = interleave ? 1 : C;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    // the tile in list units: rows of a channel, or records in natural order
    const int64_t lo = interleave ? row0 * C : row0, hi = interleave ? row0 * C + nrec : row0 + nrows;
    for (int l = threadIdx.x >> 5; l < nlist; l += nw) {
        const int base = chan_base[l];
        const int first = base + tile_off[tile * C + l];
        const int end = tile + 1 < n_tiles ? base + tile_off[(tile + 1) * C + l] : chan_base[l + 1];
        for (int e = first - 1 + lane; e < end; e += 32) {
            if (e < base) continue;
            const int2 run = runs[e];
            const int64_t a = max((int64_t)run.x, lo), b = min((int64_t)run.y + 1, hi);
            if (a >= b) continue;
            float2 m[P];
#pragma unroll
            for (int p = 0; p < P; ++p) m[p] = acc[(int64_t)e * P + p];
            for (int64_t r = a; r < b; ++r) {
                const int j = interleave ? (int)(r - lo) : (int)(r - row0) * C + l;
#pragma unroll
                for (int p = 0; p < P; ++p) s_out[j * P + p] = m[p];
            }
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nrec; j += blockDim.x) {
        const int64_t rec = row0 * C + j;
        const bool neg = (rclass[rec] >> 3) & 1;
        float2 v[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            // with cross-hand swapping, output pol 1 of a take-conjugate record comes from grid
            // pol 2 and pol 2 from pol 1 (the adjoint of the swap is the swap)
            const int src = (P == 4 && cross_swap && neg && (p == 1 || p == 2)) ? 3 - p : p;
            const float2 a = s_out[j * P + src];
            v[p] = neg ? make_float2(a.x, -a.y) : a;
            if (adjoint) {
                const float wf = weight[rec * P + p] * (1.0f - (float)flag[rec * P + p]);
                v[p].x *= wf;
                v[p].y *= wf;
            }
        }
        float2* o = out + rec * P;
        if (P == 1 || !vec) {
#pragma unroll
            for (int p = 0; p < P; ++p) o[p] = v[p];
        } else {
#pragma unroll
            for (int h = 0; h < P; h += 2)
                *reinterpret_cast<float4*>(o + h) = make_float4(v[h].x, v[h].y, v[(h + 1) % P].x, v[(h + 1) % P].y);
        }
    }
}

template <int P>
static int degrid_sum_launch(const Grid& g, const Table& t, const WorkList& wl, cudaStream_t s)
{
    static int blocks_per_sm = 0;
    const int smem = (int)(kWarps * kDegridSmem<P>);
    if (blocks_per_sm == 0) {
        WG_CUDA(cudaFuncSetAttribute(k_degrid_sum<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, k_degrid_sum<P>, kWarps * 32, smem) != cudaSuccess ||
            blocks_per_sm < 1)
            blocks_per_sm = 1;
    }
    k_degrid_sum<P><<<num_sms() * blocks_per_sm, kWarps * 32, smem, s>>>(
        task_params(g, t, wl, wl.task_counter + 1), reinterpret_cast<const char*>(t.pairs), g.data,
        reinterpret_cast<float*>(wl.dacc));
    WG_LAUNCHED("k_degrid_sum");
    return WG_OK;
}

template <int P>
static int degrid_impl(const Grid& g, const Table& t, const wg_vis_in& in, const WorkList& wl, int mode, float2* out,
                       cudaStream_t s)
{
    if (!wl.dacc) return fail(WG_E_INVALID_ARG, "degrid_vis: the work list has no degridding accumulator");
    const int zb = num_sms() * 4;
    k_degrid_zero<<<zb, 256, 0, s>>>(reinterpret_cast<float4*>(wl.dacc), wl.scal, P, wl.task_counter + 1);
    WG_LAUNCHED("k_degrid_zero");
    const int rc = degrid_sum_launch<P>(g, t, wl, s);
    if (rc != WG_OK) return rc;
    const int tile_smem = (int)(sizeof(float2) * (size_t)wl.rpb * in.n_chan * P);
    static bool attr_set[5] = {false, false, false, false, false};
    if (!attr_set[P]) {
        WG_CUDA(cudaFuncSetAttribute(k_degrid_tile<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(sizeof(float2) * (size_t)kTileCap * P)));
        attr_set[P] = true;
    }
    if (tile_smem > (int)(sizeof(float2) * (size_t)kTileCap * P))
        return fail(WG_E_CAPACITY, "degrid_vis: %d records per preparation tile exceed %d", wl.rpb * in.n_chan, kTileCap);
    if (wl.n_tiles == 0) return WG_OK;     // no records
    k_degrid_tile<P><<<(unsigned)wl.n_tiles, 512, tile_smem, s>>>(
        wl.runs, wl.dacc, wl.tile_cnt, wl.chan_base, wl.rclass, in.weight, in.flag, mode == WG_DEGRID_ADJOINT ? 1 : 0,
        wl.cross_swap ? 1 : 0, wl.interleave ? 1 : 0, reinterpret_cast<uintptr_t>(out) % 16 == 0 ? 1 : 0,
        in.n_rows, wl.rpb, in.n_chan, wl.n_tiles, out);
    WG_LAUNCHED("k_degrid_tile");
    return WG_OK;
}

int launch_degrid(const Grid& g, const Table& t, const wg_vis_in& in, const WorkList& wl, int mode, float2* out,
                  cudaStream_t s)
{
    switch (g.n_pol) {
        case 1: return degrid_impl<1>(g, t, in, wl, mode, out, s);
        case 2: return degrid_impl<2>(g, t, in, wl, mode, out, s);
        case 4: return degrid_impl<4>(g, t, in, wl, mode, out, s);
        default: return fail(WG_E_INVALID_ARG, "n_pol must be 1, 2 or 4");
    }
}

}  // namespace wg

// Device code shared by the gridder and the degridder: packed FP32 arithmetic, the paired kernel
// samples, and the staging of a task's entries.
//
// Pixel pairs.  Both kernels work on pairs of a footprint's points: with H = (S + 1) / 2, pair (i, c)
// holds the points of rows i and i + H in column c.  (S is odd: row S, one past the footprint, completes the
// last row of pairs, with zero samples.)  The kernel table is kept in that form as well (k_table_pairs): per
// sub-kernel, H rows of S sample pairs {re, re', im, im'}.  One 16-byte load then gives two points'
// samples as two packed FP32 pairs, which feed the packed FMAs (fma.rn.f32x2) as they are: with samples
// as (re, im) each point cost three or four moves to broadcast its two parts, on the same pipe as the FMAs.
// Pairs of adjacent columns would need a second copy of the table for odd origins; it did not fit
// L2 at 64 planes up to support 129 (2 x 200 MB: 48 % L2 hits, 125 GB of DRAM reads in one launch of 31 G updates).
//
// Ownership is Romein's (thesis Sec. 2.5) on pairs: a lane owns pairs by their class (column mod S, row
// mod H), so exactly one pair of each class lies in every footprint.  When the footprint moves by one
// column, one class column wraps; when it moves by one row, one class row does (one of the two pixels of
// its pairs has left and the other changes its place: both are flushed, rows are long and wrap rarely).  The
// pairs of a support are dealt out in units of 32 (one per lane, along the rows: a column move touches
// 32 / S of the units); the ceil(S^2 / slots) task blocks of the plan share the units evenly.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "internal.cuh"

namespace wg {

namespace {

typedef unsigned long long f32x2;   // a packed FP32 pair (Blackwell f32x2 arithmetic)

__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void cp_async8(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_addr(dst)), "l"(src));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src));
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }

// one pair of samples: the two real parts and the two imaginary parts
struct KPair {
    f32x2 re, im;
};

// the pair at byte offset `off` from a sub-kernel's first pair; TS is the stored sample type
// (float2: 16 bytes a pair; __half2 and __nv_bfloat162: 8 bytes a pair, widened)
template <typename TS>
constexpr int kPairBytes = 4 * (int)sizeof(TS) / 2;

__device__ __forceinline__ KPair load_pair(const float2*, const char* kz, unsigned off)
{
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(kz + off));
    return {v.x, v.y};
}
__device__ __forceinline__ KPair load_pair(const __half2*, const char* kz, unsigned off)
{
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(kz + off));
    __half2 a, b;
    memcpy(&a, &v.x, 4);
    memcpy(&b, &v.y, 4);
    const float2 re = __half22float2(a), im = __half22float2(b);
    return {pack2(re.x, re.y), pack2(im.x, im.y)};
}
__device__ __forceinline__ KPair load_pair(const __nv_bfloat162*, const char* kz, unsigned off)
{
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(kz + off));
    __nv_bfloat162 a, b;
    memcpy(&a, &v.x, 4);
    memcpy(&b, &v.y, 4);
    const float2 re = __bfloat1622float2(a), im = __bfloat1622float2(b);
    return {pack2(re.x, re.y), pack2(im.x, im.y)};
}

// what the staging needs of the table and the grid
struct TaskParams {
    const int4* entries;
    const float2* gamma;
    const int* seg_off;
    const long long* scal;
    const long long* n_tasks;
    const int* supports;
    const int* offsets;          // C-1 offset of each plane (entries' z refer to it)
    const unsigned* poffsets;    // first pair of each plane in the paired table
    int N, K, C, beta2;
    int64_t n_samples;
    int seg_len, slots;
    unsigned* counter;
    long long* dropped;
};

// One entry as it is staged in shared memory.
//   x: fp, the footprint's origin, column | row << 16
//   y: cuv, (-column) mod S | (-row) mod H << 16: class (0, 0)'s place in the footprint
//   z: the first pair of its sub-kernel in the paired table
//   w: key, support << 16 | grid channel; -1: rejected by the bounds checks
typedef int4 Staged;
__device__ __forceinline__ int key_support(int key) { return key >> 16; }
__device__ __forceinline__ int key_chan(int key) { return key & 0xFFFF; }

// Checks an entry against the grid and the table (never failing for a work list written by
// vis_compress for them) and finds its sub-kernel in the paired table.
__device__ __forceinline__ Staged stage_entry(const int4& E, const TaskParams& tp)
{
    const Staged bad = make_int4(0, 0, 0, -1);
    const int k = E.w & 0xFFF, ch = (E.w >> 16) & 0xFFFF;
    if (E.w < 0 || k >= tp.K || ch >= tp.C || E.z < 0) return bad;
    const int S = __ldg(&tp.supports[k]), s2 = S * S;
    const int x0 = E.x & 0xFFFF, y0 = (E.x >> 16) & 0xFFFF;
    const int rel = E.z - __ldg(&tp.offsets[k]);
    if (x0 + S > tp.N || y0 + S > tp.N || rel < 0 || (int64_t)E.z + s2 > tp.n_samples) return bad;
    // sub-kernel index rel / S^2 <= beta^2 <= 4096: the float quotient is within one of it
    int sub = __float2int_rz((float)rel * __frcp_rn((float)s2));
    int rem = rel - sub * s2;
    if (rem < 0) { --sub; rem += s2; }
    if (rem >= s2) { ++sub; rem -= s2; }
    if (rem != 0 || sub >= tp.beta2) return bad;
    const int H = (S + 1) >> 1;
    const unsigned z = __ldg(&tp.poffsets[k]) + (unsigned)sub * (unsigned)(S * H);
    const int rx = divmod_small(x0, S, __frcp_rn((float)S)).y, ry = divmod_small(y0, H, __frcp_rn((float)H)).y;
    return make_int4(x0 | (y0 << 16), (rx ? S - rx : 0) | ((ry ? H - ry : 0) << 16), (int)z, (S << 16) | ch);
}

// Gives a lane its classes (column mod S | row mod H << 16, in cls[u][lane]) of a support's units from
// unit0 up to unit1, and places them in the footprint of entry E: the pairs' offsets in a sub-kernel (in bytes,
// PB a pair) and the first pixel of each (column | row << 16 in cur[u][lane]; -1 past the last pair or unit: such
// a lane follows class (0, 0), which keeps its loads inside the sub-kernel, and holds no pixel).
template <int NU, int PB>
__device__ __forceinline__ void place_classes(unsigned (&toff)[NU], int (*cls)[32], int (*cur)[32], const Staged& E, int S,
                                              int unit0, int unit1, int lane)
{
    const int H = (S + 1) >> 1;
    const float inv_s = 1.0f / (float)S;
    const int cu = E.y & 0xFFFF, cv = E.y >> 16, end = min(H * S, unit1 * 32);
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        const int i = (unit0 + u) * 32 + lane;
        const bool in = i < end;
        const int2 vu = divmod_small(in ? i : 0, S, inv_s);
        int du = vu.y + cu, dv = vu.x + cv;
        du -= (du >= S) ? S : 0;
        dv -= (dv >= H) ? H : 0;
        cls[u][lane] = vu.y | (vu.x << 16);
        cur[u][lane] = in ? E.x + (du | (dv << 16)) : -1;
        toff[u] = (unsigned)(dv * S + du) * PB;
    }
}

// Places a pair of class cl (column | row << 16) in the footprint of entry E: its column | row << 16 there.  Each
// half of cl + E.y is less than twice its modulus, so that the smaller of it and it less the modulus (as an unsigned
// 16-bit number) is the remainder; minus_sh = minus_moduli(S, H).
__device__ __forceinline__ unsigned minus_moduli(int S, int H) { return (unsigned)(0x10000 - S) | ((unsigned)(0x10000 - H) << 16); }
__device__ __forceinline__ int place_class(int cl, const Staged& E, unsigned minus_sh)
{
    const unsigned t = (unsigned)cl + (unsigned)E.y;
    return (int)__viaddmin_u16x2(t, minus_sh, t);
}

// column + row * pitch of a packed column | row << 16 (modulo 2^32), times scale
__device__ __forceinline__ unsigned linear(int packed, int pitch, unsigned scale)
{
    return (unsigned)packed * scale + (unsigned)(packed >> 16) * ((unsigned)(pitch - 0x10000) * scale);
}

constexpr int kPartMin = 4;   // entries of the shortest part of a segment

// Units a warp holds in registers in one pass over its entries.
constexpr int kUnitsMax = 4;

// The units [x, y) of task block blk of a support with nb blocks (units of 32 pairs, shared evenly).
__device__ __forceinline__ int2 block_units(int S, int blk, int nb)
{
    const int units = (S * ((S + 1) >> 1) + 31) >> 5;
    return make_int2(blk * units / nb, (blk + 1) * units / nb);
}

// A warp's walk over the entries of its work item, 32 at a time.  Each lane stages one entry: its
// checks, residues and sub-kernel are worked out once, in parallel, and the warp keeps bit masks of the entries at which something changes, so that the record loops run
// over stretches without a test.  The next 32 entries are on their way (cp.async) meanwhile.
// With GAMMA the weighted visibilities are staged too.
template <int P, bool GAMMA>
struct Chunk {
    static constexpr int kG = GAMMA ? 32 * P * (int)sizeof(float2) : 0;
    static constexpr int kBytes = 64 * (int)sizeof(int4) + 2 * kG + (3 * kUnitsMax + 1) * 32 * (int)sizeof(int);
    int4* raw_e;             // [32] as copied
    Staged* e;               // [32]
    float2* raw_g;           // [32][P]
    float2* g;               // [32][P] weighted visibilities
    unsigned* z;             // [32] the entries' z again
    int (*cls)[32];          // [kUnitsMax][32] the lanes' classes
    int (*cur)[32];          // [kUnitsMax][32] the first pixels of the pairs they hold
    int (*nxt)[32];          // [kUnitsMax][32] the first pixels after a move (the gridder's)
    int lane;
    int e0, left, cnt;       // the chunk's first entry in the lists, entries from there to the item's end, its entries
    unsigned kc;             // entries that start a run: another support or channel, or around a slow one
    unsigned mv;             // entries whose footprint differs from their predecessor's (and kc)
    unsigned slow;           // entries with an infinite or NaN visibility

    __device__ __forceinline__ Chunk(unsigned char* base, int lane_)
        : raw_e(reinterpret_cast<int4*>(base)), e(raw_e + 32), raw_g(reinterpret_cast<float2*>(e + 32)),
          g(raw_g + kG / sizeof(float2)), z(reinterpret_cast<unsigned*>(g + kG / sizeof(float2))),
          cls(reinterpret_cast<int (*)[32]>(z + 32)), cur(cls + kUnitsMax), nxt(cls + 2 * kUnitsMax), lane(lane_)
    {
    }

    // copies the entries from list place e on, `count` of them left
    __device__ __forceinline__ void issue(const TaskParams& tp, int e, int count)
    {
        if (lane < count) {
            const size_t i = (size_t)(e + lane);
            cp_async16(&raw_e[lane], tp.entries + i);
            if constexpr (GAMMA) {
                if constexpr (P == 1) {
                    cp_async8(&raw_g[lane], tp.gamma + i);
                } else {
#pragma unroll
                    for (int p = 0; p < P; p += 2) cp_async16(&raw_g[lane * P + p], tp.gamma + i * P + p);
                }
            }
        }
        cp_commit();
    }

    // starts on entries [first, first + count) of the lists: next() then stages the first 32
    __device__ __forceinline__ void begin(const TaskParams& tp, int first, int count)
    {
        e0 = first - 32;
        left = count + 32;
        cnt = 0;
        slow = 0;
        kc = 0;
        __syncwarp();                // the item before has been read
        if (lane == 31) e[31] = make_int4(0, 0, 0, -1);
        __syncwarp();
        issue(tp, first, count);
    }

    // stages the next 32 entries; false at the end
    __device__ __forceinline__ bool next(const TaskParams& tp, bool report)
    {
        if (left <= 32) return false;
        const Staged last = e[31];
        const int pkey = last.w;
        const bool pslow = slow >> 31;
        e0 += 32;
        left -= 32;
        cnt = min(32, left);
        const bool in = lane < cnt;
        cp_wait_all();               // each lane reads only what it copied itself
        Staged s = make_int4(0, 0, 0, -1);
        if (in) s = stage_entry(raw_e[lane], tp);
        if (report && in && s.w < 0) atomicAdd(reinterpret_cast<unsigned long long*>(tp.dropped), 1ull);
        bool sl = false;
        float2 v[P];
        if constexpr (GAMMA) {
            float t = 0.f;           // 0 unless some part is infinite or NaN
#pragma unroll
            for (int p = 0; p < P; ++p) {
                v[p] = in ? raw_g[lane * P + p] : make_float2(0.f, 0.f);
                t = fmaf(v[p].x, 0.f, fmaf(v[p].y, 0.f, t));
            }
            sl = !(t == 0.f);
        }
        __syncwarp();                // the previous chunk has been read
        slow = __ballot_sync(0xffffffffu, in && sl);
        int qk = __shfl_up_sync(0xffffffffu, s.w, 1), qf = __shfl_up_sync(0xffffffffu, s.x, 1);
        bool qs = lane ? (slow >> (lane - 1)) & 1 : pslow;
        if (lane == 0) {
            qk = pkey;
            qf = last.x;
        }
        const bool k = s.w != qk || sl || qs;
        kc = __ballot_sync(0xffffffffu, in && k);
        mv = __ballot_sync(0xffffffffu, in && (k || s.x != qf));
        e[lane] = s;
        z[lane] = (unsigned)s.z;
        if constexpr (GAMMA) {
#pragma unroll
            for (int p = 0; p < P; ++p) g[lane * P + p] = v[p];
        }
        __syncwarp();
        issue(tp, e0 + 32, left - 32);
        return true;
    }

    // the first entry after j at which a run starts, or the chunk's end
    __device__ __forceinline__ int run_end(int j) const
    {
        const unsigned later = kc & (0xFFFFFFFEu << j);
        return later ? __ffs(later) - 1 : cnt;
    }
};

// A persistent kernel's next work item: a task, or part of one.  With fewer tasks than warps each
// segment is cut into parts, so that every warp has something to do (17 tasks on 2432 warps: 204 -> 25 us).
struct Item {
    int blk, e0, n;          // block of the footprint, first entry, entries
};

__device__ __forceinline__ int item_parts(const TaskParams& tp)
{
    const long long n_tasks = *tp.n_tasks, warps = (long long)gridDim.x * (blockDim.x >> 5);
    if (n_tasks <= 0 || n_tasks >= warps) return 1;
    return (int)min((long long)(tp.seg_len / kPartMin), (warps + n_tasks - 1) / n_tasks);
}

// the next item, handed out by a global counter; false when there is none left
__device__ __forceinline__ bool next_item(const TaskParams& tp, int parts, int lane, Item& it)
{
    unsigned w = 0;
    if (lane == 0) w = atomicAdd(tp.counter, 1u);
    w = __shfl_sync(0xffffffffu, w, 0);
    const unsigned t = parts > 1 ? w / (unsigned)parts : w;
    if ((long long)t >= *tp.n_tasks) return false;
    // the task's segment: each step probes 32 places
    int lo = 0, hi = (int)tp.scal[2];
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) >> 5, at = lo + lane * step;
        const unsigned m = __ballot_sync(0xffffffffu, at < hi && __ldg(&tp.seg_off[at]) <= (int)t);
        lo += (31 - __clz(m)) * step;          // (offsets grow: the probes that pass are the first ones)
        hi = min(hi, lo + step);
    }
    it.blk = (int)t - __ldg(&tp.seg_off[lo]);
    it.e0 = lo * tp.seg_len;
    it.n = (int)min((long long)tp.seg_len, tp.scal[0] - it.e0);
    if (parts > 1) {
        const int part = (int)(w - t * (unsigned)parts);
        const int a = it.n * part / parts;
        it.n = it.n * (part + 1) / parts - a;
        it.e0 += a;
    }
    return true;
}

inline TaskParams task_params(const Grid& g, const Table& t, const WorkList& wl, unsigned* counter)
{
    return {wl.entries, wl.gamma, wl.seg_off,         wl.scal,     wl.scal + 1, t.supports_d, t.offsets_d, t.poffsets_d, g.n, t.K,
            g.n_chan,   t.beta * t.beta, t.n_samples, wl.seg_len,  wl.slots,    counter,      wl.scal + 3};
}

}  // namespace

}  // namespace wg

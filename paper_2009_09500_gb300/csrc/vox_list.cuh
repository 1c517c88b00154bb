// vox_list.cuh -- the packed voxel list, one row of 32 voxels per warp and step (sm_103a).
//
// The list of Fig. 3 / Section 4 (every voxel of every segment, in segment order,
// at offsets[s] + k). Voxel k does not depend on voxel k - 1 (Section 3), and with
// a fixed-point slope it needs no division either, so lane l of a warp computes
// voxel g + l of a row of 32 consecutive voxels outright and the row is stored
// coalesced: no run per lane, no stage in shared memory, no transposition.
//
// Per axis the coordinate is the integer part of X0 + k T (mod 2^bits), with F
// fraction bits and S = ceil(|d| 2^F / N):
//   d >= 0:  X0 = S0 2^F + 2^(F-1),      T = S      floor(S0 + 1/2 + k S / 2^F)
//   d <  0:  X0 = S0 2^F + 2^(F-1) - 1,  T = -S     floor(S0 + 1/2 - k S / 2^F - 2^-F)
// The exact position S0 + 1/2 +- k |d| / N is a multiple of 1 / 2N, so its integer
// part is unchanged by an error below 1 / 2N away from the side where a tie falls;
// the error is below k 2^-F (plus 2^-F when d < 0), so F with (N + 1) 2^-F <= 1 / 2N
// gives Eq. (3) with ties away from S, exactly:
//   32-bit lists (edges <= 1024, N <= 1023): F = 22, one 32-bit word per axis;
//   64-bit lists (N < 2^21): F = 43, one 64-bit word per axis.
// The slopes are divided out once per staged segment (a lane per segment of the
// window), not once per run of voxels.
//
// What bounds it: HBM writes for 64-bit lists of long segments, instruction issue for
// short ones (a row is 128 32-bit or 64 64-bit voxels; most of its instructions are three
// additions and three or four shifts a voxel).
// Measured (GB300, list kernel alone), against runs of 33 voxels per lane stepped by the
// carry recurrence into a shared stage (long segments) and 32-voxel thread runs with a
// transposed stage (the rest); in the middle, rows whose lanes read a segment by eight
// 4-byte loads, start and step apart, and pack by shifts and masks:
//   4M log-uniform segments in 4096^3, 64-bit, 2.07e9 voxels   2720 -> 2301 -> 2307 us
//   1024 segments, 10^9 voxels, 64-bit                         1090 -> 1048 -> 1048 us
//   1M log-uniform segments in 1000^3, 64-bit, 1.5e8 voxels     301 ->  216 ->  208 us
//   300,000 uniform segments in 256^3, 32-bit, 4.2e7 voxels      76 ->   52 ->   43 us
//   1M segments of 64 voxels, 32-bit, 6.7e7 voxels               78 ->   75 ->   63 us
// (the last: 66 us by 64-voxel thread runs, which a tuning could ask for)
#pragma once

#include <cstdint>
#include <type_traits>

#include "vox_bricks.cuh"
#include "vox_device.cuh"
#include "vox_kernels.cuh"

namespace vox {

constexpr int kListWarps = 8;                  // warps per CTA
constexpr int kListThreads = 32 * kListWarps;
constexpr int kListCtas = 4;                   // CTAs per SM
constexpr int kListWin = 32;                   // segments per staged window, one per lane
// The list is cut into chunks of consecutive voxels, one per warp, as many as keep a chunk
// within kListChunkMax, from the total that the scan found. The grid holds a CTA for every
// chunk that the capacity allows (launch_list); CTAs beyond the total leave at once (0.3 ns
// each). The CTAs beyond the resident ones start in order as others end, so the warps at
// work at any moment write one front of the list (see the figures at k_list).
constexpr int kListChunkUnit = 128;            // chunks are multiples of a row
constexpr int kListChunkMin = 256;             // voxels per warp at least
constexpr int kListChunkMax = 6144;            // and at most, for up to kListRounds chunks per
constexpr int64_t kListRounds = 256;           // resident warp (7.6e9 voxels; then longer ones)

struct ListParams {
    const int32_t *segs;     // [n][6]
    int64_t n;
    const int64_t *offsets;  // [n + 1] exclusive offsets (workspace), offsets[n] = V
    void *list;              // uint32 or uint64 list, 16-byte aligned
    int64_t capacity;
    int32_t *status;
    int32_t resident;        // CTAs at work at a time; the grid is a multiple of it
};

// Fixed-point words of a list type: F fraction bits, integer parts on top. Packing is a
// chain of funnel shifts, (h << n) | (l >> (32 - n)). For 32-bit rows inside one segment
// shifts and masks are the better: 2.7e8 voxels in segments of 700 and 1000 171 and 168 us
// by funnel shifts, 166 and 162 by masks (of 200 and 300: 201 and 189 against 207 and 199;
// in rows with segment starts of 64 voxels 222 against 236).
template <typename PackT>
struct ListFix;

template <>
struct ListFix<uint32_t> {
    static constexpr int F = 22;
    // x | y << 10 | z << 20 from the top 10 bits of each word
    static __device__ __forceinline__ uint32_t pack(uint32_t x, uint32_t y, uint32_t z)
    {
        return __funnelshift_l(x, __funnelshift_l(y, z >> 22, 10), 10);
    }
    static __device__ __forceinline__ uint32_t pack_inside(uint32_t x, uint32_t y, uint32_t z)
    {
        return (x >> 22) | ((y >> 12) & 0x000ffc00u) | ((z >> 2) & 0x3ff00000u);
    }
};

template <>
struct ListFix<uint64_t> {
    static constexpr int F = 43;
    // x | y << 21 | z << 42 from the top 21 bits of each word, half by half
    static __device__ __forceinline__ uint64_t pack(uint64_t x, uint64_t y, uint64_t z)
    {
        const uint32_t xh = static_cast<uint32_t>(x >> 32), yh = static_cast<uint32_t>(y >> 32),
                       zh = static_cast<uint32_t>(z >> 32);
        const uint32_t lo = __funnelshift_l(xh, yh >> 11, 21);
        const uint32_t hi = __funnelshift_l(yh, zh >> 11, 10);
        return (static_cast<uint64_t>(hi) << 32) | lo;
    }
    static __device__ __forceinline__ uint64_t pack_inside(uint64_t x, uint64_t y, uint64_t z) { return pack(x, y, z); }
};

// Voxels that the resident CTAs' warps write with one chunk of at most kListChunkMax each.
__host__ __device__ inline int64_t list_round(int32_t resident)
{
    return static_cast<int64_t>(resident) * (kListWarps * kListChunkMax);
}

// Voxels per chunk of a list of V voxels, by a grid of grid_rounds times the resident CTAs.
__host__ __device__ inline int64_t list_chunk(int64_t V, int32_t resident, int64_t grid_rounds)
{
    const int64_t round = list_round(resident);
    int64_t chunks = static_cast<int64_t>(resident) * kListWarps;
    if (V > round) {
        const int64_t rounds = (V + round - 1) / round;
        chunks *= rounds < grid_rounds ? rounds : grid_rounds;
    }
    const int64_t per = ((V + chunks - 1) / chunks + kListChunkUnit - 1) & ~int64_t(kListChunkUnit - 1);
    return per > kListChunkMin ? per : int64_t(kListChunkMin);
}

// A segment of the window: coordinates X = C + p T at position p of the chunk (the
// segment's X0 less its first position times T, modulo the word), so that a voxel needs
// neither the segment's start nor its step; and the position where the next one starts.
template <typename PackT>
struct ListSeg {
    PackT C[3], T[3];
    int32_t next;
};

// The window as the lanes read it, in words of 16 bytes: two (32-bit) or three loads bring
// a segment, and lanes that read consecutive segments meet no bank twice.
template <typename PackT>
struct ListWarpSmem;

template <>
struct ListWarpSmem<uint32_t> {
    uint4 a[kListWin], b[kListWin];

    __device__ __forceinline__ void put(int j, const ListSeg<uint32_t> &g)
    {
        a[j] = make_uint4(g.C[0], g.C[1], g.C[2], static_cast<uint32_t>(g.next));
        b[j] = make_uint4(g.T[0], g.T[1], g.T[2], 0u);
    }
    __device__ __forceinline__ ListSeg<uint32_t> get(int j) const
    {
        const uint4 u = a[j], v = b[j];
        return {{u.x, u.y, u.z}, {v.x, v.y, v.z}, static_cast<int32_t>(u.w)};
    }
    __device__ __forceinline__ int32_t next(int j) const { return static_cast<int32_t>(a[j].w); }
};

template <>
struct ListWarpSmem<uint64_t> {
    ulonglong2 a[kListWin], b[kListWin], c[kListWin];
    int32_t nx[kListWin];

    __device__ __forceinline__ void put(int j, const ListSeg<uint64_t> &g)
    {
        a[j] = make_ulonglong2(g.C[0], g.C[1]);
        b[j] = make_ulonglong2(g.C[2], g.T[0]);
        c[j] = make_ulonglong2(g.T[1], g.T[2]);
        nx[j] = g.next;
    }
    __device__ __forceinline__ ListSeg<uint64_t> get(int j) const
    {
        const ulonglong2 u = a[j], v = b[j], w = c[j];
        return {{u.x, u.y, v.x}, {v.y, w.x, w.y}, nx[j]};
    }
    __device__ __forceinline__ int32_t next(int j) const { return nx[j]; }
};

// Largest s in [0, n) with offsets[s] <= g (offsets[0] <= g < offsets[n]): a
// 32-ary search in which every lane probes one position per round; called by
// the whole warp with the same arguments.
__device__ __forceinline__ int64_t warp_find_segment(const int64_t *offsets, int64_t n, int64_t g, int lane)
{
    int64_t lo = 0, hi = n;
    while (hi - lo > 1) {
        const int64_t stride = (hi - lo + 31) / 32;
        const int64_t pos = lo + static_cast<int64_t>(lane) * stride;
        const bool le = pos < hi && __ldg(offsets + pos) <= g;
        const int cnt = __popc(__ballot_sync(0xffffffffu, le));  // probes 0 .. cnt-1 hold (monotone)
        const int64_t base = lo;
        lo = base + static_cast<int64_t>(cnt - 1) * stride;
        hi = min(hi, base + static_cast<int64_t>(cnt) * stride);
    }
    return lo;
}

__device__ __forceinline__ void prefetch_l1(const void *p)
{
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

__device__ __forceinline__ int4 list_quad(const uint32_t (&v)[4])
{
    return make_int4(static_cast<int>(v[0]), static_cast<int>(v[1]), static_cast<int>(v[2]), static_cast<int>(v[3]));
}

__device__ __forceinline__ int4 list_quad(const uint64_t (&v)[2])
{
    return make_int4(static_cast<int>(v[0]), static_cast<int>(v[0] >> 32), static_cast<int>(v[1]),
                     static_cast<int>(v[1] >> 32));
}

// One chunk per warp, written front to back. What the chunks' order is worth: with
// persistent warps taking every n_warps-th chunk the warps drift apart, and 2.07e9
// 64-bit voxels take 2785 us; with CTAs started in order the writes stay one front and
// take 2308 us (7.2 TB/s), with chunks from a counter 2350 (10^9 voxels in 1024 segments
// 1053 and 1064, 2.7e8 32-bit voxels in segments of 700 171 and 187). Chunks of 8192 /
// 12288 voxels at most: 2353 / 2451 us; 2048: 3416 us (the search per chunk). Rows collected
// in shared memory and stored by 4 KB bulk copies: 2421 us, and 88 instead of 76 us on
// 64-voxel segments.
// A capacity of 1, 3, 16 times the total, and no bound: 4M log-uniform segments 2312, 2342,
// 2359, 2359 us; 10^9 voxels in 1024 segments 1051, 1055, 1055, 1055; 300,000 log-uniform
// 117 each. (With chunks cut from the capacity: 2308, 2552, 7016; 1053, 1326, 6476; 117,
// 122, 281.)
template <typename PackT>
__global__ void __launch_bounds__(kListThreads, kListCtas) k_list(ListParams p)
{
    using Fix = ListFix<PackT>;
    constexpr int kVox = 16 / sizeof(PackT);  // consecutive voxels per lane and row: one 16-byte store
    constexpr int kRow = 32 * kVox;
    __shared__ ListWarpSmem<PackT> s_win[kListWarps];
    __shared__ int32_t s_go;
    __shared__ int64_t s_chunk;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    ListWarpSmem<PackT> &sm = s_win[warp];

    // the CTAs beyond the list: whole rounds of resident CTAs that it does not reach
    const int64_t V = __ldg(p.offsets + p.n);
    const uint32_t rounds_before = blockIdx.x / static_cast<uint32_t>(p.resident);
    if (rounds_before > 0 && rounds_before * list_round(p.resident) >= V) return;

    // prologue decided by one thread so that the whole CTA agrees
    if (threadIdx.x == 0) {
        int32_t go = ld_volatile_i32(p.status) == 0;  // an earlier error: write nothing
        if (go && V > p.capacity) {
            set_status(p.status, kStCapacity);
            go = 0;
        }
        s_go = go;
        s_chunk = list_chunk(V, p.resident, gridDim.x / static_cast<uint32_t>(p.resident));
    }
    __syncthreads();
    if (!s_go) return;
    const int64_t chunk = s_chunk;
    PackT *const list = static_cast<PackT *>(p.list);
    const uint32_t lt_mask = (1u << lane) - 1u;  // the lanes below

    const int64_t g0 = (static_cast<int64_t>(blockIdx.x) * kListWarps + warp) * chunk;
    if (g0 < V) {
        const int32_t len = static_cast<int32_t>(min64(chunk, V - g0));
        PackT *const out = list + g0;
        int64_t s = warp_find_segment(p.offsets, p.n, g0, lane);
        int32_t pos = 0;  // positions are relative to g0
        while (pos < len) {
            // ---- the window: 32 segments from the one that holds `pos`
            const int32_t wcnt = static_cast<int32_t>(min64(kListWin, p.n - s));
            int32_t rel = 0x7fffffff;
            __syncwarp();  // every lane is done with the previous window
            if (lane < wcnt) {
                int32_t r[6];
                load_record(p.segs, s + lane, r);
                rel = static_cast<int32_t>(__ldg(p.offsets + s + lane) - g0);
                const uint32_t N = static_cast<uint32_t>(max(abs(r[3] - r[0]), max(abs(r[4] - r[1]), abs(r[5] - r[2]))));
                ListSeg<PackT> g;
                g.next = static_cast<int32_t>(__ldg(p.offsets + s + lane + 1) - g0);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int32_t d = r[3 + a] - r[a];
                    const PackT A = static_cast<PackT>(abs(d));
                    const PackT S = A == N ? PackT(1) << Fix::F  // the major axis, and minor ones as long
                                           : ((A << Fix::F) + (N - 1u)) / N;
                    g.T[a] = d < 0 ? PackT(0) - S : S;
                    g.C[a] = (static_cast<PackT>(r[a]) << Fix::F) + (PackT(1) << (Fix::F - 1)) - (d < 0 ? 1 : 0) -
                             static_cast<PackT>(static_cast<typename std::make_signed<PackT>::type>(rel)) * g.T[a];
                }
                sm.put(lane, g);
            }
            // the next 32 segments' records and offsets on their way to L1
            if (s + 2 * kListWin <= p.n) {
                if (lane < 24) prefetch_l1(p.segs + 6 * (s + kListWin) + 8 * lane);
                else prefetch_l1(p.offsets + s + kListWin + 4 * (lane - 24));
            }
            __syncwarp();
            const int32_t wend = sm.next(wcnt - 1);
            const int32_t lim = min(wend, len);
            int32_t j = 0;  // the window's segment that holds pos
            while (true) {
                // a row needs the window to cover it; without that the window moves on
                // to segment j, or (already there, or the list ends) 32 voxels are taken
                const bool covered = pos + kRow <= lim;
                if (!covered && j > 0 && wend < len) break;
                // the segments that start in the row after its first voxel (or right after
                // the row), by the lane that holds the voxel before the start; two of them
                // at one lane: short segments, 32 voxels at a time
                const int32_t b = rel - pos;
                const bool inside = b > 0 && b <= kRow;
                const uint32_t starts = __reduce_or_sync(0xffffffffu, inside ? 1u << ((b - 1) / kVox) : 0u);
                if (covered && starts == 0u) {  // rows inside one segment
                    const ListSeg<PackT> g = sm.get(j);
                    const PackT p0 = static_cast<PackT>(pos + kVox * lane);
                    PackT x = g.C[0] + p0 * g.T[0], y = g.C[1] + p0 * g.T[1], z = g.C[2] + p0 * g.T[2];
                    const int32_t stop = min(g.next, len) - kRow;
                    int4 *o = reinterpret_cast<int4 *>(out + pos) + lane;
#pragma unroll 2
                    for (; pos <= stop; pos += kRow) {
                        PackT v[kVox];
#pragma unroll
                        for (int i = 0; i < kVox; ++i) {
                            v[i] = Fix::pack_inside(x, y, z);
                            const uint32_t f = i + 1 < kVox ? 1u : static_cast<uint32_t>(kRow - kVox + 1);
                            x += f * g.T[0];
                            y += f * g.T[1];
                            z += f * g.T[2];
                        }
                        *o = list_quad(v);
                        o += 32;
                    }
                    if (pos >= len) break;
                    if (g.next <= pos) {
                        ++j;
                        if (j >= wcnt) break;
                    }
                    continue;
                }
                const int32_t n_in = __popc(__ballot_sync(0xffffffffu, inside));
                if (covered && __popc(starts) == n_in) {
                    // a row with segment starts, at most one per lane
                    const int32_t p0 = pos + kVox * lane;
                    const int32_t jl = j + __popc(starts & lt_mask);
                    const ListSeg<PackT> g = sm.get(jl);
                    PackT x = g.C[0] + static_cast<PackT>(p0) * g.T[0], y = g.C[1] + static_cast<PackT>(p0) * g.T[1],
                          z = g.C[2] + static_cast<PackT>(p0) * g.T[2];
                    PackT v[kVox];
#pragma unroll
                    for (int i = 0; i < kVox; ++i) {
                        v[i] = Fix::pack(x, y, z);
                        x += g.T[0];
                        y += g.T[1];
                        z += g.T[2];
                    }
                    const int32_t c = g.next - p0;  // this lane's voxels from c on are the next segment's
                    if (c < kVox) {
                        const ListSeg<PackT> h = sm.get(jl + 1);
                        const PackT p1 = static_cast<PackT>(p0 + 1);
                        x = h.C[0] + p1 * h.T[0];
                        y = h.C[1] + p1 * h.T[1];
                        z = h.C[2] + p1 * h.T[2];
#pragma unroll
                        for (int i = 1; i < kVox; ++i) {
                            if (i >= c) v[i] = Fix::pack(x, y, z);
                            x += h.T[0];
                            y += h.T[1];
                            z += h.T[2];
                        }
                    }
                    reinterpret_cast<int4 *>(out + pos)[lane] = list_quad(v);
                    pos += kRow;
                    j += n_in;
                } else {
                    // 32 voxels, one per lane (the window covers them: 32 segments hold at
                    // least 32 voxels): a bit for each start, and each lane counts the bits
                    // before its own position
                    if (wend < len && pos + 32 > wend) break;
                    const uint32_t bits = __reduce_or_sync(0xffffffffu, (b > 0 && b <= 32) ? 1u << (b - 1) : 0u);
                    const ListSeg<PackT> g = sm.get(j + __popc(bits & lt_mask));
                    const PackT p0 = static_cast<PackT>(pos + lane);
                    if (pos + lane < len)
                        out[pos + lane] = Fix::pack(g.C[0] + p0 * g.T[0], g.C[1] + p0 * g.T[1], g.C[2] + p0 * g.T[2]);
                    pos += 32;
                    j += __popc(bits);
                }
                if (pos >= lim) {  // the list's end, or the window's
                    j = wcnt;
                    break;
                }
            }
            s += j;
        }
    }
}

}  // namespace vox

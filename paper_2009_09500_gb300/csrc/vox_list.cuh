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
// What bounds it: HBM writes for 64-bit lists of long segments, instruction issue
// for short ones (75 % of issue slots on 64-voxel segments; about 110 instructions a
// row that holds segment starts, a row being 128 32-bit or 64 64-bit voxels).
// Measured (GB300, list kernel alone), against runs of 33 voxels per lane stepped by
// the carry recurrence into a shared stage (long segments) and 32-voxel thread runs
// with a transposed stage (the rest):
//   4M log-uniform segments in 4096^3, 64-bit, 2.07e9 voxels   2720 -> 2308 us
//   1024 segments, 10^9 voxels, 64-bit                         1090 -> 1051 us
//   1M log-uniform segments in 1000^3, 64-bit, 1.4e8 voxels     301 ->  208 us
//   300,000 uniform segments in 256^3, 32-bit, 4.2e7 voxels      76 ->   54 us
//   1M segments of 64 voxels, 32-bit, 6.7e7 voxels               78 ->   76 us
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
// The list is cut into chunks of consecutive voxels: as many per resident warp as keep a
// chunk within kListChunkMax, from the total that the scan found (never from the caller's
// capacity). A warp's first chunk goes by its index, further ones by a counter, so the
// warps at work at any moment write one front of the list (see the figures at k_list).
constexpr int kListChunkUnit = 128;            // chunks are multiples of a row
constexpr int kListChunkMin = 256;             // voxels per warp at least
constexpr int kListChunkMax = 6144;            // and at most

struct ListParams {
    const int32_t *segs;     // [n][6]
    int64_t n;
    const int64_t *offsets;  // [n + 1] exclusive offsets (workspace), offsets[n] = V
    void *list;              // uint32 or uint64 list, 16-byte aligned
    int64_t capacity;
    int32_t *status;
    uint32_t *counter;       // chunks taken beyond the warps' first (workspace; zero before
                             // the launch where the total may take more than one per warp)
};

// Fixed-point words of a list type: F fraction bits, integer parts on top.
template <typename PackT>
struct ListFix;

template <>
struct ListFix<uint32_t> {
    static constexpr int F = 22;
    // x | y << 10 | z << 20 from the top 10 bits of each word
    static __device__ __forceinline__ uint32_t pack(uint32_t x, uint32_t y, uint32_t z)
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
        const uint32_t lo = (xh >> 11) | ((yh << 10) & 0xffe00000u);
        const uint32_t hi = (yh >> 22) | ((zh >> 1) & 0x7ffffc00u);
        return (static_cast<uint64_t>(hi) << 32) | lo;
    }
};

// Voxels per chunk of a list of V voxels written by n_warps warps.
__host__ __device__ inline int32_t list_chunk(int64_t V, int64_t n_warps)
{
    const int64_t round = n_warps * kListChunkMax;  // voxels of one chunk per warp at most
    const int64_t chunks = V <= round ? n_warps : n_warps * ((V + round - 1) / round);
    const int64_t per = ((V + chunks - 1) / chunks + kListChunkUnit - 1) & ~int64_t(kListChunkUnit - 1);
    return static_cast<int32_t>(per > kListChunkMin ? per : int64_t(kListChunkMin));
}

// A window of segments as the lanes read it: field by field, so that lanes reading
// different segments hit different banks.
template <typename PackT>
struct ListWarpSmem {
    PackT X0[3][kListWin];        // coordinates of voxel 0 (fixed point, half added)
    PackT T[3][kListWin];         // per-voxel steps
    int32_t rel[kListWin + 1];    // first voxel of each segment, relative to the chunk (+ the next)
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

// k t for a signed step count k given in two's complement (modulo the word).
__device__ __forceinline__ uint32_t mul_signed(uint32_t k, uint32_t t) { return k * t; }
__device__ __forceinline__ uint64_t mul_signed(uint32_t k, uint64_t t)
{
    return static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(k))) * t;
}

// Chunks in list order, each written front to back by one warp. What the order is worth:
// with persistent warps taking every n_warps-th chunk the warps drift apart, and 2.07e9
// 64-bit voxels take 2785 us; with chunks from a counter the writes stay one front and
// take 2335 us (7.1 TB/s), whatever the list's capacity. (One chunk per warp of a grid sized
// from the capacity, its CTAs started in order: 2308 us with a capacity of V, but 2552
// with 3 V and 7016 with 16 V, whose chunks are of 384 voxels.) Chunks of 8192 / 12288
// voxels at most: 2353 / 2451 us; 2048: 3416 us (the search per chunk). Rows collected in
// shared memory and stored by 4 KB bulk copies: 2421 us, and 88 instead of 76 us on
// 64-voxel segments.
template <typename PackT>
__global__ void __launch_bounds__(kListThreads, kListCtas) k_list(ListParams p)
{
    using Fix = ListFix<PackT>;
    constexpr int kVox = 16 / sizeof(PackT);  // consecutive voxels per lane and row: one 16-byte store
    constexpr int kRow = 32 * kVox;
    __shared__ ListWarpSmem<PackT> s_win[kListWarps];
    __shared__ int32_t s_go, s_chunk;
    __shared__ int64_t s_V;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    ListWarpSmem<PackT> &sm = s_win[warp];

    // prologue decided by one thread so that the whole CTA agrees
    if (threadIdx.x == 0) {
        int32_t go = ld_volatile_i32(p.status) == 0;  // an earlier error: write nothing
        const int64_t V = __ldg(p.offsets + p.n);
        if (go && V > p.capacity) {
            set_status(p.status, kStCapacity);
            go = 0;
        }
        s_go = go;
        s_V = V;
        s_chunk = list_chunk(V, static_cast<int64_t>(gridDim.x) * kListWarps);
    }
    __syncthreads();
    if (!s_go) return;
    const int64_t V = s_V;
    const int32_t chunk = s_chunk;
    PackT *const list = static_cast<PackT *>(p.list);
    const uint32_t n_warps = gridDim.x * kListWarps;
    const uint32_t le_mask = 0xffffffffu >> (31 - lane);  // this lane and those below

    int64_t g0 = static_cast<int64_t>(blockIdx.x * kListWarps + warp) * chunk;
    while (g0 < V) {
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
                sm.rel[lane] = rel;
                if (lane == wcnt - 1) sm.rel[wcnt] = static_cast<int32_t>(__ldg(p.offsets + s + wcnt) - g0);
                const uint32_t N = static_cast<uint32_t>(max(abs(r[3] - r[0]), max(abs(r[4] - r[1]), abs(r[5] - r[2]))));
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int32_t d = r[3 + a] - r[a];
                    const PackT A = static_cast<PackT>(abs(d));
                    const PackT S = A == N ? PackT(1) << Fix::F  // the major axis, and minor ones as long
                                           : ((A << Fix::F) + (N - 1u)) / N;
                    sm.X0[a][lane] = (static_cast<PackT>(r[a]) << Fix::F) + (PackT(1) << (Fix::F - 1)) - (d < 0 ? 1 : 0);
                    sm.T[a][lane] = d < 0 ? PackT(0) - S : S;
                }
            }
            // the next 32 segments' records and offsets on their way to L1
            if (s + 2 * kListWin <= p.n) {
                if (lane < 24) prefetch_l1(p.segs + 6 * (s + kListWin) + 8 * lane);
                else prefetch_l1(p.offsets + s + kListWin + 4 * (lane - 24));
            }
            __syncwarp();
            const int32_t wend = sm.rel[wcnt];
            int32_t j = 0;  // the window's segment that holds pos
            while (true) {
                // a row needs the window to cover it; without that the window moves on
                // to segment j, or (already there, or the list ends) 32 voxels are taken
                const bool covered = pos + kRow <= min(wend, len);
                if (!covered && j > 0 && wend < len) break;
                // the segments that start in the row after its first voxel, by the first
                // lane whose voxels all follow the start; two of them at one lane: short
                // segments, 32 voxels at a time
                const int32_t b = rel - pos;
                const bool inside = b > 0 && b < kRow;
                const uint32_t starts = __reduce_or_sync(0xffffffffu, inside ? 2u << ((b - 1) / kVox) : 0u);
                if (covered && starts == 0u) {
                    const int32_t e = sm.rel[j + 1];
                    if (e - pos >= kRow) {
                        // rows inside one segment
                        const uint32_t k = static_cast<uint32_t>(pos + kVox * lane - sm.rel[j]);
                        const PackT tx = sm.T[0][j], ty = sm.T[1][j], tz = sm.T[2][j];
                        PackT x = sm.X0[0][j] + k * tx, y = sm.X0[1][j] + k * ty, z = sm.X0[2][j] + k * tz;
                        const int32_t stop = min(e, len) - kRow;
                        int4 *o = reinterpret_cast<int4 *>(out + pos) + lane;
#pragma unroll 2
                        for (; pos <= stop; pos += kRow) {
                            PackT v[kVox];
#pragma unroll
                            for (int i = 0; i < kVox; ++i) {
                                v[i] = Fix::pack(x, y, z);
                                const uint32_t f = i + 1 < kVox ? 1u : static_cast<uint32_t>(kRow - kVox + 1);
                                x += f * tx;
                                y += f * ty;
                                z += f * tz;
                            }
                            *o = list_quad(v);
                            o += 32;
                        }
                        if (pos >= len) break;
                        if (e <= pos) {
                            ++j;
                            if (j >= wcnt) break;
                        }
                        continue;
                    }
                }
                // (a start among the last lane's voxels has no such lane)
                const int32_t n_in = __popc(__ballot_sync(0xffffffffu, inside));
                const int32_t n_last = __popc(__ballot_sync(0xffffffffu, inside && b > kRow - kVox));
                if (covered && n_last <= 1 && __popc(starts) + n_last == n_in) {
                    // a row with segment starts, at most one per lane
                    const int32_t p0 = pos + kVox * lane;
                    const int32_t jl = j + __popc(starts & le_mask);
                    const int32_t c = sm.rel[jl + 1] - p0;  // this lane's voxels from c on are the next segment's
                    const uint32_t k = static_cast<uint32_t>(p0 - sm.rel[jl]);
                    const PackT tx = sm.T[0][jl], ty = sm.T[1][jl], tz = sm.T[2][jl];
                    PackT x = sm.X0[0][jl] + k * tx, y = sm.X0[1][jl] + k * ty, z = sm.X0[2][jl] + k * tz;
                    PackT v[kVox];
#pragma unroll
                    for (int i = 0; i < kVox; ++i) {
                        v[i] = Fix::pack(x, y, z);
                        x += tx;
                        y += ty;
                        z += tz;
                    }
                    if (c < kVox) {
                        const uint32_t back = 0u - static_cast<uint32_t>(c - 1);  // voxel 1 is its step 1 - c
                        const PackT ux = sm.T[0][jl + 1], uy = sm.T[1][jl + 1], uz = sm.T[2][jl + 1];
                        x = sm.X0[0][jl + 1] + mul_signed(back, ux);
                        y = sm.X0[1][jl + 1] + mul_signed(back, uy);
                        z = sm.X0[2][jl + 1] + mul_signed(back, uz);
#pragma unroll
                        for (int i = 1; i < kVox; ++i) {
                            if (i >= c) v[i] = Fix::pack(x, y, z);
                            x += ux;
                            y += uy;
                            z += uz;
                        }
                    }
                    reinterpret_cast<int4 *>(out + pos)[lane] = list_quad(v);
                    pos += kRow;
                    j += n_in;
                } else {
                    // 32 voxels, one per lane (the window covers them: 32 segments hold at
                    // least 32 voxels): a bit for each start, and each lane counts the bits
                    // up to its own position
                    if (wend < len && pos + 32 > wend) break;
                    const uint32_t bits = __reduce_or_sync(0xffffffffu, (b > 0 && b < 32) ? 1u << b : 0u);
                    const int32_t jl = j + __popc(bits & le_mask);
                    const uint32_t k = static_cast<uint32_t>(pos + lane - sm.rel[jl]);
                    const PackT x = sm.X0[0][jl] + k * sm.T[0][jl], y = sm.X0[1][jl] + k * sm.T[1][jl],
                                z = sm.X0[2][jl] + k * sm.T[2][jl];
                    if (pos + lane < len) out[pos + lane] = Fix::pack(x, y, z);
                    pos += 32;
                    j += __popc(bits);
                }
                if (pos >= len) break;
                if (sm.rel[j + 1] <= pos) {  // the next row starts a segment
                    ++j;
                    if (j >= wcnt) break;
                }
            }
            s += j;
        }
        if (static_cast<int64_t>(n_warps) * chunk >= V) break;
        uint32_t next = 0;
        if (lane == 0) next = atomicAdd(p.counter, 1u);
        g0 = (static_cast<int64_t>(n_warps) + __shfl_sync(0xffffffffu, next, 0)) * chunk;
    }
}

}  // namespace vox

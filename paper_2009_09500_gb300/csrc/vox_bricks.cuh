// vox_bricks.cuh -- the occupancy volume by brick ownership (sm_103a).
//
// OR-ing each voxel into the volume with a global atomic costs one L2/DRAM
// read-modify-write of a 32-byte sector per voxel (the volume is far larger than
// L2 for big scenes), which makes the volume store DRAM-bound at a small fraction
// of the bandwidth. Instead the volume is cut into bricks of whole 32-bit words
// (B0 x B1 x B2 voxels, B0 a multiple of 32, at most 32768 words), every segment
// is cut into pieces that stay inside one brick, the pieces are counting-sorted
// by brick, and one CTA owns each brick: it ORs the brick's voxels into a
// shared-memory bitmap and merges the bitmap into the volume in one pass (a TMA
// tensor reduce-OR, or a store of the whole brick for a fresh volume). Each
// volume sector then crosses DRAM at most twice (read + write), whatever the
// number of voxels in it.
//
//   k_bin_count    pieces per slot of a brick (lanes walk segments' pieces, global atomics)
//   k_scan<false>  exclusive scan of the slot counts (decoupled look-back)
//   k_bin_scatter  pieces written into their slot; the segments' slope table
//   k_brick_volume one CTA per brick, or part of one with very many pieces: voxels ->
//                  shared bitmap -> volume
//   k_unbrick_tma  brick-major volume -> row-major volume
//
// A piece is (segment, first step k, length). The steps at which a segment's
// coordinate on an axis enters the next brick follow from the same exact rounding
// as the voxels themselves (Eq. (3) with nearest-lattice rounding): the offset
// q(k) = floor((2 k A + N) / (2 N)) first reaches Q at k = ceil(N (2Q - 1) / (2A)).
#pragma once

#include <cuda.h>

#include <cstdint>
#include <type_traits>

#include "vox_device.cuh"

namespace vox {

constexpr int kBrickThreads = 1024;  // one CTA per SM (the bitmap takes 128 KB)
constexpr int kBrickQuarters = 4;    // z quarters of a brick: stored and cleared by 8 warps each
constexpr int kBrickWordsMax = 32768;  // 128 KB shared bitmap per brick
constexpr int32_t kNoStep = 0x7fffffff;
constexpr int32_t kStPieces = 7;  // VOX_ERR_WORKSPACE: a brick-major volume needs every piece binned

// Edges up to which the slopes below are exact, for N = int(|d|) as well:
// N < sqrt(3) 37837 < 2^16.
constexpr int32_t kSlopeDimMax = 37837;

struct BrickGeom {
    int32_t B[3];       // brick extent in voxels per axis (powers of two, B[0] >= 32)
    int32_t logB[3];    // log2(B[a])
    int32_t nb[3];      // bricks per axis
    int32_t bxw;        // words per brick row, B[0] / 32
    int32_t log_bxw;    // log2(bxw)
    int32_t log_b1;     // log2(B[1])
    int32_t row_words;  // words per volume row, w / 32
    int32_t dim[3];     // volume extent
    int32_t words;      // words per brick, bxw * B[1] * B[2]
    int64_t n_bricks;
    // Pieces are bucketed by slot = (brick, length class, replica), brick-major,
    // classes longest first: after the scan a brick's pieces are contiguous and
    // already ordered by length, so that a warp taking 32 consecutive pieces gets
    // pieces of similar length. Each (brick, class) has `reps` counters (segment
    // s uses replica s % reps) so that atomics on one brick spread over several
    // addresses when there are few bricks with many pieces each.
    int32_t reps;       // 1, 8 or 32 (segment s uses replica s & (reps - 1))
    int32_t wide;       // an edge above kSlopeDimMax: no slope table
    int64_t n_slots;    // n_bricks * kPieceClasses * reps
};

// Slots per replica of a brick: half octaves of the piece length, longest first. Pieces of
// at most kPieceMaxLen steps fill the last 13. The others stay zero; without them single
// volumes gain a little (4M segments: scatter 1127 -> 1097 us, 200,000 in 512^3 39 -> 35), but
// the counting of a batch, whose few bricks take most updates, loses more: five served
// scenes 179 -> 310 and 98 -> 126 us, 256 uneven scenes 192 -> 234 (with 16 slots 282, 130
// and 219). It seems that the busiest counters of neighbouring bricks then share lines.
constexpr int kPieceClasses = 22;
constexpr int64_t kMaxBricks = int64_t(1) << 26;

// Counter replicas per (brick, class): a brick's counters are updated once per piece in
// it, and updates of one address go one after another, so few bricks get more of them.
// Binning of 48 scenes (1.17 M segments, 1,623 bricks in all), one counter per (brick,
// class): 128 + 110 us (scatter, count), eight: 104 + 62 us.
// More of them cost the slot scan what the counting gains (48 scenes with 32: 46 instead
// of 60 us of counting, 15 instead of 7 us of scanning).
constexpr int32_t kBricks32Replicas = 512;
constexpr int32_t kBricks8Replicas = 32768;

__host__ __device__ inline int32_t counter_replicas(int64_t bricks)
{
    return bricks <= kBricks32Replicas ? 32 : (bricks <= kBricks8Replicas ? 8 : 1);
}

// Brick shape for a volume whose rows are whole 32-bit words (w % 32 == 0):
// B0 = the largest 32 * 2^k not above min(w, 256) voxels along x (whole words),
// then B1 x B2 rows (powers of two) so that a brick has at most kBrickWordsMax
// words: 256 x 64 x 64 (128 KB) for wide volumes. Two things set the shape:
// segments in random directions cross the fewer brick faces the more cube-like
// and large the brick is (fewer pieces), and the brick's store writes one
// request per brick row, so rows of 32 bytes (B0 = 256) store about three times
// faster than rows of 16 bytes (measured: 18 against 56 us per 128 MiB volume).
// all_bricks: bricks of the whole batch that the volume belongs to (0: the volume
// alone), which set the counter replicas.
__host__ __device__ inline bool brick_geom(int32_t w, int32_t h, int32_t d, BrickGeom *G, int64_t all_bricks = 0)
{
    if (w < 1 || h < 1 || d < 1 || w % 32 != 0) return false;
    int32_t b0 = 32;
    while (2 * b0 <= w && 2 * b0 <= 256) b0 *= 2;
    G->B[0] = b0;
    G->bxw = b0 / 32;
    G->log_bxw = 0;
    while ((1 << G->log_bxw) < G->bxw) ++G->log_bxw;
    const int32_t rows = kBrickWordsMax / G->bxw;
    int32_t p2 = 1;
    while ((2 * p2) * (2 * p2) <= rows) p2 *= 2;
    G->B[1] = (2 * p2 * p2 <= rows) ? 2 * p2 : p2;
    G->B[2] = p2;
    G->log_b1 = 0;
    while ((1 << G->log_b1) < G->B[1]) ++G->log_b1;
    G->dim[0] = w;
    G->dim[1] = h;
    G->dim[2] = d;
    G->row_words = w / 32;
    G->words = G->bxw * G->B[1] * G->B[2];
    for (int a = 0; a < 3; ++a) {
        G->logB[a] = 0;
        while ((1 << G->logB[a]) < G->B[a]) ++G->logB[a];
    }
    int64_t nb = 1;
    for (int a = 0; a < 3; ++a) {
        G->nb[a] = (G->dim[a] + G->B[a] - 1) / G->B[a];
        nb *= G->nb[a];
    }
    G->n_bricks = nb;
    G->reps = counter_replicas(all_bricks > 0 ? all_bricks : nb);
    G->wide = (w > kSlopeDimMax || h > kSlopeDimMax || d > kSlopeDimMax) ? 1 : 0;
    G->n_slots = nb * kPieceClasses * G->reps;
    return nb <= kMaxBricks && G->words <= kBrickWordsMax;
}

// A scene of a batch as the brick path sees it: its geometry, its
// first brick and first slot in the batch's numbering, and its volume.
struct SceneBricks {
    BrickGeom G;
    int64_t brick_base;
    int64_t slot_base;
    uint32_t *mask;
};

// Length class of a piece, longest first: 0 for the longest half octave.
__device__ __forceinline__ int32_t piece_class_desc(int32_t len)
{
    const uint32_t l = static_cast<uint32_t>(len);
    const int32_t oct = 31 - __clz(l);
    const int32_t cls = 2 * oct + (oct > 0 ? static_cast<int32_t>((l >> (oct - 1)) & 1u) : 0);
    return kPieceClasses - 1 - cls;
}

// The first slot of a piece of the brick (the replica is added to it). Slots fit 31 bits:
// with replicas there are at most 32768 bricks, else at most 2^26 bricks and one replica.
__device__ __forceinline__ uint32_t piece_slot(int32_t reps, int32_t brick, int32_t len)
{
    return (static_cast<uint32_t>(brick) * kPieceClasses + static_cast<uint32_t>(piece_class_desc(len))) *
           static_cast<uint32_t>(reps);
}

// A segment as the brick kernel enters it, one 32-byte sector, written once by the
// scattering pass: its start, directions and per axis the slope S = ceil(A 2^40 / N), so
// that a piece is entered at any step k by a multiplication per axis,
//   q(k) = floor((2 k A + N) / (2 N)) = floor((k S + 2^39) / 2^40),
// and walked by 32-bit fractions. The exact positions are multiples of 1 / 2N and the
// computed ones are above by less than k 2^-40 <= 2^-24, and by 2^-32 more for each of
// the (at most 63) steps walked from there: below 1 / 2N for N < 2^16, so every floor
// and carry is exact. A slope of 1 (A = N) is held as 1 - 2^-40: from the fraction 1/2
// it gives the same floors. Volumes with larger edges enter by division instead.
// Against the segment's record and a division per minor axis (and remainders re-biased
// at every carry), the brick kernel takes 2823 instead of 3087 us on the 4M-segment
// batch; the table is 128 MB there and costs the scattering pass 50 us.
struct alignas(32) SegSlopes {
    uint32_t xy;     // start x | y << 16
    uint32_t z;      // start z | 2^(16 + a) where axis a decreases | major axis << 19 (first with A = N)
    uint32_t hi;     // slopes' bits 32..39, a byte per axis
    uint32_t lo[3];  // slopes' bits 0..31
    uint32_t pad[2];
};

__device__ __forceinline__ SegSlopes make_slopes(const int32_t *rec, int32_t N)
{
    SegSlopes e;
    e.xy = static_cast<uint32_t>(rec[0]) | (static_cast<uint32_t>(rec[1]) << 16);
    e.z = static_cast<uint32_t>(rec[2]);
    e.hi = 0;
    e.pad[0] = e.pad[1] = 0;
    uint32_t major = 3;
    const float rcp = __frcp_rn(static_cast<float>(N));
#pragma unroll
    for (int a = 2; a >= 0; --a) {
        const int32_t d = rec[3 + a] - rec[a], A = abs(d);
        if (d < 0) e.z |= 0x10000u << a;
        uint64_t S = (uint64_t(1) << 40) - 1;
        if (A != N) {  // two digits of 20 bits
            int32_t q1, r1, q2, r2;
            divmod_est(static_cast<uint64_t>(A) << 20, N, rcp, q1, r1);
            divmod_est(static_cast<uint64_t>(r1) << 20, N, rcp, q2, r2);
            S = (static_cast<uint64_t>(q1) << 20) + static_cast<uint32_t>(q2) + (r2 > 0 ? 1 : 0);
        } else {
            major = a;
        }
        e.lo[a] = static_cast<uint32_t>(S);
        e.hi |= static_cast<uint32_t>(S >> 32) << (8 * a);
    }
    e.z |= major << 19;
    return e;
}

// Crossing steps of one axis. The segment's offset on the axis,
// q(k) = floor((2 k A + N) / (2 N)), first reaches Q at
// k = ceil(N (2Q - 1) / (2A)) (for 1 <= Q <= A <= N). Along the segment the
// axis enters a new brick at Q_1, Q_1 + B, Q_1 + 2B, ...: with
// T_j = N (2 Q_j - 1) + 2A - 1 = 2A k_j + rem_j, one division gives k_1 and
// rem_1, and each later crossing follows from T_{j+1} = T_j + 2NB without a
// division, 2NB = 2A qs + rs having been divided once.
struct AxisCrossings {
    int32_t left;  // crossings still ahead
    int32_t nk;    // step of the next crossing (kNoStep when none)
    int32_t rem;   // T_j mod 2A for the crossing at nk
    int32_t qs, rs;
    int32_t twoA;

    // From a voxel whose coordinate on the axis is v on (the step at hand is not needed).
    __device__ __forceinline__ void init(int32_t S, int32_t E, int32_t v, int32_t A, int32_t N, int32_t logB)
    {
        const int32_t b0 = v >> logB, be = E >> logB;  // coordinates are inside the volume (>= 0)
        left = abs(be - b0);
        nk = kNoStep;
        rem = qs = rs = twoA = 0;
        if (left == 0) return;
        const int32_t B = 1 << logB;
        const int32_t Q = be > b0 ? (b0 + 1) * B - S : S - b0 * B + 1;
        // quotients below 2^22: nk <= N, and qs < 2N (there are two crossings B apart, A > B)
        twoA = 2 * A;
        const float rcp = __frcp_rn(static_cast<float>(twoA));
        divmod_est(static_cast<uint64_t>(N) * static_cast<uint64_t>(2 * Q - 1) + static_cast<uint64_t>(twoA - 1), twoA,
                   rcp, nk, rem);
        if (left > 1) divmod_est(2ull * static_cast<uint64_t>(N) * static_cast<uint64_t>(B), twoA, rcp, qs, rs);
    }

    // To the crossing after the one at nk, where `hit`; without a branch, since the lanes
    // of a warp cross different axes at each of their runs.
    __device__ __forceinline__ void advance(bool hit)
    {
        int32_t r = rem + rs, n = nk + qs;
        const bool over = r >= twoA;
        r -= over ? twoA : 0;
        n += over ? 1 : 0;
        left -= hit ? 1 : 0;
        nk = hit ? (left > 0 ? n : kNoStep) : nk;
        rem = hit ? r : rem;
    }
};

// The maximal runs of consecutive steps of one segment that stay in one brick,
// in increasing k: init() at a step, then next() gives one run per
// call. Endpoints must be inside the volume. Brick indices fit 32 bits (at most
// 2^26 bricks). The crossing formula holds for any number of steps N >= max |d_a| (the
// samples of the Euclidean-N variant too).
struct PieceWalker {
    AxisCrossings ax[3];
    int32_t bstep[3];
    int32_t brick, k, N;

    // At the first run that starts at step k0 or later; false when there is none (a
    // segment's first run starts at step 0).
    __device__ __forceinline__ bool init(const int32_t *rec, const BrickGeom &G, int32_t steps, int32_t k0)
    {
        N = steps;
        const float rcp2N = k0 > 1 ? __frcp_rn(static_cast<float>(2 * N)) : 0.0f;
        const int32_t stride[3] = {1, G.nb[0], G.nb[0] * G.nb[1]};
        brick = 0;
        int32_t kn = N + 1;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int32_t A = abs(rec[3 + a] - rec[a]);
            const bool up = rec[3 + a] >= rec[a];
            int32_t v = rec[a];  // the coordinate at step k0 - 1 (at step 0 when k0 is 0 or 1)
            if (k0 > 1) {
                int32_t q, r;
                axis_entry(A, N, k0 - 1, rcp2N, q, r);
                v = up ? v + q : v - q;
            }
            brick += (v >> G.logB[a]) * stride[a];
            bstep[a] = up ? stride[a] : -stride[a];
            ax[a].init(rec[a], rec[3 + a], v, A, N, G.logB[a]);
            kn = min(kn, ax[a].nk);
        }
        k = 0;
        if (k0 == 0) return true;
        if (kn > N) return false;
        enter(kn);
        return true;
    }

    // The run that starts at step kn, where some axis enters its next brick.
    __device__ __forceinline__ void enter(int32_t kn)
    {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const bool hit = ax[a].nk == kn;
            brick += hit ? bstep[a] : 0;
            ax[a].advance(hit);
        }
        k = kn;
    }

    // The current run (brick b, first step k_lo, len steps); advances to the
    // next one and returns false if this run was the segment's last.
    __device__ __forceinline__ bool next(int32_t &b, int32_t &k_lo, int32_t &len)
    {
        const int32_t kn = min(min(ax[0].nk, ax[1].nk), min(ax[2].nk, N + 1));
        b = brick;
        k_lo = k;
        len = kn - k;
        if (kn > N) return false;
        enter(kn);
        return true;
    }
};

// Pieces are at most kPieceMaxLen steps long: a longer run in one brick is cut
// into parts of kPieceMaxLen (the last one shorter), so that no lane of the
// brick kernel walks a long piece while the rest of its CTA waits.
constexpr int32_t kPieceMaxLen = 64;

// piece = segment (32 bits) | first step (22 bits) | length - 1 (10 bits)
__device__ __forceinline__ uint64_t pack_piece(uint32_t seg, int32_t k_lo, int32_t len)
{
    return static_cast<uint64_t>(seg) | (static_cast<uint64_t>(k_lo) << 32) |
           (static_cast<uint64_t>(len - 1) << 54);
}

__device__ __forceinline__ bool endpoints_inside(const int32_t *r, const BrickGeom &G)
{
    return (unsigned)r[0] < (unsigned)G.dim[0] && (unsigned)r[3] < (unsigned)G.dim[0] &&
           (unsigned)r[1] < (unsigned)G.dim[1] && (unsigned)r[4] < (unsigned)G.dim[1] &&
           (unsigned)r[2] < (unsigned)G.dim[2] && (unsigned)r[5] < (unsigned)G.dim[2];
}

// A brick with more than hot_pieces(total) pieces is walked in parts of about that many
// by several CTAs, whose bitmaps are OR-ed into the volume (cleared beforehand when it
// is a fresh one): scenes in small volumes put all their pieces into a few bricks, and
// one CTA walks a piece in about 4 ns. Brick kernel, us, whole bricks against parts:
// 50,000 segments in 64^3 (one brick) 202 -> 18; 100,000 in 256^3 (16 bricks) 173 -> 32;
// 48 uneven scenes 500 -> 240; 200,000 in 512^3 (128 bricks) 105 -> 87. With 1/256 of
// all pieces as the limit there are at most 2 * 256 parts (1/128: 43 us in 256^3).
constexpr int64_t kHotMin = 1024;
constexpr int kHotParts = 512;
struct HotPart {
    int64_t brick, lo, hi;  // the pieces [lo, hi) of a brick
};

__device__ __forceinline__ int64_t hot_pieces(int64_t total) { return max(kHotMin, (total + kHotParts / 2 - 1) / (kHotParts / 2)); }

struct BinParams {
    const int32_t *segs;
    int64_t n;
    BrickGeom G;
    int32_t *brick_count;     // [n_slots], zeroed before k_bin_count
    int64_t *cursor;          // [n_slots], exclusive offsets (k_bin_scatter bumps them)
    const int64_t *brick_off; // [n_slots + 1]; brick_off[n_slots] = number of pieces
    uint64_t *pieces;         // [capacity]
    int64_t capacity;
    const int32_t *status;
    SegSlopes *slopes;        // [n], written by the scattering pass
    HotPart *hot;             // [kHotParts] and their number (zeroed before the launch)
    uint32_t *n_hot;
    uint32_t *mask;           // the volume, and how it is written (as in BrickParams)
    int32_t fresh, bricked;
    const SceneBricks *sb;    // batched: each scene's geometry and numbering (else null)
    const int32_t *scene_of;  // batched: scene of every segment
    const int32_t *brick_scene;  // batched: scene of every brick
    int32_t n_scenes;
};

// The geometry a segment's pieces follow and the first slot of its volume, or
// null for a segment outside every scene (only after a table error, which the
// status word holds; the batched kernels check it first).
template <bool kBatched>
__device__ __forceinline__ const BrickGeom *segment_geom(const BinParams &p, int64_t s, int64_t &slot_base)
{
    if constexpr (kBatched) {
        const int32_t k = __ldg(p.scene_of + s);
        if (static_cast<uint32_t>(k) >= static_cast<uint32_t>(p.n_scenes)) return nullptr;
        slot_base = p.sb[k].slot_base;
        return &p.sb[k].G;
    } else {
        slot_base = 0;
        return &p.G;
    }
}

// Binning work loop, shared by the counting and the scattering pass (CTAs of
// kBinThreads threads, persistent grid). A warp takes batches of 32 kPer consecutive
// segments and cuts their steps into units of kBinUnit, the last one of a segment
// shorter; a lane walks a unit: the runs (maximal runs of steps in one brick) that start
// in it, entering the segment there by one division per axis. The whole units first,
// 32 a round, dealt out over the lanes whichever segment they belong to, then every
// segment's last unit, ordered by length octave: the lanes of a round walk about as many
// runs each, whatever the mix of lengths (log-uniform lengths span three orders of
// magnitude). emit(slot, seg, k_lo, len) is called for every piece (runs cut to at most
// kPieceMaxLen steps) with its slot in the batch's slot numbering. A segment with an
// endpoint outside its volume has no pieces (the count kernel reports it).
// Bound by the L2's atomics where segments are long (counting 57 M pieces: 1.4e11
// updates/s), else by the walk's instructions. Counting + scattering pass, us, against
// a lane per segment in batches of 128 sorted by octave, with a branch per axis at
// every run's end and four reservations in flight:
//   4M log-uniform segments, 4096^3 (57 M pieces)   461 + 1295 -> 415 + 1072
//   1M log-uniform segments, 2048^3                  73 +  222 ->  83 +  187
//   48 uneven scenes (1.17 M segments)              132 +  196 ->  59 +  100
//   200,000 uniform segments, 512^3                  35 +   50 ->  22 +   30
//   1,000 uniform segments, 512 x 300 x 200          13 +   33 ->   7 +   13
// kPer segments per lane and batch: more of them fill the rounds of equal octaves
// better, fewer keep more warps busy. launch_bin_t scatters with two at any size (with
// four: 48 uneven scenes 110 against 100 us, 5 scenes of 1.3 M segments 241 against 203, 1M
// 64-voxel segments 51 against 49, log-uniform 3M 859 against 839; 4M with one 1191). It
// counts with two up to 2^20 segments and with four beyond (two against four, us):
//   log-uniform, 2048^3   0.7M 61 : 65,  1.1M  91 :  92,  1.3M 106 :  97,  2.5M 195 : 180,  5M 384 : 342
//   64 voxels, 1024^3     0.7M 22 : 25,  1.1M  30 :  32,  1.3M  31 :  31,  2.5M  54 :  54,  5M 108 : 107
//   uniform, 512^3        0.7M 60 : 64,  1.1M 113 : 114,  1.3M 120 : 122,  2.5M 249 : 248,  5M 475 : 478
//   five served scenes    1.3M 156 : 159,  1.7M 139 : 139, 228 : 210, 232 : 214 and 212 : 194,  2.2M 252 : 240
//   40, 60, 80, 110, 256 uneven scenes   40 : 41,  59 : 60,  76 : 82,  107 : 104,  218 : 207
// A lane per piece, its step and brick found by fixed-point slopes, takes about 300
// instructions a piece (779 + 1128 us on the first).
constexpr int kBinThreads = 256;
constexpr int kBinWarps = kBinThreads / 32;
constexpr int kBinCtas = 4;                // CTAs per SM
constexpr int kBinUnit = 512;              // steps
constexpr int kBinOctaves = 10;            // of a last unit's steps, 1 .. kBinUnit

template <int kPer>
struct BinWarpSmem {
    static constexpr int kBatch = 32 * kPer;
    int32_t rec[6][kBatch];   // the batch's segments
    int32_t N[kBatch];
    uint8_t last[kBatch];     // segments by the octave of their last unit, longest first
    uint8_t longs[kBatch];    // segments with whole units
    int32_t hist[32];
};

// Volumes of at most kFewBricks bricks: the lanes of a warp mostly ask for a few slots,
// so those that ask for the same one together share one update (and the segments of a
// warp one replica). Scattering and counting pass, us: 50,000 segments in 64^3 14 + 8 ->
// 9 + 4, 48 uneven scenes 117 + 59 -> 106 + 53.
constexpr int64_t kFewBricks = 8;

// The lanes active here with the same slot: the group, its leader, and the lane's rank.
struct SlotGroup {
    uint32_t lanes;
    int leader, rank;

    __device__ __forceinline__ explicit SlotGroup(int64_t slot)
    {
        lanes = __match_any_sync(__activemask(), static_cast<unsigned long long>(slot));
        leader = __ffs(lanes) - 1;
        rank = __popc(lanes & ((1u << (threadIdx.x & 31)) - 1u));
    }
};

// One lane's unit: the runs of segment j (in the batch) that start at steps
// k0 .. k0 + kBinUnit - 1.
template <bool kBatched, int kPer, typename Emit>
__device__ __forceinline__ void bin_unit(const BinParams &p, const BinWarpSmem<kPer> &sm, int64_t b0, int j, int32_t k0,
                                         Emit &emit)
{
    const int64_t s = b0 + j;
    int64_t slot_base;
    const BrickGeom *Gp = segment_geom<kBatched>(p, s, slot_base);
    const bool few = Gp->n_bricks <= kFewBricks;
    const int32_t reps = Gp->reps;
    const int64_t base = slot_base + (static_cast<int32_t>(few ? s >> 5 : s) & (reps - 1));
    int32_t r[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) r[a] = sm.rec[a][j];
    PieceWalker pw;
    bool more = pw.init(r, *Gp, sm.N[j], k0);
    int32_t b = 0, k_lo = 0, len = 0;
    while (true) {  // a piece per iteration
        if (len == 0) {
            if (!more || pw.k >= k0 + kBinUnit) break;
            more = pw.next(b, k_lo, len);
        }
        const int32_t part = min(len, kPieceMaxLen);
        emit(base + piece_slot(reps, b, part), static_cast<uint32_t>(s), k_lo, part, few);
        k_lo += part;
        len -= part;
    }
}

template <bool kEuclid, bool kBatched, bool kSlopes, int kPer, typename Emit>
__device__ __forceinline__ void bin_loop(const BinParams &p, Emit &&emit)
{
    constexpr int kBatch = 32 * kPer;
    __shared__ BinWarpSmem<kPer> s_bin[kBinWarps];
    const int lane = threadIdx.x & 31;
    BinWarpSmem<kPer> &sm = s_bin[threadIdx.x >> 5];
    const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const uint32_t lt_mask = (1u << lane) - 1u, le_mask = lt_mask | (1u << lane);
    for (int64_t b0 = gw * kBatch; b0 < p.n; b0 += nw * kBatch) {
        sm.hist[lane] = 0;
        __syncwarp();
        // ---- the batch's segments; those with whole units; each one's rank in the
        // octave of its last unit
        int32_t oct[kPer], rank[kPer];
        int32_t n_long = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int j = i * 32 + lane;
            oct[i] = -1;
            rank[i] = 0;
            bool is_long = false;
            if (b0 + j < p.n) {
                int32_t r[6];
                load_record(p.segs, b0 + j, r);
                int64_t slot_base;
                const BrickGeom *G = segment_geom<kBatched>(p, b0 + j, slot_base);
                if (G != nullptr && endpoints_inside(r, *G)) {
                    int32_t N = max(abs(r[3] - r[0]), max(abs(r[4] - r[1]), abs(r[5] - r[2])));
                    if constexpr (kEuclid) N = euclid_steps(r);
#pragma unroll
                    for (int a = 0; a < 6; ++a) sm.rec[a][j] = r[a];
                    sm.N[j] = N;
                    if (kSlopes && G->wide == 0) p.slopes[b0 + j] = make_slopes(r, N);
                    is_long = N >= kBinUnit;
                    oct[i] = kBinOctaves - 1 - (31 - __clz(N % kBinUnit + 1));
                    rank[i] = atomicAdd(&sm.hist[oct[i]], 1);
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, is_long);
            if (is_long) sm.longs[n_long + __popc(m & lt_mask)] = static_cast<uint8_t>(j);
            n_long += __popc(m);
        }
        __syncwarp();
        // octave starts: exclusive scan of the octave counts (one per lane)
        const int32_t h = sm.hist[lane];
        int32_t inc = h;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int32_t n_valid = __shfl_sync(0xffffffffu, inc, 31);
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int32_t start = __shfl_sync(0xffffffffu, inc - h, max(oct[i], 0));
            if (oct[i] >= 0) sm.last[start + rank[i]] = static_cast<uint8_t>(i * 32 + lane);
        }
        __syncwarp();
        // ---- whole units: 32 long segments at a time, 32 units a round
#pragma unroll 1
        for (int32_t l0 = 0; l0 < n_long; l0 += 32) {
            const int32_t own = l0 + lane < n_long ? sm.N[sm.longs[l0 + lane]] / kBinUnit : 0;
            int32_t end = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, end, o);
                if (lane >= o) end += y;
            }
            const int32_t total = __shfl_sync(0xffffffffu, end, 31);
            const int32_t pre = own > 0 ? end - own : 0x7fffffff;  // units of the segments before it
#pragma unroll 1
            for (int32_t base = 0; base < total; base += 32) {
                // the lane's segment: the last one whose first unit is at or before its unit
                const int32_t d = pre - base;
                const uint32_t starts = __reduce_or_sync(0xffffffffu, (d > 0 && d < 32) ? 1u << d : 0u);
                const int32_t c = __popc(__ballot_sync(0xffffffffu, d <= 0)) - 1 + __popc(starts & le_mask);
                const int32_t first = __shfl_sync(0xffffffffu, pre, c);
                if (base + lane < total)
                    bin_unit<kBatched>(p, sm, b0, sm.longs[l0 + c], (base + lane - first) * kBinUnit, emit);
                __syncwarp();
            }
        }
        // ---- every segment's last unit
#pragma unroll 1
        for (int32_t q = lane; q < n_valid; q += 32) {
            const int j = sm.last[q];
            bin_unit<kBatched>(p, sm, b0, j, sm.N[j] & ~(kBinUnit - 1), emit);
        }
        __syncwarp();  // the warp's shared arrays are free for the next batch
    }
}

// Pieces per slot (persistent grid).
template <bool kEuclid, bool kBatched, int kPer>
__global__ void __launch_bounds__(kBinThreads, kBinCtas) k_bin_count(BinParams p)
{
    // single volume: no status check (this pass may run beside the count + scan
    // that resets the status word); it reads only the segments and the host's
    // geometry, writes only the slot counts, and skips segments with endpoints
    // outside the volume (reported by the count kernel)
    // a batch reads the scene map and numbering, valid only without an error
    // (decided by the whole warp: the walk's shuffles and votes need every lane)
    if (kBatched && __any_sync(0xffffffffu, ld_volatile_i32(p.status) != 0)) return;
    bin_loop<kEuclid, kBatched, false, kPer>(p, [&](int64_t slot, uint32_t, int32_t, int32_t, bool few) {
        if (few) {
            const SlotGroup g(slot);
            if (g.rank == 0) atomicAdd(p.brick_count + slot, __popc(g.lanes));
        } else {
            atomicAdd(p.brick_count + slot, 1);
        }
    });
}

// Part c of n of a brick's words in a fresh volume set to zero, by a warp.
__device__ __forceinline__ void clear_brick(const BrickGeom &G, int64_t lb, uint32_t *mask, bool bricked, int32_t c,
                                            int32_t n)
{
    const int lane = threadIdx.x & 31;
    const int64_t rest = lb / G.nb[0];
    const int32_t X = static_cast<int32_t>(lb - rest * G.nb[0]) * G.bxw;
    const int32_t Y0 = static_cast<int32_t>(rest % G.nb[1]) * G.B[1], Z0 = static_cast<int32_t>(rest / G.nb[1]) * G.B[2];
    const int32_t plane = G.words / G.B[2];  // words per z
    const int32_t nz = bricked ? G.B[2] : min(G.B[2], G.dim[2] - Z0);
    const int32_t q0 = plane * (nz * c / n), q1 = plane * (nz * (c + 1) / n);
    const bool quads = bricked || ((G.bxw & 3) == 0 && (G.row_words & 3) == 0 && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0);
    const int32_t unit = quads ? 4 : 1;
#pragma unroll 4
    for (int32_t q = q0 + lane * unit; q < q1; q += 32 * unit) {
        uint32_t *w = mask + lb * G.words + q;
        if (!bricked) {
            const int32_t row = q >> G.log_bxw, x = X + (q & (G.bxw - 1));
            const int32_t y = Y0 + (row & (G.B[1] - 1)), z = Z0 + (row >> G.log_b1);
            if (y >= G.dim[1] || x >= G.row_words) continue;
            w = mask + x + static_cast<int64_t>(G.row_words) * (y + static_cast<int64_t>(G.dim[1]) * z);
        }
        if (quads) *reinterpret_cast<uint4 *>(w) = make_uint4(0u, 0u, 0u, 0u);
        else *w = 0u;
    }
}

// A hot brick of a fresh volume is cleared by 2^clear_split warps (one clears 64 KB in 20
// to 150 us).
__host__ __device__ inline int32_t clear_split(bool fresh, int64_t n_bricks) { return fresh && n_bricks <= 4096 ? 5 : 0; }

// The bricks to be walked in parts: their parts listed, their words of a fresh volume
// cleared. Task i = (brick, part of the clearing) goes to warp i mod (warps of the grid),
// a lane each; the grid has a lane for every task as far as the CTAs are resident
// (launch_bin_t), since a round costs two dependent loads: 500 segments in a fresh 1024^3
// volume (1,024 bricks) took 183 us a call by the one CTA that their number fills, 130 so.
template <bool kBatched>
__device__ __forceinline__ void find_hot(const BinParams &p)
{
    const int lane = threadIdx.x & 31;
    const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    const int64_t total = __ldg(p.brick_off + p.G.n_slots), limit = hot_pieces(total);
    if (total <= limit) return;  // no brick has more
    const int64_t slots = static_cast<int64_t>(kPieceClasses) * p.G.reps;
    const int32_t log_split = clear_split(p.fresh != 0, p.G.n_bricks), split = 1 << log_split;
    const int64_t tasks = p.G.n_bricks << log_split;
    for (int64_t i0 = gw; i0 < tasks; i0 += 32 * nw) {
        const int64_t i = i0 + lane * nw, b = i >> log_split;
        int64_t lo = 0, hi = 0;
        if (i < tasks) {
            lo = __ldg(p.brick_off + b * slots);
            hi = __ldg(p.brick_off + (b + 1) * slots);
        }
        uint32_t hot = __ballot_sync(0xffffffffu, hi - lo > limit);
        if (hi - lo > limit && (i & (split - 1)) == 0) {
            const int32_t parts = static_cast<int32_t>((hi - lo + limit - 1) / limit);
            const int64_t per = ((hi - lo + parts - 1) / parts + 31) & ~int64_t(31);
            const uint32_t at = atomicAdd(p.n_hot, static_cast<uint32_t>(parts));
            for (int32_t e = 0; e < parts; ++e)  // in bounds: see kHotParts
                p.hot[at + e] = HotPart{b, min64(lo + e * per, hi), min64(lo + (e + 1) * per, hi)};
        }
        while (p.fresh && hot) {
            const int64_t t = i0 + (__ffs(hot) - 1) * nw, hb = t >> log_split;
            const int32_t c = static_cast<int32_t>(t & (split - 1));
            hot &= hot - 1;
            if constexpr (kBatched) {
                const int32_t k = __ldg(p.brick_scene + hb);
                if (p.sb[k].mask != nullptr)
                    clear_brick(p.sb[k].G, hb - p.sb[k].brick_base, p.sb[k].mask, false, c, split);
            } else {
                clear_brick(p.G, hb, p.mask, p.bricked != 0, c, split);
            }
        }
    }
}

// Pieces written into their slots (persistent grid), and the slope table. p.G.n_slots: the number of
// slots (all scenes' when batched). Bound by the latency of the returning atomics:
// slot reservations of two pieces of a lane are in flight together before their
// stores (4M log-uniform segments: 1134 us; one: 1198; four, or one held while the walk
// goes on: 9 to 10 % more). The first of the two waits in shared memory: in registers the
// batched instance spills (serve-sized batches of five scenes 219 -> 206 us, 48 uneven
// scenes 103 -> 98).
template <bool kEuclid, bool kBatched, int kPer>
__global__ void __launch_bounds__(kBinThreads, kBinCtas) k_bin_scatter(BinParams p)
{
    // an earlier error: write nothing (decided by the whole warp, whose walk takes
    // shuffles and votes; the status word may be set by a kernel on another stream)
    if (__any_sync(0xffffffffu, ld_volatile_i32(p.status) != 0)) return;
    if (__ldg(p.brick_off + p.G.n_slots) > p.capacity) return;  // the volume falls back to atomics
    find_hot<kBatched>(p);
    __shared__ ulonglong2 s_pending[kBinThreads];  // a slot and its piece per thread
    bool pending = false;
    auto reserve = [&](uint64_t slot, uint64_t pieces) {
        return atomicAdd(reinterpret_cast<unsigned long long *>(p.cursor + slot), static_cast<unsigned long long>(pieces));
    };
    bin_loop<kEuclid, kBatched, true, kPer>(p, [&](int64_t slot, uint32_t seg, int32_t k, int32_t len, bool few) {
        if (few) {
            const SlotGroup g(slot);
            unsigned long long at = 0;
            if (g.rank == 0) at = reserve(slot, __popc(g.lanes));
            at = __shfl_sync(g.lanes, at, g.leader);
            p.pieces[at + g.rank] = pack_piece(seg, k, len);
            return;
        }
        const uint64_t piece = pack_piece(seg, k, len);
        if (pending) {
            const ulonglong2 first = s_pending[threadIdx.x];
            const unsigned long long at0 = reserve(first.x, 1), at1 = reserve(slot, 1);
            p.pieces[at0] = first.y;
            p.pieces[at1] = piece;
        } else {
            s_pending[threadIdx.x] = make_ulonglong2(static_cast<uint64_t>(slot), piece);
        }
        pending = !pending;
    });
    if (pending) p.pieces[reserve(s_pending[threadIdx.x].x, 1)] = s_pending[threadIdx.x].y;
}

struct BrickParams {
    const int32_t *segs;
    const SegSlopes *slopes;
    BrickGeom G;
    const int64_t *brick_off;  // [n_slots + 1]
    const uint64_t *pieces;
    int64_t capacity;
    uint32_t *mask;
    int32_t *status;
    uint32_t *ticket;  // zeroed before launch
    const HotPart *hot;      // bricks walked in parts, and the number of parts
    const uint32_t *n_hot;
    int32_t use_tma;   // merge by one TMA tensor reduce-OR (or store) per brick (tensor map valid)
    int32_t fresh;     // write every brick (zeros included) instead of OR-ing into the volume
    int32_t bricked;   // brick-major volume: brick b is words `words` at mask + b * words (one bulk copy)
    const SceneBricks *sb;       // batched: each scene's geometry, numbering and volume (G.n_slots,
    int32_t n_scenes;            // G.n_bricks: the batch's totals; merged by plain stores)
    const int32_t *brick_scene;  // batched: the scene of every brick
};

// TMA tensor reduction of a whole brick tile from shared memory into the volume:
// every word of the box (bxw x B1 x B2 words at word coordinates x, y, z) is
// OR-ed into global memory by the L2, asynchronously; parts of the box outside
// the volume are skipped by the hardware.
__device__ __forceinline__ void tma_reduce_or_3d(const CUtensorMap *tmap, const void *smem, int32_t x, int32_t y,
                                                 int32_t z)
{
    asm volatile(
        "cp.reduce.async.bulk.tensor.3d.global.shared::cta.or.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
            reinterpret_cast<uint64_t>(tmap)),
        "r"(x), "r"(y), "r"(z), "r"(smem_addr(smem))
        : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// ... and the 1-D form, OR-ing into global memory.
__device__ __forceinline__ void bulk_reduce_or_1d(void *gmem, const void *smem, uint32_t bytes)
{
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.or.b32 [%0], [%1], %2;" ::"l"(
                     reinterpret_cast<uint64_t>(gmem)),
                 "r"(smem_addr(smem)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// 1-D bulk copy of a whole brick bitmap to global memory (brick-major volume);
// both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_store_1d(void *gmem, const void *smem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(reinterpret_cast<uint64_t>(gmem)),
                 "r"(smem_addr(smem)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// TMA tensor store of a whole brick tile (the volume's previous content there is
// replaced); parts of the box outside the volume are skipped by the hardware.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *tmap, const void *smem, int32_t x, int32_t y, int32_t z)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(z), "r"(smem_addr(smem))
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ bool is_zero(uint32_t v) { return v == 0u; }
__device__ __forceinline__ bool is_zero(uint4 v) { return (v.x | v.y | v.z | v.w) == 0u; }
__device__ __forceinline__ uint32_t or_units(uint32_t a, uint32_t b) { return a | b; }
__device__ __forceinline__ uint4 or_units(uint4 a, uint4 b)
{
    return make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w);
}

// A brick's bitmap into the volume, in units T of 2^log_t words, kGroup units per thread
// at a time: OR-ed into the units that it touches (their loads are all issued before the
// stores, so DRAM latency is paid once per group, not once per unit), or (kFresh) every
// unit inside the volume stored. (The arrays start as zeros: left undefined, the kernel
// spills 500 bytes.)
template <typename T, int log_t, int kGroup, bool kFresh>
__device__ __forceinline__ void merge_units(const uint32_t *bits, const BrickGeom &G, int32_t X0, int32_t Y0, int32_t Z0,
                                            uint32_t *mask)
{
    const T *const from = reinterpret_cast<const T *>(bits);
    T *const to = reinterpret_cast<T *>(mask);
    const int32_t units = G.words >> log_t, log_bx = G.log_bxw - log_t, row_units = G.row_words >> log_t;
    const int32_t x0 = X0 / (32 << log_t);
    for (int q0 = 0; q0 < units; q0 += kGroup * kBrickThreads) {
        T v[kGroup], old[kGroup];
        int64_t at[kGroup];
        bool wr[kGroup];
#pragma unroll
        for (int e = 0; e < kGroup; ++e) {
            const int q = q0 + e * kBrickThreads + static_cast<int>(threadIdx.x);
            v[e] = old[e] = T{};
            at[e] = 0;
            wr[e] = false;
            if (q < units) {
                v[e] = from[q];
                const int32_t row = q >> log_bx, col = q & ((1 << log_bx) - 1);
                const int32_t y = Y0 + (row & (G.B[1] - 1)), z = Z0 + (row >> G.log_b1);
                if ((kFresh || !is_zero(v[e])) && y < G.dim[1] && z < G.dim[2] && x0 + col < row_units) {
                    wr[e] = true;
                    at[e] = x0 + col + static_cast<int64_t>(row_units) * (y + static_cast<int64_t>(G.dim[1]) * z);
                }
            }
        }
        if constexpr (!kFresh) {
#pragma unroll
            for (int e = 0; e < kGroup; ++e)
                if (wr[e]) old[e] = to[at[e]];
        }
#pragma unroll
        for (int e = 0; e < kGroup; ++e)
            if (wr[e]) to[at[e]] = kFresh ? v[e] : or_units(old[e], v[e]);
    }
}

// Merge a brick's shared bitmap into the volume. Brick row (ly, lz) holds bxw words that
// are contiguous in the volume; a warp covers 32 consecutive words, or 32 consecutive
// 16-byte units where rows and the volume allow them: the brick's first word in a row,
// X0 / 32, is a multiple of bxw and the volume's rows are whole units, so every unit is
// aligned and lies in or beyond the row as a whole. The brick owns its words: plain loads
// and stores suffice.
// Units per thread at a time: two of 16 bytes, of words four to store and six to OR (with
// eight the batched kernel spills). Brick kernel, us, against one loop for both kinds of
// volume with four units of 16 bytes or eight words: 3,000 segments in 1600^3 (words)
// fresh 299 -> 263, OR-ed into 272 -> 276; 200,000 380 -> 343 and 470 -> 467; 40 scenes in
// 512 x 500 x 480 fresh 247 -> 231, 324 -> 313.
__device__ __forceinline__ void merge_brick(const uint32_t *bits, const BrickGeom &G, int32_t X0, int32_t Y0,
                                            int32_t Z0, uint32_t *mask, bool fresh)
{
    if ((G.bxw & 3) == 0 && (G.row_words & 3) == 0 && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0) {
        if (fresh) merge_units<uint4, 2, 2, true>(bits, G, X0, Y0, Z0, mask);
        else merge_units<uint4, 2, 2, false>(bits, G, X0, Y0, Z0, mask);
    } else {
        if (fresh) merge_units<uint32_t, 0, 4, true>(bits, G, X0, Y0, Z0, mask);
        else merge_units<uint32_t, 0, 6, false>(bits, G, X0, Y0, Z0, mask);
    }
}

// Merge the bitmap of a part of a brick: its nonzero words OR-ed into the volume by
// reductions (other parts' CTAs do the same).
__device__ __forceinline__ void merge_part(const uint32_t *bits, const BrickGeom &G, int32_t X0, int32_t Y0, int32_t Z0,
                                           uint32_t *mask)
{
    for (int q = threadIdx.x; q < G.words; q += kBrickThreads) {
        const uint32_t v = bits[q];
        const int32_t row = q >> G.log_bxw, x = X0 / 32 + (q & (G.bxw - 1));
        const int32_t y = Y0 + (row & (G.B[1] - 1)), z = Z0 + (row >> G.log_b1);
        if (v != 0u && y < G.dim[1] && z < G.dim[2] && x < G.row_words)
            atomicOr(mask + x + static_cast<int64_t>(G.row_words) * (y + static_cast<int64_t>(G.dim[1]) * z), v);
    }
}

// A brick taken from the ticket counter: its index, its pieces [lo, hi) and its
// origin (and, in a batch, its scene's geometry and volume).
struct BrickInfo {
    int64_t brick;       // (n_bricks when there is none left)
    int32_t part;        // a part of a brick
    int32_t skip;        // a brick that is walked in parts
    int64_t lo, hi;
    int32_t origin[3];
    BrickGeom geom;      // batched: the brick's scene geometry
    uint32_t *bmask;     // batched: the scene's volume
};

struct BrickSmem {
    alignas(128) uint32_t bits[kBrickWordsMax];  // also the TMA source tile (128-byte aligned)
    BrickInfo info[3];   // a ring: the brick in hand, the next one, and the one after (taken ahead)
    int32_t next_group;  // next group of 32 pieces of the brick to hand to a warp
    int32_t n_hot;       // parts of bricks (the first tickets), and the pieces beyond which
    int64_t hot_limit;   // a brick is walked in parts (both for the thread that takes tickets)
};

// Take the next brick ticket and describe the brick (one thread).
template <bool kBatched>
__device__ __forceinline__ void take_brick(const BrickParams &p, bool overflow, BrickSmem &sm, BrickInfo &I)
{
    const int64_t ticket = atomicAdd(p.ticket, 1u);
    const int64_t n_hot = sm.n_hot;
    I.part = ticket < n_hot;
    const int64_t b = I.part ? p.hot[ticket].brick : min64(ticket - n_hot, p.G.n_bricks);
    I.brick = b;
    if (b >= p.G.n_bricks) return;
    int64_t lb = b;  // the brick's index in its volume
    const BrickGeom *Gt = &p.G;
    int64_t first_slot;
    if constexpr (kBatched) {  // the brick's scene and its geometry
        const int32_t k = __ldg(p.brick_scene + b);
        // word by word: the thread's walk waits with its state in registers
        const int32_t *from = reinterpret_cast<const int32_t *>(&p.sb[k].G);
        int32_t *to = reinterpret_cast<int32_t *>(&I.geom);
#pragma unroll 1
        for (int i = 0; i < static_cast<int>(sizeof(BrickGeom) / 4); ++i) to[i] = from[i];
        I.bmask = p.sb[k].mask;
        lb = b - p.sb[k].brick_base;
        first_slot = p.sb[k].slot_base + lb * kPieceClasses * I.geom.reps;
        Gt = &I.geom;
    } else {
        first_slot = b * kPieceClasses * p.G.reps;
    }
    const int64_t rest = lb / Gt->nb[0];
    I.origin[0] = static_cast<int32_t>(lb - rest * Gt->nb[0]) * Gt->B[0];
    I.origin[1] = static_cast<int32_t>(rest % Gt->nb[1]) * Gt->B[1];
    I.origin[2] = static_cast<int32_t>(rest / Gt->nb[1]) * Gt->B[2];
    const int64_t slots_per_brick = static_cast<int64_t>(kPieceClasses) * Gt->reps;
    if (I.part) {
        I.lo = p.hot[ticket].lo;
        I.hi = p.hot[ticket].hi;
        I.skip = 0;
    } else {
        I.lo = overflow ? 0 : __ldg(p.brick_off + first_slot);
        I.hi = overflow ? 0 : __ldg(p.brick_off + first_slot + slots_per_brick);
        I.skip = I.hi - I.lo > sm.hot_limit;
    }
}

// One CTA per brick, or part of a brick (HotPart; dynamic tickets, the parts first, taken
// two bricks ahead by the last warp while the others walk, so that no barrier waits for
// a ticket). The brick's
// pieces arrive ordered by length class, longest first (the bucket order of the
// binning). Group w of 32 consecutive pieces goes to warp w, further groups to
// the warps that ask a shared counter first: the lanes of a warp walk pieces of
// similar length (at most kPieceMaxLen steps), longest groups first. A
// warp's first group of the next brick is loaded while it walks the current one
// (its pieces during the walk, their segments' slopes after it), so that, with
// about as many groups per brick as warps, most groups start without waiting
// for global memory. Each lane enters its piece's segment at the piece's first
// step and steps through the piece by the carries of its fractions (SegSlopes),
// OR-ing bits into the brick's shared bitmap; the bitmap is then merged into the
// volume, each z quarter by a copy of its own, so that the next brick clears a
// quarter while the others are still being read.
// Bound by the shared memory's atomics (32 random words take 3.5 wavefronts of two
// cycles: 4.8 voxels per cycle and SM, 1.37 ms of the 4M-segment batch's 2.68 ms), and
// by the CTA's wait for its longest group and for its own store between bricks. The
// walk must not spill: 24 bytes at 64 registers cost 2.89 -> 3.29 ms. No instance does
// (the batched one spilled 28 bytes, most of them where bricks are merged and tickets
// taken: 48 uneven scenes 243 -> 231 us without, five served scenes 378 -> 369).
template <bool kEuclid, bool kBatched, bool kWide>
__global__ void __launch_bounds__(kBrickThreads) k_brick_volume(const __grid_constant__ BrickParams p,
                                                                const __grid_constant__ CUtensorMap tmap)
{
    extern __shared__ __align__(128) unsigned char brick_smem_raw[];
    BrickSmem &sm = *reinterpret_cast<BrickSmem *>(brick_smem_raw);
    const int t = threadIdx.x;
    const int lane = t & 31;
    const int warp = t >> 5;
    // an earlier error: write nothing, decided by the whole CTA (the status word may
    // be set meanwhile by a kernel on another stream, and the CTA meets at barriers)
    if (__syncthreads_or(ld_volatile_i32(p.status) != 0)) return;
    // pieces that did not fit: the gated atomics pass ORs the voxels in (after a
    // fresh volume has been cleared here, brick by brick)
    const bool overflow = __ldg(p.brick_off + p.G.n_slots) > p.capacity;
    if (!kBatched && overflow && p.bricked) {  // no atomics fallback for this layout
        if (blockIdx.x == 0 && t == 0) set_status(p.status, kStPieces);
        return;
    }
    if (overflow && !p.fresh) return;
    const bool async_store = !kBatched && (p.use_tma || p.bricked);  // the bitmap leaves by the bulk-copy unit
    const int64_t total_bricks = p.G.n_bricks;
    using St = typename std::conditional<kEuclid, EuclidStepper<uint32_t, uint32_t>, Stepper<uint32_t, uint32_t>>::type;
    // a piece's slope table entry (in a wide volume the piece's segment is entered by division)
    auto load_slopes = [&](uint64_t piece, uint4 &a, uint2 &b) {
        const uint4 *e = reinterpret_cast<const uint4 *>(p.slopes + (piece & 0xffffffffull));
        a = __ldg(e);
        b = __ldg(reinterpret_cast<const uint2 *>(e + 1));
    };
    // this warp's first group of the brick in hand, when loaded ahead
    bool have_pref = false;
    uint64_t pc_pref = 0;
    uint4 sa_pref = make_uint4(0u, 0u, 0u, 0u);
    uint2 sb_pref = make_uint2(0u, 0u);
    // the quarter of the bitmap that this thread's 8 warps store and clear
    const int quarter = t / (kBrickThreads / kBrickQuarters);
    const bool leader = t % (kBrickThreads / kBrickQuarters) == 0;
    // ring positions of the brick in hand, the next one and the one after
    int cur = 0, nxt = 1, aft = 2;
    const bool taker = t == kBrickThreads - 32;  // lane 0 of the last warp takes the tickets
    if (taker) {
        sm.n_hot = overflow ? 0 : static_cast<int32_t>(__ldg(p.n_hot));
        sm.hot_limit = hot_pieces(__ldg(p.brick_off + p.G.n_slots));
        take_brick<kBatched>(p, overflow, sm, sm.info[0]);
        take_brick<kBatched>(p, overflow, sm, sm.info[1]);
    }
    while (true) {
        __syncthreads();
        const BrickInfo &I = sm.info[cur];
        const BrickInfo &NI = sm.info[nxt];
        const int64_t b = I.brick;
        if (b >= total_bricks) break;
        const BrickGeom &G = kBatched ? I.geom : p.G;
        const bool wide = kBatched ? G.wide != 0 : kWide;
        const int32_t X0 = I.origin[0], Y0 = I.origin[1], Z0 = I.origin[2];
        const uint32_t bw = static_cast<uint32_t>(G.B[0]);
        const uint32_t bwh = static_cast<uint32_t>(G.B[0]) * static_cast<uint32_t>(G.B[1]);
        // below 2^31: a brick beyond the limit of hot_pieces is walked in parts
        const uint64_t *const pieces = p.pieces + I.lo;
        const int32_t cnt = static_cast<int32_t>(I.hi - I.lo);
        const bool next_ok = NI.brick < total_bricks;
        const int32_t cnt_n = next_ok ? static_cast<int32_t>(NI.hi - NI.lo) : 0;
        if ((cnt == 0 && !p.fresh) || I.skip) {
            have_pref = false;
            if (taker) take_brick<kBatched>(p, overflow, sm, sm.info[aft]);  // read by no one now
            const int c = cur;
            cur = nxt;
            nxt = aft;
            aft = c;
            continue;
        }
        // the warp's first group (group `warp`): loaded ahead, or its pieces now
        // (their records after the clear, so that the latency overlaps it)
        int32_t grp = warp;
        int32_t j = t;
        uint64_t pc = have_pref ? pc_pref : (j < cnt ? __ldg(pieces + j) : 0ull);
        uint4 sa = sa_pref;
        uint2 sb = sb_pref;
        // the next brick's first group for this warp: its pieces now, consumed after the walk
        const uint64_t pc_n = t < cnt_n ? __ldg(p.pieces + NI.lo + t) : 0ull;
        if (t == 0) sm.next_group = kBrickThreads / 32;  // groups beyond the first round, on demand
        // each quarter is cleared as soon as its own copy has been read
        if (async_store) {
            if (leader) bulk_wait_read_all();
            asm volatile("bar.sync %0, %1;" ::"r"(quarter + 1), "n"(kBrickThreads / kBrickQuarters) : "memory");
        }
        {  // a quarter's words are a multiple of 4
            const int n4 = G.words / kBrickQuarters / 4;
            uint4 *z = reinterpret_cast<uint4 *>(sm.bits) + quarter * n4;
            for (int q = t % (kBrickThreads / kBrickQuarters); q < n4; q += kBrickThreads / kBrickQuarters)
                z[q] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (!have_pref && j < cnt && !wide) load_slopes(pc, sa, sb);
        __syncthreads();
        // the brick after the next one: its ticket is taken while the CTA walks this
        // one (its ring slot held the brick before this one, read by no one now)
        if (taker) take_brick<kBatched>(p, overflow, sm, sm.info[aft]);
        // brick-local bit index of (x, y, z): (x - X0) + B0 (y - Y0) + B0 B1 (z - Z0),
        // kept modulo 2^32 while stepping (only the local value is ever used)
        const uint32_t origin = static_cast<uint32_t>(X0) + static_cast<uint32_t>(Y0) * bw +
                                static_cast<uint32_t>(Z0) * bwh;
        // one shared-memory atomic per voxel: cheaper than branching to merge runs of the
        // same word (measured on both workload shapes); repeated samples of the Euclidean
        // variant set the same bit again
        auto put = [&](uint32_t L) { atomicOr(sm.bits + (L >> 5), 1u << (L & 31u)); };
#pragma unroll 1
        while (grp * 32 < cnt) {
            if (j < cnt) {
                const int32_t len = static_cast<int32_t>(pc >> 54) + 1;
                const int32_t k = static_cast<int32_t>((pc >> 32) & 0x3fffffull);
                if (wide) {
                    int32_t rec[6];
                    load_record(p.segs, static_cast<int64_t>(pc & 0xffffffffull), rec);
                    St st;
                    st.enter(rec, k, bw, bwh);
                    st.L -= origin;
                    for (int32_t e = 0; e < len; ++e) {
                        put(st.L);
                        st.template step<false, true>();
                    }
                } else {
                    // the voxel at step k, its fractions and the signed strides
                    uint32_t f[3], s[3], d[3];
                    const uint32_t v[3] = {sa.x & 0xffffu, sa.x >> 16, sa.y & 0xffffu}, lo[3] = {sa.w, sb.x, sb.y},
                                   st[3] = {1u, bw, bwh};
                    uint32_t L = 0u - origin;
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const uint32_t hi = (sa.z >> (8 * a)) & 0xffu;
                        const uint64_t P = static_cast<uint64_t>(static_cast<uint32_t>(k)) * lo[a] + (uint64_t(1) << 39) +
                                           (static_cast<uint64_t>(static_cast<uint32_t>(k) * hi) << 32);
                        const bool down = (sa.y & (0x10000u << a)) != 0u;
                        const uint32_t q = static_cast<uint32_t>(P >> 40);
                        L += (down ? v[a] - q : v[a] + q) * st[a];
                        d[a] = down ? 0u - st[a] : st[a];
                        f[a] = static_cast<uint32_t>(P >> 8) + 1u;
                        s[a] = (hi << 24) | (lo[a] >> 8);
                        s[a] += s[a] != 0xffffffffu && (lo[a] & 0xffu) != 0u ? 1u : 0u;
                    }
                    if constexpr (kEuclid) {
#pragma unroll 4
                        for (int32_t e = 0; e < len; ++e) {
                            put(L);
#pragma unroll
                            for (int a = 0; a < 3; ++a) L += add_carry(f[a], s[a]) * d[a];
                        }
                    } else {
                        // the major axis moves at every step
                        const uint32_t m = sa.y >> 19;
                        const uint32_t dm = m == 0 ? d[0] : (m == 1 ? d[1] : d[2]);
                        const uint32_t db = m == 0 ? d[1] : d[0], dc = m == 2 ? d[1] : d[2];
                        uint32_t fb = m == 0 ? f[1] : f[0], fc = m == 2 ? f[1] : f[2];
                        const uint32_t sb_ = m == 0 ? s[1] : s[0], sc = m == 2 ? s[1] : s[2];
                        int32_t e = 0;
                        for (; e + 8 <= len; e += 8) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                put(L);
                                const uint32_t cb = add_carry(fb, sb_), cc = add_carry(fc, sc);
                                L += dm + cb * db + cc * dc;
                            }
                        }
                        for (; e < len; ++e) {
                            put(L);
                            const uint32_t cb = add_carry(fb, sb_), cc = add_carry(fc, sc);
                            L += dm + cb * db + cc * dc;
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) grp = atomicAdd(&sm.next_group, 1);
            grp = __shfl_sync(0xffffffffu, grp, 0);
            j = grp * 32 + lane;
            if (j < cnt) {
                pc = __ldg(pieces + j);
                if (!wide) load_slopes(pc, sa, sb);
            }
        }
        // the next brick's first group: its pieces have arrived, now their slopes
        have_pref = next_ok;
        pc_pref = pc_n;
        if (t < cnt_n && !(kBatched ? NI.geom.wide != 0 : kWide)) load_slopes(pc_n, sa_pref, sb_pref);
        __syncthreads();
        if (async_store) {
            const int32_t part = G.words / kBrickQuarters;
            const int32_t z = Z0 + quarter * (G.B[2] / kBrickQuarters);
            if (leader) {
                fence_proxy_async_smem();  // the bitmap's generic writes, visible to the bulk-copy unit
                if (p.bricked) {
                    uint32_t *const dst = p.mask + b * G.words + quarter * part;
                    if (I.part) bulk_reduce_or_1d(dst, sm.bits + quarter * part, static_cast<uint32_t>(part) * 4u);
                    else bulk_store_1d(dst, sm.bits + quarter * part, static_cast<uint32_t>(part) * 4u);
                } else if (z >= G.dim[2]) {
                    // the quarter lies beyond the volume
                } else if (p.fresh && !I.part)
                    tma_store_3d(&tmap, sm.bits + quarter * part, X0 / 64, Y0, z);
                else
                    tma_reduce_or_3d(&tmap, sm.bits + quarter * part, X0 / 64, Y0, z);
            }
        } else {
            uint32_t *const mask = kBatched ? I.bmask : p.mask;
            if (mask != nullptr) {
                if (I.part) merge_part(sm.bits, G, X0, Y0, Z0, mask);
                else merge_brick(sm.bits, G, X0, Y0, Z0, mask, p.fresh != 0);
            }
            __syncthreads();
        }
        const int c = cur;
        cur = nxt;
        nxt = aft;
        aft = c;
    }
    if (async_store && leader) bulk_wait_all();  // copies complete before the CTA's memory goes
}

// Brick-major volume -> row-major volume: one warp per volume row (y, z), lanes
// over the row's words; each word comes from its brick's row (bxw contiguous
// words), so reads stay sector-sized and writes are coalesced.
__global__ void __launch_bounds__(256) k_unbrick(const uint32_t *bricked, BrickGeom G, uint32_t *mask)
{
    const int lane = threadIdx.x & 31;
    const int64_t rows = static_cast<int64_t>(G.dim[1]) * G.dim[2];
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5); r < rows; r += warps) {
        const int32_t y = static_cast<int32_t>(r % G.dim[1]);
        const int32_t z = static_cast<int32_t>(r / G.dim[1]);
        const int64_t bbase = static_cast<int64_t>(G.nb[0]) * ((y >> G.logB[1]) + static_cast<int64_t>(G.nb[1]) * (z >> G.logB[2]));
        const int64_t inrow = static_cast<int64_t>(G.bxw) * ((y & (G.B[1] - 1)) + static_cast<int64_t>(G.B[1]) * (z & (G.B[2] - 1)));
        uint32_t *out = mask + r * G.row_words;
        for (int32_t xw = lane; xw < G.row_words; xw += 32) {
            const int64_t brick = bbase + (xw >> G.log_bxw);
            out[xw] = __ldg(bricked + brick * G.words + inrow + (xw & (G.bxw - 1)));
        }
    }
}

// Brick-major -> row-major through the bulk-copy unit: each CTA (one warp, of
// which thread 0 works) takes quarter bricks in a grid-stride order; a quarter brick
// is contiguous in the brick-major layout (z is the slowest axis inside a
// brick), so it arrives in shared memory with one 1-D bulk copy and leaves with
// one TMA tensor store of a quarter-brick box. Several CTAs per SM keep loads and
// stores in flight together. Bound by HBM (read and written once): 2048^3 362 us, 0.89
// of the copy peak; half bricks, three CTAs per SM, one brick after another 473 us;
// eighths 374 us; quarters brick after brick 395 us (the stores are 32 bytes a row).
// Every wait is bounded; on expiry the status (if any) records a timeout and the CTA
// stops after one more bounded wait for its copy in flight.
constexpr int kUnbrickSplit = 4;

__global__ void __launch_bounds__(32) k_unbrick_tma(const uint32_t *bricked, BrickGeom G,
                                                    const __grid_constant__ CUtensorMap tmap, int32_t *status,
                                                    uint64_t wait_ns)
{
    extern __shared__ __align__(128) unsigned char unbrick_smem_raw[];
    uint32_t *buf = reinterpret_cast<uint32_t *>(unbrick_smem_raw);
    __shared__ uint64_t bar;
    if (threadIdx.x != 0) return;
    const int32_t part_words = G.words / kUnbrickSplit;
    const int32_t part_rows = G.B[2] / kUnbrickSplit;
    mbar_init(&bar, 1);
    fence_barrier_init();
    uint32_t phase = 0;
    const int64_t n_parts = G.n_bricks * kUnbrickSplit;
    for (int64_t q = blockIdx.x; q < n_parts; q += gridDim.x) {
        // the bricks of a row of bricks side by side: their copies fill whole volume rows
        const int64_t qr = q / G.nb[0];
        const int32_t bx = static_cast<int32_t>(q - qr * G.nb[0]);
        const int64_t rest = qr / kUnbrickSplit;
        const int32_t h = static_cast<int32_t>(qr - rest * kUnbrickSplit);
        const int64_t b = rest * G.nb[0] + bx;
        const int32_t X0 = bx * G.B[0];
        const int32_t Y0 = static_cast<int32_t>(rest % G.nb[1]) * G.B[1];
        const int32_t Z0 = static_cast<int32_t>(rest / G.nb[1]) * G.B[2];
        bulk_wait_read_all();  // the previous store has read the buffer
        mbar_arrive_expect_tx(&bar, static_cast<uint32_t>(part_words) * 4u);
        bulk_copy_g2s(buf, bricked + b * G.words + static_cast<int64_t>(h) * part_words,
                      static_cast<uint32_t>(part_words) * 4u, &bar);
        if (!mbar_wait_bounded(&bar, phase, wait_ns)) {
            if (status != nullptr) set_status(status, 5);  // VOX_ERR_TIMEOUT
            mbar_wait_bounded(&bar, phase, wait_ns);
            break;
        }
        phase ^= 1u;
        tma_store_3d(&tmap, buf, X0 / 64, Y0, Z0 + h * part_rows);
    }
    bulk_wait_all();
}

}  // namespace vox

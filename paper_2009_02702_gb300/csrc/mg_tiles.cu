// mg_tiles.cu -- exact segment counts of plane tiles, for the box queries.
//
// Most cubes of a box's footprint lie in slabs one cube thick: blocks whose
// smallest run level l is met on one axis only, the other two being long (of
// the 100,000-box batch on 2048x2048x300, 66 % of all cubes are level-0 cubes
// of blocks at least 16 x 16 x 1).  A plane tile of level l and edge 2^T is
// the group of 2^T x 2^T x 1 aligned cubes of level l, a line tile one of
// 16 x 1 x 1; a record holds the level-0 voxels of every segment in its tile,
// so a slab is counted by one 16-byte record per 64 or 256 cubes instead of an
// ID per cube.  Every cube of a footprint is interior, hence its mixture is
// the exact count of its voxels and a record is the exact sum over its cubes,
// the integers that the cubes' own pushes deliver.
//
// Plane tiles are kept for the levels 0-3 with edge 8 and 0-2 with edge 16,
// for each of the three thickness axes in the axis order of the copy whose
// slowest axis it is (copy 0: tiles of (x, y), copy 1: (y, z), copy 2:
// (z, x)): counts stay below 2^16 up to those levels, and higher levels hold
// under 0.2 % of the cubes.  Line tiles, along the fastest axis of each copy,
// take the narrow blocks (two extents under 8) of the levels 1-3, whose cubes
// are mixtures that cost a table row each; at level 0 a cube is a segment, 16
// of which are read as 32 bytes anyway.
//
// Record (uint4): up to four words segment | count << 16, unused ones zero;
// a tile of more than four segments holds {0xFFFF, first, n, 0}: n uint4
// blocks of such words at `first` in the pool.
//
// Edge-8 tiles of level 0 and lines of level 1 are counted from the IDs: a
// thread holds its tile in registers and takes its segments in ascending order,
// one pass over the tile each that counts the IDs equal to this segment and
// finds the least ID above it (three instructions a word of two IDs and the
// sum), so that a warp's 32 tiles advance together whatever they hold.  Tiles
// of more than kOwnSegments segments are left to the warp, which counts one at
// a time in a table in shared memory.  Edge-8 tiles / lines, us: 512x512x384
// cells 118 / 125, 614x961x600 fibres 1,062 / 903, 255x256x257 bricks of five to
// eight segments a tile 49 / 79 (125 / 163, 3,101 / 3,403 and 264 / 843 with the
// warp counting all tiles of more than two segments, by reductions).
//
// An edge-16 tile is the sum of four edge-8 ones, an edge-8 tile of level l + 1
// the sum of two edge-16 ones of level l, and a line of level l + 1 the sum of
// eight lines: a thread collects its children's words, the warp those of tiles
// with more than kOwnWords (the fibres, all merges: 3,360 -> 1,780 us; 12, 16
// and 24 words 2,201 / 1,834 / 1,767), or of every list where there are few tiles.
//
// A stage whose lists find no room in the pool ends there, and those made from
// it at once: they are not used.
#include "mg_internal.cuh"

#include <algorithm>
#include <vector>

namespace mg {
namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kReserve = 32;       // pool blocks a warp reserves at a time
constexpr uint32_t kOwnSegments = 16;   // segments that a thread counts by itself
constexpr uint32_t kOwnWords = 24;      // distinct words that a thread collects by itself
constexpr uint32_t kMaxMerge = 256;     // words merged into distinct segments; longer lists are joined as they are
constexpr uint32_t kSegMask = 0xFFFFu;

struct Counters {
    unsigned long long used;            // pool blocks handed out (and asked for past the end)
    unsigned failed[kTileStages];       // a list of the stage did not fit the pool
};

// a warp's part of the pool: [cur, end), refilled by one atomic per kReserve blocks
struct PoolCursor {
    uint4* pool;
    unsigned long long cap, cur, end;
    Counters* cnt;
    int stage;
    bool full;   // no room for a list: the stage is not used, its warps leave
    __device__ __forceinline__ PoolCursor(uint4* p, unsigned long long c, Counters* n, int st)
        : pool(p), cap(c), cur(0), end(0), cnt(n), stage(st), full(false) {}
    // `need` blocks (same value in every lane), or ~0 when the pool is full
    __device__ __forceinline__ unsigned long long take(uint32_t need) {
        if (full) return ~0ull;
        if (cur + need > end) {
            const uint32_t r = max(need, kReserve);
            unsigned long long b = 0;
            if ((threadIdx.x & 31) == 0) b = atomicAdd(&cnt->used, (unsigned long long)r);
            b = __shfl_sync(0xffffffffu, b, 0);
            if (b + r > cap) {
                if ((threadIdx.x & 31) == 0) cnt->failed[stage] = 1u;
                full = true;
                return ~0ull;
            }
            cur = b;
            end = b + r;
        }
        const unsigned long long at = cur;
        cur += need;
        return at;
    }
};

// A warp's table of segments: words segment | count << 16 at the segment's hash
// or the next free place, zero where there is none and between tiles.  It holds
// at most half of its 2^lg places.
struct Table {
    uint32_t* at;
    int lg;
    __device__ __forceinline__ void add(uint32_t w) const {
        const uint32_t mask = (1u << lg) - 1u, s = w & kSegMask;
        for (uint32_t h = (s * 0x9E3779B1u) >> (32 - lg);; h = (h + 1) & mask) {
            const uint32_t old = atomicCAS(at + h, 0u, w);
            if (old == 0u) return;
            if ((old & kSegMask) == s) {
                atomicAdd(at + h, w & ~kSegMask);
                return;
            }
        }
    }
    // its words into buf (warp); returns their number
    __device__ __forceinline__ uint32_t take(uint32_t* buf) const {
        const int lane = threadIdx.x & 31;
        uint32_t n = 0;
        __syncwarp();
        for (uint32_t h = lane; h < 1u << lg; h += 32) {
            const uint32_t w = at[h];
            const unsigned m = __ballot_sync(0xffffffffu, w != 0u);
            if (w) {
                buf[n + __popc(m & ((1u << lane) - 1u))] = w;
                at[h] = 0u;
            }
            n += __popc(m);
        }
        return n;
    }
};

// the record of a tile whose n words are in buf (warp)
__device__ __forceinline__ uint4 finish(PoolCursor& P, const uint32_t* buf, uint32_t n) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    uint4 rec = make_uint4(0u, 0u, 0u, 0u);
    if (n <= 4) {
        rec = make_uint4(buf[0], n > 1 ? buf[1] : 0u, n > 2 ? buf[2] : 0u, n > 3 ? buf[3] : 0u);
    } else {
        const uint32_t need = (n + 3) / 4;
        const unsigned long long at = P.take(need);
        if (at != ~0ull) {
            uint32_t* out = reinterpret_cast<uint32_t*>(P.pool + at);
            for (uint32_t i = lane; i < 4 * need; i += 32) out[i] = i < n ? buf[i] : 0u;
            rec = make_uint4(kTileList, (uint32_t)at, need, 0u);
        }
    }
    __syncwarp();
    return rec;
}

// The records of the warp's tiles, each with n words at w (shared memory,
// kThreads apart): lists of more than four go to the pool, with one atomic for
// the warp.  n = 0: none (the warp path's).
__device__ __forceinline__ uint4 emit(PoolCursor& P, const uint32_t* w, uint32_t n) {
    const int lane = threadIdx.x & 31;
    const uint32_t need = n > 4 ? (n + 3) / 4 : 0u;
    uint4 rec = make_uint4(n > 0 ? w[0] : 0u, n > 1 ? w[kThreads] : 0u, n > 2 ? w[2 * kThreads] : 0u,
                           n > 3 ? w[3 * kThreads] : 0u);
    if (__any_sync(0xffffffffu, need != 0u)) {
        uint32_t incl = need;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&P.cnt->used, (unsigned long long)total);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base + total > P.cap) {
            if (lane == 0) P.cnt->failed[P.stage] = 1u;
            P.full = true;
        } else if (need) {
            const uint32_t first = (uint32_t)base + incl - need;
            for (uint32_t k = 0; k < n; k += 4)
                P.pool[first + k / 4] = make_uint4(w[k * kThreads], k + 1 < n ? w[(k + 1) * kThreads] : 0u,
                                                   k + 2 < n ? w[(k + 2) * kThreads] : 0u,
                                                   k + 3 < n ? w[(k + 3) * kThreads] : 0u);
            rec = make_uint4(kTileList, first, need, 0u);
        }
    }
    return rec;
}

// the level-0 IDs of each copy and the records counted from them
struct Level0 {
    const uint16_t* ids[3];
    uint4* out[3];
    int64_t st2[3];             // IDs between slabs
    uint32_t st1[3];            // IDs between rows
    uint32_t na[3], nb[3];      // tiles along the copy's first and second axis
    uint32_t tiles[3];
    int vec[3];                 // rows start on 16-byte boundaries
};

// LINE = false: edge-8 tiles, 8 rows of 8 IDs.  LINE = true: lines of level 1,
// 4 rows (2 x 2 in the second and third axis) of 32 IDs.
template <bool LINE>
__global__ void __launch_bounds__(kThreads) tile_ids_kernel(const __grid_constant__ Level0 A, uint4* pool,
                                                            unsigned long long cap, Counters* cnt, int stage,
                                                            uint32_t per) {
    constexpr int ROWS = LINE ? 4 : 8, VECS = LINE ? 4 : 1;   // rows of a tile, 16-byte vectors of a row
    constexpr int PER = LINE ? 4 : 2;                         // IDs per lane of a warp's tile
    constexpr uint32_t VOX = ROWS * VECS * 8;
    constexpr int LG = LINE ? 8 : 7;                          // places of the warp's table: twice the IDs
    static_assert(2 * VOX == 1u << LG, "a table is at most half full");
    constexpr int WORDS = VOX / 2;
    if (cnt->used >= cap) {   // no list has room
        if (threadIdx.x == 0) cnt->failed[stage] = 1u;
        return;
    }
    __shared__ uint32_t s_buf[kWarps][VOX], s_tab[kWarps][1 << LG], s_own[kOwnSegments * kThreads];
    uint32_t* own = s_own + threadIdx.x;
    const int c = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tiles = A.tiles[c], na = A.na[c], nb = A.nb[c], st1 = A.st1[c];
    const int64_t st2 = A.st2[c];
    auto row = [&](int k) -> int64_t {
        return LINE ? (int64_t)(k >> 1) * st2 + (int64_t)(k & 1) * st1 : (int64_t)k * st1;
    };
    PoolCursor P(pool, cap, cnt, stage);
    const Table table{s_tab[warp], LG};
    for (int h = lane; h < 1 << LG; h += 32) s_tab[warp][h] = 0u;
    __syncwarp();
    const uint32_t step = gridDim.x * kWarps * per;
    for (uint32_t i0 = (blockIdx.x * kWarps + warp) * per; i0 < tiles && !P.full; i0 += step) {
        const uint32_t i = (uint32_t)lane < per ? i0 + lane : tiles;
        const uint16_t* p = A.ids[c];
        uint32_t x[WORDS];
        if (i < tiles) {
            const uint32_t a = i % na, r = i / na, b = r % nb, t = r / nb;
            p += LINE ? (int64_t)(2 * t) * st2 + (int64_t)(2 * b) * st1 + 32 * a
                      : (int64_t)t * st2 + (int64_t)(8 * b) * st1 + 8 * a;
            if (A.vec[c]) {
#pragma unroll
                for (int k = 0; k < ROWS; k++)
#pragma unroll
                    for (int v = 0; v < VECS; v++) {
                        const uint4 u = __ldg(reinterpret_cast<const uint4*>(p + row(k)) + v);
                        const int e = 4 * (k * VECS + v);
                        x[e] = u.x;
                        x[e + 1] = u.y;
                        x[e + 2] = u.z;
                        x[e + 3] = u.w;
                    }
            } else {
#pragma unroll
                for (int k = 0; k < ROWS; k++)
#pragma unroll
                    for (int v = 0; v < 4 * VECS; v++)
                        x[4 * k * VECS + v] = (uint32_t)__ldg(p + row(k) + 2 * v) |
                                              (uint32_t)__ldg(p + row(k) + 2 * v + 1) << 16;
            }
        } else {
#pragma unroll
            for (int e = 0; e < WORDS; e++) x[e] = 0u;
        }
        // the least ID, then the segments in ascending order
        uint32_t m2 = x[0], cur = 0, n = 0;
#pragma unroll
        for (int e = 1; e < WORDS; e++) m2 = __vminu2(m2, x[e]);
        cur = min(m2 & kSegMask, m2 >> 16);
        bool more = true;
        while (more && n < kOwnSegments) {
            const uint32_t pat = cur * 0x10001u, below = ((0xFFFFu - cur) & kSegMask) * 0x10001u;
            uint32_t other = 0, above = 0xFFFFFFFFu;
#pragma unroll
            for (int e = 0; e < WORDS; e++) {
                other += __vminu2(x[e] ^ pat, 0x10001u);                // 1 per ID that is not cur
                above = __viaddmin_u16x2(x[e], below, above);           // ID - cur - 1 modulo 2^16
            }
            own[n * kThreads] = cur | (VOX - (other & kSegMask) - (other >> 16)) << 16;
            n++;
            const uint32_t next = min(above & kSegMask, above >> 16) + cur + 1u;   // past 2^16: none above cur
            more = next <= kSegMask;
            cur = next;
        }
        const uint32_t d = more ? 1u : 0u;   // the warp counts it
        uint4 rec = emit(P, own, more || i >= tiles ? 0u : n);
        if (P.full) break;
        for (unsigned m = __ballot_sync(0xffffffffu, d != 0); m && !P.full; m &= m - 1) {
            const int j = __ffs(m) - 1;
            const uint16_t* q = reinterpret_cast<const uint16_t*>(
                __shfl_sync(0xffffffffu, (unsigned long long)reinterpret_cast<uintptr_t>(p), j));
            const int at = lane * PER;   // this lane's IDs: PER consecutive ones of a row
            q += row(at / (8 * VECS)) + at % (8 * VECS);
            uint32_t v[PER];
            if (A.vec[c]) {
#pragma unroll
                for (int e = 0; e < PER; e += 2) {
                    const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(q) + e / 2);
                    v[e] = w & kSegMask;
                    v[e + 1] = w >> 16;
                }
            } else {
#pragma unroll
                for (int e = 0; e < PER; e++) v[e] = (uint32_t)__ldg(q + e);
            }
            uint32_t run = v[0] | 1u << 16;
#pragma unroll
            for (int e = 1; e < PER; e++) {
                if (v[e] == (run & kSegMask)) {
                    run += 1u << 16;
                } else {
                    table.add(run);
                    run = v[e] | 1u << 16;
                }
            }
            table.add(run);
            const uint4 lr = finish(P, s_buf[warp], table.take(s_buf[warp]));
            if (lane == j) rec = lr;
        }
        if (i < tiles) A.out[c][i] = rec;
    }
}

// tiles from the records of CH smaller ones: four edge-8 tiles (2 x 2 in the
// plane) of one level, two edge-16 tiles (adjacent slabs) of the level below,
// or eight lines (2 along the line, 2 x 2 across) of the level below
struct Merge {
    const uint4* in[3];
    uint4* out[3];
    uint32_t in1[3], in2[3];    // strides of the input records
    uint32_t na[3], nb[3], tiles[3];
};

template <int CH>
__global__ void __launch_bounds__(kThreads) tile_merge_kernel(const __grid_constant__ Merge A, uint4* pool,
                                                              unsigned long long cap, Counters* cnt, int stage,
                                                              int from, uint32_t per) {
    if (cnt->failed[from] || cnt->used >= cap) {   // the records read here are not all there, or no list has room
        if (threadIdx.x == 0) cnt->failed[stage] = 1u;
        return;
    }
    __shared__ uint32_t s_buf[kWarps][kMaxMerge], s_tab[kWarps][2 * kMaxMerge], s_own[kOwnWords * kThreads];
    uint32_t* own = s_own + threadIdx.x;
    const int c = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t tiles = A.tiles[c], na = A.na[c], nb = A.nb[c];
    PoolCursor P(pool, cap, cnt, stage);
    for (uint32_t h = lane; h < 2 * kMaxMerge; h += 32) s_tab[warp][h] = 0u;
    __syncwarp();
    const uint32_t step = gridDim.x * kWarps * per;
    for (uint32_t i0 = (blockIdx.x * kWarps + warp) * per; i0 < tiles && !P.full; i0 += step) {
        const uint32_t i = (uint32_t)lane < per ? i0 + lane : tiles;
        uint4 in[CH];
        // (where a warp has few tiles, its lanes are better spent on one each time)
        const uint32_t most = per == 32 ? kOwnWords : 4u;
        uint32_t n = 0, total = 0;
        bool over = false;
#pragma unroll
        for (int k = 0; k < CH; k++) in[k] = make_uint4(0u, 0u, 0u, 0u);
        if (i < tiles) {
            const uint32_t a = i % na, r = i / na, b = r % nb, t = r / nb;
#pragma unroll
            for (int k = 0; k < CH; k++) {
                const uint32_t ka = CH == 2 ? a : 2 * a + (k & 1), kb = CH == 2 ? b : 2 * b + ((k >> 1) & 1);
                const uint32_t kt = CH == 2 ? 2 * t + k : CH == 8 ? 2 * t + (k >> 2) : t;
                const size_t at = (size_t)kt * A.in2[c] + (size_t)kb * A.in1[c] + ka;
                in[k] = __ldg(A.in[c] + at);
            }
#pragma unroll
            for (int k = 0; k < CH; k++) total += in[k].x == kTileList ? 4u * in[k].z : 4u;
            over = total > 4 * most;
        }
        auto collect = [&](uint32_t w) {
            if (!(w >> 16)) return;
            uint32_t q = 0;
            while (q < n && ((own[q * kThreads] ^ w) & kSegMask)) q++;
            if (q < n) {
                own[q * kThreads] += w & ~kSegMask;
            } else if (n < most) {
                own[n * kThreads] = w;
                n++;
            } else {
                over = true;
            }
        };
#pragma unroll
        for (int k = 0; k < CH; k++) {
            const bool list = in[k].x == kTileList;
            const uint32_t blocks = over ? 0u : list ? in[k].z : 1u;
            for (uint32_t q = 0; q < blocks && !over; q++) {
                const uint4 w = list ? pool[in[k].y + q] : in[k];
                collect(w.x);
                collect(w.y);
                collect(w.z);
                collect(w.w);
            }
        }
        uint4 rec = emit(P, own, over ? 0u : n);
        if (P.full) break;
        for (unsigned m = __ballot_sync(0xffffffffu, over); m && !P.full; m &= m - 1) {
            const int j = __ffs(m) - 1;
            // the children's words as one sequence: four of an inline record, the pool's of a list
            uint4 ch[CH];
            uint32_t end[CH];
            total = 0;
#pragma unroll
            for (int k = 0; k < CH; k++) {
                ch[k] = make_uint4(__shfl_sync(0xffffffffu, in[k].x, j), __shfl_sync(0xffffffffu, in[k].y, j),
                                   __shfl_sync(0xffffffffu, in[k].z, j), __shfl_sync(0xffffffffu, in[k].w, j));
                total += ch[k].x == kTileList ? 4u * ch[k].z : 4u;
                end[k] = total;
            }
            auto word = [&](uint32_t s) -> uint32_t {
                uint32_t first = 0, v = 0;
#pragma unroll
                for (int k = 0; k < CH; k++) {
                    if (s >= first && s < end[k]) {
                        const uint32_t e = s - first;
                        if (ch[k].x == kTileList) v = reinterpret_cast<const uint32_t*>(pool + ch[k].y)[e];
                        else v = e == 0 ? ch[k].x : e == 1 ? ch[k].y : e == 2 ? ch[k].z : ch[k].w;
                    }
                    first = end[k];
                }
                return v;
            };
            uint4 lr;
            if (total <= kMaxMerge) {
                const Table table{s_tab[warp], max(5, 32 - __clz(2 * total - 1))};
                for (uint32_t e = lane; e < total; e += 32) {
                    const uint32_t w = word(e);
                    if (w >> 16) table.add(w);
                }
                lr = finish(P, s_buf[warp], table.take(s_buf[warp]));
            } else {
                // long lists are joined: a segment may appear twice, its counts still add up
                const unsigned long long at = P.take(total / 4);
                lr = make_uint4(0u, 0u, 0u, 0u);
                if (at != ~0ull) {
                    uint32_t* out = reinterpret_cast<uint32_t*>(pool + at);
                    for (uint32_t s = lane; s < total; s += 32) out[s] = word(s);
                    lr = make_uint4(kTileList, (uint32_t)at, total / 4, 0u);
                }
            }
            if (lane == j) rec = lr;
        }
        if (i < tiles) A.out[c][i] = rec;
    }
}

// Record of every node in the mixture table, for the cubes that no tile
// covers: up to four segments inline, so that a cube costs one gather instead
// of the row header and then its entries; longer rows {0xFFFF, first entry,
// entries, 3 lmin} in the table; zero for nodes without a row.  Rows average
// two entries; lmin <= 5 for an inline record, whose counts have 16 bits.  Rows
// past the table's `entries` (a damaged image) are not read.
__global__ void node_records_kernel(const uint2* __restrict__ meta, const uint2* __restrict__ lut, int64_t entries,
                                    int64_t N, uint4* __restrict__ rec) {
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
        const uint2 m = meta[n];
        const uint32_t lmin = m.y & 255u, len = m.x + (int64_t)(m.y >> 8) <= entries ? m.y >> 8 : 0u;
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (len > 4 || (len && lmin > 5)) {
            r = make_uint4(kTileList, m.x, len, 3 * lmin);
        } else if (len) {
            uint32_t w[4];
#pragma unroll
            for (uint32_t e = 0; e < 4; e++) {
                w[e] = 0;
                if (e < len) {
                    const uint2 t = __ldg(lut + m.x + e);
                    w[e] = t.x | t.y << 16;
                }
            }
            r = make_uint4(w[0], w[1], w[2], w[3]);
        }
        rec[n] = r;
    }
}

// The shares of a node's weight that its sources receive when the weight is
// pushed through the lerp tree with 16-bit alphas and fp32 arithmetic, one per
// entry of the node's table row (whose sources are in the same depth-first
// order, p before q).  Pushing 8^l scales every step by a power of two, so
// 8^l times a share is what that push delivers, bit for bit; only the walk is
// saved.  Two-source rows, the most frequent, are whole in the record.
template <typename AT>
__global__ void node_shares_kernel(const uint2* __restrict__ pq, const AT* __restrict__ alpha,
                                   const uint2* __restrict__ meta, int64_t entries, int64_t N, uint32_t S,
                                   float* __restrict__ frac,
                                   uint4* __restrict__ rec) {
    constexpr int kStack = 64;
    for (int64_t n0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n0 < N; n0 += (int64_t)gridDim.x * blockDim.x) {
        const uint2 m = meta[n0];
        const uint32_t len = m.x + (int64_t)(m.y >> 8) <= entries ? m.y >> 8 : 0u;
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (len) {
            uint32_t sn[kStack];
            float sw[kStack];
            int sp = 0;
            uint32_t n = (uint32_t)n0, k = 0;
            float w = 1.f;
            for (;;) {
                if (n < S) {
                    if (k < len) frac[m.x + k] = w;
                    if (k == 0) {
                        r.x = n;
                        r.y = __float_as_uint(w);
                    } else if (k == 1) {
                        r.x |= n << 16;
                        r.z = __float_as_uint(w);
                    }
                    k++;
                    if (sp == 0) break;
                    --sp;
                    n = sn[sp];
                    w = sw[sp];
                    continue;
                }
                const uint2 e = __ldg(pq + n);
                const float al = (float)alpha[n];
                // the weight of q, or of p when the sign says they are swapped
                const float wb = w * fabsf(al), wa = w - wb;
                if (sp >= kStack || k > len) break;   // (a valid row has len leaves and a shallow tree)
                sn[sp] = e.y;
                sw[sp] = al < 0.f ? wa : wb;
                sp++;
                n = e.x;
                w = al < 0.f ? wb : wa;
            }
            if (k != len) r = make_uint4(0u, 0u, 0u, 0u);   // walked by the query
            else if (len == 2) r.w = kFracPair;
            else r = make_uint4(m.x, len, 0u, kFracList);
        }
        rec[n0] = r;
    }
}

// memory that the queries can do without: null when there is none
bool try_alloc(Buf& b, const Alloc* al, size_t n, cudaStream_t s) {
    b.release();
    void* p = al->get(n, s);
    if (!p) return false;
    if (reinterpret_cast<uintptr_t>(p) % 256) {
        al->put(p, n, s);
        return false;
    }
    b.al = al;
    b.s = s;
    b.p = p;
    b.bytes = n;
    return true;
}

}  // namespace

mg_status build_tiles(mg_graph* g, cudaStream_t s) {
    TileGeom& T = g->tgeom;
    T = TileGeom{};
    if (g->id0_bytes != 2 || g->S > kMaxSharedSegments) return MG_OK;   // no box queries on such graphs
    if (g->lut_meta.p && !g->quantised && try_alloc(g->lut_rec, &g->al, (size_t)g->N * sizeof(uint4), s)) {
        node_records_kernel<<<grid_for(g->N, 256, 152 * 32), 256, 0, s>>>(g->lut_meta.as<uint2>(), g->lut.as<uint2>(),
                                                                         g->lut_entries, g->N, g->lut_rec.as<uint4>());
        MG_CUDA(cudaGetLastError());
    }
    // levels >= 1 replace pushes through exact nodes with table rows
    const int levels = std::min(g->L, g->quantised || !g->lut_meta.p ? 1 : kTileLevels);
    struct Stage {
        int kind, l;            // kind 0 / 1: edge-8 / edge-16 tiles of level l; 2: lines
        int from_kind, from_l;  // the records it sums (from_l < 0: the IDs)
        int64_t dim[3][3], count[3], all;
    };
    std::vector<Stage> stages;
    for (int l = 0; l < levels; l++) {
        stages.push_back(Stage{0, l, 1, l - 1, {}, {}, 0});
        if (l < kTileLevels - 1) stages.push_back(Stage{1, l, 0, l, {}, {}, 0});
    }
    for (int l = 1; l < levels; l++) stages.push_back(Stage{2, l, 2, l == 1 ? -1 : l - 1, {}, {}, 0});
    int64_t total = 0;
    for (Stage& st : stages)
        for (int c = 0; c < 3; c++) {
            const int l = st.l, e = st.kind == 0 ? 3 : 4;
            for (int k = 0; k < 3; k++) st.dim[c][k] = g->geom.dims[0][(c + k) % 3] >> l;
            st.dim[c][0] >>= e;
            if (st.kind < 2) st.dim[c][1] >>= e;
            st.count[c] = st.dim[c][0] * st.dim[c][1] * st.dim[c][2];
            st.all += st.count[c];
            T.off[l][st.kind][c] = total;
            T.st1[l][st.kind][c] = (uint32_t)st.dim[c][0];
            T.st2[l][st.kind][c] = (uint32_t)(st.dim[c][0] * st.dim[c][1]);
            total += st.count[c];
        }
    if (total == 0) return MG_OK;
    const int64_t V = (int64_t)g->geom.dims[0][0] * g->geom.dims[0][1] * g->geom.dims[0][2];
    // room for lists of 2 bytes per voxel (noise would need 12 and gets no
    // tiles); the part that is used is kept
    const unsigned long long cap = (unsigned long long)std::max<int64_t>(V / 8, 1 << 16);
    Buf pool;   // the blocks, then the counters
    if (!try_alloc(g->tiles, &g->al, (size_t)total * sizeof(uint4), s) ||
        !try_alloc(pool, &g->al, (size_t)cap * sizeof(uint4) + sizeof(Counters), s)) {
        g->tiles.release();
        return MG_OK;
    }
    Counters* cnt = reinterpret_cast<Counters*>(pool.as<uint4>() + cap);
    MG_CUDA(cudaMemsetAsync(cnt, 0, sizeof(Counters), s));
    uint4* rec = g->tiles.as<uint4>();
    for (size_t k = 0; k < stages.size(); k++) {
        const Stage& st = stages[k];
        if (st.all == 0) continue;
        const int l = st.l;
        // a warp's tiles that need it whole are taken in turn, so few tiles are
        // spread over more warps (a small volume's stage: 50 -> 5 us)
        const int64_t most = std::max(st.count[0], std::max(st.count[1], st.count[2]));
        uint32_t per = 32;
        while (per > 1 && most / per < 152 * 8) per /= 2;
        const dim3 grid(grid_for(most, (int)per * kWarps, 152 * 8), 3);
        if (st.from_l < 0) {
            Level0 A{};
            for (int c = 0; c < 3; c++) {
                A.ids[c] = (g->mip0x[c].p ? g->mip0x[c] : g->mip0).as<uint16_t>();
                A.out[c] = rec + T.off[l][st.kind][c];
                A.st1[c] = (uint32_t)g->qpitch[0][c];
                A.st2[c] = (int64_t)g->qpitch[0][c] * g->geom.dims[0][(c + 1) % 3];
                A.na[c] = (uint32_t)st.dim[c][0];
                A.nb[c] = (uint32_t)st.dim[c][1];
                A.tiles[c] = (uint32_t)st.count[c];
                A.vec[c] = A.st1[c] % 8 == 0;
            }
            if (st.kind == 2) tile_ids_kernel<true><<<grid, kThreads, 0, s>>>(A, pool.as<uint4>(), cap, cnt, (int)k, per);
            else tile_ids_kernel<false><<<grid, kThreads, 0, s>>>(A, pool.as<uint4>(), cap, cnt, (int)k, per);
        } else {
            Merge A{};
            for (int c = 0; c < 3; c++) {
                A.in[c] = rec + T.off[st.from_l][st.from_kind][c];
                A.in1[c] = T.st1[st.from_l][st.from_kind][c];
                A.in2[c] = T.st2[st.from_l][st.from_kind][c];
                A.out[c] = rec + T.off[l][st.kind][c];
                A.na[c] = (uint32_t)st.dim[c][0];
                A.nb[c] = (uint32_t)st.dim[c][1];
                A.tiles[c] = (uint32_t)st.count[c];
            }
            auto kernel = st.kind == 0 ? tile_merge_kernel<2> : st.kind == 1 ? tile_merge_kernel<4> : tile_merge_kernel<8>;
            int from = 0;
            while (stages[from].kind != st.from_kind || stages[from].l != st.from_l) from++;
            kernel<<<grid, kThreads, 0, s>>>(A, pool.as<uint4>(), cap, cnt, (int)k, from, per);
        }
        MG_CUDA(cudaGetLastError());
    }
    Counters h;
    MG_CUDA(cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    // a stage whose lists did not fit, and those made from it, are not used
    // (nor read: their records are not all written)
    bool ok[kTileLevels][3] = {};
    for (size_t k = 0; k < stages.size(); k++) {
        const Stage& st = stages[k];
        ok[st.l][st.kind] = !h.failed[k] && (st.from_l < 0 || ok[st.from_l][st.from_kind]);
        if (!ok[st.l][st.kind]) continue;
        if (st.kind < 2) T.edge[st.l] = 3 + st.kind;
        else T.line[st.l] = 1;
    }
    if (T.edge[0] == 0 && T.line[1] == 0) {
        g->tiles.release();
        return MG_OK;
    }
    const size_t kept = (size_t)std::min(h.used, cap) * sizeof(uint4);
    if (kept == 0) return MG_OK;
    // (a megabyte is not worth another allocation and copy: importing 64^3 takes 0.2 ms)
    if (kept < pool.bytes / 4 * 3 && pool.bytes - kept > (1u << 20) && try_alloc(g->tile_pool, &g->al, kept, s))
        MG_CUDA(cudaMemcpyAsync(g->tile_pool.p, pool.p, kept, cudaMemcpyDeviceToDevice, s));
    else
        g->tile_pool = std::move(pool);
    return MG_OK;
}

int64_t spare_tile_bytes(mg_graph* g) {
    std::lock_guard<std::mutex> lk(g->tiles_mu);
    return g->tiles_held ? 0 : (int64_t)(g->tiles.bytes + g->tile_pool.bytes + g->lut_rec.bytes);
}

bool drop_tiles(mg_graph* g) {
    std::lock_guard<std::mutex> lk(g->tiles_mu);
    if (g->tiles_held) return false;
    g->tgeom = TileGeom{};
    g->tiles.release();
    g->tile_pool.release();
    g->lut_rec.release();
    return true;
}

mg_status ensure_records16(mg_graph* g, mg_dtype dt, cudaStream_t s) {
    if (!g->lut_meta.p || g->quantised || g->S > kMaxSharedSegments) return MG_OK;
    const int k = dt == MG_BF16;
    std::lock_guard<std::mutex> lk(g->rec16_mu);
    if (g->rec16[k].p || is_capturing(s)) return MG_OK;
    Buf frac, rec;
    if (!try_alloc(frac, &g->al, (size_t)std::max<int64_t>(g->lut_entries, 1) * 4, s) ||
        !try_alloc(rec, &g->al, (size_t)g->N * sizeof(uint4), s))
        return MG_OK;
    const unsigned gb = grid_for(g->N, 256, 152 * 32);
    if (k)
        node_shares_kernel<<<gb, 256, 0, s>>>(g->pq.as<uint2>(), g->alphab16.as<__nv_bfloat16>(), g->lut_meta.as<uint2>(),
                                              g->lut_entries, g->N, g->S, frac.as<float>(), rec.as<uint4>());
    else
        node_shares_kernel<<<gb, 256, 0, s>>>(g->pq.as<uint2>(), g->alpha16.as<__half>(), g->lut_meta.as<uint2>(),
                                              g->lut_entries, g->N, g->S, frac.as<float>(), rec.as<uint4>());
    MG_CUDA(cudaGetLastError());
    MG_CUDA(cudaStreamSynchronize(s));   // read from other streams from here on
    frac.s = rec.s = nullptr;
    g->frac16[k] = std::move(frac);
    g->rec16[k] = std::move(rec);
    return MG_OK;
}

}  // namespace mg

// mg_query.cu -- segment histograms of boxes: footprint assembly (Sec. 3.6,
// Algorithm 1) and the reverse weight push through the Mixture Graph.
//
// Plan: clip the box, split each axis range into aligned power-of-two runs
// (footprint_1d), count the blocks of the runs' tensor product and the cubes
// tiling them (a block of run levels (lx, ly, lz) sits at level l = min and
// holds 2^(lx-l) * 2^(ly-l) * 2^(lz-l) cubes), then write one 12-byte record
// per block: first item, the index of its first item in its array, array, and
// log2 extents.  Blocks follow Algorithm 1's loop order (z, y, x).  A block one
// cube thick or 16 cubes long is read as tile records (mg_tiles.cu), each the
// exact segment counts of 16, 64 or 256 cubes; the others as the cubes' IDs.
// Every level is stored three times (x-, y- and z-fastest); a block reads the
// copy whose fastest axis is its longest side, so even a one-voxel-thick line
// reads contiguous IDs.
//
// Main (persistent CTAs, MG_SCHED_BATCHED): a global ticket hands out chunks of
// `chunk` consecutive items of one box to a warp with its own histogram in
// shared memory (few segments), or to a CTA that shares one (many).  A source
// adds its voxels to the histogram; a mixture node adds the segments of its
// record or table row, or is queued and pushed down its lerp tree (p gets
// W*a/(a+b), q gets W*b/(a+b), exact u32 arithmetic).  At the end of a chunk
// the touched bins are added to the box's row in global memory -- the only
// global atomics.  100,000 boxes on 2048x2048x300: 58,000 cubes a box become
// 890 units (280 tile records, 480 vectors and 120 cubes), 5.41 -> 1.08 ms;
// what is left is the latency of a chunk's dependent loads and its flush.
//
// MG_SCHED_PLAIN is the baseline: one launch and one CTA per box, walking the
// blocks in order.
#include "mg_internal.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

namespace mg {
namespace {

constexpr int kMaxRuns = 40;
constexpr int kMaxStack = 64;
constexpr uint32_t kMaxPushSteps = 1u << 24;   // a valid table never needs this many

// A block is read either as its cubes' IDs or as tiles (mg_tiles.cu): "array"
// l < 32 holds the IDs of level l, array tile_array(l, kind) the records of
// level l's tiles of that kind.
constexpr int kArrays = MG_MAX_LEVELS + 3 * kTileLevels;
__host__ __device__ __forceinline__ int tile_array(int l, int kind) { return MG_MAX_LEVELS + 3 * l + kind; }

struct Geom {
    int L;
    int id0_bytes;
    uint32_t S;
    int32_t dims[MG_MAX_LEVELS][3];
    // offset of level l >= 1 in copy c's concatenated levels, of a tile array
    // in the records
    int64_t off[kArrays][3];
    // strides of the second and third axis of each copy (copy 0: x, y, z;
    // copy 1: y, z, x; copy 2: z, x, y): the row pitch and pitch x middle dim
    uint32_t st1[kArrays][3], st2[kArrays][3];
    // tiles of the levels 0-3, four bits a level: log2 of the largest plane
    // edge (0, 3 or 4), plus 8 where the level has lines
    uint32_t tiles;
    // bit l of vec_ok[c] / vec32_ok[c]: every row of copy c at level l starts
    // on a 16-byte / 32-byte boundary (row pitch and level offset multiples)
    uint32_t vec_ok[3], vec32_ok[3];
};

struct Ids {
    const void* l0[3];       // level 0 copies (uint16 or uint32)
    const uint32_t* hi[3];   // levels >= 1 copies, concatenated at Geom::off
    const uint4* tiles;      // tile records
    const uint4* pool;       // their lists
};

struct Blk {
    uint32_t start;   // first item (cube or tile) of the block within its box
    uint32_t base;    // index of the block's first item in its copy of the array
    uint32_t meta;    // array | copy << 6 | e0 << 8 | e1 << 13 | e2 << 18 (log2 extents, copy axis order)
};

// tile_levels: levels whose tiles the caller's pushes may take (0: cubes only;
// 1: level 0, whose cubes are segments whatever the weights; kTileLevels:
// exact weights)
Geom make_geom(const mg_graph* g, int tile_levels) {
    Geom G;
    G.L = g->L;
    G.id0_bytes = g->id0_bytes;
    G.S = g->S;
    for (int l = 0; l < MG_MAX_LEVELS; l++) {
        for (int k = 0; k < 3; k++) G.dims[l][k] = g->geom.dims[l][k];
        const uint32_t dx = (uint32_t)G.dims[l][0], dy = (uint32_t)G.dims[l][1], dz = (uint32_t)G.dims[l][2];
        const uint32_t mid[3] = {dy, dz, dx};
        for (int c = 0; c < 3; c++) {
            G.off[l][c] = g->qoff[l][c];
            const uint32_t pitch = l < g->L ? (uint32_t)g->qpitch[l][c] : 1u;
            G.st1[l][c] = pitch;
            G.st2[l][c] = pitch * mid[c];
        }
    }
    G.tiles = 0;
    for (int l = 0; l < kTileLevels; l++) {
        if (l < tile_levels) G.tiles |= (uint32_t)(g->tgeom.edge[l] | (g->tgeom.line[l] ? 8 : 0)) << (4 * l);
        for (int k = 0; k < 3; k++)
            for (int c = 0; c < 3; c++) {
                const int a = tile_array(l, k);
                G.off[a][c] = g->tgeom.off[l][k][c];
                G.st1[a][c] = g->tgeom.st1[l][k][c];
                G.st2[a][c] = g->tgeom.st2[l][k][c];
            }
    }
    for (int c = 0; c < 3; c++) {
        G.vec_ok[c] = G.vec32_ok[c] = 0;
        for (int l = 0; l < G.L && l < MG_MAX_LEVELS; l++) {
            const uint32_t per16 = l == 0 ? 16u / (uint32_t)G.id0_bytes : 4u;   // IDs per 16 bytes
            const bool ok = G.st1[l][c] % per16 == 0 && G.st2[l][c] % per16 == 0 &&
                            (l == 0 || G.off[l][c] % per16 == 0);
            const uint32_t per32 = 2 * per16;
            const bool ok32 = G.st1[l][c] % per32 == 0 && G.st2[l][c] % per32 == 0 &&
                              (l == 0 || G.off[l][c] % per32 == 0);
            if (ok) G.vec_ok[c] |= 1u << l;
            if (ok32) G.vec32_ok[c] |= 1u << l;
        }
    }
    return G;
}

// 16-bit weights and quantised graphs push rounded weights through the trees:
// their levels >= 1 stay cubes
int tile_levels(const mg_graph* g, mg_dtype weights) {
    return weights == MG_F32 && !g->quantised && g->lut_meta.p ? kTileLevels : 1;
}

Ids make_ids(const mg_graph* g) {
    Ids I;
    for (int c = 0; c < 3; c++) {
        I.l0[c] = g->mip0x[c].p ? g->mip0x[c].p : g->mip0.p;   // copy 0 may be mip0 itself
        I.hi[c] = g->mipx[c].as<uint32_t>();
    }
    I.tiles = g->tiles.as<uint4>();
    I.pool = g->tile_pool.as<uint4>();
    return I;
}

// How a block of run levels (lx, ly, lz) is read: T = 3 or 4, as plane tiles
// of edge 2^T (one cube thick, the other two extents reaching 2^T; then the
// thickness axis is unique; the larger edge wherever the shorter side reaches
// it); T = 2, as lines of 16 (2^(2 T) cubes too: two extents under 8, the
// longest at least 16); T = 0, as cubes.
__device__ __forceinline__ int block_tile(uint32_t tiles, int lx, int ly, int lz) {
    const int lo = min(lx, ly), hi = max(lx, ly), l = min(lo, lz);
    const int mid = max(lo, min(hi, lz)) - l, most = max(hi, lz) - l;
    const int t = l < kTileLevels ? (int)(tiles >> (4 * l)) & 15 : 0;
    return mid >= 3 ? min(mid, t & 7) : (t & 8) && most >= 4 ? 2 : 0;
}

// items of a block: cubes, or tiles of 2^(2 T) cubes
__device__ __forceinline__ uint32_t block_items(int lx, int ly, int lz, int T) {
    const int l = min(lx, min(ly, lz));
    return 1u << (lx + ly + lz - 3 * l - 2 * T);
}

// block of run levels (lx, ly, lz) whose origin is the level-0 voxel (x0, y0,
// z0), read as T says
__device__ __forceinline__ Blk make_blk(const Geom& G, uint32_t start, int32_t x0, int32_t y0, int32_t z0, int lx,
                                        int ly, int lz, int T) {
    const int l = min(lx, min(ly, lz));
    // plane tiles lie in the copy whose slowest axis is the thickness, all
    // else in the copy whose fastest axis is the longest side
    const int c = T >= 3 ? (lz == l ? 0 : lx == l ? 1 : 2) : (lx >= ly && lx >= lz) ? 0 : ly >= lz ? 1 : 2;
    const int v = T == 0 ? l : tile_array(l, T == 2 ? 2 : T - 3);
    const int32_t a0 = c == 0 ? x0 : c == 1 ? y0 : z0, b0 = c == 0 ? y0 : c == 1 ? z0 : x0;
    const int32_t t0 = c == 0 ? z0 : c == 1 ? x0 : y0;
    const int la = c == 0 ? lx : c == 1 ? ly : lz, lb = c == 0 ? ly : c == 1 ? lz : lx;
    const int lt = c == 0 ? lz : c == 1 ? lx : ly;
    const int sa = l + (T == 2 ? 4 : T), sb = l + (T == 2 ? 0 : T);   // log2 item extents
    Blk B;
    B.start = start;
    B.base = ((uint32_t)t0 >> l) * G.st2[v][c] + ((uint32_t)b0 >> sb) * G.st1[v][c] + ((uint32_t)a0 >> sa);
    B.meta = (uint32_t)(v | c << 6 | (la - sa) << 8 | (lb - sb) << 13 | (lt - l) << 18);
    return B;
}

// Algorithm 1, footprint_1d: aligned power-of-two steps covering [i, i+di)
// clipped to [0, dim); tzcnt(0) is infinite.
__device__ __forceinline__ int footprint_1d(int64_t i, int64_t di, int64_t dim, uint8_t* r, int32_t* start) {
    int n = 0;
    di = min(i + di, dim) - i;
    while (di > 0 && n < kMaxRuns) {
        const int a = 63 - __clzll(di);
        const int b = i == 0 ? 63 : __ffsll(i) - 1;
        const int l = min(a, b);
        r[n] = (uint8_t)l;
        start[n] = (int32_t)i;
        n++;
        di -= (int64_t)1 << l;
        i += (int64_t)1 << l;
    }
    return n;
}

__device__ __forceinline__ bool box_ok(const int32_t* b, const Geom& G) {
    return b[0] >= 0 && b[0] < G.dims[0][0] && b[1] >= 0 && b[1] < G.dims[0][1] && b[2] >= 0 &&
           b[2] < G.dims[0][2] && b[3] >= 1 && b[4] >= 1 && b[5] >= 1;
}

struct Runs {
    uint8_t lx[kMaxRuns], ly[kMaxRuns], lz[kMaxRuns];
    int32_t sx[kMaxRuns], sy[kMaxRuns], sz[kMaxRuns];
    int nx, ny, nz;
};

__device__ __forceinline__ void make_runs(const int32_t* b, const Geom& G, Runs& R) {
    R.nx = footprint_1d(b[0], b[3], G.dims[0][0], R.lx, R.sx);
    R.ny = footprint_1d(b[1], b[4], G.dims[0][1], R.ly, R.sy);
    R.nz = footprint_1d(b[2], b[5], G.dims[0][2], R.lz, R.sz);
}

// the runs of a warp's box, one axis per lane, into the warp's shared slot
__device__ __forceinline__ void make_runs_warp(const int32_t* b, const Geom& G, Runs& R) {
    const int lane = threadIdx.x & 31;
    if (lane == 0) R.nx = footprint_1d(b[0], b[3], G.dims[0][0], R.lx, R.sx);
    else if (lane == 1) R.ny = footprint_1d(b[1], b[4], G.dims[0][1], R.ly, R.sy);
    else if (lane == 2) R.nz = footprint_1d(b[2], b[5], G.dims[0][2], R.lz, R.sz);
    __syncwarp();
}

constexpr int kPlanThreads = 256;   // plan kernels: one warp per box

__device__ __forceinline__ uint32_t block_cubes(int lx, int ly, int lz) {
    const int l = min(lx, min(ly, lz));
    return 1u << (lx + ly + lz - 3 * l);
}

// Footprint cubes of a box in closed form.  On each axis let F(m) be the sum
// over its runs of level a >= m of 2^(a-m), and P(m) = Fx(m) Fy(m) Fz(m).  A
// block of run levels (a, b, c) with minimum m0 adds 2^(a+b+c-3m) to P(m) for
// every m <= m0, so the blocks' cubes, sum 2^(a+b+c-3 m0), equal
// P(0) - 7 * sum over m >= 1 of P(m).  Algorithm 1's steps on one axis rise
// to a peak and fall again, so no level occurs more than twice and two bit
// masks hold an axis's levels: F(m) = (once >> m) + (twice >> m).
struct Masks {
    uint32_t once, twice;   // levels below 32: an axis's voxels are counted in int32
    __device__ __forceinline__ uint32_t sum(int m) const { return (once >> m) + (twice >> m); }            // F(m)
    __device__ __forceinline__ uint32_t runs(int l) const { return ((once >> l) & 1) + ((twice >> l) & 1); }
};

__device__ __forceinline__ Masks level_masks(const uint8_t* l, int n) {
    Masks M{0u, 0u};
    for (int i = 0; i < n; i++) {
        const uint32_t bit = 1u << l[i];
        if (M.once & bit) M.twice |= bit;
        else M.once |= bit;
    }
    return M;
}

// level m's term of that sum
__device__ __forceinline__ uint64_t cube_term(int m, const Masks& x, const Masks& y, const Masks& z) {
    const uint64_t p = (uint64_t)x.sum(m) * y.sum(m) * z.sum(m);
    return m == 0 ? p : 0ull - 7 * p;
}

// Items of the same footprint: level l's change to the count of cubes.  A
// block of level l on axis t and extents 2^a, 2^b >= 8 cubes on the others
// counts 2^(a+b) cubes but 2^(a+b-6) tiles of edge 8, or 2^(a+b-8) of edge 16
// where both extents reach 16: summed over such blocks, with n_t(l) the runs
// of level l on axis t, n_t(l) (63 F(l+3) F'(l+3) + 3 F(l+4) F'(l+4)) less, the
// last term with edge 16.  Lines along axis t replace 16 cubes each where the
// other axes' levels lie within l..l+2 and one of them is l: 15 F(l+4) times
// the sum over such pairs less.
__device__ __forceinline__ uint64_t tile_term(uint32_t tiles, int l, const Masks& x, const Masks& y, const Masks& z) {
    const uint32_t t = l < kTileLevels ? (tiles >> (4 * l)) & 15u : 0u;
    if (!t) return 0;
    const uint64_t nx = x.runs(l), ny = y.runs(l), nz = z.runs(l);
    const uint64_t fx = x.sum(l + 3), fy = y.sum(l + 3), fz = z.sum(l + 3);
    const uint64_t gx = x.sum(l + 4), gy = y.sum(l + 4), gz = z.sum(l + 4);
    uint64_t less = 0;
    if (t & 7u) less += 63 * (nx * fy * fz + ny * fz * fx + nz * fx * fy);
    if ((t & 7u) == 4u) less += 3 * (nx * gy * gz + ny * gz * gx + nz * gx * gy);
    if (t & 8u) {
        // cubes across of the runs of levels l + 1 and l + 2, per axis
        const uint64_t wx = 2 * x.runs(l + 1) + 4 * x.runs(l + 2), wy = 2 * y.runs(l + 1) + 4 * y.runs(l + 2),
                       wz = 2 * z.runs(l + 1) + 4 * z.runs(l + 2);
        less += 15 * (gx * (ny * nz + ny * wz + wy * nz) + gy * (nz * nx + nz * wx + wz * nx) +
                      gz * (nx * ny + nx * wy + wx * ny));
    }
    return 0ull - less;
}

constexpr int kMaxAxisLevels = 32;

// cubes of a footprint, or its items (tiles = G.tiles; 0: cubes)
__device__ __forceinline__ uint64_t footprint_count(const Runs& R, uint32_t tiles) {
    const Masks x = level_masks(R.lx, R.nx), y = level_masks(R.ly, R.ny), z = level_masks(R.lz, R.nz);
    uint64_t n = 0;
    for (int m = 0; m < kMaxAxisLevels && (x.once >> m) && (y.once >> m) && (z.once >> m); m++)
        n += cube_term(m, x, y, z) + tile_term(tiles, m, x, y, z);
    return n;
}

// A batch planned by the fused kernel: the footprint must fit the buffers, and
// the batch size is known (Qd == nullptr) or, for plans replayed as CUDA
// graphs, read on the device: the launches then cover Q boxes, *Qd of them live.
struct Lim {
    const int64_t* Qd;
    uint64_t cap_blocks, cap_chunks;
};

__device__ __forceinline__ int64_t live_q(const Lim& lim, int64_t Q) { return lim.Qd ? *lim.Qd : Q; }

// ---------------------------------------------------------------------------
// plan
// ---------------------------------------------------------------------------
__global__ void plan_count_kernel(Geom G, const int32_t* __restrict__ boxes, int64_t Q, uint32_t chunk,
                                  uint32_t* __restrict__ nblk, uint64_t* __restrict__ ncube,
                                  uint64_t* __restrict__ nchunk, unsigned* __restrict__ status, bool items) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= Q) return;
    int32_t b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
    if (!box_ok(b, G)) {
        if (lane == 0) {
            set_status(status, kStatBadInput);
            if (nblk) nblk[q] = 0;
            ncube[q] = 0;
            if (nchunk) nchunk[q] = 0;
        }
        return;
    }
    __shared__ Runs wr[kPlanThreads / 32];
    Runs& R = wr[threadIdx.x >> 5];
    make_runs_warp(b, G, R);
    if (lane == 0) {
        const uint64_t cubes = footprint_count(R, items ? G.tiles : 0u);
        if (nblk) nblk[q] = (uint32_t)(R.nx * R.ny * R.nz);
        ncube[q] = cubes;
        if (nchunk) nchunk[q] = (cubes + chunk - 1) / chunk;
    }
}

// Block records of every box, and for every work chunk of `chunk` cubes its
// box and the block holding its first cube.
__global__ void plan_write_kernel(Geom G, const int32_t* __restrict__ boxes, int64_t Q,
                                  const uint64_t* __restrict__ blk_off, Blk* __restrict__ blk,
                                  const uint64_t* __restrict__ chunk_off, uint32_t chunk,
                                  uint32_t* __restrict__ chunk_q, uint32_t* __restrict__ chunk_b) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= Q) return;
    int32_t b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
    if (!box_ok(b, G)) return;
    __shared__ Runs wr[kPlanThreads / 32];
    Runs& R = wr[threadIdx.x >> 5];
    make_runs_warp(b, G, R);
    const uint64_t base = blk_off[q], cbase = chunk_off[q];
    const int npairs = R.ny * R.nz;
    uint32_t running = 0;
    for (int pbase = 0; pbase < npairs; pbase += 32) {
        const int pr = pbase + lane;
        const bool valid = pr < npairs;
        const int j = valid ? pr % R.ny : 0, k = valid ? pr / R.ny : 0;
        uint32_t row = 0;
        if (valid)
            for (int i = 0; i < R.nx; i++)
                row += block_items(R.lx[i], R.ly[j], R.lz[k], block_tile(G.tiles, R.lx[i], R.ly[j], R.lz[k]));
        // exclusive warp scan of the row totals
        uint32_t incl = row;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        if (valid) {
            uint32_t start = running + incl - row;
            for (int i = 0; i < R.nx; i++) {
                const uint64_t bi = base + (uint64_t)pr * R.nx + i;
                const int T = block_tile(G.tiles, R.lx[i], R.ly[j], R.lz[k]);
                const uint32_t n = block_items(R.lx[i], R.ly[j], R.lz[k], T);
                blk[bi] = make_blk(G, start, R.sx[i], R.sy[j], R.sz[k], R.lx[i], R.ly[j], R.lz[k], T);
                // the chunks whose first cube lies in this block
                for (uint64_t c = ((uint64_t)start + chunk - 1) / chunk; c * chunk < (uint64_t)start + n; c++) {
                    chunk_q[cbase + c] = (uint32_t)q;
                    chunk_b[cbase + c] = (uint32_t)bi;
                }
                start += n;
            }
        }
        running += tot;
    }
}

// ---------------------------------------------------------------------------
// The plan of a query-plan run in one launch: the footprint counts of every
// box, both exclusive scans in a single pass, the zeroing of the batch's
// output rows, the block records and the chunk map.  CTAs take tiles of `tb`
// boxes in ticket order (tb chosen on the host so that the tiles of a full
// batch fill the GPU once); a tile publishes its own totals, then sums its
// predecessors' words backwards until it meets one that holds an inclusive
// prefix, and publishes its own prefix.  The tile words and the ticket are zero
// at launch: the main kernel, which starts reading once this one has ended,
// zeroes them for the next batch.
// ---------------------------------------------------------------------------
constexpr int kTileMax = 64;                     // boxes per tile at most
constexpr int kFusedThreads = 512;
constexpr int kFusedWarps = kFusedThreads / 32;
constexpr int kBoxLanes = 8;                     // lanes per box in the count phase (three build runs)
constexpr int kBoxGroups = kFusedThreads / kBoxLanes;
constexpr int kScanPerLane = kTileMax / 32;      // boxes per lane in the tile scan
constexpr int kFusedItems = 6;                   // blocks per thread and round, interleaved
constexpr int kLookWindows = 4;                  // look-back windows of 32 tiles loaded per poll
constexpr uint64_t kTileAgg = 1ull << 62;        // the word holds the tile's own total
constexpr uint64_t kTilePre = 2ull << 62;        // the word holds the inclusive prefix
constexpr uint64_t kTileVal = (1ull << 62) - 1;
constexpr unsigned kLookbackLimit = 1u << 20;    // polls before the look-back gives up

// boxes per tile for a batch of Q: about one tile per resident CTA
int tile_boxes(int64_t Q, int sms) {
    const int64_t slots = (int64_t)sms * 2;
    return (int)std::min<int64_t>(kTileMax, std::max<int64_t>(1, (Q + slots - 1) / slots));
}

struct FusedOut {
    uint64_t* ncube;
    uint64_t* blk_off;
    uint64_t* chunk_off;
    Blk* blk;
    uint32_t* chunk_q;
    uint32_t* chunk_b;
    uint64_t* tiles;               // two words per tile: blocks, chunks
    unsigned long long* ticket;    // tile order; [1]: the main kernel's, zeroed here
    uint32_t* acc;                 // rows zeroed for the live batch
    float* accf;                   // likewise (fp32 histograms), or nullptr
    void* const* io;               // io[0]: the boxes; io[1]: the output (acc for u32, accf for fp32)
};

// Algorithm 1's steps on one axis (as footprint_1d) together with the axis's
// level masks (levels seen once, levels seen twice)
// (0 <= i < dim <= 65535, di >= 1)
__device__ __forceinline__ int axis_runs(int32_t i, int32_t di, int32_t dim, uint8_t* r, int32_t* start, Masks& M) {
    int n = 0;
    M = Masks{0u, 0u};
    di = min(di, dim - i);
    while (di > 0 && n < kMaxRuns) {
        const int a = 31 - __clz(di);
        const int l = i == 0 ? a : min(a, __ffs(i) - 1);
        const uint32_t bit = 1u << l;
        M.twice |= M.once & bit;
        M.once |= bit;
        r[n] = (uint8_t)l;
        start[n] = i;
        n++;
        di -= (int32_t)bit;
        i += (int32_t)bit;
    }
    return n;
}

// zero a[r0, r1) of 4-byte elements (a 4-byte aligned) with 16-byte stores
// between the unaligned ends
template <typename T>
__device__ __forceinline__ void zero_span(T* a, size_t r0, size_t r1) {
    static_assert(sizeof(T) == 4, "4-byte elements");
    const size_t lead = ((16u - (reinterpret_cast<uintptr_t>(a + r0) & 15u)) & 15u) / 4u;
    const size_t a0 = min(r0 + lead, r1), a1 = a0 + ((r1 - a0) & ~(size_t)3);
    for (size_t i = r0 + threadIdx.x; i < a0; i += kFusedThreads) a[i] = T(0);
    for (size_t i = a1 + threadIdx.x; i < r1; i += kFusedThreads) a[i] = T(0);
    uint4* v = reinterpret_cast<uint4*>(a + a0);
    for (size_t i = threadIdx.x; i < (a1 - a0) / 4; i += kFusedThreads) v[i] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(kFusedThreads, 2) plan_fused_kernel(const __grid_constant__ Geom G,
                                                                      const int32_t* __restrict__ boxes,
                                                                      int64_t Q, int tb, uint32_t chunk,
                                                                      int chunk_shift, Lim lim, FusedOut F,
                                                                      unsigned* __restrict__ status) {
    __shared__ Runs wr[kTileMax];
    __shared__ uint32_t s_nblk[kTileMax];
    __shared__ uint64_t s_ncube[kTileMax];
    __shared__ uint64_t s_mx[kTileMax], s_my[kTileMax];   // ceil(2^32 / nx), ceil(2^32 / ny)
    __shared__ uint32_t s_boff[kTileMax + 1];   // tile-local block offsets, total last
    __shared__ uint64_t s_coff[kTileMax + 1];   // tile-local chunk offsets, total last
    __shared__ uint32_t s_cube[kTileMax];       // tile-local cube offsets, mod 2^32
    __shared__ uint32_t s_wsum[kFusedWarps][kFusedItems];
    __shared__ uint32_t s_rtot[kFusedItems];
    __shared__ unsigned long long s_tile;
    __shared__ uint64_t s_pre_b, s_pre_c;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        s_tile = gridDim.x == 1 ? 0ull : atomicAdd(F.ticket, 1ull);
        if (s_tile == 0) F.ticket[1] = 0;
    }
    // the main kernel may be scheduled once every tile has started; it waits
    // for this grid's completion before it reads anything written here
    grid_dependents_launch();
    __syncthreads();
    const int64_t tile = (int64_t)s_tile;
    const int64_t Qe = live_q(lim, Q);
    const int64_t q0 = tile * tb;
    if (q0 >= Qe) return;   // no tile of the live batch waits on this one
    uint32_t* acc = F.acc;
    float* accf = F.accf;
    if (F.io) {
        boxes = static_cast<const int32_t*>(F.io[0]);
        if (accf) accf = static_cast<float*>(F.io[1]);
        else acc = static_cast<uint32_t*>(F.io[1]);
    }

    // 1. blocks and cubes of every box: kBoxLanes lanes per box, lanes 0-2 of
    // a group building one axis's runs each
    const int grp = threadIdx.x / kBoxLanes, bl = threadIdx.x % kBoxLanes;
    for (int w0 = 0; w0 < tb; w0 += kBoxGroups) {
        const int w = w0 + grp;
        const int64_t q = q0 + w;
        const bool live = w < tb && q < Qe;
        bool ok = false;
        Masks M{0u, 0u};
        if (live) {
            int32_t b[6];
#pragma unroll
            for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
            ok = box_ok(b, G);
            if (!ok && bl == 0) set_status(status, kStatBadInput);
            if (ok && bl < 3) {
                Runs& R = wr[w];
                const int32_t i0 = bl == 0 ? b[0] : bl == 1 ? b[1] : b[2];
                const int32_t di = bl == 0 ? b[3] : bl == 1 ? b[4] : b[5];
                const int32_t dim = bl == 0 ? G.dims[0][0] : bl == 1 ? G.dims[0][1] : G.dims[0][2];
                uint8_t* lv = bl == 0 ? R.lx : bl == 1 ? R.ly : R.lz;
                int32_t* sv = bl == 0 ? R.sx : bl == 1 ? R.sy : R.sz;
                const int n = axis_runs(i0, di, dim, lv, sv, M);
                if (bl == 0) R.nx = n;
                else if (bl == 1) R.ny = n;
                else R.nz = n;
            }
        }
        // the group's lanes take the levels of the closed form in turn
        const Masks x{__shfl_sync(0xffffffffu, M.once, 0, kBoxLanes), __shfl_sync(0xffffffffu, M.twice, 0, kBoxLanes)};
        const Masks y{__shfl_sync(0xffffffffu, M.once, 1, kBoxLanes), __shfl_sync(0xffffffffu, M.twice, 1, kBoxLanes)};
        const Masks z{__shfl_sync(0xffffffffu, M.once, 2, kBoxLanes), __shfl_sync(0xffffffffu, M.twice, 2, kBoxLanes)};
        __syncwarp();
        uint64_t items = tile_term(G.tiles, bl, x, y, z);
        for (int m = bl; m < kMaxAxisLevels; m += kBoxLanes) items += cube_term(m, x, y, z);
#pragma unroll
        for (int o = kBoxLanes / 2; o > 0; o >>= 1) items += __shfl_xor_sync(0xffffffffu, items, o, kBoxLanes);
        if (w < tb) {
            if (bl == 0) {
                if (live) F.ncube[q] = items;
                s_ncube[w] = items;
                s_nblk[w] = ok ? (uint32_t)(wr[w].nx * wr[w].ny * wr[w].nz) : 0u;
            } else if (bl <= 2 && ok) {
                // ceil(2^32 / n)
                const uint32_t n = (uint32_t)(bl == 1 ? wr[w].nx : wr[w].ny);
                (bl == 1 ? s_mx : s_my)[w] = (uint64_t)(0xffffffffu / n) + 1;
            }
        }
    }
    {   // the tile's live output rows are one contiguous span
        const size_t r0 = (size_t)q0 * G.S, r1 = (size_t)min(q0 + tb, Qe) * G.S;
        zero_span(acc, r0, r1);
        if (accf) zero_span(accf, r0, r1);
    }
    __syncthreads();

    // 2. offsets within the tile (kScanPerLane consecutive boxes per lane),
    // then the prefix of all earlier tiles
    if (warp == 0) {
        uint64_t nbk[kScanPerLane], nck[kScanPerLane], nqk[kScanPerLane];
        uint64_t xb = 0, xc = 0, xq = 0;
#pragma unroll
        for (int k = 0; k < kScanPerLane; k++) {
            const int w = lane * kScanPerLane + k;
            nbk[k] = w < tb ? s_nblk[w] : 0u;
            nqk[k] = w < tb ? s_ncube[w] : 0u;
            nck[k] = chunk_shift >= 0 ? (nqk[k] + chunk - 1) >> chunk_shift : (nqk[k] + chunk - 1) / chunk;
            xb += nbk[k];
            xc += nck[k];
            xq += nqk[k];
        }
        uint64_t ib = xb, ic = xc, iq = xq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t yb = __shfl_up_sync(0xffffffffu, ib, o);
            const uint64_t yc = __shfl_up_sync(0xffffffffu, ic, o);
            const uint64_t yq = __shfl_up_sync(0xffffffffu, iq, o);
            if (lane >= o) {
                ib += yb;
                ic += yc;
                iq += yq;
            }
        }
        uint64_t ob = ib - xb, oc = ic - xc, oq = iq - xq;
#pragma unroll
        for (int k = 0; k < kScanPerLane; k++) {
            s_boff[lane * kScanPerLane + k] = (uint32_t)ob;
            s_coff[lane * kScanPerLane + k] = oc;
            s_cube[lane * kScanPerLane + k] = (uint32_t)oq;
            ob += nbk[k];
            oc += nck[k];
            oq += nqk[k];
        }
        const uint64_t agg_b = __shfl_sync(0xffffffffu, ib, 31), agg_c = __shfl_sync(0xffffffffu, ic, 31);
        if (lane == 0) {
            s_boff[kTileMax] = (uint32_t)agg_b;
            s_coff[kTileMax] = agg_c;
        }
        uint64_t* word = F.tiles + 2 * tile;
        if (lane == 0) {
            const uint64_t flag = tile == 0 ? kTilePre : kTileAgg;
            st_relaxed_u64(word, flag | agg_b);
            st_relaxed_u64(word + 1, flag | agg_c);
        }
        // look back kLookWindows windows of 32 tiles per poll; a word pair
        // counts once both words carry the same flag
        uint64_t eb = 0, ec = 0;
        int64_t top = tile - 1;
        unsigned polls = 0;
        bool done = top < 0;
        while (!done) {
            uint64_t wb[kLookWindows], wc[kLookWindows];
#pragma unroll
            for (int k = 0; k < kLookWindows; k++) {
                const int64_t t = top - lane - 32 * k;
                wb[k] = wc[k] = kTilePre;   // before the first tile: prefix 0
                if (t >= 0) {
                    wb[k] = ld_relaxed_u64(F.tiles + 2 * t);
                    wc[k] = ld_relaxed_u64(F.tiles + 2 * t + 1);
                }
            }
            bool late_seen = false;
#pragma unroll
            for (int k = 0; k < kLookWindows; k++) {
                if (done || late_seen) continue;
                const bool ready = (wb[k] >> 62) != 0 && (wb[k] >> 62) == (wc[k] >> 62);
                const unsigned pre = __ballot_sync(0xffffffffu, ready && (wb[k] >> 62) == 2u);
                const unsigned late = __ballot_sync(0xffffffffu, !ready);
                // the lanes up to the nearest tile holding its prefix are needed
                const unsigned need = pre ? ((pre & (0u - pre)) << 1) - 1u : 0xffffffffu;
                if (late & need) {
                    late_seen = true;
                    continue;
                }
                const bool use = (need >> lane) & 1u;
                uint64_t vb = use ? wb[k] & kTileVal : 0u, vc = use ? wc[k] & kTileVal : 0u;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    vb += __shfl_xor_sync(0xffffffffu, vb, o);
                    vc += __shfl_xor_sync(0xffffffffu, vc, o);
                }
                eb += vb;
                ec += vc;
                if (pre) done = true;
                else top -= 32;
            }
            if (late_seen && !done) {
                if (++polls > kLookbackLimit) {
                    if (lane == 0) set_status(status, kStatTimeout);
                    break;
                }
                __nanosleep(64);
            }
        }
        if (lane == 0) {
            if (tile > 0) {
                st_relaxed_u64(word, kTilePre | (eb + agg_b));
                st_relaxed_u64(word + 1, kTilePre | (ec + agg_c));
            }
            s_pre_b = eb;
            s_pre_c = ec;
        }
    }
    __syncthreads();
    const uint64_t pre_b = s_pre_b, pre_c = s_pre_c;
    const uint64_t tot_b = pre_b + s_boff[kTileMax], tot_c = pre_c + s_coff[kTileMax];
    for (int w = threadIdx.x; w < tb; w += kFusedThreads) {
        const int64_t q = q0 + w;
        if (q >= Qe) break;
        F.blk_off[q] = pre_b + s_boff[w];
        F.chunk_off[q] = pre_c + s_coff[w];
        if (q == Qe - 1) {
            F.blk_off[Qe] = tot_b;
            F.chunk_off[Qe] = tot_c;
            if (tot_b > lim.cap_blocks || tot_c > lim.cap_chunks) set_status(status, kStatCapacity);
        }
    }
    // past the plan's buffers: the last tile has flagged the batch, nothing is written
    if (tot_b > lim.cap_blocks || tot_c > lim.cap_chunks) return;

    // 3. block records and the chunk map; item `it` of thread t is the tile's
    // block r0 + it * kFusedThreads + t.  A box's block t is row pr = t / nx,
    // column i = t - pr nx; the quotients by nx, ny < 2^16 of numerators
    // < 2^16 are exact as (n * ceil(2^32 / d)) >> 32.
    const uint32_t nbt = s_boff[kTileMax];
    uint32_t carry = 0;   // cubes of the earlier rounds, mod 2^32
    for (uint32_t r0 = 0; r0 < nbt; r0 += kFusedThreads * kFusedItems) {
        uint32_t n[kFusedItems], incl[kFusedItems];
        int wk[kFusedItems], ik[kFusedItems], jk[kFusedItems], kk[kFusedItems], tk[kFusedItems];
#pragma unroll
        for (int it = 0; it < kFusedItems; it++) {
            const uint32_t idx = r0 + it * kFusedThreads + threadIdx.x;
            n[it] = 0;
            wk[it] = ik[it] = jk[it] = kk[it] = tk[it] = 0;
            if (idx < nbt) {
                int w = 0;   // the last box whose blocks start at or before idx
#pragma unroll
                for (int st = kTileMax / 2; st > 0; st >>= 1)
                    if (s_boff[w + st] <= idx) w += st;
                const Runs& R = wr[w];
                const uint32_t t = idx - s_boff[w];
                const uint32_t pr = (uint32_t)(((uint64_t)t * s_mx[w]) >> 32);
                const uint32_t k = (uint32_t)(((uint64_t)pr * s_my[w]) >> 32);
                wk[it] = w;
                ik[it] = (int)(t - pr * (uint32_t)R.nx);
                jk[it] = (int)(pr - k * (uint32_t)R.ny);
                kk[it] = (int)k;
                const int lx = R.lx[ik[it]], ly = R.ly[jk[it]], lz = R.lz[kk[it]];
                tk[it] = block_tile(G.tiles, lx, ly, lz);
                n[it] = block_items(lx, ly, lz, tk[it]);
            }
            uint32_t v = n[it];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += y;
            }
            incl[it] = v;
            if (lane == 31) s_wsum[warp][it] = v;
        }
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int it = 0; it < kFusedItems; it++) {
                const uint32_t x = lane < kFusedWarps ? s_wsum[lane][it] : 0u;
                uint32_t v = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
                    if (lane >= o) v += y;
                }
                __syncwarp();
                if (lane < kFusedWarps) s_wsum[lane][it] = v - x;
                if (lane == 31) s_rtot[it] = v;
            }
        }
        __syncthreads();
        uint32_t base = carry;
#pragma unroll
        for (int it = 0; it < kFusedItems; it++) {
            const uint32_t idx = r0 + it * kFusedThreads + threadIdx.x;
            if (idx < nbt) {
                const int w = wk[it], i = ik[it], j = jk[it], k = kk[it];
                const Runs& R = wr[w];
                const uint32_t start = base + s_wsum[warp][it] + incl[it] - n[it] - s_cube[w];
                const uint64_t bi = pre_b + idx;
                F.blk[bi] = make_blk(G, start, R.sx[i], R.sy[j], R.sz[k], R.lx[i], R.ly[j], R.lz[k], tk[it]);
                const uint64_t cb = pre_c + s_coff[w];
                const uint64_t first = (uint64_t)start + chunk - 1;
                for (uint64_t c = chunk_shift >= 0 ? first >> chunk_shift : first / chunk;
                     c * chunk < (uint64_t)start + n[it]; c++) {
                    F.chunk_q[cb + c] = (uint32_t)(q0 + w);
                    F.chunk_b[cb + c] = (uint32_t)bi;
                }
            }
            base += s_rtot[it];
        }
        carry = base;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// shared-memory histogram of one chunk
// ---------------------------------------------------------------------------
template <bool FP>
struct Hist {
    uint32_t* h;        // S integer bins
    float* hf;          // S fractional bins (fp32 push)
    uint16_t* touched;  // bins to flush (when tracking)
    uint32_t* ntouched;
    bool track;         // false: the flush scans all S bins, adds need no return value

    __device__ __forceinline__ void add_int(uint32_t s, uint32_t w) const {
        if (track) {
            if (atomicAdd(h + s, w) == 0u) touched[atomicAdd(ntouched, 1u)] = (uint16_t)s;
        } else {
            atomicAdd(h + s, w);
        }
    }
    __device__ __forceinline__ void add_frac(uint32_t s, float w) const {
        if (track) {
            if (atomicAdd(hf + s, w) == 0.f) touched[atomicAdd(ntouched, 1u)] = (uint16_t)s;
        } else {
            atomicAdd(hf + s, w);
        }
    }
};

// segment counts up to this are flushed by scanning every bin
constexpr uint32_t kScanFlushMax = 2048;
// segment counts up to this get one histogram per warp
constexpr uint32_t kWarpHistMax = 2048;

template <typename AT> struct AlphaCvt;
template <> struct AlphaCvt<float> {
    static __device__ __forceinline__ float to(float x) { return x; }
};
template <> struct AlphaCvt<__half> {
    static __device__ __forceinline__ float to(__half x) { return __half2float(x); }
};
template <> struct AlphaCvt<__nv_bfloat16> {
    static __device__ __forceinline__ float to(__nv_bfloat16 x) { return __bfloat162float(x); }
};

struct PushArgs {
    const uint2* pq;
    const uint2* ab32;
    const void* alpha;
    uint32_t S;
    unsigned* status;
    const uint2* lut_meta;   // mixture lookup table (null: walk the lerp trees)
    const uint2* lut;
    const uint4* rec;        // records of the nodes in the table (null: none)
    const float* frac;       // 16-bit weights: the share of each table entry
};

// The table row of node n for a push of weight w: entries (source, count)
// scaled to 8^lmin, so each source receives (w >> 3 lmin) * count.  len = 0
// when n has no row or w is not a multiple of 8^lmin (then the tree is walked).
__device__ __forceinline__ void lut_row(const PushArgs& P, uint32_t n, uint32_t w, uint32_t& off, uint32_t& len,
                                        uint32_t& k) {
    const uint2 m = __ldg(P.lut_meta + n);
    const uint32_t lm = 3u * (m.y & 255u);
    len = m.y >> 8;
    off = m.x;
    k = w >> lm;
    if (len && (k << lm) != w) len = 0;
}

// exact integer push of weight W from node n (Sec. 3.6 with the lerp tree of
// Sec. 3.2): depth-first, one branch kept in registers, the other stacked
template <bool FP>
__device__ void push_int(const PushArgs& P, const Hist<FP>& H, uint32_t n, uint32_t w) {
    uint32_t sn[kMaxStack], sw[kMaxStack];
    int sp = 0;
    for (uint32_t step = 0;; step++) {
        if (step >= kMaxPushSteps) {
            set_status(P.status, kStatInexact);
            return;
        }
        if (n < P.S) {
            H.add_int(n, w);
            if (sp == 0) return;
            --sp;
            n = sn[sp];
            w = sw[sp];
            continue;
        }
        const uint2 e = __ldg(P.pq + n);
        const uint2 ab = __ldg(P.ab32 + n);
        const uint32_t s = ab.x + ab.y;
        const uint32_t k = s ? w / s : 0u;
        if (s == 0 || k * s != w || sp >= kMaxStack) {
            set_status(P.status, kStatInexact);
            if (sp == 0) return;
            --sp;
            n = sn[sp];
            w = sw[sp];
            continue;
        }
        sn[sp] = e.y;
        sw[sp] = k * ab.y;
        sp++;
        n = e.x;
        w = k * ab.x;
    }
}

// fp32 push: q receives W*alpha, p the rest
template <typename AT>
__device__ void push_frac(const PushArgs& P, const Hist<true>& H, uint32_t n, float w) {
    uint32_t sn[kMaxStack];
    float sw[kMaxStack];
    int sp = 0;
    const AT* alpha = static_cast<const AT*>(P.alpha);
    for (uint32_t step = 0;; step++) {
        if (step >= kMaxPushSteps) {
            set_status(P.status, kStatInexact);
            return;
        }
        if (n < P.S) {
            H.add_frac(n, w);
            if (sp == 0) return;
            --sp;
            n = sn[sp];
            w = sw[sp];
            continue;
        }
        const uint2 e = __ldg(P.pq + n);
        float al = AlphaCvt<AT>::to(alpha[n]);
        uint32_t p = e.x, q = e.y;
        if (al < 0.f) {   // 16-bit weights: sign = p and q swapped, |alpha| <= 1/2
            al = -al;
            p = e.y;
            q = e.x;
        }
        if (sp >= kMaxStack) {
            set_status(P.status, kStatInexact);
            return;
        }
        const float wq = w * al;
        sn[sp] = q;
        sw[sp] = wq;
        sp++;
        n = p;
        w = w - wq;
    }
}

// the push of one (node, weight) by one lane: its mixture-table row, else its
// lerp tree
template <bool FP, typename AT>
__device__ __noinline__ void push_one(const PushArgs& P, const Hist<FP>& H, uint32_t n, uint32_t w) {
    if (std::is_same<AT, float>::value && P.lut_meta) {
        uint32_t off, len, k;
        lut_row(P, n, w, off, len, k);
        if (len) {
            for (uint32_t e = 0; e < len; e++) {
                const uint2 ent = __ldg(P.lut + off + e);
                H.add_int(ent.x, k * ent.y);
            }
            return;
        }
    }
    if constexpr (FP) push_frac<AT>(P, H, n, (float)w);
    else push_int<FP>(P, H, n, w);
}

__device__ __forceinline__ uint32_t read_id(const Geom& G, const Ids& I, int l, int c, uint32_t idx) {
    if (l == 0)
        return G.id0_bytes == 2 ? (uint32_t)__ldg(static_cast<const uint16_t*>(I.l0[c]) + idx)
                                : __ldg(static_cast<const uint32_t*>(I.l0[c]) + idx);
    return __ldg(I.hi[c] + G.off[l][c] + idx);
}

// node ID of cube o of block B
__device__ __forceinline__ uint32_t cube_node(const Geom& G, const Ids& I, const Blk& B, uint32_t o, int& l) {
    l = B.meta & 63;
    const int c = (B.meta >> 6) & 3, e0 = (B.meta >> 8) & 31, e1 = (B.meta >> 13) & 31;
    const uint32_t f = o & ((1u << e0) - 1u);
    const uint32_t sc = (o >> e0) & ((1u << e1) - 1u);
    const uint32_t t = o >> (e0 + e1);
    return read_id(G, I, l, c, B.base + f + sc * G.st1[l][c] + t * G.st2[l][c]);
}

// one warp-aggregated contribution of cube node `id` at level l
template <bool FP, typename AT>
__device__ __forceinline__ void accumulate(const PushArgs& P, const Hist<FP>& H, bool valid, uint32_t id, int l) {
    const uint64_t key = valid ? ((uint64_t)l << 32 | id) : ~0ull;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    const int lane = threadIdx.x & 31;
    if (!valid || lane != __ffs(peers) - 1) return;
    const uint32_t W = (uint32_t)__popc(peers) << (3 * l);
    if (id < P.S) {
        H.add_int(id, W);
        return;
    }
    push_one<FP, AT>(P, H, id, W);
}

template <bool FP>
__device__ __forceinline__ Hist<FP> carve(uint8_t* smem, uint32_t S, uint32_t* ntouched) {
    Hist<FP> H;
    H.h = reinterpret_cast<uint32_t*>(smem);
    H.hf = FP ? reinterpret_cast<float*>(H.h + S) : nullptr;
    H.touched = reinterpret_cast<uint16_t*>(FP ? reinterpret_cast<uint8_t*>(H.hf + S)
                                               : reinterpret_cast<uint8_t*>(H.h + S));
    H.ntouched = ntouched;
    H.track = S > kScanFlushMax;
    return H;
}

template <bool FP>
__device__ __forceinline__ void flush(const Hist<FP>& H, uint32_t S, int64_t q, uint32_t* __restrict__ acc,
                                      float* __restrict__ accf) {
    // With the fp32 push a bin can be listed twice (once when its integer part
    // and once when its fractional part became non-zero), so bins are read and
    // cleared in one atomic step: the second reader sees zero.
    if (!H.track) {
        for (uint32_t s = threadIdx.x; s < S; s += blockDim.x) {
            const uint32_t v = H.h[s];
            if (v) {
                H.h[s] = 0;
                atomicAdd(acc + q * S + s, v);
            }
            if constexpr (FP) {
                const float f = H.hf[s];
                if (f != 0.f) {
                    H.hf[s] = 0.f;
                    atomicAdd(accf + q * S + s, f);
                }
            }
        }
        return;
    }
    const uint32_t n = *H.ntouched;
    for (uint32_t t = threadIdx.x; t < n; t += blockDim.x) {
        const uint32_t s = H.touched[t];
        const uint32_t v = FP ? atomicExch(H.h + s, 0u) : H.h[s];
        if (!FP) H.h[s] = 0;
        if (v) atomicAdd(acc + q * S + s, v);
        if constexpr (FP) {
            const float f = atomicExch(H.hf + s, 0.f);
            if (f != 0.f) atomicAdd(accf + q * S + s, f);
        }
    }
}

struct MainArgs {
    Geom G;
    Ids I;
    PushArgs P;
    const Blk* blk;
    const uint64_t* blk_off;
    const uint64_t* ncube;
    const uint64_t* chunk_off;
    const uint32_t* chunk_q;     // box of every chunk
    const uint32_t* chunk_b;     // block holding every chunk's first cube
    unsigned long long total_chunks;
    bool planned;                // by the fused kernel (lim holds its batch size and capacities)
    Lim lim;
    uint64_t* clean;             // its words to zero, but for [1], this kernel's ticket
    uint32_t clean_words;
    int64_t Q;
    uint32_t chunk;
    unsigned long long* ticket;
    uint32_t* acc;
    float* accf;
    void* const* io;             // plans: io[1] is the output (acc for u32, accf for fp32)
    uint32_t qcap;               // entries of each warp's push queue (set by launch_main)
};

// the output a main kernel accumulates into: fixed, or (plans) the caller's
// buffer named in the plan's io slots
template <bool FP>
__device__ __forceinline__ void main_out(const MainArgs& A, uint32_t*& acc, float*& accf) {
    acc = A.acc;
    accf = A.accf;
    if (A.io) {
        if constexpr (FP) accf = static_cast<float*>(A.io[1]);
        else acc = static_cast<uint32_t*>(A.io[1]);
    }
}

// A warp's pending internal-node pushes: the unit loop appends (node, weight)
// to a queue in shared memory, and the queue is pushed 32 entries at a time
// (a measured alternative that summed the entries of one node in a hash
// table first was slower on every workload: its probes cost more than the
// expansions it saved).
// The queue is drained once it holds 32 entries; a step of the unit loop can
// add up to 8 per lane, and an entry that finds the queue full is pushed by
// its own lane at once (divergent, slower).  The launch takes the long queue
// unless a short one fits more CTAs on an SM: the loop is bound by load
// latency, so resident warps count for more where shared memory limits them.
constexpr uint32_t kQueueLong = 320, kQueueShort = 64;   // entries
constexpr size_t queue_bytes(uint32_t cap) { return (size_t)cap * 8 + 16; }   // nodes, weights, counter
constexpr size_t kMaxDynSmem = 227 * 1024;   // shared memory of one CTA at most
// dynamic shared memory of the batched kernels at most: 256 bytes are left for
// the static variables of query_batched_kernel
constexpr size_t kMaxMainSmem = kMaxDynSmem - 256;

// chunks of the launch: known on the host, or (planned by the fused kernel) read
// on the device, zero when the batch overflows the plan's buffers; the fused
// kernel's words are left zero for its next launch
__device__ __forceinline__ unsigned long long main_total(const MainArgs& A) {
    if (!A.planned) return A.total_chunks;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < A.clean_words; i += gridDim.x * blockDim.x)
        if (i != 1) A.clean[i] = 0;
    const int64_t Qe = live_q(A.lim, A.Q);
    const bool over = A.blk_off[Qe] > A.lim.cap_blocks || A.chunk_off[Qe] > A.lim.cap_chunks;
    return over ? 0ull : A.chunk_off[Qe];
}

struct Queue {
    uint32_t* n;       // queued nodes
    uint32_t* w;       // queued weights
    uint32_t* count;   // queued entries
    uint32_t cap;      // room
};

__device__ __forceinline__ Queue carve_queue(uint8_t* p, uint32_t cap) {
    Queue Qu;
    Qu.n = reinterpret_cast<uint32_t*>(p);
    Qu.w = Qu.n + cap;
    Qu.count = Qu.w + cap;
    Qu.cap = cap;
    return Qu;
}

// empty queue (one warp)
__device__ __forceinline__ void clear_queue(const Queue& Qu) {
    if ((threadIdx.x & 31) == 0) *Qu.count = 0u;
    __syncwarp();
}

// push one (node, weight) per lane where `valid`.  With the mixture table each
// lane adds the first two entries of its node's row itself (rows average about
// two entries: two independent loads right after the row header); the rest of
// longer rows is flattened: entry e goes to lane e % 32, which finds its row by
// a binary search over the inclusive sums of the remaining lengths.  Nodes
// without a row (and 16-bit weights) walk their lerp trees.
template <bool FP, typename AT>
__device__ __forceinline__ void push_lanes(const PushArgs& P, const Hist<FP>& H, bool valid, uint32_t n,
                                           uint32_t w) {
    const int lane = threadIdx.x & 31;
    if (std::is_same<AT, float>::value && P.lut_meta) {
        uint32_t off = 0, len = 0, k = 0;
        if (valid) {
            lut_row(P, n, w, off, len, k);
            if (!len) {
                if constexpr (FP) push_frac<AT>(P, H, n, (float)w);
                else push_int<FP>(P, H, n, w);
            }
        }
        __syncwarp();
        if (len) {
            const uint2 e0 = __ldg(P.lut + off);
            const uint2 e1 = len > 1 ? __ldg(P.lut + off + 1) : make_uint2(0u, 0u);
            H.add_int(e0.x, k * e0.y);
            if (len > 1) H.add_int(e1.x, k * e1.y);
            const uint32_t h = len > 1 ? 2u : 1u;
            off += h;
            len -= h;
        }
        if (!__any_sync(0xffffffffu, len != 0u)) {
            __syncwarp();
            return;
        }
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t excl = incl - len;
        for (uint32_t base = 0; base < total; base += 32) {
            const uint32_t e = base + lane;
            int j = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const uint32_t v = __shfl_sync(0xffffffffu, incl, j + step - 1);
                if (v <= e) j += step;
            }
            const uint32_t oj = __shfl_sync(0xffffffffu, off, j);
            const uint32_t kj = __shfl_sync(0xffffffffu, k, j);
            const uint32_t ej = __shfl_sync(0xffffffffu, excl, j);
            if (e < total) {
                const uint2 ent = __ldg(P.lut + oj + (e - ej));
                H.add_int(ent.x, kj * ent.y);
            }
        }
    } else if (valid) {
        if constexpr (FP) push_frac<AT>(P, H, n, (float)w);
        else push_int<FP>(P, H, n, w);
    }
    __syncwarp();
}

// push queued entries 32 at a time until fewer than 32 (none if `all`)
// remain, then move the rest to the front.  Inlined: as a call it made the
// main loop save and restore its live registers around every drain (100,000-box
// batch 5.79 -> 5.48 ms)
template <bool FP, typename AT>
__device__ __forceinline__ void drain(const PushArgs& P, const Hist<FP>& H, const Queue& Qu, bool all) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const uint32_t qc = min(*Qu.count, Qu.cap);   // entries past the end were pushed at once
    uint32_t done = 0;
    while (qc - done >= 32 || (all && qc > done)) {
        const uint32_t take = min(qc - done, 32u);
        const bool v = (uint32_t)lane < take;
        push_lanes<FP, AT>(P, H, v, v ? Qu.n[done + lane] : 0u, v ? Qu.w[done + lane] : 0u);
        done += take;
    }
    const uint32_t rest = qc - done;
    uint32_t tn = 0, tw = 0;
    if ((uint32_t)lane < rest) {
        tn = Qu.n[done + lane];
        tw = Qu.w[done + lane];
    }
    __syncwarp();
    if ((uint32_t)lane < rest) {
        Qu.n[lane] = tn;
        Qu.w[lane] = tw;
    }
    if (lane == 0) *Qu.count = rest;
    __syncwarp();
}

// What a lane needs to read the units of one block.  A warp keeps one of these
// per block of its window in shared memory, so that a unit costs two shared
// loads instead of a shuffle per field and an indexed parameter load per
// stride.
struct __align__(16) Desc {
    uint64_t addr;       // the block's first item
    uint32_t st1, st2;   // strides of its second and third axis, in items
    uint32_t off;        // item of unit u: off + (u << lg)
    uint32_t bits;       // e0 | e1 << 5 | lg << 10 | level << 13
    uint32_t lo, hi;     // its items inside the span
};
constexpr size_t kDescBytes = 32 * sizeof(Desc);   // per warp

// One class's units of a window, numbered through its blocks by a warp scan.
struct Units {
    uint32_t n, incl, total;   // this lane's block's units, their inclusive sum, the window's

    // number the units (n set) and lay out the blocks that have any, in order;
    // false when the window has none
    __device__ __forceinline__ bool number(Desc& D, uint32_t first, uint32_t lg, Desc* desc) {
        const int lane = threadIdx.x & 31;
        const unsigned act = __ballot_sync(0xffffffffu, n != 0u);
        if (!act) return false;
        incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        total = __shfl_sync(0xffffffffu, incl, 31);
        __syncwarp();   // the previous class's units have been read
        if (n) {
            D.off = first - ((incl - n) << lg);
            desc[__popc(act & ((1u << lane) - 1u))] = D;
        }
        __syncwarp();
        return true;
    }

    // place in desc of the block of unit ub + lane: the blocks that end at or
    // before ub, plus those that end inside this group of 32 at or before the
    // unit (blocks with units have distinct ends, so one bit each)
    __device__ __forceinline__ int block(uint32_t ub) const {
        const int lane = threadIdx.x & 31;
        const unsigned below = __ballot_sync(0xffffffffu, n != 0u && incl <= ub);
        const uint32_t te = incl - ub;
        const unsigned ends = __reduce_or_sync(0xffffffffu, n != 0u && incl > ub && te < 32u ? 1u << te : 0u);
        return __popc(below) + __popc(ends & ((2u << lane) - 1u));
    }
};

// index of item o of a block, relative to its first one
__device__ __forceinline__ uint32_t item_at(uint32_t o, uint32_t bits, uint32_t st1, uint32_t st2) {
    const uint32_t e0 = bits & 31u, e1 = (bits >> 5) & 31u;
    return (o & ((1u << e0) - 1u)) + ((o >> e0) & ((1u << e1) - 1u)) * st1 + (o >> (e0 + e1)) * st2;
}

// the words segment | count << 16 of a tile record's or list's block
template <bool FP>
__device__ __forceinline__ void add_words(const Hist<FP>& H, uint4 x) {
    H.add_int(x.x & 0xffffu, x.x >> 16);
    if (x.y) H.add_int(x.y & 0xffffu, x.y >> 16);
    if (x.z) H.add_int(x.z & 0xffffu, x.z >> 16);
    if (x.w) H.add_int(x.w & 0xffffu, x.w >> 16);
}

// a mixture node's cube of level l through the node's record r
template <bool FP, typename AT>
__device__ __forceinline__ void add_record(const PushArgs& P, const Hist<FP>& H, uint4 r, uint32_t node, uint32_t l) {
    if constexpr (!std::is_same<AT, float>::value) {
        // shares of 8^l, a power of two: the products are those of the tree walk
        const float W = (float)(1u << (3 * l));
        if (r.w == kFracPair) {
            H.add_frac(r.x & 0xffffu, W * __uint_as_float(r.y));
            H.add_frac(r.x >> 16, W * __uint_as_float(r.z));
        } else if (r.w == kFracList) {
            for (uint32_t e = 0; e < r.y; e++)
                H.add_frac(__ldg(P.lut + r.x + e).x, W * __ldg(P.frac + r.x + e));
        } else {
            push_one<FP, AT>(P, H, node, 1u << (3 * l));
        }
    } else if (r.x >> 16) {
        // counts of 8^lmin voxels: they sum to that power of two
        const uint32_t sum = (r.x >> 16) + (r.y >> 16) + (r.z >> 16) + (r.w >> 16);
        const uint32_t sh = 3 * l - (31 - __clz(sum));
        H.add_int(r.x & 0xffffu, (r.x >> 16) << sh);
        H.add_int(r.y & 0xffffu, (r.y >> 16) << sh);
        if (r.z) H.add_int(r.z & 0xffffu, (r.z >> 16) << sh);
        if (r.w) H.add_int(r.w & 0xffffu, (r.w >> 16) << sh);
    } else if (r.x == kTileList) {
        const uint32_t sh = 3 * l - r.w;
        for (uint32_t e = 0; e < r.z; e += 2) {
            const uint2 a = __ldg(P.lut + r.y + e);
            const uint2 b = e + 1 < r.z ? __ldg(P.lut + r.y + e + 1) : make_uint2(0u, 0u);
            H.add_int(a.x, a.y << sh);
            if (b.y) H.add_int(b.x, b.y << sh);
        }
    } else {
        push_one<FP, AT>(P, H, node, 1u << (3 * l));
    }
}

// Rows of more entries than this are added by the whole warp: a lane's loop over
// one holds the others up (a cube of level 3 of a volume of noise has 512; 100
// boxes of such a 64^3 volume with 32,768 segments 621 -> 144 us).
constexpr uint32_t kLongRow = 32;
template <typename AT> __device__ __forceinline__ bool long_row(uint4 r) {
    return std::is_same<AT, float>::value ? r.x == kTileList && r.z > kLongRow : r.w == kFracList && r.y > kLongRow;
}

// the long rows among the warp's cubes (record r, zero for none, level l)
template <bool FP, typename AT>
__device__ __forceinline__ void add_long_rows(const PushArgs& P, const Hist<FP>& H, uint4 r, uint32_t l) {
    const int lane = threadIdx.x & 31;
    for (unsigned m = __ballot_sync(0xffffffffu, long_row<AT>(r)); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const uint32_t lj = 3 * __shfl_sync(0xffffffffu, l, j);
        if constexpr (std::is_same<AT, float>::value) {
            const uint32_t first = __shfl_sync(0xffffffffu, r.y, j), n = __shfl_sync(0xffffffffu, r.z, j);
            const uint32_t sh = lj - __shfl_sync(0xffffffffu, r.w, j);
            for (uint32_t e = lane; e < n; e += 32) {
                const uint2 t = __ldg(P.lut + first + e);
                H.add_int(t.x, t.y << sh);
            }
        } else {
            const uint32_t first = __shfl_sync(0xffffffffu, r.x, j), n = __shfl_sync(0xffffffffu, r.y, j);
            const float W = (float)(1u << lj);
            for (uint32_t e = lane; e < n; e += 32) H.add_frac(__ldg(P.lut + first + e).x, W * __ldg(P.frac + first + e));
        }
    }
}

// Items [w0, w1) of one box by one warp, b the block holding item w0.
//
// The span is a flat stream of units.  A window holds the records of 31
// consecutive blocks, one per lane, and their units are taken class by class,
// so that the lanes of a warp do the same work at the same time: tile records,
// vectors of 16 or 8 level-0 IDs of one row (32 or 16 bytes, where rows of
// 2-byte IDs start on 16-byte boundaries and are at least 8 long; Algorithm
// 1's runs start on multiples of their own length, so only the ends of the
// span cut a vector), and single cubes.  No load waits on a block boundary.
// Voxels of one segment extend a per-lane run, added to the histogram when the
// segment changes (in uniform regions the lanes would otherwise meet in one
// bin at every step).
//
// REC: a mixture node's cube reads the node's record (mg_tiles.cu) and adds
// its segments at once, two dependent loads.  Without records (quantised
// graphs, no room for them) the cube is queued for the warp's pushes, equal
// nodes of a step merged.
//
// PAIRS (16-bit weights): a mixture of two segments extends a per-lane run of
// that pair, its two shares summed in registers (fp32 adds to shared memory are
// compare-and-swap loops, and cubes along a surface hold the same two segments).
// Only in the 128-thread instantiation, whose registers it fits: 100,000 boxes
// with 1,182 segments 14.7 -> 12.0 ms; at 256 threads it spills (2,000 boxes
// with 353 segments 189 -> 205 us).
//
// LONG: rows above kLongRow by the whole warp.  Only where a CTA shares a
// histogram: with up to 2,048 segments the rows are shorter and the chunks of
// a warp many, 2 to 12 times faster on noise than the queues without it, and
// the loop has no register to spare.
template <bool FP, typename AT, bool REC, bool PAIRS, bool LONG>
__device__ __forceinline__ void process_span(const MainArgs& A, const Hist<FP>& H, const Queue& Qu, Desc* desc,
                                             uint32_t w0, uint32_t w1, uint64_t b, uint64_t b1, uint32_t ncube) {
    const int lane = threadIdx.x & 31;
    const uint32_t S = A.P.S;
    const bool id16 = A.G.id0_bytes == 2;
    uint32_t rid = kNone, rcnt = 0;
    auto run_add = [&](uint32_t s, uint32_t n) {
        if (s == rid) {
            rcnt += n;
        } else {
            if (rcnt) H.add_int(rid, rcnt);
            rid = s;
            rcnt = n;
        }
    };
    uint32_t pair = 0;   // two different segments, so not 0 in use
    float pa = 0.f, pb = 0.f;
    auto pair_add = [&](uint4 r, float W) {
        const float a = W * __uint_as_float(r.y), c = W * __uint_as_float(r.z);
        if (r.x == pair) {
            pa += a;
            pb += c;
        } else {
            if (pair) {
                H.add_frac(pair & 0xffffu, pa);
                H.add_frac(pair >> 16, pb);
            }
            pair = r.x;
            pa = a;
            pb = c;
        }
    };
    for (uint64_t bb = b;; bb += 31) {
        const uint64_t i = bb + lane;
        uint32_t st = ncube, base = 0, meta = 0;
        if (i < b1) {
            const Blk t = A.blk[i];
            st = t.start;
            base = t.base;
            meta = t.meta;
        }
        const uint32_t nxt = __shfl_down_sync(0xffffffffu, st, 1);
        const uint32_t lo_a = max(st, w0), hi_a = min(nxt, w1);
        const bool use = lane < 31 && lo_a < hi_a;
        const int v = meta & 63, cp = (meta >> 6) & 3;
        const bool tiles = use && v >= MG_MAX_LEVELS;
        const bool vecs = use && v == 0 && id16 && ((meta >> 8) & 31u) >= 3 && (A.G.vec_ok[cp] & 1u);
        const uint32_t vlg = ((meta >> 8) & 31u) >= 4 && (A.G.vec32_ok[cp] & 1u) ? 4 : 3;
        Desc D{};
        if (use) {
            D.lo = lo_a - st;
            D.hi = hi_a - st;
            D.addr = tiles    ? reinterpret_cast<uint64_t>(A.I.tiles + A.G.off[v][cp] + base)
                     : v == 0 ? reinterpret_cast<uint64_t>(A.I.l0[cp]) + ((uint64_t)base << (id16 ? 1 : 2))
                              : reinterpret_cast<uint64_t>(A.I.hi[cp] + A.G.off[v][cp] + base);
            D.st1 = A.G.st1[v][cp];
            D.st2 = A.G.st2[v][cp];
            D.bits = ((meta >> 8) & 1023u) | (vecs ? vlg << 10 : 0u) | (uint32_t)(v & 31) << 13;
        }
        Units U;

        // tile records, two in flight per lane
        U.n = tiles ? D.hi - D.lo : 0u;
        if (U.number(D, D.lo, 0, desc)) {
            for (uint32_t u0 = 0; u0 < U.total; u0 += 64) {
                uint4 x[2];
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const uint32_t u = u0 + 32 * r + lane;
                    const int j = U.block(u0 + 32 * r);
                    x[r] = make_uint4(0u, 0u, 0u, 0u);
                    if (u < U.total) {
                        const Desc& d = desc[j];
                        const uint32_t idx = item_at(d.off + u, d.bits, d.st1, d.st2);
                        x[r] = __ldcs(reinterpret_cast<const uint4*>(d.addr) + idx);
                    }
                }
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    if (x[r].x == kTileList) {
                        const uint4* t = A.I.pool + x[r].y;
                        for (uint32_t k = 0; k < x[r].z; k++) add_words(H, __ldg(t + k));
                    } else if (x[r].y) {
                        add_words(H, x[r]);
                    } else if (x[r].x) {
                        run_add(x[r].x & 0xffffu, x[r].x >> 16);
                    }
                }
            }
        }

        // level-0 vectors
        U.n = vecs ? ((D.hi + (1u << vlg) - 1) >> vlg) - (D.lo >> vlg) : 0u;
        if (U.number(D, D.lo >> vlg << vlg, vlg, desc)) {
            for (uint32_t u0 = 0; u0 < U.total; u0 += 32) {
                const uint32_t u = u0 + lane;
                const int j = U.block(u0);
                if (u < U.total) {
                    const Desc& d = desc[j];
                    const uint32_t lg = (d.bits >> 10) & 7u, o = d.off + (u << lg);
                    const uint4* p = reinterpret_cast<const uint4*>(
                        d.addr + 2ull * item_at(o, d.bits, d.st1, d.st2));
                    // IDs are read once: streaming loads (evict first) leave L2
                    // to the records and table rows
                    const uint4 x = __ldcs(p);
                    uint4 y = x;
                    if (lg == 4) y = __ldcs(p + 1);
                    const uint32_t a = x.x & 0xffffu, pa = a * 0x10001u;
                    const uint32_t m = (x.x ^ pa) | (x.y ^ pa) | (x.z ^ pa) | (x.w ^ pa) | (y.x ^ pa) | (y.y ^ pa) |
                                       (y.z ^ pa) | (y.w ^ pa);
                    const uint32_t k0 = d.lo > o ? d.lo - o : 0u, k1 = min(d.hi - o, 1u << lg);   // IDs of the span
                    if (m == 0u) {
                        run_add(a, k1 - k0);
                    } else {
                        // a segment boundary inside: each ID is added to its
                        // bin at once, independent adds where a run would
                        // chain them
                        const uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                        for (uint32_t q = 0; q < 16; q++)
                            if (q >= k0 && q < k1) H.add_int((w[q >> 1] >> (16 * (q & 1))) & 0xffffu, 1u);
                    }
                }
            }
        }

        // single cubes, R in flight per lane
        constexpr int R = 2;
        U.n = use && !tiles && !vecs ? D.hi - D.lo : 0u;
        if (U.number(D, D.lo, 0, desc)) {
            for (uint32_t u0 = 0; u0 < U.total; u0 += 32 * R) {
                uint32_t id[R], lv[R];
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const uint32_t u = u0 + 32 * r + lane;
                    const int j = U.block(u0 + 32 * r);
                    id[r] = kNone;
                    lv[r] = 0;
                    if (u < U.total) {
                        const Desc& d = desc[j];
                        const uint32_t idx = item_at(d.off + u, d.bits, d.st1, d.st2);
                        lv[r] = d.bits >> 13;
                        id[r] = lv[r] == 0 && id16 ? (uint32_t)__ldcs(reinterpret_cast<const uint16_t*>(d.addr) + idx)
                                                   : __ldcs(reinterpret_cast<const uint32_t*>(d.addr) + idx);
                    }
                }
                if constexpr (REC) {
                    uint4 rec[R];
#pragma unroll
                    for (int r = 0; r < R; r++) {
                        rec[r] = make_uint4(0u, 0u, 0u, 0u);
                        if (id[r] >= S && id[r] != kNone) rec[r] = __ldg(A.P.rec + id[r]);
                    }
#pragma unroll
                    for (int r = 0; r < R; r++) {
                        if (id[r] < S) run_add(id[r], 1u << (3 * lv[r]));
                        else if (id[r] != kNone && !(LONG && long_row<AT>(rec[r]))) {
                            if (PAIRS && rec[r].w == kFracPair) pair_add(rec[r], (float)(1u << (3 * lv[r])));
                            else add_record<FP, AT>(A.P, H, rec[r], id[r], lv[r]);
                        }
                    }
                    if constexpr (LONG) {
#pragma unroll
                        for (int r = 0; r < R; r++) add_long_rows<FP, AT>(A.P, H, rec[r], lv[r]);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < R; r++) {
                        const bool node = id[r] >= S && id[r] != kNone;
                        if (id[r] < S) run_add(id[r], 1u << (3 * lv[r]));
                        // one queue entry for the equal nodes of the step
                        const unsigned peers =
                            __match_any_sync(0xffffffffu, node ? (uint64_t)lv[r] << 32 | id[r] : ~0ull);
                        if (node && lane == __ffs(peers) - 1) {
                            const uint32_t W = (uint32_t)__popc(peers) << (3 * lv[r]);
                            const uint32_t pos = atomicAdd(Qu.count, 1u);
                            if (pos < Qu.cap) {
                                Qu.n[pos] = id[r];
                                Qu.w[pos] = W;
                            } else {
                                push_one<FP, AT>(A.P, H, id[r], W);
                            }
                        }
                    }
                    __syncwarp();
                    if (*Qu.count >= 32) drain<FP, AT>(A.P, H, Qu, false);
                }
            }
        }
        const uint32_t st31 = __shfl_sync(0xffffffffu, st, 31);
        if (bb + 31 >= b1 || st31 >= w1) break;
    }
    if (rcnt) H.add_int(rid, rcnt);
    if constexpr (PAIRS) {
        if (pair) {
            H.add_frac(pair & 0xffffu, pa);
            H.add_frac(pair >> 16, pb);
        }
    }
    __syncwarp();
}

// Few segments: every warp owns a histogram in shared memory and takes whole
// chunks from the global ticket, so warps never wait for each other.
// Register budget by CTA size NT: 256 threads, at most 51 registers (5 CTAs
// per SM); 128 threads, at most 56 (9 CTAs).  The loop is bound by load
// latency, so resident warps count; neither spills.
template <int NT> struct WarpKernelBounds;
template <> struct WarpKernelBounds<128> { static constexpr int min_ctas = 9; };
template <> struct WarpKernelBounds<256> { static constexpr int min_ctas = 5; };

template <bool FP, typename AT, int NT, bool REC>
__global__ void __launch_bounds__(NT, WarpKernelBounds<NT>::min_ctas) query_warp_kernel(
    const __grid_constant__ MainArgs A) {
    constexpr bool kPairs = REC && NT == 128 && !std::is_same<AT, float>::value;
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t S = A.P.S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t S4 = (S + 3) & ~3u;   // a histogram is flushed four bins at a time
    const size_t hist_bytes = (size_t)S4 * 4 * (FP ? 2 : 1);
    Desc* desc = reinterpret_cast<Desc*>(smem + warp * kDescBytes);
    uint8_t* mine = smem + (blockDim.x >> 5) * kDescBytes + warp * (hist_bytes + (REC ? 0 : queue_bytes(A.qcap)));
    Hist<FP> H;
    H.h = reinterpret_cast<uint32_t*>(mine);
    H.hf = FP ? reinterpret_cast<float*>(H.h + S4) : nullptr;
    H.touched = nullptr;
    H.ntouched = nullptr;
    H.track = false;
    const Queue Qu = carve_queue(mine + hist_bytes, A.qcap);
    for (uint32_t i = lane; i < S4; i += 32) {
        H.h[i] = 0;
        if constexpr (FP) H.hf[i] = 0.f;
    }
    if constexpr (!REC) clear_queue(Qu);
    __syncwarp();
    grid_dependency_wait();
    uint32_t* acc;
    float* accf;
    main_out<FP>(A, acc, accf);
    const uint32_t total = (uint32_t)main_total(A);   // (below 2^32: the chunk map's bound)
    // A warp's first chunk is its own number, the ticket hands out the rest.
    // (Taking the next one while the current chunk runs left the last chunks
    // to busy warps: 125 -> 140 us for 10,000 boxes of 512x512x384.)
    const uint32_t all = gridDim.x * (NT / 32);
    uint32_t c = blockIdx.x * (NT / 32) + warp;
    while (c < total) {
        const uint32_t q = __ldg(A.chunk_q + c);
        const uint32_t ncube = (uint32_t)A.ncube[q];
        const uint32_t c0 = (c - (uint32_t)A.chunk_off[q]) * A.chunk;
        const uint32_t c1 = min(c0 + A.chunk, ncube);
        process_span<FP, AT, REC, kPairs, false>(A, H, Qu, desc, c0, c1, __ldg(A.chunk_b + c), A.blk_off[q + 1], ncube);
        if constexpr (!REC) drain<FP, AT>(A.P, H, Qu, true);
        uint32_t* row = acc + (size_t)q * S;
        for (uint32_t s = 4 * lane; s < S4; s += 128) {
            const uint4 v = *reinterpret_cast<const uint4*>(H.h + s);
            if (v.x | v.y | v.z | v.w) {
                *reinterpret_cast<uint4*>(H.h + s) = make_uint4(0u, 0u, 0u, 0u);
                if (v.x) atomicAdd(row + s, v.x);
                if (v.y) atomicAdd(row + s + 1, v.y);
                if (v.z) atomicAdd(row + s + 2, v.z);
                if (v.w) atomicAdd(row + s + 3, v.w);
            }
        }
        if constexpr (FP) {
            for (uint32_t s = lane; s < S; s += 32) {
                const float f = H.hf[s];
                if (f != 0.f) {
                    H.hf[s] = 0.f;
                    atomicAdd(accf + (size_t)q * S + s, f);
                }
            }
        }
        __syncwarp();
        if (total <= all) break;
        if (lane == 0) {   // (compared before the sum, which could pass 2^32)
            const uint32_t t = atomicAdd(reinterpret_cast<uint32_t*>(A.ticket), 1u);
            c = t < total - all ? all + t : total;
        }
        c = __shfl_sync(0xffffffffu, c, 0);
    }
}

// Many segments: one histogram per CTA; the CTA takes a chunk and its warps
// take sub-spans of it (about two each) from a shared counter.
template <bool FP, typename AT, bool REC>
__global__ void __launch_bounds__(512, 2) query_batched_kernel(const __grid_constant__ MainArgs A) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_ntouched;
    __shared__ unsigned long long s_chunk;
    __shared__ uint32_t s_q;
    __shared__ uint32_t s_next;
    const uint32_t S = A.P.S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Desc* desc = reinterpret_cast<Desc*>(smem + warp * kDescBytes);
    const Hist<FP> H = carve<FP>(smem + nw * kDescBytes, S, &s_ntouched);
    // per-warp queues follow the touched list
    const size_t touched_bytes = (size_t)S * 2 * (FP ? 2 : 1);
    uint8_t* qbase = reinterpret_cast<uint8_t*>(H.touched) + ((touched_bytes + 15) & ~(size_t)15);
    const Queue Qu = carve_queue(qbase + warp * queue_bytes(A.qcap), A.qcap);
    for (uint32_t i = threadIdx.x; i < S; i += blockDim.x) {
        H.h[i] = 0;
        if constexpr (FP) H.hf[i] = 0.f;
    }
    if (threadIdx.x == 0) s_ntouched = 0;
    if constexpr (!REC) clear_queue(Qu);
    grid_dependency_wait();
    uint32_t* acc;
    float* accf;
    main_out<FP>(A, acc, accf);
    const unsigned long long total = main_total(A);
    for (bool own = true;; own = false) {   // a CTA's first chunk is its own number
        if (threadIdx.x == 0) {
            const unsigned long long c = own ? blockIdx.x : gridDim.x + atomicAdd(A.ticket, 1ull);
            s_chunk = c;
            s_next = 0;
            if (c < total) s_q = A.chunk_q[c];
        }
        __syncthreads();
        const unsigned long long c = s_chunk;
        if (c >= total) break;
        const uint32_t q = s_q;
        const uint32_t ncube = (uint32_t)A.ncube[q];
        const uint32_t c0 = (uint32_t)(c - A.chunk_off[q]) * A.chunk;
        const uint32_t c1 = min(c0 + A.chunk, ncube);
        const uint64_t b1 = A.blk_off[q + 1];
        const uint32_t sub = max(32u, (((c1 - c0) + 2 * nw - 1) / (2 * nw) + 31) & ~31u);
        uint64_t bhint = __ldg(A.chunk_b + c);   // a warp's sub-spans only move forward
        for (;;) {
            uint32_t k = 0;
            if (lane == 0) k = atomicAdd(&s_next, 1u);
            k = __shfl_sync(0xffffffffu, k, 0);
            if ((uint64_t)k * sub >= (uint64_t)(c1 - c0)) break;
            const uint32_t w0 = c0 + k * sub;
            const uint32_t w1 = min(w0 + sub, c1);
            uint64_t b = bhint;
            if (lane == 0) {   // block of the sub-span's first cube
                uint64_t lo = bhint, hi = b1;   // blk[lo].start <= w0 < blk[hi].start
                while (hi - lo > 1) {
                    const uint64_t mid = (lo + hi) >> 1;
                    if (__ldg(&A.blk[mid].start) <= w0) lo = mid;
                    else hi = mid;
                }
                b = lo;
            }
            b = __shfl_sync(0xffffffffu, b, 0);
            bhint = b;
            process_span<FP, AT, REC, false, true>(A, H, Qu, desc, w0, w1, b, b1, ncube);
        }
        if constexpr (!REC) drain<FP, AT>(A.P, H, Qu, true);
        __syncthreads();
        flush<FP>(H, S, q, acc, accf);
        __syncthreads();
        if (threadIdx.x == 0) s_ntouched = 0;
    }
}

// Baseline (MG_SCHED_PLAIN): one launch per box, unbatched.  The launch has
// as many CTAs as the box's footprint needs (about 4,096 cubes each, at most
// a few per SM); CTA b walks the blocks in order and counts cubes
// [b * per_cta, (b + 1) * per_cta) of the box into its shared histogram, then
// adds it to the box's row.
template <bool FP, typename AT>
__global__ void __launch_bounds__(256) query_plain_kernel(MainArgs A, const int32_t* __restrict__ boxes, int64_t q,
                                                          uint32_t per_cta) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_ntouched;
    __shared__ Runs R;
    const uint32_t S = A.P.S;
    const Hist<FP> H = carve<FP>(smem, S, &s_ntouched);
    for (uint32_t i = threadIdx.x; i < S; i += blockDim.x) {
        H.h[i] = 0;
        if constexpr (FP) H.hf[i] = 0.f;
    }
    int32_t b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
    if (!box_ok(b, A.G)) {
        if (threadIdx.x == 0 && blockIdx.x == 0) set_status(A.P.status, kStatBadInput);
        return;
    }
    if (threadIdx.x == 0) {
        s_ntouched = 0;
        make_runs(b, A.G, R);
    }
    __syncthreads();
    const uint64_t c0 = (uint64_t)blockIdx.x * per_cta, c1 = c0 + per_cta;
    uint64_t start = 0;
    for (int k = 0; k < R.nz && start < c1; k++)
        for (int j = 0; j < R.ny && start < c1; j++)
            for (int i = 0; i < R.nx && start < c1; i++) {
                const uint32_t n = block_cubes(R.lx[i], R.ly[j], R.lz[k]);
                const uint64_t lo = max(start, c0), hi = min(start + n, c1);
                if (lo < hi) {
                    const Blk B = make_blk(A.G, 0, R.sx[i], R.sy[j], R.sz[k], R.lx[i], R.ly[j], R.lz[k], 0);
                    for (uint64_t base = lo - start; base < hi - start; base += blockDim.x) {
                        const uint32_t o = (uint32_t)base + threadIdx.x;
                        const bool valid = o < hi - start;
                        uint32_t id = 0;
                        int lv = 0;
                        if (valid) id = cube_node(A.G, A.I, B, o, lv);
                        accumulate<FP, AT>(A.P, H, valid, id, lv);
                    }
                }
                start += n;
            }
    __syncthreads();
    flush<FP>(H, S, q, A.acc, A.accf);
}

// Baseline (MG_SCHED_NAIVE): no footprint assembly, every level-0 voxel of
// the clipped box counted.  A box is read in the level-0 copy whose fastest
// axis is its longest side, so its rows are as long as its shape allows.  Its
// rows are cut into slabs of about kNaiveSlab voxels, taken from a global
// ticket by persistent CTAs; each CTA counts its slab into a shared histogram
// and adds it to the box's row.  A slab is one flat stream of (row, vector)
// slots, the 16-byte vectors (8 uint16 or 4 uint32 IDs) that its rows touch;
// each thread takes four consecutive slots per step (64 contiguous bytes) and
// keeps one run of equal IDs across them; a vector that is not uniform (or is
// cut by the row's ends) adds its in-row IDs one by one.  At most 51 registers
// (five CTAs of 256 threads per SM): the loop is bound by loads in flight
// (1,000 boxes of the 100,000-box recipe: 2.75 ms at 74 registers, 2.30 ms at
// 64, 2.13 ms at 51).
constexpr uint32_t kNaiveSlab = 1u << 16;

// the clipped box in the axis order of the copy it is read from: row length
// L along the copy's fastest axis, n1 rows along the second, n2 along the third
struct NaiveBox {
    int c;
    uint32_t L, n1, n2;
    uint32_t o0, o1, o2;   // origin in the copy's axis order
};
__device__ __forceinline__ NaiveBox naive_box(const int32_t* b, const Geom& G) {
    const uint32_t dx = (uint32_t)(min((int64_t)b[0] + b[3], (int64_t)G.dims[0][0]) - b[0]);
    const uint32_t dy = (uint32_t)(min((int64_t)b[1] + b[4], (int64_t)G.dims[0][1]) - b[1]);
    const uint32_t dz = (uint32_t)(min((int64_t)b[2] + b[5], (int64_t)G.dims[0][2]) - b[2]);
    NaiveBox B;
    if (dx >= dy && dx >= dz) {
        B = NaiveBox{0, dx, dy, dz, (uint32_t)b[0], (uint32_t)b[1], (uint32_t)b[2]};
    } else if (dy >= dz) {
        B = NaiveBox{1, dy, dz, dx, (uint32_t)b[1], (uint32_t)b[2], (uint32_t)b[0]};
    } else {
        B = NaiveBox{2, dz, dx, dy, (uint32_t)b[2], (uint32_t)b[0], (uint32_t)b[1]};
    }
    return B;
}
__device__ __forceinline__ uint32_t naive_rows_per(const NaiveBox& B) { return max(1u, kNaiveSlab / B.L); }

// slabs of every box (0 for a malformed box, whose row stays zero)
__global__ void naive_count_kernel(Geom G, const int32_t* __restrict__ boxes, int64_t Q, uint64_t* __restrict__ items,
                                   unsigned* __restrict__ status) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= Q) return;
    int32_t b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
    if (!box_ok(b, G)) {
        set_status(status, kStatBadInput);
        items[q] = 0;
        return;
    }
    const NaiveBox B = naive_box(b, G);
    const uint64_t rows = (uint64_t)B.n1 * B.n2, per = naive_rows_per(B);
    items[q] = (rows + per - 1) / per;
}

template <bool FP, typename T>
__global__ void __launch_bounds__(256, 5) query_naive_kernel(Geom G, Ids I, const int32_t* __restrict__ boxes, int64_t Q,
                                                          const uint64_t* __restrict__ item_off,
                                                          unsigned long long* __restrict__ ticket,
                                                          uint32_t* __restrict__ acc, float* __restrict__ accf) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ unsigned long long s_item;
    uint32_t* h = reinterpret_cast<uint32_t*>(smem);
    const uint32_t S = G.S;
    constexpr int E = 16 / (int)sizeof(T);   // IDs per 16-byte vector
    const unsigned long long total = item_off[Q];
    for (uint32_t i = threadIdx.x; i < S; i += blockDim.x) h[i] = 0;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(ticket, 1ull);
        __syncthreads();
        const unsigned long long w = s_item;
        if (w >= total) break;
        int64_t lo = 0, hi = Q;   // item_off[lo] <= w < item_off[hi]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if (item_off[mid] <= w) lo = mid;
            else hi = mid;
        }
        const int64_t q = lo;
        int32_t b[6];
#pragma unroll
        for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
        const NaiveBox B = naive_box(b, G);
        const int c = B.c;
        const T* ids = static_cast<const T*>(I.l0[c]);
        const uint64_t st1 = G.st1[0][c], st2 = G.st2[0][c];
        const int third = c == 0 ? 2 : c == 1 ? 0 : 1;   // the copy's third axis
        const uint64_t V0 = st2 * (uint64_t)G.dims[0][third];   // IDs in the copy's array
        const uint32_t per = naive_rows_per(B);
        const uint32_t r0 = (uint32_t)(w - item_off[q]) * per;
        const uint32_t r1 = (uint32_t)min((uint64_t)r0 + per, (uint64_t)B.n1 * B.n2);
        const uint32_t vpr = (B.L + E - 1) / E + 1;   // vectors a row of L IDs can touch
        const uint32_t nf = (r1 - r0) * vpr;          // <= 2^16 / E + 2^17, or one row of a longer box
        uint32_t rid = kNone, rcnt = 0;
        auto flush_run = [&]() {
            if (rcnt) atomicAdd(h + rid, rcnt);
        };
        for (uint32_t f0 = 4u * threadIdx.x; f0 < nf; f0 += 4u * blockDim.x) {
            // the first slot's row and vector; the others follow
            uint32_t row = f0 / vpr, vi = f0 - row * vpr;
            uint64_t e0 = 0;
            uint32_t rrow = kNone;
            uint4 u[4];
            uint64_t p0s[4], e0s[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                u[j] = make_uint4(0u, 0u, 0u, 0u);
                p0s[j] = ~0ull;
                e0s[j] = 0;
                if (f0 + j < nf) {
                    if (row != rrow) {
                        const uint32_t r = r0 + row, a2 = r / B.n1, a1 = r - a2 * B.n1;
                        e0 = (uint64_t)(B.o2 + a2) * st2 + (uint64_t)(B.o1 + a1) * st1 + B.o0;
                        rrow = row;
                    }
                    const uint64_t v = e0 / E + vi;
                    if (v * E < e0 + B.L) {
                        e0s[j] = e0;
                        p0s[j] = v * E;
                        if ((v + 1) * E <= V0) {
                            u[j] = __ldcs(reinterpret_cast<const uint4*>(ids) + v);
                        } else {   // the array's last vector, cut at its end
                            T* x = reinterpret_cast<T*>(&u[j]);
                            for (int k = 0; k < E && v * E + k < V0; k++) x[k] = __ldg(ids + v * E + k);
                        }
                    }
                }
                if (++vi == vpr) {
                    vi = 0;
                    row++;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint64_t p0 = p0s[j], e0j = e0s[j], e1 = e0j + B.L;
                if (p0 == ~0ull) continue;
                const uint4 x = u[j];
                uint32_t a, d;
                if (E == 8) {
                    a = x.x & 0xffffu;
                    const uint32_t pr = a * 0x10001u;
                    d = (x.x ^ pr) | (x.y ^ pr) | (x.z ^ pr) | (x.w ^ pr);
                } else {
                    a = x.x;
                    d = (x.y ^ a) | (x.z ^ a) | (x.w ^ a);
                }
                if (d == 0u && p0 >= e0j && p0 + E <= e1) {
                    if (rcnt && rid == a) {
                        rcnt += E;
                    } else {
                        flush_run();
                        rid = a;
                        rcnt = E;
                    }
                    continue;
                }
                // a mixed vector, or the cut end of a row: every in-row ID is
                // added to its bin at once (independent adds, no run chain)
                const int k0 = p0 < e0j ? (int)(e0j - p0) : 0;
                const int k1 = p0 + E > e1 ? (int)(e1 - p0) : E;
                const T* xs = reinterpret_cast<const T*>(&x);
#pragma unroll
                for (int k = 0; k < E; k++)
                    if (k >= k0 && k < k1) atomicAdd(h + (uint32_t)xs[k], 1u);
            }
        }
        flush_run();
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < S; i += blockDim.x) {
            const uint32_t cnt = h[i];
            if (cnt) {
                h[i] = 0;
                if (FP) atomicAdd(accf + q * S + i, (float)cnt);
                else atomicAdd(acc + q * S + i, cnt);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// finalisation
// ---------------------------------------------------------------------------
__global__ void dense_f32_rows_kernel(const uint32_t* __restrict__ acc, void* const* __restrict__ io,
                                      const int64_t* __restrict__ Qd, int64_t S) {
    float* out = static_cast<float*>(io[1]);
    const int64_t n = *Qd * S;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)acc[i] + out[i];
}

__global__ void dense_f32_kernel(const uint32_t* __restrict__ acc, float* __restrict__ out, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)acc[i] + out[i];
}

template <bool FP>
__global__ void csr_count_kernel(const uint32_t* __restrict__ acc, const float* __restrict__ accf, int64_t Q,
                                 uint32_t S, uint64_t* __restrict__ cnt) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= Q) return;
    uint64_t c = 0;
    for (uint32_t s = lane; s < S; s += 32) {
        bool nz = acc[q * S + s] != 0;
        if constexpr (FP) nz = nz || accf[q * S + s] != 0.f;
        c += nz;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[q] = c;
}

template <bool FP>
__global__ void csr_write_kernel(const uint32_t* __restrict__ acc, const float* __restrict__ accf, int64_t Q,
                                 uint32_t S, const uint64_t* __restrict__ off, uint32_t* __restrict__ seg,
                                 void* __restrict__ out) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= Q) return;
    uint64_t pos = off[q];
    for (uint32_t sb = 0; sb < S; sb += 32) {
        const uint32_t s = sb + lane;
        uint32_t v = 0;
        float f = 0.f;
        bool nz = false;
        if (s < S) {
            v = acc[q * S + s];
            nz = v != 0;
            if constexpr (FP) {
                f = accf[q * S + s];
                nz = nz || f != 0.f;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, nz);
        if (nz) {
            const uint64_t o = pos + __popc(m & ((1u << lane) - 1u));
            seg[o] = s;
            if constexpr (FP) static_cast<float*>(out)[o] = (float)v + f;
            else static_cast<uint32_t*>(out)[o] = v;
        }
        pos += __popc(m);
    }
}

// box and first block of every chunk
// Exclusive scans of the per-box block and chunk counts for batches of up to
// kFusedScanMax boxes in one CTA: offsets[q] and the totals at [Q]; for plans
// the capacity check of the batch (entries past the live batch are zero).
constexpr int kScanThreads = 1024;
constexpr int64_t kFusedScanMax = 1 << 18;

__global__ void __launch_bounds__(kScanThreads) plan_scan_kernel(const uint32_t* __restrict__ nblk,
                                                                 const uint64_t* __restrict__ nchunk, int64_t Q,
                                                                 uint64_t* __restrict__ blk_off,
                                                                 uint64_t* __restrict__ chunk_off) {
    __shared__ unsigned long long sb[32], sc[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long carry_b = 0, carry_c = 0;
    // tiles of kScanThreads consecutive boxes, one per thread (coalesced)
    for (int64_t t0 = 0; t0 < Q; t0 += kScanThreads) {
        const int64_t i = t0 + t;
        const unsigned long long xb = i < Q ? nblk[i] : 0ull, xc = i < Q ? nchunk[i] : 0ull;
        unsigned long long ib = xb, ic = xc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long yb = __shfl_up_sync(0xffffffffu, ib, o);
            const unsigned long long yc = __shfl_up_sync(0xffffffffu, ic, o);
            if (lane >= o) {
                ib += yb;
                ic += yc;
            }
        }
        if (lane == 31) {
            sb[warp] = ib;
            sc[warp] = ic;
        }
        __syncthreads();
        if (warp == 0) {
            unsigned long long wb = sb[lane], wc = sc[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long yb = __shfl_up_sync(0xffffffffu, wb, o);
                const unsigned long long yc = __shfl_up_sync(0xffffffffu, wc, o);
                if (lane >= o) {
                    wb += yb;
                    wc += yc;
                }
            }
            sb[lane] = wb;
            sc[lane] = wc;
        }
        __syncthreads();
        const unsigned long long pb = warp ? sb[warp - 1] : 0ull, pc = warp ? sc[warp - 1] : 0ull;
        if (i < Q) {
            blk_off[i] = carry_b + pb + ib - xb;
            chunk_off[i] = carry_c + pc + ic - xc;
        }
        carry_b += sb[31];
        carry_c += sc[31];
        __syncthreads();
    }
    if (t == 0) {
        blk_off[Q] = carry_b;
        chunk_off[Q] = carry_c;
    }
}

__global__ void widen_kernel(const uint32_t* __restrict__ a, uint64_t* __restrict__ b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = a[i];
}

int sm_count(int dev) {
    static std::mutex mu;
    static std::vector<int> cache;
    std::lock_guard<std::mutex> lk(mu);
    if ((int)cache.size() <= dev) cache.resize(dev + 1, 0);
    if (!cache[dev]) cudaDeviceGetAttribute(&cache[dev], cudaDevAttrMultiProcessorCount, dev);
    return cache[dev] ? cache[dev] : 1;
}

// Whether a CTA's warps have a histogram each (few segments) or share one.
bool warp_hists(const mg_graph* g, bool FP, int threads) {
    const size_t hist = (size_t)g->S * 4 * (FP ? 2 : 1);
    return g->S <= kWarpHistMax && threads <= 256 && (hist + queue_bytes(kQueueShort)) * (threads / 32) <= 96 * 1024;
}

// Items per work chunk of an untuned batch of Q boxes.  A batch is bound by the
// latency of its longest chunk (one warp walks it alone, or a CTA whose warps
// share a histogram) until it holds enough chunks to fill the GPU, then by what
// each chunk costs beyond its items (descriptors, the flush).  The best length
// grows with the square root of Q, and more slowly with the area of the volume's
// sides, which a box's items follow.  us of a plan run at 128 / 256 / 512 /
// 1,024 / 2,048 items, the rule's choice in brackets, uint32 counts:
//   64^3, 64 segments: 1,000 boxes [24] / 26 / 32 / 41 / 52; 10,000 boxes
//     55 / [50] / 48 / 55 / 67; 30,000 boxes 135 / 108 / [101] / 101 / 113
//   251x187x113, 90 segments: 777 boxes [31] / 32 / 36 / 46 / 58; 10,000 boxes
//     113 / 87 / [77] / 83 / 96
//   512x512x384, 353 segments: 100 boxes [23] / 26 / 31 / 39 / 55; 1,000 boxes
//     42 / [40] / 46 / 65 / 86; 10,000 boxes 212 / 150 / [127] / 127 / 134
//   2048x2048x300, 1,182 segments: 1,000 boxes 57 / [49] / 52 / 58 / 85; 10,000
//     boxes 377 / 255 / 197 / [181] / 190; 100,000 boxes - / - / - / 1472 / [1328]
//   614x961x600, 15,917 segments, a histogram per CTA: 10 boxes 33 / [33] / 35 /
//     41 / 53; 100 boxes 76 / 59 / [52] / 50 / 63; 1,000 boxes - / - / 311 /
//     250 / [229]
// fp32 histograms flush two bins a segment: a third longer (2048x2048x300,
// 10,000 boxes: - / - / 335 / 289 / [283]).  With 16-bit weights a chunk's items
// touch more bins too: longer in proportion above 750 segments, and at least one
// item per five segments in a warp's (1,182 segments: 100 boxes 64 / [52] / 58 /
// 85 / 108, 1,000 boxes 337 / 241 / 194 / [186] / 197; 64^3, 10,000 boxes 77 /
// [77] / 86 / 98 / 134).
constexpr uint32_t kDefaultChunk = 2048, kMinChunk = 128, kMinSharedChunk = 256;
double ideal_chunk(const mg_graph* g, bool FP, mg_dtype weights, bool own, int64_t Q) {
    const double x = g->geom.dims[0][0], y = g->geom.dims[0][1], z = g->geom.dims[0][2];
    const double per = !own ? (FP ? 3.6 : 2.0) : !FP ? 0.33 : weights == MG_F32 ? 0.45 : 0.45 * std::max(1.0, g->S / 750.0);
    return per * std::sqrt((double)Q * std::sqrt(x * y + y * z + z * x));
}
uint32_t default_chunk(const mg_graph* g, bool FP, mg_dtype weights, int threads, int64_t Q) {
    const bool own = warp_hists(g, FP, threads);
    const double best = ideal_chunk(g, FP, weights, own, Q);
    const uint32_t least = !own                ? kMinSharedChunk
                           : weights == MG_F32 ? kMinChunk
                                               : std::max(kMinChunk, g->S / 5);
    uint32_t c = kDefaultChunk;
    while (c / 2 >= least && c > best) c /= 2;
    return c;
}

// Most blocks and work chunks that Q boxes of the volume can have.  An axis of
// d voxels splits into at most 2 ceil(log2(d + 1)) runs, two of each level; the
// cubes of level l whose thickness lies on an axis are at most 2 (area across
// it) / 4^l, so a footprint holds at most 8/3 of the three areas.
uint64_t block_bound(const mg_graph* g, int64_t Q) {
    uint64_t n = (uint64_t)Q;
    for (int k = 0; k < 3; k++) {
        int bits = 0;
        while ((g->geom.dims[0][k] >> bits) > 0) bits++;
        n *= 2 * (uint64_t)bits;
    }
    return n;
}
uint64_t chunk_bound(const mg_graph* g, int64_t Q, uint32_t chunk) {
    const uint64_t x = g->geom.dims[0][0], y = g->geom.dims[0][1], z = g->geom.dims[0][2];
    return (uint64_t)Q * ((3 * (x * y + y * z + z * x)) / chunk + 1);
}

template <typename K>
mg_status prepare_kernel(K kernel, size_t smem) {
    MG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return MG_OK;
}

size_t hist_smem(uint32_t S, bool FP) {   // histogram and touched list of a CTA
    const size_t touched = (size_t)S * 2 * (FP ? 2 : 1);
    return (size_t)S * 4 * (FP ? 2 : 1) + ((touched + 15) & ~(size_t)15) + 16;
}

// the batched kernel for a graph and a CTA size
struct MainShape {
    void (*k)(const MainArgs) = nullptr;
    int threads = 0, full = 0;     // CTAs that fill the GPU
    int chunks_per_cta = 1;        // chunks a CTA works on at a time
    size_t smem = 0;
    uint32_t qcap = 0;
};

template <bool FP, typename AT>
mg_status main_shape(const mg_graph* g, bool rec, int threads, MainShape* out) {
    // few segments: a private histogram per warp; else one per CTA (smem
    // is then the histogram's part); the warps' block descriptors and, without
    // node records, their queues come on top
    int warps = threads / 32;
    const size_t smem = hist_smem(g->S, FP);
    const size_t hist_s = (size_t)((g->S + 3) & ~3u) * 4 * (FP ? 2 : 1);
    const bool warp_mode = warp_hists(g, FP, threads);
    auto k = !warp_mode       ? (rec ? query_batched_kernel<FP, AT, true> : query_batched_kernel<FP, AT, false>)
             : threads <= 128 ? (rec ? query_warp_kernel<FP, AT, 128, true> : query_warp_kernel<FP, AT, 128, false>)
                              : (rec ? query_warp_kernel<FP, AT, 256, true> : query_warp_kernel<FP, AT, 256, false>);
    auto smem_for = [&](uint32_t cap) {
        const size_t each = kDescBytes + (rec ? 0 : queue_bytes(cap));
        return warp_mode ? (hist_s + each) * warps : smem + warps * each;
    };
    int per_sm = 0, per_long = 0;
    if (!warp_mode) {
        // the shape asked for has to fit with its queues alone; the descriptors
        // of the last few segment counts that do take fewer warps
        if (smem + warps * queue_bytes(kQueueShort) > kMaxDynSmem)
            return fail(MG_ERR_UNSUPPORTED, "query kernel does not fit on an SM");
        while (warps > 1 && smem_for(kQueueShort) > kMaxMainSmem) warps /= 2;
        threads = warps * 32;
    }
    // one limit for every launch of the kernel, the most that any shape asks
    // for: callers of several shapes never lower each other's
    MG_TRY(prepare_kernel(k, kMaxMainSmem));
    MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem_for(kQueueShort)));
    if (per_sm < 1) return fail(MG_ERR_UNSUPPORTED, "query kernel does not fit on an SM");
    if (!rec && smem_for(kQueueLong) <= kMaxMainSmem)
        MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_long, k, threads, smem_for(kQueueLong)));
    out->k = k;
    out->threads = threads;
    out->full = per_sm * sm_count(g->device);
    out->chunks_per_cta = warp_mode ? warps : 1;
    out->qcap = per_long >= per_sm ? kQueueLong : kQueueShort;
    out->smem = smem_for(out->qcap);
    return MG_OK;
}

// pdl: with programmatic stream serialisation (its CTAs start while the plan
// kernel finishes and wait for it on the device)
mg_status launch_shape(const mg_graph* g, const MainArgs& A, const MainShape& M, cudaStream_t s, bool pdl) {
    MainArgs A2 = A;
    A2.qcap = M.qcap;
    // no more CTAs than chunks the batch can have
    const uint64_t most = chunk_bound(g, A.Q, A.chunk);
    const unsigned grid = (unsigned)std::min<uint64_t>(M.full, (most + M.chunks_per_cta - 1) / M.chunks_per_cta);
    if (!pdl) {
        M.k<<<grid, M.threads, M.smem, s>>>(A2);
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)M.threads);
    cfg.dynamicSmemBytes = M.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    MG_CUDA(cudaLaunchKernelEx(&cfg, M.k, A2));
    return MG_OK;
}

template <bool FP, typename AT>
mg_status launch_main(const mg_graph* g, const MainArgs& A, const mg_query_opts& o, const int32_t* boxes,
                      size_t smem, int threads, cudaStream_t s, const Alloc* scratch) {
    if (o.schedule == MG_SCHED_NAIVE) {
        // slabs per box, their offsets, then one persistent launch
        if (!scratch) return fail(MG_ERR_INVALID_ARG, "naive schedule without scratch");
        Buf items, off, ticket;
        MG_TRY(items.alloc(scratch, (size_t)A.Q * 8, s));
        MG_TRY(off.alloc(scratch, (size_t)(A.Q + 1) * 8, s));
        MG_TRY(ticket.alloc(scratch, 8, s));
        naive_count_kernel<<<grid_for(A.Q, 256), 256, 0, s>>>(A.G, boxes, A.Q, items.as<uint64_t>(), A.P.status);
        MG_CUDA(cudaGetLastError());
        MG_TRY(scan_exclusive_u64(items.as<uint64_t>(), off.as<uint64_t>(), A.Q, off.as<uint64_t>() + A.Q, *scratch,
                                  s));
        MG_CUDA(cudaMemsetAsync(ticket.p, 0, 8, s));
        const size_t sm = (size_t)g->S * 4;
        auto launch = [&](auto k) -> mg_status {
            MG_TRY(prepare_kernel(k, sm));
            int per_sm = 0;
            MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, sm));
            const int grid = std::max(per_sm, 1) * sm_count(g->device);
            k<<<grid, 256, sm, s>>>(A.G, A.I, boxes, A.Q, off.as<uint64_t>(), ticket.as<unsigned long long>(), A.acc,
                                    A.accf);
            MG_CUDA(cudaGetLastError());
            return MG_OK;
        };
        if (g->id0_bytes == 2) return launch(&query_naive_kernel<FP, uint16_t>);
        return launch(&query_naive_kernel<FP, uint32_t>);
    }
    if (o.schedule == MG_SCHED_PLAIN) {
        // footprint cubes of every box, read back to size each box's launch
        if (!scratch) return fail(MG_ERR_INVALID_ARG, "plain schedule without scratch");
        Buf cubes;
        MG_TRY(cubes.alloc(scratch, (size_t)A.Q * 8, s));
        plan_count_kernel<<<grid_for(A.Q * 32, kPlanThreads), kPlanThreads, 0, s>>>(
            A.G, boxes, A.Q, 1, nullptr, cubes.as<uint64_t>(), nullptr, A.P.status, false);
        MG_CUDA(cudaGetLastError());
        std::vector<uint64_t> nc((size_t)A.Q);
        MG_CUDA(cudaMemcpyAsync(nc.data(), cubes.p, (size_t)A.Q * 8, cudaMemcpyDeviceToHost, s));
        MG_CUDA(cudaStreamSynchronize(s));
        auto k = query_plain_kernel<FP, AT>;
        MG_TRY(prepare_kernel(k, smem));
        const uint64_t max_ctas = 4ull * sm_count(g->device);
        for (int64_t q = 0; q < A.Q; q++) {
            const uint64_t n = std::max<uint64_t>(nc[q], 1);
            const uint64_t ctas = std::min<uint64_t>(max_ctas, (n + 4095) / 4096);
            const uint32_t per = (uint32_t)((n + ctas - 1) / ctas);
            k<<<(unsigned)ctas, 256, smem, s>>>(A, boxes, q, per);
        }
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    MainShape M;
    MG_TRY((main_shape<FP, AT>(g, A.P.rec != nullptr, threads, &M)));
    return launch_shape(g, A, M, s, false);
}

// Box histograms summed from the mixture table (Sec. 3.6) with error bars
// (Sec. 3.5): one CTA per box walks its footprint blocks; every cube adds
// 8^l mu and (8^l dmu)^2 of each entry of its node's row into shared fp64
// accumulators; the row's error bars are the square roots.
__global__ void __launch_bounds__(256) query_lut_kernel(Geom G, Ids I, const int32_t* __restrict__ boxes,
                                                        const uint64_t* __restrict__ off,
                                                        const uint32_t* __restrict__ src, const double* __restrict__ mu,
                                                        const double* __restrict__ dmu, double* __restrict__ hist,
                                                        double* __restrict__ err, unsigned* __restrict__ status) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ Runs R;
    const uint32_t S = G.S;
    double* h = reinterpret_cast<double*>(smem);
    double* e2 = h + S;
    const int64_t q = blockIdx.x;
    for (uint32_t i = threadIdx.x; i < 2 * S; i += blockDim.x) h[i] = 0.0;
    int32_t b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = boxes[q * 6 + k];
    const bool ok = box_ok(b, G);
    if (threadIdx.x == 0) {
        if (ok) make_runs(b, G, R);
        else set_status(status, kStatBadInput);
    }
    __syncthreads();
    if (ok) {
        // warps take the footprint's blocks in turn; a lane takes a contiguous
        // range of its block's cubes (consecutive cubes of a row) and keeps a
        // run of equal nodes, so a row of k cubes of node n at level l adds
        // k 8^l mu(n) and k (8^l dmu(n))^2 with one pass over n's row
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
        const int nb = R.nx * R.ny * R.nz;
        uint32_t rn = 0xffffffffu, rc = 0;
        int rl = 0;
        auto flush_run = [&]() {
            if (!rc) return;
            const double W = ldexp((double)rc, 3 * rl), W2 = ldexp((double)rc, 6 * rl);
            for (uint64_t t = off[rn]; t < off[rn + 1]; t++) {
                const uint32_t s = src[t];
                if (s >= S) continue;
                atomicAdd(h + s, W * mu[t]);
                const double x = dmu[t];
                if (x != 0.0) atomicAdd(e2 + s, W2 * x * x);
            }
        };
        for (int bi = warp; bi < nb; bi += nwarps) {
            const int i = bi % R.nx, j = (bi / R.nx) % R.ny, k = bi / (R.nx * R.ny);
            const Blk B = make_blk(G, 0, R.sx[i], R.sy[j], R.sz[k], R.lx[i], R.ly[j], R.lz[k], 0);
            const uint32_t n = block_cubes(R.lx[i], R.ly[j], R.lz[k]);
            const uint32_t per = (n + 31) / 32, o0 = min(n, lane * per), o1 = min(n, o0 + per);
            const int lv = B.meta & 63, cp = (B.meta >> 6) & 3;
            const uint32_t bits = (B.meta >> 8) & 1023u, st1 = G.st1[lv][cp], st2 = G.st2[lv][cp];
            const uint16_t* ids16 = static_cast<const uint16_t*>(I.l0[cp]) + B.base;
            const uint32_t* ids32 = (lv ? I.hi[cp] + G.off[lv][cp] : static_cast<const uint32_t*>(I.l0[cp])) + B.base;
            const bool half = lv == 0 && G.id0_bytes == 2;
            for (uint32_t o = o0; o < o1; o++) {
                const uint32_t at = item_at(o, bits, st1, st2);
                const uint32_t node = half ? (uint32_t)__ldg(ids16 + at) : __ldg(ids32 + at);
                if (node == rn && lv == rl) {
                    rc++;
                } else {
                    flush_run();
                    rn = node;
                    rl = lv;
                    rc = 1;
                }
            }
        }
        flush_run();
    }
    __syncthreads();
    for (uint32_t s = threadIdx.x; s < S; s += blockDim.x) {
        hist[q * S + s] = h[s];
        if (err) err[q * S + s] = sqrt(e2[s]);
    }
}

}  // namespace

mg_status query_lut(const mg_graph* g, const int32_t* boxes, int64_t Q, double* hist, double* err, cudaStream_t s) {
    if (!g->err_off.p) return fail(MG_ERR_INVALID_ARG, "build the mixture table first (mg_error_table_build)");
    const size_t sm = (size_t)g->S * 16;
    if (sm > 200 * 1024) return fail(MG_ERR_UNSUPPORTED, "too many segments for the shared fp64 accumulators");
    if (Q == 0) return MG_OK;
    MG_CUDA(cudaFuncSetAttribute(query_lut_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    query_lut_kernel<<<(unsigned)Q, 256, sm, s>>>(make_geom(g, 0), make_ids(g), boxes, g->err_off.as<uint64_t>(),
                                                   g->err_src.as<uint32_t>(), g->err_mu.as<double>(),
                                                   g->err_dmu.as<double>(), hist, err, g->status.as<unsigned>());
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

mg_status count_cubes(const mg_graph* g, const int32_t* boxes, int64_t Q, uint64_t* cubes, cudaStream_t s) {
    const Geom G = make_geom(g, 0);
    plan_count_kernel<<<grid_for(Q * 32, kPlanThreads), kPlanThreads, 0, s>>>(G, boxes, Q, 1, nullptr, cubes, nullptr,
                                                            g->status.as<unsigned>(), false);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

namespace {

int64_t tile_count(int64_t Q, int dev) {
    const int tb = tile_boxes(Q, sm_count(dev));
    return (Q + tb - 1) / tb;
}

// buffers of a batch planned by the fused kernel
struct QueryBufs {
    uint64_t *ncube, *blk_off, *chunk_off;
    Blk* blk;
    uint32_t *chunk_q, *chunk_b;
    uint64_t* words;        // two tickets (fused kernel, main kernel), then the tile words; zero between batches
    uint32_t* acc;          // fp32 histograms: the integer part
    uint64_t cap_blocks, cap_chunks;
    uint32_t chunk;
    MainShape shape;
};

// the batch itself: boxes, size and output given here (Qd, io null), or read on
// the device from Qd and io = {boxes, output} (replayed graphs), Q the most
struct BatchRun {
    const int32_t* boxes;
    int64_t Q;
    const int64_t* Qd;
    void* const* io;
    void* out;
};

// The fused plan kernel and the main kernel, the latter launched with
// programmatic stream serialisation; fp32 histograms then get their integer
// part added (unless `parts`: the caller takes both parts).  ev: events after
// the plan, after the main kernel.
template <bool FP, typename AT>
mg_status enqueue_batch(const mg_graph* g, const QueryBufs& B, const BatchRun& R, bool parts, cudaEvent_t* ev,
                        cudaStream_t s) {
    const mg_dtype weights = std::is_same<AT, __half>::value          ? MG_F16
                             : std::is_same<AT, __nv_bfloat16>::value ? MG_BF16
                                                                      : MG_F32;
    const Geom G = make_geom(g, tile_levels(g, weights));
    unsigned* status = g->status.as<unsigned>();
    const Lim lim{R.Qd, B.cap_blocks, B.cap_chunks};
    uint32_t* acc = FP ? B.acc : static_cast<uint32_t*>(R.out);
    float* accf = FP ? static_cast<float*>(R.out) : nullptr;
    const int64_t tiles = tile_count(R.Q, g->device);
    const int tb = tile_boxes(R.Q, sm_count(g->device));
    const int chunk_shift = (B.chunk & (B.chunk - 1)) == 0 ? __builtin_ctz(B.chunk) : -1;
    FusedOut F;
    F.ncube = B.ncube;
    F.blk_off = B.blk_off;
    F.chunk_off = B.chunk_off;
    F.blk = B.blk;
    F.chunk_q = B.chunk_q;
    F.chunk_b = B.chunk_b;
    F.tiles = B.words + 2;
    F.ticket = reinterpret_cast<unsigned long long*>(B.words);
    F.acc = acc;
    F.accf = accf;
    F.io = R.io;
    plan_fused_kernel<<<(unsigned)tiles, kFusedThreads, 0, s>>>(G, R.boxes, R.Q, tb, B.chunk, chunk_shift, lim, F,
                                                                status);
    MG_CUDA(cudaGetLastError());
    const cudaError_t mark = ev ? cudaEventRecord(ev[0], s) : cudaSuccess;

    const int w16 = weights == MG_BF16;
    MainArgs A;
    A.G = G;
    A.I = make_ids(g);
    A.P.pq = g->pq.as<uint2>();
    A.P.ab32 = g->ab32.as<uint2>();
    A.P.lut_meta = g->lut_meta.as<uint2>();
    A.P.lut = g->lut.as<uint2>();
    A.P.rec = weights == MG_F32 ? g->lut_rec.as<uint4>() : g->rec16[w16].as<uint4>();
    A.P.frac = weights == MG_F32 ? nullptr : g->frac16[w16].as<float>();
    A.P.alpha = weights == MG_F16 ? g->alpha16.p : weights == MG_BF16 ? g->alphab16.p : g->alpha.p;
    A.P.S = g->S;
    A.P.status = status;
    A.blk = B.blk;
    A.blk_off = B.blk_off;
    A.ncube = B.ncube;
    A.chunk_off = B.chunk_off;
    A.chunk_q = B.chunk_q;
    A.chunk_b = B.chunk_b;
    A.total_chunks = 0;
    A.planned = true;
    A.lim = lim;
    A.clean = B.words;
    A.clean_words = (uint32_t)(2 + 2 * tiles);
    A.Q = R.Q;
    A.chunk = B.chunk;
    A.ticket = F.ticket + 1;
    A.acc = acc;
    A.accf = accf;
    A.io = R.io;
    A.qcap = 0;   // the shape's
    const mg_status st =
        mark == cudaSuccess ? launch_shape(g, A, B.shape, s, !ev) : cuda_fail(mark, "cudaEventRecord");
    if (st != MG_OK) {   // it is the main kernel that zeroes the words for the next batch
        cudaMemsetAsync(B.words, 0, (size_t)A.clean_words * 8, s);
        return st;
    }
    if (ev) MG_CUDA(cudaEventRecord(ev[1], s));
    if (FP && !parts) {
        const int64_t cells = R.Q * (int64_t)g->S;
        const unsigned gb = grid_for(cells, 256, 152 * 64);
        if (R.io) dense_f32_rows_kernel<<<gb, 256, 0, s>>>(acc, R.io, R.Qd, g->S);
        else dense_f32_kernel<<<gb, 256, 0, s>>>(acc, accf, cells);
        MG_CUDA(cudaGetLastError());
    }
    return MG_OK;
}

mg_status enqueue_any(const mg_graph* g, const QueryBufs& B, const BatchRun& R, bool FP, mg_dtype weights, bool parts,
                      cudaEvent_t* ev, cudaStream_t s) {
    if (!FP) return enqueue_batch<false, float>(g, B, R, parts, ev, s);
    if (weights == MG_F16) return enqueue_batch<true, __half>(g, B, R, parts, ev, s);
    if (weights == MG_BF16) return enqueue_batch<true, __nv_bfloat16>(g, B, R, parts, ev, s);
    return enqueue_batch<true, float>(g, B, R, parts, ev, s);
}

mg_status shape_of(const mg_graph* g, bool FP, mg_dtype weights, int threads, MainShape* out) {
    const bool rec = (weights == MG_F32 ? g->lut_rec : g->rec16[weights == MG_BF16]).p != nullptr;
    if (!FP) return main_shape<false, float>(g, rec, threads, out);
    if (weights == MG_F16) return main_shape<true, __half>(g, rec, threads, out);
    if (weights == MG_BF16) return main_shape<true, __nv_bfloat16>(g, rec, threads, out);
    return main_shape<true, float>(g, rec, threads, out);
}

// Threads of an untuned batch's CTAs.  256 have the smaller register budget and
// the faster loop; where their histograms leave shared memory for a quarter
// fewer warps per SM than CTAs of 128 (the loop is bound by latency, so resident
// warps count), 128.  fp32 histograms of 1,182 segments, 16 against 20 warps:
// 100,000 boxes 2.98 -> 2.60 ms, with 16-bit weights 17.7 -> 14.7, 1,000 boxes
// 307 -> 274 us; uint32 counts, 32 against 36: 1.66 at 256, 1.70 at 128; fp32
// histograms of 353, 40 against 36: 547 us at 256, 574 at 128 (10,000 boxes).
int default_threads(const mg_graph* g, bool FP, mg_dtype weights) {
    const bool rec = (weights == MG_F32 ? g->lut_rec : g->rec16[weights == MG_BF16]).p != nullptr;
    const size_t bins = FP ? 2 : 1, queue = queue_bytes(kQueueShort);
    if ((g->S * 4 * bins + queue) * 8 > 96 * 1024) return 256;   // a histogram per CTA
    const size_t each = ((g->S + 3) & ~(size_t)3) * 4 * bins + kDescBytes + (rec ? 0 : queue);
    const size_t sm = kMaxDynSmem + 1024;                        // a CTA takes 1 KiB more than it asks for
    auto warps = [&](size_t w, size_t most) { return w * std::min<size_t>(most, sm / (w * each + 1024)); };
    return 4 * warps(4, WarpKernelBounds<128>::min_ctas) >= 5 * warps(8, WarpKernelBounds<256>::min_ctas) ? 128 : 256;
}

// The launch shape of a batch: what the caller names, else what
// mg_query_autotune or mg_query_set_tuning recorded, else the defaults.  The
// tuner's shape holds for the weights it was tuned with (16-bit weights want
// other CTAs and longer chunks than fp32 ones).  It tries 1,024 items and more:
// where the best length is nearer to 512 (or below 512 with a histogram per CTA,
// whose CTAs of 512 threads gain on long chunks), a batch has too few of those,
// whatever batch they were tuned on (us a run untuned / tuned: 1,000 boxes of
// 64^3 25 / 41, of 512x512x384 40 / 65, 3,000 of these 61 / 69, 10,000 beside a
// frame's propagation 160 / 150; 15,917 segments, 100 boxes 53 / 44).
struct Shape {
    int threads;
    uint32_t chunk;
    uint32_t longest;   // the chunks that capacities are counted in
    bool recorded;      // the chunk is a recorded one
};
// whether a batch has enough recorded chunks
bool takes_recorded(const mg_graph* g, bool FP, mg_dtype weights, int threads, int64_t Q) {
    const bool own = warp_hists(g, FP, threads);
    return ideal_chunk(g, FP, weights, own, Q) >= (own ? 1024 / std::sqrt(2.0) : 512.0);
}
Shape launch_shape_of(const mg_graph* g, bool FP, mg_dtype weights, int chunk_cubes, int block_threads, int64_t Q) {
    if (!FP) weights = MG_F32;
    const bool told = !FP || g->tuned_weights < 0 || g->tuned_weights == (int)weights;
    uint32_t tuned = told ? (uint32_t)g->tuned_chunk[FP] : 0u;
    int threads = told ? g->tuned_threads[FP] : 0;
    const int usual = default_threads(g, FP, weights);
    Shape R;
    R.longest = chunk_cubes > 0 ? (uint32_t)chunk_cubes : tuned ? tuned : kDefaultChunk;
    const uint32_t c = default_chunk(g, FP, weights, block_threads > 0 ? block_threads : usual, Q);
    if (chunk_cubes <= 0 && tuned > c && !takes_recorded(g, FP, weights, usual, Q)) {
        tuned = 0;
        threads = 0;
    }
    R.threads = block_threads > 0 ? block_threads : threads > 0 ? threads : usual;
    R.recorded = chunk_cubes <= 0 && tuned != 0;
    R.chunk = chunk_cubes > 0 ? R.longest : tuned ? tuned : default_chunk(g, FP, weights, R.threads, Q);
    return R;
}

// Scratch comes from `al`; `words` are two host words for readbacks; `room`,
// when not null, returns the bytes `al` can still hand out (fixed pools).
mg_status query_boxes_impl(const mg_graph* g, const int32_t* boxes, int64_t Q, const mg_query_opts& o, void* out,
                           size_t cap, uint32_t* seg, uint64_t* offsets, size_t* required, cudaStream_t s,
                           const Alloc& al, uint64_t* words, size_t (*room)(const Alloc&)) {
    const uint32_t S = g->S;
    const bool FP = o.hist_type == MG_HIST_F32;
    const bool csr = o.layout == MG_LAYOUT_CSR;
    if (S > kMaxSharedSegments) return fail(MG_ERR_UNSUPPORTED, "more than 32768 segments");
    const_cast<mg_graph*>(g)->hold_tiles();
    if (required) *required = 0;
    if (Q == 0) {
        if (csr) MG_CUDA(cudaMemsetAsync(offsets, 0, sizeof(uint64_t), s));
        return MG_OK;
    }
    if (FP && o.alpha_dtype != MG_F32) {
        MG_TRY(ensure_alpha16(const_cast<mg_graph*>(g), (mg_dtype)o.alpha_dtype, s));
        MG_TRY(ensure_records16(const_cast<mg_graph*>(g), (mg_dtype)o.alpha_dtype, s));
    }
    const Shape shape = launch_shape_of(g, FP, (mg_dtype)o.alpha_dtype, o.chunk_cubes, o.block_threads, Q);
    const int threads = o.schedule == MG_SCHED_BATCHED || o.block_threads > 0 ? shape.threads
                        : g->tuned_threads[FP] > 0                            ? g->tuned_threads[FP]
                                                                              : 256;
    const uint32_t longest = shape.longest;
    uint32_t chunk = shape.chunk;
    // the room of a fixed pool is counted in long chunks: shorter ones are taken
    // where the batch fits with them too, and there is one scan to repeat
    if (room && Q > kFusedScanMax) chunk = longest;
    // Where the most that this many boxes can have fits a modest buffer, the
    // footprint is planned in one launch and nothing is read back: 1,000 boxes
    // of a 64^3 volume took 69 us with three plan kernels and the read-back of
    // their totals, 34 with this.  That is worth somewhat longer chunks (300
    // boxes of 512x512x384, 16-bit weights: 97 us with 128 items and the
    // read-back, 59 with 256).
    constexpr uint64_t kMostUnread = 1u << 22;
    const uint64_t most_blocks = block_bound(g, Q);
    bool fused = o.schedule == MG_SCHED_BATCHED && !room && most_blocks < kMostUnread;
    while (fused && chunk < longest && chunk_bound(g, Q, chunk) >= kMostUnread) chunk = std::min(2 * chunk, longest);
    const uint64_t most_chunks = chunk_bound(g, Q, chunk);
    fused = fused && most_chunks < kMostUnread;
    const Geom G = make_geom(g, tile_levels(g, (mg_dtype)o.alpha_dtype));
    unsigned* status = g->status.as<unsigned>();
    mg_graph* gm = const_cast<mg_graph*>(g);
    const bool timed = o.timing != 0;
    if (timed) {
        for (auto& e : gm->qev)
            if (!e) MG_CUDA(cudaEventCreate(&e));
        gm->qev_valid = false;
        MG_CUDA(cudaEventRecord(gm->qev[0], s));
    }

    // accumulators: the dense u32 output itself, else scratch
    Buf acc_b, accf_b;
    uint32_t* acc = nullptr;
    float* accf = nullptr;
    const size_t cells = (size_t)Q * S;
    if (!csr && !FP) {
        acc = static_cast<uint32_t*>(out);
    } else {
        MG_TRY(acc_b.alloc(&al, cells * 4, s));
        acc = acc_b.as<uint32_t>();
    }
    if (FP) {
        if (!csr) {
            accf = static_cast<float*>(out);
        } else {
            MG_TRY(accf_b.alloc(&al, cells * 4, s));
            accf = accf_b.as<float>();
        }
    }

    const mg_dtype weights = (mg_dtype)o.alpha_dtype;
    const int w16 = weights == MG_BF16;
    MainArgs A;
    A.G = G;
    A.I = make_ids(g);
    A.P.pq = g->pq.as<uint2>();
    A.P.ab32 = g->ab32.as<uint2>();
    A.P.lut_meta = g->lut_meta.as<uint2>();
    A.P.lut = g->lut.as<uint2>();
    A.P.rec = weights == MG_F32 ? g->lut_rec.as<uint4>() : g->rec16[w16].as<uint4>();
    A.P.frac = weights == MG_F32 ? nullptr : g->frac16[w16].as<float>();
    A.P.alpha = o.alpha_dtype == MG_F16 ? g->alpha16.p : o.alpha_dtype == MG_BF16 ? g->alphab16.p : g->alpha.p;
    A.P.S = S;
    A.P.status = status;
    A.Q = Q;
    A.chunk = chunk;
    A.acc = acc;
    A.accf = accf;
    A.blk = nullptr;
    A.blk_off = nullptr;
    A.ncube = nullptr;
    A.chunk_off = nullptr;
    A.chunk_q = nullptr;
    A.chunk_b = nullptr;
    A.total_chunks = 0;
    A.lim = Lim{nullptr, 0, 0};
    A.planned = false;
    A.clean = nullptr;
    A.clean_words = 0;
    A.ticket = nullptr;
    A.io = nullptr;
    A.qcap = kQueueShort;

    const size_t smem = hist_smem(S, FP);
    if (smem > 220 * 1024) return fail(MG_ERR_UNSUPPORTED, "too many segments for the shared-memory histogram");
    Buf nblk, ncube, nchunk, blk_off, chunk_off, blk, ticket, chunk_q, chunk_b, tiles;
    const size_t words_bytes = 16 + 16 * (size_t)tile_count(Q, g->device);
    if (fused) {
        // buffers of that size are more than the batch needs: where there is no
        // memory for them, it is planned with a read-back
        auto got = [&](Buf& b, size_t n) { return b.alloc(&al, n, s) == MG_OK; };
        fused = got(ncube, (size_t)Q * 8) && got(blk_off, (size_t)(Q + 1) * 8) && got(chunk_off, (size_t)(Q + 1) * 8) &&
                got(blk, (size_t)most_blocks * sizeof(Blk)) && got(chunk_q, (size_t)most_chunks * 4) &&
                got(chunk_b, (size_t)most_chunks * 4) && got(tiles, words_bytes);
        if (!fused) {
            for (Buf* b : {&ncube, &blk_off, &chunk_off, &blk, &chunk_q, &chunk_b, &tiles}) b->release();
            set_error("");
        }
    }
    if (fused) {
        QueryBufs B;
        B.cap_blocks = most_blocks;
        B.cap_chunks = most_chunks;
        B.chunk = chunk;
        MG_TRY(shape_of(g, FP, weights, threads, &B.shape));
        B.ncube = ncube.as<uint64_t>();
        B.blk_off = blk_off.as<uint64_t>();
        B.chunk_off = chunk_off.as<uint64_t>();
        B.blk = blk.as<Blk>();
        B.chunk_q = chunk_q.as<uint32_t>();
        B.chunk_b = chunk_b.as<uint32_t>();
        B.words = tiles.as<uint64_t>();
        B.acc = acc;
        MG_CUDA(cudaMemsetAsync(B.words, 0, words_bytes, s));
        const BatchRun run{boxes, Q, nullptr, nullptr, FP ? static_cast<void*>(accf) : static_cast<void*>(acc)};
        cudaEvent_t* ev = timed ? gm->qev + 1 : nullptr;
        MG_TRY(enqueue_any(g, B, run, FP, weights, csr, ev, s));
    } else if (o.schedule == MG_SCHED_BATCHED) {
        MG_TRY(nblk.alloc(&al, (size_t)Q * 4, s));
        MG_TRY(ncube.alloc(&al, (size_t)Q * 8, s));
        MG_TRY(nchunk.alloc(&al, (size_t)Q * 8, s));
        MG_TRY(blk_off.alloc(&al, (size_t)(Q + 1) * 8, s));
        MG_TRY(chunk_off.alloc(&al, (size_t)(Q + 1) * 8, s));
        MG_TRY(ticket.alloc(&al, 8, s));
        uint64_t* totals = words;   // blocks, chunks
        for (;;) {
            plan_count_kernel<<<grid_for(Q * 32, kPlanThreads), kPlanThreads, 0, s>>>(G, boxes, Q, chunk, nblk.as<uint32_t>(),
                                                                    ncube.as<uint64_t>(), nchunk.as<uint64_t>(),
                                                                    status, true);
            MG_CUDA(cudaGetLastError());
            if (Q <= kFusedScanMax) {
                plan_scan_kernel<<<1, kScanThreads, 0, s>>>(nblk.as<uint32_t>(), nchunk.as<uint64_t>(), Q,
                                                            blk_off.as<uint64_t>(), chunk_off.as<uint64_t>());
                MG_CUDA(cudaGetLastError());
            } else {
                // block offsets are 64-bit sums of the 32-bit per-box counts
                MG_TRY(scan_exclusive_u64(nchunk.as<uint64_t>(), chunk_off.as<uint64_t>(), Q,
                                          chunk_off.as<uint64_t>() + Q, al, s));
                Buf nb64;
                MG_TRY(nb64.alloc(&al, (size_t)Q * 8, s));
                widen_kernel<<<grid_for(Q, 256, 152 * 64), 256, 0, s>>>(nblk.as<uint32_t>(), nb64.as<uint64_t>(), Q);
                MG_CUDA(cudaGetLastError());
                MG_TRY(scan_exclusive_u64(nb64.as<uint64_t>(), blk_off.as<uint64_t>(), Q, blk_off.as<uint64_t>() + Q, al,
                                          s));
            }
            MG_CUDA(cudaMemcpyAsync(&totals[0], blk_off.as<uint64_t>() + Q, 8, cudaMemcpyDeviceToHost, s));
            MG_CUDA(cudaMemcpyAsync(&totals[1], chunk_off.as<uint64_t>() + Q, 8, cudaMemcpyDeviceToHost, s));
            MG_CUDA(cudaStreamSynchronize(s));
            if (totals[0] >= (1ull << 32) || totals[1] >= (1ull << 32))
                return fail(MG_ERR_UNSUPPORTED, "more than 2^32 footprint blocks or work chunks in one call");
            if (room) {
                const size_t need = (((size_t)std::max<uint64_t>(totals[0], 1) * sizeof(Blk) + 255) & ~(size_t)255) +
                                    2 * (((size_t)std::max<uint64_t>(totals[1], 1) * 4 + 255) & ~(size_t)255);
                if (need > room(al) && chunk < longest) {
                    chunk = longest;
                    continue;
                }
                if (need > room(al))
                    return fail(MG_ERR_CAPACITY, "these boxes need " + std::to_string(need >> 10) +
                                                     " KiB of footprint scratch; " + std::to_string(room(al) >> 10) +
                                                     " KiB of the fixed scratch remain: split the batch");
            }
            break;
        }
        A.chunk = chunk;
        MG_TRY(blk.alloc(&al, (size_t)std::max<uint64_t>(totals[0], 1) * sizeof(Blk), s));
        MG_TRY(chunk_q.alloc(&al, (size_t)std::max<uint64_t>(totals[1], 1) * 4, s));
        MG_TRY(chunk_b.alloc(&al, (size_t)std::max<uint64_t>(totals[1], 1) * 4, s));
        plan_write_kernel<<<grid_for(Q * 32, kPlanThreads), kPlanThreads, 0, s>>>(
            G, boxes, Q, blk_off.as<uint64_t>(), blk.as<Blk>(), chunk_off.as<uint64_t>(), chunk,
            chunk_q.as<uint32_t>(), chunk_b.as<uint32_t>());
        MG_CUDA(cudaGetLastError());
        A.chunk_q = chunk_q.as<uint32_t>();
        A.chunk_b = chunk_b.as<uint32_t>();
        A.total_chunks = totals[1];
        MG_CUDA(cudaMemsetAsync(ticket.p, 0, 8, s));
        A.blk = blk.as<Blk>();
        A.blk_off = blk_off.as<uint64_t>();
        A.ncube = ncube.as<uint64_t>();
        A.chunk_off = chunk_off.as<uint64_t>();
        A.ticket = ticket.as<unsigned long long>();
    }
    // the accumulators are cleared only once the footprint is known to fit, so
    // a refused call leaves the caller's output as it was
    if (!fused) {
        if (FP) MG_CUDA(cudaMemsetAsync(accf, 0, cells * 4, s));
        MG_CUDA(cudaMemsetAsync(acc, 0, cells * 4, s));
        if (timed) MG_CUDA(cudaEventRecord(gm->qev[1], s));
    }
    if (!fused && FP) {
        if (o.alpha_dtype == MG_F16)
            MG_TRY((launch_main<true, __half>(g, A, o, boxes, smem, threads, s, &al)));
        else if (o.alpha_dtype == MG_BF16)
            MG_TRY((launch_main<true, __nv_bfloat16>(g, A, o, boxes, smem, threads, s, &al)));
        else
            MG_TRY((launch_main<true, float>(g, A, o, boxes, smem, threads, s, &al)));
    } else if (!fused) {
        MG_TRY((launch_main<false, float>(g, A, o, boxes, smem, threads, s, &al)));
    }

    if (timed && !fused) MG_CUDA(cudaEventRecord(gm->qev[2], s));
    if (!csr) {
        if (FP && !fused) {
            dense_f32_kernel<<<grid_for((int64_t)cells, 256, 152 * 64), 256, 0, s>>>(acc, accf, (int64_t)cells);
            MG_CUDA(cudaGetLastError());
        }
        if (timed) {
            MG_CUDA(cudaEventRecord(gm->qev[3], s));
            gm->qev_valid = true;
        }
        return MG_OK;
    }
    // CSR: count, scan, capacity check, write
    Buf cnt;
    MG_TRY(cnt.alloc(&al, (size_t)Q * 8, s));
    if (FP)
        csr_count_kernel<true><<<grid_for(Q * 32, 256), 256, 0, s>>>(acc, accf, Q, S, cnt.as<uint64_t>());
    else
        csr_count_kernel<false><<<grid_for(Q * 32, 256), 256, 0, s>>>(acc, accf, Q, S, cnt.as<uint64_t>());
    MG_CUDA(cudaGetLastError());
    MG_TRY(scan_exclusive_u64(cnt.as<uint64_t>(), offsets, Q, offsets + Q, al, s));
    uint64_t* nnz_p = words;
    MG_CUDA(cudaMemcpyAsync(nnz_p, offsets + Q, 8, cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    const uint64_t nnz = *nnz_p;
    if (required) *required = (size_t)nnz;
    if (nnz > cap) return fail(MG_ERR_CAPACITY, "CSR output needs " + std::to_string(nnz) + " entries");
    if (FP)
        csr_write_kernel<true><<<grid_for(Q * 32, 256), 256, 0, s>>>(acc, accf, Q, S, offsets, seg, out);
    else
        csr_write_kernel<false><<<grid_for(Q * 32, 256), 256, 0, s>>>(acc, accf, Q, S, offsets, seg, out);
    MG_CUDA(cudaGetLastError());
    if (timed) {
        MG_CUDA(cudaEventRecord(gm->qev[3], s));
        gm->qev_valid = true;
    }
    return MG_OK;
}

}  // namespace

mg_status query_boxes(const mg_graph* g, const int32_t* boxes, int64_t Q, const mg_query_opts& o, void* out,
                      size_t cap, uint32_t* seg, uint64_t* offsets, size_t* required, cudaStream_t s) {
    Arena* arena = nullptr;
    MG_TRY(arena_begin(const_cast<mg_graph*>(g), s, &arena));
    uint64_t local[2] = {0, 0};
    return query_boxes_impl(g, boxes, Q, o, out, cap, seg, offsets, required, s, arena->view,
                            arena->pinned ? arena->pinned : local, nullptr);
}

mg_status query_timing(const mg_graph* g, float* plan_ms, float* main_ms, float* out_ms) {
    if (!g->qev_valid) return fail(MG_ERR_INVALID_ARG, "no timed query call on this graph");
    MG_CUDA(cudaEventSynchronize(g->qev[3]));
    float t[3];
    for (int i = 0; i < 3; i++) MG_CUDA(cudaEventElapsedTime(&t[i], g->qev[i], g->qev[i + 1]));
    if (plan_ms) *plan_ms = t[0];
    if (main_ms) *main_ms = t[1];
    if (out_ms) *out_ms = t[2];
    return MG_OK;
}

}  // namespace mg

// ---------------------------------------------------------------------------
// Box histograms for callers that cannot allocate device memory: the same
// exact dense query with its scratch in a fixed array compiled into the
// library instead of memory from the allocator.
// ---------------------------------------------------------------------------
namespace mg {
namespace {

// Fixed scratch of mg_query_boxes_noalloc.  Every GPU that loads the library
// holds these 64 MiB until the process exits.
constexpr size_t kNoAllocBytes = 64ull << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

std::mutex g_noalloc_mu;
void* g_noalloc_addr[256] = {};   // device address of the array, per device

// Host code only knows a stand-in for the array's name; the device address is
// looked up once per device, with that device current.
mg_status noalloc_scratch(int dev, unsigned char** out) {
    if (dev < 0 || dev >= 256) return fail(MG_ERR_UNSUPPORTED, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(fixed query scratch)");
        g_noalloc_addr[dev] = p;
    }
    *out = static_cast<unsigned char*>(g_noalloc_addr[dev]);
    return MG_OK;
}

// bump allocation from the fixed array for one call
struct Pool {
    unsigned char* base;
    size_t cap, used;
};

void* pool_alloc(void* ctx, size_t bytes, mg_stream) {
    Pool* pl = static_cast<Pool*>(ctx);
    const size_t n = (bytes + 255) & ~(size_t)255;
    if (pl->used + n > pl->cap) return nullptr;
    void* p = pl->base + pl->used;
    pl->used += n;
    return p;
}

void pool_free(void*, void*, size_t, mg_stream) {}

size_t pool_room(const Alloc& al) {
    const Pool* pl = static_cast<const Pool*>(al.a.ctx);
    return pl->cap - pl->used;
}

size_t rounded(size_t n) { return (n + 255) & ~(size_t)255; }

// scratch of the per-box plan arrays and their scans, before the footprint blocks
size_t per_box_scratch(int64_t Q) {
    const size_t q = (size_t)Q;
    const size_t parts = rounded(8 * ((q + 2047) / 2048)) * 2;   // one scan level's partial sums
    return rounded(4 * q) + 5 * rounded(8 * (q + 1)) + rounded(8) + 2 * (parts + 2 * rounded(8)) + 4096;
}

}  // namespace
}  // namespace mg

extern "C" MG_API mg_status mg_query_boxes_noalloc(const mg_graph* g, const int32_t* boxes, int64_t Q, uint32_t* out,
                                                   size_t out_capacity, mg_stream stream) {
    MG_RANGE("mg_query_boxes_noalloc");
    using namespace mg;
    if (!g) return fail(MG_ERR_INVALID_ARG, "graph is NULL");
    if (Q < 0) return fail(MG_ERR_INVALID_ARG, "Q must be >= 0");
    if (Q == 0) return MG_OK;
    if (!boxes || !out) return fail(MG_ERR_INVALID_ARG, "NULL argument");
    if ((uint64_t)out_capacity < (uint64_t)Q * g->S) return fail(MG_ERR_INVALID_ARG, "out_capacity must be >= Q*S");
    if (g->S > kMaxSharedSegments) return fail(MG_ERR_UNSUPPORTED, "more than 32768 segments");
    if (g->quantised) return fail(MG_ERR_UNSUPPORTED, "a quantised graph has no exact weights");
    if (per_box_scratch(Q) > kNoAllocBytes / 2) {
        int64_t qmax = 1;
        while (per_box_scratch(qmax * 2) <= kNoAllocBytes / 2) qmax *= 2;
        return fail(MG_ERR_CAPACITY, "at most about " + std::to_string(qmax) +
                                         " boxes fit the fixed query scratch in one call: split the batch");
    }
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device) MG_CUDA(cudaSetDevice(g->device));
    unsigned char* base = nullptr;
    mg_status st = noalloc_scratch(g->device, &base);
    if (st == MG_OK) {
        Pool pool{base, kNoAllocBytes, 0};
        Alloc al;
        al.a.ctx = &pool;
        al.a.alloc = pool_alloc;
        al.a.free = pool_free;
        al.custom = true;
        mg_query_opts o{};   // exact uint32 counts, dense, batched, default tuning
        uint64_t words[2] = {0, 0};
        st = query_boxes_impl(g, boxes, Q, o, out, out_capacity, nullptr, nullptr, nullptr,
                              reinterpret_cast<cudaStream_t>(stream), al, words, pool_room);
    }
    if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    return st;
}

// ---------------------------------------------------------------------------
// Query plans: every buffer of a batch of up to max_Q boxes, allocated once; a
// run is two launches (three for fp32 histograms) on the caller's boxes and
// output, with no host synchronisation.  The request loop replays the same
// launches as a CUDA graph on the plan's own buffers.
// ---------------------------------------------------------------------------
struct mg_query_plan {
    mg_graph* g = nullptr;
    int64_t max_Q = 0;
    bool fp = false;
    mg_dtype weights = MG_F32;
    int threads = 0;
    bool told = false, recorded = false;   // the chunk is the caller's, a recorded one
    mg::QueryBufs bufs{};
    mg::Buf pool;
    mg::Pool bump{nullptr, 0, 0};
    int32_t* boxes = nullptr;
    int64_t* Qd = nullptr;
    void* result = nullptr;   // max_Q x S, uint32 or fp32
    void** io = nullptr;      // device slots: the run's boxes and output (default: boxes, result)
    cudaStream_t cap_stream = nullptr;
    cudaGraph_t graph[2] = {nullptr, nullptr};         // any batch; a few boxes
    cudaGraphExec_t exec[2] = {nullptr, nullptr};
    bool timed = false, ran = false;
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};   // graph start, plan done, main done
    ~mg_query_plan() {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        for (cudaGraphExec_t e : exec)
            if (e) cudaGraphExecDestroy(e);
        for (cudaGraph_t e : graph)
            if (e) cudaGraphDestroy(e);
        if (cap_stream) cudaStreamDestroy(cap_stream);
    }
};

namespace mg {
uint32_t longest_chunk(const mg_graph* g, int hist_type) {
    const int tuned = g->tuned_chunk[hist_type == MG_HIST_F32];
    return tuned > 0 ? (uint32_t)tuned : kDefaultChunk;
}

PlanChunk plan_chunk(const mg_graph* g, int hist_type, mg_dtype weights, int chunk_cubes, int block_threads,
                     int64_t max_Q, uint64_t cap_chunks) {
    const Shape R = launch_shape_of(g, hist_type == MG_HIST_F32, weights, chunk_cubes, block_threads, max_Q);
    for (uint32_t c = R.chunk; c < R.longest; c *= 2) {
        const uint64_t n = std::min(cap_chunks * ((R.longest + c - 1) / c), chunk_bound(g, max_Q, c));
        if (n <= std::max<uint64_t>(cap_chunks, 1u << 23)) return PlanChunk{c, n, R.threads, R.recorded};
    }
    return PlanChunk{R.longest, cap_chunks, R.threads, R.recorded};
}

// Chunk length of a run of Q boxes: the plan's, or a shorter one that suits so
// few boxes where the plan's chunk map holds the most that they can have (one
// box with 15,917 segments and fp32 histograms by a plan for 10,000: 55 -> 33 us).
static uint32_t run_chunk(const mg_query_plan* p, int64_t Q) {
    const QueryBufs& B = p->bufs;
    if (p->told || Q == p->max_Q) return B.chunk;
    const int threads = B.shape.threads;
    uint32_t c = default_chunk(p->g, p->fp, p->fp ? p->weights : MG_F32, threads, Q);
    if (p->recorded && takes_recorded(p->g, p->fp, p->fp ? p->weights : MG_F32, threads, Q)) return B.chunk;
    while (c < B.chunk && chunk_bound(p->g, Q, c) > B.cap_chunks) c *= 2;
    return std::min(c, B.chunk);
}

mg_status plan_parts(mg_query_plan* p, PlanParts* out) {
    if (!p->exec[0]) {
        MG_CUDA(cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
        for (int k = 0; k < 2; k++) {
            const int64_t Q = k == 0 ? p->max_Q : std::min<int64_t>(p->max_Q, kFewBoxes);
            QueryBufs B = p->bufs;
            if (k == 1) B.chunk = run_chunk(p, Q);
            MG_CUDA(cudaStreamBeginCapture(p->cap_stream, cudaStreamCaptureModeThreadLocal));
            const BatchRun run{p->boxes, Q, p->Qd, p->io, p->result};
            const mg_status st = enqueue_any(p->g, B, run, p->fp, p->weights, false, nullptr, p->cap_stream);
            const cudaError_t e = cudaStreamEndCapture(p->cap_stream, &p->graph[k]);
            if (st != MG_OK) return st;
            if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
            MG_CUDA(cudaGraphInstantiate(&p->exec[k], p->graph[k], 0));
        }
    }
    *out = PlanParts{p->boxes, p->Qd, p->result, p->exec[0], p->exec[1],
                     p->bufs.chunk, p->bufs.cap_blocks, p->bufs.cap_chunks};
    return MG_OK;
}
}  // namespace mg

using mg::fail;

extern "C" {

MG_API mg_status mg_query_plan_create(mg_graph* g, int64_t max_Q, const mg_query_opts* opts, int64_t max_blocks,
                                      int64_t max_chunks, mg_query_plan** out) {
    MG_RANGE("mg_query_plan_create");
    using namespace mg;
    if (!g || !out) return fail(MG_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    if (max_Q < 1 || max_Q >= (1ll << 31)) return fail(MG_ERR_INVALID_ARG, "max_Q must be in 1..2^31-1");
    if (max_blocks < 0 || max_chunks < 0) return fail(MG_ERR_INVALID_ARG, "negative capacity");
    mg_query_opts o{};
    if (opts) o = *opts;
    if (o.layout != MG_LAYOUT_DENSE || o.schedule != MG_SCHED_BATCHED)
        return fail(MG_ERR_UNSUPPORTED, "plans hold the dense layout and the batched schedule");
    if (o.hist_type != MG_HIST_U32 && o.hist_type != MG_HIST_F32) return fail(MG_ERR_INVALID_ARG, "bad hist_type");
    if (g->quantised && o.hist_type == MG_HIST_U32)
        return fail(MG_ERR_UNSUPPORTED, "a quantised graph has no exact weights: use MG_HIST_F32");
    if (o.alpha_dtype != MG_F32 && (o.hist_type == MG_HIST_U32 || (o.alpha_dtype != MG_F16 && o.alpha_dtype != MG_BF16)))
        return fail(MG_ERR_INVALID_ARG, "bad alpha_dtype");
    if (o.block_threads && o.block_threads != 128 && o.block_threads != 256 && o.block_threads != 512)
        return fail(MG_ERR_INVALID_ARG, "block_threads must be 128, 256 or 512");
    if (o.chunk_cubes < 0) return fail(MG_ERR_INVALID_ARG, "negative chunk_cubes");
    if (g->S > kMaxSharedSegments) return fail(MG_ERR_UNSUPPORTED, "more than 32768 segments");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device) MG_CUDA(cudaSetDevice(g->device));
    std::unique_ptr<mg_query_plan> p(new (std::nothrow) mg_query_plan());
    mg_status st = p ? MG_OK : fail(MG_ERR_OOM, "host allocation failed");
    g->hold_tiles();
    if (st == MG_OK && o.hist_type == MG_HIST_F32 && o.alpha_dtype != MG_F32) {   // (the launch shape depends on them)
        st = ensure_alpha16(g, (mg_dtype)o.alpha_dtype, nullptr);
        if (st == MG_OK) st = ensure_records16(g, (mg_dtype)o.alpha_dtype, nullptr);
    }
    if (st == MG_OK) {
        const bool FP = o.hist_type == MG_HIST_F32;
        p->g = g;
        p->max_Q = max_Q;
        p->fp = FP;
        p->weights = (mg_dtype)o.alpha_dtype;
        QueryBufs& B = p->bufs;
        B.cap_blocks = max_blocks > 0 ? (uint64_t)max_blocks : (uint64_t)max_Q * 1024;
        B.cap_chunks = max_chunks > 0 ? (uint64_t)max_chunks : (uint64_t)max_Q * 256;
        const PlanChunk pc = plan_chunk(g, o.hist_type, p->weights, o.chunk_cubes, o.block_threads, max_Q, B.cap_chunks);
        B.chunk = pc.chunk;
        B.cap_chunks = pc.cap_chunks;
        p->threads = pc.threads;
        p->told = o.chunk_cubes > 0;
        p->recorded = pc.recorded;
        if (B.cap_blocks >= (1ull << 32) || B.cap_chunks >= (1ull << 32))
            st = fail(MG_ERR_UNSUPPORTED, "plan capacities must be below 2^32");
    }
    if (st == MG_OK) {
        QueryBufs& B = p->bufs;
        const size_t S = g->S, Q = (size_t)max_Q;
        auto r = [](size_t n) { return (n + 255) & ~(size_t)255; };
        // boxes, batch size, io slots, results (+ the integer part of fp32
        // ones), cube counts, both offset arrays, blocks, chunk map, tile words
        // (a pair per box at most), tickets
        const size_t bytes = r(Q * 24) + r(8) + r(16) + r(Q * S * 4) * (p->fp ? 2 : 1) + r(8 * Q) + 2 * r(8 * (Q + 1)) +
                             r(B.cap_blocks * sizeof(Blk)) + 2 * r(B.cap_chunks * 4) + r(16 * Q + 16) + 65536;
        st = p->pool.alloc(&g->al, bytes, nullptr);
        if (st == MG_OK) {
            p->bump = Pool{p->pool.as<unsigned char>(), p->pool.bytes, 0};
            auto take = [&](size_t n) { return pool_alloc(&p->bump, n, nullptr); };
            p->boxes = static_cast<int32_t*>(take(Q * 24));
            p->Qd = static_cast<int64_t*>(take(8));
            p->result = take(Q * S * 4);
            p->io = static_cast<void**>(take(16));
            B.acc = p->fp ? static_cast<uint32_t*>(take(Q * S * 4)) : nullptr;
            B.ncube = static_cast<uint64_t*>(take(Q * 8));
            B.blk_off = static_cast<uint64_t*>(take((Q + 1) * 8));
            B.chunk_off = static_cast<uint64_t*>(take((Q + 1) * 8));
            B.blk = static_cast<Blk*>(take(B.cap_blocks * sizeof(Blk)));
            B.chunk_q = static_cast<uint32_t*>(take(B.cap_chunks * 4));
            B.chunk_b = static_cast<uint32_t*>(take(B.cap_chunks * 4));
            B.words = static_cast<uint64_t*>(take(16 * Q + 16));
            void* io0[2] = {p->boxes, p->result};
            cudaError_t e = cudaMemcpy(p->io, io0, sizeof(io0), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = cudaMemsetAsync(B.words, 0, 16 * Q + 16, nullptr);
            if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
            if (e != cudaSuccess) st = cuda_fail(e, "plan buffers");
            p->pool.s = nullptr;
        }
    }
    if (st == MG_OK)
        st = shape_of(g, p->fp, p->weights, p->threads, &p->bufs.shape);
    if (st == MG_OK && o.timing) {
        p->timed = true;
        for (cudaEvent_t& ev : p->ev) {
            const cudaError_t e = cudaEventCreate(&ev);
            if (e != cudaSuccess && st == MG_OK) st = cuda_fail(e, "cudaEventCreate");
        }
    }
    if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    if (st != MG_OK) return st;
    *out = p.release();
    return MG_OK;
}

MG_API mg_status mg_query_plan_run(mg_query_plan* p, const int32_t* boxes, int64_t Q, void* out, size_t out_capacity,
                                   mg_stream stream) {
    MG_RANGE("mg_query_plan_run");
    using namespace mg;
    if (!p) return fail(MG_ERR_INVALID_ARG, "plan is NULL");
    if (Q < 0 || Q > p->max_Q) return fail(MG_ERR_INVALID_ARG, "Q must be in 0..max_Q");
    if (Q == 0) return MG_OK;
    if (!boxes || !out) return fail(MG_ERR_INVALID_ARG, "NULL argument");
    if ((uint64_t)out_capacity < (uint64_t)Q * p->g->S) return fail(MG_ERR_INVALID_ARG, "out_capacity must be >= Q*S");
    if (reinterpret_cast<uintptr_t>(boxes) % 4 || reinterpret_cast<uintptr_t>(out) % 4)
        return fail(MG_ERR_INVALID_ARG, "boxes and out must be 4-byte aligned");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != p->g->device) MG_CUDA(cudaSetDevice(p->g->device));
    mg_status st = MG_OK;
    if (p->timed) {
        const cudaError_t e = cudaEventRecord(p->ev[0], s);
        if (e != cudaSuccess) st = cuda_fail(e, "mg_query_plan_run");
    }
    const BatchRun run{boxes, Q, nullptr, nullptr, out};
    QueryBufs B = p->bufs;
    B.chunk = run_chunk(p, Q);
    if (st == MG_OK) st = enqueue_any(p->g, B, run, p->fp, p->weights, false, p->timed ? p->ev + 1 : nullptr, s);
    if (st == MG_OK) p->ran = true;
    if (prev >= 0 && prev != p->g->device) cudaSetDevice(prev);
    return st;
}

MG_API mg_status mg_query_plan_timing(const mg_query_plan* p, float* plan_ms, float* main_ms) {
    using namespace mg;
    if (!p || !plan_ms || !main_ms) return fail(MG_ERR_INVALID_ARG, "NULL argument");
    if (!p->timed) return fail(MG_ERR_INVALID_ARG, "plan created without opts->timing");
    if (!p->ran) return fail(MG_ERR_INVALID_ARG, "plan has not run");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != p->g->device) MG_CUDA(cudaSetDevice(p->g->device));
    cudaError_t e = cudaEventSynchronize(p->ev[2]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(plan_ms, p->ev[0], p->ev[1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(main_ms, p->ev[1], p->ev[2]);
    if (prev >= 0 && prev != p->g->device) cudaSetDevice(prev);
    if (e != cudaSuccess) return cuda_fail(e, "mg_query_plan_timing");
    return MG_OK;
}

MG_API void mg_query_plan_free(mg_query_plan* p) {
    if (!p) return;
    const int dev = p->g->device;
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
    cudaDeviceSynchronize();
    delete p;
    if (prev >= 0 && prev != dev) cudaSetDevice(prev);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Autotuner: time the batched query over work-chunk sizes and CTA sizes on the
// caller's own batch and keep the fastest for later calls on this graph.
// ---------------------------------------------------------------------------
extern "C" MG_API mg_status mg_query_autotune(mg_graph* g, const int32_t* boxes, int64_t Q, mg_query_opts* opts,
                                              float* best_ms, mg_stream stream) {
    MG_RANGE("mg_query_autotune");
    using namespace mg;
    if (!g || !opts) return fail(MG_ERR_INVALID_ARG, "NULL argument");
    if (Q < 1 || !boxes) return fail(MG_ERR_INVALID_ARG, "autotuning needs a non-empty batch");
    if (opts->hist_type != MG_HIST_U32 && opts->hist_type != MG_HIST_F32) return fail(MG_ERR_INVALID_ARG, "bad hist_type");
    if (g->quantised && opts->hist_type == MG_HIST_U32)
        return fail(MG_ERR_UNSUPPORTED, "a quantised graph has no exact weights: use MG_HIST_F32");
    const bool FP = opts->hist_type == MG_HIST_F32;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device) MG_CUDA(cudaSetDevice(g->device));
    mg_status st = MG_OK;
    Buf outb;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float best = 1e30f;
    int best_c = 0, best_t = 0;
    st = outb.alloc(&g->al, (size_t)Q * g->S * 4, s);
    if (st == MG_OK && (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess))
        st = fail(MG_ERR_CUDA, "cudaEventCreate");
    // 512 threads matter when one histogram per CTA fills shared memory
    // (many segments): two CTAs per SM then hold 32 warps instead of 8
    const int chunks[] = {1024, 2048, 4096, 8192, 16384};
    const int threads[] = {128, 256, 512};
    const int nc = (int)(sizeof(chunks) / sizeof(chunks[0])), nt = (int)(sizeof(threads) / sizeof(threads[0]));
    for (int ci = 0; st == MG_OK && ci < nc; ci++) {
        for (int ti = 0; st == MG_OK && ti < nt; ti++) {
            mg_query_opts o = *opts;
            o.layout = MG_LAYOUT_DENSE;
            o.schedule = MG_SCHED_BATCHED;
            o.chunk_cubes = chunks[ci];
            o.block_threads = threads[ti];
            o.timing = 0;
            float ms = 0.f;
            for (int rep = 0; st == MG_OK && rep < 3; rep++) {   // first run warms up
                cudaEventRecord(e0, s);
                st = query_boxes(g, boxes, Q, o, outb.p, (size_t)Q * g->S, nullptr, nullptr, nullptr, s);
                cudaEventRecord(e1, s);
                if (st == MG_OK && cudaEventSynchronize(e1) != cudaSuccess) st = fail(MG_ERR_CUDA, "autotune sync");
                float t = 0.f;
                if (st == MG_OK) cudaEventElapsedTime(&t, e0, e1);
                if (rep > 0) ms += t;
            }
            if (st == MG_OK && ms < best) {
                best = ms;
                best_c = chunks[ci];
                best_t = threads[ti];
            }
        }
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st == MG_OK) {
        g->tuned_chunk[FP ? 1 : 0] = best_c;
        g->tuned_threads[FP ? 1 : 0] = best_t;
        if (FP) g->tuned_weights = opts->alpha_dtype;
        opts->chunk_cubes = best_c;
        opts->block_threads = best_t;
        if (best_ms) *best_ms = best / 2.f;
    }
    if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    return st;
}

// Record a launch shape found earlier (for example, read from a cache file).
extern "C" MG_API mg_status mg_query_set_tuning(mg_graph* g, int hist_type, int chunk_cubes, int block_threads) {
    using namespace mg;
    if (!g) return fail(MG_ERR_INVALID_ARG, "graph is NULL");
    if (hist_type != MG_HIST_U32 && hist_type != MG_HIST_F32) return fail(MG_ERR_INVALID_ARG, "bad hist_type");
    if (chunk_cubes < 0 || (block_threads && block_threads != 128 && block_threads != 256 && block_threads != 512))
        return fail(MG_ERR_INVALID_ARG, "bad launch shape");
    g->tuned_chunk[hist_type] = chunk_cubes;
    g->tuned_threads[hist_type] = block_threads;
    if (hist_type == MG_HIST_F32) g->tuned_weights = -1;
    return MG_OK;
}

// mg_build.cu -- Mixture Graph construction on the GPU.
//
//  A1  Sec. 3.1, Eq. 4: normalised histogram mipmap.  Each level is a CSR of
//      (segment id, integer weight) lists, weight = 8^l * H; a parent's list is
//      the merge of its <= 8 children's lists scaled by 8/N, N the children in
//      support (1, 2, 4 or 8).  Count pass, scan, write pass per level.
//  A2  Sec. 3.2-3.3, Eq. 5-7: every list longer than one entry is factorised
//      into binary lerps, pairing positions (0,1),(2,3),... per round with an
//      odd last entry carried.  A lerp is the key (p, q, a, b) with a:b the
//      reduced weight ratio; a global open-addressing hash returns the existing
//      node for a key or publishes a new one (lock-free: the node row is written
//      first, then its index is CAS-ed into the slot).
//  A3  Sec. 3.4, Fig. 5: topological level = max(level of p, level of q) + 1;
//      nodes are renumbered in ascending (level, p', q', a, b) with p', q' the
//      new IDs of the predecessors, by a stable radix sort per level; bucket
//      offsets delimit the levels; mip IDs are rewritten.
#include "mg_internal.cuh"

#include <algorithm>
#include <vector>

namespace mg {
namespace {

struct Dims3 {
    int32_t x, y, z;
};

__host__ __device__ __forceinline__ int64_t nvox(Dims3 d) { return (int64_t)d.x * d.y * d.z; }

// ---------------------------------------------------------------------------
// level 0 checks and copy
// ---------------------------------------------------------------------------
template <typename IdT, typename OutT>
__global__ void copy_ids_kernel(const IdT* __restrict__ in, OutT* __restrict__ out, int64_t n, uint32_t S,
                                unsigned* __restrict__ status) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t v = (uint32_t)in[i];
        if (v >= S) {
            set_status(status, kStatBadInput);
            v = 0;
        }
        out[i] = (OutT)v;
    }
}

// ---------------------------------------------------------------------------
// A1: level 0 -> level 1 (sort <= 8 IDs per parent)
// ---------------------------------------------------------------------------
// the <= 8 IDs under a parent, ascending: a compare-exchange network on
// registers (an index into a local array would spill it), absent children as
// kNone, which sorts last
template <typename IdT>
__device__ __forceinline__ int gather_l0(const IdT* __restrict__ ids, Dims3 d0, int X, int Y, int Z, uint32_t (&v)[8]) {
    int n = 0;
    const bool x1 = 2 * X + 1 < d0.x;
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const int y = 2 * Y + (r & 1), z = 2 * Z + (r >> 1);
        v[2 * r] = v[2 * r + 1] = kNone;
        if (y < d0.y && z < d0.z) {
            const IdT* p = ids + ((int64_t)z * d0.y + y) * d0.x + 2 * X;
            v[2 * r] = (uint32_t)__ldg(p);
            n++;
            if (x1) {
                v[2 * r + 1] = (uint32_t)__ldg(p + 1);
                n++;
            }
        }
    }
    return n;
}

__device__ __forceinline__ void sort8(uint32_t (&v)[8]) {
    // Batcher's odd-even merge network for eight (19 exchanges)
    constexpr int A[19] = {0, 2, 4, 6, 0, 1, 4, 5, 1, 5, 0, 1, 2, 3, 2, 3, 1, 3, 5};
    constexpr int B[19] = {1, 3, 5, 7, 2, 3, 6, 7, 2, 6, 4, 5, 6, 7, 4, 5, 2, 4, 6};
#pragma unroll
    for (int k = 0; k < 19; k++) {
        const uint32_t lo = min(v[A[k]], v[B[k]]), hi = max(v[A[k]], v[B[k]]);
        v[A[k]] = lo;
        v[B[k]] = hi;
    }
}

// parent coordinates of voxel v (32-bit arithmetic: volumes hold < 2^32 voxels)
__device__ __forceinline__ void parent_at(uint32_t v, Dims3 d, int& X, int& Y, int& Z) {
    const uint32_t r = v / (uint32_t)d.x;
    X = (int)(v - r * (uint32_t)d.x);
    Z = (int)(r / (uint32_t)d.y);
    Y = (int)(r - (uint32_t)Z * (uint32_t)d.y);
}

template <typename IdT>
__global__ void l1_count_kernel(const IdT* __restrict__ ids, Dims3 d0, Dims3 d1, uint32_t* __restrict__ nnz) {
    const int64_t V1 = nvox(d1);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V1; v += (int64_t)gridDim.x * blockDim.x) {
        int X, Y, Z;
        parent_at((uint32_t)v, d1, X, Y, Z);
        uint32_t s[8];
        gather_l0(ids, d0, X, Y, Z, s);
        bool one = true;
#pragma unroll
        for (int a = 1; a < 8; a++) one = one && (s[a] == s[0] || s[a] == kNone);
        uint32_t c = 1;
        if (!one) {
            sort8(s);
#pragma unroll
            for (int a = 1; a < 8; a++) c += s[a] != s[a - 1] && s[a] != kNone;
        }
        nnz[v] = c;
    }
}

template <typename IdT>
__global__ void l1_write_kernel(const IdT* __restrict__ ids, Dims3 d0, Dims3 d1, const uint32_t* __restrict__ off,
                                uint32_t* __restrict__ out_ids, uint64_t* __restrict__ out_w) {
    const int64_t V1 = nvox(d1);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V1; v += (int64_t)gridDim.x * blockDim.x) {
        uint32_t o = off[v];
        int X, Y, Z;
        parent_at((uint32_t)v, d1, X, Y, Z);
        uint32_t s[8];
        const int n = gather_l0(ids, d0, X, Y, Z, s);
        if (off[v + 1] - o == 1) {
            out_ids[o] = s[0];
            out_w[o] = 8;   // n children of weight 8 / n
            continue;
        }
        const uint64_t scale = 8u / (unsigned)n;   // Eq. 4: divide by N, times 8^l
        sort8(s);
        uint32_t run = 1;
#pragma unroll
        for (int a = 1; a <= 8; a++) {
            if (a < 8 && s[a] == s[a - 1]) {
                run++;
                continue;
            }
            if (s[a - 1] != kNone) {
                out_ids[o] = s[a - 1];
                out_w[o] = (uint64_t)run * scale;
                o++;
            }
            run = 1;
        }
    }
}

// ---------------------------------------------------------------------------
// A1: level l -> level l+1 (merge <= 8 sorted child lists)
// ---------------------------------------------------------------------------
struct Heads {
    uint32_t pos[8], end[8], head[8];
    int n;
};

__device__ __forceinline__ void load_children(const uint32_t* __restrict__ off, const uint32_t* __restrict__ ids,
                                              Dims3 dl, int X, int Y, int Z, Heads& h) {
    h.n = 0;
#pragma unroll
    for (int k = 0; k < 2; k++)
#pragma unroll
        for (int j = 0; j < 2; j++)
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const int x = 2 * X + i, y = 2 * Y + j, z = 2 * Z + k;
                const int c = 4 * k + 2 * j + i;
                if (x < dl.x && y < dl.y && z < dl.z) {
                    const int64_t cv = ((int64_t)z * dl.y + y) * dl.x + x;
                    h.pos[c] = off[cv];
                    h.end[c] = off[cv + 1];
                    h.n++;
                } else {
                    h.pos[c] = 0;
                    h.end[c] = 0;
                }
                h.head[c] = h.pos[c] < h.end[c] ? ids[h.pos[c]] : kNone;
            }
}

__device__ __forceinline__ uint32_t heads_min(const Heads& h) {
    uint32_t m = kNone;
#pragma unroll
    for (int c = 0; c < 8; c++) m = min(m, h.head[c]);
    return m;
}

__global__ void next_count_kernel(const uint32_t* __restrict__ off, const uint32_t* __restrict__ ids, Dims3 dl,
                                  Dims3 dn, uint32_t* __restrict__ nnz) {
    const int64_t Vn = nvox(dn);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < Vn; v += (int64_t)gridDim.x * blockDim.x) {
        int X, Y, Z;
        parent_at((uint32_t)v, dn, X, Y, Z);
        Heads h;
        load_children(off, ids, dl, X, Y, Z, h);
        uint32_t cnt = 0;
        for (;;) {
            const uint32_t m = heads_min(h);
            if (m == kNone) break;
            cnt++;
#pragma unroll
            for (int c = 0; c < 8; c++) {
                if (h.head[c] == m) {
                    h.pos[c]++;
                    h.head[c] = h.pos[c] < h.end[c] ? ids[h.pos[c]] : kNone;
                }
            }
        }
        nnz[v] = cnt;
    }
}

__global__ void next_write_kernel(const uint32_t* __restrict__ off, const uint32_t* __restrict__ ids,
                                  const uint64_t* __restrict__ w, Dims3 dl, Dims3 dn,
                                  const uint32_t* __restrict__ noff, uint32_t* __restrict__ nids,
                                  uint64_t* __restrict__ nw) {
    const int64_t Vn = nvox(dn);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < Vn; v += (int64_t)gridDim.x * blockDim.x) {
        int X, Y, Z;
        parent_at((uint32_t)v, dn, X, Y, Z);
        Heads h;
        load_children(off, ids, dl, X, Y, Z, h);
        const uint64_t scale = 8u / (unsigned)h.n;   // Eq. 4
        uint32_t o = noff[v];
        for (;;) {
            const uint32_t m = heads_min(h);
            if (m == kNone) break;
            uint64_t sum = 0;
#pragma unroll
            for (int c = 0; c < 8; c++) {
                if (h.head[c] == m) {
                    sum += w[h.pos[c]];
                    h.pos[c]++;
                    h.head[c] = h.pos[c] < h.end[c] ? ids[h.pos[c]] : kNone;
                }
            }
            nids[o] = m;
            nw[o] = sum * scale;
            o++;
        }
    }
}

// The coarse levels: few parents with long lists.  A CTA sums the children's
// lists of one parent in a table of all segments in shared memory and reads it
// out in order (a thread merging eight lists of hundreds of entries takes
// about 150 ns an entry: the last five levels of 512x512x384 cost 440 us,
// this 78).  Taken for at most kDenseParents parents and segment counts whose
// table fits.
constexpr int kDenseThreads = 256;
constexpr int64_t kDenseParents = 2048;
constexpr uint32_t kDenseSegments = 24 * 1024;   // 192 KB of 64-bit sums

// the sums of parent v's children in `sum` (zeroed here); returns the children in support
__device__ __forceinline__ int dense_sum(const uint32_t* __restrict__ off, const uint32_t* __restrict__ ids,
                                         const uint64_t* __restrict__ w, Dims3 dl, int X, int Y, int Z, uint32_t S,
                                         unsigned long long* sum) {
    for (uint32_t s = threadIdx.x; s < S; s += kDenseThreads) sum[s] = 0;
    __syncthreads();
    int n = 0;
    for (int c = 0; c < 8; c++) {
        const int x = 2 * X + (c & 1), y = 2 * Y + ((c >> 1) & 1), z = 2 * Z + (c >> 2);
        if (x >= dl.x || y >= dl.y || z >= dl.z) continue;
        n++;
        const int64_t cv = ((int64_t)z * dl.y + y) * dl.x + x;
        const uint32_t e1 = off[cv + 1];
        for (uint32_t e = off[cv] + threadIdx.x; e < e1; e += kDenseThreads) atomicAdd(sum + ids[e], w[e]);
    }
    __syncthreads();
    return n;
}

// WRITE = false: entries of every parent's list; true: the lists
template <bool WRITE>
__global__ void __launch_bounds__(kDenseThreads) dense_next_kernel(const uint32_t* __restrict__ off,
                                                                   const uint32_t* __restrict__ ids,
                                                                   const uint64_t* __restrict__ w, Dims3 dl, Dims3 dn,
                                                                   uint32_t S, uint32_t* __restrict__ noff,
                                                                   uint32_t* __restrict__ nids,
                                                                   uint64_t* __restrict__ nw) {
    extern __shared__ __align__(16) unsigned long long s_sum[];
    __shared__ uint32_t s_warp[kDenseThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t Vn = nvox(dn);
    for (int64_t v = blockIdx.x; v < Vn; v += gridDim.x) {
        int X, Y, Z;
        parent_at((uint32_t)v, dn, X, Y, Z);
        const int n = dense_sum(off, ids, w, dl, X, Y, Z, S, s_sum);
        const uint64_t scale = 8u / (unsigned)n;   // Eq. 4
        uint32_t at = WRITE ? noff[v] : 0u;
        for (uint32_t s0 = 0; s0 < S; s0 += kDenseThreads) {
            const uint32_t s = s0 + threadIdx.x;
            const unsigned long long x = s < S ? s_sum[s] : 0ull;
            const unsigned m = __ballot_sync(0xffffffffu, x != 0);
            if (lane == 0) s_warp[warp] = __popc(m);
            __syncthreads();
            uint32_t before = 0, all = 0;
#pragma unroll
            for (int k = 0; k < kDenseThreads / 32; k++) {
                if (k < warp) before += s_warp[k];
                all += s_warp[k];
            }
            if (WRITE && x) {
                const uint32_t o = at + before + __popc(m & ((1u << lane) - 1u));
                nids[o] = s;
                nw[o] = x * scale;
            }
            at += all;
            __syncthreads();
        }
        if (!WRITE && threadIdx.x == 0) noff[v] = at;
    }
}

// ---------------------------------------------------------------------------
// A2: node table with lock-free hash pruning
// ---------------------------------------------------------------------------
struct NodeTab {
    uint32_t* p;
    uint32_t* q;
    uint64_t* a;
    uint64_t* b;
    uint8_t* depth;
    uint32_t* slots;       // node index or kNone
    uint64_t mask;         // slots - 1
    unsigned long long* count;
    uint64_t cap;
    unsigned* status;
};

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
    x ^= x >> 31;
    x *= 0x7fb5d329728ea185ull;
    x ^= x >> 27;
    x *= 0x81dadef4bc2dd44dull;
    x ^= x >> 33;
    return x;
}

__device__ __forceinline__ uint64_t key_hash(uint32_t p, uint32_t q, uint64_t a, uint64_t b) {
    return mix64(mix64(((uint64_t)p << 32 | q) ^ 0x9e3779b97f4a7c15ull) ^ a * 0xc2b2ae3d27d4eb4full ^
                 (b + 0x165667b19e3779f9ull) * 0x27d4eb2f165667c5ull);
}

__device__ __forceinline__ uint64_t gcd64(uint64_t u, uint64_t v) {
    if (u == 0) return v;
    if (v == 0) return u;
    const int shift = __ffsll((long long)(u | v)) - 1;
    u >>= __ffsll((long long)u) - 1;
    do {
        v >>= __ffsll((long long)v) - 1;
        if (u > v) {
            uint64_t t = u;
            u = v;
            v = t;
        }
        v -= u;
    } while (v);
    return u << shift;
}

__device__ __forceinline__ uint32_t gcd32(uint32_t u, uint32_t v) {
    if (u == 0) return v;
    if (v == 0) return u;
    const int shift = __ffs((int)(u | v)) - 1;
    u >>= __ffs((int)u) - 1;
    do {
        v >>= __ffs((int)v) - 1;
        const uint32_t lo = min(u, v);
        v = max(u, v) - lo;
        u = lo;
    } while (v);
    return u << shift;
}

// Eq. 5-6 with Sec. 3.3 re-use: node for the lerp of (p, wp) and (q, wq).
__device__ uint32_t node_get(const NodeTab& t, uint32_t p, uint32_t q, uint64_t wp, uint64_t wq) {
    if (p >= kDead || q >= kDead) return kNone;   // an earlier failure propagates
    uint64_t a, b;
    if (((wp | wq) >> 32) == 0) {   // nearly all: a fraction of the 64-bit steps' latency
        const uint32_t g = gcd32((uint32_t)wp, (uint32_t)wq);
        a = (uint32_t)wp / g;
        b = (uint32_t)wq / g;
    } else {
        const uint64_t g = gcd64(wp, wq);
        a = wp / g;
        b = wq / g;
    }
    uint64_t h = key_hash(p, q, a, b) & t.mask;
    uint32_t mine = kNone;
    for (uint64_t probe = 0; probe <= t.mask; probe++) {
        uint32_t s = ld_acquire_u32(t.slots + h);
        if (s == kNone) {
            if (mine == kNone) {
                const unsigned long long k = atomicAdd(t.count, 1ull);
                if (k >= t.cap) {
                    set_status(t.status, kStatCapacity);
                    return kNone;
                }
                mine = (uint32_t)k;
                t.p[mine] = p;
                t.q[mine] = q;
                t.a[mine] = a;
                t.b[mine] = b;
                // Sec. 3.4: topological level, the predecessors are complete
                const uint8_t dp = ld_relaxed_u8(t.depth + p), dq = ld_relaxed_u8(t.depth + q);
                t.depth[mine] = (uint8_t)(max(dp, dq) + 1);
                __threadfence();
            }
            const uint32_t old = atomicCAS(t.slots + h, kNone, mine);
            if (old == kNone) return mine;
            s = old;
            __threadfence();
        }
        if (ld_relaxed_u32(t.p + s) == p && ld_relaxed_u32(t.q + s) == q && ld_relaxed_u64(t.a + s) == a &&
            ld_relaxed_u64(t.b + s) == b) {
            if (mine != kNone) t.p[mine] = kDead;   // our unpublished row is never referenced
            return s;
        }
        h = (h + 1) & t.mask;
    }
    set_status(t.status, kStatCapacity);
    return kNone;
}

// Lists are factorised by a thread (up to kShortList entries), a warp (up to
// kWarpList) or a CTA: a round's pairs are independent, while a node costs a
// chain of dependent table accesses (2-4 us), so a thread that walked 16
// entries alone held its level up.
constexpr int kShortList = 4;
constexpr int64_t kWarpList = 256;
constexpr int kFactorThreads = 256;
constexpr int kFactorPer = 8;       // voxels per thread and block at most (one where a level has few)

// Lists of one entry are copied; the others of a block are gathered first, so
// that a warp's lanes factorise together (one voxel in seven of level 1 has
// more than one entry: nearly every warp held some).
__global__ void __launch_bounds__(kFactorThreads) factor_short_kernel(
    NodeTab t, const uint32_t* __restrict__ off, const uint32_t* __restrict__ ids, const uint64_t* __restrict__ w,
    int64_t V, uint32_t* __restrict__ mip_out, uint32_t* __restrict__ long_list, unsigned* __restrict__ long_count,
    unsigned* __restrict__ longest, int per) {
    __shared__ uint32_t s_list[kFactorThreads * kFactorPer];
    __shared__ unsigned s_count;
    unsigned most = 0;   // longest list seen (statistics)
    const int64_t span = (int64_t)kFactorThreads * per;
    for (int64_t base = (int64_t)blockIdx.x * span; base < V; base += (int64_t)gridDim.x * span) {
        if (threadIdx.x == 0) s_count = 0;
        __syncthreads();
        for (int k = 0; k < per; k++) {
            const int64_t v = base + k * kFactorThreads + threadIdx.x;
            if (v >= V) break;
            const uint32_t b = off[v], n = off[v + 1] - b;
            most = max(most, n);
            if (n == 1) mip_out[v] = ids[b];
            else if (n <= kShortList) s_list[atomicAdd(&s_count, 1u)] = (uint32_t)v;
            else long_list[atomicAdd(long_count, 1u)] = (uint32_t)v;
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < s_count; i += kFactorThreads) {
            const uint32_t v = s_list[i], b = off[v], n = off[v + 1] - b;
            const uint64_t w0 = w[b], w1 = w[b + 1];
            uint32_t r = node_get(t, ids[b], ids[b + 1], w0, w1);
            if (n == 3) {
                r = node_get(t, r, ids[b + 2], w0 + w1, w[b + 2]);
            } else if (n == 4) {
                const uint64_t w2 = w[b + 2], w3 = w[b + 3];
                const uint32_t r2 = node_get(t, ids[b + 2], ids[b + 3], w2, w3);
                r = node_get(t, r, r2, w0 + w1, w2 + w3);
            }
            mip_out[v] = r;
        }
        __syncthreads();
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0 && most > ld_relaxed_u32(longest)) atomicMax(longest, most);
}

// One warp (or CTA) per list; rounds in place in the level's CSR arrays (all
// reads of a round's slice happen before its writes, separated by a barrier).
// The warps pass the lists above kWarpList on to the CTAs.
template <bool CTA>
__global__ void __launch_bounds__(kFactorThreads) factor_long_kernel(NodeTab t, const uint32_t* __restrict__ off,
                                                                     uint32_t* ids, uint64_t* w,
                                                                     const uint32_t* __restrict__ list,
                                                                     const unsigned* __restrict__ count,
                                                                     uint32_t* __restrict__ next,
                                                                     unsigned* __restrict__ next_count,
                                                                     uint32_t* __restrict__ mip_out) {
    constexpr int G = CTA ? kFactorThreads : 32;   // threads on a list
    const int me = threadIdx.x % G;
    const unsigned groups = gridDim.x * (kFactorThreads / G), nlong = *count;
    auto sync = [] {
        if constexpr (CTA) __syncthreads();
        else __syncwarp();
    };
    for (unsigned i = blockIdx.x * (kFactorThreads / G) + threadIdx.x / G; i < nlong; i += groups) {
        const uint32_t v = list[i];
        const uint32_t b = off[v];
        int64_t n = (int64_t)(off[v + 1] - b);
        if (!CTA && n > kWarpList) {
            if (me == 0) next[atomicAdd(next_count, 1u)] = v;
            continue;
        }
        uint32_t* nd = ids + b;
        uint64_t* ww = w + b;
        while (n > 1) {
            const int64_t half = n / 2;
            for (int64_t base = 0; base < half; base += G) {
                const int64_t k = base + me;
                uint32_t n0 = 0, n1 = 0;
                uint64_t w0 = 0, w1 = 0;
                if (k < half) {
                    n0 = nd[2 * k];
                    n1 = nd[2 * k + 1];
                    w0 = ww[2 * k];
                    w1 = ww[2 * k + 1];
                }
                sync();
                if (k < half) {
                    nd[k] = node_get(t, n0, n1, w0, w1);
                    ww[k] = w0 + w1;
                }
                sync();
            }
            if (n & 1) {
                if (me == 0) {
                    nd[half] = nd[n - 1];
                    ww[half] = ww[n - 1];
                }
                sync();
            }
            n = (n + 1) / 2;
        }
        if (me == 0) mip_out[v] = nd[0];
        sync();
    }
}

__global__ void rehash_kernel(NodeTab t, uint64_t lo, uint64_t hi) {
    for (uint64_t k = lo + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < hi;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t p = t.p[k];
        if (p >= kDead) continue;
        uint64_t h = key_hash(p, t.q[k], t.a[k], t.b[k]) & t.mask;
        for (uint64_t probe = 0; probe <= t.mask; probe++) {
            if (atomicCAS(t.slots + h, kNone, (uint32_t)k) == kNone) break;
            h = (h + 1) & t.mask;
        }
    }
}

// ---------------------------------------------------------------------------
// A3: canonical relabel
// ---------------------------------------------------------------------------
// nodes per topological level, and the OR of each level's weights (the digits
// its sort has to look at)
struct LevelStats {
    unsigned long long count[MG_MAX_DEPTH + 1], weights[MG_MAX_DEPTH + 1];
};
__global__ void depth_hist_kernel(const uint32_t* __restrict__ p, const uint8_t* __restrict__ depth,
                                  const uint64_t* __restrict__ a, const uint64_t* __restrict__ b, uint64_t lo,
                                  uint64_t hi, LevelStats* __restrict__ st) {
    __shared__ unsigned int sh[MG_MAX_DEPTH + 1];
    __shared__ unsigned long long sw[MG_MAX_DEPTH + 1];
    for (int i = threadIdx.x; i <= MG_MAX_DEPTH; i += blockDim.x) {
        sh[i] = 0;
        sw[i] = 0;
    }
    __syncthreads();
    for (uint64_t k = lo + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < hi;
         k += (uint64_t)gridDim.x * blockDim.x) {
        if (p[k] < kDead) {
            const int d = min((int)depth[k], MG_MAX_DEPTH);
            atomicAdd(&sh[d], 1u);
            const unsigned long long w = a[k] | b[k];
            if (w & ~sw[d]) atomicOr(&sw[d], w);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= MG_MAX_DEPTH; i += blockDim.x)
        if (sh[i]) {
            atomicAdd(&st->count[i], (unsigned long long)sh[i]);
            atomicOr(&st->weights[i], sw[i]);
        }
}

// The nodes of each level gathered (in any order: the sort's key is unique).
// Places are handed out per CTA and level, not per node: a global atomic each
// on the same few cursors took 130 us for 230,000 nodes, this takes 5.
__global__ void __launch_bounds__(256) scatter_depth_kernel(const uint32_t* __restrict__ p,
                                                            const uint8_t* __restrict__ depth, uint64_t lo, uint64_t hi,
                                                            unsigned long long* __restrict__ cursor,
                                                            uint32_t* __restrict__ order) {
    __shared__ unsigned int sh[MG_MAX_DEPTH + 1];
    __shared__ unsigned long long s_base[MG_MAX_DEPTH + 1];
    for (uint64_t k0 = lo + (uint64_t)blockIdx.x * blockDim.x; k0 < hi; k0 += (uint64_t)gridDim.x * blockDim.x) {
        for (int i = threadIdx.x; i <= MG_MAX_DEPTH; i += blockDim.x) sh[i] = 0;
        __syncthreads();
        const uint64_t k = k0 + threadIdx.x;
        const bool live = k < hi && p[k] < kDead;
        const int d = live ? depth[k] : 0;
        unsigned at = 0;
        if (live) at = atomicAdd(&sh[d], 1u);
        __syncthreads();
        for (int i = threadIdx.x; i <= MG_MAX_DEPTH; i += blockDim.x)
            if (sh[i]) s_base[i] = atomicAdd(&cursor[i], (unsigned long long)sh[i]);
        __syncthreads();
        if (live) order[s_base[d] + at] = (uint32_t)k;
        __syncthreads();
    }
}

// key for the stable sort: field 0 = b, 1 = a, 2 = a<<sh | b, 3 = p'<<sh | q'
__global__ void sort_key_kernel(const uint32_t* __restrict__ perm, int64_t n, int field, int sh,
                                const uint32_t* __restrict__ p, const uint32_t* __restrict__ q,
                                const uint64_t* __restrict__ a, const uint64_t* __restrict__ b,
                                const uint32_t* __restrict__ canon, uint64_t* __restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = perm[i];
        uint64_t key;
        if (field == 0) key = b[k];
        else if (field == 1) key = a[k];
        else if (field == 2) key = a[k] << sh | b[k];
        else key = (uint64_t)canon[p[k]] << sh | canon[q[k]];
        keys[i] = key;
    }
}

__global__ void assign_kernel(const uint32_t* __restrict__ perm, int64_t n, uint32_t first,
                              const uint32_t* __restrict__ p, const uint32_t* __restrict__ q,
                              const uint64_t* __restrict__ a, const uint64_t* __restrict__ b,
                              uint32_t* __restrict__ canon, uint2* __restrict__ pq, ulonglong2* __restrict__ ab) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = perm[i];
        const uint32_t c = first + (uint32_t)i;
        canon[k] = c;
        pq[c] = make_uint2(canon[p[k]], canon[q[k]]);
        ab[c] = make_ulonglong2(a[k], b[k]);
    }
}

// The levels from `first` on, all of at most kTailMax nodes, sorted and
// numbered by one CTA, level after level (a level's key reads the numbers of
// the levels below it): bitonic in shared memory on the whole key (p', q', a,
// b).  The last levels hold a few nodes each, and a radix sort of any size
// costs some 60 launches a level: 84 sort passes of the 512x512x384 volume
// became 22, 1.27 -> 0.53 ms.
constexpr int kTailThreads = 1024;
constexpr int kTailMax = 4096;
struct TailLevels {
    int first, last;
    int64_t bucket[MG_MAX_DEPTH + 2];
};
struct TailKey {
    uint64_t pq, a, b;
};
constexpr size_t kTailSmem = (size_t)kTailMax * (sizeof(TailKey) + sizeof(uint32_t));

__global__ void __launch_bounds__(kTailThreads) sort_tail_kernel(TailLevels T, uint32_t S, const uint32_t* order,
                                                                 const uint32_t* __restrict__ p,
                                                                 const uint32_t* __restrict__ q,
                                                                 const uint64_t* __restrict__ a,
                                                                 const uint64_t* __restrict__ b, uint32_t* canon,
                                                                 uint2* __restrict__ pq, ulonglong2* __restrict__ ab) {
    extern __shared__ __align__(16) uint8_t smem[];
    TailKey* key = reinterpret_cast<TailKey*>(smem);
    uint32_t* idx = reinterpret_cast<uint32_t*>(key + kTailMax);
    for (int k = T.first; k <= T.last; k++) {
        const int n = (int)(T.bucket[k + 1] - T.bucket[k]);
        const uint32_t* perm = order + (T.bucket[k] - S);
        int m = 1;
        while (m < n) m *= 2;
        for (int i = threadIdx.x; i < m; i += kTailThreads) {
            idx[i] = (uint32_t)i;
            if (i < n) {
                const uint32_t t = perm[i];
                key[i] = TailKey{(uint64_t)canon[p[t]] << 32 | canon[q[t]], a[t], b[t]};
            } else {
                key[i] = TailKey{~0ull, ~0ull, ~0ull};
            }
        }
        __syncthreads();
        for (int w = 2; w <= m; w *= 2)
            for (int h = w / 2; h > 0; h /= 2) {
                for (int t = threadIdx.x; t < m / 2; t += kTailThreads) {
                    const int i = 2 * t - (t & (h - 1)), j = i + h;
                    const uint32_t x = idx[i], y = idx[j];
                    const TailKey &kx = key[x], &ky = key[y];
                    const bool more = kx.pq != ky.pq ? kx.pq > ky.pq : kx.a != ky.a ? kx.a > ky.a : kx.b > ky.b;
                    if (more == ((i & w) == 0)) {
                        idx[i] = y;
                        idx[j] = x;
                    }
                }
                __syncthreads();
            }
        for (int i = threadIdx.x; i < n; i += kTailThreads) {
            const uint32_t x = idx[i], t = perm[x], c = (uint32_t)T.bucket[k] + (uint32_t)i;
            canon[t] = c;
            pq[c] = make_uint2((uint32_t)(key[x].pq >> 32), (uint32_t)key[x].pq);
            ab[c] = make_ulonglong2(key[x].a, key[x].b);
        }
        __syncthreads();   // the next level's keys read these numbers
    }
}

__global__ void sources_kernel(uint32_t S, uint32_t* __restrict__ canon, uint2* __restrict__ pq,
                               ulonglong2* __restrict__ ab) {
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
        canon[s] = s;
        pq[s] = make_uint2(kNone, kNone);
        ab[s] = make_ulonglong2(0, 0);
    }
}

__global__ void remap_kernel(uint32_t* __restrict__ mip, int64_t n, const uint32_t* __restrict__ canon,
                             unsigned* __restrict__ status) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = mip[i];
        if (t >= kDead) {
            set_status(status, kStatCapacity);
            mip[i] = 0;
        } else {
            mip[i] = canon[t];
        }
    }
}

__global__ void weights_kernel(const ulonglong2* __restrict__ ab, int64_t N, uint32_t S, uint2* __restrict__ ab32,
                               float* __restrict__ alpha) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < (int64_t)S) {
            ab32[i] = make_uint2(0, 0);
            alpha[i] = 0.f;
            continue;
        }
        const ulonglong2 w = ab[i];
        const uint64_t s = w.x + w.y;
        ab32[i] = s < (1ull << 32) ? make_uint2((uint32_t)w.x, (uint32_t)w.y) : make_uint2(0, 0);
        alpha[i] = (float)((double)w.y / (double)s);   // weight of q, rounded to fp32
    }
}

// ---------------------------------------------------------------------------
// axis-major copies: copy 0 orders (x, y, z), copy 1 (y, z, x), copy 2
// (z, x, y); rows of `pitch` IDs, the ones past the row's end set to 0
// ---------------------------------------------------------------------------
// One job is one copy of one level; a launch runs a list of jobs, so the nine
// small levels of a volume cost one launch.  Copies 1 and 2 are batched 2-D
// transposes (x against the new fastest axis, one per index of the third
// axis) through a shared-memory tile, because x is the fast axis of the
// source and the slow or middle one of the copy: a thread-per-element copy
// read one ID per 32-byte sector.  HBM bound once both sides move whole rows:
// 512x512x384, both level-0 copies 1.04 -> 0.16 ms, levels >= 1 0.28 -> 0.07 ms.
struct AxisJob {
    const void* src;
    void* dst;
    int64_t tile0;            // first tile of the job in the launch
    int32_t x, y, z;          // dims of the level
    int32_t copy, pitch;
    int32_t tx, tf;           // tiles along x (copy 0: parts of a row) and along the copy's fastest axis (rows)
};
constexpr int kMaxJobs = 3 * MG_MAX_LEVELS;
struct AxisJobs {
    int n;
    int64_t tiles;
    AxisJob job[kMaxJobs];
};

constexpr int kTransThreads = 256;
// tile edge: 64 two-byte or 32 four-byte IDs, 128 bytes of a row on both sides
template <typename T> constexpr int trans_edge() { return 128 / (int)sizeof(T); }

template <typename T>
__global__ void __launch_bounds__(kTransThreads) transpose_kernel(const __grid_constant__ AxisJobs J) {
    constexpr int E = trans_edge<T>();
    constexpr int PW = 4 / (int)sizeof(T);   // IDs per 4-byte word
    // one spare word per row: a column read then meets every bank (two lanes
    // per bank for the two-byte IDs, whose words hold two columns)
    __shared__ __align__(4) T tile[E][E + PW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t b = blockIdx.x; b < J.tiles; b += gridDim.x) {
        int j = 0;
        while (j + 1 < J.n && J.job[j + 1].tile0 <= b) j++;
        const AxisJob& A = J.job[j];
        const uint32_t t = (uint32_t)(b - A.tile0);   // < 2^32 tiles: a tile holds at least one ID
        const uint32_t ix = t % (uint32_t)A.tx, r = t / (uint32_t)A.tx;
        const uint32_t jf = r % (uint32_t)A.tf, o = r / (uint32_t)A.tf;
        const int x0 = (int)ix * E, f0 = (int)jf * E;
        const int nf = A.copy == 1 ? A.y : A.z;
        // source: ID (x, f, o) at o * so + f * sf + x; copy: at x * dx + o * dn + f
        const int64_t sf = A.copy == 1 ? A.x : (int64_t)A.x * A.y, so = A.copy == 1 ? (int64_t)A.x * A.y : A.x;
        const int64_t dx = A.copy == 1 ? (int64_t)A.z * A.pitch : A.pitch;
        const int64_t dn = A.copy == 1 ? A.pitch : (int64_t)A.x * A.pitch;
        const T* src = static_cast<const T*>(A.src) + (int64_t)o * so;
        T* dst = static_cast<T*>(A.dst) + (int64_t)o * dn;
        const bool even = PW == 1 || (A.x % 2 == 0);   // two-byte rows readable as words
        constexpr int N = E / (kTransThreads / 32);     // rows per warp, all in flight
        const int x = x0 + lane * PW;
        uint32_t w[N];
        if (even) {
#pragma unroll
            for (int k = 0; k < N; k++) {
                const int f = f0 + warp + k * (kTransThreads / 32);
                w[k] = 0;
                if (f < nf && x < A.x) w[k] = __ldcs(reinterpret_cast<const uint32_t*>(src + (int64_t)f * sf + x));
            }
        } else {
#pragma unroll
            for (int k = 0; k < N; k++) {
                const int f = f0 + warp + k * (kTransThreads / 32);
                const T* p = src + (int64_t)f * sf + x;
                w[k] = 0;
                if (f < nf && x < A.x) w[k] = (uint32_t)__ldcs(p) | (x + 1 < A.x ? (uint32_t)__ldcs(p + 1) << 16 : 0u);
            }
        }
#pragma unroll
        for (int k = 0; k < N; k++)
            *reinterpret_cast<uint32_t*>(&tile[warp + k * (kTransThreads / 32)][lane * PW]) = w[k];
        __syncthreads();
        const bool words = PW == 1 || (A.pitch % 2 == 0);
        const int f = lane * PW;
#pragma unroll
        for (int k = 0; k < N; k++) {
            const int c = warp + k * (kTransThreads / 32);
            if (x0 + c >= A.x || f0 + f >= A.pitch) continue;
            T* p = dst + (int64_t)(x0 + c) * dx + f0 + f;
            if constexpr (PW == 1) {
                *p = tile[f][c];
            } else {
                const uint32_t u = (uint32_t)tile[f][c] | (uint32_t)tile[f + 1][c] << 16;
                if (words) {
                    *reinterpret_cast<uint32_t*>(p) = u;
                } else {
                    p[0] = (T)u;
                    if (f0 + f + 1 < A.pitch) p[1] = (T)(u >> 16);
                }
            }
        }
        __syncthreads();
    }
}

// copy 0: the x-fastest rows re-spaced to their pitch, one warp for kRowPart of
// a row (a volume of one row, 60,000 voxels long: 408 -> 19 us)
constexpr int kRowPart = 1024;
template <typename T>
__global__ void __launch_bounds__(kTransThreads) repitch_kernel(const __grid_constant__ AxisJobs J) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (kTransThreads / 32);
    for (int64_t b = (int64_t)blockIdx.x * (kTransThreads / 32) + (threadIdx.x >> 5); b < J.tiles; b += warps) {
        int j = 0;
        while (j + 1 < J.n && J.job[j + 1].tile0 <= b) j++;
        const AxisJob& A = J.job[j];
        const uint32_t t = (uint32_t)(b - A.tile0);   // < 2^32: a part holds at least one ID
        const int64_t row = t / (uint32_t)A.tx;
        const int f0 = (int)(t - (uint32_t)row * (uint32_t)A.tx) * kRowPart, f1 = min(f0 + kRowPart, A.pitch);
        const T* src = static_cast<const T*>(A.src) + row * A.x;
        T* dst = static_cast<T*>(A.dst) + row * A.pitch;
        for (int f = f0 + lane; f < f1; f += 32) dst[f] = f < A.x ? __ldcs(src + f) : T(0);
    }
}

// ---------------------------------------------------------------------------
// host orchestration
// ---------------------------------------------------------------------------
struct HostTable {
    Buf p, q, a, b, depth, slots;
    uint64_t cap = 0, nslots = 0;
    Buf count;   // unsigned long long
};

unsigned grid_n(int64_t n, int threads = 256) { return grid_for(n, threads, 152 * 64); }

mg_status grow_table(HostTable& t, uint64_t need, uint64_t used, const Alloc& al, cudaStream_t s) {
    if (need <= t.cap) return MG_OK;
    uint64_t ncap = std::max<uint64_t>(need, t.cap * 2);
    if (ncap >= (uint64_t)kDead) return fail(MG_ERR_UNSUPPORTED, "more than 2^32-2 nodes");
    Buf np, nq, na, nb, nd;
    MG_TRY(np.alloc(&al, ncap * 4, s));
    MG_TRY(nq.alloc(&al, ncap * 4, s));
    MG_TRY(na.alloc(&al, ncap * 8, s));
    MG_TRY(nb.alloc(&al, ncap * 8, s));
    MG_TRY(nd.alloc(&al, ncap, s));
    if (used) {
        MG_CUDA(cudaMemcpyAsync(np.p, t.p.p, used * 4, cudaMemcpyDeviceToDevice, s));
        MG_CUDA(cudaMemcpyAsync(nq.p, t.q.p, used * 4, cudaMemcpyDeviceToDevice, s));
        MG_CUDA(cudaMemcpyAsync(na.p, t.a.p, used * 8, cudaMemcpyDeviceToDevice, s));
        MG_CUDA(cudaMemcpyAsync(nb.p, t.b.p, used * 8, cudaMemcpyDeviceToDevice, s));
        MG_CUDA(cudaMemcpyAsync(nd.p, t.depth.p, used, cudaMemcpyDeviceToDevice, s));
    }
    t.p = std::move(np);
    t.q = std::move(nq);
    t.a = std::move(na);
    t.b = std::move(nb);
    t.depth = std::move(nd);
    t.cap = ncap;
    uint64_t ns = 1024;
    while (ns < 2 * ncap) ns <<= 1;
    if (ns != t.nslots) {
        MG_TRY(t.slots.alloc(&al, ns * 4, s));
        MG_CUDA(cudaMemsetAsync(t.slots.p, 0xFF, ns * 4, s));
        t.nslots = ns;
    }
    return MG_OK;
}

NodeTab view(HostTable& t, unsigned* status) {
    NodeTab v;
    v.p = t.p.as<uint32_t>();
    v.q = t.q.as<uint32_t>();
    v.a = t.a.as<uint64_t>();
    v.b = t.b.as<uint64_t>();
    v.depth = t.depth.as<uint8_t>();
    v.slots = t.slots.as<uint32_t>();
    v.mask = t.nslots - 1;
    v.count = t.count.as<unsigned long long>();
    v.cap = t.cap;
    v.status = status;
    return v;
}

template <typename T>
mg_status read_scalar(T* host, const void* dev, cudaStream_t s) {
    MG_CUDA(cudaMemcpyAsync(host, dev, sizeof(T), cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    return MG_OK;
}

int bits_for(uint64_t maxval) {
    int b = 0;
    while (b < 64 && (maxval >> b)) b++;
    return b;
}

}  // namespace

mg_status build_graph(mg_graph* g, const void* ids, int id_bytes, int64_t nx, int64_t ny, int64_t nz,
                      cudaStream_t s) {
    const Alloc& al = g->al;
    const uint32_t S = g->S;
    LevelGeom& G = g->geom;

    // ---- Eq. 4 level geometry: round up until 1^3 ----
    int64_t d[3] = {nx, ny, nz};
    int L = 0;
    for (;;) {
        if (L >= MG_MAX_LEVELS) return fail(MG_ERR_UNSUPPORTED, "too many mip levels");
        for (int k = 0; k < 3; k++) G.dims[L][k] = (int32_t)d[k];
        L++;
        if (d[0] == 1 && d[1] == 1 && d[2] == 1) break;
        for (int k = 0; k < 3; k++) d[k] = (d[k] + 1) / 2;
    }
    G.L = g->L = L;
    auto dims_of = [&](int l) { return Dims3{G.dims[l][0], G.dims[l][1], G.dims[l][2]}; };
    int64_t total_hi = 0;
    G.off[0] = 0;
    for (int l = 1; l < L; l++) {
        G.off[l] = total_hi;
        total_hi += nvox(dims_of(l));
    }

    MG_TRY(g->status.alloc(&al, sizeof(unsigned), s));
    MG_CUDA(cudaMemsetAsync(g->status.p, 0, sizeof(unsigned), s));
    unsigned* status = g->status.as<unsigned>();

    // ---- level 0: the IDs themselves (lossless, Sec. 3.4) ----
    const int64_t V0 = nx * ny * nz;
    g->id0_bytes = S <= 65536u ? 2 : 4;
    MG_TRY(g->mip0.alloc(&al, (size_t)V0 * g->id0_bytes, s));
    {
        const unsigned gb = grid_n(V0);
        if (id_bytes == 2 && g->id0_bytes == 2)
            copy_ids_kernel<uint16_t, uint16_t><<<gb, 256, 0, s>>>((const uint16_t*)ids, g->mip0.as<uint16_t>(), V0, S, status);
        else if (id_bytes == 2)
            copy_ids_kernel<uint16_t, uint32_t><<<gb, 256, 0, s>>>((const uint16_t*)ids, g->mip0.as<uint32_t>(), V0, S, status);
        else if (g->id0_bytes == 2)
            copy_ids_kernel<uint32_t, uint16_t><<<gb, 256, 0, s>>>((const uint32_t*)ids, g->mip0.as<uint16_t>(), V0, S, status);
        else
            copy_ids_kernel<uint32_t, uint32_t><<<gb, 256, 0, s>>>((const uint32_t*)ids, g->mip0.as<uint32_t>(), V0, S, status);
        MG_CUDA(cudaGetLastError());
        unsigned bits = 0;
        MG_TRY(read_scalar(&bits, status, s));
        if (bits & kStatBadInput) return fail(MG_ERR_INVALID_ARG, "a segment ID is >= num_segments");
    }

    // ---- node table: sources 0..S-1 ----
    HostTable t;
    MG_TRY(t.count.alloc(&al, 2 * sizeof(unsigned long long), s));   // nodes; entries of the newest lists
    {
        const unsigned long long c0[2] = {S, 0};
        MG_CUDA(cudaMemcpyAsync(t.count.p, c0, sizeof(c0), cudaMemcpyHostToDevice, s));
    }
    MG_TRY(grow_table(t, (uint64_t)S + 4096, 0, al, s));
    MG_CUDA(cudaMemsetAsync(t.p.p, 0xFF, (size_t)S * 4, s));
    MG_CUDA(cudaMemsetAsync(t.q.p, 0xFF, (size_t)S * 4, s));
    MG_CUDA(cudaMemsetAsync(t.a.p, 0, (size_t)S * 8, s));
    MG_CUDA(cudaMemsetAsync(t.b.p, 0, (size_t)S * 8, s));
    MG_CUDA(cudaMemsetAsync(t.depth.p, 0, (size_t)S, s));
    uint64_t used = S;

    if (total_hi > 0) MG_TRY(g->mip.alloc(&al, (size_t)total_hi * 4, s));
    Buf maxlen;
    MG_TRY(maxlen.alloc(&al, sizeof(unsigned), s));
    MG_CUDA(cudaMemsetAsync(maxlen.p, 0, sizeof(unsigned), s));
    Buf long_list, huge_list, long_count;   // counts: warp lists, CTA lists
    MG_TRY(long_count.alloc(&al, 2 * sizeof(unsigned), s));

    // ---- A1 + A2, level by level ----
    struct Lists {
        Buf off, ids, w;
        int64_t V = 0;
        uint32_t nnz = 0;
    };
    // the newest lists' entries and the node count, in one read-back
    unsigned long long counts[2] = {S, 0};
    auto read_counts = [&](Lists& out) -> mg_status {
        MG_CUDA(cudaMemcpyAsync(t.count.as<unsigned long long>() + 1, out.off.as<uint32_t>() + out.V, sizeof(uint32_t),
                                cudaMemcpyDeviceToDevice, s));
        MG_TRY(read_scalar(&counts, t.count.p, s));
        out.nnz = (uint32_t)counts[1];
        return MG_OK;
    };
    auto make_level1 = [&](Lists& out) -> mg_status {
        const Dims3 d0 = dims_of(0), d1 = dims_of(1);
        out.V = nvox(d1);
        MG_TRY(out.off.alloc(&al, (size_t)(out.V + 1) * 4, s));
        const unsigned gb = grid_n(out.V);
        if (g->id0_bytes == 2)
            l1_count_kernel<uint16_t><<<gb, 256, 0, s>>>(g->mip0.as<uint16_t>(), d0, d1, out.off.as<uint32_t>());
        else
            l1_count_kernel<uint32_t><<<gb, 256, 0, s>>>(g->mip0.as<uint32_t>(), d0, d1, out.off.as<uint32_t>());
        MG_CUDA(cudaGetLastError());
        MG_TRY(scan_exclusive_u32(out.off.as<uint32_t>(), out.off.as<uint32_t>(), out.V,
                                  out.off.as<uint32_t>() + out.V, al, s));
        MG_TRY(read_counts(out));
        MG_TRY(out.ids.alloc(&al, (size_t)out.nnz * 4, s));
        MG_TRY(out.w.alloc(&al, (size_t)out.nnz * 8, s));
        if (g->id0_bytes == 2)
            l1_write_kernel<uint16_t><<<gb, 256, 0, s>>>(g->mip0.as<uint16_t>(), d0, d1, out.off.as<uint32_t>(),
                                                         out.ids.as<uint32_t>(), out.w.as<uint64_t>());
        else
            l1_write_kernel<uint32_t><<<gb, 256, 0, s>>>(g->mip0.as<uint32_t>(), d0, d1, out.off.as<uint32_t>(),
                                                         out.ids.as<uint32_t>(), out.w.as<uint64_t>());
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    };
    auto make_next = [&](const Lists& in, int l, Lists& out) -> mg_status {
        const Dims3 dl = dims_of(l), dn = dims_of(l + 1);
        out.V = nvox(dn);
        MG_TRY(out.off.alloc(&al, (size_t)(out.V + 1) * 4, s));
        const unsigned gb = grid_n(out.V);
        const bool dense = out.V <= kDenseParents && S <= kDenseSegments;
        const unsigned db = grid_for(out.V, 1, 152 * 2);
        const size_t dsm = (size_t)S * 8;
        if (dense) {
            MG_CUDA(cudaFuncSetAttribute(dense_next_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kDenseSegments * 8)));
            MG_CUDA(cudaFuncSetAttribute(dense_next_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kDenseSegments * 8)));
            dense_next_kernel<false><<<db, kDenseThreads, dsm, s>>>(in.off.as<uint32_t>(), in.ids.as<uint32_t>(),
                                                                     in.w.as<uint64_t>(), dl, dn, S,
                                                                     out.off.as<uint32_t>(), nullptr, nullptr);
        } else next_count_kernel<<<gb, 256, 0, s>>>(in.off.as<uint32_t>(), in.ids.as<uint32_t>(), dl, dn,
                                             out.off.as<uint32_t>());
        MG_CUDA(cudaGetLastError());
        MG_TRY(scan_exclusive_u32(out.off.as<uint32_t>(), out.off.as<uint32_t>(), out.V,
                                  out.off.as<uint32_t>() + out.V, al, s));
        MG_TRY(read_counts(out));
        MG_TRY(out.ids.alloc(&al, (size_t)out.nnz * 4, s));
        MG_TRY(out.w.alloc(&al, (size_t)out.nnz * 8, s));
        if (dense)
            dense_next_kernel<true><<<db, kDenseThreads, dsm, s>>>(in.off.as<uint32_t>(), in.ids.as<uint32_t>(),
                                                                    in.w.as<uint64_t>(), dl, dn, S,
                                                                    out.off.as<uint32_t>(), out.ids.as<uint32_t>(),
                                                                    out.w.as<uint64_t>());
        else next_write_kernel<<<gb, 256, 0, s>>>(in.off.as<uint32_t>(), in.ids.as<uint32_t>(), in.w.as<uint64_t>(), dl,
                                             dn, out.off.as<uint32_t>(), out.ids.as<uint32_t>(),
                                             out.w.as<uint64_t>());
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    };

    int64_t max_list = 1;
    Lists cur;
    if (L > 1) MG_TRY(make_level1(cur));
    for (int l = 1; l < L; l++) {
        Lists nxt;
        if (l + 1 < L) MG_TRY(make_next(cur, l, nxt));
        // factorise level l (in place on cur)
        const uint64_t pairs = (uint64_t)cur.nnz - (uint64_t)cur.V;
        g->pairs += (int64_t)pairs;
        if (pairs > 0) {
            // (the last level makes no further lists: read the count alone)
            if (l + 1 == L) MG_TRY(read_scalar(&counts[0], t.count.p, s));
            used = counts[0];
            const uint64_t old_slots = t.nslots;
            MG_TRY(grow_table(t, used + pairs, used, al, s));
            if (t.nslots != old_slots && used > S) {
                rehash_kernel<<<grid_n((int64_t)(used - S)), 256, 0, s>>>(view(t, status), S, used);
                MG_CUDA(cudaGetLastError());
            }
        }
        MG_CUDA(cudaMemsetAsync(long_count.p, 0, 2 * sizeof(unsigned), s));
        if (long_list.bytes < (size_t)cur.V * 4) MG_TRY(long_list.alloc(&al, (size_t)cur.V * 4, s));
        const size_t huge = ((size_t)cur.nnz / kWarpList + 1) * 4;   // lists above kWarpList at most
        if (huge_list.bytes < huge) MG_TRY(huge_list.alloc(&al, huge, s));
        uint32_t* mip_out = g->mip.as<uint32_t>() + G.off[l];
        unsigned* counts2 = long_count.as<unsigned>();
        const int per = (int)std::min<int64_t>(kFactorPer, std::max<int64_t>(1, cur.V / (kFactorThreads * 152 * 8)));
        factor_short_kernel<<<grid_for(cur.V, kFactorThreads * per, 152 * 8), kFactorThreads, 0, s>>>(
            view(t, status), cur.off.as<uint32_t>(), cur.ids.as<uint32_t>(), cur.w.as<uint64_t>(), cur.V, mip_out,
            long_list.as<uint32_t>(), counts2, maxlen.as<unsigned>(), per);
        MG_CUDA(cudaGetLastError());
        factor_long_kernel<false><<<152 * 8, kFactorThreads, 0, s>>>(
            view(t, status), cur.off.as<uint32_t>(), cur.ids.as<uint32_t>(), cur.w.as<uint64_t>(),
            long_list.as<uint32_t>(), counts2, huge_list.as<uint32_t>(), counts2 + 1, mip_out);
        MG_CUDA(cudaGetLastError());
        if (S > kWarpList && cur.nnz > kWarpList) {   // a list holds each segment once
            factor_long_kernel<true><<<152 * 4, kFactorThreads, 0, s>>>(
                view(t, status), cur.off.as<uint32_t>(), cur.ids.as<uint32_t>(), cur.w.as<uint64_t>(),
                huge_list.as<uint32_t>(), counts2 + 1, nullptr, nullptr, mip_out);
            MG_CUDA(cudaGetLastError());
        }
        cur = std::move(nxt);
    }
    {
        unsigned long long cnt = 0;
        MG_TRY(read_scalar(&cnt, t.count.p, s));
        used = std::min<uint64_t>(cnt, t.cap);
        unsigned bits = 0;
        MG_TRY(read_scalar(&bits, status, s));
        if (bits & kStatCapacity) return fail(MG_ERR_CAPACITY, "node table overflow during factorisation");
    }
    {
        unsigned ml = 1;
        MG_TRY(read_scalar(&ml, maxlen.p, s));
        max_list = std::max<int64_t>(1, ml);
    }
    g->max_list = max_list;

    // ---- A3: topological levels and canonical numbering ----
    Buf hist;
    MG_TRY(hist.alloc(&al, sizeof(LevelStats), s));
    MG_CUDA(cudaMemsetAsync(hist.p, 0, sizeof(LevelStats), s));
    if (used > S) {
        depth_hist_kernel<<<grid_n((int64_t)(used - S)), 256, 0, s>>>(t.p.as<uint32_t>(), t.depth.as<uint8_t>(),
                                                                       t.a.as<uint64_t>(), t.b.as<uint64_t>(), S, used,
                                                                       hist.as<LevelStats>());
        MG_CUDA(cudaGetLastError());
    }
    LevelStats stats;
    MG_CUDA(cudaMemcpyAsync(&stats, hist.p, sizeof(stats), cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    const unsigned long long (&hh)[MG_MAX_DEPTH + 1] = stats.count;
    if (hh[MG_MAX_DEPTH]) return fail(MG_ERR_UNSUPPORTED, "topological depth above the supported maximum");
    int D = 0;
    for (int k = 1; k < MG_MAX_DEPTH; k++)
        if (hh[k]) D = k;
    g->D = D;
    g->bucket[0] = 0;
    g->bucket[1] = S;
    for (int k = 1; k <= D; k++) g->bucket[k + 1] = g->bucket[k] + (int64_t)hh[k];
    const int64_t N = g->N = g->bucket[D + 1];
    const int64_t NI = N - S;

    MG_TRY(g->pq.alloc(&al, (size_t)N * sizeof(uint2), s));
    MG_TRY(g->ab.alloc(&al, (size_t)N * sizeof(ulonglong2), s));
    Buf canon;
    MG_TRY(canon.alloc(&al, (size_t)std::max<uint64_t>(used, 1) * 4, s));
    sources_kernel<<<grid_n(S), 256, 0, s>>>(S, canon.as<uint32_t>(), g->pq.as<uint2>(), g->ab.as<ulonglong2>());
    MG_CUDA(cudaGetLastError());
    if (NI > 0) {
        Buf order, cursor, keys;
        MG_TRY(order.alloc(&al, (size_t)NI * 4, s));
        MG_TRY(cursor.alloc(&al, (MG_MAX_DEPTH + 1) * sizeof(unsigned long long), s));
        MG_TRY(keys.alloc(&al, (size_t)NI * 8, s));
        unsigned long long hc[MG_MAX_DEPTH + 1] = {};
        for (int k = 1; k <= D; k++) hc[k] = (unsigned long long)(g->bucket[k] - S);
        MG_CUDA(cudaMemcpyAsync(cursor.p, hc, sizeof(hc), cudaMemcpyHostToDevice, s));
        scatter_depth_kernel<<<grid_n((int64_t)(used - S)), 256, 0, s>>>(t.p.as<uint32_t>(), t.depth.as<uint8_t>(), S,
                                                                          used, cursor.as<unsigned long long>(),
                                                                          order.as<uint32_t>());
        MG_CUDA(cudaGetLastError());
        const int bits_n = bits_for((uint64_t)N);
        // the levels from `tail` on are small: sorted by one CTA after the loop
        int tail = D + 1;
        while (tail > 1 && g->bucket[tail] - g->bucket[tail - 1] <= kTailMax) tail--;
        for (int k = 1; k < tail; k++) {
            const int bits_ab = std::max(1, bits_for(stats.weights[k]));
            const int64_t n = g->bucket[k + 1] - g->bucket[k];
            uint32_t* perm = order.as<uint32_t>() + (g->bucket[k] - S);
            uint64_t* kk = keys.as<uint64_t>();
            auto key_pass = [&](int field, int sh, int bits) -> mg_status {
                sort_key_kernel<<<grid_n(n), 256, 0, s>>>(perm, n, field, sh, t.p.as<uint32_t>(), t.q.as<uint32_t>(),
                                                          t.a.as<uint64_t>(), t.b.as<uint64_t>(),
                                                          canon.as<uint32_t>(), kk);
                MG_CUDA(cudaGetLastError());
                return radix_sort_pairs(kk, perm, n, bits, al, s);
            };
            if (2 * bits_ab <= 64) {
                MG_TRY(key_pass(2, bits_ab, 2 * bits_ab));
            } else {
                MG_TRY(key_pass(0, 0, bits_ab));
                MG_TRY(key_pass(1, 0, bits_ab));
            }
            MG_TRY(key_pass(3, bits_n, 2 * bits_n));
            assign_kernel<<<grid_n(n), 256, 0, s>>>(perm, n, (uint32_t)g->bucket[k], t.p.as<uint32_t>(),
                                                    t.q.as<uint32_t>(), t.a.as<uint64_t>(), t.b.as<uint64_t>(),
                                                    canon.as<uint32_t>(), g->pq.as<uint2>(), g->ab.as<ulonglong2>());
            MG_CUDA(cudaGetLastError());
        }
        if (tail <= D) {
            TailLevels T;
            T.first = tail;
            T.last = D;
            for (int k = 0; k < MG_MAX_DEPTH + 2; k++) T.bucket[k] = g->bucket[k];
            MG_CUDA(cudaFuncSetAttribute(sort_tail_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem));
            sort_tail_kernel<<<1, kTailThreads, kTailSmem, s>>>(T, S, order.as<uint32_t>(), t.p.as<uint32_t>(),
                                                                t.q.as<uint32_t>(), t.a.as<uint64_t>(),
                                                                t.b.as<uint64_t>(), canon.as<uint32_t>(),
                                                                g->pq.as<uint2>(), g->ab.as<ulonglong2>());
            MG_CUDA(cudaGetLastError());
        }
    }
    if (total_hi > 0) {
        remap_kernel<<<grid_n(total_hi), 256, 0, s>>>(g->mip.as<uint32_t>(), total_hi, canon.as<uint32_t>(), status);
        MG_CUDA(cudaGetLastError());
    }
    MG_TRY(build_query_copies(g, s));
    MG_TRY(g->ab32.alloc(&al, (size_t)N * sizeof(uint2), s));
    MG_TRY(g->alpha.alloc(&al, (size_t)N * sizeof(float), s));
    weights_kernel<<<grid_n(N), 256, 0, s>>>(g->ab.as<ulonglong2>(), N, S, g->ab32.as<uint2>(), g->alpha.as<float>());
    MG_CUDA(cudaGetLastError());
    MG_TRY(build_lut(g, s));
    MG_TRY(build_tiles(g, s));
    unsigned bits = 0;
    MG_TRY(read_scalar(&bits, status, s));
    if (bits) return fail(MG_ERR_CAPACITY, "node table overflow during the build");
    MG_CUDA(cudaMemsetAsync(status, 0, sizeof(unsigned), s));
    return MG_OK;
}

// The padded axis-major copies of the box queries (copy c of level l: rows
// of the copy's fastest axis, qpitch[l][c] IDs apart, a multiple of 32 bytes
// unless that would take a copy past 2^32 IDs).
mg_status build_query_copies(mg_graph* g, cudaStream_t s) {
    const int L = g->L;
    auto dims_of = [&](int l) {
        Dims3 d;
        d.x = g->geom.dims[l][0];
        d.y = g->geom.dims[l][1];
        d.z = g->geom.dims[l][2];
        return d;
    };
    int64_t hi_total[3] = {0, 0, 0};
    for (int c = 0; c < 3; c++) {
        for (int l = 0; l < L; l++) {
            const Dims3 d = dims_of(l);
            const int64_t d0 = c == 0 ? d.x : c == 1 ? d.y : d.z;
            const int64_t rows = nvox(d) / d0;
            const int64_t per32 = l == 0 ? 32 / g->id0_bytes : 8;
            int64_t pitch = (d0 + per32 - 1) / per32 * per32;
            if (pitch * rows >= (1ll << 32)) pitch = d0;
            g->qpitch[l][c] = (int32_t)pitch;
            if (l >= 1) {
                g->qoff[l][c] = hi_total[c];
                hi_total[c] += pitch * rows;
            }
        }
    }
    // jobs[0]: copy 0 (rows); jobs[1]: copies 1 and 2 (tiles); level 0 and the
    // levels >= 1 apart, as their IDs differ in size
    AxisJobs jobs[2][2] = {};
    auto add = [&](AxisJobs& J, int l, int c, const void* src, void* dst, int edge) {
        AxisJob& A = J.job[J.n++];
        const Dims3 d = dims_of(l);
        A.src = src;
        A.dst = dst;
        A.tile0 = J.tiles;
        A.x = d.x;
        A.y = d.y;
        A.z = d.z;
        A.copy = c;
        A.pitch = g->qpitch[l][c];
        A.tx = c == 0 ? (A.pitch + kRowPart - 1) / kRowPart : (d.x + edge - 1) / edge;
        A.tf = c == 0 ? d.y : (A.pitch + edge - 1) / edge;
        J.tiles += (int64_t)A.tx * A.tf * (c == 2 ? d.y : d.z);
    };
    for (int c = 0; c < 3; c++) {
        const Dims3 d0 = dims_of(0);
        const int64_t pitch0 = g->qpitch[0][c];
        if (c > 0 || pitch0 != d0.x) {
            const int64_t n = pitch0 * (nvox(d0) / (c == 0 ? d0.x : c == 1 ? d0.y : d0.z));
            MG_TRY(g->mip0x[c].alloc(&g->al, (size_t)n * g->id0_bytes, s));
            add(jobs[c > 0][0], 0, c, g->mip0.p, g->mip0x[c].p, 128 / g->id0_bytes);
        }
        if (hi_total[c] > 0) {
            MG_TRY(g->mipx[c].alloc(&g->al, (size_t)hi_total[c] * 4, s));
            for (int l = 1; l < L; l++)
                add(jobs[c > 0][1], l, c, g->mip.as<uint32_t>() + g->geom.off[l],
                    g->mipx[c].as<uint32_t>() + g->qoff[l][c], 32);
        }
    }
    for (int hi = 0; hi < 2; hi++) {
        const bool wide = hi == 1 || g->id0_bytes == 4;
        const AxisJobs& R = jobs[0][hi];
        if (R.tiles > 0) {
            const unsigned gb = grid_for((R.tiles + 7) / 8, 1, 152 * 32);
            if (wide) repitch_kernel<uint32_t><<<gb, kTransThreads, 0, s>>>(R);
            else repitch_kernel<uint16_t><<<gb, kTransThreads, 0, s>>>(R);
            MG_CUDA(cudaGetLastError());
        }
        const AxisJobs& X = jobs[1][hi];
        if (X.tiles > 0) {
            const unsigned gb = grid_for(X.tiles, 1, 152 * 64);
            if (wide) transpose_kernel<uint32_t><<<gb, kTransThreads, 0, s>>>(X);
            else transpose_kernel<uint16_t><<<gb, kTransThreads, 0, s>>>(X);
            MG_CUDA(cudaGetLastError());
        }
    }
    return MG_OK;
}

}  // namespace mg

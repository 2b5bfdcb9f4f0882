// mg_propagate.cu -- forward transfer-function propagation (Sec. 3.4, Sec. 4).
//
// Sources take the TF row of their segment; then, level by level (nodes of a
// level are contiguous and independent), every node lerps the rows of its two
// predecessors:  v = v_p + alpha * (v_q - v_p), fp32.  Node records are SoA:
// (p, q) as one 8-byte load, alpha as 4 (or 2) bytes.
//
// An item is one vector (16 or 8 bytes) of one node's row, so neighbouring
// threads read and write whole rows however long they are (a thread per row
// took one 16-byte piece of 32 different rows per load: 8 RGBA TFs of a
// 217,000-node graph 104 -> 29 us).
//
// One persistent launch covers all levels: CTAs take tiles of items from a
// global ticket in level order, and a tile first waits until every tile of the
// wave before it has signalled (a counter per wave).  Tiles are handed out in
// order, so every tile waited on belongs to a CTA that is already running: the
// wait always ends.  It is bounded all the same; past the bound the kernel
// records MG_ERR_TIMEOUT and returns.  Waves: the sources and, for fp32 RGBA,
// level 1, whose nodes read the transfer function itself, so that the largest
// level waits for nothing; then one level each; the last levels, a few nodes
// each, are one tile, whose CTA walks them with no hand-off but its own barrier.
//
// Rows are gathered through L1 (nodes of a level are ordered by predecessor, so
// neighbours share rows): a CTA has acquired a wave's counter before it reads
// the wave's rows, which orders its plain loads after the stores and drops
// older lines.  The read-only path (ld.global.nc) is for the node table only.
#include "mg_internal.cuh"

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace mg {
namespace {

template <typename T> struct Cvt;
template <> struct Cvt<float> {
    static __device__ __forceinline__ float to(float x) { return x; }
    static __device__ __forceinline__ float from(float x) { return x; }
};
template <> struct Cvt<__half> {
    static __device__ __forceinline__ float to(__half x) { return __half2float(x); }
    static __device__ __forceinline__ __half from(float x) { return __float2half_rn(x); }
};
template <> struct Cvt<__nv_bfloat16> {
    static __device__ __forceinline__ float to(__nv_bfloat16 x) { return __bfloat162float(x); }
    static __device__ __forceinline__ __nv_bfloat16 from(float x) { return __float2bfloat16_rn(x); }
};

// One vector of E consecutive channels of a row, held as it is stored until
// the lerp: 16 or 8 bytes, or E elements where their size is neither.
template <typename ST, int E, int B = (int)sizeof(ST) * E> struct Vec {
    ST e[E];
    __device__ __forceinline__ void load(const ST* p) {
#pragma unroll
        for (int c = 0; c < E; c++) e[c] = p[c];
    }
    __device__ __forceinline__ void store(ST* p) const {
#pragma unroll
        for (int c = 0; c < E; c++) p[c] = e[c];
    }
    __device__ __forceinline__ float get(int c) const { return Cvt<ST>::to(e[c]); }
    __device__ __forceinline__ void set(int c, float x) { e[c] = Cvt<ST>::from(x); }
};
template <typename ST, int E, typename W> struct WideVec {
    union {
        W w;
        ST e[E];
    };
    __device__ __forceinline__ WideVec() {}
    __device__ __forceinline__ void load(const ST* p) { w = *reinterpret_cast<const W*>(p); }
    __device__ __forceinline__ void store(ST* p) const { *reinterpret_cast<W*>(p) = w; }
    __device__ __forceinline__ float get(int c) const { return Cvt<ST>::to(e[c]); }
    __device__ __forceinline__ void set(int c, float x) { e[c] = Cvt<ST>::from(x); }
};
template <typename ST, int E> struct Vec<ST, E, 16> : WideVec<ST, E, uint4> {};
template <typename ST, int E> struct Vec<ST, E, 8> : WideVec<ST, E, uint2> {};

// v_p + alpha (v_q - v_p) in fp32, rounded to the storage type
template <typename ST, int E>
__device__ __forceinline__ Vec<ST, E> lerp_vec(const Vec<ST, E>& p, const Vec<ST, E>& q, float al) {
    Vec<ST, E> out;
#pragma unroll
    for (int c = 0; c < E; c++) out.set(c, fmaf(al, q.get(c) - p.get(c), p.get(c)));
    return out;
}

// node weight: fp32 alpha, or a signed 16-bit alpha whose sign says p and q
// are swapped (alpha <= 1/2 after the swap; interpolation symmetry, Sec. 3.7)
template <typename ST> struct Weight {
    using T = ST;
};
template <> struct Weight<float> {
    using T = float;
};

constexpr int kPropThreads = 256;
constexpr int kPerThread = 2;                   // items of a tile per thread
constexpr int kTileItems = kPropThreads * kPerThread;
constexpr int kTailItems = 4 * kTileItems;      // levels up to this size may join the tail
constexpr unsigned kSpinLimit = 1u << 22;       // polls before a wait gives up

// elements of an item and items of a row: the row as 16-byte vectors, else as
// 8-byte ones, else whole
template <typename ST, int C> struct RowShape {
    static constexpr int B = (int)sizeof(ST) * C;
    static constexpr int E = B % 16 == 0 ? 16 / (int)sizeof(ST) : B % 8 == 0 ? 8 / (int)sizeof(ST) : C;
    static constexpr int items = C / E;
    static constexpr int tile_nodes = kTileItems / items;
    // resident CTAs: bound by load latency, as many as the registers allow
    // without spills (11.8 M nodes, f32 / f16 x 4 TFs: 112 / 210 us with 4, 114 /
    // 289 with 5, 118 / 202 with 3 of twice the items)
    static constexpr int min_ctas = E <= 4 ? 5 : 4;
};

// k transfer functions of cin channels each, TF j at tf + j * S * cin
struct TfRows {
    const float* tf;
    int64_t stride;   // S * cin
    int cin;
};

// segments of tiles in ticket order: the sources, the levels, the tail
enum { kSources = 0, kFromTf = 1, kFromRows = 2, kTail = 3 };
struct PropPlan {
    int segs;
    uint32_t tiles;
    uint32_t tile0[MG_MAX_DEPTH + 2];           // first tile of every segment (+ end)
    uint32_t first[MG_MAX_DEPTH + 1];           // first node
    uint32_t count[MG_MAX_DEPTH + 1];           // nodes
    int8_t kind[MG_MAX_DEPTH + 1];
    int8_t wave[MG_MAX_DEPTH + 1];
    uint32_t wave_tiles[MG_MAX_DEPTH + 1];      // tiles of every wave
    int tail_first, tail_last;                  // levels of the tail
    uint32_t bucket[MG_MAX_DEPTH + 2];
};

struct PropArgs {
    const uint2* pq;
    const void* alpha;
    TfRows F;
    void* vals;
    unsigned* sync;        // words kLine apart: ticket, CTAs that have left, signalled tiles of every wave; zero between launches
    unsigned* status;
};
// each word has a 128-byte line of its own: the polls of one wave's counter do
// not meet the ticket's atomics
constexpr int kLine = kPropLine, kSyncWords = kPropWords;

// Poll *p (acquire) until it reaches `need`: at once for the first polls, then
// with pauses; bounded like bounded_wait_geq.
__device__ __forceinline__ bool wave_wait(const unsigned* p, unsigned need, unsigned* status) {
    for (int i = 0; i < 32; i++)
        if (ld_acquire_u32(p) >= need) return true;
    return bounded_wait_geq(p, need, kSpinLimit, status);
}

// p and q in the order of the lerp (16-bit weights: sign = swapped)
__device__ __forceinline__ uint2 lerp_order(uint2 e, float al) { return al < 0.f ? make_uint2(e.y, e.x) : e; }

template <typename ST, int C>
__global__ void __launch_bounds__(kPropThreads, RowShape<ST, C>::min_ctas) propagate_kernel(const __grid_constant__ PropPlan T,
                                                                 const __grid_constant__ PropArgs A) {
    using R = RowShape<ST, C>;
    using WT = typename Weight<ST>::T;
    constexpr int E = R::E, I = R::items, TN = R::tile_nodes;
    using V = Vec<ST, E>;
    constexpr int NT = kPerThread;
    __shared__ unsigned s_next[2];
    __shared__ int s_abort;
    ST* vals = static_cast<ST*>(A.vals);
    const WT* __restrict__ alpha = static_cast<const WT*>(A.alpha);
    unsigned* ticket = A.sync;
    unsigned* done = A.sync + 2 * kLine;
    const unsigned total = T.tiles;
    // thread 0 holds the ticket after next, taken two tiles ahead so that the
    // atomic's round trip is never waited on
    unsigned ahead = 0;
    int seen = 0;        // every wave below this one is known to be complete
    int pending = -1;    // wave of the finished tile that is not yet signalled
    unsigned turn = 0;
    if (threadIdx.x == 0) {
        s_next[1] = atomicAdd(ticket, 1u);
        ahead = atomicAdd(ticket, 1u);
        s_abort = 0;
    }
    __syncthreads();
    unsigned t = s_next[1];
    // thread 0, once every thread of the CTA has stored its part of the tile
    auto signal = [&]() {
        if (threadIdx.x == 0 && pending >= 0) {
            __threadfence();
            atomicAdd(done + pending * kLine, 1u);
        }
        pending = -1;
    };
    auto segment = [&](unsigned tile) {
        int d = 0;
        while (tile >= T.tile0[d + 1]) d++;
        return d;
    };
    // item k of this thread in tile `tile` of segment d: node (past the end: none) and vector
    auto item = [&](int d, unsigned tile, int k, uint32_t& n, int& ch) {
        const uint32_t i = k * kPropThreads + threadIdx.x, r = i / I;
        ch = (int)(i - r * I);
        const uint32_t at = (tile - T.tile0[d]) * TN + r;
        n = T.first[d] + at;
        return r < TN && at < T.count[d];
    };
    auto edges = [&](unsigned tile, uint2 (&e)[NT], WT (&al)[NT]) {
        const int d = tile < total ? segment(tile) : 0;
        const bool live = tile < total && (T.kind[d] == kFromTf || T.kind[d] == kFromRows);
#pragma unroll
        for (int k = 0; k < NT; k++) {
            uint32_t n;
            int ch;
            e[k] = make_uint2(0u, 0u);
            al[k] = WT(0.f);
            if (live && item(d, tile, k, n, ch)) {   // (nothing here waits for the loads)
                e[k] = __ldg(A.pq + n);
                al[k] = alpha[n];
            }
        }
    };
    // Software pipeline over tiles: the next tile's ticket is known and its
    // (static) edges and weights are loaded while this tile waits and runs.
    // Tickets are taken in order and a tile only waits for smaller ones, so
    // the smallest unfinished ticket is always some CTA's current tile.
    uint2 e[NT];
    WT al[NT];
    edges(t, e, al);
    while (t < total) {
        const int d = segment(t);
        const int kind = T.kind[d], w = T.wave[d];
        if (w > seen) {   // wave w - 1 not yet seen complete; it may lack this CTA's last tile
            __syncthreads();
            signal();
            if (threadIdx.x == 0 && !wave_wait(done + (w - 1) * kLine, T.wave_tiles[w - 1], A.status)) s_abort = 1;
            seen = w;
        }
        if (threadIdx.x == 0) {
            s_next[turn] = ahead;
            ahead = atomicAdd(ticket, 1u);
        }
        // one barrier a tile: the last tile is stored, the next ticket known,
        // the wave's rows acquired
        __syncthreads();
        if (s_abort) break;
        const unsigned tn = s_next[turn];
        turn ^= 1u;
        uint2 en[NT];
        WT aln[NT];
        edges(tn, en, aln);
        if (kind == kSources) {
#pragma unroll
            for (int k = 0; k < NT; k++) {
                uint32_t n;
                int ch;
                if (item(d, t, k, n, ch)) {
                    V v;
                    for (int c = 0; c < E; c++) {
                        const int j = (ch * E + c) / A.F.cin;
                        v.set(c, __ldg(A.F.tf + j * A.F.stride + (int64_t)n * A.F.cin + (ch * E + c - j * A.F.cin)));
                    }
                    v.store(vals + (int64_t)n * C + ch * E);
                }
            }
        } else if (kind == kTail) {
            signal();
            for (int l = T.tail_first; l <= T.tail_last; l++) {
                const uint32_t lo = T.bucket[l];
                const int items = (int)(T.bucket[l + 1] - lo) * I;
                for (int i = (int)threadIdx.x; i < items; i += kPropThreads) {
                    const int r = i / I, ch = i - r * I;
                    const float a = Cvt<WT>::to(alpha[lo + r]);
                    const uint2 x = lerp_order(__ldg(A.pq + lo + r), a);
                    V p, q;
                    p.load(vals + (int64_t)x.x * C + ch * E);
                    q.load(vals + (int64_t)x.y * C + ch * E);
                    lerp_vec<ST, E>(p, q, fabsf(a)).store(vals + (int64_t)(lo + r) * C + ch * E);
                }
                __syncthreads();   // the next level reads these rows
            }
        } else {
            // both predecessor vectors of every item are loaded before any is
            // stored (nodes of one level never read each other)
            const ST* rows = vals;
            int64_t pitch = C, tf_ch = E;   // elements between rows, and between a row's vectors
            if (std::is_same<ST, float>::value && kind == kFromTf) {
                rows = reinterpret_cast<const ST*>(A.F.tf);
                pitch = E;
                tf_ch = A.F.stride;
            }
            V p[NT], q[NT];   // (loaded before the last tile's signal, whose fence takes as long)
#pragma unroll
            for (int k = 0; k < NT; k++) {
                uint32_t n;
                int ch;
                if (item(d, t, k, n, ch)) {
                    const uint2 x = lerp_order(e[k], Cvt<WT>::to(al[k]));
                    p[k].load(rows + (int64_t)x.x * pitch + ch * tf_ch);
                    q[k].load(rows + (int64_t)x.y * pitch + ch * tf_ch);
                }
            }
            signal();
#pragma unroll
            for (int k = 0; k < NT; k++) {
                uint32_t n;
                int ch;
                if (item(d, t, k, n, ch))
                    lerp_vec<ST, E>(p[k], q[k], fabsf(Cvt<WT>::to(al[k]))).store(vals + (int64_t)n * C + ch * E);
            }
        }
        signal();
        pending = w;
        t = tn;
#pragma unroll
        for (int k = 0; k < NT; k++) {
            e[k] = en[k];
            al[k] = aln[k];
        }
    }
    __syncthreads();
    signal();
    // The last CTA to leave (no other reads or writes the words any more)
    // zeroes them for the next launch on this stream.
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(A.sync + kLine, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last)
        for (int i = threadIdx.x; i < kSyncWords / kLine; i += kPropThreads) A.sync[i * kLine] = 0u;
}

__global__ void alpha16_kernel(const ulonglong2* __restrict__ ab, int64_t N, uint32_t S, int bf16,
                               void* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.f;
        if (i >= (int64_t)S) {
            const ulonglong2 w = ab[i];
            const double s = (double)w.x + (double)w.y;
            // alpha = b/(a+b); above 1/2 store -(a/(a+b)) meaning "swap p and q"
            v = (w.y <= w.x) ? (float)((double)w.y / s) : -(float)((double)w.x / s);
        }
        if (bf16)
            static_cast<__nv_bfloat16*>(out)[i] = __float2bfloat16_rn(v);
        else
            static_cast<__half*>(out)[i] = __float2half_rn(v);
    }
}

// the same from fp32 weights (quantised graphs: no exact a, b)
__global__ void alpha16_from_f32_kernel(const float* __restrict__ alpha, int64_t N, uint32_t S, int bf16,
                                        void* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.f;
        if (i >= (int64_t)S) {
            const float w = alpha[i];
            v = w <= 0.5f ? w : -(1.0f - w);
        }
        if (bf16)
            static_cast<__nv_bfloat16*>(out)[i] = __float2bfloat16_rn(v);
        else
            static_cast<__half*>(out)[i] = __float2half_rn(v);
    }
}

int sm_count_prop(int dev) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

template <typename ST, int C>
mg_status run(mg_graph* g, const float* tf, int cin, const void* alpha, ST* vals, cudaStream_t s) {
    using R = RowShape<ST, C>;
    PropPlan T;
    T.segs = 0;
    T.tiles = 0;
    int waves = 0;
    auto add = [&](int kind, int wave, int64_t first, int64_t count, int64_t tiles) {
        const int d = T.segs++;
        T.kind[d] = (int8_t)kind;
        T.wave[d] = (int8_t)wave;
        T.first[d] = (uint32_t)first;
        T.count[d] = (uint32_t)count;
        T.tile0[d] = T.tiles;
        T.tiles += (uint32_t)tiles;
        if (wave == waves) T.wave_tiles[waves++] = 0;
        T.wave_tiles[wave] += (uint32_t)tiles;
    };
    auto tiles_of = [](int64_t nodes) { return (nodes + R::tile_nodes - 1) / R::tile_nodes; };
    // the levels after which none is larger than kTailItems
    int tail = g->D + 1;
    while (tail > 2 && (g->bucket[tail] - g->bucket[tail - 1]) * R::items <= kTailItems) tail--;
    for (int d = 0; d <= g->D + 1; d++) T.bucket[d] = (uint32_t)g->bucket[d];
    // level 1 from the transfer function: rows of four floats on 16 bytes, the
    // vectors of a row one TF apart
    const bool quad = std::is_same<ST, float>::value && R::E == 4 && cin == 4 && aligned(tf, 16);
    for (int d = 0; d < tail && d <= g->D; d++) {
        const int64_t n = g->bucket[d + 1] - g->bucket[d];
        const bool from_tf = d == 1 && quad;
        add(d == 0 ? kSources : from_tf ? kFromTf : kFromRows, from_tf ? 0 : d == 0 ? 0 : waves, g->bucket[d], n,
            tiles_of(n));
    }
    T.tail_first = tail;
    T.tail_last = g->D;
    if (tail <= g->D) add(kTail, waves, g->bucket[tail], g->bucket[g->D + 1] - g->bucket[tail], 1);
    T.tile0[T.segs] = T.tiles;
    PropArgs A;
    A.pq = g->pq.as<uint2>();
    A.alpha = alpha;
    A.F = TfRows{tf, (int64_t)g->S * cin, cin};
    A.vals = vals;
    A.status = g->status.as<unsigned>();
    Buf own;
    MG_TRY(prop_sync_words(g, s, own, &A.sync));
    auto k = propagate_kernel<ST, C>;
    static std::atomic<int> per_sm{0};   // of this kernel (one architecture)
    int per = per_sm.load(std::memory_order_relaxed);
    if (per == 0) {
        MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kPropThreads, 0));
        per_sm.store(std::max(per, 1), std::memory_order_relaxed);
    }
    const int64_t grid = std::min<int64_t>(T.tiles, (int64_t)std::max(per, 1) * sm_count_prop(g->device));
    k<<<(unsigned)std::max<int64_t>(grid, 1), kPropThreads, 0, s>>>(T, A);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

template <typename ST>
mg_status dispatch_c(mg_graph* g, const float* tf, int C, int cin, const void* alpha, void* vals, cudaStream_t s) {
    ST* v = static_cast<ST*>(vals);
    switch (C) {
        case 1: return run<ST, 1>(g, tf, cin, alpha, v, s);
        case 2: return run<ST, 2>(g, tf, cin, alpha, v, s);
        case 3: return run<ST, 3>(g, tf, cin, alpha, v, s);
        case 4: return run<ST, 4>(g, tf, cin, alpha, v, s);
        case 5: return run<ST, 5>(g, tf, cin, alpha, v, s);
        case 6: return run<ST, 6>(g, tf, cin, alpha, v, s);
        case 7: return run<ST, 7>(g, tf, cin, alpha, v, s);
        case 8: return run<ST, 8>(g, tf, cin, alpha, v, s);
        case 12: return run<ST, 12>(g, tf, cin, alpha, v, s);
        case 16: return run<ST, 16>(g, tf, cin, alpha, v, s);
        case 20: return run<ST, 20>(g, tf, cin, alpha, v, s);
        case 24: return run<ST, 24>(g, tf, cin, alpha, v, s);
        case 28: return run<ST, 28>(g, tf, cin, alpha, v, s);
        case 32: return run<ST, 32>(g, tf, cin, alpha, v, s);
        default: break;
    }
    return fail(MG_ERR_UNSUPPORTED, "channels per node (k * C) must be 1-8, 12, 16, 20, 24, 28 or 32");
}

}  // namespace

mg_status ensure_alpha16(mg_graph* g, mg_dtype dt, cudaStream_t s) {
    Buf& b = dt == MG_BF16 ? g->alphab16 : g->alpha16;
    std::lock_guard<std::mutex> lk(g->alpha16_mu);   // until the weights are there: other threads read them at once
    if (b.p) return MG_OK;
    if (is_capturing(s))
        return fail(MG_ERR_CUDA, "the first call with 16-bit weights makes them and cannot be captured");
    Buf made;
    MG_TRY(made.alloc(&g->al, (size_t)g->N * 2, s));
    if (g->quantised)
        alpha16_from_f32_kernel<<<grid_for(g->N, 256, 152 * 32), 256, 0, s>>>(g->alpha.as<float>(), g->N, g->S,
                                                                              dt == MG_BF16, made.p);
    else
        alpha16_kernel<<<grid_for(g->N, 256, 152 * 32), 256, 0, s>>>(g->ab.as<ulonglong2>(), g->N, g->S,
                                                                    dt == MG_BF16, made.p);
    MG_CUDA(cudaGetLastError());
    MG_CUDA(cudaStreamSynchronize(s));
    made.s = nullptr;
    b = std::move(made);
    return MG_OK;
}

// ---------------------------------------------------------------------------
// Self-test of the bounded wait: one thread waits, with the propagation's
// helper, on a word that is either already set or that nothing ever sets.
// ---------------------------------------------------------------------------
namespace {
__device__ unsigned g_selftest_words[2];   // [0] the awaited flag, [1] the status word

__global__ void selftest_wait_kernel(unsigned limit) {
    if (threadIdx.x == 0 && blockIdx.x == 0) bounded_wait_geq(&g_selftest_words[0], 1u, limit, &g_selftest_words[1]);
}
}  // namespace

mg_status selftest_wait(bool satisfied, unsigned limit, cudaStream_t s) {
    const unsigned init[2] = {satisfied ? 1u : 0u, 0u};
    MG_CUDA(cudaMemcpyToSymbolAsync(g_selftest_words, init, sizeof(init), 0, cudaMemcpyHostToDevice, s));
    selftest_wait_kernel<<<1, 32, 0, s>>>(limit);
    MG_CUDA(cudaGetLastError());
    unsigned words[2] = {0, 0};
    MG_CUDA(cudaMemcpyFromSymbolAsync(words, g_selftest_words, sizeof(words), 0, cudaMemcpyDeviceToHost, s));
    MG_CUDA(cudaStreamSynchronize(s));
    return status_from_bits(words[1]);
}

mg_status propagate_multi(mg_graph* g, const float* tf, int k, int C, mg_dtype storage, void* vals, cudaStream_t s) {
    const int CT = k * C;
    const size_t esz = storage == MG_F32 ? 4 : 2;
    const size_t row = esz * (size_t)CT;
    if (row % 16 == 0 ? !aligned(vals, 16) : row % 8 == 0 ? !aligned(vals, 8) : false)
        return fail(MG_ERR_INVALID_ARG, "vals must be aligned to 16 bytes (rows of a multiple of 16 bytes) or 8");
    if (storage == MG_F32) return dispatch_c<float>(g, tf, CT, C, g->alpha.p, vals, s);
    MG_TRY(ensure_alpha16(g, storage, s));
    if (storage == MG_F16) return dispatch_c<__half>(g, tf, CT, C, g->alpha16.p, vals, s);
    return dispatch_c<__nv_bfloat16>(g, tf, CT, C, g->alphab16.p, vals, s);
}

mg_status propagate(mg_graph* g, const float* tf, int C, mg_dtype storage, void* vals, cudaStream_t s) {
    return propagate_multi(g, tf, 1, C, storage, vals, s);
}

}  // namespace mg

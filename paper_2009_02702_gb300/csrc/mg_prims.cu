// mg_prims.cu -- device-wide exclusive scan and stable LSD radix sort.
//
// Scan: reduce-then-scan over tiles of 2048 elements (256 threads x 8), the
// per-tile partial sums scanned recursively.  Sort: 8-bit digits, one
// histogram, one scan and one scatter per digit; ranks inside a tile are made
// stable with warp match + per-warp digit counts in shared memory.  Sorts of at
// most kSmallTiles tiles are bound by the latency of those launches: there the
// scatter sums the tiles' counts itself and counts the digits of the next pass
// as it places each element, one launch a digit (176,000 and 57,000 pairs, 11
// digits each: 445 us and 66 launches before, 305 us and 24 launches now).
#include "mg_internal.cuh"

namespace mg {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// exclusive prefix of v over the block; *block_total receives the sum
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* wsum, T* block_total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T x = warp_incl_scan(v, lane);
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? wsum[lane] : T(0);
        w = warp_incl_scan(w, lane);
        wsum[lane] = w;
    }
    __syncthreads();
    T pre = warp > 0 ? wsum[warp - 1] : T(0);
    *block_total = wsum[nw - 1];
    return pre + x - v;
}

template <typename T>
__global__ void scan_reduce_kernel(const T* __restrict__ in, int64_t n, T* __restrict__ partial) {
    __shared__ T wsum[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (idx < n) s += in[idx];
    }
    T tot;
    block_excl_scan(s, wsum, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <typename T>
__global__ void scan_tile_kernel(const T* in, T* out, int64_t n, const T* __restrict__ partial_ex,
                                 T* __restrict__ total) {
    __shared__ T tile[kScanTile];
    __shared__ T wsum[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
        tile[i * kScanThreads + threadIdx.x] = idx < n ? in[idx] : T(0);
    }
    __syncthreads();
    T loc[kScanItems];
    T sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        loc[i] = tile[threadIdx.x * kScanItems + i];
        sum += loc[i];
    }
    T bt;
    T ex = block_excl_scan(sum, wsum, &bt);
    const T off = partial_ex ? partial_ex[blockIdx.x] : T(0);
    T run = ex + off;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        tile[threadIdx.x * kScanItems + i] = run;
        run += loc[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
        if (idx < n) out[idx] = tile[i * kScanThreads + threadIdx.x];
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = off + bt;
}

// A few tiles in one CTA of 1,024 threads, 16 consecutive counters per thread
// and tile, with a running carry: one launch where the reduce-then-scan takes
// three (and the gaps between them), so it is taken up to 64 K counters.
constexpr int kOneThreads = 1024;
constexpr int kOneItems = 16;
constexpr int64_t kOneMax = 1 << 16;
__global__ void __launch_bounds__(kOneThreads) scan_one_kernel(const uint32_t* in, uint32_t* out, int64_t n,
                                                               uint32_t* __restrict__ total) {
    __shared__ uint32_t wsum[32];
    uint32_t carry = 0;
    for (int64_t base = 0; base < n; base += kOneThreads * kOneItems) {
        const int64_t at = base + (int64_t)threadIdx.x * kOneItems;
        uint32_t x[kOneItems], sum = 0;
        if (at + kOneItems <= n) {
#pragma unroll
            for (int k = 0; k < kOneItems / 4; k++) {
                const uint4 u = *reinterpret_cast<const uint4*>(in + at + 4 * k);
                x[4 * k] = u.x;
                x[4 * k + 1] = u.y;
                x[4 * k + 2] = u.z;
                x[4 * k + 3] = u.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < kOneItems; k++) x[k] = at + k < n ? in[at + k] : 0u;
        }
#pragma unroll
        for (int k = 0; k < kOneItems; k++) sum += x[k];
        uint32_t bt;
        uint32_t run = carry + block_excl_scan(sum, wsum, &bt);
        carry += bt;
#pragma unroll
        for (int k = 0; k < kOneItems; k++) {
            const uint32_t v = x[k];
            x[k] = run;
            run += v;
        }
        if (at + kOneItems <= n) {
#pragma unroll
            for (int k = 0; k < kOneItems / 4; k++)
                *reinterpret_cast<uint4*>(out + at + 4 * k) = make_uint4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]);
        } else {
#pragma unroll
            for (int k = 0; k < kOneItems; k++)
                if (at + k < n) out[at + k] = x[k];
        }
        __syncthreads();   // wsum is reused
    }
    if (total && threadIdx.x == 0) *total = carry;
}

template <typename T>
mg_status scan_impl(const T* in, T* out, int64_t n, T* total, const Alloc& al, cudaStream_t s) {
    if (n <= 0) {
        if (total) MG_CUDA(cudaMemsetAsync(total, 0, sizeof(T), s));
        return MG_OK;
    }
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        scan_tile_kernel<T><<<1, kScanThreads, 0, s>>>(in, out, n, nullptr, total);
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    if (n <= kOneMax && sizeof(T) == 4 && reinterpret_cast<uintptr_t>(in) % 16 == 0 &&
        reinterpret_cast<uintptr_t>(out) % 16 == 0) {
        scan_one_kernel<<<1, kOneThreads, 0, s>>>(reinterpret_cast<const uint32_t*>(in),
                                                            reinterpret_cast<uint32_t*>(out), n,
                                                            reinterpret_cast<uint32_t*>(total));
        MG_CUDA(cudaGetLastError());
        return MG_OK;
    }
    Buf part, part_ex;
    MG_TRY(part.alloc(&al, (size_t)nb * sizeof(T), s));
    MG_TRY(part_ex.alloc(&al, (size_t)nb * sizeof(T), s));
    scan_reduce_kernel<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, part.as<T>());
    MG_CUDA(cudaGetLastError());
    MG_TRY(scan_impl<T>(part.as<T>(), part_ex.as<T>(), nb, nullptr, al, s));
    scan_tile_kernel<T><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, part_ex.as<T>(), total);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

// ---------------------------------------------------------------------------
// radix sort
// ---------------------------------------------------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kSortWarps = kSortThreads / 32;

// small sorts: tiles at most, 1 KiB of counts each that every tile reads
constexpr int kSmallTiles = 128;

// counts of tile b's digits, digit d at hist[d * ds + b * bs]
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) rs_hist_kernel(const uint64_t* __restrict__ keys, int64_t n, int shift,
                                                               uint32_t* __restrict__ hist, int64_t ds, int64_t bs) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortThreads * ITEMS;
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
        int64_t idx = base + (int64_t)i * kSortThreads + threadIdx.x;
        if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[threadIdx.x * ds + blockIdx.x * bs] = h[threadIdx.x];
}

// SMALL = false: offs holds the scanned counts, digit-major.  SMALL = true:
// offs holds this pass's counts, a tile's 256 together; next (null in the last
// pass) receives those of the pass at next_shift, zero before the launch.
template <int ITEMS, bool SMALL>
__global__ void __launch_bounds__(kSortThreads) rs_scatter_kernel(
    const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, int64_t n, int shift,
    const uint32_t* __restrict__ offs, int64_t nb, uint64_t* __restrict__ kout, uint32_t* __restrict__ vout,
    uint32_t* __restrict__ next, int next_shift) {
    constexpr uint32_t TILE = kSortThreads * ITEMS;
    __shared__ uint32_t running[256];
    __shared__ uint32_t wcnt[kSortWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (SMALL) {
        // thread d: elements of digit d in all tiles, and in the tiles before this one
        __shared__ uint32_t wsum[32];
        uint32_t all = 0, before = 0;
#pragma unroll 16
        for (int b = 0; b < (int)nb; b++) {
            const uint32_t c = __ldg(offs + (size_t)b * 256 + threadIdx.x);
            all += c;
            before += b < (int)blockIdx.x ? c : 0u;
        }
        uint32_t total;
        running[threadIdx.x] = block_excl_scan(all, wsum, &total) + before;
    } else {
        running[threadIdx.x] = offs[(int64_t)threadIdx.x * nb + blockIdx.x];
    }
    const unsigned lt = (1u << lane) - 1u;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    for (int i = 0; i < ITEMS; i++) {
#pragma unroll
        for (int w = 0; w < kSortWarps; w++) wcnt[w][threadIdx.x] = 0;
        __syncthreads();
        const int64_t idx = base + (int64_t)i * kSortThreads + threadIdx.x;
        const bool valid = idx < n;
        uint64_t k = valid ? kin[idx] : 0;
        uint32_t v = valid ? vin[idx] : 0;
        const uint32_t digit = valid ? (uint32_t)((k >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, digit);
        const uint32_t rank = __popc(peers & lt);
        if (valid && lane == __ffs(peers) - 1) wcnt[warp][digit] = __popc(peers);
        __syncthreads();
        {
            uint32_t s = running[threadIdx.x];
#pragma unroll
            for (int w = 0; w < kSortWarps; w++) {
                uint32_t c = wcnt[w][threadIdx.x];
                wcnt[w][threadIdx.x] = s;
                s += c;
            }
            running[threadIdx.x] = s;
        }
        __syncthreads();
        if (valid) {
            const uint32_t pos = wcnt[warp][digit] + rank;
            kout[pos] = k;
            vout[pos] = v;
            if (SMALL && next) atomicAdd(next + (pos / TILE) * 256u + (uint32_t)((k >> next_shift) & 255u), 1u);
        }
        __syncthreads();
    }
}

// the passes of a sort of at most kSmallTiles tiles; *in_second: the result
// lies in the second pair of buffers
template <int ITEMS>
mg_status small_sort(uint64_t* keys, uint32_t* vals, uint64_t* keys2, uint32_t* vals2, int64_t n, int bits,
                     const Alloc& al, cudaStream_t s, bool* in_second) {
    const int64_t nb = (n + kSortThreads * ITEMS - 1) / (kSortThreads * ITEMS);
    const int passes = (bits + 7) / 8;
    Buf hist;   // the tiles' counts of every pass
    MG_TRY(hist.alloc(&al, (size_t)passes * nb * 256 * sizeof(uint32_t), s));
    uint32_t* h = hist.as<uint32_t>();
    if (passes > 1) MG_CUDA(cudaMemsetAsync(h + nb * 256, 0, (size_t)(passes - 1) * nb * 256 * sizeof(uint32_t), s));
    rs_hist_kernel<ITEMS><<<(unsigned)nb, kSortThreads, 0, s>>>(keys, n, 0, h, 1, 256);
    MG_CUDA(cudaGetLastError());
    for (int p = 0; p < passes; p++) {
        const bool odd = p & 1;
        rs_scatter_kernel<ITEMS, true><<<(unsigned)nb, kSortThreads, 0, s>>>(
            odd ? keys2 : keys, odd ? vals2 : vals, n, 8 * p, h + p * nb * 256, nb, odd ? keys : keys2,
            odd ? vals : vals2, p + 1 < passes ? h + (p + 1) * nb * 256 : nullptr, 8 * (p + 1));
        MG_CUDA(cudaGetLastError());
    }
    *in_second = passes & 1;
    return MG_OK;
}

}  // namespace

mg_status scan_exclusive_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total,
                             const Alloc& al, cudaStream_t s) {
    return scan_impl<uint32_t>(in, out, n, total, al, s);
}

mg_status scan_exclusive_u64(const uint64_t* in, uint64_t* out, int64_t n, uint64_t* total,
                             const Alloc& al, cudaStream_t s) {
    return scan_impl<uint64_t>(in, out, n, total, al, s);
}

mg_status radix_sort_pairs(uint64_t* keys, uint32_t* vals, int64_t n, int bits, const Alloc& al,
                           cudaStream_t s) {
    if (n <= 1 || bits <= 0) return MG_OK;
    if (n >= (int64_t)1 << 32) return fail(MG_ERR_UNSUPPORTED, "radix sort of more than 2^32 items");
    const int64_t nb = (n + kSortTile - 1) / kSortTile;
    Buf k2, v2, hist;
    MG_TRY(k2.alloc(&al, (size_t)n * sizeof(uint64_t), s));
    MG_TRY(v2.alloc(&al, (size_t)n * sizeof(uint32_t), s));
    uint64_t* ks = keys;
    uint32_t* vs = vals;
    uint64_t* kd = k2.as<uint64_t>();
    uint32_t* vd = v2.as<uint32_t>();
    if (nb <= kSmallTiles) {
        // the smallest tiles of which there are at most kSmallTiles: a tile's
        // items are a serial chain
        auto small = n <= kSmallTiles * kSortThreads * 2   ? small_sort<2>
                     : n <= kSmallTiles * kSortThreads * 4 ? small_sort<4>
                                                           : small_sort<kSortItems>;
        bool second = false;
        MG_TRY(small(ks, vs, kd, vd, n, bits, al, s, &second));
        if (second) ks = kd, vs = vd;
    } else {
        MG_TRY(hist.alloc(&al, (size_t)nb * 256 * sizeof(uint32_t), s));
        for (int shift = 0; shift < bits; shift += 8) {
            rs_hist_kernel<kSortItems><<<(unsigned)nb, kSortThreads, 0, s>>>(ks, n, shift, hist.as<uint32_t>(), nb, 1);
            MG_CUDA(cudaGetLastError());
            MG_TRY(scan_exclusive_u32(hist.as<uint32_t>(), hist.as<uint32_t>(), nb * 256, nullptr, al, s));
            rs_scatter_kernel<kSortItems, false><<<(unsigned)nb, kSortThreads, 0, s>>>(
                ks, vs, n, shift, hist.as<uint32_t>(), nb, kd, vd, nullptr, 0);
            MG_CUDA(cudaGetLastError());
            uint64_t* tk = ks; ks = kd; kd = tk;
            uint32_t* tv = vs; vs = vd; vd = tv;
        }
    }
    if (ks != keys) {
        MG_CUDA(cudaMemcpyAsync(keys, ks, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
        MG_CUDA(cudaMemcpyAsync(vals, vs, (size_t)n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    }
    return MG_OK;
}

}  // namespace mg

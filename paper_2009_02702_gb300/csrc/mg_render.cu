// mg_render.cu -- ray-sample node lookup (Sec. 4: rendering from the Mixture
// Graph is a paletted lookup).  One thread per sample: pick the level nearest
// to the sample's LOD, the voxel containing the sample at that level, read its
// node ID and copy the node's value row.  The level and voxel are decided in
// fp32, the precision of the samples.
#include "mg_internal.cuh"

namespace mg {
namespace {

struct Geom {
    int L;
    int id0_bytes;
    int32_t dims[MG_MAX_LEVELS][3];
    int64_t off[MG_MAX_LEVELS];
};

__device__ __forceinline__ int32_t floor_coord(float x, int32_t d0) {
    float xc = x;
    if (!(xc >= 0.f)) xc = 0.f;                  // negatives and NaN
    if (xc > (float)d0) xc = (float)d0;
    return (int32_t)xc;                         // truncation is the floor for xc >= 0
}

// 128-thread CTAs of at most 32 registers a thread: one fits beside a
// persistent query kernel that leaves 4,096 registers of an SM free, so a
// lookup issued on another stream runs concurrently with it
constexpr int kLookupThreads = 128;
// Samples per thread: a lookup is three dependent loads (sample, ID, row), and
// two chains in flight per thread hide more of them than one.  Rows of 32 bytes
// and more are bound by the copy, and a second one only spreads a warp's writes
// (2.07 M samples of 512x512x384: 4-byte rows 20.6 us with one, 14.4 with two;
// 64-byte rows 45.6 and 49.7).
constexpr int lookup_samples(size_t row) { return row < 32 ? 2 : 1; }

// index of the voxel of a sample in its level (32-bit: a volume holds fewer
// than 2^32 voxels), and the level
__device__ __forceinline__ uint32_t sample_voxel(const Geom& G, const float4& smp, int& l) {
    const float t = smp.w + 0.5f;                 // nearest level
    if (!(t >= 0.f)) l = 0;
    else if (t >= (float)(G.L - 1)) l = G.L - 1;
    else l = (int)t;
    uint32_t v[3];
    const float c[3] = {smp.x, smp.y, smp.z};
#pragma unroll
    for (int k = 0; k < 3; k++)
        v[k] = (uint32_t)min(floor_coord(c[k], G.dims[0][k]) >> l, G.dims[l][k] - 1);
    return (v[2] * (uint32_t)G.dims[l][1] + v[1]) * (uint32_t)G.dims[l][0] + v[0];
}

__device__ __forceinline__ uint32_t voxel_node(const Geom& G, const void* __restrict__ mip0,
                                               const uint32_t* __restrict__ mip, int l, uint32_t idx) {
    if (l == 0)
        return G.id0_bytes == 2 ? (uint32_t)__ldg(static_cast<const uint16_t*>(mip0) + idx)
                                : __ldg(static_cast<const uint32_t*>(mip0) + idx);
    return __ldg(mip + G.off[l] + idx);
}

template <typename RowT, int N>
__global__ void __launch_bounds__(kLookupThreads, 16) lookup_kernel(const __grid_constant__ Geom G,
                                                                    const void* __restrict__ mip0,
                                                                    const uint32_t* __restrict__ mip,
                                                                    const float4* __restrict__ samples, int64_t P,
                                                                    const RowT* __restrict__ vals, int words,
                                                                    RowT* __restrict__ out) {
    const int64_t i0 = (int64_t)blockIdx.x * (kLookupThreads * N) + threadIdx.x;
    uint32_t node[N];
    {
        float4 smp[N];
#pragma unroll
        for (int k = 0; k < N; k++)
            smp[k] = i0 + k * kLookupThreads < P ? __ldcs(samples + i0 + k * kLookupThreads) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < N; k++) {
            int l;
            const uint32_t idx = sample_voxel(G, smp[k], l);
            node[k] = voxel_node(G, mip0, mip, l, idx);   // (past the end: the volume's first voxel)
        }
    }
    if (words == 1) {
        RowT v[N];
#pragma unroll
        for (int k = 0; k < N; k++) v[k] = __ldg(vals + node[k]);
#pragma unroll
        for (int k = 0; k < N; k++)
            if (i0 + k * kLookupThreads < P) out[i0 + k * kLookupThreads] = v[k];
        return;
    }
#pragma unroll
    for (int k = 0; k < N; k++) {
        const int64_t i = i0 + k * kLookupThreads;
        if (i >= P) return;
        const RowT* src = vals + (int64_t)node[k] * words;
        RowT* dst = out + i * words;
        for (int w = 0; w < words; w++) dst[w] = __ldg(src + w);
    }
}

// k frames in one launch: samples [off[j], off[j+1]) belong to frame j and
// read the j-th slice of `words` words of every value row (rows of k slices,
// the layout of a k-TF propagation)
constexpr int kMaxFrames = 32;
struct FrameOffsets {
    int64_t off[kMaxFrames + 1];
};

template <typename RowT>
__global__ void __launch_bounds__(kLookupThreads, 16) lookup_multi_kernel(Geom G, const void* __restrict__ mip0,
                                                                          const uint32_t* __restrict__ mip,
                                                                          const float4* __restrict__ samples,
                                                                          FrameOffsets F, int k,
                                                                          const RowT* __restrict__ vals, int words,
                                                                          RowT* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= F.off[k]) return;
    int j = 0;
    while (j + 1 < k && F.off[j + 1] <= i) j++;
    int l;
    const uint32_t idx = sample_voxel(G, __ldg(samples + i), l);
    const uint32_t node = voxel_node(G, mip0, mip, l, idx);
    const RowT* src = vals + ((int64_t)node * k + j) * words;
    RowT* dst = out + i * words;
    for (int w = 0; w < words; w++) dst[w] = __ldg(src + w);
}

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

Geom render_geom(const mg_graph* g) {
    Geom G;
    G.L = g->L;
    G.id0_bytes = g->id0_bytes;
    for (int l = 0; l < MG_MAX_LEVELS; l++) {
        for (int a = 0; a < 3; a++) G.dims[l][a] = g->geom.dims[l][a];
        G.off[l] = g->geom.off[l];
    }
    return G;
}

}  // namespace

mg_status render_lookup_multi(const mg_graph* g, const void* vals, int k, int C, mg_dtype dt, const float* samples,
                              const int64_t* offsets, void* out, cudaStream_t s) {
    if (k < 1 || k > kMaxFrames) return fail(MG_ERR_INVALID_ARG, "k must be 1..32 frames");
    if (!aligned(samples, 16)) return fail(MG_ERR_INVALID_ARG, "samples must be 16-byte aligned");
    FrameOffsets F;
    for (int j = 0; j <= kMaxFrames; j++) F.off[j] = offsets[j <= k ? j : k];
    if (F.off[0] != 0) return fail(MG_ERR_INVALID_ARG, "offsets[0] must be 0");
    for (int j = 0; j < k; j++)
        if (F.off[j + 1] < F.off[j]) return fail(MG_ERR_INVALID_ARG, "offsets must be non-decreasing");
    const int64_t P = F.off[k];
    if (P == 0) return MG_OK;
    const Geom G = render_geom(g);
    const size_t row = (size_t)C * (dt == MG_F32 ? 4 : 2);
    const unsigned grid = grid_for(P, kLookupThreads);
    const float4* sm = reinterpret_cast<const float4*>(samples);
    const uint32_t* mip = g->mip.as<uint32_t>();
    if (row % 16 == 0 && aligned(vals, 16) && aligned(out, 16))
        lookup_multi_kernel<uint4><<<grid, kLookupThreads, 0, s>>>(G, g->mip0.p, mip, sm, F, k, (const uint4*)vals,
                                                                  (int)(row / 16), (uint4*)out);
    else if (row % 8 == 0 && aligned(vals, 8) && aligned(out, 8))
        lookup_multi_kernel<uint2><<<grid, kLookupThreads, 0, s>>>(G, g->mip0.p, mip, sm, F, k, (const uint2*)vals,
                                                                  (int)(row / 8), (uint2*)out);
    else if (row % 4 == 0 && aligned(vals, 4) && aligned(out, 4))
        lookup_multi_kernel<uint32_t><<<grid, kLookupThreads, 0, s>>>(G, g->mip0.p, mip, sm, F, k,
                                                                     (const uint32_t*)vals, (int)(row / 4),
                                                                     (uint32_t*)out);
    else
        lookup_multi_kernel<uint16_t><<<grid, kLookupThreads, 0, s>>>(G, g->mip0.p, mip, sm, F, k,
                                                                     (const uint16_t*)vals, (int)(row / 2),
                                                                     (uint16_t*)out);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

mg_status render_lookup(const mg_graph* g, const void* vals, int C, mg_dtype dt, const float* samples, int64_t P,
                        void* out, cudaStream_t s) {
    if (!aligned(samples, 16)) return fail(MG_ERR_INVALID_ARG, "samples must be 16-byte aligned");
    const Geom G = render_geom(g);
    const size_t row = (size_t)C * (dt == MG_F32 ? 4 : 2);
    const int each = lookup_samples(row);
    const unsigned grid = grid_for(P, kLookupThreads * each);
    const float4* sm = reinterpret_cast<const float4*>(samples);
    const uint32_t* mip = g->mip.as<uint32_t>();
    auto launch = [&](auto k, auto* v, auto* o) {
        k<<<grid, kLookupThreads, 0, s>>>(G, g->mip0.p, mip, sm, P, v, (int)(row / sizeof(*v)), o);
    };
    auto run = [&](auto word) {
        using W = decltype(word);
        launch(each == 2 ? lookup_kernel<W, 2> : lookup_kernel<W, 1>, static_cast<const W*>(vals), static_cast<W*>(out));
    };
    if (row % 16 == 0 && aligned(vals, 16) && aligned(out, 16)) run(uint4{});
    else if (row % 8 == 0 && aligned(vals, 8) && aligned(out, 8)) run(uint2{});
    else if (row % 4 == 0 && aligned(vals, 4) && aligned(out, 4)) run(uint32_t{});
    else run(uint16_t{});
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

}  // namespace mg

// ---------------------------------------------------------------------------
// Ray marching through the node values (Sec. 4): for every pixel a ray from
// the camera through the volume, samples on the lattice t_k = t_start +
// k * base; a sample's LOD, floor(log2(t * pixel angle)) + bias, picks level m
// (clamped to the pyramid) and the step 2^m * base (the step adjusted to the
// LOD, with opacity correction alpha' = 1 - (1 - alpha)^(2^m)); its value is
// trilinear within level m between the 8 voxel centres around it and linear
// between levels m and m+1 by the fractional LOD; front-to-back compositing
// stops at the early-termination opacity.  With node opacities (the TF's
// alpha propagated through the graph), empty space is skipped: climbing from
// level m+2 while the voxel around the sample has opacity exactly 0, the
// lattice samples inside the largest such voxel shrunk by the reach of the
// interpolation (3 * 2^m: levels m and m+1 read voxels within 1.5 of their
// widths of the sample), and before the next LOD change, are skipped; each
// would add exactly nothing, so the image is the same with and without it.
// Decisions (lattice, level, skip, termination) use one rounding per fp32
// operation (no contraction), so they are reproducible off the GPU.
// ---------------------------------------------------------------------------
namespace mg {
namespace {

// one level as the marcher reads it: 32-bit indices (a volume holds fewer than
// 2^32 voxels)
struct MarchLevel {
    const void* ids;        // uint16 or uint32 at level 0, else uint32
    const uint8_t* top;     // levels >= 2, skipping on: where a climb from a voxel ends (0: it is occupied)
    int32_t d[3];
    uint32_t slab;          // voxels between slabs
};

struct MarchArgs {
    int L;
    int id0_bytes;
    MarchLevel lev[MG_MAX_LEVELS];
    const float4* vals;
    int skip;
    mg_camera cam;
    float4* img;
    int32_t* steps;
};

__device__ __forceinline__ float rn_lerp(float a, float b, float f) { return __fadd_rn(a, __fmul_rn(f, __fsub_rn(b, a))); }

__device__ __forceinline__ float4 lerp4(float4 a, float4 b, float f) {
    return make_float4(rn_lerp(a.x, b.x, f), rn_lerp(a.y, b.y, f), rn_lerp(a.z, b.z, f), rn_lerp(a.w, b.w, f));
}

// the eight voxels of a level around a point, and the point's place between them
struct Corners {
    uint32_t n[8];
    float f[3];
};

// node IDs of the 8 voxels whose centres surround p (level-0 units), clamped to the level
__device__ __forceinline__ Corners march_corners(const MarchArgs& A, int l, const float (&p)[3]) {
    Corners K;
    const MarchLevel& V = A.lev[l];
    const float scale = __int_as_float((127 - l) << 23);   // 2^-l
    uint32_t i0[3], i1[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float u = __fsub_rn(__fmul_rn(p[c], scale), 0.5f);
        const float fl = floorf(u);
        K.f[c] = __fsub_rn(u, fl);
        const int k = fl > -1.0e9f ? min((int)fl, 1 << 30) : -(1 << 30), d = V.d[c];   // (NaN: as below the level)
        i0[c] = (uint32_t)min(max(k, 0), d - 1);
        i1[c] = (uint32_t)min(max(k + 1, 0), d - 1);
    }
    const uint32_t r[4] = {i0[2] * V.slab + i0[1] * (uint32_t)V.d[0], i0[2] * V.slab + i1[1] * (uint32_t)V.d[0],
                           i1[2] * V.slab + i0[1] * (uint32_t)V.d[0], i1[2] * V.slab + i1[1] * (uint32_t)V.d[0]};
    if (l == 0 && A.id0_bytes == 2) {
        const uint16_t* ids = static_cast<const uint16_t*>(V.ids);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            K.n[2 * k] = __ldg(ids + r[k] + i0[0]);
            K.n[2 * k + 1] = __ldg(ids + r[k] + i1[0]);
        }
    } else {
        const uint32_t* ids = static_cast<const uint32_t*>(V.ids);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            K.n[2 * k] = __ldg(ids + r[k] + i0[0]);
            K.n[2 * k + 1] = __ldg(ids + r[k] + i1[0]);
        }
    }
    return K;
}

// 2^e for -126 <= e <= 127
__device__ __forceinline__ float exp2_int(int e) { return __int_as_float((127 + e) << 23); }

// trilinear value between the corners.  Inside a segment all eight are one
// node: one gather, and one lerp instead of seven on its value.  Each would
// give a + f (a - a): a itself, or NaN for infinities and NaNs, as here.
__device__ __forceinline__ float4 march_value(const MarchArgs& A, const Corners& K) {
    const uint32_t* n = K.n;
    const uint32_t d = (n[0] ^ n[1]) | (n[0] ^ n[2]) | (n[0] ^ n[3]) | (n[0] ^ n[4]) | (n[0] ^ n[5]) | (n[0] ^ n[6]) |
                       (n[0] ^ n[7]);
    if (d == 0u) {
        const float4 v = __ldg(A.vals + n[0]);
        return lerp4(v, v, K.f[0] + K.f[1] + K.f[2]);
    }
    float4 v[8];
#pragma unroll
    for (int corner = 0; corner < 8; corner++) v[corner] = __ldg(A.vals + n[corner]);
    const float4 x00 = lerp4(v[0], v[1], K.f[0]), x10 = lerp4(v[2], v[3], K.f[0]);
    const float4 x01 = lerp4(v[4], v[5], K.f[0]), x11 = lerp4(v[6], v[7], K.f[0]);
    return lerp4(lerp4(x00, x10, K.f[1]), lerp4(x01, x11, K.f[1]), K.f[2]);
}

__global__ void __launch_bounds__(128) march_kernel(MarchArgs A) {
    const mg_camera& cam = A.cam;
    // a warp takes 8 x 4 pixels, whose rays stay closer than those of 16 x 2
    const int t = threadIdx.x;
    const int i = blockIdx.x * 16 + (t & 7) + ((t >> 2) & 8), j = blockIdx.y * 8 + ((t >> 3) & 3) + ((t >> 4) & 4);
    if (i >= cam.width || j >= cam.height) return;
    const int L = A.L;
    const float inf = 3.0e38f;
    const float sx = __fmul_rn(__fsub_rn(__fadd_rn((float)i, 0.5f), __fmul_rn(0.5f, (float)cam.width)), cam.pix);
    const float sy = __fmul_rn(__fsub_rn(__fsub_rn(__fmul_rn(0.5f, (float)cam.height), (float)j), 0.5f), cam.pix);
    float d[3];
#pragma unroll
    for (int c = 0; c < 3; c++)
        d[c] = __fadd_rn(__fadd_rn(cam.fwd[c], __fmul_rn(sx, cam.right[c])), __fmul_rn(sy, cam.up[c]));
    const float nrm = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(d[0], d[0]), __fmul_rn(d[1], d[1])), __fmul_rn(d[2], d[2])));
#pragma unroll
    for (int c = 0; c < 3; c++) d[c] = __fdiv_rn(d[c], nrm);
    float tmin = -inf, tmax = inf;
    bool miss = false;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float dim = (float)A.lev[0].d[c];
        if (d[c] == 0.0f) {
            if (cam.eye[c] < 0.0f || cam.eye[c] > dim) miss = true;
            continue;
        }
        const float t0 = __fdiv_rn(__fsub_rn(0.0f, cam.eye[c]), d[c]), t1 = __fdiv_rn(__fsub_rn(dim, cam.eye[c]), d[c]);
        const float lo = t0 < t1 ? t0 : t1, hi = t0 < t1 ? t1 : t0;
        if (lo > tmin) tmin = lo;
        if (hi < tmax) tmax = hi;
    }
    const float ts = tmin > 0.0f ? tmin : 0.0f;
    float C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, Aacc = 0.0f;
    int32_t taken = 0;
    if (!miss && tmax > ts) {
        int64_t k = 0;
        while (k < cam.max_steps) {
            const float t = __fadd_rn(ts, __fmul_rn((float)k, cam.base_step));
            if (!(t < tmax)) break;
            const float x = __fmul_rn(t, cam.pix);
            // the exponent of a normal float; ilogbf for the rest
            const int ex = x >= 1.17549435e-38f && x < inf ? (__float_as_int(x) >> 23) - 127 : x > 0.0f ? ilogbf(x) : -1000000;
            const int lam = x > 0.0f ? ex + cam.lod_bias : -1000000;
            const int m = lam < 0 ? 0 : (lam > L - 1 ? L - 1 : lam);
            float fr = 0.0f;
            if (lam >= 0 && m < L - 1) {
                fr = __fsub_rn(__fadd_rn(log2f(x), (float)cam.lod_bias), (float)lam);
                fr = fr < 0.0f ? 0.0f : (fr > 1.0f ? 1.0f : fr);
            }
            float p[3];
#pragma unroll
            for (int c = 0; c < 3; c++) p[c] = __fadd_rn(cam.eye[c], __fmul_rn(t, d[c]));
            // The end of the climb and the sample's node IDs are loaded
            // together; the node values, which a skipped sample does not use,
            // only once it is known not to skip.
            int jz = 0;
            int32_t vox[3] = {0, 0, 0};   // the level-0 voxel around the sample
            if (A.skip && m + 2 < L) {
                const MarchLevel& V = A.lev[m + 2];
                int32_t b[3];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    vox[c] = max((int)floorf(p[c]), 0);
                    b[c] = min(vox[c] >> (m + 2), V.d[c] - 1);
                }
                jz = __ldg(V.top + ((uint32_t)b[2] * V.slab + (uint32_t)b[1] * (uint32_t)V.d[0] + (uint32_t)b[0]));
            }
            const Corners K0 = march_corners(A, m, p);
            Corners K1;
            if (fr > 0.0f) K1 = march_corners(A, m + 1, p);
            if (jz > 0) {
                int32_t bz[3];
#pragma unroll
                for (int c = 0; c < 3; c++) bz[c] = min(vox[c] >> jz, A.lev[jz].d[c] - 1);
                const float size = exp2_int(jz), gap = 3.0f * exp2_int(m);
                float lo[3], hi[3];
                bool inside = true;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    lo[c] = __fadd_rn(__fmul_rn((float)bz[c], size), gap);
                    hi[c] = __fsub_rn(__fmul_rn(__fadd_rn((float)bz[c], 1.0f), size), gap);
                    if (!(p[c] > lo[c] && p[c] < hi[c])) inside = false;
                }
                if (inside) {
                    float tout = inf;
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const float te = d[c] > 0.0f ? __fdiv_rn(__fsub_rn(hi[c], cam.eye[c]), d[c])
                                         : d[c] < 0.0f ? __fdiv_rn(__fsub_rn(lo[c], cam.eye[c]), d[c]) : inf;
                        if (te < tout) tout = te;
                    }
                    const float tch = m < L - 1 ? __fdiv_rn(ldexpf(1.0f, ex + 1), cam.pix) : inf;
                    const float tl = tout < tch ? tout : tch;
                    const float len = __fmul_rn((float)((int64_t)1 << m), cam.base_step);
                    const int64_t n = (int64_t)floorf(__fdiv_rn(__fsub_rn(tl, t), len)) - 1;
                    if (n >= 1) {
                        k += n << m;
                        continue;
                    }
                }
            }
            float4 s = march_value(A, K0);
            if (fr > 0.0f) s = lerp4(s, march_value(A, K1), fr);
            float q = __fsub_rn(1.0f, s.w);
            for (int e = 0; e < m; e++) q = __fmul_rn(q, q);
            const float ap = __fsub_rn(1.0f, q);
            const float w = __fmul_rn(__fsub_rn(1.0f, Aacc), ap);
            C0 = __fadd_rn(C0, __fmul_rn(w, s.x));
            C1 = __fadd_rn(C1, __fmul_rn(w, s.y));
            C2 = __fadd_rn(C2, __fmul_rn(w, s.z));
            Aacc = __fadd_rn(Aacc, w);
            taken++;
            if (cam.ert <= 1.0f && Aacc >= cam.ert) break;
            k += (int64_t)1 << m;
        }
    }
    const int64_t o = (int64_t)j * cam.width + i;
    A.img[o] = make_float4(C0, C1, C2, Aacc);
    if (A.steps) A.steps[o] = taken;
}

// Where a climb from every voxel of a level >= 2 ends: the last of the levels l,
// l + 1, ... whose voxel around it is empty, 0 when the voxel itself is occupied
// (the opacity of its node is not zero).  A ray takes some 45 samples a pixel of
// which one or two skip, so the climb is walked once per voxel here (5.6 M of
// them for 1024x1024x300) instead of at every sample (95 M of a 1920x1080
// frame).
//
// From the coarse levels down, a climb that leaves a voxel ends where its
// parent's ends: one byte read.  The levels of at most kClimbSmall voxels are
// one launch, each voxel climbing by itself, the larger ones one launch each,
// bound by the gathers of the opacities.  (One launch for all, occupancy bits
// first and every voxel climbing over them, took 240 us for 2048x2048x300, as
// much as a frame of 160x120 pixels without skipping; this 47.)
constexpr int64_t kClimbSmall = 1 << 16;
struct ClimbLevel {
    const uint32_t* ids;
    uint8_t* top;
    int32_t d[3];
};
struct ClimbLevels {
    int first, last;
    ClimbLevel lev[MG_MAX_LEVELS];
    int64_t end[MG_MAX_LEVELS];     // voxels of the levels first..l
};

__global__ void climb_small_kernel(const __grid_constant__ ClimbLevels A, const float* __restrict__ opac) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < A.end[A.last]; v += stride) {
        int l = A.first;
        while (v >= A.end[l]) l++;
        const uint32_t i = (uint32_t)(v - (l > A.first ? A.end[l - 1] : 0));
        uint32_t r = i / (uint32_t)A.lev[l].d[0];
        uint32_t x = i - r * (uint32_t)A.lev[l].d[0], z = r / (uint32_t)A.lev[l].d[1], y = r - z * (uint32_t)A.lev[l].d[1];
        int t = 0;
        uint32_t at = i;
        for (int j = l;; j++) {
            if (__ldg(opac + __ldg(A.lev[j].ids + at)) != 0.0f) break;
            t = j;
            if (j == A.last) break;
            // (clamped: an imported image may claim any extents)
            const int32_t(&d)[3] = A.lev[j + 1].d;
            x = min(x >> 1, (uint32_t)d[0] - 1u);
            y = min(y >> 1, (uint32_t)d[1] - 1u);
            z = min(z >> 1, (uint32_t)d[2] - 1u);
            at = (z * (uint32_t)d[1] + y) * (uint32_t)d[0] + x;
        }
        A.lev[l].top[i] = (uint8_t)t;
    }
}

// level l from its parents; 2^lg threads on a row
__global__ void __launch_bounds__(256) climb_level_kernel(const __grid_constant__ ClimbLevel V,
                                                          const __grid_constant__ ClimbLevel P, int l, int lg,
                                                          const float* __restrict__ opac) {
    constexpr int N = 4;   // voxels in flight per thread
    const uint32_t w = 1u << lg, dx = (uint32_t)V.d[0], dy = (uint32_t)V.d[1], rows = dy * (uint32_t)V.d[2];
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x, step = (gridDim.x * blockDim.x) >> lg;
    for (uint32_t r = t >> lg; r < rows; r += step) {
        const uint32_t z = r / dy, y = r - z * dy;
        const uint32_t* ids = V.ids + (size_t)r * dx;
        const uint32_t uz = min(z >> 1, (uint32_t)P.d[2] - 1u), uy = min(y >> 1, (uint32_t)P.d[1] - 1u);
        const uint8_t* up = P.top + ((size_t)uz * (uint32_t)P.d[1] + uy) * (uint32_t)P.d[0];
        uint8_t* top = V.top + (size_t)r * dx;
        for (uint32_t x0 = t & (w - 1); x0 < dx; x0 += N * w) {
            uint32_t id[N];
            uint8_t u[N];
#pragma unroll
            for (int k = 0; k < N; k++) {
                const uint32_t x = x0 + k * w;
                id[k] = x < dx ? __ldg(ids + x) : 0u;   // (past the end: a node that is there)
                u[k] = x < dx ? __ldg(up + min(x >> 1, (uint32_t)P.d[0] - 1u)) : 0;
            }
            float o[N];
#pragma unroll
            for (int k = 0; k < N; k++) o[k] = __ldg(opac + id[k]);
#pragma unroll
            for (int k = 0; k < N; k++)
                if (x0 + k * w < dx) top[x0 + k * w] = o[k] != 0.0f ? (uint8_t)0 : u[k] ? u[k] : (uint8_t)l;
        }
    }
}

}  // namespace

mg_status raymarch(const mg_graph* g, const float* vals, const float* opacity, const mg_camera& cam, float* image,
                   int32_t* steps, cudaStream_t s) {
    if (!aligned(vals, 16) || !aligned(image, 16)) return fail(MG_ERR_INVALID_ARG, "vals and image must be 16-byte aligned");
    MarchArgs A;
    const Geom G = render_geom(g);
    A.L = g->L;
    A.id0_bytes = g->id0_bytes;
    A.vals = reinterpret_cast<const float4*>(vals);
    A.skip = 0;
    for (int l = 0; l < MG_MAX_LEVELS; l++) {
        MarchLevel& V = A.lev[l];
        V = MarchLevel{};
        if (l >= g->L) continue;
        V.ids = l == 0 ? g->mip0.p : static_cast<const void*>(g->mip.as<uint32_t>() + G.off[l]);
        for (int c = 0; c < 3; c++) V.d[c] = G.dims[l][c];
        V.slab = (uint32_t)V.d[0] * (uint32_t)V.d[1];
    }
    if (opacity) {
        // empty-space skipping reads where its climb ends, one byte per voxel
        // of levels >= 2 (built here, in the graph's per-stream scratch),
        // instead of a node ID and its opacity per level climbed
        int64_t bytes = 0, at[MG_MAX_LEVELS] = {};
        for (int l = 2; l < g->L; l++) {
            at[l] = bytes;
            bytes += ((int64_t)G.dims[l][0] * G.dims[l][1] * G.dims[l][2] + 31) & ~(int64_t)31;
        }
        if (bytes > 0) {
            Arena* arena = nullptr;
            MG_TRY(arena_begin(const_cast<mg_graph*>(g), s, &arena));
            Buf top;
            MG_TRY(top.alloc(&arena->view, (size_t)bytes, s));
            ClimbLevels C{};
            C.first = g->L - 1;
            C.last = g->L - 1;
            for (int l = g->L - 1; l >= 2; l--) {
                ClimbLevel& V = C.lev[l];
                V.ids = static_cast<const uint32_t*>(A.lev[l].ids);
                V.top = top.as<uint8_t>() + at[l];
                A.lev[l].top = V.top;
                for (int c = 0; c < 3; c++) V.d[c] = G.dims[l][c];
                if ((int64_t)V.d[0] * V.d[1] * V.d[2] <= kClimbSmall) C.first = l;
            }
            int64_t small = 0;
            for (int l = C.first; l < g->L; l++) {
                small += (int64_t)G.dims[l][0] * G.dims[l][1] * G.dims[l][2];
                C.end[l] = small;
            }
            climb_small_kernel<<<grid_for(small, 128, 152 * 8), 128, 0, s>>>(C, opacity);
            MG_CUDA(cudaGetLastError());
            for (int l = C.first - 1; l >= 2; l--) {
                const ClimbLevel& V = C.lev[l];
                int lg = 0;
                while (lg < 5 && (1 << lg) < V.d[0]) lg++;
                const int64_t threads = ((int64_t)V.d[1] * V.d[2]) << lg;
                climb_level_kernel<<<grid_for(threads, 256, 152 * 16), 256, 0, s>>>(V, C.lev[l + 1], l, lg, opacity);
                MG_CUDA(cudaGetLastError());
            }
            A.skip = 1;
        }
    }
    A.cam = cam;
    A.img = reinterpret_cast<float4*>(image);
    A.steps = steps;
    const dim3 grid((unsigned)((cam.width + 15) / 16), (unsigned)((cam.height + 7) / 8));
    march_kernel<<<grid, 128, 0, s>>>(A);
    MG_CUDA(cudaGetLastError());
    return MG_OK;
}

}  // namespace mg

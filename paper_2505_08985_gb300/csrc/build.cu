// Min/max normal-bound pyramid build (Sec. 4.2, Fig. 5a).
//
// A node at level l covers 2^l x 2^l quads and stores the bounding box
// (s_min, t_min, s_max, t_max) of the normals of every texel its quads touch,
// so each normal triangle below it lies inside the box.  Levels
// kLeafLevel..L are stored; level l is a (2^(L-l))^2 array in Morton order,
// so the four children of node k at level l are nodes 4k..4k+3 at level l-1
// (64 contiguous bytes in either bound format: with FP16 bounds a node's box and
// slab are one 16-byte record, with FP32 bounds the slabs are a second array).
//
// Beside the boxes, the nodes of levels 2..kSlabTop carry a slab (see
// common.cuh), and level 1 holds one 16-byte record per 2 x 2 quads, a
// binary16 box and a slab.  Nothing is stored per quad: the traversal tests a
// group's eight triangles from its nine texels.
//
// Kernel 1 (build_tiles): one CTA per 64 x 64-quad tile.  The tile's 65 x 65
// texels are staged in shared memory with 16-byte vector loads (float4 = two
// FP32 texels, uint4 = four FP16 texels) and stored unchanged into the
// hierarchy's own copy of the map (each texel by exactly one tile, so the map
// is read once per build); each thread builds one leaf node from its 5 x 5
// texels, its four groups' records and their union, warps build the slabs up to
// kSlabTop by shuffles, and levels up to 6 are reduced in shared memory.  A tile
// is a Morton-aligned square at every level, so its nodes form one contiguous
// run and the writes are fully coalesced.
// Kernel 2 (build_up): one launch per level above the tile, four contiguous
// children reduced per thread.
// FP16 bounds round outward (min toward -inf, max toward +inf) so pruning
// stays conservative: the FP16 box contains the FP32 box.
#include "common.cuh"
#include "tri.cuh"

namespace pndf {
namespace {

constexpr int kTileQuadsMax = 64;
constexpr int kTileTexMax = kTileQuadsMax + 1;
constexpr int kBuildThreads = 256;
constexpr int kBuildCtas = 3;  // per SM, 80 registers; at two (91) an 8192^2 build takes 0.25 ms longer

// Second moments of a set of normals about a reference point.
struct Moments {
    float n, s, t, ss, st, tt;
};

__device__ __forceinline__ void add_point(Moments &m, float2 p, float2 ref)
{
    const float s = p.x - ref.x, t = p.y - ref.y;
    m.n += 1.f;
    m.s += s;
    m.t += t;
    m.ss = fmaf(s, s, m.ss);
    m.st = fmaf(s, t, m.st);
    m.tt = fmaf(t, t, m.tt);
}

// Slab direction: the minor principal axis of the set, rounded to binary16
// (any direction would be valid; (0, 1) where the axis is undefined).
__device__ __forceinline__ __half2 slab_dir(const Moments &m)
{
    const float inv = __frcp_rn(fmaxf(m.n, 1.f));
    const float a = fmaf(-m.s * inv, m.s, m.ss), b = fmaf(-m.s * inv, m.t, m.st), c = fmaf(-m.t * inv, m.t, m.tt);
    const float d1 = a - c, d2 = 2.f * b;
    const float h2 = fmaf(d1, d1, d2 * d2);
    if (!(h2 > 1e-37f)) return __floats2half2_rn(0.f, 1.f);
    const float c2 = d1 * rsqrtf(h2);  // cosine of twice the major axis' angle
    const float cs = sqrtf(fmaxf(fmaf(0.5f, c2, 0.5f), 0.f)), sn = copysignf(sqrtf(fmaxf(fmaf(-0.5f, c2, 0.5f), 0.f)), d2);
    return __floats2half2_rn(-sn, cs);
}

// The stored slab of normals whose projections onto dir span [lo, hi] and
// whose |s| + |t| is at most reach: widened by reach 2^-19, more than the FP32
// rounding of the projection here (3 x 2^-24 reach), of the query's (the same),
// and of the distance by which an edge function rounded to zero can let m
// outside its triangle (2^-21 of the triangle's extent, at most 2 reach), then
// rounded outward to binary16.
__device__ __forceinline__ uint2 slab_code(__half2 dir, float lo, float hi, float reach, bool mark)
{
    const float2 d = __half22float2(dir);
    uint2 v;
    v.x = *reinterpret_cast<uint32_t *>(&dir);
    const float w = reach * 0x1p-19f;
    if (mark || !isfinite(d.x) || !isfinite(d.y) || !isfinite(lo) || !isfinite(hi) || !isfinite(w)) {
        v.x = 0u;  // direction 0: every projection is 0, inside (-inf, +inf)
        v.y = kSlabAll;
    } else {
        const __half2 iv = __halves2half2(__float2half_rd(lo - w), __float2half_ru(hi + w));
        v.y = *reinterpret_cast<const uint32_t *>(&iv);
    }
    return v;
}

__device__ __forceinline__ float project(__half2 dir, float2 p)
{
    const float2 d = __half22float2(dir);
    return fmaf(p.x, d.x, p.y * d.y);
}

__device__ __forceinline__ float box_reach(const Box &b)
{
    return fmaxf(fabsf(b.smin), fabsf(b.smax)) + fmaxf(fabsf(b.tmin), fabsf(b.tmax));
}

// A triangle that the traversal evaluates in FP64 (FP32 |cross| below
// kTinyCross, cross not exactly 0).  The groups that hold one are marked, so
// that pruning by slabs never decides whether it is reached.  Written so that
// a cross that is not a number counts.
__device__ __forceinline__ bool near_singular(float2 a, float2 b, float2 c)
{
    if (fabsf(orient(a.x, a.y, b.x, b.y, c.x, c.y)) >= kTinyCross) return false;
    if ((a.x == b.x && a.y == b.y) || (a.x == c.x && a.y == c.y)) return false;
    return !(orient_d(a.x, a.y, b.x, b.y, c.x, c.y) == 0.0);
}

template <int TFMT>
__device__ __forceinline__ float2 load_texel(const void *t, size_t idx)
{
    if (TFMT == PNDF_TEXEL_F32X2) return reinterpret_cast<const float2 *>(t)[idx];
    return __half22float2(reinterpret_cast<const __half2 *>(t)[idx]);
}

// Texel idx of src, loaded for staging and (own) stored unchanged in dst.
template <int TFMT>
__device__ __forceinline__ float2 copy_texel(const void *src, void *dst, size_t idx, bool own)
{
    if (TFMT == PNDF_TEXEL_F32X2) {
        float2 v = reinterpret_cast<const float2 *>(src)[idx];
        if (own) reinterpret_cast<float2 *>(dst)[idx] = v;
        return v;
    }
    __half2 v = reinterpret_cast<const __half2 *>(src)[idx];
    if (own) reinterpret_cast<__half2 *>(dst)[idx] = v;
    return __half22float2(v);
}

// VEC = texels per 16-byte load (2 for FP32, 4 for FP16), or 1 when rows are
// not 16-byte aligned (n not a multiple of VEC).
template <int TFMT, int BFMT, int VEC>
__global__ void __launch_bounds__(kBuildThreads, kBuildCtas) build_tiles(const void *__restrict__ src, MapDesc d, int tileQ,
                                                            int lq)
{
    __shared__ float2 tex[kTileTexMax * kTileTexMax];
    __shared__ Box box[2][(kTileQuadsMax / kLeafQuads) * (kTileQuadsMax / kLeafQuads)];

    const int n = d.n;
    const int tw = tileQ + 1;
    const int c0 = blockIdx.x * tileQ, r0 = blockIdx.y * tileQ;
    const int tid = threadIdx.x;

    // ---- stage texels: VEC-wide loads for the first tileQ columns.  The
    // hierarchy's own copy of the map is written on the way: a tile owns its
    // first tileQ rows and columns, and the map's last row or column where it
    // is the tile's shared edge, so every texel is stored exactly once ----
    void *copy = const_cast<void *>(d.texels);
    const int nvec = tileQ / VEC;
    for (int idx = tid; idx < tw * nvec; idx += kBuildThreads) {
        int r = idx / nvec, v = idx - r * nvec;
        int gr = r0 + r, gc = c0 + v * VEC;
        if (gr >= n || gc >= n) continue;
        const bool own = r < tileQ || gr == n - 1;
        size_t g = size_t(gr) * n + gc;
        float2 *dst = &tex[r * kTileTexMax + v * VEC];
        if (VEC == 2) {
            float4 p = reinterpret_cast<const float4 *>(src)[g >> 1];
            if (own) reinterpret_cast<float4 *>(copy)[g >> 1] = p;
            dst[0] = make_float2(p.x, p.y);
            dst[1] = make_float2(p.z, p.w);
        } else if (VEC == 4) {
            uint4 p = reinterpret_cast<const uint4 *>(src)[g >> 2];
            if (own) reinterpret_cast<uint4 *>(copy)[g >> 2] = p;
            dst[0] = __half22float2(*reinterpret_cast<__half2 *>(&p.x));
            dst[1] = __half22float2(*reinterpret_cast<__half2 *>(&p.y));
            dst[2] = __half22float2(*reinterpret_cast<__half2 *>(&p.z));
            dst[3] = __half22float2(*reinterpret_cast<__half2 *>(&p.w));
        } else {
            dst[0] = copy_texel<TFMT>(src, copy, g, own);
        }
    }
    // the shared last column of the tile
    for (int r = tid; r < tw; r += kBuildThreads) {
        int gr = r0 + r, gc = c0 + tileQ;
        if (gr < n && gc < n)
            tex[r * kTileTexMax + tileQ] =
                copy_texel<TFMT>(src, copy, size_t(gr) * n + gc, gc == n - 1 && (r < tileQ || gr == n - 1));
    }
    __syncthreads();

    // ---- groups (level 1) and leaf nodes: thread i owns the leaf node with
    // local Morton index i, whose 5 x 5 texels it keeps in registers ----
    const int T = tileQ / kLeafQuads;  // leaf nodes per tile side
    const uint32_t tile_m = morton2(blockIdx.x, blockIdx.y);
    int cur = T * T;
    const bool leaf = tid < cur;
    const uint32_t m2 = tile_m * uint32_t(cur) + uint32_t(tid);
    const int la = int(compact1by1(tid)) * kLeafQuads, lc = int(compact1by1(tid >> 1)) * kLeafQuads;
    // quads of the block inside the map per axis; texels past them repeat the
    // last one, which adds nothing to a box or a slab
    const int nvx = leaf ? max(0, min(kLeafQuads, n - 1 - (c0 + la))) : 0;
    const int nvy = leaf ? max(0, min(kLeafQuads, n - 1 - (r0 + lc))) : 0;
    const bool some = nvx > 0 && nvy > 0;
    float2 t[kLeafTexels][kLeafTexels];
#pragma unroll
    for (int y = 0; y < kLeafTexels; ++y)
#pragma unroll
        for (int x = 0; x < kLeafTexels; ++x)
            t[y][x] = some ? tex[(lc + min(y, nvy)) * kTileTexMax + la + min(x, nvx)] : make_float2(0.f, 0.f);
    Box b = empty_box();
    bool mark = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int gx = 2 * (k & 1), gy = 2 * (k >> 1);
        uint4 rec = make_uint4(0x7c007c00u, 0xfc00fc00u, 0u, kSlabAll);  // empty box
        if (some && nvx > gx && nvy > gy) {
            Box gb = empty_box();
            Moments mo{};
            bool gmark = false;
#pragma unroll
            for (int v = 0; v < 9; ++v) {
                const float2 p = t[gy + v / 3][gx + v % 3];
                gb.smin = fminf(gb.smin, p.x);
                gb.tmin = fminf(gb.tmin, p.y);
                gb.smax = fmaxf(gb.smax, p.x);
                gb.tmax = fmaxf(gb.tmax, p.y);
                add_point(mo, p, t[gy][gx]);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int x = gx + (v & 1), y = gy + (v >> 1);
                gmark |= near_singular(t[y][x], t[y][x + 1], t[y + 1][x]);
                gmark |= near_singular(t[y + 1][x + 1], t[y + 1][x], t[y][x + 1]);
            }
            const __half2 dir = slab_dir(mo);
            float lo = __int_as_float(0x7f800000), hi = -lo;
#pragma unroll
            for (int v = 0; v < 9; ++v) {
                const float p = project(dir, t[gy + v / 3][gx + v % 3]);
                lo = fminf(lo, p);
                hi = fmaxf(hi, p);
            }
            const uint2 sl = slab_code(dir, lo, hi, box_reach(gb), gmark);
            const __half2 bl = __halves2half2(__float2half_rd(gb.smin), __float2half_rd(gb.tmin));
            const __half2 bh = __halves2half2(__float2half_ru(gb.smax), __float2half_ru(gb.tmax));
            rec = make_uint4(*reinterpret_cast<const uint32_t *>(&bl), *reinterpret_cast<const uint32_t *>(&bh), sl.x,
                             sl.y);
            grow(b, gb);
            mark |= gmark;
        }
        if (leaf) const_cast<uint4 *>(d.groups)[4 * size_t(m2) + k] = rec;
    }
    if (leaf) {
        box[0][tid] = b;
        store_box<BFMT>(d, node_index(d.L, kLeafLevel, m2), b);
    }

    // ---- slabs of levels 2, 3 and 4: siblings are 4 lanes, then 16 ----
    {
        const int lane = tid & 31;
        float2 ref;  // one reference point per level-4 node
        ref.x = __shfl_sync(0xffffffffu, t[0][0].x, lane & 16);
        ref.y = __shfl_sync(0xffffffffu, t[0][0].y, lane & 16);
        Moments mo{};
        if (some) {
#pragma unroll
            for (int v = 0; v < 25; ++v) add_point(mo, t[v / 5][v % 5], ref);
        }
        float reach = some ? box_reach(b) : 0.f;
        unsigned any = mark ? 1u : 0u;
#pragma unroll
        for (int l = kLeafLevel; l <= kSlabTop; ++l) {
            const int sh = 2 * (l - kLeafLevel);  // 4^(l - 2) lanes per node
            if (l > kLeafLevel) {
#pragma unroll
                for (int o = (1 << sh) >> 2; o < (1 << sh); o <<= 1) {
                    mo.n += __shfl_xor_sync(0xffffffffu, mo.n, o);
                    mo.s += __shfl_xor_sync(0xffffffffu, mo.s, o);
                    mo.t += __shfl_xor_sync(0xffffffffu, mo.t, o);
                    mo.ss += __shfl_xor_sync(0xffffffffu, mo.ss, o);
                    mo.st += __shfl_xor_sync(0xffffffffu, mo.st, o);
                    mo.tt += __shfl_xor_sync(0xffffffffu, mo.tt, o);
                    reach = fmaxf(reach, __shfl_xor_sync(0xffffffffu, reach, o));
                    any |= __shfl_xor_sync(0xffffffffu, any, o);
                }
            }
            const __half2 dir = slab_dir(mo);
            float lo = __int_as_float(0x7f800000), hi = -lo;
            if (some) {
#pragma unroll
                for (int v = 0; v < 25; ++v) {
                    const float p = project(dir, t[v / 5][v % 5]);
                    lo = fminf(lo, p);
                    hi = fmaxf(hi, p);
                }
            }
#pragma unroll
            for (int o = 1; o < (1 << sh); o <<= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            }
            if (leaf && l <= d.L && (tid & ((1 << sh) - 1)) == 0)
                store_slab<BFMT>(d, node_index(d.L, l, m2 >> sh), slab_code(dir, lo, hi, reach, any != 0u));
        }
    }
    __syncthreads();

    // ---- reduce inside the tile up to level lq ----
    int s = 0;
    for (int l = kLeafLevel + 1; l <= lq; ++l) {
        cur >>= 2;
        if (tid < cur) {
            Box b = box[s][4 * tid];
            grow(b, box[s][4 * tid + 1]);
            grow(b, box[s][4 * tid + 2]);
            grow(b, box[s][4 * tid + 3]);
            box[s ^ 1][tid] = b;
            const uint32_t k = node_index(d.L, l, tile_m * uint32_t(cur) + uint32_t(tid));
            store_box<BFMT>(d, k, b);
            if (l > kSlabTop) store_slab<BFMT>(d, k, make_uint2(0u, kSlabAll));
        }
        s ^= 1;
        __syncthreads();
    }
}

// Level l > kSlabTop from level l - 1.  (With FP16 bounds the children are
// binary16 values already and the reduction is exact.)
template <int BFMT>
__global__ void build_up(MapDesc d, int l, uint32_t count)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const uint32_t k = node_index(d.L, l, i);
    Box b = load_box<BFMT>(d, 4 * k);
    grow(b, load_box<BFMT>(d, 4 * k + 1));
    grow(b, load_box<BFMT>(d, 4 * k + 2));
    grow(b, load_box<BFMT>(d, 4 * k + 3));
    store_box<BFMT>(d, k, b);
    store_slab<BFMT>(d, k, make_uint2(0u, kSlabAll));
}

template <int TFMT, int BFMT>
cudaError_t launch_tiles(const void *src, const MapDesc &d, cudaStream_t s)
{
    const int side = 1 << d.L;
    const int tileQ = side < kTileQuadsMax ? side : kTileQuadsMax;
    int lq = 0;
    while ((1 << lq) < tileQ) ++lq;
    dim3 grid(side / tileQ, side / tileQ);
    constexpr int VEC = TFMT == PNDF_TEXEL_F32X2 ? 2 : 4;
    if (d.n % VEC == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0)
        build_tiles<TFMT, BFMT, VEC><<<grid, kBuildThreads, 0, s>>>(src, d, tileQ, lq);
    else
        build_tiles<TFMT, BFMT, 1><<<grid, kBuildThreads, 0, s>>>(src, d, tileQ, lq);
    count_launches(1 + (d.L > lq ? d.L - lq : 0));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    for (int l = lq + 1; l <= d.L; ++l) {
        const uint32_t cnt = uint32_t(level_nodes(d.L, l));
        build_up<BFMT><<<(cnt + 255) / 256, 256, 0, s>>>(d, l, cnt);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_build(const void *texels_src, pndf_hierarchy *h, cudaStream_t s)
{
    const MapDesc &d = h->d;
    cudaError_t e;
    if (d.texel_fmt == PNDF_TEXEL_F32X2)
        e = d.bounds_fmt == PNDF_BOUNDS_F32 ? launch_tiles<PNDF_TEXEL_F32X2, PNDF_BOUNDS_F32>(texels_src, d, s)
                                            : launch_tiles<PNDF_TEXEL_F32X2, PNDF_BOUNDS_F16_OUTWARD>(texels_src, d, s);
    else
        e = d.bounds_fmt == PNDF_BOUNDS_F32 ? launch_tiles<PNDF_TEXEL_F16X2, PNDF_BOUNDS_F32>(texels_src, d, s)
                                            : launch_tiles<PNDF_TEXEL_F16X2, PNDF_BOUNDS_F16_OUTWARD>(texels_src, d, s);
    if (e == cudaSuccess && h->clusters) e = launch_clusters(h, s);
    return e;
}

}  // namespace pndf

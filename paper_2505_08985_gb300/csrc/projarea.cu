// Analytic projected area P(w) of a footprint (Sec. 4.3, Eq. 9-11, App. B).
//
//   P(w) = sum over footprint triangles T of k_r(T) / |cross(T)| * V_T(w),
//   V_T(w) = integral over n+(T) of (w . m~) / m~_z dm,
// where n+(T) is the part of the normal triangle whose normals see w, k_r(T)
// the kernel at T's uv centroid (cut where q > 16), cross(T) = (n_b - n_a) x
// (n_c - n_a).  Every triangle in the footprint is integrated (no pruning:
// every visible triangle contributes).
//
// Per triangle (meang.cuh): a positive quadrature of the integrand over the uv
// triangle, in FP32.
//  * all three vertices see w  =>  the whole triangle does (the visible region,
//    a right half-disk joined to a left half-ellipse, is convex; App. B): 6
//    points for small triangles, 12 for those that straddle normal regions;
//  * no vertex sees w and none of the triangle can: exactly 0 (Alg. 1 drops
//    every edge);
//  * otherwise the polygon and the cap that the visibility boundary cuts off it
//    (partial_mean);
//  * larger triangles are split in four, each part classified again; a part that
//    is still too large takes the closed form of visible.cuh in FP64 (the clip
//    of Alg. 1, Eq. 11's boundary integral, the segment form of Eq. 13).
// All but the first kind and the zeros are deferred into per-warp rings and
// evaluated 32 at a time, so that each runs lane-dense.
//
// Work decomposition: each request's footprint is cut into bands of kBand quad
// rows; one warp integrates one band (its quads inside the support's ellipse,
// row after row, one per lane), compensated sums are reduced across the warp
// and stored per band;
// a second kernel adds a request's bands in fixed order, so results do not
// depend on scheduling or on which other requests share the launch.
#include "area_step.cuh"
#include "ggx.cuh"
#include "meang.cuh"
#include "visible.cuh"

namespace pndf {

__device__ unsigned int g_status_projarea;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kGgxCtas = 4;   // per SM, of 3, 4, 5, 6 and 8 within 8% of each other
constexpr int kAreaCtas = 4;  // see pa_items
// A band is long enough to pay for its row setup and its rings' last, partly
// filled evaluations, and short enough to spread a few footprints over the SMs: 8
// / 4 / 2 rows, the same 192 requests on 16384^2 14.3 / 13.0 / 12.2 ms, 64 on 4096^2
// 0.99 / 0.64 / 0.49 ms, 1000 small ones 0.31 ms each.  Two rows are faster or
// equal, but the partial sums (and a server's scratch) double with each halving.
constexpr int kBand = 4;                 // quad rows per work item

// V_T / |cross| in closed form (visible.cuh, FP64), for the largest triangles;
// the segment form of Eq. 13 where the normals collapsed (|cross| < 1e-12).
__device__ __noinline__ float slow_ratio(float2 a, float2 b, float2 c, const Dir &wf)
{
    const vis::DirD w = vis::make_dir(wf.wx, wf.wy, wf.wz);
    const double cr = (double(b.x) - double(a.x)) * (double(c.y) - double(a.y)) -
                      (double(b.y) - double(a.y)) * (double(c.x) - double(a.x));
    if (fabs(cr) < 1e-12) return float(vis::collapsed_visible(a.x, a.y, b.x, b.y, c.x, c.y, w));
    return float(vis::tri_visible<double>(a.x, a.y, b.x, b.y, c.x, c.y, w));
}

struct Req {
    float x, y, ia, ib, ic, norm, ry;
    int j0, j1, i0, i1;
    bool valid;
};

__device__ __forceinline__ Req make_req(const pndf_query &r, int n)
{
    Req q;
    float det = r.sxx * r.syy - r.sxy * r.sxy;
    q.valid = (r.sxx > 0.f) && (r.syy > 0.f) && (det > 0.f) && isfinite(det) && isfinite(r.x) && isfinite(r.y);
    q.x = r.x;
    q.y = r.y;
    float inv = 1.f / det;
    q.ia = r.syy * inv;
    q.ib = -r.sxy * inv;
    q.ic = r.sxx * inv;
    q.norm = 1.f / (2.f * kPi * sqrtf(det));
    float rx = 4.f * sqrtf(r.sxx) * (1.f + 1e-5f) + 1e-6f;
    q.ry = 4.f * sqrtf(r.syy) * (1.f + 1e-5f) + 1e-6f;
    // quads whose centroid (i + 1/3 or 2/3) can lie in the 4-sigma box
    // clamped in float first so no int conversion can overflow
    float fi0 = fmaxf(floorf(r.x - rx) - 1.f, 0.f), fi1 = fminf(ceilf(r.x + rx), float(n - 2));
    float fj0 = fmaxf(floorf(r.y - q.ry) - 1.f, 0.f), fj1 = fminf(ceilf(r.y + q.ry), float(n - 2));
    bool empty = !(fi0 <= fi1) || !(fj0 <= fj1);
    q.i0 = empty ? 0 : int(fi0);
    q.i1 = empty ? -1 : int(fi1);
    q.j0 = empty ? 0 : int(fj0);
    q.j1 = empty ? -1 : int(fj1);
    if (!q.valid || q.i0 > q.i1 || q.j0 > q.j1) {
        q.i1 = q.i0 - 1;
        q.j1 = q.j0 - 1;
    }
    return q;
}

__device__ __forceinline__ float wq(const Req &q, float dx, float dy)
{
    return fmaf(q.ia * dx, dx, fmaf(2.f * q.ib * dx, dy, q.ic * dy * dy));
}

// Columns [x0, x0 + count) of row j whose triangles' centroids can lie in the
// ellipse q <= kQCut: at height dy, dx = -(ib / ia) dy +- sqrt(Q / ia - dy^2 det /
// ia^2), widened by a column and 1e-3 of Q (FP32 rounding of the square root's
// argument; a nearly singular S takes the whole row).
__device__ __forceinline__ void row_span(const Req &q, int j, int &x0, int &count)
{
    const float k = q.ib / q.ia, v = q.ic / q.ia - k * k, Q = kQCut * (1.0f + 1e-3f) / q.ia;
    x0 = q.i0;
    count = q.i1 - q.i0 + 1;
    if (!(v * q.ia > 1e-3f * q.ic)) return;
    float lo = __int_as_float(0x7f800000), hi = -lo;
#pragma unroll
    for (int t = 1; t <= 2; ++t) {
        const float dy = (float(j) - q.y) + float(t) * (1.f / 3.f);
        const float r2 = fmaf(-dy * dy, v, Q);
        if (r2 < 0.f) continue;
        const float r = sqrtf(r2), c = fmaf(-k, dy, q.x);
        lo = fminf(lo, c - r);
        hi = fmaxf(hi, c + r);
    }
    if (lo > hi) {  // the row misses the ellipse
        count = 0;
        return;
    }
    const float f0 = fmaxf(floorf(lo) - 2.f, float(q.i0)), f1 = fminf(ceilf(hi) + 1.f, float(q.i1));
    if (!(f0 <= f1)) {
        count = f0 > f1 ? 0 : count;
        return;
    }
    x0 = int(f0);
    count = int(f1) - x0 + 1;
}

template <int TFMT>
__device__ __forceinline__ float2 texel(const MapDesc &d, int i, int j)
{
    size_t idx = size_t(j) * d.n + i;
    if (TFMT == PNDF_TEXEL_F32X2) return __ldg(reinterpret_cast<const float2 *>(d.texels) + idx);
    return __half22float2(__ldg(reinterpret_cast<const __half2 *>(d.texels) + idx));
}

// Deferred triangles, one ring per class and warp: (i << 15) | (j << 1) | tri and
// the kernel weight; at most 31 held over plus one step's 64.
constexpr int kDefer = 128;
constexpr int kRings = 3;  // kLarge, kPartial, kSplit
struct WarpArea {
    uint32_t id[kRings][kDefer];
    float wt[kRings][kDefer];
    int off[kBand + 1], x0[kBand];  // the band's rows: first quad of each in lane order, first column
};

// Compensated sum (Neumaier).
struct Sum {
    float s, c;
};
__device__ __forceinline__ void add(Sum &a, float v)
{
    const float t = a.s + v;
    a.c += fabsf(a.s) >= fabsf(v) ? (a.s - t) + v : (v - t) + a.s;
    a.s = t;
}

__device__ __forceinline__ float longest2(float2 a, float2 b, float2 c)
{
    return fmaxf(len2(sub(b, a)), fmaxf(len2(sub(c, a)), len2(sub(c, b))));
}

// Half the mean of g over a fully visible triangle of class kSmall / kLarge.
__device__ __forceinline__ float full_mean_small(float2 a, float2 b, float2 c, const Dir &w)
{
    return fmaf(0.5f, quad4(a, sub(b, a), sub(c, a), [&](float x, float y) { return slope_at(w, x, y); }), 0.5f * w.wz);
}
__device__ __forceinline__ float full_mean_large(float2 a, float2 b, float2 c, const Dir &w)
{
    return fmaf(0.5f, quad6(a, sub(b, a), sub(c, a), [&](float x, float y) { return slope_at(w, x, y); }), 0.5f * w.wz);
}

// V_T / |cross| of a triangle of class kPartial.
__device__ __forceinline__ float partial_ratio(float2 a, float2 b, float2 c, const Dir &w)
{
    const float v = partial_mean(a, b, c, w);
    return v < 0.f ? slow_ratio(a, b, c, w) : v;
}

// V_T / |cross| of a triangle of class kSplit: the mean over its four parts.
__device__ __noinline__ float split_ratio(float2 a, float2 b, float2 c, const Dir &w)
{
    const float2 ab = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y + b.y));
    const float2 bc = make_float2(0.5f * (b.x + c.x), 0.5f * (b.y + c.y));
    const float2 ca = make_float2(0.5f * (c.x + a.x), 0.5f * (c.y + a.y));
    float sum = 0.f;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const float2 p = k == 0 ? a : k == 1 ? ab : k == 2 ? ca : ab;
        const float2 q = k == 0 ? ab : k == 1 ? b : k == 2 ? bc : bc;
        const float2 r = k == 0 ? ca : k == 1 ? bc : k == 2 ? c : ca;
        const float zp = zof(p), zq = zof(q), zr = zof(r);
        const Class cl = classify(phi_of(w, p, zp), phi_of(w, q, zq), phi_of(w, r, zr), zp, zq, zr, longest2(p, q, r), w);
        if (cl == kSmall || cl == kLarge)
            sum += full_mean_large(p, q, r, w);
        else if (cl == kPartial)
            sum += partial_ratio(p, q, r, w);
        else if (cl == kSplit)
            sum += slow_ratio(p, q, r, w);
    }
    return 0.25f * sum;
}

// Lane's deferred triangle of ring r (slot head + lane): kernel weight times
// V_T / |cross| (tri 0 = (u0, u1, u2), tri 1 = (u3, u2, u1)).
template <int TFMT>
__device__ __forceinline__ float deferred_value(const MapDesc &d, const Dir &w, const WarpArea &wa, int r,
                                                uint32_t head, int lane)
{
    const uint32_t slot = (head + uint32_t(lane)) & (kDefer - 1);
    const uint32_t id = wa.id[r][slot];
    const int i = int(id >> 15), j = int((id >> 1) & 0x3fffu), tri = int(id & 1u);
    const float2 a = texel<TFMT>(d, i + tri, j + tri);
    const float2 b = texel<TFMT>(d, i + 1 - tri, j + tri);
    const float2 c = texel<TFMT>(d, i + tri, j + 1 - tri);
    const float v = r == 0 ? full_mean_large(a, b, c, w) : r == 1 ? partial_ratio(a, b, c, w) : split_ratio(a, b, c, w);
    return wa.wt[r][slot] * v;
}

__device__ __forceinline__ uint32_t band_count(const pndf_query &r, int n)
{
    const Req q = make_req(r, n);
    const int rows = q.j1 - q.j0 + 1;
    return rows > 0 ? uint32_t((rows + kBand - 1) / kBand) : 0u;
}

__global__ void pa_bands(MapDesc d, const pndf_query *__restrict__ qs, int64_t k0, int cnt, uint32_t *__restrict__ nb)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) nb[t] = band_count(qs[k0 + t], d.n);
}

// Exclusive scan of cnt (<= 65536) values value(i) into nb, one CTA of 1024
// threads; the total goes to nb[cnt] and the work cursor to zero.  (value may
// read nb[i] itself.)
template <class F>
__device__ __forceinline__ void scan_bands(F value, uint32_t *__restrict__ nb, int cnt, unsigned int *__restrict__ cursor)
{
    __shared__ uint32_t part[1024];
    const int per = (cnt + 1023) / 1024;
    const int b0 = threadIdx.x * per;
    uint32_t sum = 0;
    for (int i = 0; i < per; ++i)
        if (b0 + i < cnt) sum += value(b0 + i);
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        uint32_t t = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += t;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - sum;
    for (int i = 0; i < per; ++i) {
        if (b0 + i < cnt) {
            uint32_t v = value(b0 + i);
            nb[b0 + i] = run;
            run += v;
        }
    }
    if (threadIdx.x == 1023) {
        nb[cnt] = part[1023];
        *cursor = 0u;
    }
}

__global__ void __launch_bounds__(1024) pa_scan(uint32_t *nb, int cnt, unsigned int *cursor)
{
    scan_bands([&](int i) { return nb[i]; }, nb, cnt, cursor);
}

// pa_bands and pa_scan of up to kPrepSmall requests in one launch.
constexpr int kPrepSmall = 4096;
__global__ void __launch_bounds__(1024) pa_prep(MapDesc d, const pndf_query *__restrict__ qs, int64_t k0, int cnt,
                                                uint32_t *nb, unsigned int *cursor)
{
    scan_bands([&](int i) { return band_count(qs[k0 + i], d.n); }, nb, cnt, cursor);
}

// Band `band` (kBand quad rows) of request (q, w) on map d, integrated by one
// warp: the band's quads inside the ellipse in row order, one per lane, both
// triangles; returns the compensated sum and its correction, reduced to lane 0
// in a fixed order.
template <int TFMT>
__device__ __forceinline__ float2 integrate_band(const MapDesc &d, const Req &q, const Dir &w, int band, int lane,
                                                 WarpArea &wa)
{
    const unsigned lt = (1u << lane) - 1u;
    const int jb0 = q.j0 + band * kBand, rows = min(q.j1 - jb0 + 1, kBand);
    {
        int x0 = 0, cnt = 0;
        if (lane < rows) row_span(q, jb0 + lane, x0, cnt);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < kBand; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        __syncwarp();
        if (lane < kBand) {
            wa.off[lane + 1] = incl;
            wa.x0[lane] = x0;
        }
        if (lane == 0) wa.off[0] = 0;
        __syncwarp();
    }
    const int total = wa.off[kBand];
    Sum sum{0.f, 0.f};
    uint32_t head[kRings] = {0u, 0u, 0u};
    int nd[kRings] = {0, 0, 0};  // triangles waiting per ring (warp-uniform)
    int row = 0;
    for (int base = 0; base < total; base += 32) {
        const int k = base + lane;
        Class cl[2] = {kNone, kNone};
        float kw[2] = {0.f, 0.f}, v[2] = {0.f, 0.f};
        int i = 0, j = 0;
        if (k < total) {
            while (k >= wa.off[row + 1]) ++row;
            i = wa.x0[row] + (k - wa.off[row]);
            j = jb0 + row;
            const float dx = float(i) - q.x, dy = float(j) - q.y;
            const float ql = wq(q, dx + (1.f / 3.f), dy + (1.f / 3.f)), qu = wq(q, dx + (2.f / 3.f), dy + (2.f / 3.f));
            if (ql <= kQCut || qu <= kQCut) {
                const float2 n1 = texel<TFMT>(d, i + 1, j), n2 = texel<TFMT>(d, i, j + 1);
                const float2 n0 = texel<TFMT>(d, i, j), n3 = texel<TFMT>(d, i + 1, j + 1);
                const float z1 = zof(n1), z2 = zof(n2);
                const float f1 = phi_of(w, n1, z1), f2 = phi_of(w, n2, z2);
                const float d12 = len2(sub(n2, n1));
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const float qk = t ? qu : ql;
                    if (qk > kQCut) continue;
                    const float2 na = t ? n3 : n0;
                    const float za = zof(na);
                    const float h2 = fmaxf(d12, fmaxf(len2(sub(n1, na)), len2(sub(n2, na))));
                    kw[t] = q.norm * expf(-0.5f * qk);
                    cl[t] = classify(phi_of(w, na, za), f1, f2, za, z1, z2, h2, w);
                    if (cl[t] == kSmall) v[t] = kw[t] * full_mean_small(na, t ? n2 : n1, t ? n1 : n2, w);
                }
            }
        }
        add(sum, v[0]);
        add(sum, v[1]);
        const bool last = base + 32 >= total;
#pragma unroll
        for (int r = 0; r < kRings; ++r) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const bool dfr = cl[t] == Class(kLarge + r);
                const unsigned m = __ballot_sync(kFull, dfr);
                if (dfr) {
                    const uint32_t pos = (head[r] + uint32_t(nd[r]) + __popc(m & lt)) & (kDefer - 1);
                    wa.id[r][pos] = (uint32_t(i) << 15) | (uint32_t(j) << 1) | uint32_t(t);
                    wa.wt[r][pos] = kw[t];
                }
                nd[r] += __popc(m);
            }
            __syncwarp();
            while (nd[r] >= (last ? 1 : 32)) {  // (one copy of each class's code)
                const int n = min(nd[r], 32);
                add(sum, lane < n ? deferred_value<TFMT>(d, w, wa, r, head[r], lane) : 0.f);
                head[r] += uint32_t(n);
                nd[r] -= n;
                __syncwarp();
            }
        }
    }
    float s = sum.s, c = sum.c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float so = __shfl_down_sync(kFull, s, o), co = __shfl_down_sync(kFull, c, o);
        float tt = s + so;
        float err = fabsf(s) >= fabsf(so) ? (s - tt) + so : (so - tt) + s;
        s = tt;
        c += co + err;
    }
    return make_float2(s, c);
}

// What bounds it: FP32 issue (86% of the slots; about 340 instructions a triangle,
// a quarter of them the six quadrature points, the rest classification, weights,
// row walk, sums and the deferred classes).  Four CTAs per SM (64 registers): the same 192
// requests on the 16384^2 mixed map 13.5 ms, at three 14.3, at five and six 13.7, at
// eight 15.8;
// with the FP64 path for every partly visible triangle it was 79 ms.  Splitting the
// larger triangles instead of taking them in FP64: 1000 small footprints on a
// scratch map, whose grooves have many, 0.49 -> 0.34 ms.
template <int TFMT>
__global__ void __launch_bounds__(256, kAreaCtas) pa_items(MapDesc d, const pndf_query *__restrict__ qs,
                                               const float *__restrict__ omega, int64_t k0, int cnt,
                                               const uint32_t *__restrict__ off, float2 *__restrict__ part,
                                               unsigned int *__restrict__ cursor)
{
    __shared__ WarpArea wa_s[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t total = off[cnt];
    while (true) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(cursor, 1u);
        it = __shfl_sync(kFull, it, 0);
        if (it >= total) break;
        // request owning this item: last t with off[t] <= it
        int lo = 0, hi = cnt - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= it)
                lo = mid;
            else
                hi = mid - 1;
        }
        const int t = lo;
        const Req q = make_req(qs[k0 + t], d.n);
        const Dir w = make_dir_f(omega[3 * (k0 + t)], omega[3 * (k0 + t) + 1], omega[3 * (k0 + t) + 2]);
        const float2 v = integrate_band<TFMT>(d, q, w, int(it - off[t]), lane, wa_s[warp]);
        if (lane == 0) part[it] = v;
    }
}

// A request's P from its bands [b0, b1): one warp, fixed-order compensated
// sum (lane 0 gets the value); NaN for an invalid covariance.
__device__ __forceinline__ bool request_valid(const pndf_query &r)
{
    const float det = r.sxx * r.syy - r.sxy * r.sxy;
    return (r.sxx > 0.f) && (r.syy > 0.f) && (det > 0.f) && isfinite(det) && isfinite(r.x) && isfinite(r.y);
}

__device__ __forceinline__ float reduce_bands(const float2 *__restrict__ part, uint32_t b0, uint32_t b1, int lane)
{
    float s = 0.f, c = 0.f;
    for (uint32_t b = b0 + lane; b < b1; b += 32) {
        float2 p = part[b];
        float tt = s + p.x;
        c += (fabsf(s) >= fabsf(p.x) ? (s - tt) + p.x : (p.x - tt) + s) + p.y;
        s = tt;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float so = __shfl_down_sync(kFull, s, o), co = __shfl_down_sync(kFull, c, o);
        float tt = s + so;
        float err = fabsf(s) >= fabsf(so) ? (s - tt) + so : (so - tt) + s;
        s = tt;
        c += co + err;
    }
    return s + c;
}

// one warp per request: fixed-order sum of its bands
__global__ void pa_reduce(const pndf_query *__restrict__ qs, int64_t k0, int cnt, const uint32_t *__restrict__ off,
                          const float2 *__restrict__ part, float *__restrict__ P, unsigned int *hier_status)
{
    const int lane = threadIdx.x & 31;
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= cnt) return;
    const float v = reduce_bands(part, off[t], off[t + 1], lane);
    if (lane == 0) {
        const bool valid = request_valid(qs[k0 + t]);
        if (!valid) record_status(hier_status, &g_status_projarea, PNDF_QF_INVALID);
        P[k0 + t] = valid ? v : __int_as_float(0x7fc00000);
    }
}

// ---- projected-area requests inside a serving step (area_step.cuh) ----

constexpr int kStepMaxMaps = kServeMaxMaps;

__global__ void area_step_bands(const MapDesc *__restrict__ maps, const uint32_t *__restrict__ count,
                                const AreaReq *__restrict__ areq, uint32_t *__restrict__ nb)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < int(*count)) nb[t] = band_count(*areq[t].q, maps[areq[t].map].n);
}

__global__ void __launch_bounds__(1024) area_step_scan(const uint32_t *__restrict__ count, uint32_t *nb, unsigned int *cursor)
{
    scan_bands([&](int i) { return nb[i]; }, nb, int(*count), cursor);
}

__global__ void __launch_bounds__(1024) area_step_prep(const MapDesc *__restrict__ maps, const uint32_t *__restrict__ count,
                                                       const AreaReq *__restrict__ areq, uint32_t *nb, unsigned int *cursor)
{
    scan_bands([&](int i) { return band_count(*areq[i].q, maps[areq[i].map].n); }, nb, int(*count), cursor);
}

template <int TFMT>
__global__ void __launch_bounds__(256, kAreaCtas) area_step_items(const MapDesc *__restrict__ maps, int nmaps,
                                                      const uint32_t *__restrict__ count,
                                                      const AreaReq *__restrict__ areq,
                                                      const uint32_t *__restrict__ off, float2 *__restrict__ part,
                                                      unsigned int *__restrict__ cursor)
{
    __shared__ WarpArea wa_s[8];
    __shared__ MapDesc smaps[kStepMaxMaps];
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(maps);
        uint32_t *dst = reinterpret_cast<uint32_t *>(smaps);
        const int words = nmaps * int(sizeof(MapDesc) / sizeof(uint32_t));
        for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cnt = int(*count);
    if (cnt == 0) return;
    const uint32_t total = off[cnt];
    while (true) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(cursor, 1u);
        it = __shfl_sync(kFull, it, 0);
        if (it >= total) break;
        int lo = 0, hi = cnt - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (off[mid] <= it)
                lo = mid;
            else
                hi = mid - 1;
        }
        const AreaReq a = areq[lo];
        const MapDesc &d = smaps[a.map];
        const Req q = make_req(*a.q, d.n);
        const Dir w = make_dir_f(a.w[0], a.w[1], a.w[2]);
        const float2 v = integrate_band<TFMT>(d, q, w, int(it - off[lo]), lane, wa_s[warp]);
        if (lane == 0) part[it] = v;
    }
}

__global__ void area_step_reduce(const MapDesc *__restrict__ maps, const uint32_t *__restrict__ count,
                                 const AreaReq *__restrict__ areq, const uint32_t *__restrict__ off,
                                 const float2 *__restrict__ part)
{
    const int lane = threadIdx.x & 31;
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= int(*count)) return;
    const float v = reduce_bands(part, off[t], off[t + 1], lane);
    if (lane == 0) {
        const AreaReq a = areq[t];
        const bool valid = request_valid(*a.q);
        if (!valid) record_status(maps[a.map].status, &g_status_projarea, PNDF_QF_INVALID);
        *a.out = valid ? v : __int_as_float(0x7fc00000);
    }
}

// ---- GGX projected-area fit per mip node (Eq. 12) ----
//
// P'(w) = (w_z + sqrt(w_z^2 + w^T Omega w)) / 2 (Eq. 12, parentheses
// restored).  A node is box-filtered over its own quads, so its projected
// area is P(w) = 4^-l sum over its triangles of V_T / |cross| (Eq. 9-11,
// exact for the box); the fit takes P at the 16 fit directions, forms a_k =
// (2 P_k - w_z)^2 - w_z^2 = w^T Omega w and solves the 3 x 3 normal
// equations in FP64.  Leaf blocks are summed by one warp each (lane =
// triangle, FP32 per-triangle values with the FP64 path where needed); a
// parent's P is the mean of its children's.

struct GgxDirs {
    Dir w[kGgxDirs];
    double fit[3][kGgxDirs];  // least squares: Omega = fit a (the normal equations' matrix depends on w alone)
};

// Omega of a node from its P at the fit directions, one per lane (direction k,
// the 16 directions on lanes that differ in the bits SH..SH + 3); every lane
// gets it.  FP64: Omega is a difference of nearly equal terms.
template <int SH>
__device__ __forceinline__ float4 ggx_fit(double P, int k, const GgxDirs &dirs)
{
    const double wz = dirs.w[k].wz, t = 2.0 * P - wz, a = t * t - wz * wz;
    double x[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        x[c] = dirs.fit[c][k] * a;
#pragma unroll
        for (int o = 1 << SH; o < (16 << SH); o <<= 1) x[c] += __shfl_xor_sync(kFull, x[c], o);
    }
    return make_float4(float(x[0]), float(x[1]), float(x[2]), 0.f);
}

__device__ __forceinline__ bool ggx_node_inside(const MapDesc &d, int l, uint32_t m)
{
    const int64_t a = int64_t(1) << l;
    return a * (compact1by1(m) + 1) <= int64_t(d.n) - 1 && a * (compact1by1(m >> 1) + 1) <= int64_t(d.n) - 1;
}

// Vertices of triangle `lane` of leaf block (i0, j0) (lane = 2 quad + tri,
// quads row-major in the 4 x 4 block; tri 0 = (u0, u1, u2), 1 = (u3, u2, u1)).
template <int TFMT>
__device__ __forceinline__ void leaf_triangle(const MapDesc &d, int i0, int j0, int lane, float2 &a, float2 &b,
                                              float2 &c)
{
    const int q = lane >> 1, tri = lane & 1;
    const int i = i0 + (q & 3), j = j0 + (q >> 2);
    a = texel<TFMT>(d, i + tri, j + tri);
    b = texel<TFMT>(d, i + 1 - tri, j + tri);
    c = texel<TFMT>(d, i + tri, j + 1 - tri);
}

// One warp per leaf block (Morton index): P at the fit directions (NaN when
// the block has a quad outside the map) and the block's fit.  A lane integrates
// m / m~_z over its triangle once and has the directions that see all of it
// from that; the (triangle, direction) pairs that the visibility boundary
// crosses are listed and spread over the warp 32 at a time, and so are the few
// to be split.  The sums over the triangles run in a fixed order.  The
// whole fit of a 2048^2 mixed map takes 1.0 ms (17.2 ms with a closed-form integral
// per direction, FP64 for every partly visible pair and the 3 x 3 solve in FP64 by
// one lane), and Omega's error against 64 bits fell from 6e-6 to 6e-7.
constexpr int kGgxLeafWarps = 8;
static_assert(kGgxDirs == 16, "two lanes per direction in the sums, four bits in a listed pair");

template <int TFMT>
__global__ void __launch_bounds__(32 * kGgxLeafWarps, kGgxCtas) ggx_leaf(MapDesc d, GgxDirs dirs,
                                                               float *__restrict__ P, float4 *__restrict__ omega,
                                                               uint32_t nleaf)
{
    __shared__ float r_s[kGgxLeafWarps][kGgxDirs][32];
    __shared__ uint16_t item_s[kGgxLeafWarps][kGgxDirs * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (m >= nleaf) return;
    float *Pm = P + size_t(m) * kGgxDirs;
    if (!ggx_node_inside(d, kLeafLevel, m)) {
        if (lane < kGgxDirs) Pm[lane] = __int_as_float(0x7fc00000);
        if (lane == 0) omega[m] = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
        return;
    }
    float(*rs)[32] = r_s[warp];
    uint16_t *items = item_s[warp];
    const int i0 = int(compact1by1(m)) * kLeafQuads, j0 = int(compact1by1(m >> 1)) * kLeafQuads;
    uint32_t need[2] = {0u, 0u};  // directions (bits) whose pair is partly visible, and those to split
    {
        float2 na, nb, nc;
        leaf_triangle<TFMT>(d, i0, j0, lane, na, nb, nc);
        const float za = zof(na), zb = zof(nb), zc = zof(nc);
        const float h2 = longest2(na, nb, nc);
        auto f = [](float x, float y) {
            const float2 r = ratio_at(x, y);
            return V2{r.x, r.y};
        };
        const float zm = fminf(za, fminf(zb, zc)), z2 = zm * zm;
        const V2 mean = h2 <= kSmallH2 * (z2 * z2) ? quad4(na, sub(nb, na), sub(nc, na), f)
                                                    : quad6(na, sub(nb, na), sub(nc, na), f);
        for (int k = 0; k < kGgxDirs; ++k) {
            const Dir &w = dirs.w[k];
            const Class cl = classify(phi_of(w, na, za), phi_of(w, nb, zb), phi_of(w, nc, zc), za, zb, zc, h2, w);
            if (cl == kPartial)
                need[0] |= 1u << k;
            else if (cl == kSplit)
                need[1] |= 1u << k;
            else
                rs[k][lane] = cl == kNone ? 0.f : 0.5f * fmaf(w.wx, mean.x, fmaf(w.wy, mean.y, w.wz));
        }
    }
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
        // list the pairs (lane-major) and evaluate them 32 at a time
        uint32_t set = need[pass];
        const int cnt = __popc(set);
        if (!__any_sync(kFull, cnt > 0)) continue;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(kFull, incl, 31);
        for (int p = incl - cnt; set; set &= set - 1) items[p++] = uint16_t((lane << 4) | (__ffs(set) - 1));
        __syncwarp();
        for (int t0 = 0; t0 < total; t0 += 32) {
            if (t0 + lane < total) {
                const int it = items[t0 + lane], src = it >> 4, k = it & 15;
                float2 a, b, c;
                leaf_triangle<TFMT>(d, i0, j0, src, a, b, c);
                rs[k][src] = pass == 0 ? partial_ratio(a, b, c, dirs.w[k]) : split_ratio(a, b, c, dirs.w[k]);
            }
        }
        __syncwarp();
    }
    __syncwarp();
    // sums over the 32 triangles, 16 directions at once: each step halves the
    // directions a lane holds, so that lanes 2k and 2k + 1 end with direction k
    float v[kGgxDirs];
#pragma unroll
    for (int k = 0; k < kGgxDirs; ++k) v[k] = rs[k][lane];
#pragma unroll
    for (int h = kGgxDirs / 2; h >= 1; h >>= 1) {
        const int o = 2 * h;
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const float got = __shfl_xor_sync(kFull, up ? v[k] : v[k + h], o);
            v[k] = (up ? v[k + h] : v[k]) + got;
        }
    }
    const float p = (v[0] + __shfl_xor_sync(kFull, v[0], 1)) * (1.0f / float(kLeafQuads * kLeafQuads));
    if ((lane & 1) == 0) Pm[lane >> 1] = p;
    const float4 o = ggx_fit<1>(p, lane >> 1, dirs);
    if (lane == 0) omega[m] = o;
}

// 16 lanes per node of level l: P = mean of the four children's, then the fit.
// Above the leaf blocks P is kept in FP64: Omega is a small difference, and a
// rounding per level would show in the coarse ones.
template <class T>
__global__ void ggx_up(MapDesc d, int l, GgxDirs dirs, const T *__restrict__ Pc, double *__restrict__ Pp,
                       float4 *__restrict__ omega, uint32_t count)
{
    const uint32_t m = (blockIdx.x * blockDim.x + threadIdx.x) / kGgxDirs;
    const int k = threadIdx.x & (kGgxDirs - 1);
    const bool live = m < count;
    double v = 0.0;
    if (live)
        for (int c = 0; c < 4; ++c) v += double(Pc[(4 * size_t(m) + c) * kGgxDirs + k]);
    const double p = 0.25 * v;
    const unsigned half = 0xffffu << (threadIdx.x & 16);  // the node's lanes
    const bool fine = (__ballot_sync(kFull, isfinite(p)) & half) == half;
    const bool ok = live && ggx_node_inside(d, l, m) && fine;
    const float4 o = ggx_fit<0>(p, k, dirs);
    if (!live) return;
    Pp[size_t(m) * kGgxDirs + k] = ok ? p : __longlong_as_double(0x7ff8000000000000ll);
    if (k == 0) omega[m] = ok ? o : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
}

GgxDirs make_ggx_dirs()
{
    GgxDirs g;
    const double r = sqrt(1.0 - double(kGgxWz) * kGgxWz);
    double row[kGgxDirs][3], A[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int k = 0; k < kGgxDirs; ++k) {
        const double ph = 2.0 * 3.14159265358979323846 * k / kGgxDirs;
        Dir &w = g.w[k];
        w.wx = float(r * cos(ph));
        w.wy = float(r * sin(ph));
        w.wz = kGgxWz;
        row[k][0] = double(w.wx) * w.wx;
        row[k][1] = 2.0 * double(w.wx) * w.wy;
        row[k][2] = double(w.wy) * w.wy;
        for (int p = 0; p < 3; ++p)
            for (int q = 0; q < 3; ++q) A[p][q] += row[k][p] * row[k][q];
    }
    // fit = A^-1 rows^T, A^-1 by cofactors (A is symmetric and well conditioned)
    const double c00 = A[1][1] * A[2][2] - A[1][2] * A[2][1], c01 = A[1][2] * A[2][0] - A[1][0] * A[2][2];
    const double c02 = A[1][0] * A[2][1] - A[1][1] * A[2][0], c11 = A[0][0] * A[2][2] - A[0][2] * A[2][0];
    const double c12 = A[0][1] * A[2][0] - A[0][0] * A[2][1], c22 = A[0][0] * A[1][1] - A[0][1] * A[1][0];
    const double det = A[0][0] * c00 + A[0][1] * c01 + A[0][2] * c02;
    const double inv[3][3] = {{c00, c01, c02}, {c01, c11, c12}, {c02, c12, c22}};
    for (int c = 0; c < 3; ++c)
        for (int k = 0; k < kGgxDirs; ++k)
            g.fit[c][k] = (inv[c][0] * row[k][0] + inv[c][1] * row[k][1] + inv[c][2] * row[k][2]) / det;
    return g;
}

// Omega at a footprint: two mip levels around lambda = log2(sqrt(12) sigma),
// each bilinear between node centres, nodes without a fit dropped.
__device__ bool ggx_omega_at(const pndf_ggx &g, float x, float y, float sxx, float syy, float3 &O)
{
    const int L = g.L;
    float lam = log2f(3.4641016f * sqrtf(fmaxf(sxx, syy)));
    lam = fminf(fmaxf(lam, 2.0f), float(L));
    const int l0 = int(floorf(lam)), l1 = l0 < L ? l0 + 1 : l0;
    const float tl = lam - float(l0);
    float ax = 0.f, ay = 0.f, az = 0.f, wsum = 0.f;
    for (int side = 0; side < 2; ++side) {
        const int l = side ? l1 : l0;
        const float wl = side ? tl : 1.0f - tl;
        if (wl == 0.f) continue;
        const float a = float(1 << l);
        const int S = 1 << (L - l);
        const float fx = x / a - 0.5f, fy = y / a - 0.5f;
        const float flx = floorf(fx), fly = floorf(fy);
        const float tx = fx - flx, ty = fy - fly;
        float lx = 0.f, ly = 0.f, lz = 0.f, lw = 0.f;
        for (int dj = 0; dj < 2; ++dj)
            for (int di = 0; di < 2; ++di) {
                const int I = int(fminf(fmaxf(flx + di, 0.f), float(S - 1)));
                const int J = int(fminf(fmaxf(fly + dj, 0.f), float(S - 1)));
                const float4 o = g.omega[l][morton2(uint32_t(I), uint32_t(J))];
                if (!isfinite(o.x)) continue;
                const float w = (di ? tx : 1.f - tx) * (dj ? ty : 1.f - ty);
                lx += w * o.x;
                ly += w * o.y;
                lz += w * o.z;
                lw += w;
            }
        if (lw > 0.f) {
            ax += wl * lx / lw;
            ay += wl * ly / lw;
            az += wl * lz / lw;
            wsum += wl;
        }
    }
    if (!(wsum > 0.f)) return false;
    O = make_float3(ax / wsum, ay / wsum, az / wsum);
    return true;
}

__device__ __forceinline__ float ggx_lambda(const float3 &O, float wx, float wy, float wz)
{
    const float qf = O.x * wx * wx + 2.0f * O.y * wx * wy + O.z * wy * wy;
    return 0.5f * (wz + sqrtf(fmaxf(wz * wz + qf, 0.f))) / wz - 1.0f;
}

__global__ void ggx_eval(pndf_ggx g, const pndf_query *__restrict__ q, const float *__restrict__ wi,
                         const float *__restrict__ wo, int64_t n, float *__restrict__ out)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const pndf_query r = q[k];
        float3 O;
        if (!(r.sxx > 0.f && r.syy > 0.f) || !ggx_omega_at(g, r.x, r.y, r.sxx, r.syy, O)) {
            out[k] = __int_as_float(0x7fc00000);
            continue;
        }
        const float ix = wi[3 * k], iy = wi[3 * k + 1], iz = wi[3 * k + 2];
        const float li = ggx_lambda(O, ix, iy, iz);
        if (!wo) {
            out[k] = li;
            continue;
        }
        // height-correlated shadow-masking with the query normal m
        const float ox = wo[3 * k], oy = wo[3 * k + 1], oz = wo[3 * k + 2];
        const float mz = sqrtf(fmaxf(0.f, 1.0f - r.ms * r.ms - r.mt * r.mt));
        const float ci = r.ms * ix + r.mt * iy + mz * iz, co = r.ms * ox + r.mt * oy + mz * oz;
        out[k] = (ci > 0.f && co > 0.f) ? 1.0f / (1.0f + li + ggx_lambda(O, ox, oy, oz)) : 0.f;
    }
}

__global__ void ggx_copy(pndf_ggx g, int l, float *__restrict__ out)
{
    const uint32_t S = 1u << (g.L - l);
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S * S) return;
    const float4 o = g.omega[l][morton2(i % S, i / S)];
    out[3 * size_t(i)] = o.x;
    out[3 * size_t(i) + 1] = o.y;
    out[3 * size_t(i) + 2] = o.z;
}

}  // namespace

pndf_status launch_ggx_build(const pndf_hierarchy *h, pndf_ggx *g, cudaStream_t s)
{
    const MapDesc &d = h->d;
    const int L = d.L;
    const uint32_t nleaf = uint32_t(level_nodes(L, kLeafLevel));
    const size_t pbytes = size_t(nleaf) * kGgxDirs * sizeof(float);
    void *scratch = nullptr;
    if (cudaMallocAsync(&scratch, 2 * pbytes, s) != cudaSuccess) {
        cudaGetLastError();
        return PNDF_ERR_OOM;
    }
    float *pa = static_cast<float *>(scratch), *pb = pa + size_t(nleaf) * kGgxDirs;
    static const GgxDirs dirs = make_ggx_dirs();
    const unsigned blocks = unsigned((size_t(nleaf) + kGgxLeafWarps - 1) / kGgxLeafWarps);
    if (d.texel_fmt == PNDF_TEXEL_F32X2)
        ggx_leaf<PNDF_TEXEL_F32X2><<<blocks, 32 * kGgxLeafWarps, 0, s>>>(d, dirs, pa, g->omega[kLeafLevel], nleaf);
    else
        ggx_leaf<PNDF_TEXEL_F16X2><<<blocks, 32 * kGgxLeafWarps, 0, s>>>(d, dirs, pa, g->omega[kLeafLevel], nleaf);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    // the leaf blocks' P are floats in pa; the levels above alternate between
    // the two halves as doubles (a quarter of the nodes, twice the size)
    double *from = reinterpret_cast<double *>(pa), *to = reinterpret_cast<double *>(pb);
    for (int l = kLeafLevel + 1; e == cudaSuccess && l <= L; ++l) {
        const uint32_t cnt = uint32_t(level_nodes(L, l));
        const unsigned grid = unsigned((size_t(cnt) * kGgxDirs + 127) / 128);
        if (l == kLeafLevel + 1)
            ggx_up<float><<<grid, 128, 0, s>>>(d, l, dirs, pa, to, g->omega[l], cnt);
        else
            ggx_up<double><<<grid, 128, 0, s>>>(d, l, dirs, from, to, g->omega[l], cnt);
        count_launches(1);
        e = cudaGetLastError();
        double *t = from;
        from = to;
        to = t;
    }
    cudaError_t ef = cudaFreeAsync(scratch, s);
    return (e == cudaSuccess && ef == cudaSuccess) ? PNDF_OK : PNDF_ERR_CUDA;
}

cudaError_t launch_ggx_eval(const pndf_ggx *g, const pndf_query *q, const float *wi, const float *wo, int64_t n,
                            float *out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (n + 255) / 256;
    if (blocks > int64_t(sms) * 16) blocks = int64_t(sms) * 16;
    ggx_eval<<<unsigned(blocks), 256, 0, s>>>(*g, q, wi, wo, n, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_ggx_copy(const pndf_ggx *g, int l, float *out, cudaStream_t s)
{
    const uint32_t n = uint32_t(level_nodes(g->L, l));
    ggx_copy<<<(n + 255) / 256, 256, 0, s>>>(*g, l, out);
    count_launches(1);
    return cudaGetLastError();
}

int area_max_bands(int n) { return (n - 1 + kBand - 1) / kBand + 1; }

cudaError_t launch_area_step(int texel_fmt, const MapDesc *maps, int nmaps, const uint32_t *count,
                             const AreaReq *areq, int cap, uint32_t *off, float2 *part, unsigned int *cursor,
                             cudaStream_t s)
{
    if (cap <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cap <= kPrepSmall) {
        area_step_prep<<<1, 1024, 0, s>>>(maps, count, areq, off, cursor);
    } else {
        area_step_bands<<<(cap + 255) / 256, 256, 0, s>>>(maps, count, areq, off);
        area_step_scan<<<1, 1024, 0, s>>>(count, off, cursor);
    }
    int occ = 0;
    if (texel_fmt == PNDF_TEXEL_F32X2) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, area_step_items<PNDF_TEXEL_F32X2>, 256, 0);
        area_step_items<PNDF_TEXEL_F32X2><<<sms * (occ > 0 ? occ : 1), 256, 0, s>>>(maps, nmaps, count, areq, off,
                                                                                    part, cursor);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, area_step_items<PNDF_TEXEL_F16X2>, 256, 0);
        area_step_items<PNDF_TEXEL_F16X2><<<sms * (occ > 0 ? occ : 1), 256, 0, s>>>(maps, nmaps, count, areq, off,
                                                                                    part, cursor);
    }
    area_step_reduce<<<(cap * 32 + 255) / 256, 256, 0, s>>>(maps, count, areq, off, part);
    return cudaGetLastError();
}

pndf_status launch_projarea(const pndf_hierarchy *h, const pndf_query *q, const float *omega, int64_t nq, float *P,
                            cudaStream_t s)
{
    if (nq == 0) return PNDF_OK;
    const MapDesc &d = h->d;
    const int maxbands = area_max_bands(d.n);
    // requests per chunk: bounded by the scan (65536) and by 256 MiB of band partials
    int64_t chunk = (int64_t(1) << 28) / (int64_t(sizeof(float2)) * maxbands);
    if (chunk > 65536) chunk = 65536;
    if (chunk < 1024) chunk = 1024;
    if (chunk > nq) chunk = nq;
    size_t off_bytes = ((size_t(chunk) + 1) * sizeof(uint32_t) + 255) & ~size_t(255);
    size_t part_bytes = size_t(chunk) * maxbands * sizeof(float2);
    void *scratch = nullptr;
    if (cudaMallocAsync(&scratch, 256 + off_bytes + part_bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return PNDF_ERR_OOM;
    }
    char *base = static_cast<char *>(scratch);
    auto *cursor = reinterpret_cast<unsigned int *>(base);
    auto *off = reinterpret_cast<uint32_t *>(base + 256);
    auto *part = reinterpret_cast<float2 *>(base + 256 + off_bytes);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaSuccess;
    for (int64_t k0 = 0; k0 < nq && e == cudaSuccess; k0 += chunk) {
        int cnt = int(nq - k0 < chunk ? nq - k0 : chunk);
        if (cnt <= kPrepSmall) {
            pa_prep<<<1, 1024, 0, s>>>(d, q, k0, cnt, off, cursor);
        } else {
            pa_bands<<<(cnt + 255) / 256, 256, 0, s>>>(d, q, k0, cnt, off);
            pa_scan<<<1, 1024, 0, s>>>(off, cnt, cursor);
            count_launches(1);
        }
        int occ = 0;
        if (d.texel_fmt == PNDF_TEXEL_F32X2) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pa_items<PNDF_TEXEL_F32X2>, 256, 0);
            pa_items<PNDF_TEXEL_F32X2><<<sms * (occ > 0 ? occ : 1), 256, 0, s>>>(d, q, omega, k0, cnt, off, part, cursor);
        } else {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pa_items<PNDF_TEXEL_F16X2>, 256, 0);
            pa_items<PNDF_TEXEL_F16X2><<<sms * (occ > 0 ? occ : 1), 256, 0, s>>>(d, q, omega, k0, cnt, off, part, cursor);
        }
        pa_reduce<<<(cnt * 32 + 255) / 256, 256, 0, s>>>(q, k0, cnt, off, part, P, d.status);
        count_launches(3);
        e = cudaGetLastError();
    }
    cudaError_t ef = cudaFreeAsync(scratch, s);
    if (e != cudaSuccess || ef != cudaSuccess) return PNDF_ERR_CUDA;
    return PNDF_OK;
}

namespace {
__global__ void take_projarea_word(unsigned int *out) { *out = atomicExch(&g_status_projarea, 0u); }
}  // namespace

cudaError_t take_status_projarea(unsigned int *out, cudaStream_t s)
{
    take_projarea_word<<<1, 1, 0, s>>>(out);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace pndf

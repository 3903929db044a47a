// Batched P-NDF evaluation over the position-normal manifold (Sec. 4.1-4.2).
//
// Per query (footprint centre x, covariance S, normal m) the result is Eq. 5:
//   D = sum over triangles abc with m in n(abc) of
//       k_r(a l0 + b l1 + c l2 - x) / |(n_b - n_a) x (n_c - n_a)|.
//
// Pipeline (all on the caller's stream):
//   key_hist  : per query a key of 4 + sub bits: the entry level (App. C; the
//               smallest level whose node side reaches the support's
//               half-width), largest footprints first, above a sub-key of 6..14
//               bits (footprint tile and/or query-normal bin); counted into a
//               global histogram with atomics.
//   key_scan  : exclusive scan of the histogram (one CTA).
//   key_place : counting-sort placement -> query order.
//   traverse  : persistent warps pull queries from an atomic cursor; one warp
//               per query.  Depth-first descent of the min/max pyramid with a
//               per-warp shared-memory stack: each step pops up to kPop nodes,
//               lane k tests child (k & 3) of popped nodes (k >> 2) + 8 r - the
//               normal box and the slab (common.cuh: the tight bound where a
//               node straddles two normal regions) against m, then the uv box
//               against the support - and ballot/popc compaction pushes the
//               survivors.  Surviving leaf blocks (4 x 4 quads) have the
//               box and slab of their four 2 x 2-quad groups tested, sixteen
//               blocks per pass; surviving groups are compacted into a
//               per-warp ring and taken 32 at a time (lane = group): the
//               group's nine texels give the edge functions of its eight
//               triangles at once (16 edges), and the triangles that may hold
//               m, nearly all of them hits, are compacted again and decided
//               and weighed 32 at a time (lane = triangle).  Each weight is
//               added exactly into the thread's 128-bit fixed-point sum;
//               the warp's sums are added exactly and the total is written in
//               caller order (the unpermute is fused into the store).  Large
//               footprints of a batch are divided into tiles of nodes, one
//               warp per tile (split_work / split_plan).  Flat mode skips
//               every box and tests all 32 triangles of every leaf block in
//               the support's bounding box.
//
// What bounds it: the descent is instruction issue and L2 latency in about equal
// parts (55% of the issue slots used, 4.7 of 11 cycles between a warp's issues
// spent on loads; the same footprints on maps from 2048^2 to 16384^2 take 18 to
// 23 ms, so DRAM is not the limit).  Per query of the 8192^2 flake workload it
// tests 10.7k nodes, 1.2k leaf blocks, 1.4k groups and 998 triangles for 990
// hits, in 59.7k warp instructions; with a box and a capsule per quad in place of
// the slabs and groups it took 187k, and 897 ms per 4M queries against 329 ms.
//
// Hit test (tie rule): m inside the closed normal bounding box and all three
// edge functions sign-consistent with the triangle orientation (>= 0 after
// orientation, i.e. closed barycentrics).  Zero-area normal triangles are a
// delta and are skipped.  Edge functions use an FMA difference of products on
// vertex-relative differences; triangles whose FP32 |cross| is below 2e-10
// (normal-space area below 1e-10) are re-tested and weighted in FP64.
#include <mutex>

#include "common.cuh"
#include "tri.cuh"

namespace pndf {

__device__ unsigned int g_status_eval;

namespace {

// Children a lane tests per step, all their loads in flight: three with FP16
// bounds, two with FP32 bounds, whose nodes take half as many registers again.
// 512k flake queries on 8192^2 at 2 / 3: FP16 50.1 / 44.9 ms, FP32 50.5 / 52.6 ms;
// 512k scratch queries, FP32, 6.9 / 7.2 ms (4 with FP16 was no better than 3).
template <int BFMT>
constexpr int kPer = BFMT == PNDF_BOUNDS_F32 ? 2 : 3;
constexpr int kPop = 24;           // nodes popped per step at most (four children each)
// DFS stack entries per warp.  A step leaves at most 3 kPop more than it found
// on the way down a level: 3 kPop per level below the entry (at most 12), the
// last step's 4 kPop and the 16 entry nodes.
constexpr int kStackCap = 36 * kPop + 4 * kPop + 16 + 16;
constexpr int kMaxSubBits = 14;                   // sub-key bits below the 4 entry-level bits
constexpr int kKeyBins = 1 << (4 + kMaxSubBits);  // largest histogram (2^18 bins)
// 3 x 256 threads per SM at 80 registers: 4 CTAs (64 registers, spills) took
// 5-10% longer on the flake map and 5 CTAs 24%
constexpr int kTraverseCtas = 3;
constexpr int kTraverseWarps = 8 * kTraverseCtas;  // resident per SM at the default launch shape
constexpr unsigned kFull = 0xffffffffu;

// MurmurHash3 32-bit finalizer (Appleby), fingerprints hit sets in stats mode.
__device__ __forceinline__ uint32_t fmix32(uint32_t h)
{
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// Internal kernel id of the Gaussian with the Jacobian clamp of Eq. 6.
constexpr int kKernGaussClamp = 3;

// Footprint kernels (pndf_kernel): the Gaussian cut at q = d^T S^-1 d <= 16,
// and the disk (q <= 1.5^2) and box (|L^-1 d|_inf <= 1.5, S = L L^T) filters
// of the (3 sigma)^2 footprints the paper pairs with it.
// The descent keeps its query in shared memory, one per warp, and reads the
// fields where it uses them: in registers they cost about 20 of each thread's.
template <int KERN>
struct alignas(16) Query {
    static constexpr int kernel = KERN == kKernGaussClamp ? PNDF_KERNEL_GAUSS : KERN;  // pndf_kernel
    float mx, my;        // query normal
    __half2 mlo, mhi;    // m rounded down / up to binary16 (exact tests against binary16 boxes)
    float x, y;          // footprint centre
    float ia, ib, ic;    // S^-1 = [[ia, ib], [ib, ic]]
    float norm;          // kernel normalisation: 1 / (2 pi, 2.25 pi or 9) sqrt(det S)
    float rx, ry;        // half-widths of the support's bounding box (slightly inflated)
    float qprune;        // the support lies in q <= qprune (16, 2.25, 4.5), with a margin
    float theta;         // r_x r_y of the support (exact half-widths); times tau for the cluster cut
    float kyx, kxy;      // -ib / ic and -ib / ia: the minimiser of q along a vertical / horizontal line
    float nprune, ncorner;  // norms sqrt(q): of the prune limit, and of the offset (1, 1) at its larger sign
    float inv_sxx;       // box: 1 / S_xx, so that (L^-1 d)_x^2 = dx^2 / S_xx
    float l11, l21, l22; // box: the Cholesky factor L of S (node tests by separating axes)
    float jac, rho;      // Eq. 6 clamp: Jacobian floor eps and the replacement's circumradius (0: off)
    bool valid;
};

template <int KERN>
__device__ __forceinline__ Query<KERN> make_query(const pndf_query &r, float jac_eps = 0.f)
{
    constexpr int kernel = Query<KERN>::kernel;
    Query<KERN> q;
    q.jac = q.rho = 0.f;
    if (KERN == kKernGaussClamp) {
        // equilateral replacement of area eps / 2: side^2 = 2 eps / sqrt(3), circumradius side / sqrt(3)
        q.jac = jac_eps;
        q.rho = sqrtf(2.0f * jac_eps / 1.7320508f) * 0.57735027f;
    }
    q.x = r.x;
    q.y = r.y;
    q.mx = r.ms;
    q.my = r.mt;
    q.mlo = __halves2half2(__float2half_rd(r.ms), __float2half_rd(r.mt));
    q.mhi = __halves2half2(__float2half_ru(r.ms), __float2half_ru(r.mt));
    float det = r.sxx * r.syy - r.sxy * r.sxy;
    q.valid = (r.sxx > 0.f) && (r.syy > 0.f) && (det > 0.f) && isfinite(det) && isfinite(r.x) &&
              isfinite(r.y) && isfinite(r.ms) && isfinite(r.mt);
    float inv = 1.0f / det;
    q.ia = r.syy * inv;
    q.ib = -r.sxy * inv;
    q.ic = r.sxx * inv;
    q.kyx = -q.ib / q.ic;
    q.kxy = -q.ib / q.ia;
    const float sx = sqrtf(r.sxx), sy = sqrtf(r.syy), sd = sqrtf(det);
    float hx, hy;
    q.inv_sxx = 0.f;
    q.l11 = q.l21 = q.l22 = 0.f;
    if (kernel == PNDF_KERNEL_DISK) {
        q.norm = 1.0f / (2.25f * kPi * sd);
        hx = 1.5f * sx;
        hy = 1.5f * sy;
        q.qprune = 2.25f * (1.0f + 1e-4f);
    } else if (kernel == PNDF_KERNEL_BOX) {
        q.norm = 1.0f / (9.0f * sd);
        const float l21 = r.sxy / sx, l22 = sqrtf(fmaxf(r.syy - l21 * l21, 0.f));
        hx = 1.5f * sx;
        hy = 1.5f * (fabsf(l21) + l22);
        q.qprune = 4.5f * (1.0f + 1e-4f);  // |v|_inf <= 1.5 implies |v|^2 <= 4.5
        q.inv_sxx = 1.0f / r.sxx;
        q.l11 = sx;
        q.l21 = l21;
        q.l22 = l22;
    } else {
        q.norm = 1.0f / (2.0f * kPi * sd);
        hx = 4.0f * sx;  // q <= 16 implies |dx| <= 4 sqrt(sxx)
        hy = 4.0f * sy;
        q.qprune = kQPrune;
    }
    q.nprune = sqrtf(q.qprune);
    q.ncorner = sqrtf(q.ia + q.ic + 2.0f * fabsf(q.ib)) * (1.0f + 1e-5f);
    q.theta = hx * hy;
    // inflate so rounding never clips the support's box
    q.rx = hx * (1.0f + 1e-5f) + 1e-6f;
    q.ry = hy * (1.0f + 1e-5f) + 1e-6f;
    return q;
}

// Kernel weight at offset d with q = d^T S^-1 d; 0 outside the support.
template <class Q>
__device__ __forceinline__ float kweight(const Q &q, float dx, float qq)
{
    if (Q::kernel == PNDF_KERNEL_GAUSS) return qq <= kQCut ? q.norm * expf(-0.5f * qq) : 0.f;
    if (Q::kernel == PNDF_KERNEL_DISK) return qq <= 2.25f ? q.norm : 0.f;
    const float v1 = dx * dx * q.inv_sxx;  // (L^-1 d)_x^2; (L^-1 d)_y^2 = q - v1
    return (v1 <= 2.25f && qq - v1 <= 2.25f) ? q.norm : 0.f;
}

template <class Q>
__device__ __forceinline__ double kweight_d(const Q &q, double dx, double qq)
{
    if (Q::kernel == PNDF_KERNEL_GAUSS) return qq <= double(kQCut) ? double(q.norm) * exp(-0.5 * qq) : 0.0;
    if (Q::kernel == PNDF_KERNEL_DISK) return qq <= 2.25 ? double(q.norm) : 0.0;
    const double v1 = dx * dx * double(q.inv_sxx);
    return (v1 <= 2.25 && qq - v1 <= 2.25) ? double(q.norm) : 0.0;
}

template <class Q>
__device__ __forceinline__ float qform(const Q &q, float dx, float dy)
{
    return fmaf(q.ia * dx, dx, fmaf(2.0f * q.ib * dx, dy, q.ic * dy * dy));
}

// Minimum of q over the box [dx0, dx1] x [dy0, dy1] (offsets from the centre).
// The quadratic is convex with its minimum at the origin; off the box, the
// minimum lies on an edge whose outer side holds the origin, where it is a
// clamped 1D minimum (along x = X at y = -(ib / ic) X, the ratio precomputed
// per query; a minimiser off by rounding raises the value only to second
// order, far inside the pruning margin).
template <class Q>
__device__ __forceinline__ float qmin_box(const Q &q, float dx0, float dx1, float dy0, float dy1)
{
    if (dx0 <= 0.f && dx1 >= 0.f && dy0 <= 0.f && dy1 >= 0.f) return 0.f;
    float best = __int_as_float(0x7f800000);
    if (dx0 > 0.f || dx1 < 0.f) {
        float X = dx0 > 0.f ? dx0 : dx1;
        float y = fminf(fmaxf(q.kyx * X, dy0), dy1);
        best = fminf(best, qform(q, X, y));
    }
    if (dy0 > 0.f || dy1 < 0.f) {
        float Y = dy0 > 0.f ? dy0 : dy1;
        float x = fminf(fmaxf(q.kxy * Y, dx0), dx1);
        best = fminf(best, qform(q, x, Y));
    }
    return best;
}

// Node k as stored: FP16 bounds, the 16-byte record; FP32 bounds, the box, with
// the slab loaded beside it.
template <int BFMT>
struct Node {
    uint4 v;
    uint2 s;  // FP32 bounds only
};

template <int BFMT>
__device__ __forceinline__ Node<BFMT> load_node(const MapDesc &d, uint32_t k)
{
    Node<BFMT> n;
    n.v = __ldg(d.nodes + k);
    if (BFMT == PNDF_BOUNDS_F32) n.s = __ldg(d.slabs + k);
    return n;
}

template <int TFMT>
__device__ __forceinline__ float2 texel(const MapDesc &d, int i, int j)
{
    size_t idx = size_t(j) * d.n + i;
    if (TFMT == PNDF_TEXEL_F32X2) return __ldg(reinterpret_cast<const float2 *>(d.texels) + idx);
    __half2 h = __ldg(reinterpret_cast<const __half2 *>(d.texels) + idx);
    return __half22float2(h);
}

// Box kernel: does [dx0, dx1] x [dy0, dy1] (offsets from the centre) meet the
// support L [-1.5, 1.5]^2?  Separating axes: x and y (the support's extents
// are the inflated half-widths rx, ry) and n = (-l21, l11), normal to L e1,
// onto which the support projects to +-1.5 l11 l22 (slightly inflated).
template <class Q>
__device__ __forceinline__ bool box_support_meets(const Q &q, float dx0, float dx1, float dy0, float dy1)
{
    if (dx0 > q.rx || dx1 < -q.rx || dy0 > q.ry || dy1 < -q.ry) return false;
    const float hn = 1.5f * q.l11 * q.l22 * (1.0f + 1e-4f) + 1e-6f;
    const float p0 = -q.l21 * dx0, p1 = -q.l21 * dx1;
    const float pmin = fminf(p0, p1) + q.l11 * dy0, pmax = fmaxf(p0, p1) + q.l11 * dy1;
    return pmin <= hn && pmax >= -hn;
}

// Node (level l, coords a, c): uv box [a 2^l, (a+1) 2^l] x [c 2^l, (c+1) 2^l].
// It can hold a contributing hit only if that box meets the kernel's support
// (the ellipse q <= qprune; for the box kernel the sheared square itself).
template <class Q>
__device__ __forceinline__ bool node_in_footprint(const Q &q, int l, uint32_t a, uint32_t c)
{
    float sz = float(1u << l);
    float dx0 = float(a) * sz - q.x, dy0 = float(c) * sz - q.y;
    if (Q::kernel == PNDF_KERNEL_BOX) return box_support_meets(q, dx0, dx0 + sz, dy0, dy0 + sz);
    return qmin_box(q, dx0, dx0 + sz, dy0, dy0 + sz) <= q.qprune;
}

// The node's uv box lies entirely inside the pruning region (the quadratic is
// convex, so its maximum over the box is at a corner; the box kernel's
// support is convex too); every descendant then passes the footprint test
// and skips it.  Claiming "inside" wrongly would only prune less.
template <class Q>
__device__ __forceinline__ bool node_inside(const Q &q, int l, uint32_t a, uint32_t c)
{
    float sz = float(1u << l);
    float dx0 = float(a) * sz - q.x, dy0 = float(c) * sz - q.y;
    float dx1 = dx0 + sz, dy1 = dy0 + sz;
    if (Q::kernel == PNDF_KERNEL_BOX) {  // the support is convex: all four corners inside it
        const float hx = 1.5f * q.l11, hv = 1.5f * q.l22, k = q.l21 / q.l11;
        return fmaxf(fabsf(dx0), fabsf(dx1)) <= hx && fabsf(dy0 - k * dx0) <= hv && fabsf(dy0 - k * dx1) <= hv &&
               fabsf(dy1 - k * dx0) <= hv && fabsf(dy1 - k * dx1) <= hv;
    }
    float m = fmaxf(fmaxf(qform(q, dx0, dy0), qform(q, dx1, dy0)), fmaxf(qform(q, dx0, dy1), qform(q, dx1, dy1)));
    return m <= q.qprune;
}

// The descent's own version of the two tests above: does node (l, a, c) meet
// the support, and does it lie inside?  N = sqrt(q) is a norm, so every point
// of the node is within N <= h ncorner of its centre (h: half its side), which
// gives both answers from one evaluation of q, looser than the exact box by
// part of a node.  It nests: a node that meets the support by this test has a
// parent that does, and the parent of a node that does not may not be inside;
// so which leaf blocks are reached does not depend on the level a descent
// starts from.  (The box kernel's support is no norm ball of q.)
template <class Q>
__device__ __forceinline__ bool node_meets(const Q &q, int l, uint32_t a, uint32_t c, bool &inside)
{
    if (Q::kernel == PNDF_KERNEL_BOX) {
        const bool meets = node_in_footprint(q, l, a, c);
        inside = meets && node_inside(q, l, a, c);
        return meets;
    }
    const float sz = float(1u << l), e = 0.5f * sz * q.ncorner;
    const float qq = qform(q, fmaf(float(a) + 0.5f, sz, -q.x), fmaf(float(c) + 0.5f, sz, -q.y));
    const float lo = fmaxf(q.nprune - e, 0.f), hi = q.nprune + e;
    inside = qq < lo * lo;
    return !(qq > hi * hi);
}

// m in the box; with the clamp (CLAMP) widened by the replacement radius (a
// replacement lies within rho of its triangle's centroid, hence of its box).
template <bool CLAMP, class Q>
__device__ __forceinline__ bool box_holds(const float4 &b, const Q &q)
{
    if (CLAMP) return q.mx >= b.x - q.rho && q.mx <= b.z + q.rho && q.my >= b.y - q.rho && q.my <= b.w + q.rho;
    return q.mx >= b.x && q.mx <= b.z && q.my >= b.y && q.my <= b.w;
}

// m in a binary16 box.  For a binary16 bound b, m >= b exactly when m rounded
// down to binary16 is, and m <= b when m rounded up is, so two packed compares
// decide what four conversions and compares of FP32 values would.
template <bool CLAMP, class Q>
__device__ __forceinline__ bool half_box_holds(uint32_t lo, uint32_t hi, const Q &q)
{
    const __half2 l = *reinterpret_cast<const __half2 *>(&lo), h = *reinterpret_cast<const __half2 *>(&hi);
    if (CLAMP) {
        const float2 lf = __half22float2(l), hf = __half22float2(h);
        return box_holds<CLAMP>(make_float4(lf.x, lf.y, hf.x, hf.y), q);
    }
    return __hbge2(q.mlo, l) && __hble2(q.mhi, h);
}

// m in a node's box.
template <int BFMT, bool CLAMP, class Q>
__device__ __forceinline__ bool node_box_holds(const Node<BFMT> &n, const Q &q)
{
    if (BFMT == PNDF_BOUNDS_F32)
        return box_holds<CLAMP>(make_float4(__uint_as_float(n.v.x), __uint_as_float(n.v.y), __uint_as_float(n.v.z),
                                            __uint_as_float(n.v.w)), q);
    return half_box_holds<CLAMP>(n.v.x, n.v.y, q);
}

// How far a slab is widened: with the clamp, a replacement lies within rho of
// its triangle's centroid (|direction| <= 1 + 2^-10).
template <bool CLAMP, class Q>
__device__ __forceinline__ float slab_slack(const Q &q)
{
    return CLAMP ? q.rho * 1.01f : 0.f;
}

template <int BFMT, bool CLAMP, class Q>
__device__ __forceinline__ bool node_slab_holds(const Node<BFMT> &n, const Q &q)
{
    return BFMT == PNDF_BOUNDS_F32 ? slab_holds(n.s.x, n.s.y, q.mx, q.my, slab_slack<CLAMP>(q))
                                   : slab_holds(n.v.z, n.v.w, q.mx, q.my, slab_slack<CLAMP>(q));
}

// Stack / leaf-queue entry: the node's index (node_index; below 2^25 for L <=
// 14) and "inside the ellipse" in bit 31.
constexpr uint32_t kInside = 0x80000000u;

__device__ __forceinline__ int node_level(uint32_t k, int L) { return L - ((31 - __clz(int(k))) >> 1); }

// A query's sum is exact: every contribution (an FP32 value >= 0) is added
// into a 128-bit fixed-point number with 64 fraction bits, value =
// (hi 2^64 + lo) 2^-64, so the result does not depend on the order in which
// the hits are found or on how the query's work is divided among warps.  A
// contribution is rounded to the nearest multiple of 2^-64 (5.4e-20) once;
// the total is rounded to FP32 once at the end.  A contribution of 2^63 or
// more, or a sum past 2^64 (only possible for normal triangles of area far
// below 1e-20), marks the query kHuge and its D is +inf.
// The sum lives in shared memory (one 128-bit slot per thread of the CTA,
// at most 256 threads), so the descent keeps its registers; the counters and
// flags stay in registers.
struct Acc {
    uint32_t hits, hash, tests, fp64, degen, leaves, nodes, quads, cchecks, clusters;
    uint32_t flags;
};
constexpr uint32_t kHuge = 1u << 30;  // internal flag bit: the sum is out of the fixed-point range
__shared__ unsigned long long s_sum_lo[256], s_sum_hi[256];

__device__ __forceinline__ void acc_zero()
{
    s_sum_lo[threadIdx.x] = 0ull;
    s_sum_hi[threadIdx.x] = 0ull;
}

__device__ __forceinline__ void acc_add(Acc &a, float w)
{
    const uint32_t b = __float_as_uint(w);
    const int ex = int(b >> 23);  // sign 0: the biased exponent
    if (ex == 0 || (b >> 31)) return;  // zero or subnormal (< 2^-126: rounds to 0)
    if (ex >= 127 + 63) {              // 2^63 or more, inf or NaN
        a.flags |= kHuge;
        return;
    }
    const unsigned long long m = (b & 0x7fffffu) | 0x800000u;  // w = m 2^(ex - 150)
    const int sh = ex - 150 + 64;                               // w 2^64 = m 2^sh
    unsigned long long dl, dh = 0ull;
    if (sh < 0) {
        if (sh < -24) return;                        // below 2^-65: rounds to 0
        dl = (m + (1ull << (-sh - 1))) >> (-sh);     // round half up
    } else if (sh < 64) {
        dl = m << sh;
        if (sh > 40) dh = m >> (64 - sh);
    } else {
        dl = 0ull;
        dh = m << (sh - 64);  // sh <= 189 - 86: dh < 2^63
    }
    const unsigned long long lo = s_sum_lo[threadIdx.x] + dl;
    s_sum_lo[threadIdx.x] = lo;
    const unsigned long long h0 = s_sum_hi[threadIdx.x];
    const unsigned long long hi = h0 + dh + (lo < dl ? 1ull : 0ull);
    s_sum_hi[threadIdx.x] = hi;
    if (hi < h0) a.flags |= kHuge;  // past 2^64
}

// 128-bit fixed point -> FP32 (through FP64: deterministic, within an ulp).
__device__ __forceinline__ float acc_value(unsigned long long lo, unsigned long long hi, uint32_t flags)
{
    if (flags & kHuge) return __int_as_float(0x7f800000);
    return float(double(hi) + double(lo) * 0x1p-64);
}

// The quad's capsule: its two normal triangles lie within distance w of the
// segment between its two farthest normals (widened by `slack`).  Near-singular triangles are
// evaluated (and flagged) only when m is in the quad's box and capsule, so the
// flag does not depend on how the traversal got there.  The segment's ends are
// 8-bit fractions of the quad's box as stored in the bound format, w is
// rounded up to binary16 with a margin over FP32 rounding.
template <int BFMT>
__device__ __forceinline__ bool capsule_holds(float2 n0, float2 n1, float2 n2, float2 n3, float mx, float my, float slack)
{
    const float2 v[4] = {n0, n1, n2, n3};
    Box b = empty_box();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        b.smin = fminf(b.smin, v[k].x);
        b.tmin = fminf(b.tmin, v[k].y);
        b.smax = fmaxf(b.smax, v[k].x);
        b.tmax = fmaxf(b.tmax, v[k].y);
    }
    if (BFMT == PNDF_BOUNDS_F16_OUTWARD)
        b = Box{__half2float(__float2half_rd(b.smin)), __half2float(__float2half_rd(b.tmin)),
                __half2float(__float2half_ru(b.smax)), __half2float(__float2half_ru(b.tmax))};
    int ip = 0, iq = 1;
    float best = -1.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i + 1; j < 4; ++j) {
            const float dx = v[j].x - v[i].x, dy = v[j].y - v[i].y;
            const float d2 = fmaf(dx, dx, dy * dy);
            if (d2 > best) {
                best = d2;
                ip = i;
                iq = j;
            }
        }
    auto snap = [](float x, float lo, float hi) {  // x as an 8-bit fraction of [lo, hi]
        const float e = hi - lo;
        const float f = e > 0.f ? fminf(fmaxf(rintf((x - lo) / e * 255.0f), 0.f), 255.f) : 0.f;
        return fmaf(e * (1.0f / 255.0f), f, lo);
    };
    float2 p = v[0], r = v[0];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (i == ip) p = v[i];
        if (i == iq) r = v[i];
    }
    const float px = snap(p.x, b.smin, b.smax), py = snap(p.y, b.tmin, b.tmax);
    const float dx = snap(r.x, b.smin, b.smax) - px, dy = snap(r.y, b.tmin, b.tmax) - py;
    const float L2 = fmaf(dx, dx, dy * dy);
    float w = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float ax = v[k].x - px, ay = v[k].y - py;
        const float t = L2 > 0.f ? fminf(fmaxf(fmaf(ax, dx, ay * dy) / L2, 0.f), 1.f) : 0.f;
        const float ex = fmaf(-t, dx, ax), ey = fmaf(-t, dy, ay);
        w = fmaxf(w, sqrtf(fmaf(ex, ex, ey * ey)));
    }
    w = __half2float(__float2half_ru(fmaf(w, 1.0f + 1.0f / 512.0f, 1.0f / 2097152.0f))) + slack;
    const float ax = mx - px, ay = my - py, t = fmaf(ax, dx, ay * dy), w2 = w * w;
    if (t <= 0.f) return fmaf(ax, ax, ay * ay) <= w2;
    if (t >= L2) {
        const float bx = ax - dx, by = ay - dy;
        return fmaf(bx, bx, by * by) <= w2;
    }
    const float cr = fmaf(ax, dy, -ay * dx);
    return cr * cr <= w2 * L2;
}

// A near-singular normal triangle (FP32 |cross| below kTinyCross) that holds m
// in its bounding box: hit test and weight in FP64.  Returns the contribution
// (0: none) and what became of it.
struct Tiny {
    float w;
    int state;  // 0: no area, 1: evaluated, 2: out of reach (support or capsule), 3: evaluated in FP32
};
template <class Q>
__device__ __forceinline__ Tiny tiny_triangle(const Q &q, float2 na, float2 nb, float2 nc, int ai, int aj, float dir)
{
    double ax = na.x, ay = na.y, bx = nb.x, by = nb.y, cx = nc.x, cy = nc.y, mx = q.mx, my = q.my;
    double dcr = orient_d(ax, ay, bx, by, cx, cy);
    if (dcr == 0.0) return Tiny{0.f, 0};
    double e0 = orient_d(bx, by, cx, cy, mx, my);
    double e1 = orient_d(cx, cy, ax, ay, mx, my);
    double e2 = orient_d(ax, ay, bx, by, mx, my);
    bool hit = dcr > 0.0 ? (e0 >= 0.0 && e1 >= 0.0 && e2 >= 0.0) : (e0 <= 0.0 && e1 <= 0.0 && e2 <= 0.0);
    if (!hit) return Tiny{0.f, 1};
    double dl1 = e1 / dcr, dl2 = e2 / dcr;
    double dx = (double(ai) - double(q.x)) + dir * dl1;
    double dy = (double(aj) - double(q.y)) + dir * dl2;
    double qq = double(q.ia) * dx * dx + 2.0 * double(q.ib) * dx * dy + double(q.ic) * dy * dy;
    double w = kweight_d(q, dx, qq);
    if (w == 0.0) return Tiny{0.f, 1};
    return Tiny{float(w / fabs(dcr)), 1};
}

template <bool STATS>
__device__ __forceinline__ void add_tiny(const Tiny &t, uint32_t id, Acc &acc)
{
    if (t.state == 0 || t.state == 2) {
        if (STATS && t.state == 0) acc.degen++;
        return;
    }
    if (STATS) acc.fp64 += t.state == 1 ? 1u : 0u;
    acc.flags |= t.state == 1 ? PNDF_QF_FP64 : 0u;
    if (t.w == 0.f) return;
    acc_add(acc, t.w);
    if (STATS) {
        acc.hits++;
        acc.hash += fmix32(id);
    }
}

// m in the closed bounding box of (a, b, c), with the clamp widened by rho.
template <bool CLAMP, class Q>
__device__ __forceinline__ bool tri_box_holds(const Q &q, float2 na, float2 nb, float2 nc)
{
    float lox = fminf(na.x, fminf(nb.x, nc.x)), hix = fmaxf(na.x, fmaxf(nb.x, nc.x));
    float loy = fminf(na.y, fminf(nb.y, nc.y)), hiy = fmaxf(na.y, fmaxf(nb.y, nc.y));
    if (CLAMP) {
        lox -= q.rho;
        hix += q.rho;
        loy -= q.rho;
        hiy += q.rho;
    }
    return !(q.mx < lox || q.mx > hix || q.my < loy || q.my > hiy);
}

// FP32 hit decision of a triangle with |cross| = |cr| >= kTinyCross.
template <class Q>
__device__ __forceinline__ bool edges_hold(const Q &q, float2 na, float2 nb, float2 nc, float cr, float &e1, float &e2)
{
    const float e0 = orient(nb.x, nb.y, nc.x, nc.y, q.mx, q.my);
    e1 = orient(nc.x, nc.y, na.x, na.y, q.mx, q.my);
    e2 = orient(na.x, na.y, nb.x, nb.y, q.mx, q.my);
    return cr > 0.f ? (e0 >= 0.f && e1 >= 0.f && e2 >= 0.f) : (e0 <= 0.f && e1 <= 0.f && e2 <= 0.f);
}

// Does an FP32 hit (cross cr, edge functions e1, e2) lie in its triangle?  Where the
// cross is rounding noise (normals on a line) so is the hit's place in uv, and it
// may lie in the support although the hit's node does not meet it, which node_meets
// lets by.  Such a hit counts only if the node meets the support by the exact test.
__device__ __forceinline__ bool in_place(float cr, float e1, float e2)
{
    return fabsf(e1 + e2) <= fabsf(cr) * (1.0f + 1e-6f);
}

// Kernel weight of an FP32 hit: cross cr and edge functions e1, e2 (so l1 = e1 / cr,
// l2 = e2 / cr) of triangle `tri` of the quad, or of the level-l cluster, at (gi,
// gj), whose uv legs are a = 2^l.
template <class Q>
__device__ __forceinline__ float kernel_at(const Q &q, int gi, int gj, int l, int tri, float cr, float e1, float e2)
{
    const float a = float(1 << l);
    const float inv = 1.0f / cr;
    const float dir = tri ? -a : a;
    const float dx = (float(gi + (tri << l)) - q.x) + dir * (e1 * inv);
    const float dy = (float(gj + (tri << l)) - q.y) + dir * (e2 * inv);
    return kweight(q, dx, qform(q, dx, dy));
}

// Add the contribution of such a hit; the Jacobian is cr / a^2.
template <bool STATS, class Q>
__device__ __forceinline__ void weigh(const Q &q, int gi, int gj, int l, int tri, float cr, float e1, float e2,
                                      uint32_t id, Acc &acc)
{
    const float a = float(1 << l);
    const float w = kernel_at(q, gi, gj, l, tri, cr, e1, e2);
    if (w == 0.f) return;
    acc_add(acc, w * (a * a) / fabsf(cr));
    if (STATS) {
        acc.hits++;
        acc.hash += fmix32(id);
    }
}

// Test triangle `tri` of quad (gi, gj) and add its contribution; tri 0: (u0,
// u1, u2) with a = (i, j), b = a + (1, 0), c = a + (0, 1); tri 1: (u3, u2, u1)
// with a = (i+1, j+1), b = a - (1, 0), c = a - (0, 1).
template <bool STATS, class Q>
__device__ __forceinline__ void test_triangle(const Q &q, float2 na, float2 nb, float2 nc, int gi, int gj, int tri,
                                              uint32_t tri_id, Acc &acc)
{
    if (STATS) acc.tests++;
    if (!tri_box_holds<false>(q, na, nb, nc)) return;
    const float cr = orient(na.x, na.y, nb.x, nb.y, nc.x, nc.y);
    if (fabsf(cr) >= kTinyCross) {
        float e1, e2;
        if (edges_hold(q, na, nb, nc, cr, e1, e2)) weigh<STATS>(q, gi, gj, 0, tri, cr, e1, e2, tri_id, acc);
        return;
    }
    add_tiny<STATS>(tiny_triangle(q, na, nb, nc, gi + tri, gj + tri, tri ? -1.f : 1.f), tri_id, acc);
}

// Hit fingerprint ids of cluster triangles (stats): this bit, the level from
// bit 27, the node's row-major index from bit 1 and the triangle.
constexpr uint32_t kClusterTag = 0x80000000u;

// Lanes 0..24 fetch the 5 x 5 texels of leaf block (a, c) (4 x 4 quads).
template <int TFMT>
__device__ __forceinline__ float2 leaf_texel(const MapDesc &d, uint32_t a, uint32_t c, int lane)
{
    const int i0 = int(a) << kLeafLevel, j0 = int(c) << kLeafLevel;
    int tc = lane % kLeafTexels, tr = lane / kLeafTexels;
    float2 tv = make_float2(0.f, 0.f);
    if (lane < kLeafTexels * kLeafTexels && i0 + tc < d.n && j0 + tr < d.n) tv = texel<TFMT>(d, i0 + tc, j0 + tr);
    return tv;
}

// All 32 lanes: test the 32 triangles of leaf block (a, c) whose texels the
// lanes hold in tv (lane t: quad t >> 1, triangle t & 1).
template <bool STATS, class Q>
__device__ __forceinline__ void test_leaf(const MapDesc &d, const Q &q, uint32_t a, uint32_t c, float2 tv,
                                          int lane, Acc &acc)
{
    const int n = d.n;
    const int i0 = int(a) << kLeafLevel, j0 = int(c) << kLeafLevel;
    int qd = lane >> 1, qx = qd & 3, qy = qd >> 2, tri = lane & 1;
    int base = qy * kLeafTexels + qx;
    int sa = tri ? base + kLeafTexels + 1 : base;
    int sb = tri ? base + kLeafTexels : base + 1;
    int sc = tri ? base + 1 : base + kLeafTexels;
    float2 na, nb, nc;
    na.x = __shfl_sync(kFull, tv.x, sa);
    na.y = __shfl_sync(kFull, tv.y, sa);
    nb.x = __shfl_sync(kFull, tv.x, sb);
    nb.y = __shfl_sync(kFull, tv.y, sb);
    nc.x = __shfl_sync(kFull, tv.x, sc);
    nc.y = __shfl_sync(kFull, tv.y, sc);
    int gi = i0 + qx, gj = j0 + qy;
    if (STATS && lane == 0) acc.leaves++;
    if (gi <= n - 2 && gj <= n - 2) {
        uint32_t id = 2u * (uint32_t(gj) * uint32_t(n - 1) + uint32_t(gi)) + uint32_t(tri);
        test_triangle<STATS>(q, na, nb, nc, gi, gj, tri, id, acc);
    }
}

// Leaf queue: up to 15 leaf blocks held over from the last step plus one
// step's children.
constexpr int kLeafQ = 16 + 4 * kPop;
// Cut ring, with the cluster cut only: cut nodes (at most 31 held over plus one
// step's children), tested 32 at a time.
constexpr int kCutRing = 128;
// Group ring: 2 x 2-quad groups whose box and slab hold m (at most 31 held over
// plus one pass's 64): Morton index at level 1 (at most 26 bits), kMarked where
// the group holds a near-singular triangle.
constexpr int kGroupRing = 128;
constexpr uint32_t kMarked = 0x80000000u;
// Triangle ring: triangles that may hold m (at most 31 held over plus 32):
// (i << 15) | (j << 1) | tri of quad (i, j).
constexpr int kTriRing = 64;
// Hit ring, with the cluster cut only: cluster triangles that hold m (few of
// those tested), waiting to be weighed 32 at a time, as (cross, e1, e2, (index
// in the box array << 1) | tri); at most 31 held over plus 32.
constexpr int kHitRing = 64;
// Shared memory per warp: DFS stack, leaf queue, the rings.
template <bool CLUSTER>
constexpr int kWarpSmemWords = kStackCap + kLeafQ + kGroupRing + kTriRing + (CLUSTER ? 4 * kHitRing + kCutRing : 0);
static_assert((kStackCap + kLeafQ + kGroupRing + kTriRing) % 4 == 0, "hit ring alignment");

// A warp's shared memory and the rings' heads and counts.
struct LeafState {
    uint32_t *groups, *tris;
    float4 *hits;
    uint32_t *cuts;
    uint32_t ghead, thead, hhead, chead;
    int ng, nt, nh, nc;
};

// Edge functions at m of the replacement of Eq. 6 for triangle (a, b, c): the
// equilateral one (vertex k at 90 + 120 k degrees around the centroid g, radius
// rho), in vertex-relative form p = m - E0.  True if it holds m.
template <class Q>
__device__ __forceinline__ bool replacement_holds(const Q &q, float2 na, float2 nb, float2 nc, float &ecr, float &e1,
                                                  float &e2)
{
    const float gx = (na.x + nb.x + nc.x) * (1.0f / 3.0f), gy = (na.y + nb.y + nc.y) * (1.0f / 3.0f);
    const float h = 0.8660254f * q.rho;  // E1 - E0 = rho (-sqrt3/2, -3/2), E2 - E0 = rho (sqrt3/2, -3/2)
    const float2 b = make_float2(-h, -1.5f * q.rho), c = make_float2(h, -1.5f * q.rho);
    const float2 p = make_float2(q.mx - gx, (q.my - gy) - q.rho);
    ecr = diff_prod(b.x, c.y, b.y, c.x);  // > 0: counter-clockwise
    const float e0 = diff_prod(c.x - b.x, p.y - b.y, c.y - b.y, p.x - b.x);
    e1 = diff_prod(p.x, c.y, p.y, c.x);
    e2 = diff_prod(b.x, p.y, b.y, p.x);
    return e0 >= 0.f && e1 >= 0.f && e2 >= 0.f;
}

// Triangle `tri` of quad (gi, gj) when it is near-singular or its hit is out of
// place: nothing unless its leaf block meets the support by the exact test, and,
// near-singular, m is in the quad's capsule.  Out of line and called from one place,
// so that the rare path costs the common one neither registers nor instruction
// fetches (with a call of its own for the hits out of place the flake workload took
// 8% longer, like this 0.1%).
template <int BFMT, int TFMT, bool CLAMP, class Q>
__device__ __noinline__ Tiny rare_triangle(const MapDesc &d, const Q &q, int gi, int gj, int tri)
{
    if (!node_in_footprint(q, kLeafLevel, uint32_t(gi) >> kLeafLevel, uint32_t(gj) >> kLeafLevel)) return Tiny{0.f, 2};
    const float2 n0 = texel<TFMT>(d, gi, gj), n1 = texel<TFMT>(d, gi + 1, gj);
    const float2 n2 = texel<TFMT>(d, gi, gj + 1), n3 = texel<TFMT>(d, gi + 1, gj + 1);
    const float2 na = tri ? n3 : n0, nb = tri ? n2 : n1, nc = tri ? n1 : n2;
    float cr = orient(na.x, na.y, nb.x, nb.y, nc.x, nc.y), e1, e2;
    const bool clamp = CLAMP && fabsf(cr) < q.jac;
    if (clamp || fabsf(cr) >= kTinyCross) {
        const bool hit = clamp ? replacement_holds(q, na, nb, nc, cr, e1, e2) : edges_hold(q, na, nb, nc, cr, e1, e2);
        const float w = hit ? kernel_at(q, gi, gj, 0, tri, cr, e1, e2) : 0.f;
        return Tiny{w == 0.f ? 0.f : w / fabsf(cr), 3};
    }
    if (!capsule_holds<BFMT>(n0, n1, n2, n3, q.mx, q.my, CLAMP ? q.rho : 0.f)) return Tiny{0.f, 2};
    // (two copies: with one, the register allocator's choices in the caller took the
    // flake workload 6% longer)
    return tri ? tiny_triangle(q, n3, n2, n1, gi + 1, gj + 1, -1.f) : tiny_triangle(q, n0, n1, n2, gi, gj, 1.f);
}

// All 32 lanes: lane k < cnt decides triangle k of the triangle ring and adds
// its contribution.
template <int BFMT, int TFMT, bool STATS, bool CLAMP, class Q>
__device__ __forceinline__ void test_tris(const MapDesc &d, const Q &q, const LeafState &ls, int cnt, int lane,
                                          Acc &acc)
{
    if (lane >= cnt) return;
    const uint32_t pk = ls.tris[(ls.thead + uint32_t(lane)) & (kTriRing - 1)];
    const int gi = int(pk >> 15), gj = int((pk >> 1) & 0x3fffu), tri = int(pk & 1u);
    const float2 na = texel<TFMT>(d, gi + tri, gj + tri);
    const float2 nb = texel<TFMT>(d, gi + 1 - tri, gj + tri), nc = texel<TFMT>(d, gi + tri, gj + 1 - tri);
    const uint32_t id = 2u * (uint32_t(gj) * uint32_t(d.n - 1) + uint32_t(gi)) + uint32_t(tri);
    if (STATS) acc.tests++;
    if (!tri_box_holds<CLAMP>(q, na, nb, nc)) return;
    const float cr = orient(na.x, na.y, nb.x, nb.y, nc.x, nc.y);
    if (CLAMP && fabsf(cr) < q.jac) {
        float ecr, e1, e2;
        if (!replacement_holds(q, na, nb, nc, ecr, e1, e2)) return;
        if (in_place(ecr, e1, e2)) {
            weigh<STATS>(q, gi, gj, 0, tri, ecr, e1, e2, id, acc);
            return;
        }
    } else if (fabsf(cr) >= kTinyCross) {
        float e1, e2;
        if (!edges_hold(q, na, nb, nc, cr, e1, e2)) return;
        if (in_place(cr, e1, e2)) {
            weigh<STATS>(q, gi, gj, 0, tri, cr, e1, e2, id, acc);
            return;
        }
    }
    add_tiny<STATS>(rare_triangle<BFMT, TFMT, CLAMP>(d, q, gi, gj, tri), id, acc);
}

// The 3 x 3 texels of group (i, j) (i, j even), rows j..j + 2; past the map's
// last row or column the last one again.  With an even n a row's first two
// FP32 (FP16) texels are one aligned 16-byte (8-byte) load.
template <int TFMT>
__device__ __forceinline__ void group_texels(const MapDesc &d, int i, int j, float2 (&t)[3][3])
{
    const int n = d.n;
    const int i2 = min(i + 2, n - 1);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int jr = min(j + r, n - 1);
        const size_t row = size_t(jr) * n;
        if ((n & 1) == 0) {  // i + 1 <= n - 1
            if (TFMT == PNDF_TEXEL_F32X2) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const float2 *>(d.texels) + row + i));
                t[r][0] = make_float2(v.x, v.y);
                t[r][1] = make_float2(v.z, v.w);
            } else {
                const uint2 v = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const __half2 *>(d.texels) + row + i));
                t[r][0] = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
                t[r][1] = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
            }
        } else {
            t[r][0] = texel<TFMT>(d, i, jr);
            t[r][1] = texel<TFMT>(d, min(i + 1, n - 1), jr);
        }
        t[r][2] = texel<TFMT>(d, i2, jr);
    }
}

// All 32 lanes: lane k < cnt takes group k of the group ring and finds the
// triangles of its four quads that may hold m.  With d_u = n_u - m, edge u -> v
// has m on its left when d_u x d_v > 0, so the group's 16 edges (12 sides, 4
// diagonals), two operations each, decide all eight triangles.  A triangle is
// dropped only when two of its edges differ in sign by more than `eps`; with M
// the largest |d| component, the rounding of these edge functions (2^-21 M^2)
// and of the exact test's (2^-21 M^2: differences of at most 2 M, each
// relative to 2^-24) add up to 2^-20 M^2, and eps is four times that.  The
// survivors (few beside the hits) are listed and decided 32 at a time.
template <int BFMT, int TFMT, bool STATS, bool CLAMP, class Q>
__device__ __forceinline__ void test_groups(const MapDesc &d, const Q &q, LeafState &ls, int cnt, int lane, Acc &acc)
{
    const unsigned lt = (1u << lane) - 1u;
    uint32_t cand = 0, base = 0;
    if (lane < cnt) {
        const uint32_t g = ls.groups[(ls.ghead + uint32_t(lane)) & (kGroupRing - 1)];
        const uint32_t m = g & ~kMarked;
        const int i = int(compact1by1(m)) * 2, j = int(compact1by1(m >> 1)) * 2;
        base = (uint32_t(i) << 15) | (uint32_t(j) << 1);
        float2 t[3][3];
        group_texels<TFMT>(d, i, j, t);
        float M = 0.f;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                t[r][c].x -= q.mx;
                t[r][c].y -= q.my;
                M = fmaxf(M, fmaxf(fabsf(t[r][c].x), fabsf(t[r][c].y)));
            }
        const float eps = M * M * 0x1p-18f;
        auto edge = [](const float2 &u, const float2 &v) { return fmaf(u.x, v.y, -(u.y * v.x)); };
        float H[3][2], V[2][3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c) H[r][c] = edge(t[r][c], t[r][c + 1]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) V[r][c] = edge(t[r][c], t[r + 1][c]);
        auto may = [&](float a, float b, float c) {
            const bool out = fminf(a, fminf(b, c)) < -eps && fmaxf(a, fmaxf(b, c)) > eps;
            // with the clamp, also whatever its cross (the edges' sum) may send to the replacement
            return !out || (CLAMP && !(fabsf(a + b + c) >= q.jac + eps));
        };
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = k >> 1, c = k & 1;
            const float dg = edge(t[r][c + 1], t[r + 1][c]);
            cand |= uint32_t(may(H[r][c], dg, -V[r][c])) << (2 * k);              // u0 u1 u2
            cand |= uint32_t(may(-H[r + 1][c], -dg, V[r][c + 1])) << (2 * k + 1);  // u3 u2 u1
        }
        if (g & kMarked) cand = 0xffu;
        // quads past the map's last row or column of quads do not exist
        if (i + 1 > d.n - 2) cand &= 0x33u;
        if (j + 1 > d.n - 2) cand &= 0x0fu;
        if (STATS) acc.quads += 4;
    }
    unsigned m = __ballot_sync(kFull, cand != 0u);
    while (m) {
        if (cand) {
            const uint32_t b = uint32_t(__ffs(int(cand)) - 1);
            cand &= cand - 1u;
            ls.tris[(ls.thead + uint32_t(ls.nt) + __popc(m & lt)) & (kTriRing - 1)] =
                base + ((b & 2u) << 14) + ((b & 4u) >> 1) + (b & 1u);
        }
        ls.nt += __popc(m);
        __syncwarp();
        if (ls.nt >= 32) {
            test_tris<BFMT, TFMT, STATS, CLAMP>(d, q, ls, 32, lane, acc);
            ls.thead += 32;
            ls.nt -= 32;
            __syncwarp();
        }
        m = __ballot_sync(kFull, cand != 0u);
    }
}

// Cluster triangle test (Sec. 4.2) in vertex-relative form: p = m - A,
// b = B - A, c = C - A.  Same rule as for a fine triangle (closed bounding box, edge
// functions sign-consistent with the orientation); the Jacobian of the
// cluster map is cross / 4^l, applied when the hit is weighed.  Triangles
// with FP32 |cross| < 2e-10 are decided and weighed here in FP64, if the node
// (l, I, J) meets the support exactly (node_meets lets some by).
template <bool STATS, class Q>
__device__ __forceinline__ bool cluster_edge_test(const Q &q, float2 p, float2 b, float2 c, int l, int ai,
                                                  int aj, float dir, uint32_t I, uint32_t J, uint32_t id, Acc &acc,
                                                  float &cr_o, float &e1_o, float &e2_o)
{
    if (STATS) acc.tests++;
    if (p.x < fminf(0.f, fminf(b.x, c.x)) || p.x > fmaxf(0.f, fmaxf(b.x, c.x)) ||
        p.y < fminf(0.f, fminf(b.y, c.y)) || p.y > fmaxf(0.f, fmaxf(b.y, c.y)))
        return false;
    float cr = diff_prod(b.x, c.y, b.y, c.x);
    if (fabsf(cr) >= kTinyCross) {
        float e0 = diff_prod(c.x - b.x, p.y - b.y, c.y - b.y, p.x - b.x);
        float e1 = diff_prod(p.x, c.y, p.y, c.x);
        float e2 = diff_prod(b.x, p.y, b.y, p.x);
        bool hit = cr > 0.f ? (e0 >= 0.f && e1 >= 0.f && e2 >= 0.f) : (e0 <= 0.f && e1 <= 0.f && e2 <= 0.f);
        cr_o = cr;
        e1_o = e1;
        e2_o = e2;
        return hit;
    }
    if (!node_in_footprint(q, l, I, J)) return false;
    double bx = b.x, by = b.y, cx = c.x, cy = c.y, px = p.x, py = p.y;
    double dcr = bx * cy - by * cx;
    if (dcr == 0.0) {
        if (STATS) acc.degen++;
        return false;
    }
    if (STATS) acc.fp64++;
    acc.flags |= PNDF_QF_FP64;
    double e0 = (cx - bx) * (py - by) - (cy - by) * (px - bx);
    double e1 = px * cy - py * cx;
    double e2 = bx * py - by * px;
    bool hit = dcr > 0.0 ? (e0 >= 0.0 && e1 >= 0.0 && e2 >= 0.0) : (e0 <= 0.0 && e1 <= 0.0 && e2 <= 0.0);
    if (!hit) return false;
    double dl1 = e1 / dcr, dl2 = e2 / dcr;
    double dx = (double(ai) - double(q.x)) + dir * dl1;
    double dy = (double(aj) - double(q.y)) + dir * dl2;
    double qq = double(q.ia) * dx * dx + 2.0 * double(q.ib) * dx * dy + double(q.ic) * dy * dy;
    const double w = kweight_d(q, dx, qq);
    if (w == 0.0) return false;
    double sc = double(1u << l);
    acc_add(acc, float(w * sc * sc / fabs(dcr)));
    if (STATS) {
        acc.hits++;
        acc.hash += fmix32(id);
    }
    return false;
}

// Node (l, a, c) meets the support by the exact test, out of line for a rare caller.
template <class Q>
__device__ __noinline__ bool meets_exactly(const Q &q, int l, uint32_t a, uint32_t c)
{
    return node_in_footprint(q, l, a, c);
}

// All 32 lanes: lane k < cnt weighs hit k of the hit ring.
template <bool STATS, class Q>
__device__ __forceinline__ void weigh_clusters(const MapDesc &d, const Q &q, const LeafState &ls, int cnt, int lane,
                                               Acc &acc)
{
    if (lane >= cnt) return;
    const float4 h = ls.hits[(ls.hhead + uint32_t(lane)) & (kHitRing - 1)];
    const uint32_t k = __float_as_uint(h.w) >> 1;
    const int tri = int(__float_as_uint(h.w) & 1u), l = node_level(k, d.L);
    const uint32_t m = k - node_index(d.L, l, 0);
    const uint32_t I = compact1by1(m), J = compact1by1(m >> 1);
    if (!in_place(h.x, h.y, h.z) && !meets_exactly(q, l, I, J)) return;
    const uint32_t id = kClusterTag | (uint32_t(l) << 27) | (((J << (d.L - l)) + I) << 1) | uint32_t(tri);
    weigh<STATS>(q, int(I << l), int(J << l), l, tri, h.x, h.y, h.z, id, acc);
}

// All 32 lanes: lane k < cnt tests the two cluster triangles of cut node k of
// the cut ring: lower (c00, c10, c01) at uv (O, O + (a,
// 0), O + (0, a)), upper (c11, c01, c10) at (O + (a, a), O + (0, a), O + (a,
// 0)), a = 2^l; hits join the hit ring.
template <bool STATS, class Q>
__device__ __forceinline__ void test_clusters(const MapDesc &d, const ClusterDesc &cd, const Q &q,
                                              LeafState &ls, int cnt, int lane, Acc &acc)
{
    const unsigned lt = (1u << lane) - 1u;
    bool h0 = false, h1 = false;
    float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
    if (lane < cnt) {
        const uint32_t k = ls.cuts[(ls.chead + uint32_t(lane)) & (kCutRing - 1)];
        const int l = node_level(k, d.L);
        const uint32_t m = k - node_index(d.L, l, 0);
        const float4 *rec = cd.cl + 2 * size_t(k);
        float4 r0 = __ldg(rec), r1 = __ldg(rec + 1);
        const uint32_t I = compact1by1(m), J = compact1by1(m >> 1);
        int ox = int(I) << l, oy = int(J) << l;
        int a = 1 << l;
        float2 p = make_float2(q.mx - r0.x, q.my - r0.y);
        float2 d10 = make_float2(r0.z, r0.w), d01 = make_float2(r1.x, r1.y), d11 = make_float2(r1.z, r1.w);
        // hit fingerprint id (stats): row-major node index at its level
        uint32_t id = kClusterTag | (uint32_t(l) << 27) | (((J << (d.L - l)) + I) << 1);
        float cr, e1, e2;
        if (STATS) acc.clusters++;
        h0 = cluster_edge_test<STATS>(q, p, d10, d01, l, ox, oy, float(a), I, J, id, acc, cr, e1, e2);
        if (h0) v0 = make_float4(cr, e1, e2, __uint_as_float(k << 1));
        float2 pu = make_float2(p.x - d11.x, p.y - d11.y);
        float2 bu = make_float2(d01.x - d11.x, d01.y - d11.y), cu = make_float2(d10.x - d11.x, d10.y - d11.y);
        h1 = cluster_edge_test<STATS>(q, pu, bu, cu, l, ox + a, oy + a, -float(a), I, J, id | 1u, acc, cr, e1, e2);
        if (h1) v1 = make_float4(cr, e1, e2, __uint_as_float((k << 1) | 1u));
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        bool h = t ? h1 : h0;
        unsigned mk = __ballot_sync(kFull, h);
        if (h) ls.hits[(ls.hhead + uint32_t(ls.nh) + __popc(mk & lt)) & (kHitRing - 1)] = t ? v1 : v0;
        ls.nh += __popc(mk);
        __syncwarp();
        if (ls.nh >= 32) {
            weigh_clusters<STATS>(d, q, ls, 32, lane, acc);
            ls.hhead += 32;
            ls.nh -= 32;
            __syncwarp();
        }
    }
}

// All 32 lanes: filter the queued leaf blocks' 2 x 2-quad groups by box and
// slab (lane t: group t & 3 of blocks p + (t >> 2) and p + 8 + (t >> 2), sixteen
// blocks per pass, both records in flight), compact the survivors into the
// ring and test them 32 groups (256 triangles) at a time.
template <int BFMT, int TFMT, bool STATS, bool CLAMP, class Q>
__device__ __forceinline__ void process_leaves(const MapDesc &d, const Q &q, const uint32_t *lq, int nleaf,
                                               LeafState &ls, int lane, Acc &acc)
{
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t morton_mask = (1u << (2 * (d.L - kLeafLevel))) - 1u;
    for (int p = 0; p < nleaf; p += 16) {
        uint32_t g[2];
        uint4 rec[2];
        bool pass[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int blk = p + 8 * r + (lane >> 2);
            pass[r] = blk < nleaf;
            if (pass[r]) {
                g[r] = ((lq[blk] & morton_mask) << 2) | uint32_t(lane & 3);
                rec[r] = __ldg(d.groups + g[r]);
                if (STATS && (lane & 3) == 0) acc.leaves++;
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (pass[r]) {
                pass[r] = half_box_holds<CLAMP>(rec[r].x, rec[r].y, q) &&
                          slab_holds(rec[r].z, rec[r].w, q.mx, q.my, slab_slack<CLAMP>(q));
                if (slab_marked(rec[r].w)) g[r] |= kMarked;
            }
            const unsigned m = __ballot_sync(kFull, pass[r]);
            if (pass[r]) ls.groups[(ls.ghead + uint32_t(ls.ng) + __popc(m & lt)) & (kGroupRing - 1)] = g[r];
            ls.ng += __popc(m);
        }
        __syncwarp();
        while (ls.ng >= 32) {
            test_groups<BFMT, TFMT, STATS, CLAMP>(d, q, ls, 32, lane, acc);
            ls.ghead += 32;
            ls.ng -= 32;
            __syncwarp();
        }
    }
}

// Nodes of size sz (S per side) whose closed extent [a sz, (a+1) sz] meets
// [x - r, x + r]; clamped in float first so no int conversion can overflow.
// Empty (a0 > a1) when the interval misses the map.
__device__ __forceinline__ void node_range(float x, float r, float sz, int S, int &a0, int &a1)
{
    float f0 = fmaxf(ceilf((x - r) / sz) - 1.0f, 0.0f);
    float f1 = fminf(floorf((x + r) / sz), float(S - 1));
    if (!(f0 <= f1)) {
        a0 = 1;
        a1 = 0;
        return;
    }
    a0 = int(f0);
    a1 = int(f1);
}

template <class Q>
__device__ __forceinline__ int entry_level(const Q &q, int L)
{
    float r = fmaxf(q.rx, q.ry);
    int l = kLeafLevel;
    while (l < L && float(1u << l) < r) ++l;
    return l;
}

// The hierarchical descent from the nodes [a0, a1] x [c0, c1] of level e
// (at most 4 x 4 of them) into the lane's accumulator: the whole query when
// they are its entry nodes, one tile of it when a large footprint is divided
// among warps.  Node boxes nest (a parent's normal box and uv box contain its
// children's), so a leaf block is reached from any level above it exactly
// when every node test on its path passes: the hit set, and with the exact
// sum the result, does not depend on the level the descent starts from.
template <int BFMT, int TFMT, bool STATS, bool CLUSTER, bool CLAMP, class Q>
__device__ __forceinline__ void eval_range(const MapDesc &d, const ClusterDesc &cd, const Q &q, int e, int a0,
                                           int a1, int c0, int c1, int lane, uint32_t *smem, Acc &acc)
{
    uint32_t *stk = smem, *lq = smem + kStackCap;
    int top = 0, nleaf = 0;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t leaf0 = node_index(d.L, kLeafLevel, 0);  // from here on a node is a leaf block
    // With the cut, a slab above the leaf level says nothing: it holds the
    // texels' normals, but a descendant may be cut and its cluster lie outside.
    // Below an uncut leaf block only exact triangles follow.
    auto in_slab = [&](const Node<BFMT> &n, uint32_t k) {
        return (CLUSTER && k < leaf0) || node_slab_holds<BFMT, CLAMP>(n, q);
    };
    // node k, child of a parent that was not inside: meets the support?  (and is it inside?)
    auto in_footprint = [&](uint32_t k, bool &ins) {
        if (ins) return true;
        const int l = node_level(k, d.L);
        const uint32_t m = k - node_index(d.L, l, 0);
        return node_meets(q, l, compact1by1(m), compact1by1(m >> 1), ins);
    };
    uint32_t *rings = lq + kLeafQ;
    float4 *hits = reinterpret_cast<float4 *>(rings + kGroupRing + kTriRing);
    LeafState ls{rings, rings + kGroupRing, hits, reinterpret_cast<uint32_t *>(hits + kHitRing), 0u, 0u, 0u, 0u, 0, 0, 0, 0};
    // entry nodes: at most 4 x 4
    {
        int a = a0 + (lane & 3), c = c0 + (lane >> 2);
        bool valid = lane < 16 && a <= a1 && c <= c1;
        const uint32_t k = node_index(d.L, e, valid ? morton2(a, c) : 0u);
        const Node<BFMT> n = load_node<BFMT>(d, k);
        bool inside = false;
        bool pass = valid && node_meets(q, e, a, c, inside) && node_box_holds<BFMT, CLAMP>(n, q);
        bool cut = false;
        if (STATS) acc.nodes += valid ? 1u : 0u;
        if (CLUSTER && pass) {  // the cut of Sec. 4.2: e <= r_x r_y tau
            cut = __ldg(cd.ce + k) <= q.theta;
            if (STATS) acc.cchecks++;
        }
        if (pass && !cut) pass = in_slab(n, k);
        unsigned mp = __ballot_sync(kFull, pass && !cut);
        unsigned mc = __ballot_sync(kFull, cut);
        if (pass && !cut) (e == kLeafLevel ? lq : stk)[__popc(mp & lt)] = k | (inside ? kInside : 0u);
        if (CLUSTER && cut) ls.cuts[__popc(mc & lt)] = k;
        if (e == kLeafLevel)
            nleaf = __popc(mp);
        else
            top = __popc(mp);
        ls.nc = __popc(mc);
        __syncwarp();
    }
    bool overflow = false;
    while (true) {
        // leaf blocks are filtered sixteen to a pass (four lanes each, twice):
        // while the stack still holds nodes only whole passes run, and the rest
        // (fewer than 16) waits at the front of the queue for the next step
        const int nrun = top == 0 ? nleaf : (nleaf & ~15);
        process_leaves<BFMT, TFMT, STATS, CLAMP>(d, q, lq, nrun, ls, lane, acc);
        if (nrun > 0 && nrun < nleaf) {
            const int rest = nleaf - nrun;  // < 16 <= nrun: source and target do not overlap
            uint32_t v = lane < rest ? lq[nrun + lane] : 0u;
            if (lane < rest) lq[lane] = v;
            __syncwarp();
        }
        nleaf -= nrun;
        if (CLUSTER)
            while (ls.nc >= (top == 0 ? 1 : 32)) {  // full warps of cut nodes, the rest at the end
                const int cnt = min(ls.nc, 32);
                test_clusters<STATS>(d, cd, q, ls, cnt, lane, acc);
                ls.chead += uint32_t(cnt);
                ls.nc -= cnt;
                __syncwarp();
            }
        if (top == 0) break;
        // pop up to 8 kPer nodes; lane k tests child (k & 3) of popped nodes
        // (k >> 2) + 8 r, so kPer loads per lane are in flight
        constexpr int per = kPer<BFMT>;
        static_assert(8 * per <= kPop, "stack and queue capacities");
        int npop = min(top, 8 * per);
        top -= npop;
        bool pass[per], ins[per], cut[per];
        uint32_t ck[per];
        Node<BFMT> nd[per];
        float ev[per];
#pragma unroll
        for (int r = 0; r < per; ++r) {
            int slot = (lane >> 2) + 8 * r;
            uint32_t ent = slot < npop ? stk[top + slot] : 0u;
            ck[r] = (ent << 2) | uint32_t(lane & 3);  // shifts "inside" out
            ins[r] = (ent & kInside) != 0u;
            pass[r] = slot < npop;
            cut[r] = false;
            if (STATS && slot < npop) acc.nodes++;
        }
        // All loads are in flight before either is tested; the uv box,
        // the costly test, only for the few children that hold m (98 ms against
        // 105 ms with the uv box first, 1M flake queries).
#pragma unroll
        for (int r = 0; r < per; ++r)
            if (pass[r]) {
                nd[r] = load_node<BFMT>(d, ck[r]);
                if (CLUSTER) ev[r] = __ldg(cd.ce + ck[r]);
            }
#pragma unroll
        for (int r = 0; r < per; ++r) {
            pass[r] = pass[r] && node_box_holds<BFMT, CLAMP>(nd[r], q);
            if (CLUSTER) {
                pass[r] = pass[r] && in_footprint(ck[r], ins[r]);
                if (pass[r]) {  // the cut of Sec. 4.2: e <= r_x r_y tau
                    cut[r] = ev[r] <= q.theta;
                    if (STATS) acc.cchecks++;
                }
                if (pass[r] && !cut[r]) pass[r] = in_slab(nd[r], ck[r]);
            } else {
                pass[r] = pass[r] && in_slab(nd[r], ck[r]) && in_footprint(ck[r], ins[r]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < per; ++r) {
            const bool keep = pass[r] && !cut[r];
            bool to_leaf = keep && ck[r] >= leaf0;
            bool to_stack = keep && ck[r] < leaf0;
            unsigned ml = __ballot_sync(kFull, to_leaf);
            unsigned ms = __ballot_sync(kFull, to_stack);
            if (CLUSTER) {
                unsigned mc = __ballot_sync(kFull, cut[r]);
                if (cut[r]) ls.cuts[(ls.chead + uint32_t(ls.nc) + __popc(mc & lt)) & (kCutRing - 1)] = ck[r];
                ls.nc += __popc(mc);
            }
            if (to_leaf) lq[nleaf + __popc(ml & lt)] = ck[r];
            if (to_stack) {
                int pos = top + __popc(ms & lt);
                if (pos < kStackCap) stk[pos] = ck[r] | (ins[r] ? kInside : 0u);
            }
            nleaf += __popc(ml);
            top += __popc(ms);
            if (top > kStackCap) {
                top = kStackCap;
                overflow = true;
            }
        }
        __syncwarp();
    }
    if (ls.ng > 0) test_groups<BFMT, TFMT, STATS, CLAMP>(d, q, ls, ls.ng, lane, acc);  // ng < 32 here
    if (ls.nt > 0) test_tris<BFMT, TFMT, STATS, CLAMP>(d, q, ls, ls.nt, lane, acc);    // nt < 32 here
    if (CLUSTER && ls.nh > 0) weigh_clusters<STATS>(d, q, ls, ls.nh, lane, acc);  // nh < 32 here
    if (overflow) acc.flags |= PNDF_QF_OVERFLOW;
}

// Warp total of the lanes' accumulators: the fixed-point sum (exact), the
// flags and, with STATS, the counters (all lanes hold the result).
template <bool STATS>
__device__ __forceinline__ void warp_total(Acc &acc, unsigned long long &lo, unsigned long long &hi, uint32_t &fl)
{
    lo = s_sum_lo[threadIdx.x];
    hi = s_sum_hi[threadIdx.x];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long lo_o = __shfl_xor_sync(kFull, lo, off);
        const unsigned long long hi_o = __shfl_xor_sync(kFull, hi, off);
        lo += lo_o;
        const unsigned long long h0 = hi;
        hi += hi_o + (lo < lo_o ? 1ull : 0ull);
        if (hi < h0) acc.flags |= kHuge;
    }
    fl = __reduce_or_sync(kFull, acc.flags);
    if (STATS) {
        acc.hits = __reduce_add_sync(kFull, acc.hits);
        acc.hash = __reduce_add_sync(kFull, acc.hash);
        acc.tests = __reduce_add_sync(kFull, acc.tests);
        acc.fp64 = __reduce_add_sync(kFull, acc.fp64);
        acc.degen = __reduce_add_sync(kFull, acc.degen);
        acc.nodes = __reduce_add_sync(kFull, acc.nodes);
        acc.leaves = __reduce_add_sync(kFull, acc.leaves);
        acc.quads = __reduce_add_sync(kFull, acc.quads);
        acc.cchecks = __reduce_add_sync(kFull, acc.cchecks);
        acc.clusters = __reduce_add_sync(kFull, acc.clusters);
    }
}

// KERN: the footprint kernel (pndf_kernel), a compile-time constant so the
// query's kernel fields and branches fold away (each kernel is its own
// instantiation).
template <int BFMT, int TFMT, bool STATS, bool FLAT, bool CLUSTER, int KERN>
__device__ void eval_one(const MapDesc &d, const ClusterDesc &cd, float tau, float jac_eps, const pndf_query &rec,
                         int lane, uint32_t *wsm, Query<KERN> &q, float &D_out, uint32_t &flags_out,
                         pndf_query_stats *st_out)
{
    constexpr bool CLAMP = KERN == kKernGaussClamp;
    Acc acc = {};
    acc_zero();
    {
        Query<KERN> r = make_query<KERN>(rec, jac_eps);
        if (CLUSTER) r.theta *= tau;  // r_x r_y tau with the support's half-widths
        __syncwarp();
        if (lane == 0) q = r;
        __syncwarp();
    }
    if (!q.valid) {
        if (lane == 0) {
            D_out = __int_as_float(0x7fc00000);
            flags_out = PNDF_QF_INVALID;
            record_status(d.status, &g_status_eval, PNDF_QF_INVALID);
            if (STATS) *st_out = pndf_query_stats{0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        }
        return;
    }
    const int L = d.L;
    if (FLAT) {
        // every leaf block meeting the 4-sigma box, no pruning
        const int S = 1 << (L - kLeafLevel);
        const float sz = float(kLeafQuads);
        int a0, a1, c0, c1;
        node_range(q.x, q.rx, sz, S, a0, a1);
        node_range(q.y, q.ry, sz, S, c0, c1);
        for (int c = c0; c <= c1; ++c)
            for (int a = a0; a <= a1; ++a)
                test_leaf<STATS>(d, q, a, c, leaf_texel<TFMT>(d, a, c, lane), lane, acc);
    } else {
        const int e = entry_level(q, L);
        const int S = 1 << (L - e);
        const float sz = float(1u << e);
        int a0, a1, c0, c1;
        node_range(q.x, q.rx, sz, S, a0, a1);
        node_range(q.y, q.ry, sz, S, c0, c1);
        eval_range<BFMT, TFMT, STATS, CLUSTER, CLAMP>(d, cd, q, e, a0, a1, c0, c1, lane, wsm, acc);
    }
    unsigned long long lo, hi;
    uint32_t fl;
    warp_total<STATS>(acc, lo, hi, fl);
    if (lane == 0) {
        D_out = acc_value(lo, hi, fl);
        fl &= ~kHuge;
        flags_out = fl;
        if (fl & PNDF_QF_OVERFLOW) record_status(d.status, &g_status_eval, PNDF_QF_OVERFLOW);
        if (STATS)
            *st_out = pndf_query_stats{acc.nodes, acc.leaves, acc.tests, acc.hits,    acc.hash,
                                       acc.fp64,  acc.degen,  acc.quads, acc.cchecks, acc.clusters};
    }
}

__constant__ ClusterDesc kNoClusters;  // never read: the variants without the cut

// ---- large footprints divided among warps ----
//
// One warp per query leaves a batch waiting on its largest footprints: a
// sigma = 1024 query on a 16384^2 map is about 100 ms of one warp, longer
// than the rest of a few-thousand-query batch together.  Before the
// traversal, split_work sums a work estimate over the batch (the area of each
// support's bounding box) and split_plan divides every query whose estimate
// is more than twice the target w_t = max(W / (4 x resident warps), 2.6e5)
// (2.6e5: the box of a sigma = 64 footprint) into tiles of at most 4 x 4
// nodes of one level, the deepest level (>= 4, at most 256 tiles) whose tile
// count reaches its estimate / w_t.  The traversal hands out the tiles first
// (largest queries first), then the undivided queries; the last warp to
// finish a query's tiles writes its result.  The sum is exact, so the
// result is the same bits whichever way the query was divided.
constexpr int kSplitMinLevel = 4;
constexpr uint32_t kSplitMaxTiles = 256;
constexpr float kSplitMinWork = 2.6e5f;
constexpr int kSplitPerWarp = 4;

struct SplitEntry {
    uint32_t qi, tiles;        // the query (caller index) and its tile count
    unsigned long long base;   // index of its first tile among all tiles
    int32_t level, pad;        // node level of the tiles
    unsigned long long lo, hi; // fixed-point sum of the finished tiles
    uint32_t done, flags;      // tiles finished; OR of their flags
    pndf_query_stats st;       // summed counters (stats launches)
};

struct SplitPlan {
    SplitEntry *entries;       // null: no division
    uint8_t *marker;           // per query (caller index): 1 = divided into tiles
    unsigned long long *ctr;   // (entries << 40) | tiles reserved
    double *work;              // the batch's summed estimate
    float *wt;                 // the target w_t (served steps: written by the plan for the step kernel)
    uint32_t cap;              // entries capacity
    int resident_warps;
    bool one_cta;              // planned by split_small, which also clears the counters
};

template <class Q>
__device__ __forceinline__ float split_estimate(const Q &q)
{
    return q.valid ? 64.f + 4.f * q.rx * q.ry : 64.f;
}

template <int KERN>
__global__ void split_work(const pndf_query *__restrict__ qs, int64_t nq, float jac_eps, double *__restrict__ work)
{
    __shared__ double red[256];
    double acc = 0.0;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < nq; k += int64_t(gridDim.x) * blockDim.x)
        acc += double(split_estimate(make_query<KERN>(qs[k], jac_eps)));
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (int(threadIdx.x) < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(work, red[0]);
}

// Tiles of level l over the support's bounding box: ceil(nx / 4) ceil(ny / 4).
template <class Q>
__device__ __forceinline__ uint32_t split_tiles(const Q &q, int L, int l, int &a0, int &a1, int &c0, int &c1)
{
    const int S = 1 << (L - l);
    const float sz = float(1u << l);
    node_range(q.x, q.rx, sz, S, a0, a1);
    node_range(q.y, q.ry, sz, S, c0, c1);
    if (a0 > a1 || c0 > c1) return 0u;
    return uint32_t((a1 - a0) / 4 + 1) * uint32_t((c1 - c0) / 4 + 1);
}

__device__ __forceinline__ float split_target(const SplitPlan &p)
{
    return fmaxf(float(*p.work / (double(kSplitPerWarp) * p.resident_warps)), kSplitMinWork);
}

// Whether query q is divided at target wt, and into which tiles: the deepest
// level (>= kSplitMinLevel) whose tile count stays <= kSplitMaxTiles, or the
// first going down whose count reaches estimate / wt; at least two tiles.
template <class Q>
__device__ __forceinline__ bool split_choice(const Q &q, int L, float wt, int &level, uint32_t &tiles)
{
    const float w = split_estimate(q);
    if (!q.valid || !(w > 2.f * wt)) return false;
    const float target = w / wt;
    int best = -1, a0, a1, c0, c1;
    uint32_t bt = 0;
    for (int l = entry_level(q, L) - 1; l >= kSplitMinLevel; --l) {
        const uint32_t t = split_tiles(q, L, l, a0, a1, c0, c1);
        if (t > kSplitMaxTiles) break;
        best = l;
        bt = t;
        if (float(t) >= target) break;
    }
    level = best;
    tiles = bt;
    return best >= 0 && bt >= 2;
}

// Reserve an entry and its tiles; false if the entries are full (never
// expected: the division bounds them by 2 x the resident warps).
__device__ __forceinline__ bool split_reserve(const SplitPlan &p, uint32_t qi, int seg, int level, uint32_t tiles)
{
    const unsigned long long old = atomicAdd(p.ctr, (1ull << 40) | tiles);
    const unsigned long long idx = old >> 40;
    if (idx >= p.cap) return false;
    SplitEntry &E = p.entries[idx];
    E.qi = qi;
    E.tiles = tiles;
    E.base = old & ((1ull << 40) - 1ull);
    E.level = level;
    E.pad = seg;
    E.lo = E.hi = 0ull;
    E.done = E.flags = 0u;
    E.st = pndf_query_stats{0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    return true;
}

template <int KERN>
__global__ void split_plan(MapDesc d, const pndf_query *__restrict__ qs, int64_t nq, float jac_eps, SplitPlan p)
{
    const float wt = split_target(p);
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < nq; k += int64_t(gridDim.x) * blockDim.x) {
        const auto q = make_query<KERN>(qs[k], jac_eps);
        int level;
        uint32_t tiles;
        p.marker[k] = split_choice(q, d.L, wt, level, tiles) && split_reserve(p, uint32_t(k), 0, level, tiles);
    }
}

// split_work and split_plan of a small batch in one CTA, which also sets the
// work cursor and the counters to zero: one launch in place of a memset and two.
constexpr int64_t kSplitSmall = 8192;

template <int KERN>
__global__ void __launch_bounds__(1024) split_small(MapDesc d, const pndf_query *__restrict__ qs, int nq, float jac_eps,
                                                    SplitPlan p, unsigned long long *__restrict__ cursor)
{
    __shared__ double red[32];
    __shared__ double total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double acc = 0.0;
    for (int k = threadIdx.x; k < nq; k += 1024) acc += double(split_estimate(make_query<KERN>(qs[k], jac_eps)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (warp == 0) {
        acc = red[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
        if (lane == 0) {
            total = acc;
            *p.ctr = 0ull;
            *cursor = 0ull;
        }
    }
    __syncthreads();
    p.work = &total;
    const float wt = split_target(p);
    for (int k = threadIdx.x; k < nq; k += 1024) {
        const auto q = make_query<KERN>(qs[k], jac_eps);
        int level;
        uint32_t tiles;
        p.marker[k] = split_choice(q, d.L, wt, level, tiles) && split_reserve(p, uint32_t(k), 0, level, tiles);
    }
}

// Work index k < ntiles: the entry of the divided query it belongs to (the
// last entry whose first tile is <= k) and the tile's node range.
__device__ __forceinline__ int tile_entry(const SplitPlan &p, int n_entries, unsigned long long k)
{
    int lo = 0, hi = n_entries - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&p.entries[mid].base) <= k)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

template <class Q>
__device__ __forceinline__ void tile_range(const Q &q, int L, int l, uint32_t j, int &a0, int &a1, int &c0, int &c1)
{
    int b0, b1, d0, d1;
    split_tiles(q, L, l, b0, b1, d0, d1);
    const int ntx = (b1 - b0) / 4 + 1;
    a0 = b0 + 4 * int(j % uint32_t(ntx));
    c0 = d0 + 4 * int(j / uint32_t(ntx));
    a1 = min(b1, a0 + 3);
    c1 = min(d1, c0 + 3);
}

// Lane 0: fold a tile's warp total into its query's entry; the warp that
// folds in the last tile writes D, the flags and the counters.
template <bool STATS>
__device__ __forceinline__ void tile_finish(const MapDesc &d, SplitEntry &E, const Acc &acc, unsigned long long lo,
                                            unsigned long long hi, uint32_t fl, float *D, uint32_t *flags,
                                            pndf_query_stats *stats)
{
    const unsigned long long old = atomicAdd(&E.lo, lo);
    const unsigned long long add_hi = hi + (old + lo < old ? 1ull : 0ull);
    const unsigned long long old_hi = atomicAdd(&E.hi, add_hi);
    if (old_hi + add_hi < old_hi) fl |= kHuge;
    if (fl) atomicOr(&E.flags, fl);
    if (STATS) {
        atomicAdd(&E.st.nodes, acc.nodes);
        atomicAdd(&E.st.leaf_blocks, acc.leaves);
        atomicAdd(&E.st.tri_tests, acc.tests);
        atomicAdd(&E.st.hits, acc.hits);
        atomicAdd(&E.st.hit_hash, acc.hash);
        atomicAdd(&E.st.fp64_tris, acc.fp64);
        atomicAdd(&E.st.degenerate, acc.degen);
        atomicAdd(&E.st.quads, acc.quads);
    }
    __threadfence();
    if (atomicAdd(&E.done, 1u) == __ldg(&E.tiles) - 1u) {
        __threadfence();
        const uint32_t qi = __ldg(&E.qi);
        const uint32_t f = __ldcg(&E.flags);
        D[qi] = acc_value(__ldcg(&E.lo), __ldcg(&E.hi), f);
        if (flags) flags[qi] = f & ~kHuge;
        if (f & PNDF_QF_OVERFLOW) record_status(d.status, &g_status_eval, PNDF_QF_OVERFLOW);
        if (STATS)
            stats[qi] = pndf_query_stats{__ldcg(&E.st.nodes),      __ldcg(&E.st.leaf_blocks), __ldcg(&E.st.tri_tests),
                                         __ldcg(&E.st.hits),       __ldcg(&E.st.hit_hash),    __ldcg(&E.st.fp64_tris),
                                         __ldcg(&E.st.degenerate), __ldcg(&E.st.quads),       0u,
                                         0u};
    }
}

template <int BFMT, int TFMT, bool STATS, bool FLAT, bool CLUSTER, int KERN>
__global__ void __launch_bounds__(256, kTraverseCtas)
    traverse_kernel(MapDesc d, ClusterDesc cd, float tau, float jac_eps, const pndf_query *__restrict__ qs,
                    const uint32_t *__restrict__ order, int64_t nq, float *__restrict__ D,
                    uint32_t *__restrict__ flags, pndf_query_stats *__restrict__ stats,
                    unsigned long long *__restrict__ cursor, SplitPlan sp)
{
    extern __shared__ uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *wsm = smem + warp * kWarpSmemWords<CLUSTER>;
    // the divided queries' tiles take the first s_ntiles work indices
    __shared__ unsigned long long s_ntiles;
    __shared__ int s_entries;
    __shared__ uint32_t s_dest[8][2];  // per warp: query, entry (-1: whole query)
    __shared__ Query<KERN> s_query[8];
    if (threadIdx.x == 0) {
        int n = 0;
        unsigned long long t = 0ull;
        if (!FLAT && !CLUSTER && sp.entries) {
            n = int(min(__ldcg(sp.ctr) >> 40, (unsigned long long)sp.cap));
            if (n > 0) t = __ldcg(&sp.entries[n - 1].base) + __ldcg(&sp.entries[n - 1].tiles);
        }
        s_entries = n;
        s_ntiles = t;
    }
    __syncthreads();
    while (true) {
        unsigned long long k = 0;
        if (lane == 0) k = atomicAdd(cursor, 1ull);
        k = __shfl_sync(kFull, k, 0);
        if (FLAT || CLUSTER) {
            if (k >= (unsigned long long)nq) break;
            const int64_t qi = order ? int64_t(order[k]) : int64_t(k);
            float Dv;
            uint32_t fv;
            eval_one<BFMT, TFMT, STATS, FLAT, CLUSTER, KERN>(d, cd, tau, jac_eps, qs[qi], lane, wsm, s_query[warp], Dv, fv,
                                                             stats ? stats + qi : nullptr);
            if (lane == 0) {
                D[qi] = Dv;
                if (flags) flags[qi] = fv;
            }
            continue;
        }
        // a tile of a divided query, or a whole query: one descent either way
        constexpr bool CLAMP = KERN == kKernGaussClamp;
        int ei = -1;  // the divided query's entry, or -1 for a whole query
        uint32_t qi;
        Query<KERN> q;
        int e, a0, a1, c0, c1;
        if (k < s_ntiles) {
            ei = tile_entry(sp, s_entries, k);
            const SplitEntry &E = sp.entries[ei];
            qi = __ldg(&E.qi);
            q = make_query<KERN>(qs[qi], jac_eps);
            e = __ldg(&E.level);
            tile_range(q, d.L, e, uint32_t(k - __ldg(&E.base)), a0, a1, c0, c1);
        } else {
            k -= s_ntiles;
            if (k >= (unsigned long long)nq) break;
            qi = order ? order[k] : uint32_t(k);
            if (s_entries > 0 && sp.marker[qi]) continue;  // evaluated as tiles
            q = make_query<KERN>(qs[qi], jac_eps);
            if (!q.valid) {
                if (lane == 0) {
                    D[qi] = __int_as_float(0x7fc00000);
                    if (flags) flags[qi] = PNDF_QF_INVALID;
                    record_status(d.status, &g_status_eval, PNDF_QF_INVALID);
                    if (STATS) stats[qi] = pndf_query_stats{0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
                }
                continue;
            }
            e = entry_level(q, d.L);
            const float sz = float(1u << e);
            node_range(q.x, q.rx, sz, 1 << (d.L - e), a0, a1);
            node_range(q.y, q.ry, sz, 1 << (d.L - e), c0, c1);
        }
        // where the result goes waits in shared memory during the descent
        __syncwarp();
        if (lane == 0) {
            s_dest[warp][0] = qi;
            s_dest[warp][1] = uint32_t(ei);
            s_query[warp] = q;
        }
        __syncwarp();
        Acc acc = {};
        acc_zero();
        eval_range<BFMT, TFMT, STATS, false, CLAMP>(d, cd, s_query[warp], e, a0, a1, c0, c1, lane, wsm, acc);
        unsigned long long lo, hi;
        uint32_t fl;
        warp_total<STATS>(acc, lo, hi, fl);
        if (lane == 0) {
            qi = s_dest[warp][0];
            ei = int(s_dest[warp][1]);
            if (ei >= 0) {
                tile_finish<STATS>(d, sp.entries[ei], acc, lo, hi, fl, D, flags, stats);
            } else {
                D[qi] = acc_value(lo, hi, fl);
                if (flags) flags[qi] = fl & ~kHuge;
                if (fl & PNDF_QF_OVERFLOW) record_status(d.status, &g_status_eval, PNDF_QF_OVERFLOW);
                if (STATS)
                    stats[qi] = pndf_query_stats{acc.nodes, acc.leaves, acc.tests, acc.hits,    acc.hash,
                                                 acc.fp64,  acc.degen,  acc.quads, acc.cchecks, acc.clusters};
            }
        }
    }
}

// ---- query keying and counting sort ----

// Sort key: entry level (largest footprints first, 4 bits), then a sub-key of
// `sub` bits (6..14, more for larger batches): the footprint centre's tile
// (mode 1), the query normal's bin over [-0.4, 0.4]^2 (mode 2), or both, tile
// major (mode 3) or normal-bin major (mode 4).  Grouping queries that share a
// region and a normal makes the warps in flight visit the same nodes and leaf
// blocks, so they share L1/L2 lines.  The order never changes a result.
__device__ __forceinline__ uint32_t sort_key(const MapDesc &d, const pndf_query &r, int mode, int sub)
{
    const auto q = make_query<PNDF_KERNEL_GAUSS>(r);
    if (!q.valid) return 0u;
    int e = entry_level(q, d.L);
    int tb, mb;  // bits per axis for the tile and the normal bin
    if (mode == 1) {
        tb = sub >> 1;
        mb = 0;
    } else if (mode == 2) {
        tb = 0;
        mb = sub >> 1;
    } else {
        tb = (sub + 2) >> 2;
        mb = (sub >> 1) - tb;
    }
    float ts = float(1 << tb) / float(d.n), ms = float(1 << mb) / 0.8f;
    uint32_t tx = uint32_t(fminf(fmaxf(r.x * ts, 0.f), float((1 << tb) - 1)));
    uint32_t ty = uint32_t(fminf(fmaxf(r.y * ts, 0.f), float((1 << tb) - 1)));
    uint32_t mx = uint32_t(fminf(fmaxf((r.ms + 0.4f) * ms, 0.f), float((1 << mb) - 1)));
    uint32_t my = uint32_t(fminf(fmaxf((r.mt + 0.4f) * ms, 0.f), float((1 << mb) - 1)));
    uint32_t t = morton2(tx, ty), m = morton2(mx, my);
    uint32_t k = mode == 4 ? (m << (2 * tb)) | t : (t << (2 * mb)) | m;
    return (uint32_t(15 - e) << sub) | k;
}

// Sub-key bits for a batch of nq queries: about 16 queries per bin on average.
inline int sort_sub_bits(int64_t nq)
{
    int b = 6;
    while (b < kMaxSubBits && (int64_t(1) << (b + 4 + 2)) * 16 <= nq) b += 2;
    return b;
}

__global__ void key_hist(MapDesc d, const pndf_query *__restrict__ qs, int64_t nq, int mode, int sub,
                         uint32_t *__restrict__ keys, uint32_t *__restrict__ hist)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < nq; k += int64_t(gridDim.x) * blockDim.x) {
        uint32_t key = sort_key(d, qs[k], mode, sub);
        keys[k] = key;
        atomicAdd(&hist[key], 1u);
    }
}

// One CTA of 1024 threads: exclusive scan of nbins (a multiple of 4096) counts
// in place, 4096 bins per round, four consecutive bins per thread.
__global__ void __launch_bounds__(1024) key_scan(uint32_t *__restrict__ hist, int nbins)
{
    __shared__ uint32_t warp_tot[32];
    __shared__ uint32_t carry_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    for (int base = 0; base < nbins; base += 4096) {
        uint4 v = reinterpret_cast<uint4 *>(hist + base)[threadIdx.x];
        uint32_t sum = v.x + v.y + v.z + v.w;
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            uint32_t t = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += t;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            uint32_t w = warp_tot[lane], wi = w;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                uint32_t t = __shfl_up_sync(kFull, wi, off);
                if (lane >= off) wi += t;
            }
            warp_tot[lane] = wi - w;  // exclusive prefix of warp totals
        }
        __syncthreads();
        uint32_t run = carry_s + warp_tot[warp] + incl - sum;
        uint4 o;
        o.x = run;
        o.y = o.x + v.x;
        o.z = o.y + v.y;
        o.w = o.z + v.z;
        reinterpret_cast<uint4 *>(hist + base)[threadIdx.x] = o;
        __syncthreads();
        if (threadIdx.x == 1023) carry_s = run + sum;
        __syncthreads();
    }
}

__global__ void key_place(const uint32_t *__restrict__ keys, int64_t nq, uint32_t *__restrict__ offsets,
                          uint32_t *__restrict__ order)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < nq; k += int64_t(gridDim.x) * blockDim.x) {
        uint32_t pos = atomicAdd(&offsets[keys[k]], 1u);
        order[pos] = uint32_t(k);
    }
}

// Key, histogram, scan and placement: order receives a permutation of 0..nq-1.
// scratch: hist (zeroed by the caller, 1 << (4 + sub) bins) and keys (nq).
cudaError_t sort_launch(const MapDesc &d, const pndf_query *q, int64_t nq, int mode, uint32_t *hist, uint32_t *keys,
                        uint32_t *order, cudaStream_t s)
{
    const int sub = sort_sub_bits(nq);
    int nbins = 1 << (4 + sub);
    if (nbins < 4096) nbins = 4096;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (nq + 255) / 256;
    if (blocks > int64_t(sms) * 8) blocks = int64_t(sms) * 8;
    key_hist<<<unsigned(blocks), 256, 0, s>>>(d, q, nq, mode, sub, keys, hist);
    key_scan<<<1, 1024, 0, s>>>(hist, nbins);
    key_place<<<unsigned(blocks), 256, 0, s>>>(keys, nq, hist, order);
    count_launches(3);
    return cudaGetLastError();
}

// Histogram bytes a batch of nq queries needs (a multiple of 16 KiB).
inline size_t sort_hist_bytes(int64_t nq)
{
    size_t bins = size_t(1) << (4 + sort_sub_bits(nq));
    if (bins < 4096) bins = 4096;
    return bins * sizeof(uint32_t);
}

template <int BFMT, int TFMT, bool STATS, bool FLAT, bool CLUSTER, int KERN>
cudaError_t launch_traverse(const MapDesc &d, const ClusterDesc &cd, float tau, float jac_eps, const pndf_query *q,
                            const uint32_t *order, int64_t nq, float *D, uint32_t *flags, pndf_query_stats *stats,
                            unsigned long long *cursor, int warps, int ctas_per_sm, SplitPlan sp, cudaStream_t s)
{
    if (FLAT || CLUSTER) sp.entries = nullptr;  // whole queries only (the cut depends on the entry level)
    auto kern = traverse_kernel<BFMT, TFMT, STATS, FLAT, CLUSTER, KERN>;
    int threads = warps * 32;
    size_t smem = size_t(warps) * kWarpSmemWords<CLUSTER> * sizeof(uint32_t);
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // with its static arrays the kernel passes the 48 KB a launch gets by default
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) occ = 1;
    if (ctas_per_sm > 0 && ctas_per_sm < occ) occ = ctas_per_sm;
    int64_t want = (nq + warps - 1) / warps;
    int64_t grid = int64_t(sms) * occ;
    if (sp.entries) {
        // the plan: the batch's work, then the division of its large footprints
        sp.resident_warps = int(grid) * warps;
        int64_t blocks = (nq + 255) / 256;
        if (blocks > int64_t(sms) * 8) blocks = int64_t(sms) * 8;
        if (sp.one_cta) {
            split_small<KERN><<<1, 1024, 0, s>>>(d, q, int(nq), jac_eps, sp, cursor);
            count_launches(1);
        } else {
            split_work<KERN><<<unsigned(blocks), 256, 0, s>>>(q, nq, jac_eps, sp.work);
            split_plan<KERN><<<unsigned(blocks), 256, 0, s>>>(d, q, nq, jac_eps, sp);
            count_launches(2);
        }
    } else if (grid > want) {
        grid = want;
    }
    if (grid < 1) grid = 1;
    kern<<<unsigned(grid), threads, smem, s>>>(d, cd, tau, jac_eps, q, order, nq, D, flags, stats, cursor, sp);
    count_launches(1);
    return cudaGetLastError();
}

template <int BFMT, int TFMT, int KERN>
cudaError_t dispatch_kernel(const MapDesc &d, const ClusterDesc &cd, const pndf_query *q, const uint32_t *order,
                            int64_t nq, float *D, uint32_t *flags, pndf_query_stats *stats,
                            unsigned long long *cursor, const pndf_eval_config &cfg, const SplitPlan &sp,
                            cudaStream_t s)
{
    const int warps = cfg.warps_per_cta > 0 ? cfg.warps_per_cta : 8;
    const int cps = cfg.ctas_per_sm;
    const float tau = cfg.tau;
    if (cfg.mode == PNDF_MODE_FLAT)
        return stats ? launch_traverse<BFMT, TFMT, true, true, false, KERN>(d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                             cursor, warps, cps, sp, s)
                     : launch_traverse<BFMT, TFMT, false, true, false, KERN>(d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                              cursor, warps, cps, sp, s);
    if (tau > 0.f)
        return stats ? launch_traverse<BFMT, TFMT, true, false, true, KERN>(d, cd, tau, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                             cursor, warps, cps, sp, s)
                     : launch_traverse<BFMT, TFMT, false, false, true, KERN>(d, cd, tau, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                              cursor, warps, cps, sp, s);
    return stats ? launch_traverse<BFMT, TFMT, true, false, false, KERN>(d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                          cursor, warps, cps, sp, s)
                 : launch_traverse<BFMT, TFMT, false, false, false, KERN>(d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats,
                                                                           cursor, warps, cps, sp, s);
}

template <int BFMT, int TFMT>
cudaError_t dispatch_stats(const MapDesc &d, const ClusterDesc &cd, const pndf_query *q, const uint32_t *order,
                           int64_t nq, float *D, uint32_t *flags, pndf_query_stats *stats,
                           unsigned long long *cursor, const pndf_eval_config &cfg, const SplitPlan &sp,
                           cudaStream_t s)
{
    if (cfg.jac_eps > 0.f)  // Gaussian, hierarchy mode, no cluster cut (checked by the caller)
        return stats ? launch_traverse<BFMT, TFMT, true, false, false, kKernGaussClamp>(
                           d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats, cursor,
                           cfg.warps_per_cta > 0 ? cfg.warps_per_cta : 8, cfg.ctas_per_sm, sp, s)
                     : launch_traverse<BFMT, TFMT, false, false, false, kKernGaussClamp>(
                           d, cd, 0.f, cfg.jac_eps, q, order, nq, D, flags, stats, cursor,
                           cfg.warps_per_cta > 0 ? cfg.warps_per_cta : 8, cfg.ctas_per_sm, sp, s);
    if (cfg.kernel == PNDF_KERNEL_DISK)
        return dispatch_kernel<BFMT, TFMT, PNDF_KERNEL_DISK>(d, cd, q, order, nq, D, flags, stats, cursor, cfg, sp, s);
    if (cfg.kernel == PNDF_KERNEL_BOX)
        return dispatch_kernel<BFMT, TFMT, PNDF_KERNEL_BOX>(d, cd, q, order, nq, D, flags, stats, cursor, cfg, sp, s);
    return dispatch_kernel<BFMT, TFMT, PNDF_KERNEL_GAUSS>(d, cd, q, order, nq, D, flags, stats, cursor, cfg, sp, s);
}

}  // namespace

pndf_status launch_eval(const pndf_hierarchy *h, const pndf_query *q, int64_t nq, float *D, uint32_t *flags,
                        pndf_query_stats *stats, const pndf_eval_config &cfg, cudaStream_t s)
{
    if (nq == 0) return PNDF_OK;
    const MapDesc &d = h->d;
    const bool split = cfg.mode == PNDF_MODE_HIERARCHY && !(cfg.tau > 0.f) && cfg.split == 0;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // The default order is left out for a batch of up to four queries per resident
    // warp whose large footprints are divided: it gains nothing there (no warp holds
    // more than a few queries, and neighbours do not stay in flight together; 4,096
    // footprints on 16384^2 and 20,011 on 8192^2: 5.10 and 5.09 ms in arrival order,
    // 5.12 and 5.14 ms sorted; 131,072: 24.6 and 19.8 ms), and the sort's four
    // launches would be most of a small call.  Another order was asked for: it is made.
    const int warps = cfg.warps_per_cta > 0 ? cfg.warps_per_cta : 8;
    const int resident = cfg.ctas_per_sm > 0 && warps * int64_t(cfg.ctas_per_sm) < kTraverseWarps
                             ? warps * cfg.ctas_per_sm : kTraverseWarps;
    const bool sort = cfg.sort != PNDF_SORT_NONE &&
                      !(cfg.sort == PNDF_SORT_DEFAULT && split && nq <= int64_t(4) * resident * sms);
    const uint32_t cap = uint32_t(2 * 64 * (sms > 0 ? sms : 1) + 64);  // >= 2 x resident warps
    // scratch: cursor, split counter and work sum (padded to 256), key
    // histogram, keys, order, split markers and entries
    const size_t hist_b = sort_hist_bytes(nq);
    size_t off_hist = 256, off_keys = off_hist + hist_b;
    size_t off_order = off_keys + ((size_t(nq) * sizeof(uint32_t) + 255) & ~size_t(255));
    size_t bytes = sort ? off_order + ((size_t(nq) * sizeof(uint32_t) + 255) & ~size_t(255)) : 256;
    const size_t off_marker = bytes, off_entries = off_marker + ((size_t(nq) + 255) & ~size_t(255));
    if (split) bytes = off_entries + size_t(cap) * sizeof(SplitEntry);
    void *scratch = nullptr;
    if (cudaMallocAsync(&scratch, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return PNDF_ERR_OOM;
    }
    char *base = static_cast<char *>(scratch);
    auto *cursor = reinterpret_cast<unsigned long long *>(base);
    SplitPlan sp{};
    if (split) {
        sp.entries = reinterpret_cast<SplitEntry *>(base + off_entries);
        sp.marker = reinterpret_cast<uint8_t *>(base + off_marker);
        sp.ctr = reinterpret_cast<unsigned long long *>(base + 8);
        sp.work = reinterpret_cast<double *>(base + 16);
        sp.cap = cap;
        sp.one_cta = !sort && nq <= kSplitSmall;
    }
    uint32_t *order = nullptr;
    cudaError_t e = sp.one_cta ? cudaSuccess : cudaMemsetAsync(base, 0, sort ? off_keys : 256, s);
    if (e == cudaSuccess && sort) {
        order = reinterpret_cast<uint32_t *>(base + off_order);
        e = sort_launch(d, q, nq, cfg.sort, reinterpret_cast<uint32_t *>(base + off_hist),
                        reinterpret_cast<uint32_t *>(base + off_keys), order, s);
    }
    if (e == cudaSuccess && cfg.ev_begin) e = cudaEventRecord(static_cast<cudaEvent_t>(cfg.ev_begin), s);
    if (e == cudaSuccess) {
        if (d.bounds_fmt == PNDF_BOUNDS_F32)
            e = d.texel_fmt == PNDF_TEXEL_F32X2
                    ? dispatch_stats<PNDF_BOUNDS_F32, PNDF_TEXEL_F32X2>(d, h->c, q, order, nq, D, flags, stats, cursor, cfg, sp, s)
                    : dispatch_stats<PNDF_BOUNDS_F32, PNDF_TEXEL_F16X2>(d, h->c, q, order, nq, D, flags, stats, cursor, cfg, sp, s);
        else
            e = d.texel_fmt == PNDF_TEXEL_F32X2
                    ? dispatch_stats<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F32X2>(d, h->c, q, order, nq, D, flags, stats, cursor,
                                                                             cfg, sp, s)
                    : dispatch_stats<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F16X2>(d, h->c, q, order, nq, D, flags, stats, cursor,
                                                                             cfg, sp, s);
    }
    if (e == cudaSuccess && cfg.ev_end) e = cudaEventRecord(static_cast<cudaEvent_t>(cfg.ev_end), s);
    cudaError_t ef = cudaFreeAsync(scratch, s);
    if (e != cudaSuccess || ef != cudaSuccess) return PNDF_ERR_CUDA;
    return PNDF_OK;
}

// ---------------------------------------------------------------------------
// Sorting a batch on its own (pndf_sort_queries).
// ---------------------------------------------------------------------------

pndf_status launch_sort(const pndf_hierarchy *h, const pndf_query *q, int64_t nq, uint32_t *order, cudaStream_t s)
{
    if (nq == 0) return PNDF_OK;
    size_t off_keys = sort_hist_bytes(nq);
    size_t bytes = off_keys + ((size_t(nq) * sizeof(uint32_t) + 255) & ~size_t(255));
    void *scratch = nullptr;
    if (cudaMallocAsync(&scratch, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return PNDF_ERR_OOM;
    }
    auto *hist = static_cast<uint32_t *>(scratch);
    auto *keys = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + off_keys);
    cudaError_t e = cudaMemsetAsync(hist, 0, off_keys, s);
    if (e == cudaSuccess) e = sort_launch(h->d, q, nq, PNDF_SORT_DEFAULT, hist, keys, order, s);
    cudaError_t ef = cudaFreeAsync(scratch, s);
    return (e == cudaSuccess && ef == cudaSuccess) ? PNDF_OK : PNDF_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// Serving step kernel: one persistent launch over a table of segments.
//
// Table layout (device): uint32 nsegs, uint32 prefix[nsegs + 1] (prefix[0] =
// 0, prefix[i] = queries in segments 0..i-1), then the pndf_segment array at
// a 16-byte boundary.  Warps pull global work indices from one cursor; index k
// belongs to the last segment i with prefix[i] <= k.
// ---------------------------------------------------------------------------

namespace {

constexpr int kServePrefixSmem = 1025;  // prefix sums of up to 1024 segments per step in shared memory

// CLUSTER / KERN: the server's evaluation variant (the cut, the footprint
// kernel or the clamp), compiled in as for traverse_kernel.
// Segment of work index k: the last segment i with prefix[i] <= k.
__device__ __forceinline__ int serve_segment(const uint32_t *prefix, int nsegs, uint32_t k)
{
    int lo = 0, hi = nsegs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= k)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The step's division of large footprints, as for pndf_eval_batch: the work
// estimate summed over the step's queries, then the plan (which also stores
// the target w_t for the step kernel, which recomputes each query's choice).
template <int KERN>
__global__ void serve_split_work(const uint32_t *__restrict__ table, const pndf_segment *__restrict__ segs,
                                 float jac_eps, double *__restrict__ work)
{
    __shared__ double red[256];
    const int nsegs = int(table[0]);
    const uint32_t *prefix = table + 1;
    const uint32_t total = prefix[nsegs];
    double acc = 0.0;
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
        const pndf_segment &sg = segs[serve_segment(prefix, nsegs, k)];
        const int64_t j = int64_t(sg.first) + int64_t(k - prefix[&sg - segs]);
        acc += double(split_estimate(make_query<KERN>(sg.q[sg.order ? int64_t(sg.order[j]) : j], jac_eps)));
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (int(threadIdx.x) < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(work, red[0]);
}

template <int KERN>
__global__ void serve_split_plan(const MapDesc *__restrict__ maps, const uint32_t *__restrict__ table,
                                 const pndf_segment *__restrict__ segs, float jac_eps, SplitPlan p)
{
    const float wt = split_target(p);
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.wt = wt;
    const int nsegs = int(table[0]);
    const uint32_t *prefix = table + 1;
    const uint32_t total = prefix[nsegs];
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
        const int i = serve_segment(prefix, nsegs, k);
        const pndf_segment &sg = segs[i];
        const int64_t j = int64_t(sg.first) + int64_t(k - prefix[i]);
        const uint32_t qi = sg.order ? sg.order[j] : uint32_t(j);
        const auto q = make_query<KERN>(sg.q[qi], jac_eps);
        int level;
        uint32_t tiles;
        if (split_choice(q, maps[sg.map].L, wt, level, tiles) && !split_reserve(p, qi, i, level, tiles))
            record_status(maps[sg.map].status, &g_status_eval, PNDF_QF_OVERFLOW);
    }
}

template <int BFMT, int TFMT, bool CLUSTER, int KERN>
__global__ void __launch_bounds__(256, kTraverseCtas)
    serve_kernel(const MapDesc *__restrict__ maps, const ClusterDesc *__restrict__ clusters, int nmaps,
                 const uint32_t *__restrict__ table, const pndf_segment *__restrict__ segs,
                 unsigned long long *__restrict__ cursor, float tau, float jac_eps, SplitPlan sp)
{
    extern __shared__ uint32_t smem[];
    __shared__ MapDesc smaps[kServeMaxMaps];
    __shared__ uint32_t sprefix[kServePrefixSmem];
    __shared__ unsigned long long s_ntiles;
    __shared__ int s_entries;
    __shared__ float s_wt;
    __shared__ uint32_t s_dest[8][3];  // per warp: segment, query, entry (-1: whole query)
    __shared__ Query<KERN> s_query[8];
    const int nsegs = int(table[0]);
    // the segment prefix sums, searched once per query, in shared memory when they fit
    const bool prefix_in_smem = nsegs < kServePrefixSmem;
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(maps);
        uint32_t *dst = reinterpret_cast<uint32_t *>(smaps);
        const int words = nmaps * int(sizeof(MapDesc) / sizeof(uint32_t));
        for (int i = threadIdx.x; i < words; i += blockDim.x) dst[i] = src[i];
        if (prefix_in_smem)
            for (int i = threadIdx.x; i <= nsegs; i += blockDim.x) sprefix[i] = table[1 + i];
        if (threadIdx.x == 0) {
            // the divided queries' tiles take the first s_ntiles work indices
            int n = 0;
            unsigned long long t = 0ull;
            float wt = __int_as_float(0x7f800000);
            if (!CLUSTER && sp.entries) {
                n = int(min(__ldcg(sp.ctr) >> 40, (unsigned long long)sp.cap));
                if (n > 0) t = __ldcg(&sp.entries[n - 1].base) + __ldcg(&sp.entries[n - 1].tiles);
                wt = __ldcg(sp.wt);
            }
            s_entries = n;
            s_ntiles = t;
            s_wt = wt;
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *wsm = smem + warp * kWarpSmemWords<CLUSTER>;
    const uint32_t *prefix = prefix_in_smem ? sprefix : table + 1;
    const uint32_t total = prefix[nsegs];
    while (true) {
        unsigned long long k = 0;
        if (lane == 0) k = atomicAdd(cursor, 1ull);
        k = __shfl_sync(kFull, k, 0);
        if (CLUSTER) {
            if (k >= total) break;
            const int i = serve_segment(prefix, nsegs, uint32_t(k));
            const pndf_segment sg = segs[i];
            const int64_t j = int64_t(sg.first) + int64_t(uint32_t(k) - prefix[i]);
            const int64_t qi = sg.order ? int64_t(sg.order[j]) : j;
            float Dv;
            uint32_t fv;
            eval_one<BFMT, TFMT, false, false, CLUSTER, KERN>(smaps[sg.map], clusters[sg.map], tau, jac_eps, sg.q[qi],
                                                               lane, wsm, s_query[warp], Dv, fv, nullptr);
            if (lane == 0) {
                sg.D[qi] = Dv;
                if (sg.flags) sg.flags[qi] = fv;
            }
            continue;
        }
        // a tile of a divided query, or a whole query: one descent either way
        constexpr bool CLAMP = KERN == kKernGaussClamp;
        int ei = -1;
        int i;
        uint32_t qi;
        Query<KERN> q;
        int e, a0, a1, c0, c1;
        if (k < s_ntiles) {
            ei = tile_entry(sp, s_entries, k);
            const SplitEntry &E = sp.entries[ei];
            i = __ldg(&E.pad);
            qi = __ldg(&E.qi);
            q = make_query<KERN>(segs[i].q[qi], jac_eps);
            e = __ldg(&E.level);
            tile_range(q, smaps[segs[i].map].L, e, uint32_t(k - __ldg(&E.base)), a0, a1, c0, c1);
        } else {
            k -= s_ntiles;
            if (k >= total) break;
            i = serve_segment(prefix, nsegs, uint32_t(k));
            const int64_t j = int64_t(segs[i].first) + int64_t(uint32_t(k) - prefix[i]);
            qi = segs[i].order ? segs[i].order[j] : uint32_t(j);
            q = make_query<KERN>(segs[i].q[qi], jac_eps);
            const int L = smaps[segs[i].map].L;
            if (!q.valid) {
                if (lane == 0) {
                    segs[i].D[qi] = __int_as_float(0x7fc00000);
                    if (segs[i].flags) segs[i].flags[qi] = PNDF_QF_INVALID;
                    record_status(smaps[segs[i].map].status, &g_status_eval, PNDF_QF_INVALID);
                }
                continue;
            }
            {
                int l;
                uint32_t t;
                if (split_choice(q, L, s_wt, l, t)) continue;  // evaluated as tiles
            }
            e = entry_level(q, L);
            const float sz = float(1u << e);
            node_range(q.x, q.rx, sz, 1 << (L - e), a0, a1);
            node_range(q.y, q.ry, sz, 1 << (L - e), c0, c1);
        }
        // where the result goes waits in shared memory during the descent
        __syncwarp();
        if (lane == 0) {
            s_dest[warp][0] = uint32_t(i);
            s_dest[warp][1] = qi;
            s_dest[warp][2] = uint32_t(ei);
            s_query[warp] = q;
        }
        __syncwarp();
        const int map = segs[i].map;
        Acc acc = {};
        acc_zero();
        eval_range<BFMT, TFMT, false, false, CLAMP>(smaps[map], kNoClusters, s_query[warp], e, a0, a1, c0, c1, lane, wsm, acc);
        unsigned long long lo, hi;
        uint32_t fl;
        warp_total<false>(acc, lo, hi, fl);
        if (lane == 0) {
            const pndf_segment &sg = segs[s_dest[warp][0]];
            const uint32_t qo = s_dest[warp][1];
            const int eo = int(s_dest[warp][2]);
            const MapDesc &md = smaps[sg.map];
            if (eo >= 0) {
                tile_finish<false>(md, sp.entries[eo], acc, lo, hi, fl, sg.D, sg.flags, nullptr);
            } else {
                sg.D[qo] = acc_value(lo, hi, fl);
                if (sg.flags) sg.flags[qo] = fl & ~kHuge;
                if (fl & PNDF_QF_OVERFLOW) record_status(md.status, &g_status_eval, PNDF_QF_OVERFLOW);
            }
        }
    }
}

template <int BFMT, int TFMT, bool CLUSTER, int KERN>
cudaError_t launch_serve_t(const ServeVariant &v, const MapDesc *maps, const ClusterDesc *clusters, int nmaps,
                           const uint32_t *table, const pndf_segment *segs, unsigned long long *cursor, int warps,
                           int ctas_per_sm, void *split, uint32_t split_cap, cudaStream_t s)
{
    auto kern = serve_kernel<BFMT, TFMT, CLUSTER, KERN>;
    int threads = warps * 32;
    size_t smem = size_t(warps) * kWarpSmemWords<CLUSTER> * sizeof(uint32_t);
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) occ = 1;
    if (ctas_per_sm > 0 && ctas_per_sm < occ) occ = ctas_per_sm;
    SplitPlan sp{};
    if (!CLUSTER && split) {
        char *b = static_cast<char *>(split);
        sp.ctr = reinterpret_cast<unsigned long long *>(b);
        sp.work = reinterpret_cast<double *>(b + 8);
        sp.wt = reinterpret_cast<float *>(b + 16);
        sp.entries = reinterpret_cast<SplitEntry *>(b + 256);
        sp.cap = split_cap;
        sp.resident_warps = sms * occ * warps;
        e = cudaMemsetAsync(split, 0, 256, s);
        if (e != cudaSuccess) return e;
        serve_split_work<KERN><<<unsigned(sms * 4), 256, 0, s>>>(table, segs, v.jac_eps, sp.work);
        serve_split_plan<KERN><<<unsigned(sms * 4), 256, 0, s>>>(maps, table, segs, v.jac_eps, sp);
    }
    kern<<<unsigned(sms * occ), threads, smem, s>>>(maps, clusters, nmaps, table, segs, cursor, v.tau, v.jac_eps, sp);
    return cudaGetLastError();
}

// Allow the variant's kernel the dynamic shared memory of `warps` warps (with
// its static tables the total passes the 48 KB a launch gets by default).
template <int BFMT, int TFMT, bool CLUSTER, int KERN>
cudaError_t serve_smem_t(int warps)
{
    return cudaFuncSetAttribute(serve_kernel<BFMT, TFMT, CLUSTER, KERN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                warps * kWarpSmemWords<CLUSTER> * int(sizeof(uint32_t)));
}

template <int BFMT, int TFMT>
cudaError_t serve_smem_v(const ServeVariant &v, int warps)
{
    if (v.tau > 0.f) return serve_smem_t<BFMT, TFMT, true, PNDF_KERNEL_GAUSS>(warps);
    if (v.jac_eps > 0.f) return serve_smem_t<BFMT, TFMT, false, kKernGaussClamp>(warps);
    if (v.kernel == PNDF_KERNEL_DISK) return serve_smem_t<BFMT, TFMT, false, PNDF_KERNEL_DISK>(warps);
    if (v.kernel == PNDF_KERNEL_BOX) return serve_smem_t<BFMT, TFMT, false, PNDF_KERNEL_BOX>(warps);
    return serve_smem_t<BFMT, TFMT, false, PNDF_KERNEL_GAUSS>(warps);
}

// The variant's instantiation: the cut (Gaussian), the plain Gaussian, disk,
// box, or the Gaussian with the Eq. 6 clamp (the server validated the mix).
template <int BFMT, int TFMT>
cudaError_t launch_serve_v(const ServeVariant &v, const MapDesc *maps, const ClusterDesc *clusters, int nmaps,
                           const uint32_t *table, const pndf_segment *segs, unsigned long long *cursor, int warps,
                           int ctas_per_sm, void *split, uint32_t split_cap, cudaStream_t s)
{
#define PNDF_SERVE(C, K)                                                                                     \
    launch_serve_t<BFMT, TFMT, C, K>(v, maps, clusters, nmaps, table, segs, cursor, warps, ctas_per_sm, split, \
                                     split_cap, s)
    if (v.tau > 0.f) return PNDF_SERVE(true, PNDF_KERNEL_GAUSS);
    if (v.jac_eps > 0.f) return PNDF_SERVE(false, kKernGaussClamp);
    if (v.kernel == PNDF_KERNEL_DISK) return PNDF_SERVE(false, PNDF_KERNEL_DISK);
    if (v.kernel == PNDF_KERNEL_BOX) return PNDF_SERVE(false, PNDF_KERNEL_BOX);
    return PNDF_SERVE(false, PNDF_KERNEL_GAUSS);
#undef PNDF_SERVE
}

}  // namespace

cudaError_t prepare_serve(int texel_fmt, int bounds_fmt, const ServeVariant &v, int warps)
{
    if (bounds_fmt == PNDF_BOUNDS_F32)
        return texel_fmt == PNDF_TEXEL_F32X2 ? serve_smem_v<PNDF_BOUNDS_F32, PNDF_TEXEL_F32X2>(v, warps)
                                             : serve_smem_v<PNDF_BOUNDS_F32, PNDF_TEXEL_F16X2>(v, warps);
    return texel_fmt == PNDF_TEXEL_F32X2 ? serve_smem_v<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F32X2>(v, warps)
                                         : serve_smem_v<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F16X2>(v, warps);
}

// Scratch of a step's division of large footprints: a 256-byte header
// (counter, work sum, target) and the entries.
uint32_t serve_split_cap()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return uint32_t(2 * 64 * (sms > 0 ? sms : 1) + 64);  // >= 2 x the resident warps
}

size_t serve_split_bytes(uint32_t cap) { return 256 + size_t(cap) * sizeof(SplitEntry); }

cudaError_t launch_serve(int texel_fmt, int bounds_fmt, const ServeVariant &v, const MapDesc *maps,
                         const ClusterDesc *clusters, int nmaps, const uint32_t *table, const pndf_segment *segs,
                         unsigned long long *cursor, int warps, int ctas_per_sm, void *split, uint32_t split_cap,
                         cudaStream_t s)
{
#define PNDF_SERVE_V(B, T) \
    launch_serve_v<B, T>(v, maps, clusters, nmaps, table, segs, cursor, warps, ctas_per_sm, split, split_cap, s)
    if (bounds_fmt == PNDF_BOUNDS_F32)
        return texel_fmt == PNDF_TEXEL_F32X2 ? PNDF_SERVE_V(PNDF_BOUNDS_F32, PNDF_TEXEL_F32X2)
                                             : PNDF_SERVE_V(PNDF_BOUNDS_F32, PNDF_TEXEL_F16X2);
    return texel_fmt == PNDF_TEXEL_F32X2 ? PNDF_SERVE_V(PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F32X2)
                                         : PNDF_SERVE_V(PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F16X2);
#undef PNDF_SERVE_V
}

// ---------------------------------------------------------------------------
// Allocation-free evaluation (pndf_eval_batch_noalloc).
//
// Some callers cannot allocate device memory while they evaluate: a renderer
// plugin whose host owns every device allocation and forbids others, a
// real-time thread that must not take cudaMalloc's implicit device-wide
// synchronisation or its latency, or code that budgets device memory exactly
// ahead of time.  For them the sort scratch lives in one fixed device array,
// defined here at file scope and held by every GPU that loads the library
// until the process exits.  The host never uses the array's name as an
// address: on the first call on each device, with that device current, the
// device address is looked up with cudaGetSymbolAddress and cached per
// device, keyed by the id of the context it was looked up in, so that after a
// device reset (which unloads the module with its array) the first call in the
// new context looks the address up again.
// Every call shares the array and it keeps the previous call's contents, so
// the cursor and histogram are cleared on the stream at the start of each
// call; calls whose work overlaps on the GPU (different streams, or work not
// yet complete on another stream) race on the array and must be serialised by
// the caller.
// ---------------------------------------------------------------------------

namespace {

constexpr int64_t kNoallocMaxQueries = int64_t(1) << 20;
constexpr size_t kNoallocHistOff = 256;
constexpr size_t kNoallocKeysOff = kNoallocHistOff + size_t(kKeyBins) * sizeof(uint32_t);
constexpr size_t kNoallocOrderOff = kNoallocKeysOff + size_t(kNoallocMaxQueries) * sizeof(uint32_t);
constexpr size_t kNoallocBytes = kNoallocOrderOff + size_t(kNoallocMaxQueries) * sizeof(uint32_t);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

struct NoallocSlot {
    unsigned long long ctx_id;  // id of the context the address belongs to
    void *ptr;                  // device address of g_noalloc_scratch there (null: not looked up)
};

std::mutex g_noalloc_mutex;
NoallocSlot g_noalloc_slot[64] = {};

// Id of the calling thread's current context (driver entry points taken
// through the runtime, so the library links no driver library); false when
// there is none yet or the driver does not provide them.
bool current_context_id(unsigned long long *id)
{
    using GetCurrent = int (*)(void **);
    using GetId = int (*)(void *, unsigned long long *);
    static GetCurrent get_current = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult r;
        return cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &r) == cudaSuccess &&
                       r == cudaDriverEntryPointSuccess
                   ? reinterpret_cast<GetCurrent>(f)
                   : nullptr;
    }();
    static GetId get_id = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult r;
        return cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &r) == cudaSuccess &&
                       r == cudaDriverEntryPointSuccess
                   ? reinterpret_cast<GetId>(f)
                   : nullptr;
    }();
    void *ctx = nullptr;
    if (!get_current || !get_id || get_current(&ctx) != 0 || !ctx) return false;
    return get_id(ctx, id) == 0;
}

// Device address of g_noalloc_scratch on the current device: looked up on
// the first call in each context (with the device current), then cached.
cudaError_t noalloc_scratch(void **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    unsigned long long id = 0;
    bool have_id = current_context_id(&id);
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoallocSlot &slot = g_noalloc_slot[dev];
    if (!have_id || !slot.ptr || slot.ctx_id != id) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        if (!have_id) have_id = current_context_id(&id);  // the lookup made the context current
        slot.ptr = p;
        slot.ctx_id = have_id ? id : 0ull;
        if (!have_id) {  // no context id to key on: look up again next time
            *out = p;
            slot.ptr = nullptr;
            return cudaSuccess;
        }
    }
    *out = slot.ptr;
    return cudaSuccess;
}

}  // namespace

int64_t noalloc_max_queries() { return kNoallocMaxQueries; }

pndf_status launch_eval_noalloc(const pndf_hierarchy *h, const pndf_query *q, int64_t nq, float *D, uint32_t *flags,
                                cudaStream_t s)
{
    if (nq > kNoallocMaxQueries) return PNDF_ERR_CAPACITY;
    if (nq == 0) return PNDF_OK;
    void *scratch = nullptr;
    if (noalloc_scratch(&scratch) != cudaSuccess) return PNDF_ERR_CUDA;
    const MapDesc &d = h->d;
    pndf_eval_config cfg{PNDF_MODE_HIERARCHY, PNDF_SORT_DEFAULT, 0, 0, 0.f, PNDF_KERNEL_GAUSS, 0.f, 0, nullptr, nullptr};
    char *base = static_cast<char *>(scratch);
    auto *cursor = reinterpret_cast<unsigned long long *>(base);
    auto *hist = reinterpret_cast<uint32_t *>(base + kNoallocHistOff);
    auto *keys = reinterpret_cast<uint32_t *>(base + kNoallocKeysOff);
    auto *order = reinterpret_cast<uint32_t *>(base + kNoallocOrderOff);
    // cursor and histogram start at zero
    cudaError_t e = cudaMemsetAsync(base, 0, kNoallocHistOff + sort_hist_bytes(nq), s);
    if (e != cudaSuccess) return PNDF_ERR_CUDA;
    e = sort_launch(d, q, nq, cfg.sort, hist, keys, order, s);
    if (e != cudaSuccess) return PNDF_ERR_CUDA;
    if (d.bounds_fmt == PNDF_BOUNDS_F32)
        e = d.texel_fmt == PNDF_TEXEL_F32X2
                ? dispatch_stats<PNDF_BOUNDS_F32, PNDF_TEXEL_F32X2>(d, h->c, q, order, nq, D, flags, nullptr, cursor, cfg, SplitPlan{}, s)
                : dispatch_stats<PNDF_BOUNDS_F32, PNDF_TEXEL_F16X2>(d, h->c, q, order, nq, D, flags, nullptr, cursor, cfg, SplitPlan{}, s);
    else
        e = d.texel_fmt == PNDF_TEXEL_F32X2
                ? dispatch_stats<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F32X2>(d, h->c, q, order, nq, D, flags, nullptr, cursor,
                                                                         cfg, SplitPlan{}, s)
                : dispatch_stats<PNDF_BOUNDS_F16_OUTWARD, PNDF_TEXEL_F16X2>(d, h->c, q, order, nq, D, flags, nullptr, cursor,
                                                                         cfg, SplitPlan{}, s);
    return e == cudaSuccess ? PNDF_OK : PNDF_ERR_CUDA;
}

namespace {
__global__ void take_eval_word(unsigned int *out) { *out = atomicExch(&g_status_eval, 0u); }
}  // namespace

cudaError_t take_status_eval(unsigned int *out, cudaStream_t s)
{
    take_eval_word<<<1, 1, 0, s>>>(out);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace pndf

// Mean of the visible integrand over one normal triangle, in FP32.
//
// With V_T of Eq. 10, V_T / |cross(T)| is half the mean over the triangle's uv
// of g(m) = max(w . m~, 0) / m~_z at m = n(u), affine in u.  g is smooth where
// it is positive, so a positive-weight quadrature of degree d leaves an error
// that falls as h^(d+1), needs no division by |cross| (slivers and collapsed
// triangles are ordinary ones) and never cancels.  h here is the longest edge
// over the smallest m~_z^2 of the triangle, its size against the distance of
// m~_z = 0, where g is singular.  Errors against a 196-point rule, random
// triangles, root mean square: 6 points (degree 4) 3e-9 at h = 0.15, 7e-8 at 0.3;
// 12 points (degree 6) 5e-9 at 0.5, 8e-8 at 0.8.  Rules: Dunavant, "High degree
// efficient symmetrical Gaussian quadrature rules for the triangle", 1985.
//
// A triangle the boundary w . m~ = 0 crosses is cut along it into a polygon and the
// cap that bows out of it, each again a positive smooth integral (partial_mean);
// the few whose cap is cut off or too oblique take the closed form.  Larger
// triangles are split in four at their edges' midpoints; what is still too
// large goes to the closed form in FP64 (visible.cuh).
#pragma once

namespace pndf {

struct Dir {
    float wx, wy, wz;  // unit direction
};

constexpr float kSmallH2 = 0.15f * 0.15f;  // h^2 up to which the 6-point rule serves
constexpr float kLargeH2 = 0.8f * 0.8f;    // and the 12-point rule and partial_mean

// Unit direction from the caller's (unit to single precision) vector, each
// component rounded once: an error here is the same for every triangle of the
// footprint.
__device__ __forceinline__ Dir make_dir_f(float x, float y, float z)
{
    const double n = rsqrt(double(x) * x + double(y) * y + double(z) * z);
    return Dir{float(x * n), float(y * n), float(z * n)};
}

__device__ __forceinline__ float zof(float2 p)
{
    return sqrtf(fmaxf(0.f, 1.f - fmaf(p.x, p.x, p.y * p.y)));
}

__device__ __forceinline__ float phi_of(const Dir &w, float2 p, float z)
{
    return fmaf(w.wx, p.x, fmaf(w.wy, p.y, w.wz * z));
}

// (w_xy . m) / m~_z at m = (x, y); g = max(w_z + this, 0).
__device__ __forceinline__ float slope_at(const Dir &w, float x, float y)
{
    const float rz = rsqrtf(fmaxf(fmaf(-x, x, fmaf(-y, y, 1.0f)), 1e-30f));
    return fmaf(w.wx, x, w.wy * y) * rz;
}

// m / m~_z at m = (x, y).
__device__ __forceinline__ float2 ratio_at(float x, float y)
{
    const float rz = rsqrtf(fmaxf(fmaf(-x, x, fmaf(-y, y, 1.0f)), 1e-30f));
    return make_float2(x * rz, y * rz);
}

// The degree-4 rule: two orbits of three points (u, u, 1 - 2u).
constexpr float kQ4u0 = 0.445948490915965f, kQ4w0 = 0.223381589678011f;
constexpr float kQ4u1 = 0.091576213509771f, kQ4w1 = 0.109951743655322f;
// The degree-6 rule: two orbits of three and one of six.
constexpr float kQ6u0 = 0.063089014491502f, kQ6w0 = 0.050844906370207f;
constexpr float kQ6u1 = 0.249286745170910f, kQ6w1 = 0.116786275726379f, kQ6w2 = 0.082851075618374f;
constexpr float kQ6a = 0.310352451033785f, kQ6b = 0.053145049844816f, kQ6c = 0.636502499121399f;

// Sum over a rule's points of weight * f(point): the point with barycentric
// coordinates (1 - s - t, s, t) is a + s e1 + t e2.
template <class F>
__device__ __forceinline__ auto quad4(float2 a, float2 e1, float2 e2, F f)
{
    auto at = [&](float s, float t) { return f(fmaf(t, e2.x, fmaf(s, e1.x, a.x)), fmaf(t, e2.y, fmaf(s, e1.y, a.y))); };
    auto o0 = at(kQ4u0, kQ4u0) + at(1.f - 2.f * kQ4u0, kQ4u0) + at(kQ4u0, 1.f - 2.f * kQ4u0);
    auto o1 = at(kQ4u1, kQ4u1) + at(1.f - 2.f * kQ4u1, kQ4u1) + at(kQ4u1, 1.f - 2.f * kQ4u1);
    return o0 * kQ4w0 + o1 * kQ4w1;
}

template <class F>
__device__ __forceinline__ auto quad6(float2 a, float2 e1, float2 e2, F f)
{
    auto at = [&](float s, float t) { return f(fmaf(t, e2.x, fmaf(s, e1.x, a.x)), fmaf(t, e2.y, fmaf(s, e1.y, a.y))); };
    auto o0 = at(kQ6u0, kQ6u0) + at(1.f - 2.f * kQ6u0, kQ6u0) + at(kQ6u0, 1.f - 2.f * kQ6u0);
    auto o1 = at(kQ6u1, kQ6u1) + at(1.f - 2.f * kQ6u1, kQ6u1) + at(kQ6u1, 1.f - 2.f * kQ6u1);
    auto o2 = at(kQ6a, kQ6b) + at(kQ6b, kQ6a) + at(kQ6a, kQ6c) + at(kQ6c, kQ6a) + at(kQ6b, kQ6c) + at(kQ6c, kQ6b);
    return o0 * kQ6w0 + o1 * kQ6w1 + o2 * kQ6w2;
}

struct V2 {
    float x, y;
};
__device__ __forceinline__ V2 operator+(V2 a, V2 b) { return V2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ V2 operator*(V2 a, float s) { return V2{a.x * s, a.y * s}; }

__device__ __forceinline__ float len2(float2 v) { return fmaf(v.x, v.x, v.y * v.y); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

// How a triangle is integrated.
enum Class : int { kNone, kSmall, kLarge, kPartial, kSplit };

// Class of a triangle with phi = w . m~ and m~_z at its vertices, longest edge
// squared h2.  m~_z is concave with second derivative at most 1 / m~_z^3, so
// phi exceeds its linear interpolant by at most w_z h2 / (6 zmin^3): below zero
// by that much at every vertex, it is negative everywhere.  (5e-7 covers the
// rounding of phi.)
__device__ __forceinline__ Class classify(float fa, float fb, float fc, float za, float zb, float zc, float h2,
                                          const Dir &w)
{
    const float zm = fminf(za, fminf(zb, zc)), z2 = zm * zm;
    const float s2 = z2 * z2;  // h^2 = h2 / s2
    if (fminf(fa, fminf(fb, fc)) >= 0.f) return h2 <= kSmallH2 * s2 ? kSmall : h2 <= kLargeH2 * s2 ? kLarge : kSplit;
    if (fmaf(fmaxf(fa, fmaxf(fb, fc)) + 5e-7f, 6.f * z2 * zm, w.wz * h2) < 0.f) return kNone;
    return h2 <= kLargeH2 * s2 ? kPartial : kSplit;
}

// Where the segment m + t d leaves (m visible) or enters (m not visible) the
// visible region: w . m~ = 0 squared is a quadratic in t whose constant term
// factors into phi(m) times -(w_z m~_z - w_xy . m), so it is as accurate as phi.
struct Ray {
    float wm, f, z;  // w_xy . m, phi(m), m~_z of the start
    float2 m;
};
__device__ __forceinline__ void ray_terms(const Dir &w, const Ray &r, float2 d, float &qa, float &qb, float &qc,
                                          float &root)
{
    const float wd = fmaf(w.wx, d.x, w.wy * d.y), wz2 = w.wz * w.wz;
    qa = fmaf(wd, wd, wz2 * len2(d));
    qb = fmaf(r.wm, wd, wz2 * fmaf(r.m.x, d.x, r.m.y * d.y));
    qc = -fmaf(w.wz, r.z, -r.wm) * r.f;
    root = sqrtf(fmaxf(fmaf(qb, qb, -qa * qc), 0.f));
}
__device__ __forceinline__ float ray_exit(const Dir &w, const Ray &r, float2 d)
{
    float qa, qb, qc, root;
    ray_terms(w, r, d, qa, qb, qc, root);
    return qb <= 0.f ? __fdividef(root - qb, qa) : __fdividef(-qc, qb + root);
}
__device__ __forceinline__ float ray_enter(const Dir &w, const Ray &r, float2 d)
{
    float qa, qb, qc, root;
    ray_terms(w, r, d, qa, qb, qc, root);
    return __fdividef(qc, root - qb);
}

// Gauss-Legendre on [0, 1]: four points across the visible polygon and five along
// it, five across a cap and two along its rays (weights 1/2).
__constant__ float kGx4[4] = {0.069431844202974f, 0.330009478207572f, 0.669990521792428f, 0.930568155797026f};
__constant__ float kGw4[4] = {0.173927422568727f, 0.326072577431273f, 0.326072577431273f, 0.173927422568727f};
__constant__ float kGx5[5] = {0.046910077030668f, 0.230765344947158f, 0.5f, 0.769234655052842f, 0.953089922969332f};
__constant__ float kGw5[5] = {0.118463442528095f, 0.239314335249683f, 0.284444444444444f, 0.239314335249683f,
                              0.118463442528095f};
__constant__ float kGx2[2] = {0.211324865405187f, 0.788675134594813f};

// Half the mean of g over a triangle of class kPartial; negative if it needs the
// closed form after all.  Let A be the vertex whose visibility differs from the
// other two and p, q the points where edges AB and AC meet the boundary.  The
// visible part is a polygon, on which g is smooth, and the cap between its chord
// pq and the boundary, which bows out of it (the visible region is convex):
//   one vertex visible: the triangle (A, p, q);
//   two: the quadrilateral (B, C, q, p);
//   none: no polygon, p and q both on the one edge that dips into view.
// The polygon is integrated along the lines from its base (A, or BC) to the chord,
// 4 x 5 points, the triangle as a quadrilateral whose base has no length; the cap
// along rays across the chord, 5 x 2 points, each ray cut at the boundary.  The
// boundary is a conic that meets the chord at its ends, so the cut follows without
// cancellation, however close p and q are to A or to each other.  E, the rays'
// direction, lies across the chord in the uv triangle; where it runs along it in
// normal space (slivers), the boundary's slopes along E at the chord's two ends
// differ, and the closed form takes the triangle once they differ by more than
// twice (up to there the cap is good to 1e-6 of itself).  So it does where an edge
// between vertices that are not visible cuts the cap off, or where two of them dip
// into view: 1 to 4 in 10,000 partly visible triangles of flake, scratch, bump and
// noise maps.
//   Error against the closed form, FP32 rounding included: at most 1.2e-7, root
// mean square 1e-9 to 6e-9, over 2.6 million such triangles of those maps, two
// thirds of them with the direction turned until a vertex or an edge came within
// 1e-8 .. 0.03 of the boundary.
//   All lanes run the same 30 points, so that a mixed warp pays for one kind of
// triangle: against a fan of rays from A alone, which missed what lies beside AC
// where q is near A, 192 requests on the 16384^2 mixed map 15.75 -> 15.52 ms, 1000
// small footprints on a scratch map 283 -> 270 us; with a fan for one vertex and two
// triangles for two (66 points for a mixed warp) 14.13 -> 14.96 ms and 341 -> 374 us
// in another run.
__device__ __noinline__ float partial_mean(float2 a, float2 b, float2 c, const Dir &w)
{
    float fa = phi_of(w, a, zof(a)), fb = phi_of(w, b, zof(b)), fc = phi_of(w, c, zof(c));
    const bool va = fa >= 0.f, vb = fb >= 0.f, vc = fc >= 0.f;
    const int seen = int(va) + int(vb) + int(vc);
    auto g = [&](float x, float y) { return fmaxf(w.wz + slope_at(w, x, y), 0.f); };
    auto ray = [&](float2 m, float f) { return Ray{fmaf(w.wx, m.x, w.wy * m.y), f, zof(m), m}; };
    // visible part [t0, t1] of the edge m -> m + e between vertices that are not visible
    auto dips = [&](float2 m, float f, float2 e, float &t0, float &t1) {
        float qa, qb, qc, root;
        ray_terms(w, ray(m, f), e, qa, qb, qc, root);
        t0 = fmaxf(__fdividef(-qb - root, qa), 0.f);
        t1 = fminf(__fdividef(root - qb, qa), 1.f);
        return root > 0.f && t0 < t1;
    };
    // the cap: chord O + x dO, rays along E; coef: |dO x E| in barycentric coordinates
    float2 O = make_float2(0.f, 0.f), dO = O, E = O;
    float coef = 0.f, poly = 0.f;
    if (seen == 0) {
        int edges = 0;
#pragma unroll 1
        for (int k = 0; k < 3; ++k) {
            const float2 e = sub(b, a);
            float t0, t1;
            if (dips(a, fa, e, t0, t1)) {
                ++edges;
                coef = t1 - t0;
                O = make_float2(fmaf(t0, e.x, a.x), fmaf(t0, e.y, a.y));
                dO = make_float2(coef * e.x, coef * e.y);
                E = make_float2(c.x - 0.5f * (a.x + b.x), c.y - 0.5f * (a.y + b.y));
            }
            const float2 t = a; a = b; b = c; c = t;  // next edge
            const float f = fa; fa = fb; fb = fc; fc = f;
        }
        if (edges == 0) return 0.f;
        if (edges > 1) return -1.f;
    } else {
        const bool one = seen == 1;
        if (vb != va && vb != vc) {  // the odd vertex to the front
            const float2 t = a; a = b; b = t;
            const float f = fa; fa = fb; fb = f;
        } else if (vc != va && vc != vb) {
            const float2 t = a; a = c; c = t;
            const float f = fa; fa = fc; fc = f;
        }
        float t0, t1;
        if (one && dips(b, fb, sub(c, b), t0, t1)) return -1.f;
        const float2 ab = sub(b, a), ac = sub(c, a);
        const Ray ra = ray(a, fa);
        const float tb = fminf(fmaxf(one ? ray_exit(w, ra, ab) : ray_enter(w, ra, ab), 0.f), 1.f);
        const float tc = fminf(fmaxf(one ? ray_exit(w, ra, ac) : ray_enter(w, ra, ac), 0.f), 1.f);
        O = make_float2(fmaf(tb, ab.x, a.x), fmaf(tb, ab.y, a.y));
        dO = make_float2(fmaf(tc, ac.x, a.x) - O.x, fmaf(tc, ac.y, a.y) - O.y);
        // (tc, tb) in barycentric coordinates, across the chord (-tb, tc); away from A, or towards it
        const float out = one ? 1.f : -1.f;
        E = make_float2(out * fmaf(tc, ab.x, tb * ac.x), out * fmaf(tc, ab.y, tb * ac.y));
        coef = fmaf(tb, tb, tc * tc);
        const float base = one ? 0.f : 1.f;
        const float2 u0 = one ? a : b, du = one ? make_float2(0.f, 0.f) : sub(c, b);
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
            const float x = kGx4[i];
            const float2 u = make_float2(fmaf(x, du.x, u0.x), fmaf(x, du.y, u0.y));
            const float2 e = make_float2(fmaf(x, dO.x, O.x) - u.x, fmaf(x, dO.y, O.y) - u.y);
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const float v = g(fmaf(kGx5[k], e.x, u.x), fmaf(kGx5[k], e.y, u.y));
                s0 = fmaf(kGw5[k], v, s0);
                s1 = fmaf(kGw5[k] * kGx5[k], v, s1);
            }
            // the map's Jacobian (barycentric) goes from j0 at the base to j1 at the chord
            const float yb = (1.f - x) * (base - tb), yc = x * (base - tc);
            const float j0 = base * (yb + yc), j1 = fmaf(tc, yb, tb * yc);
            poly = fmaf(kGw4[i], fmaf(j1 - j0, s1, j0 * s0), poly);
        }
        poly = fabsf(poly);
        if (coef < 1e-12f) return poly;  // (the cap is less than 1e-6 of the corner that A cuts off, which underflows)
    }
    // (w_z m~_z)^2 - (w_xy . m)^2 = ch x (1 - x) on the chord, ch x (1 - x) - 2 qb t - qa t^2 at t along its rays
    const float wd = fmaf(w.wx, E.x, w.wy * E.y), wc = fmaf(w.wx, dO.x, w.wy * dO.y), wz2 = w.wz * w.wz;
    const float qa = fmaf(wd, wd, wz2 * len2(E)), ch = fmaf(wc, wc, wz2 * len2(dO));
    auto slope = [&](float2 m) { return fmaf(fmaf(w.wx, m.x, w.wy * m.y), wd, wz2 * fmaf(m.x, E.x, m.y * E.y)); };
    const float q0 = slope(O), q1 = slope(make_float2(O.x + dO.x, O.y + dO.y));
    if (!(fminf(q0, q1) >= 0.5f * fmaxf(q0, q1) && q0 > 0.f)) return -1.f;
    float cap = 0.f;
#pragma unroll 1
    for (int i = 0; i < 5; ++i) {
        const float x = kGx5[i], f = ch * (x * (1.f - x)), qb = fmaf(x, q1 - q0, q0);
        const float t = __fdividef(f, qb + sqrtf(fmaf(qb, qb, qa * f)));
        const float ox = fmaf(x, dO.x, O.x), oy = fmaf(x, dO.y, O.y);
        float in = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) in += g(fmaf(kGx2[k] * t, E.x, ox), fmaf(kGx2[k] * t, E.y, oy));
        cap = fmaf(kGw5[i] * t, in, cap);
    }
    return fmaf(0.5f * coef, cap, poly);
}

}  // namespace pndf

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
// A triangle the boundary w . m~ = 0 crosses is cut along it into straight and
// curved pieces, each again a positive smooth integral (partial_mean).  Larger
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

// Gauss-Legendre on [0, 1]: six points across, five along (times the abscissa).
__constant__ float kGx6[6] = {0.033765242898424f, 0.169395306766868f, 0.380690406958402f,
                              0.619309593041599f, 0.830604693233132f, 0.966234757101576f};
__constant__ float kGw6[6] = {0.085662246189585f, 0.180380786524069f, 0.233956967286346f,
                              0.233956967286346f, 0.180380786524069f, 0.085662246189585f};
__constant__ float kGx5[5] = {0.046910077030668f, 0.230765344947158f, 0.5f, 0.769234655052842f, 0.953089922969332f};
__constant__ float kGw5[5] = {0.118463442528095f, 0.239314335249683f, 0.284444444444444f, 0.239314335249683f,
                              0.118463442528095f};

// Half the mean of g over a triangle of class kPartial; negative if it needs the
// closed form after all (two edges that both dip into view between vertices
// that do not).  Let A be the vertex whose visibility differs from the other
// two, p and q the points where edges AB and AC meet the boundary.
//   One vertex visible: the triangle (A, p, q) with the side pq bowed out to the
//     boundary (but not past BC).
//   Two: the straight triangle (p, B, C) and (C, p, q), pq again bowed out (C
//     the one that sees more).
//   None: the cap between an edge's visible part and the boundary.
// Bowed triangles are integrated along rays from their apex, caps along rays
// across the edge, each ray cut at the boundary, 6 x 5 points.  Root mean square
// error against 64 bits, FP32 rounding included, 2e-9 (h up to 0.4) to 2e-8
// (0.8).  Clipped in FP64, the same 2% of all triangles kept the kernel's FP64
// pipe 53% busy and took most of its time.
__device__ __noinline__ float partial_mean(float2 a, float2 b, float2 c, const Dir &w)
{
    float fa = phi_of(w, a, zof(a)), fb = phi_of(w, b, zof(b)), fc = phi_of(w, c, zof(c));
    const bool va = fa >= 0.f, vb = fb >= 0.f, vc = fc >= 0.f;
    const int seen = int(va) + int(vb) + int(vc);
    auto g = [&](float x, float y) { return fmaxf(w.wz + slope_at(w, x, y), 0.f); };
    auto ray = [&](float2 m, float f, float z) { return Ray{fmaf(w.wx, m.x, w.wy * m.y), f, z, m}; };
    // rays O + x dO, directions E + x dE, x in [0, 1], t up to 1 / (l + x dl)
    float2 O, dO = make_float2(0.f, 0.f), E, dE = make_float2(0.f, 0.f);
    float l, dl = 0.f, coef, rest = 0.f;
    if (seen == 0) {
        int edges = 0;
        O = E = dO;
        l = 1.f;
        coef = 0.f;
#pragma unroll 1
        for (int k = 0; k < 3; ++k) {
            const float2 e = sub(b, a);
            float qa, qb, qc, root;
            ray_terms(w, ray(a, fa, zof(a)), e, qa, qb, qc, root);
            const float tn = __fdividef(-qb - root, qa), tf = __fdividef(root - qb, qa);
            if (root > 0.f && tn > 0.f && tf < 1.f) {
                ++edges;
                O = make_float2(fmaf(tn, e.x, a.x), fmaf(tn, e.y, a.y));
                coef = tf - tn;
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
        // the odd vertex to the front, and of the other two the higher last
        if (vb != va && vb != vc) {
            const float2 t = a; a = b; b = t;
            const float f = fa; fa = fb; fb = f;
        } else if (vc != va && vc != vb) {
            const float2 t = a; a = c; c = t;
            const float f = fa; fa = fc; fc = f;
        }
        if (fb > fc) {
            const float2 t = b; b = c; c = t;
            const float f = fb; fb = fc; fc = f;
        }
        const float2 ab = sub(b, a), ac = sub(c, a);
        const Ray ra = ray(a, fa, zof(a));
        const float tb = fminf(fmaxf(one ? ray_exit(w, ra, ab) : ray_enter(w, ra, ab), 0.f), 1.f);
        const float tc = fminf(fmaxf(one ? ray_exit(w, ra, ac) : ray_enter(w, ra, ac), 0.f), 1.f);
        const float2 p = make_float2(fmaf(tb, ab.x, a.x), fmaf(tb, ab.y, a.y));
        const float2 q = make_float2(fmaf(tc, ac.x, a.x), fmaf(tc, ac.y, a.y));
        O = one ? a : c;
        E = sub(p, O);
        dE = sub(q, p);
        // areas against the triangle's: (A, p, q) tb tc, (C, p, q) tb (1 - tc), (p, B, C) 1 - tb
        coef = one ? tb * tc : tb * (1.f - tc);
        l = one ? tb : 0.25f;
        dl = one ? tc - tb : 0.f;
        if (!one) rest = 0.5f * (1.f - tb) * quad6(p, sub(b, p), sub(c, p), g);
    }
    const bool fan = seen != 0;
    float sum = 0.f;
#pragma unroll 1
    for (int i = 0; i < 6; ++i) {
        const float x = kGx6[i];
        const float2 o = make_float2(fmaf(x, dO.x, O.x), fmaf(x, dO.y, O.y));
        const float2 e = make_float2(fmaf(x, dE.x, E.x), fmaf(x, dE.y, E.y));
        const float z = zof(o), f = fmaxf(phi_of(w, o, z), 0.f);
        float t = ray_exit(w, ray(o, f, z), e);
        t = t >= 0.f ? fminf(t, fminf(4.f, __fdividef(1.f, fmaf(x, dl, l)))) : 0.f;  // (0 / 0: a point ray)
        float in = 0.f;
#pragma unroll
        for (int k = 0; k < 5; ++k)
            in = fmaf(kGw5[k] * (fan ? kGx5[k] : 1.f), g(fmaf(kGx5[k] * t, e.x, o.x), fmaf(kGx5[k] * t, e.y, o.y)), in);
        sum = fmaf(kGw6[i] * (fan ? t * t : t), in, sum);
    }
    return fmaf(coef, sum, rest);
}

}  // namespace pndf

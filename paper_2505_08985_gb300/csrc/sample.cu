// P-NDF sampling (Sec. 3, Eq. 6).
//
// A normal is drawn from D by drawing a uv point from the footprint kernel,
// u ~ k_r(u - x), and querying the map there, m = n(u) (Eq. 3); with the
// Jacobian clamp of Eq. 6 a fine triangle whose |cross| is below eps stands
// for its equilateral replacement (area eps / 2, centred at its normal
// centroid, vertex k at 90 + 120 k degrees, vertices in the uv order), so the
// density of the sampled normals is the clamped D over the kernel mass.
//
// u comes from the caller's two uniforms by the inverse CDF in the whitened
// frame v, u = x + L v with S = L L^T (Cholesky):
//   Gaussian cut at q = 16: |v|^2 = -2 ln(1 - U1 (1 - e^-8)), angle 2 pi U2;
//   disk (q <= 1.5^2): |v| = 1.5 sqrt(U1), angle 2 pi U2;
//   box (|v|_inf <= 1.5): v = 1.5 (2 U1 - 1, 2 U2 - 1).
// One thread per sample.  The position has to be as good as FP64 makes it, so that
// the triangle chosen for u agrees with a 64-bit reference except at ties; in FP64
// that bound the kernel (86% of the FP64 pipe, 395 us per million samples).  It runs
// in pairs of FP32 numbers (pair.cuh) instead, the centre's integer part kept apart
// so that only the offset within the footprint is rounded: 41 us, bound by FP32 issue and the four
// texel loads.  Largest error of the offset in sigma, pairs and FP64: Gaussian
// 3.7e-13 and 5.9e-13 (both where U1 is next to 0 and the logarithm's argument next
// to 1), disk 2.5e-14 and 7e-16, box 3.5e-14 and 6e-16, where FP64 rounds the centre
// too, to 1e-13 of a texel on a 2048^2 map and 1e-12 on a 16384^2 one.  Records
// outside the range where the pairs serve (extreme covariances or centres) take the
// FP64 form (sample_fp64).
#include <math.h>

#include "common.cuh"
#include "pair.cuh"
#include "tri.cuh"

namespace pndf {
namespace {

template <int TFMT>
__device__ __forceinline__ float2 texel_s(const MapDesc &d, int i, int j)
{
    size_t idx = size_t(j) * d.n + i;
    if (TFMT == PNDF_TEXEL_F32X2) return __ldg(reinterpret_cast<const float2 *>(d.texels) + idx);
    return __half22float2(__ldg(reinterpret_cast<const __half2 *>(d.texels) + idx));
}

struct Sampled {
    float mx, my;
    uint32_t tri, fl;
};

// The sample in FP64 throughout.
template <int TFMT>
__device__ __noinline__ Sampled sample_fp64(const MapDesc &d, const pndf_query &r, float uf1, float uf2, int kernel,
                                            float jac_eps)
{
    const double x = r.x, y = r.y, sxx = r.sxx, sxy = r.sxy, syy = r.syy;
    const double det = sxx * syy - sxy * sxy;
    Sampled o{0.f, 0.f, 0xffffffffu, 0u};
    if (!(sxx > 0.0) || !(syy > 0.0) || !(det > 0.0) || !isfinite(det) || !isfinite(x) || !isfinite(y)) {
        o.fl = PNDF_SF_INVALID;
    } else {
        const double u1 = uf1, u2 = uf2;
        double v1, v2;
        if (kernel == PNDF_KERNEL_BOX) {
            v1 = 1.5 * (2.0 * u1 - 1.0);
            v2 = 1.5 * (2.0 * u2 - 1.0);
        } else {
            const double rad = kernel == PNDF_KERNEL_DISK ? 1.5 * sqrt(u1)
                                                          : sqrt(-2.0 * log(1.0 - u1 * (1.0 - exp(-8.0))));
            double sn, cs;
            sincospi(2.0 * u2, &sn, &cs);
            v1 = rad * cs;
            v2 = rad * sn;
        }
        const double l11 = sqrt(sxx), l21 = sxy / l11, l22 = sqrt(syy - l21 * l21);
        const double ux = x + l11 * v1, uy = y + l21 * v1 + l22 * v2;
        const double fi = floor(ux), fj = floor(uy);
        if (!(fi >= 0.0 && fj >= 0.0 && fi <= d.n - 2 && fj <= d.n - 2)) {
            o.fl = PNDF_SF_OUTSIDE;
        } else {
            const int i = int(fi), j = int(fj);
            const double fu = ux - fi, fv = uy - fj;
            const int tri = fu + fv < 1.0 ? 0 : 1;
            // Tab. 1 order: (u0, u1, u2) or (u3, u2, u1), barycentric weights of u
            float2 na, nb, nc;
            double l0, lb, lc;
            if (tri == 0) {
                na = texel_s<TFMT>(d, i, j);
                nb = texel_s<TFMT>(d, i + 1, j);
                nc = texel_s<TFMT>(d, i, j + 1);
                l0 = 1.0 - fu - fv;
                lb = fu;
                lc = fv;
            } else {
                na = texel_s<TFMT>(d, i + 1, j + 1);
                nb = texel_s<TFMT>(d, i, j + 1);
                nc = texel_s<TFMT>(d, i + 1, j);
                l0 = fu + fv - 1.0;
                lb = 1.0 - fu;
                lc = 1.0 - fv;
            }
            double ax = na.x, ay = na.y, bx = nb.x, by = nb.y, cx = nc.x, cy = nc.y;
            const double cr = (bx - ax) * (cy - ay) - (by - ay) * (cx - ax);
            if (jac_eps > 0.f && fabs(cr) < double(jac_eps)) {
                const double gx = (ax + bx + cx) / 3.0, gy = (ay + by + cy) / 3.0;
                const double rho = sqrt(2.0 * double(jac_eps) / sqrt(3.0)) / sqrt(3.0);
                const double h = 0.5 * sqrt(3.0) * rho;
                ax = gx;
                ay = gy + rho;
                bx = gx - h;
                by = gy - 0.5 * rho;
                cx = gx + h;
                cy = gy - 0.5 * rho;
            }
            o.mx = float(l0 * ax + lb * bx + lc * cx);
            o.my = float(l0 * ay + lb * by + lc * cy);
            o.tri = 2u * (uint32_t(j) * uint32_t(d.n - 1) + uint32_t(i)) + uint32_t(tri);
        }
    }
    return o;
}

// Logarithm table over the mantissa's top 7 bits i.  c is near
// the reciprocal of the interval's middle (halved from i = 53 on, so that the
// reduced argument lies in [0.707, 1.414)) with 8 significant bits, so that m c -
// 1 is exact; -log c as a pair.  c = 1 at both ends, next to the argument 1.
__device__ const float4 kLog[128] = {
    {1.0f, 0.0f, 0.0f, 0.f},
    {0.98828125f, 0.0117879556f, 1.02845142e-10f, 0.f},
    {0.98046875f, 0.019724505f, 3.25610428e-10f, 0.f},
    {0.97265625f, 0.0277245473f, 7.03191227e-10f, 0.f},
    {0.96484375f, 0.035789106f, 1.81039228e-09f, 0.f},
    {0.95703125f, 0.0439192355f, -1.53307522e-09f, 0.f},
    {0.953125f, 0.0480092205f, -1.32436062e-09f, 0.f},
    {0.9453125f, 0.0562397167f, 1.61421598e-09f, 0.f},
    {0.9375f, 0.0645385236f, -2.41723086e-09f, 0.f},
    {0.9296875f, 0.0729067698f, 9.95980742e-10f, 0.f},
    {0.92578125f, 0.0771173015f, 1.82074589e-09f, 0.f},
    {0.91796875f, 0.0855919272f, 3.1646501e-09f, 0.f},
    {0.91015625f, 0.0941389874f, 3.55147711e-09f, 0.f},
    {0.90625f, 0.0984400734f, -6.17285667e-10f, 0.f},
    {0.8984375f, 0.107098132f, 3.18446469e-09f, 0.f},
    {0.890625f, 0.115831815f, 8.18796198e-10f, 0.f},
    {0.88671875f, 0.120227426f, 7.07647718e-10f, 0.f},
    {0.87890625f, 0.129077047f, -4.83446172e-09f, 0.f},
    {0.875f, 0.133531392f, 1.00388664e-09f, 0.f},
    {0.8671875f, 0.142500058f, 4.79077755e-09f, 0.f},
    {0.86328125f, 0.147014737f, 5.8325984e-09f, 0.f},
    {0.85546875f, 0.156105712f, 2.60690158e-09f, 0.f},
    {0.8515625f, 0.16068238f, 1.49104107e-09f, 0.f},
    {0.84375f, 0.169899032f, 5.27550759e-09f, 0.f},
    {0.83984375f, 0.174539417f, -6.76527445e-10f, 0.f},
    {0.83203125f, 0.183885276f, 2.45254084e-09f, 0.f},
    {0.828125f, 0.188591167f, 2.47680809e-09f, 0.f},
    {0.82421875f, 0.193319306f, 5.22594634e-09f, 0.f},
    {0.81640625f, 0.202843189f, 3.27524963e-09f, 0.f},
    {0.8125f, 0.207639366f, -1.61007641e-09f, 0.f},
    {0.80859375f, 0.212458655f, -4.02395806e-09f, 0.f},
    {0.80078125f, 0.222167462f, 3.23063487e-09f, 0.f},
    {0.796875f, 0.227057457f, -6.33486863e-09f, 0.f},
    {0.79296875f, 0.231971473f, -7.06397962e-09f, 0.f},
    {0.7890625f, 0.236909747f, -4.53605452e-11f, 0.f},
    {0.78125f, 0.246860072f, 5.91480998e-09f, 0.f},
    {0.77734375f, 0.251872629f, -9.17216081e-09f, 0.f},
    {0.7734375f, 0.256910414f, 2.81380391e-10f, 0.f},
    {0.76953125f, 0.261973709f, 6.87354706e-09f, 0.f},
    {0.765625f, 0.267062783f, 2.00777328e-09f, 0.f},
    {0.7578125f, 0.277319282f, 3.12291459e-09f, 0.f},
    {0.75390625f, 0.282487243f, 1.21607515e-08f, 0.f},
    {0.75f, 0.287682086f, -1.37775436e-08f, 0.f},
    {0.74609375f, 0.292904019f, -2.9228413e-09f, 0.f},
    {0.7421875f, 0.298153371f, 1.70025616e-09f, 0.f},
    {0.73828125f, 0.303430438f, -8.6217673e-09f, 0.f},
    {0.734375f, 0.30873549f, -8.19566282e-09f, 0.f},
    {0.73046875f, 0.314068824f, 3.57216523e-09f, 0.f},
    {0.7265625f, 0.319430768f, 2.27652364e-09f, 0.f},
    {0.72265625f, 0.324821621f, -1.77834303e-09f, 0.f},
    {0.71875f, 0.33024168f, 6.7253132e-09f, 0.f},
    {0.71484375f, 0.335691303f, -1.13766134e-08f, 0.f},
    {0.7109375f, 0.341170758f, -6.06189765e-10f, 0.f},
    {1.4140625f, -0.34646678f, 1.2362654e-08f, 0.f},
    {1.40625f, -0.340926588f, 6.11041329e-10f, 0.f},
    {1.3984375f, -0.33535555f, 8.12959744e-09f, 0.f},
    {1.390625f, -0.32975328f, -6.68649403e-09f, 0.f},
    {1.3828125f, -0.324119478f, 9.80991466e-09f, 0.f},
    {1.375f, -0.318453729f, -1.96585526e-09f, 0.f},
    {1.3671875f, -0.312755704f, -6.07781026e-09f, 0.f},
    {1.359375f, -0.307025045f, 9.86156667e-09f, 0.f},
    {1.3515625f, -0.301261336f, 5.03318143e-09f, 0.f},
    {1.34375f, -0.295464218f, 4.76897544e-09f, 0.f},
    {1.3359375f, -0.289633304f, 1.1297649e-08f, 0.f},
    {1.328125f, -0.283768177f, 3.90182597e-09f, 0.f},
    {1.3203125f, -0.27786845f, -1.31549849e-09f, 0.f},
    {1.3125f, -0.271933705f, -1.08690026e-08f, 0.f},
    {1.3125f, -0.271933705f, -1.08690026e-08f, 0.f},
    {1.3046875f, -0.265963554f, 5.88518612e-09f, 0.f},
    {1.296875f, -0.259957522f, -2.28307173e-09f, 0.f},
    {1.2890625f, -0.25391522f, 1.05180753e-08f, 0.f},
    {1.28125f, -0.247836158f, -6.22502361e-09f, 0.f},
    {1.2734375f, -0.241719931f, -5.52308554e-09f, 0.f},
    {1.2734375f, -0.241719931f, -5.52308554e-09f, 0.f},
    {1.265625f, -0.235566065f, -6.59738131e-09f, 0.f},
    {1.2578125f, -0.229374096f, -5.26730703e-09f, 0.f},
    {1.25f, -0.223143548f, -3.5408485e-09f, 0.f},
    {1.2421875f, -0.216873944f, 5.50508039e-09f, 0.f},
    {1.2421875f, -0.216873944f, 5.50508039e-09f, 0.f},
    {1.234375f, -0.210564762f, -6.75345246e-09f, 0.f},
    {1.2265625f, -0.204215541f, 5.32808485e-11f, 0.f},
    {1.21875f, -0.197825745f, 1.41819567e-09f, 0.f},
    {1.21875f, -0.197825745f, 1.41819567e-09f, 0.f},
    {1.2109375f, -0.191394851f, -2.38794273e-09f, 0.f},
    {1.203125f, -0.184922338f, -9.61968505e-10f, 0.f},
    {1.1953125f, -0.178407654f, -3.30659677e-09f, 0.f},
    {1.1953125f, -0.178407654f, -3.30659677e-09f, 0.f},
    {1.1875f, -0.171850264f, 7.1457591e-09f, 0.f},
    {1.1796875f, -0.165249571f, -1.69112169e-09f, 0.f},
    {1.1796875f, -0.165249571f, -1.69112169e-09f, 0.f},
    {1.171875f, -0.158605024f, -5.95807936e-09f, 0.f},
    {1.1640625f, -0.151916042f, -5.55889848e-11f, 0.f},
    {1.1640625f, -0.151916042f, -5.55889848e-11f, 0.f},
    {1.15625f, -0.145182014f, 3.66715991e-09f, 0.f},
    {1.1484375f, -0.138402328f, 5.03604536e-09f, 0.f},
    {1.1484375f, -0.138402328f, 5.03604536e-09f, 0.f},
    {1.140625f, -0.131576359f, 1.48328394e-09f, 0.f},
    {1.1328125f, -0.124703482f, 3.29244632e-09f, 0.f},
    {1.1328125f, -0.124703482f, 3.29244632e-09f, 0.f},
    {1.125f, -0.117783032f, -3.29869065e-09f, 0.f},
    {1.1171875f, -0.110814363f, -3.57593155e-09f, 0.f},
    {1.1171875f, -0.110814363f, -3.57593155e-09f, 0.f},
    {1.109375f, -0.103796795f, 1.32892319e-09f, 0.f},
    {1.109375f, -0.103796795f, 1.32892319e-09f, 0.f},
    {1.1015625f, -0.0967296287f, 2.28319008e-09f, 0.f},
    {1.09375f, -0.0896121562f, -2.53696197e-09f, 0.f},
    {1.09375f, -0.0896121562f, -2.53696197e-09f, 0.f},
    {1.0859375f, -0.0824436694f, 2.27287536e-10f, 0.f},
    {1.0859375f, -0.0824436694f, 2.27287536e-10f, 0.f},
    {1.078125f, -0.0752234235f, 2.30300468e-09f, 0.f},
    {1.0703125f, -0.0679506585f, -3.40831319e-09f, 0.f},
    {1.0703125f, -0.0679506585f, -3.40831319e-09f, 0.f},
    {1.0625f, -0.0606246218f, -7.90594239e-12f, 0.f},
    {1.0625f, -0.0606246218f, -7.90594239e-12f, 0.f},
    {1.0546875f, -0.0532445163f, 1.73465908e-09f, 0.f},
    {1.0546875f, -0.0532445163f, 1.73465908e-09f, 0.f},
    {1.046875f, -0.0458095372f, 1.14102328e-09f, 0.f},
    {1.0390625f, -0.038318865f, 6.99065028e-10f, 0.f},
    {1.0390625f, -0.038318865f, 6.99065028e-10f, 0.f},
    {1.03125f, -0.0307716578f, -8.42237391e-10f, 0.f},
    {1.03125f, -0.0307716578f, -8.42237391e-10f, 0.f},
    {1.0234375f, -0.0231670588f, -4.5604151e-10f, 0.f},
    {1.0234375f, -0.0231670588f, -4.5604151e-10f, 0.f},
    {1.015625f, -0.015504187f, 4.37010483e-10f, 0.f},
    {1.015625f, -0.015504187f, 4.37010483e-10f, 0.f},
    {1.0078125f, -0.00778214028f, -1.61003558e-10f, 0.f},
    {1.0078125f, -0.00778214028f, -1.61003558e-10f, 0.f},
    {1.0f, 0.0f, 0.0f, 0.f},
};

// Natural logarithm of a + e + l, a in [2^-20, 1], |e| <= 2^-25 and 0 below a = 1/2,
// |l| <= 2^-23 a: a = 2^k m, log = k ln 2 - log c + log1p(m c - 1), the last by its
// series (|m c - 1| <= 2^-7), as in the table-driven logarithm of Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic", 1990.
// e is added exactly: next to 1 the logarithm is no larger than it.
__device__ __forceinline__ Pair log_sum(float a, float e, float l)
{
    const uint32_t bits = __float_as_uint(a), i = (bits >> 16) & 127u;
    int k = int(bits >> 23) - 127;
    float m = __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
    if (i >= 53u) {
        m *= 0.5f;
        ++k;
    }
    const float4 t = __ldg(&kLog[i]);
    const float r = __fmaf_rn(m, t.x, -1.0f);
    const Pair r2 = two_prod(r, r);
    const float q = r2.h * r * fmaf(r, fmaf(r, fmaf(r, fmaf(r, 1.0f / 7.0f, -1.0f / 6.0f), 0.2f), -0.25f), 1.0f / 3.0f);
    const Pair p = two_prod(float(k), 0.693147182f);
    const Pair s0 = two_sum(p.h, t.y), s1 = two_sum(s0.h, r), s2 = two_sum(s1.h, -0.5f * r2.h), s3 = two_sum(s2.h, e);
    float lo = fmaf(float(k), -1.90465421e-09f, p.l) + t.z;
    lo += s0.l + s1.l + s2.l + s3.l - 0.5f * r2.l + q + fmaf(-0.5f * e, e, fmaf(e, 1.0f - a, l) / a);
    return quick_sum(s3.h, lo);
}

// sin and cos of 2 pi u for u in [0, 1]: an exact reduction to |f| <= 1/4 of the
// half turn, Taylor series with the leading coefficients as pairs (the sine's up to
// z^4, z = f^2: it is multiplied by f alone).
__device__ __forceinline__ void sincos_turn(float u, Pair &sn, Pair &cs)
{
    const float t = 2.0f * u, q = rintf(2.0f * t), f = __fmaf_rn(-0.5f, q, t);
    const Pair z = two_prod(f, f);
    const float t9 = z.h * fmaf(z.h, fmaf(z.h, -2.19153535e-05f, 0.000466302805f), -0.00737043098f);
    const Pair s9 = quick_sum(0.0821458846f, t9 + 1.97806404e-09f);
    Pair s = Pair{-0.599264503f, -2.67954618e-08f} + z * s9;
    s = Pair{2.55016398f, 5.55786386e-08f} + z * s;
    s = Pair{-5.16771269f, -9.16039227e-08f} + z * s;
    s = (Pair{3.14159274f, -8.74227766e-08f} + z * s) * f;
    Pair c = Pair{0.235330626f, 3.9903707e-09f} +
             z.h * fmaf(z.h, fmaf(z.h, -0.000104638105f, 0.00192957431f), -0.0258068914f);
    c = Pair{-1.33526278f, 6.56655308e-09f} + z * c;
    c = Pair{4.05871201f, 1.20801531e-07f} + z * c;
    c = Pair{-4.93480206f, -1.45185794e-07f} + z * c;
    c = z * c + 1.0f;
    const int n = int(q) & 3;
    const Pair a = n & 1 ? c : s, b = n & 1 ? s : c;
    sn = n & 2 ? -a : a;
    cs = n == 1 || n == 2 ? -b : b;
}

// Integer part (floor) of base + v, base a whole number, and the rest in [0, 1).
__device__ __forceinline__ int whole(float base, Pair v, Pair &frac)
{
    float f = floorf(v.h);
    if (f == v.h && v.l < 0.f) f -= 1.0f;
    const Pair r = two_sum(v.h, -f);  // (inexact in one FP32 number where v is negative)
    frac = quick_sum(r.h, __fadd_rn(r.l, v.l));
    return int(base) + int(f);
}

// l0 a + lb b + lc c, rounded once.
__device__ __forceinline__ float blend(Pair l0, Pair lb, Pair lc, float a, float b, float c)
{
    const Pair p0 = two_prod(l0.h, a), p1 = two_prod(lb.h, b), p2 = two_prod(lc.h, c);
    const Pair s = two_sum(p0.h, p1.h), t = two_sum(s.h, p2.h);
    const float lo = p0.l + p1.l + p2.l + s.l + t.l + fmaf(l0.l, a, fmaf(lb.l, b, lc.l * c));
    return __fadd_rn(t.h, lo);
}

__device__ __forceinline__ float third_of_sum(float a, float b, float c, float add)
{
    const Pair s = two_sum(a, b), t = two_sum(s.h, c);
    const Pair g = quick_sum(t.h, t.l + s.l) * Pair{0.333333343f, -9.93410776e-09f};
    return __fadd_rn(g.h, g.l + add);
}

// The sample in pairs; false where the record is outside their range: centres
// past 2^20, variances outside [1e-8, 2^24] (sigma 4096, where the pairs' error comes
// to 1.4e-10 of a texel with the disk and box kernels), correlation so strong that
// S_yy - l21^2 keeps less than 1e-3 of S_yy (zero, negative and infinite inputs are
// among those), normals that are not finite.
template <int TFMT>
__device__ __forceinline__ bool sample_pair(const MapDesc &d, const pndf_query &r, float u1, float u2, int kernel,
                                            float jac_eps, float rho, Sampled &o)
{
    const float cc = r.sxx * r.syy;
    if (!(fabsf(r.x) < 1048576.f && fabsf(r.y) < 1048576.f && r.sxx > 1e-8f && r.sxx <= 0x1p24f && r.syy > 1e-8f &&
          r.syy <= 0x1p24f && fmaf(-r.sxy, r.sxy, cc) > 1e-3f * cc && u1 >= 0.f && u1 <= 1.f && u2 >= 0.f && u2 <= 1.f))
        return false;
    Pair v1, v2;
    if (kernel == PNDF_KERNEL_BOX) {
        v1 = two_sum(2.0f * u1, -1.0f) * 1.5f;
        v2 = two_sum(2.0f * u2, -1.0f) * 1.5f;
    } else {
        Pair rad;
        if (kernel == PNDF_KERNEL_DISK) {
            rad = root(Pair{u1, 0.f}) * 1.5f;
        } else {  // sqrt(-2 log(1 - u1 (1 - e^-8)))
            // as (1 - u1) + u1 e^-8, which keeps its digits for u1 next to 0 and to 1
            const Pair s = two_sum(1.0f, -u1), e8 = two_prod(u1, 3.3546262e-04f), a = two_sum(s.h, e8.h);
            const Pair g = log_sum(a.h, s.l, a.l + fmaf(u1, 3.695373e-12f, e8.l));
            rad = root(Pair{-2.0f * g.h, -2.0f * g.l});
        }
        Pair sn, cs;
        sincos_turn(u2, sn, cs);
        v1 = rad * cs;
        v2 = rad * sn;
    }
    const Pair l11 = root(Pair{r.sxx, 0.f}), l21 = divide(r.sxy, l11), l22 = root(-(l21 * l21) + r.syy);
    const float bx = floorf(r.x), by = floorf(r.y);
    Pair fu, fv;
    const int i = whole(bx, l11 * v1 + (r.x - bx), fu);
    const int j = whole(by, (l21 * v1 + l22 * v2) + (r.y - by), fv);
    o = Sampled{0.f, 0.f, 0xffffffffu, 0u};
    if (i < 0 || j < 0 || i > d.n - 2 || j > d.n - 2) {
        o.fl = PNDF_SF_OUTSIDE;
        return true;
    }
    const Pair f = fu + fv;
    const int tri = f.h < 1.0f || (f.h == 1.0f && f.l < 0.f) ? 0 : 1;
    // Tab. 1 order: (u0, u1, u2) or (u3, u2, u1), barycentric weights of u
    const float2 na = texel_s<TFMT>(d, i + tri, j + tri);
    const float2 nb = texel_s<TFMT>(d, i + 1 - tri, j + tri), nc = texel_s<TFMT>(d, i + tri, j + 1 - tri);
    const Pair one{1.0f, 0.f};
    const Pair l0 = tri ? f + (-1.0f) : one - f, lb = tri ? one - fu : fu, lc = tri ? one - fv : fv;
    bool clamp = false;
    if (jac_eps > 0.f) {
        const float ax = nb.x - na.x, ay = nb.y - na.y, cx = nc.x - na.x, cy = nc.y - na.y;
        const float cr = fabsf(diff_prod(ax, cy, ay, cx));
        // FP32 differences and products: the cross is good to 2^-21 of its terms
        const float err = 0x1p-21f * fmaf(fabsf(ax), fabsf(cy), fabsf(ay) * fabsf(cx));
        clamp = cr < jac_eps;
        if (!(fabsf(cr - jac_eps) > err))
            clamp = fabs((double(nb.x) - na.x) * (double(nc.y) - na.y) - (double(nb.y) - na.y) * (double(nc.x) - na.x)) <
                    double(jac_eps);
    }
    if (clamp) {
        // the replacement's vertices are g + (0, rho), g + (-h, -rho/2), g + (h, -rho/2)
        const float h = 0.866025404f * rho;
        o.mx = third_of_sum(na.x, nb.x, nc.x, h * ((lc.h - lb.h) + (lc.l - lb.l)));
        o.my = third_of_sum(na.y, nb.y, nc.y, rho * (1.5f * (l0.h + l0.l) - 0.5f));
    } else {
        o.mx = blend(l0, lb, lc, na.x, nb.x, nc.x);
        o.my = blend(l0, lb, lc, na.y, nb.y, nc.y);
    }
    o.tri = 2u * (uint32_t(j) * uint32_t(d.n - 1) + uint32_t(i)) + uint32_t(tri);
    // (texels that are not finite or whose products are not: a pair's low part is lost with them)
    return isfinite(o.mx) && isfinite(o.my);
}

template <int TFMT>
__global__ void __launch_bounds__(256) sample_kernel(MapDesc d, const pndf_query *__restrict__ q,
                                                     const float *__restrict__ uni, int64_t n, int kernel, float jac_eps,
                                                     float rho, float *__restrict__ m_out,
                                                     uint32_t *__restrict__ tri_out, uint32_t *__restrict__ flags_out)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const pndf_query r = q[k];
        const float u1 = uni[2 * k], u2 = uni[2 * k + 1];
        Sampled o;
        if (!sample_pair<TFMT>(d, r, u1, u2, kernel, jac_eps, rho, o))
            o = sample_fp64<TFMT>(d, r, u1, u2, kernel, jac_eps);
        m_out[2 * k] = o.mx;
        m_out[2 * k + 1] = o.my;
        if (tri_out) tri_out[k] = o.tri;
        if (flags_out) flags_out[k] = o.fl;
    }
}

}  // namespace

cudaError_t launch_sample(const pndf_hierarchy *h, const pndf_query *q, const float *u, int64_t n, int kernel,
                          float jac_eps, float *m, uint32_t *tri, uint32_t *flags, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (n + 255) / 256;
    if (blocks > int64_t(sms) * 16) blocks = int64_t(sms) * 16;
    // circumradius of the Eq. 6 replacement (equilateral, area eps / 2)
    const float rho = float(sqrt(2.0 * double(jac_eps) / sqrt(3.0)) / sqrt(3.0));
    if (h->d.texel_fmt == PNDF_TEXEL_F32X2)
        sample_kernel<PNDF_TEXEL_F32X2><<<unsigned(blocks), 256, 0, s>>>(h->d, q, u, n, kernel, jac_eps, rho, m, tri,
                                                                              flags);
    else
        sample_kernel<PNDF_TEXEL_F16X2><<<unsigned(blocks), 256, 0, s>>>(h->d, q, u, n, kernel, jac_eps, rho, m, tri,
                                                                              flags);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace pndf

// Edge functions of normal-space triangles, shared by the pyramid build (which
// marks the nodes that hold near-singular triangles) and the evaluation.
#pragma once

namespace pndf {

// Kahan's difference of products a*b - c*d with one FMA correction.
__device__ __forceinline__ float diff_prod(float a, float b, float c, float d)
{
    float w = c * d;
    float e = fmaf(-c, d, w);
    float f = fmaf(a, b, -w);
    return f + e;
}

// Twice the signed area of (p, q, r): (q - p) x (r - p).
__device__ __forceinline__ float orient(float px, float py, float qx, float qy, float rx, float ry)
{
    return diff_prod(qx - px, ry - py, qy - py, rx - px);
}

__device__ __forceinline__ double orient_d(double px, double py, double qx, double qy, double rx, double ry)
{
    return (qx - px) * (ry - py) - (qy - py) * (rx - px);
}

}  // namespace pndf

// Bounds of the distance from a point to a triangle in FP32, with which the
// object grid chooses the triangles whose FP64 distance it takes.  Plain C++ as
// well, so that the bounds can be checked without a GPU.
//
// Every product and sum below is rounded as written (the units that include
// this file are compiled without contraction).
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define TRI_HD __host__ __device__ __forceinline__
#else
#define TRI_HD static inline
#endif

namespace dock {

// A triangle relative to the lattice origin: v0, the edges to v1 and v2, its
// longest edge (with a pad), the tolerance of a plane distance (infinite: no
// FP32 bound is usable) and the slack of the test that the projection falls inside.
struct TriF {
    float v0[3], e0[3], e1[3], reach, tol, slack;
    int32_t touch;
};
static_assert(sizeof(TriF) == 52, "triangle record");

// S: the lattice's extent, which bounds every coordinate of the mesh and of the
// points (relative to the origin).  eps = 2^-24.
//
// Rounding the vertices, the edges, the point and w = p - v0 moves point and
// triangle by less than 9 eps S against each other, and a distance by no more
// (it is 1-Lipschitz in both).  For the rounded triangle, distances to points of
// its edges are evaluated to within 13 eps (longest edge + |w|): the position
// along an edge is off by 4 eps (|w| + edge), the offset by a few eps of its
// terms, and no difference of nearly equal numbers enters (the third edge is
// formed from its own end points).  tri_edge_tol covers both with 1.2 to spare
// at edges and |w| of S, and an FP64 error of delta / 2 beside them.
constexpr float TRI_DELTA = 5e-7f;   // of S: about 8 eps
TRI_HD float tri_edge_tol(float S) { return 6.f * TRI_DELTA * S; }

// v: the vertices minus the origin (FP64).  cut: distances from cut on do not matter.
TRI_HD TriF tri_f32(const double v[3][3], float S, float cut, bool touch)
{
    float f[3][3];
    for (int m = 0; m < 3; ++m)
        for (int a = 0; a < 3; ++a) f[m][a] = (float)v[m][a];
    TriF r;
    float l0 = 0.f, l1 = 0.f, l2 = 0.f;
    for (int a = 0; a < 3; ++a) {
        r.v0[a] = f[0][a];
        r.e0[a] = f[1][a] - f[0][a];
        r.e1[a] = f[2][a] - f[0][a];
        const float d = f[2][a] - f[1][a];
        l0 += r.e0[a] * r.e0[a];
        l1 += r.e1[a] * r.e1[a];
        l2 += d * d;
    }
    const float n0 = r.e0[1] * r.e1[2] - r.e0[2] * r.e1[1], n1 = r.e0[2] * r.e1[0] - r.e0[0] * r.e1[2];
    const float n2 = r.e0[0] * r.e1[1] - r.e0[1] * r.e1[0];
    const float edge = sqrtf(fmaxf(l0, fmaxf(l1, l2))), area = sqrtf(n0 * n0 + n1 * n1 + n2 * n2);
    const float delta = TRI_DELTA * S, far = 2.f * cut + edge + 32.f * delta;   // far: of |w| where it matters
    const float alt = edge > 0.f ? area / edge : 0.f;   // the smallest altitude, to a few eps edge / alt of it
    r.reach = edge * 1.00001f + 4.f * delta;
    // |w . n| / |n|: n is off by 3 eps |e0||e1|, so the plane distance by 6 eps far edge / alt and 6 eps far
    r.tol = 6.f * delta + 1e-6f * far * (edge / alt);
    // u, v, u + v - den below: sums of products off by 14, 14 and 42 eps of far edge^3
    r.slack = 1.2e-6f * far * edge * edge * edge;
    // Not usable: squares or cubes near the ends of the FP32 range, an altitude
    // that is mostly rounding, or one at which the FP64 distance itself (its
    // barycentric terms cancel to 32 2^-53 (far / alt)^2) may be off by delta / 2.
    const bool sure = area >= 1e-15f && area <= 1e15f && edge * edge * edge * far <= 1e37f && alt >= 1e-5f * edge &&
                      3.6e-15f * (far / alt) * (far / alt) * edge <= 0.5f * delta;
    if (!sure) r.tol = INFINITY;
    r.touch = touch ? 1 : 0;
    return r;
}

TRI_HD float tri_clamp01(float s) { return fminf(1.f, fmaxf(0.f, s)); }

// UPPER: the distance from p to a point of the (rounded) triangle near the
// closest one, so that adding tri_edge_tol bounds the distance from above
// whatever the triangle's shape; INFINITY when it is above `skip`.
// Otherwise a lower bound of the distance, all tolerances included: from the
// edges and, unless the projection is outside by more than the slack, the plane
// (a wrong "inside" only lowers it); INFINITY when it is above `skip`.
template <bool UPPER>
TRI_HD float tri_bound_f32(const TriF &t, float px, float py, float pz, float skip, float edge_tol)
{
    const float w0 = px - t.v0[0], w1 = py - t.v0[1], w2 = pz - t.v0[2];
    const float ww = fmaf(w0, w0, fmaf(w1, w1, w2 * w2)), lim = skip + edge_tol + t.reach;
    if (ww > lim * lim) return INFINITY;
    const float *a = t.e0, *b = t.e1;
    const float aa = fmaf(a[0], a[0], fmaf(a[1], a[1], a[2] * a[2])), bb = fmaf(b[0], b[0], fmaf(b[1], b[1], b[2] * b[2]));
    const float ab = fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2]));
    const float wa = fmaf(w0, a[0], fmaf(w1, a[1], w2 * a[2])), wb = fmaf(w0, b[0], fmaf(w1, b[1], w2 * b[2]));
    const float c0 = b[0] - a[0], c1 = b[1] - a[1], c2 = b[2] - a[2];
    const float x0 = w0 - a[0], x1 = w1 - a[1], x2 = w2 - a[2];
    const float cc = fmaf(c0, c0, fmaf(c1, c1, c2 * c2)), xc = fmaf(x0, c0, fmaf(x1, c1, x2 * c2));
    // nearest points of the edges
    const float sa = aa > 0.f ? tri_clamp01(wa / aa) : 0.f, sb = bb > 0.f ? tri_clamp01(wb / bb) : 0.f;
    const float sc = cc > 0.f ? tri_clamp01(xc / cc) : 0.f;
    const float p0 = fmaf(-sa, a[0], w0), p1 = fmaf(-sa, a[1], w1), p2 = fmaf(-sa, a[2], w2);
    const float q0 = fmaf(-sb, b[0], w0), q1 = fmaf(-sb, b[1], w1), q2 = fmaf(-sb, b[2], w2);
    const float r0 = fmaf(-sc, c0, x0), r1 = fmaf(-sc, c1, x1), r2 = fmaf(-sc, c2, x2);
    float d2 = fminf(fmaf(p0, p0, fmaf(p1, p1, p2 * p2)),
                     fminf(fmaf(q0, q0, fmaf(q1, q1, q2 * q2)), fmaf(r0, r0, fmaf(r1, r1, r2 * r2))));
    // the projection is v0 + (u a + v b) / den
    const float den = fmaf(aa, bb, -ab * ab), u = fmaf(bb, wa, -ab * wb), v = fmaf(aa, wb, -ab * wa);
    if (UPPER) {
        if (den > 0.f && u >= 0.f && v >= 0.f && u + v <= den) {
            const float s = u / den, r = fminf(v / den, 1.f - s);   // in the triangle, whatever their rounding
            const float g0 = w0 - fmaf(s, a[0], r * b[0]), g1 = w1 - fmaf(s, a[1], r * b[1]);
            const float g2 = w2 - fmaf(s, a[2], r * b[2]);
            d2 = fminf(d2, fmaf(g0, g0, fmaf(g1, g1, g2 * g2)));
        }
        return sqrtf(d2);
    }
    float low = sqrtf(d2) - edge_tol;
    if (u >= -t.slack && v >= -t.slack && u + v <= den + 3.f * t.slack) {
        const float n0 = a[1] * b[2] - a[2] * b[1], n1 = a[2] * b[0] - a[0] * b[2], n2 = a[0] * b[1] - a[1] * b[0];
        const float nn = fmaf(n0, n0, fmaf(n1, n1, n2 * n2)), wn = fmaf(w0, n0, fmaf(w1, n1, w2 * n2));
        low = fminf(low, sqrtf(wn * wn / nn) - t.tol);
    }
    return low;
}

}  // namespace dock

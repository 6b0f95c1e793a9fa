// Continuous refinement (Sec. V) on the GPU.
//
// K10/K11 (k_refine_dist): distances of the probe poses of every candidate.  A
// probe pose is expressed in the object frame, the mesh BVH is walked with the
// Eq. (21) test f_p(c) < r_node + eps (eps = tau_out2, so pruned geometry
// can only have s = s' = 0), and each surviving triangle's minimum of f_p is
// found by first-order tests or by golden-section search over one barycentric
// coordinate with an inner bisection on subgradient signs (f_p is convex).  The
// block deals nodes, triangles and searches, not poses, to its threads.  From
// d*, the witness and the SDF normal (Eq. (22)-(23)) the kernel forms the exact
// sensitivities of d w.r.t. the twist (Eq. (24)-(27), rotational term through
// the left Jacobian V(w), coupling term analytic), the score s(d) of Eq. (18)
// and its derivatives, and reduces J, grad J (Eq. (28)) and the Gauss-Newton
// matrix per candidate in FP64, deterministically (per-warp partials, fixed
// order).  k_refine_ordered evaluates again the few poses whose result depends
// on the order of the walk.
// K12 (k_refine_solve): one warp per candidate, FP64: Cholesky 6x6 solve of
// the normal equations, trust-region scaling, box projection (Eq. (20)), and
// the pose data of the next iteration (Eq. (14)-(17)).
//
// 21 evaluations and 20 steps on the GB300: 8 x 200 poses 4.0 ms, 64 x 5000 poses
// on 65 k triangles 60 ms; 100 L-BFGS-B rounds of 32 x 2000 poses 36 ms.  Bound by
// the chain of a search (53 bisections of 20 steps, 156 cycles a step) while few
// poses run, by instruction issue (half of the slots), block barriers and the last
// blocks' tail at 64 x 5000.  A thread per pose, its warp waiting for the longest of
// 32 chains, takes 34, 262 to 375 and 218 ms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "dock_internal.h"

namespace cg = cooperative_groups;

namespace dock {

#define KINK_BAND 1e-3f   // distance from the medial surface within which a witness is treated as on it (mm)

// per-candidate data read by the evaluation kernel (FP32)
struct CandF {
    float R[9], p[3];   // object pose T(xi)
    float V[9];         // left Jacobian V(w)
    float Mc[9];        // d(V(w) u)/dw
    float c[3];         // pivot p0 + V u + R0 a
    float pad[3];
};

// state layout (doubles): R0[9] p0[3] a[3] xi[6] -> 21, then J at 21, pad to 24
constexpr int ST = 24;
constexpr int NACC = 28;   // J, G[6], H upper triangle [21]

// f_p of the flat-ended cylinder (tip face z = 0, body z in [0, L]) and, in g,
// the gradient of the active branch (a valid subgradient: the cap branch on
// the inside medial surface dr == dz, +x as the radial direction on the axis).
__device__ __forceinline__ float sdf_cyl(float x, float y, float z, float r, float L, float *g)
{
    float rho = sqrtf(fmaf(x, x, y * y));
    float ux = 1.f, uy = 0.f;
    if (rho > 0.f) { ux = x / rho; uy = y / rho; }
    float dr = rho - r;
    float zlo = -z, zhi = z - L;
    float dz = zlo >= zhi ? zlo : zhi;
    float cz = zlo >= zhi ? -1.f : 1.f;
    float f;
    if (dr <= 0.f && dz <= 0.f) {
        if (dr > dz) { f = dr; if (g) { g[0] = ux; g[1] = uy; g[2] = 0.f; } }
        else { f = dz; if (g) { g[0] = 0.f; g[1] = 0.f; g[2] = cz; } }
    } else if (dr > 0.f && dz > 0.f) {
        f = sqrtf(fmaf(dr, dr, dz * dz));
        if (g) { g[0] = dr * ux / f; g[1] = dr * uy / f; g[2] = dz * cz / f; }
    } else if (dr > 0.f) {
        f = dr;
        if (g) { g[0] = ux; g[1] = uy; g[2] = 0.f; }
    } else {
        f = dz;
        if (g) { g[0] = 0.f; g[1] = 0.f; g[2] = cz; }
    }
    return f;
}

// Contact normal n* (Eq. (23)): the unit gradient; where f_p is not
// differentiable (the medial surface inside, the axis) the gradient of the
// branch sdf_cyl reports (the cap on ties, +x radially on the axis).
__device__ __forceinline__ void sdf_normal(const float *x, float r, float L, float *n)
{
    float g[3];
    sdf_cyl(x[0], x[1], x[2], r, L, g);
    float gn = sqrtf(fmaf(g[0], g[0], fmaf(g[1], g[1], g[2] * g[2])));
    n[0] = g[0] / gn; n[1] = g[1] / gn; n[2] = g[2] / gn;
}

__device__ __forceinline__ float dot3f(const float *a, const float *b) { return fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2])); }

// The subgradient of f_p at the witness x (probe frame) of triangle lv that
// gives the derivative of d = min over the triangle of f_p (Sec. V-B,
// Eq. (22)-(24)): the gradient where f_p is differentiable; on the medial
// surface inside the probe, the combination lam a + (1 - lam) b of the
// radial and cap gradients whose component along the witness's face (the
// triangle's plane, or its edge when a barycentric weight is ~0) vanishes,
// the element the minimum over the triangle selects (Danskin); a vertex lies
// on the medial surface only by coincidence, so at a vertex witness the
// gradient of the active branch (sdf_normal).  Not normalised.
__device__ __noinline__ void witness_subgradient(const float *x, const float lv[3][3], float r, float L, float *n)
{
    const float rho = sqrtf(fmaf(x[0], x[0], x[1] * x[1]));
    const float dr = rho - r, zlo = -x[2], zhi = x[2] - L;
    const float dz = zlo >= zhi ? zlo : zhi;
    if (!(dr <= 0.f && dz <= 0.f && fabsf(dr - dz) <= KINK_BAND && rho > 0.f)) {
        sdf_normal(x, r, L, n);
        return;
    }
    float e1[3], e2[3], p[3];
    for (int i = 0; i < 3; ++i) { e1[i] = lv[1][i] - lv[0][i]; e2[i] = lv[2][i] - lv[0][i]; p[i] = x[i] - lv[0][i]; }
    const float d00 = dot3f(e1, e1), d01 = dot3f(e1, e2), d11 = dot3f(e2, e2), d20 = dot3f(p, e1), d21 = dot3f(p, e2);
    const float den = fmaf(d00, d11, -d01 * d01);
    float w[3];
    w[1] = den != 0.f ? fmaf(d11, d20, -d01 * d21) / den : 0.f;
    w[2] = den != 0.f ? fmaf(d00, d21, -d01 * d20) / den : 0.f;
    w[0] = 1.f - w[1] - w[2];
    int nz = 0, zi = -1;
    for (int k = 0; k < 3; ++k)
        if (w[k] <= 1e-4f) { ++nz; zi = k; }
    if (nz >= 2 || den == 0.f) {
        sdf_normal(x, r, L, n);
        return;
    }
    const float a[3] = {x[0] / rho, x[1] / rho, 0.f}, b[3] = {0.f, 0.f, zlo >= zhi ? -1.f : 1.f};
    float Pa[3], Pb[3];
    if (nz == 0) {
        const float nu[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
        const float nn = dot3f(nu, nu), an = dot3f(a, nu) / nn, bn = dot3f(b, nu) / nn;
        for (int i = 0; i < 3; ++i) { Pa[i] = a[i] - an * nu[i]; Pb[i] = b[i] - bn * nu[i]; }
    } else {
        const float *pp = lv[(zi + 1) % 3], *qq = lv[(zi + 2) % 3];
        const float e[3] = {qq[0] - pp[0], qq[1] - pp[1], qq[2] - pp[2]};
        const float ee = dot3f(e, e), ae = dot3f(a, e) / ee, be = dot3f(b, e) / ee;
        for (int i = 0; i < 3; ++i) { Pa[i] = ae * e[i]; Pb[i] = be * e[i]; }
    }
    const float df[3] = {Pa[0] - Pb[0], Pa[1] - Pb[1], Pa[2] - Pb[2]};
    const float dd = dot3f(df, df);
    const float lm = dd > 0.f ? fminf(1.f, fmaxf(0.f, -dot3f(Pb, df) / dd)) : 0.5f;
    for (int i = 0; i < 3; ++i) n[i] = fmaf(lm, a[i], (1.f - lm) * b[i]);
}

// A number with the sign of g . e, g the subgradient sdf_cyl reports at
// (x, y, z) (same branch rules), without normalising g: the bisections need
// only the sign of the directional derivative.  The three cases are selected,
// not branched to: the lanes of a warp meet all of them, and a bisection step
// is the longest chain of the refinement.
__device__ __forceinline__ float sdf_slope_sign(float x, float y, float z, float r, float L, const float *e)
{
    const float r2 = fmaf(x, x, y * y);
    const float ri = r2 > 0.f ? rsqrtf(r2) : 0.f;
    const float rho = r2 * ri;
    const float se = r2 > 0.f ? fmaf(x, e[0], y * e[1]) : e[0];   // rho (u . e_xy), u = +x on the axis
    const float dr = rho - r, zlo = -z, zhi = z - L;
    const bool lo = zlo >= zhi;
    const float dz = lo ? zlo : zhi;
    const float ce = lo ? -e[2] : e[2];                            // cz e_z
    const float corner = fmaf(dr * se, r2 > 0.f ? ri : 1.f, dz * ce);
    return (dr > 0.f && dz > 0.f) ? corner : (dr > dz ? se : ce);
}

// f_p is differentiable at x: everywhere outside the probe; inside, away
// (by more than 1e-3 mm) from the medial surfaces where two branches meet
// and from the axis.
__device__ __forceinline__ bool sdf_smooth_at(const float *x, float r, float L)
{
    float rho = sqrtf(fmaf(x[0], x[0], x[1] * x[1]));
    float dr = rho - r, zlo = -x[2], zhi = x[2] - L;
    float dz = fmaxf(zlo, zhi);
    if (dr > 0.f || dz > 0.f) return true;
    const float band = 1e-3f;
    return fabsf(dr - dz) > band && fabsf(zlo - zhi) > band && rho > band;
}

// The inner minimisation of the per-triangle search: min over v in [0, 1-u] of
// f(v0 + u e1 + v e2) by bisection on df/dv (a subgradient sign; the same steps
// for every call, so lanes that search together stay converged; an end minimum
// is approached to 2^-iters of the segment).  Returns f there, v in *v_out and
// the point in x.
//
// G = 1, 4 or 16 lanes share one search (the group's lanes hold the same
// operands; for G > 1 all 32 lanes call, idle groups with any triangle: a vote
// over part of a warp would split it for good).  A bisection step is one chain of about 25 dependent operations,
// so a warp with few searches waits, not computes: G = 4 evaluates both
// possible next midpoints beside the current one and takes 2 steps per round,
// G = 16 takes 4 (the 15 midpoints a depth-4 tree of decisions can reach).
// Every midpoint is formed by the same halvings as step by step, so the
// decisions, and with them the result, are the same bits for every G.
template <int G>
__device__ __forceinline__ float inner_min(const float *v0, const float *e1, const float *e2, float u, float r, float L,
                                           int iters, float *v_out, float *x)
{
    const float vmax = fmaxf(0.f, 1.f - u);
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = fmaf(u, e1[a], v0[a]);
    float lo = 0.f, hi = vmax;
    if (G == 1) {
#pragma unroll 1
        for (int k = 0; k < iters; ++k) {
            const float mid = 0.5f * (lo + hi);
            const bool neg = sdf_slope_sign(fmaf(mid, e2[0], x[0]), fmaf(mid, e2[1], x[1]), fmaf(mid, e2[2], x[2]), r, L,
                                            e2) < 0.f;
            lo = neg ? mid : lo;
            hi = neg ? hi : mid;
        }
    } else {
        constexpr int D = G == 16 ? 4 : 2;                 // steps per round
        const int lane = threadIdx.x & 31, g = lane & (G - 1), sh = lane & ~(G - 1);
        const int node = g + 1 < G ? g + 1 : 1;            // heap index of the lane's midpoint (the last lane idles)
        const int dep = 31 - __clz(node);
#pragma unroll 1
        for (int k = 0; k < iters; k += D) {
            float l = lo, h = hi;
#pragma unroll
            for (int t = D - 2; t >= 0; --t)
                if (t < dep) {
                    const float m = 0.5f * (l + h);
                    const bool right = (node >> t) & 1;
                    l = right ? m : l;
                    h = right ? h : m;
                }
            const float mid = 0.5f * (l + h);
            const bool neg = sdf_slope_sign(fmaf(mid, e2[0], x[0]), fmaf(mid, e2[1], x[1]), fmaf(mid, e2[2], x[2]), r, L,
                                            e2) < 0.f;
            const unsigned bits = __ballot_sync(0xFFFFFFFFu, neg) >> sh;
            int at = 1;
#pragma unroll
            for (int t = 0; t < D; ++t)
                if (k + t < iters) {
                    const float m = 0.5f * (lo + hi);
                    const bool right = (bits >> (at - 1)) & 1u;
                    lo = right ? m : lo;
                    hi = right ? hi : m;
                    at = 2 * at + (right ? 1 : 0);
                }
        }
    }
    const float v = 0.5f * (lo + hi);
#pragma unroll
    for (int a = 0; a < 3; ++a) x[a] = fmaf(v, e2[a], x[a]);
    *v_out = v;
    return sdf_cyl(x[0], x[1], x[2], r, L, nullptr);
}

// Minimum of f_p over a triangle (local coordinates).  First-order tests at its
// vertices and on its edges settle most triangles; for the rest, a
// golden-section search on phi(u) (values only: robust on the non-smooth
// medial surface), then, for a minimum outside the probe (f is C^1 there), a
// bisection on dphi/du inside a bracket that stays outside: value-based search
// locates a smooth minimum only to ~sqrt(FP32 eps), the slope to ~eps.

// A vertex where f is differentiable and no edge from it descends is the
// minimum (f convex: f(y) >= f(x) + g.(y - x) >= f(x) on the triangle).  This
// settles most triangles, which are small against the probe; fv holds f at the
// three vertices.
__device__ __forceinline__ bool vertex_minimum(const float lv[3][3], const float *fv, float r, float L, float *d,
                                               float *uo, float *vo)
{
    int ms = 0;
    if (fv[1] < fv[ms]) ms = 1;
    if (fv[2] < fv[ms]) ms = 2;
    const float *x = lv[0];
    if (ms == 1) x = lv[1];
    if (ms == 2) x = lv[2];
    const float xm[3] = {x[0], x[1], x[2]};
    if (!sdf_smooth_at(xm, r, L)) return false;
    float g[3];
    sdf_cyl(xm[0], xm[1], xm[2], r, L, g);
    bool opt = true;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const float e[3] = {lv[m][0] - xm[0], lv[m][1] - xm[1], lv[m][2] - xm[2]};
        if (m != ms && dot3f(g, e) < 0.f) opt = false;
    }
    if (!opt) return false;
    *uo = ms == 1 ? 1.f : 0.f;
    *vo = ms == 2 ? 1.f : 0.f;
    *d = ms == 0 ? fv[0] : (ms == 1 ? fv[1] : fv[2]);
    return true;
}

// A point of edge pa-pb that minimises f along the edge, where f is
// differentiable and the direction to the opposite vertex po does not descend,
// is the minimum over the triangle (same argument: the triangle lies in the
// cone of +-edge and that direction).  Typical for a line contact with the
// probe's side.  s: position on the edge.
__device__ __forceinline__ bool edge_minimum(const float *pa, const float *pb, const float *po, float r, float L,
                                             float *d, float *so)
{
    const float e[3] = {pb[0] - pa[0], pb[1] - pa[1], pb[2] - pa[2]};
    if (sdf_slope_sign(pa[0], pa[1], pa[2], r, L, e) >= 0.f) return false;   // f grows along the edge from pa
    if (sdf_slope_sign(pb[0], pb[1], pb[2], r, L, e) <= 0.f) return false;   // f falls all the way to pb
    float lo = 0.f, hi = 1.f;
#pragma unroll 1
    for (int it = 0; it < 24; ++it) {
        const float mid = 0.5f * (lo + hi);
        const bool neg = sdf_slope_sign(fmaf(mid, e[0], pa[0]), fmaf(mid, e[1], pa[1]), fmaf(mid, e[2], pa[2]), r, L,
                                        e) < 0.f;
        lo = neg ? mid : lo;
        hi = neg ? hi : mid;
    }
    const float s = 0.5f * (lo + hi);
    float x[3], gx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) x[c] = fmaf(s, e[c], pa[c]);
    if (!sdf_smooth_at(x, r, L)) return false;
    const float fx = sdf_cyl(x[0], x[1], x[2], r, L, gx);
    const float eo[3] = {po[0] - x[0], po[1] - x[1], po[2] - x[2]};
    if (dot3f(gx, eo) < 0.f) return false;
    *d = fx;
    *so = s;
    return true;
}

// barycentric (u, v) of x = (1 - u - v) v0 + u v1 + v v2 at position s of edge k (from vertex k to k + 1)
__device__ __forceinline__ void edge_bary(int k, float s, float *u, float *v)
{
    if (k == 0) { *u = s; *v = 0.f; }
    else if (k == 1) { *u = 1.f - s; *v = s; }
    else { *u = 0.f; *v = 1.f - s; }
}

// The first-order tests in order: the vertices, then edge 0, 1, 2.
__device__ bool tri_min_shortcut(const float lv[3][3], const float *fv, float r, float L, float *d, float *uo,
                                 float *vo)
{
    if (vertex_minimum(lv, fv, r, L, d, uo, vo)) return true;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        float s;
        if (edge_minimum(lv[k], lv[(k + 1) % 3], lv[(k + 2) % 3], r, L, d, &s)) {
            edge_bary(k, s, uo, vo);
            return true;
        }
    }
    return false;
}

// Minimum of f over the triangle by golden-section search on the first
// barycentric coordinate with an inner bisection (for triangles the
// first-order tests do not settle), by the G lanes of a group together.
template <int G>
__device__ __noinline__ float3 tri_min_search(float3 p0, float3 p1, float3 p2, float r, float L, int iters)
{
    const float v0[3] = {p0.x, p0.y, p0.z};
    const float e1[3] = {p1.x - p0.x, p1.y - p0.y, p1.z - p0.z};
    const float e2[3] = {p2.x - p0.x, p2.y - p0.y, p2.z - p0.z};
    // (G > 1: decisions that lead to more evaluations are taken by the warp)
    auto some = [](bool b) -> bool { return G == 1 ? b : __any_sync(0xFFFFFFFFu, b) != 0; };
    float xt[3];
    const float ig = 0.6180339887498949f;
    float a = 0.f, b = 1.f, vc, vd;
    float c = b - ig * (b - a), d = a + ig * (b - a);
    float fc = inner_min<G>(v0, e1, e2, c, r, L, iters, &vc, xt);
    float fd = inner_min<G>(v0, e1, e2, d, r, L, iters, &vd, xt);
    int steps = iters + iters / 2;
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
        // one evaluation per step on every path
        const bool left = fc <= fd;
        if (left) { b = d; d = c; fd = fc; vd = vc; }
        else { a = c; c = d; fc = fd; vc = vd; }
        const float xn = left ? b - ig * (b - a) : a + ig * (b - a);
        float vn;
        const float fn = inner_min<G>(v0, e1, e2, xn, r, L, iters, &vn, xt);
        if (left) { c = xn; fc = fn; vc = vn; }
        else { d = xn; fd = fn; vd = vn; }
    }
    float u = fc <= fd ? c : d, v = fc <= fd ? vc : vd, best = fc <= fd ? fc : fd;
    // u = 0 and u = 1 (there v is 0: the segment has no length)
    float vu0;
    const float f0 = inner_min<G>(v0, e1, e2, 0.f, r, L, iters, &vu0, xt);
#pragma unroll
    for (int k = 0; k < 3; ++k) xt[k] = fmaf(0.f, e2[k], fmaf(1.f, e1[k], v0[k]));
    const float f1 = sdf_cyl(xt[0], xt[1], xt[2], r, L, nullptr);
    if (f0 < best) { best = f0; u = 0.f; v = vu0; }
    if (f1 < best) { best = f1; u = 1.f; v = 0.f; }
    const float le = sqrtf(dot3f(e1, e1));
    const bool polish = best > 1e-4f && le > 0.f;
    if (some(polish)) {
        // dphi/du at u for the partial minimum phi(u) = min_v f(v0 + u e1 + v e2)
        // (Danskin; valid where f is differentiable at the inner minimiser)
        auto outer_slope = [&](float uu) -> float {
            float vv, x[3], g[3];
            inner_min<G>(v0, e1, e2, uu, r, L, iters, &vv, x);
            sdf_cyl(x[0], x[1], x[2], r, L, g);
            float s = dot3f(g, e1);
            if (vv >= 1.f - uu && vv > 0.f) s -= dot3f(g, e2);
            return s;
        };
        const float w = fminf(2e-3f, 0.5f * best / le);
        float lo = fmaxf(0.f, u - w), hi = fminf(1.f, u + w);
        const bool at_lo = outer_slope(lo) >= 0.f;
        bool at_hi = false;
        if (some(polish && !at_lo)) at_hi = outer_slope(hi) <= 0.f;
        const bool inside = !at_lo && !at_hi;
        if (at_lo) hi = lo;
        else if (at_hi) lo = hi;
        if (some(polish && inside)) {
#pragma unroll 1
            for (int k = 0; k < 16; ++k) {
                const float mid = 0.5f * (lo + hi);
                const bool neg = outer_slope(mid) < 0.f;
                if (inside) {
                    lo = neg ? mid : lo;
                    hi = neg ? hi : mid;
                }
            }
        }
        const float up = 0.5f * (lo + hi);
        float vp;
        const float fp = inner_min<G>(v0, e1, e2, up, r, L, iters, &vp, xt);
        if (polish && fp <= best) { best = fp; u = up; v = vp; }
    }
    return make_float3(best, u, v);
}

// Lower bound of min f over the triangle: the linearisation at the centroid
// with a subgradient there (f is convex).  Its rounding decides which of the
// triangles that share a lowest vertex a query settles, so it is written out:
// the offsets lv - c from the unrounded centroid, one rounding each.
__device__ __forceinline__ float lin_lower_bound(const float lv[3][3], float r, float L)
{
    const float third = 1.f / 3.f;
    float s[3], c[3], g[3];
    for (int a = 0; a < 3; ++a) {
        s[a] = __fadd_rn(__fadd_rn(lv[0][a], lv[1][a]), lv[2][a]);
        c[a] = __fmul_rn(s[a], third);
    }
    const float fc = sdf_cyl(c[0], c[1], c[2], r, L, g);
    float m = INFINITY;
    for (int k = 0; k < 3; ++k) {
        float d[3];
        for (int a = 0; a < 3; ++a) d[a] = fmaf(-s[a], third, lv[k][a]);
        m = fminf(m, dot3f(g, d));
    }
    return __fadd_rn(fc, m);
}

// A tighter lower bound of f over the triangle, and a point of the triangle
// where f is close to it: the minimum of max(l_r, l_z), l_r = u . (x, y) - r
// with u the radial direction at the centroid (rho >= u . (x, y) for every unit
// u) and l_z the nearer cap plane; f >= both everywhere.  The minimum lies at a
// vertex or where an edge crosses l_r = l_z.  Exact up to the curvature of the
// probe over the triangle, where the linearisation above misses the second
// branch: it leaves about one search per pose instead of three.  Valid up to
// rounding (the caller prunes with its margin).
__device__ __forceinline__ float two_plane_bound(const float lv[3][3], float r, float L, float *pt)
{
    const float cx = (lv[0][0] + lv[1][0]) + lv[2][0], cy = (lv[0][1] + lv[1][1]) + lv[2][1];
    const float zs = (lv[0][2] + lv[1][2]) + lv[2][2];
    const float r2 = fmaf(cx, cx, cy * cy), ri = r2 > 0.f ? rsqrtf(r2) : 0.f;
    // (a factor a little below one keeps l_r below rho whatever the rounding of u)
    const float ux = cx * ri * 0.9999995f, uy = cy * ri * 0.9999995f;
    const bool low = -zs >= zs - 3.f * L;
    float lr[3], lz[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lr[k] = fmaf(ux, lv[k][0], uy * lv[k][1]) - r;
        lz[k] = low ? -lv[k][2] : lv[k][2] - L;
    }
    float best = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float m = fmaxf(lr[k], lz[k]);
        if (m < best) {
            best = m;
            pt[0] = lv[k][0]; pt[1] = lv[k][1]; pt[2] = lv[k][2];
        }
        const int n = (k + 1) % 3;
        const float da = lr[k] - lz[k], db = lr[n] - lz[n];
        if (da * db < 0.f) {
            const float t = da / (da - db);
            const float at = fmaf(t, lz[n] - lz[k], lz[k]);
            if (at < best) {
                best = at;
#pragma unroll
                for (int c = 0; c < 3; ++c) pt[c] = fmaf(t, lv[n][c] - lv[k][c], lv[k][c]);
            }
        }
    }
    return best;
}

// Eq. (18): s(d), s'(d), s''(d) with r = tau_in / tau_out and C^1 coefficients
__device__ __forceinline__ void score3(const RefineDev &D, float d, float *s, float *s1, float *s2)
{
    float it = 1.f / D.tau_out;
    float t = d * it;
    if (t > 1.f) { *s = 0.f; *s1 = 0.f; *s2 = 0.f; }
    else if (t > 0.f) {
        float cs = cospif(0.5f * t), sn = sinpif(0.5f * t);
        *s = cs * cs;
        *s1 = -3.14159265358979f * cs * sn * it;
        *s2 = -0.5f * 9.8696044010893586f * cospif(t) * it * it;
    } else if (t > -D.rr) {
        *s = fmaf(D.A * t, t * t, D.B * t * t) + 1.f;
        *s1 = (3.f * D.A * t * t + 2.f * D.B * t) * it;
        *s2 = (6.f * D.A * t + 2.f * D.B) * it * it;
    } else {
        *s = D.k_slope * (t + D.rr);
        *s1 = D.k_slope * it;
        *s2 = 0.f;
    }
}

// f_p at a bounding-sphere centre c (object frame) for the probe frame (A, b).
__device__ __forceinline__ float node_sdf(const float *A, const float *bvec, const float4 &c, float r, float L)
{
    float q[3] = {c.x - bvec[0], c.y - bvec[1], c.z - bvec[2]};
    float loc[3];
    for (int k = 0; k < 3; ++k) loc[k] = fmaf(A[0 * 3 + k], q[0], fmaf(A[1 * 3 + k], q[1], A[2 * 3 + k] * q[2]));
    return sdf_cyl(loc[0], loc[1], loc[2], r, L, nullptr);
}

// One triangle of a BVH leaf: its bounding sphere, its vertices and its index
// in the mesh, in leaf order (one 64-byte record instead of four dependent
// look-ups: leaf order -> triangle -> vertex indices -> vertices).
struct LeafRec {
    float4 sph;
    float v[9];
    int32_t tri;
    float pad[2];
};
static_assert(sizeof(LeafRec) == 64, "leaf record");

size_t leaf_bytes() { return sizeof(LeafRec); }

// A BVH node on the device: its sphere, its children (left and left + 1, or
// -1; a leaf's first slot and count), and a slab: the node's vertices lie in
// [lo, hi] along the unit normal n, measured from the centre.
struct NodeRec {
    float4 sph;
    int32_t left, first, count;
    float hi;
    float4 n_lo;
};
static_assert(sizeof(NodeRec) == 48, "node record");

size_t node_bytes() { return sizeof(NodeRec); }

// Bounding sphere of points given one by one (FP64, every operation rounded as
// written): the centre of their box, the largest distance with a small pad.
struct BoxD {
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    __device__ __forceinline__ void add(const double *v)
    {
        for (int a = 0; a < 3; ++a) { lo[a] = fmin(lo[a], v[a]); hi[a] = fmax(hi[a], v[a]); }
    }
    __device__ __forceinline__ double mid(int a) const { return 0.5 * (lo[a] + hi[a]); }
};
__device__ __forceinline__ double dist2_exact(const double *v, const double *c)
{
    const double dx = v[0] - c[0], dy = v[1] - c[1], dz = v[2] - c[2];
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}
__device__ __forceinline__ float padded_radius(double d2)
{
    return (float)__dadd_rn(__dmul_rn(sqrt(d2), 1.0 + 1e-6), 1e-6);
}

__global__ void k_leaf_records(int n, const double *V, const int32_t *T, const int32_t *order, LeafRec *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int t = order[i];
    LeafRec r;
    BoxD box;
    const double *v[3];
    for (int m = 0; m < 3; ++m) {
        v[m] = V + 3 * (size_t)T[3 * t + m];
        box.add(v[m]);
        for (int a = 0; a < 3; ++a) r.v[3 * m + a] = (float)v[m][a];
    }
    const double c[3] = {box.mid(0), box.mid(1), box.mid(2)};
    double d2 = 0.0;
    for (int m = 0; m < 3; ++m) d2 = fmax(d2, dist2_exact(v[m], c));
    r.sph = make_float4((float)c[0], (float)c[1], (float)c[2], padded_radius(d2));
    r.tri = t;
    r.pad[0] = r.pad[1] = 0.f;
    out[i] = r;
}

cudaError_t launch_leaf_records(int n, const double *V, const int32_t *T, const int32_t *order, LeafRec *out,
                                cudaStream_t st)
{
    k_leaf_records<<<(n + 127) / 128, 128, 0, st>>>(n, V, T, order, out);
    return cudaGetLastError();
}

// The value all threads of the group (a warp, or a block of NT threads) agree on.
template <int NT, class X, class Op> __device__ __forceinline__ X group_all(X x, Op op, X *buf)
{
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
    if (NT > 32) {
        __syncthreads();
        if ((threadIdx.x & 31) == 0) buf[threadIdx.x / 32] = x;
        __syncthreads();
        x = buf[0];
        for (int k = 1; k < NT / 32; ++k) x = op(x, buf[k]);
    }
    return x;
}

// NT threads per node (32: a warp, four nodes a block; 1024: a block, for the
// few nodes of thousands of triangles) over its triangles: box and sphere from
// the FP64 vertices, then the slab along the area-weighted normal.
template <int NT>
__global__ void __launch_bounds__(NT == 32 ? 128 : NT)
k_node_records(int n, const int32_t *which, const BvhNode *in, const double *V, const int32_t *T, const int32_t *order,
               const LeafRec *leaf, NodeRec *out)
{
    __shared__ double buf[NT == 32 ? 1 : NT / 32];
    const int g = NT == 32 ? (blockIdx.x * blockDim.x + threadIdx.x) / 32 : blockIdx.x, lane = threadIdx.x % NT;
    if (g >= n) return;
    const int i = which ? which[g] : g;
    const BvhNode nd = in[i];
    auto mn = [](double a, double b) { return fmin(a, b); };
    auto mx = [](double a, double b) { return fmax(a, b); };
    auto sum = [](double a, double b) { return a + b; };
    BoxD box;
    double s[3] = {0.0, 0.0, 0.0};
    for (int k = lane; k < nd.count; k += NT) {
        const int t = order[nd.first + k];
        for (int m = 0; m < 3; ++m) box.add(V + 3 * (size_t)T[3 * t + m]);
        const float *v = leaf[nd.first + k].v;
        const float a[3] = {v[3] - v[0], v[4] - v[1], v[5] - v[2]}, b[3] = {v[6] - v[0], v[7] - v[1], v[8] - v[2]};
        s[0] += (double)(a[1] * b[2] - a[2] * b[1]);
        s[1] += (double)(a[2] * b[0] - a[0] * b[2]);
        s[2] += (double)(a[0] * b[1] - a[1] * b[0]);
    }
    double c[3];
    for (int a = 0; a < 3; ++a) {
        box.lo[a] = group_all<NT>(box.lo[a], mn, buf);
        box.hi[a] = group_all<NT>(box.hi[a], mx, buf);
        s[a] = group_all<NT>(s[a], sum, buf);
        c[a] = box.mid(a);
    }
    const double q = sqrt(s[0] * s[0] + s[1] * s[1] + s[2] * s[2]);
    const bool flat = q > 0.0 && q < 1e300;
    const float nrm[3] = {flat ? (float)(s[0] / q) : 1.f, flat ? (float)(s[1] / q) : 0.f, flat ? (float)(s[2] / q) : 0.f};
    const float cf[3] = {(float)c[0], (float)c[1], (float)c[2]};
    double d2 = 0.0, lo = 1e300, hi = -1e300, far = 0.0;
    for (int k = lane; k < nd.count; k += NT) {
        const int t = order[nd.first + k];
        const float *vf = leaf[nd.first + k].v;
        for (int m = 0; m < 3; ++m) {
            d2 = fmax(d2, dist2_exact(V + 3 * (size_t)T[3 * t + m], c));
            const float d[3] = {vf[3 * m] - cf[0], vf[3 * m + 1] - cf[1], vf[3 * m + 2] - cf[2]};
            const double h = (double)fmaf(d[0], nrm[0], fmaf(d[1], nrm[1], d[2] * nrm[2]));
            lo = fmin(lo, h);
            hi = fmax(hi, h);
            far = fmax(far, (double)fmaxf(fabsf(vf[3 * m]), fmaxf(fabsf(vf[3 * m + 1]), fabsf(vf[3 * m + 2]))));
        }
    }
    d2 = group_all<NT>(d2, mx, buf);
    lo = group_all<NT>(lo, mn, buf);
    hi = group_all<NT>(hi, mx, buf);
    far = group_all<NT>(far, mx, buf);
    if (lane == 0) {
        NodeRec r;
        const float rad = padded_radius(d2);
        const float pad = 1e-6f * ((float)far + rad);   // the rounding of the heights and of the unit length
        r.sph = make_float4(cf[0], cf[1], cf[2], rad);
        r.left = nd.left;
        r.first = nd.first;
        r.count = nd.left < 0 ? nd.count : 0;
        r.hi = (float)hi + pad;
        r.n_lo = make_float4(nrm[0], nrm[1], nrm[2], (float)lo - pad);
        out[i] = r;
    }
}

cudaError_t launch_node_records(int n, int n_big, const int32_t *big, const BvhNode *in, const double *V,
                                const int32_t *T, const int32_t *order, const LeafRec *leaf, NodeRec *out,
                                cudaStream_t st)
{
    if (n_big > 0)
        k_node_records<1024><<<n_big, 1024, 0, st>>>(n_big, big, in, V, T, order, leaf, out);
    k_node_records<32><<<(n - n_big + 3) / 4, 128, 0, st>>>(n - n_big, big + n_big, in, V, T, order, leaf, out);
    return cudaGetLastError();
}

// f_p at a node's centre, and a lower bound of f_p over its triangles: f is
// convex, so f(x) >= f(c) + g . (x - c) with g the gradient at c, and x - c has
// its component along the slab's normal in [lo, hi] and the rest within the
// radius.  Where the probe's face lies along the surface the sphere alone lets
// through every triangle below the face (100 triangles and 80 nodes a pose at
// 65 k triangles); the slab leaves those next to the contact.
__device__ __forceinline__ float node_bounds(const NodeRec *nd, const float *fr, float r, float L, float4 *sph,
                                             int4 *ch, float *lower)
{
    const float4 *p = reinterpret_cast<const float4 *>(nd);
    const float4 s = __ldg(p), nl = __ldg(p + 2);
    const int4 c = __ldg(reinterpret_cast<const int4 *>(p + 1));
    const float q[3] = {s.x - fr[9], s.y - fr[10], s.z - fr[11]};
    float loc[3], g[3], ln[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        loc[k] = fmaf(fr[k], q[0], fmaf(fr[3 + k], q[1], fr[6 + k] * q[2]));
        ln[k] = fmaf(fr[k], nl.x, fmaf(fr[3 + k], nl.y, fr[6 + k] * nl.z));
    }
    const float f = sdf_cyl(loc[0], loc[1], loc[2], r, L, g);
    const float gn = dot3f(g, ln);
    const float side = sqrtf(fmaxf(0.f, fmaf(-gn, gn, 1.000002f)));
    *lower = fmaxf(f - s.w, f + fminf(gn * nl.w, gn * __int_as_float(c.w)) - side * s.w);
    *sph = s;
    *ch = c;
    return f;
}

// A float as an unsigned integer of the same order, and back.
__device__ __forceinline__ uint32_t ord_f(float f)
{
    const uint32_t u = __float_as_uint(f);
    return u ^ ((u >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float unord_f(uint32_t k)
{
    return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xFFFFFFFFu));
}

// ---------------------------------------------------------------------------
// Distance queries of Q probe poses of one candidate per block of 128 threads.
//
// Work items, not poses, are dealt to the threads.  A pose needs about 60
// sphere tests, 50 triangle tests, 8 first-order tests and 1 to 3 searches, in
// numbers that differ from pose to pose; with one thread per pose a warp took
// the longest of its 32 chains, and the searches (about 50 bisections of 20
// steps each, 80 us) ran with a few lanes active: 2 to 7 million cycles per
// warp, up to 135 million where one pose met many unsettled triangles.  Here
// the block keeps the items of all its poses in shared-memory queues:
//   nodes      (pose, BVH node whose children are to be tested under Eq. (21),
//              f_p(c) < r_node + eps); taken from the top, so the walk stays
//              depth first and the stack short
//   triangles  (pose, leaf slot): sphere test, vertices, linearised bound
//   candidates (pose, leaf slot, lower bound): first-order tests, then the
//              searches of what they leave unsettled: every pose's lowest
//              bound first, then what that did not rule out, with 16, 4 or 1
//              lanes per search, as many as the queue leaves free
// A pose's upper bound of d* (smallest vertex value, sphere and search results)
// and its best (d, triangle) are shared-memory words updated by atomicMin, so
// the result does not depend on the order of the items: the smallest d, the
// lowest triangle index among equals.  Every bound prunes with a margin `mg`
// above the rounding of the values compared (where f_p is linear over a
// triangle its linearised bound is its smallest vertex value up to rounding).
// hint (the leaf slot and barycentric point of the pose's witness at the
// previous evaluation): f_p at that point of the mesh bounds d* from the start
// without a search.
// ---------------------------------------------------------------------------
template <int Q> struct DistCfg {
    static constexpr int NT = 128;
    static constexpr int NCAP = 704, RES = 64;    // node stack; reserve for a depth-first descent
    static constexpr int TCAP = NT + 8 * NT;      // <= 127 left over + two leaves of 4 per popped node
    static constexpr int CCAP = Q < 32 ? 768 : 2048;   // a second settling costs two more rounds of searches
    static constexpr int CL = Q < 32 ? 32 / Q : 1;   // CTAs whose poses share one warp's partial sum
    static constexpr int ROWS = Q < 32 ? 32 : Q;
    static_assert(Q <= NT && Q <= 128 && CCAP > NT && CCAP <= 65535, "queue sizes");
};

template <int Q> struct DistSmem {
    using C = DistCfg<Q>;
    unsigned long long best[Q];    // (ordered d) << 32 | triangle, over every candidate
    unsigned long long sbest[Q];   // the same over the strict ones (bound not above their own vertices)
    unsigned long long first[Q];   // lowest bound among the unsettled: (ordered bound) << 32 | candidate
    float fr[Q][13];               // A[9], b[3], prune margin
    uint32_t lim[Q];               // ordered upper bound of d*
    int wslot[Q];                  // leaf slot and barycentric point of the best so far
    float wu[Q], wv[Q];            // (of the strict best)
    union {
        struct {
            int nnode[C::NCAP];
            int tslot[C::TCAP];
        };
        float rec[9][C::ROWS];     // (once the queues are empty) s, s', s'', g (6) per pose for the partial sums
    };
    int cslot[C::CCAP];
    float clb[C::CCAP];
    unsigned short open[C::CCAP], l1[Q], l2[C::CCAP];
    unsigned char nq[C::NCAP], tq[C::TCAP], cq[C::CCAP];   // pose of an entry (cq: bit 7 = strict)
    int hslot[Q];                  // leaf slot of the hint (queued at once), or -1
    unsigned char edge[C::NT];     // an edge test's outcome: 0 failed, 1 passed, 2 not run
    int redo[C::ROWS / 32];        // 32 poses whose evaluation is handed to k_refine_ordered
    int n_node, n_tri, n_cand, n_open, n_1, n_2;
};

__device__ __forceinline__ void leaf_local(const LeafRec *rec, int slot, const float *fr, float lv[3][3], int *tri)
{
    const float4 *p = reinterpret_cast<const float4 *>(rec + slot);
    const float4 b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3);
    const float v[9] = {b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, d.x};
    *tri = __float_as_int(d.y);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const float q0 = v[3 * m] - fr[9], q1 = v[3 * m + 1] - fr[10], q2 = v[3 * m + 2] - fr[11];
#pragma unroll
        for (int a = 0; a < 3; ++a) lv[m][a] = fmaf(fr[a], q0, fmaf(fr[3 + a], q1, fr[6 + a] * q2));
    }
}

// A settled candidate's minimum into its pose's bounds; returns its key (~0: nothing to take).
template <int Q>
__device__ __forceinline__ unsigned long long offer(DistSmem<Q> &S, int q, int strict, float dk, int tri)
{
    if (!(dk < INFINITY)) return ~0ull;
    const uint32_t o = ord_f(dk + 0.f);
    const unsigned long long key = ((unsigned long long)o << 32) | (uint32_t)tri;
    atomicMin(&S.best[q], key);
    if (strict) atomicMin(&S.sbest[q], key);
    atomicMin(&S.lim[q], o);
    return key;
}

// (after a barrier) the candidate whose key is its pose's strict best leaves its point
template <int Q>
__device__ __forceinline__ void keep_point(DistSmem<Q> &S, int q, int strict, unsigned long long key, int slot, float u,
                                           float v)
{
    if (strict && key != ~0ull && S.sbest[q] == key) {
        S.wslot[q] = slot;
        S.wu[q] = u;
        S.wv[q] = v;
    }
}

// Candidate i's bound lies above what its pose has already.
template <int Q> __device__ __forceinline__ bool ruled_out(DistSmem<Q> &S, int i, int q)
{
    return S.clb[i] > unord_f(*(volatile uint32_t *)&S.lim[q]) + S.fr[q][12];
}

// The searches of candidates l[0..n) of the queue by groups of G lanes.
template <int Q, int G>
__device__ __forceinline__ void run_searches(DistSmem<Q> &S, const RefineDev &D, const unsigned short *l, int n)
{
    constexpr int NT = DistCfg<Q>::NT;
    const int tid = threadIdx.x, g = tid & (G - 1);
    for (int base = 0; base < n; base += NT / G) {
        const int k = base + tid / G;
        unsigned long long key = ~0ull;
        int q = 0, slot = 0;
        float3 res = make_float3(0.f, 0.f, 0.f);
        bool run = k < n;
        int i = 0, strict = 0;
        if (run) {
            i = l[k];
            q = S.cq[i] & 127;
            strict = S.cq[i] >> 7;
            run = !ruled_out(S, i, q);
        }
        // one decision for the group (the bound may fall while its lanes read it)
        if (G > 1) run = __shfl_sync(0xFFFFFFFFu, run ? 1 : 0, (tid & 31) & ~(G - 1)) != 0;
        if (G == 1 ? run : __any_sync(0xFFFFFFFFu, run) != 0) {
            float lv[3][3] = {};
            int t = 0;
            if (run) {
                slot = S.cslot[i];
                leaf_local(D.leaf, slot, S.fr[q], lv, &t);
            }
            res = tri_min_search<G>(make_float3(lv[0][0], lv[0][1], lv[0][2]), make_float3(lv[1][0], lv[1][1], lv[1][2]),
                                    make_float3(lv[2][0], lv[2][1], lv[2][2]), D.r, D.L, D.tri_iters);
            if (run && g == 0) key = offer(S, q, strict, res.x, t);
        }
        __syncthreads();
        keep_point(S, q, strict, key, slot, res.y, res.z);
    }
    __syncthreads();
}

template <int Q>
__device__ __forceinline__ void run_list(DistSmem<Q> &S, const RefineDev &D, const unsigned short *l, int n)
{
    constexpr int NT = DistCfg<Q>::NT;
    if (n <= 0) return;
    if (n * 16 <= NT) run_searches<Q, 16>(S, D, l, n);
    else if (n * 4 <= NT) run_searches<Q, 4>(S, D, l, n);
    else run_searches<Q, 1>(S, D, l, n);
}

// Settles the queued candidates: first-order tests, then searches.  Called by
// the whole block; leaves the queue empty.  The tests at the vertices come
// first, for all; the edge tests of what they leave (three bisections of 24
// steps) are dealt to three threads each.
template <int Q>
__device__ __noinline__ void resolve_candidates(DistSmem<Q> &S, const RefineDev &D, int nc)
{
    constexpr int NT = DistCfg<Q>::NT;
    const int tid = threadIdx.x;
    if (tid == 0) S.n_open = S.n_1 = S.n_2 = 0;
    for (int q = tid; q < Q; q += NT) S.first[q] = ~0ull;
    __syncthreads();
    for (int base = 0; base < nc; base += NT) {
        const int i = base + tid;
        unsigned long long key = ~0ull;
        int q = 0, slot = 0, strict = 0;
        float u = 0.f, v = 0.f;
        if (i < nc) {
            q = S.cq[i] & 127;
            strict = S.cq[i] >> 7;
            if (!ruled_out(S, i, q)) {
                float lv[3][3], fv[3], dk;
                int t;
                slot = S.cslot[i];
                leaf_local(D.leaf, slot, S.fr[q], lv, &t);
                for (int m = 0; m < 3; ++m) fv[m] = sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr);
                if (vertex_minimum(lv, fv, D.r, D.L, &dk, &u, &v)) key = offer(S, q, strict, dk, t);
                else S.open[atomicAdd(&S.n_open, 1)] = (unsigned short)i;
            }
        }
        __syncthreads();
        keep_point(S, q, strict, key, slot, u, v);
    }
    __syncthreads();
    const int no = S.n_open;
    for (int base = 0; base < no; base += NT / 3) {
        // thread 3 j + k: edge k of candidate j
        const int j = tid / 3, k = tid - 3 * j;
        const bool on = j < NT / 3 && base + j < no;
        const int i = on ? S.open[base + j] : 0, q = S.cq[i] & 127, strict = S.cq[i] >> 7, slot = S.cslot[i];
        float d = INFINITY, sk = 0.f;
        int t = 0;
        bool ok = false;
        const bool run = on && !ruled_out(S, i, q);
        if (run) {
            float lv[3][3];
            leaf_local(D.leaf, slot, S.fr[q], lv, &t);
            const float pa[3] = {k == 0 ? lv[0][0] : k == 1 ? lv[1][0] : lv[2][0],
                                 k == 0 ? lv[0][1] : k == 1 ? lv[1][1] : lv[2][1],
                                 k == 0 ? lv[0][2] : k == 1 ? lv[1][2] : lv[2][2]};
            const float pb[3] = {k == 0 ? lv[1][0] : k == 1 ? lv[2][0] : lv[0][0],
                                 k == 0 ? lv[1][1] : k == 1 ? lv[2][1] : lv[0][1],
                                 k == 0 ? lv[1][2] : k == 1 ? lv[2][2] : lv[0][2]};
            const float po[3] = {k == 0 ? lv[2][0] : k == 1 ? lv[0][0] : lv[1][0],
                                 k == 0 ? lv[2][1] : k == 1 ? lv[0][1] : lv[1][1],
                                 k == 0 ? lv[2][2] : k == 1 ? lv[0][2] : lv[1][2]};
            ok = edge_minimum(pa, pb, po, D.r, D.L, &d, &sk);
        }
        S.edge[tid] = ok ? 1 : run ? 0 : 2;
        __syncthreads();
        // the first edge that passes settles the triangle; none: a search
        unsigned long long key = ~0ull;
        float u = 0.f, v = 0.f;
        if (on) {
            const bool lower = (k > 0 && S.edge[3 * j] == 1) || (k > 1 && S.edge[3 * j + 1] == 1);
            if (ok && !lower) {
                edge_bary(k, sk, &u, &v);
                key = offer(S, q, strict, d, t);
            }
            // (a bound that fell in between may have stopped some of the three)
            if (k == 0 && S.edge[3 * j] == 0 && S.edge[3 * j + 1] == 0 && S.edge[3 * j + 2] == 0) {
                S.l2[atomicAdd(&S.n_2, 1)] = (unsigned short)i;
                atomicMin(&S.first[q], ((unsigned long long)ord_f(S.clb[i]) << 32) | (uint32_t)i);
            }
        }
        __syncthreads();
        keep_point(S, q, strict, key, slot, u, v);
    }
    __syncthreads();
    // searches: the lowest bound of every pose
    const int ns = S.n_2;
    for (int k = tid; k < ns; k += NT) {
        const int i = S.l2[k];
        if ((uint32_t)S.first[S.cq[i] & 127] == (uint32_t)i) S.l1[atomicAdd(&S.n_1, 1)] = (unsigned short)i;
    }
    if (tid == 0) S.n_open = 0;
    __syncthreads();
    run_list<Q>(S, D, S.l1, S.n_1);
    // what that left
    for (int k = tid; k < ns; k += NT) {
        const int i = S.l2[k], q = S.cq[i] & 127;
        if ((uint32_t)S.first[q] != (uint32_t)i && !ruled_out(S, i, q))
            S.open[atomicAdd(&S.n_open, 1)] = (unsigned short)i;
    }
    __syncthreads();
    run_list<Q>(S, D, S.open, S.n_open);
    if (tid == 0) S.n_cand = 0;
    __syncthreads();
}

// Sum over the 32 lanes of each of 32 values; lane k returns the sum of value
// k.  The tree is that of shuffling down by 16, 8, 4, 2, 1 (value by value),
// with the values dealt out on the way: 31 additions instead of 160, and FP64
// additions issue at a sixteenth of the FP32 rate.
__device__ __forceinline__ double warp_sum_32(double *a)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const double keep = up ? a[k + o] : a[k], give = up ? a[k] : a[k + o];
            a[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
    }
    return a[0];
}

// A witness as the next evaluation's hint: leaf slot, barycentric (u, v) in 16 bits each.
__device__ __forceinline__ int2 pack_hint(int slot, float u, float v)
{
    const uint32_t uu = (uint32_t)(fminf(fmaxf(u, 0.f), 1.f) * 65535.f + 0.5f);
    const uint32_t vv = (uint32_t)(fminf(fmaxf(v, 0.f), 1.f) * 65535.f + 0.5f);
    return make_int2(slot, (int)(uu | (vv << 16)));
}

// The probe pose in the object frame: A = R^T R_i (fr[0..9)), b = R^T (t_i - p)
// (fr[9..12)); a mesh point m maps to probe-local A^T (m - b).
__device__ __forceinline__ void pose_frame_in_object(const CandF &cf, const PoseRec &pr, float *fr)
{
    for (int a = 0; a < 3; ++a)
        for (int k = 0; k < 3; ++k)
            fr[a * 3 + k] = fmaf(cf.R[0 * 3 + a], pr.Rf[0 * 3 + k], fmaf(cf.R[1 * 3 + a], pr.Rf[1 * 3 + k], cf.R[2 * 3 + a] * pr.Rf[2 * 3 + k]));
    const float tp[3] = {pr.tf[0] - cf.p[0], pr.tf[1] - cf.p[1], pr.tf[2] - cf.p[2]};
    for (int a = 0; a < 3; ++a) fr[9 + a] = fmaf(cf.R[0 * 3 + a], tp[0], fmaf(cf.R[1 * 3 + a], tp[1], cf.R[2 * 3 + a] * tp[2]));
}

// What one pose adds to its candidate's sums.
struct PoseTerms {
    float s = -0.f, s1 = 0.f, s2 = 0.f;   // Eq. (18) (-0: the sum adds -s)
    float g[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // dd/dxi
};

// Score, sensitivities (and, when asked for, distance, witness and normal at
// index o) of a pose whose minimum d is at the local point xl of triangle lv.
template <bool GRAD>
__device__ __forceinline__ void pose_terms(const RefineDev &D, const CandF &cf, const PoseRec &pr, bool hit, float d,
                                           const float *xl, const float lv[3][3], size_t o, float *dist_out,
                                           float *wit_out, float *nrm_out, PoseTerms &out)
{
    float n[3] = {0.f, 0.f, 0.f}, w[3] = {0.f, 0.f, 0.f};
    if (hit) {
        float nl[3];
        witness_subgradient(xl, lv, D.r, D.L, nl);
        for (int a = 0; a < 3; ++a) {
            n[a] = fmaf(pr.Rf[a * 3 + 0], nl[0], fmaf(pr.Rf[a * 3 + 1], nl[1], pr.Rf[a * 3 + 2] * nl[2]));
            w[a] = fmaf(pr.Rf[a * 3 + 0], xl[0], fmaf(pr.Rf[a * 3 + 1], xl[1], fmaf(pr.Rf[a * 3 + 2], xl[2], pr.tf[a])));
        }
    }
    if (dist_out) {
        dist_out[o] = d;
        for (int a = 0; a < 3; ++a) { wit_out[3 * o + a] = w[a]; nrm_out[3 * o + a] = n[a]; }
    }
    if (hit) {
        score3(D, d, &out.s, &out.s1, &out.s2);
        if (GRAD && (out.s1 != 0.f || out.s2 != 0.f)) {
            float *g = out.g;
            for (int j = 0; j < 3; ++j) g[j] = fmaf(cf.V[0 * 3 + j], n[0], fmaf(cf.V[1 * 3 + j], n[1], cf.V[2 * 3 + j] * n[2]));
            float wc[3] = {w[0] - cf.c[0], w[1] - cf.c[1], w[2] - cf.c[2]};
            float tq[3] = {wc[1] * n[2] - wc[2] * n[1], wc[2] * n[0] - wc[0] * n[2], wc[0] * n[1] - wc[1] * n[0]};
            for (int j = 0; j < 3; ++j) {
                float a1 = fmaf(cf.V[0 * 3 + j], tq[0], fmaf(cf.V[1 * 3 + j], tq[1], cf.V[2 * 3 + j] * tq[2]));
                float a2 = fmaf(cf.Mc[0 * 3 + j], n[0], fmaf(cf.Mc[1 * 3 + j], n[1], cf.Mc[2 * 3 + j] * n[2]));
                g[3 + j] = a1 + a2;
            }
        }
    }
}

// The warp's 32 poses' terms summed in a fixed order into partial w of candidate c.
template <bool GRAD>
__device__ __forceinline__ void write_partial(const PoseTerms &o, double *acc_part, int c, int nwarp, int w)
{
    double acc[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) acc[k] = 0.0;
    acc[0] = -(double)o.s;
    if (GRAD && (o.s1 != 0.f || o.s2 != 0.f)) {
        double g[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) g[j] = (double)o.g[j];
#pragma unroll
        for (int j = 0; j < 6; ++j) acc[1 + j] = -(double)o.s1 * g[j];
        const double wgt = o.s2 < 0.f ? -(double)o.s2 : 0.0;
        int k = 7;
#pragma unroll
        for (int a = 0; a < 6; ++a)
#pragma unroll
            for (int b = a; b < 6; ++b) acc[k++] = wgt * g[a] * g[b];
    }
    const double sum = warp_sum_32(acc);
    const int lane = threadIdx.x & 31;
    if (lane < NACC) acc_part[((size_t)c * nwarp + w) * NACC + lane] = sum;
}

// Distances, scores, sensitivities and partial sums of Q poses per block,
// blockDim 128.  acc_part[(c * nwarp + w) * NACC + k]: the sums over poses
// [32 w, 32 w + 32) of candidate c, which belongs to request grp[c] (Dt[0]
// when grp is null); warps past a request's pose count leave zeros, so a
// candidate's sums do not depend on the other requests of the launch.
template <int Q, bool GRAD>
__global__ void __launch_bounds__(128, 5)
k_refine_dist(const RefineDev *Dt, const int32_t *grp, const CandF *cands, double *acc_part, int nwarp, float *dist_out,
              float *wit_out, float *nrm_out, int2 *hints, const int32_t *active, int32_t *redo_list)
{
    using C = DistCfg<Q>;
    constexpr int NT = C::NT;
    __shared__ __align__(16) unsigned char smem[sizeof(DistSmem<Q>)];
    DistSmem<Q> &S = *reinterpret_cast<DistSmem<Q> *>(smem);
    const int c = blockIdx.y, i0 = blockIdx.x * Q, tid = threadIdx.x;
    if (active && !active[c]) return;   // a finished candidate (its partials are not read); uniform over a cluster
    const RefineDev D = Dt[grp ? grp[c] : 0];
    const CandF &cf = cands[c];
    const float eps = D.tau_out;
    int2 *hp = hints ? hints + (size_t)c * nwarp * 32 + i0 : nullptr;
    if (tid == 0) S.n_node = S.n_tri = S.n_cand = 0;
    if (tid < C::ROWS / 32) S.redo[tid] = 0;
    // (a cluster's CTAs have all started before one writes into another's shared memory)
    if constexpr (C::CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    if (tid < Q) {
        S.best[tid] = S.sbest[tid] = ~0ull;
        S.hslot[tid] = -1;
        float ub = INFINITY;
        if (i0 + tid < D.P) {
            const PoseRec &pr = D.poses[i0 + tid];
            float *A = S.fr[tid];
            pose_frame_in_object(cf, pr, A);
            const float mg = 2e-6f * (D.r + D.L + fabsf(A[9]) + fabsf(A[10]) + fabsf(A[11]));
            A[12] = mg;
            const int2 h = hp ? hp[tid] : make_int2(-1, 0);
            if (h.x >= 0) {
                const float4 sph = __ldg(&D.leaf[h.x].sph);
                if (node_sdf(A, A + 9, sph, D.r, D.L) < sph.w + eps) {
                    float lv[3][3];
                    int t;
                    leaf_local(D.leaf, h.x, A, lv, &t);
                    float pt[3];
                    const int k = atomicAdd(&S.n_cand, 1);
                    S.hslot[tid] = S.cslot[k] = h.x;
                    S.cq[k] = (unsigned char)(tid | 128);   // (the ordered walk settles it first)
                    S.clb[k] = two_plane_bound(lv, D.r, D.L, pt);
                    for (int m = 0; m < 3; ++m) ub = fminf(ub, sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr));
                    const float u = (float)(h.y & 0xFFFF) * (1.f / 65535.f);
                    const float v = fminf((float)((uint32_t)h.y >> 16) * (1.f / 65535.f), 1.f - u), w = 1.f - u - v;
                    float x[3];
                    for (int a = 0; a < 3; ++a) x[a] = fmaf(w, lv[0][a], fmaf(u, lv[1][a], v * lv[2][a]));
                    ub = fminf(ub, sdf_cyl(x[0], x[1], x[2], D.r, D.L, nullptr) + mg);
                }
            }
            float4 rt;
            int4 ch;
            float low;
            const float fc = node_bounds(D.nodes, A, D.r, D.L, &rt, &ch, &low);
            if (h.x < 0 && fc < rt.w + eps) {
                // no hint: the leaf reached by taking the nearer child bounds d*
                int4 at = ch;
#pragma unroll 1
                while (at.x >= 0) {
                    float4 sl, sr;
                    int4 cl, cr;
                    float bl, br;
                    node_bounds(D.nodes + at.x, A, D.r, D.L, &sl, &cl, &bl);
                    node_bounds(D.nodes + at.x + 1, A, D.r, D.L, &sr, &cr, &br);
                    at = bl <= br ? cl : cr;
                }
                for (int m = 0; m < at.z; ++m) {
                    const float4 sph = __ldg(&D.leaf[at.y + m].sph);
                    float lv[3][3], pt[3];
                    int t;
                    leaf_local(D.leaf, at.y + m, A, lv, &t);
                    two_plane_bound(lv, D.r, D.L, pt);
                    // (only what passes Eq. (21) may bound the others)
                    if (node_sdf(A, A + 9, sph, D.r, D.L) < sph.w + eps)
                        ub = fminf(ub, sdf_cyl(pt[0], pt[1], pt[2], D.r, D.L, nullptr) + mg);
                }
                if (!(ub < eps)) ub = INFINITY;
            }
            if (fc < rt.w + eps && !(low > ub + mg)) {   // Eq. (21)
                if (ch.x >= 0) {
                    const int k = atomicAdd(&S.n_node, 1);
                    S.nnode[k] = ch.x;
                    S.nq[k] = (unsigned char)tid;
                } else {
                    const int k = atomicAdd(&S.n_tri, ch.z);
                    for (int m = 0; m < ch.z; ++m) {
                        S.tslot[k + m] = ch.y + m;
                        S.tq[k + m] = (unsigned char)tid;
                    }
                }
            }
        }
        S.lim[tid] = ord_f(ub);
    }
#pragma unroll 1
    for (;;) {
        __syncthreads();
        const int ns = S.n_node, nt = S.n_tri, nc = S.n_cand;   // block-uniform
        if (nc > C::CCAP - NT) {
            resolve_candidates<Q>(S, D, nc);
            continue;
        }
        if (nt >= NT || (ns == 0 && nt > 0)) {
            const int n = min(nt, NT);
            const bool on = tid < n;
            const int slot = on ? S.tslot[nt - 1 - tid] : 0, q = on ? S.tq[nt - 1 - tid] : 0;
            __syncthreads();
            if (tid == 0) S.n_tri = nt - n;
            if (on) {
                const float *fr = S.fr[q];
                const float mg = fr[12];
                const float4 sph = __ldg(&D.leaf[slot].sph);
                const float ft = node_sdf(fr, fr + 9, sph, D.r, D.L);
                const float lim = unord_f(*(volatile uint32_t *)&S.lim[q]);
                if (ft < sph.w + eps && !(ft - sph.w > lim + mg)) {   // Eq. (21)
                    float lv[3][3], own = INFINITY;
                    int t;
                    leaf_local(D.leaf, slot, fr, lv, &t);
                    for (int m = 0; m < 3; ++m)
                        own = fminf(own, sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr));
                    if (own < lim) atomicMin(&S.lim[q], ord_f(own));
                    const float lbt = lin_lower_bound(lv, D.r, D.L);
                    if (slot != S.hslot[q] && !(lbt > fminf(own, lim) + mg)) {
                        float pt[3];
                        const float lb2 = two_plane_bound(lv, D.r, D.L, pt);
                        if (!(lb2 > fminf(own, lim) + mg)) {
                            const float at = sdf_cyl(pt[0], pt[1], pt[2], D.r, D.L, nullptr) + mg;
                            if (at < fminf(own, lim)) atomicMin(&S.lim[q], ord_f(at));
                            const int k = atomicAdd(&S.n_cand, 1);
                            S.cslot[k] = slot;
                            S.cq[k] = (unsigned char)(q | (lbt > own ? 0 : 128));
                            S.clb[k] = fmaxf(lbt, lb2);
                        }
                    }
                }
            }
        } else if (ns > 0) {
            // at most two nodes come back for each one taken: near the end of
            // the stack only the top one is taken (a plain descent, at most
            // one more entry per level)
            const int n = max(1, min(min(ns, NT), C::NCAP - C::RES - ns));
            const bool on = tid < n;
            const int left = on ? S.nnode[ns - 1 - tid] : 0, q = on ? S.nq[ns - 1 - tid] : 0;
            __syncthreads();
            if (tid == 0) S.n_node = ns - n;
            __syncthreads();
            if (on) {
                const float *fr = S.fr[q];
                const float mg = fr[12];
                const float lim = unord_f(*(volatile uint32_t *)&S.lim[q]);
                float4 sl, sr;
                int4 cl, cr;
                float bl, br;
                const float fl = node_bounds(D.nodes + left, fr, D.r, D.L, &sl, &cl, &bl);
                const float fr_ = node_bounds(D.nodes + left + 1, fr, D.r, D.L, &sr, &cr, &br);
                const bool nl = fl < sl.w + eps && !(bl > lim + mg);   // Eq. (21)
                const bool nr = fr_ < sr.w + eps && !(br > lim + mg);
                // a sphere that reaches the mesh bounds d* from above (used
                // below eps only: then the point that attains it is in a
                // triangle that passes Eq. (21))
                float ub = INFINITY;
                if (nl) ub = fl + sl.w + mg;
                if (nr) ub = fminf(ub, fr_ + sr.w + mg);
                if (ub < eps && ub < lim) atomicMin(&S.lim[q], ord_f(ub));
                const int pl = nl && cl.x >= 0, pr = nr && cr.x >= 0;
                if (pl + pr) {
                    int k = atomicAdd(&S.n_node, pl + pr);
                    const bool lf = bl <= br;   // the nearer child on top
                    if (pl && !(pr && lf)) { S.nnode[k] = cl.x; S.nq[k++] = (unsigned char)q; }
                    if (pr) { S.nnode[k] = cr.x; S.nq[k++] = (unsigned char)q; }
                    if (pl && pr && lf) { S.nnode[k] = cl.x; S.nq[k++] = (unsigned char)q; }
                }
                const int tl = (nl && cl.x < 0) ? cl.z : 0, tr = (nr && cr.x < 0) ? cr.z : 0;
                if (tl + tr) {
                    int k = atomicAdd(&S.n_tri, tl + tr);
                    for (int m = 0; m < tl; ++m, ++k) { S.tslot[k] = cl.y + m; S.tq[k] = (unsigned char)q; }
                    for (int m = 0; m < tr; ++m, ++k) { S.tslot[k] = cr.y + m; S.tq[k] = (unsigned char)q; }
                }
            }
        } else {
            break;
        }
    }
    if (S.n_cand > 0) resolve_candidates<Q>(S, D, S.n_cand);   // (its last barrier makes the winners visible)

    // ---- scores, sensitivities and partial sums ------------------------------
    const int rank = C::CL > 1 ? (int)(blockIdx.x % C::CL) : 0;
    DistSmem<Q> *S0 = &S;   // the CTA that sums
    if constexpr (C::CL > 1) S0 = cg::this_cluster().map_shared_rank(&S, 0);
    // (rec lies over the first CTA's queues: it has emptied them too)
    if constexpr (C::CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    int2 newhint = make_int2(-1, 0);
    const bool mine = tid < Q && i0 + tid < D.P;
    if (tid < Q) {
        const int i = i0 + tid, row = rank * Q + tid;
        PoseTerms o;
        if (mine) {
            const unsigned long long key = S.sbest[tid], all = S.best[tid];
            // the strict candidates hold the smallest d, none of the bounds met
            // can have hidden the one that does, and the smallest value found
            // lies at the bound that ruled the others out: on triangles of many
            // millimetres a search may end 1e-4 above a point that gave the bound
            const float dall = all != ~0ull ? unord_f((uint32_t)(all >> 32)) : INFINITY, lim = unord_f(S.lim[tid]);
            bool hidden = (dall <= eps && (uint32_t)(key >> 32) != (uint32_t)(all >> 32)) ||
                          (lim <= eps && dall > lim + 0.5f * S.fr[tid][12]);
            const bool hit = key != ~0ull;
            float lv[3][3], xl[3] = {0.f, 0.f, 0.f};
            if (hit) {
                int t;
                leaf_local(D.leaf, S.wslot[tid], S.fr[tid], lv, &t);
                const float u = S.wu[tid], v = S.wv[tid], w0 = 1.f - u - v;
                for (int a = 0; a < 3; ++a) xl[a] = fmaf(w0, lv[0][a], fmaf(u, lv[1][a], v * lv[2][a]));
                newhint = pack_hint(S.wslot[tid], u, v);
                if (dall <= eps && S.wslot[tid] != S.hslot[tid] && lin_lower_bound(lv, D.r, D.L) > lim)
                    hidden = true;
            }
            // (beyond the cutoff the score is zero; where the distance itself is asked for, it is that of
            // the triangles its shared walk meets)
            if (hidden || (dist_out && !(dall <= eps))) S0->redo[row / 32] = 1;
            pose_terms<GRAD>(D, cf, D.poses[i], hit, hit ? unord_f((uint32_t)(key >> 32)) : INFINITY, xl, lv,
                             (size_t)c * D.P + i, dist_out, wit_out, nrm_out, o);
        }
        S0->rec[0][row] = o.s;
        if (GRAD) {
            S0->rec[1][row] = o.s1;
            S0->rec[2][row] = o.s2;
            for (int j = 0; j < 6; ++j) S0->rec[3 + j][row] = o.g[j];
        }
    }
    if constexpr (C::CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    const bool redo = S0->redo[(rank * Q + min(tid, Q - 1)) / 32] != 0;
    if (hp && mine && !redo) hp[tid] = newhint;   // (k_refine_ordered starts from the old hints)
    if constexpr (C::CL > 1) cg::this_cluster().sync();   // the flag is read before its CTA leaves
    if (rank == 0 && tid < C::ROWS) {
        PoseTerms o;
        o.s = S.rec[0][tid];
        if (GRAD) {
            o.s1 = S.rec[1][tid];
            o.s2 = S.rec[2][tid];
            for (int j = 0; j < 6; ++j) o.g[j] = S.rec[3 + j][tid];
        }
        const int w = (i0 + tid) / 32;
        write_partial<GRAD>(o, acc_part, c, nwarp, w);
        if ((tid & 31) == 0 && S.redo[tid / 32]) redo_list[1 + atomicAdd(redo_list, 1)] = c * nwarp + w;
    }
}

// ---------------------------------------------------------------------------
// Poses evaluated again in the order of a shared walk.
//
// A candidate triangle is left out when its linearised bound lies above the
// best value met so far, and at a vertex contact the bound of every triangle
// around the vertex can exceed the vertex's own value by its rounding (one pose
// in 1e5 at a contact of a flat face).  What is then reported, the next best
// triangle or none, depends on the order of the walk.  k_refine_dist sees these
// cases (the smallest d belongs to a triangle its own bound rules out, or lies
// above the bound that ruled out others) and lists their 32 poses.  Beyond the cutoff, too, what is reported is the nearest
// of the triangles that the walk met on behalf of any of the 32 poses and that
// pass the pose's own Eq. (21) test: dock_distances, which returns it, lists
// those groups as well.  Here one warp walks for 32 poses together, entering a
// node when any lane needs it, the nearer child (by the smallest bound over the
// lanes) first, and settles a lane's triangles in the order of their bounds.
// The list is short (about 5 of 10000 warps on a first evaluation of 64 x 5000
// poses, fewer afterwards), so this path is written for its order, not speed.
// ---------------------------------------------------------------------------
struct OrderedBest {
    float d = INFINITY, u = 0.f, v = 0.f;
    int slot = -1, tri = -1;
};

__device__ __forceinline__ void ordered_take(OrderedBest &b, float dk, float u, float v, int slot, int tri)
{
    if (dk < b.d || (dk == b.d && tri < b.tri)) {
        b.d = dk;
        b.u = u;
        b.v = v;
        b.slot = slot;
        b.tri = tri;
    }
}

// The searches of the lanes that need one, by the whole warp: 16 lanes to a
// search while there are one or two of them, 4 while there are up to eight.
template <int G>
__device__ __forceinline__ float3 warp_search_g(const RefineDev &D, bool need, unsigned who, const float lv[3][3])
{
    const int lane = threadIdx.x & 31, grp = lane / G;
    float3 mine = make_float3(INFINITY, 0.f, 0.f);
    const int n = __popc(who), rank = __popc(who & ((1u << lane) - 1u));
#pragma unroll 1
    for (int base = 0; base < n; base += 32 / G) {
        const int src = base + grp < n ? (int)__fns(who, 0, base + grp + 1) : 0;
        float v[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) v[k] = __shfl_sync(0xFFFFFFFFu, lv[k / 3][k % 3], src);
        const float3 r = tri_min_search<G>(make_float3(v[0], v[1], v[2]), make_float3(v[3], v[4], v[5]),
                                           make_float3(v[6], v[7], v[8]), D.r, D.L, D.tri_iters);
        const bool take = need && rank >= base && rank < base + 32 / G;
        const int from = take ? (rank - base) * G : 0;
        const float3 got = make_float3(__shfl_sync(0xFFFFFFFFu, r.x, from), __shfl_sync(0xFFFFFFFFu, r.y, from),
                                       __shfl_sync(0xFFFFFFFFu, r.z, from));
        if (take) mine = got;
    }
    return mine;
}

__device__ __noinline__ float3 warp_search(const RefineDev &D, bool need, const float lv[3][3])
{
    const unsigned who = __ballot_sync(0xFFFFFFFFu, need);
    const int n = __popc(who);
    if (n == 0) return make_float3(INFINITY, 0.f, 0.f);
    if (n <= 2) return warp_search_g<16>(D, need, who, lv);
    if (n <= 8) return warp_search_g<4>(D, need, who, lv);
    float3 r = make_float3(INFINITY, 0.f, 0.f);
    if (need)
        r = tri_min_search<1>(make_float3(lv[0][0], lv[0][1], lv[0][2]), make_float3(lv[1][0], lv[1][1], lv[1][2]),
                              make_float3(lv[2][0], lv[2][1], lv[2][2]), D.r, D.L, D.tri_iters);
    __syncwarp();
    return r;
}

__device__ __noinline__ void ordered_query(const RefineDev &D, const float *fr, bool valid, int hint, OrderedBest &B)
{
    constexpr int QC = 16, QN = 6;   // triangles a lane keeps for after the walk; searches it keeps for after those
    int sn[64], ct[QC], qt[QN];
    float sl[64], cl[QC], ql[QN];
    int nc = 0, nq = 0;
    const float eps = D.tau_out;
    float UB = valid ? INFINITY : -INFINITY;   // a lane without a pose needs nothing
    int seeded = -1;
    // the lanes with `on` settle a triangle each: first-order tests, then a
    // search now or (may_defer) later; called by the whole warp
    auto settle = [&](bool on, int slot, float lb, bool may_defer) {
        float lv[3][3] = {}, fv[3], u = 0.f, v = 0.f, dk = INFINITY;
        int t = -1;
        bool need = false;
        if (on) {
            leaf_local(D.leaf, slot, fr, lv, &t);
            for (int m = 0; m < 3; ++m) fv[m] = sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr);
            if (tri_min_shortcut(lv, fv, D.r, D.L, &dk, &u, &v)) {
                ordered_take(B, dk, u, v, slot, t);
            } else if (may_defer && nq < QN) {
                qt[nq] = slot;
                ql[nq++] = lb;
            } else {
                need = true;
            }
        }
        __syncwarp();
        const float3 r = warp_search(D, need, lv);
        if (need) ordered_take(B, r.x, r.y, r.z, slot, t);
    };
    // the triangle that held the minimum at the previous evaluation first
    {
        bool on = false;
        if (valid && hint >= 0) {
            const float4 sph = __ldg(&D.leaf[hint].sph);
            on = node_sdf(fr, fr + 9, sph, D.r, D.L) < sph.w + eps;
            if (on) {
                float lv[3][3];
                int t;
                leaf_local(D.leaf, hint, fr, lv, &t);
                for (int m = 0; m < 3; ++m) UB = fminf(UB, sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr));
                seeded = hint;
            }
        }
        settle(on, hint, 0.f, false);
    }
    int sp = 0;
    {
        const float4 rt = __ldg(&D.nodes[0].sph);
        if (__any_sync(0xFFFFFFFFu, valid && node_sdf(fr, fr + 9, rt, D.r, D.L) < rt.w + eps)) {   // Eq. (21)
            sn[0] = 0;
            sl[0] = -INFINITY;
            sp = 1;
        }
    }
#pragma unroll 1
    while (sp > 0) {
        --sp;
        const int ni = sn[sp];
        const float lim = valid ? fminf(UB, B.d) : -INFINITY;
        // the bound stored with the node is the smallest over the lanes
        if (!__any_sync(0xFFFFFFFFu, valid && !(sl[sp] > lim))) continue;
        const int4 nd = __ldg(reinterpret_cast<const int4 *>(&D.nodes[ni]) + 1);   // left, first, count
        if (nd.x < 0) {
            for (int k = 0; k < nd.z; ++k) {
                const int slot = nd.y + k;
                const float4 sph = __ldg(&D.leaf[slot].sph);
                const float ft = node_sdf(fr, fr + 9, sph, D.r, D.L);
                const float limt = valid ? fminf(UB, B.d) : -INFINITY;
                const bool cand = valid && slot != seeded && ft < sph.w + eps && !(ft - sph.w > limt);   // Eq. (21)
                bool now = false;
                float lbt = 0.f;
                if (cand) {
                    float lv[3][3];
                    int t;
                    leaf_local(D.leaf, slot, fr, lv, &t);
                    for (int m = 0; m < 3; ++m) UB = fminf(UB, sdf_cyl(lv[m][0], lv[m][1], lv[m][2], D.r, D.L, nullptr));
                    lbt = lin_lower_bound(lv, D.r, D.L);
                    if (!(lbt > fminf(UB, B.d))) {
                        if (nc < QC) {
                            int j = nc++;
                            for (; j > 0 && cl[j - 1] > lbt; --j) {   // insertion in the order of the bounds
                                ct[j] = ct[j - 1];
                                cl[j] = cl[j - 1];
                            }
                            ct[j] = slot;
                            cl[j] = lbt;
                        } else {
                            now = true;
                        }
                    }
                }
                if (__any_sync(0xFFFFFFFFu, now)) settle(now, slot, lbt, true);
            }
        } else if (sp + 2 <= 64) {
            const float4 cL = __ldg(&D.nodes[nd.x].sph), cR = __ldg(&D.nodes[nd.x + 1].sph);
            const float fl = node_sdf(fr, fr + 9, cL, D.r, D.L), fR = node_sdf(fr, fr + 9, cR, D.r, D.L);
            const float bl = fl - cL.w, br = fR - cR.w;
            const bool nl = valid && fl < cL.w + eps && !(bl > lim);   // Eq. (21)
            const bool nr = valid && fR < cR.w + eps && !(br > lim);
            const bool anyl = __any_sync(0xFFFFFFFFu, nl), anyr = __any_sync(0xFFFFFFFFu, nr);
            // smallest bound over the lanes that need the child
            const float wl = unord_f(__reduce_min_sync(0xFFFFFFFFu, ord_f(nl ? bl : INFINITY)));
            const float wr = unord_f(__reduce_min_sync(0xFFFFFFFFu, ord_f(nr ? br : INFINITY)));
            const bool lfirst = wl <= wr;
            if (anyl && anyr) {
                sn[sp] = lfirst ? nd.x + 1 : nd.x;
                sl[sp++] = lfirst ? wr : wl;
                sn[sp] = lfirst ? nd.x : nd.x + 1;
                sl[sp++] = lfirst ? wl : wr;
            } else if (anyl || anyr) {
                sn[sp] = anyl ? nd.x : nd.x + 1;
                sl[sp++] = anyl ? wl : wr;
            }
        }
    }
#pragma unroll 1
    for (int s = 0; s < QC; ++s) {
        const bool on = s < nc && !(cl[s] > fminf(UB, B.d));
        if (__any_sync(0xFFFFFFFFu, on)) settle(on, on ? ct[s] : -1, on ? cl[s] : 0.f, true);
    }
#pragma unroll 1
    for (int s = 0; s < QN; ++s) {
        const bool on = s < nq && !(ql[s] > fminf(UB, B.d));
        if (!__any_sync(0xFFFFFFFFu, on)) continue;
        float lv[3][3] = {};
        int t = -1;
        if (on) leaf_local(D.leaf, qt[s], fr, lv, &t);
        const float3 r = warp_search(D, on, lv);
        if (on) ordered_take(B, r.x, r.y, r.z, qt[s], t);
    }
}

// One warp per block over the listed partials (list[0] entries, index c nwarp + w).
template <bool GRAD>
__global__ void __launch_bounds__(32)
k_refine_ordered(const RefineDev *Dt, const int32_t *grp, const CandF *cands, double *acc_part, int nwarp,
                 float *dist_out, float *wit_out, float *nrm_out, int2 *hints, const int32_t *list)
{
    const int n = list[0], lane = threadIdx.x;
#pragma unroll 1
    for (int e = blockIdx.x; e < n; e += gridDim.x) {
        const int id = list[1 + e], c = id / nwarp, w = id % nwarp, i = 32 * w + lane;
        const RefineDev D = Dt[grp ? grp[c] : 0];
        const CandF &cf = cands[c];
        const bool valid = i < D.P;
        const PoseRec &pr = D.poses[valid ? i : D.P - 1];
        float fr[12];
        pose_frame_in_object(cf, pr, fr);
        int2 *hp = hints ? hints + (size_t)c * nwarp * 32 + i : nullptr;
        OrderedBest B;
        ordered_query(D, fr, valid, hp && valid ? hp->x : -1, B);
        __syncwarp();
        const bool hit = valid && B.slot >= 0;
        float lv[3][3], xl[3] = {0.f, 0.f, 0.f};
        if (hit) {
            int t;
            leaf_local(D.leaf, B.slot, fr, lv, &t);
            const float w0 = 1.f - B.u - B.v;
            for (int a = 0; a < 3; ++a) xl[a] = fmaf(w0, lv[0][a], fmaf(B.u, lv[1][a], B.v * lv[2][a]));
        }
        if (hp && valid) *hp = hit ? pack_hint(B.slot, B.u, B.v) : make_int2(-1, 0);
        PoseTerms o;
        if (valid)
            pose_terms<GRAD>(D, cf, pr, hit, hit ? B.d : INFINITY, xl, lv, (size_t)c * D.P + i, dist_out, wit_out,
                             nrm_out, o);
        write_partial<GRAD>(o, acc_part, c, nwarp, w);
    }
}

// ---------------------------------------------------------------------------
// FP64 per-candidate step
// ---------------------------------------------------------------------------
__device__ void vcoef(double th, double *a, double *b, double *da, double *db)
{
    if (th < 1e-4) {
        double t2 = th * th;
        *a = 0.5 - t2 / 24.0 + t2 * t2 / 720.0;
        *b = 1.0 / 6.0 - t2 / 120.0 + t2 * t2 / 5040.0;
        *da = -1.0 / 12.0 + t2 / 180.0;
        *db = -1.0 / 60.0 + t2 / 1260.0;
    } else {
        double s = sin(th), c = cos(th);
        *a = (1.0 - c) / (th * th);
        *b = (th - s) / (th * th * th);
        *da = (th * s - 2.0 * (1.0 - c)) / (th * th * th * th);
        *db = ((1.0 - c) * th - 3.0 * (th - s)) / (th * th * th * th * th);
    }
}

// Pose T(xi) (Eq. (14)-(17)) and the derivative data of the next evaluation, by
// one warp: lane 3 i + j < 9 forms entry (i, j) of each matrix, the scalars are
// formed by every lane.  An FP64 instruction holds the SM's FP64 unit for 16
// cycles whatever its active lanes, so nine entries cost what one costs.
__device__ void cand_from_state(const double *st, CandF *out)
{
    const unsigned all = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, e = lane < 9 ? lane : 8, i = e / 3, j = e % 3;
    double R0[9], p0[3], an[3], u[3], w[3];
    for (int k = 0; k < 9; ++k) R0[k] = st[k];
    for (int k = 0; k < 3; ++k) { p0[k] = st[9 + k]; an[k] = st[12 + k]; u[k] = st[15 + k]; w[k] = st[18 + k]; }
    const double th = sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    double a, b, da, db;
    vcoef(th, &a, &b, &da, &db);
    const double sA = th < 1e-4 ? 1.0 - th * th / 6.0 + th * th * th * th / 120.0 : sin(th) / th;
    // [w]x and [u]x: entry (i, j) = -eps_ijk w_k
    auto cross_entry = [](const double *v, int r, int c) -> double {
        if (r == c) return 0.0;
        const int k = 3 - r - c;
        const double x = k == 0 ? v[0] : k == 1 ? v[1] : v[2];
        return (c - r + 3) % 3 == 1 ? -x : x;
    };
    const double K = cross_entry(w, i, j);
    double K2;
    {
        const double r0 = cross_entry(w, i, 0), r1 = cross_entry(w, i, 1), r2 = cross_entry(w, i, 2);
        K2 = r0 * cross_entry(w, 0, j) + r1 * cross_entry(w, 1, j) + r2 * cross_entry(w, 2, j);
    }
    const double I = i == j ? 1.0 : 0.0;
    const double dR = I + sA * K + a * K2, V = I + a * K + b * K2;
    const double d0 = __shfl_sync(all, dR, 3 * i), d1 = __shfl_sync(all, dR, 3 * i + 1), d2 = __shfl_sync(all, dR, 3 * i + 2);
    const double v0 = __shfl_sync(all, V, 3 * i), v1 = __shfl_sync(all, V, 3 * i + 1), v2 = __shfl_sync(all, V, 3 * i + 2);
    auto col = [&](int r) -> double { return j == 0 ? R0[3 * r] : j == 1 ? R0[3 * r + 1] : R0[3 * r + 2]; };
    const double R = d0 * col(0) + d1 * col(1) + d2 * col(2);
    double Ra[3];
    for (int k = 0; k < 3; ++k) Ra[k] = R0[3 * k] * an[0] + R0[3 * k + 1] * an[1] + R0[3 * k + 2] * an[2];
    const double dRRa = d0 * Ra[0] + d1 * Ra[1] + d2 * Ra[2];
    const double Vu = v0 * u[0] + v1 * u[1] + v2 * u[2];
    // d(V u)/dw = -a [u]x + (w x u) (a'/th) w^T + b((w.u) I + w u^T - 2 u w^T) + (w x (w x u)) (b'/th) w^T
    auto at = [](const double *v, int k) -> double { return k == 0 ? v[0] : k == 1 ? v[1] : v[2]; };
    const double wi = at(w, i), wj = at(w, j), ui = at(u, i), uj = at(u, j);
    const int i1 = i == 2 ? 0 : i + 1, i2 = i == 0 ? 2 : i - 1;
    const double wxu = at(w, i1) * at(u, i2) - at(w, i2) * at(u, i1);
    const double wd = w[0] * u[0] + w[1] * u[1] + w[2] * u[2], ww = th * th;
    const double wxwxu = wi * wd - ui * ww;
    const double t1 = -a * cross_entry(u, i, j) + wxu * da * wj;
    const double t2 = b * ((wd * I + wi * uj) - 2.0 * ui * wj) + wxwxu * db * wj;
    if (lane < 9) {
        out->Mc[e] = (float)(t1 + t2);
        out->R[e] = (float)R;
        out->V[e] = (float)V;
        if (j == 0) {
            const double p = at(p0, i), ra = at(Ra, i);
            out->p[i] = (float)(((p + Vu) + ra) - dRRa);
            out->c[i] = (float)((p + Vu) + ra);
        }
    }
}

// Solves H x = b by Cholesky, H symmetric 6 x 6: lane i < 6 holds row i in h[]
// and b_i; x (all six) in every lane.  False when H is not positive definite.
__device__ bool chol6_warp(const double *h, double b, double *x)
{
    const unsigned all = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31;
    double l[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        double s = h[j];
#pragma unroll
        for (int k = 0; k < j; ++k) s -= l[k] * __shfl_sync(all, l[k], j);
        const double d = __shfl_sync(all, s, j);
        if (!(d > 0.0)) return false;   // the same in every lane
        const double r = sqrt(d);
        l[j] = lane == j ? r : s / r;
    }
    double y[6], s = b;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double sk = __shfl_sync(all, s, k), lk = __shfl_sync(all, l[k], k);
        y[k] = sk / lk;
        s -= l[k] * y[k];
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        double t = y[i];
#pragma unroll
        for (int k = i + 1; k < 6; ++k) t -= __shfl_sync(all, l[i], k) * x[k];
        x[i] = t / __shfl_sync(all, l[i], i);
    }
    return true;
}

// Sum k < n of candidate c's partials, in the order of the poses: lane k adds
// value k (the loads of a round are independent, the additions a chain), the
// sums land in acc (shared).  One warp per candidate: with one thread adding
// all 28 values this took 42 us at 8 partials and 310 us at 160.
__device__ __forceinline__ void sum_partials(const double *acc_part, int c, int nwarp, int n, double *acc)
{
    const int lane = threadIdx.x;
    const double *p = acc_part + (size_t)c * nwarp * NACC + lane;
    if (lane < n) {
        double v = 0.0;
        int q = 0;
        for (; q + 8 <= nwarp; q += 8) {
            double t[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] = p[(size_t)(q + j) * NACC];
#pragma unroll
            for (int j = 0; j < 8; ++j) v += t[j];
        }
        for (; q < nwarp; ++q) v += p[(size_t)q * NACC];
        acc[lane] = v;
    }
    __syncwarp();
}

// prm: lambda, mu, step_t, step_r, b_t, b_r
// mode 0: only refresh the candidate data from the state
// mode 1: sum the partials, record J, take one projected Gauss-Newton step
// mode 2: sum the partials and record J (final evaluation)
// One warp per candidate; the 6 x 6 system by six lanes (with one thread 33 us a
// step, most of it FP64 divisions, roots and a serial chain).
__global__ void __launch_bounds__(32) k_refine_solve(int nwarp, double *state, const double *acc_part, const double *prm,
                                                     int mode, CandF *cands)
{
    const int c = blockIdx.x, lane = threadIdx.x;
    __shared__ double acc[NACC];
    double *st = state + (size_t)c * ST;
    if (mode != 0) {
        sum_partials(acc_part, c, nwarp, NACC, acc);
        const double lam = prm[0], mu = prm[1];
        double xi[6], xx = 0.0;
        for (int j = 0; j < 6; ++j) xi[j] = st[15 + j];
        for (int j = 0; j < 6; ++j) xx += xi[j] * xi[j];
        __syncwarp();   // every lane has read xi
        if (lane == 0) st[21] = acc[0] + lam * xx;   // J (Eq. (19))
        if (mode == 1) {
            const int i = lane < 6 ? lane : 5;
            double h[6], own = 0.0;
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                const int lo = i < j ? i : j, hi = i < j ? j : i;
                h[j] = acc[7 + 6 * lo - lo * (lo - 1) / 2 + (hi - lo)];
                if (i == j) {
                    h[j] += 2.0 * lam + mu;
                    own = xi[j];
                }
            }
            const double nb = -(acc[1 + i] + 2.0 * lam * own);
            double dl[6];
            if (chol6_warp(h, nb, dl)) {
                double mt = 0.0, mr = 0.0;
                for (int j = 0; j < 3; ++j) { mt = fmax(mt, fabs(dl[j])); mr = fmax(mr, fabs(dl[3 + j])); }
                double sc = 1.0;
                if (mt > prm[2]) sc = fmin(sc, prm[2] / mt);
                if (mr > prm[3]) sc = fmin(sc, prm[3] / mr);
                double step = 0.0;
#pragma unroll
                for (int j = 0; j < 6; ++j) if (i == j) step = dl[j];
                double v = own + sc * step;
                const double bb = i < 3 ? prm[4] : prm[5];
                if (v > bb) v = bb;
                if (v < -bb) v = -bb;
                if (lane < 6) st[15 + lane] = v;
                __syncwarp();
            }
        }
    }
    cand_from_state(st, &cands[c]);
}

// ---------------------------------------------------------------------------
// L-BFGS-B (Sec. V-C as printed): one warp per candidate, FP64.  A round
// evaluates J and grad J (Eq. (19), (28)) at every active candidate's trial
// twist; this kernel then accepts or backtracks the step (Armijo), updates the
// limited-memory pairs (s, y) and builds the next trial.  The direction is the
// two-loop recursion on the variables that are not held at a bound of
// Eq. (20) (a variable is held when it sits on its bound and the gradient
// pushes it outward), steps are projected onto the box and backtracked by
// safeguarded quadratic interpolation (first step of unit length, as in
// L-BFGS-B; later ones start at alpha = 1), and a candidate stops
// when the projected gradient or the relative decrease of J is below its
// tolerance, after max_iter accepted steps, or when backtracking fails.
// ---------------------------------------------------------------------------
enum {
    LB_X = 0, LB_F = 6, LB_G = 7, LB_D = 13, LB_ALPHA = 19, LB_GTD = 20, LB_ITER = 21, LB_NBACK = 22,
    LB_NH = 23, LB_HEAD = 24, LB_STATUS = 25, LB_NEV = 26, LB_HIST = 32
};
constexpr int LB_S = LB_HIST, LB_Y = LB_HIST + 6 * LB_M, LB_RHO = LB_HIST + 12 * LB_M;
static_assert(LB_RHO + LB_M <= LB_ST, "L-BFGS state");

__device__ __forceinline__ double lb_hi(int j, const double *prm) { return j < 3 ? prm[4] : prm[5]; }

__device__ __forceinline__ double lb_clamp(double v, double hi) { return v > hi ? hi : (v < -hi ? -hi : v); }

__device__ __forceinline__ bool lb_held(const double *x, const double *g, int j, const double *prm)
{
    const double hi = lb_hi(j, prm);
    return (x[j] <= -hi && g[j] > 0.0) || (x[j] >= hi && g[j] < 0.0);
}

// d = -H g on the free variables (two-loop recursion over the stored pairs)
__device__ void lb_direction(double *L, const double *prm)
{
    const double *x = L + LB_X, *g = L + LB_G;
    double *d = L + LB_D;
    const int nh = (int)L[LB_NH], head = (int)L[LB_HEAD];
    double q[6], al[LB_M];
    for (int j = 0; j < 6; ++j) q[j] = lb_held(x, g, j, prm) ? 0.0 : g[j];
    for (int k = 0; k < nh; ++k) {
        const int i = (head - 1 - k + 2 * LB_M) % LB_M;
        const double *S = L + LB_S + 6 * i, *Y = L + LB_Y + 6 * i;
        double a = 0.0;
        for (int j = 0; j < 6; ++j) a += S[j] * q[j];
        a *= L[LB_RHO + i];
        al[k] = a;
        for (int j = 0; j < 6; ++j) q[j] -= a * Y[j];
    }
    double gam = 1.0;
    if (nh > 0) {
        const int i = (head - 1 + LB_M) % LB_M;
        const double *S = L + LB_S + 6 * i, *Y = L + LB_Y + 6 * i;
        double sy = 0.0, yy = 0.0;
        for (int j = 0; j < 6; ++j) { sy += S[j] * Y[j]; yy += Y[j] * Y[j]; }
        gam = sy / yy;
    }
    for (int j = 0; j < 6; ++j) q[j] *= gam;
    for (int k = nh - 1; k >= 0; --k) {
        const int i = (head - 1 - k + 2 * LB_M) % LB_M;
        const double *S = L + LB_S + 6 * i, *Y = L + LB_Y + 6 * i;
        double b = 0.0;
        for (int j = 0; j < 6; ++j) b += Y[j] * q[j];
        b *= L[LB_RHO + i];
        for (int j = 0; j < 6; ++j) q[j] += S[j] * (al[k] - b);
    }
    double gd = 0.0;
    for (int j = 0; j < 6; ++j) {
        d[j] = lb_held(x, g, j, prm) ? 0.0 : -q[j];
        gd += g[j] * d[j];
    }
    if (!(gd < 0.0)) {   // not a descent direction: forget the pairs, steepest descent
        L[LB_NH] = 0.0;
        for (int j = 0; j < 6; ++j) d[j] = lb_held(x, g, j, prm) ? 0.0 : -g[j];
    }
}

// trial twist x + alpha d projected onto the box; false when it does not move
__device__ bool lb_trial(double *L, double *xi, const double *prm)
{
    const double *x = L + LB_X, *g = L + LB_G, *d = L + LB_D;
    double gtd = 0.0, mv = 0.0;
    for (int j = 0; j < 6; ++j) {
        xi[j] = lb_clamp(x[j] + L[LB_ALPHA] * d[j], lb_hi(j, prm));
        gtd += g[j] * (xi[j] - x[j]);
        mv = fmax(mv, fabs(xi[j] - x[j]));
    }
    L[LB_GTD] = gtd;
    return mv > 0.0 && gtd < 0.0;
}

__device__ void lb_new_step(double *L, double *xi, const double *prm)
{
    lb_direction(L, prm);
    double dn = 0.0;
    for (int j = 0; j < 6; ++j) dn += L[LB_D + j] * L[LB_D + j];
    dn = sqrt(dn);
    L[LB_ALPHA] = (L[LB_NH] == 0.0 && dn > 1.0) ? 1.0 / dn : 1.0;
    L[LB_NBACK] = 0.0;
    if (!lb_trial(L, xi, prm)) L[LB_STATUS] = 1.0;
}

// One candidate's step (one thread).
__device__ void lbfgs_step(double *st, const double *acc, const double *prm, double *L, int32_t *active, int phase)
{
    double *xi = st + 15;
    if (phase == 0) {
        for (int k = 0; k < LB_ST; ++k) L[k] = 0.0;
        L[LB_ITER] = -1.0;
        for (int j = 0; j < 6; ++j) xi[j] = 0.0;
        *active = 1;
    } else if (phase == 1) {
        const double lam = prm[0];
        double xx = 0.0;
        for (int j = 0; j < 6; ++j) xx += xi[j] * xi[j];
        const double ft = acc[0] + lam * xx;
        double gt[6];
        for (int j = 0; j < 6; ++j) gt[j] = acc[1 + j] + 2.0 * lam * xi[j];
        L[LB_NEV] += 1.0;
        bool take = false;
        if (L[LB_ITER] < 0.0) {
            take = true;   // the starting point
        } else if (isfinite(ft) && ft <= L[LB_F] + 1e-4 * L[LB_GTD]) {
            take = true;
        }
        if (take) {
            const bool first = L[LB_ITER] < 0.0;
            const double fold = L[LB_F];
            if (!first) {
                double s[6], y[6], sy = 0.0, yy = 0.0;
                for (int j = 0; j < 6; ++j) {
                    s[j] = xi[j] - L[LB_X + j];
                    y[j] = gt[j] - L[LB_G + j];
                    sy += s[j] * y[j];
                    yy += y[j] * y[j];
                }
                if (sy > 1e-12 * yy) {
                    const int i = (int)L[LB_HEAD];
                    for (int j = 0; j < 6; ++j) { L[LB_S + 6 * i + j] = s[j]; L[LB_Y + 6 * i + j] = y[j]; }
                    L[LB_RHO + i] = 1.0 / sy;
                    L[LB_HEAD] = (double)((i + 1) % LB_M);
                    L[LB_NH] = fmin((double)LB_M, L[LB_NH] + 1.0);
                }
            }
            for (int j = 0; j < 6; ++j) { L[LB_X + j] = xi[j]; L[LB_G + j] = gt[j]; }
            L[LB_F] = ft;
            L[LB_ITER] = first ? 0.0 : L[LB_ITER] + 1.0;
            double pg = 0.0;
            for (int j = 0; j < 6; ++j) pg = fmax(pg, fabs(lb_clamp(xi[j] - gt[j], lb_hi(j, prm)) - xi[j]));
            const bool conv = pg <= prm[6] ||
                              (!first && fold - ft <= prm[7] * fmax(fmax(fabs(fold), fabs(ft)), 1.0)) ||
                              L[LB_ITER] >= prm[8];
            if (conv) L[LB_STATUS] = 1.0;
            else lb_new_step(L, xi, prm);
        } else {
            // backtrack to the minimiser of the quadratic through f, the
            // slope gtd and the trial value, kept within [0.1, 0.5] of the step
            const double gtd = L[LB_GTD], dphi = ft - L[LB_F];
            double t = (isfinite(ft) && dphi - gtd > 0.0) ? -gtd / (2.0 * (dphi - gtd)) : 0.1;
            t = fmin(fmax(t, 0.1), 0.5);
            L[LB_NBACK] += 1.0;
            L[LB_ALPHA] *= t;
            if (L[LB_NBACK] > 30.0 || !lb_trial(L, xi, prm)) L[LB_STATUS] = 1.0;
        }
        if (L[LB_STATUS] != 0.0) {
            for (int j = 0; j < 6; ++j) xi[j] = L[LB_X + j];
            *active = 0;
        }
    } else {
        if (L[LB_ITER] >= 0.0)
            for (int j = 0; j < 6; ++j) xi[j] = L[LB_X + j];
        st[21] = L[LB_F];
        st[22] = fmax(L[LB_ITER], 0.0);
        st[23] = L[LB_NEV];
        *active = 0;
    }
}

// prm: lambda, mu, step_t, step_r, b_t, b_r, pgtol, ftol, max_iter
// phase 0: start at xi = 0; phase 1: take the round's evaluation; phase 2:
// leave every candidate at its last accepted twist (J, iterations and
// evaluations in the state's slots 21, 22, 23)
// (the solver state is staged in shared memory: its steps are chains of loads
// and FP64 operations of one thread)
__global__ void __launch_bounds__(32) k_lbfgs(int nwarp, double *state, const double *acc_part, const double *prm,
                                              double *lbs, int32_t *active, CandF *cands, int phase)
{
    const int c = blockIdx.x;   // one warp per candidate
    __shared__ double acc[7];
    if (phase == 1) {
        if (!active[c]) return;   // finished: its state stays as it is
        sum_partials(acc_part, c, nwarp, 7, acc);
    }
    __shared__ double L[LB_ST];
    double *st = state + (size_t)c * ST, *Lg = lbs + (size_t)c * LB_ST;
    if (phase != 0)
        for (int k = threadIdx.x; k < LB_ST; k += 32) L[k] = Lg[k];
    __syncwarp();
    if (threadIdx.x == 0) lbfgs_step(st, acc, prm, L, active + c, phase);
    __syncwarp();
    for (int k = threadIdx.x; k < LB_ST; k += 32) Lg[k] = L[k];
    cand_from_state(st, &cands[c]);
}

cudaError_t launch_lbfgs(int K, int nwarp, double *state, const double *acc_part, const double *prm, double *lbs,
                         int32_t *active, CandF *cands, int phase, cudaStream_t st)
{
    k_lbfgs<<<K, 32, 0, st>>>(nwarp, state, acc_part, prm, lbs, active, cands, phase);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <int Q, bool GRAD>
static cudaError_t launch_dist_t(const RefineDev *Dt, const int32_t *grp, int K, int nwarp, const CandF *cands,
                                 double *acc_part, float *dist_out, float *wit_out, float *nrm_out, int2 *hints,
                                 const int32_t *active, int32_t *redo, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nwarp * 32 / Q), (unsigned)K);
    cfg.blockDim = dim3(DistCfg<Q>::NT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = DistCfg<Q>::CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = DistCfg<Q>::CL > 1 ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_refine_dist<Q, GRAD>, Dt, grp, cands, acc_part, nwarp, dist_out, wit_out,
                                       nrm_out, hints, active, redo);
    if (e != cudaSuccess) return e;
    // two one-warp blocks per SM (an empty list costs the launch); where distances are
    // asked for, every group with a pose beyond the cutoff is on the list
    const int blocks = dist_out ? (int)std::min<int64_t>((int64_t)K * nwarp, 32 * 152) : 2 * 152;
    k_refine_ordered<GRAD><<<blocks, 32, 0, st>>>(Dt, grp, cands, acc_part, nwarp, dist_out, wit_out, nrm_out, hints,
                                                  redo);
    return cudaGetLastError();
}

cudaError_t launch_refine_eval(const RefineDev *Dt, const int32_t *grp, int K, int nwarp, const CandF *cands,
                               double *acc_part, bool grad, float *dist_out, float *wit_out, float *nrm_out,
                               int32_t *redo, cudaStream_t st, int2 *hints, const int32_t *active)
{
    if (nwarp < 1 || nwarp % REF_WARPS) return cudaErrorInvalidValue;
    const size_t poses = (size_t)K * nwarp * 32;
    cudaError_t e0 = cudaMemsetAsync(redo, 0, sizeof(int32_t), st);
    if (e0 != cudaSuccess) return e0;
    const auto launch = [&](auto with_grad, auto without) {
        return (grad ? with_grad : without)(Dt, grp, K, nwarp, cands, acc_part, dist_out, wit_out, nrm_out, hints,
                                            active, redo, st);
    };
    // Fewer poses per block while there are not enough blocks to fill the SMs
    // (8: a cluster of four blocks shares a partial sum), 128 once there are.  The
    // limits are those of L-BFGS-B, most of whose candidates are finished in most
    // rounds: 100 rounds of up to 64000 queries 58 / 46 / 76 ms at 8 / 32 / 128 poses
    // per block.  21 evaluations of Gauss-Newton, all of them active, on 65 k
    // triangles: 2048 queries 4.0 / 4.9 / 9.1 ms, 5120 5.5 / 5.4 / 9.3, 19968 22.2 /
    // 13.8 / 16.5, 40960 32 / 16.9 / 15.2, 198656 130 / 63 / 41, 327680 206 / 96 / 57:
    // they would change over at 5000 and 30000.
    if (poses <= 20000) return launch(launch_dist_t<8, true>, launch_dist_t<8, false>);
    if (poses <= 200000) return launch(launch_dist_t<32, true>, launch_dist_t<32, false>);
    return launch(launch_dist_t<128, true>, launch_dist_t<128, false>);
}

cudaError_t launch_refine_solve(int K, int nwarp, double *state, const double *acc_part, const double *prm, int mode,
                                CandF *cands, cudaStream_t st)
{
    k_refine_solve<<<K, 32, 0, st>>>(nwarp, state, acc_part, prm, mode, cands);
    return cudaGetLastError();
}

size_t cand_bytes() { return sizeof(CandF); }

// Twists from a device FP32 array into the state (the differentiable form).
__global__ void k_set_xi(int B, const float *xi, double *state)
{
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    for (int j = 0; j < 6; ++j) state[(size_t)b * ST + 15 + j] = (double)xi[6 * b + j];
}

// J[b] and grad[b] (Eq. (19), (28)) from the partials.
__global__ void __launch_bounds__(32)
k_finish_objective(int nwarp, const double *state, const double *acc_part, double lam, float *J, float *grad,
                   const float *gJ)
{
    const int b = blockIdx.x;   // one warp per twist
    const double *xi = state + (size_t)b * ST + 15;
    __shared__ double acc[7];
    sum_partials(acc_part, b, nwarp, 7, acc);
    if (threadIdx.x) return;
    double xx = 0.0;
    for (int j = 0; j < 6; ++j) xx += xi[j] * xi[j];
    if (J) J[b] = (float)(acc[0] + lam * xx);
    if (grad) {
        double sc = gJ ? (double)gJ[b] : 1.0;
        for (int j = 0; j < 6; ++j) grad[6 * b + j] = (float)(sc * (acc[1 + j] + 2.0 * lam * xi[j]));
    }
}

cudaError_t launch_set_xi(int B, const float *xi, double *state, cudaStream_t st)
{
    k_set_xi<<<(B + 63) / 64, 64, 0, st>>>(B, xi, state);
    return cudaGetLastError();
}

cudaError_t launch_finish_objective(int B, int nwarp, const double *state, const double *acc_part, double lam, float *J,
                                    float *grad, const float *gJ, cudaStream_t st)
{
    k_finish_objective<<<B, 32, 0, st>>>(nwarp, state, acc_part, lam, J, grad, gJ);
    return cudaGetLastError();
}

}  // namespace dock

// Object grid (Sec. IV-A.1, Eq. (1)-(4)).
//
// This translation unit is compiled with -fmad=false: every FP64 expression
// is rounded exactly as written, so the signed distance, its sign and the band
// value O are the same numbers a plain FP64 evaluation of the definition gives.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "dock_internal.h"
#include "tri_f32.h"

namespace dock {

// Squared distance from p to triangle (a, b, c): closest point by the Voronoi
// regions of the triangle (three vertices, three edges, interior).
__device__ double tri_dist2(const double *p, const double *a, const double *b, const double *c)
{
    double e0[3], e1[3], w[3];
    for (int i = 0; i < 3; ++i) { e0[i] = b[i] - a[i]; e1[i] = c[i] - a[i]; w[i] = p[i] - a[i]; }
    double s1 = (e0[0] * w[0] + e0[1] * w[1]) + e0[2] * w[2];
    double s2 = (e1[0] * w[0] + e1[1] * w[1]) + e1[2] * w[2];
    double q[3];
    if (s1 <= 0.0 && s2 <= 0.0) {                      // vertex a
        q[0] = a[0]; q[1] = a[1]; q[2] = a[2];
    } else {
        double wb[3] = {p[0] - b[0], p[1] - b[1], p[2] - b[2]};
        double s3 = (e0[0] * wb[0] + e0[1] * wb[1]) + e0[2] * wb[2];
        double s4 = (e1[0] * wb[0] + e1[1] * wb[1]) + e1[2] * wb[2];
        double vc = s1 * s4 - s3 * s2;
        if (s3 >= 0.0 && s4 <= s3) {                   // vertex b
            q[0] = b[0]; q[1] = b[1]; q[2] = b[2];
        } else if (vc <= 0.0 && s1 >= 0.0 && s3 <= 0.0) {   // edge ab
            double t = s1 / (s1 - s3);
            for (int i = 0; i < 3; ++i) q[i] = a[i] + t * e0[i];
        } else {
            double wc[3] = {p[0] - c[0], p[1] - c[1], p[2] - c[2]};
            double s5 = (e0[0] * wc[0] + e0[1] * wc[1]) + e0[2] * wc[2];
            double s6 = (e1[0] * wc[0] + e1[1] * wc[1]) + e1[2] * wc[2];
            double vb = s5 * s2 - s1 * s6;
            double va = s3 * s6 - s5 * s4;
            if (s6 >= 0.0 && s5 <= s6) {               // vertex c
                q[0] = c[0]; q[1] = c[1]; q[2] = c[2];
            } else if (vb <= 0.0 && s2 >= 0.0 && s6 <= 0.0) {   // edge ac
                double t = s2 / (s2 - s6);
                for (int i = 0; i < 3; ++i) q[i] = a[i] + t * e1[i];
            } else if (va <= 0.0 && (s4 - s3) >= 0.0 && (s5 - s6) >= 0.0) {   // edge bc
                double t = (s4 - s3) / ((s4 - s3) + (s5 - s6));
                for (int i = 0; i < 3; ++i) q[i] = b[i] + t * (c[i] - b[i]);
            } else {                                   // interior
                double inv = 1.0 / ((va + vb) + vc);
                double v = vb * inv, u = vc * inv;
                for (int i = 0; i < 3; ++i) q[i] = (a[i] + e0[i] * v) + e1[i] * u;
            }
        }
    }
    double dx = p[0] - q[0], dy = p[1] - q[1], dz = p[2] - q[2];
    return (dx * dx + dy * dy) + dz * dz;
}

// 2-D edge function of (a -> b) at (py, pz) with the point perturbed to
// (py + eps, pz + eps^2) (simulation of simplicity): never zero for a
// non-degenerate edge, so a row through a shared edge or vertex is counted
// by exactly one triangle.
__device__ int edge_side(double ay, double az, double by, double bz, double py, double pz, double *e)
{
    double v = (by - ay) * (pz - az) - (bz - az) * (py - ay);
    *e = v;
    if (v > 0.0) return 1;
    if (v < 0.0) return -1;
    if (bz != az) return bz > az ? -1 : 1;
    if (by != ay) return by > ay ? 1 : -1;
    return 0;
}

// The cells triangle t's box meets, per axis (axis 0 is y when flat); false when none.
__device__ __forceinline__ bool tri_cells(const double *V, const int32_t *T, int64_t t, const double3 o, double cs,
                                          const int3 d, bool flat, double pad, int *lo, int *hi)
{
    const double org[3] = {o.x, o.y, o.z};
    const int dim[3] = {d.x, d.y, d.z};
    for (int a = flat ? 1 : 0; a < 3; ++a) {
        const double x0 = V[3 * (size_t)T[3 * t] + a], x1 = V[3 * (size_t)T[3 * t + 1] + a], x2 = V[3 * (size_t)T[3 * t + 2] + a];
        const double mn = fmin(x0, fmin(x1, x2)) - pad, mx = fmax(x0, fmax(x1, x2)) + pad;
        const double l = floor((mn - org[a]) / cs), h = floor((mx - org[a]) / cs);
        lo[a] = l > 0.0 ? (l < (double)dim[a] ? (int)l : dim[a]) : 0;
        hi[a] = h < (double)(dim[a] - 1) ? (h >= 0.0 ? (int)h : -1) : dim[a] - 1;
        if (lo[a] > hi[a]) return false;
    }
    if (flat) lo[0] = hi[0] = 0;
    return true;
}

// total[0] += the entries of the 3-D bins, total[1] += those of the (y, z) bins
__global__ void k_bins_total(const double *V, const int32_t *T, int64_t nt, double3 o, double cs, int3 d, double pad,
                             unsigned long long *total)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long n[2] = {0ull, 0ull};
    int lo[3], hi[3];
    if (t < nt && tri_cells(V, T, t, o, cs, d, false, pad, lo, hi))
        n[0] = (unsigned long long)(hi[0] - lo[0] + 1) * (hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);
    if (t < nt && tri_cells(V, T, t, o, cs, d, true, 0.0, lo, hi))
        n[1] = (unsigned long long)(hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);
    for (int k = 0; k < 2; ++k) {
        for (int s = 16; s > 0; s >>= 1) n[k] += __shfl_down_sync(0xFFFFFFFFu, n[k], s);
        if ((threadIdx.x & 31) == 0 && n[k]) atomicAdd(&total[k], n[k]);
    }
}

cudaError_t launch_bins_total(const double *V, const int32_t *T, int64_t nt, const double *o, double cs, const int *d,
                              double pad, unsigned long long *total, cudaStream_t st)
{
    k_bins_total<<<(unsigned)((nt + 127) / 128), 128, 0, st>>>(V, T, nt, make_double3(o[0], o[1], o[2]), cs,
                                                               make_int3(d[0], d[1], d[2]), pad, total);
    return cudaGetLastError();
}

// at[cell] += 1 per triangle and cell; with items given, the old value is the
// triangle's place (the order within a cell does not matter: minima and
// parities are taken over it).  A thread finds a triangle's box, the warp enters
// its triangles one by one, a cell per lane (and the parts of gridDim.y share a
// box): an entry waits for its atomic, and a box may hold 30 cells (a triangle
// of a fine mesh) or all two million.  With a thread entering all cells of its
// triangle, the grid of a turned cube of 12 triangles at N = 128, h = 0.6 took
// 152 ms, now 14.
__global__ void __launch_bounds__(128)
k_bins(const double *V, const int32_t *T, int64_t nt, double3 o, double cs, int3 d, bool flat, double pad, int32_t *at,
       int32_t *items)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned all = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, w = flat ? 1 : d.x;
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0}, n = 0;
    if (t < nt && tri_cells(V, T, t, o, cs, d, flat, pad, lo, hi))
        n = (hi[0] - lo[0] + 1) * (hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);   // at most 128^3
    for (unsigned left = __ballot_sync(all, n > 0); left; left &= left - 1) {
        const int src = __ffs(left) - 1, cells = __shfl_sync(all, n, src);
        const int x0 = __shfl_sync(all, lo[0], src), y0 = __shfl_sync(all, lo[1], src), z0 = __shfl_sync(all, lo[2], src);
        const int nx = __shfl_sync(all, hi[0], src) - x0 + 1, ny = __shfl_sync(all, hi[1], src) - y0 + 1;
        const int32_t tri = (int32_t)(t - lane + src);
#pragma unroll 4
        for (int e = 32 * (int)blockIdx.y + lane; e < cells; e += 32 * (int)gridDim.y) {
            const int r = e / nx, x = x0 + e - r * nx, z = r / ny, y = y0 + r - z * ny;
            const int k = atomicAdd(&at[((z0 + z) * d.y + y) * w + x], 1);
            if (items) items[k] = tri;
        }
    }
}

// parts per box: while there are too few triangles to fill the chip (a box of 128^3
// cells entered by one warp takes about 10 ms), at no cost to a fine mesh
static dim3 bins_grid(int64_t nt)
{
    const int64_t parts = std::min<int64_t>(1024, std::max<int64_t>(1, 65536 / nt));
    return dim3((unsigned)((nt + 127) / 128), (unsigned)parts);
}

// exclusive prefix sums of n counts in place (one block); at[n] gets the total
__global__ void __launch_bounds__(1024) k_bins_scan(int32_t *at, int n)
{
    __shared__ int32_t warp_sum[32];
    __shared__ int32_t carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 1024) {
        const int i = base + tid;
        const int32_t v = i < n ? at[i] : 0;
        int32_t x = v;
        for (int s = 1; s < 32; s <<= 1) {
            const int32_t y = __shfl_up_sync(0xFFFFFFFFu, x, s);
            if (lane >= s) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int32_t w = warp_sum[lane];
            for (int s = 1; s < 32; s <<= 1) {
                const int32_t y = __shfl_up_sync(0xFFFFFFFFu, w, s);
                if (lane >= s) w += y;
            }
            warp_sum[lane] = w;
        }
        __syncthreads();
        const int32_t before = carry + (warp ? warp_sum[warp - 1] : 0) + x - v;
        if (i < n) at[i] = before;
        __syncthreads();
        if (tid == 1023) carry = before + v;
        __syncthreads();
    }
    if (tid == 0) at[n] = carry;
}

cudaError_t launch_bins_count(const double *V, const int32_t *T, int64_t nt, const double *o, double cs, const int *d,
                              bool flat, double pad, int32_t *start, cudaStream_t st)
{
    k_bins<<<bins_grid(nt), 128, 0, st>>>(V, T, nt, make_double3(o[0], o[1], o[2]), cs,
                                                         make_int3(d[0], d[1], d[2]), flat, pad, start, nullptr);
    k_bins_scan<<<1, 1024, 0, st>>>(start, (flat ? 1 : d[0]) * d[1] * d[2]);
    return cudaGetLastError();
}

cudaError_t launch_bins_fill(const double *V, const int32_t *T, int64_t nt, const double *o, double cs, const int *d,
                             bool flat, double pad, int32_t *at, int32_t *items, cudaStream_t st)
{
    k_bins<<<bins_grid(nt), 128, 0, st>>>(V, T, nt, make_double3(o[0], o[1], o[2]), cs,
                                                         make_int3(d[0], d[1], d[2]), flat, pad, at, items);
    return cudaGetLastError();
}

// One block per lattice row (ky, kz); thread kx < N.  The row's crossings with
// the mesh along +x decide the sign (odd count beyond x = inside): inside[row]
// gets one bit per voxel.
__global__ void __launch_bounds__(128)
k_object_rows(const double *V, const int32_t *T, ObjBins bins, int N, double h, double o0, double o1, double o2,
              uint32_t *inside, int *err)
{
    __shared__ double xs[1024];
    __shared__ int nx;
    const int ky = blockIdx.x % N, kz = blockIdx.x / N;
    const double py = h * (double)ky + o1;
    const double pz = h * (double)kz + o2;
    if (threadIdx.x == 0) nx = 0;
    __syncthreads();
    {
        int cy = (int)floor((py - o1) / bins.cs), cz = (int)floor((pz - o2) / bins.cs);
        if (cy >= 0 && cy < bins.d2[0] && cz >= 0 && cz < bins.d2[1]) {
            int cell = cz * bins.d2[0] + cy;
            for (int k = bins.cell2_start[cell] + threadIdx.x; k < bins.cell2_start[cell + 1]; k += blockDim.x) {
                int t = bins.cell2_items[k];
                const double *v0 = V + 3 * T[3 * t], *v1 = V + 3 * T[3 * t + 1], *v2 = V + 3 * T[3 * t + 2];
                double e0, e1, e2;
                int s0 = edge_side(v1[1], v1[2], v2[1], v2[2], py, pz, &e0);
                int s1 = edge_side(v2[1], v2[2], v0[1], v0[2], py, pz, &e1);
                int s2 = edge_side(v0[1], v0[2], v1[1], v1[2], py, pz, &e2);
                if (s0 == 0 || s0 != s1 || s1 != s2) continue;
                double den = (e0 + e1) + e2;
                if (den == 0.0) continue;
                double x = ((e0 * v0[0] + e1 * v1[0]) + e2 * v2[0]) / den;
                int slot = atomicAdd(&nx, 1);
                if (slot < 1024) xs[slot] = x;
                else atomicExch(err, DOCK_E_OVERFLOW);
            }
        }
    }
    __syncthreads();
    const int n_cross = min(nx, 1024), kx = threadIdx.x;
    if (kx >= N) return;   // whole warps: N is a multiple of 32
    const double p0 = h * (double)kx + o0;
    int par = 0;
    for (int c = 0; c < n_cross; ++c) par ^= (xs[c] > p0) ? 1 : 0;
    const uint32_t w = __ballot_sync(0xFFFFFFFFu, par);
    if ((kx & 31) == 0) inside[(size_t)blockIdx.x * (N / 32) + kx / 32] = w;
}

size_t tri_f32_bytes() { return sizeof(TriF); }

__global__ void k_tri_f32(int n, const double *V, const int32_t *T, const uint8_t *touch, double o0, double o1,
                          double o2, float S, float cut, TriF *out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double o[3] = {o0, o1, o2};
    double v[3][3];
    for (int m = 0; m < 3; ++m)
        for (int a = 0; a < 3; ++a) v[m][a] = V[3 * (size_t)T[3 * t + m] + a] - o[a];
    out[t] = tri_f32(v, S, cut, touch == nullptr || touch[t]);
}

// One block per bin cell: band values of the cell's voxels.  FP64 operations
// run at a 64th of the FP32 rate, so the triangles of the cell (about 500 near
// a surface of 65 k triangles) are measured in FP32 first, and the exact FP64
// distance (whose minimum is the result) is formed only for those whose FP32
// lower bound does not lie above the smallest FP32 upper bound, a few per voxel
// (tri_f32.h: bounds for triangles of any shape; the thinnest always get their
// FP64 distance).  Two
// threads per voxel share the triangles of a tile; the voxel-triangle pairs in
// question are dealt to the block.  44.2 -> 3.1 ms (rows and cells) at N = 128 and 65 k triangles
// (with one thread per voxel and FP64 throughout, lanes of a warp walking
// different cells).
// axis[a][c]: first voxel index along axis a whose cell is >= c (d3[a] + 1 entries
// each, the axes one after another).
__global__ void __launch_bounds__(128)
k_object_cells(const double *V, const int32_t *T, const TriF *tri, ObjBins bins, const int32_t *axis, int N, double h,
               double o0, double o1, double o2, double tau_out, double tau_in, double deep, float edge_tol,
               const uint32_t *inside, float *O)
{
    constexpr int NT = 128, NV = 64, TILE = 64, PAIRS = 4096, ROOM = 8 * NT;
    __shared__ TriF tile[TILE];
    __shared__ int tidx[TILE];
    __shared__ unsigned long long best[NV], bestt[NV];
    __shared__ int pair_i[PAIRS];             // item of the cell's list
    __shared__ unsigned char pair_s[PAIRS];   // voxel slot
    __shared__ int n_pairs;
    const int tid = threadIdx.x;
    const int cx = blockIdx.x % bins.d3[0], cy = (blockIdx.x / bins.d3[0]) % bins.d3[1], cz = blockIdx.x / (bins.d3[0] * bins.d3[1]);
    const int32_t *ax = axis, *ay = ax + bins.d3[0] + 1, *az = ay + bins.d3[1] + 1;
    const int x0 = ax[cx], y0 = ay[cy], z0 = az[cz], lx = ax[cx + 1] - x0, ly = ay[cy + 1] - y0, lz = az[cz + 1] - z0;
    const int nv = lx * ly * lz;
    const int i0 = bins.cell3_start[blockIdx.x], n_items = bins.cell3_start[blockIdx.x + 1] - i0;
    const double cut = tau_out > tau_in ? tau_out : tau_in, cut2 = cut * cut;
    const float skip = (float)cut * 1.00001f;
    // exact distances of the pairs in question
    auto settle = [&](int base) {
        __syncthreads();
        const int np = n_pairs;
        for (int k = tid; k < np; k += NT) {
            const int s = pair_s[k], t = bins.cell3_items[i0 + pair_i[k]], v = base + s;
            const double p[3] = {h * (double)(x0 + v % lx) + o0, h * (double)(y0 + (v / lx) % ly) + o1,
                                 h * (double)(z0 + v / (lx * ly)) + o2};
            const double d2 = tri_dist2(p, V + 3 * (size_t)T[3 * t], V + 3 * (size_t)T[3 * t + 1], V + 3 * (size_t)T[3 * t + 2]);
            // distances are not negative: their bits are in their order (a NaN never is the smallest)
            const unsigned long long bits = (unsigned long long)__double_as_longlong(d2);
            atomicMin(&best[s], bits);
            if (tri[t].touch) atomicMin(&bestt[s], bits);
        }
        __syncthreads();
        if (tid == 0) n_pairs = 0;
        __syncthreads();
    };
    for (int base = 0; base < nv; base += NV) {
        const int s = tid >> 1, half = tid & 1, v = base + s;
        const bool on = v < nv;
        // relative to the origin, as the FP64 point rounds (for the warps that have a voxel: FP64
        // operations are what a cell of one voxel and no triangle costs)
        float px = 0.f, py = 0.f, pz = 0.f;
        if (on) {
            px = (float)((h * (double)(x0 + v % lx) + o0) - o0);
            py = (float)((h * (double)(y0 + (v / lx) % ly) + o1) - o1);
            pz = (float)((h * (double)(z0 + v / (lx * ly)) + o2) - o2);
        }
        if (tid < NV) best[tid] = bestt[tid] = 0x7FF0000000000000ull;   // +infinity
        if (tid == 0) n_pairs = 0;
        // pass 0: upper bounds of the two minima; pass 1: the pairs in question
        float ub = INFINITY, ubt = INFINITY;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
            for (int j0 = 0; j0 < n_items; j0 += TILE) {
                const int nt = min(TILE, n_items - j0);
                __syncthreads();
                for (int k = tid; k < nt; k += NT) tidx[k] = bins.cell3_items[i0 + j0 + k];
                __syncthreads();
                constexpr int W = sizeof(TriF) / 4;
                for (int k = tid; k < nt * W; k += NT)
                    reinterpret_cast<uint32_t *>(tile)[k] = reinterpret_cast<const uint32_t *>(tri + tidx[k / W])[k % W];
                __syncthreads();
                for (int k0 = 0; k0 < nt; k0 += 16) {
                    // eight triangles of the tile per thread, then room is looked for again
                    if (on)
                        for (int k = k0 + half; k < min(nt, k0 + 16); k += 2) {
                            const TriF &t = tile[k];
                            // (a triangle without a usable FP32 bound is always in question)
                            const bool sure = t.tol < INFINITY;
                            const float b = fminf(skip, fmaxf(ub, ubt));
                            if (pass == 0) {
                                if (sure) {
                                    const float d = tri_bound_f32<true>(t, px, py, pz, b, edge_tol) + edge_tol;
                                    ub = fminf(ub, d);
                                    if (t.touch) ubt = fminf(ubt, d);
                                }
                            } else {
                                const float d = sure ? tri_bound_f32<false>(t, px, py, pz, b, edge_tol) : 0.f;
                                if (!sure || d <= fminf(skip, ub) || (t.touch && d <= fminf(skip, ubt))) {
                                    const int k2 = atomicAdd(&n_pairs, 1);
                                    pair_i[k2] = j0 + k;
                                    pair_s[k2] = (unsigned char)s;
                                }
                            }
                        }
                    if (pass == 1) {
                        __syncthreads();
                        const bool full = n_pairs > PAIRS - ROOM;
                        __syncthreads();
                        if (full) settle(base);
                    }
                }
            }
            if (pass == 0) {
                ub = fminf(ub, __shfl_xor_sync(0xFFFFFFFFu, ub, 1));
                ubt = fminf(ubt, __shfl_xor_sync(0xFFFFFFFFu, ubt, 1));
            }
        }
        settle(base);
        if (tid < NV && base + tid < nv) {
            const int vv = base + tid, kx = x0 + vv % lx, ky = y0 + (vv / lx) % ly, kz = z0 + vv / (lx * ly);
            const size_t row = (size_t)kz * N + ky;
            const int par = (inside[row * (N / 32) + kx / 32] >> (kx & 31)) & 1u;
            const double b2 = __longlong_as_double((long long)best[tid]), bt2 = __longlong_as_double((long long)bestt[tid]);
            double D = b2 < cut2 ? sqrt(b2) : INFINITY;
            double Dt = bt2 < cut2 ? sqrt(bt2) : INFINITY;
            double f = par ? -D : D;
            double Ot;
            if (0.0 <= f && f < tau_out) Ot = 1.0 - f / tau_out;          // Eq. (1), first branch
            else if (-tau_in < f && f < 0.0) Ot = 1.0 + f / tau_in;      // shallow penetration
            else if (f <= -tau_in) Ot = deep;                            // deep penetration
            else Ot = 0.0;
            double Om = 1.0 - Dt / tau_out;                              // Eq. (2)
            if (!(Om > 0.0)) Om = 0.0;
            double val = Ot < Om ? Ot : Om;                              // Eq. (3)
            O[row * N + kx] = (float)val;
        }
        __syncthreads();
    }
}

cudaError_t launch_object_grid(const double *V, const int32_t *T, int64_t nt, const uint8_t *touch, const ObjBins &bins,
                               const int32_t *axis, int N, double h, const double *o, double tau_out, double tau_in,
                               double deep, void *tri, uint32_t *inside, float *O, int *err, cudaStream_t st)
{
    TriF *tf = static_cast<TriF *>(tri);
    const double cut = tau_out > tau_in ? tau_out : tau_in;
    const float S = (float)(N * h);
    k_tri_f32<<<(unsigned)((nt + 127) / 128), 128, 0, st>>>((int)nt, V, T, touch, o[0], o[1], o[2], S, (float)cut, tf);
    k_object_rows<<<N * N, 128, 0, st>>>(V, T, bins, N, h, o[0], o[1], o[2], inside, err);
    k_object_cells<<<bins.d3[0] * bins.d3[1] * bins.d3[2], 128, 0, st>>>(V, T, tf, bins, axis, N, h, o[0], o[1], o[2],
                                                                        tau_out, tau_in, deep, tri_edge_tol(S), inside, O);
    return cudaGetLastError();
}

}  // namespace dock

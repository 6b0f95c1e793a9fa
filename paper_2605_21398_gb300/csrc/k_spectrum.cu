// Canvas spectrum of a lattice grid (Eq. (9)): conj(F(O)) / M^3 (or F(S) / M^3)
// of N^3 values zero-padded to M = 2N per axis, in FP64, stored as FP32 in the
// z-pass tile order.
//
// One FP64 FFT per axis, columns of 16 neighbouring kx per block: M = R1 x R2
// (256 = 16 x 16, 192 = 16 x 12, 128 = 16 x 8, 64 = 8 x 8), the two stages as
// register DFTs of 8 to 16 values with one exchange through shared memory.
// Index n = R2 a + b in, k = k1 + R1 k2 out:
//   X[k] = sum_b w_R2^(b k2) ( w_M^(b k1) sum_a w_R1^(a k1) x[R2 a + b] ),
// where a < R1 / 2 (the upper half of every column is padding).  FP64 operations
// bound it (2 FMA lanes per SM and clock): about 22 an output value and axis, where the
// direct sums over N terms took 4 N.  At N = 128: 32.9 -> 0.8 ms for the three
// passes.
#include <cuda_runtime.h>
#include <stdint.h>

#include "dock_internal.h"

namespace dock {

namespace {

struct cd { double x, y; };

__device__ __forceinline__ cd mk(double a, double b) { cd r; r.x = a; r.y = b; return r; }
__device__ __forceinline__ cd add(cd a, cd b) { return mk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ cd sub(cd a, cd b) { return mk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ cd mul(cd a, double c, double s) { return mk(a.x * c - a.y * s, a.x * s + a.y * c); }
__device__ __forceinline__ cd mul_mi(cd a) { return mk(a.y, -a.x); }   // times -i

// forward DFT of 4; with HALF the last two inputs are zero
template <bool HALF> __device__ __forceinline__ void dft4(cd &a, cd &b, cd &c, cd &d)
{
    if (HALF) {
        const cd x = a, y = b, z = mul_mi(b);
        a = add(x, y);
        b = add(x, z);
        c = sub(x, y);
        d = sub(x, z);
    } else {
        const cd t0 = add(a, c), t1 = sub(a, c), t2 = add(b, d), t3 = mul_mi(sub(b, d));
        a = add(t0, t2);
        b = add(t1, t3);
        c = sub(t0, t2);
        d = sub(t1, t3);
    }
}

// forward DFT of R values in natural order (HALF: v[R/2 ..] are zero)
template <int R, bool HALF> struct Dft;

template <bool HALF> struct Dft<8, HALF> {
    __device__ __forceinline__ static void run(cd *v)
    {
        const double s = 0.70710678118654752440;
        cd e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft4<HALF>(e[0], e[1], e[2], e[3]);
        dft4<HALF>(o[0], o[1], o[2], o[3]);
        o[1] = mk((o[1].x + o[1].y) * s, (o[1].y - o[1].x) * s);
        o[2] = mul_mi(o[2]);
        o[3] = mk((o[3].y - o[3].x) * s, -(o[3].x + o[3].y) * s);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = add(e[k], o[k]);
            v[k + 4] = sub(e[k], o[k]);
        }
    }
};

template <bool HALF> struct Dft<16, HALF> {
    __device__ __forceinline__ static void run(cd *v)
    {
        // n = n1 + 4 n2, k = k1 + 4 k2; cos and sin of 2 pi m / 16
        const double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
        cd a[4][4];
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < 4; ++n2) a[n1][n2] = v[n1 + 4 * n2];
            dft4<HALF>(a[n1][0], a[n1][1], a[n1][2], a[n1][3]);
        }
        a[1][1] = mul(a[1][1], c1, -s1);
        a[1][2] = mul(a[1][2], h, -h);
        a[1][3] = mul(a[1][3], s1, -c1);
        a[2][1] = mul(a[2][1], h, -h);
        a[2][2] = mul_mi(a[2][2]);
        a[2][3] = mul(a[2][3], -h, -h);
        a[3][1] = mul(a[3][1], s1, -c1);
        a[3][2] = mul(a[3][2], -h, -h);
        a[3][3] = mul(a[3][3], -c1, s1);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            dft4<false>(a[0][k1], a[1][k1], a[2][k1], a[3][k1]);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = a[k2][k1];
        }
    }
};

template <> struct Dft<12, false> {
    __device__ __forceinline__ static void run(cd *v)
    {
        // n = n1 + 3 n2 (n1 < 3, n2 < 4), k = k1 + 4 k2
        const double c1 = 0.86602540378443864676;
        cd a[3][4];
#pragma unroll
        for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < 4; ++n2) a[n1][n2] = v[n1 + 3 * n2];
            dft4<false>(a[n1][0], a[n1][1], a[n1][2], a[n1][3]);
        }
        a[1][1] = mul(a[1][1], c1, -0.5);
        a[1][2] = mul(a[1][2], 0.5, -c1);
        a[1][3] = mul_mi(a[1][3]);
        a[2][1] = mul(a[2][1], 0.5, -c1);
        a[2][2] = mul(a[2][2], -0.5, -c1);
        a[2][3] = mk(-a[2][3].x, -a[2][3].y);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            const cd p = add(a[1][k1], a[2][k1]), q = sub(a[1][k1], a[2][k1]);
            const cd m = mk(a[0][k1].x - 0.5 * p.x, a[0][k1].y - 0.5 * p.y), r = mk(c1 * q.y, -c1 * q.x);   // -i sin(60 deg) q
            v[k1] = add(a[0][k1], p);
            v[k1 + 4] = add(m, r);
            v[k1 + 8] = sub(m, r);
        }
    }
};

template <int M> struct Split;
template <> struct Split<64> { static constexpr int R1 = 8, R2 = 8; };
template <> struct Split<128> { static constexpr int R1 = 16, R2 = 8; };
template <> struct Split<192> { static constexpr int R1 = 16, R2 = 12; };
template <> struct Split<256> { static constexpr int R1 = 16, R2 = 16; };

constexpr int COLS = 16;   // columns per block

// Forward transform of the block's 16 columns.  Thread (c, t), t < R1: `in(c,
// n)` gives value n < M / 2 of column c; afterwards v[k2] of thread (c, k1)
// holds output k1 + R1 k2.  xb: [M][COLS] exchange buffer.
template <int M, class In>
__device__ __forceinline__ void column_fft(In in, cd *v, cd *xb, const double2 *tw)
{
    constexpr int R1 = Split<M>::R1, R2 = Split<M>::R2;
    const int c = threadIdx.x % COLS, t = threadIdx.x / COLS;
    if (t < R2) {
        cd u[R1];
#pragma unroll
        for (int a = 0; a < R1; ++a) u[a] = a < R1 / 2 ? in(c, R2 * a + t) : mk(0.0, 0.0);
        Dft<R1, true>::run(u);
#pragma unroll
        for (int k = 0; k < R1; ++k) {
            const double2 w = tw[t * k];   // b k1 < M
            xb[(k * R2 + t) * COLS + c] = mul(u[k], w.x, w.y);
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < R2; ++b) v[b] = xb[(t * R2 + b) * COLS + c];
    Dft<R2, false>::run(v);
}

// x: rows 2 p and 2 p + 1 of the grid as one complex column p; A[row][kx], kx <= M / 2
template <int M>
__global__ void __launch_bounds__(Split<M>::R1 *COLS)
k_spec_x(const float *O, const double2 *tw, double2 *A, bool pen)
{
    constexpr int N = M / 2, H = M / 2, R1 = Split<M>::R1, R2 = Split<M>::R2;
    extern __shared__ __align__(16) unsigned char smem[];
    cd *xb = reinterpret_cast<cd *>(smem);
    const float *o = O + (size_t)blockIdx.x * 2 * COLS * N;
    cd v[R2];
    column_fft<M>([&](int c, int n) -> cd {
        double a = (double)o[(2 * c) * N + n], b = (double)o[(2 * c + 1) * N + n];
        if (pen) { a = fmin(a, 0.0); b = fmin(b, 0.0); }
        return mk(a, b);
    }, v, xb, tw);
    __syncthreads();
    const int c = threadIdx.x % COLS, k1 = threadIdx.x / COLS;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) xb[(k1 + R1 * k2) * COLS + c] = v[k2];
    __syncthreads();
    for (int e = threadIdx.x; e < COLS * (H + 1); e += blockDim.x) {
        const int p = e / (H + 1), kx = e % (H + 1);
        const cd a = xb[kx * COLS + p], r = xb[((M - kx) % M) * COLS + p];
        double2 *row = A + ((size_t)blockIdx.x * 2 * COLS + 2 * p) * (H + 1) + kx;
        row[0] = make_double2(0.5 * (a.x + r.x), 0.5 * (a.y - r.y));
        row[H + 1] = make_double2(0.5 * (a.y + r.y), -0.5 * (a.x - r.x));
    }
}

// y: B[z][ky][kx] from A[z][y][kx]
template <int M>
__global__ void __launch_bounds__(Split<M>::R1 *COLS)
k_spec_y(const double2 *A, const double2 *tw, double2 *B)
{
    constexpr int N = M / 2, H = M / 2, R1 = Split<M>::R1, R2 = Split<M>::R2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int kx = blockIdx.x * COLS + threadIdx.x % COLS, k1 = threadIdx.x / COLS, z = blockIdx.y;
    const double2 *a = A + (size_t)z * N * (H + 1) + kx;
    cd v[R2];
    column_fft<M>([&](int, int n) -> cd {
        if (kx > H) return mk(0.0, 0.0);
        const double2 x = a[(size_t)n * (H + 1)];
        return mk(x.x, x.y);
    }, v, reinterpret_cast<cd *>(smem), tw);
    if (kx > H) return;
    double2 *b = B + (size_t)z * M * (H + 1) + kx;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) b[(size_t)(k1 + R1 * k2) * (H + 1)] = make_double2(v[k2].x, v[k2].y);
}

// z: the spectrum tile, value / M^3, conjugated when cj; zero for kx in (M / 2, P)
template <int M>
__global__ void __launch_bounds__(Split<M>::R1 *COLS)
k_spec_z(const double2 *B, int P, const double2 *tw, float2 *spec, bool cj)
{
    constexpr int H = M / 2, R1 = Split<M>::R1, R2 = Split<M>::R2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int kx = blockIdx.x * COLS + threadIdx.x % COLS, k1 = threadIdx.x / COLS, ky = blockIdx.y;
    const double2 *b = B + (size_t)ky * (H + 1) + kx;
    cd v[R2];
    column_fft<M>([&](int, int n) -> cd {
        if (kx > H) return mk(0.0, 0.0);
        const double2 x = b[(size_t)n * M * (H + 1)];
        return mk(x.x, x.y);
    }, v, reinterpret_cast<cd *>(smem), tw);
    if (kx >= P) return;
    const double sc = 1.0 / ((double)M * (double)M * (double)M);
    const size_t f = (size_t)ky * P + kx, chunk = f / 32, lane = f % 32;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2)
        spec[(chunk * M + k1 + R1 * k2) * 32 + lane] =
            make_float2((float)(v[k2].x * sc), (float)((cj ? -v[k2].y : v[k2].y) * sc));
}

template <int M>
cudaError_t launch_spectrum_t(const float *O, int P, double2 *A, double2 *B, const double2 *tw, float2 *spec,
                              cudaStream_t st, bool pen, bool cj)
{
    constexpr int N = M / 2, NT = Split<M>::R1 * COLS;
    const int sm = (int)(sizeof(cd) * M * COLS);
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(k_spec_x<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_spec_y<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(k_spec_z<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm)) != cudaSuccess) return e;
    k_spec_x<M><<<N * N / (2 * COLS), NT, sm, st>>>(O, tw, A, pen);
    k_spec_y<M><<<dim3((N + 1 + COLS - 1) / COLS, N), NT, sm, st>>>(A, tw, B);
    k_spec_z<M><<<dim3((P + COLS - 1) / COLS, M), NT, sm, st>>>(B, P, tw, spec, cj);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_spectrum(const float *O, int N, int M, int P, double2 *work1, double2 *work2, const double2 *twd,
                            float2 *spec, cudaStream_t st, bool pen, bool conj)
{
    if (M != 2 * N || P != N + 2) return cudaErrorInvalidValue;
    switch (M) {
    case 64: return launch_spectrum_t<64>(O, P, work1, work2, twd, spec, st, pen, conj);
    case 128: return launch_spectrum_t<128>(O, P, work1, work2, twd, spec, st, pen, conj);
    case 192: return launch_spectrum_t<192>(O, P, work1, work2, twd, spec, st, pen, conj);
    case 256: return launch_spectrum_t<256>(O, P, work1, work2, twd, spec, st, pen, conj);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace dock

// Products with symmetric matrices stored once per pair of entries (internal to libfcm).
//
// A block factor F = A_B^+ and a cut cell's K_e are symmetric, so a product that streams them from HBM needs
// half of the entries.  Matrices of p <= 2 (at most 81 rows) are stored folded: the upper triangle in a
// rectangle of H = (n + 1) / 2 rows and W = n | 1 columns (n = 2 H or 2 H - 1 rows), row i < H of the triangle
// at the right end of rectangle row i, row i >= H reversed at the left end of row 2 H - 1 - i.  A CTA copies
// the rectangle to shared memory (one bulk copy; enough CTAs fit an SM to keep more than 100 KB in flight)
// and gives each row of the product a thread, which walks the columns in ascending
// order, as the product with the full matrix did: the same additions in the same order.  W is odd, so the 32
// rows of a warp read 32 different banks both where they walk down a column (consecutive entries of one
// rectangle row) and where they walk along their own rows (stride W).
#pragma once

#include <cuda_runtime.h>

#include "fcm_ff.cuh"
#include "fcm_tma.cuh"

namespace fcm {

__host__ __device__ constexpr int fold_h(int n) { return (n + 1) / 2; }
__host__ __device__ constexpr int fold_w(int n) { return n | 1; }
// stored entries, padded so that the matrix is a multiple of 16 bytes (float or float2 entries)
__host__ __device__ constexpr int fold_entries(int n) { return (fold_h(n) * fold_w(n) + 3) / 4 * 4; }

// entry (i, j), i <= j
__host__ __device__ __forceinline__ int fold_at(int n, int i, int j)
{
    const int H = fold_h(n), W = fold_w(n);
    return i < H ? i * W + j + (W - n) : (2 * H - 1 - i) * W + n - 1 - j;
}

// the entry (i, j), i <= j, stored at `at`; false for an unused place
__host__ __device__ __forceinline__ bool fold_entry(int n, int at, int &i, int &j)
{
    const int H = fold_h(n), W = fold_w(n), r = at / W, c = at % W;
    i = r;
    j = c - (W - n);
    if (r < H && j >= i) return true;
    i = 2 * H - 1 - r;
    j = n - 1 - c;
    return r < H && i < n && j >= i;
}

// Calls f(k, e) for the entries e of row t in column order, columns j + k of four at a time: x(j) is called
// before the four columns j .. j + 3 (fewer at the end of the row).  N: n as a constant, or 0.  Lanes of a warp
// take consecutive rows from t0 on (t = t0 + lane, clamped to n - 1 by the caller).
template <int N, class T, class X, class F>
__device__ __forceinline__ void fold_row(const T *__restrict__ m, int n_, int t0, int t, X &&x, F &&f)
{
    const int n = N > 0 ? N : n_;
    const int H = fold_h(n), W = fold_w(n), s = W - n;
    // the lane's own row of the triangle: m[own + dir * j]
    const int dir = t < H ? 1 : -1, own = t < H ? t * W + s : (2 * H - 1 - t) * W + n - 1;
    auto general = [&](int j) {
        // column t of row j below the diagonal, the lane's own row from there on
        const T *below = j < H ? m + t + (j * W + s) : m - t + ((2 * H - 1 - j) * W + n - 1);
        return j < t ? *below : m[own + dir * j];
    };
    const int t1 = min(t0 + 32, n), a1 = min(t0, H) & ~3, b0 = min((H + 3) & ~3, t0);
    int j = 0;
    {  // every lane below the diagonal, in the upper rows: down a column
        const T *p = m + t + s;
#pragma unroll 4
        for (; j < a1; j += 4) {
            x(j);
#pragma unroll
            for (int k = 0; k < 4; ++k) f(k, p[k * W]);
            p += 4 * W;
        }
    }
    for (; j < b0; j += 4) {
        x(j);
#pragma unroll
        for (int k = 0; k < 4; ++k) f(k, general(j + k));
    }
    {  // the same in the folded rows
        const T *p = m + (2 * H - 1 - j) * W + n - 1 - t;
#pragma unroll 4
        for (; j < t0; j += 4) {
            x(j);
#pragma unroll
            for (int k = 0; k < 4; ++k) f(k, p[-k * W]);
            p -= 4 * W;
        }
    }
    const int d1 = t1 & ~3;
#pragma unroll 2
    for (; j < d1; j += 4) {  // the diagonal tile
        x(j);
#pragma unroll
        for (int k = 0; k < 4; ++k) f(k, general(j + k));
    }
    // right of the diagonal: along the lane's own row (t1 < n only if t1 is a multiple of 32)
    const T *p = m + own + dir * j;
    if (t1 == n) {
        if (j < n) {
            x(j);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (j + k < n) f(k, general(j + k));
        }
        return;
    }
#pragma unroll 4
    for (; j + 4 <= n; j += 4) {
        x(j);
#pragma unroll
        for (int k = 0; k < 4; ++k) f(k, p[k * dir]);
        p += 4 * dir;
    }
    if (j < n) {
        x(j);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (j + k < n) f(k, p[k * dir]);
    }
}

// Row t of F [x_0 .. x_{NR-1}] for a folded F in FP32: xs[j][NR] in shared memory (rows up to the next
// multiple of four readable).
template <int N, int NR>
__device__ __forceinline__ void fold_dot(const float *m, int n, int t0, int t, const float *xs, float (&acc)[NR])
{
    float xv[4][NR];
    fold_row<N>(
        m, n, t0, t,
        [&](int j) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const float4 v = reinterpret_cast<const float4 *>(xs + j * NR)[q];
                const int e = 4 * q;
                xv[e / NR][e % NR] = v.x;
                xv[(e + 1) / NR][(e + 1) % NR] = v.y;
                xv[(e + 2) / NR][(e + 2) % NR] = v.z;
                xv[(e + 3) / NR][(e + 3) % NR] = v.w;
            }
        },
        [&](int k, float f) {
#pragma unroll
            for (int r = 0; r < NR; ++r) acc[r] = fmaf(f, xv[k][r], acc[r]);
        });
}

// the same for a double-float F
template <int N, int NR>
__device__ __forceinline__ void fold_dot(const float2 *m, int n, int t0, int t, const float2 *xs, float (&S)[NR],
                                         float (&C)[NR])
{
    float2 xv[NR == 1 ? 4 : 1];
    const float2 *xj = xs;
    fold_row<N>(
        m, n, t0, t,
        [&](int j) {
            if constexpr (NR == 1) {
                const float4 a = reinterpret_cast<const float4 *>(xs + j)[0], b = reinterpret_cast<const float4 *>(xs + j)[1];
                xv[0] = make_float2(a.x, a.y);
                xv[1] = make_float2(a.z, a.w);
                xv[2] = make_float2(b.x, b.y);
                xv[3] = make_float2(b.z, b.w);
            } else {
                xj = xs + j * NR;
            }
        },
        [&](int k, float2 f) {
            if constexpr (NR == 1) {
                ff_fma(f.x, f.y, xv[k].x, xv[k].y, S[0], C[0]);
            } else {
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float2 v = xj[k * NR + r];
                    ff_fma(f.x, f.y, v.x, v.y, S[r], C[r]);
                }
            }
        });
}

}  // namespace fcm

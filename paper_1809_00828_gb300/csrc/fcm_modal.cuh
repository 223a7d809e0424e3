// K_ref x_e of uncut cells in Legendre modal form (internal to libfcm; FP64 and double-float; p <= 3).
//
// The integrated-Legendre basis is a sparse combination of Legendre polynomials: along one axis, with
// v_j the coefficient of phi_j = (P_j - P_{j-2}) / sqrt(2(2j-1)) and u_0, u_1 the hats' values, twice the
// Legendre coefficients are kappa_n r_n with
//   r_0 = u_0 + u_1 - k2 v_2,  r_1 = u_1 - u_0 - k3 v_3,  r_2 = v_2,  r_3 = v_3,
// kappa_n = k_n = sqrt(2 / (2n - 1)) for n >= 2, kappa_0 = kappa_1 = 1; and the derivative's coefficient n is
// (2n + 1) sum_{m > n, m - n odd} of them, rho_n e_n with
//   e_0 = r_1 + k3 r_3,  e_1 = r_2,  e_2 = r_3   (rho = 1, k2, k3).
// Legendre polynomials are orthogonal, so the bilinear form of Eq. (1) couples only equal mode triples alpha:
// every product of derivatives is one weight per alpha (modal_tables), and no Gauss point is needed.  p = 2
// takes about 1,000 multiply-adds or additions per cell where the 1D contractions with dense tables at the
// Gauss points took 36 (p+1)^4 + 21 (p+1)^3 = 3,483 (p = 3: 3,000 against 10,560).
//
// A warp is 32 cells and one displacement component c, three warps a group of 32 cells: each thread gathers
// and transforms its component's (p+1)^3 coefficients in registers, publishes them in shared memory, forms
// the component's stress against the other two components' modes, and transforms back: one barrier in all.
// Indices are rotated so that axis 0 of the thread's arrays is axis c of the cell; what a thread reads of
// component c + 1 or c + 2 is then at a compile-time offset.  The result goes to the cells' slots of Zk, entry
// (3 node + c) of cell i at Zk[(3 node + c) ncell + i], which k_sum_kernel adds up.
//
// FP64 is bound by its pipe, 79 % of the active cycles (ncu, 32^3 p = 3: 201 us for 30,543 uncut cells, about 180 at
// 2 operations per clock and SM; 745 us before).  Double-float takes 214 us for 440k cells at 80^3 p = 2 (1,091
// before): 62 % of the issue slots and 43 % of the FP32 pipe (ncu, 64^3), the rest waits of 15 warps per SM, which
// is what 128 registers allow, for their own results.  There the loop over the mode planes of axis 2 stays rolled (90 KB of code
// otherwise, and warps that wait for instructions), a first product starts its sum instead of adding to 0, and
// the sums stay unnormalised (370 -> 214 us together).
#pragma once

#include <cuda_runtime.h>

#include "fcm_device.cuh"
#include "fcm_ff.cuh"

namespace fcm {

constexpr double kModalK2 = 0.81649658092772603273;   // sqrt(2/3)
constexpr double kModalK3 = 0.63245553203367586640;   // sqrt(2/5)
constexpr int kModalTabs = 7;                         // weight tables per component (modal_tables)

// Arithmetic of the transforms: V the stored value, Acc a running sum.
struct ModalF64 {
    using V = double;
    static constexpr int kPlanes = 0;  // planes of the stress loop unrolled (0: all)
    struct Acc {
        double s;
    };
    __device__ static __forceinline__ V load(double x) { return x; }
    __device__ static __forceinline__ Acc start(V a) { return {a}; }
    __device__ static __forceinline__ Acc zero() { return {0.0}; }
    __device__ static __forceinline__ V constant(double k) { return k; }
    __device__ static __forceinline__ V neg(V a) { return -a; }
    __device__ static __forceinline__ void add(Acc &a, V b) { a.s += b; }
    __device__ static __forceinline__ Acc mul(V b, V c) { return {b * c}; }
    __device__ static __forceinline__ void mac(Acc &a, V b, V c) { a.s = fma(b, c, a.s); }
    __device__ static __forceinline__ V get(Acc a) { return a.s; }
    __device__ static __forceinline__ V norm(V a) { return a; }
    __device__ static __forceinline__ double to_double(V a) { return a; }
};

// Sums are kept as they run, (s, c) with c the errors and low parts: a following product takes s exactly and c
// in its cross term, so the dropped c * low term is 2^-48 of the summands either way and normalising each
// intermediate (3 operations) buys nothing.
struct ModalFF {
    using V = float2;
    static constexpr int kPlanes = 1;
    struct Acc {
        float s, c;
    };
    __device__ static __forceinline__ V load(double x) { return split_ff(x); }
    __device__ static __forceinline__ Acc start(V a) { return {a.x, a.y}; }
    __device__ static __forceinline__ Acc zero() { return {0.f, 0.f}; }
    __device__ static __forceinline__ V constant(double k)
    {
        return make_float2((float)k, (float)(k - (double)(float)k));  // folded at compile time
    }
    __device__ static __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
    __device__ static __forceinline__ void add(Acc &a, V b) { ff_add(a.s, a.c, b.x, b.y); }
    __device__ static __forceinline__ Acc mul(V b, V c)
    {
        const float p = __fmul_rn(b.x, c.x);
        return {p, __fmaf_rn(b.y, c.x, __fmaf_rn(b.x, c.y, __fmaf_rn(b.x, c.x, -p)))};
    }
    __device__ static __forceinline__ void mac(Acc &a, V b, V c) { ff_fma(b.x, b.y, c.x, c.y, a.s, a.c); }
    __device__ static __forceinline__ V get(Acc a) { return make_float2(a.s, a.c); }
    __device__ static __forceinline__ V norm(V a) { return ff_norm(a.x, a.y); }
    __device__ static __forceinline__ double to_double(V a) { return ff_to_double(a); }
};

// u (lattice order of a line: left hat, phi_2 .. phi_p, right hat) -> r, in place at stride ST
template <int P, int ST, class A>
__device__ __forceinline__ void modal_forward(typename A::V *u)
{
    using V = typename A::V;
    const V u0 = u[0], u1 = u[P * ST];
    typename A::Acc r0 = A::start(u0), r1 = A::start(u1);
    A::add(r0, u1);
    A::add(r1, A::neg(u0));
    if constexpr (P >= 2) A::mac(r0, A::constant(-kModalK2), u[ST]);
    if constexpr (P >= 3) A::mac(r1, A::constant(-kModalK3), u[2 * ST]);
    V r2{}, r3{};
    if constexpr (P >= 2) r2 = u[ST];
    if constexpr (P >= 3) r3 = u[2 * ST];
    u[0] = A::get(r0);
    u[ST] = A::get(r1);
    if constexpr (P >= 2) u[2 * ST] = r2;
    if constexpr (P >= 3) u[3 * ST] = r3;
}

// the transpose: o dual to r -> forces in lattice order, in place
template <int P, int ST, class A>
__device__ __forceinline__ void modal_backward(typename A::V *o)
{
    using V = typename A::V;
    const V o0 = o[0], o1 = o[ST];
    typename A::Acc a = A::start(o0), b = A::start(o1);
    A::add(a, A::neg(o1));  // left hat
    A::add(b, o0);          // right hat
    V w[4];
    if constexpr (P >= 2) {
        typename A::Acc t = A::start(o[2 * ST]);
        A::mac(t, A::constant(-kModalK2), o0);
        w[1] = A::get(t);
    }
    if constexpr (P >= 3) {
        typename A::Acc t = A::start(o[3 * ST]);
        A::mac(t, A::constant(-kModalK3), o1);
        w[2] = A::get(t);
    }
    o[0] = A::get(a);
    o[P * ST] = A::get(b);
#pragma unroll
    for (int n = 1; n < P; ++n) o[n * ST] = w[n];
}

// e_n along an axis at stride ST (elements) from the array entry f of mode n of that axis, n < P
template <int P, int ST, class A>
__device__ __forceinline__ typename A::V modal_deriv(const typename A::V *f, int n)
{
    if constexpr (P >= 3)
        if (n == 0) {
            typename A::Acc t = A::start(f[ST]);
            A::mac(t, A::constant(kModalK3), f[3 * ST]);
            return A::get(t);
        }
    return f[ST];
}

// o += (e_n)^T t along an axis at stride ST
template <int P, int ST, class A>
__device__ __forceinline__ void modal_deriv_t(typename A::Acc *o, int n, typename A::V t)
{
    A::add(o[ST], t);
    if constexpr (P >= 3)
        if (n == 0) A::mac(o[3 * ST], A::constant(kModalK3), t);
}

constexpr int kModalThreads = 96;  // one group of 32 cells per CTA
// CTAs per SM the register budget is set for (the warps of a CTA spread over the SM's four partitions); shared
// memory allows eight at p = 2 and three at p = 3
__host__ __device__ constexpr int modal_ctas(int P) { return P <= 2 ? 5 : 2; }
__host__ __device__ constexpr int modal_smem_bytes(int P)
{
    return ((P + 1) * (P + 1) * (P + 1)) * 3 * 8 * (kModalTabs + 32);
}

template <int P, class A>
__global__ void __launch_bounds__(kModalThreads, modal_ctas(P))
    modal_apply_kernel(const double *__restrict__ x, typename A::V *__restrict__ zk, const int *__restrict__ cells,
                       int ncells, Grid3 g, int64_t nc, const typename A::V *__restrict__ tab,
                       const int *__restrict__ done)
{
    using V = typename A::V;
    using Acc = typename A::Acc;
    constexpr int Q = P + 1, Q2 = Q * Q, Q3 = Q * Q2;
    if (done && *done) return;
    extern __shared__ __align__(16) unsigned char modal_smem[];
    V *tb = reinterpret_cast<V *>(modal_smem);
    V *cs = tb + 3 * kModalTabs * Q3;
    for (int t = threadIdx.x; t < 3 * kModalTabs * Q3; t += blockDim.x) tb[t] = tab[t];
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int idx = blockIdx.x * 32 + lane;
    const int cell = cells[min(idx, ncells - 1)];  // lanes past the end repeat the last cell and do not store
    const int cx = cell % g.n[0], cy = (cell / g.n[0]) % g.n[1], cz = cell / (g.n[0] * g.n[1]);
    const int64_t node = (int64_t)P * cx + g.M[0] * ((int64_t)P * cy + g.M[1] * ((int64_t)P * cz));
    const int64_t ps[3] = {3, 3 * (int64_t)g.M[0], 3 * (int64_t)g.M[0] * g.M[1]};
    const int64_t s0 = c == 0 ? ps[0] : c == 1 ? ps[1] : ps[2], s1 = c == 0 ? ps[1] : c == 1 ? ps[2] : ps[0],
                  s2 = c == 0 ? ps[2] : c == 1 ? ps[0] : ps[1];
    V *own = cs + c * Q3 * 32 + lane;
    {
        const double *xc = x + 3 * node + c;
        double xr[Q3];
#pragma unroll
        for (int i = 0; i < Q3; ++i) xr[i] = __ldg(xc + (i % Q) * s0 + ((i / Q) % Q) * s1 + (i / Q2) * s2);
        V r[Q3];
#pragma unroll
        for (int i = 0; i < Q3; ++i) r[i] = A::load(xr[i]);
#pragma unroll
        for (int i = 0; i < Q2; ++i) modal_forward<P, 1, A>(r + Q * i);
#pragma unroll
        for (int i = 0; i < Q2; ++i) modal_forward<P, Q, A>(r + i % Q + Q2 * (i / Q));
#pragma unroll
        for (int i = 0; i < Q2; ++i) modal_forward<P, Q2, A>(r + i);
#pragma unroll
        for (int i = 0; i < Q3; ++i) own[32 * i] = A::norm(r[i]);
    }
    __syncthreads();
    // component j = c + 1 is stored in its own frame (axes j, k, c), k = c + 2 in (k, c, j)
    const V *fj = cs + (c == 2 ? 0 : c + 1) * Q3 * 32 + lane;
    const V *fk = cs + (c == 0 ? 2 : c - 1) * Q3 * 32 + lane;
    const V *T0 = tb + c * kModalTabs * Q3;
    const int64_t qs[3] = {3 * nc, 3 * Q * nc, 3 * Q2 * nc};
    const int64_t d0 = c == 0 ? qs[0] : c == 1 ? qs[1] : qs[2], d1 = c == 0 ? qs[1] : c == 1 ? qs[2] : qs[0],
                  d2 = c == 0 ? qs[2] : c == 1 ? qs[0] : qs[1];
    V *zc = zk + c * nc + cell;
    auto store = [&](int k, int i, V v) {
        if (idx < ncells) zc[(i % Q) * d0 + (i / Q) * d1 + k * d2] = v;
    };
    Acc up[P >= 3 ? 3 : 1][Q2];  // what the planes below give the planes a2, a2 + 1, a2 + 2 along axis 2
#pragma unroll
    for (int k = 0; k < (P >= 3 ? 3 : 1); ++k)
#pragma unroll
        for (int i = 0; i < Q2; ++i) up[k][i] = A::zero();
    V keep[P >= 3 ? 2 : 1][Q2];  // transformed planes 0 .. P - 2 for the backward step of axis 2
#pragma unroll (A::kPlanes == 0 ? Q : A::kPlanes)
    for (int a2 = 0; a2 < Q; ++a2) {
        const V *T = T0 + a2 * Q2, *ow = own + a2 * Q2 * 32;
        Acc o[Q2];
#pragma unroll
        for (int i = 0; i < Q2; ++i) o[i] = up[0][i];
#pragma unroll
        for (int i = 0; i < Q2; ++i) {
            if constexpr (P >= 3) {
                up[0][i] = up[1][i];
                up[1][i] = up[2][i];
                up[2][i] = A::zero();
            } else {
                up[0][i] = A::zero();
            }
        }
#pragma unroll
        for (int i = 0; i < Q2; ++i) {
            const int a0 = i % Q, a1 = i / Q;
            const V *pj = fj + 32 * (a1 + Q * (a2 + Q * a0)), *pk = fk + 32 * (a2 + Q * (a0 + Q * a1));
            if (a0 < P) {
                Acc t = A::mul(T[i], modal_deriv<P, 32, A>(ow + 32 * i, a0));
                if (a1 < P) A::mac(t, T[Q3 + i], modal_deriv<P, 32, A>(pj, a1));
                if (a2 < P) A::mac(t, T[2 * Q3 + i], modal_deriv<P, 32, A>(pk, a2));
                modal_deriv_t<P, 1, A>(o + i, a0, A::get(t));
            }
            if (a1 < P) {
                Acc t = A::mul(T[3 * Q3 + i], modal_deriv<P, 32 * Q, A>(ow + 32 * i, a1));
                if (a0 < P) A::mac(t, T[4 * Q3 + i], modal_deriv<P, 32 * Q2, A>(pj, a0));
                modal_deriv_t<P, Q, A>(o + i, a1, A::get(t));
            }
            if (a2 < P) {
                Acc t = A::mul(T[5 * Q3 + i], modal_deriv<P, 32 * Q2, A>(ow + 32 * i, a2));
                if (a0 < P) A::mac(t, T[6 * Q3 + i], modal_deriv<P, 32 * Q, A>(pk, a0));
                const V v = A::get(t);
                if constexpr (P >= 3) A::add(up[0][i], v);
                else up[0][i] = t;
                if constexpr (P >= 3)
                    if (a2 == 0) A::mac(up[2][i], A::constant(kModalK3), v);
            }
        }
        V r[Q2];
#pragma unroll
        for (int i = 0; i < Q2; ++i) r[i] = A::get(o[i]);
#pragma unroll
        for (int i = 0; i < Q; ++i) modal_backward<P, Q, A>(r + i);
#pragma unroll
        for (int i = 0; i < Q; ++i) modal_backward<P, 1, A>(r + Q * i);
        // axis 2: hats from planes 0 and 1, bubble j = a2 from planes a2 and a2 - 2
        if (a2 == 0) {
#pragma unroll
            for (int i = 0; i < Q2; ++i) keep[0][i] = r[i];
        } else if (a2 == 1) {
#pragma unroll
            for (int i = 0; i < Q2; ++i) {
                Acc lo = A::start(keep[0][i]), hi = lo;
                A::add(lo, A::neg(r[i]));
                A::add(hi, r[i]);
                store(0, i, A::get(lo));
                store(P, i, A::get(hi));
                if constexpr (P >= 3) keep[1][i] = r[i];
            }
        } else {
            const V k = a2 == 2 ? A::constant(-kModalK2) : A::constant(-kModalK3);
#pragma unroll
            for (int i = 0; i < Q2; ++i) {
                Acc t = A::start(r[i]);
                V b = keep[0][i];
                if constexpr (P >= 3) b = a2 == 3 ? keep[1][i] : b;
                A::mac(t, k, b);
                store(a2 - 1, i, A::get(t));
            }
        }
    }
}

// y = K x from the slots: every lattice node adds the entries of the (up to 8) active cells that hold it, in a
// fixed order, so the result does not depend on the launch shape; entries that are not free become 0.
//
// A warp is 32 "cells" along x (c = n: the last node plane alone) of one lattice row: a thread owns the row's
// nodes p c .. p c + p - 1, so the slots are read in runs of consecutive cells, each entry once, and the
// row's results go through shared memory so that the stores are consecutive too.  All loads of a row are
// issued before the first addition (a row per warp and predicated loads instead of a loop over the rows of a
// cell with a branch per neighbour: 171 -> 88 us at 80^3 p = 2, 111 -> 40 us at 32^3 p = 3, where
// the slots (50 MB) stay in L2).  Loads bound it (long scoreboard; 48 % of the DRAM peak at 64^3 p = 2), in FP64 also
// its pipe (57 % at 32^3 p = 3).
constexpr int kSumWarps = 4;

template <int P, class A>
__global__ void __launch_bounds__(32 * kSumWarps)
    k_sum_kernel(const typename A::V *__restrict__ zk, const int32_t *__restrict__ cell_elem,
                 const uint8_t *__restrict__ mask, double *__restrict__ y, Grid3 g, int64_t nc,
                 const int *__restrict__ done)
{
    using V = typename A::V;
    constexpr int Q = P + 1, ROW = 3 * P;
    if (done && *done) return;
    __shared__ double row[kSumWarps][32 * ROW];
    const int lane = threadIdx.x, w = threadIdx.y;
    const unsigned nbx = (g.n[0] + 32) / 32, nby = (g.M[1] + kSumWarps - 1) / kSumWarps;
    const int bx = blockIdx.x % nbx, iy = (int)((blockIdx.x / nbx) % nby) * kSumWarps + w,
              iz = (int)(blockIdx.x / (nbx * nby));
    if (iy >= g.M[1]) return;  // uniform across the warp
    const int cx = bx * 32 + lane, cy = iy / P, ly = iy - P * cy, cz = iz / P, lz = iz - P * cz;
    typename A::Acc acc[ROW];
#pragma unroll
    for (int k = 0; k < ROW; ++k) acc[k] = A::zero();
#pragma unroll
    for (int dz = 1; dz >= 0; --dz) {  // cells one back first
        if (dz && lz > 0) continue;    // uniform across the warp, as the next
#pragma unroll
        for (int dy = 1; dy >= 0; --dy) {
            if (dy && ly > 0) continue;
            const int ay = cy - dy, az = cz - dz;
            if (ay < 0 || az < 0 || ay >= g.n[1] || az >= g.n[2]) continue;
            const int64_t at = cx + (int64_t)g.n[0] * (ay + (int64_t)g.n[1] * az);
            const bool on0 = cx < g.n[0] && cell_elem[at] >= 0, on1 = cx > 0 && cx <= g.n[0] && cell_elem[at - 1] >= 0;
            const V *zq = zk + at + (int64_t)3 * Q * ((ly + dy * P) + Q * (lz + dz * P)) * nc;
            V v1[3], v0[ROW];
#pragma unroll
            for (int k = 0; k < 3; ++k) v1[k] = on1 ? __ldcs(zq - 1 + (3 * P + k) * nc) : V{};
#pragma unroll
            for (int k = 0; k < ROW; ++k) v0[k] = on0 ? __ldcs(zq + k * nc) : V{};
#pragma unroll
            for (int k = 0; k < 3; ++k) A::add(acc[k], v1[k]);
#pragma unroll
            for (int k = 0; k < ROW; ++k) A::add(acc[k], v0[k]);
        }
    }
#pragma unroll
    for (int k = 0; k < ROW; ++k) row[w][lane * ROW + k] = A::to_double(A::get(acc[k]));
    __syncwarp();
    const int nrow = min(32 * ROW, 3 * g.M[0] - bx * 32 * ROW);
    const int64_t gi = 3 * ((int64_t)bx * 32 * P + g.M[0] * (iy + g.M[1] * (int64_t)iz));
    for (int k = lane; k < nrow; k += 32) y[gi + k] = mask[gi + k] ? row[w][k] : 0.0;
}

inline unsigned k_sum_blocks(const Grid3 &g)
{
    return (unsigned)((g.n[0] + 32) / 32) * (unsigned)((g.M[1] + kSumWarps - 1) / kSumWarps) * (unsigned)g.M[2];
}

}  // namespace fcm

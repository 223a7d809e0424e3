// Stiffness apply y = K x of the finite cell Schwarz-PCG on sm_103a (Sec. 2.1 Eq. (1)).
//
// Every active cell's product K_e x_e goes to a slot of its own (uncut cells matrix-free in Legendre modal
// form, cut cells with their dense element matrix on a second stream beside them), then one kernel adds the
// slots node by node (fcm_modal.cuh): three launches, no atomics, one fixed order of additions.  Eight
// parity colours that added into y in place took 16 dependent launches, which a small grid pays in latency
// (4^3 cells, K and S together: 119.8 us, 35.9 with the slots) and a large one in tails.  (The Schwarz apply is in fcm_schwarz.cu.)
#include <cuda_runtime.h>

#include <algorithm>

#include "fcm_device.cuh"
#include "fcm_modal.cuh"

namespace fcm {

namespace {

// Threads of the cut-cell product: PARTS column ranges of a row on different warps, so that a row's chain of
// FP64 multiply-adds is short (the FP64 pipe does 2 per clock per SM; one chain per row left a 4^3 grid's
// 34 cells waiting on latency).
__host__ __device__ constexpr int round32(int v) { return (v + 31) / 32 * 32; }
__host__ __device__ constexpr int ebe_parts(int P) { return P <= 2 ? 4 : P == 3 ? 2 : 1; }
__host__ __device__ constexpr int ebe_rows(int P) { return 3 * (P + 1) * (P + 1) * (P + 1); }
__host__ __device__ constexpr int ebe_threads(int P) { return round32(ebe_rows(P)) * ebe_parts(P); }

// Zk slots of the cut cells: K_e x_e with the cell's own dense matrix (symmetric: column t read as row t, so
// consecutive threads read consecutive entries).
template <int P>
__global__ void __launch_bounds__(ebe_threads(P))
    ebe_apply_kernel(const double *__restrict__ x, double *__restrict__ zk, const double *__restrict__ elem,
                     const CutCell *__restrict__ cells, Grid3 g, int64_t nc, const uint8_t *__restrict__ xmask,
                     const int *__restrict__ done)
{
    constexpr int Q = P + 1, NE = 3 * Q * Q * Q, R32 = round32(NE), PARTS = ebe_parts(P), JP = (NE + PARTS - 1) / PARTS;
    if (done && *done) return;
    __shared__ double xe[NE], part[PARTS > 1 ? (PARTS - 1) * NE : 1];
    const CutCell ce = cells[blockIdx.x];
    const double *xc = x + ce.base;
    for (int t = threadIdx.x; t < NE; t += blockDim.x) {
        const int l = t / 3, ix = l % Q, iy = (l / Q) % Q, iz = l / (Q * Q);
        const int64_t at = 3 * (ix + g.M[0] * (iy + (int64_t)g.M[1] * iz)) + t % 3;
        xe[t] = k_input(xc + at, xmask ? xmask + ce.base + at : nullptr);
    }
    __syncthreads();
    const int t = threadIdx.x % R32, pt = threadIdx.x / R32;
    double s = 0.0;
    if (t < NE) {
        const double *__restrict__ K = elem + (size_t)ce.elem * NE * NE + t;
        const int j1 = min(NE, (pt + 1) * JP);
#pragma unroll 8
        for (int j = pt * JP; j < j1; ++j) s = fma(__ldg(K + (size_t)j * NE), xe[j], s);
        if (pt > 0) part[(pt - 1) * NE + t] = s;
    }
    if constexpr (PARTS > 1) {
        __syncthreads();
        if (pt > 0 || t >= NE) return;
#pragma unroll
        for (int k = 0; k < PARTS - 1; ++k) s += part[k * NE + t];
    }
    if (t < NE) zk[t * nc + ce.cell] = s;
}

// Zk slots K_ref x_e of uncut cells, without the matrix, by sum factorisation (p = 4).  Each displacement
// component is interpolated to the (p+1)^3 Gauss points by one-dimensional contractions along
// x, y, z (sum factorisation); its gradient there follows from the collocation derivative on
// the Gauss points (exact: the field has degree <= p per axis).  The weighted stress
// sigma = lam tr(eps) I + 2 mu eps is formed per point, and the transposed steps give the
// nodal forces.  Exact for the uncut integrand (degree <= 2p per axis), so it equals
// K_ref x_e up to rounding, with 36 (p+1)^4 FP64 multiply-adds per cell (the dense product
// takes 9 (p+1)^6) and no matrix traffic.  Threads of a cell: one per point.
template <int P>
__global__ void __launch_bounds__(256)
    sf_apply_kernel(const double *__restrict__ x, double *__restrict__ zk, const int *__restrict__ cells, int ncells,
                    Grid3 g, int64_t nc, SfTables T, const int *__restrict__ done)
{
    constexpr int Q = P + 1, Q3 = Q * Q * Q, TPC = round32(Q3), CPC = 256 / TPC;
    if (done && *done) return;
    __shared__ double sB[Q][Q], sG[3][Q][Q], sW[Q];
    __shared__ double U[CPC][3][Q3];   // nodal values; then the point values per component
    __shared__ double A[CPC][Q3], Bq[CPC][Q3];
    for (int t = threadIdx.x; t < Q * Q; t += blockDim.x) {
        const int q = t / Q, i = t % Q;
        sB[q][i] = T.B[q][i];
        for (int a = 0; a < 3; ++a) sG[a][q][i] = T.G[a][q][i];
    }
    if (threadIdx.x < Q) sW[threadIdx.x] = T.W[threadIdx.x];
    const int lc = threadIdx.x / TPC, t = threadIdx.x % TPC;
    const int cidx = blockIdx.x * CPC + lc;
    const bool on = cidx < ncells && t < Q3;
    const int tx = t % Q, ty = (t / Q) % Q, tz = t / (Q * Q);
    int64_t node = 0;
    int cell = 0;
    if (on) {
        cell = cells[cidx];
        const int cx = cell % g.n[0], cy = (cell / g.n[0]) % g.n[1], cz = cell / (g.n[0] * g.n[1]);
        node = (P * cx + tx) + (int64_t)g.M[0] * ((P * cy + ty) + (int64_t)g.M[1] * (P * cz + tz));
        for (int c = 0; c < 3; ++c) U[lc][c][t] = x[3 * node + c];
    }
    __syncthreads();
    // interpolation to the points: (ix,iy,iz) -> (qx,iy,iz) -> (qx,qy,iz) -> (qx,qy,qz)
    double uq[3];
    for (int c = 0; c < 3; ++c) {
        if (on) {
            double s0 = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) s0 = fma(sB[tx][k], U[lc][c][k + Q * (ty + Q * tz)], s0);
            A[lc][t] = s0;
        }
        __syncthreads();
        if (on) {
            double s1 = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) s1 = fma(sB[ty][k], A[lc][tx + Q * (k + Q * tz)], s1);
            Bq[lc][t] = s1;
        }
        __syncthreads();
        if (on) {
            double s2 = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) s2 = fma(sB[tz][k], Bq[lc][tx + Q * (ty + Q * k)], s2);
            uq[c] = s2;
        }
    }
    __syncthreads();  // every point has read the nodal values of its cell
    if (on)
        for (int c = 0; c < 3; ++c) U[lc][c][t] = uq[c];
    __syncthreads();
    // gradients at the point by the collocation derivative along each axis
    double gr[3][3];
    if (on) {
        for (int c = 0; c < 3; ++c) {
            double gx = 0.0, gy = 0.0, gz = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                gx = fma(sG[0][tx][k], U[lc][c][k + Q * (ty + Q * tz)], gx);
                gy = fma(sG[1][ty][k], U[lc][c][tx + Q * (k + Q * tz)], gy);
                gz = fma(sG[2][tz][k], U[lc][c][tx + Q * (ty + Q * k)], gz);
            }
            gr[c][0] = gx;
            gr[c][1] = gy;
            gr[c][2] = gz;
        }
    }
    // weighted stress at the point: F[c][j] = w detJ (lam tr(eps) delta_cj + 2 mu eps_cj)
    double F[3][3];
    if (on) {
        const double w = sW[tx] * sW[ty] * sW[tz] * T.detJ;
        const double ltr = T.lam * (gr[0][0] + gr[1][1] + gr[2][2]);
        for (int c = 0; c < 3; ++c)
            for (int j = 0; j < 3; ++j) F[c][j] = w * (T.mu * (gr[c][j] + gr[j][c]) + (c == j ? ltr : 0.0));
    }
    double out[3];
    for (int c = 0; c < 3; ++c) {
        __syncthreads();  // the previous readers of U and A are done
        if (on)
            for (int j = 0; j < 3; ++j) U[lc][j][t] = F[c][j];
        __syncthreads();
        if (on) {  // transposed collocation derivative: point values of component c's force
            double v = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                v = fma(sG[0][k][tx], U[lc][0][k + Q * (ty + Q * tz)], v);
                v = fma(sG[1][k][ty], U[lc][1][tx + Q * (k + Q * tz)], v);
                v = fma(sG[2][k][tz], U[lc][2][tx + Q * (ty + Q * k)], v);
            }
            A[lc][t] = v;
        }
        __syncthreads();
        if (on) {  // z^T: (qx, qy, iz)
            double s2 = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) s2 = fma(sB[k][tz], A[lc][tx + Q * (ty + Q * k)], s2);
            Bq[lc][t] = s2;
        }
        __syncthreads();
        if (on) {  // y^T: (qx, iy, iz)
            double s1 = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) s1 = fma(sB[k][ty], Bq[lc][tx + Q * (k + Q * tz)], s1);
            A[lc][t] = s1;
        }
        __syncthreads();
        if (on) {  // x^T: nodal force (ix, iy, iz)
            double o = 0.0;
#pragma unroll
            for (int k = 0; k < Q; ++k) o = fma(sB[k][tx], A[lc][k + Q * (ty + Q * tz)], o);
            out[c] = o;
        }
    }
    if (on)
        for (int c = 0; c < 3; ++c) zk[(3 * t + c) * nc + cell] = out[c];
}

__global__ void mask_copy_kernel(const double *__restrict__ in, double *__restrict__ out,
                                 const uint8_t *__restrict__ mask, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = mask[i] ? in[i] : 0.0;
}

// p = 4: modal arrays of 125 modes do not fit a thread's registers; the dense-table form stays there.
template <int P>
void uncut_launch(const Grid3 &g, const double *x, double *zk, const KCells &kc, const int *done, cudaStream_t s)
{
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];
    if constexpr (P <= 3) {
        modal_apply_kernel<P, ModalF64><<<(kc.n_uncut + 31) / 32, kModalThreads, modal_smem_bytes(P), s>>>(
            x, zk, kc.uncut, kc.n_uncut, g, nc, kc.modal, done);
    } else {
        constexpr int CPC = 256 / round32((P + 1) * (P + 1) * (P + 1));
        sf_apply_kernel<P><<<(kc.n_uncut + CPC - 1) / CPC, 256, 0, s>>>(x, zk, kc.uncut, kc.n_uncut, g, nc, kc.sf, done);
    }
}

template <int P>
void k_launch(const Grid3 &g, const double *x, double *y, const uint8_t *mask, const double *elem, const KCells &kc,
              const uint8_t *xmask, const int *done, cudaStream_t s, const KStreams &ks)
{
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];
    double *zk = reinterpret_cast<double *>(kc.zk);
    const bool fork = ks.side && kc.n_uncut > 0 && kc.n_cut > 0;
    if (fork) {
        cudaEventRecord(ks.fork, s);
        cudaStreamWaitEvent(ks.side, ks.fork, 0);
    }
    if (kc.n_cut > 0)
        ebe_apply_kernel<P><<<kc.n_cut, ebe_threads(P), 0, fork ? ks.side : s>>>(x, zk, elem, kc.cut, g, nc, xmask, done);
    if (kc.n_uncut > 0) uncut_launch<P>(g, x, zk, kc, done, s);
    if (fork) {
        cudaEventRecord(ks.join, ks.side);
        cudaStreamWaitEvent(s, ks.join, 0);
    }
    k_sum_kernel<P, ModalF64><<<k_sum_blocks(g), dim3(32, kSumWarps), 0, s>>>(zk, kc.cell_elem, mask, y, g, nc, done);
}

template <int P>
cudaError_t k_prepare_p()
{
    if constexpr (P <= 3)
        return cudaFuncSetAttribute(modal_apply_kernel<P, ModalF64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    modal_smem_bytes(P));
    return cudaSuccess;
}

int grid_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

void launch_k_apply(int p, const Grid3 &g, const double *x, double *y, const uint8_t *mask, const double *elem,
                    const KCells &kc, const uint8_t *xmask, const int *done, cudaStream_t s, const KStreams &ks)
{
    switch (p) {
    case 1: k_launch<1>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 2: k_launch<2>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 3: k_launch<3>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 4: k_launch<4>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    default: break;
    }
}

void launch_mask_copy(const double *in, double *out, const uint8_t *mask, int64_t n, cudaStream_t s)
{
    mask_copy_kernel<<<grid_for(n, 256), 256, 0, s>>>(in, out, mask, n);
}

cudaError_t k_prepare(int p)
{
    switch (p) {
    case 1: return k_prepare_p<1>();
    case 2: return k_prepare_p<2>();
    case 3: return k_prepare_p<3>();
    default: return k_prepare_p<4>();
    }
}

void make_modal_tables(const double *h, double E, double nu, int p, std::vector<double> &tab)
{
    tab.clear();
    if (p > 3) return;  // dense tables (SfTables)
    const int q = p + 1, q3 = q * q * q;
    const double lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)), mu = E / (2.0 * (1.0 + nu));
    const double detJ = h[0] * h[1] * h[2] / 8.0;
    const double kap[4] = {1.0, 1.0, kModalK2, kModalK3}, rho[4] = {1.0, kModalK2, kModalK3, 0.0};
    tab.assign((size_t)3 * kModalTabs * q3, 0.0);
    for (int c = 0; c < 3; ++c) {
        const double H[3] = {2.0 / h[c], 2.0 / h[(c + 1) % 3], 2.0 / h[(c + 2) % 3]};
        double *T = tab.data() + (size_t)c * kModalTabs * q3;
        for (int i = 0; i < q3; ++i) {
            const int a[3] = {i % q, (i / q) % q, i / (q * q)};
            double own[3], mass[3], mix[3];  // per axis: both sides derived, neither, one
            for (int d = 0; d < 3; ++d) {
                own[d] = 2.0 * (2 * a[d] + 1) * rho[a[d]] * rho[a[d]];
                mass[d] = kap[a[d]] * kap[a[d]] * 2.0 / (2 * a[d] + 1);
                mix[d] = 2.0 * rho[a[d]] * kap[a[d]];
            }
            const double w = detJ / 64.0;
            const double A0 = w * H[0] * H[0] * own[0] * mass[1] * mass[2], A1 = w * H[1] * H[1] * own[1] * mass[0] * mass[2],
                         A2 = w * H[2] * H[2] * own[2] * mass[0] * mass[1];
            const double B1 = w * H[0] * H[1] * mix[0] * mix[1] * mass[2], B2 = w * H[0] * H[2] * mix[0] * mix[2] * mass[1];
            T[i] = (lam + 2.0 * mu) * A0;
            T[q3 + i] = lam * B1;
            T[2 * q3 + i] = lam * B2;
            T[3 * q3 + i] = mu * A1;
            T[4 * q3 + i] = mu * B1;
            T[5 * q3 + i] = mu * A2;
            T[6 * q3 + i] = mu * B2;
        }
    }
}

}  // namespace fcm

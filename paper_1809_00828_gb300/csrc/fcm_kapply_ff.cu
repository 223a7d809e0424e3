// Stiffness apply y = K x (Sec. 2.1 Eq. (1)) in double-float arithmetic on the FP32 pipe.
//
// The same steps as fcm_kernels.cu -- uncut cells in Legendre modal form, cut cells with their own dense
// element matrix, each into its slot of Zk, then one sum per lattice node -- with every FP64 multiply-add
// replaced by a compensated double-float one (fcm_ff.cuh): values and tables are float pairs (hi, lo), a
// product is Dekker's exact product by FMA plus the cross terms, sums run by TwoSum.  Each contraction is
// accurate to about 2^-46 relative, so K x agrees with the FP64 kernels to ~1e-13, while GB300's FP32 pipe
// (128 lanes per SM) replaces its FP64 pipe (2 multiply-adds per clock per SM).  x is read and split by
// integer operations; the slots hold float pairs, and one FP64 add per DOF is left.
#include <cuda_runtime.h>

#include "fcm_device.cuh"
#include "fcm_ff.cuh"
#include "fcm_modal.cuh"
#include "fcm_sym.cuh"

namespace fcm {

namespace {

__host__ __device__ constexpr int rnd32k(int v) { return (v + 31) / 32 * 32; }
__host__ __device__ constexpr int ebe_threads(int rows) { return rnd32k(rows) < 512 ? rnd32k(rows) : 512; }

// S + C += sum over k < n of a_k b_k for double-float operands
struct FFAcc {
    float S = 0.f, C = 0.f;
    __device__ __forceinline__ void add(float2 a, float2 b) { ff_fma(a.x, a.y, b.x, b.y, S, C); }
    __device__ __forceinline__ float2 get() const { return ff_norm(S, C); }
};

// Zk slots of the cut cells: K_e x_e, K_e stored as double-float pairs (symmetric; column t read as row t).
template <int P>
__global__ void __launch_bounds__(ebe_threads(3 * (P + 1) * (P + 1) * (P + 1)))
    ebe_apply_ff_kernel(const double *__restrict__ x, float2 *__restrict__ zk, const float2 *__restrict__ elem,
                        const CutCell *__restrict__ cells, Grid3 g, int64_t nc, const uint8_t *__restrict__ xmask,
                        const int *__restrict__ done)
{
    constexpr int Q = P + 1, NE = 3 * Q * Q * Q;
    if (done && *done) return;
    __shared__ float2 xe[NE];
    const CutCell ce = cells[blockIdx.x];
    for (int t = threadIdx.x; t < NE; t += blockDim.x) {
        const int l = t / 3, ix = l % Q, iy = (l / Q) % Q, iz = l / (Q * Q);
        const int64_t at = ce.base + 3 * (ix + g.M[0] * (iy + (int64_t)g.M[1] * iz)) + t % 3;
        xe[t] = split_ff(k_input(x + at, xmask ? xmask + at : nullptr));
    }
    __syncthreads();
    const float2 *__restrict__ K = elem + (size_t)ce.elem * NE * NE;
    for (int t = threadIdx.x; t < NE; t += blockDim.x) {
        FFAcc s;
#pragma unroll 8
        for (int j = 0; j < NE; ++j) s.add(__ldcs(K + (size_t)j * NE + t), xe[j]);
        zk[t * nc + ce.cell] = s.get();
    }
}

// The same for p <= 2, K_e folded (fcm_sym.cuh): half of the matrix's bytes.  The issue slots
// bound it now (12 operations per entry and 8 around them; ncu, 64^3: 79 % of them busy, 63 % of the DRAM peak):
// 370 us for 72,180 cells (1.92 GB, 285 us at the copy rate) where streaming the full matrices took 697 us (3.8 GB).
template <int P>
__global__ void __launch_bounds__(ebe_threads(3 * (P + 1) * (P + 1) * (P + 1)))
    ebe_fold_ff_kernel(const double *__restrict__ x, float2 *__restrict__ zk, const float2 *__restrict__ elem,
                       const CutCell *__restrict__ cells, Grid3 g, int64_t nc, const uint8_t *__restrict__ xmask,
                       int *err, int wait_tries, const int *__restrict__ done)
{
    constexpr int Q = P + 1, NE = 3 * Q * Q * Q;
    if (done && *done) return;
    __shared__ __align__(16) float2 xe[(NE + 3) / 4 * 4], m[fold_entries(NE)];
    static_assert(sizeof(xe) + sizeof(m) + 1024 <= 48 * 1024, "static shared memory");
    __shared__ uint64_t bar;
    const CutCell ce = cells[blockIdx.x];
    const int t = threadIdx.x, l = t / 3, ix = l % Q, iy = (l / Q) % Q, iz = l / (Q * Q);
    if (t == 0) {
        mbar_init(&bar);
        mbar_expect(&bar, fold_entries(NE) * 8);
        bulk_g2s(m, elem + (size_t)ce.elem * fold_entries(NE), fold_entries(NE) * 8, &bar);
    }
    if (t < NE) {
        const int64_t at = ce.base + 3 * (ix + g.M[0] * (iy + (int64_t)g.M[1] * iz)) + t % 3;
        xe[t] = split_ff(k_input(x + at, xmask ? xmask + at : nullptr));
    }
    __syncthreads();
    if (!mbar_wait(&bar, 0, wait_tries)) {
        atomicExch(err, kErrElement);
        mbar_wait(&bar, 0, kDrainTries);
        return;
    }
    float S[1] = {0.f}, C[1] = {0.f};
    fold_dot<NE, 1>(m, NE, t & ~31, min(t, NE - 1), xe, S, C);
    if (t < NE) zk[t * nc + ce.cell] = ff_norm(S[0], C[0]);
}

// Zk slots K_ref x_e of the uncut cells (p = 4), matrix-free: the steps of sf_apply_kernel
// (interpolation to the Gauss points by 1D contractions, collocation derivative, weighted stress,
// transposed steps) in double-float arithmetic.  One thread per point (and node) of a cell.
template <int P>
__global__ void __launch_bounds__(256)
    sf_apply_ff_kernel(const double *__restrict__ x, float2 *__restrict__ zk, const int *__restrict__ cells, int ncells,
                       Grid3 g, int64_t nc, SfTablesFF T, const int *__restrict__ done)
{
    constexpr int Q = P + 1, Q3 = Q * Q * Q, TPC = rnd32k(Q3), CPC = 256 / TPC;
    if (done && *done) return;
    __shared__ float2 sB[Q][Q], sG[3][Q][Q], sW[Q];
    __shared__ float2 U[CPC][3][Q3];  // nodal values; then the point values per component
    __shared__ float2 A[CPC][Q3], Bq[CPC][Q3];
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
        for (int c = 0; c < 3; ++c) U[lc][c][t] = split_ff(x[3 * node + c]);
    }
    __syncthreads();
    // interpolation to the points: (ix,iy,iz) -> (qx,iy,iz) -> (qx,qy,iz) -> (qx,qy,qz)
    float2 uq[3];
    for (int c = 0; c < 3; ++c) {
        if (on) {
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[tx][k], U[lc][c][k + Q * (ty + Q * tz)]);
            A[lc][t] = s.get();
        }
        __syncthreads();
        if (on) {
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[ty][k], A[lc][tx + Q * (k + Q * tz)]);
            Bq[lc][t] = s.get();
        }
        __syncthreads();
        if (on) {
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[tz][k], Bq[lc][tx + Q * (ty + Q * k)]);
            uq[c] = s.get();
        }
    }
    __syncthreads();  // every point has read the nodal values of its cell
    if (on)
        for (int c = 0; c < 3; ++c) U[lc][c][t] = uq[c];
    __syncthreads();
    // gradients at the point by the collocation derivative along each axis
    float2 gr[3][3];
    if (on) {
        for (int c = 0; c < 3; ++c) {
            FFAcc gx, gy, gz;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                gx.add(sG[0][tx][k], U[lc][c][k + Q * (ty + Q * tz)]);
                gy.add(sG[1][ty][k], U[lc][c][tx + Q * (k + Q * tz)]);
                gz.add(sG[2][tz][k], U[lc][c][tx + Q * (ty + Q * k)]);
            }
            gr[c][0] = gx.get();
            gr[c][1] = gy.get();
            gr[c][2] = gz.get();
        }
    }
    // weighted stress at the point: F[c][j] = w detJ (lam tr(eps) delta_cj + mu (g_cj + g_jc))
    float2 F[3][3];
    if (on) {
        const float2 w = ff_mul(ff_mul(ff_mul(sW[tx], sW[ty]), sW[tz]), T.detJ);
        const float2 ltr = ff_mul(T.lam, ff_addv(ff_addv(gr[0][0], gr[1][1]), gr[2][2]));
        for (int c = 0; c < 3; ++c)
            for (int j = 0; j < 3; ++j) {
                float2 v = ff_mul(T.mu, ff_addv(gr[c][j], gr[j][c]));
                if (c == j) v = ff_addv(v, ltr);
                F[c][j] = ff_mul(w, v);
            }
    }
    float2 out[3];
    for (int c = 0; c < 3; ++c) {
        __syncthreads();  // the previous readers of U and A are done
        if (on)
            for (int j = 0; j < 3; ++j) U[lc][j][t] = F[c][j];
        __syncthreads();
        if (on) {  // transposed collocation derivative: point values of component c's force
            FFAcc v;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                v.add(sG[0][k][tx], U[lc][0][k + Q * (ty + Q * tz)]);
                v.add(sG[1][k][ty], U[lc][1][tx + Q * (k + Q * tz)]);
                v.add(sG[2][k][tz], U[lc][2][tx + Q * (ty + Q * k)]);
            }
            A[lc][t] = v.get();
        }
        __syncthreads();
        if (on) {  // z^T: (qx, qy, iz)
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[k][tz], A[lc][tx + Q * (ty + Q * k)]);
            Bq[lc][t] = s.get();
        }
        __syncthreads();
        if (on) {  // y^T: (qx, iy, iz)
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[k][ty], Bq[lc][tx + Q * (k + Q * tz)]);
            A[lc][t] = s.get();
        }
        __syncthreads();
        if (on) {  // x^T: nodal force (ix, iy, iz)
            FFAcc s;
#pragma unroll
            for (int k = 0; k < Q; ++k) s.add(sB[k][tx], A[lc][k + Q * (ty + Q * tz)]);
            out[c] = s.get();
        }
    }
    if (on)
        for (int c = 0; c < 3; ++c) zk[(3 * t + c) * nc + cell] = out[c];
}

template <int P>
void uncut_launch_ff(const Grid3 &g, const double *x, float2 *zk, const KCells &kc, const int *done, cudaStream_t s)
{
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];
    if constexpr (P <= 3) {
        modal_apply_kernel<P, ModalFF><<<(kc.n_uncut + 31) / 32, kModalThreads, modal_smem_bytes(P), s>>>(
            x, zk, kc.uncut, kc.n_uncut, g, nc, kc.modal_ff, done);
    } else {
        constexpr int CPC = 256 / rnd32k((P + 1) * (P + 1) * (P + 1));
        sf_apply_ff_kernel<P><<<(kc.n_uncut + CPC - 1) / CPC, 256, 0, s>>>(x, zk, kc.uncut, kc.n_uncut, g, nc, kc.sff,
                                                                          done);
    }
}

template <int P>
void k_launch_ff(const Grid3 &g, const double *x, double *y, const uint8_t *mask, const float2 *elem,
                 const KCells &kc, const uint8_t *xmask, const int *done, cudaStream_t s, const KStreams &ks)
{
    constexpr int NE = 3 * (P + 1) * (P + 1) * (P + 1);
    const int64_t nc = (int64_t)g.n[0] * g.n[1] * g.n[2];
    float2 *zk = reinterpret_cast<float2 *>(kc.zk);
    // the cut cells (HBM-bound) run beside the uncut ones (FP32-pipe bound)
    const bool fork = ks.side && kc.n_uncut > 0 && kc.n_cut > 0;
    if (fork) {
        cudaEventRecord(ks.fork, s);
        cudaStreamWaitEvent(ks.side, ks.fork, 0);
    }
    if (kc.n_cut > 0) {
        if constexpr (P <= 2)
            ebe_fold_ff_kernel<P><<<kc.n_cut, ebe_threads(NE), 0, fork ? ks.side : s>>>(x, zk, elem, kc.cut, g, nc, xmask,
                                                                                     kc.err, kc.wait_tries, done);
        else
            ebe_apply_ff_kernel<P><<<kc.n_cut, ebe_threads(NE), 0, fork ? ks.side : s>>>(x, zk, elem, kc.cut, g, nc, xmask,
                                                                                      done);
    }
    if (kc.n_uncut > 0) uncut_launch_ff<P>(g, x, zk, kc, done, s);
    if (fork) {
        cudaEventRecord(ks.join, ks.side);
        cudaStreamWaitEvent(s, ks.join, 0);
    }
    k_sum_kernel<P, ModalFF><<<k_sum_blocks(g), dim3(32, kSumWarps), 0, s>>>(zk, kc.cell_elem, mask, y, g, nc, done);
}

template <int P>
cudaError_t k_prepare_ff_p()
{
    if constexpr (P <= 3)
        return cudaFuncSetAttribute(modal_apply_kernel<P, ModalFF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    modal_smem_bytes(P));
    return cudaSuccess;
}

int grid_of(int64_t n)
{
    const int64_t b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : b < 152 * 16 ? b : 152 * 16);
}

// FP64 values -> double-float pairs
__global__ void to_ff_pairs_kernel(const double *__restrict__ in, float2 *__restrict__ out, int64_t n)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = split_ff(in[e]);
}

// the same with every ne x ne matrix folded (padding entries 0)
__global__ void fold_ff_pairs_kernel(const double *__restrict__ in, float2 *__restrict__ out, int ne, int64_t n)
{
    const int fe = fold_entries(ne), hw = fold_h(ne) * fold_w(ne);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * fe; e += (int64_t)gridDim.x * blockDim.x) {
        int i, j;
        const bool on = fold_entry(ne, (int)(e % fe), i, j) && (int)(e % fe) < hw;
        out[e] = on ? split_ff(in[e / fe * ne * ne + (int64_t)i * ne + j]) : make_float2(0.f, 0.f);
    }
}

}  // namespace

void launch_k_apply_ff(int p, const Grid3 &g, const double *x, double *y, const uint8_t *mask, const float2 *elem,
                       const KCells &kc, const uint8_t *xmask, const int *done, cudaStream_t s, const KStreams &ks)
{
    switch (p) {
    case 1: k_launch_ff<1>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 2: k_launch_ff<2>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 3: k_launch_ff<3>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    case 4: k_launch_ff<4>(g, x, y, mask, elem, kc, xmask, done, s, ks); break;
    default: break;
    }
}

cudaError_t k_prepare_ff(int p)
{
    switch (p) {
    case 1: return k_prepare_ff_p<1>();
    case 2: return k_prepare_ff_p<2>();
    case 3: return k_prepare_ff_p<3>();
    default: return k_prepare_ff_p<4>();
    }
}

void launch_to_ff_pairs(const double *in, float2 *out, int64_t n, cudaStream_t s)
{
    to_ff_pairs_kernel<<<grid_of(n), 256, 0, s>>>(in, out, n);
}

int64_t element_ff_entries(int p, int64_t nelem)
{
    const int ne = 3 * (p + 1) * (p + 1) * (p + 1);
    return nelem * (p <= 2 ? fold_entries(ne) : ne * ne);
}

void launch_element_ff(int p, const double *in, float2 *out, int64_t nelem, cudaStream_t s)
{
    const int ne = 3 * (p + 1) * (p + 1) * (p + 1);
    if (p <= 2)
        fold_ff_pairs_kernel<<<grid_of(element_ff_entries(p, nelem)), 256, 0, s>>>(in, out, ne, nelem);
    else
        launch_to_ff_pairs(in, out, nelem * ne * ne, s);
}

void make_sf_tables_ff(const SfTables &T, SfTablesFF &F)
{
    auto sp = [](double v) {
        const float h = (float)v;
        return make_float2(h, (float)(v - (double)h));
    };
    for (int q = 0; q < 5; ++q) {
        F.W[q] = sp(T.W[q]);
        for (int i = 0; i < 5; ++i) {
            F.B[q][i] = sp(T.B[q][i]);
            for (int a = 0; a < 3; ++a) F.G[a][q][i] = sp(T.G[a][q][i]);
        }
    }
    F.detJ = sp(T.detJ);
    F.lam = sp(T.lam);
    F.mu = sp(T.mu);
}

}  // namespace fcm

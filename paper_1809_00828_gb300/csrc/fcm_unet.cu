// Learned coarse correction: a 3D U-Net on the cell grid with hand-written
// CUDA kernels for inference and training (BF16 weights, FP32 activations
// and accumulation), the restriction / prolongation between lattice DOFs
// and cells, and Adam.  The paper's Additive-Schwarz preconditioner has no
// coarse space (Sec. 6 lists this as a limitation of local preconditioners);
// this network supplies one, used by fcm_fpcg_solve.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "fcm_device.cuh"
#include "fcm_ff.cuh"
#include "fcm_tma.cuh"

namespace fcm {
namespace {

// ---- 3x3x3 convolution on the tensor cores
//
// out[b][co][p] = bias[co] + sum_{ci, tap} w[co][ci][tap] in[b][ci][p + off(tap)], zero padding, as a product
// D[voxel][co] += A[voxel][ci] B[co][ci] per tap (tcgen05 kind::f16, BF16 operands, FP32 accumulators in tensor
// memory).  The weights are BF16; an FP32 activation is the exact sum of three BF16 values (8 significant bits
// each, cut from the top), so three products give what FP32 multiplications of the same weights give.
//
// A CTA makes 8 x 16 x ZT voxels (x, y, z) of up to 64 output channels.  Per 16 input channels it writes the
// tile with its halo of one voxel to shared memory, [split][8 channels][z][y][x] with 16 bytes per voxel:
// eight voxels along x are a core matrix of the canonical K-major layout without swizzle and a row of them a
// fixed stride, so each of the 27 taps is the same tile at another start address, and no input is gathered
// twice.  A halo plane goes through the taps of up to three output planes in one product (N up to 3 x the
// columns: the accumulators of the tile's planes lie side by side): an MMA takes 48 clocks for N <= 96 and N / 2
// beyond, so 27 (ZT + 2) of them per 16 input channels are cheaper than 81 ZT narrow ones.  Two CTAs of 512 threads
// per SM overlap one's halo loads (latency-bound: 16 warps rather than 8 took the forward pass from 0.85 to 0.75
// ms) with the other's products (half of the time).  Forward pass on 80^3 cells, channels 16 to 64 (75 GFLOP of
// convolutions): 0.75 ms; 1.19 ms with a product per plane, and 5.76 ms with FP32 arithmetic on the CUDA cores (13
// TFLOP/s).
//
// The tensor core adds into its FP32 accumulators by truncation: with one accumulator over all 81 products of
// 16 input channels the outputs were 5.6e-6 off (relative, 2-norm), 10 times the FP32 multiply-adds' error.  So
// the leading parts of each plane of taps (dz) have an accumulator of their own, the two small parts share a
// fourth, and after every 16 channels the four are added in registers with rounding to nearest.  That is also
// four independent chains of products instead of one.
//
// Around it, the loader reads the decoder's concatenation from its two sources (upsampled and skip), the
// gradient through a ReLU from the gradient and the ReLU's output, and the epilogue adds the bias and applies
// the ReLU: no pass over an activation is left between two convolutions but the pooling.
constexpr int kConvThreads = 512;
constexpr int kTX = 8, kTY = 16, kHX = kTX + 2, kHY = kTY + 2;
constexpr int kCoMax = 64;   // output channels of a CTA

__host__ __device__ constexpr int conv_hv(int ZT) { return kHX * kHY * (ZT + 2); }        // voxels with halo
__host__ __device__ constexpr int conv_a_bytes(int ZT) { return 3 * 2 * 16 * conv_hv(ZT); }
__host__ __device__ constexpr int conv_smem(int ZT, int nb) { return 1024 + conv_a_bytes(ZT) + 27 * 32 * nb; }
__host__ __device__ constexpr int up16(int n) { return (n + 15) / 16 * 16; }
// A halo plane i reaches the tile's planes z = i - 2 + s in [0, ZT) by the taps of dz = 2 - s ("slots" s): first slot,
// number of slots, and slots of the planes before it
__host__ __device__ constexpr int conv_s0(int i) { return i < 2 ? 2 - i : 0; }
__host__ __device__ constexpr int conv_ns(int ZT, int i) { return (ZT + 1 - i < 2 ? ZT + 1 - i : 2) - conv_s0(i) + 1; }
__host__ __device__ constexpr int conv_at(int ZT, int i)
{
    int n = 0;
    for (int k = 0; k < i; ++k) n += conv_ns(ZT, k);
    return n;
}
// columns (output channels) of a CTA, CTAs per voxel tile, and BF16 entries of a layer's weight tiles
__host__ __device__ constexpr int conv_nb(int n) { return n <= kCoMax ? up16(n) : kCoMax; }
__host__ __device__ constexpr int conv_blocks(int n) { return (n + kCoMax - 1) / kCoMax; }
__host__ __device__ constexpr int64_t conv_tile_entries(int cin, int cout)
{
    return (int64_t)conv_blocks(cout) * (up16(cin) / 16) * 27 * 16 * conv_nb(cout);
}

// Source of a convolution or of its weight gradient: channels 0 .. c0 - 1 at half resolution (nearest
// upsampling), then those of `full`, set to 0 where the same entry of `gate` is not positive (gate may be null).
struct ConvSrc {
    const float *half, *full, *gate;
    int c0, c1;
};

__device__ __forceinline__ float conv_load(const ConvSrc &s, int b, int ci, int x, int y, int z, int nx, int ny, int nz)
{
    if (ci < s.c0) {
        const int hx = nx >> 1, hy = ny >> 1, hz = nz >> 1;
        return __ldg(s.half + (((int64_t)b * s.c0 + ci) * hz + (z >> 1)) * hy * hx + (y >> 1) * hx + (x >> 1));
    }
    const int64_t at = (((int64_t)b * s.c1 + ci - s.c0) * nz + z) * ny * nx + (int64_t)y * nx + x;
    const float v = __ldg(s.full + at);
    return s.gate && !(__ldg(s.gate + at) > 0.f) ? 0.f : v;
}

// x = hi + mid + lo, each with 8 significant bits in its upper half word; infinities and NaN in hi alone
__device__ __forceinline__ void split3(float x, uint32_t &hi, uint32_t &mid, uint32_t &lo)
{
    const uint32_t u = __float_as_uint(x);
    hi = u & 0xFFFF0000u;
    const float r = __fsub_rn(x, __uint_as_float(hi));
    mid = __float_as_uint(r) & 0xFFFF0000u;
    lo = __float_as_uint(__fsub_rn(r, __uint_as_float(mid)));
    if ((u & 0x7F800000u) == 0x7F800000u) {
        if (u & 0x7FFFFFu) hi |= 0x00400000u;
        mid = lo = 0u;
    }
}

// A convolution's wait for the tensor core: polls before it gives up, and the flags it then sets: `err` (device) to
// `code`, `seen` (pinned host memory, may be null) to 1.
struct ConvWait {
    int *err, *seen;
    int code, tries;
};

template <int ZT>
__global__ void __launch_bounds__(kConvThreads, 2)
    conv3_tc_kernel(ConvSrc src, const uint4 *__restrict__ w, const float *__restrict__ bias, float *__restrict__ out,
                    int cin, int cout, int nx, int ny, int nz, int relu, ConvWait wait)
{
    constexpr int HV = conv_hv(ZT);
    extern __shared__ __align__(1024) unsigned char csm[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(csm);
    uint32_t *slot = reinterpret_cast<uint32_t *>(csm + 8);
    volatile int *gave_up = reinterpret_cast<int *>(csm + 12);  // the 16 channels at which a wait ran out, else nch
    unsigned char *A = csm + 1024, *W = A + conv_a_bytes(ZT);
    const int nb = conv_nb(cout), nch = up16(cin) / 16;
    const int tx = (nx + kTX - 1) / kTX, ty = (ny + kTY - 1) / kTY;
    const int x0 = (blockIdx.x % tx) * kTX, y0 = (blockIdx.x / tx % ty) * kTY, z0 = (blockIdx.x / (tx * ty)) * ZT;
    const int b = blockIdx.z, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t S = (int64_t)nx * ny * nz, S2 = (int64_t)(nx >> 1) * (ny >> 1) * (nz >> 1);
    const uint32_t cols = 4 * ZT * nb <= 64 ? 64 : 4 * ZT * nb <= 128 ? 128 : 256;
    if (tid == 0) {
        mbar_init(bar);
        *gave_up = nch;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *slot;
    // warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (rows y of four, 8 voxels along x each) of item w / 4:
    // (z, 16 channels)
    const int items = ZT * (nb / 16), it = warp >> 2, zi = it / (nb / 16), col = it % (nb / 16) * 16;
    float sum[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) sum[k] = 0.f;
    for (int ch = 0; ch < nch; ++ch) {
        for (int e = tid; e < 2 * HV; e += kConvThreads) {
            const int kc = e >= HV, v = e - kc * HV, hx = v % kHX, hy = v / kHX % kHY, hz = v / (kHX * kHY);
            const int x = x0 + hx - 1, y = y0 + hy - 1, z = z0 + hz - 1;
            const bool in = x >= 0 && y >= 0 && z >= 0 && x < nx && y < ny && z < nz;
            const int ci = 16 * ch + 8 * kc;
            float f[8];
            if (in && ci >= src.c0 && ci + 8 <= cin) {
                const int64_t at = ((int64_t)b * src.c1 + ci - src.c0) * S + ((int64_t)z * ny + y) * nx + x;
                const float *p = src.full + at;
#pragma unroll
                for (int k = 0; k < 8; ++k) f[k] = __ldg(p + k * S);
                if (src.gate) {
                    const float *q = src.gate + at;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (!(__ldg(q + k * S) > 0.f)) f[k] = 0.f;
                }
            } else if (in && ci + 8 <= src.c0) {
                const float *p = src.half + ((int64_t)b * src.c0 + ci) * S2 + ((int64_t)(z >> 1) * (ny >> 1) + (y >> 1)) * (nx >> 1) + (x >> 1);
#pragma unroll
                for (int k = 0; k < 8; ++k) f[k] = __ldg(p + k * S2);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) f[k] = in && ci + k < cin ? conv_load(src, b, ci + k, x, y, z, nx, ny, nz) : 0.f;
            }
            uint32_t s[3][8];
#pragma unroll
            for (int k = 0; k < 8; ++k) split3(f[k], s[0][k], s[1][k], s[2][k]);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                uint4 o;  // the upper half words, channel k at bytes 2 k
                o.x = __byte_perm(s[q][0], s[q][1], 0x7632);
                o.y = __byte_perm(s[q][2], s[q][3], 0x7632);
                o.z = __byte_perm(s[q][4], s[q][5], 0x7632);
                o.w = __byte_perm(s[q][6], s[q][7], 0x7632);
                reinterpret_cast<uint4 *>(A)[(2 * q + kc) * HV + v] = o;
            }
        }
        const uint4 *wc = w + ((int64_t)blockIdx.y * nch + ch) * 27 * 2 * nb;
        for (int e = tid; e < 27 * 2 * nb; e += kConvThreads) reinterpret_cast<uint4 *>(W)[e] = __ldg(wc + e);
        // the tensor core reads shared memory through the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (*gave_up < ch) break;  // the same for all threads: what they write below is at least ch
        if (warp == 0 && tc_elect()) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // FP32 accumulator, BF16 A and B, both K-major, M = 128, N = nb .. 3 nb
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24), in8 = (uint32_t)(nb >> 3) << 17;
            const uint64_t a0 = smem_desc(smem_u32(A), 16 * HV, 16 * kHX);
            uint64_t bt = smem_desc(smem_u32(W), 128, 256);
            const uint32_t small = tmem + 3 * ZT * nb;
#pragma unroll
            for (int t = 0; t < 9; ++t, bt += 6 * nb)
#pragma unroll
                for (int q = 2; q >= 0; --q)
#pragma unroll
                    for (int k = 0; k < ZT + 2; ++k) {
                        // planes 2, 5, .. first: together they write each small accumulator once
                        constexpr int n3 = (ZT + 2) / 3;
                        const int i = k < n3 ? 3 * k + 2 : (k - n3) / 2 * 3 + (k - n3) % 2;
                        const uint64_t ad = a0 + (uint64_t)(2 * q * HV + i * kHX * kHY + t / 3 * kHX + t % 3);
                        const uint64_t bd = bt + (uint64_t)(2 * conv_s0(i) * nb);
                        const uint32_t id = idesc + conv_ns(ZT, i) * in8;
                        if (q == 0) tc_mma_bf16(tmem + conv_at(ZT, i) * nb, ad, bd, id, t > 0);
                        else tc_mma_bf16(small + (i < 2 ? 0 : i - 2) * nb, ad, bd, id, t > 0 || q < 2 || k >= n3);
                    }
            tc_commit(bar);
        }
        __syncwarp();
        if (!mbar_wait(bar, ch & 1, wait.tries)) {
            *gave_up = ch;
            atomicExch(wait.err, wait.code);
            if (wait.seen) *reinterpret_cast<volatile int *>(wait.seen) = 1;
            mbar_wait(bar, ch & 1, kDrainTries);  // the products still in flight land before the CTA leaves
        }
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (it < items) {  // uniform across the warp
            const uint32_t at = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + col;
            float part[16];
#pragma unroll
            for (int q = 3; q >= 0; --q) {
                int blk = 3 * ZT + zi;  // the small parts, then the leading ones of dz = 2, 1, 0
                if (q < 3) {
                    blk = 2 - q - conv_s0(zi + q);
                    for (int k = 0; k < zi + q; ++k) blk += conv_ns(ZT, k);
                }
                uint32_t v[16];
                tc_load16(at + blk * nb, v);
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    part[k] = q == 3 ? __uint_as_float(v[k]) : __fadd_rn(part[k], __uint_as_float(v[k]));
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[k] = __fadd_rn(sum[k], part[k]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    const int vx = x0 + (lane & 7), vy = y0 + 4 * (warp & 3) + (lane >> 3), vz = z0 + zi;
    if (it < items && vx < nx && vy < ny && vz < nz) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int co = blockIdx.y * kCoMax + col + k;
            if (co < cout) {
                float f = sum[k];
                if (bias) f = __fadd_rn(f, bias[co]);
                if (relu) f = fmaxf(f, 0.f);
                out[((int64_t)b * cout + co) * S + ((int64_t)vz * ny + vy) * nx + vx] = f;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// Weight tiles of every layer in the tensor core's layout, from the FP32 weights w[co][ci][27] rounded to BF16: per
// block of 64 output channels, 16 input channels, (dy, dx) and slot 2 - dz, [channel / 8][K / 8][8 channels][8 K] (zeros
// beyond the layer).  Two sets per layer, one after the other: those of the layer, and those of the data-gradient
// convolution, w'[ci][co][26 - tap].  One launch for all of them: an Adam step on four levels takes 23 us with its
// update, 142 with a conversion and two launches per layer.
constexpr int kMaxConv = 6 * 2 + 5 * 2 + 1;
struct TileTable {
    int64_t at[2 * kMaxConv];  // first entry of each set; a set is a multiple of 256 entries
    int64_t woff[kMaxConv];
    int cin[kMaxConv], cout[kMaxConv];
    int sets;
};
static_assert(27 * 16 * 16 % 256 == 0, "a CTA's entries are of one set");

__global__ void __launch_bounds__(256)
    weight_tiles_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ t, const __grid_constant__ TileTable tab)
{
    const int64_t first = blockIdx.x * (int64_t)256;
    int s = 0;
#pragma unroll
    for (int step = 32; step > 0; step >>= 1)
        if (s + step < tab.sets && tab.at[s + step] <= first) s += step;
    const bool flip = s & 1;
    const int cin = flip ? tab.cout[s >> 1] : tab.cin[s >> 1], cout = flip ? tab.cin[s >> 1] : tab.cout[s >> 1];
    const int nb = conv_nb(cout), nch = up16(cin) / 16;
    const unsigned e = (unsigned)(first - tab.at[s]) + threadIdx.x;
    const int k = (int)(e & 7), r = (int)(e >> 3 & 7), kc = (int)(e >> 6 & 1);
    unsigned q = e >> 7;
    const int n8 = (int)(q % (nb / 8));
    q /= nb / 8;
    const int tap = 9 * (2 - (int)(q % 3)) + (int)(q / 3 % 9);
    q /= 27;
    const int ci = 16 * (int)(q % nch) + 8 * kc + k, co = kCoMax * (int)(q / nch) + 8 * n8 + r;
    const float *wl = w + tab.woff[s >> 1];
    float v = 0.f;
    if (ci < cin && co < cout) v = flip ? wl[((int64_t)ci * cout + co) * 27 + 26 - tap] : wl[((int64_t)co * cin + ci) * 27 + tap];
    t[first + threadIdx.x] = __float2bfloat16_rn(v);
}

// ---- weight gradients: gw[co][ci][tap] += sum_{b,p} gout[b][co][p] in[b][ci][p + off(tap)], gb[co] += sum gout
//
// A CTA owns 16 output x 8 input channels and walks tiles of 8 x 8 x 4 voxels; a thread owns two output channels
// and one input channel of one plane of the tile, with their 27 taps (and the bias) in registers: eight voxels
// along x cost 31 vector reads of shared memory and 448 multiply-adds (one output channel and four voxels a time
// cost 19 reads for 112).  The tiles are dealt to enough CTAs to fill the GPU, each
// writes its sums to `part`, and wgrad_sum_kernel adds them in a fixed order in FP64 (deterministic).  The more
// channels a layer has, the fewer CTAs share a channel pair's voxels (with 256 x 256 channels one), so every `fold`
// tiles the registers' FP32 sums are added to float pairs in shared memory: no chain of FP32 additions is longer
// than 64 or a 256th of the voxels (wgrad_fold), whatever the layer.  With chains over all of a CTA's voxels the gradients
// of a 256 -> 256 layer on 32^3 voxels were 9.4e-7 off (2-norm), now 1.2e-7, and those of 192 -> 64 on 48^3 3.7e-6,
// now 0.8e-6; the folds take 0.6 % of a training step.  Half of the
// instructions of a first version went into the indices of the tiles' loads: a thread now keeps its point of the
// tile and walks channels and planes, all 24 + 16 loads in flight.  One CTA per
// (co, ci) pair with 27 unshared global reads per multiply-add row took 4.9 ms for the gradients of the
// 16-to-64-channel network on four 32^3 cubes, one channel a thread 1.08 + 0.29 ms; this 0.73 + 0.12 ms.
constexpr int kWC = 8, kWO = 16, kWX = 8, kWY = 8, kWZ = 4, kWGo = kWX * kWY * kWZ + 4;
constexpr int kWRow = 12, kWPlane = kWRow * (kWY + 2), kWCh = kWPlane * (kWZ + 2) + 4;  // 4 channels: distinct banks
constexpr int kWTaps = 28, kWRun = 64 * 2 * kWTaps * 8 /* bytes of the running sums */, kHaloXY = (kWX + 2) * (kWY + 2);
constexpr int kSumParts = 16;  // parts of the slabs that wgrad_sum_kernel adds side by side

__global__ void __launch_bounds__(256, 2)
    conv3_wgrad_kernel(ConvSrc in, ConvSrc go, int cin, int cout, int B, int nx, int ny, int nz, int fold,
                       float *__restrict__ part)
{
    extern __shared__ float2 run[];  // running sums, [2 x 28][64 threads] (where a CTA folds more than once)
    __shared__ __align__(16) float si[kWC * kWCh];
    __shared__ __align__(16) float sg[kWO][kWGo];
    const int ci0 = blockIdx.x * kWC, co0 = blockIdx.y * kWO, tid = threadIdx.x;
    const int co = tid & 7, ci = tid >> 3 & 7, zq = tid >> 6;  // output channels co, co + 8; plane zq of the tile
    const int tx = (nx + kWX - 1) / kWX, ty = (ny + kWY - 1) / kWY, tz = (nz + kWZ - 1) / kWZ;
    const int64_t tiles = (int64_t)B * tx * ty * tz;
    const int64_t S = (int64_t)nx * ny * nz, S2 = (int64_t)(nx >> 1) * (ny >> 1) * (nz >> 1);
    const int half = tid >> 7, pt = tid & 127, hx = pt % (kWX + 2), hy = pt / (kWX + 2);
    static_assert(kHaloXY <= 128 && kWX * kWY * kWZ == 256 && kWZ + 2 == 6, "threads of the loads");
    float acc[2][kWTaps];
#pragma unroll
    for (int t = 0; t < kWTaps; ++t) acc[0][t] = acc[1][t] = 0.f;
    float *red = si;  // 64 x 2 x 28 floats
    static_assert(64 * 2 * kWTaps <= kWC * kWCh, "reduction buffer");
    int held = 0;  // tiles in acc
    bool first = true;
    for (int64_t tile = blockIdx.z; tile < tiles; tile += gridDim.z) {
        const int b = (int)(tile / ((int64_t)tx * ty * tz)), q = (int)(tile % ((int64_t)tx * ty * tz));
        const int x0 = q % tx * kWX, y0 = q / tx % ty * kWY, z0 = q / (tx * ty) * kWZ;
        __syncthreads();
        {  // the inputs with their halo: threads 128 h .. + 99 take a plane's points, the halves every other plane
            const int x = x0 + hx - 1, y = y0 + hy - 1;
            const bool inxy = pt < kHaloXY && x >= 0 && y >= 0 && x < nx && y < ny;
            float v[3][kWC];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int z = z0 + 2 * i + half - 1;
                const bool on = inxy && z >= 0 && z < nz;
                const float *pf = in.full + (((int64_t)b * in.c1 + ci0 - in.c0) * nz + z) * ny * nx + (int64_t)y * nx + x;
                const float *ph = in.half + (((int64_t)b * in.c0 + ci0) * (nz >> 1) + (z >> 1)) * (ny >> 1) * (nx >> 1) +
                                  (int64_t)(y >> 1) * (nx >> 1) + (x >> 1);
#pragma unroll
                for (int c = 0; c < kWC; ++c)
                    v[i][c] = on && ci0 + c < cin ? __ldg(ci0 + c < in.c0 ? ph + c * S2 : pf + c * S) : 0.f;
            }
            if (pt < kHaloXY)
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int c = 0; c < kWC; ++c) si[c * kWCh + (2 * i + half) * kWPlane + hy * kWRow + hx] = v[i][c];
        }
        {  // the gradients: a voxel per thread
            const int x = x0 + tid % kWX, y = y0 + tid / kWX % kWY, z = z0 + tid / (kWX * kWY);
            const bool on = x < nx && y < ny && z < nz;
            const int64_t at = (((int64_t)b * cout + co0) * nz + z) * ny * nx + (int64_t)y * nx + x;
            float v[kWO];
#pragma unroll
            for (int c = 0; c < kWO; ++c) v[c] = on && co0 + c < cout ? __ldg(go.full + at + c * S) : 0.f;
            if (go.gate)
#pragma unroll
                for (int c = 0; c < kWO; ++c)
                    if (!(on && co0 + c < cout && __ldg(go.gate + at + c * S) > 0.f)) v[c] = 0.f;
#pragma unroll
            for (int c = 0; c < kWO; ++c) sg[c][tid] = v[c];
        }
        __syncthreads();
        const int ye = z0 + zq < nz ? min(kWY, ny - y0) : 0;  // rows of the thread's plane inside the grid
#pragma unroll 1
        for (int y = 0; y < ye; ++y) {
            float g[2][8];
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const float4 *p = reinterpret_cast<const float4 *>(&sg[co + 8 * o][(zq * kWY + y) * kWX]);
                const float4 a = p[0], c = p[1];
                g[o][0] = a.x, g[o][1] = a.y, g[o][2] = a.z, g[o][3] = a.w;
                g[o][4] = c.x, g[o][5] = c.y, g[o][6] = c.z, g[o][7] = c.w;
                acc[o][27] += ((a.x + a.y) + (a.z + a.w)) + ((c.x + c.y) + (c.z + c.w));
            }
#pragma unroll
            for (int d = 0; d < 9; ++d) {
                const float *row = si + ci * kWCh + (zq + d / 3) * kWPlane + (y + d % 3) * kWRow;
                const float4 a = *reinterpret_cast<const float4 *>(row), c = *reinterpret_cast<const float4 *>(row + 4);
                const float2 f = *reinterpret_cast<const float2 *>(row + 8);
                const float v[10] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w, f.x, f.y};
#pragma unroll
                for (int k = 0; k < 8; ++k)
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int o = 0; o < 2; ++o) acc[o][3 * d + dx] = fmaf(g[o][k], v[k + dx], acc[o][3 * d + dx]);
            }
        }
        const bool last = tile + gridDim.z >= tiles;
        if (++held < fold && !last) continue;
        held = 0;
        // the four planes, then the running sums
#pragma unroll 1
        for (int w = 1; w < kWZ; ++w) {
            __syncthreads();
            if (zq == w)
#pragma unroll
                for (int t = 0; t < 2 * kWTaps; ++t) red[t * 64 + (tid & 63)] = acc[t / kWTaps][t % kWTaps];
            __syncthreads();
            if (zq == 0)
#pragma unroll
                for (int t = 0; t < 2 * kWTaps; ++t) acc[t / kWTaps][t % kWTaps] += red[t * 64 + tid];
        }
        if (zq == 0 && !(first && last))
#pragma unroll
            for (int t = 0; t < 2 * kWTaps; ++t) {
                float &a = acc[t / kWTaps][t % kWTaps];
                float2 r = first ? make_float2(0.f, 0.f) : run[t * 64 + tid];
                ff_add(r.x, r.y, a, 0.f);
                if (!last) run[t * 64 + tid] = r;
                else a = r.y == r.y ? r.x + r.y : r.x;  // the errors of an infinite sum are NaN
            }
        first = false;
        if (!last)
#pragma unroll
            for (int t = 0; t < kWTaps; ++t) acc[0][t] = acc[1][t] = 0.f;
    }
    // this CTA's sums: part[z][co][ci][tap]
    if (zq == 0) {
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            float4 *p = reinterpret_cast<float4 *>(
                part + ((((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * kWO + co + 8 * o) * (gridDim.x * kWC) + ci0 + ci) * kWTaps);
#pragma unroll
            for (int t = 0; t < kWTaps; t += 4) p[t / 4] = make_float4(acc[o][t], acc[o][t + 1], acc[o][t + 2], acc[o][t + 3]);
        }
    }
}

// one warp per 32 entries and part of the slabs; blockDim.y parts, so that a thread adds about eight slabs
__global__ void __launch_bounds__(32 * kSumParts)
    wgrad_sum_kernel(const float *__restrict__ part, int nslab, int cin, int cout, int cip, int cop, float *__restrict__ gw,
                     float *__restrict__ gb)
{
    const int64_t n = (int64_t)cout * cin * kWTaps, slab = (int64_t)cop * cip * kWTaps;
    __shared__ double sh[kSumParts][32];
    for (int64_t e0 = blockIdx.x * (int64_t)32; e0 < n; e0 += (int64_t)gridDim.x * 32) {
        const int64_t e = e0 + threadIdx.x;
        const int t = (int)(e % kWTaps), ci = (int)(e / kWTaps % cin), co = (int)(e / ((int64_t)kWTaps * cin));
        const bool on = e < n && (t < 27 || ci == 0);
        double s = 0.0;
        if (on) {
            const float *p = part + ((int64_t)co * cip + ci) * kWTaps + t;
#pragma unroll 8
            for (int k = threadIdx.y; k < nslab; k += blockDim.y) s += p[k * slab];
        }
        if (blockDim.y > 1) {
            sh[threadIdx.y][threadIdx.x] = s;
            __syncthreads();
        }
        if (threadIdx.y == 0 && on) {
            for (int q = 1; q < blockDim.y; ++q) s += sh[q][threadIdx.x];
            if (t < 27) gw[((int64_t)co * cin + ci) * 27 + t] += (float)s;
            else gb[co] += (float)s;
        }
        if (blockDim.y > 1) __syncthreads();
    }
}

// coarse[bc][Z][Y][X] = mean of the 8 children (2x average pooling); bc = batch * channels
__global__ void pool_fwd_kernel(const float *fine, float *coarse, int64_t bc, int nx, int ny, int nz)
{
    const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
    const int64_t n = bc * cx * cy * cz;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int X = (int)(e % cx), Y = (int)((e / cx) % cy), Z = (int)((e / ((int64_t)cx * cy)) % cz);
        const int64_t c = e / ((int64_t)cx * cy * cz);
        const float *f = fine + c * (int64_t)nx * ny * nz;
        float s = 0.f;
        for (int k = 0; k < 8; ++k) s += f[((2 * Z + (k >> 2)) * ny + 2 * Y + ((k >> 1) & 1)) * nx + 2 * X + (k & 1)];
        coarse[e] = 0.125f * s;
    }
}

// gfine += gcoarse / 8 at every child
__global__ void pool_bwd_kernel(const float *gcoarse, float *gfine, int64_t bc, int nx, int ny, int nz)
{
    const int64_t n = bc * (int64_t)nx * ny * nz;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % nx), y = (int)((e / nx) % ny), z = (int)((e / ((int64_t)nx * ny)) % nz);
        const int64_t c = e / ((int64_t)nx * ny * nz);
        gfine[e] += 0.125f * gcoarse[((c * (nz / 2) + z / 2) * (ny / 2) + y / 2) * (nx / 2) + x / 2];
    }
}

// gsrc[b][c][P] = sum over the 8 children of gdst[b][c0 + c][.]
__global__ void up_bwd_kernel(const float *gdst, float *gsrc, int B, int C, int Cdst, int c0, int nx, int ny, int nz)
{
    const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
    const int64_t S = (int64_t)nx * ny * nz, Sc = (int64_t)cx * cy * cz, n = (int64_t)B * C * Sc;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t P = e % Sc, bc = e / Sc;
        const int c = (int)(bc % C), b = (int)(bc / C);
        const int X = (int)(P % cx), Y = (int)((P / cx) % cy), Z = (int)(P / ((int64_t)cx * cy));
        const float *g = gdst + ((int64_t)b * Cdst + c0 + c) * S;
        float s = 0.f;
        for (int k = 0; k < 8; ++k) s += g[((2 * Z + (k >> 2)) * ny + 2 * Y + ((k >> 1) & 1)) * nx + 2 * X + (k & 1)];
        gsrc[e] = s;
    }
}

// dst[b][c0 + c][p] = src[b][cs0 + c][p] for c < C
__global__ void chan_copy_kernel(const float *src, int Csrc, int cs0, float *dst, int Cdst, int c0, int B, int C,
                                 int64_t S)
{
    const int64_t n = (int64_t)B * C * S;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = e % S, bc = e / S;
        const int c = (int)(bc % C), b = (int)(bc / C);
        dst[((int64_t)b * Cdst + c0 + c) * S + p] = src[((int64_t)b * Csrc + cs0 + c) * S + p];
    }
}

// Adam (Kingma & Ba, 2015) with bias correction; nothing if a convolution gave up its wait (*err): g is not valid.
__global__ void adam_kernel(float *w, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2, const int *err)
{
    if (*err) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

int blocks_for(int64_t n)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
}

}  // namespace
}  // namespace fcm

using namespace fcm;

struct UConv {
    int cin, cout;
    int64_t woff, boff;  // offsets in the parameter arrays
    int64_t toff, doff;  // offsets of its weight tiles and of its data-gradient convolution's
};

struct fcm_unet {
    cudaStream_t stream = nullptr;
    int in_ch = 0, out_ch = 0, base = 0, levels = 0;
    std::vector<UConv> conv;  // enc (2 per level), dec (2 per level above the bottom, top-down), out
    int64_t nparam = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *tiles = nullptr;  // BF16 weight tiles of every layer (weight_tiles_kernel), made whenever w changes
    int64_t ntiles = 0;              // their entries
    float *part = nullptr;           // partial sums of a weight gradient
    float *host = nullptr;           // pinned copy of parameters and gradients for fcm_unet_get (made on first use)
    std::mutex host_lock;            // held by the reader whose copies are in it
    int *err = nullptr;              // set by a convolution whose wait for the tensor core ran out, until reported
    int *seen = nullptr;             // the same in pinned host memory
    ConvWait wait = {};              // what the convolutions get: these flags, or those of the solve they run in
    // activations for the current shape
    int B = 0, n[3] = {0, 0, 0};
    std::vector<float *> act;  // owned buffers
    const float *input = nullptr;
    float *output = nullptr;
    // per level l: the pooled input, the ReLU outputs of the four convolutions, and their gradients
    std::vector<float *> xin, eA, eB, dA, dB;
    std::vector<float *> gxin, geA, geB, gcat, gdA, gdB;
    std::vector<int64_t> S;   // voxels per level
    std::vector<int> lx, ly, lz;
    // identity of this network and of its activation buffers, for graphs that captured its launches
    uint64_t serial = 0, act_gen = 0;
    int ch(int l) const { return std::min(base << l, 4 * base); }
    int enc_a(int l) const { return 2 * l; }
    int enc_b(int l) const { return 2 * l + 1; }
    int dec_a(int l) const { return 2 * levels + 2 * (levels - 2 - l); }
    int dec_b(int l) const { return dec_a(l) + 1; }
    int out_layer() const { return (int)conv.size() - 1; }
};

namespace {

void free_acts(fcm_unet *N)
{
    for (float *p : N->act) cudaFree(p);
    N->act.clear();
    N->B = 0;
}

cudaError_t falloc(fcm_unet *N, float **p, int64_t count)
{
    cudaError_t e = cudaMalloc((void **)p, sizeof(float) * std::max<int64_t>(count, 1));
    if (e == cudaSuccess) N->act.push_back(*p);
    return e;
}

cudaError_t ensure_shape(fcm_unet *N, int B, int nx, int ny, int nz)
{
    if (N->B == B && N->n[0] == nx && N->n[1] == ny && N->n[2] == nz) return cudaSuccess;
    free_acts(N);
    ++N->act_gen;
    const int L = N->levels;
    for (auto *v : {&N->xin, &N->eA, &N->eB, &N->dA, &N->dB, &N->gxin, &N->geA, &N->geB, &N->gcat, &N->gdA, &N->gdB})
        v->assign(L, nullptr);
    N->S.assign(L, 0);
    N->lx.assign(L, 0);
    N->ly.assign(L, 0);
    N->lz.assign(L, 0);
    cudaError_t e;
    for (int l = 0; l < L; ++l) {
        N->lx[l] = nx >> l;
        N->ly[l] = ny >> l;
        N->lz[l] = nz >> l;
        const int64_t S = (int64_t)N->lx[l] * N->ly[l] * N->lz[l];
        N->S[l] = S;
        const int c = N->ch(l);
        const int64_t bs = (int64_t)B * c * S;
        if (l > 0) {
            if ((e = falloc(N, &N->xin[l], (int64_t)B * N->ch(l - 1) * S)) != cudaSuccess) return e;
            if ((e = falloc(N, &N->gxin[l], (int64_t)B * N->ch(l - 1) * S)) != cudaSuccess) return e;
        }
        for (auto *v : {&N->eA, &N->eB, &N->geA, &N->geB})
            if ((e = falloc(N, &(*v)[l], bs)) != cudaSuccess) return e;
        if (l <= L - 2) {
            if ((e = falloc(N, &N->gcat[l], (int64_t)B * (N->ch(l + 1) + c) * S)) != cudaSuccess) return e;
            for (auto *v : {&N->dA, &N->dB, &N->gdA, &N->gdB})
                if ((e = falloc(N, &(*v)[l], bs)) != cudaSuccess) return e;
        }
    }
    N->B = B;
    N->n[0] = nx;
    N->n[1] = ny;
    N->n[2] = nz;
    return cudaSuccess;
}

// CTAs of a weight gradient's partial sums: two per SM over the channel tiles
int wgrad_slabs(int cin, int cout, int64_t tiles)
{
    const int64_t ch = (int64_t)((cin + kWC - 1) / kWC) * ((cout + kWO - 1) / kWO);
    return (int)std::max<int64_t>(1, std::min<int64_t>({tiles, 304 / ch, (int64_t)65535}));
}

// Tiles (64 voxels per thread) whose products a weight gradient adds in one chain of FP32 additions: a 256th of the
// voxels of a channel pair, at least one tile
int wgrad_fold(int64_t voxels) { return (int)std::max<int64_t>(1, voxels / (256 * kWX * kWY)); }

// out = [relu](bias + conv(src)) at level l with the tiles of a convolution cin -> cout
void conv_launch(fcm_unet *N, const ConvSrc &src, int64_t tiles, const float *bias, float *out, int cin, int cout, int l,
                 bool relu)
{
    const int nx = N->lx[l], ny = N->ly[l], nz = N->lz[l], nb = conv_nb(cout);
    const int64_t txy = (int64_t)((nx + kTX - 1) / kTX) * ((ny + kTY - 1) / kTY);
    const uint4 *w = reinterpret_cast<const uint4 *>(N->tiles + tiles);
    // More planes per CTA take fewer products and halo voxels per output (27 (ZT + 2) and 1.4 (ZT + 2), over ZT);
    // with 16 columns three and with 32 two still leave room for two CTAs per SM (256 of 512 tensor-memory columns
    // each).  The choice is the least number of waves of 304 CTAs times ZT + 2 (40^3 cells, 32 channels: two planes
    // are one wave, one plane two).
    const auto ctas = [&](int zt) { return txy * ((nz + zt - 1) / zt) * N->B * conv_blocks(cout); };
    const auto cost = [&](int zt) { return (ctas(zt) + 303) / 304 * (zt + 2); };
    int zt = 1;
    for (int k = 2; k <= (nb == 16 ? 3 : nb <= 32 ? 2 : 1); ++k)
        if (cost(k) < cost(zt)) zt = k;
    const auto kernel = zt == 3 ? conv3_tc_kernel<3> : zt == 2 ? conv3_tc_kernel<2> : conv3_tc_kernel<1>;
    const dim3 grid((unsigned)(txy * ((nz + zt - 1) / zt)), conv_blocks(cout), N->B);
    kernel<<<grid, kConvThreads, conv_smem(zt, nb), N->stream>>>(src, w, bias, out, cin, cout, nx, ny, nz, relu, N->wait);
}

void conv_fwd(fcm_unet *N, int layer, const ConvSrc &src, float *out, int l, bool relu)
{
    const UConv &c = N->conv[layer];
    conv_launch(N, src, c.toff, N->w + c.boff, out, c.cin, c.cout, l, relu);
}

// weight gradients of `layer` and, if gin != NULL, the data gradient (overwritten); gout is read through the
// gate (the ReLU's output; null: none)
void conv_bwd(fcm_unet *N, int layer, const ConvSrc &in, const float *gout, const float *gate, float *gin, int l)
{
    const UConv &c = N->conv[layer];
    const int nx = N->lx[l], ny = N->ly[l], nz = N->lz[l];
    const ConvSrc go{nullptr, gout, gate, 0, c.cout};
    const int64_t tiles = (int64_t)N->B * ((nx + kWX - 1) / kWX) * ((ny + kWY - 1) / kWY) * ((nz + kWZ - 1) / kWZ);
    const int cit = (c.cin + kWC - 1) / kWC, cot = (c.cout + kWO - 1) / kWO, ns = wgrad_slabs(c.cin, c.cout, tiles);
    const int fold = wgrad_fold((int64_t)N->B * N->S[l]);
    conv3_wgrad_kernel<<<dim3(cit, cot, ns), 256, (tiles + ns - 1) / ns > fold ? kWRun : 0, N->stream>>>(
        in, go, c.cin, c.cout, N->B, nx, ny, nz, fold, N->part);
    const int np = std::max(1, std::min(ns / 8, kSumParts));
    wgrad_sum_kernel<<<blocks_for((int64_t)c.cin * c.cout * kWTaps * 8), dim3(32, np), 0, N->stream>>>(
        N->part, ns, c.cin, c.cout, cit * kWC, cot * kWO, N->g + c.woff, N->g + c.boff);
    if (gin) conv_launch(N, go, c.doff, nullptr, gin, c.cout, c.cin, l, false);
}

ConvSrc plain(const float *a, int c) { return ConvSrc{nullptr, a, nullptr, 0, c}; }

// every layer's weight tiles from the parameters
void refresh_weights(fcm_unet *N)
{
    TileTable tab;
    tab.sets = 2 * (int)N->conv.size();
    for (size_t k = 0; k < N->conv.size(); ++k) {
        const UConv &c = N->conv[k];
        tab.at[2 * k] = c.toff;
        tab.at[2 * k + 1] = c.doff;
        tab.woff[k] = c.woff;
        tab.cin[k] = c.cin;
        tab.cout[k] = c.cout;
    }
    weight_tiles_kernel<<<(unsigned)(N->ntiles / 256), 256, 0, N->stream>>>(N->w, N->tiles, tab);
}

uint64_t splitmix(uint64_t &s)
{
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}


}  // namespace


namespace fcm {
void unet_identity(const fcm_unet *N, uint64_t *serial, uint64_t *gen)
{
    *serial = N ? N->serial : 0;
    *gen = N ? N->act_gen : 0;
}

cudaStream_t unet_bind(fcm_unet *N, cudaStream_t s, int *err)
{
    cudaStream_t old = N->stream;
    N->stream = s;
    N->wait.err = err ? err : N->err;
    N->wait.seen = err ? nullptr : N->seen;
    N->wait.code = kErrConv;
    return old;
}
}  // namespace fcm

#define UN_CUDA(call)                                                                         \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) {                                                              \
            fcm_unet_last_error() = std::string(#call) + ": " + cudaGetErrorString(e_);               \
            return e_ == cudaErrorMemoryAllocation ? FCM_ENOMEM : FCM_ECUDA;                  \
        }                                                                                     \
    } while (0)

namespace {

// FCM_ETIMEOUT, once, if a convolution is known to have given up its wait: takes both flags back (the device's in
// stream order, so that an Adam step queued behind the convolution still sees it)
fcm_status unet_report(fcm_unet *N)
{
    volatile int *seen = N->seen;
    if (N->wait.seen != N->seen || !*seen) return FCM_OK;
    *seen = 0;
    UN_CUDA(cudaMemsetAsync(N->err, 0, sizeof(int), N->stream));
    fcm_unet_last_error() = timeout_text("U-Net", kErrConv);
    return FCM_ETIMEOUT;
}

}  // namespace

extern "C" {

fcm_status fcm_unet_create(const fcm_unet_desc *d, void *cuda_stream, fcm_unet **out)
{
    if (!d || !out || d->in_ch < 1 || d->out_ch < 1 || d->base < 1 || d->base > 256 || d->levels < 1 ||
        d->levels > 6) {
        fcm_unet_last_error() = "fcm_unet_create: invalid description";
        return FCM_EINVAL;
    }
    *out = nullptr;
    fcm_unet *N = new fcm_unet();
    static std::atomic<uint64_t> next_serial{1};
    N->serial = next_serial++;
    N->stream = (cudaStream_t)cuda_stream;
    N->in_ch = d->in_ch;
    N->out_ch = d->out_ch;
    N->base = d->base;
    N->levels = d->levels;
    const int L = d->levels;
    for (int l = 0; l < L; ++l) {
        N->conv.push_back({l == 0 ? d->in_ch : N->ch(l - 1), N->ch(l), 0, 0, 0, 0});
        N->conv.push_back({N->ch(l), N->ch(l), 0, 0, 0, 0});
    }
    for (int l = L - 2; l >= 0; --l) {
        N->conv.push_back({N->ch(l + 1) + N->ch(l), N->ch(l), 0, 0, 0, 0});
        N->conv.push_back({N->ch(l), N->ch(l), 0, 0, 0, 0});
    }
    N->conv.push_back({N->ch(0), d->out_ch, 0, 0, 0, 0});
    int64_t off = 0, toff = 0, npart = 0;
    for (UConv &c : N->conv) {
        c.woff = off;
        off += (int64_t)c.cout * c.cin * 27;
        c.boff = off;
        off += c.cout;
        c.toff = toff;
        toff += conv_tile_entries(c.cin, c.cout);
        c.doff = toff;
        toff += conv_tile_entries(c.cout, c.cin);
        const int64_t pairs = (int64_t)((c.cin + kWC - 1) / kWC * kWC) * ((c.cout + kWO - 1) / kWO * kWO);
        npart = std::max(npart, pairs * kWTaps * wgrad_slabs(c.cin, c.cout, INT64_MAX));
    }
    N->nparam = off;
    N->ntiles = toff;
    // Kaiming-uniform weights (bound sqrt(6 / fan_in)), zero biases; the output layer 10x smaller
    std::vector<float> h(off, 0.f);
    uint64_t s = d->seed;
    for (size_t k = 0; k < N->conv.size(); ++k) {
        const UConv &c = N->conv[k];
        float bound = std::sqrt(6.0f / (c.cin * 27.0f));
        if ((int)k == N->out_layer()) bound *= 0.1f;
        for (int64_t i = 0; i < (int64_t)c.cout * c.cin * 27; ++i) {
            const double u = (splitmix(s) >> 11) * (1.0 / 9007199254740992.0);
            h[c.woff + i] = (float)((2.0 * u - 1.0) * bound);
        }
    }
    auto fail = [&](cudaError_t e) {
        fcm_unet_last_error() = std::string("fcm_unet_create: ") + cudaGetErrorString(e);
        fcm_unet_destroy(N);
        return e == cudaErrorMemoryAllocation ? FCM_ENOMEM : FCM_ECUDA;
    };
    cudaError_t e;
    float **arrs[] = {&N->w, &N->g, &N->m, &N->v};
    for (float **a : arrs) {
        if ((e = cudaMalloc((void **)a, sizeof(float) * off)) != cudaSuccess) return fail(e);
        if ((e = cudaMemsetAsync(*a, 0, sizeof(float) * off, N->stream)) != cudaSuccess) return fail(e);
    }
    if ((e = cudaMalloc((void **)&N->tiles, sizeof(__nv_bfloat16) * toff)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc((void **)&N->part, sizeof(float) * npart)) != cudaSuccess) return fail(e);
    if ((e = cudaMalloc((void **)&N->err, sizeof(int))) != cudaSuccess) return fail(e);
    if ((e = cudaMemsetAsync(N->err, 0, sizeof(int), N->stream)) != cudaSuccess) return fail(e);
    if ((e = cudaMallocHost((void **)&N->seen, sizeof(int))) != cudaSuccess) return fail(e);
    *N->seen = 0;
    N->wait.tries = kWaitTries;
    unet_bind(N, N->stream, nullptr);
    if ((e = cudaFuncSetAttribute(conv3_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWRun)) != cudaSuccess)
        return fail(e);
    if ((e = cudaFuncSetAttribute(conv3_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  conv_smem(1, kCoMax))) != cudaSuccess ||
        (e = cudaFuncSetAttribute(conv3_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, conv_smem(2, 32))) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(conv3_tc_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, conv_smem(3, 16))) !=
            cudaSuccess)
        return fail(e);
    if ((e = cudaMemcpyAsync(N->w, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice, N->stream)) != cudaSuccess)
        return fail(e);
    refresh_weights(N);
    if ((e = cudaStreamSynchronize(N->stream)) != cudaSuccess) return fail(e);
    *out = N;
    return FCM_OK;
}

fcm_status fcm_unet_params(const fcm_unet *N, int64_t *count)
{
    if (!N || !count) return FCM_EINVAL;
    *count = N->nparam;
    return FCM_OK;
}

fcm_status fcm_unet_get(fcm_unet *N, float *w_host, float *g_host)
{
    if (!N || !w_host) return FCM_EINVAL;
    // through pinned memory: a copy to the caller's pageable buffers runs at 3.4 GB/s (2 MB each, 1.2 ms)
    const size_t bytes = sizeof(float) * N->nparam;
    const std::lock_guard<std::mutex> lock(N->host_lock);
    if (!N->host) UN_CUDA(cudaMallocHost((void **)&N->host, 2 * bytes));
    UN_CUDA(cudaMemcpyAsync(N->host, N->w, bytes, cudaMemcpyDeviceToHost, N->stream));
    if (g_host) UN_CUDA(cudaMemcpyAsync(N->host + N->nparam, N->g, bytes, cudaMemcpyDeviceToHost, N->stream));
    UN_CUDA(cudaStreamSynchronize(N->stream));
    std::memcpy(w_host, N->host, bytes);
    if (g_host) std::memcpy(g_host, N->host + N->nparam, bytes);
    return unet_report(N);
}

fcm_status fcm_unet_status(fcm_unet *N)
{
    if (!N) return FCM_EINVAL;
    UN_CUDA(cudaStreamSynchronize(N->stream));
    return unet_report(N);
}

fcm_status fcm_unet_set_wait_limit(fcm_unet *N, int tries)
{
    if (!N) return FCM_EINVAL;
    N->wait.tries = tries < 0 ? kWaitTries : tries;
    ++N->act_gen;  // graphs that captured launches with another limit are captured again
    return FCM_OK;
}

fcm_status fcm_unet_set(fcm_unet *N, const float *w_host)
{
    if (!N || !w_host) return FCM_EINVAL;
    UN_CUDA(cudaMemcpyAsync(N->w, w_host, sizeof(float) * N->nparam, cudaMemcpyHostToDevice, N->stream));
    refresh_weights(N);
    UN_CUDA(cudaStreamSynchronize(N->stream));
    return FCM_OK;
}

fcm_status fcm_unet_forward(fcm_unet *N, const float *in, int B, int nx, int ny, int nz, float *out)
{
    if (!N || !in || !out || B < 1) return FCM_EINVAL;
    const int div = 1 << (N->levels - 1);
    if (nx < div || ny < div || nz < div || nx % div || ny % div || nz % div) {
        fcm_unet_last_error() = "fcm_unet_forward: spatial sizes must be positive multiples of 2^(levels-1)";
        return FCM_EINVAL;
    }
    const fcm_status s = unet_report(N);
    if (s != FCM_OK) return s;
    UN_CUDA(ensure_shape(N, B, nx, ny, nz));
    const int L = N->levels;
    N->input = in;
    N->output = out;
    for (int l = 0; l < L; ++l) {
        if (l > 0)
            pool_fwd_kernel<<<blocks_for((int64_t)B * N->ch(l - 1) * N->S[l]), 256, 0, N->stream>>>(
                N->eB[l - 1], N->xin[l], (int64_t)B * N->ch(l - 1), N->lx[l - 1], N->ly[l - 1], N->lz[l - 1]);
        conv_fwd(N, N->enc_a(l), l == 0 ? plain(in, N->in_ch) : plain(N->xin[l], N->ch(l - 1)), N->eA[l], l, true);
        conv_fwd(N, N->enc_b(l), plain(N->eA[l], N->ch(l)), N->eB[l], l, true);
    }
    const float *prev = N->eB[L - 1];
    for (int l = L - 2; l >= 0; --l) {
        conv_fwd(N, N->dec_a(l), ConvSrc{prev, N->eB[l], nullptr, N->ch(l + 1), N->ch(l)}, N->dA[l], l, true);
        conv_fwd(N, N->dec_b(l), plain(N->dA[l], N->ch(l)), N->dB[l], l, true);
        prev = N->dB[l];
    }
    conv_fwd(N, N->out_layer(), plain(prev, N->ch(0)), out, 0, false);
    UN_CUDA(cudaGetLastError());
    return FCM_OK;
}

fcm_status fcm_unet_backward(fcm_unet *N, const float *gout, float *gin)
{
    if (!N || !gout || N->B == 0 || !N->input) {
        fcm_unet_last_error() = "fcm_unet_backward: call fcm_unet_forward first";
        return N ? FCM_ESTATE : FCM_EINVAL;
    }
    const fcm_status s = unet_report(N);
    if (s != FCM_OK) return s;
    const int L = N->levels, B = N->B;
    float *gtop = (L >= 2) ? N->gdB[0] : N->geB[0];
    const float *top = (L >= 2) ? N->dB[0] : N->eB[0];
    conv_bwd(N, N->out_layer(), plain(top, N->ch(0)), gout, nullptr, gtop, 0);
    for (int l = 0; l <= L - 2; ++l) {
        const int cu = N->ch(l + 1), cs = N->ch(l), cc = cu + cs;
        const int64_t S = N->S[l], bs = (int64_t)B * cs * S;
        const float *prev = l + 1 == L - 1 ? N->eB[L - 1] : N->dB[l + 1];
        conv_bwd(N, N->dec_b(l), plain(N->dA[l], cs), N->gdB[l], N->dB[l], N->gdA[l], l);
        conv_bwd(N, N->dec_a(l), ConvSrc{prev, N->eB[l], nullptr, cu, cs}, N->gdA[l], N->dA[l], N->gcat[l], l);
        // skip part -> encoder output of level l (the pooling adds the other part below)
        chan_copy_kernel<<<blocks_for(bs), 256, 0, N->stream>>>(N->gcat[l], cc, cu, N->geB[l], cs, 0, B, cs, S);
        // upsampled part -> the level below
        float *gprev = (l + 1 == L - 1) ? N->geB[L - 1] : N->gdB[l + 1];
        up_bwd_kernel<<<blocks_for((int64_t)B * cu * N->S[l + 1]), 256, 0, N->stream>>>(
            N->gcat[l], gprev, B, cu, cc, 0, N->lx[l], N->ly[l], N->lz[l]);
    }
    for (int l = L - 1; l >= 0; --l) {
        conv_bwd(N, N->enc_b(l), plain(N->eA[l], N->ch(l)), N->geB[l], N->eB[l], N->geA[l], l);
        if (l > 0) {
            conv_bwd(N, N->enc_a(l), plain(N->xin[l], N->ch(l - 1)), N->geA[l], N->eA[l], N->gxin[l], l);
            pool_bwd_kernel<<<blocks_for((int64_t)B * N->ch(l - 1) * N->S[l - 1]), 256, 0, N->stream>>>(
                N->gxin[l], N->geB[l - 1], (int64_t)B * N->ch(l - 1), N->lx[l - 1], N->ly[l - 1], N->lz[l - 1]);
        } else {
            conv_bwd(N, N->enc_a(0), plain(N->input, N->in_ch), N->geA[0], N->eA[0], gin, 0);
        }
    }
    UN_CUDA(cudaGetLastError());
    return FCM_OK;
}

fcm_status fcm_unet_zero_grad(fcm_unet *N)
{
    if (!N) return FCM_EINVAL;
    UN_CUDA(cudaMemsetAsync(N->g, 0, sizeof(float) * N->nparam, N->stream));
    return FCM_OK;
}

fcm_status fcm_unet_adam(fcm_unet *N, float lr, float b1, float b2, float eps, int step)
{
    if (!N || step < 1) return FCM_EINVAL;
    const fcm_status s = unet_report(N);
    if (s != FCM_OK) return s;
    const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
    adam_kernel<<<blocks_for(N->nparam), 256, 0, N->stream>>>(N->w, N->g, N->m, N->v, N->nparam, lr, b1, b2, eps, c1, c2, N->err);
    refresh_weights(N);
    UN_CUDA(cudaGetLastError());
    return FCM_OK;
}

void fcm_unet_destroy(fcm_unet *N)
{
    if (!N) return;
    if (N->stream) cudaStreamSynchronize(N->stream);
    free_acts(N);
    void *ptrs[] = {N->w, N->g, N->m, N->v, N->tiles, N->part, N->err};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (N->host) cudaFreeHost(N->host);
    if (N->seen) cudaFreeHost(N->seen);
    delete N;
}

}  // extern "C"

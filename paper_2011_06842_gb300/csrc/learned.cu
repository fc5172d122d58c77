// Kernels of the learned warm start: a small convolutional network over the
// previous frames' layer coefficients (3x3 convolutions, zero padding, ReLU),
// its backward pass, the MSE loss and the Adam update.  FP32, NCHW tensors
// with an explicit batch stride (the layers of one size are a batch).
// Not part of the paper's method: a predictor of the next time step's warm
// start and deflation directions; PCG stays the solver.
#include <cuda_runtime.h>

#include "../../include/fewha.h"

namespace {

// 4-byte asynchronous copy into shared memory; `in` false writes zero (the
// source is then not read).
__device__ __forceinline__ void cp4(float *dst, const float *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(in ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr int TX = 32;    // output tile width (4 pixels per thread)
constexpr int TY = 16;    // output tile height
constexpr int PX = 4;     // adjacent pixels per thread
constexpr int CO_T = 8;   // output channels per block
constexpr int CI_T = 4;   // input channels staged per step
constexpr int NT = TX * TY / PX;
constexpr int CONV_CTAS = 6;  // CTAs per SM: 78 registers a thread (85 would fit) and 23 KB each
constexpr int TP = TX + 4;  // pitch of a staged row: x0-1 .. x0+TX plus slack, 16-byte rows

// out[b][co][y][x] = act(bias[co] + sum_ci sum_{ky,kx} w[co][ci][ky][kx] in[b][ci][y+ky-1][x+kx-1])
// (zero outside the image).  Tensors are addressed as base + b*bs + c*cs + y*W + x.
// For the data gradient the weights are read transposed and flipped
// (wt_mode = 1: w[ci][co][2-ky][2-kx] of a Cin x Cout tensor), and with
// `mask` (laid out like out) an output whose mask is not positive is 0: the
// backward pass of the ReLU that produced the convolution's input.
//
// Bound by the FP32 units once the operands are in shared memory.  Each thread
// computes four adjacent pixels for CO_T channels: per input channel and kernel
// row it reads six inputs (one 16- and one 8-byte load) and 3 x CO_T weights
// (16-byte loads, the same for every lane), 36 shared-memory wavefronts for 288
// FMAs per thread, against 60 for 288 with two vertically adjacent pixels and
// single loads.  Input tiles and weights of the next CI_T channels are copied
// asynchronously while the present ones are used.  32 -> 32 channels over 5 x
// 128^2 and 4 x 64^2 pixels: 76 us in one launch (79 + 24 us in two of eight staged
// channels and four CTAs per SM).
//
// A launch covers up to kMaxGroups groups of equal-size images (the layers of
// each size): a group of small images alone leaves most SMs idle.
constexpr int kMaxGroups = FEWHA_NET_GROUPS;

struct ConvGroup {
    const float *in, *mask;
    float *out;
    long in_bs, in_cs, out_bs, out_cs;
    int H, W, tiles_x, tiles, blk0;  // tiles per image, first block
};
struct ConvArgs {
    ConvGroup g[kMaxGroups];
    const float *w, *bias;
    int ng, Cin, Cout, relu, wt_mode;
};

__global__ void __launch_bounds__(NT, CONV_CTAS) k_conv3x3(const __grid_constant__ ConvArgs A)
{
    __shared__ __align__(16) float tile[2][CI_T][TY + 2][TP];
    __shared__ __align__(16) float wsh[2][CI_T][9][CO_T];
    int gi = 0;
    while (gi + 1 < A.ng && (int)blockIdx.x >= A.g[gi + 1].blk0) gi++;
    const ConvGroup &G = A.g[gi];
    const float *__restrict__ w = A.w, *__restrict__ bias = A.bias, *__restrict__ mask = G.mask;
    float *__restrict__ out = G.out;
    const long in_cs = G.in_cs, out_bs = G.out_bs, out_cs = G.out_cs;
    const int Cin = A.Cin, Cout = A.Cout, H = G.H, W = G.W, relu = A.relu, wt_mode = A.wt_mode;
    const int tx = (threadIdx.x % (TX / PX)) * PX, ty = threadIdx.x / (TX / PX);
    const int nco = (Cout + CO_T - 1) / CO_T, blk = (int)blockIdx.x - G.blk0;
    const int t = blk % G.tiles, z = blk / G.tiles;
    const int x0 = (t % G.tiles_x) * TX, y0 = (t / G.tiles_x) * TY;
    const int b = z / nco, co0 = (z % nco) * CO_T;
    const float *__restrict__ inb = G.in + (long)b * G.in_bs;
    auto stage = [&](int s, int ci0) {
        // a warp per row of 34 pixels: lanes 0..31, then two lanes for the rest
        static_assert(TX == 32, "a row is a warp and two pixels");
        const int lane = threadIdx.x & 31, x = x0 - 1 + lane;
        const bool okx = x >= 0 && x < W, okt = lane < 2 && x + 32 < W;
        for (int rr = threadIdx.x >> 5; rr < CI_T * (TY + 2); rr += NT / 32) {
            const int c = rr / (TY + 2), r = rr - c * (TY + 2), y = y0 + r - 1;
            const bool row = ci0 + c < Cin && y >= 0 && y < H;
            const float *src = inb + (long)(ci0 + c) * in_cs + (long)y * W + x;
            float *dst = &tile[s][c][r][lane];
            cp4(dst, row && okx ? src : inb, row && okx);
            if (lane < 2) cp4(dst + 32, row && okt ? src + 32 : inb, row && okt);
        }
        for (int e = threadIdx.x; e < CO_T * CI_T * 9; e += NT) {
            const int k = e % 9, j = wt_mode ? (e / 9) % CO_T : e / (9 * CI_T);
            const int c = wt_mode ? e / (9 * CO_T) : (e / 9) % CI_T;
            const int co = co0 + j, ci = ci0 + c;
            const bool ok = co < Cout && ci < Cin;
            const float *src = !ok ? w : wt_mode ? w + ((long)ci * Cout + co) * 9 + (8 - k)
                                                 : w + ((long)co * Cin + ci) * 9 + k;
            cp4(&wsh[s][c][k][j], src, ok);
        }
        cp_commit();
    };
    float acc[CO_T][PX];
#pragma unroll
    for (int j = 0; j < CO_T; j++)
#pragma unroll
        for (int i = 0; i < PX; i++) acc[j][i] = (bias && co0 + j < Cout) ? bias[co0 + j] : 0.f;
    stage(0, 0);
    for (int ci0 = 0, s = 0; ci0 < Cin; ci0 += CI_T, s ^= 1) {
        if (ci0 + CI_T < Cin) {
            stage(s ^ 1, ci0 + CI_T);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const int nc = Cin - ci0 < CI_T ? Cin - ci0 : CI_T;
#pragma unroll 2
        for (int c = 0; c < nc; c++) {
#pragma unroll
            for (int ky = 0; ky < 3; ky++) {
                const float *row = &tile[s][c][ty + ky][tx];
                const float4 va = *reinterpret_cast<const float4 *>(row);
                const float2 vb = *reinterpret_cast<const float2 *>(row + 4);
                const float v[6] = {va.x, va.y, va.z, va.w, vb.x, vb.y};
#pragma unroll
                for (int kx = 0; kx < 3; kx++) {
                    const float4 wa = *reinterpret_cast<const float4 *>(&wsh[s][c][3 * ky + kx][0]);
                    const float4 wb = *reinterpret_cast<const float4 *>(&wsh[s][c][3 * ky + kx][4]);
                    const float wk[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                    for (int j = 0; j < CO_T; j++)
#pragma unroll
                        for (int i = 0; i < PX; i++) acc[j][i] += wk[j] * v[i + kx];
                }
            }
        }
        __syncthreads();
    }
    const int x = x0 + tx, y = y0 + ty;
    if (y >= H) return;
#pragma unroll
    for (int j = 0; j < CO_T; j++) {
        if (co0 + j >= Cout) break;
        const long o = (long)b * out_bs + (long)(co0 + j) * out_cs + (long)y * W + x;
#pragma unroll
        for (int i = 0; i < PX; i++) {
            if (x + i < W) {
                float v = acc[j][i];
                if (relu) v = v > 0.f ? v : 0.f;
                if (mask && !(mask[o + i] > 0.f)) v = 0.f;
                out[o + i] = v;
            }
        }
    }
}

// Partial weight/bias gradients.  A CTA takes spatial tiles of TS x TH pixels
// (tile t0 + blockIdx.x, + gridDim.x, ...) and one block of 4 CG output times 2 IG
// input channels; the next tile's gradients and inputs are copied to shared
// memory while the present one is used,
// and a thread keeps 4 x 2 x 9 sums in registers for its slice of the tile's
// pixels (512 / (CG IG) slices), so four pixels cost it 4 + 12 shared loads for
// 288 FMAs (one output value per thread read two operands from shared memory
// for every FMA).  The slices are summed in slice order at the end.  With the
// parallel sum of the partials below and the four-pixel convolution above, a
// training step on the ELT layers (5 x 128^2 and 4 x 64^2) went from 1171 to
// 596 us; with the groups in one launch and 152 CTAs, to 418 us.
constexpr int TS = 16;           // width of the spatial tile; the workspace counts TS x TS tiles
constexpr int TH = 8;            // its height: 16 x 8 tiles spread over the CTAs more evenly than 16 x 16
constexpr int WG_T = 512;        // threads
constexpr int WG_CTAS = 152;     // CTAs of one launch, one per SM: the fewer, the fewer partials to add in FP64
// Most tiles of one FP32 partial: a thread of the 32 x 32 block adds 32 products a
// tile one after another, one of the narrow blocks 4 or 8 (and more slices at the
// end), so that an FP32 sum is about as long as one 16 x 16 tile's 256 products,
// whose error it is held to: against 64 bits, normal data, rms 2.1e-7 at the limit
// (16 x 16 tiles 2.1e-7; without a limit 5.2e-7 at 54 tiles).  More tiles go in
// rounds of WG_ROUND partials and one tile less each, whose FP64 sums are carried
// from round to round in the rest of the workspace, 20 us a round.
constexpr int WG_ROUND = WG_CTAS - 3;
constexpr int wg_span(int slices) { return slices > 4 ? 24 : 8; }
constexpr int GP = TH * TS + 4;  // channel pitch of the staged gradients: 8 channels on 8 different 16-byte banks
constexpr int IW = TS + 4;       // row pitch of the staged inputs
constexpr int IP = (TH + 2) * IW + 4;  // channel pitch of the staged inputs (odd multiple of 16 bytes)

struct WgradGroup {
    const float *in, *gout;
    long in_bs, in_cs, gout_bs, gout_cs;
    int H, W, tiles_x, tiles, t0;  // tiles per image, first tile
};
struct WgradArgs {
    WgradGroup g[kMaxGroups];
    float *part;
    int ng, Cin, Cout, t0, t1;  // the launch's tiles t0 .. t1 - 1
};

template <int CG, int IG>
constexpr size_t wg_smem()
{
    const size_t tiles = 2 * (size_t)(4 * CG * GP + 2 * IG * IP), sums = (size_t)WG_T * 72;
    return (tiles > sums ? tiles : sums) * sizeof(float);
}

template <int CG, int IG>
__global__ void __launch_bounds__(WG_T, 1) k_conv3x3_wgrad_partial(const __grid_constant__ WgradArgs A)
{
    extern __shared__ __align__(16) float wg_sm[];
    constexpr int COB = 4 * CG, CIB = 2 * IG, NS = WG_T / (CG * IG), BUF = COB * GP + CIB * IP;
    static_assert(NS * CG * IG == WG_T && (TH * TS / 4) % NS == 0, "slices cover the tile");
    const int co0 = blockIdx.y * COB, ci0 = blockIdx.z * CIB, Cin = A.Cin, Cout = A.Cout;
    const int cg = threadIdx.x % CG, ig = (threadIdx.x / CG) % IG, slice = threadIdx.x / (CG * IG);
    float acc[4][2][9];
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int k = 0; k < 9; k++) acc[j][i][k] = 0.f;
    constexpr int BT = WG_T / COB < 32 ? WG_T / COB : 32;  // threads per bias channel
    float bsum = 0.f;
    // asynchronous copy of tile t into buffer s
    auto stage = [&](int s, int t) {
        int gi = 0;
        while (gi + 1 < A.ng && t >= A.g[gi + 1].t0) gi++;
        const WgradGroup &G = A.g[gi];
        const int H = G.H, W = G.W, lt = t - G.t0, b = lt / G.tiles, tile = lt - b * G.tiles;
        const int x0 = (tile % G.tiles_x) * TS, y0 = (tile / G.tiles_x) * TH;
        const float *gb = G.gout + (long)b * G.gout_bs, *ib = G.in + (long)b * G.in_bs;
        float *tg = wg_sm + s * BUF, *tin = tg + COB * GP;
        for (int e = threadIdx.x; e < COB * TH * TS; e += WG_T) {
            const int c = e / (TH * TS), r = (e / TS) % TH, q = e % TS, y = y0 + r, x = x0 + q;
            const bool ok = co0 + c < Cout && y < H && x < W;
            cp4(tg + c * GP + r * TS + q, ok ? gb + (long)(co0 + c) * G.gout_cs + (long)y * W + x : gb, ok);
        }
        for (int e = threadIdx.x; e < CIB * (TH + 2) * (TS + 2); e += WG_T) {
            const int c = e / ((TH + 2) * (TS + 2)), r = (e / (TS + 2)) % (TH + 2), q = e % (TS + 2);
            const int y = y0 + r - 1, x = x0 + q - 1;
            const bool ok = ci0 + c < Cin && y >= 0 && y < H && x >= 0 && x < W;
            cp4(tin + c * IP + r * IW + q, ok ? ib + (long)(ci0 + c) * G.in_cs + (long)y * W + x : ib, ok);
        }
        cp_commit();
    };
    stage(0, A.t0 + blockIdx.x);
    for (int t = A.t0 + blockIdx.x, s = 0; t < A.t1; t += gridDim.x, s ^= 1) {
        if (t + (int)gridDim.x < A.t1) {
            stage(s ^ 1, t + gridDim.x);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const float *tg = wg_sm + s * BUF, *tin = tg + COB * GP;
#pragma unroll 1
        for (int q = slice; q < TH * TS / 4; q += NS) {  // groups of four pixels
            const int r = q / (TS / 4), x = (q % (TS / 4)) * 4;
            float4 g[4];
#pragma unroll
            for (int j = 0; j < 4; j++)
                g[j] = *reinterpret_cast<const float4 *>(tg + (cg + CG * j) * GP + r * TS + x);
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int ky = 0; ky < 3; ky++) {
                    const float *row = tin + (ig + IG * i) * IP + (r + ky) * IW + x;
                    const float4 va = *reinterpret_cast<const float4 *>(row);
                    const float2 vb = *reinterpret_cast<const float2 *>(row + 4);
                    const float v[6] = {va.x, va.y, va.z, va.w, vb.x, vb.y};
#pragma unroll
                    for (int kx = 0; kx < 3; kx++)
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            float a = acc[j][i][3 * ky + kx];
                            a += g[j].x * v[kx];
                            a += g[j].y * v[kx + 1];
                            a += g[j].z * v[kx + 2];
                            a += g[j].w * v[kx + 3];
                            acc[j][i][3 * ky + kx] = a;
                        }
                }
        }
        if (blockIdx.z == 0 && threadIdx.x < COB * BT) {  // bias: BT neighbouring threads per channel
            const float *g = tg + (threadIdx.x / BT) * GP;
            for (int q = (threadIdx.x % BT) * 4; q < TH * TS; q += BT * 4) {
                const float4 v = *reinterpret_cast<const float4 *>(g + q);
                bsum += (v.x + v.y) + (v.z + v.w);
            }
        }
        __syncthreads();
    }
    // slices side by side in shared memory, [slice][j][i][k][thread of the slice]
    constexpr int PT = CG * IG;
    const int pt = threadIdx.x % PT;
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int k = 0; k < 9; k++)
                wg_sm[(slice * 72 + (j * 2 + i) * 9 + k) * PT + pt] = acc[j][i][k];
    __syncthreads();
    const int nw = Cout * Cin * 9;
    float *dst = A.part + (long)blockIdx.x * (nw + Cout);
    for (int e = threadIdx.x; e < COB * CIB * 9; e += WG_T) {
        const int c = e / (CIB * 9), d = (e / 9) % CIB, k = e % 9;  // channels c, d of the block
        if (co0 + c < Cout && ci0 + d < Cin) {
            const float *p = wg_sm + (((c / CG) * 2 + d / IG) * 9 + k) * PT + (d % IG) * CG + c % CG;
            float a = 0.f;
#pragma unroll
            for (int sl = 0; sl < NS; sl++) a += p[(long)sl * 72 * PT];
            dst[((long)(co0 + c) * Cin + ci0 + d) * 9 + k] = a;
        }
    }
    if (blockIdx.z == 0) {
#pragma unroll
        for (int o = BT / 2; o > 0; o >>= 1) bsum += __shfl_down_sync(0xffffffffu, bsum, o, BT);
        const int c = threadIdx.x / BT;
        if (threadIdx.x < COB * BT && threadIdx.x % BT == 0 && co0 + c < Cout) dst[nw + co0 + c] = bsum;
    }
}

// Sum of the CTAs' partials (deterministic, FP64); accumulate adds to the
// gradients already stored.  Rounds of partials: carry_in adds the totals of the
// earlier ones, carry_out stores the totals instead of the gradients.  32 outputs per CTA, RG threads each: thread g of
// an output sums partials g, g + RG, ..., then the RG sums are added in order.
// One thread per output walked all partials with one load in flight.
constexpr int RG = 8;

__global__ void __launch_bounds__(32 * RG)
    k_reduce_partials(const float *__restrict__ part, int nparts, int len, float *__restrict__ gw,
                      float *__restrict__ gb, int nw, int accumulate, double *__restrict__ total, int carry_in,
                      int carry_out)
{
    __shared__ double sh[RG][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    double a = 0.0;
    if (e < len) {
        constexpr int U = 8;  // loads in flight
        for (int p0 = g; p0 < nparts; p0 += U * RG) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; u++) v[u] = p0 + u * RG < nparts ? part[(long)(p0 + u * RG) * len + e] : 0.f;
#pragma unroll
            for (int u = 0; u < U; u++) a += (double)v[u];
        }
    }
    sh[g][lane] = a;
    __syncthreads();
    if (g == 0 && e < len) {
#pragma unroll
        for (int i = 1; i < RG; i++) a += sh[i][lane];
        if (carry_in) a += total[e];
        if (carry_out) {
            total[e] = a;
            return;
        }
        float *dst = e < nw ? gw + e : gb + (e - nw);
        *dst = accumulate ? *dst + (float)a : (float)a;
    }
}

__global__ void k_relu_bwd(const float *__restrict__ act, float *__restrict__ g, long n)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        if (!(act[i] > 0.f)) g[i] = 0.f;
}

// grad = 2 (pred - target) / n; per-block partial sums of (pred - target)^2.
__global__ void k_mse(const float *__restrict__ pred, const float *__restrict__ target, float *__restrict__ grad,
                      long n, float inv_n, double *__restrict__ loss_part)
{
    __shared__ double sh[256];
    double a = 0.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float d = pred[i] - target[i];
        grad[i] = 2.f * d * inv_n;
        a += (double)d * d;
    }
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss_part[blockIdx.x] = sh[0];
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       long n, float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// y = x * sqrt(s) (mode 0), x / sqrt(s) (mode 1), y += x / sqrt(s) (mode 2)
__global__ void k_scale(const float *__restrict__ x, const float *__restrict__ sc, float *__restrict__ y, long n,
                        int mode)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float r = sqrtf(sc[i]);
        if (mode == 0)
            y[i] = x[i] * r;
        else if (mode == 1)
            y[i] = x[i] / r;
        else
            y[i] += x[i] / r;
    }
}

// Training targets of the network (channel stride n): t0 = (c_next - c_cur) * sqrt(s);
// t_k = t0 where group[i] == k, else 0 (k = 1..4, the wavelet scale groups).
__global__ void k_targets(const float *__restrict__ c_next, const float *__restrict__ c_cur,
                          const float *__restrict__ sc, const signed char *__restrict__ group, float *__restrict__ t,
                          long n)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const float d = (c_next[i] - c_cur[i]) * sqrtf(sc[i]);
        const int g = group[i];
        t[i] = d;
#pragma unroll
        for (int k = 1; k <= 4; k++) t[k * n + i] = (g == k) ? d : 0.f;
    }
}

// --- deflated warm start: Galerkin correction over predicted directions ----
constexpr int kMaxDir = FEWHA_MAX_DEFLATE;
constexpr int kChunks = 32;

// r0 = (b - b_prev) + r_prev (the warm restart of Algorithm 3)
__global__ void k_warm_residual(const float *__restrict__ b, const float *__restrict__ b_prev,
                                const float *__restrict__ r_prev, float *__restrict__ r0, long n)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        r0[i] = (b[i] - b_prev[i]) + r_prev[i];
}

struct DotPairs {
    const float *x[64], *y[64];
};

// part[p * kChunks + chunk] = partial (x_p, y_p) over one chunk (FP32 per
// thread, FP64 across the block; fixed order, deterministic).
__global__ void __launch_bounds__(256) k_dots(const __grid_constant__ DotPairs P, long n, double *__restrict__ part)
{
    __shared__ double sh[8];
    const int p = blockIdx.x, chunk = blockIdx.y;
    const long per = (n + kChunks - 1) / kChunks, lo = chunk * per, hi = min(n, lo + per);
    const float *x = P.x[p], *y = P.y[p];
    float a = 0.f;
    for (long i = lo + threadIdx.x; i < hi; i += blockDim.x) a += x[i] * y[i];
    double d = a;
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += sh[w];
        part[p * kChunks + chunk] = t;
    }
}

// One thread: G = sym(D^T Q), g = D^T r0, Cholesky of G with directions whose
// pivot falls below 1e-10 of their diagonal dropped, w = G^{-1} g;
// ||r0 - Q w||^2 = (r0,r0) - 2 w.(Q^T r0) + w^T (Q^T Q) w.  The correction is
// taken when that is below (r0, r0).
// info: [0] taken, [1] ||r0 - Q w||, [2] ||r0||, [3] kept directions, [4..4+nd) w
__global__ void k_deflate_solve(const double *__restrict__ part, int nd, double *__restrict__ info,
                                float *__restrict__ wf)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    auto sum = [&](int p) {
        double t = 0.0;
        for (int c = 0; c < kChunks; c++) t += part[p * kChunks + c];
        return t;
    };
    // pair order: (d_i, r0) i; (d_i, q_j) i,j; (q_i, r0) i; (q_i, q_j) i,j; (r0, r0)
    double G[kMaxDir][kMaxDir], QQ[kMaxDir][kMaxDir], g[kMaxDir], qr[kMaxDir], L[kMaxDir][kMaxDir], w[kMaxDir];
    int keep[kMaxDir];
    int p = 0;
    for (int i = 0; i < nd; i++) g[i] = sum(p++);
    for (int i = 0; i < nd; i++)
        for (int j = 0; j < nd; j++) G[i][j] = sum(p++);
    for (int i = 0; i < nd; i++) qr[i] = sum(p++);
    for (int i = 0; i < nd; i++)
        for (int j = 0; j < nd; j++) QQ[i][j] = sum(p++);
    const double rr = sum(p++);
    int kept = 0;
    for (int j = 0; j < nd; j++) {
        keep[j] = 0;
        double d = 0.5 * (G[j][j] + G[j][j]);
        const double dj = d;
        for (int k = 0; k < j; k++)
            if (keep[k]) d -= L[j][k] * L[j][k];
        if (!(dj > 0.0) || !(d > 1e-10 * dj)) {
            for (int k = 0; k <= j; k++) L[j][k] = 0.0;
            continue;
        }
        keep[j] = 1;
        kept++;
        L[j][j] = sqrt(d);
        for (int i = j + 1; i < nd; i++) {
            double v = 0.5 * (G[i][j] + G[j][i]);
            for (int k = 0; k < j; k++)
                if (keep[k]) v -= L[i][k] * L[j][k];
            L[i][j] = v / L[j][j];
        }
    }
    double y[kMaxDir];
    for (int i = 0; i < nd; i++) {
        y[i] = 0.0;
        if (!keep[i]) continue;
        double v = g[i];
        for (int k = 0; k < i; k++)
            if (keep[k]) v -= L[i][k] * y[k];
        y[i] = v / L[i][i];
    }
    for (int i = nd - 1; i >= 0; i--) {
        w[i] = 0.0;
        if (!keep[i]) continue;
        double v = y[i];
        for (int k = i + 1; k < nd; k++)
            if (keep[k]) v -= L[k][i] * w[k];
        w[i] = v / L[i][i];
    }
    double rr1 = rr;
    for (int i = 0; i < nd; i++) {
        rr1 -= 2.0 * w[i] * qr[i];
        for (int j = 0; j < nd; j++) rr1 += w[i] * QQ[i][j] * w[j];
    }
    bool ok = kept > 0 && rr1 < rr && rr1 == rr1;
    for (int i = 0; i < nd; i++) ok = ok && (w[i] == w[i]);
    info[0] = ok ? 1.0 : 0.0;
    info[1] = sqrt(fmax(rr1, 0.0));
    info[2] = sqrt(rr);
    info[3] = kept;
    for (int i = 0; i < nd; i++) {
        info[4 + i] = w[i];
        wf[i] = (float)w[i];
    }
}

// If taken: c += D w, r_prev <- r0 - Q w, b_prev <- b.
__global__ void k_deflate_update(const double *__restrict__ info, const float *__restrict__ wf, int nd,
                                 const float *__restrict__ D, long ldd, const float *__restrict__ Q, long ldq,
                                 const float *__restrict__ b, const float *__restrict__ r0, float *__restrict__ c,
                                 float *__restrict__ b_prev, float *__restrict__ r_prev, long n)
{
    // not taken: the plain warm restart r0 is folded into the state
    const bool taken = info[0] != 0.0;
    if (!taken) {
        for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
            r_prev[i] = r0[i];
            b_prev[i] = b[i];
        }
        return;
    }
    float w[kMaxDir];
#pragma unroll
    for (int j = 0; j < kMaxDir; j++) w[j] = j < nd ? wf[j] : 0.f;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        float cv = c[i], rv = r0[i];
        for (int j = 0; j < nd; j++) {
            cv += w[j] * D[j * ldd + i];
            rv -= w[j] * Q[j * ldq + i];
        }
        c[i] = cv;
        r_prev[i] = rv;
        b_prev[i] = b[i];
    }
}

int ck() { return cudaGetLastError() == cudaSuccess ? FEWHA_OK : FEWHA_ERR_CUDA; }

// One launch of k_conv3x3, group by group.
struct ConvLaunch {
    ConvArgs A{};
    long blocks = 0;
    ConvLaunch(const float *w, const float *bias, int Cin, int Cout, int relu, int wt_mode)
    {
        A.w = w, A.bias = bias, A.Cin = Cin, A.Cout = Cout, A.relu = relu, A.wt_mode = wt_mode;
    }
    bool add(const float *in, long in_bs, long in_cs, float *out, long out_bs, long out_cs, const float *mask, int B,
             int H, int W)
    {
        const int tx = (W + TX - 1) / TX, ty = (H + TY - 1) / TY;
        const long z = (long)B * ((A.Cout + CO_T - 1) / CO_T), tiles = (long)tx * ty;
        if (z > 65535 || tiles > 0x7FFFFFFFL || blocks + z * tiles > 0x7FFFFFFFL) return false;
        A.g[A.ng++] = ConvGroup{in, mask, out, in_bs, in_cs, out_bs, out_cs, H, W, tx, (int)tiles, (int)blocks};
        blocks += z * tiles;
        return true;
    }
    int run(cudaStream_t s) const
    {
        k_conv3x3<<<(unsigned)blocks, NT, 0, s>>>(A);
        return ck();
    }
};

// One weight gradient: partials over the tiles of all groups, then their sum.
struct WgradLaunch {
    WgradArgs A{};
    long ntiles = 0, parts = 0;  // parts: workspace capacity, TS x TS tiles
    WgradLaunch(int Cin, int Cout) { A.Cin = Cin, A.Cout = Cout; }
    bool add(const float *in, long in_bs, long in_cs, const float *gout, long gout_bs, long gout_cs, int B, int H, int W)
    {
        const long tx = (W + TS - 1) / TS, tiles = tx * ((H + TH - 1) / TH);
        if (ntiles + tiles * B > 0x7fffffffL) return false;
        A.g[A.ng++] = WgradGroup{in, gout, in_bs, in_cs, gout_bs, gout_cs, H, W, (int)tx, (int)tiles, (int)ntiles};
        ntiles += tiles * B;
        parts += tx * ((H + TS - 1) / TS) * B;
        return true;
    }
    template <int CG, int IG>
    int partials(int n, cudaStream_t s)
    {
        auto kern = k_conv3x3_wgrad_partial<CG, IG>;
        constexpr int cob = 4 * CG, cib = 2 * IG;
        constexpr size_t bytes = wg_smem<CG, IG>();
        const dim3 grid(n, (A.Cout + cob - 1) / cob, (A.Cin + cib - 1) / cib);
        if (grid.y > 65535 || grid.z > 65535) return FEWHA_ERR_ARG;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
            return FEWHA_ERR_CUDA;
        kern<<<grid, WG_T, bytes, s>>>(A);
        return ck();
    }
    template <int CG, int IG>
    int gradient(float *gw, float *gb, int accumulate, float *workspace, cudaStream_t s)
    {
        constexpr int span = wg_span(WG_T / (CG * IG));
        const int len = A.Cout * A.Cin * 9 + A.Cout;
        const bool rounds = ntiles > (long)WG_CTAS * span;
        // n <= ntiles.  With rounds the workspace holds WG_CTAS partials: the FP64
        // totals (2 len floats and one for their alignment) lie behind the first n.
        static_assert(WG_CTAS - WG_ROUND >= 3, "room for the totals");
        const int n = rounds ? WG_ROUND : (int)(parts < WG_CTAS ? parts : WG_CTAS);
        const long most = (long)n * (span - 1), nr = rounds ? (ntiles + most - 1) / most : 1;
        double *total = reinterpret_cast<double *>((reinterpret_cast<size_t>(workspace + (long)n * len) + 7) & ~(size_t)7);
        A.part = workspace;
        for (long r = 0; r < nr; r++) {
            A.t0 = (int)(r * ntiles / nr);  // rounds of equal size, n < tiles <= most
            A.t1 = (int)((r + 1) * ntiles / nr);
            int st = partials<CG, IG>(n, s);
            if (st != FEWHA_OK) return st;
            k_reduce_partials<<<(len + 31) / 32, 32 * RG, 0, s>>>(workspace, n, len, gw, gb, len - A.Cout, accumulate,
                                                                  total, r > 0, r + 1 < nr);
            if ((st = ck()) != FEWHA_OK) return st;
        }
        return FEWHA_OK;
    }
    int run(float *gw, float *gb, int accumulate, float *workspace, cudaStream_t s)
    {
        // channel block: 32 x 32, or narrow on the side with at most 8 output / 4
        // input channels (the padding would be most of the work)
        return A.Cout <= 8  ? gradient<2, 16>(gw, gb, accumulate, workspace, s)
               : A.Cin <= 4 ? gradient<8, 2>(gw, gb, accumulate, workspace, s)
                            : gradient<8, 16>(gw, gb, accumulate, workspace, s);
    }
};

}  // namespace

extern "C" {

int fewha_conv3x3_fwd(const float *in, long in_bs, long in_cs, int Cin, const float *w, const float *bias,
                      float *out, long out_bs, long out_cs, int Cout, int B, int H, int W, int relu, cudaStream_t s)
{
    if (!in || !w || !out || Cin < 1 || Cout < 1 || B < 1 || H < 1 || W < 1) return FEWHA_ERR_ARG;
    ConvLaunch L(w, bias, Cin, Cout, relu, 0);
    if (!L.add(in, in_bs, in_cs, out, out_bs, out_cs, nullptr, B, H, W)) return FEWHA_ERR_ARG;
    return L.run(s);
}

int fewha_conv3x3_bwd_data_relu(const float *gout, long gout_bs, long gout_cs, int Cout, const float *w,
                                const float *act, float *gin, long gin_bs, long gin_cs, int Cin, int B, int H, int W,
                                cudaStream_t s)
{
    if (!gout || !w || !gin || Cin < 1 || Cout < 1 || B < 1 || H < 1 || W < 1) return FEWHA_ERR_ARG;
    ConvLaunch L(w, nullptr, Cout, Cin, 0, 1);
    if (!L.add(gout, gout_bs, gout_cs, gin, gin_bs, gin_cs, act, B, H, W)) return FEWHA_ERR_ARG;
    return L.run(s);
}

int fewha_conv3x3_bwd_data(const float *gout, long gout_bs, long gout_cs, int Cout, const float *w, float *gin,
                           long gin_bs, long gin_cs, int Cin, int B, int H, int W, cudaStream_t s)
{
    return fewha_conv3x3_bwd_data_relu(gout, gout_bs, gout_cs, Cout, w, nullptr, gin, gin_bs, gin_cs, Cin, B, H, W, s);
}

long fewha_conv3x3_wgrad_workspace(int Cin, int Cout, int B, int H, int W)
{
    if (Cin < 1 || Cout < 1 || B < 1 || H < 1 || W < 1) return 0;
    const long tiles = (long)((W + TS - 1) / TS) * ((H + TS - 1) / TS) * B;
    return tiles * ((long)Cout * Cin * 9 + Cout);
}

int fewha_conv3x3_bwd_weight(const float *in, long in_bs, long in_cs, int Cin, const float *gout, long gout_bs,
                             long gout_cs, int Cout, int B, int H, int W, float *gw, float *gb, int accumulate,
                             float *workspace, cudaStream_t s)
{
    if (!in || !gout || !gw || !gb || !workspace || Cin < 1 || Cout < 1 || B < 1 || H < 1 || W < 1)
        return FEWHA_ERR_ARG;
    const long tiles = (long)((W + TS - 1) / TS) * ((H + TS - 1) / TS) * B;
    // the call's size limit (fewha.h): a whole tile's inputs and gradients in 200 KB
    const size_t smem = ((size_t)Cin * (TS + 2) * (TS + 2) + (size_t)Cout * TS * TS) * sizeof(float);
    if (smem > 200 * 1024 || tiles > 0x7fffffffL) return FEWHA_ERR_ARG;
    WgradLaunch L(Cin, Cout);
    if (!L.add(in, in_bs, in_cs, gout, gout_bs, gout_cs, B, H, W)) return FEWHA_ERR_ARG;
    return L.run(gw, gb, accumulate, workspace, s);
}

// The training network (C0 -> C -> C -> C3, ReLU after the first two) over groups
// of equal-size images: image i of group g starts off[g] + i side[g]^2 floats
// into a channel of x, y and gy; the hidden activations and their gradients are
// (count[g], C, side, side) arrays of their own.
static int net_args_ok(const fewha_net *N)
{
    if (!N || N->ngroups < 1 || N->ngroups > kMaxGroups || N->C0 < 1 || N->C < 1 || N->C3 < 1) return 0;
    for (int i = 0; i < 3; i++)
        if (!N->w[i] || !N->b[i]) return 0;
    for (int g = 0; g < N->ngroups; g++)
        if (N->count[g] < 1 || N->side[g] < 1 || N->off[g] < 0 || !N->h1[g] || !N->h2[g]) return 0;
    return 1;
}

long fewha_convnet_workspace(const fewha_net *N)
{
    if (!N || N->ngroups < 1 || N->ngroups > kMaxGroups || N->C0 < 1 || N->C < 1 || N->C3 < 1) return 0;
    long tiles = 0;
    for (int g = 0; g < N->ngroups; g++) {
        if (N->count[g] < 1 || N->side[g] < 1) return 0;
        const long t = (N->side[g] + TS - 1) / TS;
        tiles += N->count[g] * t * t;
    }
    const int C = N->C > N->C3 ? N->C : N->C3, M = C > N->C0 ? C : N->C0;  // the largest gradient of the three
    return (tiles < WG_CTAS ? tiles : WG_CTAS) * ((long)N->C * M * 9 + C);
}

int fewha_convnet_fwd(const fewha_net *N, const float *x, long x_cs, float *y, long y_cs, cudaStream_t s)
{
    if (!net_args_ok(N) || !x || !y) return FEWHA_ERR_ARG;
    ConvLaunch L1(N->w[0], N->b[0], N->C0, N->C, 1, 0), L2(N->w[1], N->b[1], N->C, N->C, 1, 0),
        L3(N->w[2], N->b[2], N->C, N->C3, 0, 0);
    for (int g = 0; g < N->ngroups; g++) {
        const int B = N->count[g], S = N->side[g];
        const long hw = (long)S * S, hb = N->C * hw;
        if (!L1.add(x + N->off[g], hw, x_cs, N->h1[g], hb, hw, nullptr, B, S, S) ||
            !L2.add(N->h1[g], hb, hw, N->h2[g], hb, hw, nullptr, B, S, S) ||
            !L3.add(N->h2[g], hb, hw, y + N->off[g], hw, y_cs, nullptr, B, S, S))
            return FEWHA_ERR_ARG;
    }
    int st = L1.run(s);
    if (st == FEWHA_OK) st = L2.run(s);
    return st == FEWHA_OK ? L3.run(s) : st;
}

int fewha_convnet_bwd(const fewha_net *N, const float *x, long x_cs, const float *gy, long gy_cs, float *workspace,
                      cudaStream_t s)
{
    if (!net_args_ok(N) || !x || !gy || !workspace) return FEWHA_ERR_ARG;
    for (int i = 0; i < 3; i++)
        if (!N->gw[i] || !N->gb[i]) return FEWHA_ERR_ARG;
    WgradLaunch W1(N->C0, N->C), W2(N->C, N->C), W3(N->C, N->C3);
    ConvLaunch D3(N->w[2], nullptr, N->C3, N->C, 0, 1), D2(N->w[1], nullptr, N->C, N->C, 0, 1);
    for (int g = 0; g < N->ngroups; g++) {
        if (!N->g1[g] || !N->g2[g]) return FEWHA_ERR_ARG;
        const int B = N->count[g], S = N->side[g];
        const long hw = (long)S * S, hb = N->C * hw;
        const float *xg = x + N->off[g], *gg = gy + N->off[g];
        if (!W3.add(N->h2[g], hb, hw, gg, hw, gy_cs, B, S, S) || !W2.add(N->h1[g], hb, hw, N->g2[g], hb, hw, B, S, S) ||
            !W1.add(xg, hw, x_cs, N->g1[g], hb, hw, B, S, S) ||
            !D3.add(gg, hw, gy_cs, N->g2[g], hb, hw, N->h2[g], B, S, S) ||
            !D2.add(N->g2[g], hb, hw, N->g1[g], hb, hw, N->h1[g], B, S, S))
            return FEWHA_ERR_ARG;
    }
    int st = W3.run(N->gw[2], N->gb[2], 0, workspace, s);
    if (st == FEWHA_OK) st = D3.run(s);
    if (st == FEWHA_OK) st = W2.run(N->gw[1], N->gb[1], 0, workspace, s);
    if (st == FEWHA_OK) st = D2.run(s);
    return st == FEWHA_OK ? W1.run(N->gw[0], N->gb[0], 0, workspace, s) : st;
}

int fewha_relu_bwd(const float *act, float *g, long n, cudaStream_t s)
{
    if (!act || !g || n < 0) return FEWHA_ERR_ARG;
    k_relu_bwd<<<512, 256, 0, s>>>(act, g, n);
    return ck();
}

int fewha_mse_grad(const float *pred, const float *target, float *grad, long n, double *loss_part512, cudaStream_t s)
{
    if (!pred || !target || !grad || !loss_part512 || n < 1) return FEWHA_ERR_ARG;
    k_mse<<<512, 256, 0, s>>>(pred, target, grad, n, 1.f / (float)n, loss_part512);
    return ck();
}

int fewha_adam_step(float *param, const float *grad, float *m, float *v, long n, float lr, float beta1, float beta2,
                    float eps, int step, cudaStream_t s)
{
    if (!param || !grad || !m || !v || n < 1 || step < 1) return FEWHA_ERR_ARG;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adam<<<512, 256, 0, s>>>(param, grad, m, v, n, lr, beta1, beta2, eps, c1, c2);
    return ck();
}

int fewha_scale(const float *x, const float *s_, float *y, long n, int mode, cudaStream_t s)
{
    if (!x || !s_ || !y || n < 1 || mode < 0 || mode > 2) return FEWHA_ERR_ARG;
    k_scale<<<512, 256, 0, s>>>(x, s_, y, n, mode);
    return ck();
}

int fewha_learned_targets(const float *c_next, const float *c_cur, const float *scale, const signed char *group,
                          float *targets5, long n, cudaStream_t s)
{
    if (!c_next || !c_cur || !scale || !group || !targets5 || n < 1) return FEWHA_ERR_ARG;
    k_targets<<<512, 256, 0, s>>>(c_next, c_cur, scale, group, targets5, n);
    return ck();
}

int fewha_deflate_warm_start(const float *b, const float *D, long ldd, const float *Q, long ldq, int nd, float *c,
                             float *b_prev, float *r_prev, long n, float *r0_work, double *work, double *info,
                             cudaStream_t s)
{
    if (!b || !D || !Q || !c || !b_prev || !r_prev || !r0_work || !work || !info || n < 1 || nd < 1 ||
        nd > kMaxDir || ldd < n || ldq < n)
        return FEWHA_ERR_ARG;
    static_assert(2 * kMaxDir + kMaxDir * kMaxDir <= 64 && kMaxDir * kMaxDir + 1 <= 64, "dot pairs per launch");
    static_assert((2 * kMaxDir + 2 * kMaxDir * kMaxDir + 1) * kChunks <= FEWHA_DEFLATE_WORK_DOUBLES, "work");
    static_assert(4 + kMaxDir + (kMaxDir + 1) / 2 <= FEWHA_DEFLATE_INFO_DOUBLES, "info");
    k_warm_residual<<<512, 256, 0, s>>>(b, b_prev, r_prev, r0_work, n);
    DotPairs P;
    int p = 0;
    for (int i = 0; i < nd; i++) P.x[p] = D + i * ldd, P.y[p++] = r0_work;
    for (int i = 0; i < nd; i++)
        for (int j = 0; j < nd; j++) P.x[p] = D + i * ldd, P.y[p++] = Q + j * ldq;
    for (int i = 0; i < nd; i++) P.x[p] = Q + i * ldq, P.y[p++] = r0_work;
    // (q_i, q_j) and (r0, r0) go in a second launch (at most 64 pairs each)
    DotPairs P2;
    int p2 = 0;
    for (int i = 0; i < nd; i++)
        for (int j = 0; j < nd; j++) P2.x[p2] = Q + i * ldq, P2.y[p2++] = Q + j * ldq;
    P2.x[p2] = r0_work, P2.y[p2++] = r0_work;
    k_dots<<<dim3(p, kChunks), 256, 0, s>>>(P, n, work);
    k_dots<<<dim3(p2, kChunks), 256, 0, s>>>(P2, n, work + (long)p * kChunks);
    float *wf = reinterpret_cast<float *>(info + 4 + kMaxDir);
    k_deflate_solve<<<1, 32, 0, s>>>(work, nd, info, wf);
    k_deflate_update<<<512, 256, 0, s>>>(info, wf, nd, D, ldd, Q, ldq, b, r0_work, c, b_prev, r_prev, n);
    return ck();
}

}  // extern "C"

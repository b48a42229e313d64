// warmstart.cu -- learned warm start of a batch (initial fields from a CNN).
//
// Time to a steady state is set by how far the initial fields are from it.
// A convolutional network maps each domain's parameters (kind, aspect ratio,
// Reynolds, Grashof and Prandtl numbers, rotation ratio), broadcast on a
// 256 (z) x 128 (r) canvas together with the normalised coordinates, to the
// steady fields u_r, u_z, u_theta (in units of the lid speed) and T.  The
// canvases are resampled onto every domain's grid and the batch starts from
// the equilibria of those fields (the same initialisation as
// axlbm_batch_set_fields_all).
//
// Network (weights in BF16, accumulation in FP32): a four-level U-Net of 3x3
// convolutions with ReLU, channels 32, 64, 96, 128 at 256 x 128, 128 x 64,
// 64 x 32 and 32 x 16 -- per level two convolutions (8 -> 32 -> 32 first),
// 2x2 average pooling between levels -- then, from the bottom up, nearest
// upsampling and concatenation with the level's skip (deep channels first),
// two convolutions per level (224 -> 96 -> 96, 160 -> 64 -> 64,
// 96 -> 32 -> 32), and a 1x1 head 32 -> 4 without activation: 0.91 M weights.
// Activations are NHWC in BF16.  Every 3x3 convolution -- forward, and in
// training the input and weight gradients -- is a kernel of this library on
// the tensor cores (ws_conv.cuh: mma.sync BF16 with FP32 accumulation); no
// im2col matrix is formed and no GEMM library is called.  The pools come out
// of the epilogue of the convolution before them, the upsampled and
// concatenated input of a decoder level is read from its two sources by the
// convolution itself.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "batch_internal.h"
#include "internal.h"
#include "ws_conv.cuh"

struct axlbm_ws_train;  // training state (warmstart.cu, below)

namespace {

constexpr int kLevels = 4;
constexpr int kCh[kLevels] = {32, 64, 96, 128};

// The activations of one pass over n canvases: x0 the input canvas; per
// encoder level the outputs of its two convolutions (a, e) and the pooled e
// (p); per decoder level the outputs of its two convolutions (b, d).
struct Acts {
    __nv_bfloat16 *x0 = nullptr;
    __nv_bfloat16 *a[kLevels] = {}, *e[kLevels] = {}, *p[kLevels - 1] = {};
    __nv_bfloat16 *b[kLevels - 1] = {}, *d[kLevels - 1] = {};
};

}  // namespace

struct axlbm_ws {
    cudaStream_t stream;
    __nv_bfloat16* w;  // all layers, packed as in include/axlbm.h
    std::vector<size_t> woff, boff;
    int num_sms;
    int chunk;  // canvases that `act` holds
    Acts act;
    axlbm_ws_train* train;  // allocated by the first training call
    std::string err;
};

namespace {

using bf16 = __nv_bfloat16;
thread_local std::string g_ws_error;

constexpr int kH = 256, kW = 128;  // canvas rows (z) and columns (r)
constexpr int kFeat = AXLBM_WS_FEATURES;

struct Layer {
    int cin, cout, k;  // k: 3 (3x3, padding 1) or 1
};
// encoder levels 0-3 (two layers each), decoder levels 2, 1, 0 (two each), head
constexpr int kLayers = 15;
constexpr Layer kNet[kLayers] = {{8, 32, 3},   {32, 32, 3},  {32, 64, 3},  {64, 64, 3},  {64, 96, 3},
                                 {96, 96, 3},  {96, 128, 3}, {128, 128, 3}, {224, 96, 3}, {96, 96, 3},
                                 {160, 64, 3}, {64, 64, 3},  {96, 32, 3},  {32, 32, 3},  {32, 4, 1}};
constexpr int enc_layer(int l) { return 2 * l; }            // first layer of encoder level l
constexpr int dec_layer(int l) { return 8 + 2 * (2 - l); }  // first layer of decoder level l (0..2)
constexpr int kHead = 14;

size_t net_values() {
    size_t n = 0;
    for (const Layer& l : kNet) n += (size_t)l.cout * l.cin * l.k * l.k + l.cout;
    return n;
}

axlbm_status wfail(axlbm_ws* w, axlbm_status st, const std::string& m) {
    if (w) w->err = m; else g_ws_error = m;
    return st;
}

// ---------------------------------------------------------------- kernels

// Input canvas: the features broadcast over the canvas plus r/R and z/H at
// the pixel centres, NHWC [n][kH][kW][8].
__global__ void k_ws_input(const float* feat, int n, bf16* x) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long total = (long long)n * kH * kW;
    if (i >= total) return;
    const int c = int(i % kW), r = int((i / kW) % kH), b = int(i / ((long long)kH * kW));
    __align__(16) bf16 o[8];
#pragma unroll
    for (int f = 0; f < kFeat; ++f) o[f] = __float2bfloat16(feat[b * kFeat + f]);
    o[6] = __float2bfloat16((c + 0.5f) / kW);
    o[7] = __float2bfloat16((r + 0.5f) / kH);
    *reinterpret_cast<uint4*>(x + i * 8) = *reinterpret_cast<const uint4*>(o);
}

// 1x1 head 32 -> 4 (no activation), to FP32 canvases [n][4][kH][kW]: one
// pixel per thread, its 64 bytes in four loads, the weights in shared memory.
__global__ void __launch_bounds__(256) k_ws_head(const bf16* x, const bf16* wt, const bf16* bias, int n, float* out) {
    __shared__ float ws[4 * 32], bs[4];
    if (threadIdx.x < 128) ws[threadIdx.x] = __bfloat162float(wt[threadIdx.x]);
    if (threadIdx.x < 4) bs[threadIdx.x] = __bfloat162float(bias[threadIdx.x]);
    __syncthreads();
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= (long long)n * kH * kW) return;
    const int b = int(p / ((long long)kH * kW));
    const long long pix = p % ((long long)kH * kW);
    float v[32];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 u = reinterpret_cast<const uint4*>(x + p * 32)[q];
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(h[e]);
            v[8 * q + 2 * e] = f.x;
            v[8 * q + 2 * e + 1] = f.y;
        }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        float s = bs[o];
#pragma unroll
        for (int c = 0; c < 32; ++c) s = fmaf(ws[o * 32 + c], v[c], s);
        out[((long long)b * 4 + o) * kH * kW + pix] = s;
    }
}

// Fields [5][nz][nr] (rho, u_r, u_z, u_theta, T) of every domain from its
// canvas, bilinear at normalised (rn, zn) in [0, 1]: pixel centres at
// ((i + 1/2)/kW, (j + 1/2)/kH), clamped at the edges.  A block takes kFieldRows
// rows of up to kFieldCols columns of one domain; a thread walks down one
// column and keeps its values interpolated along r at the two canvas rows
// around it, which several domain rows share: FP64 instructions bound this
// kernel (an SM takes 19 cycles for one of a warp), and this takes about
// 12 of them per node and 16 per new canvas row, where sampling every node
// afresh took over a hundred with its divisions.
constexpr int kFieldCols = 128, kFieldRows = 32;
struct FieldDom {
    axlbm_ws_domain d;
    long long out;  // first value of the domain's fields
    int block0;     // first block
};
// The domains of a launch are kernel arguments (22 of the 32 KB there may be): a call needs no memory for its list.
constexpr int kFieldDoms = 256;
struct FieldDoms {
    FieldDom d[kFieldDoms];
};
__global__ void __launch_bounds__(kFieldCols)
k_ws_fields(const float* canvas, const __grid_constant__ FieldDoms doms, int n, float* fields) {
    __shared__ double row_f[kFieldRows], row_g[kFieldRows];  // weights of a row's two canvas rows, and the first of them
    __shared__ int row_y[kFieldRows];
    int lo = 0, hi = n - 1;  // the domain of this block
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (doms.d[mid].block0 <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const FieldDom& F = doms.d[lo];
    const axlbm_ws_domain& D = F.d;
    const int cols = (D.nr - 1) / kFieldCols + 1, b = blockIdx.x - F.block0, rb = b / cols;
    const int j = (b - rb * cols) * kFieldCols + threadIdx.x, k0 = rb * kFieldRows, k1 = k0 + min(kFieldRows, D.nz - k0);
    if (threadIdx.x < kFieldRows) {
        const double zn = (D.z_first + ((double)k0 + threadIdx.x) - D.z_bottom) / D.height;
        const double yc = fmin(fmax(zn * kH - 0.5, 0.0), kH - 1.0);
        row_y[threadIdx.x] = min(int(yc), kH - 2);
        row_f[threadIdx.x] = yc - row_y[threadIdx.x];
        row_g[threadIdx.x] = 1 - row_f[threadIdx.x];
    }
    __syncthreads();
    if (j >= D.nr) return;
    const double rn = (D.r_first + j) / D.r_wall;
    const double xc = fmin(fmax(rn * kW - 0.5, 0.0), kW - 1.0);
    const int x0 = min(int(xc), kW - 2);
    const double fx = xc - x0, gx = 1 - fx;
    const float* cv = canvas + (long long)lo * 4 * kH * kW + x0;
    const long long nn = (long long)D.nr * D.nz;
    float* out = fields + F.out + j;
    const float rho = float(D.rho0), us = float(D.u_scale), tr = float(D.t_ref);
    auto along_r = [&](int y, int c) {
        const float* p = cv + ((long long)c * kH + y) * kW;
        return gx * p[0] + fx * p[1];
    };
    double h0[4], h1[4];
    int have = -2;  // h0, h1 are canvas rows have, have + 1
    for (int k = k0; k < k1; ++k) {
        const int y0 = row_y[k - k0];
        const double fy = row_f[k - k0], gy = row_g[k - k0];
        if (y0 != have) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                h0[c] = y0 == have + 1 ? h1[c] : along_r(y0, c);
                h1[c] = along_r(y0 + 1, c);
            }
            have = y0;
        }
        const long long i = (long long)k * D.nr;
        out[i] = rho;
#pragma unroll
        for (int c = 0; c < 3; ++c) out[(1 + c) * nn + i] = us * float(gy * h0[c] + fy * h1[c]);
        out[4 * nn + i] = tr + float(gy * h0[3] + fy * h1[3]);
    }
}

// Canvas [4][kH][kW] of one domain from its moments [4][nz][nr] (u_r, u_z,
// u_theta, T): pixel (iz, ir) sits at r = (ir + 1/2)/kW r_wall, z = z_bottom +
// (iz + 1/2)/kH height and samples the node values bilinearly, clamped to the
// grid (the inverse of k_ws_fields); velocities over the lid speed, T - T_ref.
__global__ void k_ws_to_canvas(const float* m, axlbm_ws_domain D, float* canvas) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kH * kW) return;
    const int iz = i / kW, ir = i % kW;
    const double r = (ir + 0.5) / kW * D.r_wall, z = D.z_bottom + (iz + 0.5) / kH * D.height;
    const double x = fmin(fmax(r - D.r_first, 0.0), D.nr - 1.0), y = fmin(fmax(z - D.z_first, 0.0), D.nz - 1.0);
    const int x0 = min(int(x), D.nr - 1), y0 = min(int(y), D.nz - 1);
    const int x1 = min(x0 + 1, D.nr - 1), y1 = min(y0 + 1, D.nz - 1);
    const double fx = x - x0, fy = y - y0;
    const long long n = (long long)D.nr * D.nz;
    for (int c = 0; c < 4; ++c) {
        const float* p = m + c * n;
        const double v = (1 - fy) * ((1 - fx) * p[(long long)y0 * D.nr + x0] + fx * p[(long long)y0 * D.nr + x1]) +
                         fy * ((1 - fx) * p[(long long)y1 * D.nr + x0] + fx * p[(long long)y1 * D.nr + x1]);
        canvas[(long long)c * kH * kW + i] = float(c < 3 ? v / D.u_scale : v - D.t_ref);
    }
}

unsigned blocks_for(long long n) { return (unsigned)((n + 255) / 256); }

// Launches a 3x3 convolution (ws_conv.cuh) over n images: cout in block columns
// of 32 WN channels, tiles of 16 x 16 pixels where those still give every SM
// two blocks, else of 8 x 16 (the deep levels; wide outputs of the gradients).
template <int MODE>
cudaError_t launch_conv(const axlbm_ws* w, const axl::wsconv::ConvIn& in, int n, const bf16* wt, int cout, const bf16* bias,
                        const axl::wsconv::ConvOut& to) {
    using namespace axl::wsconv;
    const int wn = cout % 96 == 0 ? 3 : (cout % 64 == 0 ? 2 : (cout % 160 == 0 ? 5 : (cout % 224 == 0 ? 7 : 1)));
    const long long px = (long long)n * in.h * in.w;
    const bool tall = wn <= 3 && px / 256 * (cout / (32 * wn)) >= 2 * w->num_sms;
    auto go = [&](auto wn_tag, auto th_tag) -> cudaError_t {
        constexpr int WN = decltype(wn_tag)::value, TH = decltype(th_tag)::value;
        auto kern = k_conv3<WN, TH, MODE>;
        const size_t smem = conv_smem<WN, TH>(in.c0 + in.c1);
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_smem<WN, TH>(224));
        if (e != cudaSuccess) return e;
        kern<<<dim3((unsigned)(px / (TH * kTW)), (unsigned)(cout / (32 * WN))), 8 * WN * TH, smem, w->stream>>>(in, wt, cout, bias, to);
        return cudaGetLastError();
    };
    using std::integral_constant;
    const integral_constant<int, 8> low;
    const integral_constant<int, 16> high;
    switch (wn) {
        case 1: return tall ? go(integral_constant<int, 1>{}, high) : go(integral_constant<int, 1>{}, low);
        case 2: return tall ? go(integral_constant<int, 2>{}, high) : go(integral_constant<int, 2>{}, low);
        case 3: return tall ? go(integral_constant<int, 3>{}, high) : go(integral_constant<int, 3>{}, low);
    }
    if constexpr (MODE == 1) {  // the inputs of the decoder's first convolutions
        if (wn == 5) return go(integral_constant<int, 5>{}, low);
        if (wn == 7) return go(integral_constant<int, 7>{}, low);
    }
    return cudaErrorInvalidValue;
}

// 3x3 convolution of layer `layer` over n canvases, with bias, ReLU and BF16
// output, and the output's 2x2 average in `pool` unless null (the forward pass).
cudaError_t conv3(axlbm_ws* w, int layer, const axl::wsconv::ConvIn& in, int n, bf16* out, bf16* pool = nullptr) {
    return launch_conv<0>(w, in, n, w->w + w->woff[layer], kNet[layer].cout, w->w + w->boff[layer],
                          {out, pool, nullptr, nullptr, 0, nullptr});
}

// Input of an encoder level's first convolution, of any level's second, and of
// a decoder level's first.
axl::wsconv::ConvIn plain_in(const bf16* x, int c, int l) { return {x, nullptr, c, 0, 0, kH >> l, kW >> l}; }
axl::wsconv::ConvIn decoder_in(const Acts& A, int l) {
    return {l + 2 < kLevels ? A.d[l + 1] : A.e[kLevels - 1], A.e[l], kCh[l + 1], kCh[l], 1, kH >> l, kW >> l};
}

// Forward pass of n canvases through the network into the activations A,
// the output canvases into `canvas` (FP32 [n][4][kH][kW]).
cudaError_t forward_acts(axlbm_ws* w, const float* feat_dev, int n, Acts& A, float* canvas) {
    cudaError_t e;
    k_ws_input<<<blocks_for((long long)n * kH * kW), 256, 0, w->stream>>>(feat_dev, n, A.x0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int l = 0; l < kLevels; ++l) {  // encoder
        e = conv3(w, enc_layer(l), l ? plain_in(A.p[l - 1], kCh[l - 1], l) : plain_in(A.x0, 8, 0), n, A.a[l]);
        if (e != cudaSuccess) return e;
        e = conv3(w, enc_layer(l) + 1, plain_in(A.a[l], kCh[l], l), n, A.e[l], l + 1 < kLevels ? A.p[l] : nullptr);
        if (e != cudaSuccess) return e;
    }
    for (int l = kLevels - 2; l >= 0; --l) {  // decoder
        if ((e = conv3(w, dec_layer(l), decoder_in(A, l), n, A.b[l])) != cudaSuccess) return e;
        if ((e = conv3(w, dec_layer(l) + 1, plain_in(A.b[l], kCh[l], l), n, A.d[l])) != cudaSuccess) return e;
    }
    k_ws_head<<<blocks_for((long long)n * kH * kW), 256, 0, w->stream>>>(A.d[0], w->w + w->woff[kHead],
                                                                          w->w + w->boff[kHead], n, canvas);
    return cudaGetLastError();
}

// Sizes (values) of the activations of n canvases, in the order acts_ptrs lists them.
std::vector<size_t> acts_sizes(int n) {
    const size_t P0 = (size_t)n * kH * kW;
    std::vector<size_t> v;
    v.push_back(P0 * 8);
    for (int l = 0; l < kLevels; ++l) {
        const size_t P = P0 >> (2 * l);
        v.push_back(P * kCh[l]);                   // a
        v.push_back(P * kCh[l]);                   // e
        if (l + 1 < kLevels) v.push_back(P / 4 * kCh[l]);  // p
    }
    for (int l = 0; l + 1 < kLevels; ++l) {
        const size_t P = P0 >> (2 * l);
        v.push_back(P * kCh[l]);                   // b
        v.push_back(P * kCh[l]);                   // d
    }
    return v;
}
std::vector<bf16**> acts_ptrs(Acts& A) {
    std::vector<bf16**> v;
    v.push_back(&A.x0);
    for (int l = 0; l < kLevels; ++l) {
        v.push_back(&A.a[l]);
        v.push_back(&A.e[l]);
        if (l + 1 < kLevels) v.push_back(&A.p[l]);
    }
    for (int l = 0; l + 1 < kLevels; ++l) {
        v.push_back(&A.b[l]);
        v.push_back(&A.d[l]);
    }
    return v;
}
bool acts_alloc(Acts& A, int n) {
    const std::vector<size_t> sz = acts_sizes(n);
    const std::vector<bf16**> ps = acts_ptrs(A);
    for (size_t i = 0; i < ps.size(); ++i) {
        if (cudaMalloc(ps[i], sz[i] * sizeof(bf16)) != cudaSuccess) {
            cudaGetLastError();
            *ps[i] = nullptr;
            return false;
        }
    }
    return true;
}
void acts_free(Acts& A) {
    for (bf16** p : acts_ptrs(A)) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
}

// ---------------------------------------------------------------- training
//
// One training step on up to kTrainMax canvases: the forward pass keeps every
// layer's output; the loss is the mean squared error over the canvases; the
// backward pass runs through the head, the ReLU masks, the convolutions (the
// weight gradient dW[o][k] = sum_p dY[p][o] A[p][k] and the input gradient,
// a convolution of dY with the mirrored taps, both kernels of ws_conv.cuh
// with FP32 accumulation), the concatenations and the pools; Adam
// then updates FP32 master weights and rewrites the BF16 weights the forward
// pass uses.  Reductions (loss, biases, head, weight gradients over pixel
// ranges) go through partials summed in a fixed order, so a step is
// deterministic.

constexpr int kTrainMax = 16;    // canvases per training step
constexpr int kPredictMax = 32;  // canvases per inference pass

// Mean-squared-error gradient 2 (out - target) / count, and per-block sums of
// (out - target)^2.
__global__ void k_ws_loss_grad(const float* out, const float* target, long long count, float* dout, double* part) {
    __shared__ double sh[256];
    double s = 0.0;
    const float scale = 2.0f / (float)count;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const float d = out[i] - target[i];
        if (dout) dout[i] = scale * d;
        s += (double)d * d;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// Sum of n doubles in a fixed order (n a multiple of 256, one block of 256).
__global__ void __launch_bounds__(256) k_ws_sum_double(const double* part, int n, double* out) {
    __shared__ double sh[256];
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) s += part[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

// out[c] = sum over blocks of part[block][c], in a fixed order: eight
// interleaved runs of blocks per value, then the runs.
__global__ void __launch_bounds__(256) k_ws_fold(const float* part, int nblocks, int cols, float* out) {
    __shared__ float sh[8][32];
    const int v = threadIdx.x & 31, run = threadIdx.x >> 5, c = blockIdx.x * 32 + v;
    float s = 0.0f;
    if (c < cols)
        for (int b = run; b < nblocks; b += 8) s += part[(long long)b * cols + c];
    sh[run][v] = s;
    __syncthreads();
    if (run == 0 && c < cols) {
        for (int g = 1; g < 8; ++g) s += sh[g][v];
        out[c] = s;
    }
}

// Head (1x1, 32 -> 4) gradients: per-block partials [132] of dW[o][c] =
// sum_p dout[o](p) x[p][c], then db[o].  A warp reads one pixel's 32 channels
// at a time, lane = channel; blocks of kHeadRows pixels of one canvas.
constexpr int kHeadRows = 512;
__global__ void __launch_bounds__(256) k_ws_head_wgrad(const float* dout, const bf16* x, float* part) {
    __shared__ float sh[8][132];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long p0 = (long long)blockIdx.x * kHeadRows, b = p0 / ((long long)kH * kW), pix0 = p0 % ((long long)kH * kW);
    const float* d = dout + b * 4 * kH * kW + pix0;
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int r = wid; r < kHeadRows; r += 8) {
        const float v = __bfloat162float(x[(p0 + r) * 32 + lane]);
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const float g = d[(long long)o * kH * kW + r];
            s[o] = fmaf(g, v, s[o]);
            sb[o] += g;
        }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        sh[wid][o * 32 + lane] = s[o];
        if (lane == 0) sh[wid][128 + o] = sb[o];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 132; t += blockDim.x) {
        float v = sh[0][t];
        for (int g = 1; g < 8; ++g) v += sh[g][t];
        part[(long long)blockIdx.x * 132 + t] = v;
    }
}

// Eight BF16 values of v where the activations are positive, else zero.
__device__ __forceinline__ uint4 ws_masked8(const float (&v)[8], const bf16* act) {
    const uint4 u = *reinterpret_cast<const uint4*>(act);
    const __nv_bfloat162* a = reinterpret_cast<const __nv_bfloat162*>(&u);
    uint4 out;
    __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        o[e].x = __float2bfloat16(__bfloat162float(a[e].x) > 0.0f ? v[2 * e] : 0.0f);
        o[e].y = __float2bfloat16(__bfloat162float(a[e].y) > 0.0f ? v[2 * e + 1] : 0.0f);
    }
    return out;
}
__device__ __forceinline__ void ws_load8(const float* p, float (&v)[8]) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// Head input gradient through the ReLU of its input x, eight channels per
// thread: dy[p][c] = (sum_o dout[o](p) W[o][c]) [x[p][c] > 0].
__global__ void __launch_bounds__(256) k_ws_head_dx(const float* dout, const bf16* wt, const bf16* x, int n, bf16* dy) {
    __shared__ float ws[4 * 32];
    if (threadIdx.x < 128) ws[threadIdx.x] = __bfloat162float(wt[threadIdx.x]);
    __syncthreads();
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)n * kH * kW * 4) return;
    const int c = int(i & 3) * 8;
    const long long p = i >> 2, b = p / ((long long)kH * kW), pix = p % ((long long)kH * kW);
    float g[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const float d = dout[(b * 4 + o) * kH * kW + pix];
#pragma unroll
        for (int e = 0; e < 8; ++e) g[e] = fmaf(d, ws[o * 32 + c + e], g[e]);
    }
    *reinterpret_cast<uint4*>(dy + p * 32 + c) = ws_masked8(g, x + p * 32 + c);
}

// Gradient of a decoder level's deep input (h x w, c channels, FP32, at the
// level's resolution) at the deeper level's: the sum of the four copies the
// upsampling made, through the ReLU of `act`; eight channels per thread.
__global__ void __launch_bounds__(256) k_ws_up_bwd(const float* g, int n, int h, int w, int c, const bf16* act, bf16* dy) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int h2 = h / 2, w2 = w / 2, nch = c / 8;
    if (i >= (long long)n * h2 * w2 * nch) return;
    const int ch = int(i % nch) * 8;
    const long long p = i / nch;
    const int x2 = int(p % w2), y2 = int((p / w2) % h2), b = int(p / ((long long)h2 * w2));
    float s[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        float v[8];
        ws_load8(g + (((long long)b * h + 2 * y2 + (d >> 1)) * w + 2 * x2 + (d & 1)) * c + ch, v);
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] += v[e];
    }
    *reinterpret_cast<uint4*>(dy + p * c + ch) = ws_masked8(s, act + p * c + ch);
}

// Gradient of an encoder level's output (h x w, c channels), which feeds the
// 2x2 average pool (gradient gp) and the skip (gradient gs), through its ReLU;
// eight channels per thread.
__global__ void __launch_bounds__(256) k_ws_pool_bwd(const float* gp, const float* gs, int n, int h, int w, int c,
                                                     const bf16* act, bf16* dy) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int nch = c / 8;
    if (i >= (long long)n * h * w * nch) return;
    const int ch = int(i % nch) * 8;
    const long long p = i / nch;
    const int xw = int(p % w), yh = int((p / w) % h), b = int(p / ((long long)h * w));
    float v[8], s[8];
    ws_load8(gp + (((long long)b * (h / 2) + yh / 2) * (w / 2) + xw / 2) * c + ch, v);
    ws_load8(gs + p * c + ch, s);
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 0.25f * v[e] + s[e];
    *reinterpret_cast<uint4*>(dy + p * c + ch) = ws_masked8(v, act + p * c + ch);
}

// Adam on FP32 master weights (bias corrections c1 = 1 - beta1^t, c2 =
// 1 - beta2^t), rewriting the BF16 weights.
__global__ void k_ws_adam(float* master, float* m, float* v, const float* grad, size_t count, float lr, float beta1,
                          float beta2, float eps, float c1, float c2, bf16* wbf) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float g = grad[i];
    const float mi = beta1 * m[i] + (1.0f - beta1) * g;
    const float vi = beta2 * v[i] + (1.0f - beta2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float x = master[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    master[i] = x;
    wbf[i] = __float2bfloat16(x);
}

__global__ void k_bf16_to_f32(const bf16* x, size_t count, float* y) {
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i < count) y[i] = __bfloat162float(x[i]);
}

}  // namespace

// Training state: FP32 master weights, their gradients and Adam moments, and
// every activation of one step's forward pass (sized for kTrainMax canvases).
struct axlbm_ws_train {
    float *master = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    int64_t step = 0;
    Acts act;            // every activation of the kept forward pass
    bf16 *dy = nullptr, *dy2 = nullptr;  // gradients of two layers' pre-activation outputs (BF16, the GEMM operands)
    bf16* wtt = nullptr; // the mirrored-tap weights of the input gradient of one layer
    float *out = nullptr, *dout = nullptr, *gx = nullptr, *part = nullptr, *wpart = nullptr, *bpart = nullptr;
    float* gs[kLevels - 1] = {};  // gradients reaching the skips
    double *dpart = nullptr, *loss = nullptr;
};

namespace {

constexpr int kLossBlocks = 1024;
// Blocks of a weight gradient, about: just under two waves of two blocks on 152 SMs.  A number of its own and not the
// device's, because the splits set the order of the sums.
constexpr int kWgradBlocks = 592;

// Splits of layer l's weight gradient over n canvases, and the pixel tiles of one.
void wgrad_splits(int l, int n, int* nsplit, int* per, int* tiles);

void train_free(axlbm_ws_train* t) {
    if (!t) return;
    acts_free(t->act);
    void* ps[] = {t->master, t->grad, t->m, t->v, t->dy, t->dy2, t->wtt, t->out, t->dout, t->gx, t->part, t->wpart,
                  t->bpart, t->gs[0], t->gs[1], t->gs[2], t->dpart, t->loss};
    for (void* p : ps)
        if (p) cudaFree(p);
    delete t;
}

int layer_level(int l) { return l < 8 ? l / 2 : 2 - (l - 8) / 2; }
int wgrad_nc(int l) { return kNet[l].cin == 8 ? 8 : 32; }

void wgrad_splits(int l, int n, int* nsplit, int* per, int* tiles) {
    const int lev = layer_level(l);
    *tiles = n * (kH >> lev) * (kW >> lev) / (axl::wsconv::kWgTH * axl::wsconv::kTW);
    const int cols = kNet[l].cin / wgrad_nc(l) * (kNet[l].cout / 32);
    int s = kWgradBlocks / cols;
    s = s < 1 ? 1 : (s > *tiles ? *tiles : s);
    *per = (*tiles + s - 1) / s;
    *nsplit = (*tiles + *per - 1) / *per;
}

// Values of the largest weight-gradient partial buffer of a training step.
size_t wpart_values(size_t* bias) {
    size_t best = 0;
    *bias = 0;
    for (int l = 0; l < kHead; ++l)
        for (int n = 1; n <= kTrainMax; ++n) {
            int nsplit, per, tiles;
            wgrad_splits(l, n, &nsplit, &per, &tiles);
            best = std::max(best, (size_t)nsplit * kNet[l].cout * 9 * kNet[l].cin);
            *bias = std::max(*bias, (size_t)nsplit * kNet[l].cout);
        }
    return best;
}

// Allocate the training state; the master weights start from the BF16 weights.
axlbm_status train_ensure(axlbm_ws* w) {
    if (w->train) return AXLBM_OK;
    axlbm_ws_train* t = new (std::nothrow) axlbm_ws_train();
    if (!t) return wfail(w, AXLBM_ENOMEM, "host allocation failed");
    const size_t count = net_values();
    const size_t P = (size_t)kTrainMax * kH * kW;  // level-0 pixels
    size_t wtt = 0;
    for (int l = 0; l < kHead; ++l) wtt = std::max(wtt, (size_t)9 * kNet[l].cin * kNet[l].cout);
    size_t bvals = 0;
    const size_t wvals = wpart_values(&bvals);
    struct Buf { void** p; size_t bytes; };
    const Buf bufs[] = {
        {(void**)&t->master, count * 4}, {(void**)&t->grad, count * 4}, {(void**)&t->m, count * 4},
        {(void**)&t->v, count * 4},      {(void**)&t->dy, P * 32 * 2},  {(void**)&t->dy2, P * 32 * 2},
        {(void**)&t->wtt, wtt * 2},      {(void**)&t->out, P * 4 * 4},  {(void**)&t->dout, P * 4 * 4},
        {(void**)&t->gx, P * 64 * 4},    {(void**)&t->part, P / kHeadRows * 132 * 4},
        {(void**)&t->wpart, wvals * 4},  {(void**)&t->bpart, bvals * 4},
        {(void**)&t->gs[0], P * kCh[0] * 4}, {(void**)&t->gs[1], P / 4 * kCh[1] * 4},
        {(void**)&t->gs[2], P / 16 * kCh[2] * 4}, {(void**)&t->dpart, kLossBlocks * 8}, {(void**)&t->loss, 8}};
    for (const Buf& b : bufs) {
        if (cudaMalloc(b.p, b.bytes) != cudaSuccess) {
            cudaGetLastError();
            *b.p = nullptr;
            train_free(t);
            return wfail(w, AXLBM_ENOMEM, "training buffers");
        }
    }
    if (!acts_alloc(t->act, kTrainMax)) {
        train_free(t);
        return wfail(w, AXLBM_ENOMEM, "training activations");
    }
    cudaError_t e = cudaMemsetAsync(t->m, 0, count * 4, w->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(t->v, 0, count * 4, w->stream);
    if (e == cudaSuccess) {
        k_bf16_to_f32<<<blocks_for((long long)count), 256, 0, w->stream>>>(w->w, count, t->master);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        train_free(t);
        return wfail(w, AXLBM_ECUDA, "training set-up");
    }
    t->step = 0;
    w->train = t;
    return AXLBM_OK;
}

// Forward pass of n <= kTrainMax canvases keeping every layer's output.
cudaError_t train_forward(axlbm_ws* w, const float* feat, int n) {
    return forward_acts(w, feat, n, w->train->act, w->train->out);
}

// Sum of squared errors of the kept prediction against target into t->loss
// (and the loss gradient into t->dout when `grad`).
cudaError_t train_loss(axlbm_ws* w, const float* target, int n, bool grad) {
    axlbm_ws_train* t = w->train;
    const long long count = (long long)n * 4 * kH * kW;
    k_ws_loss_grad<<<kLossBlocks, 256, 0, w->stream>>>(t->out, target, count, grad ? t->dout : nullptr, t->dpart);
    k_ws_sum_double<<<1, 256, 0, w->stream>>>(t->dpart, kLossBlocks, t->loss);
    return cudaGetLastError();
}

// Bias and weight gradients of 3x3 layer l (input `in`, n canvases) into
// t->grad, from the gradient dy of its pre-activation output.
cudaError_t conv_wgrad(axlbm_ws* w, int l, const axl::wsconv::ConvIn& in, int n, const bf16* dy) {
    using namespace axl::wsconv;
    axlbm_ws_train* t = w->train;
    const Layer& L = kNet[l];
    int nsplit, per, tiles;
    wgrad_splits(l, n, &nsplit, &per, &tiles);
    auto go = [&](auto nc_tag) -> cudaError_t {
        constexpr int NC = decltype(nc_tag)::value;
        auto kern = k_conv_wgrad<NC>;
        constexpr size_t smem = 2 * wgrad_stage<NC>();
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<dim3((unsigned)(L.cin / NC), (unsigned)(L.cout / 32), (unsigned)nsplit), 288, smem, w->stream>>>(
            dy, in, L.cout, tiles, per, t->wpart, t->bpart);
        return cudaGetLastError();
    };
    const cudaError_t e = wgrad_nc(l) == 8 ? go(std::integral_constant<int, 8>{}) : go(std::integral_constant<int, 32>{});
    if (e != cudaSuccess) return e;
    const long long cnt = (long long)L.cout * 9 * L.cin;
    k_fold_splits<<<(unsigned)((cnt + L.cout + kFoldVals - 1) / kFoldVals), kFoldRuns * kFoldVals, 0, w->stream>>>(
        t->wpart, t->bpart, nsplit, cnt, L.cout, t->grad + w->woff[l], t->grad + w->boff[l]);
    return cudaGetLastError();
}

// Input gradient of 3x3 layer l: dy convolved with the mirrored taps of Wt[c][tap][o].
template <int MODE>
cudaError_t conv_dgrad(axlbm_ws* w, int l, int n, const bf16* dy, const axl::wsconv::ConvOut& to) {
    using namespace axl::wsconv;
    axlbm_ws_train* t = w->train;
    const Layer& L = kNet[l];
    k_transpose_taps<<<blocks_for((long long)L.cout * 9 * L.cin), 256, 0, w->stream>>>(w->w + w->woff[l], L.cout, L.cin, t->wtt);
    return launch_conv<MODE>(w, plain_in(dy, L.cout, layer_level(l)), n, t->wtt, L.cin, nullptr, to);
}

// Backward pass of the kept forward pass from t->dout, gradients into t->grad.
// A level's second convolution passes its gradient through the ReLU of the
// first one's output within its own input gradient (dy -> dy2).
cudaError_t train_backward(axlbm_ws* w, int n) {
    axlbm_ws_train* t = w->train;
    Acts& A = t->act;
    cudaStream_t st = w->stream;
    cudaError_t e;
    const long long P0 = (long long)n * kH * kW;
    // head (packed kernel then bias: 132 contiguous values)
    const int nb = (int)(P0 / kHeadRows);
    k_ws_head_wgrad<<<nb, 256, 0, st>>>(t->dout, A.d[0], t->part);
    k_ws_fold<<<(132 + 31) / 32, 256, 0, st>>>(t->part, nb, 132, t->grad + w->woff[kHead]);
    k_ws_head_dx<<<blocks_for(P0 * 4), 256, 0, st>>>(t->dout, w->w + w->woff[kHead], A.d[0], n, t->dy);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // decoder levels 0, 1, 2; t->dy holds the gradient of the level's second convolution
    for (int l = 0; l + 1 < kLevels; ++l) {
        const int h = kH >> l, wd = kW >> l, cd = kCh[l + 1], cs = kCh[l];
        if ((e = conv_wgrad(w, dec_layer(l) + 1, plain_in(A.b[l], cs, l), n, t->dy)) != cudaSuccess) return e;
        if ((e = conv_dgrad<2>(w, dec_layer(l) + 1, n, t->dy, {t->dy2, nullptr, nullptr, nullptr, 0, A.b[l]})) != cudaSuccess)
            return e;
        if ((e = conv_wgrad(w, dec_layer(l), decoder_in(A, l), n, t->dy2)) != cudaSuccess) return e;
        if ((e = conv_dgrad<1>(w, dec_layer(l), n, t->dy2, {nullptr, nullptr, t->gx, t->gs[l], cd, nullptr})) != cudaSuccess)
            return e;
        k_ws_up_bwd<<<blocks_for((P0 >> (2 * l)) / 4 * (cd / 8)), 256, 0, st>>>(t->gx, n, h, wd, cd,
                                                                               decoder_in(A, l).x0, t->dy);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // encoder levels 3 .. 0; t->gx holds the gradient of the pooled output of the level
    for (int l = kLevels - 1; l >= 0; --l) {
        const int h = kH >> l, wd = kW >> l, c = kCh[l];
        if (l + 1 < kLevels) {  // e[l] feeds the pool and the skip
            k_ws_pool_bwd<<<blocks_for((P0 >> (2 * l)) * (c / 8)), 256, 0, st>>>(t->gx, t->gs[l], n, h, wd, c, A.e[l], t->dy);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        if ((e = conv_wgrad(w, enc_layer(l) + 1, plain_in(A.a[l], c, l), n, t->dy)) != cudaSuccess) return e;
        if ((e = conv_dgrad<2>(w, enc_layer(l) + 1, n, t->dy, {t->dy2, nullptr, nullptr, nullptr, 0, A.a[l]})) != cudaSuccess)
            return e;
        const axl::wsconv::ConvIn in = l ? plain_in(A.p[l - 1], kCh[l - 1], l) : plain_in(A.x0, 8, 0);
        if ((e = conv_wgrad(w, enc_layer(l), in, n, t->dy2)) != cudaSuccess) return e;
        if (l && (e = conv_dgrad<1>(w, enc_layer(l), n, t->dy2, {nullptr, nullptr, t->gx, t->gx, in.c0, nullptr})) != cudaSuccess)
            return e;
    }
    return cudaGetLastError();
}

}  // namespace

extern "C" {

size_t axlbm_ws_weight_count(void) { return net_values(); }

axlbm_status axlbm_ws_create(const uint16_t* weights, size_t count, void* cuda_stream, axlbm_ws** out) {
    if (!out || !weights) return wfail(nullptr, AXLBM_EINVAL, "weights and out are required");
    if (count != net_values()) return wfail(nullptr, AXLBM_EINVAL, "weight count does not match the network");
    axlbm_ws* w = new (std::nothrow) axlbm_ws();
    if (w) {
        w->w = nullptr;
        w->train = nullptr;
    }
    if (!w) return wfail(nullptr, AXLBM_ENOMEM, "host allocation failed");
    w->stream = static_cast<cudaStream_t>(cuda_stream);
    w->chunk = 8;  // (axlbm_ws_predict grows it)
    int dev = 0;
    w->num_sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&w->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (w->num_sms < 1) w->num_sms = 1;
    size_t off = 0;
    for (const Layer& l : kNet) {
        w->woff.push_back(off);
        off += (size_t)l.cout * l.cin * l.k * l.k;
        w->boff.push_back(off);
        off += l.cout;
    }
    if (cudaMalloc(&w->w, count * 2) != cudaSuccess || !acts_alloc(w->act, w->chunk)) {
        cudaGetLastError();
        axlbm_ws_destroy(w);
        return wfail(nullptr, AXLBM_ENOMEM, "device allocation failed");
    }
    cudaError_t e = cudaMemcpyAsync(w->w, weights, count * 2, cudaMemcpyHostToDevice, w->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) {
        axlbm_ws_destroy(w);
        return wfail(nullptr, AXLBM_ECUDA, "weights upload failed");
    }
    *out = w;
    return AXLBM_OK;
}

axlbm_status axlbm_ws_predict(axlbm_ws* w, const float* features, int32_t n, float* canvas) {
    if (!w || !features || !canvas || n < 0) return wfail(w, AXLBM_EINVAL, "bad arguments");
    if (n == 0) return AXLBM_OK;
    float* fd = nullptr;
    cudaError_t e = cudaMalloc(&fd, (size_t)n * kFeat * sizeof(float));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return wfail(w, AXLBM_ENOMEM, "feature buffer");
    }
    // more canvases per pass fill the SMs at the deep levels (level 3 of 8 canvases is 32 tiles); without
    // room for them the pass stays as it was
    if (n > w->chunk && w->chunk < kPredictMax) {
        Acts more;
        const int want = n < kPredictMax ? n : kPredictMax;
        e = cudaStreamSynchronize(w->stream);
        if (e == cudaSuccess && acts_alloc(more, want)) {
            acts_free(w->act);
            w->act = more;
            w->chunk = want;
        } else {
            acts_free(more);
        }
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(fd, features, (size_t)n * kFeat * sizeof(float), cudaMemcpyHostToDevice, w->stream);
    for (int b0 = 0; b0 < n && e == cudaSuccess; b0 += w->chunk) {
        const int m = n - b0 < w->chunk ? n - b0 : w->chunk;
        e = forward_acts(w, fd + (size_t)b0 * kFeat, m, w->act, canvas + (size_t)b0 * 4 * kH * kW);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    cudaFree(fd);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, std::string("forward pass: ") + cudaGetErrorString(e));
    return AXLBM_OK;
}

axlbm_status axlbm_ws_fields(axlbm_ws* w, const float* canvas, int32_t n, const axlbm_ws_domain* doms, float* fields) {
    if (!w || !canvas || !doms || !fields || n < 0) return wfail(w, AXLBM_EINVAL, "bad arguments");
    for (int d = 0; d < n; ++d)
        if (doms[d].nr < 1 || doms[d].nz < 1 || !(doms[d].r_wall > 0.0) || !(doms[d].height > 0.0))
            return wfail(w, AXLBM_EINVAL, "bad domain geometry");
    cudaError_t e = cudaSuccess;
    long long off = 0;
    for (int d0 = 0, m; d0 < n && e == cudaSuccess; d0 += m) {
        FieldDoms list;
        long long blocks = 0;
        for (m = 0; m < kFieldDoms && d0 + m < n; ++m) {
            const axlbm_ws_domain& D = doms[d0 + m];
            const long long more = ((D.nr - 1) / kFieldCols + 1ll) * ((D.nz - 1) / kFieldRows + 1);
            if (m > 0 && blocks + more > 0x7fffffffll) break;  // (a domain of more blocks than a grid holds 1.4 TB of fields)
            list.d[m] = {D, off, (int)blocks};
            off += 5 * (long long)D.nr * D.nz;
            blocks += more;
        }
        if (blocks > 0x7fffffffll) return wfail(w, AXLBM_EINVAL, "too many nodes in one domain");
        k_ws_fields<<<(unsigned)blocks, kFieldCols, 0, w->stream>>>(canvas + (size_t)d0 * 4 * kH * kW, list, m, fields);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, "resampling");
    return AXLBM_OK;
}

axlbm_status axlbm_ws_train_step(axlbm_ws* w, const float* features, const float* target, int32_t n, float lr,
                                 float beta1, float beta2, float eps, double* loss) {
    if (!w || !features || !target || n < 1 || n > kTrainMax || !(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
        !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f))
        return wfail(w, AXLBM_EINVAL, "bad arguments (n must be 1..16)");
    axlbm_status st = train_ensure(w);
    if (st != AXLBM_OK) return st;
    axlbm_ws_train* t = w->train;
    cudaError_t e = train_forward(w, features, n);
    if (e == cudaSuccess) e = train_loss(w, target, n, true);
    if (e == cudaSuccess) e = train_backward(w, n);
    if (e == cudaSuccess) {
        t->step += 1;
        const double c1 = 1.0 - pow((double)beta1, (double)t->step), c2 = 1.0 - pow((double)beta2, (double)t->step);
        const size_t count = net_values();
        k_ws_adam<<<blocks_for((long long)count), 256, 0, w->stream>>>(t->master, t->m, t->v, t->grad, count, lr, beta1,
                                                                       beta2, eps, (float)c1, (float)c2, w->w);
        e = cudaGetLastError();
    }
    double sse = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, t->loss, sizeof sse, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, std::string("training step: ") + cudaGetErrorString(e));
    if (loss) *loss = sse / ((double)n * 4 * kH * kW);
    return AXLBM_OK;
}

axlbm_status axlbm_ws_loss(axlbm_ws* w, const float* features, const float* target, int32_t n, double* loss) {
    if (!w || !features || !target || !loss || n < 1) return wfail(w, AXLBM_EINVAL, "bad arguments");
    axlbm_status st = train_ensure(w);
    if (st != AXLBM_OK) return st;
    double total = 0.0;
    for (int b0 = 0; b0 < n; b0 += kTrainMax) {
        const int m = n - b0 < kTrainMax ? n - b0 : kTrainMax;
        cudaError_t e = train_forward(w, features + (size_t)b0 * kFeat, m);
        if (e == cudaSuccess) e = train_loss(w, target + (size_t)b0 * 4 * kH * kW, m, false);
        double sse = 0.0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, w->train->loss, sizeof sse, cudaMemcpyDeviceToHost, w->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
        if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, std::string("loss: ") + cudaGetErrorString(e));
        total += sse;
    }
    *loss = total / ((double)n * 4 * kH * kW);
    return AXLBM_OK;
}

axlbm_status axlbm_ws_last_gradient(axlbm_ws* w, float* grad) {
    if (!w || !grad) return wfail(w, AXLBM_EINVAL, "bad arguments");
    if (!w->train) return wfail(w, AXLBM_EINVAL, "no training step has run");
    cudaError_t e = cudaMemcpyAsync(grad, w->train->grad, net_values() * 4, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, "gradient download");
    return AXLBM_OK;
}

axlbm_status axlbm_ws_get_weights(axlbm_ws* w, uint16_t* weights) {
    if (!w || !weights) return wfail(w, AXLBM_EINVAL, "bad arguments");
    cudaError_t e = cudaMemcpyAsync(weights, w->w, net_values() * 2, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, "weights download");
    return AXLBM_OK;
}

axlbm_status axlbm_ws_to_canvas(axlbm_ws* w, const float* moments, int32_t n, const axlbm_ws_domain* doms,
                                float* canvas) {
    if (!w || !moments || !doms || !canvas || n < 0) return wfail(w, AXLBM_EINVAL, "bad arguments");
    size_t off = 0;
    for (int d = 0; d < n; ++d) {
        const axlbm_ws_domain& D = doms[d];
        if (D.nr < 1 || D.nz < 1 || !(D.r_wall > 0.0) || !(D.height > 0.0) || !(D.u_scale != 0.0))
            return wfail(w, AXLBM_EINVAL, "bad domain geometry");
        k_ws_to_canvas<<<blocks_for(kH * kW), 256, 0, w->stream>>>(moments + off, D, canvas + (size_t)d * 4 * kH * kW);
        off += 4 * (size_t)D.nr * D.nz;
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) return wfail(w, AXLBM_ECUDA, "canvas resampling");
    return AXLBM_OK;
}

axlbm_status axlbm_ws_destroy(axlbm_ws* w) {
    if (!w) return AXLBM_EINVAL;
    train_free(w->train);
    acts_free(w->act);
    if (w->w) cudaFree(w->w);
    delete w;
    return AXLBM_OK;
}

const char* axlbm_ws_last_error(const axlbm_ws* w) { return w ? w->err.c_str() : g_ws_error.c_str(); }

}  // extern "C"

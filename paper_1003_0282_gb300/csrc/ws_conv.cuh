// ws_conv.cuh -- BF16 3x3 convolutions of the warm-start network on the
// tensor cores (mma.sync m16n8k16, FP32 accumulation).
//
// Activations are NHWC BF16; a layer's weights are packed [cout][tap][cin]
// with tap = 3 ky + kx (the layout of the weight blob in include/axlbm.h), so
// the K index of the GEMM is k = tap * cin + c.  No im2col matrix is formed:
// a block keeps a tile of pixels with its border in shared memory and takes
// the operands of every tap from it at a shifted address, by ldmatrix.
//
//   forward:       y[p][o]  = sum_k  A[p][k] W[o][k],  A[p][(tap, c)] = x[p + d(tap)][c]
//   input grad:    gx[q][c] = sum_k' B[q][k'] Wt[c][k'], B[q][(tap, o)] = dy[q - d(tap)][o]
//                  (the same kernel with the taps mirrored and Wt[c][tap][o] = W[o][tap][c])
//   weight grad:   dW[o][k] = sum_p dy[p][o] A[p][k], split over runs of tiles
//                  into partials that a fixed-order fold adds up
// with d(tap) = (ky - 1, kx - 1).  Channel counts are multiples of 8 so that
// a 16-byte chunk of k never straddles two taps.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace axl {
namespace wsconv {

using bf16 = __nv_bfloat16;

constexpr int kBK = 32;   // k per pipeline stage
constexpr int kLd = kBK + 8;  // shared-memory row stride (bf16): 80 bytes, conflict-free ldmatrix

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte global -> shared copy; src_bytes = 0 fills the 16 bytes with zeros.
__device__ __forceinline__ void cp16(void* dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(dst)), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x4_at(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}

__device__ __forceinline__ void ldsm_x4_t_at(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a));
}

// D = A (16x16, row) B (16x8, col) + D, BF16 in, FP32 accumulate.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The input of a convolution: c0 channels of x0 (stored at half the
// resolution and upsampled by nearest when up0), then c1 channels of x1
// (c1 = 0: none).  NHWC, n images of h x w pixels.
struct ConvIn {
    const bf16* x0;
    const bf16* x1;
    int c0, c1, up0, h, w;
};

// Where a convolution's result goes.  MODE 0 (forward): y, BF16 [p][cout], and
// its 2x2 average in `pool` if given.  MODE 1 (input gradient): FP32, the
// first c0 channels to g0 [p][c0], the rest to g1 [p][cout - c0].  MODE 2
// (input gradient through the ReLU that made the input): y = acc where act > 0.
struct ConvOut {
    bf16* y;
    bf16* pool;
    float* g0;
    float* g1;
    int c0;
    const bf16* act;
};

// Tiles of the 3x3 convolutions: TH rows x 16 columns of pixels with all input
// channels and a one-pixel border in shared memory, 16-byte chunks of a pixel
// at an odd stride (in chunks), so that ldmatrix rows of consecutive pixels
// fall into different banks.
constexpr int kTW = 16;
__host__ __device__ constexpr int conv_stride(int cin) { return (cin / 8) | 1; }
constexpr int kWStages = 4;  // weight stages of kBK values of k in flight
template <int WN, int TH>
__host__ __device__ constexpr size_t conv_smem(int cin) {
    const size_t tile = (size_t)(TH + 2) * (kTW + 2) * conv_stride(cin) * 16 + 16 + (size_t)kWStages * 32 * WN * kLd * 2;
    const size_t out = (size_t)TH / 4 * WN * 64 * (32 * 2 + 16);  // the epilogue's copy of the results
    return tile > out ? tile : out;
}

// v where the eight BF16 activations a are positive, else zero.
__device__ __forceinline__ uint4 relu_mask(uint4 v, uint4 a) {
    const __nv_bfloat162* ap = reinterpret_cast<const __nv_bfloat162*>(&a);
    __nv_bfloat162* vp = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (!(__bfloat162float(ap[i].x) > 0.0f)) vp[i].x = __float2bfloat16(0.0f);
        if (!(__bfloat162float(ap[i].y) > 0.0f)) vp[i].y = __float2bfloat16(0.0f);
    }
    return v;
}

// 3x3 convolution, padding 1: out[p][o], o in [32 WN blockIdx.y, +32 WN), for
// one TH x 16 tile of pixels per block.  wt: [cout][9 cin] (row o holds k =
// tap cin + c); modes other than 0 mirror the taps.
//
// The tile's input is read once (an implicit im2col gather reads it nine
// times); the A operands of every tap are the same shared memory at a shifted
// address.  A warp owns four rows of 16 pixels x 32 channels: 6 ldmatrix per
// 16 mma, below the shared-memory rate at the full mma.sync rate (605 TFLOP/s
// from registers, measured on GB300).  Weights stream through kWStages
// cp.async stages.  k ascends in steps of 16 into one
// accumulator per output, so sums round as in any other tiling.  mma.sync and
// not tcgen05.mma: with the tile as unswizzled core matrices, a tap being a
// descriptor shifted by 16-byte places, an instruction of 128 pixels took 200
// to 260 cycles for 32 to 64 channels (200 draws predicted and resampled 9.68
// against 8.96 ms on GB300, a training step of 16 canvases 2.36 against 2.30).
template <int WN, int TH, int MODE>
__global__ void __launch_bounds__(8 * WN * TH, 512 / (8 * WN * TH) > 0 ? 512 / (8 * WN * TH) : 1)
k_conv3(const ConvIn in, const bf16* __restrict__ wt, int cout, const bf16* __restrict__ bias, const ConvOut to) {
    constexpr bool FLIP = MODE != 0;
    constexpr int BN = 32 * WN, T = 8 * WN * TH;
    extern __shared__ __align__(128) unsigned char conv_sm[];
    const int cin = in.c0 + in.c1, nch = cin / 8, stride = conv_stride(cin) * 16;  // bytes of a pixel
    const int K = 9 * cin, nk = (K + kBK - 1) / kBK;
    const int h = in.h, w = in.w, tiles_x = w / kTW, tiles_y = h / TH;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, wm = wid % (TH / 4), wn = wid / (TH / 4);
    const int img = blockIdx.x / (tiles_x * tiles_y), trem = blockIdx.x - img * tiles_x * tiles_y;
    const int y0 = (trem / tiles_x) * TH, x0 = (trem % tiles_x) * kTW, n0 = blockIdx.y * BN;
    unsigned char* zero = conv_sm + (TH + 2) * (kTW + 2) * stride;  // 16 bytes of zeros
    bf16* Bs = reinterpret_cast<bf16*>(zero + 16);                 // [kWStages][BN][kLd]
    auto load_weights = [&](int kt) {
        if (kt < nk) {
            bf16* dst = Bs + (kt % kWStages) * BN * kLd;
            for (int i = tid; i < BN * (kBK / 8); i += T) {
                const int row = i >> 2, k = kt * kBK + (i & 3) * 8;
                const bool ok = k < K;
                cp16(dst + row * kLd + (i & 3) * 8, ok ? wt + (long long)(n0 + row) * K + k : wt, ok ? 16 : 0);
            }
        }
        cp_commit();
    };
    if (tid < 4) reinterpret_cast<int*>(zero)[tid] = 0;
    for (int i = tid; i < (TH + 2) * (kTW + 2) * nch; i += T) {
        const int px = i / nch, ch = i - px * nch, ly = px / (kTW + 2), lx = px - ly * (kTW + 2);
        const int y = y0 + ly - 1, x = x0 + lx - 1, c = ch * 8;
        const bool ok = y >= 0 && y < h && x >= 0 && x < w;
        const bf16* src = in.x0;
        if (ok) {
            if (c < in.c0)
                src = in.up0 ? in.x0 + (((long long)img * (h / 2) + y / 2) * (w / 2) + x / 2) * in.c0 + c
                             : in.x0 + (((long long)img * h + y) * w + x) * in.c0 + c;
            else src = in.x1 + (((long long)img * h + y) * w + x) * in.c1 + (c - in.c0);
        }
        cp16(conv_sm + px * stride + ch * 16, src, ok ? 16 : 0);
    }
    load_weights(0);  // (one group with the tile)
#pragma unroll
    for (int s = 1; s < kWStages - 1; ++s) load_weights(s);
    float acc[4][4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.0f;
    // this lane's row of the A fragments (pixel lane & 15 of the warp's rows, upper half of k for lanes 16..31)
    const uint32_t a_lane = smem_addr(conv_sm) + (uint32_t)((4 * wm * (kTW + 2) + (lane & 15)) * stride + (lane >> 4) * 16);
    const uint32_t a_row = (kTW + 2) * stride;
    auto tap_at = [&](int tap) {
        const int ky = tap / 3, kx = tap - 3 * ky;
        return (uint32_t)(((FLIP ? 2 - ky : ky) * (kTW + 2) + (FLIP ? 2 - kx : kx)) * stride);
    };
    const int bi = lane >> 3, br = lane & 7;
    const int b_lane = (wn * 32 + (bi >> 1) * 8 + br) * kLd + (bi & 1) * 8;
    int tap = 0, c = 0;
    for (int kt = 0; kt < nk; ++kt) {
        cp_wait<kWStages - 2>();
        __syncthreads();
        load_weights(kt + kWStages - 1);  // into the stage everybody has left
        const bf16* B = Bs + (kt % kWStages) * BN * kLd;
#pragma unroll
        for (int kk = 0; kk < kBK; kk += 16) {
            if (kt * kBK + kk >= K) break;
            uint32_t at[4];
            if (cin >= 16) {
                const uint32_t a = a_lane + tap_at(tap) + c * 2;
#pragma unroll
                for (int m = 0; m < 4; ++m) at[m] = a + m * a_row;
                c += 16;
                if (c == cin) c = 0, ++tap;
            } else {  // eight channels: two taps in 16 values of k, zeros past the last
                const int t = (kt * kBK + kk) / 8 + (lane >> 4);
                const uint32_t a = a_lane - (lane >> 4) * 16 + tap_at(t < 9 ? t : 0);
#pragma unroll
                for (int m = 0; m < 4; ++m) at[m] = t < 9 ? a + m * a_row : smem_addr(zero);
            }
            uint32_t af[4][4], bf[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j) ldsm_x4(bf[j], B + b_lane + j * 16 * kLd + kk);
#pragma unroll
            for (int m = 0; m < 4; ++m) ldsm_x4_at(af[m], at[m]);
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    mma16816(acc[m][2 * j], af[m], bf[j][0], bf[j][1]);
                    mma16816(acc[m][2 * j + 1], af[m], bf[j][2], bf[j][3]);
                }
        }
    }
    const int gid = lane >> 2, tig = lane & 3;
    const long long p0 = ((long long)img * h + y0 + 4 * wm) * w + x0;  // pixel of the warp's first row
    const int o0 = n0 + wn * 32;
    if (MODE == 1) {
        const bool first = o0 < to.c0;  // (both parts are multiples of 32 channels)
        float* base = first ? to.g0 + o0 : to.g1 + (o0 - to.c0);
        const int ld = first ? to.c0 : cout - to.c0;
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float* dst = base + (p0 + (long long)m * w + gid + 8 * half) * ld + tig * 2;
#pragma unroll
                for (int ni = 0; ni < 4; ++ni)
                    *reinterpret_cast<float2*>(dst + ni * 8) = make_float2(acc[m][ni][2 * half], acc[m][ni][2 * half + 1]);
            }
        return;
    }
    // bias and ReLU (or the ReLU's mask) and BF16 through shared memory: 16-byte stores of whole pixels' channels
    cp_wait<0>();
    __syncthreads();
    unsigned char* mine = conv_sm + wid * 64 * 80;
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) {
        const int o = o0 + ni * 8 + tig * 2;
        const float b0 = MODE == 0 ? __bfloat162float(bias[o]) : 0.0f, b1 = MODE == 0 ? __bfloat162float(bias[o + 1]) : 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const float v0 = acc[m][ni][2 * half] + b0, v1 = acc[m][ni][2 * half + 1] + b1;
                __nv_bfloat162 r;
                r.x = __float2bfloat16(MODE == 2 || v0 > 0.0f ? v0 : 0.0f);
                r.y = __float2bfloat16(MODE == 2 || v1 > 0.0f ? v1 : 0.0f);
                *reinterpret_cast<__nv_bfloat162*>(mine + (m * 16 + gid + 8 * half) * 80 + (ni * 8 + tig * 2) * 2) = r;
            }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = i * 32 + lane, px = e >> 2, ch = e & 3;
        const long long at = (p0 + (long long)(px >> 4) * w + (px & 15)) * cout + o0 + ch * 8;
        uint4 v = *reinterpret_cast<const uint4*>(mine + px * 80 + ch * 16);
        if (MODE == 2) v = relu_mask(v, *reinterpret_cast<const uint4*>(to.act + at));
        *reinterpret_cast<uint4*>(to.y + at) = v;
    }
    if (MODE == 0 && to.pool) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {  // 2 x 8 pooled pixels x 4 chunks
            const int e = i * 32 + lane, px = e >> 2, ch = e & 3, py = px >> 3, pxx = px & 7;
            const unsigned char* q = mine + ((2 * py) * 16 + 2 * pxx) * 80 + ch * 16;
            __nv_bfloat162 r[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const float2 a = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(q)[v]);
                const float2 b = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(q + 80)[v]);
                const float2 d = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(q + 16 * 80)[v]);
                const float2 e2 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(q + 17 * 80)[v]);
                r[v].x = __float2bfloat16(0.25f * (a.x + b.x + d.x + e2.x));
                r[v].y = __float2bfloat16(0.25f * (a.y + b.y + d.y + e2.y));
            }
            const long long pp = ((long long)img * (h / 2) + (y0 + 4 * wm) / 2 + py) * (w / 2) + x0 / 2 + pxx;
            *reinterpret_cast<uint4*>(to.pool + pp * cout + o0 + ch * 8) = *reinterpret_cast<const uint4*>(r);
        }
    }
}

// Weight gradient of a 3x3 convolution, split over runs of pixel tiles:
// part[s][o][k] = sum over the pixels of the tiles of split s (`per` tiles of 8
// x 16 each) of dy[p][o] A[p][k], and the bias gradient's partials
// bpart[s][o] = sum dy[p][o].  Block: 32 output channels (blockIdx.y) x NC
// input channels (blockIdx.x) x one split (blockIdx.z); warp t takes tap t,
// 32 x NC products, the pixels of a tile row being the 16 values of its k.
// The tile of dy and the bordered tile of x are staged pixel-major (two
// stages of cp.async) and transposed by ldmatrix.trans: x is read 1.4 times
// instead of nine times, and a warp issues four ldmatrix per eight mma.
constexpr int kWgTH = 8;
template <int NC>
__host__ __device__ constexpr int wgrad_stride() { return (NC / 8) | 1; }  // 16-byte chunks of a pixel of x
constexpr int kWgLdD = 32 + 8;
template <int NC>
__host__ __device__ constexpr size_t wgrad_stage() {
    return (size_t)kWgTH * kTW * kWgLdD * 2 + (size_t)(kWgTH + 2) * (kTW + 2) * wgrad_stride<NC>() * 16;
}
template <int NC>
__global__ void __launch_bounds__(288, 2) k_conv_wgrad(const bf16* __restrict__ dy, const ConvIn in, int cout, int tiles,
                                                       int per, float* __restrict__ part, float* __restrict__ bpart) {
    constexpr int T = 288, ST = wgrad_stride<NC>() * 16, NJ = NC / 8;
    extern __shared__ __align__(128) unsigned char conv_sm[];
    const int tid = threadIdx.x, lane = tid & 31, tap = tid >> 5;
    const int cin = in.c0 + in.c1, K = 9 * cin, h = in.h, w = in.w, tiles_x = w / kTW, tiles_y = h / kWgTH;
    const int c0 = blockIdx.x * NC, o0 = blockIdx.y * 32, t0 = blockIdx.z * per, t1 = min(t0 + per, tiles);
    const bool half = in.up0 && c0 < in.c0;  // (a block's channels lie in one of the two sources)
    const bf16* src = c0 < in.c0 ? in.x0 + c0 : in.x1 + (c0 - in.c0);
    const int sc = c0 < in.c0 ? in.c0 : in.c1;
    auto load = [&](int t) {
        if (t < t1) {
            unsigned char* sm = conv_sm + ((t - t0) & 1) * wgrad_stage<NC>();
            const int img = t / (tiles_x * tiles_y), rem = t - img * tiles_x * tiles_y;
            const int y0 = (rem / tiles_x) * kWgTH, x0 = (rem % tiles_x) * kTW;
            for (int i = tid; i < kWgTH * kTW * 4; i += T) {
                const int px = i >> 2, ch = i & 3;
                const long long p = ((long long)img * h + y0 + (px >> 4)) * w + x0 + (px & 15);
                cp16(sm + px * (kWgLdD * 2) + ch * 16, dy + p * cout + o0 + ch * 8, 16);
            }
            sm += kWgTH * kTW * kWgLdD * 2;
            for (int i = tid; i < (kWgTH + 2) * (kTW + 2) * NJ; i += T) {
                const int px = i / NJ, ch = i - px * NJ, ly = px / (kTW + 2), y = y0 + ly - 1, x = x0 + px - ly * (kTW + 2) - 1;
                const bool ok = y >= 0 && y < h && x >= 0 && x < w;
                const bf16* at = half ? src + (((long long)img * (h / 2) + y / 2) * (w / 2) + x / 2) * sc
                                      : src + (((long long)img * h + y) * w + x) * sc;
                cp16(sm + px * ST + ch * 16, ok ? at + ch * 8 : src, ok ? 16 : 0);
            }
        }
        cp_commit();
    };
    float acc[2][NJ][4], bsum = 0.0f;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < NJ; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.0f;
    const int i = lane >> 3, r = lane & 7, ky = tap / 3, kx = tap - 3 * ky;
    load(t0);
    for (int t = t0; t < t1; ++t) {
        load(t + 1);
        cp_wait<1>();
        __syncthreads();
        unsigned char* sm = conv_sm + ((t - t0) & 1) * wgrad_stage<NC>();
        const bf16* Ds = reinterpret_cast<const bf16*>(sm);
        const uint32_t xs = smem_addr(sm + kWgTH * kTW * kWgLdD * 2) + (uint32_t)((ky * (kTW + 2) + kx) * ST);
#pragma unroll
        for (int row = 0; row < kWgTH; ++row) {
            uint32_t af[2][4], bf[NJ / 2 > 0 ? NJ / 2 : 1][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
                ldsm_x4_t(af[m], Ds + (row * kTW + (i >> 1) * 8 + r) * kWgLdD + m * 16 + (i & 1) * 8);
            // pixels (i & 1) 8 + r, channels (i >> 1) 8 .. + 8 of each pair of channel groups
            const uint32_t xr = xs + (uint32_t)((row * (kTW + 2) + (i & 1) * 8 + r) * ST);
            if (NJ > 1) {
#pragma unroll
                for (int j = 0; j < NJ / 2; ++j) ldsm_x4_t_at(bf[j], xr + (uint32_t)(j * 32 + (i >> 1) * 16));
            } else {
                ldsm_x4_t_at(bf[0], xr);  // (its upper half repeats the lower)
            }
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    mma16816(acc[m][j], af[m], bf[j / 2][(j & 1) * 2], bf[j / 2][(j & 1) * 2 + 1]);
        }
        if (blockIdx.x == 0 && tid < 256) {  // 16 pixels of one channel
#pragma unroll
            for (int x = 0; x < kTW; ++x) bsum += __bfloat162float(Ds[((tid >> 5) * kTW + x) * kWgLdD + (tid & 31)]);
        }
        __syncthreads();
    }
    const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            float* dst = part + ((long long)blockIdx.z * cout + o0 + m * 16 + gid + 8 * hf) * K + tap * cin + c0 + tig * 2;
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                *reinterpret_cast<float2*>(dst + j * 8) = make_float2(acc[m][j][2 * hf], acc[m][j][2 * hf + 1]);
        }
    if (blockIdx.x == 0) {
        float* red = reinterpret_cast<float*>(conv_sm);
        if (tid < 256) red[tid] = bsum;
        __syncthreads();
        if (tid < 32) {
            float v = 0.0f;
            for (int g = 0; g < 8; ++g) v += red[g * 32 + tid];
            bpart[(long long)blockIdx.z * cout + o0 + tid] = v;
        }
    }
}

// grad[i] = sum over s of part[s][i] and gbias[o] = sum over s of bpart[s][o],
// in a fixed order: eight interleaved runs of s per value, then the runs.
constexpr int kFoldRuns = 8, kFoldVals = 32;
__global__ void __launch_bounds__(kFoldRuns * kFoldVals)
k_fold_splits(const float* __restrict__ part, const float* __restrict__ bpart, int nsplit, long long count, int cout,
              float* __restrict__ grad, float* __restrict__ gbias) {
    __shared__ float sh[kFoldRuns][kFoldVals];
    const int v = threadIdx.x % kFoldVals, run = threadIdx.x / kFoldVals;
    const long long i = blockIdx.x * (long long)kFoldVals + v;
    const bool bias = i >= count;
    const long long n = bias ? cout : count, at = bias ? i - count : i;
    const float* src = bias ? bpart : part;
    float acc = 0.0f;
    if (at < n)
        for (int s = run; s < nsplit; s += kFoldRuns) acc += src[s * n + at];
    sh[run][v] = acc;
    __syncthreads();
    if (run == 0 && at < n) {
        for (int g = 1; g < kFoldRuns; ++g) acc += sh[g][v];
        (bias ? gbias : grad)[at] = acc;
    }
}

// Wt[c][tap][o] = W[o][tap][c]: the weights of the input-gradient convolution.
__global__ void k_transpose_taps(const bf16* __restrict__ wt, int cout, int cin, bf16* __restrict__ wtt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= cout * 9 * cin) return;
    const int o = i / (9 * cin), rem = i - o * 9 * cin, tap = rem / cin, c = rem - tap * cin;
    wtt[((long long)c * 9 + tap) * cout + o] = wt[i];
}

}  // namespace wsconv
}  // namespace axl

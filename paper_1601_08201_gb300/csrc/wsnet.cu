// wsnet.cu -- the learned warm start: a small encoder-decoder (include/wsnet.h)
// trained and run with hand-written kernels. BF16 weights, FP32 activations,
// FP32 accumulation; FP32 master weights updated by Adam.
//
// Convolutions are 3x3, stride 1, zero padding, as implicit GEMMs. Three forms:
//   k_conv       inference, on the tensor cores with the precision of FP32
//                arithmetic: the weights are BF16 already, an FP32 activation is
//                the exact sum of three BF16 terms, every product is exact, and
//                only one 16-wide step of one kernel offset is summed inside the
//                matrix unit, from zero; the steps are added up in FP32
//                registers, rounded to nearest (chained in the unit, whose adds
//                truncate, 144 steps are off by 2e-6 to 6e-6; this way by 2e-7,
//                a serial FP32 multiply-add chain by 3e-7 to 6e-7)
//   k_conv_fma   the training step's forward pass and data gradients, FP32
//                multiply-adds in one fixed order per output: a training step
//                has ReLU masks and sign-like Adam updates behind it, so a
//                rounding that differs anywhere in the forward pass is a
//                different step (tried on the tensor cores: errors as above,
//                0.6 ms instead of 1.2 for the protocol's step of 8 samples, but
//                one seed in three steps to another side of some ReLU)
//   k_conv_wgrad the training step's weight gradients, the same way
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <random>
#include <string>
#include <vector>

#include "../../include/sgtv.h"
#include "../../include/wsnet.h"
#include "sgtv_rules.h"

namespace {

constexpr int kT = 256;

int blocks_for(int64_t n)
{
    int64_t b = (n + kT - 1) / kT;
    if (b > 8192) b = 8192;
    return int(b < 1 ? 1 : b);
}

// d = a * b + c on the tensor cores: a 16 x 16 (rows: output channels, columns:
// input channels), b 16 x 8 (columns: pixels), BF16 operands, FP32 sums.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint4 &a, const uint2 &b, const float (&c)[4])
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %11, %12, %13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// (x, y) = t[0] + t[1] + t[2] exactly, each word a pair of BF16 numbers (x below):
// the leading 8 bits rounded to nearest, those of the rest, and the rest of
// that. What would round to infinity is cut instead; an infinity or NaN is all
// in t[0].
__device__ __forceinline__ void split_pair(float x, float y, uint32_t (&t)[3])
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    t[0] = *reinterpret_cast<const uint32_t *>(&h);
    float rx = x - __uint_as_float(t[0] << 16), ry = y - __uint_as_float(t[0] & 0xFFFF0000u);
    if ((t[0] & 0x7F80u) == 0x7F80u || (t[0] & 0x7F800000u) == 0x7F800000u) {
        const bool fx = isfinite(x), fy = isfinite(y);
        const uint32_t cx = fx ? __float_as_uint(x) >> 16 : t[0] & 0xFFFFu;
        const uint32_t cy = fy ? __float_as_uint(y) & 0xFFFF0000u : t[0] & 0xFFFF0000u;
        t[0] = cx | cy;
        rx = fx ? x - __uint_as_float(cx << 16) : 0.f;
        ry = fy ? y - __uint_as_float(cy) : 0.f;
    }
    const __nv_bfloat162 m = __floats2bfloat162_rn(rx, ry);
    t[1] = *reinterpret_cast<const uint32_t *>(&m);
    const __nv_bfloat162 l =
        __floats2bfloat162_rn(rx - __uint_as_float(t[1] << 16), ry - __uint_as_float(t[1] & 0xFFFF0000u));
    t[2] = *reinterpret_cast<const uint32_t *>(&l);
}

// Forward convolution. A block makes 16 MT output channels of a tile of RG NT / 2 rows x
// 16 columns of one sample: warp (m, g) 16 channels of NT / 2 rows (MT x RG
// warps, NT runs of 8 pixels each). Per step of 16 input channels the block
// stages the tile with its halo as three BF16 terms, [pixel][channel], while
// the next step's values are on their way, and each warp goes through the nine
// offsets. Weights come from global memory (L2) in fragment order, one 16-byte
// load a lane and offset, one row of offsets ahead. The activations of a
// pixel's 16 channels are 32 bytes in the order that a lane's two words (pairs
// k and k + 8) lie side by side; stores and fragment loads are both contiguous
// over the lanes. The nine layers of one 64 x 64 sample: 114 us of kernels, with
// the direct convolutions on the FP32 pipes about 600.
template <int MT, int RG, int NT, bool RELU>
__global__ void __launch_bounds__(32 * MT * RG, 16 / (MT * RG))  // 128 registers
k_conv(const float *__restrict__ x, const uint4 *__restrict__ wf, const float *__restrict__ b,
       float *__restrict__ y, int Ci, int Co, int H, int W)
{
    constexpr int kThreads = 32 * MT * RG, kRows = RG * NT / 2, kPW = 18, kPix = (kRows + 2) * kPW;
    constexpr int kItems = (4 * kPix + kThreads - 1) / kThreads;  // 4 channels of a pixel each
    __shared__ uint2 xs[3][kItems * kThreads];
    const int tiles_w = (W + 15) / 16;
    const int h0 = int(blockIdx.x) / tiles_w * kRows, w0 = int(blockIdx.x) % tiles_w * 16;
    const int n = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mt = warp % MT, rg = warp / MT;
    const int nci = (Ci + 15) / 16, co16 = int(blockIdx.y) * MT + mt;
    const bool live = co16 * 16 < Co;
    const int HW = H * W;
    const float *xn = x + size_t(n) * Ci * HW;
    // this thread's staging items: channels 2 cp, + 1, + 8, + 9 of the pixels (k kThreads + thread) / 4
    const int cp = threadIdx.x & 3;
    int off[kItems];  // the pixel's offset, -1 outside the image (or past the tile)
#pragma unroll
    for (int k = 0; k < kItems; k++) {
        const int p = (k * kThreads + int(threadIdx.x)) >> 2;
        const int gy = h0 + p / kPW - 1, gx = w0 + p % kPW - 1;
        off[k] = (p < kPix && gy >= 0 && gy < H && gx >= 0 && gx < W) ? gy * W + gx : -1;
    }
    float v[kItems][4];
    auto fetch = [&](int c0) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int c = c0 + 2 * cp + (q & 1) + 8 * (q >> 1);
            const float *xc = xn + size_t(c) * HW;
#pragma unroll
            for (int k = 0; k < kItems; k++) v[k][q] = (off[k] >= 0 && c < Ci) ? __ldg(xc + off[k]) : 0.f;
        }
    };
    fetch(0);
    float acc[NT][4];
#pragma unroll
    for (int t = 0; t < NT; t++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[t][q] = 0.f;
    const uint4 *wp = wf + (size_t(live ? co16 : 0) * nci * 9) * 32 + lane;
    uint4 a[3], an[3];
#pragma unroll
    for (int k = 0; k < 3; k++) an[k] = __ldg(wp + k * 32);
    const int il = (rg * (NT / 2) * kPW + (lane >> 2)) * 4 + (lane & 3);  // this lane's words of its first pixel
#pragma unroll 1
    for (int c = 0; c < nci; c++) {
        if (c > 0) __syncthreads();
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            uint32_t t0[3], t1[3];
            split_pair(v[k][0], v[k][1], t0);
            split_pair(v[k][2], v[k][3], t1);
#pragma unroll
            for (int m = 0; m < 3; m++) xs[m][k * kThreads + threadIdx.x] = make_uint2(t0[m], t1[m]);
        }
        __syncthreads();
        if (c + 1 < nci) fetch((c + 1) * 16);
#pragma unroll 1
        for (int kh = 0; kh < 3; kh++) {
#pragma unroll
            for (int k = 0; k < 3; k++) a[k] = an[k];
            wp += 3 * 32;
            if (c * 3 + kh + 1 < nci * 3) {
#pragma unroll
                for (int k = 0; k < 3; k++) an[k] = __ldg(wp + k * 32);
            }
            const int ik = il + kh * kPW * 4;
#pragma unroll
            for (int kw = 0; kw < 3; kw++)
#pragma unroll
                for (int t = 0; t < NT; t++) {
                    const int i = ik + ((t / 2) * kPW + (t % 2) * 8 + kw) * 4;
                    // the small terms in one sum, the large one (16-bit products: hardly a bit is cut
                    // inside the unit) in another
                    float d[4] = {0.f, 0.f, 0.f, 0.f}, z[4] = {0.f, 0.f, 0.f, 0.f};
                    mma16816(d, a[kw], xs[2][i], d);
                    mma16816(d, a[kw], xs[1][i], d);
                    mma16816(z, a[kw], xs[0][i], z);
#pragma unroll
                    for (int q = 0; q < 4; q++) acc[t][q] = (acc[t][q] + d[q]) + z[q];
                }
        }
    }
    if (!live) return;
    const bool even = (W & 1) == 0;  // else (the quarter-size images of some widths) a pair is not 8-byte aligned
#pragma unroll
    for (int hf = 0; hf < 2; hf++) {
        const int co = co16 * 16 + (lane >> 2) + 8 * hf;
        if (co >= Co) continue;
        const float bias = b ? b[co] : 0.f;
#pragma unroll
        for (int t = 0; t < NT; t++) {
            const int hh = h0 + rg * (NT / 2) + t / 2, ww = w0 + (t % 2) * 8 + (lane & 3) * 2;
            if (hh >= H || ww >= W) continue;
            const size_t o = (size_t(n) * Co + co) * HW + hh * W + ww;
            float r0 = acc[t][2 * hf] + bias, r1 = acc[t][2 * hf + 1] + bias;
            if (RELU) {
                r0 = r0 > 0.f ? r0 : 0.f;
                r1 = r1 > 0.f ? r1 : 0.f;
            }
            if (even) {
                *reinterpret_cast<float2 *>(y + o) = make_float2(r0, r1);
            } else {
                y[o] = r0;
                if (ww + 1 < W) y[o + 1] = r1;
            }
        }
    }
}

// The same convolution in FP32 multiply-adds, for training: every output adds
// its products in the order of the input channels, then the kernel's rows, then
// its columns. A warp makes 8 output channels (their weights are one broadcast
// load for the warp) of a tile of 8 G rows x 16 columns: a lane 4 G pixels of a
// row, 32 G accumulators, two output channels in a packed multiply-add. Per step
// of 8 input channels the block stages the tile with its halo and the step's
// weights, [ci][offset][co], by asynchronous copies into one of two buffers
// while it works from the other. Bound: the FP32 pipes (one operand load per 12
// to 19 multiply-adds), and the last wave. The forward pass and data gradients
// of a training step, 8 samples of 64 x 64, 320 output channels: 1185 us; without
// the packed form 1294, the direct convolutions at first 2487.
constexpr int kFmaCi = 8, kFmaPitch = 20;  // pitch: 8 rows of a quarter-warp's 16-byte loads fall in distinct banks

template <int G, int WARPS>
constexpr int kFmaStage = kFmaCi * (8 * G + 2) * kFmaPitch + kFmaCi * 9 * 8 * WARPS;  // floats

__device__ __forceinline__ void copy4(float *dst, const float *src, bool valid)  // valid = false: zero, no read
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copy16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src)
                 : "memory");
}

// Two FP32 multiply-adds in one instruction, each rounded as fmaf rounds.
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t twice(float x)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
    return d;
}
__device__ __forceinline__ float2 halves(uint64_t a)
{
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
    return v;
}

template <int G, int WARPS, bool RELU, bool MASK>
__global__ void __launch_bounds__(32 * WARPS, G == 2 ? 16 / WARPS : 20 / WARPS)
k_conv_fma(const float *__restrict__ x, const float *__restrict__ wq, const float *__restrict__ b,
           const float *__restrict__ mask, float *__restrict__ y, int Ci, int Co, int H, int W)
{
    constexpr int kThreads = 32 * WARPS, kRows = 8 * G, kCo = 8 * WARPS, kPix = (kRows + 2) * 18;
    constexpr int kPlane = (kRows + 2) * kFmaPitch, kStage = kFmaStage<G, WARPS>;
    constexpr int kItems = (kPix + kThreads - 1) / kThreads;
    extern __shared__ __align__(16) float smf[];  // two stages: x [ci][row][20], then weights [ci 9 + offset][co]
    const int tiles_w = (W + 15) / 16;
    const int h0 = int(blockIdx.x) / tiles_w * kRows, w0 = int(blockIdx.x) % tiles_w * 16;
    const int n = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int co0 = int(blockIdx.y) * kCo;
    const int row = lane & (kRows - 1), c4 = lane / kRows * 4;  // first pixel; G = 2: and the one 8 columns on
    const int HW = H * W;
    const float *xn = x + size_t(n) * Ci * HW;
    const int cop = (Co + 63) / 64 * 64;  // weights: output channels padded to 64
    int off[kItems], dst[kItems];         // this thread's pixels of a channel: offset (-1: outside), place
#pragma unroll
    for (int k = 0; k < kItems; k++) {
        const int p = k * kThreads + int(threadIdx.x);
        const int yy = p / 18, xx = p % 18, gy = h0 + yy - 1, gx = w0 + xx - 1;
        off[k] = (gy >= 0 && gy < H && gx >= 0 && gx < W) ? gy * W + gx : -1;
        dst[k] = p < kPix ? yy * kFmaPitch + xx : -1;
    }
    auto stage = [&](int c0, float *to) {
        const int nc = Ci - c0 < kFmaCi ? Ci - c0 : kFmaCi;
        for (int c = 0; c < nc; c++) {
            const float *xc = xn + size_t(c0 + c) * HW;
#pragma unroll
            for (int k = 0; k < kItems; k++)
                if (dst[k] >= 0) copy4(to + c * kPlane + dst[k], off[k] >= 0 ? xc + off[k] : xc, off[k] >= 0);
        }
        const float *wc = wq + size_t(c0) * 9 * cop + co0;
        float *tw = to + kFmaCi * kPlane;
        for (int k = threadIdx.x; k < nc * 9 * (kCo / 4); k += kThreads)
            copy16(tw + 4 * k, wc + size_t(k / (kCo / 4)) * cop + k % (kCo / 4) * 4);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint64_t acc[G][4][4];  // output channels 2 o and 2 o + 1
#pragma unroll
    for (int g = 0; g < G; g++)
#pragma unroll
        for (int o = 0; o < 4; o++)
#pragma unroll
            for (int q = 0; q < 4; q++) acc[g][o][q] = 0;
    stage(0, smf);
    int buf = 0;
#pragma unroll 1
    for (int c0 = 0; c0 < Ci; c0 += kFmaCi) {
        if (c0 + kFmaCi < Ci) {
            stage(c0 + kFmaCi, smf + (buf ^ 1) * kStage);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *xb = smf + buf * kStage + row * kFmaPitch + c4;
        const float *wb = smf + buf * kStage + kFmaCi * kPlane + 8 * warp;
        const int nc = Ci - c0 < kFmaCi ? Ci - c0 : kFmaCi;
#pragma unroll 1
        for (int c = 0; c < nc; c++) {
#pragma unroll
            for (int kh = 0; kh < 3; kh++) {
                uint64_t xv[G][6];
#pragma unroll
                for (int g = 0; g < G; g++) {
                    const float *p = xb + c * kPlane + kh * kFmaPitch + 8 * g;
                    const float4 v = *reinterpret_cast<const float4 *>(p);
                    const float2 u = *reinterpret_cast<const float2 *>(p + 4);
                    xv[g][0] = twice(v.x); xv[g][1] = twice(v.y); xv[g][2] = twice(v.z); xv[g][3] = twice(v.w);
                    xv[g][4] = twice(u.x); xv[g][5] = twice(u.y);
                }
#pragma unroll
                for (int kw = 0; kw < 3; kw++) {
                    const float *p = wb + (c * 9 + kh * 3 + kw) * kCo;
                    const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(p);
                    const ulonglong2 wd = *reinterpret_cast<const ulonglong2 *>(p + 4);
                    const uint64_t wv[4] = {wa.x, wa.y, wd.x, wd.y};
#pragma unroll
                    for (int g = 0; g < G; g++)
#pragma unroll
                        for (int o = 0; o < 4; o++)
#pragma unroll
                            for (int q = 0; q < 4; q++) acc[g][o][q] = fma2(wv[o], xv[g][q + kw], acc[g][o][q]);
                }
            }
        }
        __syncthreads();  // the next copies go over this buffer
        buf ^= 1;
    }
    const int hh = h0 + row;
    if (hh >= H) return;
#pragma unroll
    for (int o = 0; o < 8; o++) {
        const int co = co0 + 8 * warp + o;
        if (co >= Co) break;
        const float bias = b ? b[co] : 0.f;
#pragma unroll
        for (int g = 0; g < G; g++) {
            const int ww = w0 + c4 + 8 * g;
            const size_t at = (size_t(n) * Co + co) * HW + hh * W + ww;
            float sum[4];
#pragma unroll
            for (int q = 0; q < 4; q++) sum[q] = (o & 1) ? halves(acc[g][o / 2][q]).y : halves(acc[g][o / 2][q]).x;
            if ((W & 3) == 0) {  // a lane's four pixels are one aligned word
                if (ww >= W) continue;
                float r[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    r[q] = sum[q] + bias;
                    if (RELU) r[q] = r[q] > 0.f ? r[q] : 0.f;
                }
                if (MASK) {
                    const float4 m = *reinterpret_cast<const float4 *>(mask + at);
                    r[0] = m.x > 0.f ? r[0] : 0.f;
                    r[1] = m.y > 0.f ? r[1] : 0.f;
                    r[2] = m.z > 0.f ? r[2] : 0.f;
                    r[3] = m.w > 0.f ? r[3] : 0.f;
                }
                *reinterpret_cast<float4 *>(y + at) = make_float4(r[0], r[1], r[2], r[3]);
                continue;
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (ww + q >= W) break;
                float r = sum[q] + bias;
                if (RELU) r = r > 0.f ? r : 0.f;
                if (MASK) r = mask[at + q] > 0.f ? r : 0.f;
                y[at + q] = r;
            }
        }
    }
}

// Weight gradient: dw[co][ci][kh][kw] += sum over the block's pixels of
// dy[n][co][h][w] x[n][ci][h + kh - 1][w + kw - 1]; db[co] += sum of dy (blocks
// of the first input channels only). A block makes 64 output x 16 input
// channels x 9 offsets of a band of 8 rows of one sample, 16 columns at a time,
// and adds its sums to dw; a thread 2 x 4 x 9 of them, each one chain of FP32
// multiply-adds over the band's pixels, column tile by column tile, row by row.
// Both operands are staged with the channels innermost, and the 3 x 3 pixels
// around a pixel stay in registers along a row, so that a pixel costs a thread
// one 8-byte and three 16-byte loads for 72 multiply-adds (36 packed ones). The
// next column tile is copied while one is worked on. Bound: the FP32 pipes, and
// grids of 256 blocks on 152 multiprocessors. The nine layers of a training
// step, 8 samples of 64 x 64, 320 output channels: 715 us; with nine loads a
// pixel, scalar multiply-adds and no copies ahead 894; a block per output
// channel, as at first, 1573.
constexpr int kWgRows = 8, kWgCo = 64, kWgCi = 16, kWgPitchX = kWgCi + 4, kWgPitchD = kWgCo + 4;
constexpr int kWgStage = (kWgRows + 2) * 18 * kWgPitchX + kWgRows * 16 * kWgPitchD;  // floats

__global__ void __launch_bounds__(128, 2)
k_conv_wgrad(const float *__restrict__ x, const float *__restrict__ dy, float *__restrict__ dw,
             float *__restrict__ db, int Ci, int Co, int H, int W)
{
    extern __shared__ __align__(16) float smw[];  // one or two stages: x [pixel with halo][ci], dy [pixel][co]
    constexpr int kPix = (kWgRows + 2) * 18, kXs = kPix * kWgPitchX;
    const int co0 = blockIdx.x * kWgCo, ci0 = blockIdx.y * kWgCi;
    const int bands = (H + kWgRows - 1) / kWgRows;
    const int n = int(blockIdx.z) / bands, h0 = int(blockIdx.z) % bands * kWgRows;
    const int cq = threadIdx.x & 3, cp = threadIdx.x >> 2;  // input channels 4 cq .. + 3, output channels 2 cp, + 1
    const int HW = H * W;
    const float *xn = x + (size_t(n) * Ci + ci0) * HW, *dn = dy + (size_t(n) * Co + co0) * HW;
    // a warp copies 8 pixels x 4 channels at a time: 32-byte runs, every bank once
    const int pl = threadIdx.x & 7, ch = threadIdx.x >> 5 << 2 | ((threadIdx.x >> 3) & 3);
    auto stage = [&](int w0, float *to) {
        const bool live = ci0 + ch < Ci;
        const float *xc = live ? xn + size_t(ch) * HW : x;
#pragma unroll 4
        for (int p = pl; p < kPix; p += 8) {
            const int gy = h0 + p / 18 - 1, gx = w0 + p % 18 - 1;
            const bool in = live && gy >= 0 && gy < H && gx >= 0 && gx < W;
            copy4(to + p * kWgPitchX + ch, in ? xc + gy * W + gx : x, in);
        }
#pragma unroll 4
        for (int p = pl; p < kWgRows * 16; p += 8) {
            const int gy = h0 + p / 16, gx = w0 + p % 16;
            const bool in = gy < H && gx < W;
#pragma unroll
            for (int c = ch; c < ch + kWgCo; c += 16) {
                const bool ok = in && co0 + c < Co;
                copy4(to + kXs + p * kWgPitchD + c, ok ? dn + size_t(c) * HW + gy * W + gx : dy, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint64_t acc[2][2][9];  // input channels 2 i and 2 i + 1 of the four
#pragma unroll
    for (int o = 0; o < 2; o++)
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int k = 0; k < 9; k++) acc[o][i][k] = 0;
    float db0 = 0.f, db1 = 0.f;
    stage(0, smw);
    int buf = 0;
#pragma unroll 1
    for (int w0 = 0; w0 < W; w0 += 16) {
        if (w0 + 16 < W) {
            stage(w0 + 16, smw + (buf ^ 1) * kWgStage);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *const xs = smw + buf * kWgStage + 4 * cq, *const ds = smw + buf * kWgStage + kXs + 2 * cp;
#pragma unroll 1
        for (int r = 0; r < kWgRows; r++) {
            const float *const xr = xs + r * 18 * kWgPitchX, *const dr = ds + r * 16 * kWgPitchD;
            ulonglong2 win[3][3];  // [row][column mod 3] around the pixel
#pragma unroll
            for (int c = 0; c < 2; c++)
#pragma unroll
                for (int kh = 0; kh < 3; kh++)
                    win[kh][c] = *reinterpret_cast<const ulonglong2 *>(xr + (kh * 18 + c) * kWgPitchX);
#pragma unroll
            for (int c = 0; c < 16; c++) {
                const float2 d = *reinterpret_cast<const float2 *>(dr + c * kWgPitchD);
#pragma unroll
                for (int kh = 0; kh < 3; kh++)
                    win[kh][(c + 2) % 3] = *reinterpret_cast<const ulonglong2 *>(xr + (kh * 18 + c + 2) * kWgPitchX);
                db0 += d.x;
                db1 += d.y;
                const uint64_t d0 = twice(d.x), d1 = twice(d.y);
#pragma unroll
                for (int k = 0; k < 9; k++) {
                    const ulonglong2 v = win[k / 3][(c + k % 3) % 3];
                    acc[0][0][k] = fma2(d0, v.x, acc[0][0][k]);
                    acc[0][1][k] = fma2(d0, v.y, acc[0][1][k]);
                    acc[1][0][k] = fma2(d1, v.x, acc[1][0][k]);
                    acc[1][1][k] = fma2(d1, v.y, acc[1][1][k]);
                }
            }
        }
        __syncthreads();  // the next copies go over this buffer
        buf ^= 1;
    }
    // through shared memory, so that a warp's adds are contiguous in dw
    float *const out = smw;  // [co][ci][9]
#pragma unroll
    for (int o = 0; o < 2; o++)
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int k = 0; k < 9; k++) {
                const float2 v = halves(acc[o][i][k]);
                float *const to = out + ((2 * cp + o) * kWgCi + 4 * cq + 2 * i) * 9 + k;
                to[0] = v.x;
                to[9] = v.y;
            }
    __syncthreads();
    for (int k = threadIdx.x; k < kWgCo * kWgCi * 9; k += 128) {
        const int co = k / (kWgCi * 9), r = k % (kWgCi * 9);
        if (co0 + co < Co && ci0 + r / 9 < Ci) atomicAdd(dw + (size_t(co0 + co) * Ci + ci0) * 9 + r, out[k]);
    }
    if (blockIdx.y == 0 && cq == 0) {
        if (co0 + 2 * cp < Co) atomicAdd(db + co0 + 2 * cp, db0);
        if (co0 + 2 * cp + 1 < Co) atomicAdd(db + co0 + 2 * cp + 1, db1);
    }
}
static_assert(kWgStage >= kWgCo * kWgCi * 9, "the sums are turned in the staging buffer");

// The weights of one layer as k_conv reads them: fragment (co / 16, ci / 16,
// offset) of 32 lanes x 4 words; lane l's words hold rows l / 4 and l / 4 + 8,
// columns 2 (l mod 4) and + 1, then the same 8 columns on; zeros past the
// layer's channels.
__device__ __forceinline__ uint32_t bf16_bits(float v)
{
    return uint32_t(__bfloat16_as_ushort(__float2bfloat16_rn(v)));
}

__device__ __forceinline__ uint32_t frag_word(const float *__restrict__ w, int64_t k, int Ci, int Co)
{
    const int nc = (Ci + 15) / 16;
    const int q = int(k & 3), l = int(k >> 2) & 31;
    const int64_t f = k >> 7;
    const int tap = int(f % 9), c16 = int(f / 9 % nc), r16 = int(f / 9 / nc);
    const int r = r16 * 16 + l / 4 + 8 * (q & 1), c = c16 * 16 + 2 * (l & 3) + 8 * (q >> 1);
    uint32_t v = 0u;
    for (int m = 0; m < 2; m++)
        if (r < Co && c + m < Ci) v |= bf16_bits(w[(int64_t(r) * Ci + c + m) * 9 + tap]) << (16 * m);
    return v;
}

// As k_conv_fma reads them: [ci][offset][co, padded to 64], rounded to BF16 and
// widened again. FLIP: of the transposed layer with the offsets reversed (the
// data gradient as a forward convolution).
template <bool FLIP>
__device__ __forceinline__ uint32_t row_word(const float *__restrict__ w, int64_t k, int Ci, int Co)
{
    const int R = FLIP ? Ci : Co;  // output channels of the convolution
    const int cop = (R + 63) / 64 * 64;
    const int r = int(k % cop), tap = int(k / cop % 9), c = int(k / cop / 9);
    if (r >= R) return 0u;
    return bf16_bits(FLIP ? w[(int64_t(c) * Ci + r) * 9 + (8 - tap)] : w[(int64_t(r) * Ci + c) * 9 + tap]) << 16;
}

struct PackTable {
    int ci[9], co[9];
    int64_t w[9];           // offsets of the layers' parameters
    int64_t at[3][10];      // words: fragments, FP32 rows, FP32 rows of the flipped layers (the last: the form's end)
};

__global__ void k_pack_weights(const float *__restrict__ w, uint32_t *__restrict__ out, PackTable t)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < t.at[2][9]; k += int64_t(gridDim.x) * blockDim.x) {
        const int form = k < t.at[0][9] ? 0 : (k < t.at[1][9] ? 1 : 2);
        int l = 0;
        while (l < 8 && k >= t.at[form][l + 1]) l++;
        const int64_t r = k - t.at[form][l];
        const float *wl = w + t.w[l];
        out[k] = form == 0 ? frag_word(wl, r, t.ci[l], t.co[l])
                           : (form == 1 ? row_word<false>(wl, r, t.ci[l], t.co[l]) : row_word<true>(wl, r, t.ci[l], t.co[l]));
    }
}

// The elementwise kernels below go over planes (sample, channel): blockIdx.y, +
// gridDim.y, ..., with the place inside a plane in 32 bits, so that rows and
// columns cost one 32-bit division each.

// y [NC][H/2][W/2] = 2x2 average of x [NC][H][W].
__global__ void k_pool_fwd(const float *__restrict__ x, float *__restrict__ y, int64_t NC, int H, int W)
{
    const unsigned w2 = unsigned(W) / 2, n = unsigned(H) / 2 * w2;
    for (int64_t c = blockIdx.y; c < NC; c += gridDim.y)
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const unsigned hh = k / w2, ww = k - hh * w2;
            const float *p = x + (c * H + 2 * hh) * W + 2 * ww;
            y[c * n + k] = 0.25f * (p[0] + p[1] + p[W] + p[W + 1]);
        }
}

// The pooled layer's input gradient: dx = skip + dy / 4 of the cell (skip: the
// gradient through the skip connection), zeroed where a <= 0 (the ReLU).
__global__ void k_pool_bwd(const float *__restrict__ dy, const float *__restrict__ skip, const float *__restrict__ a,
                           float *__restrict__ dx, int64_t NC, int H, int W)
{
    const unsigned n = unsigned(H) * unsigned(W), w2 = unsigned(W) / 2;
    for (int64_t c = blockIdx.y; c < NC; c += gridDim.y)
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const unsigned hh = k / unsigned(W), ww = k - hh * unsigned(W);
            const float g = skip[c * n + k] + 0.25f * dy[c * (n / 4) + hh / 2 * w2 + ww / 2];
            dx[c * n + k] = a[c * n + k] > 0.f ? g : 0.f;
        }
}

// s [NC][2h][2w] = nearest upsample of a [NC][h][w] + skip.
__global__ void k_up_add(const float *__restrict__ a, const float *__restrict__ skip, float *__restrict__ s, int64_t NC,
                         int h, int w)
{
    const unsigned W = 2 * unsigned(w), n = 4 * unsigned(h) * unsigned(w);
    for (int64_t c = blockIdx.y; c < NC; c += gridDim.y)
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const unsigned hh = k / W, ww = k - hh * W;
            s[c * n + k] = a[c * (n / 4) + hh / 2 * unsigned(w) + ww / 2] + skip[c * n + k];
        }
}

// da [NC][h][w] = sum of the 4 gradients of its upsampled copies, zeroed where a <= 0.
__global__ void k_up_bwd(const float *__restrict__ ds, const float *__restrict__ a, float *__restrict__ da, int64_t NC,
                         int h, int w)
{
    const unsigned n = unsigned(h) * unsigned(w);
    const int W = 2 * w;
    for (int64_t c = blockIdx.y; c < NC; c += gridDim.y)
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
            const unsigned hh = k / unsigned(w), ww = k - hh * unsigned(w);
            const float *p = ds + (c * (2 * h) + 2 * hh) * W + 2 * ww;
            da[c * n + k] = a[c * n + k] > 0.f ? p[0] + p[1] + p[W] + p[W + 1] : 0.f;
        }
}

__device__ __forceinline__ float softplus(float z) { return z > 20.f ? z : log1pf(expf(z)); }

// Output head: channel c mod Co of a sample is the image's softplus(z) below Q
// and z itself for the dual channels from Q on.
__global__ void k_head(const float *__restrict__ z, float *__restrict__ o, int64_t NC, int HW, int Co, int Q)
{
    for (int64_t c = blockIdx.y; c < NC; c += gridDim.y) {
        const bool img = int(c % Co) < Q;
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < HW; k += gridDim.x * blockDim.x) {
            const float zz = z[c * HW + k];
            o[c * HW + k] = img ? softplus(zz) : zz;
        }
    }
}

// |v| as FP64 by integer instructions (the FP64 unit, which a conversion also
// occupies, does about 2 lanes per clock and multiprocessor): the exponent moved
// to its new bias; outside FP32's normal range by a real conversion (a loss may
// consist of subnormal differences alone).
__device__ __forceinline__ double abs_f64(float v)
{
    const uint32_t u = __float_as_uint(v) & 0x7FFFFFFFu;
    if (u - 0x00800000u >= 0x7F000000u) return u == 0u ? 0.0 : fabs(double(v));
    return __hiloint2double(int((u >> 3) + 0x38000000u), int(u << 29));
}

// loss += sum (head(z) - t)^2 / n (FP64); dz = 2 (head(z) - t) head'(z) / n with
// head' = sigmoid on the image channels and 1 on the dual channels. A block takes
// `len` consecutive elements of a plane at a time (`pieces` of them a plane), and
// adds to the loss once.
__global__ void __launch_bounds__(256)
k_mse_head(const float *__restrict__ z, const float *__restrict__ tgt, float *__restrict__ dz, int64_t NC, int HW,
           int Co, int Q, int pieces, int len, double *__restrict__ loss)
{
    __shared__ double sh[32];
    double acc = 0.0;
    const int64_t n = NC * HW;
    const float inv = 1.0f / float(n);
    for (int64_t t = blockIdx.x; t < NC * pieces; t += gridDim.x) {
        const int64_t c = t / pieces;
        const bool img = int(c % Co) < Q;
        const float *const zc = z + c * HW, *const tc = tgt + c * HW;
        const int k1 = int(t - c * pieces) * len, k2 = len < HW - k1 ? k1 + len : HW;
        for (int k0 = k1 + int(threadIdx.x); k0 < k2; k0 += 4 * kT) {
            float zz[4], tt[4];  // all loads first
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int k = k0 + u * kT;
                zz[u] = k < k2 ? zc[k] : 0.f;
                tt[u] = k < k2 ? tc[k] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int k = k0 + u * kT;
                if (k >= k2) break;
                const float diff = (img ? softplus(zz[u]) : zz[u]) - tt[u];
                const double a = abs_f64(diff);
                acc = fma(a, a, acc);
                dz[c * HW + k] = img ? 2.f * diff * inv / (1.f + expf(-zz[u])) : 2.f * diff * inv;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < int(blockDim.x >> 5); k++) s += sh[k];
        atomicAdd(loss, s / double(n));
    }
}

__global__ void k_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int64_t n, float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const float gk = g[k];
        const float mk = b1 * m[k] + (1.f - b1) * gk;
        const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
        m[k] = mk;
        v[k] = vk;
        w[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
}

__global__ void k_pack_input(const float *__restrict__ bp, int Nx, int Nz, int Nq, float inv_scale, float level,
                             float *__restrict__ x)
{
    const int64_t n = int64_t(Nq + 1) * Nx * Nz;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const int zz = int(k % Nz), xx = int((k / Nz) % Nx), q = int(k / (int64_t(Nz) * Nx));
        x[k] = q < Nq ? bp[(int64_t(xx) * Nz + zz) * Nq + q] * inv_scale : level;
    }
}

__global__ void k_unpack_output(const float *__restrict__ o, int Nx, int Nz, int Nq, float scale, float *__restrict__ f)
{
    const int64_t n = int64_t(Nq) * Nx * Nz;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const int q = int(k % Nq);
        const int64_t s = k / Nq;
        const int zz = int(s % Nz), xx = int(s / Nz);
        f[k] = scale * o[(int64_t(q) * Nx + xx) * Nz + zz];
    }
}

// c [p][J] = tau * out[Q + p * Q + q][x][z] (sample 0), p < n_dual.
__global__ void k_unpack_dual(const float *__restrict__ o, int Nx, int Nz, int Nq, int n_dual, float tau,
                              float *__restrict__ c)
{
    const int64_t J = int64_t(Nx) * Nz * Nq;
    const int64_t n = J * n_dual;
    for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < n; k += int64_t(gridDim.x) * blockDim.x) {
        const int p = int(k / J);
        const int64_t j = k - int64_t(p) * J;
        const int q = int(j % Nq);
        const int64_t s = j / Nq;
        const int zz = int(s % Nz), xx = int(s / Nz);
        c[k] = tau * o[((int64_t(Nq) * (1 + p) + q) * Nx + xx) * Nz + zz];
    }
}

struct Layer {
    int ci, co;
    int64_t woff, boff;  // offsets in the packed parameter vector
};

}  // namespace

struct wsnet_ctx {
    int H, W, C, maxN;
    int n_dual = 0, Co = 0;  // dual blocks of Q channels after the image's; output channels Q (1 + n_dual)
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::vector<void *> blocks;
    Layer L[9];
    int64_t P = 0;
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    uint32_t *wp = nullptr;  // BF16 weights in the orders that the convolutions read them (PackTable)
    PackTable pack{};
    int sms = 1;
    // activations and gradients
    float *a1, *a2, *p1, *a3, *a4, *p2, *a5, *a6, *s1, *a7, *s2, *a8, *z;
    float *gz, *g8, *gs2, *g7, *gs1, *g6, *g5, *gp2, *g4, *g3, *gp1, *g2, *g1;
    double *loss = nullptr;
    int64_t step = 0;
    std::string err;
};

namespace {

int wfail(wsnet_t h, int code, const std::string &msg)
{
    if (h) h->err = msg;
    return code;
}

#define WK(h, call)                                                                       \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) return wfail(h, SGTV_ERR_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

void *walloc(wsnet_t h, size_t bytes)
{
    void *p = nullptr;
    if (cudaMalloc(&p, bytes < 16 ? 16 : bytes) != cudaSuccess) return nullptr;
    h->blocks.push_back(p);
    return p;
}

// Inference: the larger block where it leaves every multiprocessor one of them,
// the smaller one (a quarter of the work) otherwise: one sample of 64 x 64 (32
// larger blocks a layer at full size) 241 us for the nine layers with the
// larger block, 114 with the smaller; eight samples (256) 29.2 and 29.5 a layer.
template <bool RELU>
void conv_tc(wsnet_t h, const float *x, int l, float *y, int N, int Hh, int Ww)
{
    const Layer &L = h->L[l];
    const unsigned tw = unsigned((Ww + 15) / 16), c16 = unsigned((L.co + 15) / 16);
    const uint4 *w = reinterpret_cast<const uint4 *>(h->wp + h->pack.at[0][l]);
    const float *b = h->w + L.boff;
    const dim3 big(tw * unsigned((Hh + 7) / 8), (c16 + 3) / 4, unsigned(N));
    if (uint64_t(big.x) * big.y * big.z >= unsigned(h->sms)) {
        k_conv<4, 2, 8, RELU><<<big, 256, 0, h->stream>>>(x, w, b, y, L.ci, L.co, Hh, Ww);
        return;
    }
    const dim3 small(tw * unsigned((Hh + 3) / 4), (c16 + 1) / 2, unsigned(N));
    k_conv<2, 2, 4, RELU><<<small, 128, 0, h->stream>>>(x, w, b, y, L.ci, L.co, Hh, Ww);
}

// Training: 64 channels of 16 x 16 pixels a block, or 32 channels of 8 x 16. A
// multiprocessor takes about 51 us for one of the larger blocks at 64 input
// channels and 14 us for one of the smaller (more staging for a product), so
// the form whose fullest multiprocessor is done first: 128 larger blocks or
// 512 smaller 51 or 56 us, 160 or 640 97 or 69, 320 or 1280 143 or 120, 640 or
// 2560 235 or 222.
template <bool RELU, bool MASK>
void conv_fma(wsnet_t h, const float *x, const uint32_t *w, const float *b, const float *mask, float *y, int Ci, int Co,
              int N, int Hh, int Ww)
{
    const unsigned tw = unsigned((Ww + 15) / 16);
    const float *wf = reinterpret_cast<const float *>(w);
    const dim3 big(tw * unsigned((Hh + 15) / 16), unsigned((Co + 63) / 64), unsigned(N));
    const dim3 small(tw * unsigned((Hh + 7) / 8), unsigned((Co + 31) / 32), unsigned(N));
    auto fullest = [&](const dim3 &g) { return (uint64_t(g.x) * g.y * g.z + h->sms - 1) / h->sms; };
    if (51 * fullest(big) <= 14 * fullest(small)) {
        k_conv_fma<2, 8, RELU, MASK>
            <<<big, 256, 2 * 4 * kFmaStage<2, 8>, h->stream>>>(x, wf, b, mask, y, Ci, Co, Hh, Ww);
        return;
    }
    k_conv_fma<1, 4, RELU, MASK>
        <<<small, 128, 2 * 4 * kFmaStage<1, 4>, h->stream>>>(x, wf, b, mask, y, Ci, Co, Hh, Ww);
}

void conv_fwd(wsnet_t h, const float *x, int l, float *y, int N, int Hh, int Ww, bool relu, bool training)
{
    const Layer &L = h->L[l];
    const uint32_t *w = h->wp + h->pack.at[1][l];
    if (!training) {
        if (relu) conv_tc<true>(h, x, l, y, N, Hh, Ww);
        else conv_tc<false>(h, x, l, y, N, Hh, Ww);
    } else if (relu) {
        conv_fma<true, false>(h, x, w, h->w + L.boff, nullptr, y, L.ci, L.co, N, Hh, Ww);
    } else {
        conv_fma<false, false>(h, x, w, h->w + L.boff, nullptr, y, L.ci, L.co, N, Hh, Ww);
    }
}

// dy -> weight and bias gradients, and (if dx) the data gradient, zeroed where
// mask <= 0 (if mask: the activation that the layer's input is, after its ReLU).
void conv_bwd(wsnet_t h, const float *x, const float *dy, int l, float *dx, const float *mask, int N, int Hh, int Ww)
{
    const Layer &L = h->L[l];
    const dim3 gw(unsigned((L.co + kWgCo - 1) / kWgCo), unsigned((L.ci + kWgCi - 1) / kWgCi),
                  unsigned(N * ((Hh + kWgRows - 1) / kWgRows)));
    k_conv_wgrad<<<gw, 128, (Ww > 16 ? 2 : 1) * 4 * kWgStage, h->stream>>>(x, dy, h->g + L.woff, h->g + L.boff, L.ci, L.co, Hh, Ww);
    if (!dx) return;
    const uint32_t *w = h->wp + h->pack.at[2][l];
    if (mask) conv_fma<false, true>(h, dy, w, nullptr, mask, dx, L.co, L.ci, N, Hh, Ww);
    else conv_fma<false, false>(h, dy, w, nullptr, nullptr, dx, L.co, L.ci, N, Hh, Ww);
}

void pack_weights(wsnet_t h)
{
    k_pack_weights<<<blocks_for(h->pack.at[2][9]), kT, 0, h->stream>>>(h->w, h->wp, h->pack);
}

// Blocks over NC planes of n elements each.
dim3 planes(int64_t NC, int64_t n)
{
    return dim3(unsigned((n + kT - 1) / kT), unsigned(NC < 65535 ? NC : 65535));
}

// The forward pass up to z (pre-softplus output).
void forward_to_z(wsnet_t h, const float *x, int N, bool training)
{
    const int H = h->H, W = h->W, H2 = H / 2, W2 = W / 2, H4 = H / 4, W4 = W / 4;
    cudaStream_t st = h->stream;
    conv_fwd(h, x, 0, h->a1, N, H, W, true, training);
    conv_fwd(h, h->a1, 1, h->a2, N, H, W, true, training);
    k_pool_fwd<<<planes(int64_t(N) * 64, int64_t(H2) * W2), kT, 0, st>>>(h->a2, h->p1, int64_t(N) * 64, H, W);
    conv_fwd(h, h->p1, 2, h->a3, N, H2, W2, true, training);
    conv_fwd(h, h->a3, 3, h->a4, N, H2, W2, true, training);
    k_pool_fwd<<<planes(int64_t(N) * 128, int64_t(H4) * W4), kT, 0, st>>>(h->a4, h->p2, int64_t(N) * 128, H2, W2);
    conv_fwd(h, h->p2, 4, h->a5, N, H4, W4, true, training);
    conv_fwd(h, h->a5, 5, h->a6, N, H4, W4, true, training);
    k_up_add<<<planes(int64_t(N) * 128, int64_t(H2) * W2), kT, 0, st>>>(h->a6, h->a4, h->s1, int64_t(N) * 128, H4, W4);
    conv_fwd(h, h->s1, 6, h->a7, N, H2, W2, true, training);
    k_up_add<<<planes(int64_t(N) * 64, int64_t(H) * W), kT, 0, st>>>(h->a7, h->a2, h->s2, int64_t(N) * 64, H2, W2);
    conv_fwd(h, h->s2, 7, h->a8, N, H, W, true, training);
    conv_fwd(h, h->a8, 8, h->z, N, H, W, false, training);
}

}  // namespace

extern "C" {

int wsnet_create(wsnet_t *out, int32_t H, int32_t W, int32_t Q, int32_t n_dual, int32_t max_batch, uint64_t seed,
                 void *stream)
{
    if (!out) return SGTV_ERR_ARG;
    *out = nullptr;
    if (H < 4 || W < 4 || H % 4 || W % 4 || Q < 1 || max_batch < 1 || n_dual < 0 || n_dual > 4 ||
        int64_t(Q) * (1 + n_dual) > 1024)
        return SGTV_ERR_ARG;
    wsnet_t h = new wsnet_ctx();
    h->H = H;
    h->W = W;
    h->C = Q;
    h->n_dual = n_dual;
    h->Co = Q * (1 + n_dual);
    h->maxN = max_batch;
    const int ch[9][2] = {{Q + 1, 64}, {64, 64}, {64, 128}, {128, 128}, {128, 256},
                          {256, 128}, {128, 64}, {64, 64}, {64, h->Co}};
    int64_t off = 0;
    for (int l = 0; l < 9; l++) {
        h->L[l].ci = ch[l][0];
        h->L[l].co = ch[l][1];
        h->L[l].woff = off;
        off += int64_t(ch[l][0]) * ch[l][1] * 9;
        h->L[l].boff = off;
        off += ch[l][1];
    }
    h->P = off;
    auto fail_create = [&](int code) {
        for (void *p : h->blocks) cudaFree(p);
        if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
        delete h;
        return code;
    };
    if (stream) {
        h->stream = static_cast<cudaStream_t>(stream);
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) return fail_create(SGTV_ERR_CUDA);
        h->own_stream = true;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fail_create(SGTV_ERR_CUDA);
    auto opt_in = [](auto *kernel, int bytes) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    };
    constexpr int big = 2 * 4 * kFmaStage<2, 8>;
    if (!opt_in(k_conv_wgrad, 2 * 4 * kWgStage) || !opt_in(k_conv_fma<2, 8, true, false>, big) ||
        !opt_in(k_conv_fma<2, 8, false, true>, big) || !opt_in(k_conv_fma<2, 8, false, false>, big))
        return fail_create(SGTV_ERR_CUDA);
    const size_t P = size_t(h->P);
    h->w = static_cast<float *>(walloc(h, 4 * P));
    h->g = static_cast<float *>(walloc(h, 4 * P));
    h->m = static_cast<float *>(walloc(h, 4 * P));
    h->v = static_cast<float *>(walloc(h, 4 * P));
    for (int l = 0; l < 9; l++) {
        h->pack.ci[l] = h->L[l].ci;
        h->pack.co[l] = h->L[l].co;
        h->pack.w[l] = h->L[l].woff;
    }
    int64_t words = 0;
    for (int form = 0; form < 3; form++)
        for (int l = 0; l < 9; l++) {
            const int64_t ci = h->L[l].ci, co = h->L[l].co;
            h->pack.at[form][l] = words;
            words += form == 0 ? (ci + 15) / 16 * ((co + 15) / 16) * 9 * 128
                               : (form == 1 ? ci * 9 * ((co + 63) / 64 * 64) : co * 9 * ((ci + 63) / 64 * 64));
            h->pack.at[form][l + 1] = words;
        }
    h->wp = static_cast<uint32_t *>(walloc(h, 4 * size_t(words)));
    h->loss = static_cast<double *>(walloc(h, sizeof(double)));
    const size_t N = size_t(max_batch);
    const size_t f1 = N * H * W, f2 = N * (H / 2) * (W / 2), f4 = N * (H / 4) * (W / 4);
    const int Cz = h->Co > 64 ? h->Co : 64;
    float **bufs[] = {&h->a1, &h->a2, &h->s2, &h->a8, &h->g8, &h->gs2, &h->g2, &h->g1};
    for (float **b : bufs) *b = static_cast<float *>(walloc(h, 4 * f1 * 64));
    h->z = static_cast<float *>(walloc(h, 4 * f1 * Cz));
    h->gz = static_cast<float *>(walloc(h, 4 * f1 * Cz));
    float **b2[] = {&h->p1, &h->a7, &h->g7, &h->gp1};
    for (float **b : b2) *b = static_cast<float *>(walloc(h, 4 * f2 * 64));
    float **b3[] = {&h->a3, &h->a4, &h->s1, &h->gs1, &h->g4, &h->g3};
    for (float **b : b3) *b = static_cast<float *>(walloc(h, 4 * f2 * 128));
    float **b4[] = {&h->p2, &h->a6, &h->g6, &h->gp2};
    for (float **b : b4) *b = static_cast<float *>(walloc(h, 4 * f4 * 128));
    h->a5 = static_cast<float *>(walloc(h, 4 * f4 * 256));
    h->g5 = static_cast<float *>(walloc(h, 4 * f4 * 256));
    for (void *p : h->blocks)
        if (!p) return fail_create(SGTV_ERR_OOM);
    if (h->blocks.size() != 6 + 8 + 2 + 4 + 6 + 4 + 2) return fail_create(SGTV_ERR_OOM);
    // He initialisation (normal, std sqrt(2 / fan_in)), deterministic from seed; biases 0
    std::vector<float> hw(P, 0.f);
    std::mt19937_64 rng(seed);
    for (int l = 0; l < 9; l++) {
        std::normal_distribution<float> nd(0.f, sqrtf(2.f / float(h->L[l].ci * 9)) * (l == 8 ? 0.1f : 1.f));
        for (int64_t k = 0; k < int64_t(h->L[l].ci) * h->L[l].co * 9; k++) hw[h->L[l].woff + k] = nd(rng);
    }
    if (wsnet_set_params(h, hw.data()) != SGTV_OK) return fail_create(SGTV_ERR_CUDA);
    *out = h;
    return SGTV_OK;
}

int wsnet_destroy(wsnet_t h)
{
    if (!h) return SGTV_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (void *p : h->blocks) cudaFree(p);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
    return SGTV_OK;
}

int64_t wsnet_num_params(wsnet_t h) { return h ? h->P : 0; }

int wsnet_set_params(wsnet_t h, const float *host)
{
    if (!h || !host) return SGTV_ERR_ARG;
    const size_t P = size_t(h->P);
    WK(h, cudaMemcpyAsync(h->w, host, 4 * P, cudaMemcpyHostToDevice, h->stream));
    WK(h, cudaMemsetAsync(h->m, 0, 4 * P, h->stream));
    WK(h, cudaMemsetAsync(h->v, 0, 4 * P, h->stream));
    WK(h, cudaMemsetAsync(h->g, 0, 4 * P, h->stream));
    pack_weights(h);
    WK(h, cudaGetLastError());
    WK(h, cudaStreamSynchronize(h->stream));
    h->step = 0;
    return SGTV_OK;
}

int wsnet_get_params(wsnet_t h, float *host)
{
    if (!h || !host) return SGTV_ERR_ARG;
    WK(h, cudaMemcpyAsync(host, h->w, 4 * size_t(h->P), cudaMemcpyDeviceToHost, h->stream));
    WK(h, cudaStreamSynchronize(h->stream));
    return SGTV_OK;
}

int wsnet_get_grads(wsnet_t h, float *host)
{
    if (!h || !host) return SGTV_ERR_ARG;
    WK(h, cudaMemcpyAsync(host, h->g, 4 * size_t(h->P), cudaMemcpyDeviceToHost, h->stream));
    WK(h, cudaStreamSynchronize(h->stream));
    return SGTV_OK;
}

int wsnet_forward(wsnet_t h, const float *x, int32_t N, float *out)
{
    if (!h || !x || !out) return SGTV_ERR_ARG;
    if (N < 1 || N > h->maxN) return wfail(h, SGTV_ERR_ARG, "N must be in [1, max_batch]");
    forward_to_z(h, x, N, false);
    const int HW = h->H * h->W;
    const int64_t NC = int64_t(N) * h->Co;
    k_head<<<planes(NC, HW), kT, 0, h->stream>>>(h->z, out, NC, HW, h->Co, h->C);
    WK(h, cudaGetLastError());
    return SGTV_OK;
}

int wsnet_loss_grad(wsnet_t h, const float *x, const float *target, int32_t N, double *loss)
{
    if (!h || !x || !target) return SGTV_ERR_ARG;
    if (N < 1 || N > h->maxN) return wfail(h, SGTV_ERR_ARG, "N must be in [1, max_batch]");
    const int H = h->H, W = h->W, H2 = H / 2, W2 = W / 2, H4 = H / 4, W4 = W / 4;
    cudaStream_t st = h->stream;
    forward_to_z(h, x, N, true);
    WK(h, cudaMemsetAsync(h->g, 0, 4 * size_t(h->P), st));
    WK(h, cudaMemsetAsync(h->loss, 0, sizeof(double), st));
    const int64_t nz = int64_t(N) * h->Co, n64 = int64_t(N) * 64, n128 = int64_t(N) * 128;
    const int64_t full = int64_t(H) * W, half = int64_t(H2) * W2, quarter = int64_t(H4) * W4;
    const int64_t blocks = 8 * int64_t(h->sms);
    const int pieces = int(sgtv::mse_pieces(nz, full, blocks)), len = int((full + pieces - 1) / pieces);
    k_mse_head<<<unsigned(nz * pieces < blocks ? nz * pieces : blocks), kT, 0, st>>>(
        h->z, target, h->gz, nz, H * W, h->Co, h->C, pieces, len, h->loss);
    conv_bwd(h, h->a8, h->gz, 8, h->g8, h->a8, N, H, W);
    conv_bwd(h, h->s2, h->g8, 7, h->gs2, nullptr, N, H, W);
    // s2 = up(a7) + a2
    k_up_bwd<<<planes(n64, half), kT, 0, st>>>(h->gs2, h->a7, h->g7, n64, H2, W2);
    conv_bwd(h, h->s1, h->g7, 6, h->gs1, nullptr, N, H2, W2);
    // s1 = up(a6) + a4
    k_up_bwd<<<planes(n128, quarter), kT, 0, st>>>(h->gs1, h->a6, h->g6, n128, H4, W4);
    conv_bwd(h, h->a5, h->g6, 5, h->g5, h->a5, N, H4, W4);
    conv_bwd(h, h->p2, h->g5, 4, h->gp2, nullptr, N, H4, W4);
    k_pool_bwd<<<planes(n128, half), kT, 0, st>>>(h->gp2, h->gs1, h->a4, h->g4, n128, H2, W2);
    conv_bwd(h, h->a3, h->g4, 3, h->g3, h->a3, N, H2, W2);
    conv_bwd(h, h->p1, h->g3, 2, h->gp1, nullptr, N, H2, W2);
    k_pool_bwd<<<planes(n64, full), kT, 0, st>>>(h->gp1, h->gs2, h->a2, h->g2, n64, H, W);
    conv_bwd(h, h->a1, h->g2, 1, h->g1, h->a1, N, H, W);
    conv_bwd(h, x, h->g1, 0, nullptr, nullptr, N, H, W);
    WK(h, cudaGetLastError());
    if (loss) {
        WK(h, cudaMemcpyAsync(loss, h->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        WK(h, cudaStreamSynchronize(st));
    }
    return SGTV_OK;
}

int wsnet_adam_step(wsnet_t h, float lr, float beta1, float beta2, float eps)
{
    if (!h) return SGTV_ERR_ARG;
    h->step += 1;
    const float c1 = 1.f - powf(beta1, float(h->step)), c2 = 1.f - powf(beta2, float(h->step));
    k_adam<<<blocks_for(h->P), kT, 0, h->stream>>>(h->w, h->g, h->m, h->v, h->P, lr, beta1, beta2, eps, c1, c2);
    pack_weights(h);
    WK(h, cudaGetLastError());
    return SGTV_OK;
}

int wsnet_pack_input(const float *bp, int32_t Nx, int32_t Nz, int32_t Nq, float scale, float level, float *x_in,
                     void *stream)
{
    if (!bp || !x_in || Nx < 1 || Nz < 1 || Nq < 1 || !(scale > 0.f)) return SGTV_ERR_ARG;
    k_pack_input<<<blocks_for(int64_t(Nq + 1) * Nx * Nz), kT, 0, static_cast<cudaStream_t>(stream)>>>(
        bp, Nx, Nz, Nq, 1.f / scale, level, x_in);
    return cudaGetLastError() == cudaSuccess ? SGTV_OK : SGTV_ERR_CUDA;
}

int wsnet_unpack_output(const float *out, int32_t Nx, int32_t Nz, int32_t Nq, float scale, float *f, void *stream)
{
    if (!out || !f || Nx < 1 || Nz < 1 || Nq < 1) return SGTV_ERR_ARG;
    k_unpack_output<<<blocks_for(int64_t(Nq) * Nx * Nz), kT, 0, static_cast<cudaStream_t>(stream)>>>(out, Nx, Nz, Nq,
                                                                                                     scale, f);
    return cudaGetLastError() == cudaSuccess ? SGTV_OK : SGTV_ERR_CUDA;
}

int wsnet_unpack_dual(const float *out, int32_t Nx, int32_t Nz, int32_t Nq, int32_t n_dual, float tau, float *c,
                      void *stream)
{
    if (!out || !c || Nx < 1 || Nz < 1 || Nq < 1 || n_dual < 1 || n_dual > 4 || !(tau >= 0.f)) return SGTV_ERR_ARG;
    k_unpack_dual<<<blocks_for(int64_t(Nq) * Nx * Nz * n_dual), kT, 0, static_cast<cudaStream_t>(stream)>>>(
        out, Nx, Nz, Nq, n_dual, tau, c);
    return cudaGetLastError() == cudaSuccess ? SGTV_OK : SGTV_ERR_CUDA;
}

int32_t wsnet_num_outputs(wsnet_t h) { return h ? h->Co : 0; }

const char *wsnet_last_error(wsnet_t h) { return h ? h->err.c_str() : ""; }

}  // extern "C"

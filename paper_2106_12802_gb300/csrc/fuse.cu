// Fusion network of the multi-resolution sampling method (Sec. 4): I_SR from
// the LRHS render and the HRLS render + albedo / normal layers, plus the image
// metrics of Sec. 5 (sRGB PSNR via Eq. cvt_color, RelMSE) and the fallback gate
// of the hybrid renderer.
//
// Precisions: FP32 (SIMT direct convolution; reference precision), BF16
// (tcgen05 implicit GEMM, conv_tc.cu) and FP8-E4M3 (tcgen05 kind::f8f6f4 with
// per-output-channel weight scales and calibrated per-layer activation scales).
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <float.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <string>
#include <mutex>
#include <vector>

#include "conv_tc.cuh"
#include "fuse.cuh"

namespace mrs {
namespace {

constexpr int kLayers = 18;
constexpr int kFeat = 64;

struct LayerShape { int cin, cout; size_t woff, boff; };

// Layer shapes for a network whose first conv reads cin0 = 12 channels (the
// base input) or 21 (with the extra HRLS layers: diffuse, specular, variance)
const std::vector<LayerShape>& shapes(int cin0)
{
    static std::vector<LayerShape> v12, v21;
    std::vector<LayerShape>& v = cin0 == 21 ? v21 : v12;
    if (v.empty()) {
        size_t o = 0;
        for (int l = 0; l < kLayers; ++l) {
            int cin = l == 0 ? cin0 : kFeat, cout = l == kLayers - 1 ? 3 : kFeat;
            v.push_back({cin, cout, o, o + (size_t)cout * 9 * cin});
            o += (size_t)cout * 9 * cin + cout;
        }
    }
    return v;
}
constexpr size_t kParams12 = 599555;
constexpr size_t kParams21 = 604739;
constexpr int kCinMax = 21;

__host__ __device__ inline int nout_of(int l) { return l == kLayers - 1 ? 16 : 64; }

// ---- input assembly ---------------------------------------------------------
__device__ __forceinline__ void up_pixel(const float* __restrict__ lr, int h, int w, int s, int x,
                                         int y, float o[3])
{
    float inv = 1.0f / (float)s;
    float sy = fmaxf(((float)y + 0.5f) * inv - 0.5f, 0.0f);
    float sx = fmaxf(((float)x + 0.5f) * inv - 0.5f, 0.0f);
    int y0 = min((int)sy, h - 1), x0 = min((int)sx, w - 1);
    int y1 = min(y0 + 1, h - 1), x1 = min(x0 + 1, w - 1);
    float ly = sy - (float)y0, lx = sx - (float)x0;
    const float* a = lr + ((size_t)y0 * w + x0) * 3;
    const float* b = lr + ((size_t)y0 * w + x1) * 3;
    const float* c = lr + ((size_t)y1 * w + x0) * 3;
    const float* d = lr + ((size_t)y1 * w + x1) * 3;
    for (int k = 0; k < 3; ++k) {
        float top = __ldg(a + k) * (1.0f - lx) + __ldg(b + k) * lx;
        float bot = __ldg(c + k) * (1.0f - lx) + __ldg(d + k) * lx;
        o[k] = top * (1.0f - ly) + bot * ly;
    }
}

// Fusion-input channels of pixel p: up(LRHS), HRLS, albedo, normal (12) and,
// when extra != NULL (extra [P][9] = diffuse, specular, variance of the HRLS,
// Sec. 4), diffuse, specular and log(1 + max(variance, 0)) (21).  clip > 0:
// the radiance channels (up(LRHS), HRLS, diffuse, specular) are clipped at
// `clip` (the training data's firefly clipping, Sec. 3.2).  Returns the count.
__device__ __forceinline__ int input_px(const float* lrhs, const float* hrls, const float* alb,
                                        const float* nrm, const float* extra, int H, int W, int s,
                                        size_t p, float clip, float* v)
{
    int x = (int)(p % W);
    size_t r = p / W;
    int y = (int)(r % H), n = (int)(r / H);
    int h = H / s, w = W / s;
    up_pixel(lrhs + (size_t)n * h * w * 3, h, w, s, x, y, v);
    for (int k = 0; k < 3; ++k) {
        v[3 + k] = __ldg(hrls + 3 * p + k);
        v[6 + k] = __ldg(alb + 3 * p + k);
        v[9 + k] = __ldg(nrm + 3 * p + k);
    }
    if (clip > 0.0f)
        for (int k = 0; k < 6; ++k) v[k] = fminf(v[k], clip);
    if (!extra) return 12;
    for (int k = 0; k < 6; ++k) {
        float e = __ldg(extra + 9 * p + k);
        v[12 + k] = clip > 0.0f ? fminf(e, clip) : e;
    }
    for (int k = 0; k < 3; ++k) v[18 + k] = log1pf(fmaxf(__ldg(extra + 9 * p + 6 + k), 0.0f));
    return 21;
}

__global__ void k_input_f32(const float* lrhs, const float* hrls, const float* alb,
                            const float* nrm, const float* extra, int H, int W, int s, size_t P,
                            float* x0, float clip = 0.0f)
{
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P;
         p += (size_t)gridDim.x * blockDim.x) {
        float v[kCinMax];
        int c = input_px(lrhs, hrls, alb, nrm, extra, H, W, s, p, clip, v);
        for (int k = 0; k < c; ++k) x0[c * p + k] = v[k];
    }
}

// bf16 [P][64] or fp8 [P][64] scaled by inv_scale; channels past the input's
// 12 or 21 are zero (the first 24 bf16 / 32 fp8 channels are written from v,
// the rest as zero 16-byte words)
__global__ void k_input_q(const float* lrhs, const float* hrls, const float* alb,
                          const float* nrm, const float* extra, int H, int W, int s, size_t P,
                          void* x0, int fp8, float inv_scale, float clip = 0.0f)
{
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P;
         p += (size_t)gridDim.x * blockDim.x) {
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 0.0f;
        input_px(lrhs, hrls, alb, nrm, extra, H, W, s, p, clip, v);
        const uint4 z = make_uint4(0, 0, 0, 0);
        if (!fp8) {
            uint4* o = (uint4*)((__nv_bfloat16*)x0 + p * 64);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                uint4 u;
                __nv_bfloat162* h2 = (__nv_bfloat162*)&u;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    h2[e] = __floats2bfloat162_rn(v[8 * j + 2 * e], v[8 * j + 2 * e + 1]);
                o[j] = u;
            }
#pragma unroll
            for (int j = 3; j < 8; ++j) o[j] = z;
        } else {
            uint4* o = (uint4*)((uint8_t*)x0 + p * 64);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint4 u;
                uint8_t* b8 = (uint8_t*)&u;
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    b8[e] = (uint8_t)__nv_cvt_float_to_fp8(v[16 * j + e] * inv_scale, __NV_SATFINITE, __NV_E4M3);
                o[j] = u;
            }
            o[2] = z;
            o[3] = z;
        }
    }
}

// ---- FP32 SIMT direct convolution -------------------------------------------
// A block of 128 threads computes 8 OG output channels (OG = 8 or 2) of 32 x
// (32 / OG) pixels; a thread 8 consecutive pixels of one row x 8 channels, as
// packed pairs of channels (fma.rn.f32x2: each half rounds as fmaf does, so a
// value's chain over input channel, kernel row and column is that of one
// fmaf after another).  Input channels go through shared memory four at a time
// in two buffers: the weights by asynchronous copies from a packed layout
// ([c][tap][o], so that a thread's 8 are two 16-byte loads), the input through
// registers (one 16-byte load per pixel, stored channel by channel: neighbouring
// lanes store neighbouring words), both under way while the other buffer is
// used.  Per (channel, kernel row) a thread reads 3 + 6 16-byte words for 96
// packed FMAs; rows are 36 words apart, so a warp's input reads (4 pixel
// groups x 4 rows) take the two wavefronts that their bytes need.  What bounds
// it is the FMA pipe (a packed FMA holds it two cycles).  The form before (4
// pixels x 16 channels, scalar FMAs, 4-byte copies with the channel fastest)
// was bound by shared-memory wavefronts (86%), a third of them bank conflicts:
// the 21-channel network on 486 x 330 7.42 -> 3.75 ms (26 -> 52 TFLOP/s of the
// 80.5 of 152 SMs x 128 lanes), the 35 convolutions of its training step at 6 x
// 128^2 9.40 -> 5.05 ms.  Up to 16 outputs (the 3-channel heads; up to 32 on large
// images, see simt_conv3x3) run as two groups of 8 on four times the rows, so that the
// rest is not padding.
constexpr int kSC = 4;           // input channels per stage
constexpr int kSX = 32;          // pixels of a block along x
constexpr int kSPitch = 36;
__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// two FP32 values in one 64-bit register pair
typedef unsigned long long f2_t;
__device__ __forceinline__ f2_t f2_dup(float a)
{
    f2_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ f2_t f2_fma(f2_t a, f2_t b, f2_t c)
{
    f2_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ void f2_get(f2_t a, float& x, float& y)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
}

// packed weights wp[c][t][o] (c < ceil4(cin), o < cop, zero beyond cin / cout) of
// w [cout][9][cin], or, transposed, of the gradient conv's flipped taps: its
// inputs are w's outputs, wp[o][t][c] = w[o][8 - t][c]
__device__ __forceinline__ void pack_simt_body(const float* __restrict__ w, int cin, int cout, int transposed, int cop,
                                               float* __restrict__ wp)
{
    const int ci = transposed ? cout : cin, co = transposed ? cin : cout;
    const int n = ((ci + 3) & ~3) * 9 * cop;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int o = i % cop, t = (i / cop) % 9, c = i / (9 * cop);
        float v = 0.0f;
        if (c < ci && o < co)
            v = transposed ? w[((size_t)c * 9 + (8 - t)) * cin + o] : w[((size_t)o * 9 + t) * cin + c];
        wp[i] = v;
    }
}
__global__ void k_pack_simt(const float* __restrict__ w, int cin, int cout, int transposed, int cop,
                            float* __restrict__ wp)
{
    pack_simt_body(w, cin, cout, transposed, cop, wp);
}
// a network's layers, one to a blockIdx.y
__global__ void k_pack_simt_layers(const __grid_constant__ SimtLayers p)
{
    const SimtLayers::Layer& l = p.layer[blockIdx.y];
    pack_simt_body(l.w, l.cin, l.cout, 0, l.cop, l.wp);
}

// x [P][xs] (first cin channels read), out / res [P][os] / [P][rs] (first
// cout written / read): strides let a layer read a prefix of a concatenation
// buffer and write into a channel slice of another.  kVec: every pixel's
// channels start on a 16-byte boundary and come in fours
template <int OG, bool kVec>
__global__ void __launch_bounds__(128, 4)
    k_conv_simt(const float* __restrict__ x, int cin, int xs, const float* __restrict__ wp, int cop,
                const float* __restrict__ b, int cout, int mode, int relu,
                const float* __restrict__ res, int rs, float* __restrict__ out, int os,
                const float* __restrict__ lrhs, int H, int W, int s)
{
    constexpr int kRows = 32 / OG, kPx = (kRows + 2) * (kSX + 2), kNX = (kPx + 127) / 128;
    constexpr int kWChunks = kSC * 9 * OG * 2;
    __shared__ __align__(16) float sin_[2][kSC][kRows + 2][kSPitch];
    __shared__ __align__(16) float sw[2][kSC][9][OG * 8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gx = lane & 3, ty = ((lane & 15) >> 2) + (OG == 8 ? 0 : 4 * warp);
    const int og = (lane >> 4) + (OG == 8 ? 2 * warp : 0);
    // blocks along x, then y, in grid.x: grid.y would end at 65,535 rows of blocks
    const unsigned nbx = (unsigned)(W + kSX - 1) / kSX;
    const int x0 = (int)(blockIdx.x % nbx) * kSX, y0 = (int)(blockIdx.x / nbx) * kRows;
    const int ngrp = (cout + 8 * OG - 1) / (8 * OG);
    const int n = blockIdx.y / ngrp;
    const int o0 = (blockIdx.y % ngrp) * 8 * OG;
    const float* xin = x + (size_t)n * H * W * xs;
    float4 xr[kNX];
    // input channels c0 .. c0 + 3 of this thread's pixels of the tile
    auto fetch = [&](int c0) {
#pragma unroll
        for (int i = 0; i < kNX; ++i) {
            const int idx = threadIdx.x + 128 * i, px = idx % (kSX + 2), py = idx / (kSX + 2);
            const int ix = x0 + px - 1, iy = y0 + py - 1;
            xr[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (idx < kPx && ix >= 0 && ix < W && iy >= 0 && iy < H) {
                const float* q = xin + ((size_t)iy * W + ix) * xs + c0;
                if (kVec) {
                    xr[i] = __ldg((const float4*)q);
                } else {
                    if (c0 < cin) xr[i].x = __ldg(q);
                    if (c0 + 1 < cin) xr[i].y = __ldg(q + 1);
                    if (c0 + 2 < cin) xr[i].z = __ldg(q + 2);
                    if (c0 + 3 < cin) xr[i].w = __ldg(q + 3);
                }
            }
        }
    };
    auto put = [&](int q) {
#pragma unroll
        for (int i = 0; i < kNX; ++i) {
            const int idx = threadIdx.x + 128 * i, px = idx % (kSX + 2), py = idx / (kSX + 2);
            if (idx < kPx) {
                sin_[q][0][py][px] = xr[i].x;
                sin_[q][1][py][px] = xr[i].y;
                sin_[q][2][py][px] = xr[i].z;
                sin_[q][3][py][px] = xr[i].w;
            }
        }
    };
    auto weights = [&](int c0, int q) {
#pragma unroll
        for (int i = 0; i < (kWChunks + 127) / 128; ++i) {
            const int j = threadIdx.x + 128 * i, row = j / (OG * 2), col = 4 * (j % (OG * 2));
            if (j < kWChunks) cp_async16(&sw[q][0][0][0] + row * OG * 8 + col, wp + ((size_t)c0 * 9 + row) * cop + o0 + col);
        }
        cp_async_commit();
    };
    f2_t acc[8][4];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[p][o] = 0ull;
    const int nk = (cin + kSC - 1) / kSC;
    fetch(0);
    weights(0, 0);
    put(0);
    cp_async_wait_all();
    __syncthreads();
    for (int k = 0; k < nk; ++k) {
        const int q = k & 1;
        if (k + 1 < nk) {
            fetch((k + 1) * kSC);
            weights((k + 1) * kSC, q ^ 1);
        }
#pragma unroll 1
        for (int c = 0; c < kSC; ++c) {
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const float4* row = (const float4*)&sin_[q][c][ty + dy][gx * 8];
                const float4 r0 = row[0], r1 = row[1], r2 = row[2];
                const float in[10] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y};
                f2_t in2[10];
#pragma unroll
                for (int i = 0; i < 10; ++i) in2[i] = f2_dup(in[i]);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const ulonglong2* w2 = (const ulonglong2*)&sw[q][c][dy * 3 + dx][og * 8];
                    const ulonglong2 wa = w2[0], wb = w2[1];
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        acc[p][0] = f2_fma(in2[p + dx], wa.x, acc[p][0]);
                        acc[p][1] = f2_fma(in2[p + dx], wa.y, acc[p][1]);
                        acc[p][2] = f2_fma(in2[p + dx], wb.x, acc[p][2]);
                        acc[p][3] = f2_fma(in2[p + dx], wb.y, acc[p][3]);
                    }
                }
            }
        }
        if (k + 1 < nk) {
            put(q ^ 1);
            cp_async_wait_all();
        }
        // the next iteration reads what was stored here and its copies
        // overwrite the buffer read here
        __syncthreads();
    }
    const int gy = y0 + ty;
    if (gy >= H) return;
    const int ob = o0 + og * 8;
    if (ob >= cout) return;
    // 16-byte stores (and loads of res) where all 8 channels exist and are aligned
    const bool vec = ob + 8 <= cout && (os & 3) == 0 && ((uintptr_t)out & 15) == 0 &&
                     (!res || ((rs & 3) == 0 && ((uintptr_t)res & 15) == 0));
    float bias[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) bias[o] = ob + o < cout ? __ldg(b + ob + o) : 0.0f;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const int ix = x0 + gx * 8 + p;
        if (ix >= W) break;
        const size_t pp = ((size_t)n * H + gy) * W + ix;
        float v[8];
#pragma unroll
        for (int o = 0; o < 4; ++o) f2_get(acc[p][o], v[2 * o], v[2 * o + 1]);
        if (mode == SIMT_FINAL) {
            float up[3];
            const int h = H / s, wl = W / s;
            up_pixel(lrhs + (size_t)n * h * wl * 3, h, wl, s, ix, gy, up);
#pragma unroll
            for (int o = 0; o < 3; ++o)
                if (ob + o < 3) out[pp * 3 + ob + o] = (v[o] + bias[o]) + up[o];
            continue;
        }
        const float* rp = res + pp * rs + ob;
        float* op = out + pp * os + ob;
        float r[8];
        const bool reads = mode == SIMT_RESID || mode == SIMT_MASK || mode == SIMT_RESRELU;
        if (reads && vec) {
            const float4 ra = *(const float4*)rp, rb = *(const float4*)(rp + 4);
            r[0] = ra.x; r[1] = ra.y; r[2] = ra.z; r[3] = ra.w;
            r[4] = rb.x; r[5] = rb.y; r[6] = rb.z; r[7] = rb.w;
        } else if (reads) {
#pragma unroll
            for (int o = 0; o < 8; ++o) r[o] = ob + o < cout ? rp[o] : 0.0f;
        }
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            float t = v[o] + bias[o];
            if (mode == SIMT_RESID) t = r[o] + t;
            else if (mode == SIMT_MASK) t = r[o] > 0.0f ? t : 0.0f;
            else if (mode == SIMT_RESRELU) t = r[o] + fmaxf(t, 0.0f);
            else if (relu) t = fmaxf(t, 0.0f);
            v[o] = t;
        }
        if (vec) {
            *(float4*)op = make_float4(v[0], v[1], v[2], v[3]);
            *(float4*)(op + 4) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int o = 0; o < 8; ++o)
                if (ob + o < cout) op[o] = v[o];
        }
    }
}

}  // namespace

// channels of a packed row: whole groups of the kernel that runs `cout` outputs
static int simt_cop(int cout) { return cout > 16 ? (cout + 63) / 64 * 64 : 16; }
size_t simt_pack_floats(int cin, int cout) { return (size_t)((cin + 3) & ~3) * 9 * simt_cop(cout); }

mrs_status simt_pack(const float* w, int cin, int cout, int transposed, float* wp, cudaStream_t st)
{
    const int cop = simt_cop(transposed ? cin : cout);
    const size_t n = transposed ? simt_pack_floats(cout, cin) : simt_pack_floats(cin, cout);
    k_pack_simt<<<(int)std::min<size_t>((n + 255) / 256, 2048), 256, 0, st>>>(w, cin, cout, transposed, cop, wp);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "simt pack");
}

bool SimtLayers::add(const float* w, int cin, int cout, float* wp)
{
    if (n == kMax) { set_error("simt_pack_layers: too many layers"); return false; }
    layer[n++] = Layer{w, wp, cin, cout, simt_cop(cout)};
    largest = std::max(largest, simt_pack_floats(cin, cout));
    return true;
}

mrs_status simt_pack_layers(const SimtLayers& p, cudaStream_t st)
{
    k_pack_simt_layers<<<dim3((int)std::min<size_t>((p.largest + 255) / 256, 1024), p.n), 256, 0, st>>>(p);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "simt pack");
}

mrs_status simt_conv3x3(const float* x, int cin, int xs, const float* wp, const float* b, int cout,
                        int mode, int relu, const float* res, int rs, float* out, int os,
                        const float* lrhs, int N, int H, int W, int s, cudaStream_t st)
{
    const bool vec = (cin & 3) == 0 && (xs & 3) == 0 && ((uintptr_t)x & 15) == 0;
    // Groups of 16 outputs up to 16, and up to 32 where groups of 64, half of them
    // padding, would take more than a block an SM (a block of either takes as long, but
    // the higher tile's first stage takes longer): 64 -> 32 channels at 1024^2 1318 ->
    // 813 us, 144^2 (180 blocks) 102 -> 91, 128^2 (128 blocks) 79 as 64 and 91 as 16
    const int cop = simt_cop(cout);
    const long long blocks = (long long)((W + kSX - 1) / kSX) * ((H + 3) / 4) * N;
    const int og = cout > 32 || (cout > 16 && (blocks <= sm_count() || N > 32767)) ? 8 : 2, rows = 32 / og;   // grid.y
    const dim3 grid((unsigned)((W + kSX - 1) / kSX) * (unsigned)((H + rows - 1) / rows), N * ((cout + 8 * og - 1) / (8 * og)));
    auto launch = [&](auto kernel) {
        kernel<<<grid, 128, 0, st>>>(x, cin, xs, wp, cop, b, cout, mode, relu, res, rs, out, os, lrhs, H, W, s);
    };
    if (og == 8 && vec) MRS_TIMED(PK_CONV_SIMT, st, launch(k_conv_simt<8, true>));
    else if (og == 8) MRS_TIMED(PK_CONV_SIMT, st, launch(k_conv_simt<8, false>));
    else if (vec) MRS_TIMED(PK_CONV_SIMT, st, launch(k_conv_simt<2, true>));
    else MRS_TIMED(PK_CONV_SIMT, st, launch(k_conv_simt<2, false>));
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "conv_simt launch");
}

namespace {

mrs_status conv_simt(const float* x, int cin, const float* wp, const float* b, int cout, int mode,
                     int relu, const float* res, float* out, const float* lrhs, int N, int H,
                     int W, int s, cudaStream_t st)
{
    return simt_conv3x3(x, cin, cin, wp, b, cout, mode, relu, res, cout, out, cout, lrhs, N, H, W,
                        s, st);
}

// ---- weight packing ---------------------------------------------------------
// packed[tap][o][c] (o < nout, c < 64), zero padded; layer l at l * 9*64*64
__device__ __forceinline__ void pack_one_bf16(const float* __restrict__ master, size_t woff, size_t boff, int cin,
                                              int cout, int nout, __nv_bfloat16* __restrict__ wp,
                                              float* __restrict__ bp, int i)
{
    if (i < 64) bp[i] = i < cout ? master[boff + i] : 0.0f;
    if (i >= 9 * nout * 64) return;
    int c = i % 64, o = (i / 64) % nout, t = i / (64 * nout);
    float v = (o < cout && c < cin) ? master[woff + ((size_t)o * 9 + t) * cin + c] : 0.0f;
    wp[i] = __float2bfloat16_rn(v);
}
__global__ void k_pack_bf16(const float* __restrict__ master, size_t woff, size_t boff, int cin,
                            int cout, int nout, __nv_bfloat16* __restrict__ wp, float* __restrict__ bp)
{
    pack_one_bf16(master, woff, boff, cin, cout, nout, wp, bp, blockIdx.x * blockDim.x + threadIdx.x);
}
// a network's layers, for the kernels that pack them all in one launch (layer
// blockIdx.y): a training step repacks every layer, and a launch each (35 with
// the transposed ones) took 130 us of the fusion network's step, two take 6
struct PackLayers {
    long long woff[kLayers], boff[kLayers];
    int cin[kLayers], cout[kLayers];
};
PackLayers pack_layers(int cin0)
{
    const auto& L = shapes(cin0);
    PackLayers p;
    for (int l = 0; l < kLayers; ++l) {
        p.woff[l] = (long long)L[l].woff; p.boff[l] = (long long)L[l].boff;
        p.cin[l] = L[l].cin; p.cout[l] = L[l].cout;
    }
    return p;
}
__global__ void k_pack_layers_bf16(const float* __restrict__ master, const PackLayers p,
                                   __nv_bfloat16* __restrict__ wp, float* __restrict__ bp)
{
    const int l = blockIdx.y;
    pack_one_bf16(master, p.woff[l], p.boff[l], p.cin[l], p.cout[l], nout_of(l), wp + (size_t)l * 9 * 64 * 64,
                  bp + l * 64, blockIdx.x * blockDim.x + threadIdx.x);
}

// fp8: per-output-channel scale = amax / 448 over that channel's weights
__global__ void k_pack_fp8(const float* __restrict__ master, size_t woff, size_t boff, int cin,
                           int cout, int nout, uint8_t* __restrict__ wp, float* __restrict__ bp,
                           float* __restrict__ wscale)
{
    __shared__ float amax[64];
    int tid = threadIdx.x;
    if (tid < 64) {
        float m = 0.0f;
        if (tid < cout)
            for (int k = 0; k < 9 * cin; ++k) m = fmaxf(m, fabsf(master[woff + (size_t)tid * 9 * cin + k]));
        amax[tid] = m > 0.0f ? m / 448.0f : 1.0f;
        wscale[tid] = amax[tid];
        bp[tid] = tid < cout ? master[boff + tid] : 0.0f;
    }
    __syncthreads();
    for (int i = tid; i < 9 * nout * 64; i += blockDim.x) {
        int c = i % 64, o = (i / 64) % nout, t = i / (64 * nout);
        float v = (o < cout && c < cin) ? master[woff + ((size_t)o * 9 + t) * cin + c] / amax[o] : 0.0f;
        wp[i] = (uint8_t)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
    }
}

// amax of a bf16 [P][64] tensor (for fp8 activation calibration)
__global__ void k_amax_bf16(const __nv_bfloat16* __restrict__ x, size_t n, float* out)
{
    float m = 0.0f;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(__bfloat162float(x[i])));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax((int*)out, __float_as_int(m));
}

// ---- metrics ----------------------------------------------------------------
__device__ __forceinline__ double srgb(double l)
{
    if (l <= 0.0) return 0.0;
    if (l <= 0.0031308) return 12.92 * l;
    if (l < 1.0) return 1.055 * pow(l, 1.0 / 2.4) - 0.055;
    return 1.0;
}

constexpr int kRedBlocks = 1024;
static_assert(kRedBlocks == kLossParts, "loss partial sums");

__global__ void k_metrics_partial(const float* __restrict__ x, const float* __restrict__ ref,
                                  int64_t n, double l1, double l2, double* part)
{
    __shared__ double s[3][256];
    double a = 0, b = 0, c = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double xv = x[i], rv = ref[i];
        double d = srgb(xv) - srgb(rv);
        a += d * d;
        double e = xv - rv;
        b += l1 * e * e / (rv * rv + l2);
        c += e * e;
    }
    s[0][threadIdx.x] = a; s[1][threadIdx.x] = b; s[2][threadIdx.x] = c;
    __syncthreads();
    for (int w = 128; w; w >>= 1) {
        if (threadIdx.x < w)
            for (int k = 0; k < 3; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 3) part[blockIdx.x * 3 + threadIdx.x] = s[threadIdx.x][0];
}

// out[c] = sum over i of part[i k + c] (c < k <= 4), one block of 256
// threads: strided per-thread sums, then a fixed-order tree (deterministic)
__global__ void k_reduce_parts(const double* part, int nparts, int k, double* out)
{
    __shared__ double sh[4][256];
    for (int c = 0; c < k; ++c) {
        double acc = 0;
        for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[i * k + c];
        sh[c][threadIdx.x] = acc;
    }
    __syncthreads();
    for (int w = 128; w; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < k; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < k) out[threadIdx.x] = sh[threadIdx.x][0];
}

// per LR pixel: RelMSE terms of box_s(fused) vs LRHS
__global__ void k_gate_partial(const float* __restrict__ fused, const float* __restrict__ lrhs,
                               int N, int H, int W, int s, double* part)
{
    __shared__ double sh[256];
    int h = H / s, w = W / s;
    int64_t nlr = (int64_t)N * h * w;
    double acc = 0;
    double inv = 1.0 / ((double)s * s);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlr;
         i += (int64_t)gridDim.x * blockDim.x) {
        int xl = (int)(i % w);
        int64_t r = i / w;
        int yl = (int)(r % h), n = (int)(r / h);
        for (int c = 0; c < 3; ++c) {
            double m = 0;
            for (int dy = 0; dy < s; ++dy)
                for (int dx = 0; dx < s; ++dx)
                    m += fused[(((int64_t)n * H + yl * s + dy) * W + xl * s + dx) * 3 + c];
            m *= inv;
            double ref = lrhs[i * 3 + c];
            double e = m - ref;
            acc += 0.5 * e * e / (ref * ref + 0.01);
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int k = 128; k; k >>= 1) {
        if (threadIdx.x < k) sh[threadIdx.x] += sh[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// bf16 [P][64] rows of input channels c0 .. c0 + 63 of x [P][cin] (zero past cin)
__global__ void k_to_operand_chunk(const float* x, size_t P, int cin, int c0, __nv_bfloat16* o)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < P * 64;
         i += (size_t)gridDim.x * blockDim.x) {
        size_t p = i / 64;
        int c = c0 + (int)(i % 64);
        o[i] = __float2bfloat16_rn(c < cin ? x[p * cin + c] : 0.0f);
    }
}

// packed[tap][o][c] of input channels c0 .. c0 + 63 of w [cout][3][3][cin]
__global__ void k_pack_bf16_chunk(const float* __restrict__ w, int cin, int c0, int cout, int nout,
                                  __nv_bfloat16* __restrict__ wp)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 9 * nout * 64) return;
    int c = i % 64, o = (i / 64) % nout, t = i / (64 * nout);
    float v = (o < cout && c0 + c < cin) ? w[((size_t)o * 9 + t) * cin + c0 + c] : 0.0f;
    wp[i] = __float2bfloat16_rn(v);
}

// 8 channels a thread, stored at once: bound by the operand's bytes
__global__ void k_to_operand(const float* x, size_t P, int cin, void* o, int fp8, float inv)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < P * 8;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t p = i / 8;
        const int c0 = (int)(i % 8) * 8;
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = c0 + k < cin ? x[p * cin + c0 + k] : 0.0f;
        if (fp8) {
            uint2 u;
            uint8_t* b = (uint8_t*)&u;
#pragma unroll
            for (int k = 0; k < 8; ++k) b[k] = (uint8_t)__nv_cvt_float_to_fp8(v[k] * inv, __NV_SATFINITE, __NV_E4M3);
            ((uint2*)o)[i] = u;
        } else {
            uint4 u;
            __nv_bfloat16* b = (__nv_bfloat16*)&u;
#pragma unroll
            for (int k = 0; k < 8; ++k) b[k] = __float2bfloat16_rn(v[k]);
            ((uint4*)o)[i] = u;
        }
    }
}

__global__ void k_amax_f32(const float* __restrict__ x, size_t n, float* out)
{
    float m = 0.0f;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(x[i]));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax((int*)out, __float_as_int(m));
}

// ---- training kernels (FP32) -----------------------------------------------
// dW[o][t][c] = sum_p dy[p][o] * x[p shifted by tap t][c] (zero padded), db[o] = sum_p dy[p][o]
// grid (G, ntaps, otiles * ctiles): block (g, j, z) reduces pixel tiles g, g+G, ... for tap
// t = t0 + j of the 64 x 64 channel tile z = (output tile ot, input tile ct) into
// part[z][g][j][o][c] (each z a [G][ntaps][64 * 64] slab holding the tile's cout_t x cin_t
// values packed) and, for ct = 0 and j = 0, db into dbpart[ot][g][o] (a [G * 64] slab per
// ot, cout_t values per g packed)
// A block of 64 threads; a thread 8 outputs x 8 inputs as packed pairs (a
// value's chain over pixels is one FMA after another, in pixel order).  Half a
// tile of pixels at a time is copied to shared memory as it lies (16 bytes a
// copy where the channels allow), the next half under way meanwhile.  A
// thread's channels are 4 g .. 4 g + 3 and 32 + 4 g .. 35 + 4 g, so that its
// 16-byte reads are next to its neighbours': per pixel 4 of them for 32 packed
// FMAs, which bound the kernel.  (4 x 4 scalar values a thread and 4-byte
// copies through registers were bound by issue slots, 71% used, at 45% of the FMA
// pipe: 18 layers at 6 x 128^2 and their reductions took 8.97 ms, now 3.37.)
constexpr int kDwTile = 64;      // consecutive pixels of one split
constexpr int kDwHalf = 32;      // ... of a stage
template <bool kVec>
__device__ __forceinline__ void dw_copy(float (*dst)[64], const float* __restrict__ src, int ch, int n, long long row,
                                        bool ok, int px)
{
    // channels ch .. ch + 3 of a pixel (zeros where !ok)
    const float* q = src + (ok ? row : 0);
    if (kVec) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&dst[px][ch])),
                     "l"(ok ? q + ch : src), "r"(ok ? 16 : 0)
                     : "memory");
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&dst[px][ch + e])),
                         "l"(ok && ch + e < n ? q + ch + e : src), "r"(ok && ch + e < n ? 4 : 0)
                         : "memory");
    }
}

// x [P][xs] (first cin channels used), dy [P][ys] (first cout used); I indexes pixels
template <bool kVecX, bool kVecY, typename I>
__global__ void __launch_bounds__(64, 6)
    k_dw_partial(const float* __restrict__ x, int cin, int xs, const float* __restrict__ dy, int cout,
                 int ys, int N, int H, int W, float* __restrict__ part, float* __restrict__ dbpart,
                 int t0, int ctiles)
{
    __shared__ __align__(16) float sdy[2][kDwHalf][64];
    __shared__ __align__(16) float sx[2][kDwHalf][64];
    const int j = blockIdx.y, t = t0 + j, g = blockIdx.x, G = gridDim.x;
    const int ot = blockIdx.z / ctiles, ct = blockIdx.z % ctiles;
    x += 64 * ct;
    dy += 64 * ot;
    cin = min(64, cin - 64 * ct);
    cout = min(64, cout - 64 * ot);
    const bool do_db = j == 0 && ct == 0;
    const int dyo = t / 3 - 1, dxo = t % 3 - 1;
    const int og = threadIdx.x >> 3, cg = threadIdx.x & 7;
    const I P = (I)N * H * W, ntiles = (P + kDwTile - 1) / kDwTile;
    const I mine = g < ntiles ? (ntiles - g + G - 1) / G : 0;       // tiles g, g + G, ...
    const int off = dyo * W + dxo;
    // stage k: half k & 1 of this split's tile k >> 1
    auto stage = [&](I k, int q) {
        const int ch = (threadIdx.x & 15) * 4;
        int px = threadIdx.x >> 4;
        I p = (g + (k >> 1) * G) * kDwTile + (int)(k & 1) * kDwHalf + px;
        int xx = (int)(p % W), yy = (int)((p / W) % H);
#pragma unroll
        for (int i = 0; i < kDwHalf / 4; ++i) {
            const bool in = p < P;
            const bool ok = in && xx + dxo >= 0 && xx + dxo < W && yy + dyo >= 0 && yy + dyo < H;
            dw_copy<kVecY>(sdy[q], dy, ch, cout, (long long)p * ys, in && (!kVecY || ch < cout), px);
            dw_copy<kVecX>(sx[q], x, ch, cin, (long long)(p + off) * xs, ok && (!kVecX || ch < cin), px);
            px += 4;
            p += 4;
            xx += 4;
            while (xx >= W) { xx -= W; yy = yy + 1 == H ? 0 : yy + 1; }
        }
        cp_async_commit();
    };
    f2_t acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][k] = 0ull;
    float dbacc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const I stages = 2 * mine;
    if (stages) stage(0, 0);
    for (I k = 0; k < stages; ++k) {
        const int q = (int)(k & 1);
        cp_async_wait_all();
        // what the other buffer held has been read, what this one holds has landed
        __syncthreads();
        if (k + 1 < stages) stage(k + 1, q ^ 1);
#pragma unroll 2
        for (int px = 0; px < kDwHalf; ++px) {
            const float4 a0 = *(const float4*)&sdy[q][px][og * 4], a1 = *(const float4*)&sdy[q][px][32 + og * 4];
            const ulonglong2 b0 = *(const ulonglong2*)&sx[q][px][cg * 4], b1 = *(const ulonglong2*)&sx[q][px][32 + cg * 4];
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const f2_t a2 = f2_dup(av[i]);
                acc[i][0] = f2_fma(a2, b0.x, acc[i][0]);
                acc[i][1] = f2_fma(a2, b0.y, acc[i][1]);
                acc[i][2] = f2_fma(a2, b1.x, acc[i][2]);
                acc[i][3] = f2_fma(a2, b1.y, acc[i][3]);
            }
            if (do_db)
#pragma unroll
                for (int i = 0; i < 8; ++i) dbacc[i] += av[i];
        }
    }
    float* out = part + (size_t)blockIdx.z * G * gridDim.y * 4096 + ((size_t)g * gridDim.y + j) * cout * cin;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int o = (i < 4 ? 0 : 28) + og * 4 + i;
        if (o >= cout) continue;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = (k < 2 ? 0 : 28) + cg * 4 + 2 * k;
            float v0, v1;
            f2_get(acc[i][k], v0, v1);
            if (c < cin) out[(size_t)o * cin + c] = v0;
            if (c + 1 < cin) out[(size_t)o * cin + c + 1] = v1;
        }
        if (do_db && cg == 0) dbpart[(size_t)ot * G * 64 + (size_t)g * cout + o] = dbacc[i];
    }
}

// grid (G, ntaps, tiles): see k_dw_partial
void launch_dw(dim3 grid, const float* x, int cin, int xs, const float* dy, int cout, int ys, int N, int H, int W,
               float* part, float* dbpart, int t0, int ctiles, cudaStream_t st)
{
    auto four = [](const float* p, int n, int stride) { return n % 4 == 0 && stride % 4 == 0 && ((uintptr_t)p & 15) == 0; };
    const bool vx = four(x, cin, xs), vy = four(dy, cout, ys);
    auto go = [&](auto kernel) {
        kernel<<<grid, 64, 0, st>>>(x, cin, xs, dy, cout, ys, N, H, W, part, dbpart, t0, ctiles);
    };
    if ((long long)N * H * W > (1 << 30)) go(k_dw_partial<false, false, long long>);
    else if (vx && vy) go(k_dw_partial<true, true, int>);
    else if (vx) go(k_dw_partial<true, false, int>);
    else if (vy) go(k_dw_partial<false, true, int>);
    else go(k_dw_partial<false, false, int>);
}

// grad[o][t][c] (params layout) = sum_g part[g][t][o][c]; grad_b[o] = sum_g dbpart[g][o]
// (partials gstride floats apart, bias partials bstride).
// A block takes 32 consecutive values; warp w sums partials w, w + 8, ... (one
// coalesced 128-byte row per partial) and the eight sums are added in warp
// order: a fixed order, so the result is deterministic.
__global__ void __launch_bounds__(256) k_dw_reduce(const float* __restrict__ part,
                                                   const float* __restrict__ dbpart, int G,
                                                   size_t gstride, int bstride, int cin, int cout,
                                                   float* __restrict__ gw, float* __restrict__ gb)
{
    __shared__ float red[8][32];
    const int nw = cout * 9 * cin, ntot = nw + cout;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    for (int e0 = blockIdx.x * 32; e0 < ntot; e0 += gridDim.x * 32) {
        const int e = e0 + lane;
        float acc = 0.0f;
        if (e < nw) {
            const int c = e % cin, t = (e / cin) % 9, o = e / (cin * 9);
            const float* src = part + ((size_t)t * cout + o) * cin + c;
            for (int g = wp; g < G; g += 8) acc += src[(size_t)g * gstride];
        } else if (e < ntot) {
            const int o = e - nw;
            for (int g = wp; g < G; g += 8) acc += dbpart[(size_t)g * bstride + o];
        }
        red[wp][lane] = acc;
        __syncthreads();
        if (wp == 0 && e < ntot) {
            float v = red[0][lane];
            for (int k = 1; k < 8; ++k) v += red[k][lane];
            if (e < nw) gw[e] = v;
            else gb[e - nw] = v;
        }
        __syncthreads();
    }
}

// Every tile's partial sums into the gradient (see WgRed): one thread per
// value, reads coalesced along the input channels.
__device__ __forceinline__ float sum_parts(const float* __restrict__ src, size_t stride, int np)
{
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = i < np ? src[i * stride] : 0.0f;
    float acc = v[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) acc += v[i];
    return acc;
}
__global__ void __launch_bounds__(256) k_wg_reduce(const WgRed* __restrict__ reds, const float* __restrict__ part,
                                                   const float* __restrict__ dbpart, float* __restrict__ grad)
{
    const int t = blockIdx.y;
    const WgRed r = reds[t];
    const int nw = r.cout * r.KK * r.cin, e = blockIdx.x * 256 + threadIdx.x;
    if (e < nw) {
        const int c = e % r.cin, tl = (e / r.cin) % r.KK, o = e / (r.cin * r.KK);
        const float acc = sum_parts(part + (size_t)8 * t * kWgPart +
                                        ((size_t)(r.KK == 9 ? tl : 4) * r.cout + o) * r.cin + c, kWgPart, r.np);
        const int ci = r.q > 0 ? 64 + dsf_channel(c, (r.q - 1) / r.s, (r.q - 1) % r.s, r.D) : r.c0 + c;
        grad[r.gw + ((long long)(r.o_mul * o + r.o_add) * r.KK + tl) * r.CIN + ci] = acc;
    } else if (e - nw < r.cout && r.with_bias) {
        const int o = e - nw;
        grad[r.gb + r.o_mul * o + r.o_add] = sum_parts(dbpart + (size_t)8 * t * 64 + o, 64, r.np);
    }
}

// Training losses, reduced in float64 per block; dy receives dL/dy.
//   MRS_LOSS_L1LOG: L1 on slog(x) = sign(x) log1p(|x|) (= log(1 + x) for
//     x >= 0): d = slog(y) - slog(min(t, clip)); dy = sign(d) / (1 + |y|) / n
//   MRS_LOSS_ROBUST: the robust loss l_r of Sec. 3, e = y - min(t, clip),
//     |e| / (beta + |e|) per value; dy = sign(e) beta / (beta + |e|)^2 / n
__device__ __forceinline__ double slog(double x) { return x < 0.0 ? -log1p(-x) : log1p(x); }

// moves v's binary exponent (v >= 1) into e
__device__ __forceinline__ void take_exponent(double& v, int& e)
{
    const int h = __double2hiint(v);
    e += (h >> 20) - 1023;
    v = __hiloint2double((h & 0xfffff) | 0x3ff00000, __double2loint(v));
}

// log1p(x), 0 <= x < 2^-10, to a relative 2^-62
__device__ __forceinline__ double log1p_small(double x)
{
    return x * (1.0 - x * (0.5 - x * (1.0 / 3.0 - x * (0.25 - x * (0.2 - x * (1.0 / 6.0))))));
}

// L1-log is bound by the float64 units (2 lanes a clock per SM): two log1p a
// value were 164 float64 operations.  A block sums |slog(y) - slog(t)| as the
// logarithm of a quotient instead: num collects 1 + the larger magnitude and
// den 1 + the smaller one (num both, where the signs differ), their exponents
// are counted in integers, and one logarithm of each is taken per block.  1 + |x|
// is exact for a float |x| >= 2^-29, and a product's rounding, 2^-53 of the sum
// whatever the value, does not show beside a logarithm of 2^-10 and more; below
// that a series keeps the relative precision.  Equal values add nothing, so that
// the loss of an image against itself is 0.  slog is strictly increasing on floats,
// so the gradient's sign is the values' own order.  1.77 M values: 460 -> 47 us,
// 0.79 M: 189 -> 34 us.
__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ tgt, size_t n,
                       float clip, int kind, float beta, float* __restrict__ dy,
                       double* __restrict__ part)
{
    __shared__ double sh[256], sn[256], sd[256];
    __shared__ int se[256];
    double acc = 0.0, num = 1.0, den = 1.0;
    int ex = 0;                                  // exponent of num / den
    const float inv_n = 1.0f / (float)n;
    const double b = (double)beta, dinv_n = 1.0 / (double)n;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        float yp = y[i];
        float tv = clip > 0.0f ? fminf(tgt[i], clip) : tgt[i];
        float g = 0.0f;
        if (kind == MRS_LOSS_ROBUST) {
            double e = (double)yp - (double)tv, a = fabs(e);
            acc += a / (b + a);
            if (e != 0.0) g = (float)((e > 0.0 ? b : -b) / ((b + a) * (b + a)) * dinv_n);
        } else {
            const float ay = fabsf(yp), at = fabsf(tv);
            bool differ = yp != tv, above = yp > tv;
            if (!(ay <= FLT_MAX && at <= FLT_MAX)) {
                const double d = slog((double)yp) - slog((double)tv);
                acc += fabs(d);
                differ = d != 0.0;
                above = d > 0.0;
            } else if (differ) {
                const double hi = (double)fmaxf(ay, at), lo = (double)fminf(ay, at);
                const bool same = (__float_as_int(yp) ^ __float_as_int(tv)) >= 0;
                if (hi < 0x1p-10) {
                    const double l = log1p_small(lo);
                    acc += log1p_small(hi) + (same ? -l : l);
                } else {
                    num *= 1.0 + hi;
                    if (same) den *= 1.0 + lo;
                    else num *= 1.0 + lo;
                    int de = 0;
                    take_exponent(num, ex);
                    take_exponent(den, de);
                    ex -= de;
                }
            }
            if (differ) g = (above ? 1.0f : -1.0f) / (1.0f + ay) * inv_n;
        }
        dy[i] = g;
    }
    sh[threadIdx.x] = acc;
    sn[threadIdx.x] = num;
    sd[threadIdx.x] = den;
    se[threadIdx.x] = ex;
    __syncthreads();
    for (int w = 128; w; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (kind != MRS_LOSS_ROBUST && threadIdx.x < 32) {
        int de = 0;
        for (int k = threadIdx.x + 32; k < 256; k += 32) {
            num *= sn[k];
            den *= sd[k];
            ex += se[k];
            take_exponent(num, ex);
            take_exponent(den, de);
        }
        for (int w = 16; w; w >>= 1) {
            num *= __shfl_xor_sync(0xffffffffu, num, w);
            den *= __shfl_xor_sync(0xffffffffu, den, w);
        }                                        // below 2^32
        for (int w = 16; w; w >>= 1) {
            ex += __shfl_xor_sync(0xffffffffu, ex, w);
            de += __shfl_xor_sync(0xffffffffu, de, w);
        }
        if (threadIdx.x == 0) sh[0] += (double)(ex - de) * 0.693147180559945309 + (log(num) - log(den));
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_mask_inplace(float* __restrict__ d, const float* __restrict__ act, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        if (!(act[i] > 0.0f)) d[i] = 0.0f;
}

// bias-corrected Adam (Kingma & Ba): bc1 = 1 - beta1^t, bc2 = 1 - beta2^t
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps,
                       float bc1, float bc2)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        float gi = g[i];
        float mi = b1 * m[i] + (1.0f - b1) * gi;
        float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        float mh = mi / bc1, vh = vi / bc2;
        p[i] = p[i] - lr * mh / (sqrtf(vh) + eps);
    }
}

}  // namespace

// ---- training launches shared with the method's own network (rdn.cu) -------
mrs_status dw_tiles_f32(const float* x, int cin, int xs, const float* dy, int cout, int ys, int N,
                        int H, int W, int centre_only, float* part, float* dbpart, cudaStream_t st)
{
    const int ctiles = (cin + 63) / 64, otiles = (cout + 63) / 64;
    dim3 grid(kDwParts, centre_only ? 1 : 9, otiles * ctiles);
    launch_dw(grid, x, cin, xs, dy, cout, ys, N, H, W, part, dbpart, centre_only ? 4 : 0, ctiles, st);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "dw tiles");
}

mrs_status wg_reduce(const WgRed* d_reds, int ntiles, const float* part, const float* dbpart, float* grad,
                     cudaStream_t st)
{
    const dim3 grid((kWgPart + 64 + 255) / 256, ntiles);
    MRS_TIMED(PK_TRAIN, st, k_wg_reduce<<<grid, 256, 0, st>>>(d_reds, part, dbpart, grad));
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "wgrad reduce");
}

mrs_status loss_grad_f32(const float* y, const float* tgt, size_t n, float clip, int kind,
                         float beta, float* dy, double* parts, double* sum, cudaStream_t st)
{
    k_loss<<<kRedBlocks, 256, 0, st>>>(y, tgt, n, clip, kind, beta, dy, parts);
    MRS_LAUNCHED(1);
    k_reduce_parts<<<1, 256, 0, st>>>(parts, kRedBlocks, 1, sum);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "loss");
}

mrs_status adam_f32(float* p, const float* g, float* m, float* v, size_t n, float lr, int64_t step,
                    cudaStream_t st)
{
    const double b1 = 0.9, b2 = 0.999;
    float bc1 = (float)(1.0 - pow(b1, (double)step));
    float bc2 = (float)(1.0 - pow(b2, (double)step));
    size_t gsz = (n + 255) / 256;
    k_adam<<<(int)(gsz < 4096 ? (gsz ? gsz : 1) : 4096), 256, 0, st>>>(p, g, m, v, n, lr, (float)b1,
                                                                     (float)b2, 1e-8f, bc1, bc2);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "adam");
}

namespace {

// gate decision on the device: D = sum / count; use_plain = D > tau
__global__ void k_gate_decide(const double* part, int nparts, double count, double tau,
                              int use_plain_avail, int* used_plain, double* D)
{
    // the same fixed-order reduction as k_reduce_parts
    __shared__ double sh[256];
    double a = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) a += part[i];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double acc = sh[0];
        double d = acc / count;
        if (D) *D = d;
        int u = d > tau ? 1 : 0;
        used_plain[0] = u;
        used_plain[1] = u && use_plain_avail;     // whether `out` takes the plain render
    }
}

// out = plain if the gate chose it (and a plain render was given), else fused
__global__ void k_gate_select(const float* __restrict__ fused, const float* __restrict__ plain,
                              size_t n, const int* __restrict__ choice, float* __restrict__ out)
{
    const float* src = choice[1] != 0 ? plain : fused;
    if (src == out) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = src[i];
}

// transposed, tap-flipped weights of layer (cin, cout) packed as the
// tensor-core operand of dX = conv(dY): wp[t][c][o] = w[o][8 - t][c]
// (rows c < cin of nout, columns o < cout of 64, zero padded)
__device__ __forceinline__ void pack_one_bf16_T(const float* __restrict__ master, size_t woff, int cin, int cout,
                                                int nout, __nv_bfloat16* __restrict__ wp, int i)
{
    if (i >= 9 * nout * 64) return;
    int o = i % 64, c = (i / 64) % nout, t = i / (64 * nout);
    float v = (c < cin && o < cout) ? master[woff + ((size_t)o * 9 + (8 - t)) * cin + c] : 0.0f;
    wp[i] = __float2bfloat16_rn(v);
}
__global__ void k_pack_bf16_T(const float* __restrict__ master, size_t woff, int cin, int cout,
                              int nout, __nv_bfloat16* __restrict__ wp)
{
    pack_one_bf16_T(master, woff, cin, cout, nout, wp, blockIdx.x * blockDim.x + threadIdx.x);
}
// layers 1 .. of a network, one to a blockIdx.y
__global__ void k_pack_layers_bf16_T(const float* __restrict__ master, const PackLayers p,
                                     __nv_bfloat16* __restrict__ wp)
{
    const int l = 1 + blockIdx.y;
    pack_one_bf16_T(master, p.woff[l], p.cin[l], p.cout[l], 64, wp + (size_t)l * 9 * 64 * 64,
                    blockIdx.x * blockDim.x + threadIdx.x);
}

// out[p][c] = float(o[p][c]) for c < cin from bf16 [P][64] rows
__global__ void k_from_operand(const __nv_bfloat16* __restrict__ o, size_t P, int cin,
                               float* __restrict__ out)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < P * cin;
         i += (size_t)gridDim.x * blockDim.x) {
        size_t p = i / cin;
        int c = (int)(i % cin);
        out[i] = __bfloat162float(o[p * 64 + c]);
    }
}

struct Scratch {
    std::mutex mu;
    Buf b;
};
Scratch& scratch()
{
    static Scratch s;
    return s;
}

}  // namespace
}  // namespace mrs

namespace mrs {
// What a BF16 training step of one shape needs besides its data: the tensor
// maps of its activations (all inside the handle's workspace) and the
// weight-gradient tiles.  A handle keeps those of its last kStepPlans shapes
// (batches of two shapes in turn then build, allocate and upload nothing), and
// those that a recorded step reads, which are neither changed nor freed before
// the handle is.
constexpr int kStepPlans = 8;
struct StepPlan {
    int N = -1, H = -1, W = -1;
    void* act = nullptr;
    CUtensorMap x0A, dybA, hA[9], hO[9], rA[8], rO[8], dhA[9], dhO[9], daA[8], daO[8];
    WgPlan wg;
    std::vector<uint8_t> image;    // wg.blob, then the tiles' WgRed
    Buf blob;                      // ... on the device
    const WgRed* reds = nullptr;
    bool uploaded = false;         // by a step that ran (a recorded step's upload is recorded with it)
    bool recorded = false;
    uint64_t used = 0;             // the handle's plan_clock at its last step
    ~StepPlan() { blob.release(); }
};
}  // namespace mrs

using namespace mrs;

struct mrs_net_s {
    int cin0 = 12;                 // input channels of the first conv (12 or 21)
    size_t np = kParams12;         // parameter count
    Buf block;                     // holds the arrays below
    float* master = nullptr;       // [np]
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    float* grad = nullptr;
    int64_t step = 0;
    __nv_bfloat16* wbf = nullptr;  // [18][9][64][64]
    uint8_t* wf8 = nullptr;        // [18][9][64][64]
    float* bias = nullptr;         // [18][64]
    float* bias8 = nullptr;        // [18][64]
    float* wscale = nullptr;       // [18][64]
    bool bf_valid = false, f8_valid = false;
    float xscale[kLayers];         // fp8 activation scales (calibrated)
    bool xscale_valid = false;
    CUtensorMap wmap_bf[kLayers], wmap_f8[kLayers], wmap_bfT[kLayers];
    __nv_bfloat16* wbfT = nullptr; // [18][9][64][64] transposed, tap-flipped (backward)
    bool bfT_valid = false;
    float* wsimt = nullptr;        // FP32 weights as the SIMT conv reads them, layer after layer
    // wsimt holds master's values.  A call that is being recorded packs whatever
    // this says, so that its replays follow the weights; once a training step was
    // recorded, whose replays change them unseen, every call packs
    bool simt_valid = false, step_recorded = false;
    Buf act;                       // activation workspace
    Buf aux;                       // small device scratch
    Buf tact;                      // training activations
    Buf ttmp;                      // training scratch (transposed weights, dW partials, loss)
    int* err = nullptr;            // device error word
    std::vector<std::unique_ptr<mrs::StepPlan>> plans;   // of BF16 steps
    uint64_t plan_clock = 0;
    int loss_kind = MRS_LOSS_L1LOG;
    float loss_beta = 0.1f;
};

namespace mrs {
namespace {

mrs_status pack_bf16(mrs_net_s* net, cudaStream_t st)
{
    if (net->bf_valid) return MRS_OK;
    k_pack_layers_bf16<<<dim3(9 * 64 * 64 / 256, kLayers), 256, 0, st>>>(net->master, pack_layers(net->cin0), net->wbf,
                                                                         net->bias);
    MRS_LAUNCHED(1);
    for (int l = 0; l < kLayers; ++l) {
        int nout = nout_of(l);
        mrs_status s = tc_make_w_map(&net->wmap_bf[l], net->wbf + (size_t)l * 9 * 64 * 64, 9 * nout, nout, TC_BF16);
        if (s != MRS_OK) return s;
    }
    net->bf_valid = true;
    return cuda_status(cudaGetLastError(), "pack bf16");
}

mrs_status pack_fp8(mrs_net_s* net, cudaStream_t st)
{
    if (net->f8_valid) return MRS_OK;
    const auto& L = shapes(net->cin0);
    for (int l = 0; l < kLayers; ++l) {
        int nout = nout_of(l);
        k_pack_fp8<<<1, 256, 0, st>>>(net->master, L[l].woff, L[l].boff, L[l].cin, L[l].cout, nout,
                                      net->wf8 + (size_t)l * 9 * 64 * 64, net->bias8 + l * 64,
                                      net->wscale + l * 64);
        MRS_LAUNCHED(1);
        mrs_status s = tc_make_w_map(&net->wmap_f8[l], net->wf8 + (size_t)l * 9 * 64 * 64, 9 * nout, nout, TC_FP8);
        if (s != MRS_OK) return s;
    }
    net->f8_valid = true;
    return cuda_status(cudaGetLastError(), "pack fp8");
}

// packed FP32 weights of layer l (after pack_simt)
size_t simt_off(mrs_net_s* net, int l) { return l ? simt_pack_floats(net->cin0, 64) + (size_t)(l - 1) * simt_pack_floats(64, 64) : 0; }
const float* wsimt(mrs_net_s* net, int l) { return net->wsimt + simt_off(net, l); }
mrs_status pack_simt(mrs_net_s* net, cudaStream_t st)
{
    const bool rec = recording(st);
    if (net->simt_valid && !rec) return MRS_OK;
    const auto& L = shapes(net->cin0);
    SimtLayers p;
    for (int l = 0; l < kLayers; ++l)
        if (!p.add(net->master + L[l].woff, L[l].cin, L[l].cout, net->wsimt + simt_off(net, l))) return MRS_ERR_ARG;
    const mrs_status rc = simt_pack_layers(p, st);
    if (!rec) net->simt_valid = rc == MRS_OK && !net->step_recorded;
    return rc;
}

mrs_status fuse_f32(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                    const float* nrm, const float* extra, int N, int H, int W, int s, float* out,
                    cudaStream_t st)
{
    size_t P = (size_t)N * H * W;
    const int c0 = net->cin0;
    mrs_status rc = net->act.ensure(P * (c0 + 64 + 64) * 4 + 16);
    if (rc != MRS_OK) return rc;
    if ((rc = pack_simt(net, st)) != MRS_OK) return rc;
    float* x0 = net->act.as<float>();
    float* h = x0 + ((P * c0 + 3) & ~(size_t)3);     // 16-byte aligned
    float* r = h + P * 64;
    const auto& L = shapes(net->cin0);
    k_input_f32<<<(int)((P + 255) / 256 < 65535 ? (P + 255) / 256 : 65535), 256, 0, st>>>(
        lrhs, hrls, alb, nrm, extra, H, W, s, P, x0);
    MRS_LAUNCHED(1);
    rc = conv_simt(x0, c0, wsimt(net, 0), net->master + L[0].boff, 64, SIMT_PLAIN, 1,
                   nullptr, h, nullptr, N, H, W, s, st);
    for (int k = 0; k < 8 && rc == MRS_OK; ++k) {
        const LayerShape& a = L[1 + 2 * k];
        const LayerShape& b = L[2 + 2 * k];
        rc = conv_simt(h, 64, wsimt(net, 1 + 2 * k), net->master + a.boff, 64, SIMT_PLAIN, 1,
                       nullptr, r, nullptr, N, H, W, s, st);
        if (rc == MRS_OK)
            rc = conv_simt(r, 64, wsimt(net, 2 + 2 * k), net->master + b.boff, 64, SIMT_RESID, 0, h,
                           h, nullptr, N, H, W, s, st);
    }
    if (rc == MRS_OK)
        rc = conv_simt(h, 64, wsimt(net, 17), net->master + L[17].boff, 3, SIMT_FINAL, 0,
                       nullptr, out, lrhs, N, H, W, s, st);
    return rc;
}

mrs_status calibrate_fp8(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                         const float* nrm, const float* extra, int N, int H, int W, int s,
                         cudaStream_t st);

mrs_status fuse_tc(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                   const float* nrm, const float* extra, int N, int H, int W, int s, int prec, float* out,
                   cudaStream_t st, bool calib = false)
{
    size_t P = (size_t)N * H * W;
    const bool f8 = prec == MRS_PREC_FP8 && !calib;
    mrs_status rc = pack_bf16(net, st);
    if (rc != MRS_OK) return rc;
    if (f8) {
        if ((rc = pack_fp8(net, st)) != MRS_OK) return rc;
        if (!net->xscale_valid &&
            (rc = calibrate_fp8(net, lrhs, hrls, alb, nrm, extra, N, H, W, s, st)) != MRS_OK)
            return rc;
    }
    // workspace: x0, h, r in bf16 (128 B/px each); fp8 adds x0, h, r copies (64 B/px)
    size_t need = P * 128 * 3 + (f8 ? P * 64 * 3 : 0) + 1024;
    if ((rc = net->act.ensure(need)) != MRS_OK) return rc;
    uint8_t* base = net->act.as<uint8_t>();
    void* x0 = base;
    void* h = base + P * 128;
    void* r = base + P * 256;
    uint8_t* x08 = base + P * 384;
    uint8_t* h8 = x08 + P * 64;
    uint8_t* r8 = h8 + P * 64;
    int g = (int)((P + 255) / 256 < 65535 ? (P + 255) / 256 : 65535);
    k_input_q<<<g, 256, 0, st>>>(lrhs, hrls, alb, nrm, extra, H, W, s, P, f8 ? (void*)x08 : x0, f8 ? 1 : 0,
                                 f8 ? 1.0f / net->xscale[0] : 1.0f);
    MRS_LAUNCHED(1);
    if ((rc = cuda_status(cudaGetLastError(), "input")) != MRS_OK) return rc;
    // A-operand maps (bf16: 130-pixel halo boxes; fp8: 128) and the bf16
    // residual / output maps (128-pixel boxes)
    CUtensorMap mx, mh, mr, oh, orr;
    int oper = f8 ? TC_FP8 : TC_BF16;
    const int abox = tc_a_box(oper), obox = tc_out_box(oper);
    if ((rc = tc_make_act_map(&mx, f8 ? (void*)x08 : x0, N, H, W, oper, abox)) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&mh, f8 ? (void*)h8 : h, N, H, W, oper, abox)) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&mr, f8 ? (void*)r8 : r, N, H, W, oper, abox)) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&oh, h, N, H, W, TC_BF16, obox)) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&orr, r, N, H, W, TC_BF16, obox)) != MRS_OK) return rc;
    TcConvArgs a;
    memset(&a, 0, sizeof(a));
    a.N = N; a.H = H; a.W = W; a.scale = s;
    a.operand = oper;
    a.err = net->err;
    const int nl = calib ? kLayers - 1 : kLayers;
    for (int l = 0; l < nl && rc == MRS_OK; ++l) {
        a.tmap_w = f8 ? &net->wmap_f8[l] : &net->wmap_bf[l];
        a.bias = (f8 ? net->bias8 : net->bias) + l * 64;
        a.wscale = f8 ? net->wscale + l * 64 : nullptr;
        a.xscale = f8 ? net->xscale[l] : 1.0f;
        a.nout = nout_of(l);
        a.out_fp8 = nullptr;
        a.fp8_only = 0;
        a.tmap_res = nullptr;
        a.tmap_out = nullptr;
        if (l == 0) {
            a.tmap_x = &mx; a.mode = TC_RELU_BF16; a.out = h; a.res = nullptr; a.tmap_out = &oh;
            if (f8) { a.out_fp8 = h8; a.out_fp8_inv_scale = 1.0f / net->xscale[1]; }
        } else if (l == kLayers - 1) {
            a.tmap_x = &mh; a.mode = TC_FINAL_F32; a.out = out; a.lrhs = lrhs; a.cout = 3;
        } else if (l % 2 == 1) {
            a.tmap_x = &mh; a.mode = TC_RELU_BF16; a.out = r; a.res = nullptr; a.tmap_out = &orr;
            // r is read only as the next conv's operand: with fp8 operands
            // only its fp8 copy is written (not during calibration, which
            // measures the bf16 r)
            if (f8) { a.out_fp8 = r8; a.out_fp8_inv_scale = 1.0f / net->xscale[l + 1]; a.fp8_only = 1; }
        } else {
            a.tmap_x = &mr; a.mode = TC_RESID_BF16; a.out = h; a.res = h;
            a.tmap_res = &oh; a.tmap_out = &oh;
            if (f8) { a.out_fp8 = h8; a.out_fp8_inv_scale = 1.0f / net->xscale[l + 1]; }
        }
        rc = tc_conv3x3(a, st);
        if (calib && rc == MRS_OK && l < kLayers - 1) {
            // amax of the input of layer l + 1 (h after conv_in / blocks, r after conv1)
            const void* nxt = (l % 2 == 1) ? r : h;
            float* am = net->aux.as<float>() + l + 1;
            k_amax_bf16<<<512, 256, 0, st>>>((const __nv_bfloat16*)nxt, P * 64, am);
            MRS_LAUNCHED(1);
            rc = cuda_status(cudaGetLastError(), "amax");
        }
    }
    return rc;
}

// per-layer activation scales from one BF16 pass over the first input:
// xscale[l] = amax(input of layer l) / 448
mrs_status calibrate_fp8(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                         const float* nrm, const float* extra, int N, int H, int W, int s,
                         cudaStream_t st)
{
    mrs_status rc = net->aux.ensure(4096);
    if (rc != MRS_OK) return rc;
    MRS_CHECK(cudaMemsetAsync(net->aux.p, 0, 4096, st));
    size_t P = (size_t)N * H * W;
    rc = fuse_tc(net, lrhs, hrls, alb, nrm, extra, N, H, W, s, MRS_PREC_BF16, nullptr, st, true);
    (void)P;
    if (rc != MRS_OK) return rc;
    // layer 0 input: amax of the bf16 fusion input x0
    k_amax_bf16<<<512, 256, 0, st>>>(net->act.as<__nv_bfloat16>(), P * 64, net->aux.as<float>());
    MRS_LAUNCHED(1);
    float am[kLayers];
    MRS_CHECK(cudaMemcpyAsync(am, net->aux.p, sizeof(am), cudaMemcpyDeviceToHost, st));
    MRS_CHECK(cudaStreamSynchronize(st));
    for (int l = 0; l < kLayers; ++l) net->xscale[l] = am[l] > 0.0f ? am[l] / 448.0f : 1.0f;
    net->xscale_valid = true;
    return MRS_OK;
}

}  // namespace
}  // namespace mrs

extern "C" mrs_status mrs_net_create(const float* params, int32_t n_params, mrs_net* out)
{
    MRS_ARG(out != nullptr, "out is NULL");
    *out = nullptr;
    MRS_ARG(params != nullptr, "params is NULL");
    MRS_ARG(n_params == (int32_t)kParams12 || n_params == (int32_t)kParams21,
            "n_params must equal MRS_NET_NPARAMS or MRS_NET_NPARAMS_EXTRA");
    mrs_net_s* net = new mrs_net_s();
    net->np = (size_t)n_params;
    net->cin0 = n_params == (int32_t)kParams21 ? 21 : 12;
    mrs_status s = MRS_OK;
    // one allocation, carved up (a cudaMalloc each was most of the call)
    std::vector<std::pair<void**, size_t>> parts;
    auto alloc = [&](void** p, size_t bytes) { parts.push_back({p, (bytes + 255) & ~(size_t)255}); };
    alloc((void**)&net->master, net->np * 4);
    alloc((void**)&net->adam_m, net->np * 4);
    alloc((void**)&net->adam_v, net->np * 4);
    alloc((void**)&net->grad, net->np * 4);
    alloc((void**)&net->wbf, (size_t)kLayers * 9 * 64 * 64 * 2);
    alloc((void**)&net->wbfT, (size_t)kLayers * 9 * 64 * 64 * 2);
    alloc((void**)&net->wf8, (size_t)kLayers * 9 * 64 * 64);
    alloc((void**)&net->bias, kLayers * 64 * 4);
    alloc((void**)&net->bias8, kLayers * 64 * 4);
    alloc((void**)&net->wscale, kLayers * 64 * 4);
    alloc((void**)&net->err, 4);
    alloc((void**)&net->wsimt, (simt_off(net, kLayers - 1) + simt_pack_floats(64, 3)) * 4);
    size_t total = 0;
    for (const auto& p : parts) total += p.second;
    s = net->block.ensure(total);
    if (s == MRS_OK) {
        uint8_t* q = net->block.as<uint8_t>();
        for (const auto& p : parts) { *p.first = q; q += p.second; }
    }
    if (s == MRS_OK) s = mrs_net_set_params(net, params);
    if (s != MRS_OK) { mrs_net_free(net); return s; }
    *out = net;
    return MRS_OK;
}

extern "C" mrs_status mrs_net_free(mrs_net net)
{
    if (!net) return MRS_OK;
    cudaDeviceSynchronize();
    net->block.release();
    net->act.release();
    net->aux.release();
    net->tact.release();
    net->ttmp.release();
    delete net;
    return MRS_OK;
}

extern "C" mrs_status mrs_net_set_params(mrs_net net, const float* params)
{
    MRS_ARG(net && params, "NULL argument");
    MRS_CHECK(cudaMemcpy(net->master, params, net->np * 4, cudaMemcpyHostToDevice));
    MRS_CHECK(cudaMemset(net->adam_m, 0, net->np * 4));
    MRS_CHECK(cudaMemset(net->adam_v, 0, net->np * 4));
    MRS_CHECK(cudaMemset(net->err, 0, 4));
    net->step = 0;
    net->bf_valid = net->f8_valid = net->xscale_valid = net->bfT_valid = net->simt_valid = false;
    return MRS_OK;
}

extern "C" mrs_status mrs_net_get_params(mrs_net net, float* params)
{
    MRS_ARG(net && params, "NULL argument");
    MRS_CHECK(cudaMemcpy(params, net->master, net->np * 4, cudaMemcpyDeviceToHost));
    return MRS_OK;
}

extern "C" mrs_status mrs_net_input_channels(mrs_net net, int32_t* channels)
{
    MRS_ARG(net && channels, "NULL argument");
    *channels = net->cin0;
    return MRS_OK;
}

extern "C" mrs_status mrs_fuse(mrs_net net, const float* lrhs, const float* hrls,
                               const float* albedo, const float* normal, int32_t N, int32_t H,
                               int32_t W, int32_t scale, int32_t precision, float* out, void* stream)
{
    return mrs_fuse_extra(net, lrhs, hrls, albedo, normal, nullptr, N, H, W, scale, precision, out,
                          stream);
}

extern "C" mrs_status mrs_fuse_extra(mrs_net net, const float* lrhs, const float* hrls,
                                     const float* albedo, const float* normal, const float* extra,
                                     int32_t N, int32_t H, int32_t W, int32_t scale,
                                     int32_t precision, float* out, void* stream)
{
    MRS_ARG(net != nullptr, "net is NULL");
    MRS_ARG(lrhs && hrls && albedo && normal && out, "NULL image pointer");
    MRS_ARG((extra != nullptr) == (net->cin0 == 21),
            "extra layers must be given exactly for a net with MRS_NET_NPARAMS_EXTRA parameters");
    MRS_ARG(scale == 1 || scale == 2 || scale == 4 || scale == 8, "scale must be 1, 2, 4 or 8");
    MRS_ARG(N >= 1 && H >= 1 && W >= 1, "N, H, W must be >= 1");
    MRS_ARG(H % scale == 0 && W % scale == 0, "H and W must be multiples of scale");
    MRS_ARG((int64_t)N * H * W <= (int64_t(1) << 27), "N*H*W exceeds 2^27 pixels");
    MRS_ARG(precision >= MRS_PREC_FP32 && precision <= MRS_PREC_FP8, "precision");
    cudaStream_t st = (cudaStream_t)stream;
    mrs_status rc;
    if (precision == MRS_PREC_FP32)
        rc = fuse_f32(net, lrhs, hrls, albedo, normal, extra, N, H, W, scale, out, st);
    else
        rc = fuse_tc(net, lrhs, hrls, albedo, normal, extra, N, H, W, scale, precision, out, st);
    return rc;
}

extern "C" mrs_status mrs_image_metrics(const float* x, const float* ref, int64_t n, double l1,
                                        double l2, double* out, void* stream)
{
    MRS_ARG(x && ref && out, "NULL pointer");
    MRS_ARG(n >= 1, "n must be >= 1");
    cudaStream_t st = (cudaStream_t)stream;
    Scratch& S = scratch();
    std::lock_guard<std::mutex> g(S.mu);
    mrs_status rc = S.b.ensure(sizeof(double) * (kRedBlocks * 3 + 8));
    if (rc != MRS_OK) return rc;
    double* part = S.b.as<double>();
    double* res = part + kRedBlocks * 3;
    k_metrics_partial<<<kRedBlocks, 256, 0, st>>>(x, ref, n, l1, l2, part);
    MRS_LAUNCHED(1);
    k_reduce_parts<<<1, 256, 0, st>>>(part, kRedBlocks, 3, res);
    MRS_LAUNCHED(1);
    double h[3];
    MRS_CHECK(cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, st));
    MRS_CHECK(cudaStreamSynchronize(st));
    double mse_s = h[0] / (double)n;
    out[0] = mse_s == 0.0 ? INFINITY : 10.0 * log10(1.0 / mse_s);
    out[1] = h[1] / (double)n;
    out[2] = h[2] / (double)n;
    return MRS_OK;
}

extern "C" mrs_status mrs_gate(const float* fused, const float* lrhs, const float* plain,
                               int32_t N, int32_t H, int32_t W, int32_t scale, double tau,
                               float* out, int32_t* used_plain, double* D, void* stream)
{
    MRS_ARG(fused && lrhs, "NULL pointer");
    MRS_ARG(scale >= 1 && N >= 1 && H >= scale && W >= scale && H % scale == 0 && W % scale == 0,
            "bad sizes");
    cudaStream_t st = (cudaStream_t)stream;
    Scratch& S = scratch();
    std::lock_guard<std::mutex> g(S.mu);
    mrs_status rc = S.b.ensure(sizeof(double) * (kRedBlocks + 8));
    if (rc != MRS_OK) return rc;
    double* part = S.b.as<double>();
    double* res = part + kRedBlocks;
    k_gate_partial<<<kRedBlocks, 256, 0, st>>>(fused, lrhs, N, H, W, scale, part);
    MRS_LAUNCHED(1);
    k_reduce_parts<<<1, 256, 0, st>>>(part, kRedBlocks, 1, res);
    MRS_LAUNCHED(1);
    double d;
    MRS_CHECK(cudaMemcpyAsync(&d, res, sizeof(d), cudaMemcpyDeviceToHost, st));
    MRS_CHECK(cudaStreamSynchronize(st));
    d /= (double)N * (H / scale) * (W / scale) * 3;
    bool use_plain = d > tau;
    if (D) *D = d;
    if (used_plain) *used_plain = use_plain ? 1 : 0;
    size_t bytes = (size_t)N * H * W * 3 * 4;
    if (out) {
        const float* src = (use_plain && plain) ? plain : fused;
        if (src != out) MRS_CHECK(cudaMemcpyAsync(out, src, bytes, cudaMemcpyDeviceToDevice, st));
    }
    return MRS_OK;
}

namespace mrs {
namespace {
// BF16 3x3 conv over more than 64 input channels: the input is split into
// 64-channel operand tensors and ONE tensor-core launch accumulates all of
// them (multi-chunk conv, chunk maps passed in device memory)
mrs_status conv3x3_chunked(Scratch& S, const float* x, int N, int H, int W, int cin, int cout,
                           const float* w, const float* b, int relu, float* out, cudaStream_t st)
{
    const size_t P = (size_t)N * H * W;
    const int nch = (cin + 63) / 64;
    const int nout = cout > 16 ? 64 : 16;
    const size_t wbytes = (size_t)cout * 9 * cin * 4;
    const size_t chunk_el = (size_t)9 * nout * 64;               // packed bf16 weights per chunk
    const size_t wpk_bytes = ((nch * chunk_el * 2 + 1023) / 1024) * 1024;
    const size_t xq_bytes = ((P * 128 + 1023) / 1024) * 1024;    // one [P][64] bf16 operand
    size_t need = wbytes + 64 * 4 + 1024 + wpk_bytes + nch * xq_bytes + nch * sizeof(CUtensorMap) + 1024;
    mrs_status rc = S.b.ensure(need);
    if (rc != MRS_OK) return rc;
    uint8_t* base = S.b.as<uint8_t>();
    float* dw = (float*)base;
    float* db = dw + (size_t)cout * 9 * cin;
    uint8_t* wpk = (uint8_t*)(((uintptr_t)(db + 64) + 1023) & ~(uintptr_t)1023);
    uint8_t* xq = wpk + wpk_bytes;
    CUtensorMap* dmaps = (CUtensorMap*)(xq + nch * xq_bytes);
    MRS_CHECK(cudaMemsetAsync(db, 0, 64 * 4, st));
    MRS_CHECK(cudaMemcpyAsync(dw, w, wbytes, cudaMemcpyHostToDevice, st));
    MRS_CHECK(cudaMemcpyAsync(db, b, cout * 4, cudaMemcpyHostToDevice, st));
    static int* err = nullptr;
    if (!err) { MRS_CHECK(cudaMalloc(&err, 4)); MRS_CHECK(cudaMemset(err, 0, 4)); }
    std::vector<CUtensorMap> hm(nch);
    for (int j = 0; j < nch; ++j) {
        k_pack_bf16_chunk<<<(9 * nout * 64 + 255) / 256, 256, 0, st>>>(
            dw, cin, 64 * j, cout, nout, (__nv_bfloat16*)wpk + j * chunk_el);
        MRS_LAUNCHED(1);
        __nv_bfloat16* xj = (__nv_bfloat16*)(xq + j * xq_bytes);
        k_to_operand_chunk<<<1024, 256, 0, st>>>(x, P, cin, 64 * j, xj);
        MRS_LAUNCHED(1);
        if ((rc = tc_make_act_map(&hm[j], xj, N, H, W, TC_BF16, tc_a_box(TC_BF16))) != MRS_OK) return rc;
    }
    CUtensorMap wm;
    if ((rc = tc_make_w_map(&wm, wpk, nch * 9 * nout, nout, TC_BF16)) != MRS_OK) return rc;
    MRS_CHECK(cudaMemcpyAsync(dmaps, hm.data(), nch * sizeof(CUtensorMap), cudaMemcpyHostToDevice, st));
    TcConvArgs a;
    memset(&a, 0, sizeof(a));
    a.tmap_x = &hm[0]; a.tmap_w = &wm; a.amaps = dmaps; a.kc = nch; a.w_row0 = 0;
    a.bias = db; a.out = out; a.N = N; a.H = H; a.W = W; a.scale = 1; a.nout = nout;
    a.cout = cout; a.relu = relu; a.mode = TC_PLAIN_F32; a.operand = TC_BF16; a.err = err;
    rc = tc_conv3x3(a, st);
    // the host map array and the scratch stay valid until the stream is synchronised
    if (rc == MRS_OK) rc = cuda_status(cudaStreamSynchronize(st), "conv3x3 sync");
    int herr = 0;
    if (rc == MRS_OK) {
        MRS_CHECK(cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost));
        if (herr) { cudaMemset(err, 0, 4); set_error("tensor-core conv wait timed out"); return MRS_ERR_TIMEOUT; }
    }
    return rc;
}
}  // namespace
}  // namespace mrs

extern "C" mrs_status mrs_conv3x3(const float* x, int32_t N, int32_t H, int32_t W, int32_t cin,
                                  int32_t cout, const float* w, const float* b, int32_t relu,
                                  int32_t precision, float* out, void* stream)
{
    MRS_ARG(x && w && b && out, "NULL pointer");
    MRS_ARG(N >= 1 && H >= 1 && W >= 1 && cin >= 1 && cout >= 1, "sizes must be >= 1");
    MRS_ARG(precision == MRS_PREC_FP32 || cout <= 64, "tensor-core conv needs cout <= 64");
    MRS_ARG(precision == MRS_PREC_FP32 || cin <= 64 || (precision == MRS_PREC_BF16 && cin <= 1024),
            "tensor-core conv needs cin <= 64 (FP8) or cin <= 1024 (BF16)");
    cudaStream_t st = (cudaStream_t)stream;
    size_t P = (size_t)N * H * W;
    Scratch& S = scratch();
    std::lock_guard<std::mutex> g(S.mu);
    if (precision == MRS_PREC_BF16 && cin > 64)
        return conv3x3_chunked(S, x, N, H, W, cin, cout, w, b, relu, out, st);
    size_t wbytes = (size_t)cout * 9 * cin * 4;
    size_t need = wbytes + cout * 4 + 9 * 64 * 64 * 2 + 64 * 4 * 2 + 1024 +
                  (precision == MRS_PREC_FP32 ? simt_pack_floats(cin, cout) * 4 : P * 128) + 16;
    mrs_status rc = S.b.ensure(need);
    if (rc != MRS_OK) return rc;
    uint8_t* base = S.b.as<uint8_t>();
    float* dw = (float*)base;
    float* db = dw + (size_t)cout * 9 * cin;
    uint8_t* q = (uint8_t*)(((uintptr_t)(db + cout) + 255) & ~(uintptr_t)255);
    MRS_CHECK(cudaMemcpyAsync(dw, w, wbytes, cudaMemcpyHostToDevice, st));
    MRS_CHECK(cudaMemcpyAsync(db, b, cout * 4, cudaMemcpyHostToDevice, st));
    if (precision == MRS_PREC_FP32) {
        if ((rc = simt_pack(dw, cin, cout, 0, (float*)q, st)) != MRS_OK) return rc;
        rc = conv_simt(x, cin, (const float*)q, db, cout, SIMT_PLAIN, relu, nullptr, out, nullptr, N, H, W, 1, st);
        if (rc == MRS_OK) rc = cuda_status(cudaStreamSynchronize(st), "conv3x3 sync");
        return rc;
    }
    // tensor cores: pack weights and input into the operand format
    int nout = cout > 16 ? 64 : 16;
    int oper = precision == MRS_PREC_BF16 ? TC_BF16 : TC_FP8;
    void* wp = q;
    float* bp = (float*)(q + 9 * 64 * 64 * 2);
    float* ws = bp + 64;
    float* amax_slot = ws + 64;   // one float, then the operand buffer (1024-aligned)
    void* xq = (void*)(((uintptr_t)(amax_slot + 4) + 1023) & ~(uintptr_t)1023);
    static int* err = nullptr;
    if (!err) { MRS_CHECK(cudaMalloc(&err, 4)); MRS_CHECK(cudaMemset(err, 0, 4)); }
    float xscale = 1.0f;
    if (oper == TC_BF16) {
        k_pack_bf16<<<(9 * nout * 64 + 255) / 256, 256, 0, st>>>(dw, 0, (size_t)cout * 9 * cin, cin, cout, nout,
                                                                 (__nv_bfloat16*)wp, bp);
        MRS_LAUNCHED(1);
    } else {
        k_pack_fp8<<<1, 256, 0, st>>>(dw, 0, (size_t)cout * 9 * cin, cin, cout, nout, (uint8_t*)wp, bp, ws);
        MRS_LAUNCHED(1);
    }
    // input conversion: x fp32 [P][cin] -> [P][64] operand rows (fp8: per-tensor
    // scale amax / 448, computed on the device)
    if (oper == TC_FP8) {
        float* amax = amax_slot;
        MRS_CHECK(cudaMemsetAsync(amax, 0, 4, st));
        k_amax_f32<<<512, 256, 0, st>>>(x, P * cin, amax);
        MRS_LAUNCHED(1);
        float hm = 0;
        MRS_CHECK(cudaMemcpyAsync(&hm, amax, 4, cudaMemcpyDeviceToHost, st));
        MRS_CHECK(cudaStreamSynchronize(st));
        xscale = hm > 0 ? hm / 448.0f : 1.0f;
    }
    k_to_operand<<<1024, 256, 0, st>>>(x, P, cin, xq, oper == TC_FP8, 1.0f / xscale);
    MRS_LAUNCHED(1);
    CUtensorMap mx, mw;
    if ((rc = tc_make_act_map(&mx, xq, N, H, W, oper, tc_a_box(oper))) != MRS_OK) return rc;
    if ((rc = tc_make_w_map(&mw, wp, 9 * nout, nout, oper)) != MRS_OK) return rc;
    TcConvArgs a;
    memset(&a, 0, sizeof(a));
    a.tmap_x = &mx; a.tmap_w = &mw; a.bias = bp; a.wscale = ws; a.xscale = xscale;
    a.out = out; a.N = N; a.H = H; a.W = W; a.scale = 1; a.nout = nout; a.cout = cout;
    a.relu = relu; a.mode = TC_PLAIN_F32; a.operand = oper; a.err = err;
    rc = tc_conv3x3(a, st);
    if (rc == MRS_OK) rc = cuda_status(cudaStreamSynchronize(st), "conv3x3 sync");
    int herr = 0;
    if (rc == MRS_OK) {
        MRS_CHECK(cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost));
        if (herr) { cudaMemset(err, 0, 4); set_error("tensor-core conv wait timed out"); return MRS_ERR_TIMEOUT; }
    }
    return rc;
}


namespace mrs {
namespace {

constexpr int kDwSplits = 64;
constexpr float kClip = 100.0f;

__global__ void k_clip_copy(const float* __restrict__ x, size_t n, float clip, float* __restrict__ y)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        y[i] = fminf(x[i], clip);
}

inline int grid1d(size_t n) { size_t g = (n + 255) / 256; return (int)(g < 4096 ? (g ? g : 1) : 4096); }

// dW / db of layer l from its input x [P][cin] and output gradient dy [P][cout]
mrs_status layer_dw(mrs_net_s* net, int l, const float* x, const float* dy, int N, int H, int W,
                    float* part, float* dbpart, cudaStream_t st)
{
    const LayerShape& L = shapes(net->cin0)[l];
    dim3 grid(kDwSplits, 9);
    MRS_TIMED(PK_TRAIN, st, launch_dw(grid, x, L.cin, L.cin, dy, L.cout, L.cout, N, H, W, part, dbpart, 0, 1, st));
    MRS_LAUNCHED(1);
    int nw = L.cout * 9 * L.cin + L.cout;
    MRS_TIMED(PK_TRAIN, st, k_dw_reduce<<<(nw + 31) / 32, 256, 0, st>>>(part, dbpart, kDwSplits, (size_t)9 * L.cout * L.cin, L.cout,
                                                         L.cin, L.cout, net->grad + L.woff, net->grad + L.boff));
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "dw");
}

// transposed conv of layer l: dx [P][cin] = conv(dy [P][cout], flipped w^T), epilogue `mode`
mrs_status layer_dx(mrs_net_s* net, int l, const float* dy, float* wt, const float* zero,
                    int mode, const float* res, float* dx, int N, int H, int W, cudaStream_t st)
{
    const LayerShape& L = shapes(net->cin0)[l];
    mrs_status rc = simt_pack(net->master + L.woff, L.cin, L.cout, 1, wt, st);
    if (rc != MRS_OK) return rc;
    return conv_simt(dy, L.cout, wt, zero, L.cin, mode, 0, res, dx, nullptr, N, H, W, 1, st);
}

mrs_status train_step_f32(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                          const float* nrm, const float* extra, const float* target, int N, int H,
                          int W, int s, float lr, double* loss_out, cudaStream_t st)
{
    const int c0 = net->cin0;
    const size_t P = (size_t)N * H * W;
    const size_t F = P * 64;
    const size_t nlr = (size_t)N * (H / s) * (W / s) * 3;
    // activations: x0 | h0..h8 | r0..r7 | y | dy | dh | da | lrhs_clipped
    size_t need = (P * c0 + 9 * F + 8 * F + 2 * P * 3 + 2 * F + nlr) * 4 + 32;
    mrs_status rc = net->tact.ensure(need);
    if (rc != MRS_OK) return rc;
    size_t tneed = (64 * 9 * 64 + 64) * 4 + ((size_t)kDwSplits * 9 * 64 * 64 + kDwSplits * 64) * 4 +
                   (kRedBlocks + 8) * 8;
    if ((rc = net->ttmp.ensure(tneed)) != MRS_OK) return rc;
    float* x0 = net->tact.as<float>();
    float* hs = x0 + ((P * c0 + 3) & ~(size_t)3);    // 16-byte aligned
    float* rs = hs + 9 * F;
    float* y = rs + 8 * F;
    float* dy = y + P * 3;
    float* dh = y + ((2 * P * 3 + 3) & ~(size_t)3);
    float* da = dh + F;
    float* lrc = da + F;
    float* wt = net->ttmp.as<float>();
    float* zero = wt + 64 * 9 * 64;
    float* part = zero + 64;
    float* dbpart = part + (size_t)kDwSplits * 9 * 64 * 64;
    double* lparts = (double*)(dbpart + kDwSplits * 64);
    double* lres = lparts + kRedBlocks;
    MRS_CHECK(cudaMemsetAsync(zero, 0, 64 * 4, st));
    const auto& L = shapes(net->cin0);
    const float* M = net->master;
    if ((rc = pack_simt(net, st)) != MRS_OK) return rc;

    // forward, keeping every activation the backward needs
    k_clip_copy<<<grid1d(nlr), 256, 0, st>>>(lrhs, nlr, kClip, lrc);
    MRS_LAUNCHED(1);
    k_input_f32<<<grid1d(P), 256, 0, st>>>(lrc, hrls, alb, nrm, extra, H, W, s, P, x0, kClip);
    MRS_LAUNCHED(1);
    rc = conv_simt(x0, c0, wsimt(net, 0), M + L[0].boff, 64, SIMT_PLAIN, 1, nullptr, hs, nullptr, N, H, W, s, st);
    for (int k = 0; k < 8 && rc == MRS_OK; ++k) {
        const LayerShape& a = L[1 + 2 * k];
        const LayerShape& b = L[2 + 2 * k];
        rc = conv_simt(hs + k * F, 64, wsimt(net, 1 + 2 * k), M + a.boff, 64, SIMT_PLAIN, 1, nullptr, rs + k * F,
                       nullptr, N, H, W, s, st);
        if (rc == MRS_OK)
            rc = conv_simt(rs + k * F, 64, wsimt(net, 2 + 2 * k), M + b.boff, 64, SIMT_RESID, 0, hs + k * F,
                           hs + (k + 1) * F, nullptr, N, H, W, s, st);
    }
    if (rc == MRS_OK)
        rc = conv_simt(hs + 8 * F, 64, wsimt(net, 17), M + L[17].boff, 3, SIMT_FINAL, 0, nullptr, y, lrc,
                       N, H, W, s, st);
    if (rc != MRS_OK) return rc;

    // loss (float64 reduction) and dL/dy
    MRS_TIMED(PK_TRAIN, st, k_loss<<<kRedBlocks, 256, 0, st>>>(y, target, P * 3, kClip, net->loss_kind,
                                                               net->loss_beta, dy, lparts));
    MRS_LAUNCHED(1);
    k_reduce_parts<<<1, 256, 0, st>>>(lparts, kRedBlocks, 1, lres);
    MRS_LAUNCHED(1);

    // backward
    if ((rc = layer_dw(net, 17, hs + 8 * F, dy, N, H, W, part, dbpart, st)) != MRS_OK) return rc;
    if ((rc = layer_dx(net, 17, dy, wt, zero, SIMT_PLAIN, nullptr, dh, N, H, W, st)) != MRS_OK) return rc;
    for (int k = 7; k >= 0; --k) {
        int l2 = 2 + 2 * k, l1 = 1 + 2 * k;
        if ((rc = layer_dw(net, l2, rs + k * F, dh, N, H, W, part, dbpart, st)) != MRS_OK) return rc;
        if ((rc = layer_dx(net, l2, dh, wt, zero, SIMT_MASK, rs + k * F, da, N, H, W, st)) != MRS_OK) return rc;
        if ((rc = layer_dw(net, l1, hs + k * F, da, N, H, W, part, dbpart, st)) != MRS_OK) return rc;
        if ((rc = layer_dx(net, l1, da, wt, zero, SIMT_RESID, dh, dh, N, H, W, st)) != MRS_OK) return rc;
    }
    k_mask_inplace<<<grid1d(F), 256, 0, st>>>(dh, hs, F);
    MRS_LAUNCHED(1);
    if ((rc = layer_dw(net, 0, x0, dh, N, H, W, part, dbpart, st)) != MRS_OK) return rc;

    // Adam on the FP32 master weights
    net->step += 1;
    const double b1 = 0.9, b2 = 0.999;
    float bc1 = (float)(1.0 - pow(b1, (double)net->step));
    float bc2 = (float)(1.0 - pow(b2, (double)net->step));
    MRS_TIMED(PK_TRAIN, st, k_adam<<<grid1d(net->np), 256, 0, st>>>(net->master, net->grad, net->adam_m, net->adam_v,
                                                        net->np, lr, (float)b1, (float)b2, 1e-8f, bc1, bc2));
    MRS_LAUNCHED(1);
    net->bf_valid = net->f8_valid = net->xscale_valid = net->bfT_valid = net->simt_valid = false;
    if (recording(st)) net->step_recorded = true;
    if (loss_out) {
        double h = 0;
        MRS_CHECK(cudaMemcpyAsync(&h, lres, sizeof(double), cudaMemcpyDeviceToHost, st));
        MRS_CHECK(cudaStreamSynchronize(st));
        *loss_out = h / (double)(P * 3);
    }
    return cuda_status(cudaGetLastError(), "train step");
}

mrs_status pack_bf16_T(mrs_net_s* net, cudaStream_t st)
{
    if (net->bfT_valid) return MRS_OK;
    k_pack_layers_bf16_T<<<dim3(9 * 64 * 64 / 256, kLayers - 1), 256, 0, st>>>(net->master, pack_layers(net->cin0),
                                                                               net->wbfT);
    MRS_LAUNCHED(1);
    for (int l = 1; l < kLayers; ++l) {
        mrs_status rc = tc_make_w_map(&net->wmap_bfT[l], net->wbfT + (size_t)l * 9 * 64 * 64, 9 * 64, 64, TC_BF16);
        if (rc != MRS_OK) return rc;
    }
    net->bfT_valid = true;
    return cuda_status(cudaGetLastError(), "pack bf16 T");
}

// The plan of a step of this shape over the workspace tensors, on the device as
// of `st` (see StepPlan).  The upload is ordered on st, not on the legacy stream,
// which a non-blocking stream does not wait for.
mrs_status step_plan(mrs_net_s* net, int N, int H, int W, __nv_bfloat16* x0, __nv_bfloat16* hs, __nv_bfloat16* rs,
                     __nv_bfloat16* dyb, __nv_bfloat16* dhs, __nv_bfloat16* das, cudaStream_t st, StepPlan*& plan)
{
    const bool rec = recording(st);
    auto use = [&](StepPlan& p) -> mrs_status {
        if (!p.uploaded) {
            MRS_CHECK(cudaMemcpyAsync(p.blob.p, p.image.data(), p.image.size(), cudaMemcpyHostToDevice, st));
            p.uploaded = !rec;
        }
        p.recorded = p.recorded || rec;
        p.used = ++net->plan_clock;
        plan = &p;
        return MRS_OK;
    };
    // the shape's plan, and the place of the longest unused one that may go
    size_t direct = 0, oldest = net->plans.size();
    for (size_t i = 0; i < net->plans.size(); ++i) {
        StepPlan& p = *net->plans[i];
        if (p.N == N && p.H == H && p.W == W && p.act == x0) return use(p);
        if (p.recorded) continue;
        ++direct;
        if (oldest == net->plans.size() || p.used < net->plans[oldest]->used) oldest = i;
    }
    std::unique_ptr<StepPlan> pl(new StepPlan());
    const size_t F = (size_t)N * H * W * 64;
    const auto& L = shapes(net->cin0);
    mrs_status rc = MRS_OK;
    // A operands (130-pixel boxes) and residual / output (128-pixel)
    auto amap = [&](CUtensorMap* m, const void* ptr) {
        if (rc == MRS_OK) rc = tc_make_act_map(m, ptr, N, H, W, TC_BF16, tc_a_box(TC_BF16));
    };
    auto omap = [&](CUtensorMap* m, const void* ptr) {
        if (rc == MRS_OK) rc = tc_make_act_map(m, ptr, N, H, W, TC_BF16, tc_out_box(TC_BF16));
    };
    amap(&pl->x0A, x0);
    amap(&pl->dybA, dyb);
    for (int k = 0; k < 9; ++k) {
        amap(&pl->hA[k], hs + k * F); omap(&pl->hO[k], hs + k * F);
        amap(&pl->dhA[k], dhs + k * F); omap(&pl->dhO[k], dhs + k * F);
    }
    for (int k = 0; k < 8; ++k) {
        amap(&pl->rA[k], rs + k * F); omap(&pl->rO[k], rs + k * F);
        amap(&pl->daA[k], das + k * F); omap(&pl->daO[k], das + k * F);
    }
    std::vector<WgTile> tiles;
    std::vector<WgRed> reds;
    auto tile = [&](int l, const void* x, const void* dyp) {
        WgTile t;
        if (rc == MRS_OK) rc = tc_make_wg_x_map(&t.x, x, N, H, W, 128, 128LL * W, 128LL * W * H);
        if (rc == MRS_OK) rc = tc_make_wg_dy_map(&t.dy, dyp, N, H, W, 128, 128LL * W, 128LL * W * H);
        t.N = N; t.H = H; t.W = W; t.cin = L[l].cin; t.cout = L[l].cout; t.runs = sm_count();
        tiles.push_back(t);
        WgRed r;
        memset(&r, 0, sizeof(r));
        r.cin = r.CIN = L[l].cin; r.cout = L[l].cout; r.KK = 9; r.o_mul = 1; r.s = 1; r.with_bias = 1;
        r.gw = (long long)L[l].woff; r.gb = (long long)L[l].boff;
        reds.push_back(r);
    };
    tile(17, hs + 8 * F, dyb);
    for (int k = 7; k >= 0; --k) {
        tile(2 + 2 * k, rs + k * F, dhs + (k + 1) * F);
        tile(1 + 2 * k, hs + k * F, das + k * F);
    }
    tile(0, x0, dhs);
    if (rc == MRS_OK) rc = tc_wgrad_plan(tiles, 8, pl->wg);
    if (rc != MRS_OK) return rc;
    for (size_t t = 0; t < reds.size(); ++t) reds[t].np = pl->wg.np[t];
    const size_t off = (pl->wg.blob.size() + 15) & ~(size_t)15, red_bytes = reds.size() * sizeof(WgRed);
    pl->image.resize(off + red_bytes);
    memcpy(pl->image.data(), pl->wg.blob.data(), pl->wg.blob.size());
    memcpy(pl->image.data() + off, reds.data(), red_bytes);
    if (direct >= kStepPlans) {
        // the device memory of the plan that goes (in stream order: steps of a
        // handle share its workspace)
        std::swap(pl->blob, net->plans[oldest]->blob);
        net->plans.erase(net->plans.begin() + oldest);
    }
    {
        RelaxedCapture relaxed;    // a step of a new shape may be recorded
        rc = pl->blob.ensure(tc_wgrad_blob_max((int)tiles.size(), 8) + 16 + red_bytes);
    }
    if (rc != MRS_OK) return rc;
    pl->reds = (const WgRed*)((uint8_t*)pl->blob.p + off);
    pl->N = N; pl->H = H; pl->W = W; pl->act = x0;
    net->plans.push_back(std::move(pl));
    return use(*net->plans.back());
}

// BF16 training step: forward and transposed convolutions on the tensor-core
// kernel with BF16 activations / activation gradients, FP32 accumulation,
// FP32 dW / db reductions and FP32 master weights + Adam
mrs_status train_step_bf16(mrs_net_s* net, const float* lrhs, const float* hrls, const float* alb,
                           const float* nrm, const float* extra, const float* target, int N, int H,
                           int W, int s, float lr, double* loss_out, cudaStream_t st)
{
    const size_t P = (size_t)N * H * W;
    const size_t F = P * 64;                       // bf16 elements of one [P][64] tensor
    const size_t nlr = (size_t)N * (H / s) * (W / s) * 3;
    size_t need = (size_t)(1 + 9 + 8 + 1 + 9 + 8) * F * 2 + (2 * P * 3 + nlr + P * 3) * 4 + 4096;
    mrs_status rc = net->tact.ensure(need);
    if (rc != MRS_OK) return rc;
    __nv_bfloat16* x0 = net->tact.as<__nv_bfloat16>();
    __nv_bfloat16* hs = x0 + F;
    __nv_bfloat16* rs = hs + 9 * F;
    __nv_bfloat16* dyb = rs + 8 * F;
    __nv_bfloat16* dhs = dyb + F;                  // dL/dh_k, k = 0 .. 8
    __nv_bfloat16* das = dhs + 9 * F;              // dL/d(inner conv of block k), masked
    float* y = (float*)(das + 8 * F);
    float* dy = y + P * 3;
    float* lrc = dy + P * 3;
    float* hrc = lrc + nlr;
    StepPlan* plan = nullptr;
    if ((rc = step_plan(net, N, H, W, x0, hs, rs, dyb, dhs, das, st, plan)) != MRS_OK) return rc;
    const StepPlan& pl = *plan;
    size_t tneed = 64 * 4 + (pl.wg.part_floats() + pl.wg.dbpart_floats()) * 4 + (kRedBlocks + 8) * 8;
    if ((rc = net->ttmp.ensure(tneed)) != MRS_OK) return rc;
    if ((rc = pack_bf16(net, st)) != MRS_OK) return rc;
    if ((rc = pack_bf16_T(net, st)) != MRS_OK) return rc;
    double* lparts = net->ttmp.as<double>();
    double* lres = lparts + kRedBlocks;
    float* zero = (float*)(lres + 8);
    float* part = zero + 64;
    float* dbpart = part + pl.wg.part_floats();
    MRS_CHECK(cudaMemsetAsync(zero, 0, 64 * 4, st));

    TcConvArgs a;
    memset(&a, 0, sizeof(a));
    a.N = N; a.H = H; a.W = W; a.scale = s; a.operand = TC_BF16; a.err = net->err; a.nout = 64;
    auto conv = [&](const CUtensorMap* A, const CUtensorMap* Wm, const float* bias, int mode,
                    const CUtensorMap* res, const CUtensorMap* out, int nout) {
        a.tmap_x = A; a.tmap_w = Wm; a.bias = bias; a.mode = mode; a.tmap_res = res;
        a.tmap_out = out; a.nout = nout;
        return tc_conv3x3(a, st);
    };

    // forward
    k_clip_copy<<<grid1d(nlr), 256, 0, st>>>(lrhs, nlr, kClip, lrc);
    MRS_LAUNCHED(1);
    k_clip_copy<<<grid1d(P * 3), 256, 0, st>>>(hrls, P * 3, kClip, hrc);
    MRS_LAUNCHED(1);
    k_input_q<<<grid1d(P), 256, 0, st>>>(lrc, hrc, alb, nrm, extra, H, W, s, P, x0, 0, 1.0f, kClip);
    MRS_LAUNCHED(1);
    rc = conv(&pl.x0A, &net->wmap_bf[0], net->bias, TC_RELU_BF16, nullptr, &pl.hO[0], 64);
    for (int k = 0; k < 8 && rc == MRS_OK; ++k) {
        rc = conv(&pl.hA[k], &net->wmap_bf[1 + 2 * k], net->bias + (1 + 2 * k) * 64, TC_RELU_BF16,
                  nullptr, &pl.rO[k], 64);
        if (rc == MRS_OK)
            rc = conv(&pl.rA[k], &net->wmap_bf[2 + 2 * k], net->bias + (2 + 2 * k) * 64, TC_RESID_BF16,
                      &pl.hO[k], &pl.hO[k + 1], 64);
    }
    if (rc == MRS_OK) {
        a.out = y; a.lrhs = lrc; a.cout = 3;
        rc = conv(&pl.hA[8], &net->wmap_bf[17], net->bias + 17 * 64, TC_FINAL_F32, nullptr, nullptr, 16);
    }
    if (rc != MRS_OK) return rc;

    // loss
    MRS_TIMED(PK_TRAIN, st, k_loss<<<kRedBlocks, 256, 0, st>>>(y, target, P * 3, kClip, net->loss_kind,
                                                               net->loss_beta, dy, lparts));
    MRS_LAUNCHED(1);
    k_reduce_parts<<<1, 256, 0, st>>>(lparts, kRedBlocks, 1, lres);
    MRS_LAUNCHED(1);

    // backward: data gradients as convs with the flipped, transposed weights,
    // every one kept, then the weight gradients of all layers in one launch
    // (18 launches of 152 partial sums each, and their reductions, took 1.37 of
    // a step's 2.50 ms at 16 x 128^2)
    k_to_operand<<<1024, 256, 0, st>>>(dy, P, 3, dyb, 0, 1.0f);
    MRS_LAUNCHED(1);
    if ((rc = conv(&pl.dybA, &net->wmap_bfT[17], zero, TC_LIN_BF16, nullptr, &pl.dhO[8], 64)) != MRS_OK) return rc;
    for (int k = 7; k >= 0; --k) {
        int l2 = 2 + 2 * k, l1 = 1 + 2 * k;
        if ((rc = conv(&pl.dhA[k + 1], &net->wmap_bfT[l2], zero, TC_MASK_BF16, &pl.rO[k], &pl.daO[k], 64)) != MRS_OK)
            return rc;
        a.mask = k == 0 ? hs : nullptr;            // the head's ReLU
        if ((rc = conv(&pl.daA[k], &net->wmap_bfT[l1], zero, TC_RESID_BF16, &pl.dhO[k + 1], &pl.dhO[k], 64)) != MRS_OK)
            return rc;
    }
    if ((rc = tc_conv3x3_wgrad(pl.wg, pl.blob.p, part, dbpart, net->err, st)) != MRS_OK) return rc;
    if ((rc = wg_reduce(pl.reds, pl.wg.ntiles, part, dbpart, net->grad, st)) != MRS_OK) return rc;

    // Adam on the FP32 master weights
    net->step += 1;
    const double b1 = 0.9, b2 = 0.999;
    float bc1 = (float)(1.0 - pow(b1, (double)net->step));
    float bc2 = (float)(1.0 - pow(b2, (double)net->step));
    MRS_TIMED(PK_TRAIN, st, k_adam<<<grid1d(net->np), 256, 0, st>>>(net->master, net->grad, net->adam_m, net->adam_v,
                                                        net->np, lr, (float)b1, (float)b2, 1e-8f, bc1, bc2));
    MRS_LAUNCHED(1);
    net->bf_valid = net->f8_valid = net->xscale_valid = net->bfT_valid = net->simt_valid = false;
    if (recording(st)) net->step_recorded = true;
    if (loss_out) {
        double h = 0;
        MRS_CHECK(cudaMemcpyAsync(&h, lres, sizeof(double), cudaMemcpyDeviceToHost, st));
        MRS_CHECK(cudaStreamSynchronize(st));
        *loss_out = h / (double)(P * 3);
    }
    return cuda_status(cudaGetLastError(), "train step bf16");
}

}  // namespace
}  // namespace mrs

extern "C" mrs_status mrs_train_step(mrs_net net, const float* lrhs, const float* hrls,
                                     const float* albedo, const float* normal, const float* target,
                                     int32_t N, int32_t H, int32_t W, int32_t scale, float lr,
                                     int32_t precision, double* loss_out, void* stream)
{
    return mrs_train_step_extra(net, lrhs, hrls, albedo, normal, nullptr, target, N, H, W, scale,
                                lr, precision, loss_out, stream);
}

extern "C" mrs_status mrs_train_step_extra(mrs_net net, const float* lrhs, const float* hrls,
                                           const float* albedo, const float* normal,
                                           const float* extra, const float* target, int32_t N,
                                           int32_t H, int32_t W, int32_t scale, float lr,
                                           int32_t precision, double* loss_out, void* stream)
{
    MRS_ARG(net != nullptr, "net is NULL");
    MRS_ARG(lrhs && hrls && albedo && normal && target, "NULL image pointer");
    MRS_ARG((extra != nullptr) == (net->cin0 == 21),
            "extra layers must be given exactly for a net with MRS_NET_NPARAMS_EXTRA parameters");
    MRS_ARG(scale == 1 || scale == 2 || scale == 4 || scale == 8, "scale must be 1, 2, 4 or 8");
    MRS_ARG(N >= 1 && H >= 1 && W >= 1 && H % scale == 0 && W % scale == 0, "bad sizes");
    MRS_ARG((int64_t)N * H * W <= (int64_t(1) << 22), "training batch exceeds 2^22 pixels");
    MRS_ARG(lr >= 0.0f, "lr < 0");
    MRS_ARG(precision == MRS_PREC_FP32 || precision == MRS_PREC_BF16,
            "training precision must be MRS_PREC_FP32 or MRS_PREC_BF16");
    if (precision == MRS_PREC_BF16)
        return train_step_bf16(net, lrhs, hrls, albedo, normal, extra, target, N, H, W, scale, lr,
                               loss_out, (cudaStream_t)stream);
    return train_step_f32(net, lrhs, hrls, albedo, normal, extra, target, N, H, W, scale, lr,
                          loss_out, (cudaStream_t)stream);
}

extern "C" mrs_status mrs_net_get_grads(mrs_net net, float* grads)
{
    MRS_ARG(net && grads, "NULL argument");
    MRS_CHECK(cudaMemcpy(grads, net->grad, net->np * 4, cudaMemcpyDeviceToHost));
    return MRS_OK;
}

extern "C" mrs_status mrs_net_get_state(mrs_net net, float* params, float* adam_m, float* adam_v,
                                        int64_t* step)
{
    MRS_ARG(net && params && adam_m && adam_v && step, "NULL argument");
    MRS_CHECK(cudaMemcpy(params, net->master, net->np * 4, cudaMemcpyDeviceToHost));
    MRS_CHECK(cudaMemcpy(adam_m, net->adam_m, net->np * 4, cudaMemcpyDeviceToHost));
    MRS_CHECK(cudaMemcpy(adam_v, net->adam_v, net->np * 4, cudaMemcpyDeviceToHost));
    *step = net->step;
    return MRS_OK;
}

extern "C" mrs_status mrs_net_set_state(mrs_net net, const float* params, const float* adam_m,
                                        const float* adam_v, int64_t step)
{
    MRS_ARG(net && params && adam_m && adam_v, "NULL argument");
    MRS_ARG(step >= 0, "step < 0");
    MRS_CHECK(cudaMemcpy(net->master, params, net->np * 4, cudaMemcpyHostToDevice));
    MRS_CHECK(cudaMemcpy(net->adam_m, adam_m, net->np * 4, cudaMemcpyHostToDevice));
    MRS_CHECK(cudaMemcpy(net->adam_v, adam_v, net->np * 4, cudaMemcpyHostToDevice));
    net->step = step;
    net->bf_valid = net->f8_valid = net->xscale_valid = net->bfT_valid = net->simt_valid = false;
    return MRS_OK;
}

// ---- checkpoints and seeded initialisation ----------------------------------
namespace mrs {
namespace {

static_assert(__BYTE_ORDER__ == __ORDER_LITTLE_ENDIAN__, "checkpoint I/O assumes a little-endian host");

constexpr char kCkptMagic[8] = {'M', 'R', 'S', 'N', 'E', 'T', 'v', '2'};
constexpr uint32_t kCkptVersion = 2;

// header of a checkpoint file (64 bytes, little-endian, no padding)
struct CkptHeader {
    char magic[8];
    uint32_t header_bytes;   // 64
    uint32_t version;        // 2
    int64_t n_params;
    int64_t step;
    uint64_t seed;           // the caller's data / RNG seed, stored for resume
    int32_t input_channels;  // 12 or 21
    int32_t loss;            // MRS_LOSS_*
    float beta;
    uint32_t reserved;
    uint64_t checksum;       // FNV-1a 64 over the three float arrays' bytes
};
static_assert(sizeof(CkptHeader) == 64, "checkpoint header layout");

uint64_t fnv1a(uint64_t h, const void* data, size_t n)
{
    const unsigned char* p = (const unsigned char*)data;
    for (size_t i = 0; i < n; ++i) { h ^= p[i]; h *= 0x100000001B3ull; }
    return h;
}

// splitmix64 (Steele, Lea, Flood 2014): the initialiser's uniform stream
uint64_t splitmix64(uint64_t& x)
{
    uint64_t z = (x += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// zero-mean, unit-variance approximately normal draw: the sum of 12
// uniforms minus 6 (Irwin-Hall), integer and IEEE arithmetic only, so that
// the same seed gives the same weights on every host
double normal12(uint64_t& x)
{
    double s = 0.0;
    for (int i = 0; i < 12; ++i) s += (double)(splitmix64(x) >> 11) * (1.0 / 9007199254740992.0);
    return s - 6.0;
}

}  // namespace
}  // namespace mrs

extern "C" mrs_status mrs_net_save(mrs_net net, const char* path, uint64_t seed)
{
    using namespace mrs;
    MRS_ARG(net != nullptr && path != nullptr, "NULL argument");
    std::vector<float> host(3 * net->np);
    int64_t step = 0;
    mrs_status rc = mrs_net_get_state(net, host.data(), host.data() + net->np,
                                      host.data() + 2 * net->np, &step);
    if (rc != MRS_OK) return rc;
    CkptHeader h;
    memset(&h, 0, sizeof(h));
    memcpy(h.magic, kCkptMagic, 8);
    h.header_bytes = sizeof(CkptHeader);
    h.version = kCkptVersion;
    h.n_params = (int64_t)net->np;
    h.step = step;
    h.seed = seed;
    h.input_channels = net->cin0;
    h.loss = net->loss_kind;
    h.beta = net->loss_beta;
    h.checksum = fnv1a(0xCBF29CE484222325ull, host.data(), host.size() * 4);
    std::string tmp = std::string(path) + ".tmp";
    FILE* f = fopen(tmp.c_str(), "wb");
    if (!f) { set_error("cannot open %s for writing", tmp.c_str()); return MRS_ERR_IO; }
    bool ok = fwrite(&h, sizeof(h), 1, f) == 1 && fwrite(host.data(), 4, host.size(), f) == host.size();
    ok = (fclose(f) == 0) && ok;
    if (!ok || rename(tmp.c_str(), path) != 0) {
        remove(tmp.c_str());
        set_error("writing checkpoint %s failed", path);
        return MRS_ERR_IO;
    }
    return MRS_OK;
}

extern "C" mrs_status mrs_net_load(mrs_net net, const char* path, uint64_t* seed)
{
    using namespace mrs;
    MRS_ARG(net != nullptr && path != nullptr, "NULL argument");
    FILE* f = fopen(path, "rb");
    if (!f) { set_error("cannot open %s", path); return MRS_ERR_IO; }
    CkptHeader h;
    std::vector<float> host;
    mrs_status rc = MRS_OK;
    if (fread(&h, sizeof(h), 1, f) != 1 || memcmp(h.magic, kCkptMagic, 8) != 0 ||
        h.header_bytes != sizeof(CkptHeader) || h.version != kCkptVersion) {
        set_error("%s is not a version-%u fusion-network checkpoint", path, kCkptVersion);
        rc = MRS_ERR_FORMAT;
    } else if (h.n_params != (int64_t)net->np || h.input_channels != net->cin0) {
        set_error("checkpoint holds %lld parameters (%d input channels), the net %zu (%d)",
                  (long long)h.n_params, h.input_channels, net->np, net->cin0);
        rc = MRS_ERR_FORMAT;
    } else if ((h.loss != MRS_LOSS_L1LOG && h.loss != MRS_LOSS_ROBUST) || !(h.beta > 0.0f) ||
               h.step < 0) {
        set_error("checkpoint %s has an invalid loss, beta or step", path);
        rc = MRS_ERR_FORMAT;
    } else {
        host.resize(3 * net->np);
        if (fread(host.data(), 4, host.size(), f) != host.size() || fgetc(f) != EOF) {
            set_error("checkpoint %s is truncated or has trailing bytes", path);
            rc = MRS_ERR_FORMAT;
        } else if (fnv1a(0xCBF29CE484222325ull, host.data(), host.size() * 4) != h.checksum) {
            set_error("checkpoint %s fails its checksum", path);
            rc = MRS_ERR_FORMAT;
        }
    }
    fclose(f);
    if (rc != MRS_OK) return rc;
    rc = mrs_net_set_state(net, host.data(), host.data() + net->np, host.data() + 2 * net->np, h.step);
    if (rc != MRS_OK) return rc;
    net->loss_kind = h.loss;
    net->loss_beta = h.beta;
    if (seed) *seed = h.seed;
    return MRS_OK;
}

extern "C" mrs_status mrs_net_create_seeded(int32_t input_channels, uint64_t init_seed,
                                            float resid_gain, mrs_net* out)
{
    using namespace mrs;
    MRS_ARG(out != nullptr, "out is NULL");
    *out = nullptr;
    MRS_ARG(input_channels == 12 || input_channels == 21, "input_channels must be 12 or 21");
    MRS_ARG(resid_gain >= 0.0f && resid_gain <= 1.0f, "resid_gain must be in [0, 1]");
    const auto& L = shapes(input_channels);
    size_t np = input_channels == 21 ? kParams21 : kParams12;
    std::vector<float> p(np, 0.0f);
    uint64_t x = init_seed ^ 0x6D72732D6E657430ull;
    for (int l = 0; l < kLayers; ++l) {
        if (l == kLayers - 1) break;   // the 3-channel head starts at zero
        double sd = sqrt(2.0 / (9.0 * L[l].cin));
        if (l >= 1 && l % 2 == 0) sd *= resid_gain;   // second conv of a residual block
        for (size_t i = 0; i < (size_t)L[l].cout * 9 * L[l].cin; ++i)
            p[L[l].woff + i] = (float)(sd * normal12(x));
    }
    return mrs_net_create(p.data(), (int32_t)np, out);
}

extern "C" mrs_status mrs_selftest_wait_timeout(int32_t limit_us, void* stream)
{
    MRS_ARG(limit_us >= 1 && limit_us <= 100000, "limit_us must be in [1, 100000]");
    int clk_khz = 0, dev = 0;
    MRS_CHECK(cudaGetDevice(&dev));
    MRS_CHECK(cudaDeviceGetAttribute(&clk_khz, cudaDevAttrClockRate, dev));
    long long cycles = (long long)limit_us * (clk_khz > 0 ? clk_khz : 2000000) / 1000;
    int gave_up = 0;
    mrs_status rc = tc_wait_selftest(cycles, &gave_up, (cudaStream_t)stream);
    if (rc != MRS_OK) return rc;
    if (gave_up) {
        set_error("device wait gave up after %d us (self-test)", limit_us);
        return MRS_ERR_TIMEOUT;
    }
    return MRS_OK;
}

extern "C" mrs_status mrs_gate_async(const float* fused, const float* lrhs, const float* plain,
                                     int32_t N, int32_t H, int32_t W, int32_t scale, double tau,
                                     float* out, int32_t* used_plain, double* D, void* stream)
{
    MRS_ARG(fused && lrhs && out && used_plain, "NULL pointer");
    MRS_ARG(scale >= 1 && N >= 1 && H >= scale && W >= scale && H % scale == 0 && W % scale == 0,
            "bad sizes");
    cudaStream_t st = (cudaStream_t)stream;
    static std::mutex mu;
    static Buf parts;
    std::lock_guard<std::mutex> g(mu);
    mrs_status rc = parts.ensure(sizeof(double) * kRedBlocks);
    if (rc != MRS_OK) return rc;
    k_gate_partial<<<kRedBlocks, 256, 0, st>>>(fused, lrhs, N, H, W, scale, parts.as<double>());
    MRS_LAUNCHED(1);
    k_gate_decide<<<1, 256, 0, st>>>(parts.as<double>(), kRedBlocks,
                                    (double)N * (H / scale) * (W / scale) * 3, tau,
                                    plain ? 1 : 0, used_plain, D);
    MRS_LAUNCHED(1);
    size_t n = (size_t)N * H * W * 3;
    k_gate_select<<<1024, 256, 0, st>>>(fused, plain ? plain : fused, n, used_plain, out);
    MRS_LAUNCHED(1);
    return cuda_status(cudaGetLastError(), "gate_async launch");
}

extern "C" mrs_status mrs_conv3x3_wgrad(const float* x, const float* dy, int32_t N, int32_t H,
                                        int32_t W, int32_t cin, int32_t cout, int32_t precision,
                                        float* dw, float* db, void* stream)
{
    using namespace mrs;
    MRS_ARG(x && dy && dw && db, "NULL pointer");
    MRS_ARG(N >= 1 && H >= 1 && W >= 1, "sizes must be >= 1");
    MRS_ARG(cin >= 1 && cin <= 64 && cout >= 1 && cout <= 64, "cin, cout must be in [1, 64]");
    MRS_ARG(precision == MRS_PREC_FP32 || precision == MRS_PREC_BF16, "precision must be FP32 or BF16");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t P = (size_t)N * H * W;
    const size_t nw = (size_t)cout * 9 * cin;
    const size_t maxp = (size_t)std::max(kDwSplits, sm_count());
    Scratch& S = scratch();
    std::lock_guard<std::mutex> g(S.mu);
    size_t need = (nw + cout) * 4 + maxp * (9 * 64 * 64 + 64) * 4 + 4096 +
                  (precision == MRS_PREC_BF16 ? 2 * P * 128 : 0);
    mrs_status rc = S.b.ensure(need);
    if (rc != MRS_OK) return rc;
    float* gw = S.b.as<float>();
    float* gb = gw + nw;
    float* part = (float*)(((uintptr_t)(gb + cout) + 255) & ~(uintptr_t)255);
    float* dbpart = part + maxp * 9 * 64 * 64;
    static int* err = nullptr;
    if (!err) { MRS_CHECK(cudaMalloc(&err, 4)); MRS_CHECK(cudaMemset(err, 0, 4)); }
    int np = 0;
    if (precision == MRS_PREC_FP32) {
        launch_dw(dim3(kDwSplits, 9), x, cin, cin, dy, cout, cout, N, H, W, part, dbpart, 0, 1, st);
        MRS_LAUNCHED(1);
        np = kDwSplits;
    } else {
        uint8_t* xq = (uint8_t*)(((uintptr_t)(dbpart + maxp * 64) + 1023) & ~(uintptr_t)1023);
        uint8_t* dq = xq + P * 128;
        k_to_operand<<<1024, 256, 0, st>>>(x, P, cin, xq, 0, 1.0f);
        MRS_LAUNCHED(1);
        k_to_operand<<<1024, 256, 0, st>>>(dy, P, cout, dq, 0, 1.0f);
        MRS_LAUNCHED(1);
        WgTile t;
        if ((rc = tc_make_wg_x_map(&t.x, xq, N, H, W, 128, 128LL * W, 128LL * W * H)) != MRS_OK) return rc;
        if ((rc = tc_make_wg_dy_map(&t.dy, dq, N, H, W, 128, 128LL * W, 128LL * W * H)) != MRS_OK) return rc;
        t.N = N; t.H = H; t.W = W; t.cin = cin; t.cout = cout; t.runs = sm_count();   // np partials at most
        if ((rc = tc_conv3x3_wgrad(t, part, dbpart, &np, err, st)) != MRS_OK) return rc;
    }
    const size_t gstride = precision == MRS_PREC_FP32 ? nw : (size_t)kWgPart;
    k_dw_reduce<<<(int)((nw + cout + 31) / 32), 256, 0, st>>>(part, dbpart, np, gstride,
                                                              precision == MRS_PREC_FP32 ? cout : 64, cin, cout, gw, gb);
    MRS_LAUNCHED(1);
    MRS_CHECK(cudaMemcpyAsync(dw, gw, nw * 4, cudaMemcpyDeviceToHost, st));
    MRS_CHECK(cudaMemcpyAsync(db, gb, cout * 4, cudaMemcpyDeviceToHost, st));
    MRS_CHECK(cudaStreamSynchronize(st));
    int herr = 0;
    MRS_CHECK(cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost));
    if (herr) { cudaMemset(err, 0, 4); set_error("tensor-core weight-gradient wait timed out"); return MRS_ERR_TIMEOUT; }
    return MRS_OK;
}

extern "C" mrs_status mrs_conv3x3_dgrad(const float* dy, int32_t N, int32_t H, int32_t W,
                                        int32_t cin, int32_t cout, const float* w, int32_t mode,
                                        const float* aux, int32_t precision, float* out,
                                        void* stream)
{
    using namespace mrs;
    MRS_ARG(dy && w && out, "NULL pointer");
    MRS_ARG(N >= 1 && H >= 1 && W >= 1, "sizes must be >= 1");
    MRS_ARG(cin >= 1 && cin <= 64 && cout >= 1 && cout <= 64, "cin, cout must be in [1, 64]");
    MRS_ARG(mode == MRS_DGRAD_LINEAR || mode == MRS_DGRAD_RELU_MASK || mode == MRS_DGRAD_RESIDUAL,
            "unknown mode");
    MRS_ARG(mode == MRS_DGRAD_LINEAR || aux != nullptr, "aux is required by this mode");
    MRS_ARG(precision == MRS_PREC_FP32 || precision == MRS_PREC_BF16, "precision must be FP32 or BF16");
    MRS_ARG((int64_t)N * H * W <= (int64_t(1) << 26), "more than 2^26 pixels");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t P = (size_t)N * H * W;
    const size_t nw = (size_t)cout * 9 * cin;
    Scratch& S = scratch();
    std::lock_guard<std::mutex> g(S.mu);
    const size_t opb = ((P * 128 + 1023) / 1024) * 1024;   // one bf16 [P][64] operand
    size_t need = nw * 4 + 64 * 4 + 2048 + 9 * 64 * 64 * 4 + 1024 +
                  (precision == MRS_PREC_BF16 ? 3 * opb : 0);
    mrs_status rc = S.b.ensure(need);
    if (rc != MRS_OK) return rc;
    float* dw = S.b.as<float>();
    float* zero = dw + nw;
    uint8_t* q = (uint8_t*)(((uintptr_t)(zero + 64) + 1023) & ~(uintptr_t)1023);
    MRS_CHECK(cudaMemcpyAsync(dw, w, nw * 4, cudaMemcpyHostToDevice, st));
    MRS_CHECK(cudaMemsetAsync(zero, 0, 64 * 4, st));
    if (precision == MRS_PREC_FP32) {
        // the FP32 training step's transposed conv: flipped, transposed
        // weights through the SIMT convolution with the step's epilogues
        float* wt = (float*)q;
        if ((rc = simt_pack(dw, cin, cout, 1, wt, st)) != MRS_OK) return rc;
        int sm = mode == MRS_DGRAD_LINEAR ? SIMT_PLAIN : mode == MRS_DGRAD_RELU_MASK ? SIMT_MASK : SIMT_RESID;
        rc = conv_simt(dy, cout, wt, zero, cin, sm, 0, aux, out, nullptr, N, H, W, 1, st);
        if (rc == MRS_OK) rc = cuda_status(cudaStreamSynchronize(st), "conv3x3 dgrad sync");
        return rc;
    }
    // BF16: the tensor-core conv with the training step's transposed-weight
    // packing and epilogue modes (linear; ReLU mask by the layer's output;
    // residual added in place into the incoming gradient)
    __nv_bfloat16* wp = (__nv_bfloat16*)q;
    uint8_t* dyq = q + ((9 * 64 * 64 * 2 + 1023) / 1024) * 1024;
    uint8_t* auxq = dyq + opb;
    uint8_t* outq = auxq + opb;
    static int* err = nullptr;
    if (!err) { MRS_CHECK(cudaMalloc(&err, 4)); MRS_CHECK(cudaMemset(err, 0, 4)); }
    k_pack_bf16_T<<<(9 * 64 * 64 + 255) / 256, 256, 0, st>>>(dw, 0, cin, cout, 64, wp);
    MRS_LAUNCHED(1);
    k_to_operand<<<1024, 256, 0, st>>>(dy, P, cout, dyq, 0, 1.0f);
    MRS_LAUNCHED(1);
    if (mode == MRS_DGRAD_RELU_MASK) {
        k_to_operand<<<1024, 256, 0, st>>>(aux, P, cin, auxq, 0, 1.0f);
        MRS_LAUNCHED(1);
    } else if (mode == MRS_DGRAD_RESIDUAL) {
        k_to_operand<<<1024, 256, 0, st>>>(aux, P, cin, outq, 0, 1.0f);
        MRS_LAUNCHED(1);
    }
    CUtensorMap ma, mo, mr, mw;
    if ((rc = tc_make_w_map(&mw, wp, 9 * 64, 64, TC_BF16)) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&ma, dyq, N, H, W, TC_BF16, tc_a_box(TC_BF16))) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&mo, outq, N, H, W, TC_BF16, tc_out_box(TC_BF16))) != MRS_OK) return rc;
    if ((rc = tc_make_act_map(&mr, auxq, N, H, W, TC_BF16, tc_out_box(TC_BF16))) != MRS_OK) return rc;
    TcConvArgs a;
    memset(&a, 0, sizeof(a));
    a.tmap_x = &ma; a.tmap_w = &mw; a.bias = zero; a.tmap_out = &mo;
    a.N = N; a.H = H; a.W = W; a.scale = 1; a.nout = 64; a.operand = TC_BF16; a.err = err;
    if (mode == MRS_DGRAD_LINEAR) { a.mode = TC_LIN_BF16; }
    else if (mode == MRS_DGRAD_RELU_MASK) { a.mode = TC_MASK_BF16; a.tmap_res = &mr; }
    else { a.mode = TC_RESID_BF16; a.tmap_res = &mo; }
    if ((rc = tc_conv3x3(a, st)) != MRS_OK) return rc;
    k_from_operand<<<1024, 256, 0, st>>>((const __nv_bfloat16*)outq, P, cin, out);
    MRS_LAUNCHED(1);
    rc = cuda_status(cudaStreamSynchronize(st), "conv3x3 dgrad sync");
    int herr = 0;
    if (rc == MRS_OK) {
        MRS_CHECK(cudaMemcpy(&herr, err, 4, cudaMemcpyDeviceToHost));
        if (herr) { cudaMemset(err, 0, 4); set_error("tensor-core conv wait timed out"); return MRS_ERR_TIMEOUT; }
    }
    return rc;
}

extern "C" mrs_status mrs_conv_set_ring(int32_t stages)
{
    MRS_ARG(stages == 0 || (stages >= 3 && stages <= 12), "stages must be 0 or in [3, 12]");
    mrs::tc_set_ring(stages);
    return MRS_OK;
}

extern "C" mrs_status mrs_net_set_loss(mrs_net net, int32_t loss, float beta)
{
    MRS_ARG(net != nullptr, "net is NULL");
    MRS_ARG(loss == MRS_LOSS_L1LOG || loss == MRS_LOSS_ROBUST, "unknown loss");
    MRS_ARG(beta > 0.0f && beta < 1e30f, "beta must be positive and finite");
    net->loss_kind = loss;
    net->loss_beta = beta;
    return MRS_OK;
}

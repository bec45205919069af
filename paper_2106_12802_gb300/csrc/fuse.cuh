// Internal interface shared by the fusion-network translation units (fuse.cu:
// the all-high-resolution network, metrics and gate; rdn.cu: the method's own
// two-encoder network of Sec. 4).
#pragma once

#include "common.cuh"

namespace mrs {

// Epilogues of the FP32 SIMT 3x3 convolution
enum SimtMode {
    SIMT_PLAIN = 0,    // out = acc + b (optional ReLU)
    SIMT_RESID = 1,    // out = res + (acc + b)
    SIMT_FINAL = 2,    // out[p][c < 3] = (acc + b) + bilinear_up(lrhs)[p]
    SIMT_MASK = 3,     // out = res > 0 ? acc + b : 0
    SIMT_RESRELU = 4,  // out = res + relu(acc + b)
};

// whether launches on st are being recorded: what they would write does not
// exist yet when the recording call returns
inline bool recording(cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}

// device memory may be allocated while a stream of this thread is being recorded
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// FP32 3x3 convolution with zero padding 1 on [N][H][W][.] tensors:
// out[p][o] (o < cout, pixel stride os) from x[p][c] (c < cin, pixel stride
// xs) with the weights that simt_pack packed (16-byte aligned,
// simt_pack_floats(cin, cout) floats); res has pixel stride rs.  Asynchronous
// on st.
size_t simt_pack_floats(int cin, int cout);
// w [cout][9][cin]; transposed: for the gradient with respect to the input
// (inputs cout, outputs cin, taps flipped; simt_pack_floats(cout, cin) floats)
mrs_status simt_pack(const float* w, int cin, int cout, int transposed, float* wp, cudaStream_t st);
// a network's layers in one launch (each w [cout][9][cin] into its wp): a
// recorded call holds it, and replays it with the call
struct SimtLayers {
    static constexpr int kMax = 72;
    struct Layer { const float* w; float* wp; int cin, cout, cop; } layer[kMax];
    int n = 0;
    size_t largest = 0;            // floats of the largest wp
    bool add(const float* w, int cin, int cout, float* wp);
};
mrs_status simt_pack_layers(const SimtLayers& p, cudaStream_t st);
mrs_status simt_conv3x3(const float* x, int cin, int xs, const float* wp, const float* b, int cout,
                        int mode, int relu, const float* res, int rs, float* out, int os,
                        const float* lrhs, int N, int H, int W, int s, cudaStream_t st);

// ---- FP32 training launches (fuse.cu), asynchronous on st ------------------
constexpr int kDwParts = 64;       // pixel-split partial sums of dw_tiles_f32
constexpr int kLossParts = 1024;   // float64 partial sums of loss_grad_f32

// Weight / bias gradient partial sums of a convolution with zero padding 1:
// x [P][xs] (first cin channels), dy [P][ys] (first cout), any cin / cout, in
// 64 x 64 channel tiles z = ot * ceil(cin / 64) + ct.  part holds
// [z][kDwParts][ntaps][64 * 64] floats (ntaps = 9, or 1 when centre_only: the
// centre tap alone, a 1x1 conv), tile z's tap j at part[z][g][j] as
// [cout_t][cin_t];
// dbpart holds [ot][kDwParts * 64] floats, [g][cout_t] packed.  The sums over
// g are left to the caller.
mrs_status dw_tiles_f32(const float* x, int cin, int xs, const float* dy, int cout, int ys, int N,
                        int H, int W, int centre_only, float* part, float* dbpart, cudaStream_t st);
// training loss (MRS_LOSS_*) of y against min(target, clip) over n values:
// dy = dL/dy, *sum (device double) = the sum of the per-value losses,
// parts = kLossParts doubles of scratch
mrs_status loss_grad_f32(const float* y, const float* tgt, size_t n, float clip, int kind,
                         float beta, float* dy, double* parts, double* sum, cudaStream_t st);
// one bias-corrected Adam update (beta1 0.9, beta2 0.999, eps 1e-8) at step `step` (>= 1)
mrs_status adam_f32(float* p, const float* g, float* m, float* v, size_t n, float lr, int64_t step,
                    cudaStream_t st);

// ---- BF16 training: weight-gradient tiles into the gradient (fuse.cu) --------
// Where the sums of tile t of tc_conv3x3_wgrad's partials go: the gradient of
// a layer [cout][KK][CIN] at grad + gw (KK = 9, or 1 for a 1x1 layer: the tile's
// centre tap) and its bias at grad + gb.  Tile output o is layer output
// o_mul o + o_add, tile input c layer input c0 + c, or, for chunk q >= 1 of a
// deshuffled input (D steps, scale s), 64 + the deshuffled channel of (c, view
// q - 1).  Partials 8 t .. 8 t + np - 1, summed in that order (np <= 8).
struct WgRed {
    int cin, cout, KK, CIN, o_mul, o_add, c0, q, s, D, with_bias, np;
    long long gw, gb;
};
// d_reds: ntiles entries in device memory
mrs_status wg_reduce(const WgRed* d_reds, int ntiles, const float* part, const float* dbpart, float* grad,
                     cudaStream_t st);
// channel of the D-times deshuffled map that holds channel c of HR sub-pixel
// (oy, ox) of each s x s block: c s^2 + sum over steps d = 1..D of
// (2 dy_d + dx_d) 4^(D - d), dy_d / dx_d bit d - 1 of oy / ox
__host__ __device__ __forceinline__ int dsf_channel(int c, int oy, int ox, int D)
{
    int k = c;
    for (int d = 1; d <= D; ++d) k = 4 * k + 2 * ((oy >> (d - 1)) & 1) + ((ox >> (d - 1)) & 1);
    return k;
}

}  // namespace mrs

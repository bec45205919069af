// Tensor-core 3x3 convolution (implicit GEMM on tcgen05) used by the fusion
// network: internal interface between conv_tc.cu and fuse.cu.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <vector>

#include "common.cuh"

namespace mrs {

// Epilogue modes of the tensor-core convolution
enum TcMode : int {
    TC_RELU_BF16 = 0,   // out_bf16[p][64] = relu(acc + b)
    TC_RESID_BF16 = 1,  // out_bf16[p][64] = res[p] + (acc + b)   (res may alias out)
    TC_FINAL_F32 = 2,   // out_f32[p][3]  = (acc + b) + bilinear_up(lrhs)[p]
    TC_PLAIN_F32 = 3,   // out_f32[p][cout] = acc + b, optional relu
    TC_LIN_BF16 = 4,    // out_bf16[p][64] = acc + b
    TC_MASK_BF16 = 5,   // out_bf16[p][64] = mask[p] > 0 ? acc + b : 0   (mask via tmap_res)
    TC_RESRELU_BF16 = 6,// out_bf16[p][64] = res[p] + relu(acc + b)
};

enum TcOperand : int { TC_BF16 = 0, TC_FP8 = 1 };

struct TcConvBase {
    const CUtensorMap* tmap_x;   // A operand [N][H][W][64] (bf16 or fp8, kABox-pixel boxes)
    const CUtensorMap* tmap_res; // TC_RESID_BF16 residual (bf16, kOutBox-pixel boxes)
    const CUtensorMap* tmap_out; // TC_RELU_BF16 / TC_RESID_BF16 output (bf16, kOutBox-pixel boxes)
    const CUtensorMap* tmap_w;   // packed weights [9 * nout][64]
    const float* bias;           // [nout] (padded)
    const float* wscale;         // fp8 only: per-output-channel dequant scale (may be NULL)
    float xscale;                // fp8 only: activation dequant scale
    const void* res;             // TC_RESID_BF16 residual (bf16 [p][64])
    void* out;                   // output
    const float* lrhs;           // TC_FINAL_F32: [N][h][w][3]
    int N, H, W, scale;
    int nout;                    // 64 or 16 (MMA N)
    int cout;                    // valid output channels (TC_PLAIN_F32 / TC_FINAL_F32)
    int relu;                    // TC_PLAIN_F32
    int mode;
    int operand;                 // TC_BF16 / TC_FP8
    int* err;                    // device error word (timeouts)
    // TC_RELU_BF16 / TC_RESID_BF16 with fp8 operands: also emit the fp8 copy
    void* out_fp8;
    float out_fp8_inv_scale;
    // with out_fp8: write only the fp8 copy (the bf16 result has no reader)
    int fp8_only;
    // A convolution over kc > 1 input tensors of 64 channels each (the
    // concatenation of their channels) in ONE launch: amaps = DEVICE array of
    // kc A-operand maps (64-byte aligned, alive until the kernel completes),
    // weights of chunk j at rows w_row0 + (9 j + t) nout of tmap_w.  kc <= 1:
    // tmap_x, weights at rows w_row0 + t nout.
    const CUtensorMap* amaps;
    int kc;
    int w_row0;
};

// (kept apart: the kernels that know none of it take the short parameter block)
struct TcConvArgs : TcConvBase {
    // ng > 1 convolutions of ONE input in one launch (bf16 results, kc <= 1): the
    // CTAs are shared out among them.  Group g takes the weights at rows
    // w_row0 + 9 g nout, the bias at bias + 64 g where gbias is set, mode
    // gmode[min(g, 3)], and its residual and output maps from the device array
    // gmaps [2 g], [2 g + 1] (64-byte aligned, alive until the kernel completes)
    int ng;
    int gbias;
    int gmode[4];
    const CUtensorMap* gmaps;
    // TC_RESID_BF16 (of the last group): the sum is kept where mask[p] > 0, else 0
    const void* mask;            // bf16 [p][64], or NULL
    // a second bf16 result of bf16 modes, ng <= 1: out2 = x2 > 0 ? out : 0 (op2 = 1)
    // or x2 + out (op2 = 2)
    int op2;
    const void* x2;              // bf16 [p][64]
    void* out2;
};

// Box widths (pixels): the conv reads one 130-pixel A box per input row (a
// tile's 128 outputs plus a halo pixel on each side) and moves 128-pixel
// residual / output boxes.  Maps passed to tc_conv3x3 use these widths (the
// same for both operand types).
constexpr int kABox = 130;
constexpr int kOutBox = 128;
inline int tc_a_box(int /*operand*/) { return kABox; }
inline int tc_out_box(int /*operand*/) { return kOutBox; }
// Images of up to 62 pixels' width share a tile: a box then holds this many of
// them, W + 2 pixels each, and an output pixel x of the i-th is the tile's row
// i (W + 2) + x (the halo columns between them are nobody's output).  The map
// functions below make such boxes where kABox or kOutBox is asked for.
// A layer of 16 crops of 48 x 48 fills 96 of a tile's 128 rows instead of 48
// and takes 384 tiles instead of 768: the convolutions of a two-encoder
// training step 5.63 -> 4.34 ms.  63 pixels and more leave no room for a second
// image; a tile of one costs what it did.
__host__ __device__ inline int tc_images(int N, int W)
{
    const int k = kOutBox / (W + 2);
    return k < 2 || N < 2 ? 1 : (k < N ? k : N);
}
// Encode a tiled tensor map for a [N][H][W][64] activation tensor (rows of 128
// bytes in bf16, 64 in fp8): box = box_px pixels of one image row.
mrs_status tc_make_act_map(CUtensorMap* m, const void* ptr, int N, int H, int W, int operand,
                           int box_px = 128);
// Tensor map for a strided view of a bf16 activation tensor: element (x, y, n)
// of the view is the 64-channel row at ptr + x * px_stride + y * row_stride +
// n * img_stride (bytes, multiples of 16).  Views select a sub-pixel grid of
// a larger image (a deshuffle chunk as an A operand, or a shuffle target as
// an output) without moving data.
mrs_status tc_make_view_map(CUtensorMap* m, const void* ptr, int N, int H, int W,
                            long long px_stride, long long row_stride, long long img_stride,
                            int box_px, int box_rows = 1);
// Tensor map for packed weights [rows][64 (bf16) | 64 (fp8)].
mrs_status tc_make_w_map(CUtensorMap* m, const void* ptr, int rows, int nout, int operand);

mrs_status tc_conv3x3(const TcConvArgs& a, cudaStream_t st);
// input-row ring depth of every later conv launch (0: the most that fits)
void tc_set_ring(int stages);

// Weight and bias gradients of 3x3 convs (zero padding 1) on the tensor cores:
// one launch over a list of tiles (a tile: one conv's up to 64 x 64 channels),
//   dw[o][t][c] (t = ky * 3 + kx) = sum over pixels p of
//       dy[p][o] * x[p + (ky - 1, kx - 1)][c],   db[o] = sum dy[p][o]
// for o < cout, c < cin.  A tile's jobs (kWgKB pixels of one row; strips, then
// rows, then images) are cut into `runs` equal contiguous runs, each summed on
// the tensor cores; runs w, w + C, ... (class w of C = `classes`) are added in
// FP32 in that order and written as partial w of the tile's np = min(runs, C):
//   part[(slot + w) * kWgPart + (tap * cout + o) * cin + c], dbpart[(slot + w) * 64 + o]
// (slot: C times the tile's number).  The sums' order depends on the tiles alone.
// C = 8 leaves few partials of a list; one tile alone takes C = runs, whose units
// of work are enough for every SM.
constexpr int kWgKB = 64;          // pixels per job
constexpr int kWgPart = 9 * 64 * 64;
struct WgTile {
    CUtensorMap x, dy;             // tc_make_wg_x_map / tc_make_wg_dy_map
    int N, H, W, cin, cout;
    int runs;                      // at most the tile's jobs are used
};
struct WgPlan {
    int ntiles = 0, ctas = 0, units = 0, classes = 8;
    std::vector<int> np;           // per tile: its partials
    std::vector<uint8_t> blob;     // what the kernel reads: upload to 64-byte aligned device memory
    size_t part_floats() const { return (size_t)ntiles * classes * kWgPart; }
    size_t dbpart_floats() const { return (size_t)ntiles * classes * 64; }
};
mrs_status tc_wgrad_plan(const std::vector<WgTile>& tiles, int classes, WgPlan& plan);
// bytes of a plan's blob at most
size_t tc_wgrad_blob_max(int ntiles, int classes);
mrs_status tc_conv3x3_wgrad(const WgPlan& plan, const void* d_blob, float* part, float* dbpart,
                            int* err, cudaStream_t st);
// One tile alone, without a plan: C = its runs, *np of them
mrs_status tc_conv3x3_wgrad(const WgTile& tile, float* part, float* dbpart, int* np, int* err, cudaStream_t st);
// Operand maps of a tile: [N][H][W][64] bf16 with the given strides (bytes)
// between pixels, rows and images (as tc_make_view_map).
mrs_status tc_make_wg_x_map(CUtensorMap* m, const void* ptr, int N, int H, int W, long long px_stride,
                            long long row_stride, long long img_stride);
mrs_status tc_make_wg_dy_map(CUtensorMap* m, const void* ptr, int N, int H, int W, long long px_stride,
                             long long row_stride, long long img_stride);

// Launches a kernel whose bounded mbarrier wait can never complete; *gave_up
// = 1 if the wait gave up after limit_cycles and raised the error word.
mrs_status tc_wait_selftest(long long limit_cycles, int* gave_up, cudaStream_t st);

}  // namespace mrs

// Tensor-core path of the dense layers (tensor.cu): interface to the launchers in conv.cu.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#include <cuda.h>
#endif

#include "layer.h"

namespace patconv {

// How one call runs on the tensor cores: the tile, the filter chunk and the channel split.
struct TensorPlan {
    int MT = 1;             // 128-position tiles per CTA (1, 2 or 4); MT * NC <= 256
    int NC = 0;             // filters per unit (a multiple of 16)
    int KS = 1;             // input-channel splits (KS > 1: fp32 partial sums in the workspace)
    int n_cb = 0, cb_split = 0;   // 16-channel blocks, blocks per split
    int ll = 0;             // fp32: the products of the lo parts too
    int Wp = 0, Ip = 0;     // position pitch of a row, of an image (flat tiles)
    long long Q = 0;        // flat tiles: positions of the padded output grid
    int mstep = 0;          // flat tiles: positions a tile advances
    int P = 0;              // positions a tile stages
    int vec = 1, ppr = 0, n_entries = 0, items = 0;   // values a copy, copies of a staged row, table, items
    int box = 0, rw = 0, rs = 0;   // input by tensor copies of 16 channels: values of a row, stages
    int tw = 0, th = 0, tiles_x = 0, tiles_y = 0;   // rectangles of outputs (tw 0: flat tiles)
    int tiles = 0, n_fchunks = 0;   // tiles: pairs of position tiles, one per CTA of a pair
    long long units = 0;
    int xs = 0, hs = 0, ls = 0;   // input stages, slots of the hi and lo weights
    unsigned plane = 0, x_stage = 0, w_slot = 0, pool_off = 0, tab_off = 0, ring_off = 0, x_off = 0, h_off = 0, l_off = 0;
    size_t smem = 0;
    size_t ws_bytes = 0;
    double clocks = 0;      // estimated SM clocks
};

#ifdef __CUDACC__
struct TensorCall {
    const pp_layer* L;
    const void* x;
    void* y;
    const float* bias;
    int relu, N, H, W, Ho, Wo, pool, es;
    void* ws;
    unsigned* status;
    int sms;
    long long wait_limit;
    int no_fill;
    bool pdl;
    cudaStream_t st;
};
#endif

// Plan of a call, or false where the tensor-core kernel does not take it.
// ll (fp32): with the products of the lo parts, a third more work for less rounding.
bool tensor_plan(const pp_layer* L, int N, int H, int W, int pool, int es, size_t ws_bytes, int sms, TensorPlan* out,
                 int ll = 0);
#ifdef __CUDACC__
// Tensor map of fp32 x [N][C][H][W] with boxes of 16 channels of `rows` rows of `rw` values (conv.cu).
bool encode_box(CUtensorMap* map, const void* x, int N, int C, int H, int W, int rw, int rows);
cudaError_t tensor_launch(const TensorCall& c, const TensorPlan& pl);
// Builds the tensor-core weights from the bound device image.
cudaError_t tensor_build_weights(const pp_layer* L, void* dst, cudaStream_t st);
#endif

// Filters of a unit: the layer's filters in equal chunks of at most 256, a multiple of 16.
inline int tensor_chunks(const pp_layer* L) { return (L->cout + 255) / 256; }
inline int tensor_nc(const pp_layer* L) {
    const int n = tensor_chunks(L);
    return ((L->cout + n - 1) / n + 15) / 16 * 16;
}
// A chain of nine accumulator truncations takes this share of its sum away on average; it grows with the
// kept share of the kernels (measured 0.8e-7 of the result at 0.3, 1.0e-7 at 0.5, 1.3e-7 at 1).  The
// weights carry it back, in their lo parts, but for layers of weights that are fp16 values as they are:
// with integers for inputs their sums are exact, and the bias would put them off by an ulp.
inline double tensor_truncation(const pp_layer* L) { return 5.75e-8 + 7.5e-8 * ((double)L->beta / ((double)L->cout * L->cin_g)); }
inline double tensor_bias(const pp_layer* L) { return L->tc_exact ? 0.0 : tensor_truncation(L); }
// Bytes of a layer's tensor-core weights (0 where its weights have no fp16 pairs):
// [filter chunk][half][16-channel block][hi, lo][tap row][tap column][8 channels][filter][8 halves],
// so that a CTA's share of a row of taps is one contiguous copy.
inline size_t tensor_weight_bytes(const pp_layer* L) {
    if (!L->tc_ok) return 0;
    return (size_t)tensor_chunks(L) * tensor_nc(L) * ((L->cin_g + 15) / 16) * 9 * 64;
}

}  // namespace patconv

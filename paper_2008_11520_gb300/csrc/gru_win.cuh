// The fused training window (gru_win.cu, gru_win32.cu) as gru_train.cu calls it.
#pragma once

#include "common.cuh"

namespace dnnmg {

struct WinArgs {
    int n_in, ldx, n_out, nfc, T, P, ntiles;   // nfc: n_out rounded up to 16
    int pairs;                                 // rows of D and dD start on 8 bytes (n_out even)
    int xvec;                                  // rows of X start on 16 bytes
    int part_cols;                             // columns of a CTA's partial gradients (3H + nfc, then 3H for features 64 ..)
    int kx2;                                   // 16-column steps of the second 64-column chunk of features (0: one chunk)
    const float *X, *h0, *Wx, *Uh, *Wfc, *dD;
    float *D, *hT;                             // outputs of every step, state after the last
    float *z, *r, *c, *hb;                     // saved activations, [T][ntiles][H / 4][128][4]
    float *gWx, *gUh, *gWfc, *dh0, *part;
    float *GX;                                 // FP32 forward, two chunks: X W_x^T, [T][ntiles][3H / 4][128][4]
    float *dG;                                 // FP32 backward: gate gradients, [T][ntiles][3][H / 4][128][4] (may be GX)
    int *status;
};

bool win_supported(int n_in, int H, int n_out);
int win_tiles(int P);
size_t win_part_floats(int n_in, int H, int n_out, int T, int P);
cudaError_t win_forward(const WinArgs &g, int H, cudaStream_t st);        // BF16 products (gru_win.cu)
cudaError_t win_backward(const WinArgs &g, int H, cudaStream_t st);
cudaError_t win32_forward(const WinArgs &g, int H, cudaStream_t st);      // FP32 products (gru_win32.cu)
cudaError_t win32_backward(const WinArgs &g, int H, cudaStream_t st);
int win32_parts(int T, int P);
cudaError_t win_reduce(const WinArgs &g, int H, int nparts, int fc_lane, cudaStream_t st);

}  // namespace dnnmg

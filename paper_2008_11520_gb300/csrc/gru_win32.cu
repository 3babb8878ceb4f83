// The training window of the patch network with FP32 products, on the tensor
// cores: forward over T steps, backpropagation of the state gradients, and
// the weight gradients, as three persistent kernels.
//
// An FP32 operand is the sum of three BF16 values (8 significant bits each,
// so all 24), and a product of two is the sum of six BF16 products (the three
// left out are below 2^-24 of it).  Accumulation in tensor memory truncates,
// so the order matters: the small products are accumulated first and the
// leading one last, over at most 128 terms, and longer sums are added in FP32
// registers.  Measured against 64 bits on N(0, 1) operands: 0.8e-7 for K = 64
// and 1.3e-7 for K = 128, against 1.5e-7 and 2.1e-7 for FP32 FMA in sequence
// (the leading product first: 7e-7 and 1.4e-6); sums of 4096 terms drained
// every 128: 1.6e-7 against 1.1e-6.  Each accumulation at a sum's full
// magnitude, one per 16 terms of the leading product, drops up to an ulp, all of
// one sign; the average is put back (whole), so that a chain of products does not
// gather it.  Outputs and gradients of a window (65 536 rows, T = 10, H = 64) are
// off by 0.8e-7 and at most 1.2e-7, without that by 1.2e-7 and 2.0e-7, with FP32
// FMAs by 1.7e-7 and 2.2e-7 (762 rows: 0.8e-7, 1.7e-7, 1.3e-6).
//
// Six tcgen05 products of BF16 are 316 TFLOP/s of FP32 at the measured BF16
// rate; the CUDA cores' FMAs give 74.  With the fused window (see gru_win.cu,
// whose layouts these kernels share) loss and gradients of 65 536 rows, T =
// 10, H = 64 take 1.2 ms instead of 5.5 ms with one FP32 kernel per
// product, and of 762 rows, H = 32, 0.46 ms instead of 2.7 ms; with 99
// features and 50 outputs 1.8 ms instead of 6.5 ms (X W_x^T 214 us, forward
// 383, state gradients 422, weight gradients 363 and 229).
//
// An infinite operand, or a finite one beyond the BF16 range, has no such
// parts: its remainders are NaNs, and every sum it enters is one.  So results
// are looked at, and a tile (in the weight gradients: a CTA's blocks) with a
// state, output or gradient that is not finite is computed again with FP32
// FMAs (plain_*), which give FP32's infinities, NaNs and saturated gates.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "gru_win.cuh"
#include "gru_win_dev.cuh"

namespace dnnmg {
namespace {

constexpr int W32_TH = 512;   // four threads a row

// the products of the three-part operands, small ones first
__device__ constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};

// D = A B^T of two K-major operands whose parts are astep / bstep bytes apart;
// with a second pair of operands (a2, b2), whose K follows the first one's
__device__ __forceinline__ void mma3_k(uint32_t d, uint32_t a, uint32_t astep, uint32_t b, uint32_t bstep, int N, int ksteps) {
    uint32_t acc = 0;
    for (int p = 0; p < 6; ++p) {
        const uint64_t da = desc_k(a + PA[p] * astep), db = desc_k(b + PB[p] * bstep);
        for (int k = 0; k < ksteps; ++k) {
            umma(d, da + 2 * k, db + 2 * k, idesc(N, false), acc);
            acc = 1;
        }
    }
}
// D = A^T B over `rows` rows of MN-major operands; anext / bnext: the next 64 columns
__device__ __forceinline__ void mma3_mn(uint32_t d, uint32_t a, uint32_t astep, uint32_t anext, uint32_t b, uint32_t bstep,
                                        uint32_t bnext, int N, int rows) {
    uint32_t acc = 0;
    for (int p = 0; p < 6; ++p) {
        const uint64_t da = desc_mn(a + PA[p] * astep, anext), db = desc_mn(b + PB[p] * bstep, bnext);
        for (int k = 0; k < rows / 16; ++k) {
            umma(d, da + k * (2048 >> 4), db + k * (2048 >> 4), idesc(N, true), acc);
            acc = 1;
        }
    }
}

// Each accumulation at a product's full magnitude (one per 16 terms of its
// leading part) drops on average 2.1e-8 of the sum (measured on N(0, 1) operands:
// 0.85e-7 for K = 64, 1.7e-7 for K = 128, all of one sign).  That much is put
// back.  steps: those that hold data, which are the only ones that can drop
// anything: of one, it is less than half an ulp and a representable sum stays.
__device__ __forceinline__ float whole(float v, int steps) { return fmaf(v, 2.1e-8f * (float)steps, v); }
// The steps of a row that hold data: each of its four threads (part) leaves a mask
// of the 16-column steps in which it has a value other than zero, in the row's
// word of an operand's 512 bytes; to be read after a hand-over.
constexpr int STEPS = TM * 4;
__device__ __forceinline__ void put_steps(uint8_t *f, int row, int part, unsigned mask) { f[4 * row + part] = (uint8_t)mask; }
__device__ __forceinline__ int get_steps(const uint8_t *f, int row) {
    unsigned w = *reinterpret_cast<const unsigned *>(f + 4 * row);
    w |= w >> 16;
    return __popc((w | w >> 8) & 15u);
}
// of H / 4 consecutive columns a thread; bits: all its values' bits (of zeros, no more than the sign)
template <int H> __device__ __forceinline__ unsigned step_mask(unsigned bits, int part) {
    return bits << 1 ? 1u << (H == 64 ? part : part >> 1) : 0u;
}

// Whether every value seen is finite (0 x is not 0 for one that is not)
struct Finite {
    float m = 0.f;
    __device__ __forceinline__ void see(float x) { m = fmaf(0.f, x, m); }
    __device__ __forceinline__ bool failed() const { return m != 0.f; }
};
// the three parts of two values, each pair packed
__device__ __forceinline__ void split2(float x, float y, uint32_t (&o)[3]) {
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(x, y);
        o[p] = *reinterpret_cast<const uint32_t *>(&t);
        x -= __low2float(t);
        y -= __high2float(t);
    }
}
// 8 consecutive columns of a row into the three images, `step` bytes apart
__device__ __forceinline__ void put8_3(uint8_t *img, int step, int row, int c, const float *v) {
    uint32_t o[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i) split2(v[2 * i], v[2 * i + 1], o[i]);
    const uint32_t at = swz(row, c >> 3);
#pragma unroll
    for (int p = 0; p < 3; ++p)
        *reinterpret_cast<uint4 *>(img + p * step + at) = make_uint4(o[0][p], o[1][p], o[2][p], o[3][p]);
}
// 4 consecutive columns (c a multiple of 4)
__device__ __forceinline__ void put4_3(uint8_t *img, int step, int row, int c, const float *v) {
    uint32_t a[3], b[3];
    split2(v[0], v[1], a);
    split2(v[2], v[3], b);
    const uint32_t at = swz(row, c >> 3) + (c & 4) * 2;
#pragma unroll
    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2 *>(img + p * step + at) = make_uint2(a[p], b[p]);
}

template <typename F> __device__ __forceinline__ void build3(uint8_t *img, int step, int rows, F src) {
    for (int e = threadIdx.x; e < rows * 8; e += W32_TH) {
        const int r = e >> 3, c = (e & 7) * 8;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = src(r, c + i);
        put8_3(img, step, r, c, v);   // (8-row groups are 1024 bytes apart: row * 128 throughout)
    }
}
__device__ __forceinline__ void store_x3(const WinArgs &g, const XTile<W32_TH> &x, uint8_t *img, int x0 = 0) {
    const int n = g.n_in - x0;
#pragma unroll
    for (int i = 0; i < XTile<W32_TH>::NV; ++i) {
        const int e = threadIdx.x + i * W32_TH, row = e >> 4, c = (e & 15) * 4;
        const float v[4] = {x.v[i].x, c + 1 < n ? x.v[i].y : 0.f, c + 2 < n ? x.v[i].z : 0.f, c + 3 < n ? x.v[i].w : 0.f};
        put4_3(img, IMG, row, c, v);
    }
}

// ---------------------------------------------------------------- FP32 FMAs
// A tile (128 rows) with values that are not finite, computed again: a warp
// takes a row; rows past the last patch are zero.  buf: 16 x 512 floats of
// shared memory.  Called by all threads of a CTA.
__device__ __forceinline__ size_t elem(int c, int row) { return blk(c, row) + (c & 3); }
// y = W x, W [rows][n] (one dot product at a time, lanes along n)
__device__ __forceinline__ void rows_times(const float *__restrict__ W, int rows, int n, const float *x, float *y) {
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int c = 0; c < rows; ++c) {
        float a = 0.f;
        for (int k = lane; k < n; k += 32) a = fmaf(__ldg(W + (size_t)c * n + k), x[k], a);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) y[c] = a;
    }
}
// sum over k of W[k][j] x[k], rows of W H long (lanes along j)
__device__ __forceinline__ float column_times(const float *__restrict__ W, int H, int n, int j, const float *x) {
    float a = 0.f;
#pragma unroll 4
    for (int k = 0; k < n; ++k) a = fmaf(__ldg(W + (size_t)k * H + j), x[k], a);
    return a;
}

// forward of all steps
template <int H> __device__ __noinline__ void plain_fwd(const WinArgs &g, int tile, float *buf) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t tblk = (size_t)TM * H;
    float *x = buf + warp * 512, *h = x + 128, *rh = h + 64, *ax = rh + 64, *ah = ax + 64;
    for (int row = warp; row < TM; row += W32_TH / 32) {
        const int gp = tile * TM + row;
        const bool valid = gp < g.P;
        __syncwarp();
        // (h_0 as saved: the caller's array may be the state that has been written meanwhile)
        for (int j = lane; j < H; j += 32) h[j] = g.hb[(size_t)tile * tblk + elem(j, row)];
        for (int s = 0; s < g.T; ++s) {
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk, prow = (size_t)s * g.P + gp;
            if (valid)
                for (int k = lane; k < g.n_in; k += 32) x[k] = __ldg(g.X + prow * g.ldx + k);
            for (int j = lane; j < H; j += 32) g.hb[sb + elem(j, row)] = h[j];
            for (int gate = 1; gate >= 0; --gate) {   // r, then z
                __syncwarp();
                if (valid) {
                    rows_times(g.Wx + (size_t)gate * H * g.n_in, H, g.n_in, x, ax);
                    rows_times(g.Uh + (size_t)gate * H * H, H, H, h, ah);
                }
                __syncwarp();
                for (int j = lane; j < H; j += 32) {
                    const float v = valid ? sigm(ax[j] + ah[j]) : 0.f;
                    (gate ? g.r : g.z)[sb + elem(j, row)] = v;
                    if (gate) rh[j] = v * h[j];
                }
            }
            __syncwarp();
            if (valid) {
                rows_times(g.Wx + (size_t)2 * H * g.n_in, H, g.n_in, x, ax);
                rows_times(g.Uh + (size_t)2 * H * H, H, H, rh, ah);
            }
            __syncwarp();
            for (int j = lane; j < H; j += 32) {
                const float c = valid ? tanhf(ax[j] + ah[j]) : 0.f, z = g.z[sb + elem(j, row)];
                g.c[sb + elem(j, row)] = c;
                if (valid) h[j] = z * h[j] + (1.0f - z) * c;
            }
            __syncwarp();
            if (valid) rows_times(g.Wfc, g.n_out, H, h, ax);
            __syncwarp();
            if (valid)
                for (int o = lane; o < g.n_out; o += 32) g.D[prow * g.n_out + o] = ax[o];
        }
        if (valid)
            for (int j = lane; j < H; j += 32) g.hT[(size_t)gp * H + j] = h[j];
    }
}

// state gradients of all steps
template <int H> __device__ __noinline__ void plain_bwd(const WinArgs &g, int tile, float *buf) {
    constexpr int NJ = H / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const size_t tblk = (size_t)TM * H;
    float *dd = buf + warp * 512, *az = dd + 64, *ar = az + 64, *ac = ar + 64;
    for (int row = warp; row < TM; row += W32_TH / 32) {
        const int gp = tile * TM + row;
        const bool valid = gp < g.P;
        float carry[NJ];
#pragma unroll
        for (int i = 0; i < NJ; ++i) carry[i] = 0.f;
        for (int s = g.T - 1; s >= 0; --s) {
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk, gb = 3 * sb;
            __syncwarp();
            if (valid)
                for (int o = lane; o < g.n_out; o += 32) dd[o] = __ldg(g.dD + ((size_t)s * g.P + gp) * g.n_out + o);
            __syncwarp();
            float dh[NJ], drh[NJ];
#pragma unroll
            for (int i = 0; i < NJ; ++i) {
                const int j = lane + 32 * i;
                const size_t e = sb + elem(j, row);
                az[j] = ac[j] = dh[i] = 0.f;
                if (!valid) continue;
                dh[i] = column_times(g.Wfc, H, g.n_out, j, dd) + carry[i];
                const float z = g.z[e], c = g.c[e], dc = dh[i] * (1.0f - z), dz = dh[i] * (g.hb[e] - c);
                az[j] = dz * z * (1.0f - z);
                ac[j] = dc * (1.0f - c * c);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NJ; ++i) {
                const int j = lane + 32 * i;
                const size_t e = sb + elem(j, row);
                ar[j] = drh[i] = 0.f;
                if (!valid) continue;
                drh[i] = column_times(g.Uh + (size_t)2 * H * H, H, H, j, ac);
                ar[j] = drh[i] * g.hb[e] * g.r[e] * (1.0f - g.r[e]);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NJ; ++i) {
                const int j = lane + 32 * i;
                const size_t e = sb + elem(j, row), d = gb + elem(j, row);
                g.dG[d] = az[j];
                g.dG[d + tblk] = ar[j];
                g.dG[d + 2 * tblk] = ac[j];
                if (!valid) continue;
                carry[i] = dh[i] * g.z[e] + drh[i] * g.r[e];
                carry[i] += column_times(g.Uh, H, H, j, az) + column_times(g.Uh + (size_t)H * H, H, H, j, ar);
            }
        }
        if (valid && g.dh0)
#pragma unroll
            for (int i = 0; i < NJ; ++i) g.dh0[(size_t)gp * H + lane + 32 * i] = carry[i];
    }
}

// ---------------------------------------------------------------- forward
// One CTA an SM: the weights' three parts take 172 KB (H = 64), so the three
// images of one operand share the rest and h, X and r h pass through them in
// turn: the previous state for h U_zr^T and the previous step's outputs, X
// for X W_x^T, r h for the candidate.  Tensor memory: X W_x^T [0, 3H),
// h U_zr^T [3H, 5H), (r h) U_h^T [5H, 6H), outputs [6H, 6H + nfc).
// Bound by the chain of three MMA round trips a step with the splits and gate
// functions between them.  Two chunks of features (XC = 2) leave no room for
// W_x: X W_x^T comes from memory (k_win32_x).
template <int H, int XC> struct Fwd32Layout {
    static constexpr int WS = 3 * H * 128, FS = 64 * 128;   // bytes of one part
    static constexpr int WX = 0, U = WX + (XC == 1 ? 3 * WS : 0), F = U + 3 * WS, A = F + 3 * FS, SH = A + 3 * IMG, SR = SH + STEPS, BARS = SR + STEPS, BYTES = BARS + 64 + 1024;   // SH, SR: steps of h, r h
    static constexpr int COLS = H == 64 ? 512 : 256;
};

// X W_x^T of every step for two chunks of features, [step][tile][column / 4][row][4].
// Each chunk's products are accumulated apart (W_x and one chunk's images fill
// the shared memory) and added in FP32.  Bound by the chain of split, products
// and read-out, two of them a tile.
template <int H> struct X32Layout {
    static constexpr int WS = 3 * H * 128;
    static constexpr int W = 0, A = W + 6 * WS, BARS = A + 3 * IMG, BYTES = BARS + 64 + 1024;   // W: 3 parts of each chunk
    static constexpr int COLS = H == 64 ? 512 : 256;
};
template <int H>
__global__ void __launch_bounds__(W32_TH, 1) k_win32_x(const __grid_constant__ WinArgs g) {
    using L = X32Layout<H>;
    constexpr int NC = 3 * H / 4;   // columns of a thread
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw), *sA = base + L::A;
    const uint32_t u = smem_u32(base);
    for (int x = 0; x < 2; ++x)
        build3(base + L::W + 3 * x * L::WS, L::WS, 3 * H, [&](int r, int c) {
            return 64 * x + c < g.n_in ? __ldg(g.Wx + (size_t)r * g.n_in + 64 * x + c) : 0.f;
        });
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 2, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane, c0 = part * NC;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    uint32_t ph = 0;
    bool ok = true;
    const int n = g.T * g.ntiles;
    XTile<W32_TH> xt;
    if ((int)blockIdx.x < n) xt.load(g, blockIdx.x / g.ntiles, blockIdx.x % g.ntiles * TM);
    for (int it = blockIdx.x; ok && it < n; it += gridDim.x) {
        const int s = it / g.ntiles, p0 = it % g.ntiles * TM;
        store_x3(g, xt, sA);
        xt.load(g, s, p0, 64);
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma3_k(cta.tmem, u + L::A, IMG, u + L::W, L::WS, 3 * H, 4);
            tc_commit(cta.bar0);
        }
        ok = cta.wait(0, ph);
        ph ^= 1;
        store_x3(g, xt, sA, 64);
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma3_k(cta.tmem + 3 * H, u + L::A, IMG, u + L::W + 3 * L::WS, L::WS, 3 * H, g.kx2);
            tc_commit(cta.bar0);
        }
        const int nx = it + gridDim.x;
        if (nx < n) xt.load(g, nx / g.ntiles, nx % g.ntiles * TM);
        ok = cta.wait(0, ph);
        ph ^= 1;
        float *o = g.GX + (size_t)it * (3 * TM * H);
#pragma unroll
        for (int i = 0; i < NC; i += 8) {
            float a[8], b[8];
            tmem_ld8(tl + c0 + i, a);
            tmem_ld8(tl + 3 * H + c0 + i, b);
            tmem_wait();
            keep(a);
            keep(b);
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = whole(a[j], 4) + whole(b[j], g.kx2);
            st4(o + blk(c0 + i, row), a);
            st4(o + blk(c0 + i + 4, row), a + 4);
        }
    }
    ok = cta.hand_over(ok);
    cta.finish(1, L::COLS, g.status);
}

template <int H, int XC>
__global__ void __launch_bounds__(W32_TH, 1) k_win32_fwd(const __grid_constant__ WinArgs g) {
    using L = Fwd32Layout<H, XC>;
    constexpr int NC = H / 4;   // state columns of a thread
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw), *sA = base + L::A;
    const uint32_t u = smem_u32(base), uA = u + L::A;
    if (XC == 1)
        build3(base + L::WX, L::WS, 3 * H, [&](int r, int c) { return c < g.n_in ? __ldg(g.Wx + (size_t)r * g.n_in + c) : 0.f; });
    build3(base + L::U, L::WS, 3 * H, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)r * H + c) : 0.f; });
    build3(base + L::F, L::FS, g.nfc, [&](int r, int c) { return r < g.n_out && c < H ? __ldg(g.Wfc + (size_t)r * H + c) : 0.f; });
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 2, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane, c0 = part * NC;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    const size_t tblk = (size_t)TM * H;
    uint8_t *fh = base + L::SH, *fr = base + L::SR;
    const int kx = (min(g.n_in, 64) + 15) / 16;
    int kh = 0;   // steps of the state that h U^T and the outputs in tensor memory come from
    uint32_t ph = 0;
    bool ok = true;
    XTile<W32_TH> xt;
    for (int tile = blockIdx.x; ok && tile < g.ntiles; tile += gridDim.x) {
        const int p0 = tile * TM, gp = p0 + row;
        const bool valid = gp < g.P;
        float hv[NC];
#pragma unroll
        for (int i = 0; i < NC; i += 4) {
            hv[i] = hv[i + 1] = hv[i + 2] = hv[i + 3] = 0.f;
            if (g.h0 && valid) ld4(g.h0 + (size_t)gp * H + c0 + i, hv + i);
            st4(g.hb + (size_t)tile * tblk + blk(c0 + i, row), hv + i);
        }
        auto put_h = [&]() {
            unsigned any = 0;
#pragma unroll
            for (int i = 0; i < NC; ++i) any |= __float_as_uint(hv[i]);
            put_steps(fh, row, part, step_mask<H>(any, part));
        };
        put_h();
        if (XC == 1) xt.load(g, 0, p0);
#pragma unroll
        for (int i = 0; i < NC; i += 8) put8_3(sA, IMG, row, c0 + i, hv + i);
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma3_k(cta.tmem + 3 * H, uA, IMG, u + L::U, L::WS, 2 * H, H / 16);
            tc_commit(cta.bar0);
        }
        auto outputs = [&](int s) {   // of step s, from tensor memory
            float *drow = g.D + ((size_t)s * g.P + gp) * g.n_out;
            for (int b = part; b < g.nfc / 8; b += 4) {
                float v[8];
                Finite fin;
                tmem_ld8(tl + 6 * H + 8 * b, v);
                tmem_wait();
                keep(v);
                if (!valid) continue;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = whole(v[j], kh);
                    fin.see(v[j]);
                }
                if (fin.failed()) cta.mark();
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const int c = 8 * b + j;
                    if (g.pairs) {
                        if (c < g.n_out) *reinterpret_cast<float2 *>(drow + c) = make_float2(v[j], v[j + 1]);
                    } else {
                        if (c < g.n_out) drow[c] = v[j];
                        if (c + 1 < g.n_out) drow[c + 1] = v[j + 1];
                    }
                }
            }
        };
        for (int s = 0; s < g.T; ++s) {
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
            float gr[XC == 2 ? NC : 1], gz[XC == 2 ? NC : 1], gc[XC == 2 ? NC : 1];   // X W_x^T from memory
            const float *gx = g.GX + 3 * sb;
            if (XC == 2) {
#pragma unroll
                for (int i = 0; i < NC; i += 4) ld4(gx + blk(H + c0 + i, row), gr + i);
            }
            ok = cta.wait(0, ph);
            ph ^= 1;
            kh = get_steps(fh, row);
            if (XC == 1) {
                store_x3(g, xt, sA);
                if (!(ok = cta.hand_over(ok))) break;
                if (tid == 0) {
                    mma3_k(cta.tmem, uA, IMG, u + L::WX, L::WS, 3 * H, 4);
                    tc_commit(cta.bar0);
                }
                if (s > 0) outputs(s - 1);
                ok = cta.wait(0, ph);
                ph ^= 1;
            }
            unsigned any = 0;
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8], b[8], rr[8];
                if (XC == 1) tmem_ld8(tl + H + c0 + i, a);
                tmem_ld8(tl + 4 * H + c0 + i, b);
                tmem_wait();
                if (XC == 1) keep(a);
                keep(b);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    rr[j] = sigm((XC == 1 ? whole(a[j], kx) : gr[(i + j) % (XC == 2 ? NC : 1)]) + whole(b[j], kh));
                    a[j] = rr[j] * hv[i + j];
                    any |= __float_as_uint(a[j]);
                }
                st4(g.r + sb + blk(c0 + i, row), rr);
                st4(g.r + sb + blk(c0 + i + 4, row), rr + 4);
                put8_3(sA, IMG, row, c0 + i, a);
            }
            put_steps(fr, row, part, step_mask<H>(any, part));
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma3_k(cta.tmem + 5 * H, uA, IMG, u + L::U + 2 * H * 128, L::WS, H, H / 16);
                tc_commit(cta.bar0);
            }
            if (XC == 1) {
                if (s + 1 < g.T) xt.load(g, s + 1, p0);
            } else {
                if (s > 0) outputs(s - 1);
#pragma unroll
                for (int i = 0; i < NC; i += 4) {
                    ld4(gx + blk(c0 + i, row), gz + i);
                    ld4(gx + blk(2 * H + c0 + i, row), gc + i);
                }
            }
            ok = cta.wait(0, ph);
            ph ^= 1;
            const int kr = get_steps(fr, row);
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8], b[8], zz[8], cc[8];
                Finite fin;
                if (XC == 1) {
                    tmem_ld8(tl + c0 + i, a);
                    tmem_ld8(tl + 2 * H + c0 + i, zz);
                }
                tmem_ld8(tl + 3 * H + c0 + i, b);
                tmem_ld8(tl + 5 * H + c0 + i, cc);
                tmem_wait();
                if (XC == 1) {
                    keep(a);
                    keep(zz);
                }
                keep(b);
                keep(cc);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = (i + j) % (XC == 2 ? NC : 1);
                    const float z = sigm((XC == 1 ? whole(a[j], kx) : gz[k]) + whole(b[j], kh)),
                                c = tanhf((XC == 1 ? whole(zz[j], kx) : gc[k]) + whole(cc[j], kr));
                    zz[j] = z;
                    cc[j] = c;
                    hv[i + j] = z * hv[i + j] + (1.0f - z) * c;
                    fin.see(hv[i + j]);
                }
                if (fin.failed()) cta.mark();
                st4(g.z + sb + blk(c0 + i, row), zz);
                st4(g.z + sb + blk(c0 + i + 4, row), zz + 4);
                st4(g.c + sb + blk(c0 + i, row), cc);
                st4(g.c + sb + blk(c0 + i + 4, row), cc + 4);
                put8_3(sA, IMG, row, c0 + i, hv + i);
            }
            put_h();
            if (s + 1 < g.T) {
                float *hb = g.hb + ((size_t)(s + 1) * g.ntiles + tile) * tblk;
#pragma unroll
                for (int i = 0; i < NC; i += 4) st4(hb + blk(c0 + i, row), hv + i);
            } else if (valid) {
#pragma unroll
                for (int i = 0; i < NC; i += 4) st4(g.hT + (size_t)gp * H + c0 + i, hv + i);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma3_k(cta.tmem + 6 * H, uA, IMG, u + L::F, L::FS, g.nfc, H / 16);
                if (s + 1 < g.T) mma3_k(cta.tmem + 3 * H, uA, IMG, u + L::U, L::WS, 2 * H, H / 16);
                tc_commit(cta.bar0);
            }
        }
        if (ok) {
            ok = cta.wait(0, ph);
            ph ^= 1;
            kh = get_steps(fh, row);
            if (ok) outputs(g.T - 1);
        }
        ok = cta.hand_over(ok);   // (the same answer in every thread)
        if (ok && cta.marked()) {
            plain_fwd<H>(g, tile, reinterpret_cast<float *>(sA));
            cta.unmark();
        }
    }
    cta.finish(1, L::COLS, g.status);
}

// ---------------------------------------------------------------- backward
// The state gradients, last step first (as k_win_bwd), with dA written to
// memory for the weight gradients: the images of three-part operands leave no
// room for them here.  Two operands' images (B0, B1): dA_z and dA_c, then
// dD of the next step and dA_r.  Tensor memory: dD W_fc [0, H), d(r h)
// [64, 64 + H), dA_z U_z [128, ..), dA_r U_r [192, ..).
template <int H> struct Bwd32Layout {
    static constexpr int WS = H * 128;
    static constexpr int WF = 0, UC = WF + 3 * WS, UZ = UC + 3 * WS, UR = UZ + 3 * WS, B0 = UR + 3 * WS, B1 = B0 + 3 * IMG,
                         SD = B1 + 3 * IMG, BARS = SD + STEPS, BYTES = BARS + 64 + 1024;   // SD: steps of dD
    static constexpr int COLS = 256;
};

template <int H>
__global__ void __launch_bounds__(W32_TH, 1) k_win32_bwd(const __grid_constant__ WinArgs g) {
    using L = Bwd32Layout<H>;
    constexpr int NC = H / 4;
    constexpr int T_DH = 0, T_DRH = 64, T_CZ = 128, T_CR = 192;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw), *B0 = base + L::B0, *B1 = base + L::B1;
    const uint32_t u = smem_u32(base);
    build3(base + L::WF, L::WS, H, [&](int r, int c) { return c < g.n_out ? __ldg(g.Wfc + (size_t)c * H + r) : 0.f; });
    build3(base + L::UC, L::WS, H, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)(2 * H + c) * H + r) : 0.f; });
    build3(base + L::UZ, L::WS, H, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)c * H + r) : 0.f; });
    build3(base + L::UR, L::WS, H, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)(H + c) * H + r) : 0.f; });
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 2, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane, c0 = part * NC;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    const size_t tblk = (size_t)TM * H;
    const int kfc = g.nfc / 16;
    uint8_t *fd = base + L::SD;   // (dA has values in all its steps wherever it has any)
    uint32_t ph = 0;
    bool ok = true;
    // dD of a step: each thread up to 16 columns of its row (blocks of 4 dealt to the row's threads)
    constexpr int DDN = 4;
    float dd[DDN][4];
    auto load_dd = [&](int s, int gp) {
#pragma unroll
        for (int i = 0; i < DDN; ++i) {
            const int c = 4 * (part + 4 * i);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                dd[i][j] = gp < g.P && c + j < g.n_out ? __ldg(g.dD + ((size_t)s * g.P + gp) * g.n_out + c + j) : 0.f;
        }
    };
    auto put_dd = [&](uint8_t *img) {
        unsigned mask = 0;   // (block i lies in step i)
#pragma unroll
        for (int i = 0; i < DDN; ++i) {
            const int c = 4 * (part + 4 * i);
            if (c < g.nfc) put4_3(img, IMG, row, c, dd[i]);
            const unsigned any = __float_as_uint(dd[i][0]) | __float_as_uint(dd[i][1]) | __float_as_uint(dd[i][2]) | __float_as_uint(dd[i][3]);
            mask |= any << 1 ? 1u << i : 0u;
        }
        put_steps(fd, row, part, mask);
    };
    for (int tile = blockIdx.x; ok && tile < g.ntiles; tile += gridDim.x) {
        const int p0 = tile * TM, gp = p0 + row;
        float zv[NC], rv[NC], cv[NC], hp[NC], cpart[NC];
        auto load_step = [&](int s) {
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
#pragma unroll
            for (int i = 0; i < NC; i += 4) {
                const size_t o = sb + blk(c0 + i, row);
                ld4(g.z + o, zv + i);
                ld4(g.r + o, rv + i);
                ld4(g.c + o, cv + i);
                ld4(g.hb + o, hp + i);
            }
        };
        load_dd(g.T - 1, gp);
        load_step(g.T - 1);
        put_dd(B0);
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma3_k(cta.tmem + T_DH, u + L::B0, IMG, u + L::WF, L::WS, H, kfc);
            tc_commit(cta.bar0);
        }
        for (int s = g.T - 1; s >= 0; --s) {
            const size_t gb = ((size_t)s * g.ntiles + tile) * 3 * tblk;   // dA: gates z, r, c one after the other
            if (s > 0) load_dd(s - 1, gp);
            ok = cta.wait(0, ph);
            ph ^= 1;
            float dh[NC];
            const int kd = get_steps(fd, row);
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8], b[8], c[8], az[8], ac[8];
                tmem_ld8(tl + T_DH + c0 + i, a);
                tmem_ld8(tl + T_CZ + c0 + i, b);
                tmem_ld8(tl + T_CR + c0 + i, c);
                tmem_wait();
                keep(a);
                keep(b);
                keep(c);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = i + j;
                    const float carry = s == g.T - 1 ? 0.f : whole(b[j] + c[j], H / 16) + cpart[k];
                    dh[k] = whole(a[j], kd) + carry;
                    const float dc = dh[k] * (1.0f - zv[k]), dz = dh[k] * (hp[k] - cv[k]);
                    az[j] = dz * zv[k] * (1.0f - zv[k]);
                    ac[j] = dc * (1.0f - cv[k] * cv[k]);
                }
                put8_3(B0, IMG, row, c0 + i, az);
                put8_3(B1, IMG, row, c0 + i, ac);
#pragma unroll
                for (int j = 0; j < 8; j += 4) {
                    st4(g.dG + gb + blk(c0 + i + j, row), az + j);
                    st4(g.dG + gb + 2 * tblk + blk(c0 + i + j, row), ac + j);
                }
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma3_k(cta.tmem + T_DRH, u + L::B1, IMG, u + L::UC, L::WS, H, H / 16);
                mma3_k(cta.tmem + T_CZ, u + L::B0, IMG, u + L::UZ, L::WS, H, H / 16);
                tc_commit(cta.bar0);
            }
            ok = cta.wait(0, ph);
            ph ^= 1;
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8];
                Finite fin;   // (a dA that is not finite shows in the step before)
                tmem_ld8(tl + T_DRH + c0 + i, a);
                tmem_wait();
                keep(a);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = i + j;
                    a[j] = whole(a[j], H / 16);
                    cpart[k] = dh[k] * zv[k] + a[j] * rv[k];
                    fin.see(cpart[k]);
                    a[j] = a[j] * hp[k] * rv[k] * (1.0f - rv[k]);
                }
                if (fin.failed()) cta.mark();
                put8_3(B1, IMG, row, c0 + i, a);
#pragma unroll
                for (int j = 0; j < 8; j += 4) st4(g.dG + gb + tblk + blk(c0 + i + j, row), a + j);
            }
            if (s > 0) {
                put_dd(B0);
                load_step(s - 1);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma3_k(cta.tmem + T_CR, u + L::B1, IMG, u + L::UR, L::WS, H, H / 16);
                if (s > 0) mma3_k(cta.tmem + T_DH, u + L::B0, IMG, u + L::WF, L::WS, H, kfc);
                tc_commit(cta.bar0);
            }
        }
        if (ok) {
            ok = cta.wait(0, ph);
            ph ^= 1;
            if (ok && g.dh0) {
#pragma unroll
                for (int i = 0; i < NC; i += 8) {
                    float b[8], c[8];
                    Finite fin;
                    tmem_ld8(tl + T_CZ + c0 + i, b);
                    tmem_ld8(tl + T_CR + c0 + i, c);
                    tmem_wait();
                    keep(b);
                    keep(c);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        b[j] = whole(b[j] + c[j], H / 16) + cpart[i + j];
                        fin.see(b[j]);
                    }
                    if (fin.failed()) cta.mark();
                    if (gp < g.P) {
                        st4(g.dh0 + (size_t)gp * H + c0 + i, b);
                        st4(g.dh0 + (size_t)gp * H + c0 + i + 4, b + 4);
                    }
                }
            }
        }
        ok = cta.hand_over(ok);   // (the same answer in every thread)
        if (ok && cta.marked()) {
            plain_bwd<H>(g, tile, reinterpret_cast<float *>(B0));
            cta.unmark();
        }
    }
    cta.finish(1, L::COLS, g.status);
}

// ---------------------------------------------------------------- weight gradients
// [X | h_s]^T [dA_z, dA_r], [X | r h_s]^T dA_c and h_{s+1}^T dD over all
// steps and rows, in blocks of 64 rows (whose operands' three parts fill the
// shared memory): a CTA takes a contiguous range of blocks, accumulates each
// in tensor memory, adds it to FP32 registers and these, every few blocks, to
// a sum kept in tensor memory (a sum in one run of 67 blocks loses twice as much).
// Bound by memory (2.6 kB a row and step at H = 64) and the splits.  X2: the
// products of the second chunk of features with dA alone, in a launch of its
// own (their sums have no room beside the others).
constexpr int GR = 64, GIMG = GR * 128;   // rows of a block, one image
constexpr int G32_RUN = 8;                // blocks added up in registers before they join the sum in tensor memory
template <int H> struct Grad32Layout {
    // parts of one operand GIMG apart
    static constexpr int X = 0, HP = X + 3 * GIMG, RH = HP + 3 * GIMG, HN = RH + 3 * GIMG, GZ = HN + 3 * GIMG,
                         GRR = GZ + 3 * GIMG, GC = GRR + 3 * GIMG, DD = GC + 3 * GIMG, BARS = DD + 3 * GIMG,
                         BYTES = BARS + 64 + 1024;
    static constexpr int COLS = 512;        // the block's products, then sums of G32_RUN blocks from SUM on
    static constexpr int SUM = 256;
    static constexpr int NB = (3 * H + 64) / 8 / 4;   // blocks of 8 gradient columns a thread adds up
};

// A CTA's blocks [b0, b1) with FP32 FMAs, for a warp with a sum that is not finite:
// its own lanes and columns, to where the sums were.
template <int H, bool X2> __device__ __noinline__ void plain_grad(const WinArgs &g, long long b0, long long b1, uint32_t tmem) {
    const int warp = threadIdx.x >> 5, q = warp & 3, part = warp >> 2, m = q * 32 + (threadIdx.x & 31);
    const uint32_t tl = tmem + ((uint32_t)(q * 32) << 16);
    const int ncol = 3 * H + (X2 ? 0 : g.nfc), fx = (X2 ? 64 : 0) + m, mh = m - 64;   // feature and state column of this lane
    const size_t tblk = (size_t)TM * H;
    for (int c = 8 * part; c < ncol; c += 32) {
        const int gate = c / H;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = 0.f;
        for (long long it = b0; it < b1; ++it) {
            const int s = (int)(it % g.T), th = (int)(it / g.T), tile = th >> 1, r0 = (th & 1) * GR;
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
            const bool last = s + 1 == g.T;
            for (int r = r0; r < min(r0 + GR, g.P - tile * TM); ++r) {
                const int gp = tile * TM + r;
                const size_t prow = (size_t)s * g.P + gp;
                float a = 0.f;
                if (c >= 3 * H) {
                    if (m < H) a = last ? g.hT[(size_t)gp * H + m] : g.hb[sb + (size_t)g.ntiles * tblk + elem(m, r)];
                } else if (m < 64) {
                    if (fx < g.n_in) a = __ldg(g.X + prow * g.ldx + fx);
                } else if (!X2 && mh < H) {
                    a = g.hb[sb + elem(mh, r)];
                    if (gate == 2) a *= g.r[sb + elem(mh, r)];
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float b;
                    if (c < 3 * H) b = g.dG[3 * sb + gate * tblk + elem(c - gate * H + j, r)];
                    else b = c - 3 * H + j < g.n_out ? __ldg(g.dD + prow * g.n_out + c - 3 * H + j) : 0.f;
                    v[j] = fmaf(a, b, v[j]);
                }
            }
        }
        tmem_st8(tl + Grad32Layout<H>::SUM + c, v);
    }
    tmem_wait_st();
}

template <int H, bool X2>
__global__ void __launch_bounds__(W32_TH, 1) k_win32_grad(const __grid_constant__ WinArgs g) {
    using L = Grad32Layout<H>;
    constexpr int X0 = X2 ? 64 : 0, NB = X2 ? 3 * H / 32 : L::NB;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw);
    const uint32_t u = smem_u32(base);
    // columns that no block writes but products of unused gradient rows read
    for (int e = threadIdx.x; e < L::BARS / 16; e += W32_TH) reinterpret_cast<uint4 *>(base)[e] = make_uint4(0, 0, 0, 0);
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 2, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    const int ncol = 3 * H + (X2 ? 0 : g.nfc), out0 = X2 ? 3 * H + g.nfc : 0;
    const size_t tblk = (size_t)TM * H;
    float acc[NB][8];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[b][j] = 0.f;
    const long long n = 2LL * g.T * g.ntiles;   // blocks: (tile, half, step), steps fastest
    const long long i0 = n * blockIdx.x / gridDim.x, i1 = n * (blockIdx.x + 1) / gridDim.x;
    uint32_t ph = 0;
    bool ok = true;
    const long long full = (long long)g.T * (g.P / GR);   // blocks before have all their rows, those from full + T on none
    auto drain = [&](long long it) {   // the block's products into the registers
        ok = cta.wait(0, ph);
        ph ^= 1;
        auto add = [&](int steps) {
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int c = 8 * (part + 4 * b);
                if (c < ncol) {
                    float v[8];
                    tmem_ld8(tl + c, v);
                    tmem_wait();
                    keep(v);
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[b][j] += whole(v[j], steps);
                }
            }
        };
        if (it < full) add(GR / 16);
        else add(it < full + g.T ? (g.P % GR + 15) / 16 : 0);
    };
    bool summed = false;
    auto flush = [&]() {   // the registers' sums into tensor memory
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const int c = 8 * (part + 4 * b);
            if (c < ncol) {
                if (summed) {
                    float v[8];
                    tmem_ld8(tl + L::SUM + c, v);
                    tmem_wait();
                    keep(v);
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[b][j] += v[j];
                }
                tmem_st8(tl + L::SUM + c, acc[b]);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[b][j] = 0.f;
        }
        tmem_wait_st();
        summed = true;
    };
    for (long long it = i0; it < i1; ++it) {
        const int s = (int)(it % g.T), th = (int)(it / g.T), tile = th >> 1, r0 = (th & 1) * GR;
        const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
        const bool last = s + 1 == g.T;
        // the block's operands: 8 columns of a row a thread (rows fastest, so
        // that reads are contiguous); h, r and X are read while the products
        // of the block before run, the others brought into L2 meanwhile
        const bool mine = tid < GR * (H / 8);
        const int lr = tid & (GR - 1), lc = (tid / GR) * 8, tr = r0 + lr;   // row in the block and in the tile
        const size_t o = sb + blk(lc, tr), gz = ((size_t)s * g.ntiles + tile) * 3 * tblk + blk(lc, tr);
        const float *hnp = last ? g.hT + (size_t)(tile * TM + tr) * H + lc : g.hb + o + (size_t)g.ntiles * tblk;
        const int hstep = last ? 4 : 4 * TM;
        const bool hnok = !last || tile * TM + tr < g.P;
        const int xr = tid >> 3, xc = (tid & 7) * 8, fc = X0 + xc, gp = tile * TM + r0 + xr;   // X and dD: 8 threads a row
        const float *dsrc = g.dD + ((size_t)s * g.P + gp) * g.n_out + xc;
        float hp[8], rr[8], xv[8];
        if (mine) {
            if (!X2) {
                ld4(g.hb + o, hp); ld4(g.hb + o + 4 * TM, hp + 4);
                ld4(g.r + o, rr); ld4(g.r + o + 4 * TM, rr + 4);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                prefetch_l2(g.dG + gz + k * tblk);
                prefetch_l2(g.dG + gz + k * tblk + 4 * TM);
            }
            if (!X2 && hnok) {
                prefetch_l2(hnp);
                prefetch_l2(hnp + hstep);
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) xv[j] = 0.f;
        if (gp < g.P) {
            const float *src = g.X + ((size_t)s * g.P + gp) * g.ldx + fc;
            if (g.xvec) {
                if (fc < g.n_in) ld4(src, xv);
                if (fc + 4 < g.n_in) ld4(src + 4, xv + 4);
#pragma unroll
                for (int j = 0; j < 8; ++j) xv[j] = fc + j < g.n_in ? xv[j] : 0.f;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) xv[j] = fc + j < g.n_in ? __ldg(src + j) : 0.f;
            }
            if (!X2 && xc < g.n_out) prefetch_l2(dsrc);
        }
        if (it > i0) {
            drain(it - 1);   // the images are free again
            if ((it - i0) % G32_RUN == 0) flush();
        }
        float az[8], ar[8];
        if (mine) {
            ld4(g.dG + gz, az); ld4(g.dG + gz + 4 * TM, az + 4);
            ld4(g.dG + gz + tblk, ar); ld4(g.dG + gz + tblk + 4 * TM, ar + 4);
        }
        put8_3(base + L::X, GIMG, xr, xc, xv);
        if (mine) {
            if (!X2) {
                put8_3(base + L::HP, GIMG, lr, lc, hp);
#pragma unroll
                for (int j = 0; j < 8; ++j) rr[j] *= hp[j];
                put8_3(base + L::RH, GIMG, lr, lc, rr);
            }
            ld4(g.dG + gz + 2 * tblk, hp); ld4(g.dG + gz + 2 * tblk + 4 * TM, hp + 4);   // dA_c
#pragma unroll
            for (int j = 0; j < 8; ++j) rr[j] = 0.f;
            if (!X2 && hnok) {
                ld4(hnp, rr);
                ld4(hnp + hstep, rr + 4);
            }
            put8_3(base + L::GZ, GIMG, lr, lc, az);
            // H = 32: dA_z and dA_r side by side in one image
            if (H == 64) put8_3(base + L::GRR, GIMG, lr, lc, ar);
            else put8_3(base + L::GZ, GIMG, lr, H + lc, ar);
        }
        if (!X2 && xc < g.nfc) {
#pragma unroll
            for (int j = 0; j < 8; ++j) xv[j] = gp < g.P && xc + j < g.n_out ? __ldg(dsrc + j) : 0.f;
            put8_3(base + L::DD, GIMG, xr, xc, xv);
        }
        if (mine) {
            put8_3(base + L::GC, GIMG, lr, lc, hp);
            if (!X2) put8_3(base + L::HN, GIMG, lr, lc, rr);
        }
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma3_mn(cta.tmem, u + L::X, GIMG, L::HP - L::X, u + L::GZ, GIMG, L::GRR - L::GZ, 2 * H, GR);
            mma3_mn(cta.tmem + 2 * H, u + L::X, GIMG, L::RH - L::X, u + L::GC, GIMG, GIMG, H, GR);
            if (!X2) mma3_mn(cta.tmem + 3 * H, u + L::HN, GIMG, L::HP - L::X, u + L::DD, GIMG, GIMG, g.nfc, GR);
            tc_commit(cta.bar0);
        }
    }
    if (ok && i1 > i0) {
        drain(i1 - 1);
        flush();
    }
    if (ok && summed && !*cta.abort_flag) {
        float *o = g.part + (size_t)blockIdx.x * g.part_cols * TM;
        auto write = [&]() {
            Finite fin;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int c = 8 * (part + 4 * b);
                if (c >= ncol) continue;
                float v[8];
                tmem_ld8(tl + L::SUM + c, v);
                tmem_wait();
                keep(v);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    fin.see(v[j]);
                    o[(size_t)(out0 + c + j) * TM + row] = v[j];
                }
            }
            return fin.failed();
        };
        if (__any_sync(0xffffffffu, write())) {
            plain_grad<H, X2>(g, i0, i1, cta.tmem);
            write();
        }
    }
    cta.finish(1, L::COLS, g.status);
}

}  // namespace

namespace {
template <int H> cudaError_t forward(const WinArgs &g, cudaStream_t st) {
    const int sms = sm_count(), grid = std::min(g.ntiles, sms);
    if (!g.kx2) return launch(k_win32_fwd<H, 1>, grid, W32_TH, Fwd32Layout<H, 1>::BYTES, g, st);
    const cudaError_t e = launch(k_win32_x<H>, (int)std::min<long long>((long long)g.T * g.ntiles, sms), W32_TH,
                                 X32Layout<H>::BYTES, g, st);
    return e != cudaSuccess ? e : launch(k_win32_fwd<H, 2>, grid, W32_TH, Fwd32Layout<H, 2>::BYTES, g, st);
}
template <int H> cudaError_t backward(const WinArgs &g, cudaStream_t st) {
    const int grid = std::min(g.ntiles, sm_count()), ggrid = win32_parts(g.T, g.P);
    cudaError_t e = launch(k_win32_bwd<H>, grid, W32_TH, Bwd32Layout<H>::BYTES, g, st);
    if (e == cudaSuccess) e = launch(k_win32_grad<H, false>, ggrid, W32_TH, Grad32Layout<H>::BYTES, g, st);
    if (e == cudaSuccess && g.kx2) e = launch(k_win32_grad<H, true>, ggrid, W32_TH, Grad32Layout<H>::BYTES, g, st);
    return e != cudaSuccess ? e : win_reduce(g, H, ggrid, 0, st);
}
}  // namespace

cudaError_t win32_forward(const WinArgs &g, int H, cudaStream_t st) { return H == 64 ? forward<64>(g, st) : forward<32>(g, st); }
cudaError_t win32_backward(const WinArgs &g, int H, cudaStream_t st) {
    return H == 64 ? backward<64>(g, st) : backward<32>(g, st);
}

// CTAs of the weight-gradient kernel, each with a partial sum of its own
int win32_parts(int T, int P) { return (int)std::min<long long>(2LL * T * win_tiles(P), sm_count()); }

}  // namespace dnnmg

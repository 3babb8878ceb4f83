// The training window of the patch network with BF16 products, as two
// persistent kernels: forward over T steps (Eq. gru and the output layer) and
// truncated backpropagation through time with the weight gradients.
//
// Patch rows are independent, so a CTA takes 128 of them (one tensor-memory
// lane a row) through the whole window: weights stay in shared memory as
// BF16 operand images, the state and the carried gradient in registers, every
// product is a tcgen05 MMA between images the same threads wrote, and only
// the window's inputs, outputs and saved activations touch memory.  A kernel
// per product (with FP32 intermediates and BF16 copies of every operand in
// memory between them) took 4.07 ms for loss and gradients of 65 536 rows, T =
// 10, H = 64; this takes 0.62 ms, of it forward 266 us, backward 256 us and
// the sum of the partial gradients 15 us (ncu).  With 99 features (two chunks)
// and 50 outputs 4.65 ms became 0.96 ms, forward 383 us, backward 399 us.
//
// Arithmetic is that of the kernel-per-product path (gru_train.cu): operands
// are rounded to BF16 where it rounds them, X W_x^T and h U^T are accumulated
// apart and added in FP32, gates and updates are FP32.  The weight gradients
// accumulate in tensor memory over a CTA's rows and steps, and the CTAs'
// partial sums are added in a fixed order, so they repeat bit for bit.
//
// Saved activations (z, r, c and h_0 .. h_{T-1}, FP32) are laid out
// [step][tile][column / 4][row][4]: a warp, whose lanes are rows, moves 512
// contiguous bytes per 4 columns.
//
// Every wait is bounded (2 s): on time-out the kernel sets
// DNNMG_DEVERR_TIMEOUT in *status, drains its MMAs, frees its tensor memory
// and returns.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "gru_win.cuh"
#include "gru_win_dev.cuh"

namespace dnnmg {
namespace {

constexpr int BWD_TH = 512;

// ---------------------------------------------------------------- forward
// XC = 1 (n_in <= 64): two CTAs an SM (each 256 threads, two per row, and half
// the tensor memory), so that one computes while the other waits for its MMAs.
// XC = 2 (n_in <= 128): the second chunk of W_x and X leaves room for one, of
// 512 threads.  Tensor memory
// columns: X W_zr^T [0, 2H), h U_zr^T [2H, 4H); once r has been read,
// X W_h^T [H, 2H) and (r h) U_h^T [3H, 4H); then the output layer [0, nfc).
// Bound by instruction issue (gate functions and conversions) and, close
// behind, by memory (1.2 kB a row and step).
template <int H, int XC> struct FwdLayout {
    static constexpr int TH = XC == 1 ? 256 : 512, CTAS = XC == 1 ? 2 : 1;
    static constexpr int WX = 0, U = WX + XC * 3 * H * 128, F = U + 3 * H * 128, X = F + 64 * 128, HI = X + XC * IMG,
                         BARS = HI + IMG, BYTES = BARS + 64 + 1024;
    static constexpr int COLS = 4 * H;
};

template <int H, int XC>
__global__ void __launch_bounds__(FwdLayout<H, XC>::TH, FwdLayout<H, XC>::CTAS) k_win_fwd(const WinArgs g) {
    using L = FwdLayout<H, XC>;
    constexpr int TH = L::TH, PARTS = TH / TM, NH = H / PARTS;   // threads a row, state columns of each
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw);
    uint8_t *sX = base + L::X, *sH = base + L::HI;
    const uint32_t uWx = smem_u32(base + L::WX), uU = smem_u32(base + L::U), uF = smem_u32(base + L::F),
                   uX = smem_u32(sX), uH = smem_u32(sH);
    for (int x = 0; x < XC; ++x)
        build(base + L::WX + x * 3 * H * 128, 3 * H, TH, [&](int r, int c) {
            return 64 * x + c < g.n_in ? __ldg(g.Wx + (size_t)r * g.n_in + 64 * x + c) : 0.f;
        });
    build(base + L::U, 3 * H, TH, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)r * H + c) : 0.f; });
    build(base + L::F, g.nfc, TH, [&](int r, int c) { return r < g.n_out && c < H ? __ldg(g.Wfc + (size_t)r * H + c) : 0.f; });
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 2, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane, c0 = part * NH;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    uint32_t ph = 0;   // phase of the MMA barrier
    bool ok = true;
    XTile<TH> xt[XC];
    auto load_x = [&](int s, int p0) {
#pragma unroll
        for (int x = 0; x < XC; ++x) xt[x].load(g, s, p0, 64 * x);
    };
    auto store_x = [&]() {
#pragma unroll
        for (int x = 0; x < XC; ++x) xt[x].store(g, sX + x * IMG, 64 * x);
    };
    // the products of columns [n0, n0 + N) of W_x with X
    auto mma_x = [&](uint32_t d, int n0, int N) {
        mma_k(d, uX, uWx + n0 * 128, N, 4, false);
        if (XC == 2) mma_k(d, uX + IMG, uWx + (3 * H + n0) * 128, N, g.kx2, true);
    };
    for (int tile = blockIdx.x; ok && tile < g.ntiles; tile += gridDim.x) {
        const int p0 = tile * TM, gp = p0 + row;
        const bool valid = gp < g.P;
        float hv[NH];
        load_x(0, p0);
#pragma unroll
        for (int i = 0; i < NH; i += 4) {
            hv[i] = hv[i + 1] = hv[i + 2] = hv[i + 3] = 0.f;
            if (g.h0 && valid) ld4(g.h0 + (size_t)gp * H + c0 + i, hv + i);
        }
        const size_t tblk = (size_t)TM * H;
#pragma unroll
        for (int i = 0; i < NH; i += 4) st4(g.hb + (size_t)tile * tblk + blk(c0 + i, row), hv + i);
#pragma unroll
        for (int i = 0; i < NH; i += 8) put8(sH, row, c0 + i, hv + i);
        store_x();
        for (int s = 0; s < g.T; ++s) {
            const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma_x(cta.tmem, 0, 2 * H);
                mma_k(cta.tmem + 2 * H, uH, uU, 2 * H, H / 16, false);
                tc_commit(cta.bar0);
            }
            ok = cta.wait(0, ph);
            ph ^= 1;
            // r and r h
#pragma unroll
            for (int i = 0; i < NH; i += 8) {
                float a[8], b[8], rr[8];
                tmem_ld8(tl + H + c0 + i, a);
                tmem_ld8(tl + 3 * H + c0 + i, b);
                tmem_wait();
                keep(a);
                keep(b);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    rr[j] = sigm(a[j] + b[j]);
                    a[j] = rr[j] * hv[i + j];
                }
                st4(g.r + sb + blk(c0 + i, row), rr);
                st4(g.r + sb + blk(c0 + i + 4, row), rr + 4);
                put8(sH, row, c0 + i, a);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma_x(cta.tmem + H, 2 * H, H);
                mma_k(cta.tmem + 3 * H, uH, uU + 2 * H * 128, H, H / 16, false);
                tc_commit(cta.bar0);
            }
            ok = cta.wait(0, ph);
            ph ^= 1;
            // candidate and new state
#pragma unroll
            for (int i = 0; i < NH; i += 8) {
                float a[8], b[8], zz[8], cc[8];
                tmem_ld8(tl + c0 + i, a);
                tmem_ld8(tl + 2 * H + c0 + i, b);
                tmem_ld8(tl + H + c0 + i, zz);
                tmem_ld8(tl + 3 * H + c0 + i, cc);
                tmem_wait();
                keep(a);
                keep(b);
                keep(zz);
                keep(cc);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float z = sigm(a[j] + b[j]), c = tanhf(zz[j] + cc[j]);
                    zz[j] = z;
                    cc[j] = c;
                    hv[i + j] = z * hv[i + j] + (1.0f - z) * c;
                }
                st4(g.z + sb + blk(c0 + i, row), zz);
                st4(g.z + sb + blk(c0 + i + 4, row), zz + 4);
                st4(g.c + sb + blk(c0 + i, row), cc);
                st4(g.c + sb + blk(c0 + i + 4, row), cc + 4);
                put8(sH, row, c0 + i, hv + i);
            }
            if (s + 1 < g.T) {
                load_x(s + 1, p0);
                float *hb = g.hb + ((size_t)(s + 1) * g.ntiles + tile) * tblk;
#pragma unroll
                for (int i = 0; i < NH; i += 4) st4(hb + blk(c0 + i, row), hv + i);
            } else if (valid) {
#pragma unroll
                for (int i = 0; i < NH; i += 4) st4(g.hT + (size_t)gp * H + c0 + i, hv + i);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma_k(cta.tmem, uH, uF, g.nfc, H / 16, false);
                tc_commit(cta.bar0);
            }
            if (s + 1 < g.T) store_x();
            ok = cta.wait(0, ph);
            ph ^= 1;
            // outputs: blocks of 8 columns, dealt to the threads of a row
            float *drow = g.D + ((size_t)s * g.P + gp) * g.n_out;
            for (int b = part; b < g.nfc / 8; b += PARTS) {
                float v[8];
                tmem_ld8(tl + 8 * b, v);
                tmem_wait();
                keep(v);
                if (!valid) continue;
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
        }
        ok = cta.hand_over(ok);   // (the same answer in every thread)
    }
    cta.finish(1, L::COLS, g.status);
}

// ---------------------------------------------------------------- backward
// One CTA an SM, 512 threads (four per row).  Per step, last first:
//   dh = dD W_fc + carry; dA_z, dA_c; images of h_{s}, r h_{s}, h_{s+1}, dA_z, dA_c
//   MMA: d(r h) = dA_c U_h
//   dA_r and the carry's part that does not pass through U_z, U_r
//   MMA: [dA_z, dA_r] [U_z; U_r] and the next step's dD W_fc, then the
//   weight gradients [X | h]^T [dA_z, dA_r], [X | r h]^T dA_c and h_{s+1}^T dD
//   into their accumulators, which run while the next step's elements do.
// Tensor memory, XC = 1: carry part [0, H), dD W_fc [64, 64 + H), d(r h) [128,
// 128 + H), gradients [192, 192 + 2H), [320, 320 + H), [384, 384 + nfc).  XC = 2
// (features 64 ..) has gradients of its own, so the carry's products add to
// dD W_fc, and d(r h) takes their place once they have been read.
// Bound by the chain of the two MMA round trips a step and the element work
// between them; memory (1.4 kB a row and step) is close behind.
template <int H, int XC> struct BwdLayout {
    static constexpr int X = 0, HP = X + XC * IMG, RH = HP + IMG, HN = RH + IMG, GZR = HN + IMG,
                         GC = GZR + (H == 64 ? 2 : 1) * IMG, DD = GC + IMG, WF = DD + 2 * IMG, UC = WF + H * 128,
                         UZR = UC + H * 128, BARS = UZR + (H == 64 ? 2 : 1) * H * 128, BYTES = BARS + 64 + 1024;
    static constexpr int COLS = 512;
    static constexpr int CARRY = 0, DH = XC == 1 ? 64 : 0, DRH = XC == 1 ? 128 : 0;
    // [X | h]^T [dA_z dA_r], [X | r h]^T dA_c, h_{s+1}^T dD (rows 64 .. of it with XC = 2), second chunk
    static constexpr int G1 = XC == 1 ? 192 : 64, G2 = G1 + 128, G3 = XC == 1 ? 384 : 448, G4 = 256, G5 = 384;
};

template <int H, int XC>
__global__ void __launch_bounds__(BWD_TH, 1) k_win_bwd(const WinArgs g) {
    using L = BwdLayout<H, XC>;
    constexpr int NC = H / 4;   // state columns of a thread: 16 or 8
    constexpr int T_CARRY = L::CARRY, T_DH = L::DH, T_DRH = L::DRH;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = align1k(smem_raw);
    const uint32_t u = smem_u32(base);
    // operands of the state gradients: rows are the products' columns
    build(base + L::WF, H, BWD_TH, [&](int r, int c) { return c < g.n_out ? __ldg(g.Wfc + (size_t)c * H + r) : 0.f; });
    build(base + L::UC, H, BWD_TH, [&](int r, int c) { return c < H ? __ldg(g.Uh + (size_t)(2 * H + c) * H + r) : 0.f; });
    for (int k = 0; k < (H == 64 ? 2 : 1); ++k)
        build(base + L::UZR + k * H * 128, H, BWD_TH, [&](int r, int c) { return __ldg(g.Uh + (size_t)(64 * k + c) * H + r); });
    // columns that no step writes but the MMAs of unused gradient rows read
    build(base + L::HP, TM, BWD_TH, [&](int, int) { return 0.f; });
    build(base + L::RH, TM, BWD_TH, [&](int, int) { return 0.f; });
    build(base + L::HN, TM, BWD_TH, [&](int, int) { return 0.f; });
    build(base + L::GC, TM, BWD_TH, [&](int, int) { return 0.f; });
    build(base + L::DD, TM, BWD_TH, [&](int, int) { return 0.f; });
    build(base + L::DD + IMG, TM, BWD_TH, [&](int, int) { return 0.f; });
    Cta cta;
    cta.init(reinterpret_cast<uint64_t *>(base + L::BARS), 4, L::COLS);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, part = warp >> 2, row = q * 32 + lane, c0 = part * NC;
    const uint32_t tl = cta.tmem + ((uint32_t)(q * 32) << 16);
    uint32_t ph0 = 0, ph1 = 0, ph2 = 0;   // state part, gradients, d(r h)
    bool ok = true, grads = false;        // grads: the accumulators hold something
    const size_t tblk = (size_t)TM * H;
    XTile<BWD_TH> xt;
    float zv[NC], rv[NC], cv[NC], hp[NC];
    // (rows past the last patch add nothing to the weight gradients, also where
    // an infinite weight makes NaNs of them: activations and gradients of 0)
    auto load_step = [&](int s, int tile) {
        const size_t sb = ((size_t)s * g.ntiles + tile) * tblk;
        const bool valid = tile * TM + row < g.P;
#pragma unroll
        for (int i = 0; i < NC; i += 4) {
            const size_t o = sb + blk(c0 + i, row);
            if (!valid) {
#pragma unroll
                for (int j = i; j < i + 4; ++j) zv[j] = rv[j] = cv[j] = hp[j] = 0.f;
                continue;
            }
            ld4(g.z + o, zv + i);
            ld4(g.r + o, rv + i);
            ld4(g.c + o, cv + i);
            ld4(g.hb + o, hp + i);
        }
    };
    // dD rows of a step into their image (one of two), each thread a few columns of its row
    auto load_dd = [&](int s, int p0) {
        uint8_t *img = base + L::DD + (s & 1) * IMG;
        const int gp = p0 + row;
        const float *src = g.dD + ((size_t)s * g.P + gp) * g.n_out;
        if (g.pairs) {
            for (int c = 2 * part; c < g.n_out; c += 8) {
                float2 v = make_float2(0.f, 0.f);
                if (gp < g.P) v = __ldg(reinterpret_cast<const float2 *>(src + c));
                *reinterpret_cast<uint32_t *>(img + swz(row, c >> 3) + (c & 7) * 2) = pack(v.x, v.y);
            }
        } else {
            for (int c = part; c < g.n_out; c += 4) put1(img, row, c, gp < g.P ? __ldg(src + c) : 0.f);
        }
    };
    const int kfc = g.nfc / 16;
    for (int tile = blockIdx.x; ok && tile < g.ntiles; tile += gridDim.x) {
        const int p0 = tile * TM, gp = p0 + row;
        const bool valid = gp < g.P;
        float cpart[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) cpart[i] = 0.f;
        // (the previous tile's gradients have been waited for before its images are reused: below)
        if (grads) {
            ok = cta.wait(1, ph1);
            ph1 ^= 1;
        }
        if (!(ok = cta.hand_over(ok))) break;
        load_dd(g.T - 1, p0);
        load_step(g.T - 1, tile);
        xt.load(g, g.T - 1, p0);
        if (XC == 2) xt.prefetch(g, g.T - 1, p0, 64);
        if (!(ok = cta.hand_over(ok))) break;
        if (tid == 0) {
            mma_k(cta.tmem + T_DH, u + L::DD + ((g.T - 1) & 1) * IMG, u + L::WF, H, kfc, false);
            tc_commit(cta.bar0);
        }
        for (int s = g.T - 1; s >= 0; --s) {
            ok = cta.wait(0, ph0);
            ph0 ^= 1;
            float dh[NC], az[NC], ac[NC];
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8], b[8];
                tmem_ld8(tl + T_DH + c0 + i, a);
                if (XC == 1) tmem_ld8(tl + T_CARRY + c0 + i, b);
                tmem_wait();
                keep(a);
                if (XC == 1) keep(b);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = i + j;
                    const float carry = s == g.T - 1 ? 0.f : (XC == 1 ? b[j] + cpart[k] : cpart[k]);
                    dh[k] = valid ? a[j] + carry : 0.f;
                    const float dc = dh[k] * (1.0f - zv[k]), dz = dh[k] * (hp[k] - cv[k]);
                    az[k] = dz * zv[k] * (1.0f - zv[k]);
                    ac[k] = dc * (1.0f - cv[k] * cv[k]);
                }
            }
            // the images may be overwritten once the step before's gradients are done
            if (s < g.T - 1) {
                ok = cta.wait(1, ph1) && ok;
                ph1 ^= 1;
            }
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float t[8];
                put8(base + L::HP, row, c0 + i, hp + i);
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = rv[i + j] * hp[i + j];
                put8(base + L::RH, row, c0 + i, t);
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = zv[i + j] * hp[i + j] + (1.0f - zv[i + j]) * cv[i + j];
                put8(base + L::HN, row, c0 + i, t);
                put8(base + L::GZR, row, c0 + i, az + i);
                put8(base + L::GC, row, c0 + i, ac + i);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma_k(cta.tmem + T_DRH, u + L::GC, u + L::UC, H, H / 16, false);
                tc_commit(cta.bar0 + 16);
            }
            xt.store(g, base + L::X);
            if (XC == 2) {
                xt.load(g, s, p0, 64);
                xt.store(g, base + L::X + IMG, 64);
            }
            if (s > 0) load_dd(s - 1, p0);
            ok = cta.wait(2, ph2);
            ph2 ^= 1;
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float a[8];
                tmem_ld8(tl + T_DRH + c0 + i, a);
                tmem_wait();
                keep(a);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = i + j;
                    if (!valid) a[j] = 0.f;
                    cpart[k] = dh[k] * zv[k] + a[j] * rv[k];
                    a[j] = a[j] * hp[k] * rv[k] * (1.0f - rv[k]);
                }
                // columns H .. 2H-1 of [dA_z, dA_r]
                if (H == 64) put8(base + L::GZR + IMG, row, c0 + i, a);
                else put8(base + L::GZR, row, H + c0 + i, a);
            }
            if (s > 0) {
                load_step(s - 1, tile);
                xt.load(g, s - 1, p0);
                if (XC == 2) xt.prefetch(g, s - 1, p0, 64);
            }
            if (!(ok = cta.hand_over(ok))) break;
            if (tid == 0) {
                mma_k(cta.tmem + T_CARRY, u + L::GZR, u + L::UZR, H, 4, false);
                if (H == 64) mma_k(cta.tmem + T_CARRY, u + L::GZR + IMG, u + L::UZR + H * 128, H, 4, true);
                if (s > 0) mma_k(cta.tmem + T_DH, u + L::DD + ((s - 1) & 1) * IMG, u + L::WF, H, kfc, XC == 2);
                tc_commit(cta.bar0);
                mma_mn(cta.tmem + L::G1, desc_mn(u + L::X, L::HP - L::X), desc_mn(u + L::GZR, IMG), 2 * H, grads);
                mma_mn(cta.tmem + L::G2, desc_mn(u + L::X, L::RH - L::X), desc_mn(u + L::GC, IMG), H, grads);
                if (XC == 1) {
                    mma_mn(cta.tmem + L::G3, desc_mn(u + L::HN, L::HP - L::X), desc_mn(u + L::DD + (s & 1) * IMG, IMG), g.nfc, grads);
                } else {
                    const uint64_t a = desc_mn(u + L::X + IMG, L::HN - L::X - IMG);   // [X's second chunk | h_{s+1}]
                    mma_mn(cta.tmem + L::G4, a, desc_mn(u + L::GZR, IMG), 2 * H, grads);
                    mma_mn(cta.tmem + L::G5, a, desc_mn(u + L::GC, IMG), H, grads);
                    mma_mn(cta.tmem + L::G3, a, desc_mn(u + L::DD + (s & 1) * IMG, IMG), g.nfc, grads);
                }
                tc_commit(cta.bar0 + 8);
            }
            grads = true;
        }
        if (!ok) break;
        // gradient of h_0
        ok = cta.wait(0, ph0);
        ph0 ^= 1;
        if (g.dh0) {
#pragma unroll
            for (int i = 0; i < NC; i += 8) {
                float b[8];
                tmem_ld8(tl + T_CARRY + c0 + i, b);
                tmem_wait();
                keep(b);
#pragma unroll
                for (int j = 0; j < 8; ++j) b[j] += cpart[i + j];
                if (gp < g.P) {
                    st4(g.dh0 + (size_t)gp * H + c0 + i, b);
                    st4(g.dh0 + (size_t)gp * H + c0 + i + 4, b + 4);
                }
            }
        }
        ok = cta.hand_over(ok);   // (the same answer in every thread)
    }
    // this CTA's sums: [column][lane], gradients of W_x (lanes 0 .. 63) and U (64 ..), then of W_fc,
    // then of W_x's second chunk
    if (ok && grads) {
        ok = cta.wait(1, ph1);
        ph1 ^= 1;
    }
    if (ok && !*cta.abort_flag) {
        float *o = g.part + (size_t)blockIdx.x * g.part_cols * TM;
        const int ncol = g.part_cols, x2 = 3 * H + g.nfc;
        for (int b = part; b < ncol / 8; b += 4) {
            const int c = 8 * b;
            int t = c < 2 * H ? L::G1 + c : (c < 3 * H ? L::G2 + c - 2 * H : L::G3 + c - 3 * H);
            if (XC == 2 && c >= x2) t = c - x2 < 2 * H ? L::G4 + c - x2 : L::G5 + c - x2 - 2 * H;
            float v[8];
            tmem_ld8(tl + t, v);
            tmem_wait();
            keep(v);
#pragma unroll
            for (int j = 0; j < 8; ++j) o[(size_t)(c + j) * TM + row] = v[j];
        }
    }
    cta.finish(3, L::COLS, g.status);
}

// Sums of the CTAs' partial gradients, in the order of the CTAs and without
// their rounding errors (TwoSum: an FP32 sum of 152 parts in sequence is off
// by about as much as everything before it).
__global__ void __launch_bounds__(TM) k_win_reduce(const WinArgs g, int H, int nparts, int fc_lane) {
    const int c = blockIdx.x, m = threadIdx.x;
    const float *p = g.part + (size_t)c * TM + m;
    const size_t stride = (size_t)g.part_cols * TM;
    float s = 0.f, lo = 0.f;
#pragma unroll 8
    for (int i = 0; i < nparts; ++i) {
        const float x = p[i * stride], t = __fadd_rn(s, x), bb = __fsub_rn(t, s);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(x, bb)));
        s = t;
    }
    if (lo == lo) s += lo;   // (an infinite sum keeps its value)
    if (c < 3 * H) {
        if (m < g.n_in && m < 64) g.gWx[(size_t)c * g.n_in + m] = s;
        if (m >= 64 && m < 64 + H) g.gUh[(size_t)c * H + m - 64] = s;
    } else if (c < 3 * H + g.nfc) {
        if (c - 3 * H < g.n_out && m >= fc_lane && m < fc_lane + H) g.gWfc[(size_t)(c - 3 * H) * H + m - fc_lane] = s;
    } else if (m < 64 && 64 + m < g.n_in) {
        g.gWx[(size_t)(c - 3 * H - g.nfc) * g.n_in + 64 + m] = s;
    }
}

}  // namespace

// Shapes the window kernels take: one or two 64-column chunks of features, H =
// 32 or 64, up to 64 outputs (the K = 1 and K = 2 networks of one-cell
// patches); the others run one kernel per product.
bool win_supported(int n_in, int H, int n_out) { return n_in <= 128 && (H == 32 || H == 64) && n_out <= 64; }
int win_tiles(int P) { return (P + TM - 1) / TM; }
size_t win_part_floats(int n_in, int H, int n_out, int T, int P) {
    return (size_t)win32_parts(T, P) * ((n_in > 64 ? 6 : 3) * H + round_up(n_out, 16)) * TM;   // (at least win_tiles(P) or one per SM)
}

namespace {
template <int H, int XC> cudaError_t forward(const WinArgs &g, cudaStream_t st) {
    using L = FwdLayout<H, XC>;
    return launch(k_win_fwd<H, XC>, std::min(g.ntiles, L::CTAS * sm_count()), L::TH, L::BYTES, g, st);
}
template <int H, int XC> cudaError_t backward(const WinArgs &g, int grid, cudaStream_t st) {
    return launch(k_win_bwd<H, XC>, grid, BWD_TH, BwdLayout<H, XC>::BYTES, g, st);
}
}  // namespace

cudaError_t win_forward(const WinArgs &g, int H, cudaStream_t st) {
    if (H == 64) return g.kx2 ? forward<64, 2>(g, st) : forward<64, 1>(g, st);
    return g.kx2 ? forward<32, 2>(g, st) : forward<32, 1>(g, st);
}

cudaError_t win_backward(const WinArgs &g, int H, cudaStream_t st) {
    const int grid = std::min(g.ntiles, sm_count());
    cudaError_t e;
    if (H == 64) e = g.kx2 ? backward<64, 2>(g, grid, st) : backward<64, 1>(g, grid, st);
    else e = g.kx2 ? backward<32, 2>(g, grid, st) : backward<32, 1>(g, grid, st);
    if (e != cudaSuccess) return e;
    return win_reduce(g, H, grid, g.kx2 ? 64 : 0, st);
}

// fc_lane: the lane of the first row of W_fc's gradient
cudaError_t win_reduce(const WinArgs &g, int H, int nparts, int fc_lane, cudaStream_t st) {
    k_win_reduce<<<g.part_cols, TM, 0, st>>>(g, H, nparts, fc_lane);
    return cudaGetLastError();
}

}  // namespace dnnmg

// S4 on CUDA cores: GRU cell (Eq. gru, reset gate before U_h, no biases) and
// the fully connected output layer, TP patches per CTA.
//
// Weights are stored transposed (WxT [ldx][3H], UhT [H][3H], WfcT [H][n_out])
// so that consecutive threads, which own consecutive output rows, read
// consecutive addresses; the CTA's patch rows sit in shared memory and are
// read as broadcasts.  Precisions:
//   F64      double operands, double accumulation
//   F32      float operands, float accumulation
//   BF16NET  bfloat16 GEMM operands (X, weights, h, r*h and h' rounded to
//            bfloat16), float accumulation and float gate arithmetic; the
//            stored state h stays float.  This is the same arithmetic as the
//            tensor-core kernel, so the two can be compared tightly.
#include "common.cuh"

namespace dnnmg {
namespace {

template <typename TW> struct Acc { using type = TW; };
template <> struct Acc<__nv_bfloat16> { using type = float; };

template <typename A> __device__ __forceinline__ A load_as(const __nv_bfloat16 *p) {
    return (A)__bfloat162float(*p);
}
template <typename A> __device__ __forceinline__ A load_as(const float *p) { return (A)*p; }
template <typename A> __device__ __forceinline__ A load_as(const double *p) { return (A)*p; }

// value of x as the GEMM operand type sees it
template <typename TW, typename A> __device__ __forceinline__ A quant(A x) { return x; }
template <> __device__ __forceinline__ float quant<__nv_bfloat16, float>(float x) {
    return __bfloat162float(__float2bfloat16_rn(x));
}

__device__ __forceinline__ double sigm(double x) { return 1.0 / (1.0 + exp(-x)); }
__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ double tanh_(double x) { return tanh(x); }
__device__ __forceinline__ float tanh_(float x) { return tanhf(x); }

constexpr int NT = 256;

template <typename T, typename TW, int TP>
__global__ void __launch_bounds__(NT)
k_gru(int n_in, int ldx, int H, int n_out, const TW *__restrict__ X, const TW *__restrict__ WxT,
      const TW *__restrict__ UhT, const TW *__restrict__ WfcT, T *__restrict__ h,
      T *__restrict__ d, int P) {
    using A = typename Acc<TW>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    A *xs = reinterpret_cast<A *>(smem_raw);  // [TP][ldx]  features
    A *hs = xs + TP * ldx;                    // [TP][H]    previous state (float / double)
    A *hq = hs + TP * H;                      // [TP][H]    previous state as GEMM operand
    A *zs = hq + TP * H;                      // [TP][H]    update gate
    A *rh = zs + TP * H;                      // [TP][H]    r * h (operand)
    A *gh = rh + TP * H;                      // [TP][H]    W_h x
    A *hn = gh + TP * H;                      // [TP][H]    new state (operand)
    const int p0 = blockIdx.x * TP;
    const int np = min(TP, P - p0);
    const int G = 3 * H;

    for (int i = threadIdx.x; i < TP * ldx; i += blockDim.x) {
        const int p = i / ldx, k = i - p * ldx;
        xs[i] = (p < np && k < n_in) ? load_as<A>(X + (size_t)(p0 + p) * ldx + k) : A(0);
    }
    for (int i = threadIdx.x; i < TP * H; i += blockDim.x) {
        const int p = i / H;
        const A v = p < np ? (A)h[(size_t)p0 * H + i] : A(0);
        hs[i] = v;
        hq[i] = quant<TW, A>(v);
    }
    __syncthreads();

    // z, r and W_h x
    for (int j = threadIdx.x; j < G; j += blockDim.x) {
        A acc[TP];
#pragma unroll
        for (int p = 0; p < TP; ++p) acc[p] = A(0);
        for (int k = 0; k < n_in; ++k) {
            const A w = load_as<A>(WxT + (size_t)k * G + j);
#pragma unroll
            for (int p = 0; p < TP; ++p) acc[p] += w * xs[p * ldx + k];
        }
        if (j < 2 * H) {
            for (int k = 0; k < H; ++k) {
                const A w = load_as<A>(UhT + (size_t)k * G + j);
#pragma unroll
                for (int p = 0; p < TP; ++p) acc[p] += w * hq[p * H + k];
            }
        }
        if (j < H) {
#pragma unroll
            for (int p = 0; p < TP; ++p) zs[p * H + j] = sigm(acc[p]);
        } else if (j < 2 * H) {
#pragma unroll
            for (int p = 0; p < TP; ++p)
                rh[p * H + j - H] = quant<TW, A>(sigm(acc[p]) * hs[p * H + j - H]);
        } else {
#pragma unroll
            for (int p = 0; p < TP; ++p) gh[p * H + j - 2 * H] = acc[p];
        }
    }
    __syncthreads();

    // candidate and state update
    for (int j = threadIdx.x; j < H; j += blockDim.x) {
        A acc[TP];
#pragma unroll
        for (int p = 0; p < TP; ++p) acc[p] = gh[p * H + j];
        for (int k = 0; k < H; ++k) {
            const A w = load_as<A>(UhT + (size_t)k * G + 2 * H + j);
#pragma unroll
            for (int p = 0; p < TP; ++p) acc[p] += w * rh[p * H + k];
        }
#pragma unroll
        for (int p = 0; p < TP; ++p) {
            const A z = zs[p * H + j];
            const A hnew = z * hs[p * H + j] + (A(1) - z) * tanh_(acc[p]);
            hn[p * H + j] = quant<TW, A>(hnew);
            if (p < np) h[(size_t)(p0 + p) * H + j] = (T)hnew;
        }
    }
    __syncthreads();

    // output layer d = W_fc h'
    for (int o = threadIdx.x; o < n_out; o += blockDim.x) {
        A acc[TP];
#pragma unroll
        for (int p = 0; p < TP; ++p) acc[p] = A(0);
        for (int k = 0; k < H; ++k) {
            const A w = load_as<A>(WfcT + (size_t)k * n_out + o);
#pragma unroll
            for (int p = 0; p < TP; ++p) acc[p] += w * hn[p * H + k];
        }
#pragma unroll
        for (int p = 0; p < TP; ++p)
            if (p < np) d[(size_t)(p0 + p) * n_out + o] = (T)acc[p];
    }
}

// FP32 and FP64 networks with H a multiple of 4: register tiles.  A CTA takes
// TP patches; a thread owns JT consecutive gate (or output) columns of PT
// patches, so one read of JT weights and PT staged values feeds JT x PT
// multiply-adds (one column a thread read 16 staged values for 16).  Staged
// values lie patch-fastest in shared memory; the lanes of a warp take
// consecutive column groups, so weights are read along rows and staged values
// as broadcasts.  Each sum runs over the inputs, then the state, one FMA
// after the other from zero, as k_gru's does: the same bits.
// FP32: 8 patches and 4 columns a thread, operations on patch pairs in packed
// form.  16 336 patches, 99 inputs, H = 64, 50 outputs: k_gru 123 us,
// this 64 us; bound by the weights' way from L2 (each CTA reads all of them).  FP64 runs at two FMA a clock and SM, so
// there the tile is small (2 columns of 1 patch) and few patches are spread
// over the chip: 254 patches, 51 inputs, H = 32: k_gru 83 us (32 CTAs), this
// 38 us (both under ncu, cold caches).
template <typename T, int JT, int PT> struct RTile {
    T a[JT][PT];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < JT; ++j)
#pragma unroll
            for (int p = 0; p < PT; ++p) a[j][p] = T(0);
    }
    // a += W[0 .. n)[j] x[0 .. n)[p], rows of W ldw apart, of x ldp apart
    __device__ __forceinline__ void mac(const T *__restrict__ W, int ldw, const T *x, int ldp, int n);
};
template <> __device__ __forceinline__ void RTile<float, 4, 8>::mac(const float *__restrict__ W, int ldw, const float *x,
                                                                   int ldp, int n) {
    unsigned long long c[4][4];   // patch pairs
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int p = 0; p < 4; ++p) asm("mov.b64 %0, {%1, %2};" : "=l"(c[j][p]) : "f"(a[j][2 * p]), "f"(a[j][2 * p + 1]));
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const float4 w = __ldg(reinterpret_cast<const float4 *>(W + (size_t)k * ldw));
        const ulonglong2 x0 = *reinterpret_cast<const ulonglong2 *>(x + k * ldp);
        const ulonglong2 x1 = *reinterpret_cast<const ulonglong2 *>(x + k * ldp + 4);
        const unsigned long long xv[4] = {x0.x, x0.y, x1.x, x1.y};
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            unsigned long long ww;
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww) : "f"(wv[j]));
#pragma unroll
            for (int p = 0; p < 4; ++p) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c[j][p]) : "l"(ww), "l"(xv[p]));
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int p = 0; p < 4; ++p) asm("mov.b64 {%0, %1}, %2;" : "=f"(a[j][2 * p]), "=f"(a[j][2 * p + 1]) : "l"(c[j][p]));
}
template <> __device__ __forceinline__ void RTile<double, 2, 1>::mac(const double *__restrict__ W, int ldw, const double *x,
                                                                    int ldp, int n) {
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const double2 w = __ldg(reinterpret_cast<const double2 *>(W + (size_t)k * ldw));
        const double xv = x[k * ldp];
        a[0][0] = fma(w.x, xv, a[0][0]);
        a[1][0] = fma(w.y, xv, a[1][0]);
    }
}

template <typename T, int TP, int JT, int PT, int THREADS>
__global__ void __launch_bounds__(THREADS)
k_gru_rt(int n_in, int ldx, int H, int n_out, int ldo, const T *__restrict__ X, const T *__restrict__ WxT,
         const T *__restrict__ UhT, const T *__restrict__ WfcT, T *__restrict__ h, T *__restrict__ d, int P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LP = TP + (TP > 4 ? 16 / (int)sizeof(T) : 0);   // staged row length (padded against bank conflicts)
    T *xs = reinterpret_cast<T *>(smem_raw);   // [n_in][LP] features
    T *hs = xs + n_in * LP;                    // [H][LP] previous state
    T *zs = hs + H * LP;                       // [H][LP] update gate
    T *rh = zs + H * LP;                       // [H][LP] r * h
    T *gh = rh + H * LP;                       // [H][LP] W_h x, then the new state
    const int p0 = blockIdx.x * TP, np = min(TP, P - p0), G = 3 * H;
    for (int i = threadIdx.x; i < TP * n_in; i += THREADS) {
        const int p = i / n_in, k = i - p * n_in;
        xs[k * LP + p] = p < np ? __ldg(X + (size_t)(p0 + p) * ldx + k) : T(0);
    }
    for (int i = threadIdx.x; i < TP * H; i += THREADS) {
        const int p = i / H, k = i - p * H;
        hs[k * LP + p] = p < np ? h[(size_t)(p0 + p) * H + k] : T(0);
    }
    __syncthreads();
    constexpr int PG = TP / PT;
    RTile<T, JT, PT> t;
    // z, r and W_h x: a tile lies in one gate (H is a multiple of JT)
    for (int e = threadIdx.x; e < G / JT * PG; e += THREADS) {
        const int jg = e % (G / JT), pg = e / (G / JT), j = jg * JT, p = pg * PT, gate = j / H, jj = j - gate * H;
        t.zero();
        t.mac(WxT + j, G, xs + p, LP, n_in);
        if (gate < 2) t.mac(UhT + j, G, hs + p, LP, H);
#pragma unroll
        for (int a = 0; a < JT; ++a)
#pragma unroll
            for (int b = 0; b < PT; ++b) {
                const int o = (jj + a) * LP + p + b;
                if (gate == 0) zs[o] = sigm(t.a[a][b]);
                else if (gate == 1) rh[o] = sigm(t.a[a][b]) * hs[o];
                else gh[o] = t.a[a][b];
            }
    }
    __syncthreads();
    // candidate and state update
    for (int e = threadIdx.x; e < H / JT * PG; e += THREADS) {
        const int jg = e % (H / JT), pg = e / (H / JT), j = jg * JT, p = pg * PT;
#pragma unroll
        for (int a = 0; a < JT; ++a)
#pragma unroll
            for (int b = 0; b < PT; ++b) t.a[a][b] = gh[(j + a) * LP + p + b];
        t.mac(UhT + 2 * H + j, G, rh + p, LP, H);
#pragma unroll
        for (int a = 0; a < JT; ++a)
#pragma unroll
            for (int b = 0; b < PT; ++b) {
                const int o = (j + a) * LP + p + b;
                const T z = zs[o];
                gh[o] = z * hs[o] + (T(1) - z) * tanh_(t.a[a][b]);
            }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < np * H; i += THREADS) {
        const int p = i / H, k = i - p * H;
        h[(size_t)(p0 + p) * H + k] = gh[k * LP + p];
    }
    // output layer d = W_fc h' (rows of WfcT ldo long, zero past n_out)
    for (int e = threadIdx.x; e < ldo / JT * PG; e += THREADS) {
        const int og = e % (ldo / JT), pg = e / (ldo / JT), o = og * JT, p = pg * PT;
        t.zero();
        t.mac(WfcT + o, ldo, gh + p, LP, H);
#pragma unroll
        for (int b = 0; b < PT; ++b)
#pragma unroll
            for (int a = 0; a < JT; ++a)
                if (p + b < np && o + a < n_out) d[(size_t)(p0 + p + b) * n_out + o + a] = t.a[a][b];
    }
}

template <typename T, int TP, int JT, int PT, int THREADS>
cudaError_t run_rt(const Net &n, const void *X, void *h, void *d, int P, cudaStream_t st) {
    constexpr int LP = TP + (TP > 4 ? 16 / (int)sizeof(T) : 0);
    const size_t sm = sizeof(T) * (size_t)LP * (n.n_in + 4 * n.H);
    auto k = k_gru_rt<T, TP, JT, PT, THREADS>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<(P + TP - 1) / TP, THREADS, sm, st>>>(n.n_in, n.ldx, n.H, n.n_out, n.ldo, (const T *)X, (const T *)n.WxT,
                                              (const T *)n.UhT, (const T *)n.WfcTp, (T *)h, (T *)d, P);
    return cudaGetLastError();
}

template <typename T, typename TW, int TP>
cudaError_t run(const Net &n, const void *X, void *h, void *d, int P, cudaStream_t st) {
    using A = typename Acc<TW>::type;
    const size_t sm = sizeof(A) * ((size_t)TP * n.ldx + 6 * (size_t)TP * n.H);
    auto k = k_gru<T, TW, TP>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k<<<(P + TP - 1) / TP, NT, sm, st>>>(n.n_in, n.ldx, n.H, n.n_out, (const TW *)X,
                                         (const TW *)n.WxT, (const TW *)n.UhT, (const TW *)n.WfcT,
                                         (T *)h, (T *)d, P);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gru_cuda_core(const Net &n, const void *X, void *h, void *d, int P,
                                 cudaStream_t st) {
    if (P == 0) return cudaSuccess;
    // the register-tiled kernel where its staged values fit a quarter of an SM's
    // shared memory (several CTAs an SM cover the staging); else one column a thread
    if (n.WfcTp && n.H % 4 == 0 && n.n_in + 4 * n.H <= 512) {
        if (n.precision == DNNMG_F32) return run_rt<float, 32, 4, 8, 192>(n, X, h, d, P, st);
        if (n.precision == DNNMG_F64) return run_rt<double, 2, 2, 1, 128>(n, X, h, d, P, st);
    }
    if (n.precision == DNNMG_F64) return run<double, double, 8>(n, X, h, d, P, st);
    if (n.precision == DNNMG_F32) return run<float, float, 16>(n, X, h, d, P, st);
    return run<float, __nv_bfloat16, 16>(n, X, h, d, P, st);
}

}  // namespace dnnmg

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
#include <algorithm>

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
// this 57 us; bound by latency (the weights' way from L2, staging).  FP64 runs at two FMA a clock and SM, so
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
    template <bool SW> __device__ __forceinline__ void mac(const T *W, int ldw, const T *x, int ldp, int n);
};
// a weight vector from shared memory (SW) or, through the read-only path, from global
template <bool SW, typename V, typename T> __device__ __forceinline__ V load_w(const T *p) {
    if constexpr (SW) return *reinterpret_cast<const V *>(p);
    else return __ldg(reinterpret_cast<const V *>(p));
}
// PT patches (4 or 8) of 4 columns, patch pairs packed
template <bool SW, int PT>
__device__ __forceinline__ void mac_f32(float (&a)[4][PT], const float *W, int ldw, const float *x, int ldp, int n) {
    unsigned long long c[4][PT / 2];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int p = 0; p < PT / 2; ++p) asm("mov.b64 %0, {%1, %2};" : "=l"(c[j][p]) : "f"(a[j][2 * p]), "f"(a[j][2 * p + 1]));
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const float4 w = load_w<SW, float4>(W + (size_t)k * ldw);
        unsigned long long xv[PT / 2];
#pragma unroll
        for (int p = 0; p < PT / 2; p += 2) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(x + k * ldp + 2 * p);
            xv[p] = t.x;
            xv[p + 1] = t.y;
        }
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            unsigned long long ww;
            asm("mov.b64 %0, {%1, %1};" : "=l"(ww) : "f"(wv[j]));
#pragma unroll
            for (int p = 0; p < PT / 2; ++p) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c[j][p]) : "l"(ww), "l"(xv[p]));
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int p = 0; p < PT / 2; ++p) asm("mov.b64 {%0, %1}, %2;" : "=f"(a[j][2 * p]), "=f"(a[j][2 * p + 1]) : "l"(c[j][p]));
}
template <> template <bool SW>
__device__ __forceinline__ void RTile<float, 4, 8>::mac(const float *W, int ldw, const float *x, int ldp, int n) {
    mac_f32<SW, 8>(a, W, ldw, x, ldp, n);
}
template <> template <bool SW>
__device__ __forceinline__ void RTile<float, 4, 4>::mac(const float *W, int ldw, const float *x, int ldp, int n) {
    mac_f32<SW, 4>(a, W, ldw, x, ldp, n);
}
template <> template <bool SW>
__device__ __forceinline__ void RTile<double, 2, 1>::mac(const double *W, int ldw, const double *x, int ldp, int n) {
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
        const double2 w = load_w<SW, double2>(W + (size_t)k * ldw);
        const double xv = x[k * ldp];
        a[0][0] = fma(w.x, xv, a[0][0]);
        a[1][0] = fma(w.y, xv, a[1][0]);
    }
}

template <typename T, int TP, int JT, int PT, int THREADS, bool SW>
__global__ void __launch_bounds__(THREADS)
k_gru_rt(int n_in, int ldx, int H, int n_out, int ldo, const T *X, const T *WxT, const T *UhT, const T *WfcT, T *__restrict__ h, T *__restrict__ d, int P) {
    static_assert(TP % PT == 0, "whole tiles");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int LP = TP + (TP > 4 ? 16 / (int)sizeof(T) : 0);   // staged row length (padded against bank conflicts)
    T *xs = reinterpret_cast<T *>(smem_raw);   // [n_in][LP] features
    T *hs = xs + n_in * LP;                    // [H][LP] previous state
    T *zs = hs + H * LP;                       // [H][LP] update gate
    T *rh = zs + H * LP;                       // [H][LP] r * h
    T *gh = rh + H * LP;                       // [H][LP] W_h x, then the new state
    const int G = 3 * H;
    if constexpr (SW) {
        // the weights stay in shared memory for all of this CTA's patches (sizes are whole 16-byte pieces)
        T *ws = gh + H * LP;
        const T *src[3] = {WxT, UhT, WfcT};
        const int cnt[3] = {n_in * G, H * G, H * ldo};
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            constexpr int EPC = 16 / sizeof(T);
            for (int i = threadIdx.x * EPC; i < cnt[m]; i += THREADS * EPC)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(ws + i)),
                             "l"(src[m] + i)
                             : "memory");
            if (m == 0) WxT = ws;
            else if (m == 1) UhT = ws;
            else WfcT = ws;
            ws += cnt[m];
        }
    }
    pdl_wait();   // (the weights do not change: staged above before the other kernel has completed)
    // (the grid has a CTA for every tile; as straight code FP32 came out 1.3 times slower)
    for (long long q0 = (long long)blockIdx.x * TP; q0 < P; q0 += (long long)gridDim.x * TP) {
        const int p0 = (int)q0, np = min(TP, P - p0);
        for (int i = threadIdx.x; i < TP * n_in; i += THREADS) {
            const int p = i / n_in, k = i - p * n_in;
            xs[k * LP + p] = p < np ? X[(size_t)(p0 + p) * ldx + k] : T(0);
        }
        for (int i = threadIdx.x; i < TP * H; i += THREADS) {
            const int p = i / H, k = i - p * H;
            hs[k * LP + p] = p < np ? h[(size_t)(p0 + p) * H + k] : T(0);
        }
        if constexpr (SW) asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        constexpr int PG = TP / PT;
        RTile<T, JT, PT> t;
        // the two short products have a third of the columns: half the patches a tile
        constexpr int PT2 = PT > 4 ? PT / 2 : PT, PG2 = TP / PT2;
        RTile<T, JT, PT2> t2;
        // z, r and W_h x: a tile lies in one gate (H is a multiple of JT)
        for (int e = threadIdx.x; e < G / JT * PG; e += THREADS) {
            const int jg = e % (G / JT), pg = e / (G / JT), j = jg * JT, p = pg * PT, gate = j / H, jj = j - gate * H;
            t.zero();
            t.template mac<SW>(WxT + j, G, xs + p, LP, n_in);
            if (gate < 2) t.template mac<SW>(UhT + j, G, hs + p, LP, H);
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
        for (int e = threadIdx.x; e < H / JT * PG2; e += THREADS) {
            const int jg = e % (H / JT), pg = e / (H / JT), j = jg * JT, p = pg * PT2;
#pragma unroll
            for (int a = 0; a < JT; ++a)
#pragma unroll
                for (int b = 0; b < PT2; ++b) t2.a[a][b] = gh[(j + a) * LP + p + b];
            t2.template mac<SW>(UhT + 2 * H + j, G, rh + p, LP, H);
#pragma unroll
            for (int a = 0; a < JT; ++a)
#pragma unroll
                for (int b = 0; b < PT2; ++b) {
                    const int o = (j + a) * LP + p + b;
                    const T z = zs[o];
                    gh[o] = z * hs[o] + (T(1) - z) * tanh_(t2.a[a][b]);
                }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < np * H; i += THREADS) {
            const int p = i / H, k = i - p * H;
            h[(size_t)(p0 + p) * H + k] = gh[k * LP + p];
        }
        // output layer d = W_fc h' (rows of WfcT ldo long, zero past n_out)
        for (int e = threadIdx.x; e < ldo / JT * PG2; e += THREADS) {
            const int og = e % (ldo / JT), pg = e / (ldo / JT), o = og * JT, p = pg * PT2;
            t2.zero();
            t2.template mac<SW>(WfcT + o, ldo, gh + p, LP, H);
#pragma unroll
            for (int b = 0; b < PT2; ++b)
#pragma unroll
                for (int a = 0; a < JT; ++a)
                    if (p + b < np && o + a < n_out) d[(size_t)(p0 + p + b) * n_out + o + a] = t2.a[a][b];
        }
        __syncthreads();   // the staged values are free for the next patches
    }
}

size_t weight_count(const Net &n) { return (size_t)3 * n.H * (n.n_in + n.H) + (size_t)n.H * n.ldo; }
// bytes of the weights and the staged values of TP patches (row length LP)
size_t rt_bytes(const Net &n, int LP, size_t elem) {
    return elem * ((size_t)LP * (n.n_in + 4 * n.H) + weight_count(n));
}

template <typename T, int TP, int JT, int PT, int THREADS, bool SW>
cudaError_t run_rt(const Net &n, const void *X, void *h, void *d, int P, cudaStream_t st, bool chained) {
    constexpr int LP = TP + (TP > 4 ? 16 / (int)sizeof(T) : 0);
    const size_t sm = sizeof(T) * ((size_t)LP * (n.n_in + 4 * n.H) + (SW ? weight_count(n) : 0));
    auto k = k_gru_rt<T, TP, JT, PT, THREADS, SW>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const int grid = (P + TP - 1) / TP;
    if constexpr (SW && sizeof(T) == 8) {
        // FP64 keeps the weights in shared memory while every CTA has one tile; beyond that
        // the few CTAs an SM that fit beside them fall behind those that read them from L2
        // (99 -> 32 -> 50: 300 patches 30 against 44 us, 700 patches 73 against 48,
        // 16 336 patches 1209 against 553)
        int per = 1;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, THREADS, sm)) != cudaSuccess) return e;
        if (grid > std::max(1, per) * sm_count())
            return run_rt<T, TP, JT, PT, THREADS, false>(n, X, h, d, P, st, chained);
    }
    return launch_chained(chained, k, dim3(grid), THREADS, sm, st, n.n_in, n.ldx, n.H, n.n_out, n.ldo, (const T *)X,
                          (const T *)n.WxT, (const T *)n.UhT, (const T *)n.WfcTp, (T *)h, (T *)d, P);
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
                                 cudaStream_t st, bool chained) {
    if (P == 0) return cudaSuccess;
    // the register-tiled kernel, its weights in shared memory where they fit; else
    // one column a thread
    if (n.WfcTp && n.H % 4 == 0 && n.n_in + 4 * n.H <= 512) {
        constexpr size_t lim = 225 * 1024;
        if (n.precision == DNNMG_F32) {
            // one tile or less an SM: weights staged once, narrow tiles on twice the warps
            // (99 -> 64 -> 50: 4000 patches 25 against 35 us); more tiles: several CTAs an SM
            // read them from L2 (16 336 patches 58 against 78 us)
            if ((P + 31) / 32 <= sm_count() && rt_bytes(n, 36, 4) <= lim)
                return run_rt<float, 32, 4, 4, 384, true>(n, X, h, d, P, st, chained);
            return run_rt<float, 32, 4, 8, 192, false>(n, X, h, d, P, st, chained);
        }
        if (n.precision == DNNMG_F64) {
            if (rt_bytes(n, 2, 8) <= lim) return run_rt<double, 2, 2, 1, 128, true>(n, X, h, d, P, st, chained);
            return run_rt<double, 2, 2, 1, 128, false>(n, X, h, d, P, st, chained);
        }
    }
    if (n.precision == DNNMG_F64) return run<double, double, 8>(n, X, h, d, P, st);
    if (n.precision == DNNMG_F32) return run<float, float, 16>(n, X, h, d, P, st);
    return run<float, __nv_bfloat16, 16>(n, X, h, d, P, st);
}

}  // namespace dnnmg

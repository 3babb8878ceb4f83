// Device helpers of the training-window kernels (gru_win.cu: BF16 products,
// gru_win32.cu: FP32 products): operand images in shared memory, tcgen05
// products between them, tensor memory, and the CTA's start, hand-overs and
// end.  Included by those two files only.
#pragma once

#include "common.cuh"
#include "gru_win.cuh"
#include "ptx.cuh"

namespace dnnmg {
namespace {

using namespace ptx;

constexpr int TM = 128;            // rows of a tile
constexpr int IMG = TM * 128;      // one operand image: 128 rows of 64 BF16 columns, 128-byte swizzle

__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// K-major operand: rows of 64 K elements, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t desc_k(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 |
           (uint64_t)2 << 61;
}
// The same image as an MN-major operand: its 64 columns are the M (or N)
// extent, its rows the K extent; the next 64 columns are `next` bytes on.
__device__ __forceinline__ uint64_t desc_mn(uint32_t saddr, uint32_t next) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | (uint64_t)((next >> 4) & 0x3FFF) << 16 | (uint64_t)(1024 >> 4) << 32 |
           (uint64_t)1 << 46 | (uint64_t)2 << 61;
}
// kind::f16, BF16 A and B, FP32 D; mn: both operands MN-major
__host__ __device__ constexpr uint32_t idesc(int N, bool mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(TM >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
}
// D (+)= A B^T over ksteps x 16 columns of two K-major images
__device__ __forceinline__ void mma_k(uint32_t d, uint32_t a, uint32_t b, int N, int ksteps, bool acc) {
    const uint64_t da = desc_k(a), db = desc_k(b);
    for (int k = 0; k < ksteps; ++k) umma(d, da + 2 * k, db + 2 * k, idesc(N, false), (acc || k > 0) ? 1u : 0u);
}
// D (+)= A^T B over the 128 rows of the images
__device__ __forceinline__ void mma_mn(uint32_t d, uint64_t a, uint64_t b, int N, bool acc) {
#pragma unroll
    for (int k = 0; k < TM / 16; ++k)
        umma(d, a + k * (2048 >> 4), b + k * (2048 >> 4), idesc(N, true), (acc || k > 0) ? 1u : 0u);
}
__device__ __forceinline__ void tmem_ld8(uint32_t t, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(t));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st8(uint32_t t, const float (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(t), "f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// values read by tmem_ld8 may be used from here on
__device__ __forceinline__ void keep(float (&v)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) asm volatile("" : "+f"(v[i]));
}

__device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&t);
}
// byte offset of 16-byte unit u of row `row` in an image
__device__ __forceinline__ uint32_t swz(int row, int u) { return (uint32_t)(row * 128 + ((u ^ (row & 7)) << 4)); }
// 8 consecutive columns c .. c+7 (c a multiple of 8) of a row
__device__ __forceinline__ void put8(uint8_t *img, int row, int c, const float *v) {
    *reinterpret_cast<uint4 *>(img + swz(row, c / 8)) =
        make_uint4(pack(v[0], v[1]), pack(v[2], v[3]), pack(v[4], v[5]), pack(v[6], v[7]));
}
__device__ __forceinline__ void put1(uint8_t *img, int row, int c, float v) {
    *reinterpret_cast<__nv_bfloat16 *>(img + swz(row, c / 8) + (c & 7) * 2) = __float2bfloat16_rn(v);
}
// image rows [0, rows) x columns [0, 64) of src(row, col)
template <typename F> __device__ __forceinline__ void build(uint8_t *img, int rows, int nth, F src) {
    for (int e = threadIdx.x; e < rows * 8; e += nth) {
        const int r = e >> 3, c = (e & 7) * 8;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = src(r, c + i);
        *reinterpret_cast<uint4 *>(img + (r >> 3) * 1024 + (r & 7) * 128 + (((c >> 3) ^ (r & 7)) << 4)) =
            make_uint4(pack(v[0], v[1]), pack(v[2], v[3]), pack(v[4], v[5]), pack(v[6], v[7]));
    }
}

__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }

__device__ __forceinline__ void ld4(const float *p, float *v) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void st4(float *p, const float *v) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
// saved activations: element (column c, row) of a tile's block
__device__ __forceinline__ size_t blk(int c, int row) { return (size_t)(c >> 2) * (4 * TM) + 4 * row; }

__device__ __forceinline__ void prefetch_l2(const float *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// 64 columns, from x0 on, of a tile's feature rows, coalesced: 16 lanes take one row's.
template <int NTH> struct XTile {
    static constexpr int NV = TM * 16 / NTH;
    float4 v[NV];
    __device__ __forceinline__ void load(const WinArgs &g, int s, int p0, int x0 = 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = threadIdx.x + i * NTH, row = e >> 4, c = x0 + (e & 15) * 4;
            v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p0 + row >= g.P || c >= g.n_in) continue;
            const float *src = g.X + ((size_t)s * g.P + p0 + row) * g.ldx + c;
            if (g.xvec) {
                v[i] = __ldg(reinterpret_cast<const float4 *>(src));
            } else {   // rows that do not start on 16 bytes
                v[i].x = __ldg(src);
                if (c + 1 < g.n_in) v[i].y = __ldg(src + 1);
                if (c + 2 < g.n_in) v[i].z = __ldg(src + 2);
                if (c + 3 < g.n_in) v[i].w = __ldg(src + 3);
            }
        }
    }
    __device__ __forceinline__ void prefetch(const WinArgs &g, int s, int p0, int x0) const {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = threadIdx.x + i * NTH, row = e >> 4, c = x0 + (e & 15) * 4;
            if (p0 + row < g.P && c < g.n_in) prefetch_l2(g.X + ((size_t)s * g.P + p0 + row) * g.ldx + c);
        }
    }
    __device__ __forceinline__ void store(const WinArgs &g, uint8_t *img, int x0 = 0) const {
        const int n = g.n_in - x0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = threadIdx.x + i * NTH, row = e >> 4, c = (e & 15) * 4;
            const float a = v[i].x, b = c + 1 < n ? v[i].y : 0.f, d = c + 2 < n ? v[i].z : 0.f,
                        f = c + 3 < n ? v[i].w : 0.f;   // (columns past n_in are not read as features)
            *reinterpret_cast<uint2 *>(img + swz(row, c >> 3) + (c & 4) * 2) = make_uint2(pack(a, b), pack(d, f));
        }
    }
};

// Shared start and end of both kernels: barriers, tensor memory, teardown.
struct Cta {
    uint32_t bar0, tmem;
    volatile int *abort_flag;
    __device__ __forceinline__ void init(uint64_t *bars, int nbar, int cols) {
        uint32_t *slot = reinterpret_cast<uint32_t *>(bars + nbar);
        abort_flag = reinterpret_cast<volatile int *>(slot + 1);
        bar0 = smem_u32(bars);
        if (threadIdx.x == 0) {
            for (int i = 0; i < nbar; ++i) mbar_init(bar0 + 8 * i, 1);
            abort_flag[0] = abort_flag[1] = 0;
            mbar_init_fence();
        }
        if (threadIdx.x < 32) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        fence_async_smem();
        tc_before_sync();
        __syncthreads();
        tc_after_sync();
        tmem = *slot;
    }
    // images written before are visible to the MMAs issued after, and tensor
    // memory read before may be overwritten; false once a wait has run out
    __device__ __forceinline__ bool hand_over(bool ok) {
        fence_async_smem();
        tc_before_sync();
        const bool bad = __syncthreads_or(!ok);
        tc_after_sync();
        return !bad;
    }
    // a value that is not finite has been seen (read by all threads after a hand-over, and set back by one)
    __device__ __forceinline__ void mark() { abort_flag[1] = 1; }
    __device__ __forceinline__ bool marked() const { return abort_flag[1]; }
    __device__ __forceinline__ void unmark() {
        __syncthreads();
        if (threadIdx.x == 0) abort_flag[1] = 0;
    }
    __device__ __forceinline__ bool wait(int b, uint32_t parity) {
        const bool ok = mbar_wait_inl(bar0 + 8 * b, parity, abort_flag);
        __syncwarp();
        tc_after_sync();
        return ok;
    }
    __device__ __forceinline__ void finish(int drain_bar, int cols, int *status) {
        if (threadIdx.x == 0) {
            if (*abort_flag) {
                atomicOr(status, DNNMG_DEVERR_TIMEOUT);
                volatile int no_abort = 0;
                tc_commit(bar0 + 8 * drain_bar);   // every MMA issued has finished before teardown
                mbar_wait(bar0 + 8 * drain_bar, 0, &no_abort);
            }
        }
        tc_before_sync();
        __syncthreads();
        if (threadIdx.x < 32) {
            tc_after_sync();
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
        }
    }
};

__device__ __forceinline__ uint8_t *align1k(uint8_t *p) { return p + ((1024u - (smem_u32(p) & 1023u)) & 1023u); }

template <typename K> cudaError_t launch(K k, int grid, int threads, int smem, const WinArgs &g, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k<<<grid, threads, smem, st>>>(g);
    return cudaGetLastError();
}

}  // namespace
}  // namespace dnnmg

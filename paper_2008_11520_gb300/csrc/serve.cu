// Batched correction steps of many flow instances (serving).
//
// The correction step of Algorithm 2 is per instance; its network (Eq. gru + output
// layer) works patch by patch with weights shared by every instance that uses
// the same net.  A server therefore runs one step of several instances as:
//   S1, S2+S3, S5, S6, S7   one launch each over the tiles of all instances,
//                           from and into each instance's own arrays,
//   S4                      one tensor-core GRU launch over all rows of X.
// Each instance's GRU state h lives in a segment of one state pool.  Segments
// and batch rows are whole 128-row tiles, so every GRU tile belongs to one
// instance; a per-tile table gives the tile's first state row in the pool.
// A patch row's arithmetic does not depend on the other rows of its tile, and
// a stencil tile runs the code of the single-instance launch, so an instance
// gets the same bits alone (dnnmg_step) and in any batch.
//
// Launching the passes instance by instance on eight streams was bound by the
// host (six launches and their tensor maps an instance): 20 instances of
// 64 x 16 .. 512 x 128 coarse cells, K = 1, took 390 us a step; now 235 us.
// Eight of 256 x 64 .. 512 x 128, K = 2: back to back 318 and 326 us, waited for 387
// and 360.
#include <algorithm>
#include <cstring>
#include <map>
#include <new>
#include <vector>

#include "common.cuh"

namespace dnnmg {
namespace {

constexpr int kTileRows = 128;   // rows of one GRU tile
constexpr int kGroup = 8;        // v_corr scratch: this many times the largest admitted mesh's

// First-fit allocator of row ranges in units of `unit` rows; frees coalesce.
struct RowPool {
    int capacity = 0, unit = 1;
    std::map<int, int> free_;   // start -> length, disjoint, never adjacent
    std::map<int, int> used_;   // start -> length

    void init(int cap, int u) {
        unit = u;
        capacity = cap / u * u;
        free_.clear();
        used_.clear();
        if (capacity > 0) free_[0] = capacity;
    }
    int rounded(int rows) const { return (rows + unit - 1) / unit * unit; }
    // start of a free range of rounded(rows) rows, or -1
    int alloc(int rows) {
        const int n = rounded(rows);
        if (n <= 0) return -1;
        for (auto it = free_.begin(); it != free_.end(); ++it) {
            if (it->second < n) continue;
            const int start = it->first, len = it->second;
            free_.erase(it);
            if (len > n) free_[start + n] = len - n;
            used_[start] = n;
            return start;
        }
        return -1;
    }
    bool release(int start) {
        auto u = used_.find(start);
        if (u == used_.end()) return false;
        int s = start, len = u->second;
        used_.erase(u);
        auto next = free_.lower_bound(s);
        if (next != free_.end() && next->first == s + len) {
            len += next->second;
            next = free_.erase(next);
        }
        if (next != free_.begin()) {
            auto prev = std::prev(next);
            if (prev->first + prev->second == s) {
                s = prev->first;
                len += prev->second;
                free_.erase(prev);
            }
        }
        free_[s] = len;
        return true;
    }
    int used_rows() const {
        int n = 0;
        for (auto &kv : used_) n += kv.second;
        return n;
    }
    int largest_free() const {
        int m = 0;
        for (auto &kv : free_) m = std::max(m, kv.second);
        return m;
    }
};

}  // namespace
}  // namespace dnnmg

struct dnnmg_pool_s {
    dnnmg::RowPool pool;
};

struct dnnmg_server_s {
    dnnmg_net_t net = nullptr;
    int device = -1;
    int cap_rows = 0;
    dnnmg::RowPool pool;
    float *hpool = nullptr;   // [cap_rows][H]
    void *X = nullptr;        // [cap_rows][ldx] bf16
    float *d = nullptr;       // [cap_rows][n_out]
    int *tiles_dev = nullptr; // [cap_rows / 128], per tile of the batch: its first state row in the pool
    cudaStream_t side = nullptr;               // the boundary tiles, beside the closed form
    cudaEvent_t fork = nullptr, join = nullptr;
    cudaEvent_t done = nullptr;                // end of the last step: the next may run on another stream
    char *vc = nullptr;                        // v_corr of the instances whose S5 to S7 run together
    size_t vc_bytes = 0, vc_max = 0;           // vc_bytes = kGroup x the largest admitted mesh's (vc_max)
    struct Slot {
        dnnmg_mesh_t mesh;
        int start, rows;      // pool segment (multiple of 128 rows); rows = padded patch rows
        float *xcp;           // padded x_c
        bool live;
    };
    std::vector<Slot> slots;
};

namespace dnnmg {
namespace {

size_t vc_need(const dnnmg_mesh_info &I) { return align256(2 * (size_t)I.plane * I.real_bytes); }
size_t xcp_need(const dnnmg_mesh_info &I) {
    return 3 * (size_t)(I.nyc + 1) * round_up(I.nxc + 1, 32) * I.real_bytes;
}

void server_free(dnnmg_server_s *s) {
    if (!s) return;
    cudaFree(s->hpool);
    cudaFree(s->X);
    cudaFree(s->d);
    cudaFree(s->tiles_dev);
    cudaFree(s->vc);
    for (auto &sl : s->slots)
        if (sl.live) cudaFree(sl.xcp);
    if (s->side) cudaStreamDestroy(s->side);
    for (cudaEvent_t e : {s->fork, s->join, s->done})
        if (e) cudaEventDestroy(e);
    delete s;
}

int check_server(dnnmg_server_s *s) {
    if (!s) return fail(DNNMG_EINVAL, "server handle is NULL");
    int cur = -1;
    DNNMG_CUDA_TRY(cudaGetDevice(&cur));
    if (cur != s->device) return fail(DNNMG_EINVAL, "server belongs to device %d but device %d is current", s->device, cur);
    return DNNMG_OK;
}

int check_slot(dnnmg_server_s *s, int slot) {
    if (slot < 0 || slot >= (int)s->slots.size() || !s->slots[slot].live)
        return fail(DNNMG_EINVAL, "slot %d is not an admitted instance", slot);
    return DNNMG_OK;
}

}  // namespace
}  // namespace dnnmg

using namespace dnnmg;

extern "C" {

int dnnmg_pool_create(int capacity_rows, int unit, dnnmg_pool_t *out) {
    clear_error();
    if (!out) return fail(DNNMG_EINVAL, "out is NULL");
    if (capacity_rows < 0 || unit < 1) return fail(DNNMG_EINVAL, "capacity %d / unit %d", capacity_rows, unit);
    dnnmg_pool_s *p = new (std::nothrow) dnnmg_pool_s();
    if (!p) return fail(DNNMG_ENOMEM, "host allocation failed");
    p->pool.init(capacity_rows, unit);
    *out = p;
    return DNNMG_OK;
}

int dnnmg_pool_alloc(dnnmg_pool_t pool, int rows, int *start) {
    clear_error();
    if (!pool || !start) return fail(DNNMG_EINVAL, "NULL argument");
    if (rows < 1) return fail(DNNMG_EINVAL, "rows = %d", rows);
    const int s = pool->pool.alloc(rows);
    if (s < 0) return fail(DNNMG_ENOMEM, "no free range of %d rows", pool->pool.rounded(rows));
    *start = s;
    return DNNMG_OK;
}

int dnnmg_pool_free(dnnmg_pool_t pool, int start) {
    clear_error();
    if (!pool) return fail(DNNMG_EINVAL, "pool is NULL");
    if (!pool->pool.release(start)) return fail(DNNMG_EINVAL, "no range starts at row %d", start);
    return DNNMG_OK;
}

int dnnmg_pool_stats(dnnmg_pool_t pool, int *used_rows, int *largest_free) {
    clear_error();
    if (!pool) return fail(DNNMG_EINVAL, "pool is NULL");
    if (used_rows) *used_rows = pool->pool.used_rows();
    if (largest_free) *largest_free = pool->pool.largest_free();
    return DNNMG_OK;
}

void dnnmg_pool_destroy(dnnmg_pool_t pool) { delete pool; }

size_t dnnmg_server_bytes(dnnmg_net_t net, int max_rows) {
    if (!net || max_rows < 0) return 0;
    const size_t rows = (size_t)(max_rows + kTileRows - 1) / kTileRows * kTileRows;
    return align256(rows * net->H * sizeof(float)) + align256(rows * net->ldx * 2) +
           align256(rows * net->n_out * sizeof(float)) + align256(rows / kTileRows * sizeof(int));
}

int dnnmg_server_create(dnnmg_net_t net, int max_rows, dnnmg_server_t *out) {
    clear_error();
    if (!out) return fail(DNNMG_EINVAL, "out is NULL");
    *out = nullptr;
    if (!net) return fail(DNNMG_EINVAL, "net handle is NULL");
    if (!net->tc)
        return fail(DNNMG_EUNSUPPORTED, "batched steps need a tensor-core (DNNMG_BF16NET, H <= 128) network");
    if (max_rows < 1) return fail(DNNMG_EINVAL, "max_rows = %d", max_rows);
    int dev = -1;
    DNNMG_CUDA_TRY(cudaGetDevice(&dev));
    if (dev != net->device) return fail(DNNMG_EINVAL, "net belongs to device %d but device %d is current", net->device, dev);
    dnnmg_server_s *s = new (std::nothrow) dnnmg_server_s();
    if (!s) return fail(DNNMG_ENOMEM, "host allocation failed");
    s->net = net;
    s->device = dev;
    s->cap_rows = (max_rows + kTileRows - 1) / kTileRows * kTileRows;
    s->pool.init(s->cap_rows, kTileRows);
    const size_t rows = (size_t)s->cap_rows, ntiles = rows / kTileRows;
    bool ok = cudaMalloc(&s->hpool, rows * net->H * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&s->X, rows * net->ldx * 2) == cudaSuccess &&
              cudaMalloc(&s->d, rows * net->n_out * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&s->tiles_dev, ntiles * sizeof(int)) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking) == cudaSuccess;
    for (cudaEvent_t *e : {&s->fork, &s->join, &s->done})
        ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    // feature rows past an instance's patches are read by its last GRU tile:
    // keep them finite (their results land only in the instance's padding)
    ok = ok && cudaMemset(s->X, 0, rows * net->ldx * 2) == cudaSuccess;
    if (!ok) {
        server_free(s);
        cudaGetLastError();
        return fail(DNNMG_ENOMEM, "device allocation of the server's %zu bytes failed", dnnmg_server_bytes(net, max_rows));
    }
    *out = s;
    return DNNMG_OK;
}

int dnnmg_server_destroy(dnnmg_server_t server) {
    clear_error();
    if (!server) return DNNMG_OK;
    cudaDeviceSynchronize();
    server_free(server);
    return DNNMG_OK;
}

int dnnmg_server_admit(dnnmg_server_t s, dnnmg_mesh_t mesh, int *slot) {
    clear_error();
    if (int e = check_server(s)) return e;
    if (!mesh || !slot) return fail(DNNMG_EINVAL, "NULL argument");
    if (mesh->device != s->device) return fail(DNNMG_EINVAL, "mesh and server are on different devices");
    const dnnmg_mesh_info &I = mesh->info;
    const Net &n = *s->net;
    if (I.precision != DNNMG_BF16NET) return fail(DNNMG_EINVAL, "mesh precision must be DNNMG_BF16NET");
    if (I.n_in != n.n_in || I.ldx != n.ldx || I.n_out != n.n_out)
        return fail(DNNMG_EINVAL, "mesh has n_in %d / n_out %d, the net %d / %d", I.n_in, I.n_out, n.n_in, n.n_out);
    const int rows = (I.P + kTileRows - 1) / kTileRows * kTileRows;
    int start = 0;
    if (rows > 0) {
        start = s->pool.alloc(rows);
        if (start < 0)
            return fail(DNNMG_ENOMEM, "no free state segment of %d rows (largest %d of %d)", rows,
                        s->pool.largest_free(), s->cap_rows);
    }
    float *xcp = nullptr;
    char *vc = nullptr;
    const size_t need = vc_need(I);
    cudaError_t e = cudaMalloc(&xcp, xcp_need(I));
    if (e == cudaSuccess && need > s->vc_max) {
        // the scratch may be in use by steps in flight
        e = cudaDeviceSynchronize();
        if (e == cudaSuccess) e = cudaMalloc(&vc, kGroup * need);
    }
    if (e != cudaSuccess) {
        cudaFree(xcp);
        if (rows > 0) s->pool.release(start);
        cudaGetLastError();
        return fail(DNNMG_ENOMEM, "scratch of %d x %zu bytes: %s", kGroup, need, cudaGetErrorString(e));
    }
    if (vc) {
        cudaFree(s->vc);
        s->vc = vc;
        s->vc_max = need;
        s->vc_bytes = kGroup * need;
    }
    // h0 = 0 (Sec. 6.2), padding rows included
    if (rows > 0 && cudaMemset(s->hpool + (size_t)start * n.H, 0, (size_t)rows * n.H * sizeof(float)) != cudaSuccess) {
        s->pool.release(start);
        cudaFree(xcp);
        cudaGetLastError();
        return fail(DNNMG_ECUDA, "clearing the state segment failed");
    }
    int id = -1;
    for (int i = 0; i < (int)s->slots.size(); ++i)
        if (!s->slots[i].live) {
            id = i;
            break;
        }
    if (id < 0) {
        id = (int)s->slots.size();
        s->slots.push_back({});
    }
    s->slots[id] = {mesh, start, rows, xcp, true};
    *slot = id;
    return DNNMG_OK;
}

int dnnmg_server_release(dnnmg_server_t s, int slot) {
    clear_error();
    if (int e = check_server(s)) return e;
    if (int e = check_slot(s, slot)) return e;
    // a step in flight may still read or write the segment
    DNNMG_CUDA_TRY(cudaDeviceSynchronize());
    if (s->slots[slot].rows > 0) s->pool.release(s->slots[slot].start);
    cudaFree(s->slots[slot].xcp);
    s->slots[slot].xcp = nullptr;
    s->slots[slot].live = false;
    s->slots[slot].mesh = nullptr;
    return DNNMG_OK;
}

int dnnmg_server_state(dnnmg_server_t s, int slot, float **h) {
    clear_error();
    if (!s) return fail(DNNMG_EINVAL, "server handle is NULL");
    if (int e = check_slot(s, slot)) return e;
    if (!h) return fail(DNNMG_EINVAL, "h is NULL");
    *h = s->hpool + (size_t)s->slots[slot].start * s->net->H;
    return DNNMG_OK;
}

int dnnmg_server_step(dnnmg_server_t s, int n, const int *slots, const double *const *xc, void *const *bf,
                      double *const *bc, const double *t, cudaStream_t stream) {
    clear_error();
    if (int e = check_server(s)) return e;
    if (n < 1 || !slots || !xc || !bf || !bc || !t) return fail(DNNMG_EINVAL, "empty batch or NULL argument");
    std::vector<int> row0(n);
    int total = 0;
    for (int i = 0; i < n; ++i) {
        if (int e = check_slot(s, slots[i])) return e;
        for (int j = 0; j < i; ++j)
            if (slots[j] == slots[i]) return fail(DNNMG_EINVAL, "slot %d appears twice in one batch", slots[i]);
        if (!xc[i] || !bf[i] || !bc[i]) return fail(DNNMG_EINVAL, "NULL array of instance %d", i);
        if (reinterpret_cast<uintptr_t>(bf[i]) % 16) return fail(DNNMG_EINVAL, "bf of instance %d is not 16-byte aligned", i);
        row0[i] = total;
        total += s->slots[slots[i]].rows;
    }
    // the server's buffers belong to one step at a time, on whichever stream
    // (a captured step can neither wait for one outside its graph nor mark its end)
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    DNNMG_CUDA_TRY(cudaStreamIsCapturing(stream, &capture));
    const bool eager = capture == cudaStreamCaptureStatusNone;
    if (eager) DNNMG_CUDA_TRY(cudaStreamWaitEvent(stream, s->done, 0));
    const Net &net = *s->net;
    uint16_t *X = static_cast<uint16_t *>(s->X);
    std::vector<StepInst> in(n);
    for (int i = 0; i < n; ++i) {
        const dnnmg_server_s::Slot &sl = s->slots[slots[i]];
        in[i] = {sl.mesh, xc[i], t[i], static_cast<float *>(bf[i]), bc[i], X + (size_t)row0[i] * net.ldx,
                 s->d + (size_t)row0[i] * net.n_out, sl.xcp, nullptr, row0[i] / kTileRows, sl.rows / kTileRows, sl.start};
    }
    // S1 + S2 + S3, each instance into its rows of X: one launch per pass over
    // up to kBatch instances, the boundary tiles on the side stream
    const bool cf = residual_cf_supported(in[0].mesh->g, in[0].mesh->info.precision);
    for (int i = 0; i < n; i += kBatch) {
        const int m = std::min(kBatch, n - i);
        DNNMG_CUDA_TRY(launch_coarse_pad_batch(&in[i], m, s->tiles_dev, stream));
        if (cf) {
            DNNMG_CUDA_TRY(cudaEventRecord(s->fork, stream));
            DNNMG_CUDA_TRY(cudaStreamWaitEvent(s->side, s->fork, 0));
            // (in dnnmg_step's order: one request of 256 x 64 coarse cells, K = 2, waited for, 96 -> 78 us)
            const bool second = residual_step_batch_small(&in[i], m, true);
            if (second) DNNMG_CUDA_TRY(launch_residual_cf_batch(&in[i], m, stream));
            DNNMG_CUDA_TRY(launch_residual_step_batch(&in[i], m, true, s->side));
            if (!second) DNNMG_CUDA_TRY(launch_residual_cf_batch(&in[i], m, stream));
        } else {
            DNNMG_CUDA_TRY(launch_residual_step_batch(&in[i], m, false, stream));
        }
    }
    if (cf) {
        DNNMG_CUDA_TRY(cudaEventRecord(s->join, s->side));
        DNNMG_CUDA_TRY(cudaStreamWaitEvent(stream, s->join, 0));
    }
    // S4 once over every instance's rows
    if (total > 0)
        DNNMG_CUDA_TRY(launch_gru_tc_rows(net, s->X, s->hpool, s->d, total, s->tiles_dev, s->cap_rows, stream));
    // S5, S6, S7 from each instance's rows of d, over as many instances as the scratch holds v_corr of
    for (int i = 0; i < n;) {
        size_t used = 0;
        int m = 0;
        while (i + m < n && m < kBatch && used + vc_need(in[i + m].mesh->info) <= s->vc_bytes) {
            in[i + m].vc = reinterpret_cast<float *>(s->vc + used);
            used += vc_need(in[i + m].mesh->info);
            ++m;
        }
        DNNMG_CUDA_TRY(launch_scatter_avg_batch(&in[i], m, stream, total > 0 || i > 0));
        DNNMG_CUDA_TRY(launch_rhs_batch(&in[i], m, stream));
        DNNMG_CUDA_TRY(launch_restrict_batch(&in[i], m, stream));
        i += m;
    }
    if (eager) DNNMG_CUDA_TRY(cudaEventRecord(s->done, stream));
    return DNNMG_OK;
}

}  // extern "C"

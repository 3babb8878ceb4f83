// Plain geometric multigrid for the fine-level system on the GPU: the
// solver DNN-MG is compared with (Sec. 3.3 Newton iteration, Sec. 3.4
// multigrid with the Vanka smoother, Sec. 6.4 timing comparison).
//
// One time step of the plain method solves the Crank-Nicolson system of
// Eq. nonlinearshort on level L+K by Newton's method; each Newton system is
// solved by GMRES preconditioned with multigrid V-cycles over a hierarchy of
// levels, smoothed by the Vanka method: for every cell, the 12 x 12 block of
// the Newton matrix that couples the velocity and pressure unknowns of its
// four nodes is solved against the current defect.  This file holds the
// level hierarchy and the kernels of one V-cycle and of the Newton and
// GMRES iterations; the iterations themselves are driven from the host
// (mg.py).  Node fields are [3][N] (u, v, p), N = (nx + 1)(ny + 1) nodes,
// x fastest, unpadded: the layout of the host solver.
//
// The discretisation is the one of the correction step (Q1/Q1, Crank-
// Nicolson, local projection stabilisation on 2 x 2-cell patches, 2 x 2
// Gauss points), with the element constants of FemCoef.  Level 0 is the
// finest, with any cell mask (a partly solid projection patch contributes
// the integrals of its fluid cells, as on the coarse level of the host
// solver); level l+1 has half the cells of level l in each direction, and a
// patch of level l+1 is solid iff all 16 cells of level l under it are.
// Every level uses the finest level's projection coefficient alpha (alpha0
// scaled by 4^-l): the fine projection term vanishes on a prolongated
// pressure, and alpha = alpha0 h^2 / nu evaluated with a coarse h would
// outweigh the pressure coupling of the time step there and make the coarse
// pressure corrections far too small.  (Coarse levels only precondition:
// their geometry and stabilisation approximate the fine ones.)
//
// The smoother is multiplicative (block Gauss-Seidel over cells) in 16
// colours.  A cell's local defect reads the correction up to two nodes beyond
// its own (the projection patches reach two nodes from an even node), and it
// writes its own four nodes; cells with the same (ci mod 4, cj mod 4) are
// four cells apart, so none reads a node another one writes: each colour is
// one parallel pass, and a sweep is deterministic.
#include <cmath>
#include <new>
#include <vector>

#include "common.cuh"

namespace dnnmg {

void level_coefficients(double lx, double ly, int nx, int ny, double nu, double k, double alpha0,
                        FemCoef<double> *f64, FemCoef<float> *f32);

namespace {

constexpr int MG_THREADS = 256;

// A level as the kernels see it.
template <typename T>
struct MgLev {
    int nx, ny, N;
    const uint8_t *solid;   // [ny][nx] cell mask, 1 = solid
    const uint8_t *flags;   // [N]: bit 0 velocity Dirichlet, bit 1 inflow value, bit 2 pressure active
    const uint8_t *mult;    // [N]: fluid cells holding the node
    const T *lps;           // [16][9][9]: projection patch matrix by the patch's fluid cells (bit 2 cb + ca)
    double hy, ly;
    FemCoef<T> fc;
};

template <typename T> __device__ __forceinline__ bool fluid(const MgLev<T> &L, int ci, int cj) {
    return ci >= 0 && cj >= 0 && ci < L.nx && cj < L.ny && !L.solid[(size_t)cj * L.nx + ci];
}
// The fluid cells of 2 x 2-cell projection patch (m, n): bit 2 cb + ca for its
// cell (2m + ca, 2n + cb); 0 outside the mesh.  A patch contributes the
// projection integrals of its fluid cells (every cell of an all-fluid patch).
template <typename T> __device__ __forceinline__ int patch_mask(const MgLev<T> &L, int m, int n) {
    if (m < 0 || n < 0 || 2 * m + 1 >= L.nx || 2 * n + 1 >= L.ny) return 0;
    return (fluid(L, 2 * m, 2 * n) ? 1 : 0) | (fluid(L, 2 * m + 1, 2 * n) ? 2 : 0) |
           (fluid(L, 2 * m, 2 * n + 1) ? 4 : 0) | (fluid(L, 2 * m + 1, 2 * n + 1) ? 8 : 0);
}

template <typename T> __device__ __forceinline__ T inflow(const MgLev<T> &L, int J, double up) {
    const double y = J * L.hy;
    return (T)(up * 4.0 * y * (L.ly - y) / (L.ly * L.ly));
}

// Rows of one node for the operator pieces the kernels share: with the node
// at corner a of fluid cell (ci, cj), add the cell's linear velocity and
// pressure-gradient terms (mode 0: A(x); mode 1: the right-hand side's
// 1/k M - nu/2 K part, no pressure) and the divergence.
template <typename T>
__device__ __forceinline__ void linear_rows(const MgLev<T> &L, const T *u, const T *v, const T *p, int ci, int cj,
                                            int a, bool rhs, T &Au, T &Av, T &Ap) {
    const int nxn = L.nx + 1;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int n = (cj + (b >> 1)) * nxn + ci + (b & 1);
        const T ub = u[n], vb = v[n];
        if (rhs) {
            Au += L.fc.Bv[a][b] * ub;
            Av += L.fc.Bv[a][b] * vb;
        } else {
            const T pb = p[n];
            Au += L.fc.Av[a][b] * ub - L.fc.Gx[a][b] * pb;
            Av += L.fc.Av[a][b] * vb - L.fc.Gy[a][b] * pb;
            Ap += L.fc.Dx[a][b] * ub + L.fc.Dy[a][b] * vb;
        }
    }
}

// Local projection term of pressure row (I, J): the patches that hold the node.
template <typename T> __device__ __forceinline__ T lps_row(const MgLev<T> &L, const T *p, int I, int J) {
    const int nxn = L.nx + 1;
    T acc = T(0);
#pragma unroll
    for (int pn = 0; pn < 2; ++pn) {
        const int n = (J - pn) >> 1;                      // patches n with 2n <= J <= 2n + 2
        if (pn == 1 && (J & 1)) continue;                  // an odd J lies in one patch only
        if (2 * n > J || J > 2 * n + 2) continue;
#pragma unroll
        for (int pm = 0; pm < 2; ++pm) {
            const int m = (I - pm) >> 1;
            if (pm == 1 && (I & 1)) continue;
            if (2 * m > I || I > 2 * m + 2) continue;
            const int pm_ = patch_mask(L, m, n);
            if (!pm_) continue;
            const int il = 3 * (J - 2 * n) + (I - 2 * m);
            const T *S = L.lps + (pm_ * 9 + il) * 9;
#pragma unroll
            for (int kb = 0; kb < 3; ++kb)
#pragma unroll
                for (int ka = 0; ka < 3; ++ka) acc += S[3 * kb + ka] * p[(2 * n + kb) * nxn + 2 * m + ka];
        }
    }
    return acc;
}

// Values of (u, v) at the 2 x 2 Gauss points (i along x, j along y) of a cell
// and their derivatives, in tensor form: a bilinear field's x-derivative
// depends on j only, its y-derivative on i only.
template <typename T>
struct CellVel {
    T U[2][2], V[2][2], Ux[2], Uy[2], Vx[2], Vy[2];   // [j][i], [j], [i]
    static __device__ __forceinline__ void field(const FemCoef<T> &fc, const T (&w)[4], T (&W)[2][2], T (&Wx)[2],
                                                 T (&Wy)[2]) {
        const T db = w[1] - w[0], dt = w[3] - w[2], dd = dt - db;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const T g = i ? fc.cg1 : fc.cg0;
            const T b = w[0] + g * db, t = w[2] + g * dt, e = t - b;
            W[0][i] = b + fc.cg0 * e;
            W[1][i] = b + fc.cg1 * e;
            Wy[i] = e * fc.inv_hy;
            Wx[i] = (db + g * dd) * fc.inv_hx;
        }
    }
    __device__ __forceinline__ void eval(const FemCoef<T> &fc, const T *u, const T *v, int n0, int nxn) {
        const T ub[4] = {u[n0], u[n0 + 1], u[n0 + nxn], u[n0 + nxn + 1]};
        const T vb[4] = {v[n0], v[n0 + 1], v[n0 + nxn], v[n0 + nxn + 1]};
        field(fc, ub, U, Ux, Uy);
        field(fc, vb, V, Vx, Vy);
    }
};

// mode 0: F = A(x) - b on free rows, x - g(t) on fixed rows (the Newton defect).
// mode 1: F = Rhs(x) (velocity rows; Dirichlet rows and pressure rows 0).
// mode 2: F = J(x) dx, J the Newton matrix of the defect at x (fixed rows: identity).
//
// A CTA owns 32 x 4 nodes.  The convection of every cell around them is
// formed once, in the tensor form of the Gauss rule, and its four corners'
// sums go through shared memory; each node then adds its four cells' corners
// to the linear terms.  One thread a node, evaluating its four cells by
// itself, did every cell four times over (FP64 runs at two FMA a clock and
// SM): J(x) dx on 256 x 64 cells in FP64 86 -> 23 us, on
// 1024 x 256 in FP32 20.5 -> 13.9 us (ncu, cold caches).
constexpr int MR_X = 32, MR_Y = 4, MR_CX = MR_X + 1, MR_CELLS = MR_CX * (MR_Y + 1), MR_THREADS = MR_X * MR_Y;

template <typename T, int MODE>
__global__ void __launch_bounds__(MR_THREADS) k_mg_rows(const __grid_constant__ MgLev<T> L, const T *__restrict__ x,
                                                        const T *__restrict__ dx, const T *__restrict__ b, double up,
                                                        T *__restrict__ F) {
    __shared__ T cc[8][MR_CELLS];   // corner sums of 1/2 convection: u rows of SW, SE, NW, NE, then v rows
    __shared__ unsigned char cf[MR_CELLS];
    const FemCoef<T> &fc = L.fc;
    const int nxn = L.nx + 1, N = L.N;
    const int nbx = (L.nx + MR_X) / MR_X;
    const int I0 = (blockIdx.x % nbx) * MR_X, J0 = (blockIdx.x / nbx) * MR_Y;
    const T g0 = fc.cg0, g1 = fc.cg1, hq = T(0.5) * fc.qw;
    for (int e = threadIdx.x; e < MR_CELLS; e += MR_THREADS) {
        const int ey = e / MR_CX, ex = e - ey * MR_CX, ci = I0 - 1 + ex, cj = J0 - 1 + ey;
        const bool f = fluid(L, ci, cj);
        cf[e] = f;
        if (!f) continue;
        const int n0 = cj * nxn + ci;
        CellVel<T> g, h;
        g.eval(fc, x, x + N, n0, nxn);
        if constexpr (MODE == 2) h.eval(fc, dx, dx + N, n0, nxn);
        T tu[2][2], tv[2][2];   // [j][corner along x]
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            T cu[2], cv[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                if constexpr (MODE == 2) {
                    cu[i] = g.U[j][i] * h.Ux[j] + g.V[j][i] * h.Uy[i] + h.U[j][i] * g.Ux[j] + h.V[j][i] * g.Uy[i];
                    cv[i] = g.U[j][i] * h.Vx[j] + g.V[j][i] * h.Vy[i] + h.U[j][i] * g.Vx[j] + h.V[j][i] * g.Vy[i];
                } else {
                    cu[i] = g.U[j][i] * g.Ux[j] + g.V[j][i] * g.Uy[i];
                    cv[i] = g.U[j][i] * g.Vx[j] + g.V[j][i] * g.Vy[i];
                }
            }
            tu[j][0] = g1 * cu[0] + g0 * cu[1];
            tu[j][1] = g0 * cu[0] + g1 * cu[1];
            tv[j][0] = g1 * cv[0] + g0 * cv[1];
            tv[j][1] = g0 * cv[0] + g1 * cv[1];
        }
#pragma unroll
        for (int ax = 0; ax < 2; ++ax) {
            cc[ax][e] = hq * (g1 * tu[0][ax] + g0 * tu[1][ax]);
            cc[2 + ax][e] = hq * (g0 * tu[0][ax] + g1 * tu[1][ax]);
            cc[4 + ax][e] = hq * (g1 * tv[0][ax] + g0 * tv[1][ax]);
            cc[6 + ax][e] = hq * (g0 * tv[0][ax] + g1 * tv[1][ax]);
        }
    }
    __syncthreads();
    const int tx = threadIdx.x % MR_X, ty = threadIdx.x / MR_X, I = I0 + tx, J = J0 + ty;
    if (I > L.nx || J > L.ny) return;
    const int node = J * nxn + I;
    const T *d = MODE == 2 ? dx : x;   // the field of the linear terms
    const T *u = d, *v = d + N, *p = d + 2 * (size_t)N;
    const uint8_t fl = L.flags[node];
    T Au = T(0), Av = T(0), Ap = T(0);
#pragma unroll
    for (int cy = 0; cy < 2; ++cy)
#pragma unroll
        for (int cx = 0; cx < 2; ++cx) {
            const int e = (ty + cy) * MR_CX + tx + cx;
            if (!cf[e]) continue;
            const int a = (1 - cx) + 2 * (1 - cy);       // the node's corner in this cell
            linear_rows(L, u, v, p, I - 1 + cx, J - 1 + cy, a, MODE == 1, Au, Av, Ap);
            Au += MODE == 1 ? -cc[a][e] : cc[a][e];
            Av += MODE == 1 ? -cc[4 + a][e] : cc[4 + a][e];
        }
    if (MODE == 1) {
        const bool fixed = fl & 1;
        F[node] = fixed ? T(0) : Au;
        F[N + node] = fixed ? T(0) : Av;
        F[2 * (size_t)N + node] = T(0);
        return;
    }
    Ap += lps_row(L, p, I, J);
    if (MODE == 2) {
        F[node] = (fl & 1) ? u[node] : Au;
        F[N + node] = (fl & 1) ? v[node] : Av;
        F[2 * (size_t)N + node] = (fl & 4) ? Ap : p[node];
        return;
    }
    if (fl & 1) {
        F[node] = u[node] - ((fl & 2) ? inflow(L, J, up) : T(0));
        F[N + node] = v[node];
    } else {
        F[node] = Au - b[node];
        F[N + node] = Av - b[N + node];
    }
    F[2 * (size_t)N + node] = (fl & 4) ? Ap - b[2 * (size_t)N + node] : p[node];
}

// Programmatic dependent launch: the colour passes of a sweep are launched
// so that a pass may start while the one before it drains; what depends on
// that one comes after the wait (which ends when the pass before has
// completed and its writes are visible).

// One colour pass of the Vanka smoother for J(x) d = rhs: every fluid cell
// (ci, cj) with ci = cx (mod 4), cj = cy (mod 4) solves the 12 x 12 block of
// J(x) on the unknowns of its four nodes against the current defect
// rhs - J(x) d on those unknowns (rows of fixed unknowns: identity) and adds
// omega times the solution to d.  Cells of one colour
// are four cells apart: none reads a node another one writes, so the pass is
// a block Gauss-Seidel step in any order.
//
// A pass has few cells (1/16 of the level) and much serial work in each, so a
// cell is spread over 4 lanes (8 cells a warp): the lanes evaluate the Gauss
// data of the nine cells around it into shared memory, then lane a holds the
// three rows of node a in registers, and the lanes eliminate together
// (Gauss-Jordan; the pivot row comes by shuffle).  One thread a cell, with its
// 12 x 12 block in local memory, left the chip idle: one sweep of 1024 x 256
// cells in FP32 took 0.80 ms (now 0.21), of 256 x 64 in FP64 5.7 ms (now
// 0.245).  16 lanes a cell, one row each, measured 0.65 and 0.6 ms: pivot
// search and role divergence cost more instructions than the lanes save.
// What bounds it now: instruction issue on full levels (0.42 of the slots),
// on small ones the chain of 16 dependent passes (about 5 us each in FP32).
//
// Everything is indexed relative to the row's node a: (ex, ey) says whether a
// cell around the node is in the own cell's column / row (0) or the
// neighbour's (1); b = (bx, by) is the other node of a pair inside that cell,
// 0 = the node itself along that direction.  Node a ^ b of the own cell is in
// cell (ex, ey) iff (bx & ex) == (by & ey) == 0.  Gauss points count from the
// node (0 near, 1 far).
constexpr int VK_LANES = 4, VK_THREADS = 32, VK_CELLS = VK_THREADS / VK_LANES;
constexpr int VK_ROWS = 36 + 7 * 4;
// AHEAD: the block does not depend on d, so it is assembled and eliminated
// before the wait for the colour before (the next colours' CTAs do that while
// this one runs), the multipliers staying in registers and the rows that the
// defect needs in shared memory; after the wait only the defect and its
// elimination remain.  It shortens the chain of 16 colours (one sweep,
// FP64 256 x 64 cells: 535 -> 245 us, 1024 x 256: 2620 -> 2120; FP32
// 256 x 64: 145 -> 88) but takes 164 registers instead of 109 in FP32, so
// there colours that fill the chip go without: 768 x 192 cells (9216 a
// colour) 163 against 179 us, 1024 x 256 (16384) 281 against 212.
constexpr long long VK_AHEAD_CELLS = 10000;
constexpr int VK_G = 17;   // shared values per neighbour cell: U 4, V 4, Ux 2, Vx 2, Uy 2, Vy 2 (odd pitch)

// Magnitudes compared as integers: for values without their sign bit the bit
// patterns order like the values (a NaN above all), and the comparison stays
// off the FP64 pipe.
__device__ __forceinline__ int mag_key(float v) { return __float_as_int(v) & 0x7fffffff; }
__device__ __forceinline__ long long mag_key(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; }
__device__ __forceinline__ float key_mag(int k) { return __int_as_float(k); }
__device__ __forceinline__ double key_mag(long long k) { return __longlong_as_double(k); }

// The element operator of one cell around a node, row by row: products of
// 1D factors of the Gauss rule (2 x 2 points, weights folded into hq).
template <typename T>
struct RowCell {
    T X[2], Y[2];            // (v.grad phi_b, phi_a) / 2, the x and y parts, by (by, bx)
    T jx[2], jv[2];          // (d_x u phi_b, phi_a), (d_x v ...) / 2: factor along y, by by
    T iy[2], iv[2];          // (d_y u phi_b, phi_a), (d_y v ...) / 2: factor along x, by bx
    T sx, sy;                // side of the node in the cell: +1 at its right / upper edge
    __device__ __forceinline__ void set(const FemCoef<T> &fc, const T *q, int cax, int cay) {
        const T g0 = fc.cg0, g1 = fc.cg1, hq = T(0.5) * fc.qw;
        const T w11 = g1 * g1, w00 = g0 * g0, w01 = g0 * g1;
        side(cax, cay);
        T PU[2], PV[2];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int jn = n ^ cay, in = n ^ cax;
            PU[n] = g1 * q[2 * jn + cax] + g0 * q[2 * jn + 1 - cax];
            PV[n] = g1 * q[4 + 2 * cay + in] + g0 * q[4 + 2 * (1 - cay) + in];
        }
        const T cxh = sx * (hq * fc.inv_hx), cyh = sy * (hq * fc.inv_hy);
        X[0] = cxh * (w11 * PU[0] + w00 * PU[1]);
        X[1] = cxh * (w01 * (PU[0] + PU[1]));
        Y[0] = cyh * (w11 * PV[0] + w00 * PV[1]);
        Y[1] = cyh * (w01 * (PV[0] + PV[1]));
        auto pair = [&](const T *d, int near, T (&o)[2]) {
            const T n = hq * d[near], f = hq * d[1 - near];
            o[0] = w11 * n + w00 * f;
            o[1] = w01 * (n + f);
        };
        pair(q + 8, cay, jx);
        pair(q + 10, cay, jv);
        pair(q + 12, cax, iy);
        pair(q + 14, cax, iv);
    }
    __device__ __forceinline__ void side(int cax, int cay) {
        sx = cax ? T(1) : T(-1);
        sy = cay ? T(1) : T(-1);
    }
    // entries of rows (u, v, p) of node a against (u, v, p) of node b: the
    // velocity block, and those that do not depend on x
    __device__ __forceinline__ void velocity(const FemCoef<T> &fc, int bx, int by, T &uu, T &uv, T &vu, T &vv) const {
        const T g0 = fc.cg0, g1 = fc.cg1, m0 = g1 * g1 + g0 * g0, m1 = T(2) * (g0 * g1);
        const T mx = bx ? m1 : m0, my = by ? m1 : m0;
        const T nl = (bx ? -X[by] : X[by]) + (by ? -Y[bx] : Y[bx]) + fc.Av[0][bx + 2 * by];
        uu = nl + mx * jx[by];
        uv = my * iy[bx];
        vu = mx * jv[by];
        vv = nl + my * iv[bx];
    }
    __device__ __forceinline__ void constants(const FemCoef<T> &fc, int bx, int by, T &up, T &vp, T &pu, T &pv) const {
        const T gx = sx * fc.Gx[1][1 + 2 * by], gy = sy * fc.Gy[2][2 + bx];
        up = -gx;
        vp = -gy;
        pu = bx ? -gx : gx;
        pv = by ? -gy : gy;
    }
};

template <typename T, bool AHEAD>
__global__ void __launch_bounds__(VK_THREADS) k_mg_vanka(const __grid_constant__ MgLev<T> L, const T *__restrict__ x,
                                                         const T *__restrict__ rhs, T *dx, T omega, int cx, int cy) {
    __shared__ T sm[VK_CELLS][9 * VK_G];
    // AHEAD: this lane's rows of J, the own cell's columns, then the others
    __shared__ T rows[AHEAD ? VK_ROWS : 1][VK_THREADS];
    constexpr unsigned FULL = 0xffffffffu;
    if constexpr (AHEAD) pdl_trigger();   // the next colour may start on what does not depend on d
    const FemCoef<T> &fc = L.fc;
    const int nx4 = (L.nx - cx + 3) / 4, ny4 = (L.ny - cy + 3) / 4;
    const int lane = threadIdx.x, a = lane & 3, slot = lane / VK_LANES;
    const int id = blockIdx.x * VK_CELLS + slot;
    bool live = id < nx4 * ny4;
    const int cj = live ? cy + 4 * (id / nx4) : cy, ci = live ? cx + 4 * (id % nx4) : cx;
    live = live && !L.solid[(size_t)cj * L.nx + ci];
    const int nxn = L.nx + 1, N = L.N;
    T *gs = sm[slot];
    // ---- Gauss data of the nine cells at x, cell 3 (dj + 1) + di + 1 by lane (that mod 4)
    unsigned fmask = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int c9 = 4 * r + a, di = c9 % 3 - 1, dj = c9 / 3 - 1;
        const bool f = live && c9 < 9 && fluid(L, ci + di, cj + dj);
        if (f) {
            CellVel<T> g;
            g.eval(fc, x, x + N, (cj + dj) * nxn + ci + di, nxn);
            T *o = gs + c9 * VK_G;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    o[2 * j + i] = g.U[j][i];
                    o[4 + 2 * j + i] = g.V[j][i];
                }
                o[8 + j] = g.Ux[j];
                o[10 + j] = g.Vx[j];
                o[12 + j] = g.Uy[j];
                o[14 + j] = g.Vy[j];
            }
        }
        fmask |= ((__ballot_sync(FULL, f) >> (lane & 28)) & 15u) << (4 * r);
    }
    __syncwarp();
    // ---- rows of node a: columns 3 b + component, b relative to the node
    const int ax = a & 1, ay = a >> 1;
    const int I = ci + ax, J = cj + ay, node = J * nxn + I;
    const int dcx = ax ? -1 : 1, dcy = ay ? -1 : 1;   // towards the own cell's other node
    const uint8_t fl = live ? L.flags[node] : 1;      // (a dead slot solves the identity)
    T R[3][12];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < 12; ++i) R[c][i] = T(0);
    bool has[4];   // cell (ex, ey) is fluid
    {
        int o = 36;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int ex = e & 1, ey = e >> 1;
            const int c9 = 3 * ((ey ? -dcy : 0) + 1) + (ex ? -dcx : 0) + 1;
            has[e] = (fmask >> c9) & 1;
            RowCell<T> rc;
            if (has[e]) rc.set(fc, gs + c9 * VK_G, ex ? 1 - ax : ax, ey ? 1 - ay : ay);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int bx = b & 1, by = b >> 1;
                const bool outer = (bx & ex) || (by & ey);
                if (has[e]) {
                    T uu, uv, up, vu, vv, vp, pu, pv;
                    rc.velocity(fc, bx, by, uu, uv, vu, vv);
                    rc.constants(fc, bx, by, up, vp, pu, pv);
                    if (outer && AHEAD) {
                        // kept for the defect (the constant entries are formed again there)
                        rows[o][lane] = uu;
                        rows[o + 1][lane] = uv;
                        rows[o + 2][lane] = vu;
                        rows[o + 3][lane] = vv;
                    } else if (!outer) {
                        R[0][3 * b] += uu;
                        R[0][3 * b + 1] += uv;
                        R[0][3 * b + 2] += up;
                        R[1][3 * b] += vu;
                        R[1][3 * b + 1] += vv;
                        R[1][3 * b + 2] += vp;
                        R[2][3 * b] += pu;
                        R[2][3 * b + 1] += pv;
                    }
                }
                if (outer && AHEAD) o += 4;
            }
        }
    }
    if constexpr (AHEAD) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int i = 0; i < 12; ++i) rows[12 * c + i][lane] = R[c][i];
    }
    // projection term of the node's pressure row: its entries in the own cell
    // (lp), and where its (up to four) patches' rows are
    T lp[4] = {T(0), T(0), T(0), T(0)};
    const T *Sp[4];
    int pbase[4];   // first node of the patch, -1: no such patch
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int qx = q & 1, qy = q >> 1;
        const int m = (I - qx) >> 1, n = (J - qy) >> 1;   // 2m <= I <= 2m + 2, 2n <= J <= 2n + 2
        int mask = 0;
        if (live && !(qx && (I & 1)) && !(qy && (J & 1))) mask = patch_mask(L, m, n);
        const int il = I - 2 * m, jl = J - 2 * n;
        pbase[q] = mask ? 2 * n * nxn + 2 * m : -1;
        Sp[q] = L.lps + (mask ? (mask * 9 + 3 * jl + il) * 9 : 0);
        if (mask) {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int ib = il + ((b & 1) ? dcx : 0), jb = jl + ((b >> 1) ? dcy : 0);
                if (ib >= 0 && ib <= 2 && jb >= 0 && jb <= 2) lp[b] += Sp[q][3 * jb + ib];
            }
        }
    }
    // ---- the defect rhs - J(x) d on the node's unknowns (everything that
    // depends on d, which the pass before wrote)
    T z[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) z[c] = live ? rhs[(size_t)c * N + node] : T(0);
    auto defect = [&]() {
        if constexpr (!AHEAD) pdl_trigger();
        pdl_wait();
        if (!live) return;
        const T *du = dx, *dv = dx + N, *dp = dx + 2 * (size_t)N;
        const T own[3] = {du[node], dv[node], dp[node]};
        T jd[3] = {T(0), T(0), T(0)};
        // the own cell's nodes
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int n = node + ((b & 1) ? dcx : 0) + ((b >> 1) ? dcy * nxn : 0);
            const T d0 = du[n], d1 = dv[n], d2 = dp[n];
            auto at = [&](int c, int i) { return AHEAD ? rows[AHEAD ? 12 * c + i : 0][lane] : R[c][i]; };
#pragma unroll
            for (int c = 0; c < 3; ++c) jd[c] += at(c, 3 * b) * d0 + at(c, 3 * b + 1) * d1 + at(c, 3 * b + 2) * d2;
        }
        // the other nodes of the cells around the node
        int o = 36;
#pragma unroll
        for (int e = 1; e < 4; ++e) {
            const int ex = e & 1, ey = e >> 1;
            if (!has[e]) {
                o += ex && ey ? 12 : 8;
                continue;
            }
            RowCell<T> rc;
            if constexpr (AHEAD) rc.side(ex ? 1 - ax : ax, ey ? 1 - ay : ay);
            else rc.set(fc, gs + (3 * ((ey ? -dcy : 0) + 1) + (ex ? -dcx : 0) + 1) * VK_G, ex ? 1 - ax : ax, ey ? 1 - ay : ay);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int bx = b & 1, by = b >> 1;
                if (!((bx & ex) || (by & ey))) continue;
                const int n = node + (bx ? (ex ? -dcx : dcx) : 0) + (by ? (ey ? -dcy : dcy) * nxn : 0);
                const T d0 = du[n], d1 = dv[n], d2 = dp[n];
                T uu, uv, up, vu, vv, vp, pu, pv;
                rc.constants(fc, bx, by, up, vp, pu, pv);
                if constexpr (AHEAD) {
                    uu = rows[o][lane];
                    uv = rows[o + 1][lane];
                    vu = rows[o + 2][lane];
                    vv = rows[o + 3][lane];
                    o += 4;
                } else {
                    rc.velocity(fc, bx, by, uu, uv, vu, vv);
                }
                jd[0] += uu * d0 + uv * d1 + up * d2;
                jd[1] += vu * d0 + vv * d1 + vp * d2;
                jd[2] += pu * d0 + pv * d1;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (pbase[q] < 0) continue;
            const T *pp = dp + pbase[q];
#pragma unroll
            for (int kb = 0; kb < 3; ++kb)
#pragma unroll
                for (int ka = 0; ka < 3; ++ka) jd[2] += Sp[q][3 * kb + ka] * pp[kb * nxn + ka];
        }
        z[0] -= (fl & 1) ? own[0] : jd[0];
        z[1] -= (fl & 1) ? own[1] : jd[1];
        z[2] -= (fl & 4) ? jd[2] : own[2];
    };
    if constexpr (!AHEAD) defect();
#pragma unroll
    for (int b = 0; b < 4; ++b) R[2][3 * b + 2] += lp[b];
    // rows of fixed unknowns: identity; columns by absolute node, b ^ a
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const bool fixed = c < 2 ? (fl & 1) : !(fl & 4);
#pragma unroll
        for (int i = 0; i < 12; ++i) R[c][i] = fixed ? (i == c ? T(1) : T(0)) : R[c][i];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (ax) {
                const T t0 = R[c][i], t1 = R[c][6 + i];
                R[c][i] = R[c][3 + i];
                R[c][3 + i] = t0;
                R[c][6 + i] = R[c][9 + i];
                R[c][9 + i] = t1;
            }
            if (ay) {
                const T t0 = R[c][i], t1 = R[c][3 + i];
                R[c][i] = R[c][6 + i];
                R[c][6 + i] = t0;
                R[c][3 + i] = R[c][9 + i];
                R[c][9 + i] = t1;
            }
        }
    }
    // ---- Gauss-Jordan elimination with partial pivoting over the 12 rows; the
    // multipliers stay in the eliminated columns.  (As accurate as elimination
    // below the pivot with back substitution, to a few percent of the rounding
    // error.  Two sweeps against 64 bits, means of six inputs, here and there: FP32
    // 1024 x 256 cells 2.04e-7 and 1.95e-7, 512 x 128 1.50e-7 and 1.55e-7, 200 x 48
    // 1.36e-7 and 1.31e-7, FP64 256 x 64 4.11e-16 and 4.14e-16.)  A
    // block can be singular: a cell whose 4 nodes all hold Dirichlet velocities
    // couples its pressures only through the projection term, which vanishes
    // on linear functions.  A pivot below a relative threshold leaves that
    // unknown's correction 0 and drops its row.  pos is a row's place under
    // the exchanges (ties go to the first row); unk the unknown it became.
    using Key = decltype(mag_key(T(0)));
    Key scale = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < 12; ++i) scale = max(scale, mag_key(R[c][i]));
    scale = max(scale, __shfl_xor_sync(FULL, scale, 1));
    scale = max(scale, __shfl_xor_sync(FULL, scale, 2));
    const T tiny = key_mag(scale) * (sizeof(T) == 8 ? T(1e-12) : T(1e-6));
    int pos[3] = {3 * a, 3 * a + 1, 3 * a + 2}, unk[3] = {-1, -1, -1};
    T dinv[3] = {T(0), T(0), T(0)};
    unsigned long long prows = 0;   // pivot row of each column, 4 bits
    unsigned deads = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        // the largest |entry| of column k among the rows not used yet, as (value, place, row);
        // a NaN is the largest key, so every lane agrees on it and it spreads to the whole block
        Key best = -1;
        int idx = 0xffff;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const Key v = unk[c] >= 0 ? Key(-1) : mag_key(R[c][k]);
            const int iv = (pos[c] << 4) | (3 * a + c);
            if (v > best || (v == best && iv < idx)) {
                best = v;
                idx = iv;
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const Key ov = __shfl_xor_sync(FULL, best, o);
            const int oi = __shfl_xor_sync(FULL, idx, o);
            if (ov > best || (ov == best && oi < idx)) {
                best = ov;
                idx = oi;
            }
        }
        const int prow = idx & 15, ppos = idx >> 4, pl = prow / 3, pc = prow - 3 * pl;
        const bool dead = key_mag(best) <= tiny;
        prows |= (unsigned long long)prow << (4 * k);
        deads |= (dead ? 1u : 0u) << k;
        // the pivot row, from lane pl of the cell
        T pv[12];
#pragma unroll
        for (int j = k; j < 12; ++j) {
            const T v = pc == 0 ? R[0][j] : (pc == 1 ? R[1][j] : R[2][j]);
            pv[j] = __shfl_sync(FULL, v, pl, 4);
        }
        T pz = T(0);
        if constexpr (!AHEAD) pz = __shfl_sync(FULL, pc == 0 ? z[0] : (pc == 1 ? z[1] : z[2]), pl, 4);
        const T inv = dead ? T(0) : T(1) / pv[k];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const bool piv = prow == 3 * a + c;
            const T f = piv ? T(0) : R[c][k] * inv;
            R[c][k] = f;
#pragma unroll
            for (int j = k + 1; j < 12; ++j) R[c][j] -= f * pv[j];
            if constexpr (!AHEAD) z[c] -= f * pz;
            if (pos[c] == k) pos[c] = ppos;
            if (piv) {
                pos[c] = k;
                unk[c] = k;
                dinv[c] = inv;
                if (dead) {
                    if constexpr (!AHEAD) z[c] = T(0);
#pragma unroll
                    for (int j = k + 1; j < 12; ++j) R[c][j] = T(0);
                }
            }
        }
    }
    if constexpr (AHEAD) {
        // the elimination of the right-hand side
        defect();
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int prow = (int)(prows >> (4 * k)) & 15, pl = prow / 3, pc = prow - 3 * pl;
            const T pz = __shfl_sync(FULL, pc == 0 ? z[0] : (pc == 1 ? z[1] : z[2]), pl, 4);
            const bool dead = (deads >> k) & 1;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                z[c] -= R[c][k] * pz;
                if (dead && prow == 3 * a + c) z[c] = T(0);
            }
        }
    }
    if (live) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (unk[c] < 0) continue;
            const int ua = unk[c] / 3, uc = unk[c] - 3 * ua;
            dx[(size_t)uc * N + (cj + (ua >> 1)) * nxn + ci + (ua & 1)] += omega * (z[c] * dinv[c]);
        }
    }
}

// End of a Vanka sweep: every fixed unknown (an identity row of J) takes its
// exact correction, its defect: d = rhs there.  This also reaches the nodes
// that no fluid cell holds (inside an obstacle), which no cell block visits.
template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_fixed(MgLev<T> L, const T *__restrict__ rhs, T *dx) {
    pdl_wait();   // the last colour pass of the sweep
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= L.N) return;
    const uint8_t fl = L.flags[node];
    if (fl & 1) {
        dx[node] = rhs[node];
        dx[L.N + node] = rhs[L.N + node];
    }
    if (!(fl & 4)) dx[2 * L.N + node] = rhs[2 * L.N + node];
}

// Restriction rc = P^T rf from level l (fine) to l+1 (coarse): full weighting
// (weights 1, 1/2, 1/4 of the bilinear prolongation); fixed coarse rows 0.
template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_restrict(MgLev<T> F, MgLev<T> C, const T *__restrict__ rf,
                                                            T *__restrict__ rc) {
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= C.N) return;
    const int cn = C.nx + 1, i = node % cn, j = node / cn, fn = F.nx + 1;
    const uint8_t fl = C.flags[node];
    T acc[3] = {T(0), T(0), T(0)};
    for (int dj = -1; dj <= 1; ++dj) {
        const int J = 2 * j + dj;
        if (J < 0 || J > F.ny) continue;
        for (int di = -1; di <= 1; ++di) {
            const int I = 2 * i + di;
            if (I < 0 || I > F.nx) continue;
            const T w = (di ? T(0.5) : T(1)) * (dj ? T(0.5) : T(1));
            const int n = J * fn + I;
            for (int c = 0; c < 3; ++c) acc[c] += w * rf[c * F.N + n];
        }
    }
    rc[node] = (fl & 1) ? T(0) : acc[0];
    rc[C.N + node] = (fl & 1) ? T(0) : acc[1];
    rc[2 * C.N + node] = (fl & 4) ? acc[2] : T(0);
}

// df += P dc (bilinear prolongation from level l+1 to l); fixed fine rows unchanged.
template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_prolong_add(MgLev<T> F, MgLev<T> C, const T *__restrict__ dc,
                                                               T *__restrict__ df) {
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= F.N) return;
    const int fn = F.nx + 1, I = node % fn, J = node / fn, cn = C.nx + 1;
    const uint8_t fl = F.flags[node];
    const int i0 = I >> 1, j0 = J >> 1, i1 = (I + 1) >> 1, j1 = (J + 1) >> 1;
    const T h = T(0.5);
    for (int c = 0; c < 3; ++c) {
        const bool fixed = c < 2 ? (fl & 1) : !(fl & 4);
        if (fixed) continue;
        const T *d = dc + c * C.N;
        const T v = h * (h * (d[j0 * cn + i0] + d[j0 * cn + i1]) + h * (d[j1 * cn + i0] + d[j1 * cn + i1]));
        df[c * F.N + node] += v;
    }
}

// xc = x_f at the coarse nodes (the linearisation point of a coarser level).
template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_inject(MgLev<T> F, MgLev<T> C, const T *__restrict__ xf,
                                                          T *__restrict__ xc) {
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= C.N) return;
    const int cn = C.nx + 1, i = node % cn, j = node / cn;
    const int n = (2 * j) * (F.nx + 1) + 2 * i;
    for (int c = 0; c < 3; ++c) xc[c * C.N + node] = xf[c * F.N + n];
}

template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_dot(const T *__restrict__ a, const T *__restrict__ b, long long n,
                                                       double *__restrict__ out) {
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        acc += (double)a[i] * (double)b[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ double part[MG_THREADS / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = threadIdx.x < MG_THREADS / 32 ? part[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) atomicAdd(out, acc);
    }
}

template <typename T>
__global__ void __launch_bounds__(MG_THREADS) k_mg_axpby(T alpha, const T *__restrict__ x, T beta, T *__restrict__ y,
                                                         long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = alpha * x[i] + (beta == T(0) ? T(0) : beta * y[i]);
}

}  // namespace

// ---------------------------------------------------------------- host side
struct MgLevelHost {
    int nx, ny, N;
    std::vector<uint8_t> solid, flags, mult;
    uint8_t *d_solid = nullptr, *d_flags = nullptr, *d_mult = nullptr;
    double *d_lps64 = nullptr;
    float *d_lps32 = nullptr;
    FemCoef<double> f64;
    FemCoef<float> f32;
};

}  // namespace dnnmg

struct dnnmg_mg_s {
    dnnmg_mg_desc desc;
    int device;
    std::vector<dnnmg::MgLevelHost> levels;
};

namespace dnnmg {
namespace {

template <typename T> MgLev<T> dev_level(const dnnmg_mg_s &m, int l) {
    const MgLevelHost &h = m.levels[l];
    MgLev<T> L;
    L.nx = h.nx;
    L.ny = h.ny;
    L.N = h.N;
    L.solid = h.d_solid;
    L.flags = h.d_flags;
    L.mult = h.d_mult;
    if constexpr (sizeof(T) == 8) L.lps = h.d_lps64;
    else L.lps = h.d_lps32;
    L.hy = m.desc.ly / h.ny;
    L.ly = m.desc.ly;
    if constexpr (sizeof(T) == 8) L.fc = h.f64;
    else L.fc = h.f32;
    return L;
}

// Node flags (Sec. 6.1 boundary classes) and fluid-cell counts of a level.
void node_classes(MgLevelHost &h) {
    const int nx = h.nx, ny = h.ny, nxn = nx + 1;
    h.flags.assign(h.N, 0);
    h.mult.assign(h.N, 0);
    for (int J = 0; J <= ny; ++J)
        for (int I = 0; I <= nx; ++I) {
            bool touch_solid = false, touch_fluid = false;
            int m = 0;
            for (int cy = 0; cy < 2; ++cy)
                for (int cx = 0; cx < 2; ++cx) {
                    const int ci = I - 1 + cx, cj = J - 1 + cy;
                    if (ci < 0 || cj < 0 || ci >= nx || cj >= ny) continue;
                    if (h.solid[(size_t)cj * nx + ci]) touch_solid = true;
                    else {
                        touch_fluid = true;
                        ++m;
                    }
                }
            const bool wall = J == 0 || J == ny;
            const bool dir = wall || I == 0 || touch_solid;
            const bool inflow = I == 0 && !wall && !touch_solid;
            h.flags[(size_t)J * nxn + I] = (uint8_t)((dir ? 1 : 0) | (inflow ? 2 : 0) | (touch_fluid ? 4 : 0));
            h.mult[(size_t)J * nxn + I] = (uint8_t)m;
        }
}

int check_level(const dnnmg_mg_s *m, int level, int need_coarser = 0) {
    if (!m) return fail(DNNMG_EINVAL, "multigrid handle is NULL");
    if (level < 0 || level + need_coarser >= (int)m->levels.size())
        return fail(DNNMG_EINVAL, "level %d out of range (%zu levels)", level, m->levels.size());
    int cur = -1;
    DNNMG_CUDA_TRY(cudaGetDevice(&cur));
    if (cur != m->device) return fail(DNNMG_EINVAL, "handle belongs to device %d but device %d is current", m->device, cur);
    return DNNMG_OK;
}

unsigned blocks(long long n, int th) { return (unsigned)((n + th - 1) / th); }
unsigned rows_grid(const dnnmg_mg_s *m, int l) {
    return blocks(m->levels[l].nx + 1, MR_X) * blocks(m->levels[l].ny + 1, MR_Y);
}

// Projection patch matrices by the patch's fluid cells: for each subset (bit
// 2 cb + ca), the sum over its cells T of alpha (grad(p - pi p), grad(q - pi q))_T
// on the 9 patch nodes (Eq. disc:ns; a partly solid patch of a single level's
// own mask contributes its fluid cells only).  pi: the bilinear interpolant of
// the patch's 4 corners; alpha = alpha0 (hx^2 + hy^2) / nu.
void lps_tables(const FemCoef<double> &f, double hx, double hy, double alpha0, double nu, std::vector<double> *out) {
    double S[4][4];   // (grad phi_a, grad phi_b) over one cell, 2 x 2 Gauss
    for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) {
            double s = 0.0;
            for (int q = 0; q < 4; ++q) s += f.qw * (f.qdx[q][a] * f.qdx[q][b] + f.qdy[q][a] * f.qdy[q][b]);
            S[a][b] = s;
        }
    double F[9][9];   // I - pi
    for (int i = 0; i < 9; ++i)
        for (int j = 0; j < 9; ++j) F[i][j] = i == j ? 1.0 : 0.0;
    for (int b = 0; b < 3; ++b)
        for (int a = 0; a < 3; ++a) {
            const double X = a / 2.0, Y = b / 2.0;
            F[3 * b + a][0] -= (1 - X) * (1 - Y);
            F[3 * b + a][2] -= X * (1 - Y);
            F[3 * b + a][6] -= (1 - X) * Y;
            F[3 * b + a][8] -= X * Y;
        }
    const double alpha = alpha0 * (hx * hx + hy * hy) / nu;
    double Lc[4][9][9];
    for (int c = 0; c < 4; ++c) {
        const int ca = c & 1, cb = c >> 1;
        double S9[9][9] = {};
        const int ids[4] = {3 * cb + ca, 3 * cb + ca + 1, 3 * (cb + 1) + ca, 3 * (cb + 1) + ca + 1};
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b < 4; ++b) S9[ids[a]][ids[b]] = S[a][b];
        for (int i = 0; i < 9; ++i)
            for (int j = 0; j < 9; ++j) {
                double s = 0.0;
                for (int k = 0; k < 9; ++k)
                    for (int l = 0; l < 9; ++l) s += F[k][i] * S9[k][l] * F[l][j];
                Lc[c][i][j] = alpha * s;
            }
    }
    out->assign(16 * 81, 0.0);
    for (int mask = 0; mask < 16; ++mask)
        for (int c = 0; c < 4; ++c)
            if (mask & (1 << c))
                for (int i = 0; i < 81; ++i) (*out)[mask * 81 + i] += (&Lc[c][0][0])[i];
}

// One sweep: the 16 colour passes and the fixed unknowns.  Each pass may start
// while the one before it drains (programmatic launch), except the first,
// whose inputs the work before the sweep may still be writing.
template <typename T>
cudaError_t vanka_sweep(const dnnmg_mg_s &m, int level, const T *x, const T *r, T *dx, T omega, cudaStream_t st) {
    const MgLev<T> L = dev_level<T>(m, level);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cfg.attrs = &at;
    cudaError_t e;
    for (int c = 0; c < 16; ++c) {
        const int cx = c & 3, cy = c >> 2;
        const long long nc = (long long)((L.nx - cx + 3) / 4) * ((L.ny - cy + 3) / 4);
        if (nc <= 0) continue;
        cfg.gridDim = dim3(blocks(nc, VK_CELLS));
        cfg.blockDim = dim3(VK_THREADS);
        auto k = k_mg_vanka<T, true>;
        if constexpr (sizeof(T) == 4)
            if (nc > VK_AHEAD_CELLS) k = k_mg_vanka<T, false>;
        if ((e = cudaLaunchKernelEx(&cfg, k, L, x, r, dx, omega, cx, cy)) != cudaSuccess) return e;
        cfg.numAttrs = 1;
    }
    cfg.gridDim = dim3(blocks(L.N, MG_THREADS));
    cfg.blockDim = dim3(MG_THREADS);
    return cudaLaunchKernelEx(&cfg, k_mg_fixed<T>, L, r, dx);
}

}  // namespace
}  // namespace dnnmg

using namespace dnnmg;

extern "C" {

int dnnmg_mg_create(const dnnmg_mg_desc *d, dnnmg_mg_t *out) {
    clear_error();
    if (!d || !out) return fail(DNNMG_EINVAL, "NULL argument");
    *out = nullptr;
    if (d->levels < 1 || d->levels > 12) return fail(DNNMG_EINVAL, "levels=%d out of range 1..12", d->levels);
    const int div = 1 << d->levels;
    if (d->nx <= 0 || d->ny <= 0 || d->nx % div || d->ny % div)
        return fail(DNNMG_EINVAL, "nx=%d, ny=%d must be positive multiples of 2^levels = %d", d->nx, d->ny, div);
    if (!(d->lx > 0) || !(d->ly > 0) || !(d->nu > 0) || !(d->k > 0) || !(d->alpha0 >= 0))
        return fail(DNNMG_EINVAL, "lx, ly, nu, k must be > 0 and alpha0 >= 0");
    if (d->precision != DNNMG_F64 && d->precision != DNNMG_F32)
        return fail(DNNMG_EINVAL, "precision must be DNNMG_F64 or DNNMG_F32");
    if ((long long)(d->nx + 1) * (d->ny + 1) > (1LL << 30)) return fail(DNNMG_EUNSUPPORTED, "too many nodes");
    dnnmg_mg_s *m = new (std::nothrow) dnnmg_mg_s();
    if (!m) return fail(DNNMG_ENOMEM, "host allocation failed");
    m->desc = *d;
    m->desc.solid = nullptr;
    cudaGetDevice(&m->device);
    m->levels.resize(d->levels);
    for (int l = 0; l < d->levels; ++l) {
        MgLevelHost &h = m->levels[l];
        h.nx = d->nx >> l;
        h.ny = d->ny >> l;
        h.N = (h.nx + 1) * (h.ny + 1);
        h.solid.assign((size_t)h.nx * h.ny, 0);
        if (l == 0) {
            if (d->solid)
                for (size_t i = 0; i < h.solid.size(); ++i) h.solid[i] = d->solid[i] ? 1 : 0;
        } else {
            // patch (m, n) of this level is solid iff all 16 cells of the finer level under it are
            const MgLevelHost &f = m->levels[l - 1];
            for (int n = 0; n < h.ny / 2; ++n)
                for (int mm = 0; mm < h.nx / 2; ++mm) {
                    bool all = true;
                    for (int jj = 0; jj < 4 && all; ++jj)
                        for (int ii = 0; ii < 4 && all; ++ii)
                            if (!f.solid[(size_t)(4 * n + jj) * f.nx + 4 * mm + ii]) all = false;
                    for (int jj = 0; jj < 2; ++jj)
                        for (int ii = 0; ii < 2; ++ii) h.solid[(size_t)(2 * n + jj) * h.nx + 2 * mm + ii] = all ? 1 : 0;
                }
        }
        node_classes(h);
        // every level keeps the finest level's projection coefficient alpha:
        // the fine term vanishes on prolongated pressures, and a coefficient
        // growing with h^2 would swamp the coarse pressure corrections
        const double alpha0_l = d->alpha0 / (double)(1LL << (2 * l));
        level_coefficients(d->lx, d->ly, h.nx, h.ny, d->nu, d->k, alpha0_l, &h.f64, &h.f32);
        std::vector<double> lps;
        lps_tables(h.f64, d->lx / h.nx, d->ly / h.ny, alpha0_l, d->nu, &lps);
        std::vector<float> lps32(lps.begin(), lps.end());
        if (cudaMalloc(&h.d_lps64, lps.size() * sizeof(double)) != cudaSuccess ||
            cudaMalloc(&h.d_lps32, lps32.size() * sizeof(float)) != cudaSuccess ||
            cudaMemcpy(h.d_lps64, lps.data(), lps.size() * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(h.d_lps32, lps32.data(), lps32.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaGetLastError();
            dnnmg_mg_destroy(m);
            return fail(DNNMG_ENOMEM, "device allocation of level %d failed", l);
        }
        if (cudaMalloc(&h.d_solid, h.solid.size()) != cudaSuccess || cudaMalloc(&h.d_flags, h.N) != cudaSuccess ||
            cudaMalloc(&h.d_mult, h.N) != cudaSuccess ||
            cudaMemcpy(h.d_solid, h.solid.data(), h.solid.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(h.d_flags, h.flags.data(), h.N, cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(h.d_mult, h.mult.data(), h.N, cudaMemcpyHostToDevice) != cudaSuccess) {
            cudaGetLastError();
            dnnmg_mg_destroy(m);
            return fail(DNNMG_ENOMEM, "device allocation of level %d failed", l);
        }
    }
    *out = m;
    return DNNMG_OK;
}

int dnnmg_mg_destroy(dnnmg_mg_t m) {
    clear_error();
    if (!m) return DNNMG_OK;
    for (MgLevelHost &h : m->levels) {
        cudaFree(h.d_solid);
        cudaFree(h.d_flags);
        cudaFree(h.d_mult);
        cudaFree(h.d_lps64);
        cudaFree(h.d_lps32);
    }
    delete m;
    return DNNMG_OK;
}

int dnnmg_mg_level(dnnmg_mg_t m, int level, int *nx, int *ny, unsigned char *solid) {
    clear_error();
    if (!m) return fail(DNNMG_EINVAL, "multigrid handle is NULL");
    if (level < 0 || level >= (int)m->levels.size()) return fail(DNNMG_EINVAL, "level %d out of range", level);
    const MgLevelHost &h = m->levels[level];
    if (nx) *nx = h.nx;
    if (ny) *ny = h.ny;
    if (solid)
        for (size_t i = 0; i < h.solid.size(); ++i) solid[i] = h.solid[i];
    return DNNMG_OK;
}

#define MG_DISPATCH(call_f64, call_f32)                         \
    do {                                                        \
        if (m->desc.precision == DNNMG_F64) { call_f64; }       \
        else { call_f32; }                                      \
        DNNMG_CUDA_TRY(cudaGetLastError());                     \
    } while (0)

static double inflow_peak_mg(const dnnmg_mg_desc &d, double t) {
    const double w = d.ramp ? (t <= 0.5 ? 0.5 - 0.5 * std::cos(2.0 * 3.14159265358979323846 * t) : 1.0) : 1.0;
    return d.u_max * w;
}

int dnnmg_mg_defect(dnnmg_mg_t m, int level, const void *x, const void *b, double t, void *F, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level)) return e;
    if (!x || !b || !F) return fail(DNNMG_EINVAL, "NULL array");
    const double up = inflow_peak_mg(m->desc, t);
    MG_DISPATCH((k_mg_rows<double, 0><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), (const double *)x, nullptr, (const double *)b, up, (double *)F)),
                (k_mg_rows<float, 0><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), (const float *)x, nullptr, (const float *)b, up, (float *)F)));
    return DNNMG_OK;
}

int dnnmg_mg_rhs(dnnmg_mg_t m, int level, const void *x, void *b, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level)) return e;
    if (!x || !b) return fail(DNNMG_EINVAL, "NULL array");
    if (x == b) return fail(DNNMG_EINVAL, "x and b must not alias");
    MG_DISPATCH((k_mg_rows<double, 1><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), (const double *)x, nullptr, nullptr, 0.0, (double *)b)),
                (k_mg_rows<float, 1><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), (const float *)x, nullptr, nullptr, 0.0, (float *)b)));
    return DNNMG_OK;
}

int dnnmg_mg_jvp(dnnmg_mg_t m, int level, const void *x, const void *dx, void *y, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level)) return e;
    if (!x || !dx || !y) return fail(DNNMG_EINVAL, "NULL array");
    if (y == dx || y == x) return fail(DNNMG_EINVAL, "y must not alias x or dx");
    MG_DISPATCH((k_mg_rows<double, 2><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), (const double *)x, (const double *)dx, nullptr, 0.0, (double *)y)),
                (k_mg_rows<float, 2><<<rows_grid(m, level), MR_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), (const float *)x, (const float *)dx, nullptr, 0.0, (float *)y)));
    return DNNMG_OK;
}

int dnnmg_mg_vanka(dnnmg_mg_t m, int level, const void *x, const void *r, void *dx, double omega, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level)) return e;
    if (!x || !r || !dx) return fail(DNNMG_EINVAL, "NULL array");
    if (dx == r || dx == x) return fail(DNNMG_EINVAL, "dx must not alias x or r");
    DNNMG_CUDA_TRY(m->desc.precision == DNNMG_F64
                       ? vanka_sweep(*m, level, (const double *)x, (const double *)r, (double *)dx, omega, s)
                       : vanka_sweep(*m, level, (const float *)x, (const float *)r, (float *)dx, (float)omega, s));
    return DNNMG_OK;
}

int dnnmg_mg_restrict(dnnmg_mg_t m, int level, const void *rf, void *rc, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level, 1)) return e;
    if (!rf || !rc) return fail(DNNMG_EINVAL, "NULL array");
    const int Nc = m->levels[level + 1].N;
    MG_DISPATCH((k_mg_restrict<double><<<blocks(Nc, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), dev_level<double>(*m, level + 1), (const double *)rf, (double *)rc)),
                (k_mg_restrict<float><<<blocks(Nc, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), dev_level<float>(*m, level + 1), (const float *)rf, (float *)rc)));
    return DNNMG_OK;
}

int dnnmg_mg_prolong_add(dnnmg_mg_t m, int level, const void *dc, void *df, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level, 1)) return e;
    if (!dc || !df) return fail(DNNMG_EINVAL, "NULL array");
    const int Nf = m->levels[level].N;
    MG_DISPATCH((k_mg_prolong_add<double><<<blocks(Nf, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), dev_level<double>(*m, level + 1), (const double *)dc, (double *)df)),
                (k_mg_prolong_add<float><<<blocks(Nf, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), dev_level<float>(*m, level + 1), (const float *)dc, (float *)df)));
    return DNNMG_OK;
}

int dnnmg_mg_inject(dnnmg_mg_t m, int level, const void *xf, void *xc, cudaStream_t s) {
    clear_error();
    if (int e = check_level(m, level, 1)) return e;
    if (!xf || !xc) return fail(DNNMG_EINVAL, "NULL array");
    const int Nc = m->levels[level + 1].N;
    MG_DISPATCH((k_mg_inject<double><<<blocks(Nc, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<double>(*m, level), dev_level<double>(*m, level + 1), (const double *)xf, (double *)xc)),
                (k_mg_inject<float><<<blocks(Nc, MG_THREADS), MG_THREADS, 0, s>>>(
                    dev_level<float>(*m, level), dev_level<float>(*m, level + 1), (const float *)xf, (float *)xc)));
    return DNNMG_OK;
}

int dnnmg_mg_dot(dnnmg_mg_t m, long long n, const void *a, const void *b, double *out, cudaStream_t s) {
    clear_error();
    if (!m) return fail(DNNMG_EINVAL, "multigrid handle is NULL");
    if (!a || !b || !out || n < 0) return fail(DNNMG_EINVAL, "NULL array or negative size");
    DNNMG_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(double), s));
    if (n == 0) return DNNMG_OK;
    const unsigned g = blocks(n, MG_THREADS) < 152u * 8u ? blocks(n, MG_THREADS) : 152u * 8u;
    MG_DISPATCH((k_mg_dot<double><<<g, MG_THREADS, 0, s>>>((const double *)a, (const double *)b, n, out)),
                (k_mg_dot<float><<<g, MG_THREADS, 0, s>>>((const float *)a, (const float *)b, n, out)));
    return DNNMG_OK;
}

int dnnmg_mg_axpby(dnnmg_mg_t m, long long n, double alpha, const void *x, double beta, void *y, cudaStream_t s) {
    clear_error();
    if (!m) return fail(DNNMG_EINVAL, "multigrid handle is NULL");
    if (!x || !y || n < 0) return fail(DNNMG_EINVAL, "NULL array or negative size");
    if (n == 0) return DNNMG_OK;
    const unsigned g = blocks(n, MG_THREADS) < 152u * 8u ? blocks(n, MG_THREADS) : 152u * 8u;
    MG_DISPATCH((k_mg_axpby<double><<<g, MG_THREADS, 0, s>>>(alpha, (const double *)x, beta, (double *)y, n)),
                (k_mg_axpby<float><<<g, MG_THREADS, 0, s>>>((float)alpha, (const float *)x, (float)beta, (float *)y,
                                                           n)));
    return DNNMG_OK;
}

}  // extern "C"

// Fused step of small lattices without obstacles: one node per thread, plain
// loads; one step per launch, or several.
//
// A lattice whose CTAs all fit the GPU at once is bound by latency: a
// dependent launch costs 0.6 us, a global load and a store 0.5 us more, and
// then every stage of a pipeline adds to the step.  The staged kernels
// (lb_step.cuh and its FP64 and compact forms), made for bandwidth, put a
// bulk copy (0.7 us more than plain loads), its barriers and the phi of three
// rows in series in front of a row.  Here a CTA takes 32 columns x TY rows
// and has all its loads in flight at once:
//  - FP32 and FP64 full storage: a thread pulls f and g of its node and g of
//    a position of the one-node halo (those with the highest index first);
//    phi of both goes to shared memory, the CTA meets, and each thread
//    collides its node from the 3 x 3 phi around it.
//  - compact g storage: a thread loads the four compact values of positions
//    on the tile and a two-node halo, expands them to g' in shared memory;
//    then phi(t+1) of the tile and a one-node halo is formed from the g' that
//    arrive there; then the nodes collide.
//  - the smallest: FP32 (both storages) takes up to four steps per launch,
//    with a border of two nodes more per step around the tile (small_steps);
//    FP64, bound by its pipe instead, splits a node over two threads
//    (small_split64).
// us a step, staged, one step per launch, and as here: FP32 28 x 15 4.0, 2.3, 1.4,
// 200 x 100 4.4, 2.7, 1.8; compact 28 x 15 4.5, 3.4, 1.8, 200 x 100 4.9, 3.5, 2.2;
// FP64 28 x 15 8.3, 6.6, 5.1, 200 x 100 11, 7.6.
// The arithmetic is that of the staged kernels, operation for operation, and
// so are the stored populations and ghost columns, bit for bit.
#include <cuda_runtime.h>

#include "lb_internal.h"
#include "lb_node.cuh"
#include "lb_node64.cuh"
#include "lb_node_x2.cuh"
#include "lb_small.h"
#include "lb_step.cuh"

namespace lbfe {

namespace {

constexpr int kTX = 32;          // columns of a tile
constexpr int kPW = kTX + 2;     // phi array: one halo column on each side
constexpr int kEW = kTX + 4;     // g' array (compact): two

// The tile of a CTA: node columns [x0, x0 + wc), rows [y0, y0 + hc).
struct SmallTile {
    int x0, y0, wc, hc;
    __device__ __forceinline__ SmallTile(const DomDesc& D, int x0_, int y0_, int ty)
        : x0(x0_), y0(y0_), wc(min(kTX, D.nx - x0)), hc(min(ty, D.ny - y0))
    {
    }
};

// The nine pulled values of the node at column x (-1 .. nx: ghost columns
// included) and row y of population set src; a link through a wall gives the
// node's own reversed population.
template <typename Real>
__device__ __forceinline__ void pull9(const Real* __restrict__ src, int P, int pitch, int ny,
                                      bool walls, int x, int y, Real (&v)[9])
{
    const int o = y * pitch + x + kXOff;
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const int om = y == 0 ? o + (ny - 1) * pitch : o - pitch;       // row below
    const int op = y == ny - 1 ? o - (ny - 1) * pitch : o + pitch;  // row above
    v[0] = src[o];
    v[1] = src[P + o - 1];
    v[2] = src[2 * P + o + 1];
    v[3] = src[blo ? 4 * P + o : 3 * P + om];
    v[4] = src[bhi ? 3 * P + o : 4 * P + op];
    v[5] = src[blo ? 6 * P + o : 5 * P + om - 1];
    v[6] = src[bhi ? 5 * P + o : 6 * P + op + 1];
    v[7] = src[blo ? 8 * P + o : 7 * P + om + 1];
    v[8] = src[bhi ? 7 * P + o : 8 * P + op - 1];
}

// The same from a step's result in shared memory: planes of SP values, rows of 32
// columns, the node at o; its neighbours are in the array.
__device__ __forceinline__ void pull_shared(const float* s, int SP, int o, bool blo, bool bhi,
                                            float (&v)[9])
{
    const int om = o - kTX, op = o + kTX;
    v[0] = s[o];
    v[1] = s[SP + o - 1];
    v[2] = s[2 * SP + o + 1];
    v[3] = s[blo ? 4 * SP + o : 3 * SP + om];
    v[4] = s[bhi ? 3 * SP + o : 4 * SP + op];
    v[5] = s[blo ? 6 * SP + o : 5 * SP + om - 1];
    v[6] = s[bhi ? 5 * SP + o : 6 * SP + op + 1];
    v[7] = s[blo ? 8 * SP + o : 7 * SP + om + 1];
    v[8] = s[bhi ? 7 * SP + o : 8 * SP + op - 1];
}

// Store one value of a plane at offset o and its periodic ghost copies:
// logical columns 0, 1 also at nx, nx + 1 and nx - 2, nx - 1 also at -2, -1.
template <typename Real>
__device__ __forceinline__ void store_ghosts(Real* __restrict__ p, int o, int x, int nx, Real v)
{
    p[o] = v;
    if (x < 2) p[o + nx] = v;
    if (x >= nx - 2) p[o - nx] = v;
}

// Position k of the one-node halo of w x h nodes (w at most 32), relative to the
// first one: the two rows, then the two columns; false if there is none.
__device__ __forceinline__ bool halo_at(int k, int w, int h, int& hx, int& hy)
{
    if (k < 2 * kPW) {
        const bool low = k < kPW;
        hx = (low ? k : k - kPW) - 1;
        hy = low ? -1 : h;
        return hx <= w;
    }
    k -= 2 * kPW;
    hx = (k & 1) ? w : -1;
    hy = k >> 1;
    return hy < h;
}

// FP64: the scaled derivatives (see collide64) of the node whose scaled phi is
// *r0, from the phi array around it (ghost rows: DomDesc::wet_k).
__device__ __forceinline__ void deriv64(const Node64& C, const DomDesc& D, const double* r0,
                                        bool blo, bool bhi, const double* wet, double& X,
                                        double& Y, double& L)
{
    struct Row {
        double k, h, m;
    };
    auto row_of = [&](const double* r) {
        Row v;
        v.k = LB64_SUB(r[1], r[-1]);
        v.h = LB64_ADD(r[1], r[-1]);
        v.m = __fma_rn(C.four, r[0], v.h);
        return v;
    };
    const Row cur = row_of(r0);
    Row up = cur, dn = cur;
    if (!bhi) up = row_of(r0 + kPW);
    if (!blo) dn = row_of(r0 - kPW);
    if (blo) {
        const Row& v = D.wet_k == 2 ? up : cur;
        dn.k = v.k;
        dn.m = __dsub_rn(v.m, ghost_shift64(C.sig, D.wet_k, wet[0]));
    }
    if (bhi) {
        const Row& v = D.wet_k == 2 ? dn : cur;
        up.k = v.k;
        up.m = __dsub_rn(v.m, ghost_shift64(C.sig, D.wet_k, wet[1]));
    }
    X = __fma_rn(C.four, cur.k, LB64_ADD(up.k, dn.k));
    Y = LB64_SUB(up.m, dn.m);
    L = __fma_rn(C.m20, r0[0], __fma_rn(C.four, cur.h, LB64_ADD(up.m, dn.m)));
}

// FP32: the derivatives of the node whose phi is c = *r0.
__device__ __forceinline__ void deriv32(const DomDesc& D, const float* r0, float c, bool blo,
                                        bool bhi, const float* wet, float& dx, float& dy,
                                        float& lap)
{
    float n[3], s[3];
    // the row of a ghost row's phi: row k - 1 (ny - k), see DomDesc::wet_k
    const float* gp = bhi ? r0 - (D.wet_k - 1) * kPW : r0 + kPW;
    const float* gm = blo ? r0 + (D.wet_k - 1) * kPW : r0 - kPW;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        n[j] = gp[j - 1];
        s[j] = gm[j - 1];
    }
    if (bhi) {
        const float h2 = float(D.wet_k) * wet[1];
#pragma unroll
        for (int j = 0; j < 3; ++j) n[j] = n[j] - h2;
    }
    if (blo) {
        const float h2 = float(D.wet_k) * wet[0];
#pragma unroll
        for (int j = 0; j < 3; ++j) s[j] = s[j] - h2;
    }
    stencils<float>(c, r0[1], r0[-1], n[1], s[1], n[2], n[0], s[2], s[0], dx, dy, lap);
}

// FP64.  blockDim.x = 32 TY (every thread has at most a node of its own); phi,
// scaled for the stencils (lb_step64.cuh): (TY + 2) x 34 values of shared memory.
template <bool MRT>
__device__ __forceinline__ void small_step64(const DomDesc& D, int parity, const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double* ph = reinterpret_cast<double*>(smem);
    __shared__ Node64 C;
    __shared__ double wet[2];  // wetting gradients, bottom and top
    const int TY = int(blockDim.x) / kTX;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const double* __restrict__ fs = static_cast<const double*>(parity ? D.f[1] : D.f[0]);
    const double* __restrict__ gs = static_cast<const double*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x), tx = tid % kTX, ty = tid / kTX;
    const int x = T.x0 + tx, y = T.y0 + ty;
    const bool live = tx < T.wc && ty < T.hc;
    // all loads of the thread's node and of its halo position
    double f[9], g[9], gh[9];
    int hx = 0, hy = 0;
    const int nh = 2 * kPW + 2 * TY;
    int k = int(blockDim.x) - 1 - tid;
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    auto inside = [&](int r) { return !walls || (r >= 0 && r < ny); };
    bool halo = k < nh && halo_at(k, T.wc, T.hc, hx, hy) && inside(T.y0 + hy);
    if (live) pull9<double>(gs, P, pitch, ny, walls, x, y, g);
    if (halo) pull9<double>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    if (live) pull9<double>(fs, P, pitch, ny, walls, x, y, f);
    // the wetting gradients, in flight with the populations
    const double wv = tid == 0 ? wet_bottom<double>(D) : (tid == 1 ? wet_top<double>(D) : 0.0);
    load_node64(C, D.c64, tid);
    __syncthreads();
    Phi64 s;
    double c = 0.0;
    if (live) {
        c = phi64(C, g, s);
        ph[(ty + 1) * kPW + tx + 1] = LB64_MUL(C.sig, c);
    }
    for (;;) {
        if (halo) ph[(hy + 1) * kPW + hx + 1] = LB64_MUL(C.sig, phi64(C, gh));
        k += int(blockDim.x);
        if (k >= nh) break;
        halo = halo_at(k, T.wc, T.hc, hx, hy) && inside(T.y0 + hy);
        if (halo) pull9<double>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    }
    if (tid < 2) wet[tid] = wv;
    __syncthreads();
    if (!live) return;
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const bool s2 = D.step2 && (blo || bhi);
    const double* r0 = ph + (ty + 1) * kPW + tx + 1;
    double fo[9], go[9];
    double X, Y, L;
    deriv64(C, D, r0, blo, bhi, wet, X, Y, L);
    collide64<MRT>(C, f, c, s, X, Y, L, s2, D.step2_relax_j != 0,
                   [&](double (&v)[9]) {
#pragma unroll
                       for (int i = 0; i < 9; ++i) v[i] = g[i];
                   },
                   fo, go);
    double* __restrict__ fd = static_cast<double*>(parity ? D.f[0] : D.f[1]);
    double* __restrict__ gd = static_cast<double*>(parity ? D.g[0] : D.g[1]);
    const int o = y * pitch + x + kXOff;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        store_ghosts(fd + i * P, o, x, nx, fo[i]);
        store_ghosts(gd + i * P, o, x, nx, go[i]);
    }
}

// FP64, two threads per node.  A warp's FP64 operation keeps the pipe of its
// scheduler for 64 cycles, so a lattice with fewer warps of nodes than the GPU
// has schedulers waits for one warp's 140 operations in series.  Here a warp
// pulls f of 32 nodes and forms the new f, another pulls g and forms the new g;
// phi, rho - 1 and rho u pass through shared memory.  The two do u and the
// derivatives each for itself, so with warps enough for every scheduler one
// thread per node is faster (lb_api.cu, small_rows).  100 x 50 6.60 -> 5.16 us a
// step, BGK 6.86 -> 5.42; 128 x 96 6.66 -> 5.84.
// blockDim.x = 64 TY: the f warps first.  Shared memory: phi as above, then the
// exchanged values.
template <bool MRT>
__device__ __forceinline__ void small_split64(const DomDesc& D, int parity, const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double* ph = reinterpret_cast<double*>(smem);
    __shared__ Node64 C;
    __shared__ double wet[2];  // wetting gradients, bottom and top
    const int half = int(blockDim.x) / 2, TY = half / kTX;
    double* ex = ph + (TY + 2) * kPW;  // drho, jx, jy, phi: ex[i * half + node]
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const double* __restrict__ fs = static_cast<const double*>(parity ? D.f[1] : D.f[0]);
    const double* __restrict__ gs = static_cast<const double*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x);
    const bool is_g = tid >= half;
    const int node = is_g ? tid - half : tid, tx = node % kTX, ty = node / kTX;
    const int x = T.x0 + tx, y = T.y0 + ty;
    const bool live = tx < T.wc && ty < T.hc;
    // all loads of the thread's half node and of its halo position
    double v[9], gh[9];
    int hx = 0, hy = 0;
    const int nh = 2 * kPW + 2 * TY;
    int k = int(blockDim.x) - 1 - tid;
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    auto inside = [&](int r) { return !walls || (r >= 0 && r < ny); };
    bool halo = k < nh && halo_at(k, T.wc, T.hc, hx, hy) && inside(T.y0 + hy);
    if (live) pull9<double>(is_g ? gs : fs, P, pitch, ny, walls, x, y, v);
    if (halo) pull9<double>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    const double wv =
        tid == 0 ? wet_bottom<double>(D) : (tid == 1 ? wet_top<double>(D) : 0.0);
    load_node64(C, D.c64, tid);
    __syncthreads();
    double c = 0.0;
    Moments64 m;
    Phi64 s;
    if (live) {
        if (is_g) {
            c = phi64(C, v, s);
            ph[(ty + 1) * kPW + tx + 1] = LB64_MUL(C.sig, c);
            ex[3 * half + node] = c;
        } else {
            sums64(C, v, m);
            ex[node] = m.drho;
            ex[half + node] = m.jx;
            ex[2 * half + node] = m.jy;
        }
    }
    for (;;) {
        if (halo) ph[(hy + 1) * kPW + hx + 1] = LB64_MUL(C.sig, phi64(C, gh));
        k += int(blockDim.x);
        if (k >= nh) break;
        halo = halo_at(k, T.wc, T.hc, hx, hy) && inside(T.y0 + hy);
        if (halo) pull9<double>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    }
    if (tid < 2) wet[tid] = wv;
    __syncthreads();
    if (!live) return;
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const bool s2 = D.step2 && (blo || bhi);
    const double* r0 = ph + (ty + 1) * kPW + tx + 1;
    const int o = y * pitch + x + kXOff;
    double X, Y, L, out[9];
    if (is_g) {
        m.drho = ex[node];
        m.jx = ex[half + node];
        m.jy = ex[2 * half + node];
        velocity64(C, c, s2, m);
        deriv64(C, D, r0, blo, bhi, wet, X, Y, L);
        collide_g64(C, m, c, LB64_MUL(c, c), s, L,
                    [&](double (&g)[9]) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) g[i] = v[i];
                    },
                    out);
    } else {
        c = ex[3 * half + node];
        velocity64(C, c, s2, m);
        deriv64(C, D, r0, blo, bhi, wet, X, Y, L);
        collide_f64<MRT>(C, v, m, c, LB64_MUL(c, c), X, Y, L, s2, D.step2_relax_j != 0, out);
    }
    double* __restrict__ dst = static_cast<double*>(is_g ? (parity ? D.g[0] : D.g[1])
                                                         : (parity ? D.f[0] : D.f[1]));
#pragma unroll
    for (int i = 0; i < 9; ++i) store_ghosts(dst + i * P, o, x, nx, out[i]);
}

// FP32 full storage, K steps.  A launch and the loads and stores at its
// ends are 1.5 us of the 2.4 us a step of a small lattice takes, and are paid
// once for K steps here.  The region of a CTA is its tile and E = 2 (K - 1)
// nodes around it, a thread per node: 32 columns x TY + 2 E rows.  The first
// step is done on the region, from phi of the region and one node around it;
// its f and g go to shared memory, from which phi of the region less one node
// and the next step on the region less two nodes follow, and so on down to the
// tile.  blockDim.x = 32 (TY + 2 E), 96 at least.  Shared memory: phi,
// (TY + 2 E + 2) x 34; for K > 1 f and g, 18 x blockDim.x.
// PRM_SMEM (a batch): the node parameters are read from shared memory at each
// use, as in the staged batch kernel, which keeps the bits of its BGK collision
// (the compiler fuses other products there than with parameters in registers).
template <bool MRT, bool PRM_SMEM>
__device__ __forceinline__ void small_steps(const DomDesc& D, int parity, int K, const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float wet[2];  // wetting gradients, bottom and top
    __shared__ NodeParams<float> tile_prm;  // PRM_SMEM only
    float* ph = reinterpret_cast<float*>(smem);
    const int RH = int(blockDim.x) / kTX;  // rows of a full region
    float* F = ph + (RH + 2) * kPW;
    const int SP = int(blockDim.x);  // plane stride of F and G
    float* G = F + 9 * SP;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const float* __restrict__ fs = static_cast<const float*>(parity ? D.f[1] : D.f[0]);
    const float* __restrict__ gs = static_cast<const float*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x), i = tid % kTX, j = tid / kTX;
    const int E = 2 * (K - 1), xr = T.x0 - E, yr = T.y0 - E;
    const int rw = T.wc + 2 * E, rh = T.hc + 2 * E;  // the region
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    // K = 1 stays within the ghost columns
    auto col = [&](int c) { return K == 1 ? c : (c < 0 ? c + nx : (c >= nx ? c - nx : c)); };
    auto inside = [&](int r) { return !walls || (r >= 0 && r < ny); };
    const int x = xr + i, yl = yr + j, y = row(yl);
    const bool live = i < rw && j < rh && inside(yl);
    int hx, hy;
    const bool halo = halo_at(SP - 1 - tid, rw, rh, hx, hy) && inside(yr + hy);
    float f[9], g[9], gh[9];
    if (live) pull9<float>(gs, P, pitch, ny, walls, col(x), y, g);
    if (halo) pull9<float>(gs, P, pitch, ny, walls, col(xr + hx), row(yr + hy), gh);
    if (live) pull9<float>(fs, P, pitch, ny, walls, col(x), y, f);
    const float wv = tid == 0 ? wet_bottom<float>(D) : (tid == 1 ? wet_top<float>(D) : 0.f);
    float* r0 = ph + (j + 1) * kPW + i + 1;
    float c = 0.f;
    if (live) *r0 = c = phi_sum<float>(g);
    if (halo) ph[(hy + 1) * kPW + hx + 1] = phi_sum<float>(gh);
    if (tid < 2) wet[tid] = wv;
    if (PRM_SMEM && tid == 0) tile_prm = node_params<float>(D);
    __syncthreads();
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const bool s2 = D.step2 && (blo || bhi);
    const NodeParams<float> prm = node_params<float>(D);
    float fo[9], go[9];
    bool on = live;
#pragma unroll 1
    for (int m = 1;; m += 2) {
        if (on) {
            float dx, dy, lap;
            deriv32(D, r0, c, blo, bhi, wet, dx, dy, lap);
            if constexpr (PRM_SMEM) {
                const volatile NodeParams<float>& PV = tile_prm;
                collide<float, MRT>(PV, f, g, c, dx, dy, lap, s2, D.step2_relax_j != 0, fo, go);
            } else {
                collide<float, MRT>(prm, f, g, c, dx, dy, lap, s2, D.step2_relax_j != 0, fo, go);
            }
        }
        if (m > E) break;
        if (on) {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                F[q * SP + tid] = fo[q];
                G[q * SP + tid] = go[q];
            }
        }
        __syncthreads();
        on = live && i >= m && i < rw - m && j >= m && j < rh - m;
        if (on) {
            pull_shared(G, SP, tid, blo, bhi, g);
            *r0 = c = phi_sum<float>(g);
        }
        on = on && i > m && i < rw - m - 1 && j > m && j < rh - m - 1;
        if (on) pull_shared(F, SP, tid, blo, bhi, f);
        __syncthreads();
    }
    if (!on) return;
    float* __restrict__ fd = static_cast<float*>(parity ? D.f[0] : D.f[1]);
    float* __restrict__ gd = static_cast<float*>(parity ? D.g[0] : D.g[1]);
    const int o = y * pitch + x + kXOff;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        store_ghosts(fd + q * P, o, x, nx, fo[q]);
        store_ghosts(gd + q * P, o, x, nx, go[q]);
    }
}

// Compact g storage.  Shared memory: nine values (g'_1..g'_8 and their sum)
// and the phi word of (TY + 4) x 36 positions, then phi of (TY + 2) x 34.
// K steps as in small_steps: the first one from the compact values of the region
// and two nodes around it, the others from the values of the step before, which
// each thread expands for its own node.  blockDim.x = 32 (TY + 2 E); for K > 1
// f of a step follows in shared memory, 9 x blockDim.x.
// AHEAD: a thread's first two positions are loaded before either is expanded (us a
// step: 28 x 15 1.87 -> 1.78, 200 x 100 2.32 -> 2.22, 300 x 100 2.66 -> 2.51, 6 domains
// of 22 k nodes 3.9 -> 3.8; but single steps of larger lattices, which are not bound by
// latency alone, 512 x 256 5.84 -> 5.92, without).
template <bool MRT, bool AHEAD>
__device__ __forceinline__ void small_compact_steps(const DomDesc& D, int parity, int K,
                                                    const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int SP = int(blockDim.x), RH = SP / kTX;
    const int ne = (RH + 4) * kEW;
    float* E = reinterpret_cast<float*>(smem);  // E[i * ne + position], i = 0: the sum, 9: the word
    float* ph = E + 10 * ne;
    float* F = ph + (RH + 2) * kPW;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const float* __restrict__ fs = static_cast<const float*>(parity ? D.f[1] : D.f[0]);
    const float* __restrict__ cs = static_cast<const float*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x), i = tid % kTX, j = tid / kTX;
    const int rim = 2 * (K - 1), xr = T.x0 - rim, yr = T.y0 - rim;
    const int rw = T.wc + 2 * rim, rh = T.hc + 2 * rim;  // the region
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    auto col = [&](int c) { return K == 1 ? c : (c < 0 ? c + nx : (c >= nx ? c - nx : c)); };
    auto inside = [&](int r) { return !walls || (r >= 0 && r < ny); };
    const int x = xr + i, yl = yr + j, y = row(yl);
    const bool live = i < rw && j < rh && inside(yl);
    const NodeParams<float> prm = node_params<float>(D);
    float f[9];
    if (live) pull9<float>(fs, P, pitch, ny, walls, col(x), y, f);
    __shared__ float wet[2];  // wetting gradients, bottom and top
    const float wv = tid == 0 ? wet_bottom<float>(D) : (tid == 1 ? wet_top<float>(D) : 0.f);
    auto expand = [&](int k, f2 word, f2 G, f2 ux, f2 uy) {
        f2 ge[9];
        g_equilibria2(g0_value2(word), G, ux, uy, ge);
        E[k] = g_tail_sum2(ge).lane(0);
#pragma unroll
        for (int q = 1; q < 9; ++q) E[q * ne + k] = ge[q].lane(0);
        E[9 * ne + k] = word.lane(0);
    };
    // 1. expand the compact values of the region and two nodes around it
    auto source = [&](int k) -> const float* {
        const int cy = k / kEW, cx = k - cy * kEW;
        const int r = yr + cy - 2;
        if (k >= ne || cx - 2 > rw + 1 || cy - 2 > rh + 1 || !inside(r)) return nullptr;
        return cs + row(r) * pitch + col(xr + cx - 2) + kXOff;
    };
    int k0 = tid;
    if constexpr (AHEAD) {
        const float* s0 = source(tid);
        const float* s1 = source(tid + SP);
        float v0[4], v1[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (s0) v0[q] = s0[q * P];
            if (s1) v1[q] = s1[q * P];
        }
        if (s0) expand(tid, f2(v0[0]), f2(v0[1]), f2(v0[2]), f2(v0[3]));
        if (s1) expand(tid + SP, f2(v1[0]), f2(v1[1]), f2(v1[2]), f2(v1[3]));
        k0 += 2 * SP;
    }
    for (int k = k0; k < ne; k += SP)
        if (const float* s = source(k)) expand(k, f2(s[0]), f2(s[P]), f2(s[2 * P]), f2(s[3 * P]));
    __syncthreads();
    // 2. phi(t+1) = word + [(U + H) + D - sum] of the region and one node around
    //    it (lb_step_compact.cuh); the node's own word for its store
    auto phi_at = [&](int cx, int cy, f2& word) -> f2 {
        const int q = (cy + 2) * kEW + cx + 2, r = yr + cy;
        auto e = [&](int n, int dx, int dy) { return f2(E[n * ne + q + dy * kEW + dx]); };
        const f2 u = walls && r == 0 ? (e(4, 0, 0) + e(6, 0, 0)) + e(8, 0, 0)
                                     : (e(3, 0, -1) + e(5, -1, -1)) + e(7, 1, -1);
        const f2 h = e(1, -1, 0) + e(2, 1, 0);
        const f2 d = walls && r == ny - 1 ? (e(3, 0, 0) + e(5, 0, 0)) + e(7, 0, 0)
                                          : (e(4, 0, 1) + e(6, 1, 1)) + e(8, -1, 1);
        word = g0_advance2(e(9, 0, 0), ((u + h) + d) - e(0, 0, 0));
        return g0_value2(word);
    };
    f2 word(0.f), c(0.f), dump(0.f);
    float* r0 = ph + (j + 1) * kPW + i + 1;
    if (live) {
        c = phi_at(i, j, word);
        *r0 = c.lane(0);
    }
    for (int k = SP - 1 - tid; k < 2 * kPW + 2 * RH; k += SP) {
        int hx, hy;
        if (!halo_at(k, rw, rh, hx, hy) || !inside(yr + hy)) continue;
        // a periodic halo row is the row across the lattice's edge
        ph[(hy + 1) * kPW + hx + 1] = phi_at(hx, hy, dump).lane(0);
    }
    if (tid < 2) wet[tid] = wv;
    __syncthreads();
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    f2 fo[9], gmu, ux, uy;
    bool on = live;
#pragma unroll 1
    for (int m = 1;; m += 2) {
        // 3. collide
        if (on) {
            const float* gp = bhi ? r0 - (D.wet_k - 1) * kPW : r0 + kPW;
            const float* gm = blo ? r0 + (D.wet_k - 1) * kPW : r0 - kPW;
            f2 n[3], s[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                n[q] = f2(gp[q - 1]);
                s[q] = f2(gm[q - 1]);
            }
            if (bhi) {
                const f2 h(float(D.wet_k) * wet[1]);
#pragma unroll
                for (int q = 0; q < 3; ++q) n[q] = n[q] - h;
            }
            if (blo) {
                const f2 h(float(D.wet_k) * wet[0]);
#pragma unroll
                for (int q = 0; q < 3; ++q) s[q] = s[q] - h;
            }
            f2 dx, dy, lap, fi[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) fi[q] = f2(f[q]);
            stencils2(c, f2(r0[1]), f2(r0[-1]), n[1], s[1], n[2], n[0], s[2], s[0], dx, dy, lap);
            collide_f2<MRT>(prm, fi, c, dx, dy, lap, D.step2 && (blo || bhi),
                            D.step2_relax_j != 0, fo, ux, uy);
            gmu = gamma_mu2(prm, c, lap);
        }
        if (m > rim) break;
        // 4. the next step's g' and f
        if (on) {
            expand((j + 2) * kEW + i + 2, word, gmu, ux, uy);
#pragma unroll
            for (int q = 0; q < 9; ++q) F[q * SP + tid] = fo[q].lane(0);
        }
        __syncthreads();
        on = live && i >= m && i < rw - m && j >= m && j < rh - m;
        if (on) {
            c = phi_at(i, j, word);
            *r0 = c.lane(0);
        }
        on = on && i > m && i < rw - m - 1 && j > m && j < rh - m - 1;
        if (on) pull_shared(F, SP, tid, blo, bhi, f);
        __syncthreads();
    }
    if (!on) return;
    float* __restrict__ fd = static_cast<float*>(parity ? D.f[0] : D.f[1]);
    float* __restrict__ cd = static_cast<float*>(parity ? D.g[0] : D.g[1]);
    const int o = y * pitch + x + kXOff;
#pragma unroll
    for (int q = 0; q < 9; ++q) store_ghosts(fd + q * P, o, x, nx, fo[q].lane(0));
    store_ghosts(cd, o, x, nx, word.lane(0));
    store_ghosts(cd + P, o, x, nx, gmu.lane(0));
    store_ghosts(cd + 2 * P, o, x, nx, ux.lane(0));
    store_ghosts(cd + 3 * P, o, x, nx, uy.lane(0));
}

// How a tile is stored: FP64, FP32, or FP32 with compact g; FP64 on two threads
// per node.
enum class SmallKind { F64, F32, Compact, Split64 };

// threads per row of a tile
__host__ __device__ constexpr int lane_threads(SmallKind k)
{
    return k == SmallKind::Split64 ? 2 * kTX : kTX;
}

template <SmallKind K, bool MRT, bool BATCH>
__device__ __forceinline__ void small_tile(const DomDesc& D, int parity, const SmallTile& T)
{
    if constexpr (K == SmallKind::F64)
        small_step64<MRT>(D, parity, T);
    else if constexpr (K == SmallKind::Split64)
        small_split64<MRT>(D, parity, T);
    else if constexpr (K == SmallKind::F32)
        small_steps<MRT, BATCH>(D, parity, 1, T);
    else
        small_compact_steps<MRT, BATCH>(D, parity, 1, T);
}

template <SmallKind K, bool MRT>
__global__ void __launch_bounds__(kSmallMaxThreads) small_step_kernel(DomDesc D, int parity)
{
    const int ty = int(blockDim.x) / lane_threads(K);
    small_tile<K, MRT, false>(D, parity, SmallTile(D, int(blockIdx.x) * kTX, int(blockIdx.y) * ty, ty));
}

template <bool MRT, bool COMPACT>
__global__ void __launch_bounds__(kStepsMaxThreads)
    small_steps_kernel(DomDesc D, int parity, int K, int rows)
{
    const int w = kTX - 4 * (K - 1);
    SmallTile T(D, int(blockIdx.x) * w, int(blockIdx.y) * rows, rows);
    T.wc = min(T.wc, w);
    if constexpr (COMPACT)
        small_compact_steps<MRT, true>(D, parity, K, T);
    else
        small_steps<MRT, false>(D, parity, K, T);
}

// Batch form: a CTA per work item (a tile of 32 columns x TY rows of one domain).
// The CTA copies the domain's descriptor at once; its fields read from device
// memory one by one cost more registers and waits (40 domains of 623 k nodes FP32
// 27.4 -> 25.0 us a step, 6 of 22 k 3.7 -> 3.3).
template <SmallKind K, bool MRT>
__global__ void __launch_bounds__(kSmallMaxThreads)
    small_batch_kernel(const DomDesc* __restrict__ descs, const WorkItem* __restrict__ items,
                       int parity)
{
    __shared__ DomDesc sd;
    const WorkItem w = items[blockIdx.x];
    static_assert(sizeof(DomDesc) % 8 == 0, "copied in words of eight bytes");
    for (int k = threadIdx.x; k < int(sizeof(DomDesc) / 8); k += blockDim.x)
        reinterpret_cast<double*>(&sd)[k] = reinterpret_cast<const double*>(descs + w.dom)[k];
    __syncthreads();
    const DomDesc& D = sd;
    small_tile<K, MRT, true>(D, parity, SmallTile(D, w.x0, w.y0, int(blockDim.x) / lane_threads(K)));
}

size_t small_smem(SmallKind k, int rows)
{
    const size_t phi = size_t(rows + 2) * kPW;
    if (k == SmallKind::Split64) return (phi + size_t(rows) * kTX * 4) * 8;
    return k == SmallKind::F64 ? phi * 8
                               : (k == SmallKind::F32 ? phi * 4
                                                      : (size_t(rows + 4) * kEW * 10 + phi) * 4);
}

template <SmallKind K, bool MRT>
cudaError_t launch_t(const DomDesc& d, const DomDesc* descs, const WorkItem* items, int n_items,
                     int parity, int rows, cudaStream_t s)
{
    const int threads = lane_threads(K) * rows;
    const size_t smem = small_smem(K, rows);
    if (items)
        small_batch_kernel<K, MRT><<<n_items, threads, smem, s>>>(descs, items, parity);
    else
        small_step_kernel<K, MRT>
            <<<dim3((d.nx + kTX - 1) / kTX, (d.ny + rows - 1) / rows), threads, smem, s>>>(d, parity);
    return cudaGetLastError();
}

template <SmallKind K>
cudaError_t launch_c(int coll, const DomDesc& d, const DomDesc* descs, const WorkItem* items,
                     int n_items, int parity, int rows, cudaStream_t s)
{
    return coll ? launch_t<K, true>(d, descs, items, n_items, parity, rows, s)
                : launch_t<K, false>(d, descs, items, n_items, parity, rows, s);
}

}  // namespace

int launch_small_step(int precision, int coll, const DomDesc& d, const DomDesc* descs,
                      const WorkItem* items, int n_items, int parity, int rows, void* stream)
{
    // FP32 full storage: the threads take the halo in one round (small_steps)
    const int least = precision == 0 && !d.compact ? 3 : 1;
    static_assert(3 * kTX >= 2 * kPW + 2 * 3, "a thread for each position");
    if (rows < least || rows > kSmallMaxThreads / kTX) return int(cudaErrorInvalidValue);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision != 0 && rows <= kSmallSplitRows)
        return int(launch_c<SmallKind::Split64>(coll, d, descs, items, n_items, parity, rows, s));
    if (precision != 0)
        return int(launch_c<SmallKind::F64>(coll, d, descs, items, n_items, parity, rows, s));
    if (d.compact)
        return int(launch_c<SmallKind::Compact>(coll, d, descs, items, n_items, parity, rows, s));
    return int(launch_c<SmallKind::F32>(coll, d, descs, items, n_items, parity, rows, s));
}

namespace {

// The several-step kernel of a storage, and the shared memory of its CTAs.
using StepsKernel = void (*)(DomDesc, int, int, int);
StepsKernel steps_kernel(bool compact, int coll)
{
    return compact ? (coll ? StepsKernel(small_steps_kernel<true, true>)
                           : StepsKernel(small_steps_kernel<false, true>))
                   : (coll ? StepsKernel(small_steps_kernel<true, false>)
                           : StepsKernel(small_steps_kernel<false, false>));
}
size_t steps_smem(bool compact, int threads)
{
    return small_smem(compact ? SmallKind::Compact : SmallKind::F32, threads / kTX) +
           size_t(compact ? 9 : 18) * threads * 4;
}

}  // namespace

// The limit is the process's, not a launch's: the most any launch asks for, the
// same value whoever sets it.
int prepare_small_steps()
{
    for (int k = 0; k < 4; ++k) {
        const bool compact = k & 1;
        const cudaError_t e =
            cudaFuncSetAttribute(steps_kernel(compact, k >> 1),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(steps_smem(compact, kStepsMaxThreads)));
        if (e != cudaSuccess) return int(e);
    }
    return 0;
}

int launch_small_steps(int coll, const DomDesc& d, int parity, int steps, int rows, void* stream)
{
    // a region wraps around the lattice once at most
    if (steps < 2 || small_steps_cols(steps) < 1 || rows < 1 || d.nx < 2 * steps ||
        d.ny < 2 * steps || small_steps_threads(steps, rows) > kStepsMaxThreads)
        return int(cudaErrorInvalidValue);
    const int threads = small_steps_threads(steps, rows), w = small_steps_cols(steps);
    const dim3 grid((d.nx + w - 1) / w, (d.ny + rows - 1) / rows);
    steps_kernel(d.compact != 0, coll)<<<grid, threads, steps_smem(d.compact != 0, threads),
                                         static_cast<cudaStream_t>(stream)>>>(d, parity, steps, rows);
    return int(cudaGetLastError());
}

}  // namespace lbfe

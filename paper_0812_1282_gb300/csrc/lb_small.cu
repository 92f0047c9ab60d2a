// Fused step of small lattices without obstacles: one launch per step, one
// node per thread, plain loads.
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

// Store one value of a plane at offset o and its periodic ghost copies:
// logical columns 0, 1 also at nx, nx + 1 and nx - 2, nx - 1 also at -2, -1.
template <typename Real>
__device__ __forceinline__ void store_ghosts(Real* __restrict__ p, int o, int x, int nx, Real v)
{
    p[o] = v;
    if (x < 2) p[o + nx] = v;
    if (x >= nx - 2) p[o - nx] = v;
}

// Position k of the one-node halo of a tile, relative to its first node;
// false if the tile or the lattice has none there.
__device__ __forceinline__ bool halo_at(int k, const SmallTile& T, bool walls, int ny, int& hx,
                                        int& hy)
{
    if (k < 2 * kPW) {
        const bool low = k < kPW;
        hx = (low ? k : k - kPW) - 1;
        hy = low ? -1 : T.hc;
        return hx <= T.wc && !(walls && (low ? T.y0 == 0 : T.y0 + T.hc == ny));
    }
    k -= 2 * kPW;
    hx = (k & 1) ? T.wc : -1;
    hy = k >> 1;
    return hy < T.hc;
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

// Full storage.  blockDim.x = 32 TY (a multiple of a warp; every thread has
// at most a node of its own); phi: (TY + 2) x 34 values of shared memory.
// PRM_SMEM (FP32, a batch): the node parameters are read from shared memory at
// each use, as in the staged batch kernel, which keeps the bits of its BGK
// collision (the compiler fuses other products there than with parameters in
// registers).
template <typename Real, bool MRT, bool PRM_SMEM>
__device__ __forceinline__ void small_step(const DomDesc& D, int parity, const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Real* ph = reinterpret_cast<Real*>(smem);
    __shared__ Node64 C;     // FP64 only
    __shared__ Real wet[2];  // wetting gradients, bottom and top
    __shared__ NodeParams<Real> tile_prm;  // PRM_SMEM only
    const int TY = int(blockDim.x) / kTX;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const Real* __restrict__ fs = static_cast<const Real*>(parity ? D.f[1] : D.f[0]);
    const Real* __restrict__ gs = static_cast<const Real*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x), tx = tid % kTX, ty = tid / kTX;
    const int x = T.x0 + tx, y = T.y0 + ty;
    const bool live = tx < T.wc && ty < T.hc;
    // all loads of the thread's node and of its halo position
    Real f[9], g[9], gh[9];
    int hx = 0, hy = 0;
    const int nh = 2 * kPW + 2 * TY;
    int k = int(blockDim.x) - 1 - tid;
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    bool halo = k < nh && halo_at(k, T, walls, ny, hx, hy);
    if (live) pull9<Real>(gs, P, pitch, ny, walls, x, y, g);
    if (halo) pull9<Real>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    if (live) pull9<Real>(fs, P, pitch, ny, walls, x, y, f);
    // the wetting gradients, in flight with the populations
    const Real wv = tid == 0 ? wet_bottom<Real>(D) : (tid == 1 ? wet_top<Real>(D) : Real(0));
    if constexpr (sizeof(Real) == 8) {
        load_node64(C, D.c64, tid);
        __syncthreads();
    }
    // the stored value: phi, in FP64 scaled for the stencils (lb_step64.cuh)
    auto put = [&](int cx, int cy, const Real (&v)[9], Real& phi) {
        if constexpr (sizeof(Real) == 8) {
            phi = phi64(C, v);
            ph[(cy + 1) * kPW + cx + 1] = LB64_MUL(C.sig, phi);
        } else {
            phi = phi_sum<Real>(v);
            ph[(cy + 1) * kPW + cx + 1] = phi;
        }
    };
    Real c = Real(0), dump;
    if (live) put(tx, ty, g, c);
    for (;;) {
        if (halo) put(hx, hy, gh, dump);
        k += int(blockDim.x);
        if (k >= nh) break;
        halo = halo_at(k, T, walls, ny, hx, hy);
        if (halo) pull9<Real>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    }
    if (tid < 2) wet[tid] = wv;
    if (PRM_SMEM && tid == 0) tile_prm = node_params<Real>(D);
    __syncthreads();
    if (!live) return;
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const bool s2 = D.step2 && (blo || bhi);
    const Real* r0 = ph + (ty + 1) * kPW + tx + 1;
    Real fo[9], go[9];
    if constexpr (sizeof(Real) == 8) {
        double X, Y, L;
        deriv64(C, D, r0, blo, bhi, wet, X, Y, L);
        collide64<MRT>(C, f, c, X, Y, L, s2, D.step2_relax_j != 0,
                       [&](double (&v)[9]) {
#pragma unroll
                           for (int i = 0; i < 9; ++i) v[i] = g[i];
                       },
                       fo, go);
    } else {
        const NodeParams<Real> prm = node_params<Real>(D);
        Real dx, dy, lap, n[3], s[3];
        // the row of a ghost row's phi: row k - 1 (ny - k), see DomDesc::wet_k
        const Real* gp = bhi ? r0 - (D.wet_k - 1) * kPW : r0 + kPW;
        const Real* gm = blo ? r0 + (D.wet_k - 1) * kPW : r0 - kPW;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            n[j] = gp[j - 1];
            s[j] = gm[j - 1];
        }
        if (bhi) {
            const Real h2 = Real(D.wet_k) * wet[1];
#pragma unroll
            for (int j = 0; j < 3; ++j) n[j] = n[j] - h2;
        }
        if (blo) {
            const Real h2 = Real(D.wet_k) * wet[0];
#pragma unroll
            for (int j = 0; j < 3; ++j) s[j] = s[j] - h2;
        }
        stencils<Real>(c, r0[1], r0[-1], n[1], s[1], n[2], n[0], s[2], s[0], dx, dy, lap);
        if constexpr (PRM_SMEM) {
            const volatile NodeParams<Real>& PV = tile_prm;
            collide<Real, MRT>(PV, f, g, c, dx, dy, lap, s2, D.step2_relax_j != 0, fo, go);
        } else {
            collide<Real, MRT>(prm, f, g, c, dx, dy, lap, s2, D.step2_relax_j != 0, fo, go);
        }
    }
    Real* __restrict__ fd = static_cast<Real*>(parity ? D.f[0] : D.f[1]);
    Real* __restrict__ gd = static_cast<Real*>(parity ? D.g[0] : D.g[1]);
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
    bool halo = k < nh && halo_at(k, T, walls, ny, hx, hy);
    if (live) pull9<double>(is_g ? gs : fs, P, pitch, ny, walls, x, y, v);
    if (halo) pull9<double>(gs, P, pitch, ny, walls, T.x0 + hx, row(T.y0 + hy), gh);
    const double wv =
        tid == 0 ? wet_bottom<double>(D) : (tid == 1 ? wet_top<double>(D) : 0.0);
    load_node64(C, D.c64, tid);
    __syncthreads();
    double c = 0.0;
    Moments64 m;
    if (live) {
        if (is_g) {
            c = phi64(C, v);
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
        halo = halo_at(k, T, walls, ny, hx, hy);
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
        collide_g64(C, m, c, LB64_MUL(c, c), L,
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

// Compact g storage.  Shared memory: nine values (g'_1..g'_8 and their sum)
// and the phi word of (TY + 4) x 36 positions, then phi of (TY + 2) x 34.
template <bool MRT>
__device__ __forceinline__ void small_compact_step(const DomDesc& D, int parity, const SmallTile& T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int TY = int(blockDim.x) / kTX;
    const int ne = (TY + 4) * kEW;
    float* E = reinterpret_cast<float*>(smem);  // E[i * ne + position], i = 0: the sum, 9: the word
    float* ph = E + 10 * ne;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch, P = int(D.plane);
    const bool walls = D.walls != 0;
    const float* __restrict__ fs = static_cast<const float*>(parity ? D.f[1] : D.f[0]);
    const float* __restrict__ cs = static_cast<const float*>(parity ? D.g[1] : D.g[0]);
    const int tid = int(threadIdx.x), tx = tid % kTX, ty = tid / kTX;
    const int x = T.x0 + tx, y = T.y0 + ty;
    const bool live = tx < T.wc && ty < T.hc;
    auto row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    auto inside = [&](int r) { return !walls || (r >= 0 && r < ny); };
    const NodeParams<float> prm = node_params<float>(D);
    float f[9];
    if (live) pull9<float>(fs, P, pitch, ny, walls, x, y, f);
    __shared__ float wet[2];  // wetting gradients, bottom and top
    const float wv = tid == 0 ? wet_bottom<float>(D) : (tid == 1 ? wet_top<float>(D) : 0.f);
    // 1. expand the compact values of the tile and two nodes around it
    for (int k = tid; k < ne; k += int(blockDim.x)) {
        const int cy = k / kEW, cx = k - cy * kEW;
        const int r = T.y0 + cy - 2;
        if (cx - 2 > T.wc + 1 || cy - 2 > T.hc + 1 || !inside(r)) continue;
        const float* s = cs + row(r) * pitch + T.x0 + cx - 2 + kXOff;
        const f2 word(s[0]), G(s[P]), ux(s[2 * P]), uy(s[3 * P]);
        f2 ge[9];
        g_equilibria2(g0_value2(word), G, ux, uy, ge);
        E[k] = g_tail_sum2(ge).lane(0);
#pragma unroll
        for (int i = 1; i < 9; ++i) E[i * ne + k] = ge[i].lane(0);
        E[9 * ne + k] = word.lane(0);
    }
    __syncthreads();
    // 2. phi(t+1) = word + [(U + H) + D - sum] of the tile and one node around
    //    it (lb_step_compact.cuh); the node's own word for its store
    auto phi_at = [&](int cx, int cy, f2& word) -> f2 {
        const int q = (cy + 2) * kEW + cx + 2, r = T.y0 + cy;
        auto e = [&](int i, int dx, int dy) { return f2(E[i * ne + q + dy * kEW + dx]); };
        const f2 u = walls && r == 0 ? (e(4, 0, 0) + e(6, 0, 0)) + e(8, 0, 0)
                                     : (e(3, 0, -1) + e(5, -1, -1)) + e(7, 1, -1);
        const f2 h = e(1, -1, 0) + e(2, 1, 0);
        const f2 d = walls && r == ny - 1 ? (e(3, 0, 0) + e(5, 0, 0)) + e(7, 0, 0)
                                          : (e(4, 0, 1) + e(6, 1, 1)) + e(8, -1, 1);
        word = g0_advance2(e(9, 0, 0), ((u + h) + d) - e(0, 0, 0));
        return g0_value2(word);
    };
    f2 word(0.f), c(0.f), dump(0.f);
    if (live) {
        c = phi_at(tx, ty, word);
        ph[(ty + 1) * kPW + tx + 1] = c.lane(0);
    }
    for (int k = int(blockDim.x) - 1 - tid; k < 2 * kPW + 2 * TY; k += int(blockDim.x)) {
        int hx, hy;
        if (!halo_at(k, T, walls, ny, hx, hy)) continue;
        // a periodic halo row is the row across the lattice's edge
        ph[(hy + 1) * kPW + hx + 1] = phi_at(hx, hy, dump).lane(0);
    }
    if (tid < 2) wet[tid] = wv;
    __syncthreads();
    // 3. collide
    if (!live) return;
    const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
    const float* r0 = ph + (ty + 1) * kPW + tx + 1;
    const float* gp = bhi ? r0 - (D.wet_k - 1) * kPW : r0 + kPW;
    const float* gm = blo ? r0 + (D.wet_k - 1) * kPW : r0 - kPW;
    f2 n[3], s[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        n[j] = f2(gp[j - 1]);
        s[j] = f2(gm[j - 1]);
    }
    if (bhi) {
        const f2 h(float(D.wet_k) * wet[1]);
#pragma unroll
        for (int j = 0; j < 3; ++j) n[j] = n[j] - h;
    }
    if (blo) {
        const f2 h(float(D.wet_k) * wet[0]);
#pragma unroll
        for (int j = 0; j < 3; ++j) s[j] = s[j] - h;
    }
    f2 dx, dy, lap, fi[9], fo[9], ux, uy;
#pragma unroll
    for (int i = 0; i < 9; ++i) fi[i] = f2(f[i]);
    stencils2(c, f2(r0[1]), f2(r0[-1]), n[1], s[1], n[2], n[0], s[2], s[0], dx, dy, lap);
    collide_f2<MRT>(prm, fi, c, dx, dy, lap, D.step2 && (blo || bhi), D.step2_relax_j != 0, fo, ux,
                    uy);
    const f2 gmu = gamma_mu2(prm, c, lap);
    float* __restrict__ fd = static_cast<float*>(parity ? D.f[0] : D.f[1]);
    float* __restrict__ cd = static_cast<float*>(parity ? D.g[0] : D.g[1]);
    const int o = y * pitch + x + kXOff;
#pragma unroll
    for (int i = 0; i < 9; ++i) store_ghosts(fd + i * P, o, x, nx, fo[i].lane(0));
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
        small_step<double, MRT, false>(D, parity, T);
    else if constexpr (K == SmallKind::Split64)
        small_split64<MRT>(D, parity, T);
    else if constexpr (K == SmallKind::F32)
        small_step<float, MRT, BATCH>(D, parity, T);
    else
        small_compact_step<MRT>(D, parity, T);
}

template <SmallKind K, bool MRT>
__global__ void __launch_bounds__(kSmallMaxThreads) small_step_kernel(DomDesc D, int parity)
{
    const int ty = int(blockDim.x) / lane_threads(K);
    small_tile<K, MRT, false>(D, parity, SmallTile(D, int(blockIdx.x) * kTX, int(blockIdx.y) * ty, ty));
}

// Batch form: a CTA per work item (a tile of 32 columns x blockDim.x / 32
// rows of one domain).
template <SmallKind K, bool MRT>
__global__ void __launch_bounds__(kSmallMaxThreads)
    small_batch_kernel(const DomDesc* __restrict__ descs, const WorkItem* __restrict__ items,
                       int parity)
{
    const WorkItem w = items[blockIdx.x];
    const DomDesc& D = descs[w.dom];
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
    if (rows < 1 || rows > kSmallMaxThreads / kTX) return int(cudaErrorInvalidValue);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision != 0 && rows <= kSmallSplitRows)
        return int(launch_c<SmallKind::Split64>(coll, d, descs, items, n_items, parity, rows, s));
    if (precision != 0)
        return int(launch_c<SmallKind::F64>(coll, d, descs, items, n_items, parity, rows, s));
    if (d.compact)
        return int(launch_c<SmallKind::Compact>(coll, d, descs, items, n_items, parity, rows, s));
    return int(launch_c<SmallKind::F32>(coll, d, descs, items, n_items, parity, rows, s));
}

}  // namespace lbfe

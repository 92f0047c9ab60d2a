// Time step of a domain with solid obstacles (capillary filling, Sec. VI).
//
// The paper states bounce-back and the wetting boundary condition for flat
// walls only; on an obstacle map they are read node by node:
//   - a population whose pull source r - e_i is solid is the node's own
//     reversed post-collision population (mid-link bounce-back, as at walls);
//   - Step 2 (zero equilibrium velocity) applies to fluid nodes with a solid
//     node among their eight neighbours;
//   - a solid node s next to fluid carries the wetting ghost value: the
//     flat-wall mirror phi(s + 2d) - 2 h(s) (or, with the one-sided rule,
//     phi(s + d) - h(s)), averaged over the axis directions d whose
//     neighbour s + d is fluid, or over the diagonal directions if s
//     touches fluid only through a corner.  The host rejects
//     maps where a mirror node s + 2d is solid (features thinner than two
//     nodes).  On an obstacle-free lattice this is the ghost-row rule of the
//     plain step, so both paths agree there.
// With walls, the rows y = -1 and y = ny are solid with h_bot / h_top.
//
// Node bounce-back (the paper's Fig. 4b, the wall on the boundary nodes),
// class kNodeWall in row 0 or ny - 1 of a walled domain, read as the
// full-way scheme: a wall node streams like a fluid node (its pulls from
// beyond the domain bounce back) and reverses every population instead of
// colliding; its fluid neighbours see phi(x, 0) = phi(x, 1) - h_bot (phi(x,
// ny-1) = phi(x, ny-2) - h_top) and are Step-2 nodes.
//
// A step is one launch over the tiles that hold a fluid or wall node (a list
// the host makes with the map).  A CTA owns a tile of 32 x TY nodes (one per
// thread) and, in shared memory, the class map of the tile and a four-node
// halo; further warps help with halo positions and ghost values.  Then
//   1. each thread pulls f and g of its node and g of one halo position, and
//      stores the phi of both (Eq. moments).  A tile needs phi on a one-node
//      halo, and a tile with a solid neighbour somewhere on a three-node one:
//      a ghost value reads phi up to two nodes from its solid node;
//   2. in such a tile each solid node on the tile and its one-node halo gets
//      its ghost value, once, into the same phi array;
//   3. each fluid node takes its 3 x 3 phi from shared memory, collides (the
//      node arithmetic of the plain step) and stores.
// Halo nodes are formed by several CTAs with the same arithmetic, so every
// tile sees the same phi.  Solid nodes are never written by a step; they hold
// the rest state (f = t, g = 0), so they carry no fluid.
//
// The obstacle path serves small and medium geometries (the capillary set-up
// is ~10^5 nodes) whose state stays in L2: a step is bound by launch and L2
// latency rather than by HBM bandwidth, so it uses plain loads instead of
// the staged pipeline of the plain step, and one launch with one shared
// phi field instead of a phi pass through memory.  Measured, us per step:
// 1000 x 120 channel FP32 7.6 -> 3.7 (a three-node phi halo in every tile,
// ghost values formed anew for each fluid neighbour, g pulled twice, tiles of
// solid nodes launched; then as above), 2000 x 200 FP32 18 -> 9.8, 401 x 77
// FP64 22 -> 9.0 (with the arithmetic of lb_node64.cuh); a single tile 4.2 ->
// 2.5.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <vector>

#include "lb_async.cuh"
#include "lb_internal.h"
#include "lb_geo_persist.h"
#include "lb_node.cuh"
#include "lb_node64.cuh"
#include "lb_step.cuh"

namespace lbfe {

namespace {

constexpr int kGeoBlock = 128;

template <typename Real>
__device__ __forceinline__ Real class_h(const DomDesc& D, int k);
template <>
__device__ __forceinline__ float class_h<float>(const DomDesc& D, int k)
{
    return D.fhcls[k];
}
template <>
__device__ __forceinline__ double class_h<double>(const DomDesc& D, int k)
{
    return D.hcls[k];
}

// periodic index for offsets of a few nodes (|v| < 2n)
__device__ __forceinline__ int wrap_near(int v, int n)
{
    return v < 0 ? v + n : (v >= n ? v - n : v);
}

// velocity components in the paper's order
__device__ __forceinline__ int gex(int i)
{
    return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 2 || i == 6 || i == 7) ? -1 : 0);
}
__device__ __forceinline__ int gey(int i)
{
    return (i == 3 || i == 5 || i == 7) ? 1 : ((i == 4 || i == 6 || i == 8) ? -1 : 0);
}
__device__ __forceinline__ int gopp(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

struct GeoView {
    const unsigned char* cls;
    int nx, ny, walls;

    // wetting class of (x, y); 0 = fluid, -1 / -2 = the bottom / top wall row
    __device__ __forceinline__ int cls_at(int x, int y) const
    {
        if (walls && y < 0) return -1;
        if (walls && y >= ny) return -2;
        return cls[(long long)wrap_near(y, ny) * nx + wrap_near(x, nx)];
    }
    __device__ __forceinline__ bool solid(int x, int y) const { return cls_at(x, y) != 0; }
};

// Tile of a step and its halos: 32 x TY nodes, one per thread.
constexpr int kGTX = 32;
constexpr int kGH = 3;        // phi halo
constexpr int kGC = kGH + 1;  // class-map halo
constexpr int kGCX = kGTX + 2 * kGC, kGPX = kGTX + 2 * kGH;
// Rows of the multi-step forms' tiles (persistent, two steps); the per-step
// form takes 8 or 4 (GeoTiles).
constexpr int kGTY = 8;

// periodic index for any offset (halos may exceed a small lattice)
__device__ __forceinline__ int wrap_any(int v, int n)
{
    const int r = v % n;
    return r < 0 ? r + n : r;
}

// Constants of a CTA in shared memory: the wall wetting gradients
// (DomDesc::self) and, in FP64, the node constants.  A thread fetches at most
// one early and puts it down when the CTA is about to meet, so that no warp
// waits for the load in between.
template <typename Real>
struct GeoConst {
    Real h_bot, h_top;
    __device__ __forceinline__ Real fetch(const DomDesc& D) const
    {
        const int t = int(threadIdx.x);
        return t == 0 ? D.self->fh_bot : (t == 1 ? D.self->fh_top : Real(0));
    }
    __device__ __forceinline__ void put(Real v)
    {
        if (threadIdx.x < 2) (&h_bot)[threadIdx.x] = v;
    }
};
template <>
struct GeoConst<double> {
    double h_bot, h_top;
    Node64 c;
    __device__ __forceinline__ double fetch(const DomDesc& D) const
    {
        const int t = int(threadIdx.x);
        return t == 0 ? D.self->h_bot
                      : (t == 1 ? D.self->h_top : (t < kNode64 + 2 ? D.c64[t - 2] : 0.0));
    }
    __device__ __forceinline__ void put(double v)
    {
        if (threadIdx.x < kNode64 + 2) (&h_bot)[threadIdx.x] = v;
    }
};
static_assert(offsetof(GeoConst<double>, c) == 2 * sizeof(double), "put() fills it in order");

// Per-CTA tables of a tile: the wrapped halo coordinates and the class map
// with its halo.  They depend only on the geometry, so the persistent form
// builds them once per launch.
template <int TY>
struct GeoTables {
    int colx[kGCX];          // wrapped column (+ kXOff) of each halo column
    int rowo[TY + 2 * kGC];  // offset of each halo row (wrapped row x pitch)
    int rowc[TY + 2 * kGC];  // the same row in the class map (wrapped row x nx)
    signed char cl[TY + 2 * kGC][kGCX];  // 0 fluid, k > 0 solid class k, -1 / -2 wall rows
};

template <typename Real, int TY>
__device__ __forceinline__ void geo_tile_setup(const DomDesc& D, int x0, int y0, GeoTables<TY>& t,
                                               GeoConst<Real>& K)
{
    constexpr int CY = TY + 2 * kGC;
    const Real kv = K.fetch(D);
    const int nx = D.nx, ny = D.ny;
    // periodic wrap of the halo coordinates
    for (int k = threadIdx.x; k < kGCX + CY; k += blockDim.x) {
        if (k < kGCX)
            t.colx[k] = wrap_any(x0 - kGC + k, nx) + kXOff;
        else {
            const int wy = wrap_any(y0 - kGC + (k - kGCX), ny);
            t.rowo[k - kGCX] = wy * D.pitch;
            t.rowc[k - kGCX] = wy * nx;
        }
    }
    __syncthreads();
    // class map (0 fluid, k > 0 solid class k, -1 / -2 bottom / top wall row)
    for (int k = threadIdx.x; k < kGCX * CY; k += blockDim.x) {
        const int cy = k / kGCX, cx = k - cy * kGCX;
        const int y = y0 - kGC + cy;
        int c;
        if (D.walls && y < 0)
            c = -1;
        else if (D.walls && y >= ny)
            c = -2;
        else
            c = D.cls[t.rowc[cy] + (t.colx[cx] - kXOff)];
        t.cl[cy][cx] = static_cast<signed char>(c);
    }
    K.put(kv);
    __syncthreads();
}

// Load of a stored population: through L1, or (L2ONLY, the persistent form,
// whose neighbours rewrite the state within the launch) from L2.
template <bool L2ONLY, typename Real>
__device__ __forceinline__ Real geo_ld(const Real* p)
{
    if constexpr (L2ONLY)
        return __ldcg(p);
    else
        return *p;
}

// Wetting ghost value of the solid node at (x, y), or the one-sided value a
// wall node shows its fluid neighbours; false if no fluid touches it (then
// nothing reads it).  cls(x, y) and phi(x, y) read the class map and phi around
// it; y_lat is its lattice row.  The mean over the axis (or, through a corner
// only, the diagonal) directions d towards fluid of phi(s + k d) - k h, k =
// D.wet_k.
template <typename Real, class ClsF, class PhiF>
__device__ __forceinline__ bool geo_ghost(const DomDesc& D, const GeoConst<Real>& K, int x, int y,
                                          int y_lat, ClsF cls, PhiF phi, Real& value)
{
    const int k = cls(x, y);
    if (k == kNodeWall) {
        value = y_lat == 0 ? phi(x, y + 1) - K.h_bot : phi(x, y - 1) - K.h_top;
        return true;
    }
    const Real h = k == -1 ? K.h_bot : (k == -2 ? K.h_top : class_h<Real>(D, k));
    Real sum = Real(0);
    int n = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int dx = j == 0 ? 1 : (j == 1 ? -1 : 0);
        const int dy = j == 2 ? 1 : (j == 3 ? -1 : 0);
        if (cls(x + dx, y + dy) == 0) {
            sum += phi(x + D.wet_k * dx, y + D.wet_k * dy);
            ++n;
        }
    }
    if (n == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int dx = (j == 0 || j == 3) ? 1 : -1;
            const int dy = (j == 0 || j == 2) ? 1 : -1;
            if (cls(x + dx, y + dy) == 0) {
                sum += phi(x + D.wet_k * dx, y + D.wet_k * dy);
                ++n;
            }
        }
    }
    if (n == 0) return false;
    const Real mean =
        n == 1 ? sum : (n == 2 ? sum * Real(0.5) : (n == 3 ? div_const<3>(sum) : sum * Real(0.25)));
    value = mean - Real(D.wet_k) * h;
    return true;
}

// The parts of a node's phi that its collision wants (FP64).
template <typename Real>
struct GeoPhi {};
template <>
struct GeoPhi<double> : Phi64 {};

// Collision of one fluid node from its pulled f, g, its phi c and the phi of
// its eight neighbours (ghost values at solid ones), directions 1..8 in nb.
template <typename Real, bool MRT>
__device__ __forceinline__ void geo_collide(const DomDesc& D, const GeoConst<Real>& K,
                                            const Real (&f)[9], const Real (&g)[9], Real c,
                                            const GeoPhi<Real>& s, const Real (&nb)[9],
                                            bool step2, Real (&fo)[9], Real (&go)[9])
{
    if constexpr (sizeof(Real) == 8) {
        const Node64& C = K.c;
        // the stencils of Eq. (best) on scaled values (collide64)
        const double p = LB64_SUB(nb[5], nb[6]), q = LB64_SUB(nb[8], nb[7]);
        const double X = __fma_rn(C.four, LB64_SUB(nb[1], nb[2]), LB64_ADD(p, q));
        const double Y = __fma_rn(C.four, LB64_SUB(nb[3], nb[4]), LB64_SUB(p, q));
        const double a = LB64_ADD(LB64_ADD(nb[1], nb[2]), LB64_ADD(nb[3], nb[4]));
        const double d = LB64_ADD(LB64_ADD(nb[5], nb[6]), LB64_ADD(nb[7], nb[8]));
        const double L = __fma_rn(C.m20, c, __fma_rn(C.four, a, d));
        collide64<MRT>(C, f, c, s, LB64_MUL(C.sig, X), LB64_MUL(C.sig, Y), LB64_MUL(C.sig, L),
                       step2, D.step2_relax_j != 0,
                       [&](double (&v)[9]) {
#pragma unroll
                           for (int i = 0; i < 9; ++i) v[i] = g[i];
                       },
                       fo, go);
    } else {
        Real dx, dy, lap;
        // order: centre, E, W, N, S, NE, NW, SE, SW
        stencils<Real>(c, nb[1], nb[2], nb[3], nb[4], nb[5], nb[7], nb[8], nb[6], dx, dy, lap);
        const NodeParams<Real> prm = node_params<Real>(D);
        collide<Real, MRT>(prm, f, g, c, dx, dy, lap, step2, D.step2_relax_j != 0, fo, go);
    }
}

// phi = sum of the pulled g
template <typename Real>
__device__ __forceinline__ Real geo_phi(const GeoConst<Real>& K, const Real (&g)[9], GeoPhi<Real>& s)
{
    if constexpr (sizeof(Real) == 8)
        return phi64(K.c, g, s);
    else
        return phi_sum<Real>(g);
}
template <typename Real>
__device__ __forceinline__ Real geo_phi(const GeoConst<Real>& K, const Real (&g)[9])
{
    GeoPhi<Real> s;
    return geo_phi<Real>(K, g, s);
}

// Halo position k of a tile, relative to its first node: the one-node ring
// first (kRing1 positions), then the ring two and three nodes out (kRing3).
template <int TY>
struct GeoHalo {
    static constexpr int kRing1 = 2 * (kGTX + 2) + 2 * TY;
    static constexpr int kRing3 = 4 * kGPX + 4 * (TY + 2);
    __device__ __forceinline__ static void at(int k, int& dx, int& dy)
    {
        constexpr int W = kGTX + 2;
        if (k < 2 * W) {
            dy = k < W ? -1 : TY;
            dx = (k < W ? k : k - W) - 1;
            return;
        }
        k -= 2 * W;
        if (k < 2 * TY) {
            dx = (k & 1) ? kGTX : -1;
            dy = k >> 1;
            return;
        }
        k -= 2 * TY;
        if (k < 4 * kGPX) {
            const int r = k / kGPX;
            dy = r < 2 ? r - 3 : TY - 1 + r;
            dx = k - r * kGPX - 3;
            return;
        }
        k -= 4 * kGPX;
        dy = (k >> 2) - 1;
        dx = (k & 2) ? kGTX + 1 + (k & 1) : (k & 1) - 3;
    }
};

// What a thread does in a tile, from the class map alone: a launch prepares it,
// its loads' addresses too, while the step before it finishes.  us a step, with the
// class map looked at on the way and as here: 1000 x 120 channel FP32 4.3 -> 3.7,
// 401 x 77 3.5 -> 2.7, 1500 x 100 5.2 -> 4.4, 2000 x 200 10.6 -> 9.8, a single tile
// 3.1 -> 2.5; FP64 401 x 77 9.5 -> 8.9, 1000 x 120 20.7 and 20.8.
struct GeoNode {      // a node whose populations are pulled
    int col[3], row[3];  // offsets of its columns x - 1, x, x + 1 and rows
    unsigned bounce;     // bit i: the source of direction i is solid
};
template <typename Real>
struct GeoGhost {  // a solid node's ghost value (see geo_ghost)
    int at;         // its place in the phi array
    int d[2];       // offsets of the mirror nodes: d[0], -d[0], d[1], -d[1]
    unsigned mask;  // which of the four count; 0: no ghost value
    Real shift;     // k h
    bool wall;      // a node wall: phi(at + d[0]) - shift
};
template <typename Real>
struct GeoPlan {
    int cme;             // class of the thread's own node (1: none)
    bool phi_only;       // a node beyond the lattice whose phi is needed
    bool next_to_solid;  // a neighbour of it is not fluid
    GeoNode own, halo;
    int halo_at;         // place of the halo position in the phi array, -1: none
    GeoGhost<Real> ghost;
};

template <typename Real, int TY, int N>
struct GeoTile {
    static constexpr int S = kGPX;  // row stride of the phi array
    const DomDesc& D;
    const GeoConst<Real>& K;
    const GeoTables<TY>& t;
    int x0, y0;
    bool near;  // the tile holds a fluid node with a solid neighbour
    __device__ __forceinline__ GeoTile(const DomDesc& D_, const GeoConst<Real>& K_,
                                       const GeoTables<TY>& t_, int x0_, int y0_, bool near_)
        : D(D_), K(K_), t(t_), x0(x0_), y0(y0_), near(near_)
    {
    }
    // positions relative to the tile's first node
    __device__ __forceinline__ int cls(int x, int y) const { return t.cl[y + kGC][x + kGC]; }
    __device__ __forceinline__ static int at(int x, int y) { return (y + kGH) * S + x + kGH; }
    __device__ __forceinline__ GeoNode node(int x, int y) const
    {
        GeoNode n;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            n.col[k] = t.colx[x + kGC + k - 1];
            n.row[k] = t.rowo[y + kGC + k - 1];
        }
        n.bounce = 0;
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            const int c = cls(x - gex(i), y - gey(i));
            if (c != 0 && c != kNodeWall) n.bounce |= 1u << i;
        }
        return n;
    }
    // ghost position k of the tile and its one-node halo
    __device__ __forceinline__ GeoGhost<Real> ghost(int k) const
    {
        constexpr int GX = kGTX + 2;
        const int y = k / GX - 1, x = k - (y + 1) * GX - 1;
        GeoGhost<Real> g;
        g.mask = 0;
        if (k >= GX * (TY + 2)) return g;
        const int c = cls(x, y);
        if (c == 0) return g;
        g.at = at(x, y);
        g.wall = c == kNodeWall;
        if (g.wall) {
            const bool bottom = y0 + y == 0;
            g.mask = 1;
            g.d[0] = bottom ? S : -S;
            g.d[1] = 0;
            g.shift = bottom ? K.h_bot : K.h_top;
            return g;
        }
        unsigned axis = 0, diag = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ax = j == 0 ? 1 : (j == 1 ? -1 : 0), ay = j == 2 ? 1 : (j == 3 ? -1 : 0);
            const int bx = (j == 0 || j == 3) ? 1 : -1, by = (j == 0 || j == 2) ? 1 : -1;
            if (cls(x + ax, y + ay) == 0) axis |= 1u << j;
            if (cls(x + bx, y + by) == 0) diag |= 1u << j;
        }
        const int w = D.wet_k;
        g.mask = axis ? axis : diag;
        g.d[0] = axis ? w : w * (S + 1);
        g.d[1] = axis ? w * S : w * (S - 1);
        const Real h = c == -1 ? K.h_bot : (c == -2 ? K.h_top : class_h<Real>(D, c));
        g.shift = Real(w) * h;
        return g;
    }
    __device__ __forceinline__ GeoPlan<Real> plan() const
    {
        GeoPlan<Real> p;
        const int tid = int(threadIdx.x), x = tid % kGTX, y = tid / kGTX;
        const bool has_node = N == kGTX * TY || tid < kGTX * TY;
        p.cme = 1;
        p.phi_only = p.next_to_solid = false;
        if (has_node) {
            if (x0 + x < D.nx && y0 + y < D.ny)
                p.cme = cls(x, y);
            else
                p.phi_only = cls(x, y) == 0;
            p.own = node(x, y);
#pragma unroll
            for (int i = 1; i < 9; ++i)
                p.next_to_solid = p.next_to_solid || (near && cls(x + gex(i), y + gey(i)) != 0);
        }
        p.halo_at = -1;
        if (N - 1 - tid < halo_count()) halo(N - 1 - tid, p.halo, p.halo_at);
        p.ghost.mask = 0;
        if (near) p.ghost = ghost(tid);
        return p;
    }
    __device__ __forceinline__ int halo_count() const
    {
        return GeoHalo<TY>::kRing1 + (near ? GeoHalo<TY>::kRing3 : 0);
    }
    __device__ __forceinline__ void halo(int k, GeoNode& n, int& place) const
    {
        int hx, hy;
        GeoHalo<TY>::at(k, hx, hy);
        place = -1;
        if (cls(hx, hy) != 0) return;
        n = node(hx, hy);
        place = at(hx, hy);
    }
};

// Store a solid node's ghost value from phi around it.
template <typename Real>
__device__ __forceinline__ void geo_put_ghost(const GeoGhost<Real>& g, Real* __restrict__ ph)
{
    if (g.mask == 0) return;
    const Real* c = ph + g.at;
    if (g.wall) {
        ph[g.at] = c[g.d[0]] - g.shift;
        return;
    }
    const Real p[4] = {c[g.d[0]], c[-g.d[0]], c[g.d[1]], c[-g.d[1]]};
    Real sum = Real(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) sum = (g.mask >> j) & 1u ? sum + p[j] : sum;
    const int n = __popc(g.mask);
    const Real mean =
        n == 1 ? sum : (n == 2 ? sum * Real(0.5) : (n == 3 ? div_const<3>(sum) : sum * Real(0.25)));
    ph[g.at] = mean - g.shift;
}

// One time step of a tile.  Every one of the CTA's N threads calls it (it holds
// CTA barriers); those beyond the tile's nodes help with halo positions and
// ghost values.
template <typename Real, bool MRT, int TY, int N, bool L2ONLY>
__device__ __forceinline__ void geo_tile_step(const GeoTile<Real, TY, N>& T,
                                              const GeoPlan<Real>& p, int parity,
                                              Real (&phi)[TY + 2 * kGH][kGPX])
{
    const DomDesc& D = T.D;
    const GeoConst<Real>& K = T.K;
    const long long P = D.plane;
    const Real* fs = static_cast<const Real*>(parity ? D.f[1] : D.f[0]);
    const Real* gs = static_cast<const Real*>(parity ? D.g[1] : D.g[0]);
    Real* ph = &phi[0][0];
    // the nine pulled values of a fluid or wall node; a solid source bounces
    // back (the node's own reversed population), a wall node streams
    auto pull = [&](const Real* src, const GeoNode& n, Real (&v)[9]) {
        const int own = n.row[1] + n.col[1];
        v[0] = geo_ld<L2ONLY>(src + own);
#pragma unroll
        for (int i = 1; i < 9; ++i)
            v[i] = (n.bounce >> i) & 1u
                ? geo_ld<L2ONLY>(src + gopp(i) * P + own)
                : geo_ld<L2ONLY>(src + i * P + (n.row[1 - gey(i)] + n.col[1 - gex(i)]));
    };
    const int tid = int(threadIdx.x), x = tid % kGTX, y = tid / kGTX;
    const bool live = p.cme == 0 || p.cme == kNodeWall;
    // 1. own f and g, and g of halo positions
    Real f[9], g[9];
    if (live) {
        pull(gs, p.own, g);
        pull(fs, p.own, f);
    }
    if (p.halo_at >= 0) {
        Real gh[9];
        pull(gs, p.halo, gh);
        ph[p.halo_at] = geo_phi<Real>(K, gh);
    }
    for (int k = 2 * N - 1 - tid; k < T.halo_count(); k += N) {
        GeoNode n;
        int place;
        T.halo(k, n, place);
        if (place >= 0) {
            Real gh[9];
            pull(gs, n, gh);
            ph[place] = geo_phi<Real>(K, gh);
        }
    }
    // a short last tile's threads beyond the lattice take part in the phi array
    // too: their columns and rows are the wrapped ones
    Real c = Real(0);
    GeoPhi<Real> s;
    if (live) {
        c = geo_phi<Real>(K, g, s);
        ph[T.at(x, y)] = c;
    } else if (p.phi_only) {
        pull(gs, p.own, g);
        ph[T.at(x, y)] = geo_phi<Real>(K, g);
    }
    __syncthreads();
    // 2. ghost values of the solid nodes on the tile and its one-node halo
    if (T.near) {
        geo_put_ghost<Real>(p.ghost, ph);
        for (int k = tid + N; k < (kGTX + 2) * (TY + 2); k += N) geo_put_ghost<Real>(T.ghost(k), ph);
        __syncthreads();
    }
    // 3. the tile's fluid and wall nodes
    if (!live) return;
    Real fo[9], go[9];
    if (p.cme == kNodeWall) {
        // node bounce-back: every population reversed, no collision
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            fo[i] = f[gopp(i)];
            go[i] = g[gopp(i)];
        }
    } else {
        Real nb[9];
#pragma unroll
        for (int i = 1; i < 9; ++i) nb[i] = ph[T.at(x + gex(i), y + gey(i))];
        geo_collide<Real, MRT>(D, K, f, g, c, s, nb, D.step2 != 0 && p.next_to_solid, fo, go);
    }
    Real* fd = static_cast<Real*>(parity ? D.f[0] : D.f[1]);
    Real* gd = static_cast<Real*>(parity ? D.g[0] : D.g[1]);
    const int o = p.own.row[1] + p.own.col[1];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        fd[i * P + o] = fo[i];
        gd[i * P + o] = go[i];
    }
}

// Programmatic dependent launch of the per-step kernel: once every CTA of
// one step's grid has started, the next step's grid (launched with
// programmatic stream serialisation) may be scheduled; its CTAs build their
// tables from the static class map, then wait until the previous grid has
// finished and its writes are visible before they touch the state.  The
// next launch and its set-up so overlap the tail of this one.
__device__ __forceinline__ void pdl_allow_next()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// CTAs per SM the registers of a form leave room for: two and three where the
// tiles come to that (geo_extra_warps), eight where they fill the GPU (2000 x 200
// FP32 9.8 us a step, with seven 10.2, without a limit 11.7); FP64 has all the
// registers it wants.
constexpr int geo_min_ctas(bool fp64, int xw)
{
    return fp64 ? 1 : (xw == 3 ? 2 : (xw == 1 ? 3 : 8));
}

// tiles: the domain's list (make_geo_tiles).  XW warps beyond those of the nodes
// (see geo_extra_warps).
template <typename Real, bool MRT, int TY, int XW>
__global__ void __launch_bounds__(kGTX * (TY + XW), geo_min_ctas(sizeof(Real) == 8, XW))
    geo_step_kernel(DomDesc D, int parity, const int* __restrict__ tiles)
{
    __shared__ GeoTables<TY> t;
    __shared__ Real ph[TY + 2 * kGH][kGPX];
    __shared__ GeoConst<Real> K;
    pdl_allow_next();
    const int e = tiles[blockIdx.x], ntx = (D.nx + kGTX - 1) / kGTX;
    const int q = e & kGeoTileIndex;
    const int x0 = q % ntx * kGTX, y0 = q / ntx * TY;
    geo_tile_setup<Real, TY>(D, x0, y0, t, K);
    const GeoTile<Real, TY, kGTX * (TY + XW)> T(D, K, t, x0, y0, e < 0);
    const GeoPlan<Real> plan = T.plan();
    pdl_wait_prev();
    geo_tile_step<Real, MRT, TY, kGTX * (TY + XW), false>(T, plan, parity, ph);
}

// Two steps per launch (temporal blocking; the state stays in L2, so a step
// is bound by latency, and a launch costs about as much as a step): a CTA
// computes step t on its tile and a kFH-node halo into shared memory, then
// step t + 1 on the tile from there.  Step t + 1 pulls one node beyond the
// tile and takes phi three nodes beyond it, whose g pulls reach one more:
// kFH = 4.  Step t then needs phi of the state at t kFH + kGH nodes beyond
// the tile and the class map one node further.  Halo nodes are computed by
// several CTAs with the same arithmetic (geo_node_update), so the result is
// bit-identical to two single steps.  Reads buffer `parity` and writes the
// other one, which therefore holds step t + 2: the launch flips the handle's
// buffer once.
constexpr int kFH = 4;            // step-t output halo
constexpr int kFP = kFH + kGH;    // phi halo of the state at t
constexpr int kFC = kFP + 1;      // class-map halo
constexpr int kFCX = kGTX + 2 * kFC, kFCY = kGTY + 2 * kFC;
constexpr int kFPX = kGTX + 2 * kFP, kFPY = kGTY + 2 * kFP;
constexpr int kFAX = kGTX + 2 * kFH, kFAY = kGTY + 2 * kFH;


// The step of one fluid or wall node (x, y) of class cme from its pulled
// populations f, g: cls_l(x, y) reads the class map and phi_l(x, y) phi of
// the same state around the node (lattice coordinates; ghost values at solid
// neighbours are formed on the way and reach three nodes away).
template <typename Real, bool MRT, class ClsF, class PhiF>
__device__ __forceinline__ void geo_node_update(const DomDesc& D, const GeoConst<Real>& K, int x,
                                                int y, int cme, const Real (&f)[9],
                                                const Real (&g)[9], ClsF cls_l, PhiF phi_l,
                                                Real (&fo)[9], Real (&go)[9])
{
    if (cme == kNodeWall) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            fo[i] = f[gopp(i)];
            go[i] = g[gopp(i)];
        }
        return;
    }
    Real nb[9];
    bool next_to_solid = false;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const int qx = x + gex(i), qy = y + gey(i);
        if (cls_l(qx, qy) != 0) {
            next_to_solid = true;
            geo_ghost<Real>(D, K, qx, qy, qy, cls_l, phi_l, nb[i]);
        } else {
            nb[i] = phi_l(qx, qy);
        }
    }
    GeoPhi<Real> s;
    const Real c = geo_phi<Real>(K, g, s);
    geo_collide<Real, MRT>(D, K, f, g, c, s, nb, D.step2 != 0 && next_to_solid, fo, go);
}

template <typename Real>
struct GeoFused {
    Real fa[9][kFAY][kFAX];  // step-t output on the tile and its kFH halo
    Real ga[9][kFAY][kFAX];
    Real ph0[kFPY][kFPX];    // phi of the state at t
    Real ph1[kGTY + 2 * kGH][kGPX];  // phi of the state at t + 1
    GeoConst<Real> K;
    int colx[kFCX];
    int rowo[kFCY];
    int rowc[kFCY];
    signed char cl[kFCY][kFCX];
};

template <typename Real, bool MRT>
__global__ void __launch_bounds__(kGTX * kGTY, sizeof(Real) == 4 ? 4 : 2)
    geo_step2_kernel(DomDesc D, int parity)
{
    extern __shared__ __align__(16) unsigned char geo_smem[];
    GeoFused<Real>& S = *reinterpret_cast<GeoFused<Real>*>(geo_smem);
    const int x0 = blockIdx.x * kGTX, y0 = blockIdx.y * kGTY;
    const int nx = D.nx, ny = D.ny;
    const int tid = int(threadIdx.x), nthr = int(blockDim.x);
    S.K.put(S.K.fetch(D));
    // 0. wrapped halo coordinates and the class map on the tile + kFC
    for (int k = tid; k < kFCX + kFCY; k += nthr) {
        if (k < kFCX)
            S.colx[k] = wrap_any(x0 - kFC + k, nx) + kXOff;
        else {
            const int wy = wrap_any(y0 - kFC + (k - kFCX), ny);
            S.rowo[k - kFCX] = wy * D.pitch;
            S.rowc[k - kFCX] = wy * nx;
        }
    }
    __syncthreads();
    for (int k = tid; k < kFCX * kFCY; k += nthr) {
        const int cy = k / kFCX, cx = k - cy * kFCX;
        const int y = y0 - kFC + cy;
        int c;
        if (D.walls && y < 0)
            c = -1;
        else if (D.walls && y >= ny)
            c = -2;
        else
            c = D.cls[S.rowc[cy] + (S.colx[cx] - kXOff)];
        S.cl[cy][cx] = static_cast<signed char>(c);
    }
    __syncthreads();
    auto cls_l = [&](int x, int y) -> int { return S.cl[y - y0 + kFC][x - x0 + kFC]; };
    auto solid_l = [&](int x, int y) {
        const int c = cls_l(x, y);
        return c != 0 && c != kNodeWall;
    };
    auto off_l = [&](int x, int y) -> int { return S.rowo[y - y0 + kFC] + S.colx[x - x0 + kFC]; };
    const long long P = D.plane;
    const Real* fs = static_cast<const Real*>(parity ? D.f[1] : D.f[0]);
    const Real* gs = static_cast<const Real*>(parity ? D.g[1] : D.g[0]);
    // pulls from the state at t (global) and at t + 1 (shared); a solid
    // source bounces back (the node's own reversed population)
    auto pull_g = [&](const Real* src, int x, int y, Real (&v)[9]) {
        const int own = off_l(x, y);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sx = x - gex(i), sy = y - gey(i);
            v[i] = (i != 0 && solid_l(sx, sy)) ? src[gopp(i) * P + own] : src[i * P + off_l(sx, sy)];
        }
    };
    auto pull_s = [&](const Real (&a)[9][kFAY][kFAX], int x, int y, Real (&v)[9]) {
        const int ax = x - x0 + kFH, ay = y - y0 + kFH;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int sx = x - gex(i), sy = y - gey(i);
            v[i] = (i != 0 && solid_l(sx, sy)) ? a[gopp(i)][ay][ax]
                                               : a[i][sy - y0 + kFH][sx - x0 + kFH];
        }
    };
    // 1. phi of the state at t on the tile + kFP (fixed trip counts: the
    // loads of all of a thread's positions can be in flight at once)
    constexpr int kT = kGTX * kGTY;
#pragma unroll
    for (int it = 0; it < (kFPX * kFPY + kT - 1) / kT; ++it) {
        const int k = tid + it * kT;
        if (k >= kFPX * kFPY) break;
        const int py = k / kFPX, px = k - py * kFPX;
        const int x = x0 - kFP + px, y = y0 - kFP + py;
        Real v = Real(0);
        if (cls_l(x, y) == 0) {
            Real g[9];
            pull_g(gs, x, y, g);
            v = geo_phi<Real>(S.K, g);
        }
        S.ph0[py][px] = v;
    }
    __syncthreads();
    auto phi0_l = [&](int x, int y) -> Real { return S.ph0[y - y0 + kFP][x - x0 + kFP]; };
    // 2. step t on the tile + kFH, into shared memory (solid nodes: unused)
#pragma unroll
    for (int it = 0; it < (kFAX * kFAY + kT - 1) / kT; ++it) {
        const int k = tid + it * kT;
        if (k >= kFAX * kFAY) break;
        const int ay = k / kFAX, ax = k - ay * kFAX;
        const int x = x0 - kFH + ax, y = y0 - kFH + ay;
        const int cme = cls_l(x, y);
        if (cme != 0 && cme != kNodeWall) continue;
        Real f[9], g[9], fo[9], go[9];
        pull_g(fs, x, y, f);
        pull_g(gs, x, y, g);
        geo_node_update<Real, MRT>(D, S.K, x, y, cme, f, g, cls_l, phi0_l, fo, go);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            S.fa[i][ay][ax] = fo[i];
            S.ga[i][ay][ax] = go[i];
        }
    }
    __syncthreads();
    // 3. phi of the state at t + 1 on the tile + kGH
#pragma unroll
    for (int it = 0; it < (kGPX * (kGTY + 2 * kGH) + kT - 1) / kT; ++it) {
        const int k = tid + it * kT;
        if (k >= kGPX * (kGTY + 2 * kGH)) break;
        const int py = k / kGPX, px = k - py * kGPX;
        const int x = x0 - kGH + px, y = y0 - kGH + py;
        Real v = Real(0);
        if (cls_l(x, y) == 0) {
            Real g[9];
            pull_s(S.ga, x, y, g);
            v = geo_phi<Real>(S.K, g);
        }
        S.ph1[py][px] = v;
    }
    __syncthreads();
    auto phi1_l = [&](int x, int y) -> Real { return S.ph1[y - y0 + kGH][x - x0 + kGH]; };
    // 4. step t + 1 on the tile, to the other buffer
    const int x = x0 + tid % kGTX, y = y0 + tid / kGTX;
    if (x >= nx || y >= ny) return;
    const int cme = cls_l(x, y);
    if (cme != 0 && cme != kNodeWall) return;
    Real f[9], g[9], fo[9], go[9];
    pull_s(S.fa, x, y, f);
    pull_s(S.ga, x, y, g);
    geo_node_update<Real, MRT>(D, S.K, x, y, cme, f, g, cls_l, phi1_l, fo, go);
    Real* fd = static_cast<Real*>(parity ? D.f[0] : D.f[1]);
    Real* gd = static_cast<Real*>(parity ? D.g[0] : D.g[1]);
    const int o = off_l(x, y);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        fd[i * P + o] = fo[i];
        gd[i * P + o] = go[i];
    }
}

// Persistent multi-step form: a cooperative launch (every tile's CTA
// resident at once) runs n_steps steps, one tile per CTA, step s reading
// buffer parity0 ^ (s & flip).  Instead of a launch boundary per step, a tile
// waits before step s until the tiles under its halo (kGC nodes around it,
// periodic; usually its eight neighbours) have finished step s - 1: once
// they are done with step s - 1 they are also done reading what step s
// overwrites (the halo relation is symmetric).  A tile publishes its steps in
// flags[tile] (steps done in this launch) after a CTA barrier and a fence;
// neighbour data is read from L2 (the state changes within the launch).
// The waits are bounded (flag_wait); a give-up stops the CTA at the next
// step.  done[0] counts finished CTAs; the last one resets it and the flags.
// (FP32: four CTAs per SM, so that a 1000 x 120 capillary's 480 tiles are
// resident at once on 152 SMs.)  The plan is made anew for each step: held across
// the loop it spills (64 registers), as does telling plain tiles apart.  us a step,
// every tile stepping and the solid ones passed over: 1000 x 120 FP32 12.8 and 8.6,
// 401 x 77 FP32 6.3 and 6.0, FP64 13.3 and 13.1 (plan held: 13.1, 6.3, 13.4).
template <typename Real, bool MRT>
__global__ void __launch_bounds__(kGTX * kGTY, sizeof(Real) == 4 ? 4 : 2)
    geo_persist_kernel(DomDesc D, int parity0, int flip, int n_steps, int* flags, int* done)
{
    __shared__ GeoTables<kGTY> t;
    __shared__ Real ph[kGTY + 2 * kGH][kGPX];
    __shared__ GeoConst<Real> K;
    __shared__ int nbr[16];
    __shared__ int n_nbr, stop, last_cta;
    const int ntx = int(gridDim.x), nty = int(gridDim.y);
    const int tx = int(blockIdx.x), ty = int(blockIdx.y), me = ty * ntx + tx;
    const int x0 = tx * kGTX, y0 = ty * kGTY;
    geo_tile_setup<Real, kGTY>(D, x0, y0, t, K);
    if (threadIdx.x == 0) {
        // the tiles under the halo (the wrapped columns and rows of the
        // tables; a short last tile can bring a second tile within reach)
        int cx[4], cy[4], ncx = 0, ncy = 0;
        for (int k = 0; k < kGCX; ++k) {
            const int q = (t.colx[k] - kXOff) / kGTX;
            bool seen = false;
            for (int j = 0; j < ncx; ++j) seen = seen || cx[j] == q;
            if (!seen) cx[ncx++] = q;
        }
        for (int k = 0; k < kGTY + 2 * kGC; ++k) {
            const int y = y0 - kGC + k;
            if (D.walls && (y < 0 || y >= D.ny)) continue;  // wall rows: no data
            const int q = t.rowc[k] / D.nx / kGTY;
            bool seen = false;
            for (int j = 0; j < ncy; ++j) seen = seen || cy[j] == q;
            if (!seen) cy[ncy++] = q;
        }
        int n = 0;
        for (int a = 0; a < ncy; ++a)
            for (int b = 0; b < ncx; ++b) {
                const int q = cy[a] * ntx + cx[b];
                if (q != me) nbr[n++] = q;
            }
        n_nbr = n;
        stop = 0;
    }
    // a tile of solid nodes has nothing to do and nobody to wait for
    const int cme = t.cl[kGC + int(threadIdx.x) / kGTX][kGC + int(threadIdx.x) % kGTX];
    const int any = __syncthreads_or(cme == 0 || cme == kNodeWall);
    if (!any && threadIdx.x == 0) {
        stop = 1;
        st_release_gpu(flags + me, n_steps);
    }
    const GeoTile<Real, kGTY, kGTX * kGTY> T(D, K, t, x0, y0, true);
    for (int s = 0; s < n_steps; ++s) {
        if (s > 0 && int(threadIdx.x) < n_nbr && !flag_wait(flags + nbr[threadIdx.x], s, D.err))
            stop = 1;
        __syncthreads();
        if (stop) break;
        geo_tile_step<Real, MRT, kGTY, kGTX * kGTY, true>(T, T.plan(), parity0 ^ (s & flip), ph);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            st_release_gpu(flags + me, s + 1);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_cta = atomicAdd(done, 1) == ntx * nty - 1;
    }
    __syncthreads();
    if (last_cta) {
        __threadfence();
        for (int k = int(threadIdx.x); k < ntx * nty; k += int(blockDim.x)) flags[k] = 0;
        if (threadIdx.x == 0) done[0] = 0;
        __threadfence();
    }
}

// Initial equilibrium (f = f^eq, g = g^eq of phi0 with rho = 1, u = 0) on
// a domain with obstacles; phi0 in FP64 with row pitch D.pitch.  Solid nodes
// get the rest state.  Reads phi0 only at fluid nodes.
template <typename Real>
__global__ void geo_init_eq_kernel(DomDesc D, const double* __restrict__ phi0, int parity)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx) return;
    Real* fd = static_cast<Real*>(parity ? D.f[1] : D.f[0]);
    Real* gd = static_cast<Real*>(parity ? D.g[1] : D.g[0]);
    const long long P = D.plane;
    const long long o = (long long)y * D.pitch + x + kXOff;
    const GeoView G{D.cls, D.nx, D.ny, D.walls};
    double fe[9], ge[9];
    const int cme = D.cls[(long long)y * D.nx + x];
    if (cme == kNodeWall) {
        // the rest equilibrium of the wall node's wetting phi value
        const int in = y == 0 ? 1 : D.ny - 2;
        const double pw = phi0[(long long)in * D.pitch + x] - (y == 0 ? D.h_bot : D.h_top);
        NodeParams<double> prm{D.a, D.kappa, D.gamma, D.omega_phi, D.tau_c0, D.tau_c1, D.h_bot, D.h_top};
        double m7, m8;
        equilibria<double>(prm, 0.0, pw, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, fe, ge, m7, m8);
        fe[0] = -((((fe[1] + fe[2]) + (fe[3] + fe[4])) + ((fe[5] + fe[6]) + (fe[7] + fe[8]))));
        ge[0] = pw - ((((ge[1] + ge[2]) + (ge[3] + ge[4])) + ((ge[5] + ge[6]) + (ge[7] + ge[8]))));
    } else if (cme != 0) {
        for (int i = 0; i < 9; ++i) fe[i] = ge[i] = 0.0;
    } else {
        // phi0 is laid out with pitch D.pitch; wrap it into a compact view
        auto at = [&](int qx, int qy) -> double {
            return phi0[(long long)wrap_near(qy, D.ny) * D.pitch + wrap_near(qx, D.nx)];
        };
        auto ghost = [&](int qx, int qy) -> double {
            const int k = G.cls_at(qx, qy);
            const double h = k == -1 ? D.h_bot : (k == -2 ? D.h_top : D.hcls[k]);
            double sum = 0.0;
            int n = 0;
            for (int j = 0; j < 4; ++j) {
                const int ddx = j == 0 ? 1 : (j == 1 ? -1 : 0);
                const int ddy = j == 2 ? 1 : (j == 3 ? -1 : 0);
                if (!G.solid(qx + ddx, qy + ddy)) {
                    sum += at(qx + D.wet_k * ddx, qy + D.wet_k * ddy);
                    ++n;
                }
            }
            if (n == 0)
                for (int j = 0; j < 4; ++j) {
                    const int ddx = (j == 0 || j == 3) ? 1 : -1;
                    const int ddy = (j == 0 || j == 2) ? 1 : -1;
                    if (!G.solid(qx + ddx, qy + ddy)) {
                        sum += at(qx + D.wet_k * ddx, qy + D.wet_k * ddy);
                        ++n;
                    }
                }
            const double mean = n == 1 ? sum : (n == 2 ? sum * 0.5 : (n == 3 ? div_const<3>(sum) : sum * 0.25));
            return mean - D.wet_k * h;
        };
        double nb[9];
        for (int i = 1; i < 9; ++i) {
            const int qx = x + gex(i), qy = y + gey(i);
            if (qy >= 0 && qy < D.ny && G.cls_at(qx, qy) == kNodeWall)
                nb[i] = qy == 0 ? at(qx, 1) - D.h_bot : at(qx, D.ny - 2) - D.h_top;
            else
                nb[i] = G.solid(qx, qy) ? ghost(qx, qy) : at(qx, qy);
        }
        const double c = at(x, y);
        double dx, dy, lap, m7, m8;
        stencils<double>(c, nb[1], nb[2], nb[3], nb[4], nb[5], nb[7], nb[8], nb[6], dx, dy, lap);
        NodeParams<double> prm{D.a, D.kappa, D.gamma, D.omega_phi, D.tau_c0, D.tau_c1, D.h_bot, D.h_top};
        equilibria<double>(prm, 0.0, c, 0.0, 0.0, 0.0, 0.0, dx, dy, lap, fe, ge, m7, m8);
        fe[0] = -((((fe[1] + fe[2]) + (fe[3] + fe[4])) + ((fe[5] + fe[6]) + (fe[7] + fe[8]))));
        ge[0] = c - ((((ge[1] + ge[2]) + (ge[3] + ge[4])) + ((ge[5] + ge[6]) + (ge[7] + ge[8]))));
    }
    for (int i = 0; i < 9; ++i) {
        fd[i * P + o] = Real(fe[i]);
        gd[i * P + o] = i == 0 ? G0<Real>::encode(ge[0]) : Real(ge[i]);
    }
}

// Rest state at the solid nodes of buffer b.
template <typename Real>
__global__ void geo_solid_rest_kernel(DomDesc D, int b)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= D.nx || D.cls[(long long)y * D.nx + x] == 0) return;
    Real* fd = static_cast<Real*>(b ? D.f[1] : D.f[0]);
    Real* gd = static_cast<Real*>(b ? D.g[1] : D.g[0]);
    const long long P = D.plane;
    const long long o = (long long)y * D.pitch + x + kXOff;
    for (int i = 0; i < 9; ++i) {
        fd[i * P + o] = Real(0);
        gd[i * P + o] = i == 0 ? G0<Real>::encode(0.0) : Real(0);
    }
}

dim3 geo_grid(const DomDesc& d) { return dim3((d.nx + kGeoBlock - 1) / kGeoBlock, d.ny); }

// A dependent launch, except for FP64 domains of few tiles: the next grid's
// CTAs are placed while this one's still run, some of them two to an SM, and
// there the FP64 pipe of the fullest SM is the bound (401 x 77 channel, about
// one tile per SM: 9.5 us a step without, 20.9 with; 2000 x 200, twelve
// tiles per SM: 58.0 without, 56.2 with; FP32 1000 x 120: 6.4 without, 5.3
// with, before the extra warps).
constexpr int kFewTiles = 1024;

// Warps of a CTA beyond those of its nodes.  A near tile has more halo positions
// (276 with 8 rows, 252 with 4) and possible ghost values (340, 204) than nodes,
// and the second round of a few of them holds up the whole CTA.  Three more warps
// take both in one round, while two such CTAs fit each SM; with more tiles than
// that one more, which saves the second round of the halo.  us a step with none,
// one and three more (before GeoPlan): 1000 x 120 channel (230 tiles) 5.3, 5.1, 4.3; 401 x 77 4.0,
// 3.7, 3.5; 1500 x 100 (356) 5.6, 5.2, 6.8; with 4 rows, whose tiles fill the GPU
// (2000 x 200), none 10.6, two 12.7, three 14.4.  FP64, bound by the pipe: four more while
// each tile has an SM to itself (401 x 77 10.4 -> 9.5), else none (1000 x 120 20.6
// and 22.2).
int geo_extra_warps(bool fp64, int rows, int n_tiles, int sm_count)
{
    if (fp64) return n_tiles <= sm_count ? 4 : 0;
    return rows == 8 ? (n_tiles <= 2 * sm_count ? 3 : 1) : 0;
}

template <typename Real, bool MRT, int TY, int XW>
cudaError_t geo_step_t(const DomDesc& d, int parity, const int* tiles, int n_tiles, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_tiles);
    cfg.blockDim = dim3(kGTX * (TY + XW));
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = sizeof(Real) == 4 || n_tiles >= kFewTiles;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, geo_step_kernel<Real, MRT, TY, XW>, d, parity, tiles);
}

template <typename Real, bool MRT>
cudaError_t geo_step2_t(const DomDesc& d, int parity, cudaStream_t s)
{
    const dim3 grid((d.nx + kGTX - 1) / kGTX, (d.ny + kGTY - 1) / kGTY);
    geo_step2_kernel<Real, MRT><<<grid, kGTX * kGTY, sizeof(GeoFused<Real>), s>>>(d, parity);
    return cudaGetLastError();
}

template <typename Real, bool MRT>
cudaError_t geo_step2_prepare()
{
    return cudaFuncSetAttribute(geo_step2_kernel<Real, MRT>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(sizeof(GeoFused<Real>)));
}

template <typename Real, bool MRT>
cudaError_t geo_persist_t(const DomDesc& d, int parity0, int flip, int n_steps, int* flags,
                          int* done, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((d.nx + kGTX - 1) / kGTX, (d.ny + kGTY - 1) / kGTY);
    cfg.blockDim = dim3(kGTX * kGTY);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, geo_persist_kernel<Real, MRT>, d, parity0, flip, n_steps, flags,
                              done);
}

template <typename Real, bool MRT>
int geo_persist_occupancy_t()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, geo_persist_kernel<Real, MRT>, kGTX * kGTY,
                                                      0) != cudaSuccess)
        return 0;
    return n;
}

}  // namespace

int geo_tiles(int nx, int ny) { return ((nx + kGTX - 1) / kGTX) * ((ny + kGTY - 1) / kGTY); }

int geo_persist_occupancy(int precision, int coll)
{
    if (precision == 0)
        return coll ? geo_persist_occupancy_t<float, true>() : geo_persist_occupancy_t<float, false>();
    return coll ? geo_persist_occupancy_t<double, true>() : geo_persist_occupancy_t<double, false>();
}

int launch_geo_persist(int precision, int coll, const DomDesc& d, int parity0, int flip,
                       int n_steps, int* flags, int* done, void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (n_steps <= 0) return int(cudaErrorInvalidValue);
    if (precision == 0)
        return int(coll ? geo_persist_t<float, true>(d, parity0, flip, n_steps, flags, done, s)
                        : geo_persist_t<float, false>(d, parity0, flip, n_steps, flags, done, s));
    return int(coll ? geo_persist_t<double, true>(d, parity0, flip, n_steps, flags, done, s)
                    : geo_persist_t<double, false>(d, parity0, flip, n_steps, flags, done, s));
}

int launch_geo_step2(int precision, int coll, const DomDesc& d, int parity, void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 0)
        return int(coll ? geo_step2_t<float, true>(d, parity, s) : geo_step2_t<float, false>(d, parity, s));
    return int(coll ? geo_step2_t<double, true>(d, parity, s) : geo_step2_t<double, false>(d, parity, s));
}

int prepare_geo_step2()
{
    const cudaError_t r[] = {geo_step2_prepare<float, false>(), geo_step2_prepare<float, true>(),
                             geo_step2_prepare<double, false>(), geo_step2_prepare<double, true>()};
    for (cudaError_t v : r)
        if (v != cudaSuccess) return int(v);
    return 0;
}

int launch_geo_step(int precision, int coll, const DomDesc& d, int parity, int tile_rows,
                    const int* tiles, int n_tiles, int sm_count, void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    using Launch = cudaError_t (*)(const DomDesc&, int, const int*, int, cudaStream_t);
    Launch f;
    switch (geo_extra_warps(precision != 0, tile_rows, n_tiles, sm_count)) {
        case 4: f = coll ? geo_step_t<double, true, 4, 4> : geo_step_t<double, false, 4, 4>; break;
        case 3: f = coll ? geo_step_t<float, true, 8, 3> : geo_step_t<float, false, 8, 3>; break;
        case 1: f = coll ? geo_step_t<float, true, 8, 1> : geo_step_t<float, false, 8, 1>; break;
        default:
            f = precision != 0
                ? (coll ? geo_step_t<double, true, 4, 0> : geo_step_t<double, false, 4, 0>)
                : (coll ? geo_step_t<float, true, 4, 0> : geo_step_t<float, false, 4, 0>);
    }
    return int(f(d, parity, tiles, n_tiles, s));
}

size_t geo_tile_capacity(int nx, int ny)
{
    return size_t((nx + kGTX - 1) / kGTX) * size_t((ny + 3) / 4);
}

// Per lattice row and tile column: whether a fluid or wall node is there (bit 0),
// and a fluid node with a solid neighbour (bit 1).  The neighbourhoods go row by
// row: solid at x - 1, x or x + 1, then that of the three rows (lb_set_geometry of a
// 3000 x 1000 map: 108 ms with the eight neighbours looked up for each node and list
// and a division for every node the map's check looks at, 8 ms so).
static std::vector<unsigned char> tile_flags(const unsigned char* cls, int nx, int ny, int walls)
{
    const int ntx = (nx + kGTX - 1) / kGTX;
    std::vector<unsigned char> flags(size_t(ntx) * ny, 0), solid(nx + 2), side[3];
    for (auto& v : side) v.resize(nx);
    auto sides = [&](int y, std::vector<unsigned char>& out) {
        if (walls && (y < 0 || y >= ny)) {
            std::fill(out.begin(), out.end(), 1);
            return;
        }
        const unsigned char* c = cls + size_t((y + ny) % ny) * nx;
        for (int x = 0; x < nx; ++x) solid[x + 1] = c[x] != 0;
        solid[0] = solid[nx];
        solid[nx + 1] = solid[1];
        for (int x = 0; x < nx; ++x) out[x] = solid[x] | solid[x + 1] | solid[x + 2];
    };
    sides(-1, side[2]);
    sides(0, side[0]);
    for (int y = 0; y < ny; ++y) {
        sides(y + 1, side[(y + 1) % 3]);
        const unsigned char* c = cls + size_t(y) * nx;
        for (int t = 0; t < ntx; ++t) {
            unsigned char live = 0, touches = 0;
            for (int x = t * kGTX; x < std::min(t * kGTX + kGTX, nx); ++x) {
                const unsigned char fluid = c[x] == 0;
                live |= fluid | (c[x] == kNodeWall);
                touches |= fluid & (side[0][x] | side[1][x] | side[2][x]);
            }
            flags[size_t(y) * ntx + t] = live | (touches << 1);
        }
    }
    return flags;
}

static std::vector<int> live_tiles(int ty, const std::vector<unsigned char>& flags, int nx, int ny)
{
    const int ntx = (nx + kGTX - 1) / kGTX, nty = (ny + ty - 1) / ty;
    std::vector<int> near, plain;
    for (int q = 0; q < ntx * nty; ++q) {
        unsigned char f = 0;
        for (int y = q / ntx * ty; y < std::min(q / ntx * ty + ty, ny); ++y)
            f |= flags[size_t(y) * ntx + q % ntx];
        if (f & 1) ((f & 2) ? near : plain).push_back((f & 2) ? q | ~kGeoTileIndex : q);
    }
    near.insert(near.end(), plain.begin(), plain.end());
    return near;
}

GeoTiles make_geo_tiles(int precision, int sm_count, const unsigned char* cls, int nx, int ny,
                        int walls)
{
    const std::vector<unsigned char> flags = tile_flags(cls, nx, ny, walls);
    GeoTiles t;
    t.rows = 8;
    if (precision == 0) t.list = live_tiles(8, flags, nx, ny);
    if (precision != 0 || t.list.size() > 3 * size_t(sm_count)) {
        t.rows = 4;
        t.list = live_tiles(4, flags, nx, ny);
    }
    return t;
}

int launch_geo_init_eq(int precision, const DomDesc& d, const double* phi0, int parity, void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 0)
        geo_init_eq_kernel<float><<<geo_grid(d), kGeoBlock, 0, s>>>(d, phi0, parity);
    else
        geo_init_eq_kernel<double><<<geo_grid(d), kGeoBlock, 0, s>>>(d, phi0, parity);
    return int(cudaGetLastError());
}

int launch_geo_solid_rest(int precision, const DomDesc& d, int b, void* stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 0)
        geo_solid_rest_kernel<float><<<geo_grid(d), kGeoBlock, 0, s>>>(d, b);
    else
        geo_solid_rest_kernel<double><<<geo_grid(d), kGeoBlock, 0, s>>>(d, b);
    return int(cudaGetLastError());
}

}  // namespace lbfe

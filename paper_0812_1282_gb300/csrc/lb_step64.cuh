// FP64 fused step on the stage ring of lb_step.cuh (same producer, same
// stages, same strips of W = 32 NW columns).  It is bound by the FP64 pipe
// (lb_node64.cuh), so the compute warps are arranged to give it as few
// operations as possible:
//  - a row's phi is formed once per column by the CTA and shared: each warp
//    publishes its 32 columns of the row ahead, one warp (they take turns)
//    the CTA's two halo columns in one pass, into a two-row ring, and the
//    warps meet at a named barrier.  (Every warp summing its own two halo
//    columns costs 16 operations a row: an operation takes the pipe as long
//    for one lane as for 32.)
//  - the 3 x 3 stencils come from running row values: with e, w, c the
//    published phi of a column and its neighbours, a row keeps
//      k = e - w,  h = e + w,  m = 4 c + h
//    and  X = 4 k_0 + (k_+ + k_-),  Y = m_+ - m_-,
//         L = 4 h_0 - 20 c_0 + (m_+ + m_-),
//    nine operations a node instead of 21.
// The barrier is a hardware wait, not a poll, and every compute warp runs
// the same sequence of barriers whatever its bounded stage waits return.
//
// Measured (MRT, 2048^2, best tile, per step): 1828 us with per-warp halos,
// the phi ring read nine times a node and the plain arithmetic, 834 us so
// (5.03 G node updates/s, 0.925 of what 115.6 operations a node allow at the
// pipe's 628 G DFMA/s); BGK 907 us.  Wall rows take a copy of the code of
// their own: their tests and ghost values in the common one cost it 7 %
// (890 us).  128 x 8 tiles are fastest there, 64 x 16
// within 1 %; wider tiles leave too few CTAs per SM to hide the barrier.
#pragma once

#include "lb_async.cuh"
#include "lb_internal.h"
#include "lb_node64.cuh"
#include "lb_step.cuh"

namespace lbfe {

constexpr int kStages64 = 3;
constexpr int kComputeBarrier64 = 1;

// Shared memory: the stage ring (StageLayout's barriers and stages), then the
// two-row phi ring of W + 2 values.
struct Layout64 {
    StageLayout<double> L;
    __host__ __device__ explicit Layout64(int nw) : L(nw, kStages64) {}
    __host__ __device__ size_t ring_row() const { return size_t(L.W) + 2; }
    __host__ __device__ size_t total() const { return L.rings() + 2 * ring_row() * 8; }
};

template <bool MRT>
__device__ __forceinline__ void consume_tile64(const DomDesc& D, const Node64& C, int parity, int x0,
                                               int y0, int rows, unsigned char* __restrict__ smem,
                                               int NW, int cw, unsigned& q)
{
    constexpr int S = kStages64;
    double* __restrict__ fd = static_cast<double*>(parity ? D.f[0] : D.f[1]);
    double* __restrict__ gd = static_cast<double*>(parity ? D.g[0] : D.g[1]);
    const int nx = D.nx, ny = D.ny, pitch = D.pitch;
    const int P = static_cast<int>(D.plane);
    const bool walls = D.walls != 0;
    const Layout64 Y(NW);
    const StageLayout<double>& L = Y.L;
    const int segw = L.segw;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.full());
    uint64_t* empty = reinterpret_cast<uint64_t*>(smem + L.empty());
    const double* stage = reinterpret_cast<const double*>(smem + L.stages());
    double* ring = reinterpret_cast<double*>(smem + L.rings());

    const int lane = threadIdx.x & 31;
    const TileRows T(y0, rows, ny, walls);
    const unsigned qb = q;
    q += unsigned(T.count());
    const int ncols = min(32 * NW, nx - x0);  // node columns of this strip
    const int col = 32 * cw + lane;           // this lane's column within it
    const bool active = col < ncols;
    const int x = x0 + col;

    auto slot_of = [&](int p) { return (qb + unsigned(p)) % unsigned(S); };
    auto stage_ptr = [&](int p) { return stage + size_t(slot_of(p)) * L.stage_elems(); };
    auto wait_full = [&](int p) {
        const unsigned qq = qb + unsigned(p);
        mbar_wait(full + (qq % unsigned(S)), (qq / unsigned(S)) & 1u, D.err);
    };
    auto release = [&](int p) {
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + slot_of(p));
    };
    // phi of lattice row r (staged at position p): the node's own value, its
    // row values k, h, m on the scaled phi, and the scaled phi itself
    struct Row {
        double phi, s, k, h, m;
        Phi64 g;
    };
    auto publish = [&](int p, Row& v, bool blo, bool bhi) {
        const double* sg = stage_ptr(p) + 9 * segw;
        double* rr = ring + size_t(p & 1) * Y.ring_row();
        double g[9];
        if (active) {
            read9<double>(sg, segw, col + 4, blo, bhi, g);
            v.phi = phi64(C, g, v.g);
            v.s = LB64_MUL(C.sig, v.phi);
            rr[col + 1] = v.s;
        }
        if (cw == p % NW && lane < 2) {  // the strip's halo columns
            const int c = lane ? ncols : -1;
            read9<double>(sg, segw, c + 4, blo, bhi, g);
            rr[c + 1] = LB64_MUL(C.sig, phi64(C, g));
        }
    };
    auto row_of = [&](int p, int r, Row& v) {
        if (walls && (r == 0 || r == ny - 1))
            publish(p, v, r == 0, r == ny - 1);
        else
            publish(p, v, false, false);
        __syncwarp();
        named_sync(kComputeBarrier64, 32 * NW);
        const double* rr = ring + size_t(p & 1) * Y.ring_row();
        if (active) {
            const double w = rr[col], e = rr[col + 2];
            v.k = LB64_SUB(e, w);
            v.h = LB64_ADD(e, w);
            v.m = __fma_rn(C.four, v.s, v.h);
        }
    };
    auto wrap_row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    Row cur, nxt;
    double km = 0.0, mm = 0.0;  // k and m of row y - 1
    cur.phi = cur.s = cur.k = cur.h = cur.m = cur.g.g0 = cur.g.tail = 0.0;
    nxt = cur;
    // collide row y (staged at position p) from the row values around it
    auto collide_row = [&](int y, int p, bool blo, bool bhi) {
        double f[9];
        read9<double>(stage_ptr(p), segw, col + 4, blo, bhi, f);
        const double dx = __fma_rn(C.four, cur.k, LB64_ADD(nxt.k, km));
        const double dy = LB64_SUB(nxt.m, mm);
        const double lap = __fma_rn(C.m20, cur.s, __fma_rn(C.four, cur.h, LB64_ADD(nxt.m, mm)));
        double fo[9], go[9];
        collide64<MRT>(C, f, cur.phi, cur.g, dx, dy, lap, D.step2 && (blo || bhi), D.step2_relax_j != 0,
                       [&](double (&g)[9]) {
                           read9<double>(stage_ptr(p) + 9 * segw, segw, col + 4, blo, bhi, g);
                       },
                       fo, go);
        const int o = y * pitch + x + kXOff;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            fd[i * P + o] = fo[i];
            gd[i * P + o] = go[i];
        }
        // periodic ghost copies: logical 0, 1 also at nx, nx+1 and
        // logical nx-2, nx-1 also at -2, -1
        if (x < 2) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                fd[i * P + o + nx] = fo[i];
                gd[i * P + o + nx] = go[i];
            }
        }
        if (x >= nx - 2) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                fd[i * P + o - nx] = fo[i];
                gd[i * P + o - nx] = go[i];
            }
        }
    };

    const int first = T.first, y1 = T.y1;
    if (!(walls && y0 == 0)) {
        wait_full(0);
        row_of(0, wrap_row(y0 - 1), nxt);
        km = nxt.k;
        mm = nxt.m;
        release(0);
    }
    wait_full(y0 - first);
    row_of(y0 - first, y0, cur);
    for (int y = y0; y < y1; ++y) {
        const int yn = y + 1, py = y - first;
        const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
        if (!bhi) {
            wait_full(yn - first);
            row_of(yn - first, wrap_row(yn), nxt);
        }
        if (active) {
            // wall rows apart, so that the others carry none of their tests
            if (blo || bhi) {
                // a wall ghost row is row k - 1 (ny - k) less k h: its k is
                // that row's and its m that row's less 6 k h (scaled)
                const bool mirror = D.wet_k == 2;
                if (blo) {
                    km = mirror ? nxt.k : cur.k;
                    mm = __dsub_rn(mirror ? nxt.m : cur.m,
                                   ghost_shift64(C.sig, D.wet_k, wet_bottom<double>(D)));
                } else {
                    nxt.k = mirror ? km : cur.k;
                    nxt.m = __dsub_rn(mirror ? mm : cur.m,
                                      ghost_shift64(C.sig, D.wet_k, wet_top<double>(D)));
                }
                collide_row(y, py, blo, bhi);
            } else {
                collide_row(y, py, false, false);
            }
            km = cur.k;
            mm = cur.m;
            cur = nxt;
        }
        release(py);
    }
    // the last staged row (look-ahead only) is released here
    if (T.last >= y1 && !(walls && y1 == ny)) release(T.count() - 1);
}

// Launch shape: blockDim.x = W + 32 (one producer warp, NW compute warps).
template <bool MRT>
__global__ void __launch_bounds__(288) step_single64_kernel(DomDesc D, int parity, int rows)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Node64 C;
    const int NW = int(blockDim.x >> 5) - 1;
    load_node64(C, D.c64, int(threadIdx.x));
    init_stages<double, kStages64>(smem, NW);
    const int warp = int(threadIdx.x >> 5);
    const int x0 = blockIdx.x * 32 * NW, y0 = int(blockIdx.y) * rows;
    unsigned q = 0;
    if (warp == 0) {
        produce_tile<double, kStages64>(D, parity, x0, y0, rows, smem, NW, q);
        drain_stages<double, kStages64>(smem, NW, q, D.err);
    } else {
        consume_tile64<MRT>(D, C, parity, x0, y0, rows, smem, NW, warp - 1, q);
    }
}

// Work-list form (step_batch_kernel's scheduling).
template <bool MRT>
__global__ void __launch_bounds__(288) step_batch64_kernel(const DomDesc* __restrict__ descs,
                                                           const WorkItem* __restrict__ items,
                                                           int n_items, int parity, int* sched,
                                                           unsigned* err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int tags[kStages64];
    __shared__ Node64 C;  // the current tile's constants
    const int NW = int(blockDim.x >> 5) - 1;
    init_stages<double, kStages64>(smem, NW);
    const int warp = int(threadIdx.x >> 5), lane = int(threadIdx.x & 31);
    unsigned q = 0;
    if (warp == 0) {
        for (;;) {
            int it = 0;
            if (lane == 0) it = atomicAdd(sched, 1);
            it = __shfl_sync(0xffffffffu, it, 0);
            if (it >= n_items) {
                produce_end<double, kStages64>(smem, NW, q, tags, err);
                break;
            }
            const WorkItem w = items[it];
            const DomDesc D = descs[w.dom];
            produce_tile<double, kStages64>(D, parity, w.x0, w.y0, w.rows, smem, NW, q, tags, it);
        }
        drain_stages<double, kStages64>(smem, NW, q, err);
        if (lane == 0) {
            __threadfence();
            if (atomicAdd(sched + 1, 1) == int(gridDim.x) - 1) {  // last CTA: reset
                sched[0] = 0;
                sched[1] = 0;
                __threadfence();
            }
        }
    } else {
        for (;;) {
            const int it = next_tag<double, kStages64>(smem, NW, q, tags, err);
            // one decision for all compute warps (the end of the list, or a
            // failed wait on any of them), so that they meet at the same
            // barriers
            if (named_sync_or(kComputeBarrier64, 32 * NW, it < 0 || it >= n_items)) break;
            const WorkItem w = items[it];
            const DomDesc D = descs[w.dom];
            // every compute warp is past the previous tile: refresh the constants
            load_node64(C, D.c64, int(threadIdx.x) - 32);
            named_sync(kComputeBarrier64, 32 * NW);
            consume_tile64<MRT>(D, C, parity, w.x0, w.y0, w.rows, smem, NW, warp - 1, q);
        }
    }
}

}  // namespace lbfe

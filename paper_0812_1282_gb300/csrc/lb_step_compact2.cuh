// Two time steps of the compact step per pass over memory (FP32, compact g
// storage, a single domain without obstacles).
//
// The one-step kernel (lb_step_compact.cuh) moves 104 bytes per node update at
// the rate of a plain copy, so on lattices beyond L2 only fewer bytes make it
// faster.  Here a CTA carries its rows through two steps on the way: level A
// is the one-step pipeline for step t, whose new rows go to rings in shared
// memory instead of to memory, and level B, NW compute warps of its own, is
// the same pipeline for step t + 1 four rows behind, fed from those rings.
// A node's 52 bytes are read once and written once per two steps.
//
// Columns.  Level B produces the strip's W = two_step_strip(bx) node columns
// x0 .. x0 + W - 1 and needs A's new values two columns further on each side,
// for which A reads four columns further: exactly the columns the one-step
// kernel's copies hold (x0 - 4 .. x0 + W + 3).  At the domain's sides these
// are periodic ghost columns four wide, which this kernel writes with its rows
// (the others keep two; launch_wide_ghosts fills the outer ones on entry).
// Rows.  For rows y0 .. y1 - 1 of step t + 1, A steps rows y0 - 2 .. y1 + 1
// (clipped at walls): 4 rows of work and of lead-in per tile.
//
// Iteration p: A expands compact row q = clo + p, publishes phi of row q - 1
// and collides row q - 3 into the rings; B expands A's row q - 4, publishes
// phi of row q - 5 and collides row q - 7, whose pulls read A's rows q - 8 ..
// q - 6.  All compute warps of both levels meet once per iteration, at a named
// barrier: a hardware wait, and every warp runs the same sequence of meetings
// whatever its bounded stage waits return.  (Barriers of their own for the
// levels, A up to an iteration ahead of lock step: 956 us a step on 8192^2
// against 903; the copies issued by the compute warps instead of a producer
// warp: 1031; the collision's loads before the expansion: 1224, spilling.)
//
// Rings: per plane as many rows as lie between A's write and B's last read:
// planes 3, 5, 7 (pulled from the row below) six, the others five (4, 6, 8 are
// pulled from the row above, but from the row itself at the bottom wall); the
// other compact values two, and B takes A's words from A's own word ring.
//
// What bounds it is instruction issue and the latency within an iteration (4096^2:
// 62 % of issue slots, DRAM at 46 %, 10.4 warp instructions a node
// update; waits for fixed-latency results, the barrier, the FMA pipe and the stage
// in that order), with two CTAs of eight compute warps to an SM, which their shared
// memory (98 KB at NW = 4) and registers (96) allow.  Two stages: three made
// no difference.  Measured: 8192^2 1034 -> 880 us a step (64.9 -> 76.3 G node
// updates/s), 2048^2 79.7 -> 66.4.
#pragma once

#include "lb_step_kernels.cuh"

namespace lbfe {

constexpr int kStagesTwo = 2;                  // stage-ring depth
constexpr int kTwoStepF5 = 5, kTwoStepF6 = 6;  // rows of the f rings

// Shared memory of one CTA (byte offsets).
struct TwoStepLayout {
    int NW, S, segw, PC;
    __host__ __device__ TwoStepLayout(int nw, int s)
        : NW(nw), S(s), segw(64 * nw), PC(64 * nw)
    {
    }
    __host__ __device__ size_t full() const { return 0; }
    __host__ __device__ size_t empty() const { return 64; }
    __host__ __device__ size_t stages() const { return 128; }
    __host__ __device__ size_t stage_elems() const { return size_t(13) * segw; }
    // phi and word rings of a level (0: A, 1: B), four rows each
    __host__ __device__ size_t prings(int level) const
    {
        return stages() + size_t(S) * stage_elems() * 4 + size_t(level) * 8 * PC * 4;
    }
    __host__ __device__ size_t wrings(int level) const { return prings(level) + size_t(4) * PC * 4; }
    __host__ __device__ size_t cring() const { return prings(2); }  // Gamma mu, u_eq: [2][3][PC]
    __host__ __device__ size_t fring() const { return cring() + size_t(6) * PC * 4; }
    __host__ __device__ size_t total() const
    {
        return fring() + size_t(6 * kTwoStepF5 + 3 * kTwoStepF6) * PC * 4;
    }
};

// Place of plane i in the f rings: planes 0, 1, 2, 4, 6, 8 take the first six
// rings of five rows, 3, 5, 7 three of six.
__device__ __forceinline__ constexpr bool two_step_six(int i) { return i == 3 || i == 5 || i == 7; }
__device__ __forceinline__ constexpr int two_step_base(int i)
{
    return i < 3 ? i * kTwoStepF5
                 : (two_step_six(i) ? 6 * kTwoStepF5 + (i - 3) / 2 * kTwoStepF6
                                    : (3 + (i - 4) / 2) * kTwoStepF5);
}

// A level's tile: rows y0 .. y1 - 1 (logical, past the lattice's ends where y is
// periodic) from compact rows clo .. chi; stage p carries compact row clo + p
// and, from p = npro on, the f of row clo + p - 3 (TilePlanC).
struct LevelPlan {
    int y0, y1, clo, chi, npro;
    __device__ __forceinline__ LevelPlan(int y0_, int y1_, int ny, bool walls)
        : y0(y0_), y1(y1_), clo(y0_ - 2), chi(y1_ + 1)
    {
        if (walls) {
            clo = max(clo, 0);
            chi = min(chi, ny - 1);
        }
        npro = y0 + 3 - clo;
    }
    __device__ __forceinline__ int count() const { return npro + (y1 - y0); }
};

// The rows of a two-step tile: level B's y0 .. y1 - 1, level A's a0 .. a1 - 1.
struct TwoStepPlan {
    int y0, y1, a0, a1;
    __device__ __forceinline__ TwoStepPlan(int y0_, int rows, int ny, bool walls)
    {
        y0 = y0_;
        y1 = min(y0 + rows, ny);
        a0 = y0 - 2;
        a1 = y1 + 2;
        if (walls) {
            a0 = max(a0, 0);
            a1 = min(a1, ny);
        }
    }
};

// Producer warp: the stages of level A's tile T (produce_tile_c's, with
// logical rows).
template <int S, int NWC>
__device__ __forceinline__ unsigned produce_two_step(const DomDesc& D, int parity, int x0,
                                                     const LevelPlan& T,
                                                     unsigned char* __restrict__ smem)
{
    const float* __restrict__ fs = static_cast<const float*>(parity ? D.f[1] : D.f[0]);
    const float* __restrict__ cs = static_cast<const float*>(parity ? D.g[1] : D.g[0]);
    const int ny = D.ny, pitch = D.pitch;
    const size_t P = size_t(D.plane);
    const bool walls = D.walls != 0;
    const TwoStepLayout L(NWC, S);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.full());
    uint64_t* empty = reinterpret_cast<uint64_t*>(smem + L.empty());
    float* stage = reinterpret_cast<float*>(smem + L.stages());
    const int lane = threadIdx.x & 31;
    // columns x0 - 4 .. x0 + ncols + 3, from a 16-byte boundary on (x0 is even)
    // and a multiple of 16 bytes within the pitch
    const int ncols = min(two_step_strip(32 * NWC), D.nx - x0);
    const int start = x0 & ~3;
    const int seglen = min((x0 - start + ncols + 8 + 3) / 4 * 4, pitch - start);
    const uint32_t segbytes = uint32_t(seglen) * 4u;
    const int i = lane % 9;
    const int ey = ey_of(i);
    auto wrap_row = [&](int r) { return r < 0 ? r + ny : (r >= ny ? r - ny : r); };
    const int n = T.count();
    for (int p = 0; p < n; ++p) {
        const unsigned slot = unsigned(p) % unsigned(S), use = unsigned(p) / unsigned(S);
        if (use > 0) mbar_wait_idle(empty + slot, (use - 1) & 1u, D.err);
        const bool has_f = p >= T.npro, has_c = T.clo + p <= T.chi;
        if (lane == 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(full + slot, ((has_f ? 9u : 0u) + (has_c ? 4u : 0u)) * segbytes);
        }
        __syncwarp();
        float* dst = stage + size_t(slot) * L.stage_elems() + size_t(lane) * L.segw;
        if (lane < 9 && has_f) {
            const int r = T.y0 + (p - T.npro);
            int pl = i, rr = r - ey;
            if (walls && ((ey > 0 && r == 0) || (ey < 0 && r == ny - 1))) {
                pl = opp_of(i);
                rr = r;
            }
            bulk_g2s(dst, fs + size_t(pl) * P + size_t(wrap_row(rr)) * pitch + start, segbytes,
                     full + slot);
        } else if (lane >= 9 && lane < 13 && has_c) {
            bulk_g2s(dst, cs + size_t(lane - 9) * P + size_t(wrap_row(T.clo + p)) * pitch + start,
                     segbytes, full + slot);
        }
        __syncwarp();
    }
    return unsigned(n);
}

// Compute warp cw of level LEVEL (0: A, 1: B).  The steps of an iteration are
// those of consume_tile_c, numbered as there; strip column j is lattice column
// xb + j with xb = x0 - 4 (A) or x0 - 2 (B), node n is lattice column xb + 2 + n.
template <bool MRT, int S, int NWC, int LEVEL>
__device__ __forceinline__ void two_step_level(const DomDesc& D, int parity, int x0, int y0, int rows,
                                               unsigned char* __restrict__ smem, int cw)
{
    constexpr int NW = NWC;
    constexpr bool A = LEVEL == 0;
    const int nx = D.nx, ny = D.ny, pitch = D.pitch;
    const int P = static_cast<int>(D.plane);
    const bool walls = D.walls != 0;
    const NodeParams<float> prm = node_params<float>(D);
    const TwoStepLayout L(NW, S);
    const int segw = L.segw, PC = L.PC;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.full());
    uint64_t* empty = reinterpret_cast<uint64_t*>(smem + L.empty());
    const float* stage = reinterpret_cast<const float*>(smem + L.stages());
    float* pring = reinterpret_cast<float*>(smem + L.prings(LEVEL));
    float* wring = reinterpret_cast<float*>(smem + L.wrings(LEVEL));
    float* cring = reinterpret_cast<float*>(smem + L.cring());
    float* fring = reinterpret_cast<float*>(smem + L.fring());

    const int lane = threadIdx.x & 31;
    const int je = 62 * cw + 2 * lane;
    const int jn = 2 * (32 * cw + lane);
    const TwoStepPlan R(y0, rows, ny, walls);
    const int ncols = min(two_step_strip(32 * NW), nx - x0);
    // this level as a tile: its rows and node columns, the compact rows it expands
    const LevelPlan T(A ? R.a0 : R.y0, A ? R.a1 : R.y1, ny, walls);
    const int nodes = A ? ncols + 4 : ncols;
    const bool n_on = jn < nodes;
    const int clo_a = LevelPlan(R.a0, R.a1, ny, walls).clo;
    const int last = R.y1 + 6 - clo_a;  // the iteration of B's last row

    auto slot_of = [&](int p) { return unsigned(p) % unsigned(S); };
    const int shift = x0 & 3;  // of the copies' first column before x0 - 4
    auto stage_ptr = [&](int p) { return stage + size_t(slot_of(p)) * L.stage_elems() + shift; };
    // the four ring rows of phi and words in turn
    auto rslot = [&](int y) -> float* { return pring + ((y - T.y0 + 1) & 3) * PC; };
    auto wslot = [&](int y) -> float* { return wring + ((y - T.y0 + 1) & 3) * PC; };
    // row y of plane i in the f rings (y - a0 >= 0)
    auto frow = [&](int i, int y) -> float* {
        const int k = y - R.a0;
        return fring + (two_step_base(i) + (two_step_six(i) ? k % kTwoStepF6 : k % kTwoStepF5)) * PC;
    };
    auto crow = [&](int y) -> float* { return cring + ((y - R.a0) & 1) * 3 * PC; };
    // A's words of row y as B expands it, by A's node (its ring holds the row
    // until A publishes row y + 4, an iteration later)
    const float* awords = reinterpret_cast<const float*>(smem + L.wrings(0)) + 2;
    auto arow = [&](int y) -> const float* { return awords + ((y - R.a0 + 1) & 3) * PC; };

    const int pub_lo = (walls && T.y0 == 0) ? 0 : T.y0 - 1;
    const int pub_hi = walls ? min(T.y1, ny - 1) : T.y1;
    const f2 zero(0.f);
    f2 u_next = zero, uh = zero, wd = zero, tl = zero, d_wall = zero;
    const unsigned kAll = 0xffffffffu;
    for (int p = 0; p <= last; ++p) {
        const int qr = A ? clo_a + p : clo_a + p - 4;  // this level's compact row
        const bool staged = A && qr - 3 < T.y1;
        if (staged) mbar_wait(full + slot_of(p), (unsigned(p) / unsigned(S)) & 1u, D.err);
        f2 d_pub = d_wall;
        f2 uh_q = zero, wd_q = zero, tl_q = zero;
        if (qr >= T.clo && qr <= T.chi) {
            // 1. expand
            const float* sw = A ? stage_ptr(p) + 9 * segw + je : arow(qr) + je;
            const float* sc = A ? sw + segw : crow(qr) + je;  // Gamma mu, u_eq
            const int step = A ? segw : PC;
            wd_q = f2(ld_pair(sw));
            f2 ge[9];
            g_equilibria2(g0_value2(wd_q), f2(ld_pair(sc)), f2(ld_pair(sc + step)),
                          f2(ld_pair(sc + 2 * step)), ge);
            tl_q = g_tail_sum2(ge);
            // 2. sideways
            const f2 g5l(__shfl_up_sync(kAll, ge[5].v.y, 1), ge[5].v.x);
            const f2 g1l(__shfl_up_sync(kAll, ge[1].v.y, 1), ge[1].v.x);
            const f2 g8l(__shfl_up_sync(kAll, ge[8].v.y, 1), ge[8].v.x);
            const f2 g7r(ge[7].v.y, __shfl_down_sync(kAll, ge[7].v.x, 1));
            const f2 g2r(ge[2].v.y, __shfl_down_sync(kAll, ge[2].v.x, 1));
            const f2 g6r(ge[6].v.y, __shfl_down_sync(kAll, ge[6].v.x, 1));
            const f2 h_q = g1l + g2r;
            const f2 u_q = (walls && qr == 0) ? (ge[4] + ge[6]) + ge[8] : u_next;
            uh_q = u_q + h_q;
            d_pub = (ge[4] + g6r) + g8l;
            u_next = (ge[3] + g5l) + g7r;
            if (walls && qr == ny - 1) d_wall = (ge[3] + ge[5]) + ge[7];
        }
        // 3. phi(t+1) of row qr - 1
        const int r = qr - 1;
        if (r >= pub_lo && r <= pub_hi) {
            const f2 word = g0_advance2(wd, (uh + d_pub) - tl);
            const f2 phi = g0_value2(word);
            float* pr = rslot(r) + je;
            float* wr = wslot(r) + je;
            if (lane > 0 && lane < 31) {
                st_pair(pr, phi.v);
                st_pair(wr, word.v);
            } else if (lane == 0) {
                pr[1] = phi.v.y;
                wr[1] = word.v.y;
            } else {
                pr[0] = phi.v.x;
                wr[0] = word.v.x;
            }
        }
        uh = uh_q;
        wd = wd_q;
        tl = tl_q;
        // 4. collide row y = qr - 3
        const int y = qr - 3;
        if (y >= T.y0 && y < T.y1 && n_on) {
            const bool blo = walls && y == 0, bhi = walls && y == ny - 1;
            f2 fi[9];
            if constexpr (A) {
                // the stage holds what each node pulls; node n is at index n + 2
                const float* sb = stage_ptr(p) + jn + 2;
                fi[0] = ld_pair(sb);
                fi[1] = ld_two(sb + segw - 1);
                fi[2] = ld_two(sb + 2 * segw + 1);
                fi[3] = ld_pair(sb + 3 * segw);
                fi[4] = ld_pair(sb + 4 * segw);
                fi[5] = blo ? ld_pair(sb + 5 * segw) : ld_two(sb + 5 * segw - 1);
                fi[6] = bhi ? ld_pair(sb + 6 * segw) : ld_two(sb + 6 * segw + 1);
                fi[7] = blo ? ld_pair(sb + 7 * segw) : ld_two(sb + 7 * segw + 1);
                fi[8] = bhi ? ld_pair(sb + 8 * segw) : ld_two(sb + 8 * segw - 1);
            } else {
                // A's new rows; B's node n is A's node n + 2
                const int c = jn + 2;
                fi[0] = ld_pair(frow(0, y) + c);
                fi[1] = ld_two(frow(1, y) + c - 1);
                fi[2] = ld_two(frow(2, y) + c + 1);
                if (blo) {
                    fi[3] = ld_pair(frow(4, y) + c);
                    fi[5] = ld_pair(frow(6, y) + c);
                    fi[7] = ld_pair(frow(8, y) + c);
                } else {
                    fi[3] = ld_pair(frow(3, y - 1) + c);
                    fi[5] = ld_two(frow(5, y - 1) + c - 1);
                    fi[7] = ld_two(frow(7, y - 1) + c + 1);
                }
                if (bhi) {
                    fi[4] = ld_pair(frow(3, y) + c);
                    fi[6] = ld_pair(frow(5, y) + c);
                    fi[8] = ld_pair(frow(7, y) + c);
                } else {
                    fi[4] = ld_pair(frow(4, y + 1) + c);
                    fi[6] = ld_two(frow(6, y + 1) + c + 1);
                    fi[8] = ld_two(frow(8, y + 1) + c - 1);
                }
            }
            auto row3 = [&](const float* rw, f2& w, f2& c, f2& e) {
                const float2 a = ld_pair(rw + jn), b = ld_pair(rw + jn + 2),
                             d = ld_pair(rw + jn + 4);
                w = f2(a.y, b.x);
                c = f2(b);
                e = f2(b.y, d.x);
            };
            f2 cw_, cc, ce, nw_, nc, ne, sw, sc_, se;
            row3(rslot(y), cw_, cc, ce);
            if (bhi) {
                row3(rslot(ny - D.wet_k), nw_, nc, ne);
                const f2 h(float(D.wet_k) * wet_top<float>(D));
                nw_ = nw_ - h;
                nc = nc - h;
                ne = ne - h;
            } else {
                row3(rslot(y + 1), nw_, nc, ne);
            }
            if (blo) {
                row3(rslot(D.wet_k - 1), sw, sc_, se);
                const f2 h(float(D.wet_k) * wet_bottom<float>(D));
                sw = sw - h;
                sc_ = sc_ - h;
                se = se - h;
            } else {
                row3(rslot(y - 1), sw, sc_, se);
            }
            f2 dx, dy, lap;
            stencils2(cc, ce, cw_, nc, sc_, ne, nw_, se, sw, dx, dy, lap);
            const bool s2 = D.step2 && (blo || bhi);
            f2 fo2[9], uxe, uye;
            collide_f2<MRT>(prm, fi, cc, dx, dy, lap, s2, D.step2_relax_j != 0, fo2, uxe, uye);
            const f2 gmu = gamma_mu2(prm, cc, lap);
            if constexpr (A) {
#pragma unroll
                for (int i = 0; i < 9; ++i) st_pair(frow(i, y) + jn, fo2[i].v);
                st_pair(crow(y) + jn, gmu.v);
                st_pair(crow(y) + PC + jn, uxe.v);
                st_pair(crow(y) + 2 * PC + jn, uye.v);
            } else {
                const f2 co2[4] = {f2(ld_pair(wslot(y) + jn + 2)), gmu, uxe, uye};
                float* __restrict__ fd = static_cast<float*>(parity ? D.f[0] : D.f[1]);
                float* __restrict__ cd = static_cast<float*>(parity ? D.g[0] : D.g[1]);
                const int x = x0 + jn;
                const int o = y * pitch + x + kXOff;  // even: pairs are 8-byte aligned
                if (jn + 1 < ncols) {
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        *reinterpret_cast<float2*>(fd + i * P + o) = fo2[i].v;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        *reinterpret_cast<float2*>(cd + kk * P + o) = co2[kk].v;
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i) fd[i * P + o] = fo2[i].v.x;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) cd[kk * P + o] = co2[kk].v.x;
                }
                // periodic ghost copies, four wide
                if (x < 4 || x + 1 >= nx - 4) {
#pragma unroll
                    for (int l = 0; l < 2; ++l) {
                        const int xl = x + l;
                        if (jn + l >= ncols) continue;
                        const int to = xl < 4 ? nx : (xl >= nx - 4 ? -nx : 0);
                        if (to == 0) continue;
#pragma unroll
                        for (int i = 0; i < 9; ++i) fd[i * P + o + l + to] = fo2[i].lane(l);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) cd[kk * P + o + l + to] = co2[kk].lane(l);
                    }
                }
            }
        }
        __syncwarp();
        if (staged && lane == 0) mbar_arrive(empty + slot_of(p));
        named_sync(kComputeBarrier, 64 * NW);
    }
}

// blockDim.x = 64 NW + 32: the producer warp, NW warps of level A, NW of
// level B.
template <bool MRT, int NWC>
__global__ void __launch_bounds__(64 * NWC + 32, NWC >= 3 ? 2 : 4)
    step_two_compact_kernel(DomDesc D, int parity, int rows, int band_mul)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int S = kStagesTwo;
    init_stages_c<S>(smem, NWC);
    const int warp = int(threadIdx.x >> 5);
    const int x0 = blockIdx.x * two_step_strip(32 * NWC);
    const int y0 = band_of(band_mul) * rows;
    if (warp == 0) {
        // level A's tile, whose node columns start two before the strip's
        const TwoStepPlan R(y0, rows, D.ny, D.walls != 0);
        const unsigned q = produce_two_step<S, NWC>(
            D, parity, x0, LevelPlan(R.a0, R.a1, D.ny, D.walls != 0), smem);
        drain_stages<float, S, NWC>(smem, NWC, q, D.err);
    } else if (warp <= NWC) {
        two_step_level<MRT, S, NWC, 0>(D, parity, x0, y0, rows, smem, warp - 1);
    } else {
        two_step_level<MRT, S, NWC, 1>(D, parity, x0, y0, rows, smem, warp - 1 - NWC);
    }
}

}  // namespace lbfe

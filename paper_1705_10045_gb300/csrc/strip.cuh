// One-launch D2Q9 time step: a warp marches a strip of columns along y.
//
// A step of a D2Q9 node depends on the moments of a 2-ring around it
// (fused.cuh), and a row of the ring adds only four columns.  So the step
// needs no tile wider than a warp and no hand-off between warps.  Lane l of a
// warp holds column a0 - 2 + l; lanes 2..29 own the 28 columns the warp
// collides.  Per row i the warp forms the moments and Phi of row i, the force
// of row i-1 and the collision of row i-2.  Neighbour columns come from warp
// shuffles, neighbour rows from the lane's registers (a ring of four rows
// named at compile time by unrolling four rows).  A row's nine pairs come
// into shared memory by cp.async two rows ahead; each lane reads back only
// what it copied, once for the moments and once for the collision, so there
// is no barrier and every population is read once from global memory per
// strip (plus the ring columns, which a neighbouring warp of the CTA has
// brought into L1).
//
// What bounds it: 433 warp instructions per row of 28 nodes (495 per node and
// lane; the producer/consumer march of fused.cuh took 873), with the
// collision's two sets packed into f32x2 instructions, leave the step bound
// by HBM on large domains and by the instruction latency of a row
// (0.58 us) where a domain cannot fill the SMs.  Measured on one GB300 against that march, FP32: 8192 x 4608
// 1174 -> 895 us (144 B per node: 6.07 TB/s, 0.89 of the measured copy
// bandwidth), 512 x 512 18.4 -> 8.4 us, 128 x 128 18 -> 3.7 us; FP16 storage
// 8192 x 4608 707 us.  Pairs held in registers over the three rows instead of
// shared memory (168 registers, 12 warps per SM) gave 1146 us: too few loads
// in flight.  Five CTAs per SM (102 registers) 931 us, nine of two warps 947.
#pragma once

#include "node.cuh"
#include "plan.h"

namespace lbm {

// asynchronous copy of one stored pair into shared memory
template <typename S> __device__ __forceinline__ void copy_async(Pop<S>* to, const Pop<S>* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from),
                 "n"(sizeof(Pop<S>))
                 : "memory");
}

// WALL: the domain has walls on x or y (the other instance is periodic and
// carries no trace of them).
template <typename S, typename R, bool WALL> struct Strip {
    static constexpr int Q = 9;
    static constexpr int kCols = kStripCols;
    // rows a warp holds: the two loaded ahead of the moments, the row the
    // moments take and the one between it and the collision's (whose slot the
    // next load reuses)
    static constexpr int kRows = 4, kAhead = 2;
    static constexpr size_t kRingBytes = sizeof(Pop<S>) * Q * 32 * kRows;   // per warp
    using Math = NodeMath<9, S, R>;

    const Pop<S>* src;   // written by the previous launch until griddepcontrol.wait: not __restrict__
    Pop<S>* dst;
    const KParams<R>& p;
    Counters* cnt;
    size_t nn;
    int na, nm, zb, ze;
    unsigned step;
    int lane, col;          // the lane's column (wrapped, or the mirror column across a wall)
    int col_m, col_p;       // columns the pushes to x - 1 and x + 1 go to
    bool owns;
    int edge;               // walls beside the column (bit 0 low, bit 1 high)
    bool edge_strip;        // a column the warp owns lies beside a wall
    Pop<S>* ring;           // the lane's column of the warp's rows in shared memory
    int next_row;           // wrapped index of the row the next load takes

    // rows i-3 .. i, row r in slot (r - (zb - 2)) & 3
    R phi[4], phl[4], phr[4], rho[4], T[4], P[4], ua[4], um[4], E[4], da[4], dm[4];

    __device__ __forceinline__ Strip(const S* s, S* d, const KParams<R>& kp, Counters* c, int columns, int rows,
                                     int first, int last, unsigned st, int a0, Pop<S>* rows_smem)
        : src(reinterpret_cast<const Pop<S>*>(s)), dst(reinterpret_cast<Pop<S>*>(d)), p(kp), cnt(c),
          nn((size_t)kp.nn), na(columns), nm(rows), zb(first), ze(last), step(st) {
        lane = threadIdx.x & 31;
        ring = rows_smem + lane;
        const int a = a0 + lane - 2;
        col = a;
        if (WALL && p.wall_x) {
            if (col < 0) col = -1 - col;
            if (col >= na) col = 2 * na - 1 - col;
            col = col < 0 ? 0 : (col >= na ? na - 1 : col);
        } else {
            col %= na;
            if (col < 0) col += na;
        }
        owns = lane >= 2 && lane < 2 + kCols && a < na;
        edge = WALL && p.wall_x ? (a == 0 ? 1 : 0) | (a == na - 1 ? 2 : 0) : 0;
        edge_strip = WALL && p.wall_x && (a0 == 0 || a0 + kCols >= na);
        col_m = col == 0 ? na - 1 : col - 1;
        col_p = col == na - 1 ? 0 : col + 1;
        next_row = (zb - 2) % nm;
        if (next_row < 0) next_row += nm;
    }

    // rows the step reads: all when the axis is periodic, those inside the walls otherwise
    __device__ __forceinline__ bool inside(int m) const { return !WALL || !p.wall || (m >= 0 && m < nm); }

    // start the copies of row m into slot J (one group per row, empty beyond the ring)
    template <int J> __device__ __forceinline__ void load(int m) {
        if (m <= ze + 1 && inside(m)) {
            const unsigned n = (unsigned)(next_row * na + col);
#pragma unroll
            for (int k = 0; k < Q; ++k) copy_async<S>(ring + (J * Q + k) * 32, src + k * nn + n);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        next_row = next_row + 1 == nm ? 0 : next_row + 1;
    }

    template <int J> __device__ __forceinline__ void moments(int m) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
        if (inside(m)) {
            Pop<S> f[Q];
#pragma unroll
            for (int k = 0; k < Q; ++k) f[k] = ring[(J * Q + k) * 32];
            const Moments<R> o = Math::moments(f, p);
            const R inv_rho = R(1) / o.rho;
            rho[J] = o.rho;
            E[J] = o.E;
            T[J] = o.E / (o.rho * p.c_v);
            ua[J] = o.ja * inv_rho;
            um[J] = o.jm * inv_rho;
            P[J] = eos_pressure(p, o.rho, T[J]);
            phi[J] = Math::phi_of(Math::potential(o.rho, P[J]));
        }
        phl[J] = __shfl_up_sync(0xffffffffu, phi[J], 1);
        phr[J] = __shfl_down_sync(0xffffffffu, phi[J], 1);
    }

    // du of row f, in slot J
    template <int J> __device__ __forceinline__ void force(int f) {
        if (WALL && !inside(f)) return;
        constexpr int D = (J + 3) & 3, U = (J + 1) & 3;
        // a stencil row beyond a wall is the row itself
        const bool lo = WALL && p.wall && f == 0, hi = WALL && p.wall && f == nm - 1;
        const R d[3] = {lo ? phl[J] : phl[D], lo ? phi[J] : phi[D], lo ? phr[J] : phr[D]};
        const R u[3] = {hi ? phl[J] : phl[U], hi ? phi[J] : phi[U], hi ? phr[J] : phr[U]};
        const R o[3] = {phl[J], phi[J], phr[J]};
        R du[3];
        Math::force(p, [&](int a, int, int m) { return m < 0 ? d[a + 1] : (m > 0 ? u[a + 1] : o[a + 1]); }, rho[J], du);
        da[J] = du[0];
        dm[J] = du[2];
    }

    // collision and push of row c, in slot J
    template <int J> __device__ __forceinline__ void collide(int c) {
        constexpr int D = (J + 3) & 3, U = (J + 1) & 3;
        const R half = R(0.5), r = rho[J], Tc = T[J];
        const R us = ::fma(da[J], half, ua[J]);
        R uu = __shfl_down_sync(0xffffffffu, us, 1), ud = __shfl_up_sync(0xffffffffu, us, 1);
        const bool gu = WALL && p.wall && c + 1 >= nm, gd = WALL && p.wall && c == 0;
        // ghosts beyond a wall: normal velocity negated
        if (WALL && edge) {
            if (edge & 2) uu = -us;
            if (edge & 1) ud = -us;
        }
        const R own_m = -::fma(dm[J], half, um[J]);
        typename Math::Axis ax[2] = {{uu, ud, Tc, Tc, r, r},
                                     {gu ? own_m : ::fma(dm[U], half, um[U]), gd ? own_m : ::fma(dm[D], half, um[D]), Tc,
                                      Tc, r, r}};
        if (p.conduction) {
            ax[0].Tu = __shfl_down_sync(0xffffffffu, Tc, 1);
            ax[0].Td = __shfl_up_sync(0xffffffffu, Tc, 1);
            // T beyond a wall: mirrored, or reflected about the wall temperature
            ax[1].Tu = gu ? (p.T_fixed_hi ? R(2) * p.T_hi - Tc : Tc) : T[U];
            ax[1].Td = gd ? (p.T_fixed_lo ? R(2) * p.T_lo - Tc : Tc) : T[D];
            if (WALL && (edge & 2)) ax[0].Tu = p.T_fixed_x[1] ? R(2) * p.T_x[1] - Tc : Tc;
            if (WALL && (edge & 1)) ax[0].Td = p.T_fixed_x[0] ? R(2) * p.T_x[0] - Tc : Tc;
            if (p.chi_mode) {
                ax[0].ru = __shfl_down_sync(0xffffffffu, r, 1);
                ax[0].rd = __shfl_up_sync(0xffffffffu, r, 1);
                if (WALL && (edge & 2)) ax[0].ru = r;
                if (WALL && (edge & 1)) ax[0].rd = r;
                if (!gu) ax[1].ru = rho[U];
                if (!gd) ax[1].rd = rho[D];
            }
        }
        if (!owns) return;
        const R dE = Math::energy_change(p, r, Tc, P[J], ax, 2);
        const bool clamp = Math::potential(r, P[J]) >= R(0), bad = !(Math::positive(r) && Math::positive(E[J]));
        if (clamp || bad) {
            if (clamp) atomicAdd(&cnt->clamps, 1ull);
            if (bad) atomicAdd(&cnt->bad, 1ull);
        }

        const int row = c * na, n = row + col;
        const unsigned nbits = Store<S, R>::kStochastic ? node_bits(step, (unsigned)n) : 0u;
        const R u[3] = {ua[J], R(0), um[J]}, dv[3] = {da[J], R(0), dm[J]};
        const int row_m = c == 0 ? (nm - 1) * na : row - na, row_p = c == nm - 1 ? 0 : row + na;
        auto push = [&](auto wall_tag) {
            constexpr bool BOUNCE = decltype(wall_tag)::value;
            Math::collide(p, r, E[J], u, dv, dE, [&](int k) { return ring[(J * Q + k) * 32]; }, [&](int k, Two<R> out) {
                using M = MVel<9>;
                const unsigned t = Store<S, R>::kStochastic ? pair_word(nbits, k) : 0u;
                const int to = (M::m(k) == 0 ? row : (M::m(k) > 0 ? row_p : row_m)) +
                               (M::a(k) == 0 ? col : (M::a(k) > 0 ? col_p : col_m));
                // halfway bounce-back: the pair stays at its node, in the opposite direction
                const bool bounce = BOUNCE && ((M::m(k) == -1 && gd) || (M::m(k) == 1 && gu) ||
                                               (M::a(k) == -1 && (edge & 1)) || (M::a(k) == 1 && (edge & 2)));
                if (BOUNCE && bounce) store_pop(dst + opposite(k) * nn, (unsigned)n, out, t);
                else store_pop(dst + k * nn, (unsigned)to, out, t);
            });
        };
        // one instance for the whole warp: lanes apart would run both in turn
        if (WALL && (gu || gd || edge_strip)) push(std::true_type{});
        else push(std::false_type{});
    }

    template <int J> __device__ __forceinline__ void row(int i) {
        moments<J>(i);
        if (i >= zb) force<(J + 3) & 3>(i - 1);
        if (i >= zb + 2) collide<(J + 2) & 3>(i - 2);
        load<(J + kAhead) & 3>(i + kAhead);
    }

    __device__ __forceinline__ void run() {
        load<0>(zb - 2);
        load<1>(zb - 1);
        for (int i = zb - 2;; ) {
            row<0>(i);
            if (++i == ze + 2) break;
            row<1>(i);
            if (++i == ze + 2) break;
            row<2>(i);
            if (++i == ze + 2) break;
            row<3>(i);
            if (++i == ze + 2) break;
        }
    }
};

template <typename S, typename R, bool WALL>
__global__ void __launch_bounds__(32 * kStripWarps, kStripCtas)
    strip_step_kernel(const S* src, S* dst, const __grid_constant__ KParams<R> p, StripGeom G,
                      Counters* cnt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, w = blockIdx.x * kStripWarps + warp;
    const int strip = w % G.strips, zb = G.m_lo + (w / G.strips) * G.chunk;
    if (zb >= G.m_hi) return;
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the previous step's stores
    using St = Strip<S, R, WALL>;
    St s(src, dst, p, cnt, G.na, G.nm, zb, min(zb + G.chunk, G.m_hi), p.step, strip * St::kCols,
         reinterpret_cast<Pop<S>*>(smem_raw + warp * St::kRingBytes));
    s.run();
}

}  // namespace lbm

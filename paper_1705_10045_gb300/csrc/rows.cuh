// One-launch D3Q19 time step in FP32 and FP16 storage for domains periodic in
// x: a CTA marches rows of columns along z, one warp per row.
//
// The strip of strip.cuh with a second tile axis.  Warp w of a CTA holds row
// b0 - 2 + w (TY rows the CTA collides and a 2-ring of rows), lane l column
// a0 + l of the tile (28 columns and a 2-ring).  Per plane i a warp forms the
// moments and Phi of plane i, the force of plane i-1 (all rows but the
// outermost two) and the collision of plane i-2 (the TY rows).  Neighbours in
// x come from shuffles, neighbours in z from the lane's registers, neighbours
// in y from shared memory: Phi of four planes, and u*_y, T and rho of two, so
// one barrier a plane orders everything:
//   iteration i:  M(i) writes Phi(i)            barrier
//                 F(i-1) reads Phi(i-2 .. i), writes u*_y, T, rho of i-1
//                 C(i-2) reads u*_y, T, rho of i-2 (written at i-1)
// A slot is written again after the barrier that follows its last read.  A
// warp's pairs come into shared memory by 16-byte cp.async AHEAD planes ahead
// and stay there until their collision, so every population is read once from
// global memory (ring rows and columns, 1.4 to 1.7 times the nodes, come from
// L2).  The 16-byte copies bypass L1, which is what is left of the shared
// memory; 8- and 4-byte copies through it gave 3530 and 1890 us.
//
// What bounds it: instructions and the barrier a plane.  Against the producer/consumer
// march of fused.cuh, which reads every node's pairs twice (the second time
// partly from DRAM) and holds its loads in flight in registers and L1, 384 x
// 384 x 256 in us per step: FP32 2545 -> 2325 (4.94 TB/s of 304 B per node,
// 0.73 of the measured copy bandwidth), FP16 storage 2020 -> 1720.  DRAM reads
// are 1.01 times the populations (march: 1.24 to 1.30); the wait at the
// barrier comes first now (1.6 cycles per instruction), issue is 50 % busy in
// FP32 and 68 % in FP16.
#pragma once

#include "fused.cuh"

namespace lbm {

template <typename S, typename R, int TY, int AHEAD, bool WALL> struct RowMarch {
    static constexpr int Q = 19, kRows = TY + 4;
    static constexpr int kAhead = AHEAD, kOwn = AHEAD + 2, kRing = AHEAD;   // planes held by a collided and by a ring row
    static constexpr int kPer = 16 / (int)sizeof(Pop<S>), kChunks = 32 / kPer;   // pairs in 16 bytes, 16-byte parts of a row
    static constexpr int kStride = 34;   // Phi row: a column of padding on either side
    using Math = NodeMath<19, S, R>;
    using M = MVel<19>;
    static constexpr size_t kPopBytes = sizeof(Pop<S>) * Q * 32 * (size_t)(TY * kOwn + 4 * kRing);
    static constexpr size_t kBytes = kPopBytes + sizeof(R) * (size_t)(4 * kRows * kStride + 3 * 2 * kRows * 32);
    static_assert(kBytes <= 227 * 1024, "shared memory");

    const Pop<S>* src;   // written by the previous launch until griddepcontrol.wait: not __restrict__
    Pop<S>* dst;
    const KParams<R>& p;
    Counters* cnt;
    size_t nn;
    int na, nb, nm, plane_n, zb, ze;
    unsigned step;
    int lane, w, n_ab;          // n_ab: the lane's node in a plane (wrapped, or the mirror node across a wall)
    int n_vec;                  // the first node of the 16 bytes the lane copies
    int dA_m, dA_p, dB_m, dB_p; // offsets of the pushes along x and y
    bool own_row, owns;
    bool low_y, high_y;         // the warp's row lies beside a wall on y
    Pop<S>* ring;               // the lane's column of the warp's planes
    R* phi_s;                   // Phi rows
    R* ex;                      // u*_y, T, rho
    int next_plane;             // wrapped index of the plane the next load takes

    __device__ __forceinline__ RowMarch(const S* s, S* d, const KParams<R>& kp, Counters* c, const MarchGeom& G, int a0,
                                        int b0, int first, int last, unsigned st, unsigned char* smem)
        : src(reinterpret_cast<const Pop<S>*>(s)), dst(reinterpret_cast<Pop<S>*>(d)), p(kp), cnt(c),
          nn((size_t)kp.nn), na(G.na), nb(G.nb), nm(G.nm), plane_n(G.na * G.nb), zb(first), ze(last), step(st) {
        lane = threadIdx.x & 31;
        w = threadIdx.x >> 5;
        own_row = w >= 2 && w < TY + 2;
        // lane 0 stands at a multiple of 28 columns (so the last tile collides
        // columns 0 and 1)
        const int a = a0 + lane, b = b0 + w - 2;
        const int col = a % na, row = ring_coord(b, nb, WALL && p.wall_y);
        n_ab = row * na + col;
        owns = own_row && lane >= 2 && lane < 2 + kStripCols && a < na + 2 && b < nb;
        n_vec = row * na + (a0 + kPer * (lane & (kChunks - 1))) % na;
        dA_m = col == 0 ? na - 1 : -1;
        dA_p = col == na - 1 ? 1 - na : 1;
        dB_m = (row == 0 ? nb - 1 : -1) * na;
        dB_p = (row == nb - 1 ? 1 - nb : 1) * na;
        low_y = WALL && p.wall_y && b == 0;
        high_y = WALL && p.wall_y && b == nb - 1;
        // collided rows first, then the four ring rows
        const int own = w - 2, outer = w < 2 ? w : w - TY;
        ring = reinterpret_cast<Pop<S>*>(smem) +
               (own_row ? own * kOwn : TY * kOwn + outer * kRing) * (Q * 32) + lane;
        phi_s = reinterpret_cast<R*>(smem + kPopBytes);
        ex = phi_s + 4 * kRows * kStride;
        next_plane = wrapi(zb - 2, nm);
    }
    __device__ __forceinline__ bool inside(int m) const { return !WALL || !p.wall || (m >= 0 && m < nm); }
    __device__ __forceinline__ R& phi(int slot, int row, int l) const {
        return phi_s[(slot * kRows + row) * kStride + l + 1];
    }
    __device__ __forceinline__ R& exch(int f, int plane, int row) const {
        return ex[((f * 2 + (plane & 1)) * kRows + row) * 32 + lane];
    }

    // start the copies of plane m into slot (one group per plane, empty beyond the ring)
    __device__ __forceinline__ void load(int m, int slot) {
        __syncwarp();   // the warp's last reads of the slot come before any lane's copies into it
        if (m <= ze + 1 && inside(m)) {
            // a row of 32 pairs is kChunks parts of 16 bytes: lane l copies part
            // l mod kChunks of every (32 / kChunks)-th direction
            constexpr int kStep = 32 / kChunks;
            int k = lane / kChunks;
            const Pop<S>* q = src + (size_t)k * nn + (size_t)(unsigned)(next_plane * plane_n + n_vec);
            Pop<S>* at = ring - lane + (slot * Q + k) * 32 + (lane & (kChunks - 1)) * kPer;
#pragma unroll
            for (int j = 0; j < (Q + kStep - 1) / kStep; ++j) {
                if ((j + 1) * kStep <= Q || k < Q)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(at)),
                                 "l"(q)
                                 : "memory");
                q += kStep * nn;
                at += kStep * 32;
                k += kStep;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        next_plane = next_plane + 1 == nm ? 0 : next_plane + 1;
    }

    __device__ __forceinline__ void run() {
        const int held = own_row ? kOwn : kRing;
        int put = 0;   // slot of the next load; the moments' slot trails it by kAhead, the collision's by kAhead + 2
        for (int j = 0; j < kAhead; ++j) {
            load(zb - 2 + j, put);
            put = put + 1 == held ? 0 : put + 1;
        }
        int got = 0, done = 0;   // slots of plane i and (collided rows) of plane i - 2
        // plane i, i-1, i-2, i-3: suffix 0 .. 3
        R phi0 = 0, phi1 = 0, phi2 = 0, phl0 = 0, phl1 = 0, phl2 = 0, phr0 = 0, phr1 = 0, phr2 = 0;
        R rho0 = 1, rho1 = 1, rho2 = 1, rho3 = 1, T0 = 0, T1 = 0, T2 = 0, T3 = 0;
        R u0[3] = {0, 0, 0}, u1[3] = {0, 0, 0}, u2[3] = {0, 0, 0}, E0 = 1, E1 = 1, E2 = 1, P0 = 0, P1 = 0, P2 = 0;
        R du1[3] = {0, 0, 0}, du2[3] = {0, 0, 0}, us1 = 0, us2 = 0, us3 = 0;   // us: u* along z
#pragma unroll 1
        for (int i = zb - 2; i < ze + 2; ++i) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
            __syncwarp();   // every lane's part has arrived
            if (inside(i)) {
                Pop<S> f[Q];
                const Pop<S>* q = ring + got * (Q * 32);
#pragma unroll
                for (int k = 0; k < Q; ++k) f[k] = q[k * 32];
                const Moments<R> o = Math::moments(f, p);
                const R inv = R(1) / o.rho;
                rho0 = o.rho;
                E0 = o.E;
                T0 = o.E / (o.rho * p.c_v);
                u0[0] = o.ja * inv;
                u0[1] = o.jb * inv;
                u0[2] = o.jm * inv;
                P0 = eos_pressure(p, o.rho, T0);
                phi0 = Math::phi_of(Math::potential(o.rho, P0));
                phi(i & 3, w, lane) = phi0;
            }
            got = got + 1 == held ? 0 : got + 1;
            phl0 = __shfl_up_sync(0xffffffffu, phi0, 1);
            phr0 = __shfl_down_sync(0xffffffffu, phi0, 1);
            __syncthreads();

            const int f = i - 1;
            if (i >= zb && inside(f) && w >= 1 && w < kRows - 1) {
                // a stencil plane beyond a wall is the plane itself
                const bool lo = WALL && p.wall && f == 0, hi = WALL && p.wall && f == nm - 1;
                if (WALL && lo) { phl2 = phl1; phi2 = phi1; phr2 = phr1; }
                if (WALL && hi) { phl0 = phl1; phi0 = phi1; phr0 = phr1; }
                const R* s0 = &phi(f & 3, w, lane);
                const R* sm = lo ? s0 : &phi((f - 1) & 3, w, lane);
                const R* sp = hi ? s0 : &phi((f + 1) & 3, w, lane);
                const R d[3] = {phl2, phi2, phr2}, u[3] = {phl0, phi0, phr0}, o[3] = {phl1, phi1, phr1};
                Math::force(p, [&](int a, int b, int m) {
                    if (b != 0) return (m == 0 ? s0 : (m > 0 ? sp : sm))[b * kStride + a];
                    return m < 0 ? d[a + 1] : (m > 0 ? u[a + 1] : o[a + 1]);
                }, rho1, du1);
                us1 = ::fma(du1[2], R(0.5), u1[2]);
                exch(0, f, w) = ::fma(du1[1], R(0.5), u1[1]);
                exch(1, f, w) = T1;
                if (p.chi_mode) exch(2, f, w) = rho1;
            }
            if (i >= zb + 2 && own_row) {
                const int c = i - 2;
                const bool gu = WALL && p.wall && c == nm - 1, gd = WALL && p.wall && c == 0;
                const R half = R(0.5), usa = ::fma(du2[0], half, u2[0]);
                typename Math::Axis ax[3];
                ax[0] = {__shfl_down_sync(0xffffffffu, usa, 1), __shfl_up_sync(0xffffffffu, usa, 1), T2, T2, rho2, rho2};
                ax[1] = {exch(0, c, w + 1), exch(0, c, w - 1), T2, T2, rho2, rho2};
                ax[2] = {gu ? -us2 : us1, gd ? -us2 : us3, T2, T2, rho2, rho2};
                if (p.conduction) {
                    ax[0].Tu = __shfl_down_sync(0xffffffffu, T2, 1);
                    ax[0].Td = __shfl_up_sync(0xffffffffu, T2, 1);
                    ax[1].Tu = exch(1, c, w + 1);
                    ax[1].Td = exch(1, c, w - 1);
                    ax[2].Tu = gu ? (p.T_fixed_hi ? R(2) * p.T_hi - T2 : T2) : T1;
                    ax[2].Td = gd ? (p.T_fixed_lo ? R(2) * p.T_lo - T2 : T2) : T3;
                    if (p.chi_mode) {
                        ax[0].ru = __shfl_down_sync(0xffffffffu, rho2, 1);
                        ax[0].rd = __shfl_up_sync(0xffffffffu, rho2, 1);
                        ax[1].ru = exch(2, c, w + 1);
                        ax[1].rd = exch(2, c, w - 1);
                        if (!gu) ax[2].ru = rho1;
                        if (!gd) ax[2].rd = rho3;
                    }
                }
                if (WALL && (low_y || high_y)) {   // ghosts beyond walls on y
                    const R own = -::fma(du2[1], half, u2[1]);
                    if (high_y) { ax[1].uu = own; ax[1].Tu = p.T_fixed_y[1] ? R(2) * p.T_y[1] - T2 : T2; ax[1].ru = rho2; }
                    if (low_y) { ax[1].ud = own; ax[1].Td = p.T_fixed_y[0] ? R(2) * p.T_y[0] - T2 : T2; ax[1].rd = rho2; }
                }
                if (owns) {
                    const R dE = Math::energy_change(p, rho2, T2, P2, ax, 3);
                    const bool clamp = Math::potential(rho2, P2) >= R(0), bad = !(Math::positive(rho2) && Math::positive(E2));
                    if (clamp || bad) {
                        if (clamp) atomicAdd(&cnt->clamps, 1ull);
                        if (bad) atomicAdd(&cnt->bad, 1ull);
                    }
                    const int n = c * plane_n + n_ab;
                    const int dM_m = (c == 0 ? nm - 1 : -1) * plane_n, dM_p = (c == nm - 1 ? 1 - nm : 1) * plane_n;
                    const unsigned nbits = Store<S, R>::kStochastic ? node_bits(step, (unsigned)n) : 0u;
                    const Pop<S>* q = ring + done * (Q * 32);
                    Pop<S>* dk = dst + n;
                    auto push = [&](auto wall_tag) {
                        constexpr bool BOUNCE = decltype(wall_tag)::value;
                        Math::collide(p, rho2, E2, u2, du2, dE, [&](int k) { return q[k * 32]; }, [&](int k, Two<R> v) {
                            int to = 0;
                            if (M::a(k) == 1) to += dA_p; else if (M::a(k) == -1) to += dA_m;
                            if (M::b(k) == 1) to += dB_p; else if (M::b(k) == -1) to += dB_m;
                            if (M::m(k) == 1) to += dM_p; else if (M::m(k) == -1) to += dM_m;
                            // halfway bounce-back: the pair stays at its node, in the opposite direction
                            const bool bounce = BOUNCE && ((M::m(k) == -1 && gd) || (M::m(k) == 1 && gu) ||
                                                           (M::b(k) == -1 && low_y) || (M::b(k) == 1 && high_y));
                            const long long off = bounce ? (long long)(opposite(k) - k) * (long long)nn : (long long)to;
                            store_pop(dk + off, 0, v, Store<S, R>::kStochastic ? pair_word(nbits, k) : 0u);
                            dk += nn;
                        });
                    };
                    if (WALL && (gu || gd || low_y || high_y)) push(std::true_type{});
                    else push(std::false_type{});
                }
                done = done + 1 == held ? 0 : done + 1;
            } else if (i >= zb) {
                done = done + 1 == held ? 0 : done + 1;
            }
            load(i + kAhead, put);
            put = put + 1 == held ? 0 : put + 1;
            phi2 = phi1; phi1 = phi0; phl2 = phl1; phl1 = phl0; phr2 = phr1; phr1 = phr0;
            rho3 = rho2; rho2 = rho1; rho1 = rho0; T3 = T2; T2 = T1; T1 = T0;
            E2 = E1; E1 = E0; P2 = P1; P1 = P0; us3 = us2; us2 = us1;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                u2[a] = u1[a];
                u1[a] = u0[a];
                du2[a] = du1[a];
            }
        }
    }
};

// Rows a CTA collides and planes loaded ahead: what 227 KB hold with two planes
// ahead.  384 x 384 x 256 in chunks of 64 planes (the planned chunks are faster,
// see above), us per step: FP32 9 rows 2361, 8 rows 2418, 7 rows
// 2560, 6 rows with three planes ahead 2684, 10 rows with one 3470; FP16 16
// rows 1830, 14 rows 2001, 18 rows 2671 (registers), 12 rows with three ahead
// 1905.
template <typename S> struct RowShape;
template <> struct RowShape<float> { static constexpr int TY = 9, AHEAD = 2; };
template <> struct RowShape<__half> { static constexpr int TY = 16, AHEAD = 2; };

// CTA (x, y, z) takes columns from 28 x, rows from TY y and the z-th chunk of
// planes.  WALL: the domain has walls on y or z (x is periodic).
template <typename S, typename R, bool WALL>
__global__ void __launch_bounds__(32 * (RowShape<S>::TY + 4), 1)
    row_march_kernel(const S* src, S* dst, const __grid_constant__ KParams<R> p, MarchGeom G,
                     Counters* cnt) {
    using Sh = RowShape<S>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int zb = G.m_lo + blockIdx.z * G.chunk;
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the previous step's stores
    const int ze = min(zb + G.chunk, G.m_hi), a0 = blockIdx.x * kStripCols, b0 = blockIdx.y * Sh::TY;
    // a CTA none of whose ring nodes lies beyond a wall takes the periodic code
    // (384 x 384 x 256 between walls on z: FP32 2377 -> 2340 us, FP16 1851 -> 1790;
    // periodic 2325 and 1720)
    const bool walled = WALL && ((p.wall && (zb < 2 || ze + 2 > G.nm)) || (p.wall_y && (b0 < 2 || b0 + Sh::TY + 2 > G.nb)));
    if (WALL && walled) {
        RowMarch<S, R, Sh::TY, Sh::AHEAD, true> r(src, dst, p, cnt, G, a0, b0, zb, ze, p.step, smem_raw);
        r.run();
    } else {
        RowMarch<S, R, Sh::TY, Sh::AHEAD, false> r(src, dst, p, cnt, G, a0, b0, zb, ze, p.step, smem_raw);
        r.run();
    }
}

}  // namespace lbm

// Fused one-launch time step of the thermal multiphase LB method
// (arXiv:1705.10045): every node's 2Q populations are read from HBM and its
// 2Q post-collision populations written once per step.
//
// Why a march: the energy change dE at x needs u* at x +- e_a, u* needs the
// force there, and the force needs Phi one node further out, so one step of a
// node depends on the moments of a 2-ring around it.  A CTA owns a TX x TY
// tile of the plane normal to the last lattice axis (z for D3Q19, y for D2Q9)
// and marches along that axis through a chunk of planes.  Three stages work
// on a plane each:
//   M: loads the populations of the (TX+4) x (TY+4) ring region of a plane,
//      keeps Phi on that region and rho, u, T on the (TX+2) x (TY+2) 1-ring
//      region in shared-memory plane buffers;
//   F: computes du = F/rho (Sec. 3 force + gravity) on the 1-ring region;
//   C: for the TX x TY nodes of a plane forms dE by finite differences,
//      reloads the node's populations (an L2 hit: the M stage read them a few
//      planes earlier), collides N and g and pushes them to x + c_k.
// The CTA is warp-specialised: producer warps run M on plane i and F on
// plane i-1 while consumer warps (one thread per tile node) run C on plane
// i-3 or later, so population loads overlap the collision arithmetic.  The
// two roles hand planes over through mbarriers in shared memory: producers
// release iteration i when M(i) and F(i-1) are done, and consumers release
// plane c when C(c) has read its buffers, which the producers wait for before
// overwriting them.  Neither role waits for the other's whole iteration, so a
// slow plane on one side does not stall the other.  A named barrier orders M
// before F, and F before the next M, inside the producer warps.  Ring nodes
// are recomputed by neighbouring CTAs from L2 rather than exchanged.  D2Q9
// runs the same code as a lattice with one y node: its lattice y axis is the
// march axis and its tile is TX x 1 (the fault-injection form only; D2Q9
// otherwise steps strips, strip.cuh, or phases).  Batches of D3Q19 domains run
// it, and the single FP32 and FP16 domains for which it is modelled faster
// than rows.cuh and phases.cuh (plan.h).
//
// Index arithmetic is kept out of the inner loops: the wrapped ring
// coordinates of a CTA are tabulated once in shared memory, buffer slots come
// from one remainder per plane, pair pointers walk from one direction's array
// to the next, and each consumer thread precomputes the +-1 node offsets of
// its node along every axis.  The force stencil and the collision (node.cuh)
// work on opposite-direction pairs (c_{k+1} = -c_k), which share the even part
// of every term, and the collision on both sets at once (f32x2).  384 x 384 x
// 256 D3Q19, a remainder per buffer access and scalar arithmetic -> this: FP32
// 2628 -> 2545 us (43.3 -> 38.7 warp instructions per node), FP16 storage
// 2175 -> 2014 (46.5 -> 42.1).  Carrying the slots from plane to plane instead
// spilled (80 registers): 2728 / 2152.
#pragma once

#include "node.cuh"
#include "plan.h"
#include "strip.cuh"

namespace lbm {

// mbarrier helpers of the producer/consumer hand-off (shared memory, CTA scope)
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
// Wait until the phase of parity `parity` of *b has completed, for at most
// about half a second (1e9 clock cycles); false when the wait gave up.  Each
// try_wait may suspend the warp for up to kWaitHintNs nanoseconds; it resumes
// as soon as the phase completes, so the hint bounds how often a waiting warp
// polls (and takes issue slots from the working warps), not its latency.
#ifndef LBM_WAIT_HINT_NS
#define LBM_WAIT_HINT_NS 20000
#endif
constexpr unsigned kWaitHintNs = LBM_WAIT_HINT_NS;

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* b, unsigned parity) {
    unsigned done;
    if (kWaitHintNs > 0) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_addr(b)), "r"(parity), "n"(kWaitHintNs)
            : "memory");
    } else {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_addr(b)), "r"(parity)
            : "memory");
    }
    return done != 0;
}

__device__ __forceinline__ bool mbar_wait(unsigned long long* b, unsigned parity) {
    if (mbar_try_wait(b, parity)) return true;
    const long long t0 = clock64();
    do {
        if (mbar_try_wait(b, parity)) return true;
    } while (clock64() - t0 < 1000000000ll);
    return false;
}

// Plane buffers: Phi for 3 planes, rho/u/T for 5 planes, du for 4 planes
// (the consumer trails the producer by three planes).  SPLIT: the consumers
// form the moments of their own nodes three planes ahead, which takes one
// more rho/u/T plane and a third mbarrier ring.
template <int TX, int TY, bool SPLIT = false> struct FusedShape {
    static constexpr int RB = TY > 1 ? 2 : 0;           // ring width across b (none for D2Q9)
    static constexpr int RW = TX + 4;                   // 2-ring region (Phi)
    static constexpr int RH = TY + 2 * RB;
    static constexpr int R = RW * RH;
    static constexpr int FB = RB / 2;                   // 1-ring region (rho, u, T, du)
    static constexpr int FW = TX + 2;
    static constexpr int FH = TY + 2 * FB;
    static constexpr int F = FW * FH;
    static constexpr int kRut = 5;                      // rho, ua, ub, um, T
    static constexpr int kPhiSlots = 3, kRutSlots = SPLIT ? 6 : 5, kDuSlots = 4;
    static constexpr int kHandSlots = 8;   // mbarrier ring of the producer/consumer hand-off
    static constexpr int kRings = SPLIT ? 3 : 2;
    // ring nodes outside the tile: RB full rows above and below, 2 columns
    // left and right of each tile row
    static constexpr int kBorder = 2 * RB * RW + 4 * TY;
    template <typename R_> static constexpr size_t table_offset() {
        return sizeof(R_) * ((size_t)kPhiSlots * R + (size_t)kRutSlots * kRut * F + (size_t)kDuSlots * 3 * F);
    }
    template <typename R_> static constexpr size_t barrier_offset() {
        return (table_offset<R_>() + sizeof(int) * (RW + RH) + 7) & ~(size_t)7;
    }
    // plane buffers, ring tables, kRings x kHandSlots mbarriers and an abort flag
    template <typename R_> static constexpr size_t smem_bytes() {
        return barrier_offset<R_>() + 8 * (kRings * kHandSlots + 1);
    }
    // ring index of border node q < kBorder
    __device__ static int border_ring(int q) {
        if (q < 2 * RB * RW) {
            const int row = q / RW;
            return (row < RB ? row : row + TY) * RW + q % RW;
        }
        const int q2 = q - 2 * RB * RW, c = q2 & 3;
        return (RB + (q2 >> 2)) * RW + (c < 2 ? c : c + TX);
    }
};

__device__ __forceinline__ int wrapi(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

// Coordinate of a ring row or column: wrapped on a periodic axis, the mirror
// node across a wall (clamped into the axis for ring nodes of a ragged tile
// that lie further out; their values are never used).
__device__ __forceinline__ int ring_coord(int i, int n, int walled) {
    if (!walled) return wrapi(i, n);
    if (i < 0) i = -1 - i;
    if (i >= n) i = 2 * n - 1 - i;
    return i < 0 ? 0 : (i >= n ? n - 1 : i);
}

// Walls beside tile-plane node (ga, gb): bit 0 / 1 the low / high wall of axis
// a (x), bit 2 / 3 of axis b (y of D3Q19).
template <typename R>
__device__ __forceinline__ int wall_edges(const KParams<R>& p, int Q, int ga, int gb, int na, int nb) {
    int e = 0;
    if (p.wall_x) e |= (ga == 0 ? 1 : 0) | (ga == na - 1 ? 2 : 0);
    if (Q == 19 && p.wall_y) e |= (gb == 0 ? 4 : 0) | (gb == nb - 1 ? 8 : 0);
    return e;
}

// COH: read the populations through coherent loads (the persistent batch
// kernel reads, in one launch, buffers that other CTAs wrote earlier in it).
template <int Q, typename S, typename R, int TX, int TY, bool COH = false, bool SPLIT = false> struct FusedStages {
    using V = Vel<Q>;
    using M = MVel<Q>;
    using Math = NodeMath<Q, S, R>;
    using Sh = FusedShape<TX, TY, SPLIT>;
    static constexpr int RB = Sh::RB, RW = Sh::RW, RH = Sh::RH, R_ = Sh::R, FW = Sh::FW, FB = Sh::FB, F_ = Sh::F;

    R* phis;     // [kPhiSlots][R_]
    R* ruts;     // [kRutSlots][kRut][F_]
    R* dus;      // [kDuSlots][3][F_]
    int* ring_a; // wrapped a of ring column
    int* ring_b; // wrapped b * na of ring row
    const S* __restrict__ src;
    S* __restrict__ dst;
    const KParams<R>* p;
    MarchGeom G;
    size_t nn;
    int plane_n;
    unsigned step;   // step counter of this launch (seeds FP16 stochastic rounding)

    __device__ R& phi(int slot, int r) const { return phis[slot * R_ + r]; }
    __device__ R& rut(int slot, int f, int r) const { return ruts[(slot * Sh::kRut + f) * F_ + r]; }
    __device__ R& du(int slot, int c, int r) const { return dus[(slot * 3 + c) * F_ + r]; }
    // Buffer slots are keyed by the unwrapped plane index the M stage loaded
    // (a periodic plane -1 holds the data of plane nm-1): one remainder per
    // plane, the neighbouring planes' slots from it (a remainder per access
    // would cost a dozen instructions each).
    struct Slots {
        int m, phi, rut;   // plane, its Phi slot and its rho/u/T slot
        __device__ explicit Slots(int plane) : m(plane) {   // plane >= -3
            const unsigned u = (unsigned)(plane + 3 * Sh::kPhiSlots * Sh::kRutSlots);
            phi = (int)(u % Sh::kPhiSlots);
            rut = (int)(u % Sh::kRutSlots);
        }
        static_assert(Sh::kDuSlots == 4, "du slots by mask");
        __device__ int du(int d = 0) const { return (m + d) & 3; }
        __device__ int phi_at(int d) const {   // |d| < kPhiSlots
            const int s = phi + d;
            return s < 0 ? s + Sh::kPhiSlots : (s >= Sh::kPhiSlots ? s - Sh::kPhiSlots : s);
        }
        __device__ int rut_at(int d) const {   // |d| < kRutSlots
            const int s = rut + d;
            return s < 0 ? s + Sh::kRutSlots : (s >= Sh::kRutSlots ? s - Sh::kRutSlots : s);
        }
    };

    // M: moments of plane sl.m on the ring region, ring nodes t, t + nt, ...
    __device__ void m_stage(const Slots& sl, int plane_off, int t, int nt) const {
        for (int r = t; r < R_; r += nt) m_ring(sl.phi, sl.rut, plane_off, r);
    }
    // the same for the border nodes only (SPLIT: the consumers take the tile)
    __device__ void m_border(const Slots& sl, int plane_off, int t, int nt) const {
        for (int q = t; q < Sh::kBorder; q += nt) m_ring(sl.phi, sl.rut, plane_off, Sh::border_ring(q));
    }
    __device__ __forceinline__ void m_ring(int sp, int sr, int plane_off, int r) const {
        const int ra = r % RW, rb = r / RW, fa = ra - 1, fb = rb - (RB - FB);
        const bool inner = fa >= 0 && fa < FW && fb >= 0 && fb < Sh::FH;
        m_node<kUse>(plane_off + ring_b[rb] + ring_a[ra], sp, sr, r, inner ? fb * FW + fa : -1);
    }
    // Moments of node n: Phi at ring index r, and rho, u, T at 1-ring index f
    // (f < 0: the node lies outside the 1-ring region).
    template <LoadUse U> __device__ __forceinline__ void m_node(int n, int sp, int sr, int r, int f) const {
        Pop<S> w[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k] = load_pop<COH, U>(src + 2 * ((size_t)k * nn), (size_t)(unsigned)n);
        const Moments<R> o = Math::moments(w, *p);
        const R T = o.E / (o.rho * p->c_v);
        phi(sp, r) = Math::phi_of(Math::potential(o.rho, eos_pressure(*p, o.rho, T)));
        if (f >= 0) {
            const R inv = R(1) / o.rho;
            rut(sr, 0, f) = o.rho;
            rut(sr, 1, f) = o.ja * inv;
            rut(sr, 2, f) = o.jb * inv;
            rut(sr, 3, f) = o.jm * inv;
            rut(sr, 4, f) = T;
        }
    }

    // F: du = F/rho on the 1-ring region of plane sl.m, region nodes t, t + nt, ...
    // Across a wall the stencil reads the mirror plane, the plane itself.
    __device__ void f_stage(const Slots& sl, int t, int nt) const {
        const int sp0 = sl.phi, spm = p->wall && sl.m == 0 ? sp0 : sl.phi_at(-1),
                  spp = p->wall && sl.m == G.nm - 1 ? sp0 : sl.phi_at(1);
        const int sd = sl.du();
        for (int r = t; r < F_; r += nt) {
            const int at = (r / FW + (RB - FB)) * RW + r % FW + 1;
            R d[3];
            Math::force(*p, [&](int a, int b, int m) {
                return phi(m == 0 ? sp0 : (m > 0 ? spp : spm), at + b * RW + a);
            }, rut(sl.rut, 0, r), d);
            du(sd, 0, r) = d[0];
            du(sd, 1, r) = d[1];
            du(sd, 2, r) = d[2];
        }
    }

    // C: energy change, collision and push of the node at 1-ring index fc and
    // index n_ab of its plane, plane sl.m.
    // edge: walls next to the node across the tile plane (bit 0 / 1: the low /
    // high wall of axis a, bit 2 / 3: of axis b), from wall_edges().
    // XW: the domain may have walls on the tile-plane axes (false: edge is 0
    // and the wall handling across the tile compiles away).
    template <bool XW>
    __device__ void c_stage(const Slots& sl, int fc, int n_ab, int dA_m, int dA_p, int dB_m, int dB_p,
                            int edge_in, Counters* cnt) const {
        const int edge = XW ? edge_in : 0, c = sl.m;
        const int nm = G.nm;
        const bool gu = p->wall && c == nm - 1, gd = p->wall && c == 0;
        // the node's populations first: their loads are in flight while the
        // finite differences below read shared memory.  The reload is the last
        // use of these lines on this SM, so it does not allocate them in L1.
        // With FP16 storage it stays packed (one 32-bit word per pair) and
        // each half is widened where it is used.
        const int n = c * plane_n + n_ab;
        Pop<S> w[Q];
        const S* q = src + 2 * (size_t)n;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            w[k] = load_pop<COH, kUseLast>(q, 0);
            q += 2 * nn;
        }
        const int sr = sl.rut, sd = sl.du();
        const R rho = rut(sr, 0, fc), T = rut(sr, 4, fc);
        const R u[3] = {rut(sr, 1, fc), rut(sr, 2, fc), rut(sr, 3, fc)};
        const R dv[3] = {du(sd, 0, fc), du(sd, 1, fc), du(sd, 2, fc)};

        // finite-difference neighbours along a, b and the march axis: ring
        // nodes, or (only for nodes beside a wall) the node itself mirrored
        // across it: normal velocity negated, T mirrored or reflected about
        // the wall temperature
        constexpr int N = V::D;
        typename Math::Axis ax[N];
        auto across = [&](int j, int a, int step, int g, const int* fixed, const R* Tw) {
            ax[j] = {::fma(du(sd, a, fc + step), R(0.5), rut(sr, 1 + a, fc + step)),
                     ::fma(du(sd, a, fc - step), R(0.5), rut(sr, 1 + a, fc - step)), rut(sr, 4, fc + step),
                     rut(sr, 4, fc - step), rut(sr, 0, fc + step), rut(sr, 0, fc - step)};
            if (g) {
                const R own = -::fma(dv[a], R(0.5), u[a]);
                if (g & 2) { ax[j].uu = own; ax[j].Tu = fixed[1] ? R(2) * Tw[1] - T : T; ax[j].ru = rho; }
                if (g & 1) { ax[j].ud = own; ax[j].Td = fixed[0] ? R(2) * Tw[0] - T : T; ax[j].rd = rho; }
            }
        };
        across(0, 0, 1, edge & 3, p->T_fixed_x, p->T_x);
        if (Q == 19) across(1, 1, FW, (edge >> 2) & 3, p->T_fixed_y, p->T_y);
        {
            const int su = sl.rut_at(1), sdn = sl.rut_at(-1), du_u = sl.du(1), du_d = sl.du(-1);
            const R own = -::fma(dv[2], R(0.5), u[2]);
            ax[N - 1].uu = gu ? own : ::fma(du(du_u, 2, fc), R(0.5), rut(su, 3, fc));
            ax[N - 1].ud = gd ? own : ::fma(du(du_d, 2, fc), R(0.5), rut(sdn, 3, fc));
            ax[N - 1].Tu = gu ? (p->T_fixed_hi ? R(2) * p->T_hi - T : T) : rut(su, 4, fc);
            ax[N - 1].Td = gd ? (p->T_fixed_lo ? R(2) * p->T_lo - T : T) : rut(sdn, 4, fc);
            ax[N - 1].ru = gu ? rho : rut(su, 0, fc);
            ax[N - 1].rd = gd ? rho : rut(sdn, 0, fc);
        }
        const R P = eos_pressure(*p, rho, T);
        const R dE = Math::energy_change(*p, rho, T, P, ax, N);
        const R E = Math::energy(w, *p);
        const bool clamp = Math::potential(rho, P) >= R(0), bad = !(Math::positive(rho) && Math::positive(E));
        if (clamp || bad) {
            if (clamp) atomicAdd(&cnt->clamps, 1ull);
            if (bad) atomicAdd(&cnt->bad, 1ull);
        }

        // node offsets of x + c_k: +-1 along a and b (periodic), along the
        // march axis periodic or bounced at a wall
        const int dM_m = (c == 0 ? nm - 1 : -1) * plane_n, dM_p = (c == nm - 1 ? 1 - nm : 1) * plane_n;
        const unsigned nbits = Store<S, R>::kStochastic ? node_bits(step, (unsigned)n) : 0u;
        Pop<S>* out = reinterpret_cast<Pop<S>*>(dst);
        Pop<S>* dk = out + n;
        // the collision and push, instantiated once for planes next to a wall
        // (WALL: some directions bounce back) and once for all other planes
        auto collide = [&](auto wall_tag) {
            constexpr bool WALL = decltype(wall_tag)::value;
            Math::collide(*p, rho, E, u, dv, dE, [&](int k) { return w[k]; }, [&](int k, Two<R> v) {
                // push to x + c_k, or bounce back at a wall
                const bool bounce = WALL && ((M::m(k) == -1 && gd) || (M::m(k) == 1 && gu) ||
                                             (M::a(k) == -1 && (edge & 1)) || (M::a(k) == 1 && (edge & 2)) ||
                                             (M::b(k) == -1 && (edge & 4)) || (M::b(k) == 1 && (edge & 8)));
                int to = 0;
                if (M::a(k) == 1) to += dA_p; else if (M::a(k) == -1) to += dA_m;
                if (M::b(k) == 1) to += dB_p; else if (M::b(k) == -1) to += dB_m;
                if (M::m(k) == 1) to += dM_p; else if (M::m(k) == -1) to += dM_m;
                const unsigned t = Store<S, R>::kStochastic ? pair_word(nbits, k) : 0u;
                const long long off = bounce ? (long long)(opposite(k) - k) * (long long)nn : (long long)to;
                store_pop(dk + off, 0, v, t);
                dk += nn;
            });
        };
        if (gu || gd || edge) collide(std::true_type{});
        else collide(std::false_type{});
    }
};

// One CTA of the producer/consumer fused step: the tile (a0, b0) of planes
// [zb, zb + G.chunk) of one domain.  Threads [0, TX*TY) are consumers (one per
// tile node), threads [TX*TY, TX*TY + NP) producers.
// FAULT instantiates the fault-injection form: the first CTA withholds the
// hand-off of plane fault_plane (tests of the bounded waits only).
template <int Q, typename S, typename R, int TX, int TY, int NP, bool FAULT = false, bool COH = false,
          bool XW = true, bool SPLIT = false>
__device__ __forceinline__ void fused_tile(const S* __restrict__ src, S* __restrict__ dst, const KParams<R>* p,
                                           const MarchGeom& G, unsigned step, int a0, int b0, int zb,
                                           Counters* cnt, unsigned char* smem_raw, int fault_plane = -1) {
    using St = FusedStages<Q, S, R, TX, TY, COH, SPLIT>;
    using Sh = typename St::Sh;
    constexpr int NC = TX * TY, NT = NC + NP;
    St st;
    st.phis = reinterpret_cast<R*>(smem_raw);
    st.ruts = st.phis + Sh::kPhiSlots * Sh::R;
    st.dus = st.ruts + Sh::kRutSlots * Sh::kRut * Sh::F;
    st.ring_a = reinterpret_cast<int*>(st.dus + Sh::kDuSlots * 3 * Sh::F);
    st.ring_b = st.ring_a + Sh::RW;
    st.src = src;
    st.dst = dst;
    st.p = p;
    st.G = G;
    st.nn = (size_t)p->nn;
    st.plane_n = G.na * G.nb;
    st.step = step;

    const int tid = threadIdx.x;
    const int ze = min(zb + G.chunk, G.m_hi);
    const bool walls = p->wall;
    const int wa = p->wall_x, wb = Q == 19 ? p->wall_y : 0;
    for (int i = tid; i < Sh::RW; i += NT) st.ring_a[i] = ring_coord(a0 + i - 2, G.na, wa);
    for (int i = tid; i < Sh::RH; i += NT) st.ring_b[i] = ring_coord(b0 + i - Sh::RB, G.nb, wb) * G.na;

    // hand-off ring: full[s] completes when the producers finish iteration u
    // (u = i - zb + 2, s = u mod D); empty[s] when every consumer has finished
    // plane c (u = c - zb).  The k-th use of a slot completes its phase k, so
    // the wait parity is (u / D) & 1; neither side gets two phases ahead of
    // the other's wait (producers run at most 2 iterations ahead of the plane
    // they need released, consumers cannot pass the producers).
    // SPLIT adds mint[s]: every consumer has formed the moments of its node of
    // plane c + 3 (u = c - zb), which the producers' F stage of iteration
    // c + 3 reads.  A consumer forms them right after its wait for iteration
    // c + 2, into buffer slots whose last readers (F(c+1), C(c-2)) that wait
    // has ordered before it; the producers wait on every phase in order.
    constexpr int D = Sh::kHandSlots;
    unsigned long long* full = reinterpret_cast<unsigned long long*>(smem_raw + Sh::template barrier_offset<R>());
    unsigned long long* empty = full + D;
    unsigned long long* mint = empty + D;
    volatile int* aborted = reinterpret_cast<volatile int*>(full + Sh::kRings * D);
    if (tid == 0) {
        *aborted = 0;
        for (int s = 0; s < D; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, NC);
            if (SPLIT) mbar_init(mint + s, NC);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    auto wait = [&](unsigned long long* b, int u) {
        if (*aborted) return;
        if (!mbar_wait(b + (u % D), (unsigned)(u / D) & 1u)) {
            *aborted = 1;
            atomicAdd(&cnt->timeouts, 1ull);
        }
    };

    using Slots = typename St::Slots;
    if (tid >= NC) {
        // producers: iteration i builds M(i) and F(i-1).  M(i) and F(i-1)
        // overwrite the buffers that C(i-4) read last.
        // SPLIT: from plane zb + 3 on the consumers form the tile's moments
        // and the producers the border's.
        const int t = tid - NC;
        int plane = wrapi(zb - 2, G.nm);   // wrapped index of plane i
        for (int i = zb - 2; i < ze + 3; ++i) {
            const int cw = i - 4;
            if (cw >= zb && cw < ze) wait(empty, cw - zb);
            const bool m_need = i <= ze + 1 && (walls ? (i >= 0 && i < G.nm) : true);
            const bool split = SPLIT && i >= zb + 3 && i <= ze + 1;
            if (m_need) {
                const Slots sm(i);
                if (split) st.m_border(sm, plane * st.plane_n, t, NP);
                else st.m_stage(sm, plane * st.plane_n, t, NP);
            }
            if (split) wait(mint, i - zb - 3);
            asm volatile("bar.sync 1, %0;" ::"r"(NP));
            const int f = i - 1;
            const bool f_need = f >= zb - 1 && f <= ze && (walls ? (f >= 0 && f < G.nm) : true);
            if (f_need) st.f_stage(Slots(f), t, NP);
            asm volatile("bar.sync 1, %0;" ::"r"(NP));
            bool withhold = false;
            if constexpr (FAULT) withhold = i == fault_plane && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
            if (t == 0 && !withhold) mbar_arrive(full + ((i - zb + 2) % D));
            plane = plane + 1 == G.nm ? 0 : plane + 1;
        }
    } else {
        // consumers: C(c) needs M(c+2) and F(c+1), i.e. producer iteration c+2
        const int ta = tid % TX, tb = tid / TX;
        const int ga = a0 + ta, gb = b0 + tb;
        const bool owns = ga < G.na && gb < G.nb;
        const int dA_m = ga == 0 ? G.na - 1 : -1, dA_p = ga == G.na - 1 ? 1 - G.na : 1;
        const int dB_m = (gb == 0 ? G.nb - 1 : -1) * G.na, dB_p = (gb == G.nb - 1 ? 1 - G.nb : 1) * G.na;
        const int edge = XW ? wall_edges(*p, Q, ga, gb, G.na, G.nb) : 0;
        // the thread's own ring node: its column of a plane and ring indices
        const int ring_n = st.ring_b[tb + Sh::RB] + st.ring_a[ta + 2];
        const int ring_r = (tb + Sh::RB) * Sh::RW + ta + 2, ring_f = (tb + Sh::FB) * Sh::FW + ta + 1;
        int ahead = wrapi(zb + 3, G.nm);   // wrapped index of plane c + 3
        for (int c = zb; c < ze; ++c) {
            wait(full, c - zb + 4);
            const Slots sl(c);
            if (SPLIT && c + 3 <= ze + 1) {
                if (walls ? c + 3 < G.nm : true)
                    st.template m_node<kUseKeep>(ahead * st.plane_n + ring_n, sl.phi_at(0), sl.rut_at(3), ring_r, ring_f);
                mbar_arrive(mint + ((c - zb) % D));
            }
            if (owns) st.template c_stage<XW>(sl, ring_f, ring_n, dA_m, dA_p, dB_m, dB_p, edge, cnt);
            mbar_arrive(empty + ((c - zb) % D));
            ahead = ahead + 1 == G.nm ? 0 : ahead + 1;
        }
    }
}

// CTAs per SM the single-domain step is compiled for (the register cap that
// follows from it): D3Q19 keeps two 384-thread CTAs (80 registers) with FP32
// and FP16 storage and one 512-thread CTA with FP64; D2Q9 keeps four (FP32)
// or three 288-thread CTAs.
template <int Q, typename S> struct FusedOcc {
    static constexpr int kMinBlocks = Q == 19 ? (sizeof(S) == 8 ? 1 : 2) : (sizeof(S) == 4 ? 4 : 3);
};

// Single-domain fused step: CTA (x, y, z) takes tile (x TX, y TY) and the
// z-th chunk of planes.  XW: instance for domains with walls on the
// tile-plane axes (the other instance carries no trace of them).  SPLIT: the
// consumers form their own nodes' moments (fused_tile).
template <int Q, typename S, typename R, int TX, int TY, int NP, bool XW, bool SPLIT>
__global__ void __launch_bounds__(TX* TY + NP, FusedOcc<Q, S>::kMinBlocks)
    fused_step_kernel(const S* __restrict__ src, S* __restrict__ dst, KParams<R> p, MarchGeom G, Counters* cnt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fused_tile<Q, S, R, TX, TY, NP, false, false, XW, SPLIT>(src, dst, &p, G, p.step, blockIdx.x * TX,
                                                             blockIdx.y * TY, G.m_lo + blockIdx.z * G.chunk, cnt,
                                                             smem_raw);
}

// The same step with the fault-injection hook: the first CTA withholds the
// hand-off of plane fault_plane, so that its consumers' bounded wait runs out
// and the timeout is counted.  Launched only for handles created with
// the test hook lbm_test_drop_handoff set; the kernel above carries no trace
// of it.
template <int Q, typename S, typename R, int TX, int TY, int NP, bool SPLIT>
__global__ void __launch_bounds__(TX* TY + NP, FusedOcc<Q, S>::kMinBlocks)
    fused_step_fault_kernel(const S* __restrict__ src, S* __restrict__ dst, KParams<R> p, MarchGeom G, Counters* cnt,
                            int fault_plane) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fused_tile<Q, S, R, TX, TY, NP, true, false, true, SPLIT>(src, dst, &p, G, p.step, blockIdx.x * TX,
                                                              blockIdx.y * TY, G.m_lo + blockIdx.z * G.chunk, cnt,
                                                              smem_raw, fault_plane);
}

// ---------------------------------------------------------------------------
// Many domains, many steps, one persistent launch.  The work of a request is
// n steps x the table of work items (domain, tile, chunk): work index
// w = s * items + i is step s of item i.  CTAs take work indices in order from
// a global counter.  An item of step s of domain d may start once every item
// of d has finished step s - 1: its CTA waits (bounded) until the domain's
// completion counter reaches s * items(d), reading it with acquire ordering;
// a CTA that finishes an item adds 1 to the counter with release ordering.
// Every item a CTA waits for has a smaller work index, so a CTA that is
// running already holds it, and the waits always end: no deadlock, whatever
// the number of CTAs that are resident.  A domain takes part while s < left
// and reads buffer (cur + s) mod 2.  A wait that gives up counts a timeout
// on the domain and marks it aborted, so that later items of that domain skip
// their waits (and their results, which the latched LBM_ERR_TIMEOUT voids).

struct BatchItem {
    int domain, a0, b0, zb;
};

template <typename R> struct DomainDesc {
    KParams<R> kp;      // kp.step: the domain's step count at s = 0
    MarchGeom G;
    void* pop[2];
    Counters* cnt;
    int cur;            // buffer holding the state at s = 0
    int left;           // steps the domain still takes, counted from s = 0
    int n_items;        // work items of the domain in the table
};

// Scheduling state of a request in device memory: steps, the next work
// index, and per domain a completion counter and an abort flag.
struct BatchSched {
    int n_steps;
    int next;
    int pad[2];
    // followed by unsigned done[domains], int aborted[domains]
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The scheduling loop of a persistent CTA.  work(item, domain, kp, s): step s
// of a work item, by every thread of the CTA; kp: the CTA's copy of the
// domain's parameters.  FAULT: the item fault_item of step 0 does not report
// its completion (tests of the bounded waits only).
template <bool FAULT, typename R, typename W>
__device__ __forceinline__ void batch_loop(const BatchItem* __restrict__ items, const DomainDesc<R>* __restrict__ doms,
                                           int n_items, BatchSched* sched, int n_doms, int fault_item, const W& work) {
    __shared__ KParams<R> kp;   // the current item's domain parameters
    __shared__ int w_sh, go_sh;
    int kp_domain = -1;         // domain whose parameters kp holds (thread 0)
    unsigned* done = reinterpret_cast<unsigned*>(sched + 1);
    int* aborted = reinterpret_cast<int*>(done + n_doms);
    const long long total = (long long)sched->n_steps * n_items;
    for (;;) {
        if (threadIdx.x == 0) w_sh = atomicAdd(&sched->next, 1);
        __syncthreads();
        const long long w = w_sh;
        if (w >= total || w < 0) break;
        const int s = (int)(w / n_items), i = (int)(w % n_items);
        const BatchItem it = items[i];
        const DomainDesc<R>* d = doms + it.domain;
        const bool active = s < d->left;
        if (active && threadIdx.x == 0) {
            if (kp_domain != it.domain) {   // consecutive items mostly share a domain
                kp = d->kp;
                kp_domain = it.domain;
            }
            int go = 1;
            if (s > 0) {
                const unsigned target = (unsigned)s * (unsigned)d->n_items;
                const long long t0 = clock64();
                while (ld_acquire_u32(done + it.domain) < target) {
                    if (*(volatile int*)(aborted + it.domain)) {
                        go = 0;
                        break;
                    }
                    if (clock64() - t0 > 1000000000ll) {   // about half a second
                        atomicExch(aborted + it.domain, 1);
                        atomicAdd(&d->cnt->timeouts, 1ull);
                        go = 0;
                        break;
                    }
                }
            }
            go_sh = go;
        }
        __syncthreads();
        if (active && go_sh) work(it, d, kp, s);
        __syncthreads();
        if (active && threadIdx.x == 0) {
            bool report = true;
            if constexpr (FAULT) report = !(s == 0 && i == fault_item);
            if (report) {
                __threadfence();   // release: the item's stores before its completion
                atomicAdd(done + it.domain, 1u);
            }
        }
    }
}

// Items are tiles and chunks of planes of the march.  XW: some domain has
// walls on the tile-plane axes.  SPLIT: the consumers form their own nodes'
// moments.
template <int Q, typename S, typename R, int TX, int TY, int NP, int MB, bool FAULT, bool XW, bool SPLIT>
__global__ void __launch_bounds__(TX* TY + NP, MB) fused_batch_kernel(const BatchItem* __restrict__ items,
                                                                  const DomainDesc<R>* __restrict__ doms,
                                                                  int n_items, BatchSched* sched, int n_doms,
                                                                  int fault_item) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    batch_loop<FAULT, R>(items, doms, n_items, sched, n_doms, fault_item,
                         [&](const BatchItem& it, const DomainDesc<R>* d, const KParams<R>& kp, int s) {
        const int in = (d->cur + s) & 1;
        const MarchGeom G = d->G;
        fused_tile<Q, S, R, TX, TY, NP, false, true, XW, SPLIT>((const S*)d->pop[in], (S*)d->pop[in ^ 1], &kp, G,
                                                     kp.step + (unsigned)s, it.a0, it.b0, it.zb, d->cnt, smem_raw);
    });
}

// D2Q9: items are groups of W strips of a domain (strip.cuh), numbered strip
// first, then chunk of rows; it.a0 is the first of the group.  Strips copy
// their rows with cp.async, which reads what the domain's other CTAs wrote in
// the previous step: every thread issues it after the acquire that the CTA's
// first thread made and the barrier behind it.
template <typename S, typename R, int W, int MB, bool FAULT, bool WALL>
__global__ void __launch_bounds__(32 * W, MB) strip_batch_kernel(const BatchItem* __restrict__ items,
                                                                 const DomainDesc<R>* __restrict__ doms, int n_items,
                                                                 BatchSched* sched, int n_doms, int fault_item) {
    using St = Strip<S, R, WALL>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5;
    batch_loop<FAULT, R>(items, doms, n_items, sched, n_doms, fault_item,
                         [&](const BatchItem& it, const DomainDesc<R>* d, const KParams<R>& kp, int s) {
        const MarchGeom G = d->G;
        const int strips = strip_count(G.na), w = it.a0 + warp, zb = (w / strips) * G.chunk;
        if (zb >= G.nm) return;
        const int in = (d->cur + s) & 1;
        St st((const S*)d->pop[in], (S*)d->pop[in ^ 1], kp, d->cnt, G.na, G.nm, zb, min(zb + G.chunk, G.nm),
              kp.step + (unsigned)s, (w % strips) * St::kCols,
              reinterpret_cast<Pop<S>*>(smem_raw + warp * St::kRingBytes));
        st.run();
    });
}

// descriptor bookkeeping after a request of n steps: every domain took
// min(n, left) steps
template <typename R> __global__ void batch_advance_kernel(DomainDesc<R>* doms, int count, const BatchSched* sched) {
    const int n = sched->n_steps;
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < count; d += gridDim.x * blockDim.x) {
        const int taken = doms[d].left < n ? doms[d].left : n;
        doms[d].cur ^= taken & 1;
        doms[d].kp.step += (unsigned)taken;
        doms[d].left -= taken;
    }
}

}  // namespace lbm

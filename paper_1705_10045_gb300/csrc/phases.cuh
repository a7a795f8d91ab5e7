// One time step as three launches over all nodes, each value formed once:
//   phase_moments   rho, u, T, Phi (fields) and E, P (kept where the step writes) of every node
//   phase_force     du = F/rho
//   phase_collide   dE, collision, push
// with the fields in device memory between them.
//
// For FP64, and for small D3Q19 domains.  A GB300 issues FP64 at two lanes per
// clock and SM (492 G lanes/s measured, 64 cycles latency), so an FP64 step is
// bound by its FP64 instructions (about 430 a node on D3Q19, 240 on D2Q9), not by memory: 0.8 ns
// a node against 0.1 ns for the 608 bytes of populations.  The fused march
// (fused.cuh) recomputes the moments and forces of every tile's ring, which
// saves bytes that are free here and costs instructions that are not; it also
// needs tiles to fill the chip.  Field traffic (13 values a node) is nothing
// beside the arithmetic.  The per-node arithmetic is the march's
// (node.cuh): the two forms agree bit for bit.  Measured, march -> phases, us
// per step: D2Q9 128 x 128 125 -> 14.2, a row of 128 nodes 35 -> 12.7, D3Q19
// 90 x 75 x 67 with walls on every axis 1050 -> 387 (its FP64 instructions
// need about that at the measured rate).  Reciprocals for the divisions and
// shorter chains of additions would give 12.6 and 356, with other rounding.
//
// In FP32 and FP16 storage the populations are read twice and the fields add
// traffic (about 93 ps a node against the march's 56), but every node has its
// own thread and no plane waits for another: domains too small to fill 152 SMs
// with marching CTAs step faster this way (the rule and figures stand in
// backend.cuh).
//
// Each launch starts while the one before it still writes (backend.cuh,
// launch_after), so what a launch reads is not constant for its whole life:
// populations and fields come through coherent loads behind
// griddepcontrol.wait, never through const __restrict__ pointers.
#pragma once

#include "node.cuh"

namespace lbm {

// E and P of a node wait for its collision in the buffer the step writes: the
// pair of direction 0 stays at its node, so nothing but the node's own
// collision writes it.  Only nodes the launch collides use it (the others'
// pairs may be in place already, from another range of the same step).  A pair
// of FP16 storage holds E alone; P follows from rho and T as it did before.
__device__ __forceinline__ void put_scratch(Pop<float>* q, float E, float P) { q->v = make_float2(E, P); }
__device__ __forceinline__ void put_scratch(Pop<double>* q, double E, double P) { q->v = make_double2(E, P); }
__device__ __forceinline__ void put_scratch(Pop<__half>* q, float E, float) { q->v = __float_as_uint(E); }
template <typename R> struct EnergyPressure {
    R E, P;
};
__device__ __forceinline__ EnergyPressure<float> get_scratch(const Pop<float>* q, const KParams<float>&, float, float) {
    return {q->v.x, q->v.y};
}
__device__ __forceinline__ EnergyPressure<double> get_scratch(const Pop<double>* q, const KParams<double>&, double, double) {
    return {q->v.x, q->v.y};
}
__device__ __forceinline__ EnergyPressure<float> get_scratch(const Pop<__half>* q, const KParams<float>& p, float rho, float T) {
    return {__uint_as_float(q->v), eos_pressure(p, rho, T)};
}

struct PhaseGeom {
    int plane_n, nm;       // nodes of a plane of the last axis, planes
    int first, count;      // planes of the launch, from plane `first` (wrapped)
    int m_lo, m_hi;        // planes the step collides (their nodes count clamps and bad states)
};

template <int Q, typename S, typename R> struct Phase {
    using V = Vel<Q>;
    using M = MVel<Q>;
    using Math = NodeMath<Q, S, R>;
    static constexpr int D = V::D;
    using Steps = NodeSteps<Q, R>;

    // node of this thread, or -1
    __device__ static __forceinline__ int node(const PhaseGeom& G) {
        const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
        if (t >= (unsigned)G.count * (unsigned)G.plane_n) return -1;
        const unsigned all = (unsigned)G.nm * (unsigned)G.plane_n, n = (unsigned)G.first * (unsigned)G.plane_n + t;
        return (int)(n >= all ? n - all : n);
    }
    // lattice axis of march axis 0 (a), 1 (b), 2 (m)
    __device__ static constexpr int axis(int march) { return Q == 9 && march == 2 ? 1 : march; }
    __device__ static constexpr int vel(int k, int a) { return a == 0 ? V::cx(k) : (a == 1 ? V::cy(k) : V::cz(k)); }
};

template <int Q, typename S, typename R>
__global__ void __launch_bounds__(128) phase_moments_kernel(const S* src, S* dst, R* fld,
                                                            const __grid_constant__ KParams<R> p,
                                                            PhaseGeom G, Counters* cnt) {
    using Math = NodeMath<Q, S, R>;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = Phase<Q, S, R>::node(G);
    if (n < 0) return;
    const size_t nn = (size_t)p.nn;
    Pop<S> f[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) f[k] = load_pop<true>(src + 2 * ((size_t)k * nn), (size_t)n);
    const Moments<R> o = Math::moments(f, p);
    const R inv = R(1) / o.rho;
    const R T = o.E / (o.rho * p.c_v), P = eos_pressure(p, o.rho, T);
    const R U = Math::potential(o.rho, P);
    fld[F_RHO * nn + n] = o.rho;
    fld[F_UX * nn + n] = o.ja * inv;
    fld[F_UY * nn + n] = (Q == 9 ? o.jm : o.jb) * inv;
    if (Q == 19) fld[F_UZ * nn + n] = o.jm * inv;
    fld[F_T * nn + n] = T;
    fld[F_PHI * nn + n] = Math::phi_of(U);
    if (n < G.m_lo * G.plane_n || n >= G.m_hi * G.plane_n) return;
    put_scratch(reinterpret_cast<Pop<S>*>(dst) + n, o.E, P);
    // counted once a step, with the plane's collision
    if (U >= R(0)) atomicAdd(&cnt->clamps, 1ull);
    if (!(Math::positive(o.rho) && Math::positive(o.E))) atomicAdd(&cnt->bad, 1ull);
}

template <int Q, typename S, typename R>
__global__ void __launch_bounds__(128) phase_force_kernel(R* fld, const __grid_constant__ KParams<R> p, PhaseGeom G) {
    using Ph = Phase<Q, S, R>;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = Ph::node(G);
    if (n < 0) return;
    const size_t nn = (size_t)p.nn;
    const typename Ph::Steps s(p, n);
    const R* phi = fld + F_PHI * nn;
    R du[3];
    NodeMath<Q, S, R>::force(p, [&](int a, int b, int m) {
        int to = n;
        const int c[3] = {a, b, m};
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (c[j] != 0) to += c[j] > 0 ? s.hi[Ph::axis(j)] : s.lo[Ph::axis(j)];
        return phi[to];
    }, fld[F_RHO * nn + n], du);
    fld[F_DUX * nn + n] = du[0];
    fld[F_DUY * nn + n] = Q == 9 ? du[2] : du[1];
    if (Q == 19) fld[F_DUZ * nn + n] = du[2];
}

template <int Q, typename S, typename R>
__global__ void __launch_bounds__(128) phase_collide_kernel(const S* src, S* dst, const R* fld,
                                                            const __grid_constant__ KParams<R> p, PhaseGeom G) {
    using Ph = Phase<Q, S, R>;
    using Math = NodeMath<Q, S, R>;
    constexpr int D = Ph::D;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int n = Ph::node(G);
    if (n < 0) return;
    const size_t nn = (size_t)p.nn;
    const typename Ph::Steps s(p, n);
    Pop<S> f[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) f[k] = load_pop<true>(src + 2 * ((size_t)k * nn), (size_t)n);
    const R rho = fld[F_RHO * nn + n], T = fld[F_T * nn + n];
    R u[3] = {0, 0, 0}, dv[3] = {0, 0, 0};   // in march order (a, b, m)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        if (Q == 9 && j == 1) continue;
        u[j] = fld[(F_UX + Ph::axis(j)) * nn + n];
        dv[j] = fld[(F_DUX + Ph::axis(j)) * nn + n];
    }
    typename Math::Axis ax[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int j = Q == 9 && a == 1 ? 2 : a;
        const int hi = n + s.hi[a], lo = n + s.lo[a];
        const bool gh = s.g >> (2 * a) & 2, gl = s.g >> (2 * a) & 1;
        const R* ua = fld + (F_UX + a) * nn;
        const R* da = fld + (F_DUX + a) * nn;
        const R own = -::fma(dv[j], R(0.5), u[j]);   // beyond a wall: the normal velocity negated
        ax[a].uu = gh ? own : ::fma(da[hi], R(0.5), ua[hi]);
        ax[a].ud = gl ? own : ::fma(da[lo], R(0.5), ua[lo]);
        ax[a].Tu = ax[a].Td = T;
        ax[a].ru = ax[a].rd = rho;
        if (p.conduction) {
            ax[a].Tu = fld[F_T * nn + hi];
            ax[a].Td = fld[F_T * nn + lo];
            if (s.g) {
                R Tw;
                if (gh && wall_T<D>(p, a, 1, Tw)) ax[a].Tu = R(2) * Tw - T;
                if (gl && wall_T<D>(p, a, 0, Tw)) ax[a].Td = R(2) * Tw - T;
            }
            if (p.chi_mode) {
                ax[a].ru = fld[F_RHO * nn + hi];
                ax[a].rd = fld[F_RHO * nn + lo];
            }
        }
    }
    Pop<S>* out = reinterpret_cast<Pop<S>*>(dst);
    const EnergyPressure<R> ep = get_scratch(out + n, p, rho, T);
    const R dE = Math::energy_change(p, rho, T, ep.P, ax, D);
    const unsigned nbits = Store<S, R>::kStochastic ? node_bits(p.step, (unsigned)n) : 0u;
    Math::collide(p, rho, ep.E, u, dv, dE, [&](int k) { return f[k]; }, [&](int k, Two<R> v) {
        const unsigned t = Store<S, R>::kStochastic ? pair_word(nbits, k) : 0u;
        int to = n;
        bool bounce = false;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int c = Ph::vel(k, a);
            if (c == 0) continue;
            to += c > 0 ? s.wrap_hi[a] : s.wrap_lo[a];
            if (s.g >> (2 * a) & (c > 0 ? 2 : 1)) bounce = true;
        }
        // halfway bounce-back: the pair stays at its node, in the opposite direction
        if (bounce) store_pop(out + opposite(k) * nn, (unsigned)n, v, t);
        else store_pop(out + k * nn, (unsigned)to, v, t);
    });
}

}  // namespace lbm

// Per-node arithmetic of one time step (arXiv:1705.10045), written once for
// every kernel form that shares its bits: moments, equation of state and Phi,
// force, energy change, collision.  Callers supply the neighbour values and
// the stores.  Operations that feed one another are explicit fused
// multiply-adds (the build contracts nothing else), so every kernel that runs
// this code rounds alike.
#pragma once

#include <type_traits>

#include "kernels.cuh"

namespace lbm {

// Velocity of direction k in march coordinates: (a, b) across the tile,
// m along the last lattice axis.
template <int Q> struct MVel;
template <> struct MVel<9> {
    __host__ __device__ static constexpr int a(int k) { return Vel<9>::cx(k); }
    __host__ __device__ static constexpr int b(int) { return 0; }
    __host__ __device__ static constexpr int m(int k) { return Vel<9>::cy(k); }
};
template <> struct MVel<19> {
    __host__ __device__ static constexpr int a(int k) { return Vel<19>::cx(k); }
    __host__ __device__ static constexpr int b(int k) { return Vel<19>::cy(k); }
    __host__ __device__ static constexpr int m(int k) { return Vel<19>::cz(k); }
};

// Offsets of the neighbours of node n along its lattice axes.  lo / hi: the
// node a stencil reads (across a wall the mirror node, the node itself);
// wrap_lo / wrap_hi: the periodic neighbour; g: walls beside the node (bit 2a
// the low one of axis a, bit 2a + 1 the high one).
template <int Q, typename R> struct NodeSteps {
    int lo[3], hi[3], wrap_lo[3], wrap_hi[3], g;
    __device__ __forceinline__ NodeSteps(const KParams<R>& p, int n) {
        constexpr int D = Vel<Q>::D;
        int c[3];
        node_xyz(n, p.nx, p.ny, c[0], c[1], c[2]);
        const int len[3] = {p.nx, p.ny, p.nz}, stride[3] = {1, p.nx, p.nx * p.ny};
        g = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const bool wall = a == D - 1 ? p.wall : (a == 0 ? p.wall_x : p.wall_y);
            wrap_lo[a] = c[a] == 0 ? (len[a] - 1) * stride[a] : -stride[a];
            wrap_hi[a] = c[a] == len[a] - 1 ? -(len[a] - 1) * stride[a] : stride[a];
            const bool l = wall && c[a] == 0, h = wall && c[a] == len[a] - 1;
            lo[a] = l ? 0 : wrap_lo[a];
            hi[a] = h ? 0 : wrap_hi[a];
            g |= (l ? 1 : 0) << (2 * a) | (h ? 2 : 0) << (2 * a);
        }
    }
    // the node at n + c_k as a stencil reads it
    __device__ __forceinline__ int at(int n, int k) const {
        using V = Vel<Q>;
        const int c[3] = {V::cx(k), V::cy(k), V::cz(k)};
#pragma unroll
        for (int a = 0; a < V::D; ++a)
            if (c[a] != 0) n += c[a] > 0 ? hi[a] : lo[a];
        return n;
    }
};

// Two values moved through the same operation: the N and g of a direction.
// FP32 uses the packed instructions (one issue slot for both, each half
// rounded as the scalar instruction rounds it).
template <typename R> struct Two;
template <> struct Two<float> {
    unsigned long long v;
    __device__ static Two make(float a, float b) {
        Two r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    __device__ static Two dup(float a) { return make(a, a); }
    __device__ void get(float& a, float& b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
    __device__ static Two fma(Two a, Two b, Two c) {
        Two r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
        return r;
    }
    __device__ friend Two operator+(Two a, Two b) {
        Two r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    __device__ friend Two operator-(Two a, Two b) {
        Two r;
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    __device__ friend Two operator*(Two a, Two b) {
        Two r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
};
template <> struct Two<double> {
    double x, y;
    __device__ static Two make(double a, double b) { return {a, b}; }
    __device__ static Two dup(double a) { return {a, a}; }
    __device__ void get(double& a, double& b) const { a = x; b = y; }
    __device__ static Two fma(Two a, Two b, Two c) { return {::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y)}; }
    __device__ friend Two operator+(Two a, Two b) { return {a.x + b.x, a.y + b.y}; }
    __device__ friend Two operator-(Two a, Two b) { return {a.x - b.x, a.y - b.y}; }
    __device__ friend Two operator*(Two a, Two b) { return {a.x * b.x, a.y * b.y}; }
};

// A direction's pair as it is stored: N_k and g_k, or the FP16 word of both
// (shifted values; half the registers).
template <typename S> struct Pop;
template <> struct Pop<float> {
    float2 v;
    __device__ float N() const { return v.x; }
    __device__ float g() const { return v.y; }
    __device__ Two<float> two() const { return Two<float>::make(v.x, v.y); }
};
template <> struct Pop<double> {
    double2 v;
    __device__ double N() const { return v.x; }
    __device__ double g() const { return v.y; }
    __device__ Two<double> two() const { return Two<double>::make(v.x, v.y); }
};
template <> struct Pop<__half> {
    unsigned v;
    __device__ float N() const { return Store<__half, float>::lo(v); }
    __device__ float g() const { return Store<__half, float>::hi(v); }
    __device__ Two<float> two() const { return Two<float>::make(N(), g()); }
};

// The pair at pair index i of q.  COH: coherent loads, for data other CTAs of
// the same launch or the launch before it wrote while this one was resident.  KEEP: a first read of lines the same SM reads again
// soon (L2 evict-last where it pays).  LAST: the last use of the line on this
// SM (not allocated in L1).
enum LoadUse { kUse, kUseKeep, kUseLast };
template <bool COH, LoadUse U = kUse> __device__ __forceinline__ Pop<float> load_pop(const float* q, size_t i) {
    using St = Store<float, float>;
    Pop<float> r;
    if (U == kUseLast) COH ? St::load2_last_coh(q, i, 0.f, 0.f, r.v.x, r.v.y) : St::load2_last(q, i, 0.f, 0.f, r.v.x, r.v.y);
    else if (COH) St::load2_coh(q, i, 0.f, 0.f, r.v.x, r.v.y);
    else if (U == kUseKeep) St::load2_keep(q, i, 0.f, 0.f, r.v.x, r.v.y);
    else St::load2(q, i, 0.f, 0.f, r.v.x, r.v.y);
    return r;
}
template <bool COH, LoadUse U = kUse> __device__ __forceinline__ Pop<double> load_pop(const double* q, size_t i) {
    using St = Store<double, double>;
    Pop<double> r;
    if (U == kUseLast) COH ? St::load2_last_coh(q, i, 0., 0., r.v.x, r.v.y) : St::load2_last(q, i, 0., 0., r.v.x, r.v.y);
    else if (COH) St::load2_coh(q, i, 0., 0., r.v.x, r.v.y);
    else St::load2(q, i, 0., 0., r.v.x, r.v.y);
    return r;
}
template <bool COH, LoadUse U = kUse> __device__ __forceinline__ Pop<__half> load_pop(const __half* q, size_t i) {
    using St = Store<__half, float>;
    Pop<__half> r;
    if (U == kUseLast) r.v = COH ? St::word_last_coh(q, i) : St::word_last(q, i);
    else r.v = COH ? St::word_coh(q, i) : St::word(q, i);
    return r;
}

template <typename R> struct Moments {
    R rho, ja, jb, jm, E;
};

template <int Q, typename S, typename R> struct NodeMath {
    using V = Vel<Q>;
    using M = MVel<Q>;
    static constexpr bool kSh = Store<S, R>::kShifted;

    // sum over k of g_k
    __device__ static __forceinline__ R energy(const Pop<S>* f, const KParams<R>& p) {
        R E = f[0].g();
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            if constexpr (kSh) E = Store<S, R>::add_hi(f[k].v, E);   // FP16: the half enters the sum directly
            else E += f[k].g();
        }
        if constexpr (kSh) E += p.E_ref;   // sums of shifted values: sum_k w_k = 1, sum_k w_k c_k = 0
        return E;
    }

    // rho, momentum and E of a node from its pairs f[0..Q).  Opposite
    // directions k, k+1 pair up: their sum enters rho, their difference the
    // momentum along c_k (each sum starts at its first term).
    __device__ static __forceinline__ Moments<R> moments(const Pop<S>* f, const KParams<R>& p) {
        Moments<R> o;
        o.ja = o.jb = o.jm = R(0);
        bool new_a = true, new_b = true, new_m = true;
        o.rho = f[0].N();
#pragma unroll
        for (int k = 1; k < Q; k += 2) {
            R s, d;   // N_k + N_{k+1} and N_k - N_{k+1}
            if constexpr (kSh) {   // FP16: the halves enter the sums directly
                const R x = f[k].N();
                s = Store<S, R>::add_lo(f[k + 1].v, x);
                d = -Store<S, R>::sub_lo(f[k + 1].v, x);
            } else {
                s = f[k].N() + f[k + 1].N();
                d = f[k].N() - f[k + 1].N();
            }
            o.rho += s;
            if (M::a(k) != 0) { const R t = M::a(k) > 0 ? d : -d; o.ja = new_a ? t : o.ja + t; new_a = false; }
            if (M::b(k) != 0) { const R t = M::b(k) > 0 ? d : -d; o.jb = new_b ? t : o.jb + t; new_b = false; }
            if (M::m(k) != 0) { const R t = M::m(k) > 0 ? d : -d; o.jm = new_m ? t : o.jm + t; new_m = false; }
        }
        if constexpr (kSh) o.rho += p.rho_ref;
        o.E = energy(f, p);
        return o;
    }

    // U = p - rho theta, and Phi = sqrt(-U) where U < 0
    __device__ static __forceinline__ R potential(R rho, R P) { return ::fma(-rho, R(1.0 / 3.0), P); }
    __device__ static __forceinline__ R phi_of(R U) { return U < R(0) ? sqrt(-U) : R(0); }
    __device__ static __forceinline__ bool positive(R v) {
        if constexpr (sizeof(R) == 8) {   // by its bits: an FP64 comparison takes the FP64 pipe
            const long long b = __double_as_longlong(v);
            return b > 0 && b < 0x7ff0000000000000ll;
        } else {
            return finite_pos(v);
        }
    }

    // du = F/rho of a node (Sec. 3 force + gravity).  ph(a, b, m): Phi at the
    // neighbour (a, b, m); opposite directions pair up, since
    // G Phi(x+e) e + G Phi(x-e)(-e) = G (Phi+ - Phi-) e and the Phi^2 term is
    // G (Phi+ - Phi-)(Phi+ + Phi-) e.
    template <typename PH>
    __device__ static __forceinline__ void force(const KParams<R>& p, const PH& ph, R rho, R* du) {
        const R A = p.A, B = R(1) - R(2) * p.A, inv_alpha = R(1.0 / V::alpha);
        const R gv[3] = {p.g[0], Q == 9 ? R(0) : p.g[1], Q == 9 ? p.g[1] : p.g[2]};
        const R G2 = R(V::G(Q - 1));   // next-nearest weight (1/4 or 1/2)
        const R Bph0 = B * ph(0, 0, 0);
        R n1[3] = {0, 0, 0}, n2[3] = {0, 0, 0}, q1[3] = {0, 0, 0}, q2[3] = {0, 0, 0};
#pragma unroll
        for (int k = 1; k < Q; k += 2) {
            const R pp = ph(M::a(k), M::b(k), M::m(k)), pm = ph(-M::a(k), -M::b(k), -M::m(k));
            const R d = pp - pm, sum = pp + pm;
            const bool nearest = M::a(k) * M::a(k) + M::b(k) * M::b(k) + M::m(k) * M::m(k) == 1;
            R* s1 = nearest ? n1 : q1;
            R* s2 = nearest ? n2 : q2;
            // s1 += +-d (Phi+ + Phi-) as one fused multiply-add per axis
            if (M::a(k) == 1) { s1[0] = ::fma(d, sum, s1[0]); s2[0] += d; }
            else if (M::a(k) == -1) { s1[0] = ::fma(-d, sum, s1[0]); s2[0] -= d; }
            if (M::b(k) == 1) { s1[1] = ::fma(d, sum, s1[1]); s2[1] += d; }
            else if (M::b(k) == -1) { s1[1] = ::fma(-d, sum, s1[1]); s2[1] -= d; }
            if (M::m(k) == 1) { s1[2] = ::fma(d, sum, s1[2]); s2[2] += d; }
            else if (M::m(k) == -1) { s1[2] = ::fma(-d, sum, s1[2]); s2[2] -= d; }
        }
        const R scale = inv_alpha / rho;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R s1 = ::fma(G2, q1[a], n1[a]), s2 = ::fma(G2, q2[a], n2[a]);
            du[a] = ::fma(::fma(A, s1, Bph0 * s2), scale, gv[a]);
        }
    }

    // Neighbour values of one axis (upper, lower): u* along the axis, T, rho.
    struct Axis {
        R uu, ud, Tu, Td, ru, rd;
    };
    // dE of a node by centred differences (Sec. 4, Sec. 6.2) from its n axes:
    // pressure work, conduction through faces whose conductivity is the mean
    // of the two nodes', latent heat.
    __device__ static __forceinline__ R energy_change(const KParams<R>& p, R rho, R T, R P, const Axis* ax, int n) {
        R div = R(0), cond = R(0);
#pragma unroll
        for (int a = 0; a < n; ++a) div = ::fma(ax[a].uu - ax[a].ud, R(0.5), div);
        if (p.conduction) {
            const R half_lc = conductivity(p, rho) * R(0.5);
#pragma unroll
            for (int a = 0; a < n; ++a) {
                // a constant conductivity is its own mean, exactly
                const R lu = p.chi_mode ? ::fma(conductivity(p, ax[a].ru), R(0.5), half_lc) : p.lambda;
                const R ld = p.chi_mode ? ::fma(conductivity(p, ax[a].rd), R(0.5), half_lc) : p.lambda;
                cond = ::fma(-ld, T - ax[a].Td, ::fma(lu, ax[a].Tu - T, cond));
            }
        }
        R dE = R(0);
        if (p.pressure_work) dE += -P * div;
        if (p.conduction) dE += cond;
        if (p.latent != R(0)) dE += latent_heat(p, rho, T, div);
        return dE;
    }

    // Collision, Eq. (lbe)/(edm)/(gk), written per node as
    //   N*_k = (1 - omega) N_k + rho (omega e0_k + de_k)
    //   g*_k = (1 - omega_E + dE/E) g_k + E (omega_E e0_k + [pseudoforce] de_k)
    // with e0 = N^eq(rho,u)/rho and de = (N^eq(rho,u+du) - N^eq(rho,u))/rho.
    // With v = u + du, s = c_k.u and t = c_k.v, Eq. (feq) gives
    //   e0_k = w_k (b0 + 4.5 s^2 + 3 s),   de_k = w_k (db + 4.5 (t^2 - s^2) + 3 (t - s))
    // (b0 = 1 - 1.5 u.u, db = -1.5 (v.v - u.u) = -1.5 du.(2u + du)), so
    //   rho (omega e0_k + de_k) = w_k K + 4.5 w_k [P s^2 + rho t^2] + 3 w_k [P s + rho t]
    // with K = rho omega b0 + rho db and P = rho omega - rho; the same holds
    // for g with (E omega_E, E_pf) in place of (rho omega, rho), so N and g go
    // through the same operations as the two halves of a Two.  Opposite
    // directions k, k+1 (c -> -c) share the even part and flip the odd one.
    // The factors w K, 4.5 w P, ... are formed once for the nearest directions
    // and scaled by w2/w1 (1/2 on D3Q19, 1/4 on D2Q9: exact) for the
    // next-nearest.  Shifted storage: with N_k = N'_k + w_k rho_ref and
    // g_k = g'_k + w_k E_ref
    //   N*'_k = (1 - omega) N'_k + rho (omega e0_k + de_k) - omega w_k rho_ref
    //   g*'_k = fG g'_k + E (omega_E e0_k + [pf] de_k) + (fG - 1) w_k E_ref
    // so the shifts enter K as nsh and gsh.
    // emit(k, out): the pair of direction k after the collision.
    template <typename PF, typename EM>
    __device__ static __forceinline__ void collide(const KParams<R>& p, R rho, R E, const R* u, const R* dv, R dE,
                                                   const PF& pop, const EM& emit) {
        using T2 = Two<R>;
        const R dEoverE = dE / E;
        R usq = u[2] * u[2], dsq = dv[2] * ::fma(R(2), u[2], dv[2]);
        if (Q == 19) {
            usq = ::fma(u[1], u[1], usq);
            dsq = ::fma(dv[1], ::fma(R(2), u[1], dv[1]), dsq);
        }
        usq = ::fma(u[0], u[0], usq);
        dsq = ::fma(dv[0], ::fma(R(2), u[0], dv[0]), dsq);
        const R base0 = ::fma(R(-1.5), usq, R(1)), dbase = R(-1.5) * dsq;
        const R om = p.omega, omE = p.omega_E;
        const R fN = R(1) - om, fG = R(1) - omE + dEoverE;
        const R rho_om = rho * om, E_omE = E * omE, E_pf = p.pseudoforce ? E : R(0);
        const R nsh = kSh ? -om * p.rho_ref : R(0), gsh = kSh ? (fG - R(1)) * p.E_ref : R(0);
        const R KN = kSh ? ::fma(rho_om, base0, ::fma(rho, dbase, nsh)) : ::fma(rho_om, base0, rho * dbase);
        const R KG = kSh ? ::fma(E_omE, base0, ::fma(E_pf, dbase, gsh)) : ::fma(E_omE, base0, E_pf * dbase);
        const T2 f2 = T2::make(fN, fG), K = T2::make(KN, KG);
        const T2 Pp = T2::make(rho_om - rho, E_omE - E_pf), Qq = T2::make(rho, E_pf);
        emit(0, T2::fma(pop(0).two(), f2, T2::dup(R(V::w(0))) * K));
        constexpr double w1 = V::w(1);
        T2 kn = T2::dup(R(w1)) * K, pn = T2::dup(R(4.5 * w1)) * Pp, qn = T2::dup(R(4.5 * w1)) * Qq;
        T2 rn = T2::dup(R(3.0 * w1)) * Pp, sn = T2::dup(R(3.0 * w1)) * Qq;
        T2 uu[3], vv[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            uu[a] = T2::dup(u[a]);
            vv[a] = T2::dup(u[a] + dv[a]);
        }
#pragma unroll
        for (int k = 1; k < Q; k += 2) {
            if (k == (Q == 19 ? 7 : 5)) {   // first next-nearest direction
                const T2 h = T2::dup(R(V::w(Q - 1) / w1));
                kn = kn * h; pn = pn * h; qn = qn * h; rn = rn * h; sn = sn * h;
            }
            // s = c_k.u and t = c_k.v, each summed from its first term (whose
            // sign is positive for the odd k of both lattices)
            T2 s, t;
            bool first = true;
            auto add = [&](int cc, T2 x, T2 y) {
                if (cc == 0) return;
                s = first ? x : (cc > 0 ? s + x : s - x);
                t = first ? y : (cc > 0 ? t + y : t - y);
                first = false;
            };
            add(M::a(k), uu[0], vv[0]);
            add(M::b(k), uu[1], vv[1]);
            add(M::m(k), uu[2], vv[2]);
            const T2 even = T2::fma(pn, s * s, T2::fma(qn, t * t, kn)), odd = T2::fma(rn, s, sn * t);
            emit(k, T2::fma(pop(k).two(), f2, even + odd));
            emit(k + 1, T2::fma(pop(k + 1).two(), f2, even - odd));
        }
    }
};

// store a post-collision pair at q[i]; t: the FP16 random word
__device__ __forceinline__ void store_pop(Pop<float>* q, unsigned i, Two<float> x, unsigned) {
    float a, b;
    x.get(a, b);
    Store<float, float>::store2(&q[i].v.x, 0, a, b, 0.f, 0.f);
}
__device__ __forceinline__ void store_pop(Pop<double>* q, unsigned i, Two<double> x, unsigned) {
    q[i].v = make_double2(x.x, x.y);
}
__device__ __forceinline__ void store_pop(Pop<__half>* q, unsigned i, Two<float> x, unsigned t) {
    float a, b;
    x.get(a, b);
    Store<__half, float>::store2_raw(reinterpret_cast<__half*>(q + i), 0, a, b, t);
}

}  // namespace lbm

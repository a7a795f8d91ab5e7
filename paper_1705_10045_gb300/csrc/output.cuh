// Output fields (lbm_moments, lbm_moments_f): rho, the physical velocity
// u* = u + du/2 (Eq. (ustar)), T and P (EOS), as O = double or float.
//
// Two launches, bound by memory: the first reads the populations once and
// writes rho, T and P as they leave (and rho, u, Phi for the second), the
// second forms du from Phi and writes u*.  384 x 384 x 256 D3Q19 FP32, FP32
// fields: 190 B read and 44 B written per node; three launches through nine
// field planes and a narrowing pass took 2773 us.
#pragma once

#include "node.cuh"

namespace lbm {

// cnt_out: where the device counters are copied, if anywhere
template <int Q, typename S, typename R, typename O>
__global__ void __launch_bounds__(256) output_kernel(const S* __restrict__ pop, R* __restrict__ fld,
                                                     const __grid_constant__ KParams<R> p, O* __restrict__ rho_out,
                                                     O* __restrict__ T_out, O* __restrict__ P_out, int velocity,
                                                     const Counters* cnt, Counters* cnt_out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && cnt_out) *cnt_out = *cnt;
    if (i >= p.nn) return;
    const long long nn = p.nn;
    R rho, jx, jy, jz, E;
    node_moments<Q, S, R>(pop, nn, i, p, rho, jx, jy, jz, E);
    const R T = E / (rho * p.c_v), P = eos_pressure(p, rho, T);
    if (rho_out) rho_out[i] = (O)rho;
    if (T_out) T_out[i] = (O)T;
    if (P_out) P_out[i] = (O)P;
    if (!velocity) return;
    const R U = fma(-rho, R(1.0 / 3.0), P);
    fld[F_PHI * nn + i] = U < R(0) ? sqrt(-U) : R(0);
    fld[F_RHO * nn + i] = rho;
    fld[F_UX * nn + i] = jx / rho;
    fld[F_UY * nn + i] = jy / rho;
    if (Vel<Q>::D == 3) fld[F_UZ * nn + i] = jz / rho;
}

// u* from the Phi stencil: the sums of force_kernel, term by term
template <int Q, typename R, typename O>
__global__ void __launch_bounds__(256) output_velocity_kernel(const R* __restrict__ fld,
                                                              const __grid_constant__ KParams<R> p,
                                                              O* __restrict__ u_out) {
    using V = Vel<Q>;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.nn) return;
    const long long nn = p.nn;
    const NodeSteps<Q, R> st(p, (int)i);
    const R* Phi = fld + F_PHI * nn;
    R s1[3] = {0, 0, 0}, s2[3] = {0, 0, 0};
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        const R ph = Phi[st.at((int)i, k)];
        const R t1 = R(V::G(k)) * ph * ph, t2 = R(V::G(k)) * ph;
        const int c[3] = {V::cx(k), V::cy(k), V::cz(k)};
#pragma unroll
        for (int a = 0; a < V::D; ++a) {
            if (c[a] == 1) { s1[a] += t1; s2[a] += t2; }
            else if (c[a] == -1) { s1[a] -= t1; s2[a] -= t2; }
        }
    }
    const R rho = fld[F_RHO * nn + i], ph0 = Phi[i];
    const R A = p.A, B = R(1) - R(2) * p.A, inv_alpha = R(1.0 / V::alpha);
#pragma unroll
    for (int a = 0; a < V::D; ++a) {
        const R du = ((A * s1[a] + B * ph0 * s2[a]) * inv_alpha + rho * p.g[a]) / rho;
        u_out[a * nn + i] = (O)(fld[(F_UX + a) * nn + i] + du / R(2));
    }
}

}  // namespace lbm

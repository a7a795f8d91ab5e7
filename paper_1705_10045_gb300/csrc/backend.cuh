// Launch sequences of the liblbm back end for one lattice, for every storage
// format.  Included once per lattice by lbm_d2q9.cu and lbm_d3q19.cu.
//
// A time step takes one of four forms that round alike and so leave the same
// bits: strips of columns (D2Q9 FP32 and FP16, strip.cuh), rows of columns
// (rows.cuh) or the producer/consumer march (fused.cuh) for D3Q19, and three
// launches over all nodes (FP64 and small D3Q19 domains, phases.cuh).  The
// form fields -> force -> collide (LBM_STEP_THREE_LAUNCH) is kept as a second,
// independently structured statement of the same step.
#pragma once

#include "fused.cuh"
#include "internal.h"
#include "kernels.cuh"
#include "output.cuh"
#include "phases.cuh"
#include "plan.h"
#include "rows.cuh"
#include "strip.cuh"

namespace lbm {

template <typename R> KParams<R> make_kparams(const lbm_handle* h) {
    const lbm_params& q = h->p;
    KParams<R> k;
    k.nx = q.nx; k.ny = q.ny; k.nz = q.nz; k.nn = h->nn;
    k.kappa = (R)q.kappa; k.A = (R)q.A; k.T0 = (R)q.T0; k.barotropic = q.barotropic != 0;
    k.omega = (R)(1.0 / q.tau); k.omega_E = (R)(1.0 / q.tau_E);
    k.c_v = (R)q.c_v;
    k.chi_mode = q.chi_mode != 0; k.lambda = (R)q.lambda; k.chi = (R)q.chi;
    for (int a = 0; a < 3; ++a) k.g[a] = (R)q.gravity[a];
    k.wall = q.wall != 0;
    k.T_fixed_lo = q.T_fixed_lo != 0; k.T_fixed_hi = q.T_fixed_hi != 0;
    k.T_lo = (R)q.T_lo; k.T_hi = (R)q.T_hi;
    k.wall_x = q.wall_x != 0; k.wall_y = q.lattice == LBM_D3Q19 && q.wall_y != 0;
    for (int e = 0; e < 2; ++e) {
        k.T_fixed_x[e] = q.T_fixed_x[e] != 0; k.T_fixed_y[e] = q.T_fixed_y[e] != 0;
        k.T_x[e] = (R)q.T_x[e]; k.T_y[e] = (R)q.T_y[e];
    }
    k.pressure_work = q.pressure_work != 0; k.conduction = q.conduction != 0; k.pseudoforce = q.pseudoforce != 0;
    const bool shifted = q.storage == LBM_STORE_FP16;
    k.rho_ref = shifted ? (R)q.rho_ref : R(0);
    k.E_ref = shifted ? (R)q.E_ref : R(0);
    k.step = (unsigned)h->steps;
    k.latent = (R)q.latent;
    k.coex = (const R*)h->coex;
    return k;
}

inline unsigned grid_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Launch a kernel that begins with griddepcontrol.wait as a programmatic
// dependent of the stream's previous kernel: its CTAs are set up while that
// one drains.  Between ordinary launches of short kernels the step time moved
// in stairs of 2.05 us (512 x 512 D2Q9: 10.3 us for 8.4 us this way).
template <typename... P, typename... A>
void launch_after(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, args...);
}

// CTA shape of the fused kernel: a TX x TY tile of consumer threads plus NP
// producer threads.  D3Q19 uses 32 x 8 nodes with 128 producers (two CTAs per
// SM) in FP32/FP16.  FP64 (256 producers on D3Q19) and D2Q9 (rows of 128 nodes
// with 160 producers, one per node of the 132-node ring row) run it in its
// fault-injection form only.
// SPLIT: the consumers form the moments of their own nodes and the producers
// only those of the ring's border (fused_tile)
template <int Q, typename R> struct FusedTile;
template <typename R> struct FusedTile<9, R> { static constexpr int TX = 128, TY = 1, NP = 160; static constexpr bool SPLIT = false; };
template <> struct FusedTile<19, float> { static constexpr int TX = 32, TY = 8, NP = 128; static constexpr bool SPLIT = true; };
template <> struct FusedTile<19, double> { static constexpr int TX = 32, TY = 8, NP = 256; static constexpr bool SPLIT = true; };

// CTA shapes a batch may run with; the autotuner times each on the batch and
// keeps the fastest.  D2Q9: W warps of a strip each.  D3Q19: TX x TY consumers
// + NP producers of the march, its moment stage split.  MB: CTAs per SM the
// batch kernel is compiled for (its register cap).
template <int Q, int V> struct BatchShape;
template <> struct BatchShape<9, 0> { static constexpr int W = 4, MB = 4; };
template <> struct BatchShape<9, 1> { static constexpr int W = 1, MB = 16; };
template <> struct BatchShape<9, 2> { static constexpr int W = 2, MB = 8; };
template <> struct BatchShape<19, 0> { static constexpr int TX = 32, TY = 8, NP = 128, MB = 2; };
template <> struct BatchShape<19, 1> { static constexpr int TX = 32, TY = 8, NP = 160, MB = 2; };
template <> struct BatchShape<19, 2> { static constexpr int TX = 32, TY = 4, NP = 96, MB = 3; };

template <int Q, typename S, typename R> struct Impl {
    static constexpr int TX = FusedTile<Q, R>::TX, TY = FusedTile<Q, R>::TY, NP = FusedTile<Q, R>::NP;
    static constexpr bool SPLIT = FusedTile<Q, R>::SPLIT;
    // Steps in three phases (phases.cuh): FP64, and small D3Q19 domains.
    static constexpr bool kF64 = std::is_same<S, double>::value;
    static constexpr bool kPhases = kF64 || Q == 19;
    static bool phases(const lbm_handle* h) { return kPhases && h->phases && h->fault_drop <= 0; }
    static constexpr StepModel kModel = sizeof(S) == 2 ? kModelFp16 : kModelFp32;
    static_assert(kF64 || Q == 9 || (kModel.tx == TX && kModel.ty == TY), "modelled tile");
    static bool wants_phases(const lbm_params& p) {
        if (kF64) return true;
        if (!kPhases) return false;
        const MarchGeom G = {p.nx, p.ny, p.nz, 0, 0, p.nz};
        return phase_time(kModel, G) < std::min(march_chunk(kModel, G, p.nz).t, row_chunk(kModel, G, p.nz, p.wall_x).t);
    }
    static int launches(const lbm_handle* h) {
        return h->p.step_kernel == LBM_STEP_THREE_LAUNCH || phases(h) ? 3 : 1;
    }

    // D2Q9 in FP32 and FP16 storage: a warp per strip of columns (strip.cuh)
    static constexpr bool kStrips = Q == 9 && !kF64;
    static constexpr bool kRows = Q == 19 && !kF64;

    // How a step of planes [m_lo, m_hi) is launched, found once per call.
    enum Form { kFormPhases, kFormStrips, kFormRows, kFormMarch, kFormFault };
    struct Plan {
        Form form;
        MarchGeom G;     // chunk: of rows and march
        int strip_rows;
    };
    // m_hi < 0: the handle's own range (lbm_set_step_planes; all by default)
    static Plan plan(const lbm_handle* h, int m_lo = 0, int m_hi = -1) {
        Plan s{};
        MarchGeom& G = s.G;
        G.na = h->p.nx;
        G.nb = Q == 9 ? 1 : h->p.ny;
        G.nm = Q == 9 ? h->p.ny : h->p.nz;
        if (m_hi < 0) {
            G.m_lo = h->step_count > 0 ? h->step_first : 0;
            G.m_hi = h->step_count > 0 ? h->step_first + h->step_count : G.nm;
        } else {
            G.m_lo = m_lo;
            G.m_hi = m_hi;
        }
        const int len = G.m_hi - G.m_lo;
        if (h->fault_drop > 0) {   // fault-injection test hook (lbm_test_drop_handoff)
            s.form = kFormFault;
            G.chunk = std::min(kMaxChunk, len);   // long, so that the first CTA marches over the plane
        } else if (phases(h)) {
            s.form = kFormPhases;
        } else if (kStrips) {
            s.form = kFormStrips;
            s.strip_rows = strip_rows(strip_count(G.na), len, kSms);
        } else {
            const Chunk march = march_chunk(kModel, G, len), rows = row_chunk(kModel, G, len, h->p.wall_x);
            s.form = rows.t < march.t ? kFormRows : kFormMarch;
            G.chunk = rows.t < march.t ? rows.planes : march.planes;
        }
        return s;
    }

    // name of the kernel of a step in one launch
    static const char* single_name(const lbm_handle* h) {
        const Form f = plan(h).form;
        return f == kFormStrips ? "strip_step_kernel" : (f == kFormRows ? "row_march_kernel" : "fused_step_kernel");
    }

    // the step over the planes of G in three launches
    static void launch_phase(lbm_handle* h, const KParams<R>& kp, const MarchGeom& G, const S* src, S* dst, int j) {
        // the moments of two planes and the forces of one plane beyond the
        // range, or of every plane
        const int reach = 2 - j, len = G.m_hi - G.m_lo;
        PhaseGeom g;
        g.plane_n = G.na * G.nb;
        g.nm = G.nm;
        g.m_lo = G.m_lo;
        g.m_hi = G.m_hi;
        g.first = G.m_lo - reach;
        g.count = len + 2 * reach;
        if (h->p.wall) {
            const int hi = std::min(g.first + g.count, G.nm);
            g.first = std::max(g.first, 0);
            g.count = hi - g.first;
        } else if (g.count >= G.nm) {
            g.first = 0;
            g.count = G.nm;
        } else if (g.first < 0) {
            g.first += G.nm;
        }
        const unsigned grid = grid_for((long long)g.count * g.plane_n, 128);
        R* fld = (R*)h->fld;
        if (j == 0) launch_after(phase_moments_kernel<Q, S, R>, grid, 128, 0, h->stream, src, dst, fld, kp, g, (Counters*)h->cnt);
        if (j == 1) launch_after(phase_force_kernel<Q, S, R>, grid, 128, 0, h->stream, fld, kp, g);
        if (j == 2) launch_after(phase_collide_kernel<Q, S, R>, grid, 128, 0, h->stream, src, dst, fld, kp, g);
    }

    // the planned step, src -> dst (no buffer swap)
    static void launch_fused(lbm_handle* h, const KParams<R>& kp, const Plan& s, const S* src, S* dst) {
        Counters* cnt = (Counters*)h->cnt;
        const MarchGeom& G = s.G;
        const int len = G.m_hi - G.m_lo;
        if (s.form == kFormPhases) {
            if constexpr (kPhases)
                for (int j = 0; j < 3; ++j) launch_phase(h, kp, G, src, dst, j);
        } else if (s.form == kFormStrips) {
            if constexpr (kStrips) {
                const StripGeom g = {G.na, G.nm, G.m_lo, G.m_hi, s.strip_rows, strip_count(G.na)};
                const long long warps = (long long)g.strips * ((len + g.chunk - 1) / g.chunk);
                auto kern = h->p.wall || h->p.wall_x ? strip_step_kernel<S, R, true> : strip_step_kernel<S, R, false>;
                const size_t smem = kStripWarps * Strip<S, R, false>::kRingBytes;
                allow_smem(kern, smem, h->fused_ready);
                launch_after(kern, grid_for(warps, kStripWarps), 32 * kStripWarps, smem, h->stream, src, dst, kp, g, cnt);
            }
        } else if (s.form == kFormRows) {
            if constexpr (kRows) {
                using Sh = RowShape<S>;
                static_assert(Sh::TY == kModel.rows, "modelled tile");
                constexpr size_t smem = RowMarch<S, R, Sh::TY, Sh::AHEAD, true>::kBytes;
                auto kern = h->p.wall || h->p.wall_y ? row_march_kernel<S, R, true> : row_march_kernel<S, R, false>;
                allow_smem(kern, smem, h->rows_ready);
                launch_after(kern, dim3(strip_count(G.na), (G.nb + Sh::TY - 1) / Sh::TY, (len + G.chunk - 1) / G.chunk),
                             32 * (Sh::TY + 4), smem, h->stream, src, dst, kp, G, cnt);
            }
        } else {
            const size_t smem = FusedShape<TX, TY, SPLIT>::template smem_bytes<R>();
            const dim3 grid((G.na + TX - 1) / TX, (G.nb + TY - 1) / TY, (len + G.chunk - 1) / G.chunk);
            if (s.form == kFormFault) {
                auto kern = fused_step_fault_kernel<Q, S, R, TX, TY, NP, SPLIT>;
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                kern<<<grid, TX * TY + NP, smem, h->stream>>>(src, dst, kp, G, cnt, h->fault_drop - 1);
            } else if constexpr (kRows) {
                const bool xw = h->p.wall_x || h->p.wall_y;
                auto kern = xw ? fused_step_kernel<Q, S, R, TX, TY, NP, true, SPLIT>
                               : fused_step_kernel<Q, S, R, TX, TY, NP, false, SPLIT>;
                allow_smem(kern, smem, h->fused_ready);
                kern<<<grid, TX * TY + NP, smem, h->stream>>>(src, dst, kp, G, cnt);
            }
        }
    }
    // raise a kernel's shared-memory limit, once per handle
    template <typename K> static void allow_smem(K kern, size_t smem, bool& ready) {
        if (!ready) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        ready = true;
    }
    // planes [first, first + count) of the step lbm_step_begin opened: it has
    // already made the destination buffer current, so the source is the other
    static int step_range(lbm_handle* h, int first, int count) {
        KParams<R> kp = make_kparams<R>(h);
        kp.step = (unsigned)h->pending_step;
        launch_fused(h, kp, plan(h, first, first + count), (const S*)h->pop[h->cur ^ 1], (S*)h->pop[h->cur]);
        return cuda_error(cudaGetLastError(), "lbm_step_begin launch");
    }

    // launch j of one time step; the last launch of a step swaps the buffers
    static void launch(lbm_handle* h, const KParams<R>& kp, const Plan& s, int j) {
        if (h->p.step_kernel != LBM_STEP_THREE_LAUNCH) {
            const S* src = (const S*)h->pop[h->cur];
            S* dst = (S*)h->pop[h->cur ^ 1];
            if (s.form == kFormPhases) {
                if constexpr (kPhases) launch_phase(h, kp, s.G, src, dst, j);
                if (j < 2) return;
            } else {
                launch_fused(h, kp, s, src, dst);
            }
            h->cur ^= 1;
            return;
        }
        const unsigned g = grid_for(h->nn, 256);
        R* fld = (R*)h->fld;
        const S* src = (const S*)h->pop[h->cur];
        S* dst = (S*)h->pop[h->cur ^ 1];
        if (j == 0) fields_kernel<Q, S, R><<<g, 256, 0, h->stream>>>(src, fld, kp, (Counters*)h->cnt, 1);
        if (j == 1) force_kernel<Q, R><<<g, 256, 0, h->stream>>>(fld, kp);
        if (j == 2) {
            collide_kernel<Q, S, R><<<g, 256, 0, h->stream>>>(src, dst, fld, kp);
            h->cur ^= 1;
        }
    }

    static int step(lbm_handle* h, int n) {
        KParams<R> kp = make_kparams<R>(h);
        const int L = launches(h);
        const Plan how = plan(h);
        for (int s = 0; s < n; ++s) {
            kp.step = (unsigned)(h->steps + s);
            for (int j = 0; j < L; ++j) launch(h, kp, how, j);
        }
        return cuda_error(cudaGetLastError(), "lbm_step launch");
    }

    // n steps with an event pair around every launch; ms[j] = mean duration of launch j
    static int profile(lbm_handle* h, int n, double* ms, int cap) {
        KParams<R> kp = make_kparams<R>(h);
        const int L = launches(h);
        const Plan how = plan(h);
        cudaEvent_t ev[6];
        for (int e = 0; e < 2 * L; ++e)
            if (int rc = cuda_error(cudaEventCreate(&ev[e]), "event create")) return rc;
        double acc[3] = {0.0, 0.0, 0.0};
        int rc = LBM_OK;
        for (int s = 0; s < n && !rc; ++s) {
            kp.step = (unsigned)(h->steps + s);
            for (int j = 0; j < L; ++j) {
                cudaEventRecord(ev[2 * j], h->stream);
                launch(h, kp, how, j);
                cudaEventRecord(ev[2 * j + 1], h->stream);
            }
            rc = cuda_error(cudaEventSynchronize(ev[2 * L - 1]), "profile synchronize");
            for (int j = 0; j < L && !rc; ++j) {
                float t = 0.f;
                rc = cuda_error(cudaEventElapsedTime(&t, ev[2 * j], ev[2 * j + 1]), "event time");
                acc[j] += t;
            }
        }
        for (int e = 0; e < 2 * L; ++e) cudaEventDestroy(ev[e]);
        if (rc) return rc;
        for (int j = 0; j < L && j < cap; ++j) ms[j] = n > 0 ? acc[j] / n : 0.0;
        return L;
    }

    static int init(lbm_handle* h, const double* rho, const double* u, const double* eps) {
        KParams<R> kp = make_kparams<R>(h);
        kp.step = 0xFFFFFFFFu;   // rounding seed of the initial state, distinct from every step
        init_kernel<Q, S, R><<<grid_for(h->nn, 256), 256, 0, h->stream>>>((S*)h->pop[h->cur], rho, u, eps, kp,
                                                                           (Counters*)h->cnt);
        return cuda_error(cudaGetLastError(), "lbm_init launch");
    }
    template <typename O>
    static int output(lbm_handle* h, O* rho, O* u, O* T, O* P, Counters* cnt_out) {
        const KParams<R> kp = make_kparams<R>(h);
        const unsigned g = grid_for(h->nn, 256);
        R* fld = (R*)h->fld;
        output_kernel<Q, S, R, O><<<g, 256, 0, h->stream>>>((const S*)h->pop[h->cur], fld, kp, rho, T, P, u != nullptr,
                                                            (const Counters*)h->cnt, cnt_out);
        if (u) output_velocity_kernel<Q, R, O><<<g, 256, 0, h->stream>>>(fld, kp, u);
        return cuda_error(cudaGetLastError(), "lbm_moments launch");
    }
    // ---- batches ---------------------------------------------------------
    // Planes (D2Q9: rows) per work item of the domains that step in a request.
    // D2Q9: a step of a domain starts when all items of its previous step are
    // done, so an item (its rows and four more at 1.45 us with 16 warps per SM,
    // 2 us to hand over) should take no longer than 3/4 of what one step of
    // every domain takes (1.45 us per 16 x 152 warp rows), within 2 to 64 rows.
    // Measured us per step of every domain: 24 domains of 64..512 (2.9 M nodes;
    // 29 rows) 16 rows 81.5, 32 rows 75.6, 64 rows 88.8; 6 of 64..200 (2 rows) 2
    // rows 8.9, 4 rows 10.5, 8 rows 13.7; 64 of 64..512 (64 rows) 32 rows 157, 64
    // rows 153.
    // D3Q19: the chunk of up to 64 planes with the smallest modelled time of one
    // step of every domain, (planes + 4.5) times the time of a plane (as in
    // march_chunk) times the waves of CTAs; long items repeat fewer ring planes,
    // and only few or small domains need shorter ones to fill the chip.
    // Measured FP32, 64 planes -> this: 126^3 + 80^3 315 -> 215 us, four of 64^3
    // 259 -> 83, 33^3 + 46^3 + 63^3 243 -> 49, eight of 33..126 480 (64 planes).
    // FP64, whose items are bound by arithmetic, follows the same lengths: D2Q9
    // (march in items of 64 rows -> strips) 24 of 64..512 2389 -> 1571 us, 6 of
    // 64..200 722 -> 130, 2 of 1000 2142 -> 1225; D3Q19 (64 planes -> this) four
    // of 90 x 75 x 67 2837 -> 2422, 33^3 + 46^3 + 63^3 2771 -> 730, 126^3 + 80^3
    // 3746 -> 3230.
    static int batch_chunk(const lbm_batch* b) {
        std::vector<MarchGeom> in;
        for (size_t d = 0; d < b->doms.size(); ++d)
            if (d < b->in_table.size() && b->in_table[d]) in.push_back(batch_geometry(b->doms[d], 64));
        if (Q == 9) {
            double rows = 0;   // warp rows of one step of every domain
            for (const MarchGeom& G : in) rows += (double)strip_count(G.na) * G.nm;
            const double step = rows * 1.45 / (16.0 * kSms);
            const int c = (int)((0.75 * step - 2.0) / 1.45) - 4;
            return c < 2 ? 2 : (c > 64 ? 64 : c);
        }
        int best = 64;
        double best_t = 1e30;
        for (int c = 2; c <= 64; ++c) {
            long long items = 0;
            for (const MarchGeom& G : in)
                items += (long long)((G.na + TX - 1) / TX) * ((G.nb + TY - 1) / TY) * ((G.nm + c - 1) / c);
            const double t = (c + 4.5) * (items > kSms ? kModel.plane2 : kModel.plane1) *
                             std::max(1.0, (double)items / (2.0 * kSms));
            if (t <= best_t) {
                best_t = t;
                best = c;
            }
        }
        return best;
    }
    static MarchGeom batch_geometry(const lbm_handle* h, int chunk) {
        MarchGeom G;
        G.na = h->p.nx;
        G.nb = Q == 9 ? 1 : h->p.ny;
        G.nm = Q == 9 ? h->p.ny : h->p.nz;
        G.chunk = G.nm < chunk ? G.nm : chunk;
        G.m_lo = 0;
        G.m_hi = G.nm;
        return G;
    }

    // the batch kernel of shape B: with the fault-injection hook, for domains
    // with walls across the march, for the others
    static constexpr int kFault = 0, kWalls = 1, kPlain = 2;
    template <typename B> static const void* batch_kernel(int which) {
        if constexpr (Q == 9) {
            return which == kFault   ? (const void*)strip_batch_kernel<S, R, B::W, B::MB, true, true>
                   : which == kWalls ? (const void*)strip_batch_kernel<S, R, B::W, B::MB, false, true>
                                     : (const void*)strip_batch_kernel<S, R, B::W, B::MB, false, false>;
        } else {
            return which == kFault   ? (const void*)fused_batch_kernel<Q, S, R, B::TX, B::TY, B::NP, B::MB, true, true, true>
                   : which == kWalls ? (const void*)fused_batch_kernel<Q, S, R, B::TX, B::TY, B::NP, B::MB, false, true, true>
                                     : (const void*)fused_batch_kernel<Q, S, R, B::TX, B::TY, B::NP, B::MB, false, false, true>;
        }
    }
    template <typename B> static constexpr int batch_threads() {
        if constexpr (Q == 9) return 32 * B::W;
        else return B::TX * B::TY + B::NP;
    }
    template <typename B> static constexpr size_t batch_smem() {
        if constexpr (Q == 9) return B::W * Strip<S, R, true>::kRingBytes;
        else return FusedShape<B::TX, B::TY, true>::template smem_bytes<R>();
    }
    static bool has_walls(const lbm_handle* h) {
        return Q == 9 ? h->p.wall || h->p.wall_x : h->p.wall_x || h->p.wall_y;
    }

    template <typename B> static int build_shape(lbm_batch* b) {
        std::vector<BatchItem> items;
        DomainDesc<R>* descs = (DomainDesc<R>*)b->h_descs;
        const int chunk = batch_chunk(b);
        for (size_t d = 0; d < b->doms.size(); ++d) {
            lbm_handle* h = b->doms[d];
            DomainDesc<R> dd{};
            if (h) {
                dd.kp = make_kparams<R>(h);
                dd.G = batch_geometry(h, chunk);
                dd.pop[0] = h->pop[0];
                dd.pop[1] = h->pop[1];
                dd.cnt = (Counters*)h->cnt;
                dd.cur = h->cur;
                dd.left = 0;
                const int tz = (dd.G.nm + dd.G.chunk - 1) / dd.G.chunk;
                // only the domains that step in this request get work items: a
                // paused domain would cost every persistent CTA a pass over them
                const bool in = d < b->in_table.size() && b->in_table[d];
                if constexpr (Q == 9) {
                    const int warps = strip_count(dd.G.na) * tz;
                    dd.n_items = (warps + B::W - 1) / B::W;
                    for (int w = 0; in && w < warps; w += B::W) items.push_back({(int)d, w, 0, 0});
                } else {
                    const int tx = (dd.G.na + B::TX - 1) / B::TX, ty = (dd.G.nb + B::TY - 1) / B::TY;
                    dd.n_items = tx * ty * tz;
                    for (int z = 0; in && z < tz; ++z)
                        for (int y = 0; y < ty; ++y)
                            for (int x = 0; x < tx; ++x) items.push_back({(int)d, x * B::TX, y * B::TY, z * dd.G.chunk});
                }
            }
            descs[d] = dd;
        }
        if (items.size() > b->items_cap) {
            cudaFree(b->d_items);
            b->d_items = nullptr;
            b->items_cap = 0;
            if (int rc = cuda_error(cudaMalloc(&b->d_items, sizeof(BatchItem) * items.size()), "batch table")) return rc;
            b->items_cap = items.size();
        }
        b->n_items = (int)items.size();
        if (!items.empty())
            if (int rc = cuda_error(cudaMemcpyAsync(b->d_items, items.data(), sizeof(BatchItem) * items.size(),
                                                    cudaMemcpyHostToDevice, b->stream), "batch table copy"))
                return rc;
        // one persistent CTA per resident slot: occupancy times the SM count
        constexpr size_t smem = batch_smem<B>();
        b->xw = false;
        for (auto* h : b->doms) b->xw = b->xw || (h && has_walls(h));
        for (int which : {kFault, kWalls, kPlain})
            if (int rc = cuda_error(cudaFuncSetAttribute(batch_kernel<B>(which),
                                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                                    "batch kernel attribute"))
                return rc;
        int per_sm = 0, sms = 0;
        if (int rc = cuda_error(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                    &per_sm, batch_kernel<B>(b->xw ? kWalls : kPlain), batch_threads<B>(), smem),
                                "batch occupancy"))
            return rc;
        if (int rc = cuda_error(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->common.device),
                                "SM count"))
            return rc;
        b->grid = std::max(1, per_sm) * std::max(1, sms);
        return LBM_OK;
    }

    // the persistent launch of a request (steps and scheduling state already in device memory)
    template <typename B> static void launch_shape(lbm_batch* b) {
        int n_items = b->n_items, n_doms = (int)b->doms.size(), fault = b->fault_item >= 0 ? b->fault_item : -1;
        const int grid = std::max(1, b->grid);   // CTAs beyond the work of a request leave at once
        void* args[] = {&b->d_items, &b->d_descs, &n_items, &b->d_sched, &n_doms, &fault};
        cudaLaunchKernel(batch_kernel<B>(fault >= 0 ? kFault : (b->xw ? kWalls : kPlain)), dim3(grid),
                         dim3(batch_threads<B>()), args, batch_smem<B>(), b->stream);
    }

    static int batch_build(lbm_batch* b);
    static int batch_launch(lbm_batch* b, int advance);

    // sums over nodes [i0, i0 + n) and the device counters: 8 doubles at out_dev
    static int reduce(lbm_handle* h, long long i0, long long n, double* partials, double* out_dev) {
        const KParams<R> kp = make_kparams<R>(h);
        const int blocks = reduce_blocks(n);
        reduce_kernel<Q, S, R><<<blocks, kReduceThreads, 0, h->stream>>>((const S*)h->pop[h->cur], h->nn, i0, n, kp,
                                                                         partials);
        reduce_final_kernel<<<kSums, 32, 0, h->stream>>>(partials, blocks, out_dev, (const Counters*)h->cnt);
        return cuda_error(cudaGetLastError(), "conservation sums launch");
    }
};

template <int Q, typename S, typename R> int Impl<Q, S, R>::batch_build(lbm_batch* b) {
    switch (b->variant) {
        case 0: return build_shape<BatchShape<Q, 0>>(b);
        case 1: return build_shape<BatchShape<Q, 1>>(b);
        default: return build_shape<BatchShape<Q, 2>>(b);
    }
}

// One request: clear the scheduling state, the persistent launch, and (when
// `advance`) the descriptor bookkeeping of the steps taken.
template <int Q, typename S, typename R> int Impl<Q, S, R>::batch_launch(lbm_batch* b, int advance) {
    if (b->n_items > 0) {
        const size_t clear = sizeof(BatchSched) - sizeof(int) + 2 * sizeof(int) * b->doms.size();
        if (int rc = cuda_error(cudaMemsetAsync((char*)b->d_sched + sizeof(int), 0, clear, b->stream), "batch clear"))
            return rc;
        switch (b->variant) {
            case 0: launch_shape<BatchShape<Q, 0>>(b); break;
            case 1: launch_shape<BatchShape<Q, 1>>(b); break;
            default: launch_shape<BatchShape<Q, 2>>(b); break;
        }
    }
    if (advance && !b->doms.empty()) {
        const int count = (int)b->doms.size();
        batch_advance_kernel<R><<<(count + 127) / 128, 128, 0, b->stream>>>((DomainDesc<R>*)b->d_descs, count,
                                                                            (const BatchSched*)b->d_sched);
    }
    return cuda_error(cudaGetLastError(), "batch launch");
}

#define LBM_DISPATCH(h, CALL)                                                   \
    switch ((h)->p.storage) {                                                   \
        case LBM_STORE_FP64: return Impl<Q, double, double>::CALL;              \
        case LBM_STORE_FP32: return Impl<Q, float, float>::CALL;                \
        case LBM_STORE_FP16: return Impl<Q, __half, float>::CALL;               \
        default: set_error("unknown storage format"); return LBM_ERR_INVALID_ARG; \
    }

template <int Q> int Backend<Q>::step(lbm_handle* h, int n) { LBM_DISPATCH(h, step(h, n)); }
template <int Q> int Backend<Q>::step_range(lbm_handle* h, int first, int count) {
    LBM_DISPATCH(h, step_range(h, first, count));
}
template <int Q> int Backend<Q>::profile(lbm_handle* h, int n, double* ms, int cap) {
    LBM_DISPATCH(h, profile(h, n, ms, cap));
}
template <int Q> const char* Backend<Q>::launch_name(const lbm_handle* h, int j) {
    static const char* three[] = {"fields_kernel", "force_kernel", "collide_kernel"};
    if (h->p.step_kernel == LBM_STEP_THREE_LAUNCH) return j >= 0 && j < 3 ? three[j] : "";
    static const char* phase[] = {"phase_moments_kernel", "phase_force_kernel", "phase_collide_kernel"};
    if (launches(h) == 3) return j >= 0 && j < 3 ? phase[j] : "";
    if (j != 0) return "";
    switch (h->p.storage) {
        case LBM_STORE_FP64: return Impl<Q, double, double>::single_name(h);
        case LBM_STORE_FP32: return Impl<Q, float, float>::single_name(h);
        default: return Impl<Q, __half, float>::single_name(h);
    }
}
template <int Q> int Backend<Q>::launches(const lbm_handle* h) { LBM_DISPATCH(h, launches(h)); }
template <int Q> int Backend<Q>::init(lbm_handle* h, const double* rho, const double* u, const double* eps) {
    LBM_DISPATCH(h, init(h, rho, u, eps));
}
template <int Q>
int Backend<Q>::output(lbm_handle* h, const Outputs& o, Counters* cnt_out) {
    if (o.single) {
        LBM_DISPATCH(h, output(h, (float*)o.rho, (float*)o.u, (float*)o.T, (float*)o.P, cnt_out));
    }
    LBM_DISPATCH(h, output(h, (double*)o.rho, (double*)o.u, (double*)o.T, (double*)o.P, cnt_out));
}
template <int Q> int Backend<Q>::reduce(lbm_handle* h, long long i0, long long n, double* partials, double* out_dev) {
    LBM_DISPATCH(h, reduce(h, i0, n, partials, out_dev));
}
#define LBM_BATCH_DISPATCH(b, CALL)                                              \
    switch ((b)->common.storage) {                                               \
        case LBM_STORE_FP64: return Impl<Q, double, double>::CALL;               \
        case LBM_STORE_FP32: return Impl<Q, float, float>::CALL;                 \
        case LBM_STORE_FP16: return Impl<Q, __half, float>::CALL;                \
        default: set_error("unknown storage format"); return LBM_ERR_INVALID_ARG; \
    }
template <int Q> int Backend<Q>::batch_variants() { return 3; }
template <int Q> const char* Backend<Q>::batch_variant_name(int v) {
    static const char* n9[] = {"4 strips", "1 strip", "2 strips"};
    static const char* n19[] = {"32x8+128", "32x8+160", "32x4+96"};
    if (v < 0 || v > 2) return "";
    return Q == 9 ? n9[v] : n19[v];
}
template <int Q> int Backend<Q>::batch_build(lbm_batch* b) { LBM_BATCH_DISPATCH(b, batch_build(b)); }
template <int Q> int Backend<Q>::batch_launch(lbm_batch* b, int advance) { LBM_BATCH_DISPATCH(b, batch_launch(b, advance)); }
template <int Q> size_t Backend<Q>::desc_bytes(int storage) {
    return storage == LBM_STORE_FP64 ? sizeof(DomainDesc<double>) : sizeof(DomainDesc<float>);
}
#undef LBM_BATCH_DISPATCH

template <int Q> size_t Backend<Q>::field_bytes(int storage) {
    return (size_t)F_COUNT * (storage == LBM_STORE_FP64 ? sizeof(double) : sizeof(float));
}
template <int Q> bool Backend<Q>::wants_phases(const lbm_params* p) {
    switch (p->storage) {
        case LBM_STORE_FP64: return Impl<Q, double, double>::wants_phases(*p);
        case LBM_STORE_FP32: return Impl<Q, float, float>::wants_phases(*p);
        default: return Impl<Q, __half, float>::wants_phases(*p);
    }
}

#undef LBM_DISPATCH

}  // namespace lbm

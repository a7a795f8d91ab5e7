// How a step is cut: chunks of planes per CTA, rows per strip, and the modelled
// times that the choice of a form rests on (backend.cuh).  Host code without
// CUDA, so that it compiles on its own.
//
// A plan is made once per call of lbm_step or lbm_step_begin, and no search
// looks at more than kMaxChunk chunks, however long the domain.  A search over
// every chunk count on every launch bound long domains by the host: D2Q9 28 x
// 60000 230 us per step (51 now), 64 x 20000 78 (45), D3Q19 8 x 8 x 30000 346
// (181).
#pragma once

#include <algorithm>

namespace lbm {

constexpr int kSms = 152;   // SMs of a GB300

// Geometry of the march: na x nb tile plane (nb = 1 for D2Q9), nm planes.
struct MarchGeom {
    int na, nb, nm;
    int chunk;        // planes per CTA along the march axis
    int m_lo, m_hi;   // planes whose collision the launch runs (the moment and
                      // force stages reach two and one planes beyond them)
};

struct StripGeom {
    int na, nm;       // columns (x) and rows (y) of the domain
    int m_lo, m_hi;   // rows the launch collides
    int chunk;        // rows per work item
    int strips;       // ceil(na / kStripCols)
};

constexpr int kStripCols = 28;   // columns a warp collides
constexpr int strip_count(int na) { return (na + kStripCols - 1) / kStripCols; }

// A chunk longer than this loses the ring lines that neighbouring tiles share in L2.
constexpr int kMaxChunk = 64;

// f(c, n) for every way to cut len planes into n chunks of c planes, the last
// one shorter (c the least that needs no more than n), c <= kMaxChunk, longest
// chunks first, while f returns true
template <typename F> inline void each_chunk(int len, const F& f) {
    for (int c = std::min(len, kMaxChunk); c > 0; --c) {
        const int n = (len + c - 1) / c;
        if ((len + n - 1) / n == c && !f(c, n)) return;
    }
}

// D3Q19 in FP32 and FP16 storage has three forms of a step with the same
// bits, and takes the one with the smallest modelled time.  Measured us per
// step (march / row march / phases): FP32 32^3 33 / - / 7.4, 64^3 35 / 30 /
// 21.9, 80^3 54 / 42 / 51, 96^3 75 / 77 / 89, 128^3 160 / 150 / 202, 192^3 493
// / 478 / 662, 300^3 1996 / 1705 / -, 448 x 300 x 100 994 / 870 / -, 384 x 384 x
// 256 2545 / 2325 / -; FP16 64^3 33 / 24 / 18.9, 96^3 63 / 55 / 68, 128^3 140 /
// 124 / 152, 192^3 399 / 343 / 485, 384 x 384 x 256 2020 / 1710 / -.
struct StepModel {
    // phases: 4.5 us and ns per node (ns_l2 where both buffers stay in L2)
    double phase_ns, phase_ns_l2;
    // march: us of a plane while an SM holds one CTA, and two
    double plane1, plane2;
    // row march: us of a plane
    double row_plane;
    int elem;          // bytes of a stored value
    int tx, ty;        // tile of the march
    int rows;          // rows of the row march's tile
};
constexpr StepModel kModelFp32 = {0.093, 0.072, 2.7, 4.4, 2.25, 4, 32, 8, 9};
constexpr StepModel kModelFp16 = {0.070, 0.057, 2.6, 3.85, 3.1, 2, 32, 8, 16};

// Planes per CTA, and the modelled time t.
struct Chunk {
    int planes;   // 0: the form does not run
    double t;
};

// March: a CTA takes about 4.5 plane times beyond its chunk (ring planes, the
// first three planes' moments).  A plane takes plane1 us while an SM holds one
// CTA and plane2 with two (64^3 in chunks of 8 with 128 CTAs, 128^3 in chunks
// of 32 with 256), 6 % more where CTAs of several waves run out of step.  The
// chunk with the smallest modelled time avoids nearly empty last waves: FP32,
// two CTAs' worth of planes -> this: 128^3 195 -> 160 (5 -> 4 chunks), 160 x
// 128 x 96 188 -> 165, 192^3 569 -> 493.
inline Chunk march_chunk(const StepModel& m, const MarchGeom& G, int len) {
    const long long tiles = (long long)((G.na + m.tx - 1) / m.tx) * ((G.nb + m.ty - 1) / m.ty);
    Chunk best = {len, 1e30};
    each_chunk(len, [&](int c, int n) {
        const long long ctas = tiles * n, full = ctas / (2 * kSms), rest = ctas % (2 * kSms);
        const double tn = (c + 4.5) * ((double)full * m.plane2 + (rest > kSms ? m.plane2 : (rest ? m.plane1 : 0.0))) *
                          (full ? 1.06 : 1.0);
        if (tn < best.t) best = {c, tn};
        // four waves and more: the block scheduler evens out the last one
        // (384 x 384 x 256: chunks of 64 2545 us, of 52 2597)
        return tiles * ((len + kMaxChunk - 1) / kMaxChunk) < 8 * kSms;
    });
    return best;
}

// Row march (rows.cuh): one CTA per SM, (planes + 2.5) times row_plane us a
// wave.  It does not run where x has walls or a row is no multiple of 16 bytes.
inline Chunk row_chunk(const StepModel& m, const MarchGeom& G, int len, bool wall_x) {
    Chunk best = {0, 1e30};
    if (wall_x || G.na % (8 / m.elem) != 0) return best;
    const long long tiles = (long long)strip_count(G.na) * ((G.nb + m.rows - 1) / m.rows);
    each_chunk(len, [&](int c, int n) {
        const double tn = (c + 2.5) * m.row_plane * (double)((tiles * n + kSms - 1) / kSms);
        if (tn < best.t) best = {c, tn};
        return true;
    });
    return best;
}

// Phases: launches and the nodes' traffic.
inline double phase_time(const StepModel& m, const MarchGeom& G) {
    const double nodes = (double)G.na * G.nb * G.nm;
    const double ns = 4.0 * 19 * m.elem * nodes < 110e6 ? m.phase_ns_l2 : m.phase_ns;   // both buffers stay in L2
    return 4.5 + ns * 1e-3 * nodes;
}

// Warps per CTA: strips of one CTA are neighbours in x, so the ring columns
// they share come from L1.
constexpr int kStripWarps = 4;
constexpr int kStripCtas = 4;   // CTAs per SM the kernel is compiled for (128 registers)

// Rows per warp.  More rows per warp repeat fewer ring rows (the four extra
// rows of a warp cost about 1.25 full rows); fewer rows give more warps, which
// a small domain needs to fill 152 SMs.  The time of a launch is modelled as
// its waves of CTAs, each (rows + 1.25) times the time of one row with w warps
// per SM, 0.3 + 0.072 w us (measured: 0.58 us with 4, 0.85 with 8, 1.45 with
// 16), and the row count with the smallest modelled time is taken.  Measured
// us per step around the choice: 128 x 128 2 rows 3.7, 4 rows 5.0, 8 rows
// 7.5; 512 x 512 4 rows 8.4, 8 rows 9.6, 16 rows 12.7; 1000 x 1000 8 rows
// 29.3, 16 rows 27.8, 32 rows 32.8; 8192 x 4608 32 rows 903, 64 rows 895.
inline int strip_rows(int strips, int len, int sms) {
    int best = 1;
    double best_t = 1e30;
    for (int c : {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 40, 48, 64}) {
        if (c > len && c > 1) break;
        const long long warps = (long long)strips * ((len + c - 1) / c);
        const long long ctas = (warps + kStripWarps - 1) / kStripWarps;
        const long long full = ctas / ((long long)kStripCtas * sms), rest = ctas % ((long long)kStripCtas * sms);
        auto row = [&](long long per_sm) { return 0.3 + 0.072 * (double)(per_sm * kStripWarps); };
        const double t = (c + 1.25) * ((double)full * row(kStripCtas) + (rest ? row((rest + sms - 1) / sms) : 0.0));
        if (t < best_t) {
            best_t = t;
            best = c;
        }
    }
    return best;
}

}  // namespace lbm

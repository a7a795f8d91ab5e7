// The planning functions of csrc/plan.h against a search over every chunk
// count, and the time of a plan on short and long domains.
#include <chrono>
#include <cstdio>

#include "plan.h"

using namespace lbm;

// every chunk count n of len planes with chunks of at most kMaxChunk
static Chunk march_all(const StepModel& m, const MarchGeom& G, int len) {
    const long long tiles = (long long)((G.na + m.tx - 1) / m.tx) * ((G.nb + m.ty - 1) / m.ty);
    const int few = (len + 63) / 64;
    Chunk best = {len, 1e30};
    for (int n = few; n <= len; ++n) {
        const int c = (len + n - 1) / n;
        if ((len + c - 1) / c != n) continue;
        const long long ctas = tiles * n, full = ctas / 304, rest = ctas % 304;
        const double t = (c + 4.5) * ((double)full * m.plane2 + (rest > 152 ? m.plane2 : (rest ? m.plane1 : 0.0))) *
                         (full ? 1.06 : 1.0);
        if (t < best.t) best = {c, t};
        if (tiles * few >= 8 * 152) break;
    }
    return best;
}
static Chunk rows_all(const StepModel& m, const MarchGeom& G, int len) {
    Chunk best = {0, 1e30};
    if (G.na % (8 / m.elem) != 0) return best;
    const long long tiles = (long long)((G.na + 27) / 28) * ((G.nb + m.rows - 1) / m.rows);
    for (int n = (len + 63) / 64; n <= len; ++n) {
        const int c = (len + n - 1) / n;
        if ((len + c - 1) / c != n) continue;
        const double t = (c + 2.5) * m.row_plane * (double)((tiles * n + 151) / 152);
        if (t < best.t) best = {c, t};
    }
    return best;
}

static double plan_us(int nx, int ny, int nz) {
    const MarchGeom G = {nx, ny, nz, 0, 0, nz};
    double best = 1e30, sum = 0;
    for (int rep = 0; rep < 20; ++rep) {
        const auto t = std::chrono::steady_clock::now();
        for (int k = 0; k < 50; ++k)
            sum += march_chunk(kModelFp32, G, nz - (k & 1)).t + row_chunk(kModelFp32, G, nz - (k & 1), false).t +
                   strip_rows(strip_count(nx), nz - (k & 1), kSms);
        const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t).count() / 50;
        best = us < best ? us : best;
    }
    return sum > 0 ? best : 0;
}

int main() {
    int wrong = 0, checked = 0;
    for (int len : {1, 2, 3, 5, 31, 63, 64, 65, 66, 96, 127, 128, 129, 200, 256, 301, 513, 1000, 4097, 70001})
        for (int na : {2, 8, 28, 29, 64, 100, 160, 384})
            for (int nb : {1, 7, 8, 9, 16, 33, 128, 384})
                for (const StepModel* m : {&kModelFp32, &kModelFp16}) {
                    const MarchGeom G = {na, nb, len, 0, 0, len};
                    const Chunk a = march_chunk(*m, G, len), b = march_all(*m, G, len);
                    const Chunk c = row_chunk(*m, G, len, false), d = rows_all(*m, G, len);
                    wrong += a.planes != b.planes || a.t != b.t || c.planes != d.planes || c.t != d.t;
                    ++checked;
                }
    std::printf("checked %d\nwrong %d\nshort_us %.4f\nlong_us %.4f\n", checked, wrong, plan_us(8, 8, 256), plan_us(8, 8, 30000));
    return 0;
}

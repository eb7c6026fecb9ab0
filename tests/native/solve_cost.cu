// Host-side check of solve_seconds (skf_internal.cuh), the estimate by which a
// batch is dealt out to its lanes, against measured solves; prints the estimates
// and exits 1 where one is further off than a factor 1.5.
#include "../../paper_2208_11447_gb300/csrc/skf_internal.cuh"

#include <cstdio>

int main() {
    const struct {
        int m;
        double n, nnz;
        int vb, bb;
        double us;   // measured
    } solves[] = {{40, 1e4, 4.96e4, 8, 8, 663.0},       {240, 25600.0, 1.274e5, 8, 8, 4032.0},
                  {100, 4019679.0, 2.798e7, 8, 8, 16100.0}, {80, 1e6, 6.94e6, 4, 4, 2418.0},
                  {120, 16777216.0, 1.17e8, 4, 4, 28831.0}, {40, 3375000.0, 2.35e7, 4, 2, 3751.0}};
    int bad = 0;
    for (const auto &q : solves) {
        const double us = 1e6 * skf::solve_seconds(q.m, q.n, q.nnz, q.vb, q.bb);
        printf("%d %.0f: %.0f of %.0f us\n", q.m, q.n, us, q.us);
        bad += us > 1.5 * q.us || q.us > 1.5 * us;
    }
    return bad != 0;
}

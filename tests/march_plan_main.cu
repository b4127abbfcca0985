// Host program of march_plans.py. Input lines: stages flux dt precision variant sms count x y x y ...;
// output lines: columns, rows and mode of the plan, from segments that were counted one grid at a time, with others
// that came and went, and from a pass over all grids for every plan.
#include <cstdio>

#include "dugks_dvm.cuh"
#include "dugks_host.h"

using namespace dugks;
using namespace dugks::host;

namespace dugks {
int dvm_march_strips(int cols, int nx) { return cols == 2 ? DvmMarch<float2>::strips(nx) : DvmMarch<float>::strips(nx); }
}  // namespace dugks

// the rows and segments of every plan, summed over the grids anew, with the rows that the longest segment has
static MarchPlan by_passes(const MarchShape &sh, int variant, const std::vector<int2> &sizes, int precision, int sms) {
    static const int fixed[6] = {16, 8, 0, 32, 0, 64};
    const int forced = variant >= 0 && variant < 6 ? fixed[variant] : 0;
    MarchPlan best{precision == DUGKS_FP64 ? 1 : 2, 16, 0, 0, 1e300};
    for (int cols = 1; cols <= (precision == DUGKS_FP64 ? 1 : 2); cols++)
        for (int want = forced ? forced : 1; want <= (forced ? forced : 64); want++) {
            MarchWork one;
            int rows = 1;
            for (int2 q : sizes) rows = std::max(rows, march_segment_rows(want, q.y));
            for (int2 q : sizes) one.n[cols - 1][rows] += (int64_t)sh.strips(cols, q.x) * march_segments(want, q.y);
            // (the cost of one plan: every other number of rows and columns is made too dear)
            for (int c = 0; c < 2; c++)
                for (int r = 1; r <= MARCH_ROWS; r++)
                    if (c != cols - 1 || r != rows) one.n[c][r] = (int64_t)1 << 50;
            MarchPlan p = march_plan(sh, -1, one, nullptr, 0, precision, sms);
            const double n = (double)one.n[cols - 1][rows] / (4.0 * sms);
            if (precision == DUGKS_FP64 && n > 0.8 && n <= 1.0) p.cost /= 1.1;   // (added once a plan is chosen)
            if (p.cost < best.cost) best = MarchPlan{cols, want, p.early, p.one_wave, p.cost};
        }
    return best;
}

int main() {
    int stages, flux, precision, variant, sms, count;
    double dt;
    while (std::scanf("%d %d %lf %d %d %d %d", &stages, &flux, &dt, &precision, &variant, &sms, &count) == 7) {
        const MarchShape &sh = stages == 1 ? dvm_shape(dt) : march_shape(stages, flux);
        std::vector<int2> sizes(count);
        MarchWork work;
        for (int2 &q : sizes) {
            if (std::scanf("%d %d", &q.x, &q.y) != 2) return 1;
            work.count(sh, q, 1);
            work.count(sh, make_int2(q.y + 3, q.x), 1);   // a grid that leaves again
        }
        for (int2 q : sizes) work.count(sh, make_int2(q.y + 3, q.x), -1);
        const MarchPlan a = march_plan(sh, variant, work, sizes.data(), count, precision, sms);
        const MarchPlan b = by_passes(sh, variant, sizes, precision, sms);
        std::printf("%d %d %d %d %d %d\n", a.cols, a.rows, a.mode(), b.cols, b.rows, b.mode());
    }
    return 0;
}

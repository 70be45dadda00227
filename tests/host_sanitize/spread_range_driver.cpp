// Host-only check of the range of cells a brick of the spreading kernel lists (usr_internal.h, spread_cells), run by
// tests/test_host_spread_range.py: exact in single precision, over every wrapped coordinate.
//
// Along an axis, an atom at wrapped coordinate x (0 <= x <= L) has cell id cell(x) and grid coordinate floor(x gs),
// both non-decreasing in x, and its image in period k the cell cell(x) + k nc and the point floor(x gs) + k n.  For
// every brick [o, o + e), every k and the coordinates whose stencil reaches the brick, the ends of that interval
// of floats are found by binary search over bit patterns; the cells of both ends, hence of all between, have to
// lie in the range that the kernel walks, and the stencil's first point relative to the brick, plus 32, in 8 bits.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "usr_internal.h"

namespace {

float bits_to_float(uint32_t u)
{
    float f;
    std::memcpy(&f, &u, sizeof f);
    return f;
}

uint32_t float_to_bits(float f)
{
    uint32_t u;
    std::memcpy(&u, &f, sizeof u);
    return u;
}

/* The binning kernel's cell of a wrapped coordinate, and the spreading kernel's grid point. */
int cell_of(float x, float cs, int nc)
{
    const float u = x * cs;
    const int c = u >= 0.0f ? (int)u : 0;
    return c > nc - 1 ? nc - 1 : c;
}

int point_of(float x, float gs) { return (int)std::floor(x * gs); }

/* Bits of the smallest x in [0, top] with point_of(x) >= f (top + 1 if there is none). */
uint32_t first_at(int f, float gs, uint32_t top)
{
    uint32_t lo = 0, hi = top + 1;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (point_of(bits_to_float(mid), gs) >= f) hi = mid; else lo = mid + 1;
    }
    return lo;
}

long check_axis(double Ld, int n, int nc, int P, int brick, float margin)
{
    const float L = (float)Ld, cs = (float)((double)nc / Ld), gs = (float)((double)n / Ld);
    const uint32_t top = float_to_bits(L);
    const int H = P / 2;
    long bad = 0;
    for (int o = 0; o < n; o += brick) {
        const int e = std::min(brick, n - o);
        int c0, c1;
        usr::spread_cells(o, e, H, n, nc, margin, &c0, &c1);
        // points f (unwrapped) with f - H + 1 < o + e and f + H >= o; x gs may round up to n itself
        const int f0 = o - H, f1 = o + e + H - 2;
        for (int k = -3; k <= 3; ++k) {
            const int a = f0 - k * n, b = f1 - k * n;
            if (b < 0 || a > n) continue;
            const uint32_t x0 = first_at(std::max(a, 0), gs, top), x1 = first_at(b + 1, gs, top);
            if (x0 >= x1) continue;
            const float ends[2] = {bits_to_float(x0), bits_to_float(x1 - 1)};
            for (float x : ends) {
                const int c = cell_of(x, cs, nc) + k * nc, s = point_of(x, gs) + k * n - o - H + 1 + 32;
                if (c < c0 || c > c1 || s < 0 || s > 255) ++bad;
            }
        }
    }
    return bad;
}

/* A fixed pseudo-random sequence (the same everywhere). */
double uniform(uint64_t* s)
{
    *s = *s * 6364136223846793005ULL + 1442695040888963407ULL;
    return (double)(*s >> 11) * (1.0 / 9007199254740992.0);
}

}  // namespace

int main(int argc, char** argv)
{
    const float margin = argc > 1 ? (float)std::atof(argv[1]) : usr::kSpreadMargin;
    long bad = 0, axes = 0;
    // the boxes and grids of the workloads, every cell count, both brick edges, every stencil
    const double box[] = {26.0, 31.0, 47.9, 58.5, 80.0, 100.0, 126.0, 220.0};
    const int grid[] = {24, 32, 47, 48, 64, 80, 128, 176};
    for (int i = 0; i < 8; ++i)
        for (int nc = 3; nc <= grid[i]; ++nc)
            for (int P : {8, 10, 12, 14, 16})
                for (int brick : {8, 16}) {
                    if (grid[i] < P + 8) continue;
                    bad += check_axis(box[i], grid[i], nc, P, brick, margin);
                    ++axes;
                }
    // any box side up to 1e5, any grid up to 4,096 points, any cell count up to one per point
    uint64_t s = 12345;
    for (int t = 0; t < 10000; ++t) {
        const int P = 8 + 2 * (int)(5 * uniform(&s));
        const int n = std::min(4096, std::max(P + 8, (int)std::exp(std::log(16.0) + std::log(256.001) * uniform(&s))));
        const int nc = 3 + (int)((n - 2) * uniform(&s));
        const double L = std::exp(std::log(1.0) + std::log(1.0e5) * uniform(&s));
        bad += check_axis(L, n, std::min(nc, n), P, t % 3 == 0 ? 16 : 8, margin);
        ++axes;
    }
    for (double L : {1.0e5, 99999.99, 3.3333, 1024.0})
        for (int nc : {3, 7, 511, 512, 1365, 2047, 4095, 4096}) {
            bad += check_axis(L, 4096, nc, 16, 8, margin);
            ++axes;
        }
    std::printf("axes %ld violations %ld\n", axes, bad);
    return bad == 0 ? 0 : 1;
}

double usr::plan_device_bytes(const usr::Plan&) { return 0.0; }   // (declared for the plan; not used here)

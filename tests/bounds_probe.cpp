// Host build of the update formula and of the lower bounds of the cells it makes
// (lw_internal.h), over seeded operands; called by test_bounds.py.
#include "../paper_1709_06816_gb300/csrc/lw_internal.h"

#include <random>

namespace {

// The bound as the formula gives it in 64 bits, without the margin: what a
// kernel that forgot its roundings would compare with (the planted mistake).
double plain_bound(int lk, double la, double lb, double w, double h)
{
    switch (lk) {
    case 0: return la < lb ? la : lb;
    case 1: return la > lb ? la : lb;
    case 4: return 0.5 * la + 0.5 * lb;
    case 5: return w * la + (1.0 - w) * lb - w * (1.0 - w) * h;
    default: return w * la + (1.0 - w) * lb;
    }
}

template <int LK>
void check(unsigned long long seed, long long count, long long *out)
{
    std::mt19937_64 g(seed);
    auto uniform = [&](double lo, double hi) { return lo + (hi - lo) * (double)(g() >> 11) * 0x1p-53; };
    auto size = [&]() { return 1 + (int)exp2(uniform(0.0, 21.0)); };
    // x, or a value somewhat or only a few units in the last place above it
    auto above = [&](float x) -> float {
        switch (g() % 4) {
        case 0: return x;
        case 1: return lw::value_of(lw::bits_of(x) + (unsigned)(g() % 8));
        case 2: return (float)(x * (1.0 + exp2(uniform(-22.0, 0.0))));
        default: return (float)(x * exp2(uniform(0.0, 8.0)));
        }
    };
    for (long long c = 0; c < count; ++c) {
        const float h = g() % 16 ? (float)exp2(uniform(-20.0, 20.0)) : 0.0f;
        const float base = h > 0.0f ? h : (float)exp2(uniform(-20.0, 20.0));
        // bounds of the two parts' cells and the cells themselves
        const float la = above(base), lb = g() % 3 ? above(base) : la;
        const float a = above(la), b = g() % 3 ? above(lb) : lb;
        const float dmax = above(a > b ? a : b);
        const int ni = size(), nj = size(), nk = size();
        const float fi = (float)ni, fs = (float)(ni + nj);
        const float4 co = lw::merge_coefs<LK>(ni, nj, h);
        const float v = LK == 3 ? lw::ward_cell(fi, (float)nj, fs, (float)nk, h, a, b)
                                : lw::lw_sum(co.x, co.y, co.z, co.w, a, b);
        const unsigned bound =
            lw::merged_bound<LK>((int)lw::bits_of(la), (int)lw::bits_of(lb), fi, fs, h, lw::bits_of(dmax));
        const double plain = plain_bound(LK, la, lb, (double)ni / ((double)ni + nj), h);
        out[0] += lw::bits_of(v) < bound;                  // a cell below its bound
        out[1] += (double)v < plain;                       // the margin was needed
        out[2] += (double)lw::value_of(bound) < 0.999 * plain - 1e-5 * (LK == 0 ? dmax : 0.0f);  // a useless bound
        // a part without cells outside is above everything
        out[3] += lw::merged_bound<LK>(-1, -1, fi, fs, h, lw::bits_of(dmax)) != 0xffffffffu;
    }
}

}  // namespace

extern "C" void bounds_check(int linkage, unsigned long long seed, long long count, long long *out)
{
    switch (linkage) {
    case 0: check<0>(seed, count, out); break;
    case 1: check<1>(seed, count, out); break;
    case 2: check<2>(seed, count, out); break;
    case 3: check<3>(seed, count, out); break;
    case 4: check<4>(seed, count, out); break;
    default: check<5>(seed, count, out); break;
    }
}

extern "C" unsigned bound_of(int linkage, float la, float lb, float fi, float fs, float h, float dmax)
{
    const int x = (int)lw::bits_of(la), y = (int)lw::bits_of(lb);
    const unsigned d = lw::bits_of(dmax);
    switch (linkage) {
    case 0: return lw::merged_bound<0>(x, y, fi, fs, h, d);
    case 1: return lw::merged_bound<1>(x, y, fi, fs, h, d);
    case 2: return lw::merged_bound<2>(x, y, fi, fs, h, d);
    case 3: return lw::merged_bound<3>(x, y, fi, fs, h, d);
    case 4: return lw::merged_bound<4>(x, y, fi, fs, h, d);
    default: return lw::merged_bound<5>(x, y, fi, fs, h, d);
    }
}

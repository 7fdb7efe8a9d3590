// pp_sym_plan.h -- the work plan of a pair-symmetric pass (pp_sym.cuh): which target
// blocks meet which sources in one item of work, and where the partial sums go.
// Host code without CUDA headers, so that a plain C++ program can check it.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

#ifdef __CUDACC__
#define PP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define PP_HOST_DEVICE inline
#endif

namespace ppk {

// One item of work: target blocks [ib0, ib0 + nb) against sources [j0, j1)
// (multiples of the kernel's unit).
struct SymItem {
    int ib0, nb, j0, j1;
};
// The items of one group of target blocks: `items` of them from `first` on.
struct alignas(8) SymRow {
    int first, items;
};
constexpr int kSymUnit = 64;     // sources: FP32 kernels
constexpr int kSym64Unit = 32;   // all-FP64 kernel

// Partial-sum rows: at most this many groups of target blocks, so the rows take
// at most 12 * kSymMaxRows bytes per particle.
constexpr int kSymMaxRows = 128;
constexpr int kSymThreads = 128;
constexpr int kSymWarps = kSymThreads / 32;

// Doubles before the row of group g (rows are packed: row g starts at source g * bis).
PP_HOST_DEVICE size_t sym_row_offset(int g, int npad, int bis)
{
    return 3 * ((size_t)g * npad - (size_t)bis * ((size_t)g * (g - 1) / 2));
}

struct SymPlan {
    int ki = 1;                  // target blocks per group
    std::vector<SymItem> items;
    std::vector<SymRow> rows;
    size_t row_doubles = 0, part_doubles = 0;
};

// May a pass take `bytes` for its partial sums with `free` bytes left on the device?
// A quarter of them at most: what else shares the GPU (other contexts, the program's
// own arrays) still finds room, and the pass has a one-sided form that needs none.
inline bool sym_sums_fit(size_t bytes, size_t free) { return bytes <= free / 4; }

// Work items of one pass over blocks of `targets` particles with `slots` CTAs
// resident: each group of ki target blocks walks the sources from its own start to
// the end; its row is cut into ranges of half a resident warp's share of the
// remaining work (at most a quarter of its share of the whole: the warps of a
// scheduler do not advance evenly, with whole shares at the start the pass took
// 40 % longer), long ranges first, so the tail of the pass is short.
// The shortest range (`least`) is chosen by the units of work per resident warp, r:
// 64 sources where 128 would leave fewer than 1.6 rounds of items, 256 where that
// leaves about two to three and a half, else 128 (one long item too many costs a whole
// round; above, ranges hardly matter).  ms per step with 64 / 128 / 256 sources:
//   r = 2.3  hi/lo   N = 13001  0.112 / 0.142 / 0.147      2.6  guarded 14336  0.109 / 0.123 / 0.160
//   r = 3.5  single  14336      0.099 / 0.090 / 0.127      5.1  single  16385  0.145 / 0.123 / 0.163
//   r = 5.9  guarded 20481      0.201 / 0.184 / 0.225      7.0  weights 22529  0.247 / 0.228 / 0.238
//   r = 7.7  guarded 24576      0.260 / 0.243 / 0.234      9.1  Kahan   32768  0.366 / 0.353 / 0.326
//   r = 13.6 weights 32768      0.396 / 0.391 / 0.373     17.6  weights 36865  0.524 / 0.520 / 0.528
// split > 0 shortens the ranges to npad / split where they are longer; it never
// lengthens them, since the warps without work wait for the last item, and a row
// on one warp takes seconds at N = 2^20.  Each item keeps its own sums, which
// bounds how finely the work may be cut: rows and items take 4 to 7 KB per particle
// from N = 65536 on.
inline SymPlan make_sym_plan(int n, int npad, int targets, bool f64, int64_t slots, int split)
{
    SymPlan pl;
    const int unit = f64 ? kSym64Unit : kSymUnit, BU = targets / unit, nu = npad / unit;
    const int nib = (n + targets - 1) / targets;
    // the rows of partial sums take 24 bytes x npad x groups / 2
    pl.ki = std::max(1, (nib + kSymMaxRows - 1) / kSymMaxRows);
    const int groups = (nib + pl.ki - 1) / pl.ki;
    double left = 0.0;
    for (int g = 0; g < groups; ++g)
        left += (double)std::min(pl.ki, nib - g * pl.ki) * (nu - g * pl.ki * BU);
    const double warps = kSymWarps * (double)slots, most = left / (4.0 * warps);
    const double r = left / warps;
    const int least = f64 || r < 3.2 ? 1 : r >= 7.4 && r < 14.0 ? 4 : 2;
    const int cap = split > 0 ? std::max(1, (nu + split - 1) / split) : nu;
    for (int g = 0; g < groups; ++g) {
        const int ib0 = g * pl.ki, nb = std::min(pl.ki, nib - ib0);
        const int first = (int)pl.items.size();
        for (int u = ib0 * BU; u < nu;) {
            int len = (int)(std::min(left / (2.0 * warps), most) / nb);
            len = std::min({std::max(len, least), cap, nu - u});
            pl.items.push_back(SymItem{ib0, nb, u * unit, (u + len) * unit});
            left -= (double)nb * len;
            u += len;
        }
        pl.rows.push_back(SymRow{first, (int)pl.items.size() - first});
    }
    pl.row_doubles = sym_row_offset(groups, npad, pl.ki * targets);
    pl.part_doubles = pl.items.size() * pl.ki * 3 * (size_t)targets;
    return pl;
}

}  // namespace ppk

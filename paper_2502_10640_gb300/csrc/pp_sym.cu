// pp_sym.cu -- instantiations, work plan and launcher of the pair-symmetric
// force kernels (pp_sym.cuh).
#include <algorithm>

#include "pp_internal.h"
#include "pp_sym64.cuh"

namespace ppk {

namespace {

template <int PK, int TJ, int POS, bool WEIGHTED, bool KAHAN, int MINB, bool BOX = false>
Variant make_sym(const char *name)
{
    Variant v{name, WEIGHTED ? KIND_FORCE32W : KIND_FORCE32, KAHAN ? ACC_KAHAN : ACC_FP64FOLD,
              POS == POS_SINGLE ? STAGE_F32I : STAGE_F32IX2, kSymThreads, 2 * PK, TJ, 0,
              reinterpret_cast<const void *>(
                  &force_sym_kernel<PK, TJ, POS, BOX, WEIGHTED, KAHAN, MINB>),
              kSymWarps * sym_warp_smem<PK, TJ>(), 0, POS, BOX ? 1 : 0};
    v.sym = 1;
    return v;
}

template <bool WEIGHTED>
Variant make_sym64(const char *name)
{
    Variant v{name, KIND_FORCE64, ACC_FP64FULL, STAGE_F64, kSymThreads,
              kSym64Targets / 32, kSym64Unit, 0,
              reinterpret_cast<const void *>(&force_sym64_kernel<WEIGHTED>), 0, 0, POS_SINGLE};
    v.sym = 1;
    return v;
}

}  // namespace

// Registers: three CTAs of 168 (PK = 8) or 128 to 168 (PK = 4) per thread; the
// weighted PK = 8 loop holds 16 more and runs two CTAs.  rsqrt(s)^3 is two packed
// products: 1/s from the SFU in place of one of them was slower at every size (ms
// with it and without: guarded N = 40001, 8 steps 4.75 / 4.60, single 65536,
// 8 steps 9.86 / 9.53, 2^20 261.2 / 260.4).
std::vector<Variant> sym_variants()
{
    return {
#define S(nm, ...) make_sym<__VA_ARGS__>(nm)
        S("f32x2.fold64.sym4k128", 4, 128, POS_SINGLE, false, false, 3),
        S("f32x2.fold64.sym8k256", 8, 256, POS_SINGLE, false, false, 3),
        S("f32x2.fold64.sym8k512", 8, 512, POS_SINGLE, false, false, 3),
        S("f32x2.kahan.sym4k128", 4, 128, POS_SINGLE, false, true, 4),
        S("f32x2.kahan.sym8k256", 8, 256, POS_SINGLE, false, true, 3),
        S("f32x2guard.fold64.sym4k128", 4, 128, POS_GUARDED, false, false, 4),
        S("f32x2guard.fold64.sym8k128", 8, 128, POS_GUARDED, false, false, 3),
        S("f32x2guard.kahan.sym4k128", 4, 128, POS_GUARDED, false, true, 4),
        S("f32x2guard.kahan.sym8k128", 8, 128, POS_GUARDED, false, true, 3),
        S("f32x2bguard.sfold64.sym8k128", 8, 128, POS_GUARDED, false, false, 3, true),
        S("f32x2bguard.sfold64.sym8k256", 8, 256, POS_GUARDED, false, false, 3, true),
        S("f32x2bguard.kahan.sym8k256", 8, 256, POS_GUARDED, false, true, 3, true),
        S("f32x2split.fold64.sym4k128", 4, 128, POS_SPLIT, false, false, 4),
        S("f32x2split.kahan.sym4k128", 4, 128, POS_SPLIT, false, true, 4),
        S("f32x2w.fold64.sym4k128", 4, 128, POS_SINGLE, true, false, 4),
        S("f32x2w.fold64.sym8k256", 8, 256, POS_SINGLE, true, false, 2),
        S("f32x2wguard.fold64.sym4k128", 4, 128, POS_GUARDED, true, false, 4),
        S("f32x2wbguard.sfold64.sym8k256", 8, 256, POS_GUARDED, true, false, 2, true),
        S("f32x2wsplit.fold64.sym4k128", 4, 128, POS_SPLIT, true, false, 3),
#undef S
        make_sym64<false>("f64.full.symr1k32"),
        make_sym64<true>("f64w.full.symr1k32"),
    };
}

// Work items of one pass: each group of ki target blocks walks the sources from
// its own start to the end; its row is cut into ranges of half a resident warp's
// share of the remaining work (at most a quarter of its share of the whole: the
// warps of a scheduler do not advance evenly, with whole shares at the start the
// pass took 40 % longer), long ranges first, so the tail of the pass is short.
// The shortest range is 128 sources, 256 where that leaves two to four rounds
// of items (ms per step, 128 against 256: 0.104 / 0.152 at N = 16384, 0.213 /
// 0.196 at 24576, 0.339 / 0.315 at 32768, 1.16 / 1.17 at 65536).  split > 0 cuts
// every row into npad / split.  Each item keeps its own sums, which bounds how
// finely the work may be cut: rows and items take 5 KB per particle at 2^20.
SymPlan make_sym_plan(int n, int npad, const Variant &v, int64_t slots, int split)
{
    SymPlan pl;
    const bool f64 = v.kind == KIND_FORCE64;
    const int WI = 32 * v.R, unit = f64 ? kSym64Unit : kSymUnit, BU = WI / unit, nu = npad / unit;
    const int nib = (n + WI - 1) / WI;
    // the rows of partial sums take 24 bytes x npad x groups / 2
    pl.ki = std::max(1, (nib + kSymMaxRows - 1) / kSymMaxRows);
    const int groups = (nib + pl.ki - 1) / pl.ki;
    double left = 0.0;
    for (int g = 0; g < groups; ++g)
        left += (double)std::min(pl.ki, nib - g * pl.ki) * (nu - g * pl.ki * BU);
    const double warps = kSymWarps * (double)slots, most = left / (4.0 * warps);
    const int least = f64 ? 1 : n >= 20480 && n < 40960 ? 4 : 2;
    for (int g = 0; g < groups; ++g) {
        const int ib0 = g * pl.ki, nb = std::min(pl.ki, nib - ib0);
        const int first = (int)pl.items.size();
        for (int u = ib0 * BU; u < nu;) {
            int len = split > 0 ? (nu + split - 1) / split
                                : (int)(std::min(left / (2.0 * warps), most) / nb);
            len = std::max(1, std::min(std::max(len, split > 0 ? 1 : least), nu - u));
            pl.items.push_back(SymItem{ib0, nb, u * unit, (u + len) * unit});
            left -= (double)nb * len;
            u += len;
        }
        pl.rows.push_back(make_int2(first, (int)pl.items.size() - first));
    }
    pl.row_doubles = sym_row_offset(groups, npad, pl.ki * WI);
    pl.part_doubles = pl.items.size() * pl.ki * 3 * (size_t)WI;
    return pl;
}

cudaError_t launch_sym(const Variant &v, const ForceArgs &a, const SymArgs &q, int grid,
                       cudaStream_t stream)
{
    static DeviceOnce smem_attr;
    int count = 0;
    const int idx = (int)(&v - variants(&count));
    const cudaError_t e = smem_attr.run(idx, [&] {
        return cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.smem);
    });
    if (e != cudaSuccess) return e;
    ForceArgs ac = a;
    SymArgs qc = q;
    void *args[] = {&ac, &qc};
    return cudaLaunchKernel(v.fn, dim3(grid), dim3(v.T), args, v.smem, stream);
}

}  // namespace ppk

// pp_sym.cu -- instantiations and launcher of the pair-symmetric force kernels
// (pp_sym.cuh; the work plan is in pp_sym_plan.h).
#include "pp_internal.h"
#include "pp_sym64.cuh"

namespace ppk {

namespace {

template <int PK, int TJ, int POS, bool WEIGHTED, bool KAHAN, int MINB, bool BOX = false,
          bool HALF = false>
Variant make_sym(const char *name)
{
    Variant v{name, WEIGHTED ? KIND_FORCE32W : KIND_FORCE32, KAHAN ? ACC_KAHAN : ACC_FP64FOLD,
              POS == POS_SINGLE ? STAGE_F32I : STAGE_F32IX2, kSymThreads, 2 * PK, TJ, 0,
              reinterpret_cast<const void *>(
                  &force_sym_kernel<PK, TJ, POS, BOX, WEIGHTED, KAHAN, MINB, HALF>),
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
        S("f32x2.fold64.sym4k64", 4, 64, POS_SINGLE, false, false, 3),
        S("f32x2.fold64.sym8k128h", 8, 128, POS_SINGLE, false, false, 3, false, true),
        S("f32x2.fold64.sym8k256", 8, 256, POS_SINGLE, false, false, 3),
        S("f32x2.fold64.sym8k512", 8, 512, POS_SINGLE, false, false, 3),
        S("f32x2.kahan.sym4k64", 4, 64, POS_SINGLE, false, true, 4),
        S("f32x2.kahan.sym8k64", 8, 64, POS_SINGLE, false, true, 3),
        S("f32x2.kahan.sym8k256", 8, 256, POS_SINGLE, false, true, 3),
        S("f32x2guard.fold64.sym4k64", 4, 64, POS_GUARDED, false, false, 4),
        S("f32x2guard.kahan.sym4k64", 4, 64, POS_GUARDED, false, true, 4),
        S("f32x2guard.kahan.sym4k128", 4, 128, POS_GUARDED, false, true, 4),
        S("f32x2guard.kahan.sym8k128", 8, 128, POS_GUARDED, false, true, 3),
        S("f32x2bguard.sfold64.sym8k128", 8, 128, POS_GUARDED, false, false, 3, true),
        S("f32x2bguard.sfold64.sym8k256", 8, 256, POS_GUARDED, false, false, 3, true),
        S("f32x2bguard.kahan.sym8k256", 8, 256, POS_GUARDED, false, true, 3, true),
        S("f32x2split.fold64.sym4k128", 4, 128, POS_SPLIT, false, false, 4),
        S("f32x2split.kahan.sym4k128", 4, 128, POS_SPLIT, false, true, 4),
        S("f32x2w.fold64.sym4k128h", 4, 128, POS_SINGLE, true, false, 4, false, true),
        S("f32x2w.fold64.sym8k256", 8, 256, POS_SINGLE, true, false, 2),
        S("f32x2wguard.fold64.sym4k64", 4, 64, POS_GUARDED, true, false, 4),
        S("f32x2wguard.fold64.sym4k128", 4, 128, POS_GUARDED, true, false, 4),
        S("f32x2wbguard.sfold64.sym8k256", 8, 256, POS_GUARDED, true, false, 2, true),
        S("f32x2wsplit.fold64.sym4k128", 4, 128, POS_SPLIT, true, false, 3),
#undef S
        make_sym64<false>("f64.full.symr1k32"),
        make_sym64<true>("f64w.full.symr1k32"),
    };
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

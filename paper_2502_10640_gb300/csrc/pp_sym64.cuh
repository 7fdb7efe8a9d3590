// pp_sym64.cuh -- the all-FP64 Coulomb sum over unordered pairs, on the queue and
// partial sums of pp_sym.cuh.
//
// What bounds it: the FP64 pipe, which takes 64 cycles per warp instruction and
// scheduler on this GPU; everything else is free beside it.  A pair costs 18 FP64
// operations for both directions (3 sub, 3 fma for d.d + eps^2, 6 for
// s^(-3/2), 6 fma), so the inverse square root and its cube are not taken from
// the library: y0 = rsqrt.approx of the upper word of s (about 20 bits, no FP64
// operation) and, with e = 1 - s y0^2, the series
//   s^(-3/2) = y0^3 (1 - e)^(-3/2) = y0^3 (1 + 3/2 e + 15/8 e^2 + O(e^3)),
// whose next term is below 2^-55.  Masks (self, zero distance, padding) are
// integer tests on the bits of s.  The one-sided kernel with the library's
// rsqrt takes 10.4 ms per pass at N = 16385, this one 5.04, with the pipe 88 % busy.
//
// A warp owns 32 targets (one per lane, its sums in registers over a whole item)
// and rotates 32 sources at a time through its lanes, as pp_sym.cuh does; with
// two targets per lane the units of work are twice as long for nothing (5.36
// against 5.04 ms per pass at N = 16385, 0.46 against 0.32 at 4096).  Two CTAs
// per SM: the pipe needs no more than two warps per scheduler, and fewer warps
// make the last items shorter.
#pragma once

#include "pp_sym.cuh"

namespace ppk {

constexpr int kSym64Targets = 32, kSym64Ctas = 2;

// s^(-3/2) for 0 < s <= inf.
__device__ __forceinline__ double inv_cube_root2(double s)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
    const double t = y * y;   // y has at most 21 significant bits: exact
    const double e = fma(-s, t, 1.0);
    const double y3 = y * t;
    const double c = fma(y3 * e, fma(1.875, e, 1.5), y3);
    // at the ends of the range the series would give inf - inf or 0 * NaN: s below 1e-205
    // has y3 = inf, s = inf has y3 = 0 (tested by its bits)
    return (unsigned long long)__double_as_longlong(y3) - 1ull < 0x7fefffffffffffffull ? c : y3;
}

template <bool WEIGHTED>
__global__ void __launch_bounds__(kSymThreads, kSym64Ctas)
    force_sym64_kernel(const ForceArgs p, const SymArgs q)
{
    constexpr int WI = kSym64Targets;
    __shared__ double scratch[2 * 384];
    __shared__ int s_next[2];
    const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
    const double4 *src = static_cast<const double4 *>(p.src);
    const int bis = WI * q.ki;
    auto pop = [&] { return lane == 0 ? (int)atomicAdd(&q.ctl[SYM_NEXT], 1u) : 0; };
    int ahead = pop(), done = 0;
    for (;; ++done) {
        const int item = __shfl_sync(0xffffffffu, ahead, 0);
        if (item >= q.nitems) break;
        ahead = pop();
        const SymItem it = q.items[item];
        const int grp = it.ib0 / q.ki;
        double *jrow = q.jrow + sym_row_offset(grp, p.npad, bis);
        const size_t plane = (size_t)p.npad - (size_t)grp * bis;
        for (int kb = 0; kb < it.nb; ++kb) {
            const int i0 = (it.ib0 + kb) * WI, i = i0 + lane;
            const bool real = i < p.n;
            const double4 t = real ? src[i] : make_double4(0.0, 0.0, 0.0, 0.0);
            double a[3] = {0.0, 0.0, 0.0};
            for (int j = max(it.j0, i0); j < it.j1; j += 32) {
                const bool mine = j < i0 + WI;   // the sources are among the targets
                double4 s = src[j + lane];
                double f[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
                for (int r = 0; r < 32; ++r) {
                    const int jr = j + ((lane + r) & 31);
                    double dx = t.x - s.x, dy = t.y - s.y, dz = t.z - s.z;
                    const double d2 = fma(dz, dz, fma(dy, dy, fma(dx, dx, p.eps2d)));
                    // 0 < d2 <= inf by its bits; a pair with d2 not a number adds nothing at
                    // all (0 * NaN would stay in both sums)
                    const bool some = (unsigned long long)__double_as_longlong(d2) - 1ull <
                                      0x7ff0000000000000ull;
                    const bool on = some && jr < p.n && real && jr != i;
                    dx = some ? dx : 0.0;
                    dy = some ? dy : 0.0;
                    dz = some ? dz : 0.0;
                    double c = inv_cube_root2(d2);
                    c = on ? c : 0.0;
                    const double ci = WEIGHTED ? c * s.w : c;
                    a[0] = fma(ci, dx, a[0]);
                    a[1] = fma(ci, dy, a[1]);
                    a[2] = fma(ci, dz, a[2]);
                    if (!mine) {
                        const double cj = WEIGHTED ? c * t.w : c;
                        f[0] = fma(cj, dx, f[0]);
                        f[1] = fma(cj, dy, f[1]);
                        f[2] = fma(cj, dz, f[2]);
                    }
                    s.x = __shfl_sync(0xffffffffu, s.x, next);
                    s.y = __shfl_sync(0xffffffffu, s.y, next);
                    s.z = __shfl_sync(0xffffffffu, s.z, next);
                    if (WEIGHTED) s.w = __shfl_sync(0xffffffffu, s.w, next);
#pragma unroll
                    for (int c = 0; c < 3; ++c) f[c] = __shfl_sync(0xffffffffu, f[c], next);
                }
                if (mine && kb > 0) continue;   // the group's row has been started
                double *out = jrow + (j + lane - grp * bis);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double v = kb > 0 ? ld_cg(out + c * plane) : 0.0;
                    __stcg(out + c * plane, v - f[c]);
                }
            }
            double *part = q.ipart + ((size_t)item * q.ki + kb) * 3 * WI;
#pragma unroll
            for (int c = 0; c < 3; ++c) __stcg(part + c * WI + lane, a[c]);
        }
    }
    sym_collect<WI, STAGE_F64>(p, q, done, scratch, s_next);
}

}  // namespace ppk

// pp_sym.cuh -- the O(N^2) Coulomb sum over unordered pairs: every pair term is
// evaluated once and added to both particles (Newton's third law).
//
// What bounds it: the FP32 pipe.  A pair costs 14 FP32 lane operations (3 sub,
// 3 fma for d.d + eps^2, 2 mul for the cube, 3 fma into each particle) and one
// SFU rsqrt, so 7 operations per interaction against 11 of the one-sided
// kernels of pp_force.cuh.
//
// Decomposition.  A warp owns a block of WI = 64 PK targets (each lane PK packs
// of two targets, positions and FP32 sums in registers) and walks a range of
// sources at or after its block in tiles of at most TJ (64 to 512: TJ is the length of
// a target's FP32 partial sum; HALF keeps two of TJ / 2).  The 32 sources of a subtile sit
// one per lane and rotate through the lanes by shuffle together with their
// three sums, so after 32 steps each source has met all WI targets and is home
// again: no cross-lane reduction, no shared-memory traffic in the loop (9
// shuffles per 16 PK f32x2 operations).  f32x2 lanes hold two targets, so a
// source's sum splits into an even-target and an odd-target partial, each 32 PK
// terms long.  Warps are independent of one another (a barrier per tile among
// the four warps of a CTA cost 12 % of the issue slots): each pulls work items
// from a queue.
//
// Folds.  Per tile the FP32 sums of the targets go to FP64 (or compensated
// FP32) accumulators in shared memory, those of the sources to the FP64 row of
// partial sums of this group of target blocks.  A work item writes its targets'
// sums when it ends.  When all items are done (a bounded wait on a counter), the
// CTAs share out the particles, add each one's partial sums in an order fixed
// by the plan and run the push (finish_particle).  Who does what depends on the
// run, every sum and its order does not: results are bitwise reproducible, and
// the whole pass is one launch.
//
// Pairs inside one warp's own targets (the diagonal) are summed one-sided with
// zero-distance pairs skipped.
#pragma once

#include "pp_force.cuh"
#include "pp_sym_plan.h"

namespace ppk {

// The queue words of a pass, zero between launches (the last CTA to leave
// clears them).
enum SymCtl : int { SYM_NEXT = 0, SYM_DONE = 1, SYM_FINISH = 2, SYM_LEFT = 3, SYM_CTL = 4 };

// Least limit of the wait for a pass's last items (sym_collect).
constexpr uint64_t kSymMinWaitNs = 1000000000ull;

struct SymArgs {
    const SymItem *items;
    const SymRow *rows;       // per group of ki target blocks
    unsigned *ctl;            // [SYM_CTL]
    double *jrow;             // per group: [3][npad - start] sums over its targets
    double *ipart;            // per (item, block of its group): [3][WI] sums
    int nitems;
    int ki;                   // target blocks per group
};

__device__ __forceinline__ f2_t f2_shfl(f2_t v, int from)
{
    return __shfl_sync(0xffffffffu, v, from);
}

// Fold the FP32 sums of the two targets `at`, `at + 1` into their accumulators.
// acc: [3][WI] doubles, or with KAHAN [hi x, y, z, lo x, y, z][WI] floats (WI:
// the targets of the warp's block).
template <int WI, bool KAHAN>
__device__ __forceinline__ void sym_fold(double *acc, int at, const f2_t (&f)[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (KAHAN) {
            f2_t *h = reinterpret_cast<f2_t *>(reinterpret_cast<float *>(acc) + c * WI + at);
            f2_t *l = reinterpret_cast<f2_t *>(reinterpret_cast<float *>(acc) + (3 + c) * WI + at);
            // Knuth's TwoSum on both lanes: lo collects the exact rounding errors of hi
            const f2_t a = *h, s = f2_add(a, f[c]), bb = f2_sub(s, a);
            const f2_t e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(f[c], bb));
            *h = s;
            *l = f2_add(*l, e);
        } else {
            double2 *d = reinterpret_cast<double2 *>(acc + c * WI + at);
            float x0, x1;
            f2_unpack(f[c], x0, x1);
            double2 v = *d;
            v.x += (double)x0;
            v.y += (double)x1;
            *d = v;
        }
    }
}

// Where the interleaved staging keeps particle i (x at +0, y at +2, z at +4, w at +6).
__device__ __forceinline__ const float *staged_at(const float *src, int i)
{
    return src + 8 * (size_t)(i >> 1) + (i & 1);
}

// The targets i, i + 1 (i even) as f32x2 pairs; targets past n sit far from
// every source and from the padding, with weight 0.
__device__ __forceinline__ void load_targets(const float *src, int i, int n, f2_t &x, f2_t &y,
                                             f2_t &z, f2_t &w)
{
    float4 a = make_float4(-1e18f, -1e18f, -1e18f, -1e18f);
    float4 b = make_float4(-1e18f, -1e18f, 0.f, 0.f);
    if (i + 1 < n) {
        const float4 *q = reinterpret_cast<const float4 *>(src + 4 * (size_t)i);
        a = q[0];
        b = q[1];
    } else if (i < n) {
        const float *q = src + 4 * (size_t)i;
        a.x = q[0];
        a.z = q[2];
        b.x = q[4];
        b.z = q[6];
    }
    x = f2_pack(a.x, a.y);
    y = f2_pack(a.z, a.w);
    z = f2_pack(b.x, b.y);
    w = f2_pack(b.z, b.w);
}

// The lo parts of the targets i, i + 1 (0 past n).
__device__ __forceinline__ void load_lows(const float *lo, int i, int n, f2_t &x, f2_t &y, f2_t &z)
{
    x = y = z = 0ull;
    if (i + 1 < n) {
        const float4 *q = reinterpret_cast<const float4 *>(lo + 4 * (size_t)i);
        const float4 a = q[0], b = q[1];
        x = f2_pack(a.x, a.y);
        y = f2_pack(a.z, a.w);
        z = f2_pack(b.x, b.y);
    } else if (i < n) {
        const float *q = lo + 4 * (size_t)i;
        x = f2_pack(q[0], 0.f);
        y = f2_pack(q[2], 0.f);
        z = f2_pack(q[4], 0.f);
    }
}

// v with the lanes that are not `on` set to 0.
__device__ __forceinline__ f2_t f2_keep(f2_t v, bool on0, bool on1)
{
    float a, b;
    f2_unpack(v, a, b);
    return f2_pack(on0 ? a : 0.f, on1 ? b : 0.f);
}

// The slow form of one (warp, tile): pairs with s == 0 or s not a number add
// nothing (their separation is dropped with the factor: 0 * NaN would stay in both
// sums, and one particle lost in a close encounter would take the bunch with it),
// separations on hi/lo parts with SPLIT, two packs at a time so that it needs few
// registers.  Arguments as sym_tile; fold = false leaves the targets' sums alone.
template <int PK, int TJ, int WI, bool SPLIT, bool WEIGHTED, bool KAHAN, bool OWN>
__device__ __noinline__ void sym_slow(const float *__restrict__ src, size_t lo_at, int n, int i0,
                                      int j0, int count, float eps2, double *acc, int at0, float *stash, bool add,
                                      bool fold)
{
    constexpr int G = PK % 2 ? 1 : 2;
    const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
    const f2_t EPS2 = f2_pack(eps2, eps2);
    for (int p = 0; p < PK; p += G) {
        f2_t X[G], Y[G], Z[G], W[G], XL[G], YL[G], ZL[G], A[G][3];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int i = i0 + (p + g) * 64 + 2 * lane;
            load_targets(src, i, n, X[g], Y[g], Z[g], W[g]);
            XL[g] = YL[g] = ZL[g] = 0ull;
            if (SPLIT) load_lows(src + lo_at, i, n, XL[g], YL[g], ZL[g]);
            A[g][0] = A[g][1] = A[g][2] = 0ull;
        }
        for (int s = 0; s < count; s += 32) {
            const float *q = staged_at(src, j0 + s + lane);
            float xj = q[0], yj = q[2], zj = q[4], wj = WEIGHTED ? q[6] : 1.f;
            float xl = 0.f, yl = 0.f, zl = 0.f;
            if (SPLIT) {
                xl = q[lo_at];
                yl = q[lo_at + 2];
                zl = q[lo_at + 4];
            }
            f2_t FX = 0ull, FY = 0ull, FZ = 0ull;
            for (int k = 0; k < 32; ++k) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    f2_t DX = f2_sub(X[g], f2_pack(xj, xj));
                    f2_t DY = f2_sub(Y[g], f2_pack(yj, yj));
                    f2_t DZ = f2_sub(Z[g], f2_pack(zj, zj));
                    if (SPLIT) {
                        DX = f2_add(DX, f2_sub(XL[g], f2_pack(xl, xl)));
                        DY = f2_add(DY, f2_sub(YL[g], f2_pack(yl, yl)));
                        DZ = f2_add(DZ, f2_sub(ZL[g], f2_pack(zl, zl)));
                    }
                    const f2_t S = f2_fma(DZ, DZ, f2_fma(DY, DY, f2_fma(DX, DX, EPS2)));
                    float s0, s1;
                    f2_unpack(S, s0, s1);
                    const bool on0 = s0 > 0.f, on1 = s1 > 0.f;
                    const f2_t INV = f2_pack(on0 ? rsqrt_sfu(s0) : 0.f, on1 ? rsqrt_sfu(s1) : 0.f);
                    DX = f2_keep(DX, on0, on1);
                    DY = f2_keep(DY, on0, on1);
                    DZ = f2_keep(DZ, on0, on1);
                    const f2_t INV3 = f2_mul(f2_mul(INV, INV), INV);
                    const f2_t TI = WEIGHTED ? f2_mul(INV3, f2_pack(wj, wj)) : INV3;
                    A[g][0] = f2_fma(TI, DX, A[g][0]);
                    A[g][1] = f2_fma(TI, DY, A[g][1]);
                    A[g][2] = f2_fma(TI, DZ, A[g][2]);
                    if (!OWN) {
                        const f2_t TJW = WEIGHTED ? f2_mul(INV3, W[g]) : INV3;
                        FX = f2_fma(TJW, DX, FX);
                        FY = f2_fma(TJW, DY, FY);
                        FZ = f2_fma(TJW, DZ, FZ);
                    }
                }
                xj = __shfl_sync(0xffffffffu, xj, next);
                yj = __shfl_sync(0xffffffffu, yj, next);
                zj = __shfl_sync(0xffffffffu, zj, next);
                if (WEIGHTED) wj = __shfl_sync(0xffffffffu, wj, next);
                if (SPLIT) {
                    xl = __shfl_sync(0xffffffffu, xl, next);
                    yl = __shfl_sync(0xffffffffu, yl, next);
                    zl = __shfl_sync(0xffffffffu, zl, next);
                }
                if (!OWN) {
                    FX = f2_shfl(FX, next);
                    FY = f2_shfl(FY, next);
                    FZ = f2_shfl(FZ, next);
                }
            }
            if (!OWN) {
                const f2_t F[3] = {FX, FY, FZ};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float a, b;
                    f2_unpack(F[c], a, b);
                    float *t = stash + c * TJ + s + lane;
                    *t = p == 0 && !add ? a + b : *t + (a + b);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (fold) sym_fold<WI, KAHAN>(acc, at0 + (p + g) * 64 + 2 * lane, A[g]);
    }
    __syncwarp();   // sym_tile with ADD reads the stash in other lanes
}

// Add the partial sums of 32 particles and run their push.  The order of the
// additions is fixed by the plan: the rows of the groups up to the particles'
// own, then the items of that group, eight at a time, the chunks of eight dealt
// to the four warps, whose sums are added in warp order.
template <int WI, int KIND>
__device__ __forceinline__ void sym_finish(const ForceArgs &p, const SymArgs &q, int j0,
                                           double *scratch)
{
    constexpr int U = 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int bis = WI * q.ki;
    const int ib = j0 / WI, grp = ib / q.ki;
    const SymRow row = q.rows[grp];
    const int j = j0 + lane, terms = grp + 1 + row.items;
    const double *own =
        q.ipart + ((size_t)row.first * q.ki + (ib - grp * q.ki)) * 3 * WI + (j - ib * WI);
    double sum[3] = {0.0, 0.0, 0.0};
    for (int k0 = warp * U; k0 < terms; k0 += kSymWarps * U) {
        double v[3][U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = k0 + u;
            const double *b = k <= grp
                                  ? q.jrow + sym_row_offset(k, p.npad, bis) + (j - k * bis)
                                  : own + (size_t)(k - grp - 1) * q.ki * 3 * WI;
            const size_t plane = k <= grp ? (size_t)p.npad - (size_t)k * bis : WI;
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c][u] = k < terms ? ld_cg(b + c * plane) : 0.0;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
            sum[c] += ((v[c][0] + v[c][1]) + (v[c][2] + v[c][3])) +
                      ((v[c][4] + v[c][5]) + (v[c][6] + v[c][7]));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) scratch[(warp * 3 + c) * 32 + lane] = sum[c];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sum[c] = scratch[c * 32 + lane];
            for (int w = 1; w < kSymWarps; ++w) sum[c] += scratch[(w * 3 + c) * 32 + lane];
        }
        finish_particle<KIND>(p, j, sum[0], sum[1], sum[2]);
    }
}

// The end of a pass, for every warp after its last item (`done`: items it ran):
// count them, wait until all items of the pass are done, share out the
// particles.  scratch: 768 doubles of shared memory.
template <int WI, int KIND>
__device__ __forceinline__ void sym_collect(const ForceArgs &p, const SymArgs &q, int done,
                                            double *scratch, int *s_next)
{
    const int tid = threadIdx.x, lane = tid & 31;
    __threadfence();   // the sums before the count
    __syncwarp();
    if (lane == 0) atomicAdd(&q.ctl[SYM_DONE], (unsigned)done);

    // Every item has been handed out, each to a warp that runs now: wait until all are
    // done, then share out the particles.  The wait covers the other warps' last items
    // (up to 50 ms at the largest N), so it is bounded by at least a second.  Test hook
    // (PP_OPT_TEST_SKIP_COPY): wait for one item more than there are, by the limit as set.
    __syncthreads();
    if (tid == 0) {
        int ok = 1;
        const uint64_t t0 = globaltimer_ns();
        const uint64_t limit =
            p.skip_copy || p.timeout_ns > kSymMinWaitNs ? p.timeout_ns : kSymMinWaitNs;
        const unsigned want = (unsigned)q.nitems + (p.skip_copy ? 1u : 0u);
        while (ld_acquire(&q.ctl[SYM_DONE]) < want)
            if (globaltimer_ns() - t0 > limit) {
                ok = 0;
                break;
            }
        if (!ok) atomicOr(p.err, 1);
        s_next[0] = ok ? (int)atomicAdd(&q.ctl[SYM_FINISH], 1u) : (1 << 26) - 1;
    }
    __syncthreads();
    __threadfence();
    int unit = s_next[0];
    for (int turn = 1; unit * 32 < p.n; turn ^= 1) {
        if (tid == 0) s_next[turn] = (int)atomicAdd(&q.ctl[SYM_FINISH], 1u);
        sym_finish<WI, KIND>(p, q, unit * 32, scratch + turn * 384);
        unit = s_next[turn];
    }
    if (tid == 0 && atomicAdd(&q.ctl[SYM_LEFT], 1u) == gridDim.x - 1)
        for (int k = 0; k < SYM_CTL; ++k) q.ctl[k] = 0u;
}

// One (warp, tile): the fast pair loop over the 64 PK targets from i0 and the
// `count` <= TJ sources from j0 (a multiple of 32), then the fold into acc (from
// place at0 of WI).  Without OWN the sources' sums go to `stash` ([3][TJ] of this
// warp; ADD: onto what is there), every four steps, so that an FP32 partial holds
// 8 PK terms.  OWN: the sources are among the targets; each target takes its sum
// only (the pair comes again with the roles exchanged) and skips itself by index.
// Returns false (for the whole warp, nothing folded, stash void) for a tile with a
// zero-distance pair (non-finite sum) or, with POS_GUARDED, with a pair too close for
// the hi parts alone.  BOX: the caller has ruled close pairs out.  HALF (TJ = 128): the sums of the
// first 64 sources wait in local memory and are added to those of the second 64 before the
// fold, so that no FP32 partial is longer than 64 terms at half the FP64 folds of tiles of 64
// (N = 32768: 0.320 against 0.341 ms per step).  Not inlined: the loop needs every
// register for itself (inlined into the queue loop it ran 10 % slower).
template <int PK, int TJ, int WI, int POS, bool BOX, bool WEIGHTED, bool KAHAN, bool OWN, bool ADD,
          bool HALF = false>
__device__ __noinline__ bool sym_tile(const float *__restrict__ src, size_t lo_at, int n, int i0,
                                      int j0, int count, float eps2, double *acc, int at0, float *stash)
{
    constexpr bool SPLIT = POS == POS_SPLIT, GUARD = POS == POS_GUARDED && !BOX;
    const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
    const f2_t EPS2 = f2_pack(eps2, eps2);
    f2_t X[PK], Y[PK], Z[PK], W[PK], XL[PK], YL[PK], ZL[PK], A[PK][3];
    float ms[PK];
    volatile f2_t first[HALF ? 3 * PK : 1];   // volatile: not in registers
#pragma unroll
    for (int k = 0; k < PK; ++k) {
        const int i = i0 + k * 64 + 2 * lane;
        load_targets(src, i, n, X[k], Y[k], Z[k], W[k]);
        XL[k] = YL[k] = ZL[k] = 0ull;
        if (SPLIT) load_lows(src + lo_at, i, n, XL[k], YL[k], ZL[k]);
        A[k][0] = A[k][1] = A[k][2] = 0ull;
        ms[k] = 0.f;
    }
    const float *g = staged_at(src, j0 + lane);
    float nx = g[0], ny = g[2], nz = g[4], nw = WEIGHTED ? g[6] : 0.f;
    float nxl = 0.f, nyl = 0.f, nzl = 0.f;
    if (SPLIT) {
        nxl = g[lo_at];
        nyl = g[lo_at + 2];
        nzl = g[lo_at + 4];
    }
#pragma unroll 1
    for (int s = 0; s < count; s += 32) {
        float xj = nx, yj = ny, zj = nz, wj = nw, xl = nxl, yl = nyl, zl = nzl;
        g += 128;   // the next 32 sources
        if (s + 32 < count) {
            nx = g[0];
            ny = g[2];
            nz = g[4];
            if (WEIGHTED) nw = g[6];
            if (SPLIT) {
                nxl = g[lo_at];
                nyl = g[lo_at + 2];
                nzl = g[lo_at + 4];
            }
        }
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 4) {
            f2_t FX = 0ull, FY = 0ull, FZ = 0ull;
#pragma unroll
            for (int r = r0; r < r0 + 4; ++r) {
                // OWN: this source's place among the lane's targets of pack 0 (0 or 1: itself)
                const int self = OWN ? j0 + s + ((lane + r) & 31) - (i0 + 2 * lane) : 0;
                const f2_t XJ = f2_pack(xj, xj), YJ = f2_pack(yj, yj), ZJ = f2_pack(zj, zj);
                f2_t XJL = 0ull, YJL = 0ull, ZJL = 0ull, WJ = 0ull;
                if (SPLIT) {
                    XJL = f2_pack(xl, xl);
                    YJL = f2_pack(yl, yl);
                    ZJL = f2_pack(zl, zl);
                }
                if (WEIGHTED) WJ = f2_pack(wj, wj);
                xj = __shfl_sync(0xffffffffu, xj, next);
                yj = __shfl_sync(0xffffffffu, yj, next);
                zj = __shfl_sync(0xffffffffu, zj, next);
                if (WEIGHTED) wj = __shfl_sync(0xffffffffu, wj, next);
                if (SPLIT) {
                    xl = __shfl_sync(0xffffffffu, xl, next);
                    yl = __shfl_sync(0xffffffffu, yl, next);
                    zl = __shfl_sync(0xffffffffu, zl, next);
                }
#pragma unroll
                for (int k = 0; k < PK; ++k) {
                    f2_t DX = f2_sub(X[k], XJ);
                    f2_t DY = f2_sub(Y[k], YJ);
                    f2_t DZ = f2_sub(Z[k], ZJ);
                    if (SPLIT) {
                        DX = f2_add(DX, f2_sub(XL[k], XJL));
                        DY = f2_add(DY, f2_sub(YL[k], YJL));
                        DZ = f2_add(DZ, f2_sub(ZL[k], ZJL));
                    }
                    const f2_t S = f2_fma(DZ, DZ, f2_fma(DY, DY, f2_fma(DX, DX, EPS2)));
                    float s0, s1;
                    f2_unpack(S, s0, s1);
                    float q0 = rsqrt_sfu(s0), q1 = rsqrt_sfu(s1);
                    if (OWN) {
                        q0 = self == 64 * k ? 0.f : q0;
                        q1 = self == 64 * k + 1 ? 0.f : q1;
                    }
                    if (GUARD) ms[k] = fmax3(ms[k], q0, q1);
                    const f2_t INV = f2_pack(q0, q1);
                    const f2_t INV3 = f2_mul(f2_mul(INV, INV), INV);
                    const f2_t TI = WEIGHTED ? f2_mul(INV3, WJ) : INV3;
                    A[k][0] = f2_fma(TI, DX, A[k][0]);
                    A[k][1] = f2_fma(TI, DY, A[k][1]);
                    A[k][2] = f2_fma(TI, DZ, A[k][2]);
                    if (!OWN) {
                        const f2_t TS = WEIGHTED ? f2_mul(INV3, W[k]) : INV3;
                        FX = f2_fma(TS, DX, FX);
                        FY = f2_fma(TS, DY, FY);
                        FZ = f2_fma(TS, DZ, FZ);
                    }
                }
                if (!OWN && r < r0 + 3) {
                    FX = f2_shfl(FX, next);
                    FY = f2_shfl(FY, next);
                    FZ = f2_shfl(FZ, next);
                }
            }
            if (!OWN) {   // four steps' sums to the source they belong to
                const f2_t F[3] = {FX, FY, FZ};
                float *home = stash + s + ((lane + r0 + 3) & 31);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    float a, b;
                    f2_unpack(F[c], a, b);
                    home[c * TJ] = ADD || r0 > 0 ? home[c * TJ] + (a + b) : a + b;
                }
                __syncwarp();
            }
        }
        if (HALF && s == 32) {   // 64 sources done (count: 64 or 128)
#pragma unroll
            for (int k = 0; k < PK; ++k)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    first[3 * k + c] = A[k][c];
                    A[k][c] = 0ull;
                }
        }
    }
    if (HALF) {
#pragma unroll
        for (int k = 0; k < PK; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) A[k][c] = f2_add(first[3 * k + c], A[k][c]);
    }
    f2_t all = 0ull;
    bool again = false;
#pragma unroll
    for (int k = 0; k < PK; ++k) {
        all = f2_add(all, f2_add(f2_add(A[k][0], A[k][1]), A[k][2]));
        if (GUARD) {
            const f2_t P2 = f2_fma(Z[k], Z[k], f2_fma(Y[k], Y[k], f2_mul(X[k], X[k])));
            float a, b;
            f2_unpack(P2, a, b);
            again |= ms[k] > 254.f * rsqrt_sfu(fmaxf(a, b));
        }
    }
    float a, b;
    f2_unpack(all, a, b);
    again |= !isfinite(a + b);
    if (__any_sync(0xffffffffu, again)) return false;
#pragma unroll
    for (int k = 0; k < PK; ++k) sym_fold<WI, KAHAN>(acc, at0 + k * 64 + 2 * lane, A[k]);
    return true;
}

// A tile on hi/lo separations, four packs at a time (the lo parts take as many
// registers as the hi parts).
template <int PK, int TJ, int WI, bool WEIGHTED, bool KAHAN, bool OWN>
__device__ __forceinline__ void sym_split(const float *src, size_t lo_at, int n, int i0, int j0,
                                          int count, float eps2, double *acc, float *stash)
{
    constexpr int PH = PK > 4 ? 4 : PK;
    static_assert(PK == PH || PK == 2 * PH, "one or two parts");
    if (!sym_tile<PH, TJ, WI, POS_SPLIT, false, WEIGHTED, KAHAN, OWN, false>(
            src, lo_at, n, i0, j0, count, eps2, acc, 0, stash))
        sym_slow<PH, TJ, WI, true, WEIGHTED, KAHAN, OWN>(src, lo_at, n, i0, j0, count, eps2, acc, 0, stash,
                                                        false, true);
    if (PK > PH && !sym_tile<PH, TJ, WI, POS_SPLIT, false, WEIGHTED, KAHAN, OWN, true>(
                       src, lo_at, n, i0 + 64 * PH, j0, count, eps2, acc, 64 * PH, stash)) {
        // the first part's share of the source sums again, then this part
        if (!OWN)
            sym_slow<PH, TJ, WI, true, WEIGHTED, KAHAN, OWN>(src, lo_at, n, i0, j0, count, eps2, acc, 0,
                                                            stash, false, false);
        sym_slow<PH, TJ, WI, true, WEIGHTED, KAHAN, OWN>(src, lo_at, n, i0 + 64 * PH, j0, count, eps2, acc,
                                                        64 * PH, stash, true, true);
    }
}

// One (warp, tile) by whichever of the forms above it needs.  close: BOX found
// that it may hold close pairs.
template <int PK, int TJ, int POS, bool BOX, bool WEIGHTED, bool KAHAN, bool OWN, bool HALF>
__device__ __forceinline__ void sym_any(const float *src, size_t lo_at, int n, int i0, int j0,
                                        int count, float eps2, double *acc, float *stash, bool close)
{
    constexpr int WI = 64 * PK, LEN = HALF ? TJ / 2 : TJ;   // LEN: terms per FP32 partial
    static_assert(!HALF || (POS == POS_SINGLE && LEN == 64), "two halves of 64 sources");
    if (!(BOX && close) &&
        sym_tile<PK, TJ, WI, POS, BOX, WEIGHTED, KAHAN, OWN, false, HALF>(
            src, lo_at, n, i0, j0, count, eps2, acc, 0, stash))
        return;
    if (POS == POS_GUARDED)
        sym_split<PK, TJ, WI, WEIGHTED, KAHAN, OWN>(src, lo_at, n, i0, j0, count, eps2, acc, stash);
    else
        for (int s = 0; s < count; s += LEN)
            sym_slow<PK, TJ, WI, POS == POS_SPLIT, WEIGHTED, KAHAN, OWN>(
                src, lo_at, n, i0, j0 + s, min(LEN, count - s), eps2, acc, 0, stash + s, false, true);
}

// Shared memory of each warp: its targets' accumulators and its tile's source sums.
template <int PK, int TJ>
__host__ __device__ constexpr size_t sym_warp_smem()
{
    return (size_t)3 * 64 * PK * sizeof(double) + (size_t)3 * TJ * sizeof(float);
}

// Can a target of the box [lo, hi] and a source of tile t's box have a pair
// closer than |p| / 256, p the one further out?  rmax2: the largest |p|^2 the
// first box allows.  (Spatially sorted sources.)
__device__ __forceinline__ bool sym_box_close(const float4 *boxes, int t, float4 lo, float4 hi,
                                              float rmax2, float eps2)
{
    const float4 a = boxes[2 * t], b = boxes[2 * t + 1];
    const float dx = fmax3(a.x - hi.x, lo.x - b.x, 0.f);
    const float dy = fmax3(a.y - hi.y, lo.y - b.y, 0.f);
    const float dz = fmax3(a.z - hi.z, lo.z - b.z, 0.f);
    const float s = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, eps2)));
    const float mx = fmaxf(fabsf(a.x), fabsf(b.x)), my = fmaxf(fabsf(a.y), fabsf(b.y)),
                mz = fmaxf(fabsf(a.z), fabsf(b.z));
    return s * 65536.f <= fmaxf(fmaf(mz, mz, fmaf(my, my, mx * mx)), rmax2);
}

// POS: POS_SINGLE, POS_SPLIT (hi/lo separations throughout) or POS_GUARDED.
// Guarded without BOX: hi parts, with the largest rsqrt(s) of each tile kept
// per pack; a tile with a pair closer than |p_i| / 254 is summed again on hi/lo
// parts.  (A pair closer than |p_j| / 256 to the source also passes that test,
// since then |p_i| >= |p_j| (1 - 1/256): one test serves both directions.)
// BOX, on spatially sorted sources: a tile whose box comes that close to the
// box of one of the block's own tiles, and the targets' own tiles, are summed on hi/lo parts,
// every other tile on hi parts with no test per pair.
template <int PK, int TJ, int POS, bool BOX, bool WEIGHTED, bool KAHAN, int MINB, bool HALF>
__global__ void __launch_bounds__(kSymThreads, MINB)
    force_sym_kernel(const ForceArgs p, const SymArgs q)
{
    constexpr int WI = 64 * PK, BT = WI / TJ;
    static_assert(WI % TJ == 0 && TJ % 32 == 0, "tiles divide a block of targets");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_next[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *acc = reinterpret_cast<double *>(smem_raw + warp * sym_warp_smem<PK, TJ>());
    float *stash = reinterpret_cast<float *>(acc + 3 * WI);
    const float *src = static_cast<const float *>(p.src);
    const size_t lo_at = 4 * (size_t)p.npad;
    const int bis = WI * q.ki;

    // one item ahead: its number comes back while this one runs
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
            const int i0 = (it.ib0 + kb) * WI;
            for (int k = 2 * lane; k < 3 * WI; k += 64)   // KAHAN: six floats in the same bytes
                *reinterpret_cast<double2 *>(acc + k) = make_double2(0.0, 0.0);
            __syncwarp();
            // BOX: lane k < BT tests the box of the block's k-th tile of targets (an empty
            // box is close to nothing)
            float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
            float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
            float rmax2 = 0.f;
            if (BOX && lane < BT && i0 + lane * TJ < p.npad) {
                lo = p.boxes[2 * (i0 / TJ + lane)];
                hi = p.boxes[2 * (i0 / TJ + lane) + 1];
                const float mx = fmaxf(fabsf(lo.x), fabsf(hi.x)),
                            my = fmaxf(fabsf(lo.y), fabsf(hi.y)),
                            mz = fmaxf(fabsf(lo.z), fabsf(hi.z));
                rmax2 = fmaf(mz, mz, fmaf(my, my, mx * mx));
            }
            for (int j = max(it.j0, i0), len; j < it.j1; j += len) {
                const bool mine = j < i0 + WI;   // the sources are among the targets
                len = min(TJ - j % TJ, it.j1 - j);
                if (mine)
                    sym_any<PK, TJ, POS, BOX, WEIGHTED, KAHAN, true, HALF>(
                        src, lo_at, p.n, i0, j, len, p.eps2f, acc, stash, true);
                else
                    sym_any<PK, TJ, POS, BOX, WEIGHTED, KAHAN, false, HALF>(
                        src, lo_at, p.n, i0, j, len, p.eps2f, acc, stash,
                        BOX && __any_sync(0xffffffffu, sym_box_close(p.boxes, j / TJ, lo, hi, rmax2,
                                                                     p.eps2f)));
                if (mine && kb > 0) continue;   // the group's row has been started
                // the sources' sums (the pair term acts on them with the opposite sign)
                double *out = jrow + (j + lane - grp * bis);
#pragma unroll 1
                for (int s = 0; s < len; s += 64) {
                    double v[2][3];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            v[h][c] = kb > 0 ? ld_cg(out + c * plane + s + 32 * h) : 0.0;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float f = stash[c * TJ + s + 32 * h + lane];
                            if (!mine) v[h][c] -= (double)f;
                            __stcg(out + c * plane + s + 32 * h, v[h][c]);
                        }
                }
                __syncwarp();   // the next tile's sums enter the stash in other lanes
            }
            // this item's sums of the block's targets, each written by its owner
            double *part = q.ipart + ((size_t)item * q.ki + kb) * 3 * WI;
            for (int k = 0; k < PK; ++k) {
                const int at = k * 64 + 2 * lane;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    double2 v;
                    if (KAHAN) {
                        const float *f = reinterpret_cast<const float *>(acc);
                        v.x = (double)f[c * WI + at] + (double)f[(3 + c) * WI + at];
                        v.y = (double)f[c * WI + at + 1] + (double)f[(3 + c) * WI + at + 1];
                    } else {
                        v = *reinterpret_cast<const double2 *>(acc + c * WI + at);
                    }
                    __stcg(reinterpret_cast<double2 *>(part + c * WI + at), v);
                }
            }
            __syncwarp();
        }
    }
    sym_collect<WI, POS == POS_SINGLE ? STAGE_F32I : STAGE_F32IX2>(
        p, q, done, reinterpret_cast<double *>(smem_raw), s_next);
}

}  // namespace ppk

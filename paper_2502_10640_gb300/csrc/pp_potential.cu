// pp_potential.cu -- the potential energy's double sum over unordered pairs,
// for diagnostics.
//
// Only the total is wanted, so a pair is evaluated once and added to one of its
// particles.  Blocks of 64 or 256 particles are paired on a ring: block I meets blocks
// I, I + 1, ..., I + floor(nb / 2) (mod nb), every unordered pair of blocks once
// and the same number for each block; pairs inside a block come twice and count
// half.  One warp per (block, range of ring distances): one or four packs of
// two targets per lane in registers, the sources of a block broadcast from its
// shared memory.  Per pair: 7 f32x2 half-instructions and one SFU rsqrt, which
// bounds the loop (one operation per pair at 16 per clock and SM).  FP32 sums of
// 64, 128 (from N = 16384) or 256 terms (from 32768, where 128 cost 2 %) fold into
// FP64.  N = 100003: 1.19 ms, 84 % of that bound (the one-sided scalar loop with its
// index and zero tests took 4.0); N = 24001: 94 us; N = 2048: 25 us against 73.
#include "pp_internal.h"

namespace ppk {

namespace {

constexpr int kWarps = 4;

// FP32 sums of w_j / sqrt(s) of each target over the LEN sources from `first` on of
// `tile`.  MASKED: zero-distance pairs are left out, and with `self` >= 0 the pair of a
// target with itself (self: the lane).
template <int PK, int LEN, bool MASKED>
__device__ __forceinline__ void block_terms(const float4 *tile, int first, const f2_t (&X)[PK],
                                            const f2_t (&Y)[PK], const f2_t (&Z)[PK], f2_t EPS2,
                                            int self, f2_t (&F)[PK])
{
#pragma unroll
    for (int k = 0; k < PK; ++k) F[k] = 0ull;
#pragma unroll 4
    for (int j = first; j < first + LEN; ++j) {
        const float4 s = tile[j];   // padding sources carry s.w = 0
        const f2_t XJ = f2_pack(s.x, s.x), YJ = f2_pack(s.y, s.y), ZJ = f2_pack(s.z, s.z);
        const f2_t WJ = f2_pack(s.w, s.w);
#pragma unroll
        for (int k = 0; k < PK; ++k) {
            const f2_t DX = f2_sub(X[k], XJ), DY = f2_sub(Y[k], YJ), DZ = f2_sub(Z[k], ZJ);
            const f2_t S = f2_fma(DZ, DZ, f2_fma(DY, DY, f2_fma(DX, DX, EPS2)));
            float s0, s1;
            f2_unpack(S, s0, s1);
            float q0 = rsqrt_sfu(s0), q1 = rsqrt_sfu(s1);
            if (MASKED) {
                const int own = self < 0 ? -1 : k * 64 + self;
                q0 = s0 > 0.f && j != own ? q0 : 0.f;
                q1 = s1 > 0.f && (own < 0 || j != own + 32) ? q1 : 0.f;
            }
            F[k] = f2_fma(f2_pack(q0, q1), WJ, F[k]);
        }
    }
}

// LEN: terms per FP32 sum.
template <int PK, int LEN>
__global__ void __launch_bounds__(32 * kWarps, 4)
    potential_kernel(const float4 *__restrict__ src, int n, int nb, int nd, int chunk, float eps2,
                     const double *__restrict__ wts, double *partials, int count)
{
    constexpr int B = 64 * PK;   // particles per block
    static_assert(B % LEN == 0, "whole sums per block");
    __shared__ float4 sm[kWarps][B];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int id = blockIdx.x * kWarps + warp;   // this warp's (block, range) and result slot
    if (id >= count) return;
    const int ib = id % nb, d0 = (id / nb) * chunk, d1 = min(d0 + chunk, nd);
    float4 *tile = sm[warp];
    f2_t X[PK], Y[PK], Z[PK], F[PK];
    double acc[2 * PK];
#pragma unroll
    for (int k = 0; k < PK; ++k) {
        const int i = ib * B + k * 64 + lane;
        // targets past n sit far from every source and from the padding
        const float4 far = make_float4(-1e18f, -1e18f, -1e18f, 0.f);
        const float4 a = i < n ? src[i] : far, b = i + 32 < n ? src[i + 32] : far;
        X[k] = f2_pack(a.x, b.x);
        Y[k] = f2_pack(a.y, b.y);
        Z[k] = f2_pack(a.z, b.z);
        acc[2 * k] = acc[2 * k + 1] = 0.0;
    }
    const f2_t EPS2 = f2_pack(eps2, eps2);
    for (int d = d0; d < d1; ++d) {
        if (2 * d == nb && ib >= nb / 2) break;   // the antipodal block: from one side only
        const int jb = ib + d < nb ? ib + d : ib + d - nb;
        __syncwarp();
        for (int e = lane; e < B; e += 32) tile[e] = src[jb * B + e];
        __syncwarp();
        const double share = d == 0 ? 0.5 : 1.0;
#pragma unroll 1
        for (int first = 0; first < B; first += LEN) {
            bool again = d == 0;
            if (!again) {
                block_terms<PK, LEN, false>(tile, first, X, Y, Z, EPS2, -1, F);
                f2_t all = F[0];
#pragma unroll
                for (int k = 1; k < PK; ++k) all = f2_add(all, F[k]);
                float a, b;
                f2_unpack(all, a, b);
                again = __any_sync(0xffffffffu, !isfinite(a + b));   // a zero-distance pair
            }
            if (again)
                block_terms<PK, LEN, true>(tile, first, X, Y, Z, EPS2, d == 0 ? lane : -1, F);
#pragma unroll
            for (int k = 0; k < PK; ++k) {
                float a, b;
                f2_unpack(F[k], a, b);
                acc[2 * k] += share * (double)a;
                acc[2 * k + 1] += share * (double)b;
            }
        }
    }
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < 2 * PK; ++k) {
        const int i = ib * B + (k >> 1) * 64 + (k & 1) * 32 + lane;
        if (i < n) sum += wts ? wts[i] * acc[k] : acc[k];
    }
    for (int h = 16; h > 0; h >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, h);
    if (lane == 0) partials[id] = sum;
}

// The partial sums in a fixed order.
__global__ void __launch_bounds__(1024) potential_sum_kernel(const double *partials, int count,
                                                             double *out)
{
    __shared__ double sh[32];
    double sum = 0.0;
    for (int k = threadIdx.x; k < count; k += 1024) sum += partials[k];
    for (int h = 16; h > 0; h >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, h);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < 32) {
        sum = sh[threadIdx.x];
        for (int h = 16; h > 0; h >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, h);
        if (threadIdx.x == 0) *out = sum;
    }
}

template <int PK, int LEN>
int run_potential(const void *src, int n, float eps2, const double *wts, double *partials,
                  cudaStream_t s)
{
    const int nb = (n + 64 * PK - 1) / (64 * PK), nd = nb / 2 + 1;
    // ranges of ring distances: about 20000 warps (several rounds of a full GPU), and no
    // more results than partials holds (nb * 16 PK <= npad / 4)
    int ranges = 20000 / nb;
    ranges = ranges < 1 ? 1 : ranges > 16 * PK ? 16 * PK : ranges;
    const int chunk = (nd + ranges - 1) / ranges;
    const int count = nb * ((nd + chunk - 1) / chunk);
    potential_kernel<PK, LEN><<<(count + kWarps - 1) / kWarps, 32 * kWarps, 0, s>>>(
        static_cast<const float4 *>(src), n, nb, nd, chunk, eps2, wts, partials, count);
    return count;
}

}  // namespace

// Blocks of 64 particles below 16384 (more, shorter warps), of 256 above.
cudaError_t launch_potential(const void *src, int n, int npad, float eps2, const double *wts,
                             double *partials, double *out, cudaStream_t s)
{
    if (n < 1 || npad < n || npad % 256 != 0) return cudaErrorInvalidValue;
    const int count = n < 16384   ? run_potential<1, 64>(src, n, eps2, wts, partials, s)
                      : n < 32768 ? run_potential<4, 128>(src, n, eps2, wts, partials, s)
                                  : run_potential<4, 256>(src, n, eps2, wts, partials, s);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    potential_sum_kernel<<<1, 1024, 0, s>>>(partials, count, out);
    return cudaGetLastError();
}

}  // namespace ppk

// pp_noalloc.cu -- pp_fields_noalloc: the field of Eq. B for callers that
// cannot allocate device memory.
//
// Sources are staged hi/lo (two floats per coordinate, about 48 significant
// bits), so close pairs keep their separations and the field meets the 1e-5
// relative-L2 tolerance also on inputs whose closest pairs sit 1e3 times closer
// than the bunch size (single FP32 staging loses ~3e-5 there).
//
// Some callers cannot call cudaMalloc at all: code that runs inside a
// memory pool or arena owned by a host framework that forbids foreign
// allocations, code that must never trigger the allocator's implicit device
// synchronisation in a latency-critical loop, or a plug-in that may only use
// the buffers it is handed.  This entry point serves them.  It takes device
// inputs and outputs from the caller and keeps every intermediate (staged hi/lo
// sources, j-split partial sums, tickets, moment partials, frame, error words)
// in one file-scope __device__ array of fixed size.
//
// The call is latency: the pair sum itself takes 2 us at N = 900.  So the
// staging frame (centroid, RMS radius, length unit) never comes to the host:
// each kernel finishes the reduction that the one before it left per block, the
// force kernel reads its two scale factors from the array, and the host waits
// once, at the end (before: ten launches and three waits, 190 us at N = 900).
//
// The array exists on every GPU that loads this library, for the lifetime of
// the process (kScratchBytes, 3.67 MB).  All calls on a device share it
// and it keeps the last call's contents; the entry point clears the parts that
// must start at zero (tickets, error word) on every call.  Calls whose work
// overlaps on the GPU (several host threads, or several streams) race on the
// array and must be serialised by the caller.
//
// The host-side name of a __device__ array is only a stand-in for it, not a
// device address, so the first call on each device looks the address up with
// cudaGetSymbolAddress (with that device current) and caches it together with
// the identity of the device's current context; make that first call before any
// stream capture.  If the context was destroyed and recreated since (for
// example after cudaDeviceReset), the next call sees another context identity
// and looks the address up again instead of writing through a stale one.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include <cuda.h>

#include "../../include/pp.h"
#include "pp_internal.h"

using namespace ppk;

namespace {

constexpr int kNoAllocMaxN = PP_FIELDS_NOALLOC_MAX_N;    // largest N accepted
constexpr int kNoAllocMaxSplit = 8;                      // j-chunks per i-block
constexpr int kTile = 128, kStages = 4;
// Targets per block: 64 (one per thread, many CTAs) up to kWideN, 256 above.
constexpr int kWideN = 4096;
constexpr int kMaxPad = (kNoAllocMaxN + kPad - 1) / kPad * kPad;
constexpr int kMaxNib = (kNoAllocMaxN + 255) / 256;
static_assert(kMaxNib >= (kWideN + 63) / 64, "tickets for either blocking");
constexpr int kNaThreads = 256;
constexpr int kMaxBlocks = (kNoAllocMaxN + kNaThreads - 1) / kNaThreads;   // of the O(N) kernels

// What the force kernel needs of the staging frame.
struct NaFrame {
    float eps2f;
    double escale;
};

// Byte offsets of the parts of the scratch array (each 256-byte aligned).
constexpr size_t align256(size_t x) { return (x + 255) / 256 * 256; }
constexpr size_t kOffStage = 0;                                    // hi, lo: float4[2 max_pad]
constexpr size_t kOffPartial = align256(kOffStage + 2 * sizeof(float4) * kMaxPad);
constexpr size_t kOffTickets =
    align256(kOffPartial + sizeof(double) * kNoAllocMaxSplit * 3 * (size_t)kMaxNib * 256);
constexpr size_t kOffSums = align256(kOffTickets + sizeof(unsigned) * kMaxNib);  // per block: x, y, z
constexpr size_t kOffSquares = align256(kOffSums + 3 * sizeof(double) * kMaxBlocks);
constexpr size_t kOffFrame = align256(kOffSquares + sizeof(double) * kMaxBlocks);
constexpr size_t kOffErr = align256(kOffFrame + sizeof(NaFrame));
constexpr size_t kScratchBytes = align256(kOffErr + 2 * sizeof(int));

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_lock;
unsigned char *g_scratch_addr[kMaxDevices] = {};
unsigned long long g_scratch_ctx[kMaxDevices] = {};   // context identity of each address

// Errors are reported through pp_last_error(), like every other call.
pp_status na_fail(pp_status s, const char *m)
{
    set_last_error(m);
    return s;
}

pp_status na_cuda(cudaError_t e, const char *where)
{
    char msg[256];
    std::snprintf(msg, sizeof(msg), "%s: %s", where, cudaGetErrorString(e));
    set_last_error(msg);
    return PP_ERR_CUDA;
}

#define NA_CUDA(call)                                      \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return na_cuda(e_, #call);  \
    } while (0)

// Identity of the calling thread's current CUDA context (unique for the life of
// the process; a context recreated after a device reset gets a new one), or 0
// where the driver does not report one.
unsigned long long current_context_id()
{
    using GetCurrent = CUresult (*)(CUcontext *);
    using GetId = CUresult (*)(CUcontext, unsigned long long *);
    static const std::pair<GetCurrent, GetId> fns = [] {
        void *a = nullptr, *b = nullptr;
        cudaDriverEntryPointQueryResult q1{}, q2{};
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault,
                                             &q1) != cudaSuccess || q1 != cudaDriverEntryPointSuccess)
            a = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &q2) !=
                cudaSuccess || q2 != cudaDriverEntryPointSuccess)
            b = nullptr;
        return std::make_pair(reinterpret_cast<GetCurrent>(a), reinterpret_cast<GetId>(b));
    }();
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!fns.first || !fns.second || fns.first(&ctx) != CUDA_SUCCESS || !ctx ||
        fns.second(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

// Device address of the scratch array on the current device: looked up once
// per device (with that device current), and again if the device's context
// has been recreated since.
pp_status scratch_address(int dev, unsigned char **out)
{
    if (dev < 0 || dev >= kMaxDevices) return na_fail(PP_ERR_ARG, "device ordinal out of range");
    const unsigned long long ctx = current_context_id();
    std::lock_guard<std::mutex> g(g_setup_lock);
    if (!g_scratch_addr[dev] || ctx == 0 || g_scratch_ctx[dev] != ctx) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return na_cuda(e, "cudaGetSymbolAddress(scratch)");
        g_scratch_addr[dev] = static_cast<unsigned char *>(p);
        g_scratch_ctx[dev] = ctx;
    }
    *out = g_scratch_addr[dev];
    return PP_OK;
}

// Sum over the block's threads of up to three values, in a fixed order; the
// result is returned on every thread.
__device__ double3 block_sum3(double x, double y, double z)
{
    __shared__ double sh[3][kNaThreads / 32];
    for (int h = 16; h > 0; h >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, h);
        y += __shfl_xor_sync(0xffffffffu, y, h);
        z += __shfl_xor_sync(0xffffffffu, z, h);
    }
    __syncthreads();   // sh may still be read from the call before
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = x;
        sh[1][threadIdx.x >> 5] = y;
        sh[2][threadIdx.x >> 5] = z;
    }
    __syncthreads();
    x = y = z = 0.0;
    for (int w = 0; w < kNaThreads / 32; ++w) {
        x += sh[0][w];
        y += sh[1][w];
        z += sh[2][w];
    }
    return make_double3(x, y, z);
}

// The centroid from the per-block sums (every block adds them itself).
__device__ double3 centroid(const double *sums, int blocks, int n)
{
    const int t = threadIdx.x;
    const bool on = t < blocks;
    const double3 s = block_sum3(on ? sums[3 * t] : 0.0, on ? sums[3 * t + 1] : 0.0,
                                 on ? sums[3 * t + 2] : 0.0);
    return make_double3(s.x / n, s.y / n, s.z / n);
}

// Sums of the positions per block, the check that they are finite (err[1]) and the
// clear of the tickets.
__global__ void __launch_bounds__(kNaThreads)
    na_sums_kernel(const double *__restrict__ pos, int n, double *sums, unsigned *tickets,
                   int ntickets, int *err)
{
    const int i = blockIdx.x * kNaThreads + threadIdx.x;
    if (i < ntickets) tickets[i] = 0u;
    double x = 0.0, y = 0.0, z = 0.0;
    if (i < n) {
        x = pos[3 * i];
        y = pos[3 * i + 1];
        z = pos[3 * i + 2];
        if (!(isfinite(x) && isfinite(y) && isfinite(z))) err[1] = 1;
    }
    const double3 s = block_sum3(x, y, z);
    if (threadIdx.x == 0) {
        sums[3 * blockIdx.x] = s.x;
        sums[3 * blockIdx.x + 1] = s.y;
        sums[3 * blockIdx.x + 2] = s.z;
    }
}

// Sums of the squared distances from the centroid per block.
__global__ void __launch_bounds__(kNaThreads)
    na_squares_kernel(const double *__restrict__ pos, int n, const double *sums, int blocks,
                      double *squares)
{
    const double3 c = centroid(sums, blocks, n);
    const int i = blockIdx.x * kNaThreads + threadIdx.x;
    double q = 0.0;
    if (i < n) {
        const double dx = pos[3 * i] - c.x, dy = pos[3 * i + 1] - c.y, dz = pos[3 * i + 2] - c.z;
        q = dx * dx + dy * dy + dz * dz;
    }
    const double3 s = block_sum3(q, 0.0, 0.0);
    if (threadIdx.x == 0) squares[blockIdx.x] = s.x;
}

// The frame (centre = centroid, L0 = the power of two nearest the RMS radius) and
// the staged hi/lo sources with their padding.
__global__ void __launch_bounds__(kNaThreads)
    na_stage_kernel(const double *__restrict__ pos, int n, int npad, const double *sums,
                    const double *squares, int blocks, double eps, double field_scale, void *stage,
                    NaFrame *frame)
{
    const double3 c = centroid(sums, blocks, n);
    const int t = threadIdx.x;
    const double q = block_sum3(t < blocks ? squares[t] : 0.0, 0.0, 0.0).x;
    const double rms = sqrt(q / n);
    double l0 = 1.0;
    if (isfinite(rms) && rms > 0.0) {
        const int e = (int)llround(log2(rms));
        l0 = ldexp(1.0, e < -200 ? -200 : (e > 200 ? 200 : e));
    }
    const int i = blockIdx.x * kNaThreads + t;
    if (i < n)
        store_staged<STAGE_F32IX2>(stage, npad, i, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], c.x,
                                   c.y, c.z, 1.0 / l0);
    else if (i < npad)
        store_padding<STAGE_F32IX2>(stage, npad, i);
    if (i == 0) {
        const double epsl = eps / l0;
        frame->eps2f = (float)(epsl * epsl);
        frame->escale = field_scale / (l0 * l0);
    }
}

// The packed hi/lo force kernel with the frame taken from device memory; leaves
// E_out alone if the input was not finite (bad).
template <int T, int R>
__global__ void __launch_bounds__(T, 512 / T)
    na_force_kernel(const ForceArgs a, const NaFrame *frame, const int *bad)
{
    if (*bad) return;
    ForceArgs p = a;
    p.eps2f = frame->eps2f;
    p.escale = frame->escale;
    force_f32x2_body<T, R, kTile, kStages, 512 / T, false, false, true>(p);
}

}  // namespace

extern "C" pp_status pp_fields_noalloc(int64_t N, double w, double softening, const double *pos,
                                       double *E_out, void *stream_handle)
{
    if (N < 1 || N > kNoAllocMaxN)
        return na_fail(PP_ERR_ARG, "pp_fields_noalloc: N must be in [1, PP_FIELDS_NOALLOC_MAX_N = 16384]");
    if (!pos || !E_out) return na_fail(PP_ERR_ARG, "pp_fields_noalloc: null pointer");
    if (!(std::isfinite(w) && w > 0)) return na_fail(PP_ERR_ARG, "w must be finite and > 0");
    if (!(std::isfinite(softening) && softening >= 0))
        return na_fail(PP_ERR_ARG, "softening must be finite and >= 0");
    cudaStream_t st = static_cast<cudaStream_t>(stream_handle);
    int dev = 0;
    NA_CUDA(cudaGetDevice(&dev));
    unsigned char *base = nullptr;
    if (pp_status s = scratch_address(dev, &base)) return s;

    const int n = (int)N;
    const int npad = (n + kPad - 1) / kPad * kPad;
    void *stage = base + kOffStage;
    double *sums = reinterpret_cast<double *>(base + kOffSums);
    double *squares = reinterpret_cast<double *>(base + kOffSquares);
    unsigned *tickets = reinterpret_cast<unsigned *>(base + kOffTickets);
    NaFrame *frame = reinterpret_cast<NaFrame *>(base + kOffFrame);
    int *err = reinterpret_cast<int *>(base + kOffErr);

    const bool wide = n > kWideN;
    const int bi = wide ? 256 : 64;
    const int nib = (n + bi - 1) / bi;
    const int blocks = (n + kNaThreads - 1) / kNaThreads;
    NA_CUDA(cudaMemsetAsync(err, 0, 2 * sizeof(int), st));
    na_sums_kernel<<<blocks, kNaThreads, 0, st>>>(pos, n, sums, tickets, nib, err);
    NA_CUDA(cudaGetLastError());
    na_squares_kernel<<<blocks, kNaThreads, 0, st>>>(pos, n, sums, blocks, squares);
    NA_CUDA(cudaGetLastError());
    na_stage_kernel<<<npad / kNaThreads, kNaThreads, 0, st>>>(
        pos, n, npad, sums, squares, blocks, softening, -kCoulomb * kE * w, stage, frame);
    NA_CUDA(cudaGetLastError());

    // a tile per CTA while the partial sums fit (64-target blocks), at most 8 chunks above
    const int tiles = npad / kTile;
    const int most = wide ? kNoAllocMaxSplit : kNoAllocMaxSplit * kMaxNib * 256 / (nib * bi);
    const int nsplit_req = tiles < most ? tiles : most;
    const int chunk_tiles = (tiles + nsplit_req - 1) / nsplit_req;
    ForceArgs a{};
    a.src = stage;
    a.n = n;
    a.npad = npad;
    a.nib = nib;
    a.jchunk = chunk_tiles * kTile;
    a.nsplit = (tiles + chunk_tiles - 1) / chunk_tiles;
    a.mode = MODE_FIELDS;
    a.partial = reinterpret_cast<double *>(base + kOffPartial);
    a.tickets = tickets;
    a.nipad = nib * bi;
    a.out = E_out;
    a.err = err;
    a.timeout_ns = 1000000000ull;
    const size_t smem = (size_t)kStages * kTile * sizeof(float4) * 2;
    if (wide)
        na_force_kernel<128, 2><<<nib * a.nsplit, 128, smem, st>>>(a, frame, err + 1);
    else
        na_force_kernel<64, 1><<<nib * a.nsplit, 64, smem, st>>>(a, frame, err + 1);
    NA_CUDA(cudaGetLastError());
    int flags[2] = {0, 0};
    NA_CUDA(cudaMemcpyAsync(flags, err, sizeof(flags), cudaMemcpyDeviceToHost, st));
    NA_CUDA(cudaStreamSynchronize(st));
    if (flags[1]) return na_fail(PP_ERR_ARG, "non-finite position");
    if (flags[0]) return na_fail(PP_ERR_TIMEOUT, "a device-side wait ran out of time");
    return PP_OK;
}

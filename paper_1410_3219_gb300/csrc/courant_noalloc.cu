// Courant time step over caller-owned device arrays, without allocating.
//
// Some callers cannot allocate GPU memory at the point where they need a
// time step: code running inside a memory pool or arena that owns the whole
// device, and code that must not synchronise the device (cudaMalloc/cudaFree
// can).  This entry point gives them the time step of the sweep without any
// allocation: its scratch (one partial minimum per thread block and completion
// counters) lives in a file-scope __device__ array that every
// process loading the library holds on every GPU it uses, until exit.
//
// Set-up: the first call on each device looks up the array's device address
// with cudaGetSymbolAddress (in host code the array's name is only a
// host-side stand-in); make that first call before any stream capture.
// Calls share the array: calls that overlap on the GPU (different streams,
// or different host threads) race and must not be issued.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <mutex>

#include <cuda_runtime.h>

#include "../../include/rich.h"
#include "api_internal.h"
#include "chain.cuh"

namespace {

constexpr int kBlock = 256;
// cells a thread takes per pass, and the largest grid: six blocks on each of
// 152 SMs (1,536 threads with ten to fourteen loads in flight each)
constexpr int kCells = 2;
constexpr int kMaxBlocks = 6 * rich::kSMs;

// scratch: per-block minima of the cell time step as bit patterns (the
// integer order of non-negative doubles is their numeric order; kBad marks
// a block that met a cell whose time step is not a finite non-negative
// number), then counters of the blocks that have finished.  Calls take the
// counters in turn; a call leaves its own at zero, and clears the one that comes
// kCounters / 2 calls later, so that calls that overlapped against the rule, or
// a kernel that did not finish, spoil no later one.  (One counter that a memset
// cleared before each call: 1 us more of a small call's 8.  A captured call
// keeps its counter in every replay.)
constexpr int kCounters = 64;
static __device__ __align__(256) unsigned long long g_courant_scratch[kMaxBlocks + kCounters];

constexpr unsigned long long kBad = ~0ull;

// The cell time step's bits as the sweep's own reduction orders them: a
// non-negative double's bits; -0.0, negative values and NaNs (negative as an
// integer, or above the bits of +inf) are flagged instead of being skipped.
__device__ __forceinline__ unsigned long long step_key(double v, bool &bad)
{
    const long long k = __double_as_longlong(v);
    if (k < 0 || k > 0x7ff0000000000000ll) {
        bad = true;
        return kBad;
    }
    return (unsigned long long)k;
}

__device__ __forceinline__ unsigned long long key_min(unsigned long long a, unsigned long long b)
{
    return a < b ? a : b;
}

// |v| with its mantissa cut to 24 bits, for an exponent field in [1023 -
// span, 1023 + span] (span <= 100): two shifts on the integer pipe.  FP64 to
// FP32 conversions issue on the FP64 pipe.
__device__ __forceinline__ float cut(double v)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    return __uint_as_float(__funnelshift_l(lo, hi, 3) - 0xc0000000u);
}
// v positive with an exponent within 2^-span .. 2^span
__device__ __forceinline__ bool in_span(double v, unsigned span)
{
    return ((unsigned)__double2hiint(v) >> 20) - (1023u - span) <= 2u * span;
}
__device__ __forceinline__ float root(float v)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float inverse(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// Bound by DRAM (56 B per cell of a moving mesh) where evaluating every cell
// in FP64 was bound by the FP64 pipe, which issues one warp instruction per
// 16 clocks per SM: about 110 of them per cell step (three square roots and
// two divides).  Each cell's time step is first estimated in FP32 within
// 1e-6, and only cells whose estimate is within 4e-6 of the smallest in their
// block, which the smallest time step's cell always is, are evaluated in FP64
// with the formula of the sweep: the result's bits are those of evaluating
// every cell.  A thread keeps the latest such cell until the block's smallest
// estimate is known, and evaluates a second one beside it (a tie) at once.
// Cells outside the estimate's range (gamma of 2^20 and above, density or
// pressure beyond 2^+-30, area beyond 2^+-100, speeds above 2^60, and
// everything negative or not finite) are always evaluated.
__global__ void __launch_bounds__(kBlock, 6) k_courant_noalloc(
    int32_t n, double gamma, float gamma_f, double cfl, int32_t motion_static, const double *__restrict__ area,
    const double *__restrict__ rho, const double *__restrict__ vx, const double *__restrict__ vy,
    const double *__restrict__ p, const double *__restrict__ wx, const double *__restrict__ wy,
    unsigned long long *scratch, int32_t counter, double *dt_out)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) scratch[kMaxBlocks + (counter + kCounters / 2) % kCounters] = 0;
    // kMax: the bits of +inf, above every finite non-negative time step
    const unsigned long long kMax = 0x7ff0000000000000ull;
    constexpr unsigned kNone = 0x7f800000u;  // estimate of no cell
    unsigned long long k = kMax;
    bool bad = false;
    __shared__ unsigned smallest;
    if (threadIdx.x == 0) smallest = kNone;
    __syncthreads();
    float kept = __uint_as_float(kNone);  // this thread's latest candidate
    int32_t kept_cell = -1;
    auto evaluate = [&](double area_i, double rho_i, double p_i, double ux_i, double uy_i) {
        const double cs = sqrt(gamma * p_i / rho_i);
        const double R = sqrt(area_i * (1.0 / M_PI));
        k = key_min(k, step_key(R / (cs + sqrt(ux_i * ux_i + uy_i * uy_i)), bad));
    };
    for (int32_t base = blockIdx.x * kBlock * kCells; base < n; base += gridDim.x * kBlock * kCells) {
        double A[kCells], r[kCells], P[kCells], ux[kCells], uy[kCells];
        float est[kCells];
#pragma unroll
        for (int c = 0; c < kCells; c++) {
            const int32_t i = base + c * kBlock + threadIdx.x;
            if (i < n) {
                A[c] = __ldcs(area + i);
                r[c] = __ldcs(rho + i);
                P[c] = __ldcs(p + i);
                ux[c] = __ldcs(vx + i);
                uy[c] = __ldcs(vy + i);
                if (!motion_static) {
                    ux[c] -= __ldcs(wx + i);
                    uy[c] -= __ldcs(wy + i);
                }
            }
        }
        unsigned least = kNone;
#pragma unroll
        for (int c = 0; c < kCells; c++) {
            est[c] = __uint_as_float(kNone);
            if (base + c * kBlock + (int32_t)threadIdx.x >= n) continue;
            const unsigned ex = ((unsigned)__double2hiint(ux[c]) >> 20) & 0x7ffu;
            const unsigned ey = ((unsigned)__double2hiint(uy[c]) >> 20) & 0x7ffu;
            if (!(gamma_f < 1048576.0f && in_span(r[c], 30) && in_span(P[c], 30) && in_span(A[c], 100) && ex <= 1083u && ey <= 1083u)) {
                est[c] = 0.0f;  // always evaluated
                continue;
            }
            // (a speed below 2^-100 vanishes beside c_s > 2^-31)
            const float fx = ex < 923u ? 0.0f : cut(ux[c]), fy = ey < 923u ? 0.0f : cut(uy[c]);
            const float cs = root(gamma_f * cut(P[c]) * inverse(cut(r[c])));
            est[c] = root(cut(A[c]) * 0.318309886f) * inverse(cs + root(fx * fx + fy * fy));
            least = min(least, __float_as_uint(est[c]));
        }
        least = __reduce_min_sync(0xffffffffu, least);
        // (the block's smallest so far, and this warp's; other warps may lower
        // it meanwhile: any of its values does)
        const unsigned before = *(volatile unsigned *)&smallest;
        if ((threadIdx.x & 31) == 0 && least < before) atomicMin(&smallest, least);
        const float limit = __uint_as_float(min(least, before)) * 1.000004f;
#pragma unroll
        for (int c = 0; c < kCells; c++) {
            const int32_t i = base + c * kBlock + threadIdx.x;
            if (i >= n || !(est[c] <= limit)) continue;
            if (est[c] == 0.0f || kept <= limit) {
                evaluate(A[c], r[c], P[c], ux[c], uy[c]);
            } else {
                // (a kept cell above the limit cannot hold the minimum)
                kept = est[c];
                kept_cell = i;
            }
        }
    }
    __syncthreads();
    if (kept_cell >= 0 && kept <= __uint_as_float(smallest) * 1.000004f) {
        const int32_t i = kept_cell;
        evaluate(area[i], rho[i], p[i], motion_static ? vx[i] : vx[i] - wx[i], motion_static ? vy[i] : vy[i] - wy[i]);
    }
    bad = __any_sync(0xffffffffu, bad);
    for (int o = 16; o > 0; o >>= 1) k = key_min(k, __shfl_down_sync(0xffffffffu, k, o));
    __shared__ unsigned long long red[kBlock / 32];
    __shared__ int bad_block;
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) bad_block = 0;
    __syncthreads();
    if (lane == 0) {
        red[wid] = k;
        if (bad) bad_block = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long m = red[0];
        for (int q = 1; q < kBlock / 32; q++) m = key_min(m, red[q]);
        scratch[blockIdx.x] = bad_block ? kBad : m;
        __threadfence();
        last = atomicAdd(&scratch[kMaxBlocks + counter], 1ull) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    // the last block to finish reduces the per-block minima
    __threadfence();
    if (threadIdx.x == 0) scratch[kMaxBlocks + counter] = 0;
    unsigned long long m = kMax;
    bool any_bad = false;
    for (int32_t b = threadIdx.x; b < (int32_t)gridDim.x; b += blockDim.x) {
        const unsigned long long v = ((volatile unsigned long long *)scratch)[b];
        if (v == kBad) any_bad = true;
        else m = key_min(m, v);
    }
    any_bad = __any_sync(0xffffffffu, any_bad);
    for (int o = 16; o > 0; o >>= 1) m = key_min(m, __shfl_down_sync(0xffffffffu, m, o));
    __syncthreads();
    if (threadIdx.x == 0) bad_block = 0;
    __syncthreads();
    if (lane == 0) {
        red[wid] = m;
        if (any_bad) bad_block = 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long r = red[0];
        for (int q = 1; q < kBlock / 32; q++) r = key_min(r, red[q]);
        *dt_out = bad_block ? __longlong_as_double(0x7ff8000000000000ll) : cfl * __longlong_as_double((long long)r);
    }
}

std::atomic<uint32_t> g_calls{0};
std::mutex g_setup_mutex;
unsigned long long *g_scratch_addr[64] = {};

}  // namespace

extern "C" int rich_courant_dt_noalloc(const rich_config *cfg, int64_t n, const double *area, const double *rho,
                                       const double *vx, const double *vy, const double *p, const double *wx,
                                       const double *wy, double *dt_out, void *stream)
{
    if (!rich::valid_config(cfg)) return rich::set_error(RICH_EINVAL, "invalid configuration");
    if (!area || !rho || !vx || !vy || !p || !dt_out) return rich::set_error(RICH_EINVAL, "NULL array");
    if (cfg->motion != RICH_MESH_EULERIAN && (!wx || !wy))
        return rich::set_error(RICH_EINVAL, "wx, wy are needed with a moving mesh");
    if (n < 1 || n > RICH_NOALLOC_MAX_CELLS)
        return rich::set_error(RICH_EINVAL, "n must be in [1, RICH_NOALLOC_MAX_CELLS]");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return rich::set_error(RICH_ECUDA, "no device");
    unsigned long long *scratch;
    {
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_scratch_addr[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_courant_scratch) != cudaSuccess || !ptr)
                return rich::set_error(RICH_ECUDA, "cudaGetSymbolAddress failed for the scratch array");
            g_scratch_addr[dev] = static_cast<unsigned long long *>(ptr);
        }
        scratch = g_scratch_addr[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int32_t counter = (int32_t)(g_calls.fetch_add(1, std::memory_order_relaxed) % kCounters);
    const int64_t tile = (int64_t)kBlock * kCells;
    const int blocks = (int)std::min<int64_t>((n + tile - 1) / tile, kMaxBlocks);
    k_courant_noalloc<<<blocks, kBlock, 0, st>>>((int32_t)n, cfg->gamma, (float)cfg->gamma, cfg->cfl,
                                                 cfg->motion == RICH_MESH_EULERIAN ? 1 : 0, area, rho, vx, vy, p,
                                                 wx, wy, scratch, counter, dt_out);
    return cudaGetLastError() == cudaSuccess ? RICH_OK : rich::set_error(RICH_ECUDA, "launch failed");
}

// Conservation sums without any allocation (lb_conservation_static).
//
// The library's own reductions keep their per-block partial sums in device
// memory the context allocates. This variant keeps them in a fixed
// file-scope device array instead, so a caller that must not allocate
// device memory can still get the FP64 mass and momentum totals of a
// population field. The array lives on every GPU that loads the library
// until the process exits; all calls share it.
#include "../../include/lbsc.h"
#include "lb_fields.cuh"

#include <mutex>
#include <string>

namespace lbsc {

constexpr int kStaticChunks = 32;                     // most node ranges an array is cut into: 1216 blocks, one wave (64 and 96: no faster)
constexpr long long kStaticMinNodes = 2048;           // nodes of a range at least (small fields use few)
constexpr long long kStaticMaxNodes = 67108864;       // largest field
constexpr int kStaticThreads = 256;
constexpr int kStaticUnroll = 8;                      // loads in flight a thread
constexpr int kMaxDevices = 64;

// 64 KiB of partial sums: the sum of array ak = 19 a + k and range c at
// ak chunks + c, then (32-bit words) the arrays' non-finite counts in the same
// order and the fluid nodes of every range
static __device__ __align__(256) double g_static_partials[8192];
static_assert(2 * Q * kStaticChunks * 12 + kStaticChunks * 4 <= 65536, "the partial sums fit the static array");

// The sum of eight values as integers: their significands, aligned to the
// largest exponent with 7 bits below its last, fit a signed 64-bit sum exactly
// but for what lies 2^-60 below the largest value, which is less than adding
// them one by one in FP64 loses. One conversion and one FP64 fused multiply-add
// then take the eight into s. Values that are not finite, or all so small that
// the scale would not be a normal number, are added in FP64.
__device__ __forceinline__ void add_eight(const double (&v)[kStaticUnroll], double& s, int& bad)
{
    int emax = 0;
#pragma unroll
    for (int u = 0; u < kStaticUnroll; ++u) emax = max(emax, (__double2hiint(v[u]) >> 20) & 0x7FF);
    if (emax == 0x7FF || emax < 64) {
        for (int u = 0; u < kStaticUnroll; ++u) {
            bad += (__double2hiint(v[u]) & 0x7FF00000) == 0x7FF00000;  // infinity or NaN
            s += v[u];
        }
        return;
    }
    long long t = 0;
#pragma unroll
    for (int u = 0; u < kStaticUnroll; ++u) {
        const int hi = __double2hiint(v[u]);
        const int e = (hi >> 20) & 0x7FF;
        const unsigned top = ((unsigned)hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
        const unsigned long long m = ((unsigned long long)top << 32 | (unsigned)__double2loint(v[u])) << 7;
        long long w;  // PTX shifts by 64 and more give 0 (C++ leaves them undefined)
        asm("shr.u64 %0, %1, %2;" : "=l"(w) : "l"(m), "r"(emax - max(e, 1)));
        const long long neg = (long long)(hi >> 31);
        t += (w ^ neg) - neg;
    }
    // a significand of 53 bits shifted by 7 stands for 2^(emax - 1023 - 59)
    s = fma((double)t, __hiloint2double((emax - 59) << 20, 0), s);
}

// Block (c, ak) sums range c of one population array. FP64 operations run at
// about one a clock and SM here, so their number bounded the kernel: now two
// for eight values (add_eight; moments per node took 5 to 8 a value, a plain
// sum with its test for finite values 2), and a block's threads are summed by
// one warp. The moments are formed from the 38 totals in static_finish_kernel.
// 64^3: 147 us with whole nodes in 128 blocks, 39 with a plain sum, about 15
// now (both kernels, the second launched dependently, 24.6 a call; 128^3 116, 0.83 of the measured bandwidth).
__global__ void __launch_bounds__(kStaticThreads)
    static_sum_kernel(const double* __restrict__ n, const uint8_t* __restrict__ solid, long long N, int chunks,
                      double* __restrict__ part)
{
    const int c = blockIdx.x, ak = blockIdx.y;
    grid_trigger();
    const long long lo = c * N / chunks, hi = (c + 1) * N / chunks;
    const double* __restrict__ p = n + (long long)ak * N;
    double s = 0;
    int bad = 0, fluid = 0;
    // whole strips of 8 x 256 nodes without bounds tests, then the rest; a solid node's value is loaded too (its mask byte
    // and the value are in flight together) and taken as 0
    long long i = lo + threadIdx.x;
    for (; i + (kStaticUnroll - 1) * kStaticThreads < hi; i += kStaticUnroll * kStaticThreads) {
        double v[kStaticUnroll];
        uint8_t no[kStaticUnroll];
        const double* q = p + i;
#pragma unroll
        for (int u = 0; u < kStaticUnroll; ++u) v[u] = q[u * kStaticThreads];
        if (solid) {
#pragma unroll
            for (int u = 0; u < kStaticUnroll; ++u) no[u] = solid[i + u * kStaticThreads];
#pragma unroll
            for (int u = 0; u < kStaticUnroll; ++u) {
                v[u] = no[u] ? 0.0 : v[u];
                fluid += no[u] == 0;
            }
        } else {
            fluid += kStaticUnroll;
        }
        add_eight(v, s, bad);
    }
    if (i < hi) {
        double v[kStaticUnroll];
#pragma unroll
        for (int u = 0; u < kStaticUnroll; ++u) {
            const long long j = i + u * kStaticThreads;
            const bool in = j < hi && !(solid && solid[j]);
            v[u] = in ? p[j] : 0.0;
            fluid += in;
        }
        add_eight(v, s, bad);
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    fluid = __reduce_add_sync(0xffffffffu, fluid);
    __shared__ double sh[kStaticThreads];
    __shared__ int si[kStaticThreads / 32][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sh[threadIdx.x] = s;
    if (lane == 0) {
        si[warp][0] = bad;
        si[warp][1] = fluid;
    }
    __syncthreads();
    if (warp == 0) {
        double t = sh[lane];
        int b = 0, f = 0;
#pragma unroll
        for (int w = 0; w < kStaticThreads / 32; ++w) {
            if (w) t += sh[32 * w + lane];
            b += si[w][0];
            f += si[w][1];
        }
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) {
            int* count = (int*)(part + 2 * Q * chunks);
            part[ak * chunks + c] = t;
            count[ak * chunks + c] = b;
            if (ak == 0) count[2 * Q * chunks + c] = f;
        }
    }
}

// The 38 arrays' totals (warp w takes arrays w and w + 32, the ranges in a
// fixed tree), then {M_r, M_b, Px, Py, Pz, non-finite count, fluid nodes, 0},
// a warp each (a chain of FP64 additions in one thread took 12 us)
__global__ void __launch_bounds__(1024) static_finish_kernel(const double* part, int chunks,
                                                             double* __restrict__ out)
{
    __shared__ double tot[2 * Q];
    __shared__ int num[2 * Q + 1];
    const int* count = (const int*)(part + 2 * Q * chunks);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_wait();
    for (int r = warp; r <= 2 * Q; r += 32) {
        double t = 0;
        int b = 0;
        for (int c = lane; c < chunks; c += 32) {
            if (r < 2 * Q) t += part[r * chunks + c];
            b += count[r * chunks + c];
        }
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        b = __reduce_add_sync(0xffffffffu, b);
        if (lane == 0) {
            if (r < 2 * Q) tot[r] = t;
            num[r] = b;
        }
    }
    __syncthreads();
    if (warp >= 8) return;
    double x = 0;
    long long b = 0;  // 38 counts of up to 67,108,864
    for (int r = lane; r < 2 * Q; r += 32) {
        const int k = r % Q;
        if (warp < 2) x += r / Q == warp ? tot[r] : 0.0;
        // the zero products too: a total that is not finite shows in every sum of the momentum
        else if (warp < 5) x += (warp == 2 ? cx(k) : (warp == 3 ? cy(k) : cz(k))) * tot[r];
        else if (warp == 5) b += num[r];
    }
    for (int o = 16; o > 0; o >>= 1) {
        if (warp < 5) x += __shfl_down_sync(0xffffffffu, x, o);
        else b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) out[warp] = warp < 5 ? x : (warp == 5 ? (double)b : (warp == 6 ? (double)num[2 * Q] : 0.0));
}

// Device address of the static array on the current device. Host code only
// sees a host-side stand-in under the array's name, so the address is looked
// up once per device (the first call on that device) and cached.
static int static_partials(double** out, std::string& err)
{
    static std::mutex mu;
    static double* addr[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        err = std::string("lb_conservation_static: cudaGetDevice: ") + cudaGetErrorString(e);
        return LB_ERR_CUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) {
        err = "lb_conservation_static: device index beyond the supported 64";
        return LB_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_partials);
        if (e != cudaSuccess || !p) {
            err = std::string("lb_conservation_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e);
            return LB_ERR_CUDA;
        }
        addr[dev] = (double*)p;
    }
    *out = addr[dev];
    return LB_OK;
}

}  // namespace lbsc

// error message for the context-free entry point, read through lb_last_error(NULL)
void lbsc_set_global_error(const std::string& msg);

extern "C" int lb_conservation_static(const double* populations, const uint8_t* solid, int nx, int ny, int nz,
                                      double* cons, void* cuda_stream)
{
    using namespace lbsc;
    if (!populations || !cons) {
        lbsc_set_global_error("lb_conservation_static: populations and cons must be device pointers");
        return LB_ERR_ARG;
    }
    if (nx < 1 || ny < 1 || nz < 1) {
        lbsc_set_global_error("lb_conservation_static: bad lattice dimensions");
        return LB_ERR_ARG;
    }
    const long long N = (long long)nx * ny * nz;
    if (N > kStaticMaxNodes) {
        lbsc_set_global_error("lb_conservation_static: " + std::to_string(N) +
                              " nodes exceed the static scratch maximum of 67108864 nodes");
        return LB_ERR_ARG;
    }
    std::string err;
    double* part = nullptr;
    const int rc = static_partials(&part, err);
    if (rc != LB_OK) {
        lbsc_set_global_error(err);
        return rc;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const long long want = (N + kStaticMinNodes - 1) / kStaticMinNodes;
    const int chunks = (int)(want < kStaticChunks ? want : kStaticChunks);
    static_sum_kernel<<<dim3(chunks, 2 * Q), kStaticThreads, 0, st>>>(populations, solid, N, chunks, part);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_after(static_finish_kernel, dim3(1), 1024, 0, st, part, chunks, cons);
    if (e != cudaSuccess) {
        lbsc_set_global_error(std::string("lb_conservation_static: launch: ") + cudaGetErrorString(e));
        return LB_ERR_CUDA;
    }
    return LB_OK;
}

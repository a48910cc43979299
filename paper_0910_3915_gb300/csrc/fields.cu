// Non-step kernels: initial equilibrium, FP64 conservation sums, moment
// fields for readback, contact-angle reductions and population copies.
// All reductions are deterministic: the conservation sums are exact integer
// (fixed-point) sums; the others use a fixed grid, fixed per-thread ranges,
// warp shuffles and a final pass over the per-block partials in block order.
#include "lb_fields.cuh"

#include <type_traits>

namespace lbsc {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// Sum (or max) nrows partial rows of NV values: block v reduces value v,
// thread t taking rows t, t + 256, ... in order, then a fixed shuffle tree per
// warp and the warps in order. Launched as NV blocks of 256 threads.
template <int NV>
__global__ void __launch_bounds__(256) finish_rows_kernel(const double* __restrict__ part, int nrows, uint32_t is_max,
                                                          double* __restrict__ out)
{
    const int v = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (v >= NV) return;
    const bool mx = (is_max >> v) & 1u;
    double a = mx ? -1e300 : 0.0;
    for (int r = threadIdx.x; r < nrows; r += blockDim.x) {
        const double p = part[(long long)r * NV + v];
        a = mx ? fmax(a, p) : a + p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_down_sync(0xffffffffu, a, o);
        a = mx ? fmax(a, w) : a + w;
    }
    __shared__ double sw[8];
    if (lane == 0) sw[warp] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = sw[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) t = mx ? fmax(t, sw[w]) : t + sw[w];
        out[v] = t;
    }
}

// blocks for n items at `threads` per block, at most cap (grid-stride loops cover the rest)
static int grid_for(long long n, int threads, int cap)
{
    long long b = (n + threads - 1) / threads;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

template <class S>
__device__ __forceinline__ float decode_val(float v, int k, float ref)
{
    if constexpr (Codec<S>::kDeviation) return zeta(k) * (ref + v);
    else return v;
}
template <class S>
__device__ __forceinline__ float decode(const S* p, int k, float ref)
{
    return decode_val<S>(Codec<S>::load(p), k, ref);
}

// both components' n_k of one node from their paired storage
template <class S>
__device__ __forceinline__ void decode2(const S* p, int k, const float (&ref)[2], float& n0, float& n1)
{
    const float2 v = Codec<S>::load2(p);
    if constexpr (Codec<S>::kDeviation) {
        // explicitly rounded, so that no kernel fuses the product into a later
        // sum: every readback pass sees the same n_k (and the same rho)
        n0 = __fmul_rn(zeta(k), __fadd_rn(ref[0], v.x));
        n1 = __fmul_rn(zeta(k), __fadd_rn(ref[1], v.y));
    } else {
        n0 = v.x;
        n1 = v.y;
    }
}

__device__ __forceinline__ bool node_solid(const FieldArgs& F, int x, int y, int z, long long off)
{
    if (F.general) return (F.nbmask[off] & kSelfSolid) != 0;
    return z == 0 || z == F.L.nz - 1;
}

// ---------------------------------------------------------------- init
// populations at rest: n_k = zeta_k rho (Eq. Equil at u = 0). err (may be
// NULL): kErrInput is set for a density that is negative or not finite.
template <class S>
__global__ void init_kernel(FieldArgs F, S* __restrict__ f, const double* __restrict__ rr, const double* __restrict__ rb,
                            int* err)
{
    const unsigned nxy = (unsigned)F.L.nx * (unsigned)F.L.ny;
    const unsigned N = nxy * (unsigned)F.L.nz;  // below 2^31 (the layout's limit)
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const unsigned z = i / nxy, rem = i - z * nxy;
        const int y = (int)(rem / (unsigned)F.L.nx), x = (int)(rem - (unsigned)y * F.L.nx);
        const double d0 = rr[i], d1 = rb[i];
        if (err && !(isfinite(d0) && d0 >= 0.0 && isfinite(d1) && d1 >= 0.0)) atomicOr(err, kErrInput);
        const float r0 = (float)d0, r1 = (float)d1;
        const long long zoff = (long long)z * F.L.plane;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            if constexpr (Codec<S>::kDeviation)
                put_pair<S>(f + F.L.at(0, k, 0), F.L, x, y, zoff, r0 - F.P.ref[0], r1 - F.P.ref[1]);
            else
                put_pair<S>(f + F.L.at(0, k, 0), F.L, x, y, zoff, zeta(k) * r0, zeta(k) * r1);
        }
    }
}

// ---------------------------------------------------------------- conservation
// cons = {M_r, M_b, Px, Py, Pz, non-finite count, fluid nodes, -}
// A grid-stride walk over the nodes of the fluid planes, x fastest, so that a
// warp's load of one population slot covers consecutive addresses, with a
// node's 38 loads independent of each other. A node's mass and momentum are
// summed in FP32 over its 19 values per component, and each thread adds its
// nodes in FP32. The threads' sums then go into 64-bit integers in units of
// 2^-28 (kConsFix) and are added as integers: across warps, blocks and the
// whole grid, by shuffles and atomics. Integer addition is exact and
// associative, so the totals do not depend on the grid or on the order the
// blocks finish, and no FP64 arithmetic (slow on this GPU) runs per node. The
// last block to finish converts the totals to FP64 into out[0..7] and clears
// the accumulators (acc[0..7], ticket) for the next call.
__device__ __forceinline__ long long to_fix(float v) { return __float2ll_rn(v * kConsFix); }

// With phi non-NULL the same pass also writes phi = rho_r - rho_b of every
// node (0 on solid nodes), summed as the contact angle's phi pass sums it, so
// a measurement of both needs one read of the populations.
template <class S>
__global__ void __launch_bounds__(kRedThreads) cons_kernel(FieldArgs F, const S* __restrict__ f,
                                                           unsigned long long* __restrict__ acc,
                                                           unsigned int* __restrict__ ticket, double* __restrict__ out,
                                                           float* __restrict__ phi)
{
    float m[2] = {0.f, 0.f}, j[3] = {0.f, 0.f, 0.f};
    int bad = 0, fluid = 0;
    const int nx = F.L.nx, ny = F.L.ny;
    const unsigned nxy = (unsigned)nx * (unsigned)ny;
    const unsigned n = nxy * (unsigned)F.L.nz;  // below 2^31 (the layout's limit)
    const unsigned T = gridDim.x * blockDim.x;
    const float ref[2] = {F.P.ref[0], F.P.ref[1]};
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += T) {
        const unsigned zr = i / nxy, rem = i - zr * nxy;
        const int y = (int)(rem / (unsigned)nx), x = (int)(rem - (unsigned)y * nx), z = (int)zr;
        const long long off = F.L.off(x, y, z);
        if (node_solid(F, x, y, z, off)) {
            if (phi) phi[i] = 0.f;
            continue;
        }
        ++fluid;
        float v[2][Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) decode2<S>(f + F.L.at(0, k, off), k, ref, v[0][k], v[1][k]);
        float rho[2], jn[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const float nk = v[a][k];
                bad += isfinite(nk) ? 0 : 1;
                s = __fadd_rn(s, nk);  // as the phi pass
                if (cx(k)) jn[0] += cx(k) * nk;
                if (cy(k)) jn[1] += cy(k) * nk;
                if (cz(k)) jn[2] += cz(k) * nk;
            }
            rho[a] = s;
        }
        if (phi) phi[i] = rho[0] - rho[1];
        m[0] += rho[0];
        m[1] += rho[1];
#pragma unroll
        for (int d = 0; d < 3; ++d) j[d] += jn[d];
    }
    // a non-finite value would make the fixed-point conversion meaningless: it is counted instead
    const bool fin = bad == 0 && isfinite(m[0]) && isfinite(m[1]) && isfinite(j[0]) && isfinite(j[1]) && isfinite(j[2]);
    long long q[7] = {fin ? to_fix(m[0]) : 0, fin ? to_fix(m[1]) : 0, fin ? to_fix(j[0]) : 0, fin ? to_fix(j[1]) : 0,
                      fin ? to_fix(j[2]) : 0, (long long)bad + (fin ? 0 : 1) * (bad == 0), (long long)fluid};
#pragma unroll
    for (int v = 0; v < 7; ++v)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) q[v] += __shfl_down_sync(0xffffffffu, q[v], o);
    __shared__ long long sh[kRedThreads / 32][7];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int v = 0; v < 7; ++v) sh[warp][v] = q[v];
    __syncthreads();
    __shared__ bool last;
    if (threadIdx.x < 7) {
        long long t = 0;
        for (int w = 0; w < kRedThreads / 32; ++w) t += sh[w][threadIdx.x];
        atomicAdd(&acc[threadIdx.x], (unsigned long long)t);  // two's complement: signed sums wrap correctly
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && threadIdx.x < 8) {
        __threadfence();
        const int v = threadIdx.x;
        const long long t = v < 7 ? (long long)atomicExch(&acc[v], 0ull) : 0;
        out[v] = v < 5 ? (double)t / kConsFix : (double)t;
        if (v == 0) *ticket = 0u;
    }
}

// ---------------------------------------------------------------- moment fields
// rho^r, rho^b, total j and psi of every node (psi = wall pseudo-density on
// solid). Bound by the read of the populations and the write of the fields. A
// 16-bit velocity's two components come in one load (256x256x128 BF16: 136
// us, 178 with one load each); FP32 takes them apart, the second from L1, with
// 32 registers instead of 48 (128^3: 54 us against 64).
template <class S>
__global__ void __launch_bounds__(kRedThreads) fields_kernel(FieldArgs F, const S* __restrict__ f, Scratch W)
{
    const unsigned nx = (unsigned)F.L.nx, nxy = nx * (unsigned)F.L.ny, N = nxy * (unsigned)F.L.nz;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int z = (int)(i / nxy), y = (int)((i - z * nxy) / nx), x = (int)(i - z * nxy - y * nx);
        const long long off = F.L.off(x, y, z);
        float rho[2] = {0.f, 0.f}, j[3] = {0.f, 0.f, 0.f};
        const bool solid = node_solid(F, x, y, z, off);
        if (!solid) {
            float2 v[Q];
            if constexpr (sizeof(S) == 2)
#pragma unroll
                for (int k = 0; k < Q; ++k) v[k] = Codec<S>::load2(f + F.L.at(0, k, off));
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int k = 0; k < Q; ++k) {
                    float n;
                    if constexpr (sizeof(S) == 2) n = decode_val<S>(a ? v[k].y : v[k].x, k, F.P.ref[a]);
                    else n = Codec<S>::load(f + F.L.at(a, k, off));
                    rho[a] += n;
                    j[0] += cx(k) * n;
                    j[1] += cy(k) * n;
                    j[2] += cz(k) * n;
                }
        }
        W.rho[0][i] = rho[0];
        W.rho[1][i] = rho[1];
        for (int d = 0; d < 3; ++d) W.j[d][i] = j[d];
        for (int a = 0; a < 2; ++a) W.psi[a][i] = solid ? F.P.eta[a] : -expm1f(-rho[a]);
    }
}

// u = (j + F/2) / (rho_r + rho_b) of the fluid node (x, y, z) at index i, F the
// total Shan-Chen force (Eq. SCforce)
__device__ __forceinline__ void node_velocity(const FieldArgs& F, const Scratch& W, int x, int y, int z, unsigned i,
                                              float (&u)[3])
{
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    const int xo[3] = {wrapi(x - 1, nx), x, wrapi(x + 1, nx)};
    const int yo[3] = {nx * wrapi(y - 1, ny), nx * y, nx * wrapi(y + 1, ny)};
    const int zo[3] = {nx * ny * wrapi(z - 1, nz), nx * ny * z, nx * ny * wrapi(z + 1, nz)};
    const float tot = W.rho[0][i] + W.rho[1][i];
    u[0] = u[1] = u[2] = 0.f;
    if (!(tot > 0.f)) return;
    float Ft[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        float s[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            const int ip = xo[cx(k) + 1] + yo[cy(k) + 1] + zo[cz(k) + 1];
            const float G = is_axis(k) ? F.P.Gax : F.P.Gdi;
            const float ps = W.psi[1 - a][ip];
            s[0] += G * ps * cx(k);
            s[1] += G * ps * cy(k);
            s[2] += G * ps * cz(k);
        }
        const float pre = -F.P.gk * W.psi[a][i];
        for (int d = 0; d < 3; ++d) Ft[d] += pre * s[d];
    }
    for (int d = 0; d < 3; ++d) u[d] = (W.j[d][i] + 0.5f * Ft[d]) / tot;
}

__global__ void __launch_bounds__(kRedThreads) velocity_kernel(FieldArgs F, Scratch W)
{
    const unsigned nx = (unsigned)F.L.nx, nxy = nx * (unsigned)F.L.ny, N = nxy * (unsigned)F.L.nz;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int z = (int)(i / nxy), y = (int)((i - z * nxy) / nx), x = (int)(i - z * nxy - y * nx);
        float u[3] = {0.f, 0.f, 0.f};
        if (!node_solid(F, x, y, z, F.L.off(x, y, z))) node_velocity(F, W, x, y, z, i, u);
        for (int d = 0; d < 3; ++d) W.u[d][i] = u[d];
    }
}

// phi = rho_r - rho_b of every node into W.rho[0] (0 on solid nodes), the
// contact angle's only input: FP32 sums of each component's 19 values, then
// their difference
template <class S>
__global__ void phi_kernel(FieldArgs F, const S* __restrict__ f, Scratch W)
{
    const int nx = F.L.nx, ny = F.L.ny;
    const unsigned nxy = (unsigned)nx * (unsigned)ny;
    const unsigned N = nxy * (unsigned)F.L.nz;
    const unsigned T = gridDim.x * blockDim.x;
    const float ref[2] = {F.P.ref[0], F.P.ref[1]};
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += T) {
        const unsigned z = i / nxy, rem = i - z * nxy;
        const int y = (int)(rem / (unsigned)nx), x = (int)(rem - (unsigned)y * nx);
        const long long off = F.L.off(x, y, (int)z);
        float rho[2] = {0.f, 0.f};
        if (!node_solid(F, x, y, (int)z, off)) {
            float v[2][Q];
#pragma unroll
            for (int k = 0; k < Q; ++k) decode2<S>(f + F.L.at(0, k, off), k, ref, v[0][k], v[1][k]);
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int k = 0; k < Q; ++k) rho[a] = __fadd_rn(rho[a], v[a][k]);  // as the conservation pass
        }
        W.rho[0][i] = rho[0] - rho[1];
    }
}

// ---------------------------------------------------------------- contact angle
// phi - level in FP64 at a node whose phi is the FP32 value p
__device__ __forceinline__ double phi_at(float p, double level) { return (double)p - level; }

// p > level in FP64, out of line: the rare case the FP32 test below cannot decide
__device__ __noinline__ bool above_fp64(float p, double level) { return (double)p > level; }

// p > level, i.e. phi_at(p, level) > 0, taken in FP32 where that is exact: when
// level is an FP32 number, or when p is far from it (the margin exceeds the
// rounding of level to FP32 many times over); else in FP64.
__device__ __forceinline__ bool above(float p, float lf, bool lexact, double level)
{
    if (lexact || fabsf(p - lf) > 1e-6f * (fabsf(p) + fabsf(lf)) + 1e-30f) return p > lf;
    return above_fp64(p, level);
}

// Positive length along x, from a node to its +x neighbour, of the linear
// interpolant of phi - level on the reference plane z0 + fz (p: phi at the
// node, above it, at the +x neighbour and above that). Out of line, so that
// its FP64 work runs only on that plane's rows.
__device__ __noinline__ double plane_length(float p0, float p0up, float p1, float p1up, double fz, double level)
{
    const double a0 = (1 - fz) * phi_at(p0, level) + fz * phi_at(p0up, level);
    const double a1 = (1 - fz) * phi_at(p1, level) + fz * phi_at(p1up, level);
    if (a0 > 0 && a1 > 0) return 1.0;
    if (a0 <= 0 && a1 <= 0) return 0.0;
    return a0 > 0 ? a0 / (a0 - a1) : a1 / (a1 - a0);
}

// An interface crossing between node (x, y, z) (phi = p0) and its neighbour
// along axis d (phi = p1): the top crossing (along z, from phi > level
// below to phi <= level above) and the sphere-fit sums of the crossing point at
// or above the reference plane, into the thread's accumulators acc[i * stride].
// Kept out of line so that the FP64 work runs only in the warps that meet a
// crossing instead of being predicated into every node's path.
__device__ __noinline__ void add_crossing(double* acc, int stride, int x, int y, int z, int d, float p0, float p1,
                                         double level, bool s0, double zref)
{
    const double q0 = phi_at(p0, level), q1 = phi_at(p1, level);
    const double t = q0 / (q0 - q1);
    if (d == 2 && s0) acc[0] = fmax(acc[0], z + t);  // phi > level below, <= level above
    const double pxv = x + t * (d == 0), pyv = y + t * (d == 1), pzv = z + t * (d == 2);
    if (pzv < zref) return;
    const double row[4] = {2 * pxv, 2 * pyv, 2 * pzv, 1.0};
    const double rhs = pxv * pxv + pyv * pyv + pzv * pzv;
    acc[2 * stride] += 1.0;
    int m = 3;
    for (int r = 0; r < 4; ++r)
        for (int q = r; q < 4; ++q) acc[(m++) * stride] += row[r] * row[q];
    for (int r = 0; r < 4; ++r) acc[(13 + r) * stride] += row[r] * rhs;
}

// One warp per lattice row, a lane per node, reading phi at the node and at
// its +x, +y, +z neighbours (the latter from L1/L2):
//  [0]  (max) top phi = level crossing: z + p0/(p0 - p1) where phi > level
//       below and <= level above (both nodes fluid);
//  [1]  positive length along x of the reference-plane interpolant of phi
//       (the node at z0 adds its segment to x + 1, periodic);
//  [2..16] sphere-fit sums over crossings along +x, +y, +z at or above the
//       reference plane: count, the 10 upper entries of M = sum row row^T and
//       the 4 of v = sum row |p|^2, row = (2p, 1);
//  [17] (max) max of phi over fluid nodes, [18] (max) of -phi (the contrast).
// FP64 arithmetic (slow on this GPU) runs only at crossings and on the
// reference plane; a thread's FP64 sums wait in shared memory, and a warp
// reduces a value only if one of its lanes holds a contribution to it.
__global__ void __launch_bounds__(kRedThreads) angle_kernel(FieldArgs F, Scratch W, double zref, double level,
                                                            double* __restrict__ part)
{
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    __shared__ double sacc[kAngleVals][kRedThreads];
    const int tid = threadIdx.x;
#define ACC(i) sacc[i][tid]
    for (int i = 0; i < 17; ++i) ACC(i) = 0.0;
    ACC(0) = -1e300;
    float pmax = -3.0e38f, pmin = 3.0e38f;
    const int z0 = (int)floor(zref);
    const double fz = zref - z0;
    const float lf = (float)level;
    const bool lexact = (double)lf == level;
    const float* __restrict__ P = W.rho[0];
    const unsigned nxy = (unsigned)nx * (unsigned)ny;
    // Interface crossings are rare and scattered: a lane that meets one would
    // run the FP64 work of add_crossing alone, at the cost of a whole warp's.
    // So the warp queues its crossings in shared memory, in lane order, and
    // works through them 32 at a time with every lane busy; which lane sums
    // which crossing depends only on the data, so the sums are reproducible.
    __shared__ int4 qpos[kRedThreads / 32][64];     // (x, y, z, axis)
    __shared__ float2 qphi[kRedThreads / 32][64];   // (phi at the node, phi at the neighbour)
    const int lane = tid & 31, warp = tid >> 5;
    int queued = 0;
    auto drain = [&](int n) {  // lanes < n take a queued crossing each, then the queue shifts by n
        __syncwarp();
        if (lane < n) {
            const int4 q = qpos[warp][lane];
            const float2 f = qphi[warp][lane];
            const bool s0 = above(f.x, lf, lexact, level);
            add_crossing(&sacc[0][tid], kRedThreads, q.x, q.y, q.z, q.w, f.x, f.y, level, s0, zref);
        }
        __syncwarp();
        if (lane + n < queued) {  // at most 31 left, read from [n, queued), written to [0, queued - n)
            const int4 q = qpos[warp][lane + n];
            const float2 f = qphi[warp][lane + n];
            qpos[warp][lane] = q;
            qphi[warp][lane] = f;
        }
        __syncwarp();
        queued -= n;
    };
    // a warp takes lattice rows (y, z) = w, w + W, ... (W warps in the grid), its lanes x = lane, lane + 32, ...
    const int rows = ny * nz, nwarps = gridDim.x * (kRedThreads / 32);
    for (int r = blockIdx.x * (kRedThreads / 32) + warp; r < rows; r += nwarps)
    for (int xb = 0; xb < nx; xb += 32) {  // warp-uniform: the queue needs the whole warp
        const int x = xb + lane;
        const bool in = x < nx;
        const int z = r / ny, y = r - z * ny;
        const unsigned i = (unsigned)r * (unsigned)nx + (unsigned)(in ? x : nx - 1);
        // the node and its +x, +y, +z neighbours (the node itself past an edge), loaded together
        const float p0 = P[i];
        const float pn[3] = {P[in && x + 1 < nx ? i + 1 : i], P[y + 1 < ny ? i + nx : i], P[z + 1 < nz ? i + nxy : i]};
        if (in && z == z0 && z0 + 1 < nz) {  // reference plane: every column, solid or not
            const unsigned i1 = x + 1 < nx ? i + 1 : i - x;
            ACC(1) += plane_length(p0, pn[2], P[i1], P[i1 + nxy], fz, level);
        }
        const bool fluid = in && (!F.general ? !(z == 0 || z == nz - 1) : (F.nbmask[F.L.off(x, y, z)] & kSelfSolid) == 0);
        if (fluid) {
            pmax = fmaxf(pmax, p0);
            pmin = fminf(pmin, p0);
        }
        const bool s0 = above(p0, lf, lexact, level);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int x1 = x + (d == 0), y1 = y + (d == 1), z1 = z + (d == 2);
            bool cross = fluid && x1 < nx && y1 < ny && z1 < nz;
            if (cross) cross = !(F.general ? (F.nbmask[F.L.off(x1, y1, z1)] & kSelfSolid) != 0 : z1 == nz - 1);
            if (cross) cross = s0 != above(pn[d], lf, lexact, level);
            const unsigned m = __ballot_sync(0xffffffffu, cross);
            if (cross) {
                const int at = queued + __popc(m & ((1u << lane) - 1u));
                qpos[warp][at] = make_int4(x, y, z, d);
                qphi[warp][at] = make_float2(p0, pn[d]);
            }
            queued += __popc(m);
            if (queued >= 32) drain(32);
        }
    }
    if (queued > 0) drain(queued);
    // block reduction: FP32 maxima by shuffles; FP64 values only in warps that hold some
    __shared__ double sh[kRedThreads / 32][kAngleVals];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pmax = fmaxf(pmax, __shfl_down_sync(0xffffffffu, pmax, o));
        pmin = fminf(pmin, __shfl_down_sync(0xffffffffu, pmin, o));
    }
    if (lane == 0) {
        sh[warp][17] = pmax > -3.0e38f ? (double)pmax : -1e300;
        sh[warp][18] = pmin < 3.0e38f ? -(double)pmin : -1e300;
    }
    for (int v = 0; v < 17; ++v) {
        const bool is_max = v == 0;
        double val = ACC(v);
        // a contribution changed the value's bits from their start (integer test: no FP64 operation)
        const bool held = __double_as_longlong(val) != __double_as_longlong(is_max ? -1e300 : 0.0);
        if (__any_sync(0xffffffffu, held)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double w = __shfl_down_sync(0xffffffffu, val, o);
                val = is_max ? fmax(val, w) : val + w;
            }
        }
        if (lane == 0) sh[warp][v] = val;
    }
#undef ACC
    __syncthreads();
    if (tid < kAngleVals) {
        const bool is_max = (kAngleMaxMask >> tid) & 1u;
        double v = sh[0][tid];
        for (int w = 1; w < kRedThreads / 32; ++w) v = is_max ? fmax(v, sh[w][tid]) : v + sh[w][tid];
        part[(long long)blockIdx.x * kAngleVals + tid] = v;
    }
}

// ---------------------------------------------------------------- pressure tensor
// Pressure tensor of Sec. 4.1 at a node:
//   P_ij = sum_a sum_k (c_ki - u_i)(c_kj - u_j) n_k^a
//        + 1/4 sum over the two ordered component pairs (a, abar) of
//          g kappa sum_k G_k [psi^a(x) psi^abar(x+c_k) + psi^abar(x) psi^a(x+c_k)] c_ki c_kj,
// u the moments' velocity (j + F/2)/rho, psi of a solid neighbour the wall
// pseudo-density (the force's reading of the wall). Both ordered pairs give the
// same bracket, so the interaction is 1/2 g kappa sum_k G_k [..] c_ki c_kj.
// Components xx, yy, zz, xy, xz, yz; zero on solid nodes.
//
// FP64 runs at a sixtieth of the FP32 rate on this GPU, so the sums are taken
// in pairs of FP32 numbers (Dekker 1971, Knuth's two-sum): a value is h + l
// with l far below h, a sum carries the rounding error of h in l. That keeps
// about 46 bits of the sums over exact FP32 inputs, 20 more than the stored
// populations hold. With u common to both components the kinetic term is
//   S_ij - u_i K_j - u_j J_i,  S = sum c c m,  J = sum c m,  K = J - u R,
//   R = sum m,  m_k = n_k^r + n_k^b,
// and S, J need the sums and differences of opposite velocities only. A node
// whose result is not finite is taken again in FP64, so that infinities and
// NaN come out as they always did.
struct Two {
    float h, l;
};
__device__ __forceinline__ Two two(float a) { return Two{a, 0.f}; }
__device__ __forceinline__ Two two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return Two{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// l may grow to a few roundings of h: normalised by norm2 before a product
__device__ __forceinline__ Two operator+(Two a, Two b)
{
    const Two s = two_sum(a.h, b.h);
    return Two{s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ Two operator-(Two a) { return Two{-a.h, -a.l}; }
__device__ __forceinline__ Two operator-(Two a, Two b) { return a + (-b); }
__device__ __forceinline__ Two norm2(Two a)
{
    const float s = __fadd_rn(a.h, a.l);
    return Two{s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}
__device__ __forceinline__ Two mul2f(Two a, float f)  // a normalised
{
    const float p = __fmul_rn(a.h, f);
    return Two{p, __fmaf_rn(a.l, f, __fmaf_rn(a.h, f, -p))};
}
__device__ __forceinline__ Two mul22(Two a, Two b)  // both normalised
{
    const float p = __fmul_rn(a.h, b.h);
    return Two{p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ double to_f64(Two a) { return (double)a.h + (double)a.l; }

// S_ij of values s[k] = v_k + v_kbar (k odd; entry (k - 1) / 2): xx, yy, zz, xy, xz, yz
__device__ __forceinline__ void second_moment(const Two (&s)[9], Two (&S)[6], Two& XY, Two& XZ, Two& YZ)
{
    XY = s[3] + s[4];
    XZ = s[5] + s[6];
    YZ = s[7] + s[8];
    S[0] = (s[0] + XY) + XZ;
    S[1] = (s[1] + XY) + YZ;
    S[2] = (s[2] + XZ) + YZ;
    S[3] = s[3] - s[4];
    S[4] = s[5] - s[6];
    S[5] = s[7] - s[8];
}

// the tensor in FP64, operation by operation
template <class S>
__device__ __noinline__ void node_pressure_f64(const FieldArgs& F, const S* __restrict__ f, const Scratch& W, int x, int y,
                                               int z, double* P)
{
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    for (int c = 0; c < 6; ++c) P[c] = 0.0;
    const long long off = F.L.off(x, y, z);
    const long long i = (long long)x + (long long)nx * (y + (long long)ny * z);
    float uf[3];
    node_velocity(F, W, x, y, z, (unsigned)i, uf);
    const double u[3] = {uf[0], uf[1], uf[2]};
    for (int a = 0; a < 2; ++a)
        for (int k = 0; k < Q; ++k) {
            const double n = decode<S>(f + F.L.at(a, k, off), k, F.P.ref[a]);
            const double d[3] = {cx(k) - u[0], cy(k) - u[1], cz(k) - u[2]};
            P[0] += d[0] * d[0] * n;
            P[1] += d[1] * d[1] * n;
            P[2] += d[2] * d[2] * n;
            P[3] += d[0] * d[1] * n;
            P[4] += d[0] * d[2] * n;
            P[5] += d[1] * d[2] * n;
        }
    const double pr = W.psi[0][i], pb = W.psi[1][i];
    double I[6] = {0, 0, 0, 0, 0, 0};
    for (int k = 1; k < Q; ++k) {
        const long long ip = (long long)wrapi(x + cx(k), nx) + (long long)nx * (wrapi(y + cy(k), ny) + (long long)ny * wrapi(z + cz(k), nz));
        const double G = is_axis(k) ? F.P.Gax : F.P.Gdi;
        const double pair = G * (pr * (double)W.psi[1][ip] + pb * (double)W.psi[0][ip]);
        const double c3[3] = {(double)cx(k), (double)cy(k), (double)cz(k)};
        I[0] += pair * c3[0] * c3[0];
        I[1] += pair * c3[1] * c3[1];
        I[2] += pair * c3[2] * c3[2];
        I[3] += pair * c3[0] * c3[1];
        I[4] += pair * c3[0] * c3[2];
        I[5] += pair * c3[1] * c3[2];
    }
    const double h = 0.5 * (double)F.P.gk;
    for (int c = 0; c < 6; ++c) P[c] += h * I[c];
}

// the tensor at the fluid node (x, y, z), normalised; false where a component
// is not finite (the caller then takes node_pressure_f64)
template <class S>
__device__ __forceinline__ bool node_pressure(const FieldArgs& F, const S* __restrict__ f, const Scratch& W, int x, int y,
                                              int z, Two (&P)[6])
{
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    const long long off = F.L.off(x, y, z);
    const int i = x + nx * (y + ny * z);
    float u[3];
    node_velocity(F, W, x, y, z, (unsigned)i, u);
    const float ref[2] = {F.P.ref[0], F.P.ref[1]};
    Two XY, XZ, YZ;
    {
        Two s[9], d[9];
        auto m = [&](int k) {
            float n0, n1;
            decode2<S>(f + F.L.at(0, k, off), k, ref, n0, n1);
            return two_sum(n0, n1);
        };
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const Two a = m(2 * p + 1), b = m(2 * p + 2);
            s[p] = a + b;
            d[p] = a - b;
        }
        second_moment(s, P, XY, XZ, YZ);
        const Two R = norm2(((m(0) + s[0]) + (s[1] + s[2])) + ((XY + XZ) + YZ));
        // pairs 3.. are (1,1,0), (1,-1,0), (1,0,1), (1,0,-1), (0,1,1), (0,1,-1)
        const Two J[3] = {norm2((d[0] + (d[3] + d[4])) + (d[5] + d[6])), norm2((d[1] + (d[3] - d[4])) + (d[7] + d[8])),
                          norm2((d[2] + (d[5] - d[6])) + (d[7] - d[8]))};
        Two K[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) K[q] = norm2(J[q] - mul2f(R, u[q]));
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const int a = c < 3 ? c : (c < 5 ? 0 : 1), b = c < 3 ? c : (c == 3 ? 1 : 2);
            P[c] = P[c] - (mul2f(K[b], u[a]) + mul2f(J[a], u[b]));
        }
    }
    const int xo[3] = {wrapi(x - 1, nx), x, wrapi(x + 1, nx)};
    const int yo[3] = {nx * wrapi(y - 1, ny), nx * y, nx * wrapi(y + 1, ny)};
    const int zo[3] = {nx * ny * wrapi(z - 1, nz), nx * ny * z, nx * ny * wrapi(z + 1, nz)};
    const float h = 0.5f * F.P.gk;  // exact
    Two I[6];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        Two s[9], T[6];
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            const int k = 2 * p + 1;
            const float v0 = W.psi[1 - a][xo[cx(k) + 1] + yo[cy(k) + 1] + zo[cz(k) + 1]];
            const float v1 = W.psi[1 - a][xo[1 - cx(k)] + yo[1 - cy(k)] + zo[1 - cz(k)]];
            const float G = p < 3 ? F.P.Gax : F.P.Gdi;  // 1 or 2: exact
            s[p] = two_sum(__fmul_rn(G, v0), __fmul_rn(G, v1));
        }
        second_moment(s, T, XY, XZ, YZ);
        const float own = W.psi[a][i];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const Two t = mul2f(norm2(T[c]), own);
            I[c] = a ? I[c] + t : t;
        }
    }
    bool finite = true;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        P[c] = norm2(P[c] + mul2f(norm2(I[c]), h));
        finite = finite && isfinite(P[c].h) && isfinite(P[c].l);
    }
    return finite;
}

// every node: P[c*N + i] (FP64)
template <class S>
__global__ void __launch_bounds__(kPressThreads) pressure_field_kernel(FieldArgs F, const S* __restrict__ f, Scratch W,
                                                                       double* __restrict__ out)
{
    const unsigned nx = (unsigned)F.L.nx, nxy = nx * (unsigned)F.L.ny, N = nxy * (unsigned)F.L.nz;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int z = (int)(i / nxy), y = (int)((i - z * nxy) / nx), x = (int)(i - z * nxy - y * nx);
        double D[6] = {0, 0, 0, 0, 0, 0};
        if (!node_solid(F, x, y, z, F.L.off(x, y, z))) {
            Two P[6];
            if (node_pressure<S>(F, f, W, x, y, z, P)) {
                for (int c = 0; c < 6; ++c) D[c] = to_f64(P[c]);
            } else {
                node_pressure_f64<S>(F, f, W, x, y, z, D);
            }
        }
        for (int c = 0; c < 6; ++c) out[(size_t)c * N + i] = D[c];
    }
}

// Sums over the fluid nodes of a plane (blockIdx.x) and a range of its nodes
// (one of `split` equal ones, blockIdx.y) of the six components, phi = rho_r -
// rho_b and the count -> out[(z * split + range) * 8 + v]. A thread sums its
// nodes in FP32 pairs (as node_pressure), then FP64 across threads.
// Bound by the pairs' arithmetic (2180 instructions a node at half the issue rate, five blocks an SM): 110 us at 96^3; the
// sums in FP64, one block a plane, took 1480.
template <class S>
__global__ void __launch_bounds__(kPressThreads, 5) pressure_plane_kernel(FieldArgs F, const S* __restrict__ f, Scratch W,
                                                                       int split, double* __restrict__ out)
{
    const int nx = F.L.nx, nxy = nx * F.L.ny, z = blockIdx.x;
    const int lo = (int)((long long)blockIdx.y * nxy / split), hi = (int)((long long)(blockIdx.y + 1) * nxy / split);
    Two sum[7];
    for (int v = 0; v < 7; ++v) sum[v] = two(0.f);
    double odd[6] = {0, 0, 0, 0, 0, 0};  // nodes taken in FP64
    int count = 0;
    for (int c = lo + threadIdx.x; c < hi; c += kPressThreads) {
        const int y = c / nx, x = c - y * nx;
        if (node_solid(F, x, y, z, F.L.off(x, y, z))) continue;
        const int i = c + nxy * z;
        Two P[6];
        if (node_pressure<S>(F, f, W, x, y, z, P)) {
#pragma unroll
            for (int v = 0; v < 6; ++v) sum[v] = norm2(sum[v] + P[v]);
        } else {
            double D[6];
            node_pressure_f64<S>(F, f, W, x, y, z, D);
            for (int v = 0; v < 6; ++v) odd[v] += D[v];
        }
        sum[6] = norm2(sum[6] + two_sum(W.rho[0][i], -W.rho[1][i]));
        ++count;
    }
    double acc[8];
#pragma unroll
    for (int v = 0; v < 7; ++v) acc[v] = to_f64(sum[v]) + (v < 6 ? odd[v] : 0.0);
    acc[7] = (double)count;
    __shared__ double sh[kPressThreads / 32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const double t = warp_sum(acc[v]);
        if (lane == 0) sh[warp][v] = t;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        double t = 0;
        for (int w = 0; w < kPressThreads / 32; ++w) t += sh[w][threadIdx.x];
        out[((size_t)z * split + blockIdx.y) * 8 + threadIdx.x] = t;
    }
}

// out[z*8 + v] = the sum of plane z's `split` rows, in order
__global__ void plane_rows_kernel(const double* __restrict__ part, int nz, int split, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nz * 8) return;
    double t = 0;
    for (int r = 0; r < split; ++r) t += part[((size_t)(i / 8) * split + r) * 8 + i % 8];
    out[i] = t;
}

// Radial bins about a centre: per fluid node with z >= zmin at distance
// r > 0 (minimum image along x, y, and z for the mask-driven periodic
// geometry), bin floor(r/dr) < nbins collects P_N = n.P.n,
// P_T = (tr P - P_N)/2, phi and 1. Sums are kept in 64-bit fixed point
// (units of 2^-30) so that the atomic accumulation is exact and the result
// does not depend on the order the nodes are added in.
// The bin comes from an FP32 root of the FP64 r^2; only where that lies within
// its rounding of a bin's edge is it taken from the FP64 root and quotient. A
// block gathers its nodes' sums in shared memory as 32-bit words (the low 16
// and the high bits of a value apart: 64-bit adds in shared memory are loops)
// and adds them to the global bins at its end; a value too large for that
// goes to the global bins at once.
// As the plane sums, plus about 30 FP64 operations a node for the radius and the split into words: 155 us at 96^3, 1230 with
// the tensor, three divisions and 64-bit shared-memory adds in FP64.
constexpr int kRadialNodes = 32000;  // most nodes a block takes: its 32-bit sums cannot overflow (below 2^15 nodes of 2^16)

template <class S>
__global__ void __launch_bounds__(kPressThreads, 5) pressure_radial_kernel(FieldArgs F, const S* __restrict__ f, Scratch W,
                                                                        double cxx, double cyy, double czz, double dr,
                                                                        int nbins, double zmin, unsigned per,
                                                                        unsigned long long* __restrict__ out)
{
    extern __shared__ unsigned radial_sh[];  // [nbins][7]: low and high words of the three sums, count
    for (int b = threadIdx.x; b < nbins * 7; b += kPressThreads) radial_sh[b] = 0u;
    __syncthreads();
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    const unsigned nxy = (unsigned)nx * (unsigned)ny, N = nxy * (unsigned)nz;
    const unsigned lo = blockIdx.x * per, hi = N - lo < per ? N : lo + per;
    const float idr = (float)(1.0 / dr);
    const bool plain_dr = dr > 1e-6 && dr < 1e6;
    for (unsigned i = lo + threadIdx.x; i < hi; i += kPressThreads) {
        const int z = (int)(i / nxy), y = (int)((i - z * nxy) / (unsigned)nx), x = (int)(i - z * nxy - y * nx);
        if (z < zmin) continue;
        double d[3] = {x - cxx, y - cyy, z - czz};
        // v - n rint(v / n): rint is 0 up to |v| = n / 2 (a tie goes to even), where no quotient is needed
        auto image = [](double v, int n) { return 2 * fabs(v) <= (double)n ? v : v - n * rint(v / n); };
        d[0] = image(d[0], nx);
        d[1] = image(d[1], ny);
        if (F.general) d[2] = image(d[2], nz);
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        if (!(r2 > 0)) continue;
        const float q = sqrtf((float)r2) * idr;  // r / dr within 3e-7 of itself for the moderate r2 and dr that `fast` asks for
        const bool fast = plain_dr && r2 > 1e-12 && r2 < 1e12;
        float bf = floorf(q);
        if (!fast || fabsf(q - rintf(q)) <= 1e-6f * q) {
            const double be = floor(sqrt(r2) / dr);
            if (be >= nbins) continue;
            bf = (float)be;
        }
        if (!(bf < (float)nbins)) continue;
        if (node_solid(F, x, y, z, F.L.off(x, y, z))) continue;
        Two P[6];
        long long v[3];
        const double phi = (double)W.rho[0][i] - (double)W.rho[1][i];
        if (node_pressure<S>(F, f, W, x, y, z, P)) {
            // n.P.n = d.P.d / r^2 in FP32 pairs: d_i as a pair, products of pairs
            Two e[3];
#pragma unroll
            for (int q3 = 0; q3 < 3; ++q3) {
                e[q3].h = (float)d[q3];
                e[q3].l = (float)(d[q3] - (double)e[q3].h);
            }
            const Two off = (norm2(mul22(P[3], norm2(mul22(e[0], e[1])))) + mul22(P[4], norm2(mul22(e[0], e[2])))) +
                            mul22(P[5], norm2(mul22(e[1], e[2])));
            const Two dia = (mul22(P[0], norm2(mul22(e[0], e[0]))) + mul22(P[1], norm2(mul22(e[1], e[1])))) +
                            mul22(P[2], norm2(mul22(e[2], e[2])));
            const double num = to_f64(dia + (off + off));
            const double pn = num / r2;
            const double tr = to_f64((P[0] + P[1]) + P[2]);
            v[0] = __double2ll_rn(pn * kRadialFix);
            v[1] = __double2ll_rn(0.5 * (tr - pn) * kRadialFix);
        } else {
            double D[6];
            node_pressure_f64<S>(F, f, W, x, y, z, D);
            const double r = sqrt(r2);
            const double n[3] = {d[0] / r, d[1] / r, d[2] / r};
            const double T[3][3] = {{D[0], D[3], D[4]}, {D[3], D[1], D[5]}, {D[4], D[5], D[2]}};
            double pn = 0;
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b) pn += n[a] * T[a][b] * n[b];
            v[0] = __double2ll_rn(pn * kRadialFix);
            v[1] = __double2ll_rn(0.5 * (D[0] + D[1] + D[2] - pn) * kRadialFix);
        }
        v[2] = __double2ll_rn(phi * kRadialFix);
        const int b = (int)bf;
        atomicAdd(&radial_sh[b * 7 + 6], 1u);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long top = v[c] >> 16;
            if (top >= -(1ll << 16) && top < (1ll << 16)) {
                atomicAdd(&radial_sh[b * 7 + 2 * c], (unsigned)(v[c] & 0xFFFF));
                atomicAdd(&radial_sh[b * 7 + 2 * c + 1], (unsigned)(int)top);
            } else {
                atomicAdd(&out[b * 4 + c], (unsigned long long)v[c]);
            }
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nbins * 4; t += kPressThreads) {
        const int b = t >> 2, c = t & 3;
        if (radial_sh[b * 7 + 6] == 0u) continue;
        const unsigned long long s = c == 3 ? (unsigned long long)radial_sh[b * 7 + 6]
                                            : (unsigned long long)((long long)radial_sh[b * 7 + 2 * c] +
                                                                   ((long long)(int)radial_sh[b * 7 + 2 * c + 1] << 16));
        if (s) atomicAdd(&out[t], s);
    }
}

// ---------------------------------------------------------------- population copies
template <class S>
__global__ void get_pop_kernel(FieldArgs F, const S* __restrict__ f, double* __restrict__ out)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N * 2 * Q; i += (long long)gridDim.x * blockDim.x) {
        const int ak = (int)(i / N);
        const long long n = i % N;
        const int a = ak / Q, k = ak % Q;
        const int x = (int)(n % F.L.nx), y = (int)((n / F.L.nx) % F.L.ny), z = (int)(n / ((long long)F.L.nx * F.L.ny));
        const long long off = F.L.off(x, y, z);
        out[i] = decode<S>(f + F.L.at(a, k, off), k, F.P.ref[a]);
    }
}

template <class S>
__global__ void set_pop_kernel(FieldArgs F, S* __restrict__ f, const double* __restrict__ in)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N * 2 * Q; i += (long long)gridDim.x * blockDim.x) {
        const int ak = (int)(i / N);
        const long long n = i % N;
        const int a = ak / Q, k = ak % Q;
        const int x = (int)(n % F.L.nx), y = (int)((n / F.L.nx) % F.L.ny), z = (int)(n / ((long long)F.L.nx * F.L.ny));
        const long long off = F.L.off(x, y, z);
        float v = (float)in[i];
        if constexpr (Codec<S>::kDeviation) v = (float)(in[i] / (double)zeta(k) - (double)F.P.ref[a]);
        put<S>(f + F.L.at(a, k, 0), F.L, x, y, (long long)z * F.L.plane, v);
    }
}

// ---------------------------------------------------------------- launchers

__global__ void clock_set_kernel(uint32_t* clk, uint32_t v)
{
    clk[0] = v;
    clk[1] = 0;
}

cudaError_t launch_clock_set(uint32_t* clk, uint32_t v, cudaStream_t st)
{
    clock_set_kernel<<<1, 1, 0, st>>>(clk, v);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_init(const FieldArgs& F, S* f, const double* rr, const double* rb, cudaStream_t st, int* err)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    init_kernel<S><<<grid_for(N, 256, 65536), 256, 0, st>>>(F, f, rr, rb, err);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_conservation(const FieldArgs& F, const S* f, unsigned long long* acc, unsigned int* ticket,
                                double* out, cudaStream_t st, float* phi)
{
    // one wave of resident blocks (a grid-stride loop over the nodes): a partial
    // last wave of a fixed grid left most SMs idle at the end
    static int blocks = 0;
    if (!blocks) {
        int dev = 0, nsm = 0, occ = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) ==
                                                      cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, cons_kernel<S>, kRedThreads, 0) == cudaSuccess &&
            nsm * occ > 0)
            blocks = nsm * occ < kConsBlocks ? nsm * occ : kConsBlocks;
        else
            blocks = kConsBlocks;
    }
    cons_kernel<S><<<blocks, kRedThreads, 0, st>>>(F, f, acc, ticket, out, phi);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_fields(const FieldArgs& F, const S* f, const Scratch& W, bool velocity, cudaStream_t st)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    fields_kernel<S><<<grid_for(N, 256, 65536), 256, 0, st>>>(F, f, W);
    if (velocity) velocity_kernel<<<grid_for(N, 256, 65536), 256, 0, st>>>(F, W);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_phi(const FieldArgs& F, const S* f, const Scratch& W, cudaStream_t st)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    phi_kernel<S><<<grid_for(N, 256, 65536), 256, 0, st>>>(F, f, W);
    return cudaGetLastError();
}

cudaError_t launch_angle(const FieldArgs& F, const Scratch& W, double zref, double level, double* part, double* out,
                         cudaStream_t st)
{
    angle_kernel<<<kAngleBlocks, kRedThreads, 0, st>>>(F, W, zref, level, part);
    finish_rows_kernel<kAngleVals><<<kAngleVals, 256, 0, st>>>(part, kAngleBlocks, kAngleMaxMask, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_get_pop(const FieldArgs& F, const S* f, double* out, cudaStream_t st)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz * 2 * Q;
    get_pop_kernel<S><<<grid_for(N, 256, 65536), 256, 0, st>>>(F, f, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_set_pop(const FieldArgs& F, S* f, const double* in, cudaStream_t st)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz * 2 * Q;
    set_pop_kernel<S><<<grid_for(N, 256, 65536), 256, 0, st>>>(F, f, in);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_pressure_field(const FieldArgs& F, const S* f, const Scratch& W, double* out, cudaStream_t st)
{
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    pressure_field_kernel<S><<<grid_for(N, kPressThreads, 65536), kPressThreads, 0, st>>>(F, f, W, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_pressure_planes(const FieldArgs& F, const S* f, const Scratch& W, int split, double* part, double* out,
                                   cudaStream_t st)
{
    pressure_plane_kernel<S><<<dim3(F.L.nz, split), kPressThreads, 0, st>>>(F, f, W, split, part);
    plane_rows_kernel<<<(F.L.nz * 8 + 127) / 128, 128, 0, st>>>(part, F.L.nz, split, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_pressure_radial(const FieldArgs& F, const S* f, const Scratch& W, const double* centre, double dr,
                                   int nbins, double zmin, unsigned long long* out, cudaStream_t st)
{
    if (nbins < 1 || nbins > kRadialBinsMax) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long) * 4 * nbins, st);
    if (e != cudaSuccess) return e;
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    long long per = (N + kRadialBlocks - 1) / kRadialBlocks;
    per = per < kPressThreads ? kPressThreads : (per > kRadialNodes ? kRadialNodes : per);
    pressure_radial_kernel<S><<<(unsigned)((N + per - 1) / per), kPressThreads, (size_t)nbins * 7 * sizeof(unsigned), st>>>(
        F, f, W, centre[0], centre[1], centre[2], dr, nbins, zmin, (unsigned)per, out);
    return cudaGetLastError();
}

#define LBSC_INST(S)                                                                                  \
    template cudaError_t launch_init<S>(const FieldArgs&, S*, const double*, const double*, cudaStream_t, int*); \
    template cudaError_t launch_conservation<S>(const FieldArgs&, const S*, unsigned long long*, unsigned int*, \
                                                double*, cudaStream_t, float*);                                \
    template cudaError_t launch_fields<S>(const FieldArgs&, const S*, const Scratch&, bool, cudaStream_t); \
    template cudaError_t launch_phi<S>(const FieldArgs&, const S*, const Scratch&, cudaStream_t);      \
    template cudaError_t launch_get_pop<S>(const FieldArgs&, const S*, double*, cudaStream_t);       \
    template cudaError_t launch_set_pop<S>(const FieldArgs&, S*, const double*, cudaStream_t);   \
    template cudaError_t launch_pressure_field<S>(const FieldArgs&, const S*, const Scratch&, double*, cudaStream_t); \
    template cudaError_t launch_pressure_planes<S>(const FieldArgs&, const S*, const Scratch&, int, double*, double*, \
                                                   cudaStream_t);                                     \
    template cudaError_t launch_pressure_radial<S>(const FieldArgs&, const S*, const Scratch&, const double*, double, int, \
                                                   double, unsigned long long*, cudaStream_t);
LBSC_INST(float)
LBSC_INST(__half)
LBSC_INST(__nv_bfloat16)

}  // namespace lbsc

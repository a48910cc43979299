// Non-step kernels: initial equilibrium, FP64 conservation sums, moment
// fields for readback, contact-angle reductions and population copies.
// All reductions are deterministic: the conservation sums are exact integer
// (fixed-point) sums; the others use a fixed grid, fixed per-thread ranges,
// warp shuffles and a final pass over the per-block partials in block order.
#include "lb_fields.cuh"

#include <cmath>
#include <type_traits>

namespace lbsc {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
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

// ---------------------------------------------------------------- pairs of FP32 numbers
// FP64 issues about once a clock and SM on this GPU, FP32 128 times. Sums that
// need more than FP32 are taken in pairs (Dekker 1971, Knuth's two-sum): a
// value is h + l with l far below h, a sum carries the rounding error of h in
// l. That keeps about 46 bits, 7 less than FP64; what they are formed from (psi, u, phi) is FP32. Against 64 bits
// from the same populations (27 lattices of edges 24-128 and one of 1024, three precisions) the pressure tensor, its
// profile, bins and tensions are off by as much as with FP64 (6.4e-8 of the tensor's largest entry, 1.5e-7 in a plane's
// mean), the contact angle by 1e-5 degrees at most and the fitted one by 8e-6, within 0.3% of FP64's error.
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
__device__ __forceinline__ Two two_int(int i)  // exact below 2^47
{
    const float h = (float)i;
    return Two{h, (float)((long long)i - (long long)h)};
}
// a / b, both normalised: one quotient and one correction
__device__ __forceinline__ Two div22(Two a, Two b)
{
    const float q = __fdiv_rn(a.h, b.h);
    const float r = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));
    return norm2(Two{q, __fdiv_rn(r, b.h)});
}
__device__ __forceinline__ bool less2(Two a, Two b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }  // normalised

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
// cons = {M_r, M_b, Px, Py, Pz, non-finite count, fluid nodes, the status word *err}
// A grid-stride walk over the nodes of the fluid planes, x fastest, so that a
// warp's load of one population slot covers consecutive addresses, with a
// node's 38 loads independent of each other. A node's mass and momentum are
// summed in FP32 over its 19 values per component, and each thread adds its
// nodes in FP32. The threads' sums then go into 64-bit integers in units of
// 2^-28 (kConsFix) and are added as integers: across warps, blocks and the
// whole grid, by shuffles and atomics. A node's values are tested one by one
// only where its sums are not finite (testing all 38 was a quarter of the
// instructions). Integer addition is exact and
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
                                                           float* __restrict__ phi, const int* __restrict__ err)
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
                s = __fadd_rn(s, nk);  // as the phi pass
                if (cx(k)) jn[0] += cx(k) * nk;
                if (cy(k)) jn[1] += cy(k) * nk;
                if (cz(k)) jn[2] += cz(k) * nk;
            }
            rho[a] = s;
        }
        if (phi) phi[i] = rho[0] - rho[1];
        if (!isfinite(rho[0]) || !isfinite(rho[1]))  // a value that is not finite makes its component's sum so
#pragma unroll
            for (int k = 0; k < Q; ++k) bad += (isfinite(v[0][k]) ? 0 : 1) + (isfinite(v[1][k]) ? 0 : 1);
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
        out[v] = v < 5 ? (double)t / kConsFix : (v == 7 ? (double)*err : (double)t);
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
// phi > level for the FP32 value p, exactly: A.least is the least FP32 number above the FP64 level
__device__ __forceinline__ bool above(float p, const AngleArgs& A) { return p >= A.least; }

// phi - level
__device__ __forceinline__ Two over(float p, const AngleArgs& A)
{
    const Two s = two_sum(p, -A.lh);
    return norm2(Two{s.h, __fsub_rn(s.l, A.ll)});
}

// Pairs serve where a difference of phi lies well inside FP32's range: not for
// infinities, NaN or values whose differences overflow, nor where the low part
// of a product would fall below the least FP32 number. Those nodes, rare, are
// taken in FP64 out of line.
__device__ __forceinline__ bool pairs_serve(float size) { return size > 1e-20f && size < 1e37f; }
__device__ __forceinline__ Two two_f64(double v)
{
    const float h = (float)v;
    return Two{h, isfinite(h) ? (float)(v - (double)h) : 0.f};
}

// plane_length in FP64
__device__ __noinline__ Two plane_length_f64(float p0, float p0up, float p1, float p1up, const AngleArgs& A)
{
    const double a0 = (1 - A.fz) * ((double)p0 - A.level) + A.fz * ((double)p0up - A.level);
    const double a1 = (1 - A.fz) * ((double)p1 - A.level) + A.fz * ((double)p1up - A.level);
    if (a0 > 0 && a1 > 0) return two(1.0f);
    if (a0 <= 0 && a1 <= 0) return two(0.0f);
    return two_f64(a0 > 0 ? a0 / (a0 - a1) : a1 / (a1 - a0));
}

// Positive length along x, from a node to its +x neighbour, of the linear
// interpolant of phi - level on the reference plane z0 + fz (p: phi at the
// node, above it, at the +x neighbour and above that).
__device__ __forceinline__ Two plane_length(float p0, float p0up, float p1, float p1up, const AngleArgs& A)
{
    const Two f{A.fzh, A.fzl}, g = norm2(two(1.0f) - f);
    const Two a0 = norm2(mul22(g, over(p0, A)) + mul22(f, over(p0up, A)));
    const Two a1 = norm2(mul22(g, over(p1, A)) + mul22(f, over(p1up, A)));
    if (!pairs_serve(fabsf(a0.h) + fabsf(a1.h))) return plane_length_f64(p0, p0up, p1, p1up, A);
    if (a0.h > 0 && a1.h > 0) return two(1.0f);
    if (a0.h <= 0 && a1.h <= 0) return two(0.0f);
    return a0.h > 0 ? div22(a0, norm2(a0 - a1)) : div22(a1, norm2(a1 - a0));
}

__device__ __forceinline__ void add_to(float2* acc, Two v)
{
    const float2 o = *acc;
    const Two s = norm2(Two{o.x, o.y} + v);
    *acc = make_float2(s.h, s.l);
}

// add_crossing in FP64; a crossing that is not a number goes into the sums
__device__ __noinline__ void add_crossing_f64(float2* acc, int stride, int x, int y, int z, int d, float p0, float p1,
                                              const AngleArgs& A)
{
    const double q0 = (double)p0 - A.level, q1 = (double)p1 - A.level, t = q0 / (q0 - q1);
    double p[3] = {x + t * (d == 0), y + t * (d == 1), z + t * (d == 2)};
    if (d == 2 && q0 > 0) {
        const float2 top = acc[0];
        const Two v = two_f64(z + t);
        if (less2(Two{top.x, top.y}, v)) acc[0] = make_float2(v.h, v.l);
    }
    if (p[2] < A.zref) return;
    for (int q = 0; q < 3; ++q) p[q] -= A.origin[q];
    const double rr = p[0] * p[0] + p[1] * p[1] + p[2] * p[2];
    const double v[14] = {1.0,         p[0] * p[0], p[0] * p[1], p[0] * p[2], p[0],      p[1] * p[1], p[1] * p[2],
                          p[1],        p[2] * p[2], p[2],        p[0] * rr,   p[1] * rr, p[2] * rr,   rr};
    for (int i = 0; i < 14; ++i) add_to(&acc[(i + 2) * stride], two_f64(v[i]));
}

// An interface crossing between node (x, y, z) (phi = p0) and its neighbour
// along axis d (phi = p1): the top crossing (along z, from phi > level
// below to phi <= level above) and the sphere-fit sums of the crossing point p at
// or above the reference plane, less A.origin, into the thread's accumulators acc[i * stride].
// Out of line: it is reached from a few places and rarely, and the row loop
// fits the instruction cache without it.
__device__ __noinline__ void add_crossing(float2* acc, int stride, int x, int y, int z, int d, float p0, float p1,
                                          const AngleArgs& A)
{
    const Two gap = norm2(two_sum(p0, -p1));
    if (!pairs_serve(fabsf(gap.h))) return add_crossing_f64(acc, stride, x, y, z, d, p0, p1, A);
    const Two t = div22(over(p0, A), gap);
    const Two zc = d == 2 ? norm2(two_int(z) + t) : two_int(z);
    if (d == 2 && above(p0, A)) {  // phi > level below, <= level above
        const float2 top = acc[0];
        if (less2(Two{top.x, top.y}, zc)) acc[0] = make_float2(zc.h, zc.l);
    }
    if (less2(zc, Two{A.zh, A.zl})) return;
    const Two c[3] = {two_int(x - A.origin[0]), two_int(y - A.origin[1]), two_int(z - A.origin[2])};
    Two p[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) p[q] = d == q ? norm2(c[q] + t) : c[q];
    auto add = [&](int i, Two v) { add_to(&acc[i * stride], v); };
    const Two xx = norm2(mul22(p[0], p[0])), yy = norm2(mul22(p[1], p[1])), zz = norm2(mul22(p[2], p[2]));
    const Two rr = norm2((xx + yy) + zz);
    add(2, two(1.0f));
    add(3, xx);
    add(4, mul22(p[0], p[1]));
    add(5, mul22(p[0], p[2]));
    add(6, p[0]);
    add(7, yy);
    add(8, mul22(p[1], p[2]));
    add(9, p[1]);
    add(10, zz);
    add(11, p[2]);
    add(12, mul22(p[0], rr));
    add(13, mul22(p[1], rr));
    add(14, mul22(p[2], rr));
    add(15, rr);
}

// One warp per lattice row, a lane per node, four nodes of the row in flight a
// lane, reading phi at the node and at its +y, +z neighbours (the latter from
// L1/L2; +x by shuffle):
//  [0]  (max) top phi = level crossing: z + p0/(p0 - p1) where phi > level
//       below and <= level above (both nodes fluid);
//  [1]  positive length along x of the reference-plane interpolant of phi
//       (the node at z0 adds its segment to x + 1, periodic);
//  [2..15] sums over crossings along +x, +y, +z at or above the reference
//       plane, of their points less A.origin: 1, xx, xy, xz, x, yy, yz, y, zz, z, x rr, y rr, z rr, rr (rr = |p|^2);
//  [16] (max) max of phi over fluid nodes, [17] (max) of -phi (the contrast).
// All in pairs of FP32 numbers: with FP64 sums (a drained queue took about 70
// FP64 operations, 2240 cycles of an SM's one FP64 lane) the kernel took 53 us
// at 128^3, bound by the SMs that met the most crossings. A block takes rows
// gridDim apart for the same reason: the drop's rows spread over all SMs. Now 28 us at 128^3 (9 million
// instructions, a third of them for crossings; phi is 8 MB, in L2).
// A thread's sums wait in shared memory, and a warp reduces a value only if one
// of its lanes holds a contribution to it. The last block to finish adds the
// blocks' rows, in order, and writes the 18 values lb_contact_angle works with.
__global__ void __launch_bounds__(kAngleThreads, 3) angle_kernel(FieldArgs F, AngleArgs A, const float* P,
                                                              float2* __restrict__ part, unsigned int* __restrict__ ticket,
                                                              double* __restrict__ out)
{
    constexpr int kWarps = kAngleThreads / 32, kStrips = 4;
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    __shared__ float2 sacc[16][kAngleThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = 0; i < 16; ++i) sacc[i][tid] = make_float2(i == 0 ? kNoTop : 0.f, 0.f);
    grid_wait();  // for the pass that wrote phi
    float pmax = -3.0e38f, pmin = 3.0e38f;
    const unsigned nxy = (unsigned)nx * (unsigned)ny;
    // Interface crossings are rare and scattered: a lane that meets one would
    // run the arithmetic of add_crossing alone, at the cost of a whole warp's.
    // So the warp queues its crossings in shared memory, in lane order, and
    // works through them 32 at a time with every lane busy; which lane sums
    // which crossing depends only on the data, so the sums are reproducible.
    // An entry: x and the row, each with a bit of the axis on top, and phi at
    // the node and at its neighbour.
    __shared__ int4 queue[kWarps][64];
    int queued = 0;
    auto drain = [&](int n) {  // lanes < n take a queued crossing each, then the queue shifts by n
        __syncwarp();
        if (lane < n) {
            const int4 q = queue[warp][lane];
            const int r = q.y & 0x7FFFFFFF, z = r / ny;
            add_crossing(&sacc[0][tid], kAngleThreads, q.x & 0x7FFFFFFF, r - z * ny, z,
                         (int)((unsigned)q.x >> 31) | (int)((unsigned)q.y >> 31) << 1, __int_as_float(q.z), __int_as_float(q.w), A);
        }
        __syncwarp();
        if (lane + n < queued) {  // at most 31 left, read from [n, queued), written to [0, queued - n)
            const int4 q = queue[warp][lane + n];
            queue[warp][lane] = q;
        }
        __syncwarp();
        queued -= n;
    };
    const int rows = ny * nz;
    for (int r = blockIdx.x + warp * gridDim.x; r < rows; r += kWarps * gridDim.x) {
        const int z = r / ny, y = r - z * ny;
        const float* R = P + (size_t)r * nx;
        const size_t up_y = y + 1 < ny ? nx : 0, up_z = z + 1 < nz ? nxy : 0;  // past an edge: the node itself
        // planar walls: the row is all fluid or all wall, and so is the one above it
        const bool wall = !F.general && (z == 0 || z == nz - 1);
        const bool wall_up = !F.general && z + 1 == nz - 1;
        for (int xb = 0; xb < nx; xb += 32 * kStrips) {  // warp-uniform: the queue needs the whole warp
            float p0[kStrips], py[kStrips], pz[kStrips];
#pragma unroll
            for (int s = 0; s < kStrips; ++s) {
                const int x = xb + 32 * s + lane;
                const float* q = R + (x < nx ? x : nx - 1);
                p0[s] = q[0];
                py[s] = q[up_y];
                pz[s] = q[up_z];
            }
            const int xe = xb + 32 * kStrips;
            const float pe = R[xe < nx ? xe : nx - 1];  // the node after the last strip
#pragma unroll
            for (int s = 0; s < kStrips; ++s) {
                const int xs = xb + 32 * s, x = xs + lane;
                if (xs >= nx) break;
                const unsigned in = nx - xs >= 32 ? ~0u : (1u << (nx - xs)) - 1u;  // lanes on the lattice
                if (z == A.z0 && z + 1 < nz && x < nx) {  // reference plane: every column, solid or not
                    const int x1 = x + 1 < nx ? x + 1 : 0;
                    const Two len = plane_length(p0[s], pz[s], R[x1], R[x1 + up_z], A);
                    const float2 o = sacc[1][tid];
                    const Two t = norm2(Two{o.x, o.y} + len);
                    sacc[1][tid] = make_float2(t.h, t.l);
                }
                unsigned fluid = wall ? 0u : in, ok_x = in, ok_y = in, ok_z = wall_up ? 0u : in;
                if (F.general) {
                    auto open = [&](int xx, int yy, int zz) {
                        return __ballot_sync(0xffffffffu, xx < nx && yy < ny && zz < nz &&
                                                              (F.nbmask[F.L.off(xx, yy, zz)] & kSelfSolid) == 0);
                    };
                    fluid = open(x, y, z);
                    ok_x = open(x + 1, y, z);
                    ok_y = open(x, y + 1, z);
                    ok_z = open(x, y, z + 1);
                }
                if ((fluid >> lane) & 1u) {
                    pmax = fmaxf(pmax, p0[s]);
                    pmin = fminf(pmin, p0[s]);
                }
                // the lanes above the level, and their +x, +y, +z neighbours above it (a neighbour past the
                // lattice's edge is the node itself: no crossing; along x the last node's bit is cleared)
                const unsigned b0 = __ballot_sync(0xffffffffu, above(p0[s], A));
                const float next = s + 1 < kStrips ? __shfl_sync(0xffffffffu, p0[s + 1], 0) : pe;
                const unsigned bx = b0 >> 1 | (above(next, A) ? 1u << 31 : 0u);
                const unsigned by = __ballot_sync(0xffffffffu, above(py[s], A));
                const unsigned bz = __ballot_sync(0xffffffffu, above(pz[s], A));
                const unsigned in_x = nx - 1 - xs >= 32 ? ~0u : (1u << (nx - 1 - xs)) - 1u;
                const unsigned m[3] = {(b0 ^ bx) & fluid & ok_x & in_x, (b0 ^ by) & fluid & ok_y, (b0 ^ bz) & fluid & ok_z};
                if ((m[0] | m[1] | m[2]) == 0u) continue;
                const float down = __shfl_down_sync(0xffffffffu, p0[s], 1);
                const float px = lane == 31 ? next : down;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    if (m[d] == 0u) continue;
                    if ((m[d] >> lane) & 1u) {
                        const int at = queued + __popc(m[d] & ((1u << lane) - 1u));
                        queue[warp][at] = make_int4(x | (d & 1) << 31, r | (d >> 1) << 31, __float_as_int(p0[s]),
                                                    __float_as_int(d == 0 ? px : (d == 1 ? py[s] : pz[s])));
                    }
                    queued += __popc(m[d]);
                    if (queued >= 32) drain(32);
                }
            }
        }
    }
    if (queued > 0) drain(queued);
    // block reduction: maxima by shuffles; warp w sums values w, w + kWarps, ... of all threads (each warp reducing its own
    // lanes' sums took as many instructions as the rows)
    __shared__ float lim[kWarps][2];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pmax = fmaxf(pmax, __shfl_down_sync(0xffffffffu, pmax, o));
        pmin = fminf(pmin, __shfl_down_sync(0xffffffffu, pmin, o));
    }
    if (lane == 0) {
        lim[warp][0] = pmax;
        lim[warp][1] = -pmin;
    }
    auto join = [](int v, Two a, Two b) {  // the maximum (v = 0, 16, 17) or the sum
        if (v != 0 && v < 16) return norm2(a + b);
        return less2(a, b) ? b : a;
    };
    __syncthreads();
    for (int v = warp; v < 16; v += kWarps) {
        Two val{sacc[v][lane].x, sacc[v][lane].y};
#pragma unroll
        for (int w = 1; w < kWarps; ++w) {
            const float2 o = sacc[v][32 * w + lane];
            val = join(v, val, Two{o.x, o.y});
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const Two w{__shfl_down_sync(0xffffffffu, val.h, o), __shfl_down_sync(0xffffffffu, val.l, o)};
            val = join(v, val, w);
        }
        if (lane == 0) part[(size_t)v * gridDim.x + blockIdx.x] = make_float2(val.h, val.l);
    }
    if (tid < 2) {
        float v = lim[0][tid];
        for (int w = 1; w < kWarps; ++w) v = fmaxf(v, lim[w][tid]);
        part[(size_t)(16 + tid) * gridDim.x + blockIdx.x] = make_float2(v, 0.f);
    }
    __threadfence();
    __shared__ bool last;
    __syncthreads();
    if (tid == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // all blocks' values: warp w takes values w, w + kWarps, ... together, a lane the blocks lane, lane + 32, ... in
    // order, eight of each in flight (one after the other this took as long as everything before it)
    constexpr int kMine = (kAngleRow + kWarps - 1) / kWarps;
    Two t[kMine];
#pragma unroll
    for (int i = 0; i < kMine; ++i) {
        const int v = warp + i * kWarps;
        t[i] = Two{v == 0 ? kNoTop : (v >= 16 ? -3.0e38f : 0.f), 0.f};
    }
    for (unsigned b0 = lane; b0 < gridDim.x; b0 += 32 * 8) {
        float2 q[kMine][8];
#pragma unroll
        for (int i = 0; i < kMine; ++i)
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (warp + i * kWarps < kAngleRow && b0 + 32 * u < gridDim.x)
                    q[i][u] = __ldcg(&part[(size_t)(warp + i * kWarps) * gridDim.x + b0 + 32 * u]);
#pragma unroll
        for (int i = 0; i < kMine; ++i)
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (warp + i * kWarps < kAngleRow && b0 + 32 * u < gridDim.x)
                    t[i] = join(warp + i * kWarps, t[i], Two{q[i][u].x, q[i][u].y});
    }
#pragma unroll
    for (int i = 0; i < kMine; ++i) {
        const int v = warp + i * kWarps;
        if (v >= kAngleRow) break;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const Two w{__shfl_down_sync(0xffffffffu, t[i].h, o), __shfl_down_sync(0xffffffffu, t[i].l, o)};
            t[i] = join(v, t[i], w);
        }
        if (lane == 0) out[v] = v == 0 && t[i].h == kNoTop ? -1e300 : (v >= 16 && t[i].h == -3.0e38f ? -1e300 : to_f64(t[i]));
    }
    if (tid == 0) *ticket = 0u;
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
// The sums run in pairs of FP32 numbers: about 46 bits over exact FP32 inputs,
// 20 more than the stored populations hold. With u common to both components the kinetic term is
//   S_ij - u_i K_j - u_j J_i,  S = sum c c m,  J = sum c m,  K = J - u R,
//   R = sum m,  m_k = n_k^r + n_k^b,
// and S, J need the sums and differences of opposite velocities only. A node
// whose result is not finite is taken again in FP64, so that infinities and
// NaN come out as they always did.
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

// values that a plane's sums may hold as FP32 pairs: sums of fewer than 2^31 stay below FP32's largest number
constexpr float kSumLimit = 1e28f;

// the tensor at the fluid node (x, y, z), normalised; false where a component
// is not finite or too large for the sums (the caller then takes node_pressure_f64)
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
        finite = finite && fabsf(P[c].h) < kSumLimit;
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
// nodes in FP32 pairs (as node_pressure), as do the threads of a warp; then FP64 across warps.
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
    // sums of the nodes taken in FP64, per thread: rare, so not in registers
    __shared__ double odd[7][kPressThreads];
    for (int v = 0; v < 7; ++v) odd[v][threadIdx.x] = 0.0;
    int count = 0;
    bool odd_nodes = false;
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
            for (int v = 0; v < 6; ++v) odd[v][threadIdx.x] += D[v];
            odd_nodes = true;
        }
        const Two phi = two_sum(W.rho[0][i], -W.rho[1][i]);
        if (fabsf(phi.h) < kSumLimit) {
            sum[6] = norm2(sum[6] + phi);
        } else {
            odd[6][threadIdx.x] += (double)W.rho[0][i] - (double)W.rho[1][i];
            odd_nodes = true;
        }
        ++count;
    }
    __shared__ float2 sh[kPressThreads / 32][7];
    __shared__ double sodd[kPressThreads / 32][7];
    __shared__ int sn[kPressThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < 7; ++v) {
        Two t = sum[v];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const Two w{__shfl_down_sync(0xffffffffu, t.h, o), __shfl_down_sync(0xffffffffu, t.l, o)};
            t = norm2(t + w);
        }
        if (lane == 0) sh[warp][v] = make_float2(t.h, t.l);
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0) sn[warp] = count;
    const bool any_odd = __syncthreads_or(odd_nodes);
    if (any_odd) {  // uniform
        for (int v = 0; v < 7; ++v) {
            const double t = warp_sum(odd[v][threadIdx.x]);
            if (lane == 0) sodd[warp][v] = t;
        }
        __syncthreads();
    }
    if (threadIdx.x < 8) {
        const int v = threadIdx.x;
        double t = 0;
        for (int w = 0; w < kPressThreads / 32; ++w) {
            if (v < 7) t += (double)sh[w][v].x + (double)sh[w][v].y;
            else t += (double)sn[w];
            if (any_odd && v < 7) t += sodd[w][v];
        }
        out[((size_t)z * split + blockIdx.y) * 8 + v] = t;
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
// Offsets, r^2, P_N and the fixed-point values are formed in FP32 pairs too (65
// FP64 operations a node were what bounded the pass), the bin from an FP32 root;
// only where that lies within its rounding of a bin's edge, a periodic offset near
// half the box, a value out of range or not finite, is the node taken in FP64. A
// block gathers its nodes' sums in shared memory as 32-bit words (the low 16
// and the high bits of a value apart: 64-bit adds in shared memory are loops)
// and adds them to the global bins at its end; a value too large for that
// goes to the global bins at once.
// 96^3 (the call with the moment fields and the readback): 1.3 ms with the tensor, three divisions and 64-bit shared-memory
// adds in FP64, 214 us with the tensor in pairs alone, 153 now; six blocks an SM (with five 7% longer).
// round(v 2^30) of a pair below 2^20
__device__ __forceinline__ long long to_fix30(Two v)
{
    const float h = __fmul_rn(v.h, (float)kRadialFix), a = rintf(h);
    return __float2ll_rn(a) + (long long)__float2int_rn(__fmaf_rn(v.l, (float)kRadialFix, __fsub_rn(h, a)));
}

// The FP64 form of a node's values v[3] (P_N, P_T, phi in units of 2^-30) and
// bin: false where it falls in none.
template <class S>
__device__ __noinline__ bool radial_node_f64(const FieldArgs& F, const S* __restrict__ f, const Scratch& W,
                                             const RadialArgs& R, int x, int y, int z, long long* v, int* bin)
{
    double d[3] = {x - R.c[0], y - R.c[1], z - R.c[2]};
    d[0] -= F.L.nx * rint(d[0] / F.L.nx);
    d[1] -= F.L.ny * rint(d[1] / F.L.ny);
    if (F.general) d[2] -= F.L.nz * rint(d[2] / F.L.nz);
    const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    if (!(r > 0)) return false;
    const double bf = floor(r / R.dr);
    if (!(bf < R.nbins)) return false;
    double D[6];
    node_pressure_f64<S>(F, f, W, x, y, z, D);
    const double n[3] = {d[0] / r, d[1] / r, d[2] / r};
    const double T[3][3] = {{D[0], D[3], D[4]}, {D[3], D[1], D[5]}, {D[4], D[5], D[2]}};
    double pn = 0;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) pn += n[a] * T[a][b] * n[b];
    const size_t i = (size_t)x + (size_t)F.L.nx * (y + (size_t)F.L.ny * z);
    v[0] = __double2ll_rn(pn * kRadialFix);
    v[1] = __double2ll_rn(0.5 * (D[0] + D[1] + D[2] - pn) * kRadialFix);
    v[2] = __double2ll_rn(((double)W.rho[0][i] - (double)W.rho[1][i]) * kRadialFix);
    *bin = (int)bf;
    return true;
}

constexpr int kRadialNodes = 32000;  // most nodes a block takes: its 32-bit sums cannot overflow (below 2^15 nodes of 2^16)

template <class S>
__global__ void __launch_bounds__(kPressThreads, 6) pressure_radial_kernel(FieldArgs F, const S* __restrict__ f, Scratch W,
                                                                           RadialArgs R, unsigned per,
                                                                           unsigned long long* __restrict__ out)
{
    extern __shared__ unsigned radial_sh[];  // [nbins][7]: low and high words of the three sums, count
    const int nbins = R.nbins;
    for (int b = threadIdx.x; b < nbins * 7; b += kPressThreads) radial_sh[b] = 0u;
    __syncthreads();
    const int nx = F.L.nx, ny = F.L.ny, nz = F.L.nz;
    const unsigned nxy = (unsigned)nx * (unsigned)ny, N = nxy * (unsigned)nz;
    const unsigned lo = blockIdx.x * per, hi = N - lo < per ? N : lo + per;
    for (unsigned i = lo + threadIdx.x; i < hi; i += kPressThreads) {
        const int z = (int)(i / nxy), y = (int)((i - z * nxy) / (unsigned)nx), x = (int)(i - z * nxy - y * nx);
        if (z < R.z0) continue;
        // offset from the centre, the nearest image along a periodic axis
        bool plain = R.plain;
        auto offset = [&](int at, int q, int n, bool periodic) {
            Two d = two_sum((float)at, -R.ch[q]);
            d.l = __fsub_rn(d.l, R.cl[q]);
            if (periodic) {
                // near half the box FP64 decides which image it is, but for the plain tie, which keeps its side
                const float half = 0.5f * (float)n;
                if (fabsf(d.h) == half && d.l == 0.f) return d;
                const float m = rintf(d.h / (float)n), rest = fabsf(d.h - m * (float)n);
                if (fabsf(rest - half) <= 1e-5f * half) plain = false;
                d = d + two(-m * (float)n);
            }
            return norm2(d);
        };
        const Two d[3] = {offset(x, 0, nx, true), offset(y, 1, ny, true), offset(z, 2, nz, F.general != 0)};
        const Two xx = norm2(mul22(d[0], d[0])), yy = norm2(mul22(d[1], d[1])), zz = norm2(mul22(d[2], d[2]));
        const Two r2 = norm2((xx + yy) + zz);
        const float q = sqrtf(r2.h) * R.idr;  // r / dr within 3e-7 of itself
        plain = plain && r2.h > 1e-6f && r2.h < 1e12f && fabsf(q - rintf(q)) > 1e-6f * q;
        if (plain && q >= (float)nbins) continue;
        if (node_solid(F, x, y, z, F.L.off(x, y, z))) continue;
        int b = (int)q;
        long long v[3];
        Two P[6];
        plain = plain && node_pressure<S>(F, f, W, x, y, z, P);
        if (plain) {
            // n.P.n = d.P.d / r^2
            const Two off = (norm2(mul22(P[3], norm2(mul22(d[0], d[1])))) + mul22(P[4], norm2(mul22(d[0], d[2])))) +
                            mul22(P[5], norm2(mul22(d[1], d[2])));
            const Two dia = (mul22(P[0], xx) + mul22(P[1], yy)) + mul22(P[2], zz);
            const Two pn = div22(norm2(dia + (off + off)), r2);
            const Two pt = norm2(((P[0] + P[1]) + P[2]) - pn);
            const Two phi = two_sum(W.rho[0][i], -W.rho[1][i]);
            plain = fabsf(pn.h) < 1e6f && fabsf(pt.h) < 1e6f && fabsf(phi.h) < 1e6f;
            v[0] = to_fix30(pn);
            v[1] = to_fix30(Two{0.5f * pt.h, 0.5f * pt.l});
            v[2] = to_fix30(phi);
        }
        if (!plain && !radial_node_f64<S>(F, f, W, R, x, y, z, v, &b)) continue;
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
                                double* out, const int* err, cudaStream_t st, float* phi)
{
    // one wave of resident blocks (a grid-stride loop over the nodes): a partial last wave of a fixed grid left most SMs
    // idle at the end. A thread adds its nodes in FP32, so the grid is part of the result: four blocks an SM for FP32,
    // five for 16-bit storage, whatever the registers of a build would admit
    static int blocks = 0;
    if (!blocks) {
        int dev = 0, nsm = 0;
        const int per = sizeof(S) == 4 ? 4 : 5;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && nsm > 0)
            blocks = nsm * per < kConsBlocks ? nsm * per : kConsBlocks;
        else
            blocks = kConsBlocks;
    }
    cons_kernel<S><<<blocks, kRedThreads, 0, st>>>(F, f, acc, ticket, out, phi, err);
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

cudaError_t launch_angle(const FieldArgs& F, const Scratch& W, double zref, double level, const int (&origin)[3],
                         double* part, unsigned int* ticket, double* out, cudaStream_t st)
{
    AngleArgs A;
    for (int q = 0; q < 3; ++q) A.origin[q] = origin[q];
    auto split = [](double v, float& h, float& l) {
        h = (float)v;
        l = (float)(v - (double)h);
    };
    split(level, A.lh, A.ll);
    A.least = level < (double)A.lh ? A.lh : std::nextafterf(A.lh, INFINITY);
    split(zref, A.zh, A.zl);
    const double z0 = std::floor(zref);
    split(zref - z0, A.fzh, A.fzl);
    A.level = level;
    A.zref = zref;
    A.fz = zref - z0;
    A.z0 = z0 < (double)F.L.nz ? (int)z0 : F.L.nz;
    const int rows = F.L.ny * F.L.nz, warps = kAngleThreads / 32;
    const int blocks = (rows + warps - 1) / warps < kAngleBlocks ? (rows + warps - 1) / warps : kAngleBlocks;
    return launch_after(angle_kernel, dim3(blocks), kAngleThreads, 0, st, F, A, W.rho[0], (float2*)part, ticket, out);
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
    RadialArgs R;
    bool near = true;
    for (int q = 0; q < 3; ++q) {
        R.c[q] = centre[q];
        R.ch[q] = (float)centre[q];
        R.cl[q] = (float)(centre[q] - (double)R.ch[q]);
        near = near && std::fabs(centre[q]) < 1e6;
    }
    R.dr = dr;
    R.idr = (float)(1.0 / dr);
    R.nbins = nbins;
    const double z0 = std::ceil(zmin);  // z < zmin is z < z0 for whole z
    R.z0 = z0 < 0 ? 0 : (z0 > F.L.nz ? F.L.nz : (int)z0);
    // the FP32 pairs hold whole coordinates below 2^24 exactly
    R.plain = near && dr > 1e-3 && dr < 1e6 && F.L.nx < (1 << 23) && F.L.ny < (1 << 23) && F.L.nz < (1 << 23);
    const long long N = (long long)F.L.nx * F.L.ny * F.L.nz;
    long long per = (N + kRadialBlocks - 1) / kRadialBlocks;
    per = per < kPressThreads ? kPressThreads : (per > kRadialNodes ? kRadialNodes : per);
    pressure_radial_kernel<S><<<(unsigned)((N + per - 1) / per), kPressThreads, (size_t)nbins * 7 * sizeof(unsigned), st>>>(
        F, f, W, R, (unsigned)per, out);
    return cudaGetLastError();
}

#define LBSC_INST(S)                                                                                  \
    template cudaError_t launch_init<S>(const FieldArgs&, S*, const double*, const double*, cudaStream_t, int*); \
    template cudaError_t launch_conservation<S>(const FieldArgs&, const S*, unsigned long long*, unsigned int*, \
                                                double*, const int*, cudaStream_t, float*);                    \
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

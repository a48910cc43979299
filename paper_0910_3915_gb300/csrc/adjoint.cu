// Discrete adjoint of the time step (Sec. 2) with respect to the wall
// pseudo-densities (eta_wall_r, eta_wall_b), for the planar-wall geometry.
//
// Forward step at a fluid node y, component a (omega = 1/tau):
//   rho^a = sum_k n_k, j^a = sum_k n_k c_k, psi^a = 1 - exp(-rho^a)
//   F^a   = -g kappa psi^a(y) S^a,  S^a = sum_m G_m psi~^abar(y + c_m) c_m
//           (psi~ = wall pseudo-density eta_abar where y + c_m is solid)
//   u'    = sum_b omega_b j^b / D,  D = sum_b omega_b rho^b
//   u^a   = u' + tau_a F^a / rho^a
//   q_k   = zeta_k rho^a (1 + P_k(u^a)),  n*_k = (1 - omega_a) n_k + omega_a q_k
//   stream: n_k(y + c_k, t+1) = n*_k(y), or n_kbar(y, t+1) = n*_k(y) into a wall
// The adjoint runs these in reverse for lambda = dJ/dn:
//   mu_k(y) = dJ/dn*_k(y) = lambda_k(y + c_k) or lambda_kbar(y) (wall)
//   then back through BGK, the equilibrium, the velocity shift, u', the force
//   and psi, ending in lambda_k(y, t) = (1 - omega) mu_k + rhobar + c_k . jbar.
// The force couples neighbours: node y sends Sbar^a = -g kappa psi^a(y) Fbar^a
// to psi^abar of its 18 neighbours (or to eta_abar where the neighbour is a
// wall); a second pass gathers those contributions.
//
// The adjoint of n_k(t) is kept as
//   lambda_k(t) = M_k + E_k,  M_k = (1 - omega) mu_k,  E_k = rhobar + c_k . jbar,
// so a reverse step writes E's 4 values per component (32 bytes a node)
// where writing and re-reading lambda itself took 3 passes over 38 values.
// At tau = 1 M vanishes and is neither stored nor read: lambda lives in E
// alone. All fields are dense, index x + nx*(y + ny*z), and hold both
// components of a node side by side (one 8-byte access for the two).
// Gradient sums are FP64.
#include "lb_fields.cuh"

namespace lbsc {

__device__ __forceinline__ int didx(int x, int y, int z, int nx, int ny) { return x + nx * (y + ny * z); }
__device__ __forceinline__ bool wall_z(int z, int nz) { return z == 0 || z == nz - 1; }
// coordinates of dense node index i (32-bit: node counts stay below 2^31)
__device__ __forceinline__ void node_xyz(int i, int nx, int ny, int& x, int& y, int& z)
{
    const int t = i / nx;
    x = i - t * nx;
    z = t / ny;
    y = t - z * ny;
}
__device__ __forceinline__ float lane(const float2& v, int a) { return a ? v.y : v.x; }
// s + c v for a velocity component c in {-1, 0, 1} known at compile time after unrolling
__device__ __forceinline__ float add_c(float s, int c, float v) { return c == 0 ? s : (c > 0 ? s + v : s - v); }

// Forward rho, j, psi of the stored state (lattice layout L), one thread per
// node, both components of a velocity in one load: a plain one, since the step
// that writes f may still run when this kernel starts. Bound by the read of the
// populations (152 bytes a node, from L2 when it follows the step that wrote
// them): 8.5 us at 64^3 FP32 (cold caches), 11.4 with a grid-stride grid of 512
// blocks and one component at a time.
template <class S>
__global__ void __launch_bounds__(kAdjThreads) adj_forward_kernel(Layout L, KParams P, const S* f, AdjState A)
{
    grid_trigger();
    const int N = L.nx * L.ny * L.nz;
    const int i = blockIdx.x * kAdjThreads + threadIdx.x;
    grid_wait();  // every thread of a dependent launch waits, so that the launch's end implies the earlier kernels'
    if (i >= N) return;
    int x, y, z;
    node_xyz(i, L.nx, L.ny, x, y, z);
    const bool solid = wall_z(z, L.nz);
    float2 w[Q];
    if (!solid) {
        const long long off = L.off(x, y, z);
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k] = Codec<S>::val2(*(const typename Codec<S>::Pair*)(f + L.at(0, k, off)));
    }
    float r[2], j[2][3], psi[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        float s = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
        if (!solid) {
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                float v = lane(w[k], a);
                if constexpr (Codec<S>::kDeviation) v = zeta(k) * (P.ref[a] + v);
                s += v;
                jx += cx(k) * v;
                jy += cy(k) * v;
                jz += cz(k) * v;
            }
        }
        r[a] = s;
        j[a][0] = jx;
        j[a][1] = jy;
        j[a][2] = jz;
        psi[a] = solid ? P.eta[a] : -expm1f(-s);
    }
    A.rho[i] = make_float2(r[0], r[1]);
    A.psi[i] = make_float2(psi[0], psi[1]);
#pragma unroll
    for (int d = 0; d < 3; ++d) A.j[d][i] = make_float2(j[0][d], j[1][d]);
}

// Pass A of a reverse step, one thread per fluid node: mu from lambda(t+1),
// the local adjoint of BGK, equilibrium, shift, u' and force. Writes jbar and
// (before the psi term) rhobar into E(t), M(t) where tau != 1, and V and psibar
// for pass B. The wall gradient of the block is added to its own row of
// part[block][2] (FP64), which one pass sums after the last step.
// Bound by the latency of its 68 loads of neighbours' E and psi (8 bytes, both components; L1/L2 hits) and about 1400
// instructions, 25 of them divisions: packed lanes for the two components were slower (20.6 against 20.3 ms for the
// gradient below), and so were 6 to 8 blocks an SM instead of 5.
// 25 us at 64^3; 75 when it read and wrote lambda's 38 values. The passes are launched dependently: a gradient over 300
// steps at 64^3 21.8 -> 20.3 ms. One thread summed
// the blocks' rows after every step before (32 us).
template <bool kTauOne>
__global__ void __launch_bounds__(kAdjThreads)
    adj_local_kernel(AdjArgs G, AdjState A, AdjE En, const float* Mn, AdjE Ec, float* Mc,
                     AdjV W, double* __restrict__ part)
{
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int N = nx * ny * nz;
    const int i = blockIdx.x * kAdjThreads + threadIdx.x;
    grid_trigger();
    double geta[2] = {0.0, 0.0};
    bool at_wall = false;
    int x = 0, y = 0, z = 0;
    if (i < N) node_xyz(i, nx, ny, x, y, z);
    grid_wait();
    if (i < N && !wall_z(z, nz)) {
        const int xo[3] = {wrapi(x - 1, nx), x, wrapi(x + 1, nx)};
        const int yo[3] = {wrapi(y - 1, ny), y, wrapi(y + 1, ny)};
        const bool zwall[3] = {wall_z(z - 1, nz), false, wall_z(z + 1, nz)};
        at_wall = zwall[0] || zwall[2];
        float rho[2], j[2][3], psi[2], S[2][3], F[2][3];
        {
            const float2 r2 = A.rho[i], p2 = A.psi[i];
            rho[0] = r2.x, rho[1] = r2.y, psi[0] = p2.x, psi[1] = p2.y;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float2 t = A.j[d][i];
                j[0][d] = t.x, j[1][d] = t.y;
            }
        }
        // S^a = sum_m G_m psi~^abar(y + c_m) c_m
#pragma unroll
        for (int a = 0; a < 2; ++a) S[a][0] = S[a][1] = S[a][2] = 0.f;
#pragma unroll
        for (int m = 1; m < Q; ++m) {
            const float2 pn = A.psi[didx(xo[cx(m) + 1], yo[cy(m) + 1], z + cz(m), nx, ny)];
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const float ps = G.G[m] * lane(pn, 1 - a);
                S[a][0] = add_c(S[a][0], cx(m), ps);
                S[a][1] = add_c(S[a][1], cy(m), ps);
                S[a][2] = add_c(S[a][2], cz(m), ps);
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int d = 0; d < 3; ++d) F[a][d] = -G.gk * psi[a] * S[a][d];
        const float D = G.omega[0] * rho[0] + G.omega[1] * rho[1];
        float up[3] = {0.f, 0.f, 0.f};
        if (D > 0.f)
#pragma unroll
            for (int d = 0; d < 3; ++d) up[d] = (G.omega[0] * j[0][d] + G.omega[1] * j[1][d]) / D;

        float rhob[2] = {0.f, 0.f}, ub[2][3], upb[3] = {0.f, 0.f, 0.f}, u[2][3], usq[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const bool shift = rho[a] > 1e-12f;
#pragma unroll
            for (int d = 0; d < 3; ++d) u[a][d] = up[d] + (shift ? G.tau[a] * F[a][d] / rho[a] : 0.f);
            usq[a] = u[a][0] * u[a][0] + u[a][1] * u[a][1] + u[a][2] * u[a][2];
            ub[a][0] = ub[a][1] = ub[a][2] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            // mu_k = lambda_k(y + c_k), or lambda_kbar(y) when y + c_k is a wall
            const bool wall = cz(k) != 0 && zwall[cz(k) + 1];
            const int n = wall ? i : didx(xo[cx(k) + 1], yo[cy(k) + 1], z + cz(k), nx, ny);
            float2 lam = En.rb[n];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int c = d == 0 ? cx(k) : (d == 1 ? cy(k) : cz(k));
                if (c == 0) continue;
                float2 e = En.j[d][n];
                if (cz(k) != 0 && wall) e = make_float2(-e.x, -e.y);  // c_kbar = -c_k
                lam.x = add_c(lam.x, c, e.x);
                lam.y = add_c(lam.y, c, e.y);
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                float mu = lane(lam, a);
                if constexpr (!kTauOne) {
                    mu += Mn[(long long)(a * Q + (wall ? opp(k) : k)) * N + n];
                    Mc[(long long)(a * Q + k) * N + i] = (1.0f - G.omega[a]) * mu;
                }
                const float qb = G.omega[a] * mu;
                // the zero products stay: without them the compiler shares terms between opposite
                // velocities and fuses others, which moves the gradient by 1e-8 of itself
                const float cu = cx(k) * u[a][0] + cy(k) * u[a][1] + cz(k) * u[a][2];
                const float P = 3.f * cu + 4.5f * cu * cu - 1.5f * usq[a] + 4.5f * cu * cu * cu - 4.5f * usq[a] * cu;
                rhob[a] += qb * zeta(k) * (1.0f + P);
                const float Ak = 3.f + 9.f * cu + 13.5f * cu * cu - 4.5f * usq[a], Bk = -3.f - 9.f * cu;
                const float w = qb * zeta(k) * rho[a];
                ub[a][0] += w * (cx(k) * Ak + u[a][0] * Bk);
                ub[a][1] += w * (cy(k) * Ak + u[a][1] * Bk);
                ub[a][2] += w * (cz(k) * Ak + u[a][2] * Bk);
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int d = 0; d < 3; ++d) upb[d] += ub[a][d];
        float Fb[2][3];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const bool shift = rho[a] > 1e-12f;
            float dot = 0.f;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                Fb[a][d] = shift ? ub[a][d] * G.tau[a] / rho[a] : 0.f;
                dot += ub[a][d] * F[a][d];
            }
            if (shift) rhob[a] -= dot * G.tau[a] / (rho[a] * rho[a]);
        }
        float jb[2][3];
        if (D > 0.f) {
            const float updot = upb[0] * up[0] + upb[1] * up[1] + upb[2] * up[2];
#pragma unroll
            for (int a = 0; a < 2; ++a) {
#pragma unroll
                for (int d = 0; d < 3; ++d) jb[a][d] = G.omega[a] * upb[d] / D;
                rhob[a] -= G.omega[a] * updot / D;
            }
        } else {
#pragma unroll
            for (int a = 0; a < 2; ++a) jb[a][0] = jb[a][1] = jb[a][2] = 0.f;
        }
        // force: psi^a(y) factor and the neighbour sum
        float V[2][3], psib[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            float sdot = 0.f;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                V[a][d] = -G.gk * psi[a] * Fb[a][d];
                sdot += Fb[a][d] * S[a][d];
            }
            psib[a] = -G.gk * sdot;
            // wall links of the neighbour sum feed d J / d eta_abar
            if (at_wall) {
#pragma unroll
                for (int m = 1; m < Q; ++m) {
                    if (cz(m) == 0 || !zwall[cz(m) + 1]) continue;
                    float t = 0.f;
                    t = add_c(t, cx(m), V[a][0]);
                    t = add_c(t, cy(m), V[a][1]);
                    t = add_c(t, cz(m), V[a][2]);
                    geta[1 - a] += (double)(G.G[m] * t);
                }
            }
        }
        Ec.rb[i] = make_float2(rhob[0], rhob[1]);
        W.psib[i] = make_float2(psib[0], psib[1]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            Ec.j[d][i] = make_float2(jb[0][d], jb[1][d]);
            W.v[d][i] = make_float2(V[0][d], V[1][d]);
        }
    }
    // block sum of the wall gradient, in blocks that hold a node next to a wall
    if (!__syncthreads_or(at_wall)) return;
    __shared__ double sh[kAdjThreads / 32][2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        double v = geta[a];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][a] = v;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double v = 0;
        for (int w = 0; w < kAdjThreads / 32; ++w) v += sh[w][threadIdx.x];
        part[blockIdx.x * 2 + threadIdx.x] += v;  // this block's row, step after step
    }
}

// Pass B: gather the neighbours' force adjoints into psibar, then finish
// E(t)'s rhobar with psibar psi'. A neighbour's V is read only along the
// nonzero entries of its link (30 loads of 8 bytes a node, L1/L2 hits).
// 7.8 us at 64^3; 83 when it loaded all of V and rewrote lambda's 38 values.
__global__ void __launch_bounds__(kAdjThreads) adj_gather_kernel(AdjArgs G, AdjState A, AdjV W, AdjE Ec)
{
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int N = nx * ny * nz;
    const int i = blockIdx.x * kAdjThreads + threadIdx.x;
    grid_trigger();
    int x, y, z;
    node_xyz(i < N ? i : 0, nx, ny, x, y, z);
    grid_wait();
    if (i >= N) return;
    if (wall_z(z, nz)) return;
    const int xo[3] = {wrapi(x - 1, nx), x, wrapi(x + 1, nx)};
    const int yo[3] = {wrapi(y - 1, ny), y, wrapi(y + 1, ny)};
    const bool zwall[3] = {wall_z(z - 1, nz), false, wall_z(z + 1, nz)};
    const float2 p2 = W.psib[i], r2 = A.rho[i], b2 = Ec.rb[i];
    float pb[2] = {p2.x, p2.y};
    // psi^a(x) is used by F^abar(x - c_m) for every fluid x - c_m
#pragma unroll
    for (int m = 1; m < Q; ++m) {
        if (cz(m) != 0 && zwall[1 - cz(m)]) continue;
        const int s = didx(xo[1 - cx(m)], yo[1 - cy(m)], z - cz(m), nx, ny);
        float2 t = make_float2(0.f, 0.f);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int c = d == 0 ? cx(m) : (d == 1 ? cy(m) : cz(m));
            if (c == 0) continue;
            const float2 v = W.v[d][s];
            t.x = add_c(t.x, c, v.x);
            t.y = add_c(t.y, c, v.y);
        }
        pb[0] += G.G[m] * t.y;
        pb[1] += G.G[m] * t.x;
    }
    float rb[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) rb[a] = lane(b2, a) + pb[a] * expf(-lane(r2, a));
    Ec.rb[i] = make_float2(rb[0], rb[1]);
}

// out[a] = sum over the blocks' rows of part: thread t rows t, t + 256, ... in
// order, a fixed shuffle tree per warp, then the warps in order (a = blockIdx.x)
__global__ void __launch_bounds__(256) rows_sum_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ out)
{
    const int a = blockIdx.x;
    double v = 0;
    for (int b = threadIdx.x; b < nblocks; b += 256) v += part[2 * b + a];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __shared__ double sh[8];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += sh[w];
        out[a] = t;
    }
}

// Observable J of the densities and its gradient lambda(T) = dJ/drho (FP64 sums).
// obs 0: centre-of-mass height of rho_r above the wall plane, sum (z - 1/2) rho_r / sum rho_r
// obs 1: the same with weight sigma(phi / eps), phi = rho_r - rho_b (the droplet, softly)
// obs 2: wetted area, sum over the first fluid layer of sigma(phi / eps)
__device__ __forceinline__ double sigmoid(double s) { return 1.0 / (1.0 + exp(-s)); }

__global__ void obs_sums_kernel(int nx, int ny, int nz, int obs, double eps, const float2* __restrict__ rho,
                                double* __restrict__ part)
{
    const long long N = (long long)nx * ny * nz;
    double s0 = 0, s1 = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const int z = (int)(i / ((long long)nx * ny));
        if (wall_z(z, nz)) continue;
        const double h = z - 0.5;
        if (obs == 0) {
            s0 += rho[i].x;
            s1 += h * rho[i].x;
        } else {
            const double w = sigmoid(((double)rho[i].x - (double)rho[i].y) / eps);
            if (obs == 1) {
                s0 += w;
                s1 += h * w;
            } else if (z == 1) {
                s0 += w;
            }
        }
    }
    __shared__ double sh[8][2];
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, o);
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[threadIdx.x >> 5][0] = s0;
        sh[threadIdx.x >> 5][1] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sh[w][threadIdx.x];
        part[blockIdx.x * 2 + threadIdx.x] = v;
    }
}

// J = s1/s0 (obs 0, 1) or s0 (obs 2) from the reduced sums[0..1], written to sums[2]
__global__ void obs_finish_kernel(int obs, double* __restrict__ sums)
{
    if (threadIdx.x == 0) sums[2] = obs == 2 ? sums[0] : sums[1] / sums[0];
}

// lambda(T) = dJ/dn(T) as E: the same for every velocity, so rhobar = dJ/drho and jbar = 0
__global__ void obs_grad_kernel(int nx, int ny, int nz, int obs, double eps, const float2* __restrict__ rho,
                                const double* __restrict__ sums, AdjE E)
{
    const long long N = (long long)nx * ny * nz;
    const double s0 = sums[0], J = sums[2];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
        const int z = (int)(i / ((long long)nx * ny));
        double gr = 0, gb = 0;
        if (!wall_z(z, nz)) {
            const double h = z - 0.5;
            if (obs == 0) {
                gr = (h - J) / s0;
            } else {
                const double w = sigmoid(((double)rho[i].x - (double)rho[i].y) / eps);
                const double dw = w * (1.0 - w) / eps;  // d w / d phi
                double gphi = 0;
                if (obs == 1) gphi = (h - J) * dw / s0;
                else if (z == 1) gphi = dw;
                gr = gphi;
                gb = -gphi;
            }
        }
        E.rb[i] = make_float2((float)gr, (float)gb);
#pragma unroll
        for (int d = 0; d < 3; ++d) E.j[d][i] = make_float2(0.f, 0.f);
    }
}

static int adj_blocks(long long n) { return (int)((n + kAdjThreads - 1) / kAdjThreads); }

template <class S>
cudaError_t launch_adj_forward(const Layout& L, const KParams& P, const S* f, const AdjState& A, cudaStream_t st)
{
    return launch_after(adj_forward_kernel<S>, dim3(adj_blocks((long long)L.nx * L.ny * L.nz)), kAdjThreads, 0, st, L, P, f, A);
}

cudaError_t launch_adj_backstep(const AdjArgs& G, const AdjState& A, bool tau_one, const AdjE& En, const float* Mn,
                                const AdjE& Ec, float* Mc, const AdjV& W, double* part, cudaStream_t st)
{
    const int blocks = adj_blocks((long long)G.nx * G.ny * G.nz);
    const cudaError_t e = launch_after(tau_one ? adj_local_kernel<true> : adj_local_kernel<false>, dim3(blocks), kAdjThreads, 0,
                                       st, G, A, En, Mn, Ec, Mc, W, part);
    if (e != cudaSuccess) return e;
    return launch_after(adj_gather_kernel, dim3(blocks), kAdjThreads, 0, st, G, A, W, Ec);
}

cudaError_t launch_rows_sum(const double* part, int nblocks, double* out, cudaStream_t st)
{
    rows_sum_kernel<<<2, 256, 0, st>>>(part, nblocks, out);
    return cudaGetLastError();
}

cudaError_t launch_observable(int nx, int ny, int nz, int obs, double eps, const float2* rho, double* part,
                              double* sums, const AdjE* E, cudaStream_t st)
{
    obs_sums_kernel<<<kObsBlocks, 256, 0, st>>>(nx, ny, nz, obs, eps, rho, part);
    rows_sum_kernel<<<2, 256, 0, st>>>(part, kObsBlocks, sums);
    obs_finish_kernel<<<1, 32, 0, st>>>(obs, sums);
    if (E) obs_grad_kernel<<<kObsBlocks, 256, 0, st>>>(nx, ny, nz, obs, eps, rho, sums, *E);
    return cudaGetLastError();
}

template cudaError_t launch_adj_forward<float>(const Layout&, const KParams&, const float*, const AdjState&, cudaStream_t);
template cudaError_t launch_adj_forward<__half>(const Layout&, const KParams&, const __half*, const AdjState&, cudaStream_t);
template cudaError_t launch_adj_forward<__nv_bfloat16>(const Layout&, const KParams&, const __nv_bfloat16*,
                                                       const AdjState&, cudaStream_t);

}  // namespace lbsc

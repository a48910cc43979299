// Fused time step (Sec. 2) with the next planes' populations staged into
// shared memory by TMA: planar walls, and (kGeneral) any solid mask.
//
// A CTA owns a 32 x TY tile of columns and a z segment, as in the
// load-from-global kernel, but one thread streams whole planes of the tile
// plus its one-node ring (all 19 slots of paired values, one 4-D tensor box
// per plane) into an NS-deep ring of shared-memory stages with
// cp.async.bulk.tensor, completion tracked by one mbarrier per stage. The
// compute warps reduce a landed plane to rho, j and psi out of shared memory
// while the following planes are in flight, then collide and push the plane
// below. The periodic images come from small extra boxes of real nodes: two
// 16-byte column strips at the x edges, one row at the y edges (the row
// across the periodic boundary) and 16-byte corner pieces of that row, so no
// image of any node is ever stored. Every wait is bounded: a wait that gives
// up writes an error status, drains the CTA's copies in flight and leaves the
// kernel. In a general geometry the planes wrap along z, and a node's mask word
// (its own and its links' solid bits) is loaded while its plane's copy is
// awaited: 4 bytes beside the 304 of an update.
#pragma once

#include <cuda.h>

#include "lb_fields.cuh"
#include "step_common.cuh"

namespace lbsc {

constexpr uint32_t kSpinLimit = 1u << 22;  // try_wait rounds before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the completion of the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2,
                                            int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

// Geometry of one stage. The tensor maps order a buffer as (x values, storage
// row, plane, slot k), so a box of R rows and W columns lands in shared
// memory as [k][r][c][a]: element (k, r, c, a) at 2 ((k R + r) W + c) + a.
// (Ordering the slot before the row would make the layouts of all regions
// alike, but the copies would then walk the 19 slots, hundreds of megabytes
// apart, row by row: measured 16% slower.) Regions, each 128-byte aligned:
//   main     HY rows x BX columns: x = x0 - cofs + c (16 bytes of columns on
//            each side of the tile; edge tiles shift the box inward, see the
//            kernel), rows from the tile's row window;
//   xs       HY rows x SX columns (16 bytes), the same rows, for the tiles at the
//            x edges of a row of several: the first tile's holds the columns
//            around x = nx - 1 (the images of x = -1), the last one's x = 0 ..
//            SX - 1 (the images of x >= nx);
//   ys       one row x BX columns: the row across the periodic y boundary
//            (y = ny - 1 for the first row of tiles, y = 0 for the last);
//   cs       one row x SX columns: the x-edge piece of that row.
// A single tile in x holds every column from x = 0 on, and takes the images
// from there. Element offsets count values (two per node).
// The load is bound by the 128-byte lines its box rows touch (64^3: boxes of
// the 36 columns, 4 lines a row, take 14.4 of the step's 16.2 us, of 2 aligned
// lines 10.1). Tiles begun one node later, so that a row touches 3 lines, lost
// more in their misaligned stores (128^3 FP32 116.0 against 109.4 us,
// 256x256x128 BF16 292.7 against 282.0).
// FP32 4-row tiles with one stage keep psi of three planes, not four (one more
// barrier a plane): 45.5 KB, five CTAs an SM (the batched step: four, see there).
template <class S, int TY, int NS, bool kBatch = false>
struct TmaGeom {
    static constexpr int TX = 32, HX = TX + 2, HY = TY + 2;
    static constexpr int GX = edge_x<S>();                    // nodes in 16 bytes
    static constexpr int BX = TX + 2 * GX;                   // the box's nodes per row: 16 bytes of columns each side
    static constexpr int SX = GX;                            // strip width: 16 bytes of columns
    static constexpr int al(int elems) { return (elems * (int)sizeof(S) + 127) / 128 * 128 / (int)sizeof(S); }
    static constexpr int MAIN_ELEMS = 2 * Q * HY * BX;
    static constexpr int XS_ELEMS = 2 * Q * HY * SX;
    static constexpr int YS_ELEMS = 2 * Q * BX;
    static constexpr int CS_ELEMS = 2 * Q * SX;
    static constexpr int YS = al(MAIN_ELEMS), CS = YS + al(YS_ELEMS), XS = CS + al(CS_ELEMS);
    static constexpr int STAGE_ELEMS = al(XS + XS_ELEMS);
    static constexpr uint32_t MAIN_BYTES = MAIN_ELEMS * sizeof(S);
    static constexpr uint32_t XS_BYTES = XS_ELEMS * sizeof(S);
    static constexpr uint32_t YS_BYTES = YS_ELEMS * sizeof(S);
    static constexpr uint32_t CS_BYTES = CS_ELEMS * sizeof(S);
    static constexpr uint32_t STAGE_BYTES = STAGE_ELEMS * sizeof(S);
    static constexpr int PSI_PLANES = sizeof(S) == 4 && TY == 4 && NS == 1 && !kBatch ? 3 : 4;
    static constexpr int PSI_FLOATS = PSI_PLANES * 2 * HY * HX;
    // psi follows the last stage's last region without padding
    static constexpr size_t PSI_AT = ((size_t)(NS - 1) * STAGE_ELEMS + XS + XS_ELEMS) * sizeof(S);
    static constexpr size_t SMEM = PSI_AT + PSI_FLOATS * 4 + NS * 8;
    static_assert(PSI_AT % 8 == 0, "psi pairs are 8-byte accesses");
};

// Resident CTAs per SM the registers are held to (tau = 1): for 8-row tiles
// three FP32 CTAs (shared memory admits no more) and four 16-bit CTAs (64
// registers, a few words spilled: 32 warps per SM measured faster than 24);
// five CTAs of 4-row tiles; other variants take the compiler's choice.
template <class S, int TY, bool kTauOne>
constexpr int kTmaCtas = !kTauOne ? 1 : (TY == 8 ? (sizeof(S) == 2 ? 4 : 3) : (TY == 4 ? 5 : 1));

// The four tensor maps of one buffer and tile height: main box, x-edge strip,
// y-edge row, corner piece (boxes HY x BX, HY x SX, 1 x BX, 1 x SX nodes).
struct TmaMaps {
    CUtensorMap m[4];
};

// One work item: tile column `col` of the lattice A (tile row col / tiles_x,
// x tile col % tiles_x), fluid planes [za, zb), with the maps of A's source
// buffer. `stages`, `sp` and `bar` are the CTA's shared stages, psi ring and
// stage barriers; g counts the planes the CTA has consumed so far (the
// barriers' phases run on across items). The first item (started: false) waits
// for the step before, whose end its index arithmetic overlaps, and every item
// then reads the step counter into clk. Returns false when a wait gave up (the
// status word is set and the CTA's copies in flight are drained).
template <class S, int TY, int NS, bool kTauOne, bool kGeneral, bool kBatch>
__device__ __forceinline__ bool tma_item(const TmaMaps& maps, const StepArgs<S>& A, int col, int za, int zb, S* stages,
                                         float* sp, uint64_t* bar, uint32_t& g, uint32_t& clk, bool& started)
{
    using G = TmaGeom<S, TY, NS, kBatch>;
    constexpr int TX = 32, NT = TX * TY, HX = G::HX, HY = G::HY, GX = G::GX, BX = G::BX, SX = G::SX;
    constexpr int RING = 2 * HX + 2 * TY;
    constexpr int NIT = (RING + NT - 1) / NT;
    using P2 = typename Codec<S>::Pair;

    const Layout L = A.L;
    const int nx = L.nx, ny = L.ny, nz = L.nz;
    const int plane = (int)L.plane;
    S* __restrict__ dst = A.dst;
    const float eta[2] = {A.P.eta[0], A.P.eta[1]};
    const float ref[2] = {A.P.ref[0], A.P.ref[1]};
    const float tau[2] = {A.P.tau[0], A.P.tau[1]};
    const float itau[2] = {A.P.itau[0], A.P.itau[1]};
    const float gk = A.P.gk, Gax = A.P.Gax;
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;

    // rows [y0, y0 + hgt) of an even split of ny (hgt <= TY); a row past hgt is an idle warp
    const int tyi = col / A.tiles_x;
    const int x0 = (col - tyi * A.tiles_x) * TX;
    const int y0 = tile_row(tyi, ny, A.tiles_y), hgt = tile_row(tyi + 1, ny, A.tiles_y) - y0;
    const int gx = x0 + tx, gy = y0 + ty;
    const bool active = ty < hgt;
    const bool valid = active && gx < nx;
    const int np = zb - za + 2;  // planes za-1 .. zb
    // x edges: the periodic images come from the strip (column of x = nx - 1 in the first tile's), or,
    // with a single tile, from the box itself
    const bool one = A.tiles_x == 1;
    const bool left_edge = x0 == 0 && !one, right_edge = x0 + TX >= nx && !one;
    // the box's column of node x0: GX (16 bytes of ring columns on each
    // side); an edge tile takes its outer ring column from a strip, so its
    // box is shifted inward and reads no padding columns beyond the lattice
    // (0 at the left edge, 2 GX at the right edge)
    const int cofs = x0 == 0 ? 0 : (right_edge ? 2 * GX : GX);
    const int sl = (L.gx + nx - 1) / SX * SX, ol = L.gx + nx - 1 - sl;
    // y edges: the row window of the box, given by the box row of node row
    // y0 (rofs). A middle tile's box holds rows y0 - 1 .. y0 + TY; the first
    // row of tiles' rows 0 .. HY - 1 and the last row's the HY rows ending at
    // its last own row, the ring row across the boundary coming from the
    // y-edge row (ys, with its corner pieces). With a single row of tiles
    // (ny <= TY) the box holds every row and the ring rows wrap inside it.
    const bool single = A.tiles_y == 1;
    const bool first = tyi == 0 && !single, last = tyi == A.tiles_y - 1 && !single;
    const int rofs = (first || single) ? 0 : (last ? HY - hgt : 1);
    const int yrow = first ? ny - 1 : 0;  // the real row in ys (first or last row of tiles)
    // own node: the main box; the lane past x = nx - 1 of a ragged last tile
    // holds the periodic image x = 0, the +x neighbour of x = nx - 1
    const bool own_strip = right_edge && gx >= nx;
    const bool own_rd = active && gx <= nx;
    const int own_off = own_strip ? G::XS + 2 * ((ty + rofs) * SX + gx - nx)
                                  : 2 * ((ty + rofs) * BX + (one && gx == nx ? 0 : tx + cofs));
    const int own_node = (gy + 1) * L.px + L.gx + (gx < nx ? gx : 0);  // its offset in its plane (general geometry)
    // the copies' coordinates: x of the main box and of the left strip in
    // values (two per node; 16-byte aligned, as the copy requires), storage
    // row (real row + 1) of the box's first row and of the y-edge row (-1: none)
    const int xb = 2 * (x0 + L.gx - cofs), xs = 2 * sl;
    const int yb = y0 - rofs + 1, ysr = (first || last) ? yrow + 1 : -1;

    // ring items (one per ring node, both components): shared-memory
    // position, stage position of the node's slot-0 pair, and its region's
    // slot stride: 0 main box (2 HY BX), 1 x strip (2 HY SX), 2 y-edge row
    // (2 BX), 3 corner piece (2 SX)
    // (packed in one word: stage position in bits 0-16, shared-memory position in
    // bits 17-26, stride class in bits 27-28; -1 for no item)
    static_assert(G::STAGE_ELEMS <= (1 << 17) && HY * HX <= (1 << 10), "ring item fields fit their bits");
    int it_code[NIT], it_node[NIT];  // it_node (general geometry): the node's offset in its plane
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
        const int r = tid + i * NT;
        it_code[i] = -1;
        it_node[i] = 0;
        if (r < RING) {
            int it_sm, it_base, it_cls;
            int ix, iy;
            if (r < HX) { ix = r; iy = 0; }
            else if (r < 2 * HX) { ix = r - HX; iy = hgt + 1; }
            else if (r < 2 * HX + TY) { ix = 0; iy = r - 2 * HX + 1; }
            else { ix = HX - 1; iy = r - 2 * HX - TY + 1; }
            it_sm = iy * HX + ix;
            const int xr = x0 - 1 + ix, yr = y0 - 1 + iy;  // the ring node (unwrapped)
            // side columns: the tile's own rows only; nothing past x = nx
            const bool on = (r < 2 * HX || iy <= hgt) && xr <= nx;
            const bool across = (first && yr < 0) || (last && yr >= ny);  // in the y-edge row
            const int row = wrapi(yr, ny) - y0 + rofs;                   // box row otherwise
            if ((xr < 0 || xr >= nx) && !one) {
                const int c = xr < 0 ? ol : xr - nx;  // the image's column in the strip
                it_cls = across ? 3 : 1;
                it_base = across ? G::CS + 2 * c : G::XS + 2 * (row * SX + c);
            } else {
                const int c = one ? wrapi(xr, nx) : ix - 1 + cofs;
                it_cls = across ? 2 : 0;
                it_base = across ? G::YS + 2 * c : 2 * (row * BX + c);
            }
            if (on) it_code[i] = it_base | (it_sm << 17) | (it_cls << 27);
            if constexpr (kGeneral)
                if (on) it_node[i] = (wrapi(yr, ny) + 1) * L.px + L.gx + (xr < 0 ? xr + nx : xr % nx);
        }
    }

    // a wall plane of the planar geometry (a z slab's halo plane is loaded like fluid)
    auto wall_plane = [&](int zp) {
        return !kGeneral && ((zp == 0 && !(A.halo & 1)) || (zp == nz - 1 && !(A.halo & 2)));
    };
    auto issue = [&](int zu, uint32_t gi) {
        uint64_t* b = &bar[gi % NS];
        const int zp = kGeneral ? wrapi(zu, nz) : zu;
        if (wall_plane(zp)) {
            mbar_arrive(b);  // nothing to load
        } else {
            S* stg = stages + (size_t)(gi % NS) * G::STAGE_ELEMS;
            const bool ye = ysr >= 0;
            fence_proxy_async();
            const bool xe = left_edge || right_edge;
            const int xc = left_edge ? xs : 2 * L.gx;
            mbar_expect_tx(b, G::MAIN_BYTES + (xe ? G::XS_BYTES : 0u) + (ye ? G::YS_BYTES + (xe ? G::CS_BYTES : 0u) : 0u));
            tma_load_4d(stg, &maps.m[0], b, xb, yb, zp, 0);
            if (xe) tma_load_4d(stg + G::XS, &maps.m[1], b, xc, yb, zp, 0);
            if (ye) {
                tma_load_4d(stg + G::YS, &maps.m[2], b, xb, ysr, zp, 0);
                if (xe) tma_load_4d(stg + G::CS, &maps.m[3], b, xc, ysr, zp, 0);
            }
        }
    };
    // the psi ring's plane of lattice plane z
    auto psi_plane = [&](int z) {
        return (float2*)sp + (G::PSI_PLANES == 4 ? (z & 3) : (z + 3) % 3) * (HY * HX);
    };

    // wait for plane i of the item, reduce it to psi (tile + ring) and own
    // moments, then refill its stage with plane i + NS
    auto consume = [&](int i, float (&rho)[2], float (&j)[2][3], float (&v)[2][Q], float (&m)[2], uint32_t& nb) -> bool {
        const int zp = za - 1 + i;
        const uint32_t gi = g + i;
        bool solid_own = wall_plane(zp), solid_it[NIT];
#pragma unroll
        for (int q = 0; q < NIT; ++q) solid_it[q] = solid_own;
        if constexpr (kGeneral) {
            const uint32_t* mask = A.nbmask + wrapi(zp, nz) * plane;
            auto word = [&](int node) {
                if constexpr (kCheckBounds)
                    if (!in_bounds((long long)wrapi(zp, nz) * plane + node, (long long)plane * nz, A.err)) return kSelfSolid;
                return __ldg(mask + node);
            };
            nb = own_rd ? word(own_node) : kSelfSolid;
            solid_own = (nb & kSelfSolid) != 0;
#pragma unroll
            for (int q = 0; q < NIT; ++q)
                if (it_code[q] >= 0) solid_it[q] = (word(it_node[q]) & kSelfSolid) != 0;
        }
        const bool ok = mbar_wait(&bar[gi % NS], (gi / NS) & 1u);
        float2* spl = psi_plane(zp);
        // with three planes, this one takes the place of the lowest that the collision before read
        if constexpr (G::PSI_PLANES == 3) __syncthreads();
        if (ok) {
            const S* st = stages + (size_t)(gi % NS) * G::STAGE_ELEMS;
            float ps[2] = {eta[0], eta[1]};
            rho[0] = rho[1] = m[0] = m[1] = 0.f;
#pragma unroll
            for (int a = 0; a < 2; ++a) j[a][0] = j[a][1] = j[a][2] = 0.f;
            if (!solid_own && own_rd) {
                float w[2][Q];
                // both components of velocity k in one shared-memory load
                const P2* so = (const P2*)(st + own_off);
                if (!own_strip) {
#pragma unroll
                    for (int k = 0; k < Q; ++k) {
                        const float2 t = Codec<S>::val2(so[k * HY * BX]);
                        w[0][k] = t.x;
                        w[1][k] = t.y;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < Q; ++k) {
                        const float2 t = Codec<S>::val2(so[k * HY * SX]);
                        w[0][k] = t.x;
                        w[1][k] = t.y;
                    }
                }
                moments2<S>(w, ref, rho, j, m);
                const float2 p2 = psi2_of(f2(rho[0], rho[1]));
                ps[0] = p2.x;
                ps[1] = p2.y;
                if constexpr (!kTauOne) {
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int k = 0; k < Q; ++k) v[a][k] = w[a][k];
                }
            }
            if (active) {
                spl[(ty + 1) * HX + tx + 1] = psi_pair(ps[0], ps[1]);
            }
#pragma unroll
            for (int q = 0; q < NIT; ++q) {
                const int code = it_code[q];
                if (code < 0) continue;
                const int it_sm = (code >> 17) & 0x3FF;
                float2 pr = f2(eta[0], eta[1]);
                if (!solid_it[q]) {
                    // both components of velocity k in one shared-memory load
                    float2 w[Q];
                    const P2* si = (const P2*)(st + (code & 0x1FFFF));
                    const int cls = (code >> 27) & 3;
                    if (cls == 0) {
#pragma unroll
                        for (int k = 0; k < Q; ++k) w[k] = Codec<S>::val2(si[k * HY * BX]);
                    } else if (cls == 1) {
#pragma unroll
                        for (int k = 0; k < Q; ++k) w[k] = Codec<S>::val2(si[k * HY * SX]);
                    } else if (cls == 2) {
#pragma unroll
                        for (int k = 0; k < Q; ++k) w[k] = Codec<S>::val2(si[k * BX]);
                    } else {
#pragma unroll
                        for (int k = 0; k < Q; ++k) w[k] = Codec<S>::val2(si[k * SX]);
                    }
                    float2 unused;
                    pr = psi2_of(rho2_of<S>(w, f2(ref[0], ref[1]), unused));
                }
                spl[it_sm] = psi_pair(pr.x, pr.y);
            }
        }
        const bool bad = __syncthreads_or(!ok);
        if (bad) {
            if (tid == 0) {
                atomicOr(A.err, kErrWait);
                for (int k2 = i; k2 < np && k2 < i + NS; ++k2) mbar_wait(&bar[(g + k2) % NS], ((g + k2) / NS) & 1u);
            }
            return false;
        }
        if (tid == 0 && i + NS < np) issue(zp + NS, gi + NS);
        return true;
    };

    float rc[2], jc[2][3], vc[2][Q], mc[2];
    float rn[2], jn[2][3], vn[2][Q], mn[2];
    uint32_t nbc = 0, nbn = 0;  // general geometry: mask words of the current and the next plane's own node
    if (!started) {
        grid_wait();
        started = true;
    }
    if constexpr (Codec<S>::kDeviation) clk = clock_read(A.clock);
    __syncthreads();  // the previous item's collide is done with the psi ring
    if (tid == 0)
        for (int i = 0; i < NS && i < np; ++i) issue(za - 1 + i, g + i);
    if (!consume(0, rn, jn, vn, mn, nbn) || !consume(1, rc, jc, vc, mc, nbc)) return false;

    Dest<S, sizeof(S) == 4 && !kBatch> D;
    D.set_column(L, valid ? gx : 0, valid ? gy : 0);
    D.err = A.err;
    D.hoff = A.hkey;

    for (int z = za; z < zb; ++z) {
        if (!consume(z - za + 2, rn, jn, vn, mn, nbn)) return false;
        if (valid && !(kGeneral && (nbc & kSelfSolid))) {
            float F[2][3];
            sc_force<HX, HY>(psi_plane(z - 1), psi_plane(z), psi_plane(z + 1), ty, tx, gk, Gax, F);
            D.zo[0] = (kGeneral ? wrapi(z - 1, nz) : z - 1) * plane;
            D.zo[1] = z * plane;
            D.zo[2] = (kGeneral ? wrapi(z + 1, nz) : z + 1) * plane;
            D.bot = !kGeneral && z - 1 == 0 && !(A.halo & 1);  // a halo plane takes pushes like fluid
            D.top = !kGeneral && z + 1 == nz - 1 && !(A.halo & 2);
            D.nb = nbc;
            if constexpr (Codec<S>::kDeviation) {
                // rho = rho_ref + m36 / 36, as moments2 forms it: not held across the plane
                const float2 r = fma2(f2(mc[0], mc[1]), sp2(1.0f / 36.0f), f2(ref[0], ref[1]));
                const float rr[2] = {r.x, r.y};
                collide_store<S, kGeneral, kTauOne>(rr, jc, vc, F, tau, itau, ref, dst, L, D, mc, clk);
            } else {
                collide_store<S, kGeneral, kTauOne>(rc, jc, vc, F, tau, itau, ref, dst, L, D, mc, clk);
            }
        }
        nbc = nbn;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if constexpr (!Codec<S>::kDeviation) rc[a] = rn[a];
            mc[a] = mn[a];
#pragma unroll
            for (int d = 0; d < 3; ++d) jc[a][d] = jn[a][d];
            if constexpr (!kTauOne) {
#pragma unroll
                for (int k = 0; k < Q; ++k) vc[a][k] = vn[a][k];
            }
        }
    }
    g += np;
    return true;
}

template <class S, int TY, int NS, bool kTauOne, bool kGeneral>
__global__ void __launch_bounds__(32 * TY, (kTmaCtas<S, TY, kTauOne>))
    step_tma_kernel(const __grid_constant__ TmaMaps maps, const StepArgs<S> A)
{
    using G = TmaGeom<S, TY, NS>;
    static_assert(G::STAGE_BYTES % 128 == 0 && (G::XS * sizeof(S)) % 128 == 0 && (G::YS * sizeof(S)) % 128 == 0 &&
                      (G::CS * sizeof(S)) % 128 == 0,
                  "stages and their regions stay 128-byte aligned");
    static_assert((2 * G::BX * sizeof(S)) % 16 == 0 && (2 * G::SX * sizeof(S)) % 16 == 0,
                  "box rows are whole 16-byte units");
    extern __shared__ __align__(128) unsigned char smem[];
    S* stages = (S*)smem;
    float* sp = (float*)(smem + G::PSI_AT);  // psi ring [PSI_PLANES][HY][HX] of pairs (psi^b, psi^r)
    uint64_t* bar = (uint64_t*)(sp + G::PSI_FLOATS);
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) mbar_init(&bar[s], 1);
        mbar_fence_init();
    }
    __syncthreads();
    grid_trigger();  // the next step's CTAs may take the slots that free up, up to their own wait
    uint32_t g = 0;  // planes this CTA has issued and consumed so far
    uint32_t clk = 0;
    bool started = false;
    const int ncol = A.tiles_x * A.tiles_y;
    const int nzf = A.zhi - A.zlo;
    for (int item = blockIdx.x; item < ncol * A.nseg; item += gridDim.x) {
        const int col = item % ncol, seg = item / ncol;
        const int za = A.zlo + (int)((long long)seg * nzf / A.nseg);
        const int zb = A.zlo + (int)((long long)(seg + 1) * nzf / A.nseg);
        if (za >= zb) continue;
        if (!tma_item<S, TY, NS, kTauOne, kGeneral, false>(maps, A, col, za, zb, stages, sp, bar, g, clk, started)) break;
    }
    if (!started) grid_wait();
    if constexpr (Codec<S>::kDeviation) clock_tick(A.clock);
}

// Batched TMA step: a persistent grid walks a work list of (box, tile column,
// first plane, end plane) items over many planar-wall lattices with their own
// sizes and parameters; args[2 box + parity] and maps[2 box + parity] describe
// box `box` for this step (the maps live in global memory, written by the host
// before the launch). The last CTA out advances every box's step counter.
// It is launched after the step before has ended, keeps psi of four planes (four
// FP32 CTAs of 4-row tiles an SM) and stores by node offsets: an item's ring
// rows come from L2 only while neighbouring CTAs stay in step, which CTAs placed
// as slots free up, or five an SM, do not (64 boxes of edge 48-96: 1262 us a step
// FP32 and 958 BF16, launched dependently with three planes 1668 and 1511; 6
// boxes 115 and 91, 124 and 90).
template <class S, int TY, int NS, bool kTauOne>
__global__ void __launch_bounds__(32 * TY, (kTmaCtas<S, TY, kTauOne>))
    batch_tma_kernel(const TmaMaps* __restrict__ maps, const StepArgs<S>* __restrict__ args,
                     const int4* __restrict__ items, int nitems, int parity, int nbox, uint32_t* done)
{
    using G = TmaGeom<S, TY, NS, true>;
    extern __shared__ __align__(128) unsigned char smem[];
    S* stages = (S*)smem;
    float* sp = (float*)(smem + G::PSI_AT);
    uint64_t* bar = (uint64_t*)(sp + G::PSI_FLOATS);
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) mbar_init(&bar[s], 1);
        mbar_fence_init();
    }
    __syncthreads();
    uint32_t g = 0;
    bool started = true;  // launched whole, after the step before
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const int4 w = items[it];
        const StepArgs<S>& A = args[2 * w.x + parity];
        const TmaMaps& M = maps[2 * w.x + parity];
        if (threadIdx.x == 0)
            for (int i = 0; i < 4; ++i)  // the maps were written through the generic proxy
                asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&M.m[i]) : "memory");
        uint32_t clk = 0;
        if (!tma_item<S, TY, NS, kTauOne, false, true>(M, A, w.y, w.z, w.w, stages, sp, bar, g, clk, started)) break;
    }
    if constexpr (Codec<S>::kDeviation) {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(done, 1u) == gridDim.x - 1) {
                atomicExch(done, 0u);
                for (int b = 0; b < nbox; ++b) atomicAdd(args[2 * b].clock, 1u);
            }
        }
    }
}

template <class S, int TY, int NS, bool T1, bool GEN>
static long long tma_one(int op, const CUtensorMap* m, const StepArgs<S>* A, cudaStream_t st)
{
    const auto kernel = step_tma_kernel<S, TY, NS, T1, GEN>;
    constexpr size_t smem = TmaGeom<S, TY, NS>::SMEM;
    if (op == 0) {
        TmaMaps maps;
        for (int i = 0; i < 4; ++i) maps.m[i] = m[i];
        return launch_after(kernel, dim3(A->tiles_x * A->tiles_y * A->nseg), 32 * TY, smem, st, maps, *A);
    }
    if (op == 1) return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, 32 * TY, smem) != cudaSuccess) return 1;
    return n;
}

// Dispatch over the built (tile height, stages, tau == 1) combinations.
// op 0: launch; op 1: set the shared-memory attribute; op 2: occupancy.
template <class S, bool GEN>
static long long tma_dispatch(int op, int ty, int ns, bool t1, const CUtensorMap* m, const StepArgs<S>* A,
                              cudaStream_t st)
{
#define LBSC_TMA_CASE(TY_, NS_)                                                           \
    if (ty == TY_ && ns == NS_) {                                                         \
        if (op == 1) {                                                                    \
            const long long e = tma_one<S, TY_, NS_, true, GEN>(op, m, A, st);            \
            return e != cudaSuccess ? e : tma_one<S, TY_, NS_, false, GEN>(op, m, A, st); \
        }                                                                                 \
        return t1 ? tma_one<S, TY_, NS_, true, GEN>(op, m, A, st)                         \
                  : tma_one<S, TY_, NS_, false, GEN>(op, m, A, st);                       \
    }
    LBSC_TMA_CASE(4, 1)
    LBSC_TMA_CASE(4, 2)
    if constexpr (!GEN || sizeof(S) == 2) {
        LBSC_TMA_CASE(8, 1)
        LBSC_TMA_CASE(8, 2)
    }
    if constexpr (!GEN) {
        LBSC_TMA_CASE(4, 3)
        LBSC_TMA_CASE(8, 3)
    }
    if constexpr (!GEN && sizeof(S) == 2) {
        LBSC_TMA_CASE(16, 1)
        LBSC_TMA_CASE(16, 2)
    }
#undef LBSC_TMA_CASE
    return op == 2 ? 0 : (long long)cudaErrorInvalidValue;
}

// The batched TMA kernel for one stage and 4- or 8-row tiles: op 0 launches
// on `grid` CTAs (returns a cudaError_t), op 1 sets the shared-memory
// attribute, op 2 returns the CTAs per SM to launch (0 if not built).
template <class S, int TY, bool T1>
static long long tma_batch_one(int op, const TmaMaps* maps, const StepArgs<S>* args, const int4* items, int nitems,
                               int parity, int nbox, uint32_t* done, int grid, cudaStream_t st)
{
    constexpr size_t smem = TmaGeom<S, TY, 1, true>::SMEM;
    if (op == 0) {
        batch_tma_kernel<S, TY, 1, T1><<<grid, 32 * TY, smem, st>>>(maps, args, items, nitems, parity, nbox, done);
        return cudaGetLastError();
    }
    if (op == 1)
        return cudaFuncSetAttribute(batch_tma_kernel<S, TY, 1, T1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_tma_kernel<S, TY, 1, T1>, 32 * TY, smem) !=
        cudaSuccess)
        return 0;
    // three FP32 CTAs of 8-row tiles fit, but two re-read fewer ring rows: they stay nearer each other (64 boxes of edge
    // 48-96 take 1434 us a step, 1863 with three; 8 boxes of 128^3 814 and 1052)
    return TY == 8 && sizeof(S) == 4 && n > 2 ? 2 : n;
}

template <class S>
static long long tma_batch_dispatch(int op, int ty, bool t1, const void* maps, const StepArgs<S>* args,
                                    const int4* items, int nitems, int parity, int nbox, uint32_t* done, int grid,
                                    cudaStream_t st)
{
    const TmaMaps* m = (const TmaMaps*)maps;
    if (ty == 4)
        return t1 ? tma_batch_one<S, 4, true>(op, m, args, items, nitems, parity, nbox, done, grid, st)
                  : tma_batch_one<S, 4, false>(op, m, args, items, nitems, parity, nbox, done, grid, st);
    if (ty == 8)
        return t1 ? tma_batch_one<S, 8, true>(op, m, args, items, nitems, parity, nbox, done, grid, st)
                  : tma_batch_one<S, 8, false>(op, m, args, items, nitems, parity, nbox, done, grid, st);
    return op == 2 ? 0 : (long long)cudaErrorInvalidValue;
}

}  // namespace lbsc

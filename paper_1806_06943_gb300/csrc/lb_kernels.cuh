// lb_kernels.cuh -- sm_103a kernels of the two-range pseudopotential lattice
// Boltzmann step (Fei et al., arXiv:1806.06943, Sec. II), templated on the
// population format:
//   real = double : plain populations f; this instantiation is compiled
//                   without fused multiply-add and rounds every operation of a
//                   direct evaluation of the equations, in its order (lb_f64.cuh
//                   says on which pipe), so it reproduces a plain FP64 evaluation
//                   up to the last bit of exp().
//   real = float  : offset populations h_i = f_i - w_i R, R the node's density
//                   at the previous step (kept in the other density copy), so
//                   the stored numbers are the small deviations from the local
//                   equilibrium at rest and keep their low-order digits.  The
//                   stencil and momentum sums are formed from differences of
//                   opposite neighbours, which keeps them exactly antisymmetric
//                   under reflection even with fused multiply-add (no drift).
//
// One time step is two launches over a list of tiles (lattice, x0, y0):
//   k_density : rho_k = sum_i f_k,i                           (Eq. 6)
//   k_collide : stages rho_k of the tile plus a 2-node halo in shared memory,
//               psi_k = 1 - exp(-rho_k) (Sec. II B), the forces of Eqs. (8),
//               (9) and rho_k g, the moments of Eq. (6), u^eq of Eq. (3), the
//               BGK relaxation to Eq. (2) with the Guo term of Eq. (5), and
//               pushes each post-collision population to x + e_i, reflecting
//               it at a half-way bounce-back wall (Sec. III A).
// or one: k_fused, k_fused_tma (lb_tma.cu, FP32), k_small64 (small FP64 lattices).
// The populations at a node are the pre-collision values of the current time,
// so both passes read them at their own node with coalesced loads.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "lb_f64.cuh"
#include "lb_types.h"
#include "lb_vops.cuh"

#include <type_traits>

namespace lbk {

constexpr int TX = 32;           // tile width = threads in x
constexpr int TY = 4;            // tile height of the observation kernels = threads in y
constexpr int HALO = 2;          // reach of the D2Q25 stencil
constexpr int SW = TX + 2 * HALO;
constexpr int SH = TY + 2 * HALO;
constexpr int kThreads = TX * TY;
// Tile heights the time-step kernels are built for (chosen per batch by the
// autotuner); one thread per node, 32 nodes wide.
constexpr int kTileHeights[3] = {2, 4, 8};

template <typename real>
constexpr bool kOffset = sizeof(real) == 4;

// Resident blocks per SM the fused kernel is compiled for: the FP32 kernel is
// bound by HBM and needs the warps to keep enough loads in flight; the FP64
// kernel is bound by the FP64 pipe, which 16 warps fill (24 with 550 bytes of
// spill measured 7 % slower on a 1024^2 lattice).
template <typename real, int TYv>
constexpr int kCollideMinBlocks = (kOffset<real> ? 32 : 16) / TYv;

// ---- lattice tables (Sec. II A; Fig. 1; Sec. II B after Eq. 8) ------------
// D2Q9 order: rest, (1,0), (0,1), (-1,0), (0,-1), (1,1), (-1,1), (-1,-1), (1,-1).
__host__ __device__ constexpr int ex9(int i) { return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0); }
__host__ __device__ constexpr int ey9(int i) { return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0); }
__host__ __device__ constexpr int opp9(int i)
{
    return i == 0 ? 0 : i == 1 ? 3 : i == 2 ? 4 : i == 3 ? 1 : i == 4 ? 2 : i == 5 ? 7 : i == 6 ? 8 : i == 7 ? 5 : 6;
}
// w(|e|^2) class of direction i: 0 rest, 1 axis, 2 diagonal.
__host__ __device__ constexpr int cls9(int i) { return i == 0 ? 0 : (i <= 4 ? 1 : 2); }
__host__ __device__ constexpr double w9(int i) { return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0); }
// D2Q25 weights p(|e|^2).
__host__ __device__ constexpr double p25(int e2)
{
    return e2 == 0 ? 247.0 / 420.0 : e2 == 1 ? 4.0 / 63.0 : e2 == 2 ? 4.0 / 135.0 : e2 == 4 ? 1.0 / 180.0
         : e2 == 5 ? 2.0 / 945.0 : e2 == 8 ? 1.0 / 15120.0 : 0.0;
}
// the same weights rounded to FP32
struct P25f {
    __host__ __device__ constexpr float operator()(int e2) const { return (float)p25(e2); }
};
constexpr P25f p25f{};

template <typename real> __device__ __forceinline__ real psi_of(real r);
// psi = rho0 (1 - exp(-rho/rho0)), rho0 = 1 (Sec. II B)
template <> __device__ __forceinline__ double psi_of<double>(double r) { return 1.0 - exp(-r); }
// same function, written through expm1 so small densities keep their digits
template <> __device__ __forceinline__ float psi_of<float>(float r) { return -expm1f(-r); }

// a modulo n, the remainder never negative.  Slots of a tile lie one period off at
// most unless the lattice is narrower than the tile: the division, and a branch
// that lanes take apart, only there (64^2 in tiles of 2, FP32 one pass: 5.0 us a
// step with the branch for every slot beyond the edge, 4.75 so).
__device__ __forceinline__ int wrap_index(int a, int n)
{
    const int r = a < 0 ? a + n : (a >= n ? a - n : a);
    if ((unsigned)r < (unsigned)n) return r;
    a %= n;
    return a < 0 ? a + n : a;
}

// The same for a column of the FP64 step's slots, most of which lie inside: the
// row kernel takes the shorter code (films of 186 x 8 11.8 us a step, 12.0 with
// wrap_index).
__device__ __forceinline__ int wrap_column64(int a, int n)
{
    if ((unsigned)a < (unsigned)n) return a;
    a %= n;
    return a < 0 ? a + n : a;
}

// Stage rho_k and psi_k of the tile plus its halo into shared memory from the
// density copy `rho`.  Periodic copies in x (and in y without walls); beyond a
// wall the ghost rows are either mirrored from the fluid or set to the fixed
// wall densities.
template <typename real, int SHv>
__device__ __forceinline__ void stage_tile(const Lat<real> &L, const real *__restrict__ rho, int x0, int y0,
                                           real (*srho)[SHv][SW], real (*spsi)[SHv][SW], int tid, int nthreads)
{
    constexpr int TYv = SHv - 2 * HALO;
    const int nx = L.nx, ny = L.ny;
    // tiles whose halo lies inside the lattice need no wrapping or ghosts
    const bool inner = x0 >= HALO && x0 + TX + HALO <= nx && y0 >= HALO && y0 + TYv + HALO <= ny;
    if (inner) {
        const real *__restrict__ base = rho + (size_t)(y0 - HALO) * L.pitch + (x0 - HALO);
        for (int idx = tid; idx < SW * SHv; idx += nthreads) {
            const int sx = idx % SW, sy = idx / SW;
            const size_t c = (size_t)sy * L.pitch + sx;
            const real rA = base[c], rB = base[L.plane + c];
            srho[0][sy][sx] = rA;
            srho[1][sy][sx] = rB;
            spsi[0][sy][sx] = psi_of<real>(rA);
            spsi[1][sy][sx] = psi_of<real>(rB);
        }
        return;
    }
    for (int idx = tid; idx < SW * SHv; idx += nthreads) {
        const int sx = idx % SW, sy = idx / SW;
        const int gx = wrap_index(x0 + sx - HALO, nx);
        int gy = y0 + sy - HALO;
        real rA, rB;
        bool fixed = false;
        if (gy < 0 || gy >= ny) {
            if (L.walls) {
                if (L.wall_mode == 1) {
                    rA = L.wall_rho[0];
                    rB = L.wall_rho[1];
                    fixed = true;
                } else {
                    gy = gy < 0 ? -1 - gy : 2 * ny - 1 - gy;
                    gy = gy < 0 ? 0 : (gy >= ny ? ny - 1 : gy);  // rows no valid node reads
                }
            } else {
                gy = wrap_index(gy, ny);
            }
        }
        if (!fixed) {
            const size_t c = (size_t)gy * L.pitch + gx;
            rA = rho[c];
            rB = rho[L.plane + c];
        }
        srho[0][sy][sx] = rA;
        srho[1][sy][sx] = rB;
        spsi[0][sy][sx] = psi_of<real>(rA);
        spsi[1][sy][sx] = psi_of<real>(rB);
    }
}

// sum_{i=1..8} w_i s(x + e_i) e_i (Eqs. 8, 9).
// FP64: added in direction order.  FP32: differences of opposite neighbours.
template <typename real>
__device__ __forceinline__ void q9_sum(const real (*s)[SW], int cx, int cy, real &sx, real &sy)
{
    const real W1 = (real)(1.0 / 9.0), W2 = (real)(1.0 / 36.0);
    if constexpr (!kOffset<real>) {
        const real a1 = W1 * s[cy][cx + 1], a2 = W1 * s[cy + 1][cx], a3 = W1 * s[cy][cx - 1], a4 = W1 * s[cy - 1][cx];
        const real a5 = W2 * s[cy + 1][cx + 1], a6 = W2 * s[cy + 1][cx - 1];
        const real a7 = W2 * s[cy - 1][cx - 1], a8 = W2 * s[cy - 1][cx + 1];
        sx = ((((a1 - a3) + a5) - a6) - a7) + a8;
        sy = ((((a2 - a4) + a5) + a6) - a7) - a8;
    } else {
        (void)W1;
        (void)W2;
        vq9<float>([&](int dy, int dx) { return s[cy + dy][cx + dx]; }, sx, sy);
    }
}

// sum_j p_j s(x + e_j) e_j over D2Q25 (FP64), in raster order (dy outer, dx
// inner).  The FP32 step sums the psi terms with combined weights (vq25c).
template <typename real>
__device__ __forceinline__ void q25_sum(const real (*s)[SW], int cx, int cy, real &sx, real &sy)
{
    static_assert(!kOffset<real>, "FP64 only");
    sx = (real)0;
    sy = (real)0;
#pragma unroll
    for (int j = 0; j < 25; ++j) {
        const int dx = j % 5 - 2, dy = j / 5 - 2;
        if (dx == 0 && dy == 0) continue;
        const real pp = (real)p25(dx * dx + dy * dy) * s[cy + dy][cx + dx];
        if (dx != 0) sx += pp * (real)dx;
        if (dy != 0) sy += pp * (real)dy;
    }
}

// Total force on species k at the staged node (cx, cy): Eq. (8) + Eq. (9) + rho_k g.
template <typename real, int SHv>
__device__ __forceinline__ void force_at(const Lat<real> &L, const real (*srho)[SHv][SW], const real (*spsi)[SHv][SW],
                                         int k, int cx, int cy, real &Fx, real &Fy)
{
    const real psi = spsi[k][cy][cx], rho = srho[k][cy][cx];
    if constexpr (kOffset<real>) {
        // FP32: the two psi sums as one stencil with combined weights
        float msx, msy, s3x, s3y;
        const float(*sp)[SW] = spsi[k];
        vq25c<float>([&](int dy, int dx) { return sp[cy + dy][cx + dx]; }, L.cw, p25f, msx, msy);
        q9_sum<real>(srho[1 - k], cx, cy, s3x, s3y);
        vforce<float>(psi, rho, msx, msy, s3x, s3y, L.GAB, L.g[0], L.g[1], Fx, Fy);
    } else {
        real s1x, s1y, s2x, s2y, s3x, s3y;
        q9_sum<real>(spsi[k], cx, cy, s1x, s1y);
        q25_sum<real>(spsi[k], cx, cy, s2x, s2y);
        q9_sum<real>(srho[1 - k], cx, cy, s3x, s3y);
        const real G1 = L.G1, G2 = L.G2, GAB = L.GAB;
        Fx = -G1 * psi * s1x - G2 * psi * s2x - GAB * rho * s3x + rho * L.g[0];
        Fy = -G1 * psi * s1y - G2 * psi * s2y - GAB * rho * s3y + rho * L.g[1];
    }
}

// The staged pair planes as collide_site reads them: both species' forces of Eqs. (8), (9) and rho_k g, their densities, and
// the densities a push re-references with, each as an (A, B) pair.
template <int SHv>
struct PairStage {
    const float2 (*sr)[SW];
    const float2 (*sp)[SW];
    __device__ __forceinline__ float2 density2(int cy, int cx) const { return sr[cy][cx]; }
    // Eq. (8) + Eq. (9) + rho_k g, the operations of force_at on each lane
    __device__ __forceinline__ void force2(const Lat<float> &L, int cx, int cy, float2 &Fx, float2 &Fy) const
    {
        auto at_psi = [&](int dy, int dx) { return sp[cy + dy][cx + dx]; };
        auto at_rho = [&](int dy, int dx) { return sr[cy + dy][cx + dx]; };
        float2 msx, msy, s3x, s3y;
        vq25c<float2>(at_psi, L.cw, p25f, msx, msy);
        vq9<float2>(at_rho, s3x, s3y);   // lane j: sums over species j's density
        // each species is pushed by the other's density sum
        vforce<float2>(sp[cy][cx], sr[cy][cx], msx, msy, vswap(s3x), vswap(s3y), L.GAB, L.g[0], L.g[1], Fx, Fy);
    }
    template <int EX, int EY>
    __device__ __forceinline__ float2 dest(int cx, int cy) const
    {
        return sr[cy + EY][cx + EX];
    }
};

// e_i . u in the order e_x u_x + e_y u_y, zero products dropped.
template <typename real, int EX, int EY>
__device__ __forceinline__ real edot(real ux, real uy)
{
    if constexpr (EX == 0 && EY == 0) return (real)0;
    else if constexpr (EX == 0) return EY > 0 ? uy : -uy;
    else if constexpr (EY == 0) return EX > 0 ? ux : -ux;
    else return (EX > 0 ? ux : -ux) + (EY > 0 ? uy : -uy);
}

// Store the post-collision value of direction I of species k at x + e_i
// (half-way bounce-back: back to x, reversed) near an edge of the lattice.
template <int I>
__device__ __forceinline__ void push_edge(const Lat<float> &L, float *__restrict__ fn, int k, int x, int y, float v)
{
    constexpr int EX = ex9(I), EY = ey9(I);
    int xd = x + EX, yd = y + EY;
    if constexpr (EX != 0) {
        if (xd >= L.nx) xd -= L.nx;
        if (xd < 0) xd += L.nx;
    }
    int dir = I;
    if constexpr (EY != 0) {
        if (yd < 0 || yd >= L.ny) {
            if (L.walls) {       // half-way bounce-back: back to this node, reversed
                dir = opp9(I);
                xd = x;
                yd = y;
            } else {
                yd = yd < 0 ? yd + L.ny : yd - L.ny;
            }
        }
    }
    fn[(size_t)(k * 9 + dir) * L.plane + (size_t)yd * L.pitch + xd] = v;
}

// Species momentum sum_i f e_i.  FP64: direction order, zero products
// dropped.  FP32: opposite-population differences.
template <typename real>
__device__ __forceinline__ void first_moment(const real (&f)[9], real &jx, real &jy)
{
    if constexpr (!kOffset<real>) {
        jx = ((((f[1] - f[3]) + f[5]) - f[6]) - f[7]) + f[8];
        jy = ((((f[2] - f[4]) + f[5]) + f[6]) - f[7]) - f[8];
    } else {
        vfirst<float>(f, jx, jy);
    }
}

// sum_i f_i.  FP64: direction order, as fmas with the factor `one` = 1
// (lb_f64.cuh).
template <typename real>
__device__ __forceinline__ real zeroth_moment(const real (&f)[9], real one)
{
    if constexpr (!kOffset<real>) {
        const Arith64<false> A(one);
        double r = f[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) r = A.add(r, f[i]);
        return r;
    } else {
        (void)one;
        return vzeroth<float>(f);
    }
}

// ---- kernels ----------------------------------------------------------------

// Global loads of data that other blocks of the same launch may have written
// (the persistent kernel): through L2 only, never a stale L1 line.
template <bool kCG, typename real>
__device__ __forceinline__ real ldg_state(const real *p)
{
    if constexpr (kCG) return __ldcg(p);
    else return *p;
}

// rho_k = sum_i f_k,i of one tile into density copy parity^1 (FP32: R +
// sum_i h_i, R the density of the previous step in copy parity).  kPsi: psi of
// the step (FP64) as well; the observables read densities alone (with psi a
// 1000^2 lattice's pressure tensor took 1.20 ms, 1.15 without).
template <typename real, int TYv, bool kCG, bool kPsi>
__device__ __forceinline__ void density_tile(const Lat<real> *__restrict__ lats, int4 t, int parity)
{
    const Lat<real> &L = lats[t.x];
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const real *__restrict__ f = L.f[parity];
    const size_t c = (size_t)y * L.pitch + x;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        real v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = ldg_state<kCG>(&f[(size_t)(k * 9 + i) * L.plane + c]);
        real r = zeroth_moment<real>(v, L.one);
        if constexpr (kOffset<real>) r = ldg_state<kCG>(&L.rho[parity][(size_t)k * L.plane + c]) + r;
        L.rho[parity ^ 1][(size_t)k * L.plane + c] = r;
        // FP64 keeps no reference densities: copy parity holds psi, so that
        // exp() runs once per node instead of once per staged slot
        if constexpr (kPsi) L.rho[parity][(size_t)k * L.plane + c] = psi64(r, L.one, L.exp_table);
    }
}

template <typename real, int TYv, bool kPsi>
__global__ void __launch_bounds__(TX *TYv) k_density(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles,
                                                     int tile_offset, int parity)
{
    density_tile<real, TYv, false, kPsi>(lats, tiles[tile_offset + blockIdx.x], parity);
}

// Shared memory of the FP32 step kernels for a tile of height TYv: density and
// psi of the tile and its halo as (species A, species B) pairs per node, so that
// one 64-bit shared load serves both species.
template <int TYv>
struct CollideSmem {
    float2 sr[TYv + 2 * HALO][SW];
    float2 sp[TYv + 2 * HALO][SW];
    Lat<float> L;   // descriptor copy: stores to the populations cannot alias it
    __device__ __forceinline__ void put(int sy, int sx, float rA, float rB)
    {
        sr[sy][sx] = make_float2(rA, rB);
        sp[sy][sx] = make_float2(psi_of<float>(rA), psi_of<float>(rB));
    }
};

// Moments of a node's FP32 offset populations that need no force, as
// (species A, species B) pairs: the first moment, the density change rho - R
// moved into the offsets and the offsets' residual sum dg after it
// (collide_site explains both).
struct NodeMoments {
    float2 jx, jy;
    float2 delta;
    float2 dg;
};

// The NodeMoments of a node from its offset populations h (both species as
// pairs), rho its densities and Rn its references: the same operations, in
// the same order, as collide_site's own.
__device__ __forceinline__ void node_moments(const float2 (&h)[9], float2 rho, float2 Rn, NodeMoments &nm)
{
    float2 f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = h[i];
    vfirst<float2>(f, nm.jx, nm.jy);
    nm.delta = vsub(rho, Rn);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = cfma(-(float)w9(i), nm.delta, f[i]);
    nm.dg = vzeroth<float2>(f);
}

// ---- velocity-shift forcing of the original model (FP64 only) ---------------

// Second-order equilibrium of direction I (Eq. 2), the operations of relax64.
template <typename real, int I>
__device__ __forceinline__ real feq_dir(real rho, real ux, real uy, real uu)
{
    constexpr int EX = ex9(I), EY = ey9(I);
    const real eu = edot<real, EX, EY>(ux, uy);
    return (real)w9(I) * rho * ((real)1 + (real)3 * eu + (real)4.5 * eu * eu - (real)1.5 * uu);
}

// Force, moments, u^eq, collision and push of the node (x, y), staged at
// (cx, cy).  Its populations are fk (updated in place), or with kBox
// the shared-memory box: box[(k * 9 + i) * box_plane] is population i of
// species k, read again where it is used with the same density offset
// applied, which keeps 18 registers free; fk is then not used, and the
// force-free moments come precomputed in *pre (node_moments).
// The FP32 node collision: half-force momenta (Eq. 6), the offsets from the
// node's current density, u^eq and the terms shared by the directions, then
// the collision of each direction of both species and its push.
template <bool kInner, bool kBox = false, class Stage>
__device__ __forceinline__ void collide_site(const Lat<float> &L, float *__restrict__ fn, const Stage &sg,
                                             float (&fk)[2][9], const float (&Rn)[2], int x, int y, int cx, int cy,
                                             const float *__restrict__ box = nullptr, int box_plane = 0,
                                             const NodeMoments *pre = nullptr)
{
    // both species at once, as (A, B) pairs
    float2 Fx, Fy, jx, jy, delta, dg;
    sg.force2(L, cx, cy, Fx, Fy);
    const float2 rho = sg.density2(cy, cx);
    float2 h[9];
    if constexpr (kBox) {
        (void)fk;
        (void)Rn;
        jx = pre->jx;
        jy = pre->jy;
        delta = pre->delta;
        dg = pre->dg;
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = make_float2(fk[0][i], fk[1][i]);
        vfirst<float2>(h, jx, jy);   // the reference density adds no momentum
        // offsets from the node's current density: h_i - w_i (rho - R).
        // rho - R is formed from the rounded density itself (exact: the two
        // are close), so f = h + w R is kept exactly whatever rho rounded to;
        // with sum_i h_i instead, density changes below half an ulp of R
        // would be dropped at every step and mass would drift.
        delta = vsub(rho, make_float2(Rn[0], Rn[1]));
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = cfma(-(float)w9(i), delta, h[i]);
        dg = vzeroth<float2>(h);
    }
    const float2 mx = cfma(0.5f, Fx, jx);   // Eq. (6), half force
    const float2 my = cfma(0.5f, Fy, jy);
    // the lattice constants of the collision, read once: stores to the
    // populations may alias shared memory as far as the compiler knows
    const float2 om = make_float2(L.omega[0], L.omega[1]);
    const float2 aw3[3] = {make_float2(L.aw3[0][0], L.aw3[1][0]), make_float2(L.aw3[0][1], L.aw3[1][1]),
                           make_float2(L.aw3[0][2], L.aw3[1][2])};
    OffTerms t;
    off_terms(om, rho, mx, my, Fx, Fy, dg, t);
    const size_t plane = L.plane;
    const int pitch = L.pitch;
    float *node = fn + ((size_t)y * pitch + x);
    // the populations of direction I, as the moments saw them
    auto pop = [&](int I) -> float2 {
        if constexpr (kBox)
            return cfma(-(float)w9(I), delta, make_float2(box[I * box_plane], box[(9 + I) * box_plane]));
        else return h[I];
    };
    auto dir = [&](auto Ic) {
        constexpr int I = decltype(Ic)::value;
        float2 v = off_collide<I>(t, om, aw3[cls9(I)], pop(I));
        // re-reference from rho(x) to rho(x + e_i), the reference the next
        // step reads there (not for a push that bounces back from a wall)
        constexpr int EX = ex9(I), EY = ey9(I);
        if constexpr (I != 0) {
            if (kInner || !(EY != 0 && L.walls && (y + EY < 0 || y + EY >= L.ny)))
                v = cfma((float)w9(I), vsub(rho, sg.template dest<EX, EY>(cx, cy)), v);
        }
        if constexpr (kInner) {
            // destination inside the lattice: a constant offset
            node[(size_t)I * plane + (EY * pitch + EX)] = v.x;
            node[(size_t)(9 + I) * plane + (EY * pitch + EX)] = v.y;
        } else {
            push_edge<I>(L, fn, 0, x, y, v.x);
            push_edge<I>(L, fn, 1, x, y, v.y);
        }
    };
    dir(std::integral_constant<int, 0>{});
    dir(std::integral_constant<int, 1>{});
    dir(std::integral_constant<int, 2>{});
    dir(std::integral_constant<int, 3>{});
    dir(std::integral_constant<int, 4>{});
    dir(std::integral_constant<int, 5>{});
    dir(std::integral_constant<int, 6>{});
    dir(std::integral_constant<int, 7>{});
    dir(std::integral_constant<int, 8>{});
}

template <typename real>
__device__ __forceinline__ bool slot_node(const Lat<real> &G, int4 t, int sx, int sy, int &gx, int &gy);

// Fused force + collision + push-streaming + bounce-back for one tile.  Every
// thread of the block calls it and returns from it; it ends after the tile's
// pushes are issued (the caller synchronises before reusing sm).
template <int TYv, bool kCG>
__device__ __forceinline__ void collide_tile(const Lat<float> *__restrict__ lats, int4 t, int parity,
                                             CollideSmem<TYv> &sm)
{
    const Lat<float> &G = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    static_assert(sizeof(Lat<float>) % 4 == 0, "descriptor copied as 32-bit words");
    for (int i = tid; i < (int)(sizeof(Lat<float>) / 4); i += TX * TYv)
        reinterpret_cast<uint32_t *>(&sm.L)[i] = reinterpret_cast<const uint32_t *>(&G)[i];
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    const bool valid = x < G.nx && y < G.ny;
    // issue the population loads first so their latency overlaps the staging
    const float *__restrict__ fc = G.f[parity];
    float *__restrict__ fn = G.f[parity ^ 1];
    const size_t c = valid ? (size_t)y * G.pitch + x : 0;
    float fk[2][9];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < 9; ++i) fk[k][i] = valid ? ldg_state<kCG>(&fc[(size_t)(k * 9 + i) * G.plane + c]) : (float)0;
    constexpr int SHv = TYv + 2 * HALO, kSlots = (SW * SHv + TX * TYv - 1) / (TX * TYv);
    const float *__restrict__ rho = G.rho[parity ^ 1];
    // all of the thread's slots loaded before the first is staged (128 x 5 in tiles of
    // 4, LB_MODE_PERSISTENT: 9.2 us a step one after the other, 8.8 so)
    float2 r[kSlots];
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
        const int idx = tid + q * TX * TYv;
        if (idx >= SW * SHv) break;
        int gx, gy;
        r[q] = make_float2(G.wall_rho[0], G.wall_rho[1]);
        if (slot_node(G, t, idx % SW, idx / SW, gx, gy)) {
            const size_t cc = (size_t)gy * G.pitch + gx;
            r[q] = make_float2(ldg_state<kCG>(&rho[cc]), ldg_state<kCG>(&rho[G.plane + cc]));
        }
    }
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
        const int idx = tid + q * TX * TYv;
        if (idx < SW * SHv) sm.put(idx / SW, idx % SW, r[q].x, r[q].y);
    }
    __syncthreads();
    if (!valid) return;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    float Rn[2] = {(float)0, (float)0};
    Rn[0] = ldg_state<kCG>(&G.rho[parity][c]);
    Rn[1] = ldg_state<kCG>(&G.rho[parity][G.plane + c]);
    // tiles whose pushes stay inside the lattice (no wrap, no wall) take constant offsets
    const bool inner = t.y >= 1 && t.y + TX + 1 <= sm.L.nx && t.z >= 1 && t.z + TYv + 1 <= sm.L.ny;
    const PairStage<TYv + 2 * HALO> sg{sm.sr, sm.sp};
    if (inner) collide_site<true>(sm.L, fn, sg, fk, Rn, x, y, cx, cy);
    else collide_site<false>(sm.L, fn, sg, fk, Rn, x, y, cx, cy);
}

// ---- the FP64 node ----------------------------------------------------------

// What the FP64 step stages per slot and species: density, psi, and every
// product with a stencil weight that a neighbour's sums take from the slot.
// The sums of Eqs. (8), (9) use 40 such products per node and species, of
// which only these 9 per slot differ (2 p5 psi is p5 psi doubled, exactly).
enum Plane64 { sRho = 0, sPsi, sW1Psi, sW2Psi, sP1, sP2, s2P4, sP5, s2P8, sW1Rho, sW2Rho, kPlanes64 };

template <int TYv>
struct Stage64 {
    double v[2][kPlanes64][TYv + 2 * HALO][SW];
    Lat<double> L;   // descriptor copy: stores to the populations cannot alias it

    // density and psi of species k at a slot, and the slot's products;
    // nonzero where one lies outside the range of the integer products
    __device__ __forceinline__ uint32_t put(int k, int sy, int sx, double r, double p)
    {
        double(*q)[TYv + 2 * HALO][SW] = v[k];
        q[sRho][sy][sx] = r;
        q[sPsi][sy][sx] = p;
        const uint32_t outside = base_outside(r) | base_outside(p);
        if (outside) {
            q[sW1Psi][sy][sx] = (1.0 / 9.0) * p;
            q[sW2Psi][sy][sx] = (1.0 / 36.0) * p;
            q[sP1][sy][sx] = p25(1) * p;
            q[sP2][sy][sx] = p25(2) * p;
            q[s2P4][sy][sx] = (2.0 * p25(4)) * p;
            q[sP5][sy][sx] = p25(5) * p;
            q[s2P8][sy][sx] = (2.0 * p25(8)) * p;
            q[sW1Rho][sy][sx] = (1.0 / 9.0) * r;
            q[sW2Rho][sy][sx] = (1.0 / 36.0) * r;
            return outside;
        }
        const Factor fp = factor(p), fr = factor(r);
        q[sW1Psi][sy][sx] = factor_mul(fp, factor(1.0 / 9.0));
        q[sW2Psi][sy][sx] = factor_mul(fp, factor(1.0 / 36.0));
        q[sP1][sy][sx] = factor_mul(fp, factor(p25(1)));
        q[sP2][sy][sx] = factor_mul(fp, factor(p25(2)));
        q[s2P4][sy][sx] = factor_mul(fp, factor(2.0 * p25(4)));
        q[sP5][sy][sx] = factor_mul(fp, factor(p25(5)));
        q[s2P8][sy][sx] = factor_mul(fp, factor(2.0 * p25(8)));
        q[sW1Rho][sy][sx] = factor_mul(fr, factor(1.0 / 9.0));
        q[sW2Rho][sy][sx] = factor_mul(fr, factor(1.0 / 36.0));
        return 0;
    }
};

// Component AX (0: x, 1: y) of the total force on species k at the staged
// node, Eq. (8) + Eq. (9) + rho_k g: the sums in direction order (D2Q9) and
// raster order (D2Q25), as q9_sum and q25_sum form them, from the staged
// products.
template <int AX, bool kInt, int TYv>
__device__ __forceinline__ double force64(const Arith64<kInt> &A, const Stage64<TYv> &sm, int k, int cx, int cy)
{
    const double(*q)[TYv + 2 * HALO][SW] = sm.v[k];
    const double(*o)[TYv + 2 * HALO][SW] = sm.v[1 - k];
    auto signed_add = [&](double s, double t, int e) { return e > 0 ? A.add(s, t) : A.sub(s, t); };
    // D2Q9: the axis pair, then the diagonals in direction order
    auto q9 = [&](const double(*f)[TYv + 2 * HALO][SW], int w1, int w2) {
        double s = AX == 0 ? A.sub(f[w1][cy][cx + 1], f[w1][cy][cx - 1]) : A.sub(f[w1][cy + 1][cx], f[w1][cy - 1][cx]);
#pragma unroll
        for (int i = 5; i < 9; ++i) s = signed_add(s, f[w2][cy + ey9(i)][cx + ex9(i)], AX == 0 ? ex9(i) : ey9(i));
        return s;
    };
    const double s1 = q9(q, sW1Psi, sW2Psi), s3 = q9(o, sW1Rho, sW2Rho);
    // D2Q25: the planes of |e|^2 = 4, 8 hold 2 p psi, the component being +-2
    const double two = A.one + A.one;
    double s2 = 0.0;
#pragma unroll
    for (int j = 0; j < 25; ++j) {
        const int dx = j % 5 - 2, dy = j / 5 - 2, e2 = dx * dx + dy * dy, e = AX == 0 ? dx : dy;
        if (e == 0) continue;
        const int plane = e2 == 1 ? sP1 : e2 == 2 ? sP2 : e2 == 4 ? s2P4 : e2 == 5 ? sP5 : s2P8;
        const double t = q[plane][cy + dy][cx + dx];
        if (j == 0) s2 = -t;
        else if (e2 == 5 && (e == 2 || e == -2)) s2 = __fma_rn(e > 0 ? t : -t, two, s2);
        else s2 = signed_add(s2, t, e);
    }
    const double psi = q[sPsi][cy][cx], rho = q[sRho][cy][cx];
    double F = A.sub(A.sub(A.mul(A.mul(-sm.L.G1, psi), s1), A.mul(A.mul(sm.L.G2, psi), s2)),
                     A.mul(A.mul(sm.L.GAB, rho), s3));
    // + rho g; a zero component adds nothing to a finite force
    if (!kInt || sm.L.g[AX] != 0.0) F = A.add(F, A.mul(rho, sm.L.g[AX]));
    return F;
}

// Where the node's pushes go: element offsets to its neighbours, and whether
// a vertical push meets a wall.
struct Push64 {
    long long oE, oW, oN, oS;
    bool wallN, wallS;
    __device__ __forceinline__ Push64(const Lat<double> &L, int x, int y)
    {
        oE = x + 1 < L.nx ? 1 : 1 - L.nx;
        oW = x > 0 ? -1 : L.nx - 1;
        oN = y + 1 < L.ny ? (long long)L.pitch : -(long long)L.pitch * (L.ny - 1);
        oS = y > 0 ? -(long long)L.pitch : (long long)L.pitch * (L.ny - 1);
        wallN = L.walls && y + 1 >= L.ny;
        wallS = L.walls && y <= 0;
    }
    // store v, the post-collision value of direction I of the species whose
    // population planes at the node start at fk (half-way bounce-back at walls)
    template <int I>
    __device__ __forceinline__ void store(double *__restrict__ fk, size_t plane, double v) const
    {
        constexpr int EX = ex9(I), EY = ey9(I);
        long long off = (EX > 0 ? oE : EX < 0 ? oW : 0) + (EY > 0 ? oN : EY < 0 ? oS : 0);
        int dir = I;
        if constexpr (EY != 0)
            if (EY > 0 ? wallN : wallS) {
                dir = opp9(I);
                off = 0;
            }
        fk[(long long)((size_t)dir * plane) + off] = v;
    }
};

// What the directions of the collision share: the velocity's terms of the Guo
// vectors (e - u)/cs^2 + (e.u) e/cs^4 and of the equilibrium polynomial.
// Opposite directions' e.u differ by an exact sign.
template <bool kInt>
struct Dirs64 {
    double e[4];            // e.u of directions 1, 2, 5, 8
    double uu15;            // 1.5 u.u
    double g0[2];           // -3 u
    double gp[2], gm[2];    // 3 (1 - u), 3 (-1 - u)
    __device__ __forceinline__ Dirs64(const Arith64<kInt> &A, double ux, double uy)
        : e{ux, uy, A.add(ux, uy), A.sub(ux, uy)}, uu15(A.mul(1.5, A.add(A.mul(ux, ux), A.mul(uy, uy)))),
          g0{-A.mul(3.0, ux), -A.mul(3.0, uy)}, gp{A.mul(3.0, A.sub(1.0, ux)), A.mul(3.0, A.sub(1.0, uy))},
          gm{A.mul(3.0, A.sub(-1.0, ux)), A.mul(3.0, A.sub(-1.0, uy))}
    {
    }
    // Guo vector and 1 + 3 e.u + 4.5 (e.u)^2 - 1.5 u.u of direction I
    template <int I>
    __device__ __forceinline__ void terms(const Arith64<kInt> &A, double (&g)[2], double &po) const
    {
        if constexpr (I == 0) {
            g[0] = g0[0];
            g[1] = g0[1];
            po = A.sub(1.0, uu15);
        } else {
            constexpr int B = vbase9(I), S = vsign9(I) > 0 ? 1 : -1, E[2] = {ex9(I), ey9(I)};   // e.u = S e[B]
            const double e9 = A.mul(9.0, e[B]), e3 = A.mul(3.0, e[B]);
#pragma unroll
            for (int a = 0; a < 2; ++a)
                g[a] = E[a] == 0 ? g0[a]
                                 : (E[a] * S > 0 ? A.add(E[a] > 0 ? gp[a] : gm[a], e9)
                                                 : A.sub(E[a] > 0 ? gp[a] : gm[a], e9));
            const double lin = S > 0 ? A.add(1.0, e3) : A.sub(1.0, e3);
            po = A.sub(A.add(lin, A.mul(A.mul(4.5, e[B]), e[B])), uu15);
        }
    }
};

// Post-collision value of direction I of one species (Eqs. 1, 2, 5):
// f - omega (f - feq) + C, feq = w rho po, C = (1 - omega/2) w (g . F).
template <int I, bool kInt>
__device__ __forceinline__ double relax64(const Arith64<kInt> &A, double f, double wrho, double om, double aw,
                                          const double (&g)[2], double po, double Fx, double Fy)
{
    const double C = A.mul(aw, A.add(A.mul(g[0], Fx), A.mul(g[1], Fy)));
    return A.add(A.sub(f, A.mul(om, A.sub(f, A.mul(wrho, po)))), C);
}

// Force, half-force momenta, u^eq, collision with the Guo term and push of
// both species at node (x, y), staged at (cx, cy): Eqs. (1)-(3), (5), (6),
// (8), (9), each operation rounded once, in the oracle's order.  j: the
// species' momenta sum_i f e_i; fc, fn: the node's first population plane in
// the current and the next copy.  Returns whether a value lay outside the
// range the integer products cover (lb_f64.cuh; the caller then redoes the
// node with kInt = false).
template <bool kInt, int TYv, bool kCG>
__device__ __forceinline__ bool node64(const Stage64<TYv> &sm, double one, const double *__restrict__ fc,
                                       double *__restrict__ fn, const double (&j)[2][2], int x, int y, int cx, int cy)
{
    const Arith64<kInt> A(one);
    const Lat<double> &L = sm.L;
    const size_t plane = L.plane;
    uint32_t outside = 0;
    double F[2][2], m[2][2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        F[k][0] = force64<0, kInt, TYv>(A, sm, k, cx, cy);
        F[k][1] = force64<1, kInt, TYv>(A, sm, k, cx, cy);
#pragma unroll
        for (int a = 0; a < 2; ++a) m[k][a] = __fma_rn(0.5, F[k][a], j[k][a]);   // Eq. (6): F/2 is exact
    }
    const double r0 = sm.v[0][sRho][cy][cx], r1 = sm.v[1][sRho][cy][cx];
    const double om0 = L.omega[0], om1 = L.omega[1];
    const double den = A.add(A.mul(om0, r0), A.mul(om1, r1));
    const double nx = A.add(A.mul(om0, m[0][0]), A.mul(om1, m[1][0]));
    const double ny = A.add(A.mul(om0, m[0][1]), A.mul(om1, m[1][1]));
    double ux, uy;
    if constexpr (kInt) {
        const double rden = __drcp_rn(den);
        ux = quotient64(nx, den, rden);
        uy = quotient64(ny, den, rden);
        outside = velocity_outside(ux) | velocity_outside(uy);
    } else {
        ux = nx / den;
        uy = ny / den;
    }
    const Dirs64<kInt> dirs(A, ux, uy);
    const Push64 push(L, x, y);
    const double wr[2][3] = {{A.mul(4.0 / 9.0, r0), A.mul(1.0 / 9.0, r0), A.mul(1.0 / 36.0, r0)},
                             {A.mul(4.0 / 9.0, r1), A.mul(1.0 / 9.0, r1), A.mul(1.0 / 36.0, r1)}};
    // a direction of both species at once: its terms live no longer than it
    // does, and its populations are read again where they are used
    auto dir = [&](auto Ic) {
        constexpr int I = decltype(Ic)::value, c = cls9(I);
        double g[2], po;
        dirs.template terms<I>(A, g, po);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double f = ldg_state<kCG>(&fc[(size_t)(k * 9 + I) * plane]);
            if constexpr (kInt) outside |= base_outside(f);
            push.store<I>(fn + (size_t)(k * 9) * plane, plane,
                          relax64<I>(A, f, wr[k][c], k ? om1 : om0, L.aw[k][c], g, po, F[k][0], F[k][1]));
        }
    };
    // opposite directions in turn: they share the products with e.u
    dir(std::integral_constant<int, 0>{});
    dir(std::integral_constant<int, 1>{});
    dir(std::integral_constant<int, 3>{});
    dir(std::integral_constant<int, 2>{});
    dir(std::integral_constant<int, 4>{});
    dir(std::integral_constant<int, 5>{});
    dir(std::integral_constant<int, 7>{});
    dir(std::integral_constant<int, 6>{});
    dir(std::integral_constant<int, 8>{});
    return outside != 0;
}

// The species' momenta sum_i f e_i of a node.
struct Mom64 {
    double j[2][2];
};

// The velocity-shift node (Eq. 4) on the staged planes.
template <int TYv, bool kCG>
__device__ __noinline__ void shift_node64(const Stage64<TYv> &sm, double one, const double *__restrict__ fc,
                                          double *__restrict__ fn, Mom64 jj, int x, int y, int cx, int cy)
{
    const double(&j)[2][2] = jj.j;
    const Lat<double> &L = sm.L;
    const Arith64<false> A(one);
    double F[2][2], rho[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        F[k][0] = force64<0, false, TYv>(A, sm, k, cx, cy);
        F[k][1] = force64<1, false, TYv>(A, sm, k, cx, cy);
        rho[k] = sm.v[k][sRho][cy][cx];
    }
    const double om0 = L.omega[0], om1 = L.omega[1];
    const double den = om0 * rho[0] + om1 * rho[1];
    const double ux = (om0 * j[0][0] + om1 * j[1][0]) / den;
    const double uy = (om0 * j[0][1] + om1 * j[1][1]) / den;
    const double uu = ux * ux + uy * uy;
    const Push64 push(L, x, y);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double sx = ux + L.tau[k] * F[k][0] / rho[k], sy = uy + L.tau[k] * F[k][1] / rho[k];
        const double ss = sx * sx + sy * sy, om = L.omega[k];
        // relaxation to f^eq(rho, u^eq) plus (1/tau) [f^eq(rho, u^eq + tau F / rho) - f^eq(rho, u^eq)]
        auto dir = [&](auto Ic) {
            constexpr int I = decltype(Ic)::value;
            const double f = ldg_state<kCG>(&fc[(size_t)(k * 9 + I) * L.plane]);
            const double feq = feq_dir<double, I>(rho[k], ux, uy, uu), feqs = feq_dir<double, I>(rho[k], sx, sy, ss);
            push.store<I>(fn + (size_t)(k * 9) * L.plane, L.plane, f - om * (f - feq) + om * (feqs - feq));
        };
        dir(std::integral_constant<int, 0>{});
        dir(std::integral_constant<int, 1>{});
        dir(std::integral_constant<int, 2>{});
        dir(std::integral_constant<int, 3>{});
        dir(std::integral_constant<int, 4>{});
        dir(std::integral_constant<int, 5>{});
        dir(std::integral_constant<int, 6>{});
        dir(std::integral_constant<int, 7>{});
        dir(std::integral_constant<int, 8>{});
    }
}

template <int TYv, bool kCG>
__device__ __noinline__ void plain_node64(const Stage64<TYv> &sm, double one, const double *__restrict__ fc,
                                          double *__restrict__ fn, Mom64 j, int x, int y, int cx, int cy)
{
    node64<false, TYv, kCG>(sm, one, fc, fn, j.j, x, y, cx, cy);
}

// The node's step after staging, in the lattice's forcing; plain: a staged
// value of the block lies outside the range of the integer products.
template <int TYv, bool kCG>
__device__ __forceinline__ void finish64(const Stage64<TYv> &sm, const double *__restrict__ fc, double *__restrict__ fn,
                                         const Mom64 &j, int x, int y, int cx, int cy, bool plain)
{
    const double one = sm.L.one;
    if (sm.L.forcing == 1) {   // the original model (Eq. 4), a block-uniform branch
        shift_node64<TYv, kCG>(sm, one, fc, fn, j, x, y, cx, cy);
        return;
    }
    if (plain || !sm.L.products || node64<true, TYv, kCG>(sm, one, fc, fn, j.j, x, y, cx, cy))
        plain_node64<TYv, kCG>(sm, one, fc, fn, j, x, y, cx, cy);
}

// ---- one-pass step ------------------------------------------------------------

// Density of node (gx, gy) straight from its populations (FP32: plus its
// reference density): the same sum, in the same order, as the density pass.
template <typename real, bool kCG>
__device__ __forceinline__ real node_density(const Lat<real> &L, int k, int gx, int gy, int parity)
{
    const size_t c = (size_t)gy * L.pitch + gx;
    const real *__restrict__ f = L.f[parity];
    real v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = ldg_state<kCG>(&f[(size_t)(k * 9 + i) * L.plane + c]);
    real r = zeroth_moment<real>(v, L.one);
    if constexpr (kOffset<real>) r = ldg_state<kCG>(&L.rho[parity][(size_t)k * L.plane + c]) + r;
    return r;
}

// The node whose densities staged slot (sx, sy) of tile t holds (slot (HALO,
// HALO) is the tile's first node): x wraps; beyond the lattice in y, periodic
// wrap, or a wall ghost row (the mirrored fluid row, or, returning false, the
// fixed wall densities).
template <typename real>
__device__ __forceinline__ bool slot_node(const Lat<real> &G, int4 t, int sx, int sy, int &gx, int &gy)
{
    gx = t.y + sx - HALO;
    gx = kOffset<real> ? wrap_index(gx, G.nx) : wrap_column64(gx, G.nx);
    gy = t.z + sy - HALO;
    if (gy < 0 || gy >= G.ny) {
        if (!G.walls) {
            gy = wrap_index(gy, G.ny);
        } else if (G.wall_mode == 1) {
            return false;
        } else {
            gy = gy < 0 ? -1 - gy : 2 * G.ny - 1 - gy;
            gy = gy < 0 ? 0 : (gy >= G.ny ? G.ny - 1 : gy);  // rows no valid node reads
        }
    }
    return true;
}

// Density of species k at a staged slot from the populations of its node.
template <typename real, bool kCG>
__device__ __forceinline__ real slot_density(const Lat<real> &G, int4 t, int parity, int sx, int sy, int k)
{
    int gx, gy;
    return slot_node(G, t, sx, sy, gx, gy) ? node_density<real, kCG>(G, k, gx, gy, parity) : G.wall_rho[k];
}

// Both species' densities at a staged slot (FP32: as a pair, lane by lane the
// sums of node_density).
template <typename real, bool kCG>
__device__ __forceinline__ void slot_densities(const Lat<real> &G, int4 t, int parity, int sx, int sy, real &rA,
                                               real &rB)
{
    int gx, gy;
    if (!slot_node(G, t, sx, sy, gx, gy)) {
        rA = G.wall_rho[0];
        rB = G.wall_rho[1];
        return;
    }
    if constexpr (kOffset<real>) {
        const size_t c = (size_t)gy * G.pitch + gx;
        const real *__restrict__ f = G.f[parity], *__restrict__ R = G.rho[parity];
        float2 v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            v[i] = make_float2(ldg_state<kCG>(&f[(size_t)i * G.plane + c]), ldg_state<kCG>(&f[(size_t)(9 + i) * G.plane + c]));
        const float2 r = vadd(make_float2(ldg_state<kCG>(&R[c]), ldg_state<kCG>(&R[G.plane + c])), vzeroth<float2>(v));
        rA = r.x;
        rB = r.y;
    } else {
        rA = node_density<real, kCG>(G, 0, gx, gy, parity);
        rB = node_density<real, kCG>(G, 1, gx, gy, parity);
    }
}

// Staged slot (sx, sy) of the h-th position of a tile's halo ring, enumerated
// compactly: two rows above, two below, then the two columns on each side of
// the tile's rows.
template <int TYv>
constexpr int kRing = 4 * SW + 4 * TYv;
template <int TYv>
__device__ __forceinline__ void ring_slot(int h, int &sx, int &sy)
{
    if (h < 2 * SW) {
        sy = h / SW;
        sx = h % SW;
    } else if (h < 4 * SW) {
        sy = TYv + HALO + (h - 2 * SW) / SW;
        sx = (h - 2 * SW) % SW;
    } else {
        const int q = h - 4 * SW;
        sy = HALO + q / 4;
        sx = (q % 4 < 2) ? q % 4 : TX + q % 4;
    }
}

// The same, staged with psi into the tile's density and psi planes.
template <int TYv, bool kCG>
__device__ __forceinline__ void stage_slot(const Lat<float> &G, int4 t, int parity, CollideSmem<TYv> &sm, int sx,
                                           int sy)
{
    float rA, rB;
    slot_densities<float, kCG>(G, t, parity, sx, sy, rA, rB);
    sm.put(sy, sx, rA, rB);
}

// One time step of one tile in a single pass: each thread forms its node's
// densities from the populations it loads anyway; the 2-node halo (and the
// slots of a ragged tile's missing nodes) is formed from the neighbours'
// populations, mostly L2 hits.  The halo goes first, so that its loads and
// the node's own 18 populations are not held in registers at the same time.
// It writes the node's density as the next step's reference.  Then the
// fused force + collision + push of collide_site.
template <int TYv, bool kCG>
__device__ __forceinline__ void fused_tile(const Lat<float> *__restrict__ lats, int4 t, int parity,
                                           CollideSmem<TYv> &sm)
{
    constexpr int SHv = TYv + 2 * HALO;
    const Lat<float> &G = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    for (int i = tid; i < (int)(sizeof(Lat<float>) / 4); i += TX * TYv)
        reinterpret_cast<uint32_t *>(&sm.L)[i] = reinterpret_cast<const uint32_t *>(&G)[i];
    const int nx = G.nx, ny = G.ny;
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    const bool valid = x < nx && y < ny;
    const float *__restrict__ fc = G.f[parity];
    float *__restrict__ fn = G.f[parity ^ 1];
    const size_t c = valid ? (size_t)y * G.pitch + x : 0;
    // a ragged tile's nodes read no slot further than HALO beyond its last one
    const int ex = nx - t.y + 2 * HALO, ey = ny - t.z + 2 * HALO;
    for (int h = tid; h < kRing<TYv>; h += TX * TYv) {
        int sx, sy;
        ring_slot<TYv>(h, sx, sy);
        if (sx < ex && sy < ey) stage_slot<TYv, kCG>(G, t, parity, sm, sx, sy);
    }
    // and those without a node of their own among the tile's hold wrapped copies
    if (!valid && (int)threadIdx.x + HALO < ex && (int)threadIdx.y + HALO < ey)
        stage_slot<TYv, kCG>(G, t, parity, sm, threadIdx.x + HALO, threadIdx.y + HALO);
    // then the node's own populations (kept in registers for the collision)
    float fk[2][9];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < 9; ++i) fk[k][i] = valid ? ldg_state<kCG>(&fc[(size_t)(k * 9 + i) * G.plane + c]) : (float)0;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    float Rn[2] = {(float)0, (float)0};
    if (valid) {
        float2 v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = make_float2(fk[0][i], fk[1][i]);
#pragma unroll
        for (int k = 0; k < 2; ++k) Rn[k] = ldg_state<kCG>(&G.rho[parity][(size_t)k * G.plane + c]);
        const float2 r = vadd(make_float2(Rn[0], Rn[1]), vzeroth<float2>(v));
        G.rho[parity ^ 1][c] = r.x;
        G.rho[parity ^ 1][G.plane + c] = r.y;
        sm.put(cy, cx, r.x, r.y);
    }
    __syncthreads();
    if (!valid) return;
    const bool inner = t.y >= 1 && t.y + TX + 1 <= sm.L.nx && t.z >= 1 && t.z + TYv + 1 <= sm.L.ny;
    const PairStage<SHv> sg{sm.sr, sm.sp};
    if (inner) collide_site<true>(sm.L, fn, sg, fk, Rn, x, y, cx, cy);
    else collide_site<false>(sm.L, fn, sg, fk, Rn, x, y, cx, cy);
}

// ---- the FP64 tiles -------------------------------------------------------------

template <int TYv>
__device__ __forceinline__ void copy_lat64(Stage64<TYv> &sm, const Lat<double> &G, int tid)
{
    for (int i = tid; i < (int)(sizeof(Lat<double>) / 4); i += TX * TYv)
        reinterpret_cast<uint32_t *>(&sm.L)[i] = reinterpret_cast<const uint32_t *>(&G)[i];
}

// First moments of the node's populations (direction order).
template <bool kCG>
__device__ __forceinline__ void node_moments64(const double *__restrict__ fc, size_t plane, double one, Mom64 &m,
                                               double (*rho)[2])
{
    const Arith64<false> A(one);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        double f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = ldg_state<kCG>(&fc[(size_t)(k * 9 + i) * plane]);
        m.j[k][0] = A.add(A.sub(A.sub(A.add(A.sub(f[1], f[3]), f[5]), f[6]), f[7]), f[8]);
        m.j[k][1] = A.sub(A.sub(A.add(A.add(A.sub(f[2], f[4]), f[5]), f[6]), f[7]), f[8]);
        if (rho) {
            (*rho)[k] = zeroth_moment<double>(f, one);
        }
    }
}

// The fused kernel of the two-pass step in FP64: stages the densities and psi
// the density pass wrote, then the node.
template <int TYv, bool kCG>
__device__ __forceinline__ void collide_tile64(const Lat<double> *__restrict__ lats, int4 t, int parity,
                                               Stage64<TYv> &sm)
{
    constexpr int SHv = TYv + 2 * HALO;
    const Lat<double> &G = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    copy_lat64<TYv>(sm, G, tid);
    const int nx = G.nx, ny = G.ny;
    const bool inner = t.y >= HALO && t.y + TX + HALO <= nx && t.z >= HALO && t.z + TYv + HALO <= ny;
    const double *__restrict__ rho = G.rho[parity ^ 1], *__restrict__ psi = G.rho[parity];
    uint32_t outside = 0;
    for (int idx = tid; idx < SW * SHv; idx += TX * TYv) {
        const int sx = idx % SW, sy = idx / SW;
        int gx = t.y + sx - HALO, gy = t.z + sy - HALO;
        bool fixed = false;
        if (!inner) {
            gx = wrap_index(gx, nx);
            if (gy < 0 || gy >= ny) {
                if (!G.walls) {
                    gy = wrap_index(gy, ny);
                } else if (G.wall_mode == 1) {
                    fixed = true;
                } else {
                    gy = gy < 0 ? -1 - gy : 2 * ny - 1 - gy;
                    gy = gy < 0 ? 0 : (gy >= ny ? ny - 1 : gy);  // rows no valid node reads
                }
            }
        }
        const size_t c = (size_t)gy * G.pitch + gx;
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
            const double r = fixed ? G.wall_rho[k] : ldg_state<kCG>(&rho[(size_t)k * G.plane + c]);
            const double p = fixed ? psi64(r, G.one, G.exp_table) : ldg_state<kCG>(&psi[(size_t)k * G.plane + c]);
            outside |= sm.put(k, sy, sx, r, p);
        }
    }
    const bool plain = __syncthreads_or(outside != 0);
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const size_t c = (size_t)y * sm.L.pitch + x;
    const double *__restrict__ fc = sm.L.f[parity] + c;
    Mom64 m;
    node_moments64<kCG>(fc, sm.L.plane, sm.L.one, m, nullptr);
    finish64<TYv, kCG>(sm, fc, sm.L.f[parity ^ 1] + c, m, x, y, threadIdx.x + HALO, threadIdx.y + HALO, plain);
}

// One time step of one tile in a single pass in FP64: the densities of the
// halo ring (and of a ragged tile's missing nodes) from the neighbours'
// populations, the node's own from the populations its momenta need anyway.
template <int TYv, bool kCG>
__device__ __forceinline__ void fused_tile64(const Lat<double> *__restrict__ lats, int4 t, int parity,
                                             Stage64<TYv> &sm)
{
    const Lat<double> &G = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    copy_lat64<TYv>(sm, G, tid);
    const int nx = G.nx, ny = G.ny;
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    const bool valid = x < nx && y < ny;
    const size_t c = valid ? (size_t)y * G.pitch + x : 0;
    const double *__restrict__ fc = G.f[parity] + c;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    Mom64 m;
    uint32_t outside = 0;
    // own slot first (h < 0), then the thread's ring slots
#pragma unroll 1
    for (int h = tid - TX * TYv; h < kRing<TYv>; h += TX * TYv) {
        double r[2];
        int sx = cx, sy = cy;
        if (h >= 0) ring_slot<TYv>(h, sx, sy);
        if (h < 0 && valid) node_moments64<kCG>(fc, G.plane, G.one, m, &r);
        else slot_densities<double, kCG>(G, t, parity, sx, sy, r[0], r[1]);
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
            const double rk = k ? r[1] : r[0];
            outside |= sm.put(k, sy, sx, rk, psi64(rk, G.one, G.exp_table));
        }
    }
    const bool plain = __syncthreads_or(outside != 0);
    if (!valid) return;
    finish64<TYv, kCG>(sm, fc, G.f[parity ^ 1] + c, m, x, y, cx, cy, plain);
}

// Shared memory of a step kernel: static in FP32; dynamic in FP64, whose
// planes are above the 48 KB of static shared memory.
template <typename real, int TYv>
using StepSmem = std::conditional_t<kOffset<real>, CollideSmem<TYv>, Stage64<TYv>>;
template <typename real, int TYv>
constexpr size_t kStepSmem = kOffset<real> ? 0 : sizeof(Stage64<TYv>);

extern __shared__ __align__(16) unsigned char lb_step_smem[];

template <typename real, int TYv>
__device__ __forceinline__ StepSmem<real, TYv> &step_smem()
{
    if constexpr (kOffset<real>) {
        __shared__ CollideSmem<TYv> sm;
        return sm;
    } else {
        return *reinterpret_cast<Stage64<TYv> *>(lb_step_smem);
    }
}

template <typename real, int TYv, bool kCG>
__device__ __forceinline__ void collide_any(const Lat<real> *__restrict__ lats, int4 t, int parity,
                                            StepSmem<real, TYv> &sm)
{
    if constexpr (kOffset<real>) collide_tile<TYv, kCG>(lats, t, parity, sm);
    else collide_tile64<TYv, kCG>(lats, t, parity, sm);
}

template <typename real, int TYv>
__global__ void __launch_bounds__(TX *TYv, kCollideMinBlocks<real, TYv>)
    k_collide(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles, int tile_offset, int parity)
{
    collide_any<real, TYv, false>(lats, tiles[tile_offset + blockIdx.x], parity, step_smem<real, TYv>());
}

template <typename real, int TYv>
__global__ void __launch_bounds__(TX *TYv, kCollideMinBlocks<real, TYv>)
    k_fused(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles, int tile_offset, int parity)
{
    const int4 t = tiles[tile_offset + blockIdx.x];
    auto &sm = step_smem<real, TYv>();
    if constexpr (kOffset<real>) fused_tile<TYv, false>(lats, t, parity, sm);
    else fused_tile64<TYv, false>(lats, t, parity, sm);
}

// ---- the FP64 step of small lattices ------------------------------------------
//
// One warp issues an FP64 instruction every 64 clocks, whatever its
// neighbours do (each of an SM's four schedulers has a quarter of the pipe), so
// a lattice of few nodes is bound by the instructions of one warp: 13 us of
// FP64 alone.  Here a row of 32 nodes is a block of four warps, one per
// scheduler: warp (k, a) forms component a of species k's force and momentum,
// then half a's directions of species k.  A step is this one launch; the
// densities of the row's 36 x 5 slots are formed by the block itself.  Every
// operation is that of node64.  64^2: 25.6 us a step as tiles of 32 x 4 nodes
// in two launches, 13.4 here with the products on the FP64 pipe, 12.0 with
// them in integers, which fill the 64 clocks between FP64 instructions
// (unrolling the staging loop: 14.1, its code outgrows the instruction cache),
// 10.9 with exp() by table.
constexpr int kSmallWarps = 4;

struct Small64 {
    Stage64<1> st;
    double F[2][2][TX], m[2][2][TX], u[2][TX];
};

// The populations of one species at a node.
struct Pops64 {
    double f[9];
};

// Component a of species k's force and half-force momentum (Eqs. 6, 8, 9).
template <bool kInt>
__device__ __forceinline__ void small_force(Small64 &sm, const Pops64 &p, int k, int a)
{
    const Arith64<kInt> A(sm.st.L.one);
    const int lane = threadIdx.x, cx = lane + HALO, cy = HALO;
    const double(&f)[9] = p.f;
    const double j = a == 0 ? A.add(A.sub(A.sub(A.add(A.sub(f[1], f[3]), f[5]), f[6]), f[7]), f[8])
                            : A.sub(A.sub(A.add(A.add(A.sub(f[2], f[4]), f[5]), f[6]), f[7]), f[8]);
    const double F = a == 0 ? force64<0, kInt, 1>(A, sm.st, k, cx, cy) : force64<1, kInt, 1>(A, sm.st, k, cx, cy);
    sm.F[k][a][lane] = F;
    sm.m[k][a][lane] = __fma_rn(0.5, F, j);
}

// Component a of u^eq (Eq. 3).
template <bool kInt>
__device__ __forceinline__ double small_velocity(const Small64 &sm, int a)
{
    const Arith64<kInt> A(sm.st.L.one);
    const int lane = threadIdx.x, cx = lane + HALO, cy = HALO;
    const double om0 = sm.st.L.omega[0], om1 = sm.st.L.omega[1];
    const double den = A.add(A.mul(om0, sm.st.v[0][sRho][cy][cx]), A.mul(om1, sm.st.v[1][sRho][cy][cx]));
    const double n = A.add(A.mul(om0, sm.m[0][a][lane]), A.mul(om1, sm.m[1][a][lane]));
    return n / den;
}

// Collision and push of half a's directions of species k at node (x, y):
// those along e[0] and e[2] of Dirs64 and rest, or those along e[1] and e[3].
template <bool kInt>
__device__ __forceinline__ void small_push(const Small64 &sm, const Pops64 &p, double *__restrict__ nk, int k, int a,
                                           int x, int y)
{
    const Lat<double> &L = sm.st.L;
    const Arith64<kInt> A(L.one);
    const int lane = threadIdx.x;
    const Dirs64<kInt> dirs(A, sm.u[0][lane], sm.u[1][lane]);
    const double r = sm.st.v[k][sRho][HALO][lane + HALO], om = L.omega[k], Fx = sm.F[k][0][lane], Fy = sm.F[k][1][lane];
    const Push64 push(L, x, y);
    auto dir = [&](auto Ic) {
        constexpr int I = decltype(Ic)::value;
        double g[2], po;
        dirs.template terms<I>(A, g, po);
        push.store<I>(nk, L.plane, relax64<I>(A, p.f[I], A.mul(w9(I), r), om, L.aw[k][cls9(I)], g, po, Fx, Fy));
    };
    if (a == 0) {
        dir(std::integral_constant<int, 0>{});
        dir(std::integral_constant<int, 1>{});
        dir(std::integral_constant<int, 3>{});
        dir(std::integral_constant<int, 5>{});
        dir(std::integral_constant<int, 7>{});
    } else {
        dir(std::integral_constant<int, 2>{});
        dir(std::integral_constant<int, 4>{});
        dir(std::integral_constant<int, 6>{});
        dir(std::integral_constant<int, 8>{});
    }
}

// The same on the FP64 pipe, out of line: for blocks with a value outside the
// range of the integer products.
static __device__ __noinline__ void small_force_plain(Small64 &sm, Pops64 p, int k, int a) { small_force<false>(sm, p, k, a); }
static __device__ __noinline__ double small_velocity_plain(const Small64 &sm, int a) { return small_velocity<false>(sm, a); }
static __device__ __noinline__ void small_push_plain(const Small64 &sm, Pops64 p, double *nk, int k, int a, int x, int y)
{
    small_push<false>(sm, p, nk, k, a, x, y);
}

template <int kWarps>
__global__ void __launch_bounds__(TX *kWarps, 2)
    k_small64(const Lat<double> *__restrict__ lats, const int4 *__restrict__ tiles, int tile_offset, int parity)
{
    static_assert(kWarps == 4, "two species, two components");
    extern __shared__ __align__(16) unsigned char lb_step_smem[];
    Small64 &sm = *reinterpret_cast<Small64 *>(lb_step_smem);
    const int4 t = tiles[tile_offset + blockIdx.x];
    const Lat<double> &G = lats[t.x];
    const int lane = threadIdx.x, k = threadIdx.y & 1, a = threadIdx.y >> 1;
    const int tid = threadIdx.y * TX + lane;
    for (int i = tid; i < (int)(sizeof(Lat<double>) / 4); i += TX * kWarps)
        reinterpret_cast<uint32_t *>(&sm.st.L)[i] = reinterpret_cast<const uint32_t *>(&G)[i];
    const int x = t.y + lane, y = t.z;
    const bool valid = x < G.nx;
    const size_t plane = G.plane, c = valid ? (size_t)y * G.pitch + x : 0;
    const double *__restrict__ fk = G.f[parity] + (size_t)(k * 9) * plane + c;
    Pops64 p;
#pragma unroll
    for (int i = 0; i < 9; ++i) p.f[i] = fk[(size_t)i * plane];
    uint32_t outside = G.products ? 0u : 1u;
#pragma unroll 1
    for (int q = tid; q < 2 * SW * (1 + 2 * HALO); q += TX * kWarps) {
        const int sp = q / (SW * (1 + 2 * HALO)), slot = q % (SW * (1 + 2 * HALO)), sx = slot % SW, sy = slot / SW;
        const double r = slot_density<double, false>(G, t, parity, sx, sy, sp);
        outside |= sm.st.put(sp, sy, sx, r, psi64(r, G.one, G.exp_table));
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) outside |= base_outside(p.f[i]);
    const bool plain = __syncthreads_or(outside != 0);
    if (plain) small_force_plain(sm, p, k, a);
    else small_force<true>(sm, p, k, a);
    __syncthreads();
    outside = 0;
    if (k == 0) {
        const double u = plain ? small_velocity_plain(sm, a) : small_velocity<true>(sm, a);
        sm.u[a][lane] = u;
        outside = velocity_outside(u);
    }
    const bool plain_push = __syncthreads_or(outside != 0) || plain;
    if (!valid) return;
    double *nk = sm.st.L.f[parity ^ 1] + (size_t)(k * 9) * plane + c;
    if (plain_push) small_push_plain(sm, p, nk, k, a, x, y);
    else small_push<true>(sm, p, nk, k, a, x, y);
}

// ---- persistent launch over many time steps -----------------------------------

// Bounded wait until *ctr >= need.  Gives up when another block has flagged an
// error or after `limit` SM clock cycles, then flags LB_ETIMEOUT in *err.
__device__ __forceinline__ bool wait_geq(const unsigned *ctr, unsigned need, int *err, long long limit)
{
    if (need == 0) return true;
    const long long start = clock64();
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= need) return true;
        if (*(volatile int *)err) return false;
        if (clock64() - start > limit) {
            atomicExch(err, 1);
            return false;
        }
        __nanosleep(128);
    }
}

// Control block of a persistent launch (device memory, cleared before each
// launch): the work-queue head, then per-lattice counts of finished density
// and fused tiles.  The error word lives separately and survives launches.
struct PersistCtl {
    unsigned long long head;
};

// Advance nsteps time steps of every lattice in one launch.  Work items are
// (step, phase, tile) in this order, handed out by an atomic queue; an item
// waits only for the items of its own lattice it depends on (the density
// pass of step t waits for all fused tiles of step t-1, the fused tiles of
// step t for all density tiles of step t).  Every item it waits for has a
// smaller index and was claimed by a running block, so the wait always ends
// unless a block fails to signal; then the bounded wait flags the error and
// every block leaves.  drop_tile >= 0 makes that tile never signal (a test of
// the timeout path).
template <typename real, int TYv>
__global__ void __launch_bounds__(TX *TYv, kCollideMinBlocks<real, TYv>)
    k_persistent(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles, const int *__restrict__ lat_ntiles,
                 int n_tiles, int nsteps, int parity0, PersistCtl *ctl, unsigned *dens_done, unsigned *coll_done,
                 int *err, long long wait_cycles, int drop_tile)
{
    auto &sm = step_smem<real, TYv>();
    __shared__ long long s_item;
    __shared__ int s_ok;
    const int tid = threadIdx.y * TX + threadIdx.x;
    const long long total = (long long)nsteps * 2 * n_tiles;
    for (;;) {
        if (tid == 0) s_item = (long long)atomicAdd(&ctl->head, 1ull);
        __syncthreads();
        const long long item = s_item;
        if (item >= total) break;
        const int t = (int)(item / (2 * n_tiles));
        const int r = (int)(item % (2 * n_tiles));
        const int phase = r / n_tiles, tile = r % n_tiles;
        const int4 tl = tiles[tile];
        const int nt_l = lat_ntiles[tl.x];
        const int parity = (parity0 + t) & 1;
        if (tid == 0) {
            const bool ok = phase == 0 ? wait_geq(&coll_done[tl.x], (unsigned)(t * nt_l), err, wait_cycles)
                                       : wait_geq(&dens_done[tl.x], (unsigned)((t + 1) * nt_l), err, wait_cycles);
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) break;
        if (phase == 0) density_tile<real, TYv, true, !kOffset<real>>(lats, tl, parity);
        else collide_any<real, TYv, true>(lats, tl, parity, sm);
        __syncthreads();
        if (tid == 0 && tile != drop_tile) {
            __threadfence();
            atomicAdd(phase == 0 ? &dens_done[tl.x] : &coll_done[tl.x], 1u);
        }
    }
}

// ---- observables ------------------------------------------------------------

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sums over a block of kThreads threads: every thread leaves its values in
// rows of shared memory; kSumLanes threads a row then add kSumRun values each
// (rows padded so that their accesses spread over the banks) and shuffle.
constexpr int kSumRun = 16, kSumLanes = kThreads / kSumRun, kSumRow = kThreads + kSumLanes;
__device__ __forceinline__ int sum_slot(int t) { return t + t / kSumRun; }

// Per-node diagnostics (densities, momenta with half force, barycentric
// velocity, Eq. 11 bulk pressure) reduced per tile into FP64 partial sums;
// optionally also written as dense FP64 fields [..][ny][nx].  Reads the
// density copy parity^1 written by a density pass at the same time.  The sums
// of a tile go through shared memory, 16 values a thread: shuffles within the
// warps took 75 FP64 additions a node (slot kUmax: the largest |u|^2).
template <typename real>
__global__ void __launch_bounds__(kThreads) k_observe(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles,
                                                      int tile_offset, int parity, double *__restrict__ partials,
                                                      double *__restrict__ out_rho, double *__restrict__ out_mom,
                                                      double *__restrict__ out_ubar)
{
    __shared__ real srho[2][SH][SW];
    __shared__ real spsi[2][SH][SW];
    __shared__ double sacc[kNumAcc][kSumRow];
    const int4 t = tiles[tile_offset + blockIdx.x];
    const Lat<real> &L = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    stage_tile<real, SH>(L, L.rho[parity ^ 1], t.y, t.z, srho, spsi, tid, kThreads);
    __syncthreads();
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    double acc[kNumAcc];
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) acc[a] = 0.0;
    if (x < L.nx && y < L.ny) {
        const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
        const real *__restrict__ fc = L.f[parity];
        const size_t c = (size_t)y * L.pitch + x;
        double r[2], m[2][2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            real fk[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) fk[i] = fc[(size_t)(k * 9 + i) * L.plane + c];
            real Fx, Fy, jx, jy;
            force_at<real, SH>(L, srho, spsi, k, cx, cy, Fx, Fy);
            first_moment<real>(fk, jx, jy);   // FP32: the reference density adds no momentum
            r[k] = (double)srho[k][cy][cx];
            m[k][0] = (double)(jx + (real)0.5 * Fx);
            m[k][1] = (double)(jy + (real)0.5 * Fy);
        }
        const double rt = r[0] + r[1];
        const double ux = (m[0][0] + m[1][0]) / rt, uy = (m[0][1] + m[1][1]) / rt;
        acc[kMassA] = r[0];
        acc[kMassB] = r[1];
        acc[kMomAx] = m[0][0];
        acc[kMomAy] = m[0][1];
        acc[kMomBx] = m[1][0];
        acc[kMomBy] = m[1][1];
        acc[kSumUx] = ux;
        acc[kUmax] = ux * ux + uy * uy;
        acc[kNonFinite] = (isfinite(r[0]) && isfinite(r[1]) && isfinite(ux) && isfinite(uy)) ? 0.0 : 1.0;
        if (L.has_probe) {
            double dx = fabs((double)x - L.probe[0]), dy = fabs((double)y - L.probe[1]);
            if (dx > 0.5 * L.nx) dx = L.nx - dx;
            if (!L.walls && dy > 0.5 * L.ny) dy = L.ny - dy;
            const double rr = sqrt(dx * dx + dy * dy), R = L.probe[2];
            const double psiA = 1.0 - exp(-r[0]), psiB = 1.0 - exp(-r[1]);
            const double Gs = (double)L.G1 + (double)L.G2;
            const double pb = (r[0] + 0.5 * Gs * psiA * psiA) / 3.0 + (r[1] + 0.5 * Gs * psiB * psiB) / 3.0
                            + (double)L.GAB * r[0] * r[1] / 3.0;
            if (rr < 0.5 * R) { acc[kPIn] = pb; acc[kAIn] = r[0]; acc[kNIn] = 1.0; }
            if (rr > R + 6.0) { acc[kPOut] = pb; acc[kAOut] = r[0]; acc[kNOut] = 1.0; }
        }
        if (out_rho) {
            const size_t n = (size_t)L.nx * L.ny, d = (size_t)y * L.nx + x;
            out_rho[d] = r[0];
            out_rho[n + d] = r[1];
            if (out_mom) {
                out_mom[d] = m[0][0];
                out_mom[n + d] = m[0][1];
                out_mom[2 * n + d] = m[1][0];
                out_mom[3 * n + d] = m[1][1];
            }
            if (out_ubar) {
                out_ubar[d] = ux;
                out_ubar[n + d] = uy;
            }
        }
    }
    if (!partials) return;
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) sacc[a][sum_slot(tid)] = acc[a];
    __syncthreads();
    const int a = tid / kSumLanes, l = tid % kSumLanes;
    const bool on = a < kNumAcc;
    double v = on ? sacc[a][sum_slot(kSumRun * l)] : 0.0;
#pragma unroll
    for (int q = 1; q < kSumRun; ++q) {
        const double w = on ? sacc[a][sum_slot(kSumRun * l + q)] : 0.0;
        v = a == kUmax ? fmax(v, w) : v + w;
    }
#pragma unroll
    for (int o = 1; o < kSumLanes; o <<= 1) {
        const double w = __shfl_xor_sync(0xffffffffu, v, o);
        v = a == kUmax ? fmax(v, w) : v + w;
    }
    if (on && l == 0) partials[(size_t)(tile_offset + blockIdx.x) * kAccStride + a] = v;
}

// Lattices of more tiles than this have their partials folded into kFold
// records by as many blocks before k_finalize, whose one block took 5 ms of a
// 4096^2 lattice's observables.  Microseconds of a call without and with the fold:
// 512 tiles, FP32 64 and 66, FP64 115 and 115; 1024 tiles 76 and 72, 169 and 165.
constexpr int kFoldTiles = 768, kFold = 64;

// Block (b, lattice): the b-th of kFold runs of the lattice's tile partials,
// in a fixed order.
template <typename real>
__global__ void __launch_bounds__(256) k_fold(const Lat<real> *__restrict__ lats, const double *__restrict__ partials,
                                              double *__restrict__ fold)
{
    __shared__ double s[256 / 32][kAccStride];
    const Lat<real> &L = lats[blockIdx.y];
    const int nt = L.tile_end - L.tile_begin;
    if (nt <= kFoldTiles) return;
    const int run = (nt + kFold - 1) / kFold, t0 = L.tile_begin + blockIdx.x * run, t1 = min(t0 + run, L.tile_end);
    // 16 threads a tile record, 16 records at a time
    const int a = threadIdx.x % kAccStride, r = threadIdx.x / kAccStride;
    double v = 0.0;
    if (a < kNumAcc)
        for (int t = t0 + r; t < t1; t += 256 / kAccStride) {
            const double w = partials[(size_t)t * kAccStride + a];
            v = a == kUmax ? fmax(v, w) : v + w;
        }
    const double w = __shfl_xor_sync(0xffffffffu, v, 16);
    v = a == kUmax ? fmax(v, w) : v + w;
    if (threadIdx.x % 32 < kAccStride) s[threadIdx.x / 32][a] = v;
    __syncthreads();
    if (threadIdx.x < kNumAcc) {
        v = s[0][a];
        for (int q = 1; q < 256 / 32; ++q) v = a == kUmax ? fmax(v, s[q][a]) : v + s[q][a];
        fold[((size_t)blockIdx.y * kFold + blockIdx.x) * kAccStride + a] = v;
    }
}

// One block per lattice: reduce its tile partials in a fixed order and
// derive the observables.
template <typename real>
__global__ void __launch_bounds__(256) k_finalize(const Lat<real> *__restrict__ lats, const double *__restrict__ partials,
                                                  const double *__restrict__ fold, double *__restrict__ obs)
{
    __shared__ double sred[256 / 32][kAccStride];
    const Lat<real> &L = lats[blockIdx.x];
    const int tid = threadIdx.x;
    double acc[kNumAcc];
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) acc[a] = 0.0;
    const bool folded = L.tile_end - L.tile_begin > kFoldTiles;
    const double *__restrict__ rec = folded ? fold + (size_t)blockIdx.x * kFold * kAccStride
                                            : partials + (size_t)L.tile_begin * kAccStride;
    const int nrec = folded ? kFold : L.tile_end - L.tile_begin;
    for (int tl = tid; tl < nrec; tl += 256) {
#pragma unroll
        for (int a = 0; a < kNumAcc; ++a) {
            const double v = rec[(size_t)tl * kAccStride + a];
            acc[a] = (a == kUmax) ? fmax(acc[a], v) : acc[a] + v;
        }
    }
    const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) {
        const double v = (a == kUmax) ? warp_max(acc[a]) : warp_sum(acc[a]);
        if (lane == 0) sred[warp][a] = v;
    }
    __syncthreads();
    if (tid != 0) return;
    double s[kNumAcc];
    for (int a = 0; a < kNumAcc; ++a) {
        double v = sred[0][a];
        for (int w = 1; w < 8; ++w) v = (a == kUmax) ? fmax(v, sred[w][a]) : v + sred[w][a];
        s[a] = v;
    }
    double *o = obs + (size_t)blockIdx.x * kObsStride;
    o[oMassA] = s[kMassA];
    o[oMassB] = s[kMassB];
    o[oMomAx] = s[kMomAx];
    o[oMomAy] = s[kMomAy];
    o[oMomBx] = s[kMomBx];
    o[oMomBy] = s[kMomBy];
    o[oQ] = s[kSumUx] / L.nx;
    if (L.walls && L.g_x != 0.0) {
        const double H = L.ny, nuB = (L.tau_B - 0.5) / 3.0;
        const double Q0 = L.g_x * (H * H * H + 0.5 * H) / (12.0 * nuB);
        o[oMuR] = Q0 / o[oQ];
    } else {
        o[oMuR] = __longlong_as_double(0x7ff8000000000000ll);
    }
    if (L.has_probe && s[kNIn] > 0.0 && s[kNOut] > 0.0) {
        const double rin = s[kAIn] / s[kNIn], rout = s[kAOut] / s[kNOut];
        o[oDp] = s[kPIn] / s[kNIn] - s[kPOut] / s[kNOut];
        o[oReff] = sqrt((s[kMassA] - rout * (double)L.nx * (double)L.ny) / (3.14159265358979323846 * (rin - rout)));
    } else {
        o[oDp] = __longlong_as_double(0x7ff8000000000000ll);
        o[oReff] = __longlong_as_double(0x7ff8000000000000ll);
    }
    o[oUmax] = sqrt(s[kUmax]);
    o[oFinite] = s[kNonFinite] == 0.0 ? 1.0 : 0.0;
}

// ---- pressure tensor (Sec. II B-C) --------------------------------------------

// Slots of the pressure-tensor partial sums, per tile and per lattice.
enum PSlot { pKinXX = 0, pKinYY, pKinXY, pIntXX, pIntYY, pIntXY, kNumPSlots };
constexpr int kPStride = 8;

// Second moments sum_i w_i s(x + e_i) e_ia e_ib of a staged plane over the
// D2Q9 neighbours (xx, yy, xy), in FP64.
template <typename real>
__device__ __forceinline__ void q9_second(const real (*s)[SW], int cx, int cy, double (&m)[3])
{
    const double W1 = 1.0 / 9.0, W2 = 1.0 / 36.0;
    const double e = s[cy][cx + 1], w = s[cy][cx - 1], n = s[cy + 1][cx], so = s[cy - 1][cx];
    const double ne = s[cy + 1][cx + 1], nw = s[cy + 1][cx - 1], sw = s[cy - 1][cx - 1], se = s[cy - 1][cx + 1];
    const double diag = (ne + nw) + (sw + se);
    m[0] = W1 * (e + w) + W2 * diag;
    m[1] = W1 * (n + so) + W2 * diag;
    m[2] = W2 * ((ne + sw) - (nw + se));
}

// The same over the D2Q25 neighbours with the weights p(|e|^2).
template <typename real>
__device__ __forceinline__ void q25_second(const real (*s)[SW], int cx, int cy, double (&m)[3])
{
    m[0] = m[1] = m[2] = 0.0;
#pragma unroll
    for (int j = 0; j < 25; ++j) {
        const int dx = j % 5 - 2, dy = j / 5 - 2;
        if (dx == 0 && dy == 0) continue;
        const double a = p25(dx * dx + dy * dy) * (double)s[cy + dy][cx + dx];
        m[0] += a * (double)(dx * dx);
        m[1] += a * (double)(dy * dy);
        m[2] += a * (double)(dx * dy);
    }
}

// Per node, in FP64: the kinetic pressure tensor sum_k sum_i f e_a e_b of the
// pre-collision populations (Eq. 13) and the interaction tensor
//   P^int_ab = 1/2 sum_k [G1 psi_k S1_ab + G2 psi_k S2_ab + G_AB rho_k S3_ab],
// S1, S2 the D2Q9 and D2Q25 second moments of psi_k and S3 the D2Q9 second
// moment of the other species' density: each pair interaction of Eqs. (8),
// (9) shared equally by its two nodes, which gives the bulk pressure of
// Eq. (11) in a uniform state and satisfies Eq. (12) summed across a flat
// interface.  Reduced per tile into FP64 partials (slots PSlot); optionally
// also written as dense fields out[2][3][ny][nx] (kinetic, interaction; xx,
// yy, xy).  Reads the density copy parity^1 written by a density pass at the
// same time.
template <typename real>
__global__ void __launch_bounds__(kThreads) k_pressure(const Lat<real> *__restrict__ lats, const int4 *__restrict__ tiles,
                                                       int tile_offset, int parity, double *__restrict__ partials,
                                                       double *__restrict__ out)
{
    __shared__ real srho[2][SH][SW];
    __shared__ real spsi[2][SH][SW];
    __shared__ double sacc[kThreads / 32][kPStride];
    const int4 t = tiles[tile_offset + blockIdx.x];
    const Lat<real> &L = lats[t.x];
    const int tid = threadIdx.y * TX + threadIdx.x;
    stage_tile<real, SH>(L, L.rho[parity ^ 1], t.y, t.z, srho, spsi, tid, kThreads);
    __syncthreads();
    const int x = t.y + threadIdx.x, y = t.z + threadIdx.y;
    double acc[kNumPSlots];
#pragma unroll
    for (int a = 0; a < kNumPSlots; ++a) acc[a] = 0.0;
    if (x < L.nx && y < L.ny) {
        const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
        const real *__restrict__ fc = L.f[parity];
        const size_t c = (size_t)y * L.pitch + x;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double R = kOffset<real> ? (double)L.rho[parity][(size_t)k * L.plane + c] : 0.0;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const double fi = (double)fc[(size_t)(k * 9 + i) * L.plane + c] + w9(i) * R;
                acc[pKinXX] += fi * (double)(ex9(i) * ex9(i));
                acc[pKinYY] += fi * (double)(ey9(i) * ey9(i));
                acc[pKinXY] += fi * (double)(ex9(i) * ey9(i));
            }
            double s1[3], s2[3], s3[3];
            q9_second<real>(spsi[k], cx, cy, s1);
            q25_second<real>(spsi[k], cx, cy, s2);
            q9_second<real>(srho[1 - k], cx, cy, s3);
            const double psi = spsi[k][cy][cx], rho = srho[k][cy][cx];
            const double G1 = L.G1, G2 = L.G2, GAB = L.GAB;
#pragma unroll
            for (int a = 0; a < 3; ++a) acc[pIntXX + a] += 0.5 * (G1 * psi * s1[a] + G2 * psi * s2[a] + GAB * rho * s3[a]);
        }
        if (out) {
            const size_t n = (size_t)L.nx * L.ny, d = (size_t)y * L.nx + x;
#pragma unroll
            for (int a = 0; a < kNumPSlots; ++a) out[(size_t)a * n + d] = acc[a];
        }
    }
    if (!partials) return;
    const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int a = 0; a < kNumPSlots; ++a) {
        const double v = warp_sum(acc[a]);
        if (lane == 0) sacc[warp][a] = v;
    }
    __syncthreads();
    if (tid < kNumPSlots) {
        double v = sacc[0][tid];
        for (int w = 1; w < kThreads / 32; ++w) v += sacc[w][tid];
        partials[(size_t)(tile_offset + blockIdx.x) * kPStride + tid] = v;
    }
}

// One block per lattice: the pressure-tensor partials of its tiles summed in
// a fixed order into out[lattice * kPStride + slot].
template <typename real>
__global__ void __launch_bounds__(256) k_pressure_sum(const Lat<real> *__restrict__ lats,
                                                      const double *__restrict__ partials, double *__restrict__ out)
{
    __shared__ double sred[256 / 32][kPStride];
    const Lat<real> &L = lats[blockIdx.x];
    const int tid = threadIdx.x;
    double acc[kNumPSlots];
#pragma unroll
    for (int a = 0; a < kNumPSlots; ++a) acc[a] = 0.0;
    for (int tl = L.tile_begin + tid; tl < L.tile_end; tl += 256)
#pragma unroll
        for (int a = 0; a < kNumPSlots; ++a) acc[a] += partials[(size_t)tl * kPStride + a];
    const int warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int a = 0; a < kNumPSlots; ++a) {
        const double v = warp_sum(acc[a]);
        if (lane == 0) sred[warp][a] = v;
    }
    __syncthreads();
    if (tid < kNumPSlots) {
        double v = sred[0][tid];
        for (int w = 1; w < 8; ++w) v += sred[w][tid];
        out[(size_t)blockIdx.x * kPStride + tid] = v;
    }
}

// ---- initialisation and population transfer ---------------------------------

// f_k,i = f^eq_i(rho_k, u) (Eq. 2) from dense FP64 fields.  FP32 stores the
// reference R = rho (rounded) in density copy `parity` and h = f^eq - w R.
template <typename real>
__global__ void k_init(const Lat<real> *__restrict__ lats, int lat, const double *__restrict__ rho,
                       const double *__restrict__ u, int parity)
{
    const Lat<real> &L = lats[lat];
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const size_t n = (size_t)L.nx * L.ny, d = (size_t)y * L.nx + x;
    const double ux = u ? u[d] : 0.0, uy = u ? u[n + d] : 0.0;
    const double uu = ux * ux + uy * uy;
    real *f = L.f[parity];
    const size_t c = (size_t)y * L.pitch + x;
    for (int k = 0; k < 2; ++k) {
        const double r = rho[k * n + d];
        double R = 0.0;
        if constexpr (kOffset<real>) {
            const real Rr = (real)r;
            L.rho[parity][(size_t)k * L.plane + c] = Rr;
            R = (double)Rr;
        }
        for (int i = 0; i < 9; ++i) {
            const double eu = ex9(i) * ux + ey9(i) * uy;
            const double feq = w9(i) * r * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
            f[(size_t)(k * 9 + i) * L.plane + c] = (real)(feq - w9(i) * R);
        }
    }
}

// dense FP64 [2][9][ny][nx] <-> native pitched populations (FP32: the
// reference density added back, or recomputed as sum_i f_i on input).
template <typename real>
__global__ void k_get_pops(const Lat<real> *__restrict__ lats, int lat, int parity, double *__restrict__ out)
{
    const Lat<real> &L = lats[lat];
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const size_t n = (size_t)L.nx * L.ny, d = (size_t)y * L.nx + x, c = (size_t)y * L.pitch + x;
    for (int k = 0; k < 2; ++k) {
        const double R = kOffset<real> ? (double)L.rho[parity][(size_t)k * L.plane + c] : 0.0;
        for (int i = 0; i < 9; ++i)
            out[(size_t)(k * 9 + i) * n + d] = (double)L.f[parity][(size_t)(k * 9 + i) * L.plane + c] + w9(i) * R;
    }
}

template <typename real>
__global__ void k_set_pops(const Lat<real> *__restrict__ lats, int lat, int parity, const double *__restrict__ in)
{
    const Lat<real> &L = lats[lat];
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= L.nx || y >= L.ny) return;
    const size_t n = (size_t)L.nx * L.ny, d = (size_t)y * L.nx + x, c = (size_t)y * L.pitch + x;
    for (int k = 0; k < 2; ++k) {
        double R = 0.0;
        if constexpr (kOffset<real>) {
            double s = 0.0;
            for (int i = 0; i < 9; ++i) s += in[(size_t)(k * 9 + i) * n + d];
            const real Rr = (real)s;
            L.rho[parity][(size_t)k * L.plane + c] = Rr;
            R = (double)Rr;
        }
        for (int i = 0; i < 9; ++i)
            L.f[parity][(size_t)(k * 9 + i) * L.plane + c] = (real)(in[(size_t)(k * 9 + i) * n + d] - w9(i) * R);
    }
}

}  // namespace lbk

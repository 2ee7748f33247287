// lb3_kernels.cuh -- sm_103a kernels of the three-dimensional extension of the
// two-range pseudopotential lattice Boltzmann step (the paper is 2-D; its
// Sec. II carried to three dimensions):
//   fluid         D3Q19 (w = 1/3, 1/18, 1/36), BGK with Guo forcing (Eqs. 1-3,
//                 5, 6 in 3-D)
//   short range   sums of Eqs. (8) (first term) and (9) over the D3Q19
//                 neighbours with the weights w
//   mid range     sum of Eq. (8) (second term) over the 5 x 5 x 5
//                 neighbourhood with weights q(|e|^2): 47/90, 4/135, 1/63,
//                 2/315, 5/1512, 1/945, 1/1890, 1/15120 for |e|^2 = 0..6, 8
//                 (0 for 9 and 12), isotropic to eighth order with the D2Q25
//                 stencil's second and fourth moments
// Periodic in x, y and z.  Templated on the population format, as the 2-D
// kernels: real = double plain populations (this instantiation compiled
// without FMA contraction), real = float offsets h_i = f_i - w_i R from the
// node's density at the previous step R, with the stencil and momentum sums
// formed from differences of opposite neighbours.
//
// One FP64 time step is two launches over tiles of 32 x 4 x 2 nodes:
//   k3_density : rho_k = sum_i f_k,i (FP32: R + sum_i h_i, for the observables)
//                into copy parity^1
//   k3_collide : stages rho_k and psi_k of the tile plus a 2-node halo in
//                shared memory, forms the forces, moments, u^eq, relaxes with
//                the Guo term and pushes each population to x + e_i.
// FP32 steps in one launch (k3_march), which also re-references each pushed
// offset to rho(x + e_i), the destination's next R.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <type_traits>

#include "lb_f64.cuh"
#include "lb_vops.cuh"

namespace lbk3 {

using lbk::cfma;
using lbk::cmul;
using lbk::vadd;
using lbk::vdiv;
using lbk::vfma;
using lbk::vmul;
using lbk::vneg;
using lbk::vsplat;
using lbk::vsub;
using lbk::vswap;

constexpr int TX = 32, TY = 4, TZ = 2, HALO = 2;
constexpr int SX = TX + 2 * HALO, SY = TY + 2 * HALO, SZ = TZ + 2 * HALO;
constexpr int kThreads = TX * TY * TZ;
constexpr int kNumAcc = 16;   // observation partial sums per tile

// D3Q19: rest, 6 axis directions, 12 edge directions
__host__ __device__ constexpr int ex(int i)
{
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1 : ((i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0);
}
__host__ __device__ constexpr int ey(int i)
{
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1 : ((i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0);
}
__host__ __device__ constexpr int ez(int i)
{
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1 : ((i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0);
}
__host__ __device__ constexpr int e2(int i) { return ex(i) * ex(i) + ey(i) * ey(i) + ez(i) * ez(i); }
__host__ __device__ constexpr double w19(int i) { return e2(i) == 0 ? 1.0 / 3.0 : (e2(i) == 1 ? 1.0 / 18.0 : 1.0 / 36.0); }
__host__ __device__ constexpr double q125(int e2v)
{
    return e2v == 0 ? 47.0 / 90.0 : e2v == 1 ? 4.0 / 135.0 : e2v == 2 ? 1.0 / 63.0 : e2v == 3 ? 2.0 / 315.0
         : e2v == 4 ? 5.0 / 1512.0 : e2v == 5 ? 1.0 / 945.0 : e2v == 6 ? 1.0 / 1890.0 : e2v == 8 ? 1.0 / 15120.0 : 0.0;
}

template <typename real>
constexpr bool kOffset3 = sizeof(real) == 4;

// Descriptor of one 3-D lattice (device-visible).
template <typename real>
struct Lat3 {
    real *f[2];          // ping-pong populations [2][19][nz][ny][pitch]
    real *rho[2];        // densities [2][nz][ny][pitch]
    size_t plane;        // elements per [nz][ny][pitch] volume
    int32_t nx, ny, nz, pitch;
    int32_t tiles_x, tiles_y, tiles_z, has_probe;
    real omega[2];       // 1 / tau_k
    real aw3[2][3];      // 3 (1 - omega_k / 2) w(|e|^2) for |e|^2 = 0, 1, 2
    const double2 *exp_table;   // exp(-j/512) for the FP64 density pass (lb_f64.cuh)
    real cw[9];          // -(G1 w + G2 q) for |e|^2 = 0 .. 8 (the two psi sums of Eq. 8 as one)
    real G1, G2, GAB;
    real g[3];
    double probe[4];     // cx, cy, cz, R
};

template <typename real> __device__ __forceinline__ real psi3(real r);
template <> __device__ __forceinline__ double psi3<double>(double r) { return 1.0 - exp(-r); }
template <> __device__ __forceinline__ float psi3<float>(float r) { return -expm1f(-r); }

__device__ __forceinline__ int wrap3(int a, int n)
{
    a %= n;
    return a < 0 ? a + n : a;
}

// a periodic index one period off at most (a in [-n, 2n)): no division
__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

__device__ __forceinline__ void tile_origin(int tiles_x, int tiles_y, int b, int &x0, int &y0, int &z0)
{
    x0 = (b % tiles_x) * TX;
    y0 = ((b / tiles_x) % tiles_y) * TY;
    z0 = (b / (tiles_x * tiles_y)) * TZ;
}

template <typename real>
struct Stage3 {
    real rho[2][SZ][SY][SX];
    real psi[2][SZ][SY][SX];
};
static_assert(sizeof(Stage3<float>) % 16 == 0 && sizeof(Stage3<double>) % 16 == 0, "partials stay aligned");

// rows of per-thread values for the observation sums, in the stage's place
constexpr int kSumRun3 = 16, kSumRow3 = kThreads + kThreads / kSumRun3;
static_assert(kThreads == kNumAcc * kSumRun3, "a thread sums one run of one row");
constexpr size_t kSumBytes3 = (size_t)kNumAcc * kSumRow3 * sizeof(double);

template <typename real>
constexpr size_t kCollideSmem3 = sizeof(Stage3<real>);
template <typename real>
constexpr size_t kObserveSmem3 = sizeof(Stage3<real>) > kSumBytes3 ? sizeof(Stage3<real>) : kSumBytes3;

// rho and psi of the tile (x0, y0, z0) and its 2-node halo from density copy
// `rho` (periodic copies across every face).
template <typename real>
__device__ __forceinline__ void stage3(const Lat3<real> &L, const real *__restrict__ rho, int x0, int y0, int z0,
                                       Stage3<real> &sm, int tid)
{
    // the slots' coordinates lie within one period of the lattice when each
    // side is at least a tile plus both halos (a block-uniform choice)
    const bool near = L.nx >= SX && L.ny >= SY && L.nz >= SZ;
    for (int idx = tid; idx < SX * SY * SZ; idx += kThreads) {
        const int sx = idx % SX, sy = (idx / SX) % SY, sz = idx / (SX * SY);
        const int ax = x0 + sx - HALO, ay = y0 + sy - HALO, az = z0 + sz - HALO;
        const int gx = near ? wrap1(ax, L.nx) : wrap3(ax, L.nx), gy = near ? wrap1(ay, L.ny) : wrap3(ay, L.ny);
        const int gz = near ? wrap1(az, L.nz) : wrap3(az, L.nz);
        const size_t c = ((size_t)gz * L.ny + gy) * L.pitch + gx;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const real r = rho[(size_t)k * L.plane + c];
            sm.rho[k][sz][sy][sx] = r;
            sm.psi[k][sz][sy][sx] = psi3<real>(r);
        }
    }
}

// sum_i w_i s(x + e_i) e_i over D3Q19 (FP64: direction order; FP32:
// differences of opposite neighbours)
template <typename real>
__device__ __forceinline__ void q19_sum(const real (*s)[SY][SX], int cx, int cy, int cz, real (&out)[3])
{
    out[0] = out[1] = out[2] = (real)0;
    if constexpr (!kOffset3<real>) {
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const real a = (real)w19(i) * s[cz + ez(i)][cy + ey(i)][cx + ex(i)];
            if (ex(i)) out[0] += a * (real)ex(i);
            if (ey(i)) out[1] += a * (real)ey(i);
            if (ez(i)) out[2] += a * (real)ez(i);
        }
    } else {
#pragma unroll
        for (int i = 1; i < 19; i += 2) {   // directions come in opposite pairs (i, i + 1)
            const real d = s[cz + ez(i)][cy + ey(i)][cx + ex(i)] - s[cz - ez(i)][cy - ey(i)][cx - ex(i)];
            const real wd = (real)w19(i) * d;
            if (ex(i)) out[0] += ex(i) > 0 ? wd : -wd;
            if (ey(i)) out[1] += ey(i) > 0 ? wd : -wd;
            if (ez(i)) out[2] += ez(i) > 0 ? wd : -wd;
        }
    }
}

// sum_j q_j s(x + e_j) e_j over the 5 x 5 x 5 neighbourhood (FP64: raster
// order dz, dy, dx; FP32: differences of opposite neighbours, each pair once)
template <typename real>
__device__ __forceinline__ void q125_sum(const real (*s)[SY][SX], int cx, int cy, int cz, real (&out)[3])
{
    out[0] = out[1] = out[2] = (real)0;
#pragma unroll
    for (int j = 0; j < 125; ++j) {
        const int dx = j % 5 - 2, dy = (j / 5) % 5 - 2, dz = j / 25 - 2;
        const double qw = q125(dx * dx + dy * dy + dz * dz);
        if (qw == 0.0 || (dx == 0 && dy == 0 && dz == 0)) continue;
        if constexpr (!kOffset3<real>) {
            const real a = (real)qw * s[cz + dz][cy + dy][cx + dx];
            if (dx) out[0] += a * (real)dx;
            if (dy) out[1] += a * (real)dy;
            if (dz) out[2] += a * (real)dz;
        } else {
            // each opposite pair once: the member with dz > 0, or dz = 0 and
            // dy > 0, or dz = dy = 0 and dx > 0
            if (!(dz > 0 || (dz == 0 && dy > 0) || (dz == 0 && dy == 0 && dx > 0))) continue;
            const real d = (real)qw * (s[cz + dz][cy + dy][cx + dx] - s[cz - dz][cy - dy][cx - dx]);
            if (dx) out[0] += d * (real)dx;
            if (dy) out[1] += d * (real)dy;
            if (dz) out[2] += d * (real)dz;
        }
    }
}

// ---- stencil sums from differences of opposite neighbours -----------------------

// Arithmetic on both species at once (FP32) and on one value (FP64).
struct Pair32 {
    using V = float2;
    using S = float;
    __device__ __forceinline__ V zero() const { return make_float2(0.f, 0.f); }
    __device__ __forceinline__ V add(V a, V b) const { return vadd(a, b); }
    __device__ __forceinline__ V sub(V a, V b) const { return vsub(a, b); }
    __device__ __forceinline__ V scale(S c, V a) const { return cmul(c, a); }
    __device__ __forceinline__ V fma(S c, V a, V b) const { return cfma(c, a, b); }
};
// FP64: sums as fmas with the factor 1 in a register, the cheapest FP64
// instruction of the chip (lb_f64.cuh).
struct One64 {
    using V = double;
    using S = double;
    double one;
    __device__ __forceinline__ V zero() const { return 0.0; }
    __device__ __forceinline__ V add(V a, V b) const { return __fma_rn(a, one, b); }
    __device__ __forceinline__ V sub(V a, V b) const { return __fma_rn(-b, one, a); }
    __device__ __forceinline__ V scale(S c, V a) const { return c * a; }
    __device__ __forceinline__ V fma(S c, V a, V b) const { return __fma_rn(c, a, b); }
};

// sum_j c_j s(x + e_j) e_j over the 5 x 5 x 5 neighbourhood from differences
// D(dx, dy, dz) = s(x + e) - s(x - e), outer shells first; c[|e|^2].
template <class Ops, class Diff>
__device__ __forceinline__ void psi_sums3(const Ops &o, const Diff &D, const typename Ops::S (&c)[9], typename Ops::V (&s)[3])
{
    using V = typename Ops::V;
    using S = typename Ops::S;
    s[0] = s[1] = s[2] = o.zero();
    // in-plane pairs (a, b) of the axes (A, B): (e_A, e_B) and (e_A, -e_B)
    auto plane = [&](auto Ac, auto Bc, int a, int b, S w) {
        constexpr int A = decltype(Ac)::value, B = decltype(Bc)::value;
        int e[3] = {0, 0, 0};
        e[A] = a;
        e[B] = b;
        const V p = D(e[0], e[1], e[2]);
        e[B] = -b;
        const V m = D(e[0], e[1], e[2]);
        s[A] = o.fma(w * (S)a, o.add(p, m), s[A]);
        s[B] = o.fma(w * (S)b, o.sub(p, m), s[B]);
    };
    auto corner = [&](int a, int b, int d, S w) {
        const V d1 = D(a, b, d), d2 = D(a, b, -d), d3 = D(a, -b, d), d4 = D(a, -b, -d);
        const V s12 = o.add(d1, d2), s34 = o.add(d3, d4), m12 = o.sub(d1, d2), m34 = o.sub(d3, d4);
        s[0] = o.fma(w * (S)a, o.add(s12, s34), s[0]);
        s[1] = o.fma(w * (S)b, o.sub(s12, s34), s[1]);
        s[2] = o.fma(w * (S)d, o.add(m12, m34), s[2]);
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    auto planes = [&](int a, int b, S w) {
        plane(I0{}, I1{}, a, b, w);
        plane(I0{}, I2{}, a, b, w);
        plane(I1{}, I2{}, a, b, w);
    };
    planes(2, 2, c[8]);
    corner(2, 1, 1, c[6]);
    corner(1, 2, 1, c[6]);
    corner(1, 1, 2, c[6]);
    planes(2, 1, c[5]);
    planes(1, 2, c[5]);
    s[0] = o.fma((S)2 * c[4], D(2, 0, 0), s[0]);
    s[1] = o.fma((S)2 * c[4], D(0, 2, 0), s[1]);
    s[2] = o.fma((S)2 * c[4], D(0, 0, 2), s[2]);
    corner(1, 1, 1, c[3]);
    planes(1, 1, c[2]);
    s[0] = o.fma(c[1], D(1, 0, 0), s[0]);
    s[1] = o.fma(c[1], D(0, 1, 0), s[1]);
    s[2] = o.fma(c[1], D(0, 0, 1), s[2]);
}

// sum_i w_i s(x + e_i) e_i over D3Q19 from the same differences.
template <class Ops, class Diff>
__device__ __forceinline__ void rho_sums3(const Ops &o, const Diff &D, typename Ops::V (&s)[3])
{
    using V = typename Ops::V;
    using S = typename Ops::S;
    const S w1 = (S)(1.0 / 18.0), w2 = (S)(1.0 / 36.0);
    const V xy = D(1, 1, 0), xm = D(1, -1, 0), xz = D(1, 0, 1), xn = D(1, 0, -1), yz = D(0, 1, 1), yn = D(0, 1, -1);
    s[0] = o.fma(w1, D(1, 0, 0), o.scale(w2, o.add(o.add(xy, xm), o.add(xz, xn))));
    s[1] = o.fma(w1, D(0, 1, 0), o.scale(w2, o.add(o.sub(xy, xm), o.add(yz, yn))));
    s[2] = o.fma(w1, D(0, 0, 1), o.scale(w2, o.add(o.sub(xz, xn), o.sub(yz, yn))));
}

// total force on species k at the staged node: Eq. (8) + Eq. (9) + rho_k g
template <typename real>
__device__ __forceinline__ void force3(const Lat3<real> &L, const Stage3<real> &sm, int k, int cx, int cy, int cz,
                                       real (&F)[3])
{
    real s1[3], s2[3], s3[3];
    q19_sum<real>(sm.psi[k], cx, cy, cz, s1);
    q125_sum<real>(sm.psi[k], cx, cy, cz, s2);
    q19_sum<real>(sm.rho[1 - k], cx, cy, cz, s3);
    const real psi = sm.psi[k][cz][cy][cx], rho = sm.rho[k][cz][cy][cx];
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a] = -L.G1 * psi * s1[a] - L.G2 * psi * s2[a] - L.GAB * rho * s3[a] + rho * L.g[a];
}

// kPsi: psi of the step (FP64) as well.
template <typename real, bool kPsi>
__global__ void __launch_bounds__(kThreads) k3_density(const Lat3<real> L, int parity)
{
    int x0, y0, z0;
    tile_origin(L.tiles_x, L.tiles_y, blockIdx.x, x0, y0, z0);
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    if (x >= L.nx || y >= L.ny || z >= L.nz) return;
    const size_t c = ((size_t)z * L.ny + y) * L.pitch + x;
    const real *__restrict__ f = L.f[parity];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        real r = (real)0;
#pragma unroll
        for (int i = 0; i < 19; ++i) r += f[(size_t)(k * 19 + i) * L.plane + c];
        if constexpr (kOffset3<real>) r = L.rho[parity][(size_t)k * L.plane + c] + r;
        L.rho[parity ^ 1][(size_t)k * L.plane + c] = r;
        // FP64 keeps no reference densities: copy parity holds psi for the
        // collide kernel, so that exp() runs once per node
        if constexpr (kPsi) L.rho[parity][(size_t)k * L.plane + c] = lbk::psi64(r, lbk::opaque_one(), L.exp_table);
    }
}

// Dynamic shared memory of the staging kernels (the FP64 stage is above the
// 48 KB of static shared memory): the stage, then the observation partials.
extern __shared__ __align__(16) unsigned char lb3_smem[];

// The FP64 step after its density pass.  It is bound by the FP64 pipe (one
// warp instruction per 16 to 19 clocks and SM), so what counts is the number
// of FP64 instructions: the two psi sums of Eq. (8) as one stencil of paired
// differences, products fused into the sums that take them, the terms of the
// directions shared by opposite ones and by the species, psi from the density
// pass.  704 a node (2132 as direct sums in raster order with every product on
// its own), the pipe 86 % busy; a 61 x 66 x 70 step 1.22 -> 0.44 ms, 32^3
// 160 -> 64 us.
template <typename real>
__global__ void __launch_bounds__(kThreads, 2) k3_collide(const Lat3<real> L, int parity)
{
    static_assert(!kOffset3<real>, "FP32 steps in one pass (k3_march)");
    Stage3<real> &sm = *reinterpret_cast<Stage3<real> *>(lb3_smem);
    int x0, y0, z0;
    tile_origin(L.tiles_x, L.tiles_y, blockIdx.x, x0, y0, z0);
    const int tid = (threadIdx.z * TY + threadIdx.y) * TX + threadIdx.x;
    {
        const real *__restrict__ rho = L.rho[parity ^ 1], *__restrict__ psi = L.rho[parity];
        const bool near = L.nx >= SX && L.ny >= SY && L.nz >= SZ;
        for (int idx = tid; idx < SX * SY * SZ; idx += kThreads) {
            const int sx = idx % SX, sy = (idx / SX) % SY, sz = idx / (SX * SY);
            const int ax = x0 + sx - HALO, ay = y0 + sy - HALO, az = z0 + sz - HALO;
            const int gx = near ? wrap1(ax, L.nx) : wrap3(ax, L.nx), gy = near ? wrap1(ay, L.ny) : wrap3(ay, L.ny);
            const int gz = near ? wrap1(az, L.nz) : wrap3(az, L.nz);
            const size_t c = ((size_t)gz * L.ny + gy) * L.pitch + gx;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                sm.rho[k][sz][sy][sx] = rho[(size_t)k * L.plane + c];
                sm.psi[k][sz][sy][sx] = psi[(size_t)k * L.plane + c];
            }
        }
    }
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    if (x >= L.nx || y >= L.ny || z >= L.nz) return;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO, cz = threadIdx.z + HALO;
    const size_t c = ((size_t)z * L.ny + y) * L.pitch + x;
    const real *__restrict__ fc = L.f[parity] + c;
    const One64 o{lbk::opaque_one()};
    real F[2][3], m[2][3];
    const real rho[2] = {sm.rho[0][cz][cy][cx], sm.rho[1][cz][cy][cx]};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        real p[3], s[3];
        auto dpsi = [&](int dx, int dy, int dz) {
            return o.sub(sm.psi[k][cz + dz][cy + dy][cx + dx], sm.psi[k][cz - dz][cy - dy][cx - dx]);
        };
        auto drho = [&](int dx, int dy, int dz) {
            return o.sub(sm.rho[1 - k][cz + dz][cy + dy][cx + dx], sm.rho[1 - k][cz - dz][cy - dy][cx - dx]);
        };
        psi_sums3(o, dpsi, L.cw, p);
        rho_sums3(o, drho, s);
        const real psi = sm.psi[k][cz][cy][cx], cr = -L.GAB * rho[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) F[k][a] = __fma_rn(psi, p[a], __fma_rn(cr, s[a], rho[k] * L.g[a]));
        // half-force momenta (Eq. 6) from differences of opposite populations
        real j[3];
#pragma unroll
        for (int q = 1; q < 10; ++q) {
            const real d = o.sub(fc[(size_t)(k * 19 + 2 * q - 1) * L.plane], fc[(size_t)(k * 19 + 2 * q) * L.plane]);
            const int e[3] = {ex(2 * q - 1), ey(2 * q - 1), ez(2 * q - 1)};
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (e[a] != 0) j[a] = q == a + 1 ? d : (e[a] > 0 ? o.add(j[a], d) : o.sub(j[a], d));
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) m[k][a] = __fma_rn((real)0.5, F[k][a], j[a]);
    }
    // Eq. (3)
    const real om0 = L.omega[0], om1 = L.omega[1];
    const real den = __fma_rn(om0, rho[0], om1 * rho[1]);
    real u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = __fma_rn(om0, m[0][a], om1 * m[1][a]) / den;
    const real m15uu = (real)-1.5 * __fma_rn(u[0], u[0], __fma_rn(u[1], u[1], u[2] * u[2]));
    const int oE = x + 1 < L.nx ? 1 : 1 - L.nx, oW = x > 0 ? -1 : L.nx - 1;
    const long long oN = y + 1 < L.ny ? (long long)L.pitch : -(long long)L.pitch * (L.ny - 1);
    const long long oS = y > 0 ? -(long long)L.pitch : (long long)L.pitch * (L.ny - 1);
    const long long pxy = (long long)L.ny * L.pitch;
    const long long oU = z + 1 < L.nz ? pxy : -pxy * (L.nz - 1), oD = z > 0 ? -pxy : pxy * (L.nz - 1);
    real *__restrict__ fn = L.f[parity ^ 1] + c;
    real wr[2][3], uF[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        uF[k] = __fma_rn(u[0], F[k][0], __fma_rn(u[1], F[k][1], u[2] * F[k][2]));
        wr[k][0] = (real)w19(0) * rho[k];
        wr[k][1] = (real)w19(1) * rho[k];
        wr[k][2] = (real)w19(7) * rho[k];
    }
    // direction I of both species: f + omega (w rho q - f) + 3 (1 - omega/2) w X,
    // q the polynomial of Eq. (2) and X = (e.F)(1 + 3 e.u) - u.F (Eqs. 1, 2, 5)
    auto push = [&](auto Ic, real q, real XA, real XB) {
        constexpr int I = decltype(Ic)::value, C = e2(I);
        const long long off = (long long)(ex(I) > 0 ? oE : ex(I) < 0 ? oW : 0) + (ey(I) > 0 ? oN : ey(I) < 0 ? oS : 0) +
                              (ez(I) > 0 ? oU : ez(I) < 0 ? oD : 0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const size_t pl = (size_t)(k * 19 + I) * L.plane;
            const real f = fc[pl];
            const real v = __fma_rn(k ? om1 : om0, __fma_rn(wr[k][C], q, -f), f);
            fn[(long long)pl + off] = __fma_rn(L.aw3[k][C], k ? XB : XA, v);
        }
    };
    const real c0 = o.add((real)1, m15uu);
    push(std::integral_constant<int, 0>{}, c0, -uF[0], -uF[1]);
    auto pair = [&](auto Ic) {
        constexpr int I = decltype(Ic)::value, E[3] = {ex(I), ey(I), ez(I)};
        real eu = (real)0, eF[2] = {(real)0, (real)0};
        bool first = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (E[a] == 0) continue;
            eu = first ? u[a] : (E[a] > 0 ? o.add(eu, u[a]) : o.sub(eu, u[a]));
#pragma unroll
            for (int k = 0; k < 2; ++k)
                eF[k] = first ? F[k][a] : (E[a] > 0 ? o.add(eF[k], F[k][a]) : o.sub(eF[k], F[k][a]));
            first = false;
        }
        const real sq = __fma_rn((real)4.5 * eu, eu, c0);
        const real tp = __fma_rn((real)3, eu, (real)1), tm = __fma_rn((real)3, eu, (real)-1);
        push(Ic, __fma_rn((real)3, eu, sq), __fma_rn(eF[0], tp, -uF[0]), __fma_rn(eF[1], tp, -uF[1]));
        push(std::integral_constant<int, I + 1>{}, __fma_rn((real)-3, eu, sq), __fma_rn(eF[0], tm, -uF[0]),
             __fma_rn(eF[1], tm, -uF[1]));
    };
    pair(std::integral_constant<int, 1>{});
    pair(std::integral_constant<int, 3>{});
    pair(std::integral_constant<int, 5>{});
    pair(std::integral_constant<int, 7>{});
    pair(std::integral_constant<int, 9>{});
    pair(std::integral_constant<int, 11>{});
    pair(std::integral_constant<int, 13>{});
    pair(std::integral_constant<int, 15>{});
    pair(std::integral_constant<int, 17>{});
}

// ---- the FP32 step in one pass ------------------------------------------------
//
// A block owns a column of 32 x 8 nodes in (x, y) and marches along z.  Per
// plane it forms the densities and psi of the 36 x 12 slots two planes ahead
// from their populations (into a ring of six planes in shared memory, both
// species as a pair), then, one barrier later, the forces, the collision and
// the pushes of its own plane, whose populations it reads a second time out
// of L2.  A step is one launch; the density pass and collide kernel before it
// moved 160 bytes a node more and formed the stencils once per species and as
// two sums each, 3021 instructions a node against 1592 here.  160^3: 660 us a
// step before, 421 now; 64^3: 50 and 37.  What bounds it is latency at 16 warps
// per SM (39 % of the issue slots, 42 % of HBM): three blocks of 80 registers
// spill (566 us); the populations by cp.async into shared memory a plane ahead
// (436 us, 462 at three blocks), an L2 prefetch of the planes ahead (440 us) and
// the density as a pass of its own before the same march (424 us) gained nothing.
constexpr int RY = 8;                       // tile height in y
constexpr int RW = TX + 2 * HALO, RH = RY + 2 * HALO;
constexpr int kRing3 = 6;                   // planes z-2 .. z+2, and the one being written
constexpr int kRingSlots = RW * RH - TX * RY;

struct March3 {
    float2 rho[kRing3][RH][RW];
    float2 psi[kRing3][RH][RW];
};

// Densities (both species) of a node from its offset populations, in the
// order of k3_density; f, R: the node in the first population plane and in
// the reference densities.
__device__ __forceinline__ float2 node_density3(const float *__restrict__ f, const float *__restrict__ R, size_t plane)
{
    float2 v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = make_float2(f[(size_t)i * plane], f[(size_t)(19 + i) * plane]);
    const float2 r0 = make_float2(R[0], R[plane]);
    float2 r = v[0];
#pragma unroll
    for (int i = 1; i < 19; ++i) r = vadd(r, v[i]);
    return vadd(r0, r);
}

template <int kBlocks>
__global__ void __launch_bounds__(TX *RY, kBlocks) k3_march(const Lat3<float> L, int parity, int tiles_y, int lz)
{
    March3 &sm = *reinterpret_cast<March3 *>(lb3_smem);
    const int tid = threadIdx.y * TX + threadIdx.x;
    const int bx = blockIdx.x % L.tiles_x, by = (blockIdx.x / L.tiles_x) % tiles_y;
    const int z0 = (blockIdx.x / (L.tiles_x * tiles_y)) * lz, z1 = min(z0 + lz, L.nz);
    const int x0 = bx * TX, y0 = by * RY;
    const size_t plane = L.plane, pxy = (size_t)L.ny * L.pitch;
    const float *__restrict__ f = L.f[parity], *__restrict__ R = L.rho[parity];
    // the thread's slots: its own node's, and one of the halo ring's
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    const bool valid = x < L.nx && y < L.ny, ring = tid < kRingSlots;
    const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO;
    int rx = 0, ry = 0;
    if (tid < 2 * RW) {
        ry = tid / RW;
        rx = tid % RW;
    } else if (tid < 4 * RW) {
        ry = RY + HALO + (tid - 2 * RW) / RW;
        rx = (tid - 2 * RW) % RW;
    } else if (ring) {
        const int q = tid - 4 * RW;
        ry = HALO + q / 4;
        rx = (q % 4 < 2) ? q % 4 : TX + q % 4;
    }
    const size_t own = (size_t)wrap3(y, L.ny) * L.pitch + wrap3(x, L.nx);
    const size_t rim = (size_t)wrap3(y0 + ry - HALO, L.ny) * L.pitch + wrap3(x0 + rx - HALO, L.nx);
    // densities and psi of plane z (any integer) into ring plane q
    auto stage = [&](int z, int q) {
        const size_t zo = (size_t)wrap3(z, L.nz) * pxy;
        if (ring) {
            const float2 r = node_density3(f + zo + rim, R + zo + rim, plane);
            sm.rho[q][ry][rx] = r;
            sm.psi[q][ry][rx] = make_float2(psi3<float>(r.x), psi3<float>(r.y));
        }
        const float2 r = node_density3(f + zo + own, R + zo + own, plane);
        sm.rho[q][cy][cx] = r;
        sm.psi[q][cy][cx] = make_float2(psi3<float>(r.x), psi3<float>(r.y));
        if (valid && z >= z0 && z < z1) {   // the next step's reference density
            float *rn = L.rho[parity ^ 1] + zo + own;
            rn[0] = r.x;
            rn[plane] = r.y;
        }
    };
#pragma unroll 1
    for (int z = z0 - 2; z < z0 + 2; ++z) stage(z, z - z0 + 2);
    int q = 4;   // ring plane of z + 2
    // push offsets in x and y
    const int oE = x + 1 < L.nx ? 1 : 1 - L.nx, oW = x > 0 ? -1 : L.nx - 1;
    const long long oN = y + 1 < L.ny ? (long long)L.pitch : -(long long)L.pitch * (L.ny - 1);
    const long long oS = y > 0 ? -(long long)L.pitch : (long long)L.pitch * (L.ny - 1);
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        stage(z + 2, q);
        __syncthreads();
        // ring planes of z - 2 .. z + 2
        int rp[5];
#pragma unroll
        for (int d = 0; d < 5; ++d) rp[d] = q + d - 4 + (q + d - 4 < 0 ? kRing3 : 0);
        q = q == kRing3 - 1 ? 0 : q + 1;
        if (!valid) continue;
        const size_t c = (size_t)z * pxy + own;
        float2 h[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) h[i] = make_float2(f[(size_t)i * plane + c], f[(size_t)(19 + i) * plane + c]);
        const float2 R2 = make_float2(R[c], R[plane + c]);
        auto dpsi = [&](int dx, int dy, int dz) {
            return vsub(sm.psi[rp[2 + dz]][cy + dy][cx + dx], sm.psi[rp[2 - dz]][cy - dy][cx - dx]);
        };
        auto drho = [&](int dx, int dy, int dz) {
            return vsub(sm.rho[rp[2 + dz]][cy + dy][cx + dx], sm.rho[rp[2 - dz]][cy - dy][cx - dx]);
        };
        const float2 rho = sm.rho[rp[2]][cy][cx];
        float2 F[3];
        {
            float2 m[3], s[3];
            psi_sums3(Pair32{}, dpsi, L.cw, m);
            rho_sums3(Pair32{}, drho, s);
            const float2 psi = sm.psi[rp[2]][cy][cx], cr = cmul(-L.GAB, rho);
#pragma unroll
            for (int a = 0; a < 3; ++a) F[a] = vfma(psi, m[a], vfma(cr, vswap(s[a]), cmul(L.g[a], rho)));
        }
        // first moment from differences of opposite offsets; then the offsets
        // from the node's current density and their sum (as in 2-D)
        float2 j[3];
        {
            float2 d[10];
#pragma unroll
            for (int p = 1; p < 10; ++p) d[p] = vsub(h[2 * p - 1], h[2 * p]);
            // pairs: 1 x, 2 y, 3 z, 4 xy, 5 x-y, 6 xz, 7 x-z, 8 yz, 9 y-z
            j[0] = vadd(d[1], vadd(vadd(d[4], d[5]), vadd(d[6], d[7])));
            j[1] = vadd(d[2], vadd(vsub(d[4], d[5]), vadd(d[8], d[9])));
            j[2] = vadd(d[3], vadd(vsub(d[6], d[7]), vsub(d[8], d[9])));
        }
        const float2 delta = vsub(rho, R2);
#pragma unroll
        for (int i = 0; i < 19; ++i) h[i] = cfma(-(float)w19(i), delta, h[i]);
        float2 dg = h[0];
#pragma unroll
        for (int p = 1; p < 10; ++p) dg = vadd(dg, vadd(h[2 * p - 1], h[2 * p]));
        // u^eq of Eq. (3) from the half-force momenta (Eq. 6)
        const float2 om = make_float2(L.omega[0], L.omega[1]);
        const float den = vfma(om.y, rho.y, vmul(om.x, rho.x));
        float u[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float2 m = cfma(0.5f, F[a], j[a]);
            u[a] = vdiv(vfma(om.y, m.y, vmul(om.x, m.x)), den);
        }
        const float m15uu = cmul(-1.5f, vfma(u[2], u[2], vfma(u[1], u[1], vmul(u[0], u[0]))));
        float2 nuF = vmul(vsplat(u[0], F[0]), F[0]);
        nuF = vneg(vfma(vsplat(u[2], F[2]), F[2], vfma(vsplat(u[1], F[1]), F[1], nuF)));
        const size_t zp = (size_t)(z + 1 < L.nz ? z + 1 : 0) * pxy + own, zm = (size_t)(z > 0 ? z - 1 : L.nz - 1) * pxy + own;
        float *__restrict__ fn = L.f[parity ^ 1];
        // post-collision value of direction i: Eq. (2) less w rho as geq,
        // Eq. (5) as 3 (1 - omega/2) w [(e.F)(1 + 3 e.u) - u.F], re-referenced
        // to the destination's density
        auto push = [&](auto Ic, float qv, float2 X) {
            constexpr int I = decltype(Ic)::value, EX = ex(I), EY = ey(I), EZ = ez(I), C = e2(I);
            constexpr float w = (float)w19(I);
            const float2 aw3 = make_float2(L.aw3[0][C], L.aw3[1][C]);
            const float2 geq = vfma(cmul(w, rho), vsplat(qv, rho), cmul(w, dg));
            float2 v = vfma(aw3, X, vfma(om, vsub(geq, h[I]), h[I]));
            if constexpr (I != 0) v = cfma(w, vsub(rho, sm.rho[rp[2 + EZ]][cy + EY][cx + EX]), v);
            float *d = fn + ((EZ > 0 ? zp : EZ < 0 ? zm : c) + (long long)(EX > 0 ? oE : EX < 0 ? oW : 0) +
                             (EY > 0 ? oN : EY < 0 ? oS : 0));
            d[(size_t)I * plane] = v.x;
            d[(size_t)(19 + I) * plane] = v.y;
        };
        push(std::integral_constant<int, 0>{}, m15uu, nuF);
        auto pair = [&](auto Ic) {
            constexpr int I = decltype(Ic)::value, E[3] = {ex(I), ey(I), ez(I)};
            // e.u and e.F of direction I; its opposite has them negated
            float eu = 0.f;
            float2 eF = make_float2(0.f, 0.f);
            bool first = true;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (E[a] == 0) continue;
                eu = first ? u[a] : (E[a] > 0 ? vadd(eu, u[a]) : vsub(eu, u[a]));
                eF = first ? F[a] : (E[a] > 0 ? vadd(eF, F[a]) : vsub(eF, F[a]));
                first = false;
            }
            const float sq = vfma(cmul(4.5f, eu), eu, m15uu);
            push(Ic, cfma(3.f, eu, sq), vfma(eF, vsplat(cfma(3.f, eu, 1.f), eF), nuF));
            push(std::integral_constant<int, I + 1>{}, cfma(-3.f, eu, sq), vfma(eF, vsplat(cfma(3.f, eu, -1.f), eF), nuF));
        };
        pair(std::integral_constant<int, 1>{});
        pair(std::integral_constant<int, 3>{});
        pair(std::integral_constant<int, 5>{});
        pair(std::integral_constant<int, 7>{});
        pair(std::integral_constant<int, 9>{});
        pair(std::integral_constant<int, 11>{});
        pair(std::integral_constant<int, 13>{});
        pair(std::integral_constant<int, 15>{});
        pair(std::integral_constant<int, 17>{});
    }
}

// Per-node diagnostics reduced per tile into FP64 partials: masses, momenta
// with half force (Eq. 6), max |ubar| (Eq. 7), non-finite count, and the
// Laplace probe's inside / outside sums of the Eq. (11) bulk pressure and of
// rho_A; optional dense FP64 fields rho [2][nz][ny][nx], ubar [3][..].
template <typename real>
__global__ void __launch_bounds__(kThreads) k3_observe(const Lat3<real> L, int parity, double *__restrict__ partials,
                                                       double *__restrict__ out_rho, double *__restrict__ out_u)
{
    Stage3<real> &sm = *reinterpret_cast<Stage3<real> *>(lb3_smem);
    double(*sacc)[kSumRow3] = reinterpret_cast<double(*)[kSumRow3]>(lb3_smem);
    int x0, y0, z0;
    tile_origin(L.tiles_x, L.tiles_y, blockIdx.x, x0, y0, z0);
    const int tid = (threadIdx.z * TY + threadIdx.y) * TX + threadIdx.x;
    stage3<real>(L, L.rho[parity ^ 1], x0, y0, z0, sm, tid);
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, z = z0 + threadIdx.z;
    double acc[kNumAcc];
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) acc[a] = 0.0;
    if (x < L.nx && y < L.ny && z < L.nz) {
        const int cx = threadIdx.x + HALO, cy = threadIdx.y + HALO, cz = threadIdx.z + HALO;
        const size_t c = ((size_t)z * L.ny + y) * L.pitch + x;
        double r[2], m[2][3];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            real F[3];
            force3<real>(L, sm, k, cx, cy, cz, F);
            double j[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                const double fi = (double)L.f[parity][(size_t)(k * 19 + i) * L.plane + c];
                j[0] += fi * ex(i);
                j[1] += fi * ey(i);
                j[2] += fi * ez(i);
            }
            r[k] = (double)sm.rho[k][cz][cy][cx];
#pragma unroll
            for (int a = 0; a < 3; ++a) m[k][a] = j[a] + 0.5 * (double)F[a];
        }
        const double rt = r[0] + r[1];
        double ub[3], u2 = 0.0;
        bool fin = isfinite(r[0]) && isfinite(r[1]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ub[a] = (m[0][a] + m[1][a]) / rt;
            u2 += ub[a] * ub[a];
            fin = fin && isfinite(ub[a]);
        }
        acc[0] = r[0];
        acc[1] = r[1];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc[2 + a] = m[0][a];
            acc[5 + a] = m[1][a];
        }
        acc[8] = u2;   // the square root is taken of the largest
        acc[9] = fin ? 0.0 : 1.0;
        if (L.has_probe) {
            const int Ls[3] = {L.nx, L.ny, L.nz};
            const int p[3] = {x, y, z};
            double rr2 = 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double d = fabs((double)p[a] - L.probe[a]);
                if (d > 0.5 * Ls[a]) d = Ls[a] - d;
                rr2 += d * d;
            }
            const double rr = sqrt(rr2), R = L.probe[3];
            const double psiA = 1.0 - exp(-r[0]), psiB = 1.0 - exp(-r[1]);
            const double Gs = (double)L.G1 + (double)L.G2;
            const double pb = (r[0] + 0.5 * Gs * psiA * psiA) / 3.0 + (r[1] + 0.5 * Gs * psiB * psiB) / 3.0
                            + (double)L.GAB * r[0] * r[1] / 3.0;
            if (rr < 0.5 * R) { acc[10] = pb; acc[11] = r[0]; acc[12] = 1.0; }
            if (rr > R + 6.0) { acc[13] = pb; acc[14] = r[0]; acc[15] = 1.0; }
        }
        if (out_rho) {
            const size_t n = (size_t)L.nx * L.ny * L.nz, d = ((size_t)z * L.ny + y) * L.nx + x;
            out_rho[d] = r[0];
            out_rho[n + d] = r[1];
            if (out_u)
#pragma unroll
                for (int a = 0; a < 3; ++a) out_u[a * n + d] = ub[a];
        }
    }
    if (!partials) return;
    // through shared memory, 16 values a thread (as the 2-D observables)
    __syncthreads();   // the stage has been read
#pragma unroll
    for (int a = 0; a < kNumAcc; ++a) sacc[a][tid + tid / kSumRun3] = acc[a];
    __syncthreads();
    const int a = tid / kSumRun3, l = tid % kSumRun3;
    double v = sacc[a][l * (kSumRun3 + 1)];
#pragma unroll
    for (int q = 1; q < kSumRun3; ++q) {
        const double w = sacc[a][l * (kSumRun3 + 1) + q];
        v = a == 8 ? fmax(v, w) : v + w;
    }
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const double w = __shfl_xor_sync(0xffffffffu, v, o);
        v = a == 8 ? fmax(v, w) : v + w;
    }
    if (l == 0) partials[(size_t)blockIdx.x * kNumAcc + a] = v;
}

// Block b: the b-th of gridDim.x runs of the records, summed (max for |u|^2)
// in a fixed order into out[b].
static __global__ void __launch_bounds__(256) k3_reduce(const double *__restrict__ partials, int n_rec,
                                                        double *__restrict__ out)
{
    __shared__ double s[256 / 32][kNumAcc];
    const int run = (n_rec + gridDim.x - 1) / gridDim.x, t0 = blockIdx.x * run, t1 = min(t0 + run, n_rec);
    const int a = threadIdx.x % kNumAcc;   // 16 threads a record
    double v = 0.0;
    for (int t = t0 + threadIdx.x / kNumAcc; t < t1; t += 256 / kNumAcc) {
        const double w = partials[(size_t)t * kNumAcc + a];
        v = a == 8 ? fmax(v, w) : v + w;
    }
    const double w = __shfl_xor_sync(0xffffffffu, v, 16);
    v = a == 8 ? fmax(v, w) : v + w;
    if (threadIdx.x % 32 < kNumAcc) s[threadIdx.x / 32][a] = v;
    __syncthreads();
    if (threadIdx.x < kNumAcc) {
        v = s[0][a];
        for (int q = 1; q < 256 / 32; ++q) v = a == 8 ? fmax(v, s[q][a]) : v + s[q][a];
        out[(size_t)blockIdx.x * kNumAcc + a] = v;
    }
}

// f = f^eq(rho_k, u) (Eq. 2) from dense FP64 fields; FP32 stores R = rho
// (rounded) and the offsets f^eq - w R
template <typename real>
__global__ void k3_init(const Lat3<real> L, const double *__restrict__ rho, const double *__restrict__ u, int parity)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= L.nx) return;
    const size_t n = (size_t)L.nx * L.ny * L.nz, d = ((size_t)z * L.ny + y) * L.nx + x;
    const size_t c = ((size_t)z * L.ny + y) * L.pitch + x;
    const double ux = u ? u[d] : 0.0, uy = u ? u[n + d] : 0.0, uz = u ? u[2 * n + d] : 0.0;
    const double uu = ux * ux + uy * uy + uz * uz;
    for (int k = 0; k < 2; ++k) {
        const double r = rho[k * n + d];
        double R = 0.0;
        if constexpr (kOffset3<real>) {
            const real Rr = (real)r;
            L.rho[parity][(size_t)k * L.plane + c] = Rr;
            R = (double)Rr;
        }
        for (int i = 0; i < 19; ++i) {
            const double eu = ex(i) * ux + ey(i) * uy + ez(i) * uz;
            const double feq = w19(i) * r * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
            L.f[parity][(size_t)(k * 19 + i) * L.plane + c] = (real)(feq - w19(i) * R);
        }
    }
}

// populations as dense FP64 [2][19][nz][ny][nx] (FP32: w_i R added back)
template <typename real>
__global__ void k3_get_pops(const Lat3<real> L, int parity, double *__restrict__ out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= L.nx) return;
    const size_t n = (size_t)L.nx * L.ny * L.nz, d = ((size_t)z * L.ny + y) * L.nx + x;
    const size_t c = ((size_t)z * L.ny + y) * L.pitch + x;
    for (int k = 0; k < 2; ++k) {
        const double R = kOffset3<real> ? (double)L.rho[parity][(size_t)k * L.plane + c] : 0.0;
        for (int i = 0; i < 19; ++i)
            out[(size_t)(k * 19 + i) * n + d] = (double)L.f[parity][(size_t)(k * 19 + i) * L.plane + c] + w19(i) * R;
    }
}

}  // namespace lbk3

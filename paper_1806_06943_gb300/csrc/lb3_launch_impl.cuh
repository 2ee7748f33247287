// lb3_launch_impl.cuh -- definitions of the 3-D launchers; included once per
// population format.
#pragma once

#include "lb3_launch.h"

namespace lbk3 {

template <typename real>
cudaError_t Launch3<real>::density(const Lat3<real> &L, int parity, bool step, cudaStream_t s)
{
    const unsigned n = (unsigned)L.tiles_x * L.tiles_y * L.tiles_z;
    if constexpr (!kOffset3<real>)
        if (step) {
            k3_density<real, true><<<n, dim3(TX, TY, TZ), 0, s>>>(L, parity);
            return cudaGetLastError();
        }
    k3_density<real, false><<<n, dim3(TX, TY, TZ), 0, s>>>(L, parity);
    return cudaGetLastError();
}

// Resident blocks per SM of the marching kernel.
constexpr int kMarchBlocks = 2;

// Planes a block marches along z: the whole column, or segments of it where
// columns alone do not fill the device evenly.  A segment forms the densities of
// 4 more planes than it steps, 0.4 of a plane's work each, and a wave of two
// blocks per SM takes 1.45 times as long as one of a single block.  Microseconds
// a step by planes (blocks): 33 x 33 x 32 3 (110) 21.0, 2 (160) 24.8, 1 (320) 24.8;
// 75 x 38 x 32 2 (240) 24.8, 4 (120) 26.8; 64^3 4 (256) 36.9, 8 (128) 42.2; 160^3
// 54 (300) 422, 27 (600) 417, 20 (800) 455.
inline int march_planes(int64_t columns, int nz, int sms)
{
    constexpr double kRim = 4 * 0.4, kPair = 1.45;
    static_assert(kMarchBlocks == 2, "the cost of a wave counts one or two blocks per SM");
    int best = nz;
    double cost = 1e300;
    for (int segs = 1; segs <= nz; ++segs) {
        const int lz = (nz + segs - 1) / segs;
        if ((nz + lz - 1) / lz != segs) continue;
        const int64_t blocks = columns * segs, waves = blocks / (2 * sms), rest = blocks % (2 * sms);
        const double c = (kPair * (double)waves + (rest == 0 ? 0.0 : rest <= sms ? 1.0 : kPair)) * (lz + kRim);
        if (c < cost * 0.999) {
            cost = c;
            best = lz;
        }
    }
    return best;
}

template <typename real>
cudaError_t Launch3<real>::prepare(const Lat3<real> &L, int sms, int &march)
{
    if constexpr (kOffset3<real>) {
        march = march_planes((int64_t)L.tiles_x * ((L.ny + RY - 1) / RY), L.nz, sms);
        return cudaFuncSetAttribute(k3_march<kMarchBlocks>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(March3));
    } else {
        march = 0;
        return cudaFuncSetAttribute(k3_collide<real>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kCollideSmem3<real>);
    }
}

template <typename real>
cudaError_t Launch3<real>::step(const Lat3<real> &L, int parity, int march, cudaStream_t s)
{
    if constexpr (kOffset3<real>) {
        const int tiles_y = (L.ny + RY - 1) / RY;
        const unsigned n = (unsigned)((int64_t)L.tiles_x * tiles_y * ((L.nz + march - 1) / march));
        k3_march<kMarchBlocks><<<n, dim3(TX, RY), sizeof(March3), s>>>(L, parity, tiles_y, march);
        return cudaGetLastError();
    } else {
        cudaError_t e = density(L, parity, true, s);
        if (e == cudaSuccess) e = collide3(L, parity, s);
        return e;
    }
}

template <typename real>
cudaError_t Launch3<real>::observe(const Lat3<real> &L, int parity, double *partials, double *rho, double *u,
                                   cudaStream_t s)
{
    const unsigned n = (unsigned)L.tiles_x * L.tiles_y * L.tiles_z;
    cudaError_t e = cudaFuncSetAttribute(k3_observe<real>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kObserveSmem3<real>);
    if (e != cudaSuccess) return e;
    k3_observe<real><<<n, dim3(TX, TY, TZ), kObserveSmem3<real>, s>>>(L, parity, partials, rho, u);
    return cudaGetLastError();
}

template <typename real>
cudaError_t Launch3<real>::init(const Lat3<real> &L, const double *rho, const double *u, int parity, cudaStream_t s)
{
    k3_init<real><<<dim3((L.nx + 127) / 128, L.ny, L.nz), 128, 0, s>>>(L, rho, u, parity);
    return cudaGetLastError();
}

template <typename real>
cudaError_t Launch3<real>::get_pops(const Lat3<real> &L, int parity, double *out, cudaStream_t s)
{
    k3_get_pops<real><<<dim3((L.nx + 127) / 128, L.ny, L.nz), 128, 0, s>>>(L, parity, out);
    return cudaGetLastError();
}

}  // namespace lbk3

// lb3_fp64.cu -- FP64 instantiation of the 3-D kernels.  Compiled with
// -fmad=false: every FP64 operation rounds once, in the order written.
#include "lb3_launch_impl.cuh"

namespace lbk3 {
template struct Launch3<double>;

cudaError_t collide3(const Lat3<double> &L, int parity, cudaStream_t s)
{
    const unsigned n = (unsigned)L.tiles_x * L.tiles_y * L.tiles_z;
    k3_collide<double><<<n, dim3(TX, TY, TZ), kCollideSmem3<double>, s>>>(L, parity);
    return cudaGetLastError();
}

cudaError_t reduce3(double *partials, int n_tiles, double *out, cudaStream_t s)
{
    // one block took 1.5 ms over a 160^3 lattice's 16000 tiles: fold them first
    // (observables without and with the fold: 512 tiles 104 and 105 us, 1024 164 and 154)
    double *fold = partials + (size_t)n_tiles * kNumAcc;
    const int blocks = n_tiles > 768 ? kFold3 : 1;
    if (blocks > 1) {
        k3_reduce<<<blocks, 256, 0, s>>>(partials, n_tiles, fold);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    k3_reduce<<<1, 256, 0, s>>>(blocks > 1 ? fold : partials, blocks > 1 ? blocks : n_tiles, out);
    return cudaGetLastError();
}
}  // namespace lbk3

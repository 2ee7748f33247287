// lb3_launch.h -- host-side launchers of the 3-D kernels, one explicit
// instantiation per population format (lb3_fp64.cu, lb3_fp32.cu).
#pragma once

#include <cuda_runtime.h>

#include "lb3_kernels.cuh"

namespace lbk3 {

template <typename real>
struct Launch3 {
    // shared memory of the step's kernel on the current device, and the planes
    // a block marches (FP32); call before the first step
    static cudaError_t prepare(const Lat3<real> &L, int sms, int &march);
    // one time step: FP32 in one pass (k3_march), FP64 density pass + collide
    static cudaError_t step(const Lat3<real> &L, int parity, int march, cudaStream_t s);
    // step: the density pass of a step (FP64: leaves psi as well), else of the observables
    static cudaError_t density(const Lat3<real> &L, int parity, bool step, cudaStream_t s);
    static cudaError_t observe(const Lat3<real> &L, int parity, double *partials, double *rho, double *u,
                               cudaStream_t s);
    static cudaError_t init(const Lat3<real> &L, const double *rho, const double *u, int parity, cudaStream_t s);
    static cudaError_t get_pops(const Lat3<real> &L, int parity, double *out, cudaStream_t s);
};

// The tile partials' sums into out; partials has room for kFold3 records
// behind the n_tiles.
constexpr int kFold3 = 64;
cudaError_t reduce3(double *partials, int n_tiles, double *out, cudaStream_t s);

// the FP64 step after its density pass
cudaError_t collide3(const Lat3<double> &L, int parity, cudaStream_t s);

extern template struct Launch3<double>;
extern template struct Launch3<float>;

}  // namespace lbk3

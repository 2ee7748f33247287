// lb_tables.cu -- the table of exp(-j/512) the FP64 kernels read (lb_f64.cuh),
// formed once per process in extended precision and kept by each handle on its
// device.
#include <cmath>
#include <mutex>
#include <vector>

#include "lb_f64.cuh"
#include "lb_launch.h"

namespace lbk {

cudaError_t make_exp_table(double2 **out, cudaStream_t s)
{
    static std::vector<double2> host;
    static std::once_flag once;
    std::call_once(once, [] {
        host.resize(kExpSize);
        for (int j = 0; j < kExpSize; ++j) {
            const long double e = expl(-(long double)j / kExpSteps);
            host[j].x = (double)e;
            host[j].y = (double)(e - (long double)host[j].x);
        }
    });
    cudaError_t e = cudaMalloc((void **)out, kExpSize * sizeof(double2));
    if (e == cudaSuccess) e = cudaMemcpyAsync(*out, host.data(), kExpSize * sizeof(double2), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    return e;
}

}  // namespace lbk

// lb_tables.cu -- the table of exp(-j/512) the FP64 kernels read (lb_f64.cuh),
// formed once per process in extended precision and kept by each handle on its
// device.
#include <array>
#include <cmath>

#include "lb_f64.cuh"
#include "lb_launch.h"

namespace lbk {

cudaError_t make_exp_table(double2 **out, cudaStream_t s)
{
    static const std::array<double2, kExpSize> host = [] {
        std::array<double2, kExpSize> t{};
        for (int j = 0; j < kExpSize; ++j) {
            const long double e = expl(-(long double)j / kExpSteps);
            t[j].x = (double)e;
            t[j].y = (double)(e - (long double)t[j].x);
        }
        return t;
    }();
    double2 *table = nullptr;
    cudaError_t e = cudaMalloc((void **)&table, kExpSize * sizeof(double2));
    if (e != cudaSuccess) {
        cudaGetLastError();   // not left for the next launch's check to find
        return e;
    }
    e = cudaMemcpyAsync(table, host.data(), kExpSize * sizeof(double2), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) *out = table;
    else cudaFree(table);
    return e;
}

}  // namespace lbk

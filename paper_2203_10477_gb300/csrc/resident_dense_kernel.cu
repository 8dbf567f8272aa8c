// resident_dense_kernel.cu -- the resident kernel for runs with more than two
// probes in some window (resident.cuh, DENSE), a translation unit of its own.

#include "resident.cuh"

namespace rswr {

using namespace resident;

const void* res_dense_kernel(int dtype, int P)
{
#define RSWR_DENSE(DT, Real, FORM, N) \
    if (dtype == DT && P == N) return reinterpret_cast<const void*>(&resident_kernel<Real, FORM, N, true>);
    RSWR_DENSE(kF32, float, kIncrement, 4)
    RSWR_DENSE(kF32, float, kIncrement, 8)
    RSWR_DENSE(kF32, float, kIncrement, 16)
    RSWR_DENSE(kF32, float, kIncrement, 32)
    RSWR_DENSE(kF64, double, kCanonical, 1)
    RSWR_DENSE(kF64, double, kCanonical, 2)
    RSWR_DENSE(kF64, double, kCanonical, 4)
    RSWR_DENSE(kF64, double, kCanonical, 8)
    RSWR_DENSE(kF64, double, kCanonical, 12)
    RSWR_DENSE(kF64, double, kCanonical, 16)
#undef RSWR_DENSE
    return nullptr;
}

}  // namespace rswr

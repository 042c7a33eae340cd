// Instances of the on-chip CG kernel (resident.cuh): FP64, L <= 20.
#include "resident.cuh"

namespace hol {

ResKernel resident_kernel_f64(int L, int K)
{
    switch (L) {
#define X(LL) case LL: return resident_instance<double, LL>(K, false);
        X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20)
#undef X
    }
    return ResKernel{0, 0, 0, nullptr};
}

}  // namespace hol

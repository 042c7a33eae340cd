// Instances of the on-chip CG kernel (resident.cuh): FP32, L <= 12.
#include "resident.cuh"

namespace hol {

ResKernel resident_kernel_f32_small(int L, int K, bool tm)
{
    switch (L) {
#define X(LL) case LL: return resident_instance<float, LL>(K, tm);
        X(4) X(6) X(8) X(10) X(12)
#undef X
    }
    return ResKernel{0, 0, 0, nullptr};
}

}  // namespace hol

// Instances of the on-chip CG kernel (resident.cuh): FP32, 14 <= L <= 22.
#include "resident.cuh"

namespace hol {

ResKernel resident_kernel_f32_mid(int L, int K, bool tm)
{
    switch (L) {
#define X(LL) case LL: return resident_instance<float, LL>(K, tm);
        X(14) X(16) X(18) X(20) X(22)
#undef X
    }
    return ResKernel{0, 0, 0, nullptr};
}

}  // namespace hol

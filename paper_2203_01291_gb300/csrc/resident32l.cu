// Instances of the on-chip CG kernel (resident.cuh): FP32, L >= 24.
#include "resident.cuh"

namespace hol {

ResKernel resident_kernel_f32_large(int L, int K, bool tm)
{
    switch (L) {
#define X(LL) case LL: return resident_instance<float, LL>(K, tm);
        X(24) X(26) X(28) X(30) X(32)
#undef X
    }
    return ResKernel{0, 0, 0, nullptr};
}

}  // namespace hol

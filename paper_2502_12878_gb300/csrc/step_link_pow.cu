// Linked persistent launch of the power iteration (link_kernel with
// MODE_POWER64, step_link.cuh): the stencil sizes of step_link.cu.
#include "step_link.cuh"

namespace rbffd {

template <int TH>
static StepFn pick_pow(int n) {
#define RBFFD_PCASE(NN) \
    case NN: return link_kernel<NN, MODE_POWER64, TH>;
    switch (n) {
        RBFFD_PCASE(12)
        RBFFD_PCASE(13)
        RBFFD_PCASE(16)
        RBFFD_PCASE(20)
        RBFFD_PCASE(24)
        RBFFD_PCASE(30)
        RBFFD_PCASE(31)
        default: break;
    }
    if constexpr (TH == RES_THREADS_HOST) {
        switch (n) {
            RBFFD_PCASE(6)
            RBFFD_PCASE(40)
            RBFFD_PCASE(48)
            RBFFD_PCASE(56)
            RBFFD_PCASE(57)
            RBFFD_PCASE(70)
            RBFFD_PCASE(71)
            default: return link_kernel<0, MODE_POWER64, TH>;
        }
    }
    return nullptr;
#undef RBFFD_PCASE
}

StepFn pick_link_power(int n, int threads) {
    return threads == RES_THREADS_WIDE ? pick_pow<RES_THREADS_WIDE>(n)
                                       : pick_pow<RES_THREADS_HOST>(n);
}

}  // namespace rbffd

// Linked persistent launch: the kernel instantiations (the kernel itself is in
// step_link.cuh) - 512-thread blocks for every compiled stencil size, 1024
// threads where the kernel fits 64 registers (n <= 31) - and the shared memory
// of a launch.
#include "step_link.cuh"

namespace rbffd {

template <int MODE>
static StepFn pick_link_512(int n) {
#define RBFFD_LCASE(NN) \
    case NN: return link_kernel<NN, MODE, RES_THREADS_HOST>;
    switch (n) {
        RBFFD_LCASE(6)
        RBFFD_LCASE(12)
        RBFFD_LCASE(13)
        RBFFD_LCASE(16)
        RBFFD_LCASE(20)
        RBFFD_LCASE(24)
        RBFFD_LCASE(30)
        RBFFD_LCASE(31)
        RBFFD_LCASE(40)
        RBFFD_LCASE(48)
        RBFFD_LCASE(56)
        RBFFD_LCASE(57)
        RBFFD_LCASE(70)
        RBFFD_LCASE(71)
        default: return link_kernel<0, MODE, RES_THREADS_HOST>;
    }
#undef RBFFD_LCASE
}

template <int MODE>
static StepFn pick_link_1024(int n) {
#define RBFFD_LCASE(NN) \
    case NN: return link_kernel<NN, MODE, RES_THREADS_WIDE>;
    switch (n) {
        RBFFD_LCASE(12)
        RBFFD_LCASE(13)
        RBFFD_LCASE(16)
        RBFFD_LCASE(20)
        RBFFD_LCASE(24)
        RBFFD_LCASE(30)
        RBFFD_LCASE(31)
        default: return nullptr;
    }
#undef RBFFD_LCASE
}

StepFn pick_link(int mode, int n, int threads) {
    if (threads == RES_THREADS_WIDE)
        return mode == MODE_SWEEP64 ? pick_link_1024<MODE_SWEEP64>(n)
                                    : pick_link_1024<MODE_INNER32>(n);
    return mode == MODE_SWEEP64 ? pick_link_512<MODE_SWEEP64>(n) : pick_link_512<MODE_INNER32>(n);
}

unsigned link_smem(int64_t nslices, int n, int mode, int grid, int64_t halo) {
    return link_layout((nslices + grid - 1) / grid, n, mode == MODE_SWEEP64 ? 8 : 4, halo).total;
}

}  // namespace rbffd

// Instances of the persistent kernel for variant 9: the column path of the
// exact (6, 4, 3) variant with one-byte flip words (no layered schedule).
#include "bpsf_persistent.cuh"

namespace bpsf {

typedef void (*KernelFn)(KernelParams);

KernelFn kernel_fn_v9(bool debug, bool lay) {
    if (lay) return nullptr;
    return debug ? bpsf_persistent<6, 4, 3, true, 1, false, 1, false, true>
                 : bpsf_persistent<6, 4, 3, false, 1, false, 1, false, true>;
}

}  // namespace bpsf

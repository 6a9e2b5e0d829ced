// Instances of the persistent kernel for variant 11: the column path of codes
// of exactly ten ones per row and five per column with one-byte flip words.
#include "bpsf_persistent.cuh"

namespace bpsf {

typedef void (*KernelFn)(KernelParams);

KernelFn kernel_fn_v11(bool debug, bool lay) {
    if (lay) return nullptr;
    return debug ? bpsf_persistent<10, 8, 5, true, 1, false, 1, false, true>
                 : bpsf_persistent<10, 8, 5, false, 1, false, 1, false, true>;
}

}  // namespace bpsf

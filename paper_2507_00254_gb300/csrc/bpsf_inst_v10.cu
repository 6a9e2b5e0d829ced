// Instances of the persistent kernel for variant 10: the column path of codes
// of exactly ten ones per row and five per column with two-byte flip words.
#include "bpsf_persistent.cuh"

namespace bpsf {

typedef void (*KernelFn)(KernelParams);

KernelFn kernel_fn_v10(bool debug, bool lay) {
    if (lay) return nullptr;
    return debug ? bpsf_persistent<10, 8, 5, true, 1, false, 2, false, true>
                 : bpsf_persistent<10, 8, 5, false, 1, false, 2, false, true>;
}

}  // namespace bpsf

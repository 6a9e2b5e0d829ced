// Instances of the persistent kernel for variant 12: the column path of long
// codes (up to eight ones per row, three per column), two-byte flip words.
#include "bpsf_persistent.cuh"

namespace bpsf {

typedef void (*KernelFn)(KernelParams);

KernelFn kernel_fn_v12(bool debug, bool lay) {
    if (lay) return nullptr;
    return debug ? bpsf_persistent<8, 4, 0, true, 1, false, 2, false, true>
                 : bpsf_persistent<8, 4, 0, false, 1, false, 2, false, true>;
}

}  // namespace bpsf

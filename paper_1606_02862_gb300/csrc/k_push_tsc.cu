// k_push_tsc.cu -- the push kernel for contexts whose mobile species are all TSC
// with the momentum-conserving gather.
#include "k_push.cuh"

namespace pic {

PIC_PUSH_DEFINE(2, PIC_PUSH_CASES_G1)

}  // namespace pic

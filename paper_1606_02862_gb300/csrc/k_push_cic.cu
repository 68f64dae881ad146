// k_push_cic.cu -- the push kernel for contexts whose mobile species are all CIC
// with the momentum-conserving gather.
#include "k_push.cuh"

namespace pic {

PIC_PUSH_DEFINE(1, PIC_PUSH_CASES_G1)

}  // namespace pic

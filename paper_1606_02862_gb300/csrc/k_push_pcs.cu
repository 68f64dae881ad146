// k_push_pcs.cu -- the push kernel for contexts whose mobile species are all PCS
// with the momentum-conserving gather.
#include "k_push.cuh"

namespace pic {

PIC_PUSH_DEFINE(3, PIC_PUSH_CASES_G2)

}  // namespace pic

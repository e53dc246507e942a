// ed_matvec_slot_f64_torus.cu -- the slot-index matvec for f64 vectors, torus translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_f64_torus(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<double, false, 2, 1>(a, track, el, s);
}
}  // namespace edk

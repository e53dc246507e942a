// ed_matvec_slot_f32_torus.cu -- the slot-index matvec for f32 vectors, torus translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_f32_torus(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, false, 2, 1>(a, track, el, s);
}
}  // namespace edk

// ed_matvec_slot_c64_torus.cu -- the slot-index matvec for c64 vectors, torus translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_c64_torus(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, true, 2, 1>(a, track, el, s);
}
}  // namespace edk

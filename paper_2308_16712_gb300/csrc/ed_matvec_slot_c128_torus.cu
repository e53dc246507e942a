// ed_matvec_slot_c128_torus.cu -- the slot-index matvec for c128 vectors, torus translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_c128_torus(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<double, true, 2, 1>(a, track, el, s);
}
}  // namespace edk

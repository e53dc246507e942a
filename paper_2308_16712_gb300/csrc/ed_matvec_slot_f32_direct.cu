// ed_matvec_slot_f32_direct.cu -- the slot-order matvec without the slotted copy, f32 vectors.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_direct_f32(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, false, 0, 1, true>(a, track, el, s);
}
cudaError_t slotn_direct_f32(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, false, 0, kMaxSectors, true>(a, track, el, s);
}
}  // namespace edk

// ed_matvec_slot_f32_ring.cu -- the slot-index matvec for f32 vectors, ring translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_f32_ring(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, false, 1, 1>(a, track, el, s);
}
cudaError_t slotn_f32_ring(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, false, 1, kMaxSectors>(a, track, el, s);
}
}  // namespace edk

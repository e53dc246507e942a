// ed_matvec_slot_c64_ring.cu -- the slot-index matvec for c64 vectors, ring translations.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_c64_ring(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, true, 1, 1>(a, track, el, s);
}
cudaError_t slotn_c64_ring(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<float, true, 1, kMaxSectors>(a, track, el, s);
}
}  // namespace edk

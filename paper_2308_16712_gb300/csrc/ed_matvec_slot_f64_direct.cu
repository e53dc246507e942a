// ed_matvec_slot_f64_direct.cu -- the slot-order matvec without the slotted copy, f64 vectors.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_direct_f64(const SlotArgs<1> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<double, false, 0, 1, true>(a, track, el, s);
}
cudaError_t slotn_direct_f64(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s)
{
    return slot_dispatch<double, false, 0, kMaxSectors, true>(a, track, el, s);
}
}  // namespace edk

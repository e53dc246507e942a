// ed_matvec_slot_c128.cu -- the slot-index matvec for c128 vectors: the choice of
// search, and the variants that visit every element of the group.
#include "ed_matvec_slot.cuh"

namespace edk {
cudaError_t slot1_c128_ring(const SlotArgs<1> &a, bool track, int el, cudaStream_t s);
cudaError_t slot1_c128_torus(const SlotArgs<1> &a, bool track, int el, cudaStream_t s);
cudaError_t slotn_c128_ring(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s);

cudaError_t slot1_c128(const SlotArgs<1> &a, int search, bool track, int el, cudaStream_t s)
{
    return search == 1   ? slot1_c128_ring(a, track, el, s)
           : search == 2 ? slot1_c128_torus(a, track, el, s)
                         : slot_dispatch<double, true, 0, 1>(a, track, el, s);
}

// a batch on a torus takes the general search
cudaError_t slotn_c128(const SlotArgs<kMaxSectors> &a, int search, bool track, int el, cudaStream_t s)
{
    return search == 1 ? slotn_c128_ring(a, track, el, s) : slot_dispatch<double, true, 0, kMaxSectors>(a, track, el, s);
}
}  // namespace edk

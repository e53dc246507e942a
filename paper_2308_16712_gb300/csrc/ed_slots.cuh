// ed_slots.cuh -- slot index: the position of a state's value in a copy of x
// laid out for gathering, found from the state with one byte of table.
//
// A product over a sector beyond L2 is bound by random DRAM reads (about 5e10
// per second on GB300 whatever their size up to 32 bytes), and stateToIndex
// through a hash or bucketed index costs one such read per matrix element
// before the read of x.  Every representative that a term can produce is known
// when the basis is built, so a perfect hash function does without the states.
// The range of states is cut into equal cells (s >> shift), in their order; the
// keys of a cell fall by hash into its partitions of about kSlotPartKeys, a
// partition into 2^kSlotLogB buckets of 3.5 keys on average, and each bucket
// stores one pilot byte chosen so that hash(key, pilot) gives all keys of the
// partition distinct slots.  The table takes 2.3 bits per key (18 MB at 6.3e7
// states), stays in L2, and leaves one random DRAM read per matrix element, of
// x itself.  The cells (some 10^5 keys each) keep the sorted basis's locality:
// rows are processed in ascending order, and the terms that change only low
// bits find their slots where the neighbouring rows found theirs.
//
// The function maps states that are no keys to arbitrary slots, so it may only
// be asked for keys: the representatives of the sector's popcount.  Those whose
// orbit carries no weight in the sector (norm 0, not in the basis) are keys
// too, with value 0 in the slotted copy of x.
#pragma once

#include <stdint.h>

#include <cstring>

namespace edk {

constexpr int kSlotLogB = 11;                 // buckets per partition
constexpr uint32_t kSlotPartKeys = 7168;      // keys per partition (average, at most)
constexpr uint32_t kSlotSmallKeys = 2560;     // the same for up to kSlotSmallMax keys: at load 0.3 the
constexpr uint64_t kSlotSmallMax = 1u << 18;  // longest pilot search of a partition takes 0.05 ms, not 0.3
constexpr uint32_t kSlotCap = 8533;           // slots per partition: load 0.84, and room for any
                                              // partition (16 sigma above the average)
constexpr uint32_t kPilotEscape = 255;        // pilot kept in the exception table instead

struct SlotView {
    const uint8_t *pilots;      // null: the basis has no slot index
    const uint2 *cells;         // {first bucket, buckets} of each cell
    int shift;                  // cell of a state: s >> shift
    uint32_t n_cells;
    const uint2 *exc;           // exceptions: open addressing, {bucket, pilot}, ~0 empty
    uint32_t exc_mask;
    const uint64_t *ghosts;     // representatives of norm 0
    uint32_t n_ghost;
    uint64_t n_slots;
};

struct SlotKey {
    uint32_t hi, lo;
};

// 64 well-mixed bits of a state
__host__ __device__ __forceinline__ SlotKey slot_key(uint64_t s)
{
    uint64_t t = s * 0x9E3779B97F4A7C15ULL;
    t ^= t >> 32;
    t *= 0xD6E8FEB86659FD93ULL;
    return SlotKey{(uint32_t)(t >> 32), (uint32_t)t};
}

__host__ __device__ __forceinline__ uint32_t mul_high(uint32_t a, uint32_t b)
{
    return (uint32_t)(((uint64_t)a * b) >> 32);
}

__host__ __device__ __forceinline__ uint32_t slot_cell(uint64_t s, const SlotView &v)
{
    const uint32_t c = (uint32_t)(s >> v.shift);
    return c < v.n_cells ? c : v.n_cells - 1;
}

// slot of a key within its partition under a pilot; both words enter through
// products that depend on the pilot, so two keys that differ at all part ways
// under some pilot
__host__ __device__ __forceinline__ uint32_t slot_place(SlotKey k, uint32_t pilot)
{
    const uint32_t x = (k.lo ^ (pilot * 0x9E3779B1u)) * 0x85EBCA6Bu + k.hi * (pilot * 0xC2B2AE36u + 1u);
    return mul_high(x, kSlotCap);
}

__host__ __device__ __forceinline__ uint32_t exc_start(uint32_t bucket, uint32_t mask) { return (bucket * 0x9E3779B1u >> 7) & mask; }

#ifdef __CUDACC__
__device__ __forceinline__ uint32_t slot_bucket(uint64_t s, SlotKey k, const SlotView &v)
{
    const uint2 c = __ldg(v.cells + slot_cell(s, v));
    return c.x + mul_high(k.hi, c.y);
}

// L2 eviction policy of the pilots: they stay
__device__ __forceinline__ uint64_t policy_keep()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint32_t load_pilot(const uint8_t *p, uint64_t policy)
{
    uint32_t v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u8 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(policy));
    return v;
}
// kBytes (4, 8 or 16) of a row that is read at random: not kept in L1
template <int kBytes>
__device__ __forceinline__ void load_random(void *out, const void *p)
{
    if constexpr (kBytes == 4) {
        uint32_t a;
        asm("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(a) : "l"(p));
        memcpy(out, &a, 4);
    } else if constexpr (kBytes == 8) {
        uint64_t a;
        asm("ld.global.nc.L1::no_allocate.u64 %0, [%1];" : "=l"(a) : "l"(p));
        memcpy(out, &a, 8);
    } else {
        uint4 a;
        asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w)
                     : "l"(p));
        memcpy(out, &a, 16);
    }
}

// the pilot of a bucket whose byte says kPilotEscape (about 1 bucket in 10^4);
// the table is at most half full, so a probe sequence ends
__device__ __noinline__ static uint32_t slot_exception(uint32_t bucket, const SlotView &v)
{
    uint32_t at = exc_start(bucket, v.exc_mask);
    for (uint32_t i = 0; i <= v.exc_mask; ++i) {
        const uint2 e = __ldg(v.exc + at);
        if (e.x == bucket || e.x == ~0u)
            return e.y;
        at = (at + 1) & v.exc_mask;
    }
    return 0;
}

__device__ __forceinline__ uint32_t slot_finish(SlotKey k, uint32_t bucket, uint32_t pilot, const SlotView &v)
{
    if (pilot == kPilotEscape)
        pilot = slot_exception(bucket, v);
    return (bucket >> kSlotLogB) * kSlotCap + slot_place(k, pilot);
}

__device__ __forceinline__ uint32_t slot_of(uint64_t s, const SlotView &v)
{
    const SlotKey k = slot_key(s);
    const uint32_t b = slot_bucket(s, k, v);
    return slot_finish(k, b, __ldg(v.pilots + b), v);
}
#endif

}  // namespace edk

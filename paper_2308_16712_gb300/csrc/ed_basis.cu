// ed_basis.cu -- basis build (Sec. "States enumeration"): the fixed-popcount
// states whose top bits can begin a representative (k_prefix_viable; all states
// in small sectors) are split into chunks of consecutive combinations; each
// thread unranks its chunk start (combinatorial number system, colex order =
// ascending integers) and walks the chunk with Gosper's next-combination step,
// keeping the states that are their orbit's minimum with nonzero norm.  A count
// pass, an exclusive scan and a write pass give an order-preserving compaction,
// so the result is ascending without a sort.  Then the prefix table used by
// "stateToIndex" is built over it.
#include <cuda_runtime.h>

#include <algorithm>

#include "ed_kernels.cuh"

namespace edk {
namespace {

constexpr int kEnumThreads = 256;

// Device-detected invariant violations of the kernels in this file (bit 0:
// a chunk's write pass disagreed with its count pass).  Read and cleared by
// ed_stream_status.
__device__ unsigned int g_basis_status;

__device__ __forceinline__ uint64_t unrank_colex(uint64_t rank, int n, int k, const uint64_t *binom)
{
    uint64_t s = 0;
    int hi = n;
    for (int i = k; i >= 1; --i) {
        int c = hi - 1;
        while (__ldg(binom + c * 65 + i) > rank)
            --c;
        s |= 1ULL << c;
        rank -= __ldg(binom + c * 65 + i);
        hi = c;
    }
    return s;
}

// Gosper's hack: the next larger integer with the same popcount.
__device__ __forceinline__ uint64_t next_combination(uint64_t s)
{
    const uint64_t u = s & (~s + 1ULL);
    const uint64_t v = s + u;
    return v | (((v ^ s) >> 2) >> (__ffsll((long long)s) - 1));
}

// Orbit norm of s if s is the minimum of its orbit, else 0.  Norm = number of
// group elements fixing s; -1 for a minimum without weight (a fixing element has
// chi != 1: norm 0, not in the basis).
template <typename W>
__device__ __forceinline__ int rep_norm(W s, const W *sm_masks, const uint32_t *sm_one, int n_perm,
                                        int flip, W full)
{
    int stab = 0;
    bool ok = true;
    for (int p = 0; p < n_perm; ++p) {
        const W q = benes_apply(s, sm_masks + p * kMaskStride);
        if (q < s)
            return 0;
        if (q == s) {
            ++stab;
            ok = ok && chi_is_one(sm_one, p);
        }
        if (flip) {
            const W f = q ^ full;
            if (f < s)
                return 0;
            if (f == s) {
                ++stab;
                ok = ok && chi_is_one(sm_one, p + n_perm);
            }
        }
    }
    return ok ? stab : -1;
}

// Same test over the factored group (rotation subgroup x coset representatives).
template <typename W>
__device__ __forceinline__ int rep_norm_fact(W s, const uint8_t *kinds, const W *masks,
                                             const uint32_t *one, const GroupView &g, W full)
{
    int stab = 0;
    bool ok = true, rep = true;
    for_each_image<W>(s, kinds, masks, g.n_cos, g.rot_L, g.rot_d, g.n_sites, g.n_perm, g.flip, full,
                      [&](W q, int gi) {
                          if (q < s) {
                              rep = false;
                              return true;
                          }
                          if (q == s) {
                              ++stab;
                              ok = ok && chi_is_one(one, gi);
                          }
                          return false;
                      });
    return rep ? (ok ? stab : -1) : 0;
}

// Not decided by rep_norm_rot1.
constexpr int kNormOpen = -2;

// Same test for the translations of a ring: s is a representative if no coset
// image has a smaller minimum (rep_search_rot1, one coset at a time), and only
// the identity fixes it if no other coset reaches s, no rotation by n / p (p a
// prime factor of n, plan.turn) does, and the half turn does not complement it:
// any further element of the stabiliser has one of these as a power.  The few
// states with more symmetry are left to rep_norm_fact (kNormOpen).  known: s is
// a representative.  Bound by integer issue slots like the search: some 250
// instructions against 3000 for the 72 images of ring N=36 (a warp always holds
// a state for which every image counts): both passes of its basis 37 -> 10 ms.
template <typename W>
__device__ __forceinline__ int rep_norm_rot1(W s, const uint8_t *kinds, const W *masks, const uint32_t *one,
                                             const GroupView &g, const EnumPlan &plan, W full, bool known)
{
    const int n = g.n_sites;
    GroupView ring = g;  // the rotations alone
    ring.cos_rev = -1;
    ring.n_cos = 0;
    bool alone = true;
    for (int c = 0; c < g.n_cos; ++c) {
        const bool id = c == g.cos_id;
        if (id && known)
            continue;
        W best;
        int gbest;
        rep_search_rot1<W, false>(coset_image(s, (int)kinds[c], masks + c * kMaskStride, n), kinds, masks, ring,
                                  g.flip, full, best, gbest);
        if (best < s)
            return 0;
        alone = alone && (id || best != s);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        alone = alone && (!plan.turn[i] || rotl_n(s, plan.turn[i], n, full) != s);
    if (g.flip && n % 2 == 0)
        alone = alone && rotl_n(s, n / 2, n, full) != (W)(s ^ full);
    return !alone ? kNormOpen : chi_is_one(one, g.cos_id * n) ? 1 : -1;
}

// Same test for the translations of a torus, over the candidates of
// rep_search_blocks: every element that makes the minimum is one of them.
template <typename W>
__device__ __forceinline__ int rep_norm_blocks(W s, const W *masks, const uint32_t *one, const GroupView &g, W full)
{
    int stab = 0;
    bool ok = true;
    const bool rep = blocks_candidates<W>(s, masks, g, g.flip, full, [&](W q, int gi) {
        if (q == s) {
            ++stab;
            ok = ok && chi_is_one(one, gi);
        }
        return q >= s;
    });
    return rep ? (ok ? stab : -1) : 0;
}

__host__ __device__ inline size_t enum_smem_bytes(const GroupView &g, size_t wbytes, bool fact)
{
    const int nm = fact ? g.n_cos : g.n_perm;
    return (size_t)nm * kMaskStride * wbytes + ((g.order + 31) / 32) * 4 + ((nm + 15) / 16) * 16;
}

// The states of a chunk in ascending order: one run of combinations, or the
// segments of an enumeration plan one after the other.
template <bool kU1>
struct StateWalk {
    uint64_t part, left;  // current combination of the low bits, states left in the segment
    uint64_t top;         // the other bits
    uint32_t seg;
    int shift;
    __device__ __forceinline__ uint64_t state() const { return top | part << shift; }
    __device__ __forceinline__ int ones(const EnumPlan &p) const
    {
        return p.n_up - p.odd - __popc(p.seg_prefix[seg]);
    }
    __device__ void set_segment(const EnumPlan &p)
    {
        top = (uint64_t)p.seg_prefix[seg] << p.low_bits | (uint64_t)p.odd;
    }
    __device__ void begin(const EnumPlan &p, uint64_t rank)
    {
        if (!p.seg_prefix) {
            part = kU1 ? unrank_colex(rank, p.n_sites, p.n_up, p.binom) : rank;
            left = ~0ULL;
            top = 0;
            seg = 0;
            shift = 0;
            return;
        }
        uint32_t lo = 0, hi = p.n_seg - 1;  // last segment that starts at or below rank
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo + 1) / 2;
            if (__ldg(p.seg_start + mid) <= rank)
                lo = mid;
            else
                hi = mid - 1;
        }
        seg = lo;
        shift = p.odd;
        set_segment(p);
        rank -= p.seg_start[seg];
        left = p.seg_start[seg + 1] - p.seg_start[seg] - rank;
        part = kU1 ? unrank_colex(rank, p.low_bits - p.odd, ones(p), p.binom) : rank;
    }
    __device__ __forceinline__ void next(const EnumPlan &p)
    {
        if (--left == 0) {
            ++seg;
            set_segment(p);
            left = p.seg_start[seg + 1] - p.seg_start[seg];
            part = kU1 ? (1ULL << ones(p)) - 1 : 0;
        } else {
            part = kU1 ? next_combination(part) : part + 1;
        }
    }
};

template <typename W, bool kU1, bool kWrite, bool kFact>
__global__ void __launch_bounds__(kEnumThreads) k_enumerate(EnumPlan plan, GroupView g,
                                                            uint32_t *counts,
                                                            const uint64_t *offsets,
                                                            uint64_t *states, uint16_t *norms)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nm = kFact ? g.n_cos : g.n_perm;
    W *sm_masks = reinterpret_cast<W *>(smem);
    uint32_t *sm_one = reinterpret_cast<uint32_t *>(smem + (size_t)nm * kMaskStride * sizeof(W));
    uint8_t *sm_kind = reinterpret_cast<uint8_t *>(sm_one + (g.order + 31) / 32);
    const W *gm;
    if (kFact)
        gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(g.cos_masks32)
                            : reinterpret_cast<const W *>(g.cos_masks64);
    else
        gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(g.masks32)
                            : reinterpret_cast<const W *>(g.masks64);
    for (int e = threadIdx.x; e < nm * kMaskStride; e += blockDim.x)
        sm_masks[e] = gm[e];
    for (int e = threadIdx.x; e < (g.order + 31) / 32; e += blockDim.x)
        sm_one[e] = kFact ? g.fchi_one[e] : g.chi_one[e];
    if (kFact)
        for (int e = threadIdx.x; e < g.n_cos; e += blockDim.x)
            sm_kind[e] = g.cos_kind[e];
    __syncthreads();
    const W full = (W)g.full;
    auto norm_of = [&](W s, bool known) {
        if constexpr (kFact) {
            int nrm = kNormOpen;
            if (g.prune == 1)
                nrm = rep_norm_rot1<W>(s, sm_kind, sm_masks, sm_one, g, plan, full, known);
            else if (g.prune == 2)
                nrm = rep_norm_blocks<W>(s, sm_masks, sm_one, g, full);
            return nrm != kNormOpen ? nrm : rep_norm_fact<W>(s, sm_kind, sm_masks, sm_one, g, full);
        } else {
            return rep_norm<W>(s, sm_masks, sm_one, g.n_perm, g.flip, full);
        }
    };
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < plan.n_chunks;
         c += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r0 = c * plan.chunk;
        const uint64_t cnt = min(plan.chunk, plan.total - r0);
        StateWalk<kU1> walk;
        walk.begin(plan, r0);
        uint32_t kept = 0;
        uint64_t out = kWrite ? offsets[c] : 0;
        uint32_t *cflags = plan.flags ? plan.flags + c * plan.flag_words : nullptr;
        uint32_t word = 0;
        for (uint64_t q = 0; q < cnt; ++q) {
            const uint64_t s = walk.state();
            int nrm = 0;
            if (kWrite && cflags) {  // only the states the count pass kept
                if ((q & 31) == 0)
                    word = cflags[q >> 5];
                if ((word >> (q & 31)) & 1u)
                    nrm = norm_of((W)s, true);
            } else {
                nrm = norm_of((W)s, false);
            }
            if (!kWrite && nrm < 0 && plan.ghosts) {
                const uint32_t at = atomicAdd(plan.ghost_count, 1u);
                if (at < plan.ghost_cap)
                    plan.ghosts[at] = s;
            }
            if (nrm > 0) {
                if (kWrite) {
                    states[out] = s;
                    norms[out] = (uint16_t)nrm;
                    ++out;
                }
                ++kept;
            }
            if (!kWrite && cflags) {
                word |= (nrm > 0 ? 1u : 0u) << (q & 31);
                if ((q & 31) == 31 || q + 1 == cnt) {
                    cflags[q >> 5] = word;
                    word = 0;
                }
            }
            if (q + 1 < cnt)
                walk.next(plan);
        }
        if (!kWrite)
            counts[c] = kept;
        else if (offsets[c] + kept != offsets[c + 1])
            atomicOr(&g_basis_status, 1u);
    }
}

template <typename W, bool kU1, bool kWrite, bool kFact>
cudaError_t enum_launch(const EnumPlan &plan, const GroupView &g, uint32_t *counts,
                        const uint64_t *offsets, uint64_t *states, uint16_t *norms,
                        cudaStream_t stream)
{
    auto kern = k_enumerate<W, kU1, kWrite, kFact>;
    const size_t smem = enum_smem_bytes(g, sizeof(W), kFact);
    int sms = 0, per_sm = 0;
    const cudaError_t e = kernel_occupancy((const void *)kern, kEnumThreads, smem, &sms, &per_sm);
    if (e != cudaSuccess)
        return e;
    const uint64_t want = (plan.n_chunks + kEnumThreads - 1) / kEnumThreads;
    const int grid = (int)std::min<uint64_t>(want, (uint64_t)sms * std::max(per_sm, 1));
    kern<<<std::max(grid, 1), kEnumThreads, smem, stream>>>(plan, g, counts, offsets, states, norms); count_launch();
    return cudaGetLastError();
}

template <bool kWrite>
cudaError_t enum_dispatch(EnumPlan plan, const GroupView &g, uint32_t *counts,
                          const uint64_t *offsets, uint64_t *states, uint16_t *norms,
                          cudaStream_t stream)
{
    int m = plan.n_sites, at = 0;
    for (int p = 2; p <= m; ++p) {  // at most three prime factors up to 64 sites
        if (m % p == 0)
            plan.turn[at++] = plan.n_sites / p;
        while (m % p == 0)
            m /= p;
    }
    const bool u1 = plan.n_up >= 0;
#define ED_ENUM(W, U1)                                                                           \
    return g.fact ? enum_launch<W, U1, kWrite, true>(plan, g, counts, offsets, states, norms, stream) \
                  : enum_launch<W, U1, kWrite, false>(plan, g, counts, offsets, states, norms, stream)
    if (plan.n_sites <= 32) {
        if (u1)
            ED_ENUM(uint32_t, true);
        ED_ENUM(uint32_t, false);
    }
    if (u1)
        ED_ENUM(uint64_t, true);
    ED_ENUM(uint64_t, false);
#undef ED_ENUM
}

// ---------------------------------------------------------------------------
// exclusive scan, uint32 or uint64 -> uint64 (reduce per block, scan block sums in one
// block with a running carry, rescan each block)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024, kScanItems = 4, kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t *sm_warp, uint64_t &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o)
            inc += t;
    }
    if (lane == 31)
        sm_warp[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint64_t w = lane < (int)(blockDim.x >> 5) ? sm_warp[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o)
                w += t;
        }
        sm_warp[lane] = w;  // inclusive warp-total prefix
    }
    __syncthreads();
    total = sm_warp[(blockDim.x >> 5) - 1];
    const uint64_t before = wid ? sm_warp[wid - 1] : 0;
    __syncthreads();
    return before + inc - v;
}

template <typename In>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const In *in, uint64_t n, uint64_t *bsum)
{
    __shared__ uint64_t sm[32];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint64_t v = 0;
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n)
            v += in[base + k];
    uint64_t total;
    block_exclusive_scan(v, sm, total);
    if (threadIdx.x == 0)
        bsum[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_bsums(uint64_t *bsum, uint64_t nb, uint64_t *grand)
{
    __shared__ uint64_t sm[32];
    uint64_t carry = 0;
    for (uint64_t b0 = 0; b0 < nb; b0 += kScanThreads) {
        const uint64_t i = b0 + threadIdx.x;
        const uint64_t v = i < nb ? bsum[i] : 0;
        uint64_t total;
        const uint64_t ex = block_exclusive_scan(v, sm, total);
        if (i < nb)
            bsum[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0)
        *grand = carry;
}

template <typename In>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(const In *in, uint64_t n, const uint64_t *bsum,
                                                            uint64_t *out)
{
    __shared__ uint64_t sm[32];
    const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    In items[kScanItems];
    uint64_t v = 0;
    for (int k = 0; k < kScanItems; ++k) {
        items[k] = base + k < n ? in[base + k] : 0;
        v += items[k];
    }
    uint64_t total;
    uint64_t run = bsum[blockIdx.x] + block_exclusive_scan(v, sm, total);
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n)
            out[base + k] = run;
        run += items[k];
    }
}

// ---------------------------------------------------------------------------
// Top bits that can begin a representative (see launch_prefix_filter).  At 22 of
// 36 ring sites 1 value in 40 is left, and with the lowest bit fixed the
// enumeration visits 3 states per representative instead of 144.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_prefix_viable(int n, int n_up, int odd, int bits, const uint8_t *inv,
                                                       int n_perm, int flip, uint32_t *viable)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >> bits)
        return;
    const int low = n - bits;
    bool ok = true;
    if (n_up >= 0) {
        const int rest = n_up - odd - __popc(v);
        ok = rest >= 0 && rest <= low - odd;
    }
    for (int g = 0; g < n_perm && ok; ++g) {
        const uint8_t *src = inv + g * n;
        for (int f = 0; f <= flip && ok; ++f) {
            for (int j = n - 1; j >= low; --j) {
                const int i = src[j];
                if (i < low)
                    break;  // not known
                const int a = (int)((v >> (i - low)) & 1u) ^ f, b = (int)((v >> (j - low)) & 1u);
                if (a != b) {
                    ok = a > b;
                    break;
                }
            }
        }
    }
    viable[v] = ok ? 1u : 0u;
}

__global__ void __launch_bounds__(256) k_prefix_collect(int n, int n_up, int odd, int bits, const uint32_t *viable,
                                                        const uint64_t *at, const uint64_t *binom, uint32_t *prefix,
                                                        uint64_t *count, uint32_t *n_seg)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >> bits)
        return;
    if (v == 0)
        *n_seg = (uint32_t)at[1u << bits];
    if (!viable[v])
        return;
    const int low = n - bits - odd;
    prefix[at[v]] = v;
    count[at[v]] = n_up < 0 ? 1ULL << low : binom[low * 65 + (n_up - odd - __popc(v))];
}

// ---------------------------------------------------------------------------
// prefix table, sortedness check, state -> index
// ---------------------------------------------------------------------------
__global__ void k_prefix_table(IndexView ix, uint32_t *tab)
{
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t > ix.tab_size)
        return;
    uint64_t lo = 0, hi = ix.dim;  // first i with key(states[i]) >= t
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (prefix_key(ix.states[mid], ix.e_lo, ix.mbits) < t)
            lo = mid + 1;
        else
            hi = mid;
    }
    tab[t] = (uint32_t)lo;
}

__global__ void k_hash_count(const uint64_t *states, uint64_t dim, int hbits, uint32_t *counts)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < dim;
         i += (uint64_t)gridDim.x * blockDim.x)
        atomicAdd(counts + hash_bucket(states[i], hbits), 1u);
}

__global__ void k_offsets_to_u32(const uint64_t *offsets, uint64_t n, uint32_t *out)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = (uint32_t)offsets[i];
}

// The order of entries inside a bucket depends on atomic timing; lookups
// compare states, so the result of a lookup does not.
__global__ void k_hash_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int hbits,
                            uint32_t *cursor, void *entries, int wide, int norm_bits)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < dim;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = states[i];
        const uint32_t pos = atomicAdd(cursor + hash_bucket(s, hbits), 1u);
        if (wide)
            reinterpret_cast<ulonglong2 *>(entries)[pos] =
                make_ulonglong2(s, (uint64_t)i | ((uint64_t)norms[i] << 32));
        else
            reinterpret_cast<uint2 *>(entries)[pos] =
                make_uint2((uint32_t)s, ((uint32_t)i << norm_bits) | norms[i]);
    }
}

// Slot order inside a bucket depends on atomic timing; a lookup compares the
// tag, so its result does not.
__global__ void k_bucket_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int n, int bbits,
                              int brem, uint32_t *cnt, uint64_t *bkt, ulonglong2 *stash, uint32_t *n_stash,
                              uint32_t stash_cap)
{
    const uint32_t bmask = (uint32_t)((1ULL << bbits) - 1);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < dim;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = states[i];
        const uint64_t m = bucket_mix(s, n);
        const uint32_t rem = (uint32_t)m & ((1u << brem) - 1u);
        uint32_t b = (uint32_t)(m >> brem);
        const uint64_t hi = ((uint64_t)norms[i] << (brem + 1)) | ((uint64_t)rem << 1);
        const uint64_t e = i | (hi << 32);
        uint32_t slot = atomicAdd(cnt + b, 1u);
        if (slot < kBucketSlots) {
            bkt[((uint64_t)b << 2) + slot] = e;
            continue;
        }
        b ^= bucket_alt(rem, bmask);
        slot = atomicAdd(cnt + b, 1u);
        if (slot < kBucketSlots) {
            bkt[((uint64_t)b << 2) + slot] = e | (1ULL << 32);
            continue;
        }
        const uint32_t k = atomicAdd(n_stash, 1u);
        if (k < stash_cap)
            stash[k] = make_ulonglong2(s, i | ((uint64_t)norms[i] << 32));
    }
}

__global__ void k_max_bucket(const uint32_t *tab, uint64_t tab_size, uint32_t *out)
{
    uint32_t m = 0;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tab_size;
         t += (uint64_t)gridDim.x * blockDim.x)
        m = max(m, tab[t + 1] - tab[t]);
    for (int o = 16; o > 0; o >>= 1)
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, m);
}

__global__ void k_pack_keys(const uint64_t *states, const uint16_t *norms, uint64_t dim, uint64_t *keys)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < dim;
         i += (uint64_t)gridDim.x * blockDim.x)
        keys[i] = (states[i] << 16) | norms[i];
}

__global__ void k_check_sorted(const uint64_t *states, uint64_t dim, int *flag)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; i < dim;
         i += (uint64_t)gridDim.x * blockDim.x)
        if (states[i - 1] >= states[i])
            atomicOr(flag, 1);
}

__global__ void k_index(IndexView ix, const uint64_t *q, int64_t *out, uint64_t n)
{
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        out[i] = find_index(q[i], ix);
}

}  // namespace

cudaError_t basis_status_take(unsigned int *status)
{
    unsigned int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(status, g_basis_status, sizeof(unsigned int));
    if (e == cudaSuccess && *status)
        e = cudaMemcpyToSymbol(g_basis_status, &zero, sizeof(unsigned int));
    return e;
}

cudaError_t launch_enum_count(const EnumPlan &plan, const GroupView &g, uint32_t *counts,
                              cudaStream_t stream)
{
    return enum_dispatch<false>(plan, g, counts, nullptr, nullptr, nullptr, stream);
}

cudaError_t launch_enum_write(const EnumPlan &plan, const GroupView &g, const uint64_t *offsets,
                              uint64_t *states, uint16_t *norms, cudaStream_t stream)
{
    return enum_dispatch<true>(plan, g, nullptr, offsets, states, norms, stream);
}

size_t scan_tmp_words(uint64_t n)
{
    return (n + kScanTile - 1) / kScanTile + 1;
}

cudaError_t launch_scan(const uint32_t *counts, uint64_t n, uint64_t *offsets, uint64_t *tmp,
                        cudaStream_t stream)
{
    const uint64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 0)
        return cudaMemsetAsync(offsets, 0, sizeof(uint64_t), stream);
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, stream>>>(counts, n, tmp); count_launch();
    k_scan_bsums<<<1, kScanThreads, 0, stream>>>(tmp, nb, offsets + n); count_launch();
    k_scan_down<<<(unsigned)nb, kScanThreads, 0, stream>>>(counts, n, tmp, offsets); count_launch();
    return cudaGetLastError();
}

size_t prefix_filter_bytes(int bits)
{
    const size_t n = (size_t)1 << bits;  // flags, their scan, counts, the scan's work area
    return n * 4 + (n + 1) * 8 + n * 8 + scan_tmp_words(n) * 8 + 1024;
}

cudaError_t launch_prefix_filter(int n_sites, int n_up, int odd, int bits, const uint8_t *inv, int n_perm, int flip,
                                 const uint64_t *binom, void *tmp, uint32_t *prefix, uint64_t *start,
                                 uint32_t *n_seg, cudaStream_t stream)
{
    const uint64_t n = 1ULL << bits, nb = (n + kScanTile - 1) / kScanTile;
    uint64_t *at = (uint64_t *)tmp, *count = at + ((n + 2) & ~1ULL), *work = count + n;
    uint32_t *viable = (uint32_t *)(work + ((scan_tmp_words(n) + 1) & ~1ULL));
    const unsigned grid = (unsigned)((n + 255) / 256);
    k_prefix_viable<<<grid, 256, 0, stream>>>(n_sites, n_up, odd, bits, inv, n_perm, flip, viable); count_launch();
    cudaError_t e = launch_scan(viable, n, at, work, stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(count, 0, n * sizeof(uint64_t), stream);
    if (e != cudaSuccess)
        return e;
    k_prefix_collect<<<grid, 256, 0, stream>>>(n_sites, n_up, odd, bits, viable, at, binom, prefix, count, n_seg);
    count_launch();
    // entries past the last segment count nothing: start[n_seg ..] is the total
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, stream>>>(count, n, work); count_launch();
    k_scan_bsums<<<1, kScanThreads, 0, stream>>>(work, nb, start + n); count_launch();
    k_scan_down<<<(unsigned)nb, kScanThreads, 0, stream>>>(count, n, work, start); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_prefix_table(const IndexView &ix, uint32_t *tab, cudaStream_t stream)
{
    const uint64_t n = ix.tab_size + 1;
    k_prefix_table<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(ix, tab); count_launch();
    return cudaGetLastError();
}

static unsigned grid_for(uint64_t n)
{
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + 255) / 256, 65536));
}

cudaError_t launch_hash_count(const uint64_t *states, uint64_t dim, int hbits, uint32_t *counts,
                              cudaStream_t stream)
{
    if (!dim)
        return cudaSuccess;
    k_hash_count<<<grid_for(dim), 256, 0, stream>>>(states, dim, hbits, counts); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_offsets_to_u32(const uint64_t *offsets, uint64_t n, uint32_t *out, cudaStream_t stream)
{
    k_offsets_to_u32<<<grid_for(n), 256, 0, stream>>>(offsets, n, out); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_hash_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int hbits,
                             uint32_t *cursor, void *entries, int wide, int norm_bits,
                             cudaStream_t stream)
{
    if (!dim)
        return cudaSuccess;
    k_hash_fill<<<grid_for(dim), 256, 0, stream>>>(states, norms, dim, hbits, cursor, entries, wide,
                                                    norm_bits); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_bucket_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int n_sites,
                               int bbits, int brem, uint32_t *cnt, uint64_t *bkt, ulonglong2 *stash,
                               uint32_t *n_stash, uint32_t stash_cap, cudaStream_t stream)
{
    if (!dim)
        return cudaSuccess;
    k_bucket_fill<<<grid_for(dim), 256, 0, stream>>>(states, norms, dim, n_sites, bbits, brem, cnt, bkt, stash,
                                                      n_stash, stash_cap); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_max_bucket(const uint32_t *tab, uint64_t tab_size, uint32_t *out, cudaStream_t stream)
{
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((tab_size + 255) / 256, 4096));
    k_max_bucket<<<(unsigned)blocks, 256, 0, stream>>>(tab, tab_size, out); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_pack_keys(const uint64_t *states, const uint16_t *norms, uint64_t dim, uint64_t *keys,
                             cudaStream_t stream)
{
    if (dim == 0)
        return cudaSuccess;
    const uint64_t blocks = std::min<uint64_t>((dim + 255) / 256, 65536);
    k_pack_keys<<<(unsigned)blocks, 256, 0, stream>>>(states, norms, dim, keys); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_check_sorted(const uint64_t *states, uint64_t dim, int *flag, cudaStream_t stream)
{
    if (dim < 2)
        return cudaSuccess;
    const uint64_t blocks = std::min<uint64_t>((dim + 255) / 256, 65536);
    k_check_sorted<<<(unsigned)blocks, 256, 0, stream>>>(states, dim, flag); count_launch();
    return cudaGetLastError();
}

cudaError_t launch_index(const IndexView &ix, const uint64_t *query, int64_t *out, uint64_t n,
                         cudaStream_t stream)
{
    k_index<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(ix, query, out, n); count_launch();
    return cudaGetLastError();
}

}  // namespace edk

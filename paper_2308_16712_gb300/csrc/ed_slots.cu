// ed_slots.cu -- building the slot index of a basis (ed_slots.cuh) and filling
// the slotted copy of a vector.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "ed_kernels.cuh"

namespace edk {
namespace {

constexpr int kSlotThreads = 512;
constexpr uint32_t kSlotBuckets = 1u << kSlotLogB;
constexpr uint32_t kMaxBucketKeys = 32;
constexpr uint32_t kMaxPilot = 1u << 20;  // exceptions: pilots tried before the build gives up

// keys of every cell: the basis states by binary search for the cell's ends,
// the weightless representatives one by one (count zeroed)
__global__ void __launch_bounds__(256) k_cell_count(SlotView v, const uint64_t *states, uint64_t dim, uint32_t *count)
{
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < v.n_cells) {
        uint64_t at[2];
        for (int q = 0; q < 2; ++q) {
            uint64_t lo = 0, hi = dim;  // first state of cell t + q or above
            while (lo < hi) {
                const uint64_t mid = (lo + hi) >> 1;
                if (slot_cell(states[mid], v) < t + q)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            at[q] = lo;
        }
        atomicAdd(count + t, (uint32_t)(at[1] - at[0]));
    }
    for (uint64_t i = t; i < v.n_ghost; i += (uint64_t)gridDim.x * blockDim.x)
        atomicAdd(count + slot_cell(v.ghosts[i], v), 1u);
}

// Every key (basis states, then the weightless representatives) appended to its
// partition's list; cursors beyond kSlotCap raise the error flag.
__global__ void __launch_bounds__(256) k_slot_scatter(SlotView v, const uint64_t *states, uint64_t dim,
                                                      uint32_t *cursor, uint2 *list, int *err)
{
    const uint64_t n = dim + v.n_ghost;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = i < dim ? states[i] : v.ghosts[i - dim];
        const SlotKey k = slot_key(s);
        const uint32_t p = slot_bucket(s, k, v) >> kSlotLogB;
        const uint32_t at = atomicAdd(cursor + p, 1u);
        if (at < kSlotCap)
            list[(uint64_t)p * kSlotCap + at] = make_uint2(k.hi, k.lo);
        else
            *err = 1;
    }
}

struct SlotBuild {
    uint2 keys[kSlotCap];                    // the partition's keys, grouped by bucket
    uint32_t start[kSlotBuckets + 1];        // first key of each bucket
    uint32_t fill[kSlotBuckets];
    uint16_t order[kSlotBuckets];            // buckets, fullest first
    uint32_t used[(kSlotCap + 31) / 32];
    uint32_t of_size[kMaxBucketKeys + 2];
    uint32_t scan[kSlotThreads / 32];
    int bad;
};

// One block per partition.  Buckets are placed fullest first; the buckets of
// one size are tried by all threads at once: a thread looks for a pilot whose
// slots are free, claims them bit by bit, and gives them back and goes on when
// another thread was faster.  Which of several valid pilots a bucket gets
// depends on timing; the slots of the keys are distinct in any case, and
// results do not depend on which slot a value lies in.
// Bound by shared-memory latency (a dozen probes per bucket); two blocks per SM.
// Ring N=36 (6.3e7 states): 9.9 ms.
__global__ void __launch_bounds__(kSlotThreads) k_slot_pilots(const uint2 *list, const uint32_t *cursor,
                                                              const uint32_t *part_cell, const uint2 *cells,
                                                              uint8_t *pilots, uint2 *exc,
                                                              uint32_t exc_mask, int *err)
{
    extern __shared__ __align__(16) unsigned char smem[];
    SlotBuild &b = *reinterpret_cast<SlotBuild *>(smem);
    const uint32_t part = blockIdx.x;
    const uint32_t count = min(cursor[part], kSlotCap);
    const uint2 *keys = list + (uint64_t)part * kSlotCap;
    const uint32_t tid = threadIdx.x;
    const uint32_t n_buckets = cells[part_cell[part]].y;  // whole partitions: the cell's first bucket drops out
    for (uint32_t e = tid; e < kSlotBuckets; e += kSlotThreads)
        b.fill[e] = 0;
    for (uint32_t e = tid; e < (kSlotCap + 31) / 32; e += kSlotThreads)
        b.used[e] = 0;
    for (uint32_t e = tid; e < kMaxBucketKeys + 2; e += kSlotThreads)
        b.of_size[e] = 0;
    if (tid == 0)
        b.bad = 0;
    __syncthreads();
    for (uint32_t i = tid; i < count; i += kSlotThreads)
        atomicAdd(b.fill + (mul_high(keys[i].x, n_buckets) & (kSlotBuckets - 1)), 1u);
    __syncthreads();
    {  // exclusive scan of the bucket sizes, four consecutive buckets per thread
        constexpr uint32_t kPer = kSlotBuckets / kSlotThreads;
        uint32_t sz[kPer], sum = 0;
        for (uint32_t e = 0; e < kPer; ++e) {
            sz[e] = b.fill[tid * kPer + e];
            sum += sz[e];
            if (sz[e] > kMaxBucketKeys)
                b.bad = 1;
            else
                atomicAdd(b.of_size + sz[e], 1u);
        }
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)(tid & 31) >= o)
                incl += v;
        }
        if ((tid & 31) == 31)
            b.scan[tid >> 5] = incl;
        __syncthreads();
        uint32_t before = incl - sum;
        for (uint32_t w = 0; w < (tid >> 5); ++w)
            before += b.scan[w];
        for (uint32_t e = 0; e < kPer; ++e) {
            b.start[tid * kPer + e] = before;
            before += sz[e];
        }
        if (tid == kSlotThreads - 1)
            b.start[kSlotBuckets] = before;
    }
    __syncthreads();
    if (b.bad) {
        if (tid == 0)
            *err = 1;
        return;
    }
    if (tid == 0) {  // of_size[k] becomes the first place of the buckets of k keys, fullest first
        uint32_t at = 0;
        for (int k = kMaxBucketKeys; k >= 0; --k) {
            const uint32_t c = b.of_size[k];
            b.of_size[k] = at;
            at += c;
        }
    }
    for (uint32_t e = tid; e < kSlotBuckets; e += kSlotThreads)
        b.fill[e] = b.start[e];
    __syncthreads();
    for (uint32_t i = tid; i < count; i += kSlotThreads) {
        const uint2 k = keys[i];
        b.keys[atomicAdd(b.fill + (mul_high(k.x, n_buckets) & (kSlotBuckets - 1)), 1u)] = k;
    }
    for (uint32_t e = tid; e < kSlotBuckets; e += kSlotThreads) {
        const uint32_t k = b.start[e + 1] - b.start[e];
        b.order[atomicAdd(b.of_size + k, 1u)] = (uint16_t)e;  // of_size[k] ends as the end of size k
    }
    __syncthreads();
    for (int k = kMaxBucketKeys; k >= 0; --k) {
        const uint32_t first = k == (int)kMaxBucketKeys ? 0u : b.of_size[k + 1], end = b.of_size[k];
        if (first == end)
            continue;
        for (uint32_t q = first + tid; q < end; q += kSlotThreads) {
            const uint32_t e = b.order[q], s0 = b.start[e];
            uint32_t pilot = 0;
            bool done = k == 0;
            while (!done && pilot < kMaxPilot) {
                if (pilot == kPilotEscape)
                    ++pilot;
                bool ok = true;
                for (int i = 0; i < k && ok; ++i) {
                    const uint2 x = b.keys[s0 + i];
                    const uint32_t sl = slot_place(SlotKey{x.x, x.y}, pilot);
                    ok = !((*(volatile uint32_t *)(b.used + (sl >> 5)) >> (sl & 31)) & 1u);
                }
                int got = 0;
                for (; ok && got < k; ++got) {
                    const uint2 x = b.keys[s0 + got];
                    const uint32_t sl = slot_place(SlotKey{x.x, x.y}, pilot), bit = 1u << (sl & 31);
                    if (atomicOr(b.used + (sl >> 5), bit) & bit) {
                        ok = false;  // another key (of this bucket, too) has it
                        break;
                    }
                }
                if (ok) {
                    done = true;
                } else {
                    for (int i = 0; i < got; ++i) {
                        const uint2 x = b.keys[s0 + i];
                        const uint32_t sl = slot_place(SlotKey{x.x, x.y}, pilot);
                        atomicAnd(b.used + (sl >> 5), ~(1u << (sl & 31)));
                    }
                    ++pilot;
                }
            }
            const uint32_t gb = part * kSlotBuckets + e;
            pilots[gb] = (uint8_t)(pilot < kPilotEscape ? pilot : kPilotEscape);
            if (!done) {
                *err = 1;
            } else if (pilot > kPilotEscape) {
                uint32_t at = exc_start(gb, exc_mask), i = 0;
                for (; i <= exc_mask / 2; ++i) {  // at most half full: lookups end at an empty entry
                    if (atomicCAS(&exc[at].x, ~0u, gb) == ~0u) {
                        exc[at].y = pilot;
                        break;
                    }
                    at = (at + 1) & exc_mask;
                }
                if (i > exc_mask / 2)
                    *err = 1;
            }
        }
        __syncthreads();
    }
}

// xs[slot(state_i)] = sqrt(n_i) x_i for one sector or several: one thread per EL
// scalars of a row, 2^log_lanes threads per row (those beyond the row's scalars
// idle).  One random write per row against some twenty random reads per row of
// the product that follows; the state and norm streams are coalesced.  Also
// zeroes the tile queue of that product.
template <int kSec>
struct FillArgs {
    int n_sectors, scalars, stride, log_lanes;
    unsigned long long *queue;
    SlotFill sec[kSec];
    uint32_t first_block[kSec + 1];  // blocks of each sector
};

template <typename T, int EL, int kSec>
__global__ void __launch_bounds__(256) k_slot_fill(const __grid_constant__ FillArgs<kSec> a)
{
    if (a.queue && blockIdx.x == 0 && threadIdx.x == 0)
        *a.queue = 0;
    int sec = 0;
    if (kSec > 1) {  // last sector whose blocks begin at or below this one
        int lo = 0, hi = a.n_sectors - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.first_block[mid] <= blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        sec = lo;
    }
    const SlotFill &f = a.sec[sec];
    const uint32_t block = blockIdx.x - a.first_block[sec], blocks = a.first_block[sec + 1] - a.first_block[sec];
    const int scalars = a.scalars;
    const int part = ((int)threadIdx.x & ((1 << a.log_lanes) - 1)) * EL;
    const uint64_t step = ((uint64_t)blocks * blockDim.x) >> a.log_lanes;
    const bool whole = scalars % EL == 0;
    const T *x = reinterpret_cast<const T *>(f.x);
    T *xs = reinterpret_cast<T *>(f.xs);
    for (uint64_t i = ((uint64_t)block * blockDim.x + threadIdx.x) >> a.log_lanes; i < f.dim + f.v.n_ghost; i += step) {
        const bool ghost = i >= f.dim;
        const uint64_t s = ghost ? f.v.ghosts[i - f.dim] : __ldcs(f.states + i);
        T w = T(0);
        if (!ghost) {
            const uint32_t n = __ldcs(f.norms + i);
            w = n == 1 ? T(1) : sqrt((T)n);
        }
        const uint64_t at = (uint64_t)slot_of(s, f.v) * a.stride + part;
        if (part >= scalars)
            continue;
        struct __align__(sizeof(T) * EL) Vec { T e[EL]; } r;
        if (ghost) {
#pragma unroll
            for (int e = 0; e < EL; ++e)
                r.e[e] = T(0);
        } else if (whole) {
            r = *reinterpret_cast<const Vec *>(x + i * scalars + part);
#pragma unroll
            for (int e = 0; e < EL; ++e)
                r.e[e] *= w;
        } else {
#pragma unroll
            for (int e = 0; e < EL; ++e)
                r.e[e] = part + e < scalars ? w * x[i * scalars + part + e] : T(0);
        }
        *reinterpret_cast<Vec *>(xs + at) = r;
    }
}

template <typename T, int EL, int kSec>
cudaError_t fill_launch(const SlotFill *sec, int n, const SlotRow &r, unsigned long long *queue, cudaStream_t s)
{
    static thread_local FillArgs<kSec> a;  // host staging; copied at launch
    a.n_sectors = n;
    a.scalars = r.scalars;
    a.stride = r.stride;
    a.log_lanes = 0;
    while ((1 << a.log_lanes) * EL < r.scalars)
        ++a.log_lanes;
    a.queue = queue;
    uint32_t blocks = 0;
    for (int k = 0; k < n; ++k) {
        a.sec[k] = sec[k];
        a.first_block[k] = blocks;
        const uint64_t threads = (sec[k].dim + sec[k].v.n_ghost) << a.log_lanes;
        blocks += (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((threads + 255) / 256, 152 * 64));
    }
    a.first_block[n] = blocks;
    k_slot_fill<T, EL, kSec><<<blocks, 256, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int kSec>
cudaError_t fill_dispatch(const SlotFill *sec, int n, const SlotRow &r, ed_dtype dtype, unsigned long long *queue,
                          cudaStream_t s)
{
    if (dtype == ED_F64 || dtype == ED_C128)
        return r.el == 1 ? fill_launch<double, 1, kSec>(sec, n, r, queue, s)
                         : fill_launch<double, 2, kSec>(sec, n, r, queue, s);
    return r.el == 1   ? fill_launch<float, 1, kSec>(sec, n, r, queue, s)
           : r.el == 2 ? fill_launch<float, 2, kSec>(sec, n, r, queue, s)
                       : fill_launch<float, 4, kSec>(sec, n, r, queue, s);
}

}  // namespace

// Scalars per row, scalars per 1 / 2 / 4-wide access and padded row stride of the
// slotted copy: rows of up to 64 bytes on a power of two, longer ones on a
// multiple of 32 bytes, so that a row never straddles a sector needlessly.
SlotRow slot_row(int nvec, ed_dtype dtype)
{
    const bool cplx = dtype == ED_C128 || dtype == ED_C64, dbl = dtype == ED_F64 || dtype == ED_C128;
    const int size = dbl ? 8 : 4;
    SlotRow r;
    r.scalars = nvec * (cplx ? 2 : 1);
    r.el = std::min(dbl ? 2 : 4, r.scalars > 2 ? 4 : r.scalars);
    int bytes = r.scalars * size;
    if (bytes <= 64) {
        int p = size * r.el;
        while (p < bytes)
            p *= 2;
        bytes = p;
    } else {
        bytes = (bytes + 31) / 32 * 32;
    }
    r.stride = bytes / size;
    return r;
}

size_t slot_copy_bytes(const SlotView &v, int nvec, ed_dtype dtype)
{
    return (v.n_slots * slot_row(nvec, dtype).stride * (dtype == ED_F64 || dtype == ED_C128 ? 8 : 4) + 255) / 256 * 256;
}

cudaError_t launch_slot_fill(const SlotFill *sec, int n, int nvec, ed_dtype dtype, unsigned long long *queue,
                             cudaStream_t s)
{
    const SlotRow r = slot_row(nvec, dtype);
    return n == 1 ? fill_dispatch<1>(sec, n, r, dtype, queue, s) : fill_dispatch<kSlotMaxBatch>(sec, n, r, dtype, queue, s);
}

// Builds the slot index over the basis states and the weightless
// representatives (ghosts: ownership passes to the basis on success).  False,
// with nothing kept, when memory is short or the slots exceed 32 bits; *err
// (device, zero) becomes 1 when no pilots were found: the caller then takes the
// index back.  The products then use the other index kinds.  cells: the caller's,
// to be kept until the stream has been waited for, whatever the outcome: its
// copy to the device is asynchronous, and from pageable memory CUDA does not
// promise that the call has read the source when it returns.
bool build_slot_index(ed_basis *b, uint64_t *ghosts, uint32_t n_ghost, int *err, std::vector<uint2> &cells,
                      cudaStream_t stream)
{
    if (!b->dim)
        return false;
    cudaError_t e = cudaSuccess;
    SlotView v{};
    v.ghosts = ghosts;
    v.n_ghost = n_ghost;
    int lg = 0;  // log2 of the cells: some 65536 states each, at most 8192 (64 KB of table)
    while (lg < 13 && (b->dim >> 17) >> lg)
        ++lg;
    v.shift = 63;
    v.n_cells = 1;
    std::vector<uint32_t> count(1, (uint32_t)(b->dim + n_ghost)), part_cell;
    if (lg) {
        uint64_t top = 0;  // the last state; weightless ones beyond it share the last cell
        e = cudaMemcpyAsync(&top, b->d_states + b->dim - 1, sizeof(top), cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(stream);
        const int bits = top ? 64 - __builtin_clzll(top) : 1;
        v.shift = std::min(63, std::max(0, bits - lg));
        v.n_cells = (uint32_t)(top >> v.shift) + 1;
        count.resize(v.n_cells);
        uint32_t *d_count = nullptr;
        if (e == cudaSuccess)
            e = ws_alloc_optional((void **)&d_count, v.n_cells * sizeof(uint32_t), stream);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(d_count, 0, v.n_cells * sizeof(uint32_t), stream);
        if (e == cudaSuccess) {
            const uint64_t n = std::max<uint64_t>(v.n_cells, std::min<uint64_t>(n_ghost, 1 << 18));
            k_cell_count<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(v, b->d_states, b->dim, d_count);
            count_launch();
            e = cudaMemcpyAsync(count.data(), d_count, v.n_cells * sizeof(uint32_t), cudaMemcpyDeviceToHost, stream);
        }
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(stream);
        ws_free(d_count, stream);
    }
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    cells.resize(v.n_cells);
    uint64_t parts = 0;
    const uint32_t part_keys = b->dim + n_ghost <= kSlotSmallMax ? kSlotSmallKeys : kSlotPartKeys;
    for (uint32_t c = 0; c < v.n_cells; ++c) {
        const uint64_t p = ((uint64_t)count[c] + part_keys - 1) / part_keys;
        // a cell without keys is never asked for; its entry stays in bounds
        cells[c] = p ? make_uint2((uint32_t)(parts << kSlotLogB), (uint32_t)(p << kSlotLogB)) : make_uint2(0, 1);
        part_cell.insert(part_cell.end(), p, c);
        parts += p;
    }
    const uint64_t n_slots = parts * kSlotCap, keys = b->dim + n_ghost;
    if (n_slots >= (1ULL << 32) || (parts << kSlotLogB) >= (1ULL << 32))
        return false;
    uint32_t exc_n = 64;
    while (exc_n < 8 * parts)  // some 0.3 exceptions per partition
        exc_n *= 2;
    uint8_t *pilots = nullptr;
    uint2 *exc = nullptr, *list = nullptr, *d_cells = nullptr;
    uint32_t *cursor = nullptr;
    e = ws_alloc_optional((void **)&pilots, parts << kSlotLogB, stream);
    if (e == cudaSuccess)
        e = ws_alloc_optional((void **)&exc, exc_n * sizeof(uint2), stream);
    // cells, and behind them the cell of each partition (build only)
    cells.resize(v.n_cells + (parts + 1) / 2);
    std::memcpy(cells.data() + v.n_cells, part_cell.data(), parts * sizeof(uint32_t));
    if (e == cudaSuccess)
        e = ws_alloc_optional((void **)&d_cells, cells.size() * sizeof(uint2), stream);
    if (e == cudaSuccess)
        e = ws_alloc_optional((void **)&list, n_slots * sizeof(uint2), stream);
    if (e == cudaSuccess)
        e = ws_alloc_optional((void **)&cursor, parts * sizeof(uint32_t), stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_cells, cells.data(), cells.size() * sizeof(uint2), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(cursor, 0, parts * sizeof(uint32_t), stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(exc, 0xFF, exc_n * sizeof(uint2), stream);
    v.pilots = pilots;
    v.cells = d_cells;
    v.exc = exc;
    v.exc_mask = exc_n - 1;
    v.n_slots = n_slots;
    if (e == cudaSuccess) {
        const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((keys + 255) / 256, 152 * 32));
        k_slot_scatter<<<grid, 256, 0, stream>>>(v, b->d_states, b->dim, cursor, list, err);
        count_launch();
        int sms = 0, per_sm = 0;
        e = kernel_occupancy((const void *)k_slot_pilots, kSlotThreads, sizeof(SlotBuild), &sms, &per_sm);
    }
    if (e == cudaSuccess) {
        k_slot_pilots<<<(unsigned)parts, kSlotThreads, sizeof(SlotBuild), stream>>>(list, cursor, (const uint32_t *)(d_cells + v.n_cells), d_cells, pilots,
                                                                                   exc, exc_n - 1, err);
        count_launch();
        e = cudaGetLastError();
    }
    ws_free(list, stream);
    ws_free(cursor, stream);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        ws_free(pilots, stream);
        ws_free(exc, stream);
        ws_free(d_cells, stream);
        return false;
    }
    b->slots = v;
    return true;
}

void free_slot_index(ed_basis *b)
{
    ws_free(const_cast<uint8_t *>(b->slots.pilots), 0);
    ws_free(const_cast<uint2 *>(b->slots.exc), 0);
    ws_free(const_cast<uint2 *>(b->slots.cells), 0);
    ws_free(const_cast<uint64_t *>(b->slots.ghosts), 0);
    b->slots = SlotView{};
}

}  // namespace edk

// ed_matvec.cu -- kernel choice and dtype dispatch of the matvec.
#include "ed_matvec_slot.cuh"

namespace edk {

int g_kernel_policy = 0;

// The rule where the slot kernel does not run (launch_matvec_v), for one vector of
// an exchange-only operator: the term-parallel kernel in single precision, and in double precision for
// 64-bit words (ring N=36 / 40 fp64: 42.5 / 714 ms against 45.1 / 750 ms
// row-per-lane); row-per-lane otherwise.
bool use_term_parallel(int nvec, const OpView &op, ed_dtype dtype, int n_sites)
{
    if (nvec != 1 || !op.exchange_only || g_kernel_policy == 1)
        return false;
    return g_kernel_policy == 2 || dtype == ED_F32 || dtype == ED_C64 || n_sites > 32;
}

static TpArgs<1> single_tp_args(const OpView &op, const GroupView &g, const IndexView &ix, const void *x,
                                void *y)
{
    TpArgs<1> t;
    t.op = op;
    t.g = g;
    t.ctl = BatchCtl{nullptr, nullptr, nullptr};  // one sector: static tiles, no gate
    t.n_sectors = 1;
    t.max_order = g.order;
    t.total_tiles = (ix.dim + 31) / 32;
    SectorDesc &d = t.sec[0];
    d.keys = ix.keys;
    d.states = ix.states;
    d.norms = ix.norms;
    d.htab = ix.htab;
    d.hent = ix.hent;
    d.chi = g.fact ? g.fchi : g.chi;
    d.chif = g.fact ? g.fchif : g.chif;
    d.x = x;
    d.y = y;
    d.dim = ix.dim;
    d.tile_begin = 0;
    d.hbits = ix.hbits;
    d.hwide = ix.hwide;
    d.norm_bits = ix.norm_bits;
    d.bkt = ix.bkt;
    d.stash = ix.stash;
    d.n_stash = ix.n_stash;
    d.bbits = ix.bbits;
    d.brem = ix.brem;
    d.flip = g.flip;
    return t;
}

// The push form (ablation): y = 0, then every term scattered atomically.
cudaError_t launch_matvec_push(const OpView &op, const GroupView &g, const IndexView &ix, bool track,
                               const void *x, void *y, ed_dtype dtype, cudaStream_t stream)
{
    const size_t vb = (dtype == ED_F64 || dtype == ED_C64) ? 8 : dtype == ED_F32 ? 4 : 16;
    cudaError_t e = cudaMemsetAsync(y, 0, ix.dim * vb, stream);
    if (e != cudaSuccess)
        return e;
    const TpArgs<1> t = single_tp_args(op, g, ix, x, y);
    return tp_push(t, track, tp_index_kind(t.sec[0]), dtype, stream);
}

cudaError_t launch_matvec(const OpView &op, const GroupView &g, const IndexView &ix, bool track,
                          const void *x, void *y, int nvec, ed_dtype dtype, cudaStream_t stream)
{
    return launch_matvec_v(op, g, ix, track, x, y, nvec, dtype, MatvecVariant{}, stream);
}

// ---- the slot kernel -----------------------------------------------------------
namespace {

constexpr uint64_t kSlotBlockMinDim = 1024;
// Up to this many states a product of one vector goes without the slotted copy: one
// launch instead of two that wait for each other, and everything is in L2 (8-site
// ring, 7 states, fp32 13.2 -> 8.7 us, 10.3 by the term-parallel kernel; 20 sites,
// momentum 1, 9225 states, complex128 41.3 -> 38.2; 4x6 torus, 56664 states, fp64 73
// with the copy, 89 without).
constexpr uint64_t kSlotDirectDim = 16384;

int slot_search(const GroupView &g) { return g.fact ? g.prune : 0; }

}  // namespace

// Lanes of a row: as few as keep the terms of 32 / lanes rows within the list.
int slot_log_group(const OpView &op)
{
    int lg = 1;
    while (lg < 5 && (op.max_terms << (5 - lg)) > kSlTerms)
        ++lg;
    return lg;
}

// Tiles a warp takes from the queue at a time: one, unless there are so many that
// the end of the launch is still balanced with several (at 8 chunks per warp ring
// N=32 fp32 lost 4 %).
int slot_chunk(uint64_t tiles) { return (int)std::max<uint64_t>(1, std::min<uint64_t>(8, tiles / (152 * 40 * 128))); }

bool slot_applies(const OpView &op, const GroupView &g, const IndexView &ix, bool track, int nvec, ed_dtype dtype)
{
    if (!ix.slots.pilots || !(ix.htab || ix.bkt) || !op.exchange_only || op.max_terms > kSlTerms)
        return false;
    if (g_kernel_policy != 0 && g_kernel_policy != 3)
        return false;
    // blocks of vectors over the smallest sectors stay with the row-per-lane
    // kernel, whose columns are those of its single products bit for bit; it does
    // not serve blocks of 8 in fp32 (16 sites, 415 states: 21.2 us term-parallel, 9.7
    // here)
    if (nvec > 1 && ix.dim < kSlotBlockMinDim && !(nvec == 8 && dtype == ED_F32) && g_kernel_policy != 3)
        return false;
    // the coefficient table: in shared memory, its entries counted in 16 bits
    const int order = track ? g.order : 1;
    OpView all = op;
    all.even = 0;
    const size_t bytes = dtype == ED_F64 || dtype == ED_C128 ? slot_table_bytes<double>(all, order, false)
                                                             : slot_table_bytes<float>(all, order, false);
    return bytes <= (size_t)kSlMaxTable && (size_t)op.n_mats * 2 * g.order < 65536 &&
           (size_t)op.n_fam * sizeof(OpFamily) <= 16384;
}

SlotSector slot_sector(const OpView &op, const GroupView &g, const IndexView &ix, const void *x, const void *xs,
                       void *y, bool alone)
{
    SlotSector d;
    if (xs)
        d.v = ix.slots;
    else
        d.find = SlotFind{ix.htab, ix.hent, ix.bkt, ix.stash, ix.n_stash, ix.hbits, ix.hwide, ix.norm_bits,
                          ix.bbits, ix.brem};
    d.states = ix.states;
    d.norms = ix.norms;
    d.chi = g.fact ? g.fchi : g.chi;
    d.chif = g.fact ? g.fchif : g.chif;
    d.x = x;
    d.xs = xs;
    d.y = y;
    d.dim = ix.dim;
    d.tile_begin = 0;
    // rows of a tile: all the lanes have room for; fewer where a sector alone
    // would not give every resident warp (152 x 32) a tile
    d.log_rows = 5 - slot_log_group(op);
    while (alone && d.log_rows > 0 && (ix.dim >> d.log_rows) < 152 * 32)
        --d.log_rows;
    d.flip = g.flip;
    return d;
}

uint64_t slot_tiles(const SlotSector &d) { return (d.dim + (1ull << d.log_rows) - 1) >> d.log_rows; }

bool stream_captured(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return st != cudaStreamCaptureStatusNone;
}

// xs: the slotted copy with the tile queue behind it, or null (gather from x)
static cudaError_t launch_slot(const OpView &op, const GroupView &g, const IndexView &ix, bool track, const void *x,
                               void *y, void *xs, int nvec, ed_dtype dtype, cudaStream_t stream)
{
    unsigned long long *queue = nullptr;
    if (xs) {
        queue = (unsigned long long *)((char *)xs + slot_copy_bytes(ix.slots, nvec, dtype));
        const SlotFill fill{ix.slots, ix.states, ix.norms, ix.dim, x, xs};
        const cudaError_t e = launch_slot_fill(&fill, 1, nvec, dtype, queue, stream);
        if (e != cudaSuccess)
            return e;
    }
    const SlotRow row = slot_row(nvec, dtype);
    SlotArgs<1> a;
    a.op = op;
    a.g = g;
    a.n_sectors = 1;
    a.max_order = g.order;
    a.order = track ? g.order : 1;
    a.op.even = track && op.even;
    a.byte = slot_entries(a.op) * a.order <= 256;
    a.scalars = row.scalars;
    a.stride = row.stride;
    a.log_parts = 0;
    while ((row.el << a.log_parts) < row.scalars)
        ++a.log_parts;
    a.beyond_l2 = slot_copy_bytes(ix.slots, nvec, dtype) > kSlotL2Bytes;
    a.ctl = BatchCtl{queue, nullptr, nullptr};
    a.log_group = slot_log_group(op);
    a.sec[0] = slot_sector(op, g, ix, x, xs, y, true);
    a.total_tiles = slot_tiles(a.sec[0]);
    a.chunk = slot_chunk(a.total_tiles);
    const int search = slot_search(g);
    count_product(xs ? kProductSlots : kProductDirect);
    if (!xs) {
        switch (dtype) {
        case ED_F64: return slot1_direct_f64(a, track, row.el, stream);
        case ED_F32: return slot1_direct_f32(a, track, row.el, stream);
        case ED_C128: return slot1_direct_c128(a, track, row.el, stream);
        case ED_C64: return slot1_direct_c64(a, track, row.el, stream);
        }
        return cudaErrorInvalidValue;
    }
    switch (dtype) {
    case ED_F64: return slot1_f64(a, search, track, row.el, stream);
    case ED_F32: return slot1_f32(a, search, track, row.el, stream);
    case ED_C128: return slot1_c128(a, search, track, row.el, stream);
    case ED_C64: return slot1_c64(a, search, track, row.el, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_matvec_v(const OpView &op, GroupView g, const IndexView &ix, bool track, const void *x,
                            void *y, int nvec, ed_dtype dtype, MatvecVariant v, cudaStream_t stream)
{
    if (v.prune >= 0 && g.fact && g.rot_d == 1)
        g.prune = v.prune;  // ring translations: pruned or exhaustive (autotuner)
    // the slot kernel wherever the sector has a slot index (ring N=32 fp32 / N=36
    // fp64 / 6x6 torus complex128: see ed_matvec_slot.cuh), without the slotted
    // copy where that cannot be had; else the kernels below
    if (v.kernel == 0 && slot_applies(op, g, ix, track, nvec, dtype)) {
        const size_t bytes = slot_scratch_bytes(ix.slots, nvec, dtype);
        const bool direct = g_kernel_policy == 0 && ix.dim <= (nvec == 1 ? kSlotDirectDim : kSlotBlockMinDim - 1);
        void *xs = !direct && v.scratch_bytes >= bytes ? v.scratch : nullptr;
        void *own = nullptr;
        if (!xs && !direct && v.alloc && !stream_captured(stream) && ws_alloc_optional(&own, bytes, stream) == cudaSuccess)
            xs = own;
        const cudaError_t e = launch_slot(op, g, ix, track, x, y, xs, nvec, dtype, stream);
        const cudaError_t e2 = ws_free(own, stream);
        return e != cudaSuccess ? e : e2;
    }
    // the term-parallel kernel: one vector (use_term_parallel), or a real
    // block of 8 vectors: by default in fp32 (ring N=32 / 36 / 40: 1.69 /
    // 43.6 / 724 ms against 2.04 / 48.4 / 788 ms row-per-lane), in fp64 when
    // the autotuner or the test policy chooses it (its segmented scan adds on
    // the slow fp64 pipe)
    const bool block8 = nvec == 8 && (dtype == ED_F64 || dtype == ED_F32);
    const bool tp_ok = (ix.htab || ix.bkt) && (nvec == 1 || block8) && op.exchange_only;
    const bool rule = block8 ? (g_kernel_policy == 2 || (g_kernel_policy == 0 && dtype == ED_F32))
                             : use_term_parallel(nvec, op, dtype, g.n_sites);
    const bool tp = tp_ok && (v.kernel == 2 || ((v.kernel == 0 || v.kernel == 4) && rule));
    count_product(tp ? kProductTerms : kProductRows);
    if (v.prune < 0)
        g.prune = tp ? terms_prune(g, block8) : rows_prune(g, ix.dim);
    if (tp) {
        const TpArgs<1> t = single_tp_args(op, g, ix, x, y);
        const int k = tp_index_kind(t.sec[0]);
        if (block8)
            return dtype == ED_F64 ? tp_single_f64_nv8(t, track, k, stream) : tp_single_f32_nv8(t, track, k, stream);
        switch (dtype) {
        case ED_F64: return tp_single_f64(t, track, k, stream);
        case ED_F32: return tp_single_f32(t, track, k, stream);
        case ED_C128: return tp_single_c128(t, track, k, stream);
        case ED_C64: return tp_single_c64(t, track, k, stream);
        }
        return cudaErrorInvalidValue;
    }
    const MatvecArgs a{op, g, ix, x, y, nvec};
    switch (dtype) {
    case ED_F64: return matvec_f64(a, track, stream);
    case ED_F32: return matvec_f32(a, track, stream);
    case ED_C128: return matvec_c128(a, track, stream);
    case ED_C64: return matvec_c64(a, track, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace edk

// ---------------------------------------------------------------------------
// Exact count of the stored nonzeros of H in a sector: every off-diagonal term
// whose representative is in the basis, plus one diagonal entry per row.  One
// thread per row; counts are summed with integer atomics (order-independent).
// ---------------------------------------------------------------------------
namespace edk {
namespace {

template <typename W, bool kFact>
__global__ void __launch_bounds__(256) k_count_nnz(const OpView op, const GroupView g, const IndexView ix,
                                                   unsigned long long *total)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nm = kFact ? g.n_cos : g.n_perm;
    W *sm_masks = reinterpret_cast<W *>(smem);
    uint8_t *sm_kind = reinterpret_cast<uint8_t *>(sm_masks + (size_t)nm * kMaskStride);
    const W *gm;
    if (kFact)
        gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(g.cos_masks32) : reinterpret_cast<const W *>(g.cos_masks64);
    else
        gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(g.masks32) : reinterpret_cast<const W *>(g.masks64);
    for (int e = threadIdx.x; e < nm * kMaskStride; e += blockDim.x)
        sm_masks[e] = gm[e];
    if (kFact)
        for (int e = threadIdx.x; e < g.n_cos; e += blockDim.x)
            sm_kind[e] = g.cos_kind[e];
    __syncthreads();
    const W full = (W)g.full;
    const int n = g.n_sites;
    unsigned long long cnt = 0;
    for (uint64_t row = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; row < ix.dim;
         row += (uint64_t)gridDim.x * blockDim.x) {
        const W r = (W)ix.states[row];
        cnt += 1;  // the diagonal entry
        for (int q = 0; q < op.n_fam; ++q) {
            const OpFamily fm = op.fams[q];
            int j = 0;
            const W tq = (W)(((uint64_t)r >> fm.delta | (uint64_t)r << (n - fm.delta)) & g.full);
            for (int cc = 0; cc < 4; ++cc) {
                const uint32_t targets = op.offmask[fm.mat * 4 + cc];
                if (!targets)
                    continue;
                const W a = (cc & 2) ? r : (W)~r, b = (cc & 1) ? tq : (W)~tq;
                W bits = a & b & (W)fm.mask;
                while (bits) {
                    const int i = sizeof(W) == 4 ? __ffs((uint32_t)bits) - 1 : __ffsll((long long)bits) - 1;
                    bits &= bits - 1;
                    j = i + (int)fm.delta;
                    j -= j >= n ? n : 0;
                    uint32_t tg = targets;
                    while (tg) {
                        const int cp = __ffs(tg) - 1;
                        tg &= tg - 1;
                        const int fl = cc ^ cp;
                        const W s = r ^ (W((fl >> 1) & 1) << i) ^ (W(fl & 1) << j);
                        W best;
                        int gb;
                        if (kFact && g.prune == 1)
                            rep_search_rot1<W, false>(s, sm_kind, sm_masks, g, g.flip, full, best, gb);
                        else if (kFact && g.prune == 2)
                            rep_search_blocks<W, false>(s, sm_masks, g, g.flip, full, best, gb);
                        else if (kFact)
                            rep_search_fact<W, false>(s, sm_kind, sm_masks, g.n_cos, g.rot_L, g.rot_d, n, g.n_perm,
                                                      g.flip, full, best, gb);
                        else
                            rep_search<W, false>(s, sm_masks, g.n_perm, g.flip, full, best, gb);
                        cnt += find_index((uint64_t)best, ix) >= 0 ? 1 : 0;
                    }
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1)
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0)
        atomicAdd(total, cnt);
}

template <typename W, bool kFact>
cudaError_t nnz_launch(const OpView &op, const GroupView &g, const IndexView &ix, unsigned long long *total,
                       cudaStream_t stream)
{
    const int nm = kFact ? g.n_cos : g.n_perm;
    const size_t smem = (size_t)nm * kMaskStride * sizeof(W) + (size_t)g.n_cos + 16;
    auto kern = k_count_nnz<W, kFact>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((ix.dim + 255) / 256, 152 * 16));
    kern<<<(unsigned)blocks, 256, smem, stream>>>(op, g, ix, total); count_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_count_nnz(const OpView &op, const GroupView &g, const IndexView &ix,
                             unsigned long long *total, cudaStream_t stream)
{
    if (g.n_sites <= 32)
        return g.fact ? nnz_launch<uint32_t, true>(op, g, ix, total, stream)
                      : nnz_launch<uint32_t, false>(op, g, ix, total, stream);
    return g.fact ? nnz_launch<uint64_t, true>(op, g, ix, total, stream)
                  : nnz_launch<uint64_t, false>(op, g, ix, total, stream);
}

}  // namespace edk

extern "C" void edx_kernel_policy(int policy) { edk::g_kernel_policy = policy; }

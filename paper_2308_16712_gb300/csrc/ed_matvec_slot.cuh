// ed_matvec_slot.cuh -- the pull matvec over the slot index (Sec. "Matrix-vector
// product": y_i = sum_j H_ij x_j with getRow and stateToIndex), for operators
// whose two-site terms only exchange antiparallel spins, 1 to 16 interleaved
// vectors of any type, one sector or a batch of sectors.
//
// A launch works on a slotted copy xs of the vectors (k_slot_fill: xs[slot(s)]
// = sqrt(n(s)) x(s)), so that a term needs its representative, one pilot byte
// from L2 and one read of xs; neither the representative's index nor its norm
// nor a check of membership.
//
// Work decomposition.  The grid is persistent; a warp takes a tile of R = 1 ..
// 16 consecutive rows (about 300 terms) and goes through three phases:
//   A  a group of lanes per row (2 for a ring, 8 for a J1-J2 torus, see
//      slot_log_group) shares the row's bond families: they form the diagonal,
//      count the antiparallel bonds, and (after a warp scan) list them in
//      shared memory, the terms of a row contiguous;
//   B  one term per lane and round: the flipped state, its representative, its
//      slot and its coefficient index go back to the list.  Every lane has
//      work in every round but the tile's last; the pilot is read one round
//      ahead of its use;
//   C  the rows are summed from the list: the row's lanes split its terms (and,
//      for several vectors, its columns), each lane gathers with 4 reads in
//      flight and accumulates in registers; a shuffle tree joins the group.
// Summing in phase C takes one addition per term and vector spread over all
// lanes, in chains short enough that no sum is less accurate than by the scan
// (ring N=32 fp32 5.0e-8 of the 64-bit value either way; 5.7e-8 in one chain a lane).  The segmented warp scan of the term-parallel kernel it replaces took
// 5 shuffles and 5 additions per round of 32 terms and vector (and 4 fp64
// multiplications for the coefficients), which on the 1/74-rate fp64 pipe was
// half of an fp64 product and, for 8 vectors, 80 shuffles per round.  Matrix
// entries and characters come multiplied from a table; where all off-diagonal
// entries are one real number it is factored out of the sum, and no
// multiplication is left when the characters are 1.
//
// Beyond L2 the reads of xs are bound by DRAM's rate of random accesses (5.1e10 /s
// over 0.5 GB, 4.1e10 /s over 2 GB, whatever the load's form): ring N=36 fp64
// 25.9 ms of 23, ring N=38 8 vectors fp32 126 of 116.  Within L2 issue slots and the
// L2's 2.9e11 random reads /s overlap in part (ring N=32 fp32: 71 % of the issue
// slots, 0.90 ms against 0.53 for the reads alone).  Against the kernels it
// replaced: those three 41.0, 181 and 1.18 ms; ring N=33 3 vectors complex128
// 99.8 -> 21.1, 6x6 torus complex128 838 -> 184.
//
// The order of every sum depends only on the operator, the type and the number of
// vectors, not on R: results are deterministic, and the same for a sector alone
// (small R, when it is small: one round of terms per tile) or in a batch.
#pragma once

#include "ed_matvec_tp.cuh"

namespace edk {

constexpr int kSlThreads = 256;
constexpr int kSlWarps = kSlThreads / 32;
constexpr int kSlTerms = 640;      // terms of a tile, at most: rows x off-diagonal entries of a row
constexpr int kSlMaxRows = 16;
constexpr int kSlMaxTable = 16384; // bytes of the coefficient table
// Slotted copies beyond this size are gathered without allocating in L1: 6x6 torus
// complex128 486 -> 396 ms; below it that costs (ring N=32 fp32 1.26 -> 1.51 ms,
// 8 vectors, 180 MB, 1.8 -> 2.2 ms), and at 600 MB (ring N=36 fp64) it is even.
constexpr size_t kSlotL2Bytes = 512ull << 20;

// Index of a basis as a launch without the slotted copy reads it (the fields of
// IndexView).
struct SlotFind {
    const uint32_t *htab;
    const void *hent;
    const uint64_t *bkt;
    const ulonglong2 *stash;
    uint32_t n_stash;
    int hbits, hwide, norm_bits, bbits, brem;
};

struct SlotSector {
    union {
        SlotView v;
        SlotFind find;        // launches without the slotted copy
    };
    const uint64_t *states;
    const uint16_t *norms;
    const double2 *chi;       // characters in the order of the search used
    const float2 *chif;
    const void *x;
    const void *xs;           // slotted copy (null: gathered from x)
    void *y;
    uint64_t dim;
    uint64_t tile_begin;      // first tile of this sector in the batch
    int log_rows;             // log2 R
    int flip;
};

template <int kSec>
struct SlotArgs {
    OpView op;
    GroupView g;              // lattice permutations; flip and characters per sector
    int n_sectors;
    int max_order;            // largest expanded group order among the sectors
    int order;                // characters per coefficient table row: 1 when all are 1
    int scalars, stride;      // per row: scalars of a vector row, of a row of xs
    int log_parts;            // lanes that share a row's scalars
    int log_group;            // lanes of a row: 32 >> log2 of the most rows a tile may have
    int chunk;                // tiles taken from the queue at a time
    int beyond_l2;            // the slotted copies exceed L2: gather past L1
    int byte;                 // the coefficient table has at most 256 entries
    uint64_t total_tiles;
    BatchCtl ctl;             // tile queue (zeroed by the fill; null: static tiles), status word and gate
    SlotSector sec[kSec];     // read from the launch parameters (constant bank)
};

// A warp's shared memory: this, the term list (phase A: site | row << 6 |
// (2 family + c) << 10, phase B: slot), and the terms' coefficient indices unless
// the sum has none (a byte each where that is enough).  The list is sized for
// the operator, because what is left of an SM's 256 KB is its L1, and every
// gather on its way occupies a line there: with a list of 640 terms and 16-bit
// indices for all (196 KB at five or six blocks) the 6x6 torus complex128 took
// 372 instead of 207 ms (188 with bytes), ring N=32 fp32 1.07 instead of 0.96,
// and 48 of its products of 8 vectors 74 instead of 47.
template <typename W, typename T>
struct __align__(16) SlotWarp {
    W r[kSlMaxRows];
    uint32_t off[kSlMaxRows + 1];
    T rinv[kSlMaxRows];
    Cplx<T> diag[kSlMaxRows];
};

// Coefficient table: conj(h) chi for (matrix, c = |01> or |10>) x characters, chi
// alone when h is factored out.  Characters of a batch differ by sector and
// are read from there; its table holds conj(h) only.  For a single sector with
// characters the two c share an entry where they can (op.even, cleared by the
// launch otherwise).
__host__ __device__ inline int slot_entries(const OpView &op)
{
    return op.uniform ? 1 : op.even ? op.n_mats : op.n_mats * 2;
}

template <typename T>
__host__ __device__ inline size_t slot_table_bytes(const OpView &op, int order, bool batch)
{
    return (size_t)slot_entries(op) * (batch ? 1 : order) * sizeof(Cplx<T>);
}

// a b with the same rounding wherever it is used (no contraction left to the
// compiler): the products of a sector alone and in a batch must agree in every bit
template <typename T>
__device__ __forceinline__ Cplx<T> coef_mul(Cplx<T> a, Cplx<T> b)
{
    return {fma(a.re, b.re, -(a.im * b.im)), fma(a.re, b.im, a.im * b.re)};
}

template <typename W, typename T, bool kFact>
__host__ __device__ inline void slot_smem_layout(const GroupView &g, const OpView &op, int order, int max_order,
                                                 bool batch, size_t off[7])
{
    const int nm = kFact ? g.n_cos : g.n_perm;
    off[0] = 0;                                                                  // masks
    off[1] = align16(off[0] + (size_t)nm * kMaskStride * sizeof(W));             // families
    off[2] = align16(off[1] + (size_t)op.n_fam * sizeof(OpFamily));              // diagonal entries
    off[3] = align16(off[2] + (size_t)op.n_mats * 4 * sizeof(Cplx<T>));          // coefficients, offmask
    off[4] = align16(off[3] + slot_table_bytes<T>(op, order, batch) + (size_t)op.n_mats * 4);  // coset kinds
    off[5] = align16(off[4] + (kFact ? (size_t)g.n_cos : 0));                    // 1 / sqrt table
    off[6] = align16(off[5] + (size_t)(max_order + 1) * sizeof(T));              // warps
}

__host__ __device__ inline uint32_t slot_list_terms(const OpView &op, int log_group)
{
    return (uint32_t)op.max_terms << (5 - log_group);
}

template <typename W, typename T>
__host__ __device__ inline size_t slot_warp_bytes(const OpView &op, int log_group, bool plain, bool byte,
                                                  bool direct = false)
{
    const size_t terms = slot_list_terms(op, log_group);
    if (direct)  // coefficient index and norm of every term
        return align16(sizeof(SlotWarp<W, T>) + terms * 8);
    return align16(sizeof(SlotWarp<W, T>) + terms * 4 + (plain ? 0 : byte ? terms : terms * 2));
}

template <typename W, typename T, bool kFact>
__host__ __device__ inline size_t slot_smem_bytes(const GroupView &g, const OpView &op, int order, int max_order,
                                                  int log_group, bool batch, bool plain, bool byte,
                                                  bool direct)
{
    size_t off[7];
    slot_smem_layout<W, T, kFact>(g, op, order, max_order, batch, off);
    return off[6] + kSlWarps * slot_warp_bytes<W, T>(op, log_group, plain, byte, direct);
}

// kSearch: 0 every element of the group (factored or not), 1 ring runs, 2 torus
// row keys.  EL: scalars per lane and access.
// Blocks per SM.  By registers: a word of 32 bits and single precision fit 32 of
// them (a few spill; ring N=32 fp32 0.96 -> 0.90 ms), in double precision that
// costs more than the warps give (lanczos of ring N=32 fp64 115 -> 130 ms), and a
// sixth block for 64-bit words changes nothing (they wait for DRAM).  The torus
// with characters gains more from L1 than from a fifth block (186 -> 180 ms).
template <typename W, typename T, bool kTrack, int kSearch>
constexpr int kSlBlocks = sizeof(W) == 8 ? (kTrack && kSearch == 2 ? 4 : 5) : sizeof(T) == 4 && !kTrack ? 8 : 6;

// a b rounded by itself, never contracted into a following addition
__device__ __forceinline__ float mul_alone(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_alone(double a, double b) { return __dmul_rn(a, b); }

// kDirect: without the slotted copy, for calls that cannot have it (no memory, or
// a product that is being captured: a graph with an allocation in it can
// neither be a child of another nor be instantiated twice, and takes its memory
// only when it is launched).  Phase B finds a term's row and norm through the
// basis's own index, phase C forms sqrt(n) x with the rounding of the fill, and
// all else is the same, so the result is the one with the copy bit for bit.  The
// price is a second random read per term, waited for in its round: with the copy
// / without / by the kernels below, ring N=36 fp64 25.9 / 33.2 / 41.0 ms, ring N=38
// 8 vectors fp32 104 / 151 / 180, 6x6 torus complex128 179 / 332 / 837, ring N=32
// fp32 0.91 / 1.32 / 1.21, the batch of XXZ N=28 43 / 63 / 57.  Four blocks per SM
// (ring N=36: five, with spills and less L1, 41.1; three 32.6 but N=32 1.51).
template <typename W, typename T, bool kC, bool kTrack, int kSearch, int EL, int kSec, bool kDirect = false>
__global__ void __launch_bounds__(kSlThreads, kDirect ? 4 : kSlBlocks<W, T, kTrack, kSearch>) k_matvec_slot(const __grid_constant__ SlotArgs<kSec> a)
{
    static_assert(!kC || EL % 2 == 0, "a complex number per lane at least");
    static_assert(!kDirect || kSearch == 0, "the search is chosen at run time");
    constexpr bool kBatch = kSec > 1;
    constexpr bool kWhole = kC || (sizeof(T) == 8 && EL > 1);  // two sums of a row's terms with coefficients
    extern __shared__ __align__(16) unsigned char smem[];
    const bool fact = kSearch > 0 || a.g.fact;
    size_t off[7];
    if (fact)
        slot_smem_layout<W, T, true>(a.g, a.op, a.order, a.max_order, kBatch, off);
    else
        slot_smem_layout<W, T, false>(a.g, a.op, a.order, a.max_order, kBatch, off);
    W *sm_masks = reinterpret_cast<W *>(smem + off[0]);
    OpFamily *sm_fam = reinterpret_cast<OpFamily *>(smem + off[1]);
    Cplx<T> *sm_diag = reinterpret_cast<Cplx<T> *>(smem + off[2]);
    Cplx<T> *sm_coef = reinterpret_cast<Cplx<T> *>(smem + off[3]);
    uint8_t *sm_off = smem + off[3] + slot_table_bytes<T>(a.op, a.order, kBatch);
    uint8_t *sm_kind = smem + off[4];
    T *sm_isq = reinterpret_cast<T *>(smem + off[5]);
    const bool uniform = a.op.uniform != 0;
    const bool plain = !kTrack && uniform;  // no coefficients at all
    const bool byte = kTrack && !kBatch && !kDirect && a.byte, even = kTrack && !kBatch && a.op.even;
    SlotWarp<W, T> &ws = *reinterpret_cast<SlotWarp<W, T> *>(
        smem + off[6] + (threadIdx.x >> 5) * slot_warp_bytes<W, T>(a.op, a.log_group, plain, byte, kDirect));
    uint32_t *term = reinterpret_cast<uint32_t *>(&ws + 1);
    uint16_t *coef = reinterpret_cast<uint16_t *>(term + slot_list_terms(a.op, a.log_group));
    uint8_t *coef8 = reinterpret_cast<uint8_t *>(coef);
    uint16_t *norm = coef + slot_list_terms(a.op, a.log_group);  // kDirect
    {
        const int nm = fact ? a.g.n_cos : a.g.n_perm;
        const W *gm;
        if (fact)
            gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(a.g.cos_masks32)
                                : reinterpret_cast<const W *>(a.g.cos_masks64);
        else
            gm = sizeof(W) == 4 ? reinterpret_cast<const W *>(a.g.masks32)
                                : reinterpret_cast<const W *>(a.g.masks64);
        auto mat = [&](int e) {
            if constexpr (sizeof(T) == 8)
                return load_c<T>(a.op.mats + e);
            else
                return load_cf<T>(a.op.matsf + e);
        };
        for (int e = threadIdx.x; e < nm * kMaskStride; e += blockDim.x)
            sm_masks[e] = gm[e];
        if (fact)
            for (int e = threadIdx.x; e < a.g.n_cos; e += blockDim.x)
                sm_kind[e] = a.g.cos_kind[e];
        for (int e = threadIdx.x; e < a.op.n_fam; e += blockDim.x)
            sm_fam[e] = a.op.fams[e];
        for (int e = threadIdx.x; e < a.op.n_mats * 4; e += blockDim.x) {
            sm_diag[e] = mat(e / 4 * 16 + e % 4 * 5);
            sm_off[e] = a.op.offmask[e];
        }
        const int per = kBatch ? 1 : a.order;
        for (int e = threadIdx.x; e < slot_entries(a.op) * per; e += blockDim.x) {
            const int cc = even ? 1 : 1 + e / per % 2;
            Cplx<T> c = {T(1), T(0)};
            if (!a.op.uniform)
                c = conjc(mat((even ? e / per : e / per / 2) * 16 + (3 - cc) * 4 + cc));
            if (kTrack && !kBatch) {
                Cplx<T> ch;
                if constexpr (sizeof(T) == 8)
                    ch = load_c<T>(a.sec[0].chi + e % per);
                else
                    ch = load_cf<T>(a.sec[0].chif + e % per);
                c = a.op.uniform ? ch : coef_mul(c, ch);
            }
            sm_coef[e] = c;
        }
        for (int e = threadIdx.x; e <= a.max_order; e += blockDim.x)
            sm_isq[e] = e ? T(1) / sqrt((T)e) : T(0);
    }
    if (!pass_gate(a.ctl))  // includes the barrier after the table loads
        return;

    const unsigned kAll = 0xffffffffu;
    const int n_items = 2 * a.op.n_fam;
    const int n = a.g.n_sites;
    const W full = (W)a.g.full;
    const int lane = threadIdx.x & 31;
    const bool real_op = a.op.real != 0;
    const uint64_t keep = policy_keep();
    const uint32_t mat0 = sm_fam[0].mat, delta0 = sm_fam[0].delta;  // operators of one family

    // Tiles from a queue: dealt statically, the warps of an SM drift apart (the
    // scheduler favours some) and a third of them had finished for most of the
    // launch (ring N=36: 45 % of the warp slots in use on average, 62 % resident).
    // Without a fill to zero a queue (kDirect) they are dealt all the same.
    uint64_t tile = 0, tile_end = 0;
    uint64_t dealt = ((uint64_t)blockIdx.x * kSlWarps + (threadIdx.x >> 5)) * (uint64_t)a.chunk;
    while (true) {
        if (tile == tile_end) {
            if constexpr (kDirect) {
                tile = dealt;
                dealt += (uint64_t)gridDim.x * kSlWarps * (uint64_t)a.chunk;
            } else {
                unsigned long long t = 0;
                if (lane == 0)
                    t = atomicAdd(a.ctl.queue, (unsigned long long)a.chunk);
                tile = __shfl_sync(kAll, t, 0);
            }
            tile_end = min(tile + (uint64_t)a.chunk, a.total_tiles);
            if (tile >= a.total_tiles)
                break;
        }
        int sec = 0;
        if (kBatch) {  // last sector with tile_begin <= tile (warp-uniform)
            int lo = 0, hi = a.n_sectors - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.sec[mid].tile_begin <= tile)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            sec = lo;
        }
        const SlotSector &sd = a.sec[sec];
        const int flip = sd.flip;
        const int log_rows = sd.log_rows;
        const uint64_t row0 = (tile - sd.tile_begin) << log_rows;
        ++tile;

        // ---- A: the rows and their terms ----
        const int per_row = 1 << a.log_group;  // lanes per row
        const int rows = 1 << log_rows;
        const int my = lane >> a.log_group, sub = lane & (per_row - 1);
        const bool valid = my < rows && row0 + my < sd.dim;
        W r = 0;
        uint32_t nt = 0;
        Cplx<T> d = {T(0), T(0)};
        if (valid) {
            r = (W)__ldg(sd.states + row0 + my);
            for (int it = sub; it < n_items; it += per_row) {
                const OpFamily fm = sm_fam[it >> 1];
                const W tq = rot_down(r, (int)fm.delta, n, full);
                const int cc = 1 + (it & 1);  // |01> then |10>, and one of the parallel pairs
                const int cp = (it & 1) * 3;
                const int cnt = popc(config_mask(r, tq, (W)fm.mask, cc));
                const int cnp = popc(config_mask(r, tq, (W)fm.mask, cp));
                const Cplx<T> h = sm_diag[fm.mat * 4 + cc], hp = sm_diag[fm.mat * 4 + cp];
                d.re += h.re * (T)cnt + hp.re * (T)cnp;
                if (!real_op)
                    d.im += h.im * (T)cnt + hp.im * (T)cnp;
                if (sm_off[fm.mat * 4 + cc])
                    nt += (uint32_t)cnt;
            }
        }
        for (int o = per_row >> 1; o > 0; o >>= 1) {
            d.re += __shfl_xor_sync(kAll, d.re, o);
            if (!real_op)
                d.im += __shfl_xor_sync(kAll, d.im, o);
        }
        uint32_t incl = nt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kAll, incl, o);
            if (lane >= o)
                incl += v;
        }
        const uint32_t total = __shfl_sync(kAll, incl, 31);
        if (sub == 0 && my < rows) {
            ws.r[my] = r;
            ws.off[my] = incl - nt;
            ws.diag[my] = d;
            ws.rinv[my] = valid ? sm_isq[__ldg(sd.norms + row0 + my)] : T(0);
        }
        if (lane == 31)
            ws.off[rows] = total;
        if (nt) {
            uint32_t k = incl - nt;
            for (int it = sub; it < n_items; it += per_row) {
                const OpFamily fm = sm_fam[it >> 1];
                const int cc = 1 + (it & 1);
                if (!sm_off[fm.mat * 4 + cc])
                    continue;
                W bits = config_mask(r, rot_down(r, (int)fm.delta, n, full), (W)fm.mask, cc);
                const uint32_t code = (uint32_t)my << 6 | (uint32_t)it << 10;
                while (bits) {
                    term[k++] = code | (uint32_t)lowest_bit(bits);
                    bits &= bits - 1;
                }
            }
        }
        __syncwarp();

        // ---- B: representative, slot and coefficient of every term ----
        SlotKey key = {0, 0};
        uint32_t bucket = 0, pilot = 0;
        for (uint32_t base = 0; base < total + 32; base += 32) {
            const uint32_t t = base + lane;
            const SlotKey key_p = key;
            const uint32_t bucket_p = bucket, pilot_p = pilot;
            if (t < total) {
                const uint32_t code = term[t];
                uint32_t mat = mat0, delta = delta0;
                if (n_items > 2) {
                    mat = sm_fam[code >> 11].mat;
                    delta = sm_fam[code >> 11].delta;
                }
                const int i = (int)(code & 63u);
                int j = i + (int)delta;
                j -= j >= n ? n : 0;
                const W s = ws.r[(code >> 6) & 15u] ^ (W(1) << i) ^ (W(1) << j);
                W best;
                int gbest = 0;
                if constexpr (kSearch == 1) {
                    rep_search_rot1<W, kTrack>(s, sm_kind, sm_masks, a.g, flip, full, best, gbest);
                } else if constexpr (kSearch == 2) {
                    rep_search_blocks<W, kTrack>(s, sm_masks, a.g, flip, full, best, gbest);
                } else if (kDirect && a.g.fact && a.g.prune == 1) {
                    rep_search_rot1<W, kTrack>(s, sm_kind, sm_masks, a.g, flip, full, best, gbest);
                } else if ((kBatch || kDirect) && a.g.fact && a.g.prune == 2) {
                    rep_search_blocks<W, kTrack>(s, sm_masks, a.g, flip, full, best, gbest);
                } else if (a.g.fact) {
                    if (kTrack)
                        rep_search_fact<W, true>(s, sm_kind, sm_masks, a.g.n_cos, a.g.rot_L, a.g.rot_d, n, a.g.n_perm,
                                                 flip, full, best, gbest);
                    else
                        best = rep_min_fact<W>(s, sm_kind, sm_masks, a.g.n_cos, a.g.rot_L, a.g.rot_d, n, flip, full);
                } else {
                    rep_search<W, kTrack>(s, sm_masks, a.g.n_perm, flip, full, best, gbest);
                }
                if (!plain) {
                    const uint32_t entry = uniform ? 0u : even ? mat : mat * 2 + ((code >> 10) & 1u);
                    const uint32_t at = entry * (uint32_t)a.order + (uint32_t)gbest;
                    if (byte)
                        coef8[t] = (uint8_t)at;
                    else
                        coef[t] = (uint16_t)at;
                }
                if constexpr (kDirect) {
                    uint32_t row = 0, nj = 0;
                    bool found;
                    if (sd.find.bkt) {
                        found = find_bucketed((uint64_t)best, sd.find.bkt, sd.find.stash, sd.find.n_stash, n,
                                              sd.find.bbits, sd.find.brem, row, nj);
                    } else {
                        IndexView ix;
                        ix.htab = sd.find.htab;
                        ix.hent = sd.find.hent;
                        ix.hbits = sd.find.hbits;
                        ix.hwide = sd.find.hwide;
                        ix.norm_bits = sd.find.norm_bits;
                        found = find_hashed((uint64_t)best, ix, row, nj);
                    }
                    term[t] = row;
                    norm[t] = found ? (uint16_t)nj : (uint16_t)0;  // 0: without weight, not in the basis
                } else {
                    key = slot_key((uint64_t)best);
                    bucket = slot_bucket((uint64_t)best, key, sd.v);
                    pilot = load_pilot(sd.v.pilots + bucket, keep);
                }
            }
            if (!kDirect && base && t - 32 < total)
                term[t - 32] = slot_finish(key_p, bucket_p, pilot_p, sd.v);
        }
        __syncwarp();

        // ---- C: gather and sum ----
        const int parts = 1 << a.log_parts;                       // lanes that share a row's scalars
        const int log_split = max(0, a.log_group - a.log_parts);  // lanes that share a part's terms
        const int split = 1 << log_split;
        const int part = lane & (parts - 1);
        const int sp = (lane >> a.log_parts) & (split - 1);
        const int e0 = part * EL;
        struct __align__(sizeof(T) * EL) Vec { T e[EL]; };
        const T *xs = reinterpret_cast<const T *>(sd.xs) + e0;
        const T *x = reinterpret_cast<const T *>(sd.x);
        T *y = reinterpret_cast<T *>(sd.y);
        const bool whole = a.scalars % EL == 0;
        const int group = a.log_parts + log_split;
        for (int first = 0; first < rows; first += 32 >> group) {  // same trip count for all lanes
            const int rr = first + (lane >> group);
            const bool mine = rr < rows && e0 < a.scalars;
            T acc[2][EL];
#pragma unroll
            for (int e = 0; e < EL; ++e)
                acc[0][e] = acc[1][e] = T(0);
            if (mine) {
                const uint32_t k1 = ws.off[rr + 1];
                for (uint32_t k = ws.off[rr] + sp; k < k1; k += 4 * split) {
                    Vec v[4];
                    uint32_t ci[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t q = k + u * split;
                        if (kDirect && q < k1) {
                            // row 0 stands in for a state that is not in the basis
                            const T *from = x + (uint64_t)term[q] * (uint32_t)a.scalars + e0;
                            if (whole) {
                                v[u] = *reinterpret_cast<const Vec *>(from);
                            } else {
#pragma unroll
                                for (int e = 0; e < EL; ++e)
                                    v[u].e[e] = e0 + e < a.scalars ? from[e] : T(0);
                            }
                            ci[u] = plain ? 0u : coef[q];
                        } else if (q < k1) {
                            const T *from = xs + (uint64_t)term[q] * (uint32_t)a.stride;
                            if (a.beyond_l2)
                                load_random<sizeof(Vec)>(&v[u], from);
                            else
                                v[u] = *reinterpret_cast<const Vec *>(from);
                            ci[u] = plain ? 0u : byte ? coef8[q] : coef[q];
                        } else {
                            ci[u] = 0;
#pragma unroll
                            for (int e = 0; e < EL; ++e)
                                v[u].e[e] = T(0);
                        }
                    }
                    if constexpr (kDirect) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint32_t q = k + u * split;
                            const uint32_t nj = q < k1 ? norm[q] : 1u;
                            if (nj != 1) {  // few states of a large sector
                                const T sq = sqrt((T)nj);
#pragma unroll
                                for (int e = 0; e < EL; ++e)
                                    v[u].e[e] = nj ? mul_alone(sq, v[u].e[e]) : T(0);
                            }
                        }
                    }
                    // short chains of additions: four terms as a tree; with
                    // coefficients two sums for alternate terms, for the whole row, or
                    // (real, but for several fp64 vectors) for the four.  Two per four
                    // terms add 12 % to a complex sum and half to a real one, which the
                    // fp64 pipe feels (5x6 torus, 8 vectors fp64, 3.72 -> 4.95 ms); one
                    // fp64 vector does not (2.76 ms either way), and on the 6x6 torus
                    // took 199 ms with them and 362 with the longer-lived two
                    if (plain) {
#pragma unroll
                        for (int e = 0; e < EL; ++e)
                            acc[0][e] += (v[0].e[e] + v[1].e[e]) + (v[2].e[e] + v[3].e[e]);
                    } else {
                        T four[2][EL];
#pragma unroll
                        for (int e = 0; e < EL; ++e)
                            four[0][e] = four[1][e] = T(0);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            T (&sum)[EL] = kWhole ? acc[u & 1] : four[u & 1];
                            Cplx<T> c;
                            if (kBatch && kTrack) {
                                const uint32_t m = uniform ? 0u : ci[u] / (uint32_t)a.order;
                                const uint32_t q = ci[u] - m * (uint32_t)a.order;
                                if constexpr (sizeof(T) == 8)
                                    c = load_c<T>(sd.chi + q);
                                else
                                    c = load_cf<T>(sd.chif + q);
                                if (!uniform)
                                    c = coef_mul(sm_coef[m], c);
                            } else {
                                c = sm_coef[ci[u]];
                            }
                            if constexpr (kC) {
#pragma unroll
                                for (int e = 0; e < EL; e += 2) {
                                    sum[e] = fma(c.re, v[u].e[e], fma(-c.im, v[u].e[e + 1], sum[e]));
                                    sum[e + 1] = fma(c.re, v[u].e[e + 1], fma(c.im, v[u].e[e], sum[e + 1]));
                                }
                            } else {
#pragma unroll
                                for (int e = 0; e < EL; ++e)
                                    sum[e] = fma(c.re, v[u].e[e], sum[e]);
                            }
                        }
                        if constexpr (!kWhole) {
#pragma unroll
                            for (int e = 0; e < EL; ++e)
                                acc[0][e] += four[0][e] + four[1][e];
                        }
                    }
                }
                if (kWhole && !plain) {
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        acc[0][e] += acc[1][e];
                }
            }
            for (int o = split >> 1; o > 0; o >>= 1)
#pragma unroll
                for (int e = 0; e < EL; ++e)
                    acc[0][e] += __shfl_xor_sync(kAll, acc[0][e], o << a.log_parts);
            if (sp == 0 && mine && row0 + rr < sd.dim) {
                const uint64_t at = (row0 + rr) * (uint32_t)a.scalars + e0;
                Vec xv;
                if (whole) {
                    xv = *reinterpret_cast<const Vec *>(x + at);
                } else {
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        xv.e[e] = e0 + e < a.scalars ? x[at + e] : T(0);
                }
                const Cplx<T> dg = ws.diag[rr];
                const T w = uniform ? ws.rinv[rr] * (T)a.op.scale : ws.rinv[rr];
                Vec out;
                if constexpr (kC) {
#pragma unroll
                    for (int e = 0; e < EL; e += 2) {  // conj(d) x + w acc
                        out.e[e] = fma(w, acc[0][e], dg.re * xv.e[e]);
                        out.e[e + 1] = fma(w, acc[0][e + 1], dg.re * xv.e[e + 1]);
                        if (!real_op) {
                            out.e[e] = fma(dg.im, xv.e[e + 1], out.e[e]);
                            out.e[e + 1] = fma(-dg.im, xv.e[e], out.e[e + 1]);
                        }
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        out.e[e] = fma(w, acc[0][e], dg.re * xv.e[e]);
                }
                if (whole) {
                    *reinterpret_cast<Vec *>(y + at) = out;
                } else {
#pragma unroll
                    for (int e = 0; e < EL; ++e)
                        if (e0 + e < a.scalars)
                            y[at + e] = out.e[e];
                }
            }
        }
        __syncwarp();
    }
}

template <typename W, typename T, bool kC, bool kTrack, int kSearch, int EL, int kSec, bool kDirect>
cudaError_t slot_launch(const SlotArgs<kSec> &a, cudaStream_t stream)
{
    auto kern = k_matvec_slot<W, T, kC, kTrack, kSearch, EL, kSec, kDirect>;
    const bool plain = !kTrack && a.op.uniform, byte = kTrack && kSec == 1 && a.byte;
    const size_t smem = kSearch > 0 || a.g.fact
                            ? slot_smem_bytes<W, T, true>(a.g, a.op, a.order, a.max_order, a.log_group, kSec > 1, plain, byte, kDirect)
                            : slot_smem_bytes<W, T, false>(a.g, a.op, a.order, a.max_order, a.log_group, kSec > 1, plain, byte, kDirect);
    int sms = 0, per_sm = 0;
    const cudaError_t e = kernel_occupancy((const void *)kern, kSlThreads, smem, &sms, &per_sm);
    if (e != cudaSuccess)
        return e;
    const uint64_t blocks_needed = (a.total_tiles + kSlWarps - 1) / kSlWarps;
    if (!kDirect)
        per_sm = std::min(per_sm, kSlBlocks<W, T, kTrack, kSearch>);
    const int grid = (int)std::min<uint64_t>(blocks_needed, (uint64_t)sms * std::max(1, per_sm));
    kern<<<std::max(grid, 1), kSlThreads, smem, stream>>>(a); count_launch();
    return cudaGetLastError();
}

template <typename T, bool kC, int kSearch, int kSec, bool kDirect = false>
cudaError_t slot_dispatch(const SlotArgs<kSec> &a, bool track, int el, cudaStream_t s)
{
    const bool w32 = a.g.n_sites <= 32;
#define ED_SL_W(EL)                                                                                  \
    do {                                                                                             \
        if (w32)                                                                                     \
            return track ? slot_launch<uint32_t, T, kC, true, kSearch, EL, kSec, kDirect>(a, s)      \
                         : slot_launch<uint32_t, T, kC, false, kSearch, EL, kSec, kDirect>(a, s);    \
        return track ? slot_launch<uint64_t, T, kC, true, kSearch, EL, kSec, kDirect>(a, s)          \
                     : slot_launch<uint64_t, T, kC, false, kSearch, EL, kSec, kDirect>(a, s);        \
    } while (0)
    if constexpr (!kC)
        if (el == 1)
            ED_SL_W(1);
    if (el == 2)
        ED_SL_W(2);
    if constexpr (sizeof(T) == 4)
        if (el == 4)
            ED_SL_W(4);
#undef ED_SL_W
    return cudaErrorInvalidValue;
}

// ed_matvec.cu: lanes of a row (log2), a sector's descriptor (tile_begin 0; xs
// null: without the copy) and its number of tiles; alone: tiles small enough to
// occupy the GPU; whether the stream is being captured
bool stream_captured(cudaStream_t s);
int slot_log_group(const OpView &op);
SlotSector slot_sector(const OpView &op, const GroupView &g, const IndexView &ix, const void *x, const void *xs,
                       void *y, bool alone);
int slot_chunk(uint64_t tiles);
uint64_t slot_tiles(const SlotSector &d);

// one sector / a batch, per dtype and search, and without the copy, in the
// ed_matvec_slot_*.cu units
#define ED_SLOT_DECL(NAME)                                                                        \
    cudaError_t slot1_##NAME(const SlotArgs<1> &a, int search, bool track, int el, cudaStream_t s); \
    cudaError_t slotn_##NAME(const SlotArgs<kMaxSectors> &a, int search, bool track, int el, cudaStream_t s); \
    cudaError_t slot1_direct_##NAME(const SlotArgs<1> &a, bool track, int el, cudaStream_t s);    \
    cudaError_t slotn_direct_##NAME(const SlotArgs<kMaxSectors> &a, bool track, int el, cudaStream_t s);
ED_SLOT_DECL(f64)
ED_SLOT_DECL(f32)
ED_SLOT_DECL(c128)
ED_SLOT_DECL(c64)
#undef ED_SLOT_DECL

}  // namespace edk

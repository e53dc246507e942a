// ed_kernels.cuh -- launch wrappers exported by the kernel translation units to
// the host API (ed_api.cu).  All functions enqueue on `stream` and return the
// CUDA error of the launch.
#pragma once

#include "ed_internal.cuh"

namespace edk {

// Library-owned, stream-ordered device memory (see ed_pool.cu): allocations
// and frees are ordered on stream s; freed memory stays cached for later calls.
cudaError_t ws_alloc(void **p, size_t bytes, cudaStream_t s);
// The same for memory that the caller can do without: no error is left pending
// and *p is null when it cannot be had.
cudaError_t ws_alloc_optional(void **p, size_t bytes, cudaStream_t s);
cudaError_t ws_free(void *p, cudaStream_t s);
// Bytes the pool holds freed and ready for reuse (counted as free memory when
// a solver decides whether its vectors fit).
size_t ws_cached_bytes();

// Kernel launches issued by the library since it was loaded (diagnostics).
void count_launch(unsigned n = 1);
// Takes back n counted launches (kernels recorded into a graph by stream
// capture are counted again each time the graph is launched).
void uncount_launch(unsigned n);
// Products issued (a captured one counts once), by the kernel that serves them;
// one batched launch is one product (diagnostics).
enum ProductKernel { kProductRows, kProductTerms, kProductSlots, kProductDirect, kProductKinds };
void count_product(ProductKernel k);
unsigned long long launches_so_far();

// ---- basis build (Sec. "States enumeration") --------------------------------
struct EnumPlan {
    int n_sites;
    int n_up;            // -1: all 2^n_sites states
    uint64_t total;      // states to visit
    uint64_t chunk;      // states per thread
    uint64_t n_chunks;
    const uint64_t *binom;  // device (65 x 65) binomial table
    // Optional: one bit per visited state, set by the count pass for the
    // states it keeps (flag_words 32-bit words per chunk); the write pass then
    // tests only those states again (for their norms) instead of all of them.
    uint32_t *flags = nullptr;
    uint32_t flag_words = 0;
    // Optional: the count pass lists the representatives of norm 0 here (at
    // most ghost_cap of them; *ghost_count counts all)
    uint64_t *ghosts = nullptr;
    uint32_t *ghost_count = nullptr;
    uint32_t ghost_cap = 0;
    // Optional: only the states whose top n_sites - low_bits bits can belong to a
    // representative (see launch_prefix_filter), segment by segment in
    // ascending order; total then counts the states of the segments.
    const uint32_t *seg_prefix = nullptr;  // the top bits
    const uint64_t *seg_start = nullptr;   // n_seg + 1: states before each segment
    uint32_t n_seg = 0;
    int low_bits = 0;
    int odd = 0;                           // 1: bit 0 is set in every state
    int turn[3] = {0, 0, 0};               // set by the launch: n_sites / p for its prime factors p
};

// The values of the top `bits` bits (bits < n_sites) a representative can
// have, by the bits alone: a value is out when some group element, compared
// with the identity from the top bit down through bits that are known, makes a
// smaller word.  prefix / start (2^bits and 2^bits + 1 entries) get the
// remaining ones in ascending order and the running number of their states
// (popcount n_up; n_up < 0: all; bit 0 set if odd), *n_seg their number.  inv:
// n_perm x n_sites bytes, the site that goes to each site.  tmp: work memory of
// prefix_filter_bytes(bits) bytes.
size_t prefix_filter_bytes(int bits);
cudaError_t launch_prefix_filter(int n_sites, int n_up, int odd, int bits, const uint8_t *inv, int n_perm, int flip,
                                 const uint64_t *binom, void *tmp, uint32_t *prefix, uint64_t *start,
                                 uint32_t *n_seg, cudaStream_t stream);

// Reads and clears the basis kernels' device status word (synchronous).
cudaError_t basis_status_take(unsigned int *status);
// Status word of the batched matvec launches: kStatusTimeout = a block gave up
// a bounded wait.  Reads and clears the word of the current device.
constexpr unsigned kStatusTimeout = 2u;
cudaError_t batch_status_take(unsigned int *st);
// Pass 1: per-chunk representative counts.
cudaError_t launch_enum_count(const EnumPlan &plan, const GroupView &g, uint32_t *counts,
                              cudaStream_t stream);
// Pass 2: write representatives and norms at offsets[chunk].
cudaError_t launch_enum_write(const EnumPlan &plan, const GroupView &g, const uint64_t *offsets,
                              uint64_t *states, uint16_t *norms, cudaStream_t stream);
// Exclusive scan of n uint32 counts into n + 1 uint64 offsets (offsets[n] = total).
// `tmp` must hold scan_tmp_words(n) uint64 words.
size_t scan_tmp_words(uint64_t n);
cudaError_t launch_scan(const uint32_t *counts, uint64_t n, uint64_t *offsets, uint64_t *tmp,
                        cudaStream_t stream);
// Prefix table over the ascending basis.
cudaError_t launch_prefix_table(const IndexView &ix, uint32_t *tab, cudaStream_t stream);
// Hash index build: counts[b] += 1 for every state's bucket (counts zeroed),
// then (after an exclusive scan into offsets) entries scattered into buckets.
cudaError_t launch_hash_count(const uint64_t *states, uint64_t dim, int hbits, uint32_t *counts,
                              cudaStream_t stream);
cudaError_t launch_offsets_to_u32(const uint64_t *offsets, uint64_t n, uint32_t *out, cudaStream_t stream);
cudaError_t launch_hash_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int hbits,
                             uint32_t *cursor, void *entries, int wide, int norm_bits,
                             cudaStream_t stream);
// Bucketed index build: every basis state into the first free slot of its
// primary bucket, else of its alternative bucket, else appended to the stash
// (at most stash_cap entries; *n_stash counts every stash insertion, so a value
// above stash_cap means entries were dropped).  bkt must be all ones (empty),
// cnt (2^bbits counters) zero.
cudaError_t launch_bucket_fill(const uint64_t *states, const uint16_t *norms, uint64_t dim, int n_sites,
                               int bbits, int brem, uint32_t *cnt, uint64_t *bkt, ulonglong2 *stash,
                               uint32_t *n_stash, uint32_t stash_cap, cudaStream_t stream);
// *out = max over buckets of tab[t+1] - tab[t] (*out must start at 0)
cudaError_t launch_max_bucket(const uint32_t *tab, uint64_t tab_size, uint32_t *out, cudaStream_t stream);
// keys[i] = states[i] << 16 | norms[i]
cudaError_t launch_pack_keys(const uint64_t *states, const uint16_t *norms, uint64_t dim, uint64_t *keys,
                             cudaStream_t stream);
// Sets *flag to 1 if the basis is not strictly ascending.
cudaError_t launch_check_sorted(const uint64_t *states, uint64_t dim, int *flag, cudaStream_t stream);

// ---- state -> index -----------------------------------------------------------
cudaError_t launch_index(const IndexView &ix, const uint64_t *query, int64_t *out, uint64_t n,
                         cudaStream_t stream);

// ---- matvec (Sec. "Matrix-vector product") --------------------------------------
struct OpView {
    int n_fam;
    int n_mats;
    int max_terms;           // most off-diagonal terms one row can produce
    const OpFamily *fams;    // rotation families
    const double2 *mats;     // n_mats x 16, coeff * h
    const float2 *matsf;
    const uint8_t *offmask;  // n_mats x 4: bit c' set if h[c'][c] != 0, c' != c
    int exchange_only;       // every off-diagonal entry couples |01> and |10>
    int real;                // every entry is real
    int uniform;             // every nonzero off-diagonal entry is the real number `scale`
    double scale;
    int even;                // every matrix has the same entry for |01> and |10>
};

// Host tables (generic group search) for counting a sector; validates the group.
ed_status count_tables_host(int n_sites, int n_up, int spin_inversion, int n_elems,
                            const int32_t *perms, const double *chars,
                            std::vector<uint32_t> &masks32, std::vector<uint64_t> &masks64,
                            std::vector<uint32_t> &chi_one);
uint64_t binomial_host(int n, int k);

// The index ed_basis_build makes (test hook and autotuner): 0 automatic,
// 1 hash index, 2 bucketed index where its entry fits.
int index_policy_get();
void index_policy_set(int policy);

// Operator/basis compatibility check (n_sites, symmetry); the outcome is kept per group.
ed_status check_pair(const ed_operator *op, const ed_basis *b);
OpView make_op_view(const ed_operator *op);

// *total += stored nonzeros of H in the sector (off-diagonal terms found in
// the basis plus one diagonal entry per row)
cudaError_t launch_count_nnz(const OpView &op, const GroupView &g, const IndexView &ix,
                             unsigned long long *total, cudaStream_t stream);

cudaError_t launch_matvec(const OpView &op, const GroupView &g, const IndexView &ix, bool track,
                          const void *x, void *y, int nvec, ed_dtype dtype, cudaStream_t stream);
// A product variant: kernel 0 = the library's rule (use_term_parallel),
// 1 = row-per-lane, 2 = term-parallel (where it applies), 4 = the rule without
// the slot kernel; prune -1 = the
// group's own setting, 0 = every rotation, 1 = the pruned search (rotation
// step one site only).
struct MatvecVariant {
    int kernel = 0;
    int prune = -1;
    void *scratch = nullptr;   // the caller's memory for the slotted copy of x, if any
    size_t scratch_bytes = 0;
    bool alloc = true;         // the product may take that memory from the pool
};
// The search of the row-per-lane and term-parallel kernels, from the group's own
// (GroupView::prune).  The pruned searches take fewer instructions in longer
// chains, which loses where a product is latency.  Rows: every element up to 17
// of them on a ring (16 sites without reflection, 415 states, 8 vectors fp64 34.1
// against 36.0 us; 18 sites at momentum 1, 2700 states, complex128 36.4 against
// 36.2), and on a torus below kRowsTableDim states (4x4, 441 states, 8 vectors
// fp64 128 against 167 us; 4x10, 96045 states, fp64 297 against 416; 4x9, 231880
// states, 589 against 530; in a batch each sector by its own dimension).  Terms: every
// element for blocks of 8 on a ring of up to 24 elements (16 sites, 21.7 against
// 23.2 us), and on tori whose table keys are one row or rows of two sites, which
// leave many candidates (8x8, 4 up, fp64 184 against 311 us; 2x8 102 against 110).
constexpr uint64_t kRowsTableDim = 1ULL << 17;
inline int rows_prune(const GroupView &g, uint64_t dim)
{
    return (g.prune == 1 && g.n_perm < 18) || (g.prune == 2 && dim < kRowsTableDim) ? 0 : g.prune;
}
inline int terms_prune(const GroupView &g, bool block8)
{
    return (g.prune == 1 && block8 && g.n_perm <= 24) || (g.prune == 2 && (g.blk_rows == 1 || g.rot_d == 2))
               ? 0 : g.prune;
}
cudaError_t launch_matvec_v(const OpView &op, GroupView g, const IndexView &ix, bool track, const void *x,
                            void *y, int nvec, ed_dtype dtype, MatvecVariant v, cudaStream_t stream);
// ---- slot index (ed_slots.cu) and the product over it (ed_matvec_slot.cuh) --------
bool build_slot_index(ed_basis *b, uint64_t *ghosts, uint32_t n_ghost, int *err, std::vector<uint2> &cells,
                      cudaStream_t stream);
void free_slot_index(ed_basis *b);
// Layout of a row of the slotted copy: scalars of a row, scalars per access, row stride.
struct SlotRow {
    int scalars, el, stride;
};
SlotRow slot_row(int nvec, ed_dtype dtype);
size_t slot_copy_bytes(const SlotView &v, int nvec, ed_dtype dtype);
// scratch of one product: the copy and, behind it, the tile queue
constexpr size_t kSlotQueueBytes = 256;
inline size_t slot_scratch_bytes(const SlotView &v, int nvec, ed_dtype dtype)
{
    return slot_copy_bytes(v, nvec, dtype) + kSlotQueueBytes;
}
// Whether a solver whose vectors are allocated takes that scratch for its call:
// free device memory (what the pool holds cached included) less what the call
// still allocates, with room left for what the driver loads at a first launch.
// Ring N=40, 8 vectors in single precision: 32.9 of some 56 GB; a block step takes
// 0.61 s with it, 0.91 s by the term-parallel kernel.
constexpr size_t kSlotReserve = 512ull << 20;
inline bool slot_scratch_fits(size_t want, size_t free_bytes, size_t later)
{
    return want + later + kSlotReserve <= free_bytes;
}
// One sector's part of a fill: x (rows of nvec values) into xs.
struct SlotFill {
    SlotView v;
    const uint64_t *states;
    const uint16_t *norms;
    uint64_t dim;
    const void *x;
    void *xs;
};
constexpr int kSlotMaxBatch = 160;
cudaError_t launch_slot_fill(const SlotFill *sec, int n, int nvec, ed_dtype dtype, unsigned long long *queue,
                             cudaStream_t s);
// Whether the slot kernel serves products of this operator over this basis.
bool slot_applies(const OpView &op, const GroupView &g, const IndexView &ix, bool track, int nvec, ed_dtype dtype);

// Multiprocessors of the current device and resident blocks of a kernel on one
// of them at this block size and dynamic shared memory (set as its limit);
// asked of the driver once per device, kernel and size.
cudaError_t kernel_occupancy(const void *kern, int threads, size_t smem, int *sms, int *per_sm);

// The variant ed_autotune found fastest for this basis, nvec and dtype on the
// current GPU (the default variant when none was tuned).
MatvecVariant tuned_variant(const ed_basis *b, int nvec, ed_dtype dtype);
// The index kind (1 hash, 2 bucketed) ed_autotune_index found faster for
// sectors like this one on the current GPU, or 0 when none was tuned.
int tuned_index_kind(int n_sites, int order, int flip, uint64_t dim);
// The transposed (push) form, one vector, for the ablation hook: y zeroed,
// then every contribution added atomically (order-dependent rounding).
cudaError_t launch_matvec_push(const OpView &op, const GroupView &g, const IndexView &ix, bool track,
                               const void *x, void *y, ed_dtype dtype, cudaStream_t stream);

// Kernel choice for exchange-only operators (test hook): 0 = the slot kernel where
// slot_applies, without the copy for the smallest sectors, else use_term_parallel's
// rule; 1 = always row-per-lane; 2 = term-parallel (one vector, real blocks of 8);
// 3 = the slot kernel for every block of vectors, with the copy where it can be had.
extern int g_kernel_policy;
// The rule without the slot kernel, for one vector.
bool use_term_parallel(int nvec, const OpView &op, ed_dtype dtype, int n_sites);

}  // namespace edk

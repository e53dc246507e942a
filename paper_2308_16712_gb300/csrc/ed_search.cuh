// ed_search.cuh -- representative searches that prune the group instead of
// visiting every element: for ring translations (rep_search_rot1) and for torus
// translations (rep_search_blocks).  Included by ed_internal.cuh.
//
// Both are bound by integer issue slots (no memory in the ring search, a few
// table reads in the torus search), so what counts is instructions per warp:
// every loop below either has a trip count that is the same for all lanes or
// one whose maximum over the lanes is small.
#pragma once

namespace edk {

// Low 32 bits of the 64-bit word hi:lo shifted right by s mod 32.
__host__ __device__ __forceinline__ uint32_t funnel_right(uint32_t lo, uint32_t hi, int s)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> (s & 31));
#endif
}

template <typename W>
__host__ __device__ __forceinline__ int lowest_set(W v)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(W) == 4)
        return __ffs((int)v) - 1;
    else
        return __ffsll((long long)v) - 1;
#else
    return __builtin_ctzll((unsigned long long)v);
#endif
}

__host__ __device__ __forceinline__ uint32_t reverse_bits(uint32_t s, int n)
{
#ifdef __CUDA_ARCH__
    return __brev(s) >> (32 - n);
#else
    uint32_t r = 0;
    for (int i = 0; i < n; ++i)
        r |= ((s >> i) & 1u) << (n - 1 - i);
    return r;
#endif
}
__host__ __device__ __forceinline__ uint64_t reverse_bits(uint64_t s, int n)
{
#ifdef __CUDA_ARCH__
    return __brevll(s) >> (64 - n);
#else
    uint64_t r = 0;
    for (int i = 0; i < n; ++i)
        r |= ((s >> i) & 1ull) << (n - 1 - i);
    return r;
#endif
}

// rotation of the n-bit word x up by b (0 <= b < n): bit p goes to p + b mod n
template <typename W>
__host__ __device__ __forceinline__ W rotl_n(W x, int b, int n, W full)
{
    if constexpr (sizeof(W) == 4) {
        if (n == 32)
            return funnel_right(x, x, 32 - b);
        return ((x << b) | (x >> (n - b))) & full;
    } else {
        if (n == 64)
            return (x << b) | (x >> ((64 - b) & 63));
        return ((x << b) | (x >> (n - b))) & full;
    }
}

// ---------------------------------------------------------------------------
// Pruned search for a rotation step of one site (every translation of a ring).
//
// Compared as unsigned integers, a rotation of an n-bit word h is the smaller
// the longer the run of zeros it starts with (at bit n-1).  The minimum over
// all n rotations therefore brings the top of one of the LONGEST zero runs of
// h to bit n-1, and only those rotations need to be formed and compared.  With
// spin inversion the complement of a rotation starts with the complemented
// bits, so a longest run of ones qualifies as well: the candidates are the
// longest runs of equal bits.  The bit reversal maps a run to its mirror image,
// so the candidates of the reversal coset are the same runs read from the other
// end.  The minimum equals the brute-force minimum over the rotations of every
// coset image; the minimiser may differ only by an element of the stabiliser of
// the minimum.
// ---------------------------------------------------------------------------

// Lowest bits p of the longest cyclic runs of ones of the n-bit word b (p, p+1,
// ..., p+g-1 mod n), and their length g; b neither empty nor full.  With
// P_k = {p : bits p .. p+k-1 are set}, P_{j+k} = P_j & (P_k rotated down by j):
// P_2, P_4, P_8 by doubling, then the length bit by bit from 8 down to 1 (a
// fixed number of steps for all lanes; the linear search P_{k+1} = P_k &
// rot(P_k) takes as many as the longest run of the 32 lanes, about 9), longer
// runs one at a time.  rot(x, k): x rotated down by k.  Only the bits of `keep`
// count: those above may be wrong (they are, in a word repeated by shifting).
template <typename X, typename F>
__host__ __device__ __forceinline__ X longest_ones(X p1, X keep, int &g, F &&rot)
{
    const X p2 = p1 & rot(p1, 1);
    const X p4 = p2 & rot(p2, 2);
    const X p8 = p4 & rot(p4, 4);
    X cur = p8 & keep ? p8 : ~X(0);
    int len = p8 & keep ? 8 : 0;
    X t = p4 & rot(cur, 4);
    if (t & keep) {
        cur = t;
        len += 4;
    }
    t = p2 & rot(cur, 2);
    if (t & keep) {
        cur = t;
        len += 2;
    }
    t = p1 & rot(cur, 1);
    if (t & keep) {
        cur = t;
        len += 1;
    }
    g = len;
    return cur;
}

// Lowest bits of the longest runs of equal bits of h (of zeros only when
// !flip), and the length len of those runs.  A word without such a run
// structure (all bits equal; no two equal neighbours with spin inversion; no
// zero without it) has one candidate word: bit 0 stands for it.
template <typename W>
__host__ __device__ __forceinline__ W longest_runs(W h, uint64_t twice, int n, int flip, W full, int &len)
{
    int g = 0;
    W found;
    if constexpr (sizeof(W) == 4) {
        if (n == 32) {
            const uint32_t b = flip ? ~(h ^ funnel_right(h, h, 1)) : ~h;
            auto rot = [](uint32_t x, int k) { return funnel_right(x, x, k); };
            uint32_t cur = longest_ones(b, ~0u, g, rot);
            if (b == 0 || b == ~0u) {
                cur = 1;
                g = 0;
            } else {
                while (g >= 15) {
                    const uint32_t t = b & rot(cur, 1);
                    if (!t)
                        break;
                    cur = t;
                    ++g;
                }
            }
            len = g + (flip ? 1 : 0);
            return cur;
        }
    }
    if (sizeof(W) == 4 || n <= 48) {
        // h repeated with period n in a 64-bit word (`twice`): a rotation down by
        // k is a shift right by k, valid on the low n bits while the shifts of
        // a chain add up to at most 64 - n (16 here, and at most n matter)
        const uint64_t keep = (uint64_t)full;
        const uint64_t p = flip ? ~(twice ^ (twice >> 1)) : ~twice;
        if (!(p & keep) || !(~p & keep)) {
            len = 1;
            return W(1);
        }
        uint64_t cur = longest_ones(p, keep, g, [](uint64_t x, int k) { return x >> k; });
        while (g >= 15) {
            cur &= keep;
            cur |= cur << n;
            const uint64_t t = p & (cur >> 1) & keep;
            if (!t)
                break;
            cur = t;
            ++g;
        }
        found = (W)cur & full;
    } else {
        const W b = (flip ? ~(h ^ ((h >> 1) | (h << (n - 1)))) : ~h) & full;
        if (b == 0 || b == full) {
            len = 1;
            return W(1);
        }
        W cur = b;
        g = 1;
        while (true) {
            const W t = b & rotl_n(cur, n - 1, n, full);
            if (!t)
                break;
            cur = t;
            ++g;
        }
        found = cur;
    }
    len = g + (flip ? 1 : 0);
    return found;
}

// Thins out candidates before they are formed one by one: of the runs whose
// lowest bits are c, keeps those whose continuation can be the smallest.  Read
// downwards from a run the next bit differs from it; of the kNarrow bits after
// that, one after the other, candidates that continue with the run's own value
// (a zero of the candidate word; any zero without spin inversion) win over the
// others.  `down` gets the survivors read downwards, as lowest bit - kNarrow - 1;
// `up` those read upwards (the mirrored candidates).  Each step is the same few
// instructions for all lanes and halves the candidates beyond the first; the
// loop over candidates then takes one pass for most warps instead of the four
// or five of the lane with the most runs.  rot as in longest_ones; words
// repeated with period n, valid on the bits of `keep`.
constexpr int kNarrow = 4;
template <typename X, typename F>
__host__ __device__ __forceinline__ void narrow_runs(X h, X c, X keep, int len, int flip, bool mirrored, F &&rot,
                                                     X &down, X &up)
{
    X d = rot(c, kNarrow + 1) & keep;
    X ref = flip ? rot(h, kNarrow + 1) : X(0);
#pragma unroll
    for (int k = 1; k <= kNarrow; ++k) {
        const X t = d & ~(rot(h, kNarrow - k) ^ ref);
        d = t ? t : d;
    }
    down = d;
    if (!mirrored)
        return;
    d = c & keep;
    ref = flip ? h : X(0);
    const X q = rot(h, len);
#pragma unroll
    for (int k = 1; k <= kNarrow; ++k) {
        const X t = d & ~(rot(q, k) ^ ref);
        d = t ? t : d;
    }
    up = d;
}

template <typename W>
__host__ __device__ __forceinline__ int highest_set(W v)
{
#ifdef __CUDA_ARCH__
    if constexpr (sizeof(W) == 4)
        return 31 - __clz((int)v);
    else
        return 63 - __clzll((long long)v);
#else
    return 63 - __builtin_clzll((unsigned long long)v);
#endif
}

// The word h twice in a row; get(s) = h rotated down by s (0 <= s < n).
template <typename W> struct TwiceWord;
template <> struct TwiceWord<uint32_t> {
    uint32_t lo, hi, full;
    __host__ __device__ __forceinline__ TwiceWord(uint32_t h, int n, uint32_t f) : full(f)
    {
        lo = n == 32 ? h : h | (h << n);
        hi = n == 32 ? h : h >> (32 - n);
    }
    __host__ __device__ __forceinline__ uint32_t get(int s) const { return funnel_right(lo, hi, s) & full; }
    __host__ __device__ __forceinline__ uint64_t low() const { return (uint64_t)hi << 32 | lo; }
};
template <> struct TwiceWord<uint64_t> {
    uint32_t w[4], full_hi;
    __host__ __device__ __forceinline__ TwiceWord(uint64_t h, int n, uint64_t f) : full_hi((uint32_t)(f >> 32))
    {
        const uint64_t a = n == 64 ? h : h | (h << n), b = n == 64 ? h : h >> (64 - n);
        w[0] = (uint32_t)a;
        w[1] = (uint32_t)(a >> 32);
        w[2] = (uint32_t)b;
        w[3] = (uint32_t)(b >> 32);
    }
    __host__ __device__ __forceinline__ uint64_t get(int s) const  // n > 32: the low word is complete
    {
        const bool up = (s & 32) != 0;
        const uint32_t a = up ? w[1] : w[0], b = up ? w[2] : w[1], c = up ? w[3] : w[2];
        return ((uint64_t)(funnel_right(b, c, s) & full_hi) << 32) | funnel_right(a, b, s);
    }
    __host__ __device__ __forceinline__ uint64_t low() const { return (uint64_t)w[1] << 32 | w[0]; }
};

// keep the smaller of best and q; complemented when its top bit is set and the
// group has the spin inversion (the complement then starts with the zero run)
template <typename W, bool kTrack>
__host__ __device__ __forceinline__ void take_candidate(W q, int gi, int n, int n_perm, int flip, W full, W &best,
                                                        int &gbest)
{
    if (!kTrack && sizeof(W) == 4) {
        best = min(best, q);
        best = flip ? min(best, (W)(q ^ full)) : best;
        return;
    }
    if (flip && ((q >> (n - 1)) & 1)) {
        q ^= full;
        gi += n_perm;
    }
    if (kTrack) {
        if (q < best) {
            best = q;
            gbest = gi;
        }
    } else {
        best = q < best ? q : best;
    }
}

// rotation within blocks of d bits: masks = {bits reached from below, shift up
// a, shift down d - a, bits reached from above}
template <typename W>
__host__ __device__ __forceinline__ W rotate_blocks(W s, const W *m)
{
    return ((s << (int)m[1]) & m[0]) | ((s >> (int)m[2]) & m[3]);
}

template <typename W>
__host__ __device__ __forceinline__ W coset_image(W s, int kind, const W *masks, int n)
{
    if (kind == 0)
        return s;
    if (kind == 1)
        return reverse_bits(s, n);
    if (kind == 3)
        return rotate_blocks(s, masks);
    return benes_apply(s, masks);
}

// Minimum over the factored group when its rotations step by one site (rot_L
// = n); gbest is a factored index of a minimiser.  `flip` may differ per lane.
// Against the linear run search with a candidate loop per coset (64-bit words)
// and the minimum over all 128 rotations (32-bit words) that it replaced: ring
// N=36 fp64 product 42.3 -> 41.0 ms, ring N=32 fp32 1.248 -> 1.178 ms.
template <typename W, bool kTrack>
__host__ __device__ __forceinline__ void rep_search_rot1(W s, const uint8_t *kinds, const W *masks,
                                                         const GroupView &g, int flip, W full, W &best, int &gbest)
{
    const int n = g.n_sites, n_perm = g.n_perm;
    W bst = ~W(0);
    int gb = 0, len;
    {
        const TwiceWord<W> two(s, n, full);
        const W runs = longest_runs(s, two.low(), n, flip, full, len);
        const int base = g.cos_id * n, base_rev = g.cos_rev * n;
        const bool mirrored = base_rev >= 0;
        W down = runs, up = mirrored ? runs : W(0);
        int below = 0;  // a bit of `down` stands for the run that many bits above
        const int room = n < 64 - n ? n : 64 - n;  // bits by which a doubled word may be shifted
        if (sizeof(W) == 4 && n == 32) {
            uint32_t d, u;
            narrow_runs((uint32_t)s, (uint32_t)runs, ~0u, len, flip, mirrored,
                        [](uint32_t x, int k) { return funnel_right(x, x, k); }, d, u);
            down = (W)d;
            if (mirrored)
                up = (W)u;
            below = kNarrow + 1;
        } else if (n <= 48 && kNarrow + 1 <= room) {
            uint64_t d, u;
            narrow_runs(two.low(), (uint64_t)runs | ((uint64_t)runs << n), (uint64_t)full, len, flip, mirrored,
                        [](uint64_t x, int k) { return x >> k; }, d, u);
            down = (W)d;
            if (mirrored && len + kNarrow <= room)
                up = (W)u;
            below = kNarrow + 1;
        }
        auto take_down = [&]() {
            const int p = highest_set(down);
            down ^= W(1) << p;
            int t = p + below + len;  // rotated down by t, the run's top is bit n - 1
            t -= t >= n ? n : 0;
            t -= t >= n ? n : 0;
            take_candidate<W, kTrack>(two.get(t), base + (t ? n - t : 0), n, n_perm, flip, full, bst, gb);
        };
        auto take_up = [&]() {  // mirrored: rotated down by p and reversed
            const int p = highest_set(up);
            up ^= W(1) << p;
            take_candidate<W, kTrack>(reverse_bits(two.get(p), n), base_rev + p, n, n_perm, flip, full, bst, gb);
        };
        take_down();  // there is always one; the loop is for the few words with more
        if (mirrored)
            take_up();
        while (down | up) {
            if (down)
                take_down();
            if (up)
                take_up();
        }
    }
    for (int c = 0; c < g.n_cos; ++c) {
        if (kinds[c] < 2)
            continue;
        const W h = coset_image(s, (int)kinds[c], masks + c * kMaskStride, n);
        const TwiceWord<W> two(h, n, full);
        W runs = longest_runs(h, two.low(), n, flip, full, len);
        while (runs) {
            const int p = lowest_set(runs);
            runs &= runs - 1;
            int t = p + len;
            t -= t >= n ? n : 0;
            take_candidate<W, kTrack>(two.get(t), c * n + (t ? n - t : 0), n, n_perm, flip, full, bst, gb);
        }
    }
    best = bst;
    gbest = gb;
}

// ---------------------------------------------------------------------------
// Pruned search for the translations of a torus whose rows are blocks of d =
// rot_d bits: the group is {rotation of the word by b d} x {rotation by a
// within every block} (x spin inversion), coset c = a.  Compared as unsigned
// integers, candidates are decided by their top blk_rows rows.  For every
// possible value v of those rows a table holds the smallest value that the
// rotations within blocks (and the complement) make of it (low 16 bits) and
// which of them do (bit 16 + a, bit 16 + d + a with the complement).  The rows
// that reach the smallest table value give the only candidates; with two rows
// of six that is 1.2 on average where the exhaustive search forms 72 (6x6 torus
// complex128 product, fp64-bound otherwise: 949 -> 838 ms).  The table
// without spin inversion comes first, then the one with it.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint32_t read_table(const uint32_t *p)
{
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// Visits those candidates, f(image, factored index), until f returns false;
// returns whether it never did.
template <typename W, typename F>
__host__ __device__ __forceinline__ bool blocks_candidates(W s, const W *masks, const GroupView &g, int flip, W full,
                                                           F &&f)
{
    const uint32_t *tab = g.blk_tab + (flip ? 1u << g.blk_bits : 0u);
    const int n = g.n_sites, d = g.rot_d, L = g.rot_L;
    const uint32_t kmask = (1u << g.blk_bits) - 1u;
    const uint64_t twice = (uint64_t)s | (n < 64 ? (uint64_t)s << n : 0);
    uint32_t low = 0xffffu, at = 0;  // smallest key, rows (lowest of the key) that have it
    for (int z = 0; z < L; ++z) {
        const uint32_t k = read_table(tab + ((uint32_t)(twice >> (z * d)) & kmask)) & 0xffffu;
        at = k < low ? 0u : at;
        low = k < low ? k : low;
        at |= (k == low ? 1u : 0u) << z;
    }
    int b = 0;
    uint32_t who = 0;
    while (who | at) {
        if (!who) {
            const int z = lowest_set(at);
            at &= at - 1;
            who = read_table(tab + ((uint32_t)(twice >> (z * d)) & kmask)) >> 16;
            b = 2 * L - g.blk_rows - z;  // rotation that brings those rows to the top
            b -= b >= L ? L : 0;
        }
        const int t = lowest_set(who);
        who &= who - 1;
        const bool inv = t >= d;
        const int a = inv ? t - d : t;
        W q = rotl_n(rotate_blocks(s, masks + a * kMaskStride), b * d, n, full);
        if (inv)
            q ^= full;
        if (!f(q, a * L + b + (inv ? g.n_perm : 0)))
            return false;
    }
    return true;
}

template <typename W, bool kTrack>
__host__ __device__ __forceinline__ void rep_search_blocks(W s, const W *masks, const GroupView &g, int flip, W full,
                                                           W &best, int &gbest)
{
    W bst = ~W(0);
    int gb = 0;
    blocks_candidates<W>(s, masks, g, flip, full, [&](W q, int gi) {
        if (kTrack) {
            if (q < bst) {
                bst = q;
                gb = gi;
            }
        } else {
            bst = q < bst ? q : bst;
        }
        return true;
    });
    best = bst;
    gbest = gb;
}

}  // namespace edk

// count_impl.cuh -- device templates of the counting phase (included by count.cu and by the
// per-k translation units count_k*.cu, which instantiate them in parallel builds).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "common.cuh"
#include "dense.cuh"

namespace citron {


constexpr int kMaxK = CITRON_MAX_K;
constexpr uint32_t kBitmapCap = 1024;  // largest root handled by the bitmap path
constexpr int kSmallWarps = 8;         // warps per block of k_count_small
constexpr int kListWarps = 4;          // warps per block of k_count_list
constexpr uint32_t kMidWindow = 32768;  // ids in a block's membership bitmap (k_count_mid)

struct CountStats {
    uint32_t n_small, n_mid, n_big;
    uint32_t max_mid, max_big, max_all;
    uint32_t n_high;  // bitmap-path roots of the launch of large blocks, the first n_high of the queue
    uint32_t n_low;   // host copy only: the others, or an upper bound of them
    uint32_t down;    // k >= 5: some row reaches below its own id (a DAG that keeps vertex ids)
};

// Bitmap-path roots of at most kLowMax out-neighbours run in a launch of their own, in blocks of 8 warps,
// several per SM: a block of 32 warps has a handful of rows per warp to build for them and waits at
// its barriers instead.  R-MAT 15, k = 6: 0.70 ms in one launch, 0.64 in two (0.79 with 4 warps).
constexpr uint32_t kLowMax = 128;
constexpr uint32_t kLowWarps = 8;
// From k = 5 on that launch needs a root for every block of 8 warps that the chip holds, kLowIds times as
// many in a DAG that keeps ids, whose sets are enumerated: with fewer a root is left to 8 warps while
// others idle, and what is a short launch of its own comes after the tail of the other one.  40 roots of
// 99, k = 6, ids kept: 2.4 ms in small blocks, 1.4 in large ones; 2,000 roots in rank order (R-MAT 14,
// factor 8), k = 6: 0.41 against 0.43.  At k = 3 and 4 the build is most of the work and small blocks are
// better with any number (R-MAT 12, k = 3: 99 us against 113).
// Where the counting outweighs the rows' build, two launches end in two tails: from k = 7 on (R-MAT 15,
// k = 8: 69 ms in one launch, 129 in two), and at k = 6 where sets are enumerated (a DAG that keeps ids, no
// re-encoding; R-MAT 15, ids kept, 10.9 ms against 13.9).  There the small blocks are for graphs without
// larger roots (200,000 vertices of degree 50, k = 6, ids kept: 1.8 ms against 3.5; k = 7: 1.7
// against 3.3).
constexpr uint32_t kLowSlotsPerSm = 4, kLowIds = 4;
// Under a cap on the blocks, that launch's blocks hold up to kMaxTeams teams of 8 warps, each with roots
// of its own: as many blocks of 8 warps as the cap's warps are spread over all SMs, and no block of
// 32 warps of another stream finds an empty one.  114 blocks, 180,000 roots of at most 119, k = 4..6,
// and counts of 0.13 ms on another stream: these take 4 to 21 ms at worst beside blocks of 8 warps,
// 0.25 to 1.6 ms beside teams.  (Blocks of 32 warps on one root each leave the SMs free too, but
// k = 3 on R-MAT 18 takes 1.7 ms with them, 1.3 with teams.)
constexpr int kMaxTeams = 4;

// ------------------------------------------------------------------------------------------
// Warp-register path (D <= 32).

// Number of R-cliques inside the warp-uniform candidate mask `cand` (bit j = j-th out-neighbour
// of the root); lane i holds row i of the local subgraph.  Adds lane-partial sums to acc.
template <int R>
__device__ __forceinline__ void small_dfs(uint32_t cand, uint32_t myrow, int lane,
                                          unsigned long long &acc)
{
    if constexpr (R == 1) {
        if (lane == 0) acc += __popc(cand);
    } else if constexpr (R == 2) {
        if ((cand >> lane) & 1) acc += __popc(cand & myrow);
    } else {
        uint32_t c = cand;
        while (c) {
            const int a = __ffs(c) - 1;
            c &= c - 1;
            const uint32_t c2 = cand & __shfl_sync(kFull, myrow, a);
            if (__popc(c2) >= R - 1) small_dfs<R - 1>(c2, myrow, lane, acc);
        }
    }
}

__device__ __forceinline__ uint32_t lower_bound_smem(const uint32_t *a, uint32_t n, uint32_t x)
{
    uint32_t lo = 0, len = n;
    while (len > 0) {
        const uint32_t half = len >> 1;
        if (a[lo + half] < x) {
            lo += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return lo;
}

// Membership of ids in a sorted list L[0..D) (the out-neighbours of a root), for the intersections
// N+(u) ∩ N+(a).  The ids of the largest `span` values below L's maximum are looked up in a bitmap
// (one load and a bit test; the place in L is the place of the word's first member plus the bits
// below), the smaller ones by binary search.  In a degree-ordered, relabelled DAG the heads of the
// paths u -> a -> y crowd at the top ranks: on R-MAT 20 97 % of them (by paths) lie in the last 2^14
// ranks below the root's largest neighbour and 99 % in the last 2^15, where a binary search took
// log2 D dependent loads.
template <typename Place>
struct Window {
    uint32_t *bits;   // bitmap words
    Place *first;     // place in L of each word's first member
    uint32_t base;    // id of bit 0
    uint32_t span;    // ids base .. base + span - 1 are in the bitmap
    uint32_t nlow;    // members below base

    __device__ __forceinline__ bool has(uint32_t y) const
    {
        const uint32_t p = y - base;
        return p < span && ((bits[p >> 5] >> (p & 31u)) & 1u);
    }
    __device__ __forceinline__ uint32_t place(uint32_t y) const
    {
        const uint32_t p = y - base;
        return first[p >> 5] + __popc(bits[p >> 5] & ((1u << (p & 31u)) - 1u));
    }
};

// ------------------------------------------------------------------------------------------
// Shared-memory bitmap path (small_max < D <= 1024).

// Per-warp view of the block's local subgraph and the warp's private scratch.
//   rows : D x RS words, row i = bits j with L[j] in N+(L[i]) (RS odd: column reads by
//          different rows fall in different banks)
//   tri  : every row only has bits above its own index (true for a DAG relabelled to ranks, whose
//          rows are sorted in the DAG order); lets the loops skip the words below an element.
//   elem : the current candidate set as a list of indices (compaction buffer)
//   cbuf : the current candidate set's words
//   lbuf : one candidate set per lane, word-major ([w * 32 + lane]), so that lanes reading
//          their own word w always hit 32 different banks

struct WarpCtx {
    const uint32_t *rows;
    uint32_t RS, W;
    bool tri;
    uint16_t *elem;
    uint32_t *cbuf;
    uint32_t *lbuf;
    uint32_t *mv;    // compress masks: 5 per candidate word, then the member prefix per word
    uint32_t *mbuf;  // compact rows, 4 words each (16-byte aligned); aliases lbuf
    uint32_t compact_max;  // largest candidate set re-encoded compactly by one warp (0 or 128) ...
    uint32_t compact3_max;  // ... and at R = 3 (as many members as its buffer holds packed rows of, up to 192)
    uint32_t pair_cap;     // uint16 entries of elem
    uint32_t *err;
};

// One lane's running count plus a set's total (the sum of the lanes is checked by warp_sum_u64).
__device__ __forceinline__ void add_acc(unsigned long long &acc, unsigned long long n, uint32_t *err)
{
    const unsigned long long t = acc + n;
    if (t < acc) set_error(err, kDevOverflow);
    acc = t;
}

// Number of DAG arcs inside the lane's own candidate set lb (words [lo, hi)): the penultimate
// level of Counting, which only adds subgraph degrees.  WORK adds the 32-bit word operations
// (AND + POPC) performed to `work`.
template <bool WORK>
__device__ __forceinline__ uint32_t lane_arcs(const WarpCtx &x, const uint32_t *lb, int lo, int hi,
                                              unsigned long long &work)
{
    uint32_t s = 0, ones = 0;
    for (int w = lo; w < hi; w++) {
        uint32_t y = lb[w * 32];
        if (WORK) work += (unsigned long long)__popc(y) * (uint32_t)(hi - (x.tri ? w : lo));
        // two members per step (the highest and the lowest bit): independent scans and loads
        while (y & (y - 1u)) {
            const uint32_t b1 = 31u - __clz(y);
            const uint32_t lbit = y & (0u - y);
            const uint32_t b2 = 31u - __clz(lbit);
            y ^= (1u << b1) | lbit;
            const uint32_t *r1 = x.rows + ((uint32_t)(w << 5) + b1) * x.RS;
            const uint32_t *r2 = x.rows + ((uint32_t)(w << 5) + b2) * x.RS;
            for (int w2 = x.tri ? w : lo; w2 < hi; w2++) {
                const uint32_t l = lb[w2 * 32];
                csa_add(ones, l & r1[w2], l & r2[w2], s);
            }
        }
        if (y) {
            const uint32_t b = (uint32_t)(w << 5) + 31u - __clz(y);
            const uint32_t *rb = x.rows + b * x.RS;
            int w2 = x.tri ? w : lo;
            for (; w2 + 1 < hi; w2 += 2) csa_add(ones, lb[w2 * 32] & rb[w2], lb[w2 * 32 + 32] & rb[w2 + 1], s);
            if (w2 < hi) s += __popc(lb[w2 * 32] & rb[w2]);
        }
    }
    return s + __popc(ones);
}

// Writes the candidate set (lane word c) to cbuf and its member indices to elem; returns the
// member count and the range [clo, chi) of its non-zero words.  The members are listed one word at
// a time, lane l taking bit l: a lane that lists its own word takes up to 32 steps.
__device__ __forceinline__ uint32_t compact(const WarpCtx &x, uint32_t c, int lane, int &clo, int &chi)
{
    if (lane < (int)x.W) x.cbuf[lane] = c;
    const uint32_t nz = __ballot_sync(kFull, c != 0);
    uint32_t total = 0;
    for (uint32_t r = nz; r; r &= r - 1) {
        const int w = __ffs(r) - 1;
        const uint32_t m = __shfl_sync(kFull, c, w);
        if ((m >> lane) & 1u) x.elem[total + __popc(m & lanemask_lt())] = (uint16_t)((w << 5) + lane);
        total += __popc(m);
    }
    clo = nz ? __ffs(nz) - 1 : 0;
    chi = nz ? 32 - __clz(nz) : 0;
    __syncwarp();
    return total;
}

// Triangular layout only (every row holds bits above its own index).  Sum over the members
// b = elem[j], j in [j0, total), that lie in the candidate words cw (broadcast-readable shared
// words) of |cw ∧ row_b|, restricted to words below hi.  Members are taken 32 at a time in
// index order; within such a round every lane loops over the same words [word(first), hi):
// rows have no bits below their own word, so the lanes whose member starts higher only add
// zeros, and the loop stays uniform (no divergence).  Consecutive members sit in different
// banks because the row stride is odd.  MASK: members outside cw contribute nothing.
template <bool MASK, bool WORK>
__device__ __forceinline__ uint32_t tri_rounds(const WarpCtx &x, const uint32_t *cw, uint32_t j0,
                                               uint32_t total, int hi, int lane,
                                               unsigned long long &work)
{
    uint32_t s = 0, ones = 0;
    const uint32_t lim = (uint32_t)hi << 5;
    for (; j0 < total; j0 += 32) {
        const uint32_t j = j0 + lane;
        const uint32_t b = j < total ? x.elem[j] : 0xffffu;
        const uint32_t first = __shfl_sync(kFull, b, 0);
        if (first >= lim) break;
        bool in = b < lim;
        if (MASK && in) in = (cw[b >> 5] >> (b & 31)) & 1;
        if (WORK && in) work += (uint32_t)(hi - (int)(b >> 5));
        const uint32_t *rb = x.rows + (in ? b : first) * x.RS;
        int w = (int)(first >> 5);
        for (; w + 1 < hi; w += 2) {
            const uint32_t r0 = in ? rb[w] : 0u, r1 = in ? rb[w + 1] : 0u;
            csa_add(ones, cw[w] & r0, cw[w + 1] & r1, s);
        }
        if (w < hi) s += __popc(cw[w] & (in ? rb[w] : 0u));
    }
    return s + __popc(ones);
}

// ---- Compact re-encoding of a candidate set ------------------------------------------------
// A candidate set with s members (listed in elem) is re-encoded as the s x s adjacency of its
// induced subgraph: bit j of row i is member j, so that the remaining levels work on ceil(s/32)
// words per set instead of the root-wide span.  Dense sets are counted on the symmetric COMPLEMENT
// (dense.cuh), the others enumerated on upper-triangular adjacency rows (cdfs below).  Sets of at
// most 128 members are handled by one warp, one uint4 per row.  Wider edge tasks that are dense are
// counted by a group of warps (wide_row); at R = 3 the others of up to 192 members take packed rows of 5
// or 6 words (below), and the rest stays on the root-wide bitmap.
//
// The line between the sides, in 64ths of a set's pairs that may be missing.  Where the sides cross
// (G(n, p), every set on either side): sets of one warp at p = 0.55 (k = 6: 183 us on either side at
// 0.5, 240 against 254 at 0.6; for k = 5 they stay within 5 % from 0.5 to 0.8), small sets of deep walks
// later, because a 4-clique form costs a few hundred instructions however small its set is (k = 8, 40
// copies of G(100, 0.5): 0.65 ms with the line at one half, 0.47 now).  Wide sets pay for the groups and
// barriers: at k = 5 packed rows are better to p = 0.77 (G(400, 0.7) 0.50 -> 0.31 ms), root-wide ones to
// 0.65; at k = 6 0.57 (G(400, 0.5) 0.77 -> 0.41); from k = 7 on, where the set's own members are walked
// first, 0.73 (G(700, 0.5) 72 -> 29 ms, G(400, 0.7) 82 -> 42).
__host__ __device__ constexpr uint32_t dense_line(int R, uint32_t s)
{
    if (s <= kNarrow) return R == 3 ? 28 : R >= 6 && s <= 32 ? 20 : 28;
    return R == 3 ? (s <= 192 ? 14 : 22) : R == 4 ? 28 : 17;
}
// Whether a set of s members of which `missing` of `pairs` pairs (all, or a sample) are not adjacent is
// counted on its complement.
template <int R>
__device__ __forceinline__ bool is_dense(uint32_t s, uint32_t missing, uint32_t pairs)
{
    return 64 * missing <= dense_line(R, s) * pairs;
}

// Compress masks and member prefix of every candidate word (lane w: word w), for the builders.
__device__ __forceinline__ void prepare_masks(const WarpCtx &x, int clo, int chi, int lane)
{
    const uint32_t m = (lane < chi && lane >= clo) ? x.cbuf[lane] : 0u;
    uint32_t mv[5];
    compress_masks(m, mv);
    const uint32_t pc = __popc(m);
    const uint32_t pre = warp_incl_scan(pc) - pc;
#pragma unroll
    for (int i = 0; i < 5; i++) x.mv[i * 32 + lane] = mv[i];
    x.mv[160 + lane] = pre;
    __syncwarp();
}

// The bits of row word `bits` at the members of candidate word w (mask m), packed to the low end.
__device__ __forceinline__ uint32_t member_bits(const WarpCtx &x, uint32_t bits, uint32_t m, int w)
{
    uint32_t mv[5];
#pragma unroll
    for (int t = 0; t < 5; t++) mv[t] = x.mv[t * 32 + w];
    return compress_with(bits, m, mv);
}

// Complement rows of the members 32a .. 32a + 31 of a set of s members (words in cbuf, members in
// elem, masks prepared, no words from chi on; triangular layout) in m32 (rows of S per chunk), from
// their own blocks on, and the mirror images below.  The packed row words are streamed: the member
// prefix of a candidate word is the same on every lane, so the words fill and leave at warp-uniform
// places.  Returns the complement's bits written by this lane (over all rounds, twice its edges).
// (Setting the missing pairs one by one in both rows instead: k = 5 on R-MAT 20 65 ms against 33.)
__device__ __forceinline__ uint32_t complement_round(const WarpCtx &x, uint32_t *m32, uint32_t S, uint32_t s, uint32_t a,
                                                     int chi, int lane)
{
    const uint32_t i0 = a << 5, i = i0 + lane;
    const uint32_t *row = x.rows + (uint32_t)x.elem[i < s ? i : s - 1] * x.RS;
    uint32_t bits = 0;
    // rows hold bits above their own member only: start at the word of the first member
    int w = (int)(x.elem[i0] >> 5);
    uint32_t ow = x.mv[160 + w] >> 5, sh = x.mv[160 + w] & 31u, cur = 0;
    for (; w < chi; w++) {
        const uint32_t m = x.cbuf[w];
        if (!m) continue;
        const uint32_t piece = member_bits(x, row[w], m, w);
        cur |= piece << sh;
        const uint32_t end = sh + __popc(m);
        if (end >= 32) {
            if (ow >= a) bits += put_block(m32, S, s, a, ow, cur, lane);
            ow++;
            cur = sh ? piece >> (32 - sh) : 0u;
        }
        sh = end & 31u;
    }
    if (sh && ow >= a) bits += put_block(m32, S, s, a, ow, cur, lane);
    return bits;
}

// Upper-triangular adjacency rows of the s <= 128 members of a set (words in cbuf, members in elem;
// triangular layout) by one warp, one uint4 per row in mbuf.  Returns this lane's arcs.
__device__ __forceinline__ uint32_t build_rows(const WarpCtx &x, uint32_t s, int clo, int chi, int lane)
{
    prepare_masks(x, clo, chi, lane);
    uint4 *M = reinterpret_cast<uint4 *>(x.mbuf);
    uint32_t arcs = 0;
    for (uint32_t i0 = 0; i0 < s; i0 += 32) {
        const uint32_t i = i0 + lane;
        const uint32_t *row = x.rows + (uint32_t)x.elem[i < s ? i : i0] * x.RS;
        uint32_t o[4] = {0, 0, 0, 0};
        // rows hold bits above their own member only: start at the word of the first member
        int w = (int)(x.elem[i0] >> 5);
        uint32_t ow = x.mv[160 + w] >> 5, sh = x.mv[160 + w] & 31u, cur = 0;
        // (the member prefix is the same on every lane: the words fill and leave at uniform places)
        auto leave = [&]() {
            if (ow == 0) o[0] = cur;
            else if (ow == 1) o[1] = cur;
            else if (ow == 2) o[2] = cur;
            else o[3] = cur;
        };
        for (; w < chi; w++) {
            const uint32_t m = x.cbuf[w];
            if (!m) continue;
            const uint32_t piece = member_bits(x, row[w], m, w);
            cur |= piece << sh;
            const uint32_t end = sh + __popc(m);
            if (end >= 32) {
                leave();
                ow++;
                cur = sh ? piece >> (32 - sh) : 0u;
            }
            sh = end & 31u;
        }
        if (sh) leave();
        if (i < s) {
            M[i] = make_uint4(o[0], o[1], o[2], o[3]);
            arcs += __popc(o[0]) + __popc(o[1]) + __popc(o[2]) + __popc(o[3]);
        }
    }
    __syncwarp();
    return arcs;
}

// mbuf from upper-triangular adjacency rows to complement rows of the s <= 128 members (a word of a
// row is read before its mirror image is written by the same lane: block rows in order).
__device__ __forceinline__ void rows_to_complement(const WarpCtx &x, uint32_t s, int lane)
{
    const uint4 *M = reinterpret_cast<const uint4 *>(x.mbuf);
    const uint32_t nblk = (s + 31) >> 5;
    for (uint32_t a = 0; a < nblk; a++) {
        const uint32_t i = (a << 5) + lane;
        const uint4 r = M[i < s ? i : s - 1];
        const uint32_t g[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (uint32_t ow = 0; ow < 4; ow++)
            if (ow >= a && ow < nblk) put_block(x.mbuf, 0, s, a, ow, g[ow], lane);
        __syncwarp();
    }
}

// Complement rows of the s <= 128 members of a set by one warp, one uint4 per row in mbuf.  Returns
// the complement's bits written by this lane (over all lanes, twice its edges).
__device__ __forceinline__ uint32_t build_complement(const WarpCtx &x, uint32_t s, int clo, int chi, int lane)
{
    prepare_masks(x, clo, chi, lane);
    uint32_t bits = 0;
    for (uint32_t a = 0; a << 5 < s; a++) bits += complement_round(x, x.mbuf, 0, s, a, chi, lane);
    __syncwarp();
    return bits;
}

// mbuf from complement rows to upper-triangular adjacency rows of the s <= 128 members.
__device__ __forceinline__ void complement_to_rows(const WarpCtx &x, uint32_t s, int lane)
{
    uint4 *M = reinterpret_cast<uint4 *>(x.mbuf);
    for (uint32_t i = lane; i < s; i += 32) {
        const uint4 h = M[i];
        uint32_t g[4] = {~h.x, ~h.y, ~h.z, ~h.w};
#pragma unroll
        for (uint32_t t = 0; t < 4; t++)
            g[t] &= word_mask(s, t) & (t > (i >> 5) ? kFull : (t == (i >> 5) ? above_bit(i & 31u) : 0u));
        M[i] = make_uint4(g[0], g[1], g[2], g[3]);
    }
    __syncwarp();
}

// Iteration mask of a leaf set: its members except the highest one.  In the triangular layout a
// member's row has no bits at or below its own index, so the highest member of a set adds no
// arc inside it and is not visited.
template <int CW>
__device__ __forceinline__ void drop_top(uint32_t (&Y)[CW])
{
    bool done = false;
#pragma unroll
    for (int q = CW - 1; q >= 0; q--) {
        if (!done && Y[q]) {
            Y[q] &= ~(0x80000000u >> __clz(Y[q]));
            done = true;
        }
    }
}

// o[q] |= lo, o[q + 1] |= hi for a warp-uniform q (the member prefix of a candidate word is the
// same on every lane): a uniform branch instead of a select per output word.
template <int NW>
__device__ __forceinline__ void place_piece(uint32_t (&o)[NW], uint32_t q, uint32_t lo, uint32_t hi)
{
#pragma unroll
    for (int t = 0; t < NW; t++) {
        if (q == (uint32_t)t) {
            o[t] |= lo;
            if (t + 1 < NW) o[t + 1] |= hi;
        }
    }
}

// Packed triangular compact rows for R = 3 sets of 129..192 members (CW = 5 or 6 words): the row
// of member i holds only its words q = i/32 .. CW-1 (the words below are zero in an
// upper-triangular sub-DAG), so 192 rows take 672 words instead of 1152 and fit the warp's
// scratch.  Rows of the members of word q start at packed_base(q) and are (CW - q) words long.
template <int CW>
__host__ __device__ constexpr uint32_t packed_base(int q)
{
    return q <= 0 ? 0u : packed_base<CW>(q - 1) + 32u * (uint32_t)(CW - (q - 1));
}

__host__ __device__ constexpr uint32_t packed_words(int cw) { return 16u * (uint32_t)(cw * (cw + 1)); }

template <int CW>
__device__ __forceinline__ void build_packed(const WarpCtx &x, uint32_t s, int clo, int chi, int lane)
{
    prepare_masks(x, clo, chi, lane);
#pragma unroll
    for (int q = 0; q < CW; q++) {
        const uint32_t i0 = (uint32_t)q * 32;
        if (i0 >= s) break;
        const uint32_t i = i0 + lane;
        const bool act = i < s;
        const uint32_t ei = act ? x.elem[i] : x.elem[i0];
        const uint32_t *row = x.rows + ei * x.RS;
        uint32_t o[CW];
#pragma unroll
        for (int t = 0; t < CW; t++) o[t] = 0;
        for (int w = (int)(x.elem[i0] >> 5); w < chi; w++) {
            const uint32_t m = x.cbuf[w];
            if (!m) continue;
            uint32_t mv[5];
#pragma unroll
            for (int t = 0; t < 5; t++) mv[t] = x.mv[t * 32 + w];
            const uint32_t pre = x.mv[160 + w];
            const uint32_t piece = compress_with(row[w], m, mv);
            const uint32_t qq = pre >> 5, sh = pre & 31;
            const uint32_t lo = piece << sh, hi = sh ? (piece >> (32 - sh)) : 0u;
            place_piece<CW>(o, qq, lo, hi);
        }
        if (act) {
            uint32_t *dst = x.mbuf + packed_base<CW>(q) + (uint32_t)lane * (CW - q);
#pragma unroll
            for (int t = q; t < CW; t++) dst[t - q] = o[t];
        }
    }
    __syncwarp();
}

// Arcs inside the lane's set D (CW words; zero below word Q2) on packed rows; Y = the members
// to visit (D without its highest member).
template <int CW, bool WORK, int Q2>
__device__ __forceinline__ void packed_leaf(const uint32_t *P, const uint32_t (&D)[CW],
                                            const uint32_t (&Y)[CW], uint32_t &ones, uint32_t &s,
                                            unsigned long long &work)
{
    if constexpr (Q2 < CW) {
        uint32_t y = Y[Q2];
        if (WORK) work += (unsigned long long)__popc(y) * (CW - Q2);
        // two members per step (the highest and the lowest), their words paired in the adder
        while (y & (y - 1u)) {
            const uint32_t j1 = 31u - __clz(y);
            const uint32_t lb = y & (0u - y);
            const uint32_t j2 = 31u - __clz(lb);
            y ^= (1u << j1) | lb;
            const uint32_t *r1 = P + packed_base<CW>(Q2) + j1 * (CW - Q2);
            const uint32_t *r2 = P + packed_base<CW>(Q2) + j2 * (CW - Q2);
#pragma unroll
            for (int w = Q2; w < CW; w++) csa_add(ones, D[w] & r1[w - Q2], D[w] & r2[w - Q2], s);
        }
        if (y) {
            const uint32_t *rj = P + packed_base<CW>(Q2) + (31u - __clz(y)) * (CW - Q2);
#pragma unroll
            for (int w = Q2; w + 1 < CW; w += 2) csa_add(ones, D[w] & rj[w - Q2], D[w + 1] & rj[w + 1 - Q2], s);
            if ((CW - Q2) & 1) s += __popc(D[CW - 1] & rj[CW - 1 - Q2]);
        }
        packed_leaf<CW, WORK, Q2 + 1>(P, D, Y, ones, s, work);
    }
}

// Triangles of a dense compact set of s members (members 0..s-1) on packed rows: lane l takes
// member 32q + l of each word q, forms D = C ∧ row and adds the arcs inside D.
template <int CW, bool WORK, int Q>
__device__ __forceinline__ void packed_r3(const uint32_t *P, uint32_t s_members, int lane,
                                          uint32_t &s, unsigned long long &work)
{
    if constexpr (Q < CW) {
        const uint32_t m = (uint32_t)Q * 32 + lane;
        if (m < s_members) {
            const uint32_t *rm = P + packed_base<CW>(Q) + (uint32_t)lane * (CW - Q);
            uint32_t D[CW];
#pragma unroll
            for (int w = 0; w < CW; w++) {
                const uint32_t cw = (uint32_t)w * 32 >= s_members ? 0u
                                    : (s_members >= (uint32_t)w * 32 + 32 ? kFull : ((1u << (s_members - w * 32)) - 1));
                D[w] = w < Q ? 0u : (cw & rm[w - Q]);
            }
            uint32_t Y[CW];
#pragma unroll
            for (int w = 0; w < CW; w++) Y[w] = D[w];
            drop_top<CW>(Y);
            uint32_t ones = 0, t = 0;
            packed_leaf<CW, WORK, Q>(P, D, Y, ones, t, work);
            s += t + __popc(ones);
        }
        packed_r3<CW, WORK, Q + 1>(P, s_members, lane, s, work);
    }
}

// Sum of popc(a[w] & b[w]) over words w in [FROM, CW).
template <int CW, int FROM>
__device__ __forceinline__ uint32_t popc_and(const uint32_t (&a)[CW], const uint4 &b)
{
    uint32_t s = 0;
    if (FROM <= 0) s += __popc(a[0] & b.x);
    if (CW > 1 && FROM <= 1) s += __popc(a[1] & b.y);
    if (CW > 2 && FROM <= 2) s += __popc(a[2] & b.z);
    if (CW > 3 && FROM <= 3) s += __popc(a[3] & b.w);
    return s;
}

template <int CW, bool TRI>
__device__ __forceinline__ void leaf_word_any(const uint4 *M, const uint32_t (&D)[CW], uint32_t y, int q2,
                                              uint32_t &ones, uint32_t &s)
{
    const uint32_t base = (uint32_t)q2 << 5;
    if (!TRI || q2 == 0) leaf_word<CW, 0>(M, D, y, base, ones, s);
    else if (q2 == 1) leaf_word<CW, (CW > 1 ? 1 : 0)>(M, D, y, base, ones, s);
    else if (q2 == 2) leaf_word<CW, (CW > 2 ? 2 : 0)>(M, D, y, base, ones, s);
    else leaf_word<CW, (CW > 3 ? 3 : 0)>(M, D, y, base, ones, s);
}

// Word q of the members' bits: for R = 2 and 3 lanes take the members of word q (lane l <->
// member 32q + l).  TRI: compact rows are upper-triangular, so a member's row (and any set
// derived from it) has no bits in words below the member's own word; those words are skipped
// at compile time.
template <int R, int CW, bool TRI, bool WORK, int Q>
__device__ __forceinline__ void cdfs_word(const uint4 *M, const uint32_t (&C)[CW], int lane,
                                          uint32_t &s, uint32_t &ones, unsigned long long &work)
{
    if constexpr (Q < CW) {
        if ((C[Q] >> lane) & 1) {
            const uint4 mi = M[Q * 32 + lane];
            if constexpr (R == 2) {
                s += popc_and<CW, TRI ? Q : 0>(C, mi);
                if (WORK) work += TRI ? CW - Q : CW;
            } else {
                uint32_t D[CW];
                D[0] = C[0] & mi.x;
                if (CW > 1) D[1] = C[1] & mi.y;
                if (CW > 2) D[2] = C[2] & mi.z;
                if (CW > 3) D[3] = C[3] & mi.w;
                uint32_t Y[CW];
#pragma unroll
                for (int w = 0; w < CW; w++) Y[w] = D[w];
                if (TRI) drop_top<CW>(Y);
#pragma unroll
                for (int q2 = TRI ? Q : 0; q2 < CW; q2++) {
                    uint32_t y = Y[q2];
                    if (WORK) work += (unsigned long long)__popc(y) * (TRI ? CW - q2 : CW);
                    leaf_word_any<CW, TRI>(M, D, y, q2, ones, s);
                }
            }
        }
        cdfs_word<R, CW, TRI, WORK, Q + 1>(M, C, lane, s, ones, work);
    }
}

// Triangles (R = 3) inside a compact set C whose members are scattered over its CW words (a set
// derived from a wider one, C ∧ row).  Member m_r (in index order) goes to lane r mod 32, so that
// every lane of a round holds a member (dealing by bit position would leave the lanes of the
// absent members idle); lane r forms D = C ∧ row(m_r) and adds the arcs inside D.
template <int CW, bool TRI, bool WORK>
__device__ __forceinline__ void cdfs3_dealt(const uint4 *M, uint16_t *elem, const uint32_t (&C)[CW], int lane,
                                            unsigned long long &acc, unsigned long long &work)
{
    uint32_t total = 0;
#pragma unroll
    for (int q = 0; q < CW; q++) {
        if ((C[q] >> lane) & 1) elem[total + __popc(C[q] & lanemask_lt())] = (uint16_t)(q * 32 + lane);
        total += __popc(C[q]);
    }
    __syncwarp();
    uint32_t s = 0, ones = 0;
    for (uint32_t r0 = 0; r0 < total; r0 += 32) {
        if (r0 + lane < total) {
            const uint32_t m = elem[r0 + lane];
            const uint4 mi = M[m];
            uint32_t D[CW];
            D[0] = C[0] & mi.x;
            if (CW > 1) D[1] = C[1] & mi.y;
            if (CW > 2) D[2] = C[2] & mi.z;
            if (CW > 3) D[3] = C[3] & mi.w;
            uint32_t Y[CW];
#pragma unroll
            for (int w = 0; w < CW; w++) Y[w] = D[w];
            if (TRI) drop_top<CW>(Y);
#pragma unroll
            for (int q2 = 0; q2 < CW; q2++) {
                uint32_t y = Y[q2];  // zero below the member's own word when TRI
                if (WORK) work += (unsigned long long)__popc(y) * (TRI ? CW - q2 : CW);
                leaf_word_any<CW, TRI>(M, D, y, q2, ones, s);
            }
        }
    }
    acc += s + __popc(ones);
    __syncwarp();
}

// R-cliques inside the compact set C (CW words, the same on every lane) on rows M.
template <int R, int CW, bool TRI, bool WORK>
__device__ __forceinline__ void cdfs(const uint4 *M, uint16_t *elem, const uint32_t (&C)[CW], int lane,
                                     unsigned long long &acc, unsigned long long &work)
{
    if constexpr (R == 1) {
        if (lane == 0) {
            uint32_t t = 0;
#pragma unroll
            for (int q = 0; q < CW; q++) t += __popc(C[q]);
            acc += t;
        }
    } else if constexpr (R == 2 || R == 3) {
        uint32_t s = 0, ones = 0;
        cdfs_word<R, CW, TRI, WORK, 0>(M, C, lane, s, ones, work);
        acc += s + __popc(ones);
    } else {
        // members in order; one recursive call site per level keeps the code linear in R
        uint32_t rem[CW];
#pragma unroll
        for (int t = 0; t < CW; t++) rem[t] = C[t];
        for (;;) {
            int q = -1;
            uint32_t word = 0;
#pragma unroll
            for (int t = CW - 1; t >= 0; t--)
                if (rem[t]) {
                    q = t;
                    word = rem[t];
                }
            if (q < 0) break;
            const uint32_t i = (uint32_t)(q << 5) + __ffs(word) - 1;
#pragma unroll
            for (int t = 0; t < CW; t++)
                if (t == q) rem[t] &= rem[t] - 1;
            const uint4 mi = M[i];
            uint32_t C2[CW];
            C2[0] = C[0] & mi.x;
            if (CW > 1) C2[1] = C[1] & mi.y;
            if (CW > 2) C2[2] = C[2] & mi.z;
            if (CW > 3) C2[3] = C[3] & mi.w;
            uint32_t cnt = 0;
#pragma unroll
            for (int t = 0; t < CW; t++) cnt += __popc(C2[t]);
            if (WORK && lane == 0) work += CW;
            if (cnt >= R - 1) {
                if constexpr (R == 4) cdfs3_dealt<CW, TRI, WORK>(M, elem, C2, lane, acc, work);
                else cdfs<R - 1, CW, TRI, WORK>(M, elem, C2, lane, acc, work);
            }
        }
    }
}

// 4-cliques of a dense compact set of s members (upper-triangular rows M): every arc (i, j) of
// the set is a pair queued in elem (i << 8 | j), and the queue is worked 32 pairs at a time, lane
// p forming D = M[i] ∧ M[j] and adding the arcs inside D.  Dealing the members of each C ∧ M[i]
// on its own leaves the lanes above |C ∧ M[i]| idle; pairs of many i fill every lane.
template <int CW, bool WORK>
__device__ __forceinline__ void cdfs4_pairs(const uint4 *M, uint16_t *pairs, uint32_t s, uint32_t cap, int lane,
                                            unsigned long long &acc, unsigned long long &work)
{
    uint32_t sum = 0, ones = 0, n = 0;
    auto drain = [&]() {
        __syncwarp();
        for (uint32_t r0 = 0; r0 < n; r0 += 32) {
            if (r0 + lane < n) {
                const uint32_t p = pairs[r0 + lane];
                const uint4 mi = M[p >> 8], mj = M[p & 255u];
                uint32_t D[CW];
                D[0] = mi.x & mj.x;
                if (CW > 1) D[1] = mi.y & mj.y;
                if (CW > 2) D[2] = mi.z & mj.z;
                if (CW > 3) D[3] = mi.w & mj.w;
                uint32_t Y[CW];
#pragma unroll
                for (int w = 0; w < CW; w++) Y[w] = D[w];
                drop_top<CW>(Y);
#pragma unroll
                for (int q2 = 0; q2 < CW; q2++) {
                    uint32_t y = Y[q2];
                    if (WORK) work += (unsigned long long)__popc(y) * (CW - q2);
                    leaf_word_any<CW, true>(M, D, y, q2, ones, sum);
                }
            }
        }
        __syncwarp();
        n = 0;
    };
    for (uint32_t i = 0; i + 3 < s; i++) {  // a 4-clique needs three members above i
        if (n + s > cap) drain();
        const uint4 mi = M[i];
        const uint32_t w4[4] = {mi.x, mi.y, mi.z, mi.w};
        if (WORK && lane == 0) work += CW;
        uint32_t cnt = 0;
#pragma unroll
        for (int q = 0; q < CW; q++) cnt += __popc(w4[q]);
        if (cnt < 3) continue;  // prune: fewer than three members above i
#pragma unroll
        for (int q = 0; q < CW; q++) {
            const uint32_t m = w4[q];
            if ((m >> lane) & 1) pairs[n + __popc(m & lanemask_lt())] = (uint16_t)((i << 8) | (uint32_t)(q * 32 + lane));
            n += __popc(m);
        }
    }
    drain();
    acc += sum + __popc(ones);
}

template <int R, int CW, bool TRI, bool WORK>
__device__ __forceinline__ void cdfs_all(const uint4 *M, uint16_t *elem, uint32_t cap, uint32_t s, int lane,
                                         unsigned long long &acc, unsigned long long &work)
{
    uint32_t C[CW];
#pragma unroll
    for (int q = 0; q < CW; q++) {
        const uint32_t lo = q * 32;
        C[q] = s >= lo + 32 ? kFull : (s > lo ? ((1u << (s - lo)) - 1) : 0u);
    }
    if constexpr (R == 4 && TRI) cdfs4_pairs<CW, WORK>(M, elem, s, cap, lane, acc, work);
    else cdfs<R, CW, TRI, WORK>(M, elem, C, lane, acc, work);
}

// A compact set's complement rows (chunk-major, dense.cuh): S rows per chunk, nch chunks.
struct CompSet {
    uint32_t *m32;
    uint32_t S, nch;
};

// Lane word of (set c) ∧ (members adjacent to b, above b); c has its words on the lanes below 4 nch.
__device__ __forceinline__ uint32_t adjacent_above(const CompSet &cs, uint32_t c, uint32_t b, int lane)
{
    if ((uint32_t)lane < (b >> 5) || (uint32_t)lane >= cs.nch * 4) return 0u;
    const uint32_t r = c & ~comp_word(cs.m32, cs.S, b, lane);
    return (uint32_t)lane == (b >> 5) ? r & above_bit(b & 31u) : r;
}

struct LaneSums {
    unsigned long long acc, work;
};

template <int R, int CW, bool WORK>
__device__ __noinline__ LaneSums packed_dfs(const WarpCtx x, uint32_t *m32, uint32_t s, int lane);

// R-cliques (R >= 4) of the compact set c (lane word) on complement rows: warp-uniform walk over
// the members down to R = 4, which is counted in one step.  CW: words of the sets (1..4), or 0 for
// a wide set.  Totals are added on lane 0.
template <int R, int CW, bool WORK>
__device__ __forceinline__ void dense_dfs(const WarpCtx &x, const CompSet &cs, uint32_t c, uint32_t cnt, int lane,
                                          unsigned long long &acc, unsigned long long &work)
{
    if constexpr (R == 4) {
        uint32_t *Bs = x.cbuf;
        __syncwarp();
        Bs[lane] = c;
        __syncwarp();
        const uint4 *M = reinterpret_cast<const uint4 *>(cs.m32);
        if constexpr (CW > 0) {
            const CompCount o = comp4<CW, WORK>(M, Bs, cnt, x.mv, lane);
            if (lane == 0) add_acc(acc, o.n, x.err);
            if (WORK && lane == 0) work += o.work;
        } else {
            const uint32_t ng = 32 - __clz(__ballot_sync(kFull, c != 0));
            CompSums o = comp4_wide<WORK>(M, cs.S, cs.nch, Bs, cnt, ng, 0, 1, x.mv, lane);
            if (WORK) work += o.work;
            unsigned long long n = 0;
            if (__any_sync(kFull, o.over)) {
                // a complement degree beyond the planes: one level further down
                for (uint32_t b = 0; b < ng * 32; b++) {
                    if (!((__shfl_sync(kFull, c, b >> 5) >> (b & 31u)) & 1u)) continue;
                    const uint32_t nc = adjacent_above(cs, c, b, lane);
                    const uint32_t m = __reduce_add_sync(kFull, __popc(nc));
                    if (m < 3) continue;
                    __syncwarp();
                    Bs[lane] = nc;
                    __syncwarp();
                    const CompCount t = comp3_wide<WORK>(M, cs.S, cs.nch, Bs, m, ng, 0, 1, lane);
                    if (WORK) work += t.work;
                    n += n3_finish(m, __reduce_add_sync(kFull, t.n));
                }
            } else {
                unsigned long long sl = o.sl;
#pragma unroll
                for (int k = 16; k > 0; k >>= 1) sl += __shfl_xor_sync(kFull, sl, k);
                n = n4_finish(cnt, __reduce_add_sync(kFull, o.sd), __reduce_add_sync(kFull, o.st), sl);
            }
            if (lane == 0) add_acc(acc, n, x.err);
        }
    } else {
        uint32_t rem = c;
        for (;;) {
            const uint32_t nz = __ballot_sync(kFull, rem != 0);
            if (!nz) break;
            const int wl = __ffs(nz) - 1;
            const uint32_t word = __shfl_sync(kFull, rem, wl);
            const uint32_t b = wl * 32 + __ffs(word) - 1;
            if (lane == wl) rem &= rem - 1;
            const uint32_t nc = adjacent_above(cs, c, b, lane);
            if (WORK && (uint32_t)lane < cs.nch * 4) work += 1;
            const uint32_t m = __reduce_add_sync(kFull, __popc(nc));
            if (m < R - 1) continue;
            if constexpr (R >= 6 && (CW == 4 || CW == 2)) {
                // two or more levels to go on a set that fits fewer words: packed first, so that
                // the R = 4 sets below have their lanes full (k = 8 on R-MAT 15: 69 -> 55 ms)
                if (m <= 16 * CW) {
                    uint32_t *sub = x.mbuf + kNarrow * 4 + (CW == 4 ? 0 : 256);
                    pack_subset<CW>(reinterpret_cast<const uint4 *>(cs.m32), nc, m, x.mv, sub, lane);
                    LaneSums o;
                    if (CW == 2 || m <= 32) o = packed_dfs<R - 1, 1, WORK>(x, sub, m, lane);
                    else o = packed_dfs<R - 1, 2, WORK>(x, sub, m, lane);
                    if (lane == 0) add_acc(acc, o.acc, x.err);
                    if (WORK) work += o.work;
                    continue;
                }
            }
            dense_dfs<R - 1, CW, WORK>(x, cs, nc, m, lane, acc, work);
        }
    }
}

// dense_dfs on a whole set of s members packed by pack_subset (the count on lane 0).
template <int R, int CW, bool WORK>
__device__ __noinline__ LaneSums packed_dfs(const WarpCtx x, uint32_t *m32, uint32_t s, int lane)
{
    LaneSums o = {0, 0};
    const CompSet cs = {m32, 0, 1};
    dense_dfs<R, CW, WORK>(x, cs, word_mask(s, lane), s, lane, o.acc, o.work);
    return o;
}

// C(s, R) for s <= 128 and R <= 10 (below 2^48).
template <int R>
__device__ __forceinline__ unsigned long long choose(uint32_t s)
{
    unsigned long long v = 1;
#pragma unroll
    for (uint32_t i = 0; i < (uint32_t)R; i++) v = v * (s - i) / (i + 1);
    return v;
}

// A set that is not dense, on its rows in mbuf.  Out of line: the sets of a dense core's edge tasks are
// seldom sparse, and the code would push the others' out of the instruction cache.
template <int R, int CW, bool WORK>
__device__ __noinline__ LaneSums sparse_count(const uint4 *M, uint16_t *elem, uint32_t cap, uint32_t s, int lane)
{
    LaneSums o = {0, 0};
    cdfs_all<R, CW, true, WORK>(M, elem, cap, s, lane, o.acc, o.work);
    return o;
}

// Counts a set of s members with CW words: its complement rows are in mbuf.
template <int R, int CW, bool WORK>
__device__ __forceinline__ void compact_count(const WarpCtx &x, uint32_t s, int lane, unsigned long long &acc,
                                              unsigned long long &work)
{
    if constexpr (R == 3) {
        x.cbuf[lane] = word_mask(s, lane);
        __syncwarp();
        const CompCount o = comp3<CW, WORK>(reinterpret_cast<const uint4 *>(x.mbuf), x.cbuf, s, lane);
        if (lane == 0) add_acc(acc, o.n, x.err);
        if (WORK && lane == 0) work += o.work;
    } else {
        const CompSet cs = {x.mbuf, 0, 1};
        dense_dfs<R, CW, WORK>(x, cs, word_mask(s, lane), s, lane, acc, work);
    }
}

// Triangles of a set of 129..192 members (lane word c) on packed rows.
template <bool WORK>
__device__ __forceinline__ LaneSums packed_count(const WarpCtx &x, uint32_t s, int clo, int chi, int lane)
{
    LaneSums o = {0, 0};
    uint32_t t = 0;
    if (s <= 160) {
        build_packed<5>(x, s, clo, chi, lane);
        packed_r3<5, WORK, 0>(x.mbuf, s, lane, t, o.work);
    } else {
        build_packed<6>(x, s, clo, chi, lane);
        packed_r3<6, WORK, 0>(x.mbuf, s, lane, t, o.work);
    }
    o.acc = t;
    return o;
}

// packed_count out of line, for the walks of k >= 6 (their kernels are short of registers).
template <bool WORK>
__device__ __noinline__ LaneSums packed_call(const WarpCtx x, uint32_t s, int clo, int chi, int lane)
{
    return packed_count<WORK>(x, s, clo, chi, lane);
}

// Entry for a candidate set of at most compact_max members (R = 3: compact3_max; lane word c),
// triangular layout.  TASK: the set is an edge task's.
template <int R, bool WORK, bool TASK>
__device__ __forceinline__ void compact_entry(const WarpCtx &x, uint32_t c, int lane,
                                              unsigned long long &acc, unsigned long long &work)
{
    int clo, chi;
    const uint32_t s = compact(x, c, lane, clo, chi);
    if (R == 3 && s > kNarrow) {
        const LaneSums o = TASK ? packed_count<WORK>(x, s, clo, chi, lane) : packed_call<WORK>(x, s, clo, chi, lane);
        acc += o.acc;
        if (WORK) work += o.work;
    } else if (s >= (uint32_t)R) {
        // An edge task's own set at k = 5 is packed as it is and mirrored when it is dense; deeper
        // walks pack the complement and turn it back when it is not.
        constexpr bool kRowsFirst = R == 3 && TASK;
        const uint32_t pairs = s * (s - 1) / 2;
        const uint32_t missing =
            kRowsFirst ? pairs - __reduce_add_sync(kFull, build_rows(x, s, clo, chi, lane))
                       : __reduce_add_sync(kFull, build_complement(x, s, clo, chi, lane)) / 2;
        if (!is_dense<R>(s, missing, pairs)) {
            if (!kRowsFirst) complement_to_rows(x, s, lane);
            const uint4 *M = reinterpret_cast<const uint4 *>(x.mbuf);
            const LaneSums o = s <= 32   ? sparse_count<R, 1, WORK>(M, x.elem, x.pair_cap, s, lane)
                               : s <= 64 ? sparse_count<R, 2, WORK>(M, x.elem, x.pair_cap, s, lane)
                               : s <= 96 ? sparse_count<R, 3, WORK>(M, x.elem, x.pair_cap, s, lane)
                                         : sparse_count<R, 4, WORK>(M, x.elem, x.pair_cap, s, lane);
            acc += o.acc;
            if (WORK) work += o.work;
        } else if (missing == 0) {  // a clique
            if (lane == 0) add_acc(acc, choose<R>(s), x.err);
        } else {
            if (kRowsFirst) rows_to_complement(x, s, lane);
            if (s <= 32) compact_count<R, 1, WORK>(x, s, lane, acc, work);
            else if (s <= 64) compact_count<R, 2, WORK>(x, s, lane, acc, work);
            else compact_count<R, 4, WORK>(x, s, lane, acc, work);
        }
    }
    __syncwarp();
}

// Counts the R-cliques inside the candidate set whose word w sits in lane w (words >= W are
// zero); adds lane-partial sums to acc.
//   R >= 3, triangular layout, at most compact_max (R = 3: compact3_max) members: re-encoded
//           compactly (compact_entry) and finished on the compact rows.
//   R >= 4: warp-uniform walk over the members a; the next candidate set c ∧ row_a is again
//           spread over the lanes (one shared-memory load per lane).
//   R == 3: members are compacted and dealt to lanes; each lane builds its own c ∧ row_a and
//           sums its arcs (the last two levels run lane-parallel).
//   R == 2: members dealt to lanes, each adds |c ∧ row_a|.
template <int R, bool WORK, bool TASK = false>
__device__ __forceinline__ void warp_dfs(const WarpCtx &x, uint32_t c, int lane,
                                         unsigned long long &acc, unsigned long long &work)
{
    if constexpr (R >= 3) {
        if (x.tri && __reduce_add_sync(kFull, __popc(c)) <= (R == 3 ? x.compact3_max : x.compact_max)) {
            compact_entry<R, WORK, TASK>(x, c, lane, acc, work);
            return;
        }
    }
    if constexpr (R == 1) {
        acc += __popc(c);
    } else if constexpr (R == 2) {
        const uint32_t nz = __ballot_sync(kFull, c != 0);
        if (__popc(nz) <= 4) {
            // few words: lane l takes bit l of each non-zero word in turn
            if (lane < (int)x.W) x.cbuf[lane] = c;
            __syncwarp();
            const int chi = 32 - __clz(nz);
            uint32_t outer = nz, s = 0;
            while (outer) {
                const int w = __ffs(outer) - 1;
                outer &= outer - 1;
                const uint32_t cw = x.cbuf[w];
                if ((cw >> lane) & 1) {
                    const uint32_t *ra = x.rows + (uint32_t)(w * 32 + lane) * x.RS;
                    const int w0 = x.tri ? w : (__ffs(nz) - 1);
                    if (WORK) work += (uint32_t)(chi - w0);
                    for (int w2 = w0; w2 < chi; w2++) s += __popc(x.cbuf[w2] & ra[w2]);
                }
            }
            acc += s;
            __syncwarp();
        } else if (x.tri) {
            int clo, chi;
            const uint32_t total = compact(x, c, lane, clo, chi);
            acc += tri_rounds<false, WORK>(x, x.cbuf, 0, total, chi, lane, work);
            __syncwarp();
        } else {
            int clo, chi;
            const uint32_t total = compact(x, c, lane, clo, chi);
            uint32_t s = 0;
            for (uint32_t i = lane; i < total; i += 32) {
                const uint32_t a = x.elem[i];
                const uint32_t *ra = x.rows + a * x.RS;
                const int w0 = x.tri ? (int)(a >> 5) : clo;
                if (WORK) work += (uint32_t)(chi - w0);
                for (int w = w0; w < chi; w++) s += __popc(x.cbuf[w] & ra[w]);
            }
            acc += s;
            __syncwarp();
        }
    } else if constexpr (R == 3) {
        int clo, chi;
        const uint32_t total = compact(x, c, lane, clo, chi);
        uint32_t *lb = x.lbuf + lane;
        for (uint32_t i = lane; i < total; i += 32) {
            const uint32_t a = x.elem[i];
            const uint32_t *ra = x.rows + a * x.RS;
            uint32_t cnt = 0;
            int nlo = 32, nhi = 0;
            const int w0 = x.tri ? (int)(a >> 5) : clo;
            if (WORK) work += (uint32_t)(chi - w0);
            for (int w = w0; w < chi; w++) {
                const uint32_t v = x.cbuf[w] & ra[w];
                lb[w * 32] = v;
                if (v) {
                    cnt += __popc(v);
                    nlo = min(nlo, w);
                    nhi = w + 1;
                }
            }
            if (cnt >= 2) acc += lane_arcs<WORK>(x, lb, nlo, nhi, work);
        }
        __syncwarp();
    } else {
        uint32_t rem = c;
        for (;;) {
            const uint32_t nz = __ballot_sync(kFull, rem != 0);
            if (!nz) break;
            const int wl = __ffs(nz) - 1;
            const uint32_t word = __shfl_sync(kFull, rem, wl);
            const uint32_t a = wl * 32 + __ffs(word) - 1;
            if (lane == wl) rem &= rem - 1;
            const uint32_t c2 = lane < (int)x.W ? (c & x.rows[a * x.RS + lane]) : 0u;
            if (WORK && lane < (int)x.W) work += 1;
            const uint32_t cnt = __reduce_add_sync(kFull, __popc(c2));
            if (cnt >= R - 1) warp_dfs<R - 1, WORK>(x, c2, lane, acc, work);
        }
    }
}

// Shared-memory words one warp needs for roots of out-degree <= dcap (dcap multiple of 32), in two
// parts: its own lists, cbuf (32) | mv (compress masks, 192) | the member list of a neighbourhood |
// elem (dcap uint16, or the rows of a neighbourhood once the set's rows are built), and its
// lbuf/mbuf, which holds compact_max rows of 4 words.  The second parts of all warps are
// consecutive, so that a group of neighbouring warps can take its members' parts as one buffer.
__host__ __device__ __forceinline__ uint32_t warp_list_words(uint32_t dcap, uint32_t compact_max)
{
    return 32 + kMaskWords + kNbhdList + (compact_max && kNbhdWords > dcap / 2 ? kNbhdWords : dcap / 2);
}
// (deep, k >= 8: also room for the rows of a subset of 64 members and of one of 32 in it)
__host__ __device__ __forceinline__ uint32_t warp_buf_words(uint32_t dcap, uint32_t compact_max, bool deep)
{
    const uint32_t m = compact_max ? compact_max * 4 + (deep ? 256 + 128 : 0) : 0u;
    return dcap > m ? dcap : m;
}

constexpr int kMidMaxWarps = 32;
constexpr uint32_t kMidStaticSmem = 2048;  // room left for the kernel's static shared memory
constexpr uint32_t kNoHelpSlot = 0xffffffffu;
constexpr uint32_t kHelpSlots = 8192;    // heavy roots that can take help, per launch
constexpr uint32_t kUnitMask = (1u << 21) - 1;  // units of a heavy root besides its wide rows (HeavySlot)
constexpr uint32_t kCursorEnd = 32768;   // where either wide cursor of a heavy root ends (HeavySlot)
constexpr uint32_t kSplitMembers = 128;  // heavy roots: rows above this many members are cut by member
constexpr uint32_t kMaxGroups = 15;      // pairs of warps that can head a group (named barriers 1..15)

// Words of the complement rows of a wide set of s members.
__host__ __device__ __forceinline__ uint32_t wide_words(uint32_t s) { return ((s + 127) >> 7) * s * 4; }

// Position of the r-th (from 0) set bit of x (r < popc(x)).
__device__ __forceinline__ uint32_t select_bit(uint32_t x, uint32_t r)
{
    uint32_t pos = 0;
#pragma unroll
    for (int width = 16; width > 0; width >>= 1) {
        const uint32_t low = __popc(x & ((1u << width) - 1u));
        if (r >= low) {
            r -= low;
            x >>= width;
            pos += width;
        }
    }
    return pos;
}

// Warp 0: the published heavy root with the most units left (kNoHelpSlot when none has any).
__device__ __forceinline__ uint32_t pick_help_slot(const HelpTable &ht, int lane)
{
    const uint32_t ns = min(*(volatile uint32_t *)ht.nslots, ht.cap);
    uint32_t best = kNoHelpSlot, best_rem = 0;
    for (uint32_t s0 = 0; s0 < ns; s0 += 32) {
        const uint32_t sl = s0 + lane;
        uint32_t rem = 0;
        if (sl < ns) {
            cuda::atomic_ref<uint32_t, cuda::thread_scope_device> units(ht.slots[sl].units);
            const uint32_t un = units.load(cuda::memory_order_acquire);
            const uint32_t cw = *(volatile uint32_t *)&ht.slots[sl].wide_cursor;
            const uint32_t cn = *(volatile uint32_t *)&ht.slots[sl].cursor;
            const uint32_t cb = cw & 0xffffu, cm = cw >> 16, other = un & kUnitMask;
            if (un)
                rem = (cb < kCursorEnd ? kCursorEnd - cb : 0u) + (cm < kCursorEnd ? kCursorEnd - cm : 0u) +
                      (cn < other ? other - cn : 0u);
        }
        uint32_t bsl = sl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint32_t r2 = __shfl_xor_sync(kFull, rem, o), s2 = __shfl_xor_sync(kFull, bsl, o);
            if (r2 > rem || (r2 == rem && s2 < bsl)) {
                rem = r2;
                bsl = s2;
            }
        }
        if (rem > best_rem) {
            best_rem = rem;
            best = bsl;
        }
    }
    return best;
}

// Shared state of a group of warps on a wide row.
struct GroupShared {
    unsigned long long sl;
    uint32_t unit, sd, st, next, over;
};

// A group's place: gw warps (a power of two), this warp's index gi, its named barrier.
struct Group {
    GroupShared *sh;
    uint32_t *buf;  // the members' scratch buffers as one
    uint32_t *lists;  // the first warp's lists
    uint32_t gw, gi, bar;

    __device__ __forceinline__ void sync() const
    {
        __syncwarp();
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(gw * 32u) : "memory");
    }
};

// Member number r (from 0, in index order) of a set whose word w sits in lane w.
__device__ __forceinline__ uint32_t select_member(uint32_t c, uint32_t r)
{
    const uint32_t pc = __popc(c);
    const uint32_t incl = warp_incl_scan(pc);
    const int wl = __ffs(__ballot_sync(kFull, incl > r)) - 1;
    const uint32_t before = __shfl_sync(kFull, incl - pc, wl);
    const uint32_t word = __shfl_sync(kFull, c, wl);
    return (uint32_t)wl * 32 + select_bit(word, r - before);
}

// R-cliques (R >= 3) of a dense row c (lane word, more than 128 members; triangular layout), counted by
// the warps of a group together: they build the complement rows (32 members per round), then R = 3
// and R = 4 are one pass over (32 members, chunk of 128 codegrees) units, and for R >= 5 the warps
// take the members one at a time and walk down from there.  Every warp of the group calls this.
// k = 5 (R = 3), k_count_mid: R-MAT 20 32.8 ms, Chung-Lu 4M 120.1 ms when every warp made the lists for
// itself, the rows were built 32 x 32 block by block and each pair of a triangle's edges was seen
// twice; 32.0 and 114.3 with the pairs seen once and sets sparser than one half counted as they
// are; 30.9 and 107.0 with shared lists and whole rounds.
template <int R, bool WORK>
__device__ __forceinline__ void wide_row(const WarpCtx &x, const Group &g, uint32_t c, int lane,
                                         unsigned long long &acc, unsigned long long &work)
{
    // the set's lists are made once, in the first warp's scratch: its words and masks by that warp,
    // the members by all
    WarpCtx y = x;
    y.cbuf = g.lists;
    y.mv = g.lists + 32;
    y.elem = reinterpret_cast<uint16_t *>(g.lists + 32 + kMaskWords + kNbhdList);
    const uint32_t nz = __ballot_sync(kFull, c != 0);
    const int chi = 32 - __clz(nz);
    const uint32_t pc = __popc(c), incl = warp_incl_scan(pc), s = __shfl_sync(kFull, incl, 31);
    if (g.gi == 0) {
        uint32_t mv[5];
        compress_masks(c, mv);
        y.cbuf[lane] = c;
#pragma unroll
        for (int i = 0; i < 5; i++) y.mv[i * 32 + lane] = mv[i];
        y.mv[160 + lane] = incl - pc;
    }
    for (uint32_t rest = nz; rest; rest &= rest - 1) {
        const int w = __ffs(rest) - 1;
        const uint32_t m = __shfl_sync(kFull, c, w), at = __shfl_sync(kFull, incl - pc, w);
        if (((uint32_t)w & (g.gw - 1)) == g.gi && ((m >> lane) & 1u))
            y.elem[at + __popc(m & lanemask_lt())] = (uint16_t)((w << 5) + lane);
    }
    g.sync();
    const CompSet cs = {g.buf, s, (s + 127) >> 7};
    const uint32_t nblk = (s + 31) >> 5;
    // rounds get shorter: dealt forth and back
    for (uint32_t a = 0; a < nblk; a++) {
        const uint32_t p = a & (g.gw - 1);
        if ((a & g.gw ? g.gw - 1 - p : p) == g.gi) complement_round(y, cs.m32, s, s, a, chi, lane);
    }
    g.sync();
    x.cbuf[lane] = word_mask(s, lane);
    __syncwarp();
    const uint4 *M = reinterpret_cast<const uint4 *>(cs.m32);
    bool counted = false;
    if constexpr (R == 3) {
        CompCount o = comp3_wide<WORK>(M, s, cs.nch, x.cbuf, s, nblk, g.gi, g.gw, lane);
        if (WORK) work += o.work;
        o.n = __reduce_add_sync(kFull, o.n);
        if (lane == 0) atomicAdd(&g.sh->sd, o.n);
        g.sync();
        if (g.gi == 0 && lane == 0) add_acc(acc, n3_finish(s, g.sh->sd), x.err);
        counted = true;
    } else if constexpr (R == 4) {
        CompSums o = comp4_wide<WORK>(M, s, cs.nch, x.cbuf, s, nblk, g.gi, g.gw, x.mv, lane);
        if (WORK) work += o.work;
        const bool over = __any_sync(kFull, o.over);
        o.sd = __reduce_add_sync(kFull, o.sd);
        o.st = __reduce_add_sync(kFull, o.st);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) o.sl += __shfl_xor_sync(kFull, o.sl, k);
        if (lane == 0) {
            if (over) atomicOr(&g.sh->over, 1u);
            atomicAdd(&g.sh->sd, o.sd);
            atomicAdd(&g.sh->st, o.st);
            atomicAdd(&g.sh->sl, o.sl);
        }
        g.sync();
        counted = !g.sh->over;
        if (counted && g.gi == 0 && lane == 0)
            add_acc(acc, n4_finish(s, g.sh->sd, g.sh->st, g.sh->sl), x.err);
    }
    if constexpr (R >= 4) {
        while (!counted) {  // member by member
            uint32_t r = 0;
            if (lane == 0) r = atomicAdd(&g.sh->next, 1u);
            r = __shfl_sync(kFull, r, 0);
            if (r >= s) break;
            const uint32_t nc = adjacent_above(cs, word_mask(s, lane), r, lane);
            const uint32_t m = __reduce_add_sync(kFull, __popc(nc));
            if (m < R - 1) continue;
            if constexpr (R == 4) {
                __syncwarp();
                x.cbuf[lane] = nc;
                __syncwarp();
                const CompCount o = comp3_wide<WORK>(M, s, cs.nch, x.cbuf, m, nblk, 0, 1, lane);
                if (WORK) work += o.work;
                const uint32_t sum = __reduce_add_sync(kFull, o.n);
                if (lane == 0) add_acc(acc, n3_finish(m, sum), x.err);
            } else {
                dense_dfs<R - 1, 0, WORK>(x, cs, nc, m, lane, acc, work);
            }
        }
    }
}

// Whether the set of m > 128 members whose word w sits in lane w (triangular layout) is dense enough
// for a group of warps: the arcs above 32 of its members, spread evenly, against the line.
template <int R>
__device__ __noinline__ bool wide_dense(const uint32_t *rows, uint32_t RS, uint32_t c, uint32_t m, int lane)
{
    // member r of the set in lane l: the word in which r falls (binary search over the lanes' prefix
    // sums), then the bit
    const uint32_t r = (uint32_t)lane * m >> 5, pc = __popc(c), excl = warp_incl_scan(pc) - pc;
    uint32_t o = 0;
#pragma unroll
    for (uint32_t step = 16; step > 0; step >>= 1) {
        const uint32_t e = __shfl_sync(kFull, excl, (o + step) & 31u);
        if (e <= r) o += step;
    }
    // (empty words share their prefix with the next: the search ends at the last of them, which holds r)
    const uint32_t word = __shfl_sync(kFull, c, o), before = __shfl_sync(kFull, excl, o);
    const uint32_t *row = rows + (o * 32 + select_bit(word, r - before)) * RS;
    uint32_t arcs = 0;
    for (uint32_t nz = __ballot_sync(kFull, c != 0); nz; nz &= nz - 1) {
        const int w = __ffs(nz) - 1;
        arcs += __popc(__shfl_sync(kFull, c, w) & row[w]);
    }
    const uint32_t pairs = __reduce_add_sync(kFull, m - 1 - r);
    return is_dense<R>(m, pairs - __reduce_add_sync(kFull, arcs), pairs);
}

// Bitmap path (small_max < D <= dcap): one block (or one of its `teams`) per root, roots taken largest-D first from the
// queue.  The block builds the root's local subgraph as D x D bitmap rows in shared memory
// (row i = V(g_u) ∩ N+(a_i), Algorithm GenSub-CITRON by sorted-list intersection) and its warps
// count the (K-2)-cliques of every row: the edge tasks (u, a_t).
//   K >= 5, triangular layout: dense rows of more than 128 members (wide rows) are counted first, each
//       by a group of warps whose scratch buffers together hold its complement rows: as many warps
//       as the root's widest row needs for the rows that two warps cannot hold, then two warps each;
//       the other rows by one warp each.
//   D < split_min: the rows are taken from counters in shared memory, and cut like a heavy root's where
//       there are sparse ones of more than kSplitMembers members.
//   D >= split_min (heavy roots, K >= 6): the wide rows and the units of the others are taken from
//       cursors in a global table; a unit is an edge task or, in a row of more than kSplitMembers
//       members that is not wide (sparse rows, general DAGs, no re-encoding), the sub-task (u, a_t, b) of one
//       member b: the (K-3)-cliques of row_t ∧ row_b.  Blocks that find the root queue empty pick the
//       published heavy root with the most units left, rebuild its rows and take from the same
//       cursors (work stealing across blocks); every block adds its own part of the root's count.
//       (One root of 800, k = 6, ids kept: 49 ms when whole rows were its units, 15 ms by member.)
// block_ns (optional): each block's start and end on the global timer.
// TEAMED: the block is `team_count` teams instead of one (an instance of its own: the plain kernel has no
// registers to spare).
template <int K, bool WORK, bool TEAMED>
__global__ __launch_bounds__(kMidMaxWarps * 32, 1) void k_count_mid(
    const uint64_t *__restrict__ dag_off, const uint32_t *__restrict__ dag_cols,
    const uint32_t *__restrict__ list, const CountStats *st, uint32_t *next, int low, int team_count, uint32_t dcap,
    uint32_t team_words, uint32_t buf_words, uint32_t window, uint32_t compact_max, uint32_t split_min, HelpTable ht,
    unsigned long long *result, RootSink sink, unsigned long long *work_out, unsigned long long *block_ns, Budget budget,
    uint32_t *err)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const uint32_t rs_cap = (dcap / 32) | 1;
    // this team: nw warps, of which this is number w (wb in the block); tx its thread
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
    const int nw = TEAMED ? (int)(blockDim.x >> 5) / team_count : (int)(blockDim.x >> 5);
    const int team = TEAMED ? wb / nw : 0, w = TEAMED ? wb - team * nw : wb;
    const uint32_t tx = TEAMED ? (uint32_t)w * 32 + lane : threadIdx.x, tn = TEAMED ? (uint32_t)nw * 32 : blockDim.x;
    auto sync = [&]() {
        if (!TEAMED) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(tn) : "memory");
    };
    uint32_t *sL = smem + (size_t)team * team_words;
    uint32_t *rows = sL + dcap;
    __shared__ uint32_t s_idx[kMaxTeams], s_task[kMaxTeams], s_tri[kMaxTeams], s_slot[kMaxTeams], s_u[kMaxTeams],
        s_unsorted[kMaxTeams], s_units[kMaxTeams];
    // (roots with wide rows are not counted by teams)
    __shared__ uint32_t s_wide[2], s_most, s_sparse, s_ask;
    __shared__ uint32_t s_cls[2][kBitmapCap / 32];  // wide rows of either class, one bit each
    __shared__ unsigned long long s_acc[32], s_arc[32];
    __shared__ GroupShared s_group[kMaxGroups];
    uint32_t *lists = K > 3 ? rows + (size_t)dcap * rs_cap : rows;  // k = 3 keeps no rows
    uint32_t *wscr = lists + (size_t)w * warp_list_words(dcap, compact_max);
    uint32_t *bufs = lists + (size_t)nw * warp_list_words(dcap, compact_max);
    // units before each of a heavy root's rows: it reuses sL, which is dead once the rows are built
    uint32_t *s_upre = sL;
    WarpCtx x;
    x.rows = rows;
    x.cbuf = wscr;
    x.mv = wscr + 32;
    x.elem = reinterpret_cast<uint16_t *>(wscr + 32 + kMaskWords + kNbhdList);
    x.lbuf = bufs + (size_t)w * buf_words;
    x.mbuf = x.lbuf;
    x.compact_max = compact_max;
    x.compact3_max = !compact_max ? 0u : buf_words >= packed_words(6) ? 192u : buf_words >= packed_words(5) ? 160u : 128u;
    x.pair_cap = dcap;
    x.err = err;
    // the membership window of the root being built lies over the warps' lists and buffers
    Window<uint16_t> win;
    win.bits = lists;
    win.first = reinterpret_cast<uint16_t *>(lists + window / 32);
    // this launch's part of the queue (largest out-degree first)
    const uint32_t first_root = low ? st->n_high : 0u;
    const uint32_t nlist = (low ? st->n_mid : st->n_high) - first_root;
    list += first_root;
    if (WORK && lane == 0) s_arc[wb] = 0;
    if (block_ns && threadIdx.x == 0) block_ns[2 * blockIdx.x] = global_ns();
    unsigned long long block_total = 0;  // meaningful in thread 0
    bool queue_empty = false;
    for (;;) {
        if (tx == 0) {
            s_idx[team] = queue_empty || budget.over(err) ? 0xfffffffeu : atomicAdd(next, 1u);
            s_task[team] = 0;
            s_wide[0] = s_wide[1] = 0;
            s_most = 0;
            s_sparse = 0;
            s_ask = 0;
            s_tri[team] = 1;
            s_unsorted[team] = 0;
            s_slot[team] = kNoHelpSlot;
        }
        sync();
        const uint32_t idx = s_idx[team];
        const bool owner = idx < nlist;
        if (!owner) {
            queue_empty = true;
            if (K < 6 || ht.slots == nullptr || idx == 0xfffffffeu) break;
            if (w == 0) {
                const uint32_t sl = pick_help_slot(ht, lane);
                if (lane == 0) {
                    s_slot[team] = sl;
                    if (sl != kNoHelpSlot) s_u[team] = ht.slots[sl].u;
                }
            }
            sync();
            if (s_slot[team] == kNoHelpSlot) break;
        }
        const uint32_t u = owner ? list[idx] : s_u[team];
        const uint64_t base = dag_off[u];
        const uint32_t D = (uint32_t)(dag_off[u + 1] - base);
        if (D > dcap || D == 0) {  // a root is never larger than the launch's capacity
            if (tx == 0) set_error(err, kDevBadInput);
            break;
        }
        const bool heavy = K >= 6 && (!owner || D >= split_min);
        const uint32_t W = (D + 31) >> 5, RS = W | 1;
        // the rows this warp builds (w, w + nw, ..): lane r holds the place of the r-th one's list
        const uint32_t mine = w + (uint32_t)nw * lane;
        for (uint32_t i = tx; i < D; i += tn) sL[i] = dag_cols[base + i];
        if (K > 3)
            for (uint32_t i = tx; i < D * RS; i += tn) rows[i] = 0;
        for (uint32_t i = tx; i < window / 32; i += tn) win.bits[i] = 0;
        sync();
        const uint32_t lmax = sL[D - 1];
        win.base = lmax >= window ? lmax - (window - 1) : 0u;
        win.span = lmax - win.base + 1;
        uint64_t rb = 0;
        uint32_t rlen = 0;
        if (mine < D) {
            const uint32_t a = sL[mine];
            rb = dag_off[a];
            rlen = (uint32_t)(dag_off[a + 1] - rb);
        }
        for (uint32_t i = tx; i < D; i += tn) {
            const uint32_t v = sL[i], prev = i ? sL[i - 1] : 0u;
            // the window's places hold for ascending members only, and an id above the last one's
            // would lie beyond its bitmap
            if (v < prev || v > lmax) s_unsorted[team] = 1;
            else if (v >= win.base) {
                const uint32_t p = v - win.base;
                atomicOr(&win.bits[p >> 5], 1u << (p & 31u));
                if (K > 3 && (i == 0 || prev < win.base || ((prev - win.base) >> 5) != (p >> 5)))
                    win.first[p >> 5] = (uint16_t)i;
            }
        }
        sync();
        if (s_unsorted[team]) {  // the DAG's rows have to be sorted
            if (tx == 0) set_error(err, kDevBadInput);
            break;
        }
        win.nlow = win.base ? lower_bound_smem(sL, D, win.base) : 0u;
        unsigned long long acc = 0, work = 0;
        // Build the local subgraph: row i = V(g_u) ∩ N+(a_i) (CITRON's GenSubgraph).  Each step
        // loads 128 entries of N+(a_i), four per lane in flight.  An entry found sets its bit with a
        // shared-memory atomic: gathering a step's words by ballots first cost 2.5 ms more (k = 4 on
        // R-MAT 20: 10.4 against 7.9 ms), for a few hits per step.  (A block helping with a heavy
        // root rebuilds the same rows; its triangles are not counted here.)
        bool tri = true;
        for (uint32_t i = w, r = 0; i < D; i += nw, r++) {
            if (r == 32) {  // more rows than lanes: the places of the next 32
                r = 0;
                rb = 0;
                rlen = 0;
                if (i + (uint32_t)nw * lane < D) {
                    const uint32_t a = sL[i + (uint32_t)nw * lane];
                    rb = dag_off[a];
                    rlen = (uint32_t)(dag_off[a + 1] - rb);
                }
            }
            const uint64_t b = __shfl_sync(kFull, rb, r);
            const uint32_t len = __shfl_sync(kFull, rlen, r);
            for (uint32_t p = 0; p < len; p += 128) {
                uint32_t y[4];
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    const uint32_t q = p + 32 * h + lane;
                    y[h] = q < len ? dag_cols[b + q] : 0xffffffffu;
                }
                if (__shfl_sync(kFull, y[0], 0) > lmax) break;
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    bool hit = win.has(y[h]);
                    uint32_t j = 0;
                    if (K > 3 && hit) j = win.place(y[h]);
                    if (win.nlow && y[h] < win.base) {
                        j = lower_bound_smem(sL, win.nlow, y[h]);
                        hit = j < win.nlow && sL[j] == y[h];
                    }
                    if (K == 3) {
                        acc += hit;
                        if (WORK && sink.per_arc && hit) atomicAdd(&sink.per_arc[base + i], 1ull);
                    } else {
                        tri &= !hit || j > i;
                        if (hit) atomicOr(&rows[i * RS + (j >> 5)], 1u << (j & 31u));
                    }
                }
            }
        }
        if (K > 3) {
            if (!__all_sync(kFull, tri) && lane == 0) s_tri[team] = 0;
            sync();
            x.RS = RS;
            x.W = W;
            x.tri = s_tri[team] != 0;
            // Wide rows: those that need more than two warps' buffers, then the other ones.  A root of
            // at most 129 out-neighbours has none.
            uint32_t nbig = 0, nmid = 0, units = D;
            const uint32_t most_gw = 1u << (31 - __clz(nw));  // warps of the largest group
            if constexpr (K >= 5) {
                if (x.tri && compact_max && D > kNarrow + 1) {
                    for (uint32_t q = w; q < W; q += nw) {
                        const uint32_t t = q * 32 + lane;
                        uint32_t m = 0;
                        if (t < D)
                            for (uint32_t v = q; v < W; v++) m += __popc(rows[t * RS + v]);
                        // a row too wide for the block's buffers, or sparse, is left to one warp
                        const bool fits = m > kNarrow && nw > 1 && wide_words(m) <= buf_words * most_gw;
                        const uint32_t ask = __ballot_sync(kFull, fits);
                        if (lane == 0) {
                            s_cls[0][q] = ask;
                            s_cls[1][q] = 0;
                            if (ask) s_ask = 1;
                        }
                    }
                    sync();
                    if (s_ask) {
                        for (uint32_t t = w; t < D; t += nw) {
                            if (!((*(volatile uint32_t *)&s_cls[0][t >> 5] >> (t & 31u)) & 1u)) continue;
                            const uint32_t c = lane < W ? rows[t * RS + lane] : 0u;
                            const uint32_t m = __reduce_add_sync(kFull, __popc(c));
                            const bool dense = wide_dense<K - 2>(rows, RS, c, m, lane);
                            const bool big = wide_words(m) > buf_words * 2;
                            if (lane == 0) {
                                if (!dense || !big) atomicAnd(&s_cls[0][t >> 5], ~(1u << (t & 31u)));
                                if (dense && !big) atomicOr(&s_cls[1][t >> 5], 1u << (t & 31u));
                                if (dense) atomicMax(&s_most, m);
                                else s_sparse = 1;
                            }
                        }
                        sync();
                        for (uint32_t q = 0; q < W; q++) {
                            nbig += __popc(s_cls[0][q]);
                            nmid += __popc(s_cls[1][q]);
                        }
                    }
                }
            }
            const uint32_t nwide = nbig + nmid;
            auto is_wide = [&](uint32_t t) { return ((s_cls[0][t >> 5] | s_cls[1][t >> 5]) >> (t & 31u)) & 1u; };
            const bool cut = heavy || (K >= 6 && !TEAMED && s_sparse);
            if (cut) {
                for (uint32_t t = w; t < D; t += nw) {
                    const uint32_t c = lane < W ? rows[t * RS + lane] : 0u;
                    const uint32_t m = __reduce_add_sync(kFull, __popc(c));
                    if (lane == 0)
                        s_upre[t] = m < (uint32_t)(K - 2) || (nwide && is_wide(t)) ? 0u : m > kSplitMembers ? m : 1u;
                }
                sync();
                if (w == 0) {
                    uint32_t run = 0;
                    for (uint32_t t0 = 0; t0 < D; t0 += 32) {
                        const uint32_t v = t0 + lane < D ? s_upre[t0 + lane] : 0u;
                        const uint32_t inc = warp_incl_scan(v);
                        if (t0 + lane < D) s_upre[t0 + lane] = run + inc - v;
                        run += __shfl_sync(kFull, inc, 31);
                    }
                    if (lane == 0) s_units[team] = run;
                }
                sync();
                units = s_units[team];
            }
            if (heavy) {
                if (tx == 0) {
                    const uint32_t word = 0x80000000u | (nwide << 21) | units;
                    if (owner && ht.slots) {
                        const uint32_t sl = atomicAdd(ht.nslots, 1u);
                        if (sl < ht.cap) {
                            ht.slots[sl].u = u;
                            ht.slots[sl].wide_cursor = (kCursorEnd - nmid) << 16 | (kCursorEnd - nbig);
                            cuda::atomic_ref<uint32_t, cuda::thread_scope_device> pub(ht.slots[sl].units);
                            pub.store(word, cuda::memory_order_release);
                            s_slot[team] = sl;
                        }
                    } else if (!owner && ht.slots[s_slot[team]].units != word) {
                        set_error(err, kDevBadInput);  // the rebuilt root differs from the published one
                        s_task[team] = units;          // take nothing
                        s_wide[0] = nbig;
                        s_wide[1] = nmid;
                        s_slot[team] = kNoHelpSlot;
                    }
                }
                sync();
            }
            // the units of a published heavy root are taken from its slot's cursors in global
            // memory, the others from the block's counters in shared memory
            HeavySlot *slot = s_slot[team] != kNoHelpSlot ? &ht.slots[s_slot[team]] : nullptr;
            if constexpr (K >= 5) {
                // The `count` wide rows of class cls by groups of gw warps.  A group is named by its first
                // warp (barrier and shared state), so that a warp can go on to the next class while
                // other groups are still at this one: every warp of the new group has left its old
                // group, whose last barrier it shared with the rest.
                auto run_wide = [&](int cls, uint32_t count, uint32_t gw) {
                    const uint32_t w0 = (uint32_t)w & ~(gw - 1);
                    if (w0 + gw > (uint32_t)nw || w0 >= 2 * kMaxGroups) return;
                    Group g;
                    g.gw = gw;
                    g.gi = (uint32_t)w - w0;
                    g.bar = 1 + w0 / 2;
                    g.sh = &s_group[w0 / 2];
                    g.buf = bufs + (size_t)w0 * buf_words;
                    g.lists = lists + (size_t)w0 * warp_list_words(dcap, compact_max);
                    for (;;) {
                        if (g.gi == 0 && lane == 0) {
                            uint32_t v = count;
                            if (!(heavy && budget.over(err))) {
                                if (!slot) v = atomicAdd(&s_wide[cls], 1u);
                                else
                                    v = (cls == 0 ? atomicAdd(&slot->wide_cursor, 1u) & 0xffffu
                                                  : atomicAdd(&slot->wide_cursor, 0x10000u) >> 16) -
                                        (kCursorEnd - count);
                            }
                            *g.sh = {0, v, 0, 0, 0, 0};
                        }
                        g.sync();
                        const uint32_t i = g.sh->unit;
                        if (i >= count) break;
                        const uint32_t t = select_member(lane < W ? s_cls[cls][lane] : 0u, i);
                        const uint32_t c = lane < W ? rows[t * RS + lane] : 0u;
                        wide_row<K - 2, WORK>(x, g, c, lane, acc, work);
                        if (WORK && sink.per_arc) {
                            const unsigned long long d = warp_sum_u64(acc, err);
                            if (lane == 0) {
                                if (d) atomicAdd(&sink.per_arc[base + t], d);
                                s_arc[wb] += d;
                            }
                            acc = 0;
                        }
                        g.sync();
                    }
                    g.sync();  // every warp has read the last claim before the state is used again
                };
                if (nwide) {
                    uint32_t gw = 2;
                    if (nbig) {
                        while (gw * buf_words < wide_words(s_most) && gw < most_gw) gw *= 2;
                    }
#pragma unroll 1
                    for (int cls = nbig ? 0 : 1; cls < 2; cls++)
                        run_wide(cls, cls ? nmid : nbig, cls ? 2u : gw);
                }
            }
            // k = 4, upper-triangular rows: the triangles of the local subgraph are the arcs (t, b)'s
            // |row_t ∧ row_b|.  Unit (q, v): lane l takes row t = 32q + l and its members b in word v;
            // a row-by-row walk spends a few hundred instructions per row on sets that average 33
            // members (R-MAT 20: 12.3 against 10.4 ms).
            if constexpr (K == 4) {
                if (x.tri) {
                    const uint32_t nunits = W * (W + 1) / 2;
                    for (;;) {
                        uint32_t v = 0, q = 0;
                        if (lane == 0) v = atomicAdd(&s_task[team], 1u);
                        v = __shfl_sync(kFull, v, 0);
                        if (v >= nunits) break;
                        while (v >= W - q) {
                            v -= W - q;
                            q++;
                        }
                        v += q;
                        const uint32_t t = q * 32 + lane;
                        uint32_t ones = 0, s2 = 0;
                        if (t < D) {
                            const uint32_t *own = rows + t * RS;
                            const uint32_t *block = rows + v * 32 * RS;
                            uint32_t y = own[v];
                            if (WORK) work += (unsigned long long)__popc(y) * (W - v);
                            while (y) {
                                const uint32_t b1 = 31u - __clz(y), lb = y & (0u - y), b2 = 31u - __clz(lb);
                                const uint32_t *r1 = block + b1 * RS, *r2 = block + b2 * RS;
                                const uint32_t two = b1 == b2 ? 0u : kFull;
                                y &= ~((1u << b1) | lb);
                                for (uint32_t z = v; z < W; z++) {
                                    const uint32_t o = own[z];
                                    csa_add(ones, o & r1[z], o & r2[z] & two, s2);
                                }
                            }
                            s2 += __popc(ones);
                            if (WORK && sink.per_arc && s2) atomicAdd(&sink.per_arc[base + t], (unsigned long long)s2);
                        }
                        acc += s2;
                        __syncwarp();
                    }
                    units = 0;
                }
            }
            // a warp claims its next unit before it works on the current one, so that the
            // atomic's round trip (global memory for a published heavy root) overlaps the work
            auto claim = [&]() -> uint32_t {
                uint32_t v = 0;
                if (lane == 0)
                    v = heavy && budget.over(err) ? units : (slot ? atomicAdd(&slot->cursor, 1u) : atomicAdd(&s_task[team], 1u));
                return v;
            };
            uint32_t next_i = claim();
            for (;;) {
                const uint32_t i = __shfl_sync(kFull, next_i, 0);
                if (i >= units) break;
                next_i = claim();
                uint32_t t = i, j = 0;
                bool whole = true;
                if (cut) {
                    // the row of unit i: the last t with s_upre[t] <= i
                    uint32_t lo = 0, hi = D - 1;
                    while (lo < hi) {
                        const uint32_t mid = (lo + hi + 1) >> 1;
                        if (s_upre[mid] <= i) lo = mid;
                        else hi = mid - 1;
                    }
                    t = lo;
                    j = i - s_upre[t];
                    whole = (t + 1 < D ? s_upre[t + 1] : units) - s_upre[t] == 1u;
                } else if (nwide && is_wide(t)) {
                    continue;
                }
                const uint32_t c = lane < W ? rows[t * RS + lane] : 0u;
                if (whole) {
                    const uint32_t cnt = __reduce_add_sync(kFull, __popc(c));
                    if (cnt >= K - 2) warp_dfs<K - 2, WORK, true>(x, c, lane, acc, work);
                } else if constexpr (K >= 6) {
                    // the j-th member b of row t: the sub-task (u, a_t, b)
                    const uint32_t b = select_member(c, j);
                    const uint32_t c2 = lane < W ? (c & rows[b * RS + lane]) : 0u;
                    if (WORK && lane < (int)W) work += 1;
                    const uint32_t cnt = __reduce_add_sync(kFull, __popc(c2));
                    if (cnt >= K - 3) warp_dfs<K - 3, WORK>(x, c2, lane, acc, work);
                }
                if (WORK && sink.per_arc) {
                    // debug output (instrumented kernel only): acc holds this unit's part of edge
                    // task t alone (it restarts from zero after every unit; the warp's running
                    // sum is kept in s_arc)
                    const unsigned long long d = warp_sum_u64(acc, err);
                    if (lane == 0) {
                        if (d) atomicAdd(&sink.per_arc[base + t], d);
                        s_arc[wb] += d;
                    }
                    acc = 0;
                }
            }
        }
        if (WORK) {
            const unsigned long long wsum = warp_sum_u64(work, err);
            if (lane == 0 && wsum) atomicAdd(work_out, wsum);
        }
        const unsigned long long ws = warp_sum_u64(acc, err);
        if (lane == 0) {
            s_acc[wb] = ws;
            if (WORK) {  // the per-arc mode's running sum (zero without it)
                s_acc[wb] += s_arc[wb];
                s_arc[wb] = 0;
            }
        }
        sync();
        if (tx == 0) {
            unsigned long long r = 0;
            bool wrapped = false;
            for (int i = 0; i < nw; i++) {
                const unsigned long long s2 = r + s_acc[team * nw + i];
                wrapped |= s2 < r;
                r = s2;
            }
            if (wrapped) set_error(err, kDevOverflow);
            if (sink.wants_root_total()) {
                if (heavy) sink.add(u, r, err);
                else sink.put(u, r, err);
            }
            const unsigned long long s2 = block_total + r;
            if (s2 < block_total) set_error(err, kDevOverflow);
            block_total = s2;
        }
        sync();
    }
    if (tx == 0) {
        add_checked(result, block_total, err);
        if (block_ns) atomicMax(&block_ns[2 * blockIdx.x + 1], global_ns());  // its last team's end
    }
}

// ------------------------------------------------------------------------------------------
// Warp-register path: the kernel (its recursion, small_dfs, is above).

template <int K>
constexpr bool kSmallDense = K >= 7;  // below, enumerating at most 32 members is short
constexpr uint32_t kSmallScratch = 32 + kMaskWords + kNbhdList + kNbhdWords;  // cbuf, then comp4's

// Counts a root of D > 16 members on its complement if its rows (lane i: row i) are upper-triangular and
// dense; else returns false.
template <int K>
__device__ __forceinline__ bool small_dense(uint32_t myrow, uint32_t D, int lane, bool compact, uint32_t *comp,
                                            uint32_t *scr, uint32_t *err, unsigned long long &acc)
{
    if constexpr (kSmallDense<K>) {
        if (!compact || D <= 16 || __any_sync(kFull, myrow & ~above_bit(lane))) return false;
        const uint32_t pairs = D * (D - 1) / 2, missing = pairs - __reduce_add_sync(kFull, __popc(myrow));
        if (!is_dense<K - 1>(D, missing, pairs)) return false;
        if (missing == 0) {
            if (lane == 0) add_acc(acc, choose<K - 1>(D), err);
            return true;
        }
        put_block(comp, 0, D, 0, 0, myrow, lane);
        __syncwarp();
        WarpCtx x = {};
        x.cbuf = scr;
        x.mv = scr + 32;
        x.err = err;
        const CompSet cs = {comp, 0, 1};
        unsigned long long work = 0;
        dense_dfs<K - 1, 1, false>(x, cs, word_mask(D, lane), D, lane, acc, work);
        __syncwarp();
        return true;
    } else {
        return false;
    }
}

// One warp per root; the D (D - 1) / 2 pairs of its members are looked up (binary search of one
// member in the other's list).  Scanning the members' whole lists instead costs their length:
// R-MAT 20, roots of 9..32 out-neighbours: 3061 list entries per root on average, 116 pairs.
// From k = 7 on a root whose subgraph is dense, in a DAG relabelled to its order, is counted on the
// complement (one word per row) like the bitmap path's sets; the others are enumerated.  Leaving all
// roots of more than 16 to blocks instead: 20,000 vertices of degree 40, k = 7 0.15 -> 0.23 ms; enumerating
// all of them: R-MAT 15, k = 8 13 ms in this kernel.
template <int K>
__global__ __launch_bounds__(kSmallWarps * 32) void k_count_small(
    const uint64_t *__restrict__ dag_off, const uint32_t *__restrict__ dag_cols,
    const uint32_t *__restrict__ list, const CountStats *st, unsigned long long *result,
    RootSink sink, bool compact, Budget budget, uint32_t *err)
{
    // per member: its id, its list and the list's first entry; its row as it fills
    __shared__ uint64_t s_rb[kSmallWarps][32];
    __shared__ uint32_t s_x[kSmallWarps][32], s_len[kSmallWarps][32], s_min[kSmallWarps][32], s_row[kSmallWarps][32];
    // the complement's rows (16 bytes each) and the lists of its walk
    __shared__ __align__(16) uint32_t s_comp[kSmallDense<K> ? kSmallWarps : 1][kSmallDense<K> ? 128 : 4];
    __shared__ __align__(16) uint32_t s_scr[kSmallDense<K> ? kSmallWarps : 1][kSmallDense<K> ? kSmallScratch : 4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t nlist = st->n_small;
    const uint32_t gw = blockIdx.x * kSmallWarps + w, nwarps = gridDim.x * kSmallWarps;
    unsigned long long total = 0;
    for (uint32_t idx = gw; idx < nlist; idx += nwarps) {
        int stop = 0;
        if (lane == 0) stop = budget.over(err);
        if (__shfl_sync(kFull, stop, 0)) break;
        const uint32_t u = list[idx];
        const uint64_t base = dag_off[u];
        const uint32_t D = (uint32_t)(dag_off[u + 1] - base);
        if (lane < D) {
            const uint32_t x = dag_cols[base + lane];
            const uint64_t rb = dag_off[x];
            const uint32_t len = (uint32_t)(dag_off[x + 1] - rb);
            s_x[w][lane] = x;
            s_rb[w][lane] = rb;
            s_len[w][lane] = len;
            s_min[w][lane] = len ? dag_cols[rb] : 0xffffffffu;
        }
        s_row[w][lane] = 0;
        __syncwarp();
        // The members' lists are scanned instead where that is less: a step of 32 entries (one load and a
        // search among the members in shared memory) costs about two levels of 64 pairs' searches, of
        // which a pair takes twice as many where rows reach down to smaller ids (a DAG that keeps
        // vertex ids).  20,000 vertices of degree 40, ids kept, k = 3: 158 us by pairs, 149 so; Chung-Lu
        // of 20,000, ids kept, k = 4: 150 and 123.  With the line twice and four times as high
        // 1,000,000 vertices of degree 10 take 0.64 and 0.70 ms instead of 0.57.
        const uint32_t len = lane < D ? s_len[w][lane] : 0u;
        const bool down = __any_sync(kFull, len && s_min[w][lane] < s_x[w][lane]);
        const uint32_t steps = __reduce_add_sync(kFull, (len + 31) >> 5), levels = 32 - __clz(__reduce_max_sync(kFull, len));
        const bool lists = 2 * steps <= ((D * (D - 1) / 2 + 63) / 64) * levels * (down ? 2 : 1);
        if (lists) {
            const uint32_t most = s_x[w][D - 1];
            for (uint32_t i = 0; i < D; i++) {
                const uint32_t n = s_len[w][i];
                uint32_t bits = 0;
                for (uint32_t q = 0; q < n; q += 32) {
                    const uint32_t y = q + lane < n ? dag_cols[s_rb[w][i] + q + lane] : 0xffffffffu;
                    if (__shfl_sync(kFull, y, 0) > most) break;
                    const uint32_t j = lower_bound_smem(s_x[w], D, y);
                    if (j < D && s_x[w][j] == y) bits |= 1u << j;
                }
                bits = __reduce_or_sync(kFull, bits);
                if (lane == 0) s_row[w][i] = bits;
            }
        }
        // Every pair of members once, two per lane and round: pair p is (c, c + r + 1 mod D) with
        // r = p / D, c = p mod D.  An arc between them is in the row of one of the two: the one
        // of lower index if rows only hold larger ids (a relabelled DAG), else either.
        const uint32_t npairs = lists ? 0u : D * (D - 1) / 2;
        const float inv = 1.0f / (float)D;
        for (uint32_t p0 = 0; p0 < npairs; p0 += 64) {
            uint32_t src[2], dst[2], lo[2], left[2];
            const uint32_t *row[2];
            uint32_t want[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t p = p0 + 32 * h + lane;
                const uint32_t r = (uint32_t)(((float)p + 0.5f) * inv), c = p - r * D;
                const uint32_t o = c + r + 1 >= D ? c + r + 1 - D : c + r + 1;
                const bool in = p < npairs;
                src[h] = in ? min(c, o) : 0u;
                dst[h] = in ? max(c, o) : 0u;
                lo[h] = 0;
                left[h] = in ? s_len[w][src[h]] : 0u;
                row[h] = dag_cols + s_rb[w][src[h]];
                want[h] = s_x[w][dst[h]];
            }
            for (;;) {
                // both searches step together, so that two loads are in flight
                while (left[0] | left[1]) {
                    uint32_t y[2];
#pragma unroll
                    for (int h = 0; h < 2; h++) y[h] = left[h] ? row[h][lo[h] + (left[h] >> 1)] : 0u;
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const uint32_t half = left[h] >> 1;
                        if (left[h] && y[h] == want[h]) {
                            atomicOr(&s_row[w][src[h]], 1u << dst[h]);
                            left[h] = 0;
                            dst[h] = src[h];  // found
                        } else if (y[h] < want[h]) {
                            lo[h] += left[h] ? half + 1 : 0u;
                            left[h] -= left[h] ? half + 1 : 0u;
                        } else {
                            left[h] = half;
                        }
                    }
                }
                // the other direction, where the row's ids reach down to it
                bool more = false;
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    if (dst[h] > src[h] && s_min[w][dst[h]] <= s_x[w][src[h]]) {
                        const uint32_t t = src[h];
                        src[h] = dst[h];
                        dst[h] = t;
                        lo[h] = 0;
                        left[h] = s_len[w][src[h]];
                        row[h] = dag_cols + s_rb[w][src[h]];
                        want[h] = s_x[w][t];
                        more = true;
                    }
                }
                if (!more) break;
            }
        }
        __syncwarp();
        const uint32_t myrow = s_row[w][lane];
        unsigned long long acc = 0;
        const uint32_t all = D == 32 ? kFull : ((1u << D) - 1);
        if (sink.per_arc) {
            // debug output: the root's edge tasks one at a time, each (K-2)-clique count of
            // N+(u) ∩ N+(a) stored for its arc
            for (uint32_t a = 0; a < D; a++) {
                const uint32_t c2 = all & __shfl_sync(kFull, myrow, a);
                unsigned long long t = 0;
                if (__popc(c2) >= K - 2) small_dfs<K - 2>(c2, myrow, lane, t);
                const unsigned long long tt = warp_sum_u64(t, err);
                if (lane == 0) sink.per_arc[base + a] = tt;
                acc += t;
            }
        } else if (!small_dense<K>(myrow, D, lane, compact, s_comp[kSmallDense<K> ? w : 0], s_scr[kSmallDense<K> ? w : 0], err, acc)) {
            small_dfs<K - 1>(all, myrow, lane, acc);
        }
        if (sink.wants_root_total()) {
            const unsigned long long r = warp_sum_u64(acc, err);
            if (lane == 0) sink.put(u, r, err);
        }
        total += acc;
        __syncwarp();
    }
    total = warp_sum_u64(total, err);
    if (lane == 0) add_checked(result, total, err);
}

// ------------------------------------------------------------------------------------------
// Sorted-list path (D > bitmap_max).

// R-cliques inside the sorted candidate list C[0..len); buf holds one list per deeper level.
template <int R>
__device__ void list_dfs(const uint64_t *__restrict__ dag_off, const uint32_t *__restrict__ cols,
                         const uint32_t *C, uint32_t len, uint32_t *buf, uint32_t stride, int lane,
                         unsigned long long &acc)
{
    if (len < (uint32_t)R) return;
    if constexpr (R == 1) {
        if (lane == 0) acc += len;
    } else {
        for (uint32_t i = 0; i < len; i++) {
            const uint32_t a = C[i];
            const uint64_t ab = dag_off[a], ae = dag_off[a + 1];
            uint32_t out = 0;
            for (uint32_t p = 0; p < len; p += 32) {
                bool hit = false;
                uint32_t x = 0;
                if (p + lane < len) {
                    x = C[p + lane];
                    uint64_t lo = ab, hi = ae;
                    while (lo < hi) {
                        const uint64_t mid = lo + (hi - lo) / 2;
                        if (cols[mid] < x) lo = mid + 1;
                        else hi = mid;
                    }
                    hit = lo < ae && cols[lo] == x;
                }
                const uint32_t bal = __ballot_sync(kFull, hit);
                if constexpr (R == 2) {
                    if (lane == 0) acc += __popc(bal);
                } else {
                    if (hit) buf[out + __popc(bal & lanemask_lt())] = x;
                }
                out += __popc(bal);
            }
            if constexpr (R >= 3) {
                __syncwarp();
                if (out >= (uint32_t)(R - 1))
                    list_dfs<R - 1>(dag_off, cols, buf, out, buf + stride, stride, lane, acc);
                __syncwarp();
            }
        }
    }
}

template <int K>
__global__ __launch_bounds__(kListWarps * 32) void k_count_list(
    const uint64_t *__restrict__ dag_off, const uint32_t *__restrict__ dag_cols,
    const uint32_t *__restrict__ list, const CountStats *st, uint32_t *next, uint32_t *scratch,
    uint32_t stride, unsigned long long *result, RootSink sink, Budget budget, uint32_t *err)
{
    const int lane = threadIdx.x & 31;
    const uint32_t gw = blockIdx.x * kListWarps + (threadIdx.x >> 5);
    uint32_t *buf = scratch + (size_t)gw * stride * (K > 3 ? K - 3 : 1);
    const uint32_t nlist = st->n_big;
    unsigned long long total = 0;
    for (;;) {
        uint32_t idx = 0;
        if (lane == 0) idx = budget.over(err) ? nlist : atomicAdd(next, 1u);
        idx = __shfl_sync(kFull, idx, 0);
        if (idx >= nlist) break;
        const uint32_t u = list[idx];
        const uint64_t base = dag_off[u];
        const uint32_t D = (uint32_t)(dag_off[u + 1] - base);
        if (D > stride) {
            if (lane == 0) set_error(err, kDevScratch);
            continue;
        }
        unsigned long long acc = 0;
        if (sink.per_arc) {
            // debug output: the root's edge tasks one at a time (list_dfs's first level, with
            // the intersection N+(u) ∩ N+(a) always listed in buf)
            const uint32_t *C = dag_cols + base;
            for (uint32_t i = 0; i < D; i++) {
                const uint32_t a = C[i];
                const uint64_t ab = dag_off[a], ae = dag_off[a + 1];
                uint32_t out = 0;
                for (uint32_t p = 0; p < D; p += 32) {
                    bool hit = false;
                    uint32_t y = 0;
                    if (p + lane < D) {
                        y = C[p + lane];
                        uint64_t lo = ab, hi = ae;
                        while (lo < hi) {
                            const uint64_t mid = lo + (hi - lo) / 2;
                            if (dag_cols[mid] < y) lo = mid + 1;
                            else hi = mid;
                        }
                        hit = lo < ae && dag_cols[lo] == y;
                    }
                    const uint32_t bal = __ballot_sync(kFull, hit);
                    if (hit) buf[out + __popc(bal & lanemask_lt())] = y;
                    out += __popc(bal);
                }
                __syncwarp();
                unsigned long long t = 0;
                list_dfs<K - 2>(dag_off, dag_cols, buf, out, buf + stride, stride, lane, t);
                __syncwarp();
                const unsigned long long tt = warp_sum_u64(t, err);
                if (lane == 0) sink.per_arc[base + i] = tt;
                acc += t;
            }
        } else {
            list_dfs<K - 1>(dag_off, dag_cols, dag_cols + base, D, buf, stride, lane, acc);
        }
        if (sink.wants_root_total()) {
            const unsigned long long r = warp_sum_u64(acc, err);
            if (lane == 0) sink.put(u, r, err);
        }
        total += acc;
    }
    total = warp_sum_u64(total, err);
    if (lane == 0) add_checked(result, total, err);
}

}  // namespace citron

namespace citron_host {
using namespace citron;

// Global-memory helpers of the bitmap kernel: the help table of heavy roots and the per-block
// start/end times (2 words per block, kMidBlocksPerSmCap blocks per SM and launch at most).
constexpr uint32_t kMidBlocksPerSmCap = 8;
constexpr uint32_t kMidLaunches = 2;
struct MidAux {
    HelpTable help;
    unsigned long long *block_ns = nullptr;
    Budget budget;  // the count's time budget (all of its launches)
};

struct Timer {
    cudaEvent_t a = nullptr, b = nullptr;
    bool on;
    cudaStream_t s;
    Timer(bool enable, cudaStream_t st) : on(enable), s(st)
    {
        if (on && (cudaEventCreate(&a) || cudaEventCreate(&b))) on = false;
        if (on) cudaEventRecord(a, s);
    }
    void stop() { if (on) cudaEventRecord(b, s); }
    float ms()
    {
        float t = 0;
        if (on && cudaEventSynchronize(b) == cudaSuccess) cudaEventElapsedTime(&t, a, b);
        return t;
    }
    ~Timer()
    {
        if (a) cudaEventDestroy(a);
        if (b) cudaEventDestroy(b);
    }
};

template <int K, bool WORK, bool TEAMED>
static cudaError_t launch_mid(uint32_t grid_cap, uint32_t block_cap, int low, uint32_t teams, uint32_t dcap,
                              uint32_t buf_words, uint32_t window, uint32_t compact_max, uint32_t split_min,
                              const HelpTable &ht,
                              uint32_t warps, size_t team_smem, const uint64_t *dag_off,
                              const uint32_t *dag_cols, const uint32_t *mid_list,
                              const CountStats *st, uint32_t *next, unsigned long long *result,
                              RootSink sink, unsigned long long *work, unsigned long long *block_ns,
                              Budget budget, uint32_t *grid_out, uint32_t *err, cudaStream_t s,
                              int num_sms)
{
    cudaError_t e;
    // the attribute is an upper bound on the launches' dynamic shared memory; it is always set to
    // the device's largest value, because host threads that count concurrently would otherwise
    // overwrite each other's smaller setting between the set and the launch
    int dev = 0, optin = 0;
    const size_t smem = teams * team_smem;
    warps *= teams;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    if ((size_t)optin < smem + kMidStaticSmem) return cudaErrorInvalidValue;
    if ((e = cudaFuncSetAttribute(k_count_mid<K, WORK, TEAMED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  optin - (int)kMidStaticSmem)))
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_count_mid<K, WORK, TEAMED>, warps * 32,
                                                           smem)))
        return e;
    if (per_sm < 1) per_sm = 1;
    uint32_t grid = (uint32_t)(num_sms * per_sm);
    if (grid > grid_cap) grid = grid_cap;
    if (block_cap && grid > block_cap) grid = block_cap;
    if (grid > (uint32_t)num_sms * kMidBlocksPerSmCap) grid = (uint32_t)num_sms * kMidBlocksPerSmCap;
    *grid_out = grid;
    k_count_mid<K, WORK, TEAMED><<<grid, warps * 32, smem, s>>>(dag_off, dag_cols, mid_list, st, next, low, (int)teams, dcap,
                                                        (uint32_t)(team_smem / sizeof(uint32_t)), buf_words, window, compact_max,
                                                        split_min, ht, result, sink, work, block_ns, budget, err);
    note_launches(1);
    return cudaGetLastError();
}

template <int K>
static cudaError_t launch_count_k(CountRun &run, const uint64_t *dag_off, const uint32_t *dag_cols,
                                  const CountStats &hs, const CountStats *st,
                                  const uint32_t *small_list, const uint32_t *mid_list,
                                  const uint32_t *big_list, uint32_t *next, uint32_t *list_scratch,
                                  size_t list_scratch_words, unsigned long long *result,
                                  unsigned long long *work, const MidAux &aux, uint32_t *err,
                                  cudaStream_t s, int num_sms)
{
    cudaError_t e = cudaSuccess;
    const CountPlan &plan = run.plan;
    if (hs.n_mid) {
        int smem_cap = 0, dev = 0;
        cudaGetDevice(&dev);
        if ((e = cudaDeviceGetAttribute(&smem_cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)))
            return e;
        smem_cap -= (int)kMidStaticSmem;
        // k = 4 ends at R = 2 and re-encodes no set: its warps need no room for one
        const uint32_t compact_max = K >= 5 ? plan.compact_max : 0u;
        Timer t(run.time_kernels, s);
        unsigned long long *block_ns = run.balance ? aux.block_ns : nullptr;
        const size_t ns_words = 2 * (size_t)num_sms * kMidBlocksPerSmCap;  // of one launch
        if (block_ns && (e = cudaMemsetAsync(block_ns, 0, kMidLaunches * ns_words * sizeof(*block_ns), s))) return e;
        uint32_t grid[kMidLaunches] = {0, 0};
        for (int low = 0; low < 2; low++) {
            const uint32_t n_roots = low ? hs.n_low : hs.n_high;
            if (!n_roots) continue;
            const uint32_t dmax = low && hs.max_mid > kLowMax ? kLowMax : hs.max_mid;
            const uint32_t dcap = (dmax + 31) & ~31u, rs = (dcap / 32) | 1;
            uint32_t warps = plan.warps_per_cta > (uint32_t)kMidMaxWarps ? kMidMaxWarps : plan.warps_per_cta;
            if (low && warps > kLowWarps) warps = kLowWarps;
            uint32_t buf_words = warp_buf_words(dcap, compact_max, K >= 8);
            auto scratch = [&](uint32_t nw) {  // words for the warps' lists and buffers
                return K > 3 ? (size_t)nw * (warp_list_words(dcap, compact_max) + buf_words) : (size_t)kMidWindow / 32;
            };
            auto smem_for = [&](uint32_t nw) {
                return ((size_t)dcap + (K > 3 ? (size_t)dcap * rs : 0) + scratch(nw)) * sizeof(uint32_t);
            };
            while (warps > 1 && smem_for(warps) > (size_t)smem_cap) warps--;
            // room for the packed rows of 192 members where it costs no warp
            if (const uint32_t was = buf_words; compact_max && dcap > kNarrow && was < packed_words(6)) {
                buf_words = packed_words(6);
                if (smem_for(warps) > (size_t)smem_cap) buf_words = was;
            }
            // the window's bitmap and first places (k > 3) have to fit the scratch
            uint32_t window = kMidWindow;
            while ((size_t)window / 32 + (K > 3 ? window / 64 : 0) > scratch(warps)) window /= 2;
            unsigned long long *ns = block_ns ? block_ns + low * ns_words : nullptr;
            uint32_t *queue = next + (low ? 3 : 0);
            // under a cap: teams of kLowWarps in blocks as wide as the other launch's
            uint32_t teams = 1;
            if (K <= 6 && low && plan.max_blocks && !run.count_work && !run.sink.per_arc)
                while (teams < (uint32_t)kMaxTeams && 2 * teams * kLowWarps <= plan.warps_per_cta &&
                       2 * teams * smem_for(warps) <= (size_t)smem_cap)
                    teams *= 2;
            auto launch = [&](auto kind) {
                constexpr int v = decltype(kind)::value;  // 0 plain, 1 instrumented, 2 in teams
                return launch_mid<K, v == 1, v == 2>((n_roots + teams - 1) / teams, plan.max_blocks, low, teams, dcap,
                                                     buf_words, window, compact_max, plan.split_min, aux.help, warps,
                                                     smem_for(warps), dag_off, dag_cols, mid_list, st, queue, result,
                                                     run.sink, work, ns, aux.budget, &grid[low], err, s, num_sms);
            };
            // the instrumented kernel also serves the per-arc debug output (its code is compiled
            // out of the plain kernel)
            if (run.count_work || run.sink.per_arc) {
                if constexpr (K <= (int)kInstrumentedMaxK) e = launch(std::integral_constant<int, 1>());
                else e = cudaErrorNotSupported;  // refused by citron_count_ex before any launch
            } else if (teams > 1) {
                if constexpr (K <= 6) e = launch(std::integral_constant<int, 2>());
            } else {
                e = launch(std::integral_constant<int, 0>());
            }
            if (e) return e;
        }
        t.stop();
        run.kernel_ms[1] = t.ms();
        if (block_ns) {
            // span = first block start .. last block end, over both launches; tail = first block end ..
            // last block end, of each launch
            unsigned long long s0 = ~0ull, last = 0, tails = 0;
            for (uint32_t l = 0; l < kMidLaunches; l++) {
                unsigned long long h[2 * kMidBlocksPerSmCap * 256];
                const size_t cnt = 2 * (size_t)grid[l];
                if (!cnt || cnt > sizeof(h) / sizeof(h[0])) continue;
                e = cudaMemcpyAsync(h, block_ns + l * ns_words, cnt * sizeof(h[0]), cudaMemcpyDeviceToHost, s);
                if (!e) e = cudaStreamSynchronize(s);
                if (e) return e;
                unsigned long long e0 = ~0ull, e1 = 0;
                for (uint32_t b = 0; b < grid[l]; b++) {
                    s0 = h[2 * b] < s0 ? h[2 * b] : s0;
                    e0 = h[2 * b + 1] < e0 ? h[2 * b + 1] : e0;
                    e1 = h[2 * b + 1] > e1 ? h[2 * b + 1] : e1;
                }
                last = e1 > last ? e1 : last;
                tails += e1 - e0;
            }
            if (last) {
                run.busy_ms[0] = (float)((last - s0) * 1e-6);
                run.busy_ms[1] = (float)(tails * 1e-6);
            }
        }
    }
    if (hs.n_small) {
        uint32_t grid = (hs.n_small + kSmallWarps - 1) / kSmallWarps;
        uint32_t cap = (uint32_t)num_sms * 16;
        if (plan.max_blocks && cap > plan.max_blocks * 4) cap = plan.max_blocks * 4;
        if (grid > cap) grid = cap;
        Timer t(run.time_kernels, s);
        k_count_small<K><<<grid, kSmallWarps * 32, 0, s>>>(dag_off, dag_cols, small_list, st, result, run.sink,
                                                           plan.compact_max != 0, aux.budget, err);
        note_launches(1);
        if ((e = cudaGetLastError())) return e;
        t.stop();
        run.kernel_ms[0] = t.ms();
    }
    if (hs.n_big) {
        const size_t per_warp = (size_t)hs.max_big * (K > 3 ? K - 3 : 1);
        size_t warps = per_warp ? list_scratch_words / per_warp : 0;
        if (warps < kListWarps) return cudaErrorMemoryAllocation;
        uint32_t grid = (uint32_t)(warps / kListWarps);
        uint32_t cap = (uint32_t)num_sms;
        if (plan.max_blocks && cap > plan.max_blocks) cap = plan.max_blocks;
        if (grid > cap) grid = cap;
        if (grid > (hs.n_big + kListWarps - 1) / kListWarps) grid = (hs.n_big + kListWarps - 1) / kListWarps;
        Timer t(run.time_kernels, s);
        k_count_list<K><<<grid, kListWarps * 32, 0, s>>>(dag_off, dag_cols, big_list, st, next + 1,
                                                         list_scratch, hs.max_big, result,
                                                         run.sink, aux.budget, err);
        note_launches(1);
        if ((e = cudaGetLastError())) return e;
        t.stop();
        run.kernel_ms[2] = t.ms();
    }
    return cudaSuccess;
}

// Per-k launchers, each compiled in its own translation unit (count_k*.cu).
#define CITRON_LAUNCH_K_DECL(KK)                                                                     \
    cudaError_t launch_count_##KK(CountRun &run, const uint64_t *dag_off, const uint32_t *dag_cols,  \
                                  const CountStats &hs, const CountStats *st,                       \
                                  const uint32_t *small_list, const uint32_t *mid_list,             \
                                  const uint32_t *big_list, uint32_t *next, uint32_t *list_scratch, \
                                  size_t list_scratch_words, unsigned long long *result,            \
                                  unsigned long long *work, const MidAux &aux, uint32_t *err,       \
                                  cudaStream_t s, int num_sms)
#define CITRON_LAUNCH_K_DEF(KK)                                                                      \
    CITRON_LAUNCH_K_DECL(KK)                                                                         \
    {                                                                                                \
        return launch_count_k<KK>(run, dag_off, dag_cols, hs, st, small_list, mid_list, big_list,   \
                                  next, list_scratch, list_scratch_words, result, work, aux, err,   \
                                  s, num_sms);                                                      \
    }
CITRON_LAUNCH_K_DECL(3);
CITRON_LAUNCH_K_DECL(4);
CITRON_LAUNCH_K_DECL(5);
CITRON_LAUNCH_K_DECL(6);
CITRON_LAUNCH_K_DECL(7);
CITRON_LAUNCH_K_DECL(8);
CITRON_LAUNCH_K_DECL(9);
CITRON_LAUNCH_K_DECL(10);
CITRON_LAUNCH_K_DECL(11);
CITRON_LAUNCH_K_DECL(12);

}  // namespace citron_host

// dense.cuh -- cliques of a dense candidate set, counted on its COMPLEMENT.
//
// A candidate set S of s members (N+(u) ∩ N+(a), or a deeper set) of a graph with a dense core is
// nearly a clique: on R-MAT 20 the sets of the edge tasks have a mean density of 0.85 to 0.9, and
// weighted by the arcs of their leaves 0.95.  With H the complement graph on S (a few edges per
// member), two identities replace the recursion's last levels:
//
//   3-cliques (A. W. Goodman, "On sets of acquaintances and strangers at any party", 1959):
//     2 N3 = 2 C(s,3) - sum_v d(s-1-d) - 2 t          d: degree in H, t: triangles of H
//   4-cliques = independent 4-sets of H, by inclusion-exclusion over the edges of H that lie inside
//     a 4-subset (N(X): subgraphs of H isomorphic to X, not necessarily induced):
//     N4 = C(s,4) - m C(s-2,2) + [N(P3)(s-3) + N(2K2)] - [t(s-3) + N(K1,3) + N(P4)]
//          + [N(C4) + N(paw)] - N(diamond) + N(K4)
//     m edges; N(P3) = sum C(d,2); N(2K2) = C(m,2) - N(P3); N(K1,3) = sum C(d,3);
//     N(P4) = sum over edges (d_u-1)(d_v-1) - 3t; with c the codegree of a pair:
//     N(C4) = 1/2 sum over pairs C(c,2); N(diamond) = sum over edges C(c,2);
//     N(paw) = sum_v t_v (d_v - 2), t_v = the triangles at v = 1/2 sum over neighbours c.
// Only N(K4) of the sparse H is enumerated.  The codegrees of a member v with every other member
// are the bitwise column sums of the rows of v's neighbours in H: they are kept as bit planes
// (plane j holds bit j of every codegree) and added with LOP3 full adders, so that one step adds
// one neighbour to 32 codegrees per word.
//
// What bounds it: instruction issue (and, for the 4-clique form, instruction fetch): listing a set,
// packing its rows and the adders outweigh the word operations.  k_count_mid, k = 6 on R-MAT 20:
// 683 ms enumerating the sets' arcs, 231 ms when this came in, 207 ms now; k = 8 on R-MAT 15: 577 ms,
// 69 and 57.  Where the line between the sides lies: dense_line (count_impl.cuh).
//
// All arithmetic is exact modulo 2^32 (sets of at most 128 members) or 2^64; the results are
// below the modulus.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace citron {

constexpr uint32_t kNarrow = 128;      // members of a set whose rows fit one uint4
constexpr uint32_t kWideMaxDeg = 255;  // complement degree the wide planes can hold
constexpr uint32_t kNbhdMax = 128;     // members of a neighbourhood counted by comp_nbhd
constexpr uint32_t kNbhdWords = kNbhdMax * kNbhdMax / 32;  // its rows, and ...
constexpr uint32_t kNbhdList = kNbhdMax / 2;               // ... its member list (uint16)
constexpr uint32_t kMaskWords = 192;   // compress masks (160 words) and one word per lane
constexpr uint32_t kHubNarrow = 16;    // members of a higher complement degree come last in the order
constexpr uint32_t kHubWide = 28;        // (k = 6 on R-MAT 20: 216 ms at 48, 209 at 28)
constexpr uint32_t kNbhdMin = 16;      // wide sets: larger neighbourhoods are counted by comp_nbhd

// Carry-save accumulation of bit counts (a full adder per bit position): the bits of
// ones + a + b are kept as a new `ones` word and a carry word of weight two (two LOP3s), so that
// one POPC counts two words.  POPC and the bit scans share the narrow XU pipe, which bounds the
// leaves; the LOP3s go to the wider ALU pipe.  The running total is s + popc(ones): every user
// adds popc(ones) once at the end.
__device__ __forceinline__ void csa_add(uint32_t &ones, uint32_t a, uint32_t b, uint32_t &s)
{
    const uint32_t u = ones ^ a;
    const uint32_t carry = (ones & a) | (u & b);
    ones = u ^ b;
    s += 2u * (uint32_t)__popc(carry);
}

// Bits are gathered word by word with the parallel-suffix "compress" of H. S. Warren, Hacker's
// Delight (2nd ed., Sec. 7-4): for a mask m the five move masks depend on m only, so they are
// computed once per candidate word (lane-parallel) and shared by every row.
__device__ __forceinline__ void compress_masks(uint32_t m, uint32_t mv[5])
{
    uint32_t mk = ~m << 1;
#pragma unroll
    for (int i = 0; i < 5; i++) {
        uint32_t mp = mk ^ (mk << 1);
        mp ^= mp << 2;
        mp ^= mp << 4;
        mp ^= mp << 8;
        mp ^= mp << 16;
        const uint32_t v = mp & m;
        mv[i] = v;
        m = (m ^ v) | (v >> (1 << i));
        mk &= ~mp;
    }
}

__device__ __forceinline__ uint32_t compress_with(uint32_t x, uint32_t m, const uint32_t *mv)
{
    x &= m;
#pragma unroll
    for (int i = 0; i < 5; i++) {
        const uint32_t t = x & mv[i];
        x = (x ^ t) | (t >> (1 << i));
    }
    return x;
}

// popc_and with carry-save pairs: words [FROM, CW) of a & b, two at a time.
template <int CW, int FROM>
__device__ __forceinline__ void popc_and_csa(const uint32_t (&a)[CW], const uint4 &b, uint32_t &ones, uint32_t &s)
{
    const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
    int w = FROM;
#pragma unroll
    for (int p = 0; p < 2; p++) {
        if (w + 1 < CW) {
            csa_add(ones, a[w] & bw[w], a[w + 1] & bw[w + 1], s);
            w += 2;
        }
    }
    if (w < CW) s += __popc(a[w] & bw[w]);
}

// Two leaf members at once: words [FROM, CW) of D & b1 and of D & b2 paired in the carry-save
// adder (one POPC per word pair).
template <int CW, int FROM>
__device__ __forceinline__ void popc_and_csa2(const uint32_t (&a)[CW], const uint4 &b1, const uint4 &b2,
                                              uint32_t &ones, uint32_t &s)
{
    const uint32_t v1[4] = {b1.x, b1.y, b1.z, b1.w}, v2[4] = {b2.x, b2.y, b2.z, b2.w};
#pragma unroll
    for (int w = FROM; w < CW; w++) csa_add(ones, a[w] & v1[w], a[w] & v2[w], s);
}

// Arcs from the members y of word q2 (FROM = q2 on triangular rows, else 0) into D, on compact
// rows M: two members per step, the highest and the lowest, whose bit scans and row loads are
// independent of each other.
template <int CW, int FROM>
__device__ __forceinline__ void leaf_word(const uint4 *M, const uint32_t (&D)[CW], uint32_t y, uint32_t base,
                                          uint32_t &ones, uint32_t &s)
{
    while (y & (y - 1u)) {
        const uint32_t b1 = 31u - __clz(y);
        const uint32_t lb = y & (0u - y);
        const uint32_t b2 = 31u - __clz(lb);
        y ^= (1u << b1) | lb;
        popc_and_csa2<CW, FROM>(D, M[base + b1], M[base + b2], ones, s);
    }
    if (y) popc_and_csa<CW, FROM>(D, M[base + 31u - __clz(y)], ones, s);
}

struct CompCount {
    uint32_t n;     // cliques of the set (narrow) ...
    uint32_t work;  // word operations done (instrumented kernel only)
};

// Lane-partial sums of a wide set: n4_finish turns their total into the count.
struct CompSums {
    uint32_t sd;            // sum of degrees
    uint32_t st;            // sum over members of the codegrees with their neighbours (6 t)
    unsigned long long sl;  // the terms that add up (times 4)
    uint32_t work;
    bool over;              // a degree above kWideMaxDeg: the planes cannot hold the codegrees
};

// 32 x 32 bit transpose over a warp: bit c of lane r becomes bit r of lane c.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
    uint32_t m = 0x0000ffffu;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint32_t t = __shfl_xor_sync(kFull, x, j);
        const bool up = (lane & j) != 0;
        const uint32_t keep = up ? ~m : m;
        const uint32_t moved = up ? (t >> j) : (t << j);
        x = (x & keep) | (moved & ~keep);
        m ^= m << (j >> 1);
    }
    return x;
}

// Bits above position b of a word (none for b = 31).
__device__ __forceinline__ uint32_t above_bit(uint32_t b) { return ~((2u << b) - 1u); }

// Members of word w in a set of s members numbered 0..s-1.
__device__ __forceinline__ uint32_t word_mask(uint32_t s, uint32_t w)
{
    const uint32_t lo = w << 5;
    return s >= lo + 32 ? kFull : (s > lo ? (1u << (s - lo)) - 1u : 0u);
}

// Word w of row v, rows stored in chunks of four words (chunk-major: rows of one chunk are
// consecutive uint4, so that lanes reading random rows spread over all banks).
__device__ __forceinline__ uint32_t &comp_word(uint32_t *m32, uint32_t S, uint32_t v, uint32_t w)
{
    return m32[(((w >> 2) * S + v) << 2) + (w & 3u)];
}

// The complement words of one 32 x 32 block: g holds the set's adjacency of member 32a + lane to
// the members of word ow >= a (upper-triangular).  Writes block (a, ow) and its mirror image.
// Returns the bits written by this lane.
__device__ __forceinline__ uint32_t put_block(uint32_t *m32, uint32_t S, uint32_t s, uint32_t a,
                                              uint32_t ow, uint32_t g, int lane)
{
    const uint32_t i = (a << 5) + lane;
    uint32_t h = i < s ? word_mask(s, ow) & ~g : 0u;
    if (ow == a) h &= above_bit(lane);
    const uint32_t tr = transpose32(h, lane);
    uint32_t bits;
    if (ow == a) {
        h |= tr;
        bits = __popc(h);
    } else {
        const uint32_t j = (ow << 5) + lane;
        if (j < s) comp_word(m32, S, j, a) = tr;
        bits = __popc(h) + __popc(tr);
    }
    if (i < s) comp_word(m32, S, i, ow) = h;
    return bits;
}

template <int CW>
__device__ __forceinline__ void load_row(const uint4 *M, uint32_t v, uint32_t (&r)[CW])
{
    const uint4 x = M[v];
    r[0] = x.x;
    if (CW > 1) r[1 % CW] = x.y;
    if (CW > 2) r[2 % CW] = x.z;
    if (CW > 3) r[3 % CW] = x.w;
}

// Codegree planes of one member over NW words: plane j holds bit j of the codegree with each of
// the 32 NW members.  Two neighbours are added per step: a full adder at plane 0, half adders at
// planes 1 and 2, and the deeper planes only when a carry reaches them.
template <int NW, int NP>
struct Planes {
    uint32_t p[NP][NW];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int j = 0; j < NP; j++)
#pragma unroll
            for (int w = 0; w < NW; w++) p[j][w] = 0;
    }
    __device__ __forceinline__ void add2(const uint32_t (&r1)[NW], const uint32_t (&r2)[NW])
    {
        uint32_t k[NW], any = 0;
#pragma unroll
        for (int w = 0; w < NW; w++) {
            const uint32_t a = p[0][w], b = r1[w], c = r2[w];
            const uint32_t k0 = (a & b) | (a & c) | (b & c);
            p[0][w] = a ^ b ^ c;
            const uint32_t k1 = p[1][w] & k0;
            p[1][w] ^= k0;
            k[w] = p[2][w] & k1;
            p[2][w] ^= k1;
            any |= k[w];
        }
        if (any) {
#pragma unroll
            for (int j = 3; j < NP; j++)
#pragma unroll
                for (int w = 0; w < NW; w++) {
                    const uint32_t t = p[j][w] & k[w];
                    p[j][w] ^= k[w];
                    k[w] = t;
                }
        }
    }
    // Adds the rows of the members y of the word that begins at member `base` (rows Mq).
    __device__ __forceinline__ void add_word(const uint4 *Mq, uint32_t y, uint32_t base)
    {
        while (y) {
            const uint32_t b1 = 31u - __clz(y), lb = y & (0u - y), b2 = 31u - __clz(lb);
            uint32_t r1[NW], r2[NW];
            load_row<NW>(Mq, base + b1, r1);
            load_row<NW>(Mq, base + b2, r2);
            const uint32_t two = b1 == b2 ? 0u : kFull;
#pragma unroll
            for (int w = 0; w < NW; w++) r2[w] &= two;
            y &= ~((1u << b1) | lb);
            add2(r1, r2);
        }
    }
    // Over the members of mask: the sum of C(codegree, 2); S1 adds the sum of codegrees to s1.
    template <bool S1>
    __device__ __forceinline__ uint32_t pairs(const uint32_t (&mask)[NW], bool deep, uint32_t &s1) const
    {
        uint32_t cc = 0;
#pragma unroll
        for (int w = 0; w < NW; w++) {
            const uint32_t b0 = p[0][w] & mask[w], b1 = p[1][w] & mask[w], b2 = p[2][w] & mask[w];
            const uint32_t n1 = __popc(b1), n2 = __popc(b2);
            if (S1) s1 += __popc(b0) + 2 * n1 + 4 * n2;
            cc += n1 + 6 * n2 + 2 * __popc(b0 & b1) + 4 * __popc(b0 & b2) + 8 * __popc(b1 & b2);
        }
        if (deep) {
            // codegree = lo + 8 hi: C(lo + 8 hi, 2) = C(lo, 2) + 8 lo hi + 32 hi^2 - 4 hi
#pragma unroll
            for (int w = 0; w < NW; w++) {
#pragma unroll
                for (int j = 3; j < NP; j++) {
                    const uint32_t hj = p[j][w] & mask[w];
                    if (!hj) continue;
                    const uint32_t n = __popc(hj), wj = 1u << (j - 3);
                    if (S1) s1 += 8 * wj * n;
                    cc += 8 * wj * (__popc(hj & p[0][w]) + 2 * __popc(hj & p[1][w]) + 4 * __popc(hj & p[2][w]));
                    cc += (32 * wj * wj - 4 * wj) * n;
#pragma unroll
                    for (int l = 3; l < j; l++) cc += 64 * wj * (1u << (l - 3)) * __popc(hj & p[l][w]);
                }
            }
        }
        return cc;
    }
    __device__ __forceinline__ bool deep() const
    {
        uint32_t any = 0;
#pragma unroll
        for (int j = 3; j < NP; j++)
#pragma unroll
            for (int w = 0; w < NW; w++) any |= p[j][w];
        return any != 0;
    }
};

// Triangles of the complement H inside U (lane word uw, u <= kNbhdMax members), by one warp: U's
// own adjacency rows (u bits) are gathered once and the pairs are then worked on them, one word
// load per step instead of the set's whole row.  Returns twice the triangles as lane-partial sums.
// scr: kMaskWords words (the last 32 are left alone), kNbhdList words, kNbhdWords words.
template <bool WORK>
__device__ __noinline__ CompCount comp_nbhd(const uint4 *M, uint32_t S, uint32_t nch, uint32_t uw, uint32_t u,
                                            uint32_t *scr, int lane)
{
    CompCount o = {0, 0};
    uint16_t *list = reinterpret_cast<uint16_t *>(scr + kMaskWords);
    uint32_t *L = scr + kMaskWords + kNbhdList;  // word-major: word t of member i in L[t * U32 + i]
    const uint32_t LW = (u + 31) >> 5, U32 = LW << 5;
    const uint32_t nz = __ballot_sync(kFull, uw != 0);
    {
        uint32_t mv[5];
        compress_masks(uw, mv);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 5; i++) scr[i * 32 + lane] = mv[i];
        uint32_t at = 0;
        for (uint32_t r = nz; r; r &= r - 1) {
            const int w = __ffs(r) - 1;
            const uint32_t m = __shfl_sync(kFull, uw, w);
            if ((m >> lane) & 1u) list[at + __popc(m & lanemask_lt())] = (uint16_t)((w << 5) + lane);
            at += __popc(m);
        }
        __syncwarp();
    }
    for (uint32_t r = 0; r < LW; r++) {
        const uint32_t i = (r << 5) + lane;
        const uint32_t xi = list[i < u ? i : u - 1];
        uint32_t ow = 0, sh = 0, cur = 0;
        for (uint32_t c = 0; c < nch; c++) {
            if (!((nz >> (c << 2)) & 15u)) continue;
            const uint4 x4 = M[c * S + xi];
            const uint32_t xw[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int t = 0; t < 4; t++) {
                const int w = (int)(c << 2) + t;
                const uint32_t m = __shfl_sync(kFull, uw, w);
                if (!m) continue;
                uint32_t mv[5];
#pragma unroll
                for (int k = 0; k < 5; k++) mv[k] = scr[k * 32 + w];
                const uint32_t piece = compress_with(xw[t], m, mv);
                cur |= piece << sh;
                const uint32_t end = sh + __popc(m);
                if (end >= 32) {
                    L[ow * U32 + i] = cur;
                    ow++;
                    cur = sh ? piece >> (32 - sh) : 0u;
                }
                sh = end & 31u;
            }
        }
        if (sh) L[ow * U32 + i] = cur;
    }
    __syncwarp();
    if (LW == 1) {
        const uint32_t D = (uint32_t)lane < u ? L[lane] & above_bit(lane) : 0u;
        uint32_t y = D, ones = 0;
        if (WORK) o.work += __popc(D);
        while (y & (y - 1u)) {
            const uint32_t b1 = 31u - __clz(y), lb = y & (0u - y), b2 = 31u - __clz(lb);
            y ^= (1u << b1) | lb;
            csa_add(ones, D & L[b1], D & L[b2], o.n);
        }
        if (y) o.n += __popc(D & L[31u - __clz(y)]);
        o.n += __popc(ones);
    } else {
        for (uint32_t r = 0; r < LW; r++) {
            const uint32_t i = (r << 5) + lane;
            uint32_t D[4];
#pragma unroll
            for (uint32_t t = 0; t < 4; t++) {
                D[t] = (t >= r && t < LW && i < u) ? L[t * U32 + i] : 0u;
                if (t == r) D[t] &= above_bit(lane);
            }
#pragma unroll
            for (uint32_t t = 0; t < 4; t++) {
                uint32_t y = D[t];
                while (y) {
                    const uint32_t *Lb = L + (t << 5) + 31u - __clz(y);
                    y ^= 1u << (31u - __clz(y));
#pragma unroll
                    for (uint32_t k = 0; k < 4; k++)
                        if (k < LW) o.n += __popc(D[k] & Lb[k * U32]);
                    if (WORK) o.work += LW;
                }
            }
        }
    }
    __syncwarp();
    return o;
}

// The complement rows of a subset U (lane word uw, at most 64 members) of a narrow set, packed to
// U's own numbering: rows of up to two words, one uint4 each, in out.  scr: kMaskWords and kNbhdList
// words.
template <int CW>
__device__ __noinline__ void pack_subset(const uint4 *M, uint32_t uw, uint32_t u, uint32_t *scr, uint32_t *out, int lane)
{
    uint16_t *list = reinterpret_cast<uint16_t *>(scr + kMaskWords);
    uint32_t mv[5];
    compress_masks(uw, mv);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 5; i++) scr[i * 32 + lane] = mv[i];
    uint32_t at = 0;
#pragma unroll
    for (int t = 0; t < CW; t++) {
        const uint32_t m = __shfl_sync(kFull, uw, t);
        if ((m >> lane) & 1u) list[at + __popc(m & lanemask_lt())] = (uint16_t)((t << 5) + lane);
        at += __popc(m);
    }
    __syncwarp();
    for (uint32_t i = lane; i < ((u + 31) & ~31u); i += 32) {
        uint32_t row[CW], o[2] = {0, 0};
        load_row<CW>(M, list[i < u ? i : u - 1], row);
        uint32_t pre = 0;
#pragma unroll
        for (int t = 0; t < CW; t++) {
            const uint32_t m = __shfl_sync(kFull, uw, t);
            uint32_t k[5];
#pragma unroll
            for (int q = 0; q < 5; q++) k[q] = scr[q * 32 + t];
            const unsigned long long piece = (unsigned long long)compress_with(row[t], m, k) << (pre & 31u);
            if (pre < 32) {
                o[0] |= (uint32_t)piece;
                o[1] |= (uint32_t)(piece >> 32);
            } else {
                o[1] |= (uint32_t)piece;
            }
            pre += __popc(m);
        }
        if (i < u) reinterpret_cast<uint4 *>(out)[i] = make_uint4(o[0], o[1], 0u, 0u);
    }
    __syncwarp();
}

// ---- Narrow sets (at most 128 members): one uint4 per complement row --------------------------

// Adjacent pairs (x, y) inside D (CW words), x in D's word T (bits b): y in a later word into `once`,
// y in the same word into `twice` (both orders).  Two members x per step, the highest and the
// lowest.
struct PairSums {
    uint32_t ones, once, ones2, twice;
    __device__ __forceinline__ uint32_t both() const { return 2 * (once + __popc(ones)) + twice + __popc(ones2); }
};

template <int CW, int T>
__device__ __forceinline__ void pair_word(const uint4 *M, const uint32_t (&D)[CW], uint32_t b, uint32_t base, PairSums &p)
{
    while (b) {
        const uint32_t b1 = 31u - __clz(b), lb = b & (0u - b), b2 = 31u - __clz(lb);
        const uint32_t two = b1 == b2 ? 0u : kFull;
        b &= ~((1u << b1) | lb);
        uint32_t r1[CW], r2[CW];
        load_row<CW>(M, base + b1, r1);
        load_row<CW>(M, base + b2, r2);
#pragma unroll
        for (int w = T < 0 ? 0 : T; w < CW; w++) {
            const uint32_t x1 = D[w] & r1[w], x2 = D[w] & r2[w] & two;
            if (w == T) csa_add(p.ones2, x1, x2, p.twice);
            else csa_add(p.ones, x1, x2, p.once);
        }
    }
}

template <int CW, int T>
__device__ __forceinline__ void pair_words(const uint4 *M, const uint32_t (&D)[CW], PairSums &p)
{
    if constexpr (T < CW) {
        pair_word<CW, T>(M, D, D[T], (uint32_t)T << 5, p);
        pair_words<CW, T + 1>(M, D, p);
    }
}

// 3-cliques of the set B (CW words in shared memory, s members) on complement rows M of at most
// 128 members: lane l takes member 32q + l of each word q.
template <int CW, bool WORK>
__device__ __noinline__ CompCount comp3(const uint4 *M, const uint32_t *Bs, uint32_t s, int lane)
{
    uint32_t B[CW], lin = 0, work = 0;
    PairSums p = {0, 0, 0, 0};
#pragma unroll
    for (int t = 0; t < CW; t++) B[t] = Bs[t];
#pragma unroll 1
    for (int q = 0; q < CW; q++) {
        if ((Bs[q] >> lane) & 1u) {
            uint32_t h[CW], d = 0;
            load_row<CW>(M, (uint32_t)(q << 5) + lane, h);
#pragma unroll
            for (int t = 0; t < CW; t++) {
                h[t] &= B[t];
                d += __popc(h[t]);
                h[t] &= t > q ? kFull : (t == q ? above_bit(lane) : 0u);
            }
            lin += d * (s - 1 - d);
            if (WORK) work += CW * (d + 1);
            pair_words<CW, 0>(M, h, p);
        }
        __syncwarp();
    }
    const uint32_t sum = __reduce_add_sync(kFull, lin + p.both());
    CompCount o;
    o.n = (s * (s - 1) * (s - 2) / 3 - sum) >> 1;
    o.work = WORK ? __reduce_add_sync(kFull, work) : 0u;
    return o;
}

// 4-cliques of the set B (CW words in shared memory, s members), as comp3.  Two passes: over the
// members (degrees, and the codegree planes for N(C4)), then over the edges of the complement, which
// are queued so that every lane holds one: their codegrees, and K4 of the complement as the edges
// among the common neighbours that come later than both ends.  The order of the members is: degree up
// to kHubNarrow first, then the others, by index inside both -- the few members of high degree
// would otherwise carry most of the triangles.
// scr: kMaskWords words, kNbhdList words, kNbhdWords words.
template <int CW, bool WORK>
__device__ __noinline__ CompCount comp4(const uint4 *M, const uint32_t *Bs, uint32_t s, uint32_t *scr, int lane)
{
    constexpr int NP = CW == 1 ? 5 : CW == 2 ? 6 : 7;  // codegrees below 32 CW
    constexpr uint32_t kCap = 2 * kNbhdWords;          // queued edges
    uint8_t *deg = reinterpret_cast<uint8_t *>(scr);   // degree of every member ...
    uint32_t *hub = scr + 64;                          // ... and the members of high degree, by word
    uint16_t *queue = reinterpret_cast<uint16_t *>(scr + kMaskWords + kNbhdList);
    uint32_t B[CW], sd = 0, sl = 0, st = 0, work = 0;
#pragma unroll
    for (int t = 0; t < CW; t++) B[t] = Bs[t];
    __syncwarp();
#pragma unroll 1
    for (int q = 0; q < CW; q++) {
        const uint32_t v = (uint32_t)(q << 5) + lane;
        uint32_t d = 0;
        if ((Bs[q] >> lane) & 1u) {
            uint32_t h[CW];
            load_row<CW>(M, v, h);
#pragma unroll
            for (int t = 0; t < CW; t++) {
                h[t] &= B[t];
                d += __popc(h[t]);
            }
            Planes<CW, NP> pl;
            pl.clear();
#pragma unroll
            for (int t = 0; t < CW; t++) pl.add_word(M, h[t], (uint32_t)t << 5);
            uint32_t s1 = 0;
            const uint32_t cc = pl.template pairs<false>(B, pl.deep(), s1);
            sd += d;
            // per member: terms of 4 N4 (the planes hold the member itself at codegree d)
            sl += 2 * (s - 4) * d * (d - 1) - 4 * (d * (d - 1) * (d - 2) / 6) + cc - d * (d - 1) / 2;
            if (WORK) work += CW * (d + 1);
        }
        deg[v] = (uint8_t)d;
        const uint32_t hb = __ballot_sync(kFull, d > kHubNarrow);
        if (lane == 0) hub[q] = hb;
    }
    __syncwarp();
    // members later than x in word t
    auto later = [&](uint32_t x, uint32_t t) {
        const uint32_t hw = hub[t], up = t > (x >> 5) ? kFull : (t == (x >> 5) ? above_bit(x & 31u) : 0u);
        return ((hub[x >> 5] >> (x & 31u)) & 1u) ? hw & up : hw | up;
    };
    uint32_t n = 0, ones = 0, k4 = 0;
    auto drain = [&]() {
        __syncwarp();
        for (uint32_t r0 = 0; r0 < n; r0 += 32) {
            if (r0 + lane < n) {
                const uint32_t e = queue[r0 + lane], v = e >> 8, y = e & 255u;
                uint32_t rv[CW], D[CW], c = 0;
                load_row<CW>(M, v, rv);
                load_row<CW>(M, y, D);
#pragma unroll
                for (int t = 0; t < CW; t++) {
                    D[t] &= rv[t] & B[t];
                    c += __popc(D[t]);
                }
                const uint32_t dv = deg[v], dy = deg[y];
                st += c;
                sl += 2 * c * (dv + dy) - 4 * (dv - 1) * (dy - 1) - 2 * c * (c - 1);
                if (c >= 2) {
#pragma unroll
                    for (int t = 0; t < CW; t++) D[t] &= later(v, t) & later(y, t);
#pragma unroll
                    for (int t = 0; t < CW; t++) leaf_word<CW, 0>(M, D, D[t], (uint32_t)t << 5, ones, k4);  // pairs twice
                }
                if (WORK) work += CW * (c + 1);
            }
        }
        __syncwarp();
        n = 0;
    };
#pragma unroll 1
    for (int q = 0; q < CW; q++) {
        const uint32_t v = (uint32_t)(q << 5) + lane;
#pragma unroll 1
        for (int t = 0; t < CW; t++) {
            uint32_t y = 0;
            if ((Bs[q] >> lane) & 1u) y = reinterpret_cast<const uint32_t *>(M)[v * 4 + t] & Bs[t] & later(v, t);
            if (!__ballot_sync(kFull, y != 0)) continue;
            const uint32_t cnt = __popc(y), incl = warp_incl_scan(cnt), total = __shfl_sync(kFull, incl, 31);
            if (n + total > kCap) drain();
            uint32_t at = n + incl - cnt;
            for (; y; y &= y - 1) queue[at++] = (uint16_t)((v << 8) | (uint32_t)((t << 5) + __ffs(y) - 1));
            n += total;
        }
    }
    drain();
    sl += 2 * (k4 + __popc(ones));
    sd = __reduce_add_sync(kFull, sd);
    st = __reduce_add_sync(kFull, st);  // codegrees over the edges: 3 t
    sl = __reduce_add_sync(kFull, sl);
    const uint32_t m = sd >> 1;
    CompCount o;
    // 4 C(s,4) = s(s-1)(s-2)(s-3)/6 stays below 2^32 for s <= 128 before the division
    o.n = (s * (s - 1) * (s - 2) * (s - 3) / 6 - 2 * m * (s - 2) * (s - 3) + 2 * m * (m - 1) - 4 * s * (st / 3) + sl) >> 2;
    o.work = WORK ? __reduce_add_sync(kFull, work) : 0u;
    return o;
}

// ---- Wide sets (more than 128 members): rows of nch chunks of four words ---------------------

// Bits of word w above member v.
__device__ __forceinline__ uint32_t above_word(uint32_t v, uint32_t w)
{
    return w > (v >> 5) ? kFull : (w == (v >> 5) ? above_bit(v & 31u) : 0u);
}

// Lane-partial sums for N4 of a wide set B (4 nch words in shared memory, s members), the share of
// warp u0 of ustep warps.  Unit = (member group g, chunk q): the 32 members 32g + lane and their
// codegrees with the 128 members of chunk q; then K4 of the complement as in comp4.
template <bool WORK>
__device__ __noinline__ CompSums comp4_wide(const uint4 *M, uint32_t S, uint32_t nch, const uint32_t *Bs,
                                            uint32_t s, uint32_t ngroups, uint32_t u0, uint32_t ustep,
                                            uint32_t *scr, int lane)
{
    CompSums o = {0, 0, 0, 0, false};
    const uint4 *B4 = reinterpret_cast<const uint4 *>(Bs);
    uint32_t *hubs = scr + 160;  // members of high degree, one word per group
    uint32_t nhubs = 0, nmore = 0, more = 0;
    __syncwarp();
    hubs[lane] = 0;
    __syncwarp();
    for (uint32_t g = 0; g < ngroups; g++) {
        const uint32_t v = (g << 5) + lane;
        uint32_t d = 0;
        if ((Bs[g] >> lane) & 1u)
            for (uint32_t c = 0; c < nch; c++) {
                const uint4 h = M[c * S + v], b = B4[c];
                d += __popc(h.x & b.x) + __popc(h.y & b.y) + __popc(h.z & b.z) + __popc(h.w & b.w);
            }
        o.over |= d > kWideMaxDeg;
        const uint32_t hb = __ballot_sync(kFull, d > kHubWide);
        nhubs += __popc(hb);
        if (lane == 0) hubs[g] = hb;
        const uint32_t mb = __ballot_sync(kFull, d > kNbhdMax);
        nmore += __popc(mb);
        if (lane == (int)g) more = mb;
    }
    __syncwarp();
    if (nhubs > kNbhdMax) {  // too many: draw the line at the largest neighbourhood
        hubs[lane] = more;
        nhubs = nmore;
        __syncwarp();
    }
    o.over = __any_sync(kFull, o.over) || nhubs > kNbhdMax;
    if (o.over) return o;
    const uint32_t nunits = ngroups * nch;
    for (uint32_t u = u0; u < nunits; u += ustep) {
        const uint32_t g = u / nch, q = u - g * nch;
        const uint32_t v = (g << 5) + lane;
        if ((Bs[g] >> lane) & 1u) {
            Planes<4, 8> pl;
            pl.clear();
            const uint4 *Mq = M + q * S;
            uint32_t d = 0;
            for (uint32_t c = 0; c < nch; c++) {
                const uint4 hv = M[c * S + v], bv = B4[c];
                const uint32_t h[4] = {hv.x & bv.x, hv.y & bv.y, hv.z & bv.z, hv.w & bv.w};
                d += __popc(h[0]) + __popc(h[1]) + __popc(h[2]) + __popc(h[3]);
#pragma unroll
                for (int t = 0; t < 4; t++) pl.add_word(Mq, h[t], (c << 7) + (t << 5));
            }
            const uint4 hq4 = M[q * S + v], bq4 = B4[q];
            const uint32_t bq[4] = {bq4.x, bq4.y, bq4.z, bq4.w};
            const uint32_t hq[4] = {hq4.x & bq[0], hq4.y & bq[1], hq4.z & bq[2], hq4.w & bq[3]};
            const bool deep = pl.deep();
            uint32_t s1 = 0, t1 = 0;
            uint32_t cc = pl.template pairs<true>(bq, deep, s1);
            const uint32_t ch = pl.template pairs<true>(hq, deep, t1);
            if (WORK) o.work += 4 * (d + 1);
            if (d) {
                if ((v >> 7) == q) {
                    // once per member: its degree terms, and its own place in the planes
                    o.sd += d;
                    o.sl += 2ull * (s - 4) * d * (d - 1) - 4ull * (d * (d - 1) * (d - 2) / 6) + 2ull * (d - 1) * d;
                    cc -= d * (d - 1) / 2;
                }
                o.st += t1;
                o.sl += 2ull * d * t1 + cc - 2ull * ch - 2ull * (d - 1) * s1;
            }
        }
        __syncwarp();
    }
    // K4 of the complement, at its first member in the order: neighbourhoods of more than kNbhdMin
    // later members by a warp each (comp_nbhd), the others by a lane each on their own rows of at
    // most 16 bits: entry i of lane l in tiny[32 i + l], the member above, its row below
    // members later than x in word w
    auto later = [&](uint32_t x, uint32_t w) {
        const uint32_t hw = hubs[w], up = above_word(x, w);
        return ((hubs[x >> 5] >> (x & 31u)) & 1u) ? hw & up : hw | up;
    };
    const uint32_t *M32 = reinterpret_cast<const uint32_t *>(M);
    uint32_t *tiny = scr + kMaskWords + kNbhdList + lane;
    unsigned long long k4 = 0;
    uint32_t turn = 0;
    for (uint32_t g = 0; g < ngroups; g++) {
        const uint32_t v = (g << 5) + lane;
        uint32_t u = 0;
        if ((Bs[g] >> lane) & 1u)
            for (uint32_t c = 0; c < nch; c++) {
                uint32_t h[4];
                load_row<4>(M + c * S, v, h);
#pragma unroll
                for (int t = 0; t < 4; t++) {
                    const uint32_t w = (c << 2) + t;
                    uint32_t y = h[t] & Bs[w] & later(v, w);
                    for (; y && u <= kNbhdMin; y &= y - 1) {
                        if (u < kNbhdMin) tiny[u << 5] = ((w << 5) + __ffs(y) - 1) << 16;
                        u++;
                    }
                }
            }
        if (g % ustep == u0 && u >= 3 && u <= kNbhdMin) {
            for (uint32_t i = 0; i + 1 < u; i++) {
                const uint32_t yi = tiny[i << 5] >> 16;
                uint32_t row = 0;
                for (uint32_t j = i + 1; j < u; j++) {
                    const uint32_t yj = tiny[j << 5] >> 16;
                    const uint32_t word = M32[((yj >> 7) * S + yi) * 4 + ((yj >> 5) & 3u)];
                    row |= ((word >> (yj & 31u)) & 1u) << j;
                }
                tiny[i << 5] = row;
            }
            uint32_t tri = 0;
            for (uint32_t i = 0; i + 2 < u; i++) {
                const uint32_t row = tiny[i << 5];
                for (uint32_t y = row & ~(1u << (u - 1)); y; y &= y - 1) tri += __popc(row & tiny[(__ffs(y) - 1) << 5]);
            }
            k4 += 2 * tri;
            if (WORK) o.work += u;
        }
        __syncwarp();
        for (uint32_t many = __ballot_sync(kFull, u > kNbhdMin); many; many &= many - 1) {
            if (turn++ % ustep != u0) continue;
            const int src = __ffs(many) - 1;
            const uint32_t x = (g << 5) + src;
            uint32_t uw = 0;
            if ((uint32_t)lane < nch * 4)
                uw = M32[(((uint32_t)lane >> 2) * S + x) * 4 + (lane & 3)] & Bs[lane] & later(x, lane);
            const uint32_t all = __reduce_add_sync(kFull, __popc(uw));
            const CompCount c = comp_nbhd<WORK>(M, S, nch, uw, all, scr, lane);
            k4 += c.n;
            if (WORK) o.work += c.work;
        }
    }
    o.sl += 2 * k4;
    return o;
}

// N4 of a set of s members from its sums.
__device__ __forceinline__ unsigned long long n4_finish(uint32_t s32, uint32_t sd, uint32_t st, unsigned long long sl)
{
    const unsigned long long s = s32, m = sd >> 1;
    return (s * (s - 1) * (s - 2) * (s - 3) / 6 - 2 * m * (s - 2) * (s - 3) + 2 * m * (m - 1) - 4 * s * (st / 6) + sl) >> 2;
}

// As comp4_wide, for N3: lane-partial sum over the warp's share of d(s-1-d) + 2 t (n3_finish).
template <bool WORK>
__device__ __noinline__ CompCount comp3_wide(const uint4 *M, uint32_t S, uint32_t nch, const uint32_t *Bs,
                                             uint32_t s, uint32_t ngroups, uint32_t u0, uint32_t ustep, int lane)
{
    CompCount o = {0, 0};
    const uint4 *B4 = reinterpret_cast<const uint4 *>(Bs);
    const uint32_t nunits = ngroups * nch;
    PairSums p = {0, 0, 0, 0};
    uint32_t lin = 0;
    for (uint32_t u = u0; u < nunits; u += ustep) {
        const uint32_t g = u / nch, q = u - g * nch;
        const uint32_t v = (g << 5) + lane;
        if ((Bs[g] >> lane) & 1u) {
            if ((v >> 7) == q) {
                uint32_t d = 0;
                for (uint32_t c = 0; c < nch; c++) {
                    const uint4 h = M[c * S + v], b = B4[c];
                    d += __popc(h.x & b.x) + __popc(h.y & b.y) + __popc(h.z & b.z) + __popc(h.w & b.w);
                }
                lin += d * (s - 1 - d);
                if (WORK) o.work += 4 * nch;
            }
            // v's later neighbours in chunk c
            auto later = [&](uint32_t c, uint32_t (&h)[4]) {
                const uint4 a = M[c * S + v], b = B4[c];
                const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int t = 0; t < 4; t++) h[t] = x[t] & y[t] & above_word(v, (c << 2) + t);
            };
            if (q >= (g >> 2)) {
                const uint4 *Mq = M + q * S;
                uint32_t D[4];
                later(q, D);
                if (D[0] | D[1] | D[2] | D[3]) {
                    for (uint32_t c = g >> 2; c < q; c++) {
                        uint32_t h[4];
                        later(c, h);
#pragma unroll
                        for (int t = 0; t < 4; t++) {
                            pair_word<4, -1>(Mq, D, h[t], (c << 7) + (t << 5), p);
                            if (WORK) o.work += 4 * __popc(h[t]);
                        }
                    }
                    pair_word<4, 0>(Mq, D, D[0], (q << 7), p);
                    pair_word<4, 1>(Mq, D, D[1], (q << 7) + 32, p);
                    pair_word<4, 2>(Mq, D, D[2], (q << 7) + 64, p);
                    pair_word<4, 3>(Mq, D, D[3], (q << 7) + 96, p);
                    if (WORK) o.work += 3 * (__popc(D[0]) + __popc(D[1]) + __popc(D[2]) + __popc(D[3]));
                }
            }
        }
        __syncwarp();
    }
    o.n = lin + p.both();
    return o;
}

// N3 of a set of s members from its sum.
__device__ __forceinline__ unsigned long long n3_finish(uint32_t s32, uint32_t sum)
{
    const unsigned long long s = s32;
    return ((uint32_t)(s * (s - 1) * (s - 2) / 3) - sum) >> 1;
}

}  // namespace citron

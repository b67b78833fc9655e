// lev.cuh -- edit distance (unit costs) by the bit-parallel recurrence of
// Myers (1999) in the form for global distance (Hyyrö 2001: the top row of the
// dynamic-programming table grows by one per text character, so a 1 is
// shifted into the horizontal positive-delta vector).  The pattern occupies
// W 64-bit words; words above ceil(m/64) are skipped.
//
// lev_myers returns the distance when it is <= k and some value > k
// otherwise; it stops early once the bottom-row value can no longer fall to k.
//
// lev_band is the form for a bound below the word length (Hyyrö 2003): a path
// of cost <= k from (0, 0) to (m, n) stays within floor((k - |m - n|) / 2)
// diagonals of the two that these lie on, at most k + 1 diagonals in all, so
// one word holds a column's part of that band whatever the pattern's length.
// The word slides down a row per column.  Cells outside count as one more than
// their diagonal predecessor, so every value is the cost of some path and the
// ones on a path of cost <= k are exact.  Rows above the table (bits below row
// 0) hold the column number, which makes row 0 grow by one per column.  The
// value on the diagonal of (m, n) never falls: the form stops at the first
// one above k.  Against four 32-bit words of a whole column of 96 symbols, a
// column of the band is one: the leaf stage of 50k
// reads of 96 symbols (18.7 M pairs within 13) takes 2.0 ms instead of 9.0.
#pragma once

#include <stdint.h>

#ifndef CT_HD
#define CT_HD __host__ __device__ __forceinline__
#endif

namespace ct {

inline int lev_words_for(int max_len) {
    int w = (max_len + 63) / 64;
    if (w <= 1) return 1;
    if (w <= 2) return 2;
    if (w <= 4) return 4;
    if (w <= 8) return 8;
    return 16;
}

// peq[c * W + w]: bit j set iff pattern[64 w + j] == c.
template <int W>
__device__ __forceinline__ void lev_build_peq(uint64_t *peq, const uint8_t *pat, int m) {
    for (int i = threadIdx.x; i < 256 * W; i += blockDim.x) peq[i] = 0ull;
    __syncthreads();
    for (int j = threadIdx.x; j < m; j += blockDim.x)
        atomicOr((unsigned long long *)&peq[pat[j] * W + (j >> 6)], 1ull << (j & 63));
}

// Word i of a symbol's match mask, from the 64-bit words (zero outside).
template <int W>
CT_HD uint32_t lev_word(const uint64_t *eq, int i, uint32_t) {
    return (unsigned)i < 2u * W ? (uint32_t)(eq[i >> 1] >> (32 * (i & 1))) : 0u;
}
template <int W>
CT_HD uint64_t lev_word(const uint64_t *eq, int i, uint64_t) {
    return (unsigned)i < (unsigned)W ? eq[i] : 0ull;
}
CT_HD uint32_t lev_window(uint32_t lo, uint32_t hi, int sh) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, sh);
#else
    return sh ? (lo >> sh) | (hi << (32 - sh)) : lo;
#endif
}
CT_HD uint64_t lev_window(uint64_t lo, uint64_t hi, int sh) { return sh ? (lo >> sh) | (hi << (64 - sh)) : lo; }

// The distance if it is <= k, else k + 1; m, n >= 1, |m - n| <= k < bits of T.
// sym(character) is the character's row in peq; cols: columns evaluated.
template <class T, int W, class Sym>
CT_HD int lev_band(const uint64_t *peq, Sym sym, int m, const uint8_t *txt, int n, int k, int &cols) {
    constexpr int B = 8 * sizeof(T), LB = sizeof(T) == 8 ? 6 : 5;
    const int dl = m - n;
    const int c = ((k - (dl < 0 ? -dl : dl)) >> 1) + (dl < 0 ? -dl : 0);  // bit 0: diagonal -c
    const int bf = dl + c;                                                // the bit of (m, n)'s diagonal
    T VP = ~(T)0 << c, VN = 0;
    int score = dl > 0 ? dl : 0;
    constexpr int LEV_PF = 8;  // as in lev_myers
    int nxt[LEV_PF];
#pragma unroll
    for (int u = 0; u < LEV_PF; ++u) nxt[u] = u < n ? (int)txt[u] : 0;
    for (int j0 = 0; j0 < n; j0 += LEV_PF) {
        int blk[LEV_PF];
#pragma unroll
        for (int u = 0; u < LEV_PF; ++u) {
            blk[u] = nxt[u];
            nxt[u] = j0 + LEV_PF + u < n ? (int)txt[j0 + LEV_PF + u] : 0;
        }
#pragma unroll
        for (int u = 0; u < LEV_PF; ++u) {
            const int j = j0 + u;
            if (j >= n) break;
            const uint64_t *eqr = peq + sym(blk[u]) * W;
            const int base = j - c, wi = base >> LB;  // pattern index of bit 0 (rows are 1-based)
            const T Eq = lev_window(lev_word<W>(eqr, wi, T()), lev_word<W>(eqr, wi + 1, T()), base & (B - 1));
            const T D0 = (((Eq & VP) + VP) ^ VP) | Eq | VN;
            const T HP = VN | ~(D0 | VP), HN = D0 & VP;
            score += (int)((D0 >> bf) & 1) ^ 1;
            if (score > k) {
                cols = j + 1;
                return k + 1;
            }
            VP = HN | ~((D0 >> 1) | HP);
            VN = (D0 >> 1) & HP;
        }
    }
    cols = n;
    return score;
}

template <int W>
CT_HD int lev_myers(const uint64_t *peq, int m, const uint8_t *txt, int n, int k) {
    if (k < 0) return 0 == m && 0 == n ? 0 : k + 1;
    int dl = m > n ? m - n : n - m;
    if (dl > k) return k + 1;
    if (m == 0) return n;
    if (n == 0) return m;
    if (W > 1 && k < 64) {
        int cols;
        auto same = [](int s) { return s; };
        return k < 32 ? lev_band<uint32_t, W>(peq, same, m, txt, n, k, cols)
                      : lev_band<uint64_t, W>(peq, same, m, txt, n, k, cols);
    }
    const int nw = (m + 63) >> 6;
    const int hw = (m - 1) >> 6;
    const uint64_t hbit = 1ull << ((m - 1) & 63);
    uint64_t Pv[W], Mv[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        Pv[w] = ~0ull;
        Mv[w] = 0ull;
    }
    int score = m;
    // the text is read a block of LEV_PF characters ahead of the recurrence:
    // independent loads, so that a step does not wait on its own load
    constexpr int LEV_PF = 8;
    int nxt[LEV_PF];
#pragma unroll
    for (int u = 0; u < LEV_PF; ++u) nxt[u] = u < n ? (int)txt[u] : 0;
    for (int j0 = 0; j0 < n; j0 += LEV_PF) {
        int blk[LEV_PF];
#pragma unroll
        for (int u = 0; u < LEV_PF; ++u) {
            blk[u] = nxt[u];
            nxt[u] = j0 + LEV_PF + u < n ? (int)txt[j0 + LEV_PF + u] : 0;
        }
#pragma unroll
        for (int u = 0; u < LEV_PF; ++u) {
            const int j = j0 + u;
            if (j >= n) break;
            const uint64_t *eqr = peq + blk[u] * W;
            uint64_t carry = 0ull, hp_in = 1ull, hn_in = 0ull;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (w < nw) {
                    uint64_t Eq = eqr[w];
                    uint64_t pv = Pv[w], mv = Mv[w];
                    uint64_t Xv = Eq | mv;
                    uint64_t t = Eq & pv;
                    uint64_t s1 = t + pv;
                    uint64_t c1 = s1 < t ? 1ull : 0ull;
                    uint64_t s2 = s1 + carry;
                    uint64_t c2 = s2 < s1 ? 1ull : 0ull;
                    carry = c1 | c2;
                    uint64_t Xh = (s2 ^ pv) | Eq;
                    uint64_t Ph = mv | ~(Xh | pv);
                    uint64_t Mh = pv & Xh;
                    if (w == hw) {
                        if (Ph & hbit) ++score;
                        else if (Mh & hbit) --score;
                    }
                    uint64_t ph_out = Ph >> 63, mh_out = Mh >> 63;
                    Ph = (Ph << 1) | hp_in;
                    Mh = (Mh << 1) | hn_in;
                    hp_in = ph_out;
                    hn_in = mh_out;
                    Pv[w] = Mh | ~(Xv | Ph);
                    Mv[w] = Ph & Xv;
                }
            }
            if (score - (n - 1 - j) > k) return k + 1;
        }
    }
    return score;
}

}  // namespace ct

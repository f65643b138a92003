// Super-k-mer counting: what the kernels of mh_super.cu and the lookups of
// the mercy step share.  See mh_super.cu for the method.
#pragma once

#include "mh_internal.cuh"

namespace mh {

// Minimizer length of windows of K1 symbols (0: too short for it).  The
// kernel takes window minima from blocks of 8 positions, so a window has at
// least 8 minimizer positions; within that, longer minimizers spread the
// windows over more bins and shorter ones give longer super-k-mers.  (Windows
// of 16 to 20 symbols would have room for minimizers of 9 to 13; those were not
// measured, and such sets are counted by units.)
__host__ __device__ inline int super_m(int K1) { return K1 >= 32 ? 16 : K1 >= 26 ? 14 : K1 >= 21 ? 12 : 0; }

// Windows of many words: a bin by one minimizer would get whole runs of about
// w / 2 windows at a time, times the coverage, more than a bin's table holds
// where a genome is abundant.  From 48 words on, the window's bin is by the
// smallest hash of its first and of its last half words together (swapped in
// the reverse complement, so combined by a sum): runs of about w / 8 windows.
// 0: by one minimizer, else the words of a half.
__host__ __device__ inline int super_half(int K1) {
    const int w = K1 - super_m(K1) + 1;
    return w >= 48 ? w / 2 : 0;
}

// Order of the canonical minimizer-length words: an affine map of 32-bit
// words (one multiply-add), so that runs of one symbol are not the smallest.
__host__ __device__ __forceinline__ uint32_t super_hash(uint32_t c) { return c * 0x9E3779B1u + 0x7F4A7C15u; }

// Bin of a window whose smallest hash is h.  The smallest hashes are small
// numbers, so they are mixed again (the two-multiply 32-bit mixer
// "lowbias32", C. Wellons, 2018).
__host__ __device__ __forceinline__ uint32_t super_mix(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7FEB352Du;
    x ^= x >> 15;
    x *= 0x846CA68Bu;
    return x ^ (x >> 16);
}

// Slots of a bin's table, and the windows an average bin aims at: smaller bins
// cost more rounds of barriers, larger ones leave more to the rest (3 Gbp at
// k = 31 counted in 19.6, 18.9 and 18.7 ms aiming at 2,400, 2,800 and 3,100, the
// last too full where all keys are distinct; 3 M reads at k = 61 in 7.54, 7.68
// and 7.84 at 1,200, 1,400 and 1,550, the multiple-k iteration 58.7 and 58.4 at
// the first two).
template <int NW>
struct SuperCfg {
    static constexpr int kLog = NW == 1 ? 12 : 11;
    static constexpr int kSlots = 1 << kLog;
    static constexpr uint32_t kTarget = NW == 1 ? 2800 : 1400;
    static constexpr int kWords = kSlots / 32;
    static constexpr int kRecWords = 4 * NW;  // 16-symbol words of a record: runs are cut to fit them
};

// First slot of a mixed key: an even one, since a table is probed a pair of
// slots (16 bytes) at a time, in order.
template <int NW>
__device__ __forceinline__ uint32_t super_slot(const Key<NW>& m) {
    return (uint32_t)(m.w[NW - 1] >> (64 - SuperCfg<NW>::kLog)) & ~1u;
}

// The count spectrum in bins.  Bin b's entries (mixed key, length) are those
// of its table in slot order, from off[b]; idx[b * kWords + s / 32] holds
// the occupancy bits of slots s and the entries of the bin before them, so a
// key's slot gives its place.  off[b] = kSuperDeferred: the bin's entries
// are among the last ones, [n_main, n), which are sorted by mixed key.
constexpr uint64_t kSuperDeferred = ~0ull;
struct SuperIndex {
    const uint64_t* off = nullptr;
    const uint2* idx = nullptr;
    uint32_t n_bins = 0;
    int m = 0;
    uint64_t n_main = 0, n = 0;
};

// What decides the bin of a window x of K1 symbols with reverse complement
// r: the smallest hash over its canonical minimizer-length words, or (halves)
// the sum of its halves' mixed smallest hashes.
template <int NW>
__device__ __forceinline__ uint32_t super_min(Key<NW> x, Key<NW> r, int K1, int m) {
    const uint32_t mask = m == 16 ? 0xFFFFFFFFu : (1u << (2 * m)) - 1u;
    // word j from the end: x's symbols [K1 - m - j, K1 - j), r's [j, j + m)
    uint32_t best = 0xFFFFFFFFu, last = 0xFFFFFFFFu;
    const int w = K1 - m + 1, half = super_half(K1);
    const int top = 2 * (K1 - m);
    if constexpr (NW == 1) {
        for (int j = 0; j < w; j++) {
            const uint32_t f = (uint32_t)(x.w[0] >> (2 * j)) & mask, g = (uint32_t)(r.w[0] >> (top - 2 * j)) & mask;
            const uint32_t h = super_hash(f < g ? f : g);
            best = h < best ? h : best;
        }
    } else {
        // x moved down and r, from the top of its words, up by a symbol a step
        // (gaps of 1 M reads at k = 61 walked in 2.36 ms; with shifts of both by
        // a variable at every step 2.97)
        r = key_shl<NW>(r, 64 * NW - 2 * K1);
        for (int j = 0; j < w; j++) {
            const uint32_t f = (uint32_t)x.w[0] & mask, g = (uint32_t)(r.w[NW - 1] >> 32) >> (32 - 2 * m);
            const uint32_t h = super_hash(f < g ? f : g);
            if (!half || j < half) best = h < best ? h : best;
            if (half && j >= w - half) last = h < last ? h : last;
#pragma unroll
            for (int i = 0; i < NW; i++) x.w[i] = x.w[i] >> 2 | (i + 1 < NW ? x.w[i + 1 < NW ? i + 1 : 0] << 62 : 0ull);
#pragma unroll
            for (int i = NW - 1; i >= 0; i--) r.w[i] = r.w[i] << 2 | (i ? r.w[i ? i - 1 : 0] >> 62 : 0ull);
        }
    }
    return half ? super_mix(best) + super_mix(last) : best;
}

// Run length of a window (x, its reverse complement r) in the spectrum, 0 if
// absent; mk is the mixed canonical key.
template <int NW>
__device__ __forceinline__ uint32_t super_find(const SuperIndex& S, const uint64_t* __restrict__ spec,
                                               const uint32_t* __restrict__ len, const Key<NW>& x, const Key<NW>& r,
                                               const Key<NW>& mk, int K1) {
    using C = SuperCfg<NW>;
    const uint32_t b = __umulhi(super_mix(super_min<NW>(x, r, K1, S.m)), S.n_bins);
    const uint64_t o = S.off[b];
    if (o == kSuperDeferred) {
        uint64_t lo = S.n_main, hi = S.n;
        while (lo < hi) {
            const uint64_t mid = lo + (hi - lo) / 2;
            if (key_less<NW>(load_key<NW>(spec, mid), mk)) lo = mid + 1; else hi = mid;
        }
        return lo < S.n && key_eq<NW>(load_key<NW>(spec, lo), mk) ? len[lo] : 0u;
    }
    uint32_t s = super_slot<NW>(mk);
    for (int t = 0; t < C::kSlots; t++) {
        const uint2 v = S.idx[(uint64_t)b * C::kWords + (s >> 5)];
        if (!((v.x >> (s & 31)) & 1u)) return 0;
        const uint64_t e = o + v.y + __popc(v.x & ((1u << (s & 31)) - 1u));
        if (key_eq<NW>(load_key<NW>(spec, e), mk)) return len[e];
        s = (s + 1) & (C::kSlots - 1);
    }
    return 0;
}

// Whether n windows of K1 symbols are counted by super-k-mers.
bool use_super(uint64_t n, int K1);

// False (and nothing done): too many windows would be left to the rest, the
// set is one for the unit counting.
template <int NW>
bool super_count(mh_ctx* ctx, const mh_reads* reads, int k, int d, uint64_t n, mh_kmers* out);

}  // namespace mh

// Counting by super-k-mers: the count of mh_count_kmers (paper, Sec. 2,
// third paragraph) for sets whose keys would otherwise be moved by radix
// passes.
//
// Neighbouring windows of a read share all but one symbol, so moving a key a
// window (8 to 32 bytes, several passes) moves each base some K1 times.  Here
// a window goes to the bin of its minimizer, the smallest hash among its
// canonical m-symbol words (Roberts et al., 2004, Bioinformatics 20:3363;
// binning k-mers by them: Li et al., MSPKmerCounter, 2015, and KMC 2, Deorowicz et al., 2015).
// A window and its reverse complement have the same canonical words, so equal
// canonical keys meet in one bin; neighbours mostly share their minimizer, so
// a run of them (a super-k-mer, 2 / (w + 1) a window for w words a window)
// travels as one 8-byte record: where the run starts in the packed reads and
// its number of windows.
//
//   split    tiles of 2,048 positions of the packed stream: the hashes of the
//            tile's words, the smallest over each window, the runs; a run's
//            record goes to its bin's slots at the rank one 64-bit atomic on
//            the bin's counters gives (records low, windows high)
//   place    the records past their bin's slots (half as many again as the
//            mean), from a list, to places after a scan
//   count    a CTA per bin: equal records merged, then 32 windows at a time
//            a warp; a window's mixed canonical key goes into a hash table
//            in shared memory; then each warp writes its eighth of the table
//            (the spectrum, and the kept keys of both strands) at places
//            reserved by one atomic each, and clears it for the next bin.  The kept keys are sorted afterwards, so the
//            bins' order does not matter.
//   rest     bins with more windows than one CTA should take, or whose keys
//            do not fit the table, are expanded to keys and counted by the
//            unit counting (mh_group.cu); their spectrum goes last.  Where too
//            much would go that way the whole set does (super_lost)
//
// What bounds it: the waits between a bin's barriers and instruction issue (a
// hash insertion a window), not memory: a window moves about 2 bytes of
// records and 4 of outputs instead of 8 to 32 a pass.  Equal records are
// counted once with their number (keys of one word: their records are short
// against a read, so most recur whole), which at 3 Gbp and k = 31 takes the
// count from 24.6 to 21.4 ms (18.9 since bins without a palindrome skip the
// search for them and a lane lists 16 slots at once); for wider keys most runs end with their read,
// and it would cost more than it saves.  3 Gbp, k = 31, 2.38 G windows: split
// 7.3 ms (67 thread instructions a position), count 18.9, where the
// extraction, two passes, the units and their compaction took 18.8 + 28 + 22.3
// + 5.2; 3 M reads of 100-150 bp at k = 61: 4.5 ms for 15.2.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <vector>

#include "mh_super.cuh"

namespace mh {

namespace {

constexpr int kSplitTile = 2048;                      // positions a CTA
constexpr int kSplitHalo = 128;                       // positions past it that its windows reach (w - 1 <= 112)
constexpr int kSplitWords = kSplitTile / 16 + 12;     // packed words a CTA reads
constexpr int kSplitMaxRecs = kSplitTile;
constexpr int kHashPad = (kSplitTile + kSplitHalo) / 8 * 9;  // one word of padding after 8: no bank conflicts
constexpr int kNwinBits = 12;                         // a record: start << 12 | windows (at most 2,048)
static_assert(kSplitTile < (1 << kNwinBits), "a run fits a record");

enum { T_SPEC = 0, T_SOLID = 1, T_PALIN = 2, T_DEF = 3, T_DEFWIN = 4, T_RECS = 5, T_DONE = 6, T_FULL = 7, T_LOST = 8, T_N = 9 };

}  // namespace

// first[t] = first fragment f in [0, F] with offs[f] >= t * kSplitTile.
__global__ void super_tiles_kernel(const uint64_t* __restrict__ offs, uint64_t F, uint64_t n_tiles,
                                   uint64_t* __restrict__ first) {
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < n_tiles;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t q = t * kSplitTile;
        uint64_t lo = 0, hi = F;
        while (lo < hi) {
            const uint64_t mid = lo + (hi - lo) / 2;
            if (offs[mid] < q) lo = mid + 1; else hi = mid;
        }
        first[t] = lo;
    }
}

// HALVES: bins by the smallest hashes of a window's halves (super_half).
template <int M, bool HALVES>
__global__ void __launch_bounds__(256) super_split_kernel(const uint32_t* __restrict__ packed, uint64_t n_words,
                                                          const uint64_t* __restrict__ offs, uint64_t F,
                                                          const uint64_t* __restrict__ first, int k, uint32_t n_bins,
                                                          uint32_t most, uint32_t slots, uint64_t* __restrict__ rec,
                                                          uint64_t* __restrict__ more, uint2* __restrict__ place,
                                                          uint64_t cap, unsigned long long* __restrict__ bins,
                                                          unsigned long long* __restrict__ totals) {
    constexpr int T = kSplitTile;
    constexpr uint32_t mask = M == 16 ? 0xFFFFFFFFu : (1u << (2 * M)) - 1u;
    __shared__ uint32_t words[kSplitWords];
    __shared__ __align__(16) uint32_t hash[kHashPad];  // then the positions' minima
    __shared__ uint32_t bmin[(T + kSplitHalo) / 8];
    __shared__ uint32_t inv[T / 32], stop[T / 32];     // no window starts here; a run ends before here
    __shared__ uint16_t hpos[kSplitMaxRecs];
    __shared__ uint32_t edge[8], scratch[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * T;
    const int words_all = k + 1 - M + 1;               // words a window
    const int w = HALVES ? words_all / 2 : words_all;  // words a minimum is taken over
    __shared__ uint32_t hmin[HALVES ? (T / 8 + 8) * 9 : 1];
    for (int i = tid; i < kSplitWords; i += 256) {
        const uint64_t g = base / 16 + i;
        words[i] = g < n_words ? packed[g] : 0u;
    }
    if (tid < T / 32) inv[tid] = 0;
    __syncthreads();
    // no window starts in the k positions before a fragment's start (or the
    // stream's end, offs[F])
    for (uint64_t f = first[blockIdx.x] + tid; f <= F; f += 256) {
        const uint64_t s64 = offs[f] - base;
        if (s64 > (uint64_t)(T + k)) break;
        // (past the stream's end there is none either)
        const int s = (int)s64, lo = s > k ? s - k : 0, hi = (s < T && f < F) ? s : T;
        for (int q = lo; q < hi;) {
            const int e = min(hi, (q | 31) + 1);
            const uint32_t m = (e - q == 32) ? 0xFFFFFFFFu : ((1u << (e - q)) - 1u) << (q & 31);
            atomicOr(&inv[q >> 5], m);
            q = e;
        }
    }
    // hashes of 8 positions a thread, and their smallest
    uint32_t h[8];
    const int n_blk = 256 + (words_all + (HALVES ? 20 : 6)) / 8;
    for (int blk = tid; blk < n_blk; blk += 256) {
        const int wi = blk >> 1;
        const uint64_t hi = ((uint64_t)words[wi] << 32) | words[wi + 1];
        const uint64_t x = (blk & 1) ? (hi << 16) | (words[wi + 2] >> 16) : hi;  // 32 symbols
        const uint64_t y = rev2_u64(~x);
        uint32_t v[8], b = 0xFFFFFFFFu;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const uint32_t f = (uint32_t)(x >> (64 - 2 * M - 2 * j)) & mask, g = (uint32_t)(y >> (2 * j)) & mask;
            v[j] = super_hash(min(f, g));
            hash[blk * 9 + j] = v[j];
            b = min(b, v[j]);
        }
        bmin[blk] = b;
        if (blk == tid) {
#pragma unroll
            for (int j = 0; j < 8; j++) h[j] = v[j];
        }
    }
    __syncthreads();
    // the smallest of w positions from each of 8 on (w >= 8): the block's own
    // positions from there on, the positions all eight share (whole blocks
    // by their minima), and the ones after
    uint32_t mh[8];
    auto minima = [&](int blk, const uint32_t h[8], uint32_t out[8]) {
        uint32_t mid = 0xFFFFFFFFu;
        const int nb = (w - 8) >> 3;
        for (int q = 1; q <= nb; q++) mid = min(mid, bmin[blk + q]);
        for (int p = 8 + 8 * nb; p < w; p++) mid = min(mid, hash[blk * 9 + p + (p >> 3)]);
        out[7] = h[7];
#pragma unroll
        for (int i = 6; i >= 0; i--) out[i] = min(h[i], out[i + 1]);
        out[0] = min(out[0], mid);
#pragma unroll
        for (int i = 1; i < 8; i++) {
            const int p = w - 1 + i;
            mid = min(mid, hash[blk * 9 + p + (p >> 3)]);
            out[i] = min(out[i], mid);
        }
    };
    if constexpr (HALVES) {
        const int shift = words_all - w;  // from the first half to the last
        for (int blk = tid; blk < 256 + (shift + 7) / 8; blk += 256) {
            uint32_t v[8], o[8];
#pragma unroll
            for (int j = 0; j < 8; j++) v[j] = hash[blk * 9 + j];
            minima(blk, v, o);
#pragma unroll
            for (int j = 0; j < 8; j++) {
                o[j] = super_mix(o[j]);
                hmin[blk * 9 + j] = o[j];
                if (blk == tid) mh[j] = o[j];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int p = shift + i;
            mh[i] += hmin[tid * 9 + p + (p >> 3)];
        }
    } else {
        minima(tid, h, mh);
    }
    // heads: windows whose left neighbour is none or has another minimizer
    if (lane == 31) edge[warp] = mh[7];
    __syncthreads();
    const uint32_t vb = ~(uint32_t)reinterpret_cast<const uint8_t*>(inv)[tid] & 0xFFu;
    const bool pv = tid > 0 && !(reinterpret_cast<const uint8_t*>(inv)[tid - 1] >> 7);
    uint32_t pm = __shfl_up_sync(0xFFFFFFFFu, mh[7], 1);
    if (lane == 0 && warp > 0) pm = edge[warp - 1];
    uint32_t same = (pv && pm == mh[0]) ? 1u : 0u;
#pragma unroll
    for (int i = 1; i < 8; i++) same |= (((vb >> (i - 1)) & 1u) && mh[i] == mh[i - 1]) ? 1u << i : 0u;
    const uint32_t hm = vb & ~same;
    reinterpret_cast<uint8_t*>(stop)[tid] = (uint8_t)(hm | ~vb);
    uint32_t total;
    uint32_t at = block_excl_scan_256(__popc(hm), scratch, &total);
    reinterpret_cast<uint4*>(hash)[2 * tid] = make_uint4(mh[0], mh[1], mh[2], mh[3]);
    reinterpret_cast<uint4*>(hash)[2 * tid + 1] = make_uint4(mh[4], mh[5], mh[6], mh[7]);
    for (uint32_t left = hm; left; left &= left - 1) hpos[at++] = (uint16_t)(tid * 8 + __ffs(left) - 1);
    __syncthreads();
    // a thread per run
    for (uint32_t j = tid; j < total; j += 256) {
        const uint32_t q = hpos[j];
        const uint32_t b = __umulhi(super_mix(hash[q]), n_bins);
        // (a run of more windows than a record may have, in a repeat, gives
        // several)
        uint32_t left = next_bit(stop, q + 1, T) - q, at = 0;
        while (left) {
            const uint32_t nw = min(left, most);
            const uint32_t r = (uint32_t)atomicAdd(&bins[b], 1ull | ((unsigned long long)nw << 32));
            const uint64_t v = ((base + q + at) << kNwinBits) | nw;
            if (r < slots) {
                rec[(uint64_t)b * slots + r] = v;
            } else {
                const uint64_t o = atomicAdd(&totals[T_RECS], 1ull);
                if (o < cap) {
                    more[o] = v;
                    place[o] = make_uint2(b, r - slots);
                }
            }
            left -= nw;
            at += nw;
        }
    }
}

// over[b] = records of bin b past its slots.
__global__ void super_over_kernel(const unsigned long long* __restrict__ bins, uint32_t n_bins, uint32_t slots,
                                  uint32_t* __restrict__ over) {
    for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < n_bins; b += gridDim.x * blockDim.x) {
        const uint32_t r = (uint32_t)bins[b];
        over[b] = r > slots ? r - slots : 0u;
    }
}

// Each listed record to its place past its bin's slots (nothing if the list
// overflowed).
__global__ void super_place_kernel(const uint64_t* __restrict__ more, const uint2* __restrict__ place, uint64_t cap,
                                   const unsigned long long* __restrict__ totals, const uint64_t* __restrict__ off,
                                   uint64_t* __restrict__ out) {
    const uint64_t n = totals[T_RECS];
    if (n > cap) return;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint2 p = place[i];
        out[off[p.x] + p.y] = more[i];
    }
}

// The records of the bins: bin b's first `slots` at rec[b * slots], the others
// at more[off[b]]; bins[b] counts them (low half) and their windows (high).
struct SuperRecs {
    const uint64_t* rec;
    const uint64_t* more;
    const uint64_t* off;
    const unsigned long long* bins;
    uint32_t slots;
    __device__ __forceinline__ uint64_t at(uint64_t b, uint64_t o, uint32_t i) const {
        return i < slots ? rec[b * slots + i] : more[o + i - slots];
    }
};

// Two table slots, read again each time (other lanes fill them).
__device__ __forceinline__ ulonglong2 ld_pair(const uint64_t* p) {
    ulonglong2 v;
    asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];"
                 : "=l"(v.x), "=l"(v.y)
                 : "r"((uint32_t)__cvta_generic_to_shared(p))
                 : "memory");
    return v;
}

// The windows of 32 records (a lane each; n windows in all), 32 at a time:
// body(valid, position of this lane's window) for every step.
template <class Body>
__device__ __forceinline__ uint32_t for_windows(uint64_t rec, const Body& body) {
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (uint32_t)rec & ((1u << kNwinBits) - 1u);
    uint32_t incl = nw;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t start = incl - nw, tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
    const uint64_t adj = (rec >> kNwinBits) - start;
    uint32_t before = 0;
    for (uint32_t j0 = 0; j0 < tot; j0 += 32) {
        // the record of window j0 + lane: the last one that starts at or before it
        const uint32_t rel = start - j0;
        const uint32_t m = __reduce_or_sync(0xFFFFFFFFu, (nw && rel < 32u) ? 1u << rel : 0u);
        const int idx = (int)(before + __popc(m & (0xFFFFFFFFu >> (31 - lane)))) - 1;
        before += __popc(m);
        const uint64_t p = __shfl_sync(0xFFFFFFFFu, adj, idx) + j0 + lane;
        body(j0 + lane < tot, j0 + lane, p);
    }
    return tot;
}

// Shared memory of a bin's CTA: the table (top words, other words, counts)
// and the records of a round (starts among the round's windows, symbols), over
// which the list of occupied slots goes afterwards.  For one word 56 KB, so
// that four CTAs share an SM.
template <int NW>
struct SuperSmem {
    static constexpr int kSlots = SuperCfg<NW>::kSlots;
    static constexpr int kRecs = NW == 1 ? 448 : 512 / NW;  // records a round
    static constexpr int kRW = SuperCfg<NW>::kRecWords;    // words a record's symbols take
    static constexpr int kMost = kSlots / 128 * 108;       // entries a table may hold (0.84 of its slots)
    static constexpr int kRegion = kSlots / 8;             // a warp's share of the slots
    static constexpr bool kAlike = NW == 1;                // equal records are counted once, with their number
    static constexpr int kOwners = 1024;
    static constexpr size_t kFp = 0;
    static constexpr size_t kLow = kFp + sizeof(uint64_t) * kSlots;
    static constexpr size_t kCnt = kLow + sizeof(uint64_t) * (NW - 1) * kSlots;
    static constexpr size_t kSym = kCnt + (NW == 1 ? sizeof(uint16_t) : sizeof(uint32_t)) * kSlots;
    static constexpr size_t kStart = kSym + sizeof(uint32_t) * kRW * kRecs;
    static constexpr size_t kMul = kStart + sizeof(uint32_t) * kRecs;
    static constexpr size_t kOwn = kMul + (kAlike ? sizeof(uint32_t) * kRecs : 0);
    static constexpr size_t kRecEnd = kOwn + (kAlike ? sizeof(uint32_t) * kOwners : 0);
    static constexpr size_t kListEnd = kSym + sizeof(uint16_t) * kSlots;
    static constexpr size_t kBytes = kRecEnd > kListEnd ? kRecEnd : kListEnd;
    static_assert(!kAlike || (kRecs <= kOwners / 2 && kRecs * (16 * kRW) < (1 << 16)), "records and windows of a round");
    static_assert(kSym % 16 == 0 && kOwn % 16 == 0, "aligned");
};

// Whether w windows of bins that filled their tables, of `done` counted or left
// over, are so many that the set had better be counted by units: more than 3 in
// 5, of keys of two words.  The insertions into those bins are lost, and their
// windows are written out as keys, sorted and counted all the same (a bin of
// more windows than it may have is left over before that).  By unit counting
// and by bins with what they leave over, k = 61: 5.4 and 7.2 ms with 63 % of the
// windows in full tables (300 kbp 300 times; 6.0 given up), 13.4 and 16.3 with
// 79 % (100 kbp 1,000 times; 14.1), 3.5 and 4.0 with 44 %, 5.8 and 5.6 with 54 %,
// 4.7 and 4.1 with 22 %.  Of four words 4.8 and 5.3 ms with 58 %, 9.8 and 10.3
// with 71 %, 10.2 and 10.1 with 67 %: as much as giving up costs.  Keys of one
// word are faster by bins at any depth.
constexpr uint32_t kLostBins = 32;
__host__ __device__ inline bool super_lost(uint64_t w, uint64_t done) { return 5 * w > 3 * done; }

// A CTA per bin.  The table's first word is a mixed key's top word (the whole
// key of one word); kEmpty marks a free slot: the mixed image of the
// all-ones key, which is not canonical, for one word (wider keys whose top
// word equals it are left to the rest).  Wider keys' other words are
// stored beside it by the lane that claimed the slot, which then sets the
// count's top bit; a lane that finds its top word waits for that bit
// (bounded) and compares the rest.  A key that finds no place within
// probe_max slots leaves the bin to the rest, as do more than kMost entries;
// where that takes too much of a set of give_up windows, the CTAs stop and
// totals[T_LOST] says so (0: they never do).
template <int NW>
__global__ void __launch_bounds__(256, NW == 1 ? 4 : NW == 2 ? 4 : 3)
    super_count_kernel(const uint32_t* __restrict__ packed, SuperRecs recs, uint32_t b0, uint32_t b1,
                       uint64_t rec_cap, int K1, int d, uint64_t give_up,
                       uint32_t hot, int probe_max, uint64_t spec_cap, uint64_t* __restrict__ spec_k,
                       uint32_t* __restrict__ spec_len, uint64_t solid_cap, uint64_t* __restrict__ solid_k,
                       uint32_t* __restrict__ solid_c, uint64_t* __restrict__ soff, uint2* __restrict__ sidx,
                       ulonglong2* __restrict__ deferred, unsigned long long* __restrict__ totals) {
    using C = SuperCfg<NW>;
    using L = SuperSmem<NW>;
    constexpr uint64_t kEmpty = 0ull - kMixC1;
    constexpr uint32_t kReady = 0x80000000u;
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t* fp = reinterpret_cast<uint64_t*>(smem + L::kFp);
    uint64_t* low = reinterpret_cast<uint64_t*>(smem + L::kLow);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smem + L::kCnt);
    uint32_t* sym = reinterpret_cast<uint32_t*>(smem + L::kSym);
    uint32_t* start = reinterpret_cast<uint32_t*>(smem + L::kStart);
    __shared__ uint32_t over, any_palin, lost;
    __shared__ uint32_t scratch[8], wsol[8], went[8];
    __shared__ uint64_t base[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    uint16_t* list = reinterpret_cast<uint16_t*>(smem + L::kSym) + warp * L::kRegion;  // the warp's occupied slots
    if (totals[T_RECS] > rec_cap) return;
    uint32_t palins = 0;

    // exclusive prefix over the CTA (scratch is free again after the next barrier)
    auto scan = [&](uint32_t v, uint32_t* total) {
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) scratch[warp] = x;
        __syncthreads();
        uint32_t before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < 8; w++) {
            before += w < warp ? scratch[w] : 0u;
            all += scratch[w];
        }
        *total = all;
        return before + x - v;
    };
    uint32_t* mul = reinterpret_cast<uint32_t*>(smem + L::kMul);
    uint32_t* owner = reinterpret_cast<uint32_t*>(smem + L::kOwn);
    // counts: 16 bits for one word (a bin has fewer windows than that)
    auto add = [&](uint32_t at, uint32_t c) {
        if constexpr (NW == 1) atomicAdd(&cnt[at >> 1], c << (16 * (at & 1)));
        else atomicAdd(&cnt[at], c);
    };
    auto count_at = [&](uint32_t at) -> uint32_t {
        if constexpr (NW == 1) return reinterpret_cast<const uint16_t*>(cnt)[at];
        else return cnt[at] & ~kReady;
    };
    auto insert = [&](const Key<NW>& mk, uint32_t c) {
        const uint64_t t = mk.w[NW - 1];
        if (NW > 1 && t == kEmpty) {
            over = 1;
            return;
        }
        uint32_t s = super_slot<NW>(mk);
        for (int probe = 0; probe < probe_max; probe++) {
            const ulonglong2 v = ld_pair(fp + s);
            // the first of the pair that holds the key or nothing
            uint32_t at = (v.x == t || v.x == kEmpty) ? s : s + 1;
            uint64_t cur = at == s ? v.x : v.y;
            if (cur == kEmpty) {
                cur = atomicCAS((unsigned long long*)&fp[at], (unsigned long long)kEmpty, (unsigned long long)t);
                if constexpr (NW > 1) {
                    if (cur == kEmpty) {
#pragma unroll
                        for (int q = 0; q < NW - 1; q++) low[q * C::kSlots + at] = mk.w[q];
                        __threadfence_block();
                        add(at, c | kReady);
                        return;
                    }
                } else if (cur == kEmpty) {
                    cur = t;
                }
            }
            if (cur == t) {
                bool same = true;
                if constexpr (NW > 1) {
                    int spins = 0;
                    while (!(*(volatile uint32_t*)&cnt[at] & kReady))
                        if (++spins > 4096) {
                            over = 1;
                            return;
                        }
                    __threadfence_block();
#pragma unroll
                    for (int q = 0; q < NW - 1; q++) same &= *(volatile uint64_t*)&low[q * C::kSlots + at] == mk.w[q];
                }
                if (same) {
                    add(at, c);
                    return;
                }
                over = 1;  // two wide keys with the same top word
                return;
            }
            // (a slot another lane has just taken: the pair again)
            if (at != s && cur == v.y) s = (s + 2) & (C::kSlots - 1);
        }
        over = 1;
    };

    // the next bin's counters and first round of records, fetched while the
    // bin before it is written out (those past a bin's slots later)
    constexpr int R = (L::kRecs + 255) / 256;  // records a thread
    uint64_t next_have = 0, next_off = 0, next_rr[R];
    auto fetch = [&](uint32_t b) {
        if (b >= b1) return;
        next_have = recs.bins[b];
        next_off = recs.off[b];
#pragma unroll
        for (int q = 0; q < R; q++) {
            const uint32_t i = R * tid + q;
            if (i < recs.slots) next_rr[q] = recs.rec[(uint64_t)b * recs.slots + i];
        }
    };
    auto next_hot = [&]() -> uint32_t { return (uint32_t)(next_have >> 32) > (NW == 1 ? min(hot, 0xFFFFu) : hot); };
    fetch(b0 + blockIdx.x);
    if (tid == 0) {
        over = next_hot();
        any_palin = 0;
        lost = 0;
    }
    for (int i = tid; i < C::kSlots / 2; i += 256)
        reinterpret_cast<ulonglong2*>(fp)[i] = make_ulonglong2(kEmpty, kEmpty);
    for (int i = tid; i < C::kSlots / (NW == 1 ? 8 : 4); i += 256)
        reinterpret_cast<uint4*>(cnt)[i] = make_uint4(0, 0, 0, 0);
    for (uint32_t b = b0 + blockIdx.x; b < b1; b += gridDim.x) {
        const uint64_t have = next_have, o0 = next_off;
        const uint32_t n_rec = (uint32_t)have, W = (uint32_t)(have >> 32);
        // rounds of up to kRecs records: their windows are numbered through,
        // an eighth of them to each warp, 32 at a time
        for (uint32_t rb = 0; rb < n_rec; rb += L::kRecs) {
            __syncthreads();
            if (*(volatile uint32_t*)&over) break;
            const uint32_t nr = min(n_rec - rb, (uint32_t)L::kRecs);
            uint64_t rr[R];
            uint32_t sum = 0;
#pragma unroll
            for (int q = 0; q < R; q++) {
                const uint32_t i = R * tid + q;
                rr[q] = i >= nr ? 0ull : rb == 0 && i < recs.slots ? next_rr[q] : recs.at(b, o0, rb + i);
                sum += (uint32_t)rr[q] & ((1u << kNwinBits) - 1u);
            }
            // a record's symbols from the packed reads, aligned to a word:
            // all of a thread's loads in flight at once
            auto symbols = [&](uint64_t rec, uint32_t nw, uint32_t out[L::kRW]) {
                const uint64_t p = rec >> kNwinBits;
                const uint32_t* src = packed + (p >> 4);
                const uint32_t sh = 2 * (uint32_t)(p & 15), need = ((uint32_t)(p & 15) + nw + K1 - 1 + 15) / 16;
                uint32_t v[L::kRW + 1];
#pragma unroll
                for (int i = 0; i <= L::kRW; i++) v[i] = (uint32_t)i < need ? src[i] : 0u;
#pragma unroll
                for (int i = 0; i < L::kRW; i++) out[i] = __funnelshift_l(v[i + 1], v[i], sh);
            };
            uint32_t tot, n_run;  // windows and records of the round
            if constexpr (L::kAlike) {
                // Most reads cover a place of the genome whole and without
                // error, and give equal records there.  A record is turned
                // to the smaller of its symbols and their reverse complement
                // (it has the same canonical windows), the first of equal
                // ones owns a place in a table of this round, and the others
                // only add to its number.
                for (int i = tid; i < L::kOwners / 4; i += 256) reinterpret_cast<uint4*>(owner)[i] = make_uint4(0, 0, 0, 0);
                uint64_t xh[R], xl[R];
                uint32_t nw[R];
#pragma unroll
                for (int q = 0; q < R; q++) {
                    nw[q] = (uint32_t)rr[q] & ((1u << kNwinBits) - 1u);
                    if (!nw[q]) continue;
                    uint32_t w[L::kRW];
                    symbols(rr[q], nw[q], w);
                    const int bits = 2 * ((int)nw[q] + K1 - 1);  // of 128, at the top
                    uint64_t h = (uint64_t)w[0] << 32 | w[1], l = (uint64_t)w[2] << 32 | w[3];
                    if (bits <= 64) {
                        h &= ~0ull << (64 - bits);
                        l = 0;
                    } else {
                        l &= ~0ull << (128 - bits);
                    }
                    uint64_t rh = rev2_u64(~l), rl = rev2_u64(~h);
                    const int up = 128 - bits;
                    if (up >= 64) {
                        rh = rl << (up - 64);
                        rl = 0;
                    } else if (up) {
                        rh = rh << up | rl >> (64 - up);
                        rl <<= up;
                    }
                    if (rh < h || (rh == h && rl < l)) {
                        h = rh;
                        l = rl;
                    }
                    xh[q] = h;
                    xl[q] = l;
                    const uint32_t i = R * tid + q;
                    reinterpret_cast<uint4*>(sym)[i] = make_uint4((uint32_t)(h >> 32), (uint32_t)h, (uint32_t)(l >> 32), (uint32_t)l);
                    start[i] = nw[q];
                    mul[i] = 1;
                }
                __syncthreads();
                uint32_t sums = 0;
#pragma unroll
                for (int q = 0; q < R; q++) {
                    if (!nw[q]) continue;
                    const uint32_t i = R * tid + q;
                    uint32_t o = (uint32_t)(mix_bij(xh[q] ^ mix_bij(xl[q] + nw[q])) >> 54);
                    static_assert(L::kOwners == 1 << 10, "ten bits");
                    while (true) {  // (at most half of the places are taken)
                        const uint32_t first = atomicCAS(&owner[o], 0u, i + 1);
                        if (!first) break;
                        const uint4 y = reinterpret_cast<const uint4*>(sym)[first - 1];
                        if (y.x == (uint32_t)(xh[q] >> 32) && y.y == (uint32_t)xh[q] && y.z == (uint32_t)(xl[q] >> 32) &&
                            y.w == (uint32_t)xl[q] && start[first - 1] == nw[q]) {
                            atomicAdd(&mul[first - 1], 1u);
                            nw[q] = 0;
                            break;
                        }
                        o = (o + 1) & (L::kOwners - 1);
                    }
                    if (nw[q]) sums += nw[q] | 1u << 16;
                }
                uint32_t all;
                uint32_t ex = scan(sums, &all);
                tot = all & 0xFFFFu;
                n_run = all >> 16;
#pragma unroll
                for (int q = 0; q < R; q++)
                    if (nw[q]) {
                        start[ex >> 16] = (ex & 0xFFFFu) | (uint32_t)(R * tid + q) << 16;
                        ex += nw[q] | 1u << 16;
                    }
            } else {
                uint32_t ex = scan(sum, &tot);
                n_run = nr;
#pragma unroll
                for (int q = 0; q < R; q++) {
                    const uint32_t nw = (uint32_t)rr[q] & ((1u << kNwinBits) - 1u);
                    if (nw) {
                        uint32_t w[L::kRW];
                        symbols(rr[q], nw, w);
                        uint4* dst = reinterpret_cast<uint4*>(sym + (R * tid + q) * L::kRW);
#pragma unroll
                        for (int i = 0; i < L::kRW / 4; i++)
                            dst[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
                        start[R * tid + q] = ex;
                    }
                    ex += nw;
                }
            }
            __syncthreads();
            const uint32_t per = (tot + 255) / 256 * 32;
            uint32_t j0 = warp * per;
            const uint32_t je = min(tot, j0 + per);
            if (j0 >= je) continue;
            // the last record that starts at or before window j0 (the upper
            // half of start is the record's place where equal ones are merged)
            constexpr uint32_t kAt = L::kAlike ? 0xFFFFu : 0xFFFFFFFFu;
            uint32_t cur = 0;
#pragma unroll
            for (int step = 256; step; step >>= 1)
                if (cur + step < n_run && (start[cur + step] & kAt) <= j0) cur += step;
            for (; j0 < je; j0 += 32) {
                // the record of window j0 + lane: the records after cur that
                // start among these windows, as bits
                const uint32_t nx = cur + 1 + lane, rel = (nx < n_run ? start[nx] & kAt : 0xFFFFFFFFu) - j0;
                const uint32_t m = __reduce_or_sync(0xFFFFFFFFu, rel < 32u ? 1u << rel : 0u);
                const uint32_t idx = cur + __popc(m & (0xFFFFFFFFu >> (31 - lane)));
                cur += __popc(m);
                if (j0 + lane < je) {
                    // the window's 2 NW words (and one more) of its record
                    const uint32_t st = start[idx], at = j0 + lane - (st & kAt), sh = 2 * (at & 15);
                    const uint32_t id = L::kAlike ? st >> 16 : idx;
                    const uint32_t* src = sym + id * L::kRW + (at >> 4);
                    Key<NW> x;
                    uint32_t hi = src[0];
#pragma unroll
                    for (int i = 0; i < NW; i++) {
                        const uint32_t md = src[2 * i + 1], lo = src[2 * i + 2];
                        x.w[NW - 1 - i] = ((uint64_t)__funnelshift_l(md, hi, sh) << 32) | __funnelshift_l(lo, md, sh);
                        hi = lo;
                    }
                    // the window at the top of the words, whatever follows
                    // below: shifted down it is the key; its symbols
                    // reversed and complemented, what is above the window
                    // masked off, the reverse complement
                    Key<NW> rc;
#pragma unroll
                    for (int i = 0; i < NW; i++) rc.w[i] = rev2_u64(~x.w[NW - 1 - i]);
                    rc = key_low<NW>(rc, 2 * K1);
                    x = key_shr<NW>(x, 64 * NW - 2 * K1);
                    if (key_eq<NW>(rc, x)) any_palin = 1;
                    insert(mix_key<NW>(key_less<NW>(rc, x) ? rc : x), L::kAlike ? mul[id] : 1u);
                }
            }
        }
        __syncthreads();
        // a warp an eighth of the slots: the occupied ones listed in order,
        // the occupancy bits of word q and the entries before it in lane q
        auto key_at = [&](uint32_t s) {
            Key<NW> m;
            m.w[NW - 1] = fp[s];
            if constexpr (NW > 1) {
#pragma unroll
                for (int q = 0; q < NW - 1; q++) m.w[q] = low[q * C::kSlots + s];
            }
            return m;
        };
        constexpr int WW = C::kWords / 8;
        const bool pal = any_palin != 0;  // (few bins hold a palindrome)
        uint32_t mine = 0, no = 0, my_occ = 0, my_pre = 0, my_palins = 0;
        if constexpr (NW == 1) {
            // 16 slots a lane (two reads of eight 16-bit counts)
            static_assert(L::kRegion == 512 && WW == 16, "16 slots a lane");
            const uint4* c4 = reinterpret_cast<const uint4*>(cnt) + warp * 64 + lane * 2;
            const uint4 u = c4[0], v = c4[1];
            const uint32_t c[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
            uint32_t m = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const uint32_t r = __vminu2(c[i], 0x00010001u);
                m |= ((r | r >> 15) & 3u) << (2 * i);
            }
            uint32_t incl = __popc(m);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t ex = incl - __popc(m);
            mine = __shfl_sync(0xFFFFFFFFu, incl, 31);
            uint32_t at = ex, kept = 0;
            for (uint32_t left = m; left; left &= left - 1) {
                const uint32_t s = warp * 512 + lane * 16 + __ffs(left) - 1;
                list[at++] = (uint16_t)s;
                kept += count_at(s) >= (uint32_t)d;
            }
            if (!pal) no = 2 * __reduce_add_sync(0xFFFFFFFFu, kept);
            my_occ = __shfl_sync(0xFFFFFFFFu, m, 2 * lane) | __shfl_sync(0xFFFFFFFFu, m, 2 * lane + 1) << 16;
            my_pre = __shfl_sync(0xFFFFFFFFu, ex, 2 * lane);
        } else {
#pragma unroll
            for (int q = 0; q < WW; q++) {
                const uint32_t s = (warp * WW + q) * 32 + lane, lit = count_at(s);
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, lit != 0), at = mine + __popc(m & lt);
                if (lit) list[at] = (uint16_t)s;
                if (lane == q) {
                    my_occ = m;
                    my_pre = mine;
                }
                mine += __popc(m);
                // kept keys of both strands
                if (!pal) no += 2 * __popc(__ballot_sync(0xFFFFFFFFu, lit && lit >= (uint32_t)d));
            }
        }
        __syncwarp();
        if (pal)
            for (uint32_t e0 = 0; e0 < mine; e0 += 32) {
                const uint32_t e = e0 + lane;
                bool pl = false;
                uint64_t lit = 0;
                if (e < mine) {
                    const uint32_t s = list[e];
                    lit = count_at(s);
                    const Key<NW> x = unmix_key<NW>(key_at(s));
                    pl = key_eq<NW>(key_rc<NW>(x, K1), x);
                    if (pl) lit *= 2;
                }
                const uint32_t sm = __ballot_sync(0xFFFFFFFFu, e < mine && lit >= (uint64_t)d), pm = __ballot_sync(0xFFFFFFFFu, pl);
                no += 2 * __popc(sm) - __popc(sm & pm);
                my_palins += __popc(pm);
            }
        if (lane == 0) {
            wsol[warp] = no;
            went[warp] = mine;
        }
        fetch(b + gridDim.x);
        __syncthreads();
        uint32_t po = 0, to = 0, pe = 0, ne = 0;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            po += q < warp ? wsol[q] : 0u;
            to += wsol[q];
            pe += q < warp ? went[q] : 0u;
            ne += went[q];
        }
        const bool rest = over || ne > (uint32_t)L::kMost;
        // (a warp's own slots are free once they are listed or written)
        auto clear = [&] {
            ulonglong2* f = reinterpret_cast<ulonglong2*>(fp + warp * L::kRegion);
            for (int i = lane; i < L::kRegion / 2; i += 32) f[i] = make_ulonglong2(kEmpty, kEmpty);
            constexpr int kPer = NW == 1 ? 8 : 4;  // counts in 16 bytes
            uint4* c = reinterpret_cast<uint4*>(cnt) + warp * (L::kRegion / kPer);
            for (int i = lane; i < L::kRegion / kPer; i += 32) c[i] = make_uint4(0, 0, 0, 0);
        };
        if (rest) {
            // to the rest; its place among the rest's keys
            if (tid == 0) {
                soff[b] = kSuperDeferred;
                const uint64_t q = atomicAdd(&totals[T_DEF], 1ull);
                const uint64_t w = atomicAdd(&totals[T_DEFWIN], (unsigned long long)W);
                deferred[q] = make_ulonglong2(b, w);
                if (give_up) {
                    const uint64_t done = atomicAdd(&totals[T_DONE], (unsigned long long)W);
                    const uint64_t full = atomicAdd(&totals[T_FULL], W > hot ? 0ull : (unsigned long long)W);
                    if (q >= kLostBins && full > give_up / 16 && super_lost(full, done)) totals[T_LOST] = 1;
                    lost = *(volatile unsigned long long*)&totals[T_LOST] != 0;
                }
            }
            clear();
            __syncthreads();
            if (lost) break;
            if (tid == 0) {
                over = next_hot();
                any_palin = 0;
            }
            continue;
        }
        palins += my_palins;
        // places for the entries and the kept keys, then both written
        if (tid == 0) {
            base[0] = atomicAdd(&totals[T_SPEC], (unsigned long long)ne);
            base[1] = atomicAdd(&totals[T_SOLID], (unsigned long long)to);
            soff[b] = base[0];
            if (give_up) atomicAdd(&totals[T_DONE], (unsigned long long)W);
        }
        if (lane < WW) sidx[(uint64_t)b * C::kWords + warp * WW + lane] = make_uint2(my_occ, pe + my_pre);
        __syncthreads();
        if (tid == 0) {
            over = next_hot();
            any_palin = 0;
        }
        // (past a buffer's end nothing is written: the host sees the totals)
        if (base[0] + ne <= spec_cap && base[1] + to <= solid_cap) {
            uint64_t so = base[1] + po;
            const uint64_t eo = base[0] + pe;
            for (uint32_t e0 = 0; e0 < mine; e0 += 32) {
                const uint32_t e = e0 + lane;
                bool pl = false;
                uint32_t lit = 0;
                Key<NW> x{}, r{};
                if (e < mine) {
                    const uint32_t s = list[e];
                    const Key<NW> m = key_at(s);
                    lit = count_at(s);
                    store_key<NW>(spec_k, eo + e, m);
                    spec_len[eo + e] = lit;
                    x = unmix_key<NW>(m);
                    r = key_rc<NW>(x, K1);
                    pl = pal && key_eq<NW>(r, x);
                    if (pl) lit *= 2;
                }
                const bool keep = e < mine && lit >= (uint32_t)d;
                const uint32_t sm = __ballot_sync(0xFFFFFFFFu, keep), pm = __ballot_sync(0xFFFFFFFFu, pl);
                if (keep) {
                    const uint64_t at = so + 2 * __popc(sm & lt) - __popc(sm & pm & lt);
                    store_key<NW>(solid_k, at, x);
                    solid_c[at] = lit;
                    if (!pl) {
                        store_key<NW>(solid_k, at + 1, r);
                        solid_c[at + 1] = lit;
                    }
                }
                so += 2 * __popc(sm) - __popc(sm & pm);
            }
        }
        __syncwarp();
        clear();
        // the next records on their way to L2
#pragma unroll
        for (int q = 0; q < R; q++)
            if ((uint32_t)(R * tid + q) < min((uint32_t)next_have, recs.slots))
                asm volatile("prefetch.global.L2 [%0];" ::"l"(packed + (next_rr[q] >> (kNwinBits + 4))));
    }
    if (lane == 0 && palins) atomicAdd(&totals[T_PALIN], (unsigned long long)palins);
}

// groups[q] = groups of 32 records of the q-th deferred bin.
__global__ void super_groups_kernel(SuperRecs recs, const ulonglong2* __restrict__ deferred, uint64_t n_def,
                                    uint32_t* __restrict__ groups) {
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < n_def; q += (uint64_t)gridDim.x * blockDim.x)
        groups[q] = ((uint32_t)recs.bins[deferred[q].x] + 31) / 32;
}

// The mixed canonical keys of the deferred bins, bin q's from its place on,
// in no fixed order (a warp reserves its windows' places on the bin's cursor).
// A warp a group of 32 records, wherever its bin: groups [first[q], first[q + 1])
// are bin q's.  Bins differ in size without bound; of a satellite of 171
// symbols, read 30 times, k = 61, with as many CTAs for every bin 7.6 ms, by groups
// 0.29.
template <int NW>
__global__ void __launch_bounds__(256) super_expand_kernel(const uint32_t* __restrict__ packed,
                                                           SuperRecs recs,
                                                           const ulonglong2* __restrict__ deferred, uint64_t n_def,
                                                           const uint64_t* __restrict__ first, int K1,
                                                           unsigned long long* __restrict__ cursor,
                                                           uint64_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * 8, n_groups = first[n_def];
    for (uint64_t g = blockIdx.x * 8ull + (threadIdx.x >> 5); g < n_groups; g += warps) {
        // the last bin that starts at or before group g (empty ones start with the next)
        uint64_t lo = 0, hi = n_def;
        while (hi - lo > 1) {
            const uint64_t mid = (lo + hi) / 2;
            if (first[mid] <= g) lo = mid; else hi = mid;
        }
        const uint64_t q = lo, b = deferred[q].x;
        const uint32_t n_rec = (uint32_t)recs.bins[b], i = (uint32_t)(g - first[q]) * 32 + lane;
        const uint64_t r = i < n_rec ? recs.at(b, recs.off[b], i) : 0ull;
        const uint32_t tot = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)r & ((1u << kNwinBits) - 1u));
        uint64_t at = 0;
        if (lane == 0) at = deferred[q].y + atomicAdd(&cursor[q], (unsigned long long)tot);
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        for_windows(r, [&](bool valid, uint32_t j, uint64_t p) {
            if (!valid) return;
            const Key<NW> x = load_window<NW>(packed, p, K1);
            const Key<NW> rc = key_rc<NW>(x, K1);
            store_key<NW>(out, at + j, mix_key<NW>(key_less<NW>(rc, x) ? rc : x));
        });
    }
}

// ------------------------------------------------------------------- host

static long env_long(const char* name, long dflt) {
    const char* e = std::getenv(name);
    return e ? std::strtol(e, nullptr, 10) : dflt;
}

// From 2^22 windows on, and for windows of at most 48 symbols at any number
// of them: such sets take a few launches where the unit route takes radix
// passes (whole path, windows x 10^3, unit route and this one in ms: k = 31
// 38 1.04 0.87, 376 1.28 1.05, 4,700 1.56 1.25; k = 47 62 1.34 1.02, 1,950
// 1.63 1.23).  Windows of more symbols leave bins to the rest: k = 63 248 1.48
// 1.58; k = 61 1,600 1.73 1.77; k = 99 2,600 2.45 2.65.  A plan's unit bits do not
// choose: they are those of the sets, buckets and rests that units count.  A
// variable that steers the unit counting (tests) does.  MH_SUPER=0 turns this
// route off, =1 on at any size and whatever is left to the rest (tests).  The
// counters of a bin hold 32 bits each, so fewer than 2^32 windows.
static long super_switch() {
    static const long v = env_long("MH_SUPER", -1);
    return v;
}

bool use_super(uint64_t n, int K1) {
    const long v = super_switch();
    static const bool steered = [] {
        for (const char* e : {"MH_GROUP_CAP", "MH_GROUP_UNIT_BITS", "MH_EXTRACT_SCATTER", "MH_SCATTER_CAP", "MH_SORT_CHUNK_TILES"})
            if (std::getenv(e)) return true;
        return false;
    }();
    if (v == 0 || !n || n >= (1ull << 32) || super_m(K1) == 0) return false;
    return v == 1 || (!steered && (n >= (1ull << 22) || K1 <= 48));
}

template <int NW>
bool super_count(mh_ctx* ctx, const mh_reads* reads, int k, int d, uint64_t n, mh_kmers* out) {
    using C = SuperCfg<NW>;
    const int K1 = k + 1, m = super_m(K1), w = K1 - m + 1;
    // tests: bins of more windows than MH_SUPER_HOT, or with a key that finds
    // no place in MH_SUPER_PROBES slots, are left to the rest
    static const uint32_t hot = (uint32_t)std::max(0l, env_long("MH_SUPER_HOT", 1 << 16));
    static const int most_probes = (int)std::max(1l, std::min(256l, env_long("MH_SUPER_PROBES", 128)));
    // tests: the first buffers for the other bins of a sampled set hold
    // MH_SUPER_ESTIMATE percent of the estimate (no slack), and the limit on
    // probes holds for them alone, so that the second time round bins are in
    // place that the first left to the rest
    static const long estimate = env_long("MH_SUPER_ESTIMATE", 0);
    int probes = estimate ? 128 : most_probes;
    const uint64_t F = reads->n_frags, n_words = ceil_div(reads->n_packed, 16) + kPackPad;
    const uint64_t n_tiles = ceil_div(reads->n_packed, (uint64_t)kSplitTile);
    const uint32_t n_bins = (uint32_t)std::max<uint64_t>(1, n / C::kTarget);
    const uint64_t give_up = NW == 2 && super_switch() != 1 ? n : 0;
    // records: 2 / (w + 1) a window for random sequences (about 8 / w by
    // halves), one more a fragment and a tile; each bin has slots for half as
    // many again as its share, and the list of those past them room for all:
    // where few minimizers take most windows it gets most records (again
    // with room for what there is, if there are still more)
    const double run = super_half(K1) ? w / 8.0 : (w + 1) / 2.0;
    const uint64_t expect = std::min(n, (uint64_t)((double)n / run) + F + n_tiles + 1);
    const uint32_t slots = (uint32_t)((double)expect / n_bins * 1.5) + 16;
    uint64_t cap = expect + 4096;
    const uint64_t per = d >= 2 ? 1 : 2;  // kept keys of both strands a window, at most
    // large sets: a sixteenth of the bins first, to size the outputs by
    const bool sample = n >= (1ull << 25) && n_bins >= 4096;
    // short fragments make a record of every window or two, and those beside
    // outputs with room for all windows need more than the units: a set that
    // does not fit with them is theirs
    const uint64_t out_bytes = (sample ? n / 8 : n) * (1 + per) * (8 * NW + 4);
    const uint64_t bin_bytes = 8 * n_tiles + (uint64_t)n_bins * (8 * slots + 8 * C::kWords + 64);
    const uint64_t avail = count_memory(ctx);
    auto fits = [&] { return bin_bytes + std::max(24 * cap, 8 * cap + out_bytes) + (1u << 20) <= avail; };
    if (!fits()) return false;
    Buf<uint64_t> first(ctx, n_tiles), off(ctx, (uint64_t)n_bins + 1), totals(ctx, T_N);
    Buf<unsigned long long> bins(ctx, n_bins);
    MH_LAUNCH(ctx, "super_tiles", grid_for(ctx, n_tiles, 256), 256, 0, super_tiles_kernel, reads->frag_offs, F,
              n_tiles, first.p);
    Buf<uint64_t> rec(ctx, (uint64_t)n_bins * slots);
    unsigned long long* tot = reinterpret_cast<unsigned long long*>(totals.p);
    Buf<uint64_t> more;
    SuperRecs recs{rec.p, nullptr, off.p, bins.p, slots};
    uint64_t h[T_N] = {0};
    Buf<uint64_t> spec, solid, soff(ctx, n_bins);
    Buf<uint32_t> spec_len, solid_c;
    Buf<uint2> sidx(ctx, (uint64_t)n_bins * C::kWords);
    Buf<ulonglong2> deferred(ctx, n_bins);
    uint64_t spec_cap = 0, solid_cap = 0;
    constexpr size_t smem = SuperSmem<NW>::kBytes;
    MH_CUDA(cudaFuncSetAttribute(super_count_kernel<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    MH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, super_count_kernel<NW>, 256, smem));
    auto count = [&](uint32_t b0, uint32_t b1) {
        if (b0 < b1)
            MH_LAUNCH_B(ctx, "super_count", n / 4, (unsigned)std::min<uint64_t>(b1 - b0, (uint64_t)ctx->num_sms * std::max(1, per_sm)),
                        256, smem, super_count_kernel<NW>, reads->packed, recs, b0, b1, cap, K1, d,
                        give_up, hot,
                        probes, spec_cap, spec.p, spec_len.p, solid_cap, solid.p, solid_c.p, soff.p, sidx.p,
                        deferred.p, tot);
    };
    auto room = [&](uint64_t a, uint64_t s) {
        spec_cap = a;
        solid_cap = s;
        spec = Buf<uint64_t>(ctx, a * NW);
        spec_len = Buf<uint32_t>(ctx, a);
        solid = Buf<uint64_t>(ctx, s * NW);
        solid_c = Buf<uint32_t>(ctx, s);
    };
    const uint32_t nb1 = sample ? n_bins / 16 : n_bins;
    bool all = false;
    for (int attempt = 0;; attempt++) {
        more.reset();
        more = Buf<uint64_t>(ctx, cap);
        recs.more = more.p;
        {
            Buf<uint64_t> raw(ctx, cap);
            Buf<uint2> place(ctx, cap);
            Buf<uint32_t> over(ctx, n_bins);
            bins.zero();
            totals.zero();
            const auto split = super_half(K1) ? super_split_kernel<16, true>
                               : m == 16      ? super_split_kernel<16, false>
                               : m == 14      ? super_split_kernel<14, false>
                                              : super_split_kernel<12, false>;
            MH_LAUNCH_B(ctx, "super_split", reads->n_packed / 4, (unsigned)n_tiles, 256, 0, split, reads->packed, n_words,
                        reads->frag_offs, F, first.p, k, n_bins, (uint32_t)(32 * C::kRecWords / 2 - K1 + 1), slots, rec.p,
                        raw.p, place.p, cap, bins.p, tot);
            MH_LAUNCH(ctx, "super_over", grid_for(ctx, n_bins, 256), 256, 0, super_over_kernel, bins.p, n_bins, slots,
                      over.p);
            exclusive_scan_u32(ctx, over.p, off.p, n_bins);
            MH_LAUNCH(ctx, "super_place", grid_for(ctx, cap, 256), 256, 0, super_place_kernel, raw.p, place.p, cap, tot,
                      off.p, more.p);
        }
        // (room for a sample with twice its share of the windows; with all of
        // them if it has more)
        const uint64_t n1 = sample && !all ? n / 8 : n;
        room(std::max<uint64_t>(n1, 1), std::max<uint64_t>(n1 * per, 1));
        count(0, nb1);
        read_u64(ctx, totals.p, h, T_N);
        if (h[T_LOST]) return false;
        if (h[T_RECS] <= cap && h[T_SPEC] <= spec_cap && h[T_SOLID] <= solid_cap) break;
        if (attempt >= 2) fail(MH_EDEVICE, "super-k-mer records overflow again");
        all = h[T_RECS] <= cap;
        cap = std::max(cap, h[T_RECS]);
        spec.reset();
        spec_len.reset();
        solid.reset();
        solid_c.reset();
        if (!fits()) return false;
    }
    if (sample) {
        if (give_up && h[T_DEF] > kLostBins && super_lost(h[T_FULL], h[T_DONE])) return false;
        // the other bins into buffers sized by the first ones (bins are by
        // hash: alike but for chance and the heavy ones), then the first
        // ones' entries in front of them
        Buf<uint64_t> k1 = std::move(spec), s1 = std::move(solid);
        Buf<uint32_t> l1 = std::move(spec_len), c1 = std::move(solid_c);
        const uint64_t a1 = h[T_SPEC], o1 = h[T_SOLID];
        const double f = (double)n_bins / nb1;
        uint64_t a = std::min<uint64_t>(n, (uint64_t)(1.04 * f * (double)a1) + (1u << 20));
        uint64_t s = std::min<uint64_t>(n * per, (uint64_t)(1.04 * f * (double)o1) + (1u << 20));
        if (estimate) {
            a = std::max(a1, (uint64_t)(f * (double)a1) * estimate / 100);
            s = std::max(o1, (uint64_t)(f * (double)o1) * estimate / 100);
        }
        const std::vector<uint64_t> h1(h, h + T_N);
        for (int attempt = 0;; attempt++) {
            probes = estimate && attempt ? 128 : most_probes;
            room(a, s);
            if (a1) {
                MH_CUDA(cudaMemcpyAsync(spec.p, k1.p, a1 * NW * 8, cudaMemcpyDeviceToDevice, ctx->stream));
                MH_CUDA(cudaMemcpyAsync(spec_len.p, l1.p, a1 * 4, cudaMemcpyDeviceToDevice, ctx->stream));
            }
            if (o1) {
                MH_CUDA(cudaMemcpyAsync(solid.p, s1.p, o1 * NW * 8, cudaMemcpyDeviceToDevice, ctx->stream));
                MH_CUDA(cudaMemcpyAsync(solid_c.p, c1.p, o1 * 4, cudaMemcpyDeviceToDevice, ctx->stream));
            }
            count(nb1, n_bins);
            read_u64(ctx, totals.p, h, T_N);
            if (h[T_LOST]) return false;
            if (h[T_SPEC] <= a && h[T_SOLID] <= s) break;
            if (attempt) fail(MH_EDEVICE, "super-k-mer outputs overflow twice");
            // (which bins are left to the rest depends on the order of their
            // insertions: those left out now may be in place the next time)
            a = std::min(n, h[T_SPEC] + h[T_DEFWIN]);
            s = std::min(n * per, h[T_SOLID] + per * h[T_DEFWIN]);
            MH_CUDA(cudaMemcpyAsync(totals.p, h1.data(), sizeof(uint64_t) * T_N, cudaMemcpyHostToDevice, ctx->stream));
            sync_and_check(ctx);
        }
    }
    uint64_t R = h[T_SPEC], S = h[T_SOLID], runs = R, palins = h[T_PALIN];
    const uint64_t n_main = R;
    // the outputs' buffers grow by the rest, or shrink if much too large
    auto fit = [&](Buf<uint64_t>& kb, Buf<uint32_t>& cb, uint64_t have, uint64_t& have_cap, const Buf<uint64_t>& rk,
                   const Buf<uint32_t>& rcnt, uint64_t more) {
        const uint64_t need = have + more;
        if (need > have_cap || have_cap > need + need / 4 + 4096) {
            Buf<uint64_t> k2(ctx, (need ? need : 1) * NW);
            Buf<uint32_t> c2(ctx, need ? need : 1);
            if (have) {
                MH_CUDA(cudaMemcpyAsync(k2.p, kb.p, have * NW * 8, cudaMemcpyDeviceToDevice, ctx->stream));
                MH_CUDA(cudaMemcpyAsync(c2.p, cb.p, have * 4, cudaMemcpyDeviceToDevice, ctx->stream));
            }
            kb = std::move(k2);
            cb = std::move(c2);
            have_cap = need;
        }
        if (more) {
            MH_CUDA(cudaMemcpyAsync(kb.p + have * NW, rk.p, more * NW * 8, cudaMemcpyDeviceToDevice, ctx->stream));
            MH_CUDA(cudaMemcpyAsync(cb.p + have, rcnt.p, more * 4, cudaMemcpyDeviceToDevice, ctx->stream));
        }
    };
    // the deferred bins, by the unit counting
    RunList rest;
    Buf<uint64_t> rest_k;
    Buf<uint32_t> rest_c;
    uint64_t rest_S = 0;
    if (h[T_DEF]) {
        const uint64_t nd = h[T_DEFWIN];
        // what the rest takes (keys twice, lengths, slots of kept pairs)
        // beside outputs with room for all windows can pass the 24 NW + 12
        // bytes a window that the caller's memory plan counts on: the outputs
        // are then made to fit first (else once, with the rest; it is a copy)
        const uint64_t pair = 8 * NW + 4;
        if ((spec_cap + solid_cap) * pair + nd * (16 * NW + 4 + per * pair) > n * (24 * NW + 12)) {
            fit(spec, spec_len, n_main, spec_cap, rest_k, rest_c, 0);
            fit(solid, solid_c, h[T_SOLID], solid_cap, rest_k, rest_c, 0);
        }
        Buf<uint64_t> keys(ctx, nd * NW), alt(ctx, nd * NW);
        Buf<unsigned long long> cursor(ctx, h[T_DEF]);
        cursor.zero();
        Buf<uint32_t> groups(ctx, h[T_DEF]);
        Buf<uint64_t> first_group(ctx, h[T_DEF] + 1);
        MH_LAUNCH(ctx, "super_groups", grid_for(ctx, h[T_DEF], 256), 256, 0, super_groups_kernel, recs, deferred.p,
                  h[T_DEF], groups.p);
        exclusive_scan_u32(ctx, groups.p, first_group.p, h[T_DEF]);
        MH_LAUNCH(ctx, "super_expand", grid_for(ctx, nd, 2048), 256, 0, super_expand_kernel<NW>, reads->packed, recs,
                  deferred.p, h[T_DEF], first_group.p, K1, cursor.p, keys.p);
        rec.reset();
        more.reset();
        const GroupPlan gp = group_plan(ctx, nd, 0, NW);
        if (gp.passes < 0) fail(MH_EDEVICE, "super-k-mer counting: no unit plan for the deferred bins");
        const bool in_alt = gp.passes ? radix_sort<NW>(ctx, keys.p, alt.p, nullptr, nullptr, nd, 64 * NW - 8 * gp.passes, 64 * NW)
                                      : false;
        uint64_t r2 = 0, p2 = 0;
        group_count<NW>(ctx, in_alt ? alt : keys, in_alt ? keys : alt, nd, k, d, 0, gp, rest_k, rest_c, &rest_S, &r2, &p2,
                        &rest, false);
        runs += r2;
        palins += p2;
        R += rest.n;
        S += rest_S;
    }
    rec.reset();
    more.reset();
    first.reset();
    off.reset();
    bins.reset();
    deferred.reset();
    fit(spec, spec_len, n_main, spec_cap, rest.keys, rest.lens, rest.n);
    fit(solid, solid_c, h[T_SOLID], solid_cap, rest_k, rest_c, rest_S);
    rest.keys.reset();
    rest.lens.reset();
    rest_k.reset();
    rest_c.reset();
    {
        Buf<uint64_t> alt(ctx, (S ? S : 1) * NW);
        Buf<uint32_t> calt(ctx, S ? S : 1);
        if (radix_sort_spread_kv<NW>(ctx, solid.p, alt.p, solid_c.p, calt.p, S, 64 * NW - 2 * K1)) {
            std::swap(solid, alt);
            std::swap(solid_c, calt);
        }
    }
    sync_and_check(ctx);
    out->n = S;
    out->n_distinct = 2 * runs - palins;
    out->keys = solid.release();
    out->counts = solid_c.release();
    out->n_spectrum = R;
    out->spectrum = spec.release();
    out->spectrum_len = spec_len.release();
    out->super_off = soff.release();
    out->super_idx = sidx.release();
    out->super_bins = n_bins;
    out->super_m = m;
    out->super_main = n_main;
    return true;
}

template bool super_count<1>(mh_ctx*, const mh_reads*, int, int, uint64_t, mh_kmers*);
template bool super_count<2>(mh_ctx*, const mh_reads*, int, int, uint64_t, mh_kmers*);
template bool super_count<4>(mh_ctx*, const mh_reads*, int, int, uint64_t, mh_kmers*);

}  // namespace mh

// LSD radix sort of multiword keys (optionally with a 32-bit payload) and
// device-wide exclusive scans.
//
// Sort: one histogram kernel counts every 8-bit digit of every pass in a
// single read of the keys; then each pass is one "onesweep" kernel: a CTA
// takes the next tile (dynamic tile id, so every earlier tile already runs),
// counts its keys' digits in per-warp shared-memory histograms, publishes
// the tile's per-digit counts, ranks the keys by digit (a warp match on the
// digit's top bits, ballots on the rest) with one shared atomic per group of
// equal digits (stable: rank follows input order) while staging them in
// shared memory in digit order, looks back over earlier tiles' published
// counts (decoupled look-back, every wait bounded) and writes the tile out
// in coalesced runs.  Look-back counts are 30-bit, so a pass runs in chunks of at most (2^18 - 1) tiles, one launch per chunk,
// each with its own look-back chain.  Chunk 0 starts from the global digit
// offsets of the histogram (the same for every pass); the last tile of chunk
// c writes the digit offsets where chunk c+1 starts.  The first pass may
// read a segmented input (radix_sort_segmented: the keys of each value of
// the previous digit in a segment of fixed size, as the fused extraction
// of mh_count.cu writes them); its tiles then skip the unused slots.
#include <atomic>
#include <cstdlib>
#include <vector>

#include "mh_sort_kernels.cuh"

namespace mh {

// Tiles per look-back chunk: (2^18 - 1), or MH_SORT_CHUNK_TILES (>= 1) when
// set, which tests use to run the multi-chunk path on small inputs.
static uint64_t chunk_tiles() {
    static uint64_t v = [] {
        const char* e = std::getenv("MH_SORT_CHUNK_TILES");
        uint64_t t = e ? std::strtoull(e, nullptr, 10) : 0;
        return (t >= 1 && t <= kMaxTilesPerChunk) ? t : kMaxTilesPerChunk;
    }();
    return v;
}

// Polls a look-back wait may make before it gives up (MH_SPIN_LIMIT, >= 1;
// default kSpinLimit, about a second with the back-off).
static int spin_limit() {
    static const int v = [] {
        const char* e = std::getenv("MH_SPIN_LIMIT");
        const long x = e ? std::strtol(e, nullptr, 10) : 0;
        return x >= 1 && x <= kSpinLimit ? (int)x : kSpinLimit;
    }();
    return v;
}

// Test hook: MH_TEST_WITHHOLD_TILE0=N makes the first N scatter launches of
// the process keep their tile 0 from publishing its counts, so that the
// bounded waits of the tiles after it run out (MH_ETIMEOUT); later launches
// are normal.
static int take_withhold() {
    static std::atomic<int> left{[] {
        const char* e = std::getenv("MH_TEST_WITHHOLD_TILE0");
        return e ? std::atoi(e) : 0;
    }()};
    int v = left.load();
    while (v > 0 && !left.compare_exchange_weak(v, v - 1)) {
    }
    return v > 0 ? 1 : 0;
}

// seg.cnt set: the first pass reads a segmented input of 256 * seg.cap
// slots holding the n keys (SegIn); every pass writes n contiguous keys.
template <int NW, bool HV, int ITEMS, int MINB>
static bool radix_sort_impl(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint32_t* vals, uint32_t* valt, uint64_t n,
                            int bit_lo, int bit_hi, const uint32_t* hist_in, SegIn seg = SegIn{}) {
    if (n <= 1 || bit_hi <= bit_lo) return false;
    constexpr int TILE = sort_tile<NW, ITEMS>();
    const int n_passes = (bit_hi - bit_lo + 7) / 8;
    const uint64_t chunk_len = chunk_tiles() * TILE;
    // positions pass p reads: the segment slots in the first pass
    auto span = [&](int p) { return p == 0 && seg.cnt ? 256 * seg.cap : n; };
    const int max_chunks = (int)ceil_div(span(0), chunk_len);
    Buf<uint32_t> hist(ctx, hist_in ? 1 : (size_t)n_passes * 256);
    // base[(p * max_chunks + c) * 256 + d]: where chunk c of pass p starts writing digit d
    Buf<uint64_t> base(ctx, (size_t)n_passes * max_chunks * 256);
    if (!hist_in) {
        hist.zero();
        MH_LAUNCH_B(ctx, "radix_hist", n * 8 * NW, grid_for(ctx, n, 256, 8), 256, sizeof(uint32_t) * n_passes * 256,
                    radix_hist_kernel<NW>, keys, n, bit_lo, n_passes, hist.p);
    }
    MH_LAUNCH(ctx, "radix_base", n_passes, 256, 0, radix_base_kernel, hist_in ? hist_in : hist.p, base.p,
              (uint64_t)max_chunks * 256);
    const uint64_t max_tiles = std::min<uint64_t>(chunk_tiles(), ceil_div(span(0), TILE));
    // small sorts: tile counts and counter of every pass zeroed at once (a
    // pass is otherwise three operations of the stream, 2 us each)
    const uint64_t pass_words = max_tiles * 256 + 64;
    const bool at_once = max_chunks == 1 && pass_words * n_passes <= (1u << 20);
    Buf<uint32_t> status(ctx, pass_words * (at_once ? n_passes : 1));
    if (at_once) status.zero();
    constexpr size_t smem = onesweep_smem<NW, HV, ITEMS>();
    MH_CUDA(cudaFuncSetAttribute(onesweep_kernel<NW, HV, ITEMS, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    uint64_t *kin = keys, *kout = alt;
    uint32_t *vin = vals, *vout = valt;
    for (int p = 0; p < n_passes; p++) {
        const uint64_t np = span(p);
        const int n_chunks = (int)ceil_div(np, chunk_len);
        for (int c = 0; c < n_chunks; c++) {
            uint64_t c0 = (uint64_t)c * chunk_len;
            uint64_t len = std::min(chunk_len, np - c0);
            uint64_t tiles = ceil_div(len, TILE);
            uint32_t* st = status.p + (at_once ? p * pass_words : 0);
            uint32_t* counter = st + tiles * 256;
            if (!at_once)
                MH_CUDA(cudaMemsetAsync(st, 0, (tiles * 256 + 1) * sizeof(uint32_t), ctx->stream));
            uint64_t* nb = c + 1 < n_chunks ? base.p + ((uint64_t)p * max_chunks + c + 1) * 256 : nullptr;
            if constexpr (NW == 1 && !HV) {
                if (p == 0 && seg.cnt) {
                    SegIn sp = seg;
                    sp.slot0 = c0;
                    MH_CUDA(cudaFuncSetAttribute(onesweep_kernel<NW, HV, ITEMS, MINB, true>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
                    MH_LAUNCH_B(ctx, "radix_onesweep", len * 16, (unsigned)tiles, kSortThreads, smem,
                                (onesweep_kernel<NW, HV, ITEMS, MINB, true>), kin + c0, kout, nullptr, nullptr, len,
                                bit_lo, base.p + (uint64_t)c * 256, nb, st, counter, ctx->d_status,
                                spin_limit(), take_withhold(), sp);
                    continue;
                }
            }
            MH_LAUNCH_B(ctx, "radix_onesweep", len * (16 * NW + (HV ? 8 : 0)), (unsigned)tiles, kSortThreads, smem,
                        (onesweep_kernel<NW, HV, ITEMS, MINB>), kin + c0 * NW, kout, HV ? vin + c0 : nullptr, vout, len,
                        bit_lo + 8 * p, base.p + ((uint64_t)p * max_chunks + c) * 256, nb, st, counter,
                        ctx->d_status, spin_limit(), take_withhold(), SegIn{});
        }
        std::swap(kin, kout);
        std::swap(vin, vout);
    }
    return (n_passes & 1) != 0;
}

// Tile shape of the scatter pass for 1-word keys: (items per thread,
// resident CTAs per SM).  The default, (16, 3), measured fastest on GB300 for
// keys alone and with a payload (3.3e8 pairs, with the other sorts of a path:
// 10.1 ms; (14, 3) 10.5, (12, 4) 11.5); a context's tuned shape
// (mh_run_batch's autotuner) or MH_SORT_VARIANT selects another key-only
// shape: 1 = (12, 4), 2 = (14, 3).
static int sort_variant() {
    static int v = [] {
        const char* e = std::getenv("MH_SORT_VARIANT");
        return e ? std::atoi(e) : 0;
    }();
    return v;
}

// Keys alone that fit one CTA's shared memory, by whole key: a bitonic sort
// (a power of two of slots, all-ones keys at the end).  Bound by its barriers
// (105 steps for 16,384 keys).  A pass of the radix sort costs a launch and its
// gap, six to eleven of them for whole keys: dummies and candidates of a set
// of 10,000 reads, 254 and 48 keys, 0.10 -> 0.02 ms.
template <int NW>
__host__ __device__ constexpr uint32_t tiny_sort_max() {
    return 16384 / NW;  // 128 KB
}

template <int NW>
__global__ void __launch_bounds__(1024) tiny_sort_kernel(uint64_t* __restrict__ keys, uint32_t n, uint32_t slots) {
    extern __shared__ __align__(16) uint64_t tk[];
    for (uint32_t i = threadIdx.x; i < slots; i += 1024) {
        Key<NW> x;
#pragma unroll
        for (int w = 0; w < NW; w++) x.w[w] = ~0ull;
        if (i < n) x = load_key<NW>(keys, i);
        store_key<NW>(tk, i, x);
    }
    for (uint32_t size = 2; size <= slots; size <<= 1)
        for (uint32_t step = size >> 1; step; step >>= 1) {
            __syncthreads();
            for (uint32_t q = threadIdx.x; q < slots / 2; q += 1024) {
                const uint32_t i = 2 * q - (q & (step - 1)), j = i + step;
                const Key<NW> a = load_key<NW>(tk, i), b = load_key<NW>(tk, j);
                if (key_less<NW>(b, a) == ((i & size) == 0) && !key_eq<NW>(a, b)) {
                    store_key<NW>(tk, i, b);
                    store_key<NW>(tk, j, a);
                }
            }
        }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += 1024) store_key<NW>(keys, i, load_key<NW>(tk, i));
}

// Sorts in place; n in [2, tiny_sort_max].
template <int NW>
static void tiny_sort(mh_ctx* ctx, uint64_t* keys, uint64_t n) {
    uint32_t slots = 64;
    while (slots < n) slots <<= 1;
    const size_t smem = sizeof(uint64_t) * NW * slots;
    MH_CUDA(cudaFuncSetAttribute(tiny_sort_kernel<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(sizeof(uint64_t) * NW * tiny_sort_max<NW>())));
    MH_LAUNCH(ctx, "tiny_sort", 1, 1024, smem, tiny_sort_kernel<NW>, keys, (uint32_t)n, slots);
}

// Words of keys of a sort in small tiles: 2^19, or MH_SORT_SMALL when set (tests
// run the large tiles on small inputs with 0).
static uint64_t small_words() {
    static const uint64_t v = [] {
        const char* e = std::getenv("MH_SORT_SMALL");
        return e ? (uint64_t)std::strtoull(e, nullptr, 10) : (uint64_t)1 << 19;
    }();
    return v;
}

template <int NW, bool HV>
static bool radix_sort_dispatch(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint32_t* vals, uint32_t* valt,
                                uint64_t n, int bit_lo, int bit_hi, const uint32_t* h, SegIn seg = SegIn{}) {
    // the shape of large sorts of one-word keys alone; others have one each
    const int shape = NW > 1 || HV ? 0 : ctx->sort_shape >= 0 ? ctx->sort_shape : sort_variant();
    // up to 2^19 words of keys: tiles of 1,024 words, so that a pass has some
    // for every SM (14 passes of a path of 10,000 reads 0.156 -> 0.132 ms)
    if (!seg.cnt && n * (uint64_t)NW <= small_words() && shape == 0)
        return radix_sort_impl<NW, HV, 4 / NW, 3>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
    if constexpr (NW == 1) {
        if constexpr (HV) {
            return radix_sort_impl<NW, HV, 16, 3>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
        } else {
            switch (shape) {
                case 1: return radix_sort_impl<NW, HV, 12, 4>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
                case 2: return radix_sort_impl<NW, HV, 14, 3>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
                default: return radix_sort_impl<NW, HV, 16, 3>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
            }
        }
    }
    return radix_sort_impl<NW, HV, SortItems<NW>::v, 2>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, h, seg);
}

bool radix_sort_segmented(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint64_t n,
                          const unsigned long long* seg_cnt, uint64_t seg_cap, int bit_lo, int bit_hi,
                          const uint32_t* hist) {
    if (seg_cap < (uint64_t)sort_tile<1>() || !hist) throw Error{MH_EINVAL, "segmented sort: bad segments"};
    SegIn seg;
    seg.cnt = seg_cnt;
    seg.cap = seg_cap;
    return radix_sort_dispatch<1, false>(ctx, keys, alt, nullptr, nullptr, n, bit_lo, bit_hi, hist, seg);
}

// Keys of a sort by one CTA: tiny_sort_max, or MH_TINY_SORT when set (tests
// run the passes on small inputs with 0).
template <int NW>
static uint64_t tiny_max() {
    static const long v = [] {
        const char* e = std::getenv("MH_TINY_SORT");
        return e ? std::strtol(e, nullptr, 10) : (long)tiny_sort_max<1>();
    }();
    return (uint64_t)std::max(0l, std::min(v, (long)tiny_sort_max<1>())) / NW;
}

template <int NW>
bool radix_sort(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint32_t* vals, uint32_t* valt, uint64_t n, int bit_lo,
                int bit_hi, const uint32_t* hist) {
    if (vals) return radix_sort_dispatch<NW, true>(ctx, keys, alt, vals, valt, n, bit_lo, bit_hi, hist);
    // (the bits from bit_hi on are equal in every key, so whole keys compare
    // alike)
    if (n > 1 && bit_lo == 0 && n <= tiny_max<NW>()) {
        tiny_sort<NW>(ctx, keys, n);
        return false;
    }
    return radix_sort_dispatch<NW, false>(ctx, keys, alt, nullptr, nullptr, n, bit_lo, bit_hi, hist);
}

template bool radix_sort<1>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int, int, const uint32_t*);
template bool radix_sort<2>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int, int, const uint32_t*);
template bool radix_sort<4>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int, int, const uint32_t*);

// ------------------------------------------------------------ spread sort
// The keys are mix_key images, so the top bits of their top word are evenly
// spread: LSD passes over the top P bits only (P = ceil(log2 n) rounded up
// to a digit) leave every group of equal top bits in input order, and a
// group holds more than one distinct key only where two keys collide on
// those P bits (about D^2 / 2^(P+1) groups for D distinct keys).  The fix-up
// sorts such groups.  A tile kernel reads a window of keys (2048 / nw plus
// 256 / nw past the tile, for the group that crosses its end), finds the
// groups that start in the tile and contain a descent, and sorts them: up to
// 16 keys by one thread (insertion sort), larger ones by one warp
// (successive minima: each round finds the smallest key above the previous
// one and its count, then writes that run).  Groups that do not end inside
// the window, or have more than 64 distinct keys, go to a list for a CTA
// each (successive minima over the group in global memory, written through
// the free buffer); more than 256 distinct keys there (pathological) fall
// back to a radix sort of the segment.

template <int NW>
struct Fix {
    static constexpr int kTile = 2048 / NW;
    static constexpr int kExt = 256 / NW;
    static constexpr int kWin = kTile + kExt;
    static constexpr int kWords = kWin / 32;
    static constexpr int kThreadSort = 16;
    static constexpr int kQueue = kWin / (kThreadSort + 1) + 1;  // groups of > 16 keys in a window
};
constexpr int kFixWarpRounds = 64;
constexpr int kFixBlockRounds = 256;

template <int NW>
__device__ __forceinline__ Key<NW> shfl_key(const Key<NW>& a, int src_lane_xor) {
    Key<NW> r;
#pragma unroll
    for (int w = 0; w < NW; w++) r.w[w] = __shfl_xor_sync(0xFFFFFFFFu, a.w[w], src_lane_xor);
    return r;
}

template <int NW>
__device__ __forceinline__ Key<NW> key_ones() {
    Key<NW> r;
#pragma unroll
    for (int w = 0; w < NW; w++) r.w[w] = ~0ull;
    return r;
}

template <int NW>
__global__ void __launch_bounds__(256) spread_fix_kernel(uint64_t* __restrict__ keys, uint64_t n, int lo,
                                                         uint64_t* __restrict__ big, uint64_t big_cap,
                                                         unsigned long long* __restrict__ n_big) {
    using F = Fix<NW>;
    __shared__ uint64_t K[F::kWin * NW];
    __shared__ uint32_t head[F::kWords], desc[F::kWords];
    __shared__ uint32_t queue[2 * F::kQueue];  // (start, end) of the groups for warps
    __shared__ uint32_t n_queue;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t s = blockIdx.x * (uint64_t)F::kTile;
    const uint32_t W = (uint32_t)(n - s < (uint64_t)F::kWin ? n - s : (uint64_t)F::kWin);
    const uint32_t len = W < (uint32_t)F::kTile ? W : (uint32_t)F::kTile;
    const bool window_ends_array = s + W == n;
    auto kget = [&](uint32_t i) {
        Key<NW> r;
#pragma unroll
        for (int w = 0; w < NW; w++) r.w[w] = K[i * NW + w];
        return r;
    };
    auto kset = [&](uint32_t i, const Key<NW>& x) {
#pragma unroll
        for (int w = 0; w < NW; w++) K[i * NW + w] = x.w[w];
    };
    if (W == (uint32_t)F::kWin) {
        // all loads in flight at once
        uint64_t v[F::kWin * NW / 256];
#pragma unroll
        for (int q = 0; q < F::kWin * NW / 256; q++) v[q] = keys[s * NW + tid + q * 256];
#pragma unroll
        for (int q = 0; q < F::kWin * NW / 256; q++) K[tid + q * 256] = v[q];
    } else {
        for (uint32_t i = tid; i < W * NW; i += 256) K[i] = keys[s * NW + i];
    }
    if (tid == 0) n_queue = 0;
    __syncthreads();
    // a and b share their top bits iff (a ^ b) < 2^lo in the top word
    const uint64_t same_top = 1ull << lo;
    for (uint32_t wd = warp; wd < (uint32_t)F::kWords; wd += 8) {
        const uint32_t i = wd * 32 + lane;
        bool h = false, d = false;
        if (i < W) {
            const Key<NW> x = kget(i);
            const Key<NW> y = i > 0 ? kget(i - 1) : (s > 0 ? load_key<NW>(keys, s - 1) : key_ones<NW>());
            h = i == 0 && s == 0 ? true : (x.w[NW - 1] ^ y.w[NW - 1]) >= same_top;
            d = i > 0 && !h && key_less<NW>(x, y);
        }
        const uint32_t hb = __ballot_sync(0xFFFFFFFFu, h), db = __ballot_sync(0xFFFFFFFFu, d);
        if (lane == 0) {
            head[wd] = hb;
            desc[wd] = db;
        }
    }
    __syncthreads();
    // groups starting in this tile that hold a descent, each found from its
    // first descent (a word of descent bits a thread; descents are few: a
    // group holds two distinct keys only where keys collide on the top bits)
    auto to_big = [&](uint32_t h) {
        const unsigned long long q = atomicAdd(n_big, 1ull);
        if (q < big_cap) big[q] = s + h;
    };
    if (tid == 0 && !window_ends_array) {
        // the tile's last group, if it may run past the window with no descent
        // inside it: checked by a CTA of its own
        const uint32_t h = prev_bit(head, len - 1);
        if (h != ~0u && next_bit(head, h + 1, W) == W && !any_bit(desc, h + 1, W)) to_big(h);
    }
    for (uint32_t wd = tid; wd < (uint32_t)F::kWords; wd += 256) {
        uint32_t dm = desc[wd];
        while (dm) {
            const uint32_t jd = wd * 32 + __ffs(dm) - 1;
            dm &= dm - 1;
            const uint32_t h = prev_bit(head, jd);
            if (h == ~0u || h >= len) continue;  // the group starts in another tile
            if (any_bit(desc, h + 1, jd)) continue;  // not its first descent
            const uint32_t g1 = next_bit(head, jd + 1, W);
            if (g1 == W && !window_ends_array) {
                to_big(h);  // may run past the window
                continue;
            }
            if (g1 - h <= (uint32_t)F::kThreadSort) {
                for (uint32_t j = h + 1; j < g1; j++) {
                    const Key<NW> x = kget(j);
                    uint32_t i = j;
                    while (i > h && key_less<NW>(x, kget(i - 1))) {
                        kset(i, kget(i - 1));
                        i--;
                    }
                    kset(i, x);
                }
                for (uint32_t j = h; j < g1; j++) store_key<NW>(keys, s + j, kget(j));
            } else {
                const uint32_t q = atomicAdd(&n_queue, 1u);
                queue[2 * q] = h;
                queue[2 * q + 1] = g1;
            }
        }
    }
    __syncthreads();
    // larger groups: a warp each, by successive minima, from K to keys
    const uint32_t nq = n_queue;
    for (uint32_t q = warp; q < nq; q += 8) {
        const uint32_t g0 = queue[2 * q], g1 = queue[2 * q + 1];
        uint32_t pos = g0;
        Key<NW> prev = key_zero<NW>();
        bool first = true;
        int rounds = 0;
        while (pos < g1 && rounds < kFixWarpRounds) {
            // smallest key above prev, and its count
            Key<NW> mn = key_ones<NW>();
            bool have = false;
            for (uint32_t i = g0 + lane; i < g1; i += 32) {
                const Key<NW> x = kget(i);
                if ((first || key_less<NW>(prev, x)) && (!have || key_less<NW>(x, mn))) {
                    mn = x;
                    have = true;
                }
            }
            for (int off = 16; off; off >>= 1) {
                const Key<NW> o = shfl_key<NW>(mn, off);
                const bool oh = __shfl_xor_sync(0xFFFFFFFFu, have, off);
                if (oh && (!have || key_less<NW>(o, mn))) {
                    mn = o;
                    have = true;
                }
            }
            uint32_t c = 0;
            for (uint32_t i = g0 + lane; i < g1; i += 32) c += key_eq<NW>(kget(i), mn);
            for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
            for (uint32_t i = lane; i < c; i += 32) store_key<NW>(keys, s + pos + i, mn);
            pos += c;
            prev = mn;
            first = false;
            rounds++;
        }
        if (pos < g1 && lane == 0) {
            // too many distinct keys: rewrite the group as it was and defer it
            for (uint32_t i = g0; i < g1; i++) store_key<NW>(keys, s + i, kget(i));
            const unsigned long long b = atomicAdd(n_big, 1ull);
            if (b < big_cap) big[b] = s + g0;
        }
    }
}

// A CTA per listed group start: find the group's end, skip it if sorted,
// else sort it by successive minima through tmp (the free buffer).
template <int NW>
__global__ void __launch_bounds__(256) spread_big_kernel(uint64_t* __restrict__ keys, uint64_t* __restrict__ tmp,
                                                         uint64_t n, int lo, const uint64_t* __restrict__ list,
                                                         uint64_t n_list, ulonglong2* __restrict__ rest,
                                                         unsigned long long* __restrict__ n_rest) {
    __shared__ uint64_t s_end;
    __shared__ uint64_t redk[8 * NW];
    __shared__ uint32_t redh[8];
    __shared__ uint32_t red32[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto top = [&](uint64_t i) { return keys[i * NW + NW - 1] >> lo; };
    for (uint64_t g = blockIdx.x; g < n_list; g += gridDim.x) {
        const uint64_t gs = list[g];
        if (tid == 0) {
            const uint64_t px = top(gs);
            uint64_t l = gs + 1, step = 1, h;
            while (true) {  // first index with other top bits
                const uint64_t probe = l + step - 1;
                if (probe >= n) {
                    h = n;
                    break;
                }
                if (top(probe) != px) {
                    h = probe;
                    break;
                }
                l = probe + 1;
                step <<= 1;
            }
            while (l < h) {
                const uint64_t mid = (l + h) / 2;
                if (top(mid) == px) l = mid + 1; else h = mid;
            }
            s_end = l;
        }
        __syncthreads();
        const uint64_t ge = s_end;
        // sorted already?
        uint32_t d = 0;
        for (uint64_t i = gs + 1 + tid; i < ge; i += 256)
            d |= key_less<NW>(load_key<NW>(keys, i), load_key<NW>(keys, i - 1));
        d = __syncthreads_or(d);
        if (!d) continue;
        uint64_t pos = gs;
        Key<NW> prev = key_zero<NW>();
        bool first = true;
        int rounds = 0;
        while (pos < ge && rounds < kFixBlockRounds) {
            Key<NW> mn = key_ones<NW>();
            bool have = false;
            for (uint64_t i = gs + tid; i < ge; i += 256) {
                const Key<NW> x = load_key<NW>(keys, i);
                if ((first || key_less<NW>(prev, x)) && (!have || key_less<NW>(x, mn))) {
                    mn = x;
                    have = true;
                }
            }
            for (int off = 16; off; off >>= 1) {
                const Key<NW> o = shfl_key<NW>(mn, off);
                const bool oh = __shfl_xor_sync(0xFFFFFFFFu, have, off);
                if (oh && (!have || key_less<NW>(o, mn))) {
                    mn = o;
                    have = true;
                }
            }
            if (lane == 0) {
#pragma unroll
                for (int w = 0; w < NW; w++) redk[warp * NW + w] = mn.w[w];
                redh[warp] = have;
            }
            __syncthreads();
            have = false;
            for (int wv = 0; wv < 8; wv++) {
                Key<NW> o;
#pragma unroll
                for (int w = 0; w < NW; w++) o.w[w] = redk[wv * NW + w];
                if (redh[wv] && (!have || key_less<NW>(o, mn))) {
                    mn = o;
                    have = true;
                }
            }
            uint32_t c = 0;
            for (uint64_t i = gs + tid; i < ge; i += 256) c += key_eq<NW>(load_key<NW>(keys, i), mn);
            for (int off = 16; off; off >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
            __syncthreads();
            if (lane == 0) red32[warp] = c;
            __syncthreads();
            c = 0;
            for (int w = 0; w < 8; w++) c += red32[w];
            for (uint64_t i = tid; i < c; i += 256) store_key<NW>(tmp, pos + i, mn);
            pos += c;
            prev = mn;
            first = false;
            rounds++;
            __syncthreads();
        }
        if (pos < ge) {
            if (tid == 0) rest[atomicAdd(n_rest, 1ull)] = make_ulonglong2(gs, ge);
        } else {
            for (uint64_t i = gs * NW + tid; i < ge * NW; i += 256) keys[i] = tmp[i];
        }
        __syncthreads();
    }
}

// a and b agree on every bit at or above bit lo of the whole key (bit 0 the
// lowest bit of word 0).
template <int NW>
__device__ __forceinline__ bool same_above(const Key<NW>& a, const Key<NW>& b, int lo) {
    bool eq = true;
#pragma unroll
    for (int w = 0; w < NW; w++) {
        const int b0 = 64 * w;
        if (lo >= b0 + 64) continue;
        const uint64_t x = a.w[w] ^ b.w[w];
        eq &= (lo <= b0) ? x == 0 : (x >> (lo - b0)) == 0;
    }
    return eq;
}

// Key-value fix-up (keys with a 32-bit payload): groups of up to 16 keys
// are sorted by one thread each, pairs moving together; larger groups inside
// the window by one warp (successive minima: each round writes every copy
// of the smallest key above the previous one with its payloads); groups that
// run past the window or hold more than 64 keys go to a list, each
// listed group then to a segment sort of its own (few, for spread keys).
// Where more than `most` are listed the table is sorted by other means, so
// CTAs that see that leave the rest as it is.  (With warps that went 64 rounds
// into longer groups before listing them, and without an end to it, 1.77 ms for
// 7.5 M pairs of a satellite at k = 61, now 0.11; 0.27 for 0.33 M pairs of 3 kbp,
// now 0.03.)
template <int NW>
__global__ void __launch_bounds__(256) spread_fix_kv_kernel(uint64_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                            uint64_t n, int lo, uint64_t* __restrict__ big,
                                                            uint64_t big_cap, unsigned long long* __restrict__ n_big,
                                                            uint64_t most) {
    using F = Fix<NW>;
    __shared__ uint64_t K[F::kWin * NW];
    __shared__ uint32_t V[F::kWin];
    __shared__ uint32_t head[F::kWords], desc[F::kWords];
    __shared__ uint32_t queue[2 * F::kQueue];  // (start, end) of the groups for warps
    __shared__ uint32_t n_queue, enough;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t s = blockIdx.x * (uint64_t)F::kTile;
    const uint32_t W = (uint32_t)(n - s < (uint64_t)F::kWin ? n - s : (uint64_t)F::kWin);
    const uint32_t len = W < (uint32_t)F::kTile ? W : (uint32_t)F::kTile;
    const bool window_ends_array = s + W == n;
    auto kget = [&](uint32_t i) {
        Key<NW> r;
#pragma unroll
        for (int w = 0; w < NW; w++) r.w[w] = K[i * NW + w];
        return r;
    };
    auto kset = [&](uint32_t i, const Key<NW>& x) {
#pragma unroll
        for (int w = 0; w < NW; w++) K[i * NW + w] = x.w[w];
    };
    for (uint32_t i = tid; i < W * NW; i += 256) K[i] = keys[s * NW + i];
    for (uint32_t i = tid; i < W; i += 256) V[i] = vals[s + i];
    if (tid == 0) {
        n_queue = 0;
        enough = *(volatile unsigned long long*)n_big > most;
    }
    __syncthreads();
    if (enough) return;
    for (uint32_t wd = warp; wd < (uint32_t)F::kWords; wd += 8) {
        const uint32_t i = wd * 32 + lane;
        bool h = false, d = false;
        if (i < W) {
            const Key<NW> x = kget(i);
            const Key<NW> y = i > 0 ? kget(i - 1) : (s > 0 ? load_key<NW>(keys, s - 1) : key_ones<NW>());
            h = i == 0 && s == 0 ? true : !same_above<NW>(x, y, lo);
            d = i > 0 && !h && key_less<NW>(x, y);
        }
        const uint32_t hb = __ballot_sync(0xFFFFFFFFu, h), db = __ballot_sync(0xFFFFFFFFu, d);
        if (lane == 0) {
            head[wd] = hb;
            desc[wd] = db;
        }
    }
    __syncthreads();
    // groups found from their first descent, as in spread_fix_kernel
    auto to_big = [&](uint32_t h) {
        const unsigned long long q = atomicAdd(n_big, 1ull);
        if (q < big_cap) big[q] = s + h;
    };
    if (tid == 0 && !window_ends_array) {
        const uint32_t h = prev_bit(head, len - 1);
        if (h != ~0u && next_bit(head, h + 1, W) == W && !any_bit(desc, h + 1, W)) to_big(h);
    }
    for (uint32_t wd = tid; wd < (uint32_t)F::kWords; wd += 256) {
        uint32_t dm = desc[wd];
        while (dm) {
            const uint32_t jd = wd * 32 + __ffs(dm) - 1;
            dm &= dm - 1;
            const uint32_t h = prev_bit(head, jd);
            if (h == ~0u || h >= len) continue;
            if (any_bit(desc, h + 1, jd)) continue;
            const uint32_t g1 = next_bit(head, jd + 1, W);
            // (the keys are distinct: a warp's rounds cannot finish a longer group)
            if ((g1 == W && !window_ends_array) || g1 - h > (uint32_t)kFixWarpRounds) {
                to_big(h);
                continue;
            }
            if (g1 - h > (uint32_t)F::kThreadSort) {
                const uint32_t q = atomicAdd(&n_queue, 1u);
                queue[2 * q] = h;
                queue[2 * q + 1] = g1;
                continue;
            }
            for (uint32_t j = h + 1; j < g1; j++) {
                const Key<NW> x = kget(j);
                const uint32_t v = V[j];
                uint32_t i = j;
                while (i > h && key_less<NW>(x, kget(i - 1))) {
                    kset(i, kget(i - 1));
                    V[i] = V[i - 1];
                    i--;
                }
                kset(i, x);
                V[i] = v;
            }
            for (uint32_t j = h; j < g1; j++) {
                store_key<NW>(keys, s + j, kget(j));
                vals[s + j] = V[j];
            }
        }
    }
    __syncthreads();
    // larger groups: a warp each, from K and V to keys and vals
    // (one lane's reading for the warp: others add to n_big meanwhile)
    const bool listed = __shfl_sync(0xFFFFFFFFu, lane == 0 ? *(volatile unsigned long long*)n_big > most : 0, 0);
    const uint32_t nq = listed ? 0 : n_queue;
    for (uint32_t q = warp; q < nq; q += 8) {
        const uint32_t g0 = queue[2 * q], g1 = queue[2 * q + 1];
        uint32_t pos = g0;
        Key<NW> prev = key_zero<NW>();
        bool first = true;
        while (pos < g1) {
            Key<NW> mn = key_ones<NW>();
            bool have = false;
            for (uint32_t i = g0 + lane; i < g1; i += 32) {
                const Key<NW> x = kget(i);
                if ((first || key_less<NW>(prev, x)) && (!have || key_less<NW>(x, mn))) {
                    mn = x;
                    have = true;
                }
            }
            for (int off = 16; off; off >>= 1) {
                const Key<NW> o = shfl_key<NW>(mn, off);
                const bool oh = __shfl_xor_sync(0xFFFFFFFFu, have, off);
                if (oh && (!have || key_less<NW>(o, mn))) {
                    mn = o;
                    have = true;
                }
            }
            // every copy of mn, with its payload, in group order
            for (uint32_t b0 = g0; b0 < g1; b0 += 32) {
                const uint32_t i = b0 + lane;
                const bool eq = i < g1 && key_eq<NW>(kget(i), mn);
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, eq);
                if (eq) {
                    const uint32_t o = pos + __popc(m & ((1u << lane) - 1u));
                    store_key<NW>(keys, s + o, mn);
                    vals[s + o] = V[i];
                }
                pos += __popc(m);
            }
            prev = mn;
            first = false;
        }
    }
}

// A CTA per listed group start: the group's end (the first key differing at
// or above bit lo), and (start, end) out if the group holds a descent.
template <int NW>
__global__ void __launch_bounds__(256) spread_bounds_kernel(const uint64_t* __restrict__ keys, uint64_t n, int lo,
                                                            const uint64_t* __restrict__ list, uint64_t n_list,
                                                            ulonglong2* __restrict__ rest,
                                                            unsigned long long* __restrict__ n_rest) {
    __shared__ uint64_t s_end;
    const int tid = threadIdx.x;
    for (uint64_t g = blockIdx.x; g < n_list; g += gridDim.x) {
        const uint64_t gs = list[g];
        if (tid == 0) {
            const Key<NW> px = load_key<NW>(keys, gs);
            uint64_t l = gs + 1, step = 1, h;
            while (true) {
                const uint64_t probe = l + step - 1;
                if (probe >= n) {
                    h = n;
                    break;
                }
                if (!same_above<NW>(load_key<NW>(keys, probe), px, lo)) {
                    h = probe;
                    break;
                }
                l = probe + 1;
                step <<= 1;
            }
            while (l < h) {
                const uint64_t mid = (l + h) / 2;
                if (same_above<NW>(load_key<NW>(keys, mid), px, lo)) l = mid + 1; else h = mid;
            }
            s_end = l;
        }
        __syncthreads();
        const uint64_t ge = s_end;
        uint32_t d = 0;
        for (uint64_t i = gs + 1 + tid; i < ge; i += 256)
            d |= key_less<NW>(load_key<NW>(keys, i), load_key<NW>(keys, i - 1));
        d = __syncthreads_or(d);
        if (d && tid == 0) rest[atomicAdd(n_rest, 1ull)] = make_ulonglong2(gs, ge);
        __syncthreads();
    }
}

static int ceil_log2(uint64_t n) {
    int b = 0;
    while (b < 64 && (1ull << b) < n) b++;
    return b;
}

// MH_SPREAD_BITS (a multiple of 8 in [8, 64]) fixes the number of top bits
// sorted by passes; tests use small values to run the fix-up on small inputs.
static int spread_bits(uint64_t n) {
    static int forced = [] {
        const char* e = std::getenv("MH_SPREAD_BITS");
        int v = e ? std::atoi(e) : 0;
        return (v >= 8 && v <= 64 && v % 8 == 0) ? v : 0;
    }();
    return forced ? forced : std::max(8, ((ceil_log2(n) + 7) / 8) * 8);
}

// The count sort's spread bits: the default moved by the context's plan
// (a multiple of 8, kept in [8, 64]).
int spread_pass_bits(mh_ctx* ctx, uint64_t n) {
    const int P = spread_bits(n) + (ctx ? ctx->spread_bits_delta : 0);
    return std::min(64, std::max(8, P / 8 * 8));
}

template <int NW>
bool radix_sort_spread(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint64_t n, int skip, const uint32_t* hist) {
    using F = Fix<NW>;
    const int P = spread_pass_bits(ctx, n);
    const int bits = 64 * NW;
    if (n <= tiny_max<NW>() || n <= 1 || P + skip >= 64)
        return radix_sort<NW>(ctx, keys, alt, nullptr, nullptr, n, 0, bits - skip);
    // the top `skip` bits are equal in every key: passes over the P bits below
    const int lo = 64 - skip - P;  // within the top word
    const bool in_alt = radix_sort<NW>(ctx, keys, alt, nullptr, nullptr, n, bits - skip - P, bits - skip, hist);
    uint64_t* k = in_alt ? alt : keys;
    uint64_t* other = in_alt ? keys : alt;
    const uint64_t cap = std::max<uint64_t>(1 << 16, n / 64);
    Buf<uint64_t> list(ctx, cap), cnt(ctx, 2);
    cnt.zero();
    MH_LAUNCH_B(ctx, "spread_fixup", n * 8 * NW, (unsigned)ceil_div(n, F::kTile), 256, 0, spread_fix_kernel<NW>, k,
                n, lo, list.p, cap, (unsigned long long*)cnt.p);
    uint64_t n_big = 0;
    read_u64(ctx, cnt.p, &n_big, 1);
    if (n_big > cap) {
        // far more long or crowded groups than evenly spread keys give: sort fully
        return in_alt != radix_sort<NW>(ctx, k, other, nullptr, nullptr, n, 0, bits - skip);
    }
    if (n_big) {
        Buf<ulonglong2> rest(ctx, n_big);
        MH_LAUNCH(ctx, "spread_fixup_big", (unsigned)std::min<uint64_t>(n_big, (uint64_t)ctx->num_sms * 8), 256, 0,
                  spread_big_kernel<NW>, k, other, n, lo, list.p, n_big, rest.p, (unsigned long long*)(cnt.p + 1));
        uint64_t n_rest = 0;
        read_u64(ctx, cnt.p + 1, &n_rest, 1);
        if (n_rest) {
            std::vector<ulonglong2> h(n_rest);
            MH_CUDA(cudaMemcpyAsync(h.data(), rest.p, sizeof(ulonglong2) * n_rest, cudaMemcpyDeviceToHost,
                                    ctx->stream));
            sync_and_check(ctx);
            for (const ulonglong2& seg : h) {
                const uint64_t len = seg.y - seg.x;
                if (radix_sort<NW>(ctx, k + seg.x * NW, other + seg.x * NW, nullptr, nullptr, len, 0,
                                   bits - skip - P))
                    MH_CUDA(cudaMemcpyAsync(k + seg.x * NW, other + seg.x * NW, len * 8 * NW, cudaMemcpyDeviceToDevice,
                                            ctx->stream));
            }
        }
    }
    return in_alt;
}

// Wide pairs by their `P` bits from bit lo on: a pass over (key, value) pairs
// moves 20 or 36 bytes in and out, so the bits and the pair's index go into
// one 64-bit word (P <= 32, n <= 2^32), the passes move those, and one gather
// moves the pairs, into alt and valt.  4 M reads counted at k = 99 19.6 -> 19.0
// ms, the multiple-k iteration 62.4 -> 60.2.
template <int NW>
__global__ void index_keys_kernel(const uint64_t* __restrict__ keys, uint64_t n, int lo, int P,
                                  uint64_t* __restrict__ out) {
    const uint64_t mask = (1ull << P) - 1;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = (key_shr<NW>(load_key<NW>(keys, i), lo).w[0] & mask) << 32 | i;
}

template <int NW>
__global__ void index_gather_kernel(const uint64_t* __restrict__ idx, uint64_t n, const uint64_t* __restrict__ keys,
                                    const uint32_t* __restrict__ vals, uint64_t* __restrict__ kout,
                                    uint32_t* __restrict__ vout) {
    constexpr int U = 4;  // pairs a thread has in flight
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += U * stride) {
        uint32_t j[U], v[U];
        Key<NW> x[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i + u * stride < n) j[u] = (uint32_t)idx[i + u * stride];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i + u * stride < n) {
                x[u] = load_key<NW>(keys, j[u]);
                v[u] = vals[j[u]];
            }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (i + u * stride < n) {
                store_key<NW>(kout, i + u * stride, x[u]);
                vout[i + u * stride] = v[u];
            }
    }
}

// False (and nothing done) where the two words a pair do not fit the
// context's memory: the passes then move the pairs.
template <int NW>
static bool sort_by_index(mh_ctx* ctx, const uint64_t* keys, uint64_t* alt, const uint32_t* vals, uint32_t* valt,
                          uint64_t n, int lo, int P) {
    if (n > (1ull << 32) || P > 32) return false;
    try {
        Buf<uint64_t> a(ctx, n), b(ctx, n);
        MH_LAUNCH_B(ctx, "index_keys", n * (8 * NW + 8), grid_for(ctx, n, 256), 256, 0, index_keys_kernel<NW>, keys, n,
                    lo, P, a.p);
        const bool in_b = radix_sort<1>(ctx, a.p, b.p, nullptr, nullptr, n, 32, 32 + P);
        MH_LAUNCH_B(ctx, "index_gather", n * (16 * NW + 16), grid_for(ctx, n, 1024), 256, 0, index_gather_kernel<NW>,
                    in_b ? b.p : a.p, n, keys, vals, alt, valt);
    } catch (const Error& e) {
        if (e.code != MH_ENOMEM) throw;
        return false;  // (the pairs are where they were)
    }
    return true;
}

// Distinct keys with a 32-bit payload (a solid table and its counts): the
// same spread order (passes over the top P bits of the top word below
// `skip` constant bits, then the key-value fix-up).  Keys whose top bits are
// crowded (more groups past the fix-up's sorts than `most`) are sorted fully:
// a group's own sort is ten launches and more, some 35 us, and a full sort 8 to
// 30 passes whose time grows with n.  Whole path of a sequence of 3 kbp read
// 1,000 times, k = 61, 333,534 pairs: 2.6 ms, 3.6 by up to 256 groups; of 30 kbp,
// k = 31, 3.4 M pairs, 105 groups: 2.2 for 7.8.
// Returns true when the result is in alt / valt.
template <int NW>
bool radix_sort_spread_kv(mh_ctx* ctx, uint64_t* keys, uint64_t* alt, uint32_t* vals, uint32_t* valt, uint64_t n,
                          int skip) {
    using F = Fix<NW>;
    const int P = spread_bits(n);
    const int bits = 64 * NW;
    // small tables (below 2^20 keys, or MH_SPREAD_KV_MIN for tests): the full
    // sort, which needs no read-back of the fix-up's list
    // (wide keys from 2^12 on: 17 to 32 passes cost more than the read-back)
    static const uint64_t kv_min = [] {
        const char* e = std::getenv("MH_SPREAD_KV_MIN");
        return e ? (uint64_t)std::strtoull(e, nullptr, 10) : NW == 1 ? (uint64_t)1 << 20 : (uint64_t)1 << 12;
    }();
    if (n < std::max<uint64_t>(kv_min, 2) || P + skip >= bits)
        return radix_sort<NW>(ctx, keys, alt, vals, valt, n, 0, bits - skip);
    const int lo = bits - skip - P;  // groups: keys equal at and above bit lo of the whole key
    // two words: only while the gather's reads come from L2 (beyond, it costs
    // more than three passes over pairs save: 3 M reads at k = 61 8.7 ms for 8.3)
    const bool by_index =
        (NW == 4 || (NW == 2 && n * 20 <= (96u << 20))) && sort_by_index<NW>(ctx, keys, alt, vals, valt, n, lo, P);
    const bool in_alt =
        by_index || radix_sort<NW>(ctx, keys, alt, vals, valt, n, bits - skip - P, bits - skip);
    uint64_t* k = in_alt ? alt : keys;
    uint64_t* ko = in_alt ? keys : alt;
    uint32_t* v = in_alt ? valt : vals;
    uint32_t* vo = in_alt ? vals : valt;
    constexpr uint64_t kMaxSegments = 256;
    // (MH_SPREAD_KV_MIN: tests sort the groups of small tables too)
    static const bool all_groups = std::getenv("MH_SPREAD_KV_MIN") != nullptr;
    const uint64_t most = all_groups ? kMaxSegments : std::min(kMaxSegments, std::max<uint64_t>(2, n >> 17));
    Buf<uint64_t> list(ctx, kMaxSegments), cnt(ctx, 2);
    cnt.zero();
    MH_LAUNCH_B(ctx, "spread_fixup_kv", n * (8 * NW + 4), (unsigned)ceil_div(n, F::kTile), 256, 0,
                spread_fix_kv_kernel<NW>, k, v, n, lo, list.p, kMaxSegments, (unsigned long long*)cnt.p, most);
    uint64_t n_big = 0;
    read_u64(ctx, cnt.p, &n_big, 1);
    if (n_big > most) return in_alt != radix_sort<NW>(ctx, k, ko, v, vo, n, 0, bits - skip);
    if (!n_big) return in_alt;
    Buf<ulonglong2> rest(ctx, n_big);
    MH_LAUNCH(ctx, "spread_bounds", (unsigned)n_big, 256, 0, spread_bounds_kernel<NW>, k, n, lo, list.p, n_big,
              rest.p, (unsigned long long*)(cnt.p + 1));
    uint64_t n_rest = 0;
    read_u64(ctx, cnt.p + 1, &n_rest, 1);
    if (!n_rest) return in_alt;
    std::vector<ulonglong2> h(n_rest);
    MH_CUDA(cudaMemcpyAsync(h.data(), rest.p, sizeof(ulonglong2) * n_rest, cudaMemcpyDeviceToHost, ctx->stream));
    sync_and_check(ctx);
    for (const ulonglong2& seg : h) {
        const uint64_t len = seg.y - seg.x;
        if (radix_sort<NW>(ctx, k + seg.x * NW, ko + seg.x * NW, v + seg.x, vo + seg.x, len, 0, bits - skip - P)) {
            MH_CUDA(cudaMemcpyAsync(k + seg.x * NW, ko + seg.x * NW, len * 8 * NW, cudaMemcpyDeviceToDevice,
                                    ctx->stream));
            MH_CUDA(cudaMemcpyAsync(v + seg.x, vo + seg.x, len * 4, cudaMemcpyDeviceToDevice, ctx->stream));
        }
    }
    return in_alt;
}

template bool radix_sort_spread_kv<1>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int);
template bool radix_sort_spread_kv<2>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int);
template bool radix_sort_spread_kv<4>(mh_ctx*, uint64_t*, uint64_t*, uint32_t*, uint32_t*, uint64_t, int);

template bool radix_sort_spread<1>(mh_ctx*, uint64_t*, uint64_t*, uint64_t, int, const uint32_t*);
template bool radix_sort_spread<2>(mh_ctx*, uint64_t*, uint64_t*, uint64_t, int, const uint32_t*);
template bool radix_sort_spread<4>(mh_ctx*, uint64_t*, uint64_t*, uint64_t, int, const uint32_t*);

// ------------------------------------------------------------------ scans
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__global__ void scan_reduce_kernel(const T* __restrict__ in, uint64_t n, uint64_t* __restrict__ sums) {
    uint64_t b0 = (uint64_t)blockIdx.x * kScanTile;
    uint64_t acc = 0;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
        uint64_t idx = b0 + i;
        if (idx < n) acc += (uint64_t)in[idx];
    }
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    __shared__ uint64_t ws[kScanThreads / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t t = 0;
        for (int w = 0; w < kScanThreads / 32; w++) t += ws[w];
        sums[blockIdx.x] = t;
    }
}

// In-place exclusive scan of at most kScanTile values by one block; writes the total to a[n].
__global__ void scan_small_kernel(uint64_t* a, uint64_t n) {
    __shared__ uint64_t s[kScanTile];
    __shared__ uint64_t ws[kScanThreads / 32];
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) s[i] = (uint64_t)i < n ? a[i] : 0;
    __syncthreads();
    uint64_t loc[kScanItems];
    uint64_t t = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; j++) {
        loc[j] = t;
        t += s[threadIdx.x * kScanItems + j];
    }
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = t;
    for (int off = 1; off < 32; off <<= 1) {
        uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    uint64_t wpre = 0;
    for (int w = 0; w < warp; w++) wpre += ws[w];
    uint64_t pre = wpre + x - t;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScanItems; j++) s[threadIdx.x * kScanItems + j] = pre + loc[j];
    __syncthreads();
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads)
        if ((uint64_t)i < n) a[i] = s[i];
    if (threadIdx.x == kScanThreads - 1) a[n] = pre + t;
}

// Each thread scans its own run of kScanItems consecutive inputs in
// registers (read and written straight from and to global memory: a warp's
// runs are one contiguous span), then the block adds the runs' prefixes.
template <class T>
__global__ void scan_down_kernel(const T* __restrict__ in, uint64_t n, const uint64_t* __restrict__ offs,
                                 uint64_t* __restrict__ out) {
    __shared__ uint64_t ws[kScanThreads / 32];
    const uint64_t b = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
    uint64_t loc[kScanItems];
    uint64_t t = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; j++) {
        loc[j] = t;
        t += b + j < n ? (uint64_t)in[b + j] : 0;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = t;
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    uint64_t wpre = 0;
    for (int w = 0; w < warp; w++) wpre += ws[w];
    const uint64_t pre = offs[blockIdx.x] + wpre + x - t;
#pragma unroll
    for (int j = 0; j < kScanItems; j++)
        if (b + j < n) out[b + j] = pre + loc[j];
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = offs[gridDim.x];
}

// Up to kScanOne values by one CTA: one launch where the three kernels and
// their buffer are six operations of the stream: five scans of a set of 10,000
// reads 0.12 -> 0.05 ms.
constexpr uint64_t kScanOne = 16384;
template <class T>
__global__ void __launch_bounds__(1024) scan_one_kernel(const T* __restrict__ in, uint32_t n, uint64_t* __restrict__ out) {
    constexpr uint32_t kItems = 8;
    __shared__ uint64_t ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t carry = 0;
    for (uint32_t base = 0; base < n; base += 1024 * kItems) {
        const uint32_t b = base + threadIdx.x * kItems;
        uint64_t v[kItems], t = 0;
#pragma unroll
        for (uint32_t j = 0; j < kItems; j++) v[j] = b + j < n ? (uint64_t)in[b + j] : 0;
#pragma unroll
        for (uint32_t j = 0; j < kItems; j++) {
            const uint64_t x = v[j];
            v[j] = t;
            t += x;
        }
        uint64_t x = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[warp] = x;
        __syncthreads();
        uint64_t s = ws[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= o) s += y;
        }
        const uint64_t before = __shfl_sync(0xFFFFFFFFu, s, warp ? warp - 1 : 0);
        const uint64_t pre = carry + (warp ? before : 0) + x - t;
#pragma unroll
        for (uint32_t j = 0; j < kItems; j++)
            if (b + j < n) out[b + j] = pre + v[j];
        carry += __shfl_sync(0xFFFFFFFFu, s, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = carry;
}

template <class T>
static void exclusive_scan_impl(mh_ctx* ctx, const T* in, uint64_t* out, uint64_t n) {
    if (n == 0) {
        MH_CUDA(cudaMemsetAsync(out, 0, sizeof(uint64_t), ctx->stream));
        return;
    }
    if (n <= kScanOne) {
        MH_LAUNCH(ctx, "scan_one", 1, 1024, 0, scan_one_kernel<T>, in, (uint32_t)n, out);
        return;
    }
    uint64_t nb = ceil_div(n, kScanTile);
    Buf<uint64_t> sums(ctx, nb + 1);
    MH_LAUNCH(ctx, "scan_reduce", (unsigned)nb, kScanThreads, 0, scan_reduce_kernel<T>, in, n, sums.p);
    if (nb <= (uint64_t)kScanTile) {
        MH_LAUNCH(ctx, "scan_small", 1, kScanThreads, 0, scan_small_kernel, sums.p, nb);
    } else {
        Buf<uint64_t> sums2(ctx, nb + 1);
        exclusive_scan_impl<uint64_t>(ctx, sums.p, sums2.p, nb);
        MH_CUDA(cudaMemcpyAsync(sums.p, sums2.p, sizeof(uint64_t) * (nb + 1), cudaMemcpyDeviceToDevice,
                                ctx->stream));
    }
    MH_LAUNCH(ctx, "scan_down", (unsigned)nb, kScanThreads, 0, scan_down_kernel<T>, in, n, sums.p, out);
}

void exclusive_scan_u64(mh_ctx* ctx, const uint64_t* in, uint64_t* out, uint64_t n) {
    exclusive_scan_impl<uint64_t>(ctx, in, out, n);
}
void exclusive_scan_u32(mh_ctx* ctx, const uint32_t* in, uint64_t* out, uint64_t n) {
    exclusive_scan_impl<uint32_t>(ctx, in, out, n);
}

}  // namespace mh

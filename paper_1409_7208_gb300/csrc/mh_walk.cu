// Contigs for the next k of a multiple-k iteration (the paper, Sec. 2 fourth
// paragraph and Sec. 3, builds the graph for a list of increasing k and carries
// the previous k's contigs into the next graph).  Graph cleaning and contig
// assembly are not part of this library, so a contig here is a random walk of
// the graph E = solid + mercy:
//
//   walk w   counter-based random values r(w, j) = SplitMix64 output number
//            (w << 24) + j of the stream seeded with `seed` (Steele, Lea &
//            Flood 2014: state advanced by 0x9E3779B97F4A7C15, then two
//            xor-shift-multiply rounds);
//            start edge: index r(w, 0) mod |E| of solid followed by mercy
//            (each ascending), the contig is its k+1 symbols;
//            step j = 1, 2, ...: the node is the contig's last k symbols;
//            its out-edges are the edges of E with that k-prefix, taken in
//            label order; with none the walk stops (dead end), otherwise it
//            appends the label of out-edge r(w, j) mod (their number); it
//            also stops at max_len symbols.
//
// A warp runs one walk: each step finds, in each table, the entries whose
// k-prefix is the node (node.A .. node.T) from a bucket index over the top
// bits of the keys (about 16 keys a bucket): the lanes read the bucket in one
// load and a ballot gives the first entry >= node.A, so a step costs a few
// dependent loads.  Walks write into fixed slots of max_len bytes, compacted
// afterwards.
//
// Long walks take links made beforehand instead (use_links): for every edge
// where its out-edges lie in both tables (a join of suffixes against
// prefixes, through the same index), and, by doubling, where 4 and 16 steps
// lead while every node on the way has one out-edge, with their symbols.  A
// walk is then a thread that loads its edge's link and both jumps at once and
// takes the longest that holds: one memory latency for up to 16 symbols
// instead of one for each.  (A node with one out-edge needs no random value,
// so jumps skip none that counts.)
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "mh_internal.cuh"

namespace mh {

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t c) {
    uint64_t z = seed + (c + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Top `bits` bits of a (k+1)-mer key (bits <= 2(k+1), bits <= 32).
template <int NW>
__device__ __forceinline__ uint64_t top_bits(const Key<NW>& x, int K1, int bits) {
    return key_shr<NW>(x, 2 * K1 - bits).w[0];
}

// off[b] = first entry of the sorted table whose top bits are >= b, for
// b = 0 .. 2^bits (thread per entry; each boundary written by one thread).
template <int NW>
__global__ void table_index_kernel(const uint64_t* __restrict__ T, uint64_t n, int K1, int bits,
                                   uint64_t* __restrict__ off) {
    const uint64_t nb = 1ull << bits;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t b = top_bits<NW>(load_key<NW>(T, i), K1, bits);
        const uint64_t b0 = i == 0 ? 0 : top_bits<NW>(load_key<NW>(T, i - 1), K1, bits) + 1;
        for (uint64_t x = b0; x <= b; x++) off[x] = i;
        if (i == n - 1)
            for (uint64_t x = b + 1; x <= nb; x++) off[x] = n;
    }
}

// Labels (bit c for label c) of the out-edges of node v in both tables at
// once: half-warp 0 searches the solid table, half-warp 1 the mercy table,
// each within [lo, hi), the bucket of v.A in its own table.  A half reads
// the bucket 16 entries at a time and finds the first entry >= v.A by a
// ballot (the bucket's end if none); its lanes 0..3 then read the entries
// from there (into the next bucket when the index covers the label's bits,
// for tiny k).  Every lane gets the union of both masks.
template <int NW>
__device__ __forceinline__ uint32_t out_labels(const uint64_t* __restrict__ T, uint64_t n, uint64_t lo, uint64_t hi,
                                               const Key<NW>& v, int lane) {
    const int half = lane >> 4, hl = lane & 15;
    const Key<NW> q = key_shl<NW>(v, 2);
    uint64_t pos = hi, base = lo;
    bool done = base >= hi;
    while (__ballot_sync(0xFFFFFFFFu, !done)) {
        const uint64_t i = base + hl;
        const bool ge = !done && i < hi && !key_less<NW>(load_key<NW>(T, i), q);
        const uint32_t m = (__ballot_sync(0xFFFFFFFFu, ge) >> (16 * half)) & 0xFFFFu;
        if (!done) {
            if (m) {
                pos = base + __ffs(m) - 1;
                done = true;
            } else {
                base += 16;
                done = base >= hi;
            }
        }
    }
    bool hit = false;
    uint32_t label = 0;
    if (hl < 4 && pos + hl < n) {
        const Key<NW> e = load_key<NW>(T, pos + hl);
        hit = key_eq<NW>(key_shr<NW>(e, 2), v);
        label = (uint32_t)(e.w[0] & 3u);
    }
    // entries of prefix v are consecutive from pos: lane l counts if lanes 0..l of its half all match
    const uint32_t hm = (__ballot_sync(0xFFFFFFFFu, hit) >> (16 * half)) & 0xFu;
    const uint32_t run = __ffs(~hm) - 1;  // matching entries from pos (at most 4)
    uint32_t mask = (hl < (int)run) ? (1u << label) : 0u;
    for (int o = 16; o; o >>= 1) mask |= __shfl_xor_sync(0xFFFFFFFFu, mask, o);
    return mask;
}

// One warp per walk (the searches of a step are warp-wide).  The bucket of
// the next step's node does not depend on the label the step picks when the
// index's bits stop short of the last two symbols (2 K1 - bits >= 4): its
// bounds are then loaded one step ahead, while this step searches, so that
// a step waits for one memory access (the bucket) instead of two.
template <int NW>
__global__ void walk_kernel(const uint64_t* __restrict__ S, uint64_t nS, const uint64_t* __restrict__ offS,
                            const uint64_t* __restrict__ M, uint64_t nM, const uint64_t* __restrict__ offM,
                            int bits, int k, uint64_t n_walks, uint32_t max_len, uint64_t seed,
                            uint8_t* __restrict__ slots, uint64_t* __restrict__ lens,
                            unsigned long long* __restrict__ next_walk) {
    const int K1 = k + 1;
    const int lane = threadIdx.x & 31;
    const uint64_t E = nS + nM;
    // this lane's half-warp searches one table
    const bool mer = (lane >> 4) != 0;
    const uint64_t* T = mer ? M : S;
    const uint64_t n = mer ? nM : nS;
    const uint64_t* off = mer ? offM : offS;
    const bool ahead = 2 * K1 - bits >= 4;
    // bounds of the bucket of node v's query v.A
    auto bucket = [&](const Key<NW>& v, uint64_t& lo, uint64_t& hi) {
        lo = hi = 0;
        if (n) {
            const uint64_t b = top_bits<NW>(key_shl<NW>(v, 2), K1, bits);
            lo = off[b];
            hi = off[b + 1];
        }
    };
    // walks are taken one at a time from a counter: walks differ in length
    // (a dead end ends one early), and a warp that finishes takes the next
    for (;;) {
        uint64_t w = 0;
        if (lane == 0) w = atomicAdd(next_walk, 1ull);
        w = __shfl_sync(0xFFFFFFFFu, w, 0);
        if (w >= n_walks) break;
        uint8_t* out = slots + w * max_len;
        const uint64_t s = splitmix64_at(seed, w << 24) % E;
        Key<NW> x = s < nS ? load_key<NW>(S, s) : load_key<NW>(M, s - nS);
        for (int i = lane; i < K1; i += 32) out[i] = "ACGT"[key_sym<NW>(x, K1, i)];
        uint32_t len = K1;
        Key<NW> v = key_low<NW>(x, 2 * k);
        uint64_t lo, hi;
        bucket(v, lo, hi);
        for (uint32_t j = 1; len < max_len; j++) {
            // the next node's bucket, for any label (when `ahead`)
            uint64_t nlo = 0, nhi = 0;
            if (ahead) bucket(key_low<NW>(key_shl<NW>(v, 2), 2 * k), nlo, nhi);
            const uint32_t mask = out_labels<NW>(T, n, lo, hi, v, lane);
            if (!mask) break;
            uint32_t r = (uint32_t)(splitmix64_at(seed, (w << 24) + j) % (uint64_t)__popc(mask));
            uint32_t m = mask;
            while (r--) m &= m - 1;
            const uint32_t c = __ffs(m) - 1;
            x = key_shl<NW>(v, 2);
            x.w[0] |= c;
            if (lane == 0) out[len] = "ACGT"[c];
            len++;
            v = key_low<NW>(x, 2 * k);
            if (ahead) {
                lo = nlo;
                hi = nhi;
            } else {
                bucket(v, lo, hi);
            }
        }
        if (lane == 0) lens[w] = len;
    }
}

// Where an edge leads: the first of its out-edges in the solid table (x) and
// in the mercy table (y), and their labels (z: bits 0-3 solid, 4-7 mercy).
// A jump: the edge reached (x, kNoJump if some node on the way has not
// exactly one out-edge) and the symbols appended (y, the last one lowest).
constexpr uint32_t kNoJump = 0xFFFFFFFFu;

// First entry of the table at or after q, within q's bucket.
template <int NW>
__device__ __forceinline__ uint64_t bucket_lb(const uint64_t* __restrict__ T, const uint64_t* __restrict__ off,
                                              const Key<NW>& q, int K1, int bits) {
    const uint64_t b = top_bits<NW>(q, K1, bits);
    uint64_t lo = off[b], hi = off[b + 1];
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (key_less<NW>(load_key<NW>(T, mid), q)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Links and one-step jumps of the edges T[0, n), numbered from `first`
// (thread per edge: neighbours' suffixes ascend, so neighbouring threads
// search the same buckets).
template <int NW>
__global__ void __launch_bounds__(256) walk_links_kernel(const uint64_t* __restrict__ T, uint64_t n, uint64_t first,
                                                         const uint64_t* __restrict__ S, uint64_t nS,
                                                         const uint64_t* __restrict__ offS,
                                                         const uint64_t* __restrict__ M, uint64_t nM,
                                                         const uint64_t* __restrict__ offM, int bits, int k,
                                                         uint4* __restrict__ link, uint2* __restrict__ jump) {
    const int K1 = k + 1;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const Key<NW> v = key_low<NW>(load_key<NW>(T, i), 2 * k), q = key_shl<NW>(v, 2);
        uint4 l = make_uint4(0, 0, 0, 0);
        auto find = [&](const uint64_t* __restrict__ A, uint64_t nA, const uint64_t* __restrict__ off, uint32_t& at) {
            uint32_t mask = 0;
            if (!nA) return mask;
            uint64_t p = bucket_lb<NW>(A, off, q, K1, bits);
            at = (uint32_t)p;
            for (int t = 0; t < 4 && p < nA; t++, p++) {
                const Key<NW> e = load_key<NW>(A, p);
                if (!key_eq<NW>(key_shr<NW>(e, 2), v)) break;
                mask |= 1u << (e.w[0] & 3u);
            }
            return mask;
        };
        const uint32_t ms = find(S, nS, offS, l.x), mm = find(M, nM, offM, l.y);
        l.z = ms | (mm << 4);
        link[first + i] = l;
        const uint32_t m = ms | mm;
        uint2 j = make_uint2(kNoJump, 0);
        if (__popc(m) == 1) j = make_uint2(ms ? l.x : (uint32_t)nS + l.y, __ffs(m) - 1);
        jump[first + i] = j;
    }
}

// *n_ends += edges without out-edges among kEndSamples evenly spaced ones.
constexpr uint32_t kEndSamples = 4096;
template <int NW>
__global__ void __launch_bounds__(64) walk_ends_kernel(const uint64_t* __restrict__ S, uint64_t nS,
                                                       const uint64_t* __restrict__ offS,
                                                       const uint64_t* __restrict__ M, uint64_t nM,
                                                       const uint64_t* __restrict__ offM, int bits, int k,
                                                       unsigned long long* __restrict__ n_ends) {
    const uint32_t t = blockIdx.x * 64 + threadIdx.x;
    const uint64_t i = (nS + nM) / kEndSamples * t;
    const Key<NW> v = key_low<NW>(i < nS ? load_key<NW>(S, i) : load_key<NW>(M, i - nS), 2 * k);
    const Key<NW> q = key_shl<NW>(v, 2);
    auto leaves = [&](const uint64_t* __restrict__ A, uint64_t nA, const uint64_t* __restrict__ off) {
        if (!nA) return false;
        const uint64_t p = bucket_lb<NW>(A, off, q, k + 1, bits);
        return p < nA && key_eq<NW>(key_shr<NW>(load_key<NW>(A, p), 2), v);
    };
    const bool end = !leaves(S, nS, offS) && !leaves(M, nM, offM);
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, end);
    if (m && (threadIdx.x & 31) == 0) atomicAdd(n_ends, (unsigned long long)__popc(m));
}

// Jumps of twice the steps from jumps of `steps` steps.
__global__ void __launch_bounds__(256) walk_double_kernel(const uint2* __restrict__ in, uint64_t n, int steps,
                                                          uint2* __restrict__ out) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        uint2 a = in[i];
        if (a.x != kNoJump) {
            const uint2 b = in[a.x];
            a = make_uint2(b.x, (a.y << (2 * steps)) | b.y);
        }
        out[i] = a;
    }
}

// A thread per walk, symbols packed 16 a word (first symbol highest) into
// its slot of `stride` words.  Bound by the latency of the three loads of a
// step (a few threads an SM): 16,384 walks of up to 10,000 symbols over 25 M
// edges 0.5 ms, 26.6 ms by a search a symbol.
template <int NW>
__global__ void __launch_bounds__(64) walk_linked_kernel(const uint64_t* __restrict__ S, uint64_t nS,
                                                         const uint64_t* __restrict__ M, uint64_t nM,
                                                         const uint4* __restrict__ link,
                                                         const uint2* __restrict__ jump4,
                                                         const uint2* __restrict__ jump16, int k, uint64_t n_walks,
                                                         uint32_t max_len, uint64_t seed, uint64_t stride,
                                                         uint32_t* __restrict__ slots, uint64_t* __restrict__ lens) {
    const int K1 = k + 1;
    const uint64_t E = nS + nM;
    const uint64_t w = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (w >= n_walks) return;
    uint32_t* out = slots + w * stride;
    uint64_t acc = 0;   // symbols not written yet, the last one lowest
    int pending = 0;
    auto append = [&](uint32_t syms, int n) {
        acc = (acc << (2 * n)) | syms;
        pending += n;
        if (pending >= 16) {
            pending -= 16;
            *out++ = (uint32_t)(acc >> (2 * pending));
        }
    };
    const uint64_t s = splitmix64_at(seed, w << 24) % E;
    const Key<NW> x = s < nS ? load_key<NW>(S, s) : load_key<NW>(M, s - nS);
    for (int i = 0; i < K1; i++) append(key_sym<NW>(x, K1, i), 1);
    uint32_t cur = (uint32_t)s, len = K1;
    while (len < max_len) {
        const uint2 a = jump16[cur], b = jump4[cur];
        const uint4 l = link[cur];
        if (a.x != kNoJump && len + 16 <= max_len) {
            append(a.y, 16);
            cur = a.x;
            len += 16;
        } else if (b.x != kNoJump && len + 4 <= max_len) {
            append(b.y, 4);
            cur = b.x;
            len += 4;
        } else {
            const uint32_t ms = l.z & 15u, mm = l.z >> 4, mask = ms | mm;
            if (!mask) break;
            uint32_t m = mask;
            const uint32_t n = __popc(mask);
            if (n > 1) {
                // step j appends symbol K1 + j - 1
                uint32_t r = (uint32_t)(splitmix64_at(seed, (w << 24) + (len - K1 + 1)) % (uint64_t)n);
                while (r--) m &= m - 1;
            }
            const uint32_t c = __ffs(m) - 1, below = (1u << c) - 1u;
            cur = (ms >> c) & 1u ? l.x + __popc(ms & below) : (uint32_t)nS + l.y + __popc(mm & below);
            append(c, 1);
            len++;
        }
    }
    if (pending) *out = (uint32_t)(acc << (2 * (16 - pending)));
    lens[w] = len;
}

// contig w: lens[w] symbols of its slot as letters at off[w] (block per contig)
__global__ void contig_unpack_kernel(const uint32_t* __restrict__ slots, uint64_t stride,
                                     const uint64_t* __restrict__ off, uint8_t* __restrict__ ascii) {
    const uint64_t w = blockIdx.x;
    const uint64_t o = off[w], len = off[w + 1] - o;
    const uint32_t* s = slots + w * stride;
    for (uint64_t i = threadIdx.x; i < len; i += blockDim.x)
        ascii[o + i] = "ACGT"[(s[i >> 4] >> (30 - 2 * (uint32_t)(i & 15))) & 3u];
}

// contig w: lens[w] bytes from its slot to off[w]
__global__ void contig_compact_kernel(const uint8_t* __restrict__ slots, uint32_t max_len,
                                      const uint64_t* __restrict__ off, uint8_t* __restrict__ ascii) {
    const uint64_t w = blockIdx.x;
    const uint64_t o = off[w], len = off[w + 1] - o;
    for (uint64_t i = threadIdx.x; i < len; i += blockDim.x) ascii[o + i] = slots[w * max_len + i];
}

// Whether n_walks walks of up to max_len symbols over E edges take links.
// A step by search costs about 2.7 us of dependent loads whatever E is (26.6
// ms for 10,000 steps, 16,384 walks at once); links and jumps cost about 54
// us a million edges (1.3 ms for 25 M edges) and the walks by them 0.5 ms.
// They even out near E = 49,000 max_len; the line is drawn at 20,000, since
// doubling over arrays far beyond L2 costs more an edge.
// Walks end at dead ends, so max_len is only as many steps as they could make:
// from 2^22 edges on the dead ends among some edges are counted before links are
// made (10 us), and the longest of n_walks walks is taken as ln(n_walks) times
// the mean distance of one (2,000 walks over 17.9 M edges, 1 % of them dead ends:
// 0.8 ms by search, 1.2 by links; 18.4 M edges of reads that overlap nowhere 0.26
// and 1.44).  MH_WALK_LINKS=0 / 1 decides it for tests.
static int links_switch() {
    static const int v = [] {
        const char* e = std::getenv("MH_WALK_LINKS");
        return e ? std::atoi(e) : -1;
    }();
    return v;
}

static bool links_pay(const mh_ctx* ctx, uint64_t E, uint64_t n_walks, double steps) {
    const uint64_t rounds = ceil_div(n_walks, (uint64_t)ctx->num_sms * 64);
    return (double)E <= 20000.0 * steps * (double)rounds;
}

static bool use_links(const mh_ctx* ctx, uint64_t E, uint64_t n_walks, uint64_t max_len) {
    const int v = links_switch();
    if (v == 0 || E >= kNoJump) return false;
    if (v != 1 && !links_pay(ctx, E, n_walks, (double)max_len)) return false;
    // 40 bytes an edge, beside the index: within a budget that may have room for it
    return !ctx->budget || ctx->in_use + 40 * E + n_walks * (max_len / 4 + 64) < ctx->budget;
}

template <int NW>
void walk_contigs(mh_ctx* ctx, const mh_kmers* solid, const mh_kmers* mercy, uint64_t n_walks, uint32_t max_len,
                  uint64_t seed, mh_contigs* out) {
    const int k = solid->k;
    const uint64_t nS = solid->n, nM = mercy ? mercy->n : 0, E = nS + nM;
    const uint64_t* mk = mercy ? mercy->keys : nullptr;
    if (E == 0) n_walks = 0;
    bool linked = n_walks && use_links(ctx, E, n_walks, max_len);
    Buf<uint4> link;
    Buf<uint2> a, b, c;
    Buf<uint8_t> slots;
    Buf<uint64_t> lens, off, offS, offM;
    uint64_t stride = 0;  // of a walk's slot, in words or bytes
    int bits = 1;
    auto take = [&] {
        stride = linked ? ceil_div(max_len, 16) : max_len;
        // bucket indexes over the top bits: about 16 entries a bucket (a
        // thread searching for links: 4)
        const uint64_t per = linked ? 4 : 16;
        bits = 1;
        while (bits < 32 && bits < 2 * (k + 1) && (2ull << bits) * per <= std::max(nS, nM)) bits++;
        if (linked) {
            link = Buf<uint4>(ctx, E);
            a = Buf<uint2>(ctx, E);
            b = Buf<uint2>(ctx, E);
            c = Buf<uint2>(ctx, E);
        }
        slots = Buf<uint8_t>(ctx, n_walks * stride * (linked ? 4 : 1));
        lens = Buf<uint64_t>(ctx, n_walks + 1);
        off = Buf<uint64_t>(ctx, n_walks + 1);
        if (n_walks) {
            offS = Buf<uint64_t>(ctx, (1ull << bits) + 1);
            offM = Buf<uint64_t>(ctx, (1ull << bits) + 1);
        }
    };
    try {
        take();
    } catch (const Error& e) {
        // no room for the links and what they are made with: the walks need none
        if (!linked || e.code != MH_ENOMEM) throw;
        link.reset();
        a.reset();
        b.reset();
        c.reset();
        slots.reset();
        lens.reset();
        off.reset();
        offS.reset();
        linked = false;
        take();
    }
    auto index = [&] {
        if (nS)
            MH_LAUNCH(ctx, "walk_index", grid_for(ctx, nS, 256), 256, 0, table_index_kernel<NW>, solid->keys, nS,
                      k + 1, bits, offS.p);
        if (nM)
            MH_LAUNCH(ctx, "walk_index", grid_for(ctx, nM, 256), 256, 0, table_index_kernel<NW>, mk, nM, k + 1, bits,
                      offM.p);
    };
    if (n_walks) {
        index();
        if (linked && links_switch() != 1 && E >= (1ull << 22)) {
            Buf<unsigned long long> ends(ctx, 1);
            ends.zero();
            MH_LAUNCH(ctx, "walk_ends", kEndSamples / 64, 64, 0, walk_ends_kernel<NW>, solid->keys, nS, offS.p, mk, nM,
                      offM.p, bits, k, ends.p);
            uint64_t n_ends = 0;
            read_u64(ctx, reinterpret_cast<const uint64_t*>(ends.p), &n_ends, 1);
            const double far = n_ends ? std::log((double)n_walks + 1.0) * kEndSamples / (double)n_ends : max_len;
            if (!links_pay(ctx, E, n_walks, std::min((double)max_len, far))) {
                link.reset();
                a.reset();
                b.reset();
                c.reset();
                slots.reset();
                linked = false;
                stride = max_len;
                try {
                    slots = Buf<uint8_t>(ctx, n_walks * stride);
                } catch (const Error& e) {
                    // (perhaps with the coarser index)
                    if (e.code != MH_ENOMEM) throw;
                    lens.reset();
                    off.reset();
                    offS.reset();
                    offM.reset();
                    take();
                    index();
                }
            }
        }
        if (linked) {
            if (nS)
                MH_LAUNCH(ctx, "walk_links", grid_for(ctx, nS, 256), 256, 0, walk_links_kernel<NW>, solid->keys, nS,
                          (uint64_t)0, solid->keys, nS, offS.p, mk, nM, offM.p, bits, k, link.p, a.p);
            if (nM)
                MH_LAUNCH(ctx, "walk_links", grid_for(ctx, nM, 256), 256, 0, walk_links_kernel<NW>, mk, nM, nS,
                          solid->keys, nS, offS.p, mk, nM, offM.p, bits, k, link.p, a.p);
            const int g = grid_for(ctx, E, 256);
            MH_LAUNCH(ctx, "walk_double", g, 256, 0, walk_double_kernel, a.p, E, 1, b.p);
            MH_LAUNCH(ctx, "walk_double", g, 256, 0, walk_double_kernel, b.p, E, 2, a.p);
            MH_LAUNCH(ctx, "walk_double", g, 256, 0, walk_double_kernel, a.p, E, 4, b.p);
            MH_LAUNCH(ctx, "walk_double", g, 256, 0, walk_double_kernel, b.p, E, 8, c.p);
            MH_LAUNCH(ctx, "walk", (unsigned)ceil_div(n_walks, 64), 64, 0, walk_linked_kernel<NW>, solid->keys, nS, mk,
                      nM, link.p, a.p, c.p, k, n_walks, max_len, seed, stride, reinterpret_cast<uint32_t*>(slots.p),
                      lens.p);
        } else {
            Buf<uint64_t> next_walk(ctx, 1);
            next_walk.zero();
            MH_LAUNCH(ctx, "walk", grid_for(ctx, n_walks * 32, 256, 8), 256, 0, walk_kernel<NW>, solid->keys, nS,
                      offS.p, mk, nM, offM.p, bits, k, n_walks, max_len, seed, slots.p, lens.p,
                      (unsigned long long*)next_walk.p);
        }
    }
    link.reset();
    a.reset();
    b.reset();
    c.reset();
    offS.reset();
    offM.reset();
    exclusive_scan_u64(ctx, lens.p, off.p, n_walks);
    uint64_t total = 0;
    read_u64(ctx, off.p + n_walks, &total, 1);
    Buf<uint8_t> ascii(ctx, total + 16);
    if (n_walks && linked)
        MH_LAUNCH(ctx, "contig_unpack", (unsigned)n_walks, 256, 0, contig_unpack_kernel,
                  reinterpret_cast<const uint32_t*>(slots.p), stride, off.p, ascii.p);
    else if (n_walks)
        MH_LAUNCH(ctx, "contig_compact", (unsigned)n_walks, 256, 0, contig_compact_kernel, slots.p, max_len, off.p,
                  ascii.p);
    sync_and_check(ctx);
    out->k = k;
    out->n = n_walks;
    out->n_bases = total;
    out->ascii = ascii.release();
    out->offs = off.release();
}

template void walk_contigs<1>(mh_ctx*, const mh_kmers*, const mh_kmers*, uint64_t, uint32_t, uint64_t, mh_contigs*);
template void walk_contigs<2>(mh_ctx*, const mh_kmers*, const mh_kmers*, uint64_t, uint32_t, uint64_t, mh_contigs*);
template void walk_contigs<4>(mh_ctx*, const mh_kmers*, const mh_kmers*, uint64_t, uint32_t, uint64_t, mh_contigs*);

// ------------------------------------------------ reads plus contig copies
// out_ascii = reads, then `copies` copies of every contig (copy c of contig i
// is read n_reads + i * copies + c); out_offs the matching offsets.
__global__ void append_offs_kernel(const uint64_t* __restrict__ coffs, uint64_t n_contigs, uint32_t copies,
                                   uint64_t n_reads, uint64_t n_bases, uint64_t* __restrict__ out_offs) {
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r <= n_contigs * copies;
         r += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t v;
        if (r == n_contigs * copies) {
            v = n_bases + coffs[n_contigs] * copies;
        } else {
            const uint64_t i = r / copies, c = r % copies;
            v = n_bases + coffs[i] * copies + c * (coffs[i + 1] - coffs[i]);
        }
        out_offs[n_reads + r] = v;
    }
}

__global__ void append_ascii_kernel(const uint8_t* __restrict__ cascii, const uint64_t* __restrict__ coffs,
                                    uint64_t n_contigs, uint32_t copies, uint64_t n_bases,
                                    uint8_t* __restrict__ out_ascii) {
    // block per contig
    for (uint64_t i = blockIdx.x; i < n_contigs; i += gridDim.x) {
        const uint64_t b = coffs[i], len = coffs[i + 1] - b;
        for (uint32_t c = 0; c < copies; c++) {
            uint8_t* dst = out_ascii + n_bases + b * copies + c * len;
            for (uint64_t j = threadIdx.x; j < len; j += blockDim.x) dst[j] = cascii[b + j];
        }
    }
}

void pack_reads(mh_ctx* ctx, const uint8_t* d_ascii, uint64_t n_bases, const uint64_t* d_offs, uint64_t n_reads,
                mh_reads* out);

void pack_with_contigs(mh_ctx* ctx, const uint8_t* d_ascii, uint64_t n_bases, const uint64_t* d_offs,
                       uint64_t n_reads, const mh_contigs* contigs, uint32_t copies, mh_reads* out) {
    const uint64_t nc = contigs ? contigs->n : 0;
    const uint64_t extra = contigs ? contigs->n_bases * copies : 0;
    const uint64_t N = n_bases + extra, R = n_reads + nc * copies;
    Buf<uint8_t> a(ctx, N + 16);
    Buf<uint64_t> o(ctx, R + 1);
    if (n_bases) MH_CUDA(cudaMemcpyAsync(a.p, d_ascii, n_bases, cudaMemcpyDeviceToDevice, ctx->stream));
    MH_CUDA(cudaMemcpyAsync(o.p, d_offs, sizeof(uint64_t) * (n_reads + 1), cudaMemcpyDeviceToDevice, ctx->stream));
    if (nc && copies) {
        MH_LAUNCH(ctx, "append_offs", grid_for(ctx, nc * copies + 1, 256), 256, 0, append_offs_kernel, contigs->offs,
                  nc, copies, n_reads, n_bases, o.p);
        MH_LAUNCH(ctx, "append_ascii", (unsigned)std::min<uint64_t>(nc, (uint64_t)ctx->num_sms * 16), 256, 0,
                  append_ascii_kernel, contigs->ascii, contigs->offs, nc, copies, n_bases, a.p);
    }
    pack_reads(ctx, a.p, N, o.p, R, out);
}

}  // namespace mh

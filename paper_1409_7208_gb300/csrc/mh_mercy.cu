// mh_mercy_kmers: mercy (k+1)-mers (paper, Sec. 2, third paragraph).
//
//   degrees  for every solid edge x (both orientations are in the sorted
//            solid table S): out0(x) = no solid edge starts with x[1..k];
//            in0(x) = no solid edge ends with x[0..k-1].  With P = the
//            k-prefixes of S (sorted, as S is) both are a join of the
//            suffixes x[1..k] against P: out0(x) iff x's suffix is not in P,
//            in0(y) iff no x has y's prefix as its suffix.  S is cut into
//            chunks of whole nodes; for each first symbol a, the entries
//            a.s with s in the chunk's node range are a contiguous run of S
//            (found by one search per chunk boundary), and each is looked up
//            in the chunk's prefixes held in shared memory.
//   ends     the edges with out0 or in0 (the graph's dead ends, a small
//            fraction of S) go into a small open-addressing hash table with
//            their two flags, which stays in L2.
//   probe    every window against a blocked Bloom filter of the edges without
//            outdegree, four windows a lookup by the symbols they share, and
//            the few positives against the small table; every window p
//            without outdegree is recorded as a hit (its position and the end
//            of its fragment).
//   walk     a few lanes per hit: step forward to the next solid window q; if
//            q > p+1 and q has no indegree, the windows p+1..q-1 are emitted
//            (canonical keys).  Solidity: a search of the counting spectrum
//            (distinct canonical keys as mix_key images, with their run
//            lengths), in its super-k-mer bins or, where it is ascending,
//            through a bucket index on the top bits of the top word.
//   finish   sort + dedup of the candidates, counts looked up in the
//            counting spectrum, both strands, sorted.
#include "mh_super.cuh"

namespace mh {

template <int NW>
struct Slot {
    uint64_t k[NW];
    uint32_t tag;
    uint32_t flags;
};

__device__ __forceinline__ uint32_t slot_tag(uint64_t h) { return (uint32_t)(h >> 32) | 1u; }

template <int NW>
__host__ __device__ constexpr int deg_chunk() {
    return 2048 / NW;  // entries of S per chunk (16 KB of prefixes in shared memory)
}

// First index in [0, n) with S[i] >= q.
template <int NW>
__device__ __forceinline__ uint64_t lb_key(const uint64_t* __restrict__ S, uint64_t n, const Key<NW>& q) {
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (key_less<NW>(load_key<NW>(S, mid), q)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The (k+1)-mer a followed by k symbols A (a in ACGT).
template <int NW>
__device__ __forceinline__ Key<NW> first_symbol_key(uint32_t a, int k) {
    Key<NW> q = key_zero<NW>();
    q.w[0] = a;
    return key_shl<NW>(q, 2 * k);
}

// st[t] (t = 0..n_chunks): start of chunk t, the first node start at or after
// t * chunk (st[n_chunks] = n).  xb[4t + a]: first entry of S that is >= a.P_t
// where P_t is the first node of chunk t (xb[a] = start of the entries with
// first symbol a, xb[4 n_chunks + a] = their end).
template <int NW>
__global__ void degree_bounds_kernel(const uint64_t* __restrict__ S, uint64_t n, int k, uint64_t n_chunks,
                                     uint64_t* __restrict__ st, uint64_t* __restrict__ xb) {
    constexpr int C = deg_chunk<NW>();
    for (uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; g < (n_chunks + 1) * 4;
         g += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = g >> 2;
        const uint32_t a = (uint32_t)(g & 3);
        uint64_t s = t == 0 ? 0 : (t == n_chunks ? n : t * C);
        if (t > 0)
            while (s < n && key_eq<NW>(key_shr<NW>(load_key<NW>(S, s), 2), key_shr<NW>(load_key<NW>(S, s - 1), 2)))
                s++;
        if (a == 0) st[t] = s;
        uint64_t b;
        if (t == 0) {
            b = lb_key<NW>(S, n, first_symbol_key<NW>(a, k));
        } else if (s >= n) {
            b = a == 3 ? n : lb_key<NW>(S, n, first_symbol_key<NW>(a + 1, k));
        } else {
            Key<NW> q = first_symbol_key<NW>(a, k);
            const Key<NW> p = key_shr<NW>(load_key<NW>(S, s), 2);
#pragma unroll
            for (int w = 0; w < NW; w++) q.w[w] |= p.w[w];
            b = lb_key<NW>(S, n, q);
        }
        xb[g] = b;
    }
}

// Block per chunk.  fout[j] = 1 iff entry j has no outdegree (for the
// entries whose suffix falls in the chunk's node range); flags[i] = 2 iff
// entry i of the chunk has no indegree, else 0.
template <int NW>
__global__ void __launch_bounds__(256) degree_kernel(const uint64_t* __restrict__ S, int k,
                                                     const uint64_t* __restrict__ st,
                                                     const uint64_t* __restrict__ xb, uint8_t* __restrict__ fout,
                                                     uint8_t* __restrict__ flags, uint32_t* __restrict__ err) {
    constexpr int C = deg_chunk<NW>();
    constexpr int CAP = C + 4;  // a node has at most 4 entries, so a chunk at most C + 3
    __shared__ uint64_t pk[CAP * NW];
    __shared__ uint8_t found[CAP];
    const uint64_t t = blockIdx.x;
    const uint64_t p0 = st[t], p1 = st[t + 1];
    if (p1 - p0 > (uint64_t)CAP) {
        if (threadIdx.x == 0) atomicOr(err, ST_BAD_TABLE);
        return;
    }
    const uint32_t np = (uint32_t)(p1 - p0);
    {
        // all loads of the chunk in flight at once (blockDim.x == 256)
        constexpr int R = (CAP + 255) / 256;
        Key<NW> v[R];
#pragma unroll
        for (int q = 0; q < R; q++) {
            const uint32_t i = threadIdx.x + q * 256;
            if (i < np) v[q] = load_key<NW>(S, p0 + i);
        }
#pragma unroll
        for (int q = 0; q < R; q++) {
            const uint32_t i = threadIdx.x + q * 256;
            if (i < np) {
                const Key<NW> p = key_shr<NW>(v[q], 2);
#pragma unroll
                for (int w = 0; w < NW; w++) pk[i * NW + w] = p.w[w];
                found[i] = 0;
            }
        }
    }
    __syncthreads();
    auto pkey = [&](uint32_t i) {
        Key<NW> r;
#pragma unroll
        for (int w = 0; w < NW; w++) r.w[w] = pk[i * NW + w];
        return r;
    };
    for (uint32_t a = 0; a < 4; a++) {
        const uint64_t x0 = xb[t * 4 + a], x1 = xb[(t + 1) * 4 + a];
        for (uint64_t j = x0 + threadIdx.x; j < x1; j += blockDim.x) {
            const Key<NW> sfx = key_low<NW>(load_key<NW>(S, j), 2 * k);
            uint32_t lo = 0, hi = np;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (key_less<NW>(pkey(mid), sfx)) lo = mid + 1; else hi = mid;
            }
            const bool hit = lo < np && key_eq<NW>(pkey(lo), sfx);
            if (hit) found[lo] = 1;
            fout[j] = hit ? 0 : 1;
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < np; i += blockDim.x) {
        const Key<NW> p = pkey(i);
        uint32_t f = i;
        while (f > 0 && key_eq<NW>(pkey(f - 1), p)) f--;
        flags[p0 + i] = found[f] ? 0 : 2;
    }
}

// flags[i] |= fout[i]; counts the entries with a flag.
__global__ void degree_flags_kernel(const uint8_t* __restrict__ fout, uint8_t* __restrict__ flags, uint64_t n,
                                    unsigned long long* __restrict__ n_ends) {
    uint32_t ends = 0;
    const uint64_t n4 = n / 4;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n4; i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t f = reinterpret_cast<const uint32_t*>(flags)[i] | reinterpret_cast<const uint32_t*>(fout)[i];
        reinterpret_cast<uint32_t*>(flags)[i] = f;
        ends += ((f & 0xFFu) != 0) + ((f & 0xFF00u) != 0) + ((f & 0xFF0000u) != 0) + ((f >> 24) != 0);
    }
    if (blockIdx.x == 0 && threadIdx.x < n - 4 * n4) {
        const uint64_t i = 4 * n4 + threadIdx.x;
        const uint8_t f = flags[i] | fout[i];
        flags[i] = f;
        ends += f != 0;
    }
    for (int off = 16; off; off >>= 1) ends += __shfl_xor_sync(0xFFFFFFFFu, ends, off);
    if ((threadIdx.x & 31) == 0 && ends) atomicAdd(n_ends, (unsigned long long)ends);
}

// Prefilter of the edges without outdegree: a blocked Bloom filter, three
// bits of one 32-bit word per key, so a query is one load.  Its hash is one
// multiply per key word (the table keeps key_hash): the word comes from the
// product's top 32 bits, the bit positions from three 5-bit fields of its
// middle bits.
//
// Four neighbouring windows of a read share K1 - 3 symbols, their core, and
// an edge is the j-th of such a group with its symbols [3 - j, K1 - j) as the
// core, j = 0..3.  So the filter holds every edge's four cores beside the
// edge itself: a group is looked up once, and only the groups it lets
// through (some 5% and the true ones) a window each.  At least 24 bits per dead
// end, of which about half have no outdegree: 4.8 to 19 bits a key.
constexpr int kProbeGroup = 4;
template <int NW>
__device__ __forceinline__ Key<NW> probe_core(const Key<NW>& x, int j, int K1) {
    return key_low<NW>(key_shr<NW>(x, 2 * j), 2 * (K1 - kProbeGroup + 1));
}
template <int NW>
__device__ __forceinline__ uint64_t filter_hash(const Key<NW>& x) {
    uint64_t h = x.w[0] * 0x9E3779B97F4A7C15ull;
#pragma unroll
    for (int w = 1; w < NW; w++) h ^= (x.w[w] + h) * 0xBF58476D1CE4E5B9ull;
    return h;
}
__device__ __forceinline__ uint64_t filter_word(uint64_t h, uint64_t words_mask) { return (h >> 32) & words_mask; }
__device__ __forceinline__ uint32_t filter_bits(uint64_t h) {
    return (1u << ((h >> 17) & 31)) | (1u << ((h >> 22) & 31)) | (1u << ((h >> 27) & 31));
}

// Dead-end edges (oriented) with their flags into the small table; edges
// without outdegree also into the prefilter.  A CTA lists the flagged entries
// of a tile first (a few in a hundred), so that its lanes wait for their
// insertions' round trips to memory together: 3.5e8 edges 3.5 -> 0.3 ms.
constexpr int kEndsTile = 4096;
template <int NW>
__global__ void __launch_bounds__(256) ends_insert_kernel(const uint64_t* __restrict__ S, uint64_t n, int K1,
                                                          const uint8_t* __restrict__ flags,
                                                          Slot<NW>* __restrict__ table, uint64_t cap_mask,
                                                          uint32_t* __restrict__ filter, uint64_t filter_mask,
                                                          uint32_t* __restrict__ err) {
    __shared__ uint16_t list[kEndsTile];  // entry << 2 | flags (14 bits)
    __shared__ uint32_t scratch[8];
    const uint64_t base = blockIdx.x * (uint64_t)kEndsTile;
    const uint32_t i0 = threadIdx.x * 16;
    uint32_t f[4] = {0, 0, 0, 0};
    if (base + i0 + 16 <= n) {
        const uint4 v = *reinterpret_cast<const uint4*>(flags + base + i0);
        f[0] = v.x;
        f[1] = v.y;
        f[2] = v.z;
        f[3] = v.w;
    } else {
        for (uint32_t j = 0; j < 16; j++)
            if (base + i0 + j < n) f[j >> 2] |= (uint32_t)flags[base + i0 + j] << (8 * (j & 3));
    }
    uint32_t mine = 0, total;
#pragma unroll
    for (int j = 0; j < 16; j++) mine += ((f[j >> 2] >> (8 * (j & 3))) & 3u) != 0;
    uint32_t at = block_excl_scan_256(mine, scratch, &total);
#pragma unroll
    for (int j = 0; j < 16; j++) {
        const uint32_t g = (f[j >> 2] >> (8 * (j & 3))) & 3u;
        if (g) list[at++] = (uint16_t)((i0 + j) << 2 | g);
    }
    __syncthreads();
    for (uint32_t e = threadIdx.x; e < total; e += 256) {
        const uint32_t fl = list[e] & 3u;
        const Key<NW> x = load_key<NW>(S, base + (list[e] >> 2));
        if (fl & 1u) {
            uint64_t fh = filter_hash<NW>(x);
            atomicOr(&filter[filter_word(fh, filter_mask)], filter_bits(fh));
#pragma unroll
            for (int j = 0; j < kProbeGroup; j++) {
                fh = filter_hash<NW>(probe_core<NW>(x, j, K1));
                atomicOr(&filter[filter_word(fh, filter_mask)], filter_bits(fh));
            }
        }
        const uint64_t h = key_hash<NW>(x);
        const uint32_t tag = slot_tag(h);
        uint64_t s = h & cap_mask;
        bool placed = false;
        for (uint64_t probe = 0; probe <= cap_mask; probe++) {
            if (atomicCAS(&table[s].tag, 0u, tag) == 0u) {
#pragma unroll
                for (int w = 0; w < NW; w++) table[s].k[w] = x.w[w];
                table[s].flags = fl;
                placed = true;
                break;
            }
            s = (s + 1) & cap_mask;
        }
        if (!placed) atomicOr(err, ST_TABLE_FULL);
    }
}

// Flags of the oriented key x if it is a dead-end edge, else 0.
template <int NW>
__device__ __forceinline__ uint32_t ends_find(const Slot<NW>* __restrict__ table, uint64_t cap_mask,
                                              const Key<NW>& x) {
    uint64_t h = key_hash<NW>(x);
    uint32_t tag = slot_tag(h);
    uint64_t s = h & cap_mask;
    for (uint64_t probe = 0; probe <= cap_mask; probe++) {
        uint32_t t = table[s].tag;
        if (t == 0u) return 0;
        if (t == tag) {
            bool eq = true;
#pragma unroll
            for (int w = 0; w < NW; w++) eq &= table[s].k[w] == x.w[w];
            if (eq) return table[s].flags;
        }
        s = (s + 1) & cap_mask;
    }
    return 0;
}

// Bucket index over the ascending mixed spectrum keys: off[b] = first index
// whose top `bits` bits (of the top word) are >= b, for b = 0..2^bits
// (thread per key; each bucket boundary is written by exactly one thread).
template <int NW>
__global__ void canon_index_kernel(const uint64_t* __restrict__ canon, uint64_t n, int bits,
                                   uint64_t* __restrict__ off) {
    const int sh = 64 - bits;
    const uint64_t nb = 1ull << bits;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t b = canon[i * NW + NW - 1] >> sh;
        const uint64_t b0 = i == 0 ? 0 : (canon[(i - 1) * NW + NW - 1] >> sh) + 1;
        for (uint64_t x = b0; x <= b; x++) off[x] = i;
        if (i == n - 1)
            for (uint64_t x = b + 1; x <= nb; x++) off[x] = n;
    }
}

// Run length of the mixed key m in the ascending spectrum (bucket index
// off over `bits` top bits of the top word), 0 if absent.
template <int NW>
__device__ __forceinline__ uint32_t spec_find(const uint64_t* __restrict__ spec, const uint32_t* __restrict__ len,
                                              const uint64_t* __restrict__ off, int bits, const Key<NW>& m) {
    const uint64_t b = m.w[NW - 1] >> (64 - bits);
    uint64_t i = off[b];
    const uint64_t e = off[b + 1];
    for (; i < e; i++) {
        const Key<NW> v = load_key<NW>(spec, i);
        if (!key_less<NW>(v, m)) return key_eq<NW>(v, m) ? len[i] : 0u;
    }
    return 0u;
}

// Probe every window; record windows without outdegree as (position, end).
// A warp takes up to 32 fragments and numbers their groups of four windows through,
// a group a lane and step: its core is the end of its first window.  The
// groups the filter lets through queue in shared memory until eight of them
// give every lane one window to look up.  Bound by the random filter reads (a
// line of L1 a lane): four windows a lookup took 2.38e9 windows from 9.3 to
// 3.7 ms, 3 M reads at k = 31 from 1.27 to 0.56.
template <int NW>
__global__ void __launch_bounds__(256) mercy_probe_kernel(const uint32_t* __restrict__ packed,
                                                          const uint64_t* __restrict__ frag_offs, uint64_t n_frags,
                                                          int take_frags, int k, const Slot<NW>* __restrict__ ends,
                                                          uint64_t cap_mask, const uint32_t* __restrict__ filter,
                                                          uint64_t filter_mask, ulonglong2* __restrict__ hits,
                                                          uint64_t hit_cap, unsigned long long* __restrict__ n_hits) {
    constexpr int G = kProbeGroup, B = 32 / G;
    __shared__ ulonglong2 frags[8][32];      // first group's position less G x its number; end of the windows
    __shared__ ulonglong2 queue[8][32 + B];  // groups let through: position, end of the windows
    __shared__ uint64_t starts[8][32];       // number of the fragment's first group
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const int K1 = k + 1;
    auto in_filter = [&](const Key<NW>& x) {
        const uint64_t h = filter_hash<NW>(x);
        const uint32_t fm = filter_bits(h);
        return (__ldg(&filter[filter_word(h, filter_mask)]) & fm) == fm;
    };
    // the last B groups (or fewer) of the queue's n: a window a lane, their
    // hits placed by one atomic
    auto probe = [&](uint32_t n) {
        const uint32_t take = n < (uint32_t)B ? n : (uint32_t)B, e = lane / G;
        bool hit = false;
        uint64_t p = 0, end = 0;
        if (e < take) {
            const ulonglong2 q = queue[wid][n - take + e];
            p = q.x + lane % G;
            end = q.y;
            if (p < end) {
                const Key<NW> x = load_window<NW>(packed, p, K1);
                hit = in_filter(x) && (ends_find<NW>(ends, cap_mask, x) & 1u);
            }
        }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, hit);
        if (m) {
            uint64_t first = 0;
            if (lane == 0) first = atomicAdd(n_hits, (unsigned long long)__popc(m));
            first = __shfl_sync(0xFFFFFFFFu, first, 0);
            const uint64_t idx = first + __popc(m & lt);
            if (hit && idx < hit_cap) hits[idx] = make_ulonglong2(p, end);
        }
        __syncwarp();
        return n - take;
    };
    uint32_t queued = 0;
    for (uint64_t g = warp; g * take_frags < n_frags; g += n_warps) {
        const uint64_t f = g * take_frags + lane;
        uint64_t b = 0, nwin = 0;
        if (lane < take_frags && f < n_frags) {
            b = frag_offs[f];
            const uint64_t L = frag_offs[f + 1] - b;
            nwin = L > (uint64_t)k ? L - k : 0;
        }
        const uint64_t mine = (nwin + G - 1) / G;
        uint64_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint64_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
        // the fragments that have windows, side by side
        const uint32_t some = __ballot_sync(0xFFFFFFFFu, mine != 0);
        if (mine) {
            const int r = __popc(some & lt);
            starts[wid][r] = incl - mine;
            frags[wid][r] = make_ulonglong2(b - G * (incl - mine), b + nwin);
        }
        __syncwarp();
        const uint64_t start = lane < __popc(some) ? starts[wid][lane] : ~0ull;
        uint32_t before = 0;
        for (uint64_t j0 = 0; j0 < tot; j0 += 32) {
            // the fragment of group j0 + lane: the last one that starts at or before it
            const uint64_t rel = start - j0;
            const uint32_t m = __reduce_or_sync(0xFFFFFFFFu, rel < 32u ? 1u << (uint32_t)rel : 0u);
            const uint32_t idx = before + __popc(m & (0xFFFFFFFFu >> (31 - lane))) - 1;
            before += __popc(m);
            bool pass = false;
            ulonglong2 q = make_ulonglong2(0, 0);
            if (j0 + lane < tot) {
                q = frags[wid][idx];
                q.x += G * (j0 + lane);
                pass = in_filter(probe_core<NW>(load_window<NW>(packed, q.x, K1), 0, K1));
            }
            const uint32_t pm = __ballot_sync(0xFFFFFFFFu, pass);
            if (pass) queue[wid][queued + __popc(pm & lt)] = q;
            __syncwarp();
            queued += __popc(pm);
            while (queued >= (uint32_t)B) queued = probe(queued);
        }
        __syncwarp();
    }
    if (queued) probe(queued);
}

// Walk from each hit to the next solid window; emit the gap if it qualifies.
// G lanes a hit look G windows up at a time: a lookup is a chain of
// dependent reads, and an error makes K1 windows in a row unsolid.  3 Gbp at
// k = 31 3.9 ms with a lane a hit; 2.79, 2.55, 2.49 and 2.63 with 4, 8, 16 and
// 32; one job's 450 k reads 0.48, and 0.17, 0.12, 0.09 and 0.08.
// Candidates go out as mix_key images; solidity from the counting spectrum
// (run length, doubled for a palindrome, >= d) in its super-k-mer bins (BINS)
// or through its bucket index.
constexpr int kWalkLanes = 16;
template <int NW, bool BINS, int G>
__global__ void __launch_bounds__(256) mercy_walk_kernel(const uint32_t* __restrict__ packed,
                                                         const ulonglong2* __restrict__ hits, uint64_t n_hits, int k,
                                                         const Slot<NW>* __restrict__ ends, uint64_t ends_mask,
                                                         const uint64_t* __restrict__ spec,
                                                         const uint32_t* __restrict__ spec_len,
                                                         const uint64_t* __restrict__ spec_off, int spec_bits,
                                                         SuperIndex super, int d, uint64_t* __restrict__ out, uint64_t out_cap,
                                                         unsigned long long* __restrict__ counter) {
    const int K1 = k + 1, lane = threadIdx.x & 31, gl = lane % G;
    const uint32_t group = (G == 32 ? 0xFFFFFFFFu : ((1u << (G & 31)) - 1u)) << (lane - gl);
    for (uint64_t h = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) / G; h < n_hits;
         h += (uint64_t)gridDim.x * blockDim.x / G) {
        const ulonglong2 hp = hits[h];
        const uint64_t p = hp.x, end = hp.y;
        uint64_t q = end;
        bool closes = false;  // window q has no indegree
        for (uint64_t q0 = p + 1; q0 < end; q0 += G) {
            const uint64_t mine = q0 + gl;
            bool present = false;
            Key<NW> x;
            if (mine < end) {
                x = load_window<NW>(packed, mine, K1);
                const Key<NW> r = key_rc<NW>(x, K1);
                const Key<NW> c = key_less<NW>(r, x) ? r : x;
                const uint32_t len = BINS ? super_find<NW>(super, spec, spec_len, x, r, mix_key<NW>(c), K1)
                                          : spec_find<NW>(spec, spec_len, spec_off, spec_bits, mix_key<NW>(c));
                present = (uint64_t)len * (key_eq<NW>(r, x) ? 2 : 1) >= (uint64_t)d;
            }
            const uint32_t m = __ballot_sync(group, present);
            if (m) {
                const int src = __ffs(m) - 1;
                q = q0 + (src - (lane - gl));
                const bool none = lane == src && (ends_find<NW>(ends, ends_mask, x) & 2u);
                closes = __ballot_sync(group, none) != 0;
                break;
            }
        }
        if (!closes || q == p + 1) continue;
        uint64_t idx = 0;
        if (gl == 0) idx = atomicAdd(counter, (unsigned long long)(q - p - 1));
        idx = __shfl_sync(group, idx, lane - gl) + gl;
        for (uint64_t j = p + 1 + gl; j < q; j += G, idx += G) {
            if (idx >= out_cap) continue;
            Key<NW> z = load_window<NW>(packed, j, K1);
            Key<NW> rz = key_rc<NW>(z, K1);
            Key<NW> c = key_less<NW>(rz, z) ? rz : z;
            store_key<NW>(out, idx, mix_key<NW>(c));
        }
    }
}

static uint64_t next_pow2(uint64_t x) {
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

template <int NW>
void mercy_kmers(mh_ctx* ctx, const mh_reads* reads, const mh_kmers* solid, mh_kmers* out) {
    const int k = solid->k;
    const uint64_t S = solid->n;
    Buf<uint8_t> flags(ctx, S ? S : 1);
    Buf<uint64_t> stats(ctx, 2);
    stats.zero();
    if (S) {
        const uint64_t n_chunks = ceil_div(S, deg_chunk<NW>());
        Buf<uint64_t> st(ctx, n_chunks + 1), xb(ctx, 4 * (n_chunks + 1));
        Buf<uint8_t> fout(ctx, S);
        MH_LAUNCH(ctx, "mercy_degree_bounds", grid_for(ctx, 4 * (n_chunks + 1), 256), 256, 0,
                  degree_bounds_kernel<NW>, solid->keys, S, k, n_chunks, st.p, xb.p);
        MH_LAUNCH_B(ctx, "mercy_degree", 2 * S * 8 * NW + 2 * S, (unsigned)n_chunks, 256, 0, degree_kernel<NW>,
                    solid->keys, k, st.p, xb.p, fout.p, flags.p, ctx->d_status);
        MH_LAUNCH(ctx, "mercy_degree_flags", grid_for(ctx, ceil_div(S, 4), 256), 256, 0, degree_flags_kernel, fout.p,
                  flags.p, S, (unsigned long long*)stats.p);
    }
    uint64_t n_ends = 0;
    read_u64(ctx, stats.p, &n_ends, 1);
    const uint64_t cap = next_pow2(std::max<uint64_t>(2 * n_ends, 64));
    Buf<Slot<NW>> table(ctx, cap);
    table.zero();
    // prefilter: at least 24 bits per dead end and 2^20 in all
    const uint64_t fbits = next_pow2(std::max<uint64_t>(24 * n_ends, 1u << 20));
    Buf<uint32_t> filter(ctx, fbits / 32);
    filter.zero();
    if (n_ends)
        MH_LAUNCH(ctx, "mercy_ends_insert", (unsigned)ceil_div(S, (uint64_t)kEndsTile), 256, 0, ends_insert_kernel<NW>,
                  solid->keys, S, k + 1, flags.p, table.p, cap - 1, filter.p, fbits / 32 - 1, ctx->d_status);
    flags.reset();
    // solidity: the counting handle's spectrum in its bins, or ascending with
    // a bucket index (4 to 8 keys a bucket)
    if (!solid->spectrum_mixed) fail(MH_EINVAL, "mercy: the spectrum's keys are not mixed");
    Buf<uint64_t> spec_off;
    int spec_bits = 1;
    const bool super = solid->super_idx != nullptr;
    SuperIndex sx;
    if (super) {
        sx = SuperIndex{solid->super_off, solid->super_idx, solid->super_bins, solid->super_m, solid->super_main,
                        solid->n_spectrum};
    } else {
        while (spec_bits < 40 && (2ull << spec_bits) * 4 <= solid->n_spectrum) spec_bits++;
        spec_off = Buf<uint64_t>(ctx, (1ull << spec_bits) + 1);
        spec_off.zero();
        if (solid->n_spectrum)
            MH_LAUNCH(ctx, "mercy_spectrum_index", grid_for(ctx, solid->n_spectrum, 256), 256, 0,
                      canon_index_kernel<NW>, solid->spectrum, solid->n_spectrum, spec_bits, spec_off.p);
    }
    // windows without outdegree
    uint64_t hit_cap = std::max<uint64_t>(1u << 20, reads->n_packed / 256);
    // (few fragments: fewer a warp, so that there are warps for every SM)
    const int take_frags =
        (int)std::max<uint64_t>(4, std::min<uint64_t>(32, reads->n_frags / ((uint64_t)ctx->num_sms * 64)));
    Buf<ulonglong2> hits;
    uint64_t n_hits = 0;
    for (int attempt = 0; attempt < 2; attempt++) {
        hits = Buf<ulonglong2>(ctx, hit_cap);
        MH_CUDA(cudaMemsetAsync(stats.p + 1, 0, sizeof(uint64_t), ctx->stream));
        if (reads->n_frags && n_ends)
            MH_LAUNCH_B(ctx, "mercy_probe", reads->n_packed / 4,
                        grid_for(ctx, ceil_div(reads->n_frags, (uint64_t)take_frags) * 32, 256, 8), 256, 0,
                        mercy_probe_kernel<NW>, reads->packed, reads->frag_offs, reads->n_frags, take_frags, k, table.p, cap - 1,
                        filter.p, fbits / 32 - 1, hits.p, hit_cap, (unsigned long long*)(stats.p + 1));
        read_u64(ctx, stats.p + 1, &n_hits, 1);
        if (n_hits <= hit_cap) break;
        hit_cap = n_hits;
    }
    // the gaps behind the hits
    // candidates in the spectrum's order (mix_key images), so that their
    // sorted spectrum lookups ascend
    uint64_t out_cap = std::max<uint64_t>(1u << 20, 16 * n_hits);
    const auto walk = super ? mercy_walk_kernel<NW, true, kWalkLanes> : mercy_walk_kernel<NW, false, kWalkLanes>;
    Buf<uint64_t> cand;
    uint64_t n_cand = 0;
    for (int attempt = 0; attempt < 2; attempt++) {
        cand = Buf<uint64_t>(ctx, out_cap * NW);
        MH_CUDA(cudaMemsetAsync(stats.p + 1, 0, sizeof(uint64_t), ctx->stream));
        if (n_hits)
            MH_LAUNCH(ctx, "mercy_walk", grid_for(ctx, n_hits * kWalkLanes, 256, 8), 256, 0, walk, reads->packed,
                      hits.p, n_hits, k, table.p, cap - 1, solid->spectrum, solid->spectrum_len,
                      spec_off.p, spec_bits, sx, solid->d,
                      cand.p, out_cap, (unsigned long long*)(stats.p + 1));
        read_u64(ctx, stats.p + 1, &n_cand, 1);
        if (n_cand <= out_cap) break;
        out_cap = n_cand;
    }
    hits.reset();
    spec_off.reset();
    table.reset();
    Buf<uint64_t> alt(ctx, (n_cand ? n_cand : 1) * NW);
    const bool in_alt = radix_sort_spread<NW>(ctx, cand.p, alt.p, n_cand);
    Buf<uint64_t>& sorted = in_alt ? alt : cand;
    Buf<uint64_t> mk;
    Buf<uint32_t> mc;
    uint64_t M = 0, runs = 0, palins = 0;
    expand_runs<NW>(ctx, sorted.p, n_cand, k, 1, mk, mc, &M, &runs, &palins, solid->spectrum, solid->spectrum_len,
                    solid->n_spectrum, true, true, nullptr, super ? &sx : nullptr);
    sync_and_check(ctx);
    out->k = k;
    out->nw = NW;
    out->d = solid->d;
    out->n = M;
    out->n_kmers = n_cand;
    out->n_distinct = M;
    out->keys = mk.release();
    out->counts = mc.release();
}

template void mercy_kmers<1>(mh_ctx*, const mh_reads*, const mh_kmers*, mh_kmers*);
template void mercy_kmers<2>(mh_ctx*, const mh_reads*, const mh_kmers*, mh_kmers*);
template void mercy_kmers<4>(mh_ctx*, const mh_reads*, const mh_kmers*, mh_kmers*);

}  // namespace mh

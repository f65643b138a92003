// mh_build_sdbg: the BOSS arrays of E = solid + mercy (paper, Sec. 2, first
// and second paragraphs).
//
//   colex     ck(e) = (e[k-1], ..., e[0], e[k]) packed, so integer order of ck
//             is colex order of the k-prefix, then the label
//   order     no sort: eight sorted runs of the tables, one merge (mh_colex.cu)
//   degrees   zero outdegree: a join of the targets against the nodes, both in
//             colex order; zero indegree: their reverse complements
//   padding   dummy entries (node $ v[0..k-2], label v[k-1]) sorted by
//             (v[k-2..0], v[k-1]); $ entries in the order of their nodes
//   place     final position of every dummy and $ entry: its rank in its own
//             list plus the number of entries of the other lists below it
//   emit      one sweep over the final positions: W with minus flag, last,
//             dummy, valid, mult, from the keys and the padding's positions;
//             aux; F by bisection
#include "mh_internal.cuh"

namespace mh {

// ck -> group G = ck >> 4 (node symbols k-1..1), tail = pos0' * 5 + label',
// with pos0' = node symbol 0 + 1 and label' = label + 1 ($ = 0 for both).
template <int NW>
__device__ __forceinline__ bool ext_less(const Key<NW>& ga, uint32_t ta, const Key<NW>& gb, uint32_t tb) {
    if (!key_eq<NW>(ga, gb)) return key_less<NW>(ga, gb);
    return ta < tb;
}

template <int NW>
__device__ __forceinline__ void ext_of_ck(const Key<NW>& ck, Key<NW>& g, uint32_t& tail) {
    g = key_shr<NW>(ck, 4);
    uint32_t lo = (uint32_t)(ck.w[0] & 15u);
    tail = ((lo >> 2) + 1) * 5 + (lo & 3) + 1;
}

// dummy key dk = (v[k-2], ..., v[0], v[k-1]) (k symbols): G = dk >> 2, tail = label'
template <int NW>
__device__ __forceinline__ void ext_of_dummy(const Key<NW>& dk, Key<NW>& g, uint32_t& tail) {
    g = key_shr<NW>(dk, 2);
    tail = (uint32_t)(dk.w[0] & 3u) + 1;
}

// $ entry of reversed node u_rev = (u[k-1], ..., u[0]): G = u_rev >> 2, tail = (u[0]+1)*5
template <int NW>
__device__ __forceinline__ void ext_of_dollar(const Key<NW>& ur, Key<NW>& g, uint32_t& tail) {
    g = key_shr<NW>(ur, 2);
    tail = ((uint32_t)(ur.w[0] & 3u) + 1) * 5;
}

// Lower bound of (g, t) in a sorted list whose i-th element's ext key is given by ExtOf.
template <int NW, int KIND>
__device__ __forceinline__ uint64_t lb_ext(const uint64_t* __restrict__ a, uint64_t n, const Key<NW>& g, uint32_t t) {
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
        uint64_t mid = (lo + hi) >> 1;
        Key<NW> x = load_key<NW>(a, mid), gx;
        uint32_t tx;
        if (KIND == 0) ext_of_ck<NW>(x, gx, tx);
        else if (KIND == 1) ext_of_dummy<NW>(x, gx, tx);
        else ext_of_dollar<NW>(x, gx, tx);
        if (ext_less<NW>(gx, tx, g, t)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Zero-outdegree nodes.  In colex order the targets of the edges with label c
// are c followed by their groups (e[k-1], ..., e[1]), ascending; so a tile of
// whole groups of the order meets, for each label, one contiguous range of
// the order's nodes.  The tile's groups and the labels each holds stay in
// shared memory, the four ranges are streamed past them, and a node c.g
// clears label c of group g: what is left are targets that no edge leaves.
// Reads every key twice and writes next to nothing; bound by the searches in
// shared memory, a lane a key and eight CTAs an SM to hide them (four
// searches a lane 4.0 ms, two warps a label walking on from a search in eight
// 4.4 and more).  3.5e8 edges of one word: 3.3 ms, where writing the sorted
// nodes and targets, one radix pass and the merge of their differences took
// 12.6.
template <int NW>
struct ZeroTile {
    static constexpr int kItems = 8 / NW;             // entries a thread
    static constexpr int kCap = 256 * kItems;
    // a group holds at most 16 edges, each once a table: a solid and a mercy
    // table that share edges are built too
    static constexpr int kTile = kCap - 32;
};

// st[t] = the first group start at or after t * kTile (t = 0..n_tiles; E at
// the end); tb[4 t + c] = the first entry whose node is c.g or above, g the
// group at st[t] (the end of c's block for t = n_tiles or no such group).
template <int NW>
__global__ void zero_bounds_kernel(const uint64_t* __restrict__ ck, uint64_t E, int k, uint64_t n_tiles,
                                   uint64_t* __restrict__ st, uint64_t* __restrict__ tb) {
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < (n_tiles + 1) * 4;
         q += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = q >> 2;
        const uint32_t c = (uint32_t)(q & 3);
        uint64_t s = t < n_tiles ? t * ZeroTile<NW>::kTile : E;
        if (s > 0)
            while (s < E && key_eq<NW>(key_shr<NW>(load_key<NW>(ck, s), 4), key_shr<NW>(load_key<NW>(ck, s - 1), 4))) s++;
        if (c == 0) st[t] = s;
        Key<NW> x = key_zero<NW>();
        uint64_t b = E;
        if (!(s >= E && c == 3)) {
            x.w[0] = s >= E ? c + 1 : c;
            x = key_shl<NW>(x, 2 * k);
            if (t > 0 && s < E) {
                const Key<NW> g = key_shl<NW>(key_shr<NW>(load_key<NW>(ck, s), 4), 2);
#pragma unroll
                for (int w = 0; w < NW; w++) x.w[w] |= g.w[w];
            }
            uint64_t lo = 0;
            while (lo < b) {
                const uint64_t mid = (lo + b) >> 1;
                if (key_less<NW>(load_key<NW>(ck, mid), x)) lo = mid + 1; else b = mid;
            }
        }
        tb[q] = b;
    }
}

// Tile t's targets without out-edges, as reversed nodes: cnt[c * n_tiles + t]
// of them with label c, ascending, from found[at[t]] on, label after label.
template <int NW>
__global__ void __launch_bounds__(256, NW == 4 ? 4 : 8) zero_out_kernel(const uint64_t* __restrict__ ck, int k, uint64_t n_tiles,
                                                       const uint64_t* __restrict__ st,
                                                       const uint64_t* __restrict__ tb, uint64_t* __restrict__ found,
                                                       uint64_t* __restrict__ at, uint32_t* __restrict__ cnt,
                                                       unsigned long long* __restrict__ n_found) {
    using Z = ZeroTile<NW>;
    constexpr int I = Z::kItems;
    __shared__ __align__(16) uint64_t gk[bisect_at<NW>(Z::kCap) * NW];  // the groups
    __shared__ __align__(16) uint32_t gm[Z::kCap];       // a byte a label: 1 where it is left
    __shared__ uint32_t scratch[8];
    __shared__ uint64_t wsum[8], base;
    uint8_t* left = reinterpret_cast<uint8_t*>(gm);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t t = blockIdx.x, s0 = st[t];
    const uint32_t n = (uint32_t)min(st[t + 1] - s0, (uint64_t)Z::kCap);  // at most kTile + 31
    // groups, numbered in order: a warp 32 I entries, 32 at a time
    uint32_t ng = 0;
    {
        Key<NW> x[I];
        uint32_t heads[I], mine = 0;
        const uint32_t w0 = warp * 32 * I + lane;
#pragma unroll
        for (int j = 0; j < I; j++) {
            gm[tid + j * 256] = 0;
            x[j] = key_zero<NW>();
            if (w0 + j * 32 < n) x[j] = load_key<NW>(ck, s0 + w0 + j * 32);
        }
        Key<NW> before = key_zero<NW>();
        if (lane == 0 && w0 && w0 < n) before = load_key<NW>(ck, s0 + w0 - 1);
#pragma unroll
        for (int j = 0; j < I; j++) {
            Key<NW> y;
#pragma unroll
            for (int w = 0; w < NW; w++) {
                y.w[w] = __shfl_up_sync(0xFFFFFFFFu, x[j].w[w], 1);
                const uint64_t last = j ? __shfl_sync(0xFFFFFFFFu, x[j > 0 ? j - 1 : 0].w[w], 31) : before.w[w];
                if (lane == 0) y.w[w] = last;
            }
            const uint32_t i = w0 + j * 32;
            heads[j] = __ballot_sync(0xFFFFFFFFu,
                                     i < n && (i == 0 || !key_eq<NW>(key_shr<NW>(x[j], 4), key_shr<NW>(y, 4))));
            mine += __popc(heads[j]);
        }
        if (lane == 0) scratch[warp] = mine;
        __syncthreads();
        uint32_t g = 0;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            g += q < warp ? scratch[q] : 0u;
            ng += scratch[q];
        }
#pragma unroll
        for (int j = 0; j < I; j++) {
            if (w0 + j * 32 < n) {
                const uint32_t mg = g + __popc(heads[j] & (0xFFFFFFFFu >> (31 - lane))) - 1;
                if ((heads[j] >> lane) & 1u) store_key<NW>(gk, bisect_at<NW>(mg), key_shr<NW>(x[j], 4));
                left[4 * mg + (uint32_t)(x[j].w[0] & 3u)] = 1;
            }
            g += __popc(heads[j]);
        }
    }
    const uint32_t i0 = tid * I;
    __syncthreads();
    // the nodes with first symbol c, c = 0..3, numbered through
    {
        uint64_t from[4], end[4], total = 0;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const uint64_t b0 = tb[4 * t + c], b1 = tb[4 * (t + 1) + c];
            from[c] = b0 - total;
            total += b1 > b0 ? b1 - b0 : 0;
            end[c] = total;
        }
        for (uint64_t q = tid; q < total; q += 256) {
            const uint32_t c = q < end[0] ? 0u : q < end[1] ? 1u : q < end[2] ? 2u : 3u;
            const uint64_t f = c == 0 ? from[0] : c == 1 ? from[1] : c == 2 ? from[2] : from[3];
            const Key<NW> y = key_low<NW>(key_shr<NW>(load_key<NW>(ck, q + f), 2), 2 * (k - 1));
            const uint32_t p = bisect_shared<NW>(gk, ng, y);
            if (p < ng && key_eq<NW>(load_key<NW>(gk, bisect_at<NW>(p)), y)) left[4 * p + c] = 0;
        }
    }
    __syncthreads();
    // what is left, label by label (the four counts in one 64-bit scan)
    uint64_t mine = 0;
    uint32_t m[I];
#pragma unroll
    for (int j = 0; j < I; j++) {
        m[j] = i0 + j < ng ? gm[i0 + j] : 0u;
#pragma unroll
        for (int c = 0; c < 4; c++) mine += (uint64_t)((m[j] >> (8 * c)) & 1u) << (16 * c);
    }
    uint64_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint64_t pre = incl - mine, tot = 0;
    for (int q = 0; q < 8; q++) {
        pre += q < warp ? wsum[q] : 0ull;
        tot += wsum[q];
    }
    uint32_t tc[4], to[4], all = 0;
#pragma unroll
    for (int c = 0; c < 4; c++) {
        tc[c] = (uint32_t)(tot >> (16 * c)) & 0xFFFFu;
        to[c] = all;
        all += tc[c];
    }
    if (tid == 0) {
        base = all ? atomicAdd(n_found, (unsigned long long)all) : 0ull;
        at[t] = base;
#pragma unroll
        for (int c = 0; c < 4; c++) cnt[c * n_tiles + t] = tc[c];
    }
    if (!all) return;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; c++) {
        uint64_t o = base + to[c] + ((uint32_t)(pre >> (16 * c)) & 0xFFFFu);
#pragma unroll
        for (int j = 0; j < I; j++)
            if ((m[j] >> (8 * c)) & 1u) {
                Key<NW> v = key_zero<NW>();
                v.w[0] = (uint64_t)c;
                v = key_shl<NW>(v, 2 * (k - 1));
                const Key<NW> gg = load_key<NW>(gk, bisect_at<NW>(i0 + j));
#pragma unroll
                for (int w = 0; w < NW; w++) v.w[w] |= gg.w[w];
                store_key<NW>(found, o++, v);
            }
    }
}

// The tiles' finds in order: those of (label c, tile t) to off[c * n_tiles + t]
// (thread per tile: a few finds each).
template <int NW>
__global__ void zero_gather_kernel(const uint64_t* __restrict__ found, const uint64_t* __restrict__ at,
                                   const uint32_t* __restrict__ cnt, const uint64_t* __restrict__ off,
                                   uint64_t n_tiles, uint64_t* __restrict__ out) {
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < n_tiles;
         t += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t a = at[t];
        for (int c = 0; c < 4; c++) {
            const uint32_t m = cnt[c * n_tiles + t];
            const uint64_t o = off[c * n_tiles + t];
            for (uint32_t j = 0; j < m; j++) store_key<NW>(out, o + j, load_key<NW>(found, a + j));
            a += m;
        }
    }
}

// The zero-indegree nodes are the reverse complements v of the zero-outdegree
// nodes u (the edges are closed under reverse complement): reversed node u ->
// dummy key (v[k-2], ..., v[0], v[k-1]).
template <int NW>
__global__ void dummy_keys_kernel(const uint64_t* __restrict__ zout, uint64_t t, int k, uint64_t* __restrict__ dk) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < t; i += (uint64_t)gridDim.x * blockDim.x) {
        // v reversed = the complement of u
        Key<NW> v = key_rev<NW>(load_key<NW>(zout, i), k);
#pragma unroll
        for (int w = 0; w < NW; w++) v.w[w] = ~v.w[w];
        Key<NW> low = key_low<NW>(v, 2 * (k - 1));
        Key<NW> top = key_shr<NW>(v, 2 * (k - 1));
        store_key<NW>(dk, i, key_or_low<NW>(key_shl<NW>(low, 2), top.w[0] & 3u));
    }
}

// Final positions of dummy (KIND 1) or $ (KIND 2) entries.
template <int NW, int KIND>
__global__ void place_pad_kernel(const uint64_t* __restrict__ own, uint64_t n_own, const uint64_t* __restrict__ ck,
                                 uint64_t E, const uint64_t* __restrict__ other, uint64_t n_other,
                                 uint64_t* __restrict__ final_pos) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n_own;
         i += (uint64_t)gridDim.x * blockDim.x) {
        Key<NW> x = load_key<NW>(own, i), g;
        uint32_t t;
        if (KIND == 1) ext_of_dummy<NW>(x, g, t); else ext_of_dollar<NW>(x, g, t);
        uint64_t le = lb_ext<NW, 0>(ck, E, g, t);
        uint64_t lo = KIND == 1 ? lb_ext<NW, 2>(other, n_other, g, t) : lb_ext<NW, 1>(other, n_other, g, t);
        final_pos[i] = le + i + lo;
    }
}

// aux[i]: the node v of dummy i (dk = (v[k-2], ..., v[0], v[k-1])).
template <int NW>
__global__ void aux_kernel(const uint64_t* __restrict__ dk, uint64_t t, int k, uint64_t* __restrict__ aux) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < t; i += (uint64_t)gridDim.x * blockDim.x) {
        const Key<NW> x = load_key<NW>(dk, i);
        // v = reverse of v_rev, v_rev = (v[k-1], v[k-2], ..., v[0]) = label * 4^(k-1) + dk >> 2
        Key<NW> top = key_zero<NW>();
        top.w[0] = x.w[0] & 3u;
        top = key_shl<NW>(top, 2 * (k - 1));
        Key<NW> vr = key_shr<NW>(x, 2);
#pragma unroll
        for (int w = 0; w < NW; w++) vr.w[w] |= top.w[w];
        store_key<NW>(aux, i, key_rev<NW>(vr, k));
    }
}

// hist[c - 1] = entries whose node's last symbol (the top one of every list's
// keys) is below c, for c = 1, 2, 3.
template <int NW>
__global__ void symbol_starts_kernel(const uint64_t* __restrict__ ck, uint64_t E, const uint64_t* __restrict__ dk,
                                     uint64_t t, const uint64_t* __restrict__ ur, uint64_t u, int k,
                                     unsigned long long* __restrict__ hist) {
    const int q = threadIdx.x;
    if (q >= 9) return;
    const uint64_t* a = q < 3 ? ck : q < 6 ? dk : ur;
    const uint64_t n = q < 3 ? E : q < 6 ? t : u;
    Key<NW> x = key_zero<NW>();
    x.w[0] = (uint64_t)(q % 3 + 1);
    x = key_shl<NW>(x, q < 3 ? 2 * k : 2 * (k - 1));
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (key_less<NW>(load_key<NW>(a, mid), x)) lo = mid + 1; else hi = mid;
    }
    if (lo) atomicAdd(&hist[q % 3], (unsigned long long)lo);
}

// Emission: a CTA per kEmitTile final positions.  The tile's dummies and $
// entries (few) are set down in shared memory first; the slots between them
// are the edges from a known one on, in order, so a lane finds its edge by a
// count of bits, its minus flag (an earlier entry of its group e[1..k-1] has
// the same label; a group holds at most 16) and whether it ends its node from
// the neighbours, and a warp's ballots are words of the bit-vectors.
// Reads each key once from memory (the neighbours come from L1) and writes
// each output once; bound by the loads in flight (one word: two keys a thread
// at eight CTAs an SM; four at five 1.8 ms for 3.5e8 edges, eight at two 2.7;
// two words: two at five, 0.34 ms for 4.1e7, at eight 0.37).  3.5e8 edges of
// one word: 1.6 ms, where flags, insertion counts, their scan, bytes and their
// packing (53 bytes an edge) took 6.5; build of 3 M reads at k = 47 with
// multiplicities: 0.34 ms.
constexpr int kEmitTile = 2048;

// pb[2 b] / pb[2 b + 1]: dummies / $ entries placed before position b * kEmitTile.
__global__ void emit_bounds_kernel(const uint64_t* __restrict__ pos_d, uint64_t t, const uint64_t* __restrict__ pos_u,
                                   uint64_t u, uint64_t n_tiles, uint64_t* __restrict__ pb) {
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < 2 * (n_tiles + 1);
         q += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t* a = (q & 1) ? pos_u : pos_d;
        const uint64_t p = (q >> 1) * kEmitTile;
        uint64_t lo = 0, hi = (q & 1) ? u : t;
        while (lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (a[mid] < p) lo = mid + 1; else hi = mid;
        }
        pb[q] = lo;
    }
}

template <int NW>
__global__ void __launch_bounds__(256, NW == 1 ? 8 : NW == 2 ? 5 : 3) emit_kernel(const uint64_t* __restrict__ ck, const uint32_t* __restrict__ cv,
                                                   uint64_t E, const uint64_t* __restrict__ dk, uint64_t t,
                                                   const uint64_t* __restrict__ pos_d,
                                                   const uint64_t* __restrict__ pos_u, uint64_t m,
                                                   const uint64_t* __restrict__ pb, uint8_t* __restrict__ W,
                                                   uint32_t* __restrict__ last, uint32_t* __restrict__ dummy,
                                                   uint32_t* __restrict__ valid, uint32_t* __restrict__ mult,
                                                   unsigned long long* __restrict__ n_last) {
    constexpr int kWords = kEmitTile / 32;  // 32 positions each, eight a warp
    constexpr int U = 2;
    __shared__ uint8_t pad[kEmitTile];      // where pmask is set: W code, bit 4 last, bit 5 dummy
    __shared__ uint32_t pmask[kWords], pre[kWords], sum_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t b = blockIdx.x, base = b * kEmitTile;
    const uint32_t n = (uint32_t)(m - base < (uint64_t)kEmitTile ? m - base : (uint64_t)kEmitTile);
    const uint64_t d0 = pb[2 * b], u0 = pb[2 * b + 1], d1 = pb[2 * b + 2], u1 = pb[2 * b + 3];
    const uint64_t e0 = base - d0 - u0;     // the tile's first edge
    if (tid < kWords) pmask[tid] = 0;
    if (tid == 0) sum_last = 0;
    __syncthreads();
    for (uint64_t i = d0 + tid; i < d1; i += 256) {
        const Key<NW> x = load_key<NW>(dk, i);
        const bool ends =
            i + 1 == t || !key_eq<NW>(key_shr<NW>(load_key<NW>(dk, i + 1), 2), key_shr<NW>(x, 2));
        const uint64_t p = pos_d[i] - base;
        if (p >= n) continue;  // (never so in sorted tables)
        pad[p] = (uint8_t)(((uint32_t)(x.w[0] & 3u) + 1) | (ends ? 16 : 0) | 32);
        atomicOr(&pmask[p >> 5], 1u << (p & 31));
    }
    for (uint64_t i = u0 + tid; i < u1; i += 256) {
        const uint64_t p = pos_u[i] - base;
        if (p >= n) continue;
        pad[p] = 16;
        atomicOr(&pmask[p >> 5], 1u << (p & 31));
    }
    __syncthreads();
    if (warp == 0) {
        static_assert(kWords == 64, "two words a lane");
        const uint32_t c0 = __popc(pmask[2 * lane]), c = c0 + __popc(pmask[2 * lane + 1]);
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        pre[2 * lane] = x - c;
        pre[2 * lane + 1] = x - c + c0;
    }
    __syncthreads();
    uint32_t ends = 0;
    for (int r = 0; r < 8; r += U) {
        Key<NW> x[U], lf[U], rt[U];
        uint64_t at[U];
        uint32_t kind[U];  // 0 past the end, 1 padding, 2 edge
#pragma unroll
        for (int j = 0; j < U; j++) {
            const uint32_t wd = (r + j) * 8 + warp, p = wd * 32 + lane, pm = pmask[wd];
            kind[j] = p >= n ? 0u : ((pm >> lane) & 1u) ? 1u : 2u;
            at[j] = e0 + p - pre[wd] - __popc(pm & ((1u << lane) - 1u));
            if (kind[j] == 2 && at[j] >= E) kind[j] = 0;  // (never so in sorted tables)
            if (kind[j] == 2) {
                x[j] = load_key<NW>(ck, at[j]);
                if (at[j] > 0) lf[j] = load_key<NW>(ck, at[j] - 1);
                if (at[j] + 1 < E) rt[j] = load_key<NW>(ck, at[j] + 1);
            }
        }
#pragma unroll
        for (int j = 0; j < U; j++) {
            const uint32_t wd = (r + j) * 8 + warp, p = wd * 32 + lane;
            uint32_t code = 0;
            if (kind[j] == 1) code = pad[p];
            if (kind[j] == 2) {
                const Key<NW> g = key_shr<NW>(x[j], 4);
                const uint32_t lab = (uint32_t)(x[j].w[0] & 3u);
                bool minus = false;
                Key<NW> y = lf[j];
                for (uint64_t i = at[j]; i > 0; y = load_key<NW>(ck, i - 1)) {
                    if (!key_eq<NW>(key_shr<NW>(y, 4), g)) break;
                    if ((uint32_t)(y.w[0] & 3u) == lab) {
                        minus = true;
                        break;
                    }
                    if (--i == 0) break;
                }
                const bool ends_node =
                    at[j] + 1 == E || !key_eq<NW>(key_shr<NW>(rt[j], 2), key_shr<NW>(x[j], 2));
                code = lab + 1 + (minus ? 4 : 0) + (ends_node ? 16 : 0);
            }
            const uint32_t lb = __ballot_sync(0xFFFFFFFFu, (code & 16) != 0);
            const uint32_t db = __ballot_sync(0xFFFFFFFFu, (code & 32) != 0);
            const uint32_t vb = __ballot_sync(0xFFFFFFFFu, kind[j] != 0);
            if (kind[j]) W[base + p] = (uint8_t)(code & 15);
            if (mult && kind[j]) mult[base + p] = kind[j] == 2 ? cv[at[j]] : 0u;
            if (lane == 0 && vb) {
                const uint64_t o = base / 32 + wd;
                last[o] = lb;
                dummy[o] = db;
                valid[o] = vb;
            }
            ends += __popc(lb);
        }
    }
    if (lane == 0 && ends) atomicAdd(&sum_last, ends);
    __syncthreads();
    if (tid == 0 && sum_last) atomicAdd(n_last, (unsigned long long)sum_last);
}

template <int NW>
void build_sdbg(mh_ctx* ctx, const mh_kmers* solid, const mh_kmers* mercy, mh_sdbg* out) {
    const int k = solid->k, K1 = k + 1;
    const uint64_t nS = solid->n, nM = mercy ? mercy->n : 0, E = nS + nM;
    const bool want_mult = ctx->with_mult != 0;
    out->k = k;
    out->nw = NW;
    // the edges in colex order
    Buf<uint64_t> ck(ctx, (E ? E : 1) * NW);
    Buf<uint32_t> cv;
    if (want_mult) cv = Buf<uint32_t>(ctx, E ? E : 1);
    if (E) colex_merge<NW>(ctx, solid, mercy, k, ck.p, want_mult ? cv.p : nullptr);
    // zero outdegree, ascending (as many nodes have zero indegree)
    Buf<uint64_t> zout;
    uint64_t u = 0;
    if (E) {
        const uint64_t tiles = ceil_div(E, (uint64_t)ZeroTile<NW>::kTile);
        Buf<uint64_t> st(ctx, tiles + 1), tb(ctx, 4 * (tiles + 1)), found(ctx, E * NW), at(ctx, tiles + 1),
            off(ctx, 4 * tiles + 1);
        Buf<uint32_t> cnt(ctx, 4 * tiles);
        Buf<unsigned long long> n_found(ctx, 1);
        n_found.zero();
        MH_LAUNCH(ctx, "zero_bounds", grid_for(ctx, 4 * (tiles + 1), 256), 256, 0, zero_bounds_kernel<NW>, ck.p, E, k,
                  tiles, st.p, tb.p);
        MH_LAUNCH_B(ctx, "zero_out", 2 * E * 8 * NW, (unsigned)tiles, 256, 0, zero_out_kernel<NW>, ck.p, k, tiles, st.p,
                    tb.p, found.p, at.p, cnt.p, n_found.p);
        exclusive_scan_u32(ctx, cnt.p, off.p, 4 * tiles);
        read_u64(ctx, off.p + 4 * tiles, &u, 1);
        zout = Buf<uint64_t>(ctx, (u ? u : 1) * NW);
        if (u)
            MH_LAUNCH(ctx, "zero_gather", grid_for(ctx, tiles, 256), 256, 0, zero_gather_kernel<NW>, found.p, at.p,
                      cnt.p, off.p, tiles, zout.p);
    } else {
        zout = Buf<uint64_t>(ctx, NW);
    }
    const uint64_t t = u;
    // dummy entries in colex order
    Buf<uint64_t> dk(ctx, (t ? t : 1) * NW), dk2(ctx, (t ? t : 1) * NW);
    if (t) MH_LAUNCH(ctx, "dummy_keys", grid_for(ctx, t, 256), 256, 0, dummy_keys_kernel<NW>, zout.p, t, k, dk.p);
    // (many wide keys: by their top bits and a fix-up, not 2 k bits of passes)
    if (NW > 1 && t >= (1u << 14)) {
        Buf<uint32_t> v(ctx, t), v2(ctx, t);
        v.zero();
        if (radix_sort_spread_kv<NW>(ctx, dk.p, dk2.p, v.p, v2.p, t, 64 * NW - 2 * k)) std::swap(dk, dk2);
    } else if (radix_sort<NW>(ctx, dk.p, dk2.p, nullptr, nullptr, t, 0, 2 * k)) {
        std::swap(dk, dk2);
    }
    dk2.reset();
    // merge positions of the padding
    const uint64_t m = E + t + u;
    Buf<uint64_t> pos_d(ctx, t ? t : 1), pos_u(ctx, u ? u : 1);
    if (t)
        MH_LAUNCH(ctx, "place_dummy", grid_for(ctx, t, 256), 256, 0, (place_pad_kernel<NW, 1>), dk.p, t, ck.p, E,
                  zout.p, u, pos_d.p);
    if (u)
        MH_LAUNCH(ctx, "place_dollar", grid_for(ctx, u, 256), 256, 0, (place_pad_kernel<NW, 2>), zout.p, u, ck.p, E,
                  dk.p, t, pos_u.p);
    // emit
    Buf<unsigned long long> hist(ctx, 8);
    hist.zero();
    Buf<uint32_t> mult;
    if (want_mult) mult = Buf<uint32_t>(ctx, m ? m : 1);
    const uint64_t nwk = (uint64_t)NW;
    Buf<uint64_t> aux(ctx, (t ? t : 1) * nwk);
    if (t) MH_LAUNCH(ctx, "aux", grid_for(ctx, t, 256), 256, 0, aux_kernel<NW>, dk.p, t, k, aux.p);
    const uint64_t n_words = ceil_div(m, 32);
    Buf<uint8_t> W(ctx, m ? m : 1);
    Buf<uint32_t> last(ctx, n_words ? n_words : 1), dummy(ctx, n_words ? n_words : 1), valid(ctx, n_words ? n_words : 1);
    if (m) {
        const uint64_t tiles = ceil_div(m, (uint64_t)kEmitTile);
        Buf<uint64_t> pb(ctx, 2 * (tiles + 1));
        MH_LAUNCH(ctx, "symbol_starts", 1, 32, 0, symbol_starts_kernel<NW>, ck.p, E, dk.p, t, zout.p, u, k, hist.p);
        MH_LAUNCH(ctx, "emit_bounds", grid_for(ctx, 2 * (tiles + 1), 256), 256, 0, emit_bounds_kernel, pos_d.p, t,
                  pos_u.p, u, tiles, pb.p);
        MH_LAUNCH_B(ctx, "emit", E * (8 * NW + (want_mult ? 4 : 0)) + m * (want_mult ? 5 : 1), (unsigned)tiles, 256, 0,
                    emit_kernel<NW>, ck.p, want_mult ? cv.p : nullptr, E, dk.p, t, pos_d.p, pos_u.p, m, pb.p, W.p,
                    last.p, dummy.p, valid.p, want_mult ? mult.p : nullptr, hist.p + 4);
    }
    uint64_t h[5];
    read_u64(ctx, reinterpret_cast<const uint64_t*>(hist.p), h, 5);
    out->m = m;
    out->t = t;
    out->u = u;
    out->n_nodes = h[4];
    out->F[0] = 0;
    out->F[1] = 0;
    out->F[2] = h[0];
    out->F[3] = h[1];
    out->F[4] = h[2];
    out->F[5] = m;
    out->W = W.release();
    out->last = last.release();
    out->dummy = dummy.release();
    out->valid = valid.release();
    out->aux = aux.release();
    out->mult = want_mult ? mult.release() : nullptr;
}

template void build_sdbg<1>(mh_ctx*, const mh_kmers*, const mh_kmers*, mh_sdbg*);
template void build_sdbg<2>(mh_ctx*, const mh_kmers*, const mh_kmers*, mh_sdbg*);
template void build_sdbg<4>(mh_ctx*, const mh_kmers*, const mh_kmers*, mh_sdbg*);

}  // namespace mh

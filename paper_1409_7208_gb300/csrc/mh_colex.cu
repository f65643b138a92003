// The edges in colex order, by one merge.
//
// For f = rc(e), ck(e) = (e[k-1], ..., e[0], e[k]) is ~f rotated by one symbol
// ((f[1..k] complemented, then comp f[0])), so each block of equal first
// symbol of a lex-sorted table closed under reverse complement, read
// backwards, is a sorted run of colex keys: eight runs, four of the solid and
// four of the mercy table.
//
//   runs     where they start (one small kernel: the host does not wait for it)
//   samples  every kQ-th key of each run
//   split    each sample's rank among all of them, by bisection in the other
//            runs' samples; those of a rank divisible by kP are splitters
//   bounds   where each splitter falls in each run
//   merge    a CTA per interval between splitters: at most
//            (kP + 1) kQ + 8 (kQ - 1) keys, made from the tables on the way
//            in, merged in shared memory by three levels of two-way merges
//            (a thread finds its diagonal, then merges kItems keys), written
//            out once
//
// Reads and writes every key once; bound by the shared-memory reads and the
// waits of the serial merges (seven CTAs an SM; six 0.3 ms more, four keys a
// thread 1.8 more).  3.5e8 edges of one word: 5.0 ms with the splitters, where
// writing the colex keys and a tree of three two-way merges (64 bytes an edge)
// took 7.1; build of 3 M reads at k = 47 with multiplicities: 1.24 for 1.74.
#include "mh_internal.cuh"

namespace mh {

namespace {

template <int NW>
struct Colex {
    static constexpr int kThreads = 256;
    static constexpr int kItems = NW == 1 ? 8 : NW == 2 ? 4 : 2;
    static constexpr int kCap = kThreads * kItems;
    static constexpr int kQ = 64 / NW;
    static constexpr int kP = 21;
    // a level's pairs start at threads of their own: four of them at most
    // half empty
    static_assert((kP + 1) * kQ + 8 * (kQ - 1) + 4 * kItems <= kCap, "an interval fits a CTA");
};

// Where the runs start in the tables read backwards (solid, then mercy), and
// where their samples do.
struct ColexRuns {
    uint64_t off[9];
    uint64_t samp[9];
};

// The tables as one list of colex keys read backwards.
template <int NW>
struct ColexView {
    const uint64_t* s;
    const uint32_t* sc;
    const uint64_t* m;
    const uint32_t* mc;
    uint64_t ns, nm;
    int k;
    __device__ __forceinline__ Key<NW> key(uint64_t i) const {
        Key<NW> f = i < ns ? load_key<NW>(s, ns - 1 - i) : load_key<NW>(m, nm - 1 - (i - ns));
#pragma unroll
        for (int w = 0; w < NW; w++) f.w[w] = ~f.w[w];
        f = key_low<NW>(f, 2 * (k + 1));
        const uint32_t top = (uint32_t)(key_shr<NW>(f, 2 * k).w[0] & 3u);
        return key_or_low<NW>(key_low<NW>(key_shl<NW>(f, 2), 2 * (k + 1)), top);
    }
    __device__ __forceinline__ uint32_t count(uint64_t i) const { return i < ns ? sc[ns - 1 - i] : mc[nm - 1 - (i - ns)]; }
};

// Thread (t, c): the first entry of table t (0 solid, 1 mercy) with first
// symbol >= c; then the runs.
template <int NW>
__global__ void colex_runs_kernel(ColexView<NW> v, ColexRuns* __restrict__ runs) {
    __shared__ uint64_t b[8];
    const int t = threadIdx.x >> 2, c = threadIdx.x & 3;
    if (t < 2) {
        const uint64_t* a = t == 0 ? v.s : v.m;
        uint64_t lo = 0, hi = t == 0 ? v.ns : v.nm;
        Key<NW> q = key_zero<NW>();
        q.w[0] = (uint64_t)c;
        q = key_shl<NW>(q, 2 * v.k);
        while (c && lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (key_less<NW>(load_key<NW>(a, mid), q)) lo = mid + 1; else hi = mid;
        }
        b[threadIdx.x] = lo;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t at = 0;
        for (int r = 0; r <= 8; r++) {
            // run r of a table is its block of first symbol 3 - r % 4
            const uint64_t o = r == 8 ? v.ns + v.nm : r < 4 ? (r ? v.ns - b[4 - r] : 0) : v.ns + (r > 4 ? v.nm - b[12 - r] : 0);
            runs->off[r] = o;
            if (r) at += ceil_div(o - runs->off[r - 1], (uint64_t)Colex<NW>::kQ);
            runs->samp[r] = at;
        }
    }
}

__device__ __forceinline__ int run_of(const uint64_t* off, uint64_t i) {
    int r = 0;
#pragma unroll
    for (int q = 1; q < 8; q++) r += i >= off[q];
    return r;
}

template <int NW>
__global__ void colex_samples_kernel(ColexView<NW> v, const ColexRuns* __restrict__ runs, uint64_t* __restrict__ samples) {
    __shared__ ColexRuns R;
    if (threadIdx.x < 18) (threadIdx.x < 9 ? R.off[threadIdx.x] : R.samp[threadIdx.x - 9]) =
        threadIdx.x < 9 ? runs->off[threadIdx.x] : runs->samp[threadIdx.x - 9];
    __syncthreads();
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < R.samp[8]; j += (uint64_t)gridDim.x * blockDim.x) {
        const int r = run_of(R.samp, j);
        store_key<NW>(samples, j, v.key(R.off[r] + (j - R.samp[r]) * Colex<NW>::kQ));
    }
}

// Rank of each sample: those of equal keys go by run.
template <int NW>
__global__ void colex_split_kernel(const ColexRuns* __restrict__ runs, const uint64_t* __restrict__ samples,
                                   uint64_t* __restrict__ splitters) {
    __shared__ uint64_t samp[9];
    if (threadIdx.x < 9) samp[threadIdx.x] = runs->samp[threadIdx.x];
    __syncthreads();
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < samp[8]; j += (uint64_t)gridDim.x * blockDim.x) {
        const int r = run_of(samp, j);
        const Key<NW> x = load_key<NW>(samples, j);
        uint64_t rank = j - samp[r];
        for (int q = 0; q < 8; q++) {
            if (q == r) continue;
            uint64_t lo = samp[q], hi = samp[q + 1];
            while (lo < hi) {
                const uint64_t mid = (lo + hi) >> 1;
                const Key<NW> y = load_key<NW>(samples, mid);
                const bool below = q < r ? !key_less<NW>(x, y) : key_less<NW>(y, x);
                if (below) lo = mid + 1; else hi = mid;
            }
            rank += lo - samp[q];
        }
        if (rank % Colex<NW>::kP == 0) store_key<NW>(splitters, rank / Colex<NW>::kP, x);
    }
}

// bnd[8 t + r]: the first key of run r not below splitter t (the run's ends
// for the first and past the last).
template <int NW>
__global__ void colex_bounds_kernel(ColexView<NW> v, const ColexRuns* __restrict__ runs,
                                    const uint64_t* __restrict__ splitters, uint64_t* __restrict__ bnd) {
    const uint64_t tiles = ceil_div(runs->samp[8], (uint64_t)Colex<NW>::kP);
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < 8 * (tiles + 1);
         q += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = q >> 3;
        const int r = (int)(q & 7);
        uint64_t lo = runs->off[r], hi = runs->off[r + 1];
        if (t == tiles) lo = hi;
        if (t > 0 && t < tiles) {
            const Key<NW> x = load_key<NW>(splitters, t);
            while (lo < hi) {
                const uint64_t mid = (lo + hi) >> 1;
                if (key_less<NW>(v.key(mid), x)) lo = mid + 1; else hi = mid;
            }
        }
        bnd[q] = lo;
    }
}

template <int NW, bool HV>
__global__ void __launch_bounds__(256, NW == 4 ? 4 : 7) colex_merge_kernel(ColexView<NW> v, const ColexRuns* __restrict__ runs,
                                                          const uint64_t* __restrict__ bnd, uint64_t* __restrict__ ck,
                                                          uint32_t* __restrict__ cv, uint32_t* __restrict__ err) {
    using C = Colex<NW>;
    constexpr int I = C::kItems;
    // a word of padding after 8: the threads' heads lie a few keys apart
    constexpr int kPadded = C::kCap / 8 * 9;
    __shared__ __align__(16) uint64_t sk[kPadded * NW];
    __shared__ uint32_t sv[HV ? kPadded : 1];
    __shared__ uint64_t from[8], base;
    __shared__ uint32_t end[9];
    auto pad = [](uint32_t i) { return i + (i >> 3); };
    const int tid = threadIdx.x;
    const uint64_t tiles = ceil_div(runs->samp[8], (uint64_t)C::kP);
    if (blockIdx.x >= tiles) return;
    if (tid < 32) {
        const int r = tid & 7;
        const uint64_t b0 = bnd[8 * blockIdx.x + r], b1 = bnd[8 * blockIdx.x + 8 + r];
        // (slices longer than a tile are no merge of sorted tables: cut, and reported)
        uint32_t n = (uint32_t)min(b1 - b0, (uint64_t)C::kCap), incl = n;
        uint64_t before = b0 - runs->off[r];
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o, 8);
            if (r >= o) incl += y;
            before += __shfl_xor_sync(0xFFFFFFFFu, before, o, 8);
        }
        if (tid < 8) {
            from[r] = b0 - (incl - n);
            end[r + 1] = incl;
        }
        if (tid == 0) {
            end[0] = 0;
            base = before;
        }
    }
    __syncthreads();
    const uint32_t n = end[8];
    if (n + 4 * I > (uint32_t)C::kCap) {
        if (tid == 0) atomicOr(err, ST_BAD_TABLE);
        return;
    }
    // the slices side by side, all of a thread's loads in flight
    {
        Key<NW> x[I];
        uint32_t c[HV ? I : 1];
#pragma unroll
        for (int q = 0; q < I; q++) {
            const uint32_t i = tid + q * 256;
            if (i < n) {
                int r = 0;
#pragma unroll
                for (int j = 1; j < 8; j++) r += i >= end[j];
                x[q] = v.key(from[r] + i);
                if constexpr (HV) c[q] = v.count(from[r] + i);
            }
        }
#pragma unroll
        for (int q = 0; q < I; q++) {
            const uint32_t i = tid + q * 256;
            if (i < n) {
                store_key<NW>(sk, pad(i), x[q]);
                if constexpr (HV) sv[pad(i)] = c[q];
            }
        }
    }
    __syncthreads();
    for (int level = 1; level <= 4; level <<= 1) {
        // pair p merges runs [2 p level, (2 p + 1) level) and the level after them
        uint32_t t0 = 0, d = ~0u, a0 = 0, b0 = 0, b1 = 0;
        for (int p = 0; p < 4 / level; p++) {
            const uint32_t x0 = end[2 * p * level], x1 = end[(2 * p + 1) * level], x2 = end[(2 * p + 2) * level];
            const uint32_t threads = (x2 - x0 + I - 1) / I;
            if ((uint32_t)tid - t0 < threads) {
                d = (tid - t0) * I;
                a0 = x0;
                b0 = x1;
                b1 = x2;
            }
            t0 += threads;
        }
        Key<NW> ok[I];
        uint32_t ov[HV ? I : 1];
        const uint32_t na = b0 - a0, nb = b1 - b0;
        const uint32_t mine = d == ~0u ? 0u : min((uint32_t)I, na + nb - d);
        if (mine) {
            uint32_t lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (!key_less<NW>(load_key<NW>(sk, pad(b0 + d - 1 - mid)), load_key<NW>(sk, pad(a0 + mid)))) lo = mid + 1;
                else hi = mid;
            }
            uint32_t ia = a0 + lo, ib = b0 + d - lo;
            Key<NW> ka = key_zero<NW>(), kb = key_zero<NW>();
            if (ia < b0) ka = load_key<NW>(sk, pad(ia));
            if (ib < b1) kb = load_key<NW>(sk, pad(ib));
#pragma unroll
            for (int q = 0; q < I; q++) {
                if (q < (int)mine) {
                    const bool take_a = ib >= b1 || (ia < b0 && !key_less<NW>(kb, ka));
                    ok[q] = take_a ? ka : kb;
                    if constexpr (HV) ov[q] = sv[pad(take_a ? ia : ib)];
                    if (take_a) {
                        if (++ia < b0) ka = load_key<NW>(sk, pad(ia));
                    } else {
                        if (++ib < b1) kb = load_key<NW>(sk, pad(ib));
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < I; q++)
            if (q < (int)mine) {
                store_key<NW>(sk, pad(a0 + d + q), ok[q]);
                if constexpr (HV) sv[pad(a0 + d + q)] = ov[q];
            }
        __syncthreads();
    }
    for (uint32_t i = tid; i < n; i += 256) {
        store_key<NW>(ck, base + i, load_key<NW>(sk, pad(i)));
        if constexpr (HV) cv[base + i] = sv[pad(i)];
    }
}

}  // namespace

template <int NW>
void colex_merge(mh_ctx* ctx, const mh_kmers* solid, const mh_kmers* mercy, int k, uint64_t* ck, uint32_t* cv) {
    using C = Colex<NW>;
    const uint64_t ns = solid->n, nm = mercy ? mercy->n : 0, E = ns + nm;
    const ColexView<NW> v{solid->keys, solid->counts, mercy ? mercy->keys : nullptr, mercy ? mercy->counts : nullptr, ns, nm, k};
    const uint64_t samples = E / C::kQ + 8, tiles = ceil_div(samples, (uint64_t)C::kP);  // at most
    Buf<ColexRuns> runs(ctx, 1);
    Buf<uint64_t> samp(ctx, samples * NW), split(ctx, tiles * NW), bnd(ctx, 8 * (tiles + 1));
    MH_LAUNCH(ctx, "colex_runs", 1, 32, 0, colex_runs_kernel<NW>, v, runs.p);
    MH_LAUNCH(ctx, "colex_samples", grid_for(ctx, samples, 256), 256, 0, colex_samples_kernel<NW>, v, runs.p, samp.p);
    MH_LAUNCH(ctx, "colex_split", grid_for(ctx, samples, 256), 256, 0, colex_split_kernel<NW>, runs.p, samp.p, split.p);
    MH_LAUNCH(ctx, "colex_bounds", grid_for(ctx, 8 * (tiles + 1), 256), 256, 0, colex_bounds_kernel<NW>, v, runs.p,
              split.p, bnd.p);
    if (cv)
        MH_LAUNCH_B(ctx, "colex_merge", E * (16 * NW + 8), (unsigned)tiles, 256, 0, (colex_merge_kernel<NW, true>), v,
                    runs.p, bnd.p, ck, cv, ctx->d_status);
    else
        MH_LAUNCH_B(ctx, "colex_merge", E * 16 * NW, (unsigned)tiles, 256, 0, (colex_merge_kernel<NW, false>), v, runs.p,
                    bnd.p, ck, nullptr, ctx->d_status);
}

template void colex_merge<1>(mh_ctx*, const mh_kmers*, const mh_kmers*, int, uint64_t*, uint32_t*);
template void colex_merge<2>(mh_ctx*, const mh_kmers*, const mh_kmers*, int, uint64_t*, uint32_t*);
template void colex_merge<4>(mh_ctx*, const mh_kmers*, const mh_kmers*, int, uint64_t*, uint32_t*);

}  // namespace mh

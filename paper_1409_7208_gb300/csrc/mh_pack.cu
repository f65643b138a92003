// mh_pack_reads: ASCII reads -> 2-bit packed fragments.
//
// One thread per 16 input bytes: a 16-byte vector load, per-byte code and
// validity with SIMD byte compares, one 32-bit output word (base j at bits
// 31-2(j%16)).  When every byte is a base and no read is empty, fragments are
// the reads and the packed words are the output.  Otherwise the valid bases
// are compacted (scan of per-chunk valid counts) and fragment starts are
// found from the validity masks and the read starts.
#include <cstdlib>

#include "mh_internal.cuh"

namespace mh {

// byte codes: A/a 0, C/c 1, G/g 2, T/t 3 (((c >> 1) ^ (c >> 2)) & 3 on those letters)
__device__ __forceinline__ uint32_t codes4(uint32_t x) { return ((x >> 1) ^ (x >> 2)) & 0x03030303u; }

// The letters (upper case) of four codes: the codes as nibbles select bytes.
__device__ __forceinline__ uint32_t letters4(uint32_t c) {
    return __byte_perm(0x54474341u, 0, __byte_perm(c | c >> 4, 0, 0x4420));
}

// Zero in each byte lane holding one of ACGTacgt: a byte is a base if it is
// the letter of the code that it would have.
__device__ __forceinline__ uint32_t invalid4(uint32_t x) { return letters4(codes4(x)) ^ (x & 0xDFDFDFDFu); }

// valid lanes (0xFF bytes) -> 4-bit mask, bit j = byte j
__device__ __forceinline__ uint32_t mask4(uint32_t v) {
    return (v & 1u) | ((v >> 7) & 2u) | ((v >> 14) & 4u) | ((v >> 21) & 8u);
}

// 16 bytes -> the packed word of their codes (first base most significant;
// four codes go to the top byte of a product) and the mask of the valid ones.
// Some 50 instructions for bases alone, where byte compares took 150.
__device__ __forceinline__ void encode16(const uint32_t x[4], uint32_t* word, uint32_t* valid) {
    uint32_t p[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const uint32_t c = codes4(x[q]);
        p[q] = c * 0x40100401u;  // 2^30 + 2^20 + 2^10 + 1
        d[q] = letters4(c) ^ (x[q] & 0xDFDFDFDFu);
    }
    *word = __byte_perm(__byte_perm(p[3], p[2], 0x73), __byte_perm(p[1], p[0], 0x73), 0x5410);
    *valid = 0xFFFFu;
    if (d[0] | d[1] | d[2] | d[3]) {
        *valid = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) *valid |= mask4(__vcmpeq4(d[q], 0u)) << (4 * q);
    }
}

// Load the 16 bytes of chunk c as four words (zero past n_bases).
__device__ __forceinline__ void load16(const uint8_t* __restrict__ a, uint64_t n_bases, uint64_t c, bool vec,
                                       uint32_t x[4], uint32_t* present) {
    uint64_t b = c * 16;
    if (vec && b + 16 <= n_bases) {
        uint4 v = reinterpret_cast<const uint4*>(a)[c];
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        *present = 0xFFFFu;
        return;
    }
    uint32_t pm = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        uint32_t w = 0;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            uint64_t i = b + 4 * q + j;
            if (i < n_bases) {
                w |= (uint32_t)a[i] << (8 * j);
                pm |= 1u << (4 * q + j);
            }
        }
        x[q] = w;
    }
    *present = pm;
}

// Fast-path pack: code word per chunk; sets *any_invalid if a byte is not a base.
__global__ void pack_chunks_kernel(const uint8_t* __restrict__ ascii, uint64_t n_bases, bool vec,
                                   uint32_t* __restrict__ packed, uint32_t* __restrict__ any_invalid) {
    const uint64_t n_chunks = ceil_div(n_bases, 16), stride = (uint64_t)gridDim.x * blockDim.x;
    bool bad = false;
    auto pack = [&](uint64_t c, const uint32_t x[4], uint32_t present) {
        uint32_t word, vmask;
        encode16(x, &word, &vmask);
        packed[c] = word;
        bad |= (vmask & present) != present;
    };
    // four loads in flight a thread (3 Gbp 0.61 ms; with byte compares and one load
    // 1.71, four loads 1.59)
    constexpr int U = 4;
    uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    for (; c + (U - 1) * stride < n_chunks; c += U * stride) {
        uint32_t x[U][4], present[U];
#pragma unroll
        for (int u = 0; u < U; u++) load16(ascii, n_bases, c + u * stride, vec, x[u], &present[u]);
#pragma unroll
        for (int u = 0; u < U; u++) pack(c + u * stride, x[u], present[u]);
    }
    for (; c < n_chunks; c += stride) {
        uint32_t x[4], present;
        load16(ascii, n_bases, c, vec, x, &present);
        pack(c, x, present);
    }
    if (__any_sync(0xFFFFFFFFu, bad) && (threadIdx.x & 31) == 0) atomicOr(any_invalid, 1u);
}

// Validate offsets; flag empty reads: bit 0 of *any_empty if there is one, bit 1
// if kEmptyRun in a row are.
constexpr uint64_t kEmptyRun = 1024;
__global__ void check_offs_kernel(const uint64_t* __restrict__ offs, uint64_t n_reads, uint64_t n_bases,
                                  uint32_t* __restrict__ any_empty, uint32_t* __restrict__ err) {
    uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i == 0 && (offs[0] != 0 || offs[n_reads] != n_bases)) atomicOr(err, ST_BAD_INPUT);
    uint32_t found = 0;
    for (; i < n_reads; i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t a = offs[i], b = offs[i + 1];
        if (b < a || b > n_bases) atomicOr(err, ST_BAD_INPUT);
        if (a == b) found |= i + kEmptyRun <= n_reads && offs[i + kEmptyRun] == a ? 3u : 1u;
    }
    found = __reduce_or_sync(0xFFFFFFFFu, found);
    if (found && (threadIdx.x & 31) == 0) atomicOr(any_empty, found);
}

__global__ void iota_u32_kernel(uint32_t* __restrict__ a, uint64_t n) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        a[i] = (uint32_t)i;
}

// --------------------------------------------------------- slow path
// Invalid bytes or empty reads: tiles of 4,096 input bases, a chunk of 16 a
// thread, in two sweeps over the input.  The first counts a tile's valid bases
// and fragment starts, the second (after a scan of the tiles' counts) finds
// them again, writes the fragments and sets the valid codes side by side in
// shared memory.  A tile reads its reads' starts once, so a fragment's read
// comes from a rank among them.  Two sweeps of 16-byte loads and one small
// scan, bound by memory latency; 5 M trimmed reads with Ns (450 Mbp): 0.76 ms,
// where masks, counts and prefixes a chunk in memory and a bisection of all
// offsets a fragment took 2.0 ms.
constexpr uint32_t kPackTile = 4096;

// first[t] = the first read with offs[r] >= t * kPackTile (n_reads if none).
__global__ void tile_reads_kernel(const uint64_t* __restrict__ offs, uint64_t n_reads, uint64_t n_tiles,
                                  uint64_t* __restrict__ first) {
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < n_tiles;
         t += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t lo = 0, hi = n_reads;
        while (lo < hi) {
            const uint64_t mid = (lo + hi) >> 1;
            if (offs[mid] < t * kPackTile) lo = mid + 1; else hi = mid;
        }
        first[t] = lo;
    }
}

// Read r starts at the tile's base q: its bit in rs, or (read_of) its number at
// its rank among the tile's non-empty reads.
__device__ __forceinline__ void tile_read(uint64_t r, uint64_t q, uint32_t* rs, const uint32_t* before,
                                          uint32_t* read_of) {
    if (read_of)
        read_of[before[q >> 5] + __popc(rs[q >> 5] & ((1u << (q & 31)) - 1u))] = (uint32_t)r;
    else
        atomicOr(&rs[q >> 5], 1u << (q & 31));
}

// tile_read of every non-empty read in [r0, n_reads) that starts in the tile at
// `base`, by a CTA, 32 reads a warp at a time.  A run of empty reads is passed
// over by a search for its end.  (Not inlined, and in kernels of its own: its
// registers cost two CTAs an SM, 1.14 -> 1.22 ms for 5 M trimmed reads.)
__device__ __noinline__ void sparse_tile_reads(const uint64_t* __restrict__ offs, uint64_t n_reads, uint64_t r0,
                                               uint64_t base, uint32_t* rs, const uint32_t* before,
                                               uint32_t* read_of) {
    const int lane = threadIdx.x & 31;
    for (uint64_t w0 = r0 + (threadIdx.x & ~31u); w0 < n_reads;) {
        const uint64_t r = w0 + lane;
        const uint64_t o = r < n_reads ? offs[r] : base + (uint64_t)kPackTile;
        const bool in = o - base < kPackTile;
        const uint64_t e = in ? offs[r + 1] : o;
        if (e > o) tile_read(r, o - base, rs, before, read_of);
        if (__ballot_sync(0xFFFFFFFFu, in) != 0xFFFFFFFFu) break;
        uint64_t skip = 256;
        const uint64_t o0 = __shfl_sync(0xFFFFFFFFu, o, 0);
        if (__shfl_sync(0xFFFFFFFFu, e, 31) == o0) {
            // 32 empty reads: the first offset past o0 is in (lo, hi], its
            // read the one before; steps of 1, 2, 4, ... reads, then of 32nds
            uint64_t lo = w0 + 32, hi = n_reads + 1;
            uint64_t at = lo + (1ull << lane);
            uint32_t m = __ballot_sync(0xFFFFFFFFu, at >= hi || offs[at] > o0);
            if (m) {
                const int j = __ffs(m) - 1;
                hi = min(hi, lo + ((uint64_t)1 << j));
                if (j) lo += 1ull << (j - 1);
            } else {
                lo += 1ull << 31;
            }
            while (hi - lo > 1) {
                const uint64_t step = (hi - lo + 31) / 32;
                at = lo + (lane + 1) * step;
                m = __ballot_sync(0xFFFFFFFFu, at >= hi || offs[at] > o0);
                const int j = __ffs(m) - 1;  // (the last lane's is past the end)
                hi = min(hi, lo + (uint64_t)(j + 1) * step);
                lo += (uint64_t)j * step;
            }
            if (hi > n_reads) break;  // none but empty reads
            skip = max(skip, (hi - 1 - w0) / 256 * 256);
        }
        w0 += skip;
    }
}

// The same, a read a thread.  RUNS (some empty reads lie in a row): unless the
// tile's reads are so many that most are empty.  A million empty reads in one
// tile, with a million of 150 bases around them: 5.1 ms -> 0.43.
template <bool RUNS>
__device__ __forceinline__ void tile_reads(const uint64_t* __restrict__ offs, uint64_t n_reads, uint64_t r0,
                                           uint64_t base, uint32_t* rs, const uint32_t* before, uint32_t* read_of) {
    if constexpr (RUNS) {
        const uint64_t far = r0 + 2 * kPackTile;
        if (far < n_reads && offs[far] - base < kPackTile) {
            sparse_tile_reads(offs, n_reads, r0, base, rs, before, read_of);
            return;
        }
    }
    for (uint64_t r = r0 + threadIdx.x; r < n_reads; r += 256) {
        const uint64_t o = offs[r];
        if (o - base >= kPackTile) break;
        if (offs[r + 1] > o) tile_read(r, o - base, rs, before, read_of);
    }
}

// A thread's chunk of tile t: its packed codes, valid bases and fragment
// starts (a valid base at a read's start or after an invalid one).  Also the
// starts of the tile's non-empty reads as bits in rs (after the barriers).
template <bool RUNS>
__device__ __forceinline__ void tile_chunk(const uint8_t* __restrict__ ascii, uint64_t n_bases, bool vec,
                                           const uint64_t* __restrict__ offs, uint64_t n_reads, uint64_t r0, uint64_t t,
                                           uint32_t* rs, uint8_t* tops, uint32_t* codes, uint32_t* valid,
                                           uint32_t* starts) {
    const int tid = threadIdx.x;
    const uint64_t base = t * kPackTile;
    if (tid < (int)kPackTile / 32) rs[tid] = 0;
    uint32_t x[4], present;
    load16(ascii, n_bases, t * (kPackTile / 16) + tid, vec, x, &present);
    uint32_t word, m;
    encode16(x, &word, &m);
    m &= present;
    tops[tid + 1] = (uint8_t)(m >> 15);
    if (tid == 0) tops[0] = t && !(invalid4(ascii[base - 1]) & 0xFFu) ? 1 : 0;
    __syncthreads();
    tile_reads<RUNS>(offs, n_reads, r0, base, rs, nullptr, nullptr);
    __syncthreads();
    const uint32_t rb = (rs[tid >> 1] >> (16 * (tid & 1))) & 0xFFFFu;
    *codes = word;
    *valid = m;
    *starts = m & (rb | ~(m << 1 | tops[tid])) & 0xFFFFu;
}

template <bool RUNS>
__global__ void __launch_bounds__(256) tile_count_kernel(const uint8_t* __restrict__ ascii, uint64_t n_bases, bool vec,
                                                         const uint64_t* __restrict__ offs, uint64_t n_reads,
                                                         const uint64_t* __restrict__ first,
                                                         uint32_t* __restrict__ n_valid,
                                                         uint32_t* __restrict__ n_starts) {
    __shared__ uint32_t rs[kPackTile / 32], ws[8];
    __shared__ uint8_t tops[257];
    uint32_t codes, m, fs;
    tile_chunk<RUNS>(ascii, n_bases, vec, offs, n_reads, first[blockIdx.x], blockIdx.x, rs, tops, &codes, &m, &fs);
    // (both counts at most 4,096: one sum)
    const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(m) << 16 | __popc(fs));
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t all = 0;
        for (int w = 0; w < 8; w++) all += ws[w];
        n_valid[blockIdx.x] = all >> 16;
        n_starts[blockIdx.x] = all & 0xFFFFu;
    }
}

template <bool RUNS>
__global__ void __launch_bounds__(256) tile_pack_kernel(const uint8_t* __restrict__ ascii, uint64_t n_bases, bool vec,
                                                        const uint64_t* __restrict__ offs, uint64_t n_reads,
                                                        const uint64_t* __restrict__ first,
                                                        const uint64_t* __restrict__ dst,
                                                        const uint64_t* __restrict__ fidx,
                                                        uint64_t* __restrict__ frag_offs,
                                                        uint32_t* __restrict__ frag_read,
                                                        uint32_t* __restrict__ packed) {
    __shared__ uint32_t rs[kPackTile / 32], before[kPackTile / 32], scratch[8];
    __shared__ uint32_t read_of[kPackTile];  // the tile's non-empty reads, then its output words
    __shared__ uint8_t tops[257];
    const int tid = threadIdx.x;
    const uint64_t t = blockIdx.x, base = t * kPackTile, r0 = first[t];
    uint32_t codes, m, fs;
    tile_chunk<RUNS>(ascii, n_bases, vec, offs, n_reads, r0, t, rs, tops, &codes, &m, &fs);
    // reads that start before each word of rs (at most 128 words)
    uint32_t all;
    const uint32_t reads = block_excl_scan_256(tid < (int)kPackTile / 32 ? __popc(rs[tid]) : 0u, scratch, &all);
    if (tid < (int)kPackTile / 32) before[tid] = reads;
    uint32_t tot;
    const uint32_t ex = block_excl_scan_256((uint32_t)__popc(m) << 16 | __popc(fs), scratch, &tot);
    tile_reads<RUNS>(offs, n_reads, r0, base, rs, before, read_of);
    __syncthreads();
    const uint64_t d0 = dst[t];
    uint64_t f = fidx[t] + (ex & 0xFFFFu);
    const uint32_t at = ex >> 16;  // the chunk's first valid base among the tile's
    while (fs) {
        const int j = __ffs(fs) - 1;
        fs &= fs - 1;
        const uint32_t q = tid * 16 + j;
        const uint32_t rank = before[q >> 5] + __popc(rs[q >> 5] & (0xFFFFFFFFu >> (31 - (q & 31))));
        frag_offs[f] = d0 + at + __popc(m & ((1u << j) - 1u));
        frag_read[f] = rank ? read_of[rank - 1] : (uint32_t)(r0 - 1);
        f++;
    }
    __syncthreads();
    // the valid codes side by side, placed as in the output's words
    uint32_t* out = read_of;
    for (int i = tid; i < (int)kPackTile / 16 + 2; i += 256) out[i] = 0;
    __syncthreads();
    const uint32_t n = tot >> 16, shift = (uint32_t)(d0 & 15);
    if (m) {
        uint32_t w = codes;
        for (uint32_t inv = ~m & 0xFFFFu; inv;) {  // the last invalid code taken out first
            const int j = 31 - __clz(inv);
            inv ^= 1u << j;
            const uint32_t low = 0xFFFFFFFFu >> (2 * j);
            w = (w & ~low) | (w << 2 & low);
        }
        const uint32_t p = shift + at, o = 2 * (p & 15);
        atomicOr(&out[p >> 4], w >> o);
        if (o) atomicOr(&out[(p >> 4) + 1], w << (32 - o));
    }
    __syncthreads();
    // the first and the last word may be shared with the tiles beside
    const uint32_t words = n ? (shift + n + 15) / 16 : 0;
    for (uint32_t i = tid; i < words; i += 256) {
        if (i == 0 || i + 1 == words) atomicOr(&packed[d0 / 16 + i], out[i]);
        else packed[d0 / 16 + i] = out[i];
    }
}

void pack_reads(mh_ctx* ctx, const uint8_t* d_ascii, uint64_t n_bases, const uint64_t* d_offs, uint64_t n_reads,
                mh_reads* out) {
    const uint64_t n_chunks = ceil_div(n_bases, 16);
    const bool vec = (reinterpret_cast<uintptr_t>(d_ascii) & 15) == 0;
    out->n_reads = n_reads;
    out->n_bases = n_bases;
    Buf<uint32_t> flags(ctx, 2);  // [0] any invalid byte, [1] empty reads
    flags.zero();
    Buf<uint32_t> packed(ctx, n_chunks + kPackPad);
    MH_CUDA(cudaMemsetAsync(packed.p + n_chunks, 0, kPackPad * sizeof(uint32_t), ctx->stream));
    MH_LAUNCH(ctx, "check_offs", grid_for(ctx, n_reads, 256), 256, 0, check_offs_kernel, d_offs, n_reads, n_bases,
              flags.p + 1, ctx->d_status);
    if (n_chunks)
        MH_LAUNCH(ctx, "pack_chunks", grid_for(ctx, n_chunks, 256), 256, 0, pack_chunks_kernel, d_ascii, n_bases, vec,
                  packed.p, flags.p);
    uint64_t fl[1];
    read_u64(ctx, reinterpret_cast<const uint64_t*>(flags.p), fl, 1);
    const bool any_invalid = (fl[0] & 0xFFFFFFFFull) != 0, any_empty = (fl[0] >> 32) != 0;
    const bool runs = (fl[0] >> 33) != 0;
    if (!any_invalid && !any_empty) {
        Buf<uint64_t> fo(ctx, n_reads + 1);
        MH_CUDA(cudaMemcpyAsync(fo.p, d_offs, sizeof(uint64_t) * (n_reads + 1), cudaMemcpyDeviceToDevice,
                                ctx->stream));
        Buf<uint32_t> fr(ctx, n_reads);
        if (n_reads) MH_LAUNCH(ctx, "iota", grid_for(ctx, n_reads, 256), 256, 0, iota_u32_kernel, fr.p, n_reads);
        out->n_frags = n_reads;
        out->n_packed = n_bases;
        out->packed = packed.release();
        out->frag_offs = fo.release();
        out->frag_read = fr.release();
        return;
    }
    // compaction of valid bases and fragment discovery
    packed.reset();
    const uint64_t n_tiles = ceil_div(n_bases, (uint64_t)kPackTile);
    Buf<uint64_t> first(ctx, n_tiles), dst(ctx, n_tiles + 1), fidx(ctx, n_tiles + 1);
    Buf<uint32_t> n_valid(ctx, n_tiles), n_starts(ctx, n_tiles);
    if (n_tiles) {
        MH_LAUNCH(ctx, "tile_reads", grid_for(ctx, n_tiles, 256), 256, 0, tile_reads_kernel, d_offs, n_reads, n_tiles,
                  first.p);
        MH_LAUNCH_B(ctx, "tile_count", n_bases, (unsigned)n_tiles, 256, 0,
                    (runs ? tile_count_kernel<true> : tile_count_kernel<false>), d_ascii, n_bases, vec,
                    d_offs, n_reads, first.p, n_valid.p, n_starts.p);
    }
    exclusive_scan_u32(ctx, n_valid.p, dst.p, n_tiles);
    exclusive_scan_u32(ctx, n_starts.p, fidx.p, n_tiles);
    uint64_t tot[2];
    Buf<uint64_t> both(ctx, 2);
    MH_CUDA(cudaMemcpyAsync(both.p, dst.p + n_tiles, sizeof(uint64_t), cudaMemcpyDeviceToDevice, ctx->stream));
    MH_CUDA(cudaMemcpyAsync(both.p + 1, fidx.p + n_tiles, sizeof(uint64_t), cudaMemcpyDeviceToDevice, ctx->stream));
    read_u64(ctx, both.p, tot, 2);
    const uint64_t n_packed = tot[0], n_frags = tot[1];
    Buf<uint64_t> fo(ctx, n_frags + 1);
    Buf<uint32_t> fr(ctx, n_frags);
    Buf<uint32_t> cp(ctx, ceil_div(n_packed, 16) + kPackPad);
    cp.zero();
    if (n_tiles)
        MH_LAUNCH_B(ctx, "tile_pack", n_bases + n_packed / 4 + 12 * n_frags, (unsigned)n_tiles, 256, 0,
                    (runs ? tile_pack_kernel<true> : tile_pack_kernel<false>), d_ascii, n_bases, vec, d_offs, n_reads,
                    first.p, dst.p, fidx.p, fo.p, fr.p, cp.p);
    MH_CUDA(cudaMemcpyAsync(fo.p + n_frags, dst.p + n_tiles, sizeof(uint64_t), cudaMemcpyDeviceToDevice,
                            ctx->stream));
    sync_and_check(ctx);
    out->n_frags = n_frags;
    out->n_packed = n_packed;
    out->packed = cp.release();
    out->frag_offs = fo.release();
    out->frag_read = fr.release();
}

// Reads in host memory (pinned for overlap): up to one piece (kPiece bytes)
// is uploaded on the context stream and packed as from the device.  Larger
// inputs stream through two device staging buffers of kPiece bytes on the
// context's copy stream while the context stream packs the piece before
// (piece starts are multiples of 16 bases, so every piece fills whole
// packed words of its own); only the packed stream and the offsets stay on
// the device.  If some byte is not a base or some read is empty, the
// fragments must be found and the bases compacted: the ASCII is then
// uploaded whole and packed as from the device.
constexpr uint64_t kPiece = 256ull << 20;

// staging piece in bytes: kPiece, or MH_PACK_PIECE (a multiple of 16; tests)
static uint64_t piece_bytes() {
    static const uint64_t v = [] {
        const char* e = std::getenv("MH_PACK_PIECE");
        const long long x = e ? std::atoll(e) : 0;
        return x >= 16 ? (uint64_t)x / 16 * 16 : kPiece;
    }();
    return v;
}

static cudaStream_t copy_stream(mh_ctx* ctx) {
    if (!ctx->copy_stream) MH_CUDA(cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
    return ctx->copy_stream;
}

void pack_reads_host(mh_ctx* ctx, const uint8_t* h_ascii, uint64_t n_bases, const uint64_t* h_offs, uint64_t n_reads,
                     mh_reads* out) {
    if (n_bases <= piece_bytes()) {
        // one piece: a plain upload on the context stream, then the device path
        Buf<uint8_t> da(ctx, n_bases + 16);
        Buf<uint64_t> doff(ctx, n_reads + 1);
        if (n_bases) MH_CUDA(cudaMemcpyAsync(da.p, h_ascii, n_bases, cudaMemcpyHostToDevice, ctx->stream));
        MH_CUDA(cudaMemcpyAsync(doff.p, h_offs, sizeof(uint64_t) * (n_reads + 1), cudaMemcpyHostToDevice,
                                ctx->stream));
        pack_reads(ctx, da.p, n_bases, doff.p, n_reads, out);
        return;
    }
    cudaStream_t cs = copy_stream(ctx);
    const uint64_t n_chunks = ceil_div(n_bases, 16);
    const uint64_t piece = piece_bytes();
    const uint64_t n_pieces = ceil_div(n_bases, piece);
    Buf<uint64_t> doff(ctx, n_reads + 1);
    Buf<uint32_t> flags(ctx, 2);  // [0] any invalid byte, [1] any empty read
    flags.zero();
    Buf<uint32_t> packed(ctx, n_chunks + kPackPad);
    MH_CUDA(cudaMemsetAsync(packed.p + n_chunks, 0, kPackPad * sizeof(uint32_t), ctx->stream));
    Buf<uint8_t> stage[2] = {Buf<uint8_t>(ctx, piece), Buf<uint8_t>(ctx, piece)};
    cudaEvent_t* ev = ctx->pack_ev;  // created once a context
    for (int i = 0; i < 5; i++)
        if (!ev[i]) MH_CUDA(cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming));
    {
        // the copy stream writes buffers just allocated on the context stream
        MH_CUDA(cudaEventRecord(ev[4], ctx->stream));
        MH_CUDA(cudaStreamWaitEvent(cs, ev[4], 0));
        MH_CUDA(cudaMemcpyAsync(doff.p, h_offs, sizeof(uint64_t) * (n_reads + 1), cudaMemcpyHostToDevice, cs));
        MH_CUDA(cudaEventRecord(ev[4], cs));
        MH_CUDA(cudaStreamWaitEvent(ctx->stream, ev[4], 0));
        MH_LAUNCH(ctx, "check_offs", grid_for(ctx, n_reads, 256), 256, 0, check_offs_kernel, doff.p, n_reads,
                  n_bases, flags.p + 1, ctx->d_status);
        for (uint64_t q = 0; q < n_pieces; q++) {
            const int s = (int)(q & 1);
            const uint64_t b = q * piece, len = n_bases - b < piece ? n_bases - b : piece;
            if (q >= 2) MH_CUDA(cudaStreamWaitEvent(cs, ev[2 + s], 0));  // piece q-2 packed
            MH_CUDA(cudaMemcpyAsync(stage[s].p, h_ascii + b, len, cudaMemcpyHostToDevice, cs));
            MH_CUDA(cudaEventRecord(ev[s], cs));
            MH_CUDA(cudaStreamWaitEvent(ctx->stream, ev[s], 0));
            MH_LAUNCH(ctx, "pack_chunks", grid_for(ctx, ceil_div(len, 16), 256), 256, 0, pack_chunks_kernel,
                      stage[s].p, len, true, packed.p + b / 16, flags.p);
            MH_CUDA(cudaEventRecord(ev[2 + s], ctx->stream));
        }
    }
    stage[0].reset();
    stage[1].reset();
    uint64_t fl[1];
    read_u64(ctx, reinterpret_cast<const uint64_t*>(flags.p), fl, 1);
    if ((fl[0] & 0xFFFFFFFFull) == 0 && (fl[0] >> 32) == 0) {
        Buf<uint32_t> fr(ctx, n_reads);
        if (n_reads) MH_LAUNCH(ctx, "iota", grid_for(ctx, n_reads, 256), 256, 0, iota_u32_kernel, fr.p, n_reads);
        out->n_reads = n_reads;
        out->n_bases = n_bases;
        out->n_frags = n_reads;
        out->n_packed = n_bases;
        out->packed = packed.release();
        out->frag_offs = doff.release();
        out->frag_read = fr.release();
        return;
    }
    packed.reset();
    Buf<uint8_t> da(ctx, n_bases + 16);
    if (n_bases) MH_CUDA(cudaMemcpyAsync(da.p, h_ascii, n_bases, cudaMemcpyHostToDevice, ctx->stream));
    pack_reads(ctx, da.p, n_bases, doff.p, n_reads, out);
}

}  // namespace mh

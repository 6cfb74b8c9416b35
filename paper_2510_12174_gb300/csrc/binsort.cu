// Binning: a depth order of the kept pairs, emission, a stable sort by tile,
// ranges; and the 64-bit pair sort of unigs_sort_pairs_static.
//
// The paper extends the tile pipeline of 3DGS (Sec. 3.4): each Gaussian is
// duplicated once per tile its 3-sigma rectangle overlaps, keyed by
// (global tile id << 32 | float32 bits of its camera-frame centre depth), and
// sorted so that every tile holds a front-to-back list, ties in depth in
// Gaussian order.  Sorting the instances by the whole key moves every one of
// them once per digit of 32 + tile bits.  Here the (camera, Gaussian) pairs
// with a kept tile, several times fewer than their instances, are sorted by
// depth first (four 8-bit passes, stable from pair order; depths are
// > z_near > 0, so their bit patterns order like the values).  The instances
// are then emitted in that order, and a stable sort by tile id alone (digits
// of at most 9 bits: one or two passes, 4-byte keys) leaves the same list.
//
// Each pass is one kernel: blocks take chunks by ticket, rank their keys in
// shared memory, and find the global position of each digit by looking back
// over the chunks before them (each chunk publishes its digit counts, then
// its inclusive prefixes).  A chunk only waits for chunks whose ticket was
// drawn earlier, so the wait ends; it is bounded all the same.
//
// Every kernel reads the instance count from device memory, so the whole
// sequence runs without a host round trip (CUDA-graph capture).
//
// What bounds it: the ranking's chain through shared memory (match, read and
// write a count, 16 times per thread) with 30 warps per SM; a tile pass issues
// in a quarter of the cycles and waits on shared memory for most of the rest,
// and moves the 16 bytes of each of 142M instances at 2.6 of the 6.8 TB/s that a
// copy reaches.  Small inputs: launches.  Against
// six or seven passes over 12-byte (key, value) pairs, each of a histogram, a
// three-kernel scan and a scatter (31 to 36 launches instead of 10 to 12):
// 16 views of 3M Gaussians, 142M instances, scan to ranges 13.3 -> 5.2 ms; one
// 1280x720 view of 1M, 2.7M instances, 0.36 -> 0.22 ms; one 256x256 view of
// 10k, 0.33 -> 0.24 ms for the whole frame.
#include "launch.h"
#include "lookback.cuh"

namespace unigs {

// ------------------------------------------------------------ block scan
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* sh_warp,
                                                         uint32_t* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = lane < (int)(blockDim.x >> 5) ? sh_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh_warp[lane] = s;  // inclusive prefix of warp totals
    }
    __syncthreads();
    const uint32_t warp_base = wid ? sh_warp[wid - 1] : 0;
    if (total) *total = sh_warp[(blockDim.x >> 5) - 1];
    const uint32_t r = warp_base + x - v;
    __syncthreads();
    return r;
}

// Phase 1: per-block sums of SCAN_ITEMS elements.
__global__ void __launch_bounds__(256)
    scan_reduce_kernel(const uint32_t* __restrict__ in, int64_t n, uint32_t* __restrict__ partial) {
    __shared__ uint32_t sw[32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_ITEMS;
    uint32_t s = 0;
    for (int j = threadIdx.x; j < SCAN_ITEMS; j += blockDim.x) {
        const int64_t i = base + j;
        if (i < n) s += in[i];
    }
    uint32_t tot;
    block_exclusive_scan(s, sw, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

// Phase 2: exclusive scan of the block sums by one block; writes the total.
__global__ void __launch_bounds__(1024)
    scan_partials_kernel(uint32_t* __restrict__ partial, int64_t nb, uint32_t* __restrict__ total_out) {
    __shared__ uint32_t sw[32];
    uint32_t carry = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += blockDim.x) {
        const int64_t i = b0 + threadIdx.x;
        const uint32_t v = i < nb ? partial[i] : 0;
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan(v, sw, &tot);
        if (i < nb) partial[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0 && total_out) *total_out = carry;
}

// Phase 3: scan within each block, offset by the scanned block sum.
__global__ void __launch_bounds__(256)
    scan_down_kernel(const uint32_t* __restrict__ in, int64_t n, const uint32_t* __restrict__ partial,
                     uint32_t* __restrict__ out) {
    __shared__ uint32_t sw[32];
    constexpr int PER = SCAN_ITEMS / 256;
    const int64_t base = (int64_t)blockIdx.x * SCAN_ITEMS + (int64_t)threadIdx.x * PER;
    uint32_t v[PER];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int64_t i = base + j;
        v[j] = i < n ? in[i] : 0;
        s += v[j];
    }
    uint32_t run = block_exclusive_scan(s, sw, nullptr) + partial[blockIdx.x];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int64_t i = base + j;
        if (i < n) out[i] = run;
        run += v[j];
    }
}

int scan_u32(const uint32_t* in, int64_t n, uint32_t* partial, uint32_t* out, uint32_t* total,
             cudaStream_t st) {
    const int64_t nb = (n + SCAN_ITEMS - 1) / SCAN_ITEMS;
    if (nb == 0) return 0;
    scan_reduce_kernel<<<(unsigned)nb, 256, 0, st>>>(in, n, partial);
    scan_partials_kernel<<<1, 1024, 0, st>>>(partial, nb, total);
    scan_down_kernel<<<(unsigned)nb, 256, 0, st>>>(in, n, partial, out);
    return 3;
}

// ------------------------------------------------------- single-kernel passes
// Stores a look-back word (look_back_walk has its layout).
__device__ __forceinline__ void lb_store(unsigned long long* w, uint32_t epoch, uint32_t state,
                                         uint32_t count) {
    const unsigned long long v = ((unsigned long long)(epoch << 2 | state) << 32) | count;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long lb_load(const unsigned long long* w) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(w) : "memory");
    return v;
}

// A word of the emission's look-back: state << 62 | count.
__device__ __forceinline__ void emit_store(unsigned long long* w, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(v) : "memory");
}

constexpr uint32_t LB_WAIT_LIMIT = 1u << 20;  // polls of one unwritten word, about a second
constexpr int LB_WIDE = 8;                    // predecessors read per step

// look_back_walk over column `col` of the look-back table (rows of `stride` words).
__device__ __forceinline__ bool look_back(const unsigned long long* words, int64_t chunk,
                                          int stride, int col, uint32_t epoch, uint32_t* sum_out) {
    return look_back_walk<LB_WIDE>(
        [&](int64_t p) { return lb_load(words + p * stride + col); }, chunk, epoch, LB_WAIT_LIMIT,
        sum_out);
}

// Digit counts of the depth keys of the pairs with a kept tile, for all four
// passes at once; clears the look-back words of the depth passes and of the
// emission, and the ranges.
__global__ void __launch_bounds__(512)
    depth_hist_kernel(const uint32_t* __restrict__ touched, const uint32_t* __restrict__ zbits,
                      int64_t total, SortState* __restrict__ st,
                      unsigned long long* __restrict__ words, int64_t n_words,
                      unsigned long long* __restrict__ emit_words, int64_t n_emit_words,
                      uint2* __restrict__ ranges, int64_t n_tiles) {
    pdl_begin();
    __shared__ uint32_t h[4][256];
    for (int j = threadIdx.x; j < 4 * 256; j += blockDim.x) (&h[0][0])[j] = 0;
    __syncthreads();
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < n_words; i += stride) words[i] = 0ull;
    for (int64_t i = i0; i < n_emit_words; i += stride) emit_words[i] = 0ull;
    for (int64_t i = i0; i < n_tiles; i += stride) ranges[i] = make_uint2(0u, 0u);
    uint32_t kept = 0;
    auto count = [&](uint32_t cnt, uint32_t z) {
        if (cnt == 0) return;
        ++kept;
#pragma unroll
        for (int p = 0; p < 4; ++p) atomicAdd(&h[p][(z >> (8 * p)) & 255u], 1u);
    };
    // four pairs a load (the regions start at multiples of 256 bytes)
    const int64_t n4 = total / 4;
#pragma unroll 2
    for (int64_t i = i0; i < n4; i += stride) {
        const uint4 c = reinterpret_cast<const uint4*>(touched)[i];
        const uint4 z = reinterpret_cast<const uint4*>(zbits)[i];
        count(c.x, z.x);
        count(c.y, z.y);
        count(c.z, z.z);
        count(c.w, z.w);
    }
    if (i0 < total - 4 * n4) count(touched[4 * n4 + i0], zbits[4 * n4 + i0]);
    kept = __reduce_add_sync(0xffffffffu, kept);
    if ((threadIdx.x & 31) == 0 && kept) atomicAdd(&st->n_kept, kept);
    __syncthreads();
    for (int j = threadIdx.x; j < 4 * 256; j += blockDim.x) {
        const uint32_t c = (&h[0][0])[j];
        if (c) atomicAdd(&st->dhist[0][0] + j, c);
    }
}

struct OnesweepParams {
    const uint32_t* kin;   // keys (FROM_PAIRS: depth bits of every pair)
    const uint32_t* vin;   // values (FROM_PAIRS: touched counts, the value is the index)
    uint32_t* kout;
    uint32_t* vout;
    const uint32_t* hist;  // digit counts of this pass
    unsigned long long* words;
    uint32_t* ticket;
    const uint32_t* n_ptr; // element count on the device (FROM_PAIRS: n_host)
    int64_t n_host;
    SortState* st;
    WsHeader* hdr;
    int shift, bits;       // digit (key >> shift) & (2^bits - 1), bits <= 9
    uint32_t epoch;
};

template <int PER>
struct OnesweepSmem {
    uint32_t sk[RS_THREADS * PER];
    uint32_t sv[RS_THREADS * PER];
    uint16_t whist[RS_WARPS][RS_BINS];
    uint32_t goff[RS_BINS];  // global position of the block's first key of a digit
    uint32_t loff[RS_BINS];  // its position in the block's staging
    uint32_t base[RS_BINS];  // global position of the digit
    uint32_t wsum[RS_WARPS];
    uint32_t chunk;
};

// Exclusive scan over RS_THREADS values, one per thread.
__device__ __forceinline__ uint32_t scan512(uint32_t v, uint32_t* wsum, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < RS_WARPS; ++i) {
        const uint32_t s = wsum[i];
        if (i < w) before += s;
        all += s;
    }
    __syncthreads();
    *total = all;
    return before + x - v;
}

// One stable radix pass.  Warp w of a block owns 32 PER consecutive keys of
// the block's chunk and walks them 32 at a time in order: __match_any_sync
// ranks equal digits inside a step, a running count per warp orders the
// steps, a prefix over the warps orders the warps.  The pairs are placed in
// shared memory in (digit, input) order and written out by consecutive
// threads, so the pairs of a digit land at consecutive addresses.
// FROM_PAIRS: the first depth pass, reading (touched, depth) of every
// (camera, Gaussian) pair in pair order and dropping those without a kept
// tile.  KEYS: also write the keys (the last depth pass needs only the order).
template <int PER, bool FROM_PAIRS, bool KEYS>
__global__ void __launch_bounds__(RS_THREADS, 2) onesweep_kernel(const OnesweepParams P) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char rs_raw[];
    OnesweepSmem<PER>& S = *reinterpret_cast<OnesweepSmem<PER>*>(rs_raw);
    constexpr int ITEMS = RS_THREADS * PER;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int bins = 1 << P.bits;
    const uint32_t dmask = (uint32_t)bins - 1u;
    const int64_t n = FROM_PAIRS ? P.n_host : (int64_t)*P.n_ptr;
    uint32_t tot;
    {
        const uint32_t e = scan512(tid < bins ? P.hist[tid] : 0u, S.wsum, &tot);
        S.base[tid] = e;
    }
    for (;;) {
        // an earlier wait that gave up leaves nothing to sort (no such chunk)
        if (tid == 0)
            S.chunk = *(volatile uint32_t*)&P.st->abort ? ~0u : atomicAdd(P.ticket, 1u);
        for (int j = tid; j < RS_WARPS * RS_BINS / 2; j += RS_THREADS)
            reinterpret_cast<uint32_t*>(&S.whist[0][0])[j] = 0u;
        __syncthreads();
        const int64_t chunk = S.chunk;
        const int64_t block0 = chunk * ITEMS;
        if (block0 >= n) break;
        const int64_t first = block0 + (int64_t)w * (32 * PER);
        uint32_t k[PER], v[PER];
        uint32_t rank[PER];  // digit << 16 | rank within the warp; ~0: no key
#pragma unroll
        for (int it = 0; it < PER; ++it) {
            const int64_t i = first + it * 32 + lane;
            bool ok = i < n;
            k[it] = ok ? P.kin[i] : 0u;
            v[it] = ok ? P.vin[i] : 0u;
            if (FROM_PAIRS) {
                ok = ok && v[it] != 0u;
                v[it] = (uint32_t)i;
            }
            rank[it] = ok ? 0u : ~0u;
        }
#pragma unroll
        for (int it = 0; it < PER; ++it) {
            const bool ok = rank[it] == 0u;
            const uint32_t d = ok ? (k[it] >> P.shift) & dmask : RS_BINS;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = ok ? S.whist[w][d] : 0u;
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1)
                S.whist[w][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            if (ok) rank[it] = (d << 16) | (before + __popc(peers & lt_mask));
        }
        __syncthreads();
        // digit tid: its count, the warps' offsets within it, its staging offset
        uint32_t cnt = 0;
#pragma unroll
        for (int w2 = 0; w2 < RS_WARPS; ++w2) {
            const uint32_t c = S.whist[w2][tid];
            S.whist[w2][tid] = (uint16_t)cnt;
            cnt += c;
        }
        unsigned long long* row = P.words + chunk * bins + tid;
        if (tid < bins) lb_store(row, P.epoch, chunk == 0 ? 2u : 1u, cnt);
        const uint32_t lo = scan512(cnt, S.wsum, &tot);
        S.loff[tid] = lo;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < PER; ++it)
            if (rank[it] != ~0u) {
                const uint32_t d = rank[it] >> 16;
                const uint32_t lp = S.loff[d] + S.whist[w][d] + (rank[it] & 0xffffu);
                S.sk[lp] = k[it];
                S.sv[lp] = v[it];
            }
        bool bad = false;
        if (tid < bins) {
            uint32_t before = 0;
            if (chunk > 0) {
                bad = !look_back(P.words, chunk, bins, tid, P.epoch, &before);
                if (!bad) lb_store(row, P.epoch, 2u, before + cnt);
            }
            S.goff[tid] = S.base[tid] + before;
        }
        if (__syncthreads_or(bad)) {
            if (tid == 0) {
                atomicExch(&P.st->abort, 1u);
                set_status(P.hdr, UNIGS_ERR_TIMEOUT);
            }
            break;
        }
        for (uint32_t j = tid; j < tot; j += RS_THREADS) {
            const uint32_t key = S.sk[j];
            const uint32_t d = (key >> P.shift) & dmask;
            const uint32_t dst = S.goff[d] + (j - S.loff[d]);
            if (KEYS) P.kout[dst] = key;
            P.vout[dst] = S.sv[j];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ emission
struct EmitParams {
    const CamTable* tab;
    int64_t n;
    int tw, th;
    int64_t capacity;
    const uint2* rect;
    const uint32_t* touched;
    const unsigned long long* masks;
    const float* cull;
    const uint32_t* keep_bits;        // kept-tile bits of the large rectangles
    const uint32_t* order;            // kept pairs by depth
    SortState* st;
    WsHeader* hdr;
    unsigned long long* emit_words;   // look-back, one word per chunk
    unsigned long long* words;        // look-back table of the tile passes, cleared here
    uint4* big;                       // pairs left to emit_big_kernel
    uint32_t* keys;                   // global tile ids
    uint32_t* vals;                   // Gaussian indices
    int passes, bits, items;          // tile passes: count, digit bits, keys per chunk
};

// Writes one instance and counts its tile digits.
__device__ __forceinline__ void put_instance(const EmitParams& P, uint32_t (*hist)[RS_BINS],
                                             uint32_t dst, uint32_t tile, uint32_t g) {
    P.keys[dst] = tile;
    P.vals[dst] = g;
    const uint32_t dmask = (1u << P.bits) - 1u;
    for (int p = 0; p < P.passes; ++p) atomicAdd(&hist[p][(tile >> (p * P.bits)) & dmask], 1u);
}

// The block's digit counts, added to the binning's.
__device__ __forceinline__ void flush_hist(const EmitParams& P, uint32_t (*hist)[RS_BINS]) {
    __syncthreads();
    for (int p = 0; p < P.passes; ++p)
        for (int j = threadIdx.x; j < (1 << P.bits); j += blockDim.x)
            if (hist[p][j]) atomicAdd(&P.st->thist[p][j], hist[p][j]);
}

// Position of set bit number r of m (r < popcount(m)).
__device__ __forceinline__ int nth_bit(unsigned long long m, int r) {
    int pos = 0;
    uint32_t x = (uint32_t)m;
    int c = __popc(x);
    if (r >= c) { r -= c; x = (uint32_t)(m >> 32); pos = 32; }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        c = __popc(x & ((1u << s) - 1u));
        if (r >= c) { r -= c; x >>= s; pos += s; }
    }
    return pos;
}

// One instance per kept tile, in (depth, pair) order.  A block takes 256
// pairs, finds the position of its first instance by look-back, and its warps
// write theirs from the preprocess's bit masks, one output slot per lane (so
// that a warp's stores are consecutive whatever the rectangles' sizes).
// Rectangles of more than MASK_TILES tiles are listed for emit_big_kernel:
// in depth order the largest ones, those nearest the camera, all fall into the
// first few blocks (emitted there, a 1280x720 view of 1M Gaussians took
// 1.18 ms; with the list 0.034 + 0.051 ms).  Also counts the tile digits and clears the
// look-back words of the chunks that its own instances start.
__global__ void __launch_bounds__(256) emit_kernel(const EmitParams P) {
    pdl_begin();
    __shared__ uint32_t hist[TILE_PASSES_MAX][RS_BINS];
    __shared__ uint32_t sw[32];
    __shared__ uint32_t s_chunk;
    __shared__ unsigned long long s_base;
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31;
    const int bins = 1 << P.bits;
    for (int j = tid; j < P.passes * RS_BINS; j += 256) (&hist[0][0])[j] = 0u;
    const int64_t n_kept = P.st->n_kept;
    for (;;) {
        if (tid == 0)
            s_chunk = *(volatile uint32_t*)&P.st->abort ? ~0u
                                                        : atomicAdd(&P.st->ticket[TICKET_EMIT], 1u);
        __syncthreads();
        const int64_t chunk = s_chunk;
        if (chunk * 256 >= n_kept) break;
        const int64_t i = chunk * 256 + tid;
        uint32_t t = 0, cnt = 0;
        if (i < n_kept) {
            t = P.order[i];
            cnt = P.touched[t];
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan(cnt, sw, &tot);
        // the instances of all chunks may exceed 32 bits (then far over the
        // capacity): the words' 62-bit counts are kept apart from the state
        // in the two top bits.  The first warp reads 64 predecessors a step
        if (tid < 32) {
            constexpr unsigned long long VAL = (1ull << 62) - 1ull;
            unsigned long long base = 0;
            unsigned long long* w = P.emit_words;
            bool bad = false;
            if (lane == 0) emit_store(w + chunk, (chunk == 0 ? 2ull : 1ull) << 62 | tot);
            PollLimit wait(LB_WAIT_LIMIT);
            for (int64_t p = chunk - 1; p >= 0;) {
                // lane l: predecessors p - 2 l and p - 2 l - 1
                const int64_t p0 = p - 2 * lane;
                const unsigned long long v0 = p0 >= 0 ? lb_load(w + p0) : 2ull << 62;
                const unsigned long long v1 = p0 >= 1 ? lb_load(w + p0 - 1) : 2ull << 62;
                const int s0 = (int)(v0 >> 62), s1 = (int)(v1 >> 62);
                // the lanes up to the first inclusive prefix or unwritten word
                const bool stop0 = s0 != 1, stop1 = s1 != 1;
                const uint32_t stops = __ballot_sync(0xffffffffu, stop0 || stop1);
                const int at = stops ? __ffs(stops) - 1 : 32;
                unsigned long long c = 0;
                if (lane < at) c = (v0 & VAL) + (v1 & VAL);
                if (lane == at) c = (s0 ? v0 & VAL : 0ull) + (s0 == 1 && s1 ? v1 & VAL : 0ull);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                base += c;
                if (at == 32) {
                    p -= 64;
                    wait.give_up(true);
                    continue;
                }
                const int a0 = __shfl_sync(0xffffffffu, s0, at), a1 = __shfl_sync(0xffffffffu, s1, at);
                if (a0 == 2 || (a0 == 1 && a1 == 2)) break;
                const int used = 2 * at + (a0 == 1 ? 1 : 0);
                p -= used;  // the unwritten word is read again
                if (wait.give_up(used > 0)) {
                    bad = true;
                    break;
                }
            }
            if (lane == 0) {
                if (!bad && chunk > 0) emit_store(w + chunk, 2ull << 62 | (base + tot));
                s_base = base;
                s_bad = bad;
            }
        }
        __syncthreads();
        if (s_bad) {
            if (tid == 0) {
                atomicExch(&P.st->abort, 1u);
                set_status(P.hdr, UNIGS_ERR_TIMEOUT);
            }
            break;
        }
        const unsigned long long end = s_base + tot;
        const bool fits = end <= (unsigned long long)P.capacity;
        if (tid == 0 && (chunk + 1) * 256 >= n_kept) {
            P.hdr->need = end;
            P.hdr->n_instances = fits ? (uint32_t)end : 0u;
            if (!fits) set_status(P.hdr, UNIGS_ERR_CAPACITY);
        }
        if (!fits) continue;  // uniform; s_base is not rewritten before the next barrier
        for (unsigned long long b = (s_base + P.items - 1) / P.items; b * P.items < end; ++b)
            for (int j = tid; j < bins; j += 256) P.words[b * bins + j] = 0ull;
        uint32_t o = (uint32_t)s_base + ex;
        int x0 = 0, y0 = 0, bw = 1, nt = 0, tiles_x = 0;
        uint32_t g = 0, toff = 0;
        unsigned long long mask = 0;
        if (cnt) {
            const int k = (int)(t / (uint32_t)P.n);
            g = t - (uint32_t)k * (uint32_t)P.n;
            const DevCam& cam = P.tab->cam[k];
            const uint2 r = P.rect[t];
            x0 = r.x & 0xffff;
            y0 = r.y & 0xffff;
            bw = (int)(r.x >> 16) - x0;
            nt = bw * ((int)(r.y >> 16) - y0);
            toff = (uint32_t)cam.tile_off;
            tiles_x = cam.tiles_x;
            if (nt <= MASK_TILES) mask = P.masks[t];
        }
        // slot q of the warp: the pair whose first slot is the last at or before q
        const uint32_t sc = nt <= MASK_TILES ? cnt : 0u;
        uint32_t incl = sc;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += y;
        }
        const uint32_t pre = incl - sc;
        const uint32_t slots = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t tile0 = toff + (uint32_t)(y0 * tiles_x + x0);
        for (uint32_t q0 = 0; q0 < slots; q0 += 32) {
            const uint32_t q = q0 + lane;
            int src = 0;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                const uint32_t pc = __shfl_sync(0xffffffffu, pre, src + s);
                if (pc <= q) src += s;
            }
            const uint32_t r = q - __shfl_sync(0xffffffffu, pre, src);
            const uint32_t so = __shfl_sync(0xffffffffu, o, src);
            const uint32_t st0 = __shfl_sync(0xffffffffu, tile0, src);
            const uint32_t sg = __shfl_sync(0xffffffffu, g, src);
            const int sbw = __shfl_sync(0xffffffffu, bw, src);
            const int stx = __shfl_sync(0xffffffffu, tiles_x, src);
            const unsigned long long sm = __shfl_sync(0xffffffffu, mask, src);
            if (q < slots) {
                const int j = nth_bit(sm, (int)r);
                const int ry = j / sbw;
                put_instance(P, hist, so + r, st0 + (uint32_t)(ry * stx + (j - ry * sbw)), sg);
            }
        }
        const bool large = nt > MASK_TILES && cnt > 0;
        const unsigned bm = __ballot_sync(0xffffffffu, large);
        if (bm) {
            uint32_t slot = 0;
            if (lane == 0) slot = atomicAdd(&P.st->n_big, (uint32_t)__popc(bm));
            slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(bm & ((1u << lane) - 1u));
            if (large) P.big[slot] = make_uint4(t, o, cnt, 0u);
        }
        __syncthreads();
    }
    flush_hist(P, hist);
}

// The rectangles of more than MASK_TILES tiles, BIG_SEG tiles per task: a
// warp takes their bits or, without them, repeats the tile test, 32 tiles
// per step, and the positions of the kept ones from the pair's own counter.  (The order of a pair's
// instances does not reach the sorted lists: each lies in another tile.)
// Task s * n_big + e is segment s of pair e; a warp's lanes look at every
// `warps`-th task for those that exist, so that neighbouring tasks (the
// largest rectangles stand together) go to different warps.
constexpr int BIG_SEG = WIDE_TILES;
__global__ void __launch_bounds__(256) emit_big_kernel(const EmitParams P, int max_segs) {
    pdl_begin();
    __shared__ uint32_t hist[TILE_PASSES_MAX][RS_BINS];
    const int lane = threadIdx.x & 31;
    const int64_t n_big = P.st->n_big;
    if (n_big == 0) return;
    for (int j = threadIdx.x; j < P.passes * RS_BINS; j += 256) (&hist[0][0])[j] = 0u;
    __syncthreads();
    const int64_t n_tasks = n_big * max_segs;
    const int64_t warps = (int64_t)gridDim.x * 8;
    // neighbouring warps in different blocks
    const int64_t warp = (threadIdx.x >> 5) * (int64_t)gridDim.x + blockIdx.x;
    for (int64_t q0 = warp; q0 < n_tasks; q0 += warps * 32) {
        const int64_t q = q0 + lane * warps;
        uint32_t t = 0, o = 0, cnt = 0, e = 0;
        int seg = 0, x0 = 0, y0 = 0, bw = 1, nt = 0;
        if (q < n_tasks) {
            seg = (int)(q / n_big);
            e = (uint32_t)(q - seg * n_big);
            const uint4 b = P.big[e];
            t = b.x;
            o = b.y;
            cnt = b.z;
            const uint2 r = P.rect[t];
            x0 = r.x & 0xffff;
            y0 = r.y & 0xffff;
            bw = (int)(r.x >> 16) - x0;
            nt = bw * ((int)(r.y >> 16) - y0);
        }
        unsigned todo = __ballot_sync(0xffffffffu, seg * BIG_SEG < nt);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t bt = __shfl_sync(0xffffffffu, t, src);
            const int k = (int)(bt / (uint32_t)P.n);
            const uint32_t g = bt - (uint32_t)k * (uint32_t)P.n;
            const DevCam& cam = P.tab->cam[k];
            const float4* cs = reinterpret_cast<const float4*>(P.cull + (size_t)bt * CULL_FLOATS);
            const float4 c0 = cs[0], c1 = cs[1];
            const float cr[CULL_FLOATS] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
            const int snt = __shfl_sync(0xffffffffu, nt, src);
            const bool wide = snt <= WIDE_TILES;
            const int j1 = __shfl_sync(0xffffffffu, seg, src) * BIG_SEG;
            // the segment's kept tiles as bits, word i in lane i, or the test
            const uint32_t at = wide ? 0u : __float_as_uint(cr[C_BITS]);
            const bool known = at != NO_BITS;
            const uint32_t* words =
                wide ? reinterpret_cast<const uint32_t*>(cs) : P.keep_bits + (known ? at : 0u) + j1 / 32;
            CullTest ct = {};
            uint32_t bits = 0;
            if (!known)
                ct = cull_test(cr);
            else if (lane < BIG_SEG / 32 && j1 + 32 * lane < snt)
                bits = words[lane];
            const int bx0 = __shfl_sync(0xffffffffu, x0, src);
            const int by0 = __shfl_sync(0xffffffffu, y0, src);
            const int bbw = __shfl_sync(0xffffffffu, bw, src);
            const int bn = min(snt, j1 + BIG_SEG);
            const uint32_t bo = __shfl_sync(0xffffffffu, o, src);
            const uint32_t bc = __shfl_sync(0xffffffffu, cnt, src);
            uint32_t* cursor = &P.big[__shfl_sync(0xffffffffu, e, src)].w;
            // where the bits are known, one addition reserves the segment's
            // positions (a wide rectangle is one segment of one warp)
            uint32_t run = 0;
            if (known && !wide) {
                const uint32_t total = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(bits));
                if (lane == 0) run = atomicAdd(cursor, total);
                run = __shfl_sync(0xffffffffu, run, 0);
            }
            for (int j0 = j1; j0 < bn; j0 += 32) {
                const int j = j0 + lane;
                const int ry = j / bbw;
                const int tx = bx0 + (j - ry * bbw), ty = by0 + ry;
                const unsigned m =
                    known ? __shfl_sync(0xffffffffu, bits, (j0 - j1) / 32)
                         : __ballot_sync(0xffffffffu,
                                         j < bn && tile_keep(ct, tx, ty, P.tw, P.th));
                const bool keep = (m >> lane) & 1u;
                if (!m) continue;
                uint32_t pos = run;
                if (known) {
                    run += __popc(m);
                } else {
                    if (lane == 0) pos = atomicAdd(cursor, (uint32_t)__popc(m));
                    pos = __shfl_sync(0xffffffffu, pos, 0);
                }
                pos += __popc(m & ((1u << lane) - 1u));
                if (keep && pos < bc)
                    put_instance(P, hist, bo + pos,
                                 (uint32_t)cam.tile_off + (uint32_t)(ty * cam.tiles_x + tx), g);
            }
        }
    }
    flush_hist(P, hist);
}

// ------------------------------------------------------------ radix sort
// (the 64-bit pair sort)
__device__ __forceinline__ uint32_t n_valid(const WsHeader* hdr) {
    return hdr->status == UNIGS_ERR_CAPACITY ? 0u : hdr->n_instances;
}

// Per-block digit counts, stored digit-major: hist[d * nb + b].  The digit of
// a key is (key >> shift) & dmask (dmask 255 for a whole byte; fewer bits on
// a last pass that must ignore the key bits above the sorted ones).
__global__ void __launch_bounds__(256)
    radix_hist_kernel(const unsigned long long* __restrict__ keys, const WsHeader* __restrict__ hdr,
                      int shift, uint32_t dmask, int nb, uint32_t* __restrict__ hist) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t n = n_valid(hdr);
    const int64_t base = (int64_t)blockIdx.x * SORT_ITEMS;
    for (int j = threadIdx.x; j < SORT_ITEMS; j += 256) {
        const int64_t i = base + j;
        if (i < n) atomicAdd(&cnt[(uint32_t)(keys[i] >> shift) & dmask], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nb + blockIdx.x] = cnt[threadIdx.x];
}

// Stable scatter.  Warp w of the block owns keys [w*256, w*256+256) of the
// block's chunk and walks them 32 at a time in order; __match_any_sync ranks
// equal digits inside each step, a per-warp running count orders the steps,
// and a prefix over warps orders the warps.  The block's pairs are first
// placed in shared memory in (digit, input order) order, then written out by
// consecutive threads: the pairs of one digit land at consecutive addresses,
// so the stores coalesce.
__global__ void __launch_bounds__(256)
    radix_scatter_kernel(const unsigned long long* __restrict__ kin,
                         const uint32_t* __restrict__ vin, unsigned long long* __restrict__ kout,
                         uint32_t* __restrict__ vout, const uint32_t* __restrict__ scanned,
                         const WsHeader* __restrict__ hdr, int shift, uint32_t dmask, int nb) {
    __shared__ uint32_t whist[8][256];
    __shared__ uint32_t goff[256];
    __shared__ uint32_t loff[256];  // first block-local position of each digit
    __shared__ uint32_t wsum[8];
    __shared__ unsigned long long sk[SORT_ITEMS];
    __shared__ uint32_t sv[SORT_ITEMS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < 8 * 256; j += 256) (&whist[0][0])[j] = 0;
    goff[threadIdx.x] = scanned[(int64_t)threadIdx.x * nb + blockIdx.x];
    __syncthreads();
    const uint32_t n = n_valid(hdr);
    const int64_t block0 = (int64_t)blockIdx.x * SORT_ITEMS;
    const int64_t base = block0 + w * 256;
    const uint32_t lt_mask = (1u << lane) - 1u;
    unsigned long long k[8];
    uint32_t v[8], rank[8], dig[8];
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const int64_t i = base + it * 32 + lane;
        const bool ok = i < n;
        k[it] = ok ? kin[i] : 0ull;
        v[it] = ok ? vin[i] : 0u;
        const uint32_t d = ok ? ((uint32_t)(k[it] >> shift) & dmask) : 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = (d < 256u) ? whist[w][d] : 0u;
        __syncwarp();
        if (d < 256u && lane == __ffs(peers) - 1) whist[w][d] = before + __popc(peers);
        __syncwarp();
        rank[it] = before + __popc(peers & lt_mask);
        dig[it] = d;
    }
    __syncthreads();
    {
        // per digit: the warps' exclusive offsets within the digit, then an
        // exclusive scan of the digit totals over the block
        const int d = threadIdx.x;
        uint32_t run = 0;
#pragma unroll
        for (int w2 = 0; w2 < 8; ++w2) {
            const uint32_t c = whist[w2][d];
            whist[w2][d] = run;
            run += c;
        }
        uint32_t x = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        uint32_t wp = 0;
        for (int w2 = 0; w2 < w; ++w2) wp += wsum[w2];
        loff[d] = wp + x - run;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < 8; ++it) {
        const uint32_t d = dig[it];
        if (d < 256u) {
            const uint32_t lp = loff[d] + whist[w][d] + rank[it];
            sk[lp] = k[it];
            sv[lp] = v[it];
        }
    }
    __syncthreads();
    // the valid pairs are a prefix of the block's chunk
    const int64_t rem = (int64_t)n - block0;
    const int cnt = rem <= 0 ? 0 : (rem < SORT_ITEMS ? (int)rem : SORT_ITEMS);
    for (int j = threadIdx.x; j < cnt; j += 256) {
        const unsigned long long key = sk[j];
        const uint32_t d = (uint32_t)(key >> shift) & dmask;
        const uint32_t dst = goff[d] + ((uint32_t)j - loff[d]);
        kout[dst] = key;
        vout[dst] = sv[j];
    }
}

// Per-tile [start, end) by boundary detection on the sorted tile ids.
__global__ void __launch_bounds__(256)
    ranges_kernel(const uint32_t* __restrict__ keys, const WsHeader* __restrict__ hdr,
                  const SortState* __restrict__ st, uint2* __restrict__ ranges) {
    pdl_begin();
    const uint32_t n = st->abort ? 0u : hdr->n_instances;
    // four tile ids per thread (the region is aligned to 256 bytes), and the
    // one before them
    for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 4; i < n;
         i += (int64_t)gridDim.x * blockDim.x * 4) {
        uint32_t t[5];
        t[0] = i ? keys[i - 1] : 0xffffffffu;
        if (i + 4 <= n) {
            const uint4 q = *reinterpret_cast<const uint4*>(keys + i);
            t[1] = q.x; t[2] = q.y; t[3] = q.z; t[4] = q.w;
        } else {
            for (int j = 0; j < 4; ++j) t[j + 1] = i + j < n ? keys[i + j] : 0u;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (i + j >= n) break;
            if (i + j == 0 || t[j] != t[j + 1]) {
                ranges[t[j + 1]].x = (uint32_t)(i + j);
                if (i + j) ranges[t[j]].y = (uint32_t)(i + j);
            }
            if (i + j == n - 1) ranges[t[j + 1]].y = n;
        }
    }
}

// Tile schedule of the persistent composite kernels: global tile ids ordered
// by descending list length, bucketed by floor(log2(length)) (one block;
// the order inside a bucket is arbitrary and affects scheduling only).
__global__ void __launch_bounds__(1024)
    tile_order_kernel(const uint2* __restrict__ ranges, int64_t n_tiles, uint32_t* __restrict__ order) {
    pdl_begin();
    __shared__ uint32_t cnt[33];
    __shared__ uint32_t base[33];
    if (threadIdx.x < 33) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const uint2 r = ranges[t];
        atomicAdd(&cnt[__clz(r.y - r.x)], 1u);  // longer lists -> fewer leading zeros
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int b = 0; b < 33; ++b) {
            base[b] = run;
            run += cnt[b];
        }
    }
    __syncthreads();
    for (int64_t t = threadIdx.x; t < n_tiles; t += blockDim.x) {
        const uint2 r = ranges[t];
        order[atomicAdd(&base[__clz(r.y - r.x)], 1u)] = (uint32_t)t;
    }
}

int radix_pass(const unsigned long long* kin, const uint32_t* vin, unsigned long long* kout,
               uint32_t* vout, uint32_t* hist, uint32_t* scan_tmp, const WsHeader* hdr,
               int shift, uint32_t dmask, int nb, cudaStream_t st) {
    radix_hist_kernel<<<nb, 256, 0, st>>>(kin, hdr, shift, dmask, nb, hist);
    int launches = 1 + scan_u32(hist, (int64_t)nb * 256, scan_tmp, hist, nullptr, st);
    radix_scatter_kernel<<<nb, 256, 0, st>>>(kin, vin, kout, vout, hist, hdr, shift, dmask, nb);
    return launches + 1;
}

template <int PER, bool FROM_PAIRS, bool KEYS>
static void launch_onesweep(const OnesweepParams& P, int64_t n_max, cudaStream_t st) {
    constexpr int ITEMS = RS_THREADS * PER;
    const int smem = (int)sizeof(OnesweepSmem<PER>);
    ensure_smem_limit(reinterpret_cast<const void*>(&onesweep_kernel<PER, FROM_PAIRS, KEYS>), smem);
    const int64_t chunks = (n_max + ITEMS - 1) / ITEMS, cap = (int64_t)sm_count() * 2;
    launch_after(&onesweep_kernel<PER, FROM_PAIRS, KEYS>, chunks < cap ? chunks : cap, RS_THREADS,
                 (size_t)smem, st, P);
}

template <bool FROM_PAIRS, bool KEYS>
static void launch_onesweep_n(const OnesweepParams& P, int64_t n_max, cudaStream_t st) {
    if (rs_per(n_max) == RS_PER_LARGE)
        launch_onesweep<RS_PER_LARGE, FROM_PAIRS, KEYS>(P, n_max, st);
    else
        launch_onesweep<RS_PER_SMALL, FROM_PAIRS, KEYS>(P, n_max, st);
}

int launch_bin_sort(const unigs_plan& p, void* ws, cudaStream_t st) {
    const int64_t total = p.n * (int64_t)p.n_cams;
    WsHeader* hdr = ws_ptr<WsHeader>(ws, p, OFF_HDR);
    uint2* ranges = ws_ptr<uint2>(ws, p, OFF_RANGES);
    if (total == 0 || p.capacity == 0) {
        // no instances: every tile is empty, the schedule is still needed
        cudaMemsetAsync(ranges, 0, sizeof(uint2) * (size_t)p.n_tiles, st);
        tile_order_kernel<<<1, 1024, 0, st>>>(ranges, p.n_tiles, ws_ptr<uint32_t>(ws, p, OFF_ORDER));
        return 1;
    }
    int launches = 0;
    const uint32_t* touched = ws_ptr<uint32_t>(ws, p, OFF_TOUCH);
    const uint32_t* zbits = ws_ptr<uint32_t>(ws, p, OFF_ZBITS);
    SortState* ss = ws_ptr<SortState>(ws, p, OFF_SCAN);
    unsigned long long* words = ws_ptr<unsigned long long>(ws, p, OFF_HIST);
    // The depth sort's buffers, dead once the instances are emitted, lie in
    // the gradient-record region, which only the backward uses.
    const int64_t pad = (total + 3) / 4 * 4;
    uint32_t* dz[2] = {ws_ptr<uint32_t>(ws, p, OFF_GREC), ws_ptr<uint32_t>(ws, p, OFF_GREC) + 2 * pad};
    uint32_t* dt[2] = {dz[0] + pad, dz[1] + pad};
    unsigned long long* emit_words = reinterpret_cast<unsigned long long*>(dz[0] + 4 * pad);
    cudaMemsetAsync(ss, 0, sizeof(SortState), st);
    {
        const int64_t items = (int64_t)RS_THREADS * rs_per(total);
        // 8 pairs per thread: each block adds up to 1024 counts to the same
        // words at its end
        const int64_t blocks = (total + 4095) / 4096, cap = (int64_t)sm_count() * 4;
        depth_hist_kernel<<<(unsigned)(blocks < cap ? blocks : cap), 512, 0, st>>>(
            touched, zbits, total, ss, words, (total + items - 1) / items * 256, emit_words,
            (total + 255) / 256, ranges, p.n_tiles);
        ++launches;
    }
    OnesweepParams P = {};
    P.words = words;
    P.st = ss;
    P.hdr = hdr;
    for (int pass = 0; pass < DEPTH_PASSES; ++pass) {
        const int src = (pass & 1) ^ 1, dst = src ^ 1;
        P.kin = pass ? dz[src] : zbits;
        P.vin = pass ? dt[src] : touched;
        P.kout = dz[dst];
        P.vout = dt[dst];
        P.hist = ss->dhist[pass];
        P.ticket = &ss->ticket[pass];
        P.n_ptr = &ss->n_kept;
        P.n_host = total;
        P.shift = 8 * pass;
        P.bits = 8;
        P.epoch = 1u + pass;
        if (pass == 0)
            launch_onesweep_n<true, true>(P, total, st);
        else if (pass < DEPTH_PASSES - 1)
            launch_onesweep_n<false, true>(P, total, st);
        else
            launch_onesweep_n<false, false>(P, total, st);
        ++launches;
    }
    const int tpasses = tile_pass_count(p.n_tiles);
    const int tb = tpasses ? (tile_id_bits(p.n_tiles) + tpasses - 1) / tpasses : 0;
    uint32_t* keys[2] = {ws_ptr<uint32_t>(ws, p, OFF_KEYS0), ws_ptr<uint32_t>(ws, p, OFF_KEYS1)};
    uint32_t* vals[2] = {ws_ptr<uint32_t>(ws, p, OFF_VALS0), ws_ptr<uint32_t>(ws, p, OFF_VALS1)};
    // the last tile pass writes buffer 0
    int cur = tpasses & 1;
    {
        EmitParams E;
        E.tab = ws_ptr<CamTable>(ws, p, OFF_CAM);
        E.n = p.n;
        E.tw = p.cfg.tile_w;
        E.th = p.cfg.tile_h;
        E.capacity = p.capacity;
        E.rect = ws_ptr<uint2>(ws, p, OFF_RECT);
        E.touched = touched;
        E.masks = cull_masks(ws, p);
        E.cull = cull_records(ws, p);
        E.keep_bits = cull_bits(ws, p);
        E.order = dt[1];
        E.st = ss;
        E.hdr = hdr;
        E.emit_words = emit_words;
        E.big = reinterpret_cast<uint4*>(emit_words + (total + 511) / 512 * 2);
        E.words = words;
        E.keys = keys[cur];
        E.vals = vals[cur];
        E.passes = tpasses;
        E.bits = tb;
        E.items = RS_THREADS * rs_per(p.capacity);
        const int64_t blocks = (total + 255) / 256, cap = (int64_t)sm_count() * 8;
        launch_after(&emit_kernel, blocks < cap ? blocks : cap, 256, 0, st, E);
        int max_tiles = 0;
        for (int k = 0; k < p.n_cams; ++k) {
            const int nt = p.tile_offset[k + 1] - p.tile_offset[k];
            max_tiles = nt > max_tiles ? nt : max_tiles;
        }
        launches += 1;
        if (max_tiles > MASK_TILES) {
            launch_after(&emit_big_kernel, blocks * 8 < cap ? blocks * 8 : cap, 256, 0, st, E,
                         (max_tiles + BIG_SEG - 1) / BIG_SEG);
            ++launches;
        }
    }
    for (int pass = 0; pass < tpasses; ++pass) {
        P.kin = keys[cur];
        P.vin = vals[cur];
        P.kout = keys[cur ^ 1];
        P.vout = vals[cur ^ 1];
        P.hist = ss->thist[pass];
        P.ticket = &ss->ticket[TICKET_EMIT + 1 + pass];
        P.n_ptr = &hdr->n_instances;
        P.shift = tb * pass;
        P.bits = tb;
        P.epoch = 5u + pass;
        launch_onesweep_n<false, true>(P, p.capacity, st);
        ++launches;
        cur ^= 1;
    }
    {
        const int64_t blocks = (p.capacity + 1023) / 1024;
        const int grid = (int)(blocks < 152 * 16 ? blocks : 152 * 16);
        launch_after(&ranges_kernel, grid, 256, 0, st, keys[0], hdr, ss, ranges);
        ++launches;
    }
    launch_after(&tile_order_kernel, 1, 1024, 0, st, ranges, p.n_tiles,
                 ws_ptr<uint32_t>(ws, p, OFF_ORDER));
    return launches + 1;
}

}  // namespace unigs

// Internal definitions shared by the sm_103a kernels of libunigs.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "unigs.h"

namespace unigs {

constexpr int TILE = UNIGS_TILE;             // default tile side
constexpr int TILE_PIX = UNIGS_TILE_PIXELS;  // pixels of every tile shape

// ----------------------------------------------------------------------------
// Per-(camera, Gaussian) forward record written by the preprocess and staged
// into shared memory by the composite kernels (52 floats = 208 bytes, a
// multiple of 16 so a bulk copy can move it).  The fields every evaluated
// (pixel, Gaussian) pair reads (warp box test and alpha) fill the first three
// 16-byte words.
//   [0..3]  projected centre split as integer part + remainder (x_hi, y_hi,
//           x_lo, y_lo); m = hi + lo, hi an integer-valued float, |lo| <= 0.5
//   [4..6]  conic (A, B, C) of the inverse 2D covariance; for an
//           ill-conditioned splat (flag [10]) instead the conditional form
//           q = P (a + rho b)^2 + e b^2: (P, rho_hi, rho_lo)
//   [7]     opacity
//   [8..9]  half-extents (x, y) of the box holding every pixel where alpha
//           can reach alpha_min (with margin): a warp whose 8x4 pixel block
//           lies outside skips the Gaussian
//   [10]    1 when the splat is ill-conditioned (alpha evaluated in
//           double-float), else 0
//   [11]    -1 when the camera is inside the 1-sigma ellipsoid (|v_s| <= 1),
//           else +1
//   [12..20] M_c = S^-1 R^T R_cw (camera ray -> local scaled), row-major
//   [21..23] v_s = S^-1 R^T (C - mu)
//   [24..32] N_w = R S^-1 (scaled-local normal -> world), row-major
//   [33]    camera-frame z of the centre
//   [34..36] ill-conditioned splat: e, pivot (1: a = x, b = y; 0: a = y,
//           b = x), 0; else 0
//   [37]    k (gradient factor)
//   [38..40] RGB
//   [41..43] P1, [44..46] P2: v_s x d_s = dx P1 + dy P2 for the pixel offset
//           (dx, dy) from the projected centre (see pair_geometry), the
//           cancellation-free form of the cross product for Gaussians far
//           from the camera
//   [47]    3-sigma radius r of the binning recipe (pixels): the Gaussian is
//           drawn only where |dx| <= r and |dy| <= r
//   [48..49] (cos theta, sin theta): the principal axes e0 = (cos, sin),
//           e1 = (-sin, cos) of the 2D covariance, the frame in which the
//           backward records the covariance gradient
//   [50..51] half-extents along e0 and e1 of the ellipse holding every pixel
//           where alpha can reach alpha_min (with margin): with [8..9] the
//           two boxes of the warp-block skip test
// ----------------------------------------------------------------------------
enum {
    R_MXH = 0, R_MYH, R_MXL, R_MYL, R_CON = 4, R_OP = 7, R_EXTX = 8, R_EXTY = 9,
    R_FLAG = 10, R_SR = 11, R_MC = 12, R_VS = 21, R_NW = 24, R_Z = 33, R_CLO = 34,
    R_K = 37, R_RGB = 38, R_P1 = 41, R_P2 = 44, R_R3 = 47, R_EC = 48, R_ES = 49,
    R_E0 = 50, R_E1 = 51, REC_FLOATS = 52
};

// Pixel of thread tid inside its tile of width tw (8, 16, 32 or 64; 256
// pixels): the tile is a grid of 8x4 warp blocks, tw / 8 per row; warp w
// covers the block at ((w % (tw/8)) * 8, (w / (tw/8)) * 4), lanes row-major
// within the block.
__device__ __forceinline__ void tile_pixel(int tid, int tw, int* lx, int* ly) {
    const int w = tid >> 5, lane = tid & 31, wpr = tw >> 3;
    *lx = (w % wpr) * 8 + (lane & 7);
    *ly = (w / wpr) * 4 + (lane >> 3);
}

// Origin of warp w's 8x4 block inside a tile of width tw.
__device__ __forceinline__ void warp_block(int w, int tw, int* bx, int* by) {
    const int wpr = tw >> 3;
    *bx = (w % wpr) * 8;
    *by = (w / wpr) * 4;
}

// True when the Gaussian cannot reach alpha_min anywhere in the warp's block
// [bx0, bx0+7] x [by0, by0+3]: the block lies
// outside the axis-aligned box of the q <= qlim ellipse, or outside the box
// along the ellipse's principal axes (separating-axis test of the block's
// half-extents 3.5 x 1.5 projected on e0, e1), which for an elongated splat
// is far smaller.
__device__ __forceinline__ bool warp_block_misses(const float* __restrict__ rc, float bx0,
                                                  float by0) {
    const float mx = rc[R_MXH] + rc[R_MXL], my = rc[R_MYH] + rc[R_MYL];
    const float ex = rc[R_EXTX], ey = rc[R_EXTY];
    if ((bx0 + 7.f < mx - ex) || (bx0 > mx + ex) || (by0 + 3.f < my - ey) || (by0 > my + ey))
        return true;
    const float cx = bx0 + 3.5f - mx, cy = by0 + 1.5f - my;
    const float c = rc[R_EC], s = rc[R_ES];
    const float ac = fabsf(c), as = fabsf(s);
    return fabsf(fmaf(c, cx, s * cy)) > rc[R_E0] + fmaf(3.5f, ac, 1.5f * as) ||
           fabsf(fmaf(-s, cx, c * cy)) > rc[R_E1] + fmaf(3.5f, as, 1.5f * ac);
}

// warp_block_misses for up to 32 staged records at once: lane l tests record
// first + l and the warp gets the bit mask of the records that can reach its
// block.  The test is some 25 instructions and most of a tile's list misses a
// given block, so one pass over 16 records costs what one or two serial tests
// did.  Records are 52 words apart: each quarter-warp's 16-byte reads fall in
// distinct banks.  Against the serial test, one 1280x720 view of 1M Gaussians
// went from 2.45 to 1.92 ms and a forward + backward of 16 of them from 110.2
// to 92.5 ms.
__device__ __forceinline__ uint32_t warp_block_hits(const float (*recs)[REC_FLOATS], int first,
                                                    int count, int lane, float bx0, float by0) {
    const int j = first + lane;
    bool hit = false;
    if (j < count) hit = !warp_block_misses(&recs[j][0], bx0, by0);
    return __ballot_sync(0xffffffffu, hit);
}

// Conic eigenvalue ratio above which alpha is evaluated in double-float: the
// float32 quadratic form loses about log2(ratio) bits along the long axis.
constexpr float KAPPA_FF = 64.f;

// Per-(camera, Gaussian) intermediate gradient record (32 float64
// accumulators, 256 bytes), filled by atomics in the backward composite and
// consumed by the preprocess backward:
// dL/d(projected centre x, y), dL/d(a', b', c') of the 2D covariance
// E^T [[a, b], [b, c]] E = [[a', b'], [b', c']] in the splat's principal frame
// E (low-pass included; see the record's [48..49]), opacity, RGB, the local-frame matrix
// B = sum g_vs (x) v_s + g_ds (x) d_s (row-major, accumulated as
// g_vs (x) w + (g_ds - t g_vs) (x) d_s, see the backward composite), v_s, N_w,
// k and the centre depth (centre-depth mode).
enum {
    G_MX = 0, G_MY, G_CA, G_CB, G_CC, G_OP, G_RGB, G_B = 9, G_VS = 18,
    G_NW = 21, G_K = 30, G_Z = 31, GREC_FLOATS = 32
};

// Camera as the kernels see it (read from the workspace).
struct DevCam {
    int32_t width, height, tiles_x, tiles_y;
    int64_t tile_off, pix_off;
    float fx, fy, cx, cy;
    float R_wc[9];
    float t_wc[3];
    float R_cw[9];
    float C[3];
    float z_near;
    int32_t tile_w, tile_h;  // tile shape of the plan (the same for every camera)
    float pad;
};
static_assert(sizeof(DevCam) == 160, "DevCam layout");

struct CamTable {
    DevCam cam[UNIGS_MAX_CAMS];
};

// Device status block at the start of the workspace.
struct WsHeader {
    uint32_t status;       // unigs_status of the first device-side error
    uint32_t n_instances;  // instances emitted (valid when not overflowed)
    unsigned long long need;  // instances required (capacity errors)
    unsigned long long n_eval;   // (pixel, Gaussian) pairs whose alpha the forward evaluated
    unsigned long long n_blend;  // pairs the forward blended (alpha >= alpha_min, not stopped)
    uint32_t work_fwd;           // tile counters of the persistent composite kernels
    uint32_t work_bwd;
    uint32_t nonfinite;          // first parameter array found non-finite (flag set)
    uint32_t n_kept;             // (camera, Gaussian) pairs with a kept tile (preprocess)
    uint32_t pad0;
    unsigned long long bit_words;  // words of the kept-tile bits in use (preprocess)
    uint32_t pad[48];
};
static_assert(sizeof(WsHeader) == 256, "WsHeader layout");

// Region indices into unigs_plan::off[].
enum {
    OFF_HDR = 0, OFF_CAM, OFF_REC, OFF_RECT, OFF_TOUCH, OFF_OFFS, OFF_ZBITS,
    OFF_SCAN, OFF_KEYS0, OFF_KEYS1, OFF_VALS0, OFF_VALS1, OFF_HIST, OFF_RANGES,
    OFF_GREC, OFF_CULL, OFF_SEM32, OFF_ORDER, OFF_LOSS, OFF_VP, OFF_END
};
static_assert(OFF_END <= 20, "unigs_plan::off holds 20 region offsets");

// Per-(camera, Gaussian) record of the opacity-aware tile test (8 floats):
// float32 projected centre, float32 conic (kA, kB, kC), qlim, no-cull flag,
// and the first word of the kept-tile bits (as bits; NO_BITS: none).
enum { C_MX = 0, C_MY, C_KA, C_KB, C_KC, C_QLIM, C_NOCULL, C_BITS, CULL_FLOATS = 8 };

// Opacity-aware tile test, float32 recipe with non-contractible operations
// (identical operation order in the oracle's binning): keep the tile when the
// minimum over its pixel-centre square of q(D) = D^T K D is <= qlim.
__device__ __forceinline__ float cull_q(float kA, float kB, float kC, float dx, float dy) {
    return __fadd_rn(__fadd_rn(__fmul_rn(__fmul_rn(kA, dx), dx),
                               __fmul_rn(__fmul_rn(__fmul_rn(2.f, kB), dx), dy)),
                     __fmul_rn(__fmul_rn(kC, dy), dy));
}

// The record's conic with correctly rounded reciprocals of its diagonal
// (0 where a reciprocal or a quotient by it could leave the normal range).
struct CullTest {
    float mx, my, kA, kB, kC, qlim, yA, yC;
    bool nocull;
};
__device__ __forceinline__ CullTest cull_test(const float* __restrict__ cr) {
    CullTest c = {cr[C_MX], cr[C_MY], cr[C_KA], cr[C_KB], cr[C_KC], cr[C_QLIM], 0.f, 0.f,
                  cr[C_NOCULL] != 0.f};
    constexpr float LO = 0x1p-60f, HI = 0x1p60f;
    if (c.kA >= LO && c.kA <= HI && c.kC >= LO && c.kC <= HI) {
        c.yA = __frcp_rn(c.kA);
        c.yC = __frcp_rn(c.kC);
    }
    return c;
}

// n / d rounded, y the correctly rounded 1 / d: the quotient n y corrected by
// its exact residual is the rounded quotient (Markstein 1990).  (For |n| below
// 2^-100 the residual may be inexact; such a step moves q by nothing.)  Three
// instructions, where the general division takes about twelve.
__device__ __forceinline__ float div_recip(float n, float d, float y) {
    const float q = __fmul_rn(n, y);
    return __fmaf_rn(__fmaf_rn(-d, q, n), y, q);
}

__device__ __forceinline__ bool tile_keep(const CullTest& c, int tx, int ty, int tw, int th) {
    if (c.nocull) return true;
    const float X0 = (float)(tx * tw), X1 = (float)(tx * tw + tw - 1);
    const float Y0 = (float)(ty * th), Y1 = (float)(ty * th + th - 1);
    if (X0 <= c.mx && c.mx <= X1 && Y0 <= c.my && c.my <= Y1) return 0.f <= c.qlim;
    const float ylo = __fsub_rn(Y0, c.my), yhi = __fsub_rn(Y1, c.my);
    const float xlo = __fsub_rn(X0, c.mx), xhi = __fsub_rn(X1, c.mx);
    const bool fast = c.yA != 0.f;
    float q[4];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float dx = e ? xhi : xlo;
        const float n = -__fmul_rn(c.kB, dx);
        const float d = fast ? div_recip(n, c.kC, c.yC) : __fdiv_rn(n, c.kC);
        q[e] = cull_q(c.kA, c.kB, c.kC, dx, fminf(fmaxf(d, ylo), yhi));
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float dy = e ? yhi : ylo;
        const float n = -__fmul_rn(c.kB, dy);
        const float d = fast ? div_recip(n, c.kA, c.yA) : __fdiv_rn(n, c.kA);
        q[2 + e] = cull_q(c.kA, c.kB, c.kC, fminf(fmaxf(d, xlo), xhi), dy);
    }
    return fminf(fminf(q[0], q[1]), fminf(q[2], q[3])) <= c.qlim;
}

constexpr int SCAN_ITEMS = 4096;   // elements per scan block (256 threads x 16)
constexpr int LOSS_MAX_BLOCKS = 2048;  // block partials of the loss reduction
// Rectangles of at most MASK_TILES tiles carry a bit mask of their kept tiles
// from the preprocess to the emission, those of at most WIDE_TILES one in the
// place of the test's record (8 words), larger ones a place in a common array
// of words (record [7], C_BITS) while it lasts: only rectangles that found it
// full are tested again.
constexpr int MASK_TILES = 64;
constexpr int WIDE_TILES = 32 * CULL_FLOATS;
constexpr int SORT_ITEMS = 2048;   // keys per block of the 64-bit pair sort (256 threads x 8)
// Blocks of the single-kernel radix passes: RS_THREADS threads (one per digit
// value at most) of RS_PER keys.
constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_BINS = 512;
constexpr int RS_PER_LARGE = 16, RS_PER_SMALL = 4;
// Keys per thread for an array of at most n keys: below about two full waves
// of large blocks (2 blocks of 8192 keys on each of 152 SMs) small blocks
// spread the keys over more SMs.
__host__ __device__ constexpr int rs_per(int64_t n) {
    return n >= 4 * 1000 * 1000 ? RS_PER_LARGE : RS_PER_SMALL;
}
constexpr int DEPTH_PASSES = 4;     // 32 depth bits, 8 at a time
constexpr int TILE_PASSES_MAX = 4;  // ceil(31 tile bits / 9)
// Bits of a tile id, and the passes that sort by them (digits of at most 9 bits).
__host__ inline int tile_id_bits(int64_t n_tiles) {
    int bits = 0;
    while (((int64_t)1 << bits) < n_tiles) ++bits;
    return bits;
}
__host__ inline int tile_pass_count(int64_t n_tiles) { return (tile_id_bits(n_tiles) + 8) / 9; }
constexpr int TICKET_EMIT = 4;      // tickets 0..3: depth passes, then emission, tile passes

// State of one binning, zeroed at its start.
struct SortState {
    uint32_t ticket[TICKET_EMIT + 1 + TILE_PASSES_MAX + 3];
    uint32_t n_kept;                 // pairs with a kept tile
    uint32_t n_big;                  // kept pairs of more than MASK_TILES tiles
    uint32_t abort;                  // a bounded wait gave up
    uint32_t pad;
    uint32_t dhist[4][256];          // depth digits of the kept pairs
    uint32_t thist[TILE_PASSES_MAX][RS_BINS];  // tile digits of the instances
};
template <typename T>
__host__ __device__ inline T* ws_ptr(void* ws, const unigs_plan& p, int region) {
    return reinterpret_cast<T*>(static_cast<char*>(ws) + p.off[region]);
}

// The tile-test region: a kept-tile mask per pair, then a test record per pair.
__host__ inline unsigned long long* cull_masks(void* ws, const unigs_plan& p) {
    return ws_ptr<unsigned long long>(ws, p, OFF_CULL);
}
__host__ inline float* cull_records(void* ws, const unigs_plan& p) {
    const size_t total = (size_t)p.n * (size_t)p.n_cams;
    return reinterpret_cast<float*>(cull_masks(ws, p) + (total + 1) / 2 * 2);
}

// Words of kept-tile bits: 4 bits per instance of the capacity (a rectangle's
// tiles are a few times its kept ones).
constexpr uint32_t NO_BITS = 0xffffffffu;
__host__ inline int64_t bit_word_count(int64_t capacity) { return capacity / 8 + 1024; }
__host__ inline uint32_t* cull_bits(void* ws, const unigs_plan& p) {
    const size_t total = (size_t)p.n * (size_t)p.n_cams;
    return reinterpret_cast<uint32_t*>(cull_records(ws, p) + total * CULL_FLOATS);
}

__device__ inline const DevCam& cam_of_tile(const CamTable* tab, int n_cams, int64_t gtile,
                                            int* cam_index) {
    int lo = 0;
    for (int k = 1; k < n_cams; ++k)
        if (gtile >= tab->cam[k].tile_off) lo = k;
    *cam_index = lo;
    return tab->cam[lo];
}

__device__ inline void set_status(WsHeader* h, uint32_t code) {
    atomicCAS(&h->status, 0u, code);
}

// Feature loads (float32 or bfloat16 storage, float32 math).
__device__ __forceinline__ float load_feat(const void* base, size_t i, int bf16) {
    if (bf16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[i]);
    return reinterpret_cast<const float*>(base)[i];
}

// N consecutive features from element i0 on, N and i0 multiples of 4 and base
// 16-byte aligned: 16 (float32) or 8 (bfloat16) bytes a load.
template <int N>
__device__ __forceinline__ void load_feats(const void* base, size_t i0, int bf16, float (&h)[N]) {
    static_assert(N % 4 == 0, "whole vectors");
    if (bf16) {
        const uint2* src = reinterpret_cast<const uint2*>(
            reinterpret_cast<const __nv_bfloat16*>(base) + i0);
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const uint2 v = src[q];
            h[4 * q] = __uint_as_float(v.x << 16);
            h[4 * q + 1] = __uint_as_float(v.x & 0xffff0000u);
            h[4 * q + 2] = __uint_as_float(v.y << 16);
            h[4 * q + 3] = __uint_as_float(v.y & 0xffff0000u);
        }
    } else {
        const float4* src = reinterpret_cast<const float4*>(
            reinterpret_cast<const float*>(base) + i0);
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float4 v = src[q];
            h[4 * q] = v.x;
            h[4 * q + 1] = v.y;
            h[4 * q + 2] = v.z;
            h[4 * q + 3] = v.w;
        }
    }
}

// ----------------------------------------------------------------------------
// mbarrier + bulk-copy (TMA engine, non-tensor) helpers, inline PTX.
// ----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// Adds to the expected transaction bytes of the current phase (no arrival).
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// One arrival (release semantics: this thread's earlier writes are visible to
// a thread whose wait observes the phase).
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Returns true once the phase with the given parity has completed.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// True when the phase with the given parity has completed; does not wait.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after max_iter polls and reports false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  uint32_t max_iter) {
    for (uint32_t i = 0; i < max_iter; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Before a CTA exits: waits (bounded) until the last bulk copy issued into
// each of the two staging buffers has landed in shared memory.  issued0/1
// count the phases started on bar[0]/bar[1]; phases complete in order and the
// producers keep at most one in flight per buffer, so the parity of the last
// one identifies it.  In a launch without timeouts every phase has already
// been waited for and this returns at once.  Returns false if a copy is still
// in flight after the limit (the caller has already recorded the timeout).
__device__ __forceinline__ bool drain_bulk(uint64_t* bar, uint32_t issued0, uint32_t issued1,
                                           uint32_t limit) {
    bool ok = true;
    if (issued0 > 0) ok &= mbar_wait_bounded(&bar[0], (issued0 - 1) & 1u, limit);
    if (issued1 > 0) ok &= mbar_wait_bounded(&bar[1], (issued1 - 1) & 1u, limit);
    return ok;
}

// 1D bulk copy global -> shared, completion counted on the mbarrier.
// dst, src 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// ----------------------------------------------------------------------------
// Warp transpose-reduction: every lane holds v[32]; afterwards lane L holds
// the warp-wide sum of element L (recursive halving, 31 shuffles).  The adds
// of neighbouring elements are issued as packed float32 pairs; each element
// still sees the same additions in the same order.
// ----------------------------------------------------------------------------
__device__ __forceinline__ float warp_reduce_transpose32(float (&v)[32], int lane) {
#pragma unroll
    for (int step = 0; step < 4; ++step) {
        const int off = 16 >> step;
        const int half = 16 >> step;  // current length is 2*half
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < half; k += 2) {
            const float2 lo = make_float2(v[k], v[k + 1]);
            const float2 hi = make_float2(v[k + half], v[k + half + 1]);
            const float2 send = upper ? lo : hi;
            const float2 keep = upper ? hi : lo;
            const float2 recv = make_float2(__shfl_xor_sync(0xffffffffu, send.x, off),
                                            __shfl_xor_sync(0xffffffffu, send.y, off));
            const float2 sum = __fadd2_rn(keep, recv);
            v[k] = sum.x;
            v[k + 1] = sum.y;
        }
    }
    const bool upper = (lane & 1) != 0;
    const float send = upper ? v[0] : v[1];
    const float keep = upper ? v[1] : v[0];
    return keep + __shfl_xor_sync(0xffffffffu, send, 1);
}

}  // namespace unigs

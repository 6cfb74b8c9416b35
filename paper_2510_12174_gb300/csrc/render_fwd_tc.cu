// Forward composite (Alg. 2) with the semantic blend of Eq. semantic_render
// on the 5th-generation tensor cores, for bfloat16 logit storage.
//
// Per tile and batch of B Gaussians the logit blend is a dense product:
// O[p][c] += sum_j W[p][j] F[j][c], with W[p][j] = alpha_j T_j at pixel p (0
// where Gaussian j is skipped, culled, or after the pixel's stop) and F the
// batch's logit rows.  Every other channel (RGB, depth, normal, k, T) and the
// per-pixel walk are those of the SIMT kernel (render_fwd.cu); only the 2C
// FMAs per blended pair move to the tensor core, which also frees the C
// per-pixel logit accumulators from the registers.
//
// Precision: F is exact in bfloat16 (the storage format).  W is split into
// bfloat16 hi + lo parts (w = hi + lo + r with |r| <= 2^-18 |w|), so two MMAs
// per K-step reproduce the float32 blend to ~4e-6 relative; products are exact
// and accumulate in float32 in tensor memory.
//
// Layout: the 256 pixels of the tile are two M = 128 tiles (pixel thread tid
// owns row tid, i.e. tensor-memory lane tid % 128 of M-tile tid / 128); the
// accumulators of the tile live in 2 NS float32 tensor-memory columns for the
// whole tile list.  Operands are K-major without swizzle (8 x 16-byte core
// matrices): each thread zeroes its W rows (both splits) and stores the two
// parts of each weight it blends.
//
// Warps 0-7 walk the pixels; warp 8 stages each batch (bulk copies of the
// records and logit rows), transposes the rows into F^T and issues the
// batch's 2 x 2 x (B/16) MMAs of 128 x NS x 16.  Per batch and buffer the
// handshake is: staged (bar) -> every pixel warp walked the batch and wrote
// its W rows (wrdy, 8 arrivals) -> MMAs done (mma_bar).  Buffers alternate, so
// a pixel warp with few Gaussians in its block runs up to a batch ahead of the
// slowest: with a barrier over the CTA after each batch of 16, 28% of a warp's
// time went into it.  A tile whose pixels are all opaque ends with an empty
// batch, which the staging warp sends once all 8 warps have reported.  At the
// end of the tile every pixel warp reads its 32 lanes back with tcgen05.ld and
// writes the logits.
#include "launch.h"
#include "splat.cuh"
#include "tcgen05.cuh"

#include <type_traits>

namespace unigs {

constexpr uint32_t TC_WAIT_LIMIT = 1u << 22;

struct FwdTcParams {
    const CamTable* tab;
    int n_cams;
    int n_sem;
    int64_t n;
    int64_t n_tiles;
    const float* rec;
    const void* sem;           // rows [n][n_sem]: bfloat16, or float32 (F32 kernels)
    const uint32_t* vals;
    const uint2* ranges;
    const uint32_t* order;
    uint32_t* work;
    WsHeader* hdr;
    unigs_outputs out;
    float alpha_min, alpha_max, T_min;
    int center_depth;
    int sem_bulk;
};

template <int NS, int B, bool F32>
struct FwdTcSmem {
    using SemT = typename std::conditional<F32, float, __nv_bfloat16>::type;
    static constexpr int SPLITS_F = F32 ? 2 : 1;  // float32 features: bfloat16 hi + lo
    static constexpr int SBO = 16 * B;            // bytes between 8-row core-matrix groups
    static constexpr int W_BYTES = 128 * B * 2;   // one split of one M-tile
    static constexpr int F_BYTES = NS * B * 2;
    __align__(128) unsigned char wa[2][2][2][W_BYTES];       // [buffer][split][M-tile]
    __align__(128) unsigned char fb[2][SPLITS_F][F_BYTES];   // [buffer][split] F^T, NS x B
    __align__(16) float rec[2][B][REC_FLOATS];
    __align__(16) SemT semb[2][B][NS];
    uint64_t bar[2];      // batch staged
    uint64_t wrdy[2];     // the 8 pixel warps are done with the batch (8 arrivals)
    uint64_t mma_bar[2];  // MMAs of the operand buffer complete
    int count[2];         // Gaussians of the staged batch; released by its arrival on bar
    int final[2];         // 1: the tile's last batch
    uint32_t done;        // pixel warps whose pixels are all opaque
    uint32_t tmem_base;
    int tile;
    uint32_t issued[2];   // staging phases started per buffer (the staging warp counts)
};

constexpr int FTC_THREADS = 288;

template <int NS>
__host__ __device__ constexpr uint32_t tmem_cols() {
    return 2 * NS < 32 ? 32u : (uint32_t)(2 * NS);
}

// Bounded wait that is skipped once this thread has given up.
__device__ __forceinline__ void ftc_wait(uint64_t* bar, uint32_t parity, bool& timed_out) {
    if (!timed_out && !mbar_wait_bounded(bar, parity, TC_WAIT_LIMIT)) timed_out = true;
}

// Starts the copies of a batch (count 0: an empty batch); the staging warp.
template <int NS, int B, bool F32>
__device__ __forceinline__ void ftc_stage(const FwdTcParams& P, FwdTcSmem<NS, B, F32>& S, int buf,
                                          uint32_t first, int count, bool last, int cam,
                                          uint32_t id) {
    using SemT = typename FwdTcSmem<NS, B, F32>::SemT;
    const int lane = threadIdx.x & 31;
    const uint32_t row_bytes = (uint32_t)(P.n_sem * sizeof(SemT));
    const uint32_t per = REC_FLOATS * 4 + (P.sem_bulk ? row_bytes : 0u);
    if (lane == 0 && count > 0) mbar_expect_tx(&S.bar[buf], per * (uint32_t)count);
    __syncwarp();
    for (int i = lane; i < count; i += 32) {
        // the first 32 indices were read a batch ahead
        const uint32_t g = i < 32 ? id : P.vals[first + i];
        const size_t r = (size_t)cam * (size_t)P.n + g;
        bulk_g2s(&S.rec[buf][i][0], P.rec + r * REC_FLOATS, REC_FLOATS * 4, &S.bar[buf]);
        const SemT* src = static_cast<const SemT*>(P.sem) + (size_t)g * P.n_sem;
        if (P.sem_bulk)
            bulk_g2s(&S.semb[buf][i][0], src, row_bytes, &S.bar[buf]);
        else
            for (int c = 0; c < P.n_sem; ++c) S.semb[buf][i][c] = src[c];
    }
    __syncwarp();
    if (lane == 0) {
        S.count[buf] = count;
        S.final[buf] = last ? 1 : 0;
        mbar_arrive(&S.bar[buf]);
        ++S.issued[buf];
    }
}

// F^T of the staged batch: channel c, Gaussians 8 jc .. 8 jc + 7 as one 16-byte
// core row (float32 features: the bfloat16 hi part and the bfloat16 rounding of
// the remainder, f = hi + lo + r with |r| <= 2^-18 |f|); the staging warp.
template <int NS, int B, bool F32>
__device__ __forceinline__ void ftc_transpose(FwdTcSmem<NS, B, F32>& S, int buf) {
    using Sm = FwdTcSmem<NS, B, F32>;
    for (int task = threadIdx.x & 31; task < NS * (B / 8); task += 32) {
        const int c = task % NS, jc = task / NS;
        const int off = (c >> 3) * Sm::SBO + jc * 128 + (c & 7) * 16;
        if (F32) {
            const float* col = reinterpret_cast<const float*>(&S.semb[buf][0][0]) + c;
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float f0 = col[(8 * jc + 2 * e) * NS];
                const float f1 = col[(8 * jc + 2 * e + 1) * NS];
                const __nv_bfloat16 h0 = __float2bfloat16_rn(f0);
                const __nv_bfloat16 h1 = __float2bfloat16_rn(f1);
                h[e] = (uint32_t)__bfloat16_as_ushort(h0) |
                       ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                l[e] = (uint32_t)__bfloat16_as_ushort(
                           __float2bfloat16_rn(f0 - __bfloat162float(h0))) |
                       ((uint32_t)__bfloat16_as_ushort(
                            __float2bfloat16_rn(f1 - __bfloat162float(h1)))
                        << 16);
            }
            *reinterpret_cast<uint4*>(&S.fb[buf][0][0] + off) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(&S.fb[buf][F32 ? 1 : 0][0] + off) =
                make_uint4(l[0], l[1], l[2], l[3]);
        } else {
            const unsigned short* col =
                reinterpret_cast<const unsigned short*>(&S.semb[buf][0][0]) + c;
            uint4 q;
            q.x = (uint32_t)col[(8 * jc + 0) * NS] | ((uint32_t)col[(8 * jc + 1) * NS] << 16);
            q.y = (uint32_t)col[(8 * jc + 2) * NS] | ((uint32_t)col[(8 * jc + 3) * NS] << 16);
            q.z = (uint32_t)col[(8 * jc + 4) * NS] | ((uint32_t)col[(8 * jc + 5) * NS] << 16);
            q.w = (uint32_t)col[(8 * jc + 6) * NS] | ((uint32_t)col[(8 * jc + 7) * NS] << 16);
            *reinterpret_cast<uint4*>(&S.fb[buf][0][0] + off) = q;
        }
    }
}

template <int NS, int B, bool F32>
// batch 16: 47 KB of shared memory and <= 56 registers, 4 CTAs per SM (4 x
// 128 accumulator columns fill the tensor memory); larger batches: 2
__global__ void __launch_bounds__(FTC_THREADS, (B <= 16 ? 4 : 2))
    render_fwd_tc_kernel(const FwdTcParams P) {
    using Sm = FwdTcSmem<NS, B, F32>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Sm& S = *reinterpret_cast<Sm*>(smem_raw);
    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const bool stager = warp == 8;
    constexpr uint32_t NCOLS = tmem_cols<NS>();
    constexpr uint32_t IDESC = idesc_bf16_f32(128, NS);

    // once per CTA: zero the staging (rows shorter than NS stay zero-padded),
    // init barriers, allocate the accumulator columns
    for (int j = tid; j < 2 * B * NS; j += FTC_THREADS)
        (&S.semb[0][0][0])[j] = typename Sm::SemT(0.f);
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&S.bar[b], 1);
            mbar_init(&S.wrdy[b], 8);
            mbar_init(&S.mma_bar[b], 1);
        }
        fence_mbar_init();
        S.issued[0] = S.issued[1] = 0u;
    }
    if (warp == 0) {
        tmem_alloc(&S.tmem_base, NCOLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = S.tmem_base;

    // Batches begun by this CTA: batch gk uses buffer gk & 1, and is phase
    // gk >> 1 of each of the buffer's barriers (every batch, empty ones too,
    // goes through all three).
    uint32_t gk = 0;
    uint32_t commits = 0;  // MMA commits (staging warp)
    bool timed_out = false;
    uint32_t n_eval = 0, n_blend = 0;
    const int ptid = tid & 255;
    const int mt = ptid >> 7, row = ptid & 127;
    const int wrow = (row >> 3) * Sm::SBO + (row & 7) * 16;

    for (;;) {
        if (tid == 0) {
            S.tile = (int)atomicAdd(P.work, 1u);
            S.done = 0u;
        }
        __syncthreads();
        const int64_t t = S.tile;
        if (t >= P.n_tiles) break;
        const int64_t gtile = P.order[t];
        int cam_idx;
        const DevCam& cam = cam_of_tile(P.tab, P.n_cams, gtile, &cam_idx);
        const uint2 range = P.ranges[gtile];
        const int n_items = (int)(range.y - range.x);
        const int n_batches = (n_items + B - 1) / B;

        if (stager) {
            // the MMAs of batch k, once every pixel warp has written its W rows:
            // per M-tile and K-step, W_hi F_hi and W_lo F_hi, plus W_hi F_lo for
            // float32 features (W_lo F_lo is below the float32 rounding of the
            // sum); nothing for an empty batch but the commit
            auto mma = [&](uint32_t k, bool first, bool empty) {
                const int bf = (int)(k & 1u);
                ftc_wait(&S.wrdy[bf], (k >> 1) & 1u, timed_out);
                if (__any_sync(0xffffffffu, timed_out)) {
                    timed_out = true;
                    return;
                }
                if (lane == 0) {
                    tc_fence_after_sync();
                    if (!empty)
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            const uint32_t d = tmem + (uint32_t)(m * NS);
#pragma unroll
                            for (int pr = 0; pr < (F32 ? 3 : 2); ++pr) {
                                const int sw = pr == 1 ? 1 : 0, sf = pr == 2 ? 1 : 0;
#pragma unroll
                                for (int s = 0; s < B / 16; ++s) {
                                    const uint64_t a = smem_desc_kmajor(
                                        &S.wa[bf][sw][m][0] + s * 256, 128, Sm::SBO);
                                    const uint64_t f = smem_desc_kmajor(
                                        &S.fb[bf][sf][0] + s * 256, 128, Sm::SBO);
                                    mma_bf16(d, a, f, IDESC,
                                             (!first || pr > 0 || s > 0) ? 1u : 0u);
                                }
                            }
                        }
                    mma_commit(&S.mma_bar[bf]);
                }
                ++commits;
            };
            bool stop = false, empty = false;
            constexpr int BL = B < 32 ? B : 32;
            // index of Gaussian `lane` of the next batch, read ahead
            uint32_t id = lane < BL && lane < n_items ? P.vals[range.x + lane] : 0u;
            for (int b = 0; b < n_batches; ++b, ++gk) {
                const int bf = (int)(gk & 1u);
                // the buffer's batch before last: its warps are done (waited for
                // by its MMAs), and its MMAs have read F^T
                if (gk >= 2) ftc_wait(&S.mma_bar[bf], ((gk >> 1) - 1) & 1u, timed_out);
                if (__any_sync(0xffffffffu, timed_out)) {
                    timed_out = true;
                    break;
                }
                empty = stop;
                const bool last = stop || b + 1 == n_batches;
                ftc_stage<NS, B, F32>(P, S, bf, range.x + (uint32_t)(b * B),
                                      empty ? 0 : min(B, n_items - b * B), last, cam_idx, id);
                {
                    const int nx = (b + 1) * B + lane;
                    if (lane < BL && nx < n_items) id = P.vals[range.x + (uint32_t)nx];
                }
                if (!empty) {
                    ftc_wait(&S.bar[bf], (gk >> 1) & 1u, timed_out);
                    if (__any_sync(0xffffffffu, timed_out)) {
                        timed_out = true;
                        break;
                    }
                    ftc_transpose<NS, B, F32>(S, bf);
                    fence_async_shared();
                    __syncwarp();
                }
                if (b > 0) {
                    mma(gk - 1u, b == 1, false);
                    if (timed_out) break;
                    stop = *(volatile uint32_t*)&S.done == 8u;
                }
                if (last) {
                    mma(gk, b == 0, empty);
                    ++gk;
                    break;
                }
            }
        } else {
            const int64_t ltile = gtile - cam.tile_off;
            const int tx = (int)(ltile % cam.tiles_x), ty = (int)(ltile / cam.tiles_x);
            int lx, ly;
            const int tw = cam.tile_w, th = cam.tile_h;
            tile_pixel(tid, tw, &lx, &ly);
            const int u = tx * tw + lx, v = ty * th + ly;
            // the warp's 8x4 pixel block, for the per-warp bounding-box skip
            int wbx, wby;
            warp_block(warp, tw, &wbx, &wby);
            const float bx0 = (float)(tx * tw + wbx);
            const float by0 = (float)(ty * th + wby);
            const bool inside = u < cam.width && v < cam.height;
            const float uf = (float)u, vf = (float)v;
            const float xt = (uf - cam.cx) / cam.fx, yt = (vf - cam.cy) / cam.fy;

            float T = 1.f;
            float crgb[3] = {0.f, 0.f, 0.f}, cdep = 0.f, cn[3] = {0.f, 0.f, 0.f}, ck = 0.f;
            uint32_t last = 0;
            bool done = !inside, reported = false;

            for (int b = 0; b < n_batches; ++b) {
                const int bf = (int)(gk & 1u);
                ftc_wait(&S.bar[bf], (gk >> 1) & 1u, timed_out);
                // W rows of this buffer were last read by the MMAs of batch gk - 2
                if (gk >= 2) ftc_wait(&S.mma_bar[bf], ((gk >> 1) - 1) & 1u, timed_out);
                if (__any_sync(0xffffffffu, timed_out)) {
                    timed_out = true;
                    break;
                }
                const int count = S.count[bf];
                const bool last_batch = S.final[bf] != 0;
                // this thread's W rows: zero, then the weights of the Gaussians it
                // blends (hi and lo bfloat16 parts)
                unsigned char* w0 = &S.wa[bf][0][mt][0] + wrow;
                unsigned char* w1 = &S.wa[bf][1][mt][0] + wrow;
#pragma unroll
                for (int jc = 0; jc < B / 8; ++jc) {
                    *reinterpret_cast<uint4*>(w0 + jc * 128) = make_uint4(0u, 0u, 0u, 0u);
                    *reinterpret_cast<uint4*>(w1 + jc * 128) = make_uint4(0u, 0u, 0u, 0u);
                }
                if (!__all_sync(0xffffffffu, done)) {
#pragma unroll 1
                    for (int j0 = 0; j0 < count; j0 += 32)
#pragma unroll 1
                    for (uint32_t hits = warp_block_hits(S.rec[bf], j0, count, lane, bx0, by0);
                         hits; hits &= hits - 1) {
                        const int j = j0 + __ffs(hits) - 1;
                        const float* rc = &S.rec[bf][j][0];
                        if (done) continue;
                        float dx, dy, Gs;
                        float wq;
                        const float alpha =
                            splat_alpha(rc, uf, vf, P.alpha_max, &dx, &dy, &Gs, &wq);
                        ++n_eval;
                        if (alpha < P.alpha_min) continue;
                        const float test_T = T * (1.f - alpha);
                        if (test_T < P.T_min) {
                            done = true;
                            continue;
                        }
                        ++n_blend;
                        const float w = alpha * T;
                        PairGeom G;
                        pair_geometry(rc, xt, yt, dx, dy, G);
                        const float depth = P.center_depth ? rc[R_Z] : G.t;
                        const float nsg = (G.inside ? -G.inv_m : G.inv_m) * w;
                        crgb[0] = fmaf(w, rc[R_RGB], crgb[0]);
                        crgb[1] = fmaf(w, rc[R_RGB + 1], crgb[1]);
                        crgb[2] = fmaf(w, rc[R_RGB + 2], crgb[2]);
                        cdep = fmaf(w, depth, cdep);
                        cn[0] = fmaf(nsg, G.m[0], cn[0]);
                        cn[1] = fmaf(nsg, G.m[1], cn[1]);
                        cn[2] = fmaf(nsg, G.m[2], cn[2]);
                        ck = fmaf(w, rc[R_K], ck);
                        T = test_T;
                        last = (uint32_t)(b * B + j + 1);
                        // w = hi + lo, both bfloat16
                        const __nv_bfloat16 wh = __float2bfloat16_rn(w);
                        const int off = (j >> 3) * 128 + (j & 7) * 2;
                        *reinterpret_cast<__nv_bfloat16*>(w0 + off) = wh;
                        *reinterpret_cast<__nv_bfloat16*>(w1 + off) =
                            __float2bfloat16_rn(w - __bfloat162float(wh));
                    }
                }
                const bool opaque = __all_sync(0xffffffffu, done);
                // this warp is done with the batch's records and W rows
                fence_async_shared();
                __syncwarp();
                if (lane == 0) {
                    if (opaque && !reported) atomicAdd(&S.done, 1u);
                    mbar_arrive(&S.wrdy[bf]);
                }
                reported = opaque;
                ++gk;
                if (last_batch) break;
            }
            // logits: the accumulators of this thread's row (zero without a
            // batch), once the tile's last MMAs are done (commits complete in order)
            if (n_batches > 0) ftc_wait(&S.mma_bar[(gk - 1u) & 1u], ((gk - 1u) >> 1) & 1u, timed_out);
            if (__any_sync(0xffffffffu, timed_out)) timed_out = true;
            tc_fence_after_sync();
            const int W = cam.width;
            const int64_t HW = (int64_t)cam.height * W;
            const int64_t pix = cam.pix_off;
            const int64_t idx = (int64_t)v * W + u;
            float* lo_out = P.out.logits + pix * (int64_t)P.n_sem + idx;
            const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
#pragma unroll
            for (int ch = 0; ch < NS / 16; ++ch) {
                float o[16];
                if (n_batches > 0) {
                    tmem_ld16(tmem + lane_base + (uint32_t)((warp >> 2) * NS + 16 * ch), o);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = 0.f;
                }
                if (inside)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (16 * ch + i < P.n_sem) lo_out[(int64_t)(16 * ch + i) * HW] = o[i];
            }
            tc_fence_before_sync();
            if (inside) {
                P.out.rgb[pix * 3 + 0 * HW + idx] = crgb[0];
                P.out.rgb[pix * 3 + 1 * HW + idx] = crgb[1];
                P.out.rgb[pix * 3 + 2 * HW + idx] = crgb[2];
                P.out.depth[pix + idx] = cdep;
                P.out.normal_g[pix * 3 + 0 * HW + idx] = cn[0];
                P.out.normal_g[pix * 3 + 1 * HW + idx] = cn[1];
                P.out.normal_g[pix * 3 + 2 * HW + idx] = cn[2];
                P.out.kmap[pix + idx] = ck;
                P.out.T_final[pix + idx] = T;
                P.out.n_contrib[pix + idx] = last;
            }
        }
        // a bounded wait that gave up ends the CTA (uniformly)
        if (__syncthreads_or(timed_out)) break;
        tc_fence_after_sync();
    }
    // Before the CTA exits: no bulk copy may still be landing in its shared
    // memory, and no MMA may still be reading its operands or writing its
    // tensor-memory columns (the staging warp waits, bounded, for the last
    // staging phase of each buffer and the last commit).  Then the columns are
    // returned: a CTA frees its tensor memory before it exits, also when a
    // wait gave up.
    if (stager) {
        if (lane == 0 && !drain_bulk(S.bar, S.issued[0], S.issued[1], TC_WAIT_LIMIT))
            timed_out = true;
        if (commits > 0 &&
            !mbar_wait_bounded(&S.mma_bar[(commits - 1u) & 1u], ((commits - 1u) >> 1) & 1u,
                               TC_WAIT_LIMIT))
            timed_out = true;
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tmem_dealloc(tmem, NCOLS);
    if (timed_out && (tid & 31) == 0) set_status(P.hdr, UNIGS_ERR_TIMEOUT);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_eval += __shfl_xor_sync(0xffffffffu, n_eval, o);
        n_blend += __shfl_xor_sync(0xffffffffu, n_blend, o);
    }
    if ((tid & 31) == 0 && n_eval) {
        atomicAdd(&P.hdr->n_eval, (unsigned long long)n_eval);
        atomicAdd(&P.hdr->n_blend, (unsigned long long)n_blend);
    }
}

template <int NS, int B, bool F32>
static void launch_fwd_tc_t(const FwdTcParams& P, int grid, cudaStream_t st) {
    const size_t smem = sizeof(FwdTcSmem<NS, B, F32>);
    // per device; a failure surfaces as the launch error the entry point returns
    ensure_smem_limit(reinterpret_cast<const void*>(&render_fwd_tc_kernel<NS, B, F32>), (int)smem);
    render_fwd_tc_kernel<NS, B, F32><<<grid, FTC_THREADS, smem, st>>>(P);
}

template <int B, bool F32>
static void launch_fwd_tc_b(const FwdTcParams& P, int grid, cudaStream_t st) {
    if (P.n_sem <= 16)
        launch_fwd_tc_t<16, B, F32>(P, grid, st);
    else if (P.n_sem <= 32)
        launch_fwd_tc_t<32, B, F32>(P, grid, st);
    else
        launch_fwd_tc_t<64, B, F32>(P, grid, st);
}

template <bool F32>
static void launch_fwd_tc_f(const FwdTcParams& P, int batch, int grid, cudaStream_t st) {
    switch (batch) {
        case 16: launch_fwd_tc_b<16, F32>(P, grid, st); break;
        case 64: launch_fwd_tc_b<64, F32>(P, grid, st); break;
        default: launch_fwd_tc_b<32, F32>(P, grid, st); break;
    }
}

static bool fwd_tc_plan(const unigs_plan& p) {
    return p.n_sem >= 9 && p.n_sem <= UNIGS_MAX_SEM && !(p.cfg.flags & UNIGS_FLAG_SIMT_LOGITS);
}

bool fwd_tc_eligible(const unigs_plan& p, const unigs_gaussians& g) {
    return fwd_tc_plan(p) && g.sem != nullptr;
}

bool sem32_needed(const unigs_plan& p) {
    if (!p.feat_dtype || p.n_sem <= 0 || p.n <= 0) return false;
    return !(fwd_tc_plan(p) && bwd_tc_selected(p));
}

int launch_render_fwd_tc(const unigs_plan& p, const unigs_gaussians& g, void* ws,
                         const unigs_outputs& out, cudaStream_t st) {
    if (p.n_tiles == 0) return 0;
    FwdTcParams P;
    P.tab = ws_ptr<CamTable>(ws, p, OFF_CAM);
    P.n_cams = p.n_cams;
    P.n_sem = p.n_sem;
    P.n = p.n;
    P.n_tiles = p.n_tiles;
    P.rec = ws_ptr<float>(ws, p, OFF_REC);
    P.sem = g.sem;
    P.vals = ws_ptr<uint32_t>(ws, p, OFF_VALS0);
    P.ranges = ws_ptr<uint2>(ws, p, OFF_RANGES);
    P.order = ws_ptr<uint32_t>(ws, p, OFF_ORDER);
    WsHeader* hdr = ws_ptr<WsHeader>(ws, p, OFF_HDR);
    P.work = &hdr->work_fwd;
    P.hdr = hdr;
    P.out = out;
    P.alpha_min = p.cfg.alpha_min;
    P.alpha_max = p.cfg.alpha_max;
    P.T_min = p.cfg.T_min;
    P.center_depth = (p.cfg.flags & UNIGS_FLAG_CENTER_DEPTH) ? 1 : 0;
    const int esz = p.feat_dtype ? 2 : 4;
    P.sem_bulk = ((p.n_sem * esz) % 16 == 0) && ((reinterpret_cast<uintptr_t>(P.sem) & 15) == 0);
    cudaMemsetAsync(P.work, 0, sizeof(uint32_t), st);
    // defaults: batch 16, 4 CTAs per SM; at most 4 CTAs per SM hold
    // accumulator columns at once (512 per SM)
    const int batch = p.cfg.batch_fwd > 0 ? p.cfg.batch_fwd : 16;
    int ctas = p.cfg.ctas_per_sm_fwd > 0 ? p.cfg.ctas_per_sm_fwd : 4;
    if (ctas > 4) ctas = 4;
    int64_t grid = (int64_t)sm_count() * ctas;
    if (grid > p.n_tiles) grid = p.n_tiles;
    if (p.feat_dtype)
        launch_fwd_tc_f<false>(P, batch, (int)grid, st);
    else
        launch_fwd_tc_f<true>(P, batch, (int)grid, st);
    return 1;
}

}  // namespace unigs

// Anchor attribute prediction (Sec. 3.1, Fig. 2 (a)): the MLPs that turn each
// anchor into its M Gaussians, forward and backward.  The definitions are in
// include/unigs_anchors.h.
//
// The five two-layer MLPs (F = H = 32) are about 11 k multiply-adds per anchor
// forward and 32 k backward, in float32; at 100k anchors of 10 Gaussians with
// 64 logits that is 30 and 90 us of the FP32 pipes, next to 35 and 70 us for
// the bytes.  Each layer is a product of a weight matrix with a tile of 128 (or
// 64, 32) anchors: a block keeps the weights, the anchors' features and one
// branch's hidden layer in shared memory (entries [unit][anchor]), and a
// thread owns a register tile of 4 units x 2 anchors.  Outputs and upstream
// gradients go through shared memory, so that consecutive threads read and
// write whole rows.  At that size decode takes 196 us and backward 530 us (913
// and 1780 with one thread per anchor, whose stores fell into 32 rows a warp;
// 236 and 941 with 8 warps of 4 x 4 tiles and global loads beside the
// products).  What bounds them now: shared-memory operand reads (55% of peak in
// decode, 45% in backward) and the latency between the phases of a tile.
//
// Backward: the same tiles give the outputs, dL/dh = W2^T g_y and dL/df = W1^T
// g_pre; the parameter gradients dL/dW2 = sum_a g_y (x) h and dL/dW1 = sum_a
// g_pre (x) f are register tiles over the block's anchors, added to
// accumulators in shared memory tile by tile, then over a cluster of blocks in
// float64; one float32 atomic per parameter and cluster adds them at the end.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "launch.h"
#include "unigs_anchors.h"
#include "unigs_internal.cuh"

namespace unigs {
namespace {

namespace cg = cooperative_groups;

constexpr int AF = UNIGS_ANCHOR_FEAT;
constexpr int AH = UNIGS_ANCHOR_HIDDEN;
constexpr int NMLP = 5;  // sem, k, opacity, color, cov
constexpr float Y00 = 0.28209479177387814f;  // 1 / (2 sqrt(pi))
// Row stride (floats) of the weight matrices in shared memory.  No padding:
// the 8 lanes of a shared-memory phase read the same row.
constexpr int WS = AH;
static_assert(WS == AH && AH == 32 && AF == 32, "the register tiles cover 32 hidden units");

// Each MLP's parameters in the shared-memory block (offsets in floats; rows
// of W1 and W2 are WS apart), its output count and its stored rows of W2: a
// multiple of 4, the surplus zero.  The covariance branch stores the scale
// outputs (row 3 m + i) first, then from row quat_row() the quaternions'
// (row quat_row() + 4 m + j).
struct WLayout {
    int w1[NMLP], b1[NMLP], w2[NMLP], b2[NMLP], out[NMLP], rows[NMLP];
    int total;
};

struct AnchorIn {
    int64_t n;
    int M, C;
    const float *pos, *scale, *offsets, *feat, *sem, *kfac;
    const float* w1[NMLP];
    const float* b1[NMLP];
    const float* w2[NMLP];
    const float* b2[NMLP];
};

struct DecodeOut {
    float *mean, *quat, *scale, *opacity, *kfac;
    void *sh, *sem;
};

// i / d for 0 <= i < 2^16, 1 <= d <= 192, inv = 1.f / d: the product of the two
// rounded factors is (i + 1/2) / d to a relative 2^-22, so at most 2^-6 / d off,
// where the exact value is at least 1 / (2 d) from an integer.  Three
// instructions against some twenty for a division by a runtime integer, one or
// two of which stood beside every output.
struct FastDiv {
    int d;
    float inv;
    __device__ __forceinline__ explicit FastDiv(int d_) : d(d_), inv(1.f / (float)d_) {}
    __device__ __forceinline__ int div(int i) const { return (int)(((float)i + 0.5f) * inv); }
    // i / d, and *rem = i % d
    __device__ __forceinline__ int divmod(int i, int* rem) const {
        const int q = div(i);
        *rem = i - q * d;
        return q;
    }
};

__device__ __forceinline__ float sigm(float y) { return 1.f / (1.f + expf(-y)); }

__device__ __forceinline__ void put_feat(void* base, int64_t i, float v, bool bf16) {
    if (bf16)
        static_cast<__nv_bfloat16*>(base)[i] = __float2bfloat16_rn(v);
    else
        static_cast<float*>(base)[i] = v;
}

__host__ __device__ __forceinline__ int quat_row(int M) { return (3 * M + 3) & ~3; }

// Row of W2 and b2 that branch X stores as row j; -1: a row of zeros.
__device__ __forceinline__ int param_row(int X, int out, int j, int M) {
    if (X != 4) return j < out ? j : -1;
    if (j < 3 * M) return 7 * (j / 3) + j % 3;
    j -= quat_row(M);
    return j < 0 ? -1 : 7 * (j / 4) + 3 + j % 4;
}

// Asynchronous copy of 4 or 16 bytes, global to shared.
template <int BYTES>
__device__ __forceinline__ void cp_async(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "n"(BYTES)
                 : "memory");
}
// Four floats; src 16-byte aligned where vec.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool vec) {
    if (vec) {
        cp_async<16>(dst, src);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) cp_async<4>(dst + e, src + e);
    }
}

// Copies every MLP's parameters into shared memory (the whole block), every
// copy in flight at once: one element per load and store, the 45 KB took
// most of the 41 us of a decode of a few hundred anchors.  Returns when this
// thread's copies have landed.
template <int NT>
__device__ void load_weights(const AnchorIn& P, const WLayout& L, float* sw) {
    for (int X = 0; X < NMLP; ++X) {
        const int out = L.out[X];
        if (out == 0) continue;
        const bool vec = ((reinterpret_cast<uintptr_t>(P.w1[X]) |
                           reinterpret_cast<uintptr_t>(P.w2[X])) & 15) == 0;
        for (int i = threadIdx.x; i < AH * AF / 4; i += NT)
            cp_async4(sw + L.w1[X] + 4 * i, P.w1[X] + 4 * i, vec);
        for (int i = threadIdx.x; i < AH; i += NT) cp_async<4>(sw + L.b1[X] + i, P.b1[X] + i);
        for (int i = threadIdx.x; i < L.rows[X] * (AH / 4); i += NT) {
            const int j = i / (AH / 4), src = param_row(X, out, j, P.M);
            float* dst = sw + L.w2[X] + 4 * i;
            if (src >= 0)
                cp_async4(dst, P.w2[X] + src * AH + 4 * (i % (AH / 4)), vec);
            else
                *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int j = threadIdx.x; j < L.rows[X]; j += NT) {
            const int src = param_row(X, out, j, P.M);
            if (src >= 0)
                cp_async<4>(sw + L.b2[X] + j, P.b2[X] + src);
            else
                sw[L.b2[X] + j] = 0.f;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// A tile of TA anchors worked on by NT threads: arrays are [row][anchor], rows
// S floats apart (16-byte aligned, and neighbouring rows start 4 banks apart).
// Thread tid owns anchors a0 .. a0 + RA - 1 of a group of 4 rows, GROUPS row
// groups at a time; a warp covers 8 anchor groups x 4 row groups.
template <int RA_, int NT_>
struct Tile {
    static constexpr int RA = RA_, NT = NT_;
    static constexpr int GROUPS = 8;
    static constexpr int TA = NT / GROUPS * RA, S = TA + 4;
    static constexpr int AW = NT / GROUPS / 8;  // warps along the anchors
    __device__ static __forceinline__ int anchor(int tid) {
        return ((tid & 7) + 8 * ((tid >> 5) % AW)) * RA;
    }
    __device__ static __forceinline__ int group(int tid) {
        return ((tid >> 3) & 3) + 4 * ((tid >> 5) / AW);
    }
};

template <int RA>
__device__ __forceinline__ void ld_anchors(const float* p, float (&v)[RA]) {
    if constexpr (RA == 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else if constexpr (RA == 2) {
        const float2 q = *reinterpret_cast<const float2*>(p);
        v[0] = q.x; v[1] = q.y;
    } else {
        v[0] = *p;
    }
}
template <int RA>
__device__ __forceinline__ void st_anchors(float* p, const float (&v)[RA]) {
    if constexpr (RA == 4)
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (RA == 2)
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else
        *p = v[0];
}

// acc[r][a] = b[r] + sum_k w[r][k] x[k][a] over 32 inputs k in order, for 4
// rows of weights (WS apart) and RA anchors of the tile x.
template <int RA, int S>
__device__ __forceinline__ void tile_rows(const float* w, const float* b, const float* x,
                                          float (&acc)[4][RA]) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int a = 0; a < RA; ++a) acc[r][a] = b[r];
#pragma unroll 2
    for (int k = 0; k < 32; k += 4) {
        float wv[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 q = *reinterpret_cast<const float4*>(w + r * WS + k);
            wv[r][0] = q.x; wv[r][1] = q.y; wv[r][2] = q.z; wv[r][3] = q.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float xv[RA];
            ld_anchors<RA>(x + (k + e) * S, xv);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int a = 0; a < RA; ++a) acc[r][a] = fmaf(wv[r][e], xv[a], acc[r][a]);
        }
    }
}

// acc[c][a] += sum_j w[j][c] x[j][a] over n rows j in order, for 4 columns of
// the weights.
template <int RA, int S>
__device__ __forceinline__ void tile_cols(const float* w, const float* x, int n,
                                          float (&acc)[4][RA]) {
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const float4 q = *reinterpret_cast<const float4*>(w + j * WS);
        const float wv[4] = {q.x, q.y, q.z, q.w};
        float xv[RA];
        ld_anchors<RA>(x + j * S, xv);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int a = 0; a < RA; ++a) acc[c][a] = fmaf(wv[c], xv[a], acc[c][a]);
    }
}

// Features of the tile's anchors, transposed (zero past the last anchor).
template <typename T>
__device__ __forceinline__ void load_feat(const AnchorIn& P, int64_t base, int rows, float* ft) {
    for (int i = threadIdx.x; i < T::TA * (AF / 4); i += T::NT) {
        const int a = i / (AF / 4), q = i % (AF / 4);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a < rows) v = reinterpret_cast<const float4*>(P.feat + (base + a) * AF)[q];
        float* dst = ft + 4 * q * T::S + a;
        dst[0] = v.x;
        dst[T::S] = v.y;
        dst[2 * T::S] = v.z;
        dst[3 * T::S] = v.w;
    }
}

// h = relu(W1 f + b1) of branch X for the tile.
template <typename T>
__device__ __forceinline__ void hidden_layer(const float* sw, const WLayout& L, int X,
                                             const float* ft, float* h) {
    constexpr int RA = T::RA;
    const int a0 = T::anchor(threadIdx.x), k0 = 4 * T::group(threadIdx.x);
    float acc[4][RA];
    tile_rows<RA, T::S>(sw + L.w1[X] + k0 * WS, sw + L.b1[X] + k0, ft + a0, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int a = 0; a < RA; ++a) acc[r][a] = fmaxf(acc[r][a], 0.f);
        st_anchors<RA>(h + (k0 + r) * T::S + a0, acc[r]);
    }
}

// Rows of the output buffer: the widest branch, padded.
__host__ __device__ inline int out_rows(const WLayout& L) {
    int m = 0;
    for (int X = 0; X < NMLP; ++X) m = L.rows[X] > m ? L.rows[X] : m;
    return m;
}

template <typename T>
__host__ __device__ inline size_t decode_floats(const WLayout& L, int M) {
    // the logits' rows are kept [anchor][channel]; the covariance branch's
    // scales and quaternions take turns
    const int sem = T::TA * (L.rows[0] + 4), y = 4 * M * T::S;
    return (size_t)L.total + 2 * 32 * T::S + (sem > y ? sem : y);
}

template <typename T>
__global__ void __launch_bounds__(T::NT) anchor_decode_kernel(const AnchorIn P, const WLayout L,
                                                              const DecodeOut O, int bf16) {
    constexpr int S = T::S, RA = T::RA, NT = T::NT, GROUPS = T::GROUPS;
    extern __shared__ __align__(16) float sw[];
    float* ft = sw + L.total;  // [AF][S] features
    float* h = ft + AF * S;    // [AH][S] hidden layer of one branch
    float* y = h + AH * S;     // [rows][S] outputs of one branch
    load_weights<NT>(P, L, sw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = P.M, C = P.C;
    const FastDiv byM(M), by3M(3 * M);
    const int64_t N = P.n * M;
    const bool fb = bf16 != 0;
    const int a0 = T::anchor(tid), g0 = T::group(tid);
    // whole 16-byte chunks of a Gaussian's logit row
    const int cstr = L.rows[0] + 4;
    const int row_bytes = C * (fb ? 2 : 4);
    const bool vec = row_bytes % 16 == 0 && (reinterpret_cast<uintptr_t>(O.sem) & 15) == 0;
    for (int64_t base = blockIdx.x * (int64_t)T::TA; base < P.n;
         base += (int64_t)gridDim.x * T::TA) {
        const int rows = (int)min((int64_t)T::TA, P.n - base);
        const int kids = rows * M;      // Gaussians of the tile
        const int64_t gb = base * M;    // the first of them
        __syncthreads();
        load_feat<T>(P, base, rows, ft);
        __syncthreads();
#pragma unroll 1
        for (int step = 0; step <= NMLP; ++step) {
            const int X = step < NMLP ? step : NMLP - 1;
            if (L.out[X] == 0) continue;  // no semantic branch without logits
            if (step != 5) {
                hidden_layer<T>(sw, L, X, ft, h);
                __syncthreads();
            }
            // the quaternions (step 5) follow the scales in the same branch
            const int jb = step == 5 ? quat_row(M) : 0;
            const int je = step == 4 ? quat_row(M) : L.rows[X];
#pragma unroll 1
            for (int j0 = jb + 4 * g0; j0 < je; j0 += 4 * GROUPS) {
                float acc[4][RA];
                tile_rows<RA, S>(sw + L.w2[X] + j0 * WS, sw + L.b2[X] + j0, h + a0, acc);
                if (X == 0) {
                    // semantic logits: o_ah (x) sigma(MLP_sem(f)), the same for every child
#pragma unroll
                    for (int a = 0; a < RA; ++a)
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            if (a0 + a < rows && j0 + r < C)
                                y[(a0 + a) * cstr + j0 + r] =
                                    P.sem[(base + a0 + a) * C + j0 + r] * sigm(acc[r][a]);
                } else {
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        st_anchors<RA>(y + (j0 - jb + r) * S + a0, acc[r]);
                }
            }
            __syncthreads();
            if (X == 0) {
                // a warp per anchor: its M equal rows are one contiguous block
                for (int a = warp; a < rows; a += NT / 32) {
                    const float* src = y + a * cstr;
                    const int64_t dst = (base + a) * M * C;
                    if (vec && fb) {
                        // (a lane's chunk of the row is the same at every step
                        // where the chunks divide 32)
                        const int cpr = C / 8;
                        uint4* d4 = reinterpret_cast<uint4*>(
                            static_cast<__nv_bfloat16*>(O.sem) + dst);
                        auto chunk = [&](int c) {
                            const float* s8 = src + c * 8;
                            uint32_t q[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                q[e] = (uint32_t)__bfloat16_as_ushort(
                                           __float2bfloat16_rn(s8[2 * e])) |
                                       ((uint32_t)__bfloat16_as_ushort(
                                            __float2bfloat16_rn(s8[2 * e + 1]))
                                        << 16);
                            return make_uint4(q[0], q[1], q[2], q[3]);
                        };
                        if (32 % cpr == 0) {
                            const uint4 v = chunk(lane % cpr);
                            for (int i = lane; i < M * cpr; i += 32) d4[i] = v;
                        } else {
                            for (int i = lane; i < M * cpr; i += 32) d4[i] = chunk(i % cpr);
                        }
                    } else if (vec) {
                        const int cpr = C / 4;
                        float4* d4 = reinterpret_cast<float4*>(static_cast<float*>(O.sem) + dst);
                        for (int i = lane; i < M * cpr; i += 32)
                            d4[i] = *reinterpret_cast<const float4*>(src + (i % cpr) * 4);
                    } else {
                        for (int i = lane; i < M * C; i += 32)
                            put_feat(O.sem, dst + i, src[i % C], fb);
                    }
                }
            } else if (X == 1) {
                // gradient factor: k_ah sigma(MLP_k(f))
                for (int i = tid; i < kids; i += NT) {
                    const int a = byM.div(i);
                    O.kfac[gb + i] = P.kfac[base + a] * sigm(y[a]);
                }
            } else if (X == 2) {
                for (int i = tid; i < kids; i += NT) {
                    int m;
                    const int a = byM.divmod(i, &m);
                    O.opacity[gb + i] = sigm(y[m * S + a]);
                }
            } else if (X == 3) {
                // colour as the degree-0 SH coefficient
                for (int i = tid; i < 3 * kids; i += NT) {
                    int j;
                    const int a = by3M.divmod(i, &j);
                    const float c = sigm(y[j * S + a]);
                    put_feat(O.sh, 3 * gb + i, (c - 0.5f) / Y00, fb);
                }
            } else if (step == 4) {
                // scale, and the position x + l (x) O_m
                for (int i = tid; i < kids; i += NT) {
                    int m;
                    const int a = byM.divmod(i, &m);
                    const int64_t g = gb + i;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        const float l = P.scale[d * P.n + base + a];
                        O.scale[d * N + g] = l * sigm(y[(3 * m + d) * S + a]);
                        O.mean[d * N + g] = fmaf(l, P.offsets[g * 3 + d], P.pos[d * P.n + base + a]);
                    }
                }
            } else {
                for (int i = tid; i < kids; i += NT) {
                    int m;
                    const int a = byM.divmod(i, &m);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        O.quat[j * N + gb + i] = y[(4 * m + j) * S + a];
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ backward
struct GradIn {
    const float *mean, *quat, *scale, *opacity, *kfac, *sh, *sem;
};

struct AnchorGradOut {
    float *pos, *scale, *offsets, *feat, *sem, *kfac;
    float* w1[NMLP];
    float* b1[NMLP];
    float* w2[NMLP];
    float* b2[NMLP];
    int accumulate;
};

template <typename T>
__host__ __device__ inline size_t bwd_floats(const WLayout& L, int M) {
    return 2 * (size_t)L.total + (size_t)T::S * (3 * 32 + out_rows(L) + 3 * M);
}

__device__ __forceinline__ float gin(const float* p, int64_t i) { return p ? p[i] : 0.f; }
__device__ __forceinline__ void put(float* p, int64_t i, float v, int acc) {
    if (acc)
        p[i] += v;
    else
        p[i] = v;
}

// s[i][j] += sum over the tile's anchors (in order) of x[i][a] z[j][a], 4 x RJ
// entries.
template <typename T, int RJ>
__device__ __forceinline__ void outer_sums(const float* x, const float* z, float* s) {
    float acc[4][RJ] = {};
    for (int a = 0; a < T::TA; a += 4) {
        float xv[4][4], zv[RJ][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) ld_anchors<4>(x + r * T::S + a, xv[r]);
#pragma unroll
        for (int r = 0; r < RJ; ++r) ld_anchors<4>(z + r * T::S + a, zv[r]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < RJ; ++j) acc[i][j] = fmaf(xv[i][e], zv[j][e], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float q[RJ];
        ld_anchors<RJ>(s + i * WS, q);
#pragma unroll
        for (int j = 0; j < RJ; ++j) q[j] += acc[i][j];
        st_anchors<RJ>(s + i * WS, q);
    }
}

// b[r] += sum over the tile's anchors of x[r][a], n rows, a warp per row (in
// the products' loop the sums cost every thread 16 additions per 32
// multiply-adds).
template <typename T>
__device__ __forceinline__ void row_sums(const float* x, int n, float* b) {
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < n; r += T::NT / 32) {
        float v = 0.f;
#pragma unroll
        for (int a = lane; a < T::TA; a += 32) v += x[r * T::S + a];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) b[r] += v;
    }
}

// dL/d(branch output) before the activation's derivative, into gy (zero past
// the tile's anchors and the branch's outputs): the upstream gradients are
// read here by consecutive threads, every load independent, ahead of the
// layers that hide their latency.  For the semantic branch the sum over the
// anchor's children, for the gradient factor likewise (row 0).
template <typename T>
__device__ __forceinline__ void load_upstream(const GradIn& G, int X, int nr, int out, int M, int C,
                                              int64_t base, int rows, int64_t N, bool vec,
                                              float* gy) {
    constexpr int S = T::S, TA = T::TA, NT = T::NT;
    const FastDiv byM(M);
    const int tid = threadIdx.x;
    const int kids = rows * M;
    const int64_t gb = base * M;
    if (X == 0) {
        // 2 chunks of 4 channels x 16 anchors per warp step: whole sectors of
        // the rows, and no two lanes of a shared store in one bank
        const int pairs = (nr / 4 + 1) / 2;
        for (int i = tid; i < pairs * 2 * TA; i += NT) {
            const int q = 2 * (i / (2 * TA)) + ((i >> 4) & 1);
            const int a = ((i >> 5) * 16 + (i & 15)) % TA;
            const int j0 = 4 * q;
            if (j0 >= nr) continue;
            float u[4] = {0.f, 0.f, 0.f, 0.f};
            if (a < rows && G.sem) {
                const float* src = G.sem + (base + a) * M * C + j0;
                if (vec) {
#pragma unroll 8
                    for (int m = 0; m < M; ++m) {
                        const float4 v = *reinterpret_cast<const float4*>(src + m * C);
                        u[0] += v.x; u[1] += v.y; u[2] += v.z; u[3] += v.w;
                    }
                } else {
#pragma unroll 4
                    for (int m = 0; m < M; ++m)
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            if (j0 + r < C) u[r] += src[m * C + r];
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) gy[(j0 + r) * S + a] = u[r];
        }
    } else if (X == 1) {
        for (int i = tid; i < 4 * TA; i += NT) {
            const int r = i / TA, a = i % TA;
            float gk = 0.f;
            if (r == 0 && a < rows && G.kfac)
#pragma unroll 4
                for (int m = 0; m < M; ++m) gk += G.kfac[gb + a * M + m];
            gy[r * S + a] = gk;
        }
    } else if (X == 4) {
        for (int i = tid; i < TA * M; i += NT) {
            int m;
            const int a = byM.divmod(i, &m);
            float v[7];
#pragma unroll
            for (int d = 0; d < 7; ++d) {
                const float* src = d < 3 ? G.scale : G.quat;
                v[d] = i < kids && src ? src[(d < 3 ? d : d - 3) * N + gb + i] : 0.f;
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) gy[(3 * m + d) * S + a] = v[d];
#pragma unroll
            for (int d = 0; d < 4; ++d) gy[(quat_row(M) + 4 * m + d) * S + a] = v[3 + d];
        }
        for (int i = tid; i < (quat_row(M) - 3 * M) * TA; i += NT)
            gy[(3 * M + i / TA) * S + i % TA] = 0.f;
    } else {
        const float* src = X == 2 ? G.opacity : G.sh;
        const FastDiv by_out(out);
        for (int i = tid; i < TA * out; i += NT) {
            int j;
            const int a = by_out.divmod(i, &j);
            gy[j * S + a] = i < rows * out && src ? src[base * out + i] : 0.f;
        }
        for (int i = tid; i < (nr - out) * TA; i += NT) gy[(out + i / TA) * S + i % TA] = 0.f;
    }
}

// Adds the parameter-gradient sums of the NC blocks of a cluster to the
// outputs, this block's share of the entries.  One pass over the layout with
// all NC peers' loads in flight: array by array and peer by peer, each entry
// waited for NC remote loads in a row, half the time of a small backward.
template <int NC, int NT>
__device__ void add_params(const cg::cluster_group& cl, const WLayout& L, const AnchorGradOut& R,
                           int M, float* sg) {
    for (int e = (int)cl.block_rank() * NT + threadIdx.x; e < L.total; e += NC * NT) {
        float v[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) v[k] = *cl.map_shared_rank(sg + e, k);
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < NC; ++k) t += (double)v[k];
        int X = 0;
#pragma unroll
        for (int x = 1; x < NMLP; ++x)
            if (L.out[x] > 0 && e >= L.w1[x]) X = x;
        float* dst;
        int i = e - L.w1[X];
        if (i < AH * AF) {
            dst = R.w1[X] + i;
        } else if ((i -= AH * AF) < AH) {
            dst = R.b1[X] + i;
        } else {
            i -= AH;
            const bool w2 = i < L.rows[X] * AH;
            const int row = param_row(X, L.out[X], w2 ? i / AH : i - L.rows[X] * AH, M);
            if (row < 0) continue;
            dst = w2 ? R.w2[X] + row * AH + i % AH : R.b2[X] + row;
        }
        atomicAdd(dst, (float)t);
    }
}

template <typename T>
__global__ void __launch_bounds__(T::NT, 1) anchor_decode_bwd_kernel(const AnchorIn P, const WLayout L,
                                                                  const GradIn G,
                                                                  const AnchorGradOut R) {
    constexpr int S = T::S, RA = T::RA, NT = T::NT, GROUPS = T::GROUPS;
    // columns of a thread's tile of parameter gradients: narrower tiles where
    // the block has the threads
    constexpr int RJ = NT >= 512 ? 2 : 4;
    extern __shared__ __align__(16) float sm[];
    float* sw = sm;               // parameters
    float* sg = sw + L.total;     // parameter gradients of this block, same layout
    float* ft = sg + L.total;     // [AF][S] features
    float* h = ft + AF * S;       // [AH][S] hidden layer of one branch
    float* gp = h + AH * S;       // [AH][S] its pre-activation gradients
    float* sv = gp + AH * S;      // [3 M][S] sigma of the scale outputs
    float* gy = sv + 3 * P.M * S; // [rows][S] output gradients of one branch
    load_weights<NT>(P, L, sw);
    for (int i = threadIdx.x; i < L.total; i += NT) sg[i] = 0.f;
    const int tid = threadIdx.x, M = P.M, C = P.C, acc_out = R.accumulate;
    const FastDiv byM(M);
    const int64_t N = P.n * M;
    const int a0 = T::anchor(tid), g0 = T::group(tid);
    const bool vec = C % 4 == 0 && (reinterpret_cast<uintptr_t>(G.sem) & 15) == 0;
    const bool fvec = !acc_out && (reinterpret_cast<uintptr_t>(R.feat) & 15) == 0;
    const bool svec = !acc_out && C % 4 == 0 && ((reinterpret_cast<uintptr_t>(R.sem) |
                                                  reinterpret_cast<uintptr_t>(P.sem)) & 15) == 0;
    for (int64_t base = blockIdx.x * (int64_t)T::TA; base < P.n;
         base += (int64_t)gridDim.x * T::TA) {
        const int rows = (int)min((int64_t)T::TA, P.n - base);
        __syncthreads();
        load_feat<T>(P, base, rows, ft);
        float gf[4][RA];  // dL/df of features 4 g0 .. 4 g0 + 3
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int a = 0; a < RA; ++a) gf[r][a] = 0.f;
        __syncthreads();
#pragma unroll 1
        for (int X = 0; X < NMLP; ++X) {
            const int out = L.out[X], nr = L.rows[X];
            if (out == 0) continue;  // uniform: no semantic branch without logits
            load_upstream<T>(G, X, nr, out, M, C, base, rows, N, vec, gy);
            hidden_layer<T>(sw, L, X, ft, h);
            __syncthreads();
            // dL/d(branch output); the quaternions' outputs are linear and are
            // not needed themselves
            const int ny = X == 4 ? quat_row(M) : nr;
#pragma unroll 1
            for (int j0 = 4 * g0; j0 < ny; j0 += 4 * GROUPS) {
                float yv[4][RA], uv[4][RA];
                tile_rows<RA, S>(sw + L.w2[X] + j0 * WS, sw + L.b2[X] + j0, h + a0, yv);
#pragma unroll
                for (int r = 0; r < 4; ++r) ld_anchors<RA>(gy + (j0 + r) * S + a0, uv[r]);
#pragma unroll
                for (int a = 0; a < RA; ++a) {
                    const bool ok = a0 + a < rows;
                    const int64_t ga = base + a0 + a;  // anchor
                    if (X == 0 && svec) {
                        // four channels at once
                        const int64_t e = ga * C + j0;
                        float4 o = make_float4(0.f, 0.f, 0.f, 0.f), g;
                        if (ok) o = *reinterpret_cast<const float4*>(P.sem + e);
                        const float os[4] = {o.x, o.y, o.z, o.w};
                        float gs[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float s = sigm(yv[r][a]), u = uv[r][a];
                            gs[r] = u * s;
                            uv[r][a] = u * os[r] * s * (1.f - s);
                        }
                        g = make_float4(gs[0], gs[1], gs[2], gs[3]);
                        if (ok) *reinterpret_cast<float4*>(R.sem + e) = g;
                        continue;
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int j = j0 + r;
                        const float u = uv[r][a];
                        float v = 0.f;
                        if (ok && j < (X == 4 ? 3 * M : out)) {
                            const float s = sigm(yv[r][a]);
                            if (X == 0) {
                                put(R.sem, ga * C + j, u * s, acc_out);
                                v = u * P.sem[ga * C + j] * s * (1.f - s);
                            } else if (X == 1) {
                                put(R.kfac, ga, u * s, acc_out);
                                v = u * P.kfac[ga] * s * (1.f - s);
                            } else if (X == 2) {
                                v = u * s * (1.f - s);
                            } else if (X == 3) {
                                v = u / Y00 * s * (1.f - s);
                            } else {
                                v = u * P.scale[(j % 3) * P.n + ga] * s * (1.f - s);
                                sv[j * S + a0 + a] = s;
                            }
                        }
                        uv[r][a] = v;
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) st_anchors<RA>(gy + (j0 + r) * S + a0, uv[r]);
            }
            __syncthreads();
            // back through the branch: dL/dh = W2^T gy, the relu
            {
                float gh[4][RA] = {};
                tile_cols<RA, S>(sw + L.w2[X] + 4 * g0, gy + a0, nr, gh);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float hv[RA];
                    ld_anchors<RA>(h + (4 * g0 + r) * S + a0, hv);
#pragma unroll
                    for (int a = 0; a < RA; ++a) gh[r][a] = hv[a] > 0.f ? gh[r][a] : 0.f;
                    st_anchors<RA>(gp + (4 * g0 + r) * S + a0, gh[r]);
                }
            }
            __syncthreads();
            // dL/df += W1^T gpre, and the parameter gradients over the tile's
            // anchors; every entry has a fixed owner thread, so the shared
            // accumulators need no atomics
            tile_cols<RA, S>(sw + L.w1[X] + 4 * g0, gp + a0, AH, gf);
            constexpr int TPR = 32 / RJ;  // tiles along a row of 32
            for (int t = tid; t < (8 + nr / 4) * TPR; t += NT) {
                const int row = 4 * (t / TPR), col = RJ * (t % TPR);
                if (row < AH)
                    outer_sums<T, RJ>(gp + row * S, ft + col * S, sg + L.w1[X] + row * WS + col);
                else
                    outer_sums<T, RJ>(gy + (row - AH) * S, h + col * S,
                                      sg + L.w2[X] + (row - AH) * WS + col);
            }
            row_sums<T>(gp, AH, sg + L.b1[X]);
            row_sums<T>(gy, nr, sg + L.b2[X]);
            __syncthreads();
        }
        // features, position, offsets and scale: mu_m = x + l (x) O_m
#pragma unroll
        for (int a = 0; a < RA; ++a)
            if (a0 + a < rows) {
                const int64_t e = (base + a0 + a) * AF + 4 * g0;
                if (fvec)
                    *reinterpret_cast<float4*>(R.feat + e) =
                        make_float4(gf[0][a], gf[1][a], gf[2][a], gf[3][a]);
                else
#pragma unroll
                    for (int r = 0; r < 4; ++r) put(R.feat, e + r, gf[r][a], acc_out);
            }
        for (int i = tid; i < 3 * T::TA; i += NT) {
            const int d = i / T::TA, a = i % T::TA;
            if (a >= rows) continue;
            const int64_t ga = base + a;
            float gl = 0.f, gx = 0.f;
            for (int m = 0; m < M; ++m)
                gl = fmaf(gin(G.scale, d * N + ga * M + m), sv[(3 * m + d) * S + a], gl);
            for (int m = 0; m < M; ++m) {
                const float gm = gin(G.mean, d * N + ga * M + m);
                gx += gm;
                gl = fmaf(gm, P.offsets[(ga * M + m) * 3 + d], gl);
            }
            put(R.pos, d * P.n + ga, gx, acc_out);
            put(R.scale, d * P.n + ga, gl, acc_out);
        }
        for (int i = tid; i < rows * M; i += NT) {
            const int64_t g = base * M + i, ga = base + byM.div(i);
#pragma unroll
            for (int d = 0; d < 3; ++d)
                put(R.offsets, g * 3 + d, gin(G.mean, d * N + g) * P.scale[d * P.n + ga], acc_out);
        }
    }
    // The blocks of a cluster add up their sums, each a share of the entries,
    // in float64; then one atomic per parameter and cluster (cleared by the
    // host without accumulate).
    const cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (cl.num_blocks() == 8)
        add_params<8, NT>(cl, L, R, M, sg);
    else
        add_params<2, NT>(cl, L, R, M, sg);
    cl.sync();  // a block's shared memory stays until its peers have read it
}

// Zeroes the parameter-gradient arrays, a block each: one launch (2 us) where
// a memset per array took 20 (22 us).
struct ParamClear {
    float* ptr[4 * NMLP];
    int count[4 * NMLP];
};
__global__ void __launch_bounds__(512) clear_params_kernel(const ParamClear Z) {
    float* p = Z.ptr[blockIdx.x];
    for (int i = threadIdx.x; i < Z.count[blockIdx.x]; i += blockDim.x) p[i] = 0.f;
}

}  // namespace
}  // namespace unigs

// ------------------------------------------------------------------ C ABI
namespace {

using unigs::AH;
using unigs::AF;
using unigs::NMLP;

bool mlp_ok(const unigs_mlp& m) { return m.w1 && m.b1 && m.w2 && m.b2; }
bool mlp_ok(const unigs_mlp_grads& m) { return m.w1 && m.b1 && m.w2 && m.b2; }

bool anchors_ok(const unigs_anchors* a) {
    if (!a || a->n < 0 || a->n_offsets < 1 || a->n_offsets > UNIGS_ANCHOR_MAX_OFFSETS ||
        a->feat_dim != UNIGS_ANCHOR_FEAT || a->hidden != UNIGS_ANCHOR_HIDDEN || a->n_sem < 0 ||
        a->n_sem > UNIGS_MAX_SEM)
        return false;
    if (a->n == 0) return true;
    if (!a->pos || !a->scale || !a->offsets || !a->feat || !a->kfac) return false;
    if (reinterpret_cast<uintptr_t>(a->feat) & 15) return false;
    if (a->n_sem > 0 && (!a->sem || !mlp_ok(a->mlp_sem))) return false;
    return mlp_ok(a->mlp_k) && mlp_ok(a->mlp_opacity) && mlp_ok(a->mlp_color) &&
           mlp_ok(a->mlp_cov);
}

void make_layout(const unigs_anchors& a, unigs::WLayout& L, unigs::AnchorIn& P) {
    const int M = a.n_offsets;
    const int outs[NMLP] = {a.n_sem, 1, M, 3 * M, 7 * M};
    const unigs_mlp* mlps[NMLP] = {&a.mlp_sem, &a.mlp_k, &a.mlp_opacity, &a.mlp_color, &a.mlp_cov};
    int off = 0;
    for (int X = 0; X < NMLP; ++X) {
        L.out[X] = outs[X];
        P.w1[X] = mlps[X]->w1;
        P.b1[X] = mlps[X]->b1;
        P.w2[X] = mlps[X]->w2;
        P.b2[X] = mlps[X]->b2;
        L.w1[X] = L.b1[X] = L.w2[X] = L.b2[X] = off;
        L.rows[X] = X == 4 ? unigs::quat_row(M) + 4 * M : (outs[X] + 3) & ~3;
        if (outs[X] == 0) continue;
        L.w1[X] = off;
        off += AH * unigs::WS;
        L.b1[X] = off;
        off += AH;
        L.w2[X] = off;
        off += L.rows[X] * unigs::WS;
        L.b2[X] = off;
        off += L.rows[X];
    }
    L.total = off;
    P.n = a.n;
    P.M = M;
    P.C = a.n_sem;
    P.pos = a.pos;
    P.scale = a.scale;
    P.offsets = a.offsets;
    P.feat = a.feat;
    P.sem = a.sem;
    P.kfac = a.kfac;
}

// 128 anchors (16 warps), 64 (16 warps) and 32 (8 warps) per tile.
using Wide = unigs::Tile<2, 512>;
using Mid = unigs::Tile<1, 512>;
using Narrow = unigs::Tile<1, 256>;

// Shared memory a block can have (sm_103a).
constexpr size_t MAX_SMEM = 232448;

// The wide tiles where that leaves every SM one of 128 anchors and the buffers
// fit, else the narrow ones, so that small sets still spread over the chip (a tile of 128
// takes about three times as long as one of 32).
bool wide_tiles(int64_t n, size_t floats) {
    return n >= (int64_t)unigs::sm_count() * 128 && floats * sizeof(float) <= MAX_SMEM;
}

// A persistent grid over the tiles, in clusters of `cluster` blocks.
template <typename T, typename... Params, typename... Args>
void launch_tiles(void (*kernel)(Params...), size_t floats, int blocks_per_sm, int cluster,
                  int64_t n, cudaStream_t st, const Args&... args) {
    const size_t smem = floats * sizeof(float);
    const int64_t tiles = (n + T::TA - 1) / T::TA;
    const int64_t cap = (int64_t)unigs::sm_count() * blocks_per_sm;
    const int64_t blocks = tiles < cap ? tiles : cap;
    unigs::ensure_smem_limit(reinterpret_cast<const void*>(kernel), (int)smem);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((blocks + cluster - 1) / cluster * cluster));
    cfg.blockDim = dim3(T::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

unigs_status launch_status() {
    return cudaGetLastError() == cudaSuccess ? UNIGS_OK : UNIGS_ERR_CUDA;
}

}  // namespace

extern "C" unigs_status unigs_anchor_decode(const unigs_anchors* a,
                                            const unigs_anchor_gaussians* out,
                                            unigs_stream stream) {
    if (!anchors_ok(a) || !out || (out->feat_dtype != 0 && out->feat_dtype != 1))
        return UNIGS_ERR_INVALID_ARG;
    if (a->n == 0) return UNIGS_OK;
    if (!out->mean || !out->quat || !out->scale || !out->opacity || !out->kfac || !out->sh ||
        (a->n_sem > 0 && !out->sem))
        return UNIGS_ERR_INVALID_ARG;
    unigs::WLayout L;
    unigs::AnchorIn P;
    make_layout(*a, L, P);
    unigs::DecodeOut O{out->mean, out->quat, out->scale, out->opacity, out->kfac, out->sh,
                       out->sem};
    cudaStream_t st = (cudaStream_t)stream;
    const size_t wide = unigs::decode_floats<Wide>(L, P.M),
                 narrow = unigs::decode_floats<Narrow>(L, P.M);
    if (wide_tiles(a->n, wide))
        launch_tiles<Wide>(&unigs::anchor_decode_kernel<Wide>, wide, 2, 1, a->n, st, P, L, O,
                           out->feat_dtype);
    else
        launch_tiles<Narrow>(&unigs::anchor_decode_kernel<Narrow>, narrow, 2, 1, a->n, st, P, L,
                             O, out->feat_dtype);
    return launch_status();
}

extern "C" unigs_status unigs_anchor_decode_bwd(const unigs_anchors* a, const unigs_param_grads* g,
                                                const unigs_anchor_grads* out,
                                                unigs_stream stream) {
    if (!anchors_ok(a) || !g || !out) return UNIGS_ERR_INVALID_ARG;
    if (!out->pos || !out->scale || !out->offsets || !out->feat || !out->kfac ||
        (a->n_sem > 0 && (!out->sem || !mlp_ok(out->mlp_sem))) || !mlp_ok(out->mlp_k) ||
        !mlp_ok(out->mlp_opacity) || !mlp_ok(out->mlp_color) || !mlp_ok(out->mlp_cov))
        return UNIGS_ERR_INVALID_ARG;
    unigs::WLayout L;
    unigs::AnchorIn P;
    make_layout(*a, L, P);
    cudaStream_t st = (cudaStream_t)stream;
    const unigs_mlp_grads* mg[NMLP] = {&out->mlp_sem, &out->mlp_k, &out->mlp_opacity,
                                       &out->mlp_color, &out->mlp_cov};
    unigs::AnchorGradOut R;
    R.pos = out->pos;
    R.scale = out->scale;
    R.offsets = out->offsets;
    R.feat = out->feat;
    R.sem = out->sem;
    R.kfac = out->kfac;
    R.accumulate = out->accumulate ? 1 : 0;
    unigs::ParamClear Z = {};
    for (int X = 0; X < NMLP; ++X) {
        R.w1[X] = mg[X]->w1;
        R.b1[X] = mg[X]->b1;
        R.w2[X] = mg[X]->w2;
        R.b2[X] = mg[X]->b2;
        if (L.out[X] == 0) continue;
        float* ptr[4] = {R.w1[X], R.b1[X], R.w2[X], R.b2[X]};
        const int count[4] = {AH * AF, AH, L.out[X] * AH, L.out[X]};
        for (int i = 0; i < 4; ++i) {
            Z.ptr[4 * X + i] = ptr[i];
            Z.count[4 * X + i] = count[i];
        }
    }
    // the parameter gradients are sums of atomics: cleared first
    if (!out->accumulate) unigs::clear_params_kernel<<<4 * NMLP, 512, 0, st>>>(Z);
    if (a->n == 0) return launch_status();
    unigs::GradIn G{g->mean, g->quat, g->scale, g->opacity, g->kfac, g->sh, g->sem};
    const size_t wide = unigs::bwd_floats<Wide>(L, P.M), mid = unigs::bwd_floats<Mid>(L, P.M),
                 narrow = unigs::bwd_floats<Narrow>(L, P.M);
    // The parameter gradients meet in one float32 atomic per cluster: 2 blocks
    // (the SMs of a pair, so that a full grid still fits), or 8 where the
    // tiles leave enough SMs free that every cluster of 8 finds its place.
    const int64_t tiles = (a->n + Narrow::TA - 1) / Narrow::TA;
    const int small = 4 * tiles <= 3 * unigs::sm_count() ? 8 : 2;
    if (wide_tiles(a->n, wide))
        launch_tiles<Wide>(&unigs::anchor_decode_bwd_kernel<Wide>, wide, 1, 2, a->n, st, P, L, G, R);
    else if (wide_tiles(a->n, mid))
        launch_tiles<Mid>(&unigs::anchor_decode_bwd_kernel<Mid>, mid, 1, 2, a->n, st, P, L, G, R);
    else
        launch_tiles<Narrow>(&unigs::anchor_decode_bwd_kernel<Narrow>, narrow, 1, small, a->n, st, P,
                             L, G, R);
    return launch_status();
}

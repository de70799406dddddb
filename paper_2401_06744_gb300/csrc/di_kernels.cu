// CUDA kernels (sm_103a) of the reduced-FMG ORAS inpainting decoder.
//
// Problem (Section 2.2, eq. 2.6): (C + (I - C) L) u = C f per channel, L the
// 5-point negated Laplacian with reflecting boundaries and unit spacing on
// every level (coarse right-hand sides carry the (H/h)^2 = 4 factor).
//
// Kernels:
//   k_pyramid_level  Section 4.3: one pyramid level in one pass (2x2 max pooling of
//                    the mask, modified or naive mask values, packed mask words,
//                    unknown count); k_mask_down and k_values_down are the
//                    separate steps of the single-step entry points
//   k_pack_mask16    the finest level's packed mask words and unknown count, 16 mask
//                    bytes per thread; k_pack_mask for rows of other widths
//   k_residual       r = b - A u with per-CTA partial sums of r^2 (Algorithm 2 step 1)
//   k_reduce         fixed-order sum of the partials (one global scalar product)
//   k_restrict       Algorithm 3 steps 2-3 fused: residual + 2x2 averaging (x4);
//                    k_restrict_c for the large levels of FP32 images (every
//                    channel of a cell by one thread)
//   k_prolong        Section 4.4 bilinear prolongation, cascadic or correction mode
//                    (where the block kernel cannot form its start by prolongation)
//   k_select         u = c ? b : 0 (or c ? b : u for a given start)
//   k_oras_2w        Algorithm 2 steps 1-3 for 32x32 blocks: two warps per (block,
//                    channel), plain CG in registers as packed FP32 pairs, tiles by
//                    TMA; optionally the start formed by prolongation inside it
//   k_oras_4w        the same with four warps per (block, channel), for launches of
//                    few local problems (the same bits)
//   k_oras_2w_h      k_oras_2w with FP16 / BF16 local iterates
//   k_oras_warp      8x8 and 16x16 blocks: one warp per (block, channel)
//   k_combine        Algorithm 2 step 3 for pixels shared by several blocks: the
//                    sums of their weighted contributions in a fixed order;
//                    k_combine_px for blocks of 8 and 16
//   k_plan, k_stop   the device-driven decode: levels in use and start, and the
//                    stop test after every V-cycle (conditional graph nodes)
//   k_batch_*        the batched form: the same steps over the segment tables of
//                    every image of a batch
//   k_cg_*           the global CG smoother of the comparison methods (Section 5)
//
// Layout: images planar [C][h][w] float32, masks [h][w] uint8.  The ORAS
// block pass writes pixels that only one block weights (weight 1) straight to
// u_out and parks weighted contributions of shared pixels in a BxB tile of its
// own per block and channel ([block][channel][B][B], so every word has one
// writer); the combine pass adds them in a fixed order, which keeps the result
// deterministic without atomics.
#include "di_internal.h"
#include "../../include/di.h"

#include <cfloat>
#include <cstring>
#include <cmath>

#include <atomic>
#include <mutex>
#include <type_traits>

#include <cuda.h>  // CUtensorMap and its enums (the encoder comes from the runtime)
#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace di {

static std::atomic<long long> g_launches{0};
// the calling thread's own launches: captures count their kernels with it, so
// that decodes finishing on other threads meanwhile do not enter the count
static thread_local long long t_launches = 0;
long long launch_count() { return g_launches.load(std::memory_order_relaxed); }
long long thread_launch_count() { return t_launches; }
void add_launches(long long k) {
    g_launches.fetch_add(k, std::memory_order_relaxed);
    t_launches += k;
}

namespace {

constexpr unsigned kFull = 0xffffffffu;

inline void count(int k = 1) {
    g_launches.fetch_add(k, std::memory_order_relaxed);
    t_launches += k;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
    return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, d));
    return v;
}

// Element access of an array stored as float, FP16 or BF16 (the narrow
// coarse-level storage); arithmetic is FP32 throughout.
template <class T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<__half>(const __half* p) { return __half2float(*p); }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
    return __bfloat162float(*p);
}
template <class T> __device__ __forceinline__ void stf(T* p, float v);
template <> __device__ __forceinline__ void stf<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<__half>(__half* p, float v) { *p = __float2half_rn(v); }
template <> __device__ __forceinline__ void stf<__nv_bfloat16>(__nv_bfloat16* p, float v) {
    *p = __float2bfloat16_rn(v);
}

// ---------------------------------------------------------------------------
// Mask pyramid (Section 4.3)
// ---------------------------------------------------------------------------

__device__ __forceinline__ void mask_down_body(const uint8_t* __restrict__ c, int w, int h,
                            uint8_t* __restrict__ cH, int wH, int hH, int bx, int by) {
    const int X = bx * blockDim.x + threadIdx.x;
    const int Y = by * blockDim.y + threadIdx.y;
    if (X >= wH || Y >= hH) return;
    const int x = 2 * X, y = 2 * Y;
    const bool x1 = x + 1 < w, y1 = y + 1 < h;
    const uint8_t* row = c + (size_t)y * w;
    bool m = row[x] != 0;
    if (x1) m |= row[x + 1] != 0;
    if (y1) {
        const uint8_t* row2 = row + w;
        m |= row2[x] != 0;
        if (x1) m |= row2[x + 1] != 0;
    }
    cH[(size_t)Y * wH + X] = m ? 1 : 0;
}

__global__ void k_mask_down(const uint8_t* __restrict__ c, int w, int h,
                            uint8_t* __restrict__ cH, int wH, int hH) {
    mask_down_body(c, w, h, cH, wH, hH, blockIdx.x, blockIdx.y);
}

// One coarse cell: weights of its (up to four) fine children.
__device__ __forceinline__ void values_down_body(const uint8_t* __restrict__ c, const float* __restrict__ b,
                              int w, int h, int C, const uint8_t* __restrict__ cH,
                              float* __restrict__ bH, int wH, int hH, int modified, int bx, int by) {
    const int X = bx * blockDim.x + threadIdx.x;
    const int Y = by * blockDim.y + threadIdx.y;
    if (X >= wH || Y >= hH) return;
    const size_t n = (size_t)w * h, nH = (size_t)wH * hH, P = (size_t)Y * wH + X;
    if (!cH[P]) {
        for (int ch = 0; ch < C; ++ch) bH[ch * nH + P] = 0.f;
        return;
    }
    float wt[4];
    size_t idx[4];
    float den = 0.f, cnt = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int x = 2 * X + (k & 1), y = 2 * Y + (k >> 1);
        wt[k] = 0.f;
        idx[k] = 0;
        if (x >= w || y >= h) continue;
        const size_t p = (size_t)y * w + x;
        idx[k] = p;
        if (!c[p]) continue;
        cnt += 1.f;
        if (!modified) { wt[k] = 1.f; continue; }
        int m = 0;
        const int xi = x ^ 1, yi = y ^ 1;               // partners inside the cell
        if (xi < w) m += c[(size_t)y * w + xi] != 0;
        if (yi < h) m += c[(size_t)yi * w + x] != 0;
        const int xo = (x & 1) ? x + 1 : x - 1;          // neighbours across the cell
        const int yo = (y & 1) ? y + 1 : y - 1;
        if (xo >= 0 && xo < w) m += cH[(size_t)Y * wH + (xo >> 1)] != 0;
        if (yo >= 0 && yo < h) m += cH[(size_t)(yo >> 1) * wH + X] != 0;
        wt[k] = (float)(4 - m);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) den += wt[k];
    if (den == 0.f) {  // gap of the printed rule: fall back to the naive average
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = 2 * X + (k & 1), y = 2 * Y + (k >> 1);
            wt[k] = (x < w && y < h && c[idx[k]]) ? 1.f : 0.f;
        }
        den = cnt;
    }
    const float inv = 1.f / fmaxf(1.f, den);
    for (int ch = 0; ch < C; ++ch) {
        const float* bc = b + ch * n;
        float num = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (wt[k] != 0.f) num = __fmaf_rn(wt[k], bc[idx[k]], num);
        bH[ch * nH + P] = num * inv;
    }
}

__global__ void k_values_down(const uint8_t* __restrict__ c, const float* __restrict__ b,
                              int w, int h, int C, const uint8_t* __restrict__ cH,
                              float* __restrict__ bH, int wH, int hH, int modified) {
    values_down_body(c, b, w, h, C, cH, bH, wH, hH, modified, blockIdx.x, blockIdx.y);
}

// One level of the pyramid in one pass (Section 4.3).  A CTA of 32 x 8 threads
// covers 32 x 8R coarse cells, (bx, by) its position, nbx the CTAs along x (one
// column per packed word of a coarse row but the padding word).  First every
// thread forms the mask of its R cells (rows 8 apart): cH = max over the
// children (four mask bytes, as byte pairs where the image allows), the packed
// words (known or beyond the image = 1; the last column's CTAs write the
// padding word too), the count of unknown cells, and bH = 0 where nothing is
// known.  Then the known cells get their mask values (MOD: modified, else naive
// downsampling, the weights and sums of values_down_body), the known children's
// values of every channel loaded together.  The modified weights take the child
// flags of the cell's four neighbours from a shared tile with a one-cell halo.
// LIST (MOD only): the known cells are collected in a list and get their values
// a thread each; otherwise each thread does its own.  values = 0: masks only (a
// given start).
// The list is there because the modified weights are most of the instructions
// and few cells are known (15 % at a mask density of 4 %): with a thread per cell
// the kernel was bound by instruction issue (474 warp instructions per 32 cells).
// Times of the kernel alone, mask density 0.04 / 0.5 (3840x2160 RGB takes about
// 10 us at the copy rate), a thread per cell and channel by channel before:
// 3840x2160 RGB 49.5 / 51.4 -> 26.6 / 36.1 us, 1920x1080 RGB 12.3 / 13.0 -> 7.9 /
// 11.5, 3001x1999 RGB 35.6 / 37.5 -> 20.4 / 28.5.
template <int R, bool LIST, bool MOD>
__device__ __forceinline__ void pyramid_level_body(
    const uint8_t* __restrict__ c, const float* __restrict__ b, int w, int h, int C,
    uint8_t* __restrict__ cH, float* __restrict__ bH, int wH, int hH, int values,
    uint32_t* __restrict__ bits, int wpr, unsigned long long* __restrict__ unknown, int bx,
    int by, int nbx) {
    static_assert(MOD || !LIST, "the naive average needs no list");
    constexpr int ROWS = 8 * R;
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * 32 + tx;
    const int X0 = bx * 32, Y0 = by * ROWS, X = X0 + tx;
    const size_t nH = (size_t)wH * hH;
    __shared__ uint8_t s_kn[MOD ? ROWS + 2 : 1][34];   // child flags (bit k: child k known)
    __shared__ uint16_t s_list[LIST ? 32 * ROWS : 1];  // known cells, 32 row + column
    __shared__ unsigned s_n, s_unk[8];
    if (LIST && t == 0) s_n = 0u;
    // flags of the children of coarse cell (Xc, Yc), 0 off the level
    const bool pairs = (w & 1) == 0 && (reinterpret_cast<uintptr_t>(c) & 1) == 0;
    auto children = [&](int Xc, int Yc) -> unsigned {
        if (Xc < 0 || Xc >= wH || Yc < 0 || Yc >= hH) return 0u;
        const int x = 2 * Xc, y = 2 * Yc;
        const uint8_t* row = c + (size_t)y * w + x;
        const bool y1 = y + 1 < h;
        unsigned c0, c1, c2, c3;
        if (pairs) {
            const unsigned r0 = *reinterpret_cast<const uint16_t*>(row);
            const unsigned r1 = y1 ? *reinterpret_cast<const uint16_t*>(row + w) : 0u;
            c0 = r0 & 0xffu;
            c1 = r0 >> 8;
            c2 = r1 & 0xffu;
            c3 = r1 >> 8;
        } else {
            const bool x1 = x + 1 < w;
            c0 = row[0];
            c1 = x1 ? row[1] : 0u;
            c2 = y1 ? row[w] : 0u;
            c3 = (x1 && y1) ? row[w + 1] : 0u;
        }
        return (c0 ? 1u : 0u) | (c1 ? 2u : 0u) | (c2 ? 4u : 0u) | (c3 ? 8u : 0u);
    };
    unsigned ck[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ck[r] = children(X, Y0 + ty + 8 * r);
    if (MOD && values) {  // the halo (uniform over the grid)
        if (ty == 0) s_kn[0][tx + 1] = (uint8_t)children(X, Y0 - 1);
        if (ty == 7) s_kn[ROWS + 1][tx + 1] = (uint8_t)children(X, Y0 + ROWS);
        for (int i = t; i < 2 * ROWS; i += 256)
            s_kn[(i >> 1) + 1][(i & 1) ? 33 : 0] =
                (uint8_t)children((i & 1) ? X0 + 32 : X0 - 1, Y0 + (i >> 1));
    }
    if constexpr (LIST) __syncthreads();  // s_n
    const size_t n = (size_t)w * h;
    auto value = [&](auto channels, int lx, int ly, unsigned f) {  // of a known cell with the flags f
        constexpr int NC = decltype(channels)::value;  // C <= NC
        const int Xc = X0 + lx, Yc = Y0 + ly;
        const float* bp = b + (size_t)(2 * Yc) * w + 2 * Xc;
        float bv[NC][4];
#pragma unroll
        for (int ch = 0; ch < NC; ++ch)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                bv[ch][k] = (NC == 1 || ch < C) && ((f >> k) & 1u)
                                ? bp[ch * n + (k >> 1) * (size_t)w + (k & 1)] : 0.f;
        unsigned side[2] = {0u, 0u}, vert[2] = {0u, 0u};  // neighbours known: left, right; above, below
        if (MOD) {
            // the flags are 0 off the level; the child columns and rows off an
            // odd image have no neighbour across the cell either, but they are
            // unknown and get no weight
            side[0] = s_kn[ly + 1][lx] != 0;
            side[1] = s_kn[ly + 1][lx + 2] != 0;
            vert[0] = s_kn[ly][lx + 1] != 0;
            vert[1] = s_kn[ly + 2][lx + 1] != 0;
        }
        float wt[4];
        float den = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned m = ((f >> (k ^ 1)) & 1u) + ((f >> (k ^ 2)) & 1u) + side[k & 1] +
                               vert[k >> 1];
            wt[k] = !((f >> k) & 1u) ? 0.f : MOD ? (float)(4 - (int)m) : 1.f;
            den += wt[k];
        }
        if (den == 0.f) {  // gap of the printed rule: the naive average
            den = (float)__popc(f);
#pragma unroll
            for (int k = 0; k < 4; ++k) wt[k] = ((f >> k) & 1u) ? 1.f : 0.f;
        }
        const float inv = 1.f / fmaxf(1.f, den);
        const size_t P = (size_t)Yc * wH + Xc;
#pragma unroll
        for (int ch = 0; ch < NC; ++ch) {
            float num = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (wt[k] != 0.f) num = __fmaf_rn(wt[k], bv[ch][k], num);
            if (NC == 1 || ch < C) bH[ch * nH + P] = num * inv;
        }
    };
    unsigned unk = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int ly = ty + 8 * r, Y = Y0 + ly;
        const bool kn = ck[r] != 0u, in = X < wH && Y < hH;
        const unsigned word = __ballot_sync(kFull, X >= wH || kn);
        if (Y < hH && tx == 0) {
            bits[(size_t)Y * wpr + bx] = word;
            if (bx == nbx - 1) bits[(size_t)Y * wpr + wpr - 1] = 0xffffffffu;  // the padding word
        }
        if (Y < hH) unk += (unsigned)__popc(~word);  // warp-uniform
        if (in) cH[(size_t)Y * wH + X] = kn ? 1 : 0;
        if (values) {
            if (MOD) s_kn[ly + 1][tx + 1] = (uint8_t)ck[r];
            if constexpr (LIST) {
                const unsigned list = __ballot_sync(kFull, kn);
                unsigned at = 0;
                if (tx == 0 && list) at = atomicAdd(&s_n, (unsigned)__popc(list));
                at = __shfl_sync(kFull, at, 0);
                if (kn)
                    s_list[at + (unsigned)__popc(list & ((1u << tx) - 1u))] = (uint16_t)(32 * ly + tx);
            }
            if (!kn && in) {
                for (int ch = 0; ch < C; ++ch) bH[ch * nH + (size_t)Y * wH + X] = 0.f;
            }
        }
    }
    auto own_values = [&](auto channels) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (ck[r]) value(channels, tx, ty + 8 * r, ck[r]);
    };
    if (!LIST && !MOD && values) {  // need no neighbours
        if (C == 1) own_values(std::integral_constant<int, 1>{});
        else own_values(std::integral_constant<int, kMaxChannels>{});
    }
    if (tx == 0) s_unk[ty] = unk;
    __syncthreads();
    if (unknown && t == 0) {
        unsigned a = 0;
        for (int i = 0; i < 8; ++i) a += s_unk[i];
        if (a) atomicAdd(unknown, (unsigned long long)a);
    }
    if (!values) return;
    if constexpr (LIST) {
        const unsigned known = s_n;
        for (unsigned i = t; i < known; i += 256) {
            const int e = s_list[i], lx = e & 31, ly = e >> 5;
            value(std::integral_constant<int, kMaxChannels>{}, lx, ly, s_kn[ly + 1][lx + 1]);
        }
    } else if constexpr (MOD) {
        own_values(std::integral_constant<int, kMaxChannels>{});
    }
}

template <int R, bool LIST, bool MOD>
__global__ void __launch_bounds__(256)
k_pyramid_level(const uint8_t* __restrict__ c, const float* __restrict__ b, int w, int h, int C,
                uint8_t* __restrict__ cH, float* __restrict__ bH, int wH, int hH, int values,
                uint32_t* __restrict__ bits, int wpr,
                unsigned long long* __restrict__ unknown) {
    pyramid_level_body<R, LIST, MOD>(c, b, w, h, C, cH, bH, wH, hH, values, bits, wpr, unknown,
                          blockIdx.x, blockIdx.y, gridDim.x);
}

// ---------------------------------------------------------------------------
// Residual and its norm (Algorithm 2 step 1; Section 2.2 "single global scalar
// product")
// ---------------------------------------------------------------------------

template <bool F64 = false>
__device__ __forceinline__ float residual_at(const float* __restrict__ u, int zero_u,
                                             const float* __restrict__ b, int rhs_zero,
                                             const uint8_t* __restrict__ c, int w, int h,
                                             int x, int y) {
    typedef typename std::conditional<F64, double, float>::type R;
    const size_t p = (size_t)y * w + x;
    if (c[p]) return b[p] - (zero_u ? 0.f : u[p]);
    const R rhs = rhs_zero ? (R)0 : (R)b[p];
    if (zero_u) return (float)rhs;
    const R uc = u[p];
    R lu = 0;
    if (x > 0) lu += uc - (R)u[p - 1];
    if (x < w - 1) lu += uc - (R)u[p + 1];
    if (y > 0) lu += uc - (R)u[p - w];
    if (y < h - 1) lu += uc - (R)u[p + w];
    return (float)(rhs - lu);
}

constexpr int kResBX = 32, kResBY = 8;

template <bool F64>
__global__ void __launch_bounds__(kResBX * kResBY)
k_residual(const float* __restrict__ u, int zero_u, const float* __restrict__ b, int rhs_zero,
           const uint8_t* __restrict__ c, int w, int h, float* __restrict__ r,
           double* __restrict__ partials) {
    const int x = blockIdx.x * kResBX + threadIdx.x;
    const int y = blockIdx.y * kResBY + threadIdx.y;
    const int ch = blockIdx.z;
    const size_t n = (size_t)w * h;
    float rv = 0.f;
    if (x < w && y < h) {
        rv = residual_at<F64>(u + ch * n, zero_u, b + ch * n, rhs_zero, c, w, h, x, y);
        if (r) r[ch * n + (size_t)y * w + x] = rv;
    }
    // FP32 within the warp, FP64 across the warps and CTAs (fixed order)
    __shared__ double s_part[kResBX * kResBY / 32];
    const int t = threadIdx.y * kResBX + threadIdx.x;
    const float v = warp_sum(rv * rv);
    if ((t & 31) == 0) s_part[t >> 5] = (double)v;
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int i = 0; i < kResBX * kResBY / 32; ++i) s += s_part[i];
        const size_t nparts = (size_t)gridDim.x * gridDim.y;
        partials[ch * nparts + (size_t)blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(256)
k_reduce(const double* __restrict__ partials, int nparts, double* __restrict__ out) {
    const int ch = blockIdx.x;
    const double* p = partials + (size_t)ch * nparts;
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += p[i];
    __shared__ double s_w[8];
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_w[i];
        out[ch] = t;
    }
}

// ---------------------------------------------------------------------------
// Global CG on one level, the comparison smoother of Section 5 (CG in place of
// ORAS, and single-level CG).  x is the correction of the iterate, r = b - A(u
// + x) is kept by recurrence; p and r vanish on known pixels.  Per channel
// the device keeps sc[ch * 4 + 0/1] = r.r of even/odd steps and sc[ch*4 + 2] =
// p.Ap, so a step needs no host round trip.
//
// The kernels stride over 32x8 pixel tiles with a fixed number of CTAs per
// channel (kCgCtas in total), so a dot product leaves one partial per CTA.
// Products are summed in FP32 within a thread and a warp and in FP64 across
// the warps and CTAs, all in a fixed order: GB300 issues FP64 at a small
// fraction of its FP32 rate, and per-element FP64 arithmetic would dominate
// these memory-bound passes.
// ---------------------------------------------------------------------------

constexpr int kCgBX = 32, kCgBY = 8, kCgCtas = 152 * 8;

// Sum of one float per thread of a 256-thread CTA, written to
// partials[ch * nparts + blockIdx.x]: FP32 within each warp, FP64 across the
// eight warps in warp order.
__device__ __forceinline__ void block_partial(float v, double* __restrict__ partials, int ch,
                                              int nparts) {
    __shared__ double s_p[kCgBX * kCgBY / 32];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    v = warp_sum(v);
    if ((t & 31) == 0) s_p[t >> 5] = (double)v;
    __syncthreads();
    if (t == 0) {
        double a = 0.0;
        for (int i = 0; i < kCgBX * kCgBY / 32; ++i) a += s_p[i];
        partials[(size_t)ch * nparts + blockIdx.x] = a;
    }
}

struct CgTiles {
    int w, h, tiles_x, ntiles;
    __device__ __forceinline__ void pixel(int t, int* X, int* Y) const {
        const int ty = t / tiles_x;
        *X = (t - ty * tiles_x) * kCgBX + threadIdx.x;
        *Y = ty * kCgBY + threadIdx.y;
    }
};

__global__ void __launch_bounds__(kCgBX * kCgBY)
k_cg_init(CgTiles g, const float* __restrict__ u, int zero_u, const float* __restrict__ b,
          int rhs_zero, const uint8_t* __restrict__ c, float* __restrict__ r,
          float* __restrict__ p, float* __restrict__ x, double* __restrict__ partials) {
    const int ch = blockIdx.y;
    const size_t n = (size_t)g.w * g.h;
    float acc = 0.f;
    for (int t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int X, Y;
        g.pixel(t, &X, &Y);
        if (X >= g.w || Y >= g.h) continue;
        const size_t pix = (size_t)Y * g.w + X, i = ch * n + pix;
        float rv = 0.f;
        if (!c[pix])
            rv = residual_at(u + ch * n, zero_u, b + ch * n, rhs_zero, c, g.w, g.h, X, Y);
        r[i] = rv;
        p[i] = rv;
        x[i] = 0.f;
        acc = fmaf(rv, rv, acc);
    }
    block_partial(acc, partials, ch, gridDim.x);
}

__global__ void __launch_bounds__(kCgBX * kCgBY)
k_cg_matvec(CgTiles g, const float* __restrict__ p, const uint8_t* __restrict__ c,
            float* __restrict__ q, double* __restrict__ partials) {
    const int ch = blockIdx.y;
    const int w = g.w, h = g.h;
    const size_t n = (size_t)w * h;
    const float* pc = p + ch * n;
    float acc = 0.f;
    for (int t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int X, Y;
        g.pixel(t, &X, &Y);
        if (X >= w || Y >= h) continue;
        const size_t pix = (size_t)Y * w + X;
        float qv = 0.f;
        if (!c[pix]) {
            const float pv = pc[pix];
            float sn = 0.f;
            int deg = 0;
            if (X > 0) { ++deg; sn += pc[pix - 1]; }
            if (X < w - 1) { ++deg; sn += pc[pix + 1]; }
            if (Y > 0) { ++deg; sn += pc[pix - w]; }
            if (Y < h - 1) { ++deg; sn += pc[pix + w]; }
            qv = (float)deg * pv - sn;  // known neighbours have p = 0
            acc = fmaf(pv, qv, acc);
        }
        q[ch * n + pix] = qv;
    }
    block_partial(acc, partials, ch, gridDim.x);
}

__global__ void __launch_bounds__(kCgBX * kCgBY)
k_cg_update(CgTiles g, const float* __restrict__ p, const float* __restrict__ q,
            float* __restrict__ x, float* __restrict__ r, const double* __restrict__ sc, int par,
            double* __restrict__ partials) {
    const int ch = blockIdx.y;
    const size_t n = (size_t)g.w * g.h;
    const double rr = sc[ch * 4 + par], pq = sc[ch * 4 + 2];
    const float a = pq > 0.0 ? (float)(rr / pq) : 0.f;
    float acc = 0.f;
    for (int t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
        int X, Y;
        g.pixel(t, &X, &Y);
        if (X >= g.w || Y >= g.h) continue;
        const size_t i = ch * n + (size_t)Y * g.w + X;
        x[i] = fmaf(a, p[i], x[i]);
        const float rv = fmaf(-a, q[i], r[i]);
        r[i] = rv;
        acc = fmaf(rv, rv, acc);
    }
    block_partial(acc, partials, ch, gridDim.x);
}

__global__ void k_cg_direction(float* __restrict__ p, const float* __restrict__ r, size_t n,
                               const double* __restrict__ sc, int par) {
    const int ch = blockIdx.y;
    const double rr_old = sc[ch * 4 + par], rr_new = sc[ch * 4 + (par ^ 1)];
    const float beta = rr_old > 0.0 ? (float)(rr_new / rr_old) : 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        p[ch * n + i] = fmaf(beta, p[ch * n + i], r[ch * n + i]);
}

// out = in + x (in may be zero); the largest |x| goes into *maxupd (nullable)
__global__ void k_cg_finish(const float* __restrict__ in, int zero_in,
                            const float* __restrict__ x, float* __restrict__ out, size_t n,
                            unsigned* __restrict__ maxupd) {
    const int ch = blockIdx.y;
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const float xv = x[ch * n + i];
        out[ch * n + i] = (zero_in ? 0.f : in[ch * n + i]) + xv;
        m = fmaxf(m, fabsf(xv));
    }
    if (maxupd) {
        m = warp_max(m);
        if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(maxupd, __float_as_uint(m));
    }
}

__global__ void __launch_bounds__(256)
k_reduce_slot(const double* __restrict__ partials, int nparts, double* __restrict__ sc, int slot) {
    const int ch = blockIdx.x;
    const double* pp = partials + (size_t)ch * nparts;
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += pp[i];
    __shared__ double s_w[8];
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_w[i];
        sc[ch * 4 + slot] = t;
    }
}

// ---------------------------------------------------------------------------
// Grid transfers (Algorithm 3, Section 4.4)
// ---------------------------------------------------------------------------

// One thread per coarse cell.  A coarse cell off the coarse mask has four
// unknown children (max pooling), so their residuals need no mask loads: the
// 4x4 patch of u around the children is read at once (zero outside the image)
// and the in-image neighbour count gives the reflecting boundary.  u is stored
// as TU, the right-hand side b as TB, rH as TO (FP16/BF16 on the coarse levels
// in the 16-bit precision modes).  F64: the children's residuals are formed
// and summed in FP64 (the finest-grid refinement residual) and rounded once.
// BESIDE (for VEC): the patch is loaded beside the cell's mask byte, not after
// it, and dropped if the cell is known.
template <bool VEC, class TU, class TB, class TO, bool F64, bool BESIDE = false>
__device__ __forceinline__ void restrict_body(const TU* __restrict__ u, const TB* __restrict__ b, int rhs_zero,
           int w, int h, const uint8_t* __restrict__ cH, TO* __restrict__ rH, int wH,
           int hH, int bx, int by, int bz) {
    typedef typename std::conditional<F64, double, float>::type R;
    const int X = bx * blockDim.x + threadIdx.x;
    const int Y = by * blockDim.y + threadIdx.y;
    const int ch = bz;
    if (X >= wH || Y >= hH) return;
    const size_t n = (size_t)w * h, nH = (size_t)wH * hH, P = (size_t)Y * wH + X;
    const uint8_t known = cH[P];
    const TU* uc = u + ch * n;
    const int x0 = 2 * X - 1, y0 = 2 * Y - 1;
    if (VEC && X >= 1 && Y >= 1 && 2 * X + 2 < w && 2 * Y + 2 < h) {
        // a cell whose 4x4 patch lies inside the image (all but the border
        // cells): every child has four neighbours and the count is 4, so the
        // same sums as below without a bounds test (the same bits)
        if (!BESIDE && known) {
            stf(rH + ch * nH + P, 0.f);
            return;
        }
        const TU* r0 = uc + (size_t)y0 * w + x0;
        float t[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 mid = *reinterpret_cast<const float2*>(r0 + (size_t)j * w + 1);
            t[j][1] = mid.x;
            t[j][2] = mid.y;
            t[j][0] = (j == 1 || j == 2) ? ldf(r0 + (size_t)j * w) : 0.f;
            t[j][3] = (j == 1 || j == 2) ? ldf(r0 + (size_t)j * w + 3) : 0.f;
        }
        R sum = 0;
#pragma unroll
        for (int j = 1; j <= 2; ++j) {
            float2 rb = make_float2(0.f, 0.f);
            if (!rhs_zero)
                rb = *reinterpret_cast<const float2*>(b + ch * n + (size_t)(y0 + j) * w + x0 + 1);
#pragma unroll
            for (int i = 1; i <= 2; ++i) {
                const R lu = (R)4 * (R)t[j][i] -
                             ((R)t[j][i - 1] + (R)t[j][i + 1] + (R)t[j - 1][i] + (R)t[j + 1][i]);
                const R rhs = rhs_zero ? (R)0 : (R)(i == 1 ? rb.x : rb.y);
                sum += rhs - lu;
            }
        }
        stf(rH + ch * nH + P, known ? 0.f : (float)sum);
        return;
    }
    if (known) { stf(rH + ch * nH + P, 0.f); return; }
    float t[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int y = y0 + j;
        const bool yok = y >= 0 && y < h;
        if (VEC) {
            // the two children's columns as one 8-byte word, the outer
            // columns (rows 1 and 2 only) as single words
            float2 mid = make_float2(0.f, 0.f);
            if (yok) mid = *reinterpret_cast<const float2*>(uc + (size_t)y * w + x0 + 1);
            t[j][1] = mid.x;
            t[j][2] = mid.y;
            const bool inner = j == 1 || j == 2;
            t[j][0] = (inner && yok && x0 >= 0) ? ldf(uc + (size_t)y * w + x0) : 0.f;
            t[j][3] = (inner && yok && x0 + 3 < w) ? ldf(uc + (size_t)y * w + x0 + 3) : 0.f;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int x = x0 + i;
                const bool corner = (i == 0 || i == 3) && (j == 0 || j == 3);
                t[j][i] = (!corner && yok && x >= 0 && x < w) ? ldf(uc + (size_t)y * w + x) : 0.f;
            }
        }
    }
    R sum = 0;
    int cnt = 0;
#pragma unroll
    for (int j = 1; j <= 2; ++j) {
        float2 rb = make_float2(0.f, 0.f);
        if (VEC && !rhs_zero && y0 + j < h)
            rb = *reinterpret_cast<const float2*>(b + ch * n + (size_t)(y0 + j) * w + x0 + 1);
#pragma unroll
        for (int i = 1; i <= 2; ++i) {
            const int x = x0 + i, y = y0 + j;
            if (x >= w || y >= h) continue;
            const int deg = (x > 0) + (x < w - 1) + (y > 0) + (y < h - 1);
            const R lu = (R)deg * (R)t[j][i] -
                         ((R)t[j][i - 1] + (R)t[j][i + 1] + (R)t[j - 1][i] + (R)t[j + 1][i]);
            const R rhs = rhs_zero ? (R)0
                          : VEC ? (R)(i == 1 ? rb.x : rb.y)
                                : (R)ldf(b + ch * n + (size_t)y * w + x);
            sum += rhs - lu;
            ++cnt;
        }
    }
    // 4 sum / cnt with cnt in {1, 2, 4} (children inside the image): an exact
    // power-of-two scaling, so a multiplication gives the quotient bit for bit
    stf(rH + ch * nH + P, (float)(sum * (R)(4 >> (cnt >> 1))));
}

// The large levels of FP32 images: one thread per coarse cell and all its
// channels, every channel's patch in flight together.  The kernel waits for
// memory, so what counts is loads in flight: CTAs of 128 threads (gray: 256, the
// small CTAs come and go too fast where there is nothing to do, 9.4 us against
// 5.9 at density 0.9), as many per SM as the registers of a thread's patches
// allow (three channels without a right-hand side 9: 27.7 us, 10: 26.8, 11:
// 28.4; with one 7: 39.3, 8: 38.2; eight everywhere, with spills: 30.4 and 39.1).
// The patch is loaded after the cell's mask byte, and not at all for a known
// cell; the mask bytes are fetched into L2 a wave of CTAs ahead, which gains 1.4
// us.  (Loaded beside the byte it is as fast where few cells are known, but where
// nearly all are it took 25.8 and 36.0 us for the 10.3 and 10.5 below.)
// 3840x2160 RGB (127 MB, 19 us at the copy rate), mask density 0.04 / 0.5 / 0.9:
// 42.0 / 40.1 / 14.4 us with a thread per cell and channel, 26.8 / 24.6 / 10.3
// here; with a right-hand side 48.8 / 43.4 / 14.4 and 38.2 / 33.0 / 10.5; gray
// 15.8 / 14.4 / 6.0 and 12.1 / 11.0 / 5.9.
// VEC: children pairs as 8-byte words.  Border cells as above.
__host__ __device__ constexpr int restrict_rows(int C) { return C == 1 ? 8 : 4; }  // of cells per CTA
constexpr int restrict_ctas(int C, bool vec, bool rhs0) {  // per SM
    if (C == 1) return 8;
    return rhs0 ? (C == 2 ? 14 : C == 3 ? (vec ? 10 : 9) : 7) : C == 2 ? 10 : C == 3 ? 8 : 6;
}
constexpr int kRestrictAhead = 152 * 8 * 128;  // cells: a wave of CTAs
template <int C, bool VEC, bool RHS0>
__global__ void __launch_bounds__(32 * restrict_rows(C), restrict_ctas(C, VEC, RHS0))
k_restrict_c(const float* __restrict__ u, const float* __restrict__ b, int w, int h,
             const uint8_t* __restrict__ cH, float* __restrict__ rH, int wH, int hH) {
    constexpr int ROWS = restrict_rows(C);
    const int X = blockIdx.x * 32 + threadIdx.x, Y = blockIdx.y * ROWS + threadIdx.y;
    if (X >= wH || Y >= hH) return;
    const size_t n = (size_t)w * h, nH = (size_t)wH * hH, P = (size_t)Y * wH + X;
    if (threadIdx.x == 0 && P + kRestrictAhead < nH)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(cH + P + kRestrictAhead));
    if (X < 1 || Y < 1 || 2 * X + 2 >= w || 2 * Y + 2 >= h) {
        for (int ch = 0; ch < C; ++ch)
            restrict_body<VEC, float, float, float, false>(u, b, RHS0, w, h, cH, rH, wH, hH,
                                                           blockIdx.x, blockIdx.y, ch);
        return;
    }
    if (cH[P]) {
        for (int ch = 0; ch < C; ++ch) rH[ch * nH + P] = 0.f;
        return;
    }
    auto pair = [](const float* p) {
        return VEC ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
    };
    float2 mid[C][4], rb[C][2];
    float l[C][2], r[C][2];
    const size_t at = (size_t)(2 * Y - 1) * w + 2 * X;  // row above the children, left child
#pragma unroll
    for (int ch = 0; ch < C; ++ch) {
        const float* p = u + ch * n + at;
#pragma unroll
        for (int j = 0; j < 4; ++j) mid[ch][j] = pair(p + (size_t)j * w);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            l[ch][j] = p[(size_t)(j + 1) * w - 1];
            r[ch][j] = p[(size_t)(j + 1) * w + 2];
            rb[ch][j] = make_float2(0.f, 0.f);
            if (!RHS0) rb[ch][j] = pair(b + ch * n + at + (size_t)(j + 1) * w);
        }
    }
#pragma unroll
    for (int ch = 0; ch < C; ++ch) {
        // the sums of restrict_body's interior path, in its order
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 up = mid[ch][j], ce = mid[ch][j + 1], dn = mid[ch][j + 2];
            const float l0 = 4.f * ce.x - (l[ch][j] + ce.y + up.x + dn.x);
            const float l1 = 4.f * ce.y - (ce.x + r[ch][j] + up.y + dn.y);
            sum += (RHS0 ? 0.f : rb[ch][j].x) - l0;
            sum += (RHS0 ? 0.f : rb[ch][j].y) - l1;
        }
        rH[ch * nH + P] = sum;
    }
}

template <bool VEC, class TU, class TB, class TO, bool F64, bool BESIDE = false>
__global__ void __launch_bounds__(256)
k_restrict(const TU* __restrict__ u, const TB* __restrict__ b, int rhs_zero,
           int w, int h, const uint8_t* __restrict__ cH, TO* __restrict__ rH, int wH,
           int hH) {
    restrict_body<VEC, TU, TB, TO, F64, BESIDE>(u, b, rhs_zero, w, h, cH, rH, wH, hH, blockIdx.x,
                                                blockIdx.y, blockIdx.z);
}

// Cell-centred bilinear prolongation.  A fine pixel takes 9/16 of its parent
// coarse cell, 3/16 of each of the two edge neighbours of the parent on the
// child's side and 1/16 of the diagonal one (coarse indices clamped at the
// border).  One thread per coarse cell (X, Y) and its up to 2x2 children:
// for the child row y = 2Y + dy the row blend takes coarse row Y three times
// and its neighbour on the child's side (Y - 1 for dy = 0, Y + 1 for dy = 1)
// once, the column blend the same with X - 1 (left child) or X + 1.
// mode 0: u = c ? b : P uH;  mode 1: u += c ? 0 : P uH (largest |P uH| over
// the updated pixels into *maxupd).  VEC: each child pair is one 8-byte word
// of u and b and one 2-byte word of c (w even, aligned base pointers; FP32 u).
// uH is stored as TC and u as TF (FP16/BF16 on the coarse levels in the
// 16-bit precision modes); b is FP32.
// The bilinear weights of one fine pixel: cc its parent coarse cell, cn the
// parent's vertical neighbour on the child's side, cs the horizontal one and
// csn the diagonal one; (3 (3 cc + cn) + (3 cs + csn)) / 16 with every
// rounding explicit, so that each kernel that prolongs gets the same bits.
__device__ __forceinline__ float prolong_blend(float cc, float cn, float cs, float csn) {
    const float vc = __fmaf_rn(3.f, cc, cn);
    const float vs = __fmaf_rn(3.f, cs, csn);
    return __fmul_rn(__fmaf_rn(3.f, vc, vs), 0.0625f);
}

template <bool VEC, class TC, class TF>
__device__ __forceinline__ void prolong_body(const TC* __restrict__ uH, int wH, int hH, const float* __restrict__ b,
          const uint8_t* __restrict__ c, int w, int h, TF* __restrict__ u, int mode,
          unsigned* __restrict__ maxupd, int bx, int by, int bz) {
    const int X = bx * blockDim.x + threadIdx.x;
    const int Y = by * blockDim.y + threadIdx.y;
    const int ch = bz;
    float amax = 0.f;
    if (X < wH && Y < hH) {
        const size_t n = (size_t)w * h, nH = (size_t)wH * hH;
        const TC* e = uH + ch * nH;
        const int Xl = max(X - 1, 0), Xr = min(X + 1, wH - 1);
        const TC* rc = e + (size_t)Y * wH;
        const TC* ru = e + (size_t)max(Y - 1, 0) * wH;
        const TC* rd = e + (size_t)min(Y + 1, hH - 1) * wH;
        const float cl = ldf(rc + Xl), cc = ldf(rc + X), cr = ldf(rc + Xr);
        const float ul = ldf(ru + Xl), uc = ldf(ru + X), ur = ldf(ru + Xr);
        const float dl = ldf(rd + Xl), dc = ldf(rd + X), dr = ldf(rd + Xr);
        const int x = 2 * X;
        TF* ucn = u + ch * n;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int y = 2 * Y + dy;
            if (y >= h) break;
            const float a0 = prolong_blend(cc, dy ? dc : uc, cl, dy ? dl : ul);
            const float a1 = prolong_blend(cc, dy ? dc : uc, cr, dy ? dr : ur);
            const size_t p = (size_t)y * w + x;
            if (VEC) {
                const uchar2 cm = *reinterpret_cast<const uchar2*>(c + p);
                float2* up = reinterpret_cast<float2*>(ucn + p);
                if (mode == 0) {
                    float2 bv = make_float2(0.f, 0.f);
                    if (cm.x | cm.y) bv = *reinterpret_cast<const float2*>(b + ch * n + p);
                    *up = make_float2(cm.x ? bv.x : a0, cm.y ? bv.y : a1);
                } else {
                    float2 uv = *up;
                    if (!cm.x) { uv.x = __fadd_rn(uv.x, a0); amax = fmaxf(amax, fabsf(a0)); }
                    if (!cm.y) { uv.y = __fadd_rn(uv.y, a1); amax = fmaxf(amax, fabsf(a1)); }
                    *up = uv;
                }
            } else {
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    if (x + dx >= w) break;
                    const float v = dx ? a1 : a0;
                    if (c[p + dx]) {
                        if (mode == 0) stf(ucn + p + dx, b[ch * n + p + dx]);
                    } else if (mode == 0) {
                        stf(ucn + p + dx, v);
                    } else {
                        stf(ucn + p + dx, __fadd_rn(ldf(ucn + p + dx), v));
                        amax = fmaxf(amax, fabsf(v));
                    }
                }
            }
        }
    }
    if (maxupd) {
        __shared__ float s_m[8];
        const int t = threadIdx.y * blockDim.x + threadIdx.x;
        amax = warp_max(amax);
        if ((t & 31) == 0) s_m[t >> 5] = amax;
        __syncthreads();
        if (t == 0) {
            float m = 0.f;
            for (int i = 0; i < (int)(blockDim.x * blockDim.y) / 32; ++i) m = fmaxf(m, s_m[i]);
            // most CTAs see a maximum already at least as large: skip their atomic
            if (m > __uint_as_float(*(volatile unsigned*)maxupd))
                atomicMax(maxupd, __float_as_uint(m));
        }
    }
}

template <bool VEC, class TC, class TF>
__global__ void __launch_bounds__(256)
k_prolong(const TC* __restrict__ uH, int wH, int hH, const float* __restrict__ b,
          const uint8_t* __restrict__ c, int w, int h, TF* __restrict__ u, int mode,
          unsigned* __restrict__ maxupd) {
    prolong_body<VEC, TC, TF>(uH, wH, hH, b, c, w, h, u, mode, maxupd, blockIdx.x, blockIdx.y,
                              blockIdx.z);
}

// keep == 0: u = c ? b : 0;  keep == 1: u = c ? b : u (a given iterate).
// u is stored as TU.
template <class TU>
__device__ __forceinline__ void select_body(const float* __restrict__ b, const uint8_t* __restrict__ c, size_t n,
                         TU* __restrict__ u, int keep, int bx, int nbx, int ch_) {
    const int ch = ch_;
    for (size_t i = (size_t)bx * blockDim.x + threadIdx.x; i < n;
         i += (size_t)nbx * blockDim.x) {
        if (c[i]) stf(u + ch * n + i, b[ch * n + i]);
        else if (!keep) stf(u + ch * n + i, 0.f);
    }
}

template <class TU>
__global__ void k_select(const float* __restrict__ b, const uint8_t* __restrict__ c, size_t n,
                         TU* __restrict__ u, int keep) {
    select_body<TU>(b, c, n, u, keep, blockIdx.x, gridDim.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// ORAS (Algorithm 2)
// ---------------------------------------------------------------------------

// ---- packed FP32 pairs (Blackwell f32x2 arithmetic) -------------------------
// A pair holds two horizontally adjacent pixels of one row (lo = even column).
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float lo2(f2 a) { return __uint_as_float((unsigned)(a & 0xffffffffull)); }
__device__ __forceinline__ float hi2(f2 a) { return __uint_as_float((unsigned)(a >> 32)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// r = b - ((deg) u_c - (up + down + left + right)) at one pixel; F64: in FP64
// (the finest-grid refinement residual), rounded once to FP32.
template <bool F64>
__device__ __forceinline__ float res_stencil(float b, float deg, float c, float up, float dn,
                                             float l, float r) {
    if (F64)
        return (float)((double)b - ((double)deg * (double)c -
                                    ((double)up + (double)dn + (double)l + (double)r)));
    return b - (deg * c - (up + dn + l + r));
}

// The same in FP64 from the negated degree nd.
__device__ __forceinline__ float res_f64(float b, float nd, float c, float up, float dn, float l,
                                         float r) {
    return res_stencil<true>(b, -nd, c, up, dn, l, r);
}

// Partition-of-unity weight of block k (of nb along an axis, stride s,
// overlap o) at local coordinate l (Section 3.1): 0 at the block's outermost
// overlap pixel, 1 at its innermost one, linear in between (1/2 for o = 1).
// The ramp end points are exact so that "weight == 1" and "weight == 0"
// agree with the integer classification of the combine pass.
__device__ __forceinline__ float ramp_weight(int l, int k, int nb, int s, int o, float inv_o1) {
    float wgt = 1.f;
    if (k > 0 && l < o)
        wgt *= (o == 1) ? 0.5f : (l == o - 1 ? 1.f : (float)l * inv_o1);
    if (k < nb - 1 && l >= s) {
        const int jj = l - s;
        wgt *= (o == 1) ? 0.5f : (jj == 0 ? 1.f : (jj == o - 1 ? 0.f : 1.f - (float)jj * inv_o1));
    }
    return wgt;
}

// Pixels shared by two blocks along one axis are the open interior of each
// overlap: local offsets 1 .. o-2 after the seam (o >= 3), or the single
// overlap pixel when o = 1.  nsh is their count per seam.
__host__ __device__ __forceinline__ int shared_per_seam(int o) { return o == 1 ? 1 : (o > 2 ? o - 2 : 0); }
__host__ __device__ __forceinline__ int shared_first(int o) { return o == 1 ? 0 : 1; }

// ---- asynchronous global -> shared copies (4-byte, zero fill) ----------------
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool ok) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    const int nbytes = ok ? 4 : 0;  // 0: nothing is read, the word is zero-filled
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sa), "l"(src), "r"(nbytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Bit-packed mask: row y, word k covers columns [32k, 32k + 32); bit set =
// known pixel or a column beyond the image.  wpr = words per row, including
// one padding word so that two consecutive words can always be read.  One
// warp per word (lane = column), four words in flight per warp, persistent
// warps; *unknown (nullable) gains the number of unknown pixels, with one
// atomic per CTA.
__device__ __forceinline__ void pack_mask_body(const uint8_t* __restrict__ c, int w, int h, uint32_t* __restrict__ bits, int wpr,
            unsigned long long* __restrict__ unknown, int bx, int nbx) {
    const int lane = threadIdx.x & 31;
    const int total = h * wpr;
    const int nwarps = (int)nbx * (int)(blockDim.x >> 5);
    unsigned unk = 0;
    for (int wid = (int)bx * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5);
         wid < total; wid += 4 * nwarps) {
        bool known[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int wk = wid + k * nwarps;
            known[k] = true;
            if (wk < total) {
                const int y = wk / wpr;
                const int x = 32 * (wk - y * wpr) + lane;
                known[k] = x >= w || c[(size_t)y * w + x] != 0;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int wk = wid + k * nwarps;
            const unsigned word = __ballot_sync(kFull, known[k]);
            if (wk < total) {  // warp-uniform
                if (lane == 0) bits[wk] = word;
                unk += (unsigned)__popc(~word);
            }
        }
    }
    if (unknown) {
        __shared__ unsigned s_u[8];
        if (lane == 0) s_u[threadIdx.x >> 5] = unk;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long a = 0;
            for (int i = 0; i < (int)(blockDim.x >> 5); ++i) a += s_u[i];
            if (a) atomicAdd(unknown, a);
        }
    }
}

__global__ void __launch_bounds__(256)
k_pack_mask(const uint8_t* __restrict__ c, int w, int h, uint32_t* __restrict__ bits, int wpr,
            unsigned long long* __restrict__ unknown) {
    pack_mask_body(c, w, h, bits, wpr, unknown, blockIdx.x, gridDim.x);
}

// The same for rows of whole 16-byte groups (w a multiple of 16, aligned
// base): a thread turns 16 mask bytes into half a word, and two threads make
// one.  3840x2160 (8.3 MB, 1.2 us at the copy rate): a byte per lane and a
// ballot per word, with a division per word, took 21.7 us; an iteration with
// its packing at that size went from 213 to 195 us.
__global__ void __launch_bounds__(256)
k_pack_mask16(const uint8_t* __restrict__ c, int w, int h, uint32_t* __restrict__ bits, int wpr,
              unsigned long long* __restrict__ unknown) {
    const int halves = 2 * wpr, groups = w >> 4;  // half words per row, those inside the image
    const int x = blockIdx.x * 32 + threadIdx.x;  // half word of the row
    unsigned unk = 0;
    const int y0 = ((int)blockIdx.y * 8 + (int)threadIdx.y) * 4;
    uint4 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
        if (x < groups && y0 + r < h)
            v[r] = __ldg(reinterpret_cast<const uint4*>(c + (size_t)(y0 + r) * w) + x);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        unsigned half = 0xffffu;
        if (x < groups && y0 + r < h) {
            // per byte 0 or 1, then the four flags of a word gathered at bit 24
            const unsigned f0 = __vminu4(v[r].x, 0x01010101u) * 0x01020408u;
            const unsigned f1 = __vminu4(v[r].y, 0x01010101u) * 0x01020408u;
            const unsigned f2_ = __vminu4(v[r].z, 0x01010101u) * 0x01020408u;
            const unsigned f3 = __vminu4(v[r].w, 0x01010101u) * 0x01020408u;
            half = ((f0 >> 24) & 15u) | ((f1 >> 20) & 0xf0u) | ((f2_ >> 16) & 0xf00u) |
                   ((f3 >> 12) & 0xf000u);
            unk += 16u - (unsigned)__popc(half);
        }
        const unsigned other = __shfl_xor_sync(kFull, half, 1);
        if (!(x & 1) && x < halves && y0 + r < h)
            bits[(size_t)(y0 + r) * wpr + (x >> 1)] = half | (other << 16);
    }
    if (unknown) {
        __shared__ unsigned s_u[8];
        const unsigned t = __reduce_add_sync(kFull, unk);
        if (threadIdx.x == 0) s_u[threadIdx.y] = t;
        __syncthreads();
        if (threadIdx.x == 0 && threadIdx.y == 0) {
            unsigned long long a = 0;
            for (int i = 0; i < 8; ++i) a += s_u[i];
            if (a) atomicAdd(unknown, a);
        }
    }
}

// One ORAS iteration, one warp per (block, channel) task.
//
// Lane layout: lane = (g, col), col = lane % B the block column and g the row
// group of R = B*B/32 rows; every CG vector is kept in registers as NP = R/2
// packed pairs, pair k = (row gR + k, row gR + k + NP) of the lane's column.
// Vertical neighbours of a pair are the neighbouring pairs (the first and the
// last pair swap one half with the other end of the column, and with the
// neighbouring row group through a shuffle); horizontal neighbours are the
// same pair of the neighbouring lanes (one 64-bit shuffle each way), with the
// block's outer columns cut by a 0/1 factor.  No shared memory and no barrier
// inside the CG loop.  Warps are persistent over a contiguous range of tasks
// (channel fastest, so the channels of one block are consecutive and share
// its mask bits and local operator); the next task's halo tile is fetched with
// cp.async while the current one is solved.
//
// Local problem (Section 3, Algorithm 2 step 2): plain CG on A_i v = R_i r
// from v = 0, A_i the rows of A for the block's unknown pixels with couplings
// to in-block neighbours only and alpha added to the diagonal for every
// in-image neighbour across the block edge (Robin), image edges reflecting.
// Vectors vanish on known pixels and outside the image, so the stencil reads
// neighbours unconditionally and only its result is masked.
template <int B>
struct WarpTile {
    static constexpr int G = 32 / B;       // row groups
    static constexpr int R = B / G;        // rows per lane
    static constexpr int NP = R / 2;       // packed pairs per lane
    static constexpr int TH = B + 2;       // tile side with the one-pixel halo
    static constexpr int P = B == 8 ? 12 : B + 2;  // tile pitch: row groups hit distinct banks
    static constexpr int TILE = TH * P;
    // per-warp shared memory (floats): two halo tiles, the 0/1 keep factors of
    // every pair (NP x 32 lanes x 2), the row weights (B), then optionally
    // two right-hand-side tiles (2 x B x B)
    static constexpr int KEEP = NP * 32 * 2;
    static constexpr int FIXED = 2 * TILE + KEEP + B;
};

template <int B>
__global__ void __launch_bounds__(32)
k_oras_warp(const float* __restrict__ u_in, int zero_in, const float* __restrict__ rhs,
            int rhs_zero, const uint32_t* __restrict__ mbits, int wpr, int w, int h, int C,
            int o, int nbx, int nby, float alpha, int iters, float rtol2,
            float* __restrict__ u_out, float* __restrict__ parked, unsigned* __restrict__ maxupd,
            int chan_inner, unsigned long long* __restrict__ step_count) {
    using WT = WarpTile<B>;
    constexpr int G = WT::G, R = WT::R, NP = WT::NP, TH = WT::TH, P = WT::P, TILE = WT::TILE;
    static_assert(G * B == 32 && R * G == B && NP * 2 == R, "warp shape");

    extern __shared__ float smem[];
    float* const s_u = smem;                                 // [2][TH][P]
    f2* const s_keep = reinterpret_cast<f2*>(smem + 2 * TILE);  // [NP][32] keep factors
    float* const s_wy = smem + 2 * TILE + WT::KEEP;          // [B] row weights of the block
    float* const s_b = smem + WT::FIXED;                     // [2][B][B], only when rhs_zero == 0

    const int lane = threadIdx.x;
    const int col = lane % B, g = lane / B;
    const int s = B - o;
    const size_t n = (size_t)w * h;
    const float inv_o1 = o > 1 ? 1.f / (float)(o - 1) : 0.f;

    // Task sequence of this warp.  chan_inner: blocks blockIdx.x, +gridDim.x,
    // ... each with all channels back to back (warps running together cover a
    // contiguous band of blocks, so halo re-reads hit L2, and a block's mask
    // bits and operator serve all its channels); otherwise (fewer blocks than
    // warps) tasks blockIdx.x, +gridDim.x, ... of the (block, channel) list.
    const int nblk = nbx * nby;
    auto task_of = [&](int i, int& blk, int& ch) {
        if (chan_inner) {
            blk = (int)blockIdx.x + (i / C) * (int)gridDim.x;
            ch = i % C;
        } else {
            const int t = (int)blockIdx.x + i * (int)gridDim.x;
            blk = t / C;
            ch = t - blk * C;
        }
        return blk < nblk;
    };

    // Issue the copies of task t into buffer `bs` (and the mask words of its
    // block into nlo/nhi when the block differs from `have_blk`).
    uint32_t nlo = 0xffffffffu, nhi = 0xffffffffu;
    auto prefetch = [&](int blk, int ch, int bs, int have_blk) {
        const int px0 = (blk % nbx) * s, py0 = (blk / nbx) * s;
        if (!zero_in) {
            // lane l copies tile column l of every row (and column 32 + l for
            // l < TH - 32); addresses advance by one image row per tile row
            const float* src = u_in + ch * n;
            float* dst = s_u + bs * TILE;
            const int gxa = px0 - 1 + lane, gxb = gxa + 32;
            const bool oka = lane < TH && gxa >= 0 && gxa < w;
            const bool okb = lane + 32 < TH && gxb < w;
            const float* row = src + (ptrdiff_t)(py0 - 1) * w;
#pragma unroll 2
            for (int ty = 0; ty < TH; ++ty, row += w) {
                const int gy = py0 - 1 + ty;
                const bool rok = gy >= 0 && gy < h;
                if (lane < TH) cp_async4(dst + ty * P + lane, (rok && oka) ? row + gxa : src, rok && oka);
                if (lane + 32 < TH) cp_async4(dst + ty * P + lane + 32, (rok && okb) ? row + gxb : src,
                                              rok && okb);
            }
        }
        if (!rhs_zero) {
            const float* src = rhs + ch * n;
            float* dst = s_b + bs * B * B;
#pragma unroll 4
            for (int e = lane; e < B * B; e += 32) {
                const int ly = e / B, lx = e - ly * B;
                const int gy = py0 + ly, gx = px0 + lx;
                const bool ok = gx < w && gy < h;
                cp_async4(dst + e, ok ? src + (size_t)gy * w + gx : src, ok);
            }
        }
        cp_async_commit();
        if (blk != have_blk && lane < B) {
            const int gy = py0 + lane;
            if (gy < h) {
                const uint32_t* row = mbits + (size_t)gy * wpr + (px0 >> 5);
                nlo = __ldg(row);
                nhi = __ldg(row + 1);
            } else {
                nlo = nhi = 0xffffffffu;
            }
        }
    };

    int blk, ch;
    if (!task_of(0, blk, ch)) return;  // warp-uniform
    prefetch(blk, ch, 0, -1);
    int buf = 0, cur_blk = -1;
    // per-block state
    uint32_t mb = 0;   // bit k: row gR + k of this lane's column is known or outside
    f2 ndg[NP];        // -(diagonal of A_i) per pair
    f2 ml2 = 0ull, mr2 = 0ull;  // 0/1: the left / right neighbour column is in the block
    float wx = 0.f, dh = 0.f;
    int x0 = 0, y0 = 0, bh = 0, kx = 0, ky = 0;
    float vmax = 0.f;
    unsigned nsteps = 0;  // completed local CG steps of this thread's tasks

    for (int i = 0;; ++i) {
        cp_async_wait_all();
        __syncwarp();
        const uint32_t mlo = nlo, mhi = nhi;
        int nblk_, nch;
        const bool more = task_of(i + 1, nblk_, nch);
        if (more) prefetch(nblk_, nch, buf ^ 1, blk);

        if (blk != cur_blk) {
            cur_blk = blk;
            kx = blk % nbx;
            ky = blk / nbx;
            x0 = kx * s;
            y0 = ky * s;
            const int bw = min(B, w - x0);
            bh = min(B, h - y0);
            // lane l < B holds the mask bits of block row l, columns x0 .. x0+31
            const uint32_t rowm = __funnelshift_r(mlo, mhi, x0 & 31);
            mb = 0;
#pragma unroll
            for (int rr = 0; rr < B; ++rr) {
                const uint32_t v = __shfl_sync(kFull, rowm, rr);
                const int k = rr - g * R;
                if (k >= 0 && k < R) mb |= ((v >> col) & 1u) << k;
            }
            const int gx = x0 + col;
            const float hc = (col > 0 ? 1.f : (gx > 0 ? alpha : 0.f)) +
                             (col + 1 < bw ? 1.f : (gx < w - 1 ? alpha : 0.f));
            dh = (float)((gx > 0) + (gx < w - 1));
            const float ml = col > 0 ? 1.f : 0.f, mr = col < B - 1 ? 1.f : 0.f;
            ml2 = pk(ml, ml);
            mr2 = pk(mr, mr);
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                float vc[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int ly = g * R + k + e * NP, gy = y0 + ly;
                    vc[e] = (ly > 0 ? 1.f : (gy > 0 ? alpha : 0.f)) +
                            (ly + 1 < bh ? 1.f : (gy < h - 1 ? alpha : 0.f));
                }
                ndg[k] = pk(-(hc + vc[0]), -(hc + vc[1]));
            }
            wx = ramp_weight(col, kx, nbx, s, o, inv_o1);
#pragma unroll
            for (int k = 0; k < NP; ++k)
                s_keep[k * 32 + lane] = pk(((mb >> k) & 1u) ? 0.f : 1.f,
                                          ((mb >> (k + NP)) & 1u) ? 0.f : 1.f);
            if (lane < B) s_wy[lane] = ramp_weight(lane, ky, nby, s, o, inv_o1);
            __syncwarp();
        }

        const float* tu = s_u + buf * TILE;
        const float* tb = s_b + buf * B * B;

        // initial residual r = R_i (b - A u), zero on known pixels
        f2 x[NP], r[NP], p[NP], q[NP];
        f2 acc0 = 0ull, acc1 = 0ull;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            float rv[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int ly = g * R + k + e * NP, gy = y0 + ly;
                float v = rhs_zero ? 0.f : tb[ly * B + col];
                if (!zero_in) {
                    const float* c0 = tu + (ly + 1) * P + col + 1;
                    const float dv = (float)((gy > 0) + (gy < h - 1));
                    v -= (dh + dv) * c0[0] - (c0[-P] + c0[P] + c0[-1] + c0[1]);
                }
                rv[e] = v;
            }
            r[k] = mul2(pk(rv[0], rv[1]), s_keep[k * 32 + lane]);
            p[k] = r[k];
            x[k] = 0ull;
            if (k & 1) acc1 = fma2(r[k], r[k], acc1);
            else acc0 = fma2(r[k], r[k], acc0);
        }
        acc0 = add2(acc0, acc1);
        float rr = warp_sum(lo2(acc0) + hi2(acc0));
        // rtol2 >= 0: relative stop (r.r <= max(rtol2, 1e-14) (r.r)_0); rtol2 < 0:
        // also stop once r.r <= -rtol2 (an absolute level, or the FP32 floor)
        const float rr_stop = rtol2 >= 0.f ? fmaxf(rtol2, 1e-14f) * rr
                                           : fmaxf(1e-14f * rr, -rtol2);

        for (int it = 0; it < iters; ++it) {
            if (!(rr > rr_stop)) break;  // rr is warp-uniform
            // the rows just above / below this lane's row group
            const float gu = __shfl_up_sync(kFull, hi2(p[NP - 1]), B);
            const float gd = __shfl_down_sync(kFull, lo2(p[0]), B);
            const f2 pu = pk(g > 0 ? gu : 0.f, lo2(p[NP - 1]));
            const f2 pd = pk(hi2(p[0]), g < G - 1 ? gd : 0.f);
            acc0 = 0ull;
            acc1 = 0ull;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const f2 left = __shfl_up_sync(kFull, p[k], 1, B);
                const f2 right = __shfl_down_sync(kFull, p[k], 1, B);
                const f2 up = k > 0 ? p[k - 1] : pu;
                const f2 dn = k < NP - 1 ? p[k + 1] : pd;
                f2 nbs = add2(up, dn);
                nbs = fma2(ml2, left, nbs);
                nbs = fma2(mr2, right, nbs);
                // -(A_i p), zero on known pixels
                const f2 qk = mul2(fma2(ndg[k], p[k], nbs), s_keep[k * 32 + lane]);
                q[k] = qk;
                if (k & 1) acc1 = fma2(p[k], qk, acc1);
                else acc0 = fma2(p[k], qk, acc0);
            }
            acc0 = add2(acc0, acc1);
            const float pq = -warp_sum(lo2(acc0) + hi2(acc0));
            if (!(pq > 0.f) || pq == INFINITY) break;
            const float a = __fdividef(rr, pq);
            const f2 a2 = pk(a, a);
            acc0 = 0ull;
            acc1 = 0ull;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                x[k] = fma2(a2, p[k], x[k]);
                r[k] = fma2(a2, q[k], r[k]);  // r - a A p
                if (k & 1) acc1 = fma2(r[k], r[k], acc1);
                else acc0 = fma2(r[k], r[k], acc0);
            }
            acc0 = add2(acc0, acc1);
            const float rrn = warp_sum(lo2(acc0) + hi2(acc0));
            const float beta = __fdividef(rrn, rr);
            rr = rrn;
            const f2 b2 = pk(beta, beta);
#pragma unroll
            for (int k = 0; k < NP; ++k) p[k] = fma2(b2, p[k], r[k]);
            ++nsteps;
        }

        // u_out = u_in + sum_i R_i^T D_i v_i: weight-1 pixels directly, the
        // weighted part of shared pixels parked in the block's tile for k_combine
        // (the first contributor of a shared pixel, smallest block index along
        // each shared axis, also carries u_in, so the combine pass only adds)
        const int nsh = shared_per_seam(o), first = shared_first(o);
        const bool xfirst = !(kx > 0 && col >= first && col < first + nsh);
        float* mine = parked + ((size_t)blk * C + ch) * (B * B) + col;
        float* uo = u_out + ch * n;
        const bool colok = x0 + col < w;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int ly = g * R + k + e * NP;
                if (ly >= bh || !colok) continue;
                const float v = e ? hi2(x[k]) : lo2(x[k]);
                const float d = wx * s_wy[ly];
                const float uold = zero_in ? 0.f : tu[(ly + 1) * P + col + 1];
                if (d == 1.f) {
                    uo[(size_t)(y0 + ly) * w + x0 + col] = uold + v;
                } else if (d > 0.f) {
                    const bool yfirst = !(ky > 0 && ly >= first && ly < first + nsh);
                    mine[ly * B] = (xfirst && yfirst) ? uold + d * v : d * v;
                }
                if (d > 0.f) vmax = fmaxf(vmax, fabsf(v));
            }
        }
        if (!more) break;
        blk = nblk_;
        ch = nch;
        buf ^= 1;
    }
    if (step_count && lane == 0) atomicAdd(step_count, (unsigned long long)nsteps);
    if (maxupd) {
        vmax = warp_max(vmax);
        if (lane == 0 && vmax > 0.f) atomicMax(maxupd, __float_as_uint(vmax));
    }
}

// One ORAS iteration for 32x32 blocks with two warps per block (warp wi owns
// rows 16wi .. 16wi+15), 16 pixels per thread.  Everything but the layout as in
// k_oras_warp.
//
// k_oras_2w_h (16-bit iterates): lane = block column; pair k of a lane = rows
// (16wi + k, 16wi + k + 8).  The FP32 kernels (k_oras_2w, k_batch_oras): see
// BlockThread.  The row pair at the seam (15 | 16) is exchanged through shared
// memory: each warp publishes its seam row of r with the r.r partial sum, and
// rebuilds the partner's seam row of p = r + beta p from it.  Two 64-thread
// barriers per CG step (p.Ap and r.r).
struct Tile2W {
    static constexpr int B = 32, TH = 34, P = 34, TILE = TH * P;
    // shared floats: two halo tiles, row weights, two rhs tiles (optional)
    static constexpr int FIXED = 2 * TILE + B;
};

// Shared-memory layout of the FP32 kernel (floats, from a 128-byte aligned
// base): two u tiles of TH rows with pitch PU (a 40-wide TMA box, or the
// 34-wide cp.async copy at column 1), the row weights, with a prolongation
// two patches of 18 x 18 coarse cells, then two right-hand side tiles of B
// rows with pitch PB (36-wide TMA box).  Tile strides are multiples of 128
// bytes, the alignment of a TMA destination.
struct Smem2W {
    static constexpr int B = 32, TH = 34, PU = 40, PB = 36;
    static constexpr int USTRIDE = 1376;            // >= TH * PU, 128-byte multiple
    static constexpr int BSTRIDE = B * PB;          // 1152 floats = 4608 bytes
    static constexpr int WY = 2 * USTRIDE;          // row weights (32 floats)
    static constexpr int RHS = WY + 32;             // 128-byte aligned
    static constexpr int EP = WY + 32;              // coarse patches (prolongation only)
    static constexpr int EW = 18, ES = EW * EW;     // patch side and cells
    static constexpr int EPW = 24, EH = 18;         // patch pitch (a 24-wide TMA box) and rows
    static constexpr int ESTRIDE = 448;             // >= EH * EPW, 128-byte multiple
    static constexpr int RHS_PRO = EP + 2 * ESTRIDE;
    static constexpr int TMA_E_BYTES = EH * EPW * 4;  // 1728
    static constexpr int TMA_U_BYTES = TH * PU * 4; // 5440
    static constexpr int TMA_B_BYTES = B * PB * 4;  // 4608
    static size_t bytes(bool rhs, bool pro = false) {
        return 128 + 4 * (size_t)((pro ? RHS_PRO : RHS) + (rhs ? 2 * BSTRIDE : 0));
    }
};

// ---- the local problem of a 32x32 block, FP32 (k_oras_2w, k_batch_oras) ------
//
// A thread owns two adjacent columns of eight rows: lane = 16 g + l, columns
// cl = 2l and 2l + 1, and the rows of lane group g of warp wi counted from r0
// in direction dr, so that local row 7 of the two groups of a warp are
// neighbours and local row 0 is the block's outer row (g = 0: rows 0.. and
// 31..) or the row at the warp seam (g = 1: rows 15.. and 16..).  A CG vector
// is eight packed pairs, pair 4c + k = local rows (k, k + 4) of column cl + c.
// Then half of the horizontal neighbours are the thread's own pairs (the other
// half one 64-bit shuffle within 16 lanes each), local row 8 is one 32-bit
// shuffle per column, local row -1 is the partner warp's seam row (kept as
// pb, zero for g = 0) and no select on the row group is left in the stencil: 28
// lane shuffles per warp and CG step, where the lane = column layout took 42
// and where shuffles and shared-memory accesses share one pipe.  Tile loads and
// the write of u are 8-byte words.  4K RGB, overlap 2: 13.6 us per CG step
// (lane = column layout: 16.0), 176 warp instructions per warp and step (221); a
// task without steps 612 (706), 937 with the prolongation.
struct BlockThread {
    int lane, wi, g, l;
    int cl;      // first of the two columns
    int r0, dr;  // block row of local row 0, direction
    __device__ __forceinline__ explicit BlockThread(int t) {
        lane = t & 31;
        wi = t >> 5;
        g = lane >> 4;
        l = lane & 15;
        cl = 2 * l;
        r0 = wi ? (g ? 16 : 31) : (g ? 15 : 0);
        dr = wi == g ? 1 : -1;
    }
};

// A_i on a thread's 16 pixels: -(diagonal) and the keep factors (0 on known
// pixels and off the image).  Blocks of full height have one diagonal per
// column but for local row 0, so d and e hold it; in blocks clipped by the
// image's lower edge d holds the horizontal part and s_nv the vertical one.
struct BlockOp {
    f2 d[2], e[2];   // per column: the pairs 1..3, pair 0
    f2 keep[8];
    f2 ml, mr;       // 0/1: the left / right neighbour column is in the block
    f2 nd;           // -(degree of A) of the two columns where both vertical neighbours exist
    bool full;       // full height
};

// rowm: in lane i < 16 the mask bits of block row 16 wi + i (columns x0 ..
// x0 + 31).
__device__ __forceinline__ void block_operator(BlockOp& op, const BlockThread& bt, uint32_t rowm,
                                               int x0, int y0, int bw, int bh, int w, int h,
                                               float alpha) {
    constexpr int B = 32;
    uint32_t kn = 0;
    const int src = bt.r0 - 16 * bt.wi;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t v = __shfl_sync(kFull, rowm, src + bt.dr * j) >> bt.cl;
        kn |= ((v & 1u) << j) | ((v & 2u) << (7 + j));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int b = 8 * (i >> 2) + (i & 3);
        op.keep[i] = pk(((kn >> b) & 1u) ? 0.f : 1.f, ((kn >> (b + 4)) & 1u) ? 0.f : 1.f);
    }
    const float ml = bt.l > 0 ? 1.f : 0.f, mr = bt.l < 15 ? 1.f : 0.f;
    op.ml = pk(ml, ml);
    op.mr = pk(mr, mr);
    op.full = bh == B;
    // vertical coupling of local row 0 in a block of full height
    const float v0 = bt.g ? 2.f
                          : 1.f + ((bt.wi == 0 ? y0 > 0 : y0 + B < h) ? alpha : 0.f);
    float dh[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int col = bt.cl + c, gx = x0 + col;
        dh[c] = (float)((gx > 0) + (gx < w - 1));
        const float hc = (col > 0 ? 1.f : (gx > 0 ? alpha : 0.f)) +
                         (col + 1 < bw ? 1.f : (gx < w - 1 ? alpha : 0.f));
        const float d = op.full ? -(hc + 2.f) : -hc;
        op.d[c] = pk(d, d);
        op.e[c] = pk(-(hc + v0), d);
    }
    op.nd = pk(-(dh[0] + 2.f), -(dh[1] + 2.f));
}
// The vertical part of a clipped block's diagonal into s_nv (16 pairs), read in
// block_cg after its first barrier; called after the barrier that ends the
// previous task's reads.
__device__ __forceinline__ void clipped_diagonal(const BlockThread& bt, int y0, int bh, int h,
                                                 float alpha, f2* s_nv) {
    if (bt.l >= 4) return;
    float vc[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int ly = bt.r0 + bt.dr * (bt.l + 4 * e), gy = y0 + ly;
        vc[e] = (ly > 0 ? 1.f : (gy > 0 ? alpha : 0.f)) +
                (ly + 1 < bh ? 1.f : (gy < h - 1 ? alpha : 0.f));
    }
    s_nv[(2 * bt.wi + bt.g) * 4 + bt.l] = pk(-vc[0], -vc[1]);
}

// Two adjacent words of a tile; EVEN: at an 8-byte boundary.
template <bool EVEN>
__device__ __forceinline__ f2 ld_pair(const float* p) {
    if (EVEN) return *reinterpret_cast<const f2*>(p);
    return pk(p[0], p[1]);
}

// r = b - A u on the block (0 on known pixels).  tc: the tile's word of local
// row 0, column cl (pitch folded into ts = dr * pitch); bc, bs: the same of the
// right-hand side tile (RHS0: 0 off the mask); INT: no row of the block on the
// image's top or bottom row, so every vertical degree is 2.  A thread walks its
// columns, so a row's centre is the next row's neighbour; the two columns of a
// row are a packed pair until the masked result goes to its CG pairs.  (A zero
// iterate is a tile of zeros: zero_tiles.)
template <bool F64, bool RHS0, bool INT, bool EVEN>
__device__ __forceinline__ void block_residual(f2 (&r)[8], const BlockOp& op,
                                               const BlockThread& bt, const float* tc, int ts,
                                               const float* bc, int bs, int y0, int h) {
    f2 rv[8];
    f2 up = ld_pair<EVEN>(tc - ts), cen = ld_pair<EVEN>(tc);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        f2 v = 0ull;
        if (!RHS0) {
            v = ld_pair<EVEN>(bc);
            bc += bs;
        }
        const float l = tc[-1], rt = tc[2];
        tc += ts;
        const f2 dn = ld_pair<EVEN>(tc);
        f2 nd = op.nd;
        if (!INT) {
            const int gy = y0 + bt.r0 + bt.dr * j;
            const float e = (float)((gy == 0) + (gy == h - 1));
            nd = add2(nd, pk(e, e));
        }
        if (F64) {
            const float b0 = lo2(v), b1 = hi2(v);
            v = pk(res_f64(b0, lo2(nd), lo2(cen), lo2(up), lo2(dn), l, hi2(cen)),
                   res_f64(b1, hi2(nd), hi2(cen), hi2(up), hi2(dn), lo2(cen), rt));
        } else {
            const f2 nb = add2(add2(up, dn), pk(l + hi2(cen), lo2(cen) + rt));
            const f2 t = fma2(nd, cen, nb);  // -(A u)
            v = RHS0 ? t : add2(v, t);
        }
        up = cen;
        cen = dn;
        rv[j] = v;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        r[k] = pk(lo2(rv[k]) * lo2(op.keep[k]), lo2(rv[k + 4]) * hi2(op.keep[k]));
        r[4 + k] = pk(hi2(rv[k]) * lo2(op.keep[4 + k]), hi2(rv[k + 4]) * hi2(op.keep[4 + k]));
    }
}

// Shared words of block_cg.
struct BlockShared {
    float red1[2], red2[2];
    float2 seam[2][16];
    f2 nv[16];
};

// a / b for normal b > 0: one approximate reciprocal (both warps of a block
// compute it from the same words, so they agree).  0 for b > 2^126, as with a
// fast division.
__device__ __forceinline__ float quotient(float a, float b) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
    return a * r;
}

// Residuals with 0 < r.r < kTinyNorm2 are solved scaled by kTinyScale, their
// solution scaled back: both powers of two, so the local solve of a scaled image
// has the bits of the image's own (until r.r is 0: |r| below 2^-75).  Without it
// r.r and p.Ap of values of 1e-17 and less would underflow before the relative
// stop (1e-14 of the first r.r) is reached.  Squares of kTinyScale times such a
// residual stay below 2^96.  The test costs the 4K RGB iteration 1 us of 187.
constexpr float kTinyNorm2 = 0x1p-64f, kTinyScale = 0x1p80f;
__device__ __forceinline__ bool tiny_residual(float rr, float rtol2) {
    // 0 < rr < kTinyNorm2 (blocks without unknown pixels have rr = 0), and not
    // stopped at once
    return __float_as_uint(rr) - 1u < __float_as_uint(kTinyNorm2) - 1u &&
           !(rtol2 < 0.f && rr <= -rtol2);
}
// -rtol2 (an absolute level of r.r) of a residual scaled by kTinyScale.
__device__ __forceinline__ float tiny_rtol2(float rtol2) {
    return rtol2 < 0.f ? (rtol2 * kTinyScale) * kTinyScale : rtol2;
}

// Sum over a warp of the two-warp form, the row groups last, so that the
// four-warp form (a warp per row group) adds in the same order.
__device__ __forceinline__ float warp_sum_block(float v) {
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
    return v + __shfl_xor_sync(kFull, v, 16);
}

// Up to `iters` CG steps on A_i x = r from x = 0 (r is overwritten); both
// warps of the block.  rtol2 >= 0: relative stop (r.r <= max(rtol2, 1e-14)
// (r.r)_0); rtol2 < 0: also stop once r.r <= -rtol2 (an absolute level, or the
// FP32 floor).  Tiny residuals are scaled (kTinyScale).  The last step updates
// x alone.  Returns the completed steps.
// Bound by the register file: an instruction takes half a cycle per 32-bit
// operand word it reads (a packed FMA of three distinct pairs 3 cycles, an
// add 2, a scalar add 1), which is why nothing here trades fewer
// instructions for more operands, and more warps per SM do not help.
template <bool FULL>
__device__ __forceinline__ unsigned block_cg_t(f2 (&x)[8], f2 (&r)[8], const BlockOp& op,
                                               const BlockThread& bt, int iters, float rtol2,
                                               BlockShared& sh) {
    f2 p[8], q[8];
    f2 acc0, acc1;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        p[i] = r[i];
        x[i] = 0ull;
        if (i == 0) acc0 = mul2(r[i], r[i]);
        else if (i == 4) acc1 = mul2(r[i], r[i]);
        else if (i < 4) acc0 = fma2(r[i], r[i], acc0);
        else acc1 = fma2(r[i], r[i], acc1);
    }
    acc0 = add2(acc0, acc1);
    if (bt.g) sh.seam[bt.wi][bt.l] = make_float2(lo2(r[0]), lo2(r[4]));
    float part = warp_sum_block(lo2(acc0) + hi2(acc0));
    if (bt.lane == 0) sh.red2[bt.wi] = part;
    __syncthreads();
    float rr = sh.red2[0] + sh.red2[1];
    float2 pb = make_float2(0.f, 0.f);  // local row -1 of p
    if (bt.g) pb = sh.seam[bt.wi ^ 1][bt.l];
    const bool tiny = tiny_residual(rr, rtol2);
    if (tiny) {  // the same in both warps
        const f2 up = pk(kTinyScale, kTinyScale);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            r[i] = mul2(r[i], up);
            p[i] = r[i];
            if (i == 0) acc0 = mul2(r[i], r[i]);
            else if (i == 4) acc1 = mul2(r[i], r[i]);
            else if (i < 4) acc0 = fma2(r[i], r[i], acc0);
            else acc1 = fma2(r[i], r[i], acc1);
        }
        acc0 = add2(acc0, acc1);
        part = warp_sum_block(lo2(acc0) + hi2(acc0));
        if (bt.lane == 0) sh.red1[bt.wi] = part;
        __syncthreads();
        rr = sh.red1[0] + sh.red1[1];
        __syncthreads();  // the first step writes red1
        pb.x *= kTinyScale;
        pb.y *= kTinyScale;
        rtol2 = tiny_rtol2(rtol2);
    }
    // never below the smallest normal, so that the quotients stay finite
    const float rr_stop = fmaxf(rtol2 >= 0.f ? fmaxf(rtol2, 1e-14f) * rr : fmaxf(1e-14f * rr, -rtol2),
                                FLT_MIN);
    const f2* nv = sh.nv + (2 * bt.wi + bt.g) * 4;
    int it = 0;
    while (it < iters && rr > rr_stop) {  // rr is identical in both warps
        const float dn0 = __shfl_xor_sync(kFull, hi2(p[3]), 16);  // local row 8
        const float dn1 = __shfl_xor_sync(kFull, hi2(p[7]), 16);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const f2 left = __shfl_up_sync(kFull, p[4 + k], 1, 16);
            const f2 right = __shfl_down_sync(kFull, p[k], 1, 16);
            // vertical neighbours: local row -1 is the partner's, local row 8 the
            // other row group's (their pairs as two scalar sums: packing the
            // halves first takes more instructions)
            f2 n0, n1;
            if (k == 0) {
                n0 = pk(pb.x + lo2(p[1]), lo2(p[3]) + hi2(p[1]));
                n1 = pk(pb.y + lo2(p[5]), lo2(p[7]) + hi2(p[5]));
            } else if (k == 3) {
                n0 = pk(lo2(p[2]) + hi2(p[0]), hi2(p[2]) + dn0);
                n1 = pk(lo2(p[6]) + hi2(p[4]), hi2(p[6]) + dn1);
            } else {
                n0 = add2(p[k - 1], p[k + 1]);
                n1 = add2(p[3 + k], p[5 + k]);
            }
            n0 = add2(n0, p[4 + k]);
            n1 = add2(n1, p[k]);
            n0 = fma2(op.ml, left, n0);
            n1 = fma2(op.mr, right, n1);
            f2 g0, g1;
            if (FULL) {
                g0 = k ? op.d[0] : op.e[0];
                g1 = k ? op.d[1] : op.e[1];
            } else {
                const f2 v = nv[k];
                g0 = add2(v, op.d[0]);
                g1 = add2(v, op.d[1]);
            }
            // -(A_i p), 0 on the mask
            q[k] = mul2(fma2(g0, p[k], n0), op.keep[k]);
            q[4 + k] = mul2(fma2(g1, p[4 + k], n1), op.keep[4 + k]);
            acc0 = k ? fma2(p[k], q[k], acc0) : mul2(p[k], q[k]);
            acc1 = k ? fma2(p[4 + k], q[4 + k], acc1) : mul2(p[4 + k], q[4 + k]);
        }
        acc0 = add2(acc0, acc1);
        part = warp_sum_block(lo2(acc0) + hi2(acc0));
        if (bt.lane == 0) sh.red1[bt.wi] = part;
        __syncthreads();
        const float pq = -(sh.red1[0] + sh.red1[1]);
        if (!(pq >= FLT_MIN && pq <= FLT_MAX)) break;
        const float a = quotient(rr, pq);
        const f2 a2 = pk(a, a);
        if (++it == iters) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = fma2(a2, p[i], x[i]);
            break;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            x[i] = fma2(a2, p[i], x[i]);
            r[i] = fma2(a2, q[i], r[i]);
            if (i == 0) acc0 = mul2(r[i], r[i]);
            else if (i == 4) acc1 = mul2(r[i], r[i]);
            else if (i < 4) acc0 = fma2(r[i], r[i], acc0);
            else acc1 = fma2(r[i], r[i], acc1);
        }
        acc0 = add2(acc0, acc1);
        if (bt.g) sh.seam[bt.wi][bt.l] = make_float2(lo2(r[0]), lo2(r[4]));
        part = warp_sum_block(lo2(acc0) + hi2(acc0));
        if (bt.lane == 0) sh.red2[bt.wi] = part;
        __syncthreads();
        const float rrn = sh.red2[0] + sh.red2[1];
        const float beta = quotient(rrn, rr);
        rr = rrn;
        const f2 b2 = pk(beta, beta);
#pragma unroll
        for (int i = 0; i < 8; ++i) p[i] = fma2(b2, p[i], r[i]);
        if (bt.g) {
            const float2 sv = sh.seam[bt.wi ^ 1][bt.l];
            pb.x = fmaf(beta, pb.x, sv.x);
            pb.y = fmaf(beta, pb.y, sv.y);
        }
    }
    if (tiny) {
        const f2 down = pk(1.f / kTinyScale, 1.f / kTinyScale);
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = mul2(x[i], down);
    }
    return (unsigned)it;
}
__device__ __forceinline__ unsigned block_cg(f2 (&x)[8], f2 (&r)[8], const BlockOp& op,
                                             const BlockThread& bt, int iters, float rtol2,
                                             BlockShared& sh) {
    return op.full ? block_cg_t<true>(x, r, op, bt, iters, rtol2, sh)
                   : block_cg_t<false>(x, r, op, bt, iters, rtol2, sh);
}

// Overlap 2: bit j of the local rows whose weight is 1 (all but a block edge
// inside the image) and that lie in the image.
__device__ __forceinline__ uint32_t own_rows(const BlockThread& bt, int ky, int nby, int bh) {
    uint32_t m = bt.g || (bt.wi == 0 ? ky == 0 : ky == nby - 1) ? 0xffu : 0xfeu;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (bt.r0 + bt.dr * j >= bh) m &= ~(1u << j);
    return m;
}

// Local row j of column c of a solution.
__device__ __forceinline__ float block_value(const f2 (&x)[8], int c, int j) {
    return j < 4 ? lo2(x[4 * c + j]) : hi2(x[4 * c + j - 4]);
}

// Stores under a predicate (written out: left to the compiler they become
// branches around each store).
__device__ __forceinline__ void st_if(bool ok, float* p, float a) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t"
                 "@p st.global.f32 [%0], %1;\n\t}" ::"l"(p), "f"(a), "r"((unsigned)ok) : "memory");
}
__device__ __forceinline__ void st_pair_if(bool ok, float* p, float a, float b) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
                 "@p st.global.v2.f32 [%0], {%1, %2};\n\t}"
                 ::"l"(p), "f"(a), "f"(b), "r"((unsigned)ok) : "memory");
}

// What a block of weight d stores of a pixel: u_in + v where the pixel is its
// own (d = 1), its weighted part elsewhere, the first contributor's (which a
// weight of 1 implies) with u_in.  Every rounding explicit, so that each block
// kernel gets the same bits.
__device__ __forceinline__ float shared_part(float d, float v, float u, bool first) {
    return __fmaf_rn(d, v, first ? u : 0.f);
}

// The tiles of a launch whose iterate is zero, which no copy fills: zeros, so
// that the code of every task is the same (the tests per row in the residual and
// the write were 24 branches and 92 of 690 instructions of a task without CG
// steps: decode of 4K RGB 1571 -> 1513 us, four in flight 4740 -> 4540).
__device__ __forceinline__ void zero_tiles(float* s_u, int t, int nt) {
    for (int i = t; i < 2 * Smem2W::USTRIDE; i += nt) s_u[i] = 0.f;
}

// The write of 0/1 weights (overlap 2): each pixel is written by the one block
// whose weight is 1 there, with u_in (the tile) added.  up: u_out
// at local row 0, column cl; us: its step to the next local row; own0, own1:
// the columns are the block's own; rows: bit j of a local row j of its own
// (ALL: rows 1 .. 7 are); VEC: up is at an 8-byte boundary in every row.  vmax
// gains the largest |x| written.  A lane with one column of its own stores a
// word, the others two, without a branch on it.
template <bool ALL, bool VEC>
__device__ __forceinline__ void block_write01_t(const f2 (&x)[8], const float* tc, int ts,
                                                float* up, ptrdiff_t us, bool own0, bool own1,
                                                uint32_t rows, float& vmax) {
    const bool two = own0 && own1, one = own0 != own1;
    float m0 = 0.f, m1 = 0.f;
    const int oc = own0 ? 0 : 1;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool ok = (ALL && j > 0) || ((rows >> j) & 1u);
        const float v0 = block_value(x, 0, j), v1 = block_value(x, 1, j);
        const f2 u = ld_pair<true>(tc);
        const float a = lo2(u) + v0, b = hi2(u) + v1;
        if (VEC) {
            if (ok && two) *reinterpret_cast<f2*>(up) = pk(a, b);
            if (ok && one) up[oc] = own0 ? a : b;
        } else {
            if (ok && own0) up[0] = a;
            if (ok && own1) up[1] = b;
        }
        if (ok) {
            m0 = fmaxf(m0, fabsf(v0));
            m1 = fmaxf(m1, fabsf(v1));
        }
        tc += ts;
        up += us;
    }
    if (own0) vmax = fmaxf(vmax, m0);
    if (own1) vmax = fmaxf(vmax, m1);
}
__device__ __forceinline__ void block_write01(const f2 (&x)[8], bool all, const float* tc, int ts,
                                              float* up, ptrdiff_t us, bool own0, bool own1,
                                              uint32_t rows, bool vec, float& vmax) {
    if (all && vec) block_write01_t<true, true>(x, tc, ts, up, us, own0, own1, rows, vmax);
    else if (vec) block_write01_t<false, true>(x, tc, ts, up, us, own0, own1, rows, vmax);
    else block_write01_t<false, false>(x, tc, ts, up, us, own0, own1, rows, vmax);
}

// The start of an iteration formed by prolongation inside a block's tile
// (Section 4.4's cell-centred weights): the thread's 16 pixels (x0 and y0 are
// even: columns cl and cl + 1 have the same parent, and local rows 2m, 2m + 1
// too; the even local row takes the coarse row before it in the thread's
// direction, the odd one the row after it), then the halo pixels the residual
// reads: warp 0 the row above the block and the column left of it, warp 1 the
// row below and the column right of it, one pixel of each per lane (block
// pixels of a neighbouring block, which counts them in the maximum).  pe: the
// block's coarse patch (cell (r, q) = coarse row y0 / 2 - 1 + r, column x0 / 2
// - 1 + q, pitch Smem2W::EPW, clamped to the level); hk: bits of the thread's
// two halo pixels (known or off the image).  ADD:
// u + P e at unknown pixels (a correction), else P e there (an interpolated
// solution); known pixels keep their tile value.  tw: the tile's word of the
// halo corner.  pmax gains the largest |P e| over the unknown block pixels.
// Branch-free (every patch index stays inside the patch); the patch rows and
// the tile values are read before anything is stored (the stores could alias
// them otherwise), so the loads are in flight together.
template <bool ADD>
__device__ __forceinline__ void prolong_into_tile(float* tw, const float* pe,
                                                  const BlockThread& bt, const BlockOp& op,
                                                  uint32_t hk, float& pmax) {
    constexpr int EW = Smem2W::EPW, P = Smem2W::PU, B = 32;
    {
        const int q = 1 + bt.l, es = bt.dr * EW, ts = bt.dr * P;
        const float* pr = pe + (1 + (bt.r0 >> 1)) * EW + q - es;  // row before the first parent
        float* tc = tw + (bt.r0 + 1) * P + bt.cl + 1;
        float el[6], ec[6], er[6];
        f2 tv[8];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            el[i] = pr[-1];
            ec[i] = pr[0];
            er[i] = pr[1];
            pr += es;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) tv[j] = ld_pair<true>(tc + j * ts);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = 1 + (j >> 1), n = (j & 1) ? i + 1 : i - 1;
            // unknown: the keep factor of the pixel is not 0
            const f2 kp0 = op.keep[j & 3], kp1 = op.keep[4 + (j & 3)];
            const bool u0 = (j < 4 ? lo2(kp0) : hi2(kp0)) != 0.f;
            const bool u1 = (j < 4 ? lo2(kp1) : hi2(kp1)) != 0.f;
            const float b0 = prolong_blend(ec[i], ec[n], el[i], el[n]);
            const float b1 = prolong_blend(ec[i], ec[n], er[i], er[n]);
            const float a0 = u0 ? b0 : 0.f, a1 = u1 ? b1 : 0.f;
            const float t0 = lo2(tv[j]), t1 = hi2(tv[j]);
            *reinterpret_cast<f2*>(tc + j * ts) =
                ADD ? pk(__fadd_rn(t0, a0), __fadd_rn(t1, a1)) : pk(u0 ? a0 : t0, u1 ? a1 : t1);
            pmax = fmaxf(pmax, fmaxf(fabsf(a0), fabsf(a1)));
        }
    }
    // x0 and y0 are even, so the parent cell of a halo pixel and the side of
    // its neighbours depend on the thread alone
    const int odd = bt.lane & 1, half = 1 + (bt.lane >> 1), far = bt.wi ? B / 2 + 1 : 0;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const float* pp = pe + (side == 0 ? far * EW + half : half * EW + far);
        // to the neighbour across the block's edge and along it
        const int in = (side == 0 ? EW : 1) * (bt.wi ? -1 : 1);
        const int al = (side == 0 ? 1 : EW) * (odd ? 1 : -1);
        const int vn = side == 0 ? in : al, hn = side == 0 ? al : in;
        const float a = prolong_blend(pp[0], pp[vn], pp[hn], pp[vn + hn]);
        float* tp = tw + (side == 0 ? (bt.wi ? (B + 1) * P : 0) + bt.lane + 1
                                    : (bt.lane + 1) * P + (bt.wi ? B + 1 : 0));
        const bool kn = (hk >> side) & 1u;  // known or off the image
        const float old = *tp;
        *tp = kn ? old : (ADD ? __fadd_rn(old, a) : a);
    }
}

// The coarse cells a task's prolongation reads, by 4-byte cp.async (all nt
// threads): rows (py0 >> 1) - 1 + r and columns (px0 >> 1) - 1 + q, r, q <
// 18, each clamped to the level as the prolongation clamps its indices,
// into dst with pitch Smem2W::EPW.  The caller commits the group.
__device__ __forceinline__ void copy_patch_clamped(float* dst, const float* e, int px0, int py0,
                                                   int wH, int hH, int t, int nt = 64) {
    const int Ys = (py0 >> 1) - 1, Xs = (px0 >> 1) - 1;
    for (int i = t; i < Smem2W::ES; i += nt) {
        const int r = i / Smem2W::EW, q = i - r * Smem2W::EW;
        const int Y = min(max(Ys + r, 0), hH - 1), X = min(max(Xs + q, 0), wH - 1);
        cp_async4(dst + r * Smem2W::EPW + q, e + (size_t)Y * wH + X, true);
    }
}

// Known bits of a thread's two halo pixels for prolong_into_tile (bit set:
// known or off the image).
__device__ __forceinline__ uint32_t halo_known_bits(const uint32_t* __restrict__ mbits, int wpr,
                                                    int w, int h, int px0, int py0, int wi,
                                                    int lane) {
    constexpr int B = 32;
    const int hy0 = wi == 0 ? py0 - 1 : py0 + B, hx0 = px0 + lane;
    const int hy1 = py0 + lane, hx1 = wi == 0 ? px0 - 1 : px0 + B;
    uint32_t k = 3u;
    if (hx0 >= 0 && hx0 < w && hy0 >= 0 && hy0 < h &&
        !((__ldg(mbits + (size_t)hy0 * wpr + (hx0 >> 5)) >> (hx0 & 31)) & 1u))
        k &= ~1u;
    if (hx1 >= 0 && hx1 < w && hy1 >= 0 && hy1 < h &&
        !((__ldg(mbits + (size_t)hy1 * wpr + (hx1 >> 5)) >> (hx1 & 31)) & 1u))
        k &= ~2u;
    return k;
}

// Bounded wait for phase `parity` of the mbarrier at shared address `bar`;
// false if it did not complete within the limit.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, int limit = 1 << 20) {
    for (int n = 0; n < limit; ++n) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Self test of the bounded wait: one CTA waits on an mbarrier that no thread
// and no copy ever completes.  *flag = 1 when the wait runs out (the expected
// outcome; the CTA then leaves normally, nothing is in flight), 2 if it
// completed.
__global__ void k_bounded_wait_selftest(unsigned* __restrict__ flag, int limit) {
    __shared__ __align__(8) unsigned long long bar;
    const unsigned a = (unsigned)__cvta_generic_to_shared(&bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const bool ok = mbar_wait(a, 0u, limit);
    const int any_out = __syncthreads_or(!ok);
    if (threadIdx.x == 0) *flag = any_out ? 1u : 2u;
}

// 3-D tiled TMA load of one box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int x, int y,
                                            int z, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];"
        :
        : "r"(dst), "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z),
          "r"(bar)
        : "memory");
}

// use_tma: the tiles come by TMA (tm_u over u_in, tm_b over rhs, both FP32
// [C][h][w] with w a multiple of 4); otherwise by 4-byte cp.async.  errflag:
// set to 1 if a TMA wait ran out (the CTA then stops).  use_tma_e (only with
// use_tma): the coarse patches of PRO come by TMA too (tm_e over eH).
// PRO = 1: the iteration starts from u_in + P eH instead of u_in, the coarse
// correction eH [C][hH][wH] prolonged as prolong_body does in mode 1 (added
// at unknown pixels only), so that the V-cycle's correction step needs no
// launch and no pass over the fine iterate of its own; the largest |P eH|
// over the unknown pixels goes to *maxpro.  PRO = 2: the start is u_in at
// the known pixels and P eH at the unknown ones (prolong_body's mode 0 with
// u_in as b: the cascade's interpolation of the coarser level's solution).
// Each block forms the start in its tile (block pixels and halo) before the
// residual.  PRO needs u_in (not zero_in) and an even block stride, so that the
// parity of a block pixel is that of its tile index.  OV: 0 overlap 2 (partition
// weights 0 and 1); blocks share pixels (overlap 1 or >= 3) and 1 the block
// stride 32 - o is even, 2 odd (block columns at odd pixels: no 8-byte words).
template <bool F64, int PRO, int OV>
__global__ void __launch_bounds__(64, 8)
k_oras_2w(const float* __restrict__ u_in, int zero_in, const float* __restrict__ rhs,
          int rhs_zero, const uint32_t* __restrict__ mbits, int wpr, int w, int h, int C, int o,
          int nbx, int nby, float alpha, int iters, float rtol2, float* __restrict__ u_out,
          float* __restrict__ parked, unsigned* __restrict__ maxupd, int chan_inner,
          const __grid_constant__ CUtensorMap tm_u, const __grid_constant__ CUtensorMap tm_b,
          int use_tma, unsigned* __restrict__ errflag,
          unsigned long long* __restrict__ step_count, const float* __restrict__ eH, int wH,
          int hH, unsigned* __restrict__ maxpro, const __grid_constant__ CUtensorMap tm_e,
          int use_tma_e) {
    constexpr int B = 32, TH = Smem2W::TH, P = Smem2W::PU, PB = Smem2W::PB;
    constexpr int TILE = Smem2W::USTRIDE;
    extern __shared__ float smem_raw[];
    float* const smem = reinterpret_cast<float*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    float* const s_u = smem;                     // [2][USTRIDE]
    float* const s_wy = smem + Smem2W::WY;       // [B]
    float* const s_e = smem + Smem2W::EP;        // [2][ES] if PRO
    float* const s_b = smem + (PRO ? Smem2W::RHS_PRO : Smem2W::RHS);  // [2][BSTRIDE] if rhs_zero == 0
    __shared__ BlockShared sh;
    __shared__ __align__(8) unsigned long long s_bar[2];

    const int t = threadIdx.x;
    const BlockThread bt(t);
    const int lane = bt.lane, wi = bt.wi;
    const int s = B - o;
    const size_t n = (size_t)w * h;
    const float inv_o1 = o > 1 ? 1.f / (float)(o - 1) : 0.f;
    // Task sequence of this CTA.  chan_inner: blocks blockIdx.x, +gridDim.x,
    // ... each with all channels back to back (the CTAs running together cover
    // a contiguous band of blocks, so halo re-reads hit L2, and a block's mask
    // bits and operator serve all its channels); otherwise (fewer blocks than
    // CTA slots) tasks blockIdx.x, +gridDim.x, ... of the (block, channel) list.
    const int nblk = nbx * nby;
    // the task after (blk, ch) in this CTA's sequence (no division on the
    // channel-inner path, which the large levels take)
    auto next_task = [&](int& blk, int& ch) {
        if (chan_inner) {
            if (++ch == C) { ch = 0; blk += (int)gridDim.x; }
        } else {
            const int tt = blk * C + ch + (int)gridDim.x;
            blk = tt / C;
            ch = tt - blk * C;
        }
        return blk < nblk;
    };
    uint32_t nlo = 0xffffffffu, nhi = 0xffffffffu;
    uint32_t nhk = 3u;  // PRO: bit i = halo pixel i of this thread (next block) is known or off the image
    int px0 = 0, py0 = 0;  // origin of the block prefetched last
    auto prefetch = [&](int blk, int ch, int bs, int have_blk) {
        if (blk != have_blk) {
            py0 = blk / nbx;
            px0 = (blk - py0 * nbx) * s;
            py0 *= s;
        }
        if constexpr (PRO != 0) {
            // the coarse cells the task's prolongation reads: rows
            // (py0 >> 1) - 1 + r and columns (px0 >> 1) - 1 + q, r, q < 18
            // (with TMA, the box issued below; here each cell is clamped to
            // the level as the prolongation clamps its indices)
            if (!use_tma_e) {
                copy_patch_clamped(s_e + bs * Smem2W::ESTRIDE, eH + (size_t)ch * wH * hH, px0,
                                   py0, wH, hH, t);
                cp_async_commit();
            }
            // this thread's two halo pixels (see the prolongation below)
            if (blk != have_blk) nhk = halo_known_bits(mbits, wpr, w, h, px0, py0, wi, lane);
        }
        if (use_tma) {
            if (t == 0) {
                const unsigned bar =
                    (unsigned)__cvta_generic_to_shared(&s_bar[bs]);
                const unsigned bytes = (zero_in ? 0u : (unsigned)Smem2W::TMA_U_BYTES) +
                                       (rhs_zero ? 0u : (unsigned)Smem2W::TMA_B_BYTES) +
                                       (PRO != 0 && use_tma_e ? (unsigned)Smem2W::TMA_E_BYTES
                                                              : 0u);
                // the buffer's previous contents were read before the loop-top barrier
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             :: "r"(bar), "r"(bytes) : "memory");
                // x must be a multiple of 4 elements (16 bytes): round the
                // halo column down; the tile is indexed from the remainder
                if (!zero_in)
                    tma_load_3d((unsigned)__cvta_generic_to_shared(s_u + bs * TILE), &tm_u,
                                (px0 - 1) & ~3, py0 - 1, ch, bar);
                if (!rhs_zero)
                    tma_load_3d((unsigned)__cvta_generic_to_shared(s_b + bs * Smem2W::BSTRIDE),
                                &tm_b, px0 & ~3, py0, ch, bar);
                // the coarse patch from the 4-aligned column at or below its
                // first one (cells off the level read 0 and are fixed up
                // where the task starts)
                if (PRO != 0 && use_tma_e)
                    tma_load_3d((unsigned)__cvta_generic_to_shared(s_e + bs * Smem2W::ESTRIDE),
                                &tm_e, ((px0 >> 1) - 1) & ~3, (py0 >> 1) - 1, ch, bar);
            }
        } else if (!zero_in) {
            // thread t copies tile column lane of the rows ty = wi, wi + 2, ...
            // (and column 32 + lane for lane < 2); one word in, as for TMA tiles
            // of an odd halo column, so that block column 0 is 8-byte aligned
            const float* src = u_in + ch * n;
            float* dst = s_u + bs * TILE + 1;
            const int gxa = px0 - 1 + lane, gxb = gxa + 32;
            const bool oka = gxa >= 0 && gxa < w;
            const bool okb = lane < TH - 32 && gxb < w;
#pragma unroll 2
            for (int ty = wi; ty < TH; ty += 2) {
                const int gy = py0 - 1 + ty;
                const bool rok = gy >= 0 && gy < h;
                const float* row = src + (ptrdiff_t)gy * w;
                cp_async4(dst + ty * P + lane, (rok && oka) ? row + gxa : src, rok && oka);
                if (lane < TH - 32)
                    cp_async4(dst + ty * P + lane + 32, (rok && okb) ? row + gxb : src, rok && okb);
            }
        }
        if (!use_tma && !rhs_zero) {
            const float* src = rhs + ch * n;
            float* dst = s_b + bs * Smem2W::BSTRIDE;
            const int gx = px0 + lane;
#pragma unroll 4
            for (int ly = wi; ly < B; ly += 2) {
                const int gy = py0 + ly;
                const bool ok = gx < w && gy < h;
                cp_async4(dst + ly * PB + lane, ok ? src + (size_t)gy * w + gx : src, ok);
            }
        }
        if (!use_tma) cp_async_commit();
        if (blk != have_blk && lane < 16) {
            const int gy = py0 + 16 * wi + lane;
            if (gy < h) {
                const uint32_t* row = mbits + (size_t)gy * wpr + (px0 >> 5);
                nlo = __ldg(row);
                nhi = __ldg(row + 1);
            } else {
                nlo = nhi = 0xffffffffu;
            }
        }
    };

    int blk = chan_inner ? (int)blockIdx.x : (int)blockIdx.x / C;
    int ch = chan_inner ? 0 : (int)blockIdx.x - blk * C;
    if (blk >= nblk) return;  // block-uniform
    if (zero_in) {
        zero_tiles(s_u, t, 64);
        __syncthreads();
    }
    if (use_tma) {
        if (t == 0) {
            for (int b = 0; b < 2; ++b)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;"
                             :: "r"((unsigned)__cvta_generic_to_shared(&s_bar[b])) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        // no thread may probe a barrier before it is initialised (the shared
        // memory still holds whatever an earlier CTA left there)
        __syncthreads();
    }
    unsigned phase = 0;  // bit b: parity of the next completion of s_bar[b]
    prefetch(blk, ch, 0, -1);
    int buf = 0, cur_blk = -1;
    BlockOp op;
    float wx0 = 0.f, wx1 = 0.f;  // column weights
    int x0 = 0, y0 = 0, bh = 0, kx = 0, ky = 0;
    uint32_t rows_w = 0;  // overlap 2, bit j: local row j is in the image with weight 1
    float vmax = 0.f, pmax = 0.f;
    unsigned nsteps = 0;  // completed local CG steps of this thread's tasks
    // 8-byte stores of u_out
    const bool vec = OV != 2 && (w & 1) == 0 && (reinterpret_cast<uintptr_t>(u_out) & 7) == 0;

    for (;;) {
        const bool new_blk = blk != cur_blk;
        if (new_blk) {
            // the local operator, while the tile is on its way
            cur_blk = blk;
            ky = blk / nbx;
            kx = blk - ky * nbx;
            x0 = kx * s;
            y0 = ky * s;
            bh = min(B, h - y0);
            // lane < 16: the mask bits of row 16 wi + lane
            block_operator(op, bt, __funnelshift_r(nlo, nhi, x0 & 31), x0, y0, min(B, w - x0), bh,
                           w, h, alpha);
            wx0 = x0 + bt.cl < w ? ramp_weight(bt.cl, kx, nbx, s, o, inv_o1) : 0.f;
            wx1 = x0 + bt.cl + 1 < w ? ramp_weight(bt.cl + 1, kx, nbx, s, o, inv_o1) : 0.f;
            if constexpr (OV == 0) rows_w = own_rows(bt, ky, nby, bh);
        }
        if (use_tma) {
            const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar[buf]);
            bool ok = mbar_wait(bar, (phase >> buf) & 1u);
            phase ^= 1u << buf;
            if constexpr (PRO != 0) cp_async_wait_all();  // the coarse patch
            if (__syncthreads_or(!ok)) {
                // give the copy one more bounded wait before the CTA leaves
                if (!ok) mbar_wait(bar, ((phase >> buf) & 1u) ^ 1u);
                if (t == 0 && errflag) atomicExch(errflag, 1u);
                return;
            }
        } else {
            cp_async_wait_all();
            __syncthreads();
        }
        const uint32_t hk = nhk;
        int nb2 = blk, nc2 = ch;
        const bool more = next_task(nb2, nc2);
        if (more) prefetch(nb2, nc2, buf ^ 1, blk);

        if (new_blk) {
            if (!op.full) clipped_diagonal(bt, y0, bh, h, alpha, sh.nv);
            // read only after the barriers of the CG below
            if (OV != 0 && t < B)
                s_wy[t] = lane < bh ? ramp_weight(lane, ky, nby, s, o, inv_o1) : 0.f;
        }

        // TMA tiles start at the 4-aligned column below the halo column
        const int du = use_tma ? ((x0 - 1) & 3) : 1;
        const int db = use_tma ? (x0 & 3) : 0;
        // local row 0, column cl of the tiles, and the steps to the next local row
        const float* tc = s_u + buf * TILE + du + (bt.r0 + 1) * P + bt.cl + 1;
        const float* bc = s_b + buf * Smem2W::BSTRIDE + db + bt.r0 * PB + bt.cl;
        const int ts = bt.dr * P, bs = bt.dr * PB;
        if constexpr (PRO != 0) {
            // the start of the iteration in the tile (prolong_into_tile)
            constexpr int EW = Smem2W::EPW;  // patch pitch
            float* tw = s_u + buf * TILE + du;
            const int Ys = (y0 >> 1) - 1, Xs = (x0 >> 1) - 1;
            // TMA patches start at the 4-aligned column at or below Xs
            const int dqe = use_tma_e ? Xs - (Xs & ~3) : 0;
            float* const pw = s_e + buf * Smem2W::ESTRIDE + dqe;
            if (use_tma_e && (Ys < 0 || Xs < 0 || Ys + Smem2W::EW > hH || Xs + Smem2W::EW > wH)) {
                // a block at the level's border: the cells off the level
                // (read as 0) take the value of their clamped cell, which is
                // on the level and not itself rewritten
                for (int i = t; i < Smem2W::ES; i += 64) {
                    const int r = i / Smem2W::EW, q = i - r * Smem2W::EW;
                    const int Yc = min(max(Ys + r, 0), hH - 1), Xc = min(max(Xs + q, 0), wH - 1);
                    if (Yc != Ys + r || Xc != Xs + q) pw[r * EW + q] = pw[(Yc - Ys) * EW + (Xc - Xs)];
                }
                __syncthreads();  // block-uniform branch
            }
            prolong_into_tile<PRO == 1>(tw, pw, bt, op, hk, pmax);
            __syncthreads();  // the residual reads the other threads' columns
        }

        f2 x[8], r[8];
        constexpr bool EV = OV != 2;
        if (y0 > 0 && y0 + B < h) {
            if (rhs_zero) block_residual<F64, true, true, EV>(r, op, bt, tc, ts, bc, bs, y0, h);
            else block_residual<F64, false, true, EV>(r, op, bt, tc, ts, bc, bs, y0, h);
        } else {
            if (rhs_zero) block_residual<F64, true, false, EV>(r, op, bt, tc, ts, bc, bs, y0, h);
            else block_residual<F64, false, false, EV>(r, op, bt, tc, ts, bc, bs, y0, h);
        }
        nsteps += block_cg(x, r, op, bt, iters, rtol2, sh);

        float* up = u_out + ch * n + (size_t)(y0 + bt.r0) * w + x0 + bt.cl;
        const ptrdiff_t us = bt.dr * (ptrdiff_t)w;
        if constexpr (OV == 0) {
            block_write01(x, op.full, tc, ts, up, us, wx0 > 0.f, wx1 > 0.f, rows_w, vec, vmax);
        } else {
            // the weighted part of shared pixels is parked in the block's tile
            // for k_combine; the first contributor of a shared pixel (smallest
            // block index along each shared axis) also carries u_in, so the
            // combine pass only adds
            // A column's class and, in a row of weight 1, where it goes are the
            // thread's; everything per row is a select or a predicate (branches
            // around the stores took 10 % of a launch without CG steps)
            const int first = shared_first(o), nsh = shared_per_seam(o);
            const bool xf0 = !(kx > 0 && bt.cl >= first && bt.cl < first + nsh);
            const bool xf1 = !(kx > 0 && bt.cl + 1 >= first && bt.cl + 1 < first + nsh);
            const bool z0 = wx0 > 0.f, z1 = wx1 > 0.f, own0 = wx0 == 1.f, own1 = wx1 == 1.f;
            const bool both = z0 && z1, same = both && own0 == own1 && (vec || !own0);
            float* part = parked + ((size_t)blk * C + ch) * (B * B) + bt.r0 * B + bt.cl;
            const float* tu = tc;
            float m0 = 0.f, m1 = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int ly = bt.r0 + bt.dr * j;
                const float wy = s_wy[ly];
                const bool rz = wy > 0.f, rp = wy == 1.f;
                const bool yf = !(ky > 0 && (unsigned)(ly - first) < (unsigned)nsh);
                const float v0 = block_value(x, 0, j), v1 = block_value(x, 1, j);
                const f2 u = ld_pair<EV>(tu);
                // weight 1 implies the first contributor
                const float a = shared_part(wx0 * wy, v0, lo2(u), xf0 && yf);
                const float b = shared_part(wx1 * wy, v1, hi2(u), xf1 && yf);
                float* const pa = rp && own0 ? up : part;
                float* const pb = rp && own1 ? up : part;
                const bool two = rp ? same : rz && both;
                st_pair_if(two, pa, a, b);
                st_if(rz && z0 && !two, pa, a);
                st_if(rz && z1 && !two, pb + 1, b);
                m0 = fmaxf(m0, rz ? fabsf(v0) : 0.f);
                m1 = fmaxf(m1, rz ? fabsf(v1) : 0.f);
                up += us;
                part += bt.dr * B;
                tu += ts;
            }
            if (z0) vmax = fmaxf(vmax, m0);
            if (z1) vmax = fmaxf(vmax, m1);
        }
        if (!more) break;
        blk = nb2;
        ch = nc2;
        buf ^= 1;
    }
    if (step_count && t == 0) atomicAdd(step_count, (unsigned long long)nsteps);
    if (maxupd) {
        vmax = warp_max(vmax);
        if (lane == 0 && vmax > 0.f) atomicMax(maxupd, __float_as_uint(vmax));
    }
    if (PRO == 1 && maxpro) {
        pmax = warp_max(pmax);
        if (lane == 0 && pmax > 0.f) atomicMax(maxpro, __float_as_uint(pmax));
    }
}


// ---- four warps per block: the same iteration where few blocks are to be solved
//
// On the small levels of a decode a launch has fewer local problems than the
// GPU has SMs and lasts as long as one of them: about 6 us at ten steps, a warp
// issuing an instruction every 4 cycles in the CG steps and every 6 to 9 in the
// code around them, which runs once and cold.  So this form gives each problem
// twice the threads and every thread half the work: warp 2 wi + g takes row
// group g of warp wi of the two-warp form (BlockThread), lane = column, one
// column of eight rows (four packed pairs) per thread.  One CTA per problem, no
// prefetch.  Every sum is formed in the order of the two-warp form, so the bits
// are the same and the launcher may choose by the number of problems alone.
// With every SM busy it is the slower one (a barrier and a sum more per pixel).
// 256x256 decode 249 -> 211 us, 481x321 RGB (overlap 6) 432 -> 394, 1920x1080 RGB
// 1115 -> 1090, 3840x2160 RGB 1606 -> 1589.
// One local problem (block blk, channel ch).  PRO: as in k_oras_2w, -1: pro_rt.
template <int PRO, int OV>
__device__ __forceinline__ void oras_4w(
    int blk, int ch, const float* __restrict__ u_in, int zero_in, const float* __restrict__ rhs,
    int rhs_zero, const uint32_t* __restrict__ mbits, int wpr, int w, int h, int C, int o, int nbx,
    int nby, float alpha, int iters, float rtol2, float* __restrict__ u_out,
    float* __restrict__ parked, unsigned* __restrict__ maxupd, const CUtensorMap* tm_u,
    const CUtensorMap* tm_b, int use_tma, unsigned* __restrict__ errflag,
    unsigned long long* __restrict__ step_count, const float* __restrict__ eH, int wH, int hH,
    unsigned* __restrict__ maxpro, const CUtensorMap* tm_e, int use_tma_e, int pro_rt) {
    const int pro = PRO >= 0 ? PRO : pro_rt;
    constexpr int B = 32, TH = Smem2W::TH, P = Smem2W::PU, PB = Smem2W::PB;
    constexpr int EW = Smem2W::EPW;
    __shared__ __align__(128) float s_u[Smem2W::USTRIDE];
    __shared__ __align__(128) float s_b[Smem2W::BSTRIDE];
    __shared__ __align__(128) float s_e[PRO != 0 ? Smem2W::ESTRIDE : 32];
    __shared__ float s_wy[B], s_row0[2][32], s_row7[4][32];
    __shared__ float4 s_red1, s_red2;
    __shared__ __align__(8) unsigned long long s_bar;

    const int t = threadIdx.x, lane = t & 31, wrp = t >> 5;
    const int wi = wrp >> 1, g = wrp & 1;
    const int r0 = wi ? (g ? 16 : 31) : (g ? 15 : 0), dr = wi == g ? 1 : -1;
    const int s = B - o;
    const int ky = blk / nbx, kx = blk - ky * nbx, x0 = kx * s, y0 = ky * s;
    const size_t n = (size_t)w * h;
    const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar);

    // the tiles: one TMA box each, or 4-byte cp.async, as in k_oras_2w
    if (use_tma) {
        if (t == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            const unsigned bytes = (zero_in ? 0u : (unsigned)Smem2W::TMA_U_BYTES) +
                                   (rhs_zero ? 0u : (unsigned)Smem2W::TMA_B_BYTES) +
                                   (pro != 0 && use_tma_e ? (unsigned)Smem2W::TMA_E_BYTES : 0u);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                         :: "r"(bar), "r"(bytes) : "memory");
            if (!zero_in)
                tma_load_3d((unsigned)__cvta_generic_to_shared(s_u), tm_u, (x0 - 1) & ~3, y0 - 1,
                            ch, bar);
            if (!rhs_zero)
                tma_load_3d((unsigned)__cvta_generic_to_shared(s_b), tm_b, x0 & ~3, y0, ch, bar);
            if (pro != 0 && use_tma_e)
                tma_load_3d((unsigned)__cvta_generic_to_shared(s_e), tm_e,
                            ((x0 >> 1) - 1) & ~3, (y0 >> 1) - 1, ch, bar);
        }
    } else {
        if (!zero_in) {
            const float* src = u_in + ch * n;
            const int gxa = x0 - 1 + lane, gxb = gxa + 32;
            const bool oka = gxa >= 0 && gxa < w, okb = lane < TH - 32 && gxb < w;
            for (int ty = wrp; ty < TH; ty += 4) {
                const int gy = y0 - 1 + ty;
                const bool rok = gy >= 0 && gy < h;
                const float* row = src + (ptrdiff_t)gy * w;
                float* dst = s_u + ty * P + 1;
                cp_async4(dst + lane, (rok && oka) ? row + gxa : src, rok && oka);
                if (lane < TH - 32)
                    cp_async4(dst + lane + 32, (rok && okb) ? row + gxb : src, rok && okb);
            }
        }
        if (!rhs_zero) {
            const float* src = rhs + ch * n;
            const int gx = x0 + lane;
            for (int ly = wrp; ly < B; ly += 4) {
                const int gy = y0 + ly;
                const bool ok = gx < w && gy < h;
                cp_async4(s_b + ly * PB + lane, ok ? src + (size_t)gy * w + gx : src, ok);
            }
        }
    }
    if (pro != 0 && !use_tma_e)
        copy_patch_clamped(s_e, eH + (size_t)ch * wH * hH, x0, y0, wH, hH, t, 128);
    cp_async_commit();

    // mask bits: lane j < 8 the row of local row j; with a prolongation, the
    // thread's pixel of the halo (warp: above, below, left, right)
    uint32_t rowm = 0xffffffffu;
    {
        const int gy = y0 + r0 + dr * lane;
        if (lane < 8 && gy < h) {
            const uint32_t* row = mbits + (size_t)gy * wpr + (x0 >> 5);
            rowm = __funnelshift_r(__ldg(row), __ldg(row + 1), x0 & 31);
        }
    }
    bool hkn = true;  // known or off the image
    if (pro != 0) {
        const int hy = wrp == 0 ? y0 - 1 : wrp == 1 ? y0 + B : y0 + lane;
        const int hx = wrp < 2 ? x0 + lane : wrp == 2 ? x0 - 1 : x0 + B;
        if (hx >= 0 && hx < w && hy >= 0 && hy < h)
            hkn = (__ldg(mbits + (size_t)hy * wpr + (hx >> 5)) >> (hx & 31)) & 1u;
    }

    // the local operator of the thread's column (block_operator's values)
    const int bw = min(B, w - x0), bh = min(B, h - y0);
    const int gx = x0 + lane;
    const float hc = (lane > 0 ? 1.f : (gx > 0 ? alpha : 0.f)) +
                     (lane + 1 < bw ? 1.f : (gx < w - 1 ? alpha : 0.f));
    f2 nd[4], keep[4];
    uint32_t own = 0;  // bit j: local row j in the image
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float d[2], kp[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int j = k + 4 * e, ly = r0 + dr * j, gy = y0 + ly;
            const float vc = (ly > 0 ? 1.f : (gy > 0 ? alpha : 0.f)) +
                             (ly + 1 < bh ? 1.f : (gy < h - 1 ? alpha : 0.f));
            d[e] = -(hc + vc);
            kp[e] = ((__shfl_sync(kFull, rowm, j) >> lane) & 1u) ? 0.f : 1.f;
            if (ly < bh) own |= 1u << j;
        }
        nd[k] = pk(d[0], d[1]);
        keep[k] = pk(kp[0], kp[1]);
    }
    const int odd = lane & 1, outer = odd ? lane + 1 : lane - 1;
    const float mo = (lane == 0 || lane == 31) ? 0.f : 1.f;  // the outer column is in the block
    const f2 mo2 = pk(mo, mo);
    const float inv_o1 = o > 1 ? 1.f / (float)(o - 1) : 0.f;
    const float wx = gx < w ? ramp_weight(lane, kx, nbx, s, o, inv_o1) : 0.f;
    if (OV != 0 && t < B) s_wy[t] = lane < bh ? ramp_weight(lane, ky, nby, s, o, inv_o1) : 0.f;

    cp_async_wait_all();
    __syncthreads();  // the mbarrier is initialised, the cp.async tiles are there
    if (use_tma) {
        const bool ok = mbar_wait(bar, 0u);
        if (__syncthreads_or(!ok)) {
            if (!ok) mbar_wait(bar, 0u);  // one more bounded wait before the CTA leaves
            if (t == 0 && errflag) atomicExch(errflag, 1u);
            return;
        }
    }
    const int du = use_tma ? ((x0 - 1) & 3) : 1, db = use_tma ? (x0 & 3) : 0;
    float* const tc = s_u + du + (r0 + 1) * P + lane + 1;  // local row 0
    const int ts = dr * P;
    float pmax = 0.f;
    if (pro != 0) {
        const int Ys = (y0 >> 1) - 1, Xs = (x0 >> 1) - 1;
        float* const pw = s_e + (use_tma_e ? Xs - (Xs & ~3) : 0);
        if (use_tma_e && (Ys < 0 || Xs < 0 || Ys + Smem2W::EW > hH || Xs + Smem2W::EW > wH)) {
            // cells off the level take the value of their clamped cell
            for (int i = t; i < Smem2W::ES; i += 128) {
                const int r = i / Smem2W::EW, q = i - r * Smem2W::EW;
                const int Yc = min(max(Ys + r, 0), hH - 1), Xc = min(max(Xs + q, 0), wH - 1);
                if (Yc != Ys + r || Xc != Xs + q) pw[r * EW + q] = pw[(Yc - Ys) * EW + (Xc - Xs)];
            }
            __syncthreads();  // block-uniform branch
        }
        // the start of the iteration in the tile, as in prolong_into_tile
        const int es = dr * EW;
        const float* pr = pw + (1 + (r0 >> 1)) * EW + 1 + (lane >> 1) - es;
        float ec[6], en[6], tv[8];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            ec[i] = pr[i * es];
            en[i] = pr[i * es + (odd ? 1 : -1)];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) tv[j] = tc[j * ts];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = 1 + (j >> 1), m = (j & 1) ? i + 1 : i - 1;
            const bool unk = (j < 4 ? lo2(keep[j]) : hi2(keep[j - 4])) != 0.f;
            const float bl = prolong_blend(ec[i], ec[m], en[i], en[m]);
            const float a = unk ? bl : 0.f;
            tc[j * ts] = pro == 1 ? __fadd_rn(tv[j], a) : (unk ? a : tv[j]);
            pmax = fmaxf(pmax, fabsf(a));
        }
        {
            const bool row = wrp < 2;
            const int half = 1 + (lane >> 1), far = (wrp & 1) ? B / 2 + 1 : 0;
            const float* pp = pw + (row ? far * EW + half : half * EW + far);
            const int in = (row ? EW : 1) * ((wrp & 1) ? -1 : 1);
            const int al = (row ? 1 : EW) * (odd ? 1 : -1);
            const int vn = row ? in : al, hn = row ? al : in;
            const float a = prolong_blend(pp[0], pp[vn], pp[hn], pp[vn + hn]);
            float* tp = s_u + du + (row ? ((wrp & 1) ? (B + 1) * P : 0) + lane + 1
                                        : (lane + 1) * P + ((wrp & 1) ? B + 1 : 0));
            const float old = *tp;
            *tp = hkn ? old : (pro == 1 ? __fadd_rn(old, a) : a);
        }
        __syncthreads();  // the residual reads the other threads' columns
    }

    // residual (block_residual's sums)
    f2 r[4];
    {
        float rv[8];
        const float* bc = s_b + db + r0 * PB + lane;
        const float dh = (float)((gx > 0) + (gx < w - 1)) + 2.f;
        float up = 0.f, cen = 0.f;
        if (!zero_in) {
            up = tc[-ts];
            cen = tc[0];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float v = rhs_zero ? 0.f : bc[j * dr * PB];
            if (!zero_in) {
                const float* c0 = tc + j * ts;
                const float dn = c0[ts];
                const int gy = y0 + r0 + dr * j;
                const float e = (float)((gy == 0) + (gy == h - 1));
                const float nb = (up + dn) + (c0[-1] + c0[1]);
                const float a = __fmaf_rn(e - dh, cen, nb);
                v = rhs_zero ? a : v + a;
                up = cen;
                cen = dn;
            }
            rv[j] = v;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            r[k] = pk(rv[k] * lo2(keep[k]), rv[k + 4] * hi2(keep[k]));
    }

    // CG (block_cg's steps); sums: the column pairs of the two-warp form's
    // threads, the warp, then the row groups and the halves
    auto block_sum4 = [&](f2 acc, float4* red) {
        acc = add2(acc, __shfl_xor_sync(kFull, acc, 1));
        float v = lo2(acc) + hi2(acc);
#pragma unroll
        for (int d = 16; d > 1; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
        if (lane == 0) reinterpret_cast<float*>(red)[wrp] = v;
        __syncthreads();
        const float4 a = *red;
        return (a.x + a.y) + (a.z + a.w);
    };
    auto publish = [&]() {  // the rows that other warps need
        if (g) s_row0[wi][lane] = lo2(r[0]);
        s_row7[wrp][lane] = hi2(r[3]);
    };
    f2 x[4], p[4], q[4];
    f2 acc = mul2(r[0], r[0]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        p[k] = r[k];
        x[k] = 0ull;
        if (k) acc = fma2(r[k], r[k], acc);
    }
    publish();
    float rr = block_sum4(acc, &s_red2);
    float pb = g ? s_row0[wi ^ 1][lane] : 0.f;  // local row -1 of p
    float p8 = s_row7[wrp ^ 1][lane];           // local row 8
    const bool tiny = tiny_residual(rr, rtol2);
    if (tiny) {  // the same in every warp
        const f2 up = pk(kTinyScale, kTinyScale);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            r[k] = mul2(r[k], up);
            p[k] = r[k];
            acc = k ? fma2(r[k], r[k], acc) : mul2(r[k], r[k]);
        }
        rr = block_sum4(acc, &s_red1);
        __syncthreads();  // the first step writes s_red1
        pb *= kTinyScale;
        p8 *= kTinyScale;
        rtol2 = tiny_rtol2(rtol2);
    }
    const float rr_stop = fmaxf(rtol2 >= 0.f ? fmaxf(rtol2, 1e-14f) * rr : fmaxf(1e-14f * rr, -rtol2),
                                FLT_MIN);
    int it = 0;
    while (it < iters && rr > rr_stop) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const f2 in = __shfl_xor_sync(kFull, p[k], 1);
            const f2 ou = __shfl_sync(kFull, p[k], outer);
            f2 nb;
            if (k == 0) nb = pk(pb + lo2(p[1]), lo2(p[3]) + hi2(p[1]));
            else if (k == 3) nb = pk(lo2(p[2]) + hi2(p[0]), hi2(p[2]) + p8);
            else nb = add2(p[k - 1], p[k + 1]);
            nb = add2(nb, in);
            nb = fma2(mo2, ou, nb);
            q[k] = mul2(fma2(nd[k], p[k], nb), keep[k]);
            acc = k ? fma2(p[k], q[k], acc) : mul2(p[k], q[k]);
        }
        const float pq = -block_sum4(acc, &s_red1);
        if (!(pq >= FLT_MIN && pq <= FLT_MAX)) break;
        const float a = quotient(rr, pq);
        const f2 a2 = pk(a, a);
        if (++it == iters) {
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = fma2(a2, p[k], x[k]);
            break;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[k] = fma2(a2, p[k], x[k]);
            r[k] = fma2(a2, q[k], r[k]);
            acc = k ? fma2(r[k], r[k], acc) : mul2(r[k], r[k]);
        }
        publish();
        const float rrn = block_sum4(acc, &s_red2);
        const float beta = quotient(rrn, rr);
        rr = rrn;
        const f2 b2 = pk(beta, beta);
#pragma unroll
        for (int k = 0; k < 4; ++k) p[k] = fma2(b2, p[k], r[k]);
        if (g) pb = fmaf(beta, pb, s_row0[wi ^ 1][lane]);
        p8 = fmaf(beta, p8, s_row7[wrp ^ 1][lane]);
    }
    if (tiny) {
        const f2 down = pk(1.f / kTinyScale, 1.f / kTinyScale);
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = mul2(x[k], down);
    }

    // the weighted write (k_oras_2w)
    float vmax = 0.f;
    float* const up = u_out + ch * n + (size_t)(y0 + r0) * w + gx;
    const ptrdiff_t us = dr * (ptrdiff_t)w;
    if constexpr (OV == 0) {
        // local row 0 of g = 0 is the block's edge row: weight 0 inside the image
        if (!g && (wi == 0 ? ky > 0 : ky < nby - 1)) own &= ~1u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float v = j < 4 ? lo2(x[j]) : hi2(x[j - 4]);
            if (wx > 0.f && ((own >> j) & 1u)) {
                up[j * us] = (zero_in ? 0.f : tc[j * ts]) + v;
                vmax = fmaxf(vmax, fabsf(v));
            }
        }
    } else {
        const int first = shared_first(o), last = first + shared_per_seam(o);
        const bool xf = !(kx > 0 && lane >= first && lane < last);
        float* const mine = parked + ((size_t)blk * C + ch) * (B * B) + lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int ly = r0 + dr * j;
            const float d = wx * s_wy[ly];
            const float v = j < 4 ? lo2(x[j]) : hi2(x[j - 4]);
            const float u = zero_in ? 0.f : tc[j * ts];
            const bool yf = !(ky > 0 && ly >= first && ly < last);
            const float a = shared_part(d, v, u, xf && yf);
            if (d == 1.f) up[j * us] = a;
            else if (d > 0.f) mine[ly * B] = a;
            if (d > 0.f) vmax = fmaxf(vmax, fabsf(v));
        }
    }
    if (step_count && t == 0) atomicAdd(step_count, (unsigned long long)it);
    if (maxupd) {
        vmax = warp_max(vmax);
        if (lane == 0 && vmax > 0.f) atomicMax(maxupd, __float_as_uint(vmax));
    }
    if (pro == 1 && maxpro) {
        pmax = warp_max(pmax);
        if (lane == 0 && pmax > 0.f) atomicMax(maxpro, __float_as_uint(pmax));
    }
}

template <int PRO, int OV>
__global__ void __launch_bounds__(128, 4)
k_oras_4w(const float* __restrict__ u_in, int zero_in, const float* __restrict__ rhs, int rhs_zero,
          const uint32_t* __restrict__ mbits, int wpr, int w, int h, int C, int o, int nbx, int nby,
          float alpha, int iters, float rtol2, float* __restrict__ u_out,
          float* __restrict__ parked, unsigned* __restrict__ maxupd,
          const __grid_constant__ CUtensorMap tm_u, const __grid_constant__ CUtensorMap tm_b,
          int use_tma, unsigned* __restrict__ errflag,
          unsigned long long* __restrict__ step_count, const float* __restrict__ eH, int wH,
          int hH, unsigned* __restrict__ maxpro, const __grid_constant__ CUtensorMap tm_e,
          int use_tma_e) {
    const int blk = (int)blockIdx.x / C;
    oras_4w<PRO, OV>(blk, (int)blockIdx.x - blk * C, u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h,
                     C, o, nbx, nby, alpha, iters, rtol2, u_out, parked, maxupd, &tm_u, &tm_b,
                     use_tma, errflag, step_count, eH, wH, hH, maxpro, &tm_e, use_tma_e, PRO);
}

// ---- 16-bit storage variant of k_oras_2w ------------------------------------
// The CG vectors, the stencil and the vector updates of each local solve run
// in packed FP16 or BF16 (one 32-bit register per pixel pair, so half the
// registers and one shuffle per pair); the dot products accumulate in FP32,
// the residual that starts each local solve and the update of u stay FP32
// (the outer FP32 iteration refines whatever the narrow local solve leaves).
// The block residual is normalised by its maximum (times 1/64 for FP16, whose
// range is small) before it is narrowed.  A block whose narrow iterate stops
// being finite contributes no correction in this iteration.
struct HalfT {
    typedef __half2 T2;
    static constexpr float kScale = 1.f / 64.f;
    __device__ static __forceinline__ T2 make(float lo, float hi) { return __floats2half2_rn(lo, hi); }
    __device__ static __forceinline__ float lo(T2 a) { return __low2float(a); }
    __device__ static __forceinline__ float hi(T2 a) { return __high2float(a); }
    __device__ static __forceinline__ f2 wide(T2 a) {
        const float2 v = __half22float2(a);
        return pk(v.x, v.y);
    }
};
struct Bf16T {
    typedef __nv_bfloat162 T2;
    static constexpr float kScale = 1.f;
    __device__ static __forceinline__ T2 make(float lo, float hi) { return __floats2bfloat162_rn(lo, hi); }
    __device__ static __forceinline__ float lo(T2 a) { return __low2float(a); }
    __device__ static __forceinline__ float hi(T2 a) { return __high2float(a); }
    __device__ static __forceinline__ f2 wide(T2 a) {
        const float2 v = __bfloat1622float2(a);
        return pk(v.x, v.y);
    }
};

// TU: storage of u_in, rhs and u_out -- float on the finest level (tiles by
// 4-byte cp.async, prefetched while the previous task solves), FP16/BF16 on
// the coarse levels in the 16-bit precision modes (tiles read and widened to
// FP32 at the start of each task).  F64: the block residual in FP64.
template <class H, class TU, bool F64>
__global__ void __launch_bounds__(64, 8)
k_oras_2w_h(const TU* __restrict__ u_in, int zero_in, const TU* __restrict__ rhs,
            int rhs_zero, const uint32_t* __restrict__ mbits, int wpr, int w, int h, int C, int o,
            int nbx, int nby, float alpha, int iters, float rtol2, TU* __restrict__ u_out,
            float* __restrict__ parked, unsigned* __restrict__ maxupd, int chan_inner,
            unsigned long long* __restrict__ step_count) {
    constexpr bool kAsync = std::is_same<TU, float>::value;
    typedef typename H::T2 T2;
    constexpr int B = 32, NP = 8, TH = Tile2W::TH, P = Tile2W::P, TILE = Tile2W::TILE;
    extern __shared__ float smem[];
    float* const s_u = smem;
    float* const s_wy = smem + 2 * TILE;
    float* const s_b = smem + Tile2W::FIXED;
    __shared__ float s_red1[2], s_red2[2], s_seam[2][32], s_mx[2];

    const int t = threadIdx.x;
    const int lane = t & 31, wi = t >> 5;
    const int col = lane;
    const int row0 = 16 * wi;
    const int s = B - o;
    const size_t n = (size_t)w * h;
    const float inv_o1 = o > 1 ? 1.f / (float)(o - 1) : 0.f;
    const int nblk = nbx * nby;
    auto task_of = [&](int i, int& blk, int& ch) {
        if (chan_inner) {
            blk = (int)blockIdx.x + (i / C) * (int)gridDim.x;
            ch = i % C;
        } else {
            const int tt = (int)blockIdx.x + i * (int)gridDim.x;
            blk = tt / C;
            ch = tt - blk * C;
        }
        return blk < nblk;
    };
    uint32_t nlo = 0xffffffffu, nhi = 0xffffffffu;
    // the u tile (block + one-pixel halo) and the right-hand-side tile of a
    // task into buffer bs: asynchronous 4-byte copies (FP32 storage) or plain
    // loads widened to FP32 (16-bit storage)
    auto tiles = [&](int blk, int ch, int bs) {
        const int px0 = (blk % nbx) * s, py0 = (blk / nbx) * s;
        if (kAsync) {
            if (!zero_in) {
                const float* src = reinterpret_cast<const float*>(u_in + ch * n);
                float* dst = s_u + bs * TILE;
                const int gxa = px0 - 1 + lane, gxb = gxa + 32;
                const bool oka = gxa >= 0 && gxa < w;
                const bool okb = lane < TH - 32 && gxb < w;
#pragma unroll 2
                for (int ty = wi; ty < TH; ty += 2) {
                    const int gy = py0 - 1 + ty;
                    const bool rok = gy >= 0 && gy < h;
                    const float* row = src + (ptrdiff_t)gy * w;
                    cp_async4(dst + ty * P + lane, (rok && oka) ? row + gxa : src, rok && oka);
                    if (lane < TH - 32)
                        cp_async4(dst + ty * P + lane + 32, (rok && okb) ? row + gxb : src,
                                  rok && okb);
                }
            }
            if (!rhs_zero) {
                const float* src = reinterpret_cast<const float*>(rhs + ch * n);
                float* dst = s_b + bs * B * B;
                const int gx = px0 + lane;
#pragma unroll 4
                for (int ly = wi; ly < B; ly += 2) {
                    const int gy = py0 + ly;
                    const bool ok = gx < w && gy < h;
                    cp_async4(dst + ly * B + lane, ok ? src + (size_t)gy * w + gx : src, ok);
                }
            }
            cp_async_commit();
            return;
        }
        // 16-bit storage: every load of the thread (its rows of both tiles)
        // before the first store, so that they wait together; two rows at a time
        // the tiles took 7 us of a small level's launch
        constexpr int NR = TH / 2, NB = B / 2;
        float ra[NR], rb[NR], vb[NB];
        const TU* su = u_in + ch * n;
        const TU* sb = rhs + ch * n;
        const int gxa = px0 - 1 + lane, gxb = gxa + 32, gx = px0 + lane;
        const bool oka = !zero_in && gxa >= 0 && gxa < w;
        const bool okb = !zero_in && lane < TH - 32 && gxb < w;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int gy = py0 - 1 + wi + 2 * i;
            const bool rok = gy >= 0 && gy < h;
            ra[i] = rok && oka ? ldf(su + (ptrdiff_t)gy * w + gxa) : 0.f;
            rb[i] = rok && okb ? ldf(su + (ptrdiff_t)gy * w + gxb) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int gy = py0 + wi + 2 * i;
            vb[i] = !rhs_zero && gx < w && gy < h ? ldf(sb + (size_t)gy * w + gx) : 0.f;
        }
        if (!zero_in) {
            float* dst = s_u + bs * TILE + wi * P;
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                dst[2 * i * P + lane] = ra[i];
                if (lane < TH - 32) dst[2 * i * P + lane + 32] = rb[i];
            }
        }
        if (!rhs_zero) {
            float* dst = s_b + bs * B * B + wi * B;
#pragma unroll
            for (int i = 0; i < NB; ++i) dst[2 * i * B + lane] = vb[i];
        }
    };
    auto prefetch = [&](int blk, int ch, int bs, int have_blk) {
        const int px0 = (blk % nbx) * s, py0 = (blk / nbx) * s;
        if (kAsync) tiles(blk, ch, bs);
        if (blk != have_blk && lane < 16) {
            const int gy = py0 + row0 + lane;
            if (gy < h) {
                const uint32_t* row = mbits + (size_t)gy * wpr + (px0 >> 5);
                nlo = __ldg(row);
                nhi = __ldg(row + 1);
            } else {
                nlo = nhi = 0xffffffffu;
            }
        }
    };

    int blk, ch;
    if (!task_of(0, blk, ch)) return;
    prefetch(blk, ch, 0, -1);
    int buf = 0, cur_blk = -1;
    T2 ndg[NP], keep[NP];
    T2 ml2 = H::make(0.f, 0.f), mr2 = H::make(0.f, 0.f);
    float wx = 0.f, dh = 0.f;
    int x0 = 0, y0 = 0, bh = 0, kx = 0, ky = 0;
    float vmax = 0.f;
    unsigned nsteps = 0;  // completed local CG steps of this thread's tasks

    for (int i = 0;; ++i) {
        if (kAsync) cp_async_wait_all();
        __syncthreads();
        if (!kAsync) {
            // the previous readers of this buffer finished before the barrier
            tiles(blk, ch, buf);
            __syncthreads();
        }
        const uint32_t mlo = nlo, mhi = nhi;
        int nb2, nc2;
        const bool more = task_of(i + 1, nb2, nc2);
        if (more) prefetch(nb2, nc2, buf ^ 1, blk);

        if (blk != cur_blk) {
            cur_blk = blk;
            kx = blk % nbx;
            ky = blk / nbx;
            x0 = kx * s;
            y0 = ky * s;
            const int bw = min(B, w - x0);
            bh = min(B, h - y0);
            const uint32_t rowm = __funnelshift_r(mlo, mhi, x0 & 31);
            uint32_t mb = 0;
#pragma unroll
            for (int rr = 0; rr < 16; ++rr) {
                const uint32_t v = __shfl_sync(kFull, rowm, rr);
                mb |= ((v >> col) & 1u) << rr;
            }
            const int gx = x0 + col;
            const float hc = (col > 0 ? 1.f : (gx > 0 ? alpha : 0.f)) +
                             (col + 1 < bw ? 1.f : (gx < w - 1 ? alpha : 0.f));
            dh = (float)((gx > 0) + (gx < w - 1));
            const float ml = col > 0 ? 1.f : 0.f, mr = col < B - 1 ? 1.f : 0.f;
            ml2 = H::make(ml, ml);
            mr2 = H::make(mr, mr);
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                float vc[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int ly = row0 + k + 8 * e, gy = y0 + ly;
                    vc[e] = (ly > 0 ? 1.f : (gy > 0 ? alpha : 0.f)) +
                            (ly + 1 < bh ? 1.f : (gy < h - 1 ? alpha : 0.f));
                }
                ndg[k] = H::make(-(hc + vc[0]), -(hc + vc[1]));
                keep[k] = H::make(((mb >> k) & 1u) ? 0.f : 1.f, ((mb >> (k + 8)) & 1u) ? 0.f : 1.f);
            }
            wx = ramp_weight(col, kx, nbx, s, o, inv_o1);
            if (t < B) s_wy[t] = ramp_weight(t, ky, nby, s, o, inv_o1);
        }

        const float* tu = s_u + buf * TILE;
        const float* tb = s_b + buf * B * B;

        // FP32 residual of the block, then its maximum for the normalisation
        float rv[NP][2];
        float mx = 0.f;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int ly = row0 + k + 8 * e, gy = y0 + ly;
                float v = rhs_zero ? 0.f : tb[ly * B + col];
                if (!zero_in) {
                    const float* c0 = tu + (ly + 1) * P + col + 1;
                    const float dv = (float)((gy > 0) + (gy < h - 1));
                    v = res_stencil<F64>(v, dh + dv, c0[0], c0[-P], c0[P], c0[-1], c0[1]);
                }
                v *= e ? H::hi(keep[k]) : H::lo(keep[k]);
                rv[k][e] = v;
                mx = fmaxf(mx, fabsf(v));
            }
        }
        mx = warp_max(mx);
        if (lane == 0) s_mx[wi] = mx;
        __syncthreads();
        mx = fmaxf(s_mx[0], s_mx[1]);
        const float sc = mx > 0.f ? mx / H::kScale : 1.f;  // r = sc * r_narrow
        const float isc = 1.f / sc;

        T2 x[NP], r[NP], p[NP], q[NP];
        f2 acc0 = 0ull, acc1 = 0ull;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            r[k] = H::make(rv[k][0] * isc, rv[k][1] * isc);
            p[k] = r[k];
            x[k] = H::make(0.f, 0.f);
            const f2 rw = H::wide(r[k]);
            if (k & 1) acc1 = fma2(rw, rw, acc1);
            else acc0 = fma2(rw, rw, acc0);
        }
        acc0 = add2(acc0, acc1);
        s_seam[wi][lane] = wi == 0 ? H::hi(r[NP - 1]) : H::lo(r[0]);
        float part = warp_sum(lo2(acc0) + hi2(acc0));
        if (lane == 0) s_red2[wi] = part;
        __syncthreads();
        float rr = s_red2[0] + s_red2[1];
        float pb = s_seam[wi ^ 1][lane];
        // rtol2 >= 0: relative stop (r.r <= max(rtol2, 1e-14) (r.r)_0); rtol2 < 0:
        // also stop once r.r <= -rtol2 (an absolute level, or the FP32 floor). rr is
        // the normalised residual's, so the absolute level is scaled by isc^2 too.
        const float rr_stop = fmaxf(rtol2 >= 0.f ? fmaxf(rtol2, 1e-14f) * rr
                                                 : fmaxf(1e-14f * rr, -rtol2 * isc * isc),
                                    FLT_MIN);
        bool bad = !(rr < INFINITY);

        for (int it = 0; it < iters; ++it) {
            if (!(rr > rr_stop) || bad) break;  // identical in both warps
            const T2 pu = wi == 0 ? H::make(0.f, H::lo(p[NP - 1])) : H::make(pb, H::lo(p[NP - 1]));
            const T2 pd = wi == 0 ? H::make(H::hi(p[0]), pb) : H::make(H::hi(p[0]), 0.f);
            acc0 = 0ull;
            acc1 = 0ull;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const T2 left = __shfl_up_sync(kFull, p[k], 1);
                const T2 right = __shfl_down_sync(kFull, p[k], 1);
                const T2 up = k > 0 ? p[k - 1] : pu;
                const T2 dn = k < NP - 1 ? p[k + 1] : pd;
                T2 nbs = __hadd2(up, dn);
                nbs = __hfma2(ml2, left, nbs);
                nbs = __hfma2(mr2, right, nbs);
                const T2 qk = __hmul2(__hfma2(ndg[k], p[k], nbs), keep[k]);
                q[k] = qk;
                if (k & 1) acc1 = fma2(H::wide(p[k]), H::wide(qk), acc1);
                else acc0 = fma2(H::wide(p[k]), H::wide(qk), acc0);
            }
            acc0 = add2(acc0, acc1);
            part = warp_sum(lo2(acc0) + hi2(acc0));
            if (lane == 0) s_red1[wi] = part;
            __syncthreads();
            const float pq = -(s_red1[0] + s_red1[1]);
            if (!(pq >= FLT_MIN) || !(pq < INFINITY)) {
                bad = !(pq < INFINITY) || pq != pq;
                break;
            }
            const float a = quotient(rr, pq);
            const T2 a2 = H::make(a, a);
            acc0 = 0ull;
            acc1 = 0ull;
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                x[k] = __hfma2(a2, p[k], x[k]);
                r[k] = __hfma2(a2, q[k], r[k]);
                const f2 rw = H::wide(r[k]);
                if (k & 1) acc1 = fma2(rw, rw, acc1);
                else acc0 = fma2(rw, rw, acc0);
            }
            acc0 = add2(acc0, acc1);
            s_seam[wi][lane] = wi == 0 ? H::hi(r[NP - 1]) : H::lo(r[0]);
            part = warp_sum(lo2(acc0) + hi2(acc0));
            if (lane == 0) s_red2[wi] = part;
            __syncthreads();
            const float rrn = s_red2[0] + s_red2[1];
            if (!(rrn < INFINITY)) { bad = true; break; }
            const float beta = quotient(rrn, rr);
            rr = rrn;
            const T2 b2 = H::make(beta, beta);
#pragma unroll
            for (int k = 0; k < NP; ++k) p[k] = __hfma2(b2, p[k], r[k]);
            pb = fmaf(beta, pb, s_seam[wi ^ 1][lane]);
            ++nsteps;
        }

        TU* uo = u_out + ch * n;
        const bool colok = x0 + col < w;
        const int nsh = shared_per_seam(o), first = shared_first(o);
        const bool xfirst = !(kx > 0 && col >= first && col < first + nsh);
        float* const mine = parked + ((size_t)blk * C + ch) * (B * B) + col;
        const float vs = bad ? 0.f : sc;  // a non-finite narrow iterate gives no correction
#pragma unroll
        for (int k = 0; k < NP; ++k) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int ly = row0 + k + 8 * e;
                if (ly >= bh || !colok) continue;
                const float v = (e ? H::hi(x[k]) : H::lo(x[k])) * vs;
                const float d = wx * s_wy[ly];
                const float uold = zero_in ? 0.f : tu[(ly + 1) * P + col + 1];
                if (d == 1.f) {
                    stf(uo + (size_t)(y0 + ly) * w + x0 + col, uold + v);
                } else if (d > 0.f) {
                    const bool yfirst = !(ky > 0 && ly >= first && ly < first + nsh);
                    mine[ly * B] = (xfirst && yfirst) ? uold + d * v : d * v;
                }
                if (d > 0.f) vmax = fmaxf(vmax, fabsf(v));
            }
        }
        if (!more) break;
        blk = nb2;
        ch = nc2;
        buf ^= 1;
    }
    if (step_count && t == 0) atomicAdd(step_count, (unsigned long long)nsteps);
    if (maxupd) {
        vmax = warp_max(vmax);
        if (lane == 0 && vmax > 0.f) atomicMax(maxupd, __float_as_uint(vmax));
    }
}

// The sums of the pixels that several blocks share (overlap 1 or >= 3), in the
// fixed order upper left, upper right, lower left, lower right; the first term
// carries u_in; for 32x32 blocks.  A warp takes one part of a (block, channel):
// blockIdx.z = 0 the seam left of the block (two blocks), 1 the seam above it
// (two), 2 the corner where they cross (four).  One launch per iteration instead of a row and a
// column pass: with the parts in tiles by block, a warp reaches all its
// addresses from one block index.  Bound by latency (one dependent load round
// trip per warp, four rows in flight), not bytes: that is why the parts go to
// three warps instead of one after the other.  At overlap 6 an ORAS iteration
// on 1920x1080 RGB went from 116 to 107 us, a decode of that size from 1.38 to
// 1.20 ms and one of 481x321 RGB from 1.05 to 0.91 ms (one warp for all three
// parts: 1.22 ms and no gain at 481x321).
template <class TU>
__global__ void __launch_bounds__(256)
k_combine(const float* __restrict__ parked, int w, int h, int C, int o, int nbx, int nby,
          TU* __restrict__ u_out) {
    constexpr int B = 32;
    const int lane = threadIdx.x & 31;
    const int unit = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5);  // kx * C + ch
    if (unit >= nbx * C) return;
    const int kx = unit / C, ch = unit - kx * C, ky = blockIdx.y;
    const int s = B - o, x0 = kx * s, y0 = ky * s;
    const int nsh = shared_per_seam(o), first = shared_first(o);
    // lanes over the shared run of a seam: j < nsh of the next power of two
    const int js = nsh > 8 ? 4 : nsh > 4 ? 3 : nsh > 2 ? 2 : nsh > 1 ? 1 : 0;
    const int j = lane & ((1 << js) - 1), i0 = lane >> js, di = 32 >> js;
    // rows / columns of the block that only the seam's own blocks weight
    const int wlo = o == 1 ? 1 : o - 1, whi = o == 1 ? s - 1 : s;
    TU* dst = u_out + ((size_t)ch * h + y0) * w + x0;
    const float* me = parked + ((size_t)ky * nbx * C + unit) * (B * B);
    const float* lf = me - (size_t)C * (B * B) + s;            // left block, from its column s
    const float* up = me - (size_t)nbx * C * (B * B) + s * B;  // upper block, from its row s
    // rows i, i + step, ... <= hi of column x: the sum of two tiles, four rows in flight
    auto add2_rows = [&](const float* a, int i, int hi, int step, int x) {
        for (; i <= hi; i += 4 * step) {
            float v[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int r = i + m * step;
                v[m] = r <= hi ? a[r * B + x] + me[r * B + x] : 0.f;
            }
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (i + m * step <= hi) stf(dst + (size_t)(i + m * step) * w + x, v[m]);
        }
    };
    if (blockIdx.z == 0) {
        if (kx > 0 && j < nsh)
            add2_rows(lf, (ky > 0 ? wlo : 0) + i0, ky < nby - 1 ? whi : min(B, h - y0) - 1, di,
                      first + j);
    } else if (blockIdx.z == 1) {
        const int x = lane;
        if (ky > 0 && x >= (kx > 0 ? wlo : 0) && x <= (kx < nbx - 1 ? whi : min(B, w - x0) - 1))
            add2_rows(up, first, first + nsh - 1, 1, x);
    } else if (kx > 0 && ky > 0 && j < nsh) {
        const float* ul = up - (size_t)C * (B * B) + s;
        const int x = first + j;
        for (int i = first + i0; i < first + nsh; i += di)
            stf(dst + (size_t)i * w + x,
                ul[i * B + x] + up[i * B + x] + lf[i * B + x] + me[i * B + x]);
    }
}

// The same sums for blocks of 8 and 16, where a part of a block is a run of a few
// pixels and most lanes of its warp would idle: a thread per column and
// kCombineRows rows of pixels.  Bound by the sectors of the tiles (a word of
// each).  ORAS iteration of 8 steps, 3840x2160 RGB, against k_combine's warps:
// 8x8 blocks at overlap 4 2958 -> 2207 us, at overlap 1 988 -> 774; 16x16 at
// overlap 4 637 -> 604, at overlap 8 1337 -> 1174 (eight rows per thread: 1185).
// With 32x32 blocks, whose parts fill their warps, k_combine is the better one
// (overlap 4: 272 against 306).
constexpr int kCombineRows = 4;
template <int B>
__global__ void __launch_bounds__(256)
k_combine_px(const float* __restrict__ parked, int w, int h, int C, int o, int nbx, int nby,
             float* __restrict__ u_out) {
    const int x = blockIdx.x * 32 + threadIdx.x, ch = blockIdx.z;
    const int y0 = (blockIdx.y * 8 + threadIdx.y) * kCombineRows;
    if (x >= w || y0 >= h) return;
    const int s = B - o, first = shared_first(o), last = first + shared_per_seam(o);
    // the block whose own stride holds the coordinate (the lower one of a
    // shared pixel); local coordinate 0 has weight 0 there (overlap >= 3)
    int kx = min(x / s, nbx - 1), lx = x - kx * s;
    const bool sx = kx > 0 && lx >= first && lx < last;
    if (!sx && kx > 0 && lx == 0) {
        --kx;
        lx = s;
    }
    int ky = min(y0 / s, nby - 1), ly = y0 - ky * s;
    const size_t row = (size_t)nbx * C * (B * B);  // tiles of a row of blocks
    const int lf = s - C * (B * B);                // the same pixel in the left block's tile
    const ptrdiff_t up = s * B - (ptrdiff_t)row;   // and in the upper block's
    const float* col = parked + ((size_t)kx * C + ch) * (B * B) + lx;
    float v[kCombineRows];
    unsigned put = 0;
#pragma unroll
    for (int r = 0; r < kCombineRows; ++r) {
        const bool sy = ky > 0 && ly >= first && ly < last;
        const bool top = !sy && ky > 0 && ly == 0;  // weight 0: the upper block's row s
        const float* me = col + (size_t)(top ? ky - 1 : ky) * row + (top ? s : ly) * B;
        v[r] = 0.f;
        if (y0 + r < h && (sx || sy)) {
            put |= 1u << r;
            v[r] = sx && sy ? me[up + lf] + me[up] + me[lf] + me[0]
                   : sx     ? me[lf] + me[0]
                            : me[up] + me[0];
        }
        if (++ly == s && ky < nby - 1) {
            ++ky;
            ly = 0;
        }
    }
    float* dst = u_out + ((size_t)ch * h + y0) * w + x;
#pragma unroll
    for (int r = 0; r < kCombineRows; ++r)
        if ((put >> r) & 1u) dst[(size_t)r * w] = v[r];
}

// ---------------------------------------------------------------------------
// Device-driven decode: the plan and the stop test (Section 5.2 stop criterion;
// the error-estimate rule in gray levels).  One thread each; they steer the
// conditional nodes of the decode graph.
// ---------------------------------------------------------------------------

__global__ void k_plan(const unsigned long long* __restrict__ counts, StopState* __restrict__ st,
                       StopState* __restrict__ host, PlanParams p) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int L = p.L;
    const unsigned long long unk0 = counts[1];
    // levels down to the first one without unknown pixels (max pooling keeps
    // a known pixel known, so every coarser level is fully known too)
    int Leff = L;
    for (int l = 1; l < L; ++l)
        if (counts[1 + l] == 0) { Leff = l; break; }
    if (unk0 == 0) Leff = 0;
    st->cycles = 0;
    st->converged = 0;
    st->levels_used = Leff;
    st->est = 0.f;
    st->prevU = -1.f;
    st->prevQ = -1.f;
    st->unknowns = unk0;
    for (int k = 0; k < kMaxChannels; ++k) st->rel[k] = -1.f;
    const bool empty = unk0 == p.n0;
    st->status = empty ? DI_ERR_EMPTY_MASK : DI_OK;
    if (!empty && Leff == 0) st->converged = 1;  // every pixel known: u = f
    *host = *st;  // what the host sees unless a stop test follows
    if (empty) {
        cudaGraphSetConditional(p.h_sel, kSelSkip);
        return;
    }
    cudaGraphSetConditional(p.h_sel, (unsigned)Leff);
    if (Leff > 0) cudaGraphSetConditional(p.h_loop[Leff], p.max_cycles > 0 ? 1u : 0u);
}

// The stop test of the host loop, on the device: the same float arithmetic
// in the same order, so the decisions are identical.
__global__ void k_stop(unsigned* __restrict__ upd, StopState* __restrict__ st,
                       StopState* __restrict__ host, StopParams p,
                       cudaGraphConditionalHandle h_loop) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int cycles = st->cycles + 1;
    st->cycles = cycles;
    bool stop = false;
    if (upd[kMaxUpdSlots]) {
        st->status = DI_ERR_TIMEOUT;
        stop = true;
    } else if (p.rule == DI_STOP_ERROR_ESTIMATE) {
        float U = 0.f;
        for (int k = 0; k < p.nslots; ++k) U += __uint_as_float(upd[k]);
        float prevU = st->prevU, prevQ = st->prevQ, est;
        if (!isfinite(U)) {
            est = INFINITY;
            prevU = -1.f;
            prevQ = -1.f;
        } else if (prevU > 0.f) {
            // decay factor: the larger of the last two measured ratios
            const float qk = __fdiv_rn(U, prevU);
            const float q = prevQ > qk ? prevQ : qk;
            prevQ = qk;
            est = q < 1.f ? __fdiv_rn(__fmul_rn(U, q), __fsub_rn(1.f, q)) : INFINITY;
        } else {
            est = U;  // first cycle: no decay measured yet
        }
        prevU = U;
        if (U == 0.f) est = 0.f;
        st->prevU = prevU;
        st->prevQ = prevQ;
        st->est = est;
        if (cycles >= p.min_cycles && est <= 0.5f * p.tol) {
            st->converged = 1;
            stop = true;
        }
    } else if (p.rule == DI_STOP_RELATIVE_RESIDUAL) {
        bool ok = true;
        for (int k = 0; k < p.C; ++k) {
            const double b2 = st->bnorm2[k];
            const double rr = b2 > 0 ? sqrt(st->norm2[k] / b2) : 0.0;
            st->rel[k] = (float)rr;
            if (!(rr <= (double)p.tol)) ok = false;
        }
        if (cycles >= p.min_cycles && ok) {
            st->converged = 1;
            stop = true;
        }
    } else if (cycles >= p.max_cycles) {  // fixed number of cycles
        st->converged = 1;
        stop = true;
    }
    if (!stop && cycles >= p.max_cycles) {
        st->status = DI_ERR_NOT_CONVERGED;
        stop = true;
    }
    for (int k = 0; k < p.nslots; ++k) upd[k] = 0u;
    if (stop) *host = *st;
    cudaGraphSetConditional(h_loop, stop ? 0u : 1u);
}

// ---------------------------------------------------------------------------
// Batched form: the step kernels over the segments of a batch (one image's
// level each).  A CTA finds its segment by binary search over the segments'
// first CTAs, skips it if the image does not take part in this step, and runs
// the single-image body on the segment's buffers.
// ---------------------------------------------------------------------------

__device__ __forceinline__ int find_seg(const BatchSeg* __restrict__ segs, int nseg, int g) {
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (segs[mid].first <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ bool seg_active(int when, int img, int level, int L,
                                           const BatchState& bs) {
    switch (when) {
        case kWhenTopEq: return bs.top[img] == level;
        case kWhenCoarsestStart: return bs.leff[img] == L;
        case kWhenBelowTop: return level < bs.top[img];
        case kWhenCycle: return !bs.done[img] && level < bs.leff[img];
        default: return true;
    }
}

template <int KIND>
__global__ void __launch_bounds__(256)
k_batch_grid(const BatchSeg* __restrict__ segs, int nseg, BatchState bs) {
    const BatchSeg& sg = segs[find_seg(segs, nseg, (int)blockIdx.x)];
    if (!seg_active(sg.when, sg.img, sg.level, sg.L, bs)) return;  // uniform per CTA
    const int local = (int)blockIdx.x - sg.first;
    const int w = sg.w, h = sg.h;
    const int wH = (w + 1) / 2, hH = (h + 1) / 2;
    if (KIND == kBPack) {
        pack_mask_body(static_cast<const uint8_t*>(sg.in0), w, h, const_cast<uint32_t*>(sg.mbits),
                       sg.wpr, sg.counter, local, sg.gx);
        return;
    }
    if (KIND == kBSelect) {
        const int ch = local / sg.gx, bx = local - ch * sg.gx;
        const size_t n = (size_t)w * h;
        select_body<float>(static_cast<const float*>(sg.in1), static_cast<const uint8_t*>(sg.in2),
                           n, static_cast<float*>(sg.out0), sg.keep, bx, sg.gx, ch);
        if (sg.out1)
            select_body<float>(static_cast<const float*>(sg.in1),
                               static_cast<const uint8_t*>(sg.in2), n,
                               static_cast<float*>(sg.out1), sg.keep, bx, sg.gx, ch);
        return;
    }
    const int plane = sg.gx * sg.gy;
    const int bz = local / plane, rem = local - bz * plane;
    const int by = rem / sg.gx, bx = rem - by * sg.gx;
    if (KIND == kBPyramid) {
        const uint8_t* c = static_cast<const uint8_t*>(sg.in0);
        const float* b = static_cast<const float*>(sg.in1);
        uint8_t* cH = static_cast<uint8_t*>(sg.out0);
        float* bH = static_cast<float*>(sg.out1);
        uint32_t* bits = const_cast<uint32_t*>(sg.mbits);
        if (sg.mode)
            pyramid_level_body<1, true, true>(c, b, w, h, sg.C, cH, bH, wH, hH, 1, bits, sg.wpr,
                                              sg.counter, bx, by, sg.gx);
        else
            pyramid_level_body<1, false, false>(c, b, w, h, sg.C, cH, bH, wH, hH, 1, bits, sg.wpr,
                                                sg.counter, bx, by, sg.gx);
    } else if (KIND == kBRestrict) {
        const float* u = static_cast<const float*>(sg.in0);
        const float* b = static_cast<const float*>(sg.in1);
        const uint8_t* cH = static_cast<const uint8_t*>(sg.in2);
        float* rH = static_cast<float*>(sg.out0);
        // patches beside the mask bytes: whole batches are 1 % faster for it at a
        // mask density of 0.05 and 2 % slower at 0.9 (eight images of 1920x1080:
        // 2774 against 2799 us, 2054 against 2018)
        if ((w & 1) == 0 && ((reinterpret_cast<uintptr_t>(u) |
                              (sg.rhs_zero ? 0 : reinterpret_cast<uintptr_t>(b))) & 7) == 0)
            restrict_body<true, float, float, float, false, true>(u, b, sg.rhs_zero, w, h, cH, rH,
                                                                  wH, hH, bx, by, bz);
        else
            restrict_body<false, float, float, float, false>(u, b, sg.rhs_zero, w, h, cH, rH, wH,
                                                             hH, bx, by, bz);
    }
}

// The block kernel over the block units of a batch: a unit is one 32x32
// block of one image's level with all its channels back to back; CTAs are
// persistent and stride over the units of every image in the launch, skipping
// the units of images that do not take part.  Tiles by TMA through each
// segment's tensor maps, or by 4-byte cp.async where an image does not allow
// TMA (prefetched while the previous task solves; a TMA wait that runs out
// sets *bs.err and the CTA leaves); 0/1 partition weights (overlap 2: each
// pixel is written by the one block whose weight is 1 there); a segment may
// form its start by prolongation (BatchSeg).  Otherwise the local problem,
// the CG and the write are those of k_oras_2w.
__global__ void __launch_bounds__(64, 8)
k_batch_oras(const BatchSeg* __restrict__ segs, int nseg, int nunits, int split, int o,
             float alpha, BatchState bs) {
    constexpr int B = 32, TH = Smem2W::TH, P = Smem2W::PU, PB = Smem2W::PB;
    constexpr int TILE = Smem2W::USTRIDE;
    extern __shared__ float smem_raw[];
    float* const smem = reinterpret_cast<float*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    float* const s_u = smem;
    float* const s_e = smem + Smem2W::EP;  // coarse patches of prolonging segments
    float* const s_b = smem + Smem2W::RHS_PRO;
    __shared__ BlockShared sh;
    __shared__ __align__(8) unsigned long long s_bar[2];  // TMA tiles of buffer 0, 1

    const int t = threadIdx.x;
    const BlockThread bt(t);
    const int lane = bt.lane, wi = bt.wi;
    const int s = B - o;
    const float inv_o1 = o > 1 ? 1.f / (float)(o - 1) : 0.f;
    // whether a segment's tasks form their start by prolongation (uniform per task)
    auto prolongs = [&](const BatchSeg& sg) {
        return sg.pro_mode != 0 && (!sg.pro_check || sg.level + 1 < bs.leff[sg.img]);
    };

    // a task: a unit's segment and block, and a channel
    struct Task {
        int seg, blk, ch;
    };
    // the next active task after (unit g, channel ch): the next channel, else
    // the next unit of this CTA whose image takes part; split > 0 (fewer units
    // than CTA slots): g counts (unit, channel) pairs, split of them per unit
    auto advance = [&](int& g, Task& tk) {
        if (!split && tk.seg >= 0 && ++tk.ch < segs[tk.seg].C) return true;
        const int end = split ? nunits * split : nunits;
        for (g = g < 0 ? (int)blockIdx.x : g + (int)gridDim.x; g < end; g += (int)gridDim.x) {
            const int unit = split ? g / split : g;
            const int si = find_seg(segs, nseg, unit);
            const BatchSeg& sg = segs[si];
            if (!seg_active(sg.when, sg.img, sg.level, sg.L, bs)) continue;
            tk.ch = split ? g - unit * split : 0;
            if (tk.ch >= sg.C) continue;
            tk.seg = si;
            tk.blk = unit - sg.first;
            return true;
        }
        return false;
    };
    uint32_t nlo = 0xffffffffu, nhi = 0xffffffffu, nhk = 3u;
    // bit b: buffer b awaits a TMA completion; parity of its next completion
    unsigned pend_tma = 0, phase = 0;
    auto prefetch = [&](const Task& tk, int bs_, bool new_blk) {
        const BatchSeg& sg = segs[tk.seg];
        const int w = sg.w, h = sg.h, nbx = sg.nbx;
        const size_t n = (size_t)w * h;
        const int px0 = (tk.blk % nbx) * s, py0 = (tk.blk / nbx) * s;
        if (prolongs(sg)) {
            const int wH = (w + 1) / 2, hH = (h + 1) / 2;
            copy_patch_clamped(s_e + bs_ * Smem2W::ESTRIDE, sg.pro_e + (size_t)tk.ch * wH * hH,
                               px0, py0, wH, hH, t);
            if (new_blk) nhk = halo_known_bits(sg.mbits, sg.wpr, w, h, px0, py0, wi, lane);
        }
        if (sg.tma) {
            // the tiles by TMA, as in k_oras_2w (x rounded down to a multiple
            // of 4; the tile is indexed from the remainder)
            if (t == 0) {
                const CUtensorMap* maps = static_cast<const CUtensorMap*>(sg.tmaps);
                const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar[bs_]);
                const unsigned bytes = (sg.zero_in ? 0u : (unsigned)Smem2W::TMA_U_BYTES) +
                                       (sg.rhs_zero ? 0u : (unsigned)Smem2W::TMA_B_BYTES);
                // the buffer's previous contents were read before the loop-top barrier
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             :: "r"(bar), "r"(bytes) : "memory");
                if (!sg.zero_in)
                    tma_load_3d((unsigned)__cvta_generic_to_shared(s_u + bs_ * TILE), &maps[0],
                                (px0 - 1) & ~3, py0 - 1, tk.ch, bar);
                if (!sg.rhs_zero)
                    tma_load_3d((unsigned)__cvta_generic_to_shared(s_b + bs_ * Smem2W::BSTRIDE),
                                &maps[1], px0 & ~3, py0, tk.ch, bar);
            }
            pend_tma |= 1u << bs_;
        } else if (!sg.zero_in) {
            const float* src = static_cast<const float*>(sg.in0) + tk.ch * n;
            float* dst = s_u + bs_ * TILE + 1;  // block column 0 at an 8-byte boundary
            const int gxa = px0 - 1 + lane, gxb = gxa + 32;
            const bool oka = gxa >= 0 && gxa < w;
            const bool okb = lane < TH - 32 && gxb < w;
#pragma unroll 2
            for (int ty = wi; ty < TH; ty += 2) {
                const int gy = py0 - 1 + ty;
                const bool rok = gy >= 0 && gy < h;
                const float* row = src + (ptrdiff_t)gy * w;
                cp_async4(dst + ty * P + lane, (rok && oka) ? row + gxa : src, rok && oka);
                if (lane < TH - 32)
                    cp_async4(dst + ty * P + lane + 32, (rok && okb) ? row + gxb : src, rok && okb);
            }
        }
        if (!sg.tma && !sg.rhs_zero) {
            const float* src = static_cast<const float*>(sg.in1) + tk.ch * n;
            float* dst = s_b + bs_ * Smem2W::BSTRIDE;
            const int gx = px0 + lane;
#pragma unroll 4
            for (int ly = wi; ly < B; ly += 2) {
                const int gy = py0 + ly;
                const bool ok = gx < w && gy < h;
                cp_async4(dst + ly * PB + lane, ok ? src + (size_t)gy * w + gx : src, ok);
            }
        }
        cp_async_commit();
        if (new_blk && lane < 16) {
            const int gy = py0 + 16 * wi + lane;
            if (gy < h) {
                const uint32_t* row = sg.mbits + (size_t)gy * sg.wpr + (px0 >> 5);
                nlo = __ldg(row);
                nhi = __ldg(row + 1);
            } else {
                nlo = nhi = 0xffffffffu;
            }
        }
    };

    int g = -1;
    Task cur{-1, 0, 0};
    if (!advance(g, cur)) return;  // block-uniform
    if (t == 0) {
        for (int k = 0; k < 2; ++k)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;"
                         :: "r"((unsigned)__cvta_generic_to_shared(&s_bar[k])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (segs[cur.seg].zero_in) zero_tiles(s_u, t, 64);  // of every segment of the launch
    // no thread may probe a barrier before it is initialised
    __syncthreads();
    prefetch(cur, 0, true);
    int buf = 0;
    int cur_seg = -1, cur_blk = -1;
    BlockOp op;
    float wx0 = 0.f, wx1 = 0.f;
    int x0 = 0, y0 = 0;
    uint32_t rows_w = 0;
    float vmax = 0.f, pmax = 0.f;
    unsigned* vmax_slot = nullptr;
    unsigned* pmax_slot = nullptr;

    for (;;) {
        cp_async_wait_all();
        if ((pend_tma >> buf) & 1u) {  // uniform: the task's segment decides
            const unsigned bar = (unsigned)__cvta_generic_to_shared(&s_bar[buf]);
            const bool ok = mbar_wait(bar, (phase >> buf) & 1u);
            phase ^= 1u << buf;
            pend_tma &= ~(1u << buf);
            if (__syncthreads_or(!ok)) {
                // give the copy one more bounded wait before the CTA leaves
                if (!ok) mbar_wait(bar, ((phase >> buf) & 1u) ^ 1u);
                if (t == 0 && bs.err) atomicExch(bs.err, 1u);
                return;
            }
        } else {
            __syncthreads();
        }
        const uint32_t mlo = nlo, mhi = nhi, hk = nhk;
        Task nxt = cur;
        int g2 = g;
        const bool more = advance(g2, nxt);
        if (more) prefetch(nxt, buf ^ 1, nxt.seg != cur.seg || nxt.blk != cur.blk);

        const BatchSeg& sg = segs[cur.seg];
        const int w = sg.w, h = sg.h, nbx = sg.nbx, nby = sg.nby;
        const int rhs_zero = sg.rhs_zero;
        const size_t n = (size_t)w * h;
        if (cur.seg != cur_seg) {
            // the image changes: flush the previous image's largest update
            if (vmax_slot) {
                const float m = warp_max(vmax);
                if (lane == 0 && m > 0.f) atomicMax(vmax_slot, __float_as_uint(m));
            }
            if (pmax_slot) {
                const float m = warp_max(pmax);
                if (lane == 0 && m > 0.f) atomicMax(pmax_slot, __float_as_uint(m));
            }
            vmax = 0.f;
            pmax = 0.f;
            vmax_slot = sg.maxupd;
            pmax_slot = sg.pro_mode == 1 ? sg.pro_max : nullptr;
            cur_seg = cur.seg;
            cur_blk = -1;
        }
        if (cur.blk != cur_blk) {
            cur_blk = cur.blk;
            const int kx = cur.blk % nbx, ky = cur.blk / nbx;
            x0 = kx * s;
            y0 = ky * s;
            const int bh = min(B, h - y0);
            block_operator(op, bt, __funnelshift_r(mlo, mhi, x0 & 31), x0, y0, min(B, w - x0), bh,
                           w, h, alpha);
            if (!op.full) clipped_diagonal(bt, y0, bh, h, alpha, sh.nv);
            wx0 = x0 + bt.cl < w ? ramp_weight(bt.cl, kx, nbx, s, o, inv_o1) : 0.f;
            wx1 = x0 + bt.cl + 1 < w ? ramp_weight(bt.cl + 1, kx, nbx, s, o, inv_o1) : 0.f;
            rows_w = own_rows(bt, ky, nby, bh);
        }
        // TMA tiles start at the 4-aligned column below the halo column
        const int du = sg.tma ? ((x0 - 1) & 3) : 1;
        const int db = sg.tma ? (x0 & 3) : 0;
        const float* tc = s_u + buf * TILE + du + (bt.r0 + 1) * P + bt.cl + 1;
        const float* bc = s_b + buf * Smem2W::BSTRIDE + db + bt.r0 * PB + bt.cl;
        const int ts = bt.dr * P, bs_b = bt.dr * PB;
        if (prolongs(sg)) {  // uniform per task
            const float* pe = s_e + buf * Smem2W::ESTRIDE;
            if (sg.pro_mode == 1)
                prolong_into_tile<true>(s_u + buf * TILE + du, pe, bt, op, hk, pmax);
            else
                prolong_into_tile<false>(s_u + buf * TILE + du, pe, bt, op, hk, pmax);
            __syncthreads();  // the residual reads the other threads' columns
        }

        f2 x[8], r[8];
        if (y0 > 0 && y0 + B < h) {
            if (rhs_zero)
                block_residual<false, true, true, true>(r, op, bt, tc, ts, bc, bs_b, y0, h);
            else
                block_residual<false, false, true, true>(r, op, bt, tc, ts, bc, bs_b, y0, h);
        } else {
            if (rhs_zero)
                block_residual<false, true, false, true>(r, op, bt, tc, ts, bc, bs_b, y0, h);
            else
                block_residual<false, false, false, true>(r, op, bt, tc, ts, bc, bs_b, y0, h);
        }
        block_cg(x, r, op, bt, sg.iters, sg.rtol2, sh);

        float* uo = static_cast<float*>(sg.out0);
        const bool vec = (w & 1) == 0 && (reinterpret_cast<uintptr_t>(uo) & 7) == 0;
        float* up = uo + cur.ch * n + (size_t)(y0 + bt.r0) * w + x0 + bt.cl;
        const ptrdiff_t us = bt.dr * (ptrdiff_t)w;
        block_write01(x, op.full, tc, ts, up, us, wx0 > 0.f, wx1 > 0.f, rows_w, vec, vmax);
        if (!more) break;
        g = g2;
        cur = nxt;
        buf ^= 1;
    }
    if (vmax_slot) {
        vmax = warp_max(vmax);
        if (lane == 0 && vmax > 0.f) atomicMax(vmax_slot, __float_as_uint(vmax));
    }
    if (pmax_slot) {
        pmax = warp_max(pmax);
        if (lane == 0 && pmax > 0.f) atomicMax(pmax_slot, __float_as_uint(pmax));
    }
}

// The same with four warps per local problem (oras_4w), for launches of few:
// CTA cmax * g + ch takes channel ch of block unit g.  With it, and the
// channels of a block on separate CTAs where there are fewer blocks than CTA
// slots, a batch of 12 uneven images up to 1920x1080 takes 1077 us instead of
// 1272, two cycles of 12 RGB and gray images of 640x481 984 instead of 1189.
__global__ void __launch_bounds__(128, 4)
k_batch_oras_4w(const BatchSeg* __restrict__ segs, int nseg, int cmax, int o, float alpha,
                BatchState bs) {
    const int g = (int)blockIdx.x / cmax, ch = (int)blockIdx.x - g * cmax;
    const BatchSeg& sg = segs[find_seg(segs, nseg, g)];
    if (ch >= sg.C || !seg_active(sg.when, sg.img, sg.level, sg.L, bs)) return;
    const CUtensorMap* maps = static_cast<const CUtensorMap*>(sg.tmaps);
    const bool pro = sg.pro_mode != 0 && (!sg.pro_check || sg.level + 1 < bs.leff[sg.img]);
    oras_4w<-1, 0>(g - sg.first, ch, static_cast<const float*>(sg.in0), sg.zero_in,
                   static_cast<const float*>(sg.in1), sg.rhs_zero, sg.mbits, sg.wpr, sg.w, sg.h,
                   sg.C, o, sg.nbx, sg.nby, alpha, sg.iters, sg.rtol2,
                   static_cast<float*>(sg.out0), nullptr, sg.maxupd, maps, maps + 1, sg.tma, bs.err,
                   nullptr, sg.pro_e, (sg.w + 1) / 2, (sg.h + 1) / 2,
                   sg.pro_mode == 1 ? sg.pro_max : nullptr, nullptr, 0, pro ? sg.pro_mode : 0);
}

// Plan of every image of a batch: levels in use, the cascade's start level
// and the initial stop state (as k_plan for one image).
__global__ void k_batch_plan(int n, const int* __restrict__ Ls,
                             const unsigned long long* __restrict__ n0s, BatchState bs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int L = Ls[i];
    const unsigned long long* counts = bs.counts + (size_t)i * (kMaxLevels + 1);
    const unsigned long long unk0 = counts[1];
    int Leff = L;
    for (int l = 1; l < L; ++l)
        if (counts[1 + l] == 0) { Leff = l; break; }
    if (unk0 == 0) Leff = 0;
    StopState* st = bs.st + i;
    st->cycles = 0;
    st->converged = 0;
    st->levels_used = Leff;
    st->est = 0.f;
    st->prevU = -1.f;
    st->prevQ = -1.f;
    st->unknowns = unk0;
    for (int k = 0; k < kMaxChannels; ++k) st->rel[k] = -1.f;
    const bool empty = unk0 == n0s[i];
    st->status = empty ? DI_ERR_EMPTY_MASK : DI_OK;
    bs.leff[i] = empty ? 0 : Leff;
    bs.top[i] = empty ? -1 : (Leff == 0 ? 0 : (Leff == L ? L - 1 : Leff));
    bs.done[i] = (empty || Leff == 0) ? 1 : 0;
    if (!empty && Leff == 0) st->converged = 1;
    unsigned* upd = bs.upd + (size_t)i * (kMaxUpdSlots + 1);
    for (int k = 0; k <= kMaxUpdSlots; ++k) upd[k] = 0u;
}

// The stop test of every image still running (k_stop's rule per image); the
// loop continues while any image runs.
__global__ void k_batch_stop(int n, StopParams p, BatchState bs, cudaGraphConditionalHandle h) {
    __shared__ int s_any;
    if (threadIdx.x == 0) s_any = 0;
    __syncthreads();
    int running = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        if (bs.done[i]) continue;
        StopState* st = bs.st + i;
        unsigned* upd = bs.upd + (size_t)i * (kMaxUpdSlots + 1);
        const int cycles = st->cycles + 1;
        st->cycles = cycles;
        bool stop = false;
        if (upd[kMaxUpdSlots]) {
            st->status = DI_ERR_TIMEOUT;
            stop = true;
        } else if (p.rule == DI_STOP_ERROR_ESTIMATE) {
            float U = 0.f;
            for (int k = 0; k < p.nslots; ++k) U += __uint_as_float(upd[k]);
            float prevU = st->prevU, prevQ = st->prevQ, est;
            if (!isfinite(U)) {
                est = INFINITY;
                prevU = -1.f;
                prevQ = -1.f;
            } else if (prevU > 0.f) {
                const float qk = __fdiv_rn(U, prevU);
                const float q = prevQ > qk ? prevQ : qk;
                prevQ = qk;
                est = q < 1.f ? __fdiv_rn(__fmul_rn(U, q), __fsub_rn(1.f, q)) : INFINITY;
            } else {
                est = U;
            }
            prevU = U;
            if (U == 0.f) est = 0.f;
            st->prevU = prevU;
            st->prevQ = prevQ;
            st->est = est;
            if (cycles >= p.min_cycles && est <= 0.5f * bs.tol[i]) {
                st->converged = 1;
                stop = true;
            }
        } else if (cycles >= p.max_cycles) {  // fixed number of cycles
            st->converged = 1;
            stop = true;
        }
        if (!stop && cycles >= p.max_cycles) {
            st->status = DI_ERR_NOT_CONVERGED;
            stop = true;
        }
        for (int k = 0; k < p.nslots; ++k) upd[k] = 0u;
        if (stop) bs.done[i] = 1;
        else running = 1;
    }
    if (running) atomicOr(&s_any, 1);
    __syncthreads();
    if (threadIdx.x == 0) cudaGraphSetConditional(h, s_any ? 1u : 0u);
}

// Timing event on s; inside a stream capture it becomes an event record node
// of the graph (recorded by every replay).
void record_event(cudaEvent_t e, cudaStream_t s) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
        cudaEventRecordWithFlags(e, s, cudaEventRecordExternal);
    else
        cudaEventRecord(e, s);
}

inline dim3 grid2(int w, int h, dim3 blk, int z = 1) {
    return dim3((unsigned)((w + blk.x - 1) / blk.x), (unsigned)((h + blk.y - 1) / blk.y),
                (unsigned)z);
}

template <int B>
cudaError_t launch_combine(const float* parked, int w, int h, int C, int o, int nbx, int nby,
                           float* u_out, cudaStream_t s, int stor);

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
    static std::once_flag once;
    static EncodeTiledFn fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// Tensor map of an FP32 [C][h][w] image with a (bw x bh x 1) box; false if
// the image does not meet TMA's rules (w a multiple of 4, 16-byte base).
bool make_map(CUtensorMap* m, const float* base, int w, int h, int C, int bw, int bh) {
    EncodeTiledFn fn = encode_tiled();
    if (!fn || !base || w % 4 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)C};
    const cuuint64_t strides[2] = {(cuuint64_t)w * 4, (cuuint64_t)w * h * 4};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// Resident CTAs per SM of a kernel at a shared-memory size, and the SM count,
// cached per (device, kernel, shared-memory size): a process may drive
// several GPUs.
int cached_occupancy(const void* kern, int threads, size_t smem, size_t smem_max, int* nsm_out) {
    static std::mutex occ_mu;
    constexpr int kSlots = 64;
    static int occ_dev[kSlots];
    static const void* occ_fn[kSlots] = {};
    static size_t occ_key[kSlots] = {};
    static int occ_val[kSlots] = {};
    static int occ_nsm[kSlots] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> occ_lock(occ_mu);
    for (int i = 0; i < kSlots; ++i)
        if (occ_fn[i] == kern && occ_key[i] == smem && occ_dev[i] == dev) {
            *nsm_out = occ_nsm[i];
            return occ_val[i];
        }
    int nsm = 0, oc = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&oc, kern, threads, smem);
    if (oc < 1) oc = 1;
    if (nsm < 1) nsm = 1;
    for (int i = 0; i < kSlots; ++i)
        if (occ_fn[i] == nullptr) {
            occ_fn[i] = kern;
            occ_key[i] = smem;
            occ_dev[i] = dev;
            occ_val[i] = oc;
            occ_nsm[i] = nsm;
            break;
        }
    *nsm_out = nsm;
    return oc;
}

// The 16-bit block kernel for iterate type H and storage TU.
template <class H, class TU, bool F64>
void run_oras_2w_h(int grid, size_t smem, cudaStream_t s, const float* u_in, int zero_in,
                   const float* rhs, int rhs_zero, const uint32_t* mbits, int wpr, int w, int h,
                   int C, int o, int nbx, int nby, float alpha, int iters, float rtol2,
                   float* u_out, float* parked, unsigned* maxupd, int chan_inner,
                   unsigned long long* step_count) {
    k_oras_2w_h<H, TU, F64><<<grid, 64, smem, s>>>(
        reinterpret_cast<const TU*>(u_in), zero_in, reinterpret_cast<const TU*>(rhs), rhs_zero,
        mbits, wpr, w, h, C, o, nbx, nby, alpha, iters, rtol2, reinterpret_cast<TU*>(u_out),
        parked, maxupd, chan_inner, step_count);
}

template <class H, class TU, bool F64>
const void* oras_2w_h_fn() {
    return (const void*)k_oras_2w_h<H, TU, F64>;
}

// Local problems of a launch up to which the four-warp form takes it: four per
// SM of the 152, what is resident at once (at 80 registers for six, the 256x256 decode took
// 218 us instead of 211).
// Decodes of 256x256 / 481x321 RGB / 1920x1080 RGB with the line at 0, 1, 2, 4
// and 6 per SM: 249, 212, 212, 211, 211 / 432, 404, 396, 394, 393 / 1115, 1094,
// 1094, 1091, 1088 us; four 4K decodes in flight 4764, 4749, 4755, 4771, 4769.
constexpr int kQuadTasks = 152 * 4;

// precision: 0 FP32 iterates (tiles by TMA where the image allows it), 1 FP16,
// 2 BF16 iterates; stor: storage of u_in, rhs, u_out (kF32, or the iterate
// type on the coarse levels of the 16-bit modes); f64: FP64 block residual.
// pro_e: coarser level's correction (pro_mode 1) or solution (pro_mode 0)
// prolonged into the iteration's start (FP32 only; see k_oras_2w), largest
// |P e| of mode 1 into *pro_max.
cudaError_t launch_oras_2w(const float* u_in, int zero_in, const float* rhs, int rhs_zero,
                           const uint32_t* mbits, int wpr, int w, int h, int C, int o, float alpha,
                           int iters, float rtol2, float* u_out, float* parked, unsigned* maxupd,
                           cudaStream_t s, cudaEvent_t* ev, int precision, unsigned* errflag,
                           unsigned long long* step_count, int stor, bool f64,
                           const float* pro_e, unsigned* pro_max, int pro_mode) {
    constexpr int B = 32;
    if (stor != kF32 && stor != precision) return cudaErrorInvalidValue;
    if (pro_e && (!prolong_fusable(precision, o, zero_in) || (pro_mode != 0 && pro_mode != 1)))
        return cudaErrorInvalidValue;
    const int pm = pro_e ? (pro_mode == 1 ? 1 : 2) : 0;  // the kernel's PRO
    int wH = 0, hH = 0;
    coarse_dims(w, h, &wH, &hH);
    const int nbx = axis_blocks(w, B, o), nby = axis_blocks(h, B, o);
    const int ntasks = nbx * nby * C;
    const int nblk = nbx * nby;
    int nsm = 0, oc = 0;
    size_t smem = 0;
    const void* kern = nullptr;
    decltype(&k_oras_2w<false, 0, 0>) fn = nullptr;  // the FP32 kernel
    CUtensorMap tm_u, tm_b, tm_e;
    std::memset(&tm_u, 0, sizeof tm_u);
    std::memset(&tm_b, 0, sizeof tm_b);
    std::memset(&tm_e, 0, sizeof tm_e);
    int use_tma = 0, use_tma_e = 0;
    if (precision == 0) {
        use_tma = (!zero_in || !rhs_zero) &&
                  (zero_in || make_map(&tm_u, u_in, w, h, C, Smem2W::PU, Smem2W::TH)) &&
                  (rhs_zero || make_map(&tm_b, rhs, w, h, C, Smem2W::PB, B));
        use_tma_e = use_tma && pm != 0 &&
                    make_map(&tm_e, pro_e, wH, hH, C, Smem2W::EPW, Smem2W::EH);
        smem = Smem2W::bytes(!rhs_zero, pm != 0);
#define DI_ORAS_SEL(OV)                                                               \
    (pm == 1   ? (f64 ? k_oras_2w<true, 1, OV> : k_oras_2w<false, 1, OV>)              \
     : pm == 2 ? (f64 ? k_oras_2w<true, 2, OV> : k_oras_2w<false, 2, OV>)              \
               : (f64 ? k_oras_2w<true, 0, OV> : k_oras_2w<false, 0, OV>))
        fn = o == 2          ? DI_ORAS_SEL(0)
             : (o & 1) == 0  ? DI_ORAS_SEL(1)
             : f64           ? k_oras_2w<true, 0, 2>  // no fused prolongation (prolong_fusable)
                             : k_oras_2w<false, 0, 2>;
#undef DI_ORAS_SEL
        kern = (const void*)fn;
        oc = cached_occupancy(kern, 64, smem, Smem2W::bytes(true, pm != 0), &nsm);
    } else {
        smem = ((size_t)Tile2W::FIXED + (rhs_zero ? 0 : (size_t)2 * B * B)) * sizeof(float);
        if (precision == 1)
            kern = stor != kF32 ? oras_2w_h_fn<HalfT, __half, false>()
                   : f64        ? oras_2w_h_fn<HalfT, float, true>()
                                : oras_2w_h_fn<HalfT, float, false>();
        else
            kern = stor != kF32 ? oras_2w_h_fn<Bf16T, __nv_bfloat16, false>()
                   : f64        ? oras_2w_h_fn<Bf16T, float, true>()
                                : oras_2w_h_fn<Bf16T, float, false>();
        oc = cached_occupancy(kern, 64, smem, ((size_t)Tile2W::FIXED + (size_t)2 * B * B) *
                                                  sizeof(float), &nsm);
    }
    const int slots = nsm * oc;
    const int chan_inner = nblk >= slots ? 1 : 0;
    int grid = chan_inner ? slots : (ntasks < slots ? ntasks : slots);
    if (grid < 1) grid = 1;
    if (ev) record_event(ev[0], s);
    if (precision == 0 && !f64 && (o & 1) == 0 && ntasks <= kQuadTasks) {
        auto* const fn4 = o == 2 ? (pm == 1 ? k_oras_4w<1, 0> : pm == 2 ? k_oras_4w<2, 0> : k_oras_4w<0, 0>)
                                 : (pm == 1 ? k_oras_4w<1, 1> : pm == 2 ? k_oras_4w<2, 1> : k_oras_4w<0, 1>);
        fn4<<<ntasks, 128, 0, s>>>(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, nbx, nby,
                                   alpha, iters, rtol2, u_out, parked, maxupd, tm_u, tm_b, use_tma,
                                   errflag, step_count, pro_e, wH, hH, pro_max, tm_e, use_tma_e);
    } else if (precision == 0) {
        fn<<<grid, 64, smem, s>>>(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, nbx, nby,
                                  alpha, iters, rtol2, u_out, parked, maxupd, chan_inner, tm_u,
                                  tm_b, use_tma, errflag, step_count, pro_e, wH, hH, pro_max,
                                  tm_e, use_tma_e);
    } else {
#define DI_ORAS_H(H, TU, F)                                                                     \
    run_oras_2w_h<H, TU, F>(grid, smem, s, u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, \
                            nbx, nby, alpha, iters, rtol2, u_out, parked, maxupd, chan_inner,   \
                            step_count)
        if (precision == 1) {
            if (stor != kF32) DI_ORAS_H(HalfT, __half, false);
            else if (f64) DI_ORAS_H(HalfT, float, true);
            else DI_ORAS_H(HalfT, float, false);
        } else {
            if (stor != kF32) DI_ORAS_H(Bf16T, __nv_bfloat16, false);
            else if (f64) DI_ORAS_H(Bf16T, float, true);
            else DI_ORAS_H(Bf16T, float, false);
        }
#undef DI_ORAS_H
    }
    count();
    if (ev) record_event(ev[1], s);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_combine<B>(parked, w, h, C, o, nbx, nby, u_out, s, stor);
}

template <int B>
cudaError_t launch_oras_t(const float* u_in, int zero_in, const float* rhs, int rhs_zero,
                          const uint32_t* mbits, int wpr, int w, int h, int C, int o, float alpha,
                          int iters, float rtol2, float* u_out, float* parked, unsigned* maxupd,
                          cudaStream_t s, cudaEvent_t* ev,
                          unsigned long long* step_count) {
    const int nbx = axis_blocks(w, B, o), nby = axis_blocks(h, B, o);
    const int ntasks = nbx * nby * C;
    constexpr int FIXED = WarpTile<B>::FIXED;
    const size_t smem = (size_t)FIXED * sizeof(float) +
                        (rhs_zero ? 0 : (size_t)2 * B * B * sizeof(float));
    // persistent warps: as many as fit on the GPU at once
    int nsm = 0;
    const int oc = cached_occupancy((const void*)k_oras_warp<B>, 32, smem,
                                    FIXED * sizeof(float) + 2 * B * B * sizeof(float), &nsm);
    const int slots = nsm * oc;
    const int nblk = nbx * nby;
    const int chan_inner = nblk >= slots ? 1 : 0;
    int grid = chan_inner ? slots : (ntasks < slots ? ntasks : slots);
    if (grid < 1) grid = 1;
    if (ev) record_event(ev[0], s);
    k_oras_warp<B><<<grid, 32, smem, s>>>(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o,
                                          nbx, nby, alpha, iters, rtol2, u_out, parked, maxupd,
                                          chan_inner, step_count);
    count();
    if (ev) record_event(ev[1], s);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_combine<B>(parked, w, h, C, o, nbx, nby, u_out, s, kF32);
}

template <int B>
cudaError_t launch_combine(const float* parked, int w, int h, int C, int o, int nbx, int nby,
                           float* u_out, cudaStream_t s, int stor) {
    // Overlap 2 gives 0/1 weights: no pixel is shared, nothing to add.
    if (shared_per_seam(o) == 0 || nbx * nby == 1) return cudaSuccess;
    const dim3 grid((unsigned)((nbx * C + 7) / 8), (unsigned)nby, 3);
    constexpr int kRows = 8 * kCombineRows;  // of a CTA of k_combine_px
    if constexpr (B < 32)  // FP32 only
        k_combine_px<B><<<dim3((unsigned)((w + 31) / 32), (unsigned)((h + kRows - 1) / kRows),
                               (unsigned)C),
                          dim3(32, 8), 0, s>>>(parked, w, h, C, o, nbx, nby, u_out);
    else if (stor == kF16)
        k_combine<__half><<<grid, 256, 0, s>>>(parked, w, h, C, o, nbx, nby,
                                               reinterpret_cast<__half*>(u_out));
    else if (stor == kBF16)
        k_combine<__nv_bfloat16><<<grid, 256, 0, s>>>(parked, w, h, C, o, nbx, nby,
                                                      reinterpret_cast<__nv_bfloat16*>(u_out));
    else
        k_combine<float><<<grid, 256, 0, s>>>(parked, w, h, C, o, nbx, nby, u_out);
    count();
    return cudaGetLastError();
}

}  // namespace

bool make_tile_maps(void* out, const float* u_in, int zero_in, const float* rhs, int rhs_zero,
                    int w, int h, int C) {
    CUtensorMap* m = static_cast<CUtensorMap*>(out);
    std::memset(m, 0, 2 * sizeof(CUtensorMap));
    static_assert(2 * sizeof(CUtensorMap) == kTileMapsBytes, "two tensor maps");
    return (zero_in || make_map(&m[0], u_in, w, h, C, Smem2W::PU, Smem2W::TH)) &&
           (rhs_zero || make_map(&m[1], rhs, w, h, C, Smem2W::PB, 32));
}

// ---------------------------------------------------------------------------
// Launch wrappers
// ---------------------------------------------------------------------------

cudaError_t launch_mask_down(const uint8_t* c, int w, int h, uint8_t* cH, cudaStream_t s) {
    int wH, hH;
    coarse_dims(w, h, &wH, &hH);
    dim3 blk(32, 8);
    k_mask_down<<<grid2(wH, hH, blk), blk, 0, s>>>(c, w, h, cH, wH, hH);
    count();
    return cudaGetLastError();
}

cudaError_t launch_values_down(const uint8_t* c, const float* b, int w, int h, int C,
                               const uint8_t* cH, float* bH, int modified, cudaStream_t s) {
    int wH, hH;
    coarse_dims(w, h, &wH, &hH);
    dim3 blk(32, 8);
    k_values_down<<<grid2(wH, hH, blk), blk, 0, s>>>(c, b, w, h, C, cH, bH, wH, hH, modified);
    count();
    return cudaGetLastError();
}

size_t residual_partials_per_channel(int w, int h) {
    return (size_t)((w + kResBX - 1) / kResBX) * (size_t)((h + kResBY - 1) / kResBY);
}

cudaError_t launch_residual(const float* u, int zero_u, const float* b, int rhs_zero,
                            const uint8_t* c, int w, int h, int C, float* r, double* partials,
                            int* nparts, cudaStream_t s, bool f64) {
    dim3 blk(kResBX, kResBY);
    dim3 grid = grid2(w, h, blk, C);
    *nparts = (int)(grid.x * grid.y);
    if (f64)
        k_residual<true><<<grid, blk, 0, s>>>(u, zero_u, b, rhs_zero, c, w, h, r, partials);
    else
        k_residual<false><<<grid, blk, 0, s>>>(u, zero_u, b, rhs_zero, c, w, h, r, partials);
    count();
    return cudaGetLastError();
}

// Fixed reduction scratch for callers that cannot allocate (see
// di_residual_norm_noalloc in di.h).  Host code must not pass the symbol
// itself to a kernel: on the host it names a stand-in, not device memory.
// Its device address is looked up once per device and context, with that
// device current: a context that is destroyed and created again (a device
// reset) loads the module anew, so the address is keyed on the context's
// process-unique id, not on the device ordinal alone.
static __device__ __align__(256) double g_noalloc_partials[kNoAllocPartials];

typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

// Process-unique id of the calling thread's current context (0 if none).
unsigned long long current_context_id() {
    static std::once_flag once;
    static CtxGetCurrentFn get_cur = nullptr;
    static CtxGetIdFn get_id = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            get_cur = reinterpret_cast<CtxGetCurrentFn>(p);
        p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(p);
        cudaGetLastError();
    });
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_cur || !get_id || get_cur(&ctx) != CUDA_SUCCESS || !ctx ||
        get_id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

cudaError_t launch_residual_noalloc(const float* u, const float* b, int rhs_zero,
                                    const uint8_t* c, int w, int h, int C, float* r,
                                    double* norm2, cudaStream_t s) {
    static std::mutex mu;
    static double* addr[128] = {};
    static unsigned long long addr_ctx[128] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    double* scratch;
    {
        std::lock_guard<std::mutex> lock(mu);
        unsigned long long id = current_context_id();
        if (!addr[dev] || id == 0 || id != addr_ctx[dev]) {
            // first call on this device, or its context changed: (re)load
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_partials);
            if (e != cudaSuccess) return e;
            addr[dev] = static_cast<double*>(p);
            // the lookup makes the primary context current if none was
            if (id == 0) id = current_context_id();
            addr_ctx[dev] = id;
        }
        scratch = addr[dev];
    }
    int nparts = 0;
    e = launch_residual(u, 0, b, rhs_zero, c, w, h, C, r, scratch, &nparts, s);
    if (e != cudaSuccess) return e;
    return launch_reduce_partials(scratch, nparts, C, norm2, s);
}

cudaError_t launch_reduce_partials(const double* partials, int nparts, int C, double* out,
                                   cudaStream_t s) {
    k_reduce<<<C, 256, 0, s>>>(partials, nparts, out);
    count();
    return cudaGetLastError();
}

template <class TU, class TB, class TO, bool F64>
void run_restrict(dim3 grid, dim3 blk, cudaStream_t s, const float* u, const float* b,
                  int rhs_zero, int w, int h, const uint8_t* cH, float* rH, int wH, int hH) {
    k_restrict<false, TU, TB, TO, F64><<<grid, blk, 0, s>>>(
        reinterpret_cast<const TU*>(u), reinterpret_cast<const TB*>(b), rhs_zero, w, h, cH,
        reinterpret_cast<TO*>(rH), wH, hH);
}

cudaError_t launch_restrict(const float* u, const float* b, int rhs_zero, const uint8_t* c,
                            int w, int h, int C, const uint8_t* cH, float* rH, cudaStream_t s,
                            int su, int sb, int sr, bool f64) {
    (void)c;  // children of an unmasked coarse cell are unknown by construction
    int wH, hH;
    coarse_dims(w, h, &wH, &hH);
    dim3 blk(32, 8);
    const dim3 grid = grid2(wH, hH, blk, C);
    if (rhs_zero) sb = kF32;  // b is not read
    const bool vec = su == kF32 && sb == kF32 && (w % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(u) |
                       reinterpret_cast<uintptr_t>(rhs_zero ? nullptr : b)) % 8 == 0);
    // one thread for all channels of a cell where the level's cells still fill the
    // GPU's threads (three channels, mask density 0.04 / 0.9: at 960x540 cells 7.7 /
    // 4.0 us against 10.4 / 5.0, at 1920x1080 26.8 / 10.3 against 42.0 / 14.4; at
    // 480x270 3.9 / 2.3 against 4.1 / 2.5, but with a right-hand side at 0.5 4.4
    // against 3.8)
    if (su == kF32 && sb == kF32 && sr == kF32 && !f64 &&
        (long long)wH * hH >= 152LL * 2048 && hH <= 4 * 65535) {  // grid rows of 4
        const dim3 b1(32, restrict_rows(C)), g1 = grid2(wH, hH, b1);
#define DI_RESTRICT_C(NC)                                                         \
    (vec ? (rhs_zero ? k_restrict_c<NC, true, true> : k_restrict_c<NC, true, false>) \
         : (rhs_zero ? k_restrict_c<NC, false, true> : k_restrict_c<NC, false, false>))
        auto* const kern = C == 1   ? DI_RESTRICT_C(1)
                           : C == 2 ? DI_RESTRICT_C(2)
                           : C == 3 ? DI_RESTRICT_C(3)
                                    : DI_RESTRICT_C(4);
#undef DI_RESTRICT_C
        kern<<<g1, b1, 0, s>>>(u, b, w, h, cH, rH, wH, hH);
    } else if (su == kF32 && sb == kF32 && sr == kF32) {
        if (vec && f64)
            k_restrict<true, float, float, float, true><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, rH, wH, hH);
        else if (vec && (long long)grid.x * grid.y * grid.z <= 152 * 3)
            // few CTAs: a launch lasts as long as its loads one after the other
            // (480x270 RGB, mask density 0.04 / 0.9: 2.6 / 2.0 us, after the mask
            // byte 2.9 / 1.9); larger launches read no patch of a known cell
            // (960x540 gray 2.6 / 2.0 us, beside the byte 2.4 / 2.3; RGB 4.1 / 2.5,
            // 3.8 / 3.1)
            k_restrict<true, float, float, float, false, true><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, rH, wH, hH);
        else if (vec)
            k_restrict<true, float, float, float, false><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, rH, wH, hH);
        else if (f64)
            run_restrict<float, float, float, true>(grid, blk, s, u, b, rhs_zero, w, h, cH, rH, wH, hH);
        else
            run_restrict<float, float, float, false>(grid, blk, s, u, b, rhs_zero, w, h, cH, rH, wH,
                                                     hH);
    } else if (su == kF32 && sb == kF32 && sr == kF16) {  // finest level, FP16 coarse levels
        if (vec && f64)
            k_restrict<true, float, float, __half, true><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, reinterpret_cast<__half*>(rH), wH, hH);
        else if (vec)
            k_restrict<true, float, float, __half, false><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, reinterpret_cast<__half*>(rH), wH, hH);
        else if (f64)
            run_restrict<float, float, __half, true>(grid, blk, s, u, b, rhs_zero, w, h, cH, rH, wH, hH);
        else
            run_restrict<float, float, __half, false>(grid, blk, s, u, b, rhs_zero, w, h, cH, rH, wH,
                                                      hH);
    } else if (su == kF32 && sb == kF32 && sr == kBF16) {
        if (vec && f64)
            k_restrict<true, float, float, __nv_bfloat16, true><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, reinterpret_cast<__nv_bfloat16*>(rH), wH, hH);
        else if (vec)
            k_restrict<true, float, float, __nv_bfloat16, false><<<grid, blk, 0, s>>>(
                u, b, rhs_zero, w, h, cH, reinterpret_cast<__nv_bfloat16*>(rH), wH, hH);
        else if (f64)
            run_restrict<float, float, __nv_bfloat16, true>(grid, blk, s, u, b, rhs_zero, w, h, cH,
                                                            rH, wH, hH);
        else
            run_restrict<float, float, __nv_bfloat16, false>(grid, blk, s, u, b, rhs_zero, w, h, cH,
                                                             rH, wH, hH);
    } else if (su == kF16 && (sb == kF16 || rhs_zero) && sr == kF16) {  // coarse levels
        run_restrict<__half, __half, __half, false>(grid, blk, s, u, b, rhs_zero, w, h, cH, rH, wH,
                                                    hH);
    } else if (su == kBF16 && (sb == kBF16 || rhs_zero) && sr == kBF16) {
        run_restrict<__nv_bfloat16, __nv_bfloat16, __nv_bfloat16, false>(grid, blk, s, u, b,
                                                                         rhs_zero, w, h, cH, rH,
                                                                         wH, hH);
    } else {
        return cudaErrorInvalidValue;
    }
    count();
    return cudaGetLastError();
}

template <bool VEC, class TC, class TF>
void run_prolong(dim3 grid, dim3 blk, cudaStream_t s, const float* uH, int wH, int hH,
                 const float* b, const uint8_t* c, int w, int h, float* u, int mode,
                 unsigned* maxupd) {
    k_prolong<VEC, TC, TF><<<grid, blk, 0, s>>>(reinterpret_cast<const TC*>(uH), wH, hH, b, c, w,
                                                h, reinterpret_cast<TF*>(u), mode, maxupd);
}

cudaError_t launch_prolong(const float* uH, const float* b, const uint8_t* c, int w, int h,
                           int C, float* u, int mode, unsigned* maxupd, cudaStream_t s, int suH,
                           int su) {
    int wH, hH;
    coarse_dims(w, h, &wH, &hH);
    dim3 blk(32, 8);
    const dim3 grid = grid2(wH, hH, blk, C);  // one thread per coarse cell
    const bool vec = su == kF32 && (w % 2 == 0) &&
                     ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(b)) % 8 == 0) &&
                     reinterpret_cast<uintptr_t>(c) % 2 == 0;
    unsigned* mu = mode == 1 ? maxupd : nullptr;
    if (su == kF32) {
        if (suH == kF32) {
            if (vec) run_prolong<true, float, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u, mode, mu);
            else run_prolong<false, float, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u, mode, mu);
        } else if (suH == kF16) {
            if (vec) run_prolong<true, __half, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u, mode, mu);
            else run_prolong<false, __half, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u, mode, mu);
        } else {
            if (vec)
                run_prolong<true, __nv_bfloat16, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u,
                                                        mode, mu);
            else
                run_prolong<false, __nv_bfloat16, float>(grid, blk, s, uH, wH, hH, b, c, w, h, u,
                                                         mode, mu);
        }
    } else if (su == kF16 && suH == kF16) {
        run_prolong<false, __half, __half>(grid, blk, s, uH, wH, hH, b, c, w, h, u, mode, mu);
    } else if (su == kBF16 && suH == kBF16) {
        run_prolong<false, __nv_bfloat16, __nv_bfloat16>(grid, blk, s, uH, wH, hH, b, c, w, h, u,
                                                         mode, mu);
    } else {
        return cudaErrorInvalidValue;
    }
    count();
    return cudaGetLastError();
}

cudaError_t launch_select(const float* b, const uint8_t* c, int w, int h, int C, float* u,
                          cudaStream_t s, int keep, int su) {
    const size_t n = (size_t)w * h;
    size_t blocks = (n + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    if (blocks < 1) blocks = 1;
    const dim3 grid((unsigned)blocks, (unsigned)C);
    if (su == kF16)
        k_select<__half><<<grid, 256, 0, s>>>(b, c, n, reinterpret_cast<__half*>(u), keep);
    else if (su == kBF16)
        k_select<__nv_bfloat16><<<grid, 256, 0, s>>>(b, c, n, reinterpret_cast<__nv_bfloat16*>(u),
                                                     keep);
    else
        k_select<float><<<grid, 256, 0, s>>>(b, c, n, u, keep);
    count();
    return cudaGetLastError();
}

// Global CG smoother on one level: `steps` CG steps on A x = b - A in (known
// pixels fixed), out = in + x.  With restart == 0 the state in (r, p, sc) of
// the previous call on the same level continues (single-level CG).
cudaError_t launch_cg_smooth(const float* in, int zero_in, const float* b, int rhs_zero,
                             const uint8_t* c, int w, int h, int C, int steps, int restart,
                             float* r, float* p, float* q, float* x, double* partials, double* sc,
                             int* step_par, float* out, unsigned* maxupd, cudaStream_t s) {
    CgTiles g;
    g.w = w;
    g.h = h;
    g.tiles_x = (w + kCgBX - 1) / kCgBX;
    g.ntiles = g.tiles_x * ((h + kCgBY - 1) / kCgBY);
    int per_ch = kCgCtas / C;
    if (per_ch > g.ntiles) per_ch = g.ntiles;
    if (per_ch < 1) per_ch = 1;
    const dim3 grid((unsigned)per_ch, (unsigned)C), blk(kCgBX, kCgBY);
    const size_t n = (size_t)w * h;
    size_t nb = (n + 255) / 256;
    if (nb > 8192) nb = 8192;
    cudaError_t e;
    if (restart) {
        k_cg_init<<<grid, blk, 0, s>>>(g, in, zero_in, b, rhs_zero, c, r, p, x, partials);
        count();
        k_reduce_slot<<<C, 256, 0, s>>>(partials, per_ch, sc, 0);
        count();
        *step_par = 0;
    } else {
        // continue: the correction restarts from zero on top of the new iterate
        e = cudaMemsetAsync(x, 0, n * C * sizeof(float), s);
        if (e != cudaSuccess) return e;
    }
    for (int k = 0; k < steps; ++k) {
        const int par = *step_par;
        k_cg_matvec<<<grid, blk, 0, s>>>(g, p, c, q, partials);
        count();
        k_reduce_slot<<<C, 256, 0, s>>>(partials, per_ch, sc, 2);
        count();
        k_cg_update<<<grid, blk, 0, s>>>(g, p, q, x, r, sc, par, partials);
        count();
        k_reduce_slot<<<C, 256, 0, s>>>(partials, per_ch, sc, par ^ 1);
        count();
        k_cg_direction<<<dim3((unsigned)nb, (unsigned)C), 256, 0, s>>>(p, r, n, sc, par);
        count();
        *step_par = par ^ 1;
    }
    k_cg_finish<<<dim3((unsigned)nb, (unsigned)C), 256, 0, s>>>(in, zero_in, x, out, n, maxupd);
    count();
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(unsigned* flag, int limit, cudaStream_t s) {
    k_bounded_wait_selftest<<<1, 64, 0, s>>>(flag, limit);
    count();
    return cudaGetLastError();
}

int oras_quad_tasks() { return kQuadTasks; }

cudaError_t launch_pack_mask(const uint8_t* c, int w, int h, uint32_t* bits,
                             unsigned long long* unknown, cudaStream_t s) {
    const int wpr = mask_words_per_row(w);
    const long long words = (long long)h * wpr;
    if (words > 0x7fffffffLL) return cudaErrorInvalidValue;
    const unsigned rows32 = (unsigned)((h + 31) / 32);
    if (w % 16 == 0 && (reinterpret_cast<uintptr_t>(c) & 15) == 0 && rows32 <= 65535u) {
        k_pack_mask16<<<dim3((unsigned)((2 * wpr + 31) / 32), rows32), dim3(32, 8), 0, s>>>(
            c, w, h, bits, wpr, unknown);
        count();
        return cudaGetLastError();
    }
    long long blocks = (words + 31) / 32;  // 8 warps x 4 words per CTA pass
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks < 1) blocks = 1;
    k_pack_mask<<<(unsigned)blocks, 256, 0, s>>>(c, w, h, bits, wpr, unknown);
    count();
    return cudaGetLastError();
}

cudaError_t launch_oras(const float* u_in, int zero_in, const float* rhs, int rhs_zero,
                        const uint32_t* mbits, int w, int h, int C, int B, int o, float alpha,
                        int iters, float rtol2, float* u_out, float* parked, unsigned* maxupd,
                        cudaStream_t s, cudaEvent_t* ev, int precision, unsigned* errflag,
                        unsigned long long* step_count, int stor, bool f64, const float* pro_e,
                        unsigned* pro_max, int pro_mode) {
    const int wpr = mask_words_per_row(w);
    if (B != 32 && (stor != kF32 || f64 || pro_e)) return cudaErrorInvalidValue;
    switch (B) {
        case 32:
            return launch_oras_2w(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, alpha,
                                  iters, rtol2, u_out, parked, maxupd, s, ev, precision, errflag,
                                  step_count, stor, f64, pro_e, pro_max, pro_mode);
        case 16:
            return launch_oras_t<16>(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, alpha,
                                     iters, rtol2, u_out, parked, maxupd, s, ev, step_count);
        case 8:
            return launch_oras_t<8>(u_in, zero_in, rhs, rhs_zero, mbits, wpr, w, h, C, o, alpha,
                                    iters, rtol2, u_out, parked, maxupd, s, ev, step_count);
        default:
            return cudaErrorInvalidValue;
    }
}

cudaError_t launch_plan(const unsigned long long* counts, StopState* st, StopState* host,
                        const PlanParams& p, cudaStream_t s) {
    k_plan<<<1, 32, 0, s>>>(counts, st, host, p);
    count();
    return cudaGetLastError();
}

cudaError_t launch_stop(unsigned* upd, StopState* st, StopState* host, const StopParams& p,
                        unsigned long long h_loop, cudaStream_t s) {
    k_stop<<<1, 32, 0, s>>>(upd, st, host, p, (cudaGraphConditionalHandle)h_loop);
    count();
    return cudaGetLastError();
}

void batch_grid_dims(int kind, int w, int h, int* gx, int* gy) {
    if (kind == kBPack) {  // persistent warps over the packed words
        const long long words = (long long)h * mask_words_per_row(w);
        long long b = (words + 31) / 32;
        if (b > 152) b = 152;
        *gx = (int)(b < 1 ? 1 : b);
        *gy = 1;
    } else if (kind == kBSelect) {
        size_t b = ((size_t)w * h + 255) / 256;
        if (b > 1024) b = 1024;
        *gx = (int)(b < 1 ? 1 : b);
        *gy = 1;
    } else if (kind == kBRestrict || kind == kBPyramid) {  // a coarse cell per thread, 32 x 8 per CTA
        const int wH = (w + 1) / 2, hH = (h + 1) / 2;
        *gx = (wH + 31) / 32;
        *gy = (hH + 7) / 8;
    } else {
        *gx = *gy = 1;
    }
}

cudaError_t launch_batch_grid(int kind, const BatchSeg* segs, int nseg, int nctas,
                              const BatchState& bs, cudaStream_t s) {
    if (nctas < 1 || nseg < 1) return cudaSuccess;
    const dim3 blk2(32, 8), blk1(256);
    switch (kind) {
        case kBPack: k_batch_grid<kBPack><<<nctas, blk1, 0, s>>>(segs, nseg, bs); break;
        case kBSelect: k_batch_grid<kBSelect><<<nctas, blk1, 0, s>>>(segs, nseg, bs); break;
        case kBRestrict: k_batch_grid<kBRestrict><<<nctas, blk2, 0, s>>>(segs, nseg, bs); break;
        case kBPyramid: k_batch_grid<kBPyramid><<<nctas, blk2, 0, s>>>(segs, nseg, bs); break;
        default: return cudaErrorInvalidValue;
    }
    count();
    return cudaGetLastError();
}

cudaError_t launch_batch_oras(const BatchSeg* segs, int nseg, int nunits, int ntasks, int cmax,
                              int o, float alpha,
                              const BatchState& bs, cudaStream_t s) {
    if (nunits < 1 || nseg < 1) return cudaSuccess;
    if (shared_per_seam(o) != 0) return cudaErrorInvalidValue;  // 0/1 weights only
    if (ntasks <= kQuadTasks) {  // as for one image
        k_batch_oras_4w<<<nunits * cmax, 128, 0, s>>>(segs, nseg, cmax, o, alpha, bs);
        count();
        return cudaGetLastError();
    }
    int nsm = 0;
    const size_t smem = Smem2W::bytes(true, true);
    const int oc = cached_occupancy((const void*)k_batch_oras, 64, smem, smem, &nsm);
    int grid = nsm * oc;
    const int split = nunits < grid ? cmax : 0;
    const int work = split ? nunits * split : nunits;
    if (grid > work) grid = work;
    k_batch_oras<<<grid, 64, smem, s>>>(segs, nseg, nunits, split, o, alpha, bs);
    count();
    return cudaGetLastError();
}

cudaError_t launch_batch_plan(int n, const int* L, const unsigned long long* n0,
                              const BatchState& bs, cudaStream_t s) {
    k_batch_plan<<<(n + 127) / 128, 128, 0, s>>>(n, L, n0, bs);
    count();
    return cudaGetLastError();
}

cudaError_t launch_batch_stop(int n, const StopParams& p, const BatchState& bs,
                              unsigned long long h_loop, cudaStream_t s) {
    k_batch_stop<<<1, 256, 0, s>>>(n, p, bs, (cudaGraphConditionalHandle)h_loop);
    count();
    return cudaGetLastError();
}

cudaError_t launch_pyramid_level(const uint8_t* c, const float* b, int w, int h, int C,
                                 uint8_t* cH, float* bH, int modified, int values, uint32_t* bits,
                                 unsigned long long* unknown, cudaStream_t s) {
    int wH, hH;
    coarse_dims(w, h, &wH, &hH);
    const int wpr = mask_words_per_row(wH);
    // one CTA column per packed word of a coarse row but the padding word.  Once
    // one row of cells per thread would take more than one wave of CTAs: the list
    // over four rows each (longer lists fill the CTA's threads: at 3840x2160 RGB
    // 22.1 us against 24.7 with two rows), for the naive average, whose weights
    // are few instructions, two rows and no list (3840x2160 gray, mask density
    // 0.04 / 0.9: 16.8 / 18.0 us, with the list 15.8 / 26.7, one row 19.8 / 21.1;
    // RGB 29.8 / 29.7, 25.6 / 32.8, 31.9 / 31.8).  Smaller levels wait for one
    // step after the other: one row each and no list (1280x720 RGB at 0.04 / 0.9:
    // 5.8 / 5.7 us, with the list 7.2 / 7.4).
    const long long one = (long long)(wpr - 1) * ((hH + 7) / 8);
    const dim3 blk(32, 8);
    auto grid = [&](int rows) {
        return dim3((unsigned)(wpr - 1), (unsigned)((hH + 8 * rows - 1) / (8 * rows)));
    };
#define DI_PYRAMID(R, LIST, MOD)                                                                  \
    k_pyramid_level<R, LIST, MOD><<<grid(R), blk, 0, s>>>(c, b, w, h, C, cH, bH, wH, hH, values, \
                                                          bits, wpr, unknown)
    if (one > 152 * 6 && modified) DI_PYRAMID(4, true, true);
    else if (modified) DI_PYRAMID(1, false, true);
    else if (one > 152 * 6) DI_PYRAMID(2, false, false);
    else DI_PYRAMID(1, false, false);
#undef DI_PYRAMID
    count();
    return cudaGetLastError();
}

}  // namespace di

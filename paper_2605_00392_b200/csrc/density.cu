// Textual density rho of page images (Eq. 9; Appendix B): BT.601 grayscale, 3 x 3 Sobel gradient
// magnitude, threshold tau, fraction of edge pixels per token patch, mean over the patches.
//
// The counts are exact.  With 8-bit channels, 1000 * 255 * I = 299 R + 587 G + 114 B is an integer
// below 2^18, the Sobel sums are integers below 2^21 in magnitude, so all of them are exact in fp32, and
//     G >= tau   <=>   Gx_int^2 + Gy_int^2 >= (255000 tau)^2,
// the right side rounded up once by the host.  The difference of the two sides is formed in fp32 by two
// fused multiply-adds (error below 2^-22 of the threshold where it is small); a pixel that comes within 2^-21 of the
// threshold is decided again in 64-bit integers.
// Pixels outside the image take the value of the nearest pixel inside.
//
// A CTA owns a tile of up to 256 x 64 pixels.  It fetches the tile's rows and the one above and below (3 bytes per
// pixel, plus 16 bytes on either side for the ring) as one tiled TMA box (pages seen as 32-bit words); four such
// CTAs share an SM, so that one loads while the others compute.  A thread owns 16 adjacent columns of 8 rows (16 x 8
// threads: four warps, one for each scheduler of the SM) and walks down the rows:
//   * 16 pixels are 12 words of shared memory, read as three 16-byte vectors (48 bytes from lane to lane:
//     no bank conflicts); a pixel's gray value is two dp2a on the words as loaded, added to the bits of
//     1.5 x 2^23 (even rows) or subtracted from those of -1.5 x 2^23 (odd rows), so that the integer comes out as
//     a float, off by a bias that cancels in every sum below: rows u, m, d give d - u and (2 m + u) + d;
//   * from there two pixels per instruction (f32x2; pixel i is paired with pixel i + 8, so that a pixel's
//     left and right neighbours are whole register pairs too): vertical sums a = u + 2 m + d, b = d - u from
//     the two rows kept in registers, then gx, gy across, squares, comparison by the sign of the difference.
// What bounds it: 3 bytes per pixel from DRAM, 48 us for 64 pages of 1280 x 1280 at 6.55 TB/s, against 12 warp
// instructions per 32 pixels (2.8 of them dp2a, 4.4 packed fp32, which take the FMA pipes two cycles each).  Those
// pages: 141 us with integer gray values passed through shared memory and 64-bit comparisons (36 instructions per
// pixel), 70 us = 4.5 TB/s now.
#include <cstdint>
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include <cuda_runtime.h>

#include "../../include/rtprune.h"
#include "ptx.cuh"

namespace rtp {

constexpr int kDnBand = 64;                        // rows per CTA, at most
constexpr int kDnSeg = 256;                        // columns per CTA, at most: 16 threads of 16 columns
constexpr int kDnWalk = 8;                         // rows per thread
constexpr int kDnThreads = (kDnSeg / 16) * (kDnBand / kDnWalk);
constexpr int kDnRowPitch = kDnSeg * 3 + 32;       // bytes: 16 in front of the segment's first pixel, 16 behind
constexpr int kDnSmemBytes = (kDnBand + 2) * kDnRowPitch;         // 52 KB: four CTAs per SM

// 16-bit weight pairs (low half | high half << 16) for dp2a: low half times the lower byte of the selected byte pair
// of the data word, high half times the upper one.  SIGN = -1: the negative weights.
template <int SIGN> __host__ __device__ constexpr int weights(int lo, int hi) { return (SIGN * lo & 0xffff) | (int)((uint32_t)(SIGN * hi) << 16); }
// Bits of SIGN x 1.5 x 2^23: an integer n below 2^22 added to (subtracted from) them adds n to the value.
template <int SIGN> __host__ __device__ constexpr int magic() { return SIGN > 0 ? 0x4B400000 : (int)0xCB400000; }

typedef unsigned long long f32x2;                  // two floats in a register pair

__device__ inline f32x2 pack2(uint32_t lo, uint32_t hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ inline void unpack2(f32x2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ inline f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ inline f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ inline float min3_abs(float a, float b, float c)
{
    float r;
    asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ inline f32x2 both(float x) { return pack2(__float_as_uint(x), __float_as_uint(x)); }

__device__ inline int dp2a_lo(int w, uint32_t bytes, int c)
{
    int r;
    asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(bytes), "r"(c));
    return r;
}
__device__ inline int dp2a_hi(int w, uint32_t bytes, int c)
{
    int r;
    asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(bytes), "r"(c));
    return r;
}
// Bits of the (biased) gray value of the pixel whose three bytes are: the lower three of a word; the upper three;
// the top byte of a and the lower two of b; the upper two of a and the lowest of b.
template <int S> __device__ inline uint32_t gray_low3(uint32_t v)
{
    return (uint32_t)dp2a_lo(weights<S>(299, 587), v, dp2a_hi(weights<S>(114, 0), v, magic<S>()));
}
template <int S> __device__ inline uint32_t gray_high3(uint32_t v)
{
    return (uint32_t)dp2a_lo(weights<S>(0, 299), v, dp2a_hi(weights<S>(587, 114), v, magic<S>()));
}
template <int S> __device__ inline uint32_t gray_1_2(uint32_t a, uint32_t b)
{
    return (uint32_t)dp2a_hi(weights<S>(0, 299), a, dp2a_lo(weights<S>(587, 114), b, magic<S>()));
}
template <int S> __device__ inline uint32_t gray_2_1(uint32_t a, uint32_t b)
{
    return (uint32_t)dp2a_hi(weights<S>(299, 587), a, dp2a_lo(weights<S>(114, 0), b, magic<S>()));
}

// The gray values of one row at a thread's 16 pixels as floats: pair i + 1 holds pixels i and i + 8, pairs 0 and 9
// their neighbours at both ends.  `row` = shared memory of the thread's 48 bytes (16-byte aligned, a word of the
// ring before and after it).
template <int S> __device__ inline void dn_gray_row(const uint8_t *row, bool first_col, bool last_col, f32x2 (&p)[10])
{
    uint32_t w[12];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint4 v = *reinterpret_cast<const uint4 *>(row + 16 * k);
        w[4 * k] = v.x;
        w[4 * k + 1] = v.y;
        w[4 * k + 2] = v.z;
        w[4 * k + 3] = v.w;
    }
    uint32_t left = gray_high3<S>(*reinterpret_cast<const uint32_t *>(row - 4));
    uint32_t right = gray_low3<S>(*reinterpret_cast<const uint32_t *>(row + 48));
    uint32_t g[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {                  // four pixels in three words: R G B R | G B R G | B R G B
        g[4 * k] = gray_low3<S>(w[3 * k]);
        g[4 * k + 1] = gray_1_2<S>(w[3 * k], w[3 * k + 1]);
        g[4 * k + 2] = gray_2_1<S>(w[3 * k + 1], w[3 * k + 2]);
        g[4 * k + 3] = gray_high3<S>(w[3 * k + 2]);
    }
    if (first_col) left = g[0];                    // beyond the image's border: the nearest pixel inside
    if (last_col) right = g[15];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i + 1] = pack2(g[i], g[i + 8]);
    p[0] = pack2(left, g[7]);
    p[9] = pack2(g[8], right);
}

// Edge pixels of the decision in exact arithmetic minus those of the fp32 decision, over pairs whose sum of
// squares came close to the threshold.
__device__ __noinline__ int dn_exact_pair(f32x2 gx, f32x2 gy, float T, unsigned long long thr2)
{
    float x[2], y[2];
    unpack2(gx, x[0], x[1]);
    unpack2(gy, y[0], y[1]);
    int corr = 0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const long long ix = (long long)x[e], iy = (long long)y[e];
        const bool exact = (unsigned long long)(ix * ix + iy * iy) >= thr2;
        const bool fast = fmaf(x[e], x[e], fmaf(y[e], y[e], -T)) >= 0.f;
        corr += (exact ? 1 : 0) - (fast ? 1 : 0);
    }
    return corr;
}

// Zeroes the counters the tile kernel adds to and the place of its marks (its grid dependency).
__global__ void density_clear_kernel(uint32_t *__restrict__ image_counts, float *__restrict__ rho, int batch,
                                     int32_t *__restrict__ edge_counts, int patches)
{
    ptx::grid_dep_launch();
    const int n = blockDim.x * gridDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int i = i0; i < batch; i += n) {
        image_counts[i] = 0;
        rho[i] = 0.f;
    }
    for (int i = i0; i < patches; i += n) edge_counts[i] = 0;
}

// grid = (segments of seg_w columns, bands of band_h rows, batch).  Launched as a programmatic dependent of
// density_clear_kernel.  A CTA whose wait for its pixels runs out (poll_limit) marks its image's rho with NaN and waits
// once more, with the full limit, for the copy that is on its way into its shared memory.
__global__ void __launch_bounds__(kDnThreads, 4)
density_tile_kernel(const __grid_constant__ CUtensorMap map, int H, int W, int p, int seg_w, int band_h,
                    unsigned long long thr2, int32_t *__restrict__ edge_counts, uint32_t *__restrict__ image_counts,
                    float *__restrict__ rho, uint32_t poll_limit)
{
    extern __shared__ __align__(128) uint8_t tile[];
    __shared__ uint64_t s_full;
    __shared__ int s_cnt[(kDnBand / 16) * (kDnSeg / 16)], s_total;     // of each (partial) patch: [row][16 columns]
    const int walk = threadIdx.y, xt = 16 * threadIdx.x;       // rows kDnWalk * walk .., columns xt .. of the tile
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nth = blockDim.x * blockDim.y;
    const int img = blockIdx.z, x0 = blockIdx.x * seg_w, y0 = blockIdx.y * band_h;
    const int sw = min(seg_w, W - x0), bh = min(band_h, H - y0);        // multiples of 16
    const int pr = min(p, band_h);                   // rows of a patch within the band
    const int shift = 31 - __clz(p), pshift = 31 - __clz(pr);           // (powers of two)
    ptx::grid_dep_launch();
    if (tid == 0) {
        ptx::mbar_init(&s_full, 1);
        ptx::fence_mbar_init();
        s_total = 0;
    }
    for (int i = tid; i < (kDnBand / 16) * (kDnSeg / 16); i += nth) s_cnt[i] = 0;
    __syncthreads();

    // rows y0 - 1 .. y0 + band_h, 16 bytes in front of the first pixel (what lies outside the pages arrives as zeros
    // and is replaced below)
    if (tid == 0) {
        ptx::mbar_arrive_expect_tx(&s_full, (uint32_t)((band_h + 2) * kDnRowPitch));
        ptx::tma_load_3d(ptx::smem_u32(tile), &map, &s_full, (3 * x0 - 16) / 4, y0 - 1, img);
    }
    const bool landed = ptx::mbar_wait(&s_full, 0, poll_limit);
    if (!landed) {
        (void)ptx::mbar_wait(&s_full, 0);
        ptx::grid_dep_wait();                         // (rho has been cleared)
        rho[img] = __int_as_float(0x7fffffff);
    }
    if (landed && kDnWalk * walk < bh && xt < sw) {
        const bool first_col = x0 + xt == 0, last_col = x0 + xt + 16 == W;
        const uint8_t *base = tile + kDnWalk * walk * kDnRowPitch + 16 + 3 * xt;
        const float T = (float)thr2, tol = T * 4.7683716e-7f;            // 2^-21
        const f32x2 minus_T = both(-T), two = both(2.f), minus = both(-1.f);
        f32x2 r0[10], r1[10];                         // the row above and the row of the sums taken next, in turn
        int below = 0, corr = 0;                      // pixels under the threshold; exact decisions that differ
        dn_gray_row<1>(y0 + kDnWalk * walk == 0 ? base + kDnRowPitch : base, first_col, last_col, r0);
        dn_gray_row<-1>(base + kDnRowPitch, first_col, last_col, r1);
        const uint8_t *last = base + (y0 + kDnWalk * (walk + 1) == H ? kDnWalk : kDnWalk + 1) * kDnRowPitch;
        // one row of sums: u the row above, m the row itself; the row below takes u's place
        auto row_of_sums = [&](auto sign, f32x2 (&u)[10], f32x2 (&m)[10], const uint8_t *row) {
            f32x2 g[10];
            dn_gray_row<decltype(sign)::value>(row, first_col, last_col, g);
            f32x2 a0 = add2(fma2(m[0], two, u[0]), g[0]), b0 = fma2(u[0], minus, g[0]);
            f32x2 a1 = add2(fma2(m[1], two, u[1]), g[1]), b1 = fma2(u[1], minus, g[1]);
            u[0] = g[0];
            u[1] = g[1];
#pragma unroll
            for (int part = 0; part < 2; ++part) {             // four pairs at a time: gx and gy stay in registers
                float near = 3.0e38f;
                f32x2 gx[4], gy[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = 4 * part + e + 2;
                    const f32x2 a2 = add2(fma2(m[i], two, u[i]), g[i]), b2 = fma2(u[i], minus, g[i]);
                    u[i] = g[i];
                    gx[e] = fma2(a0, minus, a2);
                    gy[e] = fma2(b1, two, add2(b0, b2));
                    a0 = a1;
                    a1 = a2;
                    b0 = b1;
                    b1 = b2;
                    const f32x2 v = fma2(gx[e], gx[e], fma2(gy[e], gy[e], minus_T));
                    float x, y;
                    unpack2(v, x, y);
                    below += (int)(__float_as_uint(x) >> 31);
                    below += (int)(__float_as_uint(y) >> 31);
                    near = min3_abs(near, x, y);
                }
                if (near < tol) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) corr += dn_exact_pair(gx[e], gy[e], T, thr2);
                }
            }
        };
#pragma unroll                                        // (whole: no registers are moved from row to row)
        for (int r = 0; r < kDnWalk; r += 2) {
            row_of_sums(std::integral_constant<int, 1>(), r0, r1, base + (r + 2) * kDnRowPitch);
            row_of_sums(std::integral_constant<int, -1>(), r1, r0, r + 3 > kDnWalk ? last : base + (r + 3) * kDnRowPitch);
        }
        // eight rows of one patch row (patches are 16 rows at least)
        const int count = 16 * kDnWalk - below + corr;
        atomicAdd(&s_cnt[((kDnWalk * walk) >> pshift) * (kDnSeg / 16) + (xt >> shift)], count);
        atomicAdd(&s_total, count);
    }
    __syncthreads();
    // the band's patches are whole (stored) or shared with the bands below and above (added)
    ptx::grid_dep_wait();                             // the counters have been cleared
    if (edge_counts) {
        const int ncol = (sw + p - 1) >> shift, ncell = (bh >> pshift) * (kDnSeg / 16);
        for (int i = tid; i < ncell; i += nth) {
            const int pi = i / (kDnSeg / 16), pj = i % (kDnSeg / 16);
            if (pj >= ncol) continue;
            int32_t *e = edge_counts + ((size_t)img * (H >> shift) + ((y0 + pi * pr) >> shift)) * (W >> shift) + (x0 >> shift) + pj;
            if (pr == p) *e = s_cnt[i];
            else atomicAdd(e, s_cnt[i]);
        }
    }
    if (tid == 0) atomicAdd(image_counts + img, (uint32_t)s_total);
}

// rho = average over the patches of (edge pixels / patch pixels); the patches are equal, so this is the
// image's edge pixels over its pixels.  A marked image (NaN) stays so and counts UINT32_MAX.
__global__ void density_finish_kernel(uint32_t *__restrict__ image_counts, int batch, float inv_pixels,
                                      float *__restrict__ rho)
{
    ptx::grid_dep_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= batch) return;
    if (isnan(rho[i])) image_counts[i] = 0xffffffffu;
    else rho[i] = (float)image_counts[i] * inv_pixels;
}

// Launch that may begin while the kernel ahead of it in the stream drains (it waits for it itself).
template <typename... KArgs, typename... Args>
static cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The pages as a 3-D tensor of 32-bit words (x, row, page); boxes of one tile.
static bool pages_map(CUtensorMap *map, const uint8_t *images, int batch, int H, int W, int band_h)
{
    typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                      const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static std::atomic<void *> encode{nullptr};       // the driver's entry point, looked up once
    void *fn = encode.load(std::memory_order_relaxed);
    if (!fn) {
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            return false;
        encode.store(fn, std::memory_order_relaxed);
    }
    const cuuint64_t dims[3] = {(cuuint64_t)W * 3 / 4, (cuuint64_t)H, (cuuint64_t)batch};
    const cuuint64_t strides[2] = {(cuuint64_t)W * 3, (cuuint64_t)W * 3 * (cuuint64_t)H};
    const cuuint32_t box[3] = {kDnRowPitch / 4, (cuuint32_t)band_h + 2, 1}, unit[3] = {1, 1, 1};
    return ((EncodeTiledFn)fn)(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<uint8_t *>(images), dims, strides, box,
                               unit, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// rtprune_density, the waits for pixels giving up after poll_limit polls.
static rtprune_status_t launch_density(void *cuda_stream, const uint8_t *images, int32_t batch, int32_t height, int32_t width,
                                       int32_t patch, float tau, float *rho, uint32_t *image_counts, int32_t *edge_counts,
                                       uint32_t poll_limit)
{
    if (batch < 0 || height <= 0 || width <= 0) return RTPRUNE_ERR_INVALID_ARG;
    if (patch != 16 && patch != 32 && patch != 64) return RTPRUNE_ERR_UNSUPPORTED;
    if (height % patch || width % patch) return RTPRUNE_ERR_UNSUPPORTED;
    if (!(tau >= 0.f) || !std::isfinite(tau)) return RTPRUNE_ERR_INVALID_ARG;
    if (batch == 0) return RTPRUNE_OK;
    if (!images || !rho || !image_counts || ((uintptr_t)images & 15u)) return RTPRUNE_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // G >= tau  <=>  Gx_int^2 + Gy_int^2 >= (255000 tau)^2; the left side is an integer
    const double t = (double)tau * 255000.0;
    const double t2 = std::ceil(t * t);
    const unsigned long long thr2 = t2 >= 1.8e19 ? ~0ull : (unsigned long long)t2;
    if (batch > 65535 || (height + kDnBand - 1) / kDnBand > 65535) return RTPRUNE_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return RTPRUNE_ERR_CUDA;
    // columns: equal segments, multiples of 64 (whole patches)
    const int nseg = (width + kDnSeg - 1) / kDnSeg;
    const int seg_w = std::min(kDnSeg, ((width + nseg - 1) / nseg + 63) / 64 * 64);
    const int nx = (width + seg_w - 1) / seg_w;
    // rows: bands of 64; of 16 when those would leave half the device idle (the two extra rows of a band then cost
    // an eighth instead of a thirty-second)
    int band_h = kDnBand;
    while (band_h > 16 && (long long)batch * nx * ((height + band_h - 1) / band_h) < 2LL * sms) band_h >>= 1;
    const int patches = (edge_counts && band_h < patch) ? batch * (height / patch) * (width / patch) : 0;
    const int n_clear = std::max((int)batch, patches);
    density_clear_kernel<<<std::min((n_clear + 255) / 256, sms), 256, 0, st>>>(image_counts, rho, batch, edge_counts, patches);
    CUtensorMap map;
    if (!pages_map(&map, images, batch, height, width, band_h)) return RTPRUNE_ERR_CUDA;
    // the attribute is the function's, per device: set once on each (a bit of the mask)
    static std::atomic<unsigned long long> attribute_set{0};
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(attribute_set.load(std::memory_order_relaxed) & bit)) {
        if (cudaFuncSetAttribute(density_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDnSmemBytes) != cudaSuccess)
            return RTPRUNE_ERR_CUDA;
        if (dev < 64) attribute_set.fetch_or(bit, std::memory_order_relaxed);
    }
    const dim3 threads((unsigned)(std::min(seg_w, (int)width) / 16), (unsigned)(band_h / kDnWalk));
    const dim3 grid((unsigned)nx, (unsigned)((height + band_h - 1) / band_h), (unsigned)batch);
    if (launch_dependent(density_tile_kernel, grid, threads, (size_t)kDnSmemBytes, st, map, height, width, patch,
                         seg_w, band_h, thr2, edge_counts, image_counts, rho, poll_limit) != cudaSuccess)
        return RTPRUNE_ERR_CUDA;
    if (launch_dependent(density_finish_kernel, dim3((unsigned)(batch + 255) / 256), dim3(256), (size_t)0, st,
                         image_counts, batch, 1.f / ((float)height * (float)width), rho) != cudaSuccess)
        return RTPRUNE_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? RTPRUNE_OK : RTPRUNE_ERR_CUDA;
}

}  // namespace rtp

extern "C" rtprune_status_t rtprune_density(void *cuda_stream, const uint8_t *images, int32_t batch, int32_t height,
                                            int32_t width, int32_t patch, float tau, float *rho,
                                            uint32_t *image_counts, int32_t *edge_counts)
{
    return rtp::launch_density(cuda_stream, images, batch, height, width, patch, tau, rho, image_counts, edge_counts,
                               rtp::ptx::kSpinLimit);
}

extern "C" rtprune_status_t rtprune_test_density_expired(void *cuda_stream, const uint8_t *images, int32_t batch,
                                                         int32_t height, int32_t width, int32_t patch, float tau,
                                                         float *rho, uint32_t *image_counts, int32_t *edge_counts)
{
    return rtp::launch_density(cuda_stream, images, batch, height, width, patch, tau, rho, image_counts, edge_counts, 0u);
}

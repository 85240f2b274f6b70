// Dustbin-augmented optimal transport by Sinkhorn iterations (Eq. 5, Appendix C) in scaling form, the rows (kept
// tokens) of an image's score tile shared out over the CTAs of a cluster and, inside a CTA, over its warps: a warp
// takes whole rows.  Tiles of up to 639 pruned tokens.
//
// The duals are carried as U = e^u, V = e^{v + c/eps} against K_ij = exp((S_ij - c)/eps), c = max(1, z),
// so that U_i K_ij V_j = exp(Z_ij + u_i + v_j) (Appendix C) after any number of iterations:
//     U_i = mu_i / sum_j K_ij V_j          V_j = nu_j / sum_i K_ij U_i          mu = [1_M, B], nu = [1_B, M].
// The dustbin row and column of S-bar are the constant z (Eq. 5), kappa = exp((z - c)/eps) in K.  They are stored as a row
// and a column of ones with 1/kappa where they meet, and their duals as kappa U_d, kappa V_d: then they are rows and
// columns like the others, but for their marginals.
//
// One iteration is one pass over K.  LR lanes share a row (8 or 16 when the tile is narrow, else the warp); a lane owns
// NQ 16-byte column chunks of every row of its warp, so V and the column sums stay in registers over the pass.  RB rows
// are taken at a time: their RB row sums are completed by a halving shuffle tree (9 shuffles for 8 rows over 32
// lanes), every lane inverts one of them and the reciprocals are handed round in shared memory; multiply-adds run on
// column pairs (f32x2).  The warps' column sums meet in shared memory; with several CTAs every one sends its sums to all
// the others by asynchronous stores counted on a barrier there, and adds the parts in rank order: bit-identical duals
// everywhere, no cluster barrier in the loop.
//
// A CTA keeps as many of its rows of K as fit in shared memory (they are fetched by bulk copies, being contiguous, and
// exponentiated in place), the rest lies in the workspace tile (L2).  How many CTAs of the launched cluster work on an
// image is decided per image (sr_ctas): an exchange costs about as much as a pass over 20 000 cells.
// Large batches of narrow tiles run with half the threads and shared memory per CTA, two to an SM (the rule is where the kernel
// is launched).
//
// What bounds it: shared-memory reads of K and instruction latency; on a 300 x 100 tile on one CTA an iteration is
// 4200 cycles (pass 3000, column sums, V and two barriers the rest).  Measured by events around the kernel, against the
// kernel before it (16 warps walking rows one by one, a cluster barrier per iteration): 128 images of 456-1156 tokens
// 209 -> 149 us, 1024 x 400 at r = 0.25 288 -> 243 us, 256 x 400 in fp32 storage 119 -> 78 us, 64 images of 456-1156
// tokens at eps = 0.1 (31 iterations on average) 834 -> 475 us.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"
#include "settled.h"
#include "sinkhorn.cuh"

namespace rtp {

__device__ inline float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// exp(x) by the hardware base-2 exponential (relative error about 2^-22).
__device__ inline float exp_fast(float x) { return exp2f(x * 1.4426950408889634f); }

constexpr int kSrThreads = 512;                // of a CTA that has an SM to itself; half as many where two share one,
constexpr int kSrHalfSmemBytes = 111 * 1024;   // and half of its 228 KB then (1 KB per CTA is the system's, 1 KB static)
constexpr int kSrMaxB = 639;
constexpr int kSrMaxC = 8;                     // CTAs per image at most
constexpr int kSrChunks = 8;                   // bulk copies a CTA's rows of S arrive in

// Columns (floats) the lanes of a row cover for B pruned tokens and the dustbin.
__host__ __device__ inline int sr_width(int B) { return B < 32 ? 32 : (B < 64 ? 64 : (B + 128) & ~127); }
// Rows of a warp's batch (at most): K in shared memory is padded to whole batches.
__host__ __device__ inline int sr_batch_rows(int B) { return B < 64 ? 32 : (B < 128 ? 16 : (B < 256 ? 8 : 4)); }
// Floats of shared memory besides K: the warps' column sums (the pairing's values and indices take their place), the
// CTAs' column sums of two iterations, V, and U per row (of whole batches).
__host__ __device__ inline int sr_aux_floats(int B, int C, int rows, int warps)
{
    const int w = sr_width(B);
    return 2 * warps * w + (C > 1 ? 2 * C * w : 0) + w + ((rows + 33) & ~3);
}
// Shared-memory rows of K for `rows` kept tokens: those and the dustbin's, in whole batches.
__host__ __device__ inline int sr_smem_rows(int B, int rows)
{
    const int br = sr_batch_rows(B);
    return (rows + 1 + br - 1) / br * br;
}
// CTAs (1, 2, 4 or 8, at most C) that work on an M x B tile: enough for K to fit in their shared memory and for each to
// have at most `spread` cells.
__host__ __device__ inline int sr_ctas(int M, int B, int C, int smem_floats, int spread, int warps)
{
    int c = 1;
    while (c < C) {
        const int rows = (M + c - 1) / c;
        const long long cells = (long long)sr_smem_rows(B, rows) * score_pitch(B);
        if (cells + sr_aux_floats(B, c, rows, warps) <= smem_floats && cells <= spread) break;
        c *= 2;
    }
    return c;
}

struct SrTile {
    int M, B, Ml, row_lo;       // the image's tile; this CTA's kept tokens
    int Mr;                     // its rows: those and, on the last CTA, the dustbin's
    int C;                      // CTAs at work on the image
    uint32_t rank;
    int ld;                     // pitch of K: B columns, the dustbin's, up to a multiple of 4
    int cap;                    // rows of K in shared memory (whole batches), the others are in the workspace
    float *Ks;                  // [cap][ld]
    float *Kg;                  // this CTA's first row in the workspace tile
    float *part, *xpart, *vs, *us;
    uint64_t *xbar, *cbar;      // [2] column sums of the other CTAs; [kSrChunks] copies of S
};

typedef unsigned long long sr_f32x2;
__device__ inline sr_f32x2 sr_pack(float lo, float hi)
{
    sr_f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ inline void sr_unpack(sr_f32x2 v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ inline sr_f32x2 sr_fma2(sr_f32x2 a, sr_f32x2 b, sr_f32x2 c)
{
    sr_f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ inline sr_f32x2 sr_add2(sr_f32x2 a, sr_f32x2 b)
{
    sr_f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Sums of RB values over groups of LR lanes; lane l of a group ends up with the total of value sr_row_of_lane(l).  Every
// step over the first log2(RB) hands half of the values a lane carries to its partner.
template <int LR, int RB> __device__ inline float sr_tree(float (&s)[RB], int lane)
{
    if constexpr (RB > 1) {
        float t[RB / 2];
        const bool hi = lane & (LR / 2);
#pragma unroll
        for (int i = 0; i < RB / 2; ++i)
            t[i] = (hi ? s[i + RB / 2] : s[i]) + __shfl_xor_sync(0xffffffffu, hi ? s[i] : s[i + RB / 2], LR / 2);
        if constexpr (LR > 2) return sr_tree<LR / 2, RB / 2>(t, lane);
        else return t[0];
    } else {
        float t = s[0];
#pragma unroll
        for (int o = LR / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    }
}
// Value a lane's total belongs to.
template <int LR, int RB> __device__ inline int sr_row_of_lane(int lane)
{
    int r = 0;
#pragma unroll
    for (int b = RB / 2, o = LR / 2; b > 0; b >>= 1, o >>= 1) r |= (lane & o) ? b : 0;
    return r;
}

// One word into another CTA's shared memory, counted on a barrier there when it has landed.
__device__ inline void sr_send(uint32_t remote_addr, float v, uint32_t remote_bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(remote_addr), "r"(__float_as_uint(v)),
                 "r"(remote_bar)
                 : "memory");
}

struct SrState {
    int done;
    float last_move;
};

// exp((s - c)/eps) = 2^(a s + b), and the dustbin's column of ones in a row's last chunk.
__device__ inline float sr_exp2(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ inline float4 sr_k4(const float4 &s, float a, float b, int j, int B)
{
    float4 k = make_float4(sr_exp2(fmaf(s.x, a, b)), sr_exp2(fmaf(s.y, a, b)), sr_exp2(fmaf(s.z, a, b)), sr_exp2(fmaf(s.w, a, b)));
    if (j + 4 > B) {                               // the chunk that holds column B
        k.x = j < B ? k.x : (j == B ? 1.f : 0.f);
        k.y = j + 1 < B ? k.y : (j + 1 == B ? 1.f : 0.f);
        k.z = j + 2 < B ? k.z : (j + 2 == B ? 1.f : 0.f);
        k.w = j + 3 < B ? k.w : (j + 3 == B ? 1.f : 0.f);
    }
    return k;
}

// K of this CTA's rows.  The rows of S that stay in shared memory are contiguous in the workspace: bulk copies bring
// them (issued before the call, a lane each), every thread exponentiates in place what has landed.
__device__ inline bool sr_chunk_rows(const SrTile &t, int c, int &lo, int &hi)
{
    const int rows = min(t.cap, t.Ml), per = (rows + kSrChunks - 1) / kSrChunks;
    lo = min(rows, c * per);
    hi = min(rows, lo + per);
    return lo < hi;
}
__device__ inline void sr_fetch(const SrTile &t, int c)
{
    int lo, hi;
    if (!sr_chunk_rows(t, c, lo, hi)) return;
    const uint32_t bytes = (uint32_t)(hi - lo) * (uint32_t)t.ld * 4u;
    ptx::mbar_arrive_expect_tx(&t.cbar[c], bytes);
    ptx::bulk_load(ptx::smem_u32(t.Ks + (size_t)lo * t.ld), t.Kg + (size_t)lo * t.ld, bytes, &t.cbar[c]);
}
template <int TH>
__device__ inline void sr_build(const SrTile &t, float shift, float inv_eps, float inv_kappa, WsHeader *hdr)
{
    const int tid = threadIdx.x;
    const float a = inv_eps * 1.4426950408889634f, b = -shift * a;
    const int qpr = t.ld >> 2;
    const int dq = TH % qpr, q0 = tid % qpr;       // place in a row: of the thread's first chunk, and what a step adds
    for (int c = 0; c < kSrChunks; ++c) {
        int lo, hi;
        if (!sr_chunk_rows(t, c, lo, hi)) break;
        if (!ptx::mbar_wait(&t.cbar[c], 0)) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
        float4 *k = reinterpret_cast<float4 *>(t.Ks + (size_t)lo * t.ld);
        int q = q0;
        for (int i = tid; i < (hi - lo) * qpr; i += TH) {
            k[i] = sr_k4(k[i], a, b, 4 * q, t.B);
            q += dq;
            if (q >= qpr) q -= qpr;
        }
    }
    // rows beyond shared memory: in place in the workspace, four loads in flight
    if (t.cap < t.Ml) {
        float4 *k = reinterpret_cast<float4 *>(t.Kg + (size_t)t.cap * t.ld);
        const int n = (t.Ml - t.cap) * qpr;
        int q = q0;
        for (int i = tid; i < n; i += 4 * TH) {
            float4 v[4];
            int qq[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                qq[e] = q;
                q += dq;
                if (q >= qpr) q -= qpr;
                v[e] = i + e * TH < n ? __ldcg(k + i + e * TH) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (i + e * TH < n) k[i + e * TH] = sr_k4(v[e], a, b, 4 * qq[e], t.B);
        }
    }
    // the dustbin's row, and zeros up to a whole batch
    if (t.Mr > t.Ml) {
        float *p = (t.Ml < t.cap ? t.Ks : t.Kg) + (size_t)t.Ml * t.ld;
        for (int j = tid; j < t.ld; j += TH) p[j] = j < t.B ? 1.f : (j == t.B ? inv_kappa : 0.f);
    }
    if (t.Mr < t.cap)
        for (int j = tid; j < (t.cap - t.Mr) * t.ld; j += TH) t.Ks[(size_t)t.Mr * t.ld + j] = 0.f;
}

// A warp's work on a batch of BR rows: lane group `slot` takes the RB rows from base + RB * slot on.
template <int LR, int NQ, int RB>
struct SrPass {
    static constexpr int RPS = 32 / LR, BR = RB * RPS, W = LR * NQ * 4;
    sr_f32x2 V[NQ][2], acc[NQ][2];
    int lane, slot, my_r, off[NQ];
    bool writes_u;

    __device__ inline void init(const SrTile &t)
    {
        lane = threadIdx.x & 31;
        slot = lane / LR;
        my_r = slot * RB + sr_row_of_lane<LR, RB>(lane);
        writes_u = (lane & ((LR > RB ? LR / RB : 1) - 1)) == 0;
        // chunks past the row's end read its last one; V is zero there and nobody reads their sums
#pragma unroll
        for (int q = 0; q < NQ; ++q) off[q] = 4 * min(q * LR + lane % LR, (t.ld >> 2) - 1);
    }
    __device__ inline void begin(const float *vs)
    {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(vs + 4 * (q * LR + lane % LR));
            V[q][0] = sr_pack(v.x, v.y);
            V[q][1] = sr_pack(v.z, v.w);
            acc[q][0] = acc[q][1] = 0ull;
        }
    }
    // Row sums against V, U, column sums of the batch from row `base` on.
    __device__ inline void batch(const SrTile &t, int base, const float4 (&k)[RB][NQ])
    {
        float s[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            sr_f32x2 d0 = 0ull, d1 = 0ull;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                d0 = sr_fma2(sr_pack(k[r][q].x, k[r][q].y), V[q][0], d0);
                d1 = sr_fma2(sr_pack(k[r][q].z, k[r][q].w), V[q][1], d1);
            }
            float a, b;
            sr_unpack(sr_add2(d0, d1), a, b);
            s[r] = a + b;
        }
        const float tot = sr_tree<LR, RB>(s, lane);
        const int i = base + my_r;
        float U = rcp_fast(tot);
        if (i >= t.Ml) U = i < t.Mr ? U * (float)t.B : 0.f;        // the dustbin's row; a row that does not exist
        // every lane takes its rows' U from shared memory (two loads; eight shuffles would cost more)
        if (writes_u) t.us[i] = U;
        __syncwarp();
        float u[RB];
        if constexpr (RB >= 4) {
#pragma unroll
            for (int r = 0; r < RB; r += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(t.us + base + slot * RB + r);
                u[r] = v.x;
                u[r + 1] = v.y;
                u[r + 2] = v.z;
                u[r + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int r = 0; r < RB; ++r) u[r] = t.us[base + slot * RB + r];
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const sr_f32x2 uu = sr_pack(u[r], u[r]);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                acc[q][0] = sr_fma2(sr_pack(k[r][q].x, k[r][q].y), uu, acc[q][0]);
                acc[q][1] = sr_fma2(sr_pack(k[r][q].z, k[r][q].w), uu, acc[q][1]);
            }
        }
    }
    __device__ inline void load_smem(const SrTile &t, int base, float4 (&k)[RB][NQ]) const
    {
        const float *p = t.Ks + (size_t)(base + slot * RB) * t.ld;
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int q = 0; q < NQ; ++q) k[r][q] = *reinterpret_cast<const float4 *>(p + r * t.ld + off[q]);
    }
    __device__ inline void load_global(const SrTile &t, int base, float4 (&k)[RB][NQ]) const       // (rows clamped)
    {
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const float *p = t.Kg + (size_t)min(base + slot * RB + r, t.Mr - 1) * t.ld;
#pragma unroll
            for (int q = 0; q < NQ; ++q) k[r][q] = __ldcg(reinterpret_cast<const float4 *>(p + off[q]));
        }
    }
};

// This CTA's column sums to the other CTAs at work on the image, theirs added to them, in rank order.
template <int TH, int COLS, int W>
__device__ inline void sr_exchange(const SrTile &t, int it, float (&tot)[COLS], WsHeader *hdr)
{
    const int tid = threadIdx.x;
    const uint32_t par = (uint32_t)it & 1u, C = (uint32_t)t.C;
    const uint32_t at = ptx::smem_u32(t.xpart) + ((par * C + t.rank) * W + (uint32_t)tid) * 4u;
    const uint32_t bar = ptx::smem_u32(&t.xbar[par]);
    for (uint32_t r = 0; r < C; ++r) {
        if (r == t.rank) continue;
        const uint32_t to = ptx::map_to_rank(at, r), tobar = ptx::map_to_rank(bar, r);
#pragma unroll
        for (int e = 0; e < COLS; ++e)
            if (tid + e * TH <= t.B) sr_send(to + (uint32_t)(e * TH) * 4u, tot[e], tobar);
    }
    if (!ptx::mbar_wait(&t.xbar[par], ((uint32_t)it >> 1) & 1u)) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
#pragma unroll
    for (int e = 0; e < COLS; ++e) {
        if (tid + e * TH > t.B) continue;
        float sum = 0.f;
        for (uint32_t r = 0; r < C; ++r) sum += r == t.rank ? tot[e] : t.xpart[(par * C + r) * W + tid + e * TH];
        tot[e] = sum;
    }
}

// The iterations.  On return vs[] holds the final V (kappa V_d at [B]) and us[] the U of this CTA's rows.
template <int TH, int LR, int NQ, int RB>
__device__ inline SrState sr_iterate(const SrTile &t, const OtParams &p, float kappa, float v_init, WsHeader *hdr)
{
    typedef SrPass<LR, NQ, RB> Pass;
    constexpr int W = Pass::W, BR = Pass::BR;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float Mf = (float)t.M;
    __shared__ float2 s_range[(TH / 32)];               // smallest and largest relative move of a warp's columns
    for (int j = tid; j < W; j += TH) t.vs[j] = j < t.B ? v_init : (j == t.B ? kappa * v_init : 0.f);
    const int nbatch = (t.Mr + BR - 1) / BR, nsmem = min(nbatch, t.cap / BR);
    const int nwarps = min((TH / 32), nbatch);          // warps with rows; the others' column sums stay zero
    for (int j = nwarps * W + tid; j < (TH / 32) * W; j += TH) t.part[j] = 0.f;
    __syncthreads();                                   // K, V
    constexpr int kCols = (W + TH - 1) / TH;
    float nv[kCols], ov[kCols];                        // this thread's columns
    int before[kCols];                                 // and their values two iterations ago
#pragma unroll
    for (int e = 0; e < kCols; ++e) {
        nv[e] = ov[e] = tid + e * TH < t.B ? v_init : kappa * v_init;
        before[e] = 0;
    }
    SrState st{0, 0.f};
    Pass ps;
    ps.init(t);

    for (int it = 0; it < p.iters; ++it) {
        if (t.C > 1 && tid == 0)
            ptx::mbar_arrive_expect_tx(&t.xbar[it & 1], (uint32_t)(t.C - 1) * (uint32_t)((t.B + 1) * 4));
        if (warp < nwarps) {
            ps.begin(t.vs);
            for (int g = warp; g < nsmem; g += (TH / 32)) {
                float4 k[RB][NQ];
                ps.load_smem(t, g * BR, k);
                ps.batch(t, g * BR, k);
            }
            if (nsmem < nbatch) {
                // (the first batch past shared memory that is this warp's)
                for (int g = nsmem + (warp - nsmem % (TH / 32) + (TH / 32)) % (TH / 32); g < nbatch; g += (TH / 32)) {
                    float4 k[RB][NQ];
                    ps.load_global(t, g * BR, k);
                    ps.batch(t, g * BR, k);
                }
            }
            // this warp's column sums, over its row slots
            float4 cs[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                sr_unpack(ps.acc[q][0], cs[q].x, cs[q].y);
                sr_unpack(ps.acc[q][1], cs[q].z, cs[q].w);
            }
#pragma unroll
            for (int o = LR; o < 32; o <<= 1) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    cs[q].x += __shfl_xor_sync(0xffffffffu, cs[q].x, o);
                    cs[q].y += __shfl_xor_sync(0xffffffffu, cs[q].y, o);
                    cs[q].z += __shfl_xor_sync(0xffffffffu, cs[q].z, o);
                    cs[q].w += __shfl_xor_sync(0xffffffffu, cs[q].w, o);
                }
            }
            if (ps.slot == 0) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) *reinterpret_cast<float4 *>(t.part + warp * W + 4 * (q * LR + lane)) = cs[q];
            }
        }
        __syncthreads();

        // V: a thread completes a column (or two) over the warps and the CTAs
        int cont = 0;
        float lo = INFINITY, hi = -INFINITY;
        if (tid <= t.B) {
            float tot[kCols];
#pragma unroll
            for (int e = 0; e < kCols; ++e) {
                const float *part = t.part + min(tid + e * TH, W - 1);
                float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int w = 0; w < (TH / 32); ++w) c[w & 3] += part[w * W];
                tot[e] = (c[0] + c[1]) + (c[2] + c[3]);
            }
            if (t.C > 1) sr_exchange<TH, kCols, W>(t, it, tot, hdr);
#pragma unroll
            for (int e = 0; e < kCols; ++e) {
                const int j = tid + e * TH;
                if (j <= t.B) {
                    ov[e] = nv[e];
                    nv[e] = (j < t.B ? 1.f : Mf) * rcp_fast(tot[e]);
                    t.vs[j] = nv[e];
                    const float rel = (nv[e] - ov[e]) * rcp_fast(ov[e]);
                    lo = e == 0 ? rel : min_nan(lo, rel);
                    hi = e == 0 ? rel : max_nan(hi, rel);
                    cont |= p.tol > 0.f ? (fabsf(nv[e] - ov[e]) > p.tol * ov[e])
                                        : (!p.stop_fp || !dual_settled(__float_as_int(nv[e]), __float_as_int(ov[e]), before[e]));
                    before[e] = __float_as_int(ov[e]);
                }
            }
        }
        lo = warp_min_redux(lo);
        hi = warp_max_redux(hi);
        if (lane == 0) s_range[warp] = make_float2(lo, hi);
        ++st.done;
        const int go = __syncthreads_or(cont);
        const float2 range = s_range[lane % (TH / 32)];         // (written again after the next iteration's first barrier)
        lo = warp_min_redux(range.x);
        hi = warp_max_redux(range.y);
        st.last_move = fmaxf(-lo, hi);
        if (!go || (p.tol == 0.f && p.stop_fp && plan_settled(lo, hi))) break;
    }
    return st;
}

// This CTA has written everything it contributes to image `img`; the last of the C CTAs to say so
// appends the image to the list that the merge kernel consumes in order of completion (it may already
// be running: it was launched as a programmatic dependent).  Called by every thread of the CTA.
// by_image: the merge kernel has a CTA for every unit, which waits for its own image: the entry's place is the image's
// number, and nobody counts.
__device__ inline void sinkhorn_list(int img, int32_t *__restrict__ ready_list, WsHeader *__restrict__ hdr, bool by_image)
{
    const uint32_t slot = by_image ? (uint32_t)img : atomicAdd(&hdr->n_ready, 1u);
    ptx::st_release_gpu(ready_list + slot, img + 1);
}
__device__ inline void sinkhorn_publish(int img, uint32_t C, uint32_t *__restrict__ sink_done,
                                        int32_t *__restrict__ ready_list, WsHeader *__restrict__ hdr, bool by_image)
{
    if (!ready_list) return;
    ptx::fence_proxy_async_all();     // the plan rows are read by TMA over there
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t prev = C > 1u ? atomicAdd(&sink_done[img], 1u) : 0u;
        if (prev == C - 1u) {
            __threadfence();
            sinkhorn_list(img, ready_list, hdr, by_image);
        }
    }
}

// Where an image's results go.
struct SrOut {
    int img;
    const int32_t *ord;                        // kept tokens, then pruned tokens
    __nv_bfloat16 *Pimg;                       // plan rows of this CTA (bf16 storage), else nullptr
    int pbuf_pitch;
    int32_t *merged_seg, *partner_seg;
    float *weight_seg;
    uint32_t *sink_done;
    int32_t *ready_list;
    bool by_image;
};

// Plan P = U K V of this CTA's rows: alpha P in bf16 (row = position among the kept tokens, columns up to the next
// multiple of 64) or P in fp32 in place in the workspace tile.  In the same pass the pairing: partner_j = argmax_i P_ij
// = argmax_i K_ij U_i, ties to the lower i.  The merge kernel may take the image before the pairs are out.
template <int TH, int LR, int NQ, int RB>
__device__ inline void sr_finish(const SrTile &t, const OtParams &p, const SrOut &o, WsHeader *hdr)
{
    typedef SrPass<LR, NQ, RB> Pass;
    constexpr int W = Pass::W;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = lane % LR, slot = lane / LR;
    const int kpad = (t.B + 63) & ~63;
    Pass ps;
    ps.init(t);
    float4 V[NQ];
    float bv[NQ][4];
    int bi[NQ][4];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int col = 4 * (q * LR + sub);
        V[q] = *reinterpret_cast<const float4 *>(t.vs + col);
        V[q].x = col < t.B ? V[q].x : 0.f;             // (not the dustbin's)
        V[q].y = col + 1 < t.B ? V[q].y : 0.f;
        V[q].z = col + 2 < t.B ? V[q].z : 0.f;
        V[q].w = col + 3 < t.B ? V[q].w : 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            bv[q][e] = -INFINITY;
            bi[q][e] = 0x7fffffff;
        }
    }
    // (rows one by one: this code runs once per image, and fetching it costs more than its latencies)
    constexpr int RPW = 32 / LR;
    for (int i0 = warp * RPW; i0 < t.Ml; i0 += (TH / 32) * RPW) {
        const int i = i0 + slot;
        if (i >= t.Ml) continue;
        const float *krow = i < t.cap ? t.Ks + (size_t)i * t.ld : t.Kg + (size_t)i * t.ld;
        const float u = t.us[i];
        __nv_bfloat16 *prow = o.Pimg ? o.Pimg + (size_t)i * o.pbuf_pitch : nullptr;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int col = 4 * (q * LR + sub);
            const float4 k = *reinterpret_cast<const float4 *>(krow + ps.off[q]);
            const float ku[4] = {k.x * u, k.y * u, k.z * u, k.w * u};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (ku[e] > bv[q][e]) {                // rows ascend within a lane: strict > keeps the lower row
                    bv[q][e] = ku[e];
                    bi[q][e] = t.row_lo + i;
                }
            const float4 P = make_float4(ku[0] * V[q].x, ku[1] * V[q].y, ku[2] * V[q].z, ku[3] * V[q].w);
            if (prow) {
                if (col < kpad) {
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(p.alpha * P.x, p.alpha * P.y);
                    const __nv_bfloat162 hi = __floats2bfloat162_rn(p.alpha * P.z, p.alpha * P.w);
                    *reinterpret_cast<uint2 *>(prow + col) =
                        make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
                }
                if (W < 64) *reinterpret_cast<uint2 *>(prow + W + col) = make_uint2(0u, 0u);        // columns 32 .. 63
            } else if (col < t.ld) {
                *reinterpret_cast<float4 *>(t.Kg + (size_t)i * t.ld + col) = P;
            }
        }
    }
    sinkhorn_publish(o.img, (uint32_t)t.C, o.sink_done, o.ready_list, hdr, o.by_image);

    // pairs: over the row slots of a warp, the warps, the CTAs (ranks hold ascending rows)
#pragma unroll
    for (int s = LR; s < 32; s <<= 1) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv[q][e], s);
                const int oi = __shfl_xor_sync(0xffffffffu, bi[q][e], s);
                if (ov > bv[q][e] || (ov == bv[q][e] && oi < bi[q][e])) {
                    bv[q][e] = ov;
                    bi[q][e] = oi;
                }
            }
    }
    float *pv = t.part;
    int *pi = reinterpret_cast<int *>(t.part + (TH / 32) * W);
    if (slot == 0) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int col = 4 * (q * LR + sub);
            *reinterpret_cast<float4 *>(pv + warp * W + col) = make_float4(bv[q][0], bv[q][1], bv[q][2], bv[q][3]);
            *reinterpret_cast<int4 *>(pi + warp * W + col) = make_int4(bi[q][0], bi[q][1], bi[q][2], bi[q][3]);
        }
    }
    if (t.C > 1) ptx::cluster_sync_all();      // nobody reads xpart as column sums any more
    else __syncthreads();
    const uint32_t xp0 = ptx::smem_u32(t.xpart);
    for (int j = tid; j < t.B; j += TH) {
        float b = pv[j];
        int ib = pi[j];
#pragma unroll
        for (int w = 1; w < (TH / 32); ++w) {
            const float ob = pv[w * W + j];
            const int oi = pi[w * W + j];
            if (ob > b || (ob == b && oi < ib)) {
                b = ob;
                ib = oi;
            }
        }
        if (t.C > 1) {
            const uint32_t at = ptx::map_to_rank(xp0, 0);
            ptx::st_cluster_f32(at + (t.rank * W + (uint32_t)j) * 4u, b);
            ptx::st_cluster_u32(at + ((t.C + t.rank) * W + (uint32_t)j) * 4u, (uint32_t)ib);
        } else {
            o.merged_seg[j] = __ldcg(o.ord + t.M + j);
            o.partner_seg[j] = ib;
            o.weight_seg[j] = b * t.vs[j];         // (K U) V, the product the plan stores
        }
    }
    if (t.C > 1) {
        ptx::cluster_sync_all();                   // after this barrier nothing is written into another CTA any more
        if (t.rank == 0) {
            const int *xi = reinterpret_cast<const int *>(t.xpart + t.C * W);
            for (int j = tid; j < t.B; j += TH) {
                float b = t.xpart[j];
                int ib = xi[j];
                for (int r = 1; r < t.C; ++r) {
                    const float ob = t.xpart[r * W + j];
                    if (ob > b) {
                        b = ob;
                        ib = xi[r * W + j];
                    }
                }
                o.merged_seg[j] = __ldcg(o.ord + t.M + j);
                o.partner_seg[j] = ib;
                o.weight_seg[j] = b * t.vs[j];
            }
        }
    }
}

// grid = batch * C CTAs, clusters of C along x (C = 1: no cluster).  WIDE: tiles of up to 639 pruned tokens, else up to
// 255.  With scores_done (per-image counts of finished score tiles) a CTA starts when its image's are in; otherwise, and
// before rank 0 leaves, it waits for the grid ahead, so that this grid's end still implies that one's.
template <bool WIDE, int TH>
__global__ void __launch_bounds__(TH, kSrThreads / TH)
sinkhorn_rows_kernel(const int32_t *__restrict__ offsets, const int32_t *__restrict__ counts,
                     const int32_t *__restrict__ out_offsets, const int32_t *__restrict__ order,
                     float *__restrict__ kmat, int kmat_stride, int max_tokens, int total, OtParams p, int C,
                     int spread, int smem_floats, __nv_bfloat16 *__restrict__ pbuf, int pbuf_pitch,
                     int32_t *__restrict__ merged_idx, int32_t *__restrict__ merge_partner,
                     float *__restrict__ merge_weight, float *__restrict__ stats, uint32_t *__restrict__ sink_done,
                     int32_t *__restrict__ ready_list, WsHeader *__restrict__ hdr, const uint32_t *scores_done, int tile_ctas, int by_image)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ uint64_t s_xbar[2], s_cbar[kSrChunks];
    const int img = blockIdx.x / C, tid = threadIdx.x;
    const uint32_t rank = (uint32_t)(blockIdx.x - img * C);
    ptx::grid_dep_launch();
    if (tid == 0) {
        ptx::mbar_init(&s_xbar[0], 1);
        ptx::mbar_init(&s_xbar[1], 1);
        for (int c = 0; c < kSrChunks; ++c) ptx::mbar_init(&s_cbar[c], 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    if (!scores_done) ptx::grid_dep_wait();
    int t_begin, N;
    const bool valid = image_range(offsets, img, max_tokens, total, t_begin, N);
    if (valid && scores_done) {
        if (tid == 0) {
            const uint32_t want = (uint32_t)((N + 127) / 128 * tile_ctas);     // the scores kernel's CTAs, by 128-token tile
            // first the run's number: before it is there the counts are what the run before left
            const bool tagged = ptx::wait_equal_gpu(&hdr->run_tag, ptx::ld_acquire_gpu(&hdr->launch_seq));
            bool ok = false;
            for (uint32_t i = 0; tagged && i < ptx::kPollLimit && !ok; ++i) {
                ok = (uint32_t)ptx::ld_acquire_gpu(reinterpret_cast<const int *>(scores_done + img)) >= want;
                if (!ok) __nanosleep(40);
            }
            if (!ok) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
        }
        __syncthreads();
    }
    SrTile t;
    t.M = valid ? __ldcg(counts + img) : 0;
    const int out0 = valid ? __ldcg(out_offsets + img) : 0;
    t.B = valid ? N - t.M : 0;
    if (t.B == 0 || t.B > kSrMaxB) {           // nothing to solve, or another kernel's tile (then no list is kept)
        if (rank == 0) {
            sinkhorn_publish(img, 1u, sink_done, ready_list, hdr, by_image != 0);
            if (scores_done) ptx::grid_dep_wait();
        }
        return;
    }
    t.C = sr_ctas(t.M, t.B, C, smem_floats, spread, TH / 32);
    t.rank = rank;
    if ((int)rank >= t.C) return;
    const int rows_per = (t.M + t.C - 1) / t.C;
    t.row_lo = min(t.M, (int)rank * rows_per);
    t.Ml = min(t.M, t.row_lo + rows_per) - t.row_lo;       // (may be 0)
    t.Mr = t.Ml + ((int)rank == t.C - 1 ? 1 : 0);
    t.ld = score_pitch(t.B);
    const int br = sr_batch_rows(t.B);
    const int room = (smem_floats - sr_aux_floats(t.B, t.C, rows_per, TH / 32)) / t.ld;      // rows of K
    t.cap = min(room / br, (t.Mr + br - 1) / br) * br;
    t.Kg = kmat + kmat_offset(kmat_stride, t_begin, img) + (size_t)t.row_lo * t.ld;
    const int w = sr_width(t.B);
    t.part = sm;
    t.xpart = t.part + 2 * (TH / 32) * w;
    t.vs = t.xpart + (t.C > 1 ? 2 * t.C * w : 0);
    t.us = t.vs + w;
    t.Ks = t.us + ((rows_per + 33) & ~3);
    t.xbar = s_xbar;
    t.cbar = s_cbar;
    if (tid < kSrChunks) {
        ptx::fence_proxy_async_all();          // the scores were written with ordinary stores
        sr_fetch(t, tid);
    }
    for (int i = tid; i < t.Ml; i += TH) t.us[i] = 1.f;      // u = 0
    const float inv_eps = 1.f / p.eps;
    const float shift = fmaxf(1.f, p.z);
    const float kappa = expf((p.z - shift) * inv_eps);
    const float v_init = expf(shift * inv_eps);            // v = 0
    const int seg = t_begin - out0;
    const SrOut o{img, order + t_begin, pbuf ? pbuf + (size_t)(t_begin + t.row_lo) * pbuf_pitch : nullptr, pbuf_pitch,
                  merged_idx + seg, merge_partner + seg, merge_weight + seg, sink_done, ready_list, by_image != 0};
    auto solve = [&](auto lr, auto nq, auto rb) {
        constexpr int LR = decltype(lr)::value, NQ = decltype(nq)::value, RB = decltype(rb)::value;
        sr_build<TH>(t, shift, inv_eps, 1.f / kappa, hdr);
        // every CTA at work is running and has its barriers in place before anything is sent to it
        if (t.C > 1) ptx::cluster_sync_all();
        const SrState st = sr_iterate<TH, LR, NQ, RB>(t, p, kappa, v_init, hdr);
        if (tid == 0 && rank == 0) {
            stats[(size_t)img * kStats + 5] = (float)st.done;
            stats[(size_t)img * kStats + 6] = fmaxf(st.last_move, 0.f);      // (0 where every dual is NaN)
        }
        sr_finish<TH, LR, NQ, RB>(t, p, o, hdr);
    };
    using std::integral_constant;
    if (t.B < 32) solve(integral_constant<int, 8>(), integral_constant<int, 1>(), integral_constant<int, 8>());
    else if (t.B < 64) solve(integral_constant<int, 8>(), integral_constant<int, 2>(), integral_constant<int, 8>());
    else if (t.B < 128) solve(integral_constant<int, 16>(), integral_constant<int, 2>(), integral_constant<int, 8>());
    else if (t.B < 256) solve(integral_constant<int, 16>(), integral_constant<int, 4>(), integral_constant<int, 4>());
    else if constexpr (WIDE) {
        if (t.B < 384) solve(integral_constant<int, 32>(), integral_constant<int, 3>(), integral_constant<int, 4>());
        else if (t.B < 512) solve(integral_constant<int, 32>(), integral_constant<int, 4>(), integral_constant<int, 4>());
        else solve(integral_constant<int, 32>(), integral_constant<int, 5>(), integral_constant<int, 2>());
    }
    if (scores_done && rank == 0) ptx::grid_dep_wait();
}

}  // namespace rtp

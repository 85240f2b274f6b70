// Dustbin-augmented optimal transport by Sinkhorn iterations (Eq. 5, Appendix C) in scaling form for score tiles of 640
// to 2047 pruned tokens (images of thousands of tokens): megabytes that no cluster's shared memory holds.  One cluster of
// C CTAs (2 to 16) per image, the rows (kept tokens) split over the CTAs and, row by row, over the warps of a CTA.
// Notation, dustbin row and column and the iteration are those of sinkhorn_rows.cuh.
//
// K stays in the image's workspace tile and is read once per iteration: every warp streams its own rows through a ring of
// shared-memory stages with 1-D bulk copies (a row is 2.6 to 8 KB and contiguous), two to four rows ahead, on across the
// end of an iteration (the tile does not change).  Rows run forwards and backwards in turn, so that an iteration begins
// with what L2 still holds of the one before.  The first iteration finds the scores there, exponentiates a row in
// registers and writes it back: no pass of its own to build K.
// A lane owns NQ 16-byte column chunks of every row of its warp, so V and the column sums of the whole row stay in its
// registers; a row costs five shuffles, no barrier.  Column sums are reduce-scattered over the cluster: a CTA owns a
// slice of the columns, receives the other CTAs' parts by counted asynchronous stores, adds them in rank order, and
// sends V of its slice to everybody the same way.  Every warp of every CTA then compares V with the V in its registers:
// bit-identical values, the same decision to stop, no exchange for it and no cluster barrier in the loop.
//
// What bounds it: the read of K per iteration, from L2 while a batch's tiles fit there, else from DRAM, by the SMs that
// clusters of that size can have (96 for 16 images, 80 for 8), and the latency chain of a row (about 900 cycles, 8 or 16
// rows at a time).  16 images of 2137 tokens (899 pruned): 242 -> 120 us in this kernel, 8 of 4512 (1729 pruned): 577 ->
// 296 us, against the block-synchronous kernel of sinkhorn_tall.cuh, which still takes what is wider.
#pragma once
#include "common.cuh"
#include "ptx.cuh"
#include "sinkhorn.cuh"
#include "sinkhorn_rows.cuh"

namespace rtp {

constexpr int kStMaxWarps = 16;
// Threads: 16 warps hide a row's chain of latencies best; a warp of tiles wider than 1024 columns needs more registers
// than that leaves (V, the column sums and a row of K: 12 floats a lane per 128 columns).
__host__ __device__ inline int st_threads(int W) { return W <= 1024 ? 512 : 256; }
constexpr int kStMaxB = 2047;
constexpr int kStMaxC = 16;
constexpr int kStMaxStages = 4;                // rows in flight per warp
// The fixed-point test of this kernel: a dual here is the reciprocal of a sum of a thousand or more products, whose
// rounding noise is a few units in the last place (see kTallFixedPointTol, the same value).
constexpr float kStFixedPointTol = 4.76837158e-7f;

// Columns the lanes cover (multiples of 256: NQ even).
__host__ __device__ inline int st_width(int B) { return (B + 256) & ~255; }
__host__ __device__ inline int st_slice(int W, int C) { return (W + C - 1) / C; }
// Floats of shared memory besides the ring of rows: V, the warps' column sums (two of them share a row), the parts
// received (values, and indices for the pairing), U of every row.
__host__ __device__ inline int st_fixed_floats(int W, int C, int rows, int warps)
{
    return W + (warps / 2) * W + 2 * C * st_slice(W, C) + ((rows + 3) & ~3);
}
// The ring: at least two rows per warp; the pairing needs a value and an index per warp and column.
__host__ __device__ inline int st_min_floats(int W, int C, int rows, int warps) { return st_fixed_floats(W, C, rows, warps) + 2 * warps * W; }

struct StTile {
    int M, B, Ml, row_lo, ld;
    bool dust;                                 // this CTA has the dustbin's row
    int C;
    uint32_t rank;
    float *Kg;                                 // this CTA's first row in the workspace tile
    float *vs, *part, *xrecv, *us, *ring;
    uint64_t *full, *sbar, *vbar;              // [warps][stages] rows; column sums; V
    int stages;
};

// exp((s - c)/eps) of a chunk that lies before column B.
__device__ inline float4 st_k4(const float4 &s, float a, float b)
{
    return make_float4(sr_exp2(fmaf(s.x, a, b)), sr_exp2(fmaf(s.y, a, b)), sr_exp2(fmaf(s.z, a, b)), sr_exp2(fmaf(s.w, a, b)));
}

// 16 bytes of shared memory as two column pairs.
__device__ inline void st_load_pairs(uint32_t addr, sr_f32x2 (&v)[2])
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v[0]), "=l"(v[1]) : "r"(addr));
}

template <int NQ, int TH>
__device__ inline void st_solve(const StTile &t, const OtParams &p, const SrOut &o, float *__restrict__ stats_img, WsHeader *__restrict__ hdr)
{
    constexpr int W = NQ * 128, kWarps = TH / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sl = st_slice(W, t.C);           // columns per owner
    const float inv_eps = 1.f / p.eps, shift = fmaxf(1.f, p.z);
    const float kappa = expf((p.z - shift) * inv_eps), inv_kappa = 1.f / kappa;
    const float v_init = expf(shift * inv_eps);               // v = 0
    const float ea = inv_eps * 1.4426950408889634f, eb = -shift * ea;
    const float Bf = (float)t.B, Mf = (float)t.M;
    bool gave_up = false;

    // this warp's rows: warp, warp + 8, ...; the stream of them, iteration after iteration
    const int nrows = t.Ml > warp ? (t.Ml - warp + kWarps - 1) / kWarps : 0;
    const int NS = t.stages;
    const uint32_t row_bytes = (uint32_t)t.ld * 4u;
    const uint32_t ring = ptx::smem_u32(t.ring) + (uint32_t)(warp * t.stages) * row_bytes;
    uint64_t *full = t.full + warp * kStMaxStages;
    // Loads: thread 0 of the warp issues them, the first iteration's rows first (a row is read again only once it is K),
    // then, in turn backwards and forwards, all that the other iterations may need.
    const float *ld_src = t.Kg + (size_t)warp * t.ld;         // of the next load
    long long ld_step = (long long)kWarps * t.ld;
    int ld_left = p.iters > 0 ? nrows : 0, ld_turn = nrows;   // loads allowed now; rows until the next turn
    int ld_more = p.iters > 1 ? (int)min((long long)(p.iters - 1) * nrows, 0x3fffffffLL) : 0;      // allowed after the first iteration
    uint32_t ld_at = 0;                                       // stage
    int issued = 0;
    auto issue = [&]() {
        if (ld_left == 0) return;
        --ld_left;
        ++issued;
        ptx::mbar_arrive_expect_tx(&full[ld_at], row_bytes);
        ptx::bulk_load(ring + ld_at * row_bytes, ld_src, row_bytes, &full[ld_at]);
        if (++ld_at == (uint32_t)NS) ld_at = 0;
        if (--ld_turn == 0) {
            ld_turn = nrows;
            ld_step = -ld_step;
        } else {
            ld_src += ld_step;
        }
    };
    if (lane == 0)
        for (int s = 0; s < NS; ++s) issue();
    int taken = 0;
    int stage = 0;
    uint32_t phase = 0;

    // byte offset of this lane's chunk q in a row: only the last two can lie past the row's end; they read its last one
    const uint32_t tail0 = 16u * (uint32_t)min((NQ - 2) * 32 + lane, (t.ld >> 2) - 1);
    const uint32_t tail1 = 16u * (uint32_t)min((NQ - 1) * 32 + lane, (t.ld >> 2) - 1);
    auto off = [&](int q) { return q < NQ - 2 ? 16u * (uint32_t)lane + 512u * (uint32_t)q : (q == NQ - 2 ? tail0 : tail1); };
    sr_f32x2 V[NQ][2];                                        // column pairs, as K is loaded
    const uint32_t vs_u32 = ptx::smem_u32(t.vs) + 16u * (uint32_t)lane;
#pragma unroll
    for (int q = 0; q < NQ; ++q) st_load_pairs(vs_u32 + 512u * q, V[q]);
    // (every CTA of the cluster is running and has its barriers in place: the caller's cluster barrier)

    int done = 0;
    float last_move = 0.f;
    for (int it = 0; it < p.iters; ++it) {
        const uint32_t par = (uint32_t)it & 1u;
        if (tid == 0) {
            // what arrives here: the other CTAs' parts of my slice; V of the other slices
            const int mine = max(0, min(sl, W - (int)t.rank * sl));
            ptx::mbar_arrive_expect_tx(t.sbar, (uint32_t)((t.C - 1) * mine * 4));
            ptx::mbar_arrive_expect_tx(t.vbar, (uint32_t)((W - mine) * 4));
        }
        sr_f32x2 acc[NQ][2];
#pragma unroll
        for (int q = 0; q < NQ; ++q) acc[q][0] = acc[q][1] = 0ull;
        // one row: FIRST: the scores become K, here and in the workspace
        auto row_pass = [&](auto first, int i) {
            if (!gave_up && !ptx::mbar_wait(&full[stage], phase)) gave_up = true;
            const uint32_t src = ring + (uint32_t)stage * row_bytes;
            sr_f32x2 k[NQ][2];
#pragma unroll
            for (int q = 0; q < NQ; ++q) st_load_pairs(src + off(q), k[q]);
            ++taken;
            if (++stage == NS) {
                stage = 0;
                phase ^= 1u;
            }
            if constexpr (decltype(first)::value) {
                float *row = t.Kg + (size_t)i * t.ld;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int col = 4 * (q * 32 + lane);
                    float4 v;
                    sr_unpack(k[q][0], v.x, v.y);
                    sr_unpack(k[q][1], v.z, v.w);
                    v = q < NQ - 2 ? st_k4(v, ea, eb) : sr_k4(v, ea, eb, col, t.B);
                    if (q < NQ - 2 || col < t.ld) *reinterpret_cast<float4 *>(row + col) = v;
                    k[q][0] = sr_pack(v.x, v.y);
                    k[q][1] = sr_pack(v.z, v.w);
                }
                ptx::fence_proxy_async_all();                 // (read again by a bulk copy)
            }
            __syncwarp();                                     // every lane has its K, and has written it
            if (lane == 0) issue();
            sr_f32x2 d0 = 0ull, d1 = 0ull;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                d0 = sr_fma2(k[q][0], V[q][0], d0);
                d1 = sr_fma2(k[q][1], V[q][1], d1);
            }
            float a, b;
            sr_unpack(sr_add2(d0, d1), a, b);
            const float U = rcp_fast(warp_sum(a + b));
            if (lane == 0) t.us[i] = U;
            const sr_f32x2 uu = sr_pack(U, U);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                acc[q][0] = sr_fma2(k[q][0], uu, acc[q][0]);
                acc[q][1] = sr_fma2(k[q][1], uu, acc[q][1]);
            }
        };
        if (it == 0) {
#pragma unroll 1
            for (int r = 0; r < nrows; ++r) row_pass(std::true_type(), warp + kWarps * r);
        } else {
            const int step = (it & 1) ? -kWarps : kWarps;
            int i = (it & 1) ? warp + kWarps * (nrows - 1) : warp;
#pragma unroll 1
            for (int r = 0; r < nrows; ++r, i += step) row_pass(std::false_type(), i);
        }
        if (it == 0) {
            ld_left = ld_more;
            if (lane == 0)
                for (int s = 0; s < NS; ++s) issue();
        }
        if (t.dust && warp == kWarps - 1) {                 // the dustbin's row: ones, 1/kappa in its own column
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int col = 4 * (q * 32 + lane);
                float v[4];
                sr_unpack(V[q][0], v[0], v[1]);
                sr_unpack(V[q][1], v[2], v[3]);
#pragma unroll
                for (int e = 0; e < 4; ++e) s = fmaf(v[e], col + e == t.B ? inv_kappa : 1.f, s);       // (V is 0 past B)
            }
            const float U = Bf * rcp_fast(warp_sum(s));
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int col = 4 * (q * 32 + lane);
                const float e0 = col == t.B ? inv_kappa : 1.f, e1 = col + 1 == t.B ? inv_kappa : 1.f;
                const float e2 = col + 2 == t.B ? inv_kappa : 1.f, e3 = col + 3 == t.B ? inv_kappa : 1.f;
                acc[q][0] = sr_fma2(sr_pack(e0, e1), sr_pack(U, U), acc[q][0]);
                acc[q][1] = sr_fma2(sr_pack(e2, e3), sr_pack(U, U), acc[q][1]);
            }
        }
        // column sums over the warps: the upper four hand theirs to the lower four, then one thread per column
        if (warp >= kWarps / 2) {
            float *dst = t.part + (warp - kWarps / 2) * W + 4 * lane;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                float4 c;
                sr_unpack(acc[q][0], c.x, c.y);
                sr_unpack(acc[q][1], c.z, c.w);
                *reinterpret_cast<float4 *>(dst + 128 * q) = c;
            }
        }
        __syncthreads();
        if (warp < kWarps / 2) {
            float *dst = t.part + warp * W + 4 * lane;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const float4 h = *reinterpret_cast<const float4 *>(dst + 128 * q);
                float4 c;
                sr_unpack(acc[q][0], c.x, c.y);
                sr_unpack(acc[q][1], c.z, c.w);
                c.x += h.x;
                c.y += h.y;
                c.z += h.z;
                c.w += h.w;
                *reinterpret_cast<float4 *>(dst + 128 * q) = c;
            }
        }
        __syncthreads();
        {
            const uint32_t sb = ptx::smem_u32(t.sbar), xr = ptx::smem_u32(t.xrecv + t.rank * sl);
            for (uint32_t r = 0; r < (uint32_t)t.C; ++r) {
                const uint32_t to = ptx::map_to_rank(xr, r), tobar = ptx::map_to_rank(sb, r);
                for (int c = tid; c < sl; c += TH) {
                    const int j = (int)r * sl + c;
                    if (j >= W) break;
                    float tot[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int w = 0; w < kWarps / 2; ++w) tot[w & 3] += t.part[w * W + j];
                    const float sum = (tot[0] + tot[1]) + (tot[2] + tot[3]);
                    if (r == t.rank) t.xrecv[t.rank * sl + c] = sum;
                    else sr_send(to + 4u * (uint32_t)c, sum, tobar);
                }
            }
        }
        __syncthreads();                                      // my own parts of my slice
        // V of my slice, to everybody
        if (!gave_up && !ptx::mbar_wait(t.sbar, par)) gave_up = true;
        {
            const uint32_t vb = ptx::smem_u32(t.vbar);
            for (int c = tid; c < sl; c += TH) {
                const int j = (int)t.rank * sl + c;
                if (j >= W) break;
                float cs = 0.f;
                for (int r = 0; r < t.C; ++r) cs += t.xrecv[r * sl + c];
                const float nv = j < t.B ? rcp_fast(cs) : (j == t.B ? Mf * rcp_fast(cs) : 0.f);
                const uint32_t at = ptx::smem_u32(t.vs + j);
                for (uint32_t r = 0; r < (uint32_t)t.C; ++r) {
                    if (r == t.rank) t.vs[j] = nv;
                    else sr_send(ptx::map_to_rank(at, r), nv, ptx::map_to_rank(vb, r));
                }
            }
        }
        __syncthreads();                                      // my own slice
        if (!gave_up && !ptx::mbar_wait(t.vbar, par)) gave_up = true;
        // the new V against the old one: the same values, the same decision in every warp of every CTA
        float move = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            float nn[4], oo[4];
            sr_unpack(V[q][0], oo[0], oo[1]);
            sr_unpack(V[q][1], oo[2], oo[3]);
            st_load_pairs(vs_u32 + 512u * q, V[q]);
            sr_unpack(V[q][0], nn[0], nn[1]);
            sr_unpack(V[q][1], nn[2], nn[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float m = fabsf(nn[e] - oo[e]) * rcp_fast(fmaxf(oo[e], 1e-38f));       // (0 past column B)
                move = fmaxf(move, m);
            }
        }
        last_move = warp_max(move);
        ++done;
        const bool go = p.tol > 0.f ? last_move > p.tol : (p.stop_fp ? last_move > kStFixedPointTol : true);
        // a wait that ran out ends the loop of its own warp only at the next uniform point: below
        if (!go) break;
    }
    if (t.rank == 0 && tid == 0) {
        stats_img[5] = (float)done;
        stats_img[6] = last_move;
    }
    // loads issued for iterations that did not run: wait for them before the ring is used again
    for (; taken < __shfl_sync(0xffffffffu, issued, 0); ++taken) {
        if (!ptx::mbar_wait(&full[stage], phase)) gave_up = true;
        if (++stage == NS) {
            stage = 0;
            phase ^= 1u;
        }
    }
    if (gave_up) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
    __syncthreads();

    if (done == 0)                                            // (no iteration: the tile still holds the scores; u = 0)
        for (int r = 0; r < nrows; ++r) {
            const int i = warp + kWarps * r;
            if (lane == 0) t.us[i] = 1.f;
            for (int c = 4 * lane; c < t.ld; c += 128) {
                float4 *k = reinterpret_cast<float4 *>(t.Kg + (size_t)i * t.ld + c);
                *k = sr_k4(__ldcg(k), ea, eb, c, t.B);
            }
            __syncwarp();
        }

    // ---- plan P = U K V of this CTA's rows, and per column the best K_ij U_i over them, half of the columns at a time
    // (the values and indices of all of them would not fit the registers)
    const int kpad = (t.B + 63) & ~63;
    constexpr int NH = NQ / 2;
    float *pv = t.ring;
    int *pi = reinterpret_cast<int *>(t.ring + kWarps * W);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const bool back = (done + h) & 1;                     // (as the iterations do)
        float4 Vh[NH];
        int bv[NH][4], bi[NH][4];                             // (K U >= 0: compared as bits)
        const int col0 = 4 * (h * NH * 32 + lane);            // chunk q begins at column col0 + 128 q
#pragma unroll
        for (int q = 0; q < NH; ++q) {
            const int col = col0 + 128 * q;
            Vh[q] = *reinterpret_cast<const float4 *>(t.vs + col);
            const float f = o.Pimg ? p.alpha : 1.f;
            Vh[q].x = col < t.B ? f * Vh[q].x : 0.f;       // (not the dustbin's)
            Vh[q].y = col + 1 < t.B ? f * Vh[q].y : 0.f;
            Vh[q].z = col + 2 < t.B ? f * Vh[q].z : 0.f;
            Vh[q].w = col + 3 < t.B ? f * Vh[q].w : 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                bv[q][e] = -1;
                bi[q][e] = 0x7fffffff;
            }
        }
        // the next row's K is on its way while this one is used
        float4 kn[NH];
        auto fetch = [&](int i) {
            const float *row = t.Kg + (size_t)i * t.ld + col0;
#pragma unroll
            for (int q = 0; q < NH; ++q)
                kn[q] = q < NH - 2 || col0 + 128 * q < t.ld ? __ldcg(reinterpret_cast<const float4 *>(row + 128 * q)) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        const int step = back ? -kWarps : kWarps, tie = back ? 1 : 0;
        int i = back ? warp + kWarps * (nrows - 1) : warp;
        if (nrows > 0) fetch(i);
        for (int r = 0; r < nrows; ++r, i += step) {
            float4 k[NH];
#pragma unroll
            for (int q = 0; q < NH; ++q) k[q] = kn[q];
            if (r + 1 < nrows) fetch(i + step);
            const float u = t.us[i];
            __nv_bfloat16 *prow = o.Pimg ? o.Pimg + (size_t)i * o.pbuf_pitch + col0 : nullptr;
            float *krow = t.Kg + (size_t)i * t.ld + col0;
#pragma unroll
            for (int q = 0; q < NH; ++q) {
                const float ku[4] = {k[q].x * u, k[q].y * u, k[q].z * u, k[q].w * u};
#pragma unroll
                for (int e = 0; e < 4; ++e) {                 // ties to the lower row
                    const int key = __float_as_int(ku[e]);
                    const bool take = key + tie > bv[q][e];
                    bv[q][e] = take ? key : bv[q][e];
                    bi[q][e] = take ? t.row_lo + i : bi[q][e];
                }
                const float4 P = make_float4(ku[0] * Vh[q].x, ku[1] * Vh[q].y, ku[2] * Vh[q].z, ku[3] * Vh[q].w);
                if (prow) {                                   // (Vh holds alpha V then)
                    if (q < NH - 2 || col0 + 128 * q < kpad) {
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(P.x, P.y);
                        const __nv_bfloat162 hi = __floats2bfloat162_rn(P.z, P.w);
                        *reinterpret_cast<uint2 *>(prow + 128 * q) =
                            make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
                    }
                } else if (q < NH - 2 || col0 + 128 * q < t.ld) {
                    *reinterpret_cast<float4 *>(krow + 128 * q) = P;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NH; ++q) {
            *reinterpret_cast<int4 *>(pv + warp * W + col0 + 128 * q) = make_int4(bv[q][0], bv[q][1], bv[q][2], bv[q][3]);
            *reinterpret_cast<int4 *>(pi + warp * W + col0 + 128 * q) = make_int4(bi[q][0], bi[q][1], bi[q][2], bi[q][3]);
        }
    }
    __syncthreads();
    // over the warps, then to the owner of the column (every CTA is past its last exchange: nobody reads xrecv as sums
    // before this barrier and nobody sends into it after the next one)
    ptx::cluster_sync_all();
    {
        const uint32_t xr = ptx::smem_u32(t.xrecv), xi = xr + (uint32_t)(t.C * sl) * 4u;
        for (int j = tid; j < t.B; j += TH) {
            float b = pv[j];
            int ib = pi[j];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) {
                const float ob = pv[w * W + j];
                const int oi = pi[w * W + j];
                if (ob > b || (ob == b && oi < ib)) {
                    b = ob;
                    ib = oi;
                }
            }
            const uint32_t own = (uint32_t)(j / sl), at = (t.rank * (uint32_t)sl + (uint32_t)j - own * (uint32_t)sl) * 4u;
            ptx::st_cluster_f32(ptx::map_to_rank(xr + at, own), b);
            ptx::st_cluster_u32(ptx::map_to_rank(xi + at, own), (uint32_t)ib);
        }
    }
    ptx::cluster_sync_all();                                  // nothing is sent to another CTA after this
    const int *xi = reinterpret_cast<const int *>(t.xrecv + t.C * sl);
    for (int c = tid; c < sl; c += TH) {
        const int j = (int)t.rank * sl + c;
        if (j >= t.B) break;
        float b = t.xrecv[c];
        int ib = xi[c];
        for (int r = 1; r < t.C; ++r) {                       // ranks hold ascending rows: strict > keeps the lower one
            const float ob = t.xrecv[r * sl + c];
            if (ob > b) {
                b = ob;
                ib = xi[r * sl + c];
            }
        }
        o.merged_seg[j] = __ldcg(o.ord + t.M + j);
        o.partner_seg[j] = ib;
        o.weight_seg[j] = b * t.vs[j];                        // (K U) V, the product the plan stores
    }
}

// grid = batch * C CTAs, clusters of C along x.  Takes the images the kernel ahead of it left (those with B > rows_max_b);
// no image of the run has more than kStMaxB pruned tokens.  Every early return depends on the image only.
template <int TH>
__global__ void __launch_bounds__(TH, 1)
sinkhorn_stream_kernel(const int32_t *__restrict__ offsets, const int32_t *__restrict__ counts,
                       const int32_t *__restrict__ out_offsets, const int32_t *__restrict__ order,
                       float *__restrict__ kmat, int kmat_stride, int max_tokens, int total, OtParams p, int smem_floats,
                       __nv_bfloat16 *__restrict__ pbuf, int pbuf_pitch, int32_t *__restrict__ merged_idx,
                       int32_t *__restrict__ merge_partner, float *__restrict__ merge_weight, float *__restrict__ stats,
                       int rows_max_b, WsHeader *__restrict__ hdr)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int kWarps = TH / 32;
    __shared__ uint64_t s_full[kWarps * kStMaxStages], s_bar[2];
    StTile t;
    t.rank = ptx::cluster_ctarank();
    t.C = (int)ptx::cluster_nctarank();
    const int img = blockIdx.x / t.C, tid = threadIdx.x;
    ptx::grid_dep_launch();
    if (tid < kWarps * kStMaxStages) ptx::mbar_init(&s_full[tid], 1);
    if (tid < 2) ptx::mbar_init(&s_bar[tid], 1);
    ptx::fence_mbar_init();
    ptx::grid_dep_wait();         // scores, counts and order come from the kernels ahead
    int t_begin, N;
    if (!image_range(offsets, img, max_tokens, total, t_begin, N)) return;
    t.M = __ldcg(counts + img);
    t.B = N - t.M;
    if (t.B <= rows_max_b || t.B > kStMaxB) return;
    const int rows_per = (t.M + t.C - 1) / t.C;
    t.row_lo = min(t.M, (int)t.rank * rows_per);
    t.Ml = min(t.M, t.row_lo + rows_per) - t.row_lo;          // this CTA's rows (may be 0)
    t.dust = (int)t.rank == t.C - 1;
    t.ld = score_pitch(t.B);
    t.Kg = kmat + kmat_offset(kmat_stride, t_begin, img) + (size_t)t.row_lo * t.ld;
    const int W = st_width(t.B);
    t.vs = sm;
    t.part = t.vs + W;
    t.xrecv = t.part + (kWarps / 2) * W;
    t.us = t.xrecv + 2 * t.C * st_slice(W, t.C);
    const int fixed = (st_fixed_floats(W, t.C, rows_per, kWarps) + 3) & ~3;
    t.ring = sm + fixed;
    t.stages = min(kStMaxStages, (smem_floats - fixed) / (kWarps * t.ld));
    t.full = s_full;
    t.sbar = &s_bar[0];
    t.vbar = &s_bar[1];
    const float v_init = expf(fmaxf(1.f, p.z) / p.eps), kappa = expf((p.z - fmaxf(1.f, p.z)) / p.eps);
    for (int j = tid; j < W; j += TH) t.vs[j] = j < t.B ? v_init : (j == t.B ? kappa * v_init : 0.f);
    ptx::fence_proxy_async_all();          // the scores were written with ordinary stores
    __syncthreads();
    // every CTA of the cluster is running and has its barriers and V in place before anything is sent to it
    ptx::cluster_sync_all();
    const int seg = t_begin - __ldcg(out_offsets + img);
    const SrOut o{img, order + t_begin, pbuf ? pbuf + (size_t)(t_begin + t.row_lo) * pbuf_pitch : nullptr, pbuf_pitch,
                  merged_idx + seg, merge_partner + seg, merge_weight + seg, nullptr, nullptr, false};
    float *st = stats + (size_t)img * kStats;
    switch (W >> 8) {
    case 3: st_solve<6, TH>(t, p, o, st, hdr); break;
    case 4: st_solve<8, TH>(t, p, o, st, hdr); break;
    default:
        if constexpr (TH == 256) {
            switch (W >> 8) {
            case 5: st_solve<10, TH>(t, p, o, st, hdr); break;
            case 6: st_solve<12, TH>(t, p, o, st, hdr); break;
            case 7: st_solve<14, TH>(t, p, o, st, hdr); break;
            default: st_solve<16, TH>(t, p, o, st, hdr); break;
            }
        }
    }
}

}  // namespace rtp

// The two contractions of stage 2 in fp32 storage -- the cosine scores (Section 3.3.2) and the merge
// T_k + alpha P T_p (Eq. 7) -- on the tcgen05 tensor cores.  An fp32 value is the exact sum of three bf16
// values (hi + mid + lo, 8 bits each, the last to within 2^-27 of it), so a product of two is, to 2^-26, the sum
// of the six bf16 products hi.hi, hi.mid, mid.hi, mid.mid, hi.lo, lo.hi, each exact in fp32.  hi.hi goes to one
// fp32 accumulator in tensor memory and the five small ones to another.  The tensor core's additions are not rounded to
// nearest: every one of them may cost a unit in the last place of the running sum, always towards zero (80 additions
// of hi.hi into one accumulator left the scores 2.5e-6 low).  The scores, whose contraction is long, therefore deal
// their k-blocks out to as many accumulators as tensor memory holds; all are added in the epilogue, rounded to nearest.
//
// Both kernels: eight producer warps load fp32 rows with 16-byte loads (rows are gathered by token index:
// no compact copy), split them in registers and store the three bf16 planes in the 128-byte-swizzled layouts the
// UMMA descriptors address; one thread issues the UMMAs; the epilogue reads TMEM.
//
// What bounds them, on 256 images of 400 tokens x 1280: the scores (868 us as fp32 FMA tiles, 246 us now; 0.42 GB of
// kept rows would take 64 us) wait for the operand reads of their UMMAs from shared memory, six per 128 x 16 tile of
// A; the merge (856 us, 383 us now; 0.84 GB in and out would take 128 us) for the splitting, which takes 8 warp
// instructions per 32 elements, and for its slowest tasks.  Largest error of the plan weights against fp64: 1.8e-6
// before, 7.8e-7 now.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace rtp {

constexpr int kF3Tile = 128;                   // rows and columns of an output tile
constexpr int kF3BK = 64;                      // contraction elements per k-block (one 128-byte row of bf16)
constexpr int kF3Plane = kF3Tile * 128;        // bytes of one plane of a 128-row operand tile
constexpr int kF3Stage = 6 * kF3Plane;         // three planes of A, three of B: 96 KB
constexpr int kF3Stages = 2;
constexpr int kF3Prod = 256;                   // producer threads

// Eight fp32 values as three vectors of eight bf16.
__device__ inline void split8(const float (&x)[8], uint4 &hi, uint4 &mid, uint4 &lo)
{
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float a = x[2 * e], b = x[2 * e + 1];
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
        h[e] = *reinterpret_cast<const uint32_t *>(&h2);
        const float ra = a - __uint_as_float(h[e] << 16), rb = b - __uint_as_float(h[e] & 0xffff0000u);
        const __nv_bfloat162 m2 = __floats2bfloat162_rn(ra, rb);
        m[e] = *reinterpret_cast<const uint32_t *>(&m2);
        const __nv_bfloat162 l2 = __floats2bfloat162_rn(ra - __uint_as_float(m[e] << 16), rb - __uint_as_float(m[e] & 0xffff0000u));
        l[e] = *reinterpret_cast<const uint32_t *>(&l2);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    mid = make_uint4(m[0], m[1], m[2], m[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// 8 consecutive floats at p (16-byte aligned).  TAIL: only the first `have` exist (a multiple of 4; the rest is zero).
template <bool TAIL> __device__ inline void load8(const float *p, int have, float (&x)[8])
{
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 a = (!TAIL || have > 0) ? __ldg(reinterpret_cast<const float4 *>(p)) : zero;
    const float4 b = (!TAIL || have > 4) ? __ldg(reinterpret_cast<const float4 *>(p) + 1) : zero;
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}

// The three planes of a chunk to their places: row `row` of a tile whose rows are 128 bytes, 16-byte piece `c`.
__device__ inline void store_planes(uint32_t tile, uint32_t plane_bytes, int row, int c, const float (&x)[8])
{
    uint4 h, m, l;
    split8(x, h, m, l);
    const uint32_t at = tile + (uint32_t)(row * 128 + ((c ^ (row & 7)) << 4));
    ptx::st_shared_v4(at, h);
    ptx::st_shared_v4(at + plane_bytes, m);
    ptx::st_shared_v4(at + 2 * plane_bytes, l);
}

// Scores: the six products of one k-block, both operands K-major, planes kF3Plane apart.
__device__ inline void f3_scores_block(uint32_t a_base, uint32_t b_base, uint32_t d_main, uint32_t d_small, uint32_t idesc,
                                       bool first_main, bool first_small)
{
    constexpr uint32_t pa[6] = {0, 0, 1, 1, 0, 2}, pb[6] = {0, 1, 0, 1, 2, 0};
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
        for (int k = 0; k < kF3BK / 16; ++k) {
            const uint64_t da = ptx::smem_desc_sw128(a_base + pa[q] * kF3Plane + k * 32, 16, 1024);
            const uint64_t db = ptx::smem_desc_sw128(b_base + pb[q] * kF3Plane + k * 32, 16, 1024);
            ptx::umma_bf16(q == 0 ? d_main : d_small, da, db, idesc, !(k == 0 && (q == 0 ? first_main : q == 1 && first_small)));
        }
}

struct F3Barriers {
    uint64_t full[kF3Stages], empty[kF3Stages], accum_full[2], accum_empty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
};
constexpr int kF3SmemBytes = kF3Stages * kF3Stage + 1024 /*alignment*/ + 256 /*barriers*/;

// ---------------------------------------------------------------------------------------------
// S_ij = x_i . x_j / (|x_i| |x_j|), i in T_kept, j in T_prop.  grid = (mtiles * btiles_max, batch), one 128 x 128
// tile per CTA.  Output: kmat[i * score_pitch(B) + j].  288 threads: the producers (which also run the epilogue), then
// the UMMA warp.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kF3Prod + 32, 1)
scores_fp32_umma_kernel(const float *__restrict__ X, const int32_t *__restrict__ offsets, int d, int btiles_max,
                        const int32_t *__restrict__ counts, const int32_t *__restrict__ order,
                        const float *__restrict__ norms, float *__restrict__ kmat, int kmat_stride, int max_tokens,
                        int total, WsHeader *__restrict__ hdr)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ float s_norm[2 * kF3Tile];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    F3Barriers *bars = reinterpret_cast<F3Barriers *>(smem + kF3Stages * kF3Stage);
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int img = blockIdx.y;
    int t_begin, N;
    const int M = __ldcg(counts + img);
    if (!image_range(offsets, img, max_tokens, total, t_begin, N)) return;
    const int B = N - M;
    const int i0 = (int)(blockIdx.x / btiles_max) * kF3Tile, j0 = (int)(blockIdx.x % btiles_max) * kF3Tile;
    if (B == 0 || i0 >= M || j0 >= B) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nkb = (d + kF3BK - 1) / kF3BK;
    const int BN = min(kF3Tile, (B - j0 + 15) & ~15);
    if (tid == 0) {
        for (int s = 0; s < kF3Stages; ++s) {
            ptx::mbar_init(&bars->full[s], kF3Prod / 32);
            ptx::mbar_init(&bars->empty[s], 1);
        }
        ptx::mbar_init(&bars->accum_full[0], 1);
        bars->abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == kF3Prod / 32) {
        ptx::tmem_alloc(&bars->tmem_base, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    // accumulators: the small products, then as many of hi.hi as fit beside them
    const int acc_cols = (BN + 31) & ~31, nmain = min(512 / acc_cols - 1, nkb);

    if (warp < kF3Prod / 32) {
        // thread = (16-byte piece c of a 128-byte row, rows r0 + 32 q of either operand).  Rows past the image's
        // last kept (pruned) one repeat it: what they give is not stored.
        const int c = tid & 7, r0 = tid >> 3;
        const int32_t *ord = order + t_begin;
        const float *src[8];                       // four rows of A, four of B
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int ta = t_begin + __ldg(ord + min(i0 + r0 + 32 * q, M - 1));
            const int tb = t_begin + __ldg(ord + M + min(j0 + r0 + 32 * q, B - 1));
            src[q] = X + (size_t)ta * d + 8 * c;
            src[4 + q] = X + (size_t)tb * d + 8 * c;
            if (c == 0) {
                s_norm[r0 + 32 * q] = fmaxf(__ldcg(norms + ta), kNormFloor);
                s_norm[kF3Tile + r0 + 32 * q] = fmaxf(__ldcg(norms + tb), kNormFloor);
            }
        }
        const uint32_t ring = ptx::smem_u32(smem);
        const int whole = d / kF3BK;               // k-blocks of 64 columns
        auto fetch = [&](int kb, float (&x)[8][8]) {
            if (kb < whole) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < 4 || r0 + 32 * (q - 4) < BN) load8<false>(src[q] + kb * kF3BK, 8, x[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 8; ++q) load8<true>(src[q] + kb * kF3BK, kb < nkb ? d - kb * kF3BK - 8 * c : 0, x[q]);
            }
        };
        bool ok = true;
        auto store = [&](int kb, const float (&x)[8][8]) {
            const int s = kb % kF3Stages;
            if (ok && kb >= kF3Stages) ok = ptx::mbar_wait(&bars->empty[s], ((kb / kF3Stages) - 1) & 1);
            if (!__all_sync(0xffffffffu, ok)) return;
            const uint32_t st = ring + s * kF3Stage;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < 4 || r0 + 32 * (q - 4) < BN)
                    store_planes(st + (q < 4 ? 0 : 3 * kF3Plane), kF3Plane, r0 + 32 * (q & 3), c, x[q]);
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->full[s]);
        };
        // two k-blocks in registers on their way, two in shared memory
        float x0[8][8], x1[8][8];
        fetch(0, x0);
        fetch(1, x1);
        for (int kb = 0; kb < nkb; kb += 2) {
            store(kb, x0);
            fetch(kb + 2, x0);
            if (kb + 1 < nkb) store(kb + 1, x1);
            fetch(kb + 3, x1);
        }
        if (!__all_sync(0xffffffffu, ok)) {
            bars->abort_flag = 1;
            if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
        }
    } else if (lane == 0) {
        const uint32_t idesc = ptx::idesc_bf16(kF3Tile, BN, false, false);
        const uint32_t base = ptx::smem_u32(smem);
        for (int kb = 0; kb < nkb; ++kb) {
            const int s = kb % kF3Stages;
            if (bars->abort_flag || !ptx::mbar_wait(&bars->full[s], (kb / kF3Stages) & 1)) {
                bars->abort_flag = 1;
                atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                break;
            }
            ptx::tc_fence_after();
            f3_scores_block(base + s * kF3Stage, base + s * kF3Stage + 3 * kF3Plane,
                            tmem_base + (uint32_t)((1 + kb % nmain) * acc_cols), tmem_base, idesc, kb < nmain, kb == 0);
            ptx::umma_commit(&bars->empty[s]);
        }
        ptx::umma_commit(&bars->accum_full[0]);
    }
    __syncthreads();                                // s_norm; every producer is past the ring
    if (warp < 8) {
        // warp = (quarter of the rows, half of the columns)
        const bool ok = ptx::mbar_wait(&bars->accum_full[0], 0) && !bars->abort_flag;
        if (__all_sync(0xffffffffu, ok)) {
            ptx::tc_fence_after();
            const int row = (warp & 3) * 32 + lane;
            const uint32_t t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
            float *out = kmat + kmat_offset(kmat_stride, t_begin, img) + (size_t)(i0 + row) * score_pitch(B) + j0;
            const float ni = s_norm[row];
            for (int c0 = (warp >> 2) * 32; c0 < BN; c0 += 64) {
                float sum[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) sum[e] = 0.f;
                for (int k = nmain; k >= 0; --k) {             // the small products last
                    uint32_t a[32];
                    ptx::tmem_ld32(t + (uint32_t)(k * acc_cols + c0), a);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) sum[e] += __uint_as_float(a[e]);
                }
                if (i0 + row < M) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        float o[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) o[e] = sum[4 * g + e] / (ni * s_norm[kF3Tile + c0 + 4 * g + e]);
                        // (the row pitch is a multiple of 4 past B: what is written beside column B is never read)
                        if (j0 + c0 + 4 * g < B) *reinterpret_cast<float4 *>(out + c0 + 4 * g) = make_float4(o[0], o[1], o[2], o[3]);
                    }
                }
            }
        } else if (lane == 0) {
            atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kF3Prod / 32) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, 512);
    }
}


// ---------------------------------------------------------------------------------------------
// y_i = x_i + alpha * sum_j P_ij x_j (Eq. 7), written packed, with kept_idx.  A task is (image, 128 kept rows, a run of
// 64-column output tiles); the kernel is persistent, its CTAs draw tasks from a
// counter (images prune 0 to N / 2 tokens: tasks dealt out in turn left the busiest SM with 2.3 times the mean).  A operand: rows of P from
// the score tile, K-major, split once per task when at most 128 tokens are pruned (else again for every output tile);
// B operand: the pruned tokens' rows, rows = contraction index.  Roles (448 threads): warps 0-7 load and split; warp 8
// issues the UMMAs (two accumulator sets); warp 9 resolves tasks ahead of the others (a chain of loads from L2) and
// hands them over in shared memory; warps 10-13 run the epilogue: the kept rows' own tile comes in by cp.async one
// output tile ahead, the sum is formed where it lies (thread = row, as TMEM is read) and leaves in coalesced rows.
// ---------------------------------------------------------------------------------------------
constexpr int kM3N = 64;                                     // output columns of a tile
constexpr int kM3Epi = 4;                                    // epilogue warps
constexpr int kM3Threads = kF3Prod + 64 + 32 * kM3Epi;
constexpr int kM3Tasks = 4;                                  // depth of the scheduler's ring
constexpr int kM3Acc = 2;                                    // accumulator sets
constexpr int kM3AccCols = 3 * kM3N;                         // of three times 64 columns, see merge_fp32_block
constexpr int kM3ASlots = 2;                                 // k-blocks of P in shared memory
constexpr int kM3ABytes = 3 * kF3Plane;                      // 48 KB each
constexpr int kM3BPlane = kF3BK * 128;                       // 64 rows x 64 columns
constexpr int kM3BBytes = 3 * kM3BPlane;                     // 24 KB per stage
constexpr int kM3Pitch = kM3N * 4 + 16;                      // bytes per row of an x / y tile: conflict-free by rows
constexpr int kM3XBytes = kF3Tile * kM3Pitch;

// Merge: the six products of one k-block.  The planes of B lie side by side, so that one UMMA multiplies a plane of A
// with several of them (a 128 x 16 tile of A is read from shared memory three times, not six: at 64 columns per UMMA
// the reads, not the multiplications, would bound it): hi x [hi | mid | lo], mid x [hi | mid], lo x [hi], into the
// column sets [s0 | s1 | s2], [s1 | s2], [s1]; s0 holds the large products.
__device__ inline void merge_fp32_block(uint32_t a_base, uint32_t b_base, uint32_t d_tmem, bool first)
{
    const uint32_t idesc[3] = {ptx::idesc_bf16(kF3Tile, 3 * kM3N, false, true), ptx::idesc_bf16(kF3Tile, 2 * kM3N, false, true),
                               ptx::idesc_bf16(kF3Tile, kM3N, false, true)};
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int k = 0; k < kF3BK / 16; ++k) {
            const uint64_t da = ptx::smem_desc_sw128(a_base + q * kF3Plane + k * 32, 16, 1024);
            const uint64_t db = ptx::smem_desc_sw128(b_base + k * 2048, kM3BPlane, 1024);
            ptx::umma_bf16(d_tmem + (q ? kM3N : 0), da, db, idesc[q], !(first && q == 0 && k == 0));
        }
}

struct M3Task {
    int end, B, M, i0, rows, ct0, ct1, ld;
    const float *P, *Xi;           // the image's plan, the image's first row of X
    const int32_t *kept, *prop;    // its kept and pruned tokens
    float *Yt;                     // the task's first row of Y
    int32_t *kidx;
};
struct M3Shared {
    F3Barriers b;
    uint64_t acc_full[kM3Acc], acc_empty[kM3Acc], task_full[kM3Tasks], task_empty[kM3Tasks];
    M3Task task[kM3Tasks];
};
constexpr int kM3SmemBytes = kM3ASlots * kM3ABytes + kF3Stages * kM3BBytes + 2 * kM3XBytes + 1024 + (int)((sizeof(M3Shared) + 127) & ~127u);
static_assert(kM3SmemBytes <= 227 * 1024, "more shared memory than a CTA can have");

__global__ void __launch_bounds__(kM3Threads, 1)
merge_fp32_umma_kernel(const float *__restrict__ X, const int32_t *__restrict__ offsets, int d, int batch, int mtiles,
                       int ct_run, const int32_t *__restrict__ counts, const int32_t *__restrict__ out_offsets,
                       const int32_t *__restrict__ order, const float *__restrict__ kmat, int kmat_stride, int max_tokens,
                       int total, float alpha, float *__restrict__ Y, int32_t *__restrict__ kept_idx,
                       WsHeader *__restrict__ hdr)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *xtiles = smem + kM3ASlots * kM3ABytes + kF3Stages * kM3BBytes;
    M3Shared *sh = reinterpret_cast<M3Shared *>(xtiles + 2 * kM3XBytes);
    const uint32_t a_u32 = ptx::smem_u32(smem), b_u32 = a_u32 + kM3ASlots * kM3ABytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kProdWarps = kF3Prod / 32;
    const int nct = (d + kM3N - 1) / kM3N, nruns = (nct + ct_run - 1) / ct_run;
    const int ntasks = batch * mtiles * nruns;
    if (tid == 0) {
        for (int s = 0; s < kF3Stages; ++s) {
            ptx::mbar_init(&sh->b.full[s], kProdWarps);
            ptx::mbar_init(&sh->b.empty[s], 1);
        }
        for (int s = 0; s < kM3Acc; ++s) {
            ptx::mbar_init(&sh->acc_full[s], 1);
            ptx::mbar_init(&sh->acc_empty[s], kM3Epi);
        }
        for (int s = 0; s < kM3Tasks; ++s) {
            ptx::mbar_init(&sh->task_full[s], 1);
            ptx::mbar_init(&sh->task_empty[s], kProdWarps + 1 + kM3Epi);
        }
        sh->b.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (warp == kProdWarps) {
        ptx::tmem_alloc(&sh->b.tmem_base, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = sh->b.tmem_base;
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    auto give_up = [&]() {
        sh->b.abort_flag = 1;
        if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
    };
    // bounded wait for a use of a ring slot
    auto wait = [&](uint64_t *bar, uint32_t phase) { return !sh->b.abort_flag && ptx::mbar_wait(bar, phase & 1u); };
    auto task_wait = [&](uint32_t t) { return wait(&sh->task_full[t % kM3Tasks], t / kM3Tasks); };

    if (warp < kProdWarps) {
        const int c = tid & 7, r0 = tid >> 3;      // 16-byte piece c of rows r0 + 32 h (two of X, four of P)
        // the block fetched next: task, column tile, k-block, the tokens of this thread's two rows of it (loaded one
        // block ahead: the rows' addresses hang on them)
        uint32_t t_next = 0;
        int ct = 0, kb = 0, tok[2] = {0, 0};
        bool ok = true, more = true;
        auto load_tokens = [&](const M3Task &q) {
#pragma unroll
            for (int h = 0; h < 2; ++h) tok[h] = __ldg(q.prop + min(kb * kF3BK + r0 + 32 * h, q.B - 1));
        };
        auto settle = [&]() {                       // onto a task with blocks, or to the end
            for (;;) {
                ok = ok && task_wait(t_next);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = more = false;
                    return;
                }
                const M3Task &q = sh->task[t_next % kM3Tasks];
                if (q.end) {
                    more = false;
                    return;
                }
                if (q.B > 0) {
                    ct = q.ct0;
                    return;
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&sh->task_empty[t_next % kM3Tasks]);
                ++t_next;
            }
        };
        settle();
        if (more) load_tokens(sh->task[t_next % kM3Tasks]);
        struct Meta { uint32_t t; int kb; bool first_ct, last; };     // of a fetched block; kb = -1: none
        auto fetch = [&](float (&x)[2][8], Meta &m) {
            m.kb = -1;
            if (!more) return;
            const M3Task &q = sh->task[t_next % kM3Tasks];
            const int col = ct * kM3N + 8 * c;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float *p = q.Xi + (size_t)tok[h] * d + col;
                if (ct * kM3N + kM3N <= d) load8<false>(p, 8, x[h]);
                else load8<true>(p, d - col, x[h]);
            }
            m.t = t_next;
            m.kb = kb;
            m.first_ct = ct == q.ct0;
            m.last = false;
            if (++kb * kF3BK >= q.B) {
                kb = 0;
                if (++ct == q.ct1) {
                    m.last = true;
                    ++t_next;
                    settle();
                }
            }
            if (more) load_tokens(sh->task[t_next % kM3Tasks]);
        };
        // this thread's pieces of the block's rows of P, when the block needs them
        auto is_streamed = [&](const M3Task &q) { return q.B > kM3ASlots * kF3BK; };
        auto fetch_p = [&](float (&pv)[4][8], const Meta &m) {
            if (m.kb < 0) return;
            const M3Task &q = sh->task[m.t % kM3Tasks];
            if (!m.first_ct && !is_streamed(q)) return;
            const float *P = q.P + (size_t)q.i0 * q.ld + m.kb * kF3BK + 8 * c;
#pragma unroll
            for (int h = 0; h < 4; ++h) load8<true>(P + (size_t)min(r0 + 32 * h, q.rows - 1) * q.ld, q.B - m.kb * kF3BK - 8 * c, pv[h]);
        };
        uint32_t n = 0;                            // blocks stored
        auto store = [&](const float (&x)[2][8], float (&pv)[4][8], const Meta &m) {
            if (m.kb < 0 || !ok) return;
            const M3Task &q = sh->task[m.t % kM3Tasks];
            const bool streamed = is_streamed(q), need_p = streamed || m.first_ct;
            const uint32_t s = n % kF3Stages;
            if (n >= (uint32_t)kF3Stages) ok = wait(&sh->b.empty[s], n / kF3Stages - 1);
            // the first block of a task may overwrite a slot of P that the block before it still reads
            if (ok && need_p && m.first_ct && m.kb == 0 && n >= 1) ok = wait(&sh->b.empty[(n - 1) % kF3Stages], (n - 1) / kF3Stages);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                return;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) store_planes(b_u32 + s * kM3BBytes, kM3BPlane, r0 + 32 * h, c, x[h]);
            if (need_p) {
                const uint32_t slot = streamed ? s : (uint32_t)m.kb;
                const int left = q.B - m.kb * kF3BK - 8 * c;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (left < 8) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) pv[h][e] = e < left ? pv[h][e] : 0.f;         // columns past B hold anything
                    }
                    store_planes(a_u32 + slot * kM3ABytes, kF3Plane, r0 + 32 * h, c, pv[h]);
                }
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(&sh->b.full[s]);
                if (m.last) ptx::mbar_arrive(&sh->task_empty[m.t % kM3Tasks]);
            }
            ++n;
        };
        float x0[2][8], x1[2][8], pv[4][8];        // two blocks in registers on their way
        Meta m0, m1;
        fetch(x0, m0);
        fetch_p(pv, m0);
        fetch(x1, m1);
        while (ok && m0.kb >= 0) {
            store(x0, pv, m0);
            fetch_p(pv, m1);
            fetch(x0, m0);
            store(x1, pv, m1);
            fetch_p(pv, m0);
            fetch(x1, m1);
        }
        if (!__all_sync(0xffffffffu, ok)) give_up();
    } else if (warp == kProdWarps) {
        if (lane == 0) {
            uint32_t n = 0, acc = 0;
            bool ok = true;
            for (uint32_t t = 0; ok; ++t) {
                ok = task_wait(t);
                if (!ok) break;
                const M3Task &q = sh->task[t % kM3Tasks];
                if (q.end) break;
                const int nkb = (q.B + kF3BK - 1) / kF3BK;
                const bool streamed = nkb > kM3ASlots;
                for (int ct = q.ct0; ct < q.ct1 && nkb > 0 && ok; ++ct, ++acc) {
                    const uint32_t buf = acc % kM3Acc, dm = tmem_base + buf * kM3AccCols;
                    if (acc >= (uint32_t)kM3Acc) ok = wait(&sh->acc_empty[buf], acc / kM3Acc - 1);
                    for (int kb = 0; kb < nkb && ok; ++kb, ++n) {
                        const uint32_t s = n % kF3Stages;
                        ok = wait(&sh->b.full[s], n / kF3Stages);
                        if (!ok) break;
                        ptx::tc_fence_after();
                        merge_fp32_block(a_u32 + (streamed ? s : (uint32_t)kb) * kM3ABytes, b_u32 + s * kM3BBytes, dm, kb == 0);
                        ptx::umma_commit(&sh->b.empty[s]);
                    }
                    if (ok) ptx::umma_commit(&sh->acc_full[buf]);
                }
                ptx::mbar_arrive(&sh->task_empty[t % kM3Tasks]);
            }
            if (!ok) give_up();
        }
    } else if (warp == kProdWarps + 1) {
        uint32_t nt = 0;
        bool ok = true;
        for (;;) {
            int u = 0;
            if (lane == 0) u = (int)atomicAdd(&hdr->merge_next, 1u);
            u = __shfl_sync(0xffffffffu, u, 0);
            if (u >= ntasks) break;
            const int run = u % nruns, mt = (u / nruns) % mtiles, img = u / (nruns * mtiles);
            const int lo = __ldg(offsets + img), hi = __ldg(offsets + img + 1);
            const int M = __ldcg(counts + img), out0 = __ldcg(out_offsets + img);
            const int N = hi - lo, i0 = mt * kF3Tile;
            if (N < 1 || N > max_tokens || lo < 0 || hi > total || i0 >= M) continue;
            if (nt >= (uint32_t)kM3Tasks) ok = wait(&sh->task_empty[nt % kM3Tasks], nt / kM3Tasks - 1);
            if (!__all_sync(0xffffffffu, ok)) break;
            if (lane == 0) {
                M3Task &q = sh->task[nt % kM3Tasks];
                q.end = 0;
                q.B = N - M;
                q.M = M;
                q.i0 = i0;
                q.rows = min(kF3Tile, M - i0);
                q.ct0 = run * ct_run;
                q.ct1 = min(nct, q.ct0 + ct_run);
                q.ld = score_pitch(N - M);
                q.P = kmat + kmat_offset(kmat_stride, lo, img);
                q.Xi = X + (size_t)lo * d;
                q.kept = order + lo;
                q.prop = order + lo + M;
                q.Yt = Y + (size_t)(out0 + i0) * d;
                q.kidx = kept_idx + out0 + i0;
                ptx::mbar_arrive(&sh->task_full[nt % kM3Tasks]);
            }
            ++nt;
        }
        if (ok && nt >= (uint32_t)kM3Tasks) ok = wait(&sh->task_empty[nt % kM3Tasks], nt / kM3Tasks - 1);
        if (__all_sync(0xffffffffu, ok)) {
            if (lane == 0) {
                sh->task[nt % kM3Tasks].end = 1;
                ptx::mbar_arrive(&sh->task_full[nt % kM3Tasks]);
            }
        } else {
            give_up();
        }
    } else {
        const int quarter = warp & 3;              // TMEM lanes 32 quarter .. + 31
        const uint32_t warp_rows = ptx::smem_u32(xtiles) + (uint32_t)(32 * quarter * kM3Pitch);
        const int rsub = lane >> 4, csub = 4 * (lane & 15);      // coalesced passes: 2 rows x 16 pieces of 16 bytes
        bool ok = true, more = true;
        // the tile whose rows are fetched next
        uint32_t t_next = 0;
        int ct_next = 0, tok = 0;
        auto settle = [&]() {
            ok = __all_sync(0xffffffffu, task_wait(t_next));
            more = ok && !sh->task[t_next % kM3Tasks].end;
            if (!more) return;
            const M3Task &q = sh->task[t_next % kM3Tasks];
            ct_next = q.ct0;
            const int r = 32 * quarter + lane;
            tok = __ldg(q.kept + q.i0 + min(r, q.rows - 1));
            if (q.ct0 == 0 && r < q.rows) q.kidx[r] = tok;
        };
        auto fetch = [&](uint32_t u) {               // rows past the tile's last repeat it; not stored
            const float *Xi = sh->task[t_next % kM3Tasks].Xi;
            const int col = ct_next * kM3N + csub;
            const uint32_t dst = warp_rows + (u & 1u) * kM3XBytes + (uint32_t)csub * 4u;
#pragma unroll
            for (int it = 0; it < 16; ++it) {
                const int r = 2 * it + rsub, tr = __shfl_sync(0xffffffffu, tok, r);
                ptx::cp_async_16(dst + (uint32_t)(r * kM3Pitch), Xi + (size_t)tr * d + min(col, d - 4), 16u);
            }
        };
        settle();
        uint32_t acc = 0;
        if (more) fetch(0);
        ptx::cp_async_commit();
        for (uint32_t u = 0; more; ++u) {
            const uint32_t t = t_next;
            const int ct = ct_next;
            const M3Task &q = sh->task[t % kM3Tasks];
            const bool last = ++ct_next == q.ct1;
            if (last) {
                ++t_next;
                settle();
            }
            if (more) fetch(u + 1);
            ptx::cp_async_commit();
            ptx::cp_async_wait<1>();
            __syncwarp();
            const uint32_t tile = warp_rows + (u & 1u) * kM3XBytes;
            if (q.B > 0) {
                const uint32_t buf = acc % kM3Acc;
                ok = __all_sync(0xffffffffu, ok && wait(&sh->acc_full[buf], acc / kM3Acc));
                if (!ok) break;
                ++acc;
                ptx::tc_fence_after();
                const uint32_t tm = tmem_base + ((uint32_t)(32 * quarter) << 16) + buf * kM3AccCols;
                const uint32_t row = tile + (uint32_t)(lane * kM3Pitch);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    uint32_t a[16], b[16], e[16];
                    ptx::tmem_ld16(tm + (uint32_t)(16 * h), a);
                    ptx::tmem_ld16(tm + (uint32_t)(kM3N + 16 * h), b);
                    ptx::tmem_ld16(tm + (uint32_t)(2 * kM3N + 16 * h), e);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const uint32_t at = row + (uint32_t)(64 * h + 16 * g);
                        const float4 x = ptx::ld_shared_v4(at);
                        float y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            y[i] = fmaf(alpha, __uint_as_float(a[4 * g + i]) + (__uint_as_float(b[4 * g + i]) + __uint_as_float(e[4 * g + i])), y[i]);
                        ptx::st_shared_v4(at, make_uint4(__float_as_uint(y[0]), __float_as_uint(y[1]), __float_as_uint(y[2]), __float_as_uint(y[3])));
                    }
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&sh->acc_empty[buf]);
            }
            const int col = ct * kM3N + csub;
            float *out = q.Yt + (size_t)(32 * quarter) * d + col;
#pragma unroll
            for (int it = 0; it < 16; ++it) {
                const int r = 2 * it + rsub;
                const float4 y = ptx::ld_shared_v4(tile + (uint32_t)(r * kM3Pitch + csub * 4));
                if (32 * quarter + r < q.rows && col < d) *reinterpret_cast<float4 *>(out + (size_t)r * d) = y;
            }
            __syncwarp();
            if (last && lane == 0) ptx::mbar_arrive(&sh->task_empty[t % kM3Tasks]);
        }
        ptx::cp_async_wait<0>();
        if (!ok) give_up();
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == kProdWarps) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, 512);
    }
}

}  // namespace rtp

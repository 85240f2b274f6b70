// Merge + pack (Eq. 7 and the output of Algorithm 1): Y = T_k + alpha * P T_p, written packed, on the
// tcgen05 tensor cores (bf16 inputs, fp32 accumulation in TMEM).
//
// A work unit is (image, tile of 128 consecutive KEPT tokens, tile of 256 output columns).  The contraction
// is alpha P . T_p; the kept tokens' own rows join in the epilogue, in fp32.
//   * A operand: the plan rows alpha P[p][0..B) in bf16, K-major, by tiled TMA from the plan buffer, whose
//     rows are positions among the kept tokens.
//   * B operand: the image's pruned rows from the compact copy by tiled TMA, MN-major (row = contraction
//     index, 64-column slabs of 128 bytes, 128-byte swizzle); its zero rows pad B to a multiple of 64.
//   * D: two 128-lane x 256-column fp32 accumulators in TMEM, so that the epilogue of one unit
//     overlaps the loads and UMMAs of the next.
//   * The kept tokens' rows: gathered from X by token index with 16-byte cp.async, coalesced, half a unit's
//     columns at a time into a tile; a thread of the epilogue adds its row's accumulator in place, then its warp
//     stores the rows, coalesced.
// What bounds it is what an SM takes in through TMA (about 31 bytes per clock), so nothing comes that way that
// need not: tiles of kept rows instead of token tiles with their pruned rows (a quarter of a corpus image, two
// fifths of a long one), own rows by another path instead of as UMMA operands against an identity tile.
// Against token tiles with own rows through the tensor cores (event times): 1024 x 400 at r = 0.25 426 -> 344 us,
// 128 images of 456-1156 tokens 141 -> 113, 16 x 2137 133 -> 71, 8 x 4512 223 -> 111, 64 x 400 39 -> 37; 1014 images of 69
// tokens 91 -> 89 at r = 0.25, 89 -> 95 at a dynamic ratio (99 and 103 while a unit of up to 64 rows took two tiles of own rows).
// The kernel is persistent: CTA c takes units c, c + gridDim.x, ...  When the Sinkhorn kernel ahead
// publishes a list of finished images, the units follow that list (its s-th entry takes the place of
// image s), the CTAs draw them from a counter, and the scheduler waits, bounded, for the entry it
// needs: the kernel is launched as a programmatic dependent and merges the first images on whatever
// SMs are free while the last ones still iterate.  Warp roles (480 threads):
// warps 0-7 epilogue (two warpgroups, one for each half of a unit's columns); warp 8 issues the TMA loads (the loads of a k-block from several lanes at once); warp 9 owns TMEM and
// its lane 0 issues the UMMAs;
// warp 10 lane 0 is the scheduler: it draws the units, looks up what the other roles need to know about
// them (a chain of dependent loads from L2) a few units ahead and hands them over through a small queue
// in shared memory; warps 11-14 fetch the kept tokens' rows.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace rtp {

constexpr int kMgTileM = 128;
constexpr int kMgTileN = 256;        // output columns per unit
constexpr int kMgBK = 64;            // contraction rows per k-block
constexpr int kMgLoaders = 128;      // threads that fetch the kept tokens' rows
constexpr int kMgEpilogue = 256;
constexpr int kMgThreads = kMgEpilogue + 96 + kMgLoaders;
constexpr int kMgLookahead = 1;       // units the scheduler may be ahead of the producer
constexpr int kMgABytes = kMgTileM * 128;            // A tile: 128 rows x 64 bf16
constexpr int kMgBBytes = kMgBK * kMgTileN * 2;      // B tile: 64 rows x 256 bf16 = 32 KB
constexpr int kMgBBoxBytes = kMgBK * 128;            // one 64-column slab of it
constexpr int kMgStageBytes = kMgABytes + kMgBBytes; // a k-block: a plan tile and a tile of pruned rows
constexpr int kMgOwnCols = 128;                      // columns of a tile of own rows: 256 bytes a row, the 16-byte pieces
constexpr int kMgOwnBytes = kMgTileM * kMgOwnCols * 2;   // of row r at places xor (r & 7), conflict-free either way
constexpr int kMgShortRows = 64;                     // a unit of up to so many rows: both halves of its columns in one tile
// Shared memory is shared out between k-blocks in flight and tiles of own rows by what a unit has of each: two k-blocks (B up to
// 128) to two tiles of own rows, or many k-blocks.
constexpr int kMgMaxStages = 3, kMgMaxBufs = 4;
constexpr int kMgDeepB = 256;
__host__ __device__ constexpr int merge_smem_bytes(int stages, int bufs)
{
    return stages * kMgStageBytes + bufs * kMgOwnBytes + 1024 /*alignment*/ + 1024 /*barriers, unit queue*/;
}
constexpr int kMgSmemMax = merge_smem_bytes(2, 4) > merge_smem_bytes(3, 2) ? merge_smem_bytes(2, 4) : merge_smem_bytes(3, 2);
static_assert(kMgSmemMax <= 227 * 1024, "one CTA per SM");

constexpr int kMgQueue = 16;         // ring of units between the producer and the other roles (about 6 in flight)

struct MergeBarriers {
    uint64_t full[kMgMaxStages];        // a k-block's tiles have landed
    uint64_t empty[kMgMaxStages];       // its UMMAs have read them
    uint64_t own_full[kMgMaxBufs];   // the kept tokens' rows are there
    uint64_t own_empty[kMgMaxBufs];  // their sums have been stored
    uint64_t accum_full[2];
    uint64_t accum_empty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
};

// What every role needs to know about a unit.  img = -1 ends the queue.
struct MergeUnit {
    int img, mt, ct;
    int t_begin, N, M, B, out0;
    bool valid;
    bool timed_out;   // the image's list entry never came
};

struct MergeQueue {
    volatile uint32_t head;          // units pushed by the scheduler
    volatile uint32_t prod;          // units the producer has taken
    volatile uint32_t tail;          // units every role is done with
    MergeUnit e[kMgQueue];
};

// Whether a unit's own rows take one tile instead of two.  The threads of the epilogue without a row then pass the tile by, and a
// thread that has passed a phase of a barrier by must know it complete before it waits for the next (a wait tells phases apart by
// parity only): with four tiles the one before belongs to unit n - 2 or an earlier one, which the accumulator's barrier has shown to
// be done; with two it can belong to unit n - 1.
__device__ inline bool merge_few_rows(const MergeUnit &q, int bufs)
{
    return bufs >= 4 && q.M - q.mt * kMgTileM <= kMgShortRows;
}

// Bounded wait for the n-th unit of the queue.  false = gave up, or the kernel is being abandoned.
__device__ inline bool merge_pop(MergeQueue *mq, const MergeBarriers *bars, uint32_t n, MergeUnit &q)
{
    for (uint32_t i = 0; i < ptx::kPollLimit && !bars->abort_flag; ++i) {
        if (mq->head > n) {
            __threadfence_block();
            q = mq->e[n % kMgQueue];
            return true;
        }
        __nanosleep(40);
    }
    return false;
}

// Image in slot `slot` of the list of finished plans (bounded wait), -1 if it never shows up.
__device__ inline int merge_wait_image(const int32_t *ready_list, int slot)
{
    for (uint32_t i = 0; i < ptx::kPollLimit; ++i) {
        const int v = ptx::ld_acquire_gpu(ready_list + slot);
        if (v != 0) return v - 1;
        __nanosleep(40);
    }
    return -1;
}

__device__ inline MergeUnit merge_unit(int u, int mtiles, int nct, const int32_t *__restrict__ offsets,
                                       const int32_t *__restrict__ counts,
                                       const int32_t *__restrict__ out_offsets, int max_tokens, int total,
                                       const int32_t *ready_list)
{
    MergeUnit q;
    q.ct = u % nct;
    const int v = u / nct;
    q.mt = v % mtiles;
    q.img = v / mtiles;
    q.timed_out = false;
    if (ready_list) {
        q.img = merge_wait_image(ready_list, q.img);
        if (q.img < 0) {
            q.valid = false;
            q.timed_out = true;
            return q;
        }
    }
    // L2 loads (with a ready list this kernel may have started before the selection wrote these), all issued
    // before the first use: one trip, not one per value (img is a valid image number either way)
    const int o_lo = __ldcg(offsets + q.img), o_hi = __ldcg(offsets + q.img + 1);
    const int m_img = __ldcg(counts + q.img), out0 = __ldcg(out_offsets + q.img);
    q.t_begin = o_lo;
    q.N = o_hi - o_lo;
    q.valid = q.N >= 1 && q.N <= max_tokens && o_lo >= 0 && o_hi <= total && q.mt * kMgTileM < m_img;
    q.M = q.valid ? m_img : 0;
    q.B = q.N - q.M;
    q.out0 = q.valid ? out0 : 0;
    return q;
}

__global__ void __launch_bounds__(kMgThreads, 1)
merge_umma_kernel(const __grid_constant__ CUtensorMap tmapXp, const __grid_constant__ CUtensorMap tmapP,
                  const __nv_bfloat16 *__restrict__ X, const int32_t *__restrict__ offsets, int d,
                  int batch, int mtiles, const int32_t *__restrict__ counts,
                  const int32_t *__restrict__ out_offsets, const int32_t *__restrict__ order,
                  int max_tokens, int total, __nv_bfloat16 *__restrict__ Y, int32_t *__restrict__ kept_idx,
                  WsHeader *__restrict__ hdr, const int32_t *ready_list, int by_image, int stages, int bufs)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *own = smem + stages * kMgStageBytes;
    MergeBarriers *bars = reinterpret_cast<MergeBarriers *>(own + bufs * kMgOwnBytes);
    MergeQueue *mq = reinterpret_cast<MergeQueue *>(own + bufs * kMgOwnBytes + 256);
    static_assert(sizeof(MergeBarriers) <= 256 && sizeof(MergeQueue) <= 768, "");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nct = (d + kMgTileN - 1) / kMgTileN;
    const int nunits = batch * mtiles * nct;

    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            ptx::mbar_init(&bars->full[s], 1);
            ptx::mbar_init(&bars->empty[s], 1);
        }
        for (int b = 0; b < bufs; ++b) {
            ptx::mbar_init(&bars->own_full[b], kMgLoaders);
            ptx::mbar_init(&bars->own_empty[b], 128);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars->accum_full[b], 1);
            ptx::mbar_init(&bars->accum_empty[b], kMgEpilogue);
        }
        bars->abort_flag = 0;
        mq->head = 0;
        mq->prod = 0;
        mq->tail = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 9) {
        ptx::tmem_alloc(&bars->tmem_base, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = bars->tmem_base;
    const uint32_t smem_base = ptx::smem_u32(smem);
    // everything above is local set-up; the plan, the selection and the compact copy come from the
    // kernels ahead in the stream: wait for them to end, or, with a list of finished images, for each
    // image's entry (which is published after everything the image needs has been written)
    ptx::grid_dep_launch();
    if (!ready_list) ptx::grid_dep_wait();

    if (warp == 8) {
        // ---------------- producer: tiled TMA for both operands -------------------------------------
        // The whole warp walks the units and k-blocks in step (every lane takes the same waits); the loads of a
        // k-block are issued by as many lanes at once, one load each (lanes 0-3: the 64-column slabs of the B
        // tile, lane 4: the plan tile): one thread issuing them one after the other spent about 145 cycles in
        // each issue, 40 % of the kernel's time.
        if (lane == 0) {
            ptx::prefetch_tensormap(&tmapXp);
            ptx::prefetch_tensormap(&tmapP);
        }
        int s = 0;                                    // place in the ring of k-blocks, and its phase
        uint32_t phase = 1;                           // (the first wait on each place returns at once)
        bool alive = true;
        for (uint32_t n = 0; alive && !bars->abort_flag; ++n) {
            MergeUnit q;
            const bool got = merge_pop(mq, bars, n, q);
            if (!__all_sync(0xffffffffu, got)) {
                bars->abort_flag = 1;
                if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                break;
            }
            if (q.img < 0) break;
            __syncwarp();                             // every lane has read the entry before it may be reused
            if (lane == 0) mq->prod = n + 1;
            if (ready_list) ptx::fence_proxy_async_all();   // the plan was written with ordinary stores
            const int nkb = (q.B + kMgBK - 1) / kMgBK;
            const int row0 = q.t_begin + q.mt * kMgTileM;
            const int xp0 = xp_row0(q.t_begin, q.img);
            const int col0 = q.ct * kMgTileN;
            const int nslab = min(kMgTileN, d - col0 + 63) / 64;   // 64-column slabs with any column < d
            for (int kb = 0; kb < nkb; ++kb) {
                const bool ok = ptx::mbar_wait(&bars->empty[s], phase);
                if (!__all_sync(0xffffffffu, ok)) {
                    bars->abort_flag = 1;
                    if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                    alive = false;
                    break;
                }
                if (lane == 0) ptx::mbar_arrive_expect_tx(&bars->full[s], kMgABytes + nslab * kMgBBoxBytes);
                __syncwarp();
                const uint32_t a_dst = smem_base + s * kMgStageBytes;
                if (lane < nslab)
                    ptx::tma_load_2d(a_dst + kMgABytes + lane * kMgBBoxBytes, &tmapXp, &bars->full[s], col0 + lane * 64, xp0 + kb * kMgBK);
                else if (lane == 4)
                    ptx::tma_load_2d(a_dst, &tmapP, &bars->full[s], kb * kMgBK, row0);
                if (++s == stages) {
                    s = 0;
                    phase ^= 1u;
                }
            }
        }
    } else if (warp == 10) {
        // ---------------- scheduler -------------------------------------------------------------------
        if (lane == 0) {
            uint32_t pushed = 0, drawn = 0;
            auto push = [&](const MergeUnit &q) {
                // stay a few units ahead of the producer, no more: a unit drawn is a unit no other CTA
                // can take.  (The queue itself cannot fill up: fewer units are in flight than it holds.)
                for (uint32_t i = 0; pushed - mq->prod >= (uint32_t)kMgLookahead ||
                                     pushed - mq->tail >= (uint32_t)kMgQueue; ++i) {
                    if (i >= ptx::kPollLimit || bars->abort_flag) return false;
                    __nanosleep(100);
                }
                mq->e[pushed % kMgQueue] = q;
                __threadfence_block();
                mq->head = ++pushed;
                return true;
            };
            // with a list of finished images: not before the run's number is there (until then the list
            // and the unit counter are what the run before left)
            bool ok = !ready_list || ptx::wait_equal_gpu(&hdr->run_tag, ptx::ld_acquire_gpu(&hdr->launch_seq));
            while (ok && !bars->abort_flag) {
                // next unit: from the shared counter when the units follow the list of finished images
                const bool drawn_units = ready_list && !by_image;
                const int u = drawn_units ? (int)atomicAdd(&hdr->merge_next, 1u) : (int)(blockIdx.x + drawn++ * gridDim.x);
                if (u >= nunits) break;
                MergeUnit q = merge_unit(u, mtiles, nct, offsets, counts, out_offsets, max_tokens, total,
                                         drawn_units ? ready_list : nullptr);
                // (by image: what the unit needs to know is there before the image is)
                if (by_image && q.valid && merge_wait_image(ready_list, q.img) < 0) q.timed_out = true;
                if (q.timed_out) ok = false;
                else if (q.valid) ok = push(q);
            }
            MergeUnit end{};
            end.img = -1;
            if (ok) ok = push(end);
            if (!ok && !bars->abort_flag) {
                bars->abort_flag = 1;
                atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
            }
        }
    } else if (warp == 9) {
        // ---------------- UMMA issuer -----------------------------------------------------------------
        if (lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16(kMgTileM, kMgTileN, false, true);
            int s = 0;
            uint32_t phase = 0;
            for (uint32_t n = 0; !bars->abort_flag; ++n) {
                MergeUnit q;
                if (!merge_pop(mq, bars, n, q)) {
                    bars->abort_flag = 1;
                    atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                    break;
                }
                if (q.img < 0) break;
                const int nkb = (q.B + kMgBK - 1) / kMgBK;
                const int buf = n & 1;
                if (n >= 2) {
                    if (!ptx::mbar_wait(&bars->accum_empty[buf], ((n >> 1) - 1) & 1)) {
                        bars->abort_flag = 1;
                        atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                        break;
                    }
                    ptx::tc_fence_after();
                }
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kMgTileN);
                bool failed = false;
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!ptx::mbar_wait(&bars->full[s], phase)) {
                        failed = true;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t a_base = smem_base + s * kMgStageBytes, b_base = a_base + kMgABytes;
#pragma unroll
                    for (int k = 0; k < kMgBK / 16; ++k) {
                        // A: K-major, 32 bytes further along the 128-byte row per 16 k.
                        // B: MN-major, 16 k-rows = 2 groups of 8 rows = 2048 bytes further; 64-column
                        //    slabs are kMgBK * 128 bytes apart, 8-row groups 1024 bytes apart.
                        const uint64_t da = ptx::smem_desc_sw128(a_base + k * 32, 16, 1024);
                        const uint64_t db = ptx::smem_desc_sw128(b_base + k * 2048, kMgBK * 128, 1024);
                        ptx::umma_bf16(d_tmem, da, db, idesc, (kb | k) != 0);
                    }
                    ptx::umma_commit(&bars->empty[s]);
                    if (++s == stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
                if (failed) {
                    bars->abort_flag = 1;
                    atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                    break;
                }
                ptx::umma_commit(&bars->accum_full[buf]);    // (at once for an image with nothing pruned)
            }
        }
    } else if (warp >= 11) {
        // ---------------- loaders: the kept tokens' own rows ------------------------------------------
        // A warp fetches 32 rows, two at a time (16 lanes x 16 bytes = 128 columns each).  In a unit of up to 64 rows the second two
        // warps take the second half of the columns, into the second half of the same tile: four such units are in flight, not two.
        const int sub = lane >> 4, piece = lane & 15;
        const uint32_t own_base = ptx::smem_u32(own) + (uint32_t)(((warp - 11) * 32 + sub) * 256);
        int buf = 0;                                  // tile of own rows, and its phase
        uint32_t phase = 1;
        bool alive = true;
        for (uint32_t n = 0; alive; ++n) {
            MergeUnit q;
            const bool got = merge_pop(mq, bars, n, q);
            if (!__all_sync(0xffffffffu, got)) {
                bars->abort_flag = 1;
                if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                break;
            }
            if (q.img < 0) break;
            const bool few = merge_few_rows(q, bufs);
            const int right = few ? (warp - 11) >> 1 : 0, lrow = (few ? (warp - 11) & 1 : warp - 11) * 32;
            const int p = q.mt * kMgTileM + lrow + lane;     // position among the kept tokens
            const int tok = p < q.M ? __ldcg(order + q.t_begin + p) : -1;
            if (q.ct == 0 && right == 0 && tok >= 0) kept_idx[q.out0 + p] = tok;
            const int nrows = max(0, min(32, q.M - (q.mt * kMgTileM + lrow)));
            const int col_end = min(d, (q.ct + 1) * kMgTileN);
            // (the second half's tile also where a unit has no such columns: a thread of the epilogue that passed a tile by could
            // take an earlier phase of its barrier for a later one)
            for (int col = q.ct * kMgTileN; col < (q.ct + 1) * kMgTileN; col += few ? kMgTileN : kMgOwnCols) {
                const bool ok = ptx::mbar_wait(&bars->own_empty[buf], phase);
                if (!__all_sync(0xffffffffu, ok)) {
                    bars->abort_flag = 1;
                    if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                    alive = false;
                    break;
                }
                const int c = col + right * kMgOwnCols + piece * 8;
                const __nv_bfloat16 *src = X + (size_t)q.t_begin * d + c;
                const uint32_t dst = own_base + (uint32_t)(buf * kMgOwnBytes);
#pragma unroll 4
                for (int r = 0; r < nrows; r += 2) {
                    const int t = __shfl_sync(0xffffffffu, tok, r + sub);
                    if (t >= 0 && c < col_end)
                        ptx::cp_async_16(dst + (uint32_t)(r * 256 + ((piece ^ ((r + sub) & 7)) << 4)), src + (size_t)t * d, 16u);
                }
                ptx::cp_async_arrive(&bars->own_full[buf]);  // once this thread's copies have landed
                if (++buf == bufs) {
                    buf = 0;
                    phase ^= 1u;
                }
            }
        }
        ptx::cp_async_commit();
        ptx::cp_async_wait<0>();
    } else {
        // ---------------- warps 0-7: epilogue ---------------------------------------------------------
        const int row = tid & 127, half = tid >> 7;           // TMEM lane = row of the tile; which half of the columns
        int ob = 0;                                           // tile of own rows of the unit's first half, and its phase
        uint32_t phase = 0;
        for (uint32_t n = 0;; ++n) {
            MergeUnit q;
            const bool got = merge_pop(mq, bars, n, q);
            if (!__all_sync(0xffffffffu, got)) {
                bars->abort_flag = 1;
                if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                break;
            }
            if (q.img < 0) break;
            const int buf = n & 1;
            const int col = q.ct * kMgTileN + half * kMgOwnCols, ncols = min(kMgOwnCols, d - col);    // (may be <= 0)
            // own rows: the tile of this thread's half (rows past the kept ones of a unit of up to 64 have none)
            const bool few = merge_few_rows(q, bufs), has_own = !few || row < kMgShortRows;
            int mine = few ? ob : ob + half;
            uint32_t mine_phase = phase;
            if (mine >= bufs) {
                mine -= bufs;
                mine_phase ^= 1u;
            }
            ob += few ? 1 : 2;
            if (ob >= bufs) {
                ob -= bufs;
                phase ^= 1u;
            }
            // the TMEM loads below are warp-collective: take the go / no-go decision per warp
            bool ok = !bars->abort_flag && ptx::mbar_wait(&bars->accum_full[buf], (n >> 1) & 1) &&
                      (!has_own || ptx::mbar_wait(&bars->own_full[mine], mine_phase));
            if (!__all_sync(0xffffffffu, ok)) {
                bars->abort_flag = 1;
                if (lane == 0) atomicOr(&hdr->status, RTPRUNE_DEV_TIMEOUT);
                break;
            }
            ptx::tc_fence_after();
            // unit n's accumulator is complete, so every epilogue thread is done with unit n - 2 (its
            // accumulator buffer was handed back) and the producer, the UMMA issuer and the loaders are past it:
            // those entries are free
            if (tid == 0 && n >= 1) mq->tail = n - 1;
            const int w0 = row & ~31, prow0 = q.mt * kMgTileM + w0;      // the warp's first row of the tile, and of the kept ones
            uint8_t *const tile = own + mine * kMgOwnBytes + (few ? half * (kMgShortRows * 256) : 0);
            // a warp whose 32 rows all lie past the kept ones has nothing to add or store
            if (prow0 < q.M && q.B > 0) {
                uint8_t *const srow = tile + row * 256;
                for (int c0 = 0; c0 < ncols; c0 += 32) {
                    uint32_t r[32];
                    ptx::tmem_ld32(tmem_base + ((uint32_t)w0 << 16) + (uint32_t)(buf * kMgTileN + half * kMgOwnCols + c0), r);
                    uint4 x[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) x[g] = *reinterpret_cast<const uint4 *>(srow + (((c0 / 8 + g) ^ (row & 7)) << 4));
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        float f[8];
                        Elem<__nv_bfloat16>::unpack(x[g], f);
                        __nv_bfloat162 o[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            o[e] = __floats2bfloat162_rn(f[2 * e] + __uint_as_float(r[8 * g + 2 * e]),
                                                         f[2 * e + 1] + __uint_as_float(r[8 * g + 2 * e + 1]));
                        *reinterpret_cast<uint4 *>(srow + (((c0 / 8 + g) ^ (row & 7)) << 4)) = *reinterpret_cast<uint4 *>(o);
                    }
                }
            }
            ptx::tc_fence_before();
            ptx::mbar_arrive(&bars->accum_empty[buf]);
            __syncwarp();                                     // the warp's rows are complete
            const int sub = lane >> 4, piece = lane & 15, nrows = min(32, q.M - prow0);      // (may be <= 0)
            __nv_bfloat16 *dst = Y + (size_t)(q.out0 + prow0) * d + col + piece * 8;
            if (piece * 8 < ncols) {
#pragma unroll 8
                for (int r = sub; r < nrows; r += 2)
                    *reinterpret_cast<uint4 *>(dst + (size_t)r * d) =
                        *reinterpret_cast<const uint4 *>(tile + (w0 + r) * 256 + ((piece ^ (r & 7)) << 4));
            }
            if (has_own) ptx::mbar_arrive(&bars->own_empty[mine]);     // (after this thread's reads)
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, 512);
    }
    // keep the stream's order: this grid does not end before the ones ahead of it have
    if (ready_list) ptx::grid_dep_wait();
}

}  // namespace rtp

// The projecting CTAs of a launch that runs two layers side by side: rows of G = X Wx^T + b of the upper layer for a chunk of timesteps
// at a time, as soon as the lower layer's CTAs have stored that chunk of X (two bf16 planes).  The matrix (18 MB at 1500 x 1500)
// is too large to stay on these SMs beside the recurrences, so each chunk streams it from L2 once: a CTA owns mb blocks of rb
// rows, weights and activations arrive through a ring of tensor copies, one warp issues the products into mb accumulators of
// tensor memory, four warps read them back, add the bias and store.  A chunk costs what its bytes take at the 50 - 60 bytes a
// clock an SM draws from L2; the weights of its first stages are requested before its activations exist.
#pragma once
#include "common.cuh"
#include "device_util.cuh"

namespace lstm {
namespace {

constexpr int kSpStages = 8;                    // most stages of the ring
constexpr int kSpBar = 1;                       // named barrier of the read-back warps

// smem_raw: this CTA's dynamic shared memory.  All kThreads threads call it; `cta` counts from 0.
__device__ __forceinline__ void stack_proj_role(unsigned char *smem_raw, const CUtensorMap *tmap_w, const CUtensorMap *tmap_x, const CUtensorMap *tmap_xlo,
                                                const StackProjArgs &a, int cta)
{
    __shared__ __align__(8) unsigned long long full_bar[kSpStages], empty_bar[kSpStages], accum_bar, drained_bar;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t w_bytes = (uint32_t)a.rb * 128u, x_bytes = (uint32_t)a.nrp * 128u, stage_bytes = a.mb * w_bytes + 2 * x_bytes;
    const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int r0 = cta * a.mb * a.rb;
    LSTM_CHECK_SMEM_END((size_t)(tiles - smem_u32(smem_raw)) + (size_t)a.stages * stage_bytes + 120 * 128, a.status);     // (the last block is read as 128 rows)

    if (tid == 0) {
        abort_s = 0;
        for (int s = 0; s < a.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
        mbar_init(smem_u32(&accum_bar), 1);
        mbar_init(smem_u32(&drained_bar), 12);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_s;
    volatile int *abort_v = &abort_s;

    if (warp == 0) {
        if (lane == 0) {
            // ---- tensor copies: the K blocks of chunk after chunk.  Two cursors, one for the weights and one for the activations
            // behind it (counted up: a division by the number of stages or blocks costs more than a copy's issue).
            int w_stage = 0, w_kb = 0, w_ahead = 0, w_left = a.nchunks * a.kblocks, x_stage = 0;       // w_ahead: stages with weights and no activations
            uint32_t w_phase = 1;
            bool ok = true;
            auto request_weights = [&]() {                  // (the stage must be free)
                const uint32_t fb = smem_u32(&full_bar[w_stage]), dst = tiles + (uint32_t)w_stage * stage_bytes;
                mbar_expect_tx(fb, stage_bytes);
                for (int b = 0; b < a.mb; ++b) tma_load_2d(dst + b * w_bytes, tmap_w, fb, w_kb * 64, r0 + b * a.rb);
                if (++w_kb == a.kblocks) w_kb = 0;
                if (++w_stage == a.stages) { w_stage = 0; w_phase ^= 1u; }
                ++w_ahead;
                --w_left;
            };
            for (int chunk = 0; chunk < a.nchunks && ok; ++chunk) {
                // while the chunk is not there: the weights of the stages that are free already
                while (w_left > 0 && w_ahead < a.stages && mbar_try_wait(smem_u32(&empty_bar[w_stage]), w_phase)) request_weights();
                ok = wait_count(a.stored + chunk, a.n_stored, abort_v, a.spin_limit, a.status);
                asm volatile("fence.proxy.async;" ::: "memory");
                for (int kb = 0; kb < a.kblocks && ok; ++kb) {
                    if (w_ahead == 0) {
                        ok = mbar_wait(smem_u32(&empty_bar[w_stage]), w_phase, abort_v);
                        if (!ok) break;
                        request_weights();
                    }
                    const uint32_t fb = smem_u32(&full_bar[x_stage]), dst = tiles + (uint32_t)x_stage * stage_bytes + a.mb * w_bytes;
                    tma_load_2d(dst, tmap_x, fb, kb * 64, chunk * a.chunk_rows);
                    tma_load_2d(dst + x_bytes, tmap_xlo, fb, kb * 64, chunk * a.chunk_rows);
                    if (++x_stage == a.stages) x_stage = 0;
                    --w_ahead;
                }
            }
        }
    } else if (warp == 1) {
        // ---- products: accumulator b at column b * 2 * nrp, columns [0, nrp) with the hi plane, [nrp, 2 nrp) with the lo plane
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * a.nrp) >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int chunk = 0; chunk < a.nchunks && ok; ++chunk) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&drained_bar), (uint32_t)(chunk & 1) ^ 1u, abort_v));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int i = 0; i < a.kblocks && ok; ++i) {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[s]), ph, abort_v));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t sa = tiles + (uint32_t)s * stage_bytes;
                const uint64_t bdesc = umma_desc_sw128(sa + a.mb * w_bytes);
                if (elect_one()) {
                    for (int b = 0; b < a.mb; ++b) {
                        const uint64_t adesc = umma_desc_sw128(sa + b * w_bytes);
#pragma unroll
                        for (int k = 0; k < 4; ++k) umma_bf16(tmem + (uint32_t)(b * 2 * a.nrp), adesc + 2 * k, bdesc + 2 * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
                    }
                    umma_commit(smem_u32(&empty_bar[s]));
                    if (i == a.kblocks - 1) umma_commit(smem_u32(&accum_bar));
                }
                __syncwarp();
                if (++s == a.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp >= 4) {
        // ---- read-back: a lane is one row of Wx, one column of G; the three warps of a lane quadrant take every third batch of 16
        // columns (four warps alone take 7.5 us for 3 x 104 rows by 80, during which the products wait)
        const int lq = warp & 3, part = (warp >> 2) - 1, row = lq * 32 + lane;
        for (int chunk = 0; chunk < a.nchunks; ++chunk) {
            const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&accum_bar), (uint32_t)chunk & 1u, abort_v));
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int m0 = chunk * a.chunk_rows, nr = min(a.chunk_rows, a.M - m0);
            int turn = part;
            for (int b = 0; b < a.mb && ok; ++b) {
                const int n = r0 + b * a.rb + row;
                const bool real = row < a.rb && n < a.N;
                const float bv = real ? a.bias[n] : 0.0f;
                const uint32_t acc = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(b * 2 * a.nrp);
                for (int c0 = 0; c0 < nr; c0 += 16) {
                    if (turn != 0) { --turn; continue; }
                    turn = 2;
                    float v[16], lo[16];
                    const bool wide = c0 + 8 < a.nrp;              // (the last batch of an odd number of eights is eight columns)
                    if (wide) { tmem_ld<16>(acc + (uint32_t)c0, v); tmem_ld<16>(acc + (uint32_t)(a.nrp + c0), lo); }
                    else {
                        float v8[8], lo8[8];
                        tmem_ld<8>(acc + (uint32_t)c0, v8);
                        tmem_ld<8>(acc + (uint32_t)(a.nrp + c0), lo8);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < 8; ++i) { v[i] = v8[i]; lo[i] = lo8[i]; v[8 + i] = lo[8 + i] = 0.0f; }
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (real) {
                        float *g = a.G + (size_t)(m0 + c0) * a.N + n;
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < nr) g[(size_t)i * a.N] = v[i] + lo[i] + bv;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&drained_bar));
            // One answer for all twelve warps: a wait that gives up does so warp by warp, and one of them may see the flag just before
            // the accumulators are complete and the others just behind; none may leave while others come to this barrier.
            if (!bar_all(kSpBar, 12 * 32, ok)) break;
            if (tid == 128 && cta != a.withhold_cta) add_count(a.ready + chunk);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(*abort_v)) {
        // a wait gave up: copies and products may still be in flight; they land within microseconds
        if (tid == 0) atomicExch(a.status, kStatusTimeout);
        const long long t0 = clock64();
        while (clock64() - t0 < 200000) { }
        __syncthreads();
    }
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

}  // namespace
}  // namespace lstm

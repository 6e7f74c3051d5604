// Batched recurrent kernel for bf16 weights on the 5th-generation tensor cores: the serial half of the LSTM
// forward pass (paper, Section 4, cell equations with zero hidden layers per gate)
//     z = G[t] + Wh h_{t-1};  i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c_t = f c_{t-1} + i g;
//     h_t = o tanh(c_t)
// for several sequences at once, up to kTcMaxRows per pass, where the per-step product
// Wh_slice [4u x H] . h_{t-1} [H x B] is a real (if skinny) matrix product.
//
// One cooperative launch runs all T steps of one layer (both directions on disjoint CTA groups).  A CTA owns upc
// consecutive hidden units (upc a multiple of four, all four gate rows of a unit).  Two CTAs form a cluster: each
// keeps the weight rows of BOTH CTAs' units (2 x 4 x upc <= 128 rows) but only its half of the K range, so each
// fetches and multiplies half of h, and the partial sums of the partner's units travel through distributed shared
// memory.  What a step does, and why it is laid out like this:
//
//   * The weights sit in TENSOR MEMORY as the A operand (row = lane, two bf16 per column) for the whole sequence:
//     128 rows by up to 960 columns.  Shared memory is then free for the B operand of a whole step, and an
//     instruction reads only its small B tile from it.  The issuing thread must be elected from a converged warp and
//     take its operands from warp-uniform values: measured for 48 instructions of N = 16 / 48, 970 / 1370 cycles; the
//     same loop entered by "lane == 0" with per-thread operands took 8260.
//   * h travels between the CTAs as 32-bit words with a phase bit (device_util.cuh), in 16-byte chunks of four units
//     of one batch row; the consumers poll the words themselves, twelve warps with all their chunks in
//     flight, split them into bf16 planes and store those as the swizzled B operand (rows 0 .. Bp - 1 hi, Bp .. 2 Bp - 1
//     lo).  Pruned layers have a third plane: their lists (recur_csr.cu) multiply h in fp32, so a batch of them carries h
//     as its own 32 bits and splits it into three terms that hold all 24: with two terms the recurrent products alone were
//     off by 9e-7 (1.5e-7 with three, as with the lists).  The split and the third plane cost 5 - 16 % of a call
//     (2 x 1500, T = 35: 4 rows 233 -> 245 us, 16 rows 249 -> 286; 2 x 800, 16 rows 198 -> 219).  A step has no
//     stamps, no release or acquire fence and no second trip for the data.
//     LDG.128 reads a row range that all SMs share at 55 - 60 bytes per clock and SM (24 when a quarter warp's 128 bytes
//     straddle two lines), a tensor copy at about 20.
//   * The K range is handed to the issuing warps in groups as they arrive (a named barrier each: an issuing thread's
//     mbarrier wait queues behind its own instructions), so the products overlap the fetch.
//   * Accumulator row = 4 x unit + gate = TMEM lane: a thread reads its row's hi and lo columns for a few batch
//     rows of the partner and sends them (st.async, completes on the partner's mbarrier), then its own batch rows, adds what
//     the partner sent, applies its gate's function, and a 4 x 4 transpose inside the quad gives every thread all four gates
//     of a (unit, batch row) of its own; c stays in registers.  The pair splits this work by batch rows, not by units: all
//     lanes of a warp then have gates to compute and a thread half as many (us per step, by units -> by rows: H = 1500, 20
//     rows 3.70 -> 3.28, 50 rows 6.10 -> 5.03; H = 600, 50 rows 4.42 -> 3.34; two directions of 800, 16 rows 2.67 -> 2.40).
//   * A step is bound by the instructions on this chain (16 warps on four schedulers), so every address is a fixed
//     offset from a pointer that advances by one step.
//
// Per step (launch time / T, one layer), against the previous kernel (weights in shared memory as the A operand, h planes by
// tensor copies behind one stamp per CTA, three "lane == 0" issuing threads): H = 1500, 20 rows 5.8 -> 3.3 us; two directions of
// 800, 16 rows 4.7 -> 2.4 us; 50 rows in a pass 5.0 us (batches above 64 ran as passes of four rows before).
//
// Pair mode needs K for both halves and clusters of two; without it (few rows of narrow layers, tc_single_rows in api.cu, or
// LSTM_B200_RECUR=tc1) a CTA works alone on its own rows and all of K.  Every wait on another CTA is bounded; on expiry the CTA records a timeout status,
// stops waiting for the rest of the launch and runs to the common exit, where tensor memory is released.
#include "common.cuh"
#include "device_util.cuh"

#include <cstdio>
#include <cstring>

namespace lstm {
namespace {

constexpr int kThreads = kTcThreads;            // 128 registers a thread
constexpr int kPollers = 12;                    // warps that fetch the operand (a multiple of 4 keeps their addresses linear)
constexpr int kIssuer = 12;                     // first of the warps that issue the products; all warps finish
constexpr int kMaxGroups = 5;                   // operand groups of 16 * kPollers columns
// Clock ticks from the CTA's own barrier to its first poll: nothing can have arrived earlier, and loads that come too early
// delay the words they wait for.  Measured us per step at 0 / 600 / 1000 ticks: H = 1500, 8 rows 2.40 / 2.30 / 2.47; two
// directions of 800, 8 rows 1.97 / 1.97 / 2.11.
constexpr unsigned kPollDelay = 600;
constexpr int kGroupBar = 2;                    // named barrier of group 0: polling warps arrive, an issuing warp waits

// Batch rows the first CTA of a pair finishes, for the units of both; the second one takes the rest, so that every lane of a
// warp has gates to compute and the row groups of a line of exchange words keep one writer.  A single row group cannot be
// split like that: there each CTA finishes its own units.  A CTA alone finishes all 8 rg.
__host__ __device__ constexpr int tc_rows_of_first(int rg, bool pair) { return pair ? (rg + 1) / 2 * 8 : 8 * rg; }
// batch rows a thread finishes per accumulator row: four warps share the rows of a lane quadrant
__host__ __device__ constexpr int tc_rows_per_thread(int rows) { return rows <= 16 ? 4 : rows <= 32 ? 8 : 16; }
// operand groups a lane has in flight: 16-byte chunks of rg batch rows each, at most twelve (registers)
__host__ __device__ constexpr int tc_groups_in_flight(int rg) { return 12 / rg < kMaxGroups ? 12 / rg : kMaxGroups; }

// ---- two-CTA cluster helpers: the partner's shared memory and barriers
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_smem_addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_smem_addr), "r"(rank));
    return r;
}
// one word into another CTA's shared memory; the bytes are counted on that CTA's barrier
__device__ __forceinline__ void st_async(uint32_t remote_dst, float v, uint32_t remote_bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                 ::"r"(remote_dst), "r"(__float_as_uint(v)), "r"(remote_bar) : "memory");
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// D[tmem] += A[tmem] . B[smem]
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint4 &v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// N columns of this warp's lane quadrant (no wait)
template <int N> __device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[N])
{
    if constexpr (N == 4)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(taddr));
    else if constexpr (N == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(taddr));
    else
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                       "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]) : "r"(taddr));
}

// 4 x 4 transpose inside a quad: lane j of the quad enters with its row v[0..3] and leaves with column j
__device__ __forceinline__ void quad_transpose(float &v0, float &v1, float &v2, float &v3, int j)
{
    const bool o1 = j & 1, o2 = j & 2;
    const float s0 = o1 ? v0 : v1, s1 = o1 ? v2 : v3;
    const float r0 = __shfl_xor_sync(0xffffffffu, s0, 1), r1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    if (o1) { v0 = r0; v2 = r1; } else { v1 = r0; v3 = r1; }
    // now (v0, v1) = rows (j & ~1, j | 1) of column (j & 1), (v2, v3) the same of column 2 + (j & 1)
    const float s2 = o2 ? v0 : v2, s3 = o2 ? v1 : v3;
    const float r2 = __shfl_xor_sync(0xffffffffu, s2, 2), r3 = __shfl_xor_sync(0xffffffffu, s3, 2);
    if (o2) { v0 = r2; v1 = r3; } else { v2 = r2; v3 = r3; }
}

// RG: groups of eight batch rows of a pass; TERMS: bf16 terms of h, two from words {hi | lo}, three from words that are h itself
template <int RG, bool PAIR, int TERMS>
__global__ void __launch_bounds__(kThreads, 1) recur_tc_kernel(const RecurTcArgs a)
{
    constexpr int Bp = 8 * RG, N = tc_columns(RG, TERMS), HB = tc_rows_of_first(RG, PAIR), RS = tc_rows_per_thread(HB);
    constexpr bool UNITS = PAIR && RG == 1;
    constexpr int KI = tc_groups_in_flight(RG), NACC = tc_accumulators(RG, TERMS);
    constexpr uint32_t tmem = 0;                                            // all 512 columns are ours: they start at address 0
    constexpr uint32_t acc_col = 512u - tc_acc_columns(RG, TERMS);                 // accumulators behind the weights
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long accum_bar, partial_bar[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int H = a.H, B = a.B, T = a.T, D = a.D, upc = a.upc;
    const int d = a.dir0 + blockIdx.x / a.ncta_dir;
    const int cta = blockIdx.x % a.ncta_dir;
    const int rank = PAIR ? (int)cluster_ctarank() : 0;
    const int RT = PAIR ? 8 * upc : 4 * upc;                                // accumulator rows of the tile
    const int k_lo = rank * a.KH, k_n = min(a.KH, H - k_lo);                // this CTA's K range
    const int nk16 = (k_n + 15) >> 4;
    const int ngroups = (nk16 + kPollers - 1) / kPollers;                   // warp w fetches piece w of every group
    const int nissue = min(NACC, ngroups);                                  // issuing warps, each with an accumulator

    // shared memory: operand tiles of 64 columns [N rows][128 bytes, swizzled], then the partner's partial sums [2][HB][RT]
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *op = smem_raw + (base - smem_u32(smem_raw));
    const int tiles = (a.KH + 63) >> 6;
    float *zs2 = reinterpret_cast<float *>(op + (size_t)tiles * N * 128);
    LSTM_CHECK_SMEM_END(reinterpret_cast<unsigned char *>(zs2 + (PAIR ? 2 * RT * HB : 0)) - smem_raw, a.status);

    if (tid == 0) {
        abort_s = 0;
        mbar_init(smem_u32(&accum_bar), (uint32_t)nissue);
        mbar_init(smem_u32(&partial_bar[0]), 1);
        mbar_init(smem_u32(&partial_bar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kIssuer) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0 && tmem_base_s != 0) atomicExch(a.status, kStatusInternal);
    volatile int *abort_v = &abort_s;

    // Exchange words: this launch's set starts with every phase bit at 0, the first words carry 1; the other set, which
    // the next launch will use, is cleared here as far as the launch before wrote it.
    // Block (16 columns, 8 batch rows) = 512 contiguous bytes, [column / 4][row][4 words]: a warp's load of a block is four
    // full lines, each by eight consecutive lanes.
    const int Hq = (H + 3) & ~3, nq = Hq >> 2;                              // chunks of four units
    const unsigned slot_words = (unsigned)((H + 15) >> 4) * (RG * 128u);
    auto chunk_word = [&](int q, int b) -> unsigned { return ((unsigned)(q >> 2) * RG + (b >> 3)) * 128u + (q & 3) * 32u + (b & 7) * 4u; };
    // (buffers by place in the launch, not by direction: launches that run the directions in turn share them)
    unsigned *xch_d = a.xch + (size_t)a.set * a.set_words + (size_t)(d - a.dir0) * 2 * slot_words;
    for (unsigned i = blockIdx.x * kThreads + tid; i < a.clear_words / 4u; i += gridDim.x * kThreads)
        reinterpret_cast<uint4 *>(a.xch + (size_t)(a.set ^ 1) * a.set_words)[i] = make_uint4(0, 0, 0, 0);
    // weights into tensor memory: warp w writes lane quadrant w % 4, every fourth 8-column piece
    {
        const int row = (warp & 3) * 32 + lane, pieces = a.KH >> 3;
        const uint4 *src = a.wpack[d] + (size_t)cta * pieces * RT + row;
        const uint32_t dst = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int p0 = warp >> 2; p0 < pieces; p0 += 32) {
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = p0 + 4 * i < pieces && row < RT ? ld_nc_u4(src + (size_t)(p0 + 4 * i) * RT) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (p0 + 4 * i < pieces) tmem_st4(dst + (uint32_t)(p0 + 4 * i) * 4u, v[i]);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < tiles * N * 8; i += kThreads) reinterpret_cast<uint4 *>(op)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (PAIR) cluster_sync_all();               // the partner's barriers are initialised before anything reaches them

    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const uint64_t bdesc0 = umma_desc_sw128(base);
    // Polling: of a block a lane takes chunk qq (four columns) of batch row rr; half a warp stores eight rows by 16 bytes,
    // which the swizzle spreads over all banks.
    const int qq = lane >> 3, rr = lane & 7;
    const int q0 = (k_lo >> 2) + warp * 4 + qq;
    const unsigned *src_even = xch_d + (size_t)((k_lo >> 4) + warp) * (RG * 128) + lane * 4, *src_odd = src_even + slot_words;
    constexpr int kSrcGroup = kPollers * RG * 128;                          // words from group to group
    unsigned char *dst0 = op + (warp >> 2) * (N * 128) + rr * 128 + ((((warp & 3) * 32) + qq * 8) ^ (rr << 4));
    constexpr int kDstGroup = kPollers / 4 * N * 128;
    // groups this warp has a piece of, groups this lane has a chunk in, and whether its row of the last row group exists:
    // what does not exist is read as the zeros the buffer holds there, and not waited for
    const int n_warp = warp < kPollers ? (nk16 - warp + kPollers - 1) / kPollers : 0;
    const int n_lane = min(n_warp, (nq - q0 + 4 * kPollers - 1) / (4 * kPollers));
    const bool last_row = B - 8 * (RG - 1) > rr;
    // finishing: TMEM lane quadrant, accumulator row, batch rows [fb0, + RS); of the partner's batch rows [sb0, + RS)
    const int row = (warp & 3) * 32 + lane, sub = warp >> 2, fq = lane & 3;
    const bool mine = row < RT && (!UNITS || (row >= RT / 2) == (rank != 0)), theirs = row < RT && (!UNITS || !mine);
    const int my_lo = UNITS ? 0 : rank * HB, my_n = UNITS ? Bp : rank ? Bp - HB : HB;
    const int other_lo = UNITS ? 0 : HB - my_lo, other_n = UNITS ? Bp : PAIR ? Bp - my_n : 0;
    const bool fin = sub * RS < my_n && __any_sync(0xffffffffu, mine), snd = sub * RS < other_n && __any_sync(0xffffffffu, theirs);
    const int fb0 = my_lo + sub * RS, sb0 = other_lo + sub * RS;
    const int j = (PAIR ? cta & ~1 : cta) * upc + (row >> 2);               // unit of this row
    const bool own = fin && mine && j < Hq, real = own && j < H;
    const float act_k = (fq == 2 ? -2.0f : -1.0f) * 1.4426950408889634f, act_sc = fq == 2 ? 2.0f : 1.0f, act_of = fq == 2 ? -1.0f : 0.0f;
    const uint32_t zs2_remote = PAIR ? map_to_cta(smem_u32(zs2), (uint32_t)(rank ^ 1)) + (uint32_t)(sub * RS * RT + row) * 4u : 0u;
    const uint32_t partial_remote = PAIR ? map_to_cta(smem_u32(partial_bar), (uint32_t)(rank ^ 1)) : 0u;
    const uint32_t abort_remote = PAIR ? map_to_cta(smem_u32(&abort_s), (uint32_t)(rank ^ 1)) : 0u;
    const float *zs2_mine = zs2 + sub * RS * RT + row;
    const size_t state0 = ((size_t)d * a.Bs + a.b0) * H + j;                // element of (pass row 0, unit j) in the state arrays
    // projection terms, outputs: pointers that advance by one timestep per step
    const long long gstep = (long long)D * 4 * H, dir = d ? -1 : 1;
    const long long m0 = (long long)(d ? T - 1 : 0) * a.Bs + a.b0 + fb0;    // row of G of this thread's first batch row
    const float *gp = a.G + m0 * gstep + (long long)d * 4 * H + 4 * (long long)j + fq;
    const int nrow = real ? max(0, min(RS, B - fb0)) : 0;
    const float *gpre = a.G + (m0 + 2 * dir * a.Bs + lane) * gstep + (long long)d * 4 * H + 4 * (long long)(j - (lane >> 2));
    const bool pre = lane < RS && fb0 + lane < B && fin && j - (lane >> 2) < H;
    float *yp = a.y ? a.y + (m0 + fq) * D * H + (long long)d * H + j : nullptr;
    __nv_bfloat16 *xp = a.xb_next ? a.xb_next + (m0 + fq) * a.xb_ld + (long long)d * H + j : nullptr;
    const long long gadv = dir * a.Bs * gstep, yadv = dir * a.Bs * D * H, xadv = dir * a.Bs * a.xb_ld;
    const int ystep = 4 * D * H, xstep = 4 * a.xb_ld;
    unsigned *const out0 = xch_d + chunk_word(j >> 2, fb0 + fq) + (j & 3);
    const int nitem = own ? max(0, min(RS / 4, (B - fb0 - fq + 3) >> 2)) : 0;       // (unit, batch row) items of this thread
    const int npub = (int)blockIdx.x != a.withhold_cta ? nitem : 0, nout = real ? nitem : 0;

    // c of (unit, batch row fb0 + 4 m + fq)
    float c[RS / 4], hn[RS / 4];
#pragma unroll
    for (int m = 0; m < RS / 4; ++m) {
        c[m] = a.c0 && m < nout ? a.c0[state0 + (size_t)(fb0 + 4 * m + fq) * H] : 0.0f;
        hn[m] = 0.0f;
    }

    // outputs of a step: written while the next step's poll is under way
    auto write_outputs = [&]() {
        if (yp) {
#pragma unroll
            for (int m = 0; m < RS / 4; ++m)
                if (m < nout) yp[m * ystep] = hn[m];
            yp += yadv;
        }
        if (xp) {
#pragma unroll
            for (int m = 0; m < RS / 4; ++m)
                if (m < nout) {
                    const __nv_bfloat16 hi = __float2bfloat16_rn(hn[m]);
                    xp[m * xstep] = hi;
                    xp[a.xb_plane + m * xstep] = __float2bfloat16_rn(hn[m] - __bfloat162float(hi));
                }
            xp += xadv;
        }
    };
    // Projection terms of this thread's row, requested between the last poll and the wait for the products, which hides the
    // trip to L2; the lines are requested from HBM two steps ahead.  Requested ahead of the polls, or a whole step ahead,
    // they delayed them: 2.63 -> 3.08 us per step (two directions of 800, 16 rows).
    float g[RS];
    auto load_g = [&](int s) {
#pragma unroll
        for (int i = 0; i < RS; ++i) g[i] = i < nrow ? ld_nc_early(gp + i * gstep) : 0.0f;
        if (a.nsplit > 1) {
            // further planes of a projection split along K: all of them on their way together
            const float *p1 = gp + a.g_split_stride, *p2 = a.nsplit > 2 ? p1 + a.g_split_stride : p1, *p3 = a.nsplit > 3 ? p2 + a.g_split_stride : p1;
            const int n2 = a.nsplit > 2 ? nrow : 0, n3 = a.nsplit > 3 ? nrow : 0;
            constexpr int C = RS < 8 ? RS : 8;
#pragma unroll
            for (int i0 = 0; i0 < RS; i0 += C) {
                float v[C], u[C], w[C];
#pragma unroll
                for (int i = 0; i < C; ++i) {
                    v[i] = i0 + i < nrow ? ld_nc_early(p1 + (i0 + i) * gstep) : 0.0f;
                    u[i] = i0 + i < n2 ? ld_nc_early(p2 + (i0 + i) * gstep) : 0.0f;
                    w[i] = i0 + i < n3 ? ld_nc_early(p3 + (i0 + i) * gstep) : 0.0f;
                }
#pragma unroll
                for (int i = 0; i < C; ++i) g[i0 + i] += (v[i] + u[i]) + w[i];
            }
        }
        if (pre && s + 2 < T) asm volatile("prefetch.global.L2 [%0];" ::"l"(gpre));
        gp += gadv;
        gpre += gadv;
    };
    unsigned t_pub = 0;

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        if (s > 0) write_outputs();
        // (an aborted CTA opens no further phase: the open one never completes, and a second arrival would exceed its count)
        if (PAIR && tid == 0 && !*abort_v) mbar_expect_tx(smem_u32(&partial_bar[s & 1]), (uint32_t)((UNITS ? RT / 2 : RT) * my_n * 4));

        if (warp >= kIssuer && warp < kIssuer + nissue) {
            // ---- products: issuing warp w takes every nissue-th group, one elected thread, an accumulator of its own
            const int w = warp - kIssuer;
            for (int gi = w; gi < ngroups; gi += nissue) {
                bar_sync(kGroupBar + gi, (kPollers + 1) * 32);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int n = min(kPollers, nk16 - gi * kPollers);
                if (elect_one()) {
                    const uint64_t bd = bdesc0 + (uint64_t)(gi * (kDstGroup / 16));
                    const uint32_t ad = tmem + (uint32_t)(gi * kPollers * 8), acc = acc_col + (uint32_t)(w * N);
#pragma unroll
                    for (int k = 0; k < kPollers; ++k)
                        if (k < n)
                            umma_bf16_ta(acc, ad + k * 8, bd + (uint64_t)((k >> 2) * (N * 128 / 16) + (k & 3) * 2), idesc, gi >= nissue || k ? 1u : 0u);
                    if (gi + nissue >= ngroups) umma_commit(smem_u32(&accum_bar));
                }
                __syncwarp();
            }
        } else if (warp < kPollers) {
            // ---- operand: h_{s-1} of this CTA's K range, KI groups at a time
            auto store_piece = [&](unsigned char *dst, uint4 w, bool polled) {
                if (!LSTM_CHECK_INDEX(dst - op + (TERMS - 1) * Bp * 128 + 7, tiles * N * 128, a.status)) return;
                if constexpr (TERMS == 2) {
                    const unsigned keep = polled ? 0xbfffbfffu : 0xffffffffu;
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(__byte_perm(w.x, w.y, 0x7632u) & keep, __byte_perm(w.z, w.w, 0x7632u) & keep);
                    *reinterpret_cast<uint2 *>(dst + Bp * 128) = make_uint2(__byte_perm(w.x, w.y, 0x5410u), __byte_perm(w.z, w.w, 0x5410u));
                } else {
                    if (polled) {
                        w.x &= ~kPhaseBit; w.y &= ~kPhaseBit; w.z &= ~kPhaseBit; w.w &= ~kPhaseBit;
                        auto size = [](unsigned v) { return fabsf(__uint_as_float(v)); };
                        if (fmaxf(fmaxf(size(w.x), size(w.y)), fmaxf(size(w.z), size(w.w))) > kMaskedNan) {
                            if (size(w.x) > kMaskedNan) w.x |= kPhaseBit;
                            if (size(w.y) > kMaskedNan) w.y |= kPhaseBit;
                            if (size(w.z) > kMaskedNan) w.z |= kPhaseBit;
                            if (size(w.w) > kMaskedNan) w.w |= kPhaseBit;
                        }
                    }
                    // each term takes the upper half of what is left, eight bits of it: three hold all 24, nothing is rounded
#pragma unroll
                    for (int t = 0; t < 3; ++t) {
                        *reinterpret_cast<uint2 *>(dst + t * Bp * 128) = make_uint2(__byte_perm(w.x, w.y, 0x7632u), __byte_perm(w.z, w.w, 0x7632u));
                        if (t == 2) break;
                        auto rest = [](unsigned v) { return __float_as_uint(__uint_as_float(v) - __uint_as_float(v & 0xffff0000u)); };
                        w = make_uint4(rest(w.x), rest(w.y), rest(w.z), rest(w.w));
                    }
                }
            };
            auto word_of = [](float h) { return TERMS == 2 ? split_word(h) : __float_as_uint(h); };
            const unsigned phase = word_phase(s - 1);
            const unsigned *src = (s & 1) ? src_even : src_odd;
            if (s == 0 && a.h0) {
                for (int i = 0; i < n_lane; ++i)
                    for (int rg = 0; rg < RG; ++rg)
                        if (rg < RG - 1 || last_row) {
                            const int k = 4 * (q0 + i * 4 * kPollers);
                            const float *hp = a.h0 + ((size_t)d * a.Bs + a.b0 + rg * 8 + rr) * H + k;
                            uint4 v = make_uint4(word_of(hp[0]), 0, 0, 0);
                            if (k + 1 < H) v.y = word_of(hp[1]);
                            if (k + 2 < H) v.z = word_of(hp[2]);
                            if (k + 3 < H) v.w = word_of(hp[3]);
                            store_piece(dst0 + i * kDstGroup + rg * 1024, v, false);
                        }
            }
            if (s > 0) while ((unsigned)clock() - t_pub < kPollDelay) { }
#pragma unroll 1
            for (int i0 = 0; i0 < ngroups; i0 += KI, src += KI * kSrcGroup) {
                uint4 w[KI][RG];
                unsigned char *dst = dst0 + i0 * kDstGroup;
                if (s > 0) {
#pragma unroll
                    for (int i = 0; i < KI; ++i)
                        if (i0 + i < n_warp) {
#pragma unroll
                            for (int rg = 0; rg < RG; ++rg) w[i][rg] = ld_relaxed_v4(src + i * kSrcGroup + rg * 128);
                        }
                }
#pragma unroll
                for (int i = 0; i < KI; ++i)
                    if (i0 + i < ngroups) {
                        if (s > 0 && i0 + i < n_warp) {
                            auto missing = [&]() -> unsigned {          // row groups of this piece that are not here yet
                                unsigned m = 0;
#pragma unroll
                                for (int rg = 0; rg < RG; ++rg)
                                    if (!words_ready(w[i][rg], phase) && (rg < RG - 1 || last_row)) m |= 1u << rg;
                                return i0 + i < n_lane ? m : 0u;
                            };
                            unsigned pending = missing();
                            int polls = 0;
                            long long t_start = 0;
                            while (__any_sync(0xffffffffu, pending)) {
#pragma unroll
                                for (int rg = 0; rg < RG; ++rg)
                                    if (pending & (1u << rg)) w[i][rg] = ld_relaxed_v4(src + i * kSrcGroup + rg * 128);
                                pending = missing();
                                if ((++polls & 15) == 0 || *abort_v) {
                                    const long long now = clock64();
                                    if (t_start == 0) t_start = now;
                                    if (*abort_v) pending = 0;
                                    else if (now - t_start > a.spin_limit || ld_volatile_s32(a.status) != kStatusOk) {
                                        *abort_v = 1;
                                        atomicExch(a.status, kStatusTimeout);
                                        pending = 0;
                                    }
                                }
                            }
#pragma unroll
                            for (int rg = 0; rg < RG; ++rg) store_piece(dst + i * kDstGroup + rg * 1024, w[i][rg], true);
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        bar_arrive(kGroupBar + i0 + i, (kPollers + 1) * 32);
                    }
            }
        }

        // ---- accumulators, partner's partial sums, gates, state
        if (fin || snd) {
            load_g(s);
            mbar_wait(smem_u32(&accum_bar), (uint32_t)s & 1u, abort_v);
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            float z[RS];
            auto read_sums = [&](int b0) {                       // this row's sums for batch rows b0 .. b0 + RS - 1
                const uint32_t ta = acc_col + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)b0;
                float zl[RS];
                if constexpr (TERMS == 3) {                      // the last two terms first: their sum takes the place of the second
                    float zt[RS];
                    tmem_ld<RS>(ta + (uint32_t)Bp, zl);
                    tmem_ld<RS>(ta + (uint32_t)(2 * Bp), zt);
                    if (NACC > 1 && nissue > 1) {
                        float y[RS], yt[RS];
                        tmem_ld<RS>(ta + (uint32_t)(N + Bp), y);
                        tmem_ld<RS>(ta + (uint32_t)(N + 2 * Bp), yt);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < RS; ++i) zl[i] = (zl[i] + y[i]) + (zt[i] + yt[i]);
                        tmem_ld<RS>(ta + (uint32_t)N, y);
                        tmem_ld<RS>(ta, z);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < RS; ++i) z[i] = (z[i] + y[i]) + zl[i];
                    } else {
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < RS; ++i) zl[i] += zt[i];
                        tmem_ld<RS>(ta, z);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int i = 0; i < RS; ++i) z[i] += zl[i];
                    }
                    return;
                }
                tmem_ld<RS>(ta, z);
                tmem_ld<RS>(ta + (uint32_t)Bp, zl);
                if (NACC > 1 && nissue > 1) {
                    float y[RS], yl[RS];
                    tmem_ld<RS>(ta + (uint32_t)N, y);
                    tmem_ld<RS>(ta + (uint32_t)(N + Bp), yl);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < RS; ++i) z[i] = (z[i] + y[i]) + (zl[i] + yl[i]);
                } else {
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < RS; ++i) z[i] += zl[i];
                }
            };
            if (PAIR && snd) {
                read_sums(sb0);
                if (*abort_v) {
                    // gave up: nothing is sent any more, so the partner must not wait for it
                    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(abort_remote), "r"(1) : "memory");
                } else if (theirs) {
                    const uint32_t dst = zs2_remote + (uint32_t)((s & 1) * RT * HB) * 4u, bar = partial_remote + (uint32_t)(s & 1) * 8u;
#pragma unroll
                    for (int i = 0; i < RS; ++i) st_async(dst + (uint32_t)(i * RT) * 4u, z[i], bar);
                }
                __syncwarp();
            }
            if (fin) {
                if (!UNITS || !snd) read_sums(fb0);
                if (PAIR) {
                    mbar_wait(smem_u32(&partial_bar[s & 1]), (uint32_t)(s >> 1) & 1u, abort_v);
                    __syncwarp();
                    if (mine) {
                        const float *zp = zs2_mine + (s & 1) * RT * HB;
#pragma unroll
                        for (int i = 0; i < RS; ++i) z[i] += zp[i * RT];
                    }
                }
#pragma unroll
                for (int i = 0; i < RS; ++i) z[i] = gate_fast(z[i] + g[i], act_k, act_sc, act_of);
                unsigned *dst = out0 + (size_t)(s & 1) * slot_words;
                const unsigned phase_out = word_phase(s);
#pragma unroll
                for (int m = 0; m < RS / 4; ++m) {
                    quad_transpose(z[4 * m], z[4 * m + 1], z[4 * m + 2], z[4 * m + 3], fq);
                    c[m] = fmaf(z[4 * m + 1], c[m], z[4 * m] * z[4 * m + 2]);
                    hn[m] = z[4 * m + 3] * tanh_fast(c[m]);
                    // (fb0 is a multiple of four: of eight where a thread has more than one item)
                    if (m < npub)
                        st_relaxed_u32(dst + (m & 1) * 16 + (m >> 1) * 128,
                                       TERMS == 2 ? pack_word(hn[m], phase_out) : (__float_as_uint(hn[m]) & ~kPhaseBit) | phase_out);
                }
            }
        }
        // Nobody polls or overwrites the operand before the whole CTA has published: early polls of words that are being
        // written pull their lines to and fro between the two halves of the L2, and delay everyone.
        bar_sync(1, kThreads);
        t_pub = (unsigned)clock();
    }
    write_outputs();
#pragma unroll
    for (int m = 0; m < RS / 4; ++m)
        if (m < nout) {
            if (a.hT) a.hT[state0 + (size_t)(fb0 + 4 * m + fq) * H] = hn[m];
            if (a.cT) a.cT[state0 + (size_t)(fb0 + 4 * m + fq) * H] = c[m];
        }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(*abort_v)) {           // one answer for the whole CTA: the partner may raise the flag at any time
        // a wait gave up: products and partial sums may still be in flight; they land within microseconds
        if (tid == 0) atomicExch(a.status, kStatusTimeout);
        const long long t0 = clock64();
        while (clock64() - t0 < 200000) { }
        __syncthreads();
    }
    if (warp == kIssuer) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base_s) : "memory");
    }
    if (PAIR) cluster_sync_all();               // no CTA leaves while its partner may still write into its shared memory
}

typedef void (*KernelFn)(const RecurTcArgs);
template <bool PAIR, int TERMS>
KernelFn pick_p(int rg)
{
    switch (rg) {
        case 1: return recur_tc_kernel<1, PAIR, TERMS>;
        case 2: return recur_tc_kernel<2, PAIR, TERMS>;
        case 3: return recur_tc_kernel<3, PAIR, TERMS>;
        case 4: return recur_tc_kernel<4, PAIR, TERMS>;
        case 5: return recur_tc_kernel<5, PAIR, TERMS>;
        case 6: return recur_tc_kernel<6, PAIR, TERMS>;
        case 7: return recur_tc_kernel<7, PAIR, TERMS>;
        case 8: return recur_tc_kernel<8, PAIR, TERMS>;
        default: return nullptr;
    }
}
KernelFn pick(int rg, bool pair, int terms)
{
    return terms == 3 ? (pair ? pick_p<true, 3>(rg) : pick_p<false, 3>(rg)) : (pair ? pick_p<true, 2>(rg) : pick_p<false, 2>(rg));
}
int groups_of(int rows) { return (rows + 7) / 8; }

cudaLaunchConfig_t config(cudaLaunchAttribute (&attr)[2], int grid, size_t smem, int pair, cudaStream_t st)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = pair ? 2 : 1;
    return cfg;
}

}  // namespace

size_t recur_tc_smem_bytes(int KH, int upc, int rows, int pair, int terms)
{
    const int rg = groups_of(rows);
    return 1024 + (size_t)((KH + 63) / 64) * tc_columns(rg, terms) * 128 + (pair ? (size_t)2 * 8 * upc * tc_rows_of_first(rg, true) * 4 : 0);
}

size_t recur_tc_xch_words(int H, int rows, int dirs) { return (size_t)dirs * 2 * ((H + 15) / 16) * groups_of(rows) * 128; }

// Partition of H units over at most max_cta CTAs, and the most batch rows (<= rows_wanted) a pass can take; false when
// the slice does not fit tensor memory.
bool recur_tc_plan(int H, int max_cta, int rows_wanted, int pair, int terms, size_t max_smem, RecurTcPlan *p)
{
    if (pair && H <= 64) return false;                                  // both halves of K must exist
    int upc = 4, n = 0;
    for (; upc <= 16; upc += 4) {
        n = (H + upc - 1) / upc;
        if (pair) n = (n + 1) / 2 * 2;
        if (n <= max_cta) break;
    }
    if (upc > 16) return false;
    const int KH = ((pair ? (H + 1) / 2 : H) + 15) / 16 * 16;
    for (int rg = groups_of(rows_wanted < kTcMaxRows ? rows_wanted : kTcMaxRows); rg >= 1; --rg) {
        if (KH / 2 + tc_acc_columns(rg, terms) <= 512 && KH <= 16 * kPollers * kMaxGroups && recur_tc_smem_bytes(KH, upc, 8 * rg, pair, terms) <= max_smem) {
            p->upc = upc; p->ncta = n; p->KH = KH; p->pair = pair; p->rows = 8 * rg; p->terms = terms;
            return true;
        }
    }
    return false;
}

cudaError_t recur_tc_prepare(int terms, int max_smem)
{
    for (int rg = 1; rg <= kTcMaxRows / 8; ++rg) {
        for (int pair = 0; pair < 2; ++pair) {
            const cudaError_t e = cudaFuncSetAttribute(pick(rg, pair != 0, terms), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

// Can `grid` CTAs of this kernel be co-resident as clusters of two (pair mode needs every pair on one GPC)?
bool recur_tc_pair_supported(int grid, const RecurTcPlan &p)
{
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = config(attr, grid, recur_tc_smem_bytes(p.KH, p.upc, p.rows, 1, p.terms), 1, nullptr);
    cfg.attrs = attr + 1; cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)pick(groups_of(p.rows), true, p.terms), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters * 2 >= grid;
}

cudaError_t launch_recur_tc(const RecurTcArgs &a, cudaStream_t st)
{
    KernelFn fn = pick(groups_of(a.B), a.pair != 0, a.terms);
    if (!fn) return cudaErrorInvalidValue;
    RecurTcArgs copy = a;
    void *params[] = {&copy};
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = config(attr, a.ncta_dir * (a.ndirs ? a.ndirs : a.D), recur_tc_smem_bytes(a.KH, a.upc, a.B, a.pair, a.terms), a.pair, st);
    return cudaLaunchKernelExC(&cfg, (const void *)fn, params);
}

}  // namespace lstm

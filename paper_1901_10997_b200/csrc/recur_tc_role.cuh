// One CTA of the batched recurrence (recur_tc.cu says what a step does and why it is laid out like this), as a device function:
// recur_tc.cu launches it for one layer, recur_stack.cu for the two layers of a stack side by side.
#pragma once
#include "common.cuh"
#include "device_util.cuh"

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

// Two layers in one launch: the lower layer counts its CTAs that have stored the planes of a chunk of timesteps, the upper one waits for
// the count of CTAs that have stored that chunk's rows of its G.
enum { kTcAlone = 0, kTcLower = 1, kTcUpper = 2 };
struct TcLink {
    int chunk;                  // timesteps of a chunk (the last one may be shorter)
    unsigned *stored;           // kTcLower: [chunk] counts
    const unsigned *ready;      // kTcUpper: [chunk] counts, complete at n_ready
    unsigned n_ready;
};

// waits until *count >= n; false when it gave up (or another role did)
__device__ __forceinline__ bool wait_count(const unsigned *count, unsigned n, volatile int *abort_v, long long spin_limit, int *status)
{
    long long t_start = 0;
    for (int polls = 1;; ++polls) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
        if (v >= n) return true;
        if ((polls & 15) == 0 || *abort_v) {
            if (*abort_v) return false;
            const long long now = clock64();
            if (t_start == 0) t_start = now;
            if (now - t_start > spin_limit || ld_volatile_s32(status) != kStatusOk) break;
        }
    }
    *abort_v = 1;
    atomicExch(status, kStatusTimeout);
    return false;
}
__device__ __forceinline__ void add_count(unsigned *count)
{
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
}

// RG: groups of eight batch rows of a pass; TERMS: bf16 terms of h, two from words {hi | lo}, three from words that are h itself
// MB: blocks of accumulator rows: 128 with their weights in tensor memory, and up to 64 with theirs in shared memory; LINK: place in a stack.
// block: this CTA's place in the group of CTAs that run the layer.
// SPLIT: the projection may come in several planes along K, and few rows: see g below.
template <int RG, bool PAIR, int TERMS, int MB, int LINK, bool SPLIT>
__device__ __forceinline__ void recur_tc_role(const RecurTcArgs &a, int block, const TcLink &link)
{
    static_assert(MB == 1 || (PAIR && tc_columns(RG, TERMS) <= 64), "two blocks: an accumulator and an issuing warp each");
    constexpr int Bp = 8 * RG, N = tc_columns(RG, TERMS), HB = tc_rows_of_first(RG, PAIR), RS = tc_rows_per_thread(HB);
    constexpr bool UNITS = PAIR && RG == 1;
    constexpr int KI = tc_groups_in_flight(RG), NACC = MB == 2 ? 2 : tc_accumulators(RG, TERMS);
    constexpr uint32_t tmem = 0;                                            // all 512 columns are ours: they start at address 0
    constexpr uint32_t acc_col = 512u - (MB == 2 ? 2 * N : tc_acc_columns(RG, TERMS));      // accumulators behind the weights
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long accum_bar, partial_bar[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int H = a.H, B = a.B, T = a.T, D = a.D, upc = a.upc;
    const int d = a.dir0 + block / a.ncta_dir;
    const int cta = block % a.ncta_dir;
    const int rank = PAIR ? (int)cluster_ctarank() : 0;
    const int RT = PAIR ? 8 * upc : 4 * upc;                                // accumulator rows of the tile
    const int k_lo = rank * a.KH, k_n = min(a.KH, H - k_lo);                // this CTA's K range
    const int nk16 = (k_n + 15) >> 4;
    const int ngroups = (nk16 + kPollers - 1) / kPollers;                   // warp w fetches piece w of every group
    const int nissue = MB == 2 ? 2 : min(NACC, ngroups);                    // issuing warps, each with an accumulator

    // shared memory: weight rows from 128 on as tiles of 64 columns [R2 rows][128 bytes, swizzled] (the instruction reads 64 rows of
    // them: what follows, into lanes nobody looks at), operand tiles of 64 columns [N rows][128 bytes, swizzled], then the
    // partner's partial sums [2][HB][RT].  Cycles an instruction at N = 48: 128 rows from tensor memory 25, from shared memory 45, 64
    // rows from shared memory 32.
    const int tiles = (a.KH + 63) >> 6, R2 = MB == 2 ? RT - 128 : 0;
    const uint32_t base2 = (smem_u32(smem_raw) + 1023u) & ~1023u, base = base2 + (uint32_t)(tiles * R2 * 128);
    unsigned char *op = smem_raw + (base - smem_u32(smem_raw));
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
    for (unsigned i = blockIdx.x * kThreads + tid; LINK == kTcAlone && i < a.clear_words / 4u; i += gridDim.x * kThreads)
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
        if constexpr (MB == 2)
            for (int i = tid; i < pieces * R2; i += kThreads) {
                const int p = i / R2, r = i - p * R2;
                *reinterpret_cast<uint4 *>(smem_raw + (base2 - smem_u32(smem_raw)) + (size_t)(p >> 3) * R2 * 128 + r * 128 + (((p & 7) ^ (r & 7)) << 4)) =
                    ld_nc_u4(a.wpack[d] + ((size_t)cta * pieces + p) * RT + 128 + r);
            }
    }
    for (int i = tid; i < tiles * N * 8; i += kThreads) reinterpret_cast<uint4 *>(op)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (PAIR) cluster_sync_all();               // the partner's barriers are initialised before anything reaches them

    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    const uint32_t idesc2 = idesc - ((uint32_t)(64 >> 4) << 24);             // 64 rows
    const uint64_t bdesc0 = umma_desc_sw128(base), adesc0 = umma_desc_sw128(base2);
    // Polling: of a block a lane takes chunk qq (four columns) of batch row rr; half a warp stores eight rows by 16 bytes,
    // which the swizzle spreads over all banks.
    const int qq = lane >> 3, rr = lane & 7;
    const int q0 = (k_lo >> 2) + warp * 4 + qq;
    const unsigned *src_even = xch_d + (size_t)((k_lo >> 4) + warp) * (RG * 128) + lane * 4, *src_odd = src_even + slot_words;
    constexpr int kSrcGroup = kPollers * RG * 128;                          // words from group to group
    unsigned char *dst0 = op + (warp >> 2) * (N * 128) + rr * 128 + ((((warp & 3) * 32) + qq * 8) ^ (rr << 4));
    constexpr int kDstGroup = kPollers / 4 * N * 128;
    constexpr int kGroupThreads = (kPollers + MB) * 32;                     // of a group's barrier: polling warps and whoever multiplies it
    // groups this warp has a piece of, groups this lane has a chunk in, and whether its row of the last row group exists:
    // what does not exist is read as the zeros the buffer holds there, and not waited for
    const int n_warp = warp < kPollers ? (nk16 - warp + kPollers - 1) / kPollers : 0;
    const int n_lane = min(n_warp, (nq - q0 + 4 * kPollers - 1) / (4 * kPollers));
    const bool last_row = B - 8 * (RG - 1) > rr;
    // finishing: TMEM lane quadrant, accumulator row (of the first block; of the second one, whose 64 rows are sixteen lanes of each
    // quadrant, it is drow rows, dj units on), batch rows [fb0, + RS); of the partner's batch rows [sb0, + RS)
    const int row = (warp & 3) * 32 + lane, sub = warp >> 2, fq = lane & 3;
    const int drow = 128 - 16 * (warp & 3), dj = 32 - 4 * (warp & 3);
    auto exists = [&](int k) { return k == 0 ? row < RT : lane < 16 && row + drow < RT; };
    auto is_mine = [&](int k) { return exists(k) && (!UNITS || (row + k * drow >= RT / 2) == (rank != 0)); };
    auto is_theirs = [&](int k) { return exists(k) && (!UNITS || !is_mine(k)); };
    const int my_lo = UNITS ? 0 : rank * HB, my_n = UNITS ? Bp : rank ? Bp - HB : HB;
    const int other_lo = UNITS ? 0 : HB - my_lo, other_n = UNITS ? Bp : PAIR ? Bp - my_n : 0;
    const bool fin = sub * RS < my_n && __any_sync(0xffffffffu, is_mine(0) || (MB == 2 && is_mine(1)));
    const bool snd = sub * RS < other_n && __any_sync(0xffffffffu, is_theirs(0) || (MB == 2 && is_theirs(1)));
    const int fb0 = my_lo + sub * RS, sb0 = other_lo + sub * RS;
    const int j = (PAIR ? cta & ~1 : cta) * upc + (row >> 2);               // unit of this row
    auto is_own = [&](int k) { return fin && is_mine(k) && j + k * dj < Hq; };
    auto is_real = [&](int k) { return is_own(k) && j + k * dj < H; };
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
    const float *gpre = a.G + (m0 + 2 * dir * a.Bs + lane) * gstep + (long long)d * 4 * H + 4 * (long long)(j - (lane >> 2));
    const bool pre = LINK != kTcUpper && lane < RS && fb0 + lane < B && fin && j - (lane >> 2) < H;
    const bool pre2 = MB == 2 && j - (lane >> 2) + dj < H;                  // (the second block's units of the last pair may not exist)
    float *yp = a.y ? a.y + (m0 + fq) * D * H + (long long)d * H + j : nullptr;
    __nv_bfloat16 *xp = a.xb_next ? a.xb_next + (m0 + fq) * a.xb_ld + (long long)d * H + j : nullptr;
    const long long gadv = dir * a.Bs * gstep, yadv = dir * a.Bs * D * H, xadv = dir * a.Bs * a.xb_ld;
    const int ystep = 4 * D * H, xstep = 4 * a.xb_ld;
    unsigned *const out0 = xch_d + chunk_word(j >> 2, fb0 + fq) + (j & 3);
    unsigned *const out1 = MB == 2 ? xch_d + chunk_word((j + dj) >> 2, fb0 + fq) + (j & 3) : nullptr;      // (dj: whole chunks)
    int nrow[MB], npub[MB], nout[MB];                                       // rows of G, words, outputs of this thread
#pragma unroll
    for (int k = 0; k < MB; ++k) {
        const int nitem = is_own(k) ? max(0, min(RS / 4, (B - fb0 - fq + 3) >> 2)) : 0;       // (unit, batch row) items
        nrow[k] = is_real(k) ? max(0, min(RS, B - fb0)) : 0;
        npub[k] = (int)blockIdx.x != a.withhold_cta ? nitem : 0;
        nout[k] = is_real(k) ? nitem : 0;
    }

    // c of (unit, batch row fb0 + 4 m + fq)
    float c[MB][RS / 4], hn[MB][RS / 4];
#pragma unroll
    for (int k = 0; k < MB; ++k)
#pragma unroll
        for (int m = 0; m < RS / 4; ++m) {
            c[k][m] = a.c0 && m < nout[k] ? a.c0[state0 + k * dj + (size_t)(fb0 + 4 * m + fq) * H] : 0.0f;
            hn[k][m] = 0.0f;
        }

    // outputs of a step: written while the next step's poll is under way
    auto write_outputs = [&]() {
        if (yp) {
#pragma unroll
            for (int k = 0; k < MB; ++k)
#pragma unroll
                for (int m = 0; m < RS / 4; ++m)
                    if (m < nout[k]) yp[m * ystep + k * dj] = hn[k][m];
            yp += yadv;
        }
        if (xp) {
#pragma unroll
            for (int k = 0; k < MB; ++k)
#pragma unroll
                for (int m = 0; m < RS / 4; ++m)
                    if (m < nout[k]) {
                        const __nv_bfloat16 hi = __float2bfloat16_rn(hn[k][m]);
                        xp[m * xstep + k * dj] = hi;
                        xp[a.xb_plane + m * xstep + k * dj] = __float2bfloat16_rn(hn[k][m] - __bfloat162float(hi));
                    }
            xp += xadv;
        }
    };
    // Projection terms of this thread's row, requested between the last poll and the wait for the products, which hides the
    // trip to L2; the lines are requested from HBM two steps ahead.  Requested ahead of the polls, or a whole step ahead,
    // they delayed them: 2.63 -> 3.08 us per step (two directions of 800, 16 rows).
    // SPLIT: the further planes of a projection split along K are added behind the products, which take less time than the loads (2 x 517,
    // 3 rows: 1020 of 4600 clocks a step stood here).  A build of its own: with one plane the registers cost more (pruned 2 x
    // 1500, 16 rows 243 -> 257 us), and with more rows the products hide the sum.
    constexpr bool LATE = SPLIT && RS == 4 && LINK != kTcUpper;
    constexpr bool PLANES = (SPLIT || RG > 2) && LINK != kTcUpper;          // up to two row groups there is a build for one plane and one for several
    float g[MB][RS], gx[MB][LATE ? 3 : 1][RS];
#pragma unroll
    for (int k = 0; k < MB; ++k)
#pragma unroll
        for (int p = 0; p < (LATE ? 3 : 1); ++p)
#pragma unroll
            for (int i = 0; i < RS; ++i) gx[k][p][i] = 0.0f;
    int chunk_end = 0;                          // kTcUpper: first step whose rows of G have not been waited for
    auto load_g = [&](int s) {
        if constexpr (LINK == kTcUpper) {
            if (s == chunk_end) {
                if (lane == 0) wait_count(link.ready + s / link.chunk, link.n_ready, abort_v, a.spin_limit, a.status);
                __syncwarp();
                chunk_end += link.chunk;
            }
        }
#pragma unroll
        for (int k = 0; k < MB; ++k)
#pragma unroll
            for (int i = 0; i < RS; ++i)
                g[k][i] = i < nrow[k] ? (LINK == kTcUpper ? __uint_as_float(ld_relaxed_u32(reinterpret_cast<const unsigned *>(gp + i * gstep + 4 * k * dj)))
                                                          : ld_nc_early(gp + i * gstep + 4 * k * dj)) : 0.0f;
        if constexpr (PLANES) if (a.nsplit > 1) {
            // further planes of a projection split along K: all of them on their way together
            const float *p1 = gp + a.g_split_stride, *p2 = a.nsplit > 2 ? p1 + a.g_split_stride : p1, *p3 = a.nsplit > 3 ? p2 + a.g_split_stride : p1;
            constexpr int C = RS < 8 ? RS : 8;
#pragma unroll
            for (int k = 0; k < MB; ++k) {
                const int n2 = a.nsplit > 2 ? nrow[k] : 0, n3 = a.nsplit > 3 ? nrow[k] : 0;
#pragma unroll
                for (int i0 = 0; i0 < RS; i0 += C) {
                    float v[C], u[C], w[C];
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        v[i] = i0 + i < nrow[k] ? ld_nc_early(p1 + (i0 + i) * gstep + 4 * k * dj) : 0.0f;
                        u[i] = i0 + i < n2 ? ld_nc_early(p2 + (i0 + i) * gstep + 4 * k * dj) : 0.0f;
                        w[i] = i0 + i < n3 ? ld_nc_early(p3 + (i0 + i) * gstep + 4 * k * dj) : 0.0f;
                    }
#pragma unroll
                    for (int i = 0; i < C; ++i) {
                        if constexpr (LATE) { gx[k][0][i0 + i] = v[i]; gx[k][1][i0 + i] = u[i]; gx[k][2][i0 + i] = w[i]; }
                        else g[k][i0 + i] += (v[i] + u[i]) + w[i];
                    }
                }
            }
        }
        if (pre && s + 2 < T) {
            if (LSTM_CHECK_INDEX(gpre - a.G, (long long)T * a.Bs * gstep, a.status)) asm volatile("prefetch.global.L2 [%0];" ::"l"(gpre));
            if (pre2 && LSTM_CHECK_INDEX(gpre + 4 * dj - a.G, (long long)T * a.Bs * gstep, a.status))
                asm volatile("prefetch.global.L2 [%0];" ::"l"(gpre + 4 * dj));
        }
        gp += gadv;
        gpre += gadv;
    };
    unsigned t_pub = 0;
    int flush_at = link.chunk - 1;              // kTcLower: last step of the current chunk
    bool flushed = false;                       // the last step's outputs have been stored already

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        if (s > 0 && !(LINK == kTcLower && flushed)) write_outputs();
        flushed = false;
        // (an aborted CTA opens no further phase: the open one never completes, and a second arrival would exceed its count)
        if (PAIR && tid == 0 && !*abort_v) mbar_expect_tx(smem_u32(&partial_bar[s & 1]), (uint32_t)((UNITS ? RT / 2 : RT) * my_n * 4));

        if (warp >= kIssuer && warp < kIssuer + nissue) {
            // ---- products: issuing warp w takes every nissue-th group, one elected thread, an accumulator of its own
            // (two blocks: issuing warp w takes block w of every group)
            const int w = warp - kIssuer;
            for (int gi = MB == 2 ? 0 : w; gi < ngroups; gi += MB == 2 ? 1 : nissue) {
                bar_sync(kGroupBar + gi, kGroupThreads);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int n = min(kPollers, nk16 - gi * kPollers);
                if (elect_one()) {
                    const uint64_t bd = bdesc0 + (uint64_t)(gi * (kDstGroup / 16));
                    const uint32_t acc = acc_col + (uint32_t)(w * N);
                    if (MB == 2 && w == 1) {
                        const uint64_t ad = adesc0 + (uint64_t)(gi * (kPollers / 4) * R2 * 8);
#pragma unroll
                        for (int k = 0; k < kPollers; ++k)
                            if (k < n)
                                umma_bf16(acc, ad + (uint64_t)((k >> 2) * R2 * 8 + (k & 3) * 2), bd + (uint64_t)((k >> 2) * (N * 128 / 16) + (k & 3) * 2), idesc2, gi || k ? 1u : 0u);
                    } else {
                        const uint32_t ad = tmem + (uint32_t)(gi * kPollers * 8);
#pragma unroll
                        for (int k = 0; k < kPollers; ++k)
                            if (k < n)
                                umma_bf16_ta(acc, ad + k * 8, bd + (uint64_t)((k >> 2) * (N * 128 / 16) + (k & 3) * 2), idesc, (MB == 2 ? gi > 0 : gi >= nissue) || k ? 1u : 0u);
                    }
                    if (gi + (MB == 2 ? 1 : nissue) >= ngroups) umma_commit(smem_u32(&accum_bar));
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
                        bar_arrive(kGroupBar + i0 + i, kGroupThreads);
                    }
            }
        }

        // ---- accumulators, partner's partial sums, gates, state
        if (fin || snd) {
            load_g(s);
            mbar_wait(smem_u32(&accum_bar), (uint32_t)s & 1u, abort_v);
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            auto read_sums = [&](int b0, int k, float (&z)[RS]) {        // this row's sums for batch rows b0 .. b0 + RS - 1
                const uint32_t ta = acc_col + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b0 + (MB == 2 ? k * N : 0));
                float zl[RS];
                if constexpr (TERMS == 3) {                      // the last two terms first: their sum takes the place of the second
                    float zt[RS];
                    tmem_ld<RS>(ta + (uint32_t)Bp, zl);
                    tmem_ld<RS>(ta + (uint32_t)(2 * Bp), zt);
                    if (MB == 1 && NACC > 1 && nissue > 1) {
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
                if (MB == 1 && NACC > 1 && nissue > 1) {
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
            float z[MB][RS];
            if (PAIR && snd) {
#pragma unroll
                for (int k = 0; k < MB; ++k) {
                    read_sums(sb0, k, z[k]);
                    if (*abort_v) {
                        // gave up: nothing is sent any more, so the partner must not wait for it
                        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(abort_remote), "r"(1) : "memory");
                    } else if (is_theirs(k)) {
                        const uint32_t dst = zs2_remote + (uint32_t)((s & 1) * RT * HB + k * drow) * 4u, bar = partial_remote + (uint32_t)(s & 1) * 8u;
#pragma unroll
                        for (int i = 0; i < RS; ++i) st_async(dst + (uint32_t)(i * RT) * 4u, z[k][i], bar);
                    }
                    __syncwarp();
                }
            }
            if (fin) {
                if (!UNITS || !snd || MB == 2) {
#pragma unroll
                    for (int k = 0; k < MB; ++k) read_sums(fb0, k, z[k]);
                }
                if (PAIR) {
                    mbar_wait(smem_u32(&partial_bar[s & 1]), (uint32_t)(s >> 1) & 1u, abort_v);
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < MB; ++k)
                        if (is_mine(k)) {
                            const float *zp = zs2_mine + (s & 1) * RT * HB + k * drow;
#pragma unroll
                            for (int i = 0; i < RS; ++i) z[k][i] += zp[i * RT];
                        }
                }
                const unsigned phase_out = word_phase(s);
#pragma unroll
                for (int k = 0; k < MB; ++k) {
#pragma unroll
                    for (int i = 0; i < RS; ++i) {
                        if constexpr (LATE) g[k][i] += (gx[k][0][i] + gx[k][1][i]) + gx[k][2][i];
                        z[k][i] = gate_fast(z[k][i] + g[k][i], act_k, act_sc, act_of);
                    }
                    unsigned *dst = (MB == 2 && k ? out1 : out0) + (size_t)(s & 1) * slot_words;
#pragma unroll
                    for (int m = 0; m < RS / 4; ++m) {
                        quad_transpose(z[k][4 * m], z[k][4 * m + 1], z[k][4 * m + 2], z[k][4 * m + 3], fq);
                        c[k][m] = fmaf(z[k][4 * m + 1], c[k][m], z[k][4 * m] * z[k][4 * m + 2]);
                        hn[k][m] = z[k][4 * m + 3] * tanh_fast(c[k][m]);
                        // (fb0 is a multiple of four: of eight where a thread has more than one item)
                        if (m < npub[k])
                            st_relaxed_u32(dst + (m & 1) * 16 + (m >> 1) * 128,
                                           TERMS == 2 ? pack_word(hn[k][m], phase_out) : (__float_as_uint(hn[k][m]) & ~kPhaseBit) | phase_out);
                    }
                }
            }
        }
        if constexpr (LINK == kTcLower) {
            flushed = s == flush_at || s == T - 1;
            if (flushed) {                      // the planes of a chunk: stored before the CTA is counted, readable by tensor copies
                write_outputs();
                asm volatile("fence.proxy.async;" ::: "memory");
            }
        }
        // Nobody polls or overwrites the operand before the whole CTA has published: early polls of words that are being
        // written pull their lines to and fro between the two halves of the L2, and delay everyone.
        bar_sync(1, kThreads);
        t_pub = (unsigned)clock();
        if constexpr (LINK == kTcLower) {
            if (flushed && tid == 0) add_count(link.stored + s / link.chunk);
            if (s == flush_at) flush_at += link.chunk;
        }
    }
    if (!(LINK == kTcLower && flushed)) write_outputs();
#pragma unroll
    for (int k = 0; k < MB; ++k)
#pragma unroll
        for (int m = 0; m < RS / 4; ++m)
            if (m < nout[k]) {
                if (a.hT) a.hT[state0 + k * dj + (size_t)(fb0 + 4 * m + fq) * H] = hn[k][m];
                if (a.cT) a.cT[state0 + k * dj + (size_t)(fb0 + 4 * m + fq) * H] = c[k][m];
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

}  // namespace
}  // namespace lstm

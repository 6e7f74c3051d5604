// Recurrent kernel of the H-LSTM cell for bf16 weights: the paper's Section 4 cell equations with ONE
// hidden layer (linear map + ReLU) inside each gate.  Per step, for gate q in {i,f,g,o}:
//     r_q = relu(P[t]_q + Uh_q h_{t-1})          P[t] = a + Ux x_t, the input half, computed beforehand
//     z_q = b_q + W_q r_q
//     i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c_t = f c_{t-1} + i g;  h_t = o tanh(c_t)
//
// One cooperative launch per layer and pass of up to kHtRows batch rows.  The weights stay on-chip as operand-A fragments
// of mma.m16n8k16; a step has two exchanges (r, then h) and two products.  What makes batches cheap is that every row tile
// is sixteen units of ONE gate, so the eight operand-B columns are eight batch rows (two instructions a tile, bf16 hi and
// lo) and nothing is multiplied for a gate it does not belong to:
//   pass 1: a CTA owns N1 tiles of the 4 x ceil(Hh / 16) hidden tiles; its sixteen warps split K = H, fragments in
//           REGISTERS; the warps' partial sums meet in shared memory; relu; the tile's r values are published;
//   pass 2: a CTA owns sixteen cell units, all four gates; four warps per gate split K = Hh, fragments in SHARED memory;
//           gate functions, c/h update, h is published.
// Values travel as 32-bit words {bf16 hi | bf16 lo} with a phase bit (device_util.cuh; r >= 0, so its phase is the sign
// bit of hi).  A block of sixteen units x eight batch rows is 512 contiguous bytes in operand-B order with ONE writer: a
// lane's 16-byte load is its fragment, nothing is staged or converted.
// Measured (one layer 1500 -> 1200, Hh = 320, T = 70, 16 rows, projection included): 354 us per call against 3825 us for the
// kernel that runs the batch rows one after the other (hlstm_mma.cu, which still serves one row, for which it is the faster one,
// and slices that do not fit here).
// Every wait is bounded; on expiry the CTA records a timeout status, stops waiting and runs to the end.
#include "common.cuh"
#include "device_util.cuh"

#include <algorithm>

namespace lstm {
namespace {

constexpr int kThreads = kHtThreads, kWarps = kThreads / 32;
constexpr int kPitch = 20;                     // floats between the batch rows of a tile's partial sums: no bank conflicts
constexpr int kTileRed = 8 * kPitch;           // partial sums of 16 rows x 8 batch rows
constexpr unsigned kRPhase = 0x80000000u;

__device__ __forceinline__ bool ready(const uint4 &w, unsigned phase, unsigned bit)
{
    return (((w.x ^ phase) | (w.y ^ phase) | (w.z ^ phase) | (w.w ^ phase)) & bit) == 0;
}

// N1: hidden tiles per CTA; KT: column tiles of h per warp; MODE: 0 up to four batch rows, hi and lo planes in adjacent
// operand-B columns; 1 row groups of eight one after the other; 2 two row groups together.
template <int N1, int KT, int MODE>
__global__ void __launch_bounds__(kThreads, 1) hlstm_tile_kernel(const HlstmTileArgs a)
{
    constexpr int RGS = MODE == 2 ? 2 : 1;
    constexpr int NF1 = (N1 * RGS + 3) / 4;            // r items per thread and sub-pass
    constexpr int KB = MODE == 2 || N1 * KT > 12 ? 6 : 12;             // pass 2: column tiles in flight
    // pass 2: the weights of a batch of tiles out of shared memory ahead of its words, where row groups take turns beside large
    // fragments (us per call, T = 35: 1500, Hh = 1500, 12 rows 620 -> 552; 1400, Hh = 1200, 16 rows 582 -> 533; elsewhere the registers
    // are not there: MODE 0 298 -> 308, and spills with twelve tiles in flight)
    constexpr bool kAhead = MODE == 1 && N1 * KT > 12;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int abort_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, tig = lane & 3;
    const int H = a.H, Hh = a.Hh, B = a.B, T = a.T, D = a.D;
    const int d = blockIdx.x / a.ncta_dir, cta = blockIdx.x % a.ncta_dir;
    const int mth = (Hh + 15) >> 4, uth = (H + 15) >> 4;        // tiles of a gate's hidden layer; of the cell units
    const int t0 = cta * N1, nt = max(0, min(N1, 4 * mth - t0));
    const bool has2 = cta < uth;
    const int KT2 = (mth + 3) >> 2, q2 = warp >> 2, kq = warp & 3;
    const int nsub = (B + 8 * RGS - 1) / (8 * RGS);

    uint4 *A2 = reinterpret_cast<uint4 *>(smem);                                    // [16 warps][KT2][32]
    float *red = reinterpret_cast<float *>(A2 + (size_t)kWarps * KT2 * 32);         // pass 1 [16][N1][RGS], pass 2 [16][RGS] tiles of sums
    float *c_s = red + kWarps * N1 * RGS * kTileRed;                                // [B][16]
    LSTM_CHECK_SMEM_END(reinterpret_cast<unsigned char *>(c_s + 16 * B) - smem, a.status);

    // exchange words: [set][D][slot][tile][2 row groups][128]; the other set is cleared for the next launch
    const unsigned hslot = (unsigned)uth * 256u, rslot = (unsigned)mth * 1024u;
    unsigned *hx = a.hx + ((size_t)a.set * D + d) * 2 * hslot, *rx = a.rx + ((size_t)a.set * D + d) * 2 * rslot;
    {
        unsigned *ho = a.hx + ((size_t)(a.set ^ 1) * D + d) * 2 * hslot, *ro = a.rx + ((size_t)(a.set ^ 1) * D + d) * 2 * rslot;
        for (int i = tid; i < 512; i += kThreads)
            if (has2) ho[(size_t)(i >> 8) * hslot + cta * 256 + (i & 255)] = 0u;
        for (int i = tid; i < 512 * nt; i += kThreads) ro[(size_t)(i & 1) * rslot + t0 * 256 + (i >> 1)] = 0u;
    }
    uint4 areg[KT][N1];
    {
        const uint4 *src = a.frag1[d] + ((size_t)(cta * kWarps + warp) * KT * N1) * 32 + lane;
#pragma unroll
        for (int i = 0; i < KT; ++i)
#pragma unroll
            for (int n = 0; n < N1; ++n) areg[i][n] = n < nt ? ld_nc_u4(src + (size_t)(i * N1 + n) * 32) : make_uint4(0, 0, 0, 0);
    }
    if (has2) {
        const uint4 *src = a.frag2[d] + (size_t)cta * kWarps * KT2 * 32;
        for (int i = tid; i < kWarps * KT2 * 32; i += kThreads) A2[i] = __ldg(src + i);
    }
    for (int i = tid; i < 16 * B; i += kThreads) {
        const int b = i >> 4, u = cta * 16 + (i & 15);
        c_s[i] = a.c0 && has2 && u < H ? a.c0[((size_t)d * a.Bs + a.b0 + b) * H + u] : 0.0f;
    }
    if (tid == 0) abort_s = 0;
    __syncthreads();
    volatile int *abort_v = &abort_s;
    const bool publish = (int)blockIdx.x != a.withhold_cta;

    const int k_tiles = max(0, min(KT, uth - warp * KT));                            // this warp's column tiles, pass 1
    const int m_tiles = max(0, min(KT2, mth - kq * KT2));                            // ... pass 2
    const int lane_row = MODE == 0 ? g >> 1 : g;                                     // batch row (of a row group) of this lane's column
    const int lane_word = MODE == 0 ? ((g >> 1) * 4 + tig) * 4 : lane * 4;
    const unsigned plane = MODE == 0 && (g & 1) ? 0x5410u : 0x7632u;

    // finishing items of this thread: pass 1 (tile n, row group rg, batch row b, row), pass 2 the same without the tile
    const int frow = tid & 15, fb = (tid >> 4) & 7, frg = (tid >> 7) & (RGS - 1);
    const bool fin2 = has2 && tid < 128 * RGS;
    const int u2 = cta * 16 + frow;
    float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (fin2 && u2 < H)
        for (int q = 0; q < 4; ++q) bias[q] = a.bias_out[((size_t)d * H + u2) * 4 + q];
    const long long grow = (long long)D * 4 * Hh;                                    // floats of G per batch row
    const float *gcol[NF1];
    bool gok[NF1];
    int rword[NF1], ritem[NF1];
#pragma unroll
    for (int f = 0; f < NF1; ++f) {
        const int i = tid + f * kThreads, n = (i >> 7) / RGS, tile = t0 + n;
        const int q = tile / mth, m = (tile - q * mth) * 16 + frow;
        gok[f] = n < nt && m < Hh;
        gcol[f] = a.G + (long long)d * 4 * Hh + 4 * (long long)m + q;
        rword[f] = n < nt ? tile * 256 + (i & 127) : -1;
        ritem[f] = ((n * RGS + frg) * 8 + fb) * kPitch + frow;
    }

    // polls w[i][rg] = the lane's 16 bytes of tile i, row group rg0 + rg (`src`: tile 0), waiting for `phase` in `bit`
    // (`base`, `words`: the exchange words that src lies in)
    auto fetch = [&](auto &w, const unsigned *src, const unsigned *base, unsigned words, int tiles, int rg0, unsigned phase, unsigned bit) {
        constexpr int NT = sizeof(w) / sizeof(w[0]);
        unsigned pending = 0;
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int rg = 0; rg < RGS; ++rg) {
                w[i][rg] = make_uint4(0, 0, 0, 0);
                if (i < tiles && (rg0 + rg) * 8 + lane_row < B) pending |= 1u << (i * RGS + rg);
            }
        if (*abort_v) pending = 0;
        int polls = 0;
        long long t_start = 0;
        while (pending) {
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
                for (int rg = 0; rg < RGS; ++rg)
                    if ((pending & (1u << (i * RGS + rg))) && LSTM_CHECK_INDEX(src - base + i * 256 + (rg0 + rg) * 128 + 3, words, a.status))
                        w[i][rg] = ld_relaxed_v4(src + i * 256 + (rg0 + rg) * 128);
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
                for (int rg = 0; rg < RGS; ++rg)
                    if ((pending & (1u << (i * RGS + rg))) && ready(w[i][rg], phase, bit)) pending &= ~(1u << (i * RGS + rg));
            if (pending && ((++polls & 15) == 0)) {
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
        __syncwarp();
    };
    auto multiply = [&](float (&acc)[4], const uint4 &af, const uint4 &w, unsigned keep) {
        if (MODE == 0) {
            const unsigned m = (g & 1) ? 0xffffffffu : keep;
            mma_bf16(acc, af, __byte_perm(w.x, w.y, plane) & m, __byte_perm(w.z, w.w, plane) & m);
        } else {
            mma_bf16(acc, af, __byte_perm(w.x, w.y, 0x7632u) & keep, __byte_perm(w.z, w.w, 0x7632u) & keep);
            mma_bf16(acc, af, __byte_perm(w.x, w.y, 0x5410u), __byte_perm(w.z, w.w, 0x5410u));
        }
    };
    auto leave_sums = [&](float *dst, const float (&acc)[4]) {
        if (!LSTM_CHECK_INDEX(dst - red + (MODE == 0 ? 3 : 7) * kPitch + 15, c_s - red, a.status)) return;
        if (MODE == 0) {
            dst[tig * kPitch + g] = acc[0] + acc[1];
            dst[tig * kPitch + g + 8] = acc[2] + acc[3];
        } else {
            dst[2 * tig * kPitch + g] = acc[0];
            dst[(2 * tig + 1) * kPitch + g] = acc[1];
            dst[2 * tig * kPitch + g + 8] = acc[2];
            dst[(2 * tig + 1) * kPitch + g + 8] = acc[3];
        }
    };

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        const int t = d ? (T - 1 - s) : s;
        const unsigned h_phase = word_phase(s - 1), r_phase = word_phase(s) << 1;     // bit 30 -> bit 31
        // ---------------- pass 1: r = relu(P[t] + Uh h_{t-1})
#pragma unroll 1
        for (int sub = 0; sub < nsub; ++sub) {
            const int rg0 = sub * RGS;
            float gv[NF1];
#pragma unroll
            for (int f = 0; f < NF1; ++f) {
                const int b = (rg0 + frg) * 8 + fb;
                gv[f] = 0.0f;
                if (gok[f] && b < B) {
                    const float *gp = gcol[f] + ((long long)t * a.Bs + a.b0 + b) * grow;
                    gv[f] = ld_nc_early(gp);
                    for (int sp = 1; sp < a.nsplit; ++sp) gv[f] += ld_nc_early(gp + sp * a.g_split_stride);
                }
            }
            if (nt > 0) {
                uint4 w[KT][RGS];
                if (s == 0) {
#pragma unroll
                    for (int i = 0; i < KT; ++i)
#pragma unroll
                        for (int rg = 0; rg < RGS; ++rg) {
                            const int b = (rg0 + rg) * 8 + lane_row, k = (warp * KT + i) * 16 + 4 * tig;
                            w[i][rg] = make_uint4(0, 0, 0, 0);
                            if (a.h0 && b < B && k < H) {
                                const float *hp = a.h0 + ((size_t)d * a.Bs + a.b0 + b) * H + k;
                                w[i][rg].x = split_word(hp[0]);
                                if (k + 1 < H) w[i][rg].y = split_word(hp[1]);
                                if (k + 2 < H) w[i][rg].z = split_word(hp[2]);
                                if (k + 3 < H) w[i][rg].w = split_word(hp[3]);
                            }
                        }
                    __syncwarp();
                } else {
                    fetch(w, hx + (size_t)((s - 1) & 1) * hslot + warp * KT * 256 + lane_word, hx, 2 * hslot, k_tiles, rg0, h_phase, kPhaseBit);
                }
                const unsigned keep = s == 0 ? 0xffffffffu : 0xbfffbfffu;
                float acc[N1][RGS][4];
#pragma unroll
                for (int n = 0; n < N1; ++n)
#pragma unroll
                    for (int rg = 0; rg < RGS; ++rg)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[n][rg][e] = 0.0f;
#pragma unroll
                for (int i = 0; i < KT; ++i)
#pragma unroll
                    for (int rg = 0; rg < RGS; ++rg)
#pragma unroll
                        for (int n = 0; n < N1; ++n) multiply(acc[n][rg], areg[i][n], w[i][rg], keep);
#pragma unroll
                for (int n = 0; n < N1; ++n)
#pragma unroll
                    for (int rg = 0; rg < RGS; ++rg) leave_sums(red + ((warp * N1 + n) * RGS + rg) * kTileRed, acc[n][rg]);
            }
            __syncthreads();
#pragma unroll
            for (int f = 0; f < NF1; ++f) {
                const int b = (rg0 + frg) * 8 + fb;
                if (rword[f] >= 0 && b < B) {
                    const float *rp = red + ritem[f];
                    float p[4];
#pragma unroll
                    for (int w4 = 0; w4 < 4; ++w4)
                        p[w4] = (rp[w4 * N1 * RGS * kTileRed] + rp[(w4 + 4) * N1 * RGS * kTileRed]) +
                                (rp[(w4 + 8) * N1 * RGS * kTileRed] + rp[(w4 + 12) * N1 * RGS * kTileRed]);
                    const float r = fmaxf(((p[0] + p[1]) + (p[2] + p[3])) + gv[f], 0.0f);
                    if (publish && LSTM_CHECK_INDEX((size_t)(s & 1) * rslot + rword[f] + (rg0 + frg) * 128, 2 * rslot, a.status))
                        st_relaxed_u32(rx + (size_t)(s & 1) * rslot + rword[f] + (rg0 + frg) * 128, (split_word(r) & ~kRPhase) | r_phase);
                }
            }
            __syncthreads();                // nobody polls before the CTA has published, and the sums are free again
        }
        // ---------------- pass 2: gates
#pragma unroll 1
        for (int sub = 0; sub < nsub; ++sub) {
            const int rg0 = sub * RGS;
            if (has2) {
                float acc[RGS][4];
#pragma unroll
                for (int rg = 0; rg < RGS; ++rg)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[rg][e] = 0.0f;
                const unsigned *src = rx + (size_t)(s & 1) * rslot + (size_t)(q2 * mth + kq * KT2) * 256 + lane_word;
                const uint4 *Aw = A2 + (size_t)warp * KT2 * 32 + lane;
#pragma unroll 1
                for (int k0 = 0; k0 < m_tiles; k0 += KB) {
                    uint4 w[KB][RGS], af[kAhead ? KB : 1];
                    if (kAhead)
#pragma unroll
                        for (int i = 0; i < KB; ++i) af[kAhead ? i : 0] = k0 + i < m_tiles ? Aw[(size_t)(k0 + i) * 32] : make_uint4(0, 0, 0, 0);
                    fetch(w, src + (size_t)k0 * 256, rx, 2 * rslot, m_tiles - k0, rg0, r_phase, kRPhase);
#pragma unroll
                    for (int i = 0; i < KB; ++i)
                        if (k0 + i < m_tiles) {
                            if (!kAhead) af[0] = Aw[(size_t)(k0 + i) * 32];
#pragma unroll
                            for (int rg = 0; rg < RGS; ++rg) multiply(acc[rg], af[kAhead ? i : 0], w[i][rg], 0x7fff7fffu);
                        }
                }
#pragma unroll
                for (int rg = 0; rg < RGS; ++rg) leave_sums(red + (warp * RGS + rg) * kTileRed, acc[rg]);
            }
            __syncthreads();
            const int b = (rg0 + frg) * 8 + fb;
            float hn = 0.0f, cn = 0.0f;
            const bool live = fin2 && b < B;
            if (live) {
                float z[4];
                const float *rp = red + (frg * 8 + fb) * kPitch + frow;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    z[q] = ((rp[(4 * q) * RGS * kTileRed] + rp[(4 * q + 1) * RGS * kTileRed]) +
                            (rp[(4 * q + 2) * RGS * kTileRed] + rp[(4 * q + 3) * RGS * kTileRed])) + bias[q];
                const float gi = sigmoid_fast(z[0]), gf = sigmoid_fast(z[1]), gg = tanh_fast(z[2]), go = sigmoid_fast(z[3]);
                const bool real = u2 < H;
                cn = real ? fmaf(gf, c_s[b * 16 + frow], gi * gg) : 0.0f;
                hn = real ? go * tanh_fast(cn) : 0.0f;
                if (publish && LSTM_CHECK_INDEX((size_t)(s & 1) * hslot + cta * 256 + (rg0 + frg) * 128 + fb * 16 + frow, 2 * hslot, a.status))
                    st_relaxed_u32(hx + (size_t)(s & 1) * hslot + cta * 256 + (rg0 + frg) * 128 + fb * 16 + frow, pack_word(hn, word_phase(s)));
                c_s[b * 16 + frow] = cn;
            }
            __syncthreads();
            if (live && u2 < H) {
                const long long row = (long long)t * a.Bs + a.b0 + b;
                if (a.y) a.y[row * D * H + (long long)d * H + u2] = hn;
                if (a.xb_next) {
                    const __nv_bfloat16 hi = __float2bfloat16_rn(hn);
                    a.xb_next[row * a.xb_ld + (long long)d * H + u2] = hi;
                    a.xb_next[a.xb_plane + row * a.xb_ld + (long long)d * H + u2] = __float2bfloat16_rn(hn - __bfloat162float(hi));
                }
                if (s == T - 1) {
                    const size_t so = ((size_t)d * a.Bs + a.b0 + b) * H + u2;
                    if (a.hT) a.hT[so] = hn;
                    if (a.cT) a.cT[so] = cn;
                }
            }
        }
    }
}

typedef void (*KernelFn)(const HlstmTileArgs);
template <int MODE>
KernelFn pick_mode(int n1, int kt)
{
    switch (n1 * 16 + kt) {
        case 1 * 16 + 4: return hlstm_tile_kernel<1, 4, MODE>;
        case 2 * 16 + 4: return hlstm_tile_kernel<2, 4, MODE>;
        case 3 * 16 + 4: return hlstm_tile_kernel<3, 4, MODE>;
        case 4 * 16 + 4: if constexpr (MODE != 2) return hlstm_tile_kernel<4, 4, MODE>; else return nullptr;     // (mode_of: n1 * kt <= 12)
        case 1 * 16 + 5: return hlstm_tile_kernel<1, 5, MODE>;
        case 1 * 16 + 6: return hlstm_tile_kernel<1, 6, MODE>;
        case 2 * 16 + 5: return hlstm_tile_kernel<2, 5, MODE>;
        case 2 * 16 + 6: return hlstm_tile_kernel<2, 6, MODE>;
        case 3 * 16 + 5: if constexpr (MODE != 2) return hlstm_tile_kernel<3, 5, MODE>; else return nullptr;
        case 3 * 16 + 6: if constexpr (MODE != 2) return hlstm_tile_kernel<3, 6, MODE>; else return nullptr;
        default: return nullptr;
    }
}
KernelFn pick(int n1, int kt, int mode) { return mode == 0 ? pick_mode<0>(n1, kt) : mode == 1 ? pick_mode<1>(n1, kt) : pick_mode<2>(n1, kt); }

size_t smem_bytes(int Hh, int n1, int rows, int mode)
{
    const int kt2 = ((Hh + 15) / 16 + 3) / 4;
    return (size_t)kWarps * kt2 * 512 + (size_t)kWarps * n1 * (mode == 2 ? 2 : 1) * kTileRed * 4 + (size_t)rows * 64;
}
// two row groups together where the registers (fragments, two sets of sums, twelve chunks in flight) and shared memory allow
int mode_of(const HlstmTilePlan &p, int rows, size_t max_smem)
{
    if (rows <= 4) return 0;
    return rows > 8 && p.n1 * p.kt <= 12 && smem_bytes(p.Hh, p.n1, rows, 2) <= max_smem ? 2 : 1;
}

}  // namespace

// Partition over at most max_cta CTAs per direction; false when the slices do not fit (then hlstm_mma.cu runs).
bool hlstm_tile_plan(int H, int Hh, int max_cta, size_t max_smem, HlstmTilePlan *p)
{
    const int mt = 4 * ((Hh + 15) / 16), ut = (H + 15) / 16;
    p->H = H; p->Hh = Hh; p->max_smem = max_smem;
    p->n1 = (mt + max_cta - 1) / max_cta;
    p->kt = std::max(4, (ut + 15) / 16);
    p->ncta = (mt + p->n1 - 1) / p->n1;
    if (ut > p->ncta) p->ncta = ut;
    return ut <= max_cta && (ut + 15) / 16 <= 6 && pick(p->n1, p->kt, 0) && smem_bytes(Hh, p->n1, kHtRows, 1) <= max_smem;
}

size_t hlstm_tile_smem_bytes(const HlstmTilePlan &p, int rows) { return smem_bytes(p.Hh, p.n1, rows, mode_of(p, rows, p.max_smem)); }

cudaError_t hlstm_tile_prepare(const HlstmTilePlan &p)
{
    for (int mode = 0; mode < 3; ++mode) {
        if (!pick(p.n1, p.kt, mode)) continue;
        const cudaError_t e = cudaFuncSetAttribute(pick(p.n1, p.kt, mode), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.max_smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_hlstm_tile(const HlstmTileArgs &a, const HlstmTilePlan &p, cudaStream_t st)
{
    const int mode = mode_of(p, a.B, p.max_smem);
    HlstmTileArgs copy = a;
    void *params[] = {&copy};
    return cudaLaunchCooperativeKernel((const void *)pick(p.n1, p.kt, mode), dim3(a.ncta_dir * a.D), dim3(kThreads), params,
                                       hlstm_tile_smem_bytes(p, a.B), st);
}

}  // namespace lstm

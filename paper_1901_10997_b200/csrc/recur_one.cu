// Register-resident recurrent kernel for ONE sequence and bf16 weights: the serial half of the LSTM forward pass
// (paper, Section 4, cell equations with zero hidden layers per gate)
//     z = G[t] + Wh h_{t-1};  i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c_t = f c_{t-1} + i g;
//     h_t = o tanh(c_t)
// One cooperative launch runs all T steps of one layer (both directions side by side on disjoint CTA groups).  As in
// recur_mma.cu a CTA keeps its slice of Wh in registers as operand-A fragments of mma.sync.m16n8k16, warp w the column
// tiles of its own range; the slices of tensor memory (recur_tc.cu) do not pay for a single column.  A step is one chain
// publish -> L2 -> poll -> products -> barrier -> gates -> publish, and everything here is about keeping it short:
//   * h travels as 32-bit words with a phase bit (device_util.cuh).  A CTA owns a multiple of FOUR units, so the 16-byte
//     chunk a lane polls has one writer and a warp's whole range is one load instruction; the columns of a tile are
//     permuted at pack time so that a chunk is four adjacent columns of an operand fragment;
//   * the projection terms are requested behind the last poll and the outputs of a step are stored before the next
//     barrier, so nothing stands between a publish and the poll that follows it but the second barrier; without it the
//     warps that finish no units poll early, and early polls delay the words they wait for (H = 1500: 1.62 us a step
//     with the barrier, 1.93 without);
//   * after the barrier eight lanes per unit add the warps' partial sums (two lanes a gate), and a warp publishes the words
//     of four units in one store.
// A short call (T <= kFuseMaxT) computes its projection in the prologue (recur_parts.cuh).
// Every wait is bounded; on expiry the CTA records a timeout status, stops waiting and runs to the end.
#include "common.cuh"
#include "device_util.cuh"
#include "recur_parts.cuh"

#include <algorithm>

namespace lstm {
namespace {

constexpr int kNT = kOneThreads, kNW = kNT / 32;
constexpr int kMaxSplit = 4, kOneMinUnits = 1025;

// FUSE: projection in the prologue; PROBE: measurement build that leaves parts of the step out
template <int MT, int NKR, bool FUSE, bool PROBE>
__global__ void __launch_bounds__(kNT, 1) recur_one_kernel(const RecurOneArgs a)
{
    const int probe = PROBE ? a.probe : 0;
    constexpr int UPC = 4 * MT, RP = MT * 16 + 4;              // units per CTA; floats between the warps' partial sums
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int abort_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, tig = lane & 3;
    const int H = a.H, T = a.T, D = a.D, Hq = (H + 3) & ~3;
    const int d = a.dir0 + blockIdx.x / a.ncta_dir, cta = blockIdx.x % a.ncta_dir;
    const int u0 = cta * UPC, nu = min(UPC, H - u0);
    const int nks = a.nkw_smem, nkw = NKR + nks, kbase = warp * nkw * 16;

    // ---- shared memory: partial sums of two steps, the warps' staged operands [plane][chunk], weight tiles beyond the registers
    float *red = reinterpret_cast<float *>(smem);                                          // [2][kNW][RP]
    uint2 *hs = reinterpret_cast<uint2 *>(red + 2 * kNW * RP) + warp * 64;                 // [kNW][2][32]
    uint4 *As = reinterpret_cast<uint4 *>(red + 2 * kNW * RP + kNW * 128);                 // [kNW][nks][MT][32]
    constexpr int GP = MT * 16 + 1;
    const float *G_s = nullptr;
    LSTM_CHECK_SMEM_END(reinterpret_cast<unsigned char *>(As + (size_t)kNW * nks * MT * 32) - smem, a.status);
    if (FUSE) LSTM_CHECK_SMEM_END((size_t)a.gs_off + (size_t)kFuseMaxT * GP * 4, a.status);

    // exchange words [set][place in the launch][slot][CTA's line]; this set starts with every phase bit at 0, the other one
    // is cleared for the next launch
    const unsigned slot_words = 32u * a.ncta_dir;
    const size_t off = (size_t)(d - a.dir0) * 2 * slot_words, set_words = (size_t)2 * D * slot_words;     // a line per CTA and slot
    unsigned *xch = a.xch + (size_t)a.set * set_words + off;
    if (tid < 2 * UPC) a.xch[(size_t)(a.set ^ 1) * set_words + off + (size_t)(tid & 1) * slot_words + cta * 32 + (tid >> 1)] = 0u;

    const uint4 *wsrc = a.wfrag[d] + ((size_t)(cta * kNW + warp) * nkw) * MT * 32 + lane;
    if (FUSE) {
        // both weight streams are requested into L2 at once, so that they leave HBM side by side
        for (int i = lane; i < nkw * MT * 4; i += 32)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(wsrc - lane) + (size_t)i * 128));
        G_s = fused_projection<MT, kNW>(smem, (size_t)a.gs_off, a.X, a.xfrag[d], a.bias, a.nkw_x, a.in_l, T, H, d, cta, u0, nu, tid);
    }
    uint4 areg[NKR][MT];
#pragma unroll
    for (int i = 0; i < NKR; ++i)
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) areg[i][mt] = ld_nc_u4(wsrc + (size_t)(i * MT + mt) * 32);
    uint4 *As_w = As + (size_t)warp * nks * MT * 32 + lane;
    for (int i = 0; i < nks * MT; ++i) As_w[(size_t)i * 32] = __ldg(wsrc + (size_t)(NKR * MT + i) * 32);
    for (int i = tid; i < 2 * kNW * RP; i += kNT) red[i] = 0.0f;
    hs[lane] = make_uint2(0, 0);
    hs[32 + lane] = make_uint2(0, 0);

    // finishing: warp w < MT takes units 4 w .. 4 w + 3, eight lanes each: gate (lane >> 1) & 3, half of the warps' sums lane & 1
    const int fq = (lane >> 1) & 3, fu = warp * 4 + (lane >> 3), j = u0 + fu, role = lane & 7;
    const bool fin = warp < MT, own = fin && j < Hq, real = fin && fu < nu;
    const float act_k = (fq == 2 ? -2.0f : -1.0f) * 1.4426950408889634f, act_sc = fq == 2 ? 2.0f : 1.0f, act_of = fq == 2 ? -1.0f : 0.0f;
    float c = real && a.c0 ? a.c0[(size_t)d * H + j] : 0.0f, hn = 0.0f;
    const long long t0 = d ? T - 1 : 0, dir = d ? -1 : 1;
    const float *gp = a.G + (t0 * D + d) * 4 * H + 4 * (long long)j + fq;
    const float *gs = FUSE ? G_s + t0 * GP + 4 * fu + fq : nullptr;
    float *yp = a.y + t0 * D * H + (long long)d * H + j;
    __nv_bfloat16 *xp = a.xb_next ? a.xb_next + t0 * a.xb_ld + (long long)d * H + j : nullptr;
    const long long gadv = dir * D * 4 * H, yadv = dir * D * H, xadv = dir * a.xb_ld;
    unsigned *out = xch + cta * 32 + fu;
    const bool publish = own && role == 0 && (int)blockIdx.x != a.withhold_cta;
    if (tid == 0) abort_s = 0;
    __syncthreads();
    volatile int *abort_v = &abort_s;

    // warps beyond H poll nothing and finish nothing: they leave, their partial sums stay zero
    const int n_active = (H + nkw * 16 - 1) / (nkw * 16), nbar = 32 * max(n_active, MT);
    if (warp * 32 >= nbar) return;
    const bool has = lane < nkw * 4 && kbase + 4 * lane < Hq;                              // this lane has a chunk to poll
    const int chunk = (kbase >> 2) + lane;
    const unsigned *src = xch + (chunk / MT) * 32 + (chunk % MT) * 4;
    const uint2 *hl = hs + (g & 1) * 32 + tig;                                             // operand B: plane g & 1 in column g

    auto write_outputs = [&]() {
        if (real) {
            if (role == 1) *yp = hn;
            else if (role == 2 && xp) *xp = __float2bfloat16_rn(hn);
            else if (role == 3 && xp) xp[a.xb_plane] = __float2bfloat16_rn(hn - __bfloat162float(__float2bfloat16_rn(hn)));
        }
        yp += yadv;
        xp = xp ? xp + xadv : xp;
    };

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        // ---- this warp's columns of h_{t-1}
        uint4 w = make_uint4(0, 0, 0, 0);
        if (s == 0) {
            if (a.h0 && has) {
                const float *hp = a.h0 + (size_t)d * H + kbase + 4 * lane;
                const int left = H - (kbase + 4 * lane);
                w.x = split_word(hp[0]);
                if (left > 1) w.y = split_word(hp[1]);
                if (left > 2) w.z = split_word(hp[2]);
                if (left > 3) w.w = split_word(hp[3]);
            }
        } else {
            const unsigned phase = word_phase(s - 1);
            const unsigned *p = src + ((s - 1) & 1) * slot_words;
            if (has && LSTM_CHECK_INDEX(p - xch + 3, 2 * slot_words, a.status)) w = ld_relaxed_v4(p);
            bool wait = has && !words_ready(w, phase) && !(probe & 4);
            int polls = 0;
            long long t_start = 0;
            while (wait) {
                w = ld_relaxed_v4(p);
                wait = !words_ready(w, phase);
                if (wait && ((++polls & 31) == 0 || *abort_v)) {
                    const long long now = clock64();
                    if (t_start == 0) t_start = now;
                    if (*abort_v) wait = false;
                    else if (now - t_start > a.spin_limit || ld_volatile_s32(a.status) != kStatusOk) {
                        *abort_v = 1;
                        atomicExch(a.status, kStatusTimeout);
                        wait = false;
                    }
                }
            }
        }
        __syncwarp();
        const unsigned keep = s == 0 ? 0xffffffffu : 0xbfffbfffu;
        hs[lane] = make_uint2(__byte_perm(w.x, w.y, 0x7632u) & keep, __byte_perm(w.z, w.w, 0x7632u) & keep);
        hs[32 + lane] = make_uint2(__byte_perm(w.x, w.y, 0x5410u), __byte_perm(w.z, w.w, 0x5410u));
        __syncwarp();

        // ---- partial products: register tiles, then the shared-memory tiles
        float acc[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][e] = 0.0f;
        if (!(probe & 1)) {
#pragma unroll
            for (int i = 0; i < NKR; ++i) {
                const uint2 b = hl[4 * i];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt], areg[i][mt], b.x, b.y);
            }
            for (int i = 0; i < nks; ++i) {
                const uint2 b = hl[4 * (NKR + i)];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt], As_w[(size_t)(i * MT + mt) * 32], b.x, b.y);
            }
        }
        // accumulator columns 0 and 1 are the hi and lo products (the other columns repeat them)
        if (tig == 0 && LSTM_CHECK_INDEX(((s & 1) * kNW + warp) * RP + g + (MT - 1) * 16 + 8, 2 * kNW * RP, a.status)) {
            float *rw = red + ((s & 1) * kNW + warp) * RP + g;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                rw[mt * 16] = acc[mt][0] + acc[mt][1];
                rw[mt * 16 + 8] = acc[mt][2] + acc[mt][3];
            }
        }
        // projection term of this lane's gate: one value per split-K plane, on its way until the sums are there
        float v[kMaxSplit] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (real && (lane & 1) == 0 && !(probe & 2)) {
            if (FUSE) v[0] = *gs;
            else {
#pragma unroll
                for (int sp = 0; sp < kMaxSplit; ++sp)
                    if (sp < a.nsplit) v[sp] = ld_nc_early(gp + sp * a.g_split_stride);
                if (fq == 0 && s + 2 < T) asm volatile("prefetch.global.L2 [%0];" ::"l"(gp + 2 * gadv));
            }
        }
        gp += gadv;
        gs += FUSE ? (int)dir * GP : 0;
        if (fin && s > 0 && !(probe & 2)) write_outputs();
        bar_sync(1, nbar);

        if (probe & 2) {
            if (publish) st_relaxed_u32(out + (s & 1) * slot_words, pack_word(0.0f, word_phase(s)));
        } else if (fin) {
            const float *rp = red + ((s & 1) * kNW + (lane & 1) * 8) * RP + 4 * fu + fq;
            float p[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) p[k] = rp[k * RP] + rp[(k + 4) * RP];
            float z = ((p[0] + p[1]) + (p[2] + p[3])) + ((v[0] + v[1]) + (v[2] + v[3]));
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            const float act = gate_fast(z, act_k, act_sc, act_of);
            const int q0 = lane & ~7;
            const float vi = __shfl_sync(0xffffffffu, act, q0), vf = __shfl_sync(0xffffffffu, act, q0 + 2);
            const float vg = __shfl_sync(0xffffffffu, act, q0 + 4), vo = __shfl_sync(0xffffffffu, act, q0 + 6);
            c = fmaf(vf, c, vi * vg);
            hn = vo * tanh_fast(c);
            if (publish && LSTM_CHECK_INDEX(out - xch + (s & 1) * slot_words, 2 * slot_words, a.status))
                st_relaxed_u32(out + (s & 1) * slot_words, pack_word(hn, word_phase(s)));
        }
        __syncwarp();
        bar_sync(2, nbar);
    }
    if (fin) {
        write_outputs();
        if (real && role == 4 && a.hT) a.hT[(size_t)d * H + j] = hn;
        if (real && role == 5 && a.cT) a.cT[(size_t)d * H + j] = c;
    }
}

typedef void (*KernelFn)(const RecurOneArgs);
template <bool FUSE, bool PROBE>
KernelFn pick_f(int mt, int nkr)
{
    switch (mt * 16 + nkr) {
        case 48 + 6: return recur_one_kernel<3, 6, FUSE, PROBE>;
        case 64 + 4: return recur_one_kernel<4, 4, FUSE, PROBE>;
        default: return nullptr;
    }
}
KernelFn pick(int mt, int nkr, bool fuse, bool probe)
{
    return probe ? pick_f<false, true>(mt, nkr) : fuse ? pick_f<true, false>(mt, nkr) : pick_f<false, false>(mt, nkr);
}

}  // namespace

size_t recur_one_smem_bytes(int mt, int nks) { return (size_t)2 * kNW * (mt * 16 + 4) * 4 + (size_t)kNW * 512 + (size_t)kNW * nks * mt * 512; }
// fused projection: the warps' partial products (24 timesteps each) lie over the kernel's other shared memory, the finished
// rows of G behind whichever is larger
size_t recur_one_gs_offset(int mt, int nks)
{
    return (std::max(recur_one_smem_bytes(mt, nks), (size_t)kNW * 24 * (mt * 16 + 1) * 4) + 15) & ~(size_t)15;
}
size_t recur_one_fuse_smem_bytes(int mt, int nks) { return recur_one_gs_offset(mt, nks) + (size_t)kFuseMaxT * (mt * 16 + 1) * 4; }

// Whole groups of four units per CTA; column tiles per warp in registers as far as 128 registers allow (MT * NKR <= 18), the
// others in shared memory.
// Served: slices of more than eight units (mt 3 and 4) and 1025 .. 2048 columns.  us per step, recur_mma.cu -> here: H = 1200
// 1.78 -> 1.65, 1500 1.78 -> 1.72, 1776 2.02 -> 1.89, 2000 2.57 -> 2.33, two directions of 1100 1.92 -> 1.78.  Slices of eight
// units gain nothing (1184: 1.51 either way) or lose (1100: 1.44 -> 1.54), nor do 1024 columns and fewer (two directions of
// 800 1.50 either way, 512 1.17 -> 1.36): the shorter product no longer covers the second barrier.
bool recur_one_plan(int H, int max_cta, size_t max_smem, RecurOnePlan *p)
{
    const int upc = ((H + max_cta - 1) / max_cta + 3) / 4 * 4, need = ((H + 15) / 16 + kNW - 1) / kNW;
    p->mt = upc / 4;
    p->nkr = p->mt == 4 ? 4 : 6;
    p->nks = std::max(0, need - p->nkr);
    p->ncta = (H + upc - 1) / upc;
    return H >= kOneMinUnits && p->mt >= 3 && pick(p->mt, p->nkr, false, false) && p->nkr + p->nks <= 8 && recur_one_smem_bytes(p->mt, p->nks) <= max_smem;
}

cudaError_t recur_one_prepare(const RecurOnePlan &p, int max_smem)
{
    for (int i = 0; i < 3; ++i) {
        const cudaError_t e = cudaFuncSetAttribute(pick(p.mt, p.nkr, i == 1, i == 2), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_recur_one(const RecurOneArgs &a, const RecurOnePlan &p, bool fuse, cudaStream_t st)
{
    RecurOneArgs copy = a;
    void *params[] = {&copy};
    return cudaLaunchCooperativeKernel((const void *)pick(p.mt, p.nkr, fuse, a.probe != 0), dim3(a.ncta_dir * (a.ndirs ? a.ndirs : a.D)), dim3(kNT), params,
                                       fuse ? recur_one_fuse_smem_bytes(p.mt, p.nks) : recur_one_smem_bytes(p.mt, p.nks), st);
}

}  // namespace lstm

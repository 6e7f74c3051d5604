// Recurrent kernel for fp32 weights on the double-precision tensor instruction: the serial half of the LSTM forward pass
// (paper, Section 4, cell equations with zero hidden layers per gate)
//     z = G[t] + Wh h_{t-1};  i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c_t = f c_{t-1} + i g;
//     h_t = o tanh(c_t)
// for up to two units per CTA and 32 batch rows; sums and gate functions in fp64 (fp32 sums miss the bound on outputs near
// zero), state and outputs fp32.  Wider layers and larger batches run on recur.cu.
//
// The eight gate rows of a CTA's two units are exactly the M of mma.m8n8k4.f64, eight batch rows its N.  The sixteen warps
// split (row tile of eight batch rows) x (K range); the weights of a warp's K range sit in registers as doubles.  A lane's
// operand is ONE value of h, so it polls that word straight into its fragment: no staging, no reduction across lanes (a
// dot product per warp needed 160 shuffles a unit).  h travels as its own 32 bits: |h| <= 1, so bit 30 is free for the phase
// (device_util.cuh); a unit's 32 batch rows are one line with one writer.  After one barrier a quad per (unit, batch row) adds
// the K ranges' sums, one gate each, and applies the gate functions, each from one exponential and one division.
// Measured (2 x 200, batch 20, T = 35, per call): 480 us with recur.cu, 209 us here.
// Every wait is bounded; on expiry the CTA records a timeout status, stops waiting and runs to the end.
#include "common.cuh"
#include "device_util.cuh"

namespace lstm {
namespace {

constexpr int kThreads = kF32Threads, kWarps = kThreads / 32;

// NT: tiles of eight batch rows
template <int NT>
__global__ void __launch_bounds__(kThreads, 1) recur_f32_kernel(const RecurF32Args a)
{
    constexpr int KS = kWarps / NT;                        // K ranges
    constexpr int KW = (kF32MaxUnits / 4 + KS - 1) / KS;   // k4 steps of a range, at most
    constexpr int RB = NT * 8, P = RB + 2;                 // doubles between rows of partial sums
    __shared__ double red[KS * 8 * P];
    __shared__ int abort_s;
    __shared__ int nan_s[32];                              // batch rows with a NaN in h: every sum of theirs is one, from then on
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.H, B = a.B, T = a.T, D = a.D;
    const int d = a.dir0 + blockIdx.x / a.ncta_dir, cta = blockIdx.x % a.ncta_dir;
    int u0, nu;
    unit_range(H, a.ncta_dir, cta, u0, nu);

    // exchange words [set][direction of the launch][slot][unit][32 batch rows]; the other set is cleared for the next launch
    const unsigned slot_words = (unsigned)H * 32u;
    const size_t off = (size_t)(d - a.dir0) * 2 * slot_words, set_words = (size_t)2 * D * slot_words;
    unsigned *xch = a.xch + (size_t)a.set * set_words + off;
    for (int i = tid; i < nu * 64; i += kThreads)
        a.xch[(size_t)(a.set ^ 1) * set_words + off + (size_t)(i & 1) * slot_words + u0 * 32 + (i >> 1)] = 0u;

    const int ksteps = (H + 3) >> 2, kper = (ksteps + KS - 1) / KS;
    const int nt = warp / KS, kq = warp - nt * KS;
    const int k0 = kq * kper, kn = nt < NT ? max(0, min(kper, ksteps - k0)) : 0;
    const int kcol = 4 * k0 + (lane & 3), b_lane = nt * 8 + (lane >> 2);
    double af[KW];
    {
        const int row = lane >> 2, u = row >> 2, q = row & 3;
        const float *w = a.wh[d] + ((size_t)(u0 + u) * 4 + q) * a.Hp8 + kcol;
#pragma unroll
        for (int i = 0; i < KW; ++i) af[i] = i < kn && u < nu && kcol + 4 * i < H ? (double)w[4 * i] : 0.0;
    }
    unsigned mine = 0;                                     // k4 steps in which this lane has a value to fetch
#pragma unroll
    for (int i = 0; i < KW; ++i)
        if (i < kn && b_lane < B && kcol + 4 * i < H) mine |= 1u << i;
    const unsigned *src0 = xch + kcol * 32 + b_lane;

    // finishing: threads 4 i .. 4 i + 3 finish item i = (unit, batch row), one gate each
    const int fq = tid & 3, item = tid >> 2, fu = item / RB, fb = item - fu * RB;
    const bool fin = tid < 64 * NT, live = fin && fu < nu && fb < B;
    const double act_k = fq == 2 ? -2.0 : -1.0, act_sc = fq == 2 ? 2.0 : 1.0, act_of = fq == 2 ? -1.0 : 0.0;
    const int j = u0 + fu;
    const size_t so = ((size_t)d * B + fb) * H + j;
    float c = live && a.c0 ? a.c0[so] : 0.0f, hn = 0.0f;
    const long long t0 = d ? T - 1 : 0, dir = d ? -1 : 1;
    const float *gp = a.G + ((t0 * B + fb) * D + d) * 4 * H + 4 * (long long)j + fq;
    float *yp = a.y + (t0 * B + fb) * D * H + (long long)d * H + j;
    const long long gadv = dir * B * D * 4 * H, yadv = dir * B * D * H;
    unsigned *out = xch + (size_t)j * 32 + fb;
    const double *rp = red + (fu * 4 + fq) * P + fb;
    if (tid == 0) abort_s = 0;
    if (tid < 32) nan_s[tid] = 0;
    __syncthreads();
    volatile int *abort_v = &abort_s;

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        const float g = live ? ld_nc_early(gp) : 0.0f;
        gp += gadv;
        // ---- this lane's values of h_{t-1} as operand B
        unsigned w[KW];
#pragma unroll
        for (int i = 0; i < KW; ++i) w[i] = 0u;
        if (s == 0) {
            if (a.h0)
#pragma unroll
                for (int i = 0; i < KW; ++i)
                    if (mine & (1u << i)) w[i] = __float_as_uint(a.h0[((size_t)d * B + b_lane) * H + kcol + 4 * i]);
        } else {
            const unsigned *src = src0 + ((s - 1) & 1) * slot_words;
            const unsigned phase = word_phase(s - 1);
            unsigned pending = *abort_v ? 0u : mine;
            int polls = 0;
            long long t_start = 0;
            while (pending) {
#pragma unroll
                for (int i = 0; i < KW; ++i)
                    if ((pending & (1u << i)) && LSTM_CHECK_INDEX(src - xch + i * 128, 2 * slot_words, a.status)) w[i] = ld_relaxed_u32(src + i * 128);
#pragma unroll
                for (int i = 0; i < KW; ++i)
                    if ((pending & (1u << i)) && ((w[i] ^ phase) & kPhaseBit) == 0) pending &= ~(1u << i);
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
        }
        __syncwarp();
        float top = 0.0f;
        if (s > 0) {
#pragma unroll
            for (int i = 0; i < KW; ++i) {
                w[i] &= ~kPhaseBit;
                top = fmaxf(top, fabsf(__uint_as_float(w[i])));
            }
        }
        double acc0[2] = {0.0, 0.0}, acc1[2] = {0.0, 0.0};      // two chains: the instruction's latency exceeds its rate
#pragma unroll
        for (int i = 0; i < KW; ++i)
            if (i < kn) mma_f64(i & 1 ? acc1 : acc0, af[i], (double)__uint_as_float(w[i]));
        if (nt < NT && LSTM_CHECK_INDEX((kq * 8 + (lane >> 2)) * P + nt * 8 + 2 * (lane & 3) + 1, KS * 8 * P, a.status)) {
            double *r = red + (kq * 8 + (lane >> 2)) * P + nt * 8 + 2 * (lane & 3);
            r[0] = acc0[0] + acc1[0];
            r[1] = acc0[1] + acc1[1];
        }
        if (top > kMaskedNan) nan_s[b_lane] = 1;       // (h of the first step keeps all its bits: no mark needed)
        __syncthreads();
        if (fin) {
            double z = (double)g;
#pragma unroll
            for (int k = 0; k < KS; ++k) z += rp[k * 8 * P];
            if (nan_s[fb]) z = nan("");
            const double act = gate_f64(z, act_k, act_sc, act_of);
            const int ql = lane & ~3;
            const double vi = __shfl_sync(0xffffffffu, act, ql), vf = __shfl_sync(0xffffffffu, act, ql + 1);
            const double vg = __shfl_sync(0xffffffffu, act, ql + 2), vo = __shfl_sync(0xffffffffu, act, ql + 3);
            const double cn = fma(vf, (double)c, vi * vg);
            hn = (float)(vo * gate_f64(cn, -2.0, 2.0, -1.0));
            c = (float)cn;
            if (live && fq == 0 && (int)blockIdx.x != a.withhold_cta && LSTM_CHECK_INDEX(out - xch + (s & 1) * slot_words, 2 * slot_words, a.status))
                st_relaxed_u32(out + (s & 1) * slot_words, (__float_as_uint(hn) & ~kPhaseBit) | word_phase(s));
        }
        __syncthreads();                    // nobody polls before the CTA has published; the sums are free again
        if (live && fq == 1) *yp = hn;
        yp += yadv;
    }
    if (live && fq == 2 && a.hT) a.hT[so] = hn;
    if (live && fq == 3 && a.cT) a.cT[so] = c;
}

typedef void (*KernelFn)(const RecurF32Args);

}  // namespace

cudaError_t launch_recur_f32(const RecurF32Args &a, cudaStream_t st)
{
    static const KernelFn kernels[4] = {recur_f32_kernel<1>, recur_f32_kernel<2>, recur_f32_kernel<3>, recur_f32_kernel<4>};
    if (a.B < 1 || a.B > kF32MaxRows) return cudaErrorInvalidValue;
    RecurF32Args copy = a;
    void *params[] = {&copy};
    return cudaLaunchCooperativeKernel((const void *)kernels[(a.B - 1) / 8], dim3(a.ncta_dir * (a.ndirs ? a.ndirs : a.D)), dim3(kThreads), params, 0, st);
}

}  // namespace lstm

// All layers of a unidirectional fp32 stack in one launch, on the double-precision tensor instruction: the LSTM forward pass
// (paper, Section 4, cell equations with zero hidden layers per gate; Section 5.1: two stacked layers)
//     z = Wx x_t + Wh h_{t-1} + b;  i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c_t = f c_{t-1} + i g;  h_t = o tanh(c_t)
// where x_t is the call's input for layer 0 and h_t of the layer below for the others.  CTAs [l * ncta, (l + 1) * ncta) run
// layer l, up to four units each; layer l works on timestep t while layer l - 1 is already on t + 1, so that the call costs
// T + L - 1 serial steps instead of L x T, and no projection launch.
//
// What bounds a step is the chain publish -> L2 -> poll -> products -> barrier -> gates of the layer's own h, and beside it the
// rate of the tensor instruction (four cycles of an SM for mma.m8n8k4.f64).  As in recur_f32.cu the eight gate rows of two
// units are its M and eight batch rows its N; here a warp takes every sixteenth group of four columns for ALL row tiles, and the
// words of a unit are stored as [row within the tile][tile], so that one vector load gives a lane its operand of every tile and
// a warp reads whole lines, each once per CTA (loads of single words by the warps of each tile: 1300 to 2300 cycles a fetch).
// The products with x_t need nothing of the chain: their operand is requested a step ahead and they run in the time the words of
// h_{t-1} travel.  The weights of both halves are kept in shared memory as doubles in operand order: a fragment is one
// conflict-free 8-byte load, two cycles of shared memory beside four of the tensor instruction.
// A layer may run any number of steps ahead of the one above: its words have a slot for every timestep, which also makes the
// phase bit (device_util.cuh) a plain "written" mark; the other set is cleared for the next launch.
// Measured (us per call, T = 35, layer by layer on recur_f32.cu -> here): 2 x 200 with 20 rows 210 -> 135, 2 x 256 with 32 rows, T = 70
// 568 -> 387, 2 x 149 with 9 rows, T = 17 101 -> 60, 2 x 64 with one row, T = 4 34 -> 16, three layers of 150 with 16 rows, T = 12
// 114 -> 47.  A step of 2 x 200 with 20 rows is 3.7 us, 7100 cycles: 1400 for each half's products, 900 for the fetch of h, 1500 for sums and
// gates; the rest was not told apart.
// Every wait is bounded; on expiry the CTA records a timeout status, stops waiting and runs to the end.
#include "common.cuh"
#include "device_util.cuh"

namespace lstm {
namespace {

constexpr int kThreads = kF32Threads, kWarps = kThreads / 32;
constexpr int kStaticSmem = 256;               // static shared memory of the kernel, at most

__host__ __device__ constexpr int f32_wave_red_doubles(int nt, int mt) { return kWarps * 8 * mt * (8 * nt + 4); }

// floats between the rows of a staged x_t: four columns by eight rows of an operand on 32 different banks
__host__ __device__ constexpr int f32_wave_x_pitch(int K) { return ((K + 3) / 4 | 1) * 4; }

template <int V> __device__ __forceinline__ void ld_words(const unsigned *p, unsigned (&w)[V])
{
    if constexpr (V == 1) w[0] = ld_relaxed_u32(p);
    else if constexpr (V == 2) asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p) : "memory");
    else {
        const uint4 v = ld_relaxed_v4(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
}

// NT: tiles of eight batch rows; MT: tiles of eight gate rows (two units)
template <int NT, int MT>
__global__ void __launch_bounds__(kThreads, 1) recur_f32_wave_kernel(const RecurF32WaveArgs a)
{
    constexpr int KW = (kF32MaxUnits / 4 + kWarps - 1) / kWarps;      // groups of four columns of a warp, at most: warp, warp + 16, ..
    constexpr int RB = NT * 8, P = RB + 4;                 // doubles between rows of partial sums (no bank conflicts for the readers)
    constexpr int V = NT == 3 ? 4 : NT;                    // words of a unit: [8 rows][V tiles], batch row = 8 * tile + row
    extern __shared__ __align__(16) double smem[];
    __shared__ int abort_s;
    __shared__ int nan_s[32];                              // batch rows with a NaN in a polled h: every sum of theirs is one, from then on
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = a.H, B = a.B, T = a.T;
    const int l = blockIdx.x / a.ncta, cta = blockIdx.x - l * a.ncta;
    const int u0 = cta * a.upc, nu = max(0, min(a.upc, H - u0));
    const int Kx = l ? H : a.in_dim;
    const int k4x = (Kx + 3) >> 2, k4h = (H + 3) >> 2;
    double *ws = smem, *red = smem + (size_t)(k4x + k4h) * MT * 32;      // [k4x + k4h][MT][32 lanes]; [warp][8 MT][P]
    float *xs = reinterpret_cast<float *>(red + f32_wave_red_doubles(NT, MT));             // layer 0: x_t [2][B][XP]
    const int XP = f32_wave_x_pitch(Kx);
    LSTM_CHECK_SMEM_END(reinterpret_cast<unsigned char *>(xs + (l ? 0 : 2 * B * XP)) - reinterpret_cast<unsigned char *>(smem), a.status);

    // exchange words [set][layer][timestep (room for 32 rows)][unit][8 rows][V tiles]
    const unsigned slot_words = (unsigned)H * 32u;
    const size_t layer_words = (size_t)a.slots * slot_words, set_words = a.L * layer_words;
    unsigned *own = a.xch + (size_t)a.set * set_words + l * layer_words;
    const unsigned *below = own - (l ? layer_words : 0);
    {
        uint4 *other = reinterpret_cast<uint4 *>(a.xch + (size_t)(a.set ^ 1) * set_words + l * layer_words);
        const size_t n = (size_t)a.clear_T * slot_words / 4;
        for (size_t i = (size_t)cta * kThreads + tid; i < n; i += (size_t)a.ncta * kThreads) other[i] = make_uint4(0, 0, 0, 0);
    }
    if (l == 0)         // the whole input on its way to L2: every CTA of this layer reads all of it, step by step
        for (size_t i = (size_t)cta * kThreads + tid; i < ((size_t)T * B * Kx + 31) / 32; i += (size_t)a.ncta * kThreads)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.x + i * 32));
    for (int i = tid; i < (k4x + k4h) * MT * 32; i += kThreads) {
        const int ln = i & 31, mt = (i >> 5) % MT, k = (i >> 5) / MT;
        const int row = mt * 8 + (ln >> 2), u = row >> 2, q = row & 3;
        const bool hh = k >= k4x;
        const int col = 4 * (hh ? k - k4x : k) + (ln & 3);
        const size_t r = (size_t)(u0 + u) * 4 + q;
        ws[i] = u < nu && col < (hh ? H : Kx) ? (double)(hh ? a.wh[l][r * a.Hp8 + col] : a.wx[l][r * a.ldx[l] + col]) : 0.0;
    }

    const int kxn = max(0, (k4x - warp + kWarps - 1) / kWarps), khn = max(0, (k4h - warp + kWarps - 1) / kWarps);
    const int rr = lane >> 2, col = 4 * warp + (lane & 3); // this lane: column col + 64 i, batch rows rr + 8 tile
    const int nrows = rr < B ? (B - rr + 7) >> 3 : 0;      // tiles in which that row exists
    const double *wxs = ws + (size_t)warp * MT * 32 + lane, *whs = ws + (size_t)(k4x + warp) * MT * 32 + lane;
    constexpr int kWStep = kWarps * MT * 32;               // fragments from group to group

    // finishing: threads 4 i .. 4 i + 3 finish item i = (unit, batch row), one gate each
    const int fq = tid & 3, item = tid >> 2, fu = item / RB, fb = item - fu * RB;
    const bool fin = tid < 64 * NT * MT, live = fin && fu < nu && fb < B;
    const double act_k = fq == 2 ? -2.0 : -1.0, act_sc = fq == 2 ? 2.0 : 1.0, act_of = fq == 2 ? -1.0 : 0.0;
    const int j = u0 + fu;
    const size_t so = ((size_t)l * B + fb) * H + j;
    float c = live && a.c0 ? a.c0[so] : 0.0f, hn = 0.0f;
    const double bias = live ? (double)a.bias[l][4 * j + fq] : 0.0;
    float *yp = a.y + (size_t)fb * H + j;
    const bool write_y = live && fq == 1 && l == a.L - 1;
    unsigned *out = own + (size_t)j * (8 * V) + (fb & 7) * V + (fb >> 3);
    const double *rp = red + (fu * 4 + fq) * P + fb;
    if (tid == 0) abort_s = 0;
    if (tid < 32) nan_s[tid] = 0;
    __syncthreads();
    volatile int *abort_v = &abort_s;

    // this lane's words of one slot: requested, and later waited for; a batch row with a NaN is marked.  (This is on the chain, by
    // all warps of the CTA: one AND per word for "written", one strip, half a maximum.)
    const int lane_x = nrows ? max(0, (Kx - col + 63) >> 6) : 0, lane_h = nrows ? max(0, (H - col + 63) >> 6) : 0;   // groups of this lane
    auto request = [&](const unsigned *src, int n, unsigned (&w)[KW][V]) {
#pragma unroll
        for (int i = 0; i < KW; ++i)
            if (i < n && LSTM_CHECK_INDEX(src - a.xch + i * 64 * 8 * V + V - 1, 2 * set_words, a.status)) ld_words<V>(src + i * 64 * 8 * V, w[i]);
    };
    auto wait_words = [&](const unsigned *src, int n, unsigned (&w)[KW][V]) {
        auto missing = [&]() {
            unsigned all = kPhaseBit;
#pragma unroll
            for (int i = 0; i < KW; ++i)
#pragma unroll
                for (int t = 0; t < NT; ++t) all &= w[i][t] | (t < nrows ? 0u : kPhaseBit);
            return all == 0u;
        };
        int polls = 0;
        long long t_start = 0;
        while (missing() && !*abort_v) {
            request(src, n, w);
            if ((++polls & 15) == 0) {
                const long long now = clock64();
                if (t_start == 0) t_start = now;
                if (now - t_start > a.spin_limit || ld_volatile_s32(a.status) != kStatusOk) {
                    *abort_v = 1;
                    atomicExch(a.status, kStatusTimeout);
                }
            }
        }
        __syncwarp();
    };
    // the words as values; groups this lane has nothing of keep the phase bit, which is no value
    auto strip = [&](unsigned (&w)[KW][V], unsigned (&v)[KW][NT]) {
        float top = 0.0f;
#pragma unroll
        for (int i = 0; i < KW; ++i)
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                v[i][t] = w[i][t] & ~kPhaseBit;
                top = fmaxf(top, fabsf(__uint_as_float(v[i][t])));
            }
        if (top > kMaskedNan)
#pragma unroll
            for (int i = 0; i < KW; ++i)
#pragma unroll
                for (int t = 0; t < NT; ++t)
                    if (fabsf(__uint_as_float(v[i][t])) > kMaskedNan) nan_s[8 * t + rr] = 1;
        __syncwarp();
    };
    unsigned wx[KW][V], wh[KW][V];
#pragma unroll
    for (int i = 0; i < KW; ++i)
#pragma unroll
        for (int t = 0; t < V; ++t) wx[i][t] = wh[i][t] = kPhaseBit;
    const unsigned *below_l = below + (size_t)col * (8 * V) + rr * V, *own_l = own + (size_t)col * (8 * V) + rr * V;
    // x_t goes through shared memory: an operand's eight rows are eight lines, which a load of its own would take one by one
    const bool x16 = (Kx & 3) == 0 && (reinterpret_cast<size_t>(a.x) & 15) == 0;
    auto request_x = [&](int s) {
        if (l) return request(below_l + (size_t)s * slot_words, lane_x, wx);
        const float *src = a.x + (size_t)s * B * Kx;
        float *dst = xs + (s & 1) * B * XP;
        if (x16) {
            const int n4 = Kx >> 2;
            for (int i = tid; i < B * n4; i += kThreads) {
                const int b = i / n4, k = i - b * n4;
                cp_async_16(dst + b * XP + 4 * k, src + 4 * (size_t)i);
            }
        } else
            for (int i = tid; i < B * Kx; i += kThreads) {
                const int b = i / Kx, k = i - b * Kx;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst + b * XP + k)), "l"(src + i) : "memory");
            }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (l == 0)
        for (int i = tid; i < 2 * B * XP; i += kThreads) xs[i] = 0.0f;                  // columns beyond the input's width
    __syncthreads();
    request_x(0);
    if (l == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

#pragma unroll 1
    for (int s = 0; s < T; ++s) {
        double acc[MT][NT][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int t = 0; t < NT; ++t) acc[mt][t][0] = acc[mt][t][1] = 0.0;
        // (a jump into the sequence of groups: under a condition of its own a group becomes predicated instructions, and a tensor
        // instruction that is predicated off takes its four cycles all the same)
        auto group = [&](const double *wf, int i, const unsigned (&w)[KW][NT]) {
            double f[MT];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) f[mt] = wf[i * kWStep + mt * 32];
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const double b = (double)__uint_as_float(w[i][t]);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) mma_f64(acc[mt][t], f[mt], b);
            }
        };
        auto products = [&](const double *wf, int kn, const unsigned (&w)[KW][NT]) {
            static_assert(KW == 5, "one case per group");
            switch (kn) {
                case 5: group(wf, 4, w);
                case 4: group(wf, 3, w);
                case 3: group(wf, 2, w);
                case 2: group(wf, 1, w);
                case 1: group(wf, 0, w);
                default: break;
            }
        };
        // ---- x_t or h_t of the layer below
        unsigned v[KW][NT];
        if (l) {
            wait_words(below_l + (size_t)s * slot_words, lane_x, wx);
            strip(wx, v);
        } else {
#pragma unroll
            for (int i = 0; i < KW; ++i)
                if (i < kxn) {
#pragma unroll
                    for (int t = 0; t < NT; ++t) v[i][t] = t < nrows ? __float_as_uint(xs[((s & 1) * B + 8 * t + rr) * XP + col + 64 * i]) : 0u;
                }
        }
        products(wxs, kxn, v);
        // ---- h_{t-1}
        if (s > 0) {
            const unsigned *src = own_l + (size_t)(s - 1) * slot_words;
            request(src, lane_h, wh);
            wait_words(src, lane_h, wh);
            strip(wh, v);
        } else {
#pragma unroll
            for (int i = 0; i < KW; ++i)
#pragma unroll
                for (int t = 0; t < NT; ++t)
                    v[i][t] = a.h0 && i < lane_h && t < nrows ? __float_as_uint(a.h0[((size_t)l * B + 8 * t + rr) * H + col + 64 * i]) : 0u;
            __syncwarp();
        }
        if (s + 1 < T) request_x(s + 1);
        products(whs, khn, v);
        if (LSTM_CHECK_INDEX(((warp * MT + MT - 1) * 8 + rr) * P + (NT - 1) * 8 + 2 * (lane & 3) + 1, f32_wave_red_doubles(NT, MT), a.status)) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int t = 0; t < NT; ++t)
                    *reinterpret_cast<double2 *>(red + ((warp * MT + mt) * 8 + rr) * P + t * 8 + 2 * (lane & 3)) = make_double2(acc[mt][t][0], acc[mt][t][1]);
        }
        __syncthreads();
        if (fin) {
            double z4[4] = {bias, 0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 0; k < kWarps; ++k) z4[k & 3] += rp[k * 8 * MT * P];
            double z = (z4[0] + z4[1]) + (z4[2] + z4[3]);
            if (nan_s[fb]) z = nan("");
            const double act = gate_f64(z, act_k, act_sc, act_of);
            const int ql = lane & ~3;
            const double vi = __shfl_sync(0xffffffffu, act, ql), vf = __shfl_sync(0xffffffffu, act, ql + 1);
            const double vg = __shfl_sync(0xffffffffu, act, ql + 2), vo = __shfl_sync(0xffffffffu, act, ql + 3);
            const double cn = fma(vf, (double)c, vi * vg);
            hn = (float)(vo * gate_f64(cn, -2.0, 2.0, -1.0));
            c = (float)cn;
            if (live && fq == 0 && (int)blockIdx.x != a.withhold_cta && LSTM_CHECK_INDEX(out - own + (size_t)s * slot_words, layer_words, a.status))
                st_relaxed_u32(out + (size_t)s * slot_words, __float_as_uint(hn) | kPhaseBit);
        }
        if (l == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                    // nobody polls before the CTA has published; the sums are free again, x_{t+1} is there
        if (write_y) *yp = hn;
        yp += (size_t)B * H;
    }
    if (live && fq == 2 && a.hT) a.hT[so] = hn;
    if (live && fq == 3 && a.cT) a.cT[so] = c;
}

typedef void (*KernelFn)(const RecurF32WaveArgs);
KernelFn pick(int nt, int mt)
{
    static const KernelFn one[4] = {recur_f32_wave_kernel<1, 1>, recur_f32_wave_kernel<2, 1>, recur_f32_wave_kernel<3, 1>, recur_f32_wave_kernel<4, 1>};
    static const KernelFn two[4] = {recur_f32_wave_kernel<1, 2>, recur_f32_wave_kernel<2, 2>, recur_f32_wave_kernel<3, 2>, recur_f32_wave_kernel<4, 2>};
    return (mt == 1 ? one : two)[nt - 1];
}
size_t smem_bytes(int in_dim, int H, int nt, int mt)
{
    const int kx = (in_dim > H ? in_dim : H) + 3;
    return ((size_t)(kx / 4 + (H + 3) / 4) * mt * 32 + f32_wave_red_doubles(nt, mt)) * 8 + (size_t)2 * 8 * nt * f32_wave_x_pitch(in_dim) * 4;
}

}  // namespace

// Units per CTA so that all layers' CTAs fit the device at once, or 0: whole tiles of two units, four units at most (2 x 200, 20 rows:
// 161 us with three units on 67 CTAs a layer and 162 with four on 50 in the first form of this kernel; four leave the words with fewer readers).
int recur_f32_wave_units(int L, int H, int in_dim, int max_cta)
{
    if (L < 2 || L > kMaxWaveLayers || H > kF32MaxUnits || in_dim > kF32MaxUnits) return 0;
    for (int u = 2; u <= 4; u += 2)
        if (L * ((H + u - 1) / u) <= max_cta) return u;
    return 0;
}

// The limit is a property of the kernel, not of a handle: the most the device has, or a handle made later for less would lower it.
cudaError_t recur_f32_wave_prepare(int upc, int max_B, int smem_optin)
{
    for (int nt = 1; nt <= 4 && 8 * (nt - 1) < max_B; ++nt) {
        const cudaError_t e = cudaFuncSetAttribute(pick(nt, (upc + 1) / 2), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - kStaticSmem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

size_t recur_f32_wave_smem_bytes(const RecurF32WaveArgs &a) { return smem_bytes(a.in_dim, a.H, (a.B + 7) / 8, (a.upc + 1) / 2); }

cudaError_t launch_recur_f32_wave(const RecurF32WaveArgs &a, cudaStream_t st)
{
    if (a.B < 1 || a.B > kF32MaxRows || a.T > a.slots) return cudaErrorInvalidValue;
    const int nt = (a.B + 7) / 8, mt = (a.upc + 1) / 2;
    RecurF32WaveArgs copy = a;
    void *params[] = {&copy};
    return cudaLaunchCooperativeKernel((const void *)pick(nt, mt), dim3(a.L * a.ncta), dim3(kThreads), params, recur_f32_wave_smem_bytes(a), st);
}

}  // namespace lstm

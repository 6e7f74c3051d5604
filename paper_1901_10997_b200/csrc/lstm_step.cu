// One timestep of one LSTM layer (T = 1, bf16 dense weights, up to eight batch rows): the call of a program that generates
// token by token and carries the state itself.
//     z = b + Wx x + Wh h;  i,f,o = sigmoid(z_i,z_f,z_o), g = tanh(z_g);  c' = f c + i g;  h' = o tanh(c')
// There is nothing to exchange between CTAs and no weight is used twice, so what bounds it is the one read of both weight
// matrices from HBM (36 MB per layer at 1500 -> 1500: 5.5 us at 6.55 TB/s).  A plain launch of the recurrent kernel spends
// its time on the fragments' residency, one tile ahead, and on the cooperative launches.  Here every CTA requests its
// whole slice into L2 at once, then streams the same operand-A fragments the recurrent kernel keeps (mma.m16n8k16, up to
// eighteen 16-byte loads in flight a lane), and two CTAs fit an SM, so that with programmatic dependent launch the next
// layer's (or the next call's) requests leave while this layer finishes: what a kernel reads of its predecessor it
// reads behind griddepcontrol.wait, weights before it.  A layer above the first also multiplies Wh h0 before the wait:
// the layer below lets it start only after its own wait, i.e. when everything before the call is complete.
// Measured (2 x 1500, one sequence, per call of the binding): 49.1 us as two cooperative launches, 23.1 us here (27.6 with
// every load behind the wait).  Eight rows here / nine in two cooperative launches of the batched kernel: 2 x 64 14.5 / 25 us,
// 2 x 300 16 / 32, 2 x 700 18 / 37, 2 x 1500 35 / 47, 2 x 2000 59 / 97.
#include "common.cuh"
#include "device_util.cuh"

#include <cstring>

namespace lstm {
namespace {

constexpr int kThreads = kStepThreads, kWarps = kThreads / 32;

// MT: 16-row tiles of the CTA (4 gate rows x units).  RB: batch rows the operand is laid out for: up to 4 rows put their hi
// and lo planes into adjacent columns, 8 take one column each and two instructions a tile.
template <int MT, int RB>
__global__ void __launch_bounds__(kThreads, 2) lstm_step_kernel(const LstmStepArgs a)
{
    constexpr int U = MT == 1 ? 12 : MT == 2 ? 8 : MT == 3 ? 6 : 4;     // column tiles in flight
    constexpr int RP = MT * 16 + (RB == 8 ? 4 : 8), WS = RB * RP;       // partial sums [warp][row][RP]: no bank conflicts
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, tig = lane & 3;
    const int H = a.H, B = a.B, D = a.D;
    const int d = blockIdx.x / a.ncta_dir, cta = blockIdx.x % a.ncta_dir;
    int u0, nu;
    unit_range(H, a.ncta_dir, cta, u0, nu);
    const uint4 *fx = a.xfrag[d] + (size_t)cta * a.x_tiles * MT * 32, *fh = a.hfrag[d] + (size_t)cta * a.h_tiles * MT * 32;
    // the whole slice into L2
    for (int i = tid; i < a.h_tiles * MT * 4; i += kThreads)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(fh) + (size_t)i * 128));
    for (int i = tid; i < a.x_tiles * MT * 4; i += kThreads)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(fx) + (size_t)i * 128));
    if (!a.first) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int xk = a.x_tiles * 16, hk = a.h_tiles * 16;                 // columns of the staged operands, zero beyond the real ones
    unsigned *oph = reinterpret_cast<unsigned *>(smem);                 // [RB][hk + 16] words {bf16 hi | bf16 lo}
    unsigned *opx = oph + RB * (hk + 16);                               // [RB][xk + 16]
    float *red = reinterpret_cast<float *>(opx + RB * (xk + 16));       // [kWarps][RB][RP]
    LSTM_CHECK_SMEM_END(reinterpret_cast<unsigned char *>(red + kWarps * WS) - smem, a.status);

    float acc[MT][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[mt][e] = 0.0f;
    // columns of h: the recurrent fragments hold columns 2 tig, 2 tig + 1, 2 tig + 8, 2 tig + 9 of a tile in this lane, the
    // input fragments 4 tig .. 4 tig + 3
    const int brow = RB == 8 ? g : RB == 1 ? 0 : g >> 1;
    const unsigned sel = RB != 8 && (g & 1) ? 0x5410u : 0x7632u;
    auto stage = [&](unsigned *op, const float *src, long long row_stride, int n, int ncol) {
#pragma unroll
        for (int b = 0; b < RB; ++b)
            for (int k0 = tid; k0 < ncol; k0 += 8 * kThreads) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = b < B && k0 + i * kThreads < n ? src[b * row_stride + k0 + i * kThreads] : 0.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (k0 + i * kThreads < ncol && LSTM_CHECK_INDEX(&op[b * (ncol + 16) + k0 + i * kThreads] - oph, reinterpret_cast<unsigned *>(red) - oph, a.status))
                        op[b * (ncol + 16) + k0 + i * kThreads] = split_word(v[i]);
            }
    };
    // a warp takes every kWarps-th column tile, U of them in flight
    uint4 af[U][MT];
    auto load = [&](const uint4 *frag, int tiles, int t0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                af[u][mt] = t0 + kWarps * u < tiles ? ld_nc_u4(frag + (size_t)((t0 + kWarps * u) * MT + mt) * 32 + lane) : make_uint4(0, 0, 0, 0);
    };
    // products of all tiles of a matrix whose first U are loaded; ends with the first U of `next` on their way
    auto products = [&](const unsigned *op, int pitch, const uint4 *frag, int tiles, bool adjacent, const uint4 *next, int next_tiles) {
        const unsigned *ow = op + brow * pitch + (adjacent ? 4 : 2) * tig;
        const int second = adjacent ? 2 : 8;
#pragma unroll 1
        for (int t0 = warp; t0 < tiles; t0 += kWarps * U) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (t0 + kWarps * u < tiles && LSTM_CHECK_INDEX(ow + (t0 + kWarps * u) * 16 + second + 1 - oph, reinterpret_cast<unsigned *>(red) - oph, a.status)) {
                    const uint2 w0 = *reinterpret_cast<const uint2 *>(ow + (t0 + kWarps * u) * 16);
                    const uint2 w1 = *reinterpret_cast<const uint2 *>(ow + (t0 + kWarps * u) * 16 + second);
                    const unsigned b0 = __byte_perm(w0.x, w0.y, sel), b1 = __byte_perm(w1.x, w1.y, sel);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt], af[u][mt], b0, b1);
                    if (RB == 8) {
                        const unsigned l0 = __byte_perm(w0.x, w0.y, 0x5410u), l1 = __byte_perm(w1.x, w1.y, 0x5410u);
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) mma_bf16(acc[mt], af[u][mt], l0, l1);
                    }
                }
            const bool more = t0 + kWarps * U < tiles;
            if (more || next) load(more ? frag : next, more ? tiles : next_tiles, more ? t0 + kWarps * U : warp);
        }
    };
    // What depends on the kernel before this one is read behind the wait: for the first layer both operands, above it x.
    const bool with_h = a.h0 != nullptr;
    load(with_h ? fh : fx, with_h ? a.h_tiles : a.x_tiles, warp);
    if (a.first) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        stage(opx, a.X, a.in_l, a.in_l, xk);
    }
    if (with_h) {
        stage(oph, a.h0 + (size_t)d * B * H, H, H, hk);
        __syncthreads();
        products(oph, hk + 16, fh, a.h_tiles, false, fx, a.x_tiles);
    }
    if (!a.first) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        stage(opx, a.X, a.in_l, a.in_l, xk);
    }
    __syncthreads();
    products(opx, xk + 16, fx, a.x_tiles, true, nullptr, 0);

    float *rw = red + warp * WS + g;
    if (!LSTM_CHECK_INDEX(rw - red + (RB == 8 ? 7 : RB - 1) * RP + (MT - 1) * 16 + 8, kWarps * WS, a.status)) {
    } else if (RB == 8) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            rw[2 * tig * RP + mt * 16] = acc[mt][0];
            rw[(2 * tig + 1) * RP + mt * 16] = acc[mt][1];
            rw[2 * tig * RP + mt * 16 + 8] = acc[mt][2];
            rw[(2 * tig + 1) * RP + mt * 16 + 8] = acc[mt][3];
        }
    } else if (tig < RB) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            rw[tig * RP + mt * 16] = acc[mt][0] + acc[mt][1];
            rw[tig * RP + mt * 16 + 8] = acc[mt][2] + acc[mt][3];
        }
    }
    __syncthreads();
    // a quad per (unit, batch row): one gate each, then all four update the state and deal out the stores
    const int fq = lane & 3;
    const float act_k = (fq == 2 ? -2.0f : -1.0f) * 1.4426950408889634f, act_sc = fq == 2 ? 2.0f : 1.0f, act_of = fq == 2 ? -1.0f : 0.0f;
    for (int i0 = 0; i0 < nu * B; i0 += kThreads / 4) {
        const int item = i0 + (tid >> 2), b = item / nu, u = item - b * nu, j = u0 + u;
        const bool live = item < nu * B;
        float z = 0.0f;
        if (live) {
            z = a.bias[((size_t)d * H + j) * 4 + fq];
            const float *rp = red + b * RP + 4 * u + fq;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) z += rp[w * WS];
        }
        const float act = gate_fast(z, act_k, act_sc, act_of);
        const int q0 = lane & ~3;
        const float vi = __shfl_sync(0xffffffffu, act, q0), vf = __shfl_sync(0xffffffffu, act, q0 + 1);
        const float vg = __shfl_sync(0xffffffffu, act, q0 + 2), vo = __shfl_sync(0xffffffffu, act, q0 + 3);
        if (live) {
            const size_t so = ((size_t)d * B + b) * H + j;
            const float cn = fmaf(vf, a.c0 ? a.c0[so] : 0.0f, vi * vg);
            const float hn = vo * tanh_fast(cn);
            if (fq == 0) a.y[(size_t)b * D * H + (size_t)d * H + j] = hn;
            else if (fq == 1 && a.hT) a.hT[so] = hn;
            else if (fq == 2 && a.cT) a.cT[so] = cn;
        }
    }
}

typedef void (*KernelFn)(const LstmStepArgs);
template <int MT> KernelFn pick_rows(int B) { return B == 1 ? lstm_step_kernel<MT, 1> : B <= 4 ? lstm_step_kernel<MT, 4> : lstm_step_kernel<MT, 8>; }
KernelFn pick(int mt, int B)
{
    switch (mt) {
        case 1: return pick_rows<1>(B);
        case 2: return pick_rows<2>(B);
        case 3: return pick_rows<3>(B);
        case 4: return pick_rows<4>(B);
        default: return nullptr;
    }
}

}  // namespace

size_t lstm_step_smem_bytes(int mt, int B, int x_tiles, int h_tiles)
{
    const int rb = B == 1 ? 1 : B <= 4 ? 4 : 8;
    return (size_t)rb * ((x_tiles + h_tiles) * 16 + 32) * 4 + (size_t)kWarps * rb * (mt * 16 + 8) * 4;
}

cudaError_t lstm_step_prepare(int mt, int max_smem)
{
    for (int B = 1; B <= kStepMaxRows; B = B == 1 ? 4 : 2 * B) {
        KernelFn fn = pick(mt, B);
        if (!fn) return cudaErrorInvalidValue;
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_lstm_step(const LstmStepArgs &a, int mt, cudaStream_t st)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(a.ncta_dir * a.D); cfg.blockDim = dim3(kThreads); cfg.stream = st;
    cfg.dynamicSmemBytes = lstm_step_smem_bytes(mt, a.B, a.x_tiles, a.h_tiles);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, pick(mt, a.B), a);
}

}  // namespace lstm

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
#include "recur_tc_role.cuh"

#include <cstdio>
#include <cstring>

namespace lstm {
namespace {

template <int RG, bool PAIR, int TERMS, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1) recur_tc_kernel(const RecurTcArgs a)
{
    recur_tc_role<RG, PAIR, TERMS, 1, kTcAlone, SPLIT>(a, blockIdx.x, TcLink());
}

typedef void (*KernelFn)(const RecurTcArgs);
template <bool PAIR, int TERMS>
KernelFn pick_p(int rg, bool split)
{
    switch (rg) {
        case 1: return split ? recur_tc_kernel<1, PAIR, TERMS, true> : recur_tc_kernel<1, PAIR, TERMS, false>;
        case 2: return split ? recur_tc_kernel<2, PAIR, TERMS, true> : recur_tc_kernel<2, PAIR, TERMS, false>;
        case 3: return recur_tc_kernel<3, PAIR, TERMS, false>;
        case 4: return recur_tc_kernel<4, PAIR, TERMS, false>;
        case 5: return recur_tc_kernel<5, PAIR, TERMS, false>;
        case 6: return recur_tc_kernel<6, PAIR, TERMS, false>;
        case 7: return recur_tc_kernel<7, PAIR, TERMS, false>;
        case 8: return recur_tc_kernel<8, PAIR, TERMS, false>;
        default: return nullptr;
    }
}
KernelFn pick(int rg, bool pair, int terms, bool split)
{
    return terms == 3 ? (pair ? pick_p<true, 3>(rg, split) : pick_p<false, 3>(rg, split)) : (pair ? pick_p<true, 2>(rg, split) : pick_p<false, 2>(rg, split));
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

// (the builds that calls of up to `rows` sequences can reach)
cudaError_t recur_tc_prepare(int terms, int rows, int max_smem)
{
    for (int rg = 1; rg <= groups_of(rows < kTcMaxRows ? rows : kTcMaxRows); ++rg) {
        for (int v = 0; v < (rg <= 2 ? 4 : 2); ++v) {
            const cudaError_t e = cudaFuncSetAttribute(pick(rg, (v & 1) != 0, terms, v >= 2), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
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
    if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)pick(groups_of(p.rows), true, p.terms, false), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters * 2 >= grid;
}

cudaError_t launch_recur_tc(const RecurTcArgs &a, cudaStream_t st)
{
    KernelFn fn = pick(groups_of(a.B), a.pair != 0, a.terms, a.nsplit > 1);
    if (!fn) return cudaErrorInvalidValue;
    RecurTcArgs copy = a;
    void *params[] = {&copy};
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = config(attr, a.ncta_dir * (a.ndirs ? a.ndirs : a.D), recur_tc_smem_bytes(a.KH, a.upc, a.B, a.pair, a.terms), a.pair, st);
    return cudaLaunchKernelExC(&cfg, (const void *)fn, params);
}

}  // namespace lstm

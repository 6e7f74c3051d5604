// Two stacked layers of a batch in one launch (paper, Section 5.1: the language model is two stacked recurrent layers): the upper
// layer's recurrence runs some timesteps behind the lower one's, on SMs of its own, instead of after it.  A recurrence is bound by
// the latency of its step and not by the SMs it runs on, so T steps plus the lag take little more than half of 2 T.
//
// Three groups of CTAs: the lower layer's and the upper layer's recurrence, each the CTA pairs of recur_tc.cu with its weights
// resident (up to 192 accumulator rows a pair: the first 128 from tensor memory, the others from shared memory), and
// between them the CTAs of stack_proj.cuh, which turn a chunk of timesteps of the lower layer's h into rows of the upper layer's G.
// All three of the matrices do not fit the chip at 1500 x 1500; the one without a recurrence is streamed once per chunk.
// Measured (us per call, one after the other -> here): 2 x 517, 3 rows, T = 23 128 -> 81; 2 x 1000, 8 rows, T = 35 206 -> 134; 2 x 1500, 20
// rows, T = 35 289 -> 254; pruned, 16 rows 286 -> 233.  At 1500 and 20 rows a step takes 5.1 us (products 2650 clocks: 47 of 128 and
// 47 of 64 rows at N = 48) and a chunk of four steps 22 us of the projecting CTAs, whose products are bound by shared memory:
// 167 KB a K block, weights once in and once out, activations once in and three times out.
// The groups meet through counts in global memory, one per chunk: "planes of X stored" and "rows of G stored".
// All CTAs of the launch are resident (cooperative launch); every wait is bounded.
#include "recur_tc_role.cuh"
#include "stack_proj.cuh"

#include <algorithm>
#include <cstring>

namespace lstm {
namespace {

template <int RG, int TERMS, int MB, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
recur_stack_kernel(const __grid_constant__ RecurStackArgs a, const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                   const __grid_constant__ CUtensorMap tmap_xlo)
{
    extern __shared__ __align__(16) unsigned char smem_stack[];
    // the other set of exchange words and counts, for the next launch
    for (unsigned i = blockIdx.x * kThreads + threadIdx.x; i < a.clear_words / 4u; i += gridDim.x * kThreads)
        reinterpret_cast<uint4 *>(a.other_set)[i] = make_uint4(0, 0, 0, 0);
    const int n = a.layer[0].ncta_dir, b = blockIdx.x;
    if (b < n) recur_tc_role<RG, true, TERMS, MB, kTcLower, SPLIT>(a.layer[0], b, TcLink{a.chunk, a.proj.stored_out, nullptr, 0});
    else if (b < 2 * n) recur_tc_role<RG, true, TERMS, MB, kTcUpper, false>(a.layer[1], b - n, TcLink{a.chunk, nullptr, a.proj.ready, (unsigned)(gridDim.x - 2 * n)});
    else stack_proj_role(smem_stack, &tmap_w, &tmap_x, &tmap_xlo, a.proj, b - 2 * n);
}

// Rows packed for one partition into pairs (recur_tc.cu's) as another one wants them; the K halves are the same.
__global__ void repartition_kernel(const uint4 *src, int src_upc, uint4 *dst, int dst_upc, int H, int pieces, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int rows = 8 * dst_upc, row = (int)(i % rows), piece = (int)(i / rows % pieces), cta = (int)(i / rows / pieces);
        const int u = (cta >> 1) * 2 * dst_upc + (row >> 2), pair = u / (2 * src_upc);
        dst[i] = u < H ? src[((long long)(2 * pair + (cta & 1)) * pieces + piece) * (8 * src_upc) + (u - pair * 2 * src_upc) * 4 + (row & 3)] : make_uint4(0, 0, 0, 0);
    }
}

typedef void (*KernelFn)(const RecurStackArgs, const CUtensorMap, const CUtensorMap, const CUtensorMap);
template <int TERMS, int MB> KernelFn pick_m(int rg, bool split)
{
    switch (rg) {
        case 1: return split ? recur_stack_kernel<1, TERMS, MB, true> : recur_stack_kernel<1, TERMS, MB, false>;
        case 2: return split ? recur_stack_kernel<2, TERMS, MB, true> : recur_stack_kernel<2, TERMS, MB, false>;
        case 3: if constexpr (TERMS == 2) return recur_stack_kernel<3, TERMS, MB, false>; else return nullptr;
        case 4: if constexpr (TERMS == 2) return recur_stack_kernel<4, TERMS, MB, false>; else return nullptr;
        default: return nullptr;
    }
}
KernelFn pick(int rg, int terms, int mb, bool split)
{
    return terms == 3 ? (mb == 2 ? pick_m<3, 2>(rg, split) : pick_m<3, 1>(rg, split)) : (mb == 2 ? pick_m<2, 2>(rg, split) : pick_m<2, 1>(rg, split));
}
int groups_of(int rows) { return (rows + 7) / 8; }
int blocks_of(int upc) { return 8 * upc > 128 ? 2 : 1; }

size_t role_smem(int KH, int upc, int rows, int terms)
{
    const int rg = groups_of(rows), tiles = (KH + 63) / 64;
    return 1024 + (size_t)tiles * (std::max(0, 8 * upc - 128) + tc_columns(rg, terms)) * 128 + (size_t)2 * 8 * upc * tc_rows_of_first(rg, true) * 4;
}
constexpr size_t kProjFixedSmem = 1024 + 120 * 128;            // alignment; the last block of a stage is read as 128 rows
size_t proj_smem(const StackProjArgs &a) { return kProjFixedSmem + (size_t)a.stages * (a.mb * a.rb + 2 * a.nrp) * 128; }

cudaLaunchConfig_t config(cudaLaunchAttribute (&attr)[2], int grid, size_t smem, cudaStream_t st)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return cfg;
}

}  // namespace

size_t recur_stack_smem_bytes(const RecurTcPlan &p, int rows, const StackProjArgs &a) { return std::max(role_smem(p.KH, p.upc, rows, p.terms), proj_smem(a)); }

// Partition of a stack whose calls have up to rows_wanted rows: CTA pairs of each layer, the others project; *ctas: all of them.
// Narrow layers take no more CTAs than they gain from: up to 296 units the launches of two handles and more fit the chip at once when
// the layers run one after the other, and so they do here: pairs of 24 units, about 72 rows of G on a projecting CTA.  us per call with 1, 2,
// 3, 6 handles on streams of their own, T = 35, one layer after the other; side by side on all SMs; on these CTAs: H = 128 with 8 rows 131, 67, 46,
// 32; 96, 82, 82, 81; 93, 49, 33, 19 (32 CTAs); 200 with 20 181, 91, 73, 73; 120, 107, 103, 103; 122, 61, 43, 36 (48); 296 with 32 207, 105, 98, 95;
// 134, 120, 119, 118; 132, 67, 59, 60 (70).  One handle against all SMs: 65 to 296 units, 5 to 32 rows, T = 4 to 70 0.92 - 1.02.  Eight projecting
// CTAs at 296: up to 1.10 at T = 4; pairs of 32 units 1.03 with 32 rows; 400 units with pairs of 24 1.06 with 8 rows.
// Wider ones take the fewest units per CTA that leave 16 CTAs to project, and all SMs: 592 units with 8, 20, 32 rows on 16 units and 108 CTAs 118, 146, 157,
// on 8 and all 116, 144, 153; 517 on 16 units and 92 CTAs 116, 144, 153, on 8 and all 116, 146, 155.  Without the 16: 1000 on 136 CTAs 204, 298,
// 413, on 148 134, 179, 200.
bool recur_stack_plan(int H, int max_cta, int rows_wanted, int terms, size_t max_smem, RecurTcPlan *p, int *ctas)
{
    if (H <= 64) return false;
    const bool narrow = H <= kStackNarrow;
    const int min_proj = narrow ? std::max(8, (4 * H + 143) / 144 * 2) : kStackMinProj;
    const int KH = ((H + 1) / 2 + 15) / 16 * 16;
    for (int upc = narrow ? 12 : 4; upc <= 24; upc += 4) {
        const int n = (H + 2 * upc - 1) / (2 * upc) * 2, mb = blocks_of(upc);
        if (2 * n + min_proj > max_cta / 2 * 2) continue;
        for (int rg = std::min(terms == 3 ? 2 : 4, groups_of(rows_wanted)); rg >= 1; --rg) {
            const int acc = mb == 2 ? 2 * tc_columns(rg, terms) : tc_acc_columns(rg, terms);
            if (KH / 2 + acc > 512 || KH > 16 * kPollers * kMaxGroups || role_smem(KH, upc, 8 * rg, terms) > max_smem) continue;
            p->upc = upc; p->ncta = n; p->KH = KH; p->pair = 1; p->rows = 8 * rg; p->terms = terms;
            *ctas = narrow ? 2 * n + min_proj : max_cta / 2 * 2;
            return true;
        }
    }
    return false;
}

cudaError_t launch_repartition(const uint4 *src, const RecurTcPlan &from, uint4 *dst, const RecurTcPlan &to, int H, cudaStream_t st)
{
    const long long n = (long long)to.ncta * (to.KH / 8) * 8 * to.upc;
    repartition_kernel<<<(int)std::min<long long>((n + 255) / 256, 4096), 256, 0, st>>>(src, from.upc, dst, to.upc, H, to.KH / 8, n);
    return cudaGetLastError();
}

cudaError_t recur_stack_prepare(const RecurTcPlan &p, int ctas, int max_smem, bool *fits)
{
    *fits = false;
    for (int v = 0; v < p.rows / 8 + std::min(2, p.rows / 8); ++v) {
        KernelFn fn = v < p.rows / 8 ? pick(v + 1, p.terms, blocks_of(p.upc), false) : pick(v + 1 - p.rows / 8, p.terms, blocks_of(p.upc), true);
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
        // (each build takes all of an SM's registers and, here, of its shared memory: one answer for all of them)
        if (v > 0) continue;
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = config(attr, ctas, max_smem, nullptr);
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)fn, &cfg) != cudaSuccess) { cudaGetLastError(); clusters = 0; }
        *fits = clusters >= ctas / 2;
    }
    return cudaSuccess;
}

// Rows, blocks and chunk of the projecting CTAs of a call; false when there is no room for one timestep.  Four timesteps a chunk, as far as
// tensor memory holds its accumulators: fewer cannot keep up with the recurrences at the wider layers, more make the lag longer.  us per
// call at 2, 3, 4, 5, 6 timesteps: 2 x 1500, T = 35, 2 rows 249, 191, 187, 192, 189; 20 rows 320, 273, 259 (no room for five); 1000
// with 24 rows 208, 185, 181, 181, 179; 517 with 8 126, 120, 118, 117, 118; 700, T = 20, 6 rows 89, 87, 85, 85, 87; 517, T = 23, 3
// rows 93, 89, 89, 89, 90; 300 with 16 124, 122, 120, 122, 120; pruned 1500 with 16 300, 253, 251, 259, 257.
bool recur_stack_proj_plan(const RecurTcPlan &p, int H, int T, int B, int ctas, size_t max_smem, StackProjArgs *a, int *chunk)
{
    const int nproj = ctas - 2 * p.ncta;
    a->M = T * B; a->N = 4 * H; a->kblocks = (H + 63) / 64;
    const int rows = (a->N + nproj - 1) / nproj;
    a->mb = (rows + 127) / 128;
    a->rb = ((rows + a->mb - 1) / a->mb + 7) / 8 * 8;
    a->nrp = 0;
    for (int c = 1; c <= std::min(4, T); ++c) {
        const int nrp = (c * B + 7) / 8 * 8;
        if (nrp > 128 || a->mb * 2 * nrp > 512) break;
        a->nrp = nrp;
        a->chunk_rows = c * B;
        *chunk = c;
    }
    if (a->nrp == 0) return false;
    a->nchunks = (T + *chunk - 1) / *chunk;
    a->stages = std::min(kSpStages, (int)((max_smem - kProjFixedSmem) / ((a->mb * a->rb + 2 * a->nrp) * 128)));
    return a->stages >= 2 && a->nchunks <= kStackMaxChunks;
}

bool stack_proj_maps(StackProjMaps *m, const __nv_bfloat16 *W, const __nv_bfloat16 *X, const __nv_bfloat16 *Xlo, const StackProjArgs &a, int K, int ldk, int ldx)
{
    return encode_tmap_bf16_2d(m->w, W, a.N, K, ldk, a.rb) && encode_tmap_bf16_2d(m->x, X, a.M, K, ldx, a.nrp) &&
           encode_tmap_bf16_2d(m->xlo, Xlo, a.M, K, ldx, a.nrp);
}

cudaError_t launch_recur_stack(const RecurStackArgs &a, const StackProjMaps &maps, const RecurTcPlan &p, int ctas, cudaStream_t st)
{
    KernelFn fn = pick(groups_of(a.layer[0].B), p.terms, blocks_of(p.upc), a.layer[0].nsplit > 1);
    if (!fn) return cudaErrorInvalidValue;
    RecurStackArgs copy = a;
    StackProjMaps m = maps;
    void *params[] = {&copy, m.w, m.x, m.xlo};
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = config(attr, ctas, recur_stack_smem_bytes(p, a.layer[0].B, a.proj), st);
    return cudaLaunchKernelExC(&cfg, (const void *)fn, params);
}

}  // namespace lstm

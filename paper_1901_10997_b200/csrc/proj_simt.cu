// Input staging and the CUDA-core forms of the input projection G = X Wx^T + b (the x_t half of
// W [x_t, h_{t-1}] + b in the paper's Section 4 cell equations, hoisted out of the time loop and
// computed for all timesteps at once).  The fp32 storage type uses the tiled FFMA kernel; pruned
// weights in CSR form use the sparse kernel.  The bf16 tensor-core kernel lives in proj_tc.cu.
#include "common.cuh"
#include "device_util.cuh"

#include <algorithm>

namespace lstm {
namespace {

// A block takes whole rows, a thread four columns at a time (ld is a multiple of eight): 16-byte loads where the rows of x allow
// them, 8-byte stores.  Bound by memory: one element
// at a time with a 64-bit division each took 30 us for 6400 rows of 1312 (67 MB) and 23 for 3500 of 1500, this 16 and 14.
template <bool VEC>
__global__ void __launch_bounds__(128) stage_bf16_kernel(const float *__restrict__ x, __nv_bfloat16 *__restrict__ xb, long long plane,
                                                         long long M, int K, int ld)
{
    for (long long m = blockIdx.x; m < M; m += gridDim.x) {
        const float *row = x + m * K;
        __nv_bfloat16 *out = xb + m * ld;
        for (int k = 4 * (int)threadIdx.x; k < ld; k += 4 * 128) {
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (VEC) {
                if (k < K) v = *reinterpret_cast<const float4 *>(row + k);
            } else {
                if (k < K) v.x = row[k];
                if (k + 1 < K) v.y = row[k + 1];
                if (k + 2 < K) v.z = row[k + 2];
                if (k + 3 < K) v.w = row[k + 3];
            }
            const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
            const __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - __low2float(h0), v.y - __high2float(h0));
            const __nv_bfloat162 l1 = __floats2bfloat162_rn(v.z - __low2float(h1), v.w - __high2float(h1));
            uint2 hi, lo;
            hi.x = *reinterpret_cast<const uint32_t *>(&h0); hi.y = *reinterpret_cast<const uint32_t *>(&h1);
            lo.x = *reinterpret_cast<const uint32_t *>(&l0); lo.y = *reinterpret_cast<const uint32_t *>(&l1);
            *reinterpret_cast<uint2 *>(out + k) = hi;
            *reinterpret_cast<uint2 *>(out + plane + k) = lo;
        }
    }
}

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// 64x64 output tile, K step 16, 256 threads, 4x4 outputs per thread.
template <typename WT>
__global__ void __launch_bounds__(256) proj_simt_kernel(const float *__restrict__ X, const WT *__restrict__ W,
                                                        int ldw, const float *__restrict__ bias,
                                                        float *__restrict__ G, int M, int N, int K)
{
    __shared__ float xs[16][64 + 4];
    __shared__ float ws[16][64 + 4];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int tm = (tid / 16) * 4, tn = (tid % 16) * 4;
    typedef float AT;
    AT acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = (AT)0;

    for (int k0 = 0; k0 < K; k0 += 16) {
        // each thread loads 4 elements of each tile: row r = tid/4 (0..63), k = (tid%4)*4 .. +3
        const int r = tid >> 2, kk = (tid & 3) * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + kk + i;
            xs[kk + i][r] = (m0 + r < M && k < K) ? X[(size_t)(m0 + r) * K + k] : 0.0f;
            ws[kk + i][r] = (n0 + r < N && k < K) ? to_f32(W[(size_t)(n0 + r) * ldw + k]) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            float xv[4], wv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { xv[i] = xs[k][tm + i]; wv[i] = ws[k][tn + i]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma((AT)xv[i], (AT)wv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + tm + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tn + j;
            if (n < N) G[(size_t)m * N + n] = (float)(acc[i][j] + (AT)(bias ? bias[n] : 0.0f));
        }
    }
}

// fp32 storage: sums in fp64 on the double-precision tensor instruction.  32 x 32 output tile, K step 16, four warps of 2 x 2
// m8n8 tiles.  What bounds it is the fp64 rate (64 multiply-adds per clock and SM) once the operands are converted as they
// are stored instead of at every use and a lane's operands are single conflict-free loads; the next K step is on its way
// while this one is multiplied, and small tiles put several CTAs on an SM.  2000 x 800 x 200: 83 us with the fp64
// multiply-adds of the tile kernel above, 50 us here.
__global__ void __launch_bounds__(128) proj_f64_kernel(const float *__restrict__ X, const float *__restrict__ W, int ldw,
                                                       const float *__restrict__ bias, float *__restrict__ G, int M, int N, int K)
{
    constexpr int P = 36;                                      // doubles between K rows: a half warp's 4 x 4 operands hit all banks
    __shared__ double xs[2][16][P], ws[2][16][P];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * 32, n0 = blockIdx.y * 32, wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
    const int r = tid >> 2, kk = (tid & 3) * 4;                // this thread loads 4 adjacent elements of row r of each tile
    const bool xok = m0 + r < M, wok = n0 + r < N;
    const bool vec = (K & 3) == 0 && (ldw & 3) == 0 && ((reinterpret_cast<size_t>(X) | reinterpret_cast<size_t>(W)) & 15) == 0;
    const float *xp = X + (size_t)(m0 + r) * K + kk, *wp = W + (size_t)(n0 + r) * ldw + kk;
    float4 xn, wv;
    auto load = [&](const float *p, bool ok, int k0) -> float4 {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (ok) {
            const int left = K - k0 - kk;
            if (vec) { if (left > 0) v = *reinterpret_cast<const float4 *>(p + k0); }
            else {
                if (left > 0) v.x = p[k0];
                if (left > 1) v.y = p[k0 + 1];
                if (left > 2) v.z = p[k0 + 2];
                if (left > 3) v.w = p[k0 + 3];
            }
        }
        return v;
    };
    double acc[2][2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
    xn = load(xp, xok, 0);
    wv = load(wp, wok, 0);
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += 16, buf ^= 1) {
        xs[buf][kk][r] = xn.x; xs[buf][kk + 1][r] = xn.y; xs[buf][kk + 2][r] = xn.z; xs[buf][kk + 3][r] = xn.w;
        ws[buf][kk][r] = wv.x; ws[buf][kk + 1][r] = wv.y; ws[buf][kk + 2][r] = wv.z; ws[buf][kk + 3][r] = wv.w;
        __syncthreads();                                       // (two buffers: the one read two steps ago is written next)
        if (k0 + 16 < K) { xn = load(xp, xok, k0 + 16); wv = load(wp, wok, k0 + 16); }
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
            double a[2], b[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                a[i] = xs[buf][k + (lane & 3)][wm + 8 * i + (lane >> 2)];
                b[i] = ws[buf][k + (lane & 3)][wn + 8 * i + (lane >> 2)];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) mma_f64(acc[i][j], a[i], b[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int m = m0 + wm + 8 * i + (lane >> 2), n = n0 + wn + 8 * j + 2 * (lane & 3) + e;
                if (m < M && n < N) G[(size_t)m * N + n] = (float)(acc[i][j][e] + (double)(bias ? bias[n] : 0.0f));
            }
}

// CSR projection: a CTA stages MT = 8 activation rows (transposed so that the 8 values of one column
// are contiguous) and its warps walk CSR rows; lanes stride over a row's entries.
constexpr int kCsrMT = 8;
constexpr int kCsrUnroll = 8;
template <typename AT>
__global__ void __launch_bounds__(256) proj_csr_kernel(const float *__restrict__ X, const int *__restrict__ rowptr,
                                                       const CsrEntry *__restrict__ ent,
                                                       const float *__restrict__ bias, float *__restrict__ G,
                                                       int M, int N, int K, int rows_per_cta)
{
    extern __shared__ __align__(16) float xt[];          // [K][8]
    const int m0 = blockIdx.y * kCsrMT;
    // a thread fetches one column of all eight rows at once (eight loads in flight, coalesced over the
    // threads) and stores them as the 32 contiguous bytes the row walk reads back
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        float v[kCsrMT];
#pragma unroll
        for (int mm = 0; mm < kCsrMT; ++mm) v[mm] = (m0 + mm < M) ? X[(size_t)(m0 + mm) * K + k] : 0.0f;
        *reinterpret_cast<float4 *>(xt + (size_t)k * kCsrMT) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4 *>(xt + (size_t)k * kCsrMT + 4) = make_float4(v[4], v[5], v[6], v[7]);
    }
    __syncthreads();
    // Rows are short (a few dozen to a few hundred survivors), so a warp walks four rows at once, eight
    // lanes each: four times as many independent trips to memory are in flight per warp, and the
    // reduction runs over eight lanes instead of thirty-two.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int sub = lane & 7, grp = lane >> 3;
    const int r_begin = blockIdx.x * rows_per_cta;
    const int r_end = min(N, r_begin + rows_per_cta);
    for (int rb = r_begin + warp * 4; rb < r_end; rb += nwarps * 4) {
        const int r = rb + grp;
        const bool live = r < r_end;
        AT acc[kCsrMT];
#pragma unroll
        for (int i = 0; i < kCsrMT; ++i) acc[i] = (AT)0;
        const int e_begin = live ? rowptr[r] : 0;
        const int e_end = live ? rowptr[r + 1] : 0;
        for (int e0 = e_begin + sub; e0 < e_end; e0 += 8 * kCsrUnroll) {
            CsrEntry en[kCsrUnroll];
#pragma unroll
            for (int u = 0; u < kCsrUnroll; ++u) {
                const int e = e0 + 8 * u;
                en[u] = e < e_end ? ent[e] : CsrEntry{0.0f, 0};
            }
#pragma unroll
            for (int u = 0; u < kCsrUnroll; ++u) {
                const float4 a = *reinterpret_cast<const float4 *>(xt + (size_t)en[u].col * kCsrMT);
                const float4 b = *reinterpret_cast<const float4 *>(xt + (size_t)en[u].col * kCsrMT + 4);
                const AT v = (AT)en[u].val;
                acc[0] = fma(v, (AT)a.x, acc[0]); acc[1] = fma(v, (AT)a.y, acc[1]);
                acc[2] = fma(v, (AT)a.z, acc[2]); acc[3] = fma(v, (AT)a.w, acc[3]);
                acc[4] = fma(v, (AT)b.x, acc[4]); acc[5] = fma(v, (AT)b.y, acc[5]);
                acc[6] = fma(v, (AT)b.z, acc[6]); acc[7] = fma(v, (AT)b.w, acc[7]);
            }
        }
#pragma unroll
        for (int i = 0; i < kCsrMT; ++i)
#pragma unroll
            for (int o = 4; o >= 1; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        if (live && m0 + sub < M) {
            AT v = (AT)0;
#pragma unroll
            for (int i = 0; i < kCsrMT; ++i) v = (sub == i) ? acc[i] : v;
            G[(size_t)(m0 + sub) * N + r] = (float)(v + (AT)(bias ? bias[r] : 0.0f));
        }
    }
}

__global__ void proj_export_kernel(const float *__restrict__ G, int nsplit, long long split_stride,
                                   float *__restrict__ out, long long M, int D, int Hg)
{
    const long long total = M * D * 4 * Hg;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        // i enumerates the public layout [m][d][q][j]
        const int j = (int)(i % Hg);
        const int q = (int)((i / Hg) % 4);
        const long long md = i / (4 * Hg);
        const long long src = (md * Hg + j) * 4 + q;
        float v = 0.0f;
        for (int sp = 0; sp < nsplit; ++sp) v += G[sp * split_stride + src];
        out[i] = v;
    }
}

}  // namespace

cudaError_t launch_proj_export(const float *G, int nsplit, long long split_stride, float *out, long long M, int D, int Hg,
                               cudaStream_t st)
{
    const long long total = M * D * 4 * Hg;
    if (total == 0) return cudaSuccess;
    long long blocks = (total + 255) / 256;
    if (blocks > 148LL * 16) blocks = 148LL * 16;
    proj_export_kernel<<<(int)blocks, 256, 0, st>>>(G, nsplit, split_stride, out, M, D, Hg);
    return cudaGetLastError();
}

cudaError_t launch_stage_bf16(const float *x, __nv_bfloat16 *xb, long long plane, long long M, int K, int ld,
                              cudaStream_t st)
{
    if (M == 0 || ld == 0) return cudaSuccess;
    const int blocks = (int)std::min(M, 148LL * 16);
    if (K % 4 == 0 && ((uintptr_t)x & 15) == 0) stage_bf16_kernel<true><<<blocks, 128, 0, st>>>(x, xb, plane, M, K, ld);
    else stage_bf16_kernel<false><<<blocks, 128, 0, st>>>(x, xb, plane, M, K, ld);
    return cudaGetLastError();
}

cudaError_t launch_proj_simt(const float *X, const void *W, bool bf16, int ldw, const float *bias,
                             float *G, int M, int N, int K, cudaStream_t st)
{
    if (M == 0 || N == 0) return cudaSuccess;
    dim3 grid((N + 63) / 64, (M + 63) / 64);
    if (bf16)
        proj_simt_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(X, (const __nv_bfloat16 *)W, ldw, bias, G, M, N, K);
    else
        // rows in x, which may have 2^31 blocks; y may have 65535 (columns: at most 2 x 4 x 65535 / 32)
        proj_f64_kernel<<<dim3((M + 31) / 32, (N + 31) / 32), 128, 0, st>>>(X, (const float *)W, ldw, bias, G, M, N, K);
    return cudaGetLastError();
}

cudaError_t proj_csr_prepare(int max_smem)
{
    cudaError_t e = cudaFuncSetAttribute(proj_csr_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(proj_csr_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
}

cudaError_t launch_proj_csr(const float *X, const int *rowptr, const CsrEntry *ent, const float *bias,
                            float *G, int M, int N, int K, bool f64_acc, cudaStream_t st)
{
    if (M == 0 || N == 0) return cudaSuccess;
    const size_t smem = (size_t)K * kCsrMT * sizeof(float);
    const int mtiles = (M + kCsrMT - 1) / kCsrMT;
    int ctas_x = max(1, (148 * 4) / mtiles);      // about four CTAs per SM: a warp walks few rows, one trip to memory each
    int rows_per_cta = max(8, (N + ctas_x - 1) / ctas_x);
    ctas_x = (N + rows_per_cta - 1) / rows_per_cta;
    dim3 grid(ctas_x, mtiles);
    if (f64_acc) proj_csr_kernel<double><<<grid, 256, smem, st>>>(X, rowptr, ent, bias, G, M, N, K, rows_per_cta);
    else proj_csr_kernel<float><<<grid, 256, smem, st>>>(X, rowptr, ent, bias, G, M, N, K, rows_per_cta);
    return cudaGetLastError();
}

}  // namespace lstm

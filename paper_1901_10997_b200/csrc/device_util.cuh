// Device-side helpers shared by the kernels of the lstm_b200 library: the stamped-word exchange
// primitives, named barriers, the warp-level tensor instruction, the gate functions, and the
// mbarrier / TMA / tcgen05 wrappers of the two tensor-core kernels, plus the host-side tensor-map
// encoder.  One definition each, so that a fix to a descriptor or a fence is made once.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace lstm {

// ---------------------------------------------------------------------------------------------------
// Checked build (-DLSTM_B200_CHECKED): the stand-in for a memory checker.  Index and carve-up checks compile
// into the kernels; a violation records kStatusInternal in the status word (reported as LSTM_ERR_INTERNAL) and
// the access is skipped -- nothing traps, nothing reads or writes out of range.  In the normal build the macros
// vanish.
// ---------------------------------------------------------------------------------------------------
constexpr int kStatusInternal = 6;
__device__ __forceinline__ unsigned dynamic_smem_bytes()
{
    unsigned v;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
    return v;
}
#ifdef LSTM_B200_CHECKED
__device__ __forceinline__ bool check_index(long long i, long long n, int *status)
{
    if (i >= 0 && i < n) return true;
    atomicCAS(status, 0, kStatusInternal);
    return false;
}
#define LSTM_CHECK_INDEX(i, n, status) lstm::check_index((long long)(i), (long long)(n), (status))
// end_bytes: bytes of dynamic shared memory the kernel is about to carve up (or read as an operand)
#define LSTM_CHECK_SMEM_END(end_bytes, status) \
    do { if ((unsigned long long)(end_bytes) > (unsigned long long)lstm::dynamic_smem_bytes()) atomicCAS((status), 0, lstm::kStatusInternal); } while (0)
#else
#define LSTM_CHECK_INDEX(i, n, status) true
#define LSTM_CHECK_SMEM_END(end_bytes, status) do { } while (0)
#endif

// ---------------------------------------------------------------------------------------------------
// global-memory accesses of the exchange
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_relaxed_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u32(unsigned *p, unsigned v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// ---------------------------------------------------------------------------------------------------
// Exchange words: one hidden value in 32 bits, {bf16 hi : 16 | bf16 lo : 16} with hi = bf16(h), lo = bf16(h - hi), the
// two terms the tensor cores multiply.  |h| = |o tanh(c)| <= 1, so bit 30 (the top exponent bit of hi) is always 0 in a
// value and carries a PHASE instead: step s writes slot s & 1 with phase bit 1 ^ (s >> 1 & 1), so a slot's phase flips
// every time it is rewritten and a consumer that polls the word itself can tell new from old.  A slot is reused two
// steps later, when its writer has seen every other CTA's words of the step between, i.e. when all have read it.  A NaN
// keeps its lo term (a NaN), so it still reaches every product.
// ---------------------------------------------------------------------------------------------------
constexpr unsigned kPhaseBit = 0x40000000u;
__device__ __forceinline__ unsigned word_phase(int s) { return ((s >> 1) & 1) ? 0u : kPhaseBit; }
__device__ __forceinline__ unsigned split_word(float h)
{
    const __nv_bfloat16 hi = __float2bfloat16_rn(h), lo = __float2bfloat16_rn(h - __bfloat162float(hi));
    return ((unsigned)__bfloat16_as_ushort(hi) << 16) | (unsigned)__bfloat16_as_ushort(lo);
}
__device__ __forceinline__ unsigned pack_word(float h, unsigned phase) { return (split_word(h) & ~kPhaseBit) | phase; }
// Exchange words that carry h as its own 32 bits (narrow fp32 layers, pruned layers): without bit 30 a NaN reads as 1.5 or more,
// which no h is (a fast tanh may pass 1 by a rounding): its reader puts the bit back or marks the batch row.
constexpr float kMaskedNan = 1.25f;
__device__ __forceinline__ bool words_ready(const uint4 &w, unsigned phase)
{
    return (((w.x ^ phase) | (w.y ^ phase) | (w.z ^ phase) | (w.w ^ phase)) & kPhaseBit) == 0;
}
__device__ __forceinline__ uint4 ld_relaxed_v4(const unsigned *p)
{
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_nc_u4(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ int ld_volatile_s32(const int *p)
{
    int v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// read-only loads that the compiler may not sink towards their use: issued early, consumed a step later
__device__ __forceinline__ float ld_nc_early(const float *p)
{
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// 16-byte asynchronous copy global -> shared through L2 only (never a stale L1 line)
__device__ __forceinline__ void cp_async_16(void *smem_dst, const void *gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// named barriers over n threads of the CTA
__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
// ... and was the condition true for all of them?
__device__ __forceinline__ bool bar_all(int id, int n, bool ok)
{
    int all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.s32 p, %3, 0;\n\t"
        "barrier.cta.red.and.pred q, %1, %2, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(all) : "r"(id), "r"(n), "r"((int)ok) : "memory");
    return all != 0;
}
__device__ __forceinline__ void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// D += A (8x4, row) * B (4x8, col) in double precision
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}
// D += A (16x16, row) * B (16x8, col), bf16 inputs, fp32 accumulation
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint4 &a, unsigned b0, unsigned b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------------------------------
// Gate functions from the fast exponential: absolute error of a few 1e-7, far inside the 2e-2 bound of the
// bf16 storage type.  Both are one expression, sc / (1 + 2^(-k log2(e) z)) + of: the logistic function with
// (k, sc, of) = (1, 1, 0) and tanh z = 2 logistic(2z) - 1 with (2, 2, -1): one exponential and one
// reciprocal on the path from the summed pre-activation to the published h.
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ float ex2_fast(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float gate_fast(float z, float neg_k_log2e, float sc, float of)
{
    return fmaf(sc, __fdividef(1.0f, 1.0f + ex2_fast(neg_k_log2e * z)), of);
}
__device__ __forceinline__ float sigmoid_fast(float z) { return __fdividef(1.0f, 1.0f + ex2_fast(-1.4426950408889634f * z)); }
__device__ __forceinline__ float tanh_fast(float z) { return fmaf(2.0f, __fdividef(1.0f, 1.0f + ex2_fast(-2.8853900817779268f * z)), -1.0f); }

// sc / (1 + e^(k z)) + of: the logistic function (k, sc, of = -1, 1, 0) or tanh (-2, 2, -1).  tanh of a small z is the
// difference of two nearby numbers there, which loses the digits of z (all of them near 1e-16): below 1e-4 it is z - z^3 / 3
// (off by less than 2 z^4 / 15 of it).  expm1 in place of both costs 0.4 us a step.
__device__ __forceinline__ double gate_f64(double z, double k, double sc, double of)
{
    double act = sc / (1.0 + exp(k * z)) + of;
    if (of != 0.0 && (__double2hiint(z) & 0x7fffffff) < 0x3f1a36e2) act = fma(z * z, z * (-1.0 / 3.0), z);       // |z| < 1e-4
    return act;
}

// hidden units [u0, u0 + n) of CTA c when H units are split evenly over nc CTAs
__host__ __device__ __forceinline__ void unit_range(int H, int nc, int c, int &u0, int &n)
{
    const int base = H / nc, rem = H % nc;
    n = base + (c < rem ? 1 : 0);
    u0 = c * base + (c < rem ? c : rem);
}

// ---------------------------------------------------------------------------------------------------
// mbarrier, TMA and tcgen05 wrappers
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
constexpr long long kMbarWaitTicks = 4000000000ll;   // clock64 ticks an mbarrier wait may last (about two seconds)
// Bounded wait.  Returns false when it gave up (or another role did): the caller leaves its loop.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    long long t_start = 0;
    for (long long it = 0;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255) == 255) {
            if (*abort_flag) return false;
            const long long now = clock64();
            if (t_start == 0) t_start = now;
            if (now - t_start > kMbarWaitTicks) break;
        }
    }
    *abort_flag = 1;
    return false;
}
// One lane of a converged warp.  The thread that issues tensor-core instructions must be chosen like this, and its operands be
// warp-uniform: the same loop entered by "lane == 0" issues one in 170 cycles instead of 20.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p)::"memory");
    return p != 0;
}
// tiled TMA load of one box into this CTA's shared memory (no multicast: every CTA fetches its own tiles)
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, uint32_t bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y) : "memory");
}
// K-major operand tile in shared memory, 128-byte swizzle: rows of 128 bytes, groups of 8 rows are
// 1024 bytes apart (stride byte offset); version field = 1 for this architecture.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3ffffu) >> 4);          // start address, bits [0,14)
    d |= (uint64_t)1 << 16;                                 // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                       // stride byte offset, bits [32,46)
    d |= (uint64_t)1 << 46;                                 // descriptor version
    d |= (uint64_t)2 << 61;                                 // layout type: 128-byte swizzle
    return d;
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}

// ---------------------------------------------------------------------------------------------------
// Host: tensor map of a row-major bf16 matrix [rows][ld] of which `cols` columns are valid, boxes of
// box_rows x 64 columns, 128-byte swizzle, zero fill outside.  The driver entry point is looked up through
// the runtime, so the library links against the runtime only.
// ---------------------------------------------------------------------------------------------------
inline bool encode_tmap_bf16_2d(void *map128, const void *base, long long rows, long long cols, long long ld, int box_rows)
{
    typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                 const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || !p) return false;
        fn = (EncodeFn)p;
    }
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1u, 1u};
    return fn((CUtensorMap *)map128, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace lstm

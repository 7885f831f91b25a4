// gwam_gemm.cu -- tcgen05 / TMA BF16 GEMM with fused epilogues (see gwam_gemm.cuh) and its
// self-test entry point.
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "gwam_df.cuh"
#include "gwam_gemm.cuh"

namespace gwam {

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr uint32_t kABytes = kBM * kBK * 2;          // 16 KB per stage
constexpr unsigned long long kWaitNs = 2000000000ull; // 2 s per wait

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t gtime()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounded wait for completion of the mbarrier phase with the given parity; false if it gave up
// (after limit_ns of %globaltimer time, or 2^31 polls)
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns)
{
    uint64_t t0 = 0;
    for (uint32_t it = 0; it < 0x7fffffffu; ++it) {
        uint32_t done;
        if (CLUSTER)   // arrivals of another CTA of the cluster
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                " selp.u32 %0, 1, 0, p;\n}"
                : "=r"(done)
                : "r"(bar), "r"(parity)
                : "memory");
        else
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                : "=r"(done)
                : "r"(bar), "r"(parity)
                : "memory");
        if (done) return true;
        if ((it & 63u) == 0) {
            const uint64_t t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) return false;
        }
    }
    return false;
}

__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor of a 128-byte swizzled K-major tile: start address >> 4,
// leading offset 16 B (unused for swizzled K-major), stride 1024 B between 8-row groups,
// descriptor version 1, swizzle mode 2 (128 B)
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A BF16 (bits 7-9 = 1), B BF16
// (bits 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Phi(z) = (1 + erf(z / sqrt 2)) / 2 with erf by Abramowitz & Stegun, Handbook of Mathematical
// Functions, formula 7.1.26 (absolute error <= 1.5e-7): for x = |z| / sqrt 2 >= 0,
// erf(x) = 1 - t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-x^2), t = 1 / (1 + p x).
// erf_abs returns erf(|z| / sqrt 2) and exp(-z^2 / 2); 1/sqrt 2 is folded into p, and exp(-z^2/2)
// = 2^(-z^2 log2(e) / 2).  Hardware reciprocal and base-2 exponential approximations (PTX
// rcp.approx / ex2.approx, relative errors near 2^-23 and 2^-22).
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float erf_abs(float z, float& e)
{
    const float t = rcp_approx(fmaf(0.23164189961f, fabsf(z), 1.0f));   // p / sqrt 2, p = 0.3275911
    float poly = fmaf(t, 1.061405429f, -1.453152027f);
    poly = fmaf(t, poly, 1.421413741f);
    poly = fmaf(t, poly, -0.284496736f);
    poly = fmaf(t, poly, 0.254829592f);
    e = ex2_approx(z * z * -0.72134752044f);                             // -log2(e) / 2
    return fmaf(-(t * poly), e, 1.0f);
}

// GELU(z) = z Phi(z) = z / 2 + |z| erf(|z| / sqrt 2) / 2 of two values in packed instructions (half the issue slots); the steps
// of erf_abs, with the polynomial's coefficients negated for its negated value.
__device__ __forceinline__ float2 gelu2(float2 z)
{
    const float2 az = make_float2(fabsf(z.x), fabsf(z.y));
    const float2 d = fma2(dup2(0.23164189961f), az, dup2(1.0f));
    const float2 t = make_float2(rcp_approx(d.x), rcp_approx(d.y));
    float2 p = fma2(t, dup2(-1.061405429f), dup2(1.453152027f));
    p = fma2(t, p, dup2(-1.421413741f));
    p = fma2(t, p, dup2(0.284496736f));
    p = fma2(t, p, dup2(-0.254829592f));
    const float2 q = mul2(mul2(z, z), dup2(-0.72134752044f));
    const float2 r = fma2(mul2(t, p), make_float2(ex2_approx(q.x), ex2_approx(q.y)), dup2(1.0f));
    return fma2(mul2(az, dup2(0.5f)), r, mul2(z, dup2(0.5f)));
}

// GELU'(z) = Phi(z) + z phi(z), phi(z) = exp(-z^2 / 2) / sqrt(2 pi)
__device__ __forceinline__ float gelu_grad(float z)
{
    float e;
    const float r = erf_abs(z, e);
    return fmaf(z * 0.39894228040143268f, e, fmaf(0.5f, copysignf(r, z), 0.5f));
}

// Sum of the squares of 32 errors, as accurate as the FP64 sum and over its whole range.  FP64 additions and
// conversions of every element (1/72 of the FP32 rate) had made this kernel 55 us: the exact products
// (hi, lo) go into unevaluated sums of three FP32 numbers, even and odd columns in the halves of packed pairs, the
// errors of the two larger ones carried into the next, and only the results are added in FP64 (relative error about
// 2^-53; a double-float sum, 48 bits, was 1e-14 off after 64 elements).  Where FP32 cannot hold the products to that
// -- an error beyond 2^60, a sum below 2^-90, infinities -- every one is formed in FP64.
__device__ __forceinline__ double sum_squares(const float (&d)[32])
{
    float2 s0 = dup2(0.0f), s1 = s0, s2 = s0;
    float most = 0.0f;
    auto two_sum = [](float2& s, float2 x) {
        const float2 t = add2(s, x), b = sub2(t, s);
        const float2 e = add2(sub2(s, sub2(t, b)), sub2(x, b));
        s = t;
        return e;
    };
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        const DF p = df_prod(d[j], d[j]), q = df_prod(d[j + 1], d[j + 1]);
        const float2 e = two_sum(s0, make_float2(p.hi, q.hi));
        const float2 f = two_sum(s1, e);
        s2 = add2(s2, add2(f, two_sum(s1, make_float2(p.lo, q.lo))));
        most = fmaxf(most, fmaxf(fabsf(d[j]), fabsf(d[j + 1])));
    }
    if (most <= 0x1p60f && (s0.x + s0.y >= 0x1p-90f || most == 0.0f))
        return (widen(s0.x) + widen(s0.y)) + ((widen(s1.x) + widen(s1.y)) + widen(s2.x + s2.y));
    double q = 0.0;
#pragma unroll
    for (int j = 0; j < 32; ++j) q = fma((double)d[j], (double)d[j], q);
    return q;
}

// Epilogue of 32 consecutive accumulator columns n = nb .. nb+31 of one row.  The columns' bias comes from
// shared memory (sbias), behind it EPI_DRAG's sigma and mu where they fit beside the stages (not at 8192
// outputs); EPI_DRAG_WIDE loads them from global memory (inference of 32 768 columns 121
// and 124 us).  Rows >= M only skip the stores.  zz: the prefetched
// pre-activations of EPI_BWD.
template <int MODE>
__device__ __forceinline__ void epi32(const GemmEpi& e, int row, int nb, float (&v)[32], const float* sbias,
                                      const float (&zz)[32], int rowmask, double& sq, uint32_t stg,
                                      int cc0)
{
    const bool live = row < e.M;
    const bool full = nb + 32 <= e.N;
    if (MODE == EPI_BWD) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] *= gelu_grad(zz[j]);
    } else {
        if (e.bias) {
            // the tile's bias from shared memory (zero beyond N), broadcast to every lane
            const float4* bp = reinterpret_cast<const float4*>(sbias + nb);
#pragma unroll
            for (int qq = 0; qq < 8; ++qq) {
                const float4 b = bp[qq];
                v[4 * qq] += b.x;
                v[4 * qq + 1] += b.y;
                v[4 * qq + 2] += b.z;
                v[4 * qq + 3] += b.w;
            }
        }
        if (MODE == EPI_DRAG || MODE == EPI_DRAG_WIDE) {
            const int npad = (e.N + 31) & ~31;
            // de-normalised in FP32 (one FMA, relative error 6e-8, far below the BF16 network's) and
            // widened exactly by integer operations: FP64 arithmetic and float -> double conversions
            // run at 1/72 of the FP32 rate on GB300
            if (!live || rowmask != 0) return;
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 s4 = MODE == EPI_DRAG ? *reinterpret_cast<const float4*>(sbias + npad + nb + j)
                                                   : __ldg(reinterpret_cast<const float4*>(e.ysig + nb + j));
                const float4 m4 = MODE == EPI_DRAG ? *reinterpret_cast<const float4*>(sbias + 2 * npad + nb + j)
                                                   : __ldg(reinterpret_cast<const float4*>(e.ymu + nb + j));
                const float sj[4] = {s4.x, s4.y, s4.z, s4.w}, mj[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int n = nb + j + u;
                    if (n < e.n_true) {
                        const double y = gwam::widen(__fmaf_rn(v[j + u], sj[u], mj[u]));
                        if (n < e.nlev) e.du[(size_t)n * e.ncol + row] = y;
                        else e.dv[(size_t)(n - e.nlev) * e.ncol + row] = y;
                    }
                }
            }
            return;
        }
        if (!live) return;
        if (MODE == EPI_STORE) {
            if (e.z) {
                float* p = e.z + (size_t)row * e.ldz + nb;
                if (full && (e.ldz & 3) == 0) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        reinterpret_cast<float4*>(p)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (nb + j < e.N) p[j] = v[j];
                }
            }
            if (e.act) {
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    const float2 g = gelu2(make_float2(v[j], v[j + 1]));
                    v[j] = g.x;
                    v[j + 1] = g.y;
                }
            }
        } else {  // EPI_LOSS
            if (e.cf) {
                float* p = e.cf + (size_t)row * e.ldcf + nb;
                if (full && (e.ldcf & 3) == 0) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        reinterpret_cast<float4*>(p)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (nb + j < e.N) p[j] = v[j];
                }
            }
            const float* tg = e.tgt + (size_t)row * e.ldt + nb;
            float tp[32];
            if (full && (e.ldt & 3) == 0) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 t4 = reinterpret_cast<const float4*>(tg)[q];
                    tp[4 * q] = t4.x;
                    tp[4 * q + 1] = t4.y;
                    tp[4 * q + 2] = t4.z;
                    tp[4 * q + 3] = t4.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) tp[j] = nb + j < e.n_true ? tg[j] : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = nb + j < e.n_true ? v[j] - tp[j] : 0.0f;
            sq += sum_squares(v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = e.gscale * v[j];
        }
    }
    if (!live) return;
    if (MODE == EPI_STORE && e.cf) {
        float* p = e.cf + (size_t)row * e.ldcf + nb;
        if (full && (e.ldcf & 3) == 0) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                reinterpret_cast<float4*>(p)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (nb + j < e.N) p[j] = v[j];
        }
    }
    if (e.cb && stg) {
        // this row's 64 bytes into the warp's 128-byte-swizzled staging box (16-byte chunk c of
        // row r at r * 128 + ((c ^ (r % 8)) * 16)); a TMA store writes the box out
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
            w[q] = *reinterpret_cast<const uint32_t*>(&h);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t a = stg + ((uint32_t)((cc0 + q) ^ (row & 7)) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(w[4 * q]), "r"(w[4 * q + 1]),
                         "r"(w[4 * q + 2]), "r"(w[4 * q + 3])
                         : "memory");
        }
    } else if (e.cb) {
        __nv_bfloat16* p = e.cb + (size_t)row * e.ldcb + nb;
        if (full && (e.ldcb & 7) == 0) {
            uint32_t w[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                w[q] = *reinterpret_cast<const uint32_t*>(&h);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                reinterpret_cast<uint4*>(p)[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (nb + j < e.N) p[j] = __float2bfloat16_rn(v[j]);
        }
    }
    if (e.ct) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (nb + j < e.N) e.ct[(size_t)(nb + j) * e.ldct + row] = __float2bfloat16_rn(v[j]);
    }
}

// 32 accumulator columns of this warp's 32 TMEM lanes, one row a lane
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&rr)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(rr[0]), "=r"(rr[1]), "=r"(rr[2]), "=r"(rr[3]), "=r"(rr[4]), "=r"(rr[5]), "=r"(rr[6]), "=r"(rr[7]),
          "=r"(rr[8]), "=r"(rr[9]), "=r"(rr[10]), "=r"(rr[11]), "=r"(rr[12]), "=r"(rr[13]), "=r"(rr[14]), "=r"(rr[15]),
          "=r"(rr[16]), "=r"(rr[17]), "=r"(rr[18]), "=r"(rr[19]), "=r"(rr[20]), "=r"(rr[21]), "=r"(rr[22]),
          "=r"(rr[23]), "=r"(rr[24]), "=r"(rr[25]), "=r"(rr[26]), "=r"(rr[27]), "=r"(rr[28]), "=r"(rr[29]),
          "=r"(rr[30]), "=r"(rr[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 columns likewise
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&rr)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(rr[0]), "=r"(rr[1]), "=r"(rr[2]), "=r"(rr[3]), "=r"(rr[4]), "=r"(rr[5]), "=r"(rr[6]), "=r"(rr[7]),
          "=r"(rr[8]), "=r"(rr[9]), "=r"(rr[10]), "=r"(rr[11]), "=r"(rr[12]), "=r"(rr[13]), "=r"(rr[14]), "=r"(rr[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Persistent, warp-specialised GEMM.  Warp 0 (one lane) streams the K blocks of every tile the
// CTA owns through the shared-memory ring; warp 1 allocates TMEM and (one lane) issues the MMAs of
// tile i into accumulator i % 2; warps 2 .. 2+EPW-1 drain accumulator (i % 2) while the MMAs of tile
// i + 1 run into the other one.  Epilogue warp w reads TMEM lane quarter w % 4 and, with EPW / 4
// warps per quarter, its share of the columns.  Tiles t = blockIdx.x, blockIdx.x + gridDim.x, ...
// over (m tile, n tile), n fastest.
template <int BN, int ST, int EPW, int MODE>
__global__ void __launch_bounds__(64 + 32 * EPW, 1)
    k_gemm_bf16(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                const __grid_constant__ CUtensorMap tc, int K, GemmEpi e)
{
    constexpr uint32_t kBBytes = BN * kBK * 2;
    constexpr uint32_t kStage = kABytes + kBBytes;   // a multiple of 1024
    constexpr uint32_t kAccStride = BN <= 64 ? 64 : (BN <= 128 ? 128 : 256);
    constexpr uint32_t kCols = 2 * kAccStride;
    constexpr int kEpiThreads = 32 * EPW;
    constexpr int kColsPerWarp = BN / (EPW / 4);
    static_assert(kColsPerWarp % 64 == 0, "epilogue column share must be a multiple of 64");
    constexpr uint32_t kStgWarp = 32u * kColsPerWarp * 2u;   // BF16 staging of a warp's 32 rows
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[ST], empty_bar[ST], accf_bar[2], acce_bar[2], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_tiles = (e.N + BN - 1) / BN, m_tiles = (e.M + kBM - 1) / kBM;
    const int total = n_tiles * m_tiles;
    const int nk = K / kBK;
    const uint32_t base = (saddr(smem_raw) + 1023u) & ~1023u;

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < ST; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty_bar[s])));
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accf_bar[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(&acce_bar[a])), "r"(kEpiThreads));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&done_bar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    // behind the stage ring: the epilogue warps' BF16 staging boxes (TMA-store mode), then the bias
    // of all N columns, zero-padded to a multiple of 32
    const uint32_t stg_base = base + (uint32_t)ST * kStage;
    float* sbias = reinterpret_cast<float*>(smem_raw + (base - saddr(smem_raw)) + (size_t)ST * kStage +
                                            (e.tstore ? (size_t)EPW * kStgWarp : 0));
    // programmatic dependent launch: the next kernel in the stream may start its own set-up now; this
    // one waits until the previous kernel has completed before it reads anything from global memory
    // (the set-up above touched only shared and tensor memory and the kernel parameters)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (e.bias) {
        const int npad = (e.N + 31) & ~31;
        for (int i = tid; i < npad; i += blockDim.x) {
            sbias[i] = i < e.N ? e.bias[i] : 0.0f;
            if (MODE == EPI_DRAG) {
                sbias[npad + i] = i < e.n_true ? e.ysig[i] : 0.0f;
                sbias[2 * npad + i] = i < e.n_true ? e.ymu[i] : 0.0f;
            }
        }
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = tmem_slot;
    const unsigned long long wlim = e.wait_ns ? e.wait_ns : kWaitNs;
    bool ok = true;
    double sq = 0.0;

    if (warp == 0) {
        if (lane == 0) {
            // TMA producer
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&ta)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tb)) : "memory");
            int it = 0;
            // (self-test of the give-up path: no copy is issued, so the MMA and epilogue warps wait
            // on stages that never fill and give up after wait_ns)
            for (int t = blockIdx.x; t < total && ok && !e.skip_copies; t += gridDim.x) {
                const int m0 = (t / n_tiles) * kBM, n0 = (t % n_tiles) * BN;
                for (int i = 0; i < nk; ++i, ++it) {
                    const int s = it % ST;
                    if (it >= ST && !mbar_wait(saddr(&empty_bar[s]), (uint32_t)((it / ST - 1) & 1), wlim)) {
                        ok = false;
                        break;
                    }
                    if (abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = saddr(&full_bar[s]);
                    const uint32_t dA = base + (uint32_t)s * kStage, dB = dA + kABytes;
                    const int kx = i * kBK;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(kStage)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
                        "{%2, %3}], [%4];" ::"r"(dA),
                        "l"(reinterpret_cast<uint64_t>(&ta)), "r"(kx), "r"(m0), "r"(fb)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
                        "{%2, %3}], [%4];" ::"r"(dB),
                        "l"(reinterpret_cast<uint64_t>(&tb)), "r"(kx), "r"(n0), "r"(fb)
                        : "memory");
                }
            }
            if (!ok) abort_flag = 1;
            // every issued copy has landed before the CTA may exit (immediate in the normal case)
            for (int i = it > ST ? it - ST : 0; i < it; ++i)
                if (!mbar_wait(saddr(&full_bar[i % ST]), (uint32_t)((i / ST) & 1), wlim)) ok = false;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // MMA issuer
            constexpr uint32_t idesc = idesc_bf16(kBM, BN);
            int it = 0, tl = 0;
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++tl) {
                const int acc = tl & 1;
                if (tl >= 2 && !mbar_wait(saddr(&acce_bar[acc]), (uint32_t)((tl / 2 - 1) & 1), wlim)) {
                    ok = false;
                    break;
                }
                tc_after();
                const uint32_t d = tmem + (uint32_t)acc * kAccStride;
                for (int i = 0; i < nk; ++i, ++it) {
                    const int s = it % ST;
                    if (abort_flag || !mbar_wait(saddr(&full_bar[s]), (uint32_t)((it / ST) & 1), wlim)) {
                        ok = false;
                        break;
                    }
                    tc_after();
                    const uint32_t a0 = base + (uint32_t)s * kStage, b0 = a0 + kABytes;
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk) {
                        const uint64_t ad = desc_sw128(a0 + 32u * kk), bd = desc_sw128(b0 + 32u * kk);
                        const uint32_t accum = (i > 0 || kk > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
                            : "memory");
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     saddr(&empty_bar[s]))
                                 : "memory");
                }
                if (!ok) break;
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 saddr(&accf_bar[acc]))
                             : "memory");
            }
            if (!ok) abort_flag = 1;
            // tracks every MMA issued above (also after a give-up): released TMEM is never written
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             saddr(&done_bar))
                         : "memory");
        }
        __syncwarp();
    } else {
        // epilogue warps
        constexpr int kChunks = kColsPerWarp / 32;
        const int q = warp & 3, part = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        int tl = 0;
        for (int t = blockIdx.x; t < total; t += gridDim.x, ++tl) {
            const int acc = tl & 1;
            const int m0 = (t / n_tiles) * kBM, n0 = (t % n_tiles) * BN;
            const int row = m0 + q * 32 + lane;
            const int cbeg = n0 + part * kColsPerWarp;
            const int rowmask = ((MODE == EPI_DRAG || MODE == EPI_DRAG_WIDE) && row < e.M) ? e.mask[row] : 0;
            const bool got = mbar_wait(saddr(&accf_bar[acc]), (uint32_t)((tl / 2) & 1), wlim);
            if (!__all_sync(0xffffffffu, got) || abort_flag) {
                ok = false;
                break;
            }
            tc_after();
            const uint32_t stg_warp = stg_base + (uint32_t)(warp - 2) * kStgWarp;
            if (e.tstore) {
                // the previous tile's TMA store has finished reading this warp's staging boxes
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
            }
            const uint32_t tacc = tmem + lane_base + (uint32_t)acc * kAccStride + (uint32_t)(part * kColsPerWarp);
            // the 32-column chunks as a rolled loop (one copy of the epilogue arithmetic: the epilogue
            // warps stalled on instruction fetch; GEMM chain 0.173 -> 0.165 ms per 32 768 columns)
#pragma unroll 1
            for (int k = 0; k < kChunks; ++k) {
                const int nb = cbeg + 32 * k;
                if (nb >= e.N) break;
                float zz[32];
                if (MODE == EPI_BWD) {
                    // pre-activations in flight while the accumulator is read
                    if (row < e.M && nb + 32 <= e.N && (e.ldz & 3) == 0) {
                        const float4* zp = reinterpret_cast<const float4*>(e.z + (size_t)row * e.ldz + nb);
#pragma unroll
                        for (int qq = 0; qq < 8; ++qq) {
                            const float4 w = zp[qq];
                            zz[4 * qq] = w.x;
                            zz[4 * qq + 1] = w.y;
                            zz[4 * qq + 2] = w.z;
                            zz[4 * qq + 3] = w.w;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            zz[j] = (row < e.M && nb + j < e.N) ? e.z[(size_t)row * e.ldz + nb + j] : 0.0f;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) zz[j] = 0.0f;
                }
                uint32_t rr[32];
                tmem_ld32(tacc + (uint32_t)(32 * k), rr);
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(rr[j]);
                const uint32_t stg =
                    e.tstore ? stg_warp + (uint32_t)((32 * k) / 64) * 4096u + (uint32_t)lane * 128u : 0u;
                epi32<MODE>(e, row, nb, v, sbias, zz, rowmask, sq, stg, ((32 * k) % 64) / 8);
            }
            tc_before();
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&acce_bar[acc])) : "memory");
            if (e.tstore) {
                // staging -> global by TMA (rows and columns outside the tensor are clipped)
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
#pragma unroll
                    for (int b = 0; b < kColsPerWarp / 64; ++b) {
                        const int x = cbeg + 64 * b;
                        if (x < e.N)
                            asm volatile(
                                "cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                    reinterpret_cast<uint64_t>(&tc)),
                                "r"(x), "r"(m0 + q * 32), "r"(stg_warp + (uint32_t)b * 4096u)
                                : "memory");
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
        }
        // this warp's TMA stores have completed before the CTA exits
        if (e.tstore && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
        if (!ok) abort_flag = 1;
        if (MODE == EPI_LOSS) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0 && sq != 0.0) atomicAdd(e.loss, sq);
        }
    }
    // every MMA has finished before the TMEM is released (bounded wait; immediate normally)
    const bool fin = mbar_wait(saddr(&done_bar), 0u, wlim);
    if (!__syncthreads_and(ok && fin) && tid == 0 && e.err) atomicOr(e.err, 1);
    tc_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}

// All hidden layers of the inference (gemm_hidden_launch).  Layer by layer in k_gemm_bf16 a layer of
// 32 768 x 512 x 512 reads 197 MB from L2 (8 TB/s) and takes 26 us where the tensor cores need 9.  Here a
// cluster of C = N / 128 CTAs owns the same rows through all layers, so that a layer needs nothing from other
// clusters and the layers follow one another without a launch between them.  Two CTAs are a pair
// (cta_group::2): 256 rows x 256 columns a tile, each CTA holding its 128 rows of A and 128 of the pair's 256
// rows of W, half of the shared-memory reads that the tile would cost one CTA.  W stays in shared memory
// through a layer (blocks of the next one replace it as the last tile releases them): 94 MB a layer.
// Inference of 32 768 columns through 4 x 512: 121 us, 137 layer by layer.  What bounds it: a tile takes 5 us,
// of them 3.6 the round trips of the four A stages that fit beside W (without any epilogue), the rest
// the epilogue and the wait for the previous layer's stores; multicast of A between the pairs changed nothing.
//
// Warps as in k_gemm_bf16, sixteen of them epilogue (eight: 12 us more).  full, in the pair's first CTA: A (and
// in a layer's first tile W) of a stage has landed in both CTAs; empty: the MMAs have released the stage;
// accf, acce: the accumulator is complete, drained by both CTAs.  done[w]: tiles that an epilogue warp of this
// CTA (or of its counterpart in the other pair) has finished writing to global memory, which the next layer's
// loads wait for.  Every wait is bounded; a CTA that gives up still meets the others at the end.  A pair may then
// have issued different stages: sent tells the first CTA how far each came, which accounts for the bytes that
// never left and waits (bounded) for the others before either leaves.
constexpr int kHidStages = 4;
constexpr int kHidMaxK = 512;
constexpr int kHidEpi = 16;                          // epilogue warps
constexpr uint32_t kHidStgWarp = 32u * 32u * 2u;

__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int C>
__global__ void __launch_bounds__(64 + 32 * kHidEpi, 1) k_hidden(const __grid_constant__ HiddenSet h, int M, int* err)
{
    constexpr int kRows = 2 * kBM, kStages = kHidStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], accf_bar[2], acce_bar[2], done_bar;
    __shared__ uint32_t done[kHidEpi * C / 2];
    __shared__ int sent[3];   // blocks of W loaded ahead; stages; whether all of them have been released
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x % C, cluster = blockIdx.x / C, clusters = gridDim.x / C;
    const int pair = rank >> 1, half = rank & 1, lead = rank & ~1;
    const int tiles = ((M + kRows - 1) / kRows - cluster + clusters - 1) / clusters;   // >= 1 of this cluster
    // W (up to 8 blocks of 16 KB), A stages, staging boxes of the epilogue warps
    const uint32_t wbase = (saddr(smem_raw) + 1023u) & ~1023u;
    const uint32_t abase = wbase + (kHidMaxK / kBK) * kABytes, sbase = abase + kStages * kABytes;
    const unsigned long long wlim = h.wait_ns ? h.wait_ns : kWaitNs;
    const bool mute = (h.skip_copies >> half) & 1;   // self-test: this CTA of the pair issues no copies
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty_bar[s])));
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accf_bar[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(&acce_bar[a])), "r"(2 * kHidEpi));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&done_bar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (tid < kHidEpi * C / 2) done[tid] = 0u;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(saddr(&tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
    tc_before();
    __syncthreads();
    cluster_sync();
    tc_after();
    const uint32_t tmem = tmem_slot;
    // a 64 x 128 box of W or A; its bytes are counted by the barrier of the pair's first CTA
    auto load = [](uint32_t dst, const CUtensorMap& map, int x, int y, uint32_t bar) {
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, "
            "%3}], [%4];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(&map)), "r"(x), "r"(y), "r"(bar)
            : "memory");
    };
    auto expect = [&](int s, uint32_t bytes) {
        if (half == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(&full_bar[s])), "r"(bytes) : "memory");
    };
    // the first blocks of W, while the previous kernel still runs
    const int pre = mute ? 0 : min(kStages, h.nk[0]);
    if (tid == 0)
        for (int i = 0; i < pre; ++i) {
            expect(i, 4 * kABytes);
            load(wbase + (uint32_t)i * kABytes, h.b[0], i * kBK, rank * 128, cluster_addr(saddr(&full_bar[i]), lead));
        }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    bool ok = true;

    if (warp == 0) {
        int it = 0, issued = 0;
        for (int l = 0; l < h.n && ok && !mute; ++l) {
            const int nk = h.nk[l], nkp = l ? h.nk[l - 1] : kStages;
            for (int j = 0; j < tiles && ok; ++j) {
                if (l > 0) {
                    // this tile's rows of the previous layer are in global memory
                    const uint32_t want = (uint32_t)((l - 1) * tiles + j + 1);
                    uint64_t t0 = 0;
                    for (;;) {
                        uint32_t v = want;
                        if (lane < kHidEpi * C / 2)
                            asm volatile("ld.acquire.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(saddr(&done[lane])) : "memory");
                        if (__all_sync(0xffffffffu, v >= want)) break;
                        const uint64_t t = __shfl_sync(0xffffffffu, gtime(), 0);
                        if (t0 == 0) t0 = t;
                        if (t - t0 > wlim || __any_sync(0xffffffffu, abort_flag != 0)) {
                            ok = false;
                            break;
                        }
                    }
                    if (!ok) break;
                    // every lane has acquired its flag; a vote does not order memory, so the warp barrier makes
                    // the rows behind all of them visible to lane 0, whose loads read them
                    __syncwarp();
                    asm volatile("fence.proxy.async;" ::: "memory");
                }
                if (lane == 0) {
                    const int row = (cluster + j * clusters) * kRows + half * kBM;
                    for (int i = 0; i < nk; ++i) {
                        const int q = it + i, s = q % kStages, p = q - nkp;
                        const uint32_t fb = cluster_addr(saddr(&full_bar[s]), lead);
                        if ((q >= kStages && !mbar_wait(saddr(&empty_bar[s]), (uint32_t)((q / kStages - 1) & 1), wlim)) ||
                            // the block of W that this one replaces may be read by a later stage than that
                            (l > 0 && j == 0 && nkp < kStages && i < nkp &&
                             !mbar_wait(saddr(&empty_bar[p % kStages]), (uint32_t)((p / kStages) & 1), wlim)) ||
                            abort_flag) {
                            ok = false;
                            break;
                        }
                        if (j > 0) expect(s, 2 * kABytes);
                        else if (l > 0 || i >= pre) {
                            expect(s, 4 * kABytes);
                            load(wbase + (uint32_t)i * kABytes, h.b[l], i * kBK, rank * 128, fb);
                        }
                        load(abase + (uint32_t)s * kABytes, h.a[l], i * kBK, row, fb);
                        issued = q + 1;
                    }
                }
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                it += nk;
            }
        }
        if (lane == 0) {
            if (!ok) abort_flag = 1;
            // the last stages' copies have landed and their release has arrived
            for (int i = it > kStages ? it - kStages : 0; i < it && ok; ++i)
                ok = mbar_wait(saddr(&empty_bar[i % kStages]), (uint32_t)((i / kStages) & 1), wlim);
            sent[0] = pre;
            sent[1] = issued;
            sent[2] = ok;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && half == 0) {
            constexpr uint32_t idesc = idesc_bf16(kRows, 256);
            auto commit = [](uint64_t* bar, uint16_t mask) {
                asm volatile(
                    "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                        saddr(bar)),
                    "h"(mask)
                    : "memory");
            };
            const uint16_t mine = (uint16_t)(3u << lead);
            int it = 0, tl = 0;
            for (int l = 0; l < h.n && ok; ++l) {
                const int nk = h.nk[l];
                for (int j = 0; j < tiles && ok; ++j, ++tl) {
                    const int acc = tl & 1;
                    if (tl >= 2 && !mbar_wait<true>(saddr(&acce_bar[acc]), (uint32_t)((tl / 2 - 1) & 1), wlim)) {
                        ok = false;
                        break;
                    }
                    tc_after();
                    for (int i = 0; i < nk; ++i, ++it) {
                        const int s = it % kStages;
                        const uint32_t ph = (uint32_t)((it / kStages) & 1);
                        if (abort_flag || !mbar_wait<true>(saddr(&full_bar[s]), ph, wlim)) {
                            ok = false;
                            break;
                        }
                        tc_after();
                        const uint32_t a0 = abase + (uint32_t)s * kABytes, b0 = wbase + (uint32_t)i * kABytes;
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; ++kk) {
                            const uint64_t ad = desc_sw128(a0 + 32u * kk), bd = desc_sw128(b0 + 32u * kk);
                            const uint32_t accum = (i > 0 || kk > 0) ? 1u : 0u;
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem + (uint32_t)acc * 256u),
                                "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
                                : "memory");
                        }
                        commit(&empty_bar[s], mine);
                    }
                    if (!ok) break;
                    commit(&accf_bar[acc], mine);
                }
            }
            if (!ok) abort_flag = 1;
            commit(&done_bar, mine);
        }
        __syncwarp();
    } else {
        // epilogue: 32 rows x 64 columns a warp and tile
        const int w = warp - 2, q = warp & 3, part = w >> 2;
        const uint32_t stg = sbase + (uint32_t)w * kHidStgWarp;
        const uint32_t slot = saddr(&done[kHidEpi * pair + w]);
        auto finished = [&](int n) {   // lane 0: the first n tiles of this warp are written
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            asm volatile("fence.acq_rel.cluster;" ::: "memory");
            asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(slot, rank)), "r"(n) : "memory");
            if (C == 4)
                asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(slot, rank ^ 2)), "r"(n)
                             : "memory");
        };
        const int n0 = pair * 256 + part * 64;
        int tl = 0;
        for (int l = 0; l < h.n && ok; ++l) {
            const float4* bias = reinterpret_cast<const float4*>(h.bias[l] + n0);
            for (int j = 0; j < tiles; ++j, ++tl) {
                const int acc = tl & 1, row0 = (cluster + j * clusters) * kRows + half * kBM + q * 32;
                const bool got = mbar_wait(saddr(&accf_bar[acc]), (uint32_t)((tl / 2) & 1), wlim);
                if (!__all_sync(0xffffffffu, got) || abort_flag) {
                    ok = false;
                    break;
                }
                tc_after();
                if (lane == 0) finished(tl);
                const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * 256 + part * 64);
#pragma unroll 1
                for (int b = 0; b < 2; ++b) {
                    uint32_t rr[32];
                    tmem_ld32(tacc + (uint32_t)(32 * b), rr);
                    // the first box has been read from the staging memory
                    if (b == 1 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t o[4];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float4 bb = __ldg(bias + 8 * b + 2 * c + u);
                            const uint32_t* r = rr + 8 * c + 4 * u;
                            const float2 g0 = gelu2(add2(make_float2(__uint_as_float(r[0]), __uint_as_float(r[1])), make_float2(bb.x, bb.y)));
                            const float2 g1 = gelu2(add2(make_float2(__uint_as_float(r[2]), __uint_as_float(r[3])), make_float2(bb.z, bb.w)));
                            const __nv_bfloat162 p0 = __floats2bfloat162_rn(g0.x, g0.y), p1 = __floats2bfloat162_rn(g1.x, g1.y);
                            o[2 * u] = *reinterpret_cast<const uint32_t*>(&p0);
                            o[2 * u + 1] = *reinterpret_cast<const uint32_t*>(&p1);
                        }
                        // 64-byte-swizzled box: 16-byte chunk c of row r at r * 64 + ((c ^ (r / 2 % 4)) * 16)
                        const uint32_t a = stg + (uint32_t)lane * 64u + ((uint32_t)(c ^ ((lane >> 1) & 3)) << 4);
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                                     "r"(o[3])
                                     : "memory");
                    }
                    if (b == 1) tc_before();
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        if (row0 < M)
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                             reinterpret_cast<uint64_t>(&h.c[l])),
                                         "r"(n0 + 32 * b), "r"(row0), "r"(stg)
                                         : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
                if (lane == 0) {
                    arrive_cluster(cluster_addr(saddr(&acce_bar[acc]), lead));
                    // with one or two tiles a layer the next layer's loads are due before the next tile's epilogue
                    if (tiles <= 2) finished(tl + 1);
                }
                __syncwarp();
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
        if (!ok) abort_flag = 1;
    }
    // (what is in flight is waited for with the full limit, also when a test has cut the others short)
    const bool fin = mbar_wait(saddr(&done_bar), 0u, kWaitNs);
    if (!__syncthreads_and(ok && fin) && tid == 0 && err) atomicOr(err, 1);
    tc_before();
    cluster_sync();   // nobody reads the accumulators or writes to another CTA's shared memory any more
    tc_after();
    if (half == 0 && tid == 0) {
        auto theirs = [&](int q) {
            int v;
            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(saddr(&sent[q]), lead + 1)) : "memory");
            return v;
        };
        if (!sent[2] || !theirs(2)) {
            // copies may be in flight: stage q's barrier completes once the bytes of both CTAs have arrived, those
            // that a CTA did not get to (A from stage[r] on, W in a layer's first tile unless loaded ahead) counted
            // as arrived here.  A CTA is at most kStages stages ahead of the other, so no earlier one is open.
            const int ahead[2] = {sent[0], theirs(0)}, stage[2] = {sent[1], theirs(1)};
            auto first_tile = [&](int q) {
                int l = 0;
                for (; l + 1 < h.n && q >= h.nk[l] * tiles; ++l) q -= h.nk[l] * tiles;
                return q < h.nk[l];
            };
            const int end = max(max(stage[0], stage[1]), max(ahead[0], ahead[1]));
            for (int q = min(stage[0], stage[1]); q < end; ++q) {
                const bool w = first_tile(q);
                uint32_t missing = 0;
                for (int r = 0; r < 2; ++r)
                    if (q >= stage[r]) missing += w && q >= ahead[r] ? 2 * kABytes : kABytes;
                if (q >= stage[0] && q >= ahead[0]) expect(q % kStages, (w ? 4 : 2) * kABytes);
                asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(
                                 cluster_addr(saddr(&full_bar[q % kStages]), lead)),
                             "r"(missing)
                             : "memory");
            }
            for (int q = max(0, end - kStages); q < end; ++q)
                mbar_wait<true>(saddr(&full_bar[q % kStages]), (uint32_t)((q / kStages) & 1), kWaitNs);
        }
    }
    __syncwarp();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
    cluster_sync();
}

// Weight gradients and weight updates of all layers (GradSet), the roles of the warps as in k_gemm_bf16:
// warp 0 streams K blocks, warp 1 issues the MMAs of slice after slice into kGradAcc accumulators by turns,
// the epilogue warps (a row a lane, kGradCols columns each) add each slice to FP32 registers in order
// and, after the last, run Adam on the tile.  Sixteen of them: Adam's divisions and square root are IEEE
// ones, about 100 instructions an element, which four warps took 23 us for.  The slices define the order of the sum (deterministic); adding them
// here instead of writing each to memory and summing them in another kernel (up to 64 slices, 33 MB
// per 512 x 512 layer) leaves one pass over the weights.
constexpr int kGradStages = 7;
constexpr uint32_t kGradStage = kABytes + kGradBN * kBK * 2;
constexpr int kGradPitch = kGradBN + 4;   // floats a row of the update's tile
constexpr int kGradEpi = 16;              // epilogue warps
constexpr int kGradAcc = 4;               // accumulators (slices in flight to the epilogue)
constexpr int kGradCols = kGradBN / (kGradEpi / 4);
static_assert(kGradCols == 16, "an epilogue warp reads 16 columns at a time");
__global__ void __launch_bounds__(64 + 32 * kGradEpi, 1) k_grad_update(const __grid_constant__ GradSet G, int K, int* err)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kGradStages], empty_bar[kGradStages], accf_bar[kGradAcc], acce_bar[kGradAcc], done_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    constexpr uint32_t kCols = kGradAcc * kGradBN;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t base = (saddr(smem_raw) + 1023u) & ~1023u;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)),
                     "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < kGradStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full_bar[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty_bar[s])));
        }
        for (int a = 0; a < kGradAcc; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accf_bar[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(&acce_bar[a])), "r"(kGradEpi));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&done_bar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = tmem_slot;
    const int total = G.end[G.n - 1], kb = K / kBK;
    const unsigned long long wlim = G.wait_ns ? G.wait_ns : kWaitNs;
    float* const tile = reinterpret_cast<float*>(smem_raw + (base - saddr(smem_raw)) + kGradStages * kGradStage);
    auto epi_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(32 * kGradEpi) : "memory"); };   // the epilogue warps
    bool ok = true;
    // job, corner and K blocks a slice of tile t
    auto decode = [&](int t, int& j, int& m0, int& n0) {
        j = 0;
        while (t >= G.end[j]) ++j;
        t -= j ? G.end[j - 1] : 0;
        const int nx = G.N[j] / kGradBN;
        m0 = (t / nx) * kBM;
        n0 = (t % nx) * kGradBN;
    };

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int t = blockIdx.x; t < total && ok && !G.skip_copies; t += gridDim.x) {
                int j, m0, n0;
                decode(t, j, m0, n0);
                for (int i = 0; i < kb; ++i, ++it) {
                    const int s = it % kGradStages;
                    if ((it >= kGradStages &&
                         !mbar_wait(saddr(&empty_bar[s]), (uint32_t)((it / kGradStages - 1) & 1), wlim)) ||
                        abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t fb = saddr(&full_bar[s]);
                    const uint32_t dA = base + (uint32_t)s * kGradStage, dB = dA + kABytes;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(kGradStage)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
                        "{%2, %3}], [%4];" ::"r"(dA),
                        "l"(reinterpret_cast<uint64_t>(&G.ta[j])), "r"(i * kBK), "r"(m0), "r"(fb)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
                        "{%2, %3}], [%4];" ::"r"(dB),
                        "l"(reinterpret_cast<uint64_t>(&G.tb[j])), "r"(i * kBK), "r"(n0), "r"(fb)
                        : "memory");
                }
            }
            if (!ok) abort_flag = 1;
            // every issued copy has landed before the CTA may exit (immediate in the normal case)
            for (int i = it > kGradStages ? it - kGradStages : 0; i < it; ++i)
                if (!mbar_wait(saddr(&full_bar[i % kGradStages]), (uint32_t)((i / kGradStages) & 1), kWaitNs)) ok = false;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(kBM, kGradBN);
            int it = 0, sl = 0;   // K blocks and slices so far
            for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
                int j, m0, n0;
                decode(t, j, m0, n0);
                const int nk = kb / G.S[j];
                for (int z = 0; z < G.S[j] && ok; ++z, ++sl) {
                    const int acc = sl % kGradAcc;
                    if (sl >= kGradAcc &&
                        !mbar_wait(saddr(&acce_bar[acc]), (uint32_t)((sl / kGradAcc - 1) & 1), wlim)) {
                        ok = false;
                        break;
                    }
                    tc_after();
                    for (int i = 0; i < nk; ++i, ++it) {
                        const int s = it % kGradStages;
                        if (abort_flag || !mbar_wait(saddr(&full_bar[s]), (uint32_t)((it / kGradStages) & 1), wlim)) {
                            ok = false;
                            break;
                        }
                        tc_after();
                        const uint32_t a0 = base + (uint32_t)s * kGradStage, b0 = a0 + kABytes;
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; ++kk) {
                            const uint64_t ad = desc_sw128(a0 + 32u * kk), bd = desc_sw128(b0 + 32u * kk);
                            const uint32_t accum = (i > 0 || kk > 0) ? 1u : 0u;
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
                                    tmem + (uint32_t)(acc * kGradBN)),
                                "l"(ad), "l"(bd), "r"(idesc), "r"(accum)
                                : "memory");
                        }
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                saddr(&empty_bar[s]))
                            : "memory");
                    }
                    if (!ok) break;
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     saddr(&accf_bar[acc]))
                                 : "memory");
                }
            }
            if (!ok) abort_flag = 1;
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             saddr(&done_bar))
                         : "memory");
        }
        __syncwarp();
    } else {
        const int q = warp & 3, part = (warp - 2) >> 2;
        const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * kGradCols);
        int sl = 0;
        for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
            int j, m0, n0;
            decode(t, j, m0, n0);
            __syncwarp();
            float g[kGradCols];
#pragma unroll
            for (int c = 0; c < kGradCols; ++c) g[c] = 0.0f;
#pragma unroll 1
            for (int z = 0; z < G.S[j]; ++z, ++sl) {
                const int acc = sl % kGradAcc;
                const bool got = mbar_wait(saddr(&accf_bar[acc]), (uint32_t)((sl / kGradAcc) & 1), wlim);
                if (!__all_sync(0xffffffffu, got) || abort_flag) {
                    ok = false;
                    break;
                }
                tc_after();
                uint32_t rr[16];
                tmem_ld16(tacc + (uint32_t)(acc * kGradBN), rr);
#pragma unroll
                for (int c = 0; c < kGradCols; ++c) g[c] += __uint_as_float(rr[c]);
                tc_before();
                __syncwarp();
                // one arrival a warp (512 of them a slice took as long as its MMAs)
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&acce_bar[acc])) : "memory");
            }
            // the epilogue warps go on together or give up together (the barriers below would wait for
            // a warp that had left)
            uint32_t all;
            asm volatile(
                "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n barrier.cta.red.and.pred p, 1, %2, q;\n"
                " selp.u32 %0, 1, 0, p;\n}"
                : "=r"(all)
                : "r"((uint32_t)ok), "n"(32 * kGradEpi)
                : "memory");
            ok = all != 0;
            if (!ok) break;
            // the tile's gradients through shared memory, so that the update reads and writes whole rows
            // (a row a lane, every access touched 32 lines and waited for the one before: 40 us)
            const int Mj = G.M[j], Di = G.N[j], no = G.n_o[j], ni = G.n_i[j];
            float* const mine = tile + (q * 32 + lane) * kGradPitch + part * kGradCols;
#pragma unroll
            for (int c = 0; c < kGradCols; c += 4)
                *reinterpret_cast<float4*>(mine + c) = make_float4(g[c], g[c + 1], g[c + 2], g[c + 3]);
            epi_sync();
            const bool upd = G.adam.lr > 0.0f;
            const int et = tid - 64, c0 = (et & 15) * 4;   // 16 threads a row
#pragma unroll 4
            for (int r = et >> 4; r < kBM; r += 2 * kGradEpi) {
                const int o = m0 + r;
                if (o >= Mj) break;
                float4* const gp = reinterpret_cast<float4*>(tile + r * kGradPitch + c0);
                const float4 g4 = *gp;
                const size_t at = (size_t)o * Di + n0 + c0;
                float gg[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (o >= no || n0 + c0 + u >= ni) gg[u] = 0.0f;
                *reinterpret_cast<float4*>(G.g[j] + at) = make_float4(gg[0], gg[1], gg[2], gg[3]);
                if (!upd || o >= no) {
                    *gp = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    continue;
                }
                const float4 w4 = *reinterpret_cast<const float4*>(G.W[j] + at);
                const float4 m4 = *reinterpret_cast<const float4*>(G.m[j] + at);
                const float4 v4 = *reinterpret_cast<const float4*>(G.v[j] + at);
                float w[4] = {w4.x, w4.y, w4.z, w4.w}, mm[4] = {m4.x, m4.y, m4.z, m4.w}, vv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (n0 + c0 + u < ni) w[u] = G.adam(w[u], gg[u], mm[u], vv[u]);
                const float4 wn = make_float4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<float4*>(G.W[j] + at) = wn;
                *reinterpret_cast<float4*>(G.m[j] + at) = make_float4(mm[0], mm[1], mm[2], mm[3]);
                *reinterpret_cast<float4*>(G.v[j] + at) = make_float4(vv[0], vv[1], vv[2], vv[3]);
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(w[0], w[1]), h1 = __floats2bfloat162_rn(w[2], w[3]);
                *reinterpret_cast<uint2*>(G.Wb[j] + at) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
                *gp = wn;
            }
            epi_sync();
            if (upd) {
                // the transposed copy: four rows a lane, a column a warp and pass
                const int r = 4 * lane;
                if (m0 + r < Mj) {
#pragma unroll 4
                    for (int c = warp - 2; c < kGradBN; c += kGradEpi) {
                        const float* col = tile + r * kGradPitch + c;
                        const __nv_bfloat162 h0 = __floats2bfloat162_rn(col[0], col[kGradPitch]);
                        const __nv_bfloat162 h1 = __floats2bfloat162_rn(col[2 * kGradPitch], col[3 * kGradPitch]);
                        *reinterpret_cast<uint2*>(G.WbT[j] + (size_t)(n0 + c) * Mj + m0 + r) =
                            make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
                    }
                }
            }
            epi_sync();   // the tile is free for the next one
        }
        if (!ok) abort_flag = 1;
    }
    // every MMA has finished before the TMEM is released (bounded wait; immediate normally)
    const bool fin = mbar_wait(saddr(&done_bar), 0u, kWaitNs);
    if (!__syncthreads_and(ok && fin) && tid == 0 && err) atomicOr(err, 1);
    tc_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols));
}

// Shared memory of k_gemm_bf16: the stages, with TMA stores 4 KB of staging boxes (32 rows x 64 columns) an
// epilogue warp, and the bias of all columns (in EPI_DRAG with sigma and mu behind it)
constexpr size_t gemm_smem(int bn, int stages, int warps, int N, int columns, bool staged)
{
    return (size_t)stages * (kABytes + bn * kBK * 2) + 1024 + (staged ? (size_t)warps * 4096 : 0) +
           (size_t)columns * ((N + 31) & ~31) * 4;
}
constexpr size_t kGemmMaxSmem = 232448 - 256;   // 227 KB opt-in per block, less the static part
struct GemmShape {
    int bn, stages, warps;
};
constexpr GemmShape kGemmShapes[] = {{256, 3, 16}, {192, 4, 12}, {128, 5, 8}, {64, 8, 4}};

template <int BN, int ST, int EPW, int MODE>
bool launch_mode(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tc, int K, const GemmEpi& e,
                 cudaStream_t s)
{
    static_assert(BN / (EPW / 4) == 64, "a warp's staging box");
    const size_t shm = gemm_smem(BN, ST, EPW, e.N, e.bias ? (MODE == EPI_DRAG ? 3 : 1) : 0, e.tstore);
    if (shm > kGemmMaxSmem)
        return MODE == EPI_DRAG ? launch_mode<BN, ST, EPW, MODE == EPI_DRAG ? (int)EPI_DRAG_WIDE : MODE>(ta, tb, tc, K, e, s)
                                : false;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64) return false;
    // dynamic shared memory limit raised per device to the largest size launched so far (the
    // opt-in limit counts the kernel's static shared memory too)
    static size_t configured[64] = {};
    if (shm > configured[dev]) {
        if (cudaFuncSetAttribute(k_gemm_bf16<BN, ST, EPW, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess)
            return false;
        configured[dev] = shm;
    }
    const long long tiles = (long long)((e.N + BN - 1) / BN) * ((e.M + kBM - 1) / kBM);
    const int grid = (int)std::min<long long>(tiles, gemm_sm_count());
    // launched with programmatic stream serialisation: the set-up of this GEMM (barriers, tensor
    // memory) overlaps the tail of the kernel before it, which it waits for before its first read
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(64 + 32 * EPW);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_gemm_bf16<BN, ST, EPW, MODE>, ta, tb, tc, K, e) == cudaSuccess;
}

// one kernel per epilogue mode: each holds only its own epilogue code (a smaller instruction
// footprint for the epilogue warps, whose instruction fetch otherwise stalls them)
template <int SHAPE>
bool launch(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tc, int K, const GemmEpi& e, cudaStream_t s)
{
    constexpr GemmShape g = kGemmShapes[SHAPE];
    switch (e.mode) {
    case EPI_STORE: return launch_mode<g.bn, g.stages, g.warps, EPI_STORE>(ta, tb, tc, K, e, s);
    case EPI_BWD: return launch_mode<g.bn, g.stages, g.warps, EPI_BWD>(ta, tb, tc, K, e, s);
    case EPI_LOSS: return launch_mode<g.bn, g.stages, g.warps, EPI_LOSS>(ta, tb, tc, K, e, s);
    case EPI_DRAG: return launch_mode<g.bn, g.stages, g.warps, EPI_DRAG>(ta, tb, tc, K, e, s);
    default: return false;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

}  // namespace

bool make_tmap_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows,
                    uint32_t box_cols)
{
    auto fn = encode_fn();
    if (!fn || !map || !base || rows == 0 || cols == 0 || ld < cols || (ld * 2) % 16 || box_rows == 0 ||
        box_rows > 256 || (box_cols != 64 && box_cols != 32) || (reinterpret_cast<uintptr_t>(base) & 15))
        return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {ld * 2};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int gemm_sm_count()
{
    static int sms[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 1;
    if (!sms[dev]) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms[dev] = n > 0 ? n : 1;
    }
    return sms[dev];
}

int gemm_pick_bn(int M, int N, bool bias, bool staged)
{
    const int sms = gemm_sm_count();
    int best = 256;
    long long cost = -1;
    for (const GemmShape& g : kGemmShapes) {
        if (gemm_smem(g.bn, g.stages, g.warps, N, bias, staged) > kGemmMaxSmem) continue;
        const long long tiles = (long long)((M + kBM - 1) / kBM) * ((N + g.bn - 1) / g.bn);
        const long long c = (tiles + sms - 1) / sms * (g.bn + 48);
        if (cost < 0 || c < cost) {
            cost = c;
            best = g.bn;
        }
    }
    return best;
}

namespace {

constexpr size_t kHidSmem = (size_t)(kHidMaxK / kBK + kHidStages) * kABytes + kHidEpi * kHidStgWarp + 1024;

template <int C>
cudaLaunchConfig_t hidden_config(int clusters, cudaLaunchAttribute (&attr)[2], cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * C));
    cfg.blockDim = dim3(64 + 32 * kHidEpi);
    cfg.dynamicSmemBytes = kHidSmem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// clusters of C CTAs that can be resident at once (0: the kernel cannot run)
template <int C>
int hidden_clusters()
{
    static std::atomic<int> n[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 0;
    if (!n[dev]) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = hidden_config<C>(1, attr, nullptr);
        cfg.numAttrs = 1;
        int c = 0;
        if (cudaFuncSetAttribute(k_hidden<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHidSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&c, k_hidden<C>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            c = 0;
        }
        n[dev] = c > 0 ? c : -1;
    }
    return std::max(n[dev].load(), 0);
}

template <int C>
bool hidden_launch(const HiddenSet& h, int M, int* err, cudaStream_t s)
{
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = hidden_config<C>(std::min(hidden_clusters<C>(), (M + 2 * kBM - 1) / (2 * kBM)), attr, s);
    return cudaLaunchKernelEx(&cfg, k_hidden<C>, h, M, err) == cudaSuccess;
}

}  // namespace

int gemm_hidden_clusters(int N) { return N == 256 ? hidden_clusters<2>() : N == 512 ? hidden_clusters<4>() : 0; }

bool gemm_hidden_fits(int M, int N, int K0)
{
    if (M < 1 || K0 < kBK || K0 > kHidMaxK || K0 % kBK) return false;
    // With fewer row tiles than 0.6 of the clusters the smaller tiles of k_gemm_bf16 spread better over the SMs
    // (4 x 512: 5000 rows 53.7 us here, 53.1 there; 9000 rows 58 and 63; 18 000 rows 74 and 89; 4 x 256: 9500
    // rows 50 and 47, 12 000 rows 59 and 62; the whole inference each time).
    const int clusters = gemm_hidden_clusters(N);
    return clusters > 0 && 5LL * ((M + 2 * kBM - 1) / (2 * kBM)) >= 3LL * clusters;
}

bool gemm_hidden_launch(const HiddenSet& h, int M, int N, int* err, cudaStream_t s)
{
    if (h.n < 1 || h.n > kHiddenMax || !gemm_hidden_fits(M, N, h.nk[0] * kBK)) return false;
    return N == 256 ? hidden_launch<2>(h, M, err, s) : hidden_launch<4>(h, M, err, s);
}

bool gemm_bf16_grad_launch(GradSet& g, int K, int* err, cudaStream_t s)
{
    if (g.n < 1 || g.n > kGradMax || K < kBK || K % kBK) return false;
    int tiles = 0;
    for (int j = 0; j < g.n; ++j) {
        if (g.M[j] < 64 || g.M[j] % 64 || g.N[j] < 64 || g.N[j] % 64 || g.S[j] < 1 || (K / kBK) % g.S[j]) return false;
        tiles += ((g.M[j] + kBM - 1) / kBM) * (g.N[j] / kGradBN);
        g.end[j] = tiles;
    }
    constexpr size_t shm = kGradStages * kGradStage + 1024 + kBM * kGradPitch * sizeof(float);
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64) return false;
    static bool configured[64] = {};
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(k_grad_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess)
            return false;
        configured[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(tiles, gemm_sm_count()));
    cfg.blockDim = dim3(64 + 32 * kGradEpi);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_grad_update, g, K, err) == cudaSuccess;
}

bool gemm_bf16_launch(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap* tc, int K, int bn,
                      const GemmEpi& e_in, cudaStream_t s)
{
    if (e_in.M < 1 || e_in.N < 1 || K < kBK || K % kBK) return false;
    GemmEpi e = e_in;
    e.tstore = (tc && e.cb) ? 1 : 0;
    static const CUtensorMap none{};
    const CUtensorMap& tcm = e.tstore ? *tc : none;
    if (bn == 0) bn = gemm_pick_bn(e.M, e.N, e.bias != nullptr, e.tstore != 0);
    static_assert(kGemmShapes[0].bn == 256 && kGemmShapes[1].bn == 192 && kGemmShapes[2].bn == 128 && kGemmShapes[3].bn == 64);
    switch (bn) {
    case 256: return launch<0>(ta, tb, tcm, K, e, s);
    case 192: return launch<1>(ta, tb, tcm, K, e, s);
    case 128: return launch<2>(ta, tb, tcm, K, e, s);
    case 64: return launch<3>(ta, tb, tcm, K, e, s);
    default: return false;
    }
}

}  // namespace gwam

namespace {

int gemm_selftest(const void* A, const void* B, int M, int N, int K, const float* bias, int gelu, int bn, int out_bf16,
                  void* C, unsigned long long wait_ns, int skip_copies, void* stream)
{
    if (!A || !B || !C || M < 1 || N < 1 || K < 64 || K % 64 || (bn != 0 && bn != 64 && bn != 128 && bn != 192 &&
                                                                  bn != 256))
        return -1;
    cudaStream_t s = (cudaStream_t)stream;
    const int use_bn = bn ? bn : gwam::gemm_pick_bn(M, N, bias != nullptr, out_bf16 && N % 8 == 0);
    CUtensorMap ta, tb, tc;
    if (!gwam::make_tmap_bf16(&ta, A, (uint64_t)M, (uint64_t)K, (uint64_t)K, 128) ||
        !gwam::make_tmap_bf16(&tb, B, (uint64_t)N, (uint64_t)K, (uint64_t)K, (uint32_t)use_bn))
        return -1;
    const bool have_tc = out_bf16 && N % 8 == 0 && gwam::make_tmap_bf16(&tc, C, (uint64_t)M, (uint64_t)N, (uint64_t)N, 32);
    int* err = nullptr;
    if (cudaMallocAsync((void**)&err, sizeof(int), s) != cudaSuccess) return -2;
    cudaMemsetAsync(err, 0, sizeof(int), s);
    gwam::GemmEpi e{};
    e.mode = gwam::EPI_STORE;
    e.act = gelu ? 1 : 0;
    e.M = M;
    e.N = N;
    e.bias = bias;
    if (out_bf16) {
        e.cb = (__nv_bfloat16*)C;
        e.ldcb = N;
    } else {
        e.cf = (float*)C;
        e.ldcf = N;
    }
    e.err = err;
    e.wait_ns = wait_ns;
    e.skip_copies = skip_copies;
    const bool launched = gwam::gemm_bf16_launch(ta, tb, have_tc ? &tc : nullptr, K, use_bn, e, s);
    int h = 0;
    cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(err, s);
    if (cudaStreamSynchronize(s) != cudaSuccess || !launched) return -5;
    return h ? -6 : 0;
}

}  // namespace

// Self-test entry point (declared in gwam.h): C = act(A . B^T + bias) with BF16 A [M][K] and
// B [N][K]; C FP32 [M][N], or BF16 [M][N] (written by TMA stores when N is a multiple of 8);
// bn = 0 picks the tile width.
extern "C" int gwam_gemm_bf16(const void* A, const void* B, int M, int N, int K, const float* bias, int gelu, int bn,
                              int out_bf16, void* C, void* stream)
{
    return gemm_selftest(A, B, M, N, K, bias, gelu, bn, out_bf16, C, 0ull, 0, stream);
}

// Self-test of the bounded waits (declared in gwam.h): the same GEMM with its producer told to
// issue no copies and every wait limited to wait_us microseconds; the kernel gives up, frees its
// TMEM and reports, and the call returns GWAM_ETIMEOUT.
extern "C" int gwam_selftest_gemm_timeout(const void* A, const void* B, int M, int N, int K, int bn, float* C,
                                          unsigned int wait_us, void* stream)
{
    if (wait_us < 1 || wait_us > 2000000u) return -1;
    return gemm_selftest(A, B, M, N, K, nullptr, 0, bn, 0, C, 1000ull * wait_us, 1, stream);
}

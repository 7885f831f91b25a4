// gwam_gemm.cuh -- BF16 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a) for the drag
// surrogate: C[M, N] = A[M, K] . B[N, K]^T, FP32 accumulation in tensor memory (TMEM), both
// operands K-major (row-major with K contiguous), fused epilogues.
//
// One CTA computes a 128 x BN tile (BN in {64, 128, 192, 256}).  Thread 0 is the TMA producer:
// it streams 64-wide K blocks of A and B into a ring of shared-memory stages (128-byte swizzled
// K-major layout, written by cp.async.bulk.tensor) and signals a "full" mbarrier per stage with
// the transaction byte count.  Thread 32 issues four 128 x BN x 16 tcgen05.mma per K block into
// the TMEM accumulator and commits them to the stage's "empty" mbarrier, which hands the stage
// back to the producer; a final commit signals the accumulator (two of them, so that a tile's
// epilogue overlaps the next tile's MMAs).  4 to 16 warps read it with tcgen05.ld (a warp owns 32 TMEM
// lanes = tile rows) and run the epilogue.  Every mbarrier wait is bounded in time; a wait that gives up sets the error word,
// the kernel still waits (bounded) for its own copies and MMAs and releases its TMEM.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace gwam {

enum GemmEpiMode {
    EPI_STORE = 0,  // v = acc (+ bias) (-> GELU if act); writes cf (FP32), cb (BF16), ct (BF16
                    // transposed); z receives the pre-activation
    EPI_BWD = 1,    // v = acc * GELU'(z[row][n]); writes cb and ct
    EPI_LOSS = 2,   // y = acc + bias; e = y - tgt (n < n_true, else 0); d = gscale * e -> cb, ct;
                    // y -> cf; sum of e^2 added to *loss
    EPI_DRAG = 3,   // y = acc + bias; for n < n_true and mask[row] == 0: y * ysig[n] + ymu[n]
                    // -> du[n * ncol + row] (n < nlev) or dv[(n - nlev) * ncol + row]
    EPI_DRAG_WIDE = 4,   // the launch's form of EPI_DRAG for outputs too many for shared memory
};

struct GemmEpi {
    int mode;
    int act;                  // EPI_STORE: apply GELU
    int M, N;                 // valid rows and columns of C
    const float* bias;        // [N] or null
    float* cf;                // FP32 [M][ldcf]
    int ldcf;
    __nv_bfloat16* cb;        // BF16 [M][ldcb]
    int ldcb;
    __nv_bfloat16* ct;        // BF16 transposed [N][ldct]
    int ldct;
    float* z;                 // FP32 pre-activation [M][ldz]
    int ldz;
    const float* tgt;         // EPI_LOSS: normalised targets [M][ldt]
    int ldt;
    int n_true;               // EPI_LOSS / EPI_DRAG: number of real outputs (N may be padded)
    float gscale;             // EPI_LOSS: dL/dy = gscale * (y - t)
    double* loss;             // EPI_LOSS: sum of squared errors, to FP64 accuracy and range
    const float* ysig;        // EPI_DRAG: de-normalisation (N entries, N a multiple of 32, 16-byte aligned)
    const float* ymu;
    const int* mask;          // EPI_DRAG: 1 = column goes to the ray tracer
    double* du;
    double* dv;
    int ncol, nlev;
    int* err;                 // bit 0 set when a bounded wait gave up
    int tstore;               // set by gemm_bf16_launch: cb is written through an output tensor map
    unsigned long long wait_ns;   // limit of every bounded wait (0: 2 s)
    int skip_copies;          // self-test of the give-up path only: the producer issues no copies
};

// 2-D BF16 tensor map of a row-major [rows][cols] matrix with leading dimension ld (elements),
// box = box_cols (64, or 32) columns x box_rows rows, swizzled over 128 (64) bytes.  false if the driver refuses it.
bool make_tmap_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
                    uint32_t box_rows, uint32_t box_cols = 64);

// One Adam update (Kingma & Ba 2015) of a parameter w with gradient g; returns the new value
struct Adam {
    float lr, b1, b2, eps, c1, c2;   // lr = 0: gradients only
    __device__ __forceinline__ float operator()(float w, float g, float& m, float& v) const
    {
        const float mm = __fmaf_rn(1.0f - b1, g, __fmul_rn(b1, m));
        const float vv = __fmaf_rn(__fmul_rn(1.0f - b2, g), g, __fmul_rn(b2, v));
        m = mm;
        v = vv;
        return w - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    }
};

// The weight gradients and weight updates of all layers as one launch: job j forms dW_j[M_j, N_j] =
// A_j . B_j^T over the batch (K), in S_j slices along K whose sums are added in order (K / 64 divisible by
// S_j), stores it to g and updates W, m, v and the BF16 copies (row-major and transposed).  M_j, N_j
// multiples of 64; entries outside [n_o][n_i] stay zero.
constexpr int kGradMax = 8;
constexpr int kGradBN = 64;
struct GradSet {
    CUtensorMap ta[kGradMax], tb[kGradMax];   // box rows 128 and kGradBN
    float *g[kGradMax], *W[kGradMax], *m[kGradMax], *v[kGradMax];
    __nv_bfloat16 *Wb[kGradMax], *WbT[kGradMax];
    int M[kGradMax], N[kGradMax], n_o[kGradMax], n_i[kGradMax], S[kGradMax];
    int end[kGradMax];                        // tiles of jobs 0 .. j (filled in by the launch)
    int n;
    Adam adam;
    unsigned long long wait_ns;   // as in GemmEpi
    int skip_copies;              // self-test of the give-up path only: the producer issues no copies
};
bool gemm_bf16_grad_launch(GradSet& set, int K, int* err, cudaStream_t s);

// Launch: A described by ta (box rows 128), B by tb (box rows bn); K a multiple of 64.  tc (or null): tensor map
// of the BF16 output cb (box 64 columns x 32 rows) -- the epilogue then stages each warp's rows in shared memory
// and writes them with TMA stores.  bn = 0 picks the tile width (gemm_pick_bn).  false on an unsupported
// shape.
bool gemm_bf16_launch(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap* tc, int K, int bn,
                      const GemmEpi& e, cudaStream_t s);

// All hidden layers of the inference, act_l = GELU(act_(l-1) . W_l^T + bias_l) in BF16, in one kernel with the
// weights in shared memory: N = 256 or 512 outputs a layer, 64 nk <= 512 inputs.  a: act_(l-1) and
// b: W_l with box rows 128; c: act_l in boxes of 32 rows x 32 columns.  The kernel reads the weights
// before the previous kernel of the stream has completed (programmatic dependent launch): they must be
// older than that.  gemm_hidden_fits says whether M rows should run here rather than layer by layer.
constexpr int kHiddenMax = 8;
struct HiddenSet {
    CUtensorMap a[kHiddenMax], b[kHiddenMax], c[kHiddenMax];
    const float* bias[kHiddenMax];
    int nk[kHiddenMax];
    int n;
    unsigned long long wait_ns;   // as in GemmEpi
    int skip_copies;              // self-test of the give-up path only: bit r -- CTA r of each pair issues no copies
};
bool gemm_hidden_fits(int M, int N, int K0);
// clusters of gemm_hidden_launch that are resident at once for N outputs a layer (0: N is not one of its widths)
int gemm_hidden_clusters(int N);
bool gemm_hidden_launch(const HiddenSet& h, int M, int N, int* err, cudaStream_t s);

// The tile width gemm_bf16_launch uses when bn = 0 (the caller builds tb with this box): the one with
// the least waves x (width + 48) over the GPU's SMs -- a tile's time grows with its width, 48 columns
// stand for its fixed part.  Wide tiles for large M (32 768 x 512: 256), narrow ones where wide ones
// would leave SMs idle (4096 x 512: 128 instead of 64 tiles of 256; 1000 x 512: 64).  Only widths whose
// shared memory holds the bias of all N columns (if there is one) and the staging boxes of TMA stores (`staged`)
// beside the stages: with both, 64, 192 and 256 do up to 4544 columns, 128 up to 8640.
int gemm_pick_bn(int M, int N, bool bias, bool staged);
// compute units of the current device
int gemm_sm_count();

}  // namespace gwam

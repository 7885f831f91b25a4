// gwam_common.cuh -- reductions and small helpers shared by the kernels.
#pragma once

#include "gwam_ctx.cuh"

namespace gwam {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ long long warp_sum(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The projected fields a step accumulates into, cleared by the step's ray-advance kernel instead
// of by a memset before the projection: that kernel is bound by instruction issue (FP64 form) or by
// its L1 gathers (precision form) and leaves HBM nearly idle, where the memsets were a pass over
// all the fields on the step's critical path.  Nothing reads or writes these fields between the
// advance and the projection.  The FP64 form clears with thread stores, a part in every
// iteration of its ray loop (clear_fields; after the loop they were 32 us of the kernel with the
// arithmetic idle); the precision form's gathers would compete with such stores for L1, so there one
// thread per block issues bulk copies of a zeroed shared-memory buffer to the tensor-memory-access
// unit, a few per iteration of its ray loop (clear_start / clear_issue / clear_finish).
constexpr int kClearPiece = 16384;  // bytes per bulk copy (measured: 4 KB 0.698, 8 KB 0.607, 16 KB 0.572 ms)

// (the fields lie one after another in one allocation, so a step's fields are one range)
struct ClearSet {
    double2* p;
    int64_t n;   // 16-byte elements
};

// the fields the step's projection accumulates into (the two temperature fields, the last of the
// range, only when projected)
inline ClearSet clear_set(const Context& c)
{
    const int nf = c.P.theta_flux ? NFIELD : F_TL;
    return ClearSet{reinterpret_cast<double2*>(c.field[0]), (c.field[nf - 1] - c.field[0] + c.field_len(nf - 1) + 1) / 2};
}

// All threads: 16-byte streaming stores of zeros to the elements of the range that belong to part m
// of `parts` (grid-stride within the part).
__device__ __forceinline__ void clear_fields(const ClearSet& z, int m, int parts)
{
    const int64_t per = (z.n + parts - 1) / parts;
    const int64_t end = (m + 1) * per < z.n ? (m + 1) * per : z.n;
    for (int64_t i = m * per + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end; i += (int64_t)gridDim.x * blockDim.x)
        __stcs(z.p + i, make_double2(0.0, 0.0));
}

struct ClearState {
    int64_t g;         // next piece of this block (blocks take every gridDim.x-th piece)
    int per;           // pieces issued per ray-loop iteration
    uint32_t zbuf;     // shared-memory address of the zeroed buffer
};

__device__ __forceinline__ int64_t clear_pieces(const ClearSet& z) { return (z.n * 16 + kClearPiece - 1) / kClearPiece; }

// All threads of the block: zero the buffer, make it visible to the bulk-copy unit, and spread the
// block's pieces over the ray loop of thread 0 (n rays, grid-stride loop).
__device__ __forceinline__ void clear_start(const ClearSet& z, float4* zbuf, int n, ClearState& st)
{
    for (int q = threadIdx.x; q < kClearPiece / 16; q += blockDim.x) zbuf[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    const int64_t total = clear_pieces(z);
    st.g = blockIdx.x;
    st.zbuf = (uint32_t)__cvta_generic_to_shared(zbuf);
    const int64_t mine = st.g < total ? (total - 1 - st.g) / gridDim.x + 1 : 0;
    const int64_t b0 = (int64_t)blockIdx.x * blockDim.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t iters = n > b0 ? (n - b0 + stride - 1) / stride : 0;
    st.per = iters > 0 ? (int)((mine + iters - 1) / iters) : 0;
}

// Thread 0: issue up to `count` of the block's pieces as one bulk group.
__device__ __forceinline__ void clear_issue(const ClearSet& z, ClearState& st, int count)
{
    const int64_t total = clear_pieces(z);
    int issued = 0;
    for (; issued < count && st.g < total; ++issued, st.g += gridDim.x) {
        const int64_t off = st.g * kClearPiece;
        const uint32_t bytes = (uint32_t)(z.n * 16 - off < kClearPiece ? z.n * 16 - off : kClearPiece);
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                     :: "l"(reinterpret_cast<char*>(z.p) + off), "r"(st.zbuf), "r"(bytes) : "memory");
    }
    if (issued) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Thread 0 of every block: the rest of its pieces, then wait until all its copies are done (the
// shared buffer must outlive them).
__device__ __forceinline__ void clear_finish(const ClearSet& z, ClearState& st)
{
    if (threadIdx.x != 0) return;
    clear_issue(z, st, 0x7fffffff);
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The FP64 ray step's loop: whole passes of the grid take consecutive rays block by block; the rays
// that are left over go to the blocks in groups of 32, a warp of every block before the second of any
// (the whole blocks of a partial last pass would leave most SMs idle, and a small population would run
// on a few SMs: 2600 rays on 11 of 152, 41 -> 30 us).  The precision form, bound by its gathers,
// is better off with neighbouring warps on neighbouring rays (210 K rays: 50 us, spread 54 us).  Ray of
// this thread in pass m, n or more if none.
__device__ __forceinline__ int loop_passes(int n) { return n / (int)(gridDim.x * blockDim.x) + 1; }
__device__ __forceinline__ int loop_ray(int m, int passes)
{
    const int T = gridDim.x * blockDim.x;
    if (m + 1 < passes) return m * T + blockIdx.x * blockDim.x + threadIdx.x;
    return m * T + ((int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
}

// Block sum in a fixed order (deterministic); the result is valid in thread 0.
template <typename T>
__device__ __forceinline__ T block_sum(T v)
{
    __shared__ T sh[32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    T r = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : T(0);
    if (wid == 0) r = warp_sum(r);
    return r;
}

// True when this lane's run of equal keys touches neither lane 0 nor lane 31: with the ray array
// sorted by key and a warp holding 32 consecutive entries, no other warp holds that key, so the
// run's sum may be stored instead of added atomically (fewer L2 atomics, and deterministic).
__device__ __forceinline__ bool warp_run_interior(int key)
{
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(0xffffffffu, key, 1);
    const int next = __shfl_down_sync(0xffffffffu, key, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != key);
    const unsigned tails = __ballot_sync(0xffffffffu, lane == 31 || next != key);
    const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
    const int end = __ffs(tails & (0xffffffffu << lane)) - 1;
    return start > 0 && end < 31;
}

// The cell offsets of a step: before the cap, and after it.  The second scan runs only when a column
// was over the cap; otherwise the first one's offsets stand.
struct CellOffsets {
    const int *before, *after;
    __device__ __forceinline__ const int* live(const Ctl* ctl) const { return ctl->n_over ? after : before; }
};

// All threads: zero part m of `parts` of n ints (a 16-byte aligned array), grid-stride within the part
__device__ __forceinline__ void clear_ints(int* p, int n, int m, int parts)
{
    const int per = (n / 4 + parts - 1) / parts, end = min((m + 1) * per, n / 4);
    for (int i = m * per + blockIdx.x * blockDim.x + threadIdx.x; i < end; i += gridDim.x * blockDim.x)
        reinterpret_cast<int4*>(p)[i] = make_int4(0, 0, 0, 0);
    if (m == 0 && blockIdx.x == 0 && (int)threadIdx.x < n % 4) p[n - 1 - threadIdx.x] = 0;
}

// First entry of this warp in pass m of a loop over n entries (n or more: none): consecutive entries
// block by block, except that fewer entries than the grid has threads go a warp to every block before
// the second of any (2600 ray volumes kept 11 of 152 SMs busy).
__device__ __forceinline__ int64_t loop_warp(int m, int n)
{
    const int T = gridDim.x * blockDim.x, w = threadIdx.x >> 5;
    if (n < T) return m ? n : ((int64_t)w * gridDim.x + blockIdx.x) * 32;
    return (int64_t)m * T + (int64_t)blockIdx.x * blockDim.x + w * 32;
}

// ---------------------------------------------------------------------------- per-column cap (App. B.5)

// Doubles as unsigned integers of the same order (-0 = +0, NaN above everything): comparisons on the
// integer pipe (an FP64 compare runs at GB300's FP64 rate).
__device__ __forceinline__ unsigned long long order_key(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x), top = 1ull << 63;
    if ((b & ~top) > 0x7FF0000000000000ull) return ~0ull;
    if (b & top) return b == top ? top : ~b;
    return b | top;
}
// the key of a number's multiple by f
__device__ __forceinline__ unsigned long long key_scaled(unsigned long long key, double f)
{
    const unsigned long long top = 1ull << 63;
    return order_key(__longlong_as_double((long long)((key & top) ? key ^ top : ~key)) * f);
}

constexpr int kCapThreads = 128;
constexpr int kCapKeys = 1024;   // keys held in shared memory; longer columns keep theirs in global scratch
constexpr double kCapDelta = 1.0 / (1 << 24);

// The entries [a, a + count) that the cap removes from an over-full column: the `drop` with the lowest
// energies, ties by the larger id first, as one block (kCapThreads).  energy(e) may be off by kCapDelta / 2
// relative: the drop-th lowest is found by a radix select over the keys (8 bits a pass, until one
// key is left; counting every entry's rank took count^2 FP64 comparisons), entries clearly below it go,
// entries clearly above it stay, and the few within kCapDelta of it are ranked by exact(e).
// A NaN energy always goes and counts towards nobody's rank.  remove(e) is called for each.
template <class Energy, class Exact, class Remove>
__device__ __forceinline__ void cap_column(int a, int count, int drop, const long long* __restrict__ ent_id,
                                           double* __restrict__ scratch, Energy energy, Exact exact, Remove remove)
{
    __shared__ unsigned long long sh_keys[kCapKeys];
    __shared__ int hist[256];
    __shared__ int sh_digit, sh_left, sh_bin, sh_low, sh_amb;
    __shared__ unsigned long long sh_cut;
    unsigned long long* keys = count <= kCapKeys ? sh_keys : reinterpret_cast<unsigned long long*>(scratch) + a;
    for (int e = threadIdx.x; e < count; e += kCapThreads) keys[e] = order_key(energy(a + e));
    if (threadIdx.x == 0) sh_low = sh_amb = 0;
    unsigned long long prefix = 0, mask = 0;
    int left = drop;   // the drop-th lowest key (1 .. count) among those with this prefix
    for (int shift = 56; shift >= 0; shift -= 8) {
        for (int q = threadIdx.x; q < 256; q += kCapThreads) hist[q] = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < count; e += kCapThreads)
            if ((keys[e] & mask) == prefix) atomicAdd(&hist[(int)(keys[e] >> shift) & 255], 1);
        __syncthreads();
        if (threadIdx.x < 32) {
            int h[8], sum = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                h[q] = hist[8 * threadIdx.x + q];
                sum += h[q];
            }
            int before = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, before, d);
                if ((int)threadIdx.x >= d) before += o;
            }
            before -= sum;
            if (before < left && left <= before + sum) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (before < left && left <= before + h[q]) {
                        sh_digit = 8 * threadIdx.x + q;
                        sh_left = left - before;
                        sh_bin = h[q];
                    }
                    before += h[q];
                }
            }
        }
        __syncthreads();
        prefix |= (unsigned long long)sh_digit << shift;
        mask |= 255ull << shift;
        left = sh_left;
        if (sh_bin == 1) break;
    }
    // the one key with the prefix, or the common value of those that share all its digits
    for (int e = threadIdx.x; e < count; e += kCapThreads)
        if ((keys[e] & mask) == prefix) sh_cut = keys[e];
    __syncthreads();
    const unsigned long long cut = sh_cut;
    if (cut == ~0ull) {   // more to drop than there are numbers
        for (int e = threadIdx.x; e < count; e += kCapThreads) remove(a + e);
        __syncthreads();
        return;
    }
    const unsigned long long k0 = key_scaled(cut, 1.0 - kCapDelta), k1 = key_scaled(cut, 1.0 + kCapDelta);
    const unsigned long long lo = k0 < k1 ? k0 : k1, hi = k0 < k1 ? k1 : k0;
    int low = 0, amb = 0;
    for (int e = threadIdx.x; e < count; e += kCapThreads) {
        const unsigned long long k = keys[e];
        low += k < lo;
        amb += k >= lo && k <= hi;
    }
    if (low) atomicAdd(&sh_low, low);
    if (amb) atomicAdd(&sh_amb, amb);
    __syncthreads();
    const int need = drop - sh_low;   // of the sh_amb around the cut
    if (need == sh_amb) {
        for (int e = threadIdx.x; e < count; e += kCapThreads)
            if (keys[e] <= hi || keys[e] == ~0ull) remove(a + e);
    } else {
        // entries around the cut get their exact keys, those below 0 (no double's key) and those above
        // ~0 - 1 (likewise); the exact ones are ranked among themselves
        for (int e = threadIdx.x; e < count; e += kCapThreads) {
            const unsigned long long k = keys[e];
            if (k != ~0ull) keys[e] = k < lo ? 0ull : (k > hi ? ~0ull - 1 : order_key(exact(a + e)));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < count; e += kCapThreads) {
            const unsigned long long k = keys[e];
            if (k == ~0ull - 1) continue;
            int rank = 0;
            if (k != 0ull && k != ~0ull) {
                const long long id = ent_id[a + e];
                for (int q = 0; q < count; ++q) {
                    const unsigned long long o = keys[q];
                    rank += o != 0ull && (o < k || (o == k && ent_id[a + q] > id));
                }
            }
            if (k == 0ull || k == ~0ull || rank < need) remove(a + e);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void set_status(Ctl* ctl, int code)
{
    atomicCAS(&ctl->status, 0, code);
}

}  // namespace gwam

// gwam_device.cuh -- device-side data layout and per-ray-volume arithmetic (FP64 form).
//
// Ray equations of Voelker et al. (arXiv:2309.11257):
//   dispersion relation with scale-height correction ........ Sec. 2a, Eq. dispersion
//   c_g = grad_k Omega, rdot = c_g ........................... Eq. eikonal, Eq. group-velocity
//   wavenumber tendencies with spherical metric terms ......... Eq. eikonal-sphere:1-3
//   face group velocities from first-order Taylor values ...... Sec. 3b, App. B.1
//   per-axis phase-space products P = h dX dk ................. Sec. 3a, Eq. vpvol_cons_cart, Eq. dkxdkl
//   low-storage RK3 (Williamson 1980) ......................... App. B.2
//   splitting thresholds ...................................... App. B.3
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gwam_df.cuh"

namespace gwam {

constexpr double kPi = 3.14159265358979323846;
constexpr int kThreads = 256;

// ---------------------------------------------------------------------------- arithmetic

// Reciprocal: the hardware approximation (PTX rcp.approx.ftz.f64, about 20 correct bits) refined by
// two Newton-Raphson steps y <- y + y (1 - x y), each of which doubles the number of correct bits.
// For the positive, finite, normal-range operands of the ray equations (within an ulp or so of the
// IEEE quotient, tested against it); FP64 division would cost several times as many instructions.
__device__ __forceinline__ double rcp_nr(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}

// Reciprocal square root: the hardware approximation (PTX rsqrt.approx.ftz.f64) refined by two
// Newton-Raphson steps y <- y + (y/2) (1 - x y^2).
__device__ __forceinline__ double rsqrt_nr(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double e = fma(-x * y, y, 1.0);
    y = fma(0.5 * y, e, y);
    e = fma(-x * y, y, 1.0);
    return fma(0.5 * y, e, y);
}

// ---------------------------------------------------------------------------- layouts

// Grid geometry as the kernels see it (derived once on the host).
struct Grid {
    int geometry;          // 0 f-plane, 1 sphere
    int columnar;          // single-column mode (no horizontal propagation, advection or refraction)
    int nx, ny, nz;
    int ncol, ncell;       // per member: nx*ny, nx*ny*nz
    int members;           // ensemble members (independent backgrounds and ray populations)
    int ncol_all, ncell_all;   // members * ncol, members * ncell
    double dX, dY, dz;     // coordinate spacings (radians on the sphere)
    double y0;             // southern edge (-pi/2) or 0
    double Lx, Ly;         // periods in x (2 pi or nx dx) and y (f-plane)
    double ztop;
    double f0, radius, omega, g;
    double phimax;         // carriers poleward of this latitude leave (centre of the last row)
    // precomputed reciprocals and tables (FP64 division is a long instruction sequence)
    double inv_dX, inv_dY, inv_dz, inv_nx, inv_ny, inv_g;
    const double* row_cos;      // cos(phi_j) of every row centre (sphere), 1 on the f-plane
    const double* row_inv_cos;  // 1 / row_cos
    const double* lev_inv_r;    // 1 / (a + z_k) of every level centre (sphere), 1 on the f-plane
    // FP32 copies for the precision form (a float <- double conversion runs at the FP64 rate)
    float f_dX, f_dY, f_dz, f_y0, f_radius, f_omega, f_f0, f_inv_dX, f_inv_dY, f_inv_dz;
    const float* row_cos32;     // [ny]
    const float* ivol32;        // [ny * nz]: 1 / cell volume of row j, level k
    const float* whf32;         // [ny]: row_inv_cos * inv_dX * inv_dY (solid-angle share per unit extent)
    // double-float constants and row tables of the FP64 form's ray equations
    float2 df_radius, df_2omega, df_8omega2, df_f0sq, df_f0;
    const float2* row_sc_df;    // [ny][2]: sin, cos of every row centre (sphere)
    const double* row_lat;      // [ny]: latitude of every row centre
    const float2* whf_df;       // [ny]: row_inv_cos * inv_dX * inv_dY
    const float2* ivol_df;      // [ny * nz]: 1 / cell volume of row j, level k
    const float2* row_lat_df;   // [ny]: latitude of every row centre
    float2 df_inv_dX, df_inv_dY, df_inv_dz, df_y0;
    // split thresholds (App. B.3), computed on the host in the order the device used to:
    // split_thr[2 j] = alpha_s sqrt(cos(phi_j) dX dY), split_thr[2 j + 1] = alpha_s cos(phi_j) dX dY
    const double* split_thr;
    double split_hthr;          // max(alpha_s dz, min_split_dz)
    const double* row_f2;       // [ny]: f^2 of every row centre (f0^2 on the f-plane)
};

struct Params {
    int gamma_mode, saturation, smoothing, flux_form, splitting, cap, theta_flux;
    double alpha_s, min_split_dz;
    float f_alpha_s;
};

// Ray-volume state, structure of arrays of double2 (16-byte vector loads):
//   a[0] = (x, y)  a[1] = (z, k)  a[2] = (l, m)  a[3] = (ex, ey)
//   a[4] = (ez, Px)  a[5] = (Py, Pz)  a[6] = (N, id as int64 bits)
struct RaySoA {
    double2* a[7];
};

enum { SX, SY, SZ, SK, SL, SM, SEX, SEY, SEZ, SPX, SPY, SPZ, SN, NSTATE };

// Ray ids are 64-bit: the ensemble member in the top 8 bits, a running number below.  Cells are
// global: member * ncell + (j * nx + i) * nz + k, so the canonical array is member-major.
constexpr int kMemberShift = 56;
__host__ __device__ __forceinline__ int member_of(long long id) { return (int)((unsigned long long)id >> kMemberShift); }
__host__ __device__ __forceinline__ long long with_member(int m, long long local)
{
    return (long long)(((unsigned long long)m << kMemberShift) | (unsigned long long)local);
}

__device__ __forceinline__ void load_ray(const RaySoA& R, int64_t i, double s[NSTATE], long long& id)
{
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        double2 v = __ldg(&R.a[q][i]);
        s[2 * q] = v.x;
        s[2 * q + 1] = v.y;
    }
    double2 v = __ldg(&R.a[6][i]);
    s[SN] = v.x;
    id = __double_as_longlong(v.y);
}

__device__ __forceinline__ void store_ray(const RaySoA& R, int64_t i, const double s[NSTATE], long long id)
{
#pragma unroll
    for (int q = 0; q < 6; ++q) R.a[q][i] = make_double2(s[2 * q], s[2 * q + 1]);
    R.a[6][i] = make_double2(s[SN], __longlong_as_double(id));
}

// Background nodes at cell centres, column-major: node (i, j, k) at (j*nx + i)*nz + k.
// The FP64 node holds U, V, N^2, Gamma^2 (32 bytes); the per-step gathers of the ray equations read
// the copies that also carry the node gradients (NodeDF of the FP64 form, Node32 of the precision
// form), written when the background is set (Sec. 3b, App. B.1).
struct __align__(32) Node {
    double v[4];       // U, V, N^2, Gamma^2
};

// FP32 background node of the precision form: the same 16 quantities in FP32 (64 bytes)
struct __align__(64) Node32 {
    float v[4];
    float d[4][3];
};

// FP32 ray record of the precision form, 64 bytes as four float4 arrays:
//   q[0] = (member-local cell as int bits, ox, oy, oz)    offsets in cell units, in [0, 1)
//   q[1] = (k, l, m, N)
//   q[2] = (eX, eY, eZ, Px)                               extents in coordinate units
//   q[3] = (Py, Pz, id low 32 bits, id high 32 bits)
struct Ray32SoA {
    float4* q[4];
};

__host__ __device__ __forceinline__ int64_t node_index(const Grid& G, int i, int j, int k)
{
    return ((int64_t)j * G.nx + i) * G.nz + k;
}

// ---------------------------------------------------------------------------- background gather

__device__ __forceinline__ int wrap_int(int i, int n)
{
    int r = i % n;
    return r < 0 ? r + n : r;
}

// periodic bracketing node pair; s in node units, inv_n = 1/n
__device__ __forceinline__ void bracket_periodic(double s, int n, double inv_n, int& q0, int& q1, double& t)
{
    if (!isfinite(s)) s = 0.0;
    s = s - (double)n * floor(s * inv_n);
    double fl = floor(s);
    t = s - fl;
    q0 = wrap_int((int)fl, n);
    q1 = q0 + 1 == n ? 0 : q0 + 1;
}

// clamped bracketing: every interpolated quantity held at its edge-node value outside
__device__ __forceinline__ void bracket_clamped(double s, int n, int& q0, int& q1, double& t)
{
    if (!isfinite(s)) s = 0.0;
    if (s < 0.0) {
        q0 = 0; q1 = 1; t = 0.0;
    } else if (s >= (double)(n - 1)) {
        q0 = n - 2; q1 = n - 1; t = 1.0;
    } else {
        double fl = floor(s);
        q0 = (int)fl; q1 = q0 + 1; t = s - fl;
    }
}

// The background node as 16 double-float pairs (hi, lo), in the order of Node's 16 doubles: the
// per-step gathers of the FP64 form run on the FP32 pipes (compensated sums), with about 48
// significant bits.  Filled from the FP64 nodes whenever the background is set.
struct __align__(128) NodeDF {
    float4 q[8];   // q[e] = the high parts of values 2e and 2e + 1, then their low parts
};

// s + c += (wh + wl) (vh + vl) for two node values at a time: TwoProduct of the high parts, TwoSum
// into s, all lower-order terms into the compensation c.  The product's error and the cross terms are
// formed negated, from the negated weight that a corner's sixteen values share, and subtracted (a
// packed instruction has no free negation): 12 packed operations for two values.
struct CornerWeight {
    float2 h, nh, nl;   // the weight's high part, and both parts negated, in both halves
};

__device__ __forceinline__ CornerWeight corner_weight(DF w) { return {dup2(w.hi), dup2(-w.hi), dup2(-w.lo)}; }

__device__ __forceinline__ void df_acc2(float2 vh, float2 vl, const CornerWeight& w, float2& s, float2& c)
{
    const float2 p = mul2(w.h, vh);
    float2 g = fma2(w.nh, vh, p);
    g = fma2(w.nl, vh, g);
    g = fma2(w.nh, vl, g);
    const float2 t = add2(s, p);
    const float2 bb = sub2(t, s);
    const float2 err = add2(sub2(s, sub2(t, bb)), sub2(p, bb));
    s = t;
    c = add2(c, sub2(err, g));
}

// Trilinear interpolation of the FP64 node values (U, V, N^2, Gamma^2) to (X, Y, Z).
__device__ __forceinline__ void gather_values_fp64(const Grid& G, const Node* __restrict__ bg, double X, double Y,
                                                   double Z, double v[4])
{
    int i0, i1, j0, j1, k0, k1;
    double tx, ty, tz;
    bracket_periodic(X * G.inv_dX - 0.5, G.nx, G.inv_nx, i0, i1, tx);
    if (G.geometry == 1) bracket_clamped((Y - G.y0) * G.inv_dY - 0.5, G.ny, j0, j1, ty);
    else bracket_periodic(Y * G.inv_dY - 0.5, G.ny, G.inv_ny, j0, j1, ty);
    bracket_clamped(Z * G.inv_dz - 0.5, G.nz, k0, k1, tz);
    const double ux = 1.0 - tx, uy = 1.0 - ty, uz = 1.0 - tz;
    const int dk = k1 - k0;
    const Node* cn[4] = {bg + node_index(G, i0, j0, k0), bg + node_index(G, i1, j0, k0),
                         bg + node_index(G, i0, j1, k0), bg + node_index(G, i1, j1, k0)};
    const double wc[4] = {ux * uy, tx * uy, ux * ty, tx * ty};
#pragma unroll
    for (int f = 0; f < 4; ++f) v[f] = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const Node* p = cn[q >> 1] + ((q & 1) ? dk : 0);
        const double w = wc[q >> 1] * ((q & 1) ? tz : uz);
        const double2 a = __ldg(reinterpret_cast<const double2*>(p->v));
        const double2 b = __ldg(reinterpret_cast<const double2*>(p->v) + 1);
        v[0] += w * a.x;
        v[1] += w * a.y;
        v[2] += w * b.x;
        v[3] += w * b.y;
    }
}

struct BgDF {
    DF v[4];
    DF d[4][3];
};

// Bracketing in node units on double-float coordinates (FP32 pipes only): u = node coordinate,
// q0 = floor(u) (wrapped or clamped), t = u - floor(u).  A non-finite u maps to node 0.
__device__ __forceinline__ int wrap_fast(int i, int n)
{
    if ((unsigned)i < (unsigned)n) return i;
    if (i < 0 && i >= -n) return i + n;
    return wrap_int(i, n);
}

// u - floor(u) of a renormalised u: hi - floor is exact for hi >= 0; for a negative hi (floor = -1 just
// west of the first node) its rounding error comes from FastTwoSum, |floor| >= |hi|.  The difference
// is zero or at least an ulp of hi, so the second FastTwoSum is exact too.
__device__ __forceinline__ DF frac_df(DF u, float fl)
{
    const float d = __fsub_rn(u.hi, fl);
    const float e = __fadd_rn(__fsub_rn(u.hi, __fadd_rn(d, fl)), u.lo);
    const float t = __fadd_rn(d, e);
    return {t, __fsub_rn(e, __fsub_rn(t, d))};
}

__device__ __forceinline__ void bracket_periodic_df(DF u, int n, int& q0, int& q1, DF& t)
{
    float fl = df_floor_sum(u);
    if (!(fabsf(fl) < 1e9f)) {
        fl = 0.0f;
        u = df_f(0.0f);
    }
    t = frac_df(u, fl);
    q0 = wrap_fast((int)fl, n);
    q1 = q0 + 1 == n ? 0 : q0 + 1;
}

__device__ __forceinline__ void bracket_clamped_df(DF u, int n, int& q0, int& q1, DF& t)
{
    float fl = df_floor_sum(u);
    if (!(fabsf(fl) < 1e9f)) {
        fl = 0.0f;
        u = df_f(0.0f);
    }
    const int q = (int)fl;
    if (q < 0) {
        q0 = 0; q1 = 1; t = df_f(0.0f);
    } else if (q >= n - 1) {
        q0 = n - 2; q1 = n - 1; t = df_f(1.0f);
    } else {
        q0 = q; q1 = q + 1; t = frac_df(u, fl);
    }
}

// The eight nodes around the double-float position (X, Y, Z): the lowest one's index and the steps to
// the others, the four horizontal weights and the two vertical ones; jrow = the row whose centre is
// nearest.  Corners in the order (i0 j0), (i1 j0), (i0 j1), (i1 j1), each at k0 then k1.
struct CornersDF {
    int base, ox, oy, oz;
    DF w00, w10, w01, w11, Uz, Tz;
    int jrow;
    __device__ __forceinline__ int node(int q) const { return base + ((q & 2) ? ox : 0) + ((q & 4) ? oy : 0) + ((q & 1) ? oz : 0); }
    __device__ __forceinline__ DF weight(int q) const
    {
        return df_mul2((q & 2) ? ((q & 4) ? w11 : w10) : ((q & 4) ? w01 : w00), (q & 1) ? Tz : Uz);
    }
};

__device__ __forceinline__ CornersDF corners_df(const Grid& G, DF X, DF Y, DF Z)
{
    CornersDF r;
    int i0, i1, j0, j1, k0, k1;
    DF Tx, Ty;
    const DF half = df_f(0.5f);
    bracket_periodic_df(df_sub(df_mul2(X, DF{G.df_inv_dX.x, G.df_inv_dX.y}), half), G.nx, i0, i1, Tx);
    if (G.geometry == 1)
        bracket_clamped_df(df_sub(df_mul2(df_sub(Y, DF{G.df_y0.x, G.df_y0.y}), DF{G.df_inv_dY.x, G.df_inv_dY.y}), half),
                           G.ny, j0, j1, Ty);
    else
        bracket_periodic_df(df_sub(df_mul2(Y, DF{G.df_inv_dY.x, G.df_inv_dY.y}), half), G.ny, j0, j1, Ty);
    bracket_clamped_df(df_sub(df_mul2(Z, DF{G.df_inv_dz.x, G.df_inv_dz.y}), half), G.nz, k0, k1, r.Tz);
    const DF one{1.0f, 0.0f};
    const DF Ux = df_add_fast(one, df_neg(Tx)), Uy = df_add_fast(one, df_neg(Ty));
    r.Uz = df_add_fast(one, df_neg(r.Tz));
    r.w00 = df_mul2(Ux, Uy);
    r.w10 = df_mul2(Tx, Uy);
    r.w01 = df_mul2(Ux, Ty);
    r.w11 = df_mul2(Tx, Ty);
    r.base = (j0 * G.nx + i0) * G.nz + k0;
    r.ox = (i1 - i0) * G.nz;
    r.oy = (j1 - j0) * G.nx * G.nz;
    r.oz = k1 - k0;
    r.jrow = Ty.hi < 0.5f ? j0 : j1;
    return r;
}

// All 16 quantities at the positions of a warp's 32 rays, by eight lanes a node: lane l loads the
// (l & 7)-th 16 bytes of the nodes of rays 4 j + (l >> 3), j = 0 .. 7, so every load covers whole
// 128-byte nodes, and accumulates that element's two quantities for these eight rays.  With a ray a
// lane, each of a node's eight 16-byte loads touched 32 lines where the rays of a warp sit at different
// levels, and the kernel was bound by them (256 x 128 x 90 sphere, waves aloft: 64 loads a stage x 32
// wavefronts = 0.5 ms of L1 per step).  The weights and node indices pass to the eight lanes through
// the ray's row of shared memory, the sums come back in the same row (kGatherRow floats: 128 bytes and
// a pad against bank conflicts).  All 32 lanes must call it; the row is free again after the call.
constexpr int kGatherRow = 36;

__device__ __forceinline__ void gather_warp_df(const Grid& G, const NodeDF* __restrict__ bg, int first, DF X, DF Y, DF Z,
                                               float* rows, BgDF& b, int& jrow)
{
    const int lane = threadIdx.x & 31;
    {
        const CornersDF cn = corners_df(G, X, Y, Z);
        jrow = cn.jrow;
        float* row = rows + lane * kGatherRow;
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            const DF w0 = cn.weight(q), w1 = cn.weight(q + 1);
            *reinterpret_cast<float4*>(row + 2 * q) = make_float4(w0.hi, w0.lo, w1.hi, w1.lo);
        }
        *reinterpret_cast<int4*>(row + 16) = make_int4(first + cn.base, cn.ox, cn.oy, cn.oz);
    }
    __syncwarp();
    const float4* __restrict__ el = reinterpret_cast<const float4*>(bg) + (lane & 7);
    float* row = rows + (lane >> 3) * kGatherRow;
    float4 nxt[8];
    auto fetch = [&](const float* r) {
        const int4 o = *reinterpret_cast<const int4*>(r + 16);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            nxt[q] = __ldg(el + 8 * (int64_t)(o.x + ((q & 2) ? o.y : 0) + ((q & 4) ? o.z : 0) + ((q & 1) ? o.w : 0)));
    };
    fetch(row);
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = nxt[q];
        if (j < 7) fetch(row + 4 * kGatherRow);   // the next rays' nodes, while these are summed
        float2 s = dup2(0.0f), c = dup2(0.0f);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float2 w = *reinterpret_cast<const float2*>(row + 2 * q);
            df_acc2(make_float2(v[q].x, v[q].y), make_float2(v[q].z, v[q].w), corner_weight(DF{w.x, w.y}), s, c);
        }
        const DF a0 = df_norm(s.x, c.x), a1 = df_norm(s.y, c.y);
        __syncwarp();   // the four rays' weights have been read by their eight lanes
        *reinterpret_cast<float4*>(row + 4 * (lane & 7)) = make_float4(a0.hi, a1.hi, a0.lo, a1.lo);
        row += 4 * kGatherRow;
    }
    __syncwarp();
    float4 e[8];
    const float* own = rows + lane * kGatherRow;
#pragma unroll
    for (int q = 0; q < 8; ++q) e[q] = *reinterpret_cast<const float4*>(own + 4 * q);
    auto val = [&](int q) { return (q & 1) ? DF{e[q >> 1].y, e[q >> 1].w} : DF{e[q >> 1].x, e[q >> 1].z}; };
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        b.v[f] = val(f);
#pragma unroll
        for (int q = 0; q < 3; ++q) b.d[f][q] = val(4 + 3 * f + q);
    }
    __syncwarp();
}

// N^2 and Gamma^2 (the second 16 bytes of each node) alone, as unevaluated hi + compensation pairs: what
// the intrinsic quantities need.  The loop over the corners is rolled, the corner's node and weight
// selected, not indexed (measured faster on GB300 than unrolling by 2 or 8: the kernels were stalling
// on instruction fetch).
__device__ __forceinline__ void gather_n2g2_sums(const Grid& G, const NodeDF* __restrict__ bg, DF X, DF Y, DF Z,
                                                 float2& s, float2& c, int& jrow)
{
    const CornersDF cn = corners_df(G, X, Y, Z);
    jrow = cn.jrow;
    s = c = dup2(0.0f);
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
        const float4 a = __ldg(bg[cn.node(q)].q + 1);
        df_acc2(make_float2(a.x, a.y), make_float2(a.z, a.w), corner_weight(cn.weight(q)), s, c);
    }
}

// N^2 and Gamma^2 alone (the second float4 of each node): what the intrinsic quantities need
__device__ __forceinline__ void gather_n2g2_df(const Grid& G, const NodeDF* __restrict__ bg, DF X, DF Y, DF Z,
                                               DF& n2, DF& g2, int& jrow)
{
    float2 s, c;
    gather_n2g2_sums(G, bg, X, Y, Z, s, c, jrow);
    n2 = df_norm(s.x, c.x);
    g2 = df_norm(s.y, c.y);
}

// f^2 and d(f^2)/dphi (f = 2 Omega sin phi on the sphere, f0 on the f-plane)
__device__ __forceinline__ void coriolis(const Grid& G, double sphi, double cphi, double& f2, double& df2)
{
    if (G.geometry == 1) {
        double f = 2.0 * G.omega * sphi;
        f2 = f * f;
        df2 = 8.0 * G.omega * G.omega * sphi * cphi;
    } else {
        f2 = G.f0 * G.f0;
        df2 = 0.0;
    }
}

// ---------------------------------------------------------------------------- dispersion (Eq. dispersion)

// Positive intrinsic branch: w^2 = (f^2 (m^2 + G^2) + N^2 k_h^2) / K^2, K^2 = k_h^2 + m^2 + G^2.
// The intrinsic group velocity is ch = (k, l) D (m^2 + G^2) / (w K^4), ch_r = -m D k_h^2 / (w K^4),
// D = N^2 - f^2, so each component is (its factor) * c with c = D / (w K^4).
struct Disp {
    double K2, iK2, D, w2, w, iw, c;
};

__device__ __forceinline__ void dispersion(double kh2, double mg2, double n2, double f2, Disp& d)
{
    d.K2 = kh2 + mg2;
    d.D = n2 - f2;
    d.iK2 = rcp_nr(d.K2);
    d.w2 = (f2 * mg2 + n2 * kh2) * d.iK2;
    d.iw = rsqrt_nr(d.w2);
    d.w = d.w2 * d.iw;
    d.c = d.D * d.iK2 * d.iK2 * d.iw;
}

// ---------------------------------------------------------------------------- ray equations

struct Geo {
    double r, ir, hX, ihX, hY, sphi, cphi, tphi;
};

__device__ __forceinline__ void geometry_at(const Grid& G, double Y, double Z, Geo& g)
{
    if (G.geometry == 1) {
        sincos(Y, &g.sphi, &g.cphi);
        g.r = G.radius + Z;
        g.ir = rcp_nr(g.r);
        const double ic = rcp_nr(g.cphi);
        g.hX = g.r * g.cphi;
        g.ihX = g.ir * ic;
        g.hY = g.r;
        g.tphi = g.sphi * ic;
    } else {
        g.sphi = 0.0; g.cphi = 1.0; g.tphi = 0.0;
        g.r = 1.0; g.ir = 1.0; g.hX = 1.0; g.ihX = 1.0; g.hY = 1.0;
    }
}

// ------------------------------------------------------------ the ray equations in double-float
// The ray equations -- the carrier moves with the mean of the opposing face group velocities, the
// extents with their difference (Sec. 3b, App. B.1); the wavenumber follows Eq. eikonal-sphere:1-3
// (sphere) or kdot = -grad Omega (f-plane) with the centre values -- evaluated in double-float on
// the FP32 pipes (GB300's FP64 rate is 1/72 of its FP32 rate): the state enters
// as FP64 and is split (one FP64 subtraction per component), the nine rates leave as FP64.  Every
// intermediate carries about 48 significant bits, the reciprocal and reciprocal square root one
// Newton step in DF from the FP32 hardware approximations (~2^-45).

struct DispDF {
    DF K2, iK2, D, w2, iw, c;
};

// w^2 as f^2 + D k_h^2 / K^2 (the same quantity as (f^2 (m^2 + G^2) + N^2 k_h^2) / K^2, one product fewer,
// and D / K^2 serves c too)
__device__ __forceinline__ void dispersion_df(DF kh2, DF mg2, DF n2, DF f2, DispDF& d)
{
    d.K2 = df_add_same(kh2, mg2);
    d.D = df_sub(n2, f2);
    d.iK2 = df_rcp(d.K2);
    const DF t = df_mul2(d.D, d.iK2);
    d.w2 = df_add(f2, df_mul2(t, kh2));
    d.iw = df_rsqrt(d.w2);
    d.c = df_mul2(df_mul2(t, d.iK2), d.iw);
}

struct GeoDF {
    DF ir, ihX, sphi, cphi, tphi;
};

// sin and cos of the latitude from the row-centre table and the offset d from the centre
// (|d| <= half a row): sin(p0 + d) = s0 cos d + c0 sin d, cos(p0 + d) = c0 cos d - s0 sin d, with
// sin d and cos d from their Taylor series -- the terms up to d^3 and d^4 in DF, the smaller ones
// (below 3e-8 for rows of up to 9 degrees) in FP32, truncated after d^7 and d^8
constexpr double kLatSeriesRow = 9.0 * kPi / 180.0;
__device__ __forceinline__ void lat_sincos_row_df(const Grid& G, int j, DF Y, DF& sphi, DF& cphi)
{
    const float2 rl = G.row_lat_df[j];
    const DF d = df_sub(Y, DF{rl.x, rl.y});
    const DF dd = df_mul2(d, d);
    constexpr DF sixth{1.0f / 6.0f, (float)(1.0 / 6.0 - (double)(1.0f / 6.0f))};
    constexpr DF twentyfourth{1.0f / 24.0f, (float)(1.0 / 24.0 - (double)(1.0f / 24.0f))};
    const float d2 = dd.hi;
    const float d4 = d2 * d2;
    const DF sind = df_add(df_sub(d, df_mul2(df_mul2(dd, d), sixth)),
                           df_f(d.hi * d4 * (1.0f / 120.0f - d2 * (1.0f / 5040.0f))));
    const DF cosd = df_sub(df_add(df_sub(df_f(1.0f), df_pow2(dd, 0.5f)), df_mul2(df_mul2(dd, dd), twentyfourth)),
                           df_f(d4 * d2 * (1.0f / 720.0f - d2 * (1.0f / 40320.0f))));
    const float2 sc0 = G.row_sc_df[2 * j], sc1 = G.row_sc_df[2 * j + 1];
    const DF s0{sc0.x, sc0.y}, c0{sc1.x, sc1.y};
    sphi = df_add(df_mul2(s0, cosd), df_mul2(c0, sind));
    cphi = df_sub(df_mul2(c0, cosd), df_mul2(s0, sind));
}

// the same with the row found from Y: it only selects the expansion point, so a neighbouring row near
// a boundary is as good
__device__ __forceinline__ void lat_sincos_df(const Grid& G, DF Y, DF& sphi, DF& cphi)
{
    const float fj = df_floor(df_mul2(df_sub(Y, DF{G.df_y0.x, G.df_y0.y}), DF{G.df_inv_dY.x, G.df_inv_dY.y}));
    const int j = fj < 0.0f ? 0 : (fj >= (float)(G.ny - 1) ? G.ny - 1 : (int)fj);
    lat_sincos_row_df(G, j, Y, sphi, cphi);
}

__device__ __forceinline__ void geometry_df(const Grid& G, int j, DF Y, DF Z, GeoDF& g)
{
    if (G.geometry == 1) {
        lat_sincos_row_df(G, j, Y, g.sphi, g.cphi);
        const DF r = df_add(DF{G.df_radius.x, G.df_radius.y}, Z);
        g.ir = df_rcp(r);
        const DF ic = df_rcp(g.cphi);
        g.ihX = df_mul2(g.ir, ic);
        g.tphi = df_mul2(g.sphi, ic);
    } else {
        g.sphi = df_f(0.0f);
        g.cphi = df_f(1.0f);
        g.tphi = df_f(0.0f);
        g.ir = df_f(1.0f);
        g.ihX = df_f(1.0f);
    }
}

// Where rk3 and ray_rhs_df keep a thread's nine components between the passes: shared memory, two
// components (their high parts, then their low parts) in a float4, a warp's pairs 32 lanes apart.  The
// state y, the low-storage register q, the increment sums acc and the rates r wait there instead of in
// the registers that the ray equations need; r shares its place with the gather's rows, which are
// free once the background is in registers.
constexpr int kRkPairs = 5;                                       // nine components and a spare half
constexpr int kRkWarp = 3 * kRkPairs * 32 + 32 * kGatherRow / 4;  // float4s a warp: y, q, acc, rows (or r)
constexpr size_t kRkSmem = kRkWarp * (kThreads / 32) * sizeof(float4);
static_assert(kRkPairs * 32 <= 32 * kGatherRow / 4, "the rates fit the gather's rows");

struct RkSlots {
    float4 *y, *q, *acc, *r;   // this thread's
    float* rows;               // its warp's
    __device__ __forceinline__ explicit RkSlots(void* smem)
    {
        float4* w = static_cast<float4*>(smem) + (threadIdx.x >> 5) * kRkWarp;
        y = w + (threadIdx.x & 31);
        q = y + kRkPairs * 32;
        acc = q + kRkPairs * 32;
        r = acc + kRkPairs * 32;
        rows = reinterpret_cast<float*>(w + 3 * kRkPairs * 32);
    }
};

__device__ __forceinline__ DF rk_get(const float4* p, int c)
{
    const float* f = reinterpret_cast<const float*>(p + (c >> 1) * 32) + (c & 1);
    return {f[0], f[2]};
}
__device__ __forceinline__ void rk_put(float4* p, int c, DF v)
{
    float* f = reinterpret_cast<float*>(p + (c >> 1) * 32) + (c & 1);
    f[0] = v.hi;
    f[2] = v.lo;
}
__device__ __forceinline__ DFP rk_get2(const float4* p, int pair)
{
    const float4 v = p[pair * 32];
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void rk_put2(float4* p, int pair, DFP v)
{
    p[pair * 32] = make_float4(v.hi.x, v.hi.y, v.lo.x, v.lo.y);
}

// the nine rates (into sl.r) at the state sl.y; first = the first node of the ray's ensemble member.  All
// 32 lanes of a warp must call it.
__device__ __forceinline__ void ray_rhs_df(const Grid& G, const NodeDF* __restrict__ bg, int first, const RkSlots& sl)
{
    const DFP y01 = rk_get2(sl.y, 0);
    const DF X = dfp_x(y01), Y = dfp_y(y01), Z = rk_get(sl.y, 2);
    BgDF b;
    int jrow;
    gather_warp_df(G, bg, first, X, Y, Z, sl.rows, b, jrow);
    GeoDF g;
    geometry_df(G, jrow, Y, Z, g);
    DF f2, df2;
    if (G.geometry == 1) {
        const DF f = df_mul2(DF{G.df_2omega.x, G.df_2omega.y}, g.sphi);
        f2 = df_mul2(f, f);
        df2 = df_mul2(df_mul2(DF{G.df_8omega2.x, G.df_8omega2.y}, g.sphi), g.cphi);
    } else {
        f2 = DF{G.df_f0sq.x, G.df_f0sq.y};
        df2 = df_f(0.0f);
    }
    const DFP y45 = rk_get2(sl.y, 2);
    const DF k = rk_get(sl.y, 3), l = dfp_x(y45), m = dfp_y(y45);
    const DF U = b.v[0], V = b.v[1], N2 = b.v[2], G2 = b.v[3];
    const DF kh2 = df_add_same(df_mul2(k, k), df_mul2(l, l));
    const DF mg2 = df_add_same(df_mul2(m, m), G2);
    DispDF d;
    dispersion_df(kh2, mg2, N2, f2, d);
    const DF mg2c = df_mul2(mg2, d.c);
    const DF cgx = df_add(df_mul2(k, mg2c), U);
    const DF cgy = df_add(df_mul2(l, mg2c), V);
    const DF cgz = df_neg(df_mul2(df_mul2(m, kh2), d.c));
    const DF hwK = df_pow2(df_mul2(d.iw, d.iK2), 0.5f);   // 1 / (2 w K^2)
    const DF aN = df_mul2(kh2, hwK);
    const DF aG = df_mul2(df_mul2(aN, d.D), d.iK2);
    const DF aF = df_mul2(mg2, hwK);
    DF Gq[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
        Gq[q] = df_sub(df_add(df_add(df_mul2(k, b.d[0][q]), df_mul2(l, b.d[1][q])), df_mul2(aN, b.d[2][q])),
                       df_mul2(aG, b.d[3][q]));
    Gq[1] = df_add(Gq[1], df_mul2(aF, df2));
    if (G.columnar) {
        // single-column mode: k and l fixed, m by the vertical gradient of Omega alone
        rk_put(sl.r, 3, df_f(0.0f));
        rk_put(sl.r, 4, df_f(0.0f));
        rk_put(sl.r, 5, df_neg(Gq[2]));
    } else if (G.geometry == 1) {
        const DF ir = g.ir;
        rk_put(sl.r, 3, df_add(df_neg(df_mul2(Gq[0], g.ihX)), df_mul2(df_mul2(k, ir), df_sub(df_mul2(g.tphi, cgy), cgz))));
        rk_put(sl.r, 4, df_sub(df_neg(df_mul2(Gq[1], ir)),
                               df_mul2(ir, df_add(df_mul2(l, cgz), df_mul2(df_mul2(k, g.tphi), cgx)))));
        rk_put(sl.r, 5, df_add(df_neg(Gq[2]), df_mul2(ir, df_add(df_mul2(k, cgx), df_mul2(l, cgy)))));
    } else {
        rk_put(sl.r, 3, df_neg(Gq[0]));
        rk_put(sl.r, 4, df_neg(Gq[1]));
        rk_put(sl.r, 5, df_neg(Gq[2]));
    }
    // faces: first-order Taylor values along the face's own axis, the two faces of an axis in the halves
    // of packed pairs.  Relative to the centre a face changes m^2 + G^2 and K^2 by +-tg and D by
    // +-(tn - tf), so its dispersion terms start from the centre's sums; with b = (m^2 + G^2) c the mean and
    // the difference of the two face velocities are (A (b+ + b-) / 2 + W) S and (A (b+ - b-) + 2 tw) S
    // (horizontal), -m k_h^2 times those of c (vertical).  108 operations a face instead of 197 for a
    // face evaluated from its own values.  The axes run as a rolled loop, the per-axis operands selected,
    // not indexed: unrolled, the kernel outgrew the instruction cache (a third of its stall cycles
    // were instruction fetch).
    int q0 = 0;
    if (G.columnar) {
        // no horizontal propagation or advection
        rk_put(sl.r, 0, df_f(0.0f));
        rk_put(sl.r, 1, df_f(0.0f));
        rk_put(sl.r, 6, df_f(0.0f));
        rk_put(sl.r, 7, df_f(0.0f));
        q0 = 2;
    }
    const DF mkh2 = df_neg(df_mul2(m, kh2));
#pragma unroll 1
    for (int q = q0; q < 3; ++q) {
        const DF ext = rk_get(sl.y, 6 + q);
        const DF dn = q == 0 ? b.d[2][0] : (q == 1 ? b.d[2][1] : b.d[2][2]);
        const DF dg = q == 0 ? b.d[3][0] : (q == 1 ? b.d[3][1] : b.d[3][2]);
        const DF h = df_pow2(ext, 0.5f);
        const DF tg = df_mul2(dg, h);
        DF td = df_mul2(dn, h);
        DFP f2f = dfp_dup(f2);
        if (q == 1) {   // f^2 varies along the meridional axis only
            const DF tf = df_mul2(df2, h);
            td = df_sub(td, tf);
            f2f = dfp_add(f2f, dfp_pm(tf));
        }
        const DFP iK2 = dfp_rcp(dfp_add(dfp_dup(d.K2), dfp_pm(tg)));
        const DFP t = dfp_mul(dfp_add(dfp_dup(d.D), dfp_pm(td)), iK2);
        const DFP iw = dfp_rsqrt(dfp_add(f2f, dfp_mul(t, dfp_dup(kh2))));
        DFP c = dfp_mul(dfp_mul(t, iK2), iw);
        if (q < 2) c = dfp_mul(dfp_add(dfp_dup(mg2), dfp_pm(tg)), c);
        const DF A = q == 0 ? k : (q == 1 ? l : mkh2);
        DF mean = df_mul2(A, df_pow2(df_add(dfp_x(c), dfp_y(c)), 0.5f));
        DF diff = df_mul2(A, df_sub(dfp_x(c), dfp_y(c)));
        if (q < 2) {
            const DF W = q == 0 ? U : V, S = q == 0 ? g.ihX : g.ir, dW = q == 0 ? b.d[0][0] : b.d[1][1];
            mean = df_mul2(df_add(mean, W), S);
            diff = df_mul2(df_add(diff, df_mul2(dW, ext)), S);   // dW ext = 2 tw
        }
        rk_put(sl.r, q, mean);
        rk_put(sl.r, 6 + q, diff);
    }
}

// Intrinsic quantities of a ray volume at its carrier position in double-float (the FP64 form's
// saturation and projection): wavenumbers, f^2, N^2 and the dispersion terms, from N^2 and Gamma^2
// interpolated alone.
struct IntrDF {
    DF k, l, m, kh2, m2, mg2, f, f2, n2;   // f: the signed Coriolis parameter at the ray
    DispDF d;
};

__device__ __forceinline__ void intrinsic_df(const Grid& G, const NodeDF* __restrict__ bg, const double s[NSTATE],
                                             IntrDF& in)
{
    DF g2;
    int jrow;
    const DF Y = df_split(s[SY]);
    gather_n2g2_df(G, bg, df_split(s[SX]), Y, df_split(s[SZ]), in.n2, g2, jrow);
    if (G.geometry == 1) {
        DF sphi, cphi;
        lat_sincos_row_df(G, jrow, Y, sphi, cphi);
        in.f = df_mul2(DF{G.df_2omega.x, G.df_2omega.y}, sphi);
        in.f2 = df_mul2(in.f, in.f);
    } else {
        in.f = DF{G.df_f0.x, G.df_f0.y};
        in.f2 = DF{G.df_f0sq.x, G.df_f0sq.y};
    }
    in.k = df_split(s[SK]);
    in.l = df_split(s[SL]);
    in.m = df_split(s[SM]);
    in.kh2 = df_add_same(df_mul2(in.k, in.k), df_mul2(in.l, in.l));
    in.m2 = df_mul2(in.m, in.m);
    in.mg2 = df_add_same(in.m2, g2);
    dispersion_df(in.kh2, in.mg2, in.n2, in.f2, in.d);
}

// Williamson (1980) low-storage RK3 on the 9 propagated components; background frozen.  The rates
// and the low-storage register q are double-float; the step's increments B q of the three stages
// are summed in double-float (sl.acc) and added to the FP64 state once, by the caller (rk_increment: one
// FP64 rounding per component instead of three: the sum is far smaller than the state, so its 48 bits
// are ample), and a double-float copy of the state, updated by the same B q, feeds the next
// evaluation.  The update takes two components at a time in packed pairs, as a rolled loop (a small
// kernel body: see ray_rhs_df).
__device__ __forceinline__ void rk3_start(const RkSlots& sl, const double (&s)[9])
{
#pragma unroll
    for (int c = 0; c < 9; ++c) rk_put(sl.y, c, df_split(s[c]));
    rk_put(sl.y, 9, df_f(0.0f));
}

// first: the first node of the ray's ensemble member; all 32 lanes of a warp must call it
__device__ __forceinline__ void rk3(const Grid& G, const NodeDF* __restrict__ bg, int first, double dt, const RkSlots& sl)
{
    constexpr DF A1{-5.0f / 9.0f, (float)(-5.0 / 9.0 - (double)(-5.0f / 9.0f))};
    constexpr DF A2{-153.0f / 128.0f, 0.0f};
    constexpr DF B0{1.0f / 3.0f, (float)(1.0 / 3.0 - (double)(1.0f / 3.0f))};
    constexpr DF B1{15.0f / 16.0f, 0.0f};
    constexpr DF B2{8.0f / 15.0f, (float)(8.0 / 15.0 - (double)(8.0f / 15.0f))};
    const DF dtd = df_split(dt);
#pragma unroll 1
    for (int st = 0; st < 3; ++st) {
        ray_rhs_df(G, bg, first, sl);
        rk_put(sl.r, 9, df_f(0.0f));
        const DFP a = dfp_dup(st == 1 ? A1 : A2);
        const DFP b = dfp_dup(st == 0 ? B0 : (st == 1 ? B1 : B2));
        const DFP h = dfp_dup(dtd);
#pragma unroll 1
        for (int p = 0; p < kRkPairs; ++p) {
            DFP q = dfp_mul(h, rk_get2(sl.r, p));
            if (st > 0) q = dfp_add(dfp_mul(a, rk_get2(sl.q, p)), q);
            const DFP bq = dfp_mul(b, q);
            if (st < 2) {   // the last stage's state is not evaluated
                rk_put2(sl.q, p, q);
                rk_put2(sl.y, p, dfp_add(rk_get2(sl.y, p), bq));
            }
            rk_put2(sl.acc, p, st > 0 ? dfp_add(rk_get2(sl.acc, p), bq) : bq);
        }
        __syncwarp();   // the rates have been read: their place is the next stage's gather rows
    }
}

// the step's increment of component c
__device__ __forceinline__ double rk_increment(const RkSlots& sl, int c) { return df_to_double(rk_get(sl.acc, c)); }

// ---------------------------------------------------------------------------- bookkeeping

__device__ __forceinline__ double wrap_period(double x, double L)
{
    double w = x - L * floor(x / L);
    if (w < 0.0) w += L;
    if (w >= L) w = 0.0;
    return w;
}

__device__ __forceinline__ void wrap_position(const Grid& G, double s[NSTATE])
{
    // most carriers stay inside the period: skip the division then
    if (!(s[SX] >= 0.0 && s[SX] < G.Lx)) s[SX] = wrap_period(s[SX], G.Lx);
    if (G.geometry == 0 && !(s[SY] >= 0.0 && s[SY] < G.Ly)) s[SY] = wrap_period(s[SY], G.Ly);
}

__device__ __forceinline__ double ray_action(const double s[NSTATE])
{
    return s[SN] * s[SPX] * s[SPY] * s[SPZ];
}

// 0 inside, 1 left the domain, 2 not a valid ray volume
__device__ __forceinline__ int ray_status(const Grid& G, const double s[NSTATE])
{
    // finiteness from the exponent bits (integer pipe): all ones means infinity or NaN
    unsigned allf = 0u;
#pragma unroll
    for (int c = 0; c < NSTATE; ++c) allf |= ((((unsigned)__double2hiint(s[c]) >> 20) & 0x7FFu) + 1u) & 0x800u;
    if (allf) return 2;
    if (!(s[SEX] > 0.0 && s[SEY] > 0.0 && s[SEZ] > 0.0)) return 2;
    if (!(s[SZ] >= 0.0 && s[SZ] < G.ztop)) return 1;
    if (G.geometry == 1 && !(fabs(s[SY]) <= G.phimax)) return 1;
    return 0;
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ void cell_ijk(const Grid& G, const double s[NSTATE], int& i, int& j, int& k)
{
    i = clampi((int)floor(s[SX] * G.inv_dX), 0, G.nx - 1);
    j = clampi((int)floor((s[SY] - G.y0) * G.inv_dY), 0, G.ny - 1);
    k = clampi((int)floor(s[SZ] * G.inv_dz), 0, G.nz - 1);
}

__device__ __forceinline__ int cell_of(const Grid& G, const double s[NSTATE])
{
    int i, j, k;
    cell_ijk(G, s, i, j, k);
    return (j * G.nx + i) * G.nz + k;
}

// latitude of row j's centre, multiply then add (never contracted into an FMA)
__device__ __forceinline__ double row_lat(const Grid& G, int j) { return __dadd_rn(G.y0, __dmul_rn(j + 0.5, G.dY)); }

// Split decision (App. B.3): bit 0 vertical, bit 1 horizontal, bit 2 horizontal axis is y.
__device__ __forceinline__ int split_code(const Grid& G, const Params& P, const double s[NSTATE])
{
    if (!P.splitting) return 0;
    int code = 0;
    if (s[SEZ] > G.split_hthr) code |= 1;
    double xlen, ylen, thr, area, athr;
    if (G.geometry == 1) {
        int i, j, k;
        cell_ijk(G, s, i, j, k);
        DF sphi, cphi;
        lat_sincos_df(G, df_split(s[SY]), sphi, cphi);
        const double cp = df_to_double(cphi);
        xlen = cp * s[SEX];
        ylen = s[SEY];
        thr = G.split_thr[2 * j];
        area = cp * s[SEX] * s[SEY];
        athr = G.split_thr[2 * j + 1];
    } else {
        xlen = s[SEX];
        ylen = s[SEY];
        thr = G.split_thr[0];
        area = s[SEX] * s[SEY];
        athr = G.split_thr[1];
    }
    if (xlen > thr || ylen > thr || area > athr) code |= (xlen >= ylen) ? 2 : 6;
    return code;
}

__device__ __forceinline__ int num_children(int code) { return ((code & 1) ? 2 : 1) * ((code & 2) ? 2 : 1); }

// one axis of a split: the half at +-1/4 of the extent, half the extent and half the product
__device__ __forceinline__ void halve(double& x, double& ext, double& P, bool plus)
{
    x += (plus ? 0.25 : -0.25) * ext;
    ext *= 0.5;
    P *= 0.5;
}

// Child c of a split parent: children are ordered (lower, upper) x (minus, plus) with the
// vertical index fastest; child 0 keeps the parent id, child c > 0 takes the (c-1)-th new id.
__device__ __forceinline__ void make_child(const Grid& G, const double p[NSTATE], int code, int c, double s[NSTATE])
{
#pragma unroll
    for (int q = 0; q < NSTATE; ++q) s[q] = p[q];
    const int nv = (code & 1) ? 2 : 1;
    if (code & 1) halve(s[SZ], s[SEZ], s[SPZ], (c % nv) == 1);
    if (code & 2) {
        const bool plus = (c / nv) == 1;
        if (code & 4) halve(s[SY], s[SEY], s[SPY], plus);
        else halve(s[SX], s[SEX], s[SPX], plus);
    }
    if (code) wrap_position(G, s);
}


// Intrinsic properties of a ray volume at its carrier position (saturation, projection, cap).
struct Intr {
    double kh2, m2, mg2, K2, iK2, D, w, iw, w2, c, f2, n2;
};

__device__ __forceinline__ void intrinsic_at(const Grid& G, const NodeDF* __restrict__ bg, const double s[NSTATE],
                                             Geo& g, Intr& in)
{
    float2 sum, cmp;
    int jrow;
    gather_n2g2_sums(G, bg, df_split(s[SX]), df_split(s[SY]), df_split(s[SZ]), sum, cmp, jrow);
    const double n2 = widen(sum.x) + widen(cmp.x), g2 = widen(sum.y) + widen(cmp.y);
    geometry_at(G, s[SY], s[SZ], g);
    double df2;
    coriolis(G, g.sphi, g.cphi, in.f2, df2);
    in.kh2 = s[SK] * s[SK] + s[SL] * s[SL];
    in.m2 = s[SM] * s[SM];
    in.n2 = n2;
    in.mg2 = in.m2 + g2;
    Disp d;
    dispersion(in.kh2, in.mg2, n2, in.f2, d);
    in.K2 = d.K2;
    in.iK2 = d.iK2;
    in.D = d.D;
    in.w = d.w;
    in.iw = d.iw;
    in.w2 = d.w2;
    in.c = d.c;
}

}  // namespace gwam

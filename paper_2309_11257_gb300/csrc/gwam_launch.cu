// gwam_launch.cu -- background upload, explicit ray volumes, and the wave sources.
//
//   background: column-major node fields + Gamma^2 from rho (Sec. 2a; Gamma^2 = (d ln rho / dz)^2 / 4,
//               centred differences between node levels, one-sided at the ends)
//   sources:    background source of Sec. 3c (alpha(phi), F_sol, F_am) and explicit spectral bins;
//               intrinsic frequency w = |k_h| c - k.U, bins outside |f| < w < N or with m^2 <= 0 are
//               filtered, m from the inverted Eq. dispersion, m < 0 (upward group velocity),
//               A = F / (|k_h| ch_r).
#include "gwam_common.cuh"
#include "gwam_fp32.cuh"

namespace gwam {

enum { BG_NONFINITE = 1, BG_RHO = 2, BG_N2F2 = 4 };

// exponent bits all ones: infinity or NaN (integer pipe)
__device__ __forceinline__ bool nonfinite_bits(double x)
{
    return ((((unsigned)__double2hiint(x) >> 20) & 0x7FFu) == 0x7FFu);
}

// caller [nz][ny][nx] -> column-major node values (U, V, N^2, Gamma^2) and rho, transposed through
// shared memory (kBgTile columns of a row per block: 8 columns, 23 KB of shared memory, eight blocks
// per SM; 16 columns, four blocks per SM, took 37 us more of the set-up).  Gamma^2 =
// (d ln rho / dz)^2 / 4 by centred differences of ln rho (one-sided at the bottom and top), each
// difference taken as the logarithm of the density ratio in double-float (df_log_ratio); 1/rho by
// the Newton reciprocal; f^2 of the row from the host table.
constexpr int kBgTile = 8;
__global__ void k_set_background(Grid G, int gamma_mode, const double* __restrict__ u, const double* __restrict__ v,
                                 const double* __restrict__ n2, const double* __restrict__ rho, Node* __restrict__ bg,
                                 double* __restrict__ rho_c, double* __restrict__ rho_inv, int* flags)
{
    extern __shared__ double sh[];   // 4 arrays x nz x kBgTile: U, V, N^2, rho
    const int TW = kBgTile;
    const int nz = G.nz;
    const int ntx = (G.nx + TW - 1) / TW;
    const int j = blockIdx.x / ntx, i0 = (blockIdx.x % ntx) * TW;
    double* su = sh;
    double* sv = sh + nz * TW;
    double* sn = sh + 2 * nz * TW;
    double* sr = sh + 3 * nz * TW;
    int bad = 0;
    for (int t = threadIdx.x; t < nz * TW; t += blockDim.x) {
        const int ii = t % TW, k = t / TW, i = i0 + ii;
        if (i >= G.nx) continue;
        const int64_t o = ((int64_t)k * G.ny + j) * G.nx + i;
        const double a = u[o], b = v[o], c = n2[o], d = rho[o];
        su[k * TW + ii] = a;
        sv[k * TW + ii] = b;
        sn[k * TW + ii] = c;
        sr[k * TW + ii] = d;
        if (nonfinite_bits(a) || nonfinite_bits(b) || nonfinite_bits(c) || nonfinite_bits(d)) bad |= BG_NONFINITE;
        else if (__double_as_longlong(d) <= 0) bad |= BG_RHO;   // rho <= 0 (or -0)
    }
    __syncthreads();
    const double f2 = G.row_f2[j];
    const DF h1{G.df_inv_dz.x, G.df_inv_dz.y};
    const DF h2 = df_pow2(h1, 0.5f);
    for (int t = threadIdx.x; t < nz * TW; t += blockDim.x) {
        const int k = t % nz, ii = t / nz, i = i0 + ii;
        if (i >= G.nx) continue;
        const double r = sr[k * TW + ii];
        const bool rok = __double_as_longlong(r) > 0 && !nonfinite_bits(r);
        double g2 = 0.0;
        if (gamma_mode) {
            const int ku = k == nz - 1 ? k : k + 1, kd = k == 0 ? 0 : k - 1;
            const double ru = sr[ku * TW + ii], rd = sr[kd * TW + ii];
            if (rok && __double_as_longlong(ru) > 0 && __double_as_longlong(rd) > 0 && !nonfinite_bits(ru) &&
                !nonfinite_bits(rd)) {
                const DF dl = df_mul2(df_log_ratio(ru, rd), (k == 0 || k == nz - 1) ? h1 : h2);
                g2 = df_to_double(df_pow2(df_mul2(dl, dl), 0.25f));
            }
        }
        const double nn = sn[k * TW + ii];
        if (!(nn > f2)) bad |= BG_N2F2;
        const int64_t c = node_index(G, i, j, k);
        *reinterpret_cast<double4*>(bg[c].v) = make_double4(su[k * TW + ii], sv[k * TW + ii], nn, g2);
        rho_c[c] = r;
        rho_inv[c] = rok ? rcp_nr(r) : 0.0;
    }
    if (bad) atomicOr(flags, bad);
}

// Node gradients by centred differences: periodic in x (and y on the f-plane), one-sided at the
// pole rows and at the bottom and top levels.  The same pass writes the per-step gather copies of
// the node: double-float pairs (FP64 form, bgdf) or FP32 (precision form, bg32), whichever is given.
// At most 85 registers, three blocks per SM: the pass waits on its neighbour loads (at 88 registers
// and two blocks per SM the whole set-up took 0.267 ms, with three 0.241 ms).
__global__ void __launch_bounds__(256, 3) k_node_gradients(Grid G, Node* __restrict__ bg, NodeDF* __restrict__ bgdf,
                                                          Node32* __restrict__ bg32)
{
    const int64_t total = (int64_t)G.ncell;
    const DF idx{G.df_inv_dX.x, G.df_inv_dX.y}, idy{G.df_inv_dY.x, G.df_inv_dY.y}, idz{G.df_inv_dz.x, G.df_inv_dz.y};
    const DF sx = df_pow2(idx, 0.5f);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < total; c += (int64_t)gridDim.x * blockDim.x) {
        const int k = (int)(c % G.nz);
        const int col = (int)(c / G.nz);
        const int i = col % G.nx, j = col / G.nx;
        const Node* e = bg + node_index(G, i + 1 == G.nx ? 0 : i + 1, j, k);
        const Node* w = bg + node_index(G, i == 0 ? G.nx - 1 : i - 1, j, k);
        const Node *nn, *ss;
        DF sy;
        if (G.geometry == 0) {
            nn = bg + node_index(G, i, j + 1 == G.ny ? 0 : j + 1, k);
            ss = bg + node_index(G, i, j == 0 ? G.ny - 1 : j - 1, k);
            sy = df_pow2(idy, 0.5f);
        } else if (j == 0) {
            nn = bg + node_index(G, i, 1, k);
            ss = bg + node_index(G, i, 0, k);
            sy = idy;
        } else if (j == G.ny - 1) {
            nn = bg + node_index(G, i, G.ny - 1, k);
            ss = bg + node_index(G, i, G.ny - 2, k);
            sy = idy;
        } else {
            nn = bg + node_index(G, i, j + 1, k);
            ss = bg + node_index(G, i, j - 1, k);
            sy = df_pow2(idy, 0.5f);
        }
        const Node *up, *dn;
        DF sz;
        if (k == 0) {
            up = bg + c + 1; dn = bg + c; sz = idz;
        } else if (k == G.nz - 1) {
            up = bg + c; dn = bg + c - 1; sz = idz;
        } else {
            up = bg + c + 1; dn = bg + c - 1; sz = df_pow2(idz, 0.5f);
        }
        auto vals = [](const Node* p) { return *reinterpret_cast<const double4*>(p->v); };
        const double4 ve = vals(e), vw = vals(w), vn = vals(nn), vs = vals(ss), vu = vals(up), vd = vals(dn),
                      vc = vals(bg + c);
        // differences in FP64 (one rounding), scaled in double-float by the spacing reciprocals
        const double dx[4] = {ve.x - vw.x, ve.y - vw.y, ve.z - vw.z, ve.w - vw.w};
        const double dy[4] = {vn.x - vs.x, vn.y - vs.y, vn.z - vs.z, vn.w - vs.w};
        const double dz[4] = {vu.x - vd.x, vu.y - vd.y, vu.z - vd.z, vu.w - vd.w};
        const double val[4] = {vc.x, vc.y, vc.z, vc.w};
        DF q[16];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            q[f] = df_split(val[f]);
            q[4 + 3 * f] = df_mul2(df_split(dx[f]), sx);
            q[5 + 3 * f] = df_mul2(df_split(dy[f]), sy);
            q[6 + 3 * f] = df_mul2(df_split(dz[f]), sz);
        }
        if (bgdf) {
            NodeDF o;
#pragma unroll
            for (int el = 0; el < 8; ++el) o.q[el] = make_float4(q[2 * el].hi, q[2 * el + 1].hi, q[2 * el].lo, q[2 * el + 1].lo);
            bgdf[c] = o;
        }
        if (bg32) {
            // the FP32 node: each quantity rounded once to nearest (hi + lo rounded as a pair)
            Node32 o;
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                o.v[f] = narrow(val[f]);
#pragma unroll
                for (int d = 0; d < 3; ++d) o.d[f][d] = __fadd_rn(q[4 + 3 * f + d].hi, q[4 + 3 * f + d].lo);
            }
            bg32[c] = o;
        }
    }
}

void launch_set_background(Context& c, int member, const double* u, const double* v, const double* n2,
                           const double* rho)
{
    const int TW = kBgTile;
    const int ntx = (c.G.nx + TW - 1) / TW;
    const size_t shm = sizeof(double) * 4 * (size_t)c.G.nz * TW;
    const int64_t o = (int64_t)member * c.G.ncell;
    k_set_background<<<ntx * c.G.ny, kThreads, shm, c.stream>>>(c.G, c.P.gamma_mode, u, v, n2, rho, c.bg + o,
                                                                c.rho + o, c.rho_inv + o, c.flag_dev);
    const int blocks = (int)std::min<int64_t>((c.G.ncell + kThreads - 1) / kThreads, 16384);
    k_node_gradients<<<blocks, kThreads, 0, c.stream>>>(c.G, c.bg + o, c.bgdf ? c.bgdf + o : nullptr,
                                                        c.f32 ? c.bg32 + o : nullptr);
}

// double-float nodes of a precision-form context (its ghost-layer launch integrates the ghost in the
// FP64 form's double-float RK3): from the FP64 node values already set
void node_gradients_df(Context& c, int member)
{
    const int64_t o = (int64_t)member * c.G.ncell;
    const int blocks = (int)std::min<int64_t>((c.G.ncell + kThreads - 1) / kThreads, 16384);
    k_node_gradients<<<blocks, kThreads, 0, c.stream>>>(c.G, c.bg + o, c.bgdf + o, nullptr);
}

// asynchronous background: an invalid value becomes the sticky context status (GWAM_ENUMERIC),
// reported by the next synchronising call; the steps in between do nothing
__global__ void k_flag_to_status(const int* flag, Ctl* ctl)
{
    if (*flag) set_status(ctl, GWAM_ENUMERIC);
}

void launch_flag_to_status(Context& c) { k_flag_to_status<<<1, 1, 0, c.stream>>>(c.flag_dev, c.ctl); }

// 1/rho of restored nodes (checkpoint load), by the Newton reciprocal as in k_set_background
__global__ void k_rho_inv(const double* __restrict__ rho, double* __restrict__ rho_inv, int64_t n)
{
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x) {
        const double r = rho[c];
        rho_inv[c] = (__double_as_longlong(r) > 0 && !nonfinite_bits(r)) ? rcp_nr(r) : 0.0;
    }
}

void restore_background(Context& c, int member)
{
    const int64_t o = (int64_t)member * c.G.ncell;
    const int blocks = (int)std::min<int64_t>((c.G.ncell + kThreads - 1) / kThreads, 16384);
    k_rho_inv<<<blocks, kThreads, 0, c.stream>>>(c.rho + o, c.rho_inv + o, c.G.ncell);
    k_node_gradients<<<blocks, kThreads, 0, c.stream>>>(c.G, c.bg + o, c.bgdf ? c.bgdf + o : nullptr,
                                                        c.f32 ? c.bg32 + o : nullptr);
}

// caller [members][nz][ny][nx] -> column-major reference potential temperature; flags values that
// are not positive and finite
__global__ void k_set_theta(Grid G, const double* __restrict__ theta, double* __restrict__ out, int* flags)
{
    const int64_t total = (int64_t)G.ncell_all;
    int bad = 0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t mem = t / G.ncell, r = t - mem * G.ncell;
        const int i = (int)(r % G.nx), j = (int)((r / G.nx) % G.ny), k = (int)(r / G.ncol);
        const double v = theta[t];
        if (!(v > 0.0) || nonfinite_bits(v)) bad = 1;
        out[mem * G.ncell + node_index(G, i, j, k)] = v;
    }
    if (bad) atomicOr(flags, BG_NONFINITE);
}

void launch_set_theta(Context& c, const double* theta)
{
    const int blocks = (int)std::min<int64_t>((c.G.ncell_all + kThreads - 1) / kThreads, 16384);
    k_set_theta<<<blocks, kThreads, 0, c.stream>>>(c.G, theta, c.theta, c.flag_dev);
}

// Eq. mean-flow-impact-t: d theta/dt = -div <u'theta'>, <u'theta'> = theta-bar / (g rho-bar) T per cell
// from the (smoothed) integrals T_l, T_p; horizontal centred differences as in the momentum
// divergence (flux zero beyond the pole rows), zero in the columnar mode.  Output in the caller's
// [members][nz][ny][nx].  FP64: an on-demand diagnostic, not a per-step kernel.
__global__ void k_theta_div(Grid G, const double* __restrict__ tl, const double* __restrict__ tp,
                            const double* __restrict__ theta, const double* __restrict__ rho_inv,
                            double* __restrict__ out)
{
    const int64_t total = (int64_t)G.ncell_all;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t mem = t / G.ncell, r = t - mem * G.ncell;
        const int i = (int)(r % G.nx), j = (int)((r / G.nx) % G.ny), k = (int)(r / G.ncol);
        if (G.columnar) {
            out[t] = 0.0;
            continue;
        }
        const int64_t o = mem * G.ncell;
        auto thf = [&](const double* a, int ii, int jj) {
            const int64_t c = o + node_index(G, ii, jj, k);
            return a[c] * theta[c] * rho_inv[c] * G.inv_g;
        };
        const int ie = i + 1 == G.nx ? 0 : i + 1, iw = i == 0 ? G.nx - 1 : i - 1;
        double div;
        if (G.geometry == 1) {
            const double yn = j + 1 < G.ny ? G.row_cos[j + 1] * thf(tp, i, j + 1) : 0.0;
            const double ys = j - 1 >= 0 ? G.row_cos[j - 1] * thf(tp, i, j - 1) : 0.0;
            const double dl = (thf(tl, ie, j) - thf(tl, iw, j)) * (0.5 * G.inv_dX);
            const double dp = (yn - ys) * (0.5 * G.inv_dY);
            div = (dl + dp) * G.row_inv_cos[j] * G.lev_inv_r[k];
        } else {
            const int jn = j + 1 == G.ny ? 0 : j + 1, js = j == 0 ? G.ny - 1 : j - 1;
            div = (thf(tl, ie, j) - thf(tl, iw, j)) * (0.5 * G.inv_dX) + (thf(tp, i, jn) - thf(tp, i, js)) * (0.5 * G.inv_dY);
        }
        out[t] = -div;
    }
}

void launch_theta_div(Context& c, const double* tl, const double* tp, double* out)
{
    const int blocks = (int)std::min<int64_t>((c.G.ncell_all + kThreads - 1) / kThreads, 16384);
    k_theta_div<<<blocks, kThreads, 0, c.stream>>>(c.G, tl, tp, c.theta, c.rho_inv, out);
}

// ----------------------------------------------------------------------------- explicit rays

// pass 0 validates, pass 1 writes at n + q with id next_id + q
struct RayInputPtrs {
    const double* p[13];
};

__global__ void k_add_rays(Grid G, RaySoA A, Ray32SoA A32, bool f32, Ctl* ctl, int64_t max_rays, RayInputPtrs in,
                           int n_add, int pass, int* flags, double* partials, int pstride)
{
    const int n0 = ctl->n;
    const long long next = ctl->next_id;
    double w = 0.0;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n_add; q += gridDim.x * blockDim.x) {
        double s[NSTATE];
        s[SX] = in.p[0][q]; s[SY] = in.p[1][q]; s[SZ] = in.p[2][q];
        s[SK] = in.p[3][q]; s[SL] = in.p[4][q]; s[SM] = in.p[5][q];
        s[SEX] = in.p[6][q]; s[SEY] = in.p[7][q]; s[SEZ] = in.p[8][q];
        Geo g;
        geometry_at(G, s[SY], s[SZ], g);
        s[SPX] = g.hX * s[SEX] * in.p[9][q];
        s[SPY] = g.hY * s[SEY] * in.p[10][q];
        s[SPZ] = s[SEZ] * in.p[11][q];
        s[SN] = in.p[12][q];
        wrap_position(G, s);
        if (ray_status(G, s) != 0) {
            atomicOr(flags, 1);
            continue;
        }
        if (pass == 1) {
            const int64_t pos = (int64_t)n0 + q;
            if (pos >= max_rays) {
                set_status(ctl, GWAM_ECAPACITY);
                continue;
            }
            if (f32) {
                S32 r;
                from_double(G, s, next + q, r);
                store32(G, A32, pos, r);
                w += (double)action32(r);
            } else {
                store_ray(A, pos, s, next + q);
                w += ray_action(s);
            }
        }
    }
    const double wb = block_sum(w);
    if (threadIdx.x == 0 && pass == 1) partials[T_LAUNCH * pstride + blockIdx.x] = wb;
}

void launch_add_rays(Context& c, const double* const in[13], int64_t n)
{
    RayInputPtrs d_in;
    for (int q = 0; q < 13; ++q) d_in.p[q] = in[q];
    cudaMemsetAsync(c.flag_dev, 0, sizeof(int), c.stream);
    k_add_rays<<<c.grid_blocks, kThreads, 0, c.stream>>>(c.G, c.A, c.A32, c.f32, c.ctl, c.max_rays, d_in, (int)n, 0,
                                                         c.flag_dev, c.partials, c.max_blocks);
    cudaMemcpyAsync(c.flag_host, c.flag_dev, sizeof(int), cudaMemcpyDeviceToHost, c.stream);
    cudaStreamSynchronize(c.stream);
    if (*c.flag_host) {
        c.err = "gwam_add_rays: a ray volume lies outside the domain or is invalid";
        throw (int)GWAM_EINVAL;
    }
    k_add_rays<<<c.grid_blocks, kThreads, 0, c.stream>>>(c.G, c.A, c.A32, c.f32, c.ctl, c.max_rays, d_in, (int)n, 1,
                                                         c.flag_dev, c.partials, c.max_blocks);
    finalize_launch(c, c.grid_blocks, nullptr, (int)n);
}

// ----------------------------------------------------------------------------- sources (Sec. 3c)

// latitudinal profile alpha(phi), phi in degrees north
__device__ __forceinline__ double alpha_profile(double p)
{
    if (p >= 80.0) return fmin(1.0, fmax(0.0, 1.0 - (p - 80.0) / 5.0));
    if (p >= 50.0) return 1.0;
    if (p >= 20.0) return 0.5 * (1.0 - cos(kPi * (p - 20.0) / 30.0));
    return 0.0;
}

__device__ __forceinline__ double f_am(double p, double tau, double fs, double fw)
{
    const double sol_p = alpha_profile(p) * fs + alpha_profile(-p) * fw;
    const double sol_m = alpha_profile(-p) * fs + alpha_profile(p) * fw;
    const double ct = cos(tau);
    return 0.5 * (sol_p * (1.0 + ct) + sol_m * (1.0 - ct));
}

// What a launch needs of its column at the launch level; flux = the flux of one bin, hY = 0 where the
// source does not launch.  64 bytes.
struct LaunchColumn {
    double U, V, N2, G2, f2, hX, hY, flux;
};

__device__ __forceinline__ void launch_column(const Grid& G, const Node* __restrict__ bg, int i, int j, double Z,
                                              LaunchColumn& col)
{
    const double X = __dmul_rn(i + 0.5, G.dX), Y = row_lat(G, j);
    double v[4];
    gather_values_fp64(G, bg, X, Y, Z, v);
    Geo g;
    geometry_at(G, Y, Z, g);
    double df2;
    coriolis(G, g.sphi, g.cphi, col.f2, df2);
    col.U = v[0]; col.V = v[1]; col.N2 = v[2]; col.G2 = v[3];
    col.hX = g.hX; col.hY = g.hY;
}

// The launch state of a bin (horizontal wavenumber kh in direction (ct, st), phase speed c) in column
// (i, j): 0 = filtered, 1 = launched (state in s)
__device__ __forceinline__ int launch_state(const Grid& G, const LaunchColumn& col, int i, int j, double z_launch,
                                            double dz_launch, double kh, double st, double ct, double c,
                                            double flux, double frac, double s[NSTATE])
{
    const double U = col.U, V = col.V, N2 = col.N2, G2 = col.G2, f2 = col.f2;
    const double k = kh * ct, l = kh * st;
    const double w = kh * c - (k * U + l * V);
    if (!(w > 0.0 && w * w > f2 && w * w < N2)) return 0;
    const double m2 = kh * kh * (N2 - w * w) / (w * w - f2) - G2;
    if (!(m2 > 0.0)) return 0;
    const double m = -sqrt(m2);
    Disp d;
    dispersion(kh * kh, m2 + G2, N2, f2, d);
    const double chr = -m * kh * kh * d.c;
    const double A = flux / (kh * chr);   // once per launched ray: IEEE division is fine here
    const double dk = frac * kh, dl = frac * kh, dm = frac * fabs(m);
    s[SX] = __dmul_rn(i + 0.5, G.dX); s[SY] = row_lat(G, j); s[SZ] = z_launch + 0.5 * dz_launch;
    s[SK] = k; s[SL] = l; s[SM] = m;
    s[SEX] = G.dX; s[SEY] = G.dY; s[SEZ] = dz_launch;
    s[SPX] = col.hX * G.dX * dk;
    s[SPY] = col.hY * G.dY * dl;
    s[SPZ] = dz_launch * dm;
    s[SN] = A / (dk * dl * dm);
    return ray_status(G, s) == 0 ? 1 : 0;
}

// The background source's columns, a thread each: the trilinear values, the metric and the seasonal
// flux are FP64 work that all bins of a column share (they took most of a launch while every bin
// repeated them).
__global__ void k_launch_columns(Grid G, const Node* __restrict__ bg, gwam_bg_source src, LaunchColumn* __restrict__ cols)
{
    const double Z = src.z_launch + 0.5 * src.dz_launch;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G.ncol_all; g += gridDim.x * blockDim.x) {
        const int mem = g / G.ncol, col = g - mem * G.ncol;
        const int j = col / G.nx, i = col - j * G.nx;
        const double pdeg = row_lat(G, j) * (180.0 / kPi);
        LaunchColumn o{};
        bool on = !(fabs(pdeg) > src.phi_max_deg);
        if (on) {
            const double fbin = f_am(pdeg, src.tau, src.f_s, src.f_w) / (src.n_az * src.n_c);
            on = !(fbin == 0.0 && !src.launch_zero_flux);
            if (on) {
                launch_column(G, bg + (int64_t)mem * G.ncell, i, j, Z, o);
                o.flux = fbin;
            }
        }
        cols[g] = o;
    }
}

// device-resident specs are not seen by the host: a column or member outside the grid is an
// input error (status GWAM_EINVAL, read at the next synchronising call), never an index
__device__ __forceinline__ bool spec_in_grid(const Grid& G, Ctl* ctl, const gwam_spec& sp)
{
    if (sp.i >= 0 && sp.i < G.nx && sp.j >= 0 && sp.j < G.ny && sp.member >= 0 && sp.member < G.members) return true;
    set_status(ctl, GWAM_EINVAL);
    return false;
}

// Ghost-layer emission (Sec. 3c): the launch state s fills the layer [z_launch, z_launch + dz_launch]
// and propagates vertically only over the launch interval dt (single-column RK3: G.columnar is set
// on the grid this kernel is given).  Returns 1 with s = the part above the layer top (vertical
// extent from the layer top, or the ghost's own bottom if it left whole, to its top; P_z in
// proportion; the ghost's m), 0 when the ghost was reflected in the layer (m no longer negative) or
// the part lies outside the domain, 2 when nothing has left the layer.  All 32 lanes of a warp must
// call it (their stages gather together); lanes without a launch state (on = false) return 0.
__device__ __forceinline__ int ghost_emit(const Grid& G, const NodeDF* __restrict__ bgdf, bool on, int member,
                                          double z_launch, double dz_launch, double dt, double s[NSTATE],
                                          const RkSlots& sl)
{
    double y[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) y[c] = on ? s[c] : 0.0;
    rk3_start(sl, y);
    rk3(G, bgdf, on ? member * G.ncell : 0, dt, sl);
    if (!on) return 0;
#pragma unroll
    for (int c = 0; c < 9; ++c) y[c] += rk_increment(sl, c);
    if (!(y[SM] < 0.0)) return 0;
    const double layer_top = z_launch + dz_launch;
    const double top = y[SZ] + 0.5 * y[SEZ], bot = y[SZ] - 0.5 * y[SEZ];
    if (!(top > layer_top)) return 2;
    const double lo = bot > layer_top ? bot : layer_top;
    s[SM] = y[SM];
    s[SZ] = 0.5 * (lo + top);
    s[SEZ] = top - lo;
    s[SPZ] = s[SPZ] * s[SEZ] / y[SEZ];   // once per emitted ray: IEEE division is fine here
    return ray_status(G, s) == 0 ? 1 : 0;
}

// Launch states of all bins: flag[t] = launched, the state (record of the context's form, id = the
// member alone) staged at position t of S / S32, filtered bins counted; k_launch_place then moves the
// launched ones behind the live rays.  (While both passes computed the states, a ghost-layer launch
// into 8192 columns took 2 x 390 us.)  kGhost: what left the ghost layer over ghost_dt instead of
// the launch state itself.  The source's bins are counted from bin0 of column col0 on.  Dynamic shared
// memory: the ghost's kRkWarp a warp, then the source's sines and cosines of the azimuths and its phase speeds
// (2 n_az + n_c doubles).
template <bool kSpec, bool kGhost>
__global__ void __launch_bounds__(kThreads, 2) k_launch(Grid G, const Node* __restrict__ bg,
                                                        const NodeDF* __restrict__ bgdf, RaySoA S, Ray32SoA S32s, bool f32,
                                                        Ctl* ctl, gwam_bg_source src,
                                                        const LaunchColumn* __restrict__ cols,
                                                        const gwam_spec* __restrict__ specs, int col0, int bin0, int total,
                                                        double ghost_dt, int* __restrict__ flag)
{
    extern __shared__ float4 sh_launch[];
    double* const az = reinterpret_cast<double*>(sh_launch + (kGhost ? kRkWarp * (blockDim.x / 32) : 0));
    double* const speed = az + 2 * src.n_az;
    const int nbins = kSpec ? 1 : src.n_az * src.n_c;
    if (!kSpec) {
        for (int a = threadIdx.x; a < src.n_az; a += blockDim.x) sincos(2.0 * kPi * a / src.n_az, &az[2 * a], &az[2 * a + 1]);
        for (int q = threadIdx.x; q < src.n_c; q += blockDim.x)
            speed[q] = src.n_c == 1 ? src.c_min : src.c_min * pow(src.c_max / src.c_min, (double)q / (src.n_c - 1));
        __syncthreads();
    }
    const double kh_src = kSpec ? 0.0 : 2.0 * kPi / src.lambda_h;
    long long filtered = 0;
    for (int t0 = blockIdx.x * blockDim.x; t0 < total; t0 += gridDim.x * blockDim.x) {
        const int t = t0 + threadIdx.x;
        double s[NSTATE];
        bool eligible = t < total;
        int ok = 0, mem = 0;
        double z_launch = src.z_launch, dz_launch = src.dz_launch;
        if (eligible && kSpec) {
            const gwam_spec sp = specs[t];
            eligible = spec_in_grid(G, ctl, sp);
            if (eligible) {
                mem = sp.member;
                z_launch = sp.z_launch;
                dz_launch = sp.dz_launch;
                LaunchColumn col;
                launch_column(G, bg + (int64_t)mem * G.ncell, sp.i, sp.j, z_launch + 0.5 * dz_launch, col);
                double st, ct;
                sincos(sp.theta, &st, &ct);
                ok = launch_state(G, col, sp.i, sp.j, z_launch, dz_launch, 2.0 * kPi / sp.lambda_h, st, ct, sp.c, sp.flux,
                                  sp.spectral_frac, s);
            }
        } else if (eligible) {
            const int q = (bin0 + t) / nbins, g = col0 + q, bin = bin0 + t - q * nbins;
            const LaunchColumn col = cols[g];
            eligible = col.hY != 0.0;
            if (eligible) {
                mem = g / G.ncol;
                const int c = g - mem * G.ncol, j = c / G.nx, a = bin / src.n_c;
                ok = launch_state(G, col, c - j * G.nx, j, z_launch, dz_launch, kh_src, az[2 * a], az[2 * a + 1],
                                  speed[bin - a * src.n_c], col.flux, src.spectral_frac, s);
            }
        }
        if (kGhost && __any_sync(0xffffffffu, ok)) {
            const int e = ghost_emit(G, bgdf, ok != 0, mem, z_launch, dz_launch, ghost_dt, s, RkSlots(sh_launch));
            if (e == 2) eligible = false;      // nothing left the layer: neither launched nor filtered
            ok = e == 1;
        }
        if (t >= total) continue;
        if (eligible && !ok) ++filtered;
        flag[t] = ok;
        if (!ok) continue;
        if (f32) {
            S32 r;
            from_double(G, s, with_member(mem, 0), r);
            store32(G, S32s, t, r);
        } else {
            store_ray(S, t, s, with_member(mem, 0));
        }
    }
    const long long fb = block_sum(filtered);
    if (threadIdx.x == 0 && fb) atomicAdd((unsigned long long*)&ctl->n_filtered, (unsigned long long)fb);
}

// The staged launches t with off[t + 1] > off[t] to position n + off[t], id next_id + off[t]
__global__ void k_launch_place(Grid G, RaySoA S, Ray32SoA S32s, RaySoA A, Ray32SoA A32, bool f32, Ctl* ctl,
                               int64_t max_rays, int total, const int* __restrict__ off, double* __restrict__ partials,
                               int pstride)
{
    const int n0 = ctl->n;
    const long long next = ctl->next_id;
    double w = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int o = off[t];
        if (off[t + 1] == o) continue;
        const int64_t pos = (int64_t)n0 + o;
        if (pos >= max_rays) {
            set_status(ctl, GWAM_ECAPACITY);
            continue;
        }
        if (f32) {
            S32 r;
            load32(G, S32s, t, r);
            r.id += next + o;
            store32(G, A32, pos, r);
            w += (double)action32(r);
        } else {
            double s[NSTATE];
            long long id;
            load_ray(S, t, s, id);
            store_ray(A, pos, s, id + next + o);
            w += ray_action(s);
        }
    }
    const double wb = block_sum(w);
    if (threadIdx.x == 0) partials[T_LAUNCH * pstride + blockIdx.x] = wb;
}

void configure_launch_kernels()
{
    cudaFuncSetAttribute(k_set_background, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    // a source has at most 1024 bins, so n_az + n_c <= 1025
    cudaFuncSetAttribute(k_launch<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kRkSmem + 2050 * sizeof(double)));
    cudaFuncSetAttribute(k_launch<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRkSmem);
}

// Launches of more bins than the context holds ray volumes (most bins filtered, or an overflow to be reported)
// go in parts: of this many bins, or of max_rays, whichever is more
constexpr int64_t kLaunchPart = 1 << 18;

static void launch_common(Context& c, const gwam_bg_source* src, const gwam_spec* specs, int64_t total,
                          double ghost_dt = 0.0)
{
    if (total <= 0) return;
    const int nb = c.grid_blocks;
    const bool ghost = ghost_dt > 0.0;
    // The re-binned ray buffer is free between steps: launch states of up to max_rays bins are staged
    // there, their flags in the per-ray scratch.  A part of more bins than that brings its own (30 MB; for
    // all bins at once it would be 116 bytes each, gigabytes on a large grid with many bins), or, where that
    // cannot be had, is cut down until it can or fits the free buffer.
    RaySoA S = c.B;
    Ray32SoA S32s = c.B32;
    int* flag = c.newid;
    char* own = nullptr;
    int64_t part = std::min(total, std::max(c.max_rays, kLaunchPart));
    const size_t rec = c.f32 ? 4 * sizeof(float4) : 7 * sizeof(double2);
    while (part > c.max_rays) {
        if (cudaMallocAsync((void**)&own, rec * (size_t)part + sizeof(int) * (size_t)(part + 1), c.stream) == cudaSuccess) {
            for (int q = 0; q < 7; ++q) S.a[q] = reinterpret_cast<double2*>(own) + q * part;
            for (int q = 0; q < 4; ++q) S32s.q[q] = reinterpret_cast<float4*>(own) + q * part;
            flag = reinterpret_cast<int*>(own + rec * (size_t)part);
            break;
        }
        cudaGetLastError();
        own = nullptr;
        part = std::max(c.max_rays, part / 2);
    }
    gwam_bg_source s0{};
    if (src) s0 = *src;
    // the ghost layer propagates vertically only: the single-column equations on this grid copy
    Grid G = c.G;
    if (ghost) G.columnar = 1;
    if (!specs) {
        const int cb = std::min((c.G.ncol_all + 31) / 32, 32 * c.num_sms);
        k_launch_columns<<<cb, 32, 0, c.stream>>>(c.G, c.bg, s0, reinterpret_cast<LaunchColumn*>(c.launch_cols));
    }
    const int nbins = specs ? 1 : s0.n_az * s0.n_c;
    auto* kernel = specs ? (ghost ? k_launch<true, true> : k_launch<true, false>)
                         : (ghost ? k_launch<false, true> : k_launch<false, false>);
    for (int64_t first = 0; first < total; first += part) {
        const int64_t n = std::min(part, total - first);
        // one wave of two blocks per SM; few bins in blocks of a warp, spread over the SMs (the bins' FP64
        // chains share an SM's FP64 pipe: 200 bins in one block took 16 us)
        const int threads = n >= 2 * (int64_t)c.num_sms * kThreads ? kThreads : 32;
        const int blocks = (int)std::min<int64_t>((int64_t)nb * (kThreads / threads), (n + threads - 1) / threads);
        const size_t shm =
            (ghost ? kRkSmem / (kThreads / threads) : 0) + (specs ? 0 : (2 * s0.n_az + s0.n_c) * sizeof(double));
        kernel<<<blocks, threads, shm, c.stream>>>(
            G, c.bg, c.bgdf, S, S32s, c.f32, c.ctl, s0, reinterpret_cast<const LaunchColumn*>(c.launch_cols),
            specs ? specs + first : nullptr, (int)(first / nbins), (int)(first % nbins), (int)n, ghost_dt, flag);
        exclusive_scan(c, flag, flag, n, nullptr);
        const int pb = std::min<int>(nb, (int)((n + kThreads - 1) / kThreads));
        k_launch_place<<<pb, kThreads, 0, c.stream>>>(c.G, S, S32s, c.A, c.A32, c.f32, c.ctl, c.max_rays, (int)n, flag,
                                                      c.partials, c.max_blocks);
        finalize_launch(c, pb, flag, (int)n);
    }
    if (own) cudaFreeAsync(own, c.stream);
}

void launch_background_source(Context& c, const gwam_bg_source& src)
{
    const int64_t total = (int64_t)c.G.ncol_all * src.n_az * src.n_c;
    launch_common(c, &src, nullptr, total);
}

void launch_spectral(Context& c, const gwam_spec* specs, int64_t n) { launch_common(c, nullptr, specs, n); }

void launch_ghost_source(Context& c, const gwam_bg_source& src, double dt)
{
    const int64_t total = (int64_t)c.G.ncol_all * src.n_az * src.n_c;
    launch_common(c, &src, nullptr, total, dt);
}

void launch_ghost_spectral(Context& c, const gwam_spec* specs, int64_t n, double dt)
{
    launch_common(c, nullptr, specs, n, dt);
}

}  // namespace gwam

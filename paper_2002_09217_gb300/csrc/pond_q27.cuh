// pond_q27.cuh -- the PonD van der Waals time step in three dimensions on the D3Q27
// lattice for sm_103a.
//
// The model is written for D dimensions (D enters the energy equilibrium and the
// heat-flux correction); D3Q27 = C1 x C1 x C1 with C1 = {-1, 0, 1}, weights 1/6, 2/3,
// 1/6 per axis and T_L = 1/3.  The transfer map G = M_lambda'^-1 M_lambda over the 27
// moments M_lmn (l, m, n <= 2) is the product of three 3-node Lagrange maps, one per axis
// (SM "Transfer matrix"); reconstruction uses the 4 x 4 x 4 cubic stencil (one cubic
// factor per axis, SM "Reconstruction").  The forced g equilibrium takes its 3-D tensors
// I_ab = uhat_a F_b + F_a uhat_b + dt F_a F_b E/(2P), M_a = (dt rho/P)(F_a H - I_ab u_b),
// N_ab = rho delta_ab + (dt rho/(2P)) I_ab.
//
// Layout: one record of SL27 = 68 values per node (node = (z*ny + y)*nx + x), in 16-byte
// chunks with chunk c of all nodes together (rec27_at):
//   [0] theta, [1..3] u, [4..30] f_0..f_26, [31..57] g_0..g_26, [58] rho, [59] T,
//   [60..62] uhat, [63] mass lo, [64..66] momentum lo, [67] energy lo
// with population i = 9*jz + 3*jy + jx, c = j - 1.  The lo values (FP32 form only) are what
// storage rounding took from the node's exact mass, momentum and energy (as on D2Q9 and
// D2Q16).
//
// One step is four launches: p/rho; the Korteweg stress and heat-flux vector of the state
// the non-local terms come from; their divergences; and the node step.
//
// The node step streams as the D2Q9 step does (pond_step.cuh): a block's tile of 8 x 4 x 4
// nodes with a halo of two is carried once into a common gauge in shared memory, and each
// thread contracts its node's 5 x 5 x 5 window axis by axis (x, y, z) with weights that
// combine the cubic Lagrange weights and the rows of the map into the arrival gauge: 12,560
// (FP32) or 10,530 (FP64) multiply-adds a population family, where carrying each of 125
// nodes into the arrival gauge and spreading it over 27 directions took about 45,000.  One family at a time is
// staged (two blocks per SM in FP32, one in FP64, by shared memory); a further stream of
// the frame search starts with the family that is already staged.  The sums of populations,
// the moments, the EoS and the non-local terms are float-float in the FP32 form.
// Measured: two mixed steps of a 96 x 96 x 64 droplet (with init and read-out) 29.3 -> 6.0
// ms, two FP64 steps of 33 x 29 x 21 nodes 152 -> 21 ms.  With two warps per scheduler the
// shared-memory latency decides: a row's slots are replaced by the next row's as they are
// used (3.78 -> 2.88 ms a step; issue 41 -> 53 %, FMA pipe 53 % busy).
#pragma once

#include "pond_kernels.cuh"
#include "pond_step.cuh"   // float-float and wide values, map helpers

namespace pond {

constexpr int Q27 = 27;
constexpr int NP27 = 2 * Q27 + 9;   // planes of the exchanged D3Q27 state
constexpr int SL27 = 68;
enum : int { R_TH = 0, R_UX = 1, R_F = 4, R_G = 31, R_RHO = 58, R_T = 59, R_UHX = 60, R_MLO = 63,
             R_JLO = 64, R_GLO = 67 };
// 8-byte scratch planes of the non-local terms (FP64; float-float pairs in the FP32 form)
enum : int { N3_K = 0 /* xx, xy, xz, yy, yz, zz */, N3_Q = 6, N3_REL = 9, N3_F = 10, N3_M0 = 13, N3_PI = 14,
             N3_PLANES = 15 };

// record offset of plane p of the exchanged state (f, g, theta, u, rho, T, uhat)
__host__ __device__ constexpr int rec27_off(int p) { return p < 54 ? p + 4 : (p < 58 ? p - 54 : p); }

#define REC27(buf, n, off) (buf)[rec_at(buf, (size_t)(n), (off), (size_t)p.N)]
#define NL3(buf, plane, n, N) (buf)[(size_t)(plane) * (size_t)(N) + (size_t)(n)]

struct Grid3 {
    int nz, bcz;
};

__device__ __forceinline__ long long node27(const DevParams &p, const Grid3 &g, int x, int y, int z)
{
    return ((long long)bc_wrap(z, g.nz, g.bcz) * p.ny + bc_wrap(y, p.ny, p.bcy)) * p.nx + bc_wrap(x, p.nx, p.bcx);
}

template <typename A>
__device__ __forceinline__ A sel3(const A (&v)[3], int k)
{
    return k == 0 ? v[0] : (k == 1 ? v[1] : v[2]);
}

// Row k of a per-axis 3-node transfer map in increment form (nodes -1, 0, 1 in the
// target's units; source velocities at c_j + eps_j): D[k][j] = l_k(c_j + eps_j) - delta_kj,
// off-diagonal entries carry the exact factor eps_j, the diagonal is
// (1 + eps_k/(c_k - o0))(1 + eps_k/(c_k - o1)) - 1 expanded.
template <typename A>
__device__ __forceinline__ void inc_row3(int k, const A (&eps)[3], A (&out)[3])
{
    // l_k(xi) = prod_{m != k} (xi - c_m) / (c_k - c_m), c = -1, 0, 1: the inverse
    // denominators (1/2, -1, 1/2) and 1/(c_k - o_m) are exact binary constants
    const A id = k == 1 ? A(-1) : A(0.5);
    const A r0 = k == 0 ? A(-1) : (k == 1 ? A(1) : A(0.5));     // 1/(c_k - o0), o0 < o1
    const A r1 = k == 0 ? A(-0.5) : (k == 1 ? A(-1) : A(1));    // 1/(c_k - o1)
    const A ek = sel3(eps, k);
    const A t0 = ek * r0, t1 = ek * r1;
    const A diag = (t0 + t1) + t0 * t1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        // the factors (c_j - c_m) + eps_j for m = 0, 1, 2 (the one with m = j is eps_j)
        const A f0 = A(j) + eps[j], f1 = A(j - 1) + eps[j], f2 = A(j - 2) + eps[j];
        const A prod = k == 0 ? f1 * f2 : (k == 1 ? f0 * f2 : f0 * f1);
        out[j] = j == k ? diag : id * prod;
    }
}

template <typename A>
__host__ __device__ __forceinline__ void cubic_w(A xi, A a[4])
{
    const A x0 = xi, x1 = xi - A(1), x2 = xi - A(2), x3 = xi - A(3);
    a[0] = -(x1 * x2 * x3) / A(6);
    a[1] = (x0 * x2 * x3) * A(0.5);
    a[2] = -(x0 * x1 * x3) * A(0.5);
    a[3] = (x0 * x1 * x2) / A(6);
}

template <typename A>
__host__ __device__ __forceinline__ int depart(int X, A v, A dt, A w[4])
{
    const A d = -v * dt;
    const A fl = floor(d);
    cubic_w<A>(d - fl + A(1), w);
    return stencil_start(X, fl);
}

__device__ __forceinline__ double w27(int i) { return w1d(i % 3) * w1d((i / 3) % 3) * w1d(i / 9); }

// Values OFF .. OFF + CNT - 1 of node nd's record, by the 16-byte chunks that cover them.
template <int OFF, int CNT>
__device__ __forceinline__ void load27(const float *__restrict__ b, size_t nd, size_t N, float *v)
{
    const float4 *q = reinterpret_cast<const float4 *>(b) + nd;
#pragma unroll
    for (int c = OFF / 4; c <= (OFF + CNT - 1) / 4; ++c) {
        const float4 t = __ldg(q + (size_t)c * N);
        const float x[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = 4 * c + e - OFF;
            if (i >= 0 && i < CNT) v[i] = x[e];
        }
    }
}
template <int OFF, int CNT>
__device__ __forceinline__ void load27(const double *__restrict__ b, size_t nd, size_t N, double *v)
{
    const double2 *q = reinterpret_cast<const double2 *>(b) + nd;
#pragma unroll
    for (int c = OFF / 2; c <= (OFF + CNT - 1) / 2; ++c) {
        const double2 t = __ldg(q + (size_t)c * N);
        const double x[2] = {t.x, t.y};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = 2 * c + e - OFF;
            if (i >= 0 && i < CNT) v[i] = x[e];
        }
    }
}

// ---------------------------------------------------------------------------
// Non-local terms, stage 0: p/rho of every node of `src`.
template <typename R>
__global__ void k_q27_pi(DevParams p, const R *__restrict__ src, typename Wide<R>::type *__restrict__ nl)
{
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    NL3(nl, N3_PI, n, p.N) = w_p_over_rho(p, REC27(src, n, R_RHO), REC27(src, n, R_T));
}

// First differences of a field over the 3 x 3 x 3 neighbourhood by the isotropic stencils,
// unnormalised: with D = phi(+1) - phi(-1) and S = phi(-1) + 4 phi(0) + phi(+1) per axis,
// d[a] = D along a and S along the other axes, s = S along all three.  The stencils are
// products over the axes, so nine lines, three planes and one column replace 27 weighted
// terms for each.
template <typename A> struct Diff3 { A d[3], s; };
template <typename A, typename Get>
__device__ __forceinline__ Diff3<A> diff3(Get get)
{
    A SD[3], DS[3], SS[3];
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        A D[3], S[3];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const auto a = get(z, y, 0), b = get(z, y, 1), c = get(z, y, 2);
            D[y] = w_sub(c, a);
            S[y] = w_add(w_add(a, c), w_x4(b));
        }
        SD[z] = w_add(w_add(D[0], D[2]), w_x4(D[1]));
        DS[z] = w_sub(S[2], S[0]);
        SS[z] = w_add(w_add(S[0], S[2]), w_x4(S[1]));
    }
    Diff3<A> o;
    o.d[0] = w_add(w_add(SD[0], SD[2]), w_x4(SD[1]));
    o.d[1] = w_add(w_add(DS[0], DS[2]), w_x4(DS[1]));
    o.d[2] = w_sub(SS[2], SS[0]);
    o.s = w_add(w_add(SS[0], SS[2]), w_x4(SS[1]));
    return o;
}

// Indices of the 27 neighbours of a node after the boundary rules.
struct Near27 {
    int x[3];
    long long row[3][3];   // [z][y]
    __device__ __forceinline__ Near27(const DevParams &p, const Grid3 &g, long long n)
    {
        const int X = (int)(n % p.nx), Y = (int)((n / p.nx) % p.ny), Z = (int)(n / ((long long)p.nx * p.ny));
#pragma unroll
        for (int k = 0; k < 3; ++k) x[k] = bc_wrap(X + k - 1, p.nx, p.bcx);
#pragma unroll
        for (int z = 0; z < 3; ++z)
#pragma unroll
            for (int y = 0; y < 3; ++y)
                row[z][y] = ((long long)bc_wrap(Z + z - 1, g.nz, g.bcz) * p.ny + bc_wrap(Y + y - 1, p.ny, p.bcy)) * p.nx;
    }
    __device__ __forceinline__ long long at(int z, int y, int k) const { return row[z][y] + x[k]; }
};

// Stage 1 (rho, T of `src`): K = -kappa (rho lap rho + |grad rho|^2/2) I + kappa grad rho
// (x) grad rho, q = -mu grad h + k grad T (h = C_v T - a rho + p/rho), rho E_lambda = kappa
// |grad rho|^2 / 2, with grad = 3 sum W c phi(x + c) = d / 72 and lap = 6 sum W (phi(x + c)
// - phi(x)) = s / 36 of the differences to the centre.
template <typename R>
__global__ void k_q27_nonlocal1(DevParams p, Grid3 g3, const R *__restrict__ src, typename Wide<R>::type *__restrict__ nl)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const long long N = p.N;
    const Near27 nb(p, g3, n);
    const R r0 = REC27(src, n, R_RHO);
    const A pi0 = NL3(nl, N3_PI, n, N);
    const Diff3<A> dr = diff3<A>([&](int z, int y, int k) { return w_sub(REC27(src, nb.at(z, y, k), R_RHO), r0); });
    const Diff3<A> dT = diff3<A>([&](int z, int y, int k) { return REC27(src, nb.at(z, y, k), R_T); });
    const Diff3<A> dp = diff3<A>([&](int z, int y, int k) { return NL3(nl, N3_PI, nb.at(z, y, k), N); });
    const A g = w_const<A>(1.0 / 72.0), kap = wide_param<A>(p.kappa, p.ff_kap);
    A gr[3], gT[3], gh[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        gr[a] = w_mul(dr.d[a], g);
        gT[a] = w_mul(dT.d[a], g);
        gh[a] = w_add(w_sub(w_mul(gT[a], wide_param<A>(p.cv, p.ff_cv)), w_mul(gr[a], wide_param<A>(p.a, p.ff_a))), w_mul(dp.d[a], g));
    }
    const A lap = w_mul(dr.s, w_const<A>(1.0 / 36.0));
    const A g2 = w_add(w_add(w_mul(gr[0], gr[0]), w_mul(gr[1], gr[1])), w_mul(gr[2], gr[2]));
    const A kg2 = w_mul(kap, w_mul(g2, w_const<A>(0.5)));   // rho E_lambda
    const A iso = w_sub(w_mul(w_mul(kap, w_mul(lap, r0)), w_const<A>(-1.0)), kg2);
    const A pr = w_mul(pi0, r0);
    const A mu = w_mul(w_less(wide_p_floor<A>(p), pr) ? pr : wide_p_floor<A>(p), wide_param<A>(p.pd.mu_coef, p.ff_mu));
    const A kc = p.k_cond >= 0.0 ? wide_param<A>(p.k_cond, p.ff_kc) : w_mul(mu, wide_param<A>(p.pd.cvR, p.ff_cvR));
    const int ab[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int a = ab[k][0], b = ab[k][1];
        const A gg = w_mul(kap, w_mul(gr[a], gr[b]));
        NL3(nl, N3_K + k, n, N) = a == b ? w_add(iso, gg) : gg;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) NL3(nl, N3_Q + a, n, N) = w_sub(w_mul(kc, gT[a]), w_mul(mu, gh[a]));
    NL3(nl, N3_REL, n, N) = kg2;
}

// Stage 2: F_a = -d_b K_ab and M_0 = 2 div q (the same stencils).
template <typename R>
__global__ void k_q27_nonlocal2(DevParams p, Grid3 g3, typename Wide<R>::type *__restrict__ nl)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const long long N = p.N;
    const Near27 nb(p, g3, n);
    auto diff = [&](int plane) { return diff3<A>([&](int z, int y, int k) { return NL3(nl, plane, nb.at(z, y, k), N); }); };
    A F[3], dq;
    {
        const Diff3<A> xx = diff(N3_K), xy = diff(N3_K + 1);
        F[0] = w_add(xx.d[0], xy.d[1]);
        F[1] = xy.d[0];
    }
    {
        const Diff3<A> xz = diff(N3_K + 2), yy = diff(N3_K + 3);
        F[0] = w_add(F[0], xz.d[2]);
        F[2] = xz.d[0];
        F[1] = w_add(F[1], yy.d[1]);
    }
    {
        const Diff3<A> yz = diff(N3_K + 4), zz = diff(N3_K + 5);
        F[1] = w_add(F[1], yz.d[2]);
        F[2] = w_add(w_add(F[2], yz.d[1]), zz.d[2]);
    }
    {
        const Diff3<A> qx = diff(N3_Q), qy = diff(N3_Q + 1), qz = diff(N3_Q + 2);
        dq = w_add(w_add(qx.d[0], qy.d[1]), qz.d[2]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) NL3(nl, N3_F + a, n, N) = w_mul(F[a], w_const<A>(-1.0 / 72.0));
    NL3(nl, N3_M0, n, N) = w_mul(dq, w_const<A>(2.0 / 72.0));
}

// ---------------------------------------------------------------------------
// Streaming into node (X, Y, Z) in gauge (th, u): for direction i = (ix, iy, iz) the
// departure point x - v_i dt is reconstructed from the 4 x 4 x 4 nodes around it, each
// carried into the arrival gauge by the three per-axis maps in increment form.  Returns
// the increments of the streamed f_i, g_i over the node's own stored values.
template <typename R>
__device__ void q27_stream(const DevParams &p, const Grid3 &g3, const R *__restrict__ in, int X, int Y,
                           int Z, R th, const R (&u)[3], R *fi, R *gi)
{
    const long long nself = ((long long)Z * p.ny + Y) * p.nx + X;
    const R s = sqrt_(th), is = R(1) / s, dt = (R)p.dt;
#pragma unroll 1
    for (int i = 0; i < Q27; ++i) {
        const int ix = i % 3, iy = (i / 3) % 3, iz = i / 9;
        R ax[4], ay[4], az[4];
        const int x0 = depart<R>(X, s * R(ix - 1) + u[0], dt, ax);
        const int y0 = depart<R>(Y, s * R(iy - 1) + u[1], dt, ay);
        const int z0 = depart<R>(Z, s * R(iz - 1) + u[2], dt, az);
        const R refF = REC27(in, nself, R_F + i), refG = REC27(in, nself, R_G + i);
        R sf = R(0), sg = R(0);
#pragma unroll 2
        for (int q = 0; q < 64; ++q) {
            const int k = q & 3, m = (q >> 2) & 3, l = q >> 4;
            const R wgt = ax[k] * ay[m] * az[l];
            const size_t nd = (size_t)node27(p, g3, x0 + k, y0 + m, z0 + l);
            R gv[4];
            load27<R_TH, 4>(in, nd, (size_t)p.N, gv);
            const R ths = gv[0];
            const R ds = (ths - th) / (sqrt_(ths) + s) * is;   // (s' - s)/s
            R ex[3], ey[3], ez[3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                ex[j] = ds * R(j - 1) + (gv[1] - u[0]) * is;
                ey[j] = ds * R(j - 1) + (gv[2] - u[1]) * is;
                ez[j] = ds * R(j - 1) + (gv[3] - u[2]) * is;
            }
            R Dx[3], Dy[3], Dz[3];
            inc_row3<R>(ix, ex, Dx);
            inc_row3<R>(iy, ey, Dy);
            inc_row3<R>(iz, ez, Dz);
            R v[54];
            load27<R_F, 54>(in, nd, (size_t)p.N, v);
#pragma unroll
            for (int pg = 0; pg < 2; ++pg) {
                const R *f = v + 27 * pg;
                // rows (jz, jy): base f_(jz, jy, ix) and x-increment
                R b[3][3], xr[3][3];
#pragma unroll
                for (int jz = 0; jz < 3; ++jz)
#pragma unroll
                    for (int jy = 0; jy < 3; ++jy) {
                        const R r0 = f[9 * jz + 3 * jy], r1 = f[9 * jz + 3 * jy + 1], r2 = f[9 * jz + 3 * jy + 2];
                        const R row[3] = {r0, r1, r2};
                        b[jz][jy] = sel3(row, ix);
                        xr[jz][jy] = Dx[0] * r0 + Dx[1] * r1 + Dx[2] * r2;
                    }
                // y-increment per jz plane, then the z-increment
                R yz[3], tz[3];
#pragma unroll
                for (int jz = 0; jz < 3; ++jz) {
                    R a = R(0);
#pragma unroll
                    for (int jy = 0; jy < 3; ++jy) a += Dy[jy] * (b[jz][jy] + xr[jz][jy]);
                    yz[jz] = a;
                    const R bb[3] = {b[jz][0], b[jz][1], b[jz][2]}, xx[3] = {xr[jz][0], xr[jz][1], xr[jz][2]};
                    tz[jz] = sel3(bb, iy) + sel3(xx, iy) + a;
                }
                const R zinc = Dz[0] * tz[0] + Dz[1] * tz[1] + Dz[2] * tz[2];
                // [G f]_i - ref = (f_i - ref) + x-inc + y-inc + z-inc of row (iz, iy)
                R bi, xi_, yi;
                {
                    const R b0[3] = {b[0][0], b[0][1], b[0][2]}, b1[3] = {b[1][0], b[1][1], b[1][2]},
                            b2[3] = {b[2][0], b[2][1], b[2][2]};
                    const R x0r[3] = {xr[0][0], xr[0][1], xr[0][2]}, x1r[3] = {xr[1][0], xr[1][1], xr[1][2]},
                            x2r[3] = {xr[2][0], xr[2][1], xr[2][2]};
                    const R bsel[3] = {sel3(b0, iy), sel3(b1, iy), sel3(b2, iy)};
                    const R xsel[3] = {sel3(x0r, iy), sel3(x1r, iy), sel3(x2r, iy)};
                    bi = sel3(bsel, iz);
                    xi_ = sel3(xsel, iz);
                    yi = sel3(yz, iz);
                }
                const R ref = pg == 0 ? refF : refG;
                const R dv = ((bi - ref) + xi_) + yi + zinc;
                if (pg == 0) sf += wgt * dv;
                else sg += wgt * dv;
            }
        }
        fi[i] = sf;
        gi[i] = sg;
    }
}

// full per-axis increment map D[k][j] at offsets eps_j = ds c_j + du
template <typename A>
__device__ __forceinline__ void axis3(A ds, A du, A D[3][3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const A eps[3] = {-ds + du, du, ds + du};
        inc_row3<A>(k, eps, D[k]);
    }
}

// ---------------------------------------------------------------------------
// General stream, for departure points beyond the staged halo (|v| dt >= 1), tiles whose
// velocities spread too far (FAR_SPEED) and non-finite gauges: reads the stencil nodes'
// records from global memory.  On the tensor lattice the union of a node's 27 departure
// stencils (4 x 4 x 4 each) is the product of the per-axis unions: W x H x D nodes, each side
// 4 + the spread of its axis's three departure floors (5 x 5 x 5 while |v| dt < 1).  Each
// region node is carried into the arrival gauge once for all 27 directions and every
// direction adds its Lagrange-weighted share, with the per-(direction, node) arithmetic of
// q27_stream: the region form transforms about 125 nodes per stream against 1,728 pairs.

// Largest region side the region stream takes; wider regions take q27_stream, which earlier
// kernels did faster (us a step of 32 x 32 x 16 nodes at 2.7 T_cr and dt = 1, three quarters of
// the streams per pair, earlier / this: mixed 13,550 / 17,600, FP64 247,000 / 263,000; at 1.6 T_cr,
// none of them, 1,320 / 274 and 45,800 / 8,500).
constexpr int Q27_REGION_MAX = 6;

// A thread's Lagrange weight tables.  Entries 0..17: x, (k * Q27_REGION_MAX + c) = weight
// of region column c in the stencil of x component k (c_x = k - 1), zero outside it;
// entries 18..41: y then z, (18 + (axis - 1) * 12 + k * 4 + j) = cubic weight j of
// component k, placed by the component's offset in the region (kept in registers).
constexpr int Q27_WT_ENTRIES = 3 * Q27_REGION_MAX + 2 * 12;
// Departure floors and cubic weights of the three components of one axis (as in
// `depart`) for the gauge velocity u; the region's first coordinate lo = X + min floor - 1,
// its side, and each component's offset in it.  False, with nothing written, when the side
// exceeds Q27_REGION_MAX or a floor is not finite or not within 2^20 (checked as reals
// before any conversion to int).  PADDED: zero-padded table entries (x), else the four
// weights per component.
template <typename R, bool PADDED>
__device__ __forceinline__ bool q27_region_axis(int X, R s, R u, R dt, R *wt, int &lo, int &side, int (&off)[3])
{
    R fl[3], a[3][4];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const R d = -(s * R(k - 1) + u) * dt;
        fl[k] = floor(d);
        cubic_w<R>(d - fl[k] + R(1), a[k]);
    }
    const R flo = fmin(fmin(fl[0], fl[1]), fl[2]);
    const R fhi = fmax(fmax(fl[0], fl[1]), fl[2]);
    if (!(fhi - flo <= R(Q27_REGION_MAX - 4)) || !(fabs(flo) <= R(1 << 20)) || !(fabs(fhi) <= R(1 << 20)))
        return false;
    lo = X + (int)flo - 1;
    side = (int)(fhi - flo) + 4;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        off[k] = (int)(fl[k] - flo);   // 0 .. side - 4
        if (PADDED) {
#pragma unroll
            for (int c = 0; c < Q27_REGION_MAX; ++c) {
                const int j = c - off[k];
                wt[(k * Q27_REGION_MAX + c)] =
                    j == 0 ? a[k][0] : (j == 1 ? a[k][1] : (j == 2 ? a[k][2] : (j == 3 ? a[k][3] : R(0))));
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) wt[(k * 4 + j)] = a[k][j];
        }
    }
    return true;
}

// weight of region row (plane) c for component k of an unpadded axis table
template <typename R>
__device__ __forceinline__ R q27_wt_at(const R *wt, int k, int o, int c)
{
    const int j = c - o;
    return (j >= 0 && j < 4) ? wt[(k * 4 + j)] : R(0);
}

// One population set (27 values at record offset OFF) of a region node carried by the
// per-axis increment maps: t1 = x-increments, t2 = y-increments of h + t1, z = the
// z-increments of h + t1 + t2, and acc_i += w_i (((h_i - ref_i) + t1_i) + t2_i + z_i) with
// the weight w_i = wx[ix] (wy[iy] wz[iz]) (wyz[3 iz + iy] = wy[iy] wz[iz]).
template <typename R, int OFF>
__device__ __forceinline__ void q27_region_pop(const R (&Dx)[3][3], const R (&Dy)[3][3], const R (&Dz)[3][3],
                                               const R *__restrict__ in, size_t nd, size_t N, const R (&ref)[Q27],
                                               const R (&wx)[3], const R (&wyz)[9], R (&acc)[Q27])
{
    R h[Q27];
    load27<OFF, Q27>(in, nd, N, h);
    R a[Q27], u[Q27];
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        const int ix = i % 3, r = i - ix;
        const R t1 = Dx[ix][0] * h[r] + Dx[ix][1] * h[r + 1] + Dx[ix][2] * h[r + 2];
        a[i] = (h[i] - ref[i]) + t1;
        u[i] = h[i] + t1;
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        const int iy = (i / 3) % 3, r = i - 3 * iy;
        // y-increments from h + t1 (held in u before the update below reads it)
        const R t2 = Dy[iy][0] * u[r] + Dy[iy][1] * u[r + 3] + Dy[iy][2] * u[r + 6];
        h[i] = t2;
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        a[i] += h[i];
        u[i] += h[i];
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        const int iz = i / 9, r = i - 9 * iz;
        const R z = Dz[iz][0] * u[r] + Dz[iz][1] * u[r + 9] + Dz[iz][2] * u[r + 18];
        acc[i] += (wx[i % 3] * wyz[i / 3]) * (a[i] + z);
    }
}

// The region pass for one population set (record offset OFF: R_F or R_G) over the region
// at (xlo, ylo, zlo) of sides W, H, D, skipping region entry `skip` (-1: none): writes the
// increments of the streamed populations over the node's own (node self) into out.
template <typename R, int OFF>
__device__ __noinline__ void q27_region_pass(const DevParams &p, const Grid3 &g3, const R *__restrict__ in,
                                             size_t self, int xlo, int ylo, int zlo, int W, int H, int D,
                                             const int (&oy)[3], const int (&oz)[3], int skip, R th,
                                             const R (&u)[3], const R *wt, R *out)
{
    const R s = sqrt_(th), is = R(1) / s;
    R ref[Q27], acc[Q27];
#pragma unroll
    for (int i = 0; i < Q27; ++i) acc[i] = R(0);
    load27<OFF, Q27>(in, self, (size_t)p.N, ref);
    const R *wty = wt + 3 * Q27_REGION_MAX, *wtz = wty + 12;
    int e = 0;   // region entry index (z-major, then y, then x)
#pragma unroll 1
    for (int cz = 0; cz < D; ++cz) {
        const int zz = bc_wrap(zlo + cz, g3.nz, g3.bcz);
        R wz[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) wz[k] = q27_wt_at(wtz, k, oz[k], cz);
#pragma unroll 1
        for (int cy = 0; cy < H; ++cy) {
            const long long row = ((long long)zz * p.ny + bc_wrap(ylo + cy, p.ny, p.bcy)) * p.nx;
            R wyz[9];   // wy[m] wz[l] at 3 l + m (population i = 9 l + 3 m + k)
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const R wy = q27_wt_at(wty, m, oy[m], cy);
#pragma unroll
                for (int l = 0; l < 3; ++l) wyz[3 * l + m] = wy * wz[l];
            }
#pragma unroll 1
            for (int cx = 0; cx < W; ++cx, ++e) {
                if (e == skip) continue;
                const size_t nd = (size_t)(row + bc_wrap(xlo + cx, p.nx, p.bcx));
                R gv[4];
                load27<R_TH, 4>(in, nd, (size_t)p.N, gv);   // theta, u_x, u_y, u_z of the region node
                const R ds = (gv[0] - th) / (sqrt_(gv[0]) + s) * is;   // (s' - s)/s
                R Dx[3][3], Dy[3][3], Dz[3][3];
                axis3<R>(ds, (gv[1] - u[0]) * is, Dx);
                axis3<R>(ds, (gv[2] - u[1]) * is, Dy);
                axis3<R>(ds, (gv[3] - u[2]) * is, Dz);
                R wx[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) wx[k] = wt[(k * Q27_REGION_MAX + cx)];
                q27_region_pop<R, OFF>(Dx, Dy, Dz, in, nd, (size_t)p.N, ref, wx, wyz, acc);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i) out[i] = acc[i];
}

// Streaming of node (X, Y, Z) into gauge (th, u) by the region stream where the region
// fits, else by q27_stream; skip_own leaves out the node's own region entry (valid when
// the gauge is the node's stored gauge: the map is then the identity and the entry adds
// exactly zero).  Adds the region entries transformed to nreg, or 1 to npair.
template <typename R>
__device__ __noinline__ void q27_stream_any(const DevParams &p, const Grid3 &g3, const R *__restrict__ in, int X,
                                            int Y, int Z, R th, const R (&u)[3], bool skip_own, R *fi, R *gi,
                                            unsigned &nreg, unsigned &npair)
{
    R wt[Q27_WT_ENTRIES];
    const R s = sqrt_(th), dt = (R)p.dt;
    int xlo, ylo, zlo, W, H, D, ox[3], oy[3], oz[3];
    R *wty = wt + 3 * Q27_REGION_MAX, *wtz = wty + 12;
    if (q27_region_axis<R, true>(X, s, u[0], dt, wt, xlo, W, ox) &&
        q27_region_axis<R, false>(Y, s, u[1], dt, wty, ylo, H, oy) &&
        q27_region_axis<R, false>(Z, s, u[2], dt, wtz, zlo, D, oz)) {
        const int cxo = X - xlo, cyo = Y - ylo, czo = Z - zlo;
        const int skip = (skip_own && cxo >= 0 && cxo < W && cyo >= 0 && cyo < H && czo >= 0 && czo < D)
                             ? (czo * H + cyo) * W + cxo : -1;
        const size_t self = (size_t)(((long long)Z * p.ny + Y) * p.nx + X);
        q27_region_pass<R, R_F>(p, g3, in, self, xlo, ylo, zlo, W, H, D, oy, oz, skip, th, u, wt, fi);
        q27_region_pass<R, R_G>(p, g3, in, self, xlo, ylo, zlo, W, H, D, oy, oz, skip, th, u, wt, gi);
        nreg += (unsigned)(W * H * D - (skip >= 0 ? 1 : 0));
    } else {
        q27_stream<R>(p, g3, in, X, Y, Z, th, u, fi, gi);
        npair += 1;
    }
}

// ---------------------------------------------------------------------------
// Sums of 27 values v and their first moments: out = sum v, sum v c_x, sum v c_y, sum v c_z
// (the last three with MOM).  Lines, planes, then the column; FP32 values in float-float
// (exact up to ~2^-48).
template <bool MOM>
__device__ __forceinline__ void sums27(const float *v, ffv *out)
{
    ffv S = {0.f, 0.f}, D = S, Y = S, S0 = S, S2 = S;
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        ffv pS = {0.f, 0.f}, pD = pS, l0 = pS, l2 = pS;
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const float *r = v + 9 * z + 3 * y;
            const ffv line = ff_add(ff_pair(r[0], r[1]), r[2]);
            pS = y == 0 ? line : ff_add(pS, line);
            if (MOM) {
                const ffv d = ff_pair(r[2], -r[0]);
                pD = y == 0 ? d : ff_add(pD, d);
                if (y == 0) l0 = line;
                if (y == 2) l2 = line;
            }
        }
        S = z == 0 ? pS : ff_add(S, pS);
        if (MOM) {
            const ffv dy = ff_add(l2, ff_neg(l0));
            D = z == 0 ? pD : ff_add(D, pD);
            Y = z == 0 ? dy : ff_add(Y, dy);
            if (z == 0) S0 = pS;
            if (z == 2) S2 = pS;
        }
    }
    out[0] = S;
    if (MOM) {
        out[1] = D;
        out[2] = Y;
        out[3] = ff_add(S2, ff_neg(S0));
    }
}
template <bool MOM>
__device__ __forceinline__ void sums27(const double *v, double *out)
{
    double S = 0, D = 0, Y = 0, S0 = 0, S2 = 0;
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        double pS = 0, l0 = 0, l2 = 0;
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const double *r = v + 9 * z + 3 * y;
            const double line = (r[0] + r[1]) + r[2];
            pS += line;
            if (MOM) {
                D += r[2] - r[0];
                if (y == 0) l0 = line;
                if (y == 2) l2 = line;
            }
        }
        S += pS;
        if (MOM) {
            Y += l2 - l0;
            if (z == 0) S0 = pS;
            if (z == 2) S2 = pS;
        }
    }
    out[0] = S;
    if (MOM) {
        out[1] = D;
        out[2] = Y;
        out[3] = S2 - S0;
    }
}

// increment of (I + Dz)(I + Dy)(I + Dx) applied to h (27 values)
template <typename A>
__device__ __forceinline__ void apply3_inc(const A (&Dx)[3][3], const A (&Dy)[3][3], const A (&Dz)[3][3], const A *h,
                                           A *out)
{
    A t1[27], t2[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const int ix = i % 3, r = i - ix;
        t1[i] = Dx[ix][0] * h[r] + Dx[ix][1] * h[r + 1] + Dx[ix][2] * h[r + 2];
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const int iy = (i / 3) % 3, r = i - 3 * iy;
        t2[i] = Dy[iy][0] * (h[r] + t1[r]) + Dy[iy][1] * (h[r + 3] + t1[r + 3]) + Dy[iy][2] * (h[r + 6] + t1[r + 6]);
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const int iz = i / 9, r = i - 9 * iz;
        const A z = Dz[iz][0] * (h[r] + t1[r] + t2[r]) + Dz[iz][1] * (h[r + 9] + t1[r + 9] + t2[r + 9]) +
                    Dz[iz][2] * (h[r + 18] + t1[r + 18] + t2[r + 18]);
        out[i] = t1[i] + t2[i] + z;
    }
}

// ---------------------------------------------------------------------------
// Staging.  The tile of a block and its staged slots.
constexpr int Q27_THREADS = STEP_THREADS, T27X = 8, T27Y = 4, T27Z = 4, HALO27 = 2;
constexpr int S27X = T27X + 2 * HALO27, S27Y = T27Y + 2 * HALO27, S27Z = T27Z + 2 * HALO27;
constexpr int SLOTS27 = S27X * S27Y * S27Z;
constexpr int PY27 = S27X, PZ27 = S27X * S27Y + 8;   // slots per row, per plane (padded: the two planes
                                                     // a half warp reads start 16 banks apart)
constexpr int SLOT_SPACE27 = PZ27 * S27Z;
__host__ __device__ constexpr int slot27(int k) { return k + 8 * (k / (S27X * S27Y)); }   // place of staged node k
// Values per slot.  FP32: ten words for each source plane p: the pairs (n = 0, 1) of m = 0,
// 1, 2, then the three values of n = 2, then a pad (8-byte loads; sixteen consecutive slots
// fall on distinct pairs of banks).  FP64: 27 values.
template <typename R> struct Slot27;
template <> struct Slot27<float> { static constexpr int stride = 30; };
template <> struct Slot27<double> { static constexpr int stride = 27; };
// What a thread keeps in shared memory across the FP32 stream: y weights and rows.
enum : int { K27_WY = 0, K27_LY = 15, K27_N = 24 };
template <typename R>
constexpr size_t q27_smem_bytes()
{
    return (size_t)SLOT_SPACE27 * Slot27<R>::stride * sizeof(R) + (sizeof(R) == 4 ? (size_t)K27_N * Q27_THREADS * sizeof(R) : 0);
}

struct Tile27 { int X0, Y0, Z0; };
__device__ __forceinline__ size_t slot_node27(const DevParams &p, const Grid3 &g3, const Tile27 &t, int k)
{
    const int x = k % S27X, y = (k / S27X) % S27Y, z = k / (S27X * S27Y);
    return (size_t)node27(p, g3, t.X0 - HALO27 + x, t.Y0 - HALO27 + y, t.Z0 - HALO27 + z);
}

// The map of one axis applied to 27 values along it (stride 1, 3 or 9).
template <int ST, typename A>
__device__ __forceinline__ void apply_axis27(const A (&G)[3][3], A (&h)[27])
{
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int i = ST == 1 ? 3 * q : (ST == 3 ? (q / 3) * 9 + q % 3 : q);
        const A a = h[i], b = h[i + ST], c = h[i + 2 * ST];
#pragma unroll
        for (int k = 0; k < 3; ++k) h[i + k * ST] = G[k][0] * a + G[k][1] * b + G[k][2] * c;
    }
}

// Stages one family (record offset OFF): its populations carried into the tile's gauge gb
// = (sqrt theta, u), theta = thb; inc (FP32): less those of node `nbase`, whose gauge gb
// then is, in increment form (see the head of pond_step.cuh).
template <int OFF, typename R>
__device__ __forceinline__ void stage27(const DevParams &p, const Grid3 &g3, const R *__restrict__ in,
                                        const Tile27 &t, size_t nbase, const R (&gb)[4], R thb, bool inc, R *slots)
{
    constexpr int DS = Slot27<R>::stride;
    const size_t N = (size_t)p.N;
    const R inv_sb = R(1) / gb[0];
#pragma unroll 1
    for (int k = threadIdx.x; k < SLOTS27; k += Q27_THREADS) {
        const size_t nd = slot_node27(p, g3, t, k);
        R gv[4], h[27];
        load27<R_TH, 4>(in, nd, N, gv);
        load27<OFF, 27>(in, nd, N, h);
        const R e = fdiv_(gv[0] - thb, (sqrt_(gv[0]) + gb[0]) * gb[0]);
        const R w[3] = {(gv[1] - gb[1]) * inv_sb, (gv[2] - gb[2]) * inv_sb, (gv[3] - gb[3]) * inv_sb};
        R D[3][3][3];
        if (sizeof(R) == 4 && inc) {
            R o[27], base[27];
#pragma unroll
            for (int a = 0; a < 3; ++a) axis_map<R>(e, w[a], D[a]);
            apply3_inc<R>(D[0], D[1], D[2], h, o);
            load27<OFF, 27>(in, nbase, N, base);
#pragma unroll
            for (int i = 0; i < 27; ++i) h[i] = (h[i] - base[i]) + o[i];
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) axis_rows<R>(e, w[a], D[a]);
            apply_axis27<1>(D[0], h);
            apply_axis27<3>(D[1], h);
            apply_axis27<9>(D[2], h);
        }
        R *dst = slots + (size_t)slot27(k) * DS;
        if constexpr (sizeof(R) == 4) {
            f32x2 *d2 = reinterpret_cast<f32x2 *>(dst);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const R *hp = h + 9 * q;
#pragma unroll
                for (int m = 0; m < 3; ++m) d2[5 * q + m] = pack2(hp[m], hp[3 + m]);
                d2[5 * q + 3] = pack2(hp[6], hp[7]);
                d2[5 * q + 4] = pack2(hp[8], 0.0f);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 27; ++i) dst[i] = h[i];
        }
    }
}

// The stream of one family as a contraction over the staged window of the slot `own` (see
// the head of pond_step.cuh): a, near0 = each axis's Lagrange weights and departure floors,
// L = the rows of the map from the tile's gauge.  FP32: five columns, rows and planes with
// zero weights outside a component's four nodes, and differences to the node's own slot
// (see the head of pond_step.cuh).
// One source plane p at a time, so that the accumulators and a row's five slots fit the
// registers and the loads of a row go out together; n = 0 and 1 share packed instructions.
__device__ __forceinline__ void contract27(const float *own, const float (&a)[3][3][4], const bool (&near0)[3][3],
                                           const float (&L)[3][3][3], float *keep, float (&acc)[27])
{
    constexpr int DS = Slot27<float>::stride;
    f32x2 wl[3][5][3];
    float wz[3][5];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const int lo = c > 3 ? 3 : c, hi = c < 1 ? 0 : c - 1;
            const float w = near0[0][k] ? (c == 0 ? 0.0f : a[0][k][hi]) : (c == 4 ? 0.0f : a[0][k][lo]);
            keep[(K27_WY + 5 * k + c) * Q27_THREADS] = near0[1][k] ? (c == 0 ? 0.0f : a[1][k][hi]) : (c == 4 ? 0.0f : a[1][k][lo]);
            wz[k][c] = near0[2][k] ? (c == 0 ? 0.0f : a[2][k][hi]) : (c == 4 ? 0.0f : a[2][k][lo]);
#pragma unroll
            for (int m = 0; m < 3; ++m) wl[k][c][m] = pack2(w * L[0][k][m], w * L[0][k][m]);
        }
#pragma unroll
    for (int i = 0; i < 9; ++i) keep[(K27_LY + i) * Q27_THREADS] = L[1][i / 3][i % 3];
#pragma unroll
    for (int i = 0; i < 27; ++i) acc[i] = 0.0f;
    const float *plane = own - (2 * PZ27 + 2 * PY27 + 2) * DS;
#pragma unroll 1
    for (int cz = 0; cz < 5; ++cz, plane += PZ27 * DS) {
#pragma unroll 1
        for (int q = 0; q < 3; ++q) {
            const f32x2 *op = reinterpret_cast<const f32x2 *>(own) + 5 * q;
            f32x2 dp[3], b2[9];   // b: 3 l + k, the shares of n = 0, 1 apart
            float ds[3], b1[9];   // n = 2
            {
                float x, y;
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    unpack2(op[m], x, y);
                    dp[m] = pack2(-x, -y);
                }
                unpack2(op[3], ds[0], ds[1]);
                unpack2(op[4], ds[2], y);
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) { b2[i] = 0ull; b1[i] = 0.0f; }
            const f32x2 *row = reinterpret_cast<const f32x2 *>(plane) + 5 * q;
            f32x2 v[5][5];   // the row's slots; each is replaced by the next row's once it is used
#pragma unroll
            for (int cx = 0; cx < 5; ++cx)
#pragma unroll
                for (int e = 0; e < 5; ++e) v[cx][e] = row[cx * (DS / 2) + e];
#pragma unroll 1
            for (int cy = 0; cy < 5; ++cy) {
                f32x2 tp[3] = {0ull, 0ull, 0ull};
                float ts[3] = {0.0f, 0.0f, 0.0f};
                if (cy < 4) row += PY27 * (DS / 2);   // (the last row loads itself again)
#pragma unroll
                for (int cx = 0; cx < 5; ++cx) {
                    float x[3], pad;
                    unpack2(v[cx][3], x[0], x[1]);
                    unpack2(v[cx][4], x[2], pad);
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        const f32x2 vp = add2(v[cx][m], dp[m]);
                        const float vs = x[m] - ds[m];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            float w, w_;
                            unpack2(wl[k][cx][m], w, w_);
                            tp[k] = fma2(wl[k][cx][m], vp, tp[k]);
                            ts[k] = fmaf(w, vs, ts[k]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 5; ++e) v[cx][e] = row[cx * (DS / 2) + e];
                }
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    const float w = keep[(K27_WY + 5 * l + cy) * Q27_THREADS];
                    const f32x2 wp = pack2(w * keep[(K27_LY + 3 * l) * Q27_THREADS], w * keep[(K27_LY + 3 * l + 1) * Q27_THREADS]);
                    const float ws = w * keep[(K27_LY + 3 * l + 2) * Q27_THREADS];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        b2[3 * l + k] = fma2(wp, tp[k], b2[3 * l + k]);
                        b1[3 * l + k] = fmaf(ws, ts[k], b1[3 * l + k]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                float x, y;
                unpack2(b2[i], x, y);
                b1[i] += x + y;
            }
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float w = wz[r][0] * sel3(q, L[2][r][0], L[2][r][1], L[2][r][2]);
#pragma unroll
                for (int i = 0; i < 9; ++i) acc[9 * r + i] = fmaf(w, b1[i], acc[9 * r + i]);
            }
        }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) wz[r][c] = wz[r][c + 1];   // the next plane's weight moves to the front
    }
}
// FP64: each component's own four columns; acc = streamed populations.
__device__ __forceinline__ void contract27(const double *own, const double (&a)[3][3][4], const bool (&near0)[3][3],
                                           const double (&L)[3][3][3], double *, double (&acc)[27])
{
    constexpr int DS = Slot27<double>::stride;
    double wl[3][4][3], wy[3][5], wz[3][5];
    int off[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        off[k] = near0[0][k] ? DS : 0;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int m = 0; m < 3; ++m) wl[k][c][m] = a[0][k][c] * L[0][k][m];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const int lo = c > 3 ? 3 : c, hi = c < 1 ? 0 : c - 1;
            wy[k][c] = near0[1][k] ? (c == 0 ? 0.0 : a[1][k][hi]) : (c == 4 ? 0.0 : a[1][k][lo]);
            wz[k][c] = near0[2][k] ? (c == 0 ? 0.0 : a[2][k][hi]) : (c == 4 ? 0.0 : a[2][k][lo]);
        }
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) acc[i] = 0.0;
    const double *plane = own - (2 * PZ27 + 2 * PY27 + 2) * DS;
#pragma unroll 1
    for (int cz = 0; cz < 5; ++cz, plane += PZ27 * DS) {
        double b[3][9];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int i = 0; i < 9; ++i) b[q][i] = 0.0;
        const double *row = plane;
#pragma unroll 1
        for (int cy = 0; cy < 5; ++cy, row += PY27 * DS) {
            double wn[3][3];
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                const double w = wy[l][0];
#pragma unroll
                for (int c = 0; c < 4; ++c) wy[l][c] = wy[l][c + 1];
                wy[l][4] = w;
#pragma unroll
                for (int n = 0; n < 3; ++n) wn[l][n] = w * L[1][l][n];
            }
#pragma unroll
            for (int q = 0; q < 9; ++q)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double *r = row + off[k] + 3 * q;
                    double t = 0.0;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int m = 0; m < 3; ++m) t = fma(wl[k][c][m], r[c * DS + m], t);
#pragma unroll
                    for (int l = 0; l < 3; ++l) b[q / 3][3 * l + k] = fma(wn[l][q % 3], t, b[q / 3][3 * l + k]);
                }
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const double w = wz[r][0];
#pragma unroll
            for (int c = 0; c < 4; ++c) wz[r][c] = wz[r][c + 1];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const double wn2 = w * L[2][r][q];
#pragma unroll
                for (int i = 0; i < 9; ++i) acc[9 * r + i] = fma(wn2, b[q][i], acc[9 * r + i]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Collision of one node in type R, equilibria as increments over their co-moving form
// (ft, gt = streamed populations, mc = the last corrector's fields, th, u = the streaming
// gauge); writes the record.  Returns whether the results are finite.
template <typename R>
__device__ __forceinline__ bool q27_collide(const DevParams &p, R *__restrict__ out, size_t n, R th, const R (&u)[3],
                                            const Macro<3, R> &mc, const typename Wide<R>::type (&F)[3],
                                            typename Wide<R>::type M0, R (&ft)[27], R (&gt)[27])
{
    using A = typename Wide<R>::type;
    const size_t N = (size_t)p.N;
    const TypedParams<R> &q = typed<R>(p);
    const R rho = w_round(mc.rho), E = w_round(mc.E), Pg = w_round(mc.P);
    const R uu[3] = {w_round(mc.uu[0]), w_round(mc.uu[1]), w_round(mc.uu[2])};
    const R uh[3] = {w_round(mc.uh[0]), w_round(mc.uh[1]), w_round(mc.uh[2])};
    const R f3[3] = {w_round(F[0]), w_round(F[1]), w_round(F[2])}, m0 = w_round(M0), dt = q.dt, om = q.omega;
    const A sA = w_sqrt(th);
    const R s = w_round(sA), is = R(1) / s, sst = sqrt_(w_round(mc.ths));
    const R ds = fdiv_(mc.dth, (sst + s) * s);             // (s* - s)/s
    const R irho = R(1) / rho, ihP = R(1) / (R(2) * Pg);   // 1/rho, 1/(2P)
    R D[3][3][3], h[Q27], inc[Q27], fo[Q27];
    {
        R Es[3][3][3], shi[Q27];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R du = w_round(mc.du[a]) * is;
            axis3<R>(ds, du, D[a]);
            axis3<R>(ds, du + f3[a] * dt * irho * is, Es[a]);
        }
#pragma unroll
        for (int i = 0; i < Q27; ++i) h[i] = rho * (R)w27(i);
        apply3_inc<R>(D[0], D[1], D[2], h, inc);
        apply3_inc<R>(Es[0], Es[1], Es[2], h, shi);
#pragma unroll
        for (int i = 0; i < Q27; ++i) fo[i] = ft[i] + om * ((h[i] - ft[i]) + inc[i]) + (shi[i] - inc[i]);
    }
    bool finite = inc[0] - inc[0] == R(0);
    A sm[4];
    sums27<true>(fo, sm);
    // mass and momentum defects (sum f = rho, sum f (v - u) = rho (u* - u) + F dt exactly),
    // spread by W_i and W_i c_i / (s T_L)
    const R mdef = w_round(w_sub(mc.rho, sm[0]));
    A jex[3];
    R jd[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        jex[a] = w_add(w_mul(mc.rho, mc.du[a]), w_mul(F[a], wide_dt<A>(p)));
        jd[a] = w_round(w_sub(jex[a], w_mul(sA, sm[1 + a]))) * (is * R(3));
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i)
        fo[i] += (R)w27(i) * (mdef + jd[0] * R(i % 3 - 1) + jd[1] * R((i / 3) % 3 - 1) + jd[2] * R(i / 9 - 1));
    R mlo = R(0), jlo[3] = {R(0), R(0), R(0)};
    if constexpr (sizeof(R) == 4) {
        sums27<true>(fo, sm);
        mlo = w_round(w_sub(mc.rho, sm[0]));
#pragma unroll
        for (int a = 0; a < 3; ++a) jlo[a] = w_round(w_sub(jex[a], w_mul(sA, sm[1 + a])));
    }

    const R Prh = Pg * irho, H = E + Prh;
    const R k2 = dt * rho * ihP;   // dt rho / (2P)
    R I[3][3], Mv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) I[a][b] = uh[a] * f3[b] + f3[a] * uh[b] + dt * f3[a] * f3[b] * E * ihP;
#pragma unroll
    for (int a = 0; a < 3; ++a) Mv[a] = (R(2) * k2) * (f3[a] * H - (I[a][0] * uu[0] + I[a][1] * uu[1] + I[a][2] * uu[2]));
    const R work = uh[0] * f3[0] + uh[1] * f3[1] + uh[2] * f3[2];
    const R rhP = rho * ihP;
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        const R c[3] = {R(i % 3 - 1), R((i / 3) % 3 - 1), R(i / 9 - 1)};
        R v[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = sst * c[a] + uu[a];
        R g = R(2) * rho * E;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            g += Mv[a] * (v[a] - uu[a]);
#pragma unroll
            for (int b = 0; b < 3; ++b)
                g += ((a == b ? rho : R(0)) + k2 * I[a][b]) * (v[a] * v[b] - (a == b ? Prh : R(0)) - uu[a] * uu[b]);
        }
        const R W = (R)w27(i);
        const R uc = uu[0] * c[0] + uu[1] * c[1] + uu[2] * c[2];
        const R v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        const R gc = m0 * W * (R(1) + rhP * uc * uc * R(3) - rhP * v2 + R(1.5));
        h[i] = om * W * g + dt * (gc + R(2) * W * work);
    }
    apply3_inc<R>(D[0], D[1], D[2], h, inc);
    finite = finite && inc[0] - inc[0] == R(0);
#pragma unroll
    for (int i = 0; i < Q27; ++i) gt[i] = gt[i] - om * gt[i] + (h[i] + inc[i]);
    // energy: sum g_out = sum g~ + dt (M_0 + 2 uhat . F) exactly; the same defect spreading
    A wk = w_mul(mc.uh[0], F[0]);
    wk = w_add(w_add(wk, w_mul(mc.uh[1], F[1])), w_mul(mc.uh[2], F[2]));
    const A g_tot = w_add(mc.gs, w_mul(w_add(M0, w_mul(wk, R(2))), wide_dt<A>(p)));
    sums27<false>(gt, sm);
    const R gdef = w_round(w_sub(g_tot, sm[0]));
#pragma unroll
    for (int i = 0; i < Q27; ++i) gt[i] += gdef * (R)w27(i);
    R glo = R(0);
    if constexpr (sizeof(R) == 4) {
        sums27<false>(gt, sm);
        glo = w_round(w_sub(g_tot, sm[0]));
    }
    R rec[SL27];
    rec[R_TH] = th;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        rec[R_UX + a] = u[a];
        rec[R_UHX + a] = uh[a];
        rec[R_JLO + a] = jlo[a];
    }
#pragma unroll
    for (int i = 0; i < Q27; ++i) {
        rec[R_F + i] = fo[i];
        rec[R_G + i] = gt[i];
    }
    rec[R_RHO] = rho;
    const R T = w_round(mc.T);
    rec[R_T] = T;
    rec[R_MLO] = mlo;
    rec[R_GLO] = glo;
    store_chunks<SL27>(out, n, N, rec);
    return finite && rho - rho == R(0) && T - T == R(0);
}

// The node step, one thread per node of the block's tile; bx, by: blocks along x and y (in
// one launch dimension, since the others hold 65,535 blocks only).  Two resident blocks per SM
// in FP32 (255 registers; the shared memory of one staged family each), one in FP64.
template <typename R>
__global__ void __launch_bounds__(Q27_THREADS, sizeof(R) == 4 ? 2 : 1)
    k_q27_step(DevParams p, Grid3 g3, int bx, int by, const R *__restrict__ in, typename Wide<R>::type *nl,
               R *__restrict__ out, DevStats *stats)
{
    using A = typename Wide<R>::type;
    extern __shared__ __align__(128) unsigned char q27_dyn_smem[];
    R *slots = reinterpret_cast<R *>(q27_dyn_smem);
    R *keep = slots + (size_t)SLOT_SPACE27 * Slot27<R>::stride + threadIdx.x;   // this thread's column (FP32)
    __shared__ StepCounts counts;
    __shared__ uint4 best[BEST];
    const int tid = threadIdx.x;
    const size_t N = (size_t)p.N;
    const int b = (int)blockIdx.x;
    const Tile27 tl{b % bx * T27X, b / bx % by * T27Y, b / bx / by * T27Z};
    // a warp takes 8 x 1 x 4 nodes: the half warps' slots then fall on distinct banks
    const int tx = tid % T27X, tz = (tid / T27X) % T27Z, ty = tid / (T27X * T27Z);
    const int X = tl.X0 + tx, Y = tl.Y0 + ty, Z = tl.Z0 + tz;
    const bool valid = X < p.nx && Y < p.ny && Z < g3.nz;
    const size_t n = valid ? ((size_t)Z * p.ny + Y) * p.nx + X : 0;
    if (tid == 0) counts = StepCounts{};

    // the tile's common gauge
    Extremes<3> ex;
    for (int k = tid; k < SLOTS27; k += Q27_THREADS) {
        R gv[4];
        load27<R_TH, 4>(in, slot_node27(p, g3, tl, k), N, gv);
        ex.offer(gv[0], gv + 1, k);
    }
    ex = tile_extremes(ex, best);
    bool inc = sizeof(R) == 4 && ex.smooth();
    const size_t nbase = slot_node27(p, g3, tl, min((int)ex.at, SLOTS27 - 1));
    R gb[4], thb;
    {
        R hot[4], cold[4];
        load27<R_TH, 4>(in, nbase, N, hot);
        load27<R_TH, 4>(in, slot_node27(p, g3, tl, min((int)ex.lat, SLOTS27 - 1)), N, cold);
        common_gauge<R, 4>(inc, hot, cold, gb);
        thb = inc ? hot[0] : gb[0] * gb[0];
    }
    R dt_b = typed<R>(p).dt;   // infinite in a tile whose velocities spread too far (no contraction)
    if (__syncthreads_or(ex.spread(gb, sqrtf(ex.hottest())))) {
        inc = false;
        if (!middle_gauge<R, 3>(ex, best, gb)) dt_b = R(1) / R(0);
        thb = gb[0] * gb[0];
    }

    R th = R(1), u[3] = {R(0), R(0), R(0)};
    if (valid) {
        R gv[4], v[27];
        load27<R_TH, 4>(in, n, N, gv);
        th = gv[0]; u[0] = gv[1]; u[1] = gv[2]; u[2] = gv[3];
        // sums of the node's own stored populations and kept remainders {f, f c, g, momentum
        // lo}: they wait in the stress and flux planes, which the divergences are done with
        A own[5];
        R lo[5];
        load27<R_F, 27>(in, n, N, v);
        sums27<true>(v, own);
        load27<R_G, 27>(in, n, N, v);
        sums27<false>(v, own + 4);
        load27<R_MLO, 5>(in, n, N, lo);
        own[0] = w_add(own[0], lo[0]);
        own[4] = w_add(own[4], lo[4]);
#pragma unroll
        for (int k = 0; k < 5; ++k) NL3(nl, N3_K + k, n, N) = own[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) NL3(nl, N3_K + 5 + a, n, N) = w_wide(lo[1 + a]);
    }

    unsigned its = 0, nreg = 0, npair = 0;
    bool active = valid, conv = true, floored = false, bad = false;
    R fi[27], gi[27];   // increments of the streamed populations
    Macro<3, R> m;
    int staged = -1;    // family in the slots
    const R *own_slot = slots + (size_t)((tz + HALO27) * PZ27 + (ty + HALO27) * PY27 + tx + HALO27) * Slot27<R>::stride;
    for (unsigned it = 1; __syncthreads_or(active); ++it) {
        const R s = sqrt_(th), inv_s = R(1) / s;
        R a[3][3][4], L[3][3][3];
        bool near0[3][3], fast = true;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const bool ok = axis_weights<R>(s, u[x], dt_b, a[x], near0[x]);
            fast = fast && ok;
            axis_rows<R>((gb[0] - s) * inv_s, (gb[1 + x] - u[x]) * inv_s, L[x]);
        }
        if (active) {
            its = it;
            if (fast) {
                int side = 1;
#pragma unroll
                for (int x = 0; x < 3; ++x)
                    side *= (near0[x][0] == near0[x][1] && near0[x][1] == near0[x][2]) ? 4 : 5;
                nreg += (unsigned)(side - (it == 1 ? 1 : 0));
            } else {
                R f2[27], g2[27];
                q27_stream_any<R>(p, g3, in, X, Y, Z, th, u, it == 1, f2, g2, nreg, npair);
#pragma unroll
                for (int i = 0; i < 27; ++i) { fi[i] = f2[i]; gi[i] = g2[i]; }
            }
        }
        // odd streams take f then g, even ones g then f: the second family of one is the
        // first of the next and stays in the slots
#pragma unroll 1
        for (int ps = 0; ps < 2; ++ps) {
            const int fam = (it & 1) ? ps : 1 - ps;
            if (staged != fam) {
                __syncthreads();
                if (fam == 0) stage27<R_F>(p, g3, in, tl, nbase, gb, thb, inc, slots);
                else stage27<R_G>(p, g3, in, tl, nbase, gb, thb, inc, slots);
                __syncthreads();
                staged = fam;
            }
            if (!active || !fast) continue;
            R acc[27];
            contract27(own_slot, a, near0, L, keep, acc);
            if (sizeof(R) == 8 || it > 1) {
                R v[27];
                if (fam == 0) load27<R_F, 27>(in, n, N, v);
                else load27<R_G, 27>(in, n, N, v);
                if constexpr (sizeof(R) == 8) {
#pragma unroll
                    for (int i = 0; i < 27; ++i) acc[i] -= v[i];
                } else {
                    // the node's own populations carried from their stored gauge into this one
                    R gv[4], Dx[3][3], Dy[3][3], Dz[3][3], o[27];
                    load27<R_TH, 4>(in, n, N, gv);
                    const R e = fdiv_(gv[0] - th, (sqrt_(gv[0]) + s) * s);
                    axis_map<R>(e, (gv[1] - u[0]) * inv_s, Dx);
                    axis_map<R>(e, (gv[2] - u[1]) * inv_s, Dy);
                    axis_map<R>(e, (gv[3] - u[2]) * inv_s, Dz);
                    apply3_inc<R>(Dx, Dy, Dz, v, o);
#pragma unroll
                    for (int i = 0; i < 27; ++i) acc[i] += o[i];
                }
            }
            if (fam == 0) {
#pragma unroll
                for (int i = 0; i < 27; ++i) fi[i] = acc[i];
            } else {
#pragma unroll
                for (int i = 0; i < 27; ++i) gi[i] = acc[i];
            }
        }
        if (active) {
            A d[5], own[8], F[3];
            sums27<true>(fi, d);
            sums27<false>(gi, d + 4);
#pragma unroll
            for (int k = 0; k < 8; ++k) own[k] = NL3(nl, N3_K + k, n, N);
#pragma unroll
            for (int k = 0; k < 3; ++k) F[k] = NL3(nl, N3_F + k, n, N);
            m.update(p, th, u, own, d, F, NL3(nl, N3_REL, n, N), 3.0);
            const float res = m.change(th);
            conv = sizeof(R) == 4 ? res <= p.tol_f : (double)res <= p.tol;
            if (conv || it >= (unsigned)p.max_iter || !(res == res)) {
                active = false;
            } else {
                th = w_round(m.ths);
#pragma unroll
                for (int x = 0; x < 3; ++x) u[x] = w_round(m.uu[x]);
            }
        }
    }
    if (valid) {
        R v[27];
        load27<R_F, 27>(in, n, N, v);
#pragma unroll
        for (int i = 0; i < 27; ++i) fi[i] += v[i];
        load27<R_G, 27>(in, n, N, v);
#pragma unroll
        for (int i = 0; i < 27; ++i) gi[i] += v[i];
        const A F[3] = {NL3(nl, N3_F, n, N), NL3(nl, N3_F + 1, n, N), NL3(nl, N3_F + 2, n, N)};
        bad = !q27_collide<R>(p, out, n, th, u, m, F, NL3(nl, N3_M0, n, N), fi, gi);
        floored = w_double(m.pr) < p.p_floor;
    }
    add_counts(counts, stats, its, nreg, npair, valid && !conv, false, floored, bad);
}

// Output fields: rho, uhat (3), T, p in FP64.
template <typename R>
__global__ void k_q27_moments(DevParams p, const R *__restrict__ st, double *rho, double *ux, double *uy,
                              double *uz, double *T, double *pr)
{
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const double r = (double)REC27(st, n, R_RHO), t = (double)REC27(st, n, R_T);
    if (rho) rho[n] = r;
    if (ux) ux[n] = (double)REC27(st, n, R_UHX);
    if (uy) uy[n] = (double)REC27(st, n, R_UHX + 1);
    if (uz) uz[n] = (double)REC27(st, n, R_UHX + 2);
    if (T) T[n] = t;
    if (pr) pr[n] = pressure_d(p, r, t);
}

// Conservation sums, stage 1: {rho, rho uhat_x, rho uhat_y, sum g / 2} per block.
template <typename R>
__global__ void k_q27_conserve1(DevParams p, const R *__restrict__ st, double *part)
{
    const long long N = p.N;
    double s[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0};
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        const double r = (double)REC27(st, n, R_RHO);
        double eg = (double)REC27(st, n, R_GLO);
        for (int i = 0; i < Q27; ++i) eg += (double)REC27(st, n, R_G + i);
        const double v[4] = {r, r * (double)REC27(st, n, R_UHX), r * (double)REC27(st, n, R_UHX + 1), 0.5 * eg};
        for (int k = 0; k < 4; ++k) pair_add(s[k], c[k], v[k], 0.0);
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int k = 0; k < 4; ++k) {
            const double s2 = __shfl_xor_sync(0xffffffffu, s[k], o);
            const double c2 = __shfl_xor_sync(0xffffffffu, c[k], o);
            pair_add(s[k], c[k], s2, c2);
        }
    __shared__ double sh[32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int k = 0; k < 4; ++k) { sh[warp][2 * k] = s[k]; sh[warp][2 * k + 1] = c[k]; }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int k = 0; k < 4; ++k) {
            double ss = sh[0][2 * k], cc = sh[0][2 * k + 1];
            for (int w = 1; w < nw; ++w) pair_add(ss, cc, sh[w][2 * k], sh[w][2 * k + 1]);
            part[blockIdx.x * 8 + 2 * k] = ss;
            part[blockIdx.x * 8 + 2 * k + 1] = cc;
        }
    }
}

}  // namespace pond

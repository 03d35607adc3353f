// pond_q16.cuh -- the PonD van der Waals time step on the D2Q16 lattice for sm_103a.
//
// The model holds for any tensor lattice C1 x C1 with weights W_i = W_jx W_jy and lattice
// temperature T_L = sum W c^2 (SM "Equilibrium").  D2Q16 takes for C1 the four roots
// -+sqrt(3 +- sqrt 6) of the Hermite polynomial He_4(c) = c^4 - 6 c^2 + 3 with the
// Gauss-Hermite weights (3 -+ sqrt 6)/12, so that T_L = 1.  The transfer map
// G = M_lambda'^-1 M_lambda (SM "Transfer matrix") is then the product of two 4-node
// Lagrange maps, one per axis, and keeps the sixteen moments M_mn, m, n <= 3.
//
// Layout: one record of SLQ = 44 values per node (node = y*nx + x), in 16-byte chunks with
// chunk c of all nodes together (rec_at), in the ABI state's plane order:
//   [0..15] f_0..f_15, [16..31] g_0..g_15, [32] theta, [33] u_x, [34] u_y, [35] rho,
//   [36] T, [37] uhat_x, [38] uhat_y, [39] mass lo, [40] momentum_x lo,
//   [41] momentum_y lo, [42] energy lo, [43] unused
// with population i = 4*jy + jx, c_i = (C1[jx], C1[jy]).  The lo values (FP32 form only;
// zero in FP64) are what the storage rounding of the populations took from the node's
// exact post-collision mass, momentum (sum f v) and energy (sum g); the next step's moments
// add them back, so that changes below half an ulp of the populations (the weak edge of an
// acoustic pulse) are not lost.
//
// One step is three launches: the Korteweg stress K and heat-flux vector q of the state
// the non-local terms come from, their divergences F = -div K and M_0 = 2 div q, and the
// node step (frame search with semi-Lagrangian streaming, then BGK collision with the
// force, heat-flux and force-work sources).  R = float (FP32 storage and streaming /
// collision arithmetic; sums, moments, EoS and non-local terms in float-float) or double.
//
// The node step streams as the D2Q9 step does (pond_step.cuh): the block's tile with a halo
// of two is carried once into a common gauge in shared memory and each thread contracts
// its node's 5 x 5 window along x, then y: 2,240 (FP32) or 1,600 (FP64) multiply-adds a
// population family, where carrying each of 25 nodes into the arrival gauge and spreading it
// over sixteen directions took about 7,000.
// Measured (with init and read-out): four mixed steps of a 1024 x 512 droplet 7.94 -> 1.90 ms,
// three FP64 steps of a 257 x 127 shock-droplet 29 -> 5.5 ms.  The mixed contraction runs on
// packed pairs, rolled over the source rows so that its code stays in the instruction cache
// (609 -> 457 us a step); its FP64 pipe, 22 % busy with the moments and EoS before they went
// to float-float, is idle.  The FP64 form is bound by the FP64 pipe.
#pragma once

#include "pond_kernels.cuh"
#include "pond_step.cuh"   // float-float and wide values, tiles

namespace pond {

constexpr int Q16 = 16;
constexpr int NP16 = 2 * Q16 + 7;   // planes of a D2Q16 state
enum : int { Q_F = 0, Q_G = 16, Q_TH = 32, Q_UX = 33, Q_UY = 34, Q_RHO = 35, Q_T = 36, Q_UHX = 37,
             Q_UHY = 38 };
// 8-byte planes of the non-local scratch (FP64, or float-float pairs): K_xx, K_xy, K_yy,
// q_x, q_y, rho E_lambda, F_x, F_y, M_0
enum : int { NL_KXX = 0, NL_KXY, NL_KYY, NL_QX, NL_QY, NL_REL, NL_FX, NL_FY, NL_M0, NL_PLANES };

constexpr int SLQ = 44;   // values per node record (43 used)
enum : int { Q_MLO = 39, Q_JXLO = 40, Q_JYLO = 41, Q_GLO = 42 };
// value `off` of node n's record, and plane `plane` of the non-local scratch
#define REC16(buf, n, off) (buf)[rec_at(buf, (size_t)(n), (off), (size_t)p.N)]
#define NLP(buf, plane, n, N) (buf)[(size_t)(plane) * (size_t)(N) + (size_t)(n)]

// Four record values from offset off (a multiple of four) of node nd, sixteen, and stores.
__device__ __forceinline__ void ld4(const float *__restrict__ b, size_t nd, size_t N, int off, float (&o)[4])
{
    const float4 t = __ldg(reinterpret_cast<const float4 *>(b) + (size_t)(off / 4) * N + nd);
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld4(const double *__restrict__ b, size_t nd, size_t N, int off, double (&o)[4])
{
    const double2 *q = reinterpret_cast<const double2 *>(b) + (size_t)(off / 2) * N + nd;
    const double2 x = __ldg(q), y = __ldg(q + N);
    o[0] = x.x; o[1] = x.y; o[2] = y.x; o[3] = y.y;
}
template <typename R>
__device__ __forceinline__ void ld16(const R *__restrict__ b, size_t nd, size_t N, int off, R (&o)[16])
{
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        R q[4];
        ld4(b, nd, N, off + 4 * r, q);
#pragma unroll
        for (int k = 0; k < 4; ++k) o[4 * r + k] = q[k];
    }
}
__device__ __forceinline__ void st4(float *b, size_t nd, size_t N, int off, float a, float c, float d, float e)
{
    reinterpret_cast<float4 *>(b)[(size_t)(off / 4) * N + nd] = make_float4(a, c, d, e);
}
__device__ __forceinline__ void st4(double *b, size_t nd, size_t N, int off, double a, double c, double d, double e)
{
    double2 *q = reinterpret_cast<double2 *>(b) + (size_t)(off / 2) * N + nd;
    q[0] = make_double2(a, c);
    q[N] = make_double2(d, e);
}
template <typename R>
__device__ __forceinline__ void st16(R *b, size_t nd, size_t N, int off, const R (&v)[16])
{
#pragma unroll
    for (int r = 0; r < 4; ++r) st4(b, nd, N, off + 4 * r, v[4 * r], v[4 * r + 1], v[4 * r + 2], v[4 * r + 3]);
}

// C1, its weights, and per node k: 1 / prod_{j != k} (c_k - c_j) (the Lagrange
// denominator), the three other nodes o_m (in increasing order) and 1 / (c_k - o_m).
template <typename A>
struct Lat16 {
    A c[4], w[4], inv_den[4];
    A o0[4], o1[4], o2[4], r0[4], r1[4], r2[4];
};

template <typename A>
__device__ __forceinline__ Lat16<A> make_lat16()
{
    const double s6 = sqrt(6.0);
    const double ci = sqrt(3.0 - s6), co = sqrt(3.0 + s6);
    const double c[4] = {-co, -ci, ci, co};
    const double wi = (3.0 + s6) / 12.0, wo = (3.0 - s6) / 12.0;
    Lat16<A> L;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double d = 1.0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j != k) d *= c[k] - c[j];
        L.c[k] = (A)c[k];
        L.w[k] = (A)((k == 0 || k == 3) ? wo : wi);
        L.inv_den[k] = (A)(1.0 / d);
        const double o0 = k == 0 ? c[1] : c[0], o1 = k <= 1 ? c[2] : c[1], o2 = k <= 2 ? c[3] : c[2];
        L.o0[k] = (A)o0; L.o1[k] = (A)o1; L.o2[k] = (A)o2;
        L.r0[k] = (A)(1.0 / (c[k] - o0)); L.r1[k] = (A)(1.0 / (c[k] - o1)); L.r2[k] = (A)(1.0 / (c[k] - o2));
    }
    return L;
}

// element k (runtime, 0..3) of a 4-array held in registers
template <typename A>
__device__ __forceinline__ A sel4(const A (&v)[4], int k)
{
    return k == 0 ? v[0] : (k == 1 ? v[1] : (k == 2 ? v[2] : v[3]));
}

// Row k of a per-axis transfer map in increment form.  With the source velocities at
// xi_j = c_j + eps_j in the target's units, G[k][j] = l_k(c_j + eps_j) and the increment
// D[k][j] = G[k][j] - delta_kj is
//   j != k: inv_den_k prod_m ((c_j - o_m) + eps_j)   (one factor is eps_j exactly),
//   j == k: prod_m (1 + eps_k / (c_k - o_m)) - 1, expanded in the three small terms,
// so that it carries full relative precision however small the gauge change is (FP32
// arithmetic would otherwise lose the change under the rounding of G ~ I).
template <typename A>
struct IncRow {
    A id, r0, r1, r2;
    A d[4][3];   // c_j - o_m (exactly 0 where o_m = c_j)
    int k;
    // the whole row at the offsets eps[0..3]
    __device__ __forceinline__ void row(const A (&eps)[4], A (&out)[4]) const
    {
        const A ek = sel4(eps, k);
        const A t0 = ek * r0, t1 = ek * r1, t2 = ek * r2;
        const A diag = (t0 + t1 + t2) + (t0 * t1 + t0 * t2 + t1 * t2) + t0 * t1 * t2;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const A off = id * ((d[j][0] + eps[j]) * (d[j][1] + eps[j]) * (d[j][2] + eps[j]));
            out[j] = j == k ? diag : off;
        }
    }
};

template <typename A>
__device__ __forceinline__ IncRow<A> inc_row(const Lat16<A> &L, int k)
{
    IncRow<A> b;
    b.id = sel4(L.inv_den, k);
    const A o0 = sel4(L.o0, k), o1 = sel4(L.o1, k), o2 = sel4(L.o2, k);
    b.r0 = sel4(L.r0, k); b.r1 = sel4(L.r1, k); b.r2 = sel4(L.r2, k);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        b.d[j][0] = L.c[j] - o0;
        b.d[j][1] = L.c[j] - o1;
        b.d[j][2] = L.c[j] - o2;
    }
    b.k = k;
    return b;
}

// Cubic Lagrange weights on the nodes 0, 1, 2, 3 at xi (SM "Reconstruction").
template <typename A>
__host__ __device__ __forceinline__ void cubic_weights(A xi, A a[4])
{
    const A x0 = xi, x1 = xi - A(1), x2 = xi - A(2), x3 = xi - A(3);
    a[0] = -(x1 * x2 * x3) / A(6);
    a[1] = (x0 * x2 * x3) / A(2);
    a[2] = -(x0 * x1 * x3) / A(2);
    a[3] = (x0 * x1 * x2) / A(6);
}

// Departure stencil along one axis of a node at integer coordinate X for the velocity v:
// the departure point X - v dt lies at stencil coordinate xi in [1, 2) of the four nodes
// x0 .. x0 + 3 (x0 = floor(X - v dt) - 1); computed from the displacement so that FP32
// keeps full precision on large grids.
template <typename A>
__host__ __device__ __forceinline__ int departure(int X, A v, A dt, A w[4])
{
    const A d = -v * dt;
    const A fl = floor(d);
    cubic_weights<A>(d - fl + A(1), w);
    return stencil_start(X, fl);
}

// ---------------------------------------------------------------------------
// First differences of a field over the 3 x 3 neighbourhood by the isotropic D2Q9 grid
// stencils, unnormalised (D = phi(+1) - phi(-1), S = phi(-1) + 4 phi(0) + phi(+1) per axis):
// dx = S_y D_x, dy = D_y S_x, s = S_y S_x.
template <typename A> struct Diff2 { A dx, dy, s; };
template <typename A, typename Get>
__device__ __forceinline__ Diff2<A> diff2(Get get)
{
    A D[3], S[3];
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const auto a = get(y, 0), b = get(y, 1), c = get(y, 2);
        D[y] = w_sub(c, a);
        S[y] = w_add(w_add(a, c), w_x4(b));
    }
    Diff2<A> o;
    o.dx = w_add(w_add(D[0], D[2]), w_x4(D[1]));
    o.dy = w_sub(S[2], S[0]);
    o.s = w_add(w_add(S[0], S[2]), w_x4(S[1]));
    return o;
}

// Indices of the nine neighbours of a node after the boundary rules.
struct Near9 {
    int x[3];
    long long row[3];
    __device__ __forceinline__ Near9(const DevParams &p, long long n)
    {
        const int X = (int)(n % p.nx), Y = (int)(n / p.nx);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = bc_wrap(X + k - 1, p.nx, p.bcx);
            row[k] = (long long)bc_wrap(Y + k - 1, p.ny, p.bcy) * p.nx;
        }
    }
    __device__ __forceinline__ size_t at(int y, int k) const { return (size_t)(row[y] + x[k]); }
};

// Non-local terms, stage 1 (rho, T of `src`; FP64, or float-float in the FP32 form): with
// grad = 3 sum W c phi(x + c) = d / 12 and lap = 6 sum W (phi(x + c) - phi(x)) = s / 6 of
// the differences to the centre,
//   K = -kappa (rho lap rho + |grad rho|^2 / 2) I + kappa grad rho (x) grad rho  (Eq. korteweg)
//   q = -mu grad h + k grad T, mu = (tau - 1/2) P dt, h = e + p/rho              (Eq. gtilde)
//   rho E_lambda = kappa |grad rho|^2 / 2.
// A block of bx by by nodes (256 threads) stages rho, T and p/rho of its nodes and their
// neighbours once: 1.3 equations of state a node instead of nine (1024 x 512 mixed nodes
// 53 -> 42 us, 20 with the parameters split on the host).  across: blocks along x.
constexpr int NL16_STAGED = 3 * 258;   // (bx + 2) (by + 2) at most, for 256 x 1 and 32 x 8
template <typename R>
__global__ void k_q16_nonlocal1(DevParams p, const R *__restrict__ src, typename Wide<R>::type *__restrict__ nl, int across)
{
    using A = typename Wide<R>::type;
    __shared__ R sr[NL16_STAGED], st[NL16_STAGED];
    __shared__ A sp[NL16_STAGED];
    const int bx = blockDim.x, by = blockDim.y, X0 = (int)(blockIdx.x % across) * bx, Y0 = (int)(blockIdx.x / across) * by, W = bx + 2;
    for (int k = threadIdx.y * bx + threadIdx.x; k < W * (by + 2); k += bx * by) {
        const size_t m = (size_t)bc_wrap(Y0 + k / W - 1, p.ny, p.bcy) * p.nx + bc_wrap(X0 + k % W - 1, p.nx, p.bcx);
        const R r = REC16(src, m, Q_RHO), t = REC16(src, m, Q_T);
        sr[k] = r;
        st[k] = t;
        sp[k] = w_p_over_rho(p, r, t);
    }
    __syncthreads();
    const int X = X0 + threadIdx.x, Y = Y0 + threadIdx.y;
    if (X >= p.nx || Y >= p.ny) return;
    const long long N = p.N, n = (long long)Y * p.nx + X;
    R r[3][3], t[3][3];
    A pi[3][3];
#pragma unroll
    for (int y = 0; y < 3; ++y)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int m = (threadIdx.y + y) * W + threadIdx.x + k;
            r[y][k] = sr[m];
            t[y][k] = st[m];
            pi[y][k] = sp[m];
        }
    const R r0 = r[1][1];
    const Diff2<A> dr = diff2<A>([&](int y, int k) { return w_sub(r[y][k], r0); });
    const Diff2<A> dT = diff2<A>([&](int y, int k) { return t[y][k]; });
    const Diff2<A> dp = diff2<A>([&](int y, int k) { return pi[y][k]; });
    const A g = w_const<A>(1.0 / 12.0), kap = wide_param<A>(p.kappa, p.ff_kap);
    const A gr[2] = {w_mul(dr.dx, g), w_mul(dr.dy, g)}, gT[2] = {w_mul(dT.dx, g), w_mul(dT.dy, g)};
    const A dpi[2] = {dp.dx, dp.dy};
    const A lap = w_mul(dr.s, w_const<A>(1.0 / 6.0));
    const A g2 = w_add(w_mul(gr[0], gr[0]), w_mul(gr[1], gr[1]));
    const A kg2 = w_mul(kap, w_mul(g2, w_const<A>(0.5)));   // rho E_lambda
    const A iso = w_sub(w_mul(w_mul(kap, w_mul(lap, r0)), w_const<A>(-1.0)), kg2);
    const A pr = w_mul(pi[1][1], r0);
    const A mu = w_mul(w_less(wide_p_floor<A>(p), pr) ? pr : wide_p_floor<A>(p), wide_param<A>(p.pd.mu_coef, p.ff_mu));
    const A kc = p.k_cond >= 0.0 ? wide_param<A>(p.k_cond, p.ff_kc) : w_mul(mu, wide_param<A>(p.pd.cvR, p.ff_cvR));
    NLP(nl, NL_KXX, n, N) = w_add(iso, w_mul(kap, w_mul(gr[0], gr[0])));
    NLP(nl, NL_KXY, n, N) = w_mul(kap, w_mul(gr[0], gr[1]));
    NLP(nl, NL_KYY, n, N) = w_add(iso, w_mul(kap, w_mul(gr[1], gr[1])));
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const A gh = w_add(w_sub(w_mul(gT[a], wide_param<A>(p.cv, p.ff_cv)), w_mul(gr[a], wide_param<A>(p.a, p.ff_a))), w_mul(dpi[a], g));
        NLP(nl, NL_QX + a, n, N) = w_sub(w_mul(kc, gT[a]), w_mul(mu, gh));
    }
    NLP(nl, NL_REL, n, N) = kg2;
}

// Stage 2: F = -div K and M_0 = 2 div q with the same gradient stencil.
template <typename R>
__global__ void k_q16_nonlocal2(DevParams p, typename Wide<R>::type *__restrict__ nl)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const long long N = p.N;
    const Near9 nb(p, n);
    auto diff = [&](int plane) { return diff2<A>([&](int y, int k) { return NLP(nl, plane, nb.at(y, k), N); }); };
    const Diff2<A> xx = diff(NL_KXX), xy = diff(NL_KXY), yy = diff(NL_KYY), qx = diff(NL_QX), qy = diff(NL_QY);
    NLP(nl, NL_FX, n, N) = w_mul(w_add(xx.dx, xy.dy), w_const<A>(-1.0 / 12.0));
    NLP(nl, NL_FY, n, N) = w_mul(w_add(xy.dx, yy.dy), w_const<A>(-1.0 / 12.0));
    NLP(nl, NL_M0, n, N) = w_mul(w_add(qx.dx, qy.dy), w_const<A>(2.0 / 12.0));
}

// ---------------------------------------------------------------------------
// Semi-Lagrangian streaming into node (X, Y) in gauge (th, ux, uy) (Eqs. f/g streaming):
// for direction i the departure point x - v_i dt is reconstructed from the 4 x 4 nodes
// around it, each node's populations first carried from its own gauge into (th, u) by
// the transfer map.  Only component i of G f is needed: with the per-axis maps
// Gx[ix][jx] = l_ix((s' c_jx + u'_x - u_x)/s) (s' = sqrt(theta') and u' the neighbour's
// gauge) it is sum_jy Gy[iy][jy] sum_jx Gx[ix][jx] f_(4 jy + jx), evaluated as f_i plus
// increments (G = I + D per axis).  Returns the increments fi, gi of the streamed
// populations over the node's own stored f_i, g_i (streamed f_i = own f_i + fi[i]).
template <typename R>
__device__ void q16_stream(const DevParams &p, const Lat16<R> &L, const R *__restrict__ in, int X,
                           int Y, R th, R ux, R uy, R *fi, R *gi)
{
    const long long nself = (long long)Y * p.nx + X;
    const R s = sqrt_(th), is = R(1) / s, dt = (R)p.dt;
#pragma unroll 1
    for (int iy = 0; iy < 4; ++iy) {
        const IncRow<R> by = inc_row(L, iy);
        R ay[4];
        const int y0 = departure<R>(Y, s * sel4(L.c, iy) + uy, dt, ay);
        long long rows[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) rows[m] = (long long)bc_wrap(y0 + m, p.ny, p.bcy) * p.nx;
#pragma unroll 1
        for (int ix = 0; ix < 4; ++ix) {
            const IncRow<R> bx = inc_row(L, ix);
            R ax[4];
            const int x0 = departure<R>(X, s * sel4(L.c, ix) + ux, dt, ax);
            int cols[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) cols[k] = bc_wrap(x0 + k, p.nx, p.bcx);
            // interpolated as ref + sum w (v - ref) with ref = the node's own f_i, g_i: the
            // weights' rounded sum then only scales the small differences
            const int i = 4 * iy + ix;
            const R refF = REC16(in, nself, Q_F + i), refG = REC16(in, nself, Q_G + i);
            R sf = R(0), sg = R(0);
            // the 16 stencil nodes as a loop unrolled by two only (fully unrolled, the body
            // overflows the instruction cache; two iterations give independent chains)
#pragma unroll 2
            for (int mk = 0; mk < 16; ++mk) {
                const int m = mk >> 2, k = mk & 3;
                const size_t nd = (size_t)(sel4(rows, m) + sel4(cols, k));
                R gv[4];   // theta, u_x, u_y, rho of the stencil node
                ld4(in, nd, (size_t)p.N, Q_TH, gv);
                const R ths = gv[0];
                const R ds = (ths - th) / (sqrt_(ths) + s) * is;   // (s' - s)/s
                const R ex = (gv[1] - ux) * is, ey = (gv[2] - uy) * is;
                R epx[4], epy[4], gx[4], gy[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    epx[j] = ds * L.c[j] + ex;
                    epy[j] = ds * L.c[j] + ey;
                }
                bx.row(epx, gx);
                by.row(epy, gy);
                // per row jy: base = f_(jy, ix), inc = sum_jx Dx[ix][jx] f_(jy, jx)
                R bf[4], bg[4], xf[4], xg[4];
#pragma unroll
                for (int jy = 0; jy < 4; ++jy) {
                    R fr[4], gr[4];
                    ld4(in, nd, (size_t)p.N, Q_F + 4 * jy, fr);
                    ld4(in, nd, (size_t)p.N, Q_G + 4 * jy, gr);
                    R df = R(0), dg = R(0);
#pragma unroll
                    for (int jx = 0; jx < 4; ++jx) { df += gx[jx] * fr[jx]; dg += gx[jx] * gr[jx]; }
                    bf[jy] = sel4(fr, ix); bg[jy] = sel4(gr, ix);
                    xf[jy] = df; xg[jy] = dg;
                }
                R df = R(0), dg = R(0);
#pragma unroll
                for (int jy = 0; jy < 4; ++jy) {
                    df += gy[jy] * (bf[jy] + xf[jy]);
                    dg += gy[jy] * (bg[jy] + xg[jy]);
                }
                // [G f]_i - ref = (f_i - ref) + x-increment of row iy + y-increment
                const R wgt = sel4(ax, k) * sel4(ay, m);
                sf += wgt * (((sel4(bf, iy) - refF) + sel4(xf, iy)) + df);
                sg += wgt * (((sel4(bg, iy) - refG) + sel4(xg, iy)) + dg);
            }
            fi[4 * iy + ix] = sf;
            gi[4 * iy + ix] = sg;
        }
    }
}

// The FP32 form's population sums in float-float on the FP32 pipes (GB300 runs FP64 at
// 1/64 of the FP32 rate, and these sums were most of the step's FP64 work).  C1's outer and
// inner nodes co = sqrt(3 + sqrt 6), ci = sqrt(3 - sqrt 6) as hi + lo (hi their FP32
// rounding, lo the FP32 rounding of the rest: together within 2^-48 relative).
__device__ __forceinline__ ffv q16_co() { return {0x1.2ace16p+1f, -0x1.b3aab0p-26f}; }
__device__ __forceinline__ ffv q16_ci() { return {0x1.7be2aep-1f, -0x1.4e69e0p-26f}; }

// Moments of 16 values v (i = 4 jy + jx) in the wide type: out[0] = sum v and, with
// WEIGHTED, out[1] = sum v c_jx and out[2] = sum v c_jy, from the column sums C_k and
// row sums R_r (sum v c_jx = co (C_3 - C_0) + ci (C_2 - C_1), the same over rows for y).
// Each float-float addition is exact up to ~2^-48 of its result (TwoSum, the error terms
// added in FP32), far below what the kept remainders resolve (FP32 storage rounding).
template <bool WEIGHTED>
__device__ __forceinline__ void sums16(const float *v, ffv *out)
{
    ffv C[4], Rw[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        C[k] = {v[k], 0.0f};
#pragma unroll
        for (int r = 1; r < 4; ++r) C[k] = ff_add(C[k], v[4 * r + k]);
    }
    const ffv s = ff_add(ff_add(C[0], C[1]), ff_add(C[2], C[3]));
    out[0] = s;
    if (WEIGHTED) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            Rw[r] = {v[4 * r], 0.0f};
#pragma unroll
            for (int k = 1; k < 4; ++k) Rw[r] = ff_add(Rw[r], v[4 * r + k]);
        }
        const ffv co = q16_co(), ci = q16_ci();
        const ffv sx = ff_add(ff_mul(ff_add(C[3], ff_neg(C[0])), co), ff_mul(ff_add(C[2], ff_neg(C[1])), ci));
        const ffv sy = ff_add(ff_mul(ff_add(Rw[3], ff_neg(Rw[0])), co), ff_mul(ff_add(Rw[2], ff_neg(Rw[1])), ci));
        out[1] = sx;
        out[2] = sy;
    }
}
template <bool WEIGHTED>
__device__ __forceinline__ void sums16(const double *v, double *out)
{
    double C[4], W[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        C[k] = (v[k] + v[4 + k]) + (v[8 + k] + v[12 + k]);
        if (WEIGHTED) W[k] = (v[4 * k] + v[4 * k + 1]) + (v[4 * k + 2] + v[4 * k + 3]);
    }
    out[0] = (C[0] + C[1]) + (C[2] + C[3]);
    if (WEIGHTED) {
        const double s6 = sqrt(6.0), ci = sqrt(3.0 - s6), co = sqrt(3.0 + s6);
        out[1] = co * (C[3] - C[0]) + ci * (C[2] - C[1]);
        out[2] = co * (W[3] - W[0]) + ci * (W[2] - W[1]);
    }
}

// Per-axis transfer map from gauge (s_src, u_src) into (s_dst, u_dst) in increment
// form: D[i][j] = l_i(c_j + eps_j) - delta_ij with eps_j = ((s_src - s_dst) c_j + du)/s_dst;
// ds = (s_src - s_dst)/s_dst and du / s_dst are passed in.
template <typename A>
__device__ __forceinline__ void axis_inc(const Lat16<A> &L, A ds, A du, A D[4][4])
{
    A eps[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) eps[j] = ds * L.c[j] + du;
#pragma unroll
    for (int i = 0; i < 4; ++i) inc_row(L, i).row(eps, D[i]);
}

// Increment of (I + Dy) (x) (I + Dx) applied to h: out_(4 iy + ix) = [G h]_i - h_i.
template <typename A>
__device__ __forceinline__ void apply_inc(const A Dx[4][4], const A Dy[4][4], const A h[16], A out[16])
{
    A t[16];
#pragma unroll
    for (int jy = 0; jy < 4; ++jy)
#pragma unroll
        for (int ix = 0; ix < 4; ++ix) {
            A a = A(0);
#pragma unroll
            for (int jx = 0; jx < 4; ++jx) a += Dx[ix][jx] * h[4 * jy + jx];
            t[4 * jy + ix] = a;
        }
#pragma unroll
    for (int iy = 0; iy < 4; ++iy)
#pragma unroll
        for (int ix = 0; ix < 4; ++ix) {
            A a = A(0);
#pragma unroll
            for (int jy = 0; jy < 4; ++jy) a += Dy[iy][jy] * (h[4 * jy + ix] + t[4 * jy + ix]);
            out[4 * iy + ix] = t[4 * iy + ix] + a;
        }
}

// ---------------------------------------------------------------------------
// General stream, for departure points beyond the staged halo (|v| dt >= 1), tiles whose
// velocities spread too far (FAR_SPEED) and non-finite gauges: reads the stencil nodes'
// records from global memory.  On a tensor lattice the union of a node's sixteen 4 x 4
// departure stencils is the product of the per-axis unions: W x H nodes with W (H) = 4 + the
// spread of the four departure floors along the axis, 5 x 5 while |v| dt < 1 in every direction.
// Each region node is carried into the arrival gauge once for all sixteen directions
// (G f = f + [(I + Dy) (x) (I + Dx) - I] f), and direction i takes its Lagrange-weighted
// share of component i.  The arithmetic per (direction, stencil node) pair is that of
// q16_stream, so the two agree up to the rounding of zero-weight terms; the region form
// transforms about 25 nodes per stream against 256 pairs.

// Largest region side the region stream takes; wider regions take q16_stream.  Departures
// beyond the halo are the one thing that earlier kernels, which streamed every node this way,
// did faster (us a step of 128 x 128 nodes at dt = 1, earlier / this, mixed: a droplet at 1.4
// T_cr 174 / 192, at 1.9 T_cr, a seventh of the streams per pair, 629 / 838; a flow at |v| dt = 1.3
// 183 / 204; FP64 within 4 %): f and g take two passes, and the weight tables lie in local
// memory.  One pass over both gave 168 and 175 us but cost every other step 3.7 %, by the
// registers of the calling kernel.
constexpr int Q16_REGION_MAX = 6;
// Entries of a thread's Lagrange weight tables: (axis * 4 + k) * Q16_REGION_MAX + c is the
// weight of region column (row) c in the stencil of axis component k, zero outside it.
constexpr int Q16_WT_ENTRIES = 2 * 4 * Q16_REGION_MAX;

// Departure floors and Lagrange weights of the four axis components for the gauge
// velocity u along one axis (as in `departure`), the table entries of that axis, and the
// region's first coordinate lo (= X + min floor - 1) and side. False, with nothing
// written, when the side exceeds Q16_REGION_MAX or a floor is not finite or not within
// 2^20 (the floors are checked as reals before any conversion to int).
template <typename R>
__device__ __forceinline__ bool q16_region_axis(const Lat16<R> &L, int X, R s, R u, R dt, R *wt, int &lo,
                                                int &side)
{
    R fl[4], a[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const R d = -(s * L.c[k] + u) * dt;
        fl[k] = floor(d);
        cubic_weights<R>(d - fl[k] + R(1), a[k]);
    }
    const R flo = fmin(fmin(fl[0], fl[1]), fmin(fl[2], fl[3]));
    const R fhi = fmax(fmax(fl[0], fl[1]), fmax(fl[2], fl[3]));
    if (!(fhi - flo <= R(Q16_REGION_MAX - 4)) || !(fabs(flo) <= R(1 << 20)) || !(fabs(fhi) <= R(1 << 20)))
        return false;
    lo = X + (int)flo - 1;
    side = (int)(fhi - flo) + 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int o = (int)(fl[k] - flo);   // 0 .. side - 4
#pragma unroll
        for (int c = 0; c < Q16_REGION_MAX; ++c) {
            const int j = c - o;
            wt[(k * Q16_REGION_MAX + c)] =
                j == 0 ? a[k][0] : (j == 1 ? a[k][1] : (j == 2 ? a[k][2] : (j == 3 ? a[k][3] : R(0))));
        }
    }
    return true;
}

// One population set (16 values at record offset off) of a region node: x-increments t = (I (x) Dx) h, the
// y-increment of each component, and acc_i += wx_ix wy_iy ((h_i - ref_i) + t_i + dy_i).
template <typename R>
__device__ __forceinline__ void q16_region_pop(const R (&Dx)[4][4], const R (&Dy)[4][4], const R *__restrict__ in,
                                               size_t nd, size_t N, int off, const R (&ref)[Q16], const R (&wx)[4], const R (&wy)[4],
                                               R (&acc)[Q16])
{
    R h[Q16], t[Q16];
    ld16(in, nd, N, off, h);
#pragma unroll
    for (int jy = 0; jy < 4; ++jy)
#pragma unroll
        for (int ix = 0; ix < 4; ++ix) {
            R a = R(0);
#pragma unroll
            for (int jx = 0; jx < 4; ++jx) a += Dx[ix][jx] * h[4 * jy + jx];
            t[4 * jy + ix] = a;
        }
#pragma unroll
    for (int iy = 0; iy < 4; ++iy)
#pragma unroll
        for (int ix = 0; ix < 4; ++ix) {
            R dy = R(0);
#pragma unroll
            for (int jy = 0; jy < 4; ++jy) dy += Dy[iy][jy] * (h[4 * jy + ix] + t[4 * jy + ix]);
            const int i = 4 * iy + ix;
            acc[i] += (wx[ix] * wy[iy]) * (((h[i] - ref[i]) + t[i]) + dy);
        }
}

// The region pass over the W x H region at (xlo, ylo), skipping region entry `skip` (-1:
// none): the increments of the streamed populations over the node's own (node self) for
// the population set at record offset `off` (Q_F or Q_G) into out.
template <typename R>
__device__ __forceinline__ void q16_region_pass(const DevParams &p, const Lat16<R> &L, const R *__restrict__ in,
                                                size_t self, int xlo, int ylo, int W, int H, int skip,
                                                R th, R ux, R uy, const R *wt, int off, R *out)
{
    const R s = sqrt_(th), is = R(1) / s;
    const size_t N = (size_t)p.N;
    R ref[Q16], acc[Q16];
    ld16(in, self, N, off, ref);
#pragma unroll
    for (int i = 0; i < Q16; ++i) acc[i] = R(0);
#pragma unroll 1
    for (int cy = 0; cy < H; ++cy) {
        const long long row = (long long)bc_wrap(ylo + cy, p.ny, p.bcy) * p.nx;
        R wy[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) wy[k] = wt[(4 + k) * Q16_REGION_MAX + cy];
#pragma unroll 1
        for (int cx = 0; cx < W; ++cx) {
            if (cy * W + cx == skip) continue;
            const size_t nd = (size_t)(row + bc_wrap(xlo + cx, p.nx, p.bcx));
            R wx[4], gv[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) wx[k] = wt[k * Q16_REGION_MAX + cx];
            ld4(in, nd, N, Q_TH, gv);   // theta, u_x, u_y, rho of the region node
            const R ds = (gv[0] - th) / (sqrt_(gv[0]) + s) * is;   // (s' - s)/s
            R Dx[4][4], Dy[4][4];
            axis_inc<R>(L, ds, (gv[1] - ux) * is, Dx);
            axis_inc<R>(L, ds, (gv[2] - uy) * is, Dy);
            q16_region_pop<R>(Dx, Dy, in, nd, N, off, ref, wx, wy, acc);
        }
    }
#pragma unroll
    for (int i = 0; i < Q16; ++i) out[i] = acc[i];
}

// Streaming of node (X, Y) into gauge (th, ux, uy) by the region stream where the region
// fits, else by q16_stream; skip_own leaves out the node's own region entry (valid when
// the gauge is the node's stored gauge: the map is then the identity and the entry adds
// exactly zero).  Adds the region entries transformed to nreg, or 1 to npair.
template <typename R>
__device__ __noinline__ void q16_stream_any(const DevParams &p, const R *__restrict__ in, int X, int Y, R th, R ux,
                                            R uy, bool skip_own, R *fi, R *gi, unsigned &nreg, unsigned &npair)
{
    const Lat16<R> L = make_lat16<R>();
    const R s = sqrt_(th), dt = (R)p.dt;
    R wt[Q16_WT_ENTRIES];
    int xlo, ylo, W, H;
    if (q16_region_axis<R>(L, X, s, ux, dt, wt, xlo, W) &&
        q16_region_axis<R>(L, Y, s, uy, dt, wt + 4 * Q16_REGION_MAX, ylo, H)) {
        const int cxo = X - xlo, cyo = Y - ylo;
        const int skip = (skip_own && cxo >= 0 && cxo < W && cyo >= 0 && cyo < H) ? cyo * W + cxo : -1;
        const size_t self = (size_t)Y * p.nx + X;
        // one population set per pass, the pass's code once (a rolled loop)
#pragma unroll 1
        for (int ps = 0; ps < 2; ++ps)
            q16_region_pass<R>(p, L, in, self, xlo, ylo, W, H, skip, th, ux, uy, wt, ps == 0 ? Q_F : Q_G,
                               ps == 0 ? fi : gi);
        nreg += (unsigned)(W * H - (skip >= 0 ? 1 : 0));
    } else {
        q16_stream<R>(p, L, in, X, Y, th, ux, uy, fi, gi);
        npair += 1;
    }
}

// ---------------------------------------------------------------------------
// Staging and contraction (the form of the D2Q9 step, see the head of pond_step.cuh, with
// four velocities per axis).  Values per staged slot: 32 carried populations (f, g), padded
// so that slots start on distinct banks.
template <typename R> struct Slot16;
template <> struct Slot16<float> { static constexpr int stride = 36; };
template <> struct Slot16<double> { static constexpr int stride = 33; };
// place of population i of family fam (0 f, 1 g): side by side in FP32 (see contract in
// pond_step.cuh)
template <typename R> __host__ __device__ constexpr int slot16_at(int fam, int i) { return sizeof(R) == 4 ? 2 * i + fam : 16 * fam + i; }
// What a thread keeps in shared memory across the stream: wide values (own sums, F, rho
// E_lambda, M_0), then the y weights and rows of the map in R.
enum : int { KW_OWN = 0, KW_F = 6, KW_REL = 8, KW_M0 = 9, KW_N = 10, KR_WY = 0, KR_LY = 20, KR_N = 36 };
template <typename R>
constexpr size_t q16_smem_bytes(int tx, int ty)
{
    return (size_t)STEP_THREADS * (KW_N * 8 + KR_N * sizeof(R)) + (size_t)step_slots(tx, ty) * Slot16<R>::stride * sizeof(R);
}

// The rows of a per-axis map, G[k][j] = l_k(xi_j) at xi_j = (1 + q) c_j + w, as products.
template <typename A>
__device__ __forceinline__ void axis_rows16(const Lat16<A> &L, A q, A w, A (&G)[4][4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const A x = (A(1) + q) * L.c[j] + w;
        const A g0 = x - L.c[0], g1 = x - L.c[1], g2 = x - L.c[2], g3 = x - L.c[3];
        const A a = g0 * g1, b = g2 * g3;
        G[0][j] = L.inv_den[0] * g1 * b; G[1][j] = L.inv_den[1] * g0 * b;
        G[2][j] = L.inv_den[2] * g3 * a; G[3][j] = L.inv_den[3] * g2 * a;
    }
}

// Departure points of the four components of an axis and their cubic weights; true when
// every floor is -1 or 0 (the stencils then lie within two nodes of the arrival node).
template <typename R>
__host__ __device__ __forceinline__ bool axis_weights16(const Lat16<R> &L, R s, R u, R dt, R (&a)[4][4], bool (&near0)[4])
{
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const R d = -(s * L.c[j] + u) * dt;
        const R f = floor(d);
        near0[j] = f == R(0);
        ok = ok && (f == R(0) || f == R(-1));
        const R t0 = d - f + R(1), t1 = t0 - R(1), t2 = t0 - R(2), t3 = t0 - R(3);
        const R p12 = t1 * t2, p03 = t0 * t3;
        a[j][0] = p12 * t3 * R(-1.0 / 6.0);
        a[j][1] = p03 * t2 * R(0.5);
        a[j][2] = p03 * t1 * R(-0.5);
        a[j][3] = p12 * t0 * R(1.0 / 6.0);
    }
    return ok;
}

// The stream over the staged slots: acc = sums over the window of the node's slot `own`
// (FP32: of differences to the own slot, i.e. increments; FP64: the streamed populations);
// keep = the thread's y weights and rows.  FP32: f and g in one instruction (packed pairs),
// five columns and rows with zero weights outside a component's four nodes; the x weights
// are kept apart from the rows of the map (96 instead of 80 multiply-adds a row and source
// index, but 72 registers of pairs instead of 160).
__device__ __forceinline__ void contract16(const float *own, int pitch, const float (&ax)[4][4], const bool (&nx0)[4],
                                           const float (&Lx)[4][4], const float *keep, float (&acc)[2][16])
{
    constexpr int DS = Slot16<float>::stride;
    f32x2 wx[4][5], L2[4][4], a2[16];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const int lo = c > 3 ? 3 : c, hi = c < 1 ? 0 : c - 1;
            const float w = nx0[k] ? (c == 0 ? 0.0f : ax[k][hi]) : (c == 4 ? 0.0f : ax[k][lo]);
            wx[k][c] = pack2(w, w);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) L2[k][m] = pack2(Lx[k][m], Lx[k][m]);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) a2[i] = 0ull;
    const float *row = own - (2 * pitch + 2) * DS;
#pragma unroll 1
    for (int cy = 0; cy < 5; ++cy, row += pitch * DS) {
#pragma unroll 1
        for (int n = 0; n < 4; ++n) {   // rolled: the body stays in the instruction cache
            f32x2 v[5][4], d[4];
            {
                float t[8];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    float x[4];
                    lds4(own + 8 * n + 4 * q, x);
#pragma unroll
                    for (int e = 0; e < 4; ++e) t[4 * q + e] = x[e];
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) d[m] = pack2(-t[2 * m], -t[2 * m + 1]);
            }
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                const ulonglong2 x = reinterpret_cast<const ulonglong2 *>(row + c * DS + 8 * n)[0];
                const ulonglong2 y = reinterpret_cast<const ulonglong2 *>(row + c * DS + 8 * n)[1];
                v[c][0] = add2(x.x, d[0]); v[c][1] = add2(x.y, d[1]);
                v[c][2] = add2(y.x, d[2]); v[c][3] = add2(y.y, d[3]);
            }
            f32x2 wn[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                const float w = keep[(KR_WY + 5 * l + cy) * STEP_THREADS] * keep[(KR_LY + 4 * l + n) * STEP_THREADS];
                wn[l] = pack2(w, w);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                f32x2 t = 0ull;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    f32x2 q = 0ull;
#pragma unroll
                    for (int c = 0; c < 5; ++c) q = fma2(wx[k][c], v[c][m], q);
                    t = fma2(L2[k][m], q, t);
                }
#pragma unroll
                for (int l = 0; l < 4; ++l) a2[4 * l + k] = fma2(wn[l], t, a2[4 * l + k]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) unpack2(a2[i], acc[0][i], acc[1][i]);
}
// FP64: each component's own four columns.
__device__ __forceinline__ void contract16(const double *own, int pitch, const double (&ax)[4][4], const bool (&nx0)[4],
                                           const double (&Lx)[4][4], const double *keep, double (&acc)[2][16])
{
    constexpr int DS = Slot16<double>::stride;
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[0][i] = acc[1][i] = 0.0;
    const double *row = own - (2 * pitch + 2) * DS;
#pragma unroll 1
    for (int cy = 0; cy < 5; ++cy, row += pitch * DS) {
        double wn[4][4];
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const double w = keep[(KR_WY + 5 * l + cy) * STEP_THREADS];
#pragma unroll
            for (int n = 0; n < 4; ++n) wn[l][n] = w * keep[(KR_LY + 4 * l + n) * STEP_THREADS];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double wl[4][4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int m = 0; m < 4; ++m) wl[c][m] = ax[k][c] * Lx[k][m];
            const double *r = row + (nx0[k] ? DS : 0);
#pragma unroll
            for (int fam = 0; fam < 2; ++fam)
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    double t = 0.0;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int m = 0; m < 4; ++m) t = fma(wl[c][m], r[c * DS + 16 * fam + 4 * n + m], t);
#pragma unroll
                    for (int l = 0; l < 4; ++l) acc[fam][4 * l + k] = fma(wn[l][n], t, acc[fam][4 * l + k]);
                }
        }
    }
}

// Apply the rows Gx, Gy to 16 values h (i = 4 jy + jx), in place.
template <typename A>
__device__ __forceinline__ void apply_rows16(const A (&Gx)[4][4], const A (&Gy)[4][4], A (&h)[16])
{
    A t[16];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            t[4 * j + k] = Gx[k][0] * h[4 * j] + Gx[k][1] * h[4 * j + 1] + Gx[k][2] * h[4 * j + 2] + Gx[k][3] * h[4 * j + 3];
#pragma unroll
    for (int l = 0; l < 4; ++l)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            h[4 * l + k] = Gy[l][0] * t[k] + Gy[l][1] * t[4 + k] + Gy[l][2] * t[8 + k] + Gy[l][3] * t[12 + k];
}

// ---------------------------------------------------------------------------
// The node step, one thread per node of the block's tile.  in: state at t - dt; nl:
// non-local terms (F, rho E_lambda, M_0) of the state they are taken from; out: state at
// t.  Frame search: predictor = the node's stored gauge; corrector = re-stream with
// (theta*, u) of the streamed moments until the relative change is <= tol or after
// max_iter streams.  Collision: equilibria built in the co-moving frame lambda* =
// (theta*, u) and carried into the streaming gauge (Eqs. f collision with S_i, g collision
// with gtilde and phi, new geq).
constexpr int Q16_MIN_BLOCKS = 3;   // FP32 blocks per SM (168 registers)
template <typename R>
__global__ void __launch_bounds__(STEP_THREADS, sizeof(R) == 4 ? Q16_MIN_BLOCKS : 2)
    k_q16_step(DevParams p, const R *__restrict__ in, const typename Wide<R>::type *__restrict__ nl,
               R *__restrict__ out, DevStats *stats)
{
    using A = typename Wide<R>::type;
    constexpr int DS = Slot16<R>::stride;
    extern __shared__ __align__(128) unsigned char q16_dyn_smem[];
    A *keep_w = reinterpret_cast<A *>(q16_dyn_smem) + threadIdx.x;   // this thread's columns
    R *keep = reinterpret_cast<R *>(q16_dyn_smem + (size_t)STEP_THREADS * KW_N * 8) + threadIdx.x;
    R *slots = reinterpret_cast<R *>(q16_dyn_smem + (size_t)STEP_THREADS * (KW_N * 8 + KR_N * sizeof(R)));
    __shared__ StepCounts counts;
    __shared__ uint4 best[BEST];
    const int tid = threadIdx.x;
    const size_t N = (size_t)p.N;
    const int TX = p.tile_x, TY = p.tile_y, WT = TX + 2 * HALO, nslots = step_slots(TX, TY);
    const int X0 = (blockIdx.x % p.tiles_x) * TX, Y0 = (blockIdx.x / p.tiles_x) * TY;
    if (tid == 0) counts = StepCounts{};
    const Lat16<R> L = make_lat16<R>();
    const float iwt = 1.0f / (float)WT;
    auto node_of = [&](int k) -> size_t {
        const int cv = (int)(((float)k + 0.5f) * iwt), cu = k - cv * WT;
        return (size_t)bc_wrap(Y0 - HALO + cv, p.ny, p.bcy) * p.nx + bc_wrap(X0 - HALO + cu, p.nx, p.bcx);
    };

    // ---- staging: every record of the tile and its halo carried into the common gauge
    Extremes<2> ex;
    for (int k = tid; k < nslots; k += STEP_THREADS) {
        R g4[4];
        ld4(in, node_of(k), N, Q_TH, g4);
        ex.offer(g4[0], g4 + 1, k);
    }
    ex = tile_extremes(ex, best);
    bool inc = sizeof(R) == 4 && ex.smooth();
    const size_t nbase = node_of(min((int)ex.at, nslots - 1));
    R gb[3];     // sqrt(theta), u_x, u_y of the tile's gauge
    R dt_b = typed<R>(p).dt;   // infinite in a tile whose velocities spread too far (no contraction)
    {
        R g4[4], cold[4];
        ld4(in, nbase, N, Q_TH, g4);
        ld4(in, node_of(min((int)ex.lat, nslots - 1)), N, Q_TH, cold);
        common_gauge<R, 3>(inc, g4, cold, gb);
        if (__syncthreads_or(ex.spread(gb, sqrtf(ex.hottest())))) {
            inc = false;
            if (!middle_gauge<R, 2>(ex, best, gb)) dt_b = R(1) / R(0);
        }
        const R thb = inc ? g4[0] : gb[0] * gb[0], inv_sb = R(1) / gb[0];
#pragma unroll 1
        for (int k = tid; k < nslots; k += STEP_THREADS) {
            const size_t nd = node_of(k);
            ld4(in, nd, N, Q_TH, g4);
            const R e = fdiv_(g4[0] - thb, (sqrt_(g4[0]) + gb[0]) * gb[0]);
            const R wx = (g4[1] - gb[1]) * inv_sb, wy = (g4[2] - gb[2]) * inv_sb;
            R Gx[4][4], Gy[4][4];
            if (inc) {
                axis_inc<R>(L, e, wx, Gx);
                axis_inc<R>(L, e, wy, Gy);
            } else {
                axis_rows16<R>(L, e, wx, Gx);
                axis_rows16<R>(L, e, wy, Gy);
            }
#pragma unroll 1
            for (int fam = 0; fam < 2; ++fam) {
                R h[16];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    R q[4];
                    ld4(in, nd, N, 16 * fam + 4 * r, q);
#pragma unroll
                    for (int c = 0; c < 4; ++c) h[4 * r + c] = q[c];
                }
                if (inc) {
                    R o[16];
                    apply_inc<R>(Gx, Gy, h, o);
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        R q[4];
                        ld4(in, nbase, N, 16 * fam + 4 * r, q);
#pragma unroll
                        for (int c = 0; c < 4; ++c) h[4 * r + c] = (h[4 * r + c] - q[c]) + o[4 * r + c];
                    }
                } else {
                    apply_rows16<R>(Gx, Gy, h);
                }
                R *dst = slots + (size_t)k * DS;
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[slot16_at<R>(0, i) + fam * slot16_at<R>(1, 0)] = h[i];
            }
        }
    }
    __syncthreads();

    const int tx = tid % TX, ty = tid / TX;
    const int X = X0 + tx, Y = Y0 + ty;
    const bool valid = X < p.nx && Y < p.ny;
    unsigned its = 0, nreg = 0, npair = 0;
    bool conv = true, floored = false, bad = false;
    if (valid) {
        const size_t n = (size_t)Y * p.nx + X;
        const R *own_slot = slots + (size_t)((ty + HALO) * WT + tx + HALO) * DS;
        keep_w[KW_F * STEP_THREADS] = NLP(nl, NL_FX, n, N);
        keep_w[(KW_F + 1) * STEP_THREADS] = NLP(nl, NL_FY, n, N);
        keep_w[KW_REL * STEP_THREADS] = NLP(nl, NL_REL, n, N);
        keep_w[KW_M0 * STEP_THREADS] = NLP(nl, NL_M0, n, N);
        // sums of the node's stored populations and its kept remainders: sum f + mass lo,
        // sum f c_x, sum f c_y, sum g + energy lo, momentum lo (absolute)
        R th, u[2];
        {
            A own[6];
            R v[16], lo[4];
            ld16(in, n, N, Q_F, v);
            sums16<true>(v, own);
            ld16(in, n, N, Q_G, v);
            sums16<false>(v, own + 3);
            ld4(in, n, N, Q_T, lo);
            own[0] = w_add(own[0], lo[3]);
            ld4(in, n, N, Q_JXLO, lo);
            own[3] = w_add(own[3], lo[2]);
            own[4] = w_wide(lo[0]);
            own[5] = w_wide(lo[1]);
#pragma unroll
            for (int k = 0; k < 6; ++k) keep_w[(KW_OWN + k) * STEP_THREADS] = own[k];
            R g4[4];
            ld4(in, n, N, Q_TH, g4);
            th = g4[0]; u[0] = g4[1]; u[1] = g4[2];
        }
        R fi[16], gi[16];   // increments of the streamed populations
        Macro<2, R> m;
        for (;;) {
            ++its;
            const R s = sqrt_(th), inv_s = R(1) / s;
            R ax[4][4], ay[4][4];
            bool nx0[4], ny0[4];
            const bool okx = axis_weights16<R>(L, s, u[0], dt_b, ax, nx0), oky = axis_weights16<R>(L, s, u[1], dt_b, ay, ny0);
            if (okx && oky) {
                auto side = [](const bool (&z)[4]) { return (z[0] == z[1] && z[1] == z[2] && z[2] == z[3]) ? 4 : 5; };
                nreg += (unsigned)(side(nx0) * side(ny0) - (its == 1 ? 1 : 0));
                R Lx[4][4], acc[2][16];
                const R q = (gb[0] - s) * inv_s;
                {
                    R Ly[4][4];
                    axis_rows16<R>(L, q, (gb[2] - u[1]) * inv_s, Ly);
#pragma unroll
                    for (int l = 0; l < 4; ++l) {
#pragma unroll
                        for (int c = 0; c < 5; ++c) {
                            const int lo = c > 3 ? 3 : c, hi = c < 1 ? 0 : c - 1;
                            keep[(KR_WY + 5 * l + c) * STEP_THREADS] =
                                ny0[l] ? (c == 0 ? R(0) : ay[l][hi]) : (c == 4 ? R(0) : ay[l][lo]);
                        }
#pragma unroll
                        for (int m2 = 0; m2 < 4; ++m2) keep[(KR_LY + 4 * l + m2) * STEP_THREADS] = Ly[l][m2];
                    }
                }
                axis_rows16<R>(L, q, (gb[1] - u[0]) * inv_s, Lx);
                contract16(own_slot, WT, ax, nx0, Lx, keep, acc);
                if constexpr (sizeof(R) == 8) {
                    R v[16];
                    ld16(in, n, N, Q_F, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[0][i] -= v[i];
                    ld16(in, n, N, Q_G, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[1][i] -= v[i];
                } else if (its > 1) {
                    // the node's own populations carried from their stored gauge
                    R g4[4], v[16], o[16], Dx[4][4], Dy[4][4];
                    ld4(in, n, N, Q_TH, g4);
                    const R e = fdiv_(g4[0] - th, (sqrt_(g4[0]) + s) * s);
                    axis_inc<R>(L, e, (g4[1] - u[0]) * inv_s, Dx);
                    axis_inc<R>(L, e, (g4[2] - u[1]) * inv_s, Dy);
#pragma unroll
                    for (int fam = 0; fam < 2; ++fam) {
                        ld16(in, n, N, 16 * fam, v);
                        apply_inc<R>(Dx, Dy, v, o);
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[fam][i] += o[i];
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    fi[i] = acc[0][i];
                    gi[i] = acc[1][i];
                }
            } else {
                R f2[16], g2[16];
                q16_stream_any<R>(p, in, X, Y, th, u[0], u[1], its == 1, f2, g2, nreg, npair);
#pragma unroll
                for (int i = 0; i < 16; ++i) { fi[i] = f2[i]; gi[i] = g2[i]; }
            }
            A d[4], own[6];
            sums16<true>(fi, d);
            sums16<false>(gi, d + 3);
#pragma unroll
            for (int k = 0; k < 6; ++k) own[k] = keep_w[(KW_OWN + k) * STEP_THREADS];
            const A F[2] = {keep_w[KW_F * STEP_THREADS], keep_w[(KW_F + 1) * STEP_THREADS]};
            m.update(p, th, u, own, d, F, keep_w[KW_REL * STEP_THREADS], 1.0);
            const float res = m.change(th);
            conv = sizeof(R) == 4 ? res <= p.tol_f : (double)res <= p.tol;
            if (conv || its >= (unsigned)p.max_iter || !(res == res)) break;
            th = w_round(m.ths);
            u[0] = w_round(m.uu[0]);
            u[1] = w_round(m.uu[1]);
        }

        // ---- collision in type R, equilibria as increments over their co-moving form
        const TypedParams<R> &q = typed<R>(p);
        const A F[2] = {keep_w[KW_F * STEP_THREADS], keep_w[(KW_F + 1) * STEP_THREADS]}, M0 = keep_w[KW_M0 * STEP_THREADS];
        {
            R v[16];
            ld16(in, n, N, Q_F, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) fi[i] += v[i];
            ld16(in, n, N, Q_G, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) gi[i] += v[i];
        }
        const R rho = w_round(m.rho), u_x = w_round(m.uu[0]), u_y = w_round(m.uu[1]);
        const R uhx = w_round(m.uh[0]), uhy = w_round(m.uh[1]), E = w_round(m.E), Pg = w_round(m.P);
        const R fx = w_round(F[0]), fy = w_round(F[1]), m0 = w_round(M0), dt = q.dt, om = q.omega;
        const A sA = w_sqrt(th);
        const R s = w_round(sA), is = R(1) / s, sst = sqrt_(w_round(m.ths));
        const R ds = fdiv_(m.dth, (sst + s) * s);                    // (s* - s)/s
        const R dux = w_round(m.du[0]) * is, duy = w_round(m.du[1]) * is;
        const R irh = R(1) / rho, ihP = R(1) / (R(2) * Pg);          // 1/rho, 1/(2P)
        const R shx = fx * dt * irh * is, shy = fy * dt * irh * is;  // du of the force
        R Dx[4][4], Dy[4][4], h[Q16], eqi[Q16], fo[Q16];
        axis_inc<R>(L, ds, dux, Dx);                                  // lambda* -> lambda
        axis_inc<R>(L, ds, duy, Dy);
#pragma unroll
        for (int i = 0; i < Q16; ++i) h[i] = rho * (L.w[i & 3] * L.w[i >> 2]);
        apply_inc<R>(Dx, Dy, h, eqi);
        {
            R Ex[4][4], Ey[4][4], shi[Q16];
            axis_inc<R>(L, ds, dux + shx, Ex);                        // lambda* + du -> lambda
            axis_inc<R>(L, ds, duy + shy, Ey);
            apply_inc<R>(Ex, Ey, h, shi);
#pragma unroll
            for (int i = 0; i < Q16; ++i) fo[i] = fi[i] + om * ((h[i] - fi[i]) + eqi[i]) + (shi[i] - eqi[i]);
        }
        bad = !(eqi[0] - eqi[0] == R(0));
        // Collision keeps the mass and adds F dt to the momentum: sum_i f_out = rho and
        // sum_i f_out (v_i - u) = rho (u* - u) + F dt exactly.  The stored values are made to
        // carry both (their sums are compared with the exact ones; the mass defect, which the
        // rounded weights and products would otherwise add every step in the same direction,
        // is spread by W_i, the momentum defect by W_i s c_i / theta, which has no mass).
        // Zero in exact arithmetic.
        A sm[3], jex[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) jex[a] = w_add(w_mul(m.rho, m.du[a]), w_mul(F[a], wide_dt<A>(p)));
        sums16<true>(fo, sm);
        const R fdef = w_round(w_sub(m.rho, sm[0]));
        // W_i s c_i J / theta = W_i c_i J / s (sum_i W_i c_i^2 = T_L = 1)
        const R jxdef = w_round(w_sub(jex[0], w_mul(sA, sm[1]))) * is;
        const R jydef = w_round(w_sub(jex[1], w_mul(sA, sm[2]))) * is;
#pragma unroll
        for (int i = 0; i < Q16; ++i)
            fo[i] += (L.w[i & 3] * L.w[i >> 2]) * (fdef + jxdef * L.c[i & 3] + jydef * L.c[i >> 2]);
        // what the stored values still miss (below their rounding) is kept beside them
        R mlo = R(0), jxlo = R(0), jylo = R(0);
        if constexpr (sizeof(R) == 4) {
            sums16<true>(fo, sm);
            mlo = w_round(w_sub(m.rho, sm[0]));
            jxlo = w_round(w_sub(jex[0], w_mul(sA, sm[1])));
            jylo = w_round(w_sub(jex[1], w_mul(sA, sm[2])));
        }
        st16(out, n, N, Q_F, fo);

        const R Prh = Pg * irh, k2 = dt * rho * ihP;            // P/rho, dt rho/(2P)
        const R H = E + Prh;
        const R Ixx = R(2) * uhx * fx + dt * fx * fx * E * ihP;
        const R Ixy = uhx * fy + fx * uhy + dt * fx * fy * E * ihP;
        const R Iyy = R(2) * uhy * fy + dt * fy * fy * E * ihP;
        const R Mx = (R(2) * k2) * (fx * H - (Ixx * u_x + Ixy * u_y));
        const R My = (R(2) * k2) * (fy * H - (Ixy * u_x + Iyy * u_y));
        const R Nxx = rho + k2 * Ixx;
        const R Nxy = k2 * Ixy;
        const R Nyy = rho + k2 * Iyy;
        const R phi = R(2) * (uhx * fx + uhy * fy);
        const R rhP = rho * ihP;                                // rho/(2P)
#pragma unroll
        for (int i = 0; i < Q16; ++i) {
            const R cx = L.c[i & 3], cy = L.c[i >> 2], W = L.w[i & 3] * L.w[i >> 2];
            const R vx = sst * cx + u_x, vy = sst * cy + u_y;
            const R Axx = vx * vx - Prh - u_x * u_x;
            const R Axy = vx * vy - u_x * u_y;
            const R Ayy = vy * vy - Prh - u_y * u_y;
            const R geq = W * (R(2) * rho * E + Mx * (vx - u_x) + My * (vy - u_y) + Nxx * Axx +
                               R(2) * Nxy * Axy + Nyy * Ayy);
            const R uc = u_x * cx + u_y * cy;
            const R gc = m0 * W * (R(1) + rhP * (uc * uc) - rhP * (vx * vx + vy * vy) + R(1));
            h[i] = om * geq + dt * (gc + W * phi);
        }
        R ginc[Q16];
        apply_inc<R>(Dx, Dy, h, ginc);
        bad = bad || !(ginc[0] - ginc[0] == R(0));
        // energy: sum_i g_out = sum_i g~ + dt (M_0 + 2 uhat . F) exactly (the heat-flux
        // correction sums to M_0, the force work to 2 uhat . F); the same defect spreading
        const A work = w_add(w_mul(m.uh[0], F[0]), w_mul(m.uh[1], F[1]));
        const A g_tot = w_add(m.gs, w_mul(w_add(M0, w_mul(work, R(2))), wide_dt<A>(p)));
#pragma unroll
        for (int i = 0; i < Q16; ++i) fo[i] = gi[i] - om * gi[i] + (h[i] + ginc[i]);
        sums16<false>(fo, sm);
        const R gdef = w_round(w_sub(g_tot, sm[0]));
#pragma unroll
        for (int i = 0; i < Q16; ++i) fo[i] += gdef * (L.w[i & 3] * L.w[i >> 2]);
        R glo = R(0);
        if constexpr (sizeof(R) == 4) {
            sums16<false>(fo, sm);
            glo = w_round(w_sub(g_tot, sm[0]));
        }
        st16(out, n, N, Q_G, fo);
        const R T = w_round(m.T);
        st4(out, n, N, Q_TH, th, u[0], u[1], rho);
        st4(out, n, N, Q_T, T, uhx, uhy, mlo);
        st4(out, n, N, Q_JXLO, jxlo, jylo, glo, R(0));
        floored = w_double(m.pr) < p.p_floor;
        bad = bad || !(rho - rho == R(0)) || !(T - T == R(0));
    }
    add_counts(counts, stats, its, nreg, npair, !conv, false, floored, bad);
}

// Output fields: rho, uhat, T, p in FP64.
template <typename R>
__global__ void k_q16_moments(DevParams p, const R *__restrict__ st, double *rho, double *ux,
                              double *uy, double *T, double *pr)
{
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const double r = (double)REC16(st, n, Q_RHO), t = (double)REC16(st, n, Q_T);
    if (rho) rho[n] = r;
    if (ux) ux[n] = (double)REC16(st, n, Q_UHX);
    if (uy) uy[n] = (double)REC16(st, n, Q_UHY);
    if (T) T[n] = t;
    if (pr) pr[n] = pressure_d(p, r, t);
}

// Conservation sums, stage 1: per-block compensated partials of
// {rho, rho uhat_x, rho uhat_y, sum_i g_i / 2} (stage 2 is k_conserve2).
template <typename R>
__global__ void k_q16_conserve1(DevParams p, const R *__restrict__ st, double *part)
{
    const long long N = p.N;
    double s[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0};
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        const double r = (double)REC16(st, n, Q_RHO);
        double eg = (double)REC16(st, n, Q_GLO);
        for (int i = 0; i < Q16; ++i) eg += (double)REC16(st, n, Q_G + i);
        const double v[4] = {r, r * (double)REC16(st, n, Q_UHX), r * (double)REC16(st, n, Q_UHY), 0.5 * eg};
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

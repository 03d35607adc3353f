// pond_init.cuh -- initial states: the co-moving equilibrium of host-given (rho, u, T) on
// each lattice (Eq. geq with the interface energy kappa |grad rho|^2 / 2 in the total
// energy).  Bound by the FP64 pipe when computed in FP64 (GB300 runs it at 1/64 of the FP32
// rate), so the FP32 form computes in float-float from the fields split once; and v^2 is a
// sum over the axes, so g_i = W_i (G + b_x(c_x) + b_y(c_y)) with b_a(c) = rho (s c + u_a)^2
// and G = rho (2 e - D P/rho) + kappa |grad rho|^2, with the gradient by differences of
// lines.  Measured (mixed, us): 2048 x 1024 D2Q9 500 -> 157, 1024 x 512 D2Q16 202 -> 45,
// 96 x 96 x 64 D3Q27 895 -> 100.
#pragma once

#include "pond_q16.cuh"
#include "pond_q27.cuh"

namespace pond {

// Thermodynamic state of a node in the wide type.
template <typename R, int D>
struct InitNode {
    using A = typename Wide<R>::type;
    A r, s, G, b[D][4];   // rho, sqrt(theta), and the parts of g (see above)
    R th, t;
    // rho, T, u in FP64; g2 = |grad rho|^2; inv_TL = 1 / T_L; c = the velocities along an axis
    template <int Q>
    __device__ __forceinline__ void set(const DevParams &p, double rho, double T, const double (&u)[D], A g2,
                                        R inv_TL, const A (&c)[Q])
    {
        r = w_const<A>(rho);
        const A tw = w_const<A>(T);
        const A pr = w_pressure(p, r, tw), fl = wide_p_floor<A>(p);
        const A P = w_less(fl, pr) ? pr : fl;
        const A theta = w_mul(w_mul(P, w_rcp(r)), inv_TL);
        s = w_sqrt(theta);
        const A e = w_sub(w_mul(tw, wide_param<A>(p.cv, p.ff_cv)), w_mul(r, wide_param<A>(p.a, p.ff_a)));
        G = w_add(w_sub(w_mul(w_mul(r, e), R(2)), w_mul(P, R(D))), w_mul(g2, wide_param<A>(p.kappa, p.ff_kap)));
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const A ua = w_const<A>(u[a]);
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                const A v = w_add(w_mul(s, c[k]), ua);
                b[a][k] = w_mul(r, w_mul(v, v));
            }
        }
        th = w_round(theta);
        t = (R)T;
    }
};

__device__ __forceinline__ void check_init(const DevParams &p, double r, double t, DevStats *stats)
{
    if (!(r > 0.0) || !(p.b * r < 1.0) || !(t > 0.0)) atomicAdd(&stats->bad_init, 1ull);
}

// |grad rho|^2 of a node by the isotropic D2Q9 stencil (zero without a Korteweg term)
template <typename A>
__device__ __forceinline__ A grad2_2d(const DevParams &p, const double *__restrict__ rho, int X, int Y)
{
    if (p.kappa == 0.0) return w_const<A>(0.0);
    double D[3], L[3];   // per row: rho(+1) - rho(-1); rho(-1) + 4 rho(0) + rho(+1)
#pragma unroll
    for (int y = 0; y < 3; ++y) {
        const long long row = (long long)bc_wrap(Y + y - 1, p.ny, p.bcy) * p.nx;
        const double a = rho[row + bc_wrap(X - 1, p.nx, p.bcx)], c = rho[row + bc_wrap(X + 1, p.nx, p.bcx)];
        D[y] = c - a;
        L[y] = (a + c) + 4.0 * rho[row + X];
    }
    const A g = w_const<A>(1.0 / 12.0);
    const A gx = w_mul(w_const<A>((D[0] + D[2]) + 4.0 * D[1]), g), gy = w_mul(w_const<A>(L[2] - L[0]), g);
    return w_add(w_mul(gx, gx), w_mul(gy, gy));
}

template <typename R>
__global__ void k_init(DevParams p, const double *__restrict__ rho, const double *__restrict__ ux,
                       const double *__restrict__ uy, const double *__restrict__ T,
                       R *__restrict__ st, DevStats *stats)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const double r = rho[n], t = T[n], u[2] = {ux[n], uy[n]};
    check_init(p, r, t, stats);
    const A c[3] = {w_wide(R(-1)), w_wide(R(0)), w_wide(R(1))};
    InitNode<R, 2> q;
    q.set(p, r, t, u, grad2_2d<A>(p, rho, (int)(n % p.nx), (int)(n / p.nx)), R(3), c);
    R rec[SL];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const A w = w_const<A>(w1d(i % 3) * w1d(i / 3));
        rec[P_F + i] = w_round(w_mul(q.r, w));
        rec[P_G + i] = w_round(w_mul(w_add(q.G, w_add(q.b[0][i % 3], q.b[1][i / 3])), w));
    }
    rec[P_TH] = q.th;
    rec[P_UX] = rec[P_UHX] = (R)u[0];
    rec[P_UY] = rec[P_UHY] = (R)u[1];
    rec[P_RHO] = w_round(q.r);
    rec[P_T] = q.t;
    rec[P_SQ] = rec[P_F4LO] = rec[P_G4LO] = rec[P_JXLO] = rec[P_JYLO] = rec[30] = rec[31] = R(0);
    store_chunks<SL>(st, (size_t)n, (size_t)p.N, rec);
}

// C1 of the D2Q16 lattice in the wide type
__device__ __forceinline__ void wide_c16(ffv (&c)[4])
{
    const ffv co = q16_co(), ci = q16_ci();
    c[0] = ff_neg(co); c[1] = ff_neg(ci); c[2] = ci; c[3] = co;
}
__device__ __forceinline__ void wide_c16(double (&c)[4])
{
    const Lat16<double> L = make_lat16<double>();
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = L.c[k];
}

template <typename R>
__global__ void k_q16_init(DevParams p, const double *__restrict__ rho, const double *__restrict__ ux,
                           const double *__restrict__ uy, const double *__restrict__ T,
                           R *__restrict__ st, DevStats *stats)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const double r = rho[n], t = T[n], u[2] = {ux[n], uy[n]};
    check_init(p, r, t, stats);
    const Lat16<double> L = make_lat16<double>();   // (its weights are constants)
    A c[4];
    wide_c16(c);
    InitNode<R, 2> q;
    q.set(p, r, t, u, grad2_2d<A>(p, rho, (int)(n % p.nx), (int)(n / p.nx)), R(1), c);
    R rec[SLQ];
#pragma unroll
    for (int i = 0; i < Q16; ++i) {
        const A w = w_const<A>(L.w[i & 3] * L.w[i >> 2]);
        rec[Q_F + i] = w_round(w_mul(q.r, w));
        rec[Q_G + i] = w_round(w_mul(w_add(q.G, w_add(q.b[0][i & 3], q.b[1][i >> 2])), w));
    }
    rec[Q_TH] = q.th;
    rec[Q_UX] = rec[Q_UHX] = (R)u[0];
    rec[Q_UY] = rec[Q_UHY] = (R)u[1];
    rec[Q_RHO] = w_round(q.r);
    rec[Q_T] = q.t;
#pragma unroll
    for (int k = Q_MLO; k < SLQ; ++k) rec[k] = R(0);
    store_chunks<SLQ>(st, (size_t)n, (size_t)p.N, rec);
}

template <typename R>
__global__ void k_q27_init(DevParams p, Grid3 g3, const double *__restrict__ rho, const double *__restrict__ ux,
                           const double *__restrict__ uy, const double *__restrict__ uz,
                           const double *__restrict__ T, R *__restrict__ st, DevStats *stats)
{
    using A = typename Wide<R>::type;
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const double r = rho[n], t = T[n], u[3] = {ux[n], uy[n], uz[n]};
    check_init(p, r, t, stats);
    A g2 = w_const<A>(0.0);
    if (p.kappa != 0.0) {
        const Near27 nb(p, g3, n);
        const Diff3<double> dr = diff3<double>([&](int z, int y, int k) { return rho[nb.at(z, y, k)]; });
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const A g = w_mul(w_const<A>(dr.d[a]), w_const<A>(1.0 / 72.0));
            g2 = w_add(g2, w_mul(g, g));
        }
    }
    const A c[3] = {w_wide(R(-1)), w_wide(R(0)), w_wide(R(1))};
    InitNode<R, 3> q;
    q.set(p, r, t, u, g2, R(3), c);
    R rec[SL27];
#pragma unroll
    for (int z = 0; z < 3; ++z)
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const A gyz = w_add(q.G, w_add(q.b[1][y], q.b[2][z]));
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const int i = 9 * z + 3 * y + x;
                const A w = w_const<A>(w27(i));
                rec[R_F + i] = w_round(w_mul(q.r, w));
                rec[R_G + i] = w_round(w_mul(w_add(gyz, q.b[0][x]), w));
            }
        }
    rec[R_TH] = q.th;
#pragma unroll
    for (int a = 0; a < 3; ++a) rec[R_UX + a] = rec[R_UHX + a] = (R)u[a];
    rec[R_RHO] = w_round(q.r);
    rec[R_T] = q.t;
#pragma unroll
    for (int k = R_MLO; k < SL27; ++k) rec[k] = R(0);
    store_chunks<SL27>(st, (size_t)n, (size_t)p.N, rec);
}

}  // namespace pond

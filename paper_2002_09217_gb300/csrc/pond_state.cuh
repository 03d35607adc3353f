// pond_state.cuh -- exchange of a context's state with the host as FP64 planes, on the
// device: the records are packed into (unpacked from) a few planes at a time in the
// context's staging buffer, so that the host only copies.  Bound by the host copies; the
// kernels move about 2 x 8 bytes a value.  (Transposing the records on the host took most
// of a call: resuming, advancing by two steps and saving 300 x 200 FP64 nodes 5.45 -> 2.31
// ms, one step of 900 x 700 138 -> 15 ms against both that and the earlier step kernel.)
#pragma once

#include "pond_q16.cuh"
#include "pond_q27.cuh"

namespace pond {

// Planes of each lattice's exchanged state, their record offsets, and how the FP32 form's
// kept remainders are exchanged: on D2Q9 with the rest populations, on the others folded
// into the populations as W_i (m + c_i . J / (s T_L)) on f and W_i G on g.
struct StateD2Q9 {
    static constexpr int planes = NPL, q = 9, values = SL, dims = 2;
    __device__ static int off(int p) { return rec_off(p); }
};
struct StateD2Q16 {
    static constexpr int planes = NP16, q = Q16, values = SLQ, dims = 2;
    static constexpr int mlo = Q_MLO, jlo = Q_JXLO, glo = Q_GLO, th = Q_TH;
    __device__ static int off(int p) { return p; }
    // weight of population i and its velocity along axis a (the host's closed forms)
    __device__ static double c1(int j)
    {
        const double s6 = sqrt(6.0), ci = sqrt(3.0 - s6), co = sqrt(3.0 + s6);
        return j == 0 ? -co : (j == 1 ? -ci : (j == 2 ? ci : co));
    }
    __device__ static double w1(int j)
    {
        const double s6 = sqrt(6.0);
        return (j == 0 || j == 3) ? (3.0 - s6) / 12.0 : (3.0 + s6) / 12.0;
    }
    __device__ static double c(int i, int a) { return c1(a == 0 ? i & 3 : i >> 2); }
    __device__ static double w(int i) { return w1(i & 3) * w1(i >> 2); }
    static constexpr double TL = 1.0;
};
struct StateD3Q27 {
    static constexpr int planes = NP27, q = Q27, values = SL27, dims = 3;
    static constexpr int mlo = R_MLO, jlo = R_JLO, glo = R_GLO, th = R_TH;
    __device__ static int off(int p) { return rec27_off(p); }
    __device__ static double c(int i, int a) { return (double)((a == 0 ? i % 3 : (a == 1 ? (i / 3) % 3 : i / 9)) - 1); }
    __device__ static double w(int i) { return w27(i); }
    static constexpr double TL = 1.0 / 3.0;
};

// Planes first .. first + count - 1 of the state into out (plane-major).
template <typename R, typename S>
__global__ void k_state_out(const R *__restrict__ st, size_t N, int first, int count, double *__restrict__ out)
{
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    for (int k = 0; k < count; ++k) {
        const int p = first + k;
        double v = (double)st[rec_at(st, n, S::off(p), N)];
        if constexpr (S::q == 9) {
            if (p == P_F + 4) v += (double)st[rec_at(st, n, P_F4LO, N)];
            if (p == P_G + 4) v += (double)st[rec_at(st, n, P_G4LO, N)];
        } else if (sizeof(R) == 4 && p < 2 * S::q) {
            const int i = p % S::q;
            if (p < S::q) {
                const double s = sqrt((double)st[rec_at(st, n, S::th, N)]);
                double cj = 0.0;
                for (int a = 0; a < S::dims; ++a) cj += S::c(i, a) * (double)st[rec_at(st, n, S::jlo + a, N)];
                v += S::w(i) * ((double)st[rec_at(st, n, S::mlo, N)] + cj / (s * S::TL));
            } else {
                v += S::w(i) * (double)st[rec_at(st, n, S::glo, N)];
            }
        }
        out[(size_t)k * N + n] = v;
    }
}

// The reverse, from planes first .. first + count - 1 (in increasing order of first).  acc:
// FP64 sums of what the FP32 populations leave out, for the D2Q16 and D3Q27 remainders:
// mass, momentum / s (dims), energy; started by first = 0, stored by k_state_finish.
template <typename R, typename S>
__global__ void k_state_in(const double *__restrict__ in, size_t N, int first, int count, R *__restrict__ st,
                           double *__restrict__ acc)
{
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    constexpr bool fold = S::q != 9 && sizeof(R) == 4;
    double sum[S::dims + 2];
    if (first == 0)
        for (int o = S::q == 9 ? P_SQ : 2 * S::q + 1 + S::dims; o < S::values; ++o) st[rec_at(st, n, o, N)] = R(0);
    if constexpr (fold)
        for (int a = 0; a < S::dims + 2; ++a) sum[a] = first == 0 ? 0.0 : acc[(size_t)a * N + n];
    for (int k = 0; k < count; ++k) {
        const int p = first + k;
        const double v = in[(size_t)k * N + n];
        const R r = (R)v;
        st[rec_at(st, n, S::off(p), N)] = r;
        if constexpr (S::q == 9) {
            // the rest populations keep the part below their float as the low word
            if (sizeof(R) == 4 && (p == P_F + 4 || p == P_G + 4))
                st[rec_at(st, n, p == P_F + 4 ? P_F4LO : P_G4LO, N)] = (R)(v - (double)r);
        } else if constexpr (fold) {
            if (p < S::q) {
                const double rf = v - (double)r;
                sum[0] += rf;
                for (int a = 0; a < S::dims; ++a) sum[1 + a] = __dadd_rn(sum[1 + a], __dmul_rn(rf, S::c(p, a)));
            } else if (p < 2 * S::q) {
                sum[1 + S::dims] += v - (double)r;
            }
        }
    }
    if constexpr (fold)
        for (int a = 0; a < S::dims + 2; ++a) acc[(size_t)a * N + n] = sum[a];
}

template <typename S>
__global__ void k_state_finish(size_t N, float *__restrict__ st, const double *__restrict__ acc)
{
    const size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const double s = sqrt((double)st[rec_at(st, n, S::th, N)]);
    st[rec_at(st, n, S::mlo, N)] = (float)acc[n];
    for (int a = 0; a < S::dims; ++a) st[rec_at(st, n, S::jlo + a, N)] = (float)(s * acc[(size_t)(1 + a) * N + n]);
    st[rec_at(st, n, S::glo, N)] = (float)acc[(size_t)(1 + S::dims) * N + n];
}

}  // namespace pond

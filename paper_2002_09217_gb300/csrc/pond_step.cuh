// pond_step.cuh -- the fused time-step kernel of the PonD van der Waals model (sm_103a).
//
// One launch per time step, one thread per node (nine lanes on small grids), a block owns a
// tile of nodes (step_shape).  Per block:
//   staging  every record of the tile and a halo of HALO = 2 nodes is read once from
//            global memory, its populations are carried into one gauge common to the tile
//            (SM "Transfer matrix": G = M_lambda'^-1 M_lambda) and left in shared memory,
//            one slot per unwrapped coordinate, so that periodic and zero-gradient
//            boundaries need no special case.
//   phase 0  non-local terms from the previous step's rho and T: the Korteweg stress K and
//            the heat flux q once per node of the tile and its ring, then F = -div K and
//            M_0 = 2 div q per node (Eq. korteweg, Eq. gtilde).
//   phase 1  frame search: each thread streams its node's 18 populations, takes the
//            moments, inverts e -> T, evaluates the EoS and the residual (FP64 in the FP64
//            form, float-float in the mixed form) until its own gauge has converged.
//   phase 2  BGK collision with the force source, heat-flux correction and forced g
//            equilibrium; the rest population takes the exact remainder of mass and
//            energy, and what storage rounding takes from the conserved sums is kept
//            beside the record.
//
// Streaming as one contraction.  The transfer map is linear, composes exactly
// (G_(n->lambda) = G_(b->lambda) G_(n->b)) and is a product over the axes, and so are the
// cubic Lagrange weights of a departure point.  With the stencil nodes already in the
// tile's common gauge b, the streamed population of direction (k, l) is
//   f~_(k,l) = sum_cy sum_n (wy[l][cy] Ly[l][n]) sum_cx sum_m (wx[k][cx] Lx[k][m]) f^b_(m,n)(cx, cy)
// (L = row of G_(b->lambda) along one axis, w = Lagrange weights): an x pass of 5 rows x 3 n
// x 3 k and a y pass, 675 multiply-adds a population family over each component's own four
// columns (FP64) and 810 over five (FP32), where carrying each of the 25 stencil nodes into
// the arrival gauge and spreading it over nine directions took about 2,700.  The tile is 128
// nodes because the halo's share of the staging falls with its size (1.9 staged nodes a
// node; 6.3 with 4 x 4 nodes and a halo of 3).
// Measured (five steps of the 2048 x 1024 shock-droplet interaction with init and read-out,
// mixed): 17.7 -> 3.90 ms, 720 us a step; two FP64 steps of a 509 x 387 droplet 22.8 ->
// 5.49 ms, 2.69 ms a step.  The mixed form is bound by instruction fetch and issue (issue 52 %
// active, FMA pipe 48 %, 1.1 warps per issue waiting for instructions), the FP64 form by the
// FP64 pipe (90 % busy); DRAM is 14 % busy.
//
// Accuracy.  A tile whose thetas differ holds the carried populations themselves in the
// gauge of geometric-mean theta and mean velocity of its hottest and coldest nodes, by
// product-form rows of the map.  Populations carried into a colder gauge are amplified (by
// (theta_b / theta) per axis for the outermost of three velocities, more for four), those
// carried into a hotter one cancel; the middle gauge splits that between the two maps.  (In
// a tile whose velocities spread it is the middle of those, see SMOOTH_SPREAD.)  On
// a 0.8 T_cr interface the worst error of a single population in FP32 is 2e-7 (D3Q27) and
// 7e-8 (D2Q16), no more than carrying each node straight into the arrival gauge; the
// hottest gauge left 3e-5 on D2Q16, the coldest 1e-6.
// The FP32 stream accumulates differences to the node's own slot, so that equal gauges and
// populations give exactly zero, rounding is proportional to local differences and not to
// the populations, and it does not accumulate as a bias.  FP32 tiles of nearly equal theta
// hold, moreover, differences to the populations of the tile's hottest node in its gauge,
// in increment form (the map as I + E with E = 0 for equal gauges), so that weak waves are
// not rounded to the populations' ulp; across an interface that form would cancel, as it
// would across a velocity jump (SMOOTH_SPREAD).
#pragma once

#include "pond_kernels.cuh"

namespace pond {

constexpr int STEP_THREADS = 128;   // threads per block
constexpr int STEP_NB = 128;        // nodes per block, one thread per node
constexpr int SPLIT_NB = 12;        // nodes per block, nine lanes per node (three nodes per warp)
constexpr int HALO = 2;       // staged halo: stencil reach for |v| dt < 1, and of the non-local terms
constexpr int HALO_FAR = 3;   // and for |v| dt < 2 (D2Q9, FP64)
// Largest side of a node's stencil region (the union of its 9 directions' 4x4 stencils)
// that the general stream handles as a region; wider ones take the per-pair stream.
constexpr int REGION_MAX = 8;
// FP32: tiles whose smallest theta is above this share of the largest are staged in
// increment form over the hottest node's populations, others as carried populations.  A
// weak wave (theta within 1e-3) needs the former; at a liquid-vapour interface (a factor of
// 4 to 6) the increment form left 6e-6 on single populations in three dimensions, the
// direct form 1.7e-7.
constexpr float SMOOTH_TILE = 0.9f;
// Velocities.  Carried populations are amplified by the velocity between a node's gauge and
// the tile's, in the increment form more than in the other.  Emulated in FP32 at uniform
// theta, a node U sqrt(theta) from the tile's gauge gets back single populations with an error
// of (D2Q9, D3Q27) 9e-8, 1e-7 in increment form at U = 0.4 and 7e-5, 3e-3 at 2; of 1.5e-7,
// 2e-7 in direct form at 0.5, 4e-7, 9e-7 at 1 and 5e-6, 3e-5 at 1.5.  So a tile in which a
// node moves faster than SMOOTH_SPREAD sqrt(theta) in the tile's gauge is staged in direct
// form around the middle of its velocities, and one in which a node then still moves faster
// than FAR_SPEED sqrt(theta) takes the general stream, which carries each node straight into
// the arrival gauge.  theta is the tile's hottest: at interfaces whose coldest nodes are at
// the pressure floor, the gauge's own theta_b is a small part of it, and tiles of ordinary
// shocks and droplets would change their gauge for nothing (their times are the same either
// way: 96 x 96 x 64 sphere 2829 us a step against theta_b, 2826 against the hottest).
constexpr float SMOOTH_SPREAD = 0.4f;
constexpr float FAR_SPEED = 1.0f;
constexpr int BEST = 8;   // uint4 of shared memory in which a block agrees on its gauge
// Mixed form: a frame-search residual below this multiple of tol that no longer halves is
// taken as the FP32 rounding floor (the EoS cancels up to ~200x inside interfaces).
constexpr float STALL_TOL_FACTOR = 16.0f;
// Resident blocks per SM the register budget is sized for: FP32 with one thread a node took
// 798, 737 and 850 us a step (2048 x 1024) with four, three and two.
#define STEP_MIN_BLOCKS(R) (sizeof(R) == 8 ? 2 : 3)
#define SPLIT_MIN_BLOCKS(R) 2

// Values per staged slot: the 18 carried populations, padded so that slots start on
// distinct banks (FP32: 16-byte loads, 20 words; FP64: 19 values).
template <typename R> struct Slot;
template <> struct Slot<float> { static constexpr int stride = 20; };
template <> struct Slot<double> { static constexpr int stride = 19; };
// place of population i of family fam (0 f, 1 g): side by side in FP32
template <typename R> __host__ __device__ constexpr int slot_at(int fam, int i) { return sizeof(R) == 4 ? 2 * i + fam : 9 * fam + i; }
constexpr int AUXW = 4;   // rho, T, p, p/rho of a staged node
constexpr int SPLIT_WORDS = SL + 9 * 18;   // nine lanes per node: the own record, the lanes' partials
constexpr int KQW = 5;    // K_xx, K_xy, K_yy, q_x, q_y of a node of the tile and its ring

__host__ __device__ constexpr int step_slots(int tx, int ty, int halo = HALO) { return (tx + 2 * halo) * (ty + 2 * halo); }

// What a thread of the one-thread-per-node form keeps in shared memory across the stream
// instead of in registers (a column of KEEP values; the contraction's weights then fit 168
// registers, three blocks per SM, without recomputing them): the node's own sums (hi, lo),
// F, rho E_lambda, M_0, and the y weights and rows of the map.
enum : int { K_HI = 0, K_LO = 4, K_F = 8, K_REL = 10, K_M0 = 11, K_WY = 12, K_LY = 27, KEEP = 36 };

// Halo that a tile's shared memory holds.  FP64: the wider one where it costs no resident
// block (16 x 8 nodes: 205 instead of 179 KB of an SM's memory for two blocks; long tiles of
// 128 nodes would lose one).  FP32 tiles do without: carrying the populations into the tile's
// gauge rounds them once more, which at the velocities of such flows doubles the error of p
// (u = 2.6, -1.9 in a droplet: 1.9e-5 -> 3.5e-5), and asking every tile cost 2 % of a step.
__host__ __device__ constexpr int widest_halo(int tx, int ty, int elem_bytes)
{
    return elem_bytes == 8 && (tx * ty < STEP_NB || (tx >= 8 && ty >= 8)) ? HALO_FAR : HALO;
}

// Dynamic shared memory of one step block: slots' rho, T, p, p/rho; populations; K and q;
// then the threads' kept values, or with nine lanes per node the partials of the general
// stream and the own records.
__host__ __device__ constexpr size_t step_smem_bytes(int tx, int ty, bool split, int slot_values, int elem_bytes)
{
    return ((size_t)step_slots(tx, ty, widest_halo(tx, ty, elem_bytes)) * (AUXW + slot_values) + (size_t)(tx + 2) * (ty + 2) * KQW +
            (split ? (size_t)SPLIT_NB * SPLIT_WORDS : (size_t)STEP_THREADS * KEEP)) * elem_bytes;
}

// Work split (8: one thread per node, 16: nine lanes per node) and tile of the D2Q9 step on an
// nx x ny grid; D2Q16 has one split and shares the tile rule.  lanes, tile_x: the caller's
// choice, 0 = by size.
//
// Nine lanes.  A step of a small grid costs one block's serial time: one thread per node
// 14.4 us (mixed) and 395 us (FP64), whatever the grid; nine lanes per node less, until their
// blocks of 12 nodes need further turns on the SMs.  Mixed: while all of them are resident at
// once, two on each SM (us a step, thread / nine lanes: 128 x 4 13.9 / 10.9, 64 x 48 14.4 /
// 13.0, 64 x 64 14.5 / 20.1).  FP64: up to five an SM (128 x 4 377 / 105, 64 x 64 395 / 265,
// 90 x 90 396 / 376, 96 x 96 395 / 424).  FP64 grids take them also where the caller asks for
// 8: the eight lanes a node of earlier kernels took 242 us on small grids, a thread 396.
//
// Tile.  One thread per node: 16 x 8, no taller than the grid for grids of few rows, and no
// wider than the grid for those of few columns once there is more than one block an SM (us a
// step in 16 x 8 / narrower tiles: 4 x 20000 mixed 118 / 46; D2Q16 mixed 1 x 4096 78.7 / 50.7,
// 2 x 2048 51.0 / 44.8, but 4 x 1024, one turn in either, 44.6 / 47.7: a narrow tile stages
// more slots).  Nine lanes: 4 x 3 and alike (1 x 2048 mixed: 29.9 in 4 x 3, 12.1 in 1 x 12).
// Strips of up to four rows or columns take tiles of 32 or 64 nodes while that is at most one
// block an SM, because the serial time falls with the slots a block stages (mixed, tiles of
// 128 / 64 / 32 nodes: 1024 x 4 15.2 / 13.9 / 13.6, 4096 x 1 17.6 / 14.9 / 13.8, 4096 x 2 16.0
// / 13.8 / 13.6, 8192 x 1 17.7 / 14.7 / 14.3, 1600 x 3 14.7 / 13.6 / 13.7, 2400 x 4 15.0 / 13.9
// / 13.9, 2048 x 4 15.5 / 13.9 / 13.9 and as a shock tube 64 nodes 3 % ahead of 32; beyond
// one block an SM, 5000 x 4 16.0 / 18.1 / 22.5).  Grids of more rows and columns gain 1 to 4 %
// from small tiles (1024 x 8 14.6 / 14.0 / 14.1, 90 x 90 14.8 / 14.6 / 14.3) and keep 128:
// they are what batches hold, where the other members fill the GPU and the wider share of the
// halo counts (128 x 128, which nearly fills it by itself, 15.3 / 19.2 / 21.1).
struct StepShape {
    int lanes, tx, ty;
    long long blocks(int nx, int ny) const { return (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty); }
};
inline StepShape step_shape(bool d2q9, bool mixed, int nx, int ny, int lanes, int tile_x, int sms)
{
    if (d2q9 && (lanes != 8 || !mixed)) {
        StepShape s{16, tile_x, 0};
        if (!s.tx) s.tx = nx < 4 ? nx : (ny == 1 ? 12 : (ny == 2 || ny == 4 ? 6 : 4));
        else if (s.tx == 8) s.tx = 6;
        else if (s.tx == 16) s.tx = 12;
        s.ty = SPLIT_NB / s.tx;
        if (lanes == 16 || s.blocks(nx, ny) <= (long long)(mixed ? SPLIT_MIN_BLOCKS(float) : 5) * sms) return s;
    }
    if (tile_x) return {8, tile_x, STEP_NB / tile_x};
    auto fit = [&](int nodes, int tx, bool narrow) {
        while (tx < nodes && nodes / (2 * tx) >= ny) tx *= 2;
        StepShape s{8, tx, nodes / tx};
        while (s.tx > 1 && s.tx / 2 >= nx && (narrow || s.blocks(nx, ny) > sms)) s = {8, s.tx / 2, 2 * s.ty};
        return s;
    };
    if (d2q9 && (nx <= 4 || ny <= 4))
        for (int nodes = 32; nodes < STEP_NB; nodes *= 2) {
            const StepShape s = fit(nodes, 8, true);
            if (s.blocks(nx, ny) <= sms) return s;
        }
    return fit(STEP_NB, 16, false);
}

// Counters of one block, summed into the context's by its last instructions.
struct StepCounts {
    unsigned streams, region_nodes, pair_streams, nonconv, stalled, clamped, nonfinite, warp_streams, max_streams;
};

// 1-D transfer-map increment E = l_k(c_a + e) - l_k(c_a) for target index k (c = k-1),
// source offset e (in units of the target spacing s) and source index a (c_a = a-1).
template <typename R>
__device__ __forceinline__ R ell_inc(int k, int a, R e)
{
    R two_c = R(2 * (a - 1));
    if (k == 1) return -e * (two_c + e);
    if (k == 0) return R(0.5) * e * (two_c + e - R(1));
    return R(0.5) * e * (two_c + e + R(1));
}

// ell_inc for a target index k known only at run time: the same arithmetic, with the
// k = 0 / k = 2 forms joined through their sign
template <typename R>
__device__ __forceinline__ R ell_inc_rt(int k, int a, R e)
{
    const R base = R(2 * (a - 1)) + e;
    return k == 1 ? -e * base : R(0.5) * e * (base + R(k - 1));
}

// 1-D lattice weights W_-1, W_0, W_+1 = 1/6, 2/3, 1/6 as values of type R whose sum is
// exactly one: in FP32 the nearest floats to 1/6 and 2/3 sum to 1 + 3e-8, a bias that every
// collision would add to the mass and energy; W_+-1 = 1/6 rounded down and W_0 = 1 - 2 W_+-1
// (both exact floats) sum to one exactly.
template <typename R> __device__ __forceinline__ R wlat(int a);
template <> __device__ __forceinline__ float wlat<float>(int a)
{
    return a == 1 ? 0x1.555556p-1f : 0x1.555554p-3f;
}
template <> __device__ __forceinline__ double wlat<double>(int a)
{
    return a == 1 ? 1.0 - 2.0 * (1.0 / 6.0) : 1.0 / 6.0;
}

// Stencil weight W_i of the isotropic D2Q9 difference operators, as a constant of type R.
template <typename R>
__device__ __forceinline__ R wst(int ex, int ey)
{
    return (ex == 0 ? R(2.0 / 3.0) : R(1.0 / 6.0)) * (ey == 0 ? R(2.0 / 3.0) : R(1.0 / 6.0));
}

// A departure offset (in nodes) limited to +-2^20, NaN mapped to the lower bound: keeps
// stencil indices derived from it in int range whatever the gauge (fmax returns the
// non-NaN operand).
template <typename R>
__device__ __forceinline__ R clamp_offset(R d)
{
    return fmin(fmax(d, R(-1048576)), R(1048576));
}

// The cubic Lagrange basis function a_j(xi) on nodes 0..3 (SM "Reconstruction") for a
// run-time j: the three factors (xi - m), m != j, picked by selects.
template <typename R>
__device__ __forceinline__ R lag1_rt(int j, R xi)
{
    const R t0 = xi, t1 = xi - R(1), t2 = xi - R(2), t3 = xi - R(3);
    const R a = j == 0 ? t1 : t0;
    const R b = j <= 1 ? t2 : t1;
    const R c = j <= 2 ? t3 : t2;
    const R inv = j == 0 ? R(-1.0 / 6.0) : (j == 1 ? R(0.5) : (j == 2 ? R(-0.5) : R(1.0 / 6.0)));
    return a * b * c * inv;
}

// a[i] for a run-time i without local-memory indexing (unrolled selects).
template <typename R, int K>
__device__ __forceinline__ R pick(const R (&a)[K], int i)
{
    R r = a[0];
#pragma unroll
    for (int j = 1; j < K; ++j) r = (i == j) ? a[j] : r;
    return r;
}

// a / b for operands of moderate range (transfer-map offsets, collision coefficients):
// the fast FP32 quotient, or a times the Newton reciprocal in FP64.
template <typename R> __device__ __forceinline__ R fdiv_(R a, R b);
template <> __device__ __forceinline__ float fdiv_(float a, float b) { return __fdividef(a, b); }
template <> __device__ __forceinline__ double fdiv_(double a, double b) { return a * rcp_d(b); }
template <typename R> __device__ __forceinline__ R frcp_(R b);
template <> __device__ __forceinline__ float frcp_(float b) { return __frcp_rn(b); }
template <> __device__ __forceinline__ double frcp_(double b) { return rcp_d(b); }

// Error-free sum of two values of type R (Knuth TwoSum).
template <typename R>
__device__ __forceinline__ void two_sum_(R a, R b, R &s, R &e)
{
    s = a + b;
    R bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Float-float ("double-word") arithmetic for the FP32 form's frame-search EoS: a value is
// an unevaluated pair hi + lo of floats.  Sums use Knuth's TwoSum, products the exact FMA
// product error (Dekker's TwoProduct with a fused multiply-add), each result renormalised
// with Dekker's Fast2Sum; relative error ~2^-44 per operation, far below the FP32 form's
// needs, on the FP32 pipes (GB300 runs FP64 at 1/64 of the FP32 rate).
struct __align__(8) ffv {
    float hi, lo;
};
__device__ __forceinline__ ffv ff_norm(float a, float b)   // |a| >= |b| or a == 0
{
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ ffv ff_pair(float a, float b)   // any a, b
{
    ffv r;
    two_sum_(a, b, r.hi, r.lo);
    return r;
}
__device__ __forceinline__ ffv ff_add(ffv a, ffv b)
{
    float s, e;
    two_sum_(a.hi, b.hi, s, e);
    return ff_norm(s, e + (a.lo + b.lo));
}
__device__ __forceinline__ ffv ff_add(ffv a, float b)
{
    float s, e;
    two_sum_(a.hi, b, s, e);
    return ff_norm(s, e + a.lo);
}
__device__ __forceinline__ ffv ff_neg(ffv a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ ffv ff_mul(ffv a, ffv b)
{
    const float p = __fmul_rn(a.hi, b.hi);   // never contracted into the sum below
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return ff_norm(p, e);
}
__device__ __forceinline__ ffv ff_mul(ffv a, float b)
{
    const float p = __fmul_rn(a.hi, b);
    float e = fmaf(a.hi, b, -p);
    e = fmaf(a.lo, b, e);
    return ff_norm(p, e);
}
// 1/a: the FP32 reciprocal and one Newton step r + r (1 - a r) with the residual in
// float-float (Newton doubles the ~24 correct bits)
__device__ __forceinline__ ffv ff_rcp(ffv a)
{
    const float r = __frcp_rn(a.hi);
    const ffv ar = ff_mul(a, r);
    const float res = (1.0f - ar.hi) - ar.lo;
    return ff_norm(r, r * res);
}

// Values 0..23 of node nd's record (f[9], g[9], theta, u_x, u_y, spare, rho, T).
__device__ __forceinline__ void load_rec24(const float *__restrict__ b, size_t nd, size_t N, float v[24])
{
    const float4 *q = reinterpret_cast<const float4 *>(b) + nd;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 t = __ldg(q + k * N);
        v[4 * k] = t.x; v[4 * k + 1] = t.y; v[4 * k + 2] = t.z; v[4 * k + 3] = t.w;
    }
}
__device__ __forceinline__ void load_rec24(const double *__restrict__ b, size_t nd, size_t N, double v[24])
{
    const double2 *q = reinterpret_cast<const double2 *>(b) + nd;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double2 t = __ldg(q + k * N);
        v[2 * k] = t.x; v[2 * k + 1] = t.y;
    }
}
// Four staged values from a 16-byte boundary.
__device__ __forceinline__ void lds4(const float *s, float (&o)[4])
{
    const float4 t = *reinterpret_cast<const float4 *>(s);
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void lds4(const double *s, double (&o)[4])
{
    const double2 a = reinterpret_cast<const double2 *>(s)[0], b = reinterpret_cast<const double2 *>(s)[1];
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}

// Contribution of stencil node `nd` to direction (jx, jy) of the arrival node, in the
// increment form.
//
// With the per-axis maps written as G = I + E (E = transfer increments, zero for equal
// gauges), [G (f_n - f_x) + (G - I) f_x]_(jx,jy) regroups exactly into
//   (f_n - f_x)_(jx,jy) + t_jy + sum_b Ey[b] (f_n(jx, b) + t_b),   t_b = sum_a Ex[a] f_n(a, b):
// the difference of the two nodes' populations plus increments that multiply the source
// values by the small E only, so the rounding stays relative to the differences and equal
// gauges still give f_n - f_x exactly.
template <typename R>
__device__ __forceinline__ R sel3(int k, R a0, R a1, R a2)
{
    return k == 0 ? a0 : (k == 1 ? a1 : a2);
}

// fxj, gxj: the arrival node's own populations of direction (jx, jy).  jx must be a
// compile-time constant after unrolling; jy may vary at run time (selects, no indexing).
template <typename R>
__device__ __forceinline__ void pair_inc(const R v[24], int jx, int jy, R th, R s, R inv_s, R ux,
                                         R uy, R fxj, R gxj, R &tf, R &tg)
{
    const R thn = v[P_TH];
    const R sn = v[P_SQ];
    // (s_n - s)/s: in FP32 without cancellation, in FP64 directly (its rounding, ~1e-16 of
    // s_n/s, stays far below what the result needs, and saves a reciprocal per pair)
    const R qm1 = sizeof(R) == 8 ? sn * inv_s - R(1) : fdiv_(thn - th, (sn + s) * s);
    const R wx = (v[P_UX] - ux) * inv_s;
    const R wy = (v[P_UY] - uy) * inv_s;
    R Ex[3], Ey[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Ex[a] = ell_inc<R>(jx, a, qm1 * R(a - 1) + wx);
        Ey[a] = ell_inc<R>(jy, a, qm1 * R(a - 1) + wy);
    }
    if constexpr (sizeof(R) == 8) {
        // FP64: the transfer applied directly, [G_n f_n]_(jx,jy) - f_x (its rounding is far
        // below what the FP64 form needs; the increment form is for FP32)
        R Gx[3], Gy[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Gx[a] = Ex[a] + (a == jx ? R(1) : R(0));
            Gy[a] = Ey[a];
        }
        R rf[3], rg[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            rf[b] = Gx[0] * v[P_F + 3 * b] + Gx[1] * v[P_F + 3 * b + 1] + Gx[2] * v[P_F + 3 * b + 2];
            rg[b] = Gx[0] * v[P_G + 3 * b] + Gx[1] * v[P_G + 3 * b + 1] + Gx[2] * v[P_G + 3 * b + 2];
        }
        // Gy = Ey + delta(b, jy): the delta picks row jy
        R sf = sel3(jy, rf[0], rf[1], rf[2]) - fxj, sg = sel3(jy, rg[0], rg[1], rg[2]) - gxj;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            sf += Gy[b] * rf[b];
            sg += Gy[b] * rg[b];
        }
        tf = sf;
        tg = sg;
        return;
    }
    R txf[3], txg[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        txf[b] = Ex[0] * v[P_F + 3 * b] + Ex[1] * v[P_F + 3 * b + 1] + Ex[2] * v[P_F + 3 * b + 2];
        txg[b] = Ex[0] * v[P_G + 3 * b] + Ex[1] * v[P_G + 3 * b + 1] + Ex[2] * v[P_G + 3 * b + 2];
    }
    R sf = (sel3(jy, v[P_F + jx], v[P_F + 3 + jx], v[P_F + 6 + jx]) - fxj) + sel3(jy, txf[0], txf[1], txf[2]);
    R sg = (sel3(jy, v[P_G + jx], v[P_G + 3 + jx], v[P_G + 6 + jx]) - gxj) + sel3(jy, txg[0], txg[1], txg[2]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        sf += Ey[b] * (v[P_F + 3 * b + jx] + txf[b]);
        sg += Ey[b] * (v[P_G + 3 * b + jx] + txg[b]);
    }
    tf = sf;
    tg = sg;
}

// One stencil node of a node's region carried into the arrival gauge for all nine
// directions of one population family, weighted and accumulated:
//   acc[(k, l)] += wx[k] wy[l] ([G_n f_n](k, l) - f_x(k, l))
// with G_n = (I + Ex) (x) (I + Ey) the separable transfer map from the stencil node's
// gauge into the arrival gauge (SM "Transfer matrix"), Ex[k][a] = l_k increments at the
// source velocities.  In FP32 the increment form (see pair_inc) keeps the rounding
// relative to the differences: (f_n - f_x)(k, l) + t(k, l) + sum_b Ey[l][b] (f_n(k, b) +
// t(k, b)), t(k, b) = sum_a Ex[k][a] f_n(a, b); in FP64 the map is applied directly.
// All indices are compile-time: each stencil node is transformed once for every
// direction whose stencil contains it.
template <typename R>
__device__ __forceinline__ void region_family(const R *v, const R *own, const R (&Ex)[3][3],
                                              const R (&Ey)[3][3], const R (&wx)[3], const R (&wy)[3],
                                              R (&acc)[9])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R t[3], u[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            t[b] = Ex[k][0] * v[3 * b] + Ex[k][1] * v[3 * b + 1] + Ex[k][2] * v[3 * b + 2];
            if constexpr (sizeof(R) == 8) t[b] += v[3 * b + k];
            u[b] = sizeof(R) == 8 ? t[b] : v[3 * b + k] + t[b];
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int i = 3 * l + k;
            R o = sizeof(R) == 8 ? t[l] - own[i] : (v[i] - own[i]) + t[l];
            o += Ey[l][0] * u[0] + Ey[l][1] * u[1] + Ey[l][2] * u[2];
            acc[i] += (wx[k] * wy[l]) * o;
        }
    }
}

// The double-well constants in the arithmetic type of a kernel.
template <typename R> __device__ __forceinline__ const R *typed_sp(const DevParams &p);
template <> __device__ __forceinline__ const float *typed_sp<float>(const DevParams &p) { return p.spf; }
template <> __device__ __forceinline__ const double *typed_sp<double>(const DevParams &p) { return p.sp; }

// Results of one corrector evaluation (moments, e -> T, EoS) of a node, in R.
template <typename R>
struct EosOut {
    R rho_hi, rho_lo;   // rho as a (hi, lo) pair
    R gs_hi, gs_lo;     // sum of the streamed g as a (hi, lo) pair (= 2 rho E)
    R uxs, uys;         // streamed velocity u* (the next gauge velocity)
    R uhx, uhy;         // actual fluid velocity uhat = u* + F dt / (2 rho)
    R E, T, P, pr;      // total energy per mass, temperature, floored and vdW pressure
    R ths;              // theta* = P / (rho T_L)
    R dth, dux, duy;    // theta* - theta, u* - u (the gauge change)
    R mx_hi, mx_lo, my_hi, my_lo;   // sum f~ c_x, sum f~ c_y as (hi, lo) pairs
};

// FP64 form: the streamed moments are the stored sums (hi + lo, rounded to FP64) plus the
// stream's increments (moments Eq.; SM "Thermodynamics": e = E - uhat^2/2 - E_lambda,
// T = (e + a rho)/C_v, p = rho R T/(1 - b rho) - a rho^2, theta = max(p, p_floor)/(rho T_L)).
__device__ __forceinline__ void eos_update(const DevParams &p, const double *bhi, const double *blo,
                                           const double *dsum, const double *nl, const double *lam,
                                           double sr, EosOut<double> &o)
{
    const double dt = p.dt;
    const double Fxd = nl[0], Fyd = nl[1], rEd = nl[2];
    const double thd = lam[0], uxd = lam[1], uyd = lam[2];
    const double rho = (bhi[0] + blo[0]) + dsum[0];
    const double irho = rcp_d(rho);
    const double mx = (bhi[1] + blo[1]) + dsum[1], my = (bhi[2] + blo[2]) + dsum[2];
    const double dux = sr * mx * irho;
    const double duy = sr * my * irho;
    o.mx_hi = mx; o.mx_lo = 0.0; o.my_hi = my; o.my_lo = 0.0;
    const double uxs = uxd + dux, uys = uyd + duy;
    const double uhx = uxs + 0.5 * Fxd * dt * irho, uhy = uys + 0.5 * Fyd * dt * irho;
    const double gs = (bhi[3] + blo[3]) + dsum[3];
    const double E = 0.5 * gs * irho;
    const double e = E - 0.5 * (uhx * uhx + uhy * uhy) - rEd * irho;
    const double T = p.isothermal ? p.T_iso : (e + p.a * rho) * p.pd.inv_cv;
    const double pr = p.eos_kind == 2
        ? rho * p.R * T * rcp_d(1.0 - p.b * rho) * exp(-p.a * rho * rcp_d(p.R * T))
        : (p.eos_kind == 3 ? p.sp[3] + well_pressure<double>(p.sp, rho)
                           : rho * p.R * T * rcp_d(1.0 - p.b * rho) - p.a * rho * rho);
    const double P = pr > p.p_floor ? pr : p.p_floor;
    const double ths = P * irho * 3.0;
    o.rho_hi = rho; o.rho_lo = 0.0; o.gs_hi = gs; o.gs_lo = 0.0;
    o.uxs = uxs; o.uys = uys; o.uhx = uhx; o.uhy = uhy;
    o.E = E; o.T = T; o.P = P; o.pr = pr; o.ths = ths;
    o.dth = ths - thd; o.dux = dux; o.duy = duy;
}

// FP32 form: the same formulas in float-float from the exact (hi, lo) stored sums and the
// FP32 increments; the results are rounded to FP32 once (the pairs of rho and sum g are
// kept for the collision's exact remainders).
__device__ __forceinline__ void eos_update(const DevParams &p, const float *bhi, const float *blo,
                                           const float *dsum, const float *nl, const float *lam,
                                           float sr, EosOut<float> &o)
{
    const float dt = p.pf.dt;
    const ffv a = {p.ff_a[0], p.ff_a[1]}, b = {p.ff_b[0], p.ff_b[1]};
    const ffv Rg = {p.ff_R[0], p.ff_R[1]}, icv = {p.ff_icv[0], p.ff_icv[1]};
    const ffv rho = ff_add(ff_pair(bhi[0], blo[0]), dsum[0]);
    const ffv irho = ff_rcp(rho);
    const ffv mx = ff_add(ff_pair(bhi[1], blo[1]), dsum[1]);
    const ffv my = ff_add(ff_pair(bhi[2], blo[2]), dsum[2]);
    const ffv dux = ff_mul(ff_mul(mx, irho), sr), duy = ff_mul(ff_mul(my, irho), sr);
    const ffv uxs = ff_add(dux, lam[1]), uys = ff_add(duy, lam[2]);
    const ffv uhx = ff_add(uxs, 0.5f * nl[0] * dt * irho.hi);
    const ffv uhy = ff_add(uys, 0.5f * nl[1] * dt * irho.hi);
    const ffv gs = ff_add(ff_pair(bhi[3], blo[3]), dsum[3]);
    const ffv E = ff_mul(ff_mul(gs, irho), 0.5f);
    const ffv kin = ff_mul(ff_add(ff_mul(uhx, uhx), ff_mul(uhy, uhy)), 0.5f);
    const ffv e = ff_add(ff_add(E, ff_neg(kin)), ff_neg(ff_mul(irho, nl[2])));
    const ffv T = p.isothermal ? ffv{p.ff_Tiso[0], p.ff_Tiso[1]} : ff_mul(ff_add(e, ff_mul(rho, a)), icv);
    const ffv den = ff_add(ff_neg(ff_mul(rho, b)), 1.0f);
    const ffv pre = ff_mul(ff_mul(ff_mul(rho, Rg), T), ff_rcp(den));
    // Dieterici: a product with no cancellation, so its exponential factor in FP32 (a few
    // ulps) is enough; van der Waals: the difference in float-float
    // double well: p0 (a float pair) plus a small polynomial part, which FP32 carries
    const ffv pr = p.eos_kind == 2
        ? ff_mul(pre, expf(-(p.pf.a * rho.hi) / (p.pf.R * T.hi)))
        : (p.eos_kind == 3 ? ff_add(ffv{p.ff_p0[0], p.ff_p0[1]}, well_pressure<float>(p.spf, rho.hi))
                           : ff_add(pre, ff_neg(ff_mul(ff_mul(rho, rho), a))));
    const bool floored = !(pr.hi > p.ff_pfl[0] || (pr.hi == p.ff_pfl[0] && pr.lo > p.ff_pfl[1]));
    const ffv P = floored ? ffv{p.ff_pfl[0], p.ff_pfl[1]} : pr;
    const ffv ths = ff_mul(ff_mul(P, irho), 3.0f);
    o.rho_hi = rho.hi; o.rho_lo = rho.lo; o.gs_hi = gs.hi; o.gs_lo = gs.lo;
    o.mx_hi = mx.hi; o.mx_lo = mx.lo; o.my_hi = my.hi; o.my_lo = my.lo;
    o.uxs = uxs.hi; o.uys = uys.hi; o.uhx = uhx.hi; o.uhy = uhy.hi;
    o.E = E.hi; o.T = T.hi; o.P = P.hi; o.pr = pr.hi; o.ths = ths.hi;
    o.dth = (ths.hi - lam[0]) + ths.lo;
    o.dux = dux.hi; o.duy = duy.hi;
}
// ---------------------------------------------------------------------------
// Wide arithmetic of the D2Q16 and D3Q27 steps: FP64 in the FP64 form, float-float in the
// FP32 form (GB300 runs an FP64 addition at the cost of 64 FP32 ones, a float-float addition
// takes about 12).
template <typename R> struct Wide;
template <> struct Wide<float> { using type = ffv; };
template <> struct Wide<double> { using type = double; };
__device__ __forceinline__ ffv w_add(float a, float b) { return ff_pair(a, b); }
__device__ __forceinline__ ffv w_add(ffv a, ffv b) { return ff_add(a, b); }
__device__ __forceinline__ ffv w_add(ffv a, float b) { return ff_add(a, b); }
__device__ __forceinline__ double w_add(double a, double b) { return a + b; }
__device__ __forceinline__ ffv w_sub(float a, float b) { return ff_pair(a, -b); }
__device__ __forceinline__ ffv w_sub(ffv a, ffv b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ double w_sub(double a, double b) { return a - b; }
__device__ __forceinline__ ffv w_mul(ffv a, ffv b) { return ff_mul(a, b); }
__device__ __forceinline__ ffv w_mul(ffv a, float b) { return ff_mul(a, b); }
__device__ __forceinline__ double w_mul(double a, double b) { return a * b; }
__device__ __forceinline__ float w_x4(float a) { return 4.0f * a; }
__device__ __forceinline__ ffv w_x4(ffv a) { return {4.0f * a.hi, 4.0f * a.lo}; }
__device__ __forceinline__ double w_x4(double a) { return 4.0 * a; }
__device__ __forceinline__ double w_double(ffv a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double w_double(double a) { return a; }
__device__ __forceinline__ float w_round(ffv a) { return a.hi; }   // (hi, lo) are kept normalised
__device__ __forceinline__ double w_round(double a) { return a; }
__device__ __forceinline__ ffv w_wide(float a) { return {a, 0.0f}; }
__device__ __forceinline__ double w_wide(double a) { return a; }
// a FP64 constant in the wide type
template <typename A> __device__ __forceinline__ A w_const(double x);
template <> __device__ __forceinline__ double w_const<double>(double x) { return x; }
template <> __device__ __forceinline__ ffv w_const<ffv>(double x)
{
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ ffv w_rcp(ffv a) { return ff_rcp(a); }
__device__ __forceinline__ double w_rcp(double a) { return rcp_d(a); }
// square root of a value of type R in the wide type (FP32: one correction step)
__device__ __forceinline__ ffv w_sqrt(float x)
{
    const float s = sqrtf(x);
    return ff_norm(s, fmaf(-s, s, x) / (2.0f * s));
}
__device__ __forceinline__ double w_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ ffv w_sqrt(ffv x)
{
    const float s = sqrtf(x.hi);
    return ff_norm(s, (fmaf(-s, s, x.hi) + x.lo) / (2.0f * s));
}
// a parameter in the wide type, from its FP64 value or its float pair (splitting an FP64
// value on the device costs as much as 25 float-float additions)
template <typename A> __device__ __forceinline__ A wide_param(double x, const float (&ff)[2]);
template <> __device__ __forceinline__ double wide_param<double>(double x, const float (&)[2]) { return x; }
template <> __device__ __forceinline__ ffv wide_param<ffv>(double, const float (&ff)[2]) { return {ff[0], ff[1]}; }
template <typename A> __device__ __forceinline__ A wide_dt(const DevParams &p);
template <> __device__ __forceinline__ double wide_dt<double>(const DevParams &p) { return p.dt; }
template <> __device__ __forceinline__ ffv wide_dt<ffv>(const DevParams &p) { return {p.ff_dt[0], p.ff_dt[1]}; }

// p/rho of the run's equation of state; the exponential factor of the Dieterici form and
// the double well's small polynomial in FP64 (rare forms, not worth a float-float one).
__device__ __forceinline__ double w_p_over_rho(const DevParams &p, double r, double t)
{
    if (p.eos_kind != 0) return eos_pressure<double>(p.eos_kind, p.a, p.b, p.R, r, t, p.sp) / r;
    return p.R * t * rcp_d(1.0 - p.b * r) - p.a * r;
}
__device__ __forceinline__ ffv w_p_over_rho(const DevParams &p, float r, float t)
{
    if (p.eos_kind != 0)
        return w_const<ffv>(eos_pressure<double>(p.eos_kind, p.a, p.b, p.R, (double)r, (double)t, p.sp) / (double)r);
    const ffv a = {p.ff_a[0], p.ff_a[1]}, b = {p.ff_b[0], p.ff_b[1]}, Rg = {p.ff_R[0], p.ff_R[1]};
    const ffv den = ff_add(ff_neg(ff_mul(b, r)), 1.0f);
    return w_sub(ff_mul(ff_mul(Rg, t), ff_rcp(den)), ff_mul(a, r));
}
// pressure p(rho, T) of wide rho, T
__device__ __forceinline__ double w_pressure(const DevParams &p, double r, double t)
{
    if (p.eos_kind != 0) return eos_pressure<double>(p.eos_kind, p.a, p.b, p.R, r, t, p.sp);
    return r * p.R * t * rcp_d(1.0 - p.b * r) - p.a * r * r;
}
__device__ __forceinline__ ffv w_pressure(const DevParams &p, ffv r, ffv t)
{
    if (p.eos_kind != 0)
        return w_const<ffv>(eos_pressure<double>(p.eos_kind, p.a, p.b, p.R, w_double(r), w_double(t), p.sp));
    const ffv a = {p.ff_a[0], p.ff_a[1]}, b = {p.ff_b[0], p.ff_b[1]}, Rg = {p.ff_R[0], p.ff_R[1]};
    const ffv den = ff_add(ff_neg(ff_mul(r, b)), 1.0f);
    return w_sub(ff_mul(ff_mul(ff_mul(r, Rg), t), ff_rcp(den)), ff_mul(ff_mul(r, r), a));
}
template <typename A> __device__ __forceinline__ A wide_p_floor(const DevParams &p);
template <> __device__ __forceinline__ double wide_p_floor<double>(const DevParams &p) { return p.p_floor; }
template <> __device__ __forceinline__ ffv wide_p_floor<ffv>(const DevParams &p) { return {p.ff_pfl[0], p.ff_pfl[1]}; }
template <typename A> __device__ __forceinline__ A wide_T(const DevParams &p, A e, A rho);   // T of e (or T_iso)
template <> __device__ __forceinline__ double wide_T<double>(const DevParams &p, double e, double rho)
{
    return p.isothermal ? p.T_iso : (e + p.a * rho) * p.pd.inv_cv;
}
template <> __device__ __forceinline__ ffv wide_T<ffv>(const DevParams &p, ffv e, ffv rho)
{
    if (p.isothermal) return {p.ff_Tiso[0], p.ff_Tiso[1]};
    return ff_mul(ff_add(e, ff_mul(rho, ffv{p.ff_a[0], p.ff_a[1]})), ffv{p.ff_icv[0], p.ff_icv[1]});
}
__device__ __forceinline__ bool w_less(ffv a, ffv b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool w_less(double a, double b) { return a < b; }

// Macroscopic fields of a node from the sums of its streamed populations in D dimensions
// (moments Eq.), in the wide type.
template <int D, typename R>
struct Macro {
    using A = typename Wide<R>::type;
    A rho, gs, E, T, pr, P, ths;   // gs = sum of the streamed g; P = max(p, p_floor)
    A uu[D], uh[D], du[D];         // streamed velocity u*, fluid velocity, u* - u
    R dth;                         // theta* - theta
    // own = stored sums {f, f c (D), g} and the momentum kept beside them (absolute, D);
    // d = the stream's increments of the first D + 2; inv_TL = 1 / T_L
    __device__ __forceinline__ void update(const DevParams &p, R th, const R (&u)[D], const A *own, const A *d,
                                           const A (&F)[D], A rEl, double inv_TL)
    {
        const A s = w_sqrt(th);
        rho = w_add(own[0], d[0]);
        const A irho = w_rcp(rho);
        const A hdt = w_mul(wide_dt<A>(p), R(0.5));
        A kin;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            // sum f v = s sum f c + u sum f: the change of velocity alone
            du[a] = w_mul(w_add(w_mul(s, w_add(own[1 + a], d[1 + a])), own[D + 2 + a]), irho);
            uu[a] = w_add(du[a], w_wide(u[a]));
            uh[a] = w_add(uu[a], w_mul(w_mul(F[a], hdt), irho));
            const A k = w_mul(uh[a], uh[a]);
            kin = a == 0 ? k : w_add(kin, k);
        }
        gs = w_add(own[D + 1], d[D + 1]);
        E = w_mul(w_mul(gs, irho), R(0.5));
        const A e = w_sub(w_sub(E, w_mul(kin, R(0.5))), w_mul(rEl, irho));
        T = wide_T<A>(p, e, rho);
        pr = w_pressure(p, rho, T);
        const A fl = wide_p_floor<A>(p);
        P = w_less(fl, pr) ? pr : fl;
        ths = w_mul(w_mul(P, irho), R(inv_TL));
        dth = w_round(w_sub(ths, w_wide(th)));
    }
    // relative change of the gauge
    __device__ __forceinline__ float change(R th) const
    {
        const float sr = (float)sqrt_(th);
        float r = fabsf((float)dth) / (float)th;
#pragma unroll
        for (int a = 0; a < D; ++a) r = fmaxf(r, fabsf((float)w_round(du[a])) / sr);
        return !(dth == dth) || !(w_round(rho) == w_round(rho)) ? __int_as_float(0x7fc00000) : r;
    }
};

// A tile's common gauge.  Each thread offers its staged nodes' gauges (those of finite
// positive theta), then the block agrees on the nodes of the largest and the smallest theta
// (every thread calls tile_extremes, which holds a barrier).  lo, hi: the velocity components
// of the thread's own nodes.
template <int D>
struct Extremes {
    unsigned top = 0, at = 0, low = 0xffffffffu, lat = 0;   // theta bits and slots
    float lo[D], hi[D];
    __device__ __forceinline__ Extremes()
    {
#pragma unroll
        for (int a = 0; a < D; ++a) { lo[a] = 1.0e38f; hi[a] = -1.0e38f; }
    }
    // u[0 .. D-1]: the velocity
    template <typename R>
    __device__ __forceinline__ void offer(R theta, const R *u, int slot)
    {
        const float th = (float)theta;
        if (!(th > 0.0f && th < 3.0e38f)) return;
        const unsigned b = __float_as_uint(th);
        if (b > top) { top = b; at = (unsigned)slot; }
        if (b < low) { low = b; lat = (unsigned)slot; }
#pragma unroll
        for (int a = 0; a < D; ++a) {
            lo[a] = fminf(lo[a], (float)u[a]);
            hi[a] = fmaxf(hi[a], (float)u[a]);
        }
    }
    __device__ __forceinline__ float hottest() const { return __uint_as_float(top); }
    // the tile's thetas lie within SMOOTH_TILE of each other
    __device__ __forceinline__ bool smooth() const { return top != 0u && __uint_as_float(low) > SMOOTH_TILE * hottest(); }
    // a node of this thread moves faster than SMOOTH_SPREAD s in the gauge gb, s = sqrt of the
    // tile's hottest theta
    template <typename R>
    __device__ __forceinline__ bool spread(const R (&gb)[D + 1], float s) const
    {
        bool far = false;
        const float lim = SMOOTH_SPREAD * s;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const float u = (float)gb[1 + a];
            far = far || hi[a] - u > lim || u - lo[a] > lim;
        }
        return far;
    }
    // with sqrt theta = s, a node of this thread moves |v| dt >= 1 along an axis
    __device__ __forceinline__ bool reach(float s, float dt) const
    {
        float m = s;
#pragma unroll
        for (int a = 0; a < D; ++a) m = fmaxf(m, fmaxf(s + hi[a], s - lo[a]));
        return m * dt >= 1.0f;
    }
};
template <int D>
__device__ __forceinline__ Extremes<D> tile_extremes(Extremes<D> t, uint4 *best)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, t.top), w = __reduce_min_sync(0xffffffffu, t.top == m ? t.at : 0xffffffffu);
    const unsigned n = __reduce_min_sync(0xffffffffu, t.low), v = __reduce_min_sync(0xffffffffu, t.low == n ? t.lat : 0xffffffffu);
    if ((threadIdx.x & 31) == 0) best[threadIdx.x >> 5] = make_uint4(m, w, n, v);
    __syncthreads();
    uint4 b = best[0];
#pragma unroll
    for (int k = 1; k < STEP_THREADS / 32; ++k) {
        const uint4 o = best[k];
        if (o.x > b.x || (o.x == b.x && o.y < b.y)) { b.x = o.x; b.y = o.y; }
        if (o.z < b.z || (o.z == b.z && o.w < b.w)) { b.z = o.z; b.w = o.w; }
    }
    t.top = b.x; t.at = b.y; t.low = b.z; t.lat = b.w;
    return t;
}
// The gauge (sqrt theta, u) of a tile from the records' gauges at its hottest and coldest
// nodes: the hottest node's own in increment form, else the geometric mean of the two
// thetas and the mean velocity (half the amplification on the way in, half on the way out).
template <typename R, int ND>
__device__ __forceinline__ void common_gauge(bool inc, const R *hot, const R *cold, R (&gb)[ND])
{
    gb[0] = inc ? sqrt_(hot[0]) : sqrt_(sqrt_(hot[0]) * sqrt_(cold[0]));
#pragma unroll
    for (int k = 1; k < ND; ++k) gb[k] = inc ? hot[k] : R(0.5) * (hot[k] + cold[k]);
}
__device__ __forceinline__ int ordered(float v)   // keeps the order of floats
{
    const int b = __float_as_int(v);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unordered(int b) { return __int_as_float(b ^ ((b >> 31) & 0x7fffffff)); }
// The gauge of a tile whose velocities spread: its extreme thetas' geometric mean and, along
// each axis, the middle of the tile's velocities (near: all of them lie within FAR_SPEED
// sqrt(hottest theta) of it).  Every thread calls it, between barriers of its own use of
// `best`; it holds one.  Apart from the step, whose code it would spread (2048 x 1024 nodes,
// us a step: 520 inline, 517 as a function).
template <typename R, int D>
struct MiddleGauge { R g[D + 1]; bool near; };
template <typename R, int D>
__device__ __noinline__ MiddleGauge<R, D> middle_gauge_of(unsigned top, unsigned low, float l0, float h0, float l1, float h1,
                                                          float l2, float h2, uint4 *best)
{
    const float lo[3] = {l0, l1, l2}, hi[3] = {h0, h1, h2};
    static_assert(STEP_THREADS / 32 * 2 * D * 4 <= BEST * (int)sizeof(uint4), "best holds the warps' velocities");
    int *w = reinterpret_cast<int *>(best);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const int l = __reduce_min_sync(0xffffffffu, ordered(lo[a])), h = __reduce_max_sync(0xffffffffu, ordered(hi[a]));
        if ((threadIdx.x & 31) == 0) {
            w[(threadIdx.x >> 5) * 2 * D + a] = l;
            w[(threadIdx.x >> 5) * 2 * D + D + a] = h;
        }
    }
    __syncthreads();
    MiddleGauge<R, D> o;
    const R hot = (R)__uint_as_float(top);
    o.g[0] = sqrt_(sqrt_(hot) * sqrt_((R)__uint_as_float(low)));
    const R lim = R(FAR_SPEED) * sqrt_(hot);
    o.near = true;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        int l = w[a], h = w[D + a];
#pragma unroll 1
        for (int k = 1; k < STEP_THREADS / 32; ++k) {
            l = min(l, w[k * 2 * D + a]);
            h = max(h, w[k * 2 * D + D + a]);
        }
        const R u = R(0.5) * (R)unordered(l), v = R(0.5) * (R)unordered(h);
        o.g[1 + a] = u + v;
        o.near = o.near && v - u <= lim;
    }
    return o;
}
template <typename R, int D>
__device__ __forceinline__ bool middle_gauge(const Extremes<D> &t, uint4 *best, R (&gb)[D + 1])
{
    const MiddleGauge<R, D> m = middle_gauge_of<R, D>(t.top, t.low, t.lo[0], t.hi[0], t.lo[1], t.hi[1], t.lo[D - 1], t.hi[D - 1], best);
#pragma unroll
    for (int a = 0; a <= D; ++a) gb[a] = m.g[a];
    return m.near;
}

// Transfer increments along one axis, E[k][a] = l_k((a - 1) + e_a) - delta_ka with
// e_a = q (a - 1) + w (q = (s_src - s)/s, w = (u_src - u)/s), from h = e/2 and
// p = h (2 c_a + e): E_0 = p - h, E_1 = -2 p, E_2 = p + h.
template <typename R>
__device__ __forceinline__ void axis_map(R q, R w, R (&E)[3][3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const R e = q * R(a - 1) + w;
        const R h = R(0.5) * e, pp = h * (R(2 * (a - 1)) + e);
        E[0][a] = pp - h; E[1][a] = R(-2) * pp; E[2][a] = pp + h;
    }
}

// The rows of the map itself, G[k][a] = l_k(xi_a) at xi_a = (1 + q) (a - 1) + w, as products
// (the identity exactly for q = w = 0): for gauges far apart, where I + E would cancel.
template <typename R>
__device__ __forceinline__ void axis_rows(R q, R w, R (&G)[3][3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const R x = a == 1 ? w : (R(1) + q) * R(a - 1) + w;
        const R h = R(0.5) * x;
        G[0][a] = h * (x - R(1)); G[1][a] = (R(1) - x) * (R(1) + x); G[2][a] = h * (x + R(1));
    }
}

// Increment of a separable map on nine values h (i = 3 b + a): [(I + Ey)(I + Ex) h]_i - h_i.
template <typename R>
__device__ __forceinline__ void map_inc(const R (&Ex)[3][3], const R (&Ey)[3][3], const R *h, R (&out)[9])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R t[3], u[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            t[b] = Ex[k][0] * h[3 * b] + Ex[k][1] * h[3 * b + 1] + Ex[k][2] * h[3 * b + 2];
            u[b] = h[3 * b + k] + t[b];
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) out[3 * l + k] = t[l] + (Ey[l][0] * u[0] + Ey[l][1] * u[1] + Ey[l][2] * u[2]);
    }
}

// Departure points of the three directions of an axis, x - (s (j - 1) + u) dt: their floors
// and the cubic Lagrange weights of the four stencil nodes.  True when every floor is -1 or
// 0 (|v| dt < 1 in general), so that the stencils lie within two nodes of the arrival node;
// false also for NaN.
template <typename R>
__host__ __device__ __forceinline__ bool axis_weights(R s, R u, R dt, R (&a)[3][4], bool (&near0)[3])
{
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const R d = -(s * R(j - 1) + u) * dt;
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

// General stream of node (X, Y) into the gauge (th, ux, uy), for departure points farther
// than the staged halo (|v| dt >= 1), tiles whose velocities spread too far (FAR_SPEED) and
// non-finite gauges: reads the stencil nodes' records from global memory.  Offsets are
// clamped to +-2^20 nodes first (a NaN offset goes to the bound), so that the floors and
// their spread stay in int range.  Regions of up to REGION_MAX nodes a side carry each node
// once for all nine directions; wider ones take each direction's 16 stencil nodes in turn.
// inc = the increments of the streamed populations over the node's own (f, then g); of
// `lanes` callers, caller `lane` adds every lanes-th stencil node only.
// One thread per node is bound by its serial chain of region nodes where few blocks fill an
// SM.  Measured (mixed, us a step, eight lanes a node over a staged halo of three, as in
// earlier kernels / this): a droplet at 1.4 T_cr and dt = 1, 256 x 256 nodes 133 / 148, 40 x 28
// 26 / 34; at 2.7 T_cr, 128 x 128 nodes 75 / 362; a flow at |v| dt = 1.3, 512 x 256 nodes 243 /
// 233, 128 x 128 51 / 98, 30 x 9 25 / 32.  (The next record's loads sent ahead: slower, 406
// instead of 362, and 7 % on a step that never comes here, by the registers.)
template <typename R>
__device__ __noinline__ void stream_general(const DevParams &p, const R *__restrict__ in, int X, int Y, R th, R ux,
                                            R uy, bool first, int lane, int lanes, R *inc, unsigned &nreg,
                                            unsigned &npair)
{
    const size_t N = (size_t)p.N;
    const R dt = typed<R>(p).dt;
    const R s = sqrt_(th), inv_s = R(1) / s;
    R own[24];
    load_rec24(in, (size_t)Y * p.nx + X, N, own);
    int fl[2][3];
    R xi[2][3];
#pragma unroll
    for (int ax = 0; ax < 2; ++ax)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const R d = clamp_offset(-(s * R(j - 1) + (ax == 0 ? ux : uy)) * dt);
            const R f = floor(d);
            fl[ax][j] = (int)f;
            xi[ax][j] = d - f + R(1);
        }
    const int lo_x = min(fl[0][0], min(fl[0][1], fl[0][2])), lo_y = min(fl[1][0], min(fl[1][1], fl[1][2]));
    const int ncols = 4 + max(fl[0][0], max(fl[0][1], fl[0][2])) - lo_x;
    const int nrows = 4 + max(fl[1][0], max(fl[1][1], fl[1][2])) - lo_y;
    R accf[9], accg[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) accf[i] = accg[i] = R(0);
    if (ncols <= REGION_MAX && nrows <= REGION_MAX) {
        // in a first stream the node's own entry is carried by the identity: it is skipped
        const bool skip = first && lo_x <= 1 && 1 - lo_x < ncols && lo_y <= 1 && 1 - lo_y < nrows;
        const int own_r = skip ? (1 - lo_y) * ncols + (1 - lo_x) : -1;
        nreg += (unsigned)(ncols * nrows - (skip ? 1 : 0));
#pragma unroll 1
        for (int r = lane; r < ncols * nrows; r += lanes) {
            if (r == own_r) continue;
            const int cy = r / ncols, cx = r - cy * ncols;
            R wx[3], wy[3], v[24];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int kx = cx - (fl[0][j] - lo_x), ky = cy - (fl[1][j] - lo_y);
                wx[j] = (kx >= 0 && kx < 4) ? lag1_rt<R>(kx, xi[0][j]) : R(0);
                wy[j] = (ky >= 0 && ky < 4) ? lag1_rt<R>(ky, xi[1][j]) : R(0);
            }
            load_rec24(in, (size_t)bc_wrap(Y + lo_y - 1 + cy, p.ny, p.bcy) * p.nx +
                               bc_wrap(X + lo_x - 1 + cx, p.nx, p.bcx), N, v);
            const R sn = sqrt_(v[P_TH]);
            const R q = sizeof(R) == 8 ? sn * inv_s - R(1) : fdiv_(v[P_TH] - th, (sn + s) * s);
            R Ex[3][3], Ey[3][3];
            axis_map<R>(q, (v[P_UX] - ux) * inv_s, Ex);
            axis_map<R>(q, (v[P_UY] - uy) * inv_s, Ey);
            region_family<R>(v + P_F, own + P_F, Ex, Ey, wx, wy, accf);
            region_family<R>(v + P_G, own + P_G, Ex, Ey, wx, wy, accg);
        }
    } else {
        npair += 1;
#pragma unroll
        for (int jy = 0; jy < 3; ++jy)
#pragma unroll
            for (int jx = 0; jx < 3; ++jx) {
                const int i = 3 * jy + jx;
#pragma unroll 1
                for (int q = lane; q < 16; q += lanes) {
                    const int kx = q & 3, ky = q >> 2;
                    const size_t nd = (size_t)bc_wrap(Y + fl[1][jy] - 1 + ky, p.ny, p.bcy) * p.nx +
                                      bc_wrap(X + fl[0][jx] - 1 + kx, p.nx, p.bcx);
                    R v[24], tf, tg;
                    load_rec24(in, nd, N, v);
                    v[P_SQ] = sqrt_(v[P_TH]);
                    pair_inc<R>(v, jx, jy, th, s, inv_s, ux, uy, own[P_F + i], own[P_G + i], tf, tg);
                    const R w = lag1_rt<R>(kx, xi[0][jx]) * lag1_rt<R>(ky, xi[1][jy]);
                    accf[i] += w * tf;
                    accg[i] += w * tg;
                }
            }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        inc[i] = accf[i];
        inc[9 + i] = accg[i];
    }
}

// Pairs of FP32 values in one 64-bit register: one instruction multiplies and adds both
// (fma.rn.f32x2: the rate of two FFMAs in one issue slot and one fetched instruction).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;\n" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The stream as a contraction over the staged slots (see the head of this file), FP32:
// own = the node's own slot, pitch = slots per staged row.  Five columns and rows with
// zero weights outside a direction's four nodes, so that every offset is a constant.  f and
// g take the same weights, so a slot holds their values side by side and each instruction
// works on both.  keep = the thread's kept values (y weights).  acc = increments over the
// node's own populations (f, then g).
__device__ __forceinline__ void contract(const float *own, int pitch, const float (&ax)[3][4],
                                         const bool (&nx0)[3], const float (&Lx)[3][3], const float *keep,
                                         float (&acc)[2][9])
{
    constexpr int DS = Slot<float>::stride;
    f32x2 wl[3][5][3], a2[9], dx[DS / 2];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const float w = nx0[k] ? (c == 0 ? 0.0f : ax[k][c - 1 < 0 ? 0 : c - 1]) : (c == 4 ? 0.0f : ax[k][c > 3 ? 3 : c]);
#pragma unroll
            for (int m = 0; m < 3; ++m) wl[k][c][m] = pack2(w * Lx[k][m], w * Lx[k][m]);
        }
#pragma unroll
    for (int q = 0; q < DS / 4; ++q) {
        float t[4];
        lds4(own + 4 * q, t);
        dx[2 * q] = pack2(-t[0], -t[1]);
        dx[2 * q + 1] = pack2(-t[2], -t[3]);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) a2[i] = 0ull;
    const float *row = own - (2 * pitch + 2) * DS;
#pragma unroll 1
    for (int cy = 0; cy < 5; ++cy, row += pitch * DS) {
        f32x2 t[3][3];   // n, k
#pragma unroll
        for (int n = 0; n < 3; ++n)
#pragma unroll
            for (int k = 0; k < 3; ++k) t[n][k] = 0ull;
#pragma unroll
        for (int cx = 0; cx < 5; ++cx) {
            f32x2 v[DS / 2];
#pragma unroll
            for (int q = 0; q < DS / 4; ++q) {
                const ulonglong2 x = reinterpret_cast<const ulonglong2 *>(row + cx * DS)[q];
                v[2 * q] = add2(x.x, dx[2 * q]);
                v[2 * q + 1] = add2(x.y, dx[2 * q + 1]);
            }
#pragma unroll
            for (int n = 0; n < 3; ++n)
#pragma unroll
                for (int m = 0; m < 3; ++m)
#pragma unroll
                    for (int k = 0; k < 3; ++k) t[n][k] = fma2(wl[k][cx][m], v[3 * n + m], t[n][k]);
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const float w = keep[(K_WY + 5 * l + cy) * STEP_THREADS];
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                const float wl_n = w * keep[(K_LY + 3 * l + n) * STEP_THREADS];
                const f32x2 wn = pack2(wl_n, wl_n);
#pragma unroll
                for (int k = 0; k < 3; ++k) a2[3 * l + k] = fma2(wn, t[n][k], a2[3 * l + k]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) unpack2(a2[i], acc[0][i], acc[1][i]);
}

// The same over the FP64 slots: the x pass reads each direction's own four
// columns (shared-memory reads are cheap beside the FP64 pipe, which runs at 1/64 of the
// FP32 rate), and a row pass costs 36 multiply-adds instead of 45.  acc = the streamed
// populations.
__device__ __forceinline__ void contract(const double *own, int pitch, const double (&ax)[3][4],
                                         const bool (&nx0)[3], const double (&Lx)[3][3], const double *keep,
                                         double (&acc)[2][9])
{
    constexpr int DS = Slot<double>::stride;
    double wl[3][4][3];
    int off[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        off[k] = nx0[k] ? DS : 0;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int m = 0; m < 3; ++m) wl[k][c][m] = ax[k][c] * Lx[k][m];
    }
#pragma unroll
    for (int fam = 0; fam < 2; ++fam)
#pragma unroll
        for (int i = 0; i < 9; ++i) acc[fam][i] = 0.0;
    const double *row = own - (2 * pitch + 2) * DS;
#pragma unroll 1
    for (int cy = 0; cy < 5; ++cy, row += pitch * DS) {
        double wn[3][3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const double w = keep[(K_WY + 5 * l + cy) * STEP_THREADS];
#pragma unroll
            for (int n = 0; n < 3; ++n) wn[l][n] = w * keep[(K_LY + 3 * l + n) * STEP_THREADS];
        }
#pragma unroll
        for (int fam = 0; fam < 2; ++fam)
#pragma unroll
            for (int n = 0; n < 3; ++n) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double *r = row + off[k] + 9 * fam + 3 * n;
                    double t = 0.0;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int m = 0; m < 3; ++m) t = fma(wl[k][c][m], r[c * DS + m], t);
#pragma unroll
                    for (int l = 0; l < 3; ++l) acc[fam][3 * l + k] = fma(wn[l][n], t, acc[fam][3 * l + k]);
                }
            }
    }
}

// The streamed populations of one direction (k, l) as a contraction over the direction's own
// 4 x 4 staged slots: first the nodes by their Lagrange weights, then the rows of the map.  For
// departure floors other than -1 and 0 (fx, fy), which the window of `contract` does not hold.
__device__ __forceinline__ void contract_one(const double *own, int pitch, const double (&ax)[4], int fx,
                                             const double (&ay)[4], int fy, const double (&Lx)[3], const double (&Ly)[3],
                                             double &of, double &og)
{
    constexpr int DS = Slot<double>::stride;
    double a[18];
#pragma unroll
    for (int i = 0; i < 18; ++i) a[i] = 0.0;
    const double *row = own + ((fy - 1) * pitch + fx - 1) * DS;
#pragma unroll 1
    for (int r = 0; r < 4; ++r, row += pitch * DS) {
        const double wr = r < 2 ? (r == 0 ? ay[0] : ay[1]) : (r == 2 ? ay[2] : ay[3]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double w = ax[c] * wr;
#pragma unroll
            for (int i = 0; i < 18; ++i) a[i] = fma(w, row[c * DS + i], a[i]);
        }
    }
    of = og = 0.0;
#pragma unroll
    for (int n = 0; n < 3; ++n) {
        of = fma(Ly[n], Lx[0] * a[3 * n] + Lx[1] * a[3 * n + 1] + Lx[2] * a[3 * n + 2], of);
        og = fma(Ly[n], Lx[0] * a[9 + 3 * n] + Lx[1] * a[9 + 3 * n + 1] + Lx[2] * a[9 + 3 * n + 2], og);
    }
}

// Weights and floor of the departure point x - v dt; whether its stencil lies within HALO_FAR
// nodes of the arrival node (false for NaN).
template <typename R>
__device__ __forceinline__ bool far_departure(R v, R dt, R (&a)[4], int &floor_)
{
    const R d = -v * dt;
    const R f = floor(d);
    const bool ok = f >= R(1 - HALO_FAR) && f <= R(HALO_FAR - 2);
    floor_ = ok ? (int)f : 0;
    const R t0 = d - f + R(1), t1 = t0 - R(1), t2 = t0 - R(2), t3 = t0 - R(3);
    const R p12 = t1 * t2, p03 = t0 * t3;
    a[0] = p12 * t3 * R(-1.0 / 6.0);
    a[1] = p03 * t2 * R(0.5);
    a[2] = p03 * t1 * R(-0.5);
    a[3] = p12 * t0 * R(1.0 / 6.0);
    return ok;
}
// Row k (run time) of the map: l_k at (1 + q) (m - 1) + w.
template <typename R>
__device__ __forceinline__ void map_row(int k, R q, R w, R (&L)[3])
{
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const R x = m == 1 ? w : (R(1) + q) * R(m - 1) + w;
        L[m] = k == 1 ? (R(1) - x) * (R(1) + x) : R(0.5) * x * (x + R(k - 1));
    }
}

// The streamed populations of direction (k, l) where the wider halo holds its stencil (ok).
struct FarOne { double f, g; int fx, fy; bool ok; };
__device__ __noinline__ FarOne far_one(const double *own, int pitch, int k, int l, double sb, double ubx, double uby,
                                       double s, double inv_s, double dt, double ux, double uy)
{
    FarOne o{0.0, 0.0, 0, 0, false};
    double ax[4], ay[4], Lx[3], Ly[3];
    const bool okx = far_departure<double>(s * (k - 1) + ux, dt, ax, o.fx), oky = far_departure<double>(s * (l - 1) + uy, dt, ay, o.fy);
    o.ok = okx && oky;
    map_row<double>(k, (sb - s) * inv_s, (ubx - ux) * inv_s, Lx);
    map_row<double>(l, (sb - s) * inv_s, (uby - uy) * inv_s, Ly);
    if (o.ok) contract_one(own, pitch, ax, o.fx, ay, o.fy, Lx, Ly, o.f, o.g);
    return o;
}

// FP64, over slots with the wider halo: streams a node whose departure points leave the window
// of `contract`, where that halo holds them as a contraction over 7 rows, of each x
// component's own four columns, else in general.  buf = the increments of the streamed
// populations over the node's own.  Measured (us a step, the eight-lane kernels / the general
// stream / this): a droplet at 1.4 T_cr, dt = 1, 256 x 256 nodes 4498 / 4607 / 2202; at 2.7
// T_cr, 128 x 128 nodes 1973 / 4145 / 1050; a flow at |v| dt = 1.3, 128 x 128 nodes 1194 / 1139
// / 580, with nine lanes 30 x 9 nodes 208 / 281 / 197.
__device__ __noinline__ void stream_far(const DevParams &p, const double *__restrict__ in, int X, int Y,
                                        const double *own, int pitch, double sb, double ubx, double uby,
                                        double dt, double th, double ux, double uy, bool first, double *buf,
                                        unsigned &nreg, unsigned &npair)
{
    constexpr int DS = Slot<double>::stride;
    const double s = sqrt_(th), inv_s = 1.0 / s;
    double wx[3][4], wy[3][4];
    int fx[3], fy[3];
    bool far = true;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        far = far_departure<double>(s * (j - 1) + ux, dt, wx[j], fx[j]) && far;
        far = far_departure<double>(s * (j - 1) + uy, dt, wy[j], fy[j]) && far;
    }
    if (!far) {
        stream_general<double>(p, in, X, Y, th, ux, uy, first, 0, 1, buf, nreg, npair);
        return;
    }
    nreg += (unsigned)((4 + max(fx[0], max(fx[1], fx[2])) - min(fx[0], min(fx[1], fx[2]))) *
                           (4 + max(fy[0], max(fy[1], fy[2])) - min(fy[0], min(fy[1], fy[2]))) - (first ? 1 : 0));
    double Lx[3][3], Ly[3][3], acc[2][9];
    const double qb = (sb - s) * inv_s;
    axis_rows<double>(qb, (ubx - ux) * inv_s, Lx);
    axis_rows<double>(qb, (uby - uy) * inv_s, Ly);
#pragma unroll
    for (int i = 0; i < 9; ++i) acc[0][i] = acc[1][i] = 0.0;
#pragma unroll 1
    for (int r = -HALO_FAR; r <= HALO_FAR; ++r) {
        double wr[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const int j = r - fy[l] + 1;   // the row's place in the stencil of component l
            wr[l] = (j >= 0 && j < 4) ? pick(wy[l], j) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double *c0 = own + (r * pitch + fx[k] - 1) * DS;
#pragma unroll
            for (int fam = 0; fam < 2; ++fam)
#pragma unroll
                for (int n = 0; n < 3; ++n) {
                    double t = 0.0;
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        double v = 0.0;
#pragma unroll
                        for (int c = 0; c < 4; ++c) v = fma(wx[k][c], c0[c * DS + 9 * fam + 3 * n + m], v);
                        t = fma(Lx[k][m], v, t);
                    }
#pragma unroll
                    for (int l = 0; l < 3; ++l) acc[fam][3 * l + k] = fma(wr[l] * Ly[l][n], t, acc[fam][3 * l + k]);
                }
        }
    }
    double v[24];
    load_rec24(in, (size_t)Y * p.nx + X, (size_t)p.N, v);
#pragma unroll
    for (int i = 0; i < 18; ++i) buf[i] = acc[i / 9][i % 9] - v[i];
}

// Streams node (X, Y) into the gauge (th, ux, uy): inc = the increments of the streamed
// populations over the node's own (f, then g).  gauge_b: the tile's common gauge
// (sqrt theta, u_x, u_y); dt: of stage_tile; FAR: the slots have a halo of HALO_FAR; keep:
// the thread's column of kept values.
template <typename R, bool FAR>
__device__ __forceinline__ void stream_node(const DevParams &p, const R *__restrict__ in, int X, int Y, const R *slot,
                                            int pitch, const R (&gauge_b)[3], R dt, R th, R ux, R uy, bool first,
                                            R *keep, R (&inc)[2][9], unsigned &nreg, unsigned &npair)
{
    const R s = sqrt_(th), inv_s = R(1) / s;
    R ax[3][4], ay[3][4];
    bool nx0[3], ny0[3];
    const bool okx = axis_weights<R>(s, ux, dt, ax, nx0), oky = axis_weights<R>(s, uy, dt, ay, ny0);
    if (!(okx && oky)) {
        R buf[18];
        if constexpr (FAR)
            stream_far(p, in, X, Y, slot, pitch, gauge_b[0], gauge_b[1], gauge_b[2], dt, th, ux, uy, first, buf, nreg, npair);
        else
            stream_general<R>(p, in, X, Y, th, ux, uy, first, 0, 1, buf, nreg, npair);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            inc[0][i] = buf[i];
            inc[1][i] = buf[9 + i];
        }
        return;
    }
    const int sx = (nx0[0] == nx0[1] && nx0[1] == nx0[2]) ? 4 : 5, sy = (ny0[0] == ny0[1] && ny0[1] == ny0[2]) ? 4 : 5;
    nreg += (unsigned)(sx * sy - (first ? 1 : 0));
    R Lx[3][3], Ly[3][3];
    const R qb = (gauge_b[0] - s) * inv_s;
    axis_rows<R>(qb, (gauge_b[1] - ux) * inv_s, Lx);
    axis_rows<R>(qb, (gauge_b[2] - uy) * inv_s, Ly);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
#pragma unroll
        for (int c = 0; c < 5; ++c)
            keep[(K_WY + 5 * l + c) * STEP_THREADS] =
                ny0[l] ? (c == 0 ? R(0) : ay[l][c - 1 < 0 ? 0 : c - 1]) : (c == 4 ? R(0) : ay[l][c > 3 ? 3 : c]);
#pragma unroll
        for (int n = 0; n < 3; ++n) keep[(K_LY + 3 * l + n) * STEP_THREADS] = Ly[l][n];
    }
    contract(slot, pitch, ax, nx0, Lx, keep, inc);
    if constexpr (sizeof(R) == 8) {
        R v[24];
        load_rec24(in, (size_t)Y * p.nx + X, (size_t)p.N, v);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            inc[0][i] -= v[P_F + i];
            inc[1][i] -= v[P_G + i];
        }
    } else {
        if (!first) {
            // the node's own populations carried from their stored gauge into this one
            R v[24], Ex[3][3], Ey[3][3], o[9];
            load_rec24(in, (size_t)Y * p.nx + X, (size_t)p.N, v);
            const R qx = fdiv_(v[P_TH] - th, (sqrt_(v[P_TH]) + s) * s);
            axis_map<R>(qx, (v[P_UX] - ux) * inv_s, Ex);
            axis_map<R>(qx, (v[P_UY] - uy) * inv_s, Ey);
#pragma unroll
            for (int fam = 0; fam < 2; ++fam) {
                map_inc<R>(Ex, Ey, v + 9 * fam, o);
#pragma unroll
                for (int i = 0; i < 9; ++i) inc[fam][i] += o[i];
            }
        }
    }
}

// Korteweg stress and heat flux of the staged node at slot s0 (K = -kappa (rho lap rho +
// |grad rho|^2/2) I + kappa grad rho (x) grad rho, q = -mu grad h + k grad T), from
// differences to the centre value (sum_i W_i c_i = 0), which keeps their FP32 rounding
// proportional to the differences.
template <typename R>
__device__ __forceinline__ void stress_and_flux(const TypedParams<R> &q, const R *aux, int s0, int pitch, R (&o)[KQW])
{
    R c[4];
    lds4(aux + (size_t)s0 * AUXW, c);
    R grx = 0, gry = 0, lap = 0, ghx = 0, ghy = 0, gTx = 0, gTy = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ex = i % 3 - 1, ey = i / 3 - 1;
        if (ex == 0 && ey == 0) continue;
        R v[4];
        lds4(aux + (s0 + ey * pitch + ex) * AUXW, v);
        const R w = wst<R>(ex, ey);
        const R dr = v[0] - c[0], dT = v[1] - c[1];
        const R dh = q.cv * dT - q.a * dr + (v[3] - c[3]);
        grx += w * R(ex) * dr;
        gry += w * R(ey) * dr;
        lap += w * dr;
        ghx += w * R(ex) * dh;
        ghy += w * R(ey) * dh;
        gTx += w * R(ex) * dT;
        gTy += w * R(ey) * dT;
    }
    grx *= R(3); gry *= R(3); lap *= R(6);
    ghx *= R(3); ghy *= R(3); gTx *= R(3); gTy *= R(3);
    const R kap = q.kappa;
    const R iso = -kap * (c[0] * lap + R(0.5) * (grx * grx + gry * gry));
    const R P0 = c[2] > q.p_floor ? c[2] : q.p_floor;
    const R mu = q.mu_coef * P0;
    const R kc = q.k_cond >= R(0) ? q.k_cond : mu * q.cvR;
    o[0] = iso + kap * grx * grx;
    o[1] = kap * grx * gry;
    o[2] = iso + kap * gry * gry;
    o[3] = -mu * ghx + kc * gTx;
    o[4] = -mu * ghy + kc * gTy;
}

// Collision of one node: ft, gt = its streamed populations (f~ = own + inc), o = the last
// corrector's results, (th, ux, uy) the streaming gauge.  Fills the record.
template <typename R>
__device__ __forceinline__ void collide(const TypedParams<R> &q, const EosOut<R> &o, R th, R ux, R uy, R Fx, R Fy,
                                        R M0, const R (&ft)[9], const R (&gt)[9], R (&rec)[SL])
{
    const R s = sqrt_(th), inv_s = R(1) / s;
    const R rr = o.rho_hi, uxr = o.uxs, uyr = o.uys, uhxr = o.uhx, uhyr = o.uhy, Er = o.E;
    const R Pr = o.P, sst = sqrt_(o.ths);
    const R qm1 = sizeof(R) == 8 ? sst * inv_s - R(1) : fdiv_(o.dth, (sst + s) * s);
    const R wsx = o.dux * inv_s, wsy = o.duy * inv_s;
    const R dtr = q.dt, om = q.omega;
    const R irr = frcp_(rr), iP2 = frcp_(R(2) * Pr);
    const R dvx = Fx * dtr * irr * inv_s, dvy = Fy * dtr * irr * inv_s;
    const R W1[3] = {wlat<R>(0), wlat<R>(1), wlat<R>(2)};
    // transfer increments from lambda* = (ths, u*) into the streaming gauge and from the
    // force-shifted frame (ths, u* + F dt/rho) (Eq. S-i): E[k][a] = l_k increments at the
    // source velocities, Ws[k] = sum_a E[k][a] W_a, Wh[k] = the shifted frame's extra weight
    R Ex[3][3], Ey[3][3], Wsx[3], Wsy[3], Whx[3], Why[3];
    auto rows = [&](R w, R dv, R (&E)[3][3], R (&Ws)[3], R (&Wh)[3]) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Ws[k] = 0;
            Wh[k] = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R e = qm1 * R(a - 1) + w;
                E[k][a] = ell_inc<R>(k, a, e);
                Ws[k] += E[k][a] * W1[a];
                Wh[k] += (ell_inc<R>(k, a, e + dv) - E[k][a]) * W1[a];
            }
        }
    };
    rows(wsx, dvx, Ex, Wsx, Whx);
    rows(wsy, dvy, Ey, Wsy, Why);
    // g: forced equilibrium (Eq. new geq), heat-flux correction (Eq. gtilde) and the
    // force-work source 2 W_i uhat.F, all in lambda*
    const R H = Er + Pr * irr;
    const R Ixx = R(2) * uhxr * Fx + dtr * Fx * Fx * Er * iP2;
    const R Ixy = uhxr * Fy + Fx * uhyr + dtr * Fx * Fy * Er * iP2;
    const R Iyy = R(2) * uhyr * Fy + dtr * Fy * Fy * Er * iP2;
    const R cM = R(2) * dtr * rr * iP2;
    const R Mx = cM * (Fx * H - (Ixx * uxr + Ixy * uyr));
    const R My = cM * (Fy * H - (Ixy * uxr + Iyy * uyr));
    const R cN = dtr * rr * iP2;
    const R Nxx = rr + cN * Ixx, Nxy = cN * Ixy, Nyy = rr + cN * Iyy;
    // P/rho in the g equilibrium as sqrt(theta*)^2 times the lattice temperature of
    // the weights in use (sum_i W_i c_ix^2 = 2 W_+-1), so that the equilibrium's zeroth
    // moment is 2 rho E to rounding also in FP32 (sum_i W_i (v_x^2 - P/rho - u_x^2) = 0)
    const R Pd = sst * sst * (R(2) * W1[0]);
    const R work = R(2) * (uhxr * Fx + uhyr * Fy);
    R Xs[9], ginc[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ix = i % 3, iy = i / 3;
        const R cx = R(ix - 1), cy = R(iy - 1);
        const R w = W1[ix] * W1[iy];
        const R ccx = sst * cx, ccy = sst * cy;                  // v - u* in lambda*
        const R Axx = ccx * ccx + R(2) * ccx * uxr - Pd;          // v v - P/rho I - u u
        const R Axy = ccx * ccy + ccx * uyr + ccy * uxr;
        const R Ayy = ccy * ccy + R(2) * ccy * uyr - Pd;
        const R geq = w * (R(2) * rr * Er + Mx * ccx + My * ccy + Nxx * Axx + R(2) * Nxy * Axy + Nyy * Ayy);
        const R vx = ccx + uxr, vy = ccy + uyr;
        const R uc = uxr * cx + uyr * cy;
        const R gc = M0 * w * (R(1) + rr * uc * uc * iP2 * R(3) - rr * (vx * vx + vy * vy) * iP2 + R(1));
        Xs[i] = om * geq + dtr * (gc + w * work);
    }
    map_inc<R>(Ex, Ey, Xs, ginc);
    // The collision conserves mass exactly and changes the energy by dt (M_0 + 2 uhat.F);
    // the rest population (i = 4) takes the remainder, summed error-free as (hi, lo)
    // pairs, so that the stored populations keep these sums up to one rounding.
    // The stored momentum (exact pair sums of the stored populations) falls short of the
    // exact post-collision momentum sum f~ c + F dt / s by its storage rounding; that
    // difference is kept beside the populations too.
    R fh = 0, fl = 0, gh = 0, gl = 0, xh = 0, xl = 0, yh = 0, yl = 0;
    auto add = [](R &h, R &l, R v) {
        R e;
        two_sum_(h, v, h, e);
        l += e;
    };
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4) continue;
        const int kx = i % 3, ky = i / 3;
        const R Wx = W1[kx] + Wsx[kx], Wy = W1[ky] + Wsy[ky];
        // f^eq - f~ with the frame-offset increments kept apart from the O(1) weights:
        // W + Ws rounded in FP32 would keep only the increment's leading bits (Ws ~ the gauge
        // change of one step, a few ulps of W), and always the same way, since W is a constant
        const R dfeq = (rr * W1[kx] * W1[ky] - ft[i]) + rr * (Wsx[kx] * W1[ky] + W1[kx] * Wsy[ky] + Wsx[kx] * Wsy[ky]);
        const R S = rr * (Whx[kx] * (Wy + Why[ky]) + Wx * Why[ky]);
        const R fo = ft[i] + om * dfeq + S;
        // X* carried into the streaming gauge
        const R go = (R(1) - om) * gt[i] + (Xs[i] + ginc[i]);
        rec[P_F + i] = fo;
        rec[P_G + i] = go;
        add(fh, fl, fo);
        add(gh, gl, go);
        if (kx != 1) add(xh, xl, R(kx - 1) * fo);
        if (ky != 1) add(yh, yl, R(ky - 1) * fo);
    }
    // target sums: rho (hi, lo) and sum g~ + dt (M_0 + work); the remainders as (hi, lo)
    // pairs: hi is stored as the population, lo beside it for the next step's sums
    R th_, tl_, s1, e1;
    two_sum_(o.gs_hi, dtr * (M0 + work), th_, tl_);
    tl_ += o.gs_lo;
    two_sum_(o.rho_hi, -fh, s1, e1);
    two_sum_(s1, e1 + (o.rho_lo - fl), rec[P_F + 4], rec[P_F4LO]);
    two_sum_(th_, -gh, s1, e1);
    two_sum_(s1, e1 + (tl_ - gl), rec[P_G + 4], rec[P_G4LO]);
    rec[P_JXLO] = ((o.mx_hi - xh) + (o.mx_lo - xl)) + Fx * dtr * inv_s;
    rec[P_JYLO] = ((o.my_hi - yh) + (o.my_lo - yl)) + Fy * dtr * inv_s;
    rec[P_TH] = th; rec[P_UX] = ux; rec[P_UY] = uy; rec[P_SQ] = 0;
    rec[P_RHO] = rr; rec[P_T] = o.T; rec[P_UHX] = uhxr; rec[P_UHY] = uhyr;
    rec[30] = rec[31] = 0;
}

// A tile of a step kernel's block: TX x TY nodes from (X0, Y0) staged with a halo of `halo`
// nodes, WT staged slots and RW ring nodes per row, and its shared memory.
template <typename R>
struct Tile {
    int X0, Y0, TX, TY, halo, WT, RW, nslots;
    R *aux, *slots, *kq, *rest;   // rest: after the others, whatever the halo
    __device__ __forceinline__ Tile(const DevParams &p, int idx, R *smem) : TX(p.tile_x), TY(p.tile_y), RW(TX + 2)
    {
        X0 = (idx % p.tiles_x) * TX;
        Y0 = (idx / p.tiles_x) * TY;
        aux = smem;
        rest = aux + (size_t)step_slots(TX, TY, widest_halo(TX, TY, sizeof(R))) * (AUXW + Slot<R>::stride) + (size_t)RW * (TY + 2) * KQW;
        set_halo(HALO);
    }
    __device__ __forceinline__ void set_halo(int h)
    {
        halo = h;
        WT = TX + 2 * h;
        nslots = step_slots(TX, TY, h);
        slots = aux + (size_t)nslots * AUXW;
        kq = slots + (size_t)nslots * Slot<R>::stride;
    }
    __device__ __forceinline__ int slot(int tx, int ty) const { return (ty + halo) * WT + tx + halo; }
};

// Stages a tile and its halo (see the head of this file) and computes K and q on the tile
// and its ring; gb = the tile's common gauge: sqrt(theta), u_x, u_y.  Returns the time step
// of the contraction's departure points: dt, or infinity, which no contraction takes, in a
// tile whose velocities spread too far for it; or 0, with nothing staged, where a node moves
// |v| dt >= 1 and the tile can hold a wider halo than tl's.  Every thread of the block calls
// it; it ends with a barrier.
template <typename R>
__device__ __forceinline__ R stage_tile(const DevParams &p, const R *__restrict__ in, const R *nlsrc,
                                           const Tile<R> &tl, StepCounts &counts, R (&gb)[3])
{
    constexpr int DS = Slot<R>::stride, ST_NT = STEP_THREADS;
    const TypedParams<R> &q = typed<R>(p);
    const size_t N = (size_t)p.N;
    const int tid = threadIdx.x;
    const int X0 = tl.X0, Y0 = tl.Y0, TX = tl.TX, TY = tl.TY, WT = tl.WT, nslots = tl.nslots;
    R *aux = tl.aux, *slots = tl.slots, *kq = tl.kq;
    __shared__ uint4 best[BEST];   // per warp: largest and smallest theta (bits) and their slots; velocities
    if (tid == 0) counts = StepCounts{};
    // k / WT through the float reciprocal: exact for k < 2^20 (the quotient's fraction
    // stays >= 0.5 / WT away from an integer)
    const float iwt = 1.0f / (float)WT;
    auto node_of = [&](int k) -> size_t {
        const int cv = (int)(((float)k + 0.5f) * iwt), cu = k - cv * WT;
        return (size_t)bc_wrap(Y0 - tl.halo + cv, p.ny, p.bcy) * p.nx + bc_wrap(X0 - tl.halo + cu, p.nx, p.bcx);
    };
    auto put_aux = [&](int k, size_t nd, R r, R t) {
        if (nlsrc != in) {   // current-time non-local terms: rho, T of the first pass's prediction
            r = nlsrc[rec_at(nlsrc, nd, P_RHO, N)];
            t = nlsrc[rec_at(nlsrc, nd, P_T, N)];
        }
        const R pr = eos_pressure<R>(p.eos_kind, q.a, q.b, q.R, r, t, typed_sp<R>(p));
        R *a = aux + (size_t)k * AUXW;
        a[0] = r; a[1] = t; a[2] = pr; a[3] = fdiv_(pr, r);
    };

    // ---------------- staging ------------------------------------------------------
    R va[24], vb[24];
    const int ka = tid, kb = tid + ST_NT;
    size_t na = 0, nb = 0;
    Extremes<2> ex;
    if (ka < nslots) { na = node_of(ka); load_rec24(in, na, N, va); }
    if (kb < nslots) { nb = node_of(kb); load_rec24(in, nb, N, vb); }
    // every slot's gauge goes to shared memory (where its rho, T will lie), so that the
    // agreed nodes' gauges and populations need no further global loads
    auto note = [&](int k, R th, R ux, R uy) {
        const R u[2] = {ux, uy};
        ex.offer(th, u, k);
        R *a = aux + (size_t)k * AUXW;
        a[0] = th; a[1] = ux; a[2] = uy;
    };
    if (ka < nslots) note(ka, va[P_TH], va[P_UX], va[P_UY]);
    if (kb < nslots) note(kb, vb[P_TH], vb[P_UX], vb[P_UY]);
    for (int k = tid + 2 * ST_NT; k < nslots; k += ST_NT) {
        const size_t nd = node_of(k);
        note(k, __ldg(in + rec_at(in, nd, P_TH, N)), __ldg(in + rec_at(in, nd, P_UX, N)), __ldg(in + rec_at(in, nd, P_UY, N)));
    }
    ex = tile_extremes(ex, best);
    bool smooth = sizeof(R) == 4 && ex.smooth();
    const int khot = min((int)ex.at, nslots - 1), kcold = min((int)ex.lat, nslots - 1);
    R thb, shot;   // theta of the gauge; sqrt theta of the hottest node
    {
        R hot[3], cold[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            hot[k] = aux[khot * AUXW + k];
            cold[k] = aux[kcold * AUXW + k];
        }
        common_gauge<R, 3>(smooth, hot, cold, gb);
        shot = sqrt_(hot[0]);
        thb = smooth ? hot[0] : gb[0] * gb[0];
    }
    __shared__ R base[18];   // the hottest node's populations
    if (smooth) {
        if (khot == ka) {
#pragma unroll
            for (int i = 0; i < 18; ++i) base[i] = va[i];
        } else if (khot == kb) {
#pragma unroll
            for (int i = 0; i < 18; ++i) base[i] = vb[i];
        } else if (khot >= 2 * ST_NT && tid == 0) {
            const size_t nd = node_of(khot);
#pragma unroll
            for (int i = 0; i < 18; ++i) base[i] = __ldg(in + rec_at(in, nd, i, N));
        }
    }
    // (the barrier: base is there, and aux may be overwritten)
    R dt = q.dt;
    const bool spread = ex.spread(gb, (float)shot), reach = ex.reach((float)shot, p.pf.dt) && tl.halo < widest_halo(TX, TY, sizeof(R));
    if (__builtin_expect(__syncthreads_or(spread || reach), 0)) {   // (rare: out of the way)
        if (__syncthreads_or(spread)) {
            smooth = false;
            if (!middle_gauge<R, 2>(ex, best, gb)) dt = R(1) / R(0);
            thb = gb[0] * gb[0];
        }
        if (sizeof(R) == 8 && __syncthreads_or(reach) && dt == q.dt) return R(0);
    }
    const R inv_sb = R(1) / gb[0];
    auto carry = [&](int k, size_t nd, const R (&v)[24]) {
        const R sn = sqrt_(v[P_TH]);
        const R e = fdiv_(v[P_TH] - thb, (sn + gb[0]) * gb[0]);
        const R wx = (v[P_UX] - gb[1]) * inv_sb, wy = (v[P_UY] - gb[2]) * inv_sb;
        R Ex[3][3], Ey[3][3], d[DS];
        if (smooth) {
            axis_map<R>(e, wx, Ex);
            axis_map<R>(e, wy, Ey);
#pragma unroll
            for (int fam = 0; fam < 2; ++fam) {
                R o[9];
                map_inc<R>(Ex, Ey, v + 9 * fam, o);
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    d[slot_at<R>(fam, i)] = (v[9 * fam + i] - base[9 * fam + i]) + o[i];
            }
        } else {
            axis_rows<R>(e, wx, Ex);
            axis_rows<R>(e, wy, Ey);
#pragma unroll
            for (int fam = 0; fam < 2; ++fam)
#pragma unroll
                for (int k2 = 0; k2 < 3; ++k2) {
                    R t[3];
#pragma unroll
                    for (int b2 = 0; b2 < 3; ++b2)
                        t[b2] = Ex[k2][0] * v[9 * fam + 3 * b2] + Ex[k2][1] * v[9 * fam + 3 * b2 + 1] +
                                Ex[k2][2] * v[9 * fam + 3 * b2 + 2];
#pragma unroll
                    for (int l2 = 0; l2 < 3; ++l2)
                        d[slot_at<R>(fam, 3 * l2 + k2)] = Ey[l2][0] * t[0] + Ey[l2][1] * t[1] + Ey[l2][2] * t[2];
                }
        }
        R *dst = slots + (size_t)k * DS;
        if constexpr (sizeof(R) == 4) {
            d[18] = d[19] = R(0);
#pragma unroll
            for (int c = 0; c < DS / 4; ++c)
                reinterpret_cast<float4 *>(dst)[c] = make_float4(d[4 * c], d[4 * c + 1], d[4 * c + 2], d[4 * c + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < 18; ++i) dst[i] = d[i];
        }
        put_aux(k, nd, v[P_RHO], v[P_T]);
    };
    // (one copy of the carrying code: it is fetched once and runs for every slot)
#pragma unroll 1
    for (int k = tid; k < nslots; k += ST_NT) {
        if (k >= 2 * ST_NT) {
            na = node_of(k);
            load_rec24(in, na, N, va);
        } else if (k >= ST_NT) {
            na = nb;
#pragma unroll
            for (int i = 0; i < 24; ++i) va[i] = vb[i];
        }
        carry(k, na, va);
    }
    __syncthreads();

    // ---------------- phase 0: non-local terms --------------------------------------
    const int RW = tl.RW;
    {
        const float irw = 1.0f / (float)RW;
        for (int k = tid; k < RW * (TY + 2); k += ST_NT) {
            const int j = (int)(((float)k + 0.5f) * irw), i = k - j * RW;
            // a zero-gradient edge clamps the node onto the grid first (its stencil is that
            // of the boundary node itself)
            const int mx = p.bcx == 0 ? X0 + i - 1 : bc_wrap(X0 + i - 1, p.nx, 1);
            const int my = p.bcy == 0 ? Y0 + j - 1 : bc_wrap(Y0 + j - 1, p.ny, 1);
            R o[KQW];
            stress_and_flux<R>(q, aux, (my - (Y0 - tl.halo)) * WT + (mx - (X0 - tl.halo)), WT, o);
#pragma unroll
            for (int c = 0; c < KQW; ++c) kq[k * KQW + c] = o[c];
        }
    }
    __syncthreads();
    return dt;
}

// Adds a block's counters (its warps' values) to the context's.  Every thread calls it.
__device__ __forceinline__ void add_counts(StepCounts &counts, DevStats *stats, unsigned its, unsigned nreg,
                                           unsigned npair, bool nonconv, bool stall, bool floored, bool bad)
{
    const int tid = threadIdx.x;
    // ---------------- statistics: warp sums, then one set of atomics per block --------
    {
        const unsigned m = 0xffffffffu;
        const unsigned w_its = __reduce_add_sync(m, its), w_reg = __reduce_add_sync(m, nreg);
        const unsigned w_pair = __reduce_add_sync(m, npair), w_max = __reduce_max_sync(m, its);
        const unsigned nc = __popc(__ballot_sync(m, nonconv)), st = __popc(__ballot_sync(m, stall));
        const unsigned cl = __popc(__ballot_sync(m, floored)), nf = __popc(__ballot_sync(m, bad));
        if ((tid & 31) == 0) {
            atomicAdd(&counts.streams, w_its);
            atomicAdd(&counts.region_nodes, w_reg);
            atomicAdd(&counts.warp_streams, w_max);
            atomicMax(&counts.max_streams, w_max);
            if (w_pair) atomicAdd(&counts.pair_streams, w_pair);
            if (nc) atomicAdd(&counts.nonconv, nc);
            if (st) atomicAdd(&counts.stalled, st);
            if (cl) atomicAdd(&counts.clamped, cl);
            if (nf) atomicAdd(&counts.nonfinite, nf);
        }
    }
    __syncthreads();
    if (tid == 0) {
        atomicAdd(&stats->streams, (unsigned long long)counts.streams);
        atomicAdd(&stats->region_nodes, (unsigned long long)counts.region_nodes);
        atomicAdd(&stats->block_streams, (unsigned long long)counts.warp_streams);
        atomicMax(&stats->max_streams, (unsigned long long)counts.max_streams);
        if (counts.pair_streams) atomicAdd(&stats->pair_streams, (unsigned long long)counts.pair_streams);
        if (counts.nonconv) atomicAdd(&stats->nonconv, (unsigned long long)counts.nonconv);
        if (counts.stalled) atomicAdd(&stats->stalled, (unsigned long long)counts.stalled);
        if (counts.clamped) atomicAdd(&stats->clamped, (unsigned long long)counts.clamped);
        if (counts.nonfinite) atomicAdd(&stats->nonfinite, (unsigned long long)counts.nonfinite);
    }
}

// Divergences of K and q at a node from the differences of opposite neighbours:
// F = -div K, M_0 = 2 div q, and grad rho (for rho E_lambda); c0, a0 = the node's entries
// of kq and aux.  Pair i < 4 of the neighbours alone (add the four).
template <typename R>
__device__ __forceinline__ void divergence_pair(const Tile<R> &tl, const R *c0, const R *a0, int i, R &Fx, R &Fy,
                                                R &M0, R &gx, R &gy)
{
    const int ex = i % 3 - 1, ey = i / 3 - 1;
    const R *a = c0 + (ey * tl.RW + ex) * KQW, *b = c0 - (ey * tl.RW + ex) * KQW;
    const R w = (ex != 0 && ey != 0) ? wst<R>(1, 1) : wst<R>(1, 0);
    const R dxy = a[1] - b[1];
    Fx -= R(3) * w * (R(ex) * (a[0] - b[0]) + R(ey) * dxy);
    Fy -= R(3) * w * (R(ex) * dxy + R(ey) * (a[2] - b[2]));
    M0 += R(6) * w * (R(ex) * (a[3] - b[3]) + R(ey) * (a[4] - b[4]));
    const R dr = a0[(ey * tl.WT + ex) * AUXW] - a0[-(ey * tl.WT + ex) * AUXW];
    gx += R(3) * w * R(ex) * dr;
    gy += R(3) * w * R(ey) * dr;
}

// Relative change of the gauge by a corrector's results o, in the gauge (th, sr = sqrt th).
template <typename R>
__device__ __forceinline__ float gauge_change(const EosOut<R> &o, R th, R sr)
{
    const float rth = fabsf((float)o.dth) / (float)th;
    const float rux = fabsf((float)o.dux) / (float)sr, ruy = fabsf((float)o.duy) / (float)sr;
    return fmaxf(rth, fmaxf(rux, ruy));
}

// Stop rules of the frame search: converged, and (FP32 form only) stalled: the streamed
// moments carry FP32 rounding that the EoS cancellation inside interfaces can lift above
// tol; once a corrector no longer halves the residual the iteration has reached that floor
// and stops.  Only a residual within STALL_TOL_FACTOR x tol counts as that floor: a larger
// one that fails to halve once (the pressure floor's kink in theta* = max(p, p_floor)/(rho
// T_L) can do that) keeps iterating, since stopping there left the gauge up to 8 % off and
// single steps 3.6e-3 off the converged result inside a compressed sub-spinodal droplet.
template <typename R>
__device__ __forceinline__ void stop_rules(const DevParams &p, float res, float last, unsigned its, bool &conv,
                                           bool &stall)
{
    conv = sizeof(R) == 4 ? res <= p.tol_f : (double)res <= p.tol;
    stall = sizeof(R) == 4 && its >= 2 && !conv && res > 0.5f * last && res < STALL_TOL_FACTOR * p.tol_f;
}

// One time step of one tile, one thread per node.  FAR (FP64): with the wider halo, apart
// from the common form, whose registers and code it would burden.
__device__ __noinline__ void step_tile_far(const DevParams &p, const double *__restrict__ in, double *__restrict__ out,
                                           DevStats *stats, int tile_idx, const double *nlsrc, double *smem);
template <typename R, bool FAR>
__device__ __forceinline__ void step_tile(const DevParams &p, const R *__restrict__ in, R *__restrict__ out,
                                          DevStats *stats, int tile_idx, const R *nlsrc, R *smem)
{
    constexpr int DS = Slot<R>::stride;
    const TypedParams<R> &q = typed<R>(p);
    const size_t N = (size_t)p.N;
    const int tid = threadIdx.x;
    __shared__ StepCounts counts;
    Tile<R> tl(p, tile_idx, smem);
    if constexpr (FAR) tl.set_halo(HALO_FAR);
    R gb[3];
    const R dt = stage_tile<R>(p, in, nlsrc, tl, counts, gb);
    if constexpr (sizeof(R) == 8 && !FAR)
        if (dt == R(0)) {
            step_tile_far(p, in, out, stats, tile_idx, nlsrc, smem);
            return;
        }
    const int tx = tid % tl.TX, ty = tid / tl.TX;
    const int X = tl.X0 + tx, Y = tl.Y0 + ty;
    const bool valid = ty < tl.TY && X < p.nx && Y < p.ny;   // (a tile may have fewer nodes than threads)
    R *keep = tl.rest + tid;   // this thread's column
    const int slot = tl.slot(tx, ty);
    unsigned its = 0, nreg = 0, npair = 0;
    bool conv = true, stall = false, floored = false, bad = false;
    if (valid) {
        R Fx = 0, Fy = 0, M0 = 0, gxn = 0, gyn = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            divergence_pair<R>(tl, tl.kq + ((ty + 1) * tl.RW + tx + 1) * KQW, tl.aux + slot * AUXW, i, Fx, Fy, M0, gxn, gyn);
        keep[K_F * STEP_THREADS] = Fx;
        keep[(K_F + 1) * STEP_THREADS] = Fy;
        keep[K_REL * STEP_THREADS] = R(0.5) * q.kappa * (gxn * gxn + gyn * gyn);
        keep[K_M0 * STEP_THREADS] = M0;
        // exact sums of the node's stored populations (error-free in R: TwoSum cascades,
        // each sum an unevaluated (hi, lo) pair); the stored low parts start the error terms
        const size_t n = (size_t)Y * p.nx + X;
        R th, ux, uy;
        {
            R hi[4] = {R(0), R(0), R(0), R(0)}, lo[4];
            R v[24];
            load_rec24(in, n, N, v);
            lo[0] = __ldg(in + rec_at(in, n, P_F4LO, N));
            lo[1] = __ldg(in + rec_at(in, n, P_JXLO, N));
            lo[2] = __ldg(in + rec_at(in, n, P_JYLO, N));
            lo[3] = __ldg(in + rec_at(in, n, P_G4LO, N));
            th = v[P_TH]; ux = v[P_UX]; uy = v[P_UY];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const R f = v[P_F + i];
                const R terms[4] = {f, R(i % 3 - 1) * f, R(i / 3 - 1) * f, v[P_G + i]};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (k == 1 && i % 3 == 1) continue;
                    if (k == 2 && i / 3 == 1) continue;
                    R e;
                    two_sum_(hi[k], terms[k], hi[k], e);
                    lo[k] += e;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                keep[(K_HI + k) * STEP_THREADS] = hi[k];
                keep[(K_LO + k) * STEP_THREADS] = lo[k];
            }
        }

        // ---------------- phase 1: frame search -------------------------------------
        R inc[2][9];
        EosOut<R> o;
        float last = 3.0e38f;   // previous residual
        for (;;) {
            ++its;
            stream_node<R, FAR>(p, in, X, Y, tl.slots + (size_t)slot * DS, tl.WT, gb, dt, th, ux, uy, its == 1, keep, inc,
                                nreg, npair);
            R sum[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                sum[0] += inc[0][i];
                if (i % 3 == 0) sum[1] -= inc[0][i];
                if (i % 3 == 2) sum[1] += inc[0][i];
                if (i / 3 == 0) sum[2] -= inc[0][i];
                if (i / 3 == 2) sum[2] += inc[0][i];
                sum[3] += inc[1][i];
            }
            const R lam[3] = {th, ux, uy};
            const R sr = sqrt_(th);
            R hi[4], lo[4], nl[3];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                hi[k] = keep[(K_HI + k) * STEP_THREADS];
                lo[k] = keep[(K_LO + k) * STEP_THREADS];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) nl[k] = keep[(K_F + k) * STEP_THREADS];
            eos_update(p, hi, lo, sum, nl, lam, sr, o);
            const float res = gauge_change<R>(o, th, sr);
            stop_rules<R>(p, res, last, its, conv, stall);
            last = res;
            if (conv || stall || !(res == res) || its >= (unsigned)p.max_iter) break;
            th = o.ths; ux = o.uxs; uy = o.uys;
        }
        conv = conv || stall;

        // ---------------- phase 2: collision ----------------------------------------
        R rec[SL];
        {
            R v[24], ft[9], gt[9];
            load_rec24(in, n, N, v);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                ft[i] = v[P_F + i] + inc[0][i];
                gt[i] = v[P_G + i] + inc[1][i];
            }
            collide<R>(q, o, th, ux, uy, keep[K_F * STEP_THREADS], keep[(K_F + 1) * STEP_THREADS],
                       keep[K_M0 * STEP_THREADS], ft, gt, rec);
        }
        store_chunks<SL>(out, n, N, rec);
        floored = o.pr < q.p_floor;
        bad = !(o.rho_hi == o.rho_hi) || !(o.T == o.T) || isinf(o.rho_hi) || isinf(o.T);
    }
    add_counts(counts, stats, its, nreg, npair, !conv, stall, floored, bad);
}

// ---------------------------------------------------------------------------
// Nine lanes per node, for grids too small to fill the GPU with one thread per node.
// Lane e = 3 n + k of a node first sums the stream's partial of direction component k over
// the source index n (an x pass of 20 slots x 3 values and a y pass onto l = 0..2), three
// lanes exchange so that lane e = 3 l + k holds the increments of population e, and the
// collision then runs one population per lane.  Three nodes per warp; lanes 27..31 repeat
// lanes 18..22.  All lanes of a node compute the moments and the EoS from the same values
// in the same order, so they agree bitwise.
template <typename R>
__device__ __forceinline__ R grp(R v, int base, int e) { return __shfl_sync(0xffffffffu, v, base + e); }

// Error-free sums over a node's nine lanes of (f, f c_x, f c_y, g) as (hi, lo) pairs, the
// same bits in every lane: rows first, then the three rows.
template <typename R>
__device__ __forceinline__ void lane_sums(R f, R g, int base, int l, R (&hi)[4], R (&lo)[4])
{
    const int r = base + 3 * l;
    const R f0 = grp(f, r, 0), f1 = grp(f, r, 1), f2 = grp(f, r, 2);
    const R g0 = grp(g, r, 0), g1 = grp(g, r, 1), g2 = grp(g, r, 2);
    R e, S, Sl, D, Dl, G, Gl;
    two_sum_(f0, f1, S, e); Sl = e;
    two_sum_(S, f2, S, e); Sl += e;
    two_sum_(f2, -f0, D, Dl);
    two_sum_(g0, g1, G, e); Gl = e;
    two_sum_(G, g2, G, e); Gl += e;
    auto fold = [&](R v, R vl, R &h, R &w) {
        const R a = grp(v, base, 0), b = grp(v, base, 3), c = grp(v, base, 6);
        const R al = grp(vl, base, 0), bl = grp(vl, base, 3), cl = grp(vl, base, 6);
        R e1, e2;
        two_sum_(a, b, h, e1);
        two_sum_(h, c, h, e2);
        w = (al + bl) + cl + (e1 + e2);
    };
    fold(S, Sl, hi[0], lo[0]);
    fold(D, Dl, hi[1], lo[1]);
    fold(G, Gl, hi[3], lo[3]);
    const R s0 = grp(S, base, 0), s2 = grp(S, base, 6), s0l = grp(Sl, base, 0), s2l = grp(Sl, base, 6);
    two_sum_(s2, -s0, hi[2], e);
    lo[2] = e + (s2l - s0l);
}

__device__ __noinline__ void step_tile_split_far(const DevParams &p, const double *__restrict__ in,
                                                 double *__restrict__ out, DevStats *stats, int tile_idx,
                                                 const double *nlsrc, double *smem);
template <typename R, bool FAR>
__device__ __forceinline__ void step_tile_split(const DevParams &p, const R *__restrict__ in, R *__restrict__ out,
                                                DevStats *stats, int tile_idx, const R *nlsrc, R *smem)
{
    constexpr int DS = Slot<R>::stride;
    constexpr unsigned ALL = 0xffffffffu;
    const TypedParams<R> &q = typed<R>(p);
    const size_t N = (size_t)p.N;
    __shared__ StepCounts counts;
    Tile<R> tl(p, tile_idx, smem);
    if constexpr (FAR) tl.set_halo(HALO_FAR);
    R gb[3];
    const R dt = stage_tile<R>(p, in, nlsrc, tl, counts, gb);
    if constexpr (sizeof(R) == 8 && !FAR)
        if (dt == R(0)) {
            step_tile_split_far(p, in, out, stats, tile_idx, nlsrc, smem);
            return;
        }

    const int ln = threadIdx.x & 31, lq = ln < 27 ? ln : ln - 9;
    const int base = lq < 9 ? 0 : (lq < 18 ? 9 : 18);
    const int e = lq - base, k = e % 3, l = e / 3;
    const int j = (threadIdx.x >> 5) * 3 + base / 9;
    const int tx = j % tl.TX, ty = j / tl.TX;
    const bool valid = tl.X0 + tx < p.nx && tl.Y0 + ty < p.ny;
    const int X = min(tl.X0 + tx, p.nx - 1), Y = min(tl.Y0 + ty, p.ny - 1);
    const size_t n = (size_t)Y * p.nx + X;
    const int slot = tl.slot(tx, ty);
    const bool writer = ln < 27;
    // the node's own record and the general stream's partials
    R *own = tl.rest + (size_t)j * SPLIT_WORDS, *part = own + SL;
    for (int v = e; v < 30; v += 9)
        if (writer) own[v] = __ldg(in + rec_at(in, n, v, N));
    R Fx = 0, Fy = 0, M0 = 0, rEl;
    {
        R gx = 0, gy = 0;
        if (e < 4)
            divergence_pair<R>(tl, tl.kq + ((ty + 1) * tl.RW + tx + 1) * KQW, tl.aux + slot * AUXW, e, Fx, Fy, M0, gx, gy);
        auto four = [&](R v) { return (grp(v, base, 0) + grp(v, base, 1)) + (grp(v, base, 2) + grp(v, base, 3)); };
        Fx = four(Fx); Fy = four(Fy); M0 = four(M0); gx = four(gx); gy = four(gy);
        rEl = R(0.5) * q.kappa * (gx * gx + gy * gy);
    }
    __syncwarp();
    const R nl[3] = {Fx, Fy, rEl};
    R th = own[P_TH], ux = own[P_UX], uy = own[P_UY];
    const R fe = own[P_F + e], ge = own[P_G + e];
    R hi[4], lo[4];
    lane_sums<R>(fe, ge, base, l, hi, lo);
    lo[0] += own[P_F4LO]; lo[1] += own[P_JXLO]; lo[2] += own[P_JYLO]; lo[3] += own[P_G4LO];
    R dx[6];   // the own slot's values this lane differences against (FP32)
    const R *sl = tl.slots + (size_t)slot * DS;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        dx[m] = sizeof(R) == 4 ? sl[slot_at<R>(0, 3 * l + m)] : R(0);
        dx[3 + m] = sizeof(R) == 4 ? sl[slot_at<R>(1, 3 * l + m)] : R(0);
    }

    // ---------------- phase 1: frame search (warp lockstep) ---------------------------
    unsigned its = 0, nreg = 0, npair = 0;
    bool conv = true, stall = false, active = valid;
    R df = 0, dg = 0;         // increments of population e
    EosOut<R> o{};
    float last = 3.0e38f;
    for (unsigned it = 1; __any_sync(ALL, active); ++it) {
        const R s = sqrt_(th), inv_s = R(1) / s;
        // departure along x of component k, along y of component l; the other y components'
        // weights come from the lanes that hold them
        R wx[4], wy[3][5], Lx[3], Ly[3];
        bool near_x, ok = true;
        {
            auto weights = [&](R v, R (&a)[4]) -> bool {   // true: floor 0, false: floor -1
                const R d = -v * dt;
                const R f = floor(d);
                ok = ok && (f == R(0) || f == R(-1));
                const R t0 = d - f + R(1), t1 = t0 - R(1), t2 = t0 - R(2), t3 = t0 - R(3);
                const R p12 = t1 * t2, p03 = t0 * t3;
                a[0] = p12 * t3 * R(-1.0 / 6.0);
                a[1] = p03 * t2 * R(0.5);
                a[2] = p03 * t1 * R(-0.5);
                a[3] = p12 * t0 * R(1.0 / 6.0);
                return f == R(0);
            };
            near_x = weights(s * R(k - 1) + ux, wx);
            R ya[4];
            const unsigned nym = __ballot_sync(ALL, weights(s * R(l - 1) + uy, ya));
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                R a[4];
#pragma unroll
                for (int j2 = 0; j2 < 4; ++j2) a[j2] = grp(ya[j2], base, 3 * c);
                const bool near = (nym >> (base + 3 * c)) & 1u;
                wy[c][0] = near ? R(0) : a[0];
                wy[c][1] = near ? a[0] : a[1];
                wy[c][2] = near ? a[1] : a[2];
                wy[c][3] = near ? a[2] : a[3];
                wy[c][4] = near ? a[3] : R(0);
            }
        }
        const unsigned okm = __ballot_sync(ALL, ok), nxm = __ballot_sync(ALL, near_x);
        const unsigned gm = 0x1ffu << base;
        bool fast = (okm & gm) == gm;
        R nf = 0, ng = 0;
        {
            // row k of the x map, column n (= l) of the y map
            const R qq = (gb[0] - s) * inv_s, w1 = (gb[1] - ux) * inv_s, w2 = (gb[2] - uy) * inv_s;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const R x = m == 1 ? w1 : (R(1) + qq) * R(m - 1) + w1;
                Lx[m] = k == 1 ? (R(1) - x) * (R(1) + x) : R(0.5) * x * (x + R(k - 1));
            }
            const R y = l == 1 ? w2 : (R(1) + qq) * R(l - 1) + w2;
            Ly[0] = R(0.5) * y * (y - R(1));
            Ly[1] = (R(1) - y) * (R(1) + y);
            Ly[2] = R(0.5) * y * (y + R(1));
            R wl[4][3];
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int m = 0; m < 3; ++m) wl[c][m] = wx[c] * Lx[m];
            R af[3] = {R(0), R(0), R(0)}, ag[3] = {R(0), R(0), R(0)};
            const R *row = sl - (2 * tl.WT + (near_x ? 1 : 2)) * DS + slot_at<R>(0, 3 * l);
            if constexpr (sizeof(R) == 4) {
                // f and g side by side (see contract)
                f32x2 w2[4][3], d2[3], a2[3] = {0ull, 0ull, 0ull};
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    d2[m] = pack2(-dx[m], -dx[3 + m]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) w2[c][m] = pack2(wl[c][m], wl[c][m]);
                }
#pragma unroll
                for (int cy = 0; cy < 5; ++cy, row += tl.WT * DS) {
                    f32x2 t = 0ull;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int m = 0; m < 3; ++m)
                            t = fma2(w2[c][m], add2(reinterpret_cast<const f32x2 *>(row + c * DS)[m], d2[m]), t);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float w = wy[c][cy] * Ly[c];
                        a2[c] = fma2(pack2(w, w), t, a2[c]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) unpack2(a2[c], af[c], ag[c]);
            } else {
#pragma unroll
                for (int cy = 0; cy < 5; ++cy, row += tl.WT * DS) {
                    R tf = 0, tg = 0;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            tf += wl[c][m] * row[c * DS + m];
                            tg += wl[c][m] * row[c * DS + 9 + m];
                        }
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const R w = wy[c][cy] * Ly[c];
                        af[c] += w * tf;
                        ag[c] += w * tg;
                    }
                }
            }
            // lane (k, n) keeps its share of l = n and sends the others to their lanes
            nf = sel3(l, af[0], af[1], af[2]);
            ng = sel3(l, ag[0], ag[1], ag[2]);
#pragma unroll
            for (int r = 1; r < 3; ++r) {
                const int to = (l + 3 - r) % 3, from = (l + r) % 3;
                nf += grp(sel3(to, af[0], af[1], af[2]), base, 3 * from + k);
                ng += grp(sel3(to, ag[0], ag[1], ag[2]), base, 3 * from + k);
            }
        }
        if (sizeof(R) == 8) {
            nf -= fe;
            ng -= ge;
        } else if (it > 1) {
            // the node's own populations carried from their stored gauge into this one
            const R tho = own[P_TH];
            const R qx = fdiv_(tho - th, (sqrt_(tho) + s) * s);
            const R w1 = (own[P_UX] - ux) * inv_s, w2 = (own[P_UY] - uy) * inv_s;
            R Er[3], Ec[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                Er[a] = ell_inc_rt<R>(k, a, qx * R(a - 1) + w1);
                Ec[a] = ell_inc_rt<R>(l, a, qx * R(a - 1) + w2);
            }
#pragma unroll
            for (int fam = 0; fam < 2; ++fam) {
                const R *h = own + 9 * fam;
                R acc = 0;
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const R t = Er[0] * h[3 * b] + Er[1] * h[3 * b + 1] + Er[2] * h[3 * b + 2];
                    acc += Ec[b] * (h[3 * b + k] + t) + (b == l ? t : R(0));
                }
                if (fam == 0) nf += acc;
                else ng += acc;
            }
        }
        unsigned add_reg = 0, add_pair = 0;
        if (fast) {
            const unsigned nx3 = (nxm >> base) & 7u;   // the row l = 0 holds all three components
            const int sx = (nx3 == 0u || nx3 == 7u) ? 4 : 5;
            const R dy0 = floor(-(s * R(-1) + uy) * dt), dy2 = floor(-(s + uy) * dt);
            add_reg = (unsigned)(sx * (dy0 == dy2 ? 4 : 5) - (it == 1 ? 1 : 0));
        }
        if (__any_sync(ALL, active && !fast)) {
            if constexpr (FAR) {
                // departure points within the wider halo: each lane streams its direction
                const FarOne o1 = far_one(sl, tl.WT, k, l, gb[0], gb[1], gb[2], s, inv_s, dt, ux, uy);
                const unsigned rm = __ballot_sync(ALL, o1.ok);
                const int x0 = grp(o1.fx, base, 0), x1 = grp(o1.fx, base, 1), x2 = grp(o1.fx, base, 2);
                const int y0 = grp(o1.fy, base, 0), y1 = grp(o1.fy, base, 3), y2 = grp(o1.fy, base, 6);
                if (!fast && (rm & gm) == gm) {
                    fast = true;
                    nf = o1.f - fe;
                    ng = o1.g - ge;
                    add_reg = (unsigned)((4 + max(x0, max(x1, x2)) - min(x0, min(x1, x2))) *
                                             (4 + max(y0, max(y1, y2)) - min(y0, min(y1, y2))) - (it == 1 ? 1 : 0));
                }
            }
            // departure points beyond the halo: the node's lanes share its stencil nodes
            if (!fast) {
                R buf[18];
                stream_general<R>(p, in, X, Y, th, ux, uy, it == 1, e, 9, buf, add_reg, add_pair);
                if (writer)
#pragma unroll
                    for (int i = 0; i < 18; ++i) part[i * 9 + e] = buf[i];
            }
            __syncwarp();
            if (!fast) {
                nf = ng = R(0);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    nf += part[e * 9 + i];
                    ng += part[(9 + e) * 9 + i];
                }
            }
            __syncwarp();
        }
        // sums of the increments, the same in every lane
        R sum[4];
        {
            const int r = base + 3 * l;
            const R f0 = grp(nf, r, 0), f1 = grp(nf, r, 1), f2 = grp(nf, r, 2);
            const R S = f0 + f1 + f2, D = f2 - f0, G = grp(ng, r, 0) + grp(ng, r, 1) + grp(ng, r, 2);
            const R s0 = grp(S, base, 0), s1 = grp(S, base, 3), s2 = grp(S, base, 6);
            sum[0] = s0 + s1 + s2;
            sum[1] = grp(D, base, 0) + grp(D, base, 3) + grp(D, base, 6);
            sum[2] = s2 - s0;
            sum[3] = grp(G, base, 0) + grp(G, base, 3) + grp(G, base, 6);
        }
        if (active) {
            its = it;
            nreg += add_reg;
            npair += add_pair;
            df = nf;
            dg = ng;
            const R lam[3] = {th, ux, uy};
            const R sr = sqrt_(th);
            eos_update(p, hi, lo, sum, nl, lam, sr, o);
            const float res = gauge_change<R>(o, th, sr);
            stop_rules<R>(p, res, last, it, conv, stall);
            last = res;
            if (conv || stall || !(res == res) || it >= (unsigned)p.max_iter) active = false;
            else { th = o.ths; ux = o.uxs; uy = o.uys; }
        }
    }
    conv = conv || stall;

    // ---------------- phase 2: collision, population e of the node per lane ------------
    // (the formulas of collide(), one population at a time)
    {
        const R s = sqrt_(th), inv_s = R(1) / s;
        const R rr = o.rho_hi, uxr = o.uxs, uyr = o.uys, uhxr = o.uhx, uhyr = o.uhy, Er = o.E;
        const R Pr = o.P, sst = sqrt_(o.ths);
        const R qm1 = sizeof(R) == 8 ? sst * inv_s - R(1) : fdiv_(o.dth, (sst + s) * s);
        const R wsx = o.dux * inv_s, wsy = o.duy * inv_s;
        const R dtr = q.dt, om = q.omega;
        const R irr = frcp_(rr), iP2 = frcp_(R(2) * Pr);
        const R dvx = Fx * dtr * irr * inv_s, dvy = Fy * dtr * irr * inv_s;
        const R W1[3] = {wlat<R>(0), wlat<R>(1), wlat<R>(2)};
        auto row = [&](int kk, R w, R dv, R (&E)[3], R &Ws, R &Wh) {
            Ws = 0;
            Wh = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R ea = qm1 * R(a - 1) + w;
                E[a] = ell_inc_rt<R>(kk, a, ea);
                Ws += E[a] * W1[a];
                Wh += (ell_inc_rt<R>(kk, a, ea + dv) - E[a]) * W1[a];
            }
        };
        R exk[3], eyl[3], Wsk, Wsl, Whk, Whl;
        row(k, wsx, dvx, exk, Wsk, Whk);
        row(l, wsy, dvy, eyl, Wsl, Whl);
        const R H = Er + Pr * irr;
        const R Ixx = R(2) * uhxr * Fx + dtr * Fx * Fx * Er * iP2;
        const R Ixy = uhxr * Fy + Fx * uhyr + dtr * Fx * Fy * Er * iP2;
        const R Iyy = R(2) * uhyr * Fy + dtr * Fy * Fy * Er * iP2;
        const R cM = R(2) * dtr * rr * iP2;
        const R Mx = cM * (Fx * H - (Ixx * uxr + Ixy * uyr));
        const R My = cM * (Fy * H - (Ixy * uxr + Iyy * uyr));
        const R cN = dtr * rr * iP2;
        const R Nxx = rr + cN * Ixx, Nxy = cN * Ixy, Nyy = rr + cN * Iyy;
        const R Pd = sst * sst * (R(2) * W1[0]);
        const R work = R(2) * (uhxr * Fx + uhyr * Fy);
        const R cx = R(k - 1), cy = R(l - 1);
        const R W1k = pick(W1, k), W1l = pick(W1, l), w = W1k * W1l;
        const R ccx = sst * cx, ccy = sst * cy;
        const R Axx = ccx * ccx + R(2) * ccx * uxr - Pd;
        const R Axy = ccx * ccy + ccx * uyr + ccy * uxr;
        const R Ayy = ccy * ccy + R(2) * ccy * uyr - Pd;
        const R geq = w * (R(2) * rr * Er + Mx * ccx + My * ccy + Nxx * Axx + R(2) * Nxy * Axy + Nyy * Ayy);
        const R vx = ccx + uxr, vy = ccy + uyr;
        const R uc = uxr * cx + uyr * cy;
        const R gc = M0 * w * (R(1) + rr * uc * uc * iP2 * R(3) - rr * (vx * vx + vy * vy) * iP2 + R(1));
        const R X_e = om * geq + dtr * (gc + w * work);
        R acc = X_e;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R x0 = grp(X_e, base, 3 * b), x1 = grp(X_e, base, 3 * b + 1), x2 = grp(X_e, base, 3 * b + 2);
            const R t = exk[0] * x0 + exk[1] * x1 + exk[2] * x2;
            acc += eyl[b] * (sel3(k, x0, x1, x2) + t) + (b == l ? t : R(0));
        }
        const R ft = fe + df, gt = ge + dg;
        const R Wx = W1k + Wsk, Wy = W1l + Wsl;
        const R dfeq = (rr * W1k * W1l - ft) + rr * (Wsk * W1l + W1k * Wsl + Wsk * Wsl);
        const R S = rr * (Whk * (Wy + Whl) + Wx * Whl);
        R fo = ft + om * dfeq + S, go = (R(1) - om) * gt + acc;
        R sh[4], sl4[4];
        lane_sums<R>(e == 4 ? R(0) : fo, e == 4 ? R(0) : go, base, l, sh, sl4);
        if (valid && writer) {
            if (e == 4) {
                R t_h, t_l, s1, e1, f4lo, g4lo;
                two_sum_(o.gs_hi, dtr * (M0 + work), t_h, t_l);
                t_l += o.gs_lo;
                two_sum_(o.rho_hi, -sh[0], s1, e1);
                two_sum_(s1, e1 + (o.rho_lo - sl4[0]), fo, f4lo);
                two_sum_(t_h, -sh[3], s1, e1);
                two_sum_(s1, e1 + (t_l - sl4[3]), go, g4lo);
                REC(out, n, P_F4LO) = f4lo;
                REC(out, n, P_G4LO) = g4lo;
                REC(out, n, P_JXLO) = ((o.mx_hi - sh[1]) + (o.mx_lo - sl4[1])) + Fx * dtr * inv_s;
                REC(out, n, P_JYLO) = ((o.my_hi - sh[2]) + (o.my_lo - sl4[2])) + Fy * dtr * inv_s;
            }
            if (e == 0) {
                REC(out, n, P_TH) = th;
                REC(out, n, P_UX) = ux;
                REC(out, n, P_UY) = uy;
                REC(out, n, P_RHO) = rr;
                REC(out, n, P_T) = o.T;
                REC(out, n, P_UHX) = uhxr;
                REC(out, n, P_UHY) = uhyr;
            }
            REC(out, n, P_F + e) = fo;
            REC(out, n, P_G + e) = go;
        }
    }
    const bool one = valid && writer && e == 0;   // one lane reports for the node
    const bool bad = !(o.rho_hi == o.rho_hi) || !(o.T == o.T) || isinf(o.rho_hi) || isinf(o.T);
    add_counts(counts, stats, one ? its : 0, one ? nreg : 0, one ? npair : 0, one && !conv, one && stall,
               one && o.pr < q.p_floor, one && bad);
}

__device__ __noinline__ void step_tile_far(const DevParams &p, const double *__restrict__ in, double *__restrict__ out,
                                           DevStats *stats, int tile_idx, const double *nlsrc, double *smem)
{
    step_tile<double, true>(p, in, out, stats, tile_idx, nlsrc, smem);
}
__device__ __noinline__ void step_tile_split_far(const DevParams &p, const double *__restrict__ in,
                                                 double *__restrict__ out, DevStats *stats, int tile_idx,
                                                 const double *nlsrc, double *smem)
{
    step_tile_split<double, true>(p, in, out, stats, tile_idx, nlsrc, smem);
}

// A simulation as one launch sees it: parameters, the buffers this step reads and writes
// (nlsrc: the state the non-local terms come from) and its counters.
template <typename R>
struct SimDesc {
    DevParams p;
    const R *in;
    R *out;
    DevStats *stats;
    const R *nlsrc;
};

// One time step.  A simulation stepped alone is one block per tile of `one` (work = null);
// a batch's blocks step tile work[b].y of simulation work[b].x of `descs` (a device
// work-list of (simulation, tile) pairs).  Both are this one kernel with the parameters
// in shared memory, so that a context gives bitwise the same result alone and in a batch.
template <typename R, bool SPLIT>
__global__ void __launch_bounds__(STEP_THREADS, SPLIT ? SPLIT_MIN_BLOCKS(R) : STEP_MIN_BLOCKS(R))
    k_pond_step(const __grid_constant__ SimDesc<R> one, const SimDesc<R> *__restrict__ descs,
                const int2 *__restrict__ work)
{
    static_assert(sizeof(SimDesc<R>) % 8 == 0, "copied by 8-byte words");
    __shared__ SimDesc<R> d;
    int tile = blockIdx.x;
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(&one);
    if (work) {
        const int2 w = work[blockIdx.x];
        tile = w.y;
        src = reinterpret_cast<const unsigned long long *>(descs + w.x);
    }
    for (int k = threadIdx.x; k < (int)(sizeof(SimDesc<R>) / 8); k += STEP_THREADS)
        reinterpret_cast<unsigned long long *>(&d)[k] = src[k];
    __syncthreads();
    // the launch may begin while the previous step still runs (its blocks, this far, only
    // copy their descriptor): wait until that step is complete and its memory visible, then
    // let the next one begin
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    extern __shared__ __align__(128) unsigned char step_dyn_smem[];
    R *smem = reinterpret_cast<R *>(step_dyn_smem);
    if constexpr (SPLIT) step_tile_split<R, false>(d.p, d.in, d.out, d.stats, tile, d.nlsrc, smem);
    else step_tile<R, false>(d.p, d.in, d.out, d.stats, tile, d.nlsrc, smem);
}

}  // namespace pond

// lat_common.cuh -- device-side state shared by the lattice kernels: the
// per-lattice constants, the FP64 scalar block that carries a(t) and the
// field-equation coefficients from one step to the next, the deterministic
// block reduction and the scale-factor update of Sec. II.B, eq. scale.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lattice.h"

namespace lat {

// Constants of one lattice, fixed at creation (program units, Sec. II.B).
struct Model {
    int n;
    int expansion;      // 0: static; 1: eq. scale; 2: the L = 1/H form (lat_lform.cu)
    int beta;           // 2 or 4: exponent of the dominant potential term
    int stencil;        // Laplacian: 7-point or 27-point (Sec. II.C)
    int split;          // 1: phi stored as FP64 homogeneous mode + fluctuation arrays
    double dx, dt, inv_dx2;
    // factor turning the stencil's integer-weight neighbour sums into the
    // Laplacian and the gradient average: 1/dx^2 (7-point, weights 1) or
    // 1/(30 dx^2) (27-point, weights 14, 3, 1 for face, edge, corner)
    double lap_scale;
    double A, B, r, s;
    double cdom0, pdom; // V_pr dominant term: cdom0 a^pdom f^beta / beta
    double kappa0, pint;// V_pr interaction: kappa0 a^pint f^2 chi^2 / 2
    double eight_pi_G;
    double g8A2;        // eight_pi_G / A^2 (eq. scale)
    double inv_sites;   // 1 / N^3
    double grad_scale;  // lap_scale / N^3: gradient sums to their averages
    double sp2, ch;     // s + 2, r (s - r + 2) (eq. scale and eq. scalar-evo)
    // the exponents of a in the coefficients (pdom, pint, -2s-2r-1, 2s+2, -2s-2)
    // as integers, valid when intpow is set (every one an integer of at most 16)
    int intpow;
    int e_dom, e_int, e_c, e_v, e_L;
};

// Step coefficients (DevScalars::kd, kf): the kick and drift of eq. scalar-evo
// and eq. evo, and the homogeneous inflaton mode the stored phi arrays are
// measured from (zero unless the lattice stores phi split, see below).
enum {
    kDtCl = 0,   // dt cL / dx^2 (times the stencil's 1/30 for 27 points)
    kDtCf,       // dt cF
    kMDtCdom,    // -dt cdom
    kMDtKap,     // -dt kappa
    kDt,         // dt
    kBg,         // P: homogeneous phi at the field time of the step
    kBg2,        // P^2
    kBgNew,      // P': homogeneous phi at the field time after the step
    kBgNew2,     // P'^2
    kCoefs = 10
};

// FP64 scalars that live on the device between steps. The step kernel reads the
// coefficients at its start and its last block writes those of the next step,
// so a captured CUDA graph of any number of steps needs no host round trip.
//
// Split storage of the inflaton (lat_params.split). phi = P + d with the
// homogeneous mode P (field time) and its momentum Pi (momentum time) kept here
// in FP64, and the arrays of field 0 holding the fluctuation d and its momentum.
// The homogeneous mode follows the same leapfrog with the homogeneous force,
// Pi_{n+1} = Pi_n + dt (cF P - cdom P^(beta-1)), P_{n+3/2} = P + dt Pi_{n+1}, and
// the kernels apply to d the rest of the force exactly:
//   cL Lap d + cF d - [cdom ((P+d)^(beta-1) - P^(beta-1)) + kappa (P+d) chi^2]
// for phi and -kappa (P+d)^2 chi for chi (the homogeneous value of chi stays
// zero: chi is stored whole), written without differences of nearby numbers
// (u = P + d; (u^3 - P^3) = d (u (u + P) + P^2)). The sum of the two parts is
// the same leapfrog step as for phi stored whole, so the scheme is unchanged;
// FP32 arrays then resolve the fluctuations of phi to FP32 precision of their
// own size rather than of phi. P = Pi = 0 is phi stored whole.
struct DevScalars {
    double t;        // program time of the momenta
    double a;        // scale factor at the field time t + dt/2
    double ad;       // a' at t
    double ad_next;  // a' at t + dt, solved from the sums at the field time
    double ad_half;  // a' at the field time, (ad + ad_next)/2
    double add;      // a'' at the field time (eq. scale)
    double S[4];     // <|grad f0|^2>, <|grad f1|^2>, <f0^beta/beta>, <f0^2 f1^2/2>
    double cL, cF;   // a^(-2s-2) and r(s-r+2) h^2 + r a''/a (eq. scalar-evo)
    double cdom, kappa; // potential coefficients at the field time
    long long step;  // parity of the ping-pong buffers = step & 1
    int status;      // sticky lat_status raised on the device
    unsigned int ticket; // last-block counter of the step kernel
    unsigned int ticket2;
    int pad;
    double kd[kCoefs]; // step coefficients (enum above)
    float kf[kCoefs];  // the same rounded once to FP32 for the FP32 kernels
    // History of the scalar blocks (the reverse-mode derivative's forward pass):
    // when set, the last block of each step also stores the block it produces,
    // the one the next step starts from, at log[step - log_base]. Null otherwise.
    DevScalars* log;
    long long log_base;
    // The L = 1/H form (expansion 2): the Hubble length l = a/a' of program time
    // at t, and l at t + dt as solved for the next step (lat_lform.cu).
    double ell, ell_next;
    // Homogeneous inflaton mode of split storage: P at the field time, Pi at the
    // momentum time, and both after the step being taken (zero when phi is
    // stored whole).
    double bgf, bgp, bgf_next, bgp_next;
};

// Step coefficient i for element type T (kd / kf above).
template <typename T>
__device__ __forceinline__ T step_coef(const DevScalars* sc, int i);
template <>
__device__ __forceinline__ float step_coef<float>(const DevScalars* sc, int i) { return sc->kf[i]; }
template <>
__device__ __forceinline__ double step_coef<double>(const DevScalars* sc, int i) { return sc->kd[i]; }

// Number of sums reduced per block: grad^2 of each field (unscaled by 1/dx^2),
// sum f0^beta/beta, sum f0^2 f1^2 / 2.
constexpr int kSums = 4;

// Deterministic reduction of kSums doubles over a block (any block shape; warps
// and lanes follow the linear thread index): a fixed shuffle tree within warps,
// then warp 0 folds the warp totals in warp order. Result valid in thread 0.
// `red` must hold 32 * kSums doubles.
__device__ __forceinline__ int linear_tid()
{
    return threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
}
__device__ __forceinline__ int block_warps() { return (blockDim.x * blockDim.y * blockDim.z + 31) >> 5; }

__device__ __forceinline__ void block_reduce(double v[kSums], double* red)
{
    const int tid = linear_tid(), lane = tid & 31, warp = tid >> 5;
    const int nwarps = block_warps();
#pragma unroll
    for (int k = 0; k < kSums; k++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (lane == 0)
        for (int k = 0; k < kSums; k++) red[warp * kSums + k] = v[k];
    __syncthreads();
    if (warp == 0) {
        for (int k = 0; k < kSums; k++) v[k] = lane < nwarps ? red[lane * kSums + k] : 0.0;
#pragma unroll
        for (int k = 0; k < kSums; k++)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    }
    __syncthreads();
}

// Block reduction of FP32 per-thread sums: a fixed FP32 shuffle tree within
// each warp (32 terms, relative rounding error a few FP32 ulp, far below that
// of the per-thread accumulations), then warp 0 folds the warp totals in FP64 in
// warp order. FP64 arithmetic runs at a small fraction of the FP32 rate, so
// only one warp of the block touches it. Result in out[] of thread 0.
__device__ __forceinline__ void block_reduce(float v[kSums], double* red, double out[kSums])
{
    const int tid = linear_tid(), lane = tid & 31, warp = tid >> 5;
    const int nwarps = block_warps();
#pragma unroll
    for (int k = 0; k < kSums; k++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < kSums; k++) red[warp * kSums + k] = (double)v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < kSums; k++) {
            double w = lane < nwarps ? red[lane * kSums + k] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
            out[k] = w;
        }
    }
}

// FP64 per-thread sums: block_reduce above in FP64 throughout.
__device__ __forceinline__ void block_reduce(double v[kSums], double* red, double out[kSums])
{
    block_reduce(v, red);
#pragma unroll
    for (int k = 0; k < kSums; k++) out[k] = v[k];
}

// The start of a kernel launched by launch_chained: everything the kernels before
// it wrote is visible after this, and the kernel after it may now be set up on
// the SMs that this one leaves. Nothing the stream's earlier work writes is read
// before it; what needs the launch arguments alone (the tile geometry) goes
// before.
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// a^p. The exponents of the two models' rescalings (Sec. II.B) are integers
// for which repeated multiplication of a (or of inv_a = 1/a for negative p) is
// exact to a few ulp and costs a handful of FP64 multiplies instead of a
// general pow, or a division, on the slow FP64 pipe.
__device__ inline double apow(double a, double inv_a, double p)
{
    if (p == rint(p) && fabs(p) <= 16.0) {
        int e = (int)fabs(p);
        double r = 1.0, b = p < 0.0 ? inv_a : a;
        while (e) {
            if (e & 1) r *= b;
            b *= b;
            e >>= 1;
        }
        return r;
    }
    return pow(a, p);
}

// <f0^beta>/beta of the homogeneous mode alone: the potential sums of split
// storage hold the rest, sum over sites of ((P+d)^beta - P^beta)/beta.
__host__ __device__ inline double bg_potential(int beta, double P)
{
    const double q = P * P;
    return beta == 4 ? 0.25 * q * q : 0.5 * q;
}

// The per-step coefficients of eq. scalar-evo as the step kernels use them, and
// one leapfrog step of the homogeneous inflaton mode under the same cL, cF,
// cdom (its force is that of the potential at (P, chi = 0)).
__device__ inline void step_coefficients(const Model& M, DevScalars* sc)
{
    const double P = sc->bgf;
    const double force = sc->cdom * (M.beta == 4 ? P * P * P : P);
    sc->bgp_next = sc->bgp + M.dt * (sc->cF * P - force);
    sc->bgf_next = P + M.dt * sc->bgp_next;
    sc->kd[kDtCl] = M.dt * sc->cL * M.lap_scale;
    sc->kd[kDtCf] = M.dt * sc->cF;
    sc->kd[kMDtCdom] = -M.dt * sc->cdom;
    sc->kd[kMDtKap] = -M.dt * sc->kappa;
    sc->kd[kDt] = M.dt;
    sc->kd[kBg] = P;
    sc->kd[kBg2] = P * P;
    sc->kd[kBgNew] = sc->bgf_next;
    sc->kd[kBgNew2] = sc->bgf_next * sc->bgf_next;
    for (int i = 0; i < kCoefs; i++) sc->kf[i] = (float)sc->kd[i];
}

// Scale-factor update of Sec. II.B, eq. scale, with the staggered a':
// a''_{n+1/2} = q a'_{n+1/2}^2 + c, q = -(s+2)/a, a'_{n+1/2} = (a'_n + a'_{n+1})/2,
// c = (8piG/A^2) a^(-2s-2r-1) ((S0+S1)/3 + a^(2s+2) <V_pr>).
// With y = a'_n + a'_{n+1} the implicit update a'_{n+1} = a'_n + dt a''_{n+1/2}
// is (dt q/4) y^2 - y + (2a'_n + dt c) = 0; the root continuous with dt -> 0 is
// y = 2 gamma / (1 + sqrt(1 - 4 alpha gamma)). Then the coefficients of the
// field equation at the field time (eq. scalar-evo, with the f coefficient
// r(s-r+2) h^2 + r a''/a that follows from eq. fe under the rescaling).
__device__ inline void scale_solve(const Model& M, DevScalars* sc)
{
    // one FP64 division (1/a) serves every negative power and quotient below
    const double a = sc->a, ia = 1.0 / a;
    sc->cdom = M.cdom0 * apow(a, ia, M.pdom);
    sc->kappa = M.kappa0 * apow(a, ia, M.pint);
    if (!M.expansion) {
        sc->ad_next = 0.0; sc->ad_half = 0.0; sc->add = 0.0;
        sc->cL = 1.0; sc->cF = 0.0;
        step_coefficients(M, sc);
        return;
    }
    const double vpr = sc->cdom * sc->S[2] + sc->kappa * sc->S[3];
    const double c = M.g8A2 * apow(a, ia, -2.0 * M.s - 2.0 * M.r - 1.0)
                   * ((sc->S[0] + sc->S[1]) * (1.0 / 3.0) + apow(a, ia, 2.0 * M.s + 2.0) * vpr);
    const double q = -(M.s + 2.0) * ia;
    const double alpha = M.dt * q * 0.25;
    const double gamma = 2.0 * sc->ad + M.dt * c;
    const double disc = 1.0 - 4.0 * alpha * gamma;
    if (!(disc >= 0.0) || !isfinite(c)) {
        sc->status = LAT_ENONFINITE;
        return;
    }
    const double y = 2.0 * gamma / (1.0 + sqrt(disc));
    sc->ad_half = 0.5 * y;
    sc->ad_next = y - sc->ad;
    sc->add = q * sc->ad_half * sc->ad_half + c;
    sc->cL = apow(a, ia, -2.0 * M.s - 2.0);
    const double h = sc->ad_half * ia;
    sc->cF = M.r * (M.s - M.r + 2.0) * h * h + M.r * sc->add * ia;
    step_coefficients(M, sc);
}

// The scalars after one step, from those before it and the volume sums S of the
// new fields: a_{n+3/2} = a_{n+1/2} + dt a'_{n+1}, a' <- a'_{n+1}, t += dt, then
// the a' solve and coefficients for the next step (scale_solve). `advance` is
// false for the sums-only pass after initialisation or a state upload. In the
// L = 1/H form the solve for the next step is a pass of its own (its sums need
// the Laplacian of the new fields), launched after this one.
__device__ inline void advance_scalars(const Model& M, DevScalars& s, const double S[kSums], bool advance)
{
    bool finite = true;
    if (advance) {
        if (M.expansion) {
            s.a = s.a + M.dt * s.ad_next;
            s.ad = s.ad_next;
            s.ell = s.ell_next;
        }
        s.bgf = s.bgf_next;
        s.bgp = s.bgp_next;
        s.t = s.t + M.dt;
        s.step = s.step + 1;
    }
    for (int k = 0; k < kSums; k++) {
        finite = finite && isfinite(S[k]);
        s.S[k] = S[k];
    }
    // the potential sums of the kernels are taken about the homogeneous mode
    s.S[2] += bg_potential(M.beta, s.bgf);
    if (!finite) s.status = LAT_ENONFINITE;
    else if (M.expansion != 2) scale_solve(M, &s);
}

// ---- The serial end of a step. GB300's FP64 units take about 64 cycles per
// warp instruction, whatever the number of active lanes and whether or not it
// depends on the one before, and each of an SM's four sub-partitions has its
// own. The update of the scalars between two steps is FP64 throughout, so its
// time is the number of FP64 instructions on its longest path. One thread
// taking the fold and advance_scalars (some 250 instructions) held every other
// SM idle; this form takes 6 to 7 us less per step (32^3 FP64: 31.1 -> 24.9 us,
// 100^3 FP32: 29.0 -> 22.3, 256^3 FP32: 110.4 -> 104.8, 512^3: 729 -> 713). Below, quantities that do not depend on one another sit in the
// lanes of one warp, so that one instruction forms all of them (the five powers
// of a, the coefficients); everything that does not depend on the volume sums
// is formed by another warp (warp 1: another sub-partition) while warp 0 folds
// its block's sums and takes the ticket; and the block partials are folded by
// four warps. What is left after the sums is about 35 instructions.

// A sum with the rounding errors of its additions beside it (two-sum, Knuth): an
// FP32 tree over a warp then loses nothing that FP64 totals would hold, at FP32
// cost. FP64 sums are kept plain.
template <typename A>
struct TreeSum;
template <>
struct TreeSum<float> {
    float s, e;
    __device__ __forceinline__ void init(float v) { s = v; e = 0.0f; }
    __device__ __forceinline__ TreeSum shfl_xor(int o) const
    {
        return TreeSum{__shfl_xor_sync(0xffffffffu, s, o), __shfl_xor_sync(0xffffffffu, e, o)};
    }
    __device__ __forceinline__ void add(TreeSum b)
    {
        const float t = __fadd_rn(s, b.s), bb = __fsub_rn(t, s);
        e = e + b.e + __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(b.s, bb));
        s = t;
    }
    __device__ __forceinline__ void store(double* red, int warp, int k) const
    {
        float* r = reinterpret_cast<float*>(red);   // 32 kSums totals, then their errors
        r[warp * kSums + k] = s;
        r[(32 + warp) * kSums + k] = e;
    }
    static __device__ __forceinline__ double fold(const double* red, int nrows, int j, int k)
    {
        const float* r = reinterpret_cast<const float*>(red);
        double t = 0.0;
        float e = 0.0f;
        for (; j < nrows; j += 8) {
            t += (double)r[j * kSums + k];
            e += r[(32 + j) * kSums + k];
        }
        return t + (double)e;
    }
};
template <>
struct TreeSum<double> {
    double s;
    __device__ __forceinline__ void init(double v) { s = v; }
    __device__ __forceinline__ TreeSum shfl_xor(int o) const { return TreeSum{__shfl_xor_sync(0xffffffffu, s, o)}; }
    __device__ __forceinline__ void add(TreeSum b) { s += b.s; }
    __device__ __forceinline__ void store(double* red, int warp, int k) const { red[warp * kSums + k] = s; }
    static __device__ __forceinline__ double fold(const double* red, int nrows, int j, int k)
    {
        double t = 0.0;
        for (; j < nrows; j += 8) t += red[j * kSums + k];
        return t;
    }
};

// The four sums over a warp: each of the first two exchanges halves the number
// of sums a lane carries, so 6 additions take the place of 20. Every lane ends
// with the total of sum (lane & 3).
template <typename A>
__device__ __forceinline__ TreeSum<A> warp_sum4(const TreeSum<A> v[kSums])
{
    const int lane = linear_tid() & 31;
    const bool b0 = lane & 1, b1 = lane & 2;
    TreeSum<A> k0 = b0 ? v[1] : v[0], k1 = b0 ? v[3] : v[2];
    const TreeSum<A> s0 = b0 ? v[0] : v[1], s1 = b0 ? v[2] : v[3];
    k0.add(s0.shfl_xor(1));
    k1.add(s1.shfl_xor(1));
    TreeSum<A> r = b1 ? k1 : k0;
    r.add((b1 ? k0 : k1).shfl_xor(2));
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) r.add(r.shfl_xor(o));
    return r;
}

template <typename A>
__device__ __forceinline__ TreeSum<A> warp_sum4(const A v[kSums])
{
    TreeSum<A> t[kSums];
#pragma unroll
    for (int k = 0; k < kSums; k++) t[k].init(v[k]);
    return warp_sum4<A>(t);
}

// The warps' totals over a block, by one warp: every lane ends with the total of
// sum (lane & 3), added in a fixed order in FP64.
template <typename A>
__device__ __forceinline__ double warp_fold4(const double* red, int nwarps)
{
    const int lane = linear_tid() & 31;
    double r = TreeSum<A>::fold(red, nwarps, lane >> 2, lane & 3);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// The partials of all blocks in device memory, folded by the first
// `warps` (at most 4) warps of the block; warp w of them returns the share of
// rows w * 8 + lane / 4 + 8 warps i.
__device__ __forceinline__ double warp_fold_partials(const double* partials, int nblocks, int warp, int warps)
{
    const int lane = linear_tid() & 31, step = 8 * warps;
    const double* p = partials + (lane & 3);
    double r = 0.0;
    int j = 8 * warp + (lane >> 2);
    for (; j + 4 * step < nblocks; j += 5 * step) {   // five loads in flight
        double x[5];
#pragma unroll
        for (int i = 0; i < 5; i++) x[i] = __ldcg(p + (size_t)(j + i * step) * kSums);
#pragma unroll
        for (int i = 0; i < 5; i++) r += x[i];
    }
    double x[5];
#pragma unroll
    for (int i = 0; i < 5; i++) x[i] = j + i * step < nblocks ? __ldcg(p + (size_t)(j + i * step) * kSums) : 0.0;
#pragma unroll
    for (int i = 0; i < 5; i++)
        if (j + i * step < nblocks) r += x[i];
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// What the update of the scalars needs beyond the scalar block itself.
struct ScalePre {
    double ia, ria;    // 1/a, r/a at the new field time
    double eb, kea;    // a^(2s+2), (8piG/A^2) a^(-2s-2r-1)
    double q, dtq;     // -(s+2)/a, dt q
    double bgpot;      // the homogeneous mode's potential term of S[2]
    double force;      // cdom P^(beta-1)
};

// The part of advance_scalars and scale_solve that does not depend on the volume
// sums, for one warp: from the block the step started with (img, in shared
// memory) its values at the new field time, cdom, kappa, cL and the step
// coefficients that follow from them alone, and pre. Same formulas and, but for
// products of constants, the same rounding as the one-thread forms.
__device__ inline void scale_pre_warp(const Model& M, DevScalars& img, ScalePre& pre, bool advance)
{
    const int lane = linear_tid() & 31;
    double a = img.a, ad = img.ad, ell = img.ell, P = img.bgf, Pi = img.bgp, t = img.t;
    if (advance) {
        if (M.expansion) {
            a = a + M.dt * img.ad_next;
            ad = img.ad_next;
            ell = img.ell_next;
        }
        P = img.bgf_next;
        Pi = img.bgp_next;
        t = t + M.dt;
    }
    double P2 = 0.0, P3 = 0.0, bgpot = 0.0;
    if (M.split) {
        P2 = P * P;
        P3 = M.beta == 4 ? P2 * P : P;
        bgpot = bg_potential(M.beta, P);
    }
    __syncwarp();
    if (lane == 0) {
        img.a = a;
        img.ad = ad;
        img.ell = ell;
        img.bgf = P;
        img.bgp = Pi;
        img.t = t;
        img.step = img.step + (advance ? 1 : 0);
        img.ticket = 0u;
        pre.bgpot = bgpot;
    }
    if (M.expansion != 2) {   // the L = 1/H form solves in its own pass
        // lanes 0..6: a^pdom, a^pint, a^(-2s-2r-1), a^(2s+2), a^(-2s-2), 1/a, 1/a
        const double ia = 1.0 / a;
        double w;
        if (M.intpow) {
            int e = lane == 0 ? M.e_dom : lane == 1 ? M.e_int : lane == 2 ? M.e_c : lane == 3 ? M.e_v : lane == 4 ? M.e_L : 0;
            double b = e < 0 ? ia : a;
            w = lane >= 5 ? ia : 1.0;
            int m = e < 0 ? -e : e;
            while (true) {
                if (m & 1) w *= b;
                m >>= 1;
                if (!__any_sync(0xffffffffu, m)) break;
                b *= b;
            }
        } else {
            const double p = lane == 0 ? M.pdom : lane == 1 ? M.pint : lane == 2 ? -2.0 * M.s - 2.0 * M.r - 1.0
                             : lane == 3 ? 2.0 * M.s + 2.0 : -2.0 * M.s - 2.0;
            w = lane >= 5 ? ia : apow(a, ia, p);
        }
        if (!M.expansion && lane == 4) w = 1.0;   // cL of static space
        // cdom, kappa, (8piG/A^2) a^(-2s-2r-1), a^(2s+2), cL, -(s+2)/a, r/a
        w = w * (lane == 0 ? M.cdom0 : lane == 1 ? M.kappa0 : lane == 2 ? M.g8A2 : lane == 5 ? -M.sp2 : lane == 6 ? M.r : 1.0);
        // -dt cdom, -dt kappa, ., ., dt cL times the Laplacian's factor, dt q
        double k = w * (lane < 2 ? -M.dt : M.dt);
        k = k * (lane == 4 ? M.lap_scale : 1.0);
        const double force = __shfl_sync(0xffffffffu, w, 0) * P3;
        if (lane == 2) k = M.dt;
        if (lane == 3) k = P;
        if (lane == 6) k = P2;
        const float kf = (float)k;
        if (lane == 0) {
            img.cdom = w;
            pre.ia = ia;
            pre.force = force;
        }
        if (lane == 1) img.kappa = w;
        if (lane == 2) pre.kea = w;
        if (lane == 3) pre.eb = w;
        if (lane == 4) img.cL = w;
        if (lane == 5) {
            pre.q = w;
            pre.dtq = k;
        }
        if (lane == 6) pre.ria = w;
        if (lane < 7 && lane != 5) {
            const int i = lane == 0 ? kMDtCdom : lane == 1 ? kMDtKap : lane == 2 ? kDt : lane == 3 ? kBg
                          : lane == 4 ? kDtCl : kBg2;
            img.kd[i] = k;
            img.kf[i] = kf;
        }
    }
    __syncwarp();
}

// y = a'_n + a'_{n+1}, the root of (dt q/4) y^2 - y + gamma = 0 that is continuous
// with dt -> 0, 2 gamma / (1 + sqrt(1 - dt q gamma)); dtq = dt q. Away from the
// double root an FP32 evaluation of that form is taken to FP64 by two Newton
// steps (the second starts at about 1e-14 and leaves the rounding of the
// residual, about an ulp of y): 9 FP64 instructions in place of the 20 of an
// FP64 square root and division. disc = 1 - dt q gamma. Error against 128-bit
// arithmetic over 2 10^6 draws of gamma and dt q: rms 7.9e-17 and at most 2.2e-16 of y
// (the square root and division: 9.8e-17 and 3.0e-16); nearer the double root 6.4e-17
// (6.9e-17 to 8.4e-17).
__device__ inline double scale_root(double dtq, double gamma, double disc)
{
    const float gf = (float)gamma, af = 0.25f * (float)dtq;
    const float yf = 2.0f * gf / (1.0f + sqrtf(1.0f - 4.0f * af * gf));
    if (disc >= 0.25 && disc <= 4.0 && fabsf(gf) >= 1e-30f && fabsf(gf) <= 1e30f) {
        const double inv = (double)(1.0f / (1.0f - 2.0f * af * yf)), alpha = 0.25 * dtq;
        double y = (double)yf;
        y = fma(fma(fma(alpha, y, -1.0), y, gamma), inv, y);
        y = fma(fma(fma(alpha, y, -1.0), y, gamma), inv, y);
        return y;
    }
    return 2.0 * gamma / (1.0 + sqrt(disc));
}

__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// The rest of the update, for one warp, from the raw volume sums of the new
// fields (lane l holds sum l & 3): img ends as advance_scalars leaves the
// scalar block.
__device__ inline void scale_finish_warp(const Model& M, DevScalars& img, const ScalePre& pre, double raw)
{
    const int lane = linear_tid() & 31, k4 = lane & 3;
    double S = raw * (k4 < 2 ? M.grad_scale : M.inv_sites);
    const bool finite = __all_sync(0xffffffffu, finite_bits(S));
    // the potential sums of the kernels are taken about the homogeneous mode
    if (M.split) S += k4 == 2 ? pre.bgpot : 0.0;
    if (lane < kSums) img.S[lane] = S;
    if (!finite) {
        if (lane == 0) img.status = LAT_ENONFINITE;
        __syncwarp();
        return;
    }
    if (M.expansion == 2) {
        __syncwarp();
        return;
    }
    double cF = 0.0, half = 0.0, next = 0.0, add = 0.0;
    if (M.expansion) {
        const double S0 = __shfl_sync(0xffffffffu, S, 0), S1 = __shfl_sync(0xffffffffu, S, 1);
        const double S2 = __shfl_sync(0xffffffffu, S, 2), S3 = __shfl_sync(0xffffffffu, S, 3);
        const double vpr = img.cdom * S2 + img.kappa * S3;
        const double c = pre.kea * ((S0 + S1) * (1.0 / 3.0) + pre.eb * vpr);
        const double ad = img.ad;
        const double gamma = (ad + ad) + M.dt * c;
        const double disc = 1.0 - pre.dtq * gamma;
        if (!(disc >= 0.0) || !finite_bits(c)) {
            if (lane == 0) img.status = LAT_ENONFINITE;
            __syncwarp();
            return;
        }
        const double y = scale_root(pre.dtq, gamma, disc);
        half = 0.5 * y;
        next = y - ad;
        add = (pre.q * half) * half + c;
        const double h = half * pre.ia;
        cF = (M.ch * h) * h + pre.ria * add;
    }
    double k = M.dt * cF, bgf = 0.0, bgp = 0.0;   // lanes 0..2: dt cF, P', P'^2
    if (M.split) {
        bgp = img.bgp + M.dt * (cF * img.bgf - pre.force);
        bgf = img.bgf + M.dt * bgp;
    }
    const double bgf2 = bgf * bgf;
    if (lane == 1) k = bgf;
    if (lane == 2) k = bgf2;
    const float kf = (float)k;
    if (lane < 3) {
        const int i = lane == 0 ? kDtCf : lane == 1 ? kBgNew : kBgNew2;
        img.kd[i] = k;
        img.kf[i] = kf;
    }
    if (lane == 0) {
        img.cF = cF;
        img.ad_half = half;
        img.ad_next = next;
        img.add = add;
        img.bgp_next = bgp;
        img.bgf_next = bgf;
    }
    __syncwarp();
}

constexpr int kScalarWords = (int)(sizeof(DevScalars) / 8);
static_assert(sizeof(DevScalars) % 8 == 0, "the scalar block is copied in 8-byte words");

// The scalar block between device and shared memory, by one warp. Reads go
// through L2: the block may have been written earlier in the same launch.
__device__ __forceinline__ void scalars_to_shared(DevScalars& img, const DevScalars* sc)
{
    const unsigned long long* s = reinterpret_cast<const unsigned long long*>(sc);
    unsigned long long* d = reinterpret_cast<unsigned long long*>(&img);
    for (int i = linear_tid() & 31; i < kScalarWords; i += 32) d[i] = __ldcg(s + i);
}
__device__ __forceinline__ void scalars_from_shared(DevScalars* sc, const DevScalars& img)
{
    const unsigned long long* s = reinterpret_cast<const unsigned long long*>(&img);
    unsigned long long* d = reinterpret_cast<unsigned long long*>(sc);
    for (int i = linear_tid() & 31; i < kScalarWords; i += 32) d[i] = s[i];
}

// One more ticket of the launch; the writes of this thread, and those that a
// barrier ordered before it, are visible to the thread that takes the last.
__device__ __forceinline__ unsigned int take_ticket(unsigned int* ticket)
{
    unsigned int t;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(ticket) : "memory");
    return t;
}

// The block's sums into its partials and its ticket (warp 0), and while that is
// on its way `meanwhile` (warp 1, or warp 0 itself in a block of one warp). True
// in every thread of the block that finished last; `red` (32 kSums doubles) is
// free again then. `before` runs on warp 1 ahead of the block's ticket.
// V: the element type A or TreeSum<A>.
template <typename A, typename V, typename Before, typename Meanwhile>
__device__ __forceinline__ bool block_ticket(const V v[kSums], double* red, double* partials, unsigned int* ticket,
                                             Before before, Meanwhile meanwhile)
{
    const int nblocks = gridDim.x * gridDim.y * gridDim.z;
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const int tid = linear_tid(), lane = tid & 31, warp = tid >> 5, nwarps = block_warps();
    const int helper = nwarps > 1 ? 1 : 0;
    __shared__ unsigned int is_last;
    if (warp == helper) before();
    const TreeSum<A> r = warp_sum4<A>(v);
    if (lane < kSums) r.store(red, warp, lane);
    __syncthreads();
    if (warp == 0) {
        const double s = warp_fold4<A>(red, nwarps);
        if (lane < kSums) partials[(size_t)bid * kSums + lane] = s;
        __syncwarp();
        if (lane == 0) is_last = take_ticket(ticket) == (unsigned int)nblocks - 1u;
    }
    if (warp == helper) meanwhile();
    __syncthreads();
    return is_last != 0u;
}

// All blocks' partials folded by the last block (every thread calls): the total
// of sum (lane & 3) in every lane of warp 0.
__device__ __forceinline__ double last_block_fold(const double* partials, double* red)
{
    const int nblocks = gridDim.x * gridDim.y * gridDim.z;
    const int tid = linear_tid(), lane = tid & 31, warp = tid >> 5;
    const int warps = block_warps() < 4 ? block_warps() : 4;
    if (warp < warps) {
        const double s = warp_fold_partials(partials, nblocks, warp, warps);
        if (lane < kSums) red[warp * kSums + lane] = s;
    }
    __syncthreads();
    double r = 0.0;
    if (warp == 0)
        for (int w = 0; w < warps; w++) r += red[w * kSums + (lane & 3)];
    return r;
}

// Write this block's partial sums, and let the last block of the launch fold
// all partials and advance the FP64 scalars: a_{n+3/2} = a_{n+1/2} + dt a'_{n+1},
// then the a' solve and coefficients for the next step. `advance` is false for
// the sums-only pass that follows initialisation or a state upload. The
// per-thread sums are float (FP32 kernels) or double.
template <typename A, typename V>
__device__ inline void finish_block_sums_of(const Model& M, DevScalars* sc, double* partials, const V* v, double* red,
                                            bool advance)
{
    __shared__ DevScalars img;
    __shared__ ScalePre pre;
    // the scalar block is read before this block's ticket: only the last block,
    // when every other has taken its own, rewrites it
    if (!block_ticket<A>(v, red, partials, &sc->ticket, [&]() { scalars_to_shared(img, sc); },
                      [&]() { scale_pre_warp(M, img, pre, advance); }))
        return;
    const double raw = last_block_fold(partials, red);
    if (linear_tid() >= 32) return;
    scale_finish_warp(M, img, pre, raw);
    scalars_from_shared(sc, img);
    if (advance && img.log) scalars_from_shared(img.log + (img.step - img.log_base), img);
}

template <typename A>
__device__ inline void finish_block(const Model& M, DevScalars* sc, double* partials, A v[kSums], double* red,
                                    bool advance)
{
    finish_block_sums_of<A>(M, sc, partials, v, red, advance);
}
// the same from sums that carry their rounding errors
template <typename A>
__device__ inline void finish_block_trees(const Model& M, DevScalars* sc, double* partials, const TreeSum<A> v[kSums],
                                          double* red, bool advance)
{
    finish_block_sums_of<A>(M, sc, partials, v, red, advance);
}

// As finish_block, for a domain that is part of a larger lattice (a z-slab):
// the last block writes the domain's share of the volume averages (sums over
// its sites / N^3) to sums_out and leaves the scalars alone; the scalars advance
// once the shares of every domain are added (advance_scalars).
template <typename A>
__device__ inline void finish_block_sums(const Model& M, DevScalars* sc, double* partials, A v[kSums], double* red,
                                         double* sums_out)
{
    if (!block_ticket<A>(v, red, partials, &sc->ticket, []() {}, []() {})) return;
    const double raw = last_block_fold(partials, red);
    const int tid = linear_tid();
    if (tid < kSums) sums_out[tid] = raw * (tid < 2 ? M.grad_scale : M.inv_sites);
    if (tid == 0) sc->ticket = 0u;
}

} // namespace lat

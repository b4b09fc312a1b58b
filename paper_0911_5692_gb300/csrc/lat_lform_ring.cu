// lat_lform_ring.cu -- the sums pass of the L = 1/H form (lat_lform.cu) in FP32,
// 7 and 27 points, over the plane ring of the step kernels (lat_xw.cuh).
//
// Per site the pass reads the four state arrays once and forms v = u + w0 f of
// lat_lform.cu, with the sums P0, Q, F2 and W; the last block solves for the next
// step's coefficients. What bounds it: the reads (40 us at 256^3 at the copy rate,
// and the step's writes still in L2 go out meanwhile: 330 MB in all; 512^3 moves 6.0
// TB/s) and what is serial around them. A vector per thread and plane with its
// neighbours through L1 took 94 us at 256^3 (27 points, a site per thread: 430),
// its 2 x 8 warps waiting for loads and some 12 us of one thread's FP64 before the
// first load and after the last. Here tiles of 32 vectors by 8 rows march along z,
// two planes in flight, two blocks to an SM (16 rows, one block: 76 us for 72): a
// warp owns two rows and carries centres and z differences in registers; one more
// warp stages the halo rows and the columns beside the tile. Runs go down in z, so
// that they start with the planes the step wrote last. The powers of a are formed
// in the lanes of that warp while the first planes are on their way, the unknowns
// are first iterated in FP32, and the coefficients are written by lanes. Step and
// pass together: 256^3 207 -> 170 us, 512^3 1264 -> 1090, 100^3 50 -> 32, 32^3 32
// -> 21; 27 points 256^3 582 -> 209, 100^3 96 -> 38.
#include <algorithm>

#include "lat_agg27.cuh"
#include "lat_async.cuh"
#include "lat_kernels.h"
#include "lat_layout.cuh"
#include "lat_pairs.cuh"

namespace lat {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// What the sites and the solve need beyond the scalar block: formed once per block.
enum { kKl, kKdom, kKkap, kKhdt = 4, kKw0, kKbgf, kKbgp, kSiteCoefs };
template <typename T>
struct LfPre {
    double cL, cdom, kappa, g, w0;   // g = (8piG/(3A^2)) a^(-2r); w0 as the sites use it
    T k[kSiteCoefs];                 // the sites' coefficients, indexed as above
};

// By one warp: powers of a in lanes 0..3.
template <typename T>
__device__ inline void lform_pre_warp(const Model& M, const DevScalars* sc, LfPre<T>& pre)
{
    const int lane = threadIdx.x & 31;
    const double a = sc->a;
    // 1/a, and r/l in lane 5
    const double quo = (lane == 5 ? M.r : 1.0) / (lane == 5 ? sc->ell : a);
    const double ia = __shfl_sync(kFull, quo, 0), rl = __shfl_sync(kFull, quo, 5);
    const double p = lane == 0 ? -2.0 * M.s - 2.0 : lane == 1 ? M.pdom : lane == 2 ? M.pint : lane == 3 ? -2.0 * M.r : 0.0;
    double w = 1.0;
    if (__all_sync(kFull, p == rint(p) && fabs(p) <= 16.0)) {   // as apow, all lanes at once
        double b = p < 0.0 ? ia : a;
        int m = (int)fabs(p);
        while (true) {
            if (m & 1) w *= b;
            m >>= 1;
            if (!__any_sync(kFull, m)) break;
            b *= b;
        }
    } else if (lane < 4) {
        w = apow(a, ia, p);
    }
    w = w * (lane == 1 ? M.cdom0 : lane == 2 ? M.kappa0 : lane == 3 ? M.g8A2 * (1.0 / 3.0) : 1.0);
    double v = lane == kKl ? w * M.lap_scale : w;
    if (lane == kKhdt) v = 0.5 * M.dt;
    if (lane == kKw0) v = 0.5 * M.dt * sc->cF - rl;
    if (lane == kKbgf) v = sc->bgf;
    if (lane == kKbgp) v = sc->bgp;
    const T k = (T)v;
    if (lane < kSiteCoefs) pre.k[lane] = k;
    if (lane == kKw0) pre.w0 = (double)k;
    if (lane == 0) pre.cL = w;
    if (lane == 1) pre.cdom = w;
    if (lane == 2) pre.kappa = w;
    if (lane == 3) pre.g = w;
}

// The implicit midpoint solve of lat_lform.cu, for one warp, from the raw sums
// (lane l holds sum l & 3); img ends as the scalar block of the next step. The
// fixed-point map (l', cF) -> (l', cF) is iterated in FP32 first, as long as it
// gains, from the same start, and its derivative J formed there; an FP64
// evaluation F is then followed by a Newton step, x + (1 - J)^-1 (F - x): the first
// leaves about 1e-14, so that the second evaluation meets the same 1e-13 (6 to 11
// without; an FP64 evaluation takes 1.2 us).
template <typename T>
__device__ inline void lform_solve_warp(const Model& M, DevScalars& img, const LfPre<T>& pre, double raw)
{
    const int lane = threadIdx.x & 31;
    const double S = raw * M.inv_sites;
    const double S0 = __shfl_sync(kFull, S, 0), S1 = __shfl_sync(kFull, S, 1), S2 = __shfl_sync(kFull, S, 2),
                 S3 = __shfl_sync(kFull, S, 3);
    const double a = img.a, dt = M.dt, r = M.r, sg = M.s, ell = img.ell, g = pre.g, w0 = pre.w0;
    bool ok = isfinite(S0) && isfinite(S1) && isfinite(S2) && isfinite(S3) && isfinite(ell) && ell != 0.0;
    double ell_next = ell, cF = 0.0, Gam = 0.0;
    bool newton = false;
    float ill = 0.0f, ilc = 0.0f, icl = 0.0f, icc = 0.0f;   // (1 - J)^-1
    if (ok) {
        const float fdt = (float)dt, fr = (float)r, fsg = (float)sg, fl = (float)ell, fg = (float)g, fw = (float)w0;
        const float f0 = (float)S0, f1 = (float)S1, f2 = (float)S2, f3 = (float)S3;
        float l = fl, c = 0.0f, change = 3.4e38f;
        float jll = 0.0f, jlc = 0.0f, jcl = 0.0f, jcc = 0.0f;
        for (int it = 0; it < 32; it++) {
            const float Lam = 0.5f * (fl + l), h = 1.0f / Lam, dw = (0.5f * fdt * c - fr * h) - fw;
            const float G = fg * ((f0 + 2.0f * dw * f1 + dw * dw * f2) - f3);
            const float cn = fr * (2.0f - fr) * h * h - fr * G, ln = fl + fdt * ((fsg + 1.0f) + G * Lam * Lam);
            const float d = fabsf(ln - l) + fabsf(cn - c);
            if (!(d < change)) break;   // no gain any more, or not finite
            const float dG = 2.0f * fg * (f1 + dw * f2), Gl = dG * 0.5f * fr * h * h, Gc = dG * 0.5f * fdt;
            jll = fdt * (Gl * Lam + G) * Lam;
            jlc = fdt * Gc * Lam * Lam;
            jcl = -fr * ((2.0f - fr) * h * h * h + Gl);
            jcc = -fr * Gc;
            change = d;
            l = ln;
            c = cn;
        }
        if (isfinite(l) && isfinite(c) && l != 0.0f && change < 1e30f) {
            ell_next = (double)l;
            cF = (double)c;
            const float all = 1.0f - jll, acc = 1.0f - jcc, det = all * acc - jlc * jcl;
            if (fabsf(det) > 0.1f && fabsf(det) < 10.0f) {
                newton = true;
                ill = acc / det;
                ilc = jlc / det;
                icl = jcl / det;
                icc = all / det;
            }
        }
    }
    bool converged = false;
    for (int it = 0; it < 200 && ok && !converged; it++) {
        const double Lam = 0.5 * (ell + ell_next), h = 1.0 / Lam;
        const double dw = (0.5 * dt * cF - r * h) - w0;
        const double P = S0 + 2.0 * dw * S1 + dw * dw * S2;
        Gam = g * (P - S3);
        const double cF_new = r * (2.0 - r) * h * h - r * Gam;
        const double ell_new = ell + dt * ((sg + 1.0) + Gam * Lam * Lam);
        ok = finite_bits(cF_new) && finite_bits(ell_new);
        // stop at 1e-13 of the size of the terms: rounding leaves a cycle of a few ulps
        converged = fabs(ell_new - ell_next) <= 1e-13 * fabs(ell_new) &&
                    fabs(cF_new - cF) <= 1e-13 * fabs(r) * (fabs(2.0 - r) * h * h + fabs(Gam));
        if (newton) {
            const float dl = (float)(ell_new - ell_next), dc = (float)(cF_new - cF);
            ell_next = ell_next + (double)(ill * dl + ilc * dc);
            cF = cF + (double)(icl * dl + icc * dc);
            newton = it < 4;
        } else {
            cF = cF_new;
            ell_next = ell_new;
        }
    }
    if (lane == 0) img.ticket = 0u;
    if (!ok || !converged) {
        if (lane == 0) img.status = LAT_ENONFINITE;
        __syncwarp();
        return;
    }
    // lanes 0, 1: 2/(l + l'), dt/l'
    const double quo = (lane == 1 ? dt : 2.0) / (lane == 1 ? ell_next : ell + ell_next);
    const double h = __shfl_sync(kFull, quo, 0), x = __shfl_sync(kFull, quo, 1);
    const double next = a * expm1(x) / dt;   // a_{n+3/2} - a_{n+1/2} = a (exp(dt/l) - 1)
    double bgf = 0.0, bgp = 0.0;
    const double P = img.bgf;
    const double force = pre.cdom * (M.beta == 4 ? P * P * P : P);
    bgp = img.bgp + dt * (cF * P - force);
    bgf = P + dt * bgp;
    // the coefficients of the step, one to a lane
    double k = 0.0;
    if (lane == kDtCl) k = dt * pre.cL * M.lap_scale;
    else {
        const double u = lane == kDtCf ? dt : lane == kMDtCdom || lane == kMDtKap ? -dt : lane == kBg2 ? P
                         : lane == kBgNew2 ? bgf : 1.0;
        const double v = lane == kDtCf ? cF : lane == kMDtCdom ? pre.cdom : lane == kMDtKap ? pre.kappa
                         : lane == kDt ? dt : lane == kBg || lane == kBg2 ? P : bgf;
        k = u * v;
    }
    __syncwarp();
    if (lane < kCoefs) {
        img.kd[lane] = k;
        img.kf[lane] = (float)k;
    }
    if (lane == 0) {
        img.cL = pre.cL;
        img.cF = cF;
        img.cdom = pre.cdom;
        img.kappa = pre.kappa;
        img.ad_half = a * h;
        img.add = a * (-sg * h * h - Gam);
        img.ad_next = next;
        img.ell_next = ell_next;
        img.bgp_next = bgp;
        img.bgf_next = bgf;
    }
    __syncwarp();
}

enum { kPair, kHalo, kIdle };   // warp roles

// EDGE: rows cut into x tiles; otherwise a row is one tile. C27: the 27-point
// Laplacian.
template <typename T, int TY, int D, bool EDGE, bool C27>
struct LR {
    typedef typename PK<T>::P P;
    static constexpr int NP = PK<T>::NP, VW = 2 * NP, W = 32 * VW;
    static constexpr int RF = D + 2, RP = D + 1;       // field and momentum plane slots
    static constexpr int ROWS = TY + 2, PAIRS = TY / 2, THREADS = (PAIRS + 1) * 32;
    static_assert(TY % 2 == 0 && ROWS <= 32, "row pairs; a lane per row for the edge columns");
    // shared memory, in elements: the field ring [slot][field][ROWS][W], the
    // momentum ring [slot][field][TY][W], the columns beside the tile
    // [slot][field][ROWS][2]
    static constexpr uint32_t FIELDF = ROWS * W, SLOTF = 2 * FIELDF, FIELDP = TY * W, SLOTP = 2 * FIELDP;
    static constexpr uint32_t P0 = RF * SLOTF, EF = 2 * ROWS, ESF = 2 * EF, E0 = P0 + RP * SLOTP;
    static constexpr uint32_t END = EDGE ? E0 + RF * ESF : E0;
    static constexpr size_t SMEM = (sizeof(T) * (size_t)END + 15) / 16 * 16;

    struct Ctx {
        T* S;
        uint32_t nn, offF, offP, rowg, rowhi, ey, exl, exr;
        int n, ty, last, row, lane, sl, sr, z0, nz;
        bool act;
        const T *f0, *f1, *p0, *p1;
    };
    struct Coef {
        P kL, hdt, cdom, kap, w0, bgf, bgp;
        bool quartic;
    };
    struct Acc {   // compensated (Kahan) sums, the halves of a pair apart
        P s[kSums], c[kSums];
        __device__ __forceinline__ void add(int k, P v)
        {
            const P y = sub2(v, c[k]), t = add2(s[k], y);
            c[k] = sub2(sub2(t, s[k]), y);
            s[k] = t;
        }
    };
    struct Slots {
        int fc, fp, fw, pc, pw;
        __device__ __forceinline__ void next()
        {
            fw = fc;
            fc = fp;
            fp = fp + 1 == RF ? 0 : fp + 1;
            pw = pc;
            pc = pc + 1 == RP ? 0 : pc + 1;
        }
    };

    // plane zrel of the run's fields, counted down from its last: a pair's rows; the
    // halo warp the rows beside
    // the tile and (lane r for staged row r) the columns beside it
    template <int ROLE>
    static __device__ __forceinline__ void fetch_f(const Ctx& C, int zrel, int slot)
    {
        const uint32_t zoff = (uint32_t)wrapn(C.z0 + C.nz - 1 - zrel, C.n) * C.nn;
        T* S = C.S + slot * SLOTF;
        if constexpr (ROLE == kPair) {
            const T *a = C.f0 + zoff + C.rowg, *b = C.f1 + zoff + C.rowg;
            T* d = S + C.offF;
            if (C.act) {
                cp_async16(d, a);
                cp_async16(d + W, a + C.n);
                cp_async16(d + FIELDF, b);
                cp_async16(d + FIELDF + W, b + C.n);
            }
        } else if constexpr (ROLE == kHalo) {
            T *lo = S + C.lane * VW, *hi = lo + (C.ty + 1) * W;
            if (C.act) {
                cp_async16(lo, C.f0 + zoff + C.rowg);
                cp_async16(lo + FIELDF, C.f1 + zoff + C.rowg);
                cp_async16(hi, C.f0 + zoff + C.rowhi);
                cp_async16(hi + FIELDF, C.f1 + zoff + C.rowhi);
            }
            if (EDGE && C.lane < C.ty + 2) {
                T* e = C.S + E0 + slot * ESF + C.lane * 2;
                const uint32_t gb = zoff + C.ey;
                cp_async_small<sizeof(T)>(e, C.f0 + gb + C.exl);
                cp_async_small<sizeof(T)>(e + 1, C.f0 + gb + C.exr);
                cp_async_small<sizeof(T)>(e + EF, C.f1 + gb + C.exl);
                cp_async_small<sizeof(T)>(e + EF + 1, C.f1 + gb + C.exr);
            }
        }
    }
    template <int ROLE>
    static __device__ __forceinline__ void fetch_p(const Ctx& C, int zrel, int slot)
    {
        if constexpr (ROLE == kPair) {
            const uint32_t g = (uint32_t)wrapn(C.z0 + C.nz - 1 - zrel, C.n) * C.nn + C.rowg;
            T* d = C.S + P0 + slot * SLOTP + C.offP;
            if (C.act) {
                cp_async16(d, C.p0 + g);
                cp_async16(d + W, C.p0 + g + C.n);
                cp_async16(d + FIELDP, C.p1 + g);
                cp_async16(d + FIELDP + W, C.p1 + g + C.n);
            }
        }
    }

    // Carried from plane to plane, for each field and row: the centre and its
    // difference to the plane below (7 points), or the pending L_z and q_z of
    // lat_step27w.cu (27).
    struct Col {
        P a[2][2][NP], b[2][2][NP];
    };

    // The Laplacian of field f at the pair's sites (x: their centres), as the step
    // kernels form it.
    static __device__ __forceinline__ void laplacian(const Ctx& C, const Slots& Z, int f, Col& Q, P (&x)[2][NP],
                                                     P (&lap)[2][NP])
    {
        const T* Fc = C.S + Z.fc * SLOTF + f * FIELDF + C.offF;
        const T* Fp = C.S + Z.fp * SLOTF + f * FIELDF + C.offF;
        if constexpr (C27) {
            const T* Ep = C.S + E0 + Z.fp * ESF + f * EF + (C.row - 1) * 2;
            const P c30 = mk2(T(30), T(30)), cm30 = mk2(T(-30), T(-30));
            P cp[2][NP], q[2][NP], r[2][NP];
            agg27<T, 2, EDGE>(Fp, W, C.lane, C.last, C.sl, C.sr, Ep, 2, cp, q, r);
#pragma unroll
            for (int i = 0; i < 2; i++) {
                PK<T>::ld(Fc + i * W, x[i]);
#pragma unroll
                for (int j = 0; j < NP; j++) {
                    const P d = sub2(cp[i][j], x[i][j]);
                    lap[i][j] = add2(fma2(c30, d, Q.a[f][i][j]), q[i][j]);
                    Q.a[f][i][j] = add2(fma2(cm30, d, Q.b[f][i][j]), r[i][j]);
                    Q.b[f][i][j] = q[i][j];
                }
            }
        } else {
            const T* Ec = C.S + E0 + Z.fc * ESF + f * EF + C.row * 2;
            P up[NP], dn[NP], zp[2][NP];
            PK<T>::ld(Fc - W, up);
            PK<T>::ld(Fc + 2 * W, dn);
#pragma unroll
            for (int i = 0; i < 2; i++) {
                PK<T>::ld(Fp + i * W, zp[i]);
#pragma unroll
                for (int j = 0; j < NP; j++) x[i][j] = Q.a[f][i][j];
            }
#pragma unroll
            for (int i = 0; i < 2; i++) {
                T left = __shfl_sync(kFull, hi2(x[i][NP - 1]), C.sl), right = __shfl_sync(kFull, lo2(x[i][0]), C.sr);
                if constexpr (EDGE) {
                    left = ld_shared_if(C.lane == 0, Ec + i * 2, left);
                    right = ld_shared_if(C.lane == C.last, Ec + i * 2 + 1, right);
                }
                T d[VW];
                xdiff<T>(x[i], right, d);
                const T dl = s_sub(lo2(x[i][0]), left);
#pragma unroll
                for (int j = 0; j < NP; j++) {
                    const P lx = mk2(s_sub(d[2 * j], j == 0 ? dl : d[2 * j - 1]), s_sub(d[2 * j + 1], d[2 * j]));
                    const P in = sub2(x[1][j], x[0][j]);
                    const P ly = i == 0 ? add2(sub2(up[j], x[i][j]), in) : sub2(sub2(dn[j], x[i][j]), in);
                    const P z = sub2(zp[i][j], x[i][j]);
                    lap[i][j] = add2(add2(lx, ly), sub2(z, Q.b[f][i][j]));
                    Q.a[f][i][j] = zp[i][j];
                    Q.b[f][i][j] = z;
                }
            }
        }
    }

    // One plane of a pair: the Laplacian, then the sites' terms, summed over the vector's pairs and the two rows before they
    // join the compensated sums.
    static __device__ __forceinline__ void pair_plane(const Ctx& C, const Coef& K, const Slots& Z, Col& Q, Acc& A)
    {
        const T* Pc = C.S + P0 + Z.pc * SLOTP + C.offP;
        P x[2][2][NP], lap[2][2][NP], mom[2][2][NP];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            laplacian(C, Z, f, Q, x[f], lap[f]);
#pragma unroll
            for (int i = 0; i < 2; i++) PK<T>::ld(Pc + f * FIELDP + i * W, mom[f][i]);
        }
        P s[kSums];
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int j = 0; j < NP; j++) {
                const P f0 = add2(x[0][i][j], K.bgf), f1 = x[1][i][j];   // whole phi (+ 0 when stored whole)
                const P p0 = add2(mom[0][i][j], K.bgp), p1 = mom[1][i][j];
                const P sq0 = mul2(f0, f0), sq1 = mul2(f1, f1), k1 = mul2(K.kap, sq1);
                const P half = mk2(T(0.5), T(0.5)), quarter = mk2(T(0.25), T(0.25));
                const P dom = K.quartic ? mul2(K.cdom, sq0) : K.cdom;
                const P u0 = mul2(f0, add2(dom, k1)), u1 = mul2(f1, mul2(K.kap, sq0));
                const P v0 = fma2(K.w0, f0, fma2(K.hdt, sub2(mul2(K.kL, lap[0][i][j]), u0), p0));
                const P v1 = fma2(K.w0, f1, fma2(K.hdt, sub2(mul2(K.kL, lap[1][i][j]), u1), p1));
                P t[kSums];
                t[0] = fma2(v0, v0, mul2(v1, v1));
                t[1] = fma2(v0, f0, mul2(v1, f1));
                t[2] = add2(sq0, sq1);
                // cdom (f^4/4 or f^2/2) + kap f^2 g^2 / 2
                t[3] = mul2(sq0, fma2(half, k1, mul2(K.quartic ? quarter : half, dom)));
#pragma unroll
                for (int q = 0; q < kSums; q++) s[q] = i == 0 && j == 0 ? t[q] : add2(s[q], t[q]);
            }
#pragma unroll
        for (int q = 0; q < kSums; q++) A.add(q, s[q]);
    }

    // One run of planes; `pre`: called by the halo warp once the first planes are on
    // their way, and then `coefs` by every warp behind a barrier.
    template <int ROLE, typename Pre, typename Coefs>
    static __device__ __forceinline__ void run(const Ctx& C, Coef& K, Acc& A, Pre pre, Coefs coefs)
    {
        fetch_f<ROLE>(C, -1, 0);
        fetch_f<ROLE>(C, 0, 1);
        fetch_f<ROLE>(C, 1, 2);
        fetch_p<ROLE>(C, 0, 0);
        cp_async_commit();
#pragma unroll
        for (int j = 1; j < D; j++) {
            if (j < C.nz) {
                fetch_f<ROLE>(C, j + 1, j + 2);
                fetch_p<ROLE>(C, j, j);
            }
            cp_async_commit();
        }
        if constexpr (ROLE == kHalo) pre();
        cp_async_wait(D - 1);
        __syncthreads();
        Col Q;
        if constexpr (ROLE == kPair) {
            coefs(K);
#pragma unroll
            for (int f = 0; f < 2; f++) {
                const T *m = C.S + f * FIELDF + C.offF, *o = m + SLOTF;   // planes -1 and 0
                P cm[2][NP];
                if constexpr (C27) {
                    const T* E = C.S + E0 + f * EF + (C.row - 1) * 2;
                    const P cm30 = mk2(T(-30), T(-30));
                    P c[2][NP], q[2][NP], r[2][NP];
                    agg27<T, 2, EDGE>(m, W, C.lane, C.last, C.sl, C.sr, E, 2, cm, Q.b[f], r);
                    agg27<T, 2, EDGE>(o, W, C.lane, C.last, C.sl, C.sr, E + ESF, 2, c, q, r);
#pragma unroll
                    for (int i = 0; i < 2; i++)
#pragma unroll
                        for (int j = 0; j < NP; j++) {
                            Q.a[f][i][j] = add2(fma2(cm30, sub2(c[i][j], cm[i][j]), Q.b[f][i][j]), r[i][j]);
                            Q.b[f][i][j] = q[i][j];
                        }
                } else {
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        PK<T>::ld(m + i * W, cm[i]);
                        PK<T>::ld(o + i * W, Q.a[f][i]);
#pragma unroll
                        for (int j = 0; j < NP; j++) Q.b[f][i][j] = sub2(Q.a[f][i][j], cm[i][j]);
                    }
                }
            }
        }
        Slots Z{1, 2, 0, 0, RP - 1};
#pragma unroll 2
        for (int k = 0; k < C.nz; k++) {
            cp_async_wait(D - 1);
            __syncthreads();
            if (k + D < C.nz) {
                fetch_f<ROLE>(C, k + D + 1, Z.fw);
                fetch_p<ROLE>(C, k + D, Z.pw);
            }
            cp_async_commit();
            if constexpr (ROLE == kPair) pair_plane(C, K, Z, Q, A);
            Z.next();
        }
    }
};

template <typename T, int TY, int D, bool EDGE, bool C27>
__global__ void __launch_bounds__(LR<T, TY, D, EDGE, C27>::THREADS, TY <= 8 ? 2 : 1)
    lform_ring_kernel(Bufs<T> B, Model M, DevScalars* sc, double* partials)
{
    typedef LR<T, TY, D, EDGE, C27> F;
    constexpr int VW = F::VW;
    __shared__ double red[32 * kSums];
    __shared__ LfPre<T> pre;
    __shared__ DevScalars img;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename F::Ctx C;
    C.S = reinterpret_cast<T*>(smem_raw);
    C.lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    // the tiles and the layout of the step kernel (lat_xw.cuh)
    const int n = M.n;
    C.n = n;
    C.nn = (uint32_t)n * n;
    const int Q = n / VW, cut = Q % 4 == 0 ? 4 : Q % 2 == 0 ? 2 : 1;
    const int nxt = EDGE ? (Q + 31) / 32 : 1, nyt = (n + TY - 1) / TY;
    const int grp = blockIdx.x / nxt, xt = blockIdx.x - grp * nxt;
    const int q0 = xt * (Q / cut) / nxt * cut, qn = (xt + 1) * (Q / cut) / nxt * cut - q0;
    const int x0 = q0 * VW, x1 = x0 + qn * VW;
    TileWalk walk(nyt, gridDim.x / nxt, grp, n);
    C.last = qn - 1;
    C.act = C.lane < qn;
    // EDGE: what the end lanes get from the shuffles is replaced by edge scalars
    C.sl = EDGE ? max(C.lane - 1, 0) : C.lane == 0 ? C.last : C.lane - 1;
    C.sr = EDGE ? min(C.lane + 1, 31) : C.lane >= C.last ? 0 : C.lane + 1;
    C.exl = (uint32_t)(x0 == 0 ? n - 1 : x0 - 1);
    C.exr = (uint32_t)(x1 == n ? 0 : x1);

    chain_begin();
    if (sc->status != LAT_OK) return;
    const int par = (int)(sc->step & 1);
    C.f0 = B.f[par][0];
    C.f1 = B.f[par][1];
    C.p0 = B.p[par][0];
    C.p1 = B.p[par][1];
    typename F::Acc A;
#pragma unroll
    for (int k = 0; k < kSums; k++) A.s[k] = A.c[k] = mk2(T(0), T(0));
    typename F::Coef K;
    auto coefs = [&](typename F::Coef& k) {
        auto two = [&](int i) { return mk2(pre.k[i], pre.k[i]); };
        k.kL = two(kKl);
        k.hdt = two(kKhdt);
        k.cdom = two(kKdom);
        k.kap = two(kKkap);
        k.w0 = two(kKw0);
        k.bgf = two(kKbgf);
        k.bgp = two(kKbgp);
        k.quartic = M.beta == 4;
    };
    const bool halo = warp == F::PAIRS;
    int yt;
    bool first = true, have = false;   // have: this warp's coefficients are read
    for (; walk.run(yt, C.z0, C.nz); first = false) {
        walk.took(C.nz);
        const int y0 = 2 * (yt * (n / 2) / nyt);
        C.ty = 2 * ((yt + 1) * (n / 2) / nyt) - y0;
        C.row = 2 * warp + 1;
        C.offF = (uint32_t)C.row * F::W + C.lane * VW;
        C.offP = (uint32_t)(C.row - 1) * F::W + C.lane * VW;
        const uint32_t xg = x0 + C.lane * VW;
        C.rowg = (uint32_t)(halo ? wrapn(y0 - 1, n) : wrapn(y0 + C.row - 1, n)) * n + xg;
        C.rowhi = (uint32_t)wrapn(y0 + C.ty, n) * n + xg;
        C.ey = (uint32_t)wrapn(y0 - 1 + min(C.lane, C.ty + 1), n) * n;
        // the previous run's last plane is read by every thread before the prologue
        // refills the ring
        if (!first) __syncthreads();
        auto form = [&]() {
            if (first) lform_pre_warp<T>(M, sc, pre);
        };
        auto get = [&](typename F::Coef& k) {
            if (!have) coefs(k);
            have = true;
        };
        if (halo) F::template run<kHalo>(C, K, A, form, get);
        else if (C.row <= C.ty) F::template run<kPair>(C, K, A, form, get);
        else F::template run<kIdle>(C, K, A, form, get);
    }
    if (first) {   // a block without work may still be the last
        if (halo) lform_pre_warp<T>(M, sc, pre);
        __syncthreads();
    }

    TreeSum<T> v[kSums];
#pragma unroll
    for (int k = 0; k < kSums; k++) {   // a sum and what its additions lost
        TreeSum<T> a{lo2(A.s[k]), -lo2(A.c[k])}, b{hi2(A.s[k]), -hi2(A.c[k])};
        a.add(b);
        v[k] = a;
        if (!C.act) v[k].init(T(0));   // nothing in this lane
    }
    if (!block_ticket<T>(v, red, partials, &sc->ticket, [&]() { scalars_to_shared(img, sc); }, []() {})) return;
    const double raw = last_block_fold(partials, red);
    if (threadIdx.x >= 32) return;
    lform_solve_warp<T>(M, img, pre, raw);
    scalars_from_shared(sc, img);
}

constexpr int kTY = 8, kDepth = 2;   // a third plane in flight: 256^3 3 us more

template <bool EDGE, bool C27>
bool ring_shape(int n, const void** fn, size_t* smem, int* threads, int* blocks)
{
    typedef LR<float, kTY, kDepth, EDGE, C27> F;
    *fn = (const void*)lform_ring_kernel<float, kTY, kDepth, EDGE, C27>;
    *smem = F::SMEM;
    *threads = F::THREADS;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (allow_dynamic_smem(*fn, F::SMEM) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    const int nxt = EDGE ? (n / 4 + 31) / 32 : 1;
    const long long units = (long long)((n + kTY - 1) / kTY) * nxt * n;
    *blocks = (int)(std::min((long long)sms * (kTY <= 8 ? 2 : 1), units) / nxt * nxt);   // whole groups of x tiles
    return *blocks >= nxt;
}

} // namespace

cudaError_t launch_lform_ring(const Bufs<float>& b, const Model& M, DevScalars* sc, double* partials, bool chain,
                              cudaStream_t st)
{
    const void* fn;
    size_t smem;
    int threads, blocks;
    auto shape = [&](auto f) { return f(M.n, &fn, &smem, &threads, &blocks); };
    const bool edge = M.n > 128;
    if (!(M.stencil == 27 ? shape(edge ? ring_shape<true, true> : ring_shape<false, true>)
                          : shape(edge ? ring_shape<true, false> : ring_shape<false, false>)))
        return cudaErrorInvalidDevice;
    void* args[] = {(void*)&b, (void*)&M, (void*)&sc, (void*)&partials};
    return launch_chained(fn, dim3(blocks), dim3(threads), args, smem, st, chain);
}

} // namespace lat

// lat_step27w.cu -- the fused leapfrog step with the 27-point Laplacian of
// Sec. II.C (Patra and Karttunen) over x tiles one warp wide, with the tile
// height TY and the prefetch depth D known at compile time and the lattice side
// taken at run time (variant 5 of the 27-point stencil).
//
// Tiles, ring and layout follow the 7-point kernel of lat_xw.cuh: a tile is at most
// W = 32 16-byte vectors wide (a row's vectors are shared evenly among its tiles)
// and at most TY rows tall. Two warps serve each pair of neighbouring rows: the step
// warp kicks and drifts it and stores its momenta; the sum warp stages the pair's
// rows, and one plane later adds up the new fields and stores them.
// One more warp stages the halo rows, kicks and drifts the look-ahead row, and,
// where the row is cut into x tiles, stages the scalars of the tile's x neighbours
// (columns x0 - 1 and the two right of the tile) and computes the new fields of
// the boundary column right of the tile, rounded exactly as the next tile computes
// its own first column. Rows of one tile reach their ends by a rotating shuffle.
//
// What bounds it. FP32: the instructions of a plane, about 480 per row of a warp (960
// per pair against some 1500 with one row per warp and 13 squared bonds per site),
// issued by 15 warps, and the step warps' chain from barrier to barrier; the copy
// itself would take 79 us of the 107 at 256^3 and 636 of the 760 at 512^3. One warp
// for both halves of a pair's work held 252 registers, two warps to a scheduler,
// and waited on its own latencies (issue slots 43 % busy, 126 us at 256^3, 913 at
// 512^3); the two halves in two warps of 128 registers overlap, with the new fields
// through shared memory (117 and 824 us), and with the copies and the fields'
// stores on the sum warps, which waited for the others at the barrier, 107 and 760.
// One row per warp took 149 and 1187. Sides that only the plane-ring kernel ran
// before: 100^3 42 -> 18 us, 292^3 1690 -> 188, 384^3 699 -> 334. FP64 is bound by
// the FP64 pipe: 256^3 4.07 -> 3.50 ms.
//
// Laplacian. In units of 1/(30 dx^2) the weights are 14 (6 faces), 3 (12 edges)
// and 1 (8 corners). Per plane p and site, with differences taken from that
// plane's own centre C:
//   v = (f(y - 1) - C) + (f(y + 1) - C)                the y pair
//   h = (f(x + 1) - C) - (C - f(x - 1))                the x pair
//   e = h + v                                          the 4 in-plane faces
//   k = v(x - 1) + v(x + 1) + 2 h                      the 4 in-plane corners
// (v(x +- 1) is taken about C(x +- 1); 2 h puts back the 2 (C(x +- 1) - C)),
//   q_p = 3 e + k    the plane's part when it is the plane below or above,
//   r_p = 14 e + 3 k its part when it is the centre plane, and
//   30 dx^2 Lap f(z) = r_z + q_{z-1} + q_{z+1} + 30 ((C_{z-1} - C_z) + (C_{z+1} - C_z)).
// Every term is a sum of differences of neighbouring values (exact for
// f = const + small). The x-shifted sums are formed by scalar operations that
// write the halves of the packed pairs, so no register moves build shifted
// pairs. Along z each field keeps three values per site in registers: C_z, the
// pending sum of plane z, L_z = (q_{z-1} - 30 (C_z - C_{z-1})) + r_z, and q_z;
// plane z + 1's aggregate, formed once, completes
// Lap(z) = (L_z + 30 (C_{z+1} - C_z)) + q_{z+1} and starts L_{z+1}. Every site's
// value depends only on its 3x3x3 neighbourhood, not on the tiling or the z
// segments.
//
// Sums of the new fields for eq. scale: -<g Lap g> is the mean over sites of
// sum_b w_b (g(x + b) - g(x))^2 over the 13 bonds a site owns. Over the whole
// lattice that is a sum over its unit cubes, and there the bond energies are
// diagonal in the cube's eight sign patterns: 15 for a pattern odd in one
// direction, 20 in two, 23 in three (each squared, over 8). With the patterns odd
// in x taken first, and their y and z sums and differences multiplied out,
//   8 E = 312 dx^2 - 32 (dx dx_y + dx dx_z) - 4 (dx dx_yz + dx_y dx_z)
//         + 70 B^2 - 10 B B_z + 15 Z^2,
// dx the x difference (dx_y, dx_z, dx_yz: of the next row, the next plane, both),
// B = dy + dy(x + 1), Z the sum of the cube's four z differences. Differences are
// still formed first. That is 8 products per site for 13 squared bonds, one
// shuffle a row for four, and only g and dx of the row above (the next pair's
// first row, from shared memory) besides the pair's own. The cube between planes P
// and P + 1 is summed at plane P + 2, after the barrier that completes P + 1.
#include <algorithm>

#include "lat_agg27.cuh"
#include "lat_async.cuh"
#include "lat_kernels.h"
#include "lat_layout.cuh"
#include "lat_pairs.cuh"
#include "lat_site.cuh"

namespace lat {

namespace {

constexpr unsigned kFull = 0xffffffffu;
enum { kStep, kSum, kAhead, kIdle };   // warp roles

// EDGE: rows cut into x tiles; otherwise a row is one tile.
template <typename T, int TY, int D, bool EDGE>
struct S27 {
    typedef typename PK<T>::P P;
    // field and momentum plane slots: planes z and z + 1 and D in flight, plane z
    // and D
    static constexpr int RF = D + 2, RP = D + 1;
    static constexpr int NP = PK<T>::NP;
    static constexpr int VW = 2 * NP;                  // elements per 16-byte vector
    static constexpr int W = 32 * VW;                  // tile width: one warp of vectors
    static constexpr int ROWS = TY + 3;                // staged rows, at most
    static constexpr int GR = TY + 1;                  // computed rows (owned + look-ahead), at most
    static constexpr int PAIRS = TY / 2;               // pairs of owned rows, two warps each
    static constexpr int THREADS = (2 * PAIRS + 1) * 32;
    static_assert(TY % 2 == 0 && ROWS <= 32, "row pairs; a lane per row for the edge columns");
    // Shared memory, in elements. The field ring [slot][field][ROWS][RS] with a
    // row stride one vector longer than the tile (the edge column reads the last
    // column of every row: the padding spreads those reads over the banks), the
    // momentum ring [slot][field][GR][W], the new fields [buf][field][GR][W]; then
    // the edge scalars: fields [slot][field][ROWS][4] (x0 - 1, x0 + W, x0 + W + 1, unused),
    // momenta at x0 + W [slot][field][GR], new fields at x0 + W [buf][field][GR].
    static constexpr int RS = W + VW;
    static constexpr uint32_t FIELDF = ROWS * RS, SLOTF = 2 * FIELDF;
    static constexpr uint32_t FIELDP = GR * W, SLOTP = 2 * FIELDP;
    static constexpr uint32_t P0 = RF * SLOTF, G0 = P0 + RP * SLOTP;
    static constexpr uint32_t EF = ROWS * 4, ESF = 2 * EF;
    static constexpr uint32_t ESP = 2 * GR;
    static constexpr uint32_t EF0 = G0 + 2 * SLOTP, EP0 = EF0 + RF * ESF, EG0 = EP0 + RP * ESP;
    static constexpr uint32_t END = EDGE ? EG0 + 2 * ESP : EF0;
    static constexpr size_t SMEM = (sizeof(T) * (size_t)END + 15) / 16 * 16;

    struct Ctx {
        T* S;
        uint32_t nn;
        int n, ty, last;                // side, owned rows of the tile (even), its last lane
        bool act;                       // this lane holds a vector of the tile
        uint32_t offF, offP;            // this thread's vector of its (first) row: field and momentum planes
        uint32_t rowg, rowlo, rowhi;    // global offsets in a plane: its (first) row; the halo rows (look-ahead warp)
        int row, lane, sl, sr, z0, nz;  // its (first) row in the staged tile; the lanes beside it
        uint32_t ey, eyp;               // edge columns: the row of staged row `lane` and of computed row lane + 1
        uint32_t exl, exr, exr1;        // the three edge columns
        const T *f0, *f1, *p0, *p1;
        T *of0, *of1, *op0, *op1;
        SiteCoefs<T> K;
    };
    struct Acc {
        P wg[2], vd, vi;                // sums of the new fields (sum warps)
    };
    // ring slots of one plane step: field planes k + 1 and the one that plane
    // k - 1 left, momentum plane k and the one that k - 1 left; new-field buffer
    struct Slots {
        int fc, fp, fw, pc, pw, g;
        __device__ __forceinline__ void next()
        {
            fw = fc;
            fc = fp;
            fp = fp + 1 == RF ? 0 : fp + 1;
            pw = pc;
            pc = pc + 1 == RP ? 0 : pc + 1;
            g ^= 1;
        }
    };
    // carried from plane to plane, for each field and row: L_z and q_z (step
    // and look-ahead warps; C_z is read again from the ring); the new fields, x differences and B of the
    // pair's rows (the row after the pair as row 2), with the new fields right of
    // the vector (sum warps)
    template <int R>
    struct Col {
        P L[2][R][NP], q[2][R][NP];
    };
    struct Cube {
        P g[2][3][NP], B[2][2][NP];
        T r[2][3];
    };
    // the boundary column (lane r - 1 for computed row r)
    struct EdgeCol {
        T L[2], q[2], c[2];
    };

    // plane z0 + zrel of the fields into ring slot `slot`
    template <int ROLE>
    static __device__ __forceinline__ void fetch_f(const Ctx& C, int zrel, int slot)
    {
        const uint32_t zoff = (uint32_t)wrapn(C.z0 + zrel, C.n) * C.nn;
        if constexpr (ROLE == kSum) {
            const T *a = C.f0 + zoff + C.rowg, *b = C.f1 + zoff + C.rowg;
            T* d = C.S + slot * SLOTF + C.offF;
            if (C.act) {
                cp_async16(d, a);
                cp_async16(d + RS, a + C.n);
                cp_async16(d + FIELDF, b);
                cp_async16(d + FIELDF + RS, b + C.n);
            }
        } else if constexpr (ROLE == kAhead) {
            T* d = C.S + slot * SLOTF + C.offF;
            T* lo = C.S + slot * SLOTF + C.lane * VW;
            if (C.act) {
                cp_async16(lo, C.f0 + zoff + C.rowlo);
                cp_async16(lo + FIELDF, C.f1 + zoff + C.rowlo);
                cp_async16(d, C.f0 + zoff + C.rowg);
                cp_async16(d + FIELDF, C.f1 + zoff + C.rowg);
                cp_async16(d + RS, C.f0 + zoff + C.rowhi);
                cp_async16(d + FIELDF + RS, C.f1 + zoff + C.rowhi);
            }
            if (EDGE && C.lane < C.ty + 3) {
                const uint32_t gb = zoff + C.ey;
                T* e = C.S + EF0 + slot * ESF + C.lane * 4;
                cp_async_small<sizeof(T)>(e + 0, C.f0 + gb + C.exl);
                cp_async_small<sizeof(T)>(e + 1, C.f0 + gb + C.exr);
                cp_async_small<sizeof(T)>(e + 2, C.f0 + gb + C.exr1);
                cp_async_small<sizeof(T)>(e + EF + 0, C.f1 + gb + C.exl);
                cp_async_small<sizeof(T)>(e + EF + 1, C.f1 + gb + C.exr);
                cp_async_small<sizeof(T)>(e + EF + 2, C.f1 + gb + C.exr1);
            }
        }
    }
    // momenta of plane z0 + zrel for the computed rows, and at x0 + W
    template <int ROLE>
    static __device__ __forceinline__ void fetch_p(const Ctx& C, int zrel, int slot)
    {
        const uint32_t zoff = (uint32_t)wrapn(C.z0 + zrel, C.n) * C.nn;
        if constexpr (ROLE == kSum || ROLE == kAhead) {
            const T *a = C.p0 + zoff + C.rowg, *b = C.p1 + zoff + C.rowg;
            T* d = C.S + P0 + slot * SLOTP + C.offP;
            if (C.act) {
                cp_async16(d, a);
                cp_async16(d + FIELDP, b);
                if constexpr (ROLE == kSum) {
                    cp_async16(d + W, a + C.n);
                    cp_async16(d + FIELDP + W, b + C.n);
                }
            }
        }
        if (EDGE && ROLE == kAhead && C.lane <= C.ty) {
            const uint32_t gb = zoff + C.eyp + C.exr;
            T* e = C.S + EP0 + slot * ESP + C.lane;
            cp_async_small<sizeof(T)>(e, C.p0 + gb);
            cp_async_small<sizeof(T)>(e + GR, C.p1 + gb);
        }
    }

    // The aggregates of one field at this lane's sites of its R rows (lat_agg27.cuh).
    // F: the field's plane in the ring, E: its edge scalars.
    template <int R>
    static __device__ __forceinline__ void aggr(const Ctx& C, const T* F, const T* E, P (&c)[R][NP], P (&q)[R][NP],
                                                P (&r)[R][NP])
    {
        agg27<T, R, EDGE>(F + C.offF, RS, C.lane, C.last, C.sl, C.sr, E + (C.row - 1) * 4, 4, c, q, r);
    }

    // The same aggregates at one site, rounded as the first site of a vector:
    // the centre row at x - 1, x, x + 1 (cl, c0, c1) and the rows y - 1 (m*) and
    // y + 1 (p*) at the same columns.
    static __device__ __forceinline__ void aggr1(T cl, T c0, T c1, T ml, T m0, T m1, T pl, T p0, T p1, T& q, T& r)
    {
        const T vl = s_add(s_sub(ml, cl), s_sub(pl, cl));
        const T v0 = s_add(s_sub(m0, c0), s_sub(p0, c0));
        const T v1 = s_add(s_sub(m1, c1), s_sub(p1, c1));
        const T h = s_sub(s_sub(c1, c0), s_sub(c0, cl));
        const T k = s_fma(T(2), h, s_add(vl, v1));
        const T eh = s_add(h, v0);
        q = s_fma(T(3), eh, k);
        r = s_fma(T(14), eh, s_mul(T(3), k));
    }

    // The aggregates at (x0 + W, row r) of one field's plane F (ring) with edge
    // scalars E; the site's centre in c.
    static __device__ __forceinline__ void aggr_edge(const Ctx& C, const T* F, const T* E, int r, T& c, T& q, T& r_)
    {
        const T* lc = F + r * RS + (C.last * VW + VW - 1);
        const T* e = E + r * 4;
        c = e[1];
        aggr1(lc[0], e[1], e[2], lc[-RS], e[-3], e[-2], lc[RS], e[5], e[6], q, r_);
    }

    // Takes the pair's new fields of plane P from G (the column right of the tile
    // from EG) and, where SUM is set, adds the cubes between plane P - 1 (in H) and
    // P, and the potential of plane P - 1; leaves plane P in H. Every lane calls
    // this.
    template <bool SUM, bool STORE>
    static __device__ __forceinline__ void cubes(const Ctx& C, Acc& A, Cube& H, const T* G, const T* EG, int k)
    {
        const bool last = C.lane == C.last;
        const T* gp = G + (C.row - 1) * W + C.lane * VW;
        const T* ep = EG + (C.row - 1);
        if constexpr (SUM) {
#pragma unroll
            for (int j = 0; j < NP; j++) {
                site_vsum<T>(C.K, H.g[0][0][j], H.g[1][0][j], A.vd, A.vi);
                site_vsum<T>(C.K, H.g[0][1][j], H.g[1][1][j], A.vd, A.vi);
            }
        }
#pragma unroll
        for (int f = 0; f < 2; f++) {
            P g[3][NP], dx[3][NP], dp[3][NP], B[2][NP];
            T re[3];
#pragma unroll
            for (int i = 0; i < 3; i++) PK<T>::ld(gp + f * FIELDP + i * W, g[i]);
            if (STORE && C.act) {
                T* o = (f ? C.of1 : C.of0) + (uint32_t)wrapn(C.z0 + k, C.n) * C.nn + C.rowg;
                PK<T>::st_stream(o, g[0]);
                PK<T>::st_stream(o + C.n, g[1]);
            }
#pragma unroll
            for (int i = 0; i < 3; i++) {
                re[i] = __shfl_sync(kFull, lo2(g[i][0]), C.sr);
                if constexpr (EDGE) re[i] = ld_shared_if(last, ep + f * GR + i, re[i]);
                T d[VW];
                xdiff<T>(g[i], re[i], d);
#pragma unroll
                for (int j = 0; j < NP; j++) dx[i][j] = mk2(d[2 * j], d[2 * j + 1]);
                if constexpr (SUM) {
                    xdiff<T>(H.g[f][i], H.r[f][i], d);
#pragma unroll
                    for (int j = 0; j < NP; j++) dp[i][j] = mk2(d[2 * j], d[2 * j + 1]);
                }
            }
            // a + a(x + 1) of a vector whose right neighbour is e
            auto xsum = [](const P(&a)[NP], T e, P(&o)[NP]) {
                T s[VW + 1];
#pragma unroll
                for (int j = 0; j < NP; j++) un2(a[j], s[2 * j], s[2 * j + 1]);
                s[VW] = e;
#pragma unroll
                for (int j = 0; j < NP; j++) o[j] = mk2(s_add(s[2 * j], s[2 * j + 1]), s_add(s[2 * j + 1], s[2 * j + 2]));
            };
#pragma unroll
            for (int i = 0; i < 2; i++) {
                P dy[NP];
#pragma unroll
                for (int j = 0; j < NP; j++) dy[j] = sub2(g[i + 1][j], g[i][j]);
                xsum(dy, s_sub(re[i + 1], re[i]), B[i]);
            }
            if constexpr (SUM) {
                P dz[3][NP];
                T de[3];
#pragma unroll
                for (int i = 0; i < 3; i++) {
#pragma unroll
                    for (int j = 0; j < NP; j++) dz[i][j] = sub2(g[i][j], H.g[f][i][j]);
                    de[i] = s_sub(re[i], H.r[f][i]);
                }
                const P zero = mk2(T(0), T(0));
                P s0 = zero, s1 = zero, s2 = zero, b1 = zero, b2 = zero, z = zero;
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    P S[NP], Z[NP];
#pragma unroll
                    for (int j = 0; j < NP; j++) S[j] = add2(dz[i][j], dz[i + 1][j]);
                    xsum(S, s_add(de[i], de[i + 1]), Z);
#pragma unroll
                    for (int j = 0; j < NP; j++) {
                        const P d = dp[i][j], dn = dp[i + 1][j];
                        s0 = fma2(d, d, s0);
                        s1 = fma2(d, add2(dn, dx[i][j]), s1);
                        s2 = fma2(d, dx[i + 1][j], fma2(dn, dx[i][j], s2));
                        b1 = fma2(H.B[f][i][j], H.B[f][i][j], b1);
                        b2 = fma2(H.B[f][i][j], B[i][j], b2);
                        z = fma2(Z[j], Z[j], z);
                    }
                }
                // this plane's cubes by weight (over 8), folded into the field's sum
                auto w = [](double c) { return mk2(T(c), T(c)); };
                P t = fma2(w(-0.5), s2, A.wg[f]);
                t = fma2(w(-1.25), b2, t);
                t = fma2(w(-4.0), s1, t);
                t = fma2(w(1.875), z, t);
                t = fma2(w(8.75), b1, t);
                A.wg[f] = fma2(w(39.0), s0, t);
            }
#pragma unroll
            for (int i = 0; i < 3; i++) {
#pragma unroll
                for (int j = 0; j < NP; j++) H.g[f][i][j] = g[i][j];
                H.r[f][i] = re[i];
            }
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < NP; j++) H.B[f][i][j] = B[i][j];
        }
    }

    // Plane k of the boundary column right of the tile at computed row r = lane + 1.
    static __device__ __forceinline__ void plane_edge(const Ctx& C, const Slots& Z, EdgeCol& E)
    {
        const int r = C.lane + 1;
        if (r > C.ty + 1) return;
        const T* Fp = C.S + Z.fp * SLOTF;
        const T* Ep = C.S + EF0 + Z.fp * ESF;
        const T* Epc = C.S + EP0 + Z.pc * ESP;
        T* EGw = C.S + EG0 + Z.g * ESP;
        T cz[2], pn[2];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            T cp, qp, rp;
            aggr_edge(C, Fp + f * FIELDF, Ep + f * EF, r, cp, qp, rp);
            const T d = s_sub(cp, E.c[f]);
            const T lap = s_add(s_fma(T(30), d, E.L[f]), qp);
            pn[f] = s_fma(C.K.dtcl, lap, s_fma(C.K.dtcf, E.c[f], Epc[f * GR + (r - 1)]));
            E.L[f] = s_add(s_fma(T(-30), d, E.q[f]), rp);
            E.q[f] = qp;
            cz[f] = E.c[f];
            E.c[f] = cp;
        }
        T g0, g1;
        site_kick_drift1<T>(C.K, cz[0], cz[1], pn[0], pn[1], g0, g1);
        EGw[r - 1] = g0;
        EGw[GR + (r - 1)] = g1;
    }

    // Plane k of a pair (R = 2; stored) or of the look-ahead row (R = 1): kick and
    // drift.
    template <int R>
    static __device__ __forceinline__ void plane_rows(const Ctx& C, const Slots& Z, Col<R>& Q, int k)
    {
        const T* Fc = C.S + Z.fc * SLOTF + C.offF;
        const T* Fp = C.S + Z.fp * SLOTF;
        const T* Pc = C.S + P0 + Z.pc * SLOTP + C.offP;
        const T* Ep = C.S + EF0 + Z.fp * ESF;
        T* Gw = C.S + G0 + Z.g * SLOTP + C.offP;
        const P c30 = mk2(T(30), T(30)), cm30 = mk2(T(-30), T(-30));
        const P dtcl2 = mk2(C.K.dtcl, C.K.dtcl), dtcf2 = mk2(C.K.dtcf, C.K.dtcf);
        P pn[2][R][NP], cz[2][R][NP], g[2][R][NP];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            P cp[R][NP], qp[R][NP], rp[R][NP];
#pragma unroll
            for (int i = 0; i < R; i++) {
                PK<T>::ld(Pc + f * FIELDP + i * W, pn[f][i]);
                PK<T>::ld(Fc + f * FIELDF + i * RS, cz[f][i]);
            }
            aggr<R>(C, Fp + f * FIELDF, Ep + f * EF, cp, qp, rp);
#pragma unroll
            for (int i = 0; i < R; i++)
#pragma unroll
                for (int j = 0; j < NP; j++) {
                    const P c = cz[f][i][j], d = sub2(cp[i][j], c);
                    const P lap = add2(fma2(c30, d, Q.L[f][i][j]), qp[i][j]);
                    pn[f][i][j] = fma2(dtcl2, lap, fma2(dtcf2, c, pn[f][i][j]));
                    Q.L[f][i][j] = add2(fma2(cm30, d, Q.q[f][i][j]), rp[i][j]);
                    Q.q[f][i][j] = qp[i][j];
                }
        }
        // potential part of the kick and the drift (lat_site.cuh)
#pragma unroll
        for (int i = 0; i < R; i++)
#pragma unroll
            for (int j = 0; j < NP; j++)
                site_kick_drift<T>(C.K, cz[0][i][j], cz[1][i][j], pn[0][i][j], pn[1][i][j], g[0][i][j], g[1][i][j]);
        if (R == 2 && k < C.nz && C.act) {
            const uint32_t gi = (uint32_t)wrapn(C.z0 + k, C.n) * C.nn + C.rowg;
#pragma unroll
            for (int i = 0; i < R; i++) {
                PK<T>::st_stream(C.op0 + gi + i * C.n, pn[0][i]);
                PK<T>::st_stream(C.op1 + gi + i * C.n, pn[1][i]);
            }
        }
#pragma unroll
        for (int i = 0; i < R; i++) {
            PK<T>::st(Gw + i * W, g[0][i]);
            PK<T>::st(Gw + FIELDP + i * W, g[1][i]);
        }
    }

    // One plane: 0, 1 or 2 planes of this run are behind it (2: or more).
    template <int ROLE, int BEHIND, int R>
    static __device__ __forceinline__ void plane(const Ctx& C, Acc& A, Slots& Z, Col<R>& Q, Cube& H, EdgeCol& E, int k)
    {
        cp_async_wait(D - 1);
        __syncthreads();
        if ((ROLE == kSum || ROLE == kAhead) && k + D <= C.nz) {
            fetch_f<ROLE>(C, k + D + 1, Z.fw);
            fetch_p<ROLE>(C, k + D, Z.pw);
        }
        cp_async_commit();
        if constexpr (ROLE == kSum && BEHIND > 0)
            cubes<(BEHIND > 1), true>(C, A, H, C.S + G0 + (Z.g ^ 1) * SLOTP, C.S + EG0 + (Z.g ^ 1) * ESP, k - 1);
        if constexpr (EDGE && ROLE == kAhead) plane_edge(C, Z, E);
        if constexpr (ROLE == kStep || ROLE == kAhead) plane_rows<R>(C, Z, Q, k);
        Z.next();
    }

    // One run of planes: the prologue (planes z0 - 1 .. z0 + D of the fields,
    // z0 .. z0 + D - 1 of the momenta, one commit group per plane step; C, L and q of
    // the first plane into registers), then the planes, and the last cubes, between
    // planes nz - 1 and nz (the look-ahead plane). Every role passes the same
    // barriers.
    template <int ROLE>
    static __device__ __forceinline__ void run(const Ctx& C, Acc& A)
    {
        constexpr int R = ROLE == kStep ? 2 : 1;
        fetch_f<ROLE>(C, -1, 0);
        fetch_f<ROLE>(C, 0, 1);
        fetch_f<ROLE>(C, 1, 2);
        fetch_p<ROLE>(C, 0, 0);
        cp_async_commit();
#pragma unroll
        for (int j = 1; j < D; j++) {
            if (j <= C.nz) {
                fetch_f<ROLE>(C, j + 1, j + 2);
                fetch_p<ROLE>(C, j, j);
            }
            cp_async_commit();
        }
        cp_async_wait(D - 1);
        __syncthreads();
        Col<R> Q;
        Cube H;
        EdgeCol E;
        if constexpr (ROLE == kStep || ROLE == kAhead) {
            const P cm30 = mk2(T(-30), T(-30));
            P cm[R][NP], c[R][NP], q[R][NP], r[R][NP];
#pragma unroll
            for (int f = 0; f < 2; f++) {
                aggr<R>(C, C.S + f * FIELDF, C.S + EF0 + f * EF, cm, Q.q[f], r);
                aggr<R>(C, C.S + SLOTF + f * FIELDF, C.S + EF0 + ESF + f * EF, c, q, r);
#pragma unroll
                for (int i = 0; i < R; i++)
#pragma unroll
                    for (int j = 0; j < NP; j++) {
                        Q.L[f][i][j] = add2(fma2(cm30, sub2(c[i][j], cm[i][j]), Q.q[f][i][j]), r[i][j]);
                        Q.q[f][i][j] = q[i][j];
                    }
            }
        }
        if constexpr (EDGE && ROLE == kAhead) {
            const int r = min(C.lane, C.ty) + 1;
#pragma unroll
            for (int f = 0; f < 2; f++) {
                T cm, qm, rm, cc, qc, rc;
                aggr_edge(C, C.S + f * FIELDF, C.S + EF0 + f * EF, r, cm, qm, rm);
                aggr_edge(C, C.S + SLOTF + f * FIELDF, C.S + EF0 + ESF + f * EF, r, cc, qc, rc);
                E.L[f] = s_add(s_fma(T(-30), s_sub(cc, cm), qm), rc);
                E.q[f] = qc;
                E.c[f] = cc;
            }
        }
        // planes 0 and 1 have fewer cubes to add; the rest is one straight body
        Slots Z{1, 2, 0, 0, RP - 1, 0};
        plane<ROLE, 0>(C, A, Z, Q, H, E, 0);
        plane<ROLE, 1>(C, A, Z, Q, H, E, 1);
        // (unrolled by two it was 120 us against 117 at 256^3, with spills)
#pragma unroll 1
        for (int k = 2; k <= C.nz; k++) plane<ROLE, 2>(C, A, Z, Q, H, E, k);
        __syncthreads();
        if constexpr (ROLE == kSum)
            cubes<true, false>(C, A, H, C.S + G0 + (Z.g ^ 1) * SLOTP, C.S + EG0 + (Z.g ^ 1) * ESP, C.nz);
    }

    // The runs of the block's group, for a warp of pair row `row` (look-ahead warp:
    // 0) of its tiles.
    template <int ROLE>
    static __device__ __forceinline__ void walk(Ctx& C, Acc& A, TileWalk runs, int nyt, int x0, int row)
    {
        const int n = C.n;
        int yt;
        for (bool first = true; runs.run(yt, C.z0, C.nz); first = false) {
            runs.took(C.nz);
            const int y0 = 2 * (yt * (n / 2) / nyt);
            C.ty = 2 * ((yt + 1) * (n / 2) / nyt) - y0;
            C.row = ROLE == kAhead ? C.ty + 1 : row;
            C.offF = (uint32_t)C.row * RS + C.lane * VW;
            C.offP = (uint32_t)(C.row - 1) * W + C.lane * VW;
            const uint32_t xg = x0 + C.lane * VW;
            C.rowg = (uint32_t)wrapn(y0 + C.row - 1, n) * n + xg;
            C.rowlo = (uint32_t)wrapn(y0 - 1, n) * n + xg;
            C.rowhi = (uint32_t)wrapn(y0 + C.ty + 1, n) * n + xg;
            C.ey = (uint32_t)wrapn(y0 - 1 + min(C.lane, C.ty + 2), n) * n;
            C.eyp = (uint32_t)wrapn(y0 + min(C.lane, C.ty), n) * n;
            // every thread is done with the previous segment's ring before the
            // prologue refills it
            if (!first) __syncthreads();
            if (ROLE == kAhead || row <= C.ty) run<ROLE>(C, A);
            else run<kIdle>(C, A);
        }
    }
};

template <typename T, int TY, int D, bool EDGE>
__global__ void __launch_bounds__(S27<T, TY, D, EDGE>::THREADS, 1)
    step27w_kernel(Bufs<T> B, Model M, DevScalars* sc, double* partials)
{
    typedef S27<T, TY, D, EDGE> F;
    constexpr int VW = F::VW;
    __shared__ double red[32 * kSums];
    extern __shared__ __align__(16) unsigned char smem_raw[];

    typename F::Ctx C;
    C.S = reinterpret_cast<T*>(smem_raw);
    const int warp = threadIdx.x >> 5;
    // warps: a step warp for each pair, then the look-ahead warp, then a
    // sum warp for each pair
    C.lane = threadIdx.x & 31;
    // groups of nxt blocks: the x tiles of one y tile, marching the same (y tile, z
    // plane) units (lat_layout.cuh); the row's vectors are shared
    // evenly among the x tiles, cut at multiples of 64 bytes where the row is one,
    // the pairs of rows among the y tiles
    const int n = M.n;
    C.n = n;
    C.nn = (uint32_t)n * n;
    const int Q = n / VW, cut = Q % 4 == 0 ? 4 : Q % 2 == 0 ? 2 : 1;
    const int nxt = EDGE ? (Q + 31) / 32 : 1, nyt = (n + TY - 1) / TY;
    const int ngroups = gridDim.x / nxt;
    const int grp = blockIdx.x / nxt, xt = blockIdx.x - grp * nxt;
    const int q0 = xt * (Q / cut) / nxt * cut, qn = (xt + 1) * (Q / cut) / nxt * cut - q0;
    const int x0 = q0 * VW, x1 = x0 + qn * VW;
    C.last = qn - 1;
    C.act = C.lane < qn;
    // EDGE: what the end lanes get from the shuffles is replaced by edge scalars
    C.sl = EDGE ? max(C.lane - 1, 0) : C.lane == 0 ? C.last : C.lane - 1;
    C.sr = EDGE ? min(C.lane + 1, 31) : C.lane >= C.last ? 0 : C.lane + 1;
    C.exl = (uint32_t)(x0 == 0 ? n - 1 : x0 - 1);
    C.exr = (uint32_t)(x1 == n ? 0 : x1);
    C.exr1 = (uint32_t)(x1 + 1 >= n ? x1 + 1 - n : x1 + 1);
    TileWalk runs(nyt, ngroups, grp, n);

    chain_begin();
    if (sc->status != LAT_OK) return;
    const bool par = (sc->step & 1) != 0;
    C.f0 = par ? B.f[1][0] : B.f[0][0];
    C.f1 = par ? B.f[1][1] : B.f[0][1];
    C.p0 = par ? B.p[1][0] : B.p[0][0];
    C.p1 = par ? B.p[1][1] : B.p[0][1];
    C.of0 = par ? B.f[0][0] : B.f[1][0];
    C.of1 = par ? B.f[0][1] : B.f[1][1];
    C.op0 = par ? B.p[0][0] : B.p[1][0];
    C.op1 = par ? B.p[0][1] : B.p[1][1];
    C.K = site_coefs<T>(sc, M.beta);
    typename F::Acc A;
    A.wg[0] = A.wg[1] = A.vd = A.vi = mk2(T(0), T(0));
    if (warp < F::PAIRS) F::template walk<kStep>(C, A, runs, nyt, x0, 2 * warp + 1);
    else if (warp == F::PAIRS) F::template walk<kAhead>(C, A, runs, nyt, x0, 0);
    else {
        typename F::Acc S = A;
        F::template walk<kSum>(C, S, runs, nyt, x0, 2 * (warp - F::PAIRS) - 1);
        if (C.act) A = S;   // nothing in the other lanes
    }

    // the pairs' two halves are added with their rounding errors beside them
    TreeSum<T> v[kSums];
    const T vf = site_vsum_factor<T>(C.K.quartic);   // factors of 1/2 and 1/4 are exact
    auto both = [](typename F::P p, T f) {
        TreeSum<T> a, b;
        a.init(f * lo2(p));
        b.init(f * hi2(p));
        a.add(b);
        return a;
    };
    v[0] = both(A.wg[0], T(1));
    v[1] = both(A.wg[1], T(1));
    v[2] = both(A.vd, vf);
    v[3] = both(A.vi, T(0.5));
    finish_block_trees<T>(M, sc, partials, v, red, true);
}

// The compiled instance for a side, tile height and prefetch depth, or null.
template <typename T>
const void* s27w_fn(int n, int ty, int depth, size_t* smem)
{
    constexpr bool kRows = sizeof(T) == 4;   // sides up to 64 are the plane-ring kernel's: FP64 rows are always cut
    const bool edge = n > 32 * (int)(16 / sizeof(T));
#define LAT_S27W_CASE(TT, DD)                                                  \
    if (ty == TT && depth == DD) {                                             \
        *smem = edge ? S27<T, TT, DD, true>::SMEM : S27<T, TT, DD, !kRows>::SMEM; \
        return edge ? (const void*)step27w_kernel<T, TT, DD, true>             \
                    : (const void*)step27w_kernel<T, TT, DD, !kRows>;          \
    }
    LAT_S27W_CASE(14, 2) LAT_S27W_CASE(16, 1)
#undef LAT_S27W_CASE
    return nullptr;
}

} // namespace

bool s27w_config(int n, int elem_bytes, int ty, int zr, int depth, MarchConfig* cfg)
{
    // FP32: tiles of 14 rows, two planes in flight (15 warps, 128 registers each,
    // nothing spilled): 256^3 107 us per step against 151 with 16 rows and one plane
    // (17 warps, 96 registers), 512^3 760 against 1108, 100^3 17.9 against 18.8; 14 rows
    // with one plane in flight 120 and 879, with three 111 and 770. FP64 is bound by its FP64 pipe, so the rows computed count: 16
    // where they divide a larger side (128^3 496 against 538 us, 160^3 1070 against
    // 1118, 256^3 3497 against 3539), else 14 (96^3 289 against 302, 132^3 790
    // against 831).
    const int best = elem_bytes == 8 && n % 16 == 0 && n >= 128 ? 16 : 14;
    const int tyv = ty > 0 ? ty : depth > 0 ? (depth == 1 ? 16 : 14) : best;
    const int d = depth > 0 ? depth : tyv == 14 ? 2 : 1;
    size_t smem = 0;
    const void* fn = elem_bytes == 4 ? s27w_fn<float>(n, tyv, d, &smem) : s27w_fn<double>(n, tyv, d, &smem);
    // up to 64 the plane-ring kernel (variant 2) runs every side
    if (!fn || smem > 227 * 1024 - 2048 || n <= 64) return false;
    const int vw = 16 / elem_bytes, nxt = (n / vw + 31) / 32;
    const int threads = (tyv + 1) * 32;
    if (allow_dynamic_smem(fn, smem) != cudaSuccess) return false;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess || occ < 1) return false;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return false;
    const int nyt = (n + tyv - 1) / tyv;
    const long long tiles = (long long)nyt * nxt, units = tiles * n;
    long long blocks = 0;
    // whole groups of nxt blocks (the x tiles of a y tile, marching together)
    if (zr > 0) blocks = tiles * ((n + std::min(zr, n) - 1) / std::min(zr, n));
    else blocks = std::min((long long)sms * occ, units) / nxt * nxt;
    if (blocks < nxt) return false;
    const long long groups = blocks / nxt;
    cfg->ty = tyv;
    const Layout L0 = tile_layout(nyt, (int)groups, 0, n);   // the first group's first run
    cfg->zr = std::min(L0.uend - L0.ubeg, L0.zspan);
    cfg->nzc = (int)((groups + nyt - 1) / nyt);
    cfg->depth = d;
    cfg->threads = threads;
    cfg->maxt = threads;
    cfg->fast = 1;
    cfg->smem = smem;
    cfg->nyt = nyt;
    cfg->blocks = (int)blocks;
    cfg->nzl = 0;
    cfg->zbase = 0;
    cfg->s27 = 1;
    cfg->xt = 0;
    cfg->xw = 1;
    cfg->nxt = nxt;
    return true;
}

template <typename T>
cudaError_t launch_step27w(const Bufs<T>& b, const Model& M, DevScalars* sc, double* partials, const MarchConfig& cfg,
                           cudaStream_t st)
{
    size_t smem = 0;
    const void* fn = s27w_fn<T>(M.n, cfg.ty, cfg.depth, &smem);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {(void*)&b, (void*)&M, (void*)&sc, (void*)&partials};
    return launch_chained(fn, dim3(cfg.blocks), dim3(cfg.threads), args, cfg.smem, st, cfg.chain);
}

template cudaError_t launch_step27w<float>(const Bufs<float>&, const Model&, DevScalars*, double*, const MarchConfig&,
                                           cudaStream_t);
template cudaError_t launch_step27w<double>(const Bufs<double>&, const Model&, DevScalars*, double*,
                                            const MarchConfig&, cudaStream_t);

} // namespace lat

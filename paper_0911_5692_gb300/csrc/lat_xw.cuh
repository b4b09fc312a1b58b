// lat_xw.cuh -- the fused 7-point step over x tiles one warp wide (variant 5),
// with the tile height TY and the prefetch depth D known at compile time and the
// lattice side taken at run time.
//
// The same step as the other plane-ring kernels (Sec. II.B, eq. evo with eq.
// scalar-evo; the sums of the new fields for eq. scale from the +y row and +z
// plane look-ahead; the FP64 a(t) update in the last block). A tile is at most W
// = 32 16-byte vectors wide (128 FP32 or 64 FP64 columns; a row's vectors are
// shared evenly among its tiles) and at most TY rows tall. Each of TY / 2 warps
// owns two neighbouring rows, a lane one vector of each, and marches them along
// z; one more warp stages the halo rows and kicks and drifts the look-ahead row;
// and the edge warp stages, per row and plane, the scalars the tile needs from
// its x neighbours: f at x0 - 1 (left Laplacian neighbour of lane 0), right of
// the tile and one further, and the momenta right of the tile. From them it
// kicks and drifts the boundary column of the owned rows, rounded exactly as the
// neighbouring tile rounds the same sites, for the x differences of the sums.
//
// What bounds it. Per plane and owned row a thread reads its vectors of the new
// plane, of the momenta and, for a pair of rows, of the two rows beside the
// pair; the centre, the difference to the plane below and the new field stay in
// registers from plane to plane, and the new field crosses warps for one row of
// the pair only. That is about half the shared-memory traffic and 15 % fewer
// instructions than one row per warp with every neighbour read from the ring
// (33.9 M against 40 M warp instructions per 256^3 launch), and a third of the
// warps in each barrier. In its steady state the kernel now moves a plane of
// full tiles at the copy rate (256^3: 1.55 us per plane of every block, 6.4 TB/s);
// what is left at 256^3 is the ramp at both ends. 512^3 FP32 713 -> 685 us (93 %
// of the measured copy rate), 256^3 102.7 -> 98, and the sides that no instance
// was compiled for before: 384^3 435 -> 298, 320^3 232 -> 209, 200^3 73 -> 62.
// The side as a compile-time constant was slower (512^3: 737 against 692 us),
// and so were longer unrolled plane loops (see run()).
//
// The x tiles of a y tile are taken by consecutive blocks that march the same (y
// tile, z plane) units at the same time, so the scalars one tile reads from its
// neighbours' columns lie in memory lines the neighbouring blocks are reading
// too (L2 hits); and neighbouring y tiles are marched at the same planes at the
// same time (lat_layout.cuh), so that a tile's halo rows, its neighbours' owned
// rows, are L2 hits too. The new state is written with streaming stores: only
// the next step reads it.
//
// SLAB instances step z ranges of the owned planes of one or several z-slabs
// (stored planes with their halos, no wrap in z; each slab with its own
// arrays), laid end to end in z for the block layout, and write the ranges'
// summed shares of the volume averages instead of advancing the scalars
// (lat_slab.cu).
#pragma once

#include <algorithm>

#include "lat_async.cuh"
#include "lat_layout.cuh"
#include "lat_kernels.h"
#include "lat_pairs.cuh"
#include "lat_site.cuh"

namespace lat {

namespace xw {

enum { kPair, kAhead, kEdge, kIdle };   // warp roles

// SW = 0: x tiles of up to 32 vectors and an edge warp. SW = 8, 16 or 32: rows of
// one tile of at most SW vectors, 32 / SW pairs of rows to a warp; the row's ends
// are each other's neighbours, reached by a shuffle, and there is no edge warp.
template <typename T, int TY, int D, bool SLAB, int SW = 0>
struct XW {
    typedef typename PK<T>::P P;
    static constexpr int RF = D + 2, RP = D + 1;       // field and momentum plane slots
    static constexpr int NP = PK<T>::NP;
    static constexpr int VW = 2 * NP;                  // elements per 16-byte vector
    static constexpr bool EDGE = SW == 0;
    static constexpr int LW = EDGE ? 32 : SW;          // lanes of a row
    static constexpr int RPW = 32 / LW;                // pairs of rows to a warp
    static constexpr int W = LW * VW;                  // tile width
    static constexpr int ROWS = TY + 3;                // staged rows
    static constexpr int PAIRS = TY / 2;               // pairs of owned rows
    static constexpr int PWARPS = PAIRS / RPW;         // warps that own them
    static constexpr int THREADS = (PWARPS + (EDGE ? 2 : 1)) * 32;   // and the look-ahead and edge warps
    static_assert(TY % 2 == 0 && PAIRS % RPW == 0, "row pairs");
    static_assert(!EDGE || ROWS <= 32, "the edge warp has a lane per row");
    // shared memory, in elements: the field ring [slot][field][ROWS][W], the
    // momentum ring [slot][field][TY + 1][W], the new fields of each pair's first
    // row and of the look-ahead row [buf][field][PAIRS + 1][W]; then the edge
    // scalars: fields [slot][field][ROWS][4] (x0 - 1, x0 + W, x0 + W + 1, unused),
    // momenta [slot][field][TY] at x0 + W, new fields [buf][field][TY] at x0 + W
    static constexpr uint32_t FIELDF = ROWS * W, SLOTF = 2 * FIELDF;
    static constexpr uint32_t FIELDP = (TY + 1) * W, SLOTP = 2 * FIELDP;
    static constexpr uint32_t FIELDG = (PAIRS + 1) * W, BUFG = 2 * FIELDG;
    static constexpr uint32_t P0 = RF * SLOTF, G0 = P0 + RP * SLOTP;
    static constexpr uint32_t EF = ROWS * 4, ESF = 2 * EF;
    static constexpr uint32_t EPF = TY, ESP = 2 * EPF;
    static constexpr uint32_t EF0 = G0 + 2 * BUFG, EP0 = EF0 + RF * ESF, EG0 = EP0 + RP * ESP;
    static constexpr uint32_t END = EDGE ? EG0 + 2 * 2 * TY : EF0;
    static constexpr size_t SMEM = (sizeof(T) * (size_t)END + 15) / 16 * 16;

    struct Ctx {
        T* S;
        uint32_t nn;                     // n^2
        int n, ty, last;                 // side, owned rows of the tile (even), its last lane
        bool act;                        // this lane holds a vector of the tile
        uint32_t offF, offP, offG;       // this thread's vector of its (first) row: field, momentum, new-field planes
        uint32_t rowg, rowlo, rowhi;     // global offsets in a plane: its (first) row; the halo rows (look-ahead warp)
        int lx, sl, sr;                  // its vector in the row; SW: the lanes of the neighbouring vectors
        int row, lane, z0, nz;           // its (first) row in the staged tile
        int zb;                          // SLAB: stored plane of the run's z = 0
        uint32_t ey, eyp;                // edge warp: offsets in a plane of its staged row and of owned row lane + 1
        uint32_t exl, exr, exr1;         // the three edge columns
        const T *f0, *f1, *p0, *p1;
        T *of0, *of1, *op0, *op1;
        P dtcl2, dtcf2;
        SiteCoefs<T> K;
    };
    // A lane of the pair warps or of the look-ahead warp in a tile of ty rows and qn
    // vectors: its (first) row in the staged tile, whether it holds a vector of it (lx
    // in its row), and where that lies in the new-field plane.
    static __host__ __device__ __forceinline__ int pair_of(int warp, int lane) { return warp * RPW + lane / LW; }
    static __host__ __device__ __forceinline__ int row_of(bool ahead, int pair, int ty) { return ahead ? ty + 1 : 2 * pair + 1; }
    static __host__ __device__ __forceinline__ bool holds(bool ahead, int pair, int lane, int lx, int qn, int ty)
    {
        return EDGE ? lx < qn : lx < qn && (ahead ? lane < LW : 2 * pair < ty);
    }
    static __host__ __device__ __forceinline__ uint32_t off_g(int row, int lx) { return (uint32_t)((row - 1) / 2) * W + lx * VW; }
    // Whether it stores its new field for the other warps. With several pairs to a warp
    // the last warp may reach past the tile's last row, and a pair just past it lies
    // where the look-ahead row does: the lanes that hold nothing store nothing, so that
    // every vector of the plane has one writer. (With x tiles those lanes' vectors are
    // their own.)
    static __host__ __device__ __forceinline__ bool shares(bool act) { return EDGE || act; }
    // the ring slots of one plane step, as offsets: field plane k, k + 1 and the
    // slot that plane k - 1 left; momentum plane k and the slot that k - 1 left
    struct Slots {
        int fc, fp, fw, pc, pw;
    };
    // carried from plane to plane in registers, for each field and row: the
    // centre vector, its difference to the plane below, the new field
    template <int R>
    struct Col {
        P c[2][R][NP], dz[2][R][NP], g[2][R][NP];
    };
    struct Acc {
        P g[2][2], vd[2], vi[2];   // [field][row] and [row], both pairs of a vector together
        __device__ __forceinline__ void zero()
        {
            const P z = mk2(T(0), T(0));
#pragma unroll
            for (int r = 0; r < 2; r++) g[0][r] = g[1][r] = vd[r] = vi[r] = z;
        }
        __device__ __forceinline__ void add(const Acc& b)
        {
#pragma unroll
            for (int r = 0; r < 2; r++) {
                g[0][r] = add2(g[0][r], b.g[0][r]);
                g[1][r] = add2(g[1][r], b.g[1][r]);
                vd[r] = add2(vd[r], b.vd[r]);
                vi[r] = add2(vi[r], b.vi[r]);
            }
        }
    };

    // array plane of run plane z0 + zrel: periodic in z for a whole lattice; a
    // slab's stored planes carry the halos, so no wrap
    static __device__ __forceinline__ uint32_t zplane(const Ctx& C, int zrel)
    {
        if constexpr (SLAB) return (uint32_t)(C.z0 + zrel + C.zb);
        else return (uint32_t)wrapn(C.z0 + zrel, C.n);
    }

    // plane z0 + zrel of the fields into slot `slot`: a pair's two rows; the
    // look-ahead warp its row and the two halo rows; the edge warp (lane r for
    // staged row r) the three edge scalars of each field
    template <int ROLE>
    static __device__ __forceinline__ void fetch_f(const Ctx& C, int zrel, int slot)
    {
        const uint32_t zoff = zplane(C, zrel) * C.nn;
        if constexpr (ROLE == kPair) {
            const T *a = C.f0 + zoff + C.rowg, *b = C.f1 + zoff + C.rowg;
            T* d = C.S + slot * SLOTF + C.offF;
            if (C.act) {
                cp_async16(d, a);
                cp_async16(d + W, a + C.n);
                cp_async16(d + FIELDF, b);
                cp_async16(d + FIELDF + W, b + C.n);
            }
        } else if constexpr (ROLE == kAhead) {
            T* d = C.S + slot * SLOTF + C.offF;
            T* lo = C.S + slot * SLOTF + C.lx * VW;
            if (C.act) {
                cp_async16(lo, C.f0 + zoff + C.rowlo);
                cp_async16(lo + FIELDF, C.f1 + zoff + C.rowlo);
                cp_async16(d, C.f0 + zoff + C.rowg);
                cp_async16(d + FIELDF, C.f1 + zoff + C.rowg);
                cp_async16(d + W, C.f0 + zoff + C.rowhi);
                cp_async16(d + FIELDF + W, C.f1 + zoff + C.rowhi);
            }
        } else if constexpr (ROLE == kEdge) {
            if (C.lane < C.ty + 3) {
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
    // momenta of plane z0 + zrel: the computing rows' vectors, and the momenta at
    // x0 + W of the owned rows (edge warp, lane r - 1 for row r)
    template <int ROLE>
    static __device__ __forceinline__ void fetch_p(const Ctx& C, int zrel, int slot)
    {
        const uint32_t zoff = zplane(C, zrel) * C.nn;
        if constexpr (ROLE == kPair || ROLE == kAhead) {
            const T *a = C.p0 + zoff + C.rowg, *b = C.p1 + zoff + C.rowg;
            T* d = C.S + P0 + slot * SLOTP + C.offP;
            if (C.act) {
                cp_async16(d, a);
                cp_async16(d + FIELDP, b);
                if constexpr (ROLE == kPair) {
                    cp_async16(d + W, a + C.n);
                    cp_async16(d + FIELDP + W, b + C.n);
                }
            }
        } else if constexpr (ROLE == kEdge) {
            if (C.lane < C.ty) {
                const uint32_t gb = zoff + C.eyp + C.exr;
                T* e = C.S + EP0 + slot * ESP + C.lane;
                cp_async_small<sizeof(T)>(e, C.p0 + gb);
                cp_async_small<sizeof(T)>(e + EPF, C.p1 + gb);
            }
        }
    }

    // The boundary column x0 + W of owned row r = lane + 1, rounded as the
    // neighbouring tile rounds its own first column (edge warp; cc and dzp carry
    // its centre and the difference to the plane below).
    template <int J>
    static __device__ __forceinline__ void edge_column(const Ctx& C, const Slots& Z, T (&cc)[2], T (&dzp)[2], bool ahead)
    {
        const T* Fc = C.S + Z.fc * SLOTF;
        const T* Ec = C.S + EF0 + Z.fc * ESF;
        const T* Ep = C.S + EF0 + Z.fp * ESF;
        const T* Epc = C.S + EP0 + Z.pc * ESP;
        T* EGw = C.S + EG0 + J * 2 * TY;
        const int r = C.lane + 1;
        if (r > C.ty || ahead) return;
        T pn[2], zp[2];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            const T* e = Ec + f * EF;
            const T left = Fc[f * FIELDF + r * W + C.last * VW + VW - 1];
            const T right = e[r * 4 + 2];
            const T up = e[(r - 1) * 4 + 1], dn = e[(r + 1) * 4 + 1];
            zp[f] = Ep[f * EF + r * 4 + 1];
            const T dz = s_sub(zp[f], cc[f]);
            const T lap = s_add(s_add(s_add(s_sub(left, cc[f]), s_sub(right, cc[f])),
                                      s_add(s_sub(up, cc[f]), s_sub(dn, cc[f]))), s_sub(dz, dzp[f]));
            dzp[f] = dz;
            pn[f] = s_fma(C.K.dtcl, lap, s_fma(C.K.dtcf, cc[f], Epc[f * EPF + (r - 1)]));
        }
        T g0, g1;
        site_kick_drift1<T>(C.K, cc[0], cc[1], pn[0], pn[1], g0, g1);
        EGw[r - 1] = g0;
        EGw[TY + (r - 1)] = g1;
        cc[0] = zp[0];
        cc[1] = zp[1];
    }

    // One plane of a row pair (R = 2) or of the look-ahead row (R = 1).
    template <int J, int R>
    static __device__ __forceinline__ void rows_plane(const Ctx& C, const Slots& Z, Col<R>& Q, Acc& A, int k, bool ahead)
    {
        constexpr bool own = R == 2;
        const T* Fc = C.S + Z.fc * SLOTF + C.offF;
        const T* Fp = C.S + Z.fp * SLOTF + C.offF;
        const T* Pc = C.S + P0 + Z.pc * SLOTP + C.offP;
        T* Gw = C.S + G0 + J * BUFG + C.offG;
        const T* Gr = C.S + G0 + (1 - J) * BUFG + C.offG;
        const T* Ec = C.S + EF0 + Z.fc * ESF + C.row * 4;
        const T* EGr = C.S + EG0 + (1 - J) * 2 * TY + (C.row - 1);

        if (!own && ahead) return;   // the look-ahead row of the look-ahead plane is not needed
        P g[2][R][NP], pn[2][R][NP];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            P zp[R][NP], up[NP], dn[NP];
            PK<T>::ld(Fc + f * FIELDF - W, up);
            PK<T>::ld(Fc + f * FIELDF + R * W, dn);
#pragma unroll
            for (int r = 0; r < R; r++) PK<T>::ld(Fp + f * FIELDF + r * W, zp[r]);
#pragma unroll
            for (int r = 0; r < R; r++) PK<T>::ld(Pc + f * FIELDP + r * W, pn[f][r]);
#pragma unroll
            for (int r = 0; r < R; r++) {
                P(&c)[NP] = Q.c[f][r];
                // the neighbours in x of the vector's ends: the next lanes', or the
                // tile's edge values (a predicated load, no branch on the lane)
                T left, right;
                if constexpr (EDGE) {
                    left = ld_shared_if(C.lane == 0, Ec + f * EF + r * 4, __shfl_up_sync(0xffffffffu, hi2(c[NP - 1]), 1));
                    right = ld_shared_if(C.lane == C.last, Ec + f * EF + r * 4 + 1,
                                         __shfl_down_sync(0xffffffffu, lo2(c[0]), 1));
                } else {
                    left = __shfl_sync(0xffffffffu, hi2(c[NP - 1]), C.sl);
                    right = __shfl_sync(0xffffffffu, lo2(c[0]), C.sr);
                }
                T d[VW];
                xdiff<T>(c, right, d);
                const T dl = s_sub(lo2(c[0]), left);
#pragma unroll
                for (int v = 0; v < NP; v++) {
                    const P lx = mk2(s_sub(d[2 * v], v == 0 ? dl : d[2 * v - 1]), s_sub(d[2 * v + 1], d[2 * v]));
                    // Laplacian as a sum of neighbour differences (exact
                    // differences for f = const + small), each formed once: the
                    // y difference inside the pair serves both rows, the z
                    // difference this plane and the next
                    P ly;
                    if constexpr (R == 2) {
                        const P in = sub2(Q.c[f][1][v], Q.c[f][0][v]);
                        ly = r == 0 ? add2(sub2(up[v], c[v]), in) : sub2(sub2(dn[v], c[v]), in);
                    } else {
                        ly = add2(sub2(up[v], c[v]), sub2(dn[v], c[v]));
                    }
                    const P dz = sub2(zp[r][v], c[v]);
                    const P lap = add2(add2(lx, ly), sub2(dz, Q.dz[f][r][v]));
                    Q.dz[f][r][v] = dz;
                    pn[f][r][v] = fma2(C.dtcl2, lap, fma2(C.dtcf2, c[v], pn[f][r][v]));
                }
            }
            // the centres of the next plane; this plane's are needed once more below
#pragma unroll
            for (int r = 0; r < R; r++)
#pragma unroll
                for (int v = 0; v < NP; v++) g[f][r][v] = Q.c[f][r][v], Q.c[f][r][v] = zp[r][v];
        }
        // potential part of the kick and the drift (lat_site.cuh)
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
            for (int v = 0; v < NP; v++) {
                const P c0 = g[0][r][v], c1 = g[1][r][v];
                site_kick_drift<T>(C.K, c0, c1, pn[0][r][v], pn[1][r][v], g[0][r][v], g[1][r][v]);
            }
        if (!ahead) {
            if (own && C.act) {
                const uint32_t gi = zplane(C, k) * C.nn + C.rowg;
                // the new state is read again only by the next step
#pragma unroll
                for (int r = 0; r < R; r++) {
                    PK<T>::st_stream(C.op0 + gi + r * C.n, pn[0][r]);
                    PK<T>::st_stream(C.op1 + gi + r * C.n, pn[1][r]);
                    PK<T>::st_stream(C.of0 + gi + r * C.n, g[0][r]);
                    PK<T>::st_stream(C.of1 + gi + r * C.n, g[1][r]);
                }
            }
            if (shares(C.act)) {
                PK<T>::st(Gw, g[0][0]);
                PK<T>::st(Gw + FIELDG, g[1][0]);
            }
        }
        // sums over the owned rows of plane k-1 (x and y pairs, potential) and
        // the z pair (k-1, k); the row after the pair's second is the next pair's
        // first, written to shared memory one plane ago; the last lane's x pair
        // ends on the boundary column the edge warp computed
        if constexpr (own) {
            if (k > 0) {
#pragma unroll
                for (int f = 0; f < 2; f++) {
                    P yn[NP];
                    PK<T>::ld(Gr + f * FIELDG + W, yn);
#pragma unroll
                    for (int r = 0; r < R; r++) {
                        P(&q)[NP] = Q.g[f][r];
                        T right;
                        if constexpr (EDGE)
                            right = ld_shared_if(C.lane == C.last, EGr + f * TY + r, __shfl_down_sync(0xffffffffu, lo2(q[0]), 1));
                        else right = __shfl_sync(0xffffffffu, lo2(q[0]), C.sr);
                        T d[VW];
                        xdiff<T>(q, right, d);
#pragma unroll
                        for (int v = 0; v < NP; v++) {
                            const P dxv = mk2(d[2 * v], d[2 * v + 1]);
                            const P dyv = sub2(r + 1 < R ? Q.g[f][R - 1][v] : yn[v], q[v]);
                            const P dzv = sub2(g[f][r][v], q[v]);
                            A.g[f][r] = fma2(dxv, dxv, fma2(dyv, dyv, fma2(dzv, dzv, A.g[f][r])));
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < R; r++)
#pragma unroll
                    for (int v = 0; v < NP; v++) site_vsum<T>(C.K, Q.g[0][r][v], Q.g[1][r][v], A.vd[r], A.vi[r]);
            }
#pragma unroll
            for (int f = 0; f < 2; f++)
#pragma unroll
                for (int r = 0; r < R; r++)
#pragma unroll
                    for (int v = 0; v < NP; v++) Q.g[f][r][v] = g[f][r][v];
        }
    }

    // what a warp of each role carries, and its plane
    template <int ROLE>
    struct Carry {
        Col<ROLE == kPair ? 2 : 1> q;
        T cc[2], dzp[2];   // edge warp
    };

    // J = k & 1: the new-field buffer of the plane
    template <int J, int ROLE>
    static __device__ __forceinline__ void plane(const Ctx& C, Slots& Z, Carry<ROLE>& Y, Acc& A, int k)
    {
        cp_async_wait(D - 1);
        __syncthreads();
        if (ROLE != kIdle && k + D <= C.nz) {
            fetch_f<ROLE>(C, k + D + 1, Z.fw);
            fetch_p<ROLE>(C, k + D, Z.pw);
        }
        cp_async_commit();
        if constexpr (ROLE == kEdge) edge_column<J>(C, Z, Y.cc, Y.dzp, k == C.nz);
        else if constexpr (ROLE == kPair) rows_plane<J, 2>(C, Z, Y.q, A, k, k == C.nz);
        else if constexpr (ROLE == kAhead) rows_plane<J, 1>(C, Z, Y.q, A, k, k == C.nz);
        Z.fw = Z.fc;
        Z.fc = Z.fp;
        Z.fp = Z.fp + 1 == RF ? 0 : Z.fp + 1;
        Z.pw = Z.pc;
        Z.pc = Z.pc + 1 == RP ? 0 : Z.pc + 1;
    }

    // one run of planes: the prologue (planes z0 - 1 .. z0 + D of the fields,
    // z0 .. z0 + D - 1 of the momenta, one commit group per plane step; the first
    // two planes into registers), then the planes; every role passes the same
    // barriers
    template <int ROLE>
    static __device__ __forceinline__ void run(const Ctx& C, Acc& A)
    {
        fetch_f<ROLE>(C, -1, 0);
        fetch_f<ROLE>(C, 0, 1);
        fetch_f<ROLE>(C, 1, 2);
        fetch_p<ROLE>(C, 0, 0);
        cp_async_commit();
#pragma unroll
        for (int j = 1; j < D; j++) {
            if (j <= C.nz) {   // a run shorter than the depth prefetches up to its look-ahead plane
                fetch_f<ROLE>(C, j + 1, j + 2);
                fetch_p<ROLE>(C, j, j);
            }
            cp_async_commit();
        }
        cp_async_wait(D - 1);
        __syncthreads();
        Carry<ROLE> Y;
        if constexpr (ROLE == kPair || ROLE == kAhead) {
            constexpr int R = ROLE == kPair ? 2 : 1;
#pragma unroll
            for (int f = 0; f < 2; f++)
#pragma unroll
                for (int r = 0; r < R; r++) {
                    P zm[NP];
                    PK<T>::ld(C.S + C.offF + f * FIELDF + r * W, zm);
                    PK<T>::ld(C.S + SLOTF + C.offF + f * FIELDF + r * W, Y.q.c[f][r]);
#pragma unroll
                    for (int v = 0; v < NP; v++) Y.q.dz[f][r][v] = sub2(Y.q.c[f][r][v], zm[v]);
                }
        } else if constexpr (ROLE == kEdge) {
            const T* e = C.S + EF0 + (min(C.lane, C.ty - 1) + 1) * 4 + 1;
#pragma unroll
            for (int f = 0; f < 2; f++) {
                Y.cc[f] = e[ESF + f * EF];
                Y.dzp[f] = s_sub(Y.cc[f], e[f * EF]);
            }
        }
        // two planes per turn: the carried registers and the new-field buffers
        // alternate without moves. More (the ring's period, with constant slots)
        // overflows the instruction cache: 0.71 ms per 512^3 step with 4 planes,
        // 1.04 ms with 6, 1.27 ms with 10.
        Slots Z{1, 2, 0, 0, RP - 1};
        for (int k = 0;; k += 2) {
            plane<0, ROLE>(C, Z, Y, A, k);
            if (k + 1 > C.nz) break;
            plane<1, ROLE>(C, Z, Y, A, k + 1);
            if (k + 2 > C.nz) break;
        }
    }

    // March planes C.z0 .. C.z0 + C.nz - 1 of the tile of rows y0 .. y0 + ty - 1 (ty
    // even) and vectors q0 .. q0 + qn - 1. `first`: no earlier run of this block is
    // still reading the ring.
    static __device__ __forceinline__ void march(Ctx& C, int warp, int q0, int qn, int y0, int ty, bool first, Acc& A)
    {
        const int n = C.n;
        const bool ahead = warp == PWARPS;
        C.lane = threadIdx.x & 31;
        C.lx = C.lane % LW;
        C.ty = ty;
        C.last = qn - 1;
        const int pair = pair_of(warp, C.lane);
        C.act = holds(ahead, pair, C.lane, C.lx, qn, ty);
        C.row = row_of(ahead, pair, ty);
        if constexpr (!EDGE) {
            C.sl = C.lane - C.lx + (C.lx == 0 ? qn - 1 : C.lx - 1);
            C.sr = C.lane - C.lx + (C.lx + 1 >= qn ? 0 : C.lx + 1);
        }
        C.offF = (uint32_t)C.row * W + C.lx * VW;
        C.offP = (uint32_t)(C.row - 1) * W + C.lx * VW;
        C.offG = off_g(C.row, C.lx);
        const int x0 = q0 * VW, x1 = x0 + qn * VW;
        const uint32_t xg = x0 + C.lx * VW;
        C.rowg = (uint32_t)wrapn(y0 + C.row - 1, n) * n + xg;
        C.rowlo = (uint32_t)wrapn(y0 - 1, n) * n + xg;
        C.rowhi = (uint32_t)wrapn(y0 + ty + 1, n) * n + xg;
        if constexpr (EDGE) {
            C.ey = (uint32_t)wrapn(y0 - 1 + min(C.lane, ty + 2), n) * n;
            C.eyp = (uint32_t)wrapn(y0 + min(C.lane, ty - 1), n) * n;
            // edge columns (periodic in x)
            C.exl = (uint32_t)(x0 == 0 ? n - 1 : x0 - 1);
            C.exr = (uint32_t)(x1 == n ? 0 : x1);
            C.exr1 = (uint32_t)(x1 + 1 >= n ? x1 + 1 - n : x1 + 1);
        }
        // the previous segment's last plane is read by every thread before the
        // prologue refills the ring
        if (!first) __syncthreads();
        if (ahead) run<kAhead>(C, A);
        else if (EDGE && warp == PWARPS + 1) run<kEdge>(C, A);
        else if (2 * warp * RPW < ty) run<kPair>(C, A);
        else run<kIdle>(C, A);
    }

    // the four sums of this thread in the element type (1/beta and 1/2 are powers
    // of two, exact)
    static __device__ __forceinline__ void totals(const Acc& A, bool quartic, T (&v)[kSums])
    {
        v[0] = (lo2(A.g[0][0]) + hi2(A.g[0][0])) + (lo2(A.g[0][1]) + hi2(A.g[0][1]));
        v[1] = (lo2(A.g[1][0]) + hi2(A.g[1][0])) + (lo2(A.g[1][1]) + hi2(A.g[1][1]));
        v[2] = ((lo2(A.vd[0]) + hi2(A.vd[0])) + (lo2(A.vd[1]) + hi2(A.vd[1]))) * site_vsum_factor<T>(quartic);
        v[3] = T(0.5) * ((lo2(A.vi[0]) + hi2(A.vi[0])) + (lo2(A.vi[1]) + hi2(A.vi[1])));
    }
};

template <typename T, int TY, int D, bool SLAB, int SW = 0>
__global__ void __launch_bounds__(XW<T, TY, D, SLAB, SW>::THREADS, XW<T, TY, D, SLAB, SW>::THREADS <= 192 ? 2 : 1)
    step_xw_kernel(Bufs<T> B, Model M, DevScalars* sc, double* partials, SlabRun R)
{
    typedef XW<T, TY, D, SLAB, SW> F;
    constexpr int VW = F::VW;
    __shared__ double red[32 * kSums];
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename F::Ctx C;
    C.S = reinterpret_cast<T*>(smem_raw);
    const int warp = threadIdx.x >> 5;

    // groups of nxt blocks: the x tiles of one y tile, marching the same
    // (y tile, z plane) units
    const int n = M.n;
    C.n = n;
    C.nn = (uint32_t)n * n;
    const int nxt = F::EDGE ? (n / VW + 31) / 32 : 1, nyt = (n + TY - 1) / TY;
    const int ngroups = gridDim.x / nxt;
    const int grp = blockIdx.x / nxt, xt = blockIdx.x - grp * nxt;
    TileWalk walk(nyt, ngroups, grp, SLAB ? R.nz : n);
    // the row's vectors are shared evenly among the x tiles, cut at multiples of
    // 64 bytes where the row is one (tiles that share a 32-byte sector write it in
    // two parts: 0.826 against 0.710 ms at N = 496), the pairs of rows among the y
    // tiles; lanes past the tile's last vector stage and store nothing
    const int Q = n / VW, cut = Q % 4 == 0 ? 4 : Q % 2 == 0 ? 2 : 1;
    const int q0 = xt * (Q / cut) / nxt * cut, qn = (xt + 1) * (Q / cut) / nxt * cut - q0;

    chain_begin();
    if (sc->status != LAT_OK) return;
    const bool par = (sc->step & 1) != 0;
    if constexpr (!SLAB) {
        C.f0 = par ? B.f[1][0] : B.f[0][0];
        C.f1 = par ? B.f[1][1] : B.f[0][1];
        C.p0 = par ? B.p[1][0] : B.p[0][0];
        C.p1 = par ? B.p[1][1] : B.p[0][1];
        C.of0 = par ? B.f[0][0] : B.f[1][0];
        C.of1 = par ? B.f[0][1] : B.f[1][1];
        C.op0 = par ? B.p[0][0] : B.p[1][0];
        C.op1 = par ? B.p[0][1] : B.p[1][1];
    }
    C.K = site_coefs<T>(sc, M.beta);
    C.dtcl2 = mk2(C.K.dtcl, C.K.dtcl);
    C.dtcf2 = mk2(C.K.dtcf, C.K.dtcf);
    typename F::Acc A;
    A.zero();
    C.zb = 0;
    int yt;
    for (bool first = true; walk.run(yt, C.z0, C.nz); first = false) {
        if constexpr (SLAB) {
            // the range holding plane z0 of the end-to-end z space: the run stays
            // within it, on its slab's arrays, from its stored planes
            int r = 0;
            while (r + 1 < R.nranges && C.z0 >= R.rz[r + 1]) r++;
            C.z0 -= R.rz[r];
            C.nz = min(C.nz, R.rn[r] - C.z0);
            C.zb = R.rzb[r];
            void* const* bs = R.buf[R.rslab[r]];
            C.f0 = (const T*)bs[par ? 4 : 0];
            C.f1 = (const T*)bs[par ? 5 : 1];
            C.p0 = (const T*)bs[par ? 6 : 2];
            C.p1 = (const T*)bs[par ? 7 : 3];
            C.of0 = (T*)bs[par ? 0 : 4];
            C.of1 = (T*)bs[par ? 1 : 5];
            C.op0 = (T*)bs[par ? 2 : 6];
            C.op1 = (T*)bs[par ? 3 : 7];
        }
        walk.took(C.nz);
        const int y0 = 2 * (yt * (n / 2) / nyt), ty = 2 * ((yt + 1) * (n / 2) / nyt) - y0;
        if constexpr (F::EDGE) {
            F::march(C, warp, q0, qn, y0, ty, first, A);
        } else {   // a lane's pair of rows may lie past this tile's last
            typename F::Acc S;
            S.zero();
            F::march(C, warp, q0, qn, y0, ty, first, S);
            if (C.act) A.add(S);
        }
    }
    if (F::EDGE && (int)(threadIdx.x & 31) >= qn) A.zero();   // nothing in this lane

    T v[kSums];
    F::totals(A, C.K.quartic, v);
    if constexpr (SLAB) finish_block_sums(M, sc, partials, v, red, R.sums_out);
    else finish_block(M, sc, partials, v, red, true);
}

} // namespace xw

} // namespace lat

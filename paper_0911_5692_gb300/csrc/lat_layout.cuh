// lat_layout.cuh -- how the step kernels that march x tiles one warp wide (variant
// 5, lat_xw.cuh and lat_step27w.cu) share the (y tile, z plane) units of one step
// among their block groups.
#pragma once

namespace lat {

// The (y tile, z plane) units of one step, T y tiles of zn planes, shared among
// the block groups so that neighbouring y tiles are marched at the same planes
// at the same time: a tile's halo rows are its neighbours' owned rows, staged by
// the neighbouring group moments before, and so come from L2. With c = ngroups /
// T >= 1, group j T + t of the first c T takes z chunk j of tile t. Of three
// ways the one whose busiest group has the least to do is taken, a plane
// counting 1 and each run a group starts beyond its first about 2.5:
//   chunks: the first c T groups cut every tile into c equal chunks, the other
//     groups (fewer than T) idle: zn / c planes;
//   chunks and shared: the chunks take M = c T (zn + 2.5) / ngroups planes of
//     every tile, and the other groups share the planes [M, zn) of all tiles in
//     (tile, z) order;
//   shared: all units in (tile, z) order (the only way for fewer groups than
//     tiles).
// The second is the best for the long runs of large lattices (256^3: 55 planes
// against 64; 384^3: 186, and 198 when M was a multiple of c, 0.343 against
// 0.33 ms); with few planes per group its rounding loses (100^3 in 7 tiles on
// 152 groups: 5 planes in equal chunks against 4 and a last shared run of 22,
// 18.9 against 48 us). A group's units are [ubeg, uend) of a space of T tiles x zspan planes
// starting at plane zoff.
struct Layout {
    int ubeg, uend;   // at most T zn units: 32-bit
    int zspan, zoff;
};

__host__ __device__ __forceinline__ Layout tile_layout(int T, int ngroups, int grp, int zn)
{
    Layout L;
    const int c = ngroups / T, U = T * zn;
    // twice the busiest group's cost of each way
    const int per = (U + ngroups - 1) / ngroups, even = 2 * per + (U % ngroups || zn % per ? 5 : 0);
    const int equal = c >= 1 && zn >= c ? 2 * ((zn + c - 1) / c) : 0x7fffffff;
    const int gm = c * T, gt = ngroups - gm;
    int M = 0, mixed = 0x7fffffff;   // planes of every tile that the chunks take
    if (c >= 1 && gt > 0 && zn > c) {
        // c T (zn + 2.5) / ngroups rounded either way, a plane per chunk at least and one left to share
        const int m1 = (int)(((long long)c * T * (2 * zn + 5)) / (2LL * ngroups));
        for (int i = 0; i < 2; i++) {
            const int m = m1 + i < c ? c : (m1 + i > zn - 1 ? zn - 1 : m1 + i);
            const int shared = 2 * ((T * (zn - m) + gt - 1) / gt) + 5 * ((T - 1) / gt), chunk = 2 * ((m + c - 1) / c);
            const int cost = shared > chunk ? shared : chunk;
            if (cost < mixed) {
                mixed = cost;
                M = m;
            }
        }
    }
    if (even < equal && even < mixed) {
        L.ubeg = (int)((long long)grp * U / ngroups);
        L.uend = (int)(((long long)grp + 1) * U / ngroups);
        L.zspan = zn;
        L.zoff = 0;
        return L;
    }
    if (grp < gm) {
        const int j = grp / T, t = grp - j * T;
        const int m = mixed < equal ? M : zn;
        const int zb = (int)((long long)j * m / c), ze = (int)(((long long)j + 1) * m / c);
        L.zspan = ze - zb;
        L.zoff = zb;
        L.ubeg = t * L.zspan;
        L.uend = L.ubeg + L.zspan;
        return L;
    }
    if (mixed >= equal) {   // a group without work
        L.ubeg = L.uend = L.zoff = 0;
        L.zspan = zn;
        return L;
    }
    const int zt = zn - M, g = grp - gm;
    L.ubeg = (int)((long long)g * T * zt / gt);
    L.uend = (int)(((long long)g + 1) * T * zt / gt);
    L.zspan = zt;
    L.zoff = M;
    return L;
}

// The runs of one group over T y tiles, also for more tiles than groups: in each
// of the first T / ngroups turns every group marches one whole tile, so that
// neighbouring tiles are marched side by side there too, and the layout above
// shares the rest of the tiles (1024^3 in 64 tiles on 19 groups: 6.81 -> 6.46 ms
// per step; 576^3, 36 tiles on 30 groups: 1.45 -> 1.13). A run may be taken in
// parts (a z-slab's range ends).
struct TileWalk {
    Layout L;
    int ngroups, grp, zn, waves, wave, zw, u;

    __host__ __device__ __forceinline__ TileWalk(int T, int ngroups_, int grp_, int zn_)
        : ngroups(ngroups_), grp(grp_), zn(zn_), waves(T / ngroups_), wave(0), zw(0)
    {
        const int rest = T - waves * ngroups;
        if (rest > 0) L = tile_layout(rest, ngroups, grp, zn);
        else {
            L.ubeg = L.uend = L.zoff = 0;
            L.zspan = zn;
        }
        u = L.ubeg;
    }
    // the next run: y tile, first plane, planes; false when there is none left
    __host__ __device__ __forceinline__ bool run(int& yt, int& z0, int& nz) const
    {
        if (wave < waves) {
            yt = wave * ngroups + grp;
            z0 = zw;
            nz = zn - zw;
            return true;
        }
        if (u >= L.uend) return false;
        const int t = u / L.zspan, zrel = u - t * L.zspan;
        yt = waves * ngroups + t;
        z0 = L.zoff + zrel;
        nz = L.zspan - zrel < L.uend - u ? L.zspan - zrel : L.uend - u;
        return true;
    }
    // nz planes of it are done
    __host__ __device__ __forceinline__ void took(int nz)
    {
        if (wave < waves) {
            zw += nz;
            if (zw == zn) {
                wave++;
                zw = 0;
            }
        } else {
            u += nz;
        }
    }
};

} // namespace lat

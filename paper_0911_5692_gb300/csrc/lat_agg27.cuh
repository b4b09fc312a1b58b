// lat_agg27.cuh -- the per-plane aggregates of the 27-point Laplacian
// (lat_step27w.cu explains them) at a vector of R neighbouring rows (1 or 2).
#pragma once

#include "lat_async.cuh"
#include "lat_pairs.cuh"
#include "lat_site.cuh"

namespace lat {

// row: the lane's vector of the first row in a plane whose rows are `rs` elements
// apart, with the rows above and below staged beside it. sl, sr: the lanes that
// hold the vectors left and right of it. EDGE: lane 0 and lane `last` take what
// lies beyond the tile from e, e + 1 (left and right of the tile, the row before
// the first), es elements a row. Centres c, q = 3 e + k and r = 14 e + 3 k. Every
// lane calls this.
template <typename T, int R, bool EDGE>
__device__ __forceinline__ void agg27(const T* row, int rs, int lane, int last_lane, int sl, int sr, const T* e, int es,
                                      typename PK<T>::P (&c)[R][PK<T>::NP], typename PK<T>::P (&q)[R][PK<T>::NP],
                                      typename PK<T>::P (&r)[R][PK<T>::NP])
{
    typedef typename PK<T>::P P;
    constexpr int NP = PK<T>::NP, VW = 2 * NP;
    P up[NP], dn[NP], v[R][NP];
    PK<T>::ld(row - rs, up);
#pragma unroll
    for (int i = 0; i < R; i++) PK<T>::ld(row + i * rs, c[i]);
    PK<T>::ld(row + R * rs, dn);
    // the column beside the tile's end that this lane is at, from the row before
    // the first to the one after the last, and its y pairs
    T ec[R + 2], ev[R];
    const bool first = lane == 0, last = lane == last_lane;
    if constexpr (EDGE) {
        const T* ep = e + (first ? 0 : 1);
#pragma unroll
        for (int i = 0; i < R + 2; i++) ec[i] = ld_shared_if(first || last, ep + es * i, T(0));
#pragma unroll
        for (int i = 0; i < R; i++) ev[i] = s_add(s_sub(ec[i], ec[i + 1]), s_sub(ec[i + 2], ec[i + 1]));
    }
    // the y difference inside a pair serves both rows
#pragma unroll
    for (int j = 0; j < NP; j++) {
        if constexpr (R == 2) {
            const P in = sub2(c[1][j], c[0][j]);
            v[0][j] = add2(sub2(up[j], c[0][j]), in);
            v[1][j] = sub2(sub2(dn[j], c[1][j]), in);
        } else {
            v[0][j] = add2(sub2(up[j], c[0][j]), sub2(dn[j], c[0][j]));
        }
    }
    const P two = mk2(T(2), T(2)), three = mk2(T(3), T(3)), fourteen = mk2(T(14), T(14));
#pragma unroll
    for (int i = 0; i < R; i++) {
        T cs[VW + 2], vs[VW + 2];
#pragma unroll
        for (int j = 0; j < NP; j++) {
            un2(c[i][j], cs[1 + 2 * j], cs[2 + 2 * j]);
            un2(v[i][j], vs[1 + 2 * j], vs[2 + 2 * j]);
        }
        cs[0] = __shfl_sync(0xffffffffu, cs[VW], sl);
        cs[VW + 1] = __shfl_sync(0xffffffffu, cs[1], sr);
        vs[0] = __shfl_sync(0xffffffffu, vs[VW], sl);
        vs[VW + 1] = __shfl_sync(0xffffffffu, vs[1], sr);
        if constexpr (EDGE) {
            cs[0] = first ? ec[i + 1] : cs[0];
            vs[0] = first ? ev[i] : vs[0];
            cs[VW + 1] = last ? ec[i + 1] : cs[VW + 1];
            vs[VW + 1] = last ? ev[i] : vs[VW + 1];
        }
        T dd[VW + 1];   // differences of consecutive sites
#pragma unroll
        for (int x = 0; x <= VW; x++) dd[x] = s_sub(cs[x + 1], cs[x]);
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const int a = 1 + 2 * j, b = 2 + 2 * j;   // positions of the pair's sites in cs and vs
            const P h = mk2(s_sub(dd[a], dd[a - 1]), s_sub(dd[b], dd[b - 1]));
            const P t = mk2(s_add(vs[a - 1], vs[a + 1]), s_add(vs[b - 1], vs[b + 1]));
            const P k = fma2(two, h, t);
            const P eh = add2(h, v[i][j]);
            q[i][j] = fma2(three, eh, k);
            r[i][j] = fma2(fourteen, eh, mul2(three, k));
        }
    }
}

} // namespace lat

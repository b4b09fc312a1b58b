// lat_diag.cu -- diagnostics off the timed path: energy density and pressure
// parts (Sec. II.B, eq. rho-pres) and the shell-binned power spectrum that
// Sec. IV names as future work.
#include <cufft.h>

#include <algorithm>
#include <type_traits>

#include "lat_grid.h"
#include "lat_kernels.h"
#include "lat_stencil27.cuh"

namespace lat {

namespace {

__device__ __forceinline__ size_t sidx(int n, int x, int y, int z) { return ((size_t)z * n + y) * n + x; }

// The block's totals of NS per-thread FP64 sums into its row of the partials:
// shuffle tree, then warp totals in order (any fixed block of whole warps).
template <int NS>
__device__ __forceinline__ void energy_partials(double (&acc)[NS], double* partials)
{
    __shared__ double red[32][NS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < NS; k++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
        if (lane == 0) red[warp][k] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x < NS) {
        double s = 0.0;
        for (int w = 0; w < nwarps; w++) s += red[w][threadIdx.x];
        partials[(size_t)blockIdx.x * NS + threadIdx.x] = s;
    }
}

// Per-block FP64 partials (one thread per (x, y) column, z marched in order; the
// 27-point stencil): [kin0, kin1, grad0, grad1, pot, sum f0, sum f1], where the
// momenta at the field time are f' + (dt/2) F(f) (the average of the stored f' and
// the next kick's), kin_i = (f'_i - r h f_i)^2 / 2 with h = a'/a at the field time,
// grad_i = the stencil's gradient sum before its factor M.lap_scale (7 points:
// sum_d (forward difference)^2; 27 points: the 13 owned weighted bonds),
// pot = V_pr.
template <typename T>
__global__ void __launch_bounds__(256) energies_kernel(Bufs<T> B, Model M, const DevScalars* sc, double* partials)
{
    const int n = M.n;
    const int par = (int)(sc->step & 1);
    const T* f0 = B.f[par][0];
    const T* f1 = B.f[par][1];
    const T* p0 = B.p[par][0];
    const T* p1 = B.p[par][1];
    const double cL = sc->cL, cF = sc->cF, cdom = sc->cdom, kap = sc->kappa, dt = M.dt;
    const double h = M.expansion ? sc->ad_half / sc->a : 0.0;
    // split storage: phi = P + stored, its momentum = Pi + stored (P = Pi = 0 otherwise)
    const double bgf = sc->bgf, bgp = sc->bgp;
    double acc[kEnergySums] = {0, 0, 0, 0, 0, 0, 0};
    const long long cols = (long long)n * n;
    for (long long col = (long long)blockIdx.x * blockDim.x + threadIdx.x; col < cols;
         col += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(col % n), y = (int)(col / n);
        const int xm = x == 0 ? n - 1 : x - 1, xp = x == n - 1 ? 0 : x + 1;
        const int ym = y == 0 ? n - 1 : y - 1, yp = y == n - 1 ? 0 : y + 1;
        for (int z = 0; z < n; z++) {
            const size_t c = sidx(n, x, y, z);
            const double s0 = (double)f0[c], a1 = (double)f1[c];
            const double a0 = s0 + bgf;
            double lap0, lap1, gs0, gs1;
            lap0 = lap27_sum(f0, n, x, y, z) * M.lap_scale;
            lap1 = lap27_sum(f1, n, x, y, z) * M.lap_scale;
            gs0 = bonds27_sum(f0, n, x, y, z);
            gs1 = bonds27_sum(f1, n, x, y, z);
            const double a0b = M.beta == 4 ? a0 * a0 * a0 : a0;
            const double F0 = cL * lap0 + cF * a0 - (cdom * a0b + kap * a0 * a1 * a1);
            const double F1 = cL * lap1 + cF * a1 - kap * a0 * a0 * a1;
            const double q0 = ((double)p0[c] + bgp) + 0.5 * dt * F0 - M.r * h * a0;
            const double q1 = (double)p1[c] + 0.5 * dt * F1 - M.r * h * a1;
            acc[0] += 0.5 * q0 * q0;
            acc[1] += 0.5 * q1 * q1;
            acc[2] += gs0;
            acc[3] += gs1;
            const double sq = a0 * a0;
            acc[4] += cdom * (M.beta == 4 ? 0.25 * sq * sq : 0.5 * sq) + 0.5 * kap * sq * a1 * a1;
            acc[5] += a0;
            acc[6] += a1;
        }
    }
    energy_partials(acc, partials);
}

// The same sums for 7 points. Bound by the FP64 pipes (64 cycles per warp
// instruction, conversions from FP32 included), so every difference and
// conversion is formed once where its neighbours are at hand: a thread marches
// one 16-byte vector of x sites of two neighbouring rows along z, carrying the
// centres and their differences to the plane below; a forward difference serves
// its own site's gradient sum and Laplacian and the next site's Laplacian; and the
// momenta at the field time take the coefficients as three products formed once.
// About 50 FP64 instructions per site where one column per thread and one
// difference at a time took about 95: 256^3 FP32 3.1 -> 1.55 ms.
template <typename T>
__global__ void __launch_bounds__(256, 1) energies7_kernel(Bufs<T> B, Model M, const DevScalars* sc, double* partials,
                                                           int nzc)
{
    constexpr int V = 16 / sizeof(T);
    using Raw = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    const int n = M.n, q = n / V;
    const int par = (int)(sc->step & 1);
    const T* __restrict__ f[2] = {par ? B.f[1][0] : B.f[0][0], par ? B.f[1][1] : B.f[0][1]};
    const T* __restrict__ p[2] = {par ? B.p[1][0] : B.p[0][0], par ? B.p[1][1] : B.p[0][1]};
    const double hdt = 0.5 * M.dt, h = M.expansion ? sc->ad_half / sc->a : 0.0;
    const double bgf = sc->bgf, bgp = sc->bgp;   // split storage: phi = P + stored, its momentum = Pi + stored
    const bool quartic = M.beta == 4;
    // q_0 = p_0 + k1 Lap + (k2 - [c3 f0^2 +] c4 f1^2) f0, q_1 = p_1 + k1 Lap + (k2 - c4 f0^2) f1
    const double k1 = hdt * sc->cL * M.inv_dx2, k2 = hdt * sc->cF - M.r * h;
    const double c3 = quartic ? hdt * sc->cdom : 0.0, c4 = hdt * sc->kappa, k20 = quartic ? k2 : k2 - hdt * sc->cdom;
    const double v0 = quartic ? 0.25 * sc->cdom : 0.0, v1 = quartic ? 0.0 : 0.5 * sc->cdom, v2 = 0.5 * sc->kappa;
    double acc[kEnergySums] = {0, 0, 0, 0, 0, 0, 0};
    auto vec = [&](const T* a, int x, int y, int z, double (&o)[V]) {
        const Raw r = __ldg(reinterpret_cast<const Raw*>(a + sidx(n, x, y, z)));
        T v[V];
        *reinterpret_cast<Raw*>(v) = r;
#pragma unroll
        for (int j = 0; j < V; j++) o[j] = (double)v[j];
    };
    const long long cols = (long long)q * (n / 2), items = cols * nzc;
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
         it += (long long)gridDim.x * blockDim.x) {
        const long long col = it % cols;
        const int zc = (int)(it / cols);
        const int x = V * (int)(col % q), y = 2 * (int)(col / q);
        const int xl = x == 0 ? n - 1 : x - 1, xr = x + V == n ? 0 : x + V;
        const int ym = y == 0 ? n - 1 : y - 1, yp = y + 2 == n ? 0 : y + 2;
        const int zb = (int)((long long)zc * n / nzc), ze = (int)((long long)(zc + 1) * n / nzc);
        double c[2][2][V], dzp[2][2][V];   // [field][row]
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int r = 0; r < 2; r++) {
                double m[V];
                vec(f[i], x, y + r, zb == 0 ? n - 1 : zb - 1, m);
                vec(f[i], x, y + r, zb, c[i][r]);
#pragma unroll
                for (int j = 0; j < V; j++) dzp[i][r][j] = c[i][r][j] - m[j];
            }
        for (int z = zb; z < ze; z++) {
            const int zp = z == n - 1 ? 0 : z + 1;
            double u[2][2][V];   // p_i + k1 Lap f_i
            double w[2][2][V];   // this plane's centres
#pragma unroll
            for (int i = 0; i < 2; i++) {
                double up[V], dn[V];
                vec(f[i], x, ym, z, up);
                vec(f[i], x, yp, z, dn);
                double g = acc[2 + i];
                double in[V];
#pragma unroll
                for (int j = 0; j < V; j++) in[j] = c[i][1][j] - c[i][0][j];
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    double nx[V], pv[V];
                    vec(f[i], x, y + r, zp, nx);
                    vec(p[i], x, y + r, z, pv);
                    const double left = (double)__ldg(f[i] + sidx(n, xl, y + r, z));
                    const double right = (double)__ldg(f[i] + sidx(n, xr, y + r, z));
                    double dl = c[i][r][0] - left;
#pragma unroll
                    for (int j = 0; j < V; j++) {
                        const double cc = c[i][r][j];
                        const double dx = (j + 1 < V ? c[i][r][j + 1 < V ? j + 1 : j] : right) - cc;
                        const double dz = nx[j] - cc;
                        const double dy = r == 0 ? in[j] : dn[j] - cc;       // forward
                        const double db = r == 0 ? cc - up[j] : in[j];       // backward
                        const double lap = ((dx - dl) + (dy - db)) + (dz - dzp[i][r][j]);
                        g = fma(dx, dx, fma(dy, dy, fma(dz, dz, g)));
                        u[i][r][j] = fma(k1, lap, pv[j]);
                        w[i][r][j] = cc;
                        dl = dx;
                        dzp[i][r][j] = dz;
                    }
                    // the next plane's centres (the in-pair difference is formed above)
#pragma unroll
                    for (int j = 0; j < V; j++) c[i][r][j] = nx[j];
                }
                acc[2 + i] = g;
            }
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
                for (int j = 0; j < V; j++) {
                    const double a0 = w[0][r][j] + bgf, a1 = w[1][r][j];
                    const double s0 = a0 * a0, s1 = a1 * a1, k = c4 * s1;
                    const double q0 = fma(k20 - fma(c3, s0, k), a0, u[0][r][j] + bgp);
                    const double q1 = fma(fma(-c4, s0, k2), a1, u[1][r][j]);
                    acc[0] = fma(q0, q0, acc[0]);
                    acc[1] = fma(q1, q1, acc[1]);
                    acc[4] = fma(s0, fma(v0, s0, fma(v2, s1, v1)), acc[4]);
                    acc[5] += a0;
                    acc[6] += a1;
                }
        }
    }
    acc[0] *= 0.5;
    acc[1] *= 0.5;
    energy_partials(acc, partials);
}

// Sums of (f_0 - mean_0)^2 and (f_1 - mean_1)^2 (per-block partials), means[0..1]
// those of the whole fields.
template <typename T>
__global__ void __launch_bounds__(256) variances_kernel(Bufs<T> B, Model M, const DevScalars* sc, double* partials,
                                                        const double* means)
{
    constexpr int V = 16 / sizeof(T);
    using Raw = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    const int par = (int)(sc->step & 1);
    const Raw* f0 = reinterpret_cast<const Raw*>(par ? B.f[1][0] : B.f[0][0]);
    const Raw* f1 = reinterpret_cast<const Raw*>(par ? B.f[1][1] : B.f[0][1]);
    const double m0 = means[0] - sc->bgf, m1 = means[1];
    double acc[2] = {0.0, 0.0};
    const long long count = (long long)M.n * M.n * M.n / V;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
        T a[V], b[V];
        *reinterpret_cast<Raw*>(a) = __ldg(f0 + i);
        *reinterpret_cast<Raw*>(b) = __ldg(f1 + i);
#pragma unroll
        for (int j = 0; j < V; j++) {
            const double d0 = (double)a[j] - m0, d1 = (double)b[j] - m1;
            acc[0] = fma(d0, d0, acc[0]);
            acc[1] = fma(d1, d1, acc[1]);
        }
    }
    energy_partials(acc, partials);
}

template <typename T>
__global__ void to_double_kernel(const T* src, double* dst, size_t count, double offset)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        const double v = (double)src[i];
        dst[i] = offset == 0.0 ? v : v + offset;   // (an FP64 addition costs more than the memory access)
    }
}

// The shell of an integer wave vector of square n2: floor(|n| + 1/2), the b with
// (2b - 1)^2 <= 4 n2 < (2b + 1)^2 (0 for n2 = 0), in integers from an FP32 root,
// which is at most one off.
__device__ __forceinline__ int shell_of(int n2)
{
    int b = (int)(sqrtf((float)n2) + 0.5f);
    if (b > 0 && 4 * n2 < (2 * b - 1) * (2 * b - 1)) b--;
    if (4 * n2 >= (2 * b + 1) * (2 * b + 1)) b++;
    return b;
}

// Shell sums of |F|^2 over the R2C half spectrum ([kz][ky][kx], kx in [0, N/2]).
// Modes with 0 < kx < N/2 stand for themselves and their conjugate partner
// (weight 2). A thread takes eight neighbouring kx of a row (one 128-byte line);
// their shells do not fall along kx, so it adds up a run of equal shells in a
// register and adds each run once to the block's shared-memory bins. FP64 bound
// the earlier form (a root, its conversions and three sums per mode, 0.70 ms at
// 256^3); this one has three FP64 operations per mode: 0.12 ms, and 0.07 for the geometry
// of the shells, from an octant of the modes.
constexpr int kBinRun = 8;
__global__ void __launch_bounds__(256) spectrum_bins_kernel(const cufftDoubleComplex* spec, int n, int nbins, double* partials)
{
    extern __shared__ double sb[];
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) sb[i] = 0.0;
    __syncthreads();
    const int nh = n / 2 + 1, runs = (nh + kBinRun - 1) / kBinRun;
    const long long items = (long long)n * n * runs;
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
         it += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(it / runs), k0 = (int)(it - (long long)row * runs) * kBinRun;
        const int ky = row % n, kz = row / n;
        const int ny = ky < n / 2 ? ky : ky - n, nz = kz < n / 2 ? kz : kz - n;
        const int nyz = ny * ny + nz * nz;
        const double2* p = reinterpret_cast<const double2*>(spec) + (size_t)row * nh;
        int cur = -1;
        double acc = 0.0;
        for (int kx = k0; kx < min(k0 + kBinRun, nh); kx++) {
            const int b = shell_of(kx * kx + nyz);   // kx = N/2 stands for -N/2: the same square
            const double2 f = p[kx];
            const double pw = f.x * f.x + f.y * f.y;
            if (b != cur) {
                if (cur >= 0 && cur < nbins) atomicAdd(&sb[cur], acc);
                cur = b;
                acc = 0.0;
            }
            // twice for a mode with a partner: the same as a weight of 2, exactly
            acc += kx == 0 || 2 * kx == n ? pw : pw + pw;
        }
        if (cur >= 0 && cur < nbins) atomicAdd(&sb[cur], acc);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) partials[(size_t)blockIdx.x * nbins + i] = sb[i];
}

// Number of modes of each shell and the sum of their |n|, over the wave vectors
// with no negative component (each standing for 2 per component that is neither
// 0 nor N/2): partials [|n| sums, counts] of each block.
__global__ void __launch_bounds__(256) shell_modes_kernel(int n, int nbins, double* partials)
{
    extern __shared__ double sb[];
    for (int i = threadIdx.x; i < 2 * nbins; i += blockDim.x) sb[i] = 0.0;
    __syncthreads();
    const int nh = n / 2 + 1, runs = (nh + kBinRun - 1) / kBinRun;
    const int items = nh * nh * runs;
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < items; it += gridDim.x * blockDim.x) {
        const int row = it / runs, k0 = (it - row * runs) * kBinRun;
        const int ky = row % nh, kz = row / nh;
        const int wyz = (ky == 0 || 2 * ky == n ? 1 : 2) * (kz == 0 || 2 * kz == n ? 1 : 2);
        int cur = -1, cnt = 0;
        double acc = 0.0;
        auto flush = [&]() {
            if (cur < 0 || cur >= nbins) return;
            atomicAdd(&sb[cur], acc);
            atomicAdd(&sb[nbins + cur], (double)cnt);
        };
        for (int kx = k0; kx < min(k0 + kBinRun, nh); kx++) {
            const int n2 = kx * kx + ky * ky + kz * kz, b = shell_of(n2);
            if (b >= nbins && cur >= nbins) continue;
            const int w = wyz * (kx == 0 || 2 * kx == n ? 1 : 2);
            if (b != cur) {
                flush();
                cur = b;
                cnt = 0;
                acc = 0.0;
            }
            cnt += w;
            acc += (double)w * sqrt((double)n2);
        }
        flush();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * nbins; i += blockDim.x) partials[(size_t)blockIdx.x * 2 * nbins + i] = sb[i];
}

// out[i] = scale of its row of `rows` partial sums of `width` values each, added in
// row order by one warp per value.
__global__ void fold_rows_kernel(const double* partials, int rows, int width, double* out, double scale, int scaled)
{
    const int i = blockIdx.x * blockDim.y + threadIdx.y;
    if (i >= width) return;
    double s = 0.0;
    for (int r = threadIdx.x; r < rows; r += 32) s += partials[(size_t)r * width + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[i] = i < scaled ? s * scale : s;
}

// Integer-weight sums over the site's stencil neighbours of the differences
// (30 dx^2 L f for 27 points, dx^2 L f for 7) and of their squares.
template <typename T>
__device__ __forceinline__ void neighbour_sums(const T* __restrict__ f, int n, int x, int y, int z, bool s27, T& lap,
                                               T& sq)
{
    const T c = __ldg(f + sidx(n, x, y, z));
    T l = T(0), g = T(0);
    if (s27) {
#pragma unroll
        for (int dz = -1; dz <= 1; dz++) {
            const int zz = wrap27(z + dz, n);
#pragma unroll
            for (int dy = -1; dy <= 1; dy++) {
                const int yy = wrap27(y + dy, n);
#pragma unroll
                for (int dx = -1; dx <= 1; dx++) {
                    const int cls = (dx != 0) + (dy != 0) + (dz != 0);
                    if (cls == 0) continue;
                    const T d = __ldg(f + sidx(n, wrap27(x + dx, n), yy, zz)) - c;
                    const T w = T(w27(cls));
                    l += w * d;
                    g += w * d * d;
                }
            }
        }
    } else {
        const int xm = x == 0 ? n - 1 : x - 1, xp = x == n - 1 ? 0 : x + 1;
        const int ym = y == 0 ? n - 1 : y - 1, yp = y == n - 1 ? 0 : y + 1;
        const int zm = z == 0 ? n - 1 : z - 1, zp = z == n - 1 ? 0 : z + 1;
        const T d[6] = {__ldg(f + sidx(n, xm, y, z)) - c, __ldg(f + sidx(n, xp, y, z)) - c,
                        __ldg(f + sidx(n, x, ym, z)) - c, __ldg(f + sidx(n, x, yp, z)) - c,
                        __ldg(f + sidx(n, x, y, zm)) - c, __ldg(f + sidx(n, x, y, zp)) - c};
#pragma unroll
        for (int k = 0; k < 6; k++) {
            l += d[k];
            g += d[k] * d[k];
        }
    }
    lap = l;
    sq = g;
}

// Energy density and pressure at every site (eq. rho-pres per site), in the
// units of lat_energies: rho = conv (sum_i [kin_i + grad_i] + V_pr),
// p = conv (sum_i [kin_i - grad_i / 3] - V_pr), kin_i = (f'_i + (dt/2) F_i - r h f_i)^2 / 2
// (the momentum at the field time), grad_i = a^(-2s-2) / 2 times half the
// weighted squared differences to all the site's stencil neighbours (each
// neighbour pair shared evenly by its two sites). One thread per (x, y) column;
// arithmetic in the lattice precision on exact neighbour differences, the
// coefficients in FP64 rounded once.
template <typename T>
struct FieldCoef {
    T cL, cF, cdom, kap, hdt, rh, gq, cv;
    T bgf, bgp;   // split storage: phi = bgf + stored, its momentum = bgp + stored
    bool quartic;
};

template <typename T>
__device__ inline FieldCoef<T> field_coefs(const Model& M, const DevScalars* sc)
{
    const double a = sc->a;
    const double h = M.expansion ? sc->ad_half / a : 0.0;
    FieldCoef<T> k;
    k.cL = (T)(sc->cL * M.lap_scale);
    k.cF = (T)sc->cF;
    k.cdom = (T)sc->cdom;
    k.kap = (T)sc->kappa;
    k.hdt = (T)(0.5 * M.dt);
    k.rh = (T)(M.r * h);
    k.gq = (T)(0.25 * pow(a, -2.0 * M.s - 2.0) * M.lap_scale);   // grad_i = gq * sum w d^2
    k.cv = (T)(M.B * M.B / (M.A * M.A) * pow(a, 2.0 * M.s - 2.0 * M.r));
    k.bgf = (T)sc->bgf;
    k.bgp = (T)sc->bgp;
    k.quartic = M.beta == 4;
    return k;
}

// rho and p at one site from its fields a0, a1, momenta m0, m1 as stored and
// the neighbour sums (l: of the differences, g: of their squares) of each field.
template <typename T>
__device__ __forceinline__ void site_energy(const FieldCoef<T>& K, T a0, T a1, T m0, T m1, T l0, T g0, T l1, T g1,
                                            T& rho, T& pres)
{
    a0 += K.bgf;   // whole phi and its momentum (unchanged when phi is stored whole)
    m0 += K.bgp;
    const T a0b = K.quartic ? a0 * a0 * a0 : a0;
    const T F0 = K.cL * l0 + K.cF * a0 - (K.cdom * a0b + K.kap * a0 * a1 * a1);
    const T F1 = K.cL * l1 + K.cF * a1 - K.kap * a0 * a0 * a1;
    const T q0 = m0 + K.hdt * F0 - K.rh * a0;
    const T q1 = m1 + K.hdt * F1 - K.rh * a1;
    const T kin = T(0.5) * (q0 * q0 + q1 * q1);
    const T grad = K.gq * (g0 + g1);
    const T sq = a0 * a0;
    const T V = K.cdom * (K.quartic ? T(0.25) * sq * sq : T(0.5) * sq) + T(0.5) * K.kap * sq * a1 * a1;
    rho = K.cv * (kin + grad + V);
    pres = K.cv * (kin - grad / T(3) - V);
}

template <typename T>
__global__ void __launch_bounds__(256) energy_field_kernel(Bufs<T> B, Model M, const DevScalars* sc, T* rho, T* pres)
{
    const int n = M.n;
    const int par = (int)(sc->step & 1);
    const T* f0 = B.f[par][0];
    const T* f1 = B.f[par][1];
    const T* p0 = B.p[par][0];
    const T* p1 = B.p[par][1];
    const FieldCoef<T> K = field_coefs<T>(M, sc);
    const bool s27 = M.stencil == 27;
    const long long cols = (long long)n * n;
    for (long long col = (long long)blockIdx.x * blockDim.x + threadIdx.x; col < cols;
         col += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(col % n), y = (int)(col / n);
        for (int z = 0; z < n; z++) {
            const size_t c = sidx(n, x, y, z);
            const T a0 = __ldg(f0 + c), a1 = __ldg(f1 + c);
            T l0, g0, l1, g1;
            neighbour_sums(f0, n, x, y, z, s27, l0, g0);
            neighbour_sums(f1, n, x, y, z, s27, l1, g1);
            site_energy(K, a0, a1, __ldg(p0 + c), __ldg(p1 + c), l0, g0, l1, g1, rho[c], pres[c]);
        }
    }
}

// The 7-point energy field with one 16-byte vector of x sites per thread,
// marching whole z runs, the loads of plane z + 1 issued before plane z is
// computed; the same per-site terms as energy_field_kernel, the six neighbour
// differences taken in the same order (-x, +x, -y, +y, -z, +z).
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
    energy_field7_kernel(Bufs<T> B, Model M, const DevScalars* sc, T* rho, T* pres, int nzc)
{
    constexpr int V = 16 / sizeof(T);
    using Raw = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    struct Vec {
        T v[V];
    };
    const int n = M.n, q = n / V;
    const int par = (int)(sc->step & 1);
    const T* __restrict__ f[2] = {B.f[par][0], B.f[par][1]};
    const T* __restrict__ p[2] = {B.p[par][0], B.p[par][1]};
    const FieldCoef<T> K = field_coefs<T>(M, sc);
    auto vec = [&](const T* a, int x, int y, int z) {
        const Raw r = __ldg(reinterpret_cast<const Raw*>(a + sidx(n, x, y, z)));
        Vec o;
        *reinterpret_cast<Raw*>(o.v) = r;
        return o;
    };
    const long long vcols = (long long)q * n, items = vcols * nzc;
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
         it += (long long)gridDim.x * blockDim.x) {
        const long long vc = it % vcols;
        const int zc = (int)(it / vcols);
        const int x = V * (int)(vc % q), y = (int)(vc / q);
        const int xl = x == 0 ? n - 1 : x - 1, xr = x + V == n ? 0 : x + V;
        const int ym = y == 0 ? n - 1 : y - 1, yp = y == n - 1 ? 0 : y + 1;
        const int zb = (int)((long long)zc * n / nzc), ze = (int)((long long)(zc + 1) * n / nzc);
        struct Plane {
            Vec cp, a, b, pv;
            T l, r;
        };
        auto load_plane = [&](int i, int z, Plane& o) {
            const int zp = z == n - 1 ? 0 : z + 1;
            o.cp = vec(f[i], x, y, zp);
            o.a = vec(f[i], x, ym, z);
            o.b = vec(f[i], x, yp, z);
            o.pv = vec(p[i], x, y, z);
            o.l = __ldg(f[i] + sidx(n, xl, y, z));
            o.r = __ldg(f[i] + sidx(n, xr, y, z));
        };
        Vec cm[2], c[2];
        Plane nx[2];
#pragma unroll
        for (int i = 0; i < 2; i++) {
            cm[i] = vec(f[i], x, y, zb == 0 ? n - 1 : zb - 1);
            c[i] = vec(f[i], x, y, zb);
            load_plane(i, zb, nx[i]);
        }
        for (int z = zb; z < ze; z++) {
            const Plane cu[2] = {nx[0], nx[1]};
            if (z + 1 < ze) {
#pragma unroll
                for (int i = 0; i < 2; i++) load_plane(i, z + 1, nx[i]);
            }
            Vec lsum[2], gsum[2];
#pragma unroll
            for (int i = 0; i < 2; i++) {
#pragma unroll
                for (int j = 0; j < V; j++) {
                    const T cc = c[i].v[j];
                    const T left = j == 0 ? cu[i].l : c[i].v[j - 1], right = j == V - 1 ? cu[i].r : c[i].v[j + 1];
                    const T d[6] = {left - cc, right - cc, cu[i].a.v[j] - cc, cu[i].b.v[j] - cc, cm[i].v[j] - cc,
                                    cu[i].cp.v[j] - cc};
                    T l = T(0), g = T(0);
#pragma unroll
                    for (int k = 0; k < 6; k++) {
                        l += d[k];
                        g += d[k] * d[k];
                    }
                    lsum[i].v[j] = l;
                    gsum[i].v[j] = g;
                }
            }
            Vec ro, pr;
#pragma unroll
            for (int j = 0; j < V; j++)
                site_energy(K, c[0].v[j], c[1].v[j], cu[0].pv.v[j], cu[1].pv.v[j], lsum[0].v[j], gsum[0].v[j],
                            lsum[1].v[j], gsum[1].v[j], ro.v[j], pr.v[j]);
            const size_t o = sidx(n, x, y, z);
            *reinterpret_cast<Raw*>(rho + o) = *reinterpret_cast<const Raw*>(ro.v);
            *reinterpret_cast<Raw*>(pres + o) = *reinterpret_cast<const Raw*>(pr.v);
#pragma unroll
            for (int i = 0; i < 2; i++) {
                cm[i] = c[i];
                c[i] = cu[i].cp;
            }
        }
    }
}

} // namespace

template <typename T>
cudaError_t launch_energy_field(const Bufs<T>& b, const Model& M, const DevScalars* sc, T* rho, T* pres,
                                cudaStream_t st)
{
    const int n = M.n;
    constexpr int V = 16 / sizeof(T);
    if (M.stencil != 27 && ((uintptr_t)rho % 16) == 0 && ((uintptr_t)pres % 16) == 0) {
        // one resident wave; runs of whole planes per thread, two planes loaded
        // before a run's first
        static int occ = 0;
        const int wave = resident_wave((const void*)energy_field7_kernel<T>, 256, &occ);
        if (wave == 0) return cudaErrorInvalidDevice;
        const long long vcols = (long long)(n / V) * n;
        const int nzc = balanced_zruns(vcols, n, (long long)wave * 256, 2.0);
        const int blocks = (int)std::min<long long>(wave, (vcols * nzc + 255) / 256);
        energy_field7_kernel<T><<<blocks, 256, 0, st>>>(b, M, sc, rho, pres, nzc);
        return cudaGetLastError();
    }
    energy_field_kernel<T><<<energies_grid_blocks(n), 256, 0, st>>>(b, M, sc, rho, pres);
    return cudaGetLastError();
}
template cudaError_t launch_energy_field<float>(const Bufs<float>&, const Model&, const DevScalars*, float*, float*,
                                                cudaStream_t);
template cudaError_t launch_energy_field<double>(const Bufs<double>&, const Model&, const DevScalars*, double*,
                                                 double*, cudaStream_t);

int energies_grid_blocks(int n)
{
    const long long cols = (long long)n * n;
    long long blocks = (cols + 255) / 256;
    return (int)(blocks < 1024 ? blocks : 1024);
}

template <typename T>
cudaError_t launch_energies(const Bufs<T>& b, const Model& M, const DevScalars* sc, double* partials, double* out,
                            cudaStream_t st)
{
    const int n = M.n;
    constexpr int V = 16 / sizeof(T);
    int blocks = energies_grid_blocks(n);
    if (M.stencil == 27) {
        energies_kernel<T><<<blocks, 256, 0, st>>>(b, M, sc, partials);
    } else {
        static int occ = 0;
        const int wave = resident_wave((const void*)energies7_kernel<T>, 256, &occ);
        if (wave == 0) return cudaErrorInvalidDevice;
        const long long cols = (long long)(n / V) * (n / 2);
        // a plane of a thread is some 14 us of FP64, so small lattices take runs of one
        const int nzc = balanced_zruns(cols, n, (long long)wave * 256, 0.3, 1);
        blocks = (int)std::min<long long>(wave, (cols * nzc + 255) / 256);
        energies7_kernel<T><<<blocks, 256, 0, st>>>(b, M, sc, partials, nzc);
    }
    const dim3 fold(32, 8);
    fold_rows_kernel<<<1, fold, 0, st>>>(partials, blocks, kEnergySums, out, M.inv_sites, kEnergySums);
    const int vb = std::min(energies_grid_blocks(n), 608);
    variances_kernel<T><<<vb, 256, 0, st>>>(b, M, sc, partials, out + 5);
    fold_rows_kernel<<<1, fold, 0, st>>>(partials, vb, 2, out + kEnergySums, M.inv_sites, 2);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_to_double(const T* src, double* dst, size_t count, double offset, cudaStream_t st)
{
    size_t blocks = (count + 255) / 256;
    to_double_kernel<T><<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(src, dst, count, offset);
    return cudaGetLastError();
}

namespace {
constexpr int kSpectrumBlocks = 608, kShellBlocks = 304;
int spectrum_blocks(int n, int most)
{
    const long long blocks = ((long long)n * n * ((n / 2 + kBinRun) / kBinRun) + 255) / 256;
    return (int)(blocks < most ? blocks : most);
}
} // namespace

size_t spectrum_scratch(int n, int nbins)
{
    (void)n;
    return (size_t)nbins * (kSpectrumBlocks + 2 * kShellBlocks);
}

cudaError_t launch_spectrum_bins(const void* spec, int n, double L, int nbins, double* scratch, double* out, cudaStream_t st)
{
    const size_t sp = (size_t)nbins * sizeof(double), sm = 2 * sp;
    if (sm > 48 * 1024) {
        cudaError_t e = allow_dynamic_smem((const void*)shell_modes_kernel, sm);
        if (e != cudaSuccess) return e;
    }
    const int nb = spectrum_blocks(n, kSpectrumBlocks), ns = spectrum_blocks(n / 2 + 1, kShellBlocks);
    double* modes = scratch + (size_t)nbins * kSpectrumBlocks;
    const dim3 fold(32, 8);
    spectrum_bins_kernel<<<nb, 256, sp, st>>>((const cufftDoubleComplex*)spec, n, nbins, scratch);
    fold_rows_kernel<<<(nbins + 7) / 8, fold, 0, st>>>(scratch, nb, nbins, out, 1.0 / ((double)n * n * n), nbins);
    shell_modes_kernel<<<ns, 256, sm, st>>>(n, nbins, modes);
    fold_rows_kernel<<<(2 * nbins + 7) / 8, fold, 0, st>>>(modes, ns, 2 * nbins, out + nbins,
                                                           2.0 * 3.14159265358979323846 / L, nbins);
    return cudaGetLastError();
}

template cudaError_t launch_energies<float>(const Bufs<float>&, const Model&, const DevScalars*, double*, double*,
                                            cudaStream_t);
template cudaError_t launch_energies<double>(const Bufs<double>&, const Model&, const DevScalars*, double*, double*,
                                             cudaStream_t);
template cudaError_t launch_to_double<float>(const float*, double*, size_t, double, cudaStream_t);
template cudaError_t launch_to_double<double>(const double*, double*, size_t, double, cudaStream_t);

} // namespace lat

// lat_init.cu -- DEFROST-style initial conditions on the device (Sec. II.B,
// last paragraph): homogeneous values plus Gaussian vacuum fluctuations.
//
// White noise: one standard normal per (seed, field, quantity, site) from
// Philox-4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) with counter
// (site, field, quantity, 0) and key (seed lo, seed hi); words 0 and 1 are mapped
// to (0,1) as (u + 1/2) 2^-32 and turned into a normal by Box-Muller's cosine
// branch. The noise is filtered in Fourier space by the vacuum amplitude
// (cuFFT does the transforms), transformed back and added to the homogeneous
// program-unit values, after which the fields are advanced by dt/2.
#include <cufft.h>

#include <cmath>

#include "lat_kernels.h"

namespace lat {

namespace {

__device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) { return __umulhi(a, b); }

// Philox-4x32-10: ten rounds, each two 32x32->64 multiplies (multipliers
// 0xD2511F53, 0xCD9E8D57) and an xor with the key; the key advances by the
// Weyl constants 0x9E3779B9, 0xBB67AE85 between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int round = 0; round < 10; round++) {
        if (round > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = mulhi32(0xD2511F53u, c[0]);
        const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = mulhi32(0xCD9E8D57u, c[2]);
        const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    }
}

// Box-Muller in FP64 from two 32-bit words: sqrt(-2 log u1) cos(2 pi u2) with
// u = (c + 1/2) 2^-32. The pass is bound by the FP64 pipe (64 cycles per warp
// instruction), so log and cos are table-driven with short polynomials, on
// arguments that are exact by construction; 256^3: 1.93 -> 1.03 ms per array.
//
// log (P. T. P. Tang, Table-driven implementation of the logarithm function in
// IEEE floating-point arithmetic, ACM TOMS 16, 1990): u1 = m 2^-33 with the odd
// integer m = 2 c + 1 = 2^e f, f in [1, 2). With g_i = 1 + (i + 1/2)/512 the
// middle of f's interval, r_i its rounded reciprocal and l_i = log(1/r_i),
// log f = l_i + log1p(t), t = fma(f, r_i, -1) (exact to rounding, |t| < 2^-9),
// log1p by its series to t^6 (the next term is below 2^-70). The upper half of
// the intervals counts f as 2 (f/2), l_i = log(1/(2 r_i)): for u1 near 1, where
// log u1 is small, the integer part is then zero and nothing cancels; the last
// one takes r = 1/2 and l = 0, so that t = f/2 - 1 alone carries the digits.
// l and the multiples of log 2 are kept as a multiple of 2^-40 and the rest, so
// that the large parts add exactly and the sum is rounded once.
//
// cos: 2 pi u2 = 2 pi (2 c + 1) 2^-33: the top 9 bits choose one of 512 points
// a_j = 2 pi (j + 1/2)/512, the other 24 bits the offset d from it, an integer
// multiple of 2 pi 2^-33 with |d| <= 2 pi/1024, and cos(a + d) = cos a cos d -
// sin a sin d with the series of cos d - 1 to d^6 and of sin d to d^5 (the next
// terms are below 2^-74 and 2^-63 of one), cos a_j with its rounding error.
//
// Error against 128-bit arithmetic over 400000 draws: rms 8.08e-17 (CUDA's log and
// cospi in the same form: 8.38e-17).
constexpr int kNoiseBits = 9, kNoiseTable = 1 << kNoiseBits;
struct NoiseTables {
    double2 lg[kNoiseTable];   // r_i, leading part of l_i
    double2 cs[kNoiseTable];   // cos a_j, sin a_j
    double lo[kNoiseTable];    // the rest of l_i
    double clo[kNoiseTable];   // the rest of cos a_j
    double2 l2[34];            // (e - 33) log 2, leading part and the rest
};

// Pairs of doubles hi + lo for the cosines of the table (two-sum and two-product,
// Dekker and Knuth).
struct DD {
    double hi, lo;
};
DD dd_norm(double a, double b)
{
    const double s = a + b, t = s - a;
    return DD{s, (a - (s - t)) + (b - t)};
}
DD dd_add(DD a, DD b)
{
    const DD s = dd_norm(a.hi, b.hi);
    return dd_norm(s.hi, s.lo + (a.lo + b.lo));
}
DD dd_mul(DD a, DD b)
{
    const double p = a.hi * b.hi;
    return dd_norm(p, std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi));
}

// The tables, formed once per process: cos and sin of (2 j + 1) pi/512 by powers
// of e^(i pi/512) (its series) in pairs of doubles.
const NoiseTables& noise_tables()
{
    static const NoiseTables tables = [] {
        NoiseTables t;
        for (int i = 0; i < kNoiseTable; i++) {
            const double r = i == kNoiseTable - 1 ? 0.5 : 1.0 / (1.0 + (i + 0.5) / kNoiseTable);
            const double l = -std::log(i >= kNoiseTable / 2 ? 2.0 * r : r), lead = std::rint(l * 0x1p40) * 0x1p-40;
            t.lg[i] = make_double2(r, lead);
            t.lo[i] = l - lead;
        }
        // log 2 to 40 bits, and the rest (log 2 less its nearest double is 2.319e-17)
        const double ln2 = 0.693147180559945309417, hi = std::rint(ln2 * 0x1p40) * 0x1p-40;
        for (int i = 0; i < 34; i++) t.l2[i] = make_double2((i - 33) * hi, (i - 33) * ((ln2 - hi) + 2.319046813846299558e-17));
        // pi = 3.141592653589793116 + 1.2246467991473532e-16
        const DD x{3.141592653589793116 / kNoiseTable, 1.2246467991473532e-16 / kNoiseTable}, x2 = dd_mul(x, x);
        DD c{1.0, 0.0}, sn = x, tc = c, ts = x;
        for (int k = 1; k <= 8; k++) {   // the next terms of the two series, (-1)^k x^(2k)/(2k)! and x^(2k+1)/(2k+1)!
            const double fc = (2.0 * k - 1) * (2 * k), fs = 2.0 * k * (2 * k + 1);
            auto over = [](DD a, double f) {
                const double q = a.hi / f;
                return dd_norm(q, (std::fma(-q, f, a.hi) + a.lo) / f);
            };
            tc = over(dd_mul(tc, x2), -fc);
            ts = over(dd_mul(ts, x2), -fs);
            c = dd_add(c, tc);
            sn = dd_add(sn, ts);
        }
        auto neg = [](DD a) { return DD{-a.hi, -a.lo}; };
        const DD wc = dd_add(dd_mul(c, c), neg(dd_mul(sn, sn))), cs = dd_mul(c, sn), ws = dd_add(cs, cs);   // (c + i sn)^2
        for (int j = 0; j < kNoiseTable; j++) {
            t.cs[j] = make_double2(c.hi, sn.hi);
            t.clo[j] = c.lo;
            const DD c1 = dd_add(dd_mul(c, wc), neg(dd_mul(sn, ws)));
            sn = dd_add(dd_mul(c, ws), dd_mul(sn, wc));
            c = c1;
        }
        return t;
    }();
    return tables;
}

__device__ __forceinline__ double noise_normal(uint32_t c0, uint32_t c1, const NoiseTables& t)
{
    // m = 2 c0 + 1 = 2^e f
    const uint64_t m = 2ull * c0 + 1ull;
    const int e = 63 - __clzll((long long)m);
    const uint64_t frac = (m << (52 - e)) & 0x000fffffffffffffull;
    const double f = __longlong_as_double((long long)(0x3ff0000000000000ull | frac));
    const int i = (int)(frac >> (52 - kNoiseBits));
    const double2 q = t.lg[i];
    const double x = fma(f, q.x, -1.0);
    const double2 b = t.l2[e + (i >= kNoiseTable / 2 ? 1 : 0)];
    double p = fma(x, -1.0 / 6.0, 1.0 / 5.0);
    p = fma(x, p, -1.0 / 4.0);
    p = fma(x, p, 1.0 / 3.0);
    p = fma(x, p, -1.0 / 2.0);
    const double lg = (b.x + q.y) + (fma(x * x, p, x) + (t.lo[i] + b.y));
    // cos(2 pi u2)
    const int j = (int)(c1 >> (32 - kNoiseBits));
    const int k = (int)(2u * (c1 & ((1u << (32 - kNoiseBits)) - 1u)) + 1u) - (1 << (32 - kNoiseBits));
    const double2 w = t.cs[j];
    const double d = (double)k * (6.283185307179586476925 / 8589934592.0), d2 = d * d;
    const double sn = fma(d * d2, fma(d2, 1.0 / 120.0, -1.0 / 6.0), d);
    const double cm = d2 * fma(d2, fma(d2, -1.0 / 720.0, 1.0 / 24.0), -0.5);   // cos d - 1
    const double cs = w.x + fma(w.x, cm, fma(-w.y, sn, t.clo[j]));
    return sqrt(-2.0 * lg) * cs;
}

__global__ void __launch_bounds__(512) white_noise_kernel(double* out, size_t count, uint64_t seed, uint32_t field,
                                                          uint32_t quantity, const NoiseTables* tables)
{
    __shared__ NoiseTables t;
    for (int i = threadIdx.x; i < (int)(sizeof(NoiseTables) / 8); i += blockDim.x)
        reinterpret_cast<double*>(&t)[i] = reinterpret_cast<const double*>(tables)[i];
    __syncthreads();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        uint32_t c[4] = {(uint32_t)i, field, quantity, 0u};
        philox4x32_10(c, (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
        out[i] = noise_normal(c[0], c[1], t);
    }
}

// s_k = sin^2(pi n_k / N) of the wave numbers n_k = k or k - N, k in [0, N).
__global__ void axis_table_kernel(double* s, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double q = sinpi((double)(k < n / 2 ? k : k - n) / n);
    s[k] = q * q;
}

// Multiply the half spectrum (kx in [0, N/2], layout [kz][ky][kx]) by the vacuum
// amplitude: fields 1/sqrt(2 w), momenta sqrt(w/2), times amp = fluct A B dx^-3/2,
// with w^2 = k_lat^2 + m_eff^2, k_lat^2 = sum_d (2/dx sin(pi n_d/N))^2. Empty for
// |n| = 0, |n| > kcut or w^2 <= 0. |n| is compared as an integer (n2max = the
// largest |n|^2 inside the cut): with the default cut of N/4 seven modes in
// eight are only cleared, and the amplitude's FP64 work (the pass's bound) is
// done for the rest, the sines from a table of one axis (256^3: 1.81 -> 0.085 ms).
__global__ void spectral_scale_kernel(cufftDoubleComplex* spec, int n, const double* __restrict__ axis, double dx,
                                      double meff2, double amp, int n2max, int quantity, int stencil)
{
    const int nh = n / 2 + 1;
    const double dx2 = dx * dx;
    for (int row = blockIdx.x * blockDim.y + threadIdx.y; row < n * n; row += gridDim.x * blockDim.y) {
        const int ky = row % n, kz = row / n;
        const int ny = ky < n / 2 ? ky : ky - n, nz = kz < n / 2 ? kz : kz - n;
        const int nyz = ny * ny + nz * nz;
        double2* p = reinterpret_cast<double2*>(spec) + (size_t)row * nh;
        for (int kx = threadIdx.x; kx < nh; kx += blockDim.x) {
            const int n2 = kx * kx + nyz;   // kx = N/2 stands for -N/2: the same square
            double scale = 0.0;
            if (n2 > 0 && n2 <= n2max) {
                // k_lat^2 = -L(k) of the stencil in s_i = sin^2(pi n_i / N) (no
                // cancellation at small k): 7-point 4 sum s_i / dx^2; 27-point
                // (4 sum s_i - 8/3 sum_{i<j} s_i s_j + 32/15 s_1 s_2 s_3) / dx^2, the weights
                // 14/30, 3/30, 1/30 of face, edge and corner neighbours written with
                // cos(k_i dx) = 1 - 2 s_i
                const double s1 = axis[kx], s2 = axis[ky], s3 = axis[kz];
                double klat = 4.0 * (s1 + s2 + s3);
                if (stencil == 27) klat += -8.0 / 3.0 * (s1 * s2 + s1 * s3 + s2 * s3) + 32.0 / 15.0 * s1 * s2 * s3;
                const double w2 = klat / dx2 + meff2;
                if (w2 > 0.0) {
                    const double w = sqrt(w2);
                    scale = amp * (quantity == 0 ? rsqrt(2.0 * w) : sqrt(0.5 * w));
                }
            }
            if (scale != 0.0) {
                const double2 v = p[kx];
                p[kx] = make_double2(v.x * scale, v.y * scale);
            } else {
                p[kx] = make_double2(0.0, 0.0);
            }
        }
    }
}

// f = fh + df + (dt/2) pi and f' = ph + dp + r h0 df, with the inverse DFT's
// 1/N^3 applied here; the half-step drift of Sec. II.B is taken in FP64 before
// rounding to the storage type. Writes ping-pong set 0.
template <typename T>
__global__ void init_combine_kernel(Bufs<T> B, int field, const double* df, const double* dp, double fh, double ph,
                                    double r_h0, double half_dt, double inv_n3, size_t count)
{
    T* f = B.f[0][field];
    T* p = B.p[0][field];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        const double d = df ? df[i] * inv_n3 : 0.0;
        const double q = dp ? dp[i] * inv_n3 : 0.0;
        const double pv = ph + q + r_h0 * d;
        const double fv = fh + d + half_dt * pv;
        f[i] = (T)fv;
        p[i] = (T)pv;
    }
}

int grid_for(size_t count)
{
    size_t b = (count + 255) / 256;
    return (int)(b < 4096 ? b : 4096);
}

} // namespace

size_t init_tables_bytes(int n) { return sizeof(NoiseTables) + sizeof(double) * (size_t)n; }

cudaError_t launch_init_tables(void* tables, int n, cudaStream_t st)
{
    cudaError_t e = cudaMemcpyAsync(tables, &noise_tables(), sizeof(NoiseTables), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    axis_table_kernel<<<(n + 63) / 64, 64, 0, st>>>((double*)((NoiseTables*)tables + 1), n);
    return cudaGetLastError();
}

cudaError_t launch_white_noise(double* out, int n, uint64_t seed, uint32_t field, uint32_t quantity,
                               const void* tables, cudaStream_t st)
{
    const size_t count = (size_t)n * n * n;
    // a few blocks per SM: each loads the tables once
    const size_t blocks = (count + 511) / 512;
    white_noise_kernel<<<(int)(blocks < 608 ? blocks : 608), 512, 0, st>>>(out, count, seed, field, quantity,
                                                                           (const NoiseTables*)tables);
    return cudaGetLastError();
}

cudaError_t launch_spectral_scale(void* spec, int n, const void* tables, double dx, double meff2, double amp, double kcut,
                                  int quantity, int stencil, cudaStream_t st)
{
    // the largest |n|^2 with sqrt(|n|^2) <= kcut
    const double most = 3.0 * (n / 2) * (n / 2);
    int n2max = (int)(kcut * kcut < most ? kcut * kcut : most);
    while (n2max > 0 && sqrt((double)n2max) > kcut) n2max--;
    while (n2max < (int)most && sqrt((double)(n2max + 1)) <= kcut) n2max++;
    const int rows = n * n, ty = 8;
    const int blocks = (rows + ty - 1) / ty;
    spectral_scale_kernel<<<blocks < 4096 ? blocks : 4096, dim3(32, ty), 0, st>>>(
        (cufftDoubleComplex*)spec, n, (const double*)((const NoiseTables*)tables + 1), dx, meff2, amp, n2max, quantity,
        stencil);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init_combine(const Bufs<T>& b, int field, const double* df, const double* dp, double fh,
                                double ph, double r_h0, double half_dt, int n, cudaStream_t st)
{
    const size_t count = (size_t)n * n * n;
    init_combine_kernel<T><<<grid_for(count), 256, 0, st>>>(b, field, df, dp, fh, ph, r_h0, half_dt,
                                                            1.0 / (double)count, count);
    return cudaGetLastError();
}

template cudaError_t launch_init_combine<float>(const Bufs<float>&, int, const double*, const double*, double,
                                                double, double, double, int, cudaStream_t);
template cudaError_t launch_init_combine<double>(const Bufs<double>&, int, const double*, const double*, double,
                                                 double, double, double, int, cudaStream_t);

} // namespace lat

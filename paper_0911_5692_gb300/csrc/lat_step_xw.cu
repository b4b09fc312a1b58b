// lat_step_xw.cu -- the compiled instances of the fused 7-point step over x
// tiles one warp wide (variant 5, lat_xw.cuh) for whole periodic lattices, and
// their launch configuration.
#include <algorithm>

#include "lat_xw.cuh"

namespace lat {

namespace {

// The compiled instance for a side, tile height and prefetch depth. FP32 sides of
// at most 128 take whole rows in tiles of 16 or 8 rows with two planes in flight:
// without the edge warp, and with two pairs of rows to a warp up to N = 64, a step is
// 1.1 us (100^3: 16.8 -> 15.7) to 1.6 us (64^3: 12.6 -> 11.0) shorter.
struct XWInst {
    const void* fn = nullptr;
    size_t smem = 0;
    int threads = 0;
};
template <typename T>
XWInst xw_inst(int n, int ty, int depth)
{
#define LAT_XW_CASE(TT, DD, SS)                                        \
    {                                                                  \
        typedef xw::XW<T, TT, DD, false, SS> F;                        \
        return XWInst{(const void*)xw::step_xw_kernel<T, TT, DD, false, SS>, F::SMEM, F::THREADS}; \
    }
    if constexpr (sizeof(T) == 4) {
        if (ty == 16 && depth == 2 && n <= 64) LAT_XW_CASE(16, 2, 16)
        if (ty == 16 && depth == 2 && n <= 128) LAT_XW_CASE(16, 2, 32)
        if (ty == 8 && depth == 2 && n <= 128) LAT_XW_CASE(8, 2, 32)
        if (ty == 16 && depth == 3) LAT_XW_CASE(16, 3, 0)
        if (ty == 8 && depth == 2) LAT_XW_CASE(8, 2, 0)
        if (ty == 8 && depth == 3) LAT_XW_CASE(8, 3, 0)
    } else {
        if (ty == 8 && depth == 1) LAT_XW_CASE(8, 1, 0)
        if (ty == 4 && depth == 1) LAT_XW_CASE(4, 1, 0)
    }
    if (ty == 16 && depth == 1) LAT_XW_CASE(16, 1, 0)
    if (ty == 16 && depth == 2) LAT_XW_CASE(16, 2, 0)
#undef LAT_XW_CASE
    return XWInst{};
}

XWInst xw_inst(int esize, int n, int ty, int depth)
{
    return esize == 4 ? xw_inst<float>(n, ty, depth) : xw_inst<double>(n, ty, depth);
}

} // namespace

bool xw_config(int n, int elem_bytes, int ty, int zr, int depth, MarchConfig* cfg)
{
    const int tyv = ty > 0 ? ty : 16;
    // the instance with the requested depth, else any compiled depth (2 first: a
    // second plane in flight takes the 512^3 FP32 step from 843 to 685 us and the
    // 256^3 step from 114 to 98; a third changes them by less than the runs differ)
    int d = depth;
    XWInst I;
    if (d > 0) I = xw_inst(elem_bytes, n, tyv, d);
    else
        for (int dd : {2, 1})
            if ((I = xw_inst(elem_bytes, n, tyv, dd)).fn) {
                d = dd;
                break;
            }
    const void* fn = I.fn;
    const size_t smem = I.smem;
    if (!fn || smem > 227 * 1024 - 2048) return false;
    const int vw = 16 / elem_bytes, nxt = (n / vw + 31) / 32;
    const int threads = I.threads;
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
    const long long groups = blocks / nxt;
    cfg->ty = tyv;
    // planes of the first group's first run (the z chunk of one tile when the
    // groups march the tiles in step, lat_layout.cuh)
    const Layout L0 = tile_layout(nyt, (int)groups, 0, n);
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
    cfg->s27 = 0;
    cfg->xt = 0;
    cfg->xw = 1;
    cfg->nxt = nxt;
    return true;
}

template <typename T>
cudaError_t launch_step_xw(const Bufs<T>& b, const Model& M, DevScalars* sc, double* partials, const MarchConfig& cfg,
                           cudaStream_t st)
{
    const void* fn = xw_inst<T>(M.n, cfg.ty, cfg.depth).fn;
    if (!fn) return cudaErrorInvalidValue;
    xw::SlabRun R{0, 0, nullptr};
    void* args[] = {(void*)&b, (void*)&M, (void*)&sc, (void*)&partials, (void*)&R};
    return launch_chained(fn, dim3(cfg.blocks), dim3(cfg.threads), args, cfg.smem, st, cfg.chain);
}

template cudaError_t launch_step_xw<float>(const Bufs<float>&, const Model&, DevScalars*, double*, const MarchConfig&,
                                           cudaStream_t);
template cudaError_t launch_step_xw<double>(const Bufs<double>&, const Model&, DevScalars*, double*,
                                            const MarchConfig&, cudaStream_t);

} // namespace lat

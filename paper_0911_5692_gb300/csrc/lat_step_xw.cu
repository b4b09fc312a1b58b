// lat_step_xw.cu -- the compiled instances of the fused 7-point step over x
// tiles one warp wide (variant 5, lat_xw.cuh) for whole periodic lattices, and
// their launch configuration.
#include <algorithm>

#include "lat_xw.cuh"

namespace lat {

namespace {

// The compiled instance of a tile height and prefetch depth, or null.
template <typename T>
const void* xw_fn(int ty, int depth, size_t* smem)
{
#define LAT_XW_CASE(TT, DD)                                 \
    if (ty == TT && depth == DD) {                          \
        *smem = xw::XW<T, TT, DD, false>::SMEM;             \
        return (const void*)xw::step_xw_kernel<T, TT, DD, false>; \
    }
    LAT_XW_CASE(16, 1) LAT_XW_CASE(16, 2)
    if constexpr (sizeof(T) == 4) { LAT_XW_CASE(16, 3) LAT_XW_CASE(8, 2) LAT_XW_CASE(8, 3) }
    else { LAT_XW_CASE(8, 1) LAT_XW_CASE(4, 1) }
#undef LAT_XW_CASE
    return nullptr;
}

const void* xw_kernel(int esize, int ty, int depth, size_t* smem)
{
    return esize == 4 ? xw_fn<float>(ty, depth, smem) : xw_fn<double>(ty, depth, smem);
}

} // namespace

bool xw_config(int n, int elem_bytes, int ty, int zr, int depth, MarchConfig* cfg)
{
    const int tyv = ty > 0 ? ty : 16;
    // the instance with the requested depth, else any compiled depth (2 first: a
    // second plane in flight takes the 512^3 FP32 step from 843 to 685 us and the
    // 256^3 step from 114 to 98; a third changes them by less than the runs differ)
    int d = depth;
    size_t smem = 0;
    const void* fn = nullptr;
    if (d > 0) fn = xw_kernel(elem_bytes, tyv, d, &smem);
    else
        for (int dd : {2, 1})
            if ((fn = xw_kernel(elem_bytes, tyv, dd, &smem))) {
                d = dd;
                break;
            }
    if (!fn || smem > 227 * 1024 - 2048) return false;
    const int vw = 16 / elem_bytes, nxt = (n / vw + 31) / 32;
    const int threads = (tyv / 2 + 2) * 32;
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
    size_t smem = 0;
    const void* fn = xw_fn<T>(cfg.ty, cfg.depth, &smem);
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

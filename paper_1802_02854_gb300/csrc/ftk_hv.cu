// Tiled H.V passes: the FP32 kernel (hv_tile_body in ftk_hv_tile.cuh; FP64 in
// ftk_hv_fix.cu, double-float in ftk_hv_df.cu) and, on the host, the layout of a
// planned pass and the launches.
#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_hv_tile.cuh"
#include "ftk_kernels.h"
#include "ftk_plan.h"

#include <algorithm>
#include <math.h>
#include <mutex>

namespace ftk {

// Grid (tiles, columns); column j at j ld elements.
template <class I, int EPI, int TB>
__global__ void __launch_bounds__(kTileThreads, 1)
hv_tile_kernel(const float2 *__restrict__ in, float2 *out, long long ld, const __grid_constant__ PassDesc pd,
               const __grid_constant__ EpiArgs ea0) {
    launch_dependents();
    hv_tile_body<I, EPI, TB>(in, out, pd, ea0, ld);
}

// ===================================================================== host
// Amplitudes per 16-byte item (log2), and the tile sizes: at most 4096 items
// (three 64 KB buffers and 32 KB of diagonal coefficients a CTA), at least 128
// (a warp of four items a thread; 256 for double-float, eight a thread). Smaller
// tiles run as gather passes.
static int item_shift(int prec) { return prec == 1 ? 1 : 0; }
int hv_max_tile_bits(int prec) { return 12 + item_shift(prec); }
bool hv_tiled(int prec, const PassDesc &pd) {
    if (prec == 2) return pd.tile_bits >= 8 && pd.tile_bits - pd.chunk_bits >= 3;
    return pd.tile_bits >= 7 + item_shift(prec) && pd.chunk_bits >= item_shift(prec) && pd.tile_bits - pd.chunk_bits >= 2;
}
static int hv_threads(int prec, const PassDesc &pd) { return 1 << (pd.tile_bits - (prec == 2 ? 3 : 2) - item_shift(prec)); }
static size_t hv_smem_bytes(int prec, const PassDesc &pd) {
    const size_t items = (size_t)1 << (pd.tile_bits - item_shift(prec));
    return items * (3 * 16 + (prec == 2 ? 0 : 8)) + (size_t)(hv_threads(prec, pd) / 32) * 2 * 8;
}

// Lay a planned pass out for the kernels: the register sites are the two
// non-chunk tile sites with the fewest bonds of the pass (the offset bits are
// renumbered chunk sites, other sites, register sites), and the bonds are
// sorted by class.
bool hv_layout_pass(PassDesc &pd, int prec) {
    const int b = pd.tile_bits, c = pd.chunk_bits, nb = pd.n_bonds;
    if (!hv_tiled(prec, pd)) return false;
    if (prec == 2) return df_layout_pass(pd);
    int degree[FTK_MAX_TILE_BITS] = {};
    for (int l = 0; l < nb; ++l) { ++degree[pd.bi[l]]; ++degree[pd.bj[l]]; }
    int reg[2] = {-1, -1};
    for (int &r : reg)
        for (int o = c; o < b; ++o)
            if (o != reg[0] && (r < 0 || degree[o] < degree[r])) r = o;
    int newpos[FTK_MAX_TILE_BITS], w = 0;
    for (int o = 0; o < b; ++o)
        if (o != reg[0] && o != reg[1]) newpos[o] = w++;
    newpos[reg[0]] = w++;
    newpos[reg[1]] = w;
    PassDesc q = pd;
    for (int o = 0; o < b; ++o) q.tile_pos[newpos[o]] = pd.tile_pos[o];
    const int sh = item_shift(prec), kbit = b - 2;
    w = 0;
    q.classes = 0;
    for (int cls = 0; cls < 24; ++cls) {
        const int w0 = w;
        for (int l = 0; l < nb; ++l) {
            const int bi = newpos[pd.bi[l]], bj = newpos[pd.bj[l]];
            const uint32_t m = (1u << bi) | (1u << bj);
            const int swap = sh && (m & 1), km = (int)(m >> kbit);
            if (bond_class(prec == 1, pd.gam[l], swap, km) != cls) continue;
            q.bi[w] = (int8_t)bi;
            q.bj[w] = (int8_t)bj;
            q.gam[w] = pd.gam[l];
            q.fdesc[w++] = ((m & ((1u << kbit) - 1)) >> sh) << 4 | (uint32_t)km << 16 | (swap ? 1u << 31 : 0u);
        }
        q.f_end[cls] = w;
        if (w > w0) q.classes |= 1u << cls;
    }
    pd = q;
    return true;
}

static TileKernel f32_kernel(int epi, bool full) {
    switch (epi) {
    case EPI_PLAIN: return full ? hv_tile_kernel<ItemF32, EPI_PLAIN, 10> : hv_tile_kernel<ItemF32, EPI_PLAIN, 0>;
    case EPI_COCG: return full ? hv_tile_kernel<ItemF32, EPI_COCG, 10> : hv_tile_kernel<ItemF32, EPI_COCG, 0>;
    case EPI_COCG_MIXED:
        return full ? hv_tile_kernel<ItemF32, EPI_COCG_MIXED, 10> : hv_tile_kernel<ItemF32, EPI_COCG_MIXED, 0>;
    default: return nullptr;
    }
}

template <typename K>
static cudaError_t opt_in(K kern) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    return e;
}

// Opt every pass kernel into the full shared memory once per process (outside
// any stream capture); thread-safe (contexts may be created from several host
// threads, as the server does).
static cudaError_t init_attributes_once() {
    cudaError_t e = cudaSuccess;
    for (int epi : {EPI_PLAIN, EPI_COCG, EPI_COCG_MIXED, EPI_TPQ, EPI_TAYLOR})
        for (bool full : {false, true}) {
            if (f32_kernel(epi, full) && e == cudaSuccess) e = opt_in(f32_kernel(epi, full));
            if (df_kernel(epi, full) && e == cudaSuccess) e = opt_in(df_kernel(epi, full));
            if (fix_kernel(epi, full) && e == cudaSuccess) e = opt_in(fix_kernel(epi, full));
        }
    return e == cudaSuccess ? fix_attributes() : e;
}

cudaError_t init_kernel_attributes() {
    static std::once_flag once;
    static cudaError_t status = cudaSuccess;
    std::call_once(once, [] { status = init_attributes_once(); });
    return status;
}

cudaError_t launch_hv_pass(int prec, int B, int epi, const void *in, void *out, const PassDesc &pd,
                           const EpiArgs &ea, int grid_cap, cudaStream_t st) {
    if (B < 1 || B > FTK_MAX_RHS || !hv_tiled(prec, pd) || pd.tile_bits > hv_max_tile_bits(prec) ||
        ((epi == EPI_TPQ || epi == EPI_TAYLOR) && (B != 1 || prec != 0)) || (epi == EPI_TAYLOR && !ea.taylor_acc) ||
        (ea.lo && prec != 1) || (prec == 2 && ea.df_lo <= 0))
        return cudaErrorInvalidConfiguration;
    const int ep = epi == EPI_COCG && ea.lo ? EPI_COCG_MIXED : epi;
    const bool full = pd.tile_bits == hv_max_tile_bits(prec);
    const int threads = hv_threads(prec, pd);
    const size_t smem = hv_smem_bytes(prec, pd);
    const TileKernel kt = prec == 1 ? f32_kernel(ep, full) : prec == 2 ? df_kernel(ep, full) : nullptr;
    const FixKernel kf = prec == 0 ? fix_kernel(ep, full) : nullptr;
    if (!kt && !kf) return cudaErrorInvalidValue;
    int per_sm = 0, dev = 0, n_sm = 0;
    cudaError_t e = kf ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kf, threads, smem)
                       : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kt, threads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    // persistent: the CTAs of all columns resident at once (within the caller's
    // partial buffers)
    long g = std::max(1L, std::min<long>((long)per_sm * n_sm, grid_cap) / B);
    g = std::min(g, 1L << pd.n_free);
    const long long ld = 1LL << pd.n_sites;
    const dim3 grid((unsigned)g, B);
    return kf ? launch_chained(kf, grid, threads, smem, st, static_cast<const double2 *>(in), static_cast<double2 *>(out),
                               ld, pd, ea)
              : launch_chained(kt, grid, threads, smem, st, static_cast<const float2 *>(in), static_cast<float2 *>(out), ld,
                               pd, ea);
}

}  // namespace ftk

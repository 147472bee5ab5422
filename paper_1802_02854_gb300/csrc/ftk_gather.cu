// The matrix-free H.V of vectors that sit in the L2 cache, in one launch: one
// thread per amplitude reads its partners x ^ m of all bonds straight from
// global memory.
//
// Why beside the tiled passes of ftk_hv.cu: a tile of 2^12 amplitudes is the
// unit of work there, so a small vector occupies few SMs (12 sites: one tile,
// hence one SM, and 36 us of its FP64 pipe; 16 sites: 16 SMs and two
// launches), while here 2^n threads spread over all of them. The price is one
// 16-byte L2 read per bond and amplitude instead of a shared-memory one, so
// the tiles win again once the reads of a launch cost more than the passes'
// launches and empty SMs (hv_use_gather, with both sides measured). Passes
// whose requested tiles are too small for the tiled kernels run here too, one
// launch per pass over the pass's bonds.
#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_kernels.h"
#include "ftk_plan.h"

#include <algorithm>
#include <type_traits>

namespace ftk {

// partners in flight per thread: the loads of a chunk are independent, and
// their latency (not their bandwidth) is what a small launch waits for
constexpr int kGatherChunk = 6;

// One column's vector in each arithmetic: load an amplitude, add c times a
// partner's, and the finished value. The order of the types, and what is summed
// apart (next_type before the second and third type, join after them), set the
// rounding. FP64 and FP32: z with its smaller coefficients, x on top of it, y from
// zero. One sum over x, y and z had 1.1 to 1.25 times the error of the tiled
// passes; so FP64 1.16e-16, FP32 6.7e-8 of the norm at 18 sites (one sum: 1.57e-16, 8.8e-8;
// tiled multiply-adds 1.27e-16, 7.1e-8), in FP64 for 2 % more time there (33.1 -> 33.9 us).
template <int PREC> struct GatherVec;
template <int PREC> __device__ constexpr int gather_type(int k) { return PREC == 2 ? k : (k + 2) % 3; }
template <> struct GatherVec<0> {
    typedef double2 amp;
    typedef double coef;
    double2 s = {0.0, 0.0}, t = {0.0, 0.0};
    __device__ static amp load(const void *p, size_t i, long long) { return static_cast<const double2 *>(p)[i]; }
    __device__ static coef c(const GatherDesc &g, int q, bool anti) { return anti ? g.tc.anti[q] : g.tc.par[q]; }
    __device__ void add(coef c, const amp &a) { s.x = fma(c, a.x, s.x); s.y = fma(c, a.y, s.y); }
    __device__ void next_type(int k) {
        if (k == 2) { t = s; s = make_double2(0.0, 0.0); }
    }
    __device__ void join() { partial(t); }
    __device__ void partial(const amp &a) { s.x += a.x; s.y += a.y; }
    __device__ void diag(const GatherDesc &g, int c0, int c1, const amp &a) {
        add((double)c0 * g.tc.dgv[0] + (double)c1 * g.tc.dgv[1], a);
    }
};
template <> struct GatherVec<1> {
    typedef float2 amp;
    typedef float coef;
    float2 s = {0.f, 0.f}, t = {0.f, 0.f};
    __device__ static amp load(const void *p, size_t i, long long) { return static_cast<const float2 *>(p)[i]; }
    __device__ static coef c(const GatherDesc &g, int q, bool anti) { return anti ? g.tc.anti_f[q] : g.tc.par_f[q]; }
    __device__ void add(coef c, const amp &a) { s = __ffma2_rn(make_float2(c, c), a, s); }
    __device__ void next_type(int k) {
        if (k == 2) { t = s; s = make_float2(0.f, 0.f); }
    }
    __device__ void join() { partial(t); }
    __device__ void partial(const amp &a) { s = __fadd2_rn(s, a); }
    __device__ void diag(const GatherDesc &g, int c0, int c1, const amp &a) {
        add((float)c0 * g.tc.dgv_f[0] + (float)c1 * g.tc.dgv_f[1], a);
    }
};
template <> struct GatherVec<2> {
    typedef float4 amp;    // (hi.re, hi.im, lo.re, lo.im)
    typedef float2 coef;   // (hi, lo)
    float2 h = {0.f, 0.f}, l = {0.f, 0.f}, th = {0.f, 0.f}, tl = {0.f, 0.f};
    __device__ static amp load(const void *p, size_t i, long long lo) {
        const float2 *q = static_cast<const float2 *>(p) + i;
        const float2 a = q[0], b = q[lo];
        return make_float4(a.x, a.y, b.x, b.y);
    }
    __device__ static coef c(const GatherDesc &g, int q, bool anti) {
        return anti ? make_float2(g.tc.anti_f[q], g.tc.anti_lo[q]) : make_float2(g.tc.par_f[q], g.tc.par_lo[q]);
    }
    __device__ void add(coef c, const amp &a) {
        df_acc2(h, l, make_float2(c.x, c.x), make_float2(-c.x, -c.x), make_float2(c.y, c.y), make_float2(a.x, a.y),
                make_float2(a.z, a.w));
    }
    // The bonds of a type are summed from zero and their renormalised pair is
    // carried to the next type's: the low parts of one sum over all bonds grow
    // and round more (18 sites: 6.2e-15 of the norm, so 4.3e-15; the tiled passes, which
    // do the same between passes, 4.7e-15).
    __device__ void next_type(int) {
        df_add_to2(h, l, th, tl);
        th = __fadd2_rn(h, l);
        tl = fsub2(l, fsub2(th, h));
        h = l = make_float2(0.f, 0.f);
    }
    __device__ void join() {}
    __device__ void partial(const amp &a) { df_add_to2(h, l, make_float2(a.x, a.y), make_float2(a.z, a.w)); }
    __device__ void diag(const GatherDesc &g, int c0, int c1, const amp &a) {
        const dfl d = dfl_add(dfl_mul({(float)c0, 0.f}, {g.tc.dgv_f[0], g.tc.dgv_lo[0]}),
                              dfl_mul({(float)c1, 0.f}, {g.tc.dgv_f[1], g.tc.dgv_lo[1]}));
        add(make_float2(d.hi, d.lo), a);
    }
    // the renormalised pair
    __device__ amp value() {
        df_add_to2(h, l, th, tl);
        const float2 hh = __fadd2_rn(h, l);
        const float2 ll = fsub2(l, fsub2(hh, h));
        return make_float4(hh.x, hh.y, ll.x, ll.y);
    }
};

// Grid (blocks, columns); element (x, j) at j 2^n + x. Reductions: per-block
// partials of the column, summed in a fixed order by its last block.
template <int PREC, int EPI>
__global__ void __launch_bounds__(128) hv_gather_kernel(const void *__restrict__ in, void *out,
                                                        const __grid_constant__ GatherDesc gd,
                                                        const __grid_constant__ EpiArgs ea) {
    typedef GatherVec<PREC> V;
    typedef typename std::conditional<PREC == 0, double, float>::type R;
    constexpr int ND = EPI == EPI_PLAIN ? 1 : 2;
    __shared__ double red[(128 / 32) * ND];
    const int j = blockIdx.y;
    if (ea.all_done && *ea.all_done) return;
    if (ea.lowp && *ea.lowp != ea.lowp_run) return;
    if (ea.col_seed && ea.col_seed[j].done != 0) return;   // finished column: no work
    const uint32_t dim = 1u << gd.n_sites;
    const size_t base = (size_t)j * dim;
    Acc<R> dot[ND];
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < dim; x += gridDim.x * blockDim.x) {
        V acc;
        int anti[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int g = gather_type<PREC>(k);
            if (k > 0) acc.next_type(k);
            for (int b = gd.off[g]; b < gd.off[g + 1]; b += kGatherChunk) {
                typename V::amp p[kGatherChunk];
#pragma unroll
                for (int u = 0; u < kGatherChunk; ++u)
                    if (b + u < gd.off[g + 1]) p[u] = V::load(in, base + (x ^ gd.mask[b + u]), ea.df_lo);
#pragma unroll
                for (int u = 0; u < kGatherChunk; ++u)
                    if (b + u < gd.off[g + 1]) {
                        const int odd = __popc(x & gd.mask[b + u]) & 1;
                        anti[g] += odd;
                        acc.add(V::c(gd, g, odd != 0), p[u]);
                    }
            }
        }
        acc.join();
        // diagonal: (parallel - antiparallel) bonds of the two classes
        const int c0 = gd.off[2] - 2 * (anti[0] + anti[1]);
        const int c1 = gd.off[3] - gd.off[2] - 2 * anti[2];
        const typename V::amp v = V::load(in, base + x, ea.df_lo);
        acc.diag(gd, c0, c1, v);
        if (!gd.first) acc.partial(V::load(out, base + x, ea.df_lo));
        if constexpr (PREC == 2) {
            const float4 w = acc.value();
            float2 *o = static_cast<float2 *>(out) + base + x;
            o[0] = make_float2(w.x, w.y);
            o[ea.df_lo] = make_float2(w.z, w.w);
            if (EPI == EPI_COCG && gd.last) {   // mu = r^T w (bilinear) from hi + lo
                dot[0].fma_pair(v.x, v.z, w.x, w.z);
                dot[0].fma_pair(-v.y, -v.w, w.y, w.w);
                dot[1].fma_pair(v.x, v.z, w.y, w.w);
                dot[1].fma_pair(v.y, v.w, w.x, w.z);
            }
        } else {
            typedef typename C2<R>::t cx;
            cx *o = static_cast<cx *>(out) + base + x;
            if (!gd.last) *o = acc.s;
            else HvEpilogue<R, EPI>(ea).apply(ea, base + x, v, acc.s, o, dot);
        }
    }
    if (EPI != EPI_PLAIN && gd.last) {
        double d[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) d[q] = dot[q].get();
        block_reduce<ND>(d, red);
        double *part = ea.partials + (size_t)j * gridDim.x * ND;
        if (threadIdx.x < ND) part[(size_t)blockIdx.x * ND + threadIdx.x] = red[threadIdx.x];
        double *res = ea.result + (EPI == EPI_TPQ || EPI == EPI_TAYLOR ? 0 : (size_t)FTK_HV_DOTS * j);
        if (!last_block_reduce<ND>(part, ea.counter + j, res, red)) return;
        if (EPI == EPI_TPQ && threadIdx.x == 0) tpq_statistics(ea, res);
    }
}

bool gather_desc(int n, const PlanBond *bonds, int nb, double K, double J, GatherDesc *gd) {
    if (n < 2 || n > FTK_MAX_SITES || nb < 1 || nb > 2 * FTK_MAX_PASS_BONDS) return false;
    GatherDesc d{};
    d.n_sites = n;
    d.first = d.last = 1;
    d.tc = type_coefficients(K, J);
    int w = 0;
    for (int g = 0; g < 3; ++g) {
        d.off[g] = w;
        for (int q = 0; q < nb; ++q)
            if (bonds[q].g == g) d.mask[w++] = (1u << bonds[q].i) | (1u << bonds[q].j);
    }
    d.off[3] = w;
    if (w != nb) return false;
    *gd = d;
    return true;
}

void gather_pass(const PassDesc &pd, GatherDesc *gd) {
    GatherDesc d{};
    d.n_sites = pd.n_sites;
    d.first = pd.first;
    d.last = pd.last;
    d.tc = pd.tc;
    int w = 0;
    for (int g = 0; g < 3; ++g) {
        d.off[g] = w;
        for (int q = 0; q < pd.n_bonds; ++q)
            if (pd.gam[q] == g) d.mask[w++] = (1u << pd.tile_pos[pd.bi[q]]) | (1u << pd.tile_pos[pd.bj[q]]);
    }
    d.off[3] = w;
    *gd = d;
}

// Where the line lies, us per product of B vectors (n sites x B), gather against
// the tiled passes in their better tile size (K = -1, J = 0.1; products queued one
// after the other):
//   all B 2^n      2^17          2^18                      2^19                      2^20
//   FP64      16x2: 18 / 30   16x4: 31 / 33, 18x1: 34 / 41   16x8: 57 / 37, 18x2: 62 / 43  18x4: 119 / 65
//   FP32      16x2:  8 /  9   16x4: 12 / 10, 18x1: 13 / 14   16x8: 21 / 13, 18x2: 21 / 14  18x4: 37 / 23
//   DF        16x2: 10 / 21   16x4: 16 / 21, 18x1: 17 / 28   16x8: 27 / 26, 18x2: 29 / 34  16x16: 49 / 41,
//                                                                   18x4: 51 / 54, 20x1: 56 / 57
//             2^21: 18x8: 99 / 94, 20x2: 105 / 96
// FP64 and FP32 cross at 2^18, where the gather's L2 reads (and, in FP64, its
// multiply-adds at the FP64 pipe's rate) cost more than the passes' launches and
// empty SMs; double-float passes are dearer and cross at 2^20. Couplings without a
// fixed-point form (fix_couplings) leave the FP64 passes to the same pipe, which
// they use no better: 18x2 62 / 97, 20x1 129 / 178, 20x2 255 / 306, 20x4 505 / 545.
bool hv_use_gather(int prec, int n, int B, bool fix) {
    int w = n;
    for (int b = 1; b < B; b <<= 1) ++w;
    return w <= (prec == 2 ? 20 : prec == 0 && !fix ? 22 : 18);
}

// Threads per block: few for the smallest vectors, so that their blocks reach
// more SMs (32 / 64 / 128 threads, FP64: 14 sites 8.1 / 7.3 / 7.3 us, 16 sites 10.5 /
// 10.4 / 12.4, 18 sites 33.1 / 34.7 / 34.0; the launch's own time hides it below). Blocks per column: one amplitude per thread, at most 1024 blocks
// where their partial dots are summed by the last one.
static int gather_threads(int n) { return n <= 12 ? 32 : n <= 14 ? 64 : 128; }

template <int PREC>
static cudaError_t launch_prec(int epi, dim3 grid, int threads, const void *in, void *out, const GatherDesc &gd,
                               const EpiArgs &ea, cudaStream_t st) {
    switch (epi) {
    case EPI_PLAIN: hv_gather_kernel<PREC, EPI_PLAIN><<<grid, threads, 0, st>>>(in, out, gd, ea); break;
    case EPI_COCG: hv_gather_kernel<PREC, EPI_COCG><<<grid, threads, 0, st>>>(in, out, gd, ea); break;
    case EPI_COCG_MIXED:
        if constexpr (PREC == 1) hv_gather_kernel<1, EPI_COCG_MIXED><<<grid, threads, 0, st>>>(in, out, gd, ea);
        else return cudaErrorInvalidValue;
        break;
       
    case EPI_TPQ:
        if constexpr (PREC == 0) hv_gather_kernel<0, EPI_TPQ><<<grid, threads, 0, st>>>(in, out, gd, ea);
        else return cudaErrorInvalidValue;
        break;
       
    case EPI_TAYLOR:
        if constexpr (PREC == 0) hv_gather_kernel<0, EPI_TAYLOR><<<grid, threads, 0, st>>>(in, out, gd, ea);
        else return cudaErrorInvalidValue;
        break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_hv_gather(int prec, int B, int epi, const void *in, void *out, const GatherDesc &gd,
                             const EpiArgs &ea, cudaStream_t st) {
    if (B < 1 || B > FTK_MAX_RHS || ((epi == EPI_TPQ || epi == EPI_TAYLOR) && B != 1) ||
        (epi == EPI_TAYLOR && !ea.taylor_acc) || (ea.lo && prec != 1) || (prec == 2 && ea.df_lo <= 0))
        return cudaErrorInvalidConfiguration;
    const int threads = gather_threads(gd.n_sites);
    uint32_t blocks = ((1u << gd.n_sites) + threads - 1) / threads;
    if (epi != EPI_PLAIN && blocks > 1024) blocks = 1024;
    const dim3 grid(blocks, B);
    const int ep = epi == EPI_COCG && ea.lo ? EPI_COCG_MIXED : epi;
    if (prec == 0) return launch_prec<0>(ep, grid, threads, in, out, gd, ea, st);
    if (prec == 1) return launch_prec<1>(ep, grid, threads, in, out, gd, ea, st);
    return launch_prec<2>(ep, grid, threads, in, out, gd, ea, st);
}

}  // namespace ftk

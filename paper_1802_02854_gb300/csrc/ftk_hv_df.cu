// The tiled double-float H.V pass (precision mode FTK_DF): FP64-class accuracy on
// the FP32 pipe, which on GB300 issues 64x the FP64 rate. A vector is a pair of
// float arrays, hi and lo (lo df_lo float2 elements after hi), value hi + lo
// (~48 significant bits). The tile holds an amplitude's hi and lo parts together
// (one float4); a bond adds c p with the exact FMA two-product of the hi parts,
// the cross terms, and Knuth's two-sum into an accumulator (hi, lo) whose lo part
// collects the rounding errors (renormalised when stored).
//
// Tiles, passes and buffers as in ftk_hv_tile.cuh; thread layout of its own: 512
// threads, thread t owns the offsets t + T k, k < 8 (the top three offset bits
// are register bits). Bonds with the same thread part of their mask form a
// group: the thread reads the partner thread's 8 amplitudes once and applies
// every bond of the group from registers (the coefficient choice is resolved
// once per thread and bond from the thread bits, and at compile time from the
// register bits). The group with mask 0 holds the bonds between register sites,
// and the diagonal.
//
// What bounds it: the latency of 10 dependent packed f32x2 instructions a term at 16
// warps an SM (24 sites, one vector: 684 us; FMA pipe 51-55 % busy, issue slots
// 50-54 %; 752 us with 12 instructions, 775 without chained launches). The layout of ftk_hv_tile.cuh (1024 threads, a
// partner read per bond) ran 812 us against 752: its gain in latency
// does not outweigh the extra instructions here. Exact float pieces (the sums of
// ftk_hv_fix.cu on three aligned floats, 4.3 packed instructions a term) ran 959
// us: 24 bytes of shared reads per bond and amplitude.
#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_hv_tile.cuh"
#include "ftk_kernels.h"

namespace ftk {

constexpr int kDfLe = 3, kDfThreads = 512;

// coefficient pairs of one bond for one thread: hi, -hi, lo of the
// coefficient at register parity 0 (s) and 1 (f)
struct DfCoef {
    float2 sh, snh, sl, fh, fnh, fl;
};
template <int KA, int KB>
struct KMask {
    static constexpr int m = (KA >= 0 ? (1 << KA) : 0) | (KB >= 0 ? (1 << KB) : 0);
};
template <int LE, int KA, int KB>
__device__ __forceinline__ void bond_apply_df(float2 (&ah)[1 << LE], float2 (&al)[1 << LE], const float2 (&ph)[1 << LE],
                                              const float2 (&pl)[1 << LE], const DfCoef &c) {
    constexpr int E = 1 << LE;
#pragma unroll
    for (int k = 0; k < E; ++k) {
        const int kpar = (KA >= 0 ? (k >> KA) & 1 : 0) ^ (KB >= 0 ? (k >> KB) & 1 : 0);
        const int kp = k ^ KMask<KA, KB>::m;
        if (kpar) df_acc2(ah[k], al[k], c.fh, c.fnh, c.fl, ph[kp], pl[kp]);
        else df_acc2(ah[k], al[k], c.sh, c.snh, c.sl, ph[kp], pl[kp]);
    }
}

#define FTK_HV_DF_CASE(ID, KA, KB)                                                                   \
    case ID:                                                                                         \
        bond_apply_df<LE, KA, KB>(ah, al, ph, pl, cf);                                               \
        break;

// TB > 0: the thread bits of the tile (tile_bits - LE) as a compile-time
// constant, so that the strides T k of the shared tile fold into immediate
// offsets (2^12-amplitude tiles: TB = 9).
template <int EPI, int TB>
__global__ void __launch_bounds__(kDfThreads, 1)
hv_df_kernel(const float2 *__restrict__ in, float2 *out, long long ld, const __grid_constant__ PassDesc pd,
             const __grid_constant__ EpiArgs ea0) {
    constexpr int LE = kDfLe, E = 1 << LE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_dependents();
    const long long lo = ea0.df_lo;
    const int b = TB > 0 ? TB + LE : pd.tile_bits;
    const int tb = b - LE;
    const int tile_n = 1 << b;
    const int T = 1 << tb;
    const int t = threadIdx.x;
    // tile buffers of (hi.re, hi.im, lo.re, lo.im): one 16-byte shared load
    // per partner amplitude
    float4 *b0 = reinterpret_cast<float4 *>(smem_raw);
    float4 *b1 = b0 + tile_n, *pb = b1 + tile_n;
    double *red = reinterpret_cast<double *>(pb + tile_n);

    uint64_t st = 0;
    for (int q = 0; q < tb; ++q)
        if ((t >> q) & 1) st |= 1ull << pd.tile_pos[q];
    long long kofs[LE];
#pragma unroll
    for (int q = 0; q < LE; ++q) kofs[q] = (long long)(1ull << pd.tile_pos[tb + q]);
    auto eofs = [&](int k) -> long long {
        long long v = (long long)st;
#pragma unroll
        for (int q = 0; q < LE; ++q)
            if ((k >> q) & 1) v += kofs[q];
        return v;
    };
    // tile offsets: the bits of the tile index deposited at the free sites.
    // Successive tiles of a CTA are gridDim.x apart; their offsets follow by
    // a masked addition (the bits outside the mask set to 1 carry across
    // them): dep(a + g) = ((dep(a) | ~mask) + dep(g)) & mask.
    auto tile_ofs = [&](long tau) -> long long {
        uint64_t v = 0;
        for (int q = 0; q < pd.n_free; ++q)
            if ((tau >> q) & 1) v |= 1ull << pd.free_pos[q];
        return (long long)v;
    };
    // (mask and step in shared memory: read once per tile, no registers held)
    __shared__ uint64_t free_mask, dep_grid;
    if (threadIdx.x == 0) {
        uint64_t m = 0;
        for (int q = 0; q < pd.n_free; ++q) m |= 1ull << pd.free_pos[q];
        free_mask = m;
        dep_grid = (uint64_t)tile_ofs(gridDim.x);
    }
    __syncthreads();
    auto next_ofs = [&](long long ofs) -> long long {
        const uint64_t m = free_mask;
        return (long long)((((uint64_t)ofs | ~m) + dep_grid) & m);
    };
    // diagonal dgv[0] c0 + dgv[1] c1 in double-float arithmetic, once per thread: c
    // counts the parallel minus the antiparallel bonds, c0 of the x and y bonds, c1 of
    // the z bonds
    float dgh[E], dgl[E];
    {
        int c0[E], c1[E];
#pragma unroll
        for (int k = 0; k < E; ++k) { c0[k] = 0; c1[k] = 0; }
        for (int l = 0; l < pd.n_bonds; ++l) {
            const int m = (1 << pd.bi[l]) | (1 << pd.bj[l]);
            const int pt = __popc(t & m & (T - 1)) & 1;
            const int km = m >> tb;
            const int cls = pd.gam[l] == 2;
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const int sg = 1 - 2 * ((pt ^ __popc(k & km)) & 1);
                c0[k] += cls ? 0 : sg;
                c1[k] += cls ? sg : 0;
            }
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const dfl d = dfl_add(dfl_mul({(float)c0[k], 0.f}, {pd.tc.dgv_f[0], pd.tc.dgv_lo[0]}),
                                  dfl_mul({(float)c1[k], 0.f}, {pd.tc.dgv_f[1], pd.tc.dgv_lo[1]}));
            dgh[k] = d.hi;
            dgl[k] = d.lo;
        }
    }
    Acc<float> dot[2];
    const bool first = pd.first != 0;
    wait_previous();
    EpiArgs ea;
    if (!hv_column(ea0, ea, ld)) return;
    in += (size_t)blockIdx.y * ld;
    out += (size_t)blockIdx.y * ld;
    auto issue = [&](const float2 *src, long long tofs, float4 *b) {
        {
            const float2 *g = src + tofs, *gl = g + lo;
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const long long e = eofs(k);
                float2 *d = reinterpret_cast<float2 *>(b + t + T * k);
                cp_async8(d, g + e);
                cp_async8(d + 1, gl + e);
            }
        }
        cp_async_commit();
    };
    const long n_tiles = 1L << pd.n_free;
    long tau = blockIdx.x;
    long long tofs = tau < n_tiles ? tile_ofs(tau) : 0;
    if (tau < n_tiles) {
        issue(in, tofs, b0);
        if (!first) issue(out, tofs, pb);
    }
    for (int it = 0; tau < n_tiles; tau += gridDim.x, ++it) {
        const float4 *cb = (it & 1) ? b1 : b0;
        float4 *nb = (it & 1) ? b0 : b1;
        const long tn = tau + gridDim.x;
        const bool more = tn < n_tiles;
        const long long tofs_n = more ? next_ofs(tofs) : 0;
        if (more) issue(in, tofs_n, nb);
        if (first) { if (more) cp_async_wait<1>(); else cp_async_wait<0>(); }
        else { if (more) cp_async_wait<2>(); else cp_async_wait<1>(); }
        __syncthreads();
        {
            float2 ah[E], al[E];   // (re, im) hi and lo parts of the accumulators
            float2 ph[E], pl[E];
#pragma unroll
            for (int k = 0; k < E; ++k) { ah[k] = make_float2(0.f, 0.f); al[k] = make_float2(0.f, 0.f); }
            int q = 0;
            for (int g = 0; g < pd.n_groups; ++g) {
                const int tm = pd.grp_tmask[g];
#pragma unroll
                for (int k = 0; k < E; ++k) {
                    const float4 v4 = cb[(t ^ tm) + T * k];
                    ph[k] = make_float2(v4.x, v4.y);
                    pl[k] = make_float2(v4.z, v4.w);
                }
                const int pt = __popc(t & tm) & 1;
                for (const int end = pd.grp_end[g]; q < end; ++q) {
                    const float parh = pd.par_f[q], parl = pd.par_lo[q], anth = pd.anti_f[q], antl = pd.anti_lo[q];
                    const float sh_ = pt ? anth : parh, sl_ = pt ? antl : parl;
                    const float fh_ = pt ? parh : anth, fl_ = pt ? parl : antl;
                    const DfCoef cf = {make_float2(sh_, sh_), make_float2(-sh_, -sh_), make_float2(sl_, sl_),
                                       make_float2(fh_, fh_), make_float2(-fh_, -fh_), make_float2(fl_, fl_)};
                    switch (pd.bcase[q]) {
                        FTK_HV_DF_CASE(0, -1, -1)
                        FTK_HV_DF_CASE(1, 0, -1)
                        FTK_HV_DF_CASE(2, 1, -1)
                        FTK_HV_DF_CASE(3, 2, -1)
                        FTK_HV_DF_CASE(9 + 0 * 8 + 1, 0, 1)
                        FTK_HV_DF_CASE(9 + 0 * 8 + 2, 0, 2)
                        FTK_HV_DF_CASE(9 + 1 * 8 + 2, 1, 2)
                        default: break;
                    }
                }
            }
            // own amplitudes (last group): diagonal
#pragma unroll
            for (int k = 0; k < E; ++k)
                df_acc2(ah[k], al[k], make_float2(dgh[k], dgh[k]), make_float2(-dgh[k], -dgh[k]),
                        make_float2(dgl[k], dgl[k]), ph[k], pl[k]);
            if (!first) {
                if (more) cp_async_wait<1>(); else cp_async_wait<0>();
#pragma unroll
                for (int k = 0; k < E; ++k) {
                    const float4 v4 = pb[t + T * k];
                    df_add_to2(ah[k], al[k], make_float2(v4.x, v4.y), make_float2(v4.z, v4.w));
                }
            }
            float2 *o = out + tofs, *ol = o + lo;
#pragma unroll
            for (int k = 0; k < E; ++k) {
                // renormalise (fast two-sum) and store hi, lo
                const float2 hh = __fadd2_rn(ah[k], al[k]);
                const float2 ll = fsub2(al[k], fsub2(hh, ah[k]));
                const long long e = eofs(k);
                o[e] = hh;
                ol[e] = ll;
                if (EPI == EPI_COCG && pd.last) {
                    // mu = r^T w (bilinear) in double-float from hi + lo
                    dot[0].fma_pair(ph[k].x, pl[k].x, hh.x, ll.x);
                    dot[0].fma_pair(-ph[k].y, -pl[k].y, hh.y, ll.y);
                    dot[1].fma_pair(ph[k].x, pl[k].x, hh.y, ll.y);
                    dot[1].fma_pair(ph[k].y, pl[k].y, hh.x, ll.x);
                }
            }
        }
        if (!first && more) issue(out, tofs_n, pb);
        tofs = tofs_n;
        __syncthreads();
    }
    cp_async_wait<0>();
    if (EPI != EPI_COCG || !pd.last) return;
    double v[2] = {dot[0].get(), dot[1].get()};
    block_reduce<2>(v, red);
    if (threadIdx.x < 2) ea.partials[(size_t)blockIdx.x * 2 + threadIdx.x] = red[threadIdx.x];
    last_block_reduce<2>(ea.partials, ea.counter, ea.result, red);
}

// ===================================================================== host
// Choose the register sites of a planned pass and order its bonds in groups.
// The register sites are three of the non-chunk tile sites, picked to minimise
// the number of groups (shared-memory reads per amplitude); the offset bits are
// renumbered chunk sites, other thread sites, register sites.
bool df_layout_pass(PassDesc &pd) {
    const int b = pd.tile_bits, c = pd.chunk_bits, nb = pd.n_bonds;
    const int le = kDfLe, tb = b - le;
    // choose the register positions among offset bits [c, b)
    const int free_n = b - c;
    int best_set = -1, best_groups = 1 << 30, best_rr = -1;
    for (int set = 0; set < (1 << free_n); ++set) {
        if (__builtin_popcount(set) != le) continue;
        // bond masks with the chosen offset bits counted as register bits
        int tms[FTK_MAX_PASS_BONDS + 1];
        int ng = 0, rr = 0;
        for (int l = 0; l < nb; ++l) {
            int tm = 0, nreg = 0;
            for (int side = 0; side < 2; ++side) {
                const int o = side ? pd.bj[l] : pd.bi[l];
                const bool reg = o >= c && ((set >> (o - c)) & 1);
                if (reg) ++nreg;
                else tm |= 1 << o;   // thread masks compared as sets of offset bits
            }
            if (nreg == 2) ++rr;
            bool seen = tm == 0;
            for (int g = 0; g < ng && !seen; ++g) seen = tms[g] == tm;
            if (!seen) tms[ng++] = tm;
        }
        ++ng;   // the own group
        if (ng < best_groups || (ng == best_groups && rr > best_rr)) {
            best_groups = ng;
            best_rr = rr;
            best_set = set;
        }
        if (free_n > 20) break;
    }
    if (best_set < 0) return false;
    // renumber offset bits: chunk bits, other thread bits, register bits
    int newpos[FTK_MAX_TILE_BITS];
    int nt = 0;
    for (int o = 0; o < c; ++o) newpos[o] = nt++;
    for (int o = c; o < b; ++o)
        if (!((best_set >> (o - c)) & 1)) newpos[o] = nt++;
    for (int o = c; o < b; ++o)
        if ((best_set >> (o - c)) & 1) newpos[o] = nt++;
    if (nt != b || (b - le) != tb) return false;
    PassDesc q = pd;
    for (int o = 0; o < b; ++o) q.tile_pos[newpos[o]] = pd.tile_pos[o];
    // bonds with their new offset bits, grouped by thread mask (own group last)
    int tmask[FTK_MAX_PASS_BONDS];
    for (int l = 0; l < nb; ++l) {
        const int bi = newpos[pd.bi[l]], bj = newpos[pd.bj[l]];
        tmask[l] = ((1 << bi) | (1 << bj)) & ((1 << tb) - 1);
    }
    // distinct nonzero masks in first-appearance order, those of z bonds alone
    // before or after the others (the smaller coefficients first: the partial
    // sums are smaller and round less), then 0
    const TypeCoef &tc = pd.tc;
    const bool z_small = tc.anti[2] * tc.anti[2] <= tc.par[0] * tc.par[0] + tc.anti[0] * tc.anti[0];
    int gm[FTK_MAX_PASS_BONDS + 1], ng = 0;
    for (const bool z : {true, false})
        for (int l = 0; l < nb; ++l) {
            if (tmask[l] == 0) continue;
            bool seen = false, only_z = true;
            for (int g = 0; g < ng; ++g) seen |= gm[g] == tmask[l];
            for (int m = 0; m < nb; ++m) only_z &= tmask[m] != tmask[l] || pd.gam[m] == 2;
            if (!seen && only_z == (z == z_small)) gm[ng++] = tmask[l];
        }
    gm[ng++] = 0;
    int w = 0;
    for (int g = 0; g < ng; ++g) {
        for (int l = 0; l < nb; ++l) {
            if (tmask[l] != gm[g]) continue;
            const int bi = newpos[pd.bi[l]], bj = newpos[pd.bj[l]];
            q.bi[w] = (int8_t)bi;
            q.bj[w] = (int8_t)bj;
            q.gam[w] = pd.gam[l];
            q.par_f[w] = pd.tc.par_f[pd.gam[l]];
            q.anti_f[w] = pd.tc.anti_f[pd.gam[l]];
            q.par_lo[w] = pd.tc.par_lo[pd.gam[l]];
            q.anti_lo[w] = pd.tc.anti_lo[pd.gam[l]];
            const int km = ((1 << bi) | (1 << bj)) >> tb;
            int ka = -1, kb = -1;
            for (int a = 0; a < le; ++a)
                if ((km >> a) & 1) { if (ka < 0) ka = a; else kb = a; }
            q.bcase[w] = (int8_t)(ka < 0 ? 0 : kb < 0 ? 1 + ka : 9 + 8 * ka + kb);
            ++w;
        }
        q.grp_tmask[g] = gm[g];
        q.grp_end[g] = w;
    }
    if (w != nb) return false;
    q.n_groups = ng;
    pd = q;
    return true;
}

TileKernel df_kernel(int epi, bool full) {
    switch (epi) {
    case EPI_PLAIN: return full ? hv_df_kernel<EPI_PLAIN, 9> : hv_df_kernel<EPI_PLAIN, 0>;
    case EPI_COCG: return full ? hv_df_kernel<EPI_COCG, 9> : hv_df_kernel<EPI_COCG, 0>;
    default: return nullptr;
    }
}

}  // namespace ftk

// The tiled FP64 H.V pass in 64-bit fixed point.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM but 64 integer additions:
// with two DFMA per bond and amplitude the product ran at the FP64 pipe's rate
// (24 sites, one vector: 2417 us, 0.82 of the pipe, HBM below 10 %). Here the
// FP64 pipe sees only the epilogue. The Hamiltonian has two couplings, so
//   H v = (K/4) A + (J/4) B,
// and A and B are sums of amplitudes of v with small integer coefficients: a
// bond adds its partner p as
//   x: A += p,          B += 2 p if the spins are antiparallel
//   y: A += +p or -p (antiparallel or parallel), B += 2 p if antiparallel
//   z:                  B += 2 p if antiparallel
// and the diagonal adds c_z v to A and (c_xy + c_z) v to B (c: parallel minus
// antiparallel bonds). The amplitudes of a vector are converted to 64-bit
// integers with one common exponent, the sums are exact, and each pass ends in
// two fixed-point multiplications by K/4 and J/4; the partial product between
// passes is the 64-bit integer result, converted to double in the last one.
//
// Accuracy: the quantum q is 2^-(53 + lsh) of 2^(e0 + 1), the power of two above
// the vector's largest component (lsh: 5 with up to 10 bonds in a pass, 4 up to
// 21, 3 up to 42), the sums add no rounding, and a component far below the largest
// has only the digits above q. An output is as good as that of a chain of
// multiply-adds only if its own terms are large against q, and outputs differ: a
// vector may hold blocks of H, or single neighbourhoods, of tiny components. So
// fix_range_kernel measures before each product, for every output and for real and
// imaginary parts apart, a lower bound of the sum of its terms' sizes, and a vector
// is admitted where the fixed-point error bound stays at every output within that
// of the chain, (bonds + 4) 2^-53 of the sum (fix_plan). Any other vector (zeros or
// tiny blocks, very wide ranges, extreme exponents, infinities, NaN) takes the
// floating-point pass (hv_tile_body), inside the same launches. (Admission by the
// mean distance of the exponents from the largest let blocks of tiny components
// come out as 0.)
//
// Measured, relative to the norm of the product, against double-double sums, random
// vectors, typical states and residuals at 18 to 24 sites: 6.0e-17 to 1.3e-16; the
// chain of multiply-adds 8.6e-17 to 1.4e-16. At the worst component of any of them 3.1
// 2^-53 of its terms; the chain 3.4, admission by the mean exponent 7.9.
//
// What bounds it now: the issue slots and the integer pipe (24 sites, three
// passes: 208, 226 and 246 us, 61-68 % of the issue slots and 48-55 % of the ALU;
// with the measuring launch 753 us per product for 2412; a vector that is not
// admitted 2362; 18 sites, four vectors: 68 for 166, not admitted 173).
//
// Layout and items as in ftk_hv_tile.cuh (1024 threads of 4 amplitudes: 32 warps
// hide the latencies that 16 warps of 8 or 8 of 16 did not). The y bonds come
// first, so that their A -= p plus a doubled D turns into A += +-p by one
// addition per amplitude. Shared memory: the next tile's doubles (cp.async),
// the integers of the current one, and the next partial products, 64 KB each.
#include <cuda_bf16.h>

#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_hv_tile.cuh"
#include "ftk_kernels.h"
#include "ftk_plan.h"

#include <algorithm>
#include <math.h>
#include <string.h>
#include <type_traits>

namespace ftk {

// ---------------------------------------------------------------- measuring
// Largest exponent of a vector's components and the smallest of its outputs'
// sums of term sizes, over the x and y bonds inside tiles of 2^13 or 2^14 amplitudes
// (12 to 14 bonds on the honeycomb clusters; a term left out only lowers the bound).
// Grid (split x persistent CTAs, columns): the outputs of a tile are shared by
// split CTAs that all load it. A tile is held as bf16 sizes (rounded down, so that
// the sums stay lower bounds; FixCoef::need holds the additions' rounding), four
// neighbouring amplitudes in 16 bytes. Sizes below the float range count as 0,
// which refuses.
// What bounds it: at 24 sites the read (50 us of 75) and, after it, the shared reads
// of 4 bytes a bond and amplitude (128 bytes a cycle and SM); below 20 sites one
// tile's time, which split shortens.
constexpr int kRangeThreads = 1024, kRangeCtas = 2, kRangeE = (1 << (kRangeBits - 2)) / kRangeThreads;   // items a thread
// the bf16 bits of a double's size, from its upper word (right below 2^128)
__device__ __forceinline__ int bf16_size(int hi) { return max((int)((unsigned)hi << 1 >> 14) - (896 << 7), 0); }
__device__ __forceinline__ __nv_bfloat162 bf16x2(uint32_t u) { return *reinterpret_cast<__nv_bfloat162 *>(&u); }

__global__ void __launch_bounds__(kRangeThreads, kRangeCtas)
fix_range_kernel(const double2 *__restrict__ in, long long ld, const __grid_constant__ RangePlan rp, FixRange *range,
                 FixRange *other, int split, const int *all_done, const CocgSeed *col_seed) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t odd_k[kRangeE], ofs_k[4 * kRangeE], s_low;
    __shared__ int s_em;
    launch_dependents();
    const int t = threadIdx.x, T = blockDim.x, tb = 31 - __clz(T), n_k = 1 << (rp.bits - 2 - tb);
    // offset of the thread's first amplitude in a tile, and the parities of its item
    // bits with the bonds' masks; both for the bits above the thread's
    uint32_t ofs = 0, odd = 0;
    for (int q = 0; q < tb; ++q)
        if ((t >> q) & 1) ofs |= 1u << rp.pos[q];
    for (int q = 0; q < kRangeBonds; ++q) odd |= (uint32_t)(__popc(t * 16 & rp.mask[q]) & 1) << q;
    if (t < 4 * n_k) {
        uint32_t o = 0, p = 0;
        for (int q = tb; q < rp.bits; ++q)
            if ((t << tb >> q) & 1) o |= 1u << rp.pos[q];
        ofs_k[t] = o;
        if (t < n_k) {
            for (int q = 0; q < kRangeBonds; ++q) p |= (uint32_t)(__popc((t << tb) * 16 & rp.mask[q]) & 1) << q;
            odd_k[t] = p;
        }
    }
    if (t == 0) { s_low = 0xffffffffu; s_em = 0; }
    wait_previous();
    if (other && blockIdx.x == 0 && blockIdx.y == 0 && t < FTK_MAX_RHS) other[t] = FixRange{0, 0};
    if (all_done && *all_done) return;
    const int j = blockIdx.y;
    if (col_seed && col_seed[j].done != 0) return;
    in += (size_t)j * ld + ofs;
    const __nv_bfloat162 par = bf16x2(rp.par), anti = bf16x2(rp.anti);
    __nv_bfloat162 low = bf16x2(0x7f807f80u);
    int em = 0;
    const int per = max(n_k / split, 1), k0 = (int)(blockIdx.x % split) * per;   // the CTA's items
    for (uint32_t tau = blockIdx.x / split; tau < 1u << rp.n_free; tau += gridDim.x / split) {
        uint32_t base = 0;
        for (int q = 0; q < rp.n_free; ++q)
            if ((tau >> q) & 1) base |= 1u << rp.free_pos[q];
        __syncthreads();   // the previous tile is read
        const double2 *v = in + base;
#pragma unroll 8
        for (int k = 0; k < 4 * n_k; ++k) {
            const double2 a = v[ofs_k[k]];
            const int x = bf16_size(__double2hiint(a.x)), y = bf16_size(__double2hiint(a.y));
            *reinterpret_cast<uint32_t *>(smem_raw + 4 * (t + k * T)) = __byte_perm(x, y, 0x5410);
            em = max(em, max(x, y));
        }
        __syncthreads();
        for (int k = k0; k < k0 + per; k += 2) {   // two items at a time (twice the same if there is one)
            const int k1 = min(k + 1, k0 + per - 1);
            const uint32_t at[2] = {16u * (t + k * T), 16u * (t + k1 * T)};
            const uint32_t w[2] = {odd ^ odd_k[k], odd ^ odd_k[k1]};
            __nv_bfloat162 s[2][4];
#pragma unroll
            for (int x = 0; x < 8; ++x) s[x >> 2][x & 3] = bf16x2(0);
            // the partner of word x of an item is word x ^ KIND of the partner item,
            // and its parity the items' with that of x & KIND; unrolled, so that masks
            // and parity bits are operands of one instruction each
            const auto walk = [&](auto kind) {
                constexpr int KIND = decltype(kind)::value;
#pragma unroll
                for (int u = 0; u < range_slots(KIND); ++u) {
                    if (u >= rp.n[KIND]) break;
                    constexpr int q0 = range_slot(KIND);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const uint4 p4 = *reinterpret_cast<const uint4 *>(smem_raw + (at[i] ^ rp.mask[q0 + u]));
                        const uint32_t p[4] = {p4.x, p4.y, p4.z, p4.w};
                        const bool o = (w[i] & (1u << (q0 + u))) != 0;
                        const __nv_bfloat162 c = o ? anti : par, f = o ? par : anti;
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            s[i][x] = __hfma2(((x & KIND & 1) != 0) != ((x & KIND & 2) != 0) ? f : c,
                                              bf16x2(p[x ^ KIND]), s[i][x]);
                    }
                }
            };
            walk(std::integral_constant<int, 0>());
            walk(std::integral_constant<int, 1>());
            walk(std::integral_constant<int, 2>());
            walk(std::integral_constant<int, 3>());
#pragma unroll
            for (int x = 0; x < 8; ++x) low = __hmin2(low, s[x >> 2][x & 3]);
        }
    }
    // integer reductions: order-independent (positive floats order as integers)
    const uint32_t lw = *reinterpret_cast<const uint32_t *>(&low);
    em = __reduce_max_sync(0xffffffffu, em);
    const uint32_t lmin = __reduce_min_sync(0xffffffffu, min(lw & 0xffffu, lw >> 16));
    if ((t & 31) == 0) {
        atomicMax(&s_em, em);
        atomicMin(&s_low, lmin);
    }
    __syncthreads();
    if (t == 0) {
        atomicMax(&range[j].emax, (s_em >> 7) + 896);
        atomicMax(&range[j].low, ~s_low);
    }
}
// Whether a column takes fixed point: its largest component well inside the float
// range (no infinity or NaN), and every output's sum as large as need asks.
__device__ __forceinline__ bool fix_admits(const FixRange &r, float need) {
    return r.emax >= 920 && r.emax <= 1120 &&
           __uint_as_float(~r.low << 16) >= need * __uint_as_float((uint32_t)(r.emax + 1 - 896) << 23);
}

// ---------------------------------------------------------------- arithmetic
// v as an integer: its 53-bit significand shifted to the common exponent e0
// (|v| < 2^(e0 + 1 - 1023) maps to at most 2^(53 + lsh)), rounded to nearest.
__device__ __forceinline__ long long to_fixed(double v, int e0, int lsh) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int sh = min(e0 - (int)((hi >> 20) & 0x7ffu), 63);   // zero: shifted out
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << (lsh + 1);
    const long long s = (long long)((m >> sh) + 1) >> 1;
    return (int)hi < 0 ? -s : s;
}
// (K/4) A + (J/4) B in units of the result's quantum, from signed 32-bit digits
// (the lowest digit products are dropped: with the roundings of the others less
// than 1 + (kl + jl) 2^-31 quanta, and one more for a shift)
__device__ __forceinline__ long long fix_combine(long long A, long long B, const FixCoef &f) {
    const int Al = (int)A, Bl = (int)B;
    const int Ah = (int)(A >> 32) - (Al >> 31), Bh = (int)(B >> 32) - (Bl >> 31);
    const long long t1 = (long long)Ah * f.kh + (long long)Bh * f.jh;
    const long long t2 = (long long)Ah * f.kl + (long long)Bh * f.jl + (1ll << 29);
    const long long t3 = (long long)Al * f.kh + (long long)Bl * f.jh + (1ll << 31);
    const long long r = t1 + (t2 >> 30) + (t3 >> 32);
    return f.sr ? r >> f.sr : r;
}
__device__ __forceinline__ double fix_to_double(long long r, int ex) {
    const double d = __ll2double_rn(r);
    return r == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (ex << 20), __double2loint(d));
}

// A += z v, B += a v for small z and a, from v's signed 32-bit digits
__device__ __forceinline__ void mac_small(long long &A, long long &B, long long v, int z, int a) {
    const int vl = (int)v, vh = (int)(v >> 32) - (vl >> 31);
    A += (long long)vl * z;
    B += (long long)vl * a;
    A += (long long)((unsigned long long)(unsigned)(vh * z) << 32);
    B += (long long)((unsigned long long)(unsigned)(vh * a) << 32);
}

// The bonds of one type (0 x, 1 y, 2 z): A += p (x) or -= p (y), D += p where
// the spins are antiparallel. The two sides of the branch on the parity touch
// complementary items; a warp whose lanes agree takes one of them.
template <int TYPE, int KM>
__device__ __forceinline__ void class_fix(longlong2 (&A)[kTileE], longlong2 (&D)[kTileE], const char *F, int at, int step, BondWalk<false> &bw) {
    bw.template run<TYPE, 0, KM, longlong2>(F, at, step, [&](const longlong2(&p)[kTileE], bool odd) {
#pragma unroll
        for (int k = 0; k < kTileE; ++k) {
            if (TYPE == 0) { A[k].x += p[k].x; A[k].y += p[k].y; }
            if (TYPE == 1) { A[k].x -= p[k].x; A[k].y -= p[k].y; }
        }
        if (odd) {
#pragma unroll
            for (int k = 0; k < kTileE; ++k)
                if (!odd_in(k, KM)) { D[k].x += p[k].x; D[k].y += p[k].y; }
        } else if (KM != 0) {
#pragma unroll
            for (int k = 0; k < kTileE; ++k)
                if (odd_in(k, KM)) { D[k].x += p[k].x; D[k].y += p[k].y; }
        }
    });
}
template <int TYPE>
__device__ __forceinline__ void bonds_fix(longlong2 (&A)[kTileE], longlong2 (&D)[kTileE], const char *F, int at, int step, BondWalk<false> &bw) {
    class_fix<TYPE, 0>(A, D, F, at, step, bw);
    class_fix<TYPE, 1>(A, D, F, at, step, bw);
    class_fix<TYPE, 2>(A, D, F, at, step, bw);
    class_fix<TYPE, 3>(A, D, F, at, step, bw);
}

// ---------------------------------------------------------------- the pass
// Returns false, having done nothing, for a vector that is not admitted.
template <int EPI, int TB>
__device__ __forceinline__ bool hv_fix_body(const double2 *__restrict__ in, double2 *out, const PassDesc &pd,
                                            const EpiArgs &ea0, long long ld) {
    constexpr int E = kTileE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tb = TB > 0 ? TB : pd.tile_bits - 2;
    const int T = 1 << tb, tile_n = T * E;
    const int t = threadIdx.x;
    double2 *raw = reinterpret_cast<double2 *>(smem_raw);
    longlong2 *F = reinterpret_cast<longlong2 *>(raw + tile_n);
    double2 *pb = reinterpret_cast<double2 *>(F + tile_n);
    double *red = reinterpret_cast<double *>(pb + tile_n);
    const TileWalk<0> w(pd, t, tb);
    // diagonal counts of the thread's amplitudes, one signed byte each
    uint32_t cz, ca;
    const unsigned long long odd = odd_bonds(pd, t);
    diag_counts(pd, odd, false, ca, cz);
    ca = __vadd4(ca, cz);
    wait_previous();
    EpiArgs ea;
    if (!hv_column(ea0, ea, ld)) return true;
    if (!fix_admits(ea0.range[blockIdx.y], pd.fx.need)) return false;
    const int e0 = ea0.range[blockIdx.y].emax;
    in += (size_t)blockIdx.y * ld;
    out += (size_t)blockIdx.y * ld;
    const HvEpilogue<double, EPI> epi(ea);
    constexpr int ND = EPI == EPI_PLAIN ? 1 : 2;
    Acc<double> dot[ND];
    const bool first = pd.first != 0, last = pd.last != 0;
    const int lsh = pd.fx.lsh;
    const int ex = e0 + pd.fx.ex;   // exponent of the result's quantum

    auto issue = [&](const double2 *src, uint32_t tofs, double2 *buf) {
        const double2 *g = src + tofs;
#pragma unroll
        for (int k = 0; k < E; ++k) cp_async16(buf + t + T * k, g + w.e[k]);
        cp_async_commit();
    };
    // Pipeline (commit order): v_0 [p_0] | per tile i: v_{i+1} once tile i is
    // converted, then p_{i+1} after its epilogue. A thread copies, converts
    // and adds its own elements only; the integers alone are shared.
    const uint32_t n_tiles = 1u << pd.n_free;
    uint32_t tau = blockIdx.x;
    uint32_t tofs = tau < n_tiles ? w.base(pd, tau) : 0;
    if (tau < n_tiles) {
        issue(in, tofs, raw);
        if (!first) issue(out, tofs, pb);
    }
    for (; tau < n_tiles; tau += gridDim.x) {
        const bool more = tau + gridDim.x < n_tiles;
        const uint32_t tofs_n = more ? w.next(tofs) : 0;
        if (first) cp_async_wait<0>(); else cp_async_wait<1>();
        __syncthreads();   // the previous tile's integers are read
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const double2 v = raw[t + T * k];
            F[t + T * k] = make_longlong2(to_fixed(v.x, e0, lsh), to_fixed(v.y, e0, lsh));
        }
        if (more) issue(in, tofs_n, raw);
        __syncthreads();
        longlong2 A[E], D[E];
#pragma unroll
        for (int k = 0; k < E; ++k) { A[k] = make_longlong2(0, 0); D[k] = make_longlong2(0, 0); }
        const char *Fb = reinterpret_cast<const char *>(F);
        BondWalk<false> bw(pd, odd);
        bonds_fix<1>(A, D, Fb, t * 16, T * 16, bw);
        // A = sum of -p, D of the antiparallel p: together +p and -p
#pragma unroll
        for (int k = 0; k < E; ++k) { A[k].x += 2 * D[k].x; A[k].y += 2 * D[k].y; }
        bonds_fix<0>(A, D, Fb, t * 16, T * 16, bw);
        bonds_fix<2>(A, D, Fb, t * 16, T * 16, bw);
        // diagonal, products
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const int z = byte_of(cz, k), a = byte_of(ca, k);
            D[k].x += D[k].x;
            D[k].y += D[k].y;
            const longlong2 p = F[t + T * k];
            mac_small(A[k].x, D[k].x, p.x, z, a);
            mac_small(A[k].y, D[k].y, p.y, z, a);
        }
        double2 v[E];   // the epilogue's exact input
        if (EPI != EPI_PLAIN && last) {
#pragma unroll
            for (int k = 0; k < E; ++k) v[k] = in[tofs + w.e[k]];
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            A[k].x = fix_combine(A[k].x, D[k].x, pd.fx);
            A[k].y = fix_combine(A[k].y, D[k].y, pd.fx);
        }
        if (!first) {   // partial product of the earlier passes (own elements)
            if (more) cp_async_wait<1>(); else cp_async_wait<0>();
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const longlong2 r = *reinterpret_cast<const longlong2 *>(pb + t + T * k);
                A[k].x += r.x;
                A[k].y += r.y;
            }
            if (more) issue(out, tofs_n, pb);
        }
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const uint32_t i = tofs + w.e[k];
            if (!last) {
                reinterpret_cast<longlong2 *>(out)[i] = A[k];
            } else {
                const double2 hv = make_double2(fix_to_double(A[k].x, ex), fix_to_double(A[k].y, ex));
                epi.apply(ea, i, v[k], hv, out + i, dot);
            }
        }
        tofs = tofs_n;
    }
    cp_async_wait<0>();
    if (EPI == EPI_PLAIN || !last) return true;
    double d[ND];
#pragma unroll
    for (int q = 0; q < ND; ++q) d[q] = dot[q].get();
    block_reduce<ND>(d, red);
    if (t < ND) ea.partials[(size_t)blockIdx.x * ND + t] = red[t];
    if (!last_block_reduce<ND>(ea.partials, ea.counter, ea.result, red)) return true;
    if (EPI == EPI_TPQ && t == 0) tpq_statistics(ea, ea.result);
    return true;
}

// Grid (tiles, columns); column j at j ld.
template <int EPI, int TB>
__global__ void __launch_bounds__(kTileThreads, 1)
hv_fix_kernel(const double2 *__restrict__ in, double2 *out, long long ld, const __grid_constant__ PassDesc pd,
              const __grid_constant__ EpiArgs ea0) {
    launch_dependents();
    if (!ea0.range) {
        hv_tile_body<ItemF64, EPI, TB>(in, out, pd, ea0, ld);
        return;
    }
    if (!hv_fix_body<EPI, TB>(in, out, pd, ea0, ld)) hv_tile_body<ItemF64, EPI, TB>(in, out, pd, ea0, ld);
}

// ===================================================================== host
// The measuring launch's tile: the lowest sites (contiguous runs of 128 bytes),
// and greedily the sites with the most x and y bonds into it; its bonds, by which
// of the sites 0 and 1 (the bits inside an item) they flip. Returns their number.
static int range_plan(int n, const PlanBond *bonds, int nb, int bits, RangePlan *rp) {
    RangePlan r{};
    r.bits = std::min(n, bits);
    r.n_free = n - r.bits;
    int at[FTK_MAX_SITES];   // offset bit of a site, -1: not in the tile
    std::fill(at, at + FTK_MAX_SITES, -1);
    for (int w = 0; w < r.bits; ++w) {
        int best = w, most = -1;
        if (w >= 3) {
            int score[FTK_MAX_SITES] = {};
            for (int q = 0; q < nb; ++q) {
                if (bonds[q].g == 2) continue;
                score[bonds[q].i] += at[bonds[q].j] >= 0 ? 17 : 1;
                score[bonds[q].j] += at[bonds[q].i] >= 0 ? 17 : 1;
            }
            for (int s = 0; s < n; ++s)
                if (at[s] < 0 && score[s] > most) { most = score[s]; best = s; }
        }
        at[best] = w;
    }
    int f = 0;
    for (int s = 0, w = 0; s < n; ++s) {   // ascending offset bits
        if (at[s] < 0) { r.free_pos[f++] = s; continue; }
        r.pos[w] = s;
        at[s] = w++;
    }
    int total = 0;
    for (int q = 0; q < nb; ++q) {
        const int i = at[bonds[q].i], j = at[bonds[q].j];
        if (bonds[q].g == 2 || i < 0 || j < 0) continue;
        const uint32_t m = (1u << i) | (1u << j);
        const int kind = m & 3;
        if (r.n[kind] == range_slots(kind)) continue;
        r.mask[range_slot(kind) + r.n[kind]++] = (m >> 2) * 16;
        ++total;
    }
    *rp = r;
    return total;
}

// Exponents stay inside the range; and the measured sums count x and y bonds, so
// both of their coefficients must differ from zero, else some state has no such
// term and no vector is admitted.
bool fix_couplings(double K, double J) {
    const double cmax = std::max(fabs(K), fabs(J)) / 4;
    double par, anti;
    bond_coefficients(0, K, J, &par, &anti);
    return cmax > 0x1p-40 && cmax < 0x1p40 && par != 0 && anti != 0;
}

// Coefficients and scales for the passes of one plan, and its measuring launch.
// Sums: a pass of nb bonds adds at most nb amplitudes to A and 3 nb to B (the
// antiparallel ones twice, and the diagonal), which has to stay below 2^63 with
// room for the signed digits. K/4 and J/4 are 61-bit integers at a common exponent
// ec. The result's quantum is 2^(ec + 2 + sr) of the input's; sr keeps the whole
// product (at most sum_b (|off-diagonal| + |diagonal|) max |v|) below 2^62.
// Admission, with q the input's quantum: an output's error is at most q / 2 for each
// unit of its coefficients (at most bound in all), and per pass the roundings of
// fix_combine. need is where that equals (nb + 3) 2^-53 of the sum of its terms'
// sizes; the result's rounding makes it nb + 4, what a chain of multiply-adds may
// lose: one for each bond, the diagonal and the partial product, two for the
// diagonal's coefficient.
bool fix_plan(PassDesc *pd, int np, const PlanBond *bonds, int nb, double K, double J, RangePlan *rp) {
    int most = 1;
    for (int p = 0; p < np; ++p) {
        pd[p].fx = FixCoef{};
        if (!hv_tiled(0, pd[p]) || pd[p].n_bonds > 60) return false;
        most = std::max(most, pd[p].n_bonds);
    }
    if (!fix_couplings(K, J)) return false;
    // tiles of 2^13 if they hold 12 bonds (18 sites, one and four vectors 6.7 and 8.4 us
    // for 8.7 and 11.0; random vectors of up to 2^27 components pass with 12), else of
    // 2^14 (20 sites: 12 bonds for 11)
    if (range_plan(pd[0].n_sites, bonds, nb, kRangeBits - 1, rp) < 12 &&
        range_plan(pd[0].n_sites, bonds, nb, kRangeBits, rp) == 0)
        return false;
    const double cmax = std::max(fabs(K), fabs(J)) / 4;
    double par, anti;
    bond_coefficients(0, K, J, &par, &anti);
    int ec = 0;
    if (frexp(cmax, &ec) == 0.5) --ec;   // cmax <= 2^ec
    double bound = 0;
    for (int q = 0; q < nb; ++q) {
        double p, a;
        bond_coefficients(bonds[q].g, K, J, &p, &a);
        bound += std::max(fabs(p), fabs(a)) + fabs(bonds[q].g == 2 ? (J + K) / 4 : J / 4);
    }
    FixCoef f{};
    while (3.0 * most * ldexp(1.0, 54 + f.lsh) <= 0x1p63 - 0x1p33) ++f.lsh;
    int eb = 0;
    frexp(bound, &eb);        // bound < 2^eb
    f.sr = std::max(0, eb + (53 + f.lsh) - (ec + 2) - 62);
    const long long ki = llrint(ldexp(K / 4, 60 - ec)), ji = llrint(ldexp(J / 4, 60 - ec));
    f.kh = (int)(ki >> 30);
    f.kl = (int)(ki & ((1 << 30) - 1));
    f.jh = (int)(ji >> 30);
    f.jl = (int)(ji & ((1 << 30) - 1));
    f.ex = 1 - 1023 - (53 + f.lsh) + ec + 2 + f.sr;
    // the coefficients' bf16 sizes, rounded down
    auto below = [](double c) -> uint32_t {
        const float x = (float)c;
        uint32_t u;
        memcpy(&u, &x, 4);
        if ((double)x > c && (u & 0xffffu) == 0) --u;   // rounded up to a bf16 number
        u >>= 16;
        return u << 16 | u;
    };
    rp->par = below(fabs(par));
    rp->anti = below(fabs(anti));
    const double combine = 1 + ((double)f.kl + f.jl) * 0x1p-31 + (f.sr > 0);
    const double need = (bound / 2 + np * combine * ldexp(1.0, ec + 2 + f.sr)) / (ldexp(1.0, f.lsh) * (nb + 3));
    f.need = (float)(need * pow(1 + 0x1p-8, rp->n[0] + rp->n[1] + rp->n[2] + rp->n[3] + 2));   // bf16 additions, the float product
    for (int p = 0; p < np; ++p) pd[p].fx = f;
    return true;
}

cudaError_t fix_attributes() {
    return cudaFuncSetAttribute(fix_range_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 << kRangeBits);
}
cudaError_t launch_fix_range(const void *in, int n, int B, FixRange *range, FixRange *other, const RangePlan &rp,
                             const EpiArgs &ea, int n_sm, cudaStream_t st) {
    const int items = 1 << (rp.bits - 2), threads = std::min(kRangeThreads, items);
    const int tiles = 1 << rp.n_free, resident = kRangeCtas * n_sm;
    int split = 1;
    while (split < items / threads && 2 * split * tiles * B <= n_sm) split *= 2;   // while SMs are idle
    const int grid = std::min(tiles, std::max(1, resident / (split * B))) * split;
    return launch_chained(fix_range_kernel, dim3(grid, B), threads, (size_t)items * 16, st,
                          static_cast<const double2 *>(in), 1LL << n, rp, range, other, split, ea.all_done, ea.col_seed);
}

template <int TB>
static FixKernel fix_kernel_tb(int epi) {
    switch (epi) {
    case EPI_PLAIN: return hv_fix_kernel<EPI_PLAIN, TB>;
    case EPI_TPQ: return hv_fix_kernel<EPI_TPQ, TB>;
    case EPI_COCG: return hv_fix_kernel<EPI_COCG, TB>;
    case EPI_TAYLOR: return hv_fix_kernel<EPI_TAYLOR, TB>;
    default: return nullptr;
    }
}
FixKernel fix_kernel(int epi, bool full) { return full ? fix_kernel_tb<10>(epi) : fix_kernel_tb<0>(epi); }

}  // namespace ftk

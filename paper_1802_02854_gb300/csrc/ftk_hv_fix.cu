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
// Accuracy: the quantum is 2^-58 of the vector's largest component, so a term's
// rounding is below that of the DFMA chain for every component above 2^-5 of
// the largest, and the sums add none. fix_range_kernel measures that before
// each product: the exponents of all nonzero components must lie within 4.5
// bits of the largest on average (3.4 for a Gaussian vector at 24 sites), with
// no infinity, NaN or extreme exponent. Any other vector takes the
// floating-point pass (hv_tile_body), inside the same launches. Relative error
// against a double-double product, Gaussian vectors: 6e-17, with the DFMA chain
// 1.2e-16.
//
// What bounds it now: the issue slots and the integer pipe (24 sites, three
// passes: 203, 221 and 243 us, 61-68 % of the issue slots and 48-55 % of the ALU;
// 709 us per product for 2417; a vector of wide range 2337).
//
// Layout and items as in ftk_hv_tile.cuh (1024 threads of 4 amplitudes: 32 warps
// hide the latencies that 16 warps of 8 or 8 of 16 did not). The y bonds come
// first, so that their A -= p plus a doubled D turns into A += +-p by one
// addition per amplitude. Shared memory: the next tile's doubles (cp.async),
// the integers of the current one, and the next partial products, 64 KB each.
#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_hv_tile.cuh"
#include "ftk_kernels.h"
#include "ftk_plan.h"

#include <algorithm>
#include <math.h>

namespace ftk {

// ---------------------------------------------------------------- exponents
// Exponents of a vector's components (grid (blocks, columns)).
__global__ void __launch_bounds__(256) fix_range_kernel(const double2 *__restrict__ in, uint64_t dim, FixRange *range,
                                                        const int *all_done, const CocgSeed *col_seed) {
    launch_dependents();
    wait_previous();
    if (all_done && *all_done) return;
    const int j = blockIdx.y;
    if (col_seed && col_seed[j].done != 0) return;
    const double2 *v = in + (size_t)j * dim;
    RangeAcc acc;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; x + 3 * stride < dim; x += 4 * stride) {
        const double2 a = v[x], b = v[x + stride], c = v[x + 2 * stride], d = v[x + 3 * stride];
        acc.add_fp64(a); acc.add_fp64(b); acc.add_fp64(c); acc.add_fp64(d);
    }
    for (; x < dim; x += stride) acc.add_fp64(v[x]);
    acc.publish_fp64(range + j, gridDim.x);
}

// ---------------------------------------------------------------- arithmetic
// v as an integer: its 53-bit significand shifted to the common exponent e0
// (|v| < 2^(e0 + 1 - 1023) maps below 2^(53 + lsh)), rounded toward zero.
__device__ __forceinline__ long long to_fixed(double v, int e0, int lsh) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int sh = min(e0 - (int)((hi >> 20) & 0x7ffu), 63);   // zero: shifted out
    const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << lsh;
    const long long s = (long long)(m >> sh);
    return (int)hi < 0 ? -s : s;
}
// (K/4) A + (J/4) B in units of the result's quantum, from signed 32-bit digits
// (the lowest digit product is below one quantum and dropped)
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
// Returns false, having done nothing, for a vector of wide range.
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
    if (ea0.range[blockIdx.y].wide) return false;
    const int e0 = ea0.range[blockIdx.y].e0;
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
// Coefficients and scales for the passes of one plan. Sums: with |F| < 2^fb and
// at most nb bonds in a pass, |A| <= nb 2^fb and |B| <= 2 nb 2^fb stay below
// 2^62. K/4 and J/4 are 61-bit integers at a common exponent ec. The result's
// quantum is 2^(ec + 2 + sr) of the input's; sr keeps the whole product (at
// most sum_b (|off-diagonal| + |diagonal|) max |v|) below 2^62.
bool fix_plan(PassDesc *pd, int np, const PlanBond *bonds, int nb, double K, double J) {
    int most = 1;
    for (int p = 0; p < np; ++p) {
        pd[p].fx = FixCoef{};
        if (!hv_tiled(0, pd[p]) || pd[p].n_bonds > 60) return false;
        most = std::max(most, pd[p].n_bonds);
    }
    const double cmax = std::max(fabs(K), fabs(J)) / 4;
    if (!(cmax > 0x1p-40) || !(cmax < 0x1p40)) return false;   // exponents stay inside the range
    int ec = 0;
    if (frexp(cmax, &ec) == 0.5) --ec;   // cmax <= 2^ec
    double bound = 0;
    for (int q = 0; q < nb; ++q) {
        double par, anti;
        bond_coefficients(bonds[q].g, K, J, &par, &anti);
        bound += std::max(fabs(par), fabs(anti)) + fabs(bonds[q].g == 2 ? (J + K) / 4 : J / 4);
    }
    int lg = 0;
    while ((1 << lg) < most) ++lg;
    const int fb = 62 - lg;   // 2 most 2^fb <= 2^63 / ... : |B| < 2^63, its signed upper digit below 2^31
    int eb = 0;
    frexp(bound, &eb);        // bound < 2^eb
    FixCoef f{};
    f.lsh = fb - 1 - 53;      // one bit of room for the signed digits
    f.sr = std::max(0, eb + (fb - 1) - (ec + 2) - 62);
    const long long ki = llrint(ldexp(K / 4, 60 - ec)), ji = llrint(ldexp(J / 4, 60 - ec));
    f.kh = (int)(ki >> 30);
    f.kl = (int)(ki & ((1 << 30) - 1));
    f.jh = (int)(ji >> 30);
    f.jl = (int)(ji & ((1 << 30) - 1));
    f.ex = 1 - 1023 - (fb - 1) + ec + 2 + f.sr;
    if (f.lsh < 0) return false;
    for (int p = 0; p < np; ++p) pd[p].fx = f;
    return true;
}

cudaError_t launch_fix_range(const void *in, uint64_t dim, int B, FixRange *range, const EpiArgs &ea, int n_sm,
                             cudaStream_t st) {
    const uint64_t want = (dim + 1023) / 1024;
    const uint64_t cap = std::max<uint64_t>(1, (uint64_t)8 * n_sm / B);
    const dim3 grid((unsigned)std::min(want, cap), B);
    return launch_chained(fix_range_kernel, grid, 256, 0, st, static_cast<const double2 *>(in), dim, range, ea.all_done,
                          ea.col_seed);
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

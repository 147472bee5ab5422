// One tiled pass of the matrix-free Kitaev-Heisenberg H.V on sm_103a (Sec.
// IV.A: every method of the paper is costed in these products), with the
// epilogues of the mTPQ step (Appendix A) and the COCG mu = r^T H r dot.
//
// Data: right-hand sides stored one after the other, element (x, j) at
// j 2^N + x. A CTA owns tiles of 2^b amplitudes: the offset bits of a tile are
// the global bits pd.tile_pos[], the other bits (pd.free_pos[]) are fixed by
// the tile index; the low offset bits are global bits 0..chunk-1, so a tile is
// a set of >= 256-byte contiguous runs. Persistent CTAs loop over tiles; the
// next tile is fetched with cp.async into the second of two shared-memory
// buffers while the current one is processed, and the partial product of
// earlier passes is prefetched into a third.
//
// Items: shared memory holds 16-byte items, an FP64 amplitude or two neighbouring
// FP32 ones (offset bit 0). A thread owns the items
// t + T k, k < 4, of at most 4096 (T = 1024), with their sums in registers. A
// bond's partner item is the item's byte offset with the bond's two bits
// flipped: one exclusive or for the thread's part, while the register part (the
// top two item bits, two sites with few bonds) only permutes the four reads. The
// bonds are sorted into classes by type and register part, each a loop of its
// own with everything but the mask known at compile time, and the parity of the
// thread's bits, which chooses the coefficient (parallel or antiparallel spins),
// is kept as one bit per bond, since it is the same for every tile.
//
// Why this layout: with 512 threads of 8 or 16 amplitudes, the partners of
// bonds with the same thread part read once and a 16-way dispatch over the
// register part, the FP32 passes issued 78-91 instructions per amplitude at 41-44 %
// of the issue slots, 16 warps a SM. Here
// 32 warps hide the latencies and a bond costs a dozen instructions per thread
// beside its reads and terms. FP32, 24 sites: 282 -> 217 us a product (three
// passes, 72-87 us, the shared-memory pipe 63-67 % busy); 26 sites 988 -> 853.
#pragma once
#include "ftk_common.cuh"
#include "ftk_device.cuh"
#include "ftk_kernels.h"

namespace ftk {

constexpr int kTileE = 4;          // items per thread
constexpr int kTileThreads = 1024;

// ------------------------------------------------------------ async copies
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// ------------------------------------------------------------ tile geometry
// Element offsets of a thread's items from the tile base, and the tile bases:
// the bits of the tile index deposited at the free sites. Successive tiles of
// a CTA are gridDim.x apart; their bases follow by a masked addition (the bits
// outside the mask set to 1 carry across them). 32 bits: a column has at most
// 2^30 elements. W: amplitudes per item (log2 in SH).
template <int SH>
struct TileWalk {
    uint32_t e[kTileE];
    uint32_t free_mask, step;
    __device__ static uint32_t base(const PassDesc &pd, uint32_t tau) {
        uint32_t v = 0;
        for (int q = 0; q < pd.n_free; ++q)
            if ((tau >> q) & 1) v |= 1u << pd.free_pos[q];
        return v;
    }
    __device__ TileWalk(const PassDesc &pd, int t, int tb) {
        uint32_t st = 0;
        for (int q = 0; q < tb; ++q)
            if ((t >> q) & 1) st |= 1u << pd.tile_pos[q + SH];
        const uint32_t k0 = 1u << pd.tile_pos[tb + SH], k1 = 1u << pd.tile_pos[tb + 1 + SH];
#pragma unroll
        for (int k = 0; k < kTileE; ++k) e[k] = st + ((k & 1) ? k0 : 0u) + ((k & 2) ? k1 : 0u);
        free_mask = 0;
        for (int q = 0; q < pd.n_free; ++q) free_mask |= 1u << pd.free_pos[q];
        step = base(pd, gridDim.x);
    }
    __device__ __forceinline__ uint32_t next(uint32_t ofs) const { return ((ofs | ~free_mask) + step) & free_mask; }
};
// Bond q of the pass: fdesc[q] holds 16 times the thread part of its item mask
// (low half), the register part (two bits from 16) and, in bit 31, whether it
// flips offset bit 0 of an FP32 pair. The bonds are sorted by class (type, swap,
// register part KM); classes has a bit per class that is not empty, f_end its
// end. FP32 (z_first): z bonds before y before x, since with the small
// coefficients first the sums round less; FP64: y before x before z (ftk_hv_fix.cu).
__host__ __device__ constexpr int bond_class(bool z_first, int type, int swap, int km) {
    return 8 * ((z_first ? 2 - type : type == 1 ? 0 : type == 0 ? 1 : 2)) + 4 * swap + km;
}
// One bit per bond: odd parity of the thread's offset bits with its mask.
__device__ __forceinline__ unsigned long long odd_bonds(const PassDesc &pd, int t) {
    unsigned long long v = 0;
    for (int q = 0; q < pd.n_bonds; ++q)
        v |= (unsigned long long)(__popc((t * 16) & (int)(pd.fdesc[q] & 0xffffu)) & 1) << q;
    return v;
}
// Walk over the bonds in their order: class by class, f(p, odd) for each bond of
// a class, p[k] the partner of item k. at: byte offset of the thread's first
// item, step: bytes between its items. An empty class costs a test of its bit
// (a loop with bounds of its own for each of up to 24 classes took 72
// instructions per FP32 pair).
template <bool ZF>
struct BondWalk {
    int q;
    unsigned long long odd;   // shifted along: bit 0 belongs to bond q
    uint32_t classes;
    const PassDesc &pd;
    __device__ BondWalk(const PassDesc &p, unsigned long long o, int start = 0)
        : q(start), odd(start < 64 ? o >> start : 0), classes(p.classes), pd(p) {}
    template <int TYPE, int SWAP, int KM, class P, class F>
    __device__ __forceinline__ void run(const char *buf, int at, int step, F f) {
        constexpr int c = bond_class(ZF, TYPE, SWAP, KM);
        if (!(classes & (1u << c))) return;
        const int end = pd.f_end[c];
#pragma unroll 1
        do {
            const char *src = buf + (at ^ (int)(pd.fdesc[q] & 0xffffu) * (int)sizeof(P) / 16);
            P p[kTileE];
#pragma unroll
            for (int k = 0; k < kTileE; ++k) p[k ^ KM] = *reinterpret_cast<const P *>(src + k * step);
            f(p, ((unsigned)odd & 1u) != 0);
            odd >>= 1;
        } while (++q < end);
    }
};
__device__ __forceinline__ constexpr bool odd_in(int k, int km) { return ((k & km & 1) ^ ((k & km) >> 1)) != 0; }

// (parallel - antiparallel) bonds of the pass at the thread's four items, one
// signed byte each: c0 of the x and y bonds, c1 of the z bonds. swapped: of the
// second halves of FP32 pairs, where a bond with offset bit 0 has the other
// sign.
__device__ __forceinline__ void diag_counts(const PassDesc &pd, unsigned long long odd, bool swapped, uint32_t &c0,
                                            uint32_t &c1) {
    c0 = c1 = 0;
    for (int l = 0; l < pd.n_bonds; ++l, odd >>= 1) {
        const uint32_t d = pd.fdesc[l];
        const int km = (d >> 16) & 3;
        // +1 or -1 by the parity of k & km, k = 0..3
        uint32_t v = km == 0 ? 0x01010101u : km == 1 ? 0xff01ff01u : km == 2 ? 0xffff0101u : 0x01ffff01u;
        if (((odd & 1) != 0) != (swapped && (d >> 31))) v = __vneg4(v);
        if (pd.gam[l] != 2) c0 = __vadd4(c0, v);
        else c1 = __vadd4(c1, v);
    }
}
__device__ __forceinline__ int byte_of(uint32_t c, int k) { return (signed char)(c >> (8 * k)); }

// ------------------------------------------------------------ item types
// amp: element type in memory; SH: log2 of the amplitudes per item; coef: a
// term's coefficient; acc: an item's sums.
struct ItemF64 {
    typedef double2 amp;
    typedef double2 item;
    typedef double coef;
    typedef double diag;
    typedef double dot;
    static constexpr int SH = 0;
    double2 s = {0.0, 0.0};
    __device__ static coef par(const PassDesc &p, int g) { return p.tc.par[g]; }
    __device__ static coef anti(const PassDesc &p, int g) { return p.tc.anti[g]; }
    __device__ static void make_diag(const PassDesc &p, unsigned long long odd, int t, int tb, diag *dg) {
        uint32_t c0, c1;
        diag_counts(p, odd, false, c0, c1);
#pragma unroll
        for (int k = 0; k < kTileE; ++k)
            dg[t + (k << tb)] = (double)byte_of(c0, k) * p.tc.dgv[0] + (double)byte_of(c1, k) * p.tc.dgv[1];
    }
    __device__ __forceinline__ void mac(coef c, const item &p) { s.x = fma(c, p.x, s.x); s.y = fma(c, p.y, s.y); }
    __device__ __forceinline__ void mac_swapped(coef, coef, const item &) {}
    __device__ __forceinline__ void mac_diag(const diag &d, const item &p) { mac(d, p); }
    __device__ __forceinline__ void add(const item &p) { s.x += p.x; s.y += p.y; }
    __device__ __forceinline__ void store(amp *o) const { *o = s; }
    template <int EPI>
    __device__ __forceinline__ void finish(const HvEpilogue<double, EPI> &epi, const EpiArgs &ea, size_t i, const item &v,
                                           amp *o, Acc<double> *d) const {
        epi.apply(ea, i, v, s, o, d);
    }
};

// two FP32 amplitudes: (a.re, a.im, b.re, b.im), b has offset bit 0 set
struct ItemF32 {
    typedef float2 amp;
    typedef float4 item;
    typedef float coef;
    typedef float2 diag;
    typedef float dot;
    static constexpr int SH = 1;
    float2 a = {0.f, 0.f}, b = {0.f, 0.f};
    __device__ static coef par(const PassDesc &p, int g) { return p.tc.par_f[g]; }
    __device__ static coef anti(const PassDesc &p, int g) { return p.tc.anti_f[g]; }
    __device__ static void make_diag(const PassDesc &p, unsigned long long odd, int t, int tb, diag *dg) {
        uint32_t a0, a1, b0, b1;
        diag_counts(p, odd, false, a0, a1);
        diag_counts(p, odd, true, b0, b1);
#pragma unroll
        for (int k = 0; k < kTileE; ++k)
            dg[t + (k << tb)] = make_float2((float)byte_of(a0, k) * p.tc.dgv_f[0] + (float)byte_of(a1, k) * p.tc.dgv_f[1],
                                            (float)byte_of(b0, k) * p.tc.dgv_f[0] + (float)byte_of(b1, k) * p.tc.dgv_f[1]);
    }
    __device__ __forceinline__ void mac(coef c, const item &p) {
        const float2 c2 = make_float2(c, c);
        a = __ffma2_rn(c2, make_float2(p.x, p.y), a);
        b = __ffma2_rn(c2, make_float2(p.z, p.w), b);
    }
    // the bond flips bit 0: a's partner is the other half; ca, cb by their parity
    __device__ __forceinline__ void mac_swapped(coef ca, coef cb, const item &p) {
        a = __ffma2_rn(make_float2(ca, ca), make_float2(p.z, p.w), a);
        b = __ffma2_rn(make_float2(cb, cb), make_float2(p.x, p.y), b);
    }
    __device__ __forceinline__ void mac_diag(const diag &d, const item &p) {
        a = __ffma2_rn(make_float2(d.x, d.x), make_float2(p.x, p.y), a);
        b = __ffma2_rn(make_float2(d.y, d.y), make_float2(p.z, p.w), b);
    }
    __device__ __forceinline__ void add(const item &p) {
        a = __fadd2_rn(a, make_float2(p.x, p.y));
        b = __fadd2_rn(b, make_float2(p.z, p.w));
    }
    __device__ __forceinline__ void store(amp *o) const {
        *reinterpret_cast<float4 *>(o) = make_float4(a.x, a.y, b.x, b.y);
    }
    template <int EPI>
    __device__ __forceinline__ void finish(const HvEpilogue<float, EPI> &epi, const EpiArgs &ea, size_t i, const item &v,
                                           amp *o, Acc<float> *d) const {
        store(o);   // every FP32 epilogue stores the product
        epi.dots(ea, i, make_float2(v.x, v.y), a, d);
        epi.dots(ea, i + 1, make_float2(v.z, v.w), b, d);
    }
};

// All bonds of one type for a thread's items.
template <int TYPE, int SWAP, int KM, class I>
__device__ __forceinline__ void tile_class(I (&acc)[kTileE], const char *buf, int at, int step,
                                           BondWalk<(I::SH > 0)> &bw) {
    const typename I::coef par = I::par(bw.pd, TYPE), anti = I::anti(bw.pd, TYPE);
    bw.template run<TYPE, SWAP, KM, typename I::item>(
        buf, at, step, [&](const typename I::item(&p)[kTileE], bool odd) {
            const typename I::coef s = odd ? anti : par, f = odd ? par : anti;
            if (TYPE == 2 && KM == 0 && !SWAP) {
                if (!odd) return;   // parallel z bonds: coefficient 0
            }
#pragma unroll
            for (int k = 0; k < kTileE; ++k) {
                if (SWAP) acc[k].mac_swapped(odd_in(k, KM) ? f : s, odd_in(k, KM) ? s : f, p[k]);
                else acc[k].mac(odd_in(k, KM) ? f : s, p[k]);
            }
        });
}
template <int TYPE, class I>
__device__ __forceinline__ void tile_bonds(I (&acc)[kTileE], const char *buf, int at, int step,
                                           BondWalk<(I::SH > 0)> &bw) {
    tile_class<TYPE, 0, 0>(acc, buf, at, step, bw);
    tile_class<TYPE, 0, 1>(acc, buf, at, step, bw);
    tile_class<TYPE, 0, 2>(acc, buf, at, step, bw);
    tile_class<TYPE, 0, 3>(acc, buf, at, step, bw);
    if constexpr (I::SH > 0) {
        tile_class<TYPE, 1, 0>(acc, buf, at, step, bw);
        tile_class<TYPE, 1, 1>(acc, buf, at, step, bw);
        tile_class<TYPE, 1, 2>(acc, buf, at, step, bw);
        tile_class<TYPE, 1, 3>(acc, buf, at, step, bw);
    }
}

// Column j of a launch with grid (tiles, columns): its arguments, or false if
// there is nothing to do.
__device__ __forceinline__ bool hv_column(const EpiArgs &ea0, EpiArgs &ea, size_t ld) {
    if (ea0.all_done && *ea0.all_done) return false;
    if (ea0.lowp && *ea0.lowp != ea0.lowp_run) return false;
    const int j = blockIdx.y;
    if (ea0.col_seed && ea0.col_seed[j].done != 0) return false;   // finished column: no work
    ea = ea0;
    ea.partials += (size_t)j * gridDim.x * 2;
    ea.counter += j;
    ea.result += (size_t)FTK_HV_DOTS * j;
    if (ea0.lo) ea.lo = static_cast<const float2 *>(ea0.lo) + (size_t)j * ld;
    return true;
}

// The pass. TB > 0: the thread bits as a compile-time constant, so that the
// strides of the shared tile fold into immediate offsets (full tiles: TB = 10).
template <class I, int EPI, int TB>
__device__ __forceinline__ void hv_tile_body(const typename I::amp *__restrict__ in, typename I::amp *out,
                                             const PassDesc &pd, const EpiArgs &ea0, long long ld) {
    typedef typename I::item item;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tb = TB > 0 ? TB : pd.tile_bits - 2 - I::SH;
    const int T = 1 << tb, n_items = T * kTileE;
    const int t = threadIdx.x;
    item *buf0 = reinterpret_cast<item *>(smem_raw), *buf1 = buf0 + n_items, *pb = buf1 + n_items;
    typename I::diag *dg = reinterpret_cast<typename I::diag *>(pb + n_items);   // per item
    double *red = reinterpret_cast<double *>(dg + n_items);
    const TileWalk<I::SH> w(pd, t, tb);
    const unsigned long long odd = odd_bonds(pd, t);
    I::make_diag(pd, odd, t, tb, dg);   // read by this thread only
    wait_previous();
    EpiArgs ea;
    if (!hv_column(ea0, ea, ld)) return;
    in += (size_t)blockIdx.y * ld;
    out += (size_t)blockIdx.y * ld;
    const HvEpilogue<typename I::dot, EPI> epi(ea);
    constexpr int ND = EPI == EPI_PLAIN ? 1 : 2;
    Acc<typename I::dot> dot[ND];
    const bool first = pd.first != 0, last = pd.last != 0;

    auto issue = [&](const typename I::amp *src, uint32_t ofs, item *buf) {
#pragma unroll
        for (int k = 0; k < kTileE; ++k) cp_async16(buf + t + T * k, src + (ofs + w.e[k]));
        cp_async_commit();
    };
    // Pipeline (commit order): v_0 [p_0] | per tile i: v_{i+1}, then after
    // tile i's sums p_{i+1}. A thread reads back only the partial items that it
    // copied itself, so pb needs no block barrier.
    const uint32_t n_tiles = 1u << pd.n_free;
    uint32_t tau = blockIdx.x;
    uint32_t ofs = tau < n_tiles ? w.base(pd, tau) : 0;
    if (tau < n_tiles) {
        issue(in, ofs, buf0);
        if (!first) issue(out, ofs, pb);
    }
    for (int it = 0; tau < n_tiles; tau += gridDim.x, ++it) {
        const item *cur = (it & 1) ? buf1 : buf0;
        item *nxt = (it & 1) ? buf0 : buf1;
        const bool more = tau + gridDim.x < n_tiles;
        const uint32_t ofs_n = more ? w.next(ofs) : 0;
        if (more) issue(in, ofs_n, nxt);
        // v of this tile: all but the newest one (first pass) or two groups
        if (first) { if (more) cp_async_wait<1>(); else cp_async_wait<0>(); }
        else { if (more) cp_async_wait<2>(); else cp_async_wait<1>(); }
        __syncthreads();
        I acc[kTileE];
        const char *cb = reinterpret_cast<const char *>(cur);
        // z bonds first, with the smaller coefficients; FP64 has them last in its
        // order, behind y and x
        BondWalk<(I::SH > 0)> bw(pd, odd);
        if constexpr (I::SH > 0) {
            tile_bonds<2>(acc, cb, t * 16, T * 16, bw);
        } else {
            BondWalk<false> bz(pd, odd, pd.f_end[bond_class(false, 2, 0, 0) - 1]);
            tile_bonds<2>(acc, cb, t * 16, T * 16, bz);
        }
        tile_bonds<1>(acc, cb, t * 16, T * 16, bw);
        tile_bonds<0>(acc, cb, t * 16, T * 16, bw);
        // the diagonal last: added first, its size would set the rounding of
        // every term after it
#pragma unroll
        for (int k = 0; k < kTileE; ++k) acc[k].mac_diag(dg[t + T * k], cur[t + T * k]);
        if (!first) {   // partial product of the earlier passes (own items)
            if (more) cp_async_wait<1>(); else cp_async_wait<0>();
#pragma unroll
            for (int k = 0; k < kTileE; ++k) acc[k].add(pb[t + T * k]);
            if (more) issue(out, ofs_n, pb);
        }
#pragma unroll
        for (int k = 0; k < kTileE; ++k) {
            const uint32_t i = ofs + w.e[k];
            if (!last) acc[k].store(out + i);
            else acc[k].finish(epi, ea, i, cur[t + T * k], out + i, dot);
        }
        ofs = ofs_n;
        __syncthreads();   // buffer `cur` is refilled two tiles later
    }
    cp_async_wait<0>();
    if (EPI == EPI_PLAIN || !last) return;
    double d[ND];
#pragma unroll
    for (int q = 0; q < ND; ++q) d[q] = dot[q].get();
    block_reduce<ND>(d, red);
    if (t < ND) ea.partials[(size_t)blockIdx.x * ND + t] = red[t];
    if (!last_block_reduce<ND>(ea.partials, ea.counter, ea.result, red)) return;
    if (EPI == EPI_TPQ && t == 0) tpq_statistics(ea, ea.result);
}

}  // namespace ftk

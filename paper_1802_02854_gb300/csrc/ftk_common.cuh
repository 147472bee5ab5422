// Shared definitions of the FTKomega CUDA path (kernels + host runtime).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#define FTK_MAX_SITES 30
#define FTK_MAX_PASS_BONDS 64
#define FTK_MAX_TILE_BITS 16
#define FTK_MAX_RHS 32
#define FTK_MAX_OMEGA 4096
#define FTK_RED_THREADS 256   // threads of the last-block reductions

// The couplings for the fixed-point FP64 passes (ftk_hv_fix.cu).
struct FixCoef {
    int32_t kh, kl, jh, jl;   // K/4 and J/4: (kh 2^30 + kl) 2^(ec - 60)
    int32_t lsh;              // left shift of the 53-bit significands
    int32_t sr;               // right shift of a pass's product
    int32_t ex;               // exponent of the result's quantum minus the input's largest
    float need;               // admitted: vectors whose smallest sum is at least need 2^(emax + 1)
};
// What the measuring launch finds in a vector (one per column).
struct FixRange {
    int32_t emax;             // largest biased exponent of its components
    uint32_t low;             // complement of the smallest sum's bf16 bits (starts from 0)
};
// Tiles and bonds of the measuring launch (fix_range_kernel in ftk_hv_fix.cu).
// Bonds by which of the offset bits 0 and 1 they flip (none, 0, 1, both): places
// of their own in mask, more of the first kind.
constexpr int kRangeBits = 14, kRangeBonds = 31;
__host__ __device__ constexpr int range_slots(int kind) { return kind == 0 ? 16 : 5; }
__host__ __device__ constexpr int range_slot(int kind) { return kind == 0 ? 0 : 11 + 5 * kind; }
struct RangePlan {
    int32_t bits, n_free;     // a tile: 2^bits amplitudes
    int32_t n[4];             // bonds of each kind
    int32_t pos[kRangeBits], free_pos[FTK_MAX_SITES];
    uint32_t mask[kRangeBonds];   // the other offset bits they flip (byte offset of the item)
    uint32_t par, anti;       // lower bounds of the coefficients' sizes, bf16 twice
};

// Matrix elements by bond type: a bond of type g adds, for parallel (par) /
// antiparallel (anti) spins i, j, the amplitude par[g] / anti[g] to
// |x ^ 2^i ^ 2^j>, and +dgv (parallel) / -dgv (antiparallel) on the diagonal,
// dgv[0] = J/4 for x and y bonds, dgv[1] = (J + K)/4 for z bonds. _f, _lo: float
// hi and lo parts.
struct TypeCoef {
    double par[3], anti[3], dgv[2];
    float par_f[3], anti_f[3], par_lo[3], anti_lo[3], dgv_f[2], dgv_lo[2];
};

// One tiled pass of H.v: a CTA owns 2^tile_bits amplitudes whose index bits
// tile_pos[] vary while the bits free_pos[] are fixed by the CTA index.
// Bonds with both sites among tile_pos are applied from shared memory.
// The low chunk_bits tile bits are global bits 0..chunk_bits-1, so a tile is
// a set of contiguous runs of 2^chunk_bits amplitudes (coalesced loads).
struct PassDesc {
    int32_t n_sites;
    int32_t tile_bits;
    int32_t chunk_bits;
    int32_t n_free;
    int32_t first;      // 1: start from zero; 0: add to the partial in out
    int32_t last;       // 1: apply the epilogue
    int32_t n_bonds;
    int32_t pad;
    int32_t tile_pos[FTK_MAX_TILE_BITS];
    int32_t free_pos[FTK_MAX_SITES];
    int8_t bi[FTK_MAX_PASS_BONDS];    // tile-offset bit of site i
    int8_t bj[FTK_MAX_PASS_BONDS];    // tile-offset bit of site j
    int8_t gam[FTK_MAX_PASS_BONDS];   // bond type
    // Kernel form of the bonds (hv_layout_pass, see BondWalk), sorted by class:
    // type, swap of an FP32 pair, register part of the mask.
    uint32_t fdesc[FTK_MAX_PASS_BONDS];
    int32_t f_end[24];
    uint32_t classes;
    // Double-float form (ftk_hv_df.cu): bonds ordered by group, those of group g
    // with the partner-thread mask grp_tmask[g] in [grp_end[g-1], grp_end[g]), the
    // last group with mask 0; bcase encodes the register part of a bond's mask: 0
    // none, 1 + a one bit a, 9 + 8a + b two bits a < b.
    int32_t n_groups;
    int32_t grp_tmask[FTK_MAX_PASS_BONDS + 1];
    int32_t grp_end[FTK_MAX_PASS_BONDS + 1];
    int8_t bcase[FTK_MAX_PASS_BONDS];
    float par_f[FTK_MAX_PASS_BONDS], anti_f[FTK_MAX_PASS_BONDS];
    float par_lo[FTK_MAX_PASS_BONDS], anti_lo[FTK_MAX_PASS_BONDS];
    TypeCoef tc;
    FixCoef fx;
};

namespace ftk {
// double complex as two doubles (16 B, layout of double2)
struct dcx { double re, im; };
}  // namespace ftk

// Device-resident state of the mTPQ iteration (one per context).
struct TpqState {
    double scale;      // s_k = 1 / ||stored psi_k||
    double logQ;       // log Q_k
    double ell;
    double n_sites;
    int32_t k;         // current step
    int32_t pad;
};

// Per-RHS seed-COCG scalars (double), written by the seed kernel.
struct CocgSeed {
    double zs_re, zs_im;        // seed shift
    double e0;                  // shift origin E_j
    double lnorm;               // ||lambda||
    double rho_re, rho_im;      // rho_k = r_k^T r_k
    double rho_prev_re, rho_prev_im;
    double alpha_re, alpha_im;  // alpha_k
    double alpha_prev_re, alpha_prev_im;
    double irho_re, irho_im;      // 1 / rho_k
    double ialpha_re, ialpha_im;  // 1 / alpha_k
    double beta_prev_re, beta_prev_im;  // beta_{k-1}
    double c_re, c_im;          // c_k = beta_{k-1} alpha_k / alpha_{k-1}
    double a1_re, a1_im;        // 1 + c_k - alpha_k z_s: coefficient of r_k in r_{k+1}
    double g_re, g_im;          // g_k = lambda^dagger r_k
    double nrm;                 // ||r_k||
    double resid;               // last max_s ||r_k|| / |pi^s_k| / ||lambda||
    double rescale;             // power of two applied to r_k, r_{k+1}, pi^s in this
                                // iteration (1: none), keeping ||r|| near ||lambda||
    int32_t k;                  // iteration index of this RHS
    int32_t done;               // 1 converged, 2 r^T r vanished, 3 alpha denominator
                                // vanished, 4 max_iter, 5 non-finite residual
    int32_t iters;              // iterations accumulated into G
    int32_t seed_idx;           // shift that is the seed system (moves when the seed switches)
    // Seed switching (the seed converged, shifts remain): this iteration the
    // slowest shift s* became the seed; r_k and w_k are scaled by s1 = 1/pi*_k,
    // r_{k-1} by s0 = 1/pi*_{k-1} (the switch kernel does it), the pi of every
    // shift likewise
    int32_t sw;                 // 1: switched in this iteration
    int32_t switches;           // number of switches so far
    double s1_re, s1_im, s0_re, s0_im;
};

// Dots produced by the vector kernels for each RHS (reduced, double).
// update kernel: [0..1] rho, [2..3] g, [4] |r|^2;  H pass: [0..1] mu
#define FTK_UPD_DOTS 6
#define FTK_HV_DOTS 2

// FP32 pair pass of the moment-based power spectrum (hip_pm_pairs.cu) and the
// fine cell list it reads (built in hip_power.cu).
#pragma once

#include "hip_internal.h"

// A cell list for the FP32 moment pass.  Frames: the box is cut into n_c^3
// coarse cells (R0 wide or more) and every offset is taken from its coarse cell's
// origin, so that it is exact (hip_cell_origin) and the candidate test rounds as
// the other FP32 paths do.  Order: particles are sorted by fine cell, g per coarse
// cell and axis, z fastest, so the fine cells of a z column are contiguous.
struct PmFine {
    const float4 *p4;     // [n] sorted: offset from the coarse cell's origin, weight
    const unsigned *cf;   // [n] fine cell (fx n_f + fy) n_f + fz; bit 31: not in the primary range
    const int *start;     // [n_f^3 + 1]
    const float2 *shift;  // [n_c][3] frame shift (hi, lo) from coarse cell c to c + d, d = -1, 0, 1 (hip_cell_shift)
    int n_c, g;
    int n;                // particles
};

#define HIP_PM_FINE_MAX (1 << 24)  // most fine cells of a list
#define HIP_PM_NO_ITEMS (1 << 30)  // more than any catalog's items
// Fine cells per coarse cell and axis.
int hip_pm_fine_grid(int64_t N, int n_c, int64_t max_cells);
// Scratch of a build that must be zero before it: int fill[n_f^3], col[n_f^2];
// then start [n_f^3 + 1], cid [N], p4 [N], cf [N], shift [3 n_c].
struct PmFineBuf {
    int *fill, *col, *start;
    int *cid;
    float4 *p4;
    unsigned *cf;
    float2 *shift;
    double *x64 = nullptr;  // FP64 pass: [N][3] sorted positions, wrapped into the box
    int *counter = nullptr;  // the moment passes' work counter (zero before), HIP_PM_NO_ITEMS on a rejected catalog
};
// Three launches.  S1 += sum of weights, wabs += sum of |weights| (both zero before;
// N for unit weights), *err |= 1 on a non-finite position or weight (the particle
// is then kept, in cell 0, so that the list stays well formed; M such particles would be
// M^2 / 2 candidates, so the work counter is moved past every item and no pass walks the list).
cudaError_t hip_build_fine(const float *pos, const float *w, int64_t N, double L, int n_c, int g, int64_t p0, int64_t p1,
                           const PmFineBuf &b, double *S1, double *wabs, int *err, cudaStream_t st);

// Sub-intervals S per moment interval and moments per sub-interval: on a
// sub-interval of half-width h, k h <= 2 / S, and the first neglected Legendre
// term of an edge function is (k h)^Q / (2Q - 1)!! of it: 9.1e-9 (S = 64, Q = 4),
// 1.0e-9 (32, 5), 3.7e-10 (16, 6), 4.5e-10 (8, 7), below the FP32 rounding of a pair's term (6e-8)
// and of varying sign from pair to pair.  The widest S whose words for three multipoles
// fit one CTA's shared memory is taken: fewer atomics per pair.  (One or two multipoles
// would fit wider ones beyond these lines; they take the same.)
struct PmSplit {
    int S, Q;
};
PmSplit hip_pm_split(int n_c);

// Constants of a catalog, made on the host: a single launch reads them as operands
// from its parameters, where they take no registers (copied into registers they made
// the kernels spill).
struct PmConst {
    float R0sq, dc, inv_dc, ihd, ihd_lo, iR, iR_lo;
    float cs, fs, inv_fs;  // coarse and fine cell side
    float reach, slack;    // R0 + slack; slack covers the rounding of offsets, cell edges and the candidate test
};

// One catalog of the pass (device-resident in a batched launch).
struct PmPairCat {
    PmConst k;             // set by hip_pm_items
    PmFine cl;
    int los, n_c;          // line-of-sight axis, moment intervals
    float R0, dc;
    double L, cs;          // box side, coarse cell side
    const double *wabs;    // sum |w|: sets the fixed-point unit
    double *G;             // [n_ell][Q][n_c S] FP64 totals (zero before the launch)
    unsigned long long *npairs;
    // work items: blocks of 32 sorted particles x n_col groups of neighbour columns x
    // n_split / n_col groups of their pieces
    int n_items, n_split, n_col;
};
// Constants and work items of a catalog for a launch of about `warps` warps, columns
// cut into pieces where they make fewer than per_warp items per warp.
void hip_pm_items(PmPairCat &c, long long warps, int per_warp = 6);
// n_ell = 1..3; full: every catalog's primary range is all its particles.  counter:
// one zeroed int per catalog.
cudaError_t hip_pm_pairs(const PmPairCat &cat, PmSplit sp, int n_ell, bool full, int *counter, cudaStream_t st);
cudaError_t hip_pm_pairs_batched(const PmPairCat *d_cats, int n_cats, int n_c_max, PmSplit sp, bool full, int warps,
                                 int *counter, cudaStream_t st);

// Warps a full launch of the pass keeps resident.
long long hip_pm_warps();

// One moment pass (FP32, or FP64 with f64) in a caller's buffer: the layout of its
// scratch and its steps.
struct Carve;
struct PmPlan {
    int n_c, g, n_f, n_e, n_ell, pm_nc;
    PmSplit sp;
    size_t o_zero, o_fill, o_col, o_G, o_start, o_cid, o_p4, o_cf, o_shift, o_acc, o_rho, o_out, zero_bytes;
    bool f64 = false;
    size_t o_x64 = 0;
    PmPlan() = default;
    // max_cells: most fine cells
    PmPlan(Carve &cv, int64_t N, double L, double R0, const double *k_edges, int n_k, int n_ell, int64_t max_cells,
           bool f64 = false);
    // S1 (double) at o_zero, sum |w| behind it, then:
    unsigned long long *npairs(char *b) const { return (unsigned long long *)(b + o_zero) + 2; }
    int *err(char *b) const { return (int *)(b + o_zero + 24); }  // error word, then the work counter
    // clears the scratch, builds the cell list (error word, S1)
    cudaError_t build(char *b, const float *pos, const float *w, int64_t N, double L, int64_t p0, int64_t p1,
                      cudaStream_t st) const;
    PmPairCat cat(char *b, int64_t N, double L, double R0, int los) const;
    // the totals G and the pair count; full: the primary range is [0, N)
    cudaError_t pairs(char *b, int64_t N, double L, double R0, int los, bool full, cudaStream_t st) const;
    // PmFinish::out at out(b), out_doubles() of them
    cudaError_t finish(char *b, double L, double R0, const double *k_edges, cudaStream_t st) const;
    double *out(char *b) const { return (double *)(b + o_out); }
    size_t out_doubles() const { return 2 * (size_t)n_ell * (n_e - 1) + 2; }
};
hip_status hip_pm_unpack(const double *h, int n, double *P_out, double *DD_out, int64_t *npairs_out);

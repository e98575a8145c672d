// Bispectrum kernels (Sec. 4 of arXiv:2005.01739): the FP64 a_lm pass, the FP64
// contraction and the C term.  The tensor-core contraction is in hip_bk_tc.cu.
//
// For every primary p (data particles, then the random catalog) the a_lm pass
// forms, over data neighbours j with 0 < |x_p - x_j| < R0,
//     A^a_lm(p) = sum_j w_j W(r/R0) jbar^a_l(r) R_lm(rhat)        (Eq. AC-def, binned)
// with real spherical harmonics R_lm scaled so that sum_m R_lm(u) R_lm(v) =
// L_l(u.v) (the addition theorem with the 4 pi / (2l+1) absorbed; real and
// complex harmonics give the same sum over m), and writes it to X[p][lm][a].
// The primary sum T^ab_l = sum_p s_p [sum_m A^a_lm A^b_lm - C^ab_l](p) (s_p = w_p
// for data primaries, -S1/N_r for random ones: the DDR^II term of Sec. 4.3 with
// a random catalog) is then the contraction sum_p s_p X_p X_p^T minus
//     sum_p s_p C^ab_l(p) = sum_(p,j) s_p w_j^2 W(r)^2 jbar^a_l(r) jbar^b_l(r),
// a pair sum of a function of r alone.  The a_lm pass accumulates it as 32
// Legendre moments of s_p w_j^2 W^2 per separation interval; the FP64 C-term
// kernels contract them with the products jbar^a_l jbar^b_l.
//
// FP64 a_lm pass (the FP32 one is hip_bk_alm32.cu): one warp owns one primary at a
// time (1 to 8 consecutive sorted primaries per work item).  Accepted neighbours are
// queued as separation vectors; 32 at a time they get one lane each for r, W, the
// 25 R_lm and the C-term moments, and are then drained with one lane per bin edge
// e: each lane evaluates F_l(r k_e), l = 0..4, from their tabulated series and
// accumulates w W F_l R_lm into its 25 registers.  At the end of the primary, adjacent edges
// give A^a_lm.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "hip_internal.h"
#include "hip_bispec.h"
#include "hip_bk_ylm.cuh"

static __constant__ HipCoeffs c_coeffs;
static cudaError_t hip_upload_cc_norm();
static cudaError_t hip_upload_tab64();
cudaError_t hip_upload_coeffs_bispec()
{
    cudaError_t e = cudaMemcpyToSymbol(c_coeffs, &hip_host_coeffs(), sizeof(HipCoeffs));
    if (e == cudaSuccess) e = hip_upload_ylm_norm();
    if (e == cudaSuccess) e = hip_upload_bk_alm32();
    if (e == cudaSuccess) e = hip_upload_cc_norm();
    if (e == cudaSuccess) e = hip_upload_tab64();
    return e;
}

// blockIdx.y = segment; warp w of block x takes data primaries x * 8 + w, stepping
// by gridDim.x * 8, lane l the bins l and l + 32 (n_k <= 64); the block's sums go
// to S with one FP64 atomic per bin.
__global__ void __launch_bounds__(256) k_bk_s_sum(const BkSeg *__restrict__ segs)
{
    __shared__ double red[8][64];
    const BkSeg sg = segs[blockIdx.y];
    if (!sg.S) return;  // block-uniform
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nk = sg.n_k;
    const double *X = (const double *)sg.X, *sp = (const double *)sg.sp;
    for (int li = 0; li < sg.n_S; ++li) {  // l = 2 li: harmonic (l, 0) is row l^2 + l, R_l0 = L_l(mu)
        const int hr = (2 * li) * (2 * li) + 2 * li;
        double s0 = 0.0, s1 = 0.0;
        for (int p = blockIdx.x * 8 + warp; p < sg.n_d; p += gridDim.x * 8) {
            const double w = sp[p];  // 0 for an excluded primary, whose row of X is not written
            if (w == 0.0) continue;
            const double *row = X + ((size_t)p * HIP_NLM + hr) * nk;
            if (lane < nk) s0 += w * row[lane];
            if (lane + 32 < nk) s1 += w * row[lane + 32];
        }
        __syncthreads();
        red[warp][lane] = s0;
        red[warp][lane + 32] = s1;
        __syncthreads();
        if (threadIdx.x < 64 && threadIdx.x < nk) {
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
            if (t != 0.0) atomicAdd(&sg.S[li * nk + threadIdx.x], t);
        }
    }
}

cudaError_t hip_bk_s_sum(const BkSeg *segs, int n_segs, cudaStream_t st)
{
    k_bk_s_sum<<<dim3(1216, n_segs), 256, 0, st>>>(segs);
    return cudaGetLastError();
}

int hip_bk_intervals(double R0, double k_max)
{
    const double q = std::ceil(R0 * k_max / 8.0);
    return q < 1.0 ? 1 : (int)q;
}

#define HIP_BK_WARPS 4  // most warps of a CTA
#define HIP_BK_SMEM 232448  // opt-in shared memory of a CTA
#define HIP_NLMP 36  // a drained pair's record: the 25 R_lm, w_j W, P_m(t) for m < HIP_BK64_M

struct BkWarpSmem {
    alignas(16) double qa[64][4];            // accepted neighbours: primary minus neighbour, w_j
    alignas(16) double qd[32][HIP_NLMP];     // drained pairs: R_lm (0..24), w_j W (25), P_m(t) (26 + m)
    double pt[32][HIP_BK_NM + 1];            // C-term weight s_p w_j^2 W^2 times R_m(t), m < 32
    int tc[32];                         // table interval of each drained pair
    int qc[32];                         // C-term interval of each drained pair
};

__global__ void k_sorted_cells(const int *__restrict__ start, int n_cells, int *__restrict__ scell)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n_cells; c += gridDim.x * blockDim.x)
        for (int i = start[c]; i < start[c + 1]; ++i) scell[i] = c;
}

cudaError_t hip_sorted_cells(const int *cell_start, int n_cells, int *scell, cudaStream_t st)
{
    const int blocks = (n_cells + 255) / 256;
    k_sorted_cells<<<blocks < 1 ? 1 : blocks, 256, 0, st>>>(cell_start, n_cells, scell);
    return cudaGetLastError();
}

// Edge functions of the FP64 pass: F_l(k_e r) as Legendre series in r on intervals
// with k_max h <= 1/4 (band-limited: the first neglected term is at most (1/4)^10 / 19!! =
// 1.5e-15, and about 1e-17 with F_l's own spectrum), tabulated as
// tab[interval][m][l][edge] for the catalogs of a chunk.  Evaluating them per
// (pair, edge) (sine, cosine and the sine integral's three ranges, all run by a warp
// whose lanes are the edges) took about 235 FP64 operations; the series take 50, and
// the table's own 12 evaluations per (interval, edge) are a fraction of a millisecond.
// Error against 64 bits (2-norm, median of 24 catalogs) by evaluation / so: 1.2e4 data
// particles 1.28e-15 / 1.26e-15, 1500 1.49e-15 / 1.48e-15.
#define HIP_BK64_NG 12
#define HIP_BK64_CB 8
static __constant__ double c_t64_x[HIP_BK64_NG], c_t64_P[HIP_BK64_NG][HIP_BK64_M];  // nodes; w_g (2m+1)/2 P_m
static cudaError_t hip_upload_tab64()
{
    void hip_gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w);
    std::vector<double> x, w;
    hip_gauss_legendre(HIP_BK64_NG, x, w);
    double P[HIP_BK64_NG][HIP_BK64_M];
    for (int g = 0; g < HIP_BK64_NG; ++g) {
        double p0 = 1.0, p1 = x[g];
        for (int m = 0; m < HIP_BK64_M; ++m) {
            P[g][m] = w[g] * (m + 0.5) * p0;
            const double p2 = ((2.0 * m + 3.0) * x[g] * p1 - (m + 1.0) * p0) / (m + 2.0);
            p0 = p1;
            p1 = p2;
        }
    }
    cudaError_t e = cudaMemcpyToSymbol(c_t64_x, x.data(), sizeof(double) * HIP_BK64_NG);
    return e == cudaSuccess ? cudaMemcpyToSymbol(c_t64_P, P, sizeof(P)) : e;
}

__global__ void __launch_bounds__(HIP_BK64_CB * HIP_BK64_NG) k_bk_tab64(const BkCat<double> *__restrict__ cats, int ci)
{
    __shared__ double f[HIP_LMAX + 1][HIP_BK64_CB][HIP_BK64_NG];
    const BkCat<double> &a = cats[ci];
    const int e = blockIdx.y, c0 = blockIdx.x * HIP_BK64_CB, ep = a.n_e <= 16 ? 16 : 32;
    {
        const int q = threadIdx.x / HIP_BK64_NG, g = threadIdx.x - q * HIP_BK64_NG;
        double F[HIP_LMAX + 1];
        hip_F_f64<31>((c0 + q + 0.5 * (1.0 + c_t64_x[g])) / a.tab_scale * a.k[e], c_coeffs, F);
#pragma unroll
        for (int l = 0; l <= HIP_LMAX; ++l) f[l][q][g] = F[l];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < HIP_BK64_CB * HIP_BK64_M * (HIP_LMAX + 1); i += blockDim.x) {
        const int l = i % (HIP_LMAX + 1), m = i / (HIP_LMAX + 1) % HIP_BK64_M, q = i / ((HIP_LMAX + 1) * HIP_BK64_M);
        if (c0 + q >= a.tab_n) continue;
        double v = 0.0;
#pragma unroll
        for (int g = 0; g < HIP_BK64_NG; ++g) v = fma(f[l][q][g], c_t64_P[g][m], v);
        a.tab[(((size_t)(c0 + q) * HIP_BK64_M + m) * (HIP_LMAX + 1) + l) * ep + e] = v;
    }
}

int hip_bk_tab64_intervals(double R0, double k_max) { return std::max(8, (int)std::ceil(2.0 * R0 * k_max)); }
size_t hip_bk_tab64_doubles(int n, int n_e) { return (size_t)n * HIP_BK64_M * (HIP_LMAX + 1) * (n_e <= 16 ? 16 : 32); }

cudaError_t hip_bk_tab64(const BkCat<double> *d_cats, int ci, int tab_n, int n_e, cudaStream_t st)
{
    k_bk_tab64<<<dim3((tab_n + HIP_BK64_CB - 1) / HIP_BK64_CB, n_e), HIP_BK64_CB * HIP_BK64_NG, 0, st>>>(d_cats, ci);
    return cudaGetLastError();
}

// Edge quantities of a lane: edge e = lane (n_e <= 32 in FP64), or lane mod 16 where 16 suffice.
struct BkEdges {
    double k3, k3n, jfac;
    int e, ep;  // edge, row length of the table
    bool on;  // the lane has an edge
};

__device__ __forceinline__ void bk_load_edges(const BkCat<double> &a, int lane, BkEdges &ed)
{
    const int n_e = a.n_e, e = n_e <= 16 ? lane & 15 : lane;
    ed.on = e < n_e;
    ed.e = e;
    ed.ep = n_e <= 16 ? 16 : 32;
    ed.k3 = e < n_e ? a.k3[e] : 0.0;
    ed.k3n = e + 1 < n_e ? a.k3[e + 1] : 0.0;
    ed.jfac = e + 1 < n_e ? a.jfac[e] : 0.0;
}

// Process the first n (<= 32) queued neighbours of the current primary: their
// geometry and harmonics (one per lane), their C-term moments (one lane per
// moment) and their contributions to the edge sums (one lane per bin edge).
__device__ __forceinline__ void bk_flush(BkWarpSmem &sm, double *cm, int n, double s_p, double iR, double iR_lo, double cc_scale, double cc_lo, int n_cc,
                                         const double *__restrict__ tab, int tab_n, double tab_scale, int n_e, const BkEdges &ed, int lane, double (&E)[HIP_NLM])
{
    if (lane < n) {
        const double dx = sm.qa[lane][0], dy = sm.qa[lane][1], dz = sm.qa[lane][2], wj = sm.qa[lane][3];
        const double r = sqrt(dx * dx + dy * dy + dz * dz);
        const double ir = 1.0 / r;
        const double W = hip_W<double>(fma(r, iR_lo, r * iR));
        double R[HIP_NLM];
        hip_real_ylm<double>(dx * ir, dy * ir, dz * ir, R);
#pragma unroll
        for (int i = 0; i < HIP_NLM; ++i) sm.qd[lane][i] = R[i];
        sm.qd[lane][25] = wj * W;
        {  // the edge functions' interval and the P_m at its position
            const double x = r * tab_scale;
            const int c = min((int)x, tab_n - 1);
            const double t = 2.0 * (x - (double)c) - 1.0;
            double p0 = 1.0, p1 = t;
            sm.tc[lane] = c;
#pragma unroll
            for (int m = 0; m < HIP_BK64_M; ++m) {
                sm.qd[lane][26 + m] = p0;
                const double p2 = ((2.0 * m + 3.0) / (m + 2.0)) * t * p1 - ((m + 1.0) / (m + 2.0)) * p0;
                p0 = p1;
                p1 = p2;
            }
        }
        // C term: interval c of width R0 / n_cc, coordinate t in [-1, 1]
        const double x = fma(r, cc_lo, r * cc_scale);
        int c = (int)x;
        if (c > n_cc - 1) c = n_cc - 1;
        double t = 2.0 * (x - (double)(c)) - 1.0;
        t = t < -1.0 ? -1.0 : (t > 1.0 ? 1.0 : t);
        const double wc = s_p * wj * wj * W * W;
        double p0 = wc, p1 = wc * t;
        sm.pt[lane][0] = p0;
        sm.pt[lane][1] = p1;
#pragma unroll
        for (int m = 1; m < HIP_BK_NM - 1; ++m) {
            const double p2 = hip_leg_alpha<double>(m) * t * p1 - hip_leg_beta<double>(m) * p0;  // R_m = d_m P_m
            sm.pt[lane][m + 1] = p2;
            p0 = p1;
            p1 = p2;
        }
        sm.qc[lane] = c;
    }
    __syncwarp();
    for (int q = 0; q < n; ++q) cm[sm.qc[q] * HIP_BK_NM + lane] += sm.pt[q][lane];
    // up to 16 edges: the half-warps take alternate pairs (their sums are joined at the
    // end of the primary), so that no lane of the FP64 pipe idles
    const int step = n_e <= 16 ? 2 : 1;
    for (int q0 = 0; q0 < n; q0 += step) {
        const int q = q0 + (step == 2 ? lane >> 4 : 0);
        const double *rec = sm.qd[min(q, n - 1)];
        const double *tb = tab + (size_t)sm.tc[min(q, n - 1)] * HIP_BK64_M * (HIP_LMAX + 1) * ed.ep + ed.e;
        const double ww = rec[25];
        double F[HIP_LMAX + 1];
#pragma unroll
        for (int l = 0; l <= HIP_LMAX; ++l) F[l] = __ldg(tb + l * ed.ep);  // P_0 = 1
#pragma unroll
        for (int m = 1; m < HIP_BK64_M; ++m) {
            const double p = rec[26 + m];
#pragma unroll
            for (int l = 0; l <= HIP_LMAX; ++l) F[l] = fma(__ldg(tb + (m * (HIP_LMAX + 1) + l) * ed.ep), p, F[l]);
        }
        if (ed.on && q < n) {
#pragma unroll
            for (int l = 0; l <= HIP_LMAX; ++l) {
                const double f = ww * F[l];
#pragma unroll
                for (int m = -l; m <= l; ++m) E[l * l + l + m] += f * rec[l * l + l + m];
            }
        }
    }
    __syncwarp();
}

// One primary g (data first, then randoms) of catalog a: the 27-cell neighbour
// scan and the queued flushes; then A^a_lm = jfac_a (k_{a+1}^3 E_{a+1} - k_a^3 E_a)
// into Xp[lm][a] and s_p into *spp.
__device__ __forceinline__ void bk_primary(const BkCat<double> &a, int g, BkWarpSmem &sm, double *cm,
                                           const BkEdges &ed, int lane, double *Xp, double *spp,
                                           unsigned long long &cnt_d, unsigned long long &cnt_r)
{
    const int n_e = a.n_e, nk = n_e - 1, n_c = a.data.n_c;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool is_rand = g >= a.n_data;
    const CellList<double> &pl = is_rand ? a.rand : a.data;
    const int p = is_rand ? g - a.n_data : g;
    const long long oi = pl.idx[p];
    const bool excluded = is_rand ? (oi < a.rp0 || oi >= a.rp1) : (oi < a.dp0 || oi >= a.dp1);
    const double s_p = excluded ? 0.0 : (is_rand ? a.rand_weight : (double)(pl.w[p]));
    if (lane == 0) *spp = s_p;
    if (excluded) return;
    const double R0sq = a.R0 * a.R0, iR = a.iR, iR_lo = a.iR_lo, cc_scale = a.cc_scale, cc_lo = a.cc_lo;
    const int n_cc = a.n_cc;
    const int c = is_rand ? a.rcell[p] : a.dcell[p];
    const int cx = c / (n_c * n_c), cy = (c / n_c) % n_c, cz = c % n_c;
    const double px = pl.x[p], py = pl.y[p], pz = pl.z[p];
    const int self = is_rand ? -1 : p;
    double E[HIP_NLM];
#pragma unroll
    for (int i = 0; i < HIP_NLM; ++i) E[i] = 0.0;
    int qn = 0;
    // cell shifts of this primary: lane 3 axis + d + 1 holds the shift of
    // neighbour offset d along that axis
    double shl = 0.0, shll = 0.0;
    if (lane < 9) {
        const int ax = lane / 3, cc = ax == 0 ? cx : (ax == 1 ? cy : cz);
        hip_cell_shift(a.data, cc, lane % 3 - 1, shl, shll);
    }
    // the 27 neighbour cells, one per lane
    int b0 = 0, bn = 0;
    if (lane < 27) {
        const int nb = (((cx + lane / 9 - 1 + n_c) % n_c) * n_c + (cy + lane / 3 % 3 - 1 + n_c) % n_c) * n_c +
                       (cz + lane % 3 - 1 + n_c) % n_c;
        b0 = a.data.cell_start[nb];
        bn = a.data.cell_start[nb + 1] - b0;
    }
    // nine rows of three z neighbours: a test of 32 candidates costs the FP64 pipe the
    // same for the 7 of one cell as for the 21 of a row
    for (int row = 0; row < 9; ++row) {
        const double ox = px - __shfl_sync(0xffffffffu, shl, row / 3), oy = py - __shfl_sync(0xffffffffu, shl, 3 + row % 3);
        const int n0 = __shfl_sync(0xffffffffu, bn, 3 * row), n1 = n0 + __shfl_sync(0xffffffffu, bn, 3 * row + 1),
                  n2 = n1 + __shfl_sync(0xffffffffu, bn, 3 * row + 2);
        for (int b = 0; b < n2; b += 32) {
            const int q = b + lane, z = (q >= n0) + (q >= n1);
            const int j = __shfl_sync(0xffffffffu, b0, 3 * row + z) + q - (z == 0 ? 0 : z == 1 ? n0 : n1);
            const double oz = pz - __shfl_sync(0xffffffffu, shl, 6 + z);
            bool ok = false;
            double ddx = 0.0, ddy = 0.0, ddz = 0.0;
            if (q < n2) {
                ddx = ox - a.data.x[j];
                ddy = oy - a.data.y[j];
                ddz = oz - a.data.z[j];
                const double r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                ok = (r2 < R0sq) && (r2 > 0.0) && (j != self);
            }
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const int slot = qn + __popc(m & lt_mask);
                sm.qa[slot][0] = ddx;
                sm.qa[slot][1] = ddy;
                sm.qa[slot][2] = ddz;
                sm.qa[slot][3] = (double)(a.data.w[j]);
            }
            const int nq = __popc(m);
            if (is_rand)
                cnt_r += nq;
            else
                cnt_d += nq;
            qn += nq;
            if (qn >= 32) {
                __syncwarp();
                bk_flush(sm, cm, 32, s_p, iR, iR_lo, cc_scale, cc_lo, n_cc, a.tab, a.tab_n, a.tab_scale, n_e, ed, lane, E);
                const int rest = qn - 32;
                double mv[4] = {0.0, 0.0, 0.0, 0.0};
                if (lane < rest) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) mv[k] = sm.qa[32 + lane][k];
                }
                __syncwarp();
                if (lane < rest) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) sm.qa[lane][k] = mv[k];
                }
                qn = rest;
                __syncwarp();
            }
        }
    }
    if (qn > 0) {
        __syncwarp();
        bk_flush(sm, cm, qn, s_p, iR, iR_lo, cc_scale, cc_lo, n_cc, a.tab, a.tab_n, a.tab_scale, n_e, ed, lane, E);
    }
#pragma unroll
    for (int i = 0; i < HIP_NLM; ++i) {
        if (n_e <= 16) E[i] += __shfl_xor_sync(0xffffffffu, E[i], 16);
        const double nxt = __shfl_down_sync(0xffffffffu, E[i], 1);
        if (lane < nk) Xp[i * nk + lane] = ed.jfac * (ed.k3n * nxt - ed.k3 * E[i]);
    }
}

// The a_lm pass: persistent CTAs of up to 4 warps; each warp takes work items (up to 8
// consecutive primaries of one span) from an atomic counter.  Per warp, the
// C-term moments of the current catalog sit in a shared array, added to the warp's
// slot after every item and to the catalog's moments when the warp leaves the catalog.
__global__ void __launch_bounds__(HIP_BK_WARPS * 32) k_bk_alm(const BkCat<double> *__restrict__ cats,
                                                              const BkSpan *__restrict__ spans, int n_spans, int n_items,
                                                              int ncc_max, double *__restrict__ X, double *__restrict__ sp,
                                                              double *__restrict__ cm_slots, int *counter)
{
    extern __shared__ __align__(16) unsigned char bk_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    BkWarpSmem &sm = reinterpret_cast<BkWarpSmem *>(bk_raw)[warp];
    double *cm = reinterpret_cast<double *>(bk_raw + n_warps * sizeof(BkWarpSmem)) + (size_t)warp * ncc_max * HIP_BK_NM;
    double *slot = cm_slots + ((size_t)blockIdx.x * n_warps + warp) * ncc_max * HIP_BK_NM;
    for (int i = lane; i < ncc_max * HIP_BK_NM; i += 32) cm[i] = 0.0;
    __syncwarp();
    BkEdges ed;
    unsigned long long cnt_d = 0, cnt_r = 0;
    int cur = -1, si = 0;
    auto leave = [&](int c) {
        const BkCat<double> &a = cats[c];
        for (int i = lane; i < a.n_cc * HIP_BK_NM; i += 32) {
            const double v = slot[i];
            if (v != 0.0) {
                atomicAdd(&a.cmom[i], v);
                slot[i] = 0.0;
            }
        }
        if (lane == 0) {  // cnt_d, cnt_r are warp-uniform
            if (cnt_d) atomicAdd(a.npairs, cnt_d);
            if (cnt_r) atomicAdd(a.npairs + 1, cnt_r);
        }
        cnt_d = cnt_r = 0;
    };
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(counter, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) break;
        while (si + 1 < n_spans && item >= spans[si].item_end) ++si;
        while (si > 0 && item < spans[si].item_begin) --si;
        const BkSpan sp_ = spans[si];
        if (sp_.cat != cur) {
            if (cur >= 0) leave(cur);
            cur = sp_.cat;
            bk_load_edges(cats[cur], lane, ed);
        }
        const BkCat<double> &a = cats[cur];
        const int nk = a.n_e - 1;
        const int g0 = sp_.g0 + (item - sp_.item_begin) * sp_.prim;
        const int g1 = min(g0 + sp_.prim, sp_.g1);
        for (int g = g0; g < g1; ++g) {
            const long long o = g - sp_.g0;
            bk_primary(a, g, sm, cm, ed, lane, X + sp_.x_off + o * HIP_NLM * nk, sp + sp_.sp_off + o, cnt_d,
                               cnt_r);
        }
        __syncwarp();
        // the item's C-term moments into the warp's FP64 slot
        for (int i = lane; i < a.n_cc * HIP_BK_NM; i += 32) {
            const double v = cm[i];
            if (v != 0.0) {
                slot[i] += (double)v;
                cm[i] = 0.0;
            }
        }
        __syncwarp();
    }
    if (cur >= 0) leave(cur);
}

int hip_bk_item_prims(long long total)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)std::max(1LL, std::min((long long)HIP_BK_PRIM, total / (8LL * 16 * sms)));
}

size_t hip_bk_alm_slot_bytes(int ncc_max)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // at most 16 CTAs per SM (the shared memory of a CTA is > 14 KB)
    return sizeof(double) * (size_t)sms * 16 * HIP_BK_WARPS * ncc_max * HIP_BK_NM;
}

cudaError_t hip_bk_alm(const BkCat<double> *cats, const BkSpan *spans, int n_spans, int n_items, int nk_max, int ncc_max,
                       double *X, double *sp, double *cm_slots, int *counter, cudaStream_t st)
{
    if (nk_max > 31) return cudaErrorInvalidValue;
    // four warps, or as many as fit beside their C-term sums: four up to 149 intervals
    // (R0 k_max 1192), one up to 830
    const size_t per_warp = sizeof(BkWarpSmem) + sizeof(double) * (size_t)ncc_max * HIP_BK_NM;
    const int warps = (int)std::max<size_t>(1, std::min<size_t>(HIP_BK_WARPS, HIP_BK_SMEM / per_warp));
    const size_t smem = warps * per_warp;
    cudaError_t e = cudaFuncSetAttribute(k_bk_alm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, nb = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bk_alm, warps * 32, smem);
    if (nb < 1) nb = 1;
    if (nb > 16) nb = 16;
    int grid = sms * nb;
    const int need = (n_items + warps - 1) / warps;
    if (grid > need) grid = need < 1 ? 1 : need;
    k_bk_alm<<<grid, warps * 32, smem, st>>>(cats, spans, n_spans, n_items, ncc_max, X, sp, cm_slots, counter);
    return cudaGetLastError();
}

// ------------------------------------------------------- FP64 contraction ----
// sum_p s_p sum_m X_p[lm][a] X_p[lm][b] for a <= b (plain path): CTAs of 256
// threads take contiguous ranges of the segments' primaries (laid end to end),
// stage four primaries' X in shared memory at a time, and keep up to
// HIP_BK64_NE upper-triangle entries (l, a <= b) per thread in FP64 registers;
// on leaving a segment they are added to its accumulator (both triangles).
#define HIP_BK64_THREADS 256
#define HIP_BK64_NE 40    // ceil(5 * 63 * 64 / 2 / 256): every upper-triangle entry up to 63 bins
#define HIP_BK64_STAGE 4  // primaries staged per step

template <typename T>
__global__ void __launch_bounds__(HIP_BK64_THREADS) k_bk_contract_f64(const BkSeg *__restrict__ segs, int n_segs,
                                                                     long long n_total)
{
    extern __shared__ __align__(16) unsigned char c64_raw[];
    double *xs = reinterpret_cast<double *>(c64_raw);  // [HIP_BK64_STAGE][25][n_k]
    __shared__ double s_sp[HIP_BK64_STAGE];
    const long long per = (n_total + gridDim.x - 1) / gridDim.x;
    const long long q0 = blockIdx.x * per, q1 = min(q0 + per, n_total);
    if (q0 >= q1) return;
    // first segment of this CTA
    int sg = 0;
    long long base = 0;
    while (sg < n_segs && base + segs[sg].n_p <= q0) base += segs[sg++].n_p;
    double acc[HIP_BK64_NE];
    int ent[HIP_BK64_NE];  // (l << 16) | (a << 8) | b, or -1
    int cur_nk = -1;
    auto setup = [&](int nk) {
        const int ntri = nk * (nk + 1) / 2;
#pragma unroll
        for (int i = 0; i < HIP_BK64_NE; ++i) {
            acc[i] = 0.0;
            const int e = threadIdx.x + HIP_BK64_THREADS * i;
            ent[i] = -1;
            if (e < (HIP_LMAX + 1) * ntri) {
                const int l = e / ntri;
                int r = e - l * ntri, aa = 0;
                while (r >= nk - aa) {
                    r -= nk - aa;
                    ++aa;
                }
                ent[i] = (l << 16) | (aa << 8) | (aa + r);
            }
        }
        cur_nk = nk;
    };
    auto flush = [&](const BkSeg &s) {
        const int nk = s.n_k;
#pragma unroll
        for (int i = 0; i < HIP_BK64_NE; ++i)
            if (ent[i] >= 0 && acc[i] != 0.0) {
                const int l = ent[i] >> 16, aa = (ent[i] >> 8) & 255, bb = ent[i] & 255;
                atomicAdd(&s.acc[((size_t)l * nk + aa) * nk + bb], acc[i]);
                if (aa != bb) atomicAdd(&s.acc[((size_t)l * nk + bb) * nk + aa], acc[i]);
                acc[i] = 0.0;
            }
    };
    long long q = q0;
    while (q < q1 && sg < n_segs) {
        const BkSeg s = segs[sg];
        const int nk = s.n_k;
        if (nk != cur_nk) setup(nk);
        const long long s_end = min(q1, base + s.n_p);
        const T *Xd = reinterpret_cast<const T *>(s.X);
        const T *spd = reinterpret_cast<const T *>(s.sp);
        while (q < s_end) {
            const int np = (int)min((long long)HIP_BK64_STAGE, s_end - q);
            const long long p0 = q - base;
            __syncthreads();
            for (int i = threadIdx.x; i < np * HIP_NLM * nk; i += HIP_BK64_THREADS)
                xs[i] = (double)Xd[p0 * HIP_NLM * nk + i];
            if (threadIdx.x < HIP_BK64_STAGE)
                s_sp[threadIdx.x] = threadIdx.x < np ? (double)spd[p0 + threadIdx.x] : 0.0;
            __syncthreads();
            for (int pp = 0; pp < np; ++pp) {
                const double spv = s_sp[pp];
                if (spv == 0.0) continue;
                const double *xp = xs + (size_t)pp * HIP_NLM * nk;
#pragma unroll
                for (int i = 0; i < HIP_BK64_NE; ++i) {
                    if (ent[i] < 0) continue;
                    const int l = ent[i] >> 16, aa = (ent[i] >> 8) & 255, bb = ent[i] & 255;
                    double d = 0.0;
                    for (int m = l * l; m <= l * l + 2 * l; ++m) d += xp[m * nk + aa] * xp[m * nk + bb];
                    acc[i] += spv * d;
                }
            }
            q += np;
        }
        flush(s);
        if (q >= base + s.n_p) {
            base += s.n_p;
            ++sg;
        }
    }
}

template <typename T>
cudaError_t hip_bk_contract_f64(const BkSeg *segs, int n_segs, long long n_p_total, int nk_max, cudaStream_t st)
{
    const size_t smem = sizeof(double) * HIP_BK64_STAGE * HIP_NLM * nk_max;
    cudaError_t e =
        cudaFuncSetAttribute(k_bk_contract_f64<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long grid = (long long)sms * 4;
    if (grid > n_p_total / 16 + 1) grid = n_p_total / 16 + 1;
    k_bk_contract_f64<T><<<(int)grid, HIP_BK64_THREADS, smem, st>>>(segs, n_segs, n_p_total);
    return cudaGetLastError();
}
template cudaError_t hip_bk_contract_f64<float>(const BkSeg *, int, long long, int, cudaStream_t);
template cudaError_t hip_bk_contract_f64<double>(const BkSeg *, int, long long, int, cudaStream_t);

// ------------------------------------------------------------ the C term ----
// sum_(p,j) s_p w_j^2 W^2 jbar^a_l(r) jbar^b_l(r) from the moments
// M[c][m] = sum over pairs in interval c of s_p w_j^2 W^2 P_m(t): on each interval
// the pair density in t is rho_c(t) = sum_m (2m+1)/2 M[c][m] P_m(t), so the sum is
// sum_c int_{-1}^{1} rho_c(t) f(r_c(t)) dt, taken by 48-point Gauss-Legendre
// (exact for the degree-31 rho times the band-limited f).  All FP64.
#define HIP_BK_CQ 48

static double s_cq_x[HIP_BK_CQ], s_cq_w[HIP_BK_CQ];
static bool s_cq_ready = false;

static void cq_nodes()
{
    if (s_cq_ready) return;
    const int n = HIP_BK_CQ;
    for (int i = 0; i < n; ++i) {
        double x = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            const double dp = n * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; ++k) {
            const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        const double dp = n * (x * p1 - p0) / (x * x - 1.0);
        s_cq_x[i] = x;
        s_cq_w[i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
    s_cq_ready = true;
}

struct BkCQ {
    double x[HIP_BK_CQ], w[HIP_BK_CQ], inv[HIP_BK_NM];  // inv[m] = 1 / (m + 1)
};

size_t hip_bk_cterm_scratch_bytes(int n_cc, int n_k)
{
    const size_t nodes = (size_t)n_cc * HIP_BK_CQ;
    return sizeof(double) * nodes * (1 + (HIP_LMAX + 1) * (size_t)n_k);
}

// Per node: its weights w_q rho_c(t_q) for each of the n_L moment sets, and
// jbar^a_l(r_q) for every l, a.  A block takes HIP_BK_CN nodes and evaluates their edge
// functions one (node, edge) per thread: FP64 runs at 1/64 of the FP32 rate here, and
// one thread per node walking the edges took 350 to 670 us whatever the size.
#define HIP_BK_CN 8
static __constant__ double c_cc_norm[HIP_BK_NM];  // (2m+1)/2 / d_m: M[m] are moments of R_m = d_m P_m
__global__ void __launch_bounds__(256) k_bk_cc_nodes(BkCTerm c, BkCQ q, int n_L, double *__restrict__ wn,
                                                     double *__restrict__ J)
{
    __shared__ double f[HIP_LMAX + 1][HIP_BMAXE][HIP_BK_CN];  // k^3 F_l(r k)
    const int n_nodes = c.n_cc * HIP_BK_CQ, nk = c.n_e - 1, i0 = blockIdx.x * HIP_BK_CN;  // HIP_BK_CQ is a multiple of HIP_BK_CN
    for (int t = threadIdx.x; t < c.n_e * HIP_BK_CN; t += 256) {
        const int e = t / HIP_BK_CN, p = t % HIP_BK_CN, i = i0 + p, cc = i / HIP_BK_CQ;
        const double r = (cc + 0.5 * (1.0 + q.x[i - cc * HIP_BK_CQ])) * (c.R0 / c.n_cc), k = c.k[e], k3 = k * k * k;
        double F[HIP_LMAX + 1];
        hip_F_f64<31>(r * k, c_coeffs, F);
#pragma unroll
        for (int l = 0; l <= HIP_LMAX; ++l) f[l][e][p] = k3 * F[l];
    }
    if (threadIdx.x < HIP_BK_CN * n_L) {
        const int L = threadIdx.x / HIP_BK_CN, i = i0 + threadIdx.x % HIP_BK_CN, cc = i / HIP_BK_CQ, iq = i - cc * HIP_BK_CQ;
        const double t = q.x[iq];
        const double *M = c.cmom + ((size_t)L * c.n_cc + cc) * HIP_BK_NM;
        double p0 = 1.0, p1 = t, rho = c_cc_norm[0] * M[0] + c_cc_norm[1] * M[1] * t;
        for (int m = 1; m < HIP_BK_NM - 1; ++m) {
            const double p2 = ((2.0 * m + 1.0) * t * p1 - m * p0) * q.inv[m];
            rho += c_cc_norm[m + 1] * M[m + 1] * p2;
            p0 = p1;
            p1 = p2;
        }
        wn[(size_t)L * n_nodes + i] = q.w[iq] * rho;
    }
    __syncthreads();
    // jbar^a_l(r) = 3 [k_{a+1}^3 F_l(r k_{a+1}) - k_a^3 F_l(r k_a)] / (k_{a+1}^3 - k_a^3)
    for (int t = threadIdx.x; t < nk * HIP_BK_CN; t += 256) {
        const int a = t / HIP_BK_CN, p = t % HIP_BK_CN;
        const double lo = c.k[a], hi = c.k[a + 1], jf = 3.0 / (hi * hi * hi - lo * lo * lo);
#pragma unroll
        for (int l = 0; l <= HIP_LMAX; ++l)
            J[((size_t)l * nk + a) * n_nodes + i0 + p] = jf * (f[l][a + 1][p] - f[l][a][p]);
    }
}

static cudaError_t hip_upload_cc_norm()
{
    double n[HIP_BK_NM];
    for (int m = 0; m < HIP_BK_NM; ++m) n[m] = (m + 0.5) / hip_leg_scale(m);
    return cudaMemcpyToSymbol(c_cc_norm, n, sizeof(n));
}

// acc[l][a][b] -= sum_q wn[q] J[l][a][q] J[l][b][q]: one warp per (l, a, b).
__global__ void k_bk_cc_contract(BkCTerm c, const double *__restrict__ wn, const double *__restrict__ J)
{
    const int nk = c.n_e - 1, n_nodes = c.n_cc * HIP_BK_CQ;
    const int lane = threadIdx.x & 31;
    const int n_out = (HIP_LMAX + 1) * nk * nk;
    for (int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; o < n_out; o += (gridDim.x * blockDim.x) >> 5) {
        const int l = o / (nk * nk), ab = o - l * nk * nk, a = ab / nk, b = ab - a * nk;
        const double *Ja = J + ((size_t)l * nk + a) * n_nodes, *Jb = J + ((size_t)l * nk + b) * n_nodes;
        double s = 0.0;
        for (int i = lane; i < n_nodes; i += 32) s += wn[i] * Ja[i] * Jb[i];
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) c.acc[o] -= s;
    }
}

cudaError_t hip_bk_cterm(const BkCTerm &c, void *scratch, cudaStream_t st)
{
    cq_nodes();
    BkCQ q;
    for (int i = 0; i < HIP_BK_CQ; ++i) {
        q.x[i] = s_cq_x[i];
        q.w[i] = s_cq_w[i];
    }
    for (int m = 0; m < HIP_BK_NM; ++m) q.inv[m] = 1.0 / (m + 1.0);
    const int n_nodes = c.n_cc * HIP_BK_CQ, nk = c.n_e - 1;
    double *wn = reinterpret_cast<double *>(scratch);
    double *J = wn + n_nodes;
    k_bk_cc_nodes<<<n_nodes / HIP_BK_CN, 256, 0, st>>>(c, q, 1, wn, J);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int n_out = (HIP_LMAX + 1) * nk * nk;
    k_bk_cc_contract<<<(n_out + 7) / 8, 256, 0, st>>>(c, wn, J);
    return cudaGetLastError();
}

// Anisotropic C term: Tc[c][a][b] -= g_c sum_q wn_{L_c}[q] J[l1_c][a][q] J[l2_c][b][q]
// (g_c = (l1 l2 L; 0 0 0)), one warp per (combination, a, b).
__global__ void k_bk_cc_contract_aniso(BkAnisoCTerm t, int nk, int n_nodes, const double *__restrict__ wn,
                                       const double *__restrict__ J, double *__restrict__ Tc)
{
    const int lane = threadIdx.x & 31;
    const int n_out = t.n_comb * nk * nk;
    for (int o = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; o < n_out; o += (gridDim.x * blockDim.x) >> 5) {
        const int ci = o / (nk * nk), ab = o - ci * nk * nk, a = ab / nk, b = ab - a * nk;
        const double *w = wn + (size_t)t.Lidx[ci] * n_nodes;
        const double *Ja = J + ((size_t)t.l1[ci] * nk + a) * n_nodes, *Jb = J + ((size_t)t.l2[ci] * nk + b) * n_nodes;
        double s = 0.0;
        for (int i = lane; i < n_nodes; i += 32) s += w[i] * Ja[i] * Jb[i];
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) Tc[o] -= t.g[ci] * s;
    }
}

size_t hip_bk_cterm_aniso_scratch_bytes(int n_cc, int n_k)
{
    const size_t nodes = (size_t)n_cc * HIP_BK_CQ;
    return sizeof(double) * nodes * (3 + (HIP_LMAX + 1) * (size_t)n_k);
}

cudaError_t hip_bk_cterm_aniso(const BkCTerm &c, const BkAnisoCTerm &t, void *scratch, double *Tc, cudaStream_t st)
{
    cq_nodes();
    BkCQ q;
    for (int i = 0; i < HIP_BK_CQ; ++i) {
        q.x[i] = s_cq_x[i];
        q.w[i] = s_cq_w[i];
    }
    for (int m = 0; m < HIP_BK_NM; ++m) q.inv[m] = 1.0 / (m + 1.0);
    const int n_nodes = c.n_cc * HIP_BK_CQ, nk = c.n_e - 1;
    double *wn = reinterpret_cast<double *>(scratch);  // [3][n_nodes]: the L = 0, 2, 4 moment sets
    double *J = wn + 3 * (size_t)n_nodes;
    k_bk_cc_nodes<<<n_nodes / HIP_BK_CN, 256, 0, st>>>(c, q, 3, wn, J);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int n_out = t.n_comb * nk * nk;
    k_bk_cc_contract_aniso<<<(n_out + 7) / 8, 256, 0, st>>>(t, nk, n_nodes, wn, J, Tc);
    return cudaGetLastError();
}

// ------------------------------------------------------------- finalize -----
// B^ab_l = (-1)^l (2l+1) T^ab_l / (V n_w^3)
//          - delta_l0 (W~^a S^b + W~^b S^a) / (V n_w^2) + 2 delta_l0 W~^a W~^b   (Sec. 4.5)
__global__ void k_bispec_final(const double *__restrict__ partials, int nparts, int nk, int lmax, double L,
                               const double *S1, const double *S, const double *Wt, double *B)
{
    const int tot = (lmax + 1) * nk * nk;
    const double V = L * L * L, nw = S1[0] / V;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += gridDim.x * blockDim.x) {
        double t = 0.0;
        for (int p = 0; p < nparts; ++p) t += partials[(size_t)p * (HIP_LMAX + 1) * nk * nk + i];
        const int l = i / (nk * nk), ab = i - l * nk * nk, aa = ab / nk, bb = ab - aa * nk;
        double b = ((l & 1) ? -1.0 : 1.0) * (2.0 * l + 1.0) * t / (V * nw * nw * nw);
        if (l == 0) b += -(Wt[aa] * S[bb] + Wt[bb] * S[aa]) / (V * nw * nw) + 2.0 * Wt[aa] * Wt[bb];
        B[i] = b;
    }
}

cudaError_t hip_bispec_finalize(const double *partials, int nparts, int nk, int lmax, double L, const double *S1,
                                const double *S, const double *Wt, double *B, cudaStream_t st)
{
    const int tot = (lmax + 1) * nk * nk;
    k_bispec_final<<<(tot + 255) / 256, 256, 0, st>>>(partials, nparts, nk, lmax, L, S1, S, Wt, B);
    return cudaGetLastError();
}

__global__ void k_bispec_sum(const double *__restrict__ partials, int nparts, int nk, int lmax, double *T)
{
    const int tot = (lmax + 1) * nk * nk;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += gridDim.x * blockDim.x) {
        double t = 0.0;
        for (int p = 0; p < nparts; ++p) t += partials[(size_t)p * (HIP_LMAX + 1) * nk * nk + i];
        T[i] = t;
    }
}

cudaError_t hip_bispec_sum(const double *partials, int nparts, int nk, int lmax, double *T, cudaStream_t st)
{
    const int tot = (lmax + 1) * nk * nk;
    k_bispec_sum<<<(tot + 255) / 256, 256, 0, st>>>(partials, nparts, nk, lmax, T);
    return cudaGetLastError();
}

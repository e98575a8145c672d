// Power-spectrum pair pass by Legendre moments of the separation.
//
// The pair sum of Sec. 3 asks, for every bin edge k_e and multipole l, for
//     S_l(k_e) = sum_pairs omega L_l(mu) f_e(r),   f_e(r) = k_e^3 F_l(r k_e),
// (omega = w_i w_j W(r/R0); the edge sums the direct kernel accumulates).  f_e is
// an entire function of r, so on a short interval [c dc, (c+1) dc) it is a
// rapidly converging Legendre series f_e(r) = sum_m a^{e}_{c m} P_m(t), t the
// position in the interval mapped to [-1, 1].  Hence
//     S_l(k_e) = sum_c sum_m a^{e l}_{c m} M^l_{c m},  M^l_{c m} = sum_{pairs in c} omega L_l(mu) P_m(t),
// and the pair loop only accumulates the moments M (HIP_PM_M per bin and l)
// instead of evaluating every edge: O(M n_l) per pair instead of O(n_e n_l).
// The coefficients a come from 24-point Gauss-Legendre projection of f_e in FP64
// (once per call), the final contraction is FP64.  f_e is band-limited (F_l(u)
// is an average of j_l(u y) over y in [0, 1], so its spectrum in r lies in
// [-k_e, k_e]); on an interval of half-width h its m-th Legendre coefficient is
// therefore at most (2m+1) max|j_m(k h)| ~ (2m+1) (k h)^m / (2m+1)!! times the
// spectral mass.  With dc = R0 / n_c (rounded up to 16 significant bits) and
// n_c >= R0 k_max / 4, k h <= 2 and the first neglected term (m = 16) is below
// ~4e-13 of f: exact for both precisions.  The moments are those of the scaled
// polynomials R_m = d_m P_m.  This file holds the FP64 pair passes, the
// coefficients, and the FP64 contraction of both precisions; the FP32 pair pass
// (hip_pm_pairs.cu) sums fewer moments on sub-intervals, which k_pm_coarse turns
// into the interval moments M.
#define HIP_PAIR_UPLOAD hip_upload_coeffs_moments
#include "hip_pair_kernel.cuh"

#include <algorithm>
#include <vector>

#include "hip_moments.h"
#include "hip_pm_search.cuh"

#define HIP_PM_NG 24
#define HIP_PM_MAXW 8      // warps of a CTA: 4 or 8 (template NW, chosen at launch)
#define HIP_PM_TILE 128    // particles per staged tile of a cell
#define HIP_PM_QCAP 64     // queue ring: < 32 pairs plus one ballot round of <= 32
#define HIP_PM_PST 17      // row stride of the P_m(t) table (odd: conflict-free stores by row)
#define HIP_PM_TWORDS (HIP_PM_M * 256)  // most entries of a k_pm_coarse table: [M][S][Q], S Q <= 256

__device__ double g_pm_T[4][HIP_PM_TWORDS];  // k_pm_coarse: (S, Q) = (64, 4), (32, 5), (16, 6), (8, 7)
__constant__ double c_pm_gw[HIP_PM_NG];           // Gauss-Legendre weights on [-1, 1]
__constant__ double c_pm_gx[HIP_PM_NG];           // and nodes
__constant__ double c_pm_P[HIP_PM_NG][HIP_PM_M];  // P_m at the nodes
__constant__ double c_pm_norm[HIP_PM_M];           // (2m+1)/2 / d_m

cudaError_t hip_upload_pm_tables()
{
    void hip_gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w);
    std::vector<double> x, w;
    hip_gauss_legendre(HIP_PM_NG, x, w);
    double P[HIP_PM_NG][HIP_PM_M];
    for (int g = 0; g < HIP_PM_NG; ++g) {
        P[g][0] = 1.0;
        P[g][1] = x[g];
        for (int m = 1; m + 1 < HIP_PM_M; ++m) P[g][m + 1] = ((2.0 * m + 1.0) * x[g] * P[g][m] - m * P[g][m - 1]) / (m + 1.0);
    }
    cudaError_t e = cudaMemcpyToSymbol(c_pm_gw, w.data(), sizeof(double) * HIP_PM_NG);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_pm_gx, x.data(), sizeof(double) * HIP_PM_NG);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_pm_P, P, sizeof(P));
    double norm[HIP_PM_M];
    for (int m = 0; m < HIP_PM_M; ++m) norm[m] = (m + 0.5) / hip_leg_scale(m);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_pm_norm, norm, sizeof(norm));
    // k_pm_coarse tables: R_m on each sub-interval, projected on P_0 .. P_{Q-1} by the
    // same nodes (exact: degree <= 15 + 6) and written in powers of t
    const PmSplit sp[4] = {{64, 4}, {32, 5}, {16, 6}, {8, 7}};
    double leg[8][8] = {{1.0}, {0.0, 1.0}};  // powers of t in P_j
    for (int j = 1; j < 7; ++j)
        for (int k = 0; k <= j + 1; ++k)
            leg[j + 1][k] = ((k ? (2.0 * j + 1.0) * leg[j][k - 1] : 0.0) - j * leg[j - 1][k]) / (j + 1.0);
    std::vector<double> T;
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
        const int S = sp[i].S, Q = sp[i].Q;
        T.assign((size_t)HIP_PM_M * S * Q, 0.0);
        for (int s = 0; s < S; ++s)
            for (int g = 0; g < HIP_PM_NG; ++g) {
                const double tc = ((2 * s + 1) + x[g]) / S - 1.0;
                double p0 = 1.0, p1 = tc;
                for (int m = 0; m < HIP_PM_M; ++m) {
                    for (int j = 0; j < Q; ++j) {
                        const double b = 0.5 * (2.0 * j + 1.0) * w[g] * P[g][j] * p0 * hip_leg_scale(m);
                        for (int q = 0; q <= j; ++q) T[((size_t)m * S + s) * Q + q] += b * leg[j][q];
                    }
                    const double p2 = ((2.0 * m + 3.0) * tc * p1 - (m + 1.0) * p0) / (m + 2.0);
                    p0 = p1;
                    p1 = p2;
                }
            }
        e = cudaMemcpyToSymbol(g_pm_T, T.data(), sizeof(double) * T.size(), sizeof(double) * (size_t)i * HIP_PM_TWORDS);
    }
    return e;
}

// a[((il n_e + e) n_c + c) M + m] = (2m+1)/2 int_{-1}^{1} f_e(r(t)) P_m(t) dt / d_m: the
// coefficients of the scaled polynomials R_m = d_m P_m whose moments the pair pass
// accumulates (batched plans, once per plan).  A block takes HIP_PM_CB intervals of
// one edge: one edge function evaluation per thread, then the projections.  FP64
// runs at 1/64 of the FP32 rate here, so the evaluations are spread over as many
// threads as there are (one thread per (edge, interval) took 340 us whatever the size).
#define HIP_PM_CB 8
__global__ void __launch_bounds__(HIP_PM_CB * HIP_PM_NG) k_pm_coeffs(const double *__restrict__ kedge, int n_e, int n_c,
                                                                    double dc, int n_ell, double *a)
{
    __shared__ double f[3][HIP_PM_CB][HIP_PM_NG];
    const int e = blockIdx.y, c0 = blockIdx.x * HIP_PM_CB;
    const double k = kedge[e], k3 = k * k * k;
    {
        const int ci = threadIdx.x / HIP_PM_NG, g = threadIdx.x - ci * HIP_PM_NG;
        double F[5];
        hip_F_f64<21>((c0 + ci + 0.5 * (1.0 + c_pm_gx[g])) * dc * k, c_coeffs, F);
        const double s = k3 * c_pm_gw[g];
        f[0][ci][g] = s * F[0];
        f[1][ci][g] = s * F[2];
        f[2][ci][g] = s * F[4];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_ell * HIP_PM_CB * HIP_PM_M; i += blockDim.x) {
        const int m = i % HIP_PM_M, ci = i / HIP_PM_M % HIP_PM_CB, il = i / (HIP_PM_M * HIP_PM_CB);
        if (c0 + ci >= n_c) continue;
        double v = 0.0;
        for (int g = 0; g < HIP_PM_NG; ++g) v = fma(f[il][ci][g], c_pm_P[g][m], v);
        a[(((size_t)il * n_e + e) * n_c + c0 + ci) * HIP_PM_M + m] = c_pm_norm[m] * v;
    }
}

// Staging of the FP64 pair pass: tiles of the two cells (shared by the CTA: offsets
// and primary flag packed, weights apart) and, per warp, a ring queue of accepted
// pairs (tile indices only) and the stage of one drain: the pairs in interval
// order with omega L_l, their interval, and P_m(t).
struct __align__(16) PmPt {
    double x, y, z;
    double in;  // 1 if the particle is in the primary range, else 0
};
struct PmTiles {
    PmPt h[HIP_PM_TILE], n[HIP_PM_TILE];
    float hw[HIP_PM_TILE], nw[HIP_PM_TILE];
};
struct __align__(16) PmRow {
    double o0, o2, o4;  // omega L_0, omega L_2, omega L_4
    int c;              // interval
};
struct PmRows {
    PmRow row[32];
    double P[32 * HIP_PM_PST];  // P_m(t) of row s at s HIP_PM_PST + m
};
struct PmStage : PmRows {
    int q[HIP_PM_QCAP];         // queued pairs: home index << 9 | neighbour index << 2 | ordered pairs counted
};

// Doubles of the CTA's moment array for n_cp intervals: [3][M][n_cp].
__host__ __device__ constexpr int hip_pm_words(int n_cp) { return 3 * HIP_PM_M * n_cp; }

// Per-launch constants of the drain: the interval width dc (a 16-bit significand),
// 1 / dc, and 2 / dc and 1 / R0 each as a rounded value plus its residual.
struct PmScale {
    double dc, inv_dc, ihd, ihd_lo, iR, iR_lo;
    __device__ PmScale(double dc_, double R0)
    {
        dc = dc_;
        inv_dc = 1.0 / dc;
        ihd = 2.0 / dc;
        ihd_lo = fma(-dc, ihd, 2.0) / dc;
        iR = 1.0 / R0;
        iR_lo = fma(-R0, iR, 1.0) / R0;
    }
};

// Frame of one work item: the neighbour cell's offset from the home cell.
struct PmShift {
    double x, y, z;
};

// The moment walk of a drain: lane 16 g + m runs over the n staged pairs in
// interval order with register sums and adds a sum to the moment array once per
// interval run (g = 0: l = 0 and l = 4, g = 1: l = 2), unrolled UNR times (the
// batched kernel, short of registers, takes 4, the single-catalog one 8).
template <int MASK, int UNR>
__device__ __forceinline__ void hip_pm_walk(const PmRows &sg, int n, int lane, double *M, int n_cp)
{
    const int m = lane & 15, g = lane >> 4;
    double *Ma = M + (size_t)(g * HIP_PM_M + m) * n_cp;
    double *Mb = M + (size_t)(2 * HIP_PM_M + m) * n_cp;
    const bool use_a = (g == 0) || (MASK & 4);
    const bool use_b = g == 0 && (MASK & 16) != 0;
    double sa = 0.0, sb = 0.0;
    int cur = sg.row[0].c;
#pragma unroll UNR
    for (int s = 0; s < n; ++s) {
        const PmRow r = sg.row[s];
        if (r.c != cur) {  // warp-uniform
            if (use_a) atomicAdd(Ma + cur, sa);
            if (use_b) atomicAdd(Mb + cur, sb);
            sa = 0.0;
            sb = 0.0;
            cur = r.c;
        }
        const double p = sg.P[s * HIP_PM_PST + m];
        sa += (g ? r.o2 : r.o0) * p;
        sb += r.o4 * p;
    }
    if (use_a) atomicAdd(Ma + cur, sa);
    if (use_b) atomicAdd(Mb + cur, sb);
}

// Moments of up to 32 pairs, one per lane (ok: this lane has one; weight product wt):
// M[(il M + m) n_cp + c] += omega L_l P_m(t).  Each lane evaluates its pair (mu, W,
// interval, t); the pairs are then sorted by interval across the warp (bitonic
// network on (interval, lane) keys), lane s tabulates P_m(t) of the s-th pair, and
// finally the lanes run over the moments, walk the sorted pairs with register sums,
// and add a sum to the shared array once per interval run.
template <int MASK, int UNR>
__device__ __forceinline__ void hip_pm_moments(PmRows &sg, bool ok, double ddx, double ddy, double ddz, double wt,
                                               int los, int lane, double *M, int n_cp, int n_c, const PmScale &ps)
{
    int key = ((HIP_PM_NCMAX + 1) << 5) | lane;  // empty lanes sort last
    double t = 0.0, o0 = 0.0, o2 = 0.0, o4 = 0.0;
    if (ok) {
        const double r = sqrt(ddx * ddx + ddy * ddy + ddz * ddz);
        const double mu = (los == 0 ? ddx : (los == 1 ? ddy : ddz)) / r;
        double l2, l4;
        hip_legendre24<double>(mu, l2, l4);
        o0 = wt * hip_W<double>(fma(r, ps.iR_lo, r * ps.iR));
        o2 = o0 * l2;
        o4 = o0 * l4;
        const int c = min((int)(r * ps.inv_dc), n_c - 1);
        const double d = r - c * ps.dc;
        t = fma(d, ps.ihd_lo, d * ps.ihd) - 1.0;
        key = (c << 5) | lane;
    }
    const int n = __popc(__ballot_sync(0xffffffffu, ok));
    if (n == 0) return;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int other = __shfl_xor_sync(0xffffffffu, key, j);
            const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
            key = keep_min ? min(key, other) : max(key, other);
        }
    const int src = key & 31;
    const double ts = __shfl_sync(0xffffffffu, t, src);
    PmRow rw;
    rw.o0 = __shfl_sync(0xffffffffu, o0, src);
    rw.o2 = __shfl_sync(0xffffffffu, o2, src);
    rw.o4 = __shfl_sync(0xffffffffu, o4, src);
    rw.c = key >> 5;
    if (lane < n) {
        double *P = sg.P + lane * HIP_PM_PST;
        double p0 = 1.0, p1 = ts;
        P[0] = p0;
        P[1] = p1;
#pragma unroll
        for (int m = 1; m + 1 < HIP_PM_M; ++m) {
            // the scaled polynomials R_m = d_m P_m (exact recurrence constants)
            const double p2 = hip_leg_alpha<double>(m) * ts * p1 - hip_leg_beta<double>(m) * p0;
            p0 = p1;
            p1 = p2;
            P[m + 1] = p2;
        }
        sg.row[lane] = rw;
    }
    __syncwarp();
    hip_pm_walk<MASK, UNR>(sg, n, lane, M, n_cp);
    __syncwarp();
}

// The n (1..32) queued pairs of the tiles at ring positions head, head + 1, ...
template <int MASK, int UNR>
__device__ __forceinline__ void hip_pm_drain(PmStage &sg, const PmTiles &tl, const PmShift &sh, int los, int head,
                                             int n, int lane, double *M, int n_cp, int n_c, const PmScale &ps,
                                             unsigned long long &cnt)
{
    double ddx = 0.0, ddy = 0.0, ddz = 0.0, wt = 0.0;
    if (lane < n) {
        const int e = sg.q[(head + lane) & (HIP_PM_QCAP - 1)];
        const int il = e >> 9, jl = (e >> 2) & 127, mult = e & 3;
        const PmPt h = tl.h[il], nb = tl.n[jl];
        ddx = (h.x - sh.x) - nb.x, ddy = (h.y - sh.y) - nb.y, ddz = (h.z - sh.z) - nb.z;
        wt = (double)tl.hw[il] * (double)tl.nw[jl] * (double)mult;
        cnt += (unsigned long long)mult;
    }
    hip_pm_moments<MASK, UNR>(sg, lane < n, ddx, ddy, ddz, wt, los, lane, M, n_cp, n_c, ps);
}

// Adds the CTA's moment array into the FP64 totals Mg ([3 M][n_c]) and clears it.
__device__ __forceinline__ void hip_pm_fold(double *M, int n_cp, int n_c, double *Mg)
{
    const int n = 3 * HIP_PM_M * n_cp;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int row = i / n_cp, c = i - row * n_cp;
        const double v = M[i];
        M[i] = 0.0;
        if (c < n_c && v != 0.0) atomicAdd(&Mg[(size_t)row * n_c + c], v);
    }
}

// One work item (home cell, half-shell shift; item counts within the catalog):
// the CTA stages the two cells' tiles, its warps take the home particles, test
// candidates one per lane and queue the accepted ones as tile indices; 32
// queued pairs (and whatever is queued when a tile pair is done) are drained
// into the CTA's moment array M.  Called by all threads of the CTA.
template <int MASK, int NW>
__device__ __forceinline__ void hip_pm_item(const CellList<double> &cl, long long p0, long long p1, int los, int item,
                                            PmTiles &tl, PmStage &sg, double *M, int n_cp, int n_c,
                                            double R0, double dc, unsigned long long &cnt)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const double R0sq = R0 * R0;
    const PmScale ps(dc, R0);
    const int n_c3 = cl.n_c;
    const int c = item / HIP_NSHIFT, q = item - c * HIP_NSHIFT;
    const int cx = c / (n_c3 * n_c3), cy = (c / n_c3) % n_c3, cz = c % n_c3;
    const int dx = c_shift[q][0], dy = c_shift[q][1], dz = c_shift[q][2];
    const int nb = (((cx + dx + n_c3) % n_c3) * n_c3 + (cy + dy + n_c3) % n_c3) * n_c3 + (cz + dz + n_c3) % n_c3;
    PmShift sh;
    double lo;
    hip_cell_shift(cl, cx, dx, sh.x, lo);
    hip_cell_shift(cl, cy, dy, sh.y, lo);
    hip_cell_shift(cl, cz, dz, sh.z, lo);
    const int a0 = cl.cell_start[c], a1 = cl.cell_start[c + 1];
    const int b0 = cl.cell_start[nb], b1 = cl.cell_start[nb + 1];
    const bool self = (q == 0);
    for (int hb = a0; hb < a1; hb += HIP_PM_TILE) {
        const int hn = min(HIP_PM_TILE, a1 - hb);
        __syncthreads();
        for (int i = threadIdx.x; i < hn; i += blockDim.x) {
            const long long oi = cl.idx[hb + i];
            PmPt p;
            p.x = cl.x[hb + i];
            p.y = cl.y[hb + i];
            p.z = cl.z[hb + i];
            p.in = (oi >= p0 && oi < p1) ? 1.0 : 0.0;
            tl.h[i] = p;
            tl.hw[i] = cl.w[hb + i];
        }
        for (int nbs = self ? hb : b0; nbs < b1; nbs += HIP_PM_TILE) {
            const int nn = min(HIP_PM_TILE, b1 - nbs);
            __syncthreads();
            for (int i = threadIdx.x; i < nn; i += blockDim.x) {
                const long long oi = cl.idx[nbs + i];
                PmPt p;
                p.x = cl.x[nbs + i];
                p.y = cl.y[nbs + i];
                p.z = cl.z[nbs + i];
                p.in = (oi >= p0 && oi < p1) ? 1.0 : 0.0;
                tl.n[i] = p;
                tl.nw[i] = cl.w[nbs + i];
            }
            __syncthreads();
            const bool same = self && (nbs == hb);
            int qn = 0;  // queued pairs of this warp (ring head 0 after each partial drain)
            int qh = 0;
            for (int il = warp; il < hn; il += NW) {
                const PmPt h = tl.h[il];
                const double xi = h.x - sh.x, yi = h.y - sh.y, zi = h.z - sh.z;
                const int ini = (int)h.in;
                for (int jb = same ? il + 1 : 0; jb < nn; jb += 32) {
                    const int jl = jb + lane;
                    bool ok = false;
                    int mult = 0;
                    if (jl < nn) {
                        const PmPt p = tl.n[jl];
                        const double ddx = xi - p.x, ddy = yi - p.y, ddz = zi - p.z;
                        const double r2 = ddx * ddx + ddy * ddy + ddz * ddz;
                        mult = ini + (int)p.in;
                        ok = (r2 < R0sq) && (r2 > 0.0) && (mult > 0);
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, ok);
                    if (ok) sg.q[(qh + qn + __popc(bal & lt_mask)) & (HIP_PM_QCAP - 1)] = (il << 9) | (jl << 2) | mult;
                    qn += __popc(bal);
                    if (qn >= 32) {
                        __syncwarp();
                        hip_pm_drain<MASK, 4>(sg, tl, sh, los, qh, 32, lane, M, n_cp, n_c, ps, cnt);
                        qh = (qh + 32) & (HIP_PM_QCAP - 1);
                        qn -= 32;
                    }
                }
            }
            if (qn > 0) {  // the tiles change after this tile pair
                __syncwarp();
                hip_pm_drain<MASK, 4>(sg, tl, sh, los, qh, qn, lane, M, n_cp, n_c, ps, cnt);
            }
        }
    }
}

// The FP64 pair pass of one catalog: the search of the FP32 pass on its records
// (hip_pm_search.cuh), whose candidate test takes every pair within R0 and a rounding
// margin; the drain forms the separation from the FP64 positions and decides.  FP64
// runs at 1/64 of the FP32 rate and a drain's 180 or so instructions are issued
// whether 3 or 32 of its lanes have a pair, so the search's full drains are what
// counts: tiles of cells drained partly filled queues at every tile pair.  5e4
// particles, 3.2 per cell of R0: 1.46 ms with tiles (of the best cell size), 0.74 so;
// 1e5 with 20 per cell: 4.22 / 2.45.  The moment array ([3][M][n_cp], n_cp = n_c
// rounded up to odd so the 16 moments of one interval fall in distinct banks) is
// folded into the FP64 totals at the end.
#define HIP_PM64_WARPS 8  // three CTAs per SM at small n_c
template <int MASK, bool FULL>
__global__ void __launch_bounds__(HIP_PM64_WARPS * 32, 3)
    k_power_moments(const __grid_constant__ PmPairCat cat, const double *__restrict__ x64, double R0, double dc, int *counter)
{
    extern __shared__ __align__(16) unsigned char pm_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_c = cat.n_c, n_cp = n_c | 1;
    PmRows &rows = reinterpret_cast<PmRows *>(pm_raw)[warp];
    PmWarp &sg = reinterpret_cast<PmWarp *>(pm_raw + HIP_PM64_WARPS * sizeof(PmRows))[warp];
    double *M = reinterpret_cast<double *>(pm_raw + HIP_PM64_WARPS * (sizeof(PmRows) + sizeof(PmWarp)));
    for (int i = threadIdx.x; i < hip_pm_words(n_cp); i += blockDim.x) M[i] = 0.0;
    __syncthreads();
    const PmScale ps(dc, R0);
    const double R0sq = R0 * R0;
    unsigned long long cnt = 0;
    int qh = 0, qn = 0;
    // image of a shift table row's neighbour cell: -1, 0, 1 box lengths
    const auto image = [&](int row) {
        const int c = row / 3 + row % 3 - 1;
        return c < 0 ? -cat.L : c >= cat.cl.n_c ? cat.L : 0.0;
    };
    const auto drain = [&](int head, int n) {
        double dx = 0.0, dy = 0.0, dz = 0.0, wt = 0.0;
        bool ok = false;
        if (lane < n) {
            const int e = (head + lane) & (HIP_PP_QCAP - 1), code = sg.qc[e], mult = code >> 27;
            const size_t i = sg.qi[e], j = sg.qj[e];
            dx = (__ldg(x64 + 3 * i) - __ldg(x64 + 3 * j)) - image(code & 511);
            dy = (__ldg(x64 + 3 * i + 1) - __ldg(x64 + 3 * j + 1)) - image((code >> 9) & 511);
            dz = (__ldg(x64 + 3 * i + 2) - __ldg(x64 + 3 * j + 2)) - image((code >> 18) & 511);
            wt = (double)__ldg(&cat.cl.p4[i].w) * (double)__ldg(&cat.cl.p4[j].w) * (double)mult;
            const double r2 = dx * dx + dy * dy + dz * dz;
            ok = r2 < R0sq && r2 > 0.0;
            if (ok) cnt += (unsigned long long)mult;
        }
        hip_pm_moments<MASK, 8>(rows, ok, dx, dy, dz, wt, cat.los, lane, M, n_cp, n_c, ps);
    };
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(counter, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= cat.n_items) break;
        const int blk = item / cat.n_split;
        hip_pp_item<FULL>(cat.cl, cat.k, blk, item - blk * cat.n_split, cat.n_col, cat.n_split / cat.n_col, sg, lane, qh, qn,
                          drain);
    }
    __syncwarp();
    if (qn > 0) drain(qh, qn);
    __syncthreads();
    // this CTA's replica of the totals
    hip_pm_fold(M, n_cp, n_c, cat.G + (size_t)(blockIdx.x % HIP_PM_REPL) * 3 * HIP_PM_M * n_c);
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (lane == 0 && cnt) atomicAdd(cat.npairs, cnt);
}

// The batched FP64 pair pass: all catalogs' work items end to end in one persistent
// launch (l = 0, 2, 4 always).  A CTA's items increase, so it moves through the
// catalogs in order; when it moves on it folds its moments and pair count into
// the catalog it leaves.  The dynamic array is sized for the largest n_c.
template <int NW>
__global__ void __launch_bounds__(NW * 32, 32 / NW)
    k_power_moments_batched(const PmCat *__restrict__ cats, int n_cats, int n_items, int n_c_max, int *counter)
{
    __shared__ PmTiles tl;
    __shared__ PmStage stages[NW];
    __shared__ int s_item;
    extern __shared__ __align__(16) unsigned char pm_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *M = reinterpret_cast<double *>(pm_raw);
    for (int i = threadIdx.x; i < hip_pm_words(n_c_max | 1); i += blockDim.x) M[i] = 0.0;
    unsigned long long cnt = 0;
    int ci = -1;
    __shared__ PmCat cat;  // the current catalog (shared: frees the registers it would take)
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        const bool done = item >= n_items;
        int nci = ci < 0 ? 0 : ci;
        if (!done)
            while (nci < n_cats - 1 && item >= cats[nci].item_end) ++nci;
        if (done || nci != ci) {  // CTA-uniform
            if (ci >= 0) {
                __syncthreads();
                hip_pm_fold(M, cat.n_c | 1, cat.n_c, cat.Mg + (size_t)(blockIdx.x % HIP_PM_REPL) * 3 * HIP_PM_M * cat.n_c);
                unsigned long long c2 = cnt;  // the fold leaves M zero
                for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
                if (lane == 0 && c2) atomicAdd(cat.npairs, c2);
                cnt = 0;
            }
            if (done) break;
            ci = nci;
            __syncthreads();  // the fold above has read the previous catalog
            if (threadIdx.x == 0) cat = cats[ci];
            __syncthreads();
        }
        hip_pm_item<21, NW>(cat.cl, cat.p0, cat.p1, cat.los, item - cat.item_begin, tl, stages[warp], M,
                                   cat.n_c | 1, cat.n_c, cat.R0, cat.dc, cnt);
    }
}

// Interval moments from the FP32 pass's sub-interval moments: R_m on interval c is,
// on sub-interval s, the polynomial sum_q T[m][s][q] t^q (its Legendre projection
// to degree < Q), so M^l_{c m} = sum_s sum_q T[m][s][q] G^l_q[c S + s].  One block of
// 128 threads per (interval, l): thread 8 m + p sums the (s, q) p, p + 8, ...
// (FP64: about 7e5 multiply-adds on 100-interval catalogs, a few microseconds).
__device__ __forceinline__ double hip_pm_coarse(const double *__restrict__ G, int n_c, int S, int Q, int c, int il)
{
    __shared__ double g[256];
    const double *T = g_pm_T[S == 64 ? 0 : S == 32 ? 1 : S == 16 ? 2 : 3];
    const int n_f = n_c * S;
    for (int i = threadIdx.x; i < S * Q; i += 128)
        g[i] = G[((size_t)il * Q + i % Q) * n_f + (size_t)c * S + i / Q];
    __syncthreads();
    const int m = threadIdx.x >> 3, p = threadIdx.x & 7;
    T += m * S * Q;
    double v = 0.0;
#pragma unroll 8
    for (int j = p; j < S * Q; j += 8) v = fma(T[j], g[j], v);  // eight table loads in flight
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;  // M_m, in all eight threads of m
}
// blockIdx.z = catalog
__global__ void __launch_bounds__(128) k_pm_coarse_batched(const PmContractCat *__restrict__ cc, int S, int Q)
{
    const PmContractCat c = cc[blockIdx.z];
    const int ic = blockIdx.x, il = blockIdx.y;
    if (ic >= c.n_c) return;
    const double v = hip_pm_coarse(c.G, c.n_c, S, Q, ic, il);
    if ((threadIdx.x & 7) == 0) c.Mg[((size_t)il * HIP_PM_M + (threadIdx.x >> 3)) * c.n_c + ic] = v;
}

// Single calls: S_l(k_e) = sum_c int rho^l_c(t) f_e(r_c(t)) dt with the pair density
// rho^l_c(t) = sum_m (2m+1)/2 M^l_{c m} P_m(t), by the 24 nodes (the same sums as the
// coefficients a, without forming them).  k_pm_rho: rho at the nodes times their
// weight, [il][c][node], one block of 128 threads per (interval, l); S = 0: M is the
// sum of the FP64 pass's replicas.
__global__ void __launch_bounds__(128) k_pm_rho(const double *__restrict__ src, int n_c, int S, int Q,
                                                double *__restrict__ rho)
{
    __shared__ double M[HIP_PM_M];
    const int c = blockIdx.x, il = blockIdx.y, t = threadIdx.x;
    double v = 0.0;
    if (S)
        v = hip_pm_coarse(src, n_c, S, Q, c, il);
    else
        for (int r = 0; r < HIP_PM_REPL; ++r)
            v += src[((size_t)(r * 3 + il) * HIP_PM_M + (t >> 3)) * n_c + c];
    if ((t & 7) == 0) M[t >> 3] = c_pm_norm[t >> 3] * v;
    __syncthreads();
    if (t < HIP_PM_NG) {
        double s = 0.0;
        for (int m = 0; m < HIP_PM_M; ++m) s = fma(M[m], c_pm_P[t][m], s);
        rho[((size_t)il * n_c + c) * HIP_PM_NG + t] = c_pm_gw[t] * s;
    }
}

// acc[e] += (S_0, S_2, S_4)(k_e) and I(k_e) = int_0^R0 r^2 F_0(r k_e) W(r/R0) dr (for W~^a):
// blockIdx.y = edge, one node per thread: the n_c 24 nodes of rho, then 24 per panel
// of the window's three polynomial pieces (panels no wider than 4 / k_max).
struct PmEdgeArgs {
    double k[HIP_MAX_EDGES];
    double R0, dc, V;
    int n_e, n_c, n_ell, np[3];  // np: panels of [0, R0/2], [R0/2, 3R0/4], [3R0/4, R0]
};
__global__ void __launch_bounds__(128) k_pm_edges(PmEdgeArgs a, const double *__restrict__ rho, double *acc)
{
    const int e = blockIdx.y, n_m = a.n_c * HIP_PM_NG, n_w = (a.np[0] + a.np[1] + a.np[2]) * HIP_PM_NG;
    const int t = blockIdx.x * 128 + threadIdx.x;
    const double k = a.k[e];
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (t < n_m + n_w) {
        const int u = t < n_m ? t : t - n_m;
        int p = u / HIP_PM_NG;
        const double x = c_pm_gx[u - p * HIP_PM_NG], w = c_pm_gw[u - p * HIP_PM_NG];
        double r, h = 0.0;
        if (t < n_m) {
            r = (p + 0.5 * (1.0 + x)) * a.dc;
        } else {
            const int q = p < a.np[0] ? 0 : p < a.np[0] + a.np[1] ? 1 : 2;
            p -= q > 0 ? a.np[0] + (q > 1 ? a.np[1] : 0) : 0;
            h = a.R0 * (q == 0 ? 0.5 : 0.25) / a.np[q];
            r = a.R0 * (q == 0 ? 0.0 : q == 1 ? 0.5 : 0.75) + h * (p + 0.5 * (1.0 + x));
        }
        double F[5];
        hip_F_f64<21>(r * k, c_coeffs, F);
        if (t < n_m) {
            const double k3 = k * k * k;
            for (int il = 0; il < a.n_ell; ++il)
                v[il] = k3 * (il == 0 ? F[0] : il == 1 ? F[2] : F[4]) * rho[(size_t)il * n_m + t];
        } else {
            v[3] = 0.5 * h * w * r * r * F[0] * hip_W<double>(r / a.R0);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
        if ((threadIdx.x & 31) == 0 && v[i] != 0.0) atomicAdd(&acc[4 * e + i], v[i]);
    }
}

// out: P [n_ell][n_k], DD [n_ell][n_k], then two words: pair count, error word.
__global__ void __launch_bounds__(256) k_pm_final(PmEdgeArgs a, const double *__restrict__ acc, const double *S1,
                                                  const unsigned long long *npairs, const int *err, double *out)
{
    const int n_k = a.n_e - 1, n = a.n_ell * n_k;
    const double nw = S1[0] / a.V;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int il = i / n_k, b = i - il * n_k;
        const double lo = a.k[b] * a.k[b] * a.k[b], hi = a.k[b + 1] * a.k[b + 1] * a.k[b + 1];
        const double dd = 3.0 * (acc[4 * (b + 1) + il] - acc[4 * b + il]) / (hi - lo);
        double p = ((il & 1) ? -1.0 : 1.0) * (4.0 * il + 1.0) * dd / (nw * nw * a.V);
        // W~^a = 4 pi int r^2 jbar^a_0 W dr from its two edges
        if (il == 0)
            p -= 4.0 * 3.14159265358979323846 * 3.0 * (hi * acc[4 * (b + 1) + 3] - lo * acc[4 * b + 3]) / (hi - lo);
        out[i] = p;
        out[n + i] = dd;
    }
    if (threadIdx.x == 0) {
        reinterpret_cast<unsigned long long *>(out)[2 * n] = *npairs;
        reinterpret_cast<unsigned long long *>(out)[2 * n + 1] = (unsigned long long)*err;
    }
}

// S[il][e] = sum_c sum_m a[il][e][c][m] Mg[il][m][c] by one 256-thread block,
// written as row[il n_e + e] (one partial row [3][n_e] of the power finalize).
__device__ __forceinline__ void hip_pm_contract_block(const double *__restrict__ a, const double *__restrict__ Mg,
                                                      int n_repl, int n_e, int n_c, int il, int e, double *row)
{
    __shared__ double red[256];
    const double *ae = a + ((size_t)il * n_e + e) * n_c * HIP_PM_M;
    const double *mg = Mg + (size_t)il * HIP_PM_M * n_c;
    const size_t rs = (size_t)3 * HIP_PM_M * n_c;  // replica stride
    double acc = 0.0;
    for (int i = threadIdx.x; i < n_c * HIP_PM_M; i += 256) {
        const int c = i / HIP_PM_M, m = i - c * HIP_PM_M;
        double v = 0.0;
        for (int r = 0; r < n_repl; ++r) v += mg[r * rs + (size_t)m * n_c + c];
        acc = fma(ae[i], v, acc);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) row[il * n_e + e] = red[0];
}

// blockIdx.y = catalog, blockIdx.x = il n_e_max + e
__global__ void __launch_bounds__(256) k_pm_contract_batched(const PmContractCat *__restrict__ cc, int n_e_max)
{
    const PmContractCat c = cc[blockIdx.y];
    const int il = blockIdx.x / n_e_max, e = blockIdx.x - il * n_e_max;
    if (il >= c.n_ell || e >= c.n_e) return;
    hip_pm_contract_block(c.coef, c.Mg, c.n_repl, c.n_e, c.n_c, il, e, c.row);
}

// ------------------------------------------------------------------ host ----
int hip_pm_intervals(double R0, double k_max)
{
    const int n = (int)std::ceil(R0 * k_max / 4.0);
    return n < 8 ? 8 : n;
}

double hip_pm_width(double R0, int n_c)
{
    int ex = 0;
    const double f = std::frexp(R0 / n_c, &ex);  // [0.5, 1)
    return std::ldexp(std::ceil(f * 65536.0) / 65536.0, ex);
}

size_t hip_pm_coef_doubles(int n_e, int n_c) { return (size_t)3 * n_e * n_c * HIP_PM_M; }

cudaError_t hip_pm_coeffs(const double *d_kedges, int n_e, int n_ell, double R0, double k_max, double *coef,
                          cudaStream_t st)
{
    const int n_c = hip_pm_intervals(R0, k_max);
    k_pm_coeffs<<<dim3((n_c + HIP_PM_CB - 1) / HIP_PM_CB, n_e), HIP_PM_CB * HIP_PM_NG, 0, st>>>(
        d_kedges, n_e, n_c, hip_pm_width(R0, n_c), n_ell, coef);
    return cudaGetLastError();
}

size_t hip_pm_rho_doubles(int n_c) { return (size_t)3 * n_c * HIP_PM_NG; }

cudaError_t hip_pm_finish(const PmFinish &f, cudaStream_t st)
{
    PmEdgeArgs a;
    for (int e = 0; e < f.n_e; ++e) a.k[e] = f.k_edges[e];
    for (int e = f.n_e; e < HIP_MAX_EDGES; ++e) a.k[e] = 0.0;
    a.R0 = f.R0;
    a.dc = hip_pm_width(f.R0, f.n_c);
    a.V = f.L * f.L * f.L;
    a.n_e = f.n_e;
    a.n_c = f.n_c;
    a.n_ell = f.n_ell;
    const double km = f.k_edges[f.n_e - 1];
    int nodes = f.n_c;
    for (int q = 0; q < 3; ++q) {
        a.np[q] = std::max(1, (int)std::ceil(f.R0 * (q == 0 ? 0.5 : 0.25) * km / 4.0));
        nodes += a.np[q];
    }
    nodes *= HIP_PM_NG;
    k_pm_rho<<<dim3(f.n_c, f.n_ell), 128, 0, st>>>(f.src, f.n_c, f.S, f.Q, f.rho);
    k_pm_edges<<<dim3((nodes + 127) / 128, f.n_e), 128, 0, st>>>(a, f.rho, f.acc);
    k_pm_final<<<1, 256, 0, st>>>(a, f.acc, f.S1, f.npairs, f.err, f.out);
    return cudaGetLastError();
}

static size_t pm_dyn_smem(int n_c) { return sizeof(double) * (size_t)hip_pm_words(n_c | 1); }

bool hip_pm_applicable(double R0, double k_max)
{
    const int n_c = hip_pm_intervals(R0, k_max);
    if (n_c > HIP_PM_NCMAX) return false;
    const size_t stat = sizeof(PmTiles) + sizeof(PmStage) * HIP_PM_MAXW;
    return pm_dyn_smem(n_c) + stat <= 220 * 1024;
}

// Warps per CTA: 8 when the cells hold enough particles to keep them busy (the
// shared tiles and moment array then serve more warps, raising occupancy), else
// 4 (sparse catalogs: fewer idle warps at each tile pair's barriers).
static int pm_warps(double per_cell) { return per_cell >= 24.0 ? 8 : 4; }

template <typename K>
static cudaError_t pm_grid(K kernel, int threads, size_t dyn, int *grid)
{
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, nb = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, dyn);
    *grid = sms * (nb < 1 ? 1 : nb);
    return cudaSuccess;
}

template <int MASK>
static cudaError_t pm_launch(PmPairCat cat, const double *x64, double R0, bool full, int *counter, cudaStream_t st)
{
    const size_t dyn = pm_dyn_smem(cat.n_c) + HIP_PM64_WARPS * (sizeof(PmRows) + sizeof(PmWarp));
    auto kernel = full ? k_power_moments<MASK, true> : k_power_moments<MASK, false>;
    int grid = 1;
    cudaError_t e = pm_grid(kernel, HIP_PM64_WARPS * 32, dyn, &grid);
    if (e != cudaSuccess) return e;
    hip_pm_items(cat, (long long)grid * HIP_PM64_WARPS, 12);
    cat.k.R0sq = cat.k.reach * cat.k.reach;  // the drain decides
    grid = std::max(1, std::min(grid, (cat.n_items + HIP_PM64_WARPS - 1) / HIP_PM64_WARPS));
    kernel<<<grid, HIP_PM64_WARPS * 32, dyn, st>>>(cat, x64, R0, hip_pm_width(R0, cat.n_c), counter);
    return cudaGetLastError();
}

cudaError_t hip_power_moments(const PmPairCat &cat, const double *x64, int n_ell, double R0, bool full, int *counter,
                              cudaStream_t st)
{
    if (n_ell == 3) return pm_launch<21>(cat, x64, R0, full, counter, st);
    if (n_ell == 2) return pm_launch<5>(cat, x64, R0, full, counter, st);
    return pm_launch<1>(cat, x64, R0, full, counter, st);
}

cudaError_t hip_pm_contract_fine_batched(const PmContractCat *cc, int n_cats, PmSplit sp, int n_c_max, int n_e_max,
                                         cudaStream_t st)
{
    k_pm_coarse_batched<<<dim3(n_c_max, 3, n_cats), 128, 0, st>>>(cc, sp.S, sp.Q);
    k_pm_contract_batched<<<dim3(3 * n_e_max, n_cats), 256, 0, st>>>(cc, n_e_max);
    return cudaGetLastError();
}

template <int NW>
static cudaError_t pm_batched_nw(const PmCat *cats, int n_cats, int n_items, int n_c_max, int *counter,
                                 cudaStream_t st)
{
    const size_t dyn = pm_dyn_smem(n_c_max);
    int grid = 1;
    cudaError_t e = pm_grid(k_power_moments_batched<NW>, NW * 32, dyn, &grid);
    if (e != cudaSuccess) return e;
    k_power_moments_batched<NW><<<grid, NW * 32, dyn, st>>>(cats, n_cats, n_items, n_c_max, counter);
    return cudaGetLastError();
}

cudaError_t hip_power_moments_batched(const PmCat *cats, int n_cats, int n_items, int n_c_max, int *counter,
                                      const PmContractCat *cc, int n_e_max, double per_cell, int warps, cudaStream_t st)
{
    const int nw = warps == 4 || warps == 8 ? warps : pm_warps(per_cell);
    cudaError_t e = nw == 8 ? pm_batched_nw<8>(cats, n_cats, n_items, n_c_max, counter, st)
                            : pm_batched_nw<4>(cats, n_cats, n_items, n_c_max, counter, st);
    if (e != cudaSuccess) return e;
    k_pm_contract_batched<<<dim3(3 * n_e_max, n_cats), 256, 0, st>>>(cc, n_e_max);
    return cudaGetLastError();
}

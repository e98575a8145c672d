// FP32 a_lm pass of the bispectrum (Eq. AC-def binned as in Sec. 4.4): per primary
// p the edge sums E_lm(e) = sum_j w_j W F_l(k_e r) R_lm, differenced into A^a_lm and
// written to X_p, and per pair the C term's moments.
//
// One warp owns one primary at a time.  Its neighbours come from nine rows of three
// cells (z neighbours; float4 records, 32 candidates per test); accepted ones are
// queued as separation vectors, 32 at a time get one lane each for r, W, the 25
// R_lm and the C-term moments, and are then drained with one lane per bin edge.
//
// The drain is the pass: 25 multiply-adds and about 60 more FP32 operations for
// F_0..F_4 per (pair, edge).  F runs on packed pairs of pairs (f32x2: each
// instruction works on pairs 2q and 2q + 1), with the records interleaved so that
// their loads are already packed and the constants stored twice: the FP32 pipe does
// the same work per operation, but at half the issue slots, which is what the
// scalar form ran out of (251 warp instructions per pair at 75 % of the issue slots;
// now 137, the FP32 pipe 52 % active; 5e5 data and 1.5e6 random primaries: 73.8 ->
// 46 ms).  The operations and their order are those of hip_F_b32.  The edge sums
// stay one running sum each: two partial sums per edge would halve their
// instructions too, but round differently (5e-8 of B).  Two packed pairs at a time
// (constants loaded once for four pairs) measured the same on this case and 10 to
// 18 % slower where more groups contain a pair below the polynomial's switch.
//
// C term: 32 Legendre moments of s_p w_j^2 W^2 in the separation per interval
// (scaled R_m, exact recurrence constants), one lane per moment, summed in FP32 over
// the primaries of one work item and then in FP64.
#include <algorithm>

#include "hip_bispec.h"
#include "hip_bk_ylm.cuh"
#include "hip_internal.h"
#include "hip_pair_geom.cuh"

#define BK32_REC 60  // floats of a packed record pair: r, w W, the 25 R_lm (2 each), padding

struct __align__(16) BkWarp32 {
    float4 qa[64];                // ring of accepted neighbours: primary minus neighbour, w_j
    float rec[16][BK32_REC];      // drained pairs 2q, 2q + 1 interleaved
    float pt[32][HIP_BK_NM + 1];  // C-term weight s_p w_j^2 W^2 times R_m(t), m < 32
    float lq[32][2];              // L_2, L_4 of each drained pair's mu (n_L = 3)
    int qc[32];                   // C-term interval of each drained pair
    float2 sh[9];                 // frame shift of neighbour offset d along an axis: [3 axis + d + 1]
    int b0[27], bn[27];           // the 27 neighbour cells: first particle, count
};

// The constants of hip_F_b32, each twice (64-bit operands of the packed operations).
struct BkF32x2 {
    float2 poly[HIP_LMAX + 1][HIP_FB_NPOLY];
    float2 sif[HIP_FB_SIDEG + 1], sig[HIP_FB_SIDEG + 1];
    float2 two_pi_inv, magic, nmagic, pa, pb, pc;        // reduction of the argument
    float2 c16, hp, hp_lo, one, m1;                      // Si
    float2 c2, m2, c3, m4, c7, c8, m15, c11, m52, c52, c75;  // closed forms
};
static __constant__ BkF32x2 c_f2;

cudaError_t hip_upload_bk_alm32()
{
    const HipCoeffs &C = hip_host_coeffs();
    BkF32x2 f;
    auto d = [](float v) { return make_float2(v, v); };
    for (int l = 0; l <= HIP_LMAX; ++l)
        for (int q = 0; q < HIP_FB_NPOLY; ++q) f.poly[l][q] = d(C.fbpoly[l][q]);
    for (int q = 0; q <= HIP_FB_SIDEG; ++q) {
        f.sif[q] = d(C.fbsif[q]);
        f.sig[q] = d(C.fbsig[q]);
    }
    f.two_pi_inv = d(0.636619746685028f);
    f.magic = d(12582912.0f);  // 1.5 2^23: x + magic holds rint(x) in its low bits
    f.nmagic = d(-12582912.0f);
    f.pa = d(-1.5707963705062866f);
    f.pb = d(4.371138828673793e-08f);
    f.pc = d(1.7151245100058819e-15f);
    f.c16 = d(16.0f);
    f.hp = d(HIP_HALF_PI_F);
    f.hp_lo = d(-HIP_HALF_PI_F_LO);
    f.one = d(1.0f);
    f.m1 = d(-1.0f);
    f.c2 = d(2.0f);
    f.m2 = d(-2.0f);
    f.c3 = d(3.0f);
    f.m4 = d(-4.0f);
    f.c7 = d(7.0f);
    f.c8 = d(8.0f);
    f.m15 = d(-15.0f);
    f.c11 = d(11.0f);
    f.m52 = d(-52.5f);
    f.c52 = d(52.5f);
    f.c75 = d(7.5f);
    cudaError_t e = cudaMemcpyToSymbol(c_f2, &f, sizeof(f));
    return e == cudaSuccess ? hip_upload_ylm_norm() : e;
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a)
{
    return make_float2(__uint_as_float(__float_as_uint(a.x) ^ 0x80000000u), __uint_as_float(__float_as_uint(a.y) ^ 0x80000000u));
}

// sin and cos from sin x, cos x and the quadrant in the low bits of n.
__device__ __forceinline__ void bk_quadrant(float sx, float cx, unsigned n, float &s, float &c)
{
    s = (n & 1) ? cx : sx;
    c = (n & 1) ? sx : cx;
    s = __uint_as_float(__float_as_uint(s) ^ ((n & 2u) << 30));
    c = __uint_as_float(__float_as_uint(c) ^ (((n + 1) & 2u) << 30));
}

// F_l(u), l = 0..4, for two arguments (hip_F_b32 on each): the closed forms.
__device__ __forceinline__ void bk_F_closed(float2 u, float2 (&F)[HIP_LMAX + 1])
{
    const float2 n = add2(mul2(u, c_f2.two_pi_inv), c_f2.magic), k = add2(n, c_f2.nmagic);
    float2 x = fma2(k, c_f2.pa, u);
    x = fma2(k, c_f2.pb, x);
    x = fma2(k, c_f2.pc, x);
    float2 s, c;
    bk_quadrant(__sinf(x.x), __cosf(x.x), __float_as_uint(n.x), s.x, c.x);
    bk_quadrant(__sinf(x.y), __cosf(x.y), __float_as_uint(n.y), s.y, c.y);
    const float2 w = make_float2(__fdividef(1.0f, u.x), __fdividef(1.0f, u.y));
    const float2 w2 = mul2(w, w), w3 = mul2(w2, w), t = mul2(c_f2.c16, w2);
    float2 pf = c_f2.sif[HIP_FB_SIDEG], pg = c_f2.sig[HIP_FB_SIDEG];
#pragma unroll
    for (int q = HIP_FB_SIDEG - 1; q >= 0; --q) {
        pf = fma2(pf, t, c_f2.sif[q]);
        pg = fma2(pg, t, c_f2.sig[q]);
    }
    // si = pi/2 - (w (pf c + w pg s) - lo)
    const float2 in = fma2(w, fma2(pf, c, mul2(mul2(w, pg), s)), c_f2.hp_lo);
    const float2 si = fma2(in, c_f2.m1, c_f2.hp);
    const float2 w2c = mul2(w2, c);
    F[0] = fma2(w3, s, neg2(w2c));
    F[1] = fma2(w3, fma2(c_f2.m2, c, c_f2.c2), neg2(mul2(w2, s)));
    F[2] = fma2(w3, fma2(c_f2.c3, si, mul2(c_f2.m4, s)), w2c);
    F[3] = fma2(w2, s, mul2(w3, fma2(c_f2.c7, c, fma2(mul2(c_f2.m15, w), s, c_f2.c8))));
    F[4] = fma2(w3, fma2(fma2(c_f2.m52, w2, c_f2.c11), s, mul2(c_f2.c75, si)), mul2(mul2(w2, fma2(c_f2.c52, w2, c_f2.m1)), c));
}

// The polynomial below HIP_FB_U, replacing F where an argument is there.
__device__ __forceinline__ void bk_F_poly(float2 u, float2 (&F)[HIP_LMAX + 1])
{
    const float2 x = mul2(u, u);
    const bool px = u.x < HIP_FB_U, py = u.y < HIP_FB_U;
    float2 ul = c_f2.one;
#pragma unroll
    for (int l = 0; l <= HIP_LMAX; ++l) {
        float2 a = c_f2.poly[l][HIP_FB_NPOLY - 1];
#pragma unroll
        for (int q = HIP_FB_NPOLY - 2; q >= 0; --q) a = fma2(a, x, c_f2.poly[l][q]);
        a = mul2(a, ul);
        F[l].x = px ? a.x : F[l].x;
        F[l].y = py ? a.y : F[l].y;
        ul = mul2(ul, u);
    }
}

// Constants of a span's catalog.
struct BkConst32 {
    float R0sq, iR, iR_lo, cc_scale, cc_lo;
    float rw;  // s_p of the random primaries
};

// Drains the first n (1..32) neighbours of the ring at head: geometry, harmonics and
// C-term moments one per lane, then the edge sums one lane per edge.
template <int NCH>
__device__ __forceinline__ void bk32_flush(BkWarp32 &sm, const BkConst32 &k, int head, int n, float s_p, int n_cc, int n_L,
                                           float *cm, int lane, const float2 (&kk)[NCH],
                                           const float2 (&kl)[NCH], float (&E)[NCH][HIP_NLM])
{
    if (lane < n) {
        const float4 q = sm.qa[(head + lane) & 63];
        const float dx = q.x, dy = q.y, dz = q.z, wj = q.w;
        const float r = sqrtf(dx * dx + dy * dy + dz * dz);
        const float ir = 1.0f / r;
        const float W = hip_W<float>(fmaf(r, k.iR_lo, r * k.iR));
        float R[HIP_NLM];
        hip_real_ylm<float>(dx * ir, dy * ir, dz * ir, R);
        float *rec = &sm.rec[lane >> 1][lane & 1];
        rec[0] = r;
        rec[2] = wj * W;
#pragma unroll
        for (int i = 0; i < HIP_NLM; ++i) rec[4 + 2 * i] = R[i];
        // C term: interval c of width R0 / n_cc, coordinate t in [-1, 1]
        const float x = fmaf(r, k.cc_lo, r * k.cc_scale);
        const int c = min((int)x, n_cc - 1);
        float t = 2.0f * (x - (float)c) - 1.0f;
        t = t < -1.0f ? -1.0f : (t > 1.0f ? 1.0f : t);
        const float wc = s_p * wj * wj * W * W;
        float p0 = wc, p1 = wc * t;
        sm.pt[lane][0] = p0;
        sm.pt[lane][1] = p1;
#pragma unroll
        for (int m = 1; m < HIP_BK_NM - 1; ++m) {
            const float p2 = hip_leg_alpha<float>(m) * t * p1 - hip_leg_beta<float>(m) * p0;  // R_m = d_m P_m
            sm.pt[lane][m + 1] = p2;
            p0 = p1;
            p1 = p2;
        }
        sm.qc[lane] = c * HIP_BK_NM;
        if (n_L > 1) {  // mu about the line of sight z (even L: the sign of dz does not matter)
            float l2, l4;
            hip_legendre24<float>(dz * ir, l2, l4);
            sm.lq[lane][0] = l2;
            sm.lq[lane][1] = l4;
        }
    } else if (lane == n) {  // n odd: an empty partner for the last pair
        float *rec = &sm.rec[lane >> 1][lane & 1];
        rec[0] = 1.0f / k.iR;
        rec[2] = 0.0f;
        for (int i = 0; i < HIP_NLM; ++i) rec[4 + 2 * i] = 0.0f;
    }
    __syncwarp();
    if (n_L > 1) {  // warp-uniform
        for (int q = 0; q < n; ++q) {
            const float v = sm.pt[q][lane];
            float *o = cm + sm.qc[q] + lane;
            o[0] += v;
            o[n_cc * HIP_BK_NM] += v * sm.lq[q][0];
            o[2 * n_cc * HIP_BK_NM] += v * sm.lq[q][1];
        }
    } else {
        for (int q = 0; q < n; ++q) cm[sm.qc[q] + lane] += sm.pt[q][lane];
    }
    for (int q = 0; 2 * q < n; ++q) {
        const float2 *rec = reinterpret_cast<const float2 *>(sm.rec[q]);
        const float4 rw = *reinterpret_cast<const float4 *>(rec);
        const float2 r = make_float2(rw.x, rw.y), ww = make_float2(rw.z, rw.w);
        constexpr int lof[HIP_NLM + 1] = {0, 1, 1, 1, 2, 2, 2, 2, 2, 3, 3, 3, 3, 3, 3, 3, 4, 4, 4, 4, 4, 4, 4, 4, 4, 4};
#pragma unroll
        for (int t = 0; t < NCH; ++t) {
            const float2 u = fma2(r, kk[t], mul2(r, kl[t]));
            float2 f[HIP_LMAX + 1];
            bk_F_closed(u, f);
            if (__any_sync(0xffffffffu, u.x < HIP_FB_U || u.y < HIP_FB_U)) bk_F_poly(u, f);
#pragma unroll
            for (int l = 0; l <= HIP_LMAX; ++l) f[l] = mul2(ww, f[l]);
#pragma unroll
            for (int i = 0; i < HIP_NLM; i += 2) {
                const float4 R = *reinterpret_cast<const float4 *>(rec + 2 + i);  // R_i, R_{i+1} of both pairs
                E[t][i] = fmaf(f[lof[i]].y, R.y, fmaf(f[lof[i]].x, R.x, E[t][i]));
                if (i + 1 < HIP_NLM) E[t][i + 1] = fmaf(f[lof[i + 1]].y, R.w, fmaf(f[lof[i + 1]].x, R.z, E[t][i + 1]));
            }
        }
    }
    __syncwarp();
}

// One primary: sorted particle p of the data (rnd false) or the randoms.
template <int NCH>
__device__ __forceinline__ void bk32_primary(const BkCat<float> &a, const BkConst32 &k, bool rnd, int p, BkWarp32 &sm,
                                             int &cell, float *cm, int lane, const float2 (&kk)[NCH],
                                             const float2 (&kl)[NCH], float *Xp, float *spp, double (&S)[NCH][3],
                                             unsigned &cnt)
{
    const unsigned cf = __ldg((rnd ? a.rcf : a.pcf) + p);
    const float4 P = __ldg((rnd ? a.r4 : a.p4) + p);
    const bool excluded = cf >> 31;
    const float s_p = excluded ? 0.0f : rnd ? k.rw : P.w;
    if (lane == 0) *spp = s_p;
    if (excluded) return;
    const int nk = a.n_e - 1, n_c = a.data.n_c, c = (int)(cf & 0x7fffffffu);
    if (c != cell) {  // neighbour table of this cell (consecutive primaries mostly share it)
        cell = c;
        const int cx = c / (n_c * n_c), cy = c / n_c % n_c, cz = c % n_c;
        __syncwarp();
        if (lane < 27) {
            int x = cx + lane / 9 - 1, y = cy + lane / 3 % 3 - 1, z = cz + lane % 3 - 1;
            x += x < 0 ? n_c : x >= n_c ? -n_c : 0;
            y += y < 0 ? n_c : y >= n_c ? -n_c : 0;
            z += z < 0 ? n_c : z >= n_c ? -n_c : 0;
            const int nb = (x * n_c + y) * n_c + z, b = __ldg(&a.data.cell_start[nb]);
            sm.b0[lane] = b;
            sm.bn[lane] = __ldg(&a.data.cell_start[nb + 1]) - b;
            if (lane < 9) sm.sh[lane] = __ldg(&a.shift[(lane / 3 == 0 ? cx : lane / 3 == 1 ? cy : cz) * 3 + lane % 3]);
        }
        __syncwarp();
    }
    const unsigned lt = (1u << lane) - 1u;
    const int self = rnd ? -1 : p;
    float E[NCH][HIP_NLM];
#pragma unroll
    for (int t = 0; t < NCH; ++t)
#pragma unroll
        for (int i = 0; i < HIP_NLM; ++i) E[t][i] = 0.0f;
    int qh = 0, qn = 0;
    // The candidate test uses the offset rounded with the cell shift; an accepted
    // neighbour's separation adds the low part (the shift's own and the rounding of
    // p - shift), which is common to all pairs across a periodic face.
    for (int row = 0; row < 9; ++row) {
        const float2 tx = sm.sh[row / 3], ty = sm.sh[3 + row % 3];
        const float ox = P.x - tx.x, oy = P.y - ty.x;
        const int n0 = sm.bn[3 * row], n1 = n0 + sm.bn[3 * row + 1], n2 = n1 + sm.bn[3 * row + 2];
        for (int b = 0; b < n2; b += 32) {
            const int q = b + lane, z = (q >= n0) + (q >= n1);
            const int j = sm.b0[3 * row + z] + q - (z == 0 ? 0 : z == 1 ? n0 : n1);
            const float2 tz = sm.sh[6 + z];
            const float oz = P.z - tz.x;
            bool ok = false;
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q < n2) {
                const float4 N = __ldg(&a.p4[j]);
                d = make_float4(ox - N.x, oy - N.y, oz - N.z, N.w);
                const float r2 = d.x * d.x + d.y * d.y + d.z * d.z;
                ok = (r2 < k.R0sq) && (r2 > 0.0f) && (j != self);
            }
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                d.x += hip_low(P.x, -tx.x, ox) - tx.y;
                d.y += hip_low(P.y, -ty.x, oy) - ty.y;
                d.z += hip_low(P.z, -tz.x, oz) - tz.y;
                sm.qa[(qh + qn + __popc(m & lt)) & 63] = d;
            }
            qn += __popc(m);
            if (qn >= 32) {
                __syncwarp();
                bk32_flush<NCH>(sm, k, qh, 32, s_p, a.n_cc, a.n_L, cm, lane, kk, kl, E);
                cnt += 32;
                qh = (qh + 32) & 63;
                qn -= 32;
            }
        }
    }
    if (qn > 0) {
        __syncwarp();
        bk32_flush<NCH>(sm, k, qh, qn, s_p, a.n_cc, a.n_L, cm, lane, kk, kl, E);
        cnt += qn;
    }
    // A^a_lm = jfac_a (k_{a+1}^3 E_{a+1} - k_a^3 E_a)
#pragma unroll
    for (int t = 0; t < NCH; ++t) {
        const int aa = lane + 32 * t;
        const bool in = aa < nk;
        const float k3 = in ? a.k3[aa] : 0.0f, k3n = in ? a.k3[aa + 1] : 0.0f, jf = in ? a.jfac[aa] : 0.0f;
#pragma unroll
        for (int i = 0; i < HIP_NLM; ++i) {
            const float e = E[t][i];
            float nxt = __shfl_down_sync(0xffffffffu, e, 1);
            if (NCH == 2 && t == 0) {
                const float wrap = __shfl_sync(0xffffffffu, E[NCH - 1][i], 0);
                if (lane == 31) nxt = wrap;
            }
            const float A = jf * (k3n * nxt - k3 * e);
            if (in) Xp[i * nk + aa] = A;
            if (!rnd && (i == 0 || i == 6 || i == 20)) S[t][i == 0 ? 0 : i == 6 ? 1 : 2] += (double)s_p * (double)A;
        }
    }
}

__device__ __forceinline__ void bk32_const(BkConst32 &k, const BkCat<float> &a)
{
    k.R0sq = a.R0 * a.R0;
    k.iR = a.iR;
    k.iR_lo = a.iR_lo;
    k.cc_scale = a.cc_scale;
    k.cc_lo = a.cc_lo;
    k.rw = a.n_rand > 0 ? (float)(-*a.S1 / (double)a.n_rand) : 0.0f;
}

// Spans one after the other, each one's primaries in groups of up to HIP_BK_PRIM from its
// own counter.  A warp's C-term sums over one group sit in FP32 shared memory, are
// added to the warp's FP64 slot after it and to the catalog at the end of the span.
template <int NCH, int NW>
__global__ void __launch_bounds__(NW * 32, 1)
    k_bk_alm32(const BkCat<float> *__restrict__ cats, const BkSpan *__restrict__ spans, int n_spans, int words,
               double *__restrict__ slots, float *__restrict__ X, float *__restrict__ spw, int *counter)
{
    extern __shared__ __align__(16) unsigned char b32_raw[];
    __shared__ BkCat<float> a;
    __shared__ BkConst32 ks;
    __shared__ int bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    BkWarp32 &sm = reinterpret_cast<BkWarp32 *>(b32_raw)[threadIdx.x >> 5];
    float *cm = reinterpret_cast<float *>(b32_raw + (blockDim.x >> 5) * sizeof(BkWarp32)) + (size_t)warp * words;
    double *slot = slots + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * words;  // zero
    for (int i = lane; i < words; i += 32) cm[i] = 0.0f;
    for (int si = 0; si < n_spans; ++si) {
        const BkSpan s = spans[si];
        for (int i = threadIdx.x; i < (int)(sizeof(a) / 4); i += blockDim.x)
            reinterpret_cast<int *>(&a)[i] = reinterpret_cast<const int *>(&cats[s.cat])[i];
        __syncthreads();
        if (threadIdx.x == 0) {
            bk32_const(ks, a);
            bad = a.err[0] | a.err[1];
        }
        __syncthreads();
        if (bad) {  // no primaries: the contraction passes over weights of zero
            for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.g1 - s.g0; i += gridDim.x * blockDim.x)
                spw[s.sp_off + i] = 0.0f;
            __syncthreads();
            continue;
        }
        const BkConst32 k = ks;
        float2 kk[NCH], kl[NCH];
#pragma unroll
        for (int t = 0; t < NCH; ++t) {  // idle lanes repeat the last edge
            const int e = min(lane + 32 * t, a.n_e - 1);
            kk[t] = make_float2(a.k[e], a.k[e]);
            kl[t] = make_float2(a.klo[e], a.klo[e]);
        }
        const int nk = a.n_e - 1;
        double S[NCH][3];
#pragma unroll
        for (int t = 0; t < NCH; ++t) S[t][0] = S[t][1] = S[t][2] = 0.0;
        unsigned cnt_d = 0, cnt_r = 0;  // warp-uniform; a warp sees fewer than 2^32 pairs of a span
        int cell = -1;
        bool did = false;
        for (;;) {
            int it = 0;
            if (lane == 0) it = atomicAdd(counter + si, 1);
            it = __shfl_sync(0xffffffffu, it, 0);
            const int g0 = s.g0 + it * s.prim;
            if (g0 >= s.g1) break;
            did = true;
            for (int g = g0; g < min(g0 + s.prim, s.g1); ++g) {
                const bool rnd = g >= a.n_data;
                const long long o = g - s.g0;
                bk32_primary<NCH>(a, k, rnd, rnd ? g - a.n_data : g, sm, cell, cm, lane, kk, kl, X + s.x_off + o * HIP_NLM * nk,
                                  spw + s.sp_off + o, S, rnd ? cnt_r : cnt_d);
            }
            __syncwarp();
            for (int i = lane; i < a.n_L * a.n_cc * HIP_BK_NM; i += 32) {
                const float v = cm[i];
                if (v != 0.0f) {
                    slot[i] += (double)v;
                    cm[i] = 0.0f;
                }
            }
            __syncwarp();
        }
        if (did)
            for (int i = lane; i < a.n_L * a.n_cc * HIP_BK_NM; i += 32) {
                const double v = slot[i];
                if (v != 0.0) {
                    atomicAdd(&a.cmom[i], v);
                    slot[i] = 0.0;
                }
            }
        if (lane == 0) {
            if (cnt_d) atomicAdd(a.npairs, (unsigned long long)cnt_d);
            if (cnt_r) atomicAdd(a.npairs + 1, (unsigned long long)cnt_r);
        }
        if (a.S && did)
#pragma unroll
            for (int t = 0; t < NCH; ++t)
                for (int l = 0; l < a.n_S; ++l)
                    if (lane + 32 * t < nk && S[t][l] != 0.0) atomicAdd(&a.S[l * nk + lane + 32 * t], S[t][l]);
        __syncthreads();  // the next span overwrites the catalog
    }
}

// ------------------------------------------------------------------ host ----
// Warps per CTA: `want`, or as many as fit with `words` C-term sums each.
static int bk32_warps(int words, int want)
{
    const int room = (232448 - 4096) / (int)(sizeof(BkWarp32) + sizeof(float) * words);
    return std::max(1, std::min(want, room));
}

#define BK32_WARPS_1 16  // one 32-edge chunk per lane: 128 registers
#define BK32_WARPS_2 8   // two: 255

static int bk32_sms()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

size_t hip_bk_alm32_slot_bytes(int words) { return sizeof(double) * (size_t)bk32_sms() * BK32_WARPS_1 * words; }

template <int NCH, int NW>
static cudaError_t launch_alm32(const BkCat<float> *cats, const BkSpan *spans, int n_spans, long long items, int words,
                                double *slots, float *X, float *spw, int *counter, cudaStream_t st)
{
    const int warps = bk32_warps(words, NW);
    const size_t smem = warps * (sizeof(BkWarp32) + sizeof(float) * (size_t)words);
    cudaError_t e = cudaFuncSetAttribute(k_bk_alm32<NCH, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::max(1LL, std::min((long long)bk32_sms(), (items + 3) / 4));
    k_bk_alm32<NCH, NW><<<grid, warps * 32, smem, st>>>(cats, spans, n_spans, words, slots, X, spw, counter);
    return cudaGetLastError();
}

cudaError_t hip_bk_alm32(const BkCat<float> *cats, const BkSpan *spans, int n_spans, long long items, int nk_max,
                         int words, double *slots, float *X, float *spw, int *counter, cudaStream_t st)
{
    if (nk_max <= 31)
        return launch_alm32<1, BK32_WARPS_1>(cats, spans, n_spans, items, words, slots, X, spw, counter, st);
    return launch_alm32<2, BK32_WARPS_2>(cats, spans, n_spans, items, words, slots, X, spw, counter, st);
}

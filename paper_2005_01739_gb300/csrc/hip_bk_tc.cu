// The bispectrum contraction on the Blackwell tensor cores (Sec. 4.4 / 4.5 of
// arXiv:2005.01739):
//
//     T^ab_l += sum_p s_p sum_m A^a_lm(p) A^b_lm(p),
//
// i.e. for each l the Gram-type product X_l diag(s) X_l^T of the per-primary
// accumulators (rows: bins a; columns: primaries p and orders m).
//
// Layout.  The rows (l, a) of all multipoles are stacked: a tile of 128 rows
// holds floor(128 / n_k) whole l blocks (all five for n_k <= 25, two tiles up to
// n_k = 42, three up to 63), so one M = 128 MMA per tile computes every diagonal block (l, l) it
// needs (the off-diagonal blocks come for free and are ignored).  The K dimension
// runs over (p, slot): each primary has 9 slots, slot m + l of row (l, a) holding
// A^a_lm and slots beyond 2l zero, so the diagonal blocks contract exactly over m.
// Slots 0..7 of primary p fill K group p (8 BF16 values, 16 bytes); slot 8 (only
// l = 4 uses it) of primaries 8g .. 8g + 7 fills K group P + g.  A stage of P
// primaries (8 for one tile, 4 for more) is K = 9P rounded up to 16.
//
// Precision: an error-free split in the manner of Ozaki et al.  The tensor core
// rounds its FP32 accumulator at the accumulator's magnitude, and a plain hi/lo
// TF32 split loses about 1e-6 of each stage's sum that way (measured), too much
// for the cancelling data and random primary sums.  Instead each row r of a stage
// is scaled by a power of two 2^e_r above its largest |value| and cut into three
// slices of 8 significant bits, x = (h + m + l) 2^e_r with h, m, l integer
// multiples of 2^-8, 2^-16, 2^-24 (|h| <= 1, |m|, |l| <= 2^-9): x to 2^-25 of the
// row's largest value.  Every slice is exact in BF16, every product of two
// slices is an exact integer multiple of its unit, and a stage's sums of at most
// 72 products stay below 2^24 units, so the three accumulators
//     A0 = h h^T,  A1 = h m^T + m h^T,  A2 = h l^T + l h^T + m m^T
// (separate tensor-memory columns; the dropped terms are below 2^-32 of A0) are
// exact whatever the accumulator's rounding (kind::f16, BF16 operands, FP32
// accumulation); after every unit of work they are added to the CTA's sums in shared
// memory, each an unevaluated sum of two floats (about 48 bits).  Primary weights enter as sqrt|s_p| before the split
// and the sign through the MMA's negate-A bit, so a unit holds primaries of one
// sign (a stage with both signs is issued twice, once per sign, with the other
// primaries zeroed).
//
// Pipeline (one CTA of 16 warps and an issuing one per SM, persistent over a contiguous range of
// stages; a unit is one (stage, sign, tile)): a bulk copy (cp.async.bulk,
// mbarrier completion) brings the next stage's X block into shared memory; four
// threads share row r of the tile (its scale and its slices, written as 16-byte K
// groups in the canonical K-major layout without swizzle: 8-row x 16-byte core
// matrices, 8-row groups 128 bytes apart, K groups 2048 bytes apart) and split
// unit u + 1 into the second slice buffer while the MMAs of unit u run; one
// thread issues the MMAs and commits them to an mbarrier; the warps read the
// accumulators back with tcgen05.ld (warp w owns lanes 32 (w mod 4)..+31, the
// four warps of a lane group split the columns) and add them to the CTA's sums,
// which go to the catalog's FP64 sums (atomics) when the CTA leaves the catalog.  Every wait is bounded (about two seconds); a wait that gives up sets
// bit 0 of *status, stops the CTA's work, and the CTA still waits (bounded) for
// its own MMAs before it frees its tensor memory.
#include <cstdint>
#include <cstdio>

#include "hip_internal.h"
#include "hip_bispec.h"

#define TC_WORK 512         // threads of the 16 warps that split and fold
#define TC_THREADS 544      // and the warp that issues copies and MMAs
#define TC_ROWB 2048        // bytes of one K group (8 bf16) of a 128-row operand
#define TC_WAIT_CYCLES 4000000000LL
#define TC_SEGS 32          // segments cached in shared memory

__device__ __forceinline__ uint32_t tc_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t tc_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(TC_ROWB >> 4) << 16;  // leading dimension (K) byte offset between core matrices
    d |= (uint64_t)(128 >> 4) << 32;      // stride dimension (M/N) byte offset between 8-row groups
    d |= (uint64_t)1 << 46;               // descriptor version of tcgen05
    return d;                             // base offset 0, relative offsets, no swizzle
}

// instruction descriptor: D f32, A and B bf16, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t tc_idesc(int n, bool negate_a)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((negate_a ? 1u : 0u) << 13) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem(bar))
                 : "memory");
}

__device__ __forceinline__ bool tc_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(tc_smem(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait on one phase of an mbarrier; false if it gave up.
__device__ __forceinline__ bool tc_wait(uint64_t *bar, uint32_t parity)
{
    if (tc_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!tc_try(bar, parity))
        if (clock64() - t0 > TC_WAIT_CYCLES) return false;
    return true;
}

// two floats that are exact in BF16 as one packed pair (x in the low half)
__device__ __forceinline__ uint32_t tc_upper(float2 v)
{
    return __byte_perm(__float_as_uint(v.x), __float_as_uint(v.y), 0x7632);
}

struct TcGeom {
    int nk, lpt, G;  // bins, l blocks per 128-row tile, tiles
    int rows[3];     // valid rows of each tile
    int ncol[3];     // N of each tile's MMA (rows rounded up to 16)
};

__device__ __forceinline__ void tc_geom(int nk, TcGeom &g)
{
    g.nk = nk;
    g.lpt = 128 / nk;
    if (g.lpt > HIP_LMAX + 1) g.lpt = HIP_LMAX + 1;
    g.G = (HIP_LMAX + 1 + g.lpt - 1) / g.lpt;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        int nl = HIP_LMAX + 1 - t * g.lpt;
        if (nl > g.lpt) nl = g.lpt;
        if (nl < 0) nl = 0;
        g.rows[t] = nl * nk;
        g.ncol[t] = ((g.rows[t] + 15) / 16) * 16;
    }
}

static int tc_tiles(int nk)
{
    int lpt = 128 / nk;
    if (lpt > HIP_LMAX + 1) lpt = HIP_LMAX + 1;
    return (HIP_LMAX + 1 + lpt - 1) / lpt;
}

// Byte offsets of the dynamic shared memory (from the 1024-byte aligned base):
// two buffers of the three slices of one tile, two staging buffers of a stage's
// X block, the sums as float pairs, three mbarriers.  The same function
// lays out the kernel and sizes (and checks) the launch.
struct TcLayout {
    size_t slice;     // bytes of one slice operand (128 rows x K bf16)
    size_t stg;       // offset of staging buffer 0 (buffer 1 follows after stg_bytes)
    size_t stg_bytes; // bytes of one staging buffer
    size_t rows;      // offset of the sums: nrow (hi, lo) float pairs
    int nrow;         // 5 n_k (n_k + 1) / 2: the upper triangle a <= b of every l, by columns b
    size_t bars;      // offset of the three mbarriers (8-byte aligned)
    size_t total;     // bytes used from the aligned base
};

__host__ __device__ __forceinline__ TcLayout tc_layout(int nk_max, int P)
{
    TcLayout t;
    const int K = ((9 * P + 15) / 16) * 16;
    t.slice = (size_t)128 * K * 2;
    t.stg = 6 * t.slice;
    t.stg_bytes = (size_t)P * HIP_NLM * nk_max * 4;
    t.rows = t.stg + 2 * t.stg_bytes;
    t.nrow = (HIP_LMAX + 1) * (nk_max * (nk_max + 1) / 2);
    t.bars = t.rows + (size_t)8 * t.nrow;
    t.total = t.bars + 3 * 8;
    return t;
}

static size_t tc_smem_bytes(int nk_max, int P) { return tc_layout(nk_max, P).total + 1024; }

#define TC_STATIC 6144  // more than the kernel's static shared memory
// Eight primaries per stage for one tile, else four.  Eight fit up to 41 bins, but a
// row's slices are cut at its largest value in the stage, and a stage of eight cuts the
// smaller ones coarser: 30 bins, 4e4 data, largest difference between two calls (order
// of the sums alone) 2.8e-9 of B, from fours to eights 6.0e-9.
int hip_bk_tc_stage_prims(int nk_max) { return 128 / nk_max >= HIP_LMAX + 1 ? 8 : 4; }

bool hip_bk_tc_supported(int nk_max) { return tc_tiles(nk_max) <= 3; }  // n_k <= 63

// One unit of work: a stage's primaries of one sign, one tile of rows.
struct TcUnit {
    int s, sgn, t;      // stage, sign (+1 / -1), tile
    int si, nk, nv;     // segment, its n_k, valid primaries of the stage
    int slot;           // geometry slot of the segment
};

template <int P>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_bk_contract_tc(const BkSeg *__restrict__ segs, int n_segs, int n_stages, int nk_max, int *status)
{
    extern __shared__ __align__(1024) unsigned char tc_dyn[];
    // operands start on a 1024-byte boundary whatever the toolchain aligns the
    // dynamic shared memory to (the launch asks for 1024 bytes of slack)
    unsigned char *tc_raw = tc_dyn + ((1024u - (tc_smem(tc_dyn) & 1023u)) & 1023u);
    constexpr int K = ((9 * P + 15) / 16) * 16, KG = K / 8;  // K groups of 8 bf16
    constexpr int GPT = (KG + 3) / 4;                          // K groups per thread
    const TcLayout lay = tc_layout(nk_max, P);
    const size_t slice = lay.slice;                            // bytes of one slice operand
    unsigned char *slices = tc_raw;                            // [2 buffers][h, m, l]
    float *stg0 = reinterpret_cast<float *>(tc_raw + lay.stg);
    const int stg_elems = P * HIP_NLM * nk_max;
    // the CTA's sums of the current catalog as unevaluated sums hi + lo of two floats
    // (FP64 arithmetic is slow on this part; two floats carry ~48 bits, more than the
    // folds need).  Element (l, a <= b) at l ntri + b (b + 1) / 2 + a: a warp's lanes
    // hold consecutive a, so they meet no bank twice.
    const int nrow = lay.nrow;
    float2 *rows = reinterpret_cast<float2 *>(tc_raw + lay.rows);
    uint64_t *bars = reinterpret_cast<uint64_t *>(tc_raw + lay.bars);  // copies 0, 1; MMA
    __shared__ uint32_t s_tmem;
    // by stage parity: a stage whose primaries are all excluded is passed over without
    // another barrier, and its flags may still be read while the next one's are written
    __shared__ float s_scale[2][8];
    __shared__ int s_sign[2][8];
    __shared__ BkSeg s_segs[TC_SEGS];  // the first segments of the table, read often
    // geometry of the segments of the units in flight (three: a new one is made while
    // slow warps still fold with the oldest), made once per segment: tiles, and
    // (l << 8) | a of every tile row (-1: padding)
    __shared__ TcGeom s_geo[3];
    __shared__ short s_row[3][3][128];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < n_segs && i < TC_SEGS; i += TC_THREADS) s_segs[i] = segs[i];
    auto SEG = [&](int i) -> const BkSeg & { return i < TC_SEGS ? s_segs[i] : segs[i]; };

    const int per = (n_stages + gridDim.x - 1) / gridDim.x;
    const int s_lo = blockIdx.x * per, s_hi = min(s_lo + per, n_stages);
    const uint32_t ncols = 512u;  // A0, A1, A2 at columns 0, 128, 256
    for (int i = tid; i < nrow; i += TC_THREADS) rows[i] = make_float2(0.f, 0.f);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&s_tmem)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < 3; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&bars[i])));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    bool ok = true;
    int n_commit = 0;

    auto seg_of = [&](int s) {
        int i = 0;
        while (i + 1 < n_segs && s >= SEG(i).stage_end) ++i;
        return i;
    };
    // the issuing thread: bulk copy of stage s's X block into staging buffer b
    auto prefetch = [&](int s, int b) {
        const BkSeg &sg = SEG(seg_of(s));
        const int j = s - sg.stage_begin;
        const int nv = min(P, sg.n_p - j * P);
        // a bulk copy moves a multiple of 16 bytes: the last stage of a segment may
        // read up to 12 bytes past its last primary (the X buffer has slack there)
        const uint32_t bytes = ((uint32_t)nv * HIP_NLM * sg.n_k * 4 + 15u) & ~15u;
        const float *src = reinterpret_cast<const float *>(sg.X) + (size_t)j * P * HIP_NLM * sg.n_k;
        float *dst = stg0 + (size_t)b * stg_elems;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem(&bars[b])), "r"(bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                tc_smem(dst)),
            "l"(src), "r"(bytes), "r"(tc_smem(&bars[b]))
            : "memory");
    };
    int has_pos = 0, has_neg = 0;
    // threads p < P: weight of stage s's primary p, read a stage ahead of its use
    auto weight = [&](int s) {
        const BkSeg &sg = SEG(seg_of(s));
        const int p = (s - sg.stage_begin) * P + tid;
        return p < sg.n_p ? reinterpret_cast<const float *>(sg.sp)[p] : 0.f;
    };
    float w_next = tid < P && s_lo < s_hi ? weight(s_lo) : 0.f;
    // make stage s current: the next stage's copy is started, this one's awaited,
    // its primaries' weights stored (all threads; CTA-uniform outcome).  Its barrier is
    // also the one between the writes before it (slices, folds) and what follows
    auto prepare = [&](int s, int slot) {  // slot >= 0: the segment's geometry goes there first
        if (slot >= 0) {
            TcGeom g;
            tc_geom(SEG(seg_of(s)).n_k, g);
            if (tid == 0) s_geo[slot] = g;
            for (int i = tid; i < 3 * 128; i += TC_THREADS) {
                const int t = i >> 7, r = i & 127, ll = r / g.nk;
                s_row[slot][t][r] = t < g.G && r < g.rows[t] ? (short)(((t * g.lpt + ll) << 8) | (r - ll * g.nk)) : (short)-1;
            }
        }
        if (s + 1 < s_hi && tid == TC_WORK) prefetch(s + 1, (s + 1 - s_lo) & 1);
        if (tid < P) {
            const float v = w_next;
            s_scale[(s - s_lo) & 1][tid] = sqrtf(fabsf(v));
            s_sign[(s - s_lo) & 1][tid] = v > 0.f ? 1 : (v < 0.f ? -1 : 0);
            w_next = s + 1 < s_hi ? weight(s + 1) : 0.f;
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        const uint32_t use = (uint32_t)((s - s_lo) >> 1);
        if (!__syncthreads_and(tc_wait(&bars[(s - s_lo) & 1], use & 1u))) {
            if (tid == 0) atomicOr(status, 1);
            ok = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int sg_p = lane < P ? s_sign[(s - s_lo) & 1][lane] : 0;
        has_pos = __any_sync(0xffffffffu, sg_p > 0);
        has_neg = __any_sync(0xffffffffu, sg_p < 0);
    };
    // the unit after u (u.s < 0: none yet); false when the CTA's stages are done.
    // `synced`: a barrier was passed (a stage was made current)
    bool synced = false;
    auto advance = [&](TcUnit &u) -> bool {
        int s = u.s, pass = u.s < 0 ? -1 : (u.sgn > 0 ? 0 : 1), t = u.t;
        synced = false;
        const int slot0 = u.slot, si0 = u.si;
        for (;;) {
            if (s >= 0 && t + 1 < s_geo[slot0].G) {
                ++t;
            } else {
                // next sign of this stage, or the next stage
                t = 0;
                bool found = false;
                while (!found) {
                    if (s >= 0 && pass == 0 && has_neg) {
                        pass = 1;
                        found = true;
                    } else {
                        s = s < 0 ? s_lo : s + 1;
                        if (s >= s_hi) return false;
                        // a new segment's geometry goes to the next slot
                        const int si = seg_of(s), slot1 = slot0 == 2 ? 0 : slot0 + 1;
                        prepare(s, si != u.si ? slot1 : -1);
                        synced = true;
                        u.si = si;
                        u.slot = si != si0 ? slot1 : slot0;
                        if (!ok) return false;
                        pass = -1;
                        if (has_pos) {
                            pass = 0;
                            found = true;
                        } else if (has_neg) {
                            pass = 1;
                            found = true;
                        }
                    }
                }
                const BkSeg &sg = SEG(u.si);
                u.nk = sg.n_k;
                u.nv = min(P, sg.n_p - (s - sg.stage_begin) * P);
            }
            u.s = s;
            u.sgn = pass == 0 ? 1 : -1;
            u.t = t;
            return true;
        }
    };
    // split unit u into slice buffer sb: four threads per row, K groups q, q + 4, ...
    // K group p < P holds slots 0..7 of primary p, group P + g slot 8 (m = 4 of
    // l = 4) of primaries 8g .. 8g + 7; the rest is zero padding
    auto transform = [&](const TcUnit &u, int sb) {
        const int nk = u.nk, row = tid >> 2, q = tid & 3;
        const int la = s_row[u.slot][u.t][row], l = la >> 8, a = la & 255;  // l = -1: padding
        const float *stg = stg0 + (size_t)((u.s - s_lo) & 1) * stg_elems;
        const float *scale = s_scale[(u.s - s_lo) & 1];
        const int *sign = s_sign[(u.s - s_lo) & 1];
        const float *col = stg + (size_t)(l > 0 ? l * l : 0) * nk + a;  // slot 0 of primary 0
        const size_t pstride = (size_t)HIP_NLM * nk;
        float v[GPT * 8];
        float vmax = 0.f;
#pragma unroll
        for (int j = 0; j < GPT; ++j) {
            const int kg = q + 4 * j;
#pragma unroll
            for (int i = 0; i < 8; ++i) v[8 * j + i] = 0.f;
            if (kg < P) {
                const int p = kg;
                const float w = (p < u.nv && sign[p] == u.sgn) ? scale[p] : 0.f;
                if (w != 0.f && l >= 0) {
                    const float *src = col + p * pstride;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (i <= 2 * l) v[8 * j + i] = src[(size_t)i * nk] * w;
                }
            } else if (kg < P + (P + 7) / 8 && l == HIP_LMAX) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int p = 8 * (kg - P) + i;
                    if (p < P && p < u.nv && sign[p] == u.sgn) v[8 * j + i] = col[p * pstride + 8 * nk] * scale[p];
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) vmax = fmaxf(vmax, fabsf(v[8 * j + i]));
        }
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, 1));
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, 2));
        // 2^e > vmax, from the exponent field (vmax = f 2^e with f in [0.5, 1)):
        // x 2^-e in (-1, 1); e is clamped so that the powers of two below are normal.
        // A row above 2^110 would be cut wrongly, but its own product in A0 leaves
        // FP32's range from 2^64 on
        int e = vmax > 0.f ? (int)((__float_as_uint(vmax) >> 23) & 0xFFu) - 126 : 0;
        e = e < -100 ? -100 : (e > 110 ? 110 : e);
        // slices by adding and subtracting 1.5 2^23 units, units 2^(e-8), 2^(e-16),
        // 2^(e-24): each rounds to the nearest multiple exactly as an integer rounding
        // of the scaled value, without scaling; every slice is exact in BF16, whose
        // bits are then the upper half of the float's
        const float M1 = __uint_as_float((uint32_t)(142 + e) << 23 | 0x400000u);
        const float M2 = __uint_as_float((uint32_t)(134 + e) << 23 | 0x400000u);
        const float M3 = __uint_as_float((uint32_t)(126 + e) << 23 | 0x400000u);
        const float2 m1 = make_float2(M1, M1), n1 = make_float2(-M1, -M1), m2 = make_float2(M2, M2),
                     n2 = make_float2(-M2, -M2), m3 = make_float2(M3, M3), n3 = make_float2(-M3, -M3),
                     neg = make_float2(-1.f, -1.f);
        unsigned char *buf = slices + (size_t)sb * 3 * slice;
#pragma unroll
        for (int j = 0; j < GPT; ++j) {
            const int kg = q + 4 * j;
            if (kg >= KG) break;
            uint32_t h[4], m[4], lo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 x = make_float2(v[8 * j + 2 * i], v[8 * j + 2 * i + 1]);
                const float2 hh = __fadd2_rn(__fadd2_rn(x, m1), n1);
                const float2 r1 = __ffma2_rn(hh, neg, x);
                const float2 mm = __fadd2_rn(__fadd2_rn(r1, m2), n2);
                const float2 r2 = __ffma2_rn(mm, neg, r1);
                const float2 ll = __fadd2_rn(__fadd2_rn(r2, m3), n3);
                h[i] = tc_upper(hh);
                m[i] = tc_upper(mm);
                lo[i] = tc_upper(ll);
            }
            const size_t off = (size_t)kg * TC_ROWB + (size_t)row * 16;
            *reinterpret_cast<uint4 *>(buf + off) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4 *>(buf + slice + off) = make_uint4(m[0], m[1], m[2], m[3]);
            *reinterpret_cast<uint4 *>(buf + 2 * slice + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        asm volatile("fence.proxy.async.shared::cta;");
    };
    // the issuing thread: the MMAs of unit u from slice buffer sb, committed to the MMA
    // barrier (it is held for most of the time the MMAs take)
    auto issue = [&](const TcUnit &u, int sb) {
        if (tid == TC_WORK) {
            const unsigned char *buf = slices + (size_t)sb * 3 * slice;
            const uint32_t ah = tc_smem(buf), am = tc_smem(buf + slice), al = tc_smem(buf + 2 * slice);
            const uint32_t idesc = tc_idesc(s_geo[u.slot].ncol[u.t], u.sgn < 0);
            // the descriptors' start-address field is addr >> 4 in the low bits:
            // a K step adds 2 TC_ROWB >> 4 to it (no carry: addresses < 256 KB)
            const uint64_t dh0 = tc_desc(ah), dm0 = tc_desc(am), dl0 = tc_desc(al);
#pragma unroll
            for (int ks = 0; ks < K / 16; ++ks) {
                const uint64_t off = (uint64_t)ks * (2 * TC_ROWB >> 4);
                const uint32_t acc = ks == 0 ? 0u : 1u;
                const uint64_t dh = dh0 + off, dm = dm0 + off, dl = dl0 + off;
                tc_mma(tmem, dh, dh, idesc, acc);
                tc_mma(tmem + 128u, dh, dm, idesc, acc);
                tc_mma(tmem + 128u, dm, dh, idesc, 1u);
                tc_mma(tmem + 256u, dh, dl, idesc, acc);
                tc_mma(tmem + 256u, dl, dh, idesc, 1u);
                tc_mma(tmem + 256u, dm, dm, idesc, 1u);
            }
            tc_commit(&bars[2]);
        }
        ++n_commit;
    };
    auto wait_mma = [&]() {
        const bool good = tc_wait(&bars[2], (uint32_t)((n_commit - 1) & 1));
        if (!__syncthreads_and(good)) {
            if (tid == 0) atomicOr(status, 1);
            ok = false;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
    };
    // A0 + A1 + A2 of unit u -> the CTA's sums (the unit's MMAs are done)
    auto fold = [&](const TcUnit &u) {
        const TcGeom &g = s_geo[u.slot];
        const short *lar = s_row[u.slot][u.t];
        const int nk = u.nk, R = g.rows[u.t], ntri = nk * (nk + 1) / 2;
        const int r0 = 32 * (warp & 3), gq = warp >> 2;
        if (r0 < R) {  // warp-uniform
            const int la = lar[r0 + lane], l = la >> 8, a = la & 255;  // l = -1: padding
            const int l0 = u.t * g.lpt;  // the tile's first l block
            const int c0 = (((lar[r0] >> 8) - l0) * nk) & ~7;
            const int c1 = min(g.ncol[u.t], ((lar[min(R - 1, r0 + 31)] >> 8) - l0 + 1) * nk);
            float2 *rl = rows + (l > 0 ? l : 0) * ntri + a;
            for (int c = c0 + 8 * gq; c < c1; c += 32) {
                uint32_t v0[8], v1[8], v2[8];
                const uint32_t ta = tmem + ((uint32_t)r0 << 16) + (uint32_t)c;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                    : "=r"(v0[0]), "=r"(v0[1]), "=r"(v0[2]), "=r"(v0[3]), "=r"(v0[4]), "=r"(v0[5]), "=r"(v0[6]),
                      "=r"(v0[7])
                    : "r"(ta));
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                    : "=r"(v1[0]), "=r"(v1[1]), "=r"(v1[2]), "=r"(v1[3]), "=r"(v1[4]), "=r"(v1[5]), "=r"(v1[6]),
                      "=r"(v1[7])
                    : "r"(ta + 128u));
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                    : "=r"(v2[0]), "=r"(v2[1]), "=r"(v2[2]), "=r"(v2[3]), "=r"(v2[4]), "=r"(v2[5]), "=r"(v2[6]),
                      "=r"(v2[7])
                    : "r"(ta + 256u));
                asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int b = c + j - (l - l0) * nk;
                    if (l >= 0 && b >= a && b < nk) {
                        // (hi, lo) += A0 + A1 + A2: A0 by an exact two-sum, the small rest into lo
                        float2 *p = rl + b * (b + 1) / 2;
                        const float2 o = *p;
                        const float x0 = __uint_as_float(v0[j]), sum = o.x + x0, bb = sum - o.x;
                        const float err = (o.x - (sum - bb)) + (x0 - bb);
                        const float rest = o.y + err + (__uint_as_float(v1[j]) + __uint_as_float(v2[j]));
                        const float nh = sum + rest;
                        *p = make_float2(nh, rest - (nh - sum));
                    }
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
    };
    // this CTA's sums -> the segment's FP64 accumulator
    auto flush = [&](int si) {
        __syncthreads();
        const BkSeg &sg = SEG(si);
        const int nk = sg.n_k, ntri = nk * (nk + 1) / 2;
        for (int i = tid; i < (HIP_LMAX + 1) * ntri; i += TC_THREADS) {
            const float2 o = rows[i];
            rows[i] = make_float2(0.f, 0.f);
            const double v = (double)o.x + (double)o.y;
            if (v == 0.0) continue;
            const int l = i / ntri, t = i - l * ntri;
            int b = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
            b += (b + 1) * (b + 2) / 2 <= t ? 1 : (b * (b + 1) / 2 > t ? -1 : 0);
            const int a = t - b * (b + 1) / 2;
            atomicAdd(&sg.acc[((size_t)l * nk + a) * nk + b], v);
            if (a != b) atomicAdd(&sg.acc[((size_t)l * nk + b) * nk + a], v);
        }
        __syncthreads();
    };

    if (s_lo < s_hi && tid == TC_WORK) prefetch(s_lo, 0);
    TcUnit cur;
    cur.s = -1;
    cur.t = 0;
    cur.sgn = 1;
    cur.si = -1;
    cur.nk = nk_max;
    cur.nv = 0;
    cur.slot = 1;
    // Unit u + 1 is split while the MMAs of u run; its own are issued after the barrier
    // of advance(u + 2), past which the other warps go on to split u + 2 at once.  Two
    // barriers a unit: the one of wait_mma (the slices of u + 1 are split, the MMAs of u
    // done), and the one after the fold.
    int sb = 0;
    const bool worker = tid < TC_WORK;
    auto sync = [&]() {
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
    };
    TcUnit nxt = cur;
    bool have = advance(cur), more = false;
    if (have) {
        if (worker) transform(cur, sb);
        sync();
        nxt = cur;
        more = advance(nxt);
        issue(cur, sb);
    }
    while (have && ok) {
        if (more && worker) transform(nxt, sb ^ 1);  // overlaps the MMAs of cur
        wait_mma();
        if (!ok) break;
        if (worker) fold(cur);
        else asm volatile("tcgen05.fence::before_thread_sync;");
        if (!more || nxt.si != cur.si) flush(cur.si);
        if (!more) break;
        sb ^= 1;
        cur = nxt;
        more = advance(nxt);
        if (!ok) break;
        if (!synced) sync();
        issue(cur, sb);
    }
    // wait (bounded) for this CTA's MMAs before freeing tensor memory
    if (n_commit > 0) tc_wait(&bars[2], (uint32_t)((n_commit - 1) & 1));
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

cudaError_t hip_bk_contract_tc(const BkSeg *segs, int n_segs, int n_stages, int nk_max, int *status, int max_grid,
                               cudaStream_t st)
{
    if (!hip_bk_tc_supported(nk_max)) return cudaErrorInvalidValue;
    if (n_stages < 1) return cudaSuccess;
    const int P = hip_bk_tc_stage_prims(nk_max);
    // the layout's alignment requirements, checked before any launch: operands
    // on 1024 bytes (descriptors), bulk-copy destinations and sizes on 16 bytes,
    // mbarriers on 8 bytes, all inside the opt-in shared memory
    const TcLayout lay = tc_layout(nk_max, P);
    int optin = 0, dev0 = 0;
    cudaGetDevice(&dev0);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev0);
    if (lay.slice % 1024 != 0 || lay.stg % 16 != 0 || lay.stg_bytes % 16 != 0 || lay.rows % 8 != 0 ||
        lay.bars % 8 != 0 || tc_smem_bytes(nk_max, P) + TC_STATIC > (size_t)optin)
        return cudaErrorInvalidValue;
    const size_t smem = tc_smem_bytes(nk_max, P);
    cudaError_t e = cudaFuncSetAttribute(P == 8 ? k_bk_contract_tc<8> : k_bk_contract_tc<4>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int grid = sms;
    if (max_grid > 0 && grid > max_grid) grid = max_grid;
    if (grid > n_stages) grid = n_stages;
    const int per = (n_stages + grid - 1) / grid;
    grid = (n_stages + per - 1) / per;  // no CTA without stages
    if (P == 8)
        k_bk_contract_tc<8><<<grid, TC_THREADS, smem, st>>>(segs, n_segs, n_stages, nk_max, status);
    else
        k_bk_contract_tc<4><<<grid, TC_THREADS, smem, st>>>(segs, n_segs, n_stages, nk_max, status);
    return cudaGetLastError();
}

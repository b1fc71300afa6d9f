// ept_build_tc.cu -- the block build (phase 1) on tcgen05 tensor cores.
//
// Algorithm 1 builds D_XX, D_YY and D_XY once (Algorithm 3 entries; the Gaussian
// kernel of Appendix A.1 for MMD).  Here the distinct entries of the pooled upper
// storage are built from the norm expansion d^2 = ||z_i||^2 + ||z_j||^2 - 2 z_i.z_j
// with the Gram term on the tensor cores in split FP16: every pooled row i is scaled
// by its own power of two c_i (so that max_k |c_i z_ik| < 2^14, inside FP16's range;
// exact) and split c_i z_i = hi_i + lo_i (hi = fp16(c z), lo = fp16(c z - hi)); then
//     c_i c_j z_i.z_j ~ hi_i.hi_j + hi_i.lo_j + lo_i.hi_j
// (three MMAs per K-step into one FP32 accumulator in tensor memory; the dropped
// lo_i.lo_j term and the residual of the split are below 2^-21 of each product, so
// the entries are about as accurate as an FP32 Gram), and the epilogue multiplies
// by 1/c_i and 1/c_j (exact).
// The epilogue forms d^2, recomputes cancellation-prone near-duplicate pairs
// (d^2 < tau (||z_i||^2 + ||z_j||^2)) from direct differences (entry_direct), applies sqrt (distances),
// exp(-d^2 / (2 sigma^2)) (Gaussian) or exp(-d / sigma) (Laplacian), forces the
// diagonal to 0 / 1, zeroes padding, and
// writes the FP32 entries into the packed upper blocks.
//
// Tile = 128 rows (half of a 256-row panel I) x 256 columns (panel J >= I, four
// K-blocks); K loop over p in steps of 32 with TMA loads of the four operand tiles
// (A hi/lo 128 x 32, B hi/lo 256 x 32, 64-byte swizzle); two TMEM accumulators so
// the epilogue of one tile overlaps the main loop of the next.  Roles (320
// threads): warp 0 TMA, warp 1 MMA + TMEM owner, warps 2-9 epilogue (two per TMEM
// lane quarter, each taking half of the tile's columns).  Every wait on an mbarrier is bounded as
// in the contraction kernel; the epilogue's named barriers follow from those (half_sync).
//
// What bounds it: up to a few hundred features the epilogue, 32768 entries a tile on
// eight warps, beyond that the tensor pipe.  A thread holds a row, so storing its entries itself
// touches 32 rows with every instruction (a 32 x 32 group took about 300 of the SM's load
// and store wavefronts); a warp now stages the group in shared memory (128-byte
// swizzle, conflict-free 16-byte stores) and one TMA store writes it, two buffers per
// warp.  Three stages of 48 KB (K = 32) leave the 64 KB for that; two of 96 KB did
// not.  The entries are formed in pairs with packed FP32 arithmetic (the same roundings).
// The epilogue also sums the entries it holds: a thread its row (two pairs at once), a warp the columns
// of each group from its buffer, the four warps of a column half through shared memory, the
// two row halves of a panel by two additions to a zeroed FP64 sum (two terms commute).  That
// spares k_blocksums and its pass over every stored entry.
// n = 20,000, p = 100: Gaussian 483 us and 197 for the sums -> 265 without sums, 434 with them; n = 5000,
// p = 200: 43 + 17 -> 38 us, p = 1000 (tensor pipe 70 % busy) 65 + 21 -> 60 us; n = 200, p = 10 (close
// pairs recomputed) 27 + 11 -> 12.5 us.  With few tiles each is shared by several CTAs (build_split).
// Sixteen epilogue warps, a K-block each, issue no more (96 registers spill; 434 -> 447 us).
#include <cuda.h>
#include <cuda_fp16.h>

#include <cstdio>
#include <cstring>

#include "ept_internal.cuh"
#include "ept_tc_common.cuh"

namespace ept {

namespace {

using namespace tc;

constexpr int BM = 128;
constexpr int BN = 256;
constexpr int BK = BUILD_STAGE_K;                     // 32
constexpr int STAGES = 3;
constexpr int A_BYTES = BM * BK * 2;                  // 8 KB
constexpr int B_BYTES = BN * BK * 2;                  // 16 KB
constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;  // 48 KB: A hi, A lo, B hi, B lo
constexpr int OUT_BYTES = 32 * 32 * 4;                // a staged 32 x 32 group of entries
constexpr int NUM_THREADS = 320;   // TMA warp, MMA warp, 8 epilogue warps
constexpr int EPI_THREADS = 256;
// stages | per-epilogue-warp output groups (8 x 2 x 4 KB) | barriers (1 KB) | per-epilogue-warp column norms and
// scales (8 x 1 KB) | per-epilogue-warp column sums (8 x 1 KB) | alignment slack
constexpr int OUT_OFF = STAGES * STAGE_BYTES;
constexpr int BAR_OFF = OUT_OFF + 8 * 2 * OUT_BYTES;
constexpr int COL_OFF = BAR_OFF + 1024;
constexpr int SUM_OFF = COL_OFF + 8 * (PANEL / 2) * 8;
constexpr int SMEM_BYTES = SUM_OFF + 8 * (PANEL / 2) * 8 + 1024;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of the build");
constexpr unsigned long long ERR_WAIT_TMA = 0x201, ERR_WAIT_MMA = 0x202, ERR_WAIT_EPI = 0x203, ERR_DRAIN = 0x205,
                             ERR_INJECTED = 0x2FE;

struct Bars {
    unsigned long long full[STAGES];      // 1 arrival + TMA transaction bytes
    unsigned long long empty[STAGES];     // 1 arrival (tcgen05.commit)
    unsigned long long acc_full[2];       // 1 arrival (tcgen05.commit)
    unsigned long long acc_empty[2];      // 128 epilogue-thread arrivals
    unsigned long long drain;
    uint32_t tmem_base;
    int abort_flag;
};

__device__ __forceinline__ const float *row_ptr(const TestDesc &d, int64_t i) {
    return (i < d.nx) ? d.X + i * d.p : d.Y + (i - d.nx) * d.p;
}

// Squared norm of a row by one warp, lane l taking elements 2l, 2l + 1 of each 64 and the lanes' sums added in
// FP64: for the rows that the pairs of k_split_rows leave open, and in the order that decides whether a row near
// FP32's limit overflows within a lane (NaN) or only in the rounding (inf).
__device__ __noinline__ double row_norm_by_warp(const float *z, int64_t p, int lane) {
    NormSum sum;
    for (int64_t k = 2 * lane; k < p; k += 64) {
        #pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float v = (k + j < p) ? z[k + j] : 0.f;
            sum.add(isfinite(v) ? v : 0.f);
        }
    }
    double acc = (double)sum.h + (double)sum.l;
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    return acc;
}

// Pooled row i of a test -> FP16 hi / lo parts of c_i z_i (zero padding up to the
// test's p_pad), the inverse scale 1/c_i, and the squared norm of the unscaled row
// (each lane's as an FP32 pair, NormSum; the lanes' pairs are added the same way wherever
// their error bound leaves one FP32 result, else in FP64: the norm is the one that the FP64
// sum gives).
// c_i = 2^k with
// max |c_i z_i| < 2^14, k clamped to [-60, 60] so that 1/c_i 1/c_j stays a normal
// FP32 number (rows above 2^74 would overflow the FP32 norms in any case).
// Non-finite inputs are counted, once a row.
//
// L lanes per row, 4 elements of it a lane and step (16 bytes read, 8 bytes written to each part; element by
// element where a row is not 16-byte aligned); the first KEEP steps stay in registers between the maximum and
// the split, so that a row of up to 16 L elements is read once.  A warp's fixed work (finding the test, scale,
// reductions: with an FP64 tree and one row a warp about 250 SM cycles, half of them FP64) was what bounded it:
// four rows a warp share it, and the pairs are added as pairs.  500 tests of 400 x 100 (212 MB of traffic,
// 31 us at the copy rate): 148 -> 57 us; 512 tests of up to 4,000 x 500: 772 -> 533 us.
template <int L>
__global__ void __launch_bounds__(256) k_split_rows(const Batch bt) {
    constexpr int R = 32 / L, KEEP = 4;
    constexpr int STEP = 4 * L;
    const int lane = threadIdx.x & 31, sub = lane % L;
    if (bt.build_sums) {   // the column sums that the build adds to
        const int64_t threads = (int64_t)gridDim.x * blockDim.x;
        for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < bt.nblk_total * KB; k += threads)
            bt.colpart[k] = 0.0;
    }
    const int64_t gr = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * R + lane / L;
    const bool row = gr < bt.nrows_total;   // every lane stays for the warp's shuffles
    const int t = row ? find_test(bt.pre.rows, bt.n_tests, gr) : 0;
    const TestDesc &d = bt.desc[t];
    const int64_t i = gr - d.row0;
    const int p = (row && i < d.n) ? (int)d.p : 0, p_pad = row ? (int)d.p_pad : 0;   // padding rows: zeros
    const float *z = p ? row_ptr(d, i) : nullptr;
    const bool vec = (p & 3) == 0 && ((uintptr_t)z & 15) == 0;   // 16-byte loads; else element by element
    auto load = [&](int k) -> float4 {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec) {
            if (k < p) v = __ldg(reinterpret_cast<const float4 *>(z + k));
        } else {
            if (k < p) v.x = z[k];
            if (k + 1 < p) v.y = z[k + 1];
            if (k + 2 < p) v.z = z[k + 2];
            if (k + 3 < p) v.w = z[k + 3];
        }
        return v;
    };
    uint32_t mx = 0;
    bool bad = false;
    auto take_max = [&](float4 v) {
        #pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t m = __float_as_uint((&v.x)[j]) & 0x7FFFFFFFu;
            if (m < 0x7F800000u) mx = max(mx, m);
            else bad = true;
        }
    };
    float4 keep[KEEP];
    #pragma unroll
    for (int q = 0; q < KEEP; ++q) keep[q] = load(4 * sub + q * STEP);
    #pragma unroll
    for (int q = 0; q < KEEP; ++q)
        if (q * STEP < p) take_max(keep[q]);
    for (int k = 4 * sub + KEEP * STEP; k < p; k += STEP) take_max(load(k));
    #pragma unroll
    for (int off = L / 2; off; off >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    const uint32_t bads = __ballot_sync(0xFFFFFFFFu, bad) >> (lane - sub) & (uint32_t)((1ull << L) - 1);
    if (bads && sub == 0) atomicAdd(&bt.ctr[t].nonfinite, 1ull);
    // 2^(e - 1) <= max < 2^e; below the normal range the clamp takes over
    int k2 = mx ? 14 - ((int)(mx >> 23) - 126) : 0;
    k2 = k2 < -60 ? -60 : (k2 > 60 ? 60 : k2);
    const float c = __uint_as_float((uint32_t)(127 + k2) << 23);
    __half *zh = (__half *)bt.Zh + gr * bt.p_stride, *zl = (__half *)bt.Zl + gr * bt.p_stride;
    NormSum sum;
    auto split = [&](int k, float4 v4) {
        __half2 h[2], l[2];
        #pragma unroll
        for (int j = 0; j < 2; ++j) {
            float v0 = (&v4.x)[2 * j], v1 = (&v4.x)[2 * j + 1];
            if (!isfinite(v0)) v0 = 0.f;
            if (!isfinite(v1)) v1 = 0.f;
            sum.add(v0);
            sum.add(v1);
            const float w0 = v0 * c, w1 = v1 * c;
            h[j] = __floats2half2_rn(w0, w1);
            const float2 hf = __half22float2(h[j]);
            l[j] = __floats2half2_rn(w0 - hf.x, w1 - hf.y);
        }
        *reinterpret_cast<uint2 *>(zh + k) = *reinterpret_cast<const uint2 *>(h);
        *reinterpret_cast<uint2 *>(zl + k) = *reinterpret_cast<const uint2 *>(l);
    };
    #pragma unroll
    for (int q = 0; q < KEEP; ++q)
        if (4 * sub + q * STEP < p_pad) split(4 * sub + q * STEP, keep[q]);
    for (int k = 4 * sub + KEEP * STEP; k < p_pad; k += STEP) split(k, load(k));
    #pragma unroll
    for (int off = L / 2; off; off >>= 1) {
        const float oh = __shfl_xor_sync(0xFFFFFFFFu, sum.h, off), ol = __shfl_xor_sync(0xFFFFFFFFu, sum.l, off);
        sum.merge(oh, ol);
    }
    // not decided by the bound (one row in 2^12 of 100 features, one in 2^10 of 1,000), or near FP32's limit
    // (past it within a lane): once more, by the whole warp.  A lane has at most p / L + 4 elements.
    float norm;
    const bool sure = sum.rounded((float)(p / L + 10), norm);
    uint32_t open = __ballot_sync(0xFFFFFFFFu, sub == 0 && !(sure && norm <= 1e38f));
    while (open) {
        const int src = __ffs(open) - 1;
        open &= open - 1;
        const float *zr = (const float *)__shfl_sync(0xFFFFFFFFu, (unsigned long long)z, src);
        const double a = row_norm_by_warp(zr, __shfl_sync(0xFFFFFFFFu, p, src), lane);
        if (lane - sub == src) norm = (float)a;
    }
    if (row && sub == 0) {
        bt.norms[gr] = norm;
        bt.iscale[gr] = __uint_as_float((uint32_t)(127 - k2) << 23);
    }
}

// Two FP32 values in one register pair: packed arithmetic with the scalar operations' roundings.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &x, float &y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// (h, l) += v on two sums at once, each an unevaluated pair (TwoSum, the rounding error kept in l)
__device__ __forceinline__ void pair_add2(f32x2 &h, f32x2 &l, f32x2 v) {
    const f32x2 s = add2(h, v), bb = sub2(s, h);
    l = add2(l, add2(sub2(h, sub2(s, bb)), sub2(v, bb)));
    h = s;
}
// the two sums added: the pair's value
__device__ __forceinline__ void pair_join(f32x2 h, f32x2 l, float &hs, float &ls) {
    float h0, h1, l0, l1, e;
    unpack2(h, h0, h1);
    unpack2(l, l0, l1);
    two_sum(h0, h1, hs, e);
    ls = (l0 + l1) + e;
}

// Barriers of the four warps that share a half of the tile's columns: 0, before a tile's column
// sums are written (the last tile's are read); 1, when they are.  They have no limit of their own: each warp
// takes both for every item that needs sums, also after it has given up, and between two of them
// only bounded waits, so the longest wait at one is the other warps' bounded wait on the accumulator.
__device__ __forceinline__ void half_sync(int half, int which) {
    if (half == 0 && which == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else if (half == 0) asm volatile("bar.sync 2, 128;" ::: "memory");
    else if (which == 0) asm volatile("bar.sync 3, 128;" ::: "memory");
    else asm volatile("bar.sync 4, 128;" ::: "memory");
}
// exp_cw of two arguments x in [-87, 0] (its operations in its order; outside the
// range the caller patches the entry)
__device__ __forceinline__ void exp_cw2(f32x2 x, float &y0, float &y1) {
    const f32x2 t = fma2(x, pack2(1.44269504f, 1.44269504f), pack2(12582912.f, 12582912.f));
    const f32x2 nk = fma2(t, pack2(-1.f, -1.f), pack2(12582912.f, 12582912.f));   // -k, exact
    f32x2 r = fma2(nk, pack2(0.693359375f, 0.693359375f), x);
    r = fma2(nk, pack2(-2.12194440e-4f, -2.12194440e-4f), r);
    f32x2 q = pack2(2.48015873e-5f, 2.48015873e-5f);
    q = fma2(q, r, pack2(1.98412698e-4f, 1.98412698e-4f));
    q = fma2(q, r, pack2(1.38888889e-3f, 1.38888889e-3f));
    q = fma2(q, r, pack2(8.33333333e-3f, 8.33333333e-3f));
    q = fma2(q, r, pack2(4.16666667e-2f, 4.16666667e-2f));
    q = fma2(q, r, pack2(1.66666667e-1f, 1.66666667e-1f));
    q = fma2(q, r, pack2(0.5f, 0.5f));
    q = fma2(q, r, pack2(1.f, 1.f));
    q = fma2(q, r, pack2(1.f, 1.f));
    float t0, t1;
    unpack2(t, t0, t1);
    const uint32_t bias = (127u - 0x4B400000u) << 23;   // (k + 127) << 23, k = low bits of t
    const f32x2 sc = pack2(__uint_as_float((__float_as_uint(t0) << 23) + bias),
                           __uint_as_float((__float_as_uint(t1) << 23) + bias));
    unpack2(mul2(q, sc), y0, y1);
}

// One row's 32 entries of a column group from the Gram accumulator v (scaled by
// c_i c_j): d^2 = n_i + n_j - 2 G_ij, the entry for kernel kind KERN (0 distance,
// 1 Gaussian, 2 Laplacian; the approximate square root is within 2^-22 of the
// exact one, below the split Gram's own error).  cg: per pair of columns, the norms and
// the inverse scales.  True when some entry needs group_patch: one with d^2 < tau (n_i
// + n_j), or a kernel value of 0.
template <int KERN>
__device__ __forceinline__ bool group_entries(const uint32_t (&v)[32], const float4 *cg, float ni, float si,
                                              float tau, float neg_inv_2s2, float inv_sigma, float (&out)[32]) {
    const f32x2 ni2 = pack2(ni, ni), si2 = pack2(si, si), tau2 = pack2(-tau, -tau), two = pack2(-2.f, -2.f);
    const float f = KERN == 1 ? neg_inv_2s2 : -inv_sigma;
    const f32x2 f2 = pack2(f, f);
    float close = 1.f, big = 0.f;   // < 0: some entry to recompute; the largest argument of exp
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        const float4 c = cg[e / 2];
        // exact rescaling by powers of two, then n_i + n_j - 2 G_ij with one rounding
        const f32x2 g = mul2(mul2(pack2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), si2), pack2(c.z, c.w));
        const f32x2 sn = add2(ni2, pack2(c.x, c.y));
        float d0, d1;
        unpack2(fma2(g, two, sn), d0, d1);
        d0 = fmaxf(0.f, d0);
        d1 = fmaxf(0.f, d1);
        float q0, q1;
        unpack2(fma2(sn, tau2, pack2(d0, d1)), q0, q1);   // tau (n_i + n_j) is exact, so the sign is
        close = fminf(close, fminf(q0, q1));
        if (KERN != 1) {
            asm("sqrt.approx.f32 %0, %1;" : "=f"(d0) : "f"(d0));
            asm("sqrt.approx.f32 %0, %1;" : "=f"(d1) : "f"(d1));
        }
        if (KERN == 0) {
            out[e] = d0;
            out[e + 1] = d1;
        } else {
            big = fmaxf(big, fmaxf(d0, d1));
            exp_cw2(mul2(pack2(d0, d1), f2), out[e], out[e + 1]);
        }
    }
    return close < 0.f || (KERN != 0 && !(big * f > -87.f));
}

// The rare rest of a group: kernel values that are 0, and the bit mask of the entries
// that need the recomputation.
__device__ __forceinline__ uint32_t group_patch(const uint32_t (&v)[32], const float4 *cg, float ni, float si,
                                                float tau, int kern, float neg_inv_2s2, float inv_sigma,
                                                float (&out)[32]) {
    uint32_t fix = 0;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        const float4 c = cg[e / 2];
        const float g = (__uint_as_float(v[e]) * si) * (e & 1 ? c.w : c.z), sn = ni + (e & 1 ? c.y : c.x);
        const float d2 = fmaxf(0.f, fmaf(-2.f, g, sn));
        fix |= (d2 < tau * sn) ? (1u << e) : 0u;
        if (kern != 0) {
            float x = d2;
            if (kern == 2) asm("sqrt.approx.f32 %0, %1;" : "=f"(x) : "f"(d2));
            x *= kern == 1 ? neg_inv_2s2 : -inv_sigma;
            if (!(x > -87.f)) out[e] = 0.f;
        }
    }
    return fix;
}

// The squared distance of two rows in FP64, feature by feature.
__device__ __forceinline__ double square_sum_fp64(const float *zi, const float *zj, int64_t p) {
    double sq = 0.0;
#pragma unroll 1
    for (int64_t k = 0; k < p; ++k) {
        const double df = (double)zi[k] - (double)zj[k];
        sq = fma(df, df, sq);
    }
    return sq;
}

// The entry of two rows by direct differences: the FP32 number that the squared distance summed in FP64
// gives.  It is summed as an FP32 pair instead, wherever the pair's error bound leaves one result: GB300's FP64
// rate is so low that eight warps' FP64 sums of 10 features took 8,000 cycles.  Eight loads of each row are in
// flight.  Left to FP64: sums near the ends of FP32's range, and the entries that the bound does not decide (one
// in 2^14 of 10 features, one in 2^8 of 1,000); equal rows are 0 in either.
__device__ __forceinline__ float entry_direct(const float *zi, const float *zj, int64_t p, int kern,
                                              float neg_inv_2s2, float inv_sigma) {
    SquareSum sum;
    float far = 0.f;
#pragma unroll 1
    for (int64_t k = 0; k < p; k += 8) {
        float a[8], b[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {   // past the end: equal values, which add nothing
            a[e] = k + e < p ? zi[k + e] : 0.f;
            b[e] = k + e < p ? zj[k + e] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            far = fmaxf(far, fabsf(a[e] - b[e]));
            sum.add(a[e], b[e]);
        }
        sum.renormalise();
    }
    const float t = sum.h + sum.l;
    if (far == 0.f) return (float)entry_from_d2(0.0, kern, neg_inv_2s2, inv_sigma);
    if (t > 1e-20f && t < 1e30f) {
        float out;
        if (kern == 0) {
            if (sum.root(p, out)) return out;
        } else {
            // a kernel value's relative error: its exponent's error, and 2^-50 of the exponent and of itself
            // for the FP64 operations on either way
            const double v = entry_from_d2((double)sum.h + (double)sum.l, kern, neg_inv_2s2, inv_sigma);
            const float x = kern == 1 ? -t * neg_inv_2s2 : sqrtf(t) * inv_sigma;
            const float rel = x * (float)(41 * p + 64) * 3.5527137e-15f + (x + 1.f) * 8.8817842e-16f;
            const double err = v * (double)(rel * 1.001f);
            out = (float)(v - err);
            if (out == (float)(v + err)) return out;
        }
    }
    return (float)entry_from_d2(square_sum_fp64(zi, zj, p), kern, neg_inv_2s2, inv_sigma);
}

// The entries of row i (this lane's) in columns j0 + e, e in `fix`, directly into the staged group.  Not inlined: with
// it in the group loop the loop's registers spill (n = 20,000, p = 100: 745 us for the build phase, 870 with it).
__device__ __noinline__ void fix_entries(uint32_t fix, uint8_t *buf, const TestDesc &d, int64_t i, int64_t j0) {
    const int lane = threadIdx.x & 31;
    const int64_t p = d.p;
    while (fix) {
        const int e = __ffs(fix) - 1;
        fix &= fix - 1u;
        const int64_t j = j0 + e;
        const float *zi = row_ptr(d, i), *zj = row_ptr(d, j);
        *reinterpret_cast<float *>(buf + lane * 128 + (((e >> 2) ^ (lane & 7)) << 4) + (e & 3) * 4) =
            entry_direct(zi, zj, p, d.kern, d.neg_inv_2s2, d.inv_sigma);
    }
}

template <bool SHARED>   // tiles shared by several CTAs (build_split); whole ones keep their constants
__global__ void __launch_bounds__(NUM_THREADS, 1)
    k_build_tc(const __grid_constant__ CUtensorMap tm_ah, const __grid_constant__ CUtensorMap tm_al,
               const __grid_constant__ CUtensorMap tm_bh, const __grid_constant__ CUtensorMap tm_bl,
               const __grid_constant__ CUtensorMap tm_d, const Batch bt, const int parts_log) {
    const int split = SHARED ? parts_log : 0;
    Counters *ctr = bt.ctr;   // bounded-wait errors are recorded in test 0's counters
    const unsigned long long wait_ns = bt.wait_ns ? bt.wait_ns : WAIT_NS;   // limit of every bounded wait
    const int nitems = (int)bt.ntiles << split;   // item t: tile t >> split, part t mod 2^split of its columns
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    Bars *bars = reinterpret_cast<Bars *>(smem + BAR_OFF);
    volatile int *abort_flag = &bars->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(su32(&bars->full[s]), 1);
            mbar_init(su32(&bars->empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(su32(&bars->acc_full[a]), 1);
            mbar_init(su32(&bars->acc_empty[a]), EPI_THREADS);
        }
        mbar_init(su32(&bars->drain), 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                         su32(&bars->tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem_base = bars->tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int armed[STAGES];
            for (int s2 = 0; s2 < STAGES; ++s2) armed[s2] = -1;
            bool ok = true;
            for (int t = blockIdx.x; t < nitems && ok; t += gridDim.x) {
                const Tile tile = bt.tiles[t >> split];
                const int64_t row0 = bt.desc[tile.t].row0;
                const int rowA = (int)row0 + tile.I * PANEL + tile.h * BM;
                const int rowB = (int)row0 + tile.J * PANEL + (t & ((1 << split) - 1)) * (BN >> split);
                const int kblocks = (int)((bt.desc[tile.t].p + BK - 1) / BK);
                for (int kk = 0; kk < kblocks; ++kk) {
                    if (!mbar_wait(su32(&bars->empty[stage]), phase ^ 1u, abort_flag, ctr, ERR_WAIT_TMA, wait_ns)) {
                        ok = false;
                        break;
                    }
                    const uint32_t full = su32(&bars->full[stage]);
                    mbar_arrive_tx(full, 2 * A_BYTES + ((2 * B_BYTES) >> split));
                    uint8_t *st = smem + stage * STAGE_BYTES;
                    tma_load_2d(su32(st), &tm_ah, kk * BK, rowA, full);
                    tma_load_2d(su32(st + A_BYTES), &tm_al, kk * BK, rowA, full);
                    tma_load_2d(su32(st + 2 * A_BYTES), &tm_bh, kk * BK, rowB, full);   // boxes of BN >> split rows
                    tma_load_2d(su32(st + 2 * A_BYTES + B_BYTES), &tm_bl, kk * BK, rowB, full);
                    armed[stage] = (int)phase;
                    if (++stage == STAGES) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            // drain: wait (bounded) for the copies under way, also where all were armed: another
            // role may give up before they have arrived
            for (int s2 = 0; s2 < STAGES; ++s2) {
                if (armed[s2] < 0) continue;
                const unsigned long long t0 = gtimer();
                while (!mbar_try(su32(&bars->full[s2]), (uint32_t)armed[s2])) {
                    if (gtimer() - t0 > wait_ns) {
                        atomicCAS(&ctr->err_code, 0ull, ERR_DRAIN);
                        break;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            const uint32_t idesc = idesc_f16_f32(BM, BN >> split);
            bool ok = true;
            for (int t = blockIdx.x; t < nitems && ok; t += gridDim.x) {
                const int kblocks = (int)((bt.desc[bt.tiles[t >> split].t].p + BK - 1) / BK);
                if (!mbar_wait(su32(&bars->acc_empty[acc]), acc_phase ^ 1u, abort_flag, ctr, ERR_WAIT_MMA, wait_ns)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                for (int kk = 0; kk < kblocks; ++kk) {
                    if (!mbar_wait(su32(&bars->full[stage]), phase, abort_flag, ctr, ERR_WAIT_MMA, wait_ns)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint32_t sa = su32(smem + stage * STAGE_BYTES);
                    const uint64_t dah = desc_sw64(sa), dal = desc_sw64(sa + A_BYTES);
                    const uint64_t dbh = desc_sw64(sa + 2 * A_BYTES), dbl = desc_sw64(sa + 2 * A_BYTES + B_BYTES);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        mma_f16(d_tmem, dah + 2 * k, dbh + 2 * k, idesc, (kk == 0 && k == 0) ? 0u : 1u);
                        mma_f16(d_tmem, dah + 2 * k, dbl + 2 * k, idesc, 1u);
                        mma_f16(d_tmem, dal + 2 * k, dbh + 2 * k, idesc, 1u);
                    }
                    mma_commit(su32(&bars->empty[stage]));
                    if (++stage == STAGES) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                mma_commit(su32(&bars->acc_full[acc]));
                if (++acc == 2) {
                    acc = 0;
                    acc_phase ^= 1u;
                }
            }
            mma_commit(su32(&bars->drain));
            const unsigned long long t0 = gtimer();
            while (!mbar_try(su32(&bars->drain), 0)) {
                if (gtimer() - t0 > wait_ns) {
                    atomicCAS(&ctr->err_code, 0ull, ERR_DRAIN);
                    break;
                }
            }
        }
    } else {
        // ---------------- epilogue: one tile row per thread ----------------
        // Each warp stages the tile's column norms and inverse scales in its own
        // shared-memory slice (read back as broadcasts), computes each group of 32
        // entries without branches, patches padding and the diagonal with selects, writes the
        // group to its output buffer, recomputes the rare cancellation-prone entries there and
        // has one TMA store take the buffer.
        // two warps per TMEM lane quarter: each takes one half (128 columns) of the tile
        const int quarter = warp & 3;
        const int half = (warp - 2) >> 2;
        const int rt = quarter * 32 + lane;   // row within the 128-row tile
        // pairs of columns: norms in x, y, inverse scales in z, w
        float *colv = reinterpret_cast<float *>(smem + COL_OFF) + (warp - 2) * PANEL;
        uint8_t *outb = smem + OUT_OFF + (warp - 2) * 2 * OUT_BYTES;
        int ob = 0;   // output buffer of the next group
        float2 *colsum = reinterpret_cast<float2 *>(smem + SUM_OFF);   // [warp][column of the half]
        int acc = 0;
        uint32_t acc_phase = 0;
        // A warp that gives up (ok false) does no more work but stays for the barriers of the items left:
        // the other three may still get an accumulator or two and wait for it there.
        bool ok = true;
        // failure-path test hook: one warp waits (bounded) on a flag that nothing sets, the others go on
        if (bt.inject_stall == STALL_BUILD && warp == 2)
            ok = __all_sync(0xFFFFFFFFu, flag_wait(&ctr->never_set, abort_flag, ctr, ERR_INJECTED, wait_ns));
        for (int t = blockIdx.x; t < nitems; t += gridDim.x) {
            const Tile tile = bt.tiles[t >> split];
            // The item's groups of 32 columns start at gi of the tile's; the warp takes `ng` from gi + gw:
            // half of the item's, or (a part is one K-block) all of them for one of the halves.
            const int part = t & ((1 << split) - 1), gi = part * (BN / 32 >> split);
            const int gw = split < 2 ? half * (BN / 64 >> split) : 0;
            const int ng = split < 2 ? BN / 64 >> split : (part & 1) == half ? 2 : 0;
            const TestDesc &d = bt.desc[tile.t];
            const int64_t n = d.n, NKB = d.NKB;
            const int kern = d.kern;
            const float neg_inv_2s2 = d.neg_inv_2s2, inv_sigma = d.inv_sigma, tau = d.tau;
            const float diag_val = (kern == 0) ? 0.f : 1.f;
            const float *norms = bt.norms + d.row0, *inv_scale = bt.iscale + d.row0;
            // first row of the warp's 32 in the block array (rows of 64 entries)
            const int64_t drow = (d.blk0 + blk_index(tile.I, (int64_t)tile.J * KB_PER_PANEL, NKB)) * PANEL +
                                 tile.h * BM + quarter * 32;
            // the blocks' row and column sums and largest entry (a median test's come from its
            // kernel values, in k_blocksums)
            const bool sums = bt.build_sums && !d.median;
            float rowh = 0.f, rowl = 0.f;   // the row's sum over a K-block's first group
            float mx = 0.f;
            if (sums) half_sync(half, 0);
            unsigned fixups = 0;
            const int rp = tile.h * BM + rt;                 // row within panel I
            const int64_t i = (int64_t)tile.I * PANEL + rp;  // pooled row of the test
            const float ni = (i < n) ? norms[i] : 0.f;
            const float si = (i < n) ? inv_scale[i] : 0.f;
            __syncwarp();
#pragma unroll
            for (int k = 0; k < BN / 64; ++k) {
                const int c = 32 * k + lane;
                if (k >= ng) break;
                const int64_t j = (int64_t)tile.J * PANEL + (gi + gw) * 32 + c;
                float *cp = colv + (c >> 1) * 4 + (c & 1);
                cp[0] = (j < n) ? norms[j] : 0.f;
                cp[2] = (j < n) ? inv_scale[j] : 0.f;
            }
            __syncwarp();
            // the warp's lanes give up together (the group loop below synchronises them)
            ok = ok && __all_sync(0xFFFFFFFFu, mbar_wait(su32(&bars->acc_full[acc]), acc_phase, abort_flag, ctr,
                                                         ERR_WAIT_EPI, wait_ns));
            if (!ok) {
                if (sums) half_sync(half, 1);
                continue;
            }
            fence_after();
            const uint32_t tbase = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
            for (int gl = 0; gl < ng; ++gl) {
                const int g = gi + gw + gl;   // column group of the tile
                uint32_t v[32];
                tmem_ld32(tbase + (uint32_t)((gw + gl) * 32), v);
                const int64_t j0 = (int64_t)tile.J * PANEL + g * 32;
                float out[32];
                const float4 *cg = reinterpret_cast<const float4 *>(colv) + gl * 16;
                const bool patch = (kern == 0)   ? group_entries<0>(v, cg, ni, si, tau, neg_inv_2s2, inv_sigma, out)
                                   : (kern == 1) ? group_entries<1>(v, cg, ni, si, tau, neg_inv_2s2, inv_sigma, out)
                                                 : group_entries<2>(v, cg, ni, si, tau, neg_inv_2s2, inv_sigma, out);
                uint32_t fix = 0;
                if (__any_sync(0xFFFFFFFFu, patch)) {
                    tmem_ld32(tbase + (uint32_t)((gw + gl) * 32), v);   // read again: no registers held for this case
                    fix = group_patch(v, cg, ni, si, tau, kern, neg_inv_2s2, inv_sigma, out);
                }
                // padding rows / columns hold 0; the diagonal is exactly 0 (ED) / 1 (MMD)
                const uint32_t jvalid =
                    (j0 >= n) ? 0u : ((j0 + 32 <= n) ? 0xFFFFFFFFu : ((1u << (uint32_t)(n - j0)) - 1u));
                const uint32_t valid = (i < n) ? jvalid : 0u;
                const int64_t dj = i - j0;
                const uint32_t diag = (dj >= 0 && dj < 32 && i < n) ? (1u << (uint32_t)dj) : 0u;
                if (valid != 0xFFFFFFFFu || diag) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        if (!((valid >> e) & 1u)) out[e] = 0.f;
                        if ((diag >> e) & 1u) out[e] = diag_val;
                    }
                }
                fix &= valid & ~diag;
                // the buffer's last store (two groups ago) has read it
                uint8_t *buf = outb + ob * OUT_BYTES;
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                __syncwarp();
#pragma unroll
                for (int c = 0; c < 8; ++c)   // row `lane`, 16-byte chunk c at c ^ (row mod 8)
                    *reinterpret_cast<float4 *>(buf + lane * 128 + ((c ^ (lane & 7)) << 4)) =
                        make_float4(out[4 * c], out[4 * c + 1], out[4 * c + 2], out[4 * c + 3]);
                // cancellation-prone pairs: d^2 by direct differences
                if (__any_sync(0xFFFFFFFFu, fix != 0u)) {
                    fixups += __popc(fix);
                    fix_entries(fix, buf, d, i, j0);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {   // every lane's, so that no entry is held in registers meanwhile
                        const float4 x = *reinterpret_cast<const float4 *>(buf + lane * 128 + ((c ^ (lane & 7)) << 4));
                        out[4 * c] = x.x;
                        out[4 * c + 1] = x.y;
                        out[4 * c + 2] = x.z;
                        out[4 * c + 3] = x.w;
                    }
                }
                if (sums) {
                    f32x2 rh = 0, rl = 0;   // even and odd columns, sixteen each, as k_blocksums' chains
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        pair_add2(rh, rl, pack2(out[e], out[e + 1]));
                        mx = fmaxf(mx, fmaxf(out[e], out[e + 1]));
                    }
                    float h, l;
                    pair_join(rh, rl, h, l);
                    if (gl & 1) {   // a K-block is complete
                        float s, e;
                        two_sum(rowh, h, s, e);
                        bt.rowpart[drow + lane + (int64_t)(g >> 1) * PANEL] = (double)s + (double)((rowl + l) + e);
                    } else {
                        rowh = h;
                        rowl = l;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                                     &tm_d),
                                 "r"((g & 1) * 32), "r"((int)(drow + (int64_t)(g >> 1) * PANEL)), "r"(su32(buf))
                                 : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                if (sums && tile.I != tile.J) {   // (the diagonal square's row sums have both triangles)
                    // column `lane` of the group over the warp's rows, even and odd rows at once
                    f32x2 ch = 0, cl = 0;
#pragma unroll 8
                    for (int r = 0; r < 32; r += 2) {
                        const float x0 = *reinterpret_cast<const float *>(buf + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) +
                                                                          (lane & 3) * 4);
                        const float x1 = *reinterpret_cast<const float *>(
                            buf + (r + 1) * 128 + (((lane >> 2) ^ ((r + 1) & 7)) << 4) + (lane & 3) * 4);
                        pair_add2(ch, cl, pack2(x0, x1));
                    }
                    float h, l;
                    pair_join(ch, cl, h, l);
                    colsum[(warp - 2) * (PANEL / 2) + gl * 32 + lane] = make_float2(h, l);
                }
                ob ^= 1;
            }
            fence_before();
            mbar_arrive(su32(&bars->acc_empty[acc]));
            if (sums) {
                for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
                if (lane == 0) atomicMax(&bt.ctr[tile.t].max_d_bits, __float_as_uint(mx));
                half_sync(half, 1);
                if (tile.I != tile.J && quarter < ng) {
                    // column c of the warps' (in their group `quarter`): the four quarters in order; the panel's
                    // two row halves (two tiles) meet in the zeroed sum, whose two terms commute
                    const int c = quarter * 32 + lane;
                    float h = 0.f, l = 0.f;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        // quarter q of this half: warps 2..9, quarter = warp mod 4, half = (warp - 2) / 4
                        const int w = 4 * half + ((q + 2) & 3);
                        const float2 x = colsum[w * (PANEL / 2) + c];
                        float sum, e;
                        two_sum(h, x.x, sum, e);
                        h = sum;
                        l += x.y + e;
                    }
                    const int64_t blk = drow / PANEL + ((gi + gw) >> 1) + (c >> 6);
                    atomicAdd(&bt.colpart[blk * KB + (c & 63)], (double)h + (double)l);
                }
            }
            if (fixups) atomicAdd(&bt.ctr[tile.t].n_fixup, (unsigned long long)fixups);
            if (++acc == 2) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // its stores are done
    }

    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

}  // namespace

// Eight lanes a row once the rows fill the chip that way; with fewer rows, or long ones, a row's own steps
// are what is waited for and the whole warp takes them.  Measured, 8 lanes against 32 (us): 4,000 rows of
// 64 features 3.9 / 4.3, 16,000 of 64 5.8 / 11.1, 400 of 500 7.8 / 3.8, 16,000 of 300 13.4 / 14.2, 32,000 of
// 300 22 / 25, 32,000 of 1,000 81 / 62.
constexpr int64_t SPLIT_NARROW_ROWS = 4096, SPLIT_WIDE_ROWS = 32768;

void launch_split_rows(const Batch &b, cudaStream_t s) {
    if (b.nrows_total <= 0) return;
    const unsigned warps = 256 / 32;
    if (b.p_stride <= 128 ? b.nrows_total >= SPLIT_NARROW_ROWS : b.p_stride <= 512 && b.nrows_total >= SPLIT_WIDE_ROWS)
        k_split_rows<8><<<(unsigned)((b.nrows_total + 4 * warps - 1) / (4 * warps)), 256, 0, s>>>(b);
    else
        k_split_rows<32><<<(unsigned)((b.nrows_total + warps - 1) / warps), 256, 0, s>>>(b);
}

cudaError_t launch_build_tc(const Batch &b, const void *tmaps, int split, int num_sms, cudaStream_t s) {
    static unsigned long long smem_set[2] = {0, 0};   // one bit per device
    const auto kernel = split ? k_build_tc<true> : k_build_tc<false>;
    cudaError_t e = smem_limit_once((const void *)kernel, SMEM_BYTES, &smem_set[split ? 1 : 0]);
    if (e != cudaSuccess) return e;
    if (b.ntiles < 1) return cudaSuccess;
    const CUtensorMap *tm = (const CUtensorMap *)tmaps;
    const int64_t items = b.ntiles << split;
    const int grid = items < num_sms ? (int)items : num_sms;
    kernel<<<grid, NUM_THREADS, SMEM_BYTES, s>>>(tm[0], tm[1], tm[2], tm[3], tm[4], b, split);
    return cudaGetLastError();
}

}  // namespace ept

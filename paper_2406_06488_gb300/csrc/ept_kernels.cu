// ept_kernels.cu -- SIMT kernels of libept: relabeling draws, the plain FP32 block
// build, centring and packing, the plain FP32 contraction and the final
// combination.  Every kernel processes a batch of tests (ept_internal.cuh).
#include "ept_internal.cuh"

#include <cuda_fp16.h>
#include <cstdint>
#include <cstdlib>

namespace ept {

// ---------------------------------------------------------------------------
// Permutation stream: Philox4x32-10 (Salmon et al., SC'11) drives Knuth's selection
// sampling; see draw_column.

// floor(u * m / 2^64) for a 64-bit u and a 32-bit m, from two 32x32->64 products:
// with u = uh 2^32 + ul, the value is floor((uh m + floor(ul m / 2^32)) / 2^32)
// (the dropped low word of ul m cannot carry across a multiple of 2^32), and
// uh m + floor(ul m / 2^32) < 2^64.  Equal to the high word of the 128-bit product.
__device__ __forceinline__ uint64_t mulhi_64x32(uint64_t u, uint32_t m) {
    const uint64_t a = (uint64_t)(uint32_t)(u >> 32) * m;
    const uint64_t b = (uint64_t)(uint32_t)u * m;
    return (a + (b >> 32)) >> 32;
}

// bits of word w that belong to real pooled rows t < n
__device__ __forceinline__ uint32_t valid_bits(int w, int n) {
    const int lo = w * 32;
    if (lo + 32 <= n) return 0xFFFFFFFFu;
    if (lo >= n) return 0u;
    return (1u << (n - lo)) - 1u;
}

// The column's part of Philox4x32-10: the round keys of the test's seed and the
// products of the first two rounds that depend on the draw alone (counter (c0, 0, blo,
// bhi): round 1 multiplies blo and c0, round 2 the two results, and the one that comes
// from blo does not change from slot to slot).
struct DrawKey {
    uint32_t kx[10], ky[10];
    uint32_t bhi, a1, qhi, qlo;
    __device__ __forceinline__ DrawKey(uint64_t seed, uint64_t b) {
        kx[0] = (uint32_t)seed;
        ky[0] = (uint32_t)(seed >> 32);
#pragma unroll
        for (int r = 1; r < 10; ++r) {
            kx[r] = kx[r - 1] + 0x9E3779B9u;
            ky[r] = ky[r - 1] + 0xBB67AE85u;
        }
        bhi = (uint32_t)(b >> 32);
        const uint64_t a = (uint64_t)0xCD9E8D57u * (uint32_t)b;
        a1 = (uint32_t)a;
        const uint64_t q = (uint64_t)0xD2511F53u * ((uint32_t)(a >> 32) ^ kx[0]);
        qhi = (uint32_t)(q >> 32);
        qlo = (uint32_t)q;
    }
    // What rounds 1 and 2 of counter c0 give whatever the draw's low word: round 1's
    // product of c0 and round 2's of its high half (columns of one high word share it).
    struct Slot { uint32_t p, sh, sl; };
    __device__ __forceinline__ Slot slot(uint32_t c0) const {
        const uint64_t p = (uint64_t)0xD2511F53u * c0;
        const uint64_t s = (uint64_t)0xCD9E8D57u * ((uint32_t)(p >> 32) ^ bhi ^ ky[0]);
        return Slot{(uint32_t)p ^ ky[1], (uint32_t)(s >> 32) ^ kx[1], (uint32_t)s};
    }
    // rounds 3..9; the last round needs x0 and x2 (and the low halves of its products, no key)
    __device__ __forceinline__ void nine(const Slot &s, uint32_t &x0, uint32_t &x1, uint32_t &x2, uint32_t &x3) const {
        x0 = s.sh ^ a1;
        x1 = s.sl;
        x2 = s.p ^ qhi;
        x3 = qlo;
#pragma unroll
        for (int r = 2; r < 9; ++r) {
            const uint64_t p0 = (uint64_t)0xD2511F53u * x0;
            const uint64_t p1 = (uint64_t)0xCD9E8D57u * x2;
            x0 = (uint32_t)(p1 >> 32) ^ x1 ^ kx[r];
            x2 = (uint32_t)(p0 >> 32) ^ x3 ^ ky[r];
            x1 = (uint32_t)p1;
            x3 = (uint32_t)p0;
        }
    }
    // high halves of the two 64-bit words of counter c0 (the low halves of the last
    // round's products: no wide multiplication, no key)
    __device__ __forceinline__ void high(const Slot &s, uint32_t &h0, uint32_t &h1) const {
        uint32_t x0, x1, x2, x3;
        nine(s, x0, x1, x2, x3);
        h0 = 0xCD9E8D57u * x2;
        h1 = 0xD2511F53u * x0;
    }
    // the two whole words of counter c0
    __device__ __forceinline__ void words(uint32_t c0, uint64_t &w0, uint64_t &w1) const {
        uint32_t x0, x1, x2, x3;
        nine(slot(c0), x0, x1, x2, x3);
        const uint64_t p0 = (uint64_t)0xD2511F53u * x0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * x2;
        w0 = (p1 << 32) | ((uint32_t)(p1 >> 32) ^ x1 ^ kx[9]);
        w1 = (p0 << 32) | ((uint32_t)(p0 >> 32) ^ x3 ^ ky[9]);
    }
};

// Rank of a slot, floor(u m / 2^64) with m = n - t slots left, from the high half uh of
// u alone: v = uh m; u m = v 2^32 + ul m, so the rank is v >> 32, plus one when the low
// half's ul m / 2^32 < m carries out of v's low word.  That takes a low word above
// 2^32 - m, which one slot in 2^32 / m has: `frac` collects the largest low word, and a
// group of slots that reaches 2^32 - n is decided again from whole words
// (DRAW_SLOW_FRAC).  Past the end (m <= 0) the rank is larger than any count.
constexpr uint32_t NO_RANK = 0x7FFFFFFFu;
__device__ __forceinline__ uint32_t rank_high(uint32_t uh, uint32_t m, uint32_t &frac) {
    const uint64_t v = (uint64_t)uh * m;
    frac = max(frac, (uint32_t)v);
    return (uint32_t)(v >> 32);
}
__device__ __forceinline__ bool draw_slow(uint32_t frac, int n) { return frac >= 0u - (uint32_t)n; }

// rank of slot t from whole words
__device__ __forceinline__ uint32_t rank_exact(uint64_t u, int t, int n) {
    return t < n ? (uint32_t)mulhi_64x32(u, (uint32_t)(n - t)) : NO_RANK;
}

// Word w of a column decided slot by slot from whole words (the rare case above).
__device__ __forceinline__ uint32_t draw_word_exact(const DrawKey &key, int n, int w, int need) {
    uint32_t bits = 0;
#pragma unroll 1
    for (int j = 0; j < 16; ++j) {
        const int t = 32 * w + 2 * j;
        uint64_t u0, u1;
        key.words((uint32_t)(t >> 1), u0, u1);
        if ((int)rank_exact(u0, t, n) < need) { bits |= 1u << (2 * j); --need; }
        if ((int)rank_exact(u1, t + 1, n) < need) { bits |= 2u << (2 * j); --need; }
    }
    return bits;
}

// Decisions of one 64-slot window: lane l holds the ranks e and o of its slots 2 l and
// 2 l + 1; returns the ballots of the kept even and odd slots and lowers `need`.  A slot is kept
// iff its rank is below need less the slots kept before it in the window; those are at
// most all `cnt` ranks below need, so when the ballots against need - cnt are the same
// they are the decisions (about six windows in seven at n = 5000).  Otherwise the
// sequential dependence is resolved by a fixed-point iteration over ballots: with
// every earlier decision known a slot's decision is determined, so iterating "decide
// from the previous guesses" reaches the unique sequential solution in at most 65
// rounds (almost always 2).
__device__ __forceinline__ void decide_window(uint32_t e, uint32_t o, unsigned lt, int &need, unsigned &me,
                                              unsigned &mo) {
    me = __ballot_sync(0xFFFFFFFFu, (int)e < need);
    mo = __ballot_sync(0xFFFFFFFFu, (int)o < need);
    const int low = need - (__popc(me) + __popc(mo));
    if (__ballot_sync(0xFFFFFFFFu, (int)e < low) == me && __ballot_sync(0xFFFFFFFFu, (int)o < low) == mo) {
        need = low;
        return;
    }
    for (int it = 0; it < 70; ++it) {
        const int be = __popc(me & lt) + __popc(mo & lt);             // kept before slot 2 l
        const int bo = be + (int)((me >> (threadIdx.x & 31)) & 1u);   // and before slot 2 l + 1
        const unsigned ne = __ballot_sync(0xFFFFFFFFu, (int)e < need - be);
        const unsigned no = __ballot_sync(0xFFFFFFFFu, (int)o < need - bo);
        const bool same = (ne == me) && (no == mo);
        me = ne;
        mo = no;
        if (same) break;
    }
    need -= __popc(me) + __popc(mo);
}

// the 16 low bits of v at the even positions
__device__ __forceinline__ uint32_t spread16(uint32_t v) {
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    return (v | (v << 1)) & 0x55555555u;
}

// One warp writes one relabeling column (words w = 0..nw-1 at col[w * stride]; nw is
// a multiple of 8).  Draw b of the stream: b = 0 is the identity; b >= 1 is Knuth's
// selection sampling (Algorithm S) over the n pooled slots, slot t kept iff
// floor(u_t (n - t) / 2^64) < need, with u_t the 64-bit word (t mod 2) of
// Philox4x32-10(counter = (t/2, 0, b lo, b hi), key = (seed lo, seed hi)).  The warp
// takes 256 consecutive slots per step, in four windows of 64: lane l runs the Philox
// call of slots 2 l and 2 l + 1 of each window (four independent chains), ballots
// decide the even and the odd slots, and the first eight lanes interleave them into
// the step's eight output words.  comp: store the complement (the y* members).
// Bound by the multiplier (a wide multiplication holds its pipe for four cycles, busy 62 %)
// and the logic pipe (53 %): per two slots 16 wide multiplications and 17 three-input
// XORs, with ranks and decisions on top.  n = 5000, 10^4 columns: 119 us (137 us with
// the last round's wide products, ranks from whole words and shuffled slots);
// 5000 columns 69 us (79).
__device__ void draw_column(uint64_t seed, int nx, int n, int64_t b, int nw, bool comp, uint32_t *col,
                            int64_t stride) {
    const int lane = threadIdx.x & 31;
    if (b == 0) {
        for (int w = lane; w < nw; w += 32) {
            const uint32_t v = valid_bits(w, nx);
            col[(int64_t)w * stride] = comp ? (~v & valid_bits(w, n)) : v;
        }
        return;
    }
    const DrawKey key(seed, (uint64_t)b);
    const unsigned lt = (1u << lane) - 1u;
    int need = nx;
    for (int base = 0; base < nw * 32; base += 256) {
        unsigned me[4] = {0u, 0u, 0u, 0u}, mo[4] = {0u, 0u, 0u, 0u};
        if (need > 0 && base < n) {
            uint32_t e[4], o[4], frac = 0;
            const int left = n - base - 2 * lane;   // slots left at this lane's first slot
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t h0, h1;
                key.high(key.slot((uint32_t)((base >> 1) + 32 * q + lane)), h0, h1);
                const int m = left - 64 * q;
                e[q] = rank_high(h0, (uint32_t)m, frac);
                o[q] = rank_high(h1, (uint32_t)(m - 1), frac);
            }
            if (base + 256 > n) {   // the last step: slots past the end are never kept
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (left - 64 * q <= 0) e[q] = NO_RANK;
                    if (left - 64 * q <= 1) o[q] = NO_RANK;
                }
            }
            if (__any_sync(0xFFFFFFFFu, draw_slow(frac, n))) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int t = base + 64 * q + 2 * lane;
                    uint64_t u0, u1;
                    key.words((uint32_t)(t >> 1), u0, u1);
                    e[q] = rank_exact(u0, t, n);
                    o[q] = rank_exact(u1, t + 1, n);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) decide_window(e[q], o[q], lt, need, me[q], mo[q]);
        }
        // word 2 q + h of the step: lanes 16 h .. 16 h + 15 of window q
        const int q = (lane >> 1) & 3, sh = (lane & 1) * 16;
        const uint32_t ve = q == 0 ? me[0] : q == 1 ? me[1] : q == 2 ? me[2] : me[3];
        const uint32_t vo = q == 0 ? mo[0] : q == 1 ? mo[1] : q == 2 ? mo[2] : mo[3];
        uint32_t v = spread16((ve >> sh) & 0xFFFFu) | (spread16((vo >> sh) & 0xFFFFu) << 1);
        if (lane < 8) {
            const int w = (base >> 5) + lane;
            if (comp) v = ~v & valid_bits(w, n);
            col[(int64_t)w * stride] = v;
        }
    }
}

// Relabeling columns of the batch, one warp per column: column 0 of a test is the
// identity, columns 1..B its draws 1..B (or the caller's relabelings, validated:
// exactly nx members among the n rows), padding columns are zero.  Warps stride over
// the columns, so the grid may be capped (MASK_CTAS_PER_SM).
__global__ void __launch_bounds__(128) k_masks(const Batch bt) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t gc = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); gc < bt.ncols_total;
         gc += nwarps) {
        const int t = find_test(bt.pre.cols, bt.n_tests, gc);
        const TestDesc &d = bt.desc[t];
        const int64_t c = gc - bt.pre.cols[t];
        const int n = (int)d.n, nw = (int)d.nw;
        const int64_t Bp = d.Bp;
        uint32_t *col = bt.maskT + d.mask0 + c;
        if (c >= d.ncols) {
            for (int w = lane; w < nw; w += 32) col[(int64_t)w * Bp] = 0u;
            continue;
        }
        if (c >= 1 && d.user_masks) {
            const int nwu = d.nwu, nx = (int)d.nx;
            const bool comp = d.comp != 0;
            const uint32_t *row = d.user_masks + (c - 1) * nwu;
            int cnt = 0;
            bool bad = false;
            for (int w = lane; w < nw; w += 32) {
                uint32_t v = (w < nwu) ? row[w] : 0u;
                const uint32_t valid = valid_bits(w, n);
                if (v & ~valid) bad = true;
                v &= valid;
                cnt += __popc(v);
                col[(int64_t)w * Bp] = comp ? (~v & valid) : v;
            }
            for (int off = 16; off; off >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, off);
            bad = __any_sync(0xFFFFFFFFu, bad);
            if (lane == 0 && (bad || cnt != nx)) atomicAdd(&bt.ctr[t].bad_mask, 1ull);
            continue;
        }
        // column 0: the identity (draw 0); column c >= 1: draw b0 + c - 1
        draw_column(d.seed, (int)d.nx, n, c == 0 ? 0 : d.b0 + c - 1, nw, d.comp != 0, col, Bp);
    }
}

// The float rank of a slot: X m with X = floor(uh / 2^9) / 2^23 (a funnel shift puts the
// 23 bits behind the exponent of 1.0), rounded once.  The slot's u m / 2^64 lies within
// m 2^-23 above X m, and the rounding moves it by at most m 2^-24, so it is below the
// integer `need` exactly when the float is, unless the two are closer than n 2^-22: one
// slot in 2^21, whose word is decided again from whole words.  Costs a shift and an FMA
// where the integer rank takes another wide multiplication.
__device__ __forceinline__ float rank_float(uint32_t uh, float m) {
    return fmaf(__uint_as_float(__funnelshift_r(uh, 0x7Fu, 9)), m, -m);
}

// The sequential decisions of one word: slot e kept iff r[e] < need.  The sign of
// r - need is shifted into the word and taken off need (-2^40 (r - need) saturated to
// [0, 1] is 1 when it is negative: a non-zero difference is at least 2^-24, and r = need
// = 0 gives 0).  near: the smallest |r - need|.  (Deciding against need - r less the
// count so far, an eight-cycle chain instead of twelve, measured 5 % faster with few
// columns and 4 % slower with many.)
__device__ __forceinline__ uint32_t word_decide(const float (&r)[32], float &need, float &near) {
    uint32_t bits = 0;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        const float d = r[e] - need;
        bits = __funnelshift_l(__float_as_uint(d), bits, 1);
        near = fminf(near, fabsf(d));
        need -= __saturatef(d * -1099511627776.f);
    }
    return __brev(bits);
}

// Relabeling columns, a lane per column, words taken in turn by a ring of warps.  A slot's
// rank depends only on the stream (the same Philox words as draw_column), and only
// the decisions "keep slot t iff its rank is below need" depend on each other: a
// warp computes the ranks of its words into registers while the other warps of its
// group do theirs, then waits for its turn at `need` (one named barrier between
// neighbours of the ring), decides its slots, passes `need` on and stores the words.
// HALVES = 2: a group is 16 columns and a turn two words, the first on lanes 0..15 and
// the second on lanes 16..31 (decided after the first; the ranks of both are computed
// at once): twice as many groups, whose number per SM then rounds up to less.
// WARPS = 1, HALVES = 1: 32 columns to a warp and no turns to wait for.  Both write the
// bits of draw_column; caller relabelings take the warp kernel.  A CTA's columns never
// straddle two tests (every test's column count is a multiple of 256).
// Bound by the multiplier's pipe: 14 wide multiplications per two slots are left (what
// rounds 1 and 2 owe to the slot alone is computed once per warp and read from shared
// memory, the last round needs low halves only), 42 cycles per slot and warp, that
// pipe busy 78 %.  n = 1000, 1.24e6 columns (WARPS = 1): 1.33 ms, 2.1 ms before with whole
// words; n = 5000, 10^4 columns (WARPS = 4): 92 us, against 119 us for the warp kernel and 182 us with one
// warp per group.
// Turns of a ring of four warps: warp k waits at named barrier 1 + k for the warp before it
// (immediate numbers, so that the CTA reserves five barriers and not all sixteen).
__device__ __forceinline__ void ring_wait(int k) {
    if (k == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
    else if (k == 1) asm volatile("bar.sync 2, 64;" ::: "memory");
    else if (k == 2) asm volatile("bar.sync 3, 64;" ::: "memory");
    else asm volatile("bar.sync 4, 64;" ::: "memory");
}
__device__ __forceinline__ void ring_pass(int k) {
    if (k == 0) asm volatile("bar.arrive 1, 64;" ::: "memory");
    else if (k == 1) asm volatile("bar.arrive 2, 64;" ::: "memory");
    else if (k == 2) asm volatile("bar.arrive 3, 64;" ::: "memory");
    else asm volatile("bar.arrive 4, 64;" ::: "memory");
}

template <int WARPS, int HALVES>
__global__ void __launch_bounds__(128, 5) k_masks_group(const Batch bt) {
    static_assert((WARPS == 1 && HALVES == 1) || (WARPS == 4 && HALVES == 2), "a ring passes one turn per step");
    constexpr int COLS = 32 / HALVES, GROUPS = 4 / WARPS;   // columns of a group, groups of a CTA
    __shared__ float need_s[COLS];                          // WARPS > 1: the group's counts, handed from warp to warp
    __shared__ uint4 slot_s[4][34];                         // per warp: the step's 32 slot pairs (halves 17 apart)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ring = warp % WARPS, half = HALVES == 2 ? lane >> 4 : 0;
    const int64_t gc0 = (int64_t)blockIdx.x * (GROUPS * COLS);   // the CTA's first batch column
    if (gc0 >= bt.ncols_total) return;                           // uniform over the CTA, before any barrier
    const int t = find_test(bt.pre.cols, bt.n_tests, gc0);
    const TestDesc &d = bt.desc[t];
    const int64_t c0 = gc0 - bt.pre.cols[t] + (warp / WARPS) * COLS;   // the group's first column
    const int64_t c = c0 + (lane & (COLS - 1));                        // this lane's column
    const int n = (int)d.n, nw = (int)d.nw;
    const int64_t Bp = d.Bp;
    const bool comp = d.comp != 0;
    const uint64_t draw = (uint64_t)(d.b0 + c - 1);   // column c >= 1 holds draw b0 + c - 1
    const bool any = c0 < d.ncols;                    // a group past the test's columns has nothing to draw
    // columns of one high word share the slot table; a group that straddles two is decided from whole words
    const bool split = (uint32_t)((uint64_t)(d.b0 + c0 - 1) >> 32) != (uint32_t)((uint64_t)(d.b0 + c0 + COLS - 2) >> 32);
    uint32_t *col = bt.maskT + d.mask0 + c;
    const DrawKey key(d.seed, draw);
    const float limit = split ? 3.0e38f : (float)n * 2.384185791015625e-7f;   // n 2^-22
    uint4 *slots = slot_s[warp];
    float need = (float)d.nx;
    for (int w0 = 2 * ring; w0 < nw; w0 += 2 * WARPS) {   // nw is a multiple of 8
        const bool some = any && 32 * w0 < n;             // uniform over the group
        if (some) {
            __syncwarp();
            const DrawKey::Slot s = key.slot((uint32_t)(16 * w0 + lane));
            slots[lane + (lane >> 4)] = make_uint4(s.p, s.sh, s.sl, 0u);
            __syncwarp();
        }
#pragma unroll 1
        for (int k = 0; k < 2; k += HALVES) {
            const int w = w0 + k + half;
            const int left = n - 32 * w;
            float r[32], near = 3.0e38f;
            if (some) {
                const float m = (float)left;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const uint4 sv = slots[17 * (k + half) + j];
                    uint32_t h0, h1;
                    key.high(DrawKey::Slot{sv.x, sv.y, sv.z}, h0, h1);
                    r[2 * j] = rank_float(h0, m - (float)(2 * j));
                    r[2 * j + 1] = rank_float(h1, m - (float)(2 * j + 1));
                }
                if (left < 32) {   // slots past the end are never kept
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (e >= left) r[e] = 1.0e30f;
                }
            }
            if (WARPS > 1 && w0 > 0) {
                __syncwarp();
                ring_wait(ring);
                need = need_s[lane & (COLS - 1)];
            }
            uint32_t bits = 0;
            if (some) {
                float before = need;
                bits = word_decide(r, need, near);
                if (HALVES == 2) {
                    if (half == 0 && near <= limit) {
                        bits = draw_word_exact(key, n, w, (int)before);
                        need = before - (float)__popc(bits);
                    }
                    // the second word starts where the first ended
                    before = __shfl_sync(0xFFFFFFFFu, need, lane & 15);
                    if (half == 1) {
                        need = before;
                        near = 3.0e38f;
                        bits = word_decide(r, need, near);
                    }
                }
                if (half == HALVES - 1 && near <= limit) {
                    bits = draw_word_exact(key, n, w, (int)before);
                    need = before - (float)__popc(bits);
                }
            }
            if (WARPS > 1 && w0 + 2 < nw) {
                if (half == HALVES - 1) need_s[lane & (COLS - 1)] = need;
                __syncwarp();
                ring_pass((ring + 1) & 3);
            }
            if (c == 0) bits = valid_bits(w, (int)d.nx);   // the identity
            if (comp) bits = ~bits & valid_bits(w, n);
            col[(int64_t)w * Bp] = c < d.ncols ? bits : 0u;
        }
    }
}

// Blocks per SM of the draw kernel: MASK_CTAS_PER_SM, or the environment's
// EPT_MASK_BLOCKS_PER_SM (0: one warp per column, no cap).
static int mask_blocks_per_sm() {
    static const int v = [] {
        const char *e = getenv("EPT_MASK_BLOCKS_PER_SM");
        if (!e || !*e) return MASK_CTAS_PER_SM;
        const int k = atoi(e);
        return k < 0 ? MASK_CTAS_PER_SM : (k > 64 ? 64 : k);
    }();
    return v;
}

void launch_masks(const Batch &b, int num_sms, int mode, cudaStream_t s) {
    if (b.ncols_total <= 0) return;
    if (mode == DRAW_RING) {
        k_masks_group<4, 2><<<(unsigned)(b.ncols_total / 16), 128, 0, s>>>(b);
        return;
    }
    if (mode == DRAW_LANES) {
        k_masks_group<1, 1><<<(unsigned)(b.ncols_total / 128), 128, 0, s>>>(b);
        return;
    }
    int64_t blocks = (b.ncols_total + 3) / 4;
    const int per_sm = mask_blocks_per_sm();
    if (per_sm > 0) {
        const int64_t cap = (int64_t)(num_sms > 0 ? num_sms : 1) * per_sm;
        if (blocks > cap) blocks = cap;
    }
    k_masks<<<(unsigned)blocks, 128, 0, s>>>(b);
}

// the stream itself, for export: column c = draw b0 + c
__global__ void __launch_bounds__(256) k_perm_masks_plain(uint64_t seed, int nx, int ny, int64_t b0, int64_t count,
                                                          int nw, uint32_t *__restrict__ maskT) {
    const int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= count) return;
    draw_column(seed, nx, nx + ny, b0 + c, nw, false, maskT + c, count);
}

void launch_perm_masks_plain(uint64_t seed, int nx, int ny, int64_t b0, int64_t count, int nw, uint32_t *maskT,
                             cudaStream_t s) {
    if (count <= 0) return;
    k_perm_masks_plain<<<(unsigned)((count + 7) / 8), 256, 0, s>>>(seed, nx, ny, b0, count, nw, maskT);
}

// maskT columns 0..count-1 -> row-major [count][nwu]
__global__ void k_masks_to_rows(const uint32_t *__restrict__ maskT, int64_t ncols, int nw, int64_t count, int nwu,
                                uint32_t *__restrict__ rows) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= count * nwu) return;
    const int64_t c = idx / nwu;
    const int w = (int)(idx % nwu);
    rows[idx] = maskT[(int64_t)w * ncols + c];
}

void launch_masks_to_rows(const uint32_t *maskT, int64_t ncols, int nw, int64_t count, int nwu, uint32_t *rows,
                          cudaStream_t s) {
    const int64_t tot = count * nwu;
    if (tot <= 0) return;
    k_masks_to_rows<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(maskT, ncols, nw, count, nwu, rows);
}

// ---------------------------------------------------------------------------
__device__ __forceinline__ const float *pooled_row(const TestDesc &d, int64_t i) {
    return (i < d.nx) ? d.X + i * d.p : d.Y + (i - d.nx) * d.p;
}

// Plain path: squared row norms ||z_i||^2 of the pooled rows, exact products summed
// in FP64 and rounded once to FP32 (padded rows: 0), and the count of non-finite
// inputs.  One warp per row of the batch.
__global__ void __launch_bounds__(256) k_norms(const Batch bt) {
    const int lane = threadIdx.x & 31;
    const int64_t gr = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (gr >= bt.nrows_total) return;
    const int t = find_test(bt.pre.rows, bt.n_tests, gr);
    const TestDesc d = bt.desc[t];
    const int64_t i = gr - d.row0;
    double acc = 0.0;
    bool bad = false;
    if (i < d.n) {
        const float *z = pooled_row(d, i);
        for (int64_t k = lane; k < d.p; k += 32) {
            const float v = z[k];
            bad |= !isfinite(v);
            acc = fma((double)v, (double)v, acc);
        }
    }
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) atomicAdd(&bt.ctr[t].nonfinite, 1ull);
    if (lane == 0) bt.norms[gr] = (float)acc;
}

void launch_norms(const Batch &b, cudaStream_t s) {
    if (b.nrows_total <= 0) return;
    k_norms<<<(unsigned)((b.nrows_total + 7) / 8), 256, 0, s>>>(b);
}

// ---------------------------------------------------------------------------
// Plain block build, SIMT FP32 (Algorithm 1 block construction; Algorithm 3 entries
// through the expansion ||x||^2 + ||y||^2 - 2 x.y).  One CTA computes half of a
// stored 256x64 block (128 rows x 64 columns): 256 threads, 8x4 outputs each,
// K-loop over p in steps of 16 staged through shared memory.
// Epilogue: d2 = max(0, n_i + n_j - 2 g_ij); a pair with d2 < tau (n_i + n_j)
// (cancellation-prone near-duplicate) is recomputed directly as sum (x - y)^2 in
// FP64; then the distance, exp(-d2 / (2 sigma^2)) (Gaussian) or exp(-d / sigma)
// (Laplacian); the diagonal is exactly 0 (distances) or 1 (kernels); padded rows and
// columns are 0.
__global__ void __launch_bounds__(256) k_build_simt(const Batch bt) {
    __shared__ float As[16][128 + 4];
    __shared__ float Bs[16][64 + 4];
    const int64_t gb = blockIdx.x;
    const int h = blockIdx.y;
    const BlkInfo bi = bt.blk[gb];
    const TestDesc d = bt.desc[bi.t];
    const int64_t n = d.n, p = d.p;
    const int64_t row0 = (int64_t)bi.I * PANEL + h * 128;
    const int64_t col0 = (int64_t)bi.kb * KB;
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    float acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = 0.f;

    for (int64_t k0 = 0; k0 < p; k0 += 16) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int idx = e * 256 + t, r = idx >> 4, k = idx & 15;
            const int64_t i = row0 + r;
            float v = 0.f;
            if (i < n && k0 + k < p) v = __ldg(pooled_row(d, i) + k0 + k);
            As[k][r] = v;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int idx = e * 256 + t, cc = idx >> 4, k = idx & 15;
            const int64_t j = col0 + cc;
            float v = 0.f;
            if (j < n && k0 + k < p) v = __ldg(pooled_row(d, j) + k0 + k);
            Bs[k][cc] = v;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const float4 a0 = *reinterpret_cast<const float4 *>(&As[k][ty * 8]);
            const float4 a1 = *reinterpret_cast<const float4 *>(&As[k][ty * 8 + 4]);
            const float4 b = *reinterpret_cast<const float4 *>(&Bs[k][tx * 4]);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[a][c] = fmaf(av[a], bv[c], acc[a][c]);
        }
        __syncthreads();
    }
    const float neg = d.neg_inv_2s2, inv_sigma = d.inv_sigma, tau = d.tau;
    const int kern = d.kern;
    unsigned fixups = 0;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int64_t i = row0 + ty * 8 + a;
        float out[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int64_t j = col0 + tx * 4 + c;
            float v = 0.f;
            if (i < n && j < n) {
                if (i == j) {
                    v = (kern == 0) ? 0.f : 1.f;
                } else {
                    const float ni = __ldg(bt.norms + d.row0 + i), nj = __ldg(bt.norms + d.row0 + j);
                    const float d2 = fmaxf(0.f, ni + nj - 2.f * acc[a][c]);
                    if (d2 < tau * (ni + nj)) {
                        const float *zi = pooled_row(d, i), *zj = pooled_row(d, j);
                        double s = 0.0;
                        for (int64_t k = 0; k < p; ++k) {
                            const double df = (double)zi[k] - (double)zj[k];
                            s = fma(df, df, s);
                        }
                        ++fixups;
                        v = (float)entry_from_d2(s, kern, neg, inv_sigma);
                    } else {
                        v = (kern == 0) ? sqrtf(d2) : (kern == 1) ? exp_cw(d2 * neg) : exp_cw(-sqrtf(d2) * inv_sigma);
                    }
                }
            }
            out[c] = v;
        }
        const int64_t off = (gb * PANEL + h * 128 + ty * 8 + a) * KB + tx * 4;
        *reinterpret_cast<float4 *>(bt.D + off) = make_float4(out[0], out[1], out[2], out[3]);
    }
    if (fixups) atomicAdd(&bt.ctr[bi.t].n_fixup, (unsigned long long)fixups);
}

void launch_build_simt(const Batch &b, cudaStream_t s) {
    if (b.nblk_total <= 0) return;
    k_build_simt<<<dim3((unsigned)b.nblk_total, 2), 256, 0, s>>>(b);
}

// ---------------------------------------------------------------------------
// (The tensor-core build sums its own entries but for median-heuristic tests.)
// Row and column partial sums of each stored block, for the row sums r = W 1
// (the lower part of W is the transpose of the stored strictly-upper blocks, so
// their column sums supply it).  Sums are accumulated as unevaluated FP32 pairs
// (hi, lo) with Knuth's TwoSum, an error-free transformation (the rounding error of
// every addition is carried in lo), then widened to FP64: about twice the FP32
// precision at FP32 cost.  One CTA per stored block of the batch, taking the block
// in four quarters of 64 rows: each quarter is read once with coalesced 16-byte loads
// into shared memory (rows padded to 65 words, so that threads walking rows or
// columns hit distinct banks), then four threads per row and four per column each
// sum 16 values, and the four pairs meet in a fixed order.

// (h, l) += (h2, l2), the rounding error of the hi addition kept in l
__device__ __forceinline__ void pair_add(float &h, float &l, float h2, float l2) {
    float s2, e;
    two_sum(h, h2, s2, e);
    h = s2;
    l += l2 + e;
}

__global__ void __launch_bounds__(256) k_blocksums(const Batch bt, int median_only) {
    constexpr int QR = 64, LD = KB + 1;   // rows per quarter, padded row length
    __shared__ float tile[QR * LD];
    __shared__ float wmax[8];
    const int64_t gb = blockIdx.x;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float *base = bt.D + gb * (int64_t)(PANEL * KB);
    const BlkInfo bi = bt.blk[gb];
    const TestDesc &d = bt.desc[bi.t];
    // median-heuristic tests: the build wrote distances; now that the bandwidth is
    // known, they become kernel values in place as they are read (padding stays 0)
    if (median_only && !d.median) return;   // the tensor-core build has summed its entries
    const bool median = d.median != 0;
    float neg = 0.f, inv = 0.f;
    if (median) {
        const float sigma = __uint_as_float(bt.ctr[bi.t].sel_prefix);
        neg = -1.f / (2.f * sigma * sigma);
        inv = 1.f / sigma;
    }
    const bool gauss = d.stat == 1;
    const int64_t n = d.n;
    float mx = 0.f;
    const int rr = t >> 2, part = t & 3;   // row rr (or column rr) of the quarter, its quarter `part`
    float ch = 0.f, cl = 0.f;               // this thread's column partial over the block's quarters
    for (int qtr = 0; qtr < PANEL / QR; ++qtr) {
        float *qbase = base + (int64_t)qtr * QR * KB;
        // coalesced load: float4 k = t + 256 i covers row k / 16, columns 4 (k % 16) ..
#pragma unroll
        for (int i = 0; i < QR * KB / 4 / 256; ++i) {
            const int k = t + 256 * i, row = k >> 4, c4 = (k & 15) * 4;
            float4 v = reinterpret_cast<const float4 *>(qbase)[k];
            if (median) {
                const int64_t gi = (int64_t)bi.I * PANEL + qtr * QR + row, gj = (int64_t)bi.kb * KB + c4;
                float e4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gi < n && gj + e < n) e4[e] = gauss ? exp_cw(e4[e] * e4[e] * neg) : exp_cw(-e4[e] * inv);
                v = make_float4(e4[0], e4[1], e4[2], e4[3]);
                reinterpret_cast<float4 *>(qbase)[k] = v;
            }
            mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            float *dst = tile + row * LD + c4;
            dst[0] = v.x;
            dst[1] = v.y;
            dst[2] = v.z;
            dst[3] = v.w;
        }
        __syncthreads();
        // row rr of the quarter: columns 16 part .. 16 part + 15, then the four parts in order
        {
            float h = 0.f, l = 0.f;
            const float *src = tile + rr * LD + 16 * part;
#pragma unroll
            for (int j = 0; j < 16; ++j) pair_add(h, l, src[j], 0.f);
            float h1 = __shfl_xor_sync(0xFFFFFFFFu, h, 1), l1 = __shfl_xor_sync(0xFFFFFFFFu, l, 1);
            if (part & 1) { const float th = h, tl = l; h = h1; l = l1; h1 = th; l1 = tl; }
            pair_add(h, l, h1, l1);   // (part 0 + part 1), (part 2 + part 3)
            float h2 = __shfl_xor_sync(0xFFFFFFFFu, h, 2), l2 = __shfl_xor_sync(0xFFFFFFFFu, l, 2);
            if (part & 2) { const float th = h, tl = l; h = h2; l = l2; h2 = th; l2 = tl; }
            pair_add(h, l, h2, l2);   // (0 + 1) + (2 + 3)
            if (part == 0) bt.rowpart[gb * PANEL + qtr * QR + rr] = (double)h + (double)l;
        }
        // column rr: rows 16 part .. 16 part + 15 of the quarter, into this thread's pair
        {
            const float *src = tile + (16 * part) * LD + rr;
#pragma unroll
            for (int i = 0; i < 16; ++i) pair_add(ch, cl, src[i * LD], 0.f);
        }
        __syncthreads();
    }
    // the column's four parts in order: (0 + 1) + (2 + 3)
    {
        float h = ch, l = cl;
        float h1 = __shfl_xor_sync(0xFFFFFFFFu, h, 1), l1 = __shfl_xor_sync(0xFFFFFFFFu, l, 1);
        if (part & 1) { const float th = h, tl = l; h = h1; l = l1; h1 = th; l1 = tl; }
        pair_add(h, l, h1, l1);
        float h2 = __shfl_xor_sync(0xFFFFFFFFu, h, 2), l2 = __shfl_xor_sync(0xFFFFFFFFu, l, 2);
        if (part & 2) { const float th = h, tl = l; h = h2; l = l2; h2 = th; l2 = tl; }
        pair_add(h, l, h2, l2);
        if (part == 0) bt.colpart[gb * KB + rr] = (double)h + (double)l;
    }
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    if (lane == 0) wmax[warp] = mx;
    __syncthreads();
    if (t == 0) {
        float m = wmax[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) m = fmaxf(m, wmax[w]);
        atomicMax(&bt.ctr[bi.t].max_d_bits, __float_as_uint(m));
    }
}

void launch_blocksums(const Batch &b, bool median_only, cudaStream_t s) {
    if (b.nblk_total <= 0) return;
    k_blocksums<<<(unsigned)b.nblk_total, 256, 0, s>>>(b, median_only ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Median heuristic (bandwidth of the MMD kernels): the lower median, rank
// k = floor((N - 1) / 2) in ascending order, of the N = n (n - 1) / 2 distances
// between distinct pooled rows (the strictly upper entries of the stored blocks).
// Exact selection on the FP32 bit patterns (non-negative floats order like their
// bits).  k_median_sample takes 16,384 entries at random and brackets the median six
// standard deviations of its sample rank to either side, about 5 % of the entries.  A pass
// (k_median_pass) counts the entries below the bracket in registers and
// histograms those inside in 2048 equal bins; the last CTA of the test finds the bin
// that holds rank k, which is the next pass's bracket, until the bins are single values.  The
// first bracket is usually within 2^22 values, so two passes do it; a median outside it
// (or a test with few pairs) starts again from all values, which takes three.  Four
// passes are launched, those left return at once.
// A pass reads every stored entry once (n = 10,500: 224 MB) and adds to shared memory for one
// entry in twenty; histograms of the leading digits of every entry took 167 us a pass,
// three times, since distances share a few leading digits; now 27 us for the sample, 83 and 75 us for the
// passes that do the work and 7 us for the two that return.
constexpr int MED_SAMPLES = 16384, MED_BINS = 2048, MED_PASSES = 4;

// state of a test's selection (Counters): values [lo, lo + nbins << shift), rank k among
// the entries from `lo` on (first pass: from 0 on)
enum { MED_SAMPLED = 1, MED_INSIDE = 2, MED_DONE = 3 };

// the 32-bit finaliser of MurmurHash3 (Appleby, public domain)
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x85EBCA6Bu;
    x ^= x >> 13;
    x *= 0xC2B2AE35u;
    return x ^ (x >> 16);
}

// The bin of h[0 .. MED_BINS) that holds rank k, and the number of entries in the bins before it
// (bin -1: k is past the end); every thread of the CTA (T threads, a multiple of 32) gets both.
template <int T, typename Bin>
__device__ __forceinline__ int find_bin(const Bin *h, unsigned long long k, unsigned long long &before) {
    constexpr int PER = MED_BINS / T;
    __shared__ unsigned long long wsum[T / 32];
    __shared__ int bin_s;
    __shared__ unsigned long long before_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long mine = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) mine += h[threadIdx.x * PER + q];
    unsigned long long inc = mine;   // inclusive over the warp
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if (lane >= off) inc += o;
    }
    if (threadIdx.x == 0) bin_s = -1;
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    unsigned long long base = 0;
    for (int w = 0; w < warp; ++w) base += wsum[w];
    unsigned long long cum = base + inc - mine;   // entries before this thread's bins
    if (k >= cum && k < cum + mine) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const unsigned long long c = h[threadIdx.x * PER + q];
            if (k >= cum && k < cum + c) {
                bin_s = threadIdx.x * PER + q;
                before_s = cum;
            }
            cum += c;
        }
    }
    __syncthreads();
    before = before_s;
    const int bin = bin_s;
    __syncthreads();
    return bin;
}

__global__ void __launch_bounds__(1024) k_median_sample(const Batch bt) {
    __shared__ uint32_t h[2][MED_BINS];
    const int t = blockIdx.x;
    const TestDesc &d = bt.desc[t];
    if (!d.median) return;
    Counters *c = bt.ctr + t;
    constexpr int PER = MED_SAMPLES / 1024;
    uint32_t v[PER];
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const uint32_t s = (uint32_t)(q * 1024 + threadIdx.x);
        const int64_t gb = d.blk0 + (int64_t)(((uint64_t)mix32(s * 2u + 1u) * (uint64_t)d.nblk) >> 32);
        const int e = (int)(mix32(s * 2u + 2u) & (PANEL * KB - 1));
        const BlkInfo bi = bt.blk[gb];
        const int64_t i = (int64_t)bi.I * PANEL + (e >> 6), j = (int64_t)bi.kb * KB + (e & 63);
        const bool take = i < d.n && j < d.n && j > i;
        v[q] = take ? __float_as_uint(bt.D[gb * (int64_t)(PANEL * KB) + e]) : 0xFFFFFFFFu;
        cnt += take;
    }
    for (int k = threadIdx.x; k < MED_BINS; k += 1024) h[0][k] = 0u;
    __shared__ int cnt_s;
    if (threadIdx.x == 0) cnt_s = 0;
    __syncthreads();
    for (int off = 16; off; off >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, off);
    if ((threadIdx.x & 31) == 0) atomicAdd(&cnt_s, cnt);
    // leading 11 of 31 bits: lanes with equal digits aggregated
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const uint32_t bin = v[q] >> 20;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, bin);
        if (bin < MED_BINS && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[0][bin], (uint32_t)__popc(peers));
    }
    __syncthreads();
    const int m = cnt_s;
    const int spread = (int)(3.f * sqrtf((float)m)) + 2;   // six standard deviations of the median's sample rank
    const int r0 = m / 2 - spread, r1 = m / 2 + spread;
    const unsigned long long npairs = (unsigned long long)d.n * (unsigned long long)(d.n - 1) / 2ull;
    uint32_t lo = 0, width = 0x80000000u;
    if (r0 > 0 && r1 < m) {
        unsigned long long b0, b1;
        const int p0 = find_bin<1024>(h[0], (unsigned long long)r0, b0);
        const int p1 = find_bin<1024>(h[0], (unsigned long long)r1, b1);
        for (int k = threadIdx.x; k < MED_BINS; k += 1024) h[0][k] = h[1][k] = 0u;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PER; ++q) {   // the next 11 bits of the entries that share either digit
            const uint32_t lead = v[q] >> 20, next = (v[q] >> 9) & (MED_BINS - 1);
            if (lead == (uint32_t)p0) atomicAdd(&h[0][next], 1u);
            if (lead == (uint32_t)p1) atomicAdd(&h[1][next], 1u);
        }
        __syncthreads();
        unsigned long long x;
        const int q0 = find_bin<1024>(h[0], (unsigned long long)r0 - b0, x);
        const int q1 = find_bin<1024>(h[1], (unsigned long long)r1 - b1, x);
        lo = ((uint32_t)p0 << 20) | ((uint32_t)q0 << 9);
        width = (((uint32_t)p1 << 20) | ((uint32_t)q1 << 9)) + 512u - lo;
    }
    if (threadIdx.x == 0) {
        int shift = 0;
        while (((width - 1u) >> shift) >= (uint32_t)MED_BINS) ++shift;
        c->sel_prefix = lo;
        c->sel_shift = shift;
        c->sel_bins = ((width - 1u) >> shift) + 1u;
        c->sel_k = (npairs - 1ull) / 2ull;
        c->sel_state = MED_SAMPLED;
    }
}

// One pass over the stored entries: a CTA takes a run of consecutive blocks, and hands its
// histogram over where the test changes and at the end.
__global__ void __launch_bounds__(256) k_median_pass(const Batch bt) {
    // a CTA's counts in 32 bits (it reads fewer entries than that), a test's in 64: above n = 92,682 there are more
    // than 2^32 pairs, and equal distances share a bin (smaller tests look their bin up in 32 bits: 0.5 us a
    // pass of a few rows)
    __shared__ unsigned long long bins_s[MED_BINS];
    uint32_t *hist = reinterpret_cast<uint32_t *>(bins_s);
    __shared__ bool last_s;
    const int64_t b0 = bt.nblk_total * (int64_t)blockIdx.x / gridDim.x;
    const int64_t b1 = bt.nblk_total * (int64_t)(blockIdx.x + 1) / gridDim.x;
    int64_t gb = b0;
    while (gb < b1) {
        const int t = bt.blk[gb].t;
        const TestDesc &d = bt.desc[t];
        const int64_t end = d.blk0 + d.nblk < b1 ? d.blk0 + d.nblk : b1;   // this test's blocks of the run
        Counters *c = bt.ctr + t;
        if (!d.median || c->sel_state == MED_DONE) {
            gb = end;
            continue;
        }
        const uint32_t lo = c->sel_prefix, shift = c->sel_shift, bins = c->sel_bins;
        const int64_t n = d.n;
        for (int k = threadIdx.x; k < MED_BINS; k += 256) hist[k] = 0u;
        __syncthreads();
        uint32_t below = 0;
        const unsigned int nb = (unsigned int)(end - gb);
        for (; gb < end; ++gb) {
            const BlkInfo bi = bt.blk[gb];
            const int64_t i0 = (int64_t)bi.I * PANEL, j0 = (int64_t)bi.kb * KB;
            const bool inside = i0 + PANEL <= n && j0 + KB <= n && j0 >= i0 + PANEL;   // every entry counts
            const float4 *base = reinterpret_cast<const float4 *>(bt.D + gb * (int64_t)(PANEL * KB));
#pragma unroll 1
            for (int q0 = 0; q0 < PANEL * KB / 4 / 256; q0 += 8) {
                float4 f[8];   // the loads first: they do not move past the histogram's atomics
#pragma unroll
                for (int q = 0; q < 8; ++q) f[q] = base[(q0 + q) * 256 + threadIdx.x];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int x = (q0 + q) * 256 + threadIdx.x;
                    const uint32_t u[4] = {__float_as_uint(f[q].x), __float_as_uint(f[q].y), __float_as_uint(f[q].z),
                                           __float_as_uint(f[q].w)};
                    const int64_t i = i0 + (x >> 4), j = j0 + (x & 15) * 4;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (!inside && !(i < n && j + e < n && j + e > i)) continue;
                        const uint32_t bin = (u[e] - lo) >> shift;   // below `lo`: wraps past the bins
                        below += u[e] < lo;
                        if (u[e] >= lo && bin < bins) atomicAdd(&hist[bin], 1u);
                    }
                }
            }
        }
        __syncthreads();
        unsigned long long *gh = bt.sel_hist + (int64_t)t * MED_BINS;
        for (int k = threadIdx.x; k < MED_BINS; k += 256)
            if (hist[k]) atomicAdd(&gh[k], (unsigned long long)hist[k]);
        for (int off = 16; off; off >>= 1) below += __shfl_xor_sync(0xFFFFFFFFu, below, off);
        if ((threadIdx.x & 31) == 0 && below) atomicAdd(&c->sel_below, (unsigned long long)below);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last_s = atomicAdd(&c->sel_blocks, nb) + nb == (unsigned int)d.nblk;
        __syncthreads();
        if (!last_s) continue;
        // the test's last CTA: the bin of rank k
        __threadfence();
        const bool wide = (unsigned long long)n * (unsigned long long)(n - 1) / 2ull >> 32 != 0ull;
        for (int k = threadIdx.x; k < MED_BINS; k += 256) {
            const unsigned long long v = __ldcg(&gh[k]);
            if (wide) bins_s[k] = v;
            else hist[k] = (uint32_t)v;
            gh[k] = 0ull;   // ready for the next pass
        }
        __syncthreads();
        const bool first = c->sel_state == MED_SAMPLED;
        const unsigned long long under = first ? __ldcg(&c->sel_below) : 0ull, k = c->sel_k;
        unsigned long long before = 0;
        const int bin = k < under ? -1   // uniform
                        : wide    ? find_bin<256>(bins_s, k - under, before)
                                  : find_bin<256>(hist, k - under, before);
        __syncthreads();
        if (threadIdx.x == 0) {
            c->sel_blocks = 0u;
            if (bin < 0) {
                // outside the sampled bracket: from all values; else the counts do not add up
                // (reported as a zero bandwidth)
                c->sel_state = first ? MED_INSIDE : MED_DONE;
                c->sel_prefix = 0u;
                c->sel_shift = 20;
                c->sel_bins = MED_BINS;
            } else {
                c->sel_prefix = lo + ((uint32_t)bin << shift);
                c->sel_k = k - under - before;
                c->sel_state = shift == 0 ? MED_DONE : MED_INSIDE;
                c->sel_shift = shift > 11 ? shift - 11 : 0;
                c->sel_bins = 1u << (shift < 11 ? shift : 11);
            }
        }
        __syncthreads();
    }
}

void launch_median_select(const Batch &b, int num_sms, cudaStream_t s) {
    if (!b.sel_hist || b.nblk_total <= 0) return;
    k_median_sample<<<(unsigned)b.n_tests, 1024, 0, s>>>(b);
    // as many CTAs as are resident at once (five of 48 registers a thread): 84 + 73 us with five per SM,
    // 117 + 102 with six (a second wave), 113 + 101 with three
    const int64_t full = (int64_t)5 * num_sms, grid = b.nblk_total < full ? b.nblk_total : full;
    for (int pass = 0; pass < MED_PASSES; ++pass) k_median_pass<<<(unsigned)grid, 256, 0, s>>>(b);
}

// r_i = sum over the stored blocks of row i's panel (its own row segments) + sum
// over the earlier panels J < panel(i) of column i's segments.  Eight threads per
// row take every eighth term and combine by a fixed shuffle tree (deterministic).
// CTA = 32 rows of one test (256 threads); Spart[CTA] = sum of its rows' r_i, by one warp's tree: as one
// thread's 32 additions in a row it was most of a small test's time (n = 200: 4.5 -> 3.5 us; 500 tests of
// n = 400: 58 -> 43 us).
__global__ void __launch_bounds__(256) k_rowsum_reduce(const Batch bt) {
    __shared__ double sh[32];
    const int sub = threadIdx.x & 7, rl = threadIdx.x >> 3;
    const int64_t gr = (int64_t)blockIdx.x * 32 + rl;
    const int t = find_test(bt.pre.rows, bt.n_tests, (int64_t)blockIdx.x * 32);
    const TestDesc &d = bt.desc[t];
    const int64_t i = gr - d.row0;
    const int64_t I = i / PANEL, rr = i % PANEL, NKB = d.NKB;
    double acc = 0.0;
    if (i < d.n) {
        const int64_t nkb = contract_nkb(d) - KB_PER_PANEL * I;   // those with real columns
        const int64_t base = d.blk0 + blk_off(I, NKB);
        for (int64_t k = sub; k < nkb; k += 8) acc += bt.rowpart[(base + k) * PANEL + rr];
        const int64_t kbi = i / KB, ci = i % KB;
        for (int64_t J = sub; J < I; J += 8) acc += bt.colpart[(d.blk0 + blk_index(J, kbi, NKB)) * KB + ci];
    }
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 4);
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
    acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
    if (sub == 0) {
        bt.r[gr] = acc;
        sh[rl] = acc;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double s = sh[threadIdx.x];
        for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
        if (threadIdx.x == 0) bt.Spart[blockIdx.x] = s;
    }
}

void launch_rowsum_reduce(const Batch &b, cudaStream_t s) {
    if (b.nrows_total <= 0) return;
    k_rowsum_reduce<<<(unsigned)(b.nrows_total / 32), 256, 0, s>>>(b);
}

// Deterministic sum of a short array in fixed order (one warp: strided lane sums,
// then a fixed shuffle tree).
__device__ __forceinline__ double warp_ordered_sum(const double *a, int64_t m) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int64_t k = lane; k < m; k += 32) s += a[k];
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
    return s;
}

__device__ __forceinline__ double block_sum_256(double v, double *sh) {
    const int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int off = 128; off; off >>= 1) {
        if (t < off) sh[t] += sh[t + off];
        __syncthreads();
    }
    return sh[0];
}

// Centring.  u_i = r_i / n - S / (2 n^2) (double centring, S = 1'W1), rounded to FP32;
// the centred matrix is W~ = W - u 1' - 1 u'.  Let s mark the contracted group (size
// m, the other group has size o; see ept_internal.cuh).  Writing Eq. 1 with
// T = s'W~s, L = s'W~1 and S~ = 1'W~1 (the sums over the other group are
// S~ - 2L + T, the cross sums L - T) gives, whatever u is,
//     ED = -cT T + cL L - S~/o^2,  cT = (n/(nx ny))^2,  cL = 2n/(m o^2),
// and MMD^2 (Eq. 2) is the same expression with the opposite sign.  Because
// s_i^2 = s_i, L = s' diag(r~) s with r~ = W~ 1 = r - n u - (1'u) 1, so
//     stat = sign * (cT s'Cs + S~/o^2),  C = W~ - kappa diag(r~),  kappa = cL/cT = 2m/n,
// sign = -1 (ED) or +1 (MMD).  dcorr_i = kappa r~_i.
// Only r~ must be exact (it is, in FP64, for the FP32 u actually stored); u itself
// may be any value, so it is formed with multiplications by precomputed reciprocals.
// Step 1 (one CTA per panel of the batch): u_i, Upart[panel] = sum of the u_i.
__global__ void __launch_bounds__(256) k_center_u(const Batch bt) {
    __shared__ double sh[256];
    __shared__ double bS;
    const int64_t gp = blockIdx.x;
    const int t = find_test(bt.pre.panels, bt.n_tests, gp);
    const TestDesc d = bt.desc[t];
    if (threadIdx.x < 32) {
        const double S = warp_ordered_sum(bt.Spart + d.sp0, d.n_pad / 32);
        if (threadIdx.x == 0) bS = S;
    }
    __syncthreads();
    const int64_t i = (gp - d.pan0) * PANEL + threadIdx.x;
    float ui = 0.f;
    if (i < d.n) ui = (float)(bt.r[d.row0 + i] * d.inv_n - bS * d.inv_2n2);
    bt.u[d.row0 + i] = ui;
    float mx = fabsf(ui);
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    if ((threadIdx.x & 31) == 0) atomicMax(&bt.ctr[t].max_u_bits, __float_as_uint(mx));
    const double tot = block_sum_256((double)ui, sh);
    if (threadIdx.x == 0) bt.Upart[gp] = tot;
}

// Step 2 (one CTA per panel): r~_i, dcorr_i = kappa r~_i, Stpart[panel] = sum of r~_i.
__global__ void __launch_bounds__(256) k_center_r(const Batch bt) {
    __shared__ double sh[256];
    __shared__ double bU;
    const int64_t gp = blockIdx.x;
    const int t = find_test(bt.pre.panels, bt.n_tests, gp);
    const TestDesc d = bt.desc[t];
    if (threadIdx.x < 32) {
        const double U = warp_ordered_sum(bt.Upart + d.pan0, d.NP);
        if (threadIdx.x == 0) bU = U;
    }
    __syncthreads();
    const int64_t i = (gp - d.pan0) * PANEL + threadIdx.x;
    double rt = 0.0;
    if (i < d.n) rt = bt.r[d.row0 + i] - (double)d.n * (double)bt.u[d.row0 + i] - bU;
    bt.dcorr[d.row0 + i] = d.kappa * rt;
    float mx = (float)fabs(d.kappa * rt);
    for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    if ((threadIdx.x & 31) == 0) atomicMax(&bt.ctr[t].max_dc_bits, __float_as_uint(mx));
    const double tot = block_sum_256(rt, sh);
    if (threadIdx.x == 0) bt.Stpart[gp] = tot;
}

// The sum of a value over the CTA's CENTER_THREADS threads, in every thread: each lane of the first warp adds
// every 32nd value in a fixed tree, then a shuffle tree (an FP64 instruction of a warp takes 16 cycles of the SM:
// one warp's 20 cost less than a tree in every warp).
constexpr int CENTER_THREADS = 512;
__device__ __forceinline__ double center_sum(double v, double *sh) {
    __syncthreads();   // the last sum has been read
    sh[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double x[CENTER_THREADS / 32];
#pragma unroll
        for (int q = 0; q < CENTER_THREADS / 32; ++q) x[q] = sh[q * 32 + threadIdx.x];
#pragma unroll
        for (int w = CENTER_THREADS / 64; w; w >>= 1)
#pragma unroll
            for (int q = 0; q < w; ++q) x[q] += x[q + w];
        for (int off = 16; off; off >>= 1) x[0] += __shfl_xor_sync(0xFFFFFFFFu, x[0], off);
        if (threadIdx.x == 0) sh[CENTER_THREADS] = x[0];
    }
    __syncthreads();
    return sh[CENTER_THREADS];
}

// k_rowsum_reduce, k_center_u and k_center_r in one launch, for batches of tests of up to CENTER_ROWS rows: a CTA
// per test, up to two rows a thread.  The three kernels are latency (a launch, a few dependent loads,
// reductions); this one is bounded by one SM's FP64 rate, which holds it to tests of this size.  n = 200: 3.5 + 4.1 +
// 4.4 -> 7.3 us and two launches fewer (a call 86.6 -> 85.0 us; n = 400 the same as before within 0.5 %); 500 tests of
// n = 400 68 -> 23 us (their run 1,327 -> 1,259 us).
constexpr int CENTER_ROWS = 2 * CENTER_THREADS;
__global__ void __launch_bounds__(CENTER_THREADS) k_center_small(const Batch bt) {
    __shared__ double sh[CENTER_THREADS + 1];
    const int t = blockIdx.x, tid = threadIdx.x;
    const TestDesc &d = bt.desc[t];
    const int n = (int)d.n, n_pad = (int)d.n_pad, nkb = (int)contract_nkb(d);
    const int rows = n_pad > CENTER_THREADS ? 2 : 1;   // of a thread
    double r[2] = {0.0, 0.0};
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        if (m >= rows) break;
        const int i = tid + m * CENTER_THREADS;
        if (i < n) {
            const int I = i / PANEL;
            const double *rp = bt.rowpart + (d.blk0 + blk_index(I, KB_PER_PANEL * I, d.NKB)) * PANEL + i % PANEL;
            double acc = rp[0];
#pragma unroll 4
            for (int k = 1; k < nkb - KB_PER_PANEL * I; ++k) acc += rp[(int64_t)k * PANEL];
            for (int J = 0; J < I; ++J) acc += bt.colpart[(d.blk0 + blk_index(J, i / KB, d.NKB)) * KB + i % KB];
            r[m] = acc;
        }
        if (i < n_pad) bt.r[d.row0 + i] = r[m];
    }
    const double S = center_sum(r[0] + r[1], sh);
    double usum = 0.0;
    float u[2] = {0.f, 0.f}, mx = 0.f;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        if (m >= rows) break;
        const int i = tid + m * CENTER_THREADS;
        u[m] = i < n ? (float)(r[m] * d.inv_n - S * d.inv_2n2) : 0.f;
        if (i < n_pad) bt.u[d.row0 + i] = u[m];
        mx = fmaxf(mx, fabsf(u[m]));
        usum += (double)u[m];
    }
    const double U = center_sum(usum, sh);
    double rsum = 0.0;
    float mxd = 0.f;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        if (m >= rows) break;
        const int i = tid + m * CENTER_THREADS;
        const double rt = i < n ? r[m] - (double)n * (double)u[m] - U : 0.0;
        if (i < n_pad) bt.dcorr[d.row0 + i] = d.kappa * rt;
        mxd = fmaxf(mxd, (float)fabs(d.kappa * rt));
        rsum += rt;
    }
    for (int off = 16; off; off >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
        mxd = fmaxf(mxd, __shfl_xor_sync(0xFFFFFFFFu, mxd, off));
    }
    if ((tid & 31) == 0) {
        atomicMax(&bt.ctr[t].max_u_bits, __float_as_uint(mx));
        atomicMax(&bt.ctr[t].max_dc_bits, __float_as_uint(mxd));
    }
    const double St = center_sum(rsum, sh);
    // the readers add the parts of a test: the whole sum and zeros
    if (tid < n_pad / 32) bt.Spart[d.sp0 + tid] = tid == 0 ? S : 0.0;
    if (tid < d.NP) {
        bt.Upart[d.pan0 + tid] = tid == 0 ? U : 0.0;
        bt.Stpart[d.pan0 + tid] = tid == 0 ? St : 0.0;
    }
}

void launch_rowsums_center(const Batch &b, int64_t max_rows, cudaStream_t s) {
    if (b.n_tests <= 0) return;
    if (max_rows <= CENTER_ROWS) {
        k_center_small<<<(unsigned)b.n_tests, CENTER_THREADS, 0, s>>>(b);
    } else {
        launch_rowsum_reduce(b, s);
        launch_center(b, s);
    }
}

void launch_center(const Batch &b, cudaStream_t s) {
    if (b.npan_total <= 0) return;
    k_center_u<<<(unsigned)b.npan_total, 256, 0, s>>>(b);
    k_center_r<<<(unsigned)b.npan_total, 256, 0, s>>>(b);
}

// Packing.  Stored entry (i, j), j >= 256*panel(i):
//   j > i:  2 * ((D_ij - u_i) - u_j)      (upper triangle counted twice: s'Cs over
//                                           the upper triangle = the full form)
//   j = i:  D_ii - 2 u_i - dcorr_i
//   j < i or padding: 0
// FP32 in place (plain path), or (tuned path) c C split into FP16 hi + lo parts,
// hi = fp16(c C), lo = fp16(c C - hi), with the test's power-of-two scale c
// (packed_scale): |c C - hi - lo| <= 2^-22 |c C|, written over the block's own FP32
// storage (Batch::Chi / Clo with block stride c_stride), so the packed operand needs
// no memory of its own.  One CTA per block.
//
// Bound by the copy (8 bytes an entry) once there are blocks enough, by the latency of one block below.
// An FP64 instruction takes a warp 16 cycles of its SM, so the diagonal's three, issued row by row for one
// lane each, were the longest part of a diagonal block: now one row a lane.  n = 200: 8.7 -> 4.8 us;
// 500 tests of n = 400 (786 MB, 116 us at the copy rate): 170 -> 120 us; 512 tests of up to 4,000 rows
// 2,085 -> 1,845 us; n = 20,000: 267 -> 257 us (of 240).
template <bool SPLIT>
__global__ void __launch_bounds__(512) k_pack(const Batch bt) {
    const int64_t gb = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the whole block is read before any of it is rewritten: the split parts are
    // written over the block's own FP32 storage (hi in its first half, lo in its second).
    // Its loads do not wait for the block's test, descriptor and vectors.
    float2 dv[16];
#pragma unroll
    for (int q = 0; q < 16; ++q)
        dv[q] = __ldcs(reinterpret_cast<const float2 *>(bt.D + (gb * PANEL + warp * 16 + q) * KB + 2 * lane));
    const BlkInfo bi = bt.blk[gb];
    const TestDesc &d = bt.desc[bi.t];
    const int64_t n = d.n;
    const int64_t j0 = (int64_t)bi.kb * KB + 2 * lane;
    if ((int64_t)bi.kb * KB >= n) return;   // a K-block of padding: the build's zeros are also the split's
    const float *u = bt.u + d.row0;
    const double *dcorr = bt.dcorr + d.row0;
    const float uj[2] = {(j0 < n) ? u[j0] : 0.f, (j0 + 1 < n) ? u[j0 + 1] : 0.f};
    const int64_t row0 = (int64_t)bi.I * PANEL + warp * 16;   // 16 warps x 16 rows
    const float cs = SPLIT ? packed_scale(bt.ctr[bi.t]) : 1.f;
    // diagonal entries, one row a lane: FP64 arithmetic once for the warp's 16 rows, not row by row
    const bool on_diag = row0 / KB == bi.kb;   // the warp's rows cross the diagonal in this block, or none does
    float diag = 0.f;
    if (on_diag && lane < 16 && row0 + lane < n) {
        const int64_t i = row0 + lane;
        const float dii = bt.D[(gb * PANEL + warp * 16 + lane) * KB + (i - (int64_t)bi.kb * KB)];
        diag = (float)((double)dii - 2.0 * (double)u[i] - dcorr[i]);
    }
    if (SPLIT) __syncthreads();
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int64_t i = row0 + q;
        const float ui = (i < n) ? u[i] : 0.f;
        const float dq[2] = {dv[q].x, dv[q].y};
        const float di = on_diag ? __shfl_sync(0xFFFFFFFFu, diag, q) : 0.f;
        float w[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int64_t j = j0 + e;
            const float v = j == i ? di : 2.f * ((dq[e] - ui) - uj[e]);
            w[e] = (i < n && j < n && j >= i) ? v : 0.f;
        }
        const int64_t r = warp * 16 + q;
        if (SPLIT) {
            const float a0 = w[0] * cs, a1 = w[1] * cs;   // exact: cs is a power of two
            const __half h0 = __float2half_rn(a0), h1 = __float2half_rn(a1);
            const __half l0 = __float2half_rn(a0 - __half2float(h0));
            const __half l1 = __float2half_rn(a1 - __half2float(h1));
            const uint32_t hv = (uint32_t)__half_as_ushort(h0) | ((uint32_t)__half_as_ushort(h1) << 16);
            const uint32_t lv = (uint32_t)__half_as_ushort(l0) | ((uint32_t)__half_as_ushort(l1) << 16);
            const int64_t off = gb * bt.c_stride + r * KB + 2 * lane;
            *reinterpret_cast<uint32_t *>(bt.Chi + off) = hv;
            *reinterpret_cast<uint32_t *>(bt.Clo + off) = lv;
        } else {
            *reinterpret_cast<float2 *>(bt.D + (gb * PANEL + r) * KB + 2 * lane) = make_float2(w[0], w[1]);
        }
    }
}

void launch_pack(const Batch &b, bool split, cudaStream_t s) {
    if (b.nblk_total <= 0) return;
    if (split) k_pack<true><<<(unsigned)b.nblk_total, 512, 0, s>>>(b);
    else k_pack<false><<<(unsigned)b.nblk_total, 512, 0, s>>>(b);
}

// ---------------------------------------------------------------------------
// Plain FP32 contraction (the comparison path).  Work item = (test, chunk q =
// (panel I, K-blocks [kb0, kb1)), half h of the panel's rows, 64 relabeling columns):
//   U[b, i] = sum_{j in chunk} s_b[j] C[i, j]     (FP32 FMA, masks as 0/1 floats)
//   partial[(2q + h)][b] = sum_{i in half} s_b[i] U[b, i]
// 256 threads, each 4 relabelings x 8 rows; columns staged 32 at a time.
__global__ void __launch_bounds__(256) k_contract_simt(const Batch bt) {
    __shared__ float Cs[32][128 + 4];
    __shared__ uint32_t Ms[64];
    const int64_t w = blockIdx.x;
    const int tt = find_test(bt.pre.simt, bt.n_tests, w);
    const TestDesc d = bt.desc[tt];
    const int64_t lw = w - bt.pre.simt[tt];
    const int64_t tiles = d.Bp / 64;
    const int64_t q = lw / (2 * tiles), rem = lw % (2 * tiles);
    const int h = (int)(rem / tiles);
    const int64_t b0 = (rem % tiles) * 64;
    const Chunk ch = bt.chunks[d.chunk0 + q];
    const uint32_t *maskT = bt.maskT + d.mask0;
    const int64_t Bp = d.Bp;
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    float acc[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[a][r] = 0.f;

    for (int kb = ch.kb0; kb < ch.kb1; ++kb) {
        const float *blkp = bt.D + (d.blk0 + blk_index(ch.I, kb, d.NKB)) * (int64_t)(PANEL * KB) + (int64_t)h * 128 * KB;
        for (int sub = 0; sub < 2; ++sub) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int idx = e * 256 + t, r = idx >> 5, j = idx & 31;
                Cs[j][r] = blkp[(int64_t)r * KB + sub * 32 + j];
            }
            if (t < 64) Ms[t] = maskT[(int64_t)(2 * kb + sub) * Bp + b0 + t];
            __syncthreads();
            uint32_t mw[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) mw[a] = Ms[ty * 4 + a];
#pragma unroll 8
            for (int j = 0; j < 32; ++j) {
                const float4 c0 = *reinterpret_cast<const float4 *>(&Cs[j][tx * 8]);
                const float4 c1 = *reinterpret_cast<const float4 *>(&Cs[j][tx * 8 + 4]);
                const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float f = ((mw[a] >> j) & 1u) ? 1.f : 0.f;
#pragma unroll
                    for (int r = 0; r < 8; ++r) acc[a][r] = fmaf(f, cv[r], acc[a][r]);
                }
            }
            __syncthreads();
        }
    }
    // rows tx*8 .. tx*8+7 of this half lie in one mask word
    const int64_t word = (int64_t)ch.I * (PANEL / 32) + h * 4 + (tx >> 2);
    const int shift = (tx & 3) * 8;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int64_t b = b0 + ty * 4 + a;
        const uint32_t bits = (maskT[word * Bp + b] >> shift) & 0xFFu;
        float v = 0.f;
#pragma unroll
        for (int r = 0; r < 8; ++r) v += ((bits >> r) & 1u) ? acc[a][r] : 0.f;
        for (int off = 8; off; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        if (tx == 0) bt.partial[d.part0 + (2 * q + h) * Bp + b] = v;
    }
}

void launch_contract_simt(const Batch &b, cudaStream_t s) {
    if (b.nsimt_total <= 0) return;
    k_contract_simt<<<(unsigned)b.nsimt_total, 256, 0, s>>>(b);
}

// ---------------------------------------------------------------------------
// Final combination (Algorithm 1, statistic and p-value lines): per relabeling
// column b, Q_b = sum of its partials, stat_b = sign * (cT Q_b + S~/o^2).  The partials are summed
// in FP32 numbers that keep the roundings (pairs of a few partials, or a TripleSum of 64),
// which then meet in FP64 in a fixed order: this GPU's FP64 pipe takes 16 cycles for a
// warp's operation, so that with FP64 per partial, or per few of them, it is the limit.
// Then k_combine_count compares against stat_0 (the identity, evaluated by the same
// kernels): stat_b >= stat_0 and near-ties |stat_b - stat_0| <= 1e-5 |stat_0|.
// the statistic and the accumulation part of its error estimate (ept_internal.cuh, refine_ka)
// from the sum q of a column's partials and the sum a of their magnitudes
__device__ __forceinline__ void finish_stat(const Batch &bt, int t, const TestDesc &d, int64_t c, double q, double a,
                                            double St) {
    // the tensor-core path accumulates c Q (packed operand scaled by c); 1/c is exact
    const double inv_c = d.scaled ? (double)(1.f / packed_scale(bt.ctr[t])) : 1.0;
    bt.stats[d.col0 + c] = d.sign * (d.cT * (q * inv_c) + St * d.inv_o2);
    if (bt.errest) bt.errest[d.col0 + c] = d.ka * REFINE_U * d.cT * (a * inv_c);
}

// Many columns (a batch): a thread per column (256 per CTA), eight partials at a time (their
// loads in flight together), 64 to a TripleSum and as many magnitudes to another, those in FP64.
// The kernel below makes 16 FP64 merges per column whatever its partials, 1.08 ms for 512
// uneven tests (2.6 million columns, 50 partials on average, 0.5 GB); this one takes 0.31 ms (0.29 with
// FP32 pairs of eight and the magnitudes in one FP32 sum, which is less than the other kernel keeps).  It
// needs two CTAs per SM to pay (COMBINE_COLUMNS_PER_SM): with few columns a thread's chain of loads
// is longer than the sixteen warps' (5000 columns of 50 partials: 8 us against 6).  Tests of more
// partials than COMBINE_THREAD_PARTS keep the other.
constexpr int64_t COMBINE_THREAD_PARTS = 1024;
constexpr int64_t COMBINE_COLUMNS_PER_SM = 512;
__global__ void __launch_bounds__(256) k_combine_columns(const Batch bt) {
    __shared__ double bSt;
    const int64_t gc0 = (int64_t)blockIdx.x * 256;
    const int t = find_test(bt.pre.cols, bt.n_tests, gc0);
    const TestDesc &d = bt.desc[t];
    const int64_t nparts = d.nparts;
    if (nparts > COMBINE_THREAD_PARTS) return;
    if (threadIdx.x < 32) {
        const double St = warp_ordered_sum(bt.Stpart + d.pan0, d.NP);
        if (threadIdx.x == 0) bSt = St;
    }
    __syncthreads();
    const int64_t c = gc0 + threadIdx.x - bt.pre.cols[t];
    if (c >= d.ncols) return;
    const int64_t Bp = d.Bp;
    const float *part = bt.partial + d.part0 + c;
    double q = 0.0, a = 0.0;
    for (int64_t k1 = 0; k1 < nparts; k1 += 64) {
        const int64_t end = k1 + 64 < nparts ? k1 + 64 : nparts;
        TripleSum sum, mag;
        for (int64_t k0 = k1; k0 < end; k0 += 8) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = k0 + k < nparts ? part[(k0 + k) * Bp] : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                sum.add(v[k]);
                mag.add(fabsf(v[k]));
            }
        }
        q += sum.value();
        a += mag.value();
    }
    finish_stat(bt, t, d, c, q, a, bSt);
}

// Tests of more partials: a CTA covers 32 columns of one test (the column padding is a multiple of
// 256): lane l of each of its 16 warps reads column l of every 16th partial (one coalesced 128-byte
// row per load, eight loads in flight), and the 16 warp sums are added in a fixed
// order (deterministic).
__global__ void __launch_bounds__(512) k_combine_stats(const Batch bt, int64_t above) {
    constexpr int NW = 16;   // warps: parts k = warp, warp + NW, ...
    __shared__ double bSt;
    __shared__ double ws[NW][32], wa[NW][32];
    const int64_t gc0 = (int64_t)blockIdx.x * 32;
    const int t = find_test(bt.pre.cols, bt.n_tests, gc0);
    const TestDesc &d = bt.desc[t];
    if (d.nparts <= above) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        const double St = warp_ordered_sum(bt.Stpart + d.pan0, d.NP);
        if (lane == 0) bSt = St;
    }
    const int64_t c = gc0 + lane - bt.pre.cols[t];
    const int64_t Bp = d.Bp, nparts = d.nparts;
    const float *part = bt.partial + d.part0 + c;
    // a warp's parts summed as an unevaluated FP32 pair (TwoSum: each addition's
    // rounding error is kept exactly), so that no FP64 operation runs per partial;
    // the pairs of the warps then meet in FP64 in a fixed order
    float h = 0.f, l = 0.f, aabs = 0.f;
#pragma unroll 8
    for (int64_t k = warp; k < nparts; k += NW) {
        const float v = part[k * Bp];
        float s2, e;
        two_sum(h, v, s2, e);
        h = s2;
        l += e;
        aabs += fabsf(v);
    }
    ws[warp][lane] = (double)h + (double)l;
    wa[warp][lane] = (double)aabs;
    __syncthreads();
    if (warp == 0) {
        double q = 0.0, a = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            q += ws[w][lane];
            a += wa[w][lane];
        }
        // the tensor-core path accumulates c Q (packed operand scaled by c); 1/c is exact
        const double inv_c = d.scaled ? 1.0 / (double)packed_scale(bt.ctr[t]) : 1.0;
        if (c < d.ncols) {
            bt.stats[d.col0 + c] = d.sign * (d.cT * (q * inv_c) + bSt * d.inv_o2);
            // accumulation part of the error estimate (ept_internal.cuh, refine_ka)
            if (bt.errest) bt.errest[d.col0 + c] = d.ka * REFINE_U * d.cT * (a * inv_c);
        }
    }
}

// Errors of test t that the host will report: non-finite data, malformed
// relabelings, a median bandwidth that is not positive and finite.
__device__ __forceinline__ bool test_failed(const Batch &bt, int t) {
    const Counters &k = bt.ctr[t];
    bool f = k.nonfinite || k.bad_mask;
    if (bt.desc[t].median) {
        const float sg = __uint_as_float(k.sel_prefix);
        f = f || !(sg > 0.f) || !isfinite(sg);
    }
    return f;
}

// Whether any test of a batch failed (one CTA): a batched call that returns an
// error writes none of its device outputs.
__global__ void __launch_bounds__(256) k_batch_status(const Batch bt) {
    int bad = 0;
    for (int t = threadIdx.x; t < bt.n_tests; t += blockDim.x) bad |= test_failed(bt, t) ? 1 : 0;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0 && bad) bt.ctr[0].batch_failed = 1ull;
}

// Counting and outputs: a CTA covers 256 columns of one test.  A caller's device
// buffer of permuted statistics is written only when the call will succeed (no
// error in any test of the call, no expired wait), so that output buffers are
// written only on success.
// With `flag` (the first count of a run), also the error criterion: statistic c is
// flagged for FP64 recomputation when E_c > REFINE_TOL |stat_c| (ept_internal.cuh).
__global__ void __launch_bounds__(256) k_combine_count(const Batch bt, int flag) {
    __shared__ double bW;
    const int64_t gc = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int t = find_test(bt.pre.cols, bt.n_tests, (int64_t)blockIdx.x * 256);
    const TestDesc d = bt.desc[t];
    const int64_t c = gc - bt.pre.cols[t];
    const double obs = bt.stats[d.col0];
    if (flag && bt.flags) {
        if (threadIdx.x < 32) {
            const double S = warp_ordered_sum(bt.Spart + d.sp0, d.n_pad / 32);
            if (threadIdx.x == 0) bW = S * d.inv_n * d.inv_n;
        }
        __syncthreads();
        int fl = 0;
        if (c < d.ncols) {
            const double v = bt.stats[d.col0 + c];
            const double rep = REFINE_KR * REFINE_U * fabs(bW) / (double)d.m;
            // errest holds refine_ka u cT A; the observed and aligned statistics take REFINE_KC_RATIO times it
            const double e0 = REFINE_KC_RATIO * bt.errest[d.col0] + rep;
            const bool aligned = c == 0 || fabs(v - obs) <= REFINE_TOL * fabs(obs) + 2.0 * e0;
            const double acc = aligned ? REFINE_KC_RATIO * bt.errest[d.col0 + c] : bt.errest[d.col0 + c];
            const double tol = REFINE_TOL * fabs(v);
            // flagged when the estimate exceeds the tolerance; 2 (rebuild the entries in FP64)
            // when the representation term exceeds REFINE_L2 of it, else 1 (re-sum the
            // packed operand exactly).  NaN-safe: a non-finite estimate takes the rebuild
            const int lvl = !(acc + rep <= tol) ? (!(rep <= REFINE_L2 * tol) ? 2 : 1) : 0;
            fl = lvl != 0;
            bt.flags[d.col0 + c] = (uint8_t)lvl;
        }
        fl = __syncthreads_count(fl);
        if (threadIdx.x == 0 && fl) atomicAdd(&bt.ctr[t].n_flag, (unsigned long long)fl);
    }
    int ge = 0, near = 0;
    if (c >= 1 && c < d.ncols) {
        const double v = bt.stats[d.col0 + c];
        ge = v >= obs;
        near = fabs(v - obs) <= 1e-5 * fabs(obs);
        if (d.out_stats) {
            if (!test_failed(bt, t) && !bt.ctr[0].err_code && !bt.ctr[0].batch_failed) d.out_stats[c - 1] = v;
        }
    }
    if (c == 0) bt.observed[t] = obs;
    ge = __syncthreads_count(ge);
    near = __syncthreads_count(near);
    if (threadIdx.x == 0) {
        if (ge) atomicAdd(&bt.ctr[t].n_ge, (unsigned long long)ge);
        if (near) atomicAdd(&bt.ctr[t].n_near, (unsigned long long)near);
    }
}

void launch_combine(const Batch &b, int num_sms, cudaStream_t s) {
    if (b.ncols_total <= 0) return;
    if (b.n_tests > 1) k_batch_status<<<1, 256, 0, s>>>(b);
    const bool columns = b.ncols_total >= COMBINE_COLUMNS_PER_SM * num_sms && b.parts_min <= COMBINE_THREAD_PARTS;
    if (columns) k_combine_columns<<<(unsigned)(b.ncols_total / 256), 256, 0, s>>>(b);
    if (!columns || b.parts_max > COMBINE_THREAD_PARTS)
        k_combine_stats<<<(unsigned)(b.ncols_total / 32), 512, 0, s>>>(b, columns ? COMBINE_THREAD_PARTS : 0);
    k_combine_count<<<(unsigned)(b.ncols_total / 256), 256, 0, s>>>(b, 1);
}

void launch_combine_count(const Batch &b, cudaStream_t s) {
    if (b.ncols_total <= 0) return;
    k_combine_count<<<(unsigned)(b.ncols_total / 256), 256, 0, s>>>(b, 0);
}

__global__ void k_reset_counts(Counters *ctr, int n_tests) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n_tests) {
        ctr[t].n_ge = 0;
        ctr[t].n_near = 0;
    }
}

void launch_reset_counts(const Batch &b, cudaStream_t s) {
    if (b.n_tests <= 0) return;
    k_reset_counts<<<(unsigned)((b.n_tests + 255) / 256), 256, 0, s>>>(b.ctr, b.n_tests);
}

// ---------------------------------------------------------------------------
// Expand one test's packed upper storage into a full row-major n x n matrix
// (checking aid).
__global__ void k_expand(const float *__restrict__ D, int64_t n, int64_t NKB, float *__restrict__ out) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * n) return;
    int64_t i = idx / n, j = idx % n;
    if (j / PANEL < i / PANEL) {
        const int64_t tmp = i;
        i = j;
        j = tmp;
    }
    const int64_t I = i / PANEL, kb = j / KB;
    out[idx] = D[(blk_index(I, kb, NKB) * PANEL + (i - I * PANEL)) * KB + (j - kb * KB)];
}

void launch_expand_blocks(const float *D, int64_t n, int64_t NKB, float *out, cudaStream_t s) {
    const int64_t tot = n * n;
    if (tot <= 0) return;
    k_expand<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(D, n, NKB, out);
}

// ---------------------------------------------------------------------------
// Debug checks: one CTA per guard band fills it with a pattern that depends on the
// band's index, or counts the words that no longer hold it.
__global__ void k_guards(uint8_t *arena, GuardList g, int check, Counters *ctr) {
    const int k = blockIdx.x;
    if (k >= g.n) return;
    uint32_t *w = reinterpret_cast<uint32_t *>(arena + g.off[k]);
    const uint32_t pat = 0xA5C3E1F0u ^ (uint32_t)(k * 0x9E3779B9u);
    unsigned bad = 0;
    for (int i = threadIdx.x; i < GUARD_BYTES / 4; i += blockDim.x) {
        if (check) bad += (w[i] != (pat ^ (uint32_t)i));
        else w[i] = pat ^ (uint32_t)i;
    }
    if (check) {
        for (int off = 16; off; off >>= 1) bad += __shfl_xor_sync(0xFFFFFFFFu, bad, off);
        if ((threadIdx.x & 31) == 0 && bad) atomicAdd(&ctr->guard_bad, (unsigned long long)bad);
    }
}

void launch_guards(uint8_t *arena, const GuardList &g, bool check, Counters *ctr, cudaStream_t s) {
    if (g.n <= 0) return;
    k_guards<<<(unsigned)g.n, 32, 0, s>>>(arena, g, check ? 1 : 0, ctr);
}

}  // namespace ept

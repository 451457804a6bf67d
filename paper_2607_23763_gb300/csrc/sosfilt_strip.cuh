// Persistent single-signal kernel for cascades whose memory is finite in float32, sm_103a: the signal
// is cut into one strip of consecutive samples per thread block, and no block takes another's state.
//
// The zero-input transition of a stable cascade over H samples, M1^H, decays to matrices whose float32
// entries are all zero; from there on a state H samples old adds nothing to the carried one (Eq. 25 with
// the terms the float32 tables hold as zeros left out).  The host finds that memory once per filter
// (warm_rows, in rows of 64 samples).  A block then starts its strip warm_rows rows early from zero state,
// which gives it the strip's true incoming state, and carries the state from unit to unit inside the
// block: no lookback across blocks, no descriptors, the same composition on every run.  Only in place
// does a block wait for another: a strip's last rows are stored once the next strip has read them as its
// warm-up (a word per strip; strips are taken from the last one down, so the block waited for is running
// or done).  Which signals are cut, and how: sosfilt_strip_rule.h.
//
// A unit is 128 rows of N = 64 samples, staged in shared memory with the 16-byte chunks of a row permuted
// by the row number (a lane reads its own row without bank conflicts).  Per unit:
//   1. terminal states of the rows under zero state (Sec. II-C).
//      kStripFma (one or two sections, short or misaligned signals): each lane multiplies its row with the
//      2 or 4 state responses by FMAs.
//      kStripStates (one or two sections, long; more, quiet): T = X G^T, the rows times the 64 state responses,
//      by tcgen05.mma with the rows in tensor memory.
//      kStripOutputs (three sections and more): [Y | T] = X [T^T | G^T], the rows' zero-state outputs by the lower
//      triangular Toeplitz matrix of the impulse response as well.
//      The products are of split operands in TF32: the samples as the nearest TF32 values (11 bits) and exact
//      remainders (12 bits, of which the tensor core reads 11), the tables as nearest TF32 values and remainders
//      rounded to TF32.  kStripStates takes all four partial products, into separate accumulators for the large and
//      the small terms, which the epilogue adds; kStripOutputs leaves remainder times remainder out (3 % of the
//      error) and takes the small terms first, into one accumulator.
//   2. lane scan (Sec. II-C's recursive doubling) of each warp's 32 rows, fold of the four groups'
//      carries, and the unit's incoming state Z' = (A_C)^4 Z + c from the previous unit's.
//   3. every row's true incoming state S_l + (M_N)^l Z (Eq. 24 at the rows' starts), and from it the outputs:
//      by the sections' recurrences over the row in place, skewed by one sample per section, 4 FMAs per section
//      and sample and no separate correction pass (the lookback kernel's particular pass and correction are 6);
//      or, kStripOutputs, by a second product onto the first, Y += St H^T with the rows' states as an operand of
//      two TF32 words (three partial products).
//   4. coalesced stores, through a staging buffer and by TMA where the outputs are in tensor memory.
// Groups of warm-up rows stop after step 2.  Samples that are not finite, or so large that their nearest TF32
// value is not: rows_again, rows_plainly; what follows a strip that ends in such a state: the last block.
//
// Warp roles (one block per SM; the first eight warps give registers to the others):
//   warps 0, 2, 3  load the units' samples: TMA where x and y are 16-byte aligned and strips long, by one thread;
//                  else cp.async (zero-filled past the end, any alignment)
//   warp 1         tensor-memory owner; issues the products
//   warps 4-7      split the rows into the products' operands, in tensor memory (two buffers)
//   warps 8 on     three or four warpgroups, one unit each in turn; warp q of a warpgroup takes rows
//                  32q .. 32q+31
// Without the tensor cores warps 0-7 all load.
// Every wait is bounded by the spin budget, and those for a block's own copies and products at its end by kStripDrain.
#pragma once
#include <cstring>

#include "sosfilt_lane.cuh"
#include "sosfilt_tcgen05.cuh"

namespace sosk {

constexpr int kStripXBytes = kStripUnit * 4;       // one staged unit: two column halves of 16 KB
constexpr int kStripHalf = kStripXBytes / 2;
constexpr int kStripDS = 4;                        // accumulator slots, ahead of the operand buffers
constexpr int kStripZ = 8;                         // units' incoming states kept (more than are in hand)
constexpr int kStripBars = 384;                    // bytes of barriers and shared words
constexpr long long kStripDrain = 2000000000LL;    // cycles a block waits for its own products at exit

// What the tensor cores do for a unit.
enum StripMode {
    kStripFma = 0,       // nothing: terminal states by FMAs, outputs by the recurrences
    kStripStates = 1,    // terminal states; outputs by the recurrences
    kStripOutputs = 2    // terminal states and outputs
};

template <int K, int MODE>
struct StripDims {
    using Dm = LaneDims<K, kStripN, kLaneW>;
    static constexpr int S = 2 * K;
    static constexpr bool TC = MODE != kStripFma, MM = MODE == kStripOutputs;
    // epilogue warpgroups, and the registers that a thread of the first two warpgroups (SREGS) and of theirs
    // (REGS) then has: 256 x 64 + 512 x 88 or 256 x 48 + 512 x 96 of 768 x 80 at launch; the recurrences of five
    // and more sections want 128: 256 x 48 + 384 x 128 of 640 x 96 (four warpgroups with 96: 5 % slower)
    static constexpr int WGS = MM || K <= 4 ? 4 : 3;
    static constexpr int SREGS = MM || K > 4 ? 48 : 64;
    static constexpr int REGS = MM ? 96 : K <= 4 ? 88 : 128;
    static constexpr int THREADS = 256 + 128 * WGS;
    static constexpr int LOADERS = TC ? 3 : 8;  // loading warps
    static constexpr int U = TC ? 1 : 8;        // chunks of the recurrences unrolled
    // tensor memory: four accumulator slots (states only: two sets of 16 + 16 columns for the large and the
    // small terms; outputs: 64, the terminal states' 16 and, in their place later, the row states' operand
    // of 16 + 16), then the samples' operands, one buffer for each half of the rows (32 columns of heads and 32
    // of remainders: while a half is multiplied the other is written)
    static constexpr int COLS = MM ? 96 : 64;
    static constexpr int ACOL = kStripDS * COLS;
    static_assert(ACOL + 2 * 64 <= 512, "tensor memory");
    // shared memory: staged units, operand image, the output staging (half a row for each of a
    // warp's rows), then floats: (M_N)^b for b = 0 .. 7 and 8, 16, 24, (A_C)^v for v = 1 .. 4, the warpgroups' local carries (two slots), group states, unit states;
    // and the barriers
    // the operand image in shared memory; with outputs, of [T | G]'s second column half only rows 32 .. 79,
    // the others being zeros that no product takes
    static constexpr int B1 = (80 + 48) * 128;  // heads or remainders of [T | G]
    static constexpr int IMG = MM ? 2 * B1 + 64 * 128 : 4 * kStripImgFloats;
    static constexpr int STAGE = MM ? 4 * WGS * 4096 : 0;
    
    // from three sections on, the rows' states are formed by two-word products (state_mv2): a warp's four group
    // states then have every word twice, at a pitch that puts the four on different banks.  Shorter cascades
    // have too few products to gain by it (order 2, 2^22 samples: 11.9 us against 11.2)
    static constexpr bool TWO = K > 2;
    static constexpr int ZW = TWO ? 2 : 1, ZP = !TWO ? S : 2 * S + (S % 8 == 6 ? 8 : 4);
    static constexpr int T_ML = 0;
    static constexpr int T_ACP = T_ML + 11 * Dm::MS;
    static constexpr int T_A = T_ACP + 4 * S * S;
    static constexpr int T_ZV = T_A + WGS * 2 * 4 * S;
    static constexpr int T_Z = T_ZV + WGS * 4 * 4 * ZP;
    // the output basis H [S][64] and the states of the signal's first group (row_part), strip 0 only
    static constexpr int T_H = T_Z + kStripZ * S;
    static constexpr int T_ST = T_H + kStripN * S;
    static constexpr int T_END = T_ST + (MM ? 0 : 32 * S);
    static constexpr int FIXED = IMG + STAGE + 4 * T_END + kStripBars;
    static constexpr int XS_FIT = (227 * 1024 - FIXED) / kStripXBytes;
    static constexpr int XS = XS_FIT > 6 ? 6 : XS_FIT;  // staged units
    static_assert(XS >= (MM ? 3 : WGS + 2), "units in the epilogue (with outputs: in the products) and two loading");
    static constexpr int OFF_IMG = XS * kStripXBytes;
    static constexpr int OFF_STAGE = OFF_IMG + IMG;
    static constexpr int OFF_TAB = OFF_STAGE + STAGE;
    static constexpr int OFF_BAR = OFF_TAB + 4 * T_END;
    static constexpr size_t SMEM = OFF_BAR + kStripBars;
};

// Strips of at least this many rows take TMA copies.
constexpr int kStripTmaRows = 4 * kStripRows;
// A signal's full rows of 64 samples as a tensor map, copied in boxes of 32 x box_rows (sosfilt_tc.cu).
bool strip_rows_map(CUtensorMap *tm, const float *base, long long rows, int box_rows);

// The recurrences' coefficients of the sections s and s + H, H = K / 2, in one word each (lane_recurrence): -a1,
// -a2, and of the sections after them b1, b2, b0 (zero past the last).
template <int K>
struct StripPairs {
    static constexpr bool TWO = K > 2 && K % 2 == 0;
    static constexpr int H = (K + 1) / 2;
    unsigned long long a1[H], a2[H], b1[H], b2[H], b0[H];
};

template <int K, int MODE>
struct StripParams {
    LaneParams<K> p;
    int in_place;      // y == x: a strip's tail is stored once the next strip has read it
    int x_aligned, y_aligned;  // 16-byte aligned
    int tma;           // tmx and tmy are set: full units are loaded, full groups' outputs stored by TMA
    CUtensorMap tmx, tmy;  // x and y as [rows][64], boxes of 32 x 128 and 32 x 32, 128-byte swizzle
    unsigned long long host_tickets;  // what the host adds to the lookback kernels' ticket base
    StripPairs<K> pk;
    float g[MODE == kStripFma ? 2 * K : 1][kStripN];  // without the tensor cores: the state responses
};

__device__ __forceinline__ bool mbar_test(unsigned long long *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// mbar_wait whose hardware suspension is never longer than the budget.
__device__ __forceinline__ bool strip_wait1(unsigned long long *bar, unsigned parity, long long budget, int *status) {
    if (mbar_test(bar, parity)) return true;
    if (budget < kSuspendHintNs / 2) {  // a budget below a suspension: no suspension
        const long long t0 = clock64();
        while (!mbar_test(bar, parity))
            if (clock64() - t0 > budget) {
                atomicOr(status, kDevErrTimeout);
                return false;
            }
        return true;
    }
    const unsigned hint = budget < kSuspendHintNs ? static_cast<unsigned>(budget) : kSuspendHintNs;
    const long long t0 = clock64();
    while (!mbar_try_wait_sleep(bar, parity, hint)) {
        if (clock64() - t0 > budget) {
            atomicOr(status, kDevErrTimeout);
            return false;
        }
    }
    return true;
}
// The same for a whole warp: one answer for its lanes.
__device__ __forceinline__ bool strip_wait(unsigned long long *bar, unsigned parity, long long budget, int *status) {
    return __all_sync(0xffffffffu, strip_wait1(bar, parity, budget, status));
}

// cp.async of 16 or 4 bytes to a shared-memory address, the bytes past `bytes` zero-filled.
__device__ __forceinline__ void cp_async16_s(unsigned dst, const float *src, unsigned bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4_s(unsigned dst, const float *src, unsigned bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Arrival on a shared-memory barrier once the thread's earlier cp.async copies have landed.
__device__ __forceinline__ void cp_async_arrive(unsigned long long *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Barrier of `threads` threads that is also a vote: true when every thread brought true.
__device__ __forceinline__ bool named_bar_and(int id, int threads, bool ok) {
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(static_cast<unsigned>(ok)), "r"(id), "r"(threads)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Two float32 in one 64-bit word, and a b + c on both at once.
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ void unpack2(unsigned long long v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

// The sections' recurrences over one row (64 samples, in place) from the row's true incoming state st
// (transposed direct form II), sections skewed by one sample each and in direct-form-I order as in
// lane_particular: a state word z1, z2 enters its section's input at the section's samples 0 and 1.
// Chunk j (four samples) of the row lies at half j / 8, 16-byte slot (j ^ row) & 7; `row` is the offset
// of chunk 0 in the shared memory sm.  Unrolled by U chunks: with U = 8 the whole row, so that a short signal's few warps overlap
// the loads and stores with the dependent FMAs of a step (one section, one warp per scheduler: 1000 cycles
// a row instead of 2800); with U = 1 the code stays small where every scheduler has work (unrolling by 2 to
// 8 cost 7 to 17 % at orders 2 to 16 on 2^26 samples and more, in instruction fetches).
//
// Four, six and eight sections (TWO): the steps take sections s and s + H, H = K / 2, in one two-word product
// each, with the coefficients from `pk` (StripPairs): the inputs of the pair s are the outputs of the pair
// s - 1 as they lie, and only the pair 0 puts two words together.  The same products in the same order, in half
// the issue slots, which is what bounds the recurrences here: 2^28 samples, order 8 486 -> 460 us, order 12
// 605 -> 586, order 16 751 -> 677.  An odd count wastes half a pair (orders 6 and 10 were 3 and 7 % slower
// so); two sections are one pair that waits on itself.
template <int K, bool NORM, int U, class Secs>
__device__ __forceinline__ void lane_recurrence(const Secs &cs, const StripPairs<K> &pk, unsigned char *sm, unsigned row,
                                                float gain, const float (&st)[2 * K]) {
    constexpr int N = kStripN, D = K - 1, R0 = (4 - (D & 3)) & 3, D4 = (D + R0) / 4;
    constexpr int C0 = ((K + 1 + 3) / 4 + U - 1) / U * U;  // chunks in which some section starts: unrolled
    float y1[K], y2[K], pipe[K];
#pragma unroll
    for (int s = 0; s < K; ++s) y1[s] = y2[s] = pipe[s] = 0.f;
    float x1 = 0.f, x2 = 0.f;
    float carry[R0 > 0 ? R0 : 1];
#pragma unroll
    for (int r = 0; r < (R0 > 0 ? R0 : 1); ++r) carry[r] = 0.f;
    unsigned at[D4 + 1];  // offsets of the last chunks read: the outputs follow D + R0 samples behind
#pragma unroll
    for (int r = 0; r <= D4; ++r) at[r] = row;
    auto section = [&](int s, float F) -> float {
        const float4 c = cs.c(s);
        const float y = fmaf(c.z, y1[s], fmaf(c.w, y2[s], F));
        if (s + 1 < K) {  // F_{s+1} before the history moves
            const float4 n = cs.c(s + 1 < K ? s + 1 : s);
            const float by = NORM ? y : cs.b0(s + 1 < K ? s + 1 : s) * y;
            pipe[s] = fmaf(n.x, y1[s], fmaf(n.y, y2[s], by));
        }
        y2[s] = y1[s];
        y1[s] = y;
        return y;
    };
    // section s at its sample m = 0 or 1, its state words still to come in
    auto section_start = [&](int s, int m, float F) -> float {
        const float4 c = cs.c(s);
        const float y = m == 0 ? F + st[2 * s] : fmaf(c.z, y1[s], F + st[2 * s + 1]);
        if (s + 1 < K) {
            const float4 n = cs.c(s + 1 < K ? s + 1 : s);
            const float by = NORM ? y : cs.b0(s + 1 < K ? s + 1 : s) * y;
            pipe[s] = m == 0 ? by : fmaf(n.x, y1[s], by);
        }
        y2[s] = y1[s];
        y1[s] = y;
        return y;
    };
    auto input = [&](float x) -> float {
        const float gx = NORM ? x * gain : x;
        const float4 c0 = cs.c(0);
        const float F = fmaf(c0.x, x1, fmaf(c0.y, x2, NORM ? gx : cs.b0(0) * gx));
        x2 = x1;
        x1 = gx;
        return F;
    };
    // one chunk of four steps, `first` its first step where that is below C0 (else only >= C0 matters)
    auto chunk = [&](unsigned a, const float4 &xv, int first) {
#pragma unroll
        for (int r = D4; r > 0; --r) at[r] = at[r - 1];
        at[0] = a;
        const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
        float out[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = first + j;
#pragma unroll
            for (int s = K - 1; s >= 1; --s) {
                if (i - s < 0) continue;
                const float w = i - s < 2 ? section_start(s, i - s, pipe[s - 1]) : section(s, pipe[s - 1]);
                if (s == K - 1) out[j] = w;
            }
            const float F = input(xs[j]);
            const float w0 = i < 2 ? section_start(0, i, F) : section(0, F);
            if (K == 1) out[j] = w0;
        }
        if (first - D - R0 >= 0) {  // out[j] is sample first + j - D
            float blk[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) blk[r] = r < R0 ? carry[r] : out[r - R0];
            *reinterpret_cast<float4 *>(sm + at[D4]) = make_float4(blk[0], blk[1], blk[2], blk[3]);
        }
#pragma unroll
        for (int r = 0; r < R0; ++r) carry[r] = out[4 - R0 + r];
    };
    // `row` carries the row's permutation in its bits 4..6, so chunk j of a half is at row ^ 16 j
    auto at_chunk = [&](int j) -> unsigned { return (row ^ ((j & 7) << 4)) + (j >> 3) * kStripHalf; };
    auto get = [&](unsigned a) { return *reinterpret_cast<const float4 *>(sm + a); };
    float4 xn = get(row);
#pragma unroll
    for (int j = 0; j < C0; ++j) {
        const float4 xv = xn;
        if (j + 1 < N / 4) xn = get(at_chunk(j + 1));
        chunk(at_chunk(j), xv, 4 * j);
    }
    if constexpr (StripPairs<K>::TWO) {
        using W = unsigned long long;
        constexpr int H = StripPairs<K>::H, LAST = H - 1;  // the pair whose second section is the last
        static_assert(U == 1);
        W Y1[H], Y2[H], PP[H];
#pragma unroll
        for (int s = 0; s < H; ++s) {
            Y1[s] = pack2(y1[s], y1[s + H]);
            Y2[s] = pack2(y2[s], y2[s + H]);
            PP[s] = pack2(pipe[s], pipe[s + H]);
        }
#pragma unroll 1
        for (int j0 = C0; j0 < N / 4; ++j0) {
            const float4 xv = xn;
            if (j0 + 1 < N / 4) xn = get(at_chunk(j0 + 1));
#pragma unroll
            for (int r = D4; r > 0; --r) at[r] = at[r - 1];
            at[0] = at_chunk(j0);
            const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
            float out[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float mid, over;  // the input of section H: what section H - 1 left in the last step
                unpack2(PP[H - 1], mid, over);
                const float F0 = input(xs[j]);
#pragma unroll
                for (int s = H - 1; s >= 0; --s) {
                    const W F = s > 0 ? PP[s > 0 ? s - 1 : 0] : pack2(F0, mid);
                    const W y = fma2(pk.a1[s], Y1[s], fma2(pk.a2[s], Y2[s], F));
                    W by = y;
                    if constexpr (!NORM) asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(by) : "l"(pk.b0[s]), "l"(y));
                    PP[s] = fma2(pk.b1[s], Y1[s], fma2(pk.b2[s], Y2[s], by));
                    Y2[s] = Y1[s];
                    Y1[s] = y;
                    if (s == LAST) unpack2(y, over, out[j]);
                }
            }
            float blk[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) blk[r] = r < R0 ? carry[r] : out[r - R0];
            *reinterpret_cast<float4 *>(sm + at[D4]) = make_float4(blk[0], blk[1], blk[2], blk[3]);
#pragma unroll
            for (int r = 0; r < R0; ++r) carry[r] = out[4 - R0 + r];
        }
#pragma unroll
        for (int s = 0; s < H; ++s) {
            unpack2(Y1[s], y1[s], y1[s + H]);
            unpack2(Y2[s], y2[s], y2[s + H]);
            unpack2(PP[s], pipe[s], pipe[s + H]);
        }
    } else {
#pragma unroll 1
    for (int j0 = C0; j0 < N / 4; j0 += U) {
        const unsigned b = at_chunk(j0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float4 xv = xn;
            if (u + 1 < U)
                xn = get(b ^ ((u + 1) << 4));
            else if (j0 + U < N / 4)
                xn = get(at_chunk(j0 + U));
            chunk(b ^ (u << 4), xv, 4 * C0);
        }
    }
    }
    // drain: steps N .. N + D - 1, in which only the sections s > step - N are still running
    if constexpr (D > 0) {
        float tail[R0 + D];
#pragma unroll
        for (int r = 0; r < R0; ++r) tail[r] = carry[r];
#pragma unroll
        for (int e = 0; e < D; ++e) {
#pragma unroll
            for (int s = K - 1; s >= e + 1; --s) {
                const float w = section(s, pipe[s - 1]);
                if (s == K - 1) tail[R0 + e] = w;
            }
        }
#pragma unroll
        for (int r = 0; r < D4; ++r)
            *reinterpret_cast<float4 *>(sm + at[D4 - 1 - r]) =
                make_float4(tail[4 * r], tail[4 * r + 1], tail[4 * r + 2], tail[4 * r + 3]);
    }
}

// The signal's first group: an initial state may be thousands of times the outputs that are left of it, and 64
// steps of the recurrences from it err by as many roundings of the coefficients; so there the recurrences run
// from zero state and the state's part (Eq. 24) is added from the output basis H ([2K][64], float64-derived),
// both in shared memory.
template <int K>
__device__ __forceinline__ void row_part(unsigned char *sm, unsigned row, const float *H, const float *st) {
#pragma unroll(K <= 2 ? 8 : 2)
    for (int j = 0; j < kStripN / 4; ++j) {
        float4 *a = reinterpret_cast<float4 *>(sm + (row ^ ((j & 7) << 4)) + (j >> 3) * kStripHalf);
        float4 v = *a;
#pragma unroll
        for (int s = 0; s < 2 * K; ++s) {
            const float4 b = *reinterpret_cast<const float4 *>(H + s * kStripN + 4 * j);
            const float z = st[s];
            v.x = fmaf(b.x, z, v.x);
            v.y = fmaf(b.y, z, v.y);
            v.z = fmaf(b.z, z, v.z);
            v.w = fmaf(b.w, z, v.w);
        }
        *a = v;
    }
}

// A chunk of four samples k .. k + 3 of a group whose own samples are from .. to - 1 (from a multiple of four).
__device__ __forceinline__ void put4(float *y, int k, int from, int to, const float4 &v) {
    if (k >= from && k + 4 <= to) {
        __stcs(reinterpret_cast<float4 *>(y + k), v);
    } else if (k >= from) {
        if (k + 0 < to) y[k] = v.x;
        if (k + 1 < to) y[k + 1] = v.y;
        if (k + 2 < to) y[k + 2] = v.z;
    }
}

// A warp's rows whose products are worth nothing (`bad`), from the signal to the output directly: by the sections one
// after the other (transposed direct form II) from the rows' states, which are in the 16 + 16 columns at d.  The group's
// first sample is `base`, its own are from .. to - 1.  Rare, and small rather than fast.
template <int K>
__device__ __noinline__ void rows_plainly(const LaneParams<K> &p, unsigned d, bool bad, long long base, int from, int to) {
    float e[16], l[16];
    tc_ldn<16>(d, e);
    tc_ldn<16>(d + 16, l);
    tc_wait_ld();
    const int k = (threadIdx.x & 31) * kStripN;
    if (bad && k >= from && k < to) {
        const long long at = base + k;
        const int count = to - k < kStripN ? to - k : kStripN;
        float z[2 * K];
        for (int s = 0; s < 2 * K; ++s) z[s] = e[s] + l[s];
        for (int m = 0; m < count; ++m) {
            float v = p.x[at + m] * p.gain;
            for (int s = 0; s < K; ++s) {
                const float4 c = p.sec[s].c;  // b1, b2, -a1, -a2
                const float y = fmaf(p.sec[s].b0, v, z[2 * s]);
                z[2 * s] = fmaf(c.x, v, fmaf(c.z, y, z[2 * s + 1]));
                z[2 * s + 1] = fmaf(c.y, v, c.w * y);
                v = y;
            }
            p.y[at + m] = v;
        }
    }
    __syncwarp();
}

// In place: a strip's warm-up samples have been read.  (Out of line, as rows_again: code that hardly ever runs costs the
// epilogue's loop a few per cent by its layout alone.)
static __device__ __noinline__ void set_flag(unsigned *flag, bool now) {
    if (!now) return;
    __threadfence();
    atomicExch(flag, 1u);
}

// The terminal states of a warp's rows (R the first of them), in the accumulator d, again: where they are not finite
// (`bad`), which samples next to the largest float32 bring about as well as ones that are not finite, from the samples by
// FMAs -- with outputs from the signal, up to the strip's end, since the stage is gone; otherwise from the row X of it.
template <int K, int MODE>
__device__ __noinline__ void rows_again(const LaneParams<K> &p, unsigned d, bool bad, long long R, long long r_end,
                                        const unsigned char *X) {
    const long long at = (R + (threadIdx.x & 31)) * kStripN, end = r_end * kStripN < p.n ? r_end * kStripN : p.n;
    constexpr int S = 2 * K;
    constexpr bool MM = MODE == kStripOutputs;
    float t[16], a[16];
    tc_ldn<16>(d + (MM ? 64 : 0), t);
    tc_wait_ld();
    if constexpr (!MM) {  // as the epilogue adds them
        float b[16];
        tc_ldn<16>(d + 32, a);
        tc_wait_ld();
        for (int j = 0; j < 16; ++j) t[j] += a[j];
        tc_ldn<16>(d + 16, a);
        tc_ldn<16>(d + 48, b);
        tc_wait_ld();
        for (int j = 0; j < 16; ++j) t[j] += a[j] + b[j];
    }
    if (bad) {
        const int r = static_cast<int>(reinterpret_cast<uintptr_t>(X) >> 7) & 7;
        for (int s = 0; s < S; ++s) {
            float v = 0.f;
            for (int j = 0; j < kStripN; ++j) {
                float x = 0.f;
                if constexpr (MM) {
                    if (at + j < end) x = p.x[at + j];
                } else {
                    const int c = j & 31;
                    x = *reinterpret_cast<const float *>(X + (j >> 5) * kStripHalf + ((((c >> 2) ^ r) << 4) | ((c & 3) << 2)));
                }
                v = fmaf(__ldg(p.gtail + s * kStripN + j), x, v);
            }
            t[s] = v;
        }
    }
    __syncwarp();
    tc_st16(d + (MM ? 64 : 0), t);
    if constexpr (!MM) {
        for (int j = 0; j < 16; ++j) a[j] = 0.f;
        tc_st16(d + 16, a);
        tc_st16(d + 32, a);
        tc_st16(d + 48, a);
    }
    tc_wait_st();
}

// Row `row` of y = A x, A dense column-major S x S and x in shared memory (read as pairs, broadcast): no
// shuffles, so that products of several vectors overlap.
template <int S>
__device__ __forceinline__ float mv_shared(const float *A, const float *x, int row) {
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int j = 0; j < S; j += 2) {
        const float2 v = *reinterpret_cast<const float2 *>(x + j);
        y0 = fmaf(A[j * S + row], v.x, y0);
        y1 = fmaf(A[(j + 1) * S + row], v.y, y1);
    }
    return y0 + y1;
}

// The epilogue's warps fill the issue slots (half of all cycles issue, a fifth of the stalls wait for
// instructions), so that fewer instructions count for more than shorter chains: order 16, 2^28 samples,
// 459 -> 421 us by two-word products here, in the scan's coupling and in the operands' remainders (order 12:
// 375 -> 356, order 8: 375 -> 349; order 16, 2^26 samples: 137 -> 122); a scan that takes the sections in
// pairs, with half the exchanges in a chain but more products, was slower (473).

// a - b, two words at a time (exact where the difference of each word is) or word by word.
template <bool TWO>
__device__ __forceinline__ float4 sub4(const float4 &a, const float4 &b) {
    if constexpr (!TWO) return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
    const unsigned long long m = pack2(-1.f, -1.f);
    float4 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(fma2(pack2(b.x, b.y), m, pack2(a.x, a.y))));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.z), "=f"(r.w) : "l"(fma2(pack2(b.z, b.w), m, pack2(a.z, a.w))));
    return r;
}

// y += A x, A packed lower block-triangular with its 2 x 2 blocks by columns, x with every word twice, both in
// shared memory: two-word products, half the instructions.
template <int K>
__device__ __forceinline__ void state_mv2(const float *A, const float *x, float (&y)[2 * K]) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
        unsigned long long v = pack2(y[2 * s], y[2 * s + 1]);
#pragma unroll
        for (int j = 0; j <= s; ++j) {
            const ulonglong2 B = *reinterpret_cast<const ulonglong2 *>(A + 4 * (s * (s + 1) / 2 + j));
            const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(x + 4 * j);
            v = fma2(B.x, z.x, fma2(B.y, z.y, v));
        }
        asm("mov.b64 {%0, %1}, %2;" : "=f"(y[2 * s]), "=f"(y[2 * s + 1]) : "l"(v));
    }
}

// lane_scan with the sections' coupling in two-word products; p.MX holds the 2 x 2 blocks by columns.
template <int K, class Secs>
__device__ __forceinline__ void scan2(const LaneParams<K> &p, const Secs &cs, const float (&t)[2 * K], float (&S)[2 * K],
                                      float *a_out, int lane) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        unsigned long long v = pack2(t[2 * k], t[2 * k + 1]);
#pragma unroll
        for (int j = 0; j < k; ++j) {
            const float4 b = p.MX[k * (k - 1) / 2 + j];
            v = fma2(pack2(b.x, b.y), pack2(S[2 * j], S[2 * j]), fma2(pack2(b.z, b.w), pack2(S[2 * j + 1], S[2 * j + 1]), v));
        }
        float u1, u2;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(u1), "=f"(u2) : "l"(v));
#pragma unroll
        for (int r = 0; r < 5; ++r) {
            const float o1 = __shfl_up_sync(0xffffffffu, u1, 1 << r);
            const float o2 = __shfl_up_sync(0xffffffffu, u2, 1 << r);
            const float4 tn = cs.tn(k, r);
            if (lane >= (1 << r)) {
                u1 = fmaf(tn.x, o1, fmaf(tn.y, o2, u1));
                u2 = fmaf(tn.z, o1, fmaf(tn.w, o2, u2));
            }
        }
        const float s1 = __shfl_up_sync(0xffffffffu, u1, 1), s2 = __shfl_up_sync(0xffffffffu, u2, 1);
        S[2 * k] = lane == 0 ? 0.f : s1;
        S[2 * k + 1] = lane == 0 ? 0.f : s2;
        if (lane == 31) *reinterpret_cast<float2 *>(a_out + 2 * k) = make_float2(u1, u2);
    }
}

// Row `lane` (< S) of A x + B y: the two products by a half of the warp each.
template <int S>
__device__ __forceinline__ float mv_two(const float *A, const float *x, const float *B, const float *y, int lane) {
    const bool h = lane >= 16;
    const float v = mv_shared<S>(h ? B : A, h ? y : x, (lane & 15) < S ? lane & 15 : 0);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

// Words of the run's workspace (LaneParams::tail), all zero between runs.
struct StripTail {
    unsigned ticket, poison, done, pad;
    float zf[2 * kMaxPass];
    unsigned flag[kStripMax];  // in place: strip's warm-up samples have been read
};
static_assert(sizeof(StripTail) <= kStripTailBytes, "workspace of a run");

// Barriers of a block: staged units, operand buffers, accumulator slots, units' incoming states.
template <int XS>
struct StripBars {
    unsigned long long full[XS], xfree[XS], afull[2], afree[2], dfull[kStripDS], dfree[kStripDS], zready[kStripZ], yfull[4], fin;
    unsigned tmem, strip, last, stop;
};

template <int K, bool NORM, int MODE>
__global__ void __launch_bounds__(StripDims<K, MODE>::THREADS, 1)
    sos_strip_kernel(const __grid_constant__ StripParams<K, MODE> P) {
    using Sd = StripDims<K, MODE>;
    using Dm = typename Sd::Dm;
    constexpr int S = Sd::S, MS = Dm::MS, XS = Sd::XS, WGS = Sd::WGS;
    const LaneParams<K> &p = P.p;
    extern __shared__ __align__(1024) unsigned char sm[];
    float *tabs = reinterpret_cast<float *>(sm + Sd::OFF_TAB);
    float *sML = tabs + Sd::T_ML;
    float *sACp = tabs + Sd::T_ACP;
    float *z_buf = tabs + Sd::T_Z;  // [kStripZ][S] units' incoming states
    StripTail *tail = reinterpret_cast<StripTail *>(p.tail);
    StripBars<XS> &bars = *reinterpret_cast<StripBars<XS> *>(sm + Sd::OFF_BAR);
    static_assert(sizeof(StripBars<XS>) <= kStripBars, "barriers");
    unsigned long long *full = bars.full, *xfree = bars.xfree, *afull = bars.afull, *afree = bars.afree,
                       *dfull = bars.dfull, *dfree = bars.dfree, *zready = bars.zready;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long budget = p.spin_budget;
    const unsigned long long t_entry = p.trace ? global_ns() : 0;
    if (tid == 0) {
        // in place, a strip's last rows are stored once the next strip has read them: strips are taken from
        // the last one down, so that the block waited on is running or done
        bars.strip = P.in_place && p.cut.n_strips > 1 ? p.cut.n_strips - 1 - atomicAdd(&tail->ticket, 1u) : blockIdx.x;
        for (int i = 0; i < XS; ++i) {
            mbar_init(&full[i], 32 * Sd::LOADERS);
            mbar_init(&xfree[i], 4);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&afull[i], 4);
            mbar_init(&afree[i], 1);
        }
        for (int i = 0; i < kStripDS; ++i) {
            mbar_init(&dfull[i], 1);
            mbar_init(&dfree[i], 4);
        }
        for (int i = 0; i < kStripZ; ++i) mbar_init(&zready[i], 1);
        for (int i = 0; i < 4; ++i) mbar_init(&bars.yfull[i], 1);
        mbar_init(&bars.fin, 1);
    }
    if (Sd::TC && warp == 1) tc_alloc512(&bars.tmem);
    if (Sd::TC) tc_fence_before();
    __syncthreads();
    if (Sd::TC) tc_fence_after();
    const unsigned tmem = Sd::TC ? bars.tmem : 0;
    const int strip = static_cast<int>(bars.strip);
    const long long r_own = static_cast<long long>(strip) * p.cut.strip_rows;
    const long long r_end = r_own + p.cut.strip_rows < p.cut.n_rows ? r_own + p.cut.strip_rows : p.cut.n_rows;
    const int n_warm = r_own < p.cut.warm_rows ? static_cast<int>(r_own) : p.cut.warm_rows;
    // units of 128 rows from r_first on; rows r_first .. r_own - 1 only warm up, rows past r_end are zeros
    const long long r_first = r_own - n_warm;
    const unsigned n_u = static_cast<unsigned>((r_end - r_first + kStripRows - 1) / kStripRows);
    // phase trace (diagnostics; nothing is written without a trace buffer): one item per unit, strip by strip
    const long long item0 = strip * ((static_cast<long long>(p.cut.strip_rows) + p.cut.warm_rows + kStripRows - 1) / kStripRows);
    auto trace = [&](unsigned i, int slot) {
        if (p.trace && lane == 0 && item0 + i < p.trace_tiles)
            p.trace[static_cast<size_t>(item0 + i) * kTraceSlots + slot] = global_ns();
    };
    if (p.trace && tid == 0 && item0 < p.trace_tiles) {
        p.trace[static_cast<size_t>(item0) * kTraceSlots + 19] = t_entry;
        trace(0, 20);
    }
    // the tables, by every warp but the loading ones, which start at once
    auto load_tables = [&]() {
        const int w = !Sd::TC ? warp - 8 : warp == 1 ? 0 : warp - 3, k = 32 * w + lane;
        constexpr int step = Sd::THREADS - 32 * Sd::LOADERS;
        if constexpr (Sd::TC) {
            const float4 *src = reinterpret_cast<const float4 *>(p.gimg);
            float4 *dst = reinterpret_cast<float4 *>(sm + Sd::OFF_IMG);
            if constexpr (Sd::MM) {
                constexpr int HALF = 80 * 8, SKIP = 32 * 8;  // 16-byte words of a column half, and of its zeros
                for (int i = k; i < 4 * HALF; i += step) {   // heads, then remainders, two halves each
                    const int part = i / HALF, w = i % HALF, odd = part & 1;
                    if (!odd) dst[(part >> 1) * (Sd::B1 / 16) + w] = __ldg(src + i);
                    else if (w >= SKIP) dst[(part >> 1) * (Sd::B1 / 16) + HALF + w - SKIP] = __ldg(src + i);
                }
                for (int i = k; i < 64 * 8; i += step) dst[2 * Sd::B1 / 16 + i] = __ldg(src + 4 * HALF + i);
            } else {
                for (int i = k; i < Sd::IMG / 16; i += step) dst[i] = __ldg(src + i);
            }
        }
        for (int i = k; i < 11 * MS / 4; i += step) {
            const int m = i / (MS / 4), lane_of = m < 8 ? m : 8 * (m - 7);
            const float4 v = __ldg(reinterpret_cast<const float4 *>(p.tab) + lane_of * (MS / 4) + i % (MS / 4));
            reinterpret_cast<float4 *>(sML)[i] = Sd::TWO ? make_float4(v.x, v.z, v.y, v.w) : v;  // blocks by columns
        }
        for (int i = k; i < 4 * S * S; i += step) sACp[i] = __ldg(p.tab + Dm::OFF_ACP + i);
        if (p.zi && r_first == 0)
            for (int i = k; i < kStripN * S; i += step) tabs[Sd::T_H + i] = __ldg(p.tab + Dm::OFF_H + i);
        if (Sd::TC) fence_proxy_async_smem();  // the image is read by the tensor cores
        named_bar_sync(8, step);
        if (warp == 8) trace(0, 21);
    };

    if (warp < 8) {
    if constexpr (Sd::TC) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Sd::SREGS));
    if (!Sd::TC || (warp < 4 && warp != 1)) {
        // ------------------------------------------------------------------ loads
        const int w = !Sd::TC || warp == 0 ? warp : warp - 1;
        if (w == 0) {
            if (lane < S) z_buf[lane] = (r_first == 0 && p.zi) ? p.zi[lane] * p.sec[lane >> 1].zscale : 0.f;
            __syncwarp();
            if (lane == 0) mbar_arrive(&zready[0]);
        }
        unsigned i = 0;
        for (; i < n_u; ++i) {
            const unsigned xs = i % XS;
            if (i >= XS && !strip_wait(&xfree[xs], (i / XS - 1) & 1, budget, p.status)) break;
            const long long base = (r_first + static_cast<long long>(i) * kStripRows) * kStripN;
            const long long avail = (r_end * kStripN < p.n ? r_end * kStripN : p.n) - base;
            const float *x = p.x + base;
            const unsigned dst = smem_u32(sm) + xs * kStripXBytes;
            if (P.tma && avail >= kStripUnit) {
                if (w == 0 && lane == 0) {
                    fence_proxy_async_smem();  // the stage's ordinary reads come before the copy
                    mbar_expect_tx(&full[xs], kStripXBytes);
                    const long long row = r_first + static_cast<long long>(i) * kStripRows;
                    tma_load_2d(sm + xs * kStripXBytes, &P.tmx, 0, row, &full[xs]);
                    tma_load_2d(sm + xs * kStripXBytes + kStripHalf, &P.tmx, 32, row, &full[xs]);
                } else {
                    mbar_arrive(&full[xs]);
                }
                if (w == 0) trace(i, 16);
                continue;
            }
            if (P.x_aligned) {
                // 16-byte copies: lane = (row parity, chunk of the row); row 8m + 2k + parity has the chunk at
                // (chunk ^ parity ^ 2k) & 7
                const unsigned c = lane & 15, r1 = lane >> 4;
                const unsigned d = dst + (c >> 3) * kStripHalf + r1 * 128 + (((c & 7) ^ r1) << 4);
                const int off = r1 * kStripN + 4 * c;
                if (avail >= kStripUnit) {
                    const float *src = x + off;
#pragma unroll 1
                    for (int m = w; m < kStripRows / 8; m += Sd::LOADERS) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            cp_async16_s((d ^ (k << 5)) + (8 * m + 2 * k) * 128, src + (8 * m + 2 * k) * kStripN, 16u);
                    }
                } else {
                    const int left = static_cast<int>(avail) - off;
#pragma unroll 4
                    for (int j = w; j < kStripRows / 2; j += Sd::LOADERS) {
                        const int rem = left - 2 * j * kStripN;
                        const unsigned bytes = rem >= 4 ? 16u : rem > 0 ? static_cast<unsigned>(4 * rem) : 0u;
                        cp_async16_s((d ^ ((j & 3) << 5)) + 2 * j * 128, bytes ? x + off + 2 * j * kStripN : p.x, bytes);
                    }
                }
            } else {
                // 4-byte copies: chunk lane / 4 of a row's half
                const int left = avail < kStripUnit ? static_cast<int>(avail) : kStripUnit;
                const unsigned d = dst + ((lane & 3) << 2);
#pragma unroll 4
                for (int j = w; j < kStripUnit / 32; j += Sd::LOADERS) {
                    const unsigned r = j >> 1;
                    const bool in = 32 * j + lane < left;
                    cp_async4_s(d + (j & 1) * kStripHalf + r * 128 + (((lane >> 2) ^ (r & 7)) << 4),
                                in ? x + 32 * j + lane : p.x, in ? 4u : 0u);
                }
            }
            cp_async_arrive(&full[xs]);
            if (w == 0) trace(i, 16);
        }
        cp_async_wait_all();
        if (Sd::TC && P.tma) {
            // where a wait gave up, the copies in flight land before the block exits, under a limit of their own: the
            // warps that issued none stopped anywhere, and arrive for what warp 0 had issued; its last XS units sit
            // in distinct stages with none issued after them, so theirs are the current phases
            if (w == 0 && lane == 0) bars.stop = i;
            named_bar_sync(13, 32 * Sd::LOADERS);
            const unsigned stop = bars.stop;
#pragma unroll 1
            for (; i < stop; ++i) mbar_arrive(&full[i % XS]);
            if (w == 0 && stop < n_u)
#pragma unroll 1
                for (i = stop > XS ? stop - XS : 0; i < stop; ++i) strip_wait(&full[i % XS], (i / XS) & 1, kStripDrain, p.status);
        }
    } else if (Sd::TC && warp == 1) {
        // ------------------------------------------------------------------ products
        load_tables();
        {
            const unsigned g = smem_u32(sm + Sd::OFF_IMG), go = tc_elect();
            for (unsigned i = 0; i < n_u; ++i) {
                const unsigned ds = i % kStripDS;
                if (i >= kStripDS && !strip_wait(&dfree[ds], (i / kStripDS - 1) & 1, budget, p.status)) break;
                const unsigned d = tmem + ds * Sd::COLS;
                bool ok = true;
#pragma unroll
                for (int h = 0; h < 2; ++h) {  // half of the rows' samples at a time
                    ok = ok && strip_wait(&afull[h], i & 1, budget, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    if (h == 0) trace(i, 17);
                    const unsigned hi = tmem + Sd::ACOL + 64 * h, lo = hi + 32;
                    if constexpr (Sd::MM) {
                        // [Y_p | T] = X [T^T | G^T]: columns 0..63 the rows' zero-state outputs, 64..79 their
                        // terminal states.  T is lower triangular, so the samples from 16 j on enter columns
                        // 16 j .. only.  The small terms first
                        auto chain = [&](unsigned a, int image, bool first) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int off = 32 * h + 16 * (k >> 1);
                                tc_mma_ts(d + off, a + 8 * k, tc_sdesc(g + image + (h ? 80 + off - 32 : off) * 128 + k * 32),
                                          tc_idesc(80 - off), first && h == 0 && k == 0 ? 0u : 1u, go);
                            }
                        };
                        chain(lo, 0, true);        // remainders of x, heads of the image
                        chain(hi, Sd::B1, false);  // heads of x, remainders of the image
                        chain(hi, 0, false);       // heads of both
                    } else {
                        // x [G_hi | G_lo]: columns 32 h .. 32 h + 31; the remainders' products join the small
                        // terms, columns 16..31
                        constexpr unsigned i32 = tc_idesc(32), i16 = tc_idesc(16);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const unsigned gk = g + h * (Sd::IMG / 2) + k * 32;
                            tc_mma_ts(d + 32 * h, hi + 8 * k, tc_sdesc(gk), i32, k ? 1u : 0u, go);
                            tc_mma_ts(d + 16, lo + 8 * k, tc_sdesc(gk), i16, 1u, go);
                            tc_mma_ts(d + 16, lo + 8 * k, tc_sdesc(gk + 16 * 128), i16, 1u, go);
                        }
                    }
                    tc_commit_if(&afree[h], go);
                }
                if (!ok) break;
                tc_commit_if(&dfull[ds], go);
                trace(i, 18);
            }
            // every product issued has completed before tensor memory is released
            __syncwarp();
            tc_commit_if(&bars.fin, go);
            strip_wait(&bars.fin, 0, kStripDrain, p.status);
        }
    } else {
        // ------------------------------------------------------------------ operands of the products
        load_tables();
        const int r = 32 * (warp - 4) + lane;  // row within the unit
        const unsigned ta = tmem + Sd::ACOL + (static_cast<unsigned>(32 * (warp - 4)) << 16);
        // heads: the nearest TF32 values; remainders: exact in 12 bits, of which the tensor core reads 11
        for (unsigned i = 0; i < n_u; ++i) {
            const unsigned xs = i % XS;
            if (!strip_wait(&full[xs], (i / XS) & 1, budget, p.status)) break;
            if (warp == 4) trace(i, 1);
            const unsigned char *X = sm + xs * kStripXBytes + r * 128;
            bool ok = true;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                ok = ok && (i == 0 || strip_wait(&afree[h], (i - 1) & 1, budget, p.status));
                if (!ok) break;
                tc_fence_after();
                if (warp == 4 && h == 0) trace(i, 2);
                const unsigned char *Xh = X + h * kStripHalf;
                const unsigned t0 = ta + 64 * h;
#pragma unroll
                for (int j = 0; j < 4; ++j) {  // eight samples at a time
                    const float4 u = *reinterpret_cast<const float4 *>(Xh + (((2 * j) ^ (r & 7)) << 4));
                    const float4 v = *reinterpret_cast<const float4 *>(Xh + (((2 * j + 1) ^ (r & 7)) << 4));
                    const float4 uh = make_float4(tf32_near(u.x), tf32_near(u.y), tf32_near(u.z), tf32_near(u.w));
                    const float4 vh = make_float4(tf32_near(v.x), tf32_near(v.y), tf32_near(v.z), tf32_near(v.w));
                    tc_st8(t0 + 8 * j, uh, vh);
                    tc_st8(t0 + 32 + 8 * j, sub4<Sd::TWO>(u, uh), sub4<Sd::TWO>(v, vh));
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&afull[h]);
            }
            if (!ok) break;
            if (Sd::MM && lane == 0) mbar_arrive(&xfree[xs]);
            if (warp == 4) trace(i, 3);
        }
    }
    } else {
        // ------------------------------------------------------------------ scan, carry, recurrences
        if constexpr (Sd::TC) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Sd::REGS));
        load_tables();
        const int wg = (warp - 8) >> 2, q = warp & 3;
        const int r = 32 * q + lane;  // row within the unit
        const unsigned tl = tmem + (static_cast<unsigned>(32 * q) << 16);
        const ParamSecs<K> cs{p};
        constexpr int ZP = Sd::ZP, ZW = Sd::ZW;
        constexpr int QC = Sd::TWO ? 1 : 3;  // the warp that forms the next unit's state
        float *zv = tabs + Sd::T_ZV + (wg * 4 + q) * 4 * ZP;  // [4][ZP], every word ZW times
        const int li = lane < S ? lane : 0;
        bool dead = false;
        unsigned par = 0, y_par = 0;
        for (unsigned i = wg; i < n_u; i += WGS, par ^= 1) {
            const unsigned ds = i % kStripDS, xs = i % XS;
            float *ab = tabs + Sd::T_A + (wg * 2 + par) * 4 * S;
            float Sl[S];
            [[maybe_unused]] bool released = false;  // the accumulator slot
            bool bad = false;  // the row's samples are not all finite (its products are then worth nothing)
            bool ok = !dead && (Sd::TC ? strip_wait(&dfull[ds], (i / kStripDS) & 1, budget, p.status)
                                       : strip_wait(&full[xs], (i / XS) & 1, budget, p.status));
            const long long R = r_first + static_cast<long long>(i) * kStripRows + 32 * q;  // the warp's first row
            if (q == 0) trace(i, 4);
            if (ok) {
                float t[S];
                if constexpr (!Sd::TC) {
                    if (P.in_place && q == 0 && lane == 0 && n_warm > 0 && static_cast<int>(i) == (n_warm - 1) / kStripRows) {
                        __threadfence();
                        atomicExch(&tail->flag[strip], 1u);  // the warm-up samples have been read
                    }
                    const unsigned o = xs * kStripXBytes + r * 128 + ((r & 7) << 4);
                    float a[S][2];
#pragma unroll
                    for (int s = 0; s < S; ++s) a[s][0] = a[s][1] = 0.f;
#pragma unroll
                    for (int j = 0; j < kStripN / 4; ++j) {
                        const float4 x = *reinterpret_cast<const float4 *>(sm + (o ^ ((j & 7) << 4)) + (j >> 3) * kStripHalf);
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            const float *g = P.g[s] + 4 * j;
                            a[s][j & 1] = fmaf(g[0], x.x, fmaf(g[1], x.y, fmaf(g[2], x.z, fmaf(g[3], x.w, a[s][j & 1]))));
                        }
                    }
#pragma unroll
                    for (int s = 0; s < S; ++s) t[s] = a[s][0] + a[s][1];
                } else {
                    tc_fence_after();
                    constexpr int C = S <= 2 ? 2 : S <= 4 ? 4 : S <= 8 ? 8 : 16;
                    const unsigned d = tl + ds * Sd::COLS;
                    auto terminal = [&]() {
                        if constexpr (Sd::MM) {
                            float a[C];
                            tc_ldn<C>(d + 64, a);
                            tc_wait_ld();
#pragma unroll
                            for (int j = 0; j < S; ++j) t[j] = a[j];
                        } else {
                            float a0[C], a1[C];
                            tc_ldn<C>(d + 16, a0);  // the small terms
                            tc_ldn<C>(d + 48, a1);
                            tc_wait_ld();
#pragma unroll
                            for (int j = 0; j < S; ++j) t[j] = a0[j] + a1[j];
                            tc_ldn<C>(d, a0);
                            tc_ldn<C>(d + 32, a1);
                            tc_wait_ld();
#pragma unroll
                            for (int j = 0; j < S; ++j) t[j] = (a0[j] + a1[j]) + t[j];
                        }
                    };
                    terminal();
                    bad = !(fabsf(t[0]) <= 3.402823466e38f);
                    if (__any_sync(0xffffffffu, bad)) {
                        rows_again<K, MODE>(p, d, bad, R, r_end, sm + xs * kStripXBytes + r * 128);
                        terminal();
                    }
                    if constexpr (!Sd::MM) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&dfree[ds]);
                    }
                }
                if (q == 0) trace(i, 5);
                if constexpr (Sd::MM) scan2<K>(p, cs, t, Sl, ab + q * S, lane);
                else lane_scan<K>(cs, t, Sl, ab + q * S, lane);
                if (q == 0) trace(i, 7);
            }
            if (!named_bar_and(1 + wg, 128, ok)) break;
            // the fold's prefix p_v (carry of the groups before this warp's under zero state), then, once
            // the unit's incoming state is known, the group's: Z_v = (A_C)^v Z + p_v
            // p_v = a_{v-1} + A_C a_{v-2} + (A_C)^2 a_{v-3} and the unit's carry c: independent products
            const float *A1 = sACp, *A2 = sACp + S * S, *A3 = sACp + 2 * S * S, *A4 = sACp + 3 * S * S;
            float pv = 0.f, cu = 0.f;
            if (q == 1) pv = ab[li];
            if (q == 2) pv = mv_shared<S>(A1, ab, li) + ab[S + li];
            constexpr bool HALVES = S > 8;  // long rows: two products at a time
            if (q == 3)
                pv = (HALVES ? mv_two<S>(A2, ab, A1, ab + S, lane) : mv_shared<S>(A2, ab, li) + mv_shared<S>(A1, ab + S, li)) + ab[2 * S + li];
            if (q == QC) {
                cu = (HALVES ? mv_two<S>(A3, ab, A2, ab + S, lane) : mv_shared<S>(A3, ab, li) + mv_shared<S>(A2, ab + S, li)) + ab[3 * S + li];
                if (!HALVES) cu += mv_shared<S>(A1, ab + 2 * S, li);
            }
            dead = !strip_wait(&zready[i % kStripZ], (i / kStripZ) & 1, budget, p.status);
            if (!Sd::MM && dead) continue;
            if (q == 0) trace(i, 9);
            const float *z0 = z_buf + (i % kStripZ) * S;
            // the unit's rows have all been read, and the ones before, by rows_again too
            if constexpr (Sd::TC)
                if (P.in_place) set_flag(&tail->flag[strip], q == 0 && lane == 0 && n_warm > 0 && static_cast<int>(i) == (n_warm - 1) / kStripRows);
            if (q == QC) {
                const float zn = (HALVES ? mv_two<S>(A4, z0, A1, ab + 2 * S, lane) : mv_shared<S>(A4, z0, li)) + cu;
                if (i + 1 < n_u) {
                    if (lane < S) z_buf[((i + 1) % kStripZ) * S + lane] = zn;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&zready[(i + 1) % kStripZ]);
                } else if (__any_sync(0xffffffffu, !(fabsf(zn) <= 3.402823466e38f)) && lane == 0 && strip + 1 < p.cut.n_strips) {
                    atomicMax(&tail->poison, static_cast<unsigned>(p.cut.n_strips - strip));
                }
            }
            // the unit's first and last own rows; with outputs its four warps stay together for the products
            const bool own = R + 32 > r_own && R < r_end;
            const bool unit_own = R - 32 * q + kStripRows > r_own;
            if (Sd::MM ? unit_own : own) {
                const float zq = q == 0 ? z0[li] : mv_shared<S>(q == 1 ? A1 : q == 2 ? A2 : A3, z0, li) + pv;
                // (M_N)^lane Z_v in two steps, lane = 8 a + b: the four (M_N)^(8 a) Z_v, a section's two words a
                // lane, then each lane's (M_N)^b of one of them (11 matrices to read instead of 32)
                if (lane < S) {
                    if constexpr (Sd::TWO) *reinterpret_cast<float2 *>(zv + 2 * lane) = make_float2(zq, zq);
                    else zv[lane] = zq;
                }
                __syncwarp();
                {
                    const int a = lane >> 3, s = lane & 7;
                    float w0 = 0.f, w1 = 0.f;
                    if (a > 0 && s < K) {
                        const float *m = sML + (7 + a) * MS + 2 * s * (s + 1);
#pragma unroll
                        for (int j = 0; j < K; ++j)
                            if (j <= s) {
                                const float4 B = *reinterpret_cast<const float4 *>(m + 4 * j);
                                const float z0 = zv[2 * ZW * j], z1 = zv[2 * ZW * j + ZW];
                                w0 = fmaf(B.x, z0, fmaf(Sd::TWO ? B.z : B.y, z1, w0));
                                w1 = fmaf(Sd::TWO ? B.y : B.z, z0, fmaf(B.w, z1, w1));
                            }
                        if constexpr (Sd::TWO) *reinterpret_cast<float4 *>(zv + a * ZP + 4 * s) = make_float4(w0, w0, w1, w1);
                        else *reinterpret_cast<float2 *>(zv + a * ZP + 2 * s) = make_float2(w0, w1);
                    }
                }
                __syncwarp();
                float st[S];
#pragma unroll
                for (int j = 0; j < S; ++j) st[j] = Sl[j];
                if constexpr (Sd::TWO) state_mv2<K>(sML + (lane & 7) * MS, zv + (lane >> 3) * ZP, st);
                else lane_state_mv<K>(sML + (lane & 7) * MS, zv + (lane >> 3) * ZP, st);
                unsigned char *X = sm + xs * kStripXBytes;
                const long long base = R * kStripN;
                if (q == 0) trace(i, 10);
                if (p.zf && r_end == p.cut.n_rows && R + 32 >= r_end) {
                    // final state: the last row's samples under zero state, taken across the lanes, plus
                    // the transition of the row's incoming state over them
                    const int lane_last = static_cast<int>(p.cut.n_rows - 1 - R);
                    const int ml = p.m_last;
                    [[maybe_unused]] const int rl = 32 * q + lane_last;
                    float acc[S], zt[S];
                    {
                        const float *gt = p.gtail + (kStripN - 1 - ml);
                        float xa = 0.f, xb = 0.f;
                        if constexpr (Sd::MM) {  // the stage is gone; the signal is still as it was here, in place too
                            const float *xr = p.x + base + lane_last * kStripN;
                            if (lane <= ml) xa = xr[lane];
                            if (lane + 32 <= ml) xb = xr[lane + 32];
                        } else {
                            if (lane <= ml) xa = *reinterpret_cast<const float *>(X + tc_swz(rl, lane));
                            if (lane + 32 <= ml) xb = *reinterpret_cast<const float *>(X + kStripHalf + tc_swz(rl, lane));
                        }
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            float v = lane <= ml ? __ldg(gt + s * kStripN + lane) * xa : 0.f;
                            if (lane + 32 <= ml) v = fmaf(__ldg(gt + s * kStripN + lane + 32), xb, v);
                            acc[s] = v;
                        }
#pragma unroll
                        for (int s = 0; s < S; ++s)
#pragma unroll
                            for (int o = 16; o; o >>= 1) acc[s] += __shfl_xor_sync(0xffffffffu, acc[s], o);
                    }
                    packed_mv_param<K>(p.A_tail, st, zt);
                    if (lane == lane_last) {
                        // with several strips the block that finishes last hands the state over, since zf
                        // may be the array another strip reads its initial state from
                        float *zf = p.cut.n_strips > 1 ? tail->zf : p.zf;
#pragma unroll
                        for (int s = 0; s < S; ++s) zf[s] = (acc[s] + zt[s]) * p.sec[s >> 1].zscale_inv;
                    }
                    __syncwarp();
                }
                if constexpr (Sd::MM) {
                    if (p.zi && r_first == 0 && i == 0 && q == 0 && !__any_sync(0xffffffffu, bad)) {
                        // the signal's first group: its states' part is added in float32 (row_part; as operands of
                        // 22 bits they would err by as much), and none are left to multiply.  (Rows that
                        // are done plainly below take theirs from the operand.)
                        const float *H = tabs + Sd::T_H;
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            float v[16];
                            tc_ldn<16>(tl + ds * Sd::COLS + 16 * c, v);
                            tc_wait_ld();
#pragma unroll
                            for (int j = 0; j < S; ++j)
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    const float4 b = *(reinterpret_cast<const float4 *>(H + j * kStripN + 16 * c) + k);
                                    v[4 * k] = fmaf(b.x, st[j], v[4 * k]);
                                    v[4 * k + 1] = fmaf(b.y, st[j], v[4 * k + 1]);
                                    v[4 * k + 2] = fmaf(b.z, st[j], v[4 * k + 2]);
                                    v[4 * k + 3] = fmaf(b.w, st[j], v[4 * k + 3]);
                                }
                            tc_st16(tl + ds * Sd::COLS + 16 * c, v);
                        }
#pragma unroll
                        for (int j = 0; j < S; ++j) st[j] = 0.f;
                    }
                    // the rows' states as an operand beside the accumulator, then Y += St H^T, small terms first,
                    // issued by the warpgroup's first warp
                    float e[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) e[j] = j < S ? tf32_near(st[j < S ? j : 0]) : 0.f;
                    tc_st16(tl + ds * Sd::COLS + 64, e);
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const float4 l = sub4<true>(make_float4(j < S ? st[j < S ? j : 0] : 0.f, j + 1 < S ? st[j + 1 < S ? j + 1 : 0] : 0.f,
                                                          j + 2 < S ? st[j + 2 < S ? j + 2 : 0] : 0.f, j + 3 < S ? st[j + 3 < S ? j + 3 : 0] : 0.f),
                                              make_float4(e[j], e[j + 1], e[j + 2], e[j + 3]));
                        e[j] = l.x; e[j + 1] = l.y; e[j + 2] = l.z; e[j + 3] = l.w;
                    }
                    tc_st16(tl + ds * Sd::COLS + 80, e);
                    tc_wait_st();
                    tc_fence_before();
                    if (!named_bar_and(9 + wg, 128, !dead)) break;
                    if (q == 0) {
                        tc_fence_after();
                        constexpr unsigned i64 = tc_idesc(64);
                        const unsigned d = tmem + ds * Sd::COLS, h = smem_u32(sm + Sd::OFF_IMG) + 2 * Sd::B1, go = tc_elect();
                        constexpr int KK = S > 8 ? 2 : 1;
#pragma unroll
                        for (int k = 0; k < KK; ++k) tc_mma_ts(d, d + 80 + 8 * k, tc_sdesc(h + 32 * k), i64, 1u, go);
#pragma unroll
                        for (int k = 0; k < KK; ++k) tc_mma_ts(d, d + 64 + 8 * k, tc_sdesc(h + 64 + 32 * k), i64, 1u, go);
#pragma unroll
                        for (int k = 0; k < KK; ++k) tc_mma_ts(d, d + 64 + 8 * k, tc_sdesc(h + 32 * k), i64, 1u, go);
                        tc_commit_if(&bars.yfull[wg], go);
                    }
                    if (!strip_wait(&bars.yfull[wg], y_par, budget, p.status)) dead = true;
                    y_par ^= 1;
                    tc_fence_after();
                } else {
                    const unsigned row = xs * kStripXBytes + r * 128 + ((r & 7) << 4);
                    const bool first = p.zi && r_first == 0 && i == 0 && q == 0;
                    if (first) {
#pragma unroll
                        for (int j = 0; j < S; ++j) {
                            tabs[Sd::T_ST + lane * S + j] = st[j];
                            st[j] = 0.f;
                        }
                    }
                    lane_recurrence<K, NORM, Sd::U>(cs, P.pk, sm, row, p.gain, st);
                    if (first) row_part<K>(sm, row, tabs + Sd::T_H, tabs + Sd::T_ST + lane * S);
                    __syncwarp();
                }
                if (q == 0) trace(i, 11);
                if (P.in_place && own && strip + 1 < p.cut.n_strips && R + 32 > r_end - p.cut.warm_rows) {
                    const long long t0 = clock64();
                    bool seen = false, late = false;
                    while (!seen && !late) {
                        seen = ld_acquire_u32(&tail->flag[strip + 1]) != 0;
                        late = clock64() - t0 > budget;
                    }
                    if (!__all_sync(0xffffffffu, seen)) {
                        if (lane == 0) atomicOr(p.status, kDevErrTimeout);
                        dead = true;
                    }
                }
                if (!Sd::MM && dead) continue;
                // the group's own samples: from .. to - 1, counted from its first row (none of a group outside)
                const int from = R < r_own ? static_cast<int>(r_own - R) * kStripN : 0;
                const long long own_end = r_end * kStripN < p.n ? r_end * kStripN : p.n;
                const int to = !own ? 0 : own_end - base < 32 * kStripN ? static_cast<int>(own_end - base) : 32 * kStripN;
                float *y = p.y + base;
                if constexpr (Sd::MM) {
                    const unsigned bad_rows = __ballot_sync(0xffffffffu, bad);
                    const unsigned sg = Sd::OFF_STAGE + (warp - 8) * 4096;  // 32 rows x 128 B, chunks permuted
                    if (bad_rows && !dead) {
                        // rows with samples that are not finite: the outputs up to the first of them are right
                        // by the recurrence, which is run from the rows' states on the signal itself
                        rows_plainly<K>(p, tl + ds * Sd::COLS + 64, bad, base, from, to);
                        __syncwarp();
                    }
                    if (!dead) {
                        float v[64];
#pragma unroll
                        for (int k = 0; k < 4; ++k) tc_ldn<16>(tl + ds * Sd::COLS + 16 * k, *reinterpret_cast<float(*)[16]>(v + 16 * k));
                        tc_wait_ld();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&dfree[ds]);
                        released = true;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {  // half a row at a time through the staging
                            if (P.tma) {  // the last store has read it
                                if (lane == 0) bulk_wait_read0();
                                __syncwarp();
                            }
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                *reinterpret_cast<float4 *>(sm + sg + lane * 128 + ((c ^ (lane & 7)) << 4)) =
                                    make_float4(v[32 * h + 4 * c], v[32 * h + 4 * c + 1], v[32 * h + 4 * c + 2], v[32 * h + 4 * c + 3]);
                            if (P.tma && from == 0 && to == 32 * kStripN && !bad_rows) {
                                fence_proxy_async_smem();
                                __syncwarp();
                                if (lane == 0) {
                                    tma_store_2d(&P.tmy, 32 * h, R, sm + sg);
                                    bulk_commit();
                                }
                                continue;
                            }
                            __syncwarp();
                            if (P.y_aligned) {
                                const int c = lane & 7, r1 = lane >> 3;
                                const int k0 = r1 * kStripN + 32 * h + 4 * c;
                                auto get = [&](int j) {
                                    const int rr = 4 * j + r1;
                                    return *reinterpret_cast<const float4 *>(sm + sg + rr * 128 + ((c ^ (rr & 7)) << 4));
                                };
                                if (from == 0 && to == 32 * kStripN && !bad_rows) {
#pragma unroll
                                    for (int j = 0; j < 8; ++j) __stcs(reinterpret_cast<float4 *>(y + k0 + 4 * j * kStripN), get(j));
                                } else {
#pragma unroll 2
                                    for (int j = 0; j < 8; ++j) {
                                        const int k = k0 + 4 * j * kStripN;
                                        if (!(bad_rows >> (4 * j + r1) & 1)) put4(y, k, from, to, get(j));
                                    }
                                }
                            } else {
#pragma unroll 4
                                for (int j = 0; j < 32; ++j) {
                                    const int k = j * kStripN + 32 * h + lane;
                                    const float v = *reinterpret_cast<const float *>(sm + sg + tc_swz(j, lane));
                                    if (k >= from && k < to && !(bad_rows >> j & 1)) __stcs(y + k, v);
                                }
                            }
                            __syncwarp();
                        }
                    }
                } else if (P.y_aligned) {
                    const int c = lane & 15, r1 = lane >> 4;
                    const unsigned src = xs * kStripXBytes + (32 * q + r1) * 128 + (c >> 3) * kStripHalf + (((c & 7) ^ r1) << 4);
                    const int k0 = r1 * kStripN + 4 * c;  // from is a multiple of 64
                    auto get = [&](int j) {
                        return *reinterpret_cast<const float4 *>(sm + (src ^ ((j & 3) << 5)) + 256 * j);
                    };
                    if (from == 0 && to == 32 * kStripN) {
#pragma unroll 8
                        for (int j = 0; j < 16; ++j) __stcs(reinterpret_cast<float4 *>(y + k0 + 2 * j * kStripN), get(j));
                    } else {
#pragma unroll 4
                        for (int j = 0; j < 16; ++j) put4(y, k0 + 2 * j * kStripN, from, to, get(j));
                    }
                } else {
                    const unsigned char *Xw = X + 32 * q * 128;
#pragma unroll 8
                    for (int j = 0; j < kStripN; ++j) {
                        const int rr = j >> 1, k = 32 * j + lane;
                        const float v = *reinterpret_cast<const float *>(Xw + (j & 1) * kStripHalf + tc_swz(rr, lane));
                        if (k >= from && k < to) __stcs(y + k, v);
                    }
                }
                __syncwarp();
            }
            if (Sd::MM && !released) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&dfree[ds]);
            }
            if (!Sd::MM) {
                // the recurrences' ordinary stores to the stage, and the loads of the outputs, come before the TMA
                // copy that overwrites it
                if (Sd::TC && P.tma) fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&xfree[xs]);
            }
            if (q == 0) {
                trace(i, 12);
                if (p.trace && lane == 0 && item0 + i < p.trace_tiles) {
                    unsigned smid;
                    asm volatile("mov.u32 %0, %smid;" : "=r"(smid));
                    p.trace[static_cast<size_t>(item0 + i) * kTraceSlots] = static_cast<unsigned long long>(item0 + i) + 1;
                    p.trace[static_cast<size_t>(item0 + i) * kTraceSlots + 13] = smid;
                }
            }
        }
        // a wait for the last products gave up: they end before tensor memory is released
        if (Sd::MM && dead) strip_wait(&bars.yfull[wg], y_par ^ 1, kStripDrain, p.status);
    }
    if (Sd::MM && P.tma && warp >= 8 && lane == 0) bulk_wait0();  // the outputs are written
    if (Sd::TC) tc_fence_before();
    __syncthreads();
    if (Sd::TC && warp == 1) {
        tc_fence_after();
        tc_dealloc512(tmem);
    }
    if (tid == 0) trace(0, 22);
    // the block that finishes last: the final state, and what follows a strip that ended in a state that
    // is not finite (the following strips, which did not see it, become NaN as the recurrence would
    // leave them); the workspace is left as it was found
    if (blockIdx.x == 0 && tid == 0 && P.host_tickets) atomicAdd(p.ticket, P.host_tickets);
    if (p.cut.n_strips == 1) return;
    if (tid == 0) {
        __threadfence();
        bars.last = atomicAdd(&tail->done, 1u) + 1 == gridDim.x;
    }
    __syncthreads();
    if (!bars.last) return;
    __threadfence();
    const unsigned poison = *reinterpret_cast<volatile unsigned *>(&tail->poison);
    const float nan = __uint_as_float(0x7fffffffu);
    if (poison) {
        const long long from = static_cast<long long>(p.cut.n_strips - poison + 1) * p.cut.strip_rows * kStripN;
        for (long long k = from + tid; k < p.n; k += Sd::THREADS) p.y[k] = nan;
    }
    if (p.zf && tid < S) p.zf[tid] = poison ? nan : *reinterpret_cast<volatile float *>(&tail->zf[tid]);
    for (int k = tid; k < p.cut.n_strips; k += Sd::THREADS) tail->flag[k] = 0;
    __syncthreads();
    if (tid == 0) tail->ticket = tail->poison = tail->done = 0;
}

// ---- launch (one set of instantiations per translation unit: sosfilt_strip_*.cu)
template <int K, bool NORM, int MODE>
KernelOnce g_strip_once;

template <int K, bool NORM, int MODE>
cudaError_t launch_strip_one(const StripParams<K, MODE> &P, cudaStream_t s) {
    using Sd = StripDims<K, MODE>;
    auto kern = sos_strip_kernel<K, NORM, MODE>;
    cudaError_t e = raise_smem_once(g_strip_once<K, NORM, MODE>, kern, Sd::SMEM);
    if (e != cudaSuccess) return e;
    kern<<<static_cast<unsigned>(P.p.cut.n_strips), Sd::THREADS, Sd::SMEM, s>>>(P);
    return cudaGetLastError();
}

template <int K, int MODE>
cudaError_t launch_strip_mode(const LaneParams<K> &p, long long grid, cudaStream_t s) {
    StripParams<K, MODE> P;
    std::memset(static_cast<void *>(&P), 0, sizeof(P));
    P.p = p;
    if constexpr (MODE == kStripOutputs)
        for (auto &b : P.p.MX) b = make_float4(b.x, b.z, b.y, b.w);  // by columns (scan2)
    P.in_place = p.x == p.y;
    P.x_aligned = reinterpret_cast<uintptr_t>(p.x) % 16 == 0;
    P.y_aligned = reinterpret_cast<uintptr_t>(p.y) % 16 == 0;
    P.host_tickets = static_cast<unsigned long long>(p.n_tiles + grid);
    if constexpr (MODE != kStripFma) {
        // the tensor maps cost a call about a microsecond on the host: for strips of several units
        if (P.x_aligned && P.y_aligned && p.cut.strip_rows >= kStripTmaRows)
            P.tma = strip_rows_map(&P.tmx, p.x, p.n / kStripN, kStripRows) &&
                    strip_rows_map(&P.tmy, p.y, p.n / kStripN, 32);
    }
    if constexpr (MODE == kStripFma) std::memcpy(P.g, p.gresp, sizeof P.g);
    if constexpr (MODE == kStripStates && StripPairs<K>::TWO) {
        constexpr int H = StripPairs<K>::H;
        auto put = [](unsigned long long &w, int half, float v) { std::memcpy(reinterpret_cast<char *>(&w) + 4 * half, &v, 4); };
        for (int k = 0; k < K; ++k) {
            const int s = k % H, half = k / H;
            put(P.pk.a1[s], half, p.sec[k].c.z);
            put(P.pk.a2[s], half, p.sec[k].c.w);
            if (k + 1 == K) continue;
            put(P.pk.b1[s], half, p.sec[k + 1].c.x);
            put(P.pk.b2[s], half, p.sec[k + 1].c.y);
            put(P.pk.b0[s], half, p.sec[k + 1].b0);
        }
    }
    return p.norm ? launch_strip_one<K, true, MODE>(P, s) : launch_strip_one<K, false, MODE>(P, s);
}

template <int K>
bool launch_strip_k(const LaneParams<K> &p, long long grid, cudaStream_t s, cudaError_t &err) {
    if (!p.cut.n_strips) return false;
    if constexpr (K <= kStripStatesK) {
        if (p.cut.fma) {
            err = launch_strip_mode<K, kStripFma>(p, grid, s);
            return true;
        }
    } else if (p.products) {
        err = launch_strip_mode<K, kStripOutputs>(p, grid, s);
        return true;
    }
    err = launch_strip_mode<K, kStripStates>(p, grid, s);
    return true;
}

#define SOSK_STRIP_INST(k)                                                                           \
    template <>                                                                                      \
    bool launch_strip<k>(const LaneParams<k> &p, long long grid, cudaStream_t s, cudaError_t &err) { \
        return launch_strip_k<k>(p, grid, s, err);                                                   \
    }

}  // namespace sosk

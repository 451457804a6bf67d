// Persistent single-signal kernel for cascades whose memory is finite in float32, sm_103a: the signal
// is cut into one strip of consecutive samples per thread block, and no block waits on another.
//
// The zero-input transition of a stable cascade over H samples, M1^H, decays to matrices whose float32
// entries are all zero; from there on a state H samples old adds nothing to the carried one (Eq. 25 with
// the terms the float32 tables hold as zeros left out).  The host finds that memory once per filter
// (warm_rows, in rows of 64 samples).  A block then starts its strip warm_rows rows early from zero state,
// which gives it the strip's true incoming state, and carries the state from unit to unit inside the
// block: no lookback across blocks, no descriptors, the same composition on every run.
//
// A unit is 128 rows of N = 64 samples, staged in shared memory with the 16-byte chunks of a row permuted
// by the row number (a lane reads its own row without bank conflicts).  Per unit:
//   1. terminal states of the rows under zero state (Sec. II-C).  With one or two sections, by FMAs: each
//      lane multiplies its row with the 2 or 4 state responses.  With more, the product of the rows with the 64
//      state responses, T = X G^T, by tcgen05.mma with the rows in tensor memory.  TF32 products of the
//      split operands: X as its upper 19 bits (what the tensor core reads) and the rounded remainder, G
//      as a TF32 value rounded to nearest and its remainder; the four partial products enter separate
//      accumulators for the large and the small terms, summed in float32 by the epilogue.
//   2. lane scan (Sec. II-C's recursive doubling) of each warp's 32 rows, fold of the four groups'
//      carries, and the unit's incoming state Z' = (A_C)^4 Z + c from the previous unit's.
//   3. every row's true incoming state S_l + (M_N)^l Z (Eq. 24 at the rows' starts), from which the
//      sections' recurrences run over the row in place, skewed by one sample per section: the outputs
//      themselves, 4 FMAs per section and sample and no separate correction pass (the lookback kernel's
//      particular pass and correction are 6).
//   4. coalesced stores.
// Groups of warm-up rows stop after step 2.
//
// Warp roles (one block per SM; the first eight warps give registers to the others):
//   warps 0, 2, 3  load the units' samples (cp.async, zero-filled past the end, any alignment)
//   warp 1         tensor-memory owner; lane 0 issues the products
//   warps 4-7      split the rows into the products' operands, in tensor memory (two buffers)
//   warps 8 on     three or four warpgroups, one unit each in turn; warp q of a warpgroup takes rows
//                  32q .. 32q+31
// Without the tensor cores warps 0-7 all load.
// Every wait is bounded by the spin budget.
#pragma once
#include <atomic>

#include "sosfilt_lane.cuh"
#include "sosfilt_tcgen05.cuh"

namespace sosk {

constexpr int kStripN = 64;                        // samples per row
constexpr int kStripRows = 128;                    // rows per unit (four groups of 32 lanes)
static_assert(kStripUnit == kStripN * kStripRows, "unit geometry");
constexpr int kStripXBytes = kStripUnit * 4;       // one staged unit: two column halves of 16 KB
constexpr int kStripHalf = kStripXBytes / 2;
constexpr int kStripCols = 64;                     // accumulator columns of a unit
constexpr int kStripDS = 4;                        // accumulator slots: columns 0 .. 255
constexpr int kStripACol = kStripDS * kStripCols;  // operand buffers: two of 64 + 64 columns behind them
constexpr int kStripImg = 8192;                    // G image: two K halves of 32 rows x 128 B
constexpr int kStripZ = 8;                         // units' incoming states kept (more than are in hand)
constexpr int kStripBars = 384;                    // bytes of barriers and shared words
constexpr long long kStripDrain = 2000000000LL;    // cycles a block waits for its own products at exit

template <int K, bool TC_>
struct StripDims {
    using Dm = LaneDims<K, kStripN, kLaneW>;
    static constexpr int S = 2 * K;
    // epilogue warpgroups, and the registers a thread of the first two warpgroups (SREGS) and of theirs
    // (REGS) has: four with 88 (768 threads of 80 at launch: 256 x 64 + 512 x 88), or three with 128 where
    // the scan and the recurrences of five and more sections need them (640 threads of 96 at launch:
    // 256 x 48 + 384 x 128)
    static constexpr int WGS = K <= 4 ? 4 : 3;
    static constexpr int SREGS = K <= 4 ? 64 : 48;
    static constexpr int REGS = K <= 4 ? 88 : 128;
    static constexpr int THREADS = 256 + 128 * WGS;
    // terminal states on the tensor cores (else by FMAs: 128 or 256 a row, which one or two sections have
    // the issue slots for, and which spare the signal's first unit the operands and products)
    static constexpr bool TC = TC_;
    static constexpr int LOADERS = TC ? 3 : 8;  // loading warps
    static constexpr int U = TC ? 1 : 8;        // chunks of the recurrences unrolled
    // shared memory after the staged units: G image, then floats: (M_N)^lane, (A_C)^v for v = 1 .. 4, the
    // warpgroups' local carries (two slots), group states, unit states; then the barriers
    static constexpr int T_ML = 0;
    static constexpr int T_ACP = T_ML + 32 * Dm::MS;
    static constexpr int T_A = T_ACP + 4 * S * S;
    static constexpr int T_ZV = T_A + WGS * 2 * 4 * S;
    static constexpr int T_Z = T_ZV + WGS * 4 * S;
    static constexpr int T_END = T_Z + kStripZ * S;
    static constexpr int FIXED = kStripImg + 4 * T_END + kStripBars;
    static constexpr int XS_FIT = (227 * 1024 - FIXED) / kStripXBytes;
    static constexpr int XS = XS_FIT > 6 ? 6 : XS_FIT;  // staged units
    static_assert(XS >= WGS + 2, "units in the epilogue and two loading");
    static constexpr int OFF_IMG = XS * kStripXBytes;
    static constexpr int OFF_TAB = OFF_IMG + kStripImg;
    static constexpr int OFF_BAR = OFF_TAB + 4 * T_END;
    static constexpr size_t SMEM = OFF_BAR + kStripBars;
};

// How a signal is cut into strips.
struct StripCut {
    long long n_rows;
    int strip_rows;    // rows per strip (the last strip may be shorter)
    int n_strips;      // strips = thread blocks
    int warm_rows;     // rows a strip starts early
};

// A signal of n samples in strips, at most one per SM.  A signal of one unit is one strip; a strip is at
// least half a unit, and no shorter than its warm-up, so that a warm-up reaches into one neighbour only.
// False where strips are not taken: the cascade remembers for longer than a strip is (its warm-up would
// then cost as much as the strip; two units of it are taken even so, since they cost less than a chain of
// lookbacks).
inline bool strip_cut(long long n, int warm_rows, StripCut &c) {
    static std::atomic<int> known[64];  // SMs of a device, 0: not asked yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    int sms = known[dev].load(std::memory_order_relaxed);
    if (!sms) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return false;
        known[dev].store(sms, std::memory_order_relaxed);
    }
    if (sms > kStripMax) sms = kStripMax;
    c.n_rows = (n + kStripN - 1) / kStripN;
    c.warm_rows = warm_rows;
    long long per = (c.n_rows + sms - 1) / sms;
    if (per > (1LL << 30)) return false;
    const long long most = per > 2 * kStripRows ? per : 2 * kStripRows;
    if (c.n_rows <= kStripRows) {
        per = c.n_rows;
        c.warm_rows = 0;
    } else {
        if (warm_rows < 1 || warm_rows > most) return false;
        if (per < kStripRows / 2) per = kStripRows / 2;
        if (per < warm_rows) per = warm_rows;
    }
    c.strip_rows = static_cast<int>(per);
    c.n_strips = static_cast<int>((c.n_rows + per - 1) / per);
    return true;
}

// One or two sections: strips of at most this many rows with their warm-up take the terminal states by FMAs
// (no operands, products or tensor memory on the way: a 4096-sample call is 0.6 of the time in the kernel),
// longer ones on the tensor cores (2^28 samples at order 2: 329 us against 354).
constexpr int kStripFmaRows = 4 * kStripRows;

template <int K, bool TC>
struct StripParams {
    LaneParams<K> p;
    StripCut cut;
    int in_place;      // y == x: a strip's tail is stored once the next strip has read it
    int x_aligned, y_aligned;  // 16-byte aligned
    unsigned long long host_tickets;  // what the host adds to the lookback kernels' ticket base
    float g[TC ? 1 : 2 * K][kStripN];  // without the tensor cores: the state responses
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

// The sections' recurrences over one row (64 samples, in place) from the row's true incoming state st
// (transposed direct form II), sections skewed by one sample each and in direct-form-I order as in
// lane_particular: a state word z1, z2 enters its section's input at the section's samples 0 and 1.
// Chunk j (four samples) of the row lies at half j / 8, 16-byte slot (j ^ row) & 7; `row` is the offset
// of chunk 0 in the shared memory sm.  Unrolled by U chunks: with U = 8 the whole row, so that a short signal's few warps overlap
// the loads and stores with the dependent FMAs of a step (one section, one warp per scheduler: 1000 cycles
// a row instead of 2800); with U = 1 the code stays small where every scheduler has work (unrolling by 2 to
// 8 cost 7 to 17 % at orders 2 to 16 on 2^26 samples and more, in instruction fetches).
template <int K, bool NORM, int U, class Secs>
__device__ __forceinline__ void lane_recurrence(const Secs &cs, unsigned char *sm, unsigned row, float gain,
                                                const float (&st)[2 * K]) {
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
    unsigned long long full[XS], xfree[XS], afull[2], afree[2], dfull[kStripDS], dfree[kStripDS], zready[kStripZ], fin;
    unsigned tmem, strip, last, pad;
};

template <int K, bool NORM, bool TC>
__global__ void __launch_bounds__(StripDims<K, TC>::THREADS, 1)
    sos_strip_kernel(const __grid_constant__ StripParams<K, TC> P) {
    using Sd = StripDims<K, TC>;
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
        bars.strip = P.in_place && P.cut.n_strips > 1 ? P.cut.n_strips - 1 - atomicAdd(&tail->ticket, 1u) : blockIdx.x;
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
        mbar_init(&bars.fin, 1);
    }
    if (Sd::TC && warp == 1) tc_alloc512(&bars.tmem);
    if (Sd::TC) tc_fence_before();
    __syncthreads();
    if (Sd::TC) tc_fence_after();
    const unsigned tmem = Sd::TC ? bars.tmem : 0;
    const int strip = static_cast<int>(bars.strip);
    const long long r_own = static_cast<long long>(strip) * P.cut.strip_rows;
    const long long r_end = r_own + P.cut.strip_rows < P.cut.n_rows ? r_own + P.cut.strip_rows : P.cut.n_rows;
    const int n_warm = r_own < P.cut.warm_rows ? static_cast<int>(r_own) : P.cut.warm_rows;
    // units of 128 rows from r_first on; rows r_first .. r_own - 1 only warm up, rows past r_end are zeros
    const long long r_first = r_own - n_warm;
    const unsigned n_u = static_cast<unsigned>((r_end - r_first + kStripRows - 1) / kStripRows);
    // phase trace (diagnostics; nothing is written without a trace buffer): one item per unit, strip by strip
    const long long item0 = strip * ((static_cast<long long>(P.cut.strip_rows) + P.cut.warm_rows + kStripRows - 1) / kStripRows);
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
            for (int i = k; i < kStripImg / 16; i += step) dst[i] = __ldg(src + i);
        }
        for (int i = k; i < 32 * MS / 4; i += step)
            reinterpret_cast<float4 *>(sML)[i] = __ldg(reinterpret_cast<const float4 *>(p.tab) + i);
        for (int i = k; i < 4 * S * S; i += step) sACp[i] = __ldg(p.tab + Dm::OFF_ACP + i);
        if (Sd::TC) fence_proxy_async_smem();  // the G image is read by the tensor cores
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
        for (unsigned i = 0; i < n_u; ++i) {
            const unsigned xs = i % XS;
            if (i >= XS && !strip_wait(&xfree[xs], (i / XS - 1) & 1, budget, p.status)) break;
            const long long base = (r_first + static_cast<long long>(i) * kStripRows) * kStripN;
            const long long avail = (r_end * kStripN < p.n ? r_end * kStripN : p.n) - base;
            const float *x = p.x + base;
            const unsigned dst = smem_u32(sm) + xs * kStripXBytes;
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
    } else if (Sd::TC && warp == 1) {
        // ------------------------------------------------------------------ products
        load_tables();
        if (lane == 0) {
            constexpr unsigned i32 = tc_idesc(32), i16 = tc_idesc(16);
            const unsigned g = smem_u32(sm + Sd::OFF_IMG);
            for (unsigned i = 0; i < n_u; ++i) {
                const unsigned ds = i % kStripDS, b = i & 1;
                if (i >= kStripDS && !strip_wait1(&dfree[ds], (i / kStripDS - 1) & 1, budget, p.status)) break;
                if (!strip_wait1(&afull[b], (i >> 1) & 1, budget, p.status)) break;
                tc_fence_after();
                trace(i, 17);
                const unsigned d = tmem + ds * kStripCols, xa = tmem + kStripACol + b * 128, lo = xa + 64;
                // x [G_hi | G_lo]: columns 0..31 over the first half of the row, 32..63 over the second; the
                // remainder's products join the small terms, columns 16..31
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const unsigned gk = g + (k >> 2) * (kStripImg / 2) + (k & 3) * 32;
                    tc_mma_ts(d + 32 * (k >> 2), xa + 8 * k, tc_sdesc(gk), i32, (k & 3) ? 1u : 0u);
                    tc_mma_ts(d + 16, lo + 8 * k, tc_sdesc(gk), i16, 1u);
                    tc_mma_ts(d + 16, lo + 8 * k, tc_sdesc(gk + 16 * 128), i16, 1u);
                }
                tc_commit(&afree[b]);
                tc_commit(&dfull[ds]);
                trace(i, 18);
            }
            // every product issued has completed before tensor memory is released
            tc_commit(&bars.fin);
            strip_wait1(&bars.fin, 0, kStripDrain, p.status);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ operands of the products
        load_tables();
        const int r = 32 * (warp - 4) + lane;  // row within the unit
        const unsigned ta = tmem + kStripACol + (static_cast<unsigned>(32 * (warp - 4)) << 16);
        // the remainder x - (upper 19 bits of x) is exact in 13 bits; half a unit of the 11 the tensor
        // core reads is added to its magnitude, so that the cut rounds to nearest
        auto rem = [](float x) {
            const float e = x - __uint_as_float(__float_as_uint(x) & 0xffffe000u);
            return __uint_as_float(__float_as_uint(e) + 0x1000u);
        };
        for (unsigned i = 0; i < n_u; ++i) {
            const unsigned xs = i % XS, b = i & 1;
            if (!strip_wait(&full[xs], (i / XS) & 1, budget, p.status)) break;
            if (warp == 4) trace(i, 1);
            if (P.in_place && warp == 4 && lane == 0 && n_warm > 0 && static_cast<int>(i) == (n_warm - 1) / kStripRows) {
                __threadfence();
                atomicExch(&tail->flag[strip], 1u);  // the warm-up samples have been read
            }
            if (i >= 2 && !strip_wait(&afree[b], ((i >> 1) - 1) & 1, budget, p.status)) break;
            tc_fence_after();
            if (warp == 4) trace(i, 2);
            const unsigned char *X = sm + xs * kStripXBytes + r * 128;
            const unsigned t0 = ta + b * 128;
#pragma unroll 2
            for (int j = 0; j < 8; ++j) {  // eight samples at a time
                const unsigned char *h = X + (j >> 2) * kStripHalf;
                const int c = 2 * (j & 3);
                const float4 u = *reinterpret_cast<const float4 *>(h + ((c ^ (r & 7)) << 4));
                const float4 v = *reinterpret_cast<const float4 *>(h + (((c + 1) ^ (r & 7)) << 4));
                tc_st8(t0 + 8 * j, u, v);
                tc_st8(t0 + 64 + 8 * j, make_float4(rem(u.x), rem(u.y), rem(u.z), rem(u.w)),
                       make_float4(rem(v.x), rem(v.y), rem(v.z), rem(v.w)));
            }
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull[b]);
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
        float *zv = tabs + Sd::T_ZV + (wg * 4 + q) * S;
        const int li = lane < S ? lane : 0;
        bool dead = false;
        unsigned par = 0;
        for (unsigned i = wg; i < n_u; i += WGS, par ^= 1) {
            const unsigned ds = i % kStripDS, xs = i % XS;
            float *ab = tabs + Sd::T_A + (wg * 2 + par) * 4 * S;
            float Sl[S];
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
                    float a0[C], a1[C];
                    tc_ldn<C>(tl + ds * kStripCols + 16, a0);  // the small terms
                    tc_ldn<C>(tl + ds * kStripCols + 48, a1);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < S; ++j) t[j] = a0[j] + a1[j];
                    tc_ldn<C>(tl + ds * kStripCols, a0);
                    tc_ldn<C>(tl + ds * kStripCols + 32, a1);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < S; ++j) t[j] = (a0[j] + a1[j]) + t[j];
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&dfree[ds]);
                }
                if (q == 0) trace(i, 5);
                lane_scan<K>(cs, t, Sl, ab + q * S, lane);
                if (q == 0) trace(i, 7);
            }
            if (!named_bar_and(1 + wg, 128, ok)) break;
            // the fold's prefix p_v (carry of the groups before this warp's under zero state), then, once
            // the unit's incoming state is known, the group's: Z_v = (A_C)^v Z + p_v
            float pv = 0.f;
            if (q >= 1) pv = ab[li];
#pragma unroll 1
            for (int v = 1; v < q; ++v) pv = lane_mv<S>(sACp, pv, lane) + ab[v * S + li];
            float cu = 0.f;
            if (q == 3) cu = lane_mv<S>(sACp, pv, lane) + ab[3 * S + li];
            if (!strip_wait(&zready[i % kStripZ], (i / kStripZ) & 1, budget, p.status)) {
                dead = true;
                continue;
            }
            if (q == 0) trace(i, 9);
            const float z0 = z_buf[(i % kStripZ) * S + li];
            if (q == 3) {
                const float zn = lane_mv<S>(sACp + 3 * S * S, z0, lane) + cu;
                if (i + 1 < n_u) {
                    if (lane < S) z_buf[((i + 1) % kStripZ) * S + lane] = zn;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&zready[(i + 1) % kStripZ]);
                } else if (__any_sync(0xffffffffu, !(fabsf(zn) <= 3.402823466e38f)) && lane == 0 && strip + 1 < P.cut.n_strips) {
                    atomicMax(&tail->poison, static_cast<unsigned>(P.cut.n_strips - strip));
                }
            }
            if (R + 32 > r_own && R < r_end) {
                const float zq = q == 0 ? z0 : lane_mv<S>(sACp + (q - 1) * S * S, z0, lane) + pv;
                if (lane < S) zv[lane] = zq;
                __syncwarp();
                float st[S];
#pragma unroll
                for (int j = 0; j < S; ++j) st[j] = Sl[j];
                lane_state_mv<K>(sML + lane * MS, zv, st);
                unsigned char *X = sm + xs * kStripXBytes;
                if (q == 0) trace(i, 10);
                if (p.zf && r_end == P.cut.n_rows && R + 32 >= r_end) {
                    // final state: the last row's samples under zero state, taken across the lanes, plus
                    // the transition of the row's incoming state over them
                    const int lane_last = static_cast<int>(P.cut.n_rows - 1 - R);
                    const int ml = p.m_last, rl = 32 * q + lane_last;
                    float acc[S], zt[S];
                    {
                        const float *gt = p.gtail + (kStripN - 1 - ml);
                        const float xa = lane <= ml ? *reinterpret_cast<const float *>(X + tc_swz(rl, lane)) : 0.f;
                        const float xb =
                            lane + 32 <= ml ? *reinterpret_cast<const float *>(X + kStripHalf + tc_swz(rl, lane)) : 0.f;
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
                        float *zf = P.cut.n_strips > 1 ? tail->zf : p.zf;
#pragma unroll
                        for (int s = 0; s < S; ++s) zf[s] = (acc[s] + zt[s]) * p.sec[s >> 1].zscale_inv;
                    }
                    __syncwarp();
                }
                lane_recurrence<K, NORM, Sd::U>(cs, sm, xs * kStripXBytes + r * 128 + ((r & 7) << 4), p.gain, st);
                __syncwarp();
                if (q == 0) trace(i, 11);
                if (P.in_place && strip + 1 < P.cut.n_strips && R + 32 > r_end - P.cut.warm_rows) {
                    const long long t0 = clock64();
                    bool seen = false, late = false;
                    while (!seen && !late) {
                        seen = ld_acquire_u32(&tail->flag[strip + 1]) != 0;
                        late = clock64() - t0 > budget;
                    }
                    if (!__all_sync(0xffffffffu, seen)) {
                        if (lane == 0) atomicOr(p.status, kDevErrTimeout);
                        dead = true;
                        continue;
                    }
                }
                // the group's own samples: from .. to - 1, counted from its first row
                const long long base = R * kStripN;
                const int from = R < r_own ? static_cast<int>(r_own - R) * kStripN : 0;
                const long long own_end = r_end * kStripN < p.n ? r_end * kStripN : p.n;
                const int to = own_end - base < 32 * kStripN ? static_cast<int>(own_end - base) : 32 * kStripN;
                float *y = p.y + base;
                const unsigned char *Xw = X + 32 * q * 128;
                if (P.y_aligned) {
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
                        for (int j = 0; j < 16; ++j) {
                            const int k = k0 + 2 * j * kStripN;
                            const float4 v = get(j);
                            if (k >= from && k + 4 <= to) {
                                __stcs(reinterpret_cast<float4 *>(y + k), v);
                            } else if (k >= from) {
                                if (k + 0 < to) y[k] = v.x;
                                if (k + 1 < to) y[k + 1] = v.y;
                                if (k + 2 < to) y[k + 2] = v.z;
                            }
                        }
                    }
                } else {
#pragma unroll 8
                    for (int j = 0; j < kStripN; ++j) {
                        const int rr = j >> 1, k = 32 * j + lane;
                        const float v = *reinterpret_cast<const float *>(Xw + (j & 1) * kStripHalf + tc_swz(rr, lane));
                        if (k >= from && k < to) __stcs(y + k, v);
                    }
                }
                __syncwarp();
            }
            if (lane == 0) mbar_arrive(&xfree[xs]);
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
    }
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
    if (P.cut.n_strips == 1) return;
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
        const long long from = static_cast<long long>(P.cut.n_strips - poison + 1) * P.cut.strip_rows * kStripN;
        for (long long k = from + tid; k < p.n; k += Sd::THREADS) p.y[k] = nan;
    }
    if (p.zf && tid < S) p.zf[tid] = poison ? nan : *reinterpret_cast<volatile float *>(&tail->zf[tid]);
    for (int k = tid; k < P.cut.n_strips; k += Sd::THREADS) tail->flag[k] = 0;
    __syncthreads();
    if (tid == 0) tail->ticket = tail->poison = tail->done = 0;
}

}  // namespace sosk

// When a pass goes by strips (sosfilt_strip.cuh) and how its signal is cut: host code, no device.
//
// A strip costs its start (tables, barriers, tensor memory: some 5 us), then its units of 128 rows, warm-up
// included; the lookback kernels a tile's latency, a few hops of the chain, and more work per sample.  So strips
// lose where a signal is short, where the warm-up is a large part of a strip, and where the samples come 4 bytes at
// a time (a misaligned x), which the lookback kernels bear better.  The lines below are where the two were measured
// equal: back-to-back launches, 2^13 to 2^28 samples by half octaves, warm-ups of 4 to 1600 rows and of 0.01 to 1
// strip, each section count, products and recurrences apart.
#pragma once

namespace sosk {

constexpr int kStripN = 64;      // samples per row
constexpr int kStripRows = 128;  // rows per unit of a strip's work (four groups of 32 lanes)
constexpr int kStripMax = 256;   // strips of a run (at most one per SM)

// How a signal is cut into strips.
struct StripCut {
    long long n_rows;
    int strip_rows;    // rows per strip (the last strip may be shorter)
    int n_strips;      // strips = thread blocks
    int warm_rows;     // rows a strip starts early
    bool fma;          // one or two sections: terminal states by FMAs, nothing on the tensor cores
};

// The lines for three and more sections.
struct StripRule {
    // x aligned: the least rows of a signal, with a warm-up of a unit or less and with a longer one.  The general
    // floor of 2048 rows (32 strips of half a unit) is where order 8 breaks even (12.3 us both, recurrences; products
    // 13.3 at 2^17 samples against 12.3 to 14.3 from device to device, 13.3 against 14.3 at 2^18).  Order 6:
    // recurrences 12.3 against 12.4 at 2^18, 10.3 at 2^17; products 13.2 to 14.3 up to 2^20.4 against 12.4 to 13.4,
    // 14.3 against 15.4 at 2^21.  With 200 rows of warm-up (strips of 200 rows and more, so fewer of them): order 8 by
    // products 16.4 against 15.4 at 2^20.6, 16.4 against 16.3 at 2^21.
    int least, least_long;
    // x misaligned: least rows; the rows that a strip's units hold, warm-up included, over its own at most; and the
    // warm-up that signals of less than kStripShortOdd rows may have whatever its share (50 below 4096, except at
    // order 16).  Order 6 by products: 7 units on 862 rows 32.8 us against 34.0, 8 on 862 36.1, 6 on 611 29 against
    // 26.7.  Order 8 by products: 3 on 305 20.5 against 22.4, 4 on 305 23.8, 5 on 514 27.7 against 27.3.  Order 16: 7 on
    // 432 (0.8 units of it warm-up) 33.1 against 35.5, 18 on 1221 76.1 against 75.4.
    int least_odd;
    float units_odd;
    int warm_odd;
};
constexpr int kStripShortOdd = 27500;

inline const StripRule &strip_rule(int K, bool products) {
    static const StripRule rec[] = {{4096, 24576, 45000, 1.26f, 0}, {2048, 4096, 4096, 1.50f, 0},
                                    {2048, 4096, 2048, 1.30f, 100}, {2048, 4096, 2048, 1.60f, 100},
                                    {2048, 4096, 2048, 1.50f, 100}, {2048, 4096, 2048, 1.85f, 100}};
    static const StripRule prod[] = {{24576, 45000, 92000, 1.10f, 0}, {4096, 32768, 45000, 1.26f, 0},
                                     {4096, 8192, 2880, 1.30f, 64},   {2048, 4096, 2880, 1.50f, 100},
                                     {2048, 4096, 2048, 1.85f, 100},  {2048, 4096, 2048, 1.85f, 100}};
    return (products ? prod : rec)[K - 3];
}

// One or two sections: a strip no longer than this many rows and its warm-up's (1600 at most), and any where x is
// misaligned, takes its terminal states by FMAs (no operands, products or tensor memory on the way, and eight warps
// load).  Longer ones on the tensor cores, with TMA.  Order 2: 2^24.5 samples 38.0 us against 40.5, 2^25 51.6 against 50.7 (with 1600
// rows of warm-up 55.5 against 57.9), 2^28 352 against 333; order 4: 2^26 93.5 against 99.1, 2^27 183 against 181.
// Misaligned, 2^28: order 2 431 against 545 (lookback 572), order 4 455 against 593 (636).
inline int strip_fma_rows(int K) { return K == 1 ? 3328 : 12288; }

// Cuts a signal of n samples, for a pass of K sections of the given mode whose state is forgotten after warm_rows
// rows (0: not in time), on a device of `sms` SMs.  odd: x is not 16-byte aligned; tc: the other way would be the
// tensor-core lookback kernel, whose start costs more than the strips' (order 6 at 2^15: 15.8 us against 13.7).
// False where strips are not taken.  A signal of one unit is one strip; a strip is at least half a unit, and no
// shorter than its warm-up, so that a warm-up reaches into one neighbour only.
inline bool strip_cut(int K, bool products, bool odd, bool tc, long long n, int warm_rows, int sms, StripCut &c) {
    if (sms < 1) return false;
    if (sms > kStripMax) sms = kStripMax;
    c.n_rows = (n + kStripN - 1) / kStripN;
    c.warm_rows = warm_rows;
    c.fma = false;
    long long per = (c.n_rows + sms - 1) / sms;
    if (per > (1LL << 30)) return false;
    if (K <= 2 && c.n_rows <= kStripRows) {
        c.strip_rows = static_cast<int>(c.n_rows);
        c.n_strips = 1;
        c.warm_rows = 0;
        c.fma = true;
        return true;
    }
    if (warm_rows < 1) return false;
    const double strip = static_cast<double>(per);
    if (K <= 2) {
        // a warm-up of 192 rows, or 256, costs less than a chain of lookbacks however short the strips (256 rows at
        // order 4, 2^15 samples: 10.2 us against 9.3; 2^18: 10.3 against 11.3).  Strips on the tensor cores meet the
        // lookback kernels at a warm-up of half a strip (2^28 samples at 0.5: order 2 415 us against 416 and 422,
        // order 4 430 against 425 and 491; at 0.4 402 and 414; order 4 at 0.7 461).  By FMAs shorter ones win
        // with one nearly as long as the strip (order 2, 2^24, 0.93: 27.3 against 38.2, misaligned 40.1 against 46.3),
        // misaligned longer ones up to 0.66 (2^24.5: 59.9 against 61.6)
        const bool costly = !tc && c.n_rows > 256 && (K == 2 ? c.n_rows < 4096 : odd && c.n_rows < 16384);
        const int least = costly ? 192 : 256;
        c.fma = odd || per - (warm_rows < 1600 ? warm_rows : 1600) <= strip_fma_rows(K);
        const double share = odd     ? (per <= 2048 ? 0.95 : 0.6)
                             : c.fma ? (per <= 2560 ? 1.0 : 0.5)
                                     : (tc ? 0.4 : K == 1 ? 0.5 : 0.8);
        if (warm_rows > least && warm_rows > share * strip) return false;
    } else {
        const StripRule &r = strip_rule(K, products);
        const int least = odd ? r.least_odd : tc ? 2048 : warm_rows > kStripRows ? r.least_long : r.least;
        if (c.n_rows < least) return false;
        if (odd) {
            const long long units = (per + warm_rows + kStripRows - 1) / kStripRows;
            const int any = c.n_rows >= kStripShortOdd ? 0 : c.n_rows < 4096 && K < 8 && r.warm_odd > 50 ? 50 : r.warm_odd;
            if (warm_rows > any && units * kStripRows > r.units_odd * strip) return false;
        } else if (warm_rows > (per > 2 * kStripRows ? per : 2 * kStripRows) ||
                   (tc && K <= 4 && per > 1024 && warm_rows > 0.7 * strip)) {
            // three and four sections against the tensor-core lookback kernel: even at 0.9 of a strip (2^28, order 6:
            // 457 us against 486 at 0.7, 507 against 484 at 1); the others win with a warm-up as long as the strip
            return false;
        }
    }
    if (per < kStripRows / 2) per = kStripRows / 2;
    if (per < warm_rows) per = warm_rows;
    c.strip_rows = static_cast<int>(per);
    c.n_strips = static_cast<int>((c.n_rows + per - 1) / per);
    return true;
}

}  // namespace sosk

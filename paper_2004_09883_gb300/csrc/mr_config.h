// mr_config.h -- shape of a composite-radix line pass (fft_mr.cuh), decided by
// its length and layout alone: radix schedule, lines per tile, threads, and
// the placement of the exchange buffers in shared memory.  Evaluated at
// compile time by the kernels and at run time by the planner.
#pragma once

namespace fbfft {

constexpr int kMrMaxStages = 4;

// Radices the kernels have.
constexpr int kMrRadices[] = {25, 20, 18, 16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
constexpr int kMrNumRadices = 14;

struct MrSchedule {
    int n;                    // stages, 0: no schedule
    int radix[kMrMaxStages];  // non-increasing (radix-1 copies apart)
};

// The best split of n into `left` non-increasing radices from kMrRadices[from]
// on: the smallest first (largest) radix, then the smallest sum -- the most even
// split.  best.n = 0 until one is found.
constexpr void mr_search(int n, int from, int left, MrSchedule cur, MrSchedule& best, int& best_sum)
{
    if (left == 0) {
        if (n != 1) return;
        int sum = 0;
        for (int i = 0; i < cur.n; ++i) sum += cur.radix[i];
        if (best.n == 0 || cur.radix[0] < best.radix[0] || (cur.radix[0] == best.radix[0] && sum < best_sum)) {
            best = cur;
            best_sum = sum;
        }
        return;
    }
    for (int k = from; k < kMrNumRadices; ++k) {
        if (n % kMrRadices[k]) continue;
        MrSchedule c = cur;
        c.radix[c.n++] = kMrRadices[k];
        mr_search(n / kMrRadices[k], k, left - 1, c, best, best_sum);
    }
}

// Schedule of an L-point line: the fewest stages, then the most even split,
// largest radix first (the first stage's loads wait for global memory: the
// more of them a thread has in flight the better).  A length of one radix ends
// with a radix-1 copy, and on contiguous lines starts with one too, so that
// global accesses stay on consecutive values.
constexpr MrSchedule mr_schedule(int L, bool contiguous)
{
    MrSchedule best{};
    int sum = 0;
    for (int n = 1; n <= kMrMaxStages && best.n == 0; ++n) mr_search(L, 0, n, MrSchedule{}, best, sum);
    if (best.n != 1) return best;
    const int r = best.radix[0];
    MrSchedule s{};
    if (contiguous) s.radix[s.n++] = 1;
    s.radix[s.n++] = r;
    s.radix[s.n++] = 1;
    return s;
}

struct MrConfig {
    int L, io;
    int n;                      // stages (>= 2), 0: the length has no schedule
    int radix[kMrMaxStages];
    int ns[kMrMaxStages];       // product of the radices before stage s
    int T;                      // lines per tile (a power of two where a side is strided)
    int threads;
    int regs;                   // register cap
    // Exchange s (1 <= s < n), written by stage s - 1, read by stage s: value
    // i of line t sits at t row[s] + i + (i / ns[s]) pad[s].  Blocks of ns[s]
    // values are what one group of butterflies writes; the writer's and the
    // reader's index both split along them.
    int pad[kMrMaxStages];
    int row[kMrMaxStages];
    int buf[2];                 // values of the two exchange buffers (exchange s uses s - 1 & 1)
    int ptw;                    // values of the tile's four-step factors, behind them (io 3)
};

constexpr bool mr_in_t(int io) { return io == 1 || io == 3; }
constexpr bool mr_out_t(int io) { return io != 0; }
// Whether stage s maps consecutive threads to consecutive lines of the tile
// (else to consecutive butterflies of a line): where it touches a strided
// side, and between the stages of tiles with a strided output.
constexpr bool mr_tfast(int io, int s) { return s == 0 ? mr_in_t(io) : mr_out_t(io); }

// Shared-memory wavefronts (8-byte words, half a warp at a time, 16 banks) of
// the first 64 threads writing and reading exchange e with rows of `row`.
constexpr int mr_wavefronts(const MrConfig& c, int e, int row)
{
    int total = 0;
    for (int side = 0; side < 2; ++side) {
        const int s = e - 1 + side, LR = c.L / c.radix[s], nb = c.T * LR < 64 ? c.T * LR : 64;
        for (int h = 0; h < nb; h += 16) {
            int count[16] = {}, worst = 0;
            for (int b = h; b < h + 16 && b < nb; ++b) {
                const int t = mr_tfast(c.io, s) ? b % c.T : b / LR, j = mr_tfast(c.io, s) ? b / c.T : b % LR;
                const int at = side ? t * row + j + j / c.ns[e] * c.pad[e]
                                    : t * row + j / c.ns[e - 1] * (c.ns[e] + c.pad[e]) + j % c.ns[e - 1];
                const int n = ++count[at & 15];
                worst = n > worst ? n : worst;
            }
            total += worst;
        }
    }
    return total;
}

constexpr MrConfig mr_config(int L, int io)
{
    MrConfig c{};
    c.L = L, c.io = io;
    const MrSchedule s = mr_schedule(L, io == 0);
    c.n = s.n;
    if (c.n == 0) return c;
    int ns = 1, rmax = 1;
    for (int i = 0; i < c.n; ++i) {
        c.radix[i] = s.radix[i];
        c.ns[i] = ns;
        ns *= s.radix[i];
        rmax = s.radix[i] > rmax ? s.radix[i] : rmax;
    }
    if (io == 0) {
        // Contiguous lines: the line count with the fewest idle lanes in the
        // last warp of a stage, among tiles of up to 2560 values (at least
        // 1000 where the length allows).
        long long best_used = 0, best_all = 1;
        const int tmax = 2560 / L > 1 ? 2560 / L : 1, tmin = (1000 + L - 1) / L < tmax ? (1000 + L - 1) / L : tmax;
        for (int T = tmin; T <= tmax; ++T) {
            long long used = 0, all = 0;
            for (int i = 0; i < c.n; ++i) {
                const int nb = T * (L / c.radix[i]);
                used += (long long)nb * c.radix[i];
                all += (long long)((nb + 31) / 32 * 32) * c.radix[i];
            }
            if (used * best_all > best_used * all) best_used = used, best_all = all, c.T = T;
        }
    } else {
        // A strided side moves rows of T values: 16 (128 bytes) up to 256
        // points, 8 up to 512, 4 (one 32-byte sector) up to 2048, then 2.
        c.T = L <= 256 ? 16 : (L <= 540 ? 8 : (L <= 2048 ? 4 : 2));
    }
    int nbmax = 1;
    for (int i = 0; i < c.n; ++i) {
        const int nb = c.T * (L / c.radix[i]);
        nbmax = nb > nbmax ? nb : nbmax;
    }
    const int rounds = (nbmax + 255) / 256;
    c.threads = ((nbmax + rounds - 1) / rounds + 31) / 32 * 32;
    c.regs = rmax <= 10 ? 64 : (rmax <= 16 ? 80 : (rmax <= 20 ? 96 : 112));
    for (int e = 1; e < c.n; ++e) {
        // Writer: groups of Nw consecutive values, the next group R Nw + pad
        // further on; half a warp covers consecutive groups without a bank
        // met twice when that stride is Nw mod 16 (8-byte words), or, for
        // Nw = 1, odd.  Tiles of 16 lines spread a half-warp over their rows
        // instead and need no pad.  The row stride is the one of 16 with the
        // fewest conflicts.
        const int Nw = c.ns[e - 1], R = c.radix[e - 1], blk = c.ns[e];
        const bool by_rows = c.T >= 16 && mr_tfast(io, e - 1) && mr_tfast(io, e);
        int pad = by_rows ? 0 : (Nw == 1 ? (R % 2 == 0) : ((Nw - Nw * R) % 16 + 16) % 16);
        if (Nw > 1 && pad * 8 > blk) pad = 0;
        c.pad[e] = pad;
        const int ext = L + (L / blk - 1) * pad;
        int row = ext, best = 1 << 30;
        for (int x = 0; x < (c.T > 1 ? 16 : 1); ++x) {
            const int cost = mr_wavefronts(c, e, ext + x);
            if (cost < best) best = cost, row = ext + x;
        }
        c.row[e] = row;
        int& b = c.buf[(e - 1) & 1];
        b = c.T * row > b ? c.T * row : b;
    }
    c.buf[0] = (c.buf[0] + 1) & ~1;
    c.ptw = io == 3 ? c.radix[c.n - 1] * c.T : 0;
    return c;
}

}  // namespace fbfft

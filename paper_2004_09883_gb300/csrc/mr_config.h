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
constexpr MrSchedule mr_schedule(int L, bool contiguous, int max_radix = 25)
{
    MrSchedule best{};
    int sum = 0, from = 0;
    while (kMrRadices[from] > max_radix) ++from;
    for (int n = 1; n <= kMrMaxStages && best.n == 0; ++n) mr_search(L, from, n, MrSchedule{}, best, sum);
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
    int buf[2];                 // values of the two exchange buffers (exchange s uses s - 1 & 1);
                                // buf[1] = 0: every exchange uses buffer 0 (see in_place)
    bool in_place;              // every stage reads all its values before any is written
    // The tile's four-step factors exp(-2 pi i c m / N) of its lines c, behind
    // the buffers (io 3): m = r ns[n-1] for the outputs of a last-stage
    // butterfly, then the two parts of its position j = a + radix[0] b: m = a,
    // m = radix[0] b (three stages and more).  T values each.
    int ptw_a, ptw_b, ptw;      // where m = a and m = radix[0] b start, and all of them
};

constexpr bool mr_in_t(int io) { return io == 1 || io == 3; }
constexpr bool mr_out_t(int io) { return io != 0; }
// Whether stage s maps consecutive threads to consecutive lines of the tile
// (else to consecutive butterflies of a line): where it touches a strided
// side, and between the stages of tiles with a strided output.
constexpr bool mr_tfast(int io, int s) { return s == 0 ? mr_in_t(io) : mr_out_t(io); }

// The first 32 threads writing (side 0) and reading (side 1) exchange e, whose
// pad is set: thread b is on line t[side][b], `at` values into it (mod 16, the
// banks of 8-byte words).  Worked out once for all the row strides tried below: the
// divisions took most of a batched-uneven plan's placement time (327 shapes of
// up to 2048 points 2.0 -> 0.8 ms).
struct MrLanes {
    int nb[2];
    unsigned char t[2][32], at[2][32];
};
constexpr MrLanes mr_lanes(const MrConfig& c, int e)
{
    MrLanes l{};
    for (int side = 0; side < 2; ++side) {
        const int s = e - 1 + side, LR = c.L / c.radix[s], nb = c.T * LR < 32 ? c.T * LR : 32;
        l.nb[side] = nb;
        for (int b = 0; b < nb; ++b) {
            int t = mr_tfast(c.io, s) ? b % c.T : b / LR, j = mr_tfast(c.io, s) ? b / c.T : b % LR;
            if (c.io == 2 && s == 0) t = b / 4 % c.T, j = b / (4 * c.T) * 4 + b % 4;  // column-tile blocks
            const int at = side ? j + j / c.ns[e] * c.pad[e]
                                : j / c.ns[e - 1] * (c.ns[e] + c.pad[e]) + j % c.ns[e - 1];
            l.t[side][b] = (unsigned char)t;
            l.at[side][b] = (unsigned char)(at & 15);
        }
    }
    return l;
}
// Shared-memory wavefronts of these threads with rows of `row` values, half a
// warp at a time; stops counting at `most`.
constexpr int mr_wavefronts(const MrLanes& l, int row, int most)
{
    int total = 0;
    for (int side = 0; side < 2; ++side) {
        for (int h = 0; h < l.nb[side] && total < most; h += 16) {
            int count[16] = {}, worst = 0;
            for (int b = h; b < h + 16 && b < l.nb[side]; ++b) {
                const int n = ++count[(l.t[side][b] * (row & 15) + l.at[side][b]) & 15];
                worst = n > worst ? n : worst;
            }
            total += worst;
        }
    }
    return total;
}

// Place the exchange buffers of a shape whose L, io, n, radix, ns and T are set.
constexpr void mr_place(MrConfig& c)
{
    const int L = c.L;
    for (int e = 1; e < c.n; ++e) {
        // Writer: groups of Nw consecutive values, the next group R Nw + pad
        // further on; half a warp covers consecutive groups without a bank
        // met twice when that stride is Nw mod 16 (8-byte words), or, for
        // Nw = 1, odd.  No pad where that is no better (tiles of 8 lines and
        // more spread a half-warp over their rows).
        const int Nw = c.ns[e - 1], R = c.radix[e - 1], blk = c.ns[e];
        int want = Nw == 1 ? (R % 2 == 0) : ((Nw - Nw * R) % 16 + 16) % 16;
        if (Nw > 1 && want * 8 > blk) want = 0;
        int row = L, best = 1 << 30, best_pad = 0;
        for (int k = 0; k < (want ? 2 : 1); ++k) {
            c.pad[e] = k ? want : 0;
            const int ext = L + (L / blk - 1) * c.pad[e];
            // The row stride: lines of 32 butterflies and more side by side
            // hardly meet, any will do; stages across the lines on both sides
            // want rows an odd multiple of H = 16 / T apart (half a warp holds H
            // positions of T lines); else the one of 16 with the fewest conflicts.
            const bool tw = mr_tfast(c.io, e - 1), tr = mr_tfast(c.io, e);
            const int H = c.T < 16 ? 16 / c.T : 1;
            int x0 = 0, x1 = 1;
            if (tw && tr)
                for (x0 = 0; (ext + x0) % (2 * H) != H;) ++x0;
            else if (c.T > 1 && (tw || tr || L / R < 32 || L / c.radix[e] < 32))
                x1 = 16;
            if (tw && tr) x1 = x0 + 1;
            const MrLanes lanes = mr_lanes(c, e);
            const int least = (lanes.nb[0] + 15) / 16 + (lanes.nb[1] + 15) / 16;  // one wavefront a half-warp
            for (int x = x0; x < x1 && best > least; ++x) {
                const int cost = mr_wavefronts(lanes, ext + x, best);
                if (cost < best) best = cost, best_pad = c.pad[e], row = ext + x;
            }
        }
        c.pad[e] = best_pad;
        c.row[e] = row;
        int& b = c.buf[c.in_place ? 0 : (e - 1) & 1];
        b = c.T * row > b ? c.T * row : b;
    }
    if (c.in_place && c.buf[0] < L * c.T) c.buf[0] = L * c.T;  // the tile itself, as copied in and out
    c.buf[0] = (c.buf[0] + 1) & ~1;
    c.ptw_a = c.T * c.radix[c.n - 1];
    c.ptw_b = c.ptw_a + c.T * c.radix[0];
    c.ptw = c.io != 3 ? 0 : c.ptw_b + (c.n > 2 ? c.T * (c.ns[c.n - 1] / c.radix[0]) : 0);
}

// Registers a thread of a CTA can have: each quarter of an SM holds 16384, and
// the CTA's warps are dealt out to the quarters one by one.
constexpr int mr_reg_cap(int threads) { return 16384 / (32 * ((threads + 127) / 128)) / 8 * 8; }

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
        // points, 8 up to 540, 4 (one 32-byte sector) up to 2048, then 2.
        c.T = L <= 256 ? 16 : (L <= 540 ? 8 : (L <= 2048 ? 4 : 2));
    }
    c.regs = rmax <= 10 ? 48 : (rmax <= 12 ? 56 : (rmax <= 16 ? 64 : (rmax <= 20 ? 80 : 96)));
    if (io == 0 || c.n == 2 || c.T >= 16 || L > 1024) {
        // Contiguous lines, and strided tiles but for those below: straight
        // between global memory and registers, small CTAs, several per SM -- the
        // fewest rounds of 320 threads (strided: 512, or 256 for the long lines'
        // large tiles), then the fewest threads.
        int rounds = 1 << 30;
        for (int th = 64; th <= (io == 0 ? 320 : (L > 1024 ? 256 : 512)); th += 32) {
            int all = 0;
            for (int i = 0; i < c.n; ++i) all += (c.T * (L / c.radix[i]) + th - 1) / th;
            if (all < rounds) rounds = all, c.threads = th;
        }
    } else {
        // Strided tiles of three stages and more, rows of 4 or 8 values: the
        // copy engine moves them, which spares the load and store path one access
        // per 32-byte piece, and every stage works in the tile's own buffer: it
        // reads all its values before any is written, so a thread holds `held`
        // values at once.  One round per stage where 1024 threads reach it (two
        // butterflies held at once spill), then the fewest threads.  10^6 points x
        // 16: 205 -> 134 us with this and the tile's own factors below (1000 x 64
        // grids x 80: 39.6 -> 34.1 us).  Slower this way: tiles of two stages (120 x
        // 150 x 144 x 4: 163 against 146 us), rows of 16 (65610 points x 200, 243-
        // point columns: 127 against 101), and lines above 1024 points, whose tile
        // then has an SM to itself (1500 x 64 grids x 50: 45 against 39).
        int held = 0, cost = 1 << 30;
        for (int th = 64; th <= 1024; th += 32) {
            int most = 0, worst = 0;
            for (int i = 0; i < c.n; ++i) {
                const int q = (c.T * (L / c.radix[i]) + th - 1) / th, h = q * c.radix[i];
                const int w = q > 1 && h > 12 ? h + 8 : h;
                most = h > most ? h : most;
                worst = w > worst ? w : worst;
            }
            if ((2 * most + 28 + 7) / 8 * 8 > mr_reg_cap(th) || worst >= cost) continue;
            cost = worst, held = most, c.threads = th;
        }
        c.in_place = true;
        const int need = (2 * held + 28 + 7) / 8 * 8, cap = mr_reg_cap(c.threads);
        c.regs = need > c.regs ? need : c.regs;
        c.regs = c.regs < cap ? c.regs : cap;
    }
    mr_place(c);
    return c;
}

}  // namespace fbfft

// Host run of the composite-radix line pass (fft_mr.cuh): for every 5-smooth
// length up to 4096 and every layout, the stages of full and ragged tiles
// butterfly by butterfly with the kernel's formulas over mr_config's shape, in
// FP32 with the kernel's own butterflies.  Counts shared-memory slots outside their buffer, slots
// written twice in one exchange, slots read that were not written, outputs
// written not exactly once, and compares every line with the DFT in double.
// Prints: cases, index failures, worst relative L2 error.
#include <cmath>
#include <complex>
#include <cstdio>
#include <utility>
#include <vector>

#include "fft_mr.cuh"
#include "fft_uneven.cuh"

using namespace fbfft;
using cd = std::complex<double>;

static void fft64(std::vector<cd>& x, int sign)
{  // recursive mixed radix by the smallest prime factor
    const int n = (int)x.size();
    if (n == 1) return;
    int p = 2;
    while (n % p) ++p;
    const int m = n / p;
    std::vector<std::vector<cd>> y(p, std::vector<cd>(m));
    for (int i = 0; i < n; ++i) y[i % p][i / p] = x[i];
    for (auto& v : y) fft64(v, sign);
    for (int k = 0; k < n; ++k) {
        cd s = 0;
        for (int a = 0; a < p; ++a) s += y[a][k % m] * std::polar(1.0, sign * 2.0 * M_PI * (double)(a * (long long)k % n) / n);
        x[k] = s;
    }
}

template <bool FWD>
static void dft_any(int R, float2* v)
{
    switch (R) {
    case 2: mr_dft<2, FWD>(v); break;
    case 3: mr_dft<3, FWD>(v); break;
    case 4: mr_dft<4, FWD>(v); break;
    case 5: mr_dft<5, FWD>(v); break;
    case 6: mr_dft<6, FWD>(v); break;
    case 8: mr_dft<8, FWD>(v); break;
    case 9: mr_dft<9, FWD>(v); break;
    case 10: mr_dft<10, FWD>(v); break;
    case 12: mr_dft<12, FWD>(v); break;
    case 15: mr_dft<15, FWD>(v); break;
    case 16: mr_dft<16, FWD>(v); break;
    case 18: mr_dft<18, FWD>(v); break;
    case 20: mr_dft<20, FWD>(v); break;
    case 25: mr_dft<25, FWD>(v); break;
    default: break;
    }
}

// One tile of Tv lines; returns index failures, the worst error in *err.
template <bool FWD>
static long long run_tile(const MrConfig& c, int Tv, double* err)
{
    long long bad = 0;
    const int L = c.L, nst = c.n;
    std::vector<std::vector<float2>> x(Tv, std::vector<float2>(L)), y = x;
    unsigned s = 12345u + (unsigned)(L * 7 + c.io);
    auto rnd = [&]() { s = s * 1664525u + 1013904223u; return (float)(s >> 8) / 8388608.0f - 1.0f; };
    for (auto& l : x)
        for (auto& v : l) v = make_float2(rnd(), rnd());
    std::vector<float2> buf[2] = {std::vector<float2>(c.buf[0]), std::vector<float2>(c.buf[1])};
    std::vector<int> mark[2] = {std::vector<int>(c.buf[0], -1), std::vector<int>(c.buf[1], -1)};
    std::vector<int> wrote(Tv * (size_t)L, 0);
    for (int st = 0; st < nst; ++st) {
        const bool first = st == 0, last = st == nst - 1;
        const bool tf = mr_tfast(c.io, st);
        const int R = c.radix[st], LR = L / R, Ns = c.ns[st];
        const int rb = c.in_place ? 0 : (st - 1) & 1, wb = c.in_place ? 0 : st & 1;
        std::vector<std::pair<long long, float2>> out;  // written once every value of the stage is read
        for (int b = 0; b < c.T * LR; ++b) {
            const int t = tf ? b % c.T : b / LR, j = tf ? b / c.T : b % LR, q = j / Ns, k = j % Ns;
            if (t >= Tv) continue;
            float2 v[25];
            for (int r = 0; r < R; ++r) {
                if (first) {
                    v[r] = x[t][j + r * LR];
                } else {
                    const long long at = (long long)t * c.row[st] + j + q * c.pad[st] + (long long)r * (LR + LR / Ns * c.pad[st]);
                    if (at < 0 || at >= c.buf[rb] || mark[rb][at] != st) { ++bad; continue; }
                    v[r] = buf[rb][at];
                    const cd w = std::polar(1.0, -2.0 * M_PI * (double)((long long)r * k % ((long long)Ns * R)) / ((double)Ns * R));
                    v[r] = twmul<FWD>(v[r], make_float2((float)w.real(), (float)w.imag()));
                }
            }
            dft_any<FWD>(R, v);
            for (int r = 0; r < R; ++r) {
                if (!last) {
                    const int blk = Ns * R + c.pad[st + 1];
                    const long long at = (long long)t * c.row[st + 1] + (long long)q * blk + k + (long long)r * Ns;
                    if (at < 0 || at >= c.buf[wb]) { ++bad; continue; }
                    out.push_back({at, v[r]});
                } else {
                    const int kk = j + r * Ns;
                    if (kk >= L || wrote[t * (size_t)L + kk]++) { ++bad; continue; }
                    y[t][kk] = v[r];
                }
            }
        }
        for (auto& o : out) {
            bad += mark[wb][o.first] == st + 1;
            mark[wb][o.first] = st + 1;
            buf[wb][o.first] = o.second;
        }
    }
    for (int w : wrote) bad += w != 1;
    for (int t = 0; t < Tv; ++t) {
        std::vector<cd> z(L);
        for (int i = 0; i < L; ++i) z[i] = cd(x[t][i].x, x[t][i].y);
        fft64(z, FWD ? -1 : 1);
        double num = 0, den = 0;
        for (int i = 0; i < L; ++i) num += std::norm(cd(y[t][i].x, y[t][i].y) - z[i]), den += std::norm(z[i]);
        *err = std::max(*err, std::sqrt(num / den));
    }
    return bad;
}

int main()
{
    long long cases = 0, bad = 0;
    double err = 0;
    for (int L = 2; L <= 4096; ++L) {
        int n = L;
        for (int p : {2, 3, 5})
            while (n % p == 0) n /= p;
        if (n != 1) continue;
        for (int io = 0; io < 4; ++io) {
            const MrConfig c = mr_config(L, io);
            bad += c.n < 2 || c.n > kMrMaxStages;
            bad += io != 0 && (c.T & (c.T - 1)) != 0;
            bad += c.threads > 1024 || c.threads % 32 != 0 || c.regs > mr_reg_cap(c.threads);
            bad += (c.buf[0] + c.buf[1]) * 8 > 227 * 1024;
            for (int Tv : {c.T, (c.T + 1) / 2, 1}) {
                bad += run_tile<true>(c, Tv, &err);
                if (Tv == 1) bad += run_tile<false>(c, Tv, &err);
                ++cases;
            }
        }
    }
    std::printf("mr_pass %lld %lld %.3e\n", cases, bad, err);
    // rows read from column-tile blocks: every value of every row once, from
    // where the column pass puts it (value n of row k: block n / 2^tl of N1 2^tl
    // values, in it row k's run)
    cases = bad = 0;
    for (int L = 16; L <= 4096; ++L) {
        int n = L;
        for (int p : {2, 3, 5})
            while (n % p == 0) n /= p;
        if (n != 1) continue;
        const MrConfig c = mr_config(L, 2);
        const int R = c.radix[0], LR = L / R;
        for (int tl = 1; tl <= 4; ++tl) {
            if (LR % (1 << tl)) continue;
            const long long N1 = 1000;
            std::vector<int> seen((size_t)c.T * L, 0);
            for (int b = 0; b < c.T * LR; ++b) {
                const int t = (b >> tl) % c.T, j = (b >> tl) / c.T << tl | (b & ((1 << tl) - 1));
                bad += j < 0 || j >= LR;
                const int lo = j & ((1 << tl) - 1);
                for (int r = 0; r < R && j < LR; ++r) {
                    const int v = j + r * LR;
                    bad += (j - lo) * N1 + (t << tl) + lo + (long long)r * LR * N1 !=
                           (v >> tl) * (N1 << tl) + (t << tl) + (v & ((1 << tl) - 1));
                    ++seen[(size_t)t * L + v];
                }
            }
            for (int x : seen) bad += x != 1;
            ++cases;
        }
    }
    std::printf("row_blocks %lld %lld 0\n", cases, bad);
    // the jobs of the batched-uneven kernel: run-time shapes, tiles of few lines
    cases = bad = 0;
    err = 0;
    for (int L = 1; L <= kUnevenMaxLen; ++L) {
        int n = L;
        for (int p : {2, 3, 5})
            while (n % p == 0) n /= p;
        if (n != 1) continue;
        for (int io = 0; io < 4; ++io)
            for (long long C : {1LL, 5LL, 100000LL}) {
                MrConfig c = uneven_shape(L, C, io);
                bad += c.n < 2 || c.n > kMrMaxStages;
                mr_place(c);
                bad += io != 0 && (c.T & (c.T - 1)) != 0;
                bad += c.T < 1 || c.T > kUnevenThreads || (long long)c.T * L > kUnevenCap;
                bad += (c.buf[0] + c.buf[1] + c.ptw) * 8 + 2 * (sizeof(PassDesc) + sizeof(UTile)) + 1024 > 233472 / kUnevenCtas;
                bad += run_tile<true>(c, c.T, &err);
                bad += run_tile<false>(c, (c.T + 1) / 2, &err);
                ++cases;
            }
    }
    std::printf("uneven_jobs %lld %lld %.3e\n", cases, bad, err);
    return 0;
}

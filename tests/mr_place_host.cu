// mr_place_host.cu -- the exchange buffers mr_place picks, against a plain search
// that counts every candidate row's bank conflicts from scratch: the same pads,
// rows and buffer sizes for every length, layout and tile height of the
// composite-radix and batched-uneven kernels, and the time both take.
// Prints: shapes, differing shapes, mr_place us, plain search us.
#include <chrono>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fft_uneven.cuh"

using namespace fbfft;

namespace {

int plain_wavefronts(const MrConfig& c, int e, int row)
{
    int total = 0;
    for (int side = 0; side < 2; ++side) {
        const int s = e - 1 + side, LR = c.L / c.radix[s], nb = c.T * LR < 32 ? c.T * LR : 32;
        for (int h = 0; h < nb; h += 16) {
            int count[16] = {}, worst = 0;
            for (int b = h; b < h + 16 && b < nb; ++b) {
                int t = mr_tfast(c.io, s) ? b % c.T : b / LR, j = mr_tfast(c.io, s) ? b / c.T : b % LR;
                if (c.io == 2 && s == 0) t = b / 4 % c.T, j = b / (4 * c.T) * 4 + b % 4;
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

void plain_place(MrConfig& c)
{
    for (int e = 1; e < c.n; ++e) {
        const int Nw = c.ns[e - 1], R = c.radix[e - 1], blk = c.ns[e];
        int want = Nw == 1 ? (R % 2 == 0) : ((Nw - Nw * R) % 16 + 16) % 16;
        if (Nw > 1 && want * 8 > blk) want = 0;
        int row = c.L, best = 1 << 30, pad = 0;
        for (int k = 0; k < (want ? 2 : 1); ++k) {
            c.pad[e] = k ? want : 0;
            const int ext = c.L + (c.L / blk - 1) * c.pad[e], H = c.T < 16 ? 16 / c.T : 1;
            const bool tw = mr_tfast(c.io, e - 1), tr = mr_tfast(c.io, e);
            int x0 = 0, x1 = 1;
            if (tw && tr) {
                while ((ext + x0) % (2 * H) != H) ++x0;
                x1 = x0 + 1;
            } else if (c.T > 1 && (tw || tr || c.L / R < 32 || c.L / c.radix[e] < 32)) {
                x1 = 16;
            }
            for (int x = x0; x < x1; ++x) {
                const int cost = plain_wavefronts(c, e, ext + x);
                if (cost < best) best = cost, pad = c.pad[e], row = ext + x;
            }
        }
        c.pad[e] = pad;
        c.row[e] = row;
        int& b = c.buf[c.in_place ? 0 : (e - 1) & 1];
        b = c.T * row > b ? c.T * row : b;
    }
    if (c.in_place && c.buf[0] < c.L * c.T) c.buf[0] = c.L * c.T;
    c.buf[0] = (c.buf[0] + 1) & ~1;
}

double now_us()
{
    return std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

}  // namespace

int main()
{
    std::vector<MrConfig> shapes;
    for (int L = 2; L <= 4096; ++L) {
        int m = L;
        for (int p : {2, 3, 5})
            while (m % p == 0) m /= p;
        if (m != 1) continue;
        for (int io = 0; io < 4; ++io) {
            MrConfig c = mr_config(L, io);
            if (c.n) {
                std::memset(c.pad, 0, sizeof(c.pad));
                std::memset(c.row, 0, sizeof(c.row));
                c.buf[0] = c.buf[1] = 0;
                shapes.push_back(c);
            }
            for (int C : {2, 3, 5, 17, 4096})
                if (L <= kUnevenMaxLen && uneven_shape(L, C, io).n >= 2) shapes.push_back(uneven_shape(L, C, io));
        }
    }
    std::vector<MrConfig> a = shapes, b = shapes;
    double best_a = 1e30, best_b = 1e30;
    for (int rep = 0; rep < 5; ++rep) {
        a = shapes, b = shapes;
        double t = now_us();
        for (MrConfig& c : a) mr_place(c);
        const double ta = now_us() - t;
        t = now_us();
        for (MrConfig& c : b) plain_place(c);
        const double tb = now_us() - t;
        best_a = ta < best_a ? ta : best_a, best_b = tb < best_b ? tb : best_b;
    }
    int bad = 0;
    for (size_t i = 0; i < shapes.size(); ++i)
        bad += std::memcmp(a[i].pad, b[i].pad, sizeof(a[i].pad)) != 0 ||
               std::memcmp(a[i].row, b[i].row, sizeof(a[i].row)) != 0 || a[i].buf[0] != b[i].buf[0] ||
               a[i].buf[1] != b[i].buf[1];
    std::printf("%d %d %.1f %.1f\n", (int)shapes.size(), bad, best_a, best_b);
    return 0;
}

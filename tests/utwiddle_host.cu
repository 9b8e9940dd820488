// utwiddle_host.cu -- stage twiddles of the batched-uneven kernel (UTwiddle), on
// the host: for every radix of its schedules and every stage size up to 2048
// points, the factors it forms from the powers it reads (each rounded to FP32, as
// the tables hold them) against exp(-+2 pi i k r / (Ns R)) in FP64.
// Prints: factors checked, wrong ones (off by more than `bound`), the largest error.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fft_uneven.cuh"

using namespace fbfft;

namespace {

long long checked = 0, wrong = 0;
double worst = 0;

template <int R, bool FWD>
void radix(double bound)
{
    const double tau = 6.283185307179586476925286766559;
    for (int Ns = 2; Ns * R <= kUnevenMaxLen; ++Ns) {
        int m = Ns;
        for (int p : {2, 3, 5})
            while (m % p == 0) m /= p;
        if (m != 1) continue;
        for (int k = 0; k < Ns; ++k) {
            UTwiddle<R> tw;
            for (int i = 0; i < tw.N; ++i) {
                const double a = -tau * ((long long)k * tw.power(i) % (Ns * R)) / (Ns * R);
                tw.w[i] = make_float2((float)std::cos(a), (float)std::sin(a));
            }
            float2 v[R];
            for (int r = 0; r < R; ++r) v[r] = make_float2(1.f, 0.f);
            tw.template apply<FWD>(v);
            for (int r = 0; r < R; ++r) {
                const double a = (FWD ? -tau : tau) * ((long long)k * r % (Ns * R)) / (Ns * R);
                const double e = std::hypot(v[r].x - std::cos(a), v[r].y - std::sin(a));
                ++checked;
                wrong += !(e <= bound);
                worst = e > worst ? e : worst;
            }
        }
    }
}

}  // namespace

int main(int, char** argv)
{
    const double bound = std::atof(argv[1]);
#define FB_RADIX(R) radix<R, true>(bound), radix<R, false>(bound)
    FB_RADIX(2), FB_RADIX(3), FB_RADIX(4), FB_RADIX(5), FB_RADIX(6), FB_RADIX(8), FB_RADIX(9), FB_RADIX(10), FB_RADIX(12),
        FB_RADIX(15), FB_RADIX(16);
    std::printf("%lld %lld %.3e\n", checked, wrong, worst);
    return 0;
}

// fft_mr.cuh -- the line pass of large composite radices (up to 25): any
// 5-smooth length up to 4096 in two or three Stockham stages (two lengths take
// four), specialised at compile time on length and layout (mr_config.h).
//
// One CTA takes one tile of T lines.  The first stage's threads load their
// butterflies straight from global memory, the stages exchange through one or
// two shared-memory buffers, the last stage stores to global memory (with the
// four-step twiddle and the 1/N scale).  There is no landing buffer and no
// copy-engine traffic, so any alignment and stride takes the same path, and
// several small CTAs per SM overlap one another's loads, stages and stores.
//
// What bounds it: instruction issue first (the kernels before it spent 160-200
// thread instructions per value on four or five small run-time radices; these
// spend 50-60), then the memory system: 1000-point lines x 20001 148.4 -> 66.6
// us (4.8 TB/s, 0.71 of the copy rate), the passes of a 120 x 150 x 144 x 4
// volume 103-127 -> 26-32 us each (5.2-6.3 TB/s).  Large radices cut the shared-
// memory round trips and the twiddle multiplies to one or two per value; a
// run-time-strided form of the same stages needed 75 instructions and 96
// registers (83 us on the 1000-point lines), which is why the length is a
// template parameter.  Power-of-two lengths stay on fft_p2.cuh, whose copy-engine
// tiles measured faster there (4096 x 16384 173 against 224 us).
#pragma once

#include "fft_device.cuh"
#include "mr_config.h"

namespace fbfft {

// ---------------------------------------------------------------------------
// Composite butterflies.  N1 and N2 coprime: the prime-factor (Good-Thomas)
// map n = N2 n1 + N1 n2, k = (N2 u k1 + N1 v k2) mod N with u = N2^-1 mod N1,
// v = N1^-1 mod N2 turns an N1 N2-point DFT into N2 DFTs of N1 points and N1
// of N2 points with no factors between them.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int mr_inv_mod(int a, int m)
{
    for (int x = 1; x < m; ++x)
        if ((a % m) * x % m == 1) return x;
    return 1;
}
template <int R, bool FWD>
__host__ __device__ __forceinline__ void mr_dft(float2* v);

template <int N1, int N2, bool FWD>
__host__ __device__ __forceinline__ void mr_pfa(float2* v)
{
    constexpr int N = N1 * N2;
    constexpr int U = mr_inv_mod(N2, N1) * N2, V = mr_inv_mod(N1, N2) * N1;
    float2 y[N];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
        float2 a[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) a[n1] = v[(N2 * n1 + N1 * n2) % N];
        mr_dft<N1, FWD>(a);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) y[k1 * N2 + n2] = a[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
        float2 a[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) a[n2] = y[k1 * N2 + n2];
        mr_dft<N2, FWD>(a);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) v[(U * k1 + V * k2) % N] = a[k2];
    }
}

// 9 = 3 x 3: n = 3 n1 + n2, k = k1 + 3 k2, factors w9^{n2 k1} between.
template <bool FWD>
__host__ __device__ __forceinline__ void mr_dft9(float2* v)
{
    // cos / sin of 2 pi m / 9, m = 1, 2, 4
    constexpr float C1 = 0.76604444311897803520f, S1 = 0.64278760968653932632f;
    constexpr float C2 = 0.17364817766693034885f, S2 = 0.98480775301220805936f;
    constexpr float C4 = -0.93969262078590838405f, S4 = 0.34202014332566873304f;
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) dft3<FWD>(v[n2], v[3 + n2], v[6 + n2]);
    // v[3 k1 + n2]
    v[4] = rot<FWD>(v[4], C1, S1);
    v[5] = rot<FWD>(v[5], C2, S2);
    v[7] = rot<FWD>(v[7], C2, S2);
    v[8] = rot<FWD>(v[8], C4, S4);
    dft3<FWD>(v[0], v[1], v[2]);
    dft3<FWD>(v[3], v[4], v[5]);
    dft3<FWD>(v[6], v[7], v[8]);
    // v[3 k1 + k2] holds Y[k1 + 3 k2]: transpose
    float2 t;
    t = v[1], v[1] = v[3], v[3] = t;
    t = v[2], v[2] = v[6], v[6] = t;
    t = v[5], v[5] = v[7], v[7] = t;
}

// 25 = 5 x 5, the same scheme.
template <bool FWD>
__host__ __device__ __forceinline__ void mr_dft25(float2* v)
{
    // cos / sin of 2 pi m / 25 for m = n2 k1 in {1, 2, 3, 4, 6, 8, 9, 12, 16}
    constexpr float C[17] = {1.f, 0.96858316112863108f, 0.87630668004386361f, 0.72896862742141155f,
                             0.53582679497899666f, 0.f, 0.062790519529313374f, 0.f, -0.42577929156507272f,
                             -0.63742398974868975f, 0.f, 0.f, -0.99211470131447788f, 0.f, 0.f, 0.f,
                             -0.63742398974868952f};
    constexpr float S[17] = {0.f, 0.24868988716485479f, 0.48175367410171532f, 0.68454710592868862f,
                             0.84432792550201508f, 0.f, 0.99802672842827156f, 0.f, 0.90482705246601958f,
                             0.77051324277578925f, 0.f, 0.f, 0.12533323356430426f, 0.f, 0.f, 0.f,
                             -0.77051324277578936f};
    float2 y[25];
#pragma unroll
    for (int n2 = 0; n2 < 5; ++n2) {
        float2 a[5];
#pragma unroll
        for (int n1 = 0; n1 < 5; ++n1) a[n1] = v[5 * n1 + n2];
        dft5<FWD>(a);
#pragma unroll
        for (int k1 = 0; k1 < 5; ++k1)
            y[5 * k1 + n2] = (n2 * k1) ? rot<FWD>(a[k1], C[n2 * k1], S[n2 * k1]) : a[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < 5; ++k1) {
        dft5<FWD>(y + 5 * k1);
#pragma unroll
        for (int k2 = 0; k2 < 5; ++k2) v[k1 + 5 * k2] = y[5 * k1 + k2];
    }
}

template <int R, bool FWD>
__host__ __device__ __forceinline__ void mr_dft(float2* v)
{
    if constexpr (R == 6) mr_pfa<2, 3, FWD>(v);
    else if constexpr (R == 18) mr_pfa<2, 9, FWD>(v);
    else if constexpr (R == 9) mr_dft9<FWD>(v);
    else if constexpr (R == 10) mr_pfa<2, 5, FWD>(v);
    else if constexpr (R == 12) mr_pfa<4, 3, FWD>(v);
    else if constexpr (R == 15) mr_pfa<3, 5, FWD>(v);
    else if constexpr (R == 20) mr_pfa<4, 5, FWD>(v);
    else if constexpr (R == 25) mr_dft25<FWD>(v);
    else if constexpr (R > 1) dft<R, FWD>(v);
}

#ifdef __CUDACC__

// Streamed global accesses: every value is read and written once per pass, so
// its lines leave L1 first (the twiddle tables stay), with the pass's L2 policy.
__device__ __forceinline__ float2 mr_ldg(const float2* p, unsigned long long pol)
{
    float2 v;
    asm volatile("ld.global.L1::evict_first.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;"
                 : "=f"(v.x), "=f"(v.y)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ void mr_stg(float2* p, float2 v, unsigned long long pol)
{
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(v.x), "f"(v.y), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ unsigned long long l2_evict_normal_policy()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// exp(-2 pi i m / N) from the split four-step tables (m < N < 2^31).
__device__ __forceinline__ float2 mr_ptw(const PassDesc& d, unsigned m)
{
    return cmul(__ldg(d.ptw_hi + (m >> d.ptw_log)), __ldg(d.ptw_lo + (m & ((1u << d.ptw_log) - 1))));
}

template <int L, int IO>
struct Mr {
    static constexpr MrConfig c = mr_config(L, IO);
    static constexpr bool IN_T = mr_in_t(IO), OUT_T = mr_out_t(IO);
    static_assert(c.n >= 2, "no schedule");
};

// Stage S of the tile whose first line starts at gin / gout.
template <bool FWD, int L, int IO, int S>
__device__ __forceinline__ void mr_stage(const PassDesc& d, const float2* gin, float2* gout, float2* buf0,
                                         float2* buf1, float2* ptw, int Tv, int c0, unsigned long long pol)
{
    constexpr MrConfig C = Mr<L, IO>::c;
    constexpr bool first = S == 0, last = S == C.n - 1;
    constexpr bool IN_T = Mr<L, IO>::IN_T, OUT_T = Mr<L, IO>::OUT_T, tfast = first ? IN_T : OUT_T;
    constexpr int R = C.radix[S], LR = L / R, Ns = C.ns[S], TH = C.threads;
    constexpr int NB = C.T * LR, Q = (NB + TH - 1) / TH;  // butterflies of a full tile, rounds
    constexpr int Q1 = first && Q * R <= (C.regs - 32) / 2 ? Q : 1;  // rounds whose loads go out together
    const float2* rd = (S & 1) ? buf0 : buf1;
    float2* wr = (S & 1) ? buf1 : buf0;
    const float2* twb = d.tw + (first ? 0 : d.twoff[S]);
    if constexpr (first && IO == 3) {  // the tile's four-step factors: last stage's r, line t
        constexpr int RL = C.radix[C.n - 1];
        for (int e = threadIdx.x; e < RL * C.T; e += TH)
            if (e % C.T < Tv)  // c < C: the product stays below N
                ptw[e] = mr_ptw(d, (unsigned)(c0 + e % C.T) * (unsigned)(e / C.T * (L / RL)));
    }
    if constexpr (!first) __syncthreads();
#pragma unroll
    for (int q0 = 0; q0 < Q; q0 += Q1) {
        float2 v[Q1][R];
        int t[Q1], j[Q1];
        bool ok[Q1];
#pragma unroll
        for (int u = 0; u < Q1; ++u) {
            const int b = threadIdx.x + (q0 + u) * TH;
            t[u] = tfast ? b % C.T : b / LR;
            j[u] = tfast ? b / C.T : b % LR;
            ok[u] = ((q0 + u + 1) * TH <= NB || b < NB) && t[u] < Tv;
            if (!ok[u]) continue;
            if constexpr (first) {
                const float2* p = IN_T ? gin + (long long)j[u] * d.in_sn + t[u] : gin + t[u] * L + j[u];
                const long long step = IN_T ? LR * d.in_sn : LR;
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = mr_ldg(p + r * step, pol);
            } else {
                constexpr int step = LR + LR / Ns * C.pad[S];
                const float2* p = rd + t[u] * C.row[S] + j[u] + j[u] / Ns * C.pad[S];
                const float2* w = twb + j[u] % Ns;
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = p[r * step];
#pragma unroll
                for (int r = 1; r < R; ++r) v[u][r] = twmul<FWD>(v[u][r], __ldg(w + (r - 1) * Ns));
            }
        }
#pragma unroll
        for (int u = 0; u < Q1; ++u) {
            if (!ok[u]) continue;
            mr_dft<R, FWD>(v[u]);
            if constexpr (!last) {
                constexpr int row = C.row[S + 1], blk = Ns * R + C.pad[S + 1];
                float2* p = wr + t[u] * row + j[u] / Ns * blk + j[u] % Ns;
#pragma unroll
                for (int r = 0; r < R; ++r) p[r * Ns] = v[u][r];
            } else {
                // Ns = L / R: the outputs of butterfly j are j + r Ns
                float2* p = OUT_T ? gout + (long long)j[u] * d.out_sk + t[u] : gout + t[u] * L + j[u];
                const long long step = OUT_T ? Ns * d.out_sk : Ns;
                if constexpr (IO == 3) {
                    // exp(-2 pi i c (j + r Ns) / N) = exp(-2 pi i c j / N), one table
                    // product per butterfly, times exp(-2 pi i c r Ns / N) from the
                    // tile's own table of R values per line
                    const float2 w = mr_ptw(d, (unsigned)(c0 + t[u]) * (unsigned)j[u]);
                    const float2* p4 = ptw + t[u];
                    v[u][0] = twmul<FWD>(v[u][0], w);
#pragma unroll
                    for (int r = 1; r < R; ++r) v[u][r] = twmul<FWD>(v[u][r], cmul(w, p4[r * C.T]));
                }
                if constexpr (!FWD) {
                    if (d.apply_scale) {
#pragma unroll
                        for (int r = 0; r < R; ++r) v[u][r] = d.scale * v[u][r];
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) mr_stg(p + r * step, v[u][r], pol);
            }
        }
    }
}

template <bool FWD, int L, int IO>
__global__ void __maxnreg__((Mr<L, IO>::c.regs)) k_fft_mr(const __grid_constant__ LineArgs a)
{
    extern __shared__ __align__(16) unsigned char mr_smem[];
    constexpr MrConfig C = Mr<L, IO>::c;
    const PassDesc& d = a.d;
    float2* buf0 = reinterpret_cast<float2*>(mr_smem);
    float2* buf1 = buf0 + C.buf[0];
    float2* ptw = buf1 + C.buf[1];
    pdl_start();
    const unsigned long long pin = d.evict_first ? l2_evict_first_policy() : l2_evict_normal_policy();
    const unsigned long long pout = d.evict_last ? l2_evict_last_policy() : l2_evict_normal_policy();
    for (long long tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) {
        // tile = o tiles_per_o + rest: below 2^32 by the reciprocal
        // ceil(2^32 / tiles_per_o), which is at most one too high
        long long o = 0;
        if (d.tpo_mag) {
            o = __umulhi((unsigned)tile, d.tpo_mag);
            if (o * d.tiles_per_o > tile) --o;
        } else if (d.tiles_per_o < d.ntiles) {
            o = tile / d.tiles_per_o;
        }
        const long long c0 = (tile - o * d.tiles_per_o) * d.T;
        const int Tv = d.C - c0 < d.T ? (int)(d.C - c0) : d.T;
        const float2* gin = d.in + o * d.in_so + c0 * d.in_sc;
        float2* gout = d.out + o * d.out_so + c0 * d.out_sc;
        if (tile != blockIdx.x) __syncthreads();  // the last tile's exchange buffers are free
        mr_stage<FWD, L, IO, 0>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0, pin);
        mr_stage<FWD, L, IO, 1>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0, pout);
        if constexpr (C.n > 2) mr_stage<FWD, L, IO, 2>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0, pout);
        if constexpr (C.n > 3) mr_stage<FWD, L, IO, 3>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0, pout);
    }
}

template <bool FWD, int L, int IO>
LineKernel mr_entry()
{
    LineKernel k = make_entry<Mr<L, IO>::c.threads>(k_fft_mr<FWD, L, IO>, FWD, L, IO);
    k.kind = 5;
    return k;
}

#endif  // __CUDACC__

}  // namespace fbfft

// fft_mr.cuh -- the line pass of large composite radices (up to 25): any
// 5-smooth length up to 4096 in two or three Stockham stages (two lengths take
// four), specialised at compile time on length and layout (mr_config.h).
//
// One CTA takes one tile of T lines.  The first stage's threads load their
// butterflies straight from global memory, the stages exchange through one or
// two shared-memory buffers, the last stage stores to global memory (with the
// four-step twiddle and the 1/N scale): any alignment and stride takes the same
// path, and several small CTAs per SM overlap one another's loads, stages and
// stores.  Strided tiles with rows of 4 or 8 values (MrConfig::in_place) move by
// TMA instead where strides and bases allow it, and all their stages work in the
// one buffer they land in.
//
// What bounds it: instruction issue first (the kernels before it spent 160-200
// thread instructions per value on four or five small run-time radices; these
// spend 40-60), then the memory system: 1000-point lines x 20001 148.4 -> 62.6
// us (5.1 TB/s, 0.75 of the copy rate), the six passes of a 120 x 150 x 144 x 4
// volume 694 -> 146 us (6.2-6.7 TB/s a pass).  Large radices cut the shared-memory
// round trips and the twiddle multiplies to one or two per value; a run-time-
// strided form of the same stages needed 75 instructions and 96 registers (83 us
// on the 1000-point lines), which is why the length is a template parameter.
// The narrow strided tiles are bound by latency and the load/store path:
// 10^6 points x 16 266 -> 134 us.  Powers of two share the work with fft_p2.cuh
// (pow2_on_mr in fb_plan.h says which goes where); its warp-specialised tiles stay
// faster on 4096 x 16384 (173 against 201 us), on the four-step passes (2^20 x 32
// 209 against 243-269) and on long strided lines.
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

// Wait for the tile's copies, at most kWaitLimitNs.  One tile per CTA and no cap
// on the grid: once a CTA of the launch has given up (error word), a wait longer
// than any copy takes ends too, or a launch of thousands of tiles whose copies
// cannot arrive would wait the limit once per wave of CTAs.
__device__ __forceinline__ bool mr_wait(unsigned long long* bar, unsigned parity, const int* err)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        const unsigned long long t = global_ns() - t0;
        if (t > kWaitLimitNs || (t > 1000000ULL && *static_cast<const volatile int*>(err) != 0)) return false;
    }
    return true;
}

// exp(-2 pi i m / N) from the split four-step tables (m < N < 2^31).
__device__ __forceinline__ float2 mr_ptw(const PassDesc& d, unsigned m)
{
    return cmul(__ldg(d.ptw_hi + (m >> d.ptw_log)), __ldg(d.ptw_lo + (m & ((1u << d.ptw_log) - 1))));
}

// How a tile's strided sides move: by its threads, by TMA, or by its threads with
// the lines of several outer indices in the tile (PassDesc::fold).  The last is a
// kernel of its own: as a run-time case of the first the line's address cost the
// short strided lines 5 to 19 % (216 points 22.0 -> 26.1 us at 2^23 values).
enum MrMode { kMrPlain = 0, kMrCopied = 1, kMrFold = 2 };

// Where line t of a strided tile starts relative to its first line (so: values
// between outer indices).
template <int MODE>
__device__ __forceinline__ long long mr_line(const PassDesc& d, int t, long long so)
{
    if constexpr (MODE != kMrFold) return t;
    const int o = (int)((unsigned)t * d.fold_mag >> 16);
    return o * so + (t - o * d.fold);
}

template <int L, int IO>
struct Mr {
    static constexpr MrConfig c = mr_config(L, IO);
    static constexpr bool IN_T = mr_in_t(IO), OUT_T = mr_out_t(IO);
    static_assert(c.n >= 2, "no schedule");
};

// Stage S of the tile whose first line starts at gin / gout.  kMrCopied: the strided
// sides of the tile are in buf0 (dense, [position][line]), moved by TMA.
template <bool FWD, int L, int IO, int MODE, int S>
__device__ __forceinline__ void mr_stage(const PassDesc& d, const float2* gin, float2* gout, float2* buf0,
                                         float2* buf1, float2* ptw, int Tv, int c0, unsigned long long pol)
{
    constexpr MrConfig C = Mr<L, IO>::c;
    constexpr bool COPIED = MODE == kMrCopied;
    constexpr bool first = S == 0, last = S == C.n - 1;
    constexpr bool IN_T = Mr<L, IO>::IN_T, OUT_T = Mr<L, IO>::OUT_T, tfast = first ? IN_T : OUT_T;
    constexpr int R = C.radix[S], LR = L / R, Ns = C.ns[S], TH = C.threads;
    constexpr int NB = C.T * LR, Q = (NB + TH - 1) / TH;  // butterflies of a full tile, rounds
    constexpr bool land = first && IN_T && COPIED, back = last && OUT_T && COPIED;
    // rounds whose loads go out together: all of a stage's where it writes the
    // buffer it reads
    constexpr bool shared = C.in_place && (first ? land : (!last || back));
    constexpr int Q1 = shared || (first && Q * R <= (C.regs - 28) / 2) ? Q : 1;
    const float2* rd = (S & 1) || C.in_place ? buf0 : buf1;
    float2* wr = (S & 1) && !C.in_place ? buf1 : buf0;
    const float2* twb = d.tw + (first ? 0 : d.twoff[S]);
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
            if constexpr (first && IO == 2) {
                // rows in column-tile blocks of 2^in_tl values of every row:
                // consecutive threads on a block's consecutive rows
                if (d.in_tl) {
                    t[u] = (b >> d.in_tl) % C.T;
                    j[u] = (b >> d.in_tl) / C.T << d.in_tl | (b & ((1 << d.in_tl) - 1));
                }
            }
            ok[u] = ((q0 + u + 1) * TH <= NB || b < NB) && t[u] < Tv;
            if ((shared || Q1 > 1) && !ok[u]) {
                // defined on every path (loaded and used under one condition,
                // which the register allocator cannot prove)
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = make_float2(0.f, 0.f);
            }
            if (!ok[u]) continue;
            if constexpr (land) {
                const float2* p = buf0 + b;  // (j + r LR) T + t, b = j T + t
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = p[r * LR * C.T];
            } else if constexpr (first) {
                const float2* p = IN_T ? gin + (long long)j[u] * d.in_sn + mr_line<MODE>(d, t[u], d.in_so)
                                       : gin + t[u] * L + j[u];
                long long step = IN_T ? LR * d.in_sn : LR;
                if constexpr (IO == 2) {
                    if (d.in_tl) {
                        const int lo = j[u] & ((1 << d.in_tl) - 1);
                        p = gin + (long long)(j[u] - lo) * d.in_sn + (t[u] << d.in_tl) + lo;
                        step = LR * d.in_sn;
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = mr_ldg(p + r * step, pol);
            } else {
                constexpr int step = LR + LR / Ns * C.pad[S];
                const float2* p = rd + t[u] * C.row[S] + j[u] + j[u] / Ns * C.pad[S];
#pragma unroll
                for (int r = 0; r < R; ++r) v[u][r] = p[r * step];
            }
        }
        if constexpr (shared) __syncthreads();  // every value of the buffer has been read
#pragma unroll
        for (int u = 0; u < Q1; ++u) {
            if (!ok[u]) continue;
            if constexpr (!first) {
                const float2* w = twb + j[u] % Ns;
#pragma unroll
                for (int r = 1; r < R; ++r) v[u][r] = twmul<FWD>(v[u][r], __ldg(w + (r - 1) * Ns));
            }
            mr_dft<R, FWD>(v[u]);
            if constexpr (!last) {
                constexpr int row = C.row[S + 1], blk = Ns * R + C.pad[S + 1];
                float2* p = wr + t[u] * row + j[u] / Ns * blk + j[u] % Ns;
#pragma unroll
                for (int r = 0; r < R; ++r) p[r * Ns] = v[u][r];
            } else {
                // Ns = L / R: the outputs of butterfly j are j + r Ns
                float2* p = OUT_T ? gout + (long long)j[u] * d.out_sk + mr_line<MODE>(d, t[u], d.out_so)
                                  : gout + t[u] * L + j[u];
                const long long step = OUT_T ? Ns * d.out_sk : Ns;
                if constexpr (IO == 3) {
                    // exp(-2 pi i c (j + r Ns) / N): products of the tile's own factors
                    // (one gather per tile entry instead of two per butterfly from
                    // tables of N, which were a quarter of this pass's L1 accesses)
                    constexpr int R0 = C.radix[0];
                    const float2* p4 = ptw + t[u];
                    float2 w = p4[C.ptw_a + j[u] % R0 * C.T];
                    if constexpr (C.n > 2) w = cmul(w, p4[C.ptw_b + j[u] / R0 * C.T]);
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
                if constexpr (back) {
                    const int b = threadIdx.x + (q0 + u) * TH;
#pragma unroll
                    for (int r = 0; r < R; ++r) buf0[b + r * Ns * C.T] = v[u][r];
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) mr_stg(p + r * step, v[u][r], pol);
                }
            }
        }
    }
    if constexpr (first && IO == 3) {  // the tile's four-step factors, behind the stage so that its loads go out first
        constexpr int RL = C.radix[C.n - 1], R0 = C.radix[0];
        for (int e = threadIdx.x; e < C.ptw; e += TH) {
            const int i = e / C.T, t = e % C.T;
            const int m = i < RL ? i * (L / RL) : (i < RL + R0 ? i - RL : (i - RL - R0) * R0);
            if (t < Tv) ptw[e] = mr_ptw(d, (unsigned)(c0 + t) * (unsigned)m);  // c < C: the product stays below N
        }
    }
}

template <bool FWD, int L, int IO, int MODE>
__device__ __forceinline__ void mr_tile(const PassDesc& d, const float2* gin, float2* gout, float2* buf0,
                                        float2* buf1, float2* ptw, int Tv, int c0, unsigned long long pin,
                                        unsigned long long pout)
{
    constexpr int n = Mr<L, IO>::c.n;
    mr_stage<FWD, L, IO, MODE, 0>(d, gin, gout, buf0, buf1, ptw, Tv, c0, pin);
    mr_stage<FWD, L, IO, MODE, 1>(d, gin, gout, buf0, buf1, ptw, Tv, c0, pout);
    if constexpr (n > 2) mr_stage<FWD, L, IO, MODE, 2>(d, gin, gout, buf0, buf1, ptw, Tv, c0, pout);
    if constexpr (n > 3) mr_stage<FWD, L, IO, MODE, 3>(d, gin, gout, buf0, buf1, ptw, Tv, c0, pout);
}

template <bool FWD, int L, int IO, bool FOLD = false>
__global__ void __maxnreg__((Mr<L, IO>::c.regs)) k_fft_mr(const __grid_constant__ LineArgs a)
{
    extern __shared__ __align__(128) unsigned char mr_smem_dyn[];
    constexpr MrConfig C = Mr<L, IO>::c;
    constexpr bool IN_T = Mr<L, IO>::IN_T, OUT_T = Mr<L, IO>::OUT_T;
    const PassDesc& d = a.d;
    // 128 bytes for the barrier, then the buffers, 128-byte aligned for the copies
    unsigned char* mr_smem = mr_smem_dyn + ((128u - (smem_u32(mr_smem_dyn) & 127u)) & 127u);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(mr_smem);
    float2* buf0 = reinterpret_cast<float2*>(mr_smem + 128);
    float2* buf1 = buf0 + C.buf[0];
    float2* ptw = buf1 + C.buf[1];
    const bool copied = !FOLD && C.in_place && d.async_io != 0;
    if constexpr (IN_T) {
        if (copied) {
            if (threadIdx.x == 0) {
                mbar_init(bar, 1);
                fence_mbar_init();
            }
            __syncthreads();
        }
    }
    pdl_start();
    const unsigned long long pin = d.evict_first ? l2_evict_first_policy() : l2_evict_normal_policy();
    const unsigned long long pout = d.evict_last ? l2_evict_last_policy() : l2_evict_normal_policy();
    unsigned phase = 0;
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
        if (tile != blockIdx.x) __syncthreads();  // the last tile's buffers are free (copies: read, below)
        if constexpr (IN_T) {
            if (copied) {
                if (threadIdx.x == 0) {
                    mbar_arrive_expect_tx(bar, (unsigned)(C.T * L) * 8u + d.debug_extra_tx);
                    for (int n0 = 0; n0 < L; n0 += d.box_rows)
                        tma_load_3d(buf0 + n0 * C.T, &a.tm_in, (int)c0, n0, (int)o, bar, d.err, true, pin);
                }
                const bool bad = !mr_wait(bar, phase, d.err);
                if (__syncthreads_or(bad)) {
                    if (threadIdx.x == 0) {
                        atomicExch(d.err, 1);
                        bulk_wait_all();
                        mr_wait(bar, phase, d.err);  // the tile's loads, once more, while its shared memory lives
                    }
                    return;
                }
                phase ^= 1u;
            }
        }
        if (!FOLD && C.in_place && copied)
            mr_tile<FWD, L, IO, !FOLD && C.in_place ? kMrCopied : kMrPlain>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0,
                                                                             pin, pout);
        else
            mr_tile<FWD, L, IO, FOLD ? kMrFold : kMrPlain>(d, gin, gout, buf0, buf1, ptw, Tv, (int)c0, pin, pout);
        if constexpr (OUT_T) {
            if (copied) {
                fence_proxy_async();  // the tile -> visible to the copy engine
                __syncthreads();
                if (threadIdx.x == 0) {
                    if (d.out_blk) {  // column-tile blocks: the tile as it lies here
                        bulk_store_1d(gout, buf0, (unsigned)(C.T * L) * 8u, d.err, true, pout);
                    } else {
                        for (int k0 = 0; k0 < L; k0 += d.box_rows)
                            tma_store_3d(&a.tm_out, (int)c0, k0, (int)o, buf0 + k0 * C.T, d.err, true, pout);
                    }
                    bulk_commit();
                    bulk_wait_read_all();  // before the buffer is written again or the CTA leaves
                }
            }
        }
    }
    if constexpr (OUT_T) {
        if (copied && threadIdx.x == 0) bulk_wait_all();
    }
}

template <bool FWD, int L, int IO, bool FOLD = false>
LineKernel mr_entry()
{
    LineKernel k = make_entry<Mr<L, IO>::c.threads>(k_fft_mr<FWD, L, IO, FOLD>, FWD, L, IO);
    k.kind = 5;
    k.mr = &Mr<L, IO>::c;
    return k;
}
// Strided lines in tiles of several outer indices: lengths whose tiles hold two
// outer indices of two lines and more.
template <bool FWD, int L>
LineKernel mr_fold_entry()
{
    if constexpr (Mr<L, 1>::c.T >= 4)
        return mr_entry<FWD, L, 1, true>();
    else
        return LineKernel{nullptr, 0, false, 0, 0};
}

#endif  // __CUDACC__

}  // namespace fbfft
